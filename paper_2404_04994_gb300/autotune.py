"""Autotuner of the batched ground state: for every group of arrays with the
same dot count and form (open / closed), the pruning threshold t and the team
width (lanes per pixel; pixels per warp = 32 / team) that the batch should use.

Threshold (Sec. III.B; the heuristic of App. F): candidate values below 1 are
1/2, 2 ||Delta||_2 and ||Delta||_F, with Cdd = D (I - Delta), D = diag(Cdd).  A
t < 1 prunes the candidate set and can change the result, so it is admitted
only if it reproduces the t = 1 charge map exactly on every pixel of the
sample rasters of the group; the smallest admitted value wins, else t = 1.
The chosen t is an output of the tuning and the batch is then exact with
respect to the method at that t (the oracle is run at the same t).

Team: the library's own choice (0: for most arrays a search with lanes of its
own) and every power of two from 1 to 32 are timed at the chosen t (CUDA
events, median of a few runs) and the fastest wins.  The sample is repeated
until its pixels fill the GPU, as the batch does: a few small arrays alone time
launches.

The decision logic takes a ``runner(specs, reps) -> (maps, ms)`` so that it can
be exercised on the CPU with a fake; the default runner drives the library's
batched entry point on the current CUDA device.
"""
from __future__ import annotations

import json
import math

import numpy as np

TEAMS = (0, 1, 2, 4, 8, 16, 32)
TIMED_PIXELS = 32768  # about four to each team of lanes the GPU holds


def delta_matrix(Cdd):
    """Delta of Cdd = D (I - Delta): minus the off-diagonal entries divided
    by their row's diagonal entry, zero on the diagonal."""
    Cdd = np.asarray(Cdd, dtype=np.float64)
    D = np.diag(Cdd)
    Dl = -Cdd / D[:, None]
    np.fill_diagonal(Dl, 0.0)
    return Dl


def threshold_candidates(Cdds):
    """Candidate thresholds below 1, ascending, for a group of arrays: 1/2
    and the two norm-based values of App. F, each taken at its largest over
    the group (the most conservative member decides)."""
    spec = max(2.0 * np.linalg.norm(delta_matrix(C), 2) for C in Cdds)
    frob = max(np.linalg.norm(delta_matrix(C), "fro") for C in Cdds)
    cands = {0.5, float(spec), float(frob)}
    return sorted(t for t in cands if 0.0 < t < 1.0)


def sample_spec(spec, side):
    """The same voltage window as ``spec`` at side x side pixels."""
    r = dict(spec["raster"])
    r["W"] = int(side)
    r["H"] = int(side)
    out = dict(spec)
    out["raster"] = r
    return out


def group_key(spec):
    return (int(np.asarray(spec["Cdd"]).shape[0]), bool(spec.get("closed", False)))


def tune(specs, runner=None, sample_side=24, arrays_per_group=4, teams=TEAMS, reps=3):
    """Returns {(N, closed): entry}, entry = {"threshold", "team",
    "arrays" (indices sampled), "rejected" {t: mismatching pixels},
    "team_ms" {team: ms}}."""
    runner = runner or gpu_runner
    groups = {}
    for i, sp in enumerate(specs):
        groups.setdefault(group_key(sp), []).append(i)
    table = {}
    for key in sorted(groups):
        idx = groups[key][:arrays_per_group]
        base = [dict(sample_spec(specs[i], sample_side), threshold=1.0, team=0) for i in idx]
        ref, _ = runner(base, 1)
        chosen, rejected = 1.0, {}
        for t in threshold_candidates([specs[i]["Cdd"] for i in idx]):
            maps, _ = runner([dict(b, threshold=t) for b in base], 1)
            bad = sum(int((m != r).any(axis=-1).sum()) for m, r in zip(maps, ref))
            if bad == 0:
                chosen = t
                break
            rejected[t] = bad
        copies = -(-TIMED_PIXELS // sum(b["raster"]["W"] * b["raster"]["H"] for b in base))
        team_ms = {}
        for T in teams:
            _, ms = runner([dict(b, threshold=chosen, team=T) for b in base] * copies, reps)
            team_ms[T] = ms
        best_team = min(team_ms, key=lambda T: (team_ms[T], T))
        table[key] = {"threshold": chosen, "team": int(best_team), "arrays": idx,
                      "rejected": rejected, "team_ms": team_ms}
    return table


def apply(specs, table):
    """Copies of specs with the tuned threshold and team of their group."""
    out = []
    for sp in specs:
        e = table[group_key(sp)]
        out.append(dict(sp, threshold=e["threshold"], t=e["threshold"], team=e["team"]))
    return out


def to_json(table):
    rows = []
    for (n, closed), e in sorted(table.items()):
        rows.append({"n_dot": n, "closed": closed, "threshold": e["threshold"],
                     "team": e["team"], "arrays": list(e["arrays"]),
                     "rejected": {repr(k): v for k, v in e["rejected"].items()},
                     "team_ms": {str(k): v for k, v in e["team_ms"].items()}})
    return json.dumps(rows, indent=1)


def from_json(text):
    table = {}
    for r in json.loads(text):
        table[(int(r["n_dot"]), bool(r["closed"]))] = {
            "threshold": float(r["threshold"]), "team": int(r["team"]),
            "arrays": r["arrays"], "rejected": r["rejected"], "team_ms": r["team_ms"]}
    return table


def gpu_runner(specs, reps):
    """Runs the sample arrays as one batched call; returns the charge maps
    (host, [H, W, N] each) and the median device time of ``reps`` runs."""
    import torch

    from .api import Batch
    b = Batch(specs)
    try:
        b.run()
        times = []
        for _ in range(max(1, reps)):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record()
            b.run()
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        maps = [o[0].cpu().numpy() for o in b.outputs]
    finally:
        b.close()
    return maps, float(np.median(times)) if times else math.nan
