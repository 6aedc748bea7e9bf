"""Timed cases: the calls a user of this package makes, over the range of
their sizes, options and directions, with FP64 values to hold them against.

A case is a dict of plain values; ``op`` says which call it is:

  ground    charge map of an open or closed array over a gate-voltage raster
  points    the same at a list of random voltage vectors (Sec. VII's benchmark)
  batch     many arrays of uneven size in one prepared batch
  soft      finite-temperature occupation of a raster (Sec. IV.B)
  softgrad  occupation, loss and gradients through torch.autograd
  fit       one fused capacitance-fitting step
  sensor    charge-sensor diagram: ground state of the dots, sensor response
  brute     exhaustive ground state (Table I)

Capacitances, offsets and voltages are drawn from the seed by the recipes of
``inputs.py`` (grids where the dot count is a grid of the paper's kind, chains
otherwise).  ``exact`` restates each call in FP64 with torch and numpy alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2404_04994_gb300 import api, autograd, inputs

GRIDS = {6: (2, 3), 8: (2, 4), 9: (3, 3), 12: (3, 4), 16: (4, 4)}
NOISE = {"width": 0.05, "white_sigma": 0.05, "pink_sigma": 0.03, "jump_amplitude": 0.2,
         "jump_prob": 0.01}
ADAM = {"lr": 2e-3, "beta1": 0.9, "beta2": 0.999, "eps": 1e-8}


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def _case(op, **kw):
    c = {"op": op, "n": 2, "extra_gates": 0, "W": 1, "H": 1, "lo": -1.0, "hi": 6.0, "t": 1.0,
         "closed": False, "n_charges": 0, "carrier": 1.0, "coupling": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest diagram a user tunes a double dot with, called over and
        # over while the voltages move: launches and host work count
        _case("ground", name="open_2dot_100x100", n=2, W=100, H=100),
        # the benchmark diagram of the paper (Sec. VII), open and closed
        _case("ground", name="open_16dot_100x100", n=16, W=100, H=100),
        _case("ground", name="closed_16dot_100x100", n=16, W=100, H=100, closed=True,
              n_charges=16),
        # the thresholded algorithm on a large array, raster of no round size
        _case("ground", name="open_16dot_257x193_t0.5", n=16, W=257, H=193, t=0.5),
        # a mid-size array at high resolution (the exhaustive search's range)
        _case("ground", name="open_12dot_400x301", n=12, W=400, H=301),
        # random voltage vectors, the shape of the paper's Fig. 4 and 5
        _case("points", name="points_16dot_10000", n=16, W=10000),
        # a data set of diagrams: arrays of 2 to 16 dots, open and closed
        _case("batch", name="batch_192_arrays", count=192),
        # thermally broadened diagram
        _case("soft", name="soft_8dot_200x200", n=8, W=200, H=200, kT=0.01),
        # a training step through torch on an array beyond 8 dots
        _case("softgrad", name="softgrad_12dot_75x60", n=12, W=75, H=60, kT=0.05),
        # the capacitance-fitting loop's step
        _case("fit", name="fit_8dot_200x200", n=8, W=200, H=200, kT=0.01),
        # the paper's Fig. 3b diagram: four dots read out by a charge sensor
        _case("sensor", name="sensor_4dot_200x200", n=4, W=200, H=200, n_sensor=1),
        # Table I's exhaustive reference at the size of its four-dot diagram
        _case("brute", name="brute_4dot_200x200_nmax7", n=4, W=200, H=200, n_max=7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _raster_size(rng, most, lo=16, hi=400):
    W, H = _log_int(rng, lo, hi), _log_int(rng, lo, hi)
    while W * H > most:
        W, H = max(lo, int(W * 0.9)), max(lo, int(H * 0.9))
        if W == lo and H == lo:
            break
    return W, H


def draw(rng):
    op = rng.choices(["ground", "points", "batch", "soft", "softgrad", "fit", "sensor", "brute"],
                     [5, 2, 1, 1, 1, 1, 1, 1])[0]
    if op == "ground":
        n = rng.randint(2, 16)
        closed = rng.random() < 0.4
        W, H = _raster_size(rng, 50000 if n > 12 else 120000)
        return _case(op, n=n, W=W, H=H, extra_gates=rng.choice([0, 0, 1, 3]), closed=closed,
                     t=rng.choice([1.0, 1.0, 0.5, round(rng.uniform(0.1, 0.9), 2)]),
                     n_charges=rng.randint(1, 2 * n) if closed else 0,
                     hi=6.0 if closed else rng.choice([6.0, 6.0, 150.0]),
                     carrier=rng.choice([1.0, 1.0, 1.0, -1.0]) if closed else 1.0,
                     coupling=rng.random() < 0.25)
    if op == "points":
        n = rng.randint(2, 16)
        closed = rng.random() < 0.4
        return _case(op, n=n, W=_log_int(rng, 100, 50000 if n <= 12 else 20000),
                     extra_gates=rng.choice([0, 0, 1, 5]), closed=closed,
                     t=rng.choice([1.0, 1.0, 0.5]), n_charges=rng.randint(1, 2 * n) if closed else 0)
    if op == "batch":
        return _case(op, count=_log_int(rng, 6, 192), t=rng.choice([1.0, 1.0, 0.5]))
    if op in ("soft", "softgrad", "fit"):
        n = rng.randint(2, 12)
        closed = op == "soft" and rng.random() < 0.4
        W, H = _raster_size(rng, min(40000, (75 * 60 << 12) >> n), hi=200)
        return _case(op, n=n, W=W, H=H, kT=round(rng.uniform(0.01, 0.05), 3), closed=closed,
                     t=rng.choice([1.0, 1.0, 0.5]) if op == "soft" else 1.0,
                     n_charges=rng.randint(1, n + 2) if closed else 0)
    if op == "sensor":
        W, H = _raster_size(rng, 60000, hi=600)
        return _case(op, n=rng.randint(2, 6), W=W, H=H, n_sensor=rng.randint(1, 2))
    n = rng.randint(2, 5)
    closed = rng.random() < 0.4
    n_max = rng.randint(2, {2: 12, 3: 12, 4: 8, 5: 5}[n])
    W, H = _raster_size(rng, min(40000, int(40000 * 8 ** 4 / (n_max + 1) ** n)), hi=200)
    return _case(op, n=n, W=W, H=H, n_max=n_max, closed=closed)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _rng(seed, k=0):
    return np.random.Generator(np.random.PCG64([seed, k]))


def _matrices(r, n, n_gate, coupling=False):
    Cdd = inputs.grid_cdd(r, *GRIDS[n]) if n in GRIDS else inputs.chain_cdd(r, n, nn=(0.05, 0.25))
    Cgd = inputs.dense_cgd(r, n, n_gate, diag=(0.5, 1.0), off=(0.0, 0.1))
    if coupling:
        Cdd = np.abs(Cdd - np.diag(np.diag(Cdd)))
    return Cdd, Cgd


def _perturbed(r, Cdd, Cgd):
    """Every entry times 1 + U[-10 %, 10 %], Cdd kept symmetric."""
    f = 1.0 + r.uniform(-0.1, 0.1, Cdd.shape)
    f = np.triu(f) + np.triu(f, 1).T
    return Cdd * f, Cgd * (1.0 + r.uniform(-0.1, 0.1, Cgd.shape))


def _raster(r, case, n, n_gate):
    gx, gy = inputs.swept_gates(n)
    V = inputs.offsets(r, n_gate, (gx, gy))
    lo, hi = case["lo"], case["hi"]
    if case["carrier"] < 0:
        V, lo, hi = -V, -hi, -lo
    return inputs.raster(n_gate, gx, gy, V, lo=lo, hi=hi, W=case["W"], H=case["H"])


def _array(case, seed):
    """Cdd, Cgd and the raster of a single-array case."""
    r = _rng(seed)
    n = case["n"] + case.get("n_sensor", 0)
    n_gate = n + case["extra_gates"]
    Cdd, Cgd = _matrices(r, n, n_gate, case["coupling"])
    if case["op"] == "sensor":
        nd = case["n"]  # each sensing dot couples weakly to every dot
        Cdd = np.eye(n)
        Cdd[:nd, :nd] = inputs.chain_cdd(r, nd, nn=(0.1, 0.3))
        Cdd[nd:, :nd] = -r.uniform(0.02, 0.08, (n - nd, nd))
        Cdd[:nd, nd:] = Cdd[nd:, :nd].T
    return Cdd, Cgd, _raster(r, case, case["n"], n_gate)


def _voltages(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    V = torch.rand((case["W"], case["n"] + case["extra_gates"]), dtype=torch.float64,
                   device="cuda", generator=g)
    return case["lo"] + (case["hi"] - case["lo"]) * V


def _specs(case, seed):
    """The arrays of a batch: N ~ U{2..16}, rasters of 64 or 128 pixels a side
    (one side in four of another length), open or closed with N charges."""
    r = _rng(seed)
    rs = _rng(0, case["count"])  # the shapes belong to the case, not to the seed
    out = []
    for _ in range(case["count"]):
        n = int(rs.integers(2, 17))
        side = int(rs.choice([64, 128]))
        H = side if rs.random() < 0.75 else int(rs.integers(33, side))
        closed = bool(rs.integers(0, 2))
        Cdd, Cgd = _matrices(r, n, n)
        gx, gy = inputs.swept_gates(n)
        V = inputs.offsets(r, n, (gx, gy))
        out.append({"Cdd": Cdd, "Cgd": Cgd, "n": n, "closed": closed, "t": case["t"],
                    "n_charges": n if closed else 0,
                    "raster": inputs.raster(n, gx, gy, V, W=side, H=H)})
    return out


def _target(case, seed, Cdd, Cgd, ras):
    """sum_i <n_i> of a perturbed model: what a fit is given."""
    Ct, Gt = _perturbed(_rng(seed, 1), Cdd, Cgd)
    with torch.no_grad():
        mean, _ = _soft(_dev(Ct), _dev(Gt), _raster_volts(ras), 1.0, case["kT"], case["t"],
                        False, 0)
    return mean.sum(1).float()


def prepare(case, seed):
    op = case["op"]
    st = {"case": case, "seed": seed}
    if op == "batch":
        specs = _specs(case, seed)
        st["models"] = [api.Model(s["Cdd"], s["Cgd"]) for s in specs]
        # one buffer for each kind of output, an array's part starting on a
        # 256-byte boundary
        parts, at_n, at_p = [], 0, 0
        for s in specs:
            P = s["raster"]["W"] * s["raster"]["H"]
            parts.append((at_n, at_p, P, P * s["n"]))
            at_n += -(-P * s["n"] // 256) * 256
            at_p += -(-P // 256) * 256
        st["n"] = torch.zeros(at_n, dtype=torch.int8, device="cuda")
        st["U"] = torch.zeros(at_p, dtype=torch.float64, device="cuda")
        st["flags"] = torch.zeros(at_p, dtype=torch.uint8, device="cuda")
        st["handle"] = api.qa_batch_create([
            dict(model=m.handle, raster=s["raster"], threshold=s["t"], closed=s["closed"],
                 n_charges=s["n_charges"], out_n=st["n"][a:a + q], out_U=st["U"][b:b + P],
                 out_flags=st["flags"][b:b + P])
            for m, s, (a, b, P, q) in zip(st["models"], specs, parts)])
        return _Owned(st)
    if op == "points":
        Cdd, Cgd, _ = _array(dict(case, H=1), seed)
        st["model"] = api.Model(Cdd, Cgd)
        st["V"] = _voltages(case, seed)
        return st
    Cdd, Cgd, st["raster"] = _array(case, seed)
    if op == "sensor":
        nd, S = case["n"], case["n_sensor"]
        st["model"] = api.Model(Cdd[:nd, :nd], Cgd[:nd])
        st["full"] = api.Model(Cdd, Cgd)
        shape = (case["H"], case["W"], S)
        st["signal"] = torch.empty(shape, dtype=torch.float32, device="cuda")
        st["n_sensor"] = torch.empty(shape, dtype=torch.int8, device="cuda")
        st["potential"] = torch.empty(shape, dtype=torch.float64, device="cuda")
        st["params"] = dict(NOISE, n_sensor=S, shape=api.QA_SENSOR_LORENTZIAN, seed=seed)
        return st
    st["model"] = api.Model(Cdd, Cgd, form=api.QA_FORM_COUPLING if case["coupling"]
                            else api.QA_FORM_MAXWELL, carrier_sign=case["carrier"])
    if op == "softgrad":
        # the parameters of a torch training loop: FP32 leaves
        for k, v in (("Cdd", Cdd), ("Cgd", Cgd)):
            st[k] = torch.tensor(v, dtype=torch.float32, device="cuda", requires_grad=True)
        st["target"] = _target(case, seed, Cdd, Cgd, st["raster"])
    elif op == "fit":
        for k, v in (("Cdd", Cdd), ("Cgd", Cgd)):
            st[k] = torch.tensor(v, dtype=torch.float64, device="cuda")
        st["target"] = _target(case, seed, Cdd, Cgd, st["raster"])
        st["opt"] = torch.zeros(api.fit_state_len(*Cgd.shape), dtype=torch.float64, device="cuda")
        st["loss"] = torch.zeros((), dtype=torch.float32, device="cuda")
        st["mean"] = torch.empty((case["W"] * case["H"], Cgd.shape[0]), dtype=torch.float32,
                                 device="cuda")
    return st


class _Owned(dict):
    """A prepared batch with its handle, released with the state."""

    def __del__(self):
        torch.cuda.synchronize()
        api.qa_batch_destroy(self["handle"])


# --------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------

def run(st):
    case = st["case"]
    op = case["op"]
    if op == "batch":
        api.qa_batch_run(st["handle"])
        return {"n": st["n"], "U": st["U"], "flags": st["flags"]}
    m = st["model"]
    if op == "ground":
        if case["hi"] > 100.0:  # charges beyond int8
            n, U, f = m.ground_state_i16(st["raster"], threshold=case["t"], closed=case["closed"],
                                         n_charges=case["n_charges"])
        elif case["closed"]:
            n, U, f = m.ground_state_closed(st["raster"], case["n_charges"], threshold=case["t"])
        else:
            n, U, f = m.ground_state_open(st["raster"], threshold=case["t"])
        return {"n": n, "U": U, "flags": f}
    if op == "points":
        n, U, f = m.ground_state_points(st["V"], threshold=case["t"], closed=case["closed"],
                                        n_charges=case["n_charges"])
        return {"n": n, "U": U, "flags": f}
    if op == "soft":
        mean, logZ = m.soft_occupation(st["raster"], case["kT"], threshold=case["t"],
                                       closed=case["closed"], n_charges=case["n_charges"])
        return {"mean": mean, "logZ": logZ}
    if op == "softgrad":
        mean = autograd.soft_occupation(st["Cdd"].double(), st["Cgd"].double(), m.handle,
                                        st["raster"], case["kT"], case["t"])
        loss = torch.mean((mean.sum(1) - st["target"]) ** 2)
        dCdd, dCgd = torch.autograd.grad(loss, (st["Cdd"], st["Cgd"]))
        return {"mean": mean.detach(), "loss": loss.detach(), "dCdd": dCdd, "dCgd": dCgd}
    if op == "fit":
        api.qa_fit_step(m.handle, st["raster"], case["kT"], case["t"], False, 0, st["target"],
                        False, st["Cdd"], st["Cgd"], st["opt"], ADAM["lr"], ADAM["beta1"],
                        ADAM["beta2"], ADAM["eps"], loss=st["loss"], out_mean=st["mean"])
        return {"loss": st["loss"], "mean": st["mean"], "Cdd": st["Cdd"], "Cgd": st["Cgd"]}
    if op == "sensor":
        n, U, f = m.ground_state_open(st["raster"], threshold=case["t"])
        api.qa_charge_sensor(st["full"].handle, st["raster"], n, st["params"], st["signal"],
                             st["n_sensor"], st["potential"])
        return {"n": n, "signal": st["signal"], "n_sensor": st["n_sensor"],
                "potential": st["potential"]}
    if case["closed"]:
        n, U, f = m.brute_force_closed(st["raster"], case["n_max"])
    else:
        n, U, f = m.brute_force_open(st["raster"], case["n_max"])
    return {"n": n, "U": U, "flags": f}


def work(case):
    """Bytes in and out, and the operations no form of the call avoids: the
    induced charge, h = M (base - c) and the energy of the answer for a ground
    state; one energy a state where every state counts (soft, brute)."""
    op, n = case["op"], case["n"]
    ng = n + case["extra_gates"]
    if op == "batch":
        b = f = 0
        for s in _specs(case, 0):
            P, k = s["raster"]["W"] * s["raster"]["H"], s["n"]
            b += P * (k + 9)
            f += P * (4 * k * k + 4 * k)
        return {"bytes": b, "flops": f}
    P = case["W"] * case["H"]
    per = 4 * n * n + 4 * n
    if op == "points":
        return {"bytes": P * (8 * ng + n + 9), "flops": P * (per + 2 * n * ng)}
    if op == "ground":
        return {"bytes": P * (n * (2 if case["hi"] > 100.0 else 1) + 9), "flops": P * per}
    if op in ("soft", "softgrad", "fit"):
        states = 2.0 ** (n if case["t"] >= 1.0 else n * math.log2(1.0 + case["t"]))
        back = op != "soft"
        return {"bytes": P * (4 * n + 4), "flops": P * (per + states * (8 if back else 4))}
    if op == "sensor":
        S = case["n_sensor"]
        return {"bytes": P * (n + 13 * S), "flops": P * (per + 4 * S * (n + S) + 30 * S)}
    states = float(case["n_max"] + 1) ** (n - 1 if case["closed"] else n)
    return {"bytes": P * (n + 9), "flops": P * (per + 2 * states)}


# --------------------------------------------------------------------------
# FP64 values
# --------------------------------------------------------------------------

def _dev(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")


def _raster_volts(ras):
    W, H = ras["W"], ras["H"]
    dx = (ras["x1"] - ras["x0"]) / (W - 1) if W > 1 else 0.0
    dy = (ras["y1"] - ras["y0"]) / (H - 1) if H > 1 else 0.0
    x = ras["x0"] + dx * torch.arange(W, dtype=torch.float64, device="cuda")
    y = ras["y0"] + dy * torch.arange(H, dtype=torch.float64, device="cuda")
    V = _dev(ras["V0"]) + x[None, :, None] * _dev(ras["u"]) + y[:, None, None] * _dev(ras["w"])
    return V.reshape(W * H, -1)


def _maxwell(case, Cdd, Cgd):
    if case["coupling"]:
        return np.diag(Cdd.sum(1) + Cgd.sum(1)) - Cdd
    return Cdd


def _relaxed(Cdd, c, closed, n_charges):
    """argmin of (x - c)^T Cdd^-1 (x - c) over x >= 0 [, sum x = n_charges]:
    x = c + Cdd (z + lambda 1) with z = 0 off the active set, the active set
    grown by negative x and shrunk by the most negative multiplier."""
    P, n = c.shape
    v = Cdd.sum(1)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    x = c + (n_charges - c.sum(1, keepdim=True)) * (v / v.sum()) if closed else c.clone()
    todo = torch.nonzero((x < 0).any(1)).flatten()
    if closed and n_charges == 0:
        return torch.zeros_like(c)
    act = x[todo] < 0
    for _ in range(8 * n + 8):
        if not len(todo):
            break
        ca, m = c[todo], act.double()
        K = Cdd * m[:, :, None] * m[:, None, :] + eye * (1 - m)[:, None, :]
        rhs = -ca * m
        if closed:
            top = torch.cat([K, (v * m)[:, :, None]], 2)
            low = torch.cat([v * m, v.sum().expand(len(todo), 1)], 1)[:, None, :]
            K = torch.cat([top, low], 1)
            rhs = torch.cat([rhs, n_charges - ca.sum(1, keepdim=True)], 1)
        z = torch.linalg.solve(K, rhs)
        xa = ca + (z[:, :n] * m) @ Cdd + (z[:, n:] * v if closed else 0.0)
        xa = torch.where(act, torch.zeros_like(xa), xa)
        neg = xa < -1e-13 * (1.0 + ca.abs().amax(1, keepdim=True))
        zz = torch.where(act, z[:, :n], torch.full_like(xa, math.inf))
        worst, at = zz.min(1)
        grow = neg.any(1)
        drop = ~grow & (worst < -1e-13 * (1.0 + ca.abs().amax(1)))
        done = ~grow & ~drop
        x[todo[done]] = xa[done].clamp_min(0.0)
        act = torch.where(grow[:, None], act | neg, act)
        act[drop, at[drop]] = False
        todo, act = todo[~done], act[~done]
    return x


def _candidates(x, t, closed, n_charges):
    """base, ambiguous mask and weight of the floor / floor + 1 sets."""
    x = x.clamp_min(0.0)
    fl = x.floor()
    fr = x - fl
    tt = torch.full((len(x), 1), float(t), dtype=torch.float64, device="cuda")
    for _ in range(40):
        amb = (fr - 0.5).abs() <= 0.5 * tt
        base = fl + (~amb & (fr >= 0.5))
        w = n_charges - base.sum(1)
        if not closed:
            break
        bad = ((w < 0) | (w > amb.sum(1))) & (tt[:, 0] < 1.0)
        if not bad.any():
            break
        tt = torch.where(bad[:, None], torch.where(tt <= 0, 1.0, (2 * tt).clamp_max(1.0)), tt)
    return base, amb, w


def _patterns(n):
    b = torch.arange(1 << n, device="cuda")
    bits = ((b[:, None] >> torch.arange(n, device="cuda")) & 1).double()
    return b, bits


def _energies(M, c, base, amb, w, closed, b, bits):
    """Energies relative to the base of every pattern, inf off the set."""
    n = c.shape[1]
    r = base - c
    E = (r @ M) @ bits.T + 0.5 * ((bits @ M) * bits).sum(1)
    if not bool(amb.all()):
        word = (amb.long() << torch.arange(n, device="cuda")).sum(1)
        E = torch.where((b[None, :] & ~word[:, None]) != 0, math.inf, E)
    if closed:
        E = torch.where(bits.sum(1)[None, :] != w[:, None], math.inf, E)
    return E, 0.5 * ((r @ M) * r).sum(1)


def _ground_U(Cdd, c, t, closed, n_charges):
    """U of the ground state of every row of c, with its charges."""
    M = torch.linalg.inv(Cdd)
    base, amb, w = _candidates(_relaxed(Cdd, c, closed, n_charges), t, closed, n_charges)
    n = c.shape[1]
    b, bits = _patterns(n)
    step = max(1, (1 << 27) >> n)
    U, nv = [], []
    for i in range(0, len(c), step):
        s = slice(i, i + step)
        E, _ = _energies(M, c[s], base[s], amb[s], w[s], closed, b, bits)
        nn = base[s] + bits[E.argmin(1)]
        r = nn - c[s]
        U.append(0.5 * ((r @ M) * r).sum(1))
        nv.append(nn)
    return torch.cat(U), torch.cat(nv)


def _soft(Cdd, Cgd, V, carrier, kT, t, closed, n_charges):
    """<n> and log Z over the frozen candidate sets, differentiable."""
    with torch.no_grad():
        c0 = carrier * V @ Cgd.T
        base, amb, w = _candidates(_relaxed(Cdd, c0, closed, n_charges), t, closed, n_charges)
    M = torch.linalg.inv(0.5 * (Cdd + Cdd.T))
    n = Cdd.shape[0]
    b, bits = _patterns(n)
    step = max(1, (1 << 25) >> n)
    mean, logZ = [], []
    for i in range(0, len(V), step):
        s = slice(i, i + step)
        E, U0 = _energies(M, carrier * V[s] @ Cgd.T, base[s], amb[s], w[s], closed, b, bits)
        mean.append(base[s] + torch.softmax(-E / kT, 1) @ bits)
        logZ.append(torch.logsumexp(-E / kT, 1) - U0 / kT)
    return torch.cat(mean), torch.cat(logZ)


def _soft_grads(case, Cdd, Cgd, V, target):
    Cdd, Cgd = _dev(Cdd).requires_grad_(), _dev(Cgd).requires_grad_()
    mean, _ = _soft(Cdd, Cgd, V, 1.0, case["kT"], case["t"], False, 0)
    loss = torch.mean((mean.sum(1) - target) ** 2)
    dCdd, dCgd = torch.autograd.grad(loss, (Cdd, Cgd))
    return mean.detach(), loss.detach(), 0.5 * (dCdd + dCdd.T), dCgd


def _philox(c, k):
    """Philox4x32-10 on arrays of counters c[4] under the key k[2]."""
    low = np.uint64(0xFFFFFFFF)
    c = [np.asarray(v, dtype=np.uint64) for v in np.broadcast_arrays(*c)]
    for r in range(10):
        if r:
            k = ((k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF)
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k[0]), p1 & low,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k[1]), p0 & low]
    return c


def _sensor_noise(case, seed, s):
    """White, 1/f and telegraph noise of sensor s, [H, W]."""
    W, H = case["W"], case["H"]
    row = np.arange(H)[:, None]
    key = (seed & 0xFFFFFFFF, seed >> 32)

    def gauss(tag, idx):
        b = _philox([tag, row, idx, 0], key)
        u1, u2 = (b[0] + 1.0) * 2.0 ** -32, b[1] * 2.0 ** -32
        return np.sqrt(-2.0 * np.log(u1)) * np.cos(2.0 * np.pi * u2)

    v = NOISE["white_sigma"] * gauss(s << 4, np.arange(W)[None, :])
    K = 1
    while (1 << (K - 1)) < W:
        K += 1
    pink = sum(gauss(1 | (s << 4) | (k << 8), np.arange(W)[None, :] >> k) for k in range(K))
    v = v + NOISE["pink_sigma"] * pink / math.sqrt(K)
    flip = np.zeros((H, W), dtype=np.int64)
    pos = np.full(H, -1.0)
    lq = math.log(1.0 - NOISE["jump_prob"])
    for j in range(W):
        u = (_philox([2 | (s << 4), np.arange(H), j, 0], key)[0] + 1.0) * 2.0 ** -32
        pos = pos + 1.0 + np.floor(np.log(u) / lq)
        on = pos < W
        if not on.any():
            break
        flip[np.nonzero(on)[0], pos[on].astype(np.int64)] ^= 1
    return v + NOISE["jump_amplitude"] * (flip.cumsum(1) & 1)


def exact(case, seed):
    op, t, closed, nc = case["op"], case["t"], case["closed"], case["n_charges"]
    if op == "batch":
        U = []
        for s in _specs(case, seed):
            c = _raster_volts(s["raster"]) @ _dev(s["Cgd"]).T
            u, _ = _ground_U(_dev(s["Cdd"]), c, s["t"], s["closed"], s["n_charges"])
            U += [u, torch.zeros(-len(u) % 256, dtype=torch.float64, device="cuda")]
        return {"n": None, "U": torch.cat(U), "flags": None}
    if op == "points":
        Cdd, Cgd, _ = _array(dict(case, H=1), seed)
        V = _voltages(case, seed)
    else:
        Cdd, Cgd, ras = _array(case, seed)
        V = _raster_volts(ras)
    if op in ("ground", "points"):
        c = case["carrier"] * V @ _dev(Cgd).T
        U, _ = _ground_U(_dev(_maxwell(case, Cdd, Cgd)), c, t, closed, nc)
        return {"n": None, "U": U, "flags": None}
    if op == "soft":
        mean, logZ = _soft(_dev(Cdd), _dev(Cgd), V, 1.0, case["kT"], t, closed, nc)
        return {"mean": mean, "logZ": logZ}
    if op in ("softgrad", "fit"):
        target = _target(case, seed, Cdd, Cgd, ras).double()
        if op == "softgrad":
            f32 = [a.astype(np.float32).astype(np.float64) for a in (Cdd, Cgd)]
            mean, loss, dCdd, dCgd = _soft_grads(case, *f32, V, target)
            return {"mean": mean, "loss": loss, "dCdd": dCdd, "dCgd": dCgd}
        mean, loss, dCdd, dCgd = _soft_grads(case, Cdd, Cgd, V, target)
        new = [_dev(p) - ADAM["lr"] * g / (g.abs() + ADAM["eps"])  # Adam's first step
               for p, g in ((Cdd, dCdd), (Cgd, dCgd))]
        return {"loss": loss, "mean": mean, "Cdd": new[0], "Cgd": new[1]}
    if op == "sensor":
        nd, S = case["n"], case["n_sensor"]
        M, c = torch.linalg.inv(_dev(Cdd)), V @ _dev(Cgd).T
        _, n = _ground_U(_dev(Cdd[:nd, :nd]), c[:, :nd], t, False, 0)
        xs = c[:, nd:] - (n - c[:, :nd]) @ M[:nd, nd:] @ torch.linalg.inv(M[nd:, nd:])
        fl = xs.clamp_min(0.0).floor()
        _, bits = _patterns(S)
        full = torch.cat([n[:, None, :].expand(-1, 1 << S, -1), fl[:, None, :] + bits], 2)
        r = full - c[:, None, :]
        r = r[torch.arange(len(r), device="cuda"), ((r @ M) * r).sum(2).argmin(1)]
        pot = (r @ M)[:, nd:]
        y = (0.5 * torch.diag(M)[nd:] - pot.abs()) / NOISE["width"]
        sig = 1.0 / (1.0 + y * y)
        noise = np.stack([_sensor_noise(case, seed, s) for s in range(S)], -1)
        shape = (case["H"], case["W"], S)
        return {"n": None, "signal": sig.reshape(shape) + _dev(noise), "n_sensor": None,
                "potential": pot.reshape(shape)}
    # brute force: every state of the box, or of the simplex sum n = n_max
    M, c = torch.linalg.inv(_dev(Cdd)), V @ _dev(Cgd).T
    states = torch.cartesian_prod(*[torch.arange(case["n_max"] + 1, device="cuda").double()
                                    for _ in range(case["n"])])
    if closed:
        states = states[states.sum(1) == case["n_max"]]
    q = 0.5 * ((states @ M) * states).sum(1)
    U, step = [], max(1, (1 << 27) // len(states))
    for i in range(0, len(c), step):
        r = states[(q - (c[i:i + step] @ M) @ states.T).argmin(1)] - c[i:i + step]
        U.append(0.5 * ((r @ M) * r).sum(1))
    return {"n": None, "U": torch.cat(U), "flags": None}
