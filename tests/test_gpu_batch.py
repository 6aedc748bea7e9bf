"""The batched ground state (persistent launches over a device work queue)
against the single-array calls and the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2404_04994_gb300 import inputs
from parity import compare

pytestmark = pytest.mark.gpu


def _mixed_specs(count, sides=(12, 17), seed=0, nmax=16):
    r = np.random.Generator(np.random.PCG64(4242 + seed))
    specs = []
    for a in range(count):
        n = int(r.integers(2, nmax + 1))
        Cdd = inputs.grid_cdd(r, 4, 4) if n == 16 else inputs.chain_cdd(r, n, nn=(0.05, 0.25))
        Cgd = inputs.dense_cgd(r, n, diag=(0.5, 1.0), off=(0.0, 0.1))
        gx, gy = inputs.swept_gates(n)
        V = inputs.offsets(r, n, (gx, gy))
        side = int(sides[int(r.integers(0, len(sides)))])
        closed = bool(r.integers(0, 2))
        t = float(r.choice([1.0, 1.0, 0.5]))
        specs.append(dict(Cdd=Cdd, Cgd=Cgd, raster=inputs.raster(n, gx, gy, V, W=side, H=side - 3),
                          threshold=t, closed=closed, n_charges=n if closed else 0))
    return specs


def test_batch_matches_oracle_and_single_calls(qa):
    specs = _mixed_specs(40)
    b = qa.Batch(specs)
    b.run()
    st = b.stats()
    assert st["pixels"] == sum(s["raster"]["W"] * s["raster"]["H"] for s in specs)
    assert st["unresolved"] == 0
    for sp, (n, U, f) in zip(specs, b.outputs):
        nd = sp["Cdd"].shape[0]
        n = n.cpu().numpy().reshape(-1, nd)
        U = U.cpu().numpy().reshape(-1)
        f = f.cpu().numpy().reshape(-1)
        rec = oracle.ground_state(sp["Cdd"], sp["Cgd"], raster=sp["raster"], t=sp["threshold"],
                                  closed=sp["closed"], n_charges=sp["n_charges"])
        compare(n, U, f, rec, sp["Cdd"], f"batch N={nd} closed={sp['closed']}",
                closed=sp["closed"])
        m = qa.Model(sp["Cdd"], sp["Cgd"])
        if sp["closed"]:
            n1, U1, _ = m.ground_state_closed(sp["raster"], sp["n_charges"], threshold=sp["threshold"])
        else:
            n1, U1, _ = m.ground_state_open(sp["raster"], threshold=sp["threshold"])
        np.testing.assert_array_equal(n, n1.cpu().numpy().reshape(-1, nd))
        np.testing.assert_allclose(U, U1.cpu().numpy(), rtol=1e-9, atol=1e-12)
        m.close()
    b.close()


def test_batch_rerun_and_team_override(qa):
    specs = _mixed_specs(10, sides=(20,), seed=1)
    for sp in specs:
        sp["team"] = 4
    b = qa.Batch(specs)
    b.run()
    first = [o[0].clone() for o in b.outputs]
    b.run()
    for o, f0 in zip(b.outputs, first):
        assert bool((o[0] == f0).all())
    b.close()


def test_batch_rejects_bad_items(qa):
    sp = _mixed_specs(1)[0]
    sp["threshold"] = 2.0
    with pytest.raises(qa.QAError) as e:
        qa.Batch([sp])
    assert e.value.code == -5


def test_full_size_batch_graph_sampled_against_oracle(qa):
    # The 4096-array workload (N ~ U{2..16}, 64^2 / 128^2 rasters, open or
    # closed with N_hat = N) in the launch configuration the benchmark times:
    # one CUDA-graph replay of the batched run.  Every dot count and both
    # forms are sampled; three rows of each sampled array (first, a middle
    # one, last) are recomputed by the oracle one by one.
    import torch
    specs = inputs.batch(4096)
    b = qa.Batch(specs)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        b.run(s)
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.run()
    for o in b.outputs:
        o[0].fill_(-1)
    g.replay()
    torch.cuda.synchronize()
    st = b.stats()
    assert st["pixels"] == b.pixels
    assert st["unresolved"] == 0 and st["overflow"] == 0
    picks = {}
    for a, sp in enumerate(specs):
        key = (sp["Cdd"].shape[0], sp["closed"])
        picks.setdefault(key, []).append(a)
    chosen = sorted(v[0] for v in picks.values()) + sorted(v[-1] for v in picks.values())
    chosen = sorted(set(chosen))
    assert len({specs[a]["Cdd"].shape[0] for a in chosen}) == 15
    compared = 0
    for a in chosen:
        sp = specs[a]
        nd = sp["Cdd"].shape[0]
        W, H = sp["raster"]["W"], sp["raster"]["H"]
        n = b.outputs[a][0].cpu().numpy().reshape(-1, nd)
        U = b.outputs[a][1].cpu().numpy().reshape(-1)
        f = b.outputs[a][2].cpu().numpy().reshape(-1)
        if sp["closed"]:
            assert (n.astype(np.int64).sum(1) == nd).all()
        for row in (0, H // 2 + a % 7, H - 1):
            p0, p1 = row * W, (row + 1) * W
            rec = oracle.ground_state(sp["Cdd"], sp["Cgd"], raster=sp["raster"], t=sp["t"],
                                      closed=sp["closed"], n_charges=sp["n_charges"],
                                      pixels=(p0, p1))
            rep = compare(n[p0:p1], U[p0:p1], f[p0:p1], rec, sp["Cdd"],
                          f"batch array {a} N={nd} closed={sp['closed']} row {row}",
                          closed=sp["closed"])
            compared += rep["comparable"]
    assert compared > 0.9 * sum(3 * specs[a]["raster"]["W"] for a in chosen)
    b.close()


def test_autotuned_batch_matches_oracle_at_the_tuned_thresholds(qa):
    from paper_2404_04994_gb300 import autotune
    specs = _mixed_specs(24, sides=(16, 21), seed=3, nmax=10)
    for sp in specs:
        sp["threshold"] = 1.0
    table = autotune.tune(specs, sample_side=16, arrays_per_group=3)
    for key, e in table.items():
        assert e["team"] in autotune.TEAMS
        if e["threshold"] < 1.0:
            base = [dict(autotune.sample_spec(specs[i], 16), threshold=1.0) for i in e["arrays"]]
            ref, _ = autotune.gpu_runner(base, 1)
            got, _ = autotune.gpu_runner([dict(b, threshold=e["threshold"]) for b in base], 1)
            for r, g in zip(ref, got):
                np.testing.assert_array_equal(r, g)
    tuned = autotune.apply(specs, table)
    b = qa.Batch(tuned)
    b.run()
    assert b.stats()["unresolved"] == 0
    for sp, (n, U, f) in zip(tuned, b.outputs):
        nd = sp["Cdd"].shape[0]
        rec = oracle.ground_state(sp["Cdd"], sp["Cgd"], raster=sp["raster"], t=sp["threshold"],
                                  closed=sp["closed"], n_charges=sp["n_charges"])
        compare(n.cpu().numpy().reshape(-1, nd), U.cpu().numpy().reshape(-1),
                f.cpu().numpy().reshape(-1), rec, sp["Cdd"],
                f"tuned N={nd} t={sp['threshold']:.3f} team={sp['team']}", closed=sp["closed"])
    b.close()


def test_batch_and_graph_see_a_model_update(qa):
    # capacitances may change between a batch's runs: the next run, and the
    # replay of a captured one, take the new Cgd with the new M
    import torch
    old, new = _mixed_specs(15, sides=(23,), seed=7), _mixed_specs(15, sides=(23,), seed=7)
    r = np.random.Generator(np.random.PCG64(1))
    for sp in new:
        sp["Cdd"] = sp["Cdd"] + 0.1 * np.diag(r.random(sp["Cdd"].shape[0]))
        sp["Cgd"] = sp["Cgd"] * r.uniform(0.6, 1.4, sp["Cgd"].shape)
    want = []
    for sp in new:
        m = qa.Model(sp["Cdd"], sp["Cgd"])
        call = m.ground_state_closed if sp["closed"] else m.ground_state_open
        arg = (sp["n_charges"],) if sp["closed"] else ()
        n, U, _ = call(sp["raster"], *arg, threshold=sp["threshold"])
        want.append((n.cpu().numpy(), U.cpu().numpy().reshape(n.shape[:2])))
        m.close()

    def check(label):
        torch.cuda.synchronize()
        for (n, U, _), (n0, U0) in zip(b.outputs, want):
            np.testing.assert_array_equal(n.cpu().numpy(), n0, err_msg=label)
            np.testing.assert_allclose(U.cpu().numpy(), U0, rtol=1e-9, atol=1e-12, err_msg=label)

    b = qa.Batch(old)
    b.run()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.run()
    for m, sp in zip(b.models, new):
        qa.qa_model_update(m.handle, sp["Cdd"], sp["Cgd"])
    b.run()
    check("run after an update")
    for o in b.outputs:
        o[0].fill_(-1)
    g.replay()
    check("replay after an update")
    for m, sp in zip(b.models, new):
        qa.qa_model_update_dev(m.handle, torch.tensor(sp["Cdd"], device="cuda"),
                               torch.tensor(sp["Cgd"], device="cuda"))
    g.replay()
    check("replay after an update on the device")
    b.close()


@pytest.mark.parametrize("launcher", ["_ZN2qa19launch_pixels_batchERKNS_8GsLaunchEP11CUstream_st",
                                      "_ZN2qa12launch_listsERKNS_8GsLaunchEP11CUstream_st"])
def test_batch_reports_the_error_of_each_stage(tmp_path, launcher):
    # a stand-in for one launcher that launches nothing and fails
    import os
    import shutil
    import subprocess
    import sys
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "fail.cpp"
    src.write_text(f'extern "C" int {launcher}(const void*, void*) {{ return 1; }}\n')
    lib = tmp_path / "fail.so"
    subprocess.check_call([gxx, "-shared", "-fPIC", "-o", str(lib), str(src)])
    code = ("import numpy as np\n"
            "from paper_2404_04994_gb300 import api, inputs\n"
            "ras = inputs.raster(4, 0, 1, np.ones(4), W=9, H=7)\n"
            "b = api.Batch([dict(Cdd=np.eye(4), Cgd=np.eye(4), raster=ras)])\n"
            "try:\n    b.run()\nexcept api.QAError as e:\n    print('code', e.code)\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=root)
    r = subprocess.run([sys.executable, "-c", code], env=env, cwd=root, capture_output=True,
                       text=True, timeout=300)
    assert r.stdout.strip() == "code -7", r.stdout + r.stderr


@pytest.mark.parametrize("n", [2, 5, 12])
def test_captured_call_sees_a_model_update(qa, n):
    # a single-array call replayed from a graph after its model changed
    import torch
    r = np.random.Generator(np.random.PCG64(n))
    Cdd, Cgd = inputs.chain_cdd(r, n), inputs.dense_cgd(r, n)
    ras = inputs.raster(n, *inputs.swept_gates(n), np.ones(n), W=60, H=50)
    m = qa.Model(Cdd, Cgd)
    out = torch.zeros((3000, n), dtype=torch.int8, device="cuda")
    qa.qa_ground_state_open(m.handle, ras, 1.0, out)  # (the workspace, before the capture)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        qa.qa_ground_state_open(m.handle, ras, 1.0, out)
    Cgd = Cgd * r.uniform(0.6, 1.4, Cgd.shape)
    qa.qa_model_update(m.handle, Cdd, Cgd)
    g.replay()
    torch.cuda.synchronize()
    m2 = qa.Model(Cdd, Cgd)
    want, _, _ = m2.ground_state_open(ras)
    assert bool((out == want.view(-1, n)).all())
    m.close()
    m2.close()
