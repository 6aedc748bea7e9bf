"""GPU brute force (Table I, brute-force row; C ABI -> CUDA) against the
FP64 oracle's exhaustive search, and against the default method where
Theorem 2 makes the default method exact."""
import math

import numpy as np
import pytest

import oracle
from paper_2404_04994_gb300 import inputs

pytestmark = pytest.mark.gpu


def _brute_gpu(qa, Cdd, Cgd, ras, closed, bound):
    m = qa.Model(Cdd, Cgd)
    if closed:
        n, U, f = m.brute_force_closed(ras, bound)
    else:
        n, U, f = m.brute_force_open(ras, bound)
    out = (n.cpu().numpy().reshape(-1, m.n_dot).astype(np.int64), U.cpu().numpy(),
           f.cpu().numpy())
    m.close()
    return out


def _check(qa, Cdd, Cgd, ras, closed, bound, label):
    n, U, f = _brute_gpu(qa, Cdd, Cgd, ras, closed, bound)
    ref = oracle.brute_force_raster(Cdd, Cgd, ras, closed=closed, n_charges=bound if closed else 0,
                                    n_max=bound)
    gap = ref["U2"] - ref["U"]
    ok = gap > 1e-9
    bad = ok & (n != ref["n"]).any(1)
    assert not bad.any(), f"{label}: {int(bad.sum())} pixels differ, first {np.where(bad)[0][:5]}"
    assert ok.sum() >= 0.9 * len(ok)
    scale = np.maximum(1.0, np.abs(ref["U"]))
    assert np.max(np.abs(U - ref["U"]) / scale) < 1e-10, label
    # flags: near ties exactly where the oracle's gap is (numerically) zero-ish
    assert not (((f & 1) != 0) & (gap > 1e-6)).any()
    if not closed:
        np.testing.assert_array_equal((f & 2) != 0, ref["hit"])
    else:
        assert (n.sum(1) == bound).all() and (n >= 0).all()
    return n, U, f, ref


def _model(seed, n, chain=True):
    r = np.random.Generator(np.random.PCG64(seed))
    Cdd = inputs.chain_cdd(r, n) if chain else inputs.grid_cdd(r, 2, n // 2)
    Cgd = inputs.dense_cgd(r, n, diag=(0.5, 1.0), off=(0.0, 0.2))
    gx, gy = inputs.swept_gates(n)
    V = inputs.offsets(r, n, (gx, gy))
    return Cdd, Cgd, gx, gy, V


@pytest.mark.parametrize("n,nmax,W,H", [(2, 8, 23, 17), (3, 5, 13, 11), (4, 4, 9, 7)])
def test_open_matches_oracle(qa, n, nmax, W, H):
    Cdd, Cgd, gx, gy, V = _model(100 + n, n)
    ras = inputs.raster(n, gx, gy, V, lo=-1.0, hi=4.0, W=W, H=H)
    _check(qa, Cdd, Cgd, ras, False, nmax, f"open N={n}")


@pytest.mark.parametrize("n,nhat,W,H", [(2, 3, 19, 13), (3, 5, 11, 9), (4, 4, 9, 7), (1, 2, 5, 3)])
def test_closed_matches_oracle(qa, n, nhat, W, H):
    Cdd, Cgd, gx, gy, V = _model(200 + n, n)
    if n == 1:
        gx, gy = 0, 0
    ras = inputs.raster(n, gx, gy, V, W=W, H=H)
    _check(qa, Cdd, Cgd, ras, True, nhat, f"closed N={n}")


def test_box_too_small_is_flagged(qa):
    Cdd, Cgd, gx, gy, V = _model(301, 3)
    ras = inputs.raster(3, gx, gy, V, lo=2.0, hi=6.0, W=8, H=6)
    n, U, f, ref = _check(qa, Cdd, Cgd, ras, False, 2, "open N=3 small box")
    assert ref["hit"].any() and ((f & 2) != 0).any()


def test_default_method_equals_brute_force_under_theorem_2(qa):
    # Theorem 2 (App. E): with kappa(M) <= 1 + 4/n and x = c >= 0 the default
    # method (t = 1) is exact; both run on the GPU here
    r = np.random.Generator(np.random.PCG64(77))
    n = 2
    while True:
        Cdd, _ = inputs.random_model(r, n, nn=(0.0, 0.2))
        ev = np.linalg.eigvalsh(np.linalg.inv(Cdd))
        if ev[-1] / ev[0] <= 1 + 4 / n:
            break
    Cgd = np.diag(r.uniform(0.5, 1.0, n))
    ras = inputs.raster(n, 0, 1, np.zeros(n), lo=0.0, hi=5.0, W=31, H=29)
    m = qa.Model(Cdd, Cgd)
    nd, Ud, fd = m.ground_state_open(ras)
    nb, Ub, fb = m.brute_force_open(ras, 9)
    nd = nd.cpu().numpy().reshape(-1, n)
    nb = nb.cpu().numpy().reshape(-1, n)
    clear = ((fb.cpu().numpy() & 1) == 0) & ((fd.cpu().numpy() & 1) == 0)
    np.testing.assert_array_equal(nd[clear], nb[clear])
    assert clear.mean() > 0.95
    m.close()


def test_brute_force_errors(qa):
    Cdd, Cgd, gx, gy, V = _model(401, 4)
    ras = inputs.raster(4, gx, gy, V, W=4, H=4)
    m = qa.Model(Cdd, Cgd)
    with pytest.raises(qa.QAError) as e:
        m.brute_force_open(ras, -1)
    assert e.value.code == -5
    with pytest.raises(qa.QAError) as e:
        m.brute_force_closed(ras, 200)
    assert e.value.code == -5
    m.close()
    r = np.random.Generator(np.random.PCG64(9))
    big = qa.Model(inputs.grid_cdd(r, 4, 4), inputs.dense_cgd(r, 16))
    gx, gy = inputs.swept_gates(16)
    with pytest.raises(qa.QAError) as e:   # 128^16 states per pixel
        big.brute_force_open(inputs.raster(16, gx, gy, np.zeros(16), W=2, H=2), 127)
    assert e.value.code == -5
    big.close()


# The FP32 line search against the oracle where it can go wrong: one state, one
# line, the largest digit range, many leading digits, closed simplices whose
# leading digits leave nothing, and exact ties (uncoupled dots at half
# charges, 2^N of equal energy), which the FP64 shortlist settles.
@pytest.mark.parametrize("n,closed,bound,W,H", [
    (1, False, 0, 7, 1), (1, False, 127, 33, 3), (1, True, 0, 3, 1), (2, False, 127, 9, 5),
    (3, False, 1, 5, 129), (6, False, 3, 7, 3), (10, False, 1, 3, 2), (2, True, 127, 9, 3),
    (5, True, 6, 11, 3), (6, True, 2, 1, 33)])
def test_line_search_edges(qa, n, closed, bound, W, H):
    r = np.random.Generator(np.random.PCG64(500 + n))
    Cdd, Cgd = inputs.random_model(r, n)
    gx, gy = (0, 0) if n == 1 else inputs.swept_gates(n)
    ras = inputs.raster(n, gx, gy, inputs.offsets(r, n, (gx, gy)), W=W, H=H,
                        hi=140.0 if bound == 127 else 5.0)
    _check(qa, Cdd, Cgd, ras, closed, bound, f"N={n} closed={closed} bound={bound}")


@pytest.mark.parametrize("n", [2, 4])
@pytest.mark.parametrize("closed", [False, True])
def test_line_search_exact_ties(qa, n, closed):
    # every dot at c = 1.5 (open: 2^n equal energies; closed with 2 n - n / 2
    # charges: n over n / 2 of them): a near tie, the lexicographically
    # smallest state
    ras = inputs.raster(n, 0, 1, np.full(n, 1.5), W=1, H=1)
    ras["V0"][:] = 1.5
    ras["u"][:] = 0.0
    ras["w"][:] = 0.0
    nh = n + n // 2
    nn, U, f = _brute_gpu(qa, np.eye(n), np.eye(n), ras, closed, nh if closed else 4)
    want = [1] * (n - n // 2) + [2] * (n // 2) if closed else [1] * n
    np.testing.assert_array_equal(nn[0], want)
    assert f[0] & 1 and abs(U[0] - 0.125 * n) < 1e-14


@pytest.mark.parametrize("n,closed,bound,W,H", [
    (1, False, 30, 40, 30), (2, True, 30, 40, 30), (2, False, 7, 40, 30), (3, False, 1, 4, 1),
    (2, False, 12, 153, 4), (3, True, 9, 19, 32)])
def test_teams_wider_than_the_hi_states(qa, n, closed, bound, W, H):
    # small rasters: lanes without a leading-digit state of their own
    r = np.random.Generator(np.random.PCG64(600 + n))
    Cdd, Cgd = inputs.random_model(r, n)
    gx, gy = (0, 0) if n == 1 else inputs.swept_gates(n)
    ras = inputs.raster(n, gx, gy, inputs.offsets(r, n, (gx, gy)), W=W, H=H, hi=5.0)
    _check(qa, Cdd, Cgd, ras, closed, bound, f"N={n} closed={closed} bound={bound}")
