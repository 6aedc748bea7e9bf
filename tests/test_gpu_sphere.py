"""The one-pass searches (sphere search, enumeration) against the FP32 search:
the same model updated from device matrices has no host factor and takes the
general path, so both run on the same inputs.  Charges and flags are equal;
energies differ by the rounding of double-float sums of at most 256 terms
(2^-44 each) and of the host's and the device's inverse (cond 2^-52)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_04994_gb300 import inputs
from parity import compare

pytestmark = pytest.mark.gpu

GRIDS = {12: (3, 4), 16: (4, 4)}


def _model(n, seed, extra=0):
    r = np.random.Generator(np.random.PCG64(seed))
    Cdd = inputs.grid_cdd(r, *GRIDS[n]) if n in GRIDS else inputs.chain_cdd(r, n)
    Cgd = inputs.dense_cgd(r, n, n + extra)
    gx, gy = inputs.swept_gates(n)
    return Cdd, Cgd, gx, gy, inputs.offsets(r, n + extra, (gx, gy))


def _both(qa, Cdd, Cgd, call, **kw):
    """call(model) on the sphere path and on the general one."""
    out = []
    for dev in (False, True):
        m = qa.Model(Cdd, Cgd, **kw)
        if dev:
            C = torch.tensor(Cdd, device="cuda")
            qa.qa_model_update_dev(m.handle, C, torch.tensor(Cgd, device="cuda"))
        out.append([x.cpu().numpy() for x in call(m)])
        m.close()
    return out


def _same(a, b, label):
    np.testing.assert_array_equal(a[0], b[0], err_msg=label)
    np.testing.assert_array_equal(a[2], b[2], err_msg=label)
    np.testing.assert_allclose(a[1], b[1], rtol=1e-11, atol=1e-12, err_msg=label)


@pytest.mark.parametrize("n,closed,t,W,H,N", [
    (15, False, 1.0, 1, 1, 0), (16, False, 1.0, 2, 1, 0), (16, False, 1.0, 3, 1, 0),
    (13, False, 1.0, 19, 7, 0), (14, False, 1.0, 64, 33, 0), (16, False, 0.8, 100, 99, 0),
    (12, False, 1.0, 200, 151, 0), (16, False, 0.65, 201, 150, 0), (13, False, 0.8, 183, 167, 0),
    (12, True, 1.0, 41, 23, 1), (13, True, 0.8, 64, 31, 13), (15, True, 1.0, 57, 40, 30),
    (16, True, 1.0, 100, 31, 16), (16, True, 0.65, 211, 143, 20),
    # the enumeration by 4, 8 and 16 lanes
    (3, False, 1.0, 1, 1, 0), (3, True, 1.0, 33, 5, 4), (4, False, 1.0, 67, 31, 0),
    (4, True, 0.5, 67, 31, 3), (5, False, 1.0, 17, 1, 0), (6, True, 1.0, 50, 41, 12),
    (8, False, 1.0, 101, 67, 0), (8, True, 0.25, 101, 67, 8), (8, True, 0.0, 31, 67, 5),
    (9, True, 1.0, 90, 67, 9), (9, False, 0.5, 90, 67, 0), (11, False, 0.65, 90, 45, 0),
    (11, True, 0.65, 90, 45, 7),
    # either by the pixel's dots
    (12, False, 0.5, 190, 160, 0), (14, False, 0.25, 60, 41, 0), (16, False, 0.5, 257, 193, 0),
    (12, True, 0.5, 60, 41, 12), (16, True, 0.5, 60, 41, 16), (14, True, 0.0, 60, 41, 14)])
def test_sphere_matches_fp32_search(qa, n, closed, t, W, H, N):
    Cdd, Cgd, gx, gy, V = _model(n, 7 * n + W)
    ras = inputs.raster(n, gx, gy, V, lo=-1.0, hi=6.0, W=W, H=H)

    def call(m):
        if closed:
            return m.ground_state_closed(ras, N, threshold=t)
        return m.ground_state_open(ras, threshold=t)
    a, b = _both(qa, Cdd, Cgd, call)
    _same(a, b, f"N={n} closed={closed} t={t}")
    q = min(W * H, 100)
    rec = oracle.ground_state(Cdd, Cgd, raster=ras, t=t, closed=closed, n_charges=N, pixels=(0, q))
    compare(a[0].reshape(-1, n)[:q], a[1].reshape(-1)[:q], a[2].reshape(-1)[:q], rec, Cdd,
            "sphere", closed=closed)


@pytest.mark.parametrize("form,carrier,i16", [("coupling", 1.0, False), ("maxwell", -1.0, False),
                                              ("maxwell", 1.0, True)])
def test_sphere_forms(qa, form, carrier, i16):
    n = 16
    Cdd, Cgd, gx, gy, V = _model(n, 5, extra=3)
    ras = inputs.raster(n + 3, gx, gy, carrier * V, lo=-1.0, hi=6.0, W=90, H=61)
    if carrier < 0:
        ras = inputs.raster(n + 3, gx, gy, -V, lo=-6.0, hi=1.0, W=90, H=61)
    if i16:
        ras = inputs.raster(n + 3, gx, gy, V, lo=100.0, hi=400.0, W=90, H=61)
    A = np.abs(Cdd - np.diag(np.diag(Cdd)))
    for closed in (False, True):
        def call(m):
            if i16:
                return m.ground_state_i16(ras, threshold=1.0, closed=closed, n_charges=9)
            if closed:
                return m.ground_state_closed(ras, 9)
            return m.ground_state_open(ras)
        if form == "coupling":
            a = _both(qa, A, Cgd, call, form=qa.QA_FORM_COUPLING)[0]
            # (the device update takes Maxwell matrices)
            Cm = np.diag(A.sum(1) + Cgd.sum(1)) - A
            b = _both(qa, Cm, Cgd, call)[1]
        else:
            a, b = _both(qa, Cdd, Cgd, call, carrier_sign=carrier)
        _same(a, b, f"{form} carrier {carrier} closed {closed}")


@pytest.mark.parametrize("n,ng,closed", [(16, 16, False), (16, 20, False), (16, 16, True),
                                         (4, 4, False), (7, 9, True)])
def test_sphere_points(qa, n, ng, closed):
    Cdd, Cgd, *_ = _model(n, 11, extra=ng - n)
    V = torch.rand((1501, ng), dtype=torch.float64, device="cuda",
                   generator=torch.Generator(device="cuda").manual_seed(3)) * 7 - 1
    a, b = _both(qa, Cdd, Cgd, lambda m: m.ground_state_points(V, closed=closed,
                                                               n_charges=n if closed else 0))
    _same(a, b, f"points {ng}")


@pytest.mark.parametrize("n,closed", [(13, False), (16, False), (14, True), (4, False),
                                      (8, False), (8, True)])
def test_exact_ties(qa, n, closed):
    # identical, uncoupled dots, all of one charge: half-integer voltages tie
    # every pattern, more than the search lists; the rest ties none or all
    Cdd, Cgd = np.eye(n), np.eye(n)
    u = np.ones(n)
    ras = dict(inputs.raster(n, 0, 1, np.zeros(n), lo=0.0, hi=2.0, W=9, H=1), u=u,
               w=np.zeros(n))
    a, b = _both(qa, Cdd, Cgd, lambda m: (m.ground_state_closed(ras, 5) if closed
                                          else m.ground_state_open(ras)))
    _same(a, b, "ties")
    # coupled pairs: a few tied candidates
    r = np.random.Generator(np.random.PCG64(n))
    Cdd = inputs.chain_cdd(r, n)
    Cdd = 0.5 * (Cdd + Cdd[::-1, ::-1])  # mirror symmetric
    a, b = _both(qa, Cdd, Cgd, lambda m: (m.ground_state_closed(dict(ras, W=61), 5) if closed
                                          else m.ground_state_open(dict(ras, W=61))))
    # the last bits of the host's and the device's inverse decide a tie, so
    # either path may name either of the tied states: of equal energy, and
    # each the energy of the state it comes with
    M = np.linalg.inv(Cdd)
    c = np.repeat(np.linspace(0.0, 2.0, 61)[:, None], n, 1)
    for x in (a, b):
        r = x[0].reshape(-1, n) - c
        np.testing.assert_allclose(0.5 * ((r @ M) * r).sum(1), x[1].reshape(-1), rtol=1e-11,
                                   atol=1e-12)
    np.testing.assert_allclose(a[1], b[1], rtol=1e-11, atol=1e-12)
    np.testing.assert_array_equal(a[2], b[2])


@pytest.mark.parametrize("n,a,N,t", [(4, 0.999, 20000, 1.0), (6, 0.99, 30000, 1.0),
                                     (8, 0.999, 50000, 1.0), (8, 0.999, 50000, 0.5),
                                     (11, 0.999, 60000, 0.6), (12, 0.999, 60000, 0.5),
                                     (14, 0.999, 60000, 1.0)])
def test_closed_far_from_the_induced_charge(qa, n, a, N, t):
    # a closed array whose total is far from sum c (lambda large, no dot at
    # zero) and whose off-diagonal capacitances are positive, so that h = M r
    # cancels: the FP32 rounding of h is 10^3 u |h| and more.  U is large
    # against its gaps: energies to the rounding of the double-float sum,
    # 2^-44 sum |r| |M| |r|
    r = np.random.Generator(np.random.PCG64(n))
    Cdd = (1.0 - a) * np.diag(r.uniform(0.8, 1.2, n)) + a
    Cgd = inputs.dense_cgd(r, n)
    ras = inputs.raster(n, *inputs.swept_gates(n), r.uniform(1.0, 3.0, n), lo=0.0, hi=3.0,
                        W=100, H=60)
    x, y = _both(qa, Cdd, Cgd, lambda m: m.ground_state_i16(ras, threshold=t, closed=True,
                                                            n_charges=N))
    assert (x[0].astype(np.int64).sum(-1) == N).all()
    assert not (x[2] & 4).any()
    np.testing.assert_array_equal(x[0], y[0])
    np.testing.assert_array_equal(x[2], y[2])
    mag = np.abs(np.linalg.inv(Cdd)).sum() * (2.0 * N / n) ** 2
    np.testing.assert_allclose(x[1], y[1], rtol=0, atol=2.0 ** -44 * mag)


@pytest.mark.parametrize("n,closed,t,W,H,N", [
    # either side of the dispatch's lines: the sizes where a small raster's rule
    # ends, 9 to 11 dots around 9.5 expected ambiguous ones
    (9, False, 1.0, 100, 60, 0), (10, False, 1.0, 60, 40, 0), (10, False, 1.0, 152, 32, 0),
    (11, False, 1.0, 9, 7, 0), (11, False, 0.8, 120, 90, 0), (11, True, 1.0, 60, 40, 11),
    (10, True, 1.0, 60, 40, 7), (12, False, 1.0, 9, 7, 0), (12, False, 1.0, 8, 8, 0),
    (12, False, 1.0, 128, 38, 0), (12, False, 1.0, 127, 38, 0), (13, False, 0.6, 100, 100, 0),
    (14, False, 0.7, 100, 100, 0), (15, False, 0.4, 60, 40, 0), (13, True, 1.0, 40, 30, 13),
    (13, True, 1.0, 38, 32, 13), (12, True, 0.0, 30, 20, 5), (13, True, 0.0, 30, 20, 5),
    (16, True, 0.7, 40, 31, 16), (16, False, 0.95, 30, 20, 0)])
def test_either_side_of_the_lines(qa, n, closed, t, W, H, N):
    Cdd, Cgd, gx, gy, V = _model(n, 3 * n + W)
    ras = inputs.raster(n, gx, gy, V, lo=-1.0, hi=6.0, W=W, H=H)
    a, b = _both(qa, Cdd, Cgd, lambda m: (m.ground_state_closed(ras, N, threshold=t) if closed
                                          else m.ground_state_open(ras, threshold=t)))
    _same(a, b, f"N={n} closed={closed} t={t} {W} x {H}")
