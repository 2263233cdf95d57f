"""Tensor-core path at the edges of its tiling: groups of 16 consecutive sorted sources (any box boundary inside a
group), blocks of 32 target boxes, windows of at most 128 targets (boxes of more than 128 points), segments of a long
entry list, right-hand sides around multiples of 8 and 64, odd leading dimensions, and strengths that are not finite.

Tolerance: the path's own per-target bound, |err_i| <= delta S_i with S_i = sum_j |G(r_ij) lambda_j| and delta = 2^-14
for hi / lo, 2^-20 for hi / mid / lo (what the guarded apply relies on), at every target and right-hand side."""
import numpy as np
import pytest

import oracle
from paper_2403_01596_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DELTA = {"tc_bf16x3": 2.0 ** -14, "tc_bf16x6": 2.0 ** -20}


def _worst(out, ref, S):
    """Largest |err| / S over targets and right-hand sides (targets without a pair must be exactly zero)."""
    err = np.abs(out - ref)
    assert (err[S == 0] == 0).all()
    return float((err[S > 0] / S[S > 0]).max()) if (S > 0).any() else 0.0


def _api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    return api


# points, boxes per axis of the unit cube: one box of 15 / 16 / 17 / 127 / 128 / 129 / 400 points, boxes of ~140
# (several windows per box, long lists), 33 and 64 boxes of a few points (block edges), ~1 point per box
@pytest.mark.parametrize("n,ng", [(15, 1), (16, 1), (17, 1), (127, 1), (128, 1), (129, 1), (400, 1), (3800, 3),
                                  (170, 4), (500, 5), (900, 10)])
@pytest.mark.parametrize("path", ["tc_bf16x3", "tc_bf16x6"])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
def test_tiles(n, ng, path, kernel):
    api = _api()
    pts = np.random.default_rng(n + ng).random((n, 3)).astype(np.float32)
    lo, h, k = (0.0, 0.0, 0.0), 1.0 / ng, (float(np.float32(2 * np.pi * ng / 5)) if kernel == "helmholtz" else 0.0)
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, kernel=kernel, max_nrhs=67)
    for nrhs in (1, 9, 33, 64, 67):
        lam = W.strengths(n, nrhs, n + nrhs).reshape(n, nrhs)
        out = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
        assert plan.async_status() == 0
        ref = oracle.p2p(pts, lam, lo, h, ng, k, kernel=kid).reshape(n, nrhs)
        S = oracle.p2p(pts, np.abs(lam).astype(np.complex64), lo, h, ng, 0.0, kernel=oracle.LAPLACE).real.reshape(n, nrhs)
        assert _worst(out, ref, S) <= DELTA[path], (nrhs, _worst(out, ref, S))


@pytest.mark.parametrize("path", ["tc_bf16x3", "tc_bf16x6"])
def test_two_sets_with_lonely_targets(path):
    """Targets with no source nearby (whole windows of them, and some in windows that have work) stay zero."""
    api = _api()
    rng = np.random.default_rng(3)
    tgt = rng.random((3000, 3)).astype(np.float32)
    src = (rng.random((500, 3)) * 0.3).astype(np.float32)
    src[:50] = tgt[np.flatnonzero((tgt < 0.3).all(1))[:50]]  # some at r = 0
    ng, lo, h, k = 10, (0.0, 0.0, 0.0), 0.1, 12.0
    plan = api.TwoSetPlan(torch.from_numpy(tgt).cuda(), torch.from_numpy(src).cuda(), lo, h, ng, k, max_nrhs=16)
    lam = W.strengths(500, 16, 4)
    out = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
    assert plan.async_status() == 0
    ref = oracle.p2p_st(tgt, src, lam, lo, h, ng, k)
    S = oracle.p2p_st(tgt, src, np.abs(lam).astype(np.complex64), lo, h, ng, 0.0, kernel=oracle.LAPLACE).real
    assert _worst(out, ref, S) <= DELTA[path]
    assert (out[np.abs(ref).max(1) == 0] == 0).all() and (np.abs(ref).max(1) == 0).any()


@pytest.mark.parametrize("path", ["tc_bf16x3", "tc_bf16x6"])
@pytest.mark.parametrize("nrhs", [17, 64])
def test_strength_that_is_not_finite_stays_local(path, nrhs):
    """An infinite or NaN strength makes NaN of the results of its own neighbourhood and right-hand side, and of
    nothing else."""
    api = _api()
    wl = W.Workload("s", W.unit_sphere(4000, 8), (-1, -1, -1), 2 / 14, 14, 30.0, 8)
    plan = api.Plan(torch.from_numpy(wl.points).cuda(), wl.lo, wl.h, wl.ng, wl.k, max_nrhs=nrhs)
    lam = W.strengths(wl.n, nrhs, 8)
    clean = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
    cell = np.clip(np.floor((wl.points.astype(np.float64) + 1) / wl.h), 0, wl.ng - 1)
    hit = np.zeros((wl.n, nrhs), bool)
    for s, r, v in ((5, 3, np.inf), (1777, 16, np.nan), (1778, 0, complex(0, -np.inf))):
        lam[s, r] = v
        hit[np.abs(cell - cell[s]).max(1) <= 1, r] = True
    out = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
    assert plan.async_status() == 0
    assert np.isnan(out.real[hit]).all() and np.isnan(out.imag[hit]).all()
    assert np.array_equal(out[~hit], clean[~hit])


@pytest.mark.parametrize("n,ng", [(15, 1), (17, 1), (128, 1), (129, 1), (400, 1), (3800, 3), (170, 4), (900, 10)])
@pytest.mark.parametrize("kernel,path,widths", [("helmholtz", "tc_bf16x3", (1, 33, 67)), ("laplace", "tc_bf16x3", (9, 64)),
                                                ("helmholtz", "tc_bf16x6", (1, 9, 32)), ("laplace", "tc_bf16x6", (24,))])
def test_tiles_in_a_large_plan(n, ng, kernel, path, widths):
    """The same boxes in the corner of a plan of 42 000 more points, about one per box, so that it is large enough for
    units of 128 targets."""
    api = _api()
    rng = np.random.default_rng(n + ng)
    ng2, h = ng + 42, 1.0 / ng
    far = rng.random((42000, 3)) * [ng2, ng2, 40] + [0, 0, ng + 2]  # in cells, at least two cells from the corner's boxes
    pts = np.concatenate([rng.random((n, 3)), far * h]).astype(np.float32)
    lo, k, m = (0.0, 0.0, 0.0), (float(np.float32(2 * np.pi * ng / 5)) if kernel == "helmholtz" else 0.0), len(pts)
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng2, k, kernel=kernel, max_nrhs=67)
    for nrhs in widths:
        lam = W.strengths(m, nrhs, n + nrhs).reshape(m, nrhs)
        out = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
        assert plan.async_status() == 0
        ref = oracle.p2p(pts, lam, lo, h, ng2, k, kernel=kid).reshape(m, nrhs)
        S = oracle.p2p(pts, np.abs(lam).astype(np.complex64), lo, h, ng2, 0.0, kernel=oracle.LAPLACE).real.reshape(m, nrhs)
        assert _worst(out, ref, S) <= DELTA[path], (nrhs, _worst(out, ref, S))


# 58 points per box in a cube: a window of 128 targets covers two or three boxes whose neighbourhoods differ, its list
# holds more than 64 entries (several segments); one box per unit (4 000 points, or wide three parts) next to it
@pytest.mark.parametrize("path,nrhs,n,ng", [("tc_bf16x3", 17, 42000, 9), ("tc_bf16x3", 64, 42000, 9), ("tc_bf16x3", 80, 42000, 9),
                                            ("tc_bf16x6", 17, 42000, 9), ("tc_bf16x6", 32, 42000, 9), ("tc_bf16x6", 64, 42000, 9),
                                            ("tc_bf16x3", 17, 4000, 4), ("tc_bf16x6", 17, 4000, 4)])
def test_strengths_at_the_ends_of_fp32(path, nrhs, n, ng):
    """Infinite and NaN strengths make NaN of their own neighbourhood and right-hand side; the largest finite ones, which
    round to infinity in BF16, give their neighbours what they are worth; every other result is what it was, bit for bit.
    Points far enough apart (r > 1) that no term overflows."""
    api = _api()
    h = 200.0
    pts = (np.random.default_rng(n).random((n, 3)) * (ng * h)).astype(np.float32)
    lo, k = (0.0, 0.0, 0.0), 2 * np.pi / 500.0
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, max_nrhs=nrhs)
    lam = W.strengths(n, nrhs, 8)
    clean = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
    cell = np.clip(np.floor(pts.astype(np.float64) / h), 0, ng - 1)
    near = lambda s: np.abs(cell - cell[s]).max(1) <= 1  # noqa: E731
    nan, huge, top = np.zeros((n, nrhs), bool), np.zeros((n, nrhs), bool), np.finfo(np.float32).max
    for s, r, v in ((5, 3, np.inf), (1777, 7, np.nan), (1778, 0, complex(0, -np.inf)), (n - 7, 5, -np.inf)):
        lam[s, r] = v
        nan[near(s), r] = True
    for s, r, v in ((9, 1, top), (n - 11, 2, complex(0, -3.397e38)), (n // 2, 11, 3.39e38), (n // 3, nrhs - 1, -top)):
        d = np.linalg.norm(pts[near(s)].astype(np.float64) - pts[s], axis=1)
        assert d[d > 0].min() > 1.0
        lam[s, r] = v
        huge[near(s), r] = True
    out = plan.apply(torch.from_numpy(lam).cuda(), path=path).cpu().numpy()
    assert plan.async_status() == 0
    assert np.isnan(out.real[nan]).all() and np.isnan(out.imag[nan]).all()
    rest = ~nan & ~huge
    assert np.array_equal(out[rest], clean[rest])
    # the FP32 kernels form the same G (whose phase is rounded in FP32: one pair may be all of a sum here)
    cols = np.unique(np.flatnonzero(huge.any(0)))
    ref = plan.apply(torch.from_numpy(lam).cuda(), path="fp32_shared").cpu().numpy()[:, cols].astype(np.complex128)
    S = oracle.p2p(pts, np.abs(lam[:, cols].astype(np.complex128)).clip(max=top).astype(np.complex64), lo, h, ng, 0.0,
                   kernel=oracle.LAPLACE).real.reshape(n, -1)
    at = huge[:, cols]
    assert np.isfinite(out[:, cols][at]).all()
    assert (np.abs(out[:, cols][at].astype(np.complex128) - ref[at]) <= DELTA[path] * S[at]).all()
