"""The hi / lo tensor-core path with more than 32 right-hand sides per launch: accumulating every product of the split in
tensor memory must not cost more than the fourth product gains, so the error stays below that of the three leading
products (hi.hi + hi.lo + lo.hi) of the same BF16 parts summed in 64 bits.

No tolerance is chosen: the bound is evaluated from the inputs themselves."""
import numpy as np
import pytest

import oracle
from paper_2403_01596_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _parts(v):
    """hi and lo of FP32 values as 64-bit arrays."""
    t = torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32))
    hi = t.to(torch.bfloat16).to(torch.float32)
    lo = (t - hi).to(torch.bfloat16).to(torch.float32)
    return hi.numpy().astype(np.float64), lo.numpy().astype(np.float64)


def _three(a, b):
    ah, al = _parts(a)
    bh, bl = _parts(b)
    return ah @ bh + ah @ bl + al @ bh


# two launches of 40, one of 64 right-hand sides; ~180 and ~430 sources per target
@pytest.mark.parametrize("nrhs,per_box", [(40, 20), (64, 20), (64, 48), (80, 20)])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
def test_error_below_the_three_products(nrhs, per_box, kernel):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    n = 60_000
    ng = max(2, round(2.0 * np.sqrt(n / per_box / (1.29 * 4.0 * np.pi))))
    pts, lo, h = W.unit_sphere(n, 3), (-1.0, -1.0, -1.0), 2.0 / ng
    k = float(np.float32(2 * np.pi * 0.25 / h)) if kernel == "helmholtz" else 0.0
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    lam = W.strengths(n, nrhs, 4)
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, kernel=kernel, max_nrhs=nrhs)
    out = plan.apply(torch.from_numpy(lam).cuda(), path="tc_bf16x3").cpu().numpy()
    assert plan.async_status() == 0
    idx = np.random.default_rng(5).choice(n, 400, replace=False)
    ref = oracle.p2p_targets(pts, lam, idx, lo, h, ng, k, kernel=kid).reshape(400, nrhs)
    cell = np.clip(np.floor((pts.astype(np.float64) - lo[0]) / h), 0, ng - 1)
    three = np.zeros_like(ref)
    for i, t in enumerate(idx):
        near = np.flatnonzero((np.abs(cell - cell[t]) <= 1).all(1))
        r = np.linalg.norm(pts[near].astype(np.float64) - pts[t].astype(np.float64), axis=1)
        near, r = near[r > 0], r[r > 0]
        gr, gi = np.cos(k * r) / r, np.sin(k * r) / r
        lr, li = lam[near].real, lam[near].imag
        three[i] = (_three(gr, lr) - _three(gi, li)) + 1j * (_three(gr, li) + _three(gi, lr))
    three /= 4.0 * np.pi
    err = np.linalg.norm(out[idx] - ref) / np.linalg.norm(ref)
    bound = np.linalg.norm(three - ref) / np.linalg.norm(ref)
    assert err <= bound, (err, bound)
