"""Several right-hand sides in FP32 at the edges of the kernel's tiling: widths around 2, 4 and 8 per launch, boxes of
one point, of just under and over 32 (a target group) and of more than 128, lists shorter than a sub-chunk and of many
chunks (added results), every target-group size, both layouts, an odd leading dimension.

Tolerance: the FP32 paths' per-target bound |err_i| <= 2^-20 S_i, S_i = sum_j |G(r_ij) lambda_j|."""
import numpy as np
import pytest

import oracle
from paper_2403_01596_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ng,tuning", [(1, 2, None), (33, 1, None), (300, 7, None), (2100, 4, {"chunk": 32}),
                                         (1500, 2, {"target_group": 128}), (4000, 5, {"target_group": 64, "chunk": 1024})])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
@pytest.mark.parametrize("layout", ["indexed", "redundant"])
def test_widths(n, ng, tuning, kernel, layout):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import _capi as C, api
    pts = np.random.default_rng(n).random((n, 3)).astype(np.float32)
    if n > 40:
        pts[:20] = pts[20:40]  # coincident points (r = 0)
    lo, h = (0.0, 0.0, 0.0), 1.0 / ng
    k = float(np.float32(2 * np.pi * ng / 4)) if kernel == "helmholtz" else 0.0
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, kernel=kernel, layout=layout, max_nrhs=15, tuning=tuning)
    lam = W.strengths(n, 15, n).reshape(n, 15)
    S = oracle.p2p(pts, np.abs(lam).astype(np.complex64), lo, h, ng, 0.0, kernel=oracle.LAPLACE).real.reshape(n, 15)
    for adjoint in (False, True):
        ref = oracle.p2p(pts, lam, lo, h, ng, k, kernel=kid, adjoint=adjoint).reshape(n, 15)
        for nrhs in (2, 3, 4, 5, 8, 9, 12, 15):
            # a window of a wider array: leading dimension 15
            lam_d = torch.from_numpy(lam).cuda()
            out = torch.full((n, 15), complex(7, 7), dtype=torch.complex64, device="cuda")
            C.p2p_apply_path(plan._plan, lam_d, out, nrhs, 15, int(adjoint), C.P2P_PATH_FP32_SHARED,
                             torch.cuda.current_stream())
            got = out.cpu().numpy()
            assert plan.async_status() == 0
            assert (np.abs(got[:, :nrhs] - ref[:, :nrhs]) <= 2.0 ** -20 * S[:, :nrhs]).all(), nrhs
            assert (got[:, nrhs:] == complex(7, 7)).all()


@pytest.mark.parametrize("n,ng,flat", [(2000, 12, False), (5000, 16, False), (55000, 46, True), (57000, 46, True)])
@pytest.mark.parametrize("kernel,layout", [("helmholtz", "indexed"), ("laplace", "redundant")])
def test_two_on_both_sides_of_the_kernel_choice(n, ng, flat, kernel, layout):
    """Two right-hand sides with few boxes, with boxes of few points, and with boxes of just under and just over the
    points at which the streamed kernel is left, against the oracle and against each alone; same bound (twice it
    between two computed results)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    pts = np.random.default_rng(n).random((n, 3)).astype(np.float32)
    if flat:
        pts[:, 2] = 0.5
    lo, h = (0.0, 0.0, 0.0), 1.0 / ng
    k = float(np.float32(2 * np.pi * ng / 4)) if kernel == "helmholtz" else 0.0
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, kernel=kernel, layout=layout, max_nrhs=2)
    lam = W.strengths(n, 2, n).reshape(n, 2)
    S = oracle.p2p(pts, np.abs(lam).astype(np.complex64), lo, h, ng, 0.0, kernel=oracle.LAPLACE).real.reshape(n, 2)
    ref = oracle.p2p(pts, lam, lo, h, ng, k, kernel=kid, adjoint=True).reshape(n, 2)
    lam_d = torch.from_numpy(lam).cuda()
    got = plan.apply(lam_d, adjoint=True).cpu().numpy()
    alone = np.stack([plan.apply(lam_d[:, q].contiguous(), adjoint=True).cpu().numpy() for q in range(2)], 1)
    assert plan.async_status() == 0
    assert (np.abs(got - ref) <= 2.0 ** -20 * S).all()
    assert (np.abs(got - alone) <= 2.0 ** -19 * S).all()


@pytest.mark.parametrize("share,radius", [(0.0, 0.0), (0.3, 0.03)])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
def test_gradient_of_even_and_clustered_geometries(share, radius, kernel):
    """The coordinate gradient on both launch shapes: points spread over a cube, and with a cluster whose box is worth many
    average warps.  Tolerance: relative L2 1e-5, as for every FP32 result against the oracle."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    n, ng = 20_000, 11
    rng = np.random.default_rng(6)
    pts = rng.random((n, 3))
    m = int(share * n)
    pts[:m] = 0.5 + radius * rng.random((m, 3))
    pts = pts.astype(np.float32)
    lo, h = (0.0, 0.0, 0.0), 1.0 / ng
    k = float(np.float32(2 * np.pi * ng / 4)) if kernel == "helmholtz" else 0.0
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, kernel=kernel)
    lam, g = W.strengths(n, 1, 7), W.strengths(n, 1, 8)
    got = plan.grad_points(torch.from_numpy(lam).cuda(), torch.from_numpy(g).cuda()).cpu().numpy()
    assert plan.async_status() == 0
    ref = oracle.grad_points(pts, lam, g, lo, h, ng, k, kernel=kid)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5


@pytest.mark.parametrize("share", [0.0, 0.3])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
def test_two_with_and_without_a_cluster(share, kernel):
    """Two right-hand sides on a plan of many boxes, streamed, and with a box that decides the time, staged; same bound."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    n, ng = 30_000, 16
    rng = np.random.default_rng(9)
    pts = rng.random((n, 3))
    m = int(share * n)
    pts[:m] = 0.5 + 0.02 * rng.random((m, 3))
    pts = pts.astype(np.float32)
    lo, h = (0.0, 0.0, 0.0), 1.0 / ng
    k = float(np.float32(2 * np.pi * ng / 4)) if kernel == "helmholtz" else 0.0
    kid = oracle.HELMHOLTZ if kernel == "helmholtz" else oracle.LAPLACE
    plan = api.Plan(torch.from_numpy(pts).cuda(), lo, h, ng, k, kernel=kernel, max_nrhs=2)
    assert plan.num_boxes >= 2048 and plan.num_boxes ** 2 >= 80 * n
    lam = W.strengths(n, 2, n).reshape(n, 2)
    got = plan.apply(torch.from_numpy(lam).cuda()).cpu().numpy()
    assert plan.async_status() == 0
    S = oracle.p2p(pts, np.abs(lam).astype(np.complex64), lo, h, ng, 0.0, kernel=oracle.LAPLACE).real.reshape(n, 2)
    ref = oracle.p2p(pts, lam, lo, h, ng, k, kernel=kid).reshape(n, 2)
    assert (np.abs(got - ref) <= 2.0 ** -20 * S).all()
