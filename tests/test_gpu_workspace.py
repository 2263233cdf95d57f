"""Plans whose work items and boxes number just under 2^18 while the workspace is sized for a bound above it, where the
radix sort needs the most scratch for its count: plan creation and the apply stay inside the workspace."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_01596_gb300 import _capi as C  # noqa: E402
from paper_2403_01596_gb300 import workloads as W  # noqa: E402

GUARD = 1 << 20


def _api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    return api


def _plate(n, seed, share=1.0):
    p = torch.rand(n, 3, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
    p[:, 0] *= share
    p[:, 2] = 0.5
    return p.contiguous()


# (targets, sources or None for one set, boxes per axis, share of the plate, kernel request): the item bound lies above
# 2^18, the boxes between 130 000 and 2^18; the scratch of the smaller plans is the last part of their workspace
@pytest.mark.parametrize("n,n_src,ng,share,request_", [(790_000, None, 512, 1.0, 0), (600_000, None, 512, 1.0, 0),
                                                       (600_000, None, 512, 1.0, -1), (1 << 20, None, 512, 1.0, 8),
                                                       (1 << 20, 2_000_000, 426, 1.0, 0), (1 << 20, 1_500_000, 512, 0.75, 4)])
def test_plan_stays_in_its_workspace(n, n_src, ng, share, request_):
    api = _api()
    lo, h, tuning = (0.0, 0.0, 0.0), 1.0 / ng, {"warp_boxes": request_}
    tgt = _plate(n, n, share)
    lam = torch.from_numpy(W.strengths(n_src or n, 1, 5)).cuda()
    if n_src:
        src = _plate(n_src, n_src + 1, share)
        st = api.TwoSetStructure(tgt, src, lo, h, ng)
        t, s = st.tgt, st.src
        ws = C.p2p_plan_workspace_size_st(n, t.num_boxes, n_src, s.num_boxes, st.nnz, st.sources, C.P2P_LAYOUT_INDEXED, 1, tuning)
        boxes = t.num_boxes
    else:
        st = api.BoxStructure(tgt, lo, h, ng)
        ws = C.p2p_plan_workspace_size(n, st.num_boxes, st.nnz, st.sources, C.P2P_LAYOUT_INDEXED, 1, tuning)
        boxes = st.num_boxes
    assert 130_000 < boxes <= 1 << 18 < st.sources // 128 + boxes + 1
    buf = torch.full((ws + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    work = buf[:ws]
    if n_src:
        plan = C.p2p_plan_create_st(t.points, t.perm, t.box_ptr, t.num_boxes, s.points, s.perm, s.box_ptr, s.num_boxes,
                                    st.nbr_ptr, st.nbr_idx, st.nbr_self, st.nnz, st.sources, C.P2P_LAPLACE, 0.0,
                                    C.P2P_LAYOUT_INDEXED, 1, tuning, work, 0)
    else:
        plan = C.p2p_plan_create(st.points, st.perm, st.box_ptr, st.num_boxes, st.nbr_ptr, st.nbr_idx, st.nnz, st.sources,
                                 C.P2P_LAPLACE, 0.0, C.P2P_LAYOUT_INDEXED, 1, tuning, work, 0)
    try:
        out = torch.empty(n, dtype=torch.complex64, device="cuda")
        C.p2p_apply_path(plan, lam, out, 1, 1, 0, C.P2P_PATH_AUTO, 0)
        assert C.p2p_last_async_status(plan, 0) == 0
        assert bool((buf[ws:] == 0xA5).all())
        # every box was computed once: a few targets against the sums over all sources near them in 64 bits
        pts, lamh = (st.src.points if n_src else tgt).double(), lam.to(torch.complex128)
        for i in np.random.default_rng(0).choice(n, 20, replace=False):
            x = tgt[int(i)].double()
            cell = torch.floor(x / h)
            near = ((torch.floor(pts / h) - cell).abs() <= 1).all(dim=1)
            r = (pts[near] - x).norm(dim=1)
            keep = r > 0
            g = 1.0 / (4.0 * np.pi * r[keep])
            ref = (g * lamh[near][keep]).sum()
            S = (g * lamh[near][keep].abs()).sum()
            assert abs(complex(out[int(i)].item()) - complex(ref.item())) <= 2.0 ** -20 * float(S) + 1e-30
    finally:
        C.p2p_plan_destroy(plan)
