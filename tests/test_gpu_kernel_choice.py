"""The kernel a plan chooses for one right-hand side, at box counts on both sides of every line of the choice, and the
batched box-group launch: results against the staged pipeline on the same plan data.

Tolerance: both evaluate the same FP32 terms in another order; each is within 2^-20 S_i of the exact sum, so they
differ by at most 2^-19 S_i, S_i = sum_j |G(r_ij) lambda_j| (the Laplace apply of |lambda|)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2403_01596_gb300 import workloads as W  # noqa: E402


def _api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_01596_gb300 import api
    return api


def _close(api, plan, pts, lo, h, ng, lam, out):
    ref = api.Plan(pts, lo, h, ng, plan.k, kernel=plan.kernel, tuning={"warp_boxes": -1}).apply(lam)
    S = api.Plan(pts, lo, h, ng, kernel="laplace", tuning={"warp_boxes": -1}).apply(lam.abs().to(torch.complex64)).real
    return bool(((out - ref).abs() <= 2.0 ** -19 * S + 1e-30).all())


# points in the unit cube, boxes per axis (all of them occupied or nearly): box counts around 2 500, 6 000, 15 000 and
# 45 000 at 1 to 30 points per box
@pytest.mark.parametrize("n,ng", [(1500, 12), (2900, 14), (6000, 13), (6500, 14), (13000, 14), (22000, 13), (24000, 14),
                                  (31000, 14), (50000, 14), (110000, 18), (125000, 19), (40000, 24), (43000, 25),
                                  (100000, 24), (106000, 25), (270000, 35), (290000, 36), (200000, 14)])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
@pytest.mark.parametrize("layout", ["indexed", "redundant"])
def test_choice(n, ng, kernel, layout):
    api = _api()
    pts = torch.rand(n, 3, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    lo, h = (0.0, 0.0, 0.0), 1.0 / ng
    lam = torch.from_numpy(W.strengths(n, 1, n)).cuda()
    plan = api.Plan(pts, lo, h, ng, 2 * np.pi * ng / 4, kernel=kernel, layout=layout)
    out = plan.apply(lam)
    assert plan.async_status() == 0
    assert _close(api, plan, pts, lo, h, ng, lam, out), plan.info


@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
def test_batched_groups(kernel):
    """Plans on the box-group kernel in one launch: every plan's rows equal its own apply bit for bit (the same
    members swept the same way), eagerly, replayed, and after the strengths change."""
    api = _api()
    plans, lams = [], []
    for i, (n, ng, request) in enumerate([(3000, 6, -2), (1, 2, -2), (17, 1, -2), (40001, 14, 0), (5000, 7, -2)]):
        pts = torch.rand(n, 3, generator=torch.Generator(device="cuda").manual_seed(i), device="cuda")
        plans.append(api.Plan(pts, (0.0, 0.0, 0.0), 1.0 / ng, ng, 2 * np.pi * ng / 4, kernel=kernel,
                              tuning={"warp_boxes": request}))
        assert plans[-1].info["tuning"]["warp_boxes"] == -2
        lams.append(torch.from_numpy(W.strengths(n, 1, i)).cuda())
    src = torch.rand(900, 3, generator=torch.Generator(device="cuda").manual_seed(9), device="cuda") * 0.4
    two = api.TwoSetPlan(plans[0].structure.points, src, (0.0, 0.0, 0.0), 1.0 / 6, 6, 9.0, kernel=kernel,
                         tuning={"warp_boxes": -2})
    plans.append(two)
    lams.append(torch.from_numpy(W.strengths(900, 1, 9)).cuda())
    batch = api.Batch(plans)
    for o, p, l in zip(batch.apply(lams), plans, lams):
        assert torch.equal(o[:, 0], p.apply(l))
    outs = batch.capture(lams)
    for scale in (1.0, 2.0):
        for l in lams:
            l.mul_(scale)
        batch.replay()
        for o, p, l in zip(outs, plans, lams):
            assert torch.equal(o[:, 0], p.apply(l)) and p.async_status() == 0


def test_batch_info_reports_the_launch():
    """A batch on the box-group launch reports its groups, blocks of 8 warps and a grid no larger than the groups; a
    caller that names the warps per block gets the staged launch of that shape, with the same results."""
    api = _api()
    plans, lams = [], []
    for i, (n, ng) in enumerate([(3000, 6), (1500, 5)]):
        pts = torch.rand(n, 3, generator=torch.Generator(device="cuda").manual_seed(i), device="cuda")
        plans.append(api.Plan(pts, (0.0, 0.0, 0.0), 1.0 / ng, ng, 9.0, tuning={"warp_boxes": -2}))
        lams.append(torch.from_numpy(W.strengths(n, 1, i)).cuda())
    group = api.Batch(plans)
    groups = sum(-(-p.num_boxes // 16) for p in plans)
    assert (group.info["work_items"], group.info["warps_per_cta"]) == (groups, 8) and 0 < group.info["grid"] <= groups
    staged = api.Batch(plans, warps_per_cta=4)
    assert staged.info["work_items"] == sum(p.info["work_items"] for p in plans) and staged.info["warps_per_cta"] == 4
    for o, s, p, l in zip(group.apply(lams), staged.apply(lams), plans, lams):
        assert torch.equal(o[:, 0], p.apply(l))
        st = p.structure
        assert _close(api, p, st.points, st.lo, st.h, st.ng, l, s[:, 0])


def test_batch_takes_groups_only_where_no_box_decides():
    """Spheres of ~18 points per box on the box-group kernel by their own choice: one alone has too little work for the
    boxes that single warps sweep and runs the staged launch, sixteen together the box-group launch; a plan whose tuning
    names the kernel keeps it."""
    api = _api()
    lo, ng = (-1.0, -1.0, -1.0), 16
    plans, lams = [], []
    for i in range(16):
        pts = torch.from_numpy(W.unit_sphere(20000, 4 + i)).cuda()
        plans.append(api.Plan(pts, lo, 2.0 / ng, ng, 9.0))
        assert plans[-1].info["tuning"]["warp_boxes"] == -2
        lams.append(torch.from_numpy(W.strengths(20000, 1, i)).cuda())
    asked = [api.Plan(plans[0].structure.points, lo, 2.0 / ng, ng, 9.0, tuning={"warp_boxes": -2})]
    groups = lambda ps: sum(-(-p.num_boxes // 16) for p in ps)  # noqa: E731
    for ps, own in ((plans[:1], False), (plans, True), (asked, True)):
        batch = api.Batch(ps)
        assert batch.info["work_items"] == (groups(ps) if own else sum(p.info["work_items"] for p in ps))
        for o, p, l in zip(batch.apply(lams[:len(ps)]), ps, lams):
            assert p.async_status() == 0 and _close(api, p, p.structure.points, lo, 2.0 / ng, ng, l, o[:, 0])


# a geometry whose mean occupancy names the direct or the box-group kernel, evenly spread and with a dense cap
@pytest.mark.parametrize("n,ng,cap,radius", [(100_000, 80, 0.0, 0.0), (100_000, 80, 0.01, 0.01), (60_000, 44, 0.0, 0.0),
                                             (60_000, 44, 0.02, 0.02), (400_000, 160, 0.01, 0.01)])
@pytest.mark.parametrize("kernel", ["helmholtz", "laplace"])
@pytest.mark.parametrize("layout", ["indexed", "redundant"])
def test_heaviest_box(n, ng, cap, radius, kernel, layout):
    """A plan left to choose takes the staged pipeline where one box holds a cluster, and what its mean occupancy says
    otherwise; a request is kept either way."""
    api = _api()
    pts = W.unit_sphere(n, 7).astype(np.float64)
    m = int(cap * n)
    if m:
        q = np.random.default_rng(8).normal(size=(m, 3)) * radius + [0.0, 0.6, 0.8]
        pts[:m] = q / np.linalg.norm(q, axis=1, keepdims=True)
    pts = torch.from_numpy(pts.astype(np.float32)).cuda()
    lo, h = (-1.0, -1.0, -1.0), 2.0 / ng
    lam = torch.from_numpy(W.strengths(n, 1, 9)).cuda()
    plan = api.Plan(pts, lo, h, ng, 2 * np.pi * 0.25 / h, kernel=kernel, layout=layout)
    even = -2 if ng == 44 and layout == "indexed" else (-1 if ng == 44 else 4)
    assert plan.info["tuning"]["warp_boxes"] == (-1 if m else even)
    out = plan.apply(lam)
    assert plan.async_status() == 0 and _close(api, plan, pts, lo, h, ng, lam, out)
    if m and n == 60_000:
        asked = api.Plan(pts, lo, h, ng, plan.k, kernel=kernel, layout=layout, tuning={"warp_boxes": 2})
        assert asked.info["tuning"]["warp_boxes"] == 2 and _close(api, asked, pts, lo, h, ng, lam, asked.apply(lam))


# shape, points, boxes per axis, kernel, layout, expected: one point on either side of the lines that depend on the list
# length (plates 9, cubes up to 27 times the occupancy), the kernel function and the layout
@pytest.mark.parametrize("shape,n,ng,kernel,layout,want", [
    ("plate", 400_001, 211, "laplace", "indexed", 4), ("plate", 400_001, 211, "helmholtz", "indexed", -2),
    ("plate", 400_001, 211, "laplace", "redundant", -1), ("plate", 250_001, 177, "laplace", "redundant", 4),
    ("plate", 400_001, 356, "laplace", "indexed", 8), ("cube", 400_001, 50, "laplace", "indexed", 4),
    ("cube", 700_001, 61, "helmholtz", "indexed", 4), ("plate", 250_001, 201, "laplace", "indexed", 4),
    ("plate", 250_001, 201, "helmholtz", "indexed", 1), ("cube", 14_301, 10, "helmholtz", "indexed", -1),
    ("cube", 34_001, 13, "helmholtz", "indexed", -2)])
def test_choice_by_list_length_kernel_and_layout(shape, n, ng, kernel, layout, want):
    api = _api()
    gen = torch.Generator(device="cuda").manual_seed(1)
    pts, lo, h = torch.rand(n, 3, generator=gen, device="cuda"), (0.0, 0.0, 0.0), 1.0 / ng
    if shape == "plate":
        pts[:, 2] = 0.5
    plan = api.Plan(pts, lo, h, ng, 2 * np.pi * 0.25 / h, kernel=kernel, layout=layout)
    assert plan.info["tuning"]["warp_boxes"] == want, (n / plan.num_boxes, plan.num_boxes, plan.structure.sources / plan.num_boxes)
    lam = torch.from_numpy(W.strengths(n, 1, n)).cuda()
    out = plan.apply(lam)
    assert plan.async_status() == 0 and _close(api, plan, pts, lo, h, ng, lam, out)
