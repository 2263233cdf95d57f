"""Workspace queries around the counts at which the radix sort takes larger tiles (2^18 and 2^22 keys): a workspace for
more points, sources or boxes is never the smaller one, so what was sized for a bound holds every count below it."""
import pytest

from paper_2403_01596_gb300 import _capi as C

STEPS = (1 << 18, 1 << 22)


@pytest.mark.parametrize("step", STEPS)
def test_binning_workspace_never_falls(step):
    sizes = [C.p2p_bin_workspace_size(n) for n in (step // 2 + 1, step - 1, step, step + 1, step + 4096, 2 * step)]
    assert sizes == sorted(sizes)


# one kernel request each: the tables of the box-group kernel are a choice of the plan that may come and go with the boxes
@pytest.mark.parametrize("step", STEPS)
@pytest.mark.parametrize("warp_boxes", [-1, 4, -2])
@pytest.mark.parametrize("two_sets", [False, True])
def test_plan_workspace_never_falls(step, warp_boxes, two_sets):
    """The item bound (sources / 128 + boxes + 1) crosses the step first with the sources, then with the boxes."""
    tuning = {"warp_boxes": warp_boxes}
    nb = int(0.9 * step)
    n, nnz, at = 3 * nb, 6 * nb, 128 * (step - nb - 1)

    def size(sources, boxes):
        if two_sets:
            return C.p2p_plan_workspace_size_st(n, boxes, n // 8, boxes // 8, nnz, sources, C.P2P_LAYOUT_INDEXED, 1, tuning)
        return C.p2p_plan_workspace_size(n, boxes, nnz, sources, C.P2P_LAYOUT_INDEXED, 1, tuning)

    by_sources = [size(at + d, nb) for d in (-128 * 4096, -128, -1, 0, 127, 128, 128 * 4096)]
    assert by_sources == sorted(by_sources)
    by_boxes = [size(at, nb + d) for d in (-4096, -1, 0, 1, 4096)]
    assert by_boxes == sorted(by_boxes)
