"""GPU test: one query gives the workspace that a call on a plan can use, the
largest of what the queries by kind of call give."""
import numpy as np
import pytest

from helpers import gpu_env, to_dev

pytestmark = pytest.mark.gpu


def test_one_query_gives_the_largest_of_the_others():
    torch = gpu_env()
    from paper_2212_10961_gb300 import field as F
    L = F.lib()
    rng = np.random.default_rng(3)
    grid = [np.ascontiguousarray(v.ravel().astype(np.float32))
            for v in np.meshgrid(np.arange(96) / 90, np.arange(80) / 80, np.arange(90) / 96, indexing="ij")[::-1]]
    cloud = list(rng.random((3, 200_000)).astype(np.float32))
    for cells, segments in ((grid, None), (cloud, None), (cloud[:2], None), ([c[:3000] for c in cloud], None),
                            (cloud, [10, 199_000, 990])):
        plan = F.CellPlan(*to_dev(torch, cells), segments=segments)
        for s in range(-1, len(segments or [1]) + 1):
            n = plan.segment_size(s)
            for modes in (100, 4096, 70_000, 2 ** 20):
                g, b = L.grf_synth_grid_workspace_bytes(plan.ptr, s, modes), L.grf_synth_band_workspace_bytes(plan.ptr, s, modes)
                assert F.synth_workspace_bytes(plan, s, modes) == max(L.grf_synth_workspace_bytes(n), g or b)
                for dim in (2, 3):
                    g = L.grf_backward_grid_workspace_bytes(plan.ptr, s, modes)
                    b = L.grf_backward_band_workspace_bytes(n, modes, dim)
                    assert F.backward_workspace_bytes(plan, s, modes, dim) == max(L.grf_backward_workspace_bytes(n, modes, dim), g or b)


@pytest.mark.parametrize("grid", [True, False])
def test_an_allocation_failure_reaches_the_call_not_the_query(grid):
    # the queries allocate nothing: the call that runs out of memory says so
    torch = gpu_env()
    from paper_2212_10961_gb300 import _abi, field as F
    c = np.random.default_rng(3).random((2, 3000)).astype(np.float32)
    if grid:
        c = np.stack([v.ravel().astype(np.float32) for v in np.meshgrid(np.arange(40) / 40, np.arange(50) / 50)])
    plan = F.CellPlan(*to_dev(torch, list(c)))
    p = F.FieldParams(family="gaussian", sigma2=1.0, ell=(0.1, 0.2), dim=2, n_modes=300, seed=4)
    gf = F.GaussianField(p)
    g = torch.ones(plan.n_cells, device="cuda")
    gf.synth(plan), F.backward(gf.table, p, plan, g)  # the plan's own check has been read
    for call in (lambda: gf.synth(plan), lambda: F.backward(gf.table, p, plan, g)):
        try:
            F.lib().grf_debug_inject_alloc_failures(1)
            with pytest.raises(_abi.GRFError) as e:
                call()
            assert e.value.code == _abi.GRF_ENOMEM
        finally:
            F.lib().grf_debug_inject_alloc_failures(0)
