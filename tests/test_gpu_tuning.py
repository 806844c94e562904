"""What the autotuner may change: an FP64 run keeps the launch shapes of the FP32 kernels,
and a plan without rows of the tiled kernels keeps its tile shape."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _autotune(plan, dtype):
    q = torch.rand(plan.n_cells, dtype=dtype, device=DEV) + 1.0
    v0 = torch.full((plan.n_rows,), 0.3, dtype=torch.float64, device=DEV)
    before = plan.tuning().as_dict()
    after = ram.autotune(plan, q, torch.empty_like(q), v0, 0.1, reps=2).as_dict()
    return {k for k in before if before[k] != after[k]}


@pytest.mark.parametrize("a4", [False, True])
def test_fp64_run_keeps_the_fp32_shapes(a4):
    n = 1024
    plan = ram.Plan(np.arange(9) * n, wl.uniform_nodes(n), order=3, shared_mesh=True, a4=a4)
    assert plan.tuning().seg_variant_f32 == 2
    assert _autotune(plan, torch.float64) <= {"uniform_kernel_f64", "rows_cells_per_thread_f64"}
    assert plan.check_errors() == 0


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("uniform", [True, False])
def test_tile_shape_stays_without_tiled_rows(dtype, uniform):
    n = 2048
    x = wl.uniform_nodes(n) if uniform else wl.random_nodes(n, seed=1)
    plan = ram.Plan(np.arange(5) * n, x, order=3, shared_mesh=True)
    t = plan.tuning()
    t.tile_cells, t.threads = 640, 96  # not among the candidates
    plan.set_tuning(t)
    assert not _autotune(plan, dtype) & {"tile_cells", "threads"}
    assert plan.check_errors() == 0
