"""The kernels that lbpc_step_timed times and lbpc_kernel_name names, for each form of a step."""

import pytest

from paper_1709_04400_gb300 import lbpc, workloads

from .helpers import RL, RV, TC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    from paper_1709_04400_gb300 import build

    build.build()
    torch.cuda.set_device(0)


# With the domain-mean buoyancy the mean is a kernel of its own, except where the last block of an unstaged fused step
# takes it.
@pytest.mark.parametrize("prec,path,n,mean,want", [
    (lbpc.FP64, lbpc.PATH_SPLIT, 64, True, ["k_macro", "k_collide_tile", "k_finish"]),
    (lbpc.DF64, lbpc.PATH_SPLIT, 64, False, ["k_macro", "k_collide_tile"]),
    (lbpc.FP32, lbpc.PATH_SPLIT, 64, True, ["k_macro", "k_force", "k_collide", "k_finish"]),
    (lbpc.FP64, lbpc.PATH_FUSED, 64, True, ["k_fused"]),
    (lbpc.FP32, lbpc.PATH_FUSED, 64, True, ["k_fused"]),
    (lbpc.FP32, lbpc.PATH_FUSED, 600, True, ["k_fused", "k_finish"]),  # staged
    (lbpc.FP32, lbpc.PATH_FUSED, 1200, True, ["k_fused", "k_finish"]),  # persistent
    (lbpc.FP16DEV, lbpc.PATH_FUSED, 64, True, ["k_fused", "k_finish"]),
    (lbpc.FP16DEV, lbpc.PATH_FUSED, 64, False, ["k_fused"]),
])
def test_each_kernel_of_a_step_is_timed(prec, path, n, mean, want):
    if mean:
        case, rho, T = workloads.mixed_small(TC, RV, RL, nx=n, ny=n)
    else:
        case, rho, T = workloads.droplet_periodic(TC, RV, RL, n=n, radius=14.0)
    sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
    sim.set_path(path)
    sim.init(rho, T)
    for _ in range(2):  # both buffers as the source
        got = sim.step_timed()
        assert list(got) == want and all(v > 0.0 for v in got.values())
    sim.close()
