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


# FP32 grids of 32 x 8 tiles are staged by tensor copies from 3/4 of a tile per resident CTA on (four CTAs per SM), with
# the domain-mean buoyancy from two tiles: the grids of 320 and 640 columns on either side of each line.
@pytest.mark.parametrize("mean,nx,per_sm", [(False, 320, 3), (True, 640, 8)], ids=["plain", "mean"])
def test_fp32_steps_on_both_sides_of_the_staging_line(mean, nx, per_sm):
    """The binary32 step against the binary64 one: 30 steps, the parity tests' 1e-4 (u against its largest value)."""
    import torch

    from .helpers import max_rel, norm_rel

    line = per_sm * torch.cuda.get_device_properties(0).multi_processor_count  # tiles
    rows = [(line - 1) // (nx // 32) * 8, -(-line // (nx // 32)) * 8]
    assert rows[0] // 8 * (nx // 32) < line <= rows[1] // 8 * (nx // 32)
    for ny, names in zip(rows, (["k_fused"], ["k_fused", "k_finish"] if mean else ["k_fused"])):
        if mean:
            case, rho, T = workloads.mixed_small(TC, RV, RL, nx=nx, ny=ny)
        else:
            case, rho, T = workloads.droplet_evaporation(TC, RV, RL, n=max(nx, ny), radius=60.0, dT_ratio=0.1)
            case, rho, T = dict(case, nx=nx, ny=ny), rho[:ny, :nx].copy(), T[:ny, :nx].copy()
        out = []
        for prec in (lbpc.FP32, lbpc.FP64):
            sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
            sim.init(rho, T)
            sim.step(29)
            got = sim.step_timed()
            assert prec == lbpc.FP64 or list(got) == names
            out.append(sim.fields())
            sim.close()
        a, b = out
        assert max_rel(a[0], b[0]) <= 1e-4 and max_rel(a[3], b[3]) <= 1e-4
        assert norm_rel(a[1], b[1]) <= 1e-4 and norm_rel(a[2], b[2]) <= 1e-4


@pytest.mark.parametrize("prec", [lbpc.FP32, lbpc.FP16DEV], ids=["fp32", "fp16"])
def test_persistent_just_above_its_line(prec):
    """More than five tiles per resident CTA (four CTAs per SM) run persistent: the first such grid of 1001 columns
    (padded rows) gives the bits of one CTA per tile."""
    import numpy as np
    import torch

    rows = 5 * 4 * torch.cuda.get_device_properties(0).multi_processor_count // 32 + 1
    case, rho, T = workloads.mixed_small(TC, RV, RL, nx=1001, ny=8 * rows - 3)
    out = []
    for tile in (4, 1):
        sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
        sim.set_fused_tile(tile)
        sim.init(rho, T)
        sim.step(8)
        out.append(sim.fields())
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
