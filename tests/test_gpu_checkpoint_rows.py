"""Checkpoints of grids with padded rows: packed and unpacked by a kernel, straight or through scratch, or by pitched
copies (device buffers that are not aligned, long rows on their way to the host); the same bytes every way, and they
resume bit for bit."""

import numpy as np
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


# 65: a warp's row with a remainder of one; 127, 129 and 161: rows that end around whole warps; 1027 rows: many blocks; 601:
# eight elements per lane, and rows of more than 1 KB, which go to the host by pitched copies.
@pytest.mark.parametrize("prec", [lbpc.FP32, lbpc.FP16DEV], ids=["fp32", "fp16"])
@pytest.mark.parametrize("nx,ny", [(65, 8), (127, 40), (129, 1027), (161, 33), (601, 17)])
def test_every_kind_of_buffer(prec, nx, ny):
    import torch

    case, rho, T = workloads.mixed_small(TC, RV, RL, nx=nx, ny=ny)
    sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
    sim.init(rho, T)
    sim.step(5)
    n = sim.checkpoint_bytes()
    host = sim.save()
    room = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")
    shifted = [room[k : k + n] for k in (0, 1, 2, 4)]
    pinned = torch.zeros(n, dtype=torch.uint8).pin_memory().numpy()
    for buf in shifted + [pinned]:
        sim.save(buf)
        assert np.array_equal(buf if buf is pinned else buf.cpu().numpy(), host)
    sim.step(6)  # the scratch that saving used is written before it is read
    want = sim.fields()
    for k in (0, 1, 2, 4, None, "pinned"):
        other = lbpc.Simulation(lbpc.params_from_case(case, prec))
        if isinstance(k, int):
            src = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")[k : k + n]
            src.copy_(torch.from_numpy(host))
        else:
            src = pinned if k else host
        other.load(src)
        assert np.array_equal(other.save(), host)
        other.step(6)
        for a, b in zip(other.fields(), want):
            assert np.array_equal(a, b)
        other.close()
    sim.close()
