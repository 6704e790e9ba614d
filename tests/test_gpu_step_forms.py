"""The forms a step can take, at the sizes where each can go wrong: the two-kernel binary64 and double-word
step at the edges of its tiles, the persistent and per-tile forms of the fused step on rows that the library
pads, the batch walked by persistent CTAs, and the sums written to each kind of memory."""

import numpy as np
import pytest

from oracle import model
from paper_1709_04400_gb300 import lbpc, workloads

from .helpers import RL, RV, TC, max_rel, norm_rel, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    from paper_1709_04400_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def _fields(case, rho, T, steps, prec, path=lbpc.PATH_AUTO, tile=None):
    sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
    sim.set_path(path)
    if tile is not None:
        sim.set_fused_tile(tile)
    sim.init(rho, T)
    sim.step(steps)
    out = sim.fields()
    sim.close()
    return out


# Tiles of the two-kernel step are 16 x 8 nodes: one below, at and above one and two of them. The bar is the parity
# tests' 1e-10.
@pytest.mark.parametrize("prec", [lbpc.FP64, lbpc.DF64], ids=["fp64", "df64"])
@pytest.mark.parametrize("nx,ny", [(15, 23), (16, 24), (17, 25), (31, 31), (33, 33)])
@pytest.mark.parametrize("walls", [False, True], ids=["ring", "walls"])
def test_two_kernel_step_at_tile_edges(prec, nx, ny, walls):
    if walls:  # wall with strip, pressure top, mean buoyancy, rates that differ, lambda = rho c_V chi
        case, rho, T = workloads.mixed_small(TC, RV, RL, nx=nx, ny=ny)
    else:
        case, rho, T = workloads.droplet_evaporation(TC, RV, RL, n=max(nx, ny), radius=4.0, dT_ratio=0.1)
        case, rho, T = dict(case, nx=nx, ny=ny), rho[:ny, :nx].copy(), T[:ny, :nx].copy()
    got = _fields(case, rho, T, 20, prec, lbpc.PATH_SPLIT)
    p, s = run_oracle(case, rho, T, 20)
    ref = model.fields(p, s)
    assert max_rel(got[0], ref[0]) <= 1e-10 and max_rel(got[3], ref[3]) <= 1e-10
    assert norm_rel(got[1], ref[1]) <= 1e-10 and norm_rel(got[2], ref[2]) <= 1e-10


def test_two_kernel_step_wide_tiles():
    """From 2^20 nodes binary64 takes 32 x 8 tiles: a ragged grid just above, against the one-kernel step. Both
    evaluate the same step in binary64 (round-off of 1e-16 per operation, three steps; u against its largest
    value)."""
    case, rho, T = workloads.droplet_evaporation(TC, RV, RL, n=1031, radius=180.0, dT_ratio=0.1)
    a = _fields(case, rho, T, 3, lbpc.FP64, lbpc.PATH_SPLIT)
    b = _fields(case, rho, T, 3, lbpc.FP64, lbpc.PATH_FUSED)
    assert max_rel(a[0], b[0]) <= 1e-13 and max_rel(a[3], b[3]) <= 1e-13
    assert norm_rel(a[1], b[1]) <= 1e-10 and norm_rel(a[2], b[2]) <= 1e-10


# More than 5 (FP32) or 12 (FP16) tiles per resident CTA run persistent; odd widths have padded rows, the last
# tiles of a row and the last rows are partial, and every edge kind occurs.
@pytest.mark.parametrize("prec,nx,ny", [(lbpc.FP32, 1023, 1101), (lbpc.FP16DEV, 1543, 1209)], ids=["fp32", "fp16"])
def test_persistent_step_on_padded_rows(prec, nx, ny):
    for case, rho, T in (workloads.mixed_small(TC, RV, RL, nx=nx, ny=ny),
                         workloads.droplet_evaporation(TC, RV, RL, n=nx, radius=0.2 * nx, dT_ratio=0.2)):
        for a, b in zip(_fields(case, rho, T, 12, prec, tile=4), _fields(case, rho, T, 12, prec, tile=1)):
            assert np.array_equal(a, b), case["name"]


@pytest.mark.parametrize("prec", [lbpc.FP32, lbpc.FP16DEV], ids=["fp32", "fp16"])
@pytest.mark.parametrize("nx", [63, 64, 65, 67, 70])
def test_checkpoint_has_no_padding(prec, nx):
    """Rows of 65, 67 and 70 elements are padded in the context but not in a checkpoint, whose bytes are the same in
    host and device memory and resume bit for bit."""
    import torch

    case, rho, T = workloads.mixed_small(TC, RV, RL, nx=nx, ny=41)
    sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
    sim.init(rho, T)
    sim.step(5)
    nodes, half = nx * 41, prec == lbpc.FP16DEV
    want = 512 + 18 * nodes * (2 if half else 4) + (8 * nodes if half else 0) + 4 * nodes + 4 * nx * 8
    assert sim.checkpoint_bytes() == want
    host = sim.save()
    dev = sim.save(torch.empty(want, dtype=torch.uint8, device="cuda"))
    assert np.array_equal(host, dev.cpu().numpy())
    sim.step(6)
    ref = sim.fields()
    for ck in (host, dev):
        other = lbpc.Simulation(lbpc.params_from_case(case, prec))
        other.load(ck)
        other.step(6)
        for a, b in zip(other.fields(), ref):
            assert np.array_equal(a, b)
        other.close()
    sim.close()


@pytest.mark.parametrize("prec", [lbpc.FP32, lbpc.FP16DEV], ids=["fp32", "fp16"])
def test_batch_walk_equals_alone(prec):
    """A batch whose launch is walked by persistent CTAs (12,288 tiles of large instances) beside instances without
    tensor maps (60 columns), with padded rows, with walls: each equals, bit for bit, its run in a batch of its own."""
    cases = [workloads.droplet_evaporation(TC, RV, RL, n=1021, radius=200.0, dT_ratio=d) for d in (0.05, 0.1, 0.2)]
    cases += [workloads.droplet_evaporation(TC, RV, RL, n=60, radius=14.0, dT_ratio=0.1),
              workloads.mixed_small(TC, RV, RL, nx=131, ny=75), workloads.droplet_periodic(TC, RV, RL, n=97, radius=20.0)]

    def run(some):
        ps = [lbpc.params_from_case(c, prec) for c, _, _ in some]
        b = lbpc.Batch(prec, sum(lbpc.Batch.instance_bytes(p) for p in ps) + (256 << 20), max_instances=8)
        ids = [b.add(p, r, t) for p, (_, r, t) in zip(ps, some)]
        b.step(20)
        b.check()
        out = [b.fields(i) for i in ids]
        b.close()
        return out

    together = run(cases)
    for k in (0, 3, 4, 5):
        for a, b in zip(together[k], run([cases[k]])[0]):
            assert np.array_equal(a, b), cases[k][0]["name"]


@pytest.mark.parametrize("prec", [lbpc.FP64, lbpc.FP32], ids=["fp64", "fp32"])
def test_sums_to_every_kind_of_memory(prec):
    """lbpc_sums_async into device, pinned and pageable memory, and lbpc_sums, give the same two numbers; the grid of
    1031 x 1029 takes four nodes per thread, the other one."""
    import torch

    for n in (45, 1031):
        case, rho, T = workloads.droplet_evaporation(TC, RV, RL, n=n, radius=0.2 * n, dT_ratio=0.1)
        sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
        sim.init(rho, T)
        sim.step(3)
        outs = [torch.zeros(2, dtype=torch.float64, device="cuda"), torch.zeros(2, dtype=torch.float64, pin_memory=True),
                torch.zeros(2, dtype=torch.float64)]
        for o in outs:
            sim.sums_async(o)
        sim.check()
        want = sim.sums()
        for o in outs:
            assert tuple(o.cpu().tolist()) == want
        got = sim.fields()
        assert abs(want[0] / got[0].sum() - 1.0) < 1e-6 and abs(want[1] / got[3].sum() - 1.0) < 1e-6
        sim.close()


@pytest.mark.parametrize("prec", [lbpc.FP64, lbpc.FP32, lbpc.FP16DEV, lbpc.DF64], ids=["fp64", "fp32", "fp16", "df64"])
@pytest.mark.parametrize("n", [11, 363, 600, 1031])
def test_sums_of_the_populations(prec, n):
    """The sums against the exported populations: one block that is partly filled (11 x 11), a last block that is, in
    rows with and without padding (363 x 363), populations widened from their bits in every storage (from 600 x 600
    on), four nodes per thread (1031 x 1031). Fewer than 100 additions lead to a total of positive numbers, so it is
    within 100 x 2^-53 = 1.1e-14 of the exact one; numpy's own pairwise sum is as good, and 1e-13 leaves room for
    both."""
    case, rho, T = workloads.droplet_evaporation(TC, RV, RL, n=n, radius=0.2 * n, dT_ratio=0.1)
    sim = lbpc.Simulation(lbpc.params_from_case(case, prec))
    sim.init(rho, T)
    sim.step(2)
    mass, heat = sim.sums()
    f, g = sim.populations()
    assert sim.sums() == (mass, heat)
    sim.close()
    assert abs(mass / f.sum() - 1.0) < 1e-13 and abs(heat / g.sum() - 1.0) < 1e-13
