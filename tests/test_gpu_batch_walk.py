"""Batches walked by persistent CTAs, against the same instances in forms that are not walked: an instance in the
block that another one of other sizes has left, and a step of which a second launch is a walk too."""

import numpy as np
import pytest

from paper_1709_04400_gb300 import lbpc, workloads

from .helpers import RL, RV, TC

pytestmark = pytest.mark.gpu

PRECS = pytest.mark.parametrize("prec", [lbpc.FP32, lbpc.FP16DEV], ids=["fp32", "fp16"])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    from paper_1709_04400_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def _batch(prec, cases, extra=128 << 20):
    ps = [lbpc.params_from_case(c, prec) for c, _, _ in cases]
    b = lbpc.Batch(prec, sum(lbpc.Batch.instance_bytes(p) for p in ps) + extra, max_instances=256)
    return b, [b.add(p, r, t) for p, (_, r, t) in zip(ps, cases)]


def _alone(prec, case, steps):
    """The instance in a batch of its own, one CTA per tile (the cases here have too few tiles to be walked alone)."""
    b, (i,) = _batch(prec, [case])
    b.step(steps)
    out = b.fields(i)
    b.close()
    return out


@PRECS
def test_instance_in_a_freed_block(prec):
    """A 97 x 1021 instance leaves a walked batch and one of 99 x 1021 takes its block: the padded rows are the same,
    so are the addresses of the tensor maps, and their widths differ. Its interior tile at x = 64 reads the columns 97
    and 98, which the first one's maps do not hold."""
    large = [workloads.droplet_evaporation(TC, RV, RL, n=1021, radius=200.0, dT_ratio=d) for d in (0.1, 0.2)]
    first, second = (workloads.mixed_small(TC, RV, RL, nx=nx, ny=1021) for nx in (97, 99))
    p, q = (lbpc.params_from_case(c, prec) for c, _, _ in (first, second))
    assert lbpc.Batch.instance_bytes(p) == lbpc.Batch.instance_bytes(q)
    b, ids = _batch(prec, [first] + large)  # the lowest block of the arena is the first instance's
    b.step(18)
    b.check()
    for got, want in zip(b.fields(ids[0]), _alone(prec, first, 18)):
        assert np.array_equal(got, want)
    free = b.free_bytes()
    b.remove(ids[0])
    i = b.add(q, second[1], second[2])
    assert b.free_bytes() == free
    b.step(18)
    b.check()
    for got, want in zip(b.fields(i), _alone(prec, second, 18)):
        assert np.array_equal(got, want)
    b.close()


def test_kernel_names_are_those_launched():
    """lbpc_batch_kernel_name tells the forms apart: the benchmark names and counts a step's launches by it."""
    large = [workloads.droplet_evaporation(TC, RV, RL, n=1021, radius=200.0, dT_ratio=d) for d in (0.1, 0.2)]
    small = [workloads.mixed_small(TC, RV, RL, nx=37, ny=29)]
    b, _ = _batch(lbpc.FP32, large)
    assert b.kernel_names() == ["k_batch_walk", "k_batch_advance"]
    b.set_config(3, 0)
    assert b.kernel_names() == ["k_batch_tiles", "k_batch_advance"]
    b.set_config(0, 4)
    assert b.kernel_names() == ["k_batch_step", "k_batch_advance"]
    b.close()
    for prec in (lbpc.FP64, lbpc.FP32, lbpc.FP16DEV):
        n = lbpc.Batch.per_tile_capacity(prec) + 1
        b, _ = _batch(prec, small * n)
        assert b.kernel_names() == ["k_batch_tiles"] * 2 + ["k_batch_advance"]
        b.close()


@PRECS
def test_second_launch_is_walked(prec):
    """More instances than a walk holds: the second walk starts while the first one ends and takes its own tickets.
    Each kind of instance equals, first, middle and last, its run alone by one CTA per tile; 20 steps are one by itself,
    a captured chunk of 16, and three more."""
    large = workloads.droplet_evaporation(TC, RV, RL, n=511, radius=100.0, dT_ratio=0.1)
    kinds = [large, workloads.mixed_small(TC, RV, RL, nx=37, ny=29), workloads.droplet_periodic(TC, RV, RL, n=97, radius=20.0)]
    cases = kinds * 24  # 24 x (1,024 + 8 + 52) tiles
    b, ids = _batch(prec, cases)
    assert b.kernel_names()[:2] == ["k_batch_walk"] * 2
    b.step(20)
    b.check()
    for k, kind in enumerate(kinds):
        one, (i,) = _batch(prec, [kind])
        assert one.kernel_names() == ["k_batch_tiles", "k_batch_advance"]
        one.step(20)
        want = one.fields(i)
        one.close()
        for j in (k, 36 + k, 69 + k):
            for got, w in zip(b.fields(ids[j]), want):
                assert np.array_equal(got, w), (kind[0]["name"], j)
    b.close()
