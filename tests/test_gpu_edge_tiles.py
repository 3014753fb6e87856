"""Edge tiles of the stored half: the passes that leave the padding columns out (z and y passes of
256 and 384 points, the step chain) against the oracle's FP64 transform and, bit for bit, against
steps that do not chain."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

# both passes with edge tiles, one of them, rows of one whole tile and of several; blocks along y
# that a tile's eight rows hold several of, one of, and half of
CASES = [
    ((256, 384, 64), (8, 8, 8)),
    ((384, 256, 64), (16, 2, 4)),
    ((256, 64, 64), (8, 16, 2)),
    ((64, 256, 128), (8, 4, 8)),
    ((128, 64, 128), (4, 16, 16)),
]


def _field(dims):
    return W.ch_initial_condition(dims, mean=0.05, seed=W.BASE_SEED).astype(np.float32)


@pytest.mark.parametrize("dims,block", CASES)
def test_transforms_match_oracle(dims, block):
    from paper_2609_03922_gb300 import spdba
    x = _field(dims)
    with spdba.Plan(dims, block, half_storage=1) as p:
        p.set_field(x)
        want = O.fftn(x.astype(np.complex128))[:, :, : dims[2] // 2 + 1]
        assert O.rel_l2(p.get_spectrum().reshape(want.shape), want) <= 2e-6
        assert O.rel_l2(p.get_field().reshape(dims), x) <= 4e-6


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("dims,block", CASES)
def test_one_call_equals_single_steps(dims, block, mode):
    from paper_2609_03922_gb300 import spdba
    x = _field(dims)
    outs = []
    for calls in ((12,), (1,) * 12):
        with spdba.Plan(dims, block, half_storage=1, threshold=0.6, reassess=5, mode=mode, dt=0.02) as p:
            p.set_field(x)
            for n in calls:
                p.step(n)
            outs.append((p.get_spectrum(), p.get_mask(), p.get_stats()["active_ratio_sum"], p.get_field()))
    a, b = outs
    assert np.array_equal(a[0].view(np.float32), b[0].view(np.float32))
    assert np.array_equal(a[1], b[1])
    assert a[2] == b[2]
    assert np.array_equal(a[3], b[3])


def test_many_block_rows():
    """2048 rows of blocks along y: the pencil liveness that prunes the forward passes. Fused steps use
    the x columns' part of it, staged ones also the z pencils'."""
    from paper_2609_03922_gb300 import spdba
    dims, block = (16, 2048, 64), (4, 1, 8)
    x = _field(dims)
    outs = []
    for fuse in (1, 0):
        with spdba.Plan(dims, block, half_storage=1, threshold=0.6, reassess=5, mode=1, dt=0.02, fuse_update=fuse) as p:
            p.set_field(x)
            p.step(8)
            outs.append((p.get_spectrum(), p.get_mask()))
    assert np.array_equal(outs[0][0].view(np.float32), outs[1][0].view(np.float32))
    assert np.array_equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("dims,block,kw", [((192, 64), (8, 16), {}), ((384, 128), (16, 8), {"force_dc": 0}),
                                           ((192, 16, 64), (8, 8, 8), {"half_spectrum": 0}),
                                           ((384, 64, 64), (16, 4, 8), {"half_storage": 1})])
def test_last_update_equals_staged(dims, block, kw, mode):
    """The fused update of a call's last step at 192 and 384 points (the chain's kernel without its
    inverse) against the staged update, bit for bit."""
    from paper_2609_03922_gb300 import spdba
    x = _field(dims)
    outs = []
    for fuse in (1, 0):
        with spdba.Plan(dims, block, threshold=0.6, reassess=3, mode=mode, dt=0.02, fuse_update=fuse, **kw) as p:
            p.set_field(x)
            for n in (1, 1, 3, 2):
                p.step(n)
            outs.append((p.get_spectrum(), p.get_mask(), p.get_stats()["active_ratio_sum"]))
    assert np.array_equal(outs[0][0].view(np.float32), outs[1][0].view(np.float32))
    assert np.array_equal(outs[0][1], outs[1][1])
    assert outs[0][2] == outs[1][2]
