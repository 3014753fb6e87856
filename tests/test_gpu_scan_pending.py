"""The activity scan's pending candidate: modes that rise through a block by steps around the
screen's error (so that each new one replaces the pending one, or ties with it), in both scan
kernels and both CTA sizes of the rows kernel, bit for bit with the FP64 maxima."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [2.0 ** -24, 2.0 ** -20, 2.0 ** -18, 2.0 ** -16])
# rows kernel with 128 and with 256 threads, warp-per-block kernel
@pytest.mark.parametrize("shape,block", [((128, 128, 64), (4, 4, 4)), ((160, 256, 256), (8, 8, 8)),
                                         ((32, 32, 32), (8, 8, 8))])
def test_rising_modes(shape, block, step):
    import torch
    from paper_2609_03922_gb300 import spdba
    r = np.random.default_rng(17)
    nb = tuple(s // b for s, b in zip(shape, block))
    # |q| rises along each block's modes, in storage order of its rows, at random phases
    rank = np.arange(int(np.prod(block))).reshape(block)
    mag = np.tile(1.0 + step * rank, nb) * np.exp2(r.integers(-40, 40, size=nb)).repeat(block[0], 0).repeat(
        block[1], 1).repeat(block[2], 2)
    q = (mag * np.exp(2j * np.pi * r.random(shape))).astype(np.complex64)
    maxsq = torch.empty(nb, dtype=torch.float64, device="cuda")
    gmax = torch.zeros(2, dtype=torch.float64, device="cuda")
    spdba.block_activity(torch.from_numpy(q).cuda(), block, maxsq, None, gmax, precision=0)
    torch.cuda.synchronize()
    q64 = q.astype(np.complex128)
    mx, _ = O.block_measures(q64, block)
    assert np.array_equal(maxsq.cpu().numpy(), mx)
    assert gmax.cpu().numpy()[0] == O.global_max_sq(q64, exclude_dc=False)
