"""Transform passes at every length, with pencil counts that take the wide tiles, the narrow
ones and the kernel for any count, against the oracle's FP64 FFT."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

TOL = {0: 2e-6, 1: 1e-13}   # rel-L2, as for the other transforms: FP32 / FP64 arithmetic
LENGTHS = [16, 32, 64, 128, 192, 256, 384, 512]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("length", LENGTHS)
# (second axis, batch): few and many strided pencils; rows in counts that no tile, a narrow
# tile and a wide tile divides (second axis 0: a 1-D batch)
@pytest.mark.parametrize("other,batch", [(16, 1), (64, 41), (0, 3), (0, 8), (0, 2560)])
def test_pass_matches_oracle(length, other, batch, precision):
    import torch
    from paper_2609_03922_gb300 import spdba
    shape = (length, other) if other else (length,)
    r = np.random.default_rng(length + 7 * other + batch)
    x = (r.standard_normal((batch,) + shape) + 1j * r.standard_normal((batch,) + shape))
    x = x.astype(np.complex64 if precision == 0 else np.complex128)
    xd = torch.from_numpy(x).cuda()
    plan = spdba.FFTPlan(shape, batch=batch, precision=precision)
    yd, zd = torch.empty_like(xd), torch.empty_like(xd)
    plan.exec(xd, yd, spdba.SPDBA_FORWARD)
    plan.exec(yd, zd, spdba.SPDBA_INVERSE)
    torch.cuda.synchronize()
    y, z = yd.cpu().numpy(), zd.cpu().numpy()
    for b in sorted({0, batch // 2, batch - 1}):
        assert O.rel_l2(y[b], O.fftn(x[b].astype(np.complex128))) <= TOL[precision], b
    assert O.rel_l2(z, x) <= 2 * TOL[precision]
    plan.close()
