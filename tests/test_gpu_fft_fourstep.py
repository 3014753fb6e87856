"""1-D transforms above 4096 points (n1 * 512) at every n1, in batches whose first pass takes the
narrow tiles and the wide ones, against the oracle's FP64 transform in either direction (forward
and back give the input also where both lack the twiddles between the passes)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

TOL = {0: 2e-6, 1: 1e-13}   # rel-L2, as for the other transforms: FP32 / FP64 arithmetic


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("batch", [1, 5, 64])
@pytest.mark.parametrize("n1", [16, 32, 64, 128, 192, 256, 384, 512])
def test_fourstep_matches_oracle(n1, batch, precision):
    import torch
    from paper_2609_03922_gb300 import spdba
    n = n1 * 512
    r = np.random.default_rng(n1 + batch)
    x = (r.standard_normal((batch, n)) + 1j * r.standard_normal((batch, n)))
    x = x.astype(np.complex64 if precision == 0 else np.complex128)
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    plan = spdba.FFTPlan((n,), batch=batch, precision=precision)
    for direction, ref in ((spdba.SPDBA_FORWARD, O.fftn), (spdba.SPDBA_INVERSE, O.ifftn)):
        plan.exec(xd, yd, direction)
        torch.cuda.synchronize()
        y = yd.cpu().numpy()
        for b in sorted({0, batch // 2, batch - 1}):
            assert O.rel_l2(y[b], ref(x[b].astype(np.complex128))) <= TOL[precision], (direction, b)
    plan.close()
