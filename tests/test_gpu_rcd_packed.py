"""complex64 reaction-cross-diffusion steps, whose transforms carry two components per complex
field, against complex128 plans, whose transforms do not, from the same rounded start."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

# every row length with a packing kernel; odd and even component counts (the last one of an
# odd count stands alone); one and two tiles of row pairs and a ragged last one; blocks of
# unequal edges; thresholds that freeze most blocks (rows and planes drop out) and none
CASES = [((16, 32), (4, 4), 2), ((64, 64), (4, 8), 3), ((16, 128), (8, 4), 5), ((32, 256), (4, 4), 4),
         ((16, 16, 32), (4, 4, 4), 5), ((16, 32, 64), (4, 8, 4), 8), ((32, 16, 128), (8, 4, 4), 7),
         ((16, 16, 256), (4, 4, 8), 2)]


@pytest.mark.parametrize("threshold", [0.0, 1e-3, 0.3])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("dims,block,M", CASES)
def test_packed_steps_match_complex128(dims, block, M, mode, threshold):
    import torch
    from paper_2609_03922_gb300 import spdba
    u0 = W.rcd_initial_condition(dims, M, W.rcd_lv_homogeneous(M), 0.1, seed=W.BASE_SEED + M).astype(np.float32)
    outs = []
    with torch.cuda.stream(torch.cuda.Stream()):
        for precision, u in ((0, u0), (1, u0.astype(np.float64))):
            with spdba.Plan(dims, block, threshold=threshold, reassess=4, precision=precision, mode=mode,
                            model=spdba.SPDBA_MODEL_RCD, components=M, dx=0.5) as p:
                p.set_field(np.ascontiguousarray(u))
                p.step(10)
                outs.append((p.get_field(), p.get_mask()))
    assert np.array_equal(outs[0][1], outs[1][1])
    # the tolerance of the complex64 fields against the FP64 oracle over such runs
    assert O.rel_l2(outs[0][0], outs[1][0]) <= 1e-5
