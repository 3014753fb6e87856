"""Half-spectrum storage with an axis of 1024 or 2048 points along z or y (strided passes of those
lengths, the staged update where no fused one exists), in lock-step with the oracle's half form,
and the lengths that are refused."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from _helpers import states_within_tie_band

pytestmark = pytest.mark.gpu

B = (8, 8, 8)


@pytest.mark.parametrize("fuse", [1, 0])
@pytest.mark.parametrize("dims", [(1024, 16, 64), (2048, 16, 64), (16, 1024, 128), (16, 2048, 64), (1024, 64, 64),
                                  (192, 1024, 64)])
def test_long_axes_against_oracle(dims, fuse):
    from paper_2609_03922_gb300 import spdba
    c0 = W.ch_initial_condition(dims, mean=0.1, seed=W.BASE_SEED + 800).astype(np.float32)
    with spdba.Plan(dims, B, threshold=0.1, reassess=2, half_storage=1, fuse_update=fuse) as plan:
        plan.set_field(np.ascontiguousarray(c0))
        spec0, field0 = plan.get_spectrum(), plan.get_field()
        plan.step(1)
        masks = {0: plan.get_mask()}
        plan.step(2)
        masks[2] = plan.get_mask()
        field, spec = plan.get_field(), plan.get_spectrum()
    c0 = c0.astype(np.float64)
    # the tolerances of the half form's other lengths: transforms, there and back, and three steps
    assert O.rel_l2(spec0, O.rfftn_half(c0)) <= 2e-6
    assert O.rel_l2(field0, c0) <= 4e-6
    assert {0, 1, 2} <= set(np.unique(masks[2]).tolist())
    cfg = O.CHConfig(dims, B, threshold=0.1, reassess=2)
    checked = []

    def on_assess(n, h, st, tau):
        _, _, meas = O.assess_states_half(h, cfg, exclude_dc=True)
        checked.append(states_within_tie_band(masks[n], meas, tau, cfg, classifier=O.classify_half)[0])
        return masks[n]

    ref_h, _ = O.run_ch_half(c0, cfg, 3, on_assess=on_assess)
    assert checked == [True, True]
    assert O.rel_l2(field, O.ch_real_field_half(ref_h, dims)) <= 1e-5
    assert O.rel_l2(spec, ref_h) <= 1e-5


@pytest.mark.parametrize("dims", [(4096, 16, 64), (16, 4096, 64), (16, 16, 1024)])
def test_longer_axes_are_refused(dims):
    from paper_2609_03922_gb300 import spdba
    with pytest.raises(spdba.SpdbaError) as e:
        spdba.Plan(dims, B, half_storage=1)
    assert e.value.status == spdba.SPDBA_ERR_UNSUPPORTED
