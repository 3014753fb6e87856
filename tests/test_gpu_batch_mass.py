"""The mass statistic of each run of a large batch of small fields, whose rows a wide tile of the
nonlinear pass would span several fields of."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,runs,precision", [((16, 64), 1300, 1), ((16, 32), 2600, 1), ((16, 16), 5200, 1),
                                                 ((16, 64), 160, 0), ((16, 16), 200, 0)])
def test_mass_of_each_run(dims, runs, precision):
    from paper_2609_03922_gb300 import spdba
    dt = np.float64 if precision else np.float32
    x = W.ch_initial_condition(dims, mean=0.0, seed=W.BASE_SEED)
    with spdba.Plan(None, (8, 8), batch_dims=[dims] * runs, precision=precision, reassess=5) as p:
        fields = [np.ascontiguousarray((x + 0.01 * (r % 97)).astype(dt)) for r in range(runs)]
        for r, f in enumerate(fields):
            p.set_field(f, run=r)
        p.step(1)
        # the field at step 0 is the transform's round trip of c0, to the transforms' tolerance a value
        tol = (2e-13 if precision else 4e-6) * x.size
        for r, f in enumerate(fields):
            assert abs(p.get_stats(run=r)["mass"] - f.astype(np.float64).sum()) <= tol, r
