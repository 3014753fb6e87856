"""The step chain (update and the next step's first inverse pass in one kernel): n steps in
one call, which chain, against n calls of one step, which do not, bit for bit."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# tiles at every pass length that has a chain kernel, single and several rows of a small grid,
# tiles with frozen blocks (large thresholds), both precisions, batches, the stored half
CASES = [
    (((64, 64),), (16, 16), 1, {}),
    (((128, 192),), (16, 16), 1, {}),
    (((192, 64), (128, 128), (192, 64)), (8, 16), 0, {}),
    (((384, 128),), (16, 8), 0, {}),
    (((512, 256),), (16, 16), 0, {"measure": 1}),
    (((256, 16, 32),), (8, 8, 8), 0, {"half_spectrum": 0}),
    (((32, 32, 64),), (8, 8, 8), 1, {}),
    (((64, 64, 64),), (8, 8, 8), 0, {"half_storage": 1}),
    (((192, 64, 128),), (8, 4, 8), 0, {"half_storage": 1, "refresh_every": 7}),
    (((16, 64, 128),), (4, 8, 8), 0, {"half_storage": 1, "transitions": 0}),
]


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_one_call_equals_single_steps(case, mode, graph):
    import torch
    from paper_2609_03922_gb300 import spdba
    runs, block, precision, kw = CASES[case]
    dt = np.float64 if precision else np.float32
    x = [W.ch_initial_condition(d, mean=0.05, seed=W.BASE_SEED + i).astype(dt) for i, d in enumerate(runs)]
    outs = []
    with torch.cuda.stream(torch.cuda.Stream()):
        for calls in ((23,), (1,) * 23, (4, 10, 9)):
            # the threshold freezes part of the blocks of the noise's spectrum
            with spdba.Plan(None, block, threshold=0.6, reassess=5, batch_dims=list(runs), precision=precision,
                            mode=mode, use_graph=graph, dt=0.02, **kw) as p:
                for r, f in enumerate(x):
                    p.set_field(np.ascontiguousarray(f), run=r)
                for n in calls:
                    p.step(n)
                outs.append([(p.get_spectrum(run=r), p.get_mask(run=r), p.get_stats(run=r)["active_ratio_sum"])
                             for r in range(len(runs))])
    for got in outs[1:]:
        for (a, ma, ra), (b, mb, rb) in zip(outs[0], got):
            assert np.array_equal(a.view(dt), b.view(dt))
            assert np.array_equal(ma, mb)
            assert ra == rb
