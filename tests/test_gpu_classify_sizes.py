"""Classification of maps on either side of the size where its CTAs grow from 256 to 1024 blocks
(ragged last CTAs among them): states, the list of non-frozen blocks and their count against the
oracle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("share", [0.002, 0.3])
@pytest.mark.parametrize("nblocks", [(1024, 2048), (1024, 2049), (129, 129, 129)])
def test_large_maps_match_oracle(nblocks, share):
    import torch
    from paper_2609_03922_gb300 import spdba
    nb = int(np.prod(nblocks))
    m = np.random.default_rng(nb).random(nblocks)
    dev = lambda dt, n: torch.empty(n, dtype=dt, device="cuda")
    states, chi, lst, cnt = dev(torch.uint8, nb), dev(torch.uint8, nb), dev(torch.int32, nb), dev(torch.int32, 1)
    scratch = dev(torch.uint8, spdba.classify_scratch_bytes(nb))
    tau = torch.tensor([1.0 - share], dtype=torch.float64, device="cuda")
    spdba.classify(nblocks, torch.from_numpy(m).cuda(), tau, 0, 1, states, chi, lst, cnt, scratch)
    torch.cuda.synchronize()
    want = O.classify(m, 1.0 - share, force_dc=False, transitions=True).reshape(-1)
    assert np.array_equal(states.cpu().numpy(), want)
    live = np.flatnonzero(want)
    assert int(cnt.item()) == live.size
    assert np.array_equal(lst[:live.size].cpu().numpy(), live)
