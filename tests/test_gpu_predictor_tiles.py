"""The predictor's voxel-tile kernels on maps that their 4 x 4 x 16 tiles do not divide,
against the CPU reference (FP64 with the same BF16 rounding points)."""
import numpy as np
import pytest

from oracle import predictor_ref as R
from test_gpu_predictor import _data, _flat, _to_dev, _unflat

pytestmark = pytest.mark.gpu


# edges of one voxel past a tile, of the smallest map, and of several maps with a ragged last tile
@pytest.mark.parametrize("shape,nmaps", [((3, 3, 3), 1), ((4, 4, 16), 2), ((5, 5, 17), 2), ((3, 9, 33), 3),
                                         ((13, 7, 15), 1)])
def test_ragged_maps_match_reference(shape, nmaps):
    import torch
    from paper_2609_03922_gb300 import spdba
    P = R.init_params(11)
    for k in ("b1", "b2", "b3"):
        P[k] = P[k] + 0.05
    params = _flat(P).astype(np.float32)
    pr = spdba.Predictor(shape, max_batch=nmaps, params=params)
    x, y = _data(shape, nmaps, 12)
    xd, yd = _to_dev(x, y)
    prob = torch.empty((nmaps,) + shape, dtype=torch.float32, device="cuda")
    pr.forward(xd, prob, nmaps=nmaps)
    torch.cuda.synchronize()
    ref, _ = R.forward(_unflat(params), x, round_bf16=True)
    assert np.max(np.abs(prob.cpu().numpy() - ref)) <= 2e-3
    loss, g = pr.gradients(xd, yd, nmaps=nmaps)
    ref_loss, G = R.backward(_unflat(params), x, y, round_bf16=True)
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    Gg = _unflat(g)
    for k in G:
        assert np.linalg.norm(Gg[k] - G[k]) <= 1e-2 * np.linalg.norm(G[k]) + 1e-9, k
    pr.close()
