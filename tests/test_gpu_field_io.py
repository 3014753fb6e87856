"""set_field and get_field from host arrays, device tensors and device tensors off a 16-byte
boundary: the same spectrum bit for bit, and the field back."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

CH = [((64, 192), 0, 0), ((512, 64), 0, 0), ((128, 32), 1, 0), ((16, 16, 64), 0, 1), ((16, 32, 128), 0, 1),
      ((32, 16, 256), 0, 1), ((16, 64, 384), 0, 1), ((16, 16, 512), 0, 1), ((16, 32, 64), 0, 0), ((64, 16), 0, 0)]


def _check(make, x, tol):
    import torch
    shape = x.shape
    got = []
    for kind in ("host", "device", "offset"):
        with make() as p:
            if kind == "host":
                p.set_field(np.ascontiguousarray(x))
                out = p.get_field()
            else:
                k = 0 if kind == "device" else 1
                buf = torch.zeros(x.size + 1, dtype=torch.from_numpy(x).dtype, device="cuda")
                buf[k:k + x.size] = torch.from_numpy(x).cuda().reshape(-1)
                dst = torch.zeros_like(buf)
                torch.cuda.synchronize()
                p.set_field(buf[k:k + x.size])
                p.get_field(dst[k:k + x.size])
                out = dst[k:k + x.size].cpu().numpy().reshape(shape)
            got.append((p.get_spectrum(), out))
    for s, f in got[1:]:
        assert np.array_equal(s, got[0][0])
        assert np.array_equal(f, got[0][1])
    assert O.rel_l2(got[0][1], x) <= tol


@pytest.mark.parametrize("dims,precision,half", CH)
def test_real_fields(dims, precision, half):
    from paper_2609_03922_gb300 import spdba
    x = W.ch_initial_condition(dims, mean=0.1, seed=3).astype(np.float64 if precision else np.float32)
    _check(lambda: spdba.Plan(dims, (8,) * len(dims), precision=precision, half_storage=half), x,
           2e-13 if precision else 4e-6)   # forward and back: twice the transforms' tolerance


@pytest.mark.parametrize("dims,M", [((16, 64), 3), ((16, 16, 32), 2)])
def test_component_fields(dims, M):
    from paper_2609_03922_gb300 import spdba
    x = W.rcd_initial_condition(dims, M, 0.3, 0.1, seed=5).astype(np.float32)
    _check(lambda: spdba.Plan(dims, (4,) * len(dims), model=spdba.SPDBA_MODEL_RCD, components=M), x, 4e-6)


@pytest.mark.parametrize("n", [1024, 4096, 8192, 65536])
@pytest.mark.parametrize("precision", [0, 1])
def test_signals(n, precision):
    from paper_2609_03922_gb300 import spdba
    x = W.nls_signal(n, seed=7).astype(np.complex128 if precision else np.complex64)
    _check(lambda: spdba.Plan((n,), (n // 64,), model=spdba.SPDBA_MODEL_NLS, precision=precision), x,
           2e-13 if precision else 4e-6)
