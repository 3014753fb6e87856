"""set_field and get_field with memory of another GPU than the plan's: it is copied, as between any
two devices, and no kernel of the plan's device takes it."""
import pytest

import _fake_device

# (dims, block, options, bytes per value): Cahn-Hilliard in each storage form and precision, with and
# without kernels for real rows, NLS of short and long signals, reaction-cross-diffusion
CASES = [((64, 64), (8, 8), {}, 4), ((64, 64), (8, 8), {"precision": 1}, 8), ((16, 32, 64), (4, 8, 8), {"half_storage": 1}, 4),
         ((1024,), (16,), {"model": 1}, 8), ((65536,), (1024,), {"model": 1}, 8), ((8192,), (128,), {"model": 1, "precision": 1}, 16),
         ((16, 64), (4, 4), {"model": 2, "components": 3}, 4)]

SNIPPET = """
dims, block, kw, size = %r
n = int(np.prod(dims)) * kw.get("components", 1) * size
own, other = (np.zeros(n + 256, dtype=np.uint8) for _ in range(2))
fake.fake_foreign(ctypes.c_void_p(other.ctypes.data), ctypes.c_size_t(other.size))
with spdba.Plan(dims, block, stream=64, **kw) as p:
    for buf, copies in ((own, 0), (other, 2)):
        at = (buf.ctypes.data + 255) // 256 * 256
        assert L.spdba_set_field(p._p, 0, at, 1) == 0
        assert L.spdba_get_field(p._p, 0, at, 1) == 0
        assert fake.fake_foreign_launches() == 0, "a kernel took the other GPU's pointer"
        assert fake.fake_foreign_copies() == copies
"""


@pytest.mark.parametrize("case", CASES)
def test_other_gpus_memory_is_copied(tmp_path, case):
    _fake_device.run(tmp_path, SNIPPET % (case,))
