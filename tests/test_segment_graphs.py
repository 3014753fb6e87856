"""How many graphs a plan captures for its segments: one where the launches are the same whatever
comes before and after a segment, and one per kind of neighbour where steps chain."""
import pytest

import _fake_device

# steps of 3 segments; (dims, block, options), graphs: Cahn-Hilliard steps chain (first, middle and last
# segment differ), the multi-size form, NLS and reaction-cross-diffusion do not
CASES = [(dict(dims=(64, 64), block=(8, 8)), 3), (dict(dims=(64, 64), block=(8, 8), fuse_update=0), 1),
         (dict(dims=None, block=(8, 8), batch_dims=[(64, 64), (128, 128)], multi_pass=1), 1),
         (dict(dims=(1024,), block=(16,), model=1), 1), (dict(dims=(16, 64), block=(4, 4), model=2, components=3), 1)]

SNIPPET = """
kw = %r
with spdba.Plan(kw.pop("dims"), kw.pop("block"), reassess=5, stream=64, **kw) as p:
    if kw.get("multi_pass"):
        assert p.get_config()["multi_pass"] == 1
    for _ in range(2):
        p.step(15)
print(fake.fake_instantiated())
"""


@pytest.mark.parametrize("kw,graphs", CASES)
def test_graphs_of_three_segments(tmp_path, kw, graphs):
    assert int(_fake_device.run(tmp_path, SNIPPET % (kw,))) == graphs
