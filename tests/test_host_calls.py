"""Host code of the library against a CUDA runtime that only writes calls down: the order of
copies on several streams, scratch after an allocation that failed, calls that failed half way."""
from tests._fake_cuda import run, unordered_copies

RING = """
import numpy as np
W = H = 64
r = hv.Renderer(W, H, 8, 16)
r.set_params(W, H, spatial="asp", T=8, stride=4, fs=20000.0, band=(1, 2))
g = hv.hv_group_open([r.h], use_graph=%(graph)s)
out = Dev((8, H, W), 4)
host = np.zeros((8, H, W), np.uint8)
log()
assert hv.hv_render_group(g, [Dev((12, H, W), 1)], [out]) == [2]
assert r.push(host, async_=True) == hv.HV_OK     # frames 12 .. 19, slots 12 .. 15, 0 .. 3
assert r.render(out) == 2
assert r.push(host, async_=True) == hv.HV_OK     # frames 20 .. 27: over the group's 8 .. 11
r.render(out)
print(json.dumps(log()))
"""


def test_pushes_follow_the_copy_of_a_groups_last_frames():
    """A group step of 12 frames copies the four that the next window reads again into slots 8
    .. 11 of the input ring, behind its images; a later push from the host overwrites the
    slots on the copy stream."""
    for graph in (False, True):
        assert unordered_copies(run(RING % dict(graph=graph))) == []
