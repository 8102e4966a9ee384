"""Which destinations the mesh copy stores to with its own kernel: device memory of
the context's GPU, with that GPU current, on a 4-byte boundary and inside its
allocation.  Everything else stays with the driver's copy, as host buffers do
(host arithmetic: no GPU, no launch)."""

import pytest

UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3          # cudaMemoryType


@pytest.fixture(scope="module")
def lib():
    from paper_1712_03084_gb300 import build, ftr
    build.build()
    return ftr.load()


@pytest.mark.parametrize("kw,want", [
    ({}, 1),
    (dict(room=120, size=120), 1),
    (dict(room=119, size=120), 0),                        # past the end of its allocation
    (dict(room=0), 0),                                    # extent not known
    (dict(address=0x7f0000000004), 1),
    (dict(address=0x7f0000000001), 0),
    (dict(address=0x7f0000000002), 0),
    (dict(device=1), 0),                                  # another GPU's memory
    (dict(current=1), 0),                                 # another GPU current: no launch on this stream
    (dict(ctx=1, device=1, current=1), 1),
    (dict(ctx=1, device=0, current=1), 0),
    (dict(type=MANAGED), 0),
    (dict(type=HOST), 0),
    (dict(type=UNREGISTERED), 0),
])
def test_route(lib, kw, want):
    d = dict(type=DEVICE, device=0, ctx=0, current=0, address=0x7f0000000000, room=1 << 20, size=1200)
    d.update(kw)
    assert lib.ftr_debug_mesh_copy_route(d["type"], d["device"], d["ctx"], d["current"], d["address"], d["room"],
                                         d["size"]) == want
