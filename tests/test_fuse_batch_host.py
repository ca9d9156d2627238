"""Host side of the batched fusion: creation does no device work and holds no device memory."""
import ctypes
import os
import re

import pytest

FAKE = 0x10000  # a 256-byte aligned stand-in address; never dereferenced here


@pytest.fixture(scope="module")
def lib():
    from paper_2505_18932_gb300 import build as b
    b.build()
    from paper_2505_18932_gb300 import gvs
    return gvs.load()


@pytest.mark.parametrize("n_items", [1, 14, 15, 1024])
def test_batch_table(lib, n_items):
    """The table is a formality of one aligned block, refused as ever when missing, short or misaligned."""
    from paper_2505_18932_gb300 import gvs
    from synth import camera_at
    cam = gvs.camera_struct(camera_at(64, 48, (0.0, 0.0, 0.0)))
    cams = (gvs.GvsCamera * 2)(cam, cam)
    item = gvs.GvsFuseItem(FAKE, lib.gvs_fuse_workspace_bytes(2, 64, 48), ctypes.pointer(cam), FAKE, None)
    items = (gvs.GvsFuseItem * n_items)(*[item] * n_items)
    p = gvs.GvsFuseParams(64, 0.5, 5.0, 0.05, 0.001, 7, 0, 0, 0, 0)
    size = lib.gvs_fuse_batch_bytes(n_items)
    assert size == 256 and lib.gvs_fuse_batch_bytes(-1) == 0

    def create(n=n_items, table=FAKE, table_bytes=size):
        h = ctypes.c_void_p()
        st = lib.gvs_fuse_batch_create(cams, 2, items, n, ctypes.byref(p), table, table_bytes, ctypes.byref(h))
        assert (st == 0) == bool(h)
        lib.gvs_fuse_batch_destroy(h)
        return st

    assert create() == 0
    assert create(table=None) == 3
    assert create(table_bytes=size - 1) == 3
    assert create(table=FAKE + 16) == 3
    assert create(n=0) == 1
    assert create(n=1025) == 1


def test_items_of_a_launch():
    """The binding counts launches with the library's own number of items."""
    from paper_2505_18932_gb300 import gvs
    h = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "gvs.h")).read()
    n = int(re.search(r"#define GVS_BATCH_LAUNCH_ITEMS (\d+)", h).group(1))
    assert gvs.FUSE_BATCH_ITEMS == n
