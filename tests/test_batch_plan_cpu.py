"""Plans and workspaces on the host: sizes that no card holds do not end the process,
and the radix form's tables and workspace go to calls that may run it."""
import ctypes

import numpy as np
import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_1611_00463_gb300 import build, pgs
    build.build()
    return pgs.load()


def workspace_bytes(lib, offsets, dtype="u64", **opts):
    from paper_1611_00463_gb300 import pgs
    off = np.ascontiguousarray(np.asarray(offsets, dtype=np.uint64))
    cfg, h = pgs.make_config(dtype=dtype, **opts), ctypes.c_void_p()
    assert lib.pgs_batch_create(off.ctypes.data, len(off) - 1, None, 1, ctypes.byref(cfg), ctypes.byref(h)) == pgs.PGS_OK
    n = lib.pgs_batch_workspace_bytes(h)
    assert lib.pgs_batch_destroy(h) == pgs.PGS_OK
    return n


@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_more_keys_than_any_card_holds(lib, dtype):
    assert workspace_bytes(lib, [0, 1 << 42], dtype) > 1 << 42


@pytest.mark.parametrize("dtype,unit", [("u32", 7680), ("u64", 6144)])
def test_radix_tables_only_where_they_serve(lib, dtype, unit):
    full = np.arange(0, 401) * unit                       # whole tiles
    sparse = np.arange(0, 20_001) * (unit // 50)          # tiles one fiftieth full
    for opts in ({"merge_ways": 2}, {"exchange": "fused"}):
        assert workspace_bytes(lib, full, dtype, **opts) < workspace_bytes(lib, full, dtype)
    # (merge_ways 0 and 2 pass alike below 2^23 keys)
    assert workspace_bytes(lib, sparse, dtype) == workspace_bytes(lib, sparse, dtype, merge_ways=2)
    few = [0, unit, 2 * unit]                             # full tiles, too few keys
    assert workspace_bytes(lib, few, dtype) == workspace_bytes(lib, few, dtype, merge_ways=2)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_no_room_for_the_radix_form_where_merges_are_asked_for(lib, dtype):
    from paper_1611_00463_gb300 import pgs
    n, P = 5_000_000, 40

    def room(**opts):
        return pgs.pgs_workspace_bytes(n, P, pgs.make_config(dtype=dtype, **opts))
    assert room(investigator="local") == room(merge_ways=2, investigator="local") < room()
    assert room(exchange="fused") == room(merge_ways=2, exchange="fused") < room()
    assert room(tile_variant=2) == room(merge_ways=2, tile_variant=2) < room()
