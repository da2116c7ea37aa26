"""The indexed search's choice of where to look, against the oracle, on key
spacings that mislead interpolation: long runs of one value, gaps that grow
geometrically inside a block, all keys equal, the key type's extremes; ragged
last lines, blocks and table cells; keys off the 16-byte boundary."""
import numpy as np
import pytest

from oracle import pgs_oracle as O

pytestmark = pytest.mark.gpu


def spaced(kind, n, dtype, g):
    w = 64 if dtype == "u64" else 32
    top = (1 << w) - 1
    i = np.arange(n, dtype=np.uint64)
    if kind == "smooth":
        k = g.integers(0, top, size=n, dtype=np.uint64, endpoint=True)
    elif kind == "runs":                                  # runs of 1 to 3000 equal keys, far apart
        k = np.repeat(g.integers(0, top, size=n, dtype=np.uint64, endpoint=True), g.integers(1, 3000, size=n) ** 2 // 3000 + 1)[:n]
    elif kind == "steep":                                 # doubling gaps inside groups of w - 20 keys
        k = np.uint64(1) << (i % np.uint64(w - 20))
        k = k + (i // np.uint64(w - 20) << np.uint64(w - 20)) if dtype == "u64" else k
    elif kind == "equal":
        k = np.full(n, 12345, np.uint64)
    else:                                                 # the type's ends and little between
        k = np.where(i < n // 2, np.uint64(0), np.uint64(top))
        k[n // 2 - 3:n // 2 + 3] = g.integers(0, top, size=6, dtype=np.uint64)
    return np.sort(k.astype(np.uint64 if dtype == "u64" else np.uint32))


@pytest.mark.parametrize("kind", ["smooth", "runs", "steep", "equal", "ends"])
@pytest.mark.parametrize("dtype,n,shift", [("u64", 65536, 0), ("u64", 65537, 1), ("u64", 1_000_063, 0),
                                           ("u32", 65536 + 63, 0), ("u32", 262_145, 3), ("u32", 700_001, 0)])
def test_misleading_spacings(kind, dtype, n, shift):
    import torch
    from paper_1611_00463_gb300 import pgs
    g = np.random.default_rng(n + shift)
    keys = spaced(kind, n, dtype, g)
    near = keys[g.integers(0, n, size=70_000)]
    ext = np.array([0, 1, np.iinfo(keys.dtype).max - 1, np.iinfo(keys.dtype).max], keys.dtype)
    q = np.concatenate([near, near + keys.dtype.type(1), near - keys.dtype.type(1), keys[-70:], keys[:70], ext])
    q = np.concatenate([q, np.sort(q)])                   # neighbours in a warp apart, then together
    assert len(q) >= 3 << 17                              # fewer queries bisect the array itself
    dk = torch.empty(n + shift, dtype=pgs.KEY_TORCH[dtype], device="cuda")[shift:]
    dk.copy_(pgs.as_device_keys(keys, dtype))
    dq = pgs.as_device_keys(q, dtype)
    ws = torch.empty(pgs.pgs_search_workspace_bytes(n, dtype), dtype=torch.uint8, device="cuda")
    for side in ("left", "right"):
        pos = torch.empty(len(q), dtype=torch.int64, device="cuda")
        pgs.pgs_search(dk, dq, pos, side=side, dtype=dtype, workspace=ws)
        torch.cuda.synchronize()
        assert np.array_equal(pos.cpu().numpy(), O.search(keys, q, dtype, side))
