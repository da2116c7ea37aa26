"""The indexed search against the oracle where its warps are ragged or split:
query counts that leave part of a warp, warps whose lanes differ in whether the
interpolated looks can serve them."""
import numpy as np
import pytest

from oracle import pgs_oracle as O

pytestmark = pytest.mark.gpu

INDEX_QUERIES = 3 << 17                                   # fewer queries bisect the array itself


def sorted_keys(n, dtype, seed):
    """Smooth keys, with runs of equal ones in the last third."""
    g = np.random.default_rng(seed)
    k = g.integers(0, 1 << (64 if dtype == "u64" else 32), size=n, dtype=np.uint64)
    k[2 * n // 3:] = k[g.integers(2 * n // 3, 2 * n // 3 + 40, size=n - 2 * n // 3)]
    return np.sort(k.astype(np.uint64 if dtype == "u64" else np.uint32))


def run(keys, q, dtype, side, e=None):
    import torch
    from paper_1611_00463_gb300 import pgs
    ws = torch.empty(pgs.pgs_search_workspace_bytes(len(keys), dtype), dtype=torch.uint8, device="cuda")
    pos = torch.full((len(q) + 64,), -1, dtype=torch.int64, device="cuda")      # nothing written past the last query
    bkt = None if e is None else torch.full((len(q) + 64,), -1, dtype=torch.int32, device="cuda")
    pgs.pgs_search(pgs.as_device_keys(keys, dtype), pgs.as_device_keys(q, dtype), pos[:len(q)], side=side, dtype=dtype,
                   workspace=ws, bucket_bounds=None if e is None else torch.from_numpy(e).cuda(),
                   bucket_out=None if e is None else bkt[:len(q)])
    torch.cuda.synchronize()
    assert (pos[len(q):] == -1).all() and (bkt is None or (bkt[len(q):] == -1).all())
    return pos[:len(q)].cpu().numpy(), None if e is None else bkt[:len(q)].cpu().numpy()


@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("more", [0, 1, 31, 33, 255, 257])
def test_ragged_query_counts_and_split_warps(dtype, more):
    n, m = 100_003, INDEX_QUERIES + more
    keys = sorted_keys(n, dtype, more)
    g = np.random.default_rng(more + 1)
    q = keys[g.integers(0, n, size=m)]
    q[::3] += keys.dtype.type(1)                          # hits and misses, runs and smooth keys in every warp
    q[::97] = np.iinfo(keys.dtype).max
    q[1::97] = 0
    for side in ("left", "right"):
        assert np.array_equal(run(keys, q, dtype, side)[0], O.search(keys, q, dtype, side))


@pytest.mark.parametrize("dtype,n", [("u64", 1 << 20), ("u64", (1 << 20) + 1), ("u32", 1 << 21), ("u32", (1 << 21) + 1)])
@pytest.mark.parametrize("kind", ["smooth", "third", "all"])
def test_by_steps_or_with_looks(dtype, n, kind):
    """Both sides of the size up to which the search only bisects (8 MB), and keys of
    which none, a third and all repeat (a quarter is where a CTA gives the looks up)."""
    keys = sorted_keys(n, dtype, n)
    g = np.random.default_rng(n + 1)
    if kind == "smooth":
        keys = np.sort(g.integers(0, np.iinfo(keys.dtype).max, size=n, dtype=keys.dtype, endpoint=True))
    elif kind == "all":
        keys = np.sort(keys[g.integers(0, 700, size=n)])
    q = np.concatenate([keys[g.integers(0, n, size=INDEX_QUERIES // 2)],
                        g.integers(0, np.iinfo(keys.dtype).max, size=INDEX_QUERIES // 2 + 5, dtype=keys.dtype)])
    g.shuffle(q)
    for side in ("left", "right"):
        assert np.array_equal(run(keys, q, dtype, side)[0], O.search(keys, q, dtype, side))


@pytest.mark.parametrize("dtype,n,P", [("u32", 300_001, 1), ("u64", 200_003, 128), ("f32", 250_000, 1023), ("u32", 400_009, 1024),
                                       ("u64", 3_000_017, 1023), ("u64", 3_000_017, 1024), ("u32", 6_000_011, 3000),
                                       ("u64", (1 << 24) + 5, 64)])
def test_buckets_through_the_index(dtype, n, P):
    """Buckets looked up in shared memory (P < 1024) and outside it; from 2^24 keys the
    index is used for half as many queries."""
    m = INDEX_QUERIES // 2 if n >= 1 << 24 else INDEX_QUERIES
    keys = sorted_keys(n, "u32" if dtype == "f32" else dtype, P)
    if dtype == "f32":                                    # order form to float bits
        keys = np.where(keys >> np.uint32(31) == 1, keys & np.uint32(0x7FFFFFFF), ~keys).astype(np.uint32)
    g = np.random.default_rng(P)
    q = keys[g.integers(0, n, size=m)]
    q[::2] = g.integers(0, np.iinfo(keys.dtype).max, size=(m + 1) // 2, dtype=keys.dtype)
    e = np.sort(np.concatenate([[0, n], g.integers(0, n + 1, size=P - 1)])).astype(np.int64)    # some buckets empty
    for side in ("left", "right"):
        pos, bkt = run(keys, q, dtype, side, e)
        want = O.search(keys, q, dtype, side)
        assert np.array_equal(pos, want)
        assert np.array_equal(bkt, O.bucket_of(want, e))
