"""Sorts of 8-byte keys whose passes leave bytes out, against the oracle: keys
that agree above the passes' bytes in segments of 2 to 600 (both sides of what
one tile orders by itself, across tiles), in large crowds that a sample of the
keys cannot see (one value, and a few others next to it), constant bytes above
and in the middle, an odd number of passes in place, and batches of them."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs
from tests.test_gpu_parity import check_against_oracle

pytestmark = pytest.mark.gpu

N = 1_900_007                                             # above the sizes of a single launch


def wide_keys(kind, n, g):
    k = g.integers(0, 1 << 64, size=n, dtype=np.uint64)
    at = g.permutation(n)

    def crowd(lo, size, base, distinct):                  # `size` keys above `base`, of so many values
        k[at[lo:lo + size]] = np.uint64(base) + g.integers(0, distinct, size=size, dtype=np.uint64)
        return lo + size

    if kind == "segments":
        lo = 0
        for i, size in enumerate([2, 3, 31, 32, 33, 255, 256, 257, 300, 600]):
            lo = crowd(lo, size, (0x1111 * (i + 1)) << 44, 1 << 20)
    elif kind == "hot":                                   # half the keys 7 << 40, 200 keys next to it
        k[at[:n // 2]] = np.uint64(7 << 40)
        crowd(n // 2, 200, (7 << 40) - 50, 100)
    elif kind == "crowd":                                 # 40,000 keys of 3 values in one place, 5,000 in another
        lo = crowd(0, 40_000, 9 << 50, 3)
        crowd(lo, 5_000, 11 << 50, 1 << 30)
    elif kind == "narrow":                                # three bytes, and a fixed one between them
        k = (k & np.uint64(0xFF00FFFF00)) | np.uint64(0x5500000000000033)
    elif kind == "normal":
        k = inputs.normal_lognormal_u64(n, 5)
    elif kind == "exponential":
        k = (g.exponential(2.0 ** 40, size=n)).astype(np.uint64)
    elif kind == "sparse":                                # all alike but 300 keys, of two bytes and of all
        k = np.full(n, 5, np.uint64)
        k[at[:150]] += g.integers(0, 1 << 16, size=150, dtype=np.uint64)
        k[at[150:300]] = g.integers(0, 1 << 64, size=150, dtype=np.uint64)
    return k


KINDS = ["segments", "hot", "crowd", "narrow", "normal", "exponential", "uniform", "sparse"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("P", [40, 300])
def test_against_oracle(kind, P):
    g = np.random.default_rng(len(kind) + P)
    check_against_oracle(wide_keys(kind, N, g), inputs.index_payload(N), P, "u64")


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [50_000, 1_000_003])
def test_one_launch_form(kind, n):
    """The same keys where every pass runs in one launch (the hot values' segments
    are still shared by all CTAs of the clean-up)."""
    check_against_oracle(wide_keys(kind, n, np.random.default_rng(n)), inputs.index_payload(n), 24, "u64")


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("with_vals", [False, True])
def test_no_bounds_in_place(kind, with_vals):
    import torch
    from paper_1611_00463_gb300 import pgs
    g = np.random.default_rng(len(kind))
    keys, vals = wide_keys(kind, N, g), inputs.index_payload(N)
    want_k, want_v = O.stable_sort(keys, vals, "u64")
    dv = torch.from_numpy(vals.view(np.int32)).cuda() if with_vals else None
    cfg = pgs.make_config(dtype="u64", workspace=pgs.workspace(N, 40, pgs.make_config(dtype="u64")))
    for in_place in (False, True):
        dk = pgs.as_device_keys(keys, "u64")
        if in_place:
            ok, ov = dk, dv
            pgs.pgs_sort(dk, dv, 40, cfg)
        else:
            ok, ov = torch.empty_like(dk), None if dv is None else torch.empty_like(dv)
            pgs.pgs_sort_copy(dk, dv, ok, ov, 40, cfg)
        assert np.array_equal(pgs.to_numpy_keys(ok, "u64"), want_k)
        if with_vals:
            assert np.array_equal(ov.cpu().numpy().view(np.uint32), want_v)


@pytest.mark.parametrize("with_vals", [False, True])
def test_batch(with_vals):
    from tests.test_gpu_batched import check, run_batch
    g = np.random.default_rng(3)
    sizes = [6144 * 9 + 1, 1, 0, 6144, 300_000, 257, 12_288, 90_001, 6143, 500_009,      # above the batches left to merges
             200_000, 120_000, 100_003, 150_000, 99_000, 81_000, 260_001]
    assert sum(sizes) >= 3 << 19
    parts = [wide_keys(KINDS[i % len(KINDS)], n, g) if n > 80_000 else
             g.integers(0, 400, n).astype(np.uint64) << np.uint64(20) for i, n in enumerate(sizes)]
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    keys = np.concatenate(parts)
    vals = inputs.index_payload(len(keys)) if with_vals else None
    P = np.array([max(1, min(64, n // 500)) for n in sizes], dtype=np.uint32)
    got_k, got_v, _ = run_batch(offsets, keys, vals, P, "u64")
    check(offsets, keys, vals, got_k, got_v, [int(p) for p in P], "u64")


@pytest.mark.parametrize("dtype,tile", [("u64", 6144), ("u32", 7680)])
@pytest.mark.parametrize("tiles,delta,P", [(312, 0, 312), (312, 1, 312), (312, -1, 312), (312, 5, 311), (312, 5, 1000)])
def test_runs_as_long_as_a_tile_and_shorter(dtype, tile, tiles, delta, P):
    """A tile that is as long as a run, one key longer or shorter, and one that holds several."""
    n = tiles * tile + delta
    gen = inputs.uniform_u32 if dtype == "u32" else inputs.uniform_u64
    check_against_oracle(gen(n, P), inputs.index_payload(n), P, dtype)
