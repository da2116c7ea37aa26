"""The clean-up of wide keys against the oracle: long segments whose keys differ in
one, two or three bytes that lie next to one another or apart (an odd number of
moves is copied back), taken by one CTA or by all, with and without payloads and
run tags; and nearly sorted keys, whose mates lie close together in the input."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs
from tests.test_gpu_parity import check_against_oracle

pytestmark = pytest.mark.gpu


def near_hot(n, size, differ, g):
    """n random keys, `size` of them one value but for 20 that differ from it in the
    bits of `differ` (so few that a sample of the keys does not tell)."""
    k = g.integers(0, 1 << 64, size=n, dtype=np.uint64)
    at = g.permutation(n)[:size]
    k[at] = np.uint64(0x5A << 40)
    k[at[:20]] |= g.integers(0, 1 << 40, size=20, dtype=np.uint64) & np.uint64(differ)
    return k


@pytest.mark.parametrize("differ", [0xFF, 0xFF00FF, 0xFFFF00, 0xFFFFFF00, 0xFFFFFFFF])
@pytest.mark.parametrize("n,size", [(300_007, 3_000), (300_007, 150_000), (2_500_003, 9_000), (2_500_003, 1_200_000)])
def test_bytes_left_out(n, size, differ):
    g = np.random.default_rng(n + size)
    keys = near_hot(n, size, differ, g)
    check_against_oracle(keys, inputs.index_payload(n), 30, "u64")
    check_against_oracle(keys, None, 30, "u64")


@pytest.mark.parametrize("n", [100_003, 2_500_003])
def test_no_runs_and_many_segments(n):
    """No tags (P = 1 and no bounds), and twenty hot values, each with neighbours."""
    from tests.gpu_helpers import gpu_sort
    g = np.random.default_rng(n)
    keys = g.integers(0, 1 << 64, size=n, dtype=np.uint64)
    at = g.permutation(n)
    for h in range(20):
        part = at[h * (n // 50):(h + 1) * (n // 50)]
        keys[part] = np.uint64((h + 3) << 44)
        keys[part[:5]] += g.integers(0, 1 << (8 * (h % 4) + 1), size=5, dtype=np.uint64)
    vals = inputs.index_payload(n)
    want_k, want_v = O.stable_sort(keys, vals, "u64")
    got = gpu_sort(keys, vals, 1, "u64")
    assert np.array_equal(got["keys"], want_k) and np.array_equal(got["vals"], want_v)
    check_against_oracle(keys, vals, 24, "u64")


@pytest.mark.parametrize("n", [100_003, 1_000_003, 4_000_037])
@pytest.mark.parametrize("noise", [1, 1 << 8, 1 << 16, 1 << 24])
def test_nearly_sorted(n, noise):
    g = np.random.default_rng(noise)
    keys = np.uint64(1_700_000_000_000_000_000) + np.arange(n, dtype=np.uint64) * np.uint64(1000) + \
        g.integers(0, noise, size=n, dtype=np.uint64)
    check_against_oracle(keys, inputs.index_payload(n), 20, "u64")
