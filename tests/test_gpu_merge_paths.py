"""Parity with the oracle on both sides of the merge pipeline's small-sort limits,
with the merge width asked for (sorts that ask for none run the radix form): cut
searches and bucket offsets at 4096 (run, splitter) slots, sample rounds worked
out by their merge CTAs, every merge tile shape."""
import pytest

from paper_1611_00463_gb300 import inputs
from tests.test_gpu_parity import check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ways", [2, 4])
@pytest.mark.parametrize("P", [64, 65])
@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_cut_search_and_offsets_either_side_of_4096_slots(P, dtype, ways):
    n = 90_001
    gen = {"u32": inputs.exponential_u32, "u64": inputs.normal_lognormal_u64}[dtype]
    check_against_oracle(gen(n, P), inputs.index_payload(n), P, dtype, merge_ways=ways)


@pytest.mark.parametrize("ways", [2, 4])
@pytest.mark.parametrize("P", [5, 16, 100])
def test_inline_sample_rounds_with_ragged_runs(P, ways):
    for n, s in [(P * 1000 + P - 1, None), (P * 37 + 3, 64), (P * 37 + 3, 37), (P * 37 + 3, 38)]:
        check_against_oracle(inputs.uniform_u32(n, n), inputs.index_payload(n), P, "u32", s=s, merge_ways=ways)


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_every_tile_shape(dtype, variant):
    n = 250_003
    gen = {"u32": inputs.exponential_u32, "u64": inputs.normal_lognormal_u64}[dtype]
    check_against_oracle(gen(n, variant), inputs.index_payload(n), 16, dtype, tile_variant=variant, merge_ways=2)
