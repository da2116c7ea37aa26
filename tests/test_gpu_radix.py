"""The radix form of the sort against the oracle, bit for bit (keys, payloads,
bucket bounds, cut matrix, splitters): one key below, at and above whole tiles
and whole counting chunks, both run widths a tag holds (P = 256 and 257), keys
that differ in one byte or not at all, every investigator, unaligned buffers,
sorts that ask for no bounds, and the merge pipeline's results for the same
calls.  Sorts with more than 64 partitions take this form at every size."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs
from tests.test_gpu_parity import check_against_oracle

pytestmark = pytest.mark.gpu

TILE = {"u32": 384 * 20, "f32": 384 * 20, "u64": 384 * 16}      # keys per tile of a pass
GEN = {"u32": inputs.uniform_u32, "u64": inputs.normal_lognormal_u64, "f32": inputs.zipf_dup_f32}


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
@pytest.mark.parametrize("tiles,delta", [(0, 70), (1, -1), (1, 0), (1, 1), (2, 5), (40, -3), (40, 0), (40, 1)])
def test_whole_and_ragged_tiles(dtype, tiles, delta):
    n = tiles * TILE[dtype] + delta
    check_against_oracle(GEN[dtype](n, n), inputs.index_payload(n), 65, dtype)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("P", [255, 256, 257, 1000])
def test_runs_either_side_of_one_byte(dtype, P):
    n = 3 * TILE[dtype] + 1001
    for variant in (0, 1, 2):
        check_against_oracle(GEN[dtype](n, P), inputs.index_payload(n), P, dtype, variant=variant)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_more_than_one_tile_per_counting_chunk(dtype):
    n = 2500 * TILE[dtype] + 17                       # above 1216 tiles a chunk holds several
    check_against_oracle(GEN[dtype](n, 3), inputs.index_payload(n), 7, dtype)


@pytest.mark.parametrize("dtype,byte", [("u32", b) for b in range(4)] + [("u64", b) for b in range(8)])
def test_keys_that_differ_in_one_byte(dtype, byte):
    n = 2 * TILE[dtype] + 33
    rng = np.random.default_rng(byte)
    kt = np.uint64 if dtype == "u64" else np.uint32
    keys = (rng.integers(0, 256, n).astype(kt) << kt(8 * byte)) | kt(0x5A5A5A5A) & ~(kt(0xFF) << kt(8 * byte))
    check_against_oracle(keys, inputs.index_payload(n), 66, dtype)
    check_against_oracle(np.full(n, keys[0]), inputs.index_payload(n), 66, dtype)


@pytest.mark.parametrize("kind", ["sorted", "reverse", "few", "extremes"])
@pytest.mark.parametrize("guaranteed", [False, True])
def test_structured_keys_and_guaranteed_samples(kind, guaranteed):
    n, P = 5 * TILE["u32"] + 91, 70
    keys = inputs.structured_u32(kind, n)
    s = max(O.paper_samples_per_run(P, 4), O.guaranteed_samples_per_run(P, 0.05)) if guaranteed else None
    check_against_oracle(keys, inputs.index_payload(n), P, "u32", s=s)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("with_vals", [False, True])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_unaligned_buffers_and_no_bounds(dtype, with_vals, offset):
    """Buffers that start 1 or 3 elements past an aligned address, a call that
    asks for no bounds (nothing depends on the runs), then the same with them;
    out of place, then in place."""
    import torch
    from paper_1611_00463_gb300 import pgs
    n, P = 4 * TILE[dtype] + 7, 100
    keys, vals = GEN[dtype](n, offset), inputs.index_payload(n)
    want_k, want_v = O.stable_sort(keys, vals, dtype)

    def shifted(a):
        t = torch.empty(n + offset + 8, dtype=a.dtype, device="cuda")
        t[offset:offset + n] = a
        return t[offset:offset + n]
    kin, vin = shifted(pgs.as_device_keys(keys, dtype)), shifted(torch.from_numpy(vals.view(np.int32)).cuda())
    ws = pgs.workspace(n, P, pgs.make_config(dtype=dtype))
    bounds = torch.zeros(P + 1, dtype=torch.int64, device="cuda")
    for b in (None, bounds):
        cfg = pgs.make_config(dtype=dtype, workspace=ws, bucket_bounds=b)
        ko, vo = shifted(torch.zeros_like(kin)), shifted(torch.zeros_like(vin))
        pgs.pgs_sort_copy(kin, vin if with_vals else None, ko, vo if with_vals else None, P, cfg)
        assert np.array_equal(pgs.to_numpy_keys(ko, dtype), want_k)
        if with_vals:
            assert np.array_equal(vo.cpu().numpy().view(np.uint32), want_v)
    assert np.array_equal(bounds.cpu().numpy(), O.buckets(keys, P, dtype)["e"])
    pgs.pgs_sort(kin, vin if with_vals else None, P, cfg)
    assert np.array_equal(pgs.to_numpy_keys(kin, dtype), want_k)


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
@pytest.mark.parametrize("per_thread", [4, 8, 16, 20])
@pytest.mark.parametrize("tiles,delta", [(1, -1), (1, 0), (1, 1), (3, 0), (304, -1), (304, 0), (304, 1)])
def test_small_and_tiny_forms_at_their_limits(dtype, per_thread, tiles, delta):
    """One CTA up to 384 x 8 and 384 x 20 (wide keys 16) keys; one cooperative
    launch of at most 304 tiles of 384 x 4, 8 and 20 (16) keys; three launches
    a pass beyond."""
    n = tiles * 384 * per_thread + delta
    for P in (66, 300) if tiles == 1 else (70,):
        check_against_oracle(GEN[dtype](n, tiles), inputs.index_payload(n), P, dtype)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("n", [1, 2, 33, 1000, 3072])
@pytest.mark.parametrize("P", [1, 2, 33, 255, 256, 257])
def test_tiny_sorts_with_every_rule(dtype, n, P):
    keys = inputs.structured_u32("few", n).astype(np.uint64 if dtype == "u64" else np.uint32)
    for variant in (0, 1, 2):
        check_against_oracle(keys, inputs.index_payload(n), P, dtype, s=3, variant=variant)
        check_against_oracle(GEN[dtype](n, P), None, P, dtype, variant=variant)


def test_small_sorts_on_two_streams_at_once():
    """Two cooperative sorts that each fill the GPU, issued on two streams
    without waiting, many times: both finish and both are right."""
    import torch
    from paper_1611_00463_gb300 import pgs
    n, P = 304 * 384 * 20, 16
    work = []
    for i in range(2):
        keys = inputs.uniform_u32(n, 40 + i)
        kin = pgs.as_device_keys(keys, "u32")
        ko = torch.empty_like(kin)
        st = torch.zeros(pgs.STATS_BYTES, dtype=torch.uint8, device="cuda")
        cfg = pgs.make_config(workspace=pgs.workspace(n, P, pgs.make_config()), stats=st, graph_cache="off")
        work.append((keys, kin, ko, st, cfg, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(20):
        for _, kin, ko, _, cfg, s in work:
            pgs.pgs_sort_copy(kin, None, ko, None, P, cfg, stream=s)
    for keys, _, ko, st, _, s in work:
        assert pgs.pgs_get_stats(st, s)["error"] == 0
        assert np.array_equal(pgs.to_numpy_keys(ko, "u32"), np.sort(keys))


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
def test_batch_of_uneven_instances_with_and_without_stats(dtype):
    from tests.test_gpu_batched import check, run_batch
    T = TILE[dtype]
    sizes = [T, T + 1, 0, 3 * T - 1, 1, 2 * T, 70 * T + 5]
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    n = int(offsets[-1])
    keys, vals = GEN[dtype](n, 5), inputs.index_payload(n)
    P = np.array([3, 70, 1, 300, 5, 1, 16], dtype=np.uint32)
    Peff = [max(1, min(int(p), s)) for p, s in zip(P, sizes)]
    got_k, got_v, st = run_batch(offsets, keys, vals, P, dtype)
    check(offsets, keys, vals, got_k, got_v, Peff, dtype)
    loads = [O.buckets(keys[int(a):int(b)], p, dtype)["stats"] for a, b, p in zip(offsets, offsets[1:], Peff) if b > a]
    assert st["max_bucket"] == max(x["max"] for x in loads)
    assert st["min_bucket"] == 0                      # the empty instance's bucket
    got_k, _, _ = run_batch(offsets, keys, None, P, dtype, graph=True)
    check(offsets, keys, None, got_k, None, Peff, dtype)


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
def test_a_workspace_sized_for_merges_still_sorts(dtype):
    """A workspace queried for a merge width (smaller than the radix form's)
    was enough for every call of that size, and still is."""
    import torch
    from paper_1611_00463_gb300 import pgs
    n, P = 300_007, 80
    keys, vals = GEN[dtype](n, 8), inputs.index_payload(n)
    small = pgs.workspace(n, P, pgs.make_config(dtype=dtype, merge_ways=2))
    full = pgs.workspace(n, P, pgs.make_config(dtype=dtype))
    out = []
    for ws in (small, full):
        kin = pgs.as_device_keys(keys, dtype)
        vin = torch.from_numpy(vals.view(np.int32)).cuda()
        bounds = torch.zeros(P + 1, dtype=torch.int64, device="cuda")
        pgs.pgs_sort(kin, vin, P, pgs.make_config(dtype=dtype, workspace=ws, bucket_bounds=bounds))
        out.append((pgs.to_numpy_keys(kin, dtype), vin.cpu().numpy(), bounds.cpu().numpy()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
