"""The radix form's bounded waits made to run out, without any GPU fault: a tile
that announces its copies and issues none, a CTA that waits at a grid barrier for
arrivals that never come.  The call reports PGS_ERR_TIMEOUT soon after
spin_limit, and the next sort in the same workspace is right, with all outputs."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs

pytestmark = pytest.mark.gpu

LIMIT_NS = 1_000_000
GEN = {"u32": inputs.uniform_u32, "u64": inputs.normal_lognormal_u64, "f32": inputs.zipf_dup_f32}


def times_out_then_right(fault, keys, P, dtype):
    import torch
    from paper_1611_00463_gb300 import pgs
    n, vals = len(keys), inputs.index_payload(len(keys))
    kin = pgs.as_device_keys(keys, dtype)
    vin = torch.from_numpy(vals.view(np.int32)).cuda()
    kout, vout = torch.empty_like(kin), torch.empty_like(vin)
    ws = pgs.workspace(n, P, pgs.make_config(dtype=dtype))
    ws.fill_(0xFF)                                        # tags that no pass wrote name no run
    st = torch.zeros(pgs.STATS_BYTES, dtype=torch.uint8, device="cuda")
    e = torch.empty(P + 1, dtype=torch.int64, device="cuda")
    cuts = torch.empty(P * (P + 1), dtype=torch.int64, device="cuda")
    spl = torch.empty(P - 1, dtype=kin.dtype, device="cuda")
    outs = dict(dtype=dtype, workspace=ws, stats=st, bucket_bounds=e, cuts=cuts, splitters_out=spl)
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    pgs.pgs_sort_copy(kin, vin, kout, vout, P,
                      pgs.make_config(spin_limit=LIMIT_NS, fault_inject=fault, graph_cache="off", **outs), stream)
    e1.record(stream)
    with pytest.raises(pgs.PgsError) as err:
        pgs.pgs_get_stats(st, stream)
    assert err.value.status == pgs.PGS_ERR_TIMEOUT
    ms = e0.elapsed_time(e1)
    assert 1.0 <= ms < 500.0, f"the injected wait took {ms} ms"
    pgs.pgs_sort_copy(kin, vin, kout, vout, P, pgs.make_config(**outs), stream)
    assert pgs.pgs_get_stats(st, stream)["error"] == 0
    want_k, want_v = O.stable_sort(keys, vals, dtype)
    ref = O.buckets(keys, P, dtype)
    assert np.array_equal(pgs.to_numpy_keys(kout, dtype), want_k)
    assert np.array_equal(vout.cpu().numpy().view(np.uint32), want_v)
    assert np.array_equal(e.cpu().numpy(), ref["e"])
    assert np.array_equal(cuts.cpu().numpy().reshape(P, P + 1), ref["cut"])
    assert np.array_equal(O.ord_bits(pgs.to_numpy_keys(spl, dtype), dtype), ref["splitters"])


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
@pytest.mark.parametrize("n,P", [(200_003, 24), (200_003, 300), (3_000_017, 24), (3_000_017, 300)])
def test_copies_that_never_come(n, P, dtype):
    times_out_then_right("radix_copies", GEN[dtype](n, n), P, dtype)


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
@pytest.mark.parametrize("n,P", [(20_003, 24), (1_000_003, 24), (1_000_003, 300)])
def test_one_launch_sorts_barrier(n, P, dtype):
    times_out_then_right("radix_barrier", GEN[dtype](n, n), P, dtype)


@pytest.mark.parametrize("P", [24, 300])
def test_clean_up_barrier(P):
    """Half the keys alike, ten next to them that a sample of 1024 misses (it meets one
    in 200 times): one long segment that all CTAs of the clean-up share."""
    n, g = 1_900_007, np.random.default_rng(P)
    keys = g.integers(0, 1 << 64, size=n, dtype=np.uint64)
    at = g.permutation(n)
    keys[at[:n // 2]] = np.uint64(7 << 40)
    keys[at[n // 2:n // 2 + 10]] = np.uint64(7 << 40) + g.integers(1, 50, size=10, dtype=np.uint64)
    times_out_then_right("radix_barrier", keys, P, "u64")


@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_batch(dtype):
    import torch
    from paper_1611_00463_gb300 import pgs
    offsets = np.array([0, 1_000_003, 1_000_003, 1_700_001, 2_500_007], dtype=np.uint64)
    keys, vals = GEN[dtype](int(offsets[-1]), 5), inputs.index_payload(int(offsets[-1]))
    bt = pgs.Batch(offsets, None, dtype=dtype, with_vals=True)
    k, v = pgs.as_device_keys(keys, dtype), torch.from_numpy(vals.view(np.int32)).cuda()
    ko, vo = torch.empty_like(k), torch.empty_like(v)
    st = torch.zeros(pgs.STATS_BYTES, dtype=torch.uint8, device="cuda")
    bt.sort_copy(k, v, ko, vo, cfg=pgs.make_config(dtype=dtype, workspace=bt.workspace, stats=st, spin_limit=LIMIT_NS,
                                                   fault_inject="radix_copies", graph_cache="off"))
    with pytest.raises(pgs.PgsError) as err:
        pgs.pgs_get_stats(st)
    assert err.value.status == pgs.PGS_ERR_TIMEOUT
    bt.sort_copy(k, v, ko, vo, cfg=bt.config(stats=st))
    assert pgs.pgs_get_stats(st)["error"] == 0
    got_k, got_v = pgs.to_numpy_keys(ko, dtype), vo.cpu().numpy().view(np.uint32)
    for a, b in zip(offsets[:-1].astype(int), offsets[1:].astype(int)):
        want_k, want_v = O.stable_sort(keys[a:b], vals[a:b], dtype)
        assert np.array_equal(got_k[a:b], want_k) and np.array_equal(got_v[a:b], want_v)
