"""Sorts under a spin_limit far below what a copy or a grid barrier takes: the
call either is right or reports PGS_ERR_TIMEOUT, the context stays usable, and
the next sort in the same workspace is right."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs

pytestmark = pytest.mark.gpu

LIMITS = [1, 1_000, 20_000]                               # ns


def short_then_right(n, P, dtype, stats, **opts):
    import torch
    from paper_1611_00463_gb300 import pgs
    keys = inputs.uniform_u32(n, n) if dtype == "u32" else inputs.normal_lognormal_u64(n, n)
    vals = inputs.index_payload(n)
    want_k, want_v = O.stable_sort(keys, vals, dtype)
    kin = pgs.as_device_keys(keys, dtype)
    vin = torch.from_numpy(vals.view(np.int32)).cuda()
    kout, vout = torch.empty_like(kin), torch.empty_like(vin)
    ws = pgs.workspace(n, P, pgs.make_config(dtype=dtype, **opts))
    outs = {}
    if stats:
        outs = {"stats": torch.zeros(pgs.STATS_BYTES, dtype=torch.uint8, device="cuda"),
                "bucket_bounds": torch.empty(P + 1, dtype=torch.int64, device="cuda"),
                "cuts": torch.empty(P * (P + 1), dtype=torch.int64, device="cuda")}

    def sort(limit):
        cfg = pgs.make_config(dtype=dtype, workspace=ws, spin_limit=limit, graph_cache="off", **outs, **opts)
        pgs.pgs_sort_copy(kin, vin, kout, vout, P, cfg)
        torch.cuda.synchronize()
        if stats:
            pgs.pgs_get_stats(outs["stats"])

    def right():
        return (np.array_equal(pgs.to_numpy_keys(kout, dtype), want_k) and
                np.array_equal(vout.cpu().numpy().view(np.uint32), want_v))

    gave_up = 0
    for limit in LIMITS:
        try:
            sort(limit)
            assert not stats or right()
        except pgs.PgsError as err:
            assert err.status == pgs.PGS_ERR_TIMEOUT
            gave_up += 1
        sort(0)
        assert right()
    return gave_up


@pytest.mark.parametrize("ways", [2, 4])
@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_merges(dtype, ways):
    short_then_right(3_000_017, 24, dtype, True, merge_ways=ways)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("n", [60_001, 1_000_003, 6_000_011])
def test_radix_keys_and_payloads_alone(n, dtype):
    short_then_right(n, 24, dtype, False)


@pytest.mark.parametrize("dtype", ["u32", "u64"])
@pytest.mark.parametrize("n,P", [(60_001, 24), (1_000_003, 200), (1_000_003, 700), (6_000_011, 24), (6_000_011, 700)])
def test_radix_with_bounds_cuts_and_stats(n, P, dtype):
    gave_up = short_then_right(n, P, dtype, True)
    # 1 ns is less than any grid barrier of several CTAs takes.
    assert gave_up > 0 or n > 1_000_003
