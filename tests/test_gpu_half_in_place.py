"""Sorts whose payloads are in place while the keys are not, and the reverse,
against the oracle: one CTA, one launch and many, plans of an odd and of an even
number of passes, single sorts and batches."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs

pytestmark = pytest.mark.gpu

GEN = {"u32": inputs.uniform_u32, "u64": inputs.uniform_u64, "wide": inputs.normal_lognormal_u64}


def half_in_place(which, keys, vals, dtype, sort):
    """Calls sort(kin, vin, kout, vout) with one of the two outputs on its input."""
    import torch
    from paper_1611_00463_gb300 import pgs
    kin = pgs.as_device_keys(keys, dtype)
    vin = torch.from_numpy(vals.view(np.int32)).cuda()
    kout = kin if which == "keys" else torch.empty_like(kin)
    vout = vin if which == "vals" else torch.empty_like(vin)
    sort(kin, vin, kout, vout)
    torch.cuda.synchronize()
    if which == "vals":
        assert np.array_equal(pgs.to_numpy_keys(kin, dtype), keys)
    else:
        assert np.array_equal(vin.cpu().numpy().view(np.uint32), vals)
    return pgs.to_numpy_keys(kout, dtype), vout.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("which", ["keys", "vals"])
@pytest.mark.parametrize("bounds", [False, True])
@pytest.mark.parametrize("kind", ["u32", "u64", "wide"])
@pytest.mark.parametrize("n,P", [(5_000, 4), (300_007, 24), (2_500_003, 24), (2_500_003, 300), (20_000_003, 40)])
def test_single(n, P, kind, bounds, which):
    import torch
    from paper_1611_00463_gb300 import pgs
    dtype = "u32" if kind == "u32" else "u64"
    keys, vals = GEN[kind](n, n + P), inputs.index_payload(n)
    ws = pgs.workspace(n, P, pgs.make_config(dtype=dtype))
    e = torch.empty(P + 1, dtype=torch.int64, device="cuda") if bounds else None
    cfg = pgs.make_config(dtype=dtype, workspace=ws, bucket_bounds=e)
    k, v = half_in_place(which, keys, vals, dtype, lambda ki, vi, ko, vo: pgs.pgs_sort_copy(ki, vi, ko, vo, P, cfg))
    want_k, want_v = O.stable_sort(keys, vals, dtype)
    assert np.array_equal(k, want_k) and np.array_equal(v, want_v)


@pytest.mark.parametrize("which", ["keys", "vals"])
@pytest.mark.parametrize("kind", ["u32", "u64", "wide"])
def test_batch(kind, which):
    from paper_1611_00463_gb300 import pgs
    dtype = "u32" if kind == "u32" else "u64"
    sizes = [2_000_003, 1, 0, 700_001, 90_000, 3_000_017]
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    keys, vals = GEN[kind](int(offsets[-1]), 7), inputs.index_payload(int(offsets[-1]))
    bt = pgs.Batch(offsets, None, dtype=dtype, with_vals=True)
    k, v = half_in_place(which, keys, vals, dtype, bt.sort_copy)
    for a, b in zip(offsets[:-1].astype(int), offsets[1:].astype(int)):
        want_k, want_v = O.stable_sort(keys[a:b], vals[a:b], dtype)
        assert np.array_equal(k[a:b], want_k) and np.array_equal(v[a:b], want_v)
