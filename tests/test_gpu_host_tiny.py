"""Host-buffer sorts of the sizes one CTA sorts: one launch, every output as the
oracle has it; one key more takes the ordinary launches."""
import numpy as np
import pytest

from oracle import pgs_oracle as O
from paper_1611_00463_gb300 import inputs
from tests.test_gpu_host import host_tensor

pytestmark = pytest.mark.gpu

GEN = {"u32": inputs.uniform_u32, "u64": inputs.normal_lognormal_u64, "f32": inputs.zipf_dup_f32}
MOST = {"u32": 960 * 8, "f32": 960 * 8, "u64": 768 * 8}


@pytest.mark.parametrize("dtype", ["u32", "u64", "f32"])
@pytest.mark.parametrize("with_vals", [False, True])
@pytest.mark.parametrize("size", [1, 384 * 8, 384 * 8 + 1, 0, -1])     # 0: the most one CTA sorts; -1: one more
@pytest.mark.parametrize("P", [1, 4, 256])
def test_tiny_host_sort(dtype, with_vals, size, P):
    import torch
    from paper_1611_00463_gb300 import pgs
    n = size if size > 0 else MOST[dtype] - size
    Pe = max(1, min(P, n))
    keys, vals = GEN[dtype](n, n + P), inputs.index_payload(n)
    hk = host_tensor(keys, dtype, True)
    hv = host_tensor(vals, "u32", True) if with_vals else None
    ko, vo = torch.empty_like(hk).pin_memory(), torch.empty(n, dtype=torch.int32).pin_memory() if with_vals else None
    ws = torch.empty(pgs.pgs_host_workspace_bytes(n, P, pgs.make_config(dtype=dtype)), dtype=torch.uint8, device="cuda")
    e = torch.empty(Pe + 1, dtype=torch.int64, device="cuda")
    cuts = torch.empty(Pe * (Pe + 1), dtype=torch.int64, device="cuda")
    st = torch.zeros(pgs.STATS_BYTES, dtype=torch.uint8, device="cuda")
    pgs.pgs_sort_host(hk, hv, ko, vo, P, pgs.make_config(dtype=dtype, workspace=ws, bucket_bounds=e, cuts=cuts, stats=st))
    torch.cuda.synchronize()
    want_k, want_v = O.stable_sort(keys, vals, dtype)
    ref = O.buckets(keys, P, dtype)
    assert np.array_equal(ko.numpy().view(want_k.dtype), want_k)
    assert not with_vals or np.array_equal(vo.numpy().view(np.uint32), want_v)
    assert np.array_equal(e.cpu().numpy(), ref["e"])
    assert np.array_equal(cuts.cpu().numpy().reshape(Pe, Pe + 1), ref["cut"])
    assert (pgs.pgs_get_stats(st)["launches"] == 1) == (size >= 0)
