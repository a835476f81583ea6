"""GPU checks of the rules by which the library picks a launch: each at the sizes where its branches meet, against
the CUDA-core kernel or the oracle."""
import numpy as np
import pytest
import torch

from gpu_util import MAX_ABS_TOL, MEAN_REL_TOL, ensure_built
from paper_2608_27875_b200 import api, workloads as wl

pytestmark = pytest.mark.gpu
INT8 = (wl.FMT_INT8,) * 3
FP8ALL = (wl.FMT_FP8_E4M3,) * 3
INT4FP8 = (wl.FMT_INT4, wl.FMT_INT4, wl.FMT_FP8_E4M3)


def _normal(shape, seed):
    return torch.randn(*shape, generator=torch.Generator("cuda").manual_seed(seed), device="cuda").bfloat16()


def _both_kernels(Q, K, V, fmts, W, k, out_dtype=torch.float32, **kw):
    """The tensor-core kernel's output and LSE and the CUDA-core kernel's, on the same codes and index sets."""
    idx = api.hyq_select_vertical(Q, K, W, k) if k else None
    qz = [api.hyq_quantize_blocks(t, f) for t, f in zip((Q, K, V), fmts)]
    res = []
    for impl in (api.IMPL_TCGEN05, api.IMPL_SIMT):
        lse = torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        out = api.hyq_hybrid_attention_prefill(Q, K, V, qz[0][0], qz[1][0], qz[2][0], qz[0][1], qz[1][1], qz[2][1], fmts, idx, W,
                                               out_dtype=out_dtype, lse=lse, status_word=status, impl=impl, **kw)
        assert int(status.item()) == 0
        res += [out.float(), lse]
    return res


def _close(tc, lse_tc, simt, lse_simt):
    diff = (tc - simt).abs()
    assert torch.isfinite(tc).all() and float(diff.max()) <= MAX_ABS_TOL
    assert float(diff.sum() / simt.abs().sum()) <= MEAN_REL_TOL
    assert float((lse_tc - lse_simt).abs().max()) <= 2e-3       # the bound of the suite's other LSE comparisons


@pytest.mark.parametrize("B,Hq,Hkv,L,Lq", [
    (1, 3, 3, 50000, 600),        # two KV heads to a group, one left over
    (2, 6, 3, 24000, 520),        # GQA, groups across the batch boundary, the last one short
    (1, 2, 1, 140000, 300),       # a KV head larger than the budget: groups of one
])
def test_heads_interleaved_in_groups(B, Hq, Hkv, L, Lq):
    ensure_built()
    Q, K, V = _normal((B, Hq, Lq, 128), L), _normal((B, Hkv, L, 128), L + 1), _normal((B, Hkv, L, 128), L + 2)
    _close(*_both_kernels(Q, K, V, INT8, 256, 100))
