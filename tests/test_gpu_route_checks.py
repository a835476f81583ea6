"""GPU checks that calls keep their results, their workspaces and their pace whatever launch the library picks for them."""
import ctypes

import pytest
import torch

from gpu_util import MAX_ABS_TOL, MEAN_REL_TOL, ensure_built
from paper_2608_27875_b200 import api, decode_api as dapi
from test_gpu_launch_shapes import FP8ALL, INT4FP8, INT8, _both_kernels, _close, _normal, _packed_calls

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmts,out", [(INT8, torch.float32), (INT4FP8, torch.bfloat16)])
def test_ctas_that_go_on_from_a_unit_with_a_ragged_end(fmts, out):
    """160 units of 200 rows (eight of their last warp's 32) shared by 148 CTAs: most CTAs write such a unit's rows from the
    buffers that their next unit's queries are loaded into."""
    ensure_built()
    Q, K, V = _normal((4, 40, 200, 128), 1), _normal((4, 8, 3000, 128), 2), _normal((4, 8, 3000, 128), 3)
    for _ in range(3):
        _close(*_both_kernels(Q, K, V, fmts, 256, 40, out))


def test_the_longest_prompts_workspace_is_enough_for_a_batch_with_shorter_ones():
    """The longest prompt's units are not shared by several CTAs and leave no partial results, the shorter one's are."""
    ensure_built()
    Hq, W, lens = 8, 256, [6016, 1536]
    qs, ks, vs = ([_normal((Hq, L, 128), 10 * h + n) for n, L in enumerate(lens)] for h in range(3))
    k_per = [(L - W) // 50 for L in lens]
    one = api.hybrid_prefill_varlen(qs, ks, vs, W, k_per, INT8)
    for r, out in zip(one, _packed_calls(qs, ks, vs, W, k_per, INT8, False)):
        assert torch.equal(r["out"], out)


def test_the_mass_selectors_workspace_of_a_longer_context_is_enough_for_a_shorter_one():
    """512 queries: the kept scores of two heads fit a group at 11000 keys, those of one do at 15000."""
    ensure_built()
    q, k = _normal((1, 2, 512, 128), 1), _normal((1, 1, 15000, 128), 2)
    n = ctypes.c_size_t(0)
    api._check(api.lib().hyq_select_vertical_mass_workspace(1, 2, 1, 512, 15000, 128, 512, 512, 200, ctypes.byref(n)), "workspace")
    ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    short = k[:, :, :11000].contiguous()
    assert torch.equal(api.hyq_select_vertical_mass(q, short, 512, 200, 512, workspace=ws), api.hyq_select_vertical_mass(q, short, 512, 200, 512))


@pytest.mark.parametrize("fmts", [INT8, FP8ALL])
def test_a_window_key_a_little_above_the_reference_gives_the_same_bits_alone_and_in_a_batch(fmts):
    """One window key whose score lies 12 to 16 log2 units above a row's reference: above what raises the reference where the
    maximum is looked at, and not enough to have the piece done again where it is not.  64 heads x 2560: not shared by CTAs."""
    ensure_built()
    u = torch.ones(128, device="cuda") / 128 ** 0.5
    def queries(L, seed):                                       # noqa: E306 (each query 6 units along u: one score for all rows)
        q = _normal((64, L, 128), seed).float()
        return (q + (6.0 - q @ u).unsqueeze(-1) * u).bfloat16()
    lens, W = [2560, 700], 512
    qs, (ks, vs) = [queries(L, n) for n, L in enumerate(lens)], ([_normal((1, L, 128), 10 * h + n) for n, L in enumerate(lens)] for h in (1, 2))
    ks[0][:, 2300] = (23.0 * u).bfloat16()
    api.hyq_test_read_attention_restarts(reset=True)
    alone = api.hybrid_prefill(qs[0][None], ks[0][None], vs[0][None], W, 0, fmts)
    batch = api.hybrid_prefill_varlen(qs, ks, vs, W, [0, 0], fmts)
    assert api.hyq_test_read_attention_restarts(reset=True) == 0
    assert torch.equal(alone["out"][0], batch[0]["out"])


def _ragged_cache(lens, Hkv, W=128):
    rc = dapi.RaggedKvCache(len(lens), 4 * Hkv, Hkv, max(lens), W, 8)
    for b, n in enumerate(lens):
        rc.freeze_sequence(b, _normal((1, Hkv, n, 128), b), _normal((1, Hkv, n, 128), 1000 + b), None)
    return rc, _normal((len(lens), 4 * Hkv, 128), 7)


def _median_us(calls, n=20, rounds=5):
    """Median device time of each call, the calls in turn."""
    times = [[] for _ in calls]
    for r in range(rounds + 1):
        for t, f in zip(times, calls):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(n):
                f()
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b) / n * 1e3)
    return [sorted(t[1:])[rounds // 2] for t in times]


@pytest.mark.parametrize("n,Hkv", [(64, 8), (74, 8), (100, 8), (300, 2)])
def test_large_ragged_batches_take_no_longer_than_with_one_slice_each(n, Hkv):
    """Sequences of 100 to 700 rows, a slice per head whichever way they are cut: what a CTA spends on finding its slice may not
    show (bound: half as long again; the search that every CTA once made took 1.9 to 25 times as long)."""
    ensure_built()
    lens = [100 + (97 * b) % 600 for b in range(n)]
    rc, q = _ragged_cache(lens, Hkv)
    outs = [torch.empty(n, 4 * Hkv, 128, device="cuda") for _ in range(2)]
    ws = [torch.empty(dapi.hyq_hybrid_attention_decode_workspace(rc.batch, s), dtype=torch.uint8, device="cuda") for s in (0, 1)]
    calls = [lambda s=s: dapi.hyq_hybrid_attention_decode_ragged(q, rc, splits=s, out=outs[s], workspace=ws[s]) for s in (0, 1)]
    share, one = _median_us(calls)
    assert share <= 1.5 * one, (share, one)
    d = (outs[0] - outs[1]).abs()
    assert float(d.max()) <= MAX_ABS_TOL and float(d.sum() / outs[1].abs().sum()) <= MEAN_REL_TOL


def _block_call(Q, K, V, fmts, W, k):
    idx = api.hyq_select_vertical(Q, K, W, k)
    qz = [api.hyq_quantize_blocks(t, f) for t, f in zip((Q, K, V), fmts)]
    out = torch.empty(Q.shape, device="cuda")
    return lambda: api.hyq_hybrid_attention_prefill(Q, K, V, qz[0][0], qz[1][0], qz[2][0], qz[0][1], qz[1][1], qz[2][1], fmts, idx, W, out=out)


@pytest.mark.parametrize("B,Hq,Hkv,L,Lq,fmts", [(1, 32, 8, 20000, 2000, INT8), (2, 32, 4, 20000, 1000, FP8ALL), (1, 40, 8, 12000, 3001, INT4FP8)])
def test_a_query_block_with_a_ragged_last_tile_takes_no_longer_than_a_full_one(B, Hq, Hkv, L, Lq, fmts):
    """Against the next multiple of 256 rows (bound: a fifth more; with its ragged tiles at half the pace 1.6 to 1.9 times)."""
    ensure_built()
    K, V = _normal((B, Hkv, L, 128), 2), _normal((B, Hkv, L, 128), 3)
    short, full = _median_us([_block_call(_normal((B, Hq, n, 128), 1), K, V, fmts, 512, 390) for n in (Lq, -(-Lq // 256) * 256)], n=5, rounds=5)
    assert short <= 1.2 * full, (short, full)


@pytest.mark.parametrize("fmts", [INT8, INT4FP8])
@pytest.mark.parametrize("B,Hq,Hkv,L,Lq,W,k", [
    (1, 2, 2, 20010, 20010, 256, 395),      # a whole prefill: CTAs with one piece at the long end, a dozen short units at the other
    (1, 4, 1, 9000, 9000, 0, 0),            # no window: units down to four tiles, shorter than the cost of beginning them
    (3, 16, 4, 5000, 700, 200, 60),         # a query block, three units per head
    (1, 1, 1, 30000, 3, 64, 300),           # one unit for all CTAs
])
def test_shares_that_count_what_a_unit_costs_to_begin(fmts, B, Hq, Hkv, L, Lq, W, k):
    ensure_built()
    Q, K, V = _normal((B, Hq, Lq, 128), L), _normal((B, Hkv, L, 128), L + 1), _normal((B, Hkv, L, 128), L + 2)
    if W == 0:                              # (the selector's tail mean needs a window or a count)
        idx = torch.arange(0, L, 97, dtype=torch.int32, device="cuda").expand(B, Hq, -1).contiguous()
    else:
        idx = api.hyq_select_vertical(Q, K, W, k)
    qz = [api.hyq_quantize_blocks(t, f) for t, f in zip((Q, K, V), fmts)]
    res = []
    for impl in (api.IMPL_TCGEN05, api.IMPL_SIMT):
        lse = torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
        out = api.hyq_hybrid_attention_prefill(Q, K, V, qz[0][0], qz[1][0], qz[2][0], qz[0][1], qz[1][1], qz[2][1], fmts, idx, W, lse=lse, impl=impl)
        res += [out, lse]
    _close(*res)


def test_an_unknown_attention_kernel_is_refused():
    ensure_built()
    q, k = _normal((1, 2, 200, 128), 1), _normal((1, 1, 200, 128), 2)
    for impl in (-1, 3):
        with pytest.raises(api.HyqError) as e:
            api.hybrid_prefill(q, k, k, 64, 3, impl=impl)
        assert e.value.code == 1
