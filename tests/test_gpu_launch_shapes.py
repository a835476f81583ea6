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
    """The tensor-core kernel's output and LSE and the CUDA-core kernel's, on the same codes and index sets.  The workspace
    starts out full of NaN patterns: nothing that the pre-pass leaves out may be read."""
    idx = api.hyq_select_vertical(Q, K, W, k) if k else None
    qz = [api.hyq_quantize_blocks(t, f) for t, f in zip((Q, K, V), fmts)]
    res = []
    for impl in (api.IMPL_TCGEN05, api.IMPL_SIMT):
        lse = torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        out = api.hyq_hybrid_attention_prefill(Q, K, V, qz[0][0], qz[1][0], qz[2][0], qz[0][1], qz[1][1], qz[2][1], fmts, idx, W,
                                               workspace=torch.full((400 << 20,), 0xFF, dtype=torch.uint8, device="cuda"),
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


@pytest.mark.parametrize("fmts", [INT8, FP8ALL, INT4FP8])
@pytest.mark.parametrize("Hq,Hkv,L,Lq,W,k,mode,out", [
    (2, 2, 2048, 2048, 128, 32, 0, torch.float32),      # a whole prefill of few units
    (1, 1, 3333, 3333, 100, 70, 0, torch.bfloat16),     # ragged last tile, bf16 rows from the merge and from whole pieces
    (4, 2, 9000, 777, 256, 200, 0, torch.float32),      # a query block, last unit of 9 rows
    (4, 1, 6000, 1500, 512, 100, 1, torch.bfloat16),    # fixed window: equal units
    (2, 2, 5003, 900, 1000, 50, 1, torch.float32),      # fixed window wider than the block, ragged last key tile
    (2, 2, 5003, 300, 2000, 50, 0, torch.float32),      # a window from the middle of a key tile on
    (1, 1, 20000, 1, 64, 300, 0, torch.float32),        # one row: most pieces have one live query tile
])
def test_units_shared_by_several_ctas(fmts, Hq, Hkv, L, Lq, W, k, mode, out):
    ensure_built()
    Q, K, V = _normal((1, Hq, Lq, 128), L), _normal((1, Hkv, L, 128), L + 1), _normal((1, Hkv, L, 128), L + 2)
    _close(*_both_kernels(Q, K, V, fmts, W, k, out, window_mode=mode))


@pytest.mark.parametrize("fmts", [INT8, FP8ALL])
@pytest.mark.parametrize("j_star,again", [(-1, False), (1336, True)])
def test_dominant_key_in_window_tiles_taken_without_their_maximum(fmts, j_star, again):
    """Quiet low-bit keys, and one key whose score lies 19 log2 units above the others', in the window of all later rows."""
    ensure_built()
    u = torch.ones(128, device="cuda") / 128 ** 0.5
    Q, K, V = _normal((1, 64, 1536, 128), 1) + (6.0 * u).bfloat16(), _normal((1, 1, 1536, 128), 2), _normal((1, 1, 1536, 128), 3)
    if j_star >= 0:
        K[:, :, j_star] = (30.0 * u).bfloat16()
    api.hyq_test_read_attention_restarts(reset=True)
    _close(*_both_kernels(Q, K, V, fmts, 512, 0))
    assert (api.hyq_test_read_attention_restarts(reset=True) > 0) == again


def _packed_calls(qs, ks, vs, W, k_per, fmts, all_in_one):
    """The three *_varlen calls on packed buffers; the attention's workspace for all prompts at once or the smallest accepted."""
    import ctypes
    lib = api.lib()
    n, Hq, Hkv = len(qs), qs[0].shape[0], ks[0].shape[0]
    (qp, cu), (kp, _), (vp, _) = (api.pack_sequences(t) for t in (qs, ks, vs))
    lens = [cu[i + 1] - cu[i] for i in range(n)]
    cu_c, k_c = api._i32(cu), api._i32(k_per)
    empty = lambda m, dt=torch.uint8: torch.empty(max(m, 16), dtype=dt, device="cuda")       # noqa: E731
    idx = empty(Hq * sum(k_per), torch.int32)
    ws = empty(max(api.hyq_select_vertical_workspace(1, Hq, Hkv, L, L, 128, W, k) for L, k in zip(lens, k_per)) * (20 if all_in_one else 1))
    api._check(lib.hyq_select_vertical_varlen(qp.data_ptr(), kp.data_ptr(), n, cu_c, Hq, Hkv, 128, W, 0, k_c, idx.data_ptr(),
                                              ws.data_ptr(), ws.numel(), api._stream()), "select")
    qz = []
    for x, H, f in ((qp, Hq, fmts[0]), (kp, Hkv, fmts[1]), (vp, Hkv, fmts[2])):
        c, sc = empty(H * cu[-1] * api.code_row_bytes(f, 128)), empty(H * sum(-(-L // 64) for L in lens), torch.float32)
        api._check(lib.hyq_quantize_blocks_varlen(x.data_ptr(), n, cu_c, H, 128, 64, f, c.data_ptr(), sc.data_ptr(), api._stream()), "quantize")
        qz.append((c, sc))
    out = torch.empty(Hq * cu[-1] * 128, device="cuda")
    a = api.AttnArgs()
    a.struct_size = ctypes.sizeof(api.AttnArgs)
    a.B, a.Hq, a.Hkv, a.L, a.D, a.window, a.block_tokens, a.out_dtype = 1, Hq, Hkv, max(lens), 128, W, 64, 1
    a.q_format, a.k_format, a.v_format = fmts
    a.k = k_per[lens.index(max(lens))]
    a.q, a.k_, a.v, a.vl_idx, a.out = qp.data_ptr(), kp.data_ptr(), vp.data_ptr(), idx.data_ptr(), out.data_ptr()
    a.q_codes, a.k_codes, a.v_codes = (c.data_ptr() for c, _ in qz)
    a.q_scales, a.k_scales, a.v_scales = (sc.data_ptr() for _, sc in qz)
    need = ctypes.c_size_t(0)
    if all_in_one:
        api._check(lib.hyq_hybrid_attention_prefill_varlen_workspace(ctypes.byref(a), n, cu_c, k_c, ctypes.byref(need)), "workspace")
    else:
        api._check(lib.hyq_hybrid_attention_prefill_workspace(ctypes.byref(a), ctypes.byref(need)), "workspace")
    ws = empty(need.value)
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    api._check(lib.hyq_hybrid_attention_prefill_varlen(ctypes.byref(a), n, cu_c, k_c, api._stream()), "attention")
    return [out[Hq * 128 * cu[i]:Hq * 128 * cu[i + 1]].view(Hq, lens[i], 128) for i in range(n)]


@pytest.mark.parametrize("fmts", [INT8, INT4FP8])
def test_ragged_batches_of_any_launch_grouping_give_the_same_bits(fmts):
    """40 prompts (more than one launch holds; among them prompts whose units are shared by several CTAs): the whole path in
    one call on the prompts where they lie, the three packed calls with all the workspace and with the longest prompt's alone
    (launches of a few prompts each), and the plain calls on a prompt by itself."""
    ensure_built()
    rng = np.random.default_rng(5)
    lens = [int(x) for x in np.exp(rng.uniform(np.log(1), np.log(3000), 39))] + [3000]
    qs, ks, vs = ([_normal((h, L, 128), 100 * h + n) for n, L in enumerate(lens)] for h in (6, 2, 2))
    k_per = [max(0, L - 128) // 40 for L in lens]
    one = api.hybrid_prefill_varlen(qs, ks, vs, 128, k_per, fmts)
    for all_in_one in (True, False):
        for r, out in zip(one, _packed_calls(qs, ks, vs, 128, k_per, fmts, all_in_one)):
            assert torch.equal(r["out"], out)
    for n in (0, 17, 39):
        alone = api.hybrid_prefill(qs[n][None], ks[n][None], vs[n][None], 128, k_per[n], fmts)
        for name in alone:
            assert torch.equal(alone[name][0], one[n][name]), name
        # stage by stage
        qz = [api.hyq_quantize_blocks(t[n][None], f) for t, f in zip((qs, ks, vs), fmts)]
        idx = api.hyq_select_vertical(qs[n][None], ks[n][None], 128, k_per[n])
        out = api.hyq_hybrid_attention_prefill(qs[n][None], ks[n][None], vs[n][None], qz[0][0], qz[1][0], qz[2][0], qz[0][1],
                                               qz[1][1], qz[2][1], fmts, idx, 128)
        assert torch.equal(out[0], one[n]["out"]) and torch.equal(idx[0], one[n]["idx"])


# ---- selection: the oracle's index sets bit for bit ---------------------------------------------------------------
def _select_is_the_oracles(Q, K, W, k, n_tail=0):
    import oracle
    got = api.hyq_select_vertical(Q.cuda(), K.cuda(), W, k, n_tail=n_tail).cpu().numpy()
    np.testing.assert_array_equal(got, oracle.select_vertical(wl.bits(Q), wl.bits(K), W, k, n_tail=n_tail))


@pytest.mark.parametrize("P,k", [(1, 1), (255, 255), (257, 3), (4096, 80), (4097, 4097), (8193, 160), (16385, 5), (40001, 900)])
def test_topk_over_one_to_eight_ctas(P, k):
    ensure_built()
    W = 64
    Q, K = _normal((1, 2, W, 128), P).cpu(), _normal((1, 1, P + W, 128), P + 1).cpu()
    _select_is_the_oracles(Q, K, W, k)


@pytest.mark.parametrize("kind", ["ties", "all_equal", "far_below_the_maximum", "narrow", "most_negative"])
def test_topk_where_one_sweep_does_not_settle_it(kind):
    """Scores are K's channel 0 times the tail mean's (the other channels are zero): equal keys, a threshold more than 16
    octaves below the maximum, scores that agree in all leading bits, a threshold among negative scores."""
    ensure_built()
    W, P = 32, 6000
    g = torch.Generator().manual_seed(11)
    c = {"ties": torch.randint(0, 4, (P,), generator=g).float(),
         "all_equal": torch.full((P,), 3.0),
         "far_below_the_maximum": torch.cat([torch.full((5,), 2.0**60), torch.rand(P - 5, generator=g)]),
         "narrow": 128.0 + torch.randint(0, 3, (P,), generator=g).float(),
         "most_negative": torch.randn(P, generator=g) - 3.0}[kind]
    K = torch.zeros(1, 1, P + W, 128)
    K[0, 0, :P, 0] = c
    Q = torch.zeros(1, 2, W, 128)
    Q[:, :, :, 0] = 1.0
    _select_is_the_oracles(Q.bfloat16(), K.bfloat16(), W, 700)


@pytest.mark.parametrize("Hq,Hkv,P", [(1, 1, 129), (2, 1, 300), (3, 1, 257), (5, 1, 700), (8, 1, 128), (9, 1, 513), (16, 8, 9000), (40, 8, 9001)])
def test_scores_for_every_group_size_and_both_key_counts_per_thread(Hq, Hkv, P):
    ensure_built()
    W = 48
    Q, K = _normal((1, Hq, W, 128), P).cpu(), _normal((1, Hkv, P + W, 128), P + 1).cpu()
    K[0, 0, 5] = 2.0**-130                     # bf16 subnormals, an all-zero row, one large row
    K[0, 0, 6] = 0.0
    K[0, 0, 7] = 2.0**100
    _select_is_the_oracles(Q, K, W, max(1, P // 10))


@pytest.mark.parametrize("t", [1, 2, 15, 16, 65, 300])
@pytest.mark.parametrize("spread", [0, 20, 34, 60])
def test_tail_mean_in_any_order_and_in_row_order(t, spread):
    """Exponent spreads on either side of what keeps every partial sum exact (53 - 8 - log2 t bits)."""
    ensure_built()
    Q, K = _normal((1, 2, 300, 128), t).cpu().float(), _normal((1, 1, 400, 128), t + 1).cpu()
    e = torch.randint(-spread // 2, spread // 2 + 1, Q.shape, generator=torch.Generator().manual_seed(t + spread))
    Q = (Q * torch.exp2(e.float())).bfloat16()
    Q[0, 0, -1, :7] = 0.0
    _select_is_the_oracles(Q, K, 100, 150, n_tail=t)


# ---- ragged decode ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("lens", [
    [300] * 3 + [9000],                       # one sequence with almost all of the bytes: slices by share
    [40 + 7 * i for i in range(131)],         # more sequences than one table of lengths holds, some shorter than the window
    [17],
])
def test_ragged_steps_with_slices_by_share(lens):
    """Appends to the first and the last sequence, then the attention: slices by share against the same slices for all
    (bounds: the suite's for the decode attention), and with a workspace that has room for the latter only."""
    from paper_2608_27875_b200 import decode_api as dapi
    ensure_built()
    B, Hq, Hkv, W = len(lens), 4, 2, 64
    rc = dapi.RaggedKvCache(B, Hq, Hkv, max(lens), W, 8, staging_capacity=4)
    for b, n in enumerate(lens):
        rc.freeze_sequence(b, _normal((1, Hkv, n, 128), b), _normal((1, Hkv, n, 128), 500 + b), None)
    for i, b in enumerate((0, B - 1, -1)):
        rc.append(b, _normal((Hkv, 128), 900 + i), _normal((Hkv, 128), 950 + i))
    assert torch.equal(rc.lengths.cpu(), rc.lengths_host) and int(rc.lengths_host[:, 3].sum()) == 3
    with pytest.raises(IndexError):
        rc.append(B, _normal((Hkv, 128), 1), _normal((Hkv, 128), 2))
    q = _normal((B, Hq, 128), 7)
    share, even = (dapi.hyq_hybrid_attention_decode_ragged(q, rc, splits=n, out_dtype=torch.float32) for n in (0, 2))
    n = dapi.hyq_hybrid_attention_decode_workspace(rc.batch, 1)
    small = torch.empty(n if B == 1 else max(n, dapi.hyq_hybrid_attention_decode_workspace(rc.batch, 0) // 2), dtype=torch.uint8, device="cuda")
    outs = [share]
    if B > 1:
        outs.append(dapi.hyq_hybrid_attention_decode_ragged(q, rc, out_dtype=torch.float32, workspace=small))
    for out in outs:
        d = (out - even).abs()
        assert float(d.max()) <= MAX_ABS_TOL and float(d.sum() / even.abs().sum()) <= MEAN_REL_TOL


# ---- column-mass selector: query counts by which the warps share the keys, key counts around its blocks ------------
@pytest.mark.parametrize("Hq,Hkv,Lq,Lk,W,nT,k", [
    (2, 1, 64, 700, 64, 4, 30), (2, 2, 64, 513, 64, 5, 449), (4, 2, 64, 512, 40, 8, 20), (2, 1, 64, 769, 30, 9, 40),
    (3, 1, 33, 1025, 33, 33, 60),
    (2, 1, 512, 16640, 512, 512, 300),                          # a head's scores fill a group: one round of launches each
])
def test_mass_selector_by_query_count(Hq, Hkv, Lq, Lk, W, nT, k):
    ensure_built()
    import oracle
    Q, K = _normal((1, Hq, Lq, 128), Lk).cpu(), _normal((1, Hkv, Lk, 128), Lk + 1).cpu()
    got = api.hyq_select_vertical_mass(Q.cuda(), K.cuda(), W, k, nT).cpu().numpy()
    np.testing.assert_array_equal(got, oracle.select_vertical_mass(wl.bits(Q), wl.bits(K), W, k, nT))
