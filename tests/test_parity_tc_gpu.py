"""GPU parity of the tensor-core scoring path (bf16, head_dim 128) and of the
fused pass on bf16 caches, against the CPU oracle."""
import math
import dataclasses

import numpy as np
import pytest
import torch

from oracle import refree_oracle as orc
from paper_2502_16886_b200 import binding, build, workloads
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BASE = workloads.CONFIGS[1]          # 32 q / 8 kv heads, d 128, bf16, window 64


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.lib()


def cfg_with(**kw):
    return dataclasses.replace(BASE, num_layers=1, **kw)


@pytest.mark.parametrize("hq,hkv,w,lens", [
    (8, 2, 64, [1000]),                    # 256 rows, several tiles and a ragged tail
    (8, 2, 64, [128, 129, 64, 65, 700]),   # tile-aligned, one over, exactly the window, window + 1
    (7, 1, 64, [900, 300]),                # 448 rows (GQA 7): two accumulators per tile
    (16, 2, 64, [520]),                    # 512 rows (GQA 8)
    (4, 2, 16, [400, 50]),                 # 32 rows: one partly filled row block
    (8, 2, 64, [40, 1, 300]),              # sequences shorter than the window
])
def test_tc_scores_match_oracle(hq, hkv, w, lens):
    cfg = cfg_with(num_q_heads=hq, num_kv_heads=hkv, window=w)
    lay = workloads.make_layer(cfg, 0, seq_lens=lens)
    p = binding.params_for(cfg, lay)
    q, k, ss, sl = [t.to(DEV) for t in (lay.q_win, lay.k, lay.seq_start, lay.seq_len)]
    total = lay.total_tokens
    ws = torch.empty(binding.refree_workspace_size(p, total), dtype=torch.uint8, device=DEV)
    scores = torch.full((hkv, total), float("nan"), device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.refree_score(p, q, k, ss, sl, total, scores, ws, st)
    torch.cuda.synchronize()
    assert st.item() == 0
    want = orc.score(parity.oracle_params(p), lay.q_win, lay.k, lay.seq_start, lay.seq_len)
    worst = parity.check_scores(scores, want)
    assert worst < 1e-4          # fp32 softmax of exact bf16 products: far inside the 1e-3 bar


@pytest.mark.parametrize("layout", ["head_major", "token_major"])
@pytest.mark.parametrize("rank_mode", [binding.RANK_POSITION, binding.RANK_SCORE])
def test_tc_fused_pass_both_layouts(layout, rank_mode):
    cfg = cfg_with(num_q_heads=8, num_kv_heads=2)
    lay = workloads.make_layer(cfg, 3, layout=layout, seq_lens=[2000, 333])
    parity.run_fused_and_check(cfg, lay, rank_mode=rank_mode)


def test_tc_padded_batch_layout_with_sequence_stride():
    """[B, Hkv, n_max, d] cache with per-sequence lengths below n_max: the token
    axis restarts at 0 for every sequence and a sequence stride is in play."""
    cfg = cfg_with(num_q_heads=8, num_kv_heads=2)
    lens, n_max = [300, 517, 64], 640
    lay = workloads.make_layer(cfg, 0, seq_lens=lens)
    B, Hkv, d = len(lens), 2, 128
    kp = torch.zeros(B, Hkv, n_max, d, dtype=torch.bfloat16)
    vp = torch.zeros(B, Hkv, n_max, d, dtype=torch.bfloat16)
    for s, n in enumerate(lens):
        a = int(lay.seq_start[s])
        kp[s, :, :n] = lay.k[:, a:a + n]
        vp[s, :, :n] = lay.v[:, a:a + n]
    strides = (Hkv * n_max * d, d, n_max * d)
    p = binding.params_for(cfg, lay, kv_tokens=n_max, k_strides=strides, v_strides=strides)
    zero = torch.zeros(B, dtype=torch.int32)
    total = sum(lens)
    res = binding.compress_layer(p, lay.q_win.to(DEV), kp.to(DEV), vp.to(DEV), zero.to(DEV), lay.seq_len.to(DEV), total)
    torch.cuda.synchronize()
    assert res.device_status.item() == 0
    ref = orc.compress_layer(parity.oracle_params(p), lay.q_win, kp, vp, zero, lay.seq_len)
    parity.check_scores(res.scores, ref.scores)
    parity.check_selection(p, lens, res.lengths, res.offsets, res.kept_idx, ref.sel, ref.scores32)
    rows = int(ref.sel.offsets[-1])
    if torch.equal(res.lengths.cpu().reshape(-1), torch.from_numpy(ref.sel.lengths.reshape(-1))):
        assert torch.equal(parity.bits(res.k_out[:rows].cpu()), parity.bits(ref.k_out))
        assert torch.equal(parity.bits(res.v_out[:rows].cpu()), parity.bits(ref.v_out))


def test_tc_large_logits_do_not_overflow():
    """Keys scaled so that logits reach the hundreds: the running reference of
    pass 1 must be refreshed when a later tile dwarfs the first one."""
    cfg = cfg_with(num_q_heads=8, num_kv_heads=2)
    lay = workloads.make_layer(cfg, 1, seq_lens=[1500])
    lay.k[:, 700:710] *= 40.0          # a few late, very loud keys
    p = binding.params_for(cfg, lay)
    q, k, ss, sl = [t.to(DEV) for t in (lay.q_win, lay.k, lay.seq_start, lay.seq_len)]
    ws = torch.empty(binding.refree_workspace_size(p, 1500), dtype=torch.uint8, device=DEV)
    scores = torch.empty(2, 1500, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.refree_score(p, q, k, ss, sl, 1500, scores, ws, st)
    torch.cuda.synchronize()
    assert st.item() == 0
    want = orc.score(parity.oracle_params(p), lay.q_win, lay.k, lay.seq_start, lay.seq_len)
    parity.check_scores(scores, want)


@pytest.mark.parametrize("hq,hkv,w,n", [(8, 2, 16, 40_000), (8, 2, 64, 30_001), (14, 2, 64, 21_000), (8, 1, 64, 60_100)])
def test_tc_logits_that_outgrow_the_reference_of_a_run(hq, hkv, w, n):
    """A row's sum over a CTA's tiles is taken against the largest logit of its first tile; keys that are far louder in
    later tiles of the run take it out of fp32's range, and the reference is renewed.  (Enough tiles that a CTA has several
    of them; 1, 2 and 4 row blocks.)"""
    cfg = cfg_with(num_q_heads=hq, num_kv_heads=hkv, window=w)
    lay = workloads.make_layer(cfg, 1, seq_lens=[n])
    for g in range(hkv):
        loud = torch.arange(5 + 300 * 128 * g // 7, n - 200, 128 * 7)
        lay.k[g, loud] *= 48.0
    p = binding.params_for(cfg, lay)
    q, k, ss, sl = [t.to(DEV) for t in (lay.q_win, lay.k, lay.seq_start, lay.seq_len)]
    ws = torch.empty(binding.refree_workspace_size(p, n), dtype=torch.uint8, device=DEV)
    scores = torch.full((hkv, n), float("nan"), device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.refree_score(p, q, k, ss, sl, n, scores, ws, st)
    torch.cuda.synchronize()
    assert st.item() == 0
    want = orc.score(parity.oracle_params(p), lay.q_win, lay.k, lay.seq_start, lay.seq_len)
    parity.check_scores(scores, want)


@pytest.mark.parametrize("hq,hkv,w", [(2, 2, 2), (16, 16, 16), (12, 4, 10), (5, 1, 6)])
def test_tc_few_query_rows_are_padded(hq, hkv, w):
    cfg = cfg_with(num_q_heads=hq, num_kv_heads=hkv, window=w)
    lay = workloads.make_layer(cfg, 2, seq_lens=[700, 3, 129])
    parity.run_fused_and_check(cfg, lay)


@pytest.mark.parametrize("hq,hkv,w,lens,layers", [(32, 8, 64, [16384], 6), (28, 4, 64, [9877, 4096, 640], 4), (8, 2, 16, [2000, 77], 11),
                                                  (48, 4, 32, [5000], 5)])
@pytest.mark.parametrize("small_workspace", [False, True])
@pytest.mark.parametrize("rank_mode", [0, 1])
def test_run_of_layers_scores_a_layer_as_alone(hq, hkv, w, lens, layers, small_workspace, rank_mode):
    """A layer's scores are the same bits whatever shares its launch (a budget on a near-tie would else depend on the length
    of the run and on the workspace).  A run does not return scores; those of its last layers are still in the workspace."""
    d, total = 128, sum(lens)
    gen = torch.Generator(device=DEV).manual_seed(11)
    mu = torch.randn(layers, 1, hkv, 1, 1, d, generator=gen, device=DEV)
    q = torch.randn(layers, len(lens), hkv, hq // hkv, w, d, generator=gen, device=DEV)
    q = list(((q + mu) / math.sqrt(2)).view(layers, len(lens), hq, w, d).to(torch.bfloat16))
    k = list(torch.randn(layers, hkv, total, d, generator=gen, device=DEV).to(torch.bfloat16))
    sl = torch.tensor(lens, dtype=torch.int32, device=DEV)
    ss = torch.tensor([sum(lens[:i]) for i in range(len(lens))], dtype=torch.int32, device=DEV)
    p = binding.Params(num_seqs=len(lens), num_q_heads=hq, num_kv_heads=hkv, head_dim=d, window=w, kv_tokens=total,
                       rank_mode=rank_mode, k_strides=(0, d, total * d), v_strides=(0, d, total * d))
    ko, vo = [list(torch.empty(layers, hkv * total, d, dtype=torch.bfloat16, device=DEV)) for _ in range(2)]
    lengths = list(torch.zeros(layers, len(lens) * hkv, dtype=torch.int32, device=DEV))
    off = list(torch.zeros(layers, len(lens) * hkv + 1, dtype=torch.int64, device=DEV))
    size = 2 * binding.refree_workspace_size(p, total) if small_workspace else binding.refree_layers_workspace_size(p, total)
    ws = torch.zeros(size // 4, dtype=torch.int32, device=DEV)
    binding.refree_compress_layers(p, binding.LayerPointers(q, k, k, ko, vo, lengths, off), ss, sl, total, hkv * total, ws)
    scores = torch.zeros(hkv, total, dtype=torch.float32, device=DEV)
    ws1 = torch.empty(binding.refree_workspace_size(p, total), dtype=torch.uint8, device=DEV)
    binding.refree_score(p, q[-1], k[-1], ss, sl, total, scores, ws1)
    torch.cuda.synchronize()
    want = parity.bits(scores).reshape(-1)
    key = want[want.numel() // 3]                      # a value from the middle says where the array may lie
    at = [int(i) - want.numel() // 3 for i in (ws == key).nonzero()]
    assert any(0 <= i <= ws.numel() - want.numel() and torch.equal(ws[i:i + want.numel()], want) for i in at)


@pytest.mark.parametrize("loud", [45.75, 46.0, 55.75, 90.0])
def test_tc_row_sums_far_above_the_reference_stay_finite(loud):
    """One long unit over every SM, each range of it quiet in its first two tiles, from which a row's reference comes, and
    loud behind them: tile sums of 2^99.4 and 2^99.9 (just inside the limit), 2^119.8 and beyond fp32, added up over some
    hundred ranges."""
    n, w = 60_100, 64
    p = binding.Params(num_seqs=1, num_q_heads=4, num_kv_heads=1, head_dim=128, window=w, kv_tokens=n,
                       k_strides=(0, 128, n * 128), v_strides=(0, 128, n * 128))
    q, k = torch.zeros(1, 4, w, 128, dtype=torch.bfloat16), torch.zeros(1, n, 128, dtype=torch.bfloat16)
    q[..., 0] = 16.0
    tiles, ctas = -(-n // 128), torch.cuda.get_device_properties(0).multi_processor_count
    begins = [-(-c * tiles // ctas) for c in range(ctas + 1)]
    for b, e in zip(begins, begins[1:]):
        k[0, 128 * (b + 2):128 * e, 0] = loud
    sl, ss = torch.tensor([n], dtype=torch.int32), torch.zeros(1, dtype=torch.int32)
    ws = torch.empty(binding.refree_workspace_size(p, n), dtype=torch.uint8, device=DEV)
    scores = torch.full((1, n), float("nan"), device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.refree_score(p, q.to(DEV), k.to(DEV), ss.to(DEV), sl.to(DEV), n, scores, ws, st)
    torch.cuda.synchronize()
    assert st.item() == 0
    parity.check_scores(scores, orc.score(parity.oracle_params(p), q, k, ss, sl))
