"""Sizes at which the short-call kernels, the score ranking, the single-row stream and the host pipeline can go wrong: edges
of tiles and row chunks, spreads of the scores, layers that share a warp, threads that share the pipelines."""
import dataclasses
import math
import threading
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2502_16886_b200 import binding, build, workloads
from tests import parity

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    binding.lib()


def cfg_like(**kw):
    return dataclasses.replace(workloads.CONFIGS[0], **kw)


@pytest.mark.parametrize("dtype,d,hq,hkv,w,lens", [
    ("fp32", 64, 4, 2, 16, [1]), ("fp32", 64, 3, 3, 5, [64, 0, 63, 65, 1]), ("bf16", 64, 6, 2, 11, [513 - 130, 64, 65]),
    ("fp32", 128, 4, 4, 33, [512]), ("fp32", 128, 16, 4, 16, [200, 64, 0, 65, 183]), ("fp32", 64, 8, 2, 16, [513]),
    ("fp32", 64, 2, 2, 65, [300]), ("bf16", 64, 2, 2, 17, [449]), ("bf16", 64, 34, 2, 1, [70, 90])])
def test_short_units_from_keys_to_budgets(dtype, d, hq, hkv, w, lens):
    """Row counts around the chunks (16, 32, 64) and one more than the most, one position, empty sequences, fewer tiles than
    blocks, the longest call and one more position."""
    cfg = cfg_like(num_q_heads=hq, num_kv_heads=hkv, head_dim=d, dtype=dtype, window=w)
    lay = workloads.make_layer(cfg, 0, seq_lens=lens)
    for rank_mode, scope in ((0, 0), (0, 1), (1, 0)):
        parity.run_fused_and_check(cfg, lay, rank_mode=rank_mode, scope=scope, threshold=0.05)


@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("fp32", 128), ("bf16", 64)])
@pytest.mark.parametrize("lens", [[544], [577, 1], [33, 640, 0]])
@pytest.mark.parametrize("extent", ["known", 0, 1 << 40])
def test_rows_and_list_whatever_extent_the_caller_gives(dtype, d, lens, extent):
    """The copy's grid follows the cache's extent: rows that end with a block's pieces and one more, an extent that is not given
    and one far beyond."""
    cfg = cfg_like(num_q_heads=4, num_kv_heads=2, head_dim=d, dtype=dtype, window=24)
    lay = workloads.make_layer(cfg, 0, seq_lens=lens)
    parity.run_fused_and_check(cfg, lay, rank_mode=0, threshold=0.05, **({} if extent == "known" else {"kv_tokens": extent}))


@pytest.mark.parametrize("dtype,d,hq,hkv,w", [("fp32", 64, 8, 2, 16), ("fp32", 128, 3, 1, 11), ("bf16", 64, 4, 4, 1), ("bf16", 64, 2, 1, 32)])
@pytest.mark.parametrize("layout", ["head_major", "token_major"])
@pytest.mark.parametrize("q_offset", [0, 1])
def test_short_units_score_as_in_a_longer_call(dtype, d, hq, hkv, w, layout, q_offset):
    """A short call takes the cluster per unit, one with a long sequence more the three kernels: same bits for the sequences
    that they share, whatever the order of the cache and wherever the queries start."""
    cfg = cfg_like(num_q_heads=hq, num_kv_heads=hkv, head_dim=d, dtype=dtype, window=w)
    lens = [65, 1, 0, 127, 300, 600]
    lay = workloads.make_layer(cfg, 0, seq_lens=lens, layout=layout)
    if w == 1 and hq // hkv <= 16:
        cfg = dataclasses.replace(cfg, window=2)                         # (a single row has a path of its own)
        lay = workloads.make_layer(cfg, 0, seq_lens=lens, layout=layout)
    p = binding.params_for(cfg, lay)
    buf = torch.empty(lay.q_win.numel() + 8, dtype=lay.q_win.dtype, device=DEV)
    q = buf[q_offset:q_offset + lay.q_win.numel()].view(lay.q_win.shape)
    q.copy_(lay.q_win)
    k, start, length = [t.to(DEV) for t in (lay.k, lay.seq_start, lay.seq_len)]
    got = []
    for seqs in (6, 5):
        p.num_seqs, total = seqs, sum(lens[:seqs])
        scores = torch.full((hkv, total), float("nan"), device=DEV)
        ws = torch.empty(binding.refree_workspace_size(p, total), dtype=torch.uint8, device=DEV)
        binding.refree_score(p, q[:seqs], k, start[:seqs], length[:seqs], total, scores, ws)
        got.append(scores)
    torch.cuda.synchronize()
    assert torch.equal(got[0][:, :sum(lens[:5])], got[1])


@pytest.mark.parametrize("hq,hkv,dtype,d", [(8, 8, "bf16", 128), (4, 2, "bf16", 64), (28, 4, "bf16", 128), (8, 8, "fp32", 64)])
@pytest.mark.parametrize("rows", [[9000, 100, 3000, 1, 700, 2500, 0, 1200, 40, 500, 4000, 900, 300], [3000, 40], [6000, 1500, 700]])
def test_decode_of_lengths_that_differ(hq, hkv, dtype, d, rows):
    """Units that a plan cuts in proportion to their rows: more units than half the SMs, a few, empty ones; two heads of a
    sequence that keep different numbers of rows."""
    from tests.test_decode_gpu import check_against_oracle
    lengths = [max(0, r - 37 * g) for r in rows for g in range(hkv)]
    check_against_oracle(len(rows), hq, hkv, d, dtype, lengths, seed=41, max_rows=max(rows), kv_tokens=sum(rows))


@pytest.mark.parametrize("dtype,d,rows,launches", [("fp32", 128, [1200, 800, 600, 400, 300, 200], 1), ("fp32", 64, [700, 1025, 411, 96, 1500, 333], 1),
                                                   ("fp32", 64, [3000, 500, 400, 300, 200, 100], 2)])
def test_decode_of_units_that_need_no_cut(dtype, d, rows, launches):
    """More units than half the SMs: each is left whole, and its rows in one launch, unless one is far longer than the rest."""
    from tests.test_decode_gpu import check_against_oracle
    before = binding.lib().refree_kernel_launch_count()
    check_against_oracle(len(rows), 16, 16, d, dtype, [r for r in rows for _ in range(16)], seed=43, max_rows=max(rows), kv_tokens=sum(rows))
    assert binding.lib().refree_kernel_launch_count() - before == launches


@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (16, 1, 128), (12, 1, 64)])
@pytest.mark.parametrize("lens", [[8193], [20_000, 255, 0, 257], [300] * 40])
def test_single_query_row_beyond_the_short_calls(hq, hkv, d, lens):
    cfg = cfg_like(num_q_heads=hq, num_kv_heads=hkv, head_dim=d, dtype="bf16", window=1)
    lay = workloads.make_layer(cfg, 1, seq_lens=lens)
    parity.run_fused_and_check(cfg, lay, rank_mode=0)


@pytest.mark.parametrize("hq,hkv,d,lens", [(16, 4, 128, [37_000, 200, 1]), (10, 2, 64, [76_000]), (24, 2, 128, [38_100, 90]), (32, 2, 64, [9000])])
def test_single_query_row_of_more_chunks_than_blocks(hq, hkv, d, lens):
    """A chunk to a block, several chunks of a unit and of two units to a block, with up to 4, 8 and 16 heads a group."""
    cfg = cfg_like(num_q_heads=hq, num_kv_heads=hkv, head_dim=d, dtype="bf16", window=1)
    lay = workloads.make_layer(cfg, 1, seq_lens=lens)
    parity.run_fused_and_check(cfg, lay, rank_mode=0)


@pytest.mark.parametrize("group,w", [(1, 257), (4, 65), (4, 75), (3, 110), (2, 192), (4, 100), (7, 64), (1, 449), (7, 73), (2, 17), (5, 13), (1, 130)])
def test_query_rows_that_do_not_fill_their_products(group, w):
    """Row blocks of 128 and column products of 256 with rows to spare: warps of the row pass without rows, chunks of the column
    pass without rows, a second product that is padded; a tile before the window, tiles inside it, one position."""
    cfg = cfg_like(num_q_heads=2 * group, num_kv_heads=2, head_dim=128, dtype="bf16", window=w)
    lay = workloads.make_layer(cfg, 2, seq_lens=[700, 129, 1])
    parity.run_fused_and_check(cfg, lay, rank_mode=0, threshold=0.05)


def _exact_rule(a, lead, w_eff, threshold):
    """Budget and kept positions of one unit ranked by score, by the documented integers (squares in fixed point, C_n in
    [2^60, 2^61))."""
    n = len(a)
    sq = [Fraction(float(x)) ** 2 for x in a]
    scale = Fraction(2) ** (60 - math.floor(math.log2(float(sum(sq)))))
    sq = [math.floor(x * scale) for x in sq]
    prot = list(range(lead)) + list(range(n - w_eff, n))
    order = prot + sorted(range(lead, n - w_eff), key=lambda i: (-float(a[i]), i))
    total = sum(sq)
    t = float(np.float32(threshold))
    c_min = total - (math.ceil(float(total) * (t * (2.0 - t))) - 1)
    c, j = 0, n
    for r, i in enumerate(order):
        c += sq[i]
        if c >= c_min:
            j = r + 1
            break
    b = max(j, len(prot))
    return b, sorted(order[:b])


@pytest.mark.parametrize("n", [700, 5000, 20_000])
@pytest.mark.parametrize("binades,threshold", [(0, 0.01), (8, 0.1), (40, 0.01), (29, 1e-18), (30, 1e-18), (30, 1e-17)])
def test_score_ranking_whatever_the_spread_of_the_scores(n, binades, threshold):
    """Scores spread evenly over 2^-binades .. 1; with a tiny threshold one large score is protected and the sum crosses
    among scores far below it, beyond the binades that the first level of the descent tells apart."""
    gen = torch.Generator().manual_seed(n + binades)
    if threshold > 1e-6:
        scores = torch.exp2(-binades * torch.rand(1, n, generator=gen)) * (1 + torch.rand(1, n, generator=gen)) / 2
    else:
        scores = 2.0 ** -binades * (1 + torch.rand(1, n, generator=gen))
        scores[0, 0] = 1.25
    p = binding.Params(num_seqs=1, num_q_heads=2, num_kv_heads=1, head_dim=64, window=4, sink=2, threshold=threshold,
                       rank_mode=binding.RANK_SCORE, dtype=binding.DTYPE_F32, kv_tokens=n, k_strides=(0, 64, n * 64),
                       v_strides=(0, 64, n * 64))
    lengths = torch.zeros(1, dtype=torch.int32, device=DEV)
    offsets = torch.zeros(2, dtype=torch.int64, device=DEV)
    kept = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    ws = torch.empty(binding.refree_workspace_size(p, n), dtype=torch.uint8, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.refree_select_budget(p, scores.to(DEV), torch.tensor([n], dtype=torch.int32, device=DEV), n, lengths, offsets, kept, n, ws, st)
    torch.cuda.synchronize()
    want_b, want = _exact_rule(scores[0].tolist(), 2, 4, threshold)
    assert int(st.item()) == 0 and int(lengths.item()) == want_b
    assert kept[:want_b].cpu().tolist() == want


@pytest.mark.parametrize("lens", [[2047], [2048], [4096], [4097], [16385], [1024, 3073], [5120, 1, 2049], [9000, 0, 1023]])
@pytest.mark.parametrize("levels", [3, 1 << 20])
def test_index_list_of_units_without_counts(lens, levels):
    """Ranked per head the selection leaves counts where the workspace has room for them, in the built-in scratch there is none:
    the same list, with ties at every step of the scores and without."""
    n, units = sum(lens), 2 * len(lens)
    scores = (torch.randint(1, levels + 1, (2, n), generator=torch.Generator().manual_seed(n + levels)).float() / levels).to(DEV)
    p = binding.Params(num_seqs=len(lens), num_q_heads=2, num_kv_heads=2, head_dim=64, window=4, sink=2, threshold=0.1,
                       rank_mode=binding.RANK_SCORE, dtype=binding.DTYPE_F32, kv_tokens=n, k_strides=(0, 64, n * 64),
                       v_strides=(0, 64, n * 64))
    length = torch.tensor(lens, dtype=torch.int32, device=DEV)
    ws = torch.empty(binding.refree_workspace_size(p, n), dtype=torch.uint8, device=DEV)
    got = []
    for static in (False, True):
        out = [torch.zeros(units, dtype=torch.int32, device=DEV), torch.zeros(units + 1, dtype=torch.int64, device=DEV),
               torch.full((2 * n,), -1, dtype=torch.int32, device=DEV)]
        if static:
            binding.refree_select_budget_static(p, scores, length, n, *out, 2 * n)
        else:
            binding.refree_select_budget(p, scores, length, n, *out, 2 * n, ws)
        got.append([t.cpu() for t in out])
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("lens", [[16_384] + [100] * 9, [90] * 8 + [16_385, 3000], [66_000] + [70] * 40, [0, 65_536] + [64] * 39])
def test_score_ranking_of_a_long_unit_among_many_short_ones(lens):
    """Units that one block holds, the next longer, the longest that four hold and one beyond: three kernels share a call."""
    cfg = cfg_like(num_q_heads=2, num_kv_heads=2, head_dim=64, dtype="bf16", window=1)
    lay = workloads.make_layer(cfg, 0, seq_lens=lens)
    parity.run_fused_and_check(cfg, lay, rank_mode=1, threshold=0.1)


@pytest.mark.parametrize("lens", [[2048], [2049, 3000], [4097]])
def test_index_list_of_a_layer_ranked_across_its_heads(lens):
    cfg = cfg_like(num_q_heads=4, num_kv_heads=2, head_dim=64, dtype="fp32", window=8)
    lay = workloads.make_layer(cfg, 0, seq_lens=lens)
    parity.run_fused_and_check(cfg, lay, rank_mode=1, scope=1, threshold=0.1)


def test_score_ranking_counts_scores_that_are_not_finite():
    n = 3000
    scores = torch.rand(1, n, generator=torch.Generator().manual_seed(3)) * 1e-3
    scores[0, 1500] = float("inf")
    p = binding.Params(num_seqs=1, num_q_heads=2, num_kv_heads=1, head_dim=64, window=4, sink=2, threshold=0.01,
                       rank_mode=binding.RANK_SCORE, dtype=binding.DTYPE_F32, kv_tokens=n, k_strides=(0, 64, n * 64),
                       v_strides=(0, 64, n * 64))
    lengths, offsets = torch.zeros(1, dtype=torch.int32, device=DEV), torch.zeros(2, dtype=torch.int64, device=DEV)
    kept = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    ws = torch.empty(binding.refree_workspace_size(p, n), dtype=torch.uint8, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.refree_select_budget(p, scores.to(DEV), torch.tensor([n], dtype=torch.int32, device=DEV), n, lengths, offsets, kept, n, ws, st)
    torch.cuda.synchronize()
    b = int(lengths.item())
    assert int(st.item()) == binding.DEV_NONFINITE and 1500 in kept[:b].cpu().tolist()        # its key is the largest
    assert torch.equal(kept[:b].cpu(), kept[:b].cpu().unique()) and b < n


def _host_run(cfg, lays, p, cap, rounds, out):
    try:
        total, units = lays[0].total_tokens, p.num_seqs * p.num_kv_heads
        arena = torch.empty(binding.refree_host_pipeline_arena_size(p, total, lays[0].k.numel(), cap), dtype=torch.uint8, device=DEV)
        for _ in range(rounds):
            ko = [torch.zeros(cap, p.head_dim, dtype=lays[0].k.dtype).pin_memory() for _ in lays]
            vo = [torch.zeros_like(t).pin_memory() for t in ko]
            ln = [torch.zeros(units, dtype=torch.int32) for _ in lays]
            of = [torch.zeros(units + 1, dtype=torch.int64) for _ in lays]
            rc = binding.refree_compress_layers_host(p, [l.q_win for l in lays], [l.k for l in lays], [l.v for l in lays], lays[0].seq_start,
                                                     lays[0].seq_len, total, ko, vo, cap, ln, of, arena, check=False)
            out.append((rc, ko, vo, ln, of))
    except Exception as e:                                               # (shown by the test)
        out.append(e)


def test_host_pipelines_of_several_threads_and_after_an_error():
    """Threads take pipelines of their own; one that ended with an error serves the next call."""
    cfg = cfg_like(window=16, dtype="bf16", head_dim=128, num_q_heads=8, num_kv_heads=2)
    lays = [workloads.make_layer(cfg, l, seq_lens=[900, 1, 333]) for l in range(3)]
    p = binding.params_for(cfg, lays[0], threshold=0.05)
    cap = p.num_kv_heads * lays[0].total_tokens
    refs = [binding.compress_layer(p, *[t.to(DEV) for t in (l.q_win, l.k, l.v, l.seq_start, l.seq_len)], l.total_tokens) for l in lays]
    torch.cuda.synchronize()
    short = []
    _host_run(cfg, lays, p, 40, 1, short)
    assert short[0][0] == binding.ERR_CAPACITY
    outs = [[] for _ in range(6)]
    threads = [threading.Thread(target=_host_run, args=(cfg, lays, p, cap, 3, o)) for o in outs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for o in outs:
        assert len(o) == 3
        for rc, ko, vo, ln, of in o:
            assert rc == 0
            for ref, k, v, n, f in zip(refs, ko, vo, ln, of):
                rows = int(f[-1])
                assert torch.equal(n, ref.lengths.cpu().reshape(-1)) and torch.equal(f, ref.offsets.cpu())
                assert torch.equal(parity.bits(k[:rows]), parity.bits(ref.k_out[:rows].cpu()))
                assert torch.equal(parity.bits(v[:rows]), parity.bits(ref.v_out[:rows].cpu()))
