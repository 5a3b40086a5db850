"""The row-wise steps of a draft at the sizes where their thread counts matter: partial lists per row and leaves per
sequence below, at and above the threads of a CTA."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_19124_b200 import synth
from helpers import LOGIT_TOL, TIE_TOL, DraftChecker, kernels_launched, small_cfg, to_oracle_weights, weights_to_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2404_19124_b200 import build
    build.build()
    from paper_2404_19124_b200 import binding
    return binding


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("topk,K", [((8, 4, 5), 160), ((7, 7, 3), 100), ((8, 4, 3, 2), 64), ((8, 4, 3, 2), 192),
                                    ((8, 8, 4), 255), ((8, 8, 4), 256), ((7, 5, 8), 1), ((8, 8, 8), 1),
                                    ((8, 8, 8), 64), ((8, 8, 8), 255), ((8, 8, 8), 256), ((8, 8, 8), 257),
                                    ((8, 8, 8, 8), 5), ((8, 8, 8, 8), 256)])
def test_prune_leaves_round_the_thread_counts(B, topk, K, fp8):
    """147 to 256 leaves: more and fewer than the 160 (or 512) threads of the CTA that ranks them; more leaves: up to 256
    kept are selected, more are sorted."""
    cfg = small_cfg(d_base=48, d_inner=64, V=96, topk=topk, K=K, B=3, seed=K)
    sw = synth.make_weights(cfg)
    ow, gw = to_oracle_weights(sw), weights_to_cuda(sw)
    ctx, tok = synth.make_draft_inputs(cfg)
    h = B.spec_create(gw)
    if fp8:
        B.spec_attach_fp8_heads(h)
        B.spec_set_option(h, B.SPEC_OPT_FP8_MAX_ROWS, 4096)
    ct = torch.full((cfg.B, K, cfg.n), -1, dtype=torch.int32, device="cuda")
    lp = torch.full((cfg.B, K), 1.0, device="cuda")
    _, _, ws = B.spec_draft(h, ctx.cuda(), tok.cuda(), topk, K, cand_tok=ct, cand_logp=lp)
    assert B.spec_poll_error(ws) == 0
    lay = B.spec_draft_layout(h, cfg.B, topk, K)
    L = cfg.leaves
    leaf = ws[lay.score[cfg.n]:lay.score[cfg.n] + 4 * cfg.B * L].view(torch.float32).view(cfg.B, L)
    want = torch.sort(leaf, dim=1, descending=True, stable=True)
    assert torch.equal(lp, want.values[:, :K])
    last = ws[lay.tok[cfg.n]:lay.tok[cfg.n] + 4 * cfg.B * L].view(torch.int32).view(cfg.B, L)
    assert torch.equal(ct[:, :, -1], torch.gather(last, 1, want.indices[:, :K]))
    if not fp8 and L <= 256:
        chk = DraftChecker(ow, topk, K)
        for b in range(cfg.B):
            chk.check(synth.bf16_bits(ctx)[b], int(tok[b]), ct[b].cpu().numpy(), lp[b].cpu().numpy())
    B.spec_destroy(h)


@pytest.mark.parametrize("V", [31 * 32, 33 * 32, 256 * 32, 256 * 32 + 1])
@pytest.mark.parametrize("topk,K,rows", [((1, 1), 1, 1), ((1, 7), 5, 1), ((4, 3, 2), 16, 12), ((6, 4, 3), 72, 24), ((6, 4, 8), 100, 24),
                                         ((5, 5, 8), 100, 25)])
def test_last_merge_and_prune_of_a_sequence(B, topk, K, rows, V):
    """The last merge is one CTA per sequence or one per row; the kept leaves are the best of the scores that it leaves in the
    workspace, in order, with the tokens of their paths."""
    assert rows * topk[-1] == np.prod(topk)
    _check_last_merge(B, topk, K, V, 3)


@pytest.mark.parametrize("topk,lists,seqs", [((7,), 160, 32), ((7,), 160, 33), ((8,), 160, 1), ((3,), 160, 33), ((4,), 160, 33),
                                             ((2, 8), 96, 30), ((2, 8), 97, 30), ((3, 4, 8), 160, 4), ((5, 2, 8), 160, 5),
                                             ((4, 3, 8), 160, 13), ((3, 5, 8), 129, 3), ((8, 2, 6), 160, 3), ((8, 2, 6), 161, 3),
                                             ((6, 4, 8), 100, 25), ((6, 4, 8), 100, 24)])
def test_last_merge_on_both_sides_of_its_rule(B, topk, lists, seqs):
    """Rounds of a row, rows of a sequence and rows in all where the last merge goes from a CTA per sequence to a CTA per row."""
    _check_last_merge(B, topk, min(12, int(np.prod(topk))), 32 * lists - 5, seqs)


def _check_last_merge(B, topk, K, V, seqs):
    cfg = small_cfg(d_base=48, d_inner=64, V=V, topk=topk, K=K, B=seqs, seed=K)
    sw = synth.make_weights(cfg)
    ctx, tok = synth.make_draft_inputs(cfg)
    h = B.spec_create(weights_to_cuda(sw))
    B.spec_set_option(h, B.SPEC_OPT_HEAD_BLOCK_N, 32)
    ct, lp, ws = B.spec_draft(h, ctx.cuda(), tok.cuda(), topk, K)
    assert B.spec_poll_error(ws) == 0
    lay = B.spec_draft_layout(h, cfg.B, topk, K)
    n, L = cfg.n, cfg.leaves
    leaf = ws[lay.score[n]:lay.score[n] + 4 * cfg.B * L].view(torch.float32).view(cfg.B, L)
    want = torch.sort(leaf, dim=1, descending=True, stable=True)
    assert torch.equal(lp, want.values[:, :K])
    per = 1
    for l in range(n):
        per *= topk[l]
        t = ws[lay.tok[l + 1]:lay.tok[l + 1] + 4 * cfg.B * per].view(torch.int32).view(cfg.B, per)
        assert torch.equal(ct[:, :, l], torch.gather(t, 1, want.indices[:, :K] // (L // per)))
    chk = DraftChecker(to_oracle_weights(sw), topk, K)
    for b in range(min(3, seqs)):
        chk.check(synth.bf16_bits(ctx)[b], int(tok[b]), ct[b].cpu().numpy(), lp[b].cpu().numpy())
    B.spec_destroy(h)


@pytest.mark.parametrize("swap", [0, 128])
@pytest.mark.parametrize("k", [1, 4, 5, 8])
@pytest.mark.parametrize("V", [159 * 32, 160 * 32, 161 * 32, 320 * 32 + 1, 80000])
def test_merge_lists_round_the_thread_counts(B, V, k, swap):
    """Tiles 32 wide: 159 to 2500 partial lists per row for 160 threads (one, two, many lists per thread)."""
    rows, d = 5, 64
    cfg = small_cfg(d_base=d, d_inner=d, V=V, topk=(2, 2), seed=V % 97 + k)
    sw = synth.make_weights(cfg)
    ow, gw = to_oracle_weights(sw), weights_to_cuda(sw)
    h = B.spec_create(gw)
    if swap:
        B.spec_set_option(h, B.SPEC_OPT_HEAD_SWAP_MAX_ROWS, swap)
    else:
        B.spec_set_option(h, B.SPEC_OPT_HEAD_BLOCK_N, 32)
    g = torch.Generator().manual_seed(k)
    S = torch.randn(rows, d, generator=g).to(torch.bfloat16)
    tok, logp, ws = B.spec_head_topk(h, 0, S.cuda(), k)
    assert B.spec_poll_error(ws) == 0
    logits = oracle.stage_logits(ow, 0, S.to(torch.float32).numpy())
    lse = torch.logsumexp(torch.from_numpy(logits).double(), 1).numpy()
    got = tok.cpu().numpy()
    for r in range(rows):
        ids, _ = oracle.topk(logits[r], k)
        near = np.abs(logits[r][got[r]] - logits[r][ids])      # (a near-tie may be ordered either way)
        assert len(set(got[r].tolist())) == k and near.max() <= TIE_TOL
        assert np.abs(logp[r].cpu().numpy() - (logits[r][got[r]] - lse[r])).max() <= LOGIT_TOL
    B.spec_destroy(h)


@pytest.mark.parametrize("rows", [1, 17, 48])
@pytest.mark.parametrize("d", [2048, 4096, 2056])
def test_equal_rows_give_equal_logits_in_every_tile(B, d, rows):
    """Nodes as MMA columns, rows of 4096 and 8192 bytes: every second CTA sums its weight tiles with the halves of the K range
    in the other order.  Copies of one head row in tiles of either kind must tie exactly, lower token first."""
    V = 20000                                            # 136 rows per CTA: two tiles each
    cfg = small_cfg(d_base=64, d_inner=d, V=V, topk=(8, 2), seed=rows + d)
    sw = synth.make_weights(cfg)
    copies = [5, 130, 140, 300, 4000, 4100, 9999, V - 1]
    for c in copies[1:]:
        sw.head[0][c] = sw.head[0][copies[0]]
    h = B.spec_create(weights_to_cuda(sw))
    B.spec_set_option(h, B.SPEC_OPT_HEAD_SWAP_MAX_ROWS, 128)
    g = torch.Generator().manual_seed(rows)
    scale = 1.0 + 0.5 * torch.rand(rows, 1, generator=g)
    S = (sw.head[0][copies[0]].float()[None] * 40 * scale + 0.01 * torch.randn(rows, d, generator=g)).to(torch.bfloat16)
    tok, logp, ws = B.spec_head_topk(h, 0, S.cuda(), 8)
    assert B.spec_poll_error(ws) == 0
    assert (tok.cpu() == torch.tensor(copies, dtype=torch.int32)).all()
    assert (logp == logp[:, :1]).all()
    want = torch.log_softmax(S.double() @ sw.head[0].double().t(), 1)[:, copies[0]]
    assert (logp[:, 0].cpu().double() - want).abs().max() <= LOGIT_TOL
    B.spec_destroy(h)


@pytest.mark.parametrize("d", [2048, 2056, 4096])
@pytest.mark.parametrize("B_,topk", [(37, (4, 2)), (18, (8, 1, 2)), (149, (1, 2)), (74, (2, 1)), (75, (2, 1))])
def test_merge_and_mix_round_one_child_per_sm(B, B_, topk, d):
    """148 children and a few more or less (a level's merge and the next level's mix are one kernel up to one child per
    SM), row widths round the two thread counts."""
    _check_every_level(B, small_cfg(d_base=64, d_inner=d, V=600, topk=topk, K=int(np.prod(topk)), B=B_, seed=B_ + d))


@pytest.mark.parametrize("swap", [0, 128])
@pytest.mark.parametrize("B_,topk,V,d", [(37, (4, 1), 600, 2048), (37, (4, 1), 600, 4096), (37, (4, 1), 600, 4112),
                                         (75, (2, 1), 600, 512), (2, (4, 3, 2), 4805, 272), (1, (8, 1, 2), 19000, 1040),
                                         (17, (1, 7), 37900, 128)])
def test_e4m3_levels_with_and_without_swapped_operands(B, B_, topk, V, d, swap):
    """Both operand orders of the e4m3 head, with one and several weight tiles per CTA and short last ones; children of a
    re-scored level below, at and above one per SM and row widths round what one CTA covers."""
    _check_every_level(B, small_cfg(d_base=64, d_inner=d, V=V, topk=topk, K=int(np.prod(topk)), B=B_, seed=B_ + d),
                       e4m3=True, swap=swap)


@pytest.mark.parametrize("chain", [False, True])
@pytest.mark.parametrize("B_,topk,V,d_base,d,one", [(1, (4, 3, 2), 1024, 256, 256, True), (16, (1, 1, 1), 1000, 64, 512, True),
                                                     (17, (1, 1), 1000, 64, 512, False), (3, (5, 1, 2), 1003, 40, 264, True),
                                                     (2, (8, 8), 2047, 8, 128, True), (1, (8, 2, 8), 600, 2048, 8, True),
                                                     (2, (8,), 16, 72, 504, True), (5, (3, 1, 2), 257, 1000, 248, True),
                                                     (1, (4, 2, 2, 2), 2048, 256, 512, True), (9, (1, 1, 4), 129, 2040, 40, True),
                                                     (1, (4, 3), 3100, 64, 512, True), (1, (4, 3), 3300, 64, 512, True),
                                                     (1, (4, 3), 3322, 64, 512, False), (1, (2, 2), 1000, 64, 520, False),
                                                     (1, (2, 2), 1000, 2056, 64, False), (16, (1, 1), 100000, 64, 8, False)])
def test_small_drafts_are_one_kernel(B, B_, topk, V, d_base, d, one, chain):
    """Node counts, widths and vocabularies at the edges of what one cluster takes: 16 and 17 nodes, fewer rows than warps,
    CTAs without any vocabulary row, K ranges that end inside a group of 32, sizes on both sides of the limits, and logits of
    16 nodes that do not fit its shared memory.  Each also as the chain of kernels that an option asks for."""
    _check_every_level(B, small_cfg(d_base=d_base, d_inner=d, V=V, topk=topk, K=int(np.prod(topk)), B=B_, seed=B_ + d),
                       pair=0 if chain else None, one_kernel=one and not chain)


def _check_every_level(B, cfg, e4m3=False, swap=None, pair=None, one_kernel=None):
    """Every level is re-derived by the oracle from the GPU's parent level for the first and the last sequence; one_kernel:
    whether the draft is to be a single kernel."""
    B_, topk, K, d = cfg.B, cfg.topk, cfg.K, cfg.d_inner
    sw = synth.make_weights(cfg)
    ow, gw = to_oracle_weights(sw), weights_to_cuda(sw)
    ctx, tok = synth.make_draft_inputs(cfg)
    h = B.spec_create(gw)
    if e4m3:
        B.spec_attach_fp8_heads(h)
    if swap is not None:
        B.spec_set_option(h, B.SPEC_OPT_HEAD_SWAP_MAX_ROWS, swap)
    if pair is not None:
        B.spec_set_option(h, B.SPEC_OPT_HEAD_PAIR, pair)
    gctx, gtok = ctx.cuda(), tok.cuda()
    ct, lp, ws = B.spec_draft(h, gctx, gtok, topk, K)
    if one_kernel is not None:
        assert one_kernel == (kernels_launched(lambda: B.spec_draft(h, gctx, gtok, topk, K, ct, lp, ws)) == 1)
    assert B.spec_poll_error(ws) == 0
    lay = B.spec_draft_layout(h, B_, topk, K)
    view = lambda off, n, dt: ws[off:off + n * torch.empty((), dtype=dt).element_size()].view(dt)
    chk = DraftChecker(ow, topk, K)
    for b in (0, B_ - 1):
        st, tk, sc = [], [], []
        for l in range(cfg.n):
            N, N1 = cfg.nodes(l), cfg.nodes(l + 1)
            S = view(lay.state[l], N * d, torch.bfloat16).view(B_, N // B_, d)
            st.append(S[b].float().cpu().numpy())
            tk.append(view(lay.tok[l + 1], N1, torch.int32).view(B_, -1)[b].cpu().numpy())
            sc.append(view(lay.score[l + 1], N1, torch.float32).view(B_, -1)[b].cpu().numpy())
        chk.check(synth.bf16_bits(ctx)[b], int(tok[b]), ct[b].cpu().numpy(), lp[b].cpu().numpy(),
                  levels={"state": st, "tok": tk, "score": sc}, force_levels=True)
    B.spec_destroy(h)


@pytest.mark.parametrize("values", [1, 2, 5])
@pytest.mark.parametrize("K", [1, 100, 256])
def test_selection_among_equal_scores(B, K, values):
    """All heads zero but for the last, whose rows repeat: 512 leaves with `values` distinct scores each; equal scores are
    kept in ascending leaf order."""
    topk = (8, 8, 8)
    cfg = small_cfg(d_base=48, d_inner=64, V=96, topk=topk, K=K, B=2, seed=values)
    sw = synth.make_weights(cfg)
    for l in range(2):
        sw.head[l].zero_()
    sw.head[2][:] = sw.head[2][:1]
    if values > 1:
        sw.head[2][:4] *= 2.0
    if values > 2:
        sw.emb[2][:] = 0.0
    h = B.spec_create(weights_to_cuda(sw))
    ctx, tok = synth.make_draft_inputs(cfg)
    ct, lp, ws = B.spec_draft(h, ctx.cuda(), tok.cuda(), topk, K)
    assert B.spec_poll_error(ws) == 0
    lay = B.spec_draft_layout(h, cfg.B, topk, K)
    leaf = ws[lay.score[3]:lay.score[3] + 4 * cfg.B * 512].view(torch.float32).view(cfg.B, 512)
    last = ws[lay.tok[3]:lay.tok[3] + 4 * cfg.B * 512].view(torch.int32).view(cfg.B, 512)
    want = torch.sort(leaf, dim=1, descending=True, stable=True)
    assert torch.equal(lp, want.values[:, :K])
    assert torch.equal(ct[:, :, -1], torch.gather(last, 1, want.indices[:, :K]))
    first = ws[lay.tok[1]:lay.tok[1] + 4 * cfg.B * 8].view(torch.int32).view(cfg.B, 8)
    assert torch.equal(ct[:, :, 0], torch.gather(first, 1, want.indices[:, :K] // 64))
    B.spec_destroy(h)


@pytest.mark.parametrize("d", [264, 512, 520, 1024, 1032, 2304, 4096])
@pytest.mark.parametrize("parents", [40, 74, 75, 150])
def test_mix_of_many_rows_round_the_thread_counts(B, d, parents):
    """More nodes than SMs, with the parents' projection split (up to 128 rows) and whole; states against the oracle."""
    topk = (4, 1)
    cfg = small_cfg(d_base=64, d_inner=d, V=64, topk=topk, K=4, B=parents, seed=d)
    sw = synth.make_weights(cfg)
    ow, gw = to_oracle_weights(sw), weights_to_cuda(sw)
    ctx, tok = synth.make_draft_inputs(cfg)
    h = B.spec_create(gw)
    B.spec_set_option(h, B.SPEC_OPT_HEAD_PAIR, 0)
    _, _, ws = B.spec_draft(h, ctx.cuda(), tok.cuda(), topk, 4)
    assert B.spec_poll_error(ws) == 0
    lay = B.spec_draft_layout(h, parents, topk, 4)
    s0 = ws[lay.state[0]:lay.state[0] + 2 * parents * d].view(torch.bfloat16).view(parents, d).float().cpu().numpy()
    s1 = ws[lay.state[1]:lay.state[1] + 8 * parents * d].view(torch.bfloat16).view(4 * parents, d).float().cpu().numpy()
    t1 = ws[lay.tok[1]:lay.tok[1] + 16 * parents].view(torch.int32).cpu().numpy()
    for r in (0, 1, 2 * parents + 1, 4 * parents - 1):
        want = oracle.stage_state(ow, 1, s0[r // 4], int(t1[r]))
        assert np.allclose(s1[r], want, rtol=0.008, atol=2e-4)
    B.spec_destroy(h)


@pytest.mark.parametrize("k,d", [(2, 1032), (2, 2048), (2, 2056), (2, 4096), (4, 1032), (4, 2048)])
def test_states_are_the_same_bits_in_every_kernel(B, k, d):
    """148 children have one CTA each; with one parent more they are computed one CTA per parent (two children per row) or by a
    kernel of their own (four).  The children that both batches have get the same states, so that a sequence's result does not
    hang on the batch it is in."""
    topk, n0 = (k, 1), 148 // k
    cfg = small_cfg(d_base=64, d_inner=d, V=600, topk=topk, K=k, B=n0 + 1, seed=d)
    sw = synth.make_weights(cfg)
    ctx, tok = synth.make_draft_inputs(cfg)
    h = B.spec_create(weights_to_cuda(sw))
    got = []
    for n in (n0, n0 + 1):
        ct, lp, ws = B.spec_draft(h, ctx[:n].cuda(), tok[:n].cuda(), topk, k)
        assert B.spec_poll_error(ws) == 0
        lay = B.spec_draft_layout(h, n, topk, k)
        got.append([ws[lay.state[l]:lay.state[l] + 2 * rows * d].view(torch.int16) for l, rows in ((0, n0), (1, 148))] +
                   [ws[lay.tok[1]:lay.tok[1] + 4 * 148].view(torch.int32)])
    for a, b in zip(*got):
        assert torch.equal(a, b)
    B.spec_destroy(h)


@pytest.mark.parametrize("k", [1, 2])
@pytest.mark.parametrize("d", [264, 1032, 2048, 2056, 3080, 4096])
def test_states_are_the_same_bits_above_and_below_one_parent_per_sm(B, k, d):
    """148 parents of one or two children: one kernel finds and computes these; 150 parents: the merge and the mix are kernels of
    their own.  The sequences that both batches have get the same states."""
    topk, n0 = (2, k, 1), 74
    cfg = small_cfg(d_base=64, d_inner=d, V=600, topk=topk, K=2 * k, B=n0 + 1, seed=d)
    sw = synth.make_weights(cfg)
    ctx, tok = synth.make_draft_inputs(cfg)
    h = B.spec_create(weights_to_cuda(sw))
    got = []
    for n in (n0, n0 + 1):
        _, _, ws = B.spec_draft(h, ctx[:n].cuda(), tok[:n].cuda(), topk, cfg.K)
        assert B.spec_poll_error(ws) == 0
        lay = B.spec_draft_layout(h, n, topk, cfg.K)
        rows = [n0, 2 * n0, 2 * k * n0]
        got.append([ws[lay.state[l]:lay.state[l] + 2 * rows[l] * d].view(torch.int16) for l in range(3)] +
                   [ws[lay.tok[l]:lay.tok[l] + 4 * rows[l]].view(torch.int32) for l in (1, 2)])
    for a, b in zip(*got):
        assert torch.equal(a, b)
    B.spec_destroy(h)


@pytest.mark.parametrize("d,what", [(256, "ln_gamma"), (256, "ln_beta"), (512, "ln_gamma"), (40, "ln_beta"), (256, "proj"), (256, "head")])
def test_a_small_draft_reads_its_weights_in_stream_order(B, d, what):
    """spec_next_ctx, whose kernel lets its dependents start at once and waits behind a long verification itself, writes into
    the weights of the draft that follows it."""
    cfg = small_cfg(d_base=256, d_inner=d, V=600, topk=(3, 2), K=6, B=1, seed=d)
    gw = weights_to_cuda(synth.make_weights(cfg))
    ctx, tok = (t.cuda() for t in synth.make_draft_inputs(cfg))
    h = B.spec_create(gw)
    target = getattr(gw, what)[0].view(torch.bfloat16).reshape(1, -1)
    old = target.clone()
    new = (getattr(gw, what)[0] * -0.75).view(torch.bfloat16).reshape(1, -1)
    state = new.view(1, 1, 1, -1).expand(1, 1, 2, -1).contiguous()
    zero = torch.zeros(1, dtype=torch.int32, device="cuda")
    logits = torch.zeros((16, 8, 4, 128256), dtype=torch.bfloat16, device="cuda")
    cand = torch.zeros((16, 8, 3), dtype=torch.int32, device="cuda")
    res = [torch.empty(16, dtype=torch.int32, device="cuda") for _ in range(3)]
    vws = B.spec_verify(cand, logits)[3]
    ct, lp, ws = B.spec_draft(h, ctx, tok, cfg.topk, cfg.K)
    before = lp.clone()
    for _ in range(5):
        target.copy_(old)
        torch.cuda.synchronize()
        B.spec_verify(cand, logits, *res, workspace=vws)
        B.spec_next_ctx(state, zero, zero, ctx_state=target)
        B.spec_draft(h, ctx, tok, cfg.topk, cfg.K, cand_tok=ct, cand_logp=lp, workspace=ws)
        torch.cuda.synchronize()
        got = ct.clone(), lp.clone()
        B.spec_draft(h, ctx, tok, cfg.topk, cfg.K, cand_tok=ct, cand_logp=lp, workspace=ws)
        torch.cuda.synchronize()
        assert torch.equal(got[0], ct) and torch.equal(got[1], lp) and not torch.equal(lp, before)
    B.spec_destroy(h)


@pytest.mark.parametrize("e4m3", [False, True])
def test_weights_rewritten_by_an_ordinary_kernel_are_seen(B, e4m3):
    """Weights, or the e4m3 copies of heads, rewritten on the stream by kernels that do not let their dependents start early,
    behind a long verification and directly before the draft."""
    cfg = small_cfg(d_base=2048, d_inner=2048, V=2048, topk=(4, 2), K=8, B=4, seed=9)
    gw = weights_to_cuda(synth.make_weights(cfg))
    ctx, tok = (t.cuda() for t in synth.make_draft_inputs(cfg))
    h = B.spec_create(gw)
    if e4m3:
        B.spec_attach_fp8_heads(h)
    logits = torch.zeros((16, 8, 4, 128256), dtype=torch.bfloat16, device="cuda")
    cand = torch.zeros((16, 8, 3), dtype=torch.int32, device="cuda")
    res = [torch.empty(16, dtype=torch.int32, device="cuda") for _ in range(3)]
    vws = B.spec_verify(cand, logits)[3]
    ct, lp, ws = B.spec_draft(h, ctx, tok, cfg.topk, cfg.K)
    for i in range(10):
        new = gw.proj[0] * -1.0
        torch.cuda.synchronize()
        before = lp.clone()
        B.spec_verify(cand, logits, *res, workspace=vws)
        if e4m3:
            for l in (1, 0):
                gw.head[l].mul_(-1.0)
                q, scale = h._fp8[l]
                assert B._lib.spec_quantize_head(h.ptr, l, q.data_ptr(), scale.data_ptr(), B._stream_ptr(None)) == B.SPEC_OK
        else:
            gw.proj[0].copy_(new)
        B.spec_draft(h, ctx, tok, cfg.topk, cfg.K, cand_tok=ct, cand_logp=lp, workspace=ws)
        torch.cuda.synchronize()
        got = ct.clone(), lp.clone()
        B.spec_draft(h, ctx, tok, cfg.topk, cfg.K, cand_tok=ct, cand_logp=lp, workspace=ws)
        torch.cuda.synchronize()
        assert torch.equal(got[0], ct) and torch.equal(got[1], lp) and not torch.equal(lp, before)
    B.spec_destroy(h)
