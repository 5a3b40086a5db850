"""The natively marshalled calls: on tensors that are not what a call takes they stand aside for the Python checks, and on the
GPU both ways of marshalling give the same results and the same errors."""
import pytest
import torch

from paper_2404_19124_b200 import build, synth
from helpers import small_cfg, weights_to_cuda


@pytest.fixture(scope="module")
def B():
    build.build()
    from paper_2404_19124_b200 import binding
    return binding


def test_anything_unusual_is_left_to_the_python_checks(B):
    if B._pycall is None:
        pytest.skip("built without the interpreter's headers")
    i32 = torch.zeros(2, 3, 1, dtype=torch.int32)
    assert B._pycall.verify(None, 1, 2, 3, 4, 5, None, False) is None
    assert B._pycall.verify(i32, i32, i32, i32, i32, i32, None, False) is None          # not on a GPU
    assert B._pycall.verify(i32) is None
    assert B._pycall.next_ctx(i32, i32, i32, i32, None, None) is None
    assert B._pycall.draft(None, 3, 8, i32, i32, (1, 1, 1), 1, i32, i32, i32, None) is None
    assert B._pycall.draft(1, 3, 8, i32, i32, (1, 1), 1, i32, i32, i32, None) is None
    with pytest.raises(ValueError, match="cand_tok"):
        B.spec_verify(i32, torch.zeros(2, 3, 2, 8), workspace=i32)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,early", [(torch.bfloat16, False), (torch.bfloat16, True), (torch.float32, False)])
def test_both_ways_of_marshalling_agree(B, monkeypatch, dtype, early):
    cfg = small_cfg(d_base=64, d_inner=64, V=512, topk=(3, 2), K=4, B=3, seed=1)
    h = B.spec_create(weights_to_cuda(synth.make_weights(cfg)))
    ctx, tok = synth.make_draft_inputs(cfg, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(1)
    state = torch.randn((cfg.B, cfg.K, cfg.n + 1, cfg.d_base), generator=g, device="cuda").to(torch.bfloat16)
    out = []
    for native in (True, False):
        if not native:
            monkeypatch.setattr(B, "_pycall", None)
        for stream in (None, torch.cuda.Stream()):
            torch.cuda.synchronize()
            ct, lp, ws = B.spec_draft(h, ctx, tok, cfg.topk, cfg.K, stream=stream)
            torch.cuda.synchronize()
            cand, logp = torch.full_like(ct, -1), torch.full_like(lp, 1.0)
            for topk in (cfg.topk, list(cfg.topk)):
                B.spec_draft(h, ctx, tok, topk, cfg.K, cand_tok=cand, cand_logp=logp, workspace=ws, stream=stream)
            logits = synth.make_base_logits(cfg, ct, device="cuda", dtype=dtype)
            res = [torch.full((cfg.B,), -1, dtype=torch.int32, device="cuda") for _ in range(3)]
            torch.cuda.synchronize()
            _, _, _, vws = B.spec_verify(cand, logits, early_exit=early, stream=stream)
            B.spec_verify(cand, logits, *res, workspace=vws, early_exit=early, stream=stream)
            torch.cuda.synchronize()
            new = torch.zeros_like(ctx)
            B.spec_next_ctx(state, res[1], res[0], ctx_state=new, err_workspace=vws, stream=stream)
            torch.cuda.synchronize()
            assert torch.equal(cand, ct) and torch.equal(logp, lp)
            out.append([ct, lp, *res, new])
            with pytest.raises(B.SpecError):
                B.spec_verify(cand, logits, *res, workspace=vws[:256], early_exit=early, stream=stream)
            with pytest.raises(ValueError, match="next_tok"):
                B.spec_verify(cand, logits, res[0], res[1], res[2][:1], workspace=vws)
            with pytest.raises(B.SpecError):
                B.spec_draft(h, ctx, tok, (3, 2, 1), cfg.K, cand_tok=cand, cand_logp=logp, workspace=ws)
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert torch.equal(a, b)
    B.spec_destroy(h)
