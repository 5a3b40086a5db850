"""The natively marshalled calls: on tensors that are not what a call takes they stand aside for the Python checks, and on the
GPU both ways of marshalling give the same results and the same errors.  The module itself: named for one interpreter, never
older than its source, and not needed."""
import os
import shutil
import sys
import sysconfig

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


def _private_tree(tmp_path, monkeypatch):
    """The build of the module alone, in a package directory of its own."""
    pkg = tmp_path / "pkg"
    pkg.mkdir()
    monkeypatch.setattr(build, "_PKG", str(pkg))
    monkeypatch.setattr(build, "PYCALL_PATH", str(pkg / os.path.basename(build.PYCALL_PATH)))
    return pkg


def test_the_module_is_named_for_this_interpreter(tmp_path, monkeypatch):
    assert sys.implementation.cache_tag in os.path.basename(build.PYCALL_PATH)
    assert build.PYCALL_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    pkg = _private_tree(tmp_path, monkeypatch)
    (pkg / "_pycall.so").write_bytes(b"of another interpreter")
    build._build_pycall(False)
    assert not (pkg / "_pycall.so").exists()


@pytest.mark.parametrize("missing", ["headers", "compiler", "working compiler"])
def test_a_module_that_cannot_be_built_is_left_out(tmp_path, monkeypatch, missing):
    pkg = _private_tree(tmp_path, monkeypatch)
    stale = pkg / os.path.basename(build.PYCALL_PATH)
    stale.write_bytes(b"of an older source")
    os.utime(stale, (1, 1))
    if missing == "headers":
        monkeypatch.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
        build._build_pycall(False)
    else:
        monkeypatch.setenv("CC", str(tmp_path / "none") if missing == "compiler" else shutil.which("false"))
        with pytest.warns(UserWarning, match="marshalled in Python"):
            build._build_pycall(False)
    assert os.listdir(pkg) == []


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,early", [(torch.bfloat16, False), (torch.bfloat16, True), (torch.float32, False)])
def test_both_ways_of_marshalling_agree(B, monkeypatch, dtype, early):
    if B._pycall is None:
        pytest.skip("built without the interpreter's headers")
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
            if native:                                       # the module itself answered, it did not stand aside
                args = (h._h.value, h.n_heads, h.d_base, ctx, tok, cfg.topk, cfg.K, cand, logp, ws, stream)
                assert B._pycall.draft(*args) == B.SPEC_OK
                assert B._pycall.verify(cand, logits, *res, vws, stream, early) == B.SPEC_OK
                assert B._pycall.next_ctx(state, res[1], res[0], new, vws, stream) == B.SPEC_OK
                torch.cuda.synchronize()
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
