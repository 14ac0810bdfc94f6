"""The native argument marshalling takes only calls of plain CUDA tensors: any other form is handed
back (None) with nothing launched, and the Python path raises its errors as it always did."""
import sys

import pytest
import torch

from paper_2602_06161_gb300 import _lib, api


def _qkv(dtype=torch.bfloat16):
    return [torch.zeros(1, 2, 16, 128, dtype=dtype) for _ in range(3)]


def test_cpu_tensors_are_handed_back_and_refused():
    q, k, v = _qkv()
    n = _lib.native()
    assert n.attn(0, q, k, v, None, None, None, 0, None, None, True, None) is None
    assert n.attn(2, q, k, v, None, None, None, 0, None, None, True, None) is None
    assert n.kv(1, k, v, torch.zeros(1, 2, dtype=torch.int32), k, v, None) is None
    with pytest.raises(ValueError, match="q must be a CUDA tensor"):
        api.cover_attn_fwd(q, k, v)
    with pytest.raises(TypeError, match="q must be torch.float32"):
        api.cover_attn_fwd_f32(q, k, v)
    with pytest.raises(ValueError, match="logits must be a CUDA tensor"):
        api.cover_score_fwd(torch.zeros(4, 8, dtype=torch.bfloat16), 1, 1)


@pytest.mark.parametrize("args", [(None,) * 12, (0, 1, 2, 3, None, None, None, 0, None, None, True, None),
                                  ("0",) + (None,) * 11])
def test_other_objects_are_handed_back(args):
    assert _lib.native().attn(*args) is None


def test_wrong_number_of_arguments():
    for fn in ("attn", "score", "decide", "mass", "kv"):
        with pytest.raises(TypeError):
            getattr(_lib.native(), fn)(1, 2)
    with pytest.raises(ValueError):
        _lib.native().bind([1, 2])


def test_not_a_tensor():
    with pytest.raises(TypeError, match="q must be a torch.Tensor"):
        api.cover_attn_fwd([1.0], None, None)


def test_forms_that_the_native_path_does_not_take_are_not_offered_to_it(monkeypatch):
    """A stream, given outputs, a missing workspace: such calls pay for one marshalling, not for two."""
    class Native:
        def __getattr__(self, name):
            raise AssertionError(name + " was offered the call")

    monkeypatch.setattr(api, "_nat", Native())
    q, k, v = _qkv()
    x, t, u = torch.zeros(4, 8, dtype=torch.bfloat16), torch.zeros(4, dtype=torch.int32), torch.zeros(4, dtype=torch.uint8)
    f32, ws = torch.zeros(1, 2, 16), torch.zeros(64, dtype=torch.int32)
    dec = dict(draft_budget=1, remask_budget=1, mask_id=0)
    calls = [lambda: api.cover_attn_fwd(q, k, v, stream=0), lambda: api.cover_attn_fwd_prefix(q, k, v, q0=0, stream=0),
             lambda: api.cover_score_fwd(x, 1, 1), lambda: api.cover_score_fwd(x, 1, 1, workspace=ws, out={}),
             lambda: api.cover_score_fwd(x, 1, 0, stream=0), lambda: api.cover_seed_kv_gather(q, q, t[None], stream=0),
             lambda: api.cover_score_decide_fwd(x, 1, t, u, u, tau_draft=0.5, **dec),
             lambda: api.cover_score_decide_fwd(x, 1, t, u, u, tau_draft=0.5, workspace=ws, out={}, **dec),
             lambda: api.cover_score_decide_fwd(x, 1, t, u, u, tau_draft=1, workspace=ws, **dec),
             lambda: api.cover_attn_mass_fwd(q, k, f32, t, u, mask_id=0, pos0=0, per=4)]
    for call in calls:
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            call()
    with pytest.raises(AssertionError, match="attn was offered"):
        api.cover_attn_fwd(q, k, v)


def test_the_binding_is_made_again_for_another_torch_or_interpreter(monkeypatch, tmp_path):
    """The object reads PyTorch's and the interpreter's structures: it serves the ones it was compiled for only."""
    from paper_2602_06161_gb300 import build

    build.build()
    assert not build._binding_stale()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build._binding_stale()
    monkeypatch.undo()
    monkeypatch.setattr(sys, "version", "9.9.9 (other)")
    assert build._binding_stale()
    monkeypatch.undo()
    # a failure leaves no object behind, is not tried again for the same pair, and does not touch the library
    monkeypatch.setattr(build, "BINDING", str(tmp_path / "_binding.so"))
    monkeypatch.setattr(build, "BINDING_TAG", str(tmp_path / "binding.tag"))
    (tmp_path / "_binding.so").write_text("of another torch")
    monkeypatch.setenv("CXX", "no-such-compiler")
    with pytest.warns(UserWarning, match="marshalled in Python"):
        assert build.build() == build.LIB
    assert not (tmp_path / "_binding.so").exists() and not build._binding_stale() and not build._stale()
    # nor is one used that belongs to another pair and cannot be replaced
    monkeypatch.setattr(build, "BINDING_TAG", str(tmp_path / "no" / "such" / "folder"))
    monkeypatch.setattr(_lib, "_native", None)
    with pytest.warns(UserWarning, match="marshalled in Python"):
        assert _lib.native() is _lib._Declines


def test_calls_work_without_the_binding(monkeypatch):
    monkeypatch.setitem(sys.modules, "paper_2602_06161_gb300._binding", None)   # its import fails
    monkeypatch.delattr("paper_2602_06161_gb300._binding", raising=False)
    monkeypatch.setattr(_lib, "_native", None)
    monkeypatch.setattr(api, "_nat", None)
    with pytest.warns(UserWarning, match="marshalled in Python"):
        with pytest.raises(ValueError, match="q must be a CUDA tensor"):   # the Python path's own check
            api.cover_attn_fwd(*_qkv())
    assert _lib.native().kv() is None
