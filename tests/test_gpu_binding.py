"""The native argument marshalling against the Python path behind it (a Stream object takes that one):
the same bits, the same objects returned, the same errors."""
import pytest
import torch

from paper_2602_06161_gb300 import CoverError, api

pytestmark = pytest.mark.gpu


def _r(*shape, dtype=torch.bfloat16, seed=0):
    return torch.randn(shape, generator=torch.Generator("cuda").manual_seed(seed + len(shape)), device="cuda").to(dtype)


def _seeds(B, S, L):
    return torch.stack([torch.randperm(L)[:S] for _ in range(B)]).to(torch.int32).cuda()


def _calls():
    calls = {}
    for name, dt, D in (("", torch.bfloat16, 128), ("_f32", torch.float32, 64)):
        k, v, km, vm = _r(2, 2, 70, D, dtype=dt), _r(2, 2, 70, D, dtype=dt, seed=1), _r(2, 2, 3, D, dtype=dt, seed=2), \
            _r(2, 2, 3, D, dtype=dt, seed=3)
        sd, q = _seeds(2, 3, 70), _r(2, 4, 70, D, dtype=dt, seed=4)
        qw = q[:, :, 20:51].contiguous()
        fn, fw = getattr(api, "cover_attn_fwd" + name), getattr(api, "cover_attn_fwd_prefix" + name)
        calls["attn" + name] = lambda fn=fn, a=(q, k, v, km, vm, sd), **kw: fn(*a, **kw)
        calls["attn_no_seeds" + name] = lambda fn=fn, a=(q, k, v), **kw: fn(*a, want_lse=False, **kw)
        calls["prefix" + name] = lambda fn=fw, a=(qw, k, v, km, vm, sd), **kw: fn(*a, q0=20, **kw)
    x = _r(12, 1003, seed=5)
    tok = torch.randint(0, 1003, (12,), device="cuda", dtype=torch.int32)
    d, e = torch.rand(12, device="cuda"), torch.rand(12, device="cuda") + 1
    ok = (torch.rand(12, device="cuda") < 0.6).to(torch.uint8)
    calls["score"] = lambda **kw: api.cover_score_fwd(x, 2, 3, workspace=api.score_workspace(2), **kw)
    calls["score_side"] = lambda **kw: api.cover_score_fwd(x, 2, 3, cur_tok=tok, d_in=d, d_out=e, eligible=ok,
                                                           workspace=api.score_workspace(2), **kw)
    calls["score_k0"] = lambda **kw: api.cover_score_fwd(x, 2, 0, **kw)
    calls["decide"] = lambda **kw: api.cover_score_decide_fwd(
        x, 2, tok.clone(), ok.clone(), ok.clone(), tau_draft=0.01, draft_budget=2, remask_budget=3, mask_id=1000, pos0=5,
        max_seeds=4, d_in=d, d_out=e, draft_ok=1 - ok, workspace=api.decide_workspace(12, 2), **kw)
    q, k, sd = _r(2, 4, 70, 128, seed=4), _r(2, 2, 70, 128), _seeds(2, 3, 70)
    lse, km = _r(2, 4, 70, dtype=torch.float32, seed=6) + 5, _r(2, 2, 3, 128, seed=2)
    t2, f2 = torch.randint(0, 9, (80,), device="cuda", dtype=torch.int32), torch.full((80,), 2, device="cuda", dtype=torch.uint8)
    ws = torch.empty(api.cover_attn_mass_workspace_bytes(2, 4, 40), dtype=torch.uint8, device="cuda")
    calls["mass"] = lambda **kw: api.cover_attn_mass_fwd(q, k, lse, t2, f2, mask_id=3, pos0=30, per=40, k_seedmask=km,
                                                         seed_idx=sd, workspace=ws, **kw)
    calls["gather"] = lambda **kw: api.cover_seed_kv_gather(k, k.clone(), sd, **kw)

    def override(**kw):
        a, b = k.clone(), k.clone()
        return api.cover_seed_kv_override(a, b, sd, km.clone(), km.clone(), **kw) + (a, b)
    calls["override"] = override
    return calls


NAMES = ["attn", "attn_no_seeds", "prefix", "attn_f32", "attn_no_seeds_f32", "prefix_f32", "score", "score_side",
         "score_k0", "decide", "mass", "gather", "override"]


def _flat(r):
    return [x for _, x in sorted(r.items())] if isinstance(r, dict) else list(r)


class _Counting:
    """The native marshalling, counting the calls that it took."""

    def __init__(self, native):
        self.native, self.took = native, 0

    def __getattr__(self, name):
        def call(*args):
            r = getattr(self.native, name)(*args)
            self.took += r is not None
            return r
        return call


@pytest.mark.parametrize("name", NAMES)
def test_native_call_equals_the_python_path(name, monkeypatch):
    torch.manual_seed(0)
    call = _calls()[name]
    counting = _Counting(api._native())
    monkeypatch.setattr(api, "_nat", counting)
    a = call()
    assert counting.took == 1
    b = call(stream=torch.cuda.current_stream())
    assert counting.took == 1
    torch.cuda.synchronize()
    assert type(a) is type(b) and (not isinstance(a, dict) or list(a) == list(b))
    for x, y in zip(_flat(a), _flat(b)):
        if x is None or y is None:
            assert x is y
            continue
        assert (x.shape, x.dtype, x.device, x.requires_grad) == (y.shape, y.dtype, y.device, y.requires_grad)
        if not (name == "score_k0" and x.numel() == 0):
            assert torch.equal(x, y)
    assert api.cover_device_status() == 0


def test_given_outputs_are_returned_and_side_streams_used():
    q, k = _r(1, 2, 64, 128), _r(1, 2, 64, 128, seed=9)
    out, lse = torch.empty_like(q), torch.empty(1, 2, 64, device="cuda")
    ref = api.cover_attn_fwd(q, k, k)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        o, m = api.cover_attn_fwd(q, k, k, out=out, lse=lse)
    side.synchronize()
    assert o is out and m is lse and torch.equal(out, ref[0]) and torch.equal(lse, ref[1])


def test_errors_are_those_of_the_python_path():
    q, k = _r(1, 2, 64, 128), _r(1, 2, 64, 128, seed=9)
    with pytest.raises(ValueError, match="q must be contiguous"):
        api.cover_attn_fwd(q.transpose(1, 2), k, k)
    with pytest.raises(TypeError, match="k_cached must be torch.bfloat16"):
        api.cover_attn_fwd(q, k.float(), k)
    with pytest.raises(ValueError, match="matching q"):
        api.cover_attn_fwd(q, k[:, :, :32].contiguous(), k)
    with pytest.raises(ValueError, match="seed_idx must be"):
        api.cover_attn_fwd(q, k, k, k, k, torch.zeros(2, 64, dtype=torch.int32, device="cuda"))
    with pytest.raises(CoverError) as e:
        api.cover_attn_fwd(*[_r(1, 2, 64, 64, seed=i) for i in range(3)])   # D = 64 has no bf16 kernel
    assert e.value.code == -2
    with pytest.raises(CoverError) as e:
        api.cover_attn_fwd_prefix(q[:, :, :8].contiguous(), k, k, q0=60)
    assert e.value.code == -1
    with pytest.raises(TypeError, match="logits must be torch.bfloat16"):
        api.cover_score_fwd(q.float()[0, 0], 1, 1, workspace=api.score_workspace(1))


class _NoTruth:
    def __bool__(self):
        raise ArithmeticError("no truth value")


def test_a_flag_without_a_truth_value_raises_before_anything_is_launched():
    q, k = _r(1, 2, 64, 128), _r(1, 2, 64, 128, seed=9)
    out = torch.zeros_like(q)
    with pytest.raises(ArithmeticError, match="no truth value"):
        api.cover_attn_fwd(q, k, k, out=out, want_lse=_NoTruth())
    x = _r(12, 1003, seed=5)
    tok, flags = torch.full((12,), 1000, device="cuda", dtype=torch.int32), torch.zeros(12, device="cuda", dtype=torch.uint8)
    with pytest.raises(ArithmeticError, match="no truth value"):
        api.cover_score_decide_fwd(x, 2, tok, flags, flags.clone(), tau_draft=0.0, draft_budget=2, remask_budget=3,
                                   mask_id=1000, min_one=_NoTruth(), workspace=api.decide_workspace(12, 2))
    torch.cuda.synchronize()
    assert not out.any() and (tok == 1000).all() and not flags.any()
