"""GPU parity of the fused scoring + top-k kernel against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_06161_gb300 import api
from paper_2602_06161_gb300 import workloads as W
from tests import _gpu as H

pytestmark = pytest.mark.gpu

TOL = 1e-5   # fp32 outputs, max |d|


def run_score(inp: W.ScoreInputs, workspace=None):
    # with a workspace the call takes the native marshalling, as a decoding program's does
    if workspace is None and inp.topk > 0:
        workspace = api.score_workspace(inp.n_seq)
    logits = H.to_dev(inp.logits, "bf16")
    kw = {}
    if inp.cur_tok is not None:
        kw["cur_tok"] = H.to_dev(inp.cur_tok, "i32")
    if inp.d_in is not None:
        kw["d_in"] = H.to_dev(inp.d_in, "f32")
        kw["d_out"] = H.to_dev(inp.d_out, "f32")
    if inp.eligible is not None:
        kw["eligible"] = torch.from_numpy(inp.eligible).cuda()
    r = api.cover_score_fwd(logits, inp.n_seq, inp.topk, workspace=workspace, **kw)
    torch.cuda.synchronize()
    assert api.cover_device_status() == 0
    return {k: v.cpu().numpy() for k, v in r.items()}


def check(inp: W.ScoreInputs, r, what=""):
    ref = oracle.score_rows(inp.logits_f64(), cur_tok=inp.cur_tok, d_in=inp.d_in, d_out=inp.d_out)
    assert np.array_equal(r["argmax"], ref["argmax"]), what
    for k in ("maxprob", "entropy", "score"):
        d = np.abs(r[k].astype(np.float64) - ref[k]).max()
        assert d <= TOL, f"{what} {k} max |d| {d:.3e}"
    # the top-k decision taken on the kernel's own fp32 scores must be bit-exact
    idx, val = oracle.topk_select(r["score"], inp.n_seq, inp.topk, inp.eligible)
    assert np.array_equal(r["topk_idx"], idx), what
    assert np.array_equal(r["topk_score"], val.astype(np.float32)), what
    # against the fp64 selection: identical wherever the oracle's margin is clear
    ref_idx, _ = oracle.topk_select(ref["score"], inp.n_seq, inp.topk, inp.eligible)
    gaps = oracle.topk_margin(ref["score"], inp.n_seq, inp.topk, inp.eligible)
    for g in range(inp.n_seq):
        if gaps[g] > 4 * TOL:
            assert set(r["topk_idx"][g].tolist()) == set(ref_idx[g].tolist()), f"{what} segment {g}"
    return ref


@pytest.mark.parametrize("N,V,n_seq,k", [
    (1, 1, 1, 1), (3, 7, 1, 2), (16, 1000, 4, 3), (64, 4099, 2, 32), (8, 8, 8, 1), (37, 20001, 1, 37),
])
def test_score_shapes(N, V, n_seq, k):
    inp = W.make_score_inputs(N, V, n_seq, k, seed=N + V, spike_frac=0.1)
    check(inp, run_score(inp), f"N{N} V{V}")


@pytest.mark.parametrize("N,V", [
    (5, 16387), (38, 20001),      # eight CTAs a row, the last slice short; the most rows on 152 SMs
    (39, 20001), (76, 8193),      # four
    (77, 65544), (152, 65537),    # two
    (153, 65544),                 # one
    (100, 20001), (153, 36355), (304, 18435), (160, 98305),   # loaded to registers
    (153, 45055),
    (305, 20001), (100, 20481), (100, 18427), (153, 45057),   # and on the other side of that rule
])
def test_score_split_rows(N, V):
    """Rows split over a cluster: sums and, with the maximum in several slices, its first index."""
    inp = W.make_score_inputs(N, V, 1, 4, seed=V, with_cur_tok=True, spike_frac=0.3)
    x = inp.logits
    for r in range(0, N, 2):
        x[r, [V // 9, V // 2, V - 1 - r % 7]] = W.f32_to_bf16_bits(np.full(3, 20.0, np.float32))
    x[1, 0] = x[1, V - 1] = W.f32_to_bf16_bits(np.full(1, 21.0, np.float32))[0]
    check(inp, run_score(inp), f"N{N} V{V}")


def test_score_side_inputs_and_eligibility():
    inp = W.make_score_inputs(96, 5003, 3, 10, seed=7, with_cur_tok=True, with_dio=True, eligible_frac=0.4)
    check(inp, run_score(inp))


@pytest.mark.parametrize("N,V", [(6, 20001), (400, 5000), (100, 20001)])   # rows split or not, to registers
def test_score_token_outside_the_vocabulary(N, V):
    """Every value outside [0, V) has no probability, the largest and smallest of the type too: u and score are NaN."""
    x = H.to_dev(W.make_score_inputs(N, V, 1, 1, seed=V).logits, "bf16")
    outside = [-1, V, 2**31 - 1, -2**31]
    tok = torch.zeros(N, dtype=torch.int32, device="cuda")
    tok[:4] = torch.tensor(outside)
    r = api.cover_score_fwd(x, 1, 0, cur_tok=tok)
    ref = api.cover_score_fwd(x, 1, 0, cur_tok=torch.zeros_like(tok))
    assert r["score"][:4].isnan().all() and torch.equal(r["score"][4:], ref["score"][4:])
    assert torch.equal(r["maxprob"], ref["maxprob"])
    # in the decision step such a row has no score: neither counted in n_t nor chosen
    t, flags = tok.clone(), torch.zeros(N, dtype=torch.uint8, device="cuda")
    d = api.cover_score_decide_fwd(x, 1, t, flags, flags.clone(), tau_draft=0.9, draft_budget=1, remask_budget=3, mask_id=3,
                                   max_seeds=N)
    assert d["score"][:4].isneginf().all() and int(d["stats"][0, 4]) == N - 4
    assert int(flags[:4].sum()) == 0 and t[:4].tolist() == outside
    assert api.cover_device_status() == 0


@pytest.mark.parametrize("N,V", [(6, 20001), (400, 5000), (100, 20001)])   # rows split or not, to registers
def test_score_rows_without_a_greedy_token(N, V):
    """A row of -inf has no greedy token: its score is NaN, not -inf, beside rows that it leaves as they are."""
    x = H.to_dev(W.make_score_inputs(N, V, 1, 1, seed=V).logits, "bf16")
    ref = api.cover_score_fwd(x, 1, 0)
    x[1] = -float("inf")
    r = api.cover_score_fwd(x, 1, 0)
    others = torch.arange(N, device="cuda") != 1
    assert r["score"][1].isnan() and torch.equal(r["score"][others], ref["score"][others])
    assert api.cover_device_status() == 0


LOWEST = float(torch.finfo(torch.bfloat16).min)


@pytest.mark.parametrize("low", [LOWEST, -1e38, -1e35, -1e30, -1e10, -1e9])
@pytest.mark.parametrize("N,V", [(4, 20001), (4, 126464), (400, 20001), (400, 5000), (100, 20001)])   # split or not, to registers
def test_score_masked_logits(N, V, low):
    """Masked logits: in the elements past the aligned vectors, in whole batches of a lane, in whole slices of
    a row, at its start and between. They have no weight. (t 2^t of the lowest value is -inf times 0: no entropy.)"""
    inp = W.make_score_inputs(N, V, 1, 1, seed=V)
    x = H.to_dev(inp.logits, "bf16")
    spans = [(V - 1, V), (V - 5, V), (V - 40, V), (2 * V // 3, V), (V // 2, V), (0, 1), (0, V // 3), (V // 4, V // 2),
             (1, V), (0, V - 1)]
    for lo, hi in spans:
        y = x.clone()
        y[:, lo:hi] = low
        r = {k: v.cpu().numpy() for k, v in api.cover_score_fwd(y, 1, 0).items()}
        ref = oracle.score_rows(y[:3].double().cpu().numpy())
        assert np.array_equal(r["argmax"][:3], ref["argmax"]), (lo, hi)
        for k in ("maxprob", "score") + (("entropy",) if low > LOWEST else ()):
            assert np.abs(r[k][:3] - ref[k]).max() <= TOL, (lo, hi, k, r[k][:3], ref[k])
    assert api.cover_device_status() == 0


@pytest.mark.parametrize("N,V", [(4, 20001), (4, 126464), (400, 20001), (400, 5000), (100, 20001)])   # split or not, to registers
def test_score_nan_logits_show(N, V):
    """One NaN logit anywhere, or a slice of them, leaves its row NaN and the other rows as they are."""
    x = H.to_dev(W.make_score_inputs(N, V, 1, 1, seed=V).logits, "bf16")
    ref = api.cover_score_fwd(x, 1, 0)
    for lo, hi in [(V - 1, V), (0, 1), (V // 2, V // 2 + 1), (V // 3, V), (V - 3, V)]:
        y = x.clone()
        y[1, lo:hi] = float("nan")
        r = api.cover_score_fwd(y, 1, 0)
        others = torch.arange(N, device="cuda") != 1
        for k in ("maxprob", "entropy", "score"):
            assert r[k][1].isnan() and torch.equal(r[k][others], ref[k][others]), (lo, hi, k)
    assert api.cover_device_status() == 0


@pytest.mark.parametrize("per,k,frac", [(1000, 32, 0.012), (300, 20, 0.012), (1000, 6, 0.003)])
def test_score_topk_fewer_eligible_than_k(per, k, frac):
    """General path with fewer eligible rows than k: the list ends in -1 / -inf."""
    inp = W.make_score_inputs(2 * per, 300, 2, k, seed=per, eligible_frac=frac)
    r = run_score(inp)
    check(inp, r)
    n_elig = inp.eligible.reshape(2, per).sum(axis=1)
    assert (n_elig < k).all()
    for g in range(2):
        assert (r["topk_idx"][g, n_elig[g]:] == -1).all() and (r["topk_idx"][g, :n_elig[g]] >= 0).all()


@pytest.mark.parametrize("N,k", [(304, 8), (304, 9), (288, 40), (200, 3)])
def test_score_topk_of_rows_loaded_to_registers(N, k):
    inp = W.make_score_inputs(N, 18435, 1, k, seed=N + k, eligible_frac=0.7)
    check(inp, run_score(inp))


@pytest.mark.parametrize("per,k", [
    (289, 2), (289, 8), (1025, 8), (4096, 3),       # found in the row kernel
    (289, 9), (512, 32), (513, 32), (1024, 32),     # the lists of 10 to 32 warps, merged
    (289, 33), (300, 300), (768, 33), (768, 700),   # ranks
    (769, 33), (1024, 1024), (1025, 33),            # sorts
    (1025, 9), (1025, 32), (4096, 32),              # warp sorts on 512 threads
])
@pytest.mark.parametrize("frac", [1.0, 0.6, 0.005])
def test_score_topk_of_long_segments(per, k, frac):
    """Segments longer than the row kernel's CTAs: lists in a launch of their own, also with fewer eligible rows."""
    inp = W.make_score_inputs(2 * per, 203, 2, k, seed=per + k, eligible_frac=frac)
    inp.logits[5] = inp.logits[7] = inp.logits[per + 3] = inp.logits[2]   # equal scores: the lower row first
    check(inp, run_score(inp, workspace=api.score_workspace(2)), f"per {per} k {k}")


def test_score_no_eligible_rows():
    inp = W.make_score_inputs(32, 512, 2, 4, seed=8, eligible_frac=0.0)
    r = run_score(inp)
    assert (r["topk_idx"] == -1).all() and np.isneginf(r["topk_score"]).all()


def test_score_ties_and_uniform_rows():
    inp = W.make_score_inputs(16, 3000, 1, 16, seed=9)
    x = inp.logits.copy()
    x[0, :] = W.f32_to_bf16_bits(np.full(3000, 0.5, np.float32))      # all equal: argmax 0
    x[1, :] = W.f32_to_bf16_bits(np.full(3000, -1.0, np.float32))
    x[1, [17, 2000, 2999]] = W.f32_to_bf16_bits(np.float32([3.0, 3.0, 3.0]))  # tie: lowest index 17
    x[2] = x[1]                                                           # equal scores: lower row first
    inp.logits = x
    r = run_score(inp)
    assert r["argmax"][0] == 0 and r["argmax"][1] == 17
    check(inp, r)


@pytest.mark.parametrize("V", [40000, 40001])   # aligned rows (V % 8 == 0), unaligned rows
def test_score_argmax_ties_across_batches(V):
    """The first index of the row maximum when it occurs several times: in different chunks, in one
    thread's batch (different vectors), in one thread's batches of different chunks, at the row's
    first and last element, and as -0.0 before +0.0."""
    placed = [
        [39999, 12345, 8192 + 3, 20000],       # several chunks: 8195
        [2 * 2048 + 5 * 8 + 3, 5 * 8 + 6],     # one thread, one batch, vectors 2 and 0: 46
        [3 * 8192 + 7 * 8 + 1, 8192 + 7 * 8 + 2],
        [0, V - 1],
        [V - 1],
        [8 * 4096 + 11, 4096 + 3, 2 * 4096 + 3],
    ]
    inp = W.make_score_inputs(len(placed) + 1, V, 1, 3, seed=V)
    x = inp.logits.copy()
    for r, pos in enumerate(placed):
        x[r, pos] = W.f32_to_bf16_bits(np.full(len(pos), 9.5, np.float32))
    zr = len(placed)
    x[zr, :] = W.f32_to_bf16_bits(np.full(V, -2.0, np.float32))
    x[zr, 30000] = np.uint16(0x8000)   # -0.0
    x[zr, 31000] = np.uint16(0x0000)   # +0.0
    x[zr, 500] = np.uint16(0x8000)
    inp.logits = x
    r = run_score(inp)
    expect = [min(p) for p in placed] + [500]
    assert r["argmax"].tolist() == expect
    check(inp, r)


def test_score_max_segment_and_workspace_reuse():
    inp = W.make_score_inputs(4096, 64, 1, 256, seed=10)
    ws = api.score_workspace(1)
    r1 = run_score(inp, workspace=ws)
    r2 = run_score(inp, workspace=ws)
    assert int(ws.abs().sum().item()) == 0
    for k in r1:
        assert np.array_equal(r1[k], r2[k])
    check(inp, r1)


@pytest.mark.parametrize("name", ["dream_gqa_l1024", "llada_b8_l2048"])
def test_score_named_workloads_full(name):
    inp = W.WORKLOADS[name].score_inputs()
    r = run_score(inp)
    ref = check(inp, r, name)
    gaps = oracle.topk_margin(ref["score"], inp.n_seq, inp.topk)
    print(f"{name}: top-k margins min {gaps.min():.3e}")


@pytest.mark.parametrize("per,V,k", [
    (288, 1000, 40),    # one row per thread of the bulk-copy kernel: selection by rank
    (289, 1000, 20),    # the general path, a short list: warp sorts and merges
    (289, 1000, 40),    # the general path, a long list: the bitonic sort
    (512, 1001, 33),    # an odd vocabulary, more rows than a CTA has threads
    (513, 1001, 32),    # and one row past it: warp sorts and merges
    (4096, 136, 32),    # the largest segment, k = 32
    (600, 300, 9),      # the fewest keys taken by warp sorts
    (600, 300, 8),      # the most taken by rounds of a CTA-wide maximum
    (777, 200, 1),      # k = 1
    (600, 1001, 5),     # an odd vocabulary, the general path, rounds
])
def test_score_topk_on_both_sides_of_the_fast_path(per, V, k):
    inp = W.make_score_inputs(2 * per, V, 2, k, seed=per + k, spike_frac=0.1, eligible_frac=0.8)
    check(inp, run_score(inp), f"per {per} V {V} k {k}")
