"""hpd_decode_step: the attention and the greedy acceptance as one step.

The acceptance reads only the logits and the drafts, so the library runs it
on the SMs that the attention kernel leaves idle (launched behind it, without
waiting for it to end).  Whatever it
chooses, the step must give exactly the results of the two calls made in
order, eagerly and inside a captured CUDA graph, and match the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_2607_18839_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

V = 32000


@pytest.fixture(scope="module")
def hpd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_18839_gb300 import build, hpd as H
    build.build()
    H.load()
    return H


def step_inputs(name, seed):
    inp = W.make_config(name)
    logits = W.make_logits(inp.B, inp.m, V, seed)
    ref_tok0, _ = oracle.pmtp_accept(logits, np.zeros((inp.B, inp.m), np.int32))
    drafts = W.mix_drafts(ref_tok0, V, 0.7, seed=seed + 1)
    return inp, logits, drafts


def to_dev(H, logits, drafts):
    lg = torch.from_numpy(logits.view(np.int16)).cuda().view(torch.bfloat16)
    dr = torch.from_numpy(drafts).cuda()
    return lg, dr


def results(op, tok, acc):
    torch.cuda.synchronize()
    return (op.out.view(torch.int16).cpu().numpy(), op.lse.cpu().numpy(),
            tok.cpu().numpy(), acc.cpu().numpy())


def separate_calls(H, inp, lg, dr):
    op = H.BranchAttn(H.DeviceInputs.from_host(inp))
    tok = torch.empty((inp.B, inp.m), dtype=torch.int32, device="cuda")
    acc = torch.empty((inp.B,), dtype=torch.int32, device="cuda")
    op()
    H.hpd_pmtp_accept(lg.data_ptr(), dr.data_ptr(), inp.B, inp.m, V, tok.data_ptr(),
                      acc.data_ptr(), H._stream_handle(None))
    return results(op, tok, acc)


def assert_same(a, b):
    for x, y, what in zip(a, b, ("out", "lse", "tokens", "accepted_len")):
        assert np.array_equal(x, y, equal_nan=(what == "lse")), what


@pytest.mark.parametrize("name", ["c2", "c3", "c4", "c5"])
def test_step_equals_the_two_calls_bitwise(hpd, name):
    inp, logits, drafts = step_inputs(name, seed=500)
    lg, dr = to_dev(hpd, logits, drafts)
    ref = separate_calls(hpd, inp, lg, dr)
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    tok = torch.full((inp.B, inp.m), -7, dtype=torch.int32, device="cuda")
    acc = torch.full((inp.B,), -7, dtype=torch.int32, device="cuda")
    for _ in range(2):
        op.step(lg, dr, tok, acc)
    got = results(op, tok, acc)
    assert op.errors() == 0
    assert_same(got, ref)


def test_step_matches_the_oracle(hpd):
    inp, logits, drafts = step_inputs("c2", seed=510)
    lg, dr = to_dev(hpd, logits, drafts)
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    tok = torch.empty((inp.B, inp.m), dtype=torch.int32, device="cuda")
    acc = torch.empty((inp.B,), dtype=torch.int32, device="cuda")
    op.step(lg, dr, tok, acc)
    _, lse, tok_np, acc_np = results(op, tok, acc)
    out = op.out.float().cpu().numpy()
    ref_out, ref_lse = oracle.branch_attn(inp)
    assert np.max(np.abs(out - ref_out.reshape(out.shape))) <= 1e-2
    fin = ~np.isneginf(ref_lse)
    assert np.array_equal(np.isneginf(lse), ~fin)
    assert np.max(np.abs(lse[fin] - ref_lse.reshape(lse.shape)[fin])) <= 1e-3
    ref_tok, ref_acc = oracle.pmtp_accept(logits, drafts)
    np.testing.assert_array_equal(tok_np, ref_tok)
    np.testing.assert_array_equal(acc_np, ref_acc)


def test_concurrency_plan(hpd):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # beside the attention when there are fewer than two work units per SM:
    # c2 60 units, c5 264 units, c4 832 units (row tiles + one per page, x KV heads x splits)
    for name, units in (("c2", 60), ("c5", 264), ("c4", 832)):
        args = hpd.make_args(hpd.DeviceInputs.from_host(W.make_config(name)))
        assert hpd.hpd_decode_step_concurrent(args) == (1 if units < 2 * sms else 0), name


@pytest.mark.parametrize("name", ["c2", "c4"])
def test_step_inside_graph_capture(hpd, name):
    inp, logits, drafts = step_inputs(name, seed=520)
    lg, dr = to_dev(hpd, logits, drafts)
    ref = separate_calls(hpd, inp, lg, dr)
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    tok = torch.full((inp.B, inp.m), -7, dtype=torch.int32, device="cuda")
    acc = torch.full((inp.B,), -7, dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    op.step(lg, dr, tok, acc, stream=s)  # eager first call
    s.synchronize()
    tok.fill_(-7)
    acc.fill_(-7)
    op.out.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for _ in range(3):
            op.step(lg, dr, tok, acc, stream=s)
    g.replay()
    got = results(op, tok, acc)
    assert op.errors() == 0
    assert_same(got, ref)


def test_step_refuses_bad_arguments_before_enqueueing(hpd):
    inp, logits, drafts = step_inputs("c2", seed=530)
    lg, dr = to_dev(hpd, logits, drafts)
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    tok = torch.empty((inp.B, inp.m), dtype=torch.int32, device="cuda")
    acc = torch.empty((inp.B,), dtype=torch.int32, device="cuda")
    op.out.fill_(3.0)
    torch.cuda.synchronize()
    lib = hpd.load()
    h = hpd._stream_handle(None)
    # no drafts, then a vocabulary of 0: refused, and the attention did not run
    assert lib.hpd_decode_step(hpd.ctypes.byref(op.args), lg.data_ptr(), None, V,
                               tok.data_ptr(), acc.data_ptr(), h) == 1
    assert lib.hpd_decode_step(hpd.ctypes.byref(op.args), lg.data_ptr(), dr.data_ptr(), 0,
                               tok.data_ptr(), acc.data_ptr(), h) == 1
    torch.cuda.synchronize()
    assert bool((op.out.float() == 3.0).all())


def special_logits(B, m, V, seed):
    """Logits with the cases the argmax must get exactly right: ties (the
    lowest index wins), -0 against +0, NaN (never wins), rows of NaN and -inf
    (the first -inf wins), a row of NaN only (token 0), and maxima at the
    last index and around index 8192."""
    rng = np.random.default_rng(seed)
    x = rng.integers(-4, 5, size=(B, m, V)).astype(np.float32)  # many ties
    x[0, 0, :] = 0.0
    x[0, 0, 7::9] = -0.0
    x[0, 1, :] = np.nan
    x[0, 1, 3] = -np.inf
    x[0, 1, 11] = -np.inf
    x[0, 2, :] = np.nan                      # all NaN -> token 0
    x[1, :, 5::13] = np.nan                  # NaN mixed with values
    x[2, 0, :] = -np.inf
    x[3, 0, V - 1] = 100.0
    if V > 8192:
        x[3, 1, 8192] = 100.0
        x[3, 2, 8191] = 100.0
    return W.f32_to_bf16_bits(x)


@pytest.mark.parametrize("name,V_", [("c4", 4096), ("c4", 20001), ("c2", 32000)])
def test_step_acceptance_special_values(hpd, name, V_):
    inp = W.make_config(name)
    logits = special_logits(inp.B, inp.m, V_, seed=V_)
    ref_tok0, _ = oracle.pmtp_accept(logits, np.zeros((inp.B, inp.m), np.int32))
    drafts = W.mix_drafts(ref_tok0, V_, 0.7, seed=V_ + 1)
    ref_tok, ref_acc = oracle.pmtp_accept(logits, drafts)
    assert ref_tok[0, 2] == 0 and ref_tok[0, 1] == 3 and ref_tok[2, 0] == 0
    lg = torch.from_numpy(logits.view(np.int16)).cuda().view(torch.bfloat16)
    dr = torch.from_numpy(drafts).cuda()
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    tok = torch.full((inp.B, inp.m), -7, dtype=torch.int32, device="cuda")
    acc = torch.full((inp.B,), -7, dtype=torch.int32, device="cuda")
    op.step(lg, dr, tok, acc)
    torch.cuda.synchronize()
    assert op.errors() == 0
    np.testing.assert_array_equal(tok.cpu().numpy(), ref_tok)
    np.testing.assert_array_equal(acc.cpu().numpy(), ref_acc)


@pytest.mark.parametrize("empty,H_kv", [(1, 1), (74, 2), (151, 1), (400, 4)])
def test_step_of_pages_without_branches(hpd, empty, H_kv):
    # Pages without branches: most CTAs of the attention find no unit (or no
    # keys) and end at once, with the copies of the offsets that they began
    # drained, and the acceptance takes their place; every step gives the bits
    # of the first, and the oracle's results.
    inp = W.build_inputs([40] * (empty + 1), [0] * empty + [3], [5, 0, 33], 2, 4 * H_kv, H_kv, 64,
                         seed=520)
    logits = W.make_logits(inp.B, inp.m, V, 521)
    ref_tok, ref_acc = oracle.pmtp_accept(logits, np.zeros((inp.B, inp.m), np.int32))
    lg, dr = to_dev(hpd, logits, np.zeros((inp.B, inp.m), np.int32))
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    tok = torch.empty((inp.B, inp.m), dtype=torch.int32, device="cuda")
    acc = torch.empty((inp.B,), dtype=torch.int32, device="cuda")
    op.step(lg, dr, tok, acc)
    first = results(op, tok, acc)
    ref_out, ref_lse = oracle.branch_attn(inp)
    assert np.max(np.abs(op.out.float().cpu().numpy() - ref_out)) <= 1e-2
    assert np.max(np.abs(first[1] - ref_lse)) <= 1e-3
    np.testing.assert_array_equal(first[2], ref_tok)
    np.testing.assert_array_equal(first[3], ref_acc)
    for _ in range(200):
        op.step(lg, dr, tok, acc)
    assert_same(results(op, tok, acc), first)
    assert op.errors() == 0


@pytest.mark.parametrize("docs,heads,vocab", [(2, 16, 9001), (16, 16, 9001), (16, 16, 33000)])
def test_acceptance_behind_an_attention_that_may_still_run(hpd, docs, heads, vocab):
    # An attention call without split keys, then an acceptance call, which may
    # be launched at the start of a small attention grid (48 units), or when the
    # CTAs of a larger one (320) end; both orders in turn.  Exact.
    inp = W.build_inputs([100] * docs, [3] * docs, [9] * (3 * docs), 8, heads, heads, 64, seed=540)
    B = 3 * docs
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    assert hpd.hpd_branch_attn_kernel_name(op.args, 1) is None
    rng = np.random.default_rng(541)
    vals = rng.integers(-40, 41, size=(B, 8, vocab)).astype(np.float32)  # many ties
    logits = W.f32_to_bf16_bits(vals)
    ref_tok, _ = oracle.pmtp_accept(logits, np.zeros((B, 8), np.int32))
    drafts = W.mix_drafts(ref_tok, vocab, 0.8, seed=542)
    ref_tok, ref_acc = oracle.pmtp_accept(logits, drafts)
    lg, dr = to_dev(hpd, logits, drafts)
    tok = torch.empty((B, 8), dtype=torch.int32, device="cuda")
    acc = torch.empty((B,), dtype=torch.int32, device="cuda")
    op()
    torch.cuda.synchronize()
    first = op.out.clone()
    for _ in range(20):
        tok.fill_(-7), acc.fill_(-7), op.out.zero_()
        for _ in range(2):
            op()
            hpd.hpd_pmtp_accept(lg.data_ptr(), dr.data_ptr(), B, 8, vocab, tok.data_ptr(),
                                acc.data_ptr(), hpd._stream_handle(None))
        torch.cuda.synchronize()
        assert torch.equal(op.out, first)
        np.testing.assert_array_equal(tok.cpu().numpy(), ref_tok)
        np.testing.assert_array_equal(acc.cpu().numpy(), ref_acc)


@pytest.mark.parametrize("B,m,D,vocab", [(38, 8, 128, 80000), (61, 5, 128, 79999), (61, 5, 128, 80000),
                                         (2, 1, 128, 152064), (61, 5, 64, 80001)])
def test_step_where_the_acceptance_goes(hpd, B, m, D, vocab):
    # one page whose keys are split: the acceptance goes before the merge (304
    # and more rows) or, with two rows, beside it; whichever it is, the bits of
    # the two calls, eagerly and from a graph
    inp = W.build_inputs([1500], [B], [(7 * b) % 50 for b in range(B)], m, 8, 2, D, seed=530)
    g = torch.Generator(device="cuda").manual_seed(531)
    lg = torch.randn((B, m, vocab), generator=g, device="cuda").to(torch.bfloat16)
    best = lg.float().argmax(2).to(torch.int32)
    dr = torch.where(torch.rand((B, m), generator=g, device="cuda") < 0.8, best, 0).contiguous()
    op = hpd.BranchAttn(hpd.DeviceInputs.from_host(inp))
    assert "merge_splits" in [hpd.hpd_branch_attn_kernel_name(op.args, k) for k in range(3)]
    op()
    tok, acc = hpd.pmtp_accept(lg, dr)
    ref = results(op, tok, acc)
    top = lg.float().gather(2, tok.long()[:, :, None])[:, :, 0]
    assert torch.equal(top, lg.float().amax(2))
    tok, acc = torch.full_like(tok, -7), torch.full_like(acc, -7)
    op.out.zero_()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    op.step(lg, dr, tok, acc, stream=s)
    s.synchronize()
    assert_same(results(op, tok, acc), ref)
    tok.fill_(-7), acc.fill_(-7), op.out.zero_()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        for _ in range(3):
            op.step(lg, dr, tok, acc, stream=s)
    graph.replay()
    assert_same(results(op, tok, acc), ref)
    assert op.errors() == 0
