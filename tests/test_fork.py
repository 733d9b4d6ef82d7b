"""Fork detection and child branches (Algorithm 1, Sec. 3.3): pins of the
oracle (hand-worked example, invariants) and bit-exact parity of
hpd_fork_children with it."""
import numpy as np
import pytest

from oracle import fork as F

FORK = 151666  # any token id serves as the fork token


def _case(rng, n_docs, per_doc, m, max_pages, p_fork):
    counts = rng.integers(0, per_doc + 1, size=n_docs)
    branch_cu = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    B = int(branch_cu[-1])
    tok = rng.integers(0, 1000, size=(B, m)).astype(np.int32)
    tok[rng.random((B, m)) < p_fork] = FORK
    acc = rng.integers(-1, m + 1, size=B).astype(np.int32)
    is_layout = np.zeros(B, np.int32)
    for d in range(n_docs):  # first branch of a page is its layout branch
        if counts[d]:
            is_layout[branch_cu[d]] = 1
    layout_pos = rng.integers(0, 3000, size=B).astype(np.int32)
    bpl = rng.integers(0, 3000, size=B).astype(np.int32)
    blen = rng.integers(0, 200, size=B).astype(np.int32)
    pt = rng.integers(0, 5000, size=(B, max_pages)).astype(np.int32)
    return tok, acc, is_layout, layout_pos, branch_cu, bpl, blen, pt


def test_hand_example():
    # page 0: branches 0 (layout), 1; page 1: branch 2 (layout)
    tok = np.array([[5, FORK, 7, FORK], [FORK, 1, 2, 3], [FORK, 9, 9, 9]], np.int32)
    acc = np.array([2, 4, 0], np.int32)  # branch 0 emits 3 tokens, branch 2 emits 1
    is_layout = np.array([1, 0, 1], np.int32)
    layout_pos = np.array([100, 0, 40], np.int32)
    cu = np.array([0, 2, 3], np.int32)
    pt = np.arange(6, dtype=np.int32).reshape(3, 2)
    new, err = F.fork_children(tok, acc, is_layout, layout_pos, FORK, cu, None,
                               np.array([10, 11, 12], np.int32), pt, cap=8)
    assert err == 0 and new["new_B"] == 5
    # page 0: old 0, old 1, child of 0 at index 1 (prefix 100 + 1 + 1); the
    # fork token at index 3 was not emitted; page 1: old 2, child of 2 (40 + 1)
    assert list(new["branch_cu"]) == [0, 3, 5]
    assert list(new["parent"]) == [0, 1, -1, 2, -3]
    assert list(new["branch_prefix_len"]) == [-1, -1, 102, -1, 41]
    assert list(new["branch_len"]) == [10, 11, 0, 12, 0]
    assert (new["page_table"][2] == -1).all() and (new["page_table"][3] == pt[2]).all()


def test_invariants_and_capacity():
    rng = np.random.default_rng(3)
    tok, acc, lay, pos, cu, bpl, blen, pt = _case(rng, 7, 9, 4, 3, 0.3)
    new, err = F.fork_children(tok, acc, lay, pos, FORK, cu, bpl, blen, pt, cap=10_000)
    assert err == 0
    B = len(blen)
    olds = new["parent"][new["parent"] >= 0]
    assert sorted(olds) == list(range(B))
    n_child = int((new["parent"] < 0).sum())
    expect = sum(int(np.sum(tok[b, :min(acc[b] + 1, 4)] == FORK)) for b in range(B)
                 if lay[b] and acc[b] >= 0)
    assert n_child == expect and new["new_B"] == B + n_child
    for d in range(len(cu) - 1):  # every child lands in its parent's page
        for i in range(new["branch_cu"][d], new["branch_cu"][d + 1]):
            par = new["parent"][i]
            b = par if par >= 0 else -1 - par
            assert cu[d] <= b < cu[d + 1]
    _, err = F.fork_children(tok, acc, lay, pos, FORK, cu, bpl, blen, pt, cap=B + n_child - 1)
    assert err == F.ERR_FORK_CAP
    _, err = F.fork_children(tok, acc, lay, pos, FORK, np.array([0, 5, 3, B], np.int32)
                             if B > 5 else np.array([0, 1, 0, B], np.int32), bpl, blen, pt, cap=10_000)
    assert err == F.ERR_BRANCH_CU


def _gpu(args, cap):
    import torch
    from paper_2607_18839_gb300 import hpd as H
    tok, acc, lay, pos, cu, bpl, blen, pt = args
    t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    new = H.fork_children(t(tok), t(acc), t(lay), t(pos), FORK, t(cu), t(bpl), t(blen), t(pt), cap)
    torch.cuda.synchronize()
    err = int(new["workspace"][:4].view(torch.int32).item())
    return {k: v.cpu().numpy() for k, v in new.items() if k != "workspace"}, err


@pytest.mark.gpu
@pytest.mark.parametrize("n_docs,per_doc,m,p_fork,layout", [
    (1, 16, 4, 0.2, True), (32, 24, 8, 0.05, True), (700, 3, 2, 0.5, False), (3, 0, 4, 0.3, True)])
def test_gpu_parity(n_docs, per_doc, m, p_fork, layout):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(n_docs * 10 + m)
    case = list(_case(rng, n_docs, per_doc, m, 5, p_fork))
    if not layout:
        case[2] = None
    cap = int(case[4][-1]) * (m + 1) + 1
    ref, err = F.fork_children(*case[:4], FORK, *case[4:], cap=cap)
    got, gerr = _gpu(case, cap)
    assert gerr == err == 0
    nb = ref["new_B"]
    assert int(got["new_B"][0]) == nb
    assert np.array_equal(got["branch_cu"], ref["branch_cu"])
    for k in ("parent", "branch_len", "branch_prefix_len", "page_table"):
        assert np.array_equal(got[k][:nb], ref[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("n_docs,per_doc,m,max_pages", [(3, 2, 1, 1), (2, 4, 16, 32),
                                                        (5, 605, 5, 33), (11, 294, 64, 65)])
def test_gpu_rows_of_the_page_table(n_docs, per_doc, m, max_pages):
    # a warp moves a row or a piece of one: rows of one word, of a warp's width
    # and one more, and more rows than warps (128 CTAs of 8); whole numbers, exact
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    case = _case(np.random.default_rng(7 * max_pages + m), n_docs, per_doc, m, max_pages, 0.1)
    cap = int(case[4][-1]) * (m + 1) + 1
    ref, err = F.fork_children(*case[:4], FORK, *case[4:], cap=cap)
    got, gerr = _gpu(case, cap)
    assert gerr == err == 0
    nb = ref["new_B"]
    assert int(got["new_B"][0]) == nb
    for k in ("parent", "branch_len", "branch_prefix_len", "page_table"):
        assert np.array_equal(got[k][:nb], ref[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("n_docs,per_doc,m,p_fork", [(3, 85, 1, 0.5), (1, 256, 64, 0.3),
                                                     (1, 257, 64, 0.3), (1500, 7, 64, 0.05),
                                                     (1, 11997, 7, 0.05), (1, 11998, 64, 0.05)])
def test_gpu_tokens_of_layout_branches_only(n_docs, per_doc, m, p_fork):
    # The tokens that count are those emitted by layout branches, whatever the
    # others hold: as many branches as a CTA has threads (256) and one more or
    # less, the largest call of one launch and the next; whole numbers, exact.
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(9 * per_doc + m)
    B = n_docs * per_doc
    lay = (rng.random(B) < 0.1).astype(np.int32)
    tok = np.where((lay[:, None] == 0) | (rng.random((B, m)) < p_fork), FORK, 5).astype(np.int32)
    ints = lambda lo, hi, *n: rng.integers(lo, hi, size=n).astype(np.int32)
    case = [tok, ints(-1, m + 1, B), lay, ints(0, 3000, B),
            (np.arange(n_docs + 1) * per_doc).astype(np.int32), ints(0, 3000, B), ints(0, 40, B),
            ints(0, 5000, B, 3)]
    cap = int(case[4][-1]) + int((case[0] == FORK)[lay == 1].sum()) + 1
    ref, err = F.fork_children(*case[:4], FORK, *case[4:], cap=cap)
    got, gerr = _gpu(case, cap)
    assert gerr == err == 0
    nb = ref["new_B"]
    assert int(got["new_B"][0]) == nb
    for k in ("parent", "branch_len", "branch_prefix_len", "page_table"):
        assert np.array_equal(got[k][:nb], ref[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("B,max_pages", [(1, 32768), (1, 32769), (3, 4097), (31, 1056), (1023, 33),
                                         (1024, 257), (1025, 256), (700, 1000)])
def test_gpu_pieces_of_wide_rows(B, max_pages):
    # a row is cut into pieces of 32 to 256 words, as few pieces as the largest
    # grid has warps (1,024) where that is enough: full and nearly empty last
    # pieces, one piece to a warp and more; whole numbers, so exact
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(B + max_pages)
    ints = lambda lo, hi, *n: rng.integers(lo, hi, size=n).astype(np.int32)
    tok = np.where(rng.random((B, 2)) < 0.2, FORK, 5).astype(np.int32)
    tok[-1, 0] = FORK
    case = [tok, np.full(B, 1, np.int32), None, ints(0, 3000, B), np.array([0, B // 2, B], np.int32),
            None, ints(0, 40, B), ints(0, 5000, B, max_pages)]
    cap = B + int((tok == FORK).sum())
    ref, err = F.fork_children(*case[:4], FORK, *case[4:], cap=cap)
    got, gerr = _gpu(case, cap)
    assert gerr == err == 0 and int(got["new_B"][0]) == ref["new_B"] == cap
    for k in ("parent", "branch_len", "branch_prefix_len", "page_table"):
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.gpu
def test_gpu_capacity_and_bad_offsets():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(5)
    case = list(_case(rng, 4, 6, 4, 2, 0.5))
    ref, _ = F.fork_children(*case[:4], FORK, *case[4:], cap=10_000)
    B = int(case[4][-1])
    got, err = _gpu(case, max(B, ref["new_B"] - 1))
    assert err == F.ERR_FORK_CAP and int(got["new_B"][0]) == -1
    bad = list(case)
    bad[4] = np.array([0, 3, 1, 4, B], np.int32)
    got, err = _gpu(bad, 10_000)
    assert err == F.ERR_BRANCH_CU and int(got["new_B"][0]) == -1
