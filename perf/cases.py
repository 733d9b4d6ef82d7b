"""What is measured of the branch-decode step: its cases, their inputs, their
work and what their results may differ by.

A case is one call (or one pair of calls) that a decoder built on libhpd makes
in every step: the branch attention (``BranchAttn.__call__``), the whole step
with the acceptance (``BranchAttn.step``), the acceptance alone
(``pmtp_accept``), the paged-KV append and rollback (``PagedKV``) and the fork
detection (``fork_children``).  Sizes are those of the presets of
``workloads.py`` and of the test suite, or generic.  Lengths (prefixes,
branches, private histories, fork positions) come from the case alone
(``len_seed``), so that the work does not depend on the seed of the inputs;
values and the physical order of the KV pages come from that seed.
"""
import math

import numpy as np
import torch

from paper_2607_18839_gb300 import hpd

PAGE = 16
FORK_TOKEN = 7
#: no drawn case may cost more than the largest listed ones
MAX_FLOPS, MAX_BYTES = 1.1e11, 0.8e9


# ---------------------------------------------------------------- the cases --

def _attn(name, **kw):
    case = dict(name=name, kind="attn", docs=1, branches_lo=16, branches_hi=16, prefix_lo=1152,
                prefix_hi=1152, suffix="uniform", suffix_lo=16, suffix_hi=256, m=4, hq=16, hkv=2,
                d=128, layout="contiguous", fork=False, layout_branch=False, vocab=0, len_seed=1)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: a short page with four branches of one token
        # each, where latency and launches are all there is
        _attn("attn_tiny", branches_lo=4, branches_hi=4, prefix_lo=256, prefix_hi=256,
              suffix_lo=8, suffix_hi=32, m=1, hq=8, hkv=2, d=64),
        # one page of the vision encoder's 1,024 tokens being read by 16
        # branches: attention and acceptance as one step (the ordinary call
        # of an interactive session)
        _attn("step_one_page", kind="step", vocab=32000),
        # a long page with many blocks of text in flight
        _attn("attn_busy_page", branches_lo=64, branches_hi=64, prefix_lo=4096, prefix_hi=4096,
              suffix="lognormal", suffix_lo=1, suffix_hi=1024, m=4, hq=32, hkv=8),
        # a serving batch: 32 pages of different lengths, each with 24
        # branches; the whole step (the largest case by tokens and bytes)
        _attn("step_serving_batch", kind="step", docs=32, branches_lo=24, branches_hi=24,
              prefix_lo=1024, prefix_hi=3072, suffix="lognormal", suffix_lo=1, suffix_hi=1024,
              m=8, vocab=32000),
        # the longest context with the most branches of one page (the largest
        # case by operations)
        _attn("attn_long_page", branches_lo=256, branches_hi=256, prefix_lo=8192, prefix_hi=8192,
              suffix="pareto", suffix_lo=8, suffix_hi=2048, m=4, hq=32, hkv=8),
        # a batch whose pages' prefixes sit in the shared KV pool, page by
        # page wherever a page was free (a pool after some hours of serving)
        _attn("attn_paged_batch", docs=16, branches_lo=8, branches_hi=32, prefix_lo=777,
              prefix_hi=2999, suffix="lognormal", suffix_lo=1, suffix_hi=1024, m=5,
              layout="paged"),
        # each page's layout branch decodes beside its content branches,
        # which forked at different positions; prefixes in runs of the pool
        _attn("attn_layout_branches", docs=8, branches_lo=5, branches_hi=25, prefix_lo=1088,
              prefix_hi=3584, suffix="lognormal", suffix_lo=1, suffix_hi=1024, layout="paged_runs",
              fork=True, layout_branch=True),
        # a head ratio of five (40 query heads on 8 KV heads), ragged sizes
        _attn("attn_ratio_five", docs=3, branches_lo=17, branches_hi=41, prefix_lo=911,
              prefix_hi=2600, suffix="lognormal", suffix_lo=1, suffix_hi=1024, m=3, hq=40, hkv=8,
              fork=True),
        # heads of 64 dimensions
        _attn("attn_head_64", docs=6, branches_lo=9, branches_hi=40, prefix_lo=500,
              prefix_hi=4000, suffix="lognormal", suffix_lo=1, suffix_hi=1024, m=4, hq=16, hkv=4,
              d=64),
        # the acceptance alone, with a vocabulary that leaves every row at
        # another alignment
        dict(name="accept_odd_vocab", kind="accept", branches=190, m=5, vocab=50257),
        # the step's rows written to the paged cache and taken back (a step
        # whose drafts were all refused), as many branches as the batch has
        dict(name="kv_append_rollback", kind="kv", branches=768, m=8, hkv=2, d=128,
             suffix_lo=1, suffix_hi=1024, len_seed=2),
        # the fork tokens of a batch's layout branches make new branches
        dict(name="fork_batch", kind="fork", docs=32, branches=24, m=8, max_pages=65, p_fork=0.25,
             len_seed=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


HEADS = ((8, 2, 64), (16, 4, 64), (4, 4, 64), (16, 2, 128), (32, 8, 128), (40, 8, 128),
         (6, 2, 128), (16, 1, 128))


def draw(rng):
    kind = rng.choice(["attn"] * 6 + ["step"] * 2 + ["accept", "kv", "fork"])
    seed = rng.randrange(1 << 30)
    if kind == "accept":
        while True:
            c = dict(kind=kind, branches=_log(rng, 1, 1024), m=rng.randint(1, 16),
                     vocab=_log(rng, 1000, 152000))
            if work(c)["bytes"] <= MAX_BYTES / 2:
                return c
    if kind == "kv":
        return dict(kind=kind, branches=_log(rng, 4, 2048), m=rng.randint(1, 16),
                    hkv=rng.choice([1, 2, 4, 8]), d=rng.choice([64, 128]), suffix_lo=1,
                    suffix_hi=_log(rng, 64, 1024), len_seed=seed)
    if kind == "fork":
        return dict(kind=kind, docs=_log(rng, 1, 64), branches=_log(rng, 1, 64),
                    m=rng.randint(1, 16), max_pages=_log(rng, 4, 129),
                    p_fork=rng.uniform(0.02, 0.4), len_seed=seed)
    while True:
        hq, hkv, d = rng.choice(HEADS)
        layout_branch = rng.random() < 0.15
        p = sorted(_log(rng, 64, 8192) for _ in range(2))
        b = sorted(_log(rng, 2, 256) for _ in range(2))
        c = _attn("", kind=kind, docs=_log(rng, 1, 32), branches_lo=b[0], branches_hi=b[1],
                  prefix_lo=p[0], prefix_hi=p[1],
                  suffix=rng.choice(["uniform", "lognormal", "pareto"]), suffix_lo=1,
                  suffix_hi=_log(rng, 32, 2048), m=rng.randint(1, 8), hq=hq, hkv=hkv, d=d,
                  layout="paged_runs" if layout_branch else
                  rng.choice(["contiguous", "contiguous", "paged", "paged_runs"]),
                  fork=layout_branch or rng.random() < 0.3, layout_branch=layout_branch,
                  vocab=_log(rng, 1000, 64000) if kind == "step" else 0, len_seed=seed)
        del c["name"]
        w = work(c)
        if w["flops"] <= MAX_FLOPS and w["bytes"] <= MAX_BYTES:
            return c


# ------------------------------------------------------------------- lengths --

def _suffixes(rng, case, n):
    lo, hi = case["suffix_lo"], case["suffix_hi"]
    if case.get("suffix") == "uniform":
        return rng.integers(lo, hi + 1, size=n)
    if case.get("suffix") == "pareto":
        return np.clip(np.floor(8.0 * (1.0 + rng.pareto(1.5, size=n))), lo, hi).astype(np.int64)
    return np.clip(np.round(rng.lognormal(4.5, 0.8, size=n)), lo, hi).astype(np.int64)


def _lengths(case):
    """Prefix length and branches of each page, private length (this step's
    m tokens included) and visible prefix of each branch."""
    rng = np.random.default_rng(case["len_seed"])
    docs, m = case["docs"], case["m"]
    P = rng.integers(case["prefix_lo"], case["prefix_hi"] + 1, size=docs)
    C = rng.integers(case["branches_lo"], case["branches_hi"] + 1, size=docs)
    B = int(C.sum())
    L = _suffixes(rng, case, B) + m
    doc = np.repeat(np.arange(docs), C)
    cu = np.concatenate([[0], np.cumsum(C)])
    fork = P[doc].copy()
    if case["fork"]:  # a branch forks in the last third of its page's tokens
        fork = rng.integers(2 * P[doc] // 3, P[doc] + 1)
    if case["layout_branch"]:
        # branch cu[d] is page d's own sequence: its fork prefix is the
        # page-aligned first two thirds, its private pages the rest of the
        # page's run, then its m drafts
        first = cu[:-1]
        fork[first] = (2 * P // 3) // PAGE * PAGE
        L[first] = P + m - fork[first]
    return P, C, cu, doc, L, fork


def _attn_work(case):
    P, C, cu, doc, L, fork = _lengths(case)
    m, hq, hkv, d = case["m"], case["hq"], case["hkv"], case["d"]
    B = len(L)
    seen = np.maximum(L[:, None] - m + 1 + np.arange(m)[None, :], 0).sum()
    flops = 4.0 * d * hq * (float(m) * fork.sum() + seen)
    keys = sum(int(fork[cu[i]:cu[i + 1]].max()) for i in range(len(P))) + int(L.sum())
    io = B * m * hq * (2 * d * 2 + 4)
    tables = 4 * (2 * len(P) + 2 + B * (1 + (1 if case["fork"] else 0)) + int(-(-L // PAGE).sum()))
    return {"bytes": float(keys * hkv * d * 2 * 2 + io + tables), "flops": float(flops)}


def _accept_bytes(B, m, V):
    return float(B * m * V * 2 + B * m * 8 + B * 4)


def work(case):
    k = case["kind"]
    if k == "accept":
        return {"bytes": _accept_bytes(case["branches"], case["m"], case["vocab"]), "flops": 0.0}
    if k == "kv":  # the rows read and written once, K and V
        return {"bytes": float(case["branches"] * (8 * case["m"] * case["hkv"] * case["d"] + 16)),
                "flops": 0.0}
    if k == "fork":
        B, m, mp = case["docs"] * case["branches"], case["m"], case["max_pages"]
        return {"bytes": float(B * (4 * (m + 3) + 4 * 3 + 8 * mp)), "flops": 0.0}
    w = _attn_work(case)
    if k == "step":
        B = int(_lengths(case)[1].sum())
        w["bytes"] += _accept_bytes(B, case["m"], case["vocab"])
    return w


def tolerance(case):
    # attention: 16-bit outputs of sums whose weights are rounded to 16 bits;
    # everything else is whole numbers and copies
    return {"rel": 0.008, "max": 0.045} if case["kind"] in ("attn", "step") else "exact"


# -------------------------------------------------------------------- inputs --

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, shape, std=0.5):
    out = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    flat = out.view(-1)
    step = 1 << 26
    for i in range(0, flat.numel(), step):
        n = min(step, flat.numel() - i)
        flat[i:i + n] = torch.randn(n, generator=g, device="cuda").mul_(std).to(torch.bfloat16)
    return out


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def _attn_inputs(case, seed):
    P, C, cu, doc, L, fork = _lengths(case)
    rng, g = np.random.default_rng(seed), _gen(seed)
    m, hq, hkv, d = case["m"], case["hq"], case["hkv"], case["d"]
    docs, B = len(P), len(L)
    paged = case["layout"] != "contiguous"
    own = -(-L // PAGE)            # private pages of each branch
    first = cu[:-1]
    if case["layout_branch"]:
        own[first] = 0             # those are the page's own
    # pages taken from the pool: each private page by itself; a page's prefix
    # (and its layout branch's drafts) as one run, or page by page
    pre = np.zeros(docs, np.int64)
    if paged:
        pre = -(-(P + (m if case["layout_branch"] else 0)) // PAGE)
    runs = case["layout"] == "paged_runs"
    sizes = np.concatenate([np.ones(int(own.sum()), np.int64),
                            pre if runs else np.ones(int(pre.sum()), np.int64)])
    order = rng.permutation(len(sizes))
    start = np.empty(len(sizes), np.int64)
    start[order] = np.concatenate([[0], np.cumsum(sizes[order])[:-1]])
    pages = max(8, int(sizes.sum()))
    total = -(-L // PAGE)
    max_pages = int(total.max())
    table = rng.integers(0, pages, size=(B, max_pages))
    at = 0
    for b in range(B):
        table[b, :own[b]] = start[at:at + own[b]]
        at += int(own[b])
    ppt = None
    if paged:
        ppt = rng.integers(0, pages, size=(docs, int(pre.max())))
        for i in range(docs):
            if runs:
                ppt[i, :pre[i]] = start[at + i] + np.arange(pre[i])
            else:
                ppt[i, :pre[i]] = start[at:at + pre[i]]
                at += int(pre[i])
    if case["layout_branch"]:
        for i, b in enumerate(first):
            table[b, :total[b]] = ppt[i, fork[b] // PAGE:fork[b] // PAGE + total[b]]
    T = int(P.sum())
    pk = None if paged else _normal(g, (T, hkv, d))
    pv = None if paged else _normal(g, (T, hkv, d))
    return hpd.DeviceInputs(
        q=_normal(g, (B * m, hq, d)), prefix_k=pk, prefix_v=pv,
        prefix_cu=_i32(np.concatenate([[0], np.cumsum(P)])), branch_cu=_i32(cu),
        branch_prefix_len=_i32(fork) if case["fork"] else None,
        k_cache=_normal(g, (pages, PAGE, hkv, d)), v_cache=_normal(g, (pages, PAGE, hkv, d)),
        page_table=_i32(table), branch_len=_i32(L), n_docs=docs, B=B, m=m, H_q=hq, H_kv=hkv, D=d,
        num_pages=pages, max_pages=max_pages, prefix_tokens=T, max_prefix_len=int(P.max()),
        scale=0.0, prefix_page_table=None if ppt is None else _i32(ppt),
        max_prefix_pages=0 if ppt is None else ppt.shape[1])


def _accept_inputs(B, m, V, seed):
    """Logits, and drafts that are the row's argmax seven times in ten."""
    g = _gen(seed + 1)
    logits = _normal(g, (B, m, V), 1.0)
    best = logits.view(B * m, V).float().argmax(1).view(B, m).to(torch.int32) if B * m * V < 1 << 28 \
        else torch.stack([x.float().argmax(1) for x in logits]).to(torch.int32)
    other = torch.randint(0, V, (B, m), generator=g, device="cuda", dtype=torch.int32)
    keep = torch.rand((B, m), generator=g, device="cuda") < 0.7
    return logits, torch.where(keep, best, other).contiguous()


def _kv_inputs(case, seed):
    B, m, hkv, d = case["branches"], case["m"], case["hkv"], case["d"]
    rng, g = np.random.default_rng(seed), _gen(seed)
    L = _suffixes(np.random.default_rng(case["len_seed"]), case, B)
    used = -(-L // PAGE)
    max_pages = int(-(-(case["suffix_hi"] + m) // PAGE))
    pages = int((-(-(L + m) // PAGE)).sum()) + B // 8 + 8
    perm = rng.permutation(pages)
    table = np.full((B, max_pages), -1, np.int64)
    at = 0
    for b in range(B):
        table[b, :used[b]] = perm[at:at + used[b]]
        at += int(used[b])
    free = np.zeros(pages, np.int64)
    free[:pages - at] = perm[at:]
    kv = hpd.PagedKV(_normal(g, (pages, PAGE, hkv, d)), _normal(g, (pages, PAGE, hkv, d)),
                     _i32(table), _i32(L), _i32(free), _i32([pages - at]), m)
    new = (_normal(g, (B, m, hkv, d)), _normal(g, (B, m, hkv, d)))
    return kv, new, _i32(np.full(B, -1))


def _fork_inputs(case, seed):
    """Page d's first branch is its layout branch; its accepted tokens hold a
    fork token with probability p_fork each, a content branch's never do."""
    docs, n, m, mp = case["docs"], case["branches"], case["m"], case["max_pages"]
    rng, sizes = np.random.default_rng(seed), np.random.default_rng(case["len_seed"])
    B = docs * n
    lay = np.zeros(B, np.int64)
    lay[::n] = 1
    tok = rng.integers(FORK_TOKEN + 1, 32000, size=(B, m))
    tok[(lay[:, None] == 1) & (sizes.random((B, m)) < case["p_fork"])] = FORK_TOKEN
    acc = sizes.integers(0, m + 1, size=B)
    emitted = np.arange(m)[None, :] < np.minimum(acc + 1, m)[:, None]
    children = int(((tok == FORK_TOKEN) & emitted).sum())
    L = sizes.integers(1, mp * PAGE + 1, size=B)
    args = dict(out_tokens=_i32(tok), accepted_len=_i32(acc), is_layout=_i32(lay),
                layout_pos=_i32(rng.integers(1024, 3000, size=B)), fork_token=FORK_TOKEN,
                branch_cu=_i32(np.arange(docs + 1) * n),
                branch_prefix_len=_i32(rng.integers(1024, 3000, size=B)), branch_len=_i32(L),
                page_table=_i32(rng.integers(0, B * mp, size=(B, mp))), cap=B + children)
    return args


def prepare(case, seed):
    k = case["kind"]
    if k == "accept":
        logits, drafts = _accept_inputs(case["branches"], case["m"], case["vocab"], seed)
        return dict(kind=k, logits=logits, drafts=drafts)
    if k == "kv":
        kv, new, acc = _kv_inputs(case, seed)
        return dict(kind=k, kv=kv, new=new, acc=acc)
    if k == "fork":
        return dict(kind=k, args=_fork_inputs(case, seed))
    d = _attn_inputs(case, seed)
    st = dict(kind=k, d=d, op=hpd.BranchAttn(d))
    if k == "step":
        logits, drafts = _accept_inputs(d.B, d.m, case["vocab"], seed)
        st.update(logits=logits, drafts=drafts,
                  tokens=torch.empty((d.B, d.m), dtype=torch.int32, device="cuda"),
                  accepted=torch.empty((d.B,), dtype=torch.int32, device="cuda"))
    return st


def run(state):
    k = state["kind"]
    if k == "accept":
        return hpd.pmtp_accept(state["logits"], state["drafts"])
    if k == "kv":
        kv = state["kv"]
        kv.append(*state["new"])
        kv.rollback(state["acc"])
        return (kv.branch_len, kv.page_table, kv.free_pages, kv.free_top, kv.k_cache, kv.v_cache)
    if k == "fork":
        new = hpd.fork_children(**state["args"])
        return {n: v for n, v in new.items() if n != "workspace"}
    if k == "step":
        out, lse = state["op"].step(state["logits"], state["drafts"], state["tokens"],
                                    state["accepted"])
        return out, lse, state["tokens"], state["accepted"]
    return state["op"]()


# -------------------------------------------------------------- in 64 bits --

def exact(case, seed):
    if case["kind"] not in ("attn", "step"):
        return None
    P, C, cu, doc, L, fork = _lengths(case)
    d = _attn_inputs(case, seed)
    m, hq, hkv, D = d.m, d.H_q, d.H_kv, d.D
    G = hq // hkv
    out = torch.zeros((d.B * m, hq, D), dtype=torch.float64, device="cuda")
    lse = torch.full((d.B * m, hq), -math.inf, dtype=torch.float64, device="cuda")
    pcu = np.concatenate([[0], np.cumsum(P)])
    kc, vc = d.k_cache.view(-1, hkv, D), d.v_cache.view(-1, hkv, D)
    slot = torch.arange(PAGE, device="cuda")
    for i in range(len(P)):
        b0, b1 = int(cu[i]), int(cu[i + 1])
        n = b1 - b0
        if d.prefix_page_table is None:
            pk, pv = (x[int(pcu[i]):int(pcu[i + 1])] for x in (d.prefix_k, d.prefix_v))
        else:
            rows = (d.prefix_page_table[i].long()[:, None] * PAGE + slot).reshape(-1)[:int(P[i])]
            pk, pv = kc[rows], vc[rows]
        # private keys, padded to the page's longest branch
        lmax = int(L[b0:b1].max())
        rows = (d.page_table[b0:b1].long()[:, :, None] * PAGE + slot).reshape(n, -1)[:, :lmax]
        Lb, fb = (torch.from_numpy(x[b0:b1].copy()).cuda() for x in (L, fork))
        see_p = torch.arange(int(P[i]), device="cuda")[None, :] < fb[:, None]         # [n, P]
        last = Lb[:, None] - m + torch.arange(m, device="cuda")[None, :]              # [n, m]
        see_s = torch.arange(lmax, device="cuda")[None, None, :] <= last[:, :, None]  # [n, m, l]
        q = d.q[b0 * m:b1 * m].view(n, m, hq, D)
        for h in range(hkv):
            qh = q[:, :, h * G:(h + 1) * G].reshape(n, m * G, D).double()
            sp = torch.matmul(qh.view(-1, D), pk[:, h].double().T).view(n, m * G, -1) / math.sqrt(D)
            sp.masked_fill_(~see_p[:, None, :], -math.inf)
            ss = torch.bmm(qh, kc[rows, h].double().transpose(1, 2)) / math.sqrt(D)
            ss.masked_fill_(~see_s.repeat_interleave(G, dim=1), -math.inf)
            top = torch.maximum(sp.amax(2) if sp.shape[2] else ss.amax(2), ss.amax(2))
            sp, ss = torch.exp(sp - top[:, :, None]), torch.exp(ss - top[:, :, None])
            z = sp.sum(2) + ss.sum(2)
            o = torch.matmul(sp.view(n * m * G, -1), pv[:, h].double()).view(n, m * G, D)
            o = (o + torch.bmm(ss, vc[rows, h].double())) / z[:, :, None]
            out[b0 * m:b1 * m, h * G:(h + 1) * G] = o.view(n * m, G, D)
            lse[b0 * m:b1 * m, h * G:(h + 1) * G] = (top + torch.log(z)).view(n * m, G)
    if case["kind"] == "step":
        return out, lse, None, None
    return out, lse
