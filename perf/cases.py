"""The work a user of this library has it do, as cases that can be timed and compared.

Two programs use the library.  One builds a trimmed vocabulary once per calibration corpus: count the
token ids, select the kept ids, gather the drafter's head (kind "build").  The other drafts tokens all
day: one head call per draft token of a chain ("chain"), one per depth of a draft tree followed by the
rerank and the verification ("tree"), one per step over the rows of many sequences ("batch"), or one
per step with the step's tensors in host memory ("host").

Sizes are those of the test configurations and the benchmark (vocabularies of 4096, 128256 and up to
several hundred thousand ids; hidden sizes 1024-4096; 5000 to 128256 kept ids; 1 to 256 hidden rows; trees of
depth 3-6, top-8 / top-10, 32 or 60 nodes; corpora of 1e5 to 1e9 ids), and odd ones between them.
"""
from __future__ import annotations

import torch

import paper_2506_22694_b200 as vt

DEV = "cuda"


# ---- cases -------------------------------------------------------------------------------------------
def _build(name, n, V, rule, K, d, p=0.0, min_count=0):
    return {"name": name, "kind": "build", "n": n, "V": V, "rule": rule, "K": K, "p": p, "min_count": min_count, "d": d}


def _chain(name, V, d, K, steps, B, topk, sample, mapped=True):
    return {"name": name, "kind": "chain", "V": V, "d": d, "K": K, "steps": steps, "B": B, "topk": topk,
            "sample": sample, "mapped": mapped}


def _tree(name, V, d, K, depth, topk, budget, sample, mapped=True):
    return {"name": name, "kind": "tree", "V": V, "d": d, "K": K, "depth": depth, "topk": topk, "budget": budget,
            "sample": sample, "mapped": mapped}


def _batch(name, V, d, K, B, topk, sample):
    return {"name": name, "kind": "batch", "V": V, "d": d, "K": K, "B": B, "topk": topk, "sample": sample}


def _host(name, V, d, K, B, topk):
    return {"name": name, "kind": "host", "V": V, "d": d, "K": K, "B": B, "topk": topk}


def listed():
    return [
        # a small vocabulary from a small sample: launches and latency are all there is
        _build("build_tiny", 100_000, 4096, "topk", 1024, 256),
        # a fine-tuning set as calibration corpus (a few million tokens): ids down to the one that completes
        # nine tenths of all tokens are kept; the host reads how many before it sizes the trimmed head
        _build("build_calibration", 3_000_017, 128256, "topp", 0, 3072, p=0.9),
        # a vocabulary too large for three counters per shared-memory word
        _build("build_large_vocab", 40_000_003, 256_000, "topk", 20_000, 0),
        # corpus scale, with the gather of the trimmed head
        _build("build_corpus", 1_000_000_000, 128256, "topk", 32768, 4096),
        # small drafter, small head: four draft tokens in a chain, greedy
        _chain("chain_small_head", 128256, 1024, 5000, 4, 1, 8, False),
        # a 3B-class head: seven draft tokens in a chain, greedy with the top-8 log-probabilities
        _chain("chain_3b_head", 128256, 3072, 32768, 7, 1, 8, False),
        # the untrimmed head two sequences at a time, sampled
        _chain("chain_full_head", 128256, 3072, 128256, 3, 2, 8, True, mapped=False),
        # the paper's tree (depth 3, top-8, 32 draft tokens) over an odd-sized head
        _tree("tree_depth3", 128256, 3072, 9_973, 3, 8, 32, False),
        # an 8B-class tree drafter: ten nodes per depth, six depths, sampled
        _tree("tree_8b_head", 128256, 4096, 32768, 6, 10, 60, True),
        # serving a few sequences: more rows than a tree has, an odd number of kept ids
        _batch("batch_40_rows", 128256, 3072, 20_001, 40, 8, True),
        # serving 64 sequences of four tree nodes each
        _batch("batch_256_rows", 128256, 4096, 32768, 256, 8, True),
        # a drafting server whose step tensors live in pinned host memory
        _host("host_step", 128256, 3072, 32768, 4, 8),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def _hidden(rng):
    return rng.choice([1024, 2048, 3072, 4096, 8 * rng.randint(64, 512)])


def draw(rng):
    kind = rng.choice(["build", "build", "build", "chain", "chain", "tree", "tree", "batch", "batch", "batch", "host"])
    V = rng.choice([128256, 128256, _log(rng, 4096, 300_000)])
    d = _hidden(rng)
    K = _log(rng, min(3000, V // 2), min(V, 100_000))
    sample = rng.random() < 0.5
    if kind == "build":
        rule = rng.choice(["topk", "topk", "topp", "minfreq"])
        c = _build("", _log(rng, 100_000, 500_000_000), V, rule, K if rule == "topk" else 0, rng.choice([0, d]),
                   p=round(rng.uniform(0.5, 0.99), 3) if rule == "topp" else 0.0,
                   min_count=_log(rng, 2, 1000) if rule == "minfreq" else 0)
    elif kind == "chain":
        mapped = rng.random() < 0.8
        c = _chain("", V, d, K if mapped else V, rng.randint(3, 7), rng.choice([1, 1, 1, 2, 3, 4, 8]),
                   rng.choice([1, 4, 8, 10, 20]), sample, mapped)
    elif kind == "tree":
        topk = rng.choice([4, 8, 8, 10, 10, 16])
        c = _tree("", V, d, K, rng.randint(3, 6), topk, rng.choice([32, 60]), sample)
    elif kind == "batch":
        c = _batch("", V, d, K, _log(rng, 9, 256), rng.choice([1, 4, 8, 10, 16]), sample)
    else:
        c = _host("", V, d, K, rng.choice([1, 1, 4, 10, 32]), rng.choice([4, 8, 10]))
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _zipf_ids(n, V, s, noise, g):
    """Zipf(s) ranks over a random permutation of the ids, a share `noise` of them replaced by uniform ids."""
    perm = torch.randperm(V, generator=g, device=DEV).to(torch.int32)
    cdf = torch.cumsum(torch.arange(1, V + 1, dtype=torch.float64, device=DEV).pow(-s), 0)
    cdf = (cdf / cdf[-1]).to(torch.float32)
    out = torch.empty(n, dtype=torch.int32, device=DEV)
    for lo in range(0, n, 1 << 26):
        m = min(1 << 26, n - lo)
        r = torch.searchsorted(cdf, torch.rand(m, generator=g, device=DEV)).clamp_(max=V - 1)
        ids = perm[r]
        coin = torch.rand(m, generator=g, device=DEV) < noise
        ids[coin] = torch.randint(0, V, (int(coin.sum()),), generator=g, device=DEV, dtype=torch.int32)
        out[lo:lo + m] = ids
    return out


def _gauss(shape, std, g):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(0.0, std, generator=g)


def _uniforms(shape, g):
    """(2x+1) * 2^-24: representable in fp32 and strictly inside (0, 1)."""
    x = torch.randint(0, 1 << 23, shape, generator=g, device=DEV, dtype=torch.int32)
    return (2.0 * x.to(torch.float32) + 1.0) * 2.0 ** -24


def _outs(B, topk, **kw):
    return (torch.empty((B, 1 + topk), dtype=torch.int32, **kw), torch.empty((B, 1 + topk), dtype=torch.float32, **kw))


def _head(case, seed):
    """The trimmed head and its index map: what a drafter keeps between calls."""
    g = _gen(seed, 1)
    W = _gauss((case["K"], case["d"]), 0.02, g)
    if case.get("mapped", True):
        map_ = torch.randperm(case["V"], generator=g, device=DEV)[:case["K"]].to(torch.int32)
    else:
        map_ = None
    return W, map_


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed, 2)
    if kind == "build":
        n, V, K, d = case["n"], case["V"], case["K"], case["d"]
        ids = _zipf_ids(n, V, 1.07, 0.05, g)
        W = _gauss((V, d), 0.02, g) if d else None
        op = vt.VT_OP_BUILD_VOCAB if case["rule"] == "topk" else vt.VT_OP_HISTOGRAM
        nbytes = max(vt.workspace_bytes(op, n, V, K or V), vt.workspace_bytes(vt.VT_OP_SELECT_TOPK, 0, V, V))
        st = {"case": case, "ids": ids, "W": W, "ws": vt.Workspace(nbytes, DEV)}
        if case["rule"] != "topk":
            # how many ids are kept is known only after the selection: tables that hold any number of them
            st["counts"] = torch.empty(V, dtype=torch.int32, device=DEV)
            st["kept"] = torch.full((V,), -1, dtype=torch.int32, device=DEV)
            st["W_trim"] = torch.zeros((V, d), dtype=torch.bfloat16, device=DEV) if d else None
        return st
    W, map_ = _head(case, seed)
    K, d, topk = case["K"], case["d"], case["topk"]
    if kind == "host":
        B = case["B"]
        h = _gauss((B, d), 1.0, g).cpu().pin_memory()
        T = torch.full((B,), 1.0).pin_memory()
        ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD_HOST, 0, case["V"], K, d, B, topk), DEV)
        return {"case": case, "W": W, "map": map_, "h": h, "T": T, "ws": ws, "out": _outs(B, topk, pin_memory=True)}
    if kind == "tree":
        rows = [1] + [topk] * (case["depth"] - 1)
        temp = (0.7, 0.7)
    else:
        rows = [case["B"]] * case.get("steps", 1)
        temp = (0.5, 1.5) if kind == "batch" else (1.0, 1.0)
    steps = []
    for B in rows:
        h = _gauss((B, d), 1.0, g)
        T = temp[0] + (temp[1] - temp[0]) * torch.rand(B, generator=g, device=DEV)
        u = _uniforms((B, K), g) if case["sample"] else None
        steps.append((h, T, u, _outs(B, topk, device=DEV)))
    nbytes = max(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk) for B in set(rows))
    st = {"case": case, "W": W, "map": map_, "steps": steps, "ws": vt.Workspace(nbytes, DEV)}
    if kind == "tree":
        total = sum(B * topk for B in rows)
        st["pool"] = vt.tree_pool(total, DEV)
        st["n"] = total
        # the target's greedy token after each node: after two nodes in three the token of one of the node's children
        # (drafted once here to know them), else another token
        N = case["budget"]
        target = torch.randint(0, case["V"], (1, N + 1), generator=g, device=DEV, dtype=torch.int32)
        token, parent = (t.tolist() for t in _draft_tree(st)[:2])
        coin = torch.rand(N, generator=g, device=DEV).tolist()
        row = target[0].tolist()
        for i in reversed(range(N)):
            if token[i] >= 0 and coin[i] < 2.0 / 3.0:
                row[parent[i] + 1] = token[i]
        st["target"] = torch.tensor([row], dtype=torch.int32, device=DEV)
    return st


# ---- one pass ----------------------------------------------------------------------------------------
def _draft_tree(s):
    case, W, map_, pool, ws = s["case"], s["W"], s["map"], s["pool"], s["ws"]
    topk, frontier, base = case["topk"], None, 0
    for h, T, u, out in s["steps"]:
        _, _, frontier = vt.vt_draft_head_expand(h, W, map_, T, topk, u, frontier, pool, base, topk, ws=ws, out=out)
        base += h.shape[0] * topk
    nodes, token, parent = vt.vt_tree_rerank(pool, s["n"], case["budget"])
    return token, parent, nodes


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "build":
        if case["rule"] == "topk":
            map_, inv = vt.vt_build_vocab(s["ids"], case["V"], case["K"], ws=s["ws"])
            return map_, inv, vt.vt_trim_head(s["W"], map_, ws=s["ws"]) if case["d"] else None
        counts = vt.vt_histogram(s["ids"], case["V"], counts=s["counts"], ws=s["ws"])
        if case["rule"] == "topp":
            k, map_, inv = vt.vt_select_topp(counts, case["p"], ws=s["ws"])
        else:
            k, map_, inv = vt.vt_select_minfreq(counts, case["min_count"], ws=s["ws"])
        K = int(k)                                         # the host sizes the head by it
        s["kept"][:K].copy_(map_[:K])
        if case["d"]:
            vt.vt_trim_head(s["W"], map_[:K], W_trim=s["W_trim"][:K], ws=s["ws"])
        return counts, k, s["kept"], inv, s["W_trim"]
    if kind == "tree":
        token, parent, nodes = _draft_tree(s)
        N = case["budget"]
        accepted = vt.vt_verify_greedy(token.view(1, N), parent.view(1, N), s["target"])
        return [out for _, _, _, out in s["steps"]], s["pool"], token, parent, nodes, accepted
    if kind == "host":
        vt.vt_draft_head_host(s["h"], s["W"], s["map"], s["T"], case["topk"], None, s["ws"], s["out"])
        torch.cuda.current_stream().synchronize()          # the program reads the ids on the host
        return s["out"]
    return [vt.vt_draft_head(h, s["W"], s["map"], T, case["topk"], u, ws=s["ws"], out=out, overlapped=True)
            for h, T, u, out in s["steps"]]


# ---- what a pass cannot do without -------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "build":
        n, V, d = case["n"], case["V"], case["d"]
        # (how many ids a data-dependent rule keeps is not known here: 0.9 of the tokens of such a stream lie in
        # a quarter of the ids)
        K = case["K"] or V // 4
        return {"bytes": 4.0 * n + 4.0 * (K + V) + 4.0 * K * d, "flops": 0.0}
    K, d, topk = case["K"], case["d"], case["topk"]
    if kind == "tree":
        rows = [1] + [topk] * (case["depth"] - 1)
    elif kind == "host":
        rows = [case["B"]]
    else:
        rows = [case["B"]] * case.get("steps", 1)
    nbytes = flops = 0.0
    for B in rows:                                          # every call reads the head: the next one needs this one's tokens
        nbytes += 2.0 * K * d + 2.0 * B * d + 4.0 * B + 8.0 * B * (1 + topk)
        nbytes += 4.0 * B * K if case.get("sample") else 0.0
        flops += 2.0 * B * K * d
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "build":
        return "exact"                                      # counting, ranking and copying whole numbers and bits
    # bf16 products summed in fp32, log-probabilities from fp32 exponentials.  Against sums in 64 bits they differ by
    # up to 9e-8 (2-norm) and 2.1e-7 (largest) for the few rows of a chain, and by 2.2e-6 and 5.6e-6 where a tile of
    # many rows is summed with fast exponentials; candidates closer than that may change places.
    if case["kind"] == "chain":
        return {"rel": 4e-7, "max": 1e-6, "differ": 0.004}
    return {"rel": 1e-5, "max": 3e-5, "differ": 0.004}
