"""Performance cases: what a decoding program has this library do, over the range it is used on.

Two kinds of case, each one pass through the public entry points of
paper_2607_05722_gb300.nld:

  step      a decoding step's attention and token decision. ``passes`` is a
            string of passes, each running every layer's attention and then
            the decision that follows it: "d" the diffusion draft
            (bidirectional block mask), then top-k unmasking; "v" the causal
            verify pass, then longest-prefix acceptance; "q" the table-mask
            pass of quadratic self-speculation, then acceptance of its drafts.
            ``layers`` layers with a paged KV pool each, since a model runs its
            other layers between two passes over the same pool (the pools of
            one state, or of the rotated states, do not fit in L2). With
            ``stage`` every attention call is preceded by the commit of the
            block's own K/V into the paged cache (so the prefix flag is not
            set), and the step ends with the commit of the accepted rows.
  decide    logits to token decisions: "plain" runs the (argmax, confidence)
            reduction on the draft logits, threshold unmasking on its
            confidences, the reduction on the verify logits and acceptance of
            the draft ids against the verify ids; "ensemble" runs the
            AR-diffusion ensemble verifier and acceptance against its ids.

``graph``: the calls are captured once and replayed, as a decoding loop with
fixed buffers does; without it they are issued one by one.

The lengths of a batch are drawn uniformly from lmin..lmax by the seed;
work() uses their mean. Each attention call and each logits reduction counts
its own inputs: the verify pass needs the draft pass's result.
"""
import math

import numpy as np
import torch

from paper_2607_05722_gb300 import nld

_PAGES = (16, 16, 32, 64, 128, 256)
_VOCABS = (32000, 32001, 50257, 65536, 100003, 131072)


def _step(name, passes, batch, hq, hkv, d, page, bl, lmin, lmax, layers=1, k=4, stage=False, graph=True):
    return {"name": name, "kind": "step", "passes": passes, "batch": batch, "hq": hq, "hkv": hkv, "d": d,
            "page": page, "bl": bl, "lmin": lmin, "lmax": lmax, "layers": layers, "k": k, "stage": stage,
            "graph": graph}


def _decide(name, what, batch, n, vocab, graph=True):
    return {"name": name, "kind": "decide", "what": what, "batch": batch, "n": n, "vocab": vocab, "graph": graph}


def listed():
    return [
        # The smallest program: one sequence, one KV head, head_dim 64, a
        # 256-token page of prefix, four calls issued one by one. Launch and
        # call overhead is what it pays for.
        _step("tiny_step_calls", "dv", 1, 4, 1, 64, 256, 8, 256, 256, k=2, graph=False),
        # One user of an 8B-class model (32 query heads over 8 KV heads): the
        # draft and the verify pass of a block of 16 over 4096 cached tokens,
        # 16 layers with a pool each, unmasking and acceptance.
        _step("8b_step_16_layers", "dv", 1, 32, 8, 128, 16, 16, 4096, 4096, layers=16),
        # The same model late in a long context: the verify pass of a block of
        # 32 (128 packed rows per KV head) over 32768 tokens, two layers.
        _step("long_verify_32k", "v", 1, 32, 8, 128, 16, 32, 32768, 32768, layers=2),
        # A 14B-class model (40 query heads over 8) serving 16 sequences of
        # 8192..16384 tokens: one denoising pass of a block of 32.
        _step("14b_draft_b16", "d", 16, 40, 8, 128, 16, 32, 8192, 16384, k=8, graph=False),
        # Ragged serving batches of the 8B heads, blocks of 8: few sequences,
        # a middle size and the largest.
        _step("serve_verify_b8", "v", 8, 32, 8, 128, 16, 8, 512, 8192),
        _step("serve_verify_b32", "v", 32, 32, 8, 128, 16, 8, 512, 8192),
        _step("serve_verify_b128", "v", 128, 32, 8, 128, 16, 8, 512, 8192, graph=False),
        # A serving step that also stages the block's K/V in the cache before
        # it attends and commits the accepted rows after it; pages of 64.
        _step("serve_commit_b24", "v", 24, 32, 8, 128, 64, 16, 256, 4096, stage=True),
        # Quadratic self-speculation with k = 3 (13 block slots, 52 packed
        # rows) on the 8B heads, an odd prefix length, 8 layers.
        _step("quadss_k3_8_layers", "q", 1, 32, 8, 128, 16, 13, 4093, 4093, layers=8, k=3),
        # One block's logits to its decisions: 16 rows of a 131072-entry
        # vocabulary, twice.
        _decide("decide_16_rows", "plain", 1, 16, 131072),
        # The same for a serving batch of 64 sequences, blocks of 8.
        _decide("decide_512_rows", "plain", 64, 8, 131072),
        # The ensemble verifier for 32 sequences of k = 5 speculative tokens,
        # a vocabulary that is not a multiple of 8.
        _decide("ensemble_160_rows", "ensemble", 32, 5, 100003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "decide"))
    if kind == "decide":
        what = rng.choice(("plain", "plain", "ensemble"))
        vocab = rng.choice(_VOCABS)
        n = rng.randint(1, 32) if what == "plain" else rng.randint(1, 5)
        batch = min(_log_int(rng, 1, 128), max(1, 1024 // n))
        c = _decide("", what, batch, n, vocab, rng.random() < 0.7)
    else:
        d = rng.choice((128, 128, 128, 64))
        group, hkv = rng.choice(((4, 8), (4, 8), (5, 8), (8, 4), (2, 8), (1, 8), (7, 4), (4, 1)))
        passes = rng.choice(("dv", "d", "v", "v", "q"))
        if passes == "q":
            k = rng.randint(1, 5)
            bl = 1 + k + k * k
            if group * bl > 256:
                group = 5
        else:
            bl = rng.randint(1, 256 // group if group > 8 else 32)
            k = rng.randint(1, bl)
        batch = _log_int(rng, 1, 96)
        lmax = _log_int(rng, 64, 32768)
        # at most 400 MB of keys and values a layer
        lmax = max(64, min(lmax, int(4e8 / (batch * hkv * d * 4))))
        lmin = rng.choice((lmax, max(1, lmax // 2), max(1, lmax // 16)))
        layers = max(1, min(8, int(2e8 / (batch * hkv * d * 4 * lmax)))) if passes != "dv" else 2
        c = _step("", passes, batch, group * hkv, hkv, d, rng.choice(_PAGES), bl, lmin, lmax, layers, k,
                  rng.random() < 0.25, rng.random() < 0.7)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _normal(gen, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)


def _lengths(case, rng):
    return rng.integers(case["lmin"], case["lmax"], size=case["batch"], endpoint=True).astype(np.int32)


def _ids(rng, batch, n, p_agree, vocab=131072):
    draft = rng.integers(0, vocab, size=(batch, n))
    other = rng.integers(0, vocab - 1, size=(batch, n))
    verify = np.where(rng.random((batch, n)) < p_agree, draft, other + (other >= draft))
    return draft.astype(np.int32), verify.astype(np.int32)


def _table(lens, lmax, bl, page, rng):
    """Every sequence's pages scattered over one pool, -1 past its last page.
    The pool and the table have room for every sequence at lmax tokens."""
    need = [-(-(int(x) + bl) // page) for x in lens]
    width = -(-(lmax + bl) // page)
    order = rng.permutation(len(need) * width).astype(np.int32)
    table = np.full((len(need), width), -1, dtype=np.int32)
    at = 0
    for b, m in enumerate(need):
        table[b, :m] = order[at:at + m]
        at += m
    return table, order.size


def _step_inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, bl, hq, hkv, d, page = (case[x] for x in ("batch", "bl", "hq", "hkv", "d", "page"))
    lens = _lengths(case, rng)
    table, pages = _table(lens, case["lmax"], bl, page, rng)
    n = case["k"] if "q" in case["passes"] else bl
    draft, verify = _ids(rng, B, n, 0.75)
    s = {"case": case, "bl": bl,
         "lens": torch.from_numpy(lens).cuda(), "table": torch.from_numpy(table).cuda(),
         "draft": torch.from_numpy(draft).cuda(), "verify": torch.from_numpy(verify).cuda(),
         "conf": torch.from_numpy(rng.random((B, bl), dtype=np.float32)).cuda(),
         "k_pages": [_normal(gen, pages, hkv, page, d) for _ in range(case["layers"])],
         "v_pages": [_normal(gen, pages, hkv, page, d) for _ in range(case["layers"])],
         "q": {p: [_normal(gen, B, bl, hq, d) for _ in range(case["layers"])] for p in case["passes"]}}
    if case["stage"]:
        s["k_new"] = [_normal(gen, B, bl, hkv, d) for _ in range(case["layers"])]
        s["v_new"] = [_normal(gen, B, bl, hkv, d) for _ in range(case["layers"])]
    return s


def _peaked_logits(gen, rng, rows, vocab, peak):
    """Unit-normal logits with one token per row raised, so that confidences
    spread over (0, 1) as a model's do. Rows are padded to a multiple of 8."""
    ld = -(-vocab // 8) * 8
    x = _normal(gen, rows, ld)
    up = torch.from_numpy(rng.uniform(6.0, 18.0, size=rows)).to(device="cuda", dtype=torch.bfloat16)
    x[torch.arange(rows, device="cuda"), torch.from_numpy(peak).cuda().long()] = up
    return x


def _decide_inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, n, vocab = case["batch"], case["n"], case["vocab"]
    draft, verify = _ids(rng, B, n, 0.75, vocab)
    if case["what"] == "ensemble":
        # the causal and the denoising row agree on most positions
        _, other = _ids(rng, B, n, 0.75, vocab)
        second = np.where(rng.random((B, n)) < 0.75, verify, other)
        a = _peaked_logits(gen, rng, B * n, vocab, verify.reshape(-1))
        b = _peaked_logits(gen, rng, B * n, vocab, second.reshape(-1))
    else:
        a = _peaked_logits(gen, rng, B * n, vocab, draft.reshape(-1))
        b = _peaked_logits(gen, rng, B * n, vocab, verify.reshape(-1))
    return {"case": case, "a": a, "b": b, "draft": torch.from_numpy(draft).cuda()}


_LAMBDA = 0.5
_THRESHOLD = 0.9


# ---------------------------------------------------------------------------
# The passes
# ---------------------------------------------------------------------------

_MODES = {"d": nld.NLD_MODE_DIFFUSION, "v": nld.NLD_MODE_VERIFY}


def _empty(*shape, dtype=torch.int32):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _prepare_step(case, seed):
    s = _step_inputs(case, seed)
    B, bl, hq, d, layers = (case[x] for x in ("batch", "bl", "hq", "d", "layers"))
    flags = 0 if case["stage"] else nld.NLD_ATTN_PREFIX_READY
    s["params"] = nld.params_for(s["q"][case["passes"][0]][0], s["k_pages"][0], s["table"], flags=flags)
    s["ws"] = nld.alloc_workspace(s["params"], bl)
    if "q" in case["passes"]:
        s["mask"] = torch.from_numpy(nld.nld_quadss_block_mask(case["k"]).view(np.int32)).cuda()
    s["out"] = {p: {"out": _empty(layers, B, bl, hq, d, dtype=torch.bfloat16),
                    "lse": _empty(layers, B, hq, bl, dtype=torch.float32)} for p in case["passes"]}
    for p in case["passes"]:
        if p == "d":
            s["out"][p]["positions"] = _empty(B, case["k"])
            s["out"][p]["selected"] = _empty(B)
        else:
            s["out"][p]["accepted"] = _empty(B)
    return s


def _run_step(s):
    case, bl, prm = s["case"], s["bl"], s["params"]
    got = s["out"]
    for p in case["passes"]:
        o = got[p]
        for i in range(case["layers"]):
            k, v = s["k_pages"][i], s["v_pages"][i]
            if case["stage"]:
                nld.nld_kv_commit(prm, s["k_new"][i], s["v_new"][i], None, s["table"], s["lens"], bl, False, k, v)
            if p == "q":
                nld.nld_block_attn_masked(prm, s["q"][p][i], k, v, s["table"], s["lens"], bl, s["mask"],
                                          o["out"][i], o["lse"][i], s["ws"])
            else:
                nld.nld_block_attn(prm, s["q"][p][i], k, v, s["table"], s["lens"], bl, _MODES[p], o["out"][i],
                                   o["lse"][i], s["ws"])
        if p == "d":
            nld.nld_unmask(s["conf"], case["k"], o["positions"], o["selected"])
        else:
            nld.nld_accept(s["draft"], s["verify"], o["accepted"])
            if case["stage"]:
                for i in range(case["layers"]):
                    nld.nld_kv_commit(prm, s["k_new"][i], s["v_new"][i], o["accepted"], s["table"], s["lens"], bl,
                                      False, s["k_pages"][i], s["v_pages"][i])
    if case["stage"]:
        return [got, s["k_pages"], s["v_pages"]]
    return [got]


def _prepare_decide(case, seed):
    s = _decide_inputs(case, seed)
    B, n = case["batch"], case["n"]
    out = {"ids": _empty(B * n), "conf": _empty(B * n, dtype=torch.float32), "accepted": _empty(B)}
    if case["what"] == "plain":
        out.update(first_ids=_empty(B * n), first_conf=_empty(B * n, dtype=torch.float32), positions=_empty(B, n),
                   selected=_empty(B))
    s["out"] = out
    return s


def _run_decide(s):
    case, o = s["case"], s["out"]
    B, n, vocab = case["batch"], case["n"], case["vocab"]
    if case["what"] == "plain":
        nld.nld_logits_argmax(s["a"], o["first_ids"], o["first_conf"], vocab)
        nld.nld_unmask_threshold(o["first_conf"].view(B, n), _THRESHOLD, o["positions"], o["selected"])
        nld.nld_logits_argmax(s["b"], o["ids"], o["conf"], vocab)
        nld.nld_accept(o["first_ids"].view(B, n), o["ids"].view(B, n), o["accepted"])
    else:
        nld.nld_logits_ensemble_argmax(s["a"], s["b"], _LAMBDA, o["ids"], o["conf"], vocab)
        nld.nld_accept(s["draft"], o["ids"].view(B, n), o["accepted"])
    return [o]


def _calls(s):
    return _run_step(s) if s["case"]["kind"] == "step" else _run_decide(s)


def prepare(case, seed):
    s = _prepare_step(case, seed) if case["kind"] == "step" else _prepare_decide(case, seed)
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _calls(s)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["returned"] = _calls(s)
    return s


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["returned"]
    return _calls(state)


# ---------------------------------------------------------------------------
# What a pass cannot do without, how exact it is, and its result in 64 bits
# ---------------------------------------------------------------------------

def work(case):
    if case["kind"] == "decide":
        rows = case["batch"] * case["n"]
        return {"bytes": 2 * rows * case["vocab"] * 2 + 4 * rows * 4, "flops": 0}
    B, bl, hq, hkv, d = (case[x] for x in ("batch", "bl", "hq", "hkv", "d"))
    tokens = B * ((case["lmin"] + case["lmax"]) / 2 + bl)
    kv = tokens * hkv * d * 2 * 2
    q_out = 2 * B * bl * hq * d * 2 + 4 * B * bl * hq
    block = B * bl * hkv * d * 2 * 2
    calls = case["layers"] * len(case["passes"])
    per_call = kv + q_out + (3 * block if case["stage"] else 0)
    return {"bytes": calls * per_call, "flops": calls * 4.0 * tokens * bl * hq * d}


def tolerance(case):
    if case["kind"] == "decide":
        return {"rel": 2e-5, "max": 2e-4, "differ": 0.01}
    # bf16 probabilities and outputs
    return {"rel": 1.2e-2, "max": 0.15}


def _exact_attention(s, p, i):
    case = s["case"]
    B, bl, hq, hkv, d, page = (case[x] for x in ("batch", "bl", "hq", "hkv", "d", "page"))
    G = hq // hkv
    out = torch.empty((B, bl, hq, d), dtype=torch.float64, device="cuda")
    lse = torch.empty((B, hq, bl), dtype=torch.float64, device="cuda")
    slot = torch.arange(bl, device="cuda")
    if p == "v":
        block = slot[None, :] <= slot[:, None]
    elif p == "d":
        block = torch.ones((bl, bl), dtype=torch.bool, device="cuda")
    else:
        # the chain (slot 0 and each group's first slot) is causal and sees no
        # mask slot; a group's k masks see the chain up to it and each other
        k = case["k"]
        spec = [0] + [1 + g * (k + 1) for g in range(k)]
        block = torch.zeros((bl, bl), dtype=torch.bool, device="cuda")
        for a, row in enumerate(spec):
            block[row, spec[:a + 1]] = True
            if a:
                for r in range(row + 1, row + 1 + k):
                    block[r, spec[:a + 1]] = True
                    block[r, row + 1:row + 1 + k] = True
    for b in range(B):
        L = int(s["lens"][b])
        T = L + bl
        pages = s["table"][b, :-(-T // page)].long()
        key, val = (x[i][pages].transpose(1, 2).reshape(-1, hkv, d)[:T].clone() for x in (s["k_pages"], s["v_pages"]))
        if case["stage"]:
            key[L:] = s["k_new"][i][b]
            val[L:] = s["v_new"][i][b]
        key, val = (x.transpose(0, 1).double() for x in (key, val))
        q = s["q"][p][i][b].double().view(bl, hkv, G, d).permute(1, 2, 0, 3).reshape(hkv, G * bl, d)
        x = torch.matmul(q, key.transpose(1, 2)) / math.sqrt(d)
        x = x.view(hkv, G, bl, T)
        x[..., L:].masked_fill_(~block, -math.inf)
        m = torch.logsumexp(x, -1)
        o = torch.matmul(torch.exp(x - m[..., None]).view(hkv, G * bl, T), val).view(hkv, G, bl, d)
        out[b] = o.permute(2, 0, 1, 3).reshape(bl, hq, d)
        lse[b] = m.view(hq, bl)
    return out, lse


def exact(case, seed):
    if case["kind"] == "decide":
        s = _decide_inputs(case, seed)
        vocab = case["vocab"]

        def softmax(x):
            return [torch.softmax(x[r:r + 16, :vocab].double(), -1) for r in range(0, x.shape[0], 16)]

        if case["what"] == "plain":
            return [{"ids": None, "conf": torch.cat([p.amax(-1) for p in softmax(s["b"])]), "accepted": None,
                     "first_ids": None, "first_conf": torch.cat([p.amax(-1) for p in softmax(s["a"])]),
                     "positions": None, "selected": None}]
        mix = torch.cat([(_LAMBDA * p + (1 - _LAMBDA) * q).amax(-1) for p, q in zip(softmax(s["a"]), softmax(s["b"]))])
        return [{"ids": None, "conf": mix, "accepted": None}]
    s = _step_inputs(case, seed)
    got = {}
    for p in case["passes"]:
        each = [_exact_attention(s, p, i) for i in range(case["layers"])]
        got[p] = {"out": torch.stack([x[0] for x in each]), "lse": torch.stack([x[1] for x in each])}
        got[p].update({"positions": None, "selected": None} if p == "d" else {"accepted": None})
    return [got, None, None] if case["stage"] else [got]
