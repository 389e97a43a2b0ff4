"""The work a decoding program has this library do, as cases to be timed and compared.

Five kinds of pass, each through the public entry points of the package:

* ``step``    one speculative block with static draft trees: the draft lists of every drafted
              context (encode side), then the target race, the walk and the scores (decode side);
              optionally top-k / top-p truncated, DISTINCT or IID lists, bf16 or fp32 logits;
* ``tree``    the dynamic IID tree: gamma sequential draft calls and expansions, then the verify;
* ``hetero``  the tree of B non-identical proposals, the same way;
* ``lmhead``  a step whose logits never reach memory: hidden states and LM-head matrices in;
* ``detect``  the detector over texts: per-token scores, per-text sums and log p-values.

Inputs are the synthetic decoding workloads of ``paper_2609_21858_gb300.synth``.  ``exact`` restates
every pass in plain torch / numpy, 64-bit, from the definitions (keyed Philox words, race keys
s = ln E - l / T, multi-arrival scores, truncation, walk, scores, null laws).
"""
import math

import numpy as np
import torch

from paper_2609_21858_gb300 import pps, synth
from paper_2609_21858_gb300.tree import HeteroTreeBuilder, TreeBuilder

DEV = "cuda"


def _step(name, family, n_seq, vocab, K, gamma, dtype="bf16", mode="distinct", temperature=1.0, top_k=0, top_p=1.0,
          static=False):
    case = {"kind": "step", "family": family, "n_seq": n_seq, "vocab": vocab, "K": K, "gamma": gamma, "dtype": dtype,
            "mode": mode, "temperature": temperature, "top_k": top_k, "top_p": top_p, "static": static}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest call: 64 short sequences of a toy vocabulary; launches and latency
        _step("tiny_fp32", "tiny", 64, 1000, 2, 1, dtype="fp32"),
        # a small-vocabulary model (V = 32000), 8 sequences of 4 chains: an ordinary small server batch
        _step("chain4x4_bf16", "chain4x4", 8, 32000, 4, 4),
        # one interactive sequence of a 128k-vocabulary model: latency of a batch of 41 rows
        _step("one_sequence_bf16", "zipf_k8", 1, 128256, 8, 5),
        # the benchmark's step: 64 sequences, 8 chains of 5, every draft and node row in bf16
        _step("zipf_k8_bf16", "zipf_k8", 64, 128256, 8, 5),
        # a vocabulary grown by one token (V = 32001): contiguous bf16 rows that start on odd offsets
        _step("odd_vocab_iid_bf16", "zipf_k8", 24, 32001, 6, 4, mode="iid"),
        # fp32 logits over the largest vocabulary, wide static branching (16, 3, 2, 1)
        _step("branch16_fp32", "branch16", 16, 152064, 16, 4, dtype="fp32", static=True),
        # the experiments' logit processing: top-k 50 before the race, the benchmark's batch
        _step("top50_bf16", "zipf_k8", 64, 128256, 8, 5, top_k=50),
        # the paper's own drafting: dynamic trees of IID samples, five sequential depths
        {"name": "iid_tree_bf16", "kind": "tree", "n_seq": 64, "vocab": 128256, "K": 8, "gamma": 5,
         "temperature": 1.0},
        # eight different draft models proposing chains
        {"name": "hetero_bf16", "kind": "hetero", "n_seq": 64, "vocab": 128256, "K": 8, "gamma": 5,
         "temperature": 1.0},
        # the LM heads of one sequence (41 target rows of d = 4096, 33 draft rows of d = 2048): a decode step
        {"name": "lmhead_one_sequence", "kind": "lmhead", "n_seq": 1, "vocab": 128256, "K": 8, "gamma": 5,
         "d_target": 4096, "d_draft": 2048, "mode": "distinct", "temperature": 1.0},
        # the LM heads of a full batch: 2624 and 2112 rows
        {"name": "lmhead_64", "kind": "lmhead", "n_seq": 64, "vocab": 128256, "K": 8, "gamma": 5, "d_target": 4096,
         "d_draft": 2048, "mode": "distinct", "temperature": 1.0},
        # scanning a corpus for the watermark: 10^7 tokens of texts of 128, half of them watermarked
        {"name": "detect_1e7", "kind": "detect", "n": 10_000_000, "text": 128, "ragged": False, "score": "aaronson"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_vocab(rng, lo, hi):
    v = _log_int(rng, lo, hi)
    return max(lo, min(hi, v - v % 64 if rng.random() < 0.5 else v))  # padded vocabularies and any others


def draw(rng):
    kind = rng.choice(["step", "step", "step", "tree", "hetero", "lmhead", "detect"])
    temperature = rng.choice([0.6, 1.0, 1.0, 1.7])
    n_seq = _log_int(rng, 1, 64)
    if kind == "step":
        vocab, dtype = _draw_vocab(rng, 1000, 152064), rng.choice(["bf16", "bf16", "fp32"])
        static = rng.random() < 0.25
        K, gamma = (16, 4) if static else (_log_int(rng, 1, 32), rng.randint(1, 5))
        family = "branch16" if static else rng.choice(["zipf_k8", "chain4x4"])
        top_k, top_p = rng.choice([(0, 1.0), (0, 1.0), (0, 1.0), (50, 1.0), (rng.randint(1, 64), 0.9)])
        case = _step("", family, n_seq, vocab, K, gamma, dtype, rng.choice(["distinct", "iid"]), temperature, top_k,
                     top_p, static)
        while case["n_seq"] > 1 and work(case)["bytes"] > 3.5e9:
            case["n_seq"] = case["n_seq"] * 2 // 3
        return case
    if kind in ("tree", "hetero"):
        return {"kind": kind, "n_seq": n_seq, "vocab": _draw_vocab(rng, 1000, 128256), "K": rng.randint(2, 8),
                "gamma": rng.randint(2, 5), "temperature": temperature}
    if kind == "lmhead":
        d = 8 * rng.randint(64, 512)
        return {"kind": kind, "n_seq": n_seq, "vocab": _draw_vocab(rng, 32000, 128256), "K": rng.randint(1, 8),
                "gamma": rng.randint(1, 5), "d_target": d, "d_draft": 8 * rng.randint(32, d // 8),
                "mode": rng.choice(["distinct", "iid"]), "temperature": temperature}
    return {"kind": kind, "n": _log_int(rng, 10_000, 10_000_000), "text": _log_int(rng, 32, 4096), "ragged": True,
            "score": rng.choice(["aaronson", "aaronson", "u", "li", "power"])}


# ---------------------------------------------------------------- inputs

class _State:
    pass


def _gpu(x):
    return torch.as_tensor(x).to(DEV).contiguous()


def _branching(case):
    return (16, 3, 2, 1) if case.get("static") else (case["K"],) + (1,) * (case["gamma"] - 1)


def _lists_out(n, K):
    e = lambda *s, dt=torch.int32: torch.empty(*s, dtype=dt, device=DEV)  # noqa: E731
    return dict(tok=e(n, K), key=e(n, K, dt=torch.float32), mult=e(n, K), ndist=e(n), samples=e(n, K))


def _walk_out(n, n_seq, W):
    e = lambda *s, dt=torch.int32: torch.empty(*s, dtype=dt, device=DEV)  # noqa: E731
    return dict(winner=e(n), word=e(n), accept_len=e(n_seq), n_emitted=e(n_seq), emitted=e(n_seq, W),
                score=e(n_seq, W, dt=torch.float32), score_sum=e(n_seq, dt=torch.float64))


def _topology(s, tree):
    s.gamma, s.K, s.n_seq = tree.gamma, tree.K, tree.n_seq
    s.seq_off, s.node_draft_row = _gpu(tree.seq_off), _gpu(tree.node_draft_row)
    s.row_k, s.child_node = _gpu(tree.row_k), _gpu(tree.child_node)
    s.draft, s.walk = _lists_out(tree.n_draft, tree.K), _walk_out(tree.n_nodes, tree.n_seq, tree.gamma + 1)
    s.status = torch.zeros(1, dtype=torch.int32, device=DEV)


def _zipf_rows(gen, rows, vocab):
    """bf16 logits -ln(rank) + N(0, 1), the ranks permuted per row."""
    out = torch.empty(rows, vocab, dtype=torch.bfloat16, device=DEV)
    base = -torch.log(torch.arange(1, vocab + 1, device=DEV, dtype=torch.float32))
    step = max(1, (1 << 26) // vocab)
    for r in range(0, rows, step):
        m = min(step, rows - r)
        perm = torch.argsort(torch.rand(m, vocab, generator=gen, device=DEV), dim=1)
        out[r:r + m] = (base[perm] + torch.randn(m, vocab, generator=gen, device=DEV)).to(torch.bfloat16)
    return out


def _ints(gen, n, bits):
    return torch.randint(0, 2 ** bits, (n,), generator=gen, device=DEV, dtype=torch.int64)


def _prepare_step(case, seed):
    s = _State()
    wl = synth.make_workload(case["family"], device=DEV, n_seq=case["n_seq"], vocab=case["vocab"],
                             branching=_branching(case), seed=seed,
                             dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)
    _topology(s, wl.tree)
    s.q, s.p = wl.q_logits.contiguous(), wl.p_logits.contiguous()
    s.draft_ids = (wl.draft_key.contiguous(), wl.draft_ctx.contiguous(), wl.draft_pos.contiguous())
    s.node_ids = (wl.node_key, wl.node_ctx, wl.node_pos)
    s.ws_q, s.ws_p = pps.workspace(wl.tree.n_draft), pps.workspace(wl.tree.n_nodes, wl.tree.n_seq)
    return s


def _run_step(case, s):
    d = pps.draft_list(s.q, *s.draft_ids, s.K, row_k=s.row_k, mode=pps.IID if case["mode"] == "iid" else pps.DISTINCT,
                       temperature=case["temperature"], ws=s.ws_q, status=s.status, out=s.draft, top_k=case["top_k"],
                       top_p=case["top_p"])
    v = pps.verify_tree(s.p, *s.node_ids, s.gamma, s.seq_off, s.node_draft_row, d["tok"], d["ndist"], s.child_node,
                        temperature=case["temperature"], ws=s.ws_p, status=s.status, out=s.walk,
                        top_k=case["top_k"], top_p=case["top_p"])
    return {"draft": d, "walk": v, "status": s.status}


def _prepare_tree(case, seed):
    s = _State()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n_seq, K, gamma, V = case["n_seq"], case["K"], case["gamma"], case["vocab"]
    hetero = case["kind"] == "hetero"
    s.builder = (HeteroTreeBuilder if hetero else TreeBuilder)(n_seq, K, gamma, DEV)
    s.n_nodes = s.builder.n_nodes
    # the draft models' logits of every depth's rows, and the target model's of every node slot
    s.depth_logits = [_zipf_rows(gen, n_seq * (K if hetero or d else 1), V) for d in range(gamma)]
    s.p = _zipf_rows(gen, s.n_nodes, V)
    s.root = (_ints(gen, n_seq, 62), _ints(gen, n_seq, 62), _ints(gen, n_seq, 12).to(torch.int32))
    s.ws, s.walk = pps.workspace(s.n_nodes, n_seq), _walk_out(s.n_nodes, n_seq, gamma + 1)
    s.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    return s


def _run_tree(case, s):
    b = s.builder.run(*s.root, lambda depth, *ids: s.depth_logits[depth], temperature=case["temperature"])
    v = b.verify(s.p, temperature=case["temperature"], ws=s.ws, out=s.walk, status=s.status)
    if case["kind"] == "hetero":
        lists = {"tok": b.list_tok, "ndist": b.list_nd, "drawn": b.draft_tok}
    else:
        lists = {"tok": b.draft_tok, "mult": b.draft_mult, "ndist": b.draft_ndist}
    return {"lists": lists, "child": b.child_node, "node_ctx": b.node_ctx, "walk": v, "status": s.status}


def _prepare_lmhead(case, seed):
    s = _State()
    wl = synth.lmhead_workload(n_seq=case["n_seq"], branching=_branching(case), vocab=case["vocab"],
                               d_target=case["d_target"], d_draft=case["d_draft"], seed=seed, device=DEV)
    _topology(s, wl.tree)
    s.hp, s.wp, s.hq, s.wq = (x.contiguous() for x in (wl.hp, wl.wp, wl.hq, wl.wq))
    s.draft_ids = (wl.draft_key.contiguous(), wl.draft_ctx.contiguous(), wl.draft_pos.contiguous())
    s.node_ids = (wl.node_key, wl.node_ctx, wl.node_pos)
    s.ws_q, s.ws_p = pps.lmhead_workspace(wl.tree.n_draft), pps.lmhead_workspace(wl.tree.n_nodes, wl.tree.n_seq)
    return s


def _run_lmhead(case, s):
    d = pps.lmhead_draft_list(s.hq, s.wq, *s.draft_ids, s.K, row_k=s.row_k,
                              mode=pps.IID if case["mode"] == "iid" else pps.DISTINCT,
                              temperature=case["temperature"], ws=s.ws_q, status=s.status, out=s.draft)
    v = pps.lmhead_verify_tree(s.hp, s.wp, *s.node_ids, s.gamma, s.seq_off, s.node_draft_row, d["tok"], d["ndist"],
                               s.child_node, temperature=case["temperature"], ws=s.ws_p, status=s.status, out=s.walk)
    return {"draft": d, "walk": v, "status": s.status}


_SCORES = {"aaronson": (pps.SCORE_AARONSON, 0.0), "u": (pps.SCORE_U, 0.0), "li": (pps.SCORE_LI, 0.1),
           "power": (pps.SCORE_POWER_LAW, 0.05)}


def _prepare_detect(case, seed):
    s = _State()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n, text = case["n"], case["text"]
    if case["ragged"]:  # as many texts as the mean length gives, of any length from 1 up
        m = max(1, n // text)
        cut = torch.sort(torch.randint(0, n - m + 1, (m - 1,), generator=gen, device=DEV)).values
        cut = cut + torch.arange(1, m, device=DEV)
        off = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), cut, torch.full((1,), n, device=DEV)])
    else:
        off = torch.arange(0, n + text, text, device=DEV, dtype=torch.int64).clamp_max_(n)
    s.seg_off = off.contiguous()
    length = off[1:] - off[:-1]
    s.key = torch.repeat_interleave(_ints(gen, length.numel(), 62), length).contiguous()  # one key per text
    s.ctx = _ints(gen, n, 62)
    s.pos = _ints(gen, n, 30).to(torch.int32)
    s.tok = torch.randint(0, 128256, (n,), generator=gen, device=DEV, dtype=torch.int64)
    # the first half is watermarked: each token the race winner among eight equally likely ones
    half = n // 2
    for a in range(0, half, 1 << 20):
        b = min(half, a + (1 << 20))
        best, word = s.tok[a:b].clone(), _word(s.tok[a:b], s.key[a:b], s.ctx[a:b], s.pos[a:b])
        for _ in range(7):
            t = torch.randint(0, 128256, (b - a,), generator=gen, device=DEV, dtype=torch.int64)
            w = _word(t, s.key[a:b], s.ctx[a:b], s.pos[a:b])
            best, word = torch.where(w > word, t, best), torch.maximum(w, word)
        s.tok[a:b] = best
    s.tok = s.tok.to(torch.int32)
    return s


def _run_detect(case, s):
    kind, param = _SCORES[case["score"]]
    score, sums, logp = pps.wm_detect(s.tok, s.key, s.ctx, s.pos, s.seg_off, kind=kind, param=param)
    return {"score": score, "sum": sums, "logp": logp}


_KINDS = {"step": (_prepare_step, _run_step), "tree": (_prepare_tree, _run_tree),
          "hetero": (_prepare_tree, _run_tree), "lmhead": (_prepare_lmhead, _run_lmhead),
          "detect": (_prepare_detect, _run_detect)}


def prepare(case, seed):
    s = _KINDS[case["kind"]][0](case, seed)
    s.case = case
    return s


def run(state):
    return _KINDS[state.case["kind"]][1](state.case, state)


def _rows(case):
    """(node rows, draft rows, list stride) of a case's trees."""
    K, n_seq = case["K"], case["n_seq"]
    if case["kind"] in ("tree", "hetero"):
        wide = K if case["kind"] == "hetero" else 1
        return n_seq * (1 + K * case["gamma"]), n_seq * (wide + K * (case["gamma"] - 1)), K
    nodes, draft, at = 1, 0, 1
    for b in _branching(case):
        draft += at
        at *= b
        nodes += at
    return nodes * n_seq, draft * n_seq, K


def work(case):
    """Bytes: every logit (or operand), identity and topology entry read once, every output written
    once.  Flops: the LM heads' products; the other kinds do integer work (a Philox block per four
    tokens, or per scored token), which no floating-point rate describes."""
    if case["kind"] == "detect":
        n_seg = max(1, case["n"] // case["text"])
        return {"bytes": case["n"] * (4 + 8 + 8 + 4 + 4) + n_seg * 24, "flops": 0}
    nodes, draft, K = _rows(case)
    V, W = case["vocab"], case["gamma"] + 1
    small = nodes * (20 + 4 + 8) + draft * (20 + 4 + K * 20) + case["n_seq"] * (4 + 16 + 8 * W)
    if case["kind"] == "lmhead":
        dt, dd = case["d_target"], case["d_draft"]
        return {"bytes": 2 * (V * (dt + dd) + nodes * dt + draft * dd) + small,
                "flops": 2 * V * (nodes * dt + draft * dd)}
    return {"bytes": (nodes + draft) * V * (4 if case.get("dtype") == "fp32" else 2) + small, "flops": 0}


def tolerance(case):
    """Tokens, words, lists and accept lengths are whole numbers and are compared as such; keys are
    fp32 estimates of s and scores fp32 roundings of fp64 values (measured against 64 bits: up to
    1.6e-7 of the norm for keys and 3e-8 for scores; the key's error bound is about 1e-5)."""
    if case["kind"] == "detect":
        # fp32 scores (7e-8 measured), their sums and log p-values (1.6e-7; about 1e-6 absolute)
        return {"rel": 1e-6, "max": 1e-4}
    if case["kind"] == "lmhead":
        # the logits are fp32 sums of d products: the tensor cores' sums move the keys by 7e-6 of
        # their norm against 64 bits, and another order of addition may turn a near tie
        return {"rel": 2.5e-5, "max": 5e-4, "differ": 1e-3}
    return {"rel": 1e-6, "max": 4e-5}


# ---------------------------------------------------------------- the same in 64 bits, from the definitions

_M32 = 0xFFFFFFFF


def _philox(c0, pos, ctx, key):
    """The four words of block c0 (unsigned 32-bit values in int64 tensors, broadcast together)."""
    x = [c0 & _M32, pos.to(torch.int64) & _M32, ctx & _M32, (ctx >> 32) & _M32]
    k0, k1 = key & _M32, (key >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        a, b = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57  # 64-bit products, wrapped like unsigned ones
        x = [((b >> 32) & _M32) ^ x[1] ^ k0, b & _M32, ((a >> 32) & _M32) ^ x[3] ^ k1, a & _M32]
    return x


def _word(tok, key, ctx, pos, arrival=1):
    key = key ^ (((arrival - 1) * 0x9E3779B9) & _M32)
    w = _philox(tok >> 2, pos, ctx, key)
    lane = tok & 3
    return torch.where(lane == 0, w[0], torch.where(lane == 1, w[1], torch.where(lane == 2, w[2], w[3])))


def _exp1(w):
    lo = -torch.log((w.double() + 0.5) * 2.0 ** -32)
    hi = -torch.log1p(-((_M32 - w).double() + 0.5) * 2.0 ** -32)
    return torch.where(w < 2 ** 31, lo, hi)


def _row_words(key, ctx, pos, vocab):
    c0 = torch.arange((vocab + 3) // 4, device=DEV)[None, :]
    w = _philox(c0, pos[:, None], ctx[:, None], key[:, None])
    return torch.stack(w, dim=2).reshape(key.numel(), -1)[:, :vocab]


def _kept(l, T, top_k, top_p):
    """Which tokens of the rows l (float64) survive top-k, then top-p by groups of equal logits."""
    keep = l >= torch.topk(l, min(top_k, l.shape[1]), dim=1).values[:, -1:]
    if top_p < 1.0:
        cut = 1.0 - float(np.float32(top_p))
        for r in range(l.shape[0]):
            v = torch.sort(l[r][keep[r]]).values.cpu().numpy()
            e = np.exp((v - v[-1]) / T)
            run, least = np.cumsum(e / e.sum()), v[0]
            for j in range(len(v)):
                if v[j] == v[-1]:
                    least = v[-1]
                    break
                if v[j + 1] != v[j]:
                    least = v[j + 1]
                    if run[j] > cut:
                        least = v[j]
                        break
            keep[r] = l[r] >= float(least)
    return keep


def _race(logits, key, ctx, pos, T, k, top_k=0, top_p=1.0, block=None, blocks=1):
    """The k smallest race keys of every row: (keys, tokens).  `logits(a, b)` gives rows a..b-1 in
    float64; `block`: the rows are proposals `block` of `blocks` on the augmented source."""
    n, T = key.numel(), float(np.float32(T))
    ks, ts = [], []
    V = logits(0, 1).shape[1]
    step = max(1, (1 << 24) // V)
    for a in range(0, n, step):
        b = min(n, a + step)
        l = logits(a, b)
        ids = key[a:b], ctx[a:b], pos[a:b]
        E = _exp1(_row_words(*ids, V))
        if block is not None:
            bk = block[a:b].long()
            J = (_row_words(ids[0] ^ 0x3C6EF372FE94F82B, *ids[1:], V) * blocks) >> 32
            mult = torch.tensor([((i + 1) * 0xBB67AE8584CAA73B + 2 ** 63) % 2 ** 64 - 2 ** 63 for i in range(blocks)],
                                dtype=torch.int64, device=DEV)
            F = _exp1(_row_words(ids[0] ^ mult[bk], *ids[1:], V))
            E = E / blocks + torch.where(J == bk[:, None], torch.zeros_like(F), F)
        s = torch.log(E) - l / T
        if top_k:
            s = torch.where(_kept(l, T, top_k, top_p), s, torch.full_like(s, math.inf))
        v, i = torch.topk(s, k, dim=1, largest=False, sorted=True)
        ks.append(v)
        ts.append(torch.where(v < math.inf, i, torch.full_like(i, -1)))
    return torch.cat(ks), torch.cat(ts)


def _lists(logits, key, ctx, pos, T, K, row_k, iid, **kw):
    """Draft lists as the draft call lays them out (numpy)."""
    s, t = _race(logits, key, ctx, pos, T, K, **kw)
    n, T = key.numel(), float(np.float32(T))
    m = torch.arange(K, device=DEV)[None, :]
    use = (m < row_k[:, None]) & (t >= 0)
    tok, out_key = torch.where(use, t, -1), torch.where(use, s, math.inf)
    mult, samples = use.long(), tok
    if iid:
        tt = t.clamp_min(0)
        ids = key[:, None], ctx[:, None], pos[:, None]
        E1 = _exp1(_word(tt, *ids))
        rest, G, cand = s - torch.log(E1), E1.clone(), []
        for j in range(1, K + 1):
            if j > 1:
                G = G + _exp1(_word(tt, *ids, arrival=j))
            cand.append(torch.where(use & (j <= row_k[:, None]), torch.log(G) + rest, math.inf))
        v, i = torch.topk(torch.stack(cand, 2).reshape(n, -1), K, dim=1, largest=False, sorted=True)
        pick = torch.where((v < math.inf) & (m < row_k[:, None]), i // K, -1)
        mult = (pick[:, :, None] == m[:, None, :]).sum(1)
        samples = torch.where(pick >= 0, torch.gather(t, 1, pick.clamp_min(0)), -1)
    return {"tok": tok.cpu().numpy(), "key": out_key.cpu().numpy(), "mult": mult.cpu().numpy(),
            "ndist": (mult > 0).sum(1).cpu().numpy(), "samples": samples.cpu().numpy()}


def _walk(logits, key, ctx, pos, T, seq_off, ndr, tok, nd, child, gamma, **kw):
    """Target winners, walks and scores as the verify call lays them out (numpy)."""
    _, y = _race(logits, key, ctx, pos, T, 1, **kw)
    y = y[:, 0]
    w = _word(y.clamp_min(0), key, ctx, pos)
    A = torch.where(w < 2 ** 31, -torch.log1p(-(w.double() + 0.5) * 2.0 ** -32),
                    -torch.log(((_M32 - w).double() + 0.5) * 2.0 ** -32)).cpu().numpy()
    y, w = y.cpu().numpy(), w.cpu().numpy()
    n_seq, W = len(seq_off) - 1, gamma + 1
    out = {"winner": y, "word": w.astype(np.uint32).view(np.int32), "accept_len": np.zeros(n_seq, np.int64),
           "n_emitted": np.zeros(n_seq, np.int64), "emitted": np.full((n_seq, W), -1), "score": np.zeros((n_seq, W)),
           "score_sum": np.zeros(n_seq)}
    for b in range(n_seq):
        c = int(seq_off[b])
        for step in range(W):
            out["emitted"][b, step], out["score"][b, step] = y[c], A[c]
            out["n_emitted"][b] = step + 1
            dr = int(ndr[c])
            hit = np.nonzero(tok[dr, :nd[dr]] == y[c])[0] if dr >= 0 and step < gamma else []
            if not len(hit) or child[dr, hit[0]] < 0:
                break
            c = int(child[dr, hit[0]])
            out["accept_len"][b] = step + 1
        out["score_sum"][b] = out["score"][b].sum()
    return out


def _mix64(z):
    with np.errstate(over="ignore"):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _child_label(ctx, tok):
    with np.errstate(over="ignore"):
        return _mix64(np.uint64(ctx) ^ (np.uint64(tok + 1) * np.uint64(0x9E3779B97F4A7C15)))


def _dense(t):
    return lambda a, b: t[a:b].double()


def _exact_step(case, s):
    kw = {"top_k": case["top_k"], "top_p": case["top_p"]}
    d = _lists(_dense(s.q), *s.draft_ids, case["temperature"], s.K, s.row_k, case["mode"] == "iid", **kw)
    v = _walk(_dense(s.p), *s.node_ids, case["temperature"], s.seq_off.cpu().numpy(), s.node_draft_row.cpu().numpy(),
              d["tok"], d["ndist"], s.child_node.cpu().numpy(), s.gamma, **kw)
    return {"draft": d, "walk": v, "status": None}


def _exact_lmhead(case, s):
    def products(h, w):
        w = w.double()
        return lambda a, b: h[a:b].double() @ w.T

    d = _lists(products(s.hq, s.wq), *s.draft_ids, case["temperature"], s.K, s.row_k, case["mode"] == "iid")
    v = _walk(products(s.hp, s.wp), *s.node_ids, case["temperature"], s.seq_off.cpu().numpy(),
              s.node_draft_row.cpu().numpy(), d["tok"], d["ndist"], s.child_node.cpu().numpy(), s.gamma)
    return {"draft": d, "walk": v, "status": None}


def _exact_tree(case, s):
    """Both tree kinds on the static slots of the fixed-capacity layout."""
    hetero = case["kind"] == "hetero"
    n_seq, K, gamma, T = case["n_seq"], case["K"], case["gamma"], case["temperature"]
    N1 = 1 + K * gamma
    ids = {"key": np.zeros((n_seq, N1), np.uint64), "ctx": np.zeros((n_seq, N1), np.uint64),
           "pos": np.zeros((n_seq, N1), np.uint32)}
    root = [x.cpu().numpy() for x in s.root]
    rk, rc, rp = root[0].view(np.uint64), root[1].view(np.uint64), root[2].view(np.uint32)
    ids["key"][:, 0], ids["ctx"][:, 0], ids["pos"][:, 0] = rk, rc, rp
    n_lists = n_seq * (1 + K * (gamma - 1))
    tok, nd = np.full((n_lists, K), -1), np.zeros(n_lists, np.int64)
    child, ndr = np.full((n_lists, K), -1), np.full((n_seq, N1), -1)
    # a depth's rows: (key, ctx, pos, draws, node slot of the depth) per sequence
    width = K if hetero else 1
    rows = [[(int(rk[b]), int(rc[b]), int(rp[b]), K, 0)] * width for b in range(n_seq)]
    first = 0
    for d in range(gamma):
        w, w_list = len(rows[0]), 1 if d == 0 else K
        flat = [r for seq in rows for r in seq]
        key, ctx = (torch.from_numpy(np.array([r[c] for r in flat], np.uint64).view(np.int64)).to(DEV) for c in (0, 1))
        pos = torch.tensor([r[2] for r in flat], dtype=torch.int64, device=DEV)
        draws = torch.tensor([max(1, min(K, r[3])) for r in flat], device=DEV)
        if hetero:
            blk = torch.arange(K, device=DEV).repeat(n_seq)
            x = _race(_dense(s.depth_logits[d]), key, ctx, pos, T, 1, block=blk, blocks=K)[1][:, 0].cpu().numpy()
        else:
            lists = _lists(_dense(s.depth_logits[d]), key, ctx, pos, T, K, draws, True)
        nxt = []
        for b in range(n_seq):
            ndr[b, (0 if d == 0 else 1 + (d - 1) * K):][:w_list] = first + b * w_list + np.arange(w_list)
            mine, kids = rows[b], []
            for i, (k, c, p, nu, slot) in enumerate(mine):
                lr = first + b * w_list + slot
                if hetero:
                    t = int(x[b * w + i])
                    at = next((j for j in range(i) if mine[j][4] == slot and int(x[b * w + j]) == t), i)
                    if at == i:
                        tok[lr, nd[lr]], child[lr, nd[lr]] = t, b * N1 + 1 + d * K + i
                        nd[lr] += 1
                    kids.append((k, int(_child_label(c, t)), p + 1, 1, at))
                    continue
                if not nu:
                    continue
                tok[lr], nd[lr] = lists["tok"][b * w + i], lists["ndist"][b * w + i]
                for m in range(int(nd[lr])):
                    child[lr, m] = b * N1 + 1 + d * K + len(kids)
                    kids.append((k, int(_child_label(c, int(tok[lr, m]))), p + 1, int(lists["mult"][b * w + i, m]),
                                 len(kids)))
            for j, (k, c, p, _, slot) in enumerate(kids):
                if not hetero or slot == j:
                    at = 1 + d * K + j
                    ids["key"][b, at], ids["ctx"][b, at], ids["pos"][b, at] = k, c, p
            kids += [(int(rk[b]), 0, 0, 0, j) for j in range(len(kids), K)]
            nxt.append(kids)
        first += n_seq * w_list
        rows = nxt
    node = [torch.from_numpy(ids[c].reshape(-1).view(t)).to(DEV)
            for c, t in (("key", np.int64), ("ctx", np.int64), ("pos", np.int32))]
    v = _walk(_dense(s.p), *node, T, np.arange(n_seq + 1) * N1, ndr.reshape(-1), tok, nd, child, gamma)
    return {"lists": None, "child": None, "node_ctx": ids["ctx"].view(np.int64).reshape(-1), "walk": v,
            "status": None}


def _exact_detect(case, s):
    tok = s.tok.long()
    w = _word(tok, s.key, s.ctx, s.pos)
    u, v = (w.double() + 0.5) * 2.0 ** -32, ((_M32 - w).double() + 0.5) * 2.0 ** -32
    lu = torch.where(u < 0.5, torch.log(u), torch.log1p(-v))
    if case["score"] == "aaronson":
        score = torch.where(u < 0.5, -torch.log1p(-u), -torch.log(v))
    elif case["score"] == "u":
        score = u
    elif case["score"] == "li":
        D = _SCORES["li"][1]
        k = math.floor(1.0 / (1.0 - D))
        q = 1.0 - k * (1.0 - D)
        score = torch.log(k * torch.exp(D / (1 - D) * lu) + (torch.exp((1 - q) / q * lu) if q > 0 else 0.0))
    else:
        e = _SCORES["power"][1]
        score = torch.clamp_max(v ** -0.5, e ** -0.5) - (2.0 - math.sqrt(e))
    off = s.seg_off
    length = off[1:] - off[:-1]
    seg = torch.repeat_interleave(torch.arange(length.numel(), device=DEV), length)
    sums = torch.zeros(length.numel(), dtype=torch.float64, device=DEV).index_add_(0, seg, score)
    M = length.double()
    if case["score"] == "aaronson":
        # ln P(Gamma(M, 1) >= S) = ln sum_{j < M} e^-S S^j / j!
        j = (torch.arange(tok.numel(), device=DEV) - off[:-1][seg]).double()
        term = -sums[seg] + j * torch.log(sums)[seg] - torch.lgamma(j + 1.0)
        top = torch.full_like(sums, -math.inf).scatter_reduce_(0, seg, term, "amax")
        logp = top + torch.log(torch.zeros_like(sums).index_add_(0, seg, torch.exp(term - top[seg])))
        logp = torch.where(length > 0, logp, torch.zeros_like(logp))
    elif case["score"] == "u":
        x = sums / M.clamp_min(1.0)
        lo, hi = torch.full_like(x, 1e-9), 2.0 / (1.0 - x) + 10.0
        for _ in range(200):  # the tilted mean 1/(1 - e^-l) - 1/l equals S/M at the minimum
            mid = 0.5 * (lo + hi)
            big = 1.0 / (-torch.expm1(-mid)) - 1.0 / mid > x
            lo, hi = torch.where(big, lo, mid), torch.where(big, mid, hi)
        b = M * torch.log(torch.expm1(lo) / lo) - lo * sums
        logp = torch.where(x > 0.5, b.clamp_max(0.0), torch.zeros_like(b))
    else:
        logp = None
    return {"score": score, "sum": sums, "logp": logp}


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "detect":
        return _exact_detect(case, s)
    if kind == "lmhead":
        return _exact_lmhead(case, s)
    return _exact_step(case, s) if kind == "step" else _exact_tree(case, s)
