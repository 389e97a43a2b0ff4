"""GPU parity of the truncated race (top-k, then top-p, before the race)
against the oracle's masking followed by its untruncated race, through the
C ABI (pps_draft_list_trunc / pps_verify_tree_trunc)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_21858_gb300 import pps, synth
from parity import TOP_P_MARGIN, check_workload, compare_draft, compare_winners, f32, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    pps.lib()


@pytest.mark.parametrize("top_k,top_p", [(50, 1.0), (1, 1.0), (5, 0.9), (64, 0.5), (20, 0.97)])
@pytest.mark.parametrize("mode", [pps.DISTINCT, pps.IID])
def test_chain4x4_truncated(top_k, top_p, mode):
    wl = synth.make_workload("chain4x4", n_seq=8)
    check_workload(wl, mode, top_k=top_k, top_p=top_p)


@pytest.mark.parametrize("top_k,top_p", [(50, 1.0), (8, 0.8)])
def test_zipf_k8_truncated_reduced(top_k, top_p):
    wl = synth.make_workload("zipf_k8", n_seq=3)
    check_workload(wl, pps.DISTINCT, top_k=top_k, top_p=top_p)
    check_workload(wl, pps.IID, top_k=top_k, top_p=top_p)


def test_fp32_tiny_and_branch16_truncated():
    check_workload(synth.make_workload("tiny"), pps.DISTINCT, top_k=50, top_p=0.9)
    check_workload(synth.make_workload("branch16", n_seq=1), pps.DISTINCT, top_k=50, top_p=1.0)


@pytest.mark.parametrize("V,dtype", [(3, torch.bfloat16), (13, torch.float32), (70, torch.bfloat16),
                                     (1003, torch.bfloat16), (4099, torch.float32)])
def test_ragged_vocab_truncated(V, dtype):
    K = min(4, V)
    wl = synth.make_workload("chain4x4", n_seq=5, vocab=V, branching=(K, 1), dtype=dtype, seed=11 + V)
    check_workload(wl, pps.DISTINCT, top_k=min(50, V), top_p=0.9)
    check_workload(wl, pps.IID, top_k=10, top_p=1.0)


def test_unaligned_rows_truncated():
    base = synth.make_workload("chain4x4", n_seq=3, vocab=2001, seed=21)
    for attr in ("p_logits", "q_logits"):
        x = getattr(base, attr)
        wide = torch.zeros(x.shape[0], x.shape[1] + 3, dtype=x.dtype)
        wide[:, 1:1 + x.shape[1]] = x
        setattr(base, attr, wide.cuda()[:, 1:1 + x.shape[1]])
    check_workload(base, pps.DISTINCT, top_k=50, top_p=0.95)


def test_temperature_truncated():
    wl = synth.make_workload("chain4x4", n_seq=3, vocab=5000, seed=41)
    wl.temperature = 0.6
    check_workload(wl, pps.DISTINCT, top_k=30, top_p=0.8)
    wl.temperature = 1.7
    check_workload(wl, pps.IID, top_k=30, top_p=0.8)


def test_masked_nan_and_short_rows_truncated():
    wl = synth.make_workload("chain4x4", n_seq=4, vocab=3000, dtype=torch.float32, seed=31)
    p, q = wl.p_logits, wl.q_logits
    rng = np.random.default_rng(0)
    for x in (p, q):
        x[torch.as_tensor(rng.random(x.shape) < 0.3)] = float("-inf")
        x[torch.as_tensor(rng.random(x.shape) < 0.01)] = float("nan")
    p[3, :] = float("-inf")       # no usable token: winner -1
    q[2, :-3] = float("-inf")     # 3 usable tokens < top_k
    p[7, :-20] = float("nan")     # 20 usable tokens
    for tk, tp in ((50, 1.0), (10, 0.7)):
        gd, gv, status = run_gpu(wl, top_k=tk, top_p=tp)
        od, ov = run_oracle(wl, top_k=tk, top_p=tp)
        assert status == 0
        compare_draft(gd, od, loose=od["loose"])
        compare_winners(gv["winner"], gv["word"], ov["winner"], ov["word"], ov["margin"], loose=ov["loose"])
        assert gv["winner"][3] == -1


def _tie_rows(wl, n_ties, top_k):
    """Rows whose top_k-th logit ties with n_ties tokens (more than the 64-entry list holds)."""
    rng = np.random.default_rng(n_ties)
    for x in (wl.p_logits, wl.q_logits):
        V = x.shape[1]
        for r in range(0, x.shape[0], 2):
            cols = torch.as_tensor(rng.choice(V, n_ties + top_k // 2, replace=False), device=x.device)
            x[r, cols[: top_k // 2]] = 8.0 + torch.arange(top_k // 2, device=x.device, dtype=x.dtype) * 0.25
            x[r, cols[top_k // 2:]] = 6.0   # the tie group at the top_k-th place


@pytest.mark.parametrize("top_p", [1.0, 0.999999, 0.6])
def test_top_k_tie_group_larger_than_the_list(top_p):
    # the tie group of l_(k) overflows the 64-entry lists: the row is finished by a
    # second pass (kept tie group: exact race over logit >= l_(k); dropped: the list)
    wl = synth.make_workload("chain4x4", n_seq=4, vocab=32000, seed=61)
    _tie_rows(wl, 300, 40)
    gd, gv, status = run_gpu(wl, top_k=40, top_p=top_p)
    od, ov = run_oracle(wl, top_k=40, top_p=top_p)
    assert status == 0
    compare_draft(gd, od, loose=od["loose"])
    compare_winners(gv["winner"], gv["word"], ov["winner"], ov["word"], ov["margin"], loose=ov["loose"])


def test_constant_rows_keep_everything():
    wl = synth.make_workload("chain4x4", n_seq=2, vocab=5000, seed=71)
    wl.p_logits[1, :] = 1.5
    wl.q_logits[0, :] = -2.0
    check_workload(wl, pps.DISTINCT, top_k=3, top_p=1.0)


def test_full_size_zipf_k8_truncated_sampled_rows():
    wl = synth.make_workload("zipf_k8", device="cuda")
    t = wl.tree
    gd, gv, status = run_gpu(wl, top_k=50, top_p=1.0)
    assert status == 0
    rng = np.random.default_rng(8)
    dr = np.sort(rng.choice(t.n_draft, 48, replace=False))
    nr = np.sort(rng.choice(t.n_nodes, 48, replace=False))
    dsel, nsel = torch.as_tensor(dr, device="cuda"), torch.as_tensor(nr, device="cuda")
    qm, _ = oracle.truncate_rows(wl.q_logits[dsel].float().cpu().numpy(), 50, 1.0, 1.0)
    pm, _ = oracle.truncate_rows(wl.p_logits[nsel].float().cpu().numpy(), 50, 1.0, 1.0)
    od = oracle.draft_rows(qm, synth.u64(wl.draft_key[dsel]), synth.u64(wl.draft_ctx[dsel]),
                           synth.u32(wl.draft_pos[dsel]), t.K, row_k=t.row_k[dr])
    sub = {k: (x[dr] if x is not None and x.ndim >= 1 and x.shape[0] == t.n_draft else x) for k, x in gd.items()}
    compare_draft(sub, od, rows=dr)
    win, wd, _, mg = oracle.target_rows(pm, synth.u64(wl.node_key[nsel]), synth.u64(wl.node_ctx[nsel]),
                                        synth.u32(wl.node_pos[nsel]))
    compare_winners(gv["winner"][nr], gv["word"][nr], win, wd, mg)
    ow = oracle.walk(t.gamma, t.seq_off, t.node_draft_row, gd["tok"], gd["ndist"], t.child_node, gv["winner"],
                     gv["word"])
    assert np.array_equal(gv["accept_len"], ow["accept_len"]) and np.array_equal(gv["emitted"], ow["emitted"])


def _hard_rows(n, V, dtype, seed):
    """Rows that a threshold guessed from 32 evenly spread chunks of 32 vectors meets badly, five kinds
    in turn: random, sorted, the largest logits all inside those chunks (the guess is too high), one
    value everywhere, fewer usable tokens than top-k."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn(n, V, generator=g, device="cuda")
    x[1::5] = -1.1 * torch.log(torch.arange(1, V + 1, device="cuda", dtype=torch.float32))
    vw = 8 if dtype == torch.bfloat16 else 4
    chunks = V // vw // 32
    at = torch.tensor([chunks * c // 32 * 32 * vw + 7 * c for c in range(32)], device="cuda")
    x[2::5, at] = 9.0 + torch.arange(32, device="cuda") / 16
    x[3::5] = 0.5
    x[4::5, 40:] = float("-inf")
    return x.to(dtype)


# rows too many to be cut (long enough for a guess) and few rows cut between warps; starts on 16-byte boundaries and not;
# the last three are long enough for a guess (6144 vectors) whole and cut in two, wherever the number of resident warps lies
@pytest.mark.parametrize("n,V,dtype,shift", [(2900, 65536, torch.bfloat16, 0), (3100, 49201, torch.bfloat16, 3),
                                             (2900, 24700, torch.float32, 1), (11, 70001, torch.bfloat16, 1),
                                             (7, 30000, torch.float32, 0), (2900, 98400, torch.bfloat16, 0),
                                             (3100, 98411, torch.bfloat16, 3), (2900, 49201, torch.float32, 1)])
def test_top_k_threshold_of_hard_rows(n, V, dtype, shift):
    wide = torch.full((n, V + (-V % 8) + 8), 50.0, dtype=dtype, device="cuda")
    x = wide[:, shift:shift + V]
    x.copy_(_hard_rows(n, V, dtype, V))
    rng = np.random.default_rng(V)
    key, ctx = rng.integers(0, 2 ** 64, n, dtype=np.uint64), rng.integers(0, 2 ** 64, n, dtype=np.uint64)
    pos = rng.integers(0, 2 ** 31, n, dtype=np.uint32)
    ids = tuple(torch.as_tensor(a.view(t)).cuda() for a, t in ((key, np.int64), (ctx, np.int64), (pos, np.int32)))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for top_k, top_p in ((50, 1.0), (64, 0.7), (1, 1.0)):
        d = pps.draft_list(x, *ids, 8, top_k=top_k, top_p=top_p, status=status)
        torch.cuda.synchronize()
        rows = np.arange(min(n, 15)) if n < 100 else np.concatenate([np.arange(10), n - 1 - np.arange(5)])
        sel = torch.as_tensor(rows, device="cuda")
        mask, margin = oracle.truncate_rows(x[sel].float().cpu().numpy(), top_k, top_p, 1.0)
        want = oracle.draft_rows(mask, key[rows], ctx[rows], pos[rows], 8)
        compare_draft({k: v[sel].cpu().numpy() for k, v in d.items()}, want, loose=margin < TOP_P_MARGIN)
    assert int(status.item()) == 0


def _random_ids(n, seed):
    rng = np.random.default_rng(seed)
    ids = (rng.integers(0, 2 ** 64, n, dtype=np.uint64), rng.integers(0, 2 ** 64, n, dtype=np.uint64),
           rng.integers(0, 2 ** 31, n, dtype=np.uint32))
    return ids, tuple(torch.as_tensor(a.view(t)).cuda() for a, t in zip(ids, (np.int64, np.int64, np.int32)))


def _exactly_the_oracles(x, ids, dev, K, mode, top_k, top_p):
    """Lists (and, for K = 1, winners) of the truncated rows, near ties included."""
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    d = pps.draft_list(torch.as_tensor(x).cuda(), *dev, K, mode=mode, top_k=top_k, top_p=top_p, status=status)
    masked, _ = oracle.truncate_rows(x, top_k, f32(top_p), 1.0)
    want = oracle.draft_rows(masked, *ids, K, mode=mode)
    assert np.array_equal(d["tok"].cpu().numpy(), want["tok"])
    assert np.array_equal(d["samples"].cpu().numpy(), want["labels"])
    if K == 1:
        n = len(x)
        off = torch.arange(n + 1, dtype=torch.int32, device="cuda")
        none = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        one = torch.zeros(1, 1, dtype=torch.int32, device="cuda")
        v = pps.verify_tree(torch.as_tensor(x).cuda(), *dev, 1, off, none, one, one[0], one, top_k=top_k, top_p=top_p,
                            status=status)
        assert np.array_equal(v["winner"].cpu().numpy(), want["tok"][:, 0])
    assert int(status.item()) == 0


# rows whose tie group at l_(k) overflows the list, the K-th key crowded (so that the row is scanned once
# more), and 400 tokens just below l_(k), many of them with smaller keys
@pytest.mark.parametrize("V,top_p", [(2000, 1.0), (2000, 0.9999), (40000, 1.0)])
@pytest.mark.parametrize("K", [8, 32])
def test_a_second_scan_of_a_crowded_row_keeps_to_the_truncated_set(K, V, top_p):
    n, top_k, tied, extra = 16, 40, 150, 20
    ids, dev = _random_ids(n, 50 + K)
    rng = np.random.default_rng(V + K)
    x = np.full((n, V), -20.0, np.float32)
    for r in range(n):
        w = oracle.words(*(a[r:r + 1] for a in ids), V)[0]
        log_e = np.log(-np.log((w + 0.5) * 2.0 ** -32))
        at = rng.permutation(V)
        x[r, at[:tied]] = 4.0
        x[r, at[tied:tied + 400]] = rng.uniform(3.2, 3.9, 400)
        last = np.sort(log_e[at[:tied]] - 4.0)[K - 1]
        rest = at[tied + 400:]
        rest = rest[log_e[rest] - last > 4.001][:extra]  # their logits come to lie above the tie group's
        x[r, rest] = log_e[rest] - last - rng.uniform(-3e-7, 3e-7, extra)
    _exactly_the_oracles(x, ids, dev, K, pps.DISTINCT, top_k, top_p)


def _crowded(ids, V, usable, lo, hi, K, seed):
    """fp32 rows whose `usable` tokens (the rest at -30) have their keys of ranks lo .. hi - 1 within 1e-6
    of the K-th smallest one, in an order that only 64 bits tell."""
    rng = np.random.default_rng(seed)
    key, ctx, pos = ids
    x = np.full((len(key), V), -30.0, np.float32)
    for r in range(len(key)):
        at = rng.choice(V, usable, replace=False)
        log_e = np.log(-np.log((oracle.words(key[r:r + 1], ctx[r:r + 1], pos[r:r + 1], V)[0, at] + 0.5) * 2.0 ** -32))
        l = rng.normal(5, 1.5, usable)
        order = np.argsort(log_e - l)
        s = (log_e - l)[order]
        l[order[lo:hi]] = log_e[order[lo:hi]] - s[K - 1] - rng.uniform(-3e-7, 3e-7, hi - lo)
        x[r, at] = l
    return x


# more keys within the fp32 error bounds of the K-th than the kept list (2 K + 1 entries, at most 32) holds
@pytest.mark.parametrize("V", [3000, 40000])
@pytest.mark.parametrize("K,mode", [(1, pps.DISTINCT), (8, pps.DISTINCT), (8, pps.IID), (15, pps.DISTINCT),
                                    (31, pps.DISTINCT), (32, pps.DISTINCT), (32, pps.IID)])
def test_lists_of_rows_crowded_at_the_last_key(K, mode, V):
    ids, dev = _random_ids(24, K)
    x = _crowded(ids, V, 64, max(0, K - 3), min(64, 2 * K + 10), K, K + V)
    _exactly_the_oracles(x, ids, dev, K, mode, 64, 1.0)


def test_proposals_of_rows_crowded_at_the_first_key():
    n, V, B, usable = 24, 900, 3, 40
    ids, dev = _random_ids(n, 9)
    block = (np.arange(n) % B).astype(np.int32)
    rng = np.random.default_rng(10)
    x = np.full((n, V), -30.0, np.float32)
    for r in range(n):
        at = rng.choice(V, usable, replace=False)
        log_e = np.log([oracle.block_e(*(int(a[r]) for a in ids), int(i), int(block[r]), B) for i in at])
        l = rng.normal(5, 1.5, usable)
        first = np.argsort(log_e - l)[:10]
        l[first] = log_e[first] - (log_e - l).min() - rng.uniform(-3e-7, 3e-7, 10)
        x[r, at] = l
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = pps.draft_hetero(torch.as_tensor(x).cuda(), *dev, torch.as_tensor(block).cuda(), B, top_k=usable, status=status)
    assert np.array_equal(got.cpu().numpy(), oracle.block_draft_rows(x, *ids, block, B)[0])
    assert int(status.item()) == 0
