"""One workspace serves calls of different sizes in turn: a call's results are those it has with a
workspace of its own, whatever larger calls left in the partial lists."""
import pytest
import torch

from paper_2609_21858_gb300 import pps

pytestmark = pytest.mark.gpu

BF, F32 = torch.bfloat16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    pps.lib()


def _rows(n, V, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = (torch.randn(n, V, generator=g, device="cuda") * 2.5).to(dtype)
    return x, (torch.randint(-2 ** 62, 2 ** 62, (n,), generator=g, device="cuda"),
               torch.randint(-2 ** 62, 2 ** 62, (n,), generator=g, device="cuda"),
               torch.randint(0, 2 ** 30, (n,), generator=g, device="cuda", dtype=torch.int32))


def _chains(n):
    """n // 5 sequences of 5 nodes: a root and its chain, each with a one-token draft row."""
    s = n // 5
    node = torch.arange(5 * s, dtype=torch.int32, device="cuda")
    child = torch.where(node % 5 < 4, node + 1, torch.full_like(node, -1))
    return 4, node[::5].tolist() + [5 * s], node, child.view(-1, 1)


def _verify(fn, n, ids, ws, **kw):
    gamma, off, draft_row, child = _chains(n)
    m = draft_row.numel()
    tok = torch.zeros(m, 1, dtype=torch.int32, device="cuda")
    nd = torch.ones(m, dtype=torch.int32, device="cuda")
    off = torch.tensor(off, dtype=torch.int32, device="cuda")
    return fn(*(x[:m] for x in ids), gamma, off, draft_row, tok, nd, child, ws=ws, **kw)


def _same(a, b):
    for k in a:
        assert (a[k] is None) == (b[k] is None) and (a[k] is None or torch.equal(a[k], b[k])), k


# rows enough that each kind of call cuts rows between warps far beyond the slots of a small call
@pytest.mark.parametrize("n,V,dtype,top_k", [(16720, 5717, BF, 50), (31000, 4000, BF, 0), (31000, 2000, F32, 0)])
def test_small_calls_after_a_large_one(n, V, dtype, top_k):
    ws = pps.workspace(n, n)
    x, ids = _rows(n, V, dtype, n)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    big = pps.draft_list(x, *ids, 8, top_k=top_k, status=status)
    _same(pps.draft_list(x, *ids, 8, top_k=top_k, ws=ws, status=status), big)
    for m, U in ((5, 40000), (303, 9001), (2500, 5000)):
        y, jds = _rows(m, U, dtype, m)
        blk = torch.arange(m, dtype=torch.int32, device="cuda") % 4
        for kw in ({}, {"top_k": 50}):
            kw["status"] = status
            _same(pps.draft_list(y, *jds, 8, ws=ws, **kw), pps.draft_list(y, *jds, 8, **kw))
            assert torch.equal(pps.draft_hetero(y, *jds, blk, 4, ws=ws, **kw), pps.draft_hetero(y, *jds, blk, 4, **kw))
            v = _verify(lambda *a, **k: pps.verify_tree(y[:m // 5 * 5], *a, **k), m, jds, ws, **kw)
            _same(v, _verify(lambda *a, **k: pps.verify_tree(y[:m // 5 * 5], *a, **k), m, jds, None, **kw))
    _same(pps.draft_list(x, *ids, 8, top_k=top_k, ws=ws, status=status), big)
    assert int(status.item()) == 0


@pytest.mark.parametrize("n", [129, 1300, 41984])
def test_small_lmhead_calls_after_a_large_one(n):
    # 41984 rows: 328 row blocks, two partial lists a row
    V, d = 700, 64
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    h = torch.randn(n, d, generator=g, device="cuda").to(BF)
    w = torch.randn(V, d, generator=g, device="cuda").to(BF)
    ids = _rows(n, 1, F32, n)[1]
    ws = pps.lmhead_workspace(n, n)
    big = pps.lmhead_draft_list(h, w, *ids, 8)
    _same(pps.lmhead_draft_list(h, w, *ids, 8, ws=ws), big)
    for m in (1000, 65, 5):
        m = min(m, n // 5 * 5)
        jds = [x[:m] for x in ids]
        _same(pps.lmhead_draft_list(h[:m], w, *jds, 4, ws=ws), pps.lmhead_draft_list(h[:m], w, *jds, 4))
        call = lambda *a, **k: pps.lmhead_verify_tree(h[:m], w, *a, **k)
        _same(_verify(call, m, jds, ws), _verify(call, m, jds, None))
    _same(pps.lmhead_draft_list(h, w, *ids, 8, ws=ws), big)
