"""Rows of any alignment and length: a row's results depend on its values alone.

Rows that start on 16-byte boundaries stream with 128-bit loads, others through aligned 32-bit
words (full race) or from their first 16-byte boundary on (truncated race), and a row's remainder
after the last whole iteration takes its own pass.  Each case places the same logits in rows of
another offset and stride and compares every output bit for bit with the aligned rows' (which
the parity suites check against the oracle), around the sizes of a vector, a pass of 32 vectors
and a fast iteration (96 vectors of bf16, 192 of fp32)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_21858_gb300 import pps
from parity import compare_draft

pytestmark = pytest.mark.gpu

BF, F32 = torch.bfloat16, torch.float32
DRAFT = ("tok", "key", "mult", "ndist", "samples")
VERIFY = ("winner", "word", "accept_len", "n_emitted", "emitted", "score", "score_sum")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    pps.lib()


def _inputs(n, V, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = (torch.randn(n, V, generator=g, device="cuda") * 2.5).to(dtype)
    if V > 40:  # some rows with masked tokens: -inf, NaN and the type's lowest value
        hole = torch.rand(n, V, generator=g, device="cuda") < 0.2
        x[1::4] = torch.where(hole[1::4], torch.tensor(float("-inf"), device="cuda").to(dtype), x[1::4])
        x[2::4] = torch.where(hole[2::4], torch.tensor(float("nan"), device="cuda").to(dtype), x[2::4])
        x[3::4] = torch.where(hole[3::4], torch.tensor(torch.finfo(dtype).min, device="cuda").to(dtype), x[3::4])
    ids = (torch.randint(-2 ** 62, 2 ** 62, (n,), generator=g, device="cuda"),
           torch.randint(-2 ** 62, 2 ** 62, (n,), generator=g, device="cuda"),
           torch.randint(0, 2 ** 30, (n,), generator=g, device="cuda", dtype=torch.int32))
    return x, ids


def _placed(x, offset, pad):
    """The rows of x at element `offset` of rows of V + pad elements, with foreign values around them."""
    n, V = x.shape
    wide = torch.full((n * (V + pad) + offset + 16,), 1e4, dtype=x.dtype, device="cuda")
    view = wide[offset:offset + n * (V + pad)].view(n, V + pad)[:, :V]
    view.copy_(x)
    return view


def _aligned(x):
    return _placed(x, 0, -x.shape[1] % 8 + 8)


def _same(a, b, names):
    for k in names:
        assert torch.equal(a[k], b[k]), k


def _verify(x, ids, **kw):
    n = x.shape[0]
    off = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    none = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    one = torch.zeros(1, 1, dtype=torch.int32, device="cuda")
    return pps.verify_tree(x, *ids, 1, off, none, one, one[0], one, **kw)


SIZES = [1, 5, 8, 33, 255, 256, 257, 767, 768, 769, 775, 1541, 6151, 40003]


@pytest.mark.parametrize("dtype,offset,pad", [(BF, 1, 0), (BF, 2, 1), (BF, 4, 4), (BF, 7, 10), (F32, 1, 0),
                                              (F32, 2, 2), (F32, 3, 5)])
def test_results_do_not_depend_on_the_rows_place(dtype, offset, pad):
    for V in SIZES:
        x, ids = _inputs(9, V, dtype, 100 + V)
        y, z = _placed(x, offset, pad), _aligned(x)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        for K, mode in ((1, pps.DISTINCT), (min(V, 8), pps.IID), (min(V, 32), pps.DISTINCT)):
            for kw in ({}, {"top_k": 5}, {"top_k": 64, "top_p": 0.9}):
                _same(pps.draft_list(y, *ids, K, mode=mode, status=status, **kw),
                      pps.draft_list(z, *ids, K, mode=mode, status=status, **kw), DRAFT)
        for kw in ({}, {"top_k": 50}):
            _same(_verify(y, ids, status=status, **kw), _verify(z, ids, status=status, **kw), VERIFY)
        blk = torch.arange(9, dtype=torch.int32, device="cuda") % 4
        for kw in ({}, {"top_k": 20}):
            a = pps.draft_hetero(y, *ids, blk, 4, status=status, **kw)
            assert torch.equal(a, pps.draft_hetero(z, *ids, blk, 4, status=status, **kw)), V
        assert int(status.item()) == 0, V


# a row cut between as many warps as it can be (60), and between a few; the whole list (K = 32: more
# entries than the merge stages of each list) in one warp's segment, or spread
@pytest.mark.parametrize("n,V,dtype", [(1, 128256, BF), (2, 40000, BF), (3, 70001, F32)])
@pytest.mark.parametrize("where", ["one", "all"])
def test_lists_of_rows_cut_between_many_warps(n, V, dtype, where):
    rng = np.random.default_rng(V + n)
    x = rng.normal(0, 1, (n, V)).astype(np.float32)
    if where == "one":
        x[:, V // 3:V // 3 + 90] += 25.0
    x = torch.as_tensor(x).to(dtype).cuda()
    ids = [rng.integers(0, 2 ** 64, n, dtype=np.uint64), rng.integers(0, 2 ** 64, n, dtype=np.uint64),
           rng.integers(0, 2 ** 31, n, dtype=np.uint32)]
    dev = [torch.as_tensor(a.view(t)).cuda() for a, t in zip(ids, (np.int64, np.int64, np.int32))]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for K, mode in ((32, pps.DISTINCT), (8, pps.IID), (1, pps.DISTINCT)):
        d = pps.draft_list(x, *dev, K, mode=mode, status=status)
        torch.cuda.synchronize()
        want = oracle.draft_rows(x.float().cpu().numpy(), *ids, K, mode=mode)
        compare_draft({k: v.cpu().numpy() for k, v in d.items()}, want)
    assert int(status.item()) == 0


# +inf logits win, the lowest index first, however many there are: more than a list holds, met by the
# lanes and warps of a row in another order than that of their indexes
@pytest.mark.parametrize("dtype,offset,pad", [(BF, 0, 0), (BF, 1, 1), (F32, 0, 0), (F32, 3, 2)])
@pytest.mark.parametrize("V,many", [(700, 20), (700, 200), (20000, 200), (20000, 3000), (128256, 4000)])
def test_rows_with_many_infinite_logits(V, many, dtype, offset, pad):
    n = 24
    rng = np.random.default_rng(V + many)
    x = rng.normal(0, 2.5, (n, V)).astype(np.float32)
    for r in range(n):
        x[r, rng.choice(V, many, replace=False)] = np.inf
    x = torch.as_tensor(x).to(dtype).cuda()
    ids = (rng.integers(0, 2 ** 64, n, dtype=np.uint64), rng.integers(0, 2 ** 64, n, dtype=np.uint64),
           rng.integers(0, 2 ** 31, n, dtype=np.uint32))
    dev = tuple(torch.as_tensor(a.view(t)).cuda() for a, t in zip(ids, (np.int64, np.int64, np.int32)))
    y = _placed(x, offset, pad)
    lowest = np.stack([np.nonzero(row == np.inf)[0][:32] for row in x.float().cpu().numpy()])
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for kw in ({}, {"top_k": 50}):
        for K in (1, 4, 8, 16):
            d = pps.draft_list(y, *dev, K, status=status, **kw)
            assert np.array_equal(d["tok"].cpu().numpy(), lowest[:, :K]), (K, kw)
        assert np.array_equal(_verify(y, dev, status=status, **kw)["winner"].cpu().numpy(), lowest[:, 0]), kw
        blk = torch.arange(n, dtype=torch.int32, device="cuda") % 5
        x1 = pps.draft_hetero(y, *dev, blk, 5, status=status, **kw)
        assert np.array_equal(x1.cpu().numpy(), lowest[:, 0]), kw
    assert int(status.item()) == 0
    want = oracle.draft_rows(x.float().cpu().numpy(), *ids, 16)
    assert np.array_equal(want["tok"], lowest[:, :16])
