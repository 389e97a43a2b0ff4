"""The tree builders take root identities of their own dtype, device and number only, on the CPU:
`run` writes them before it calls the drafter, which ends these runs."""
import pytest
import torch

from paper_2609_21858_gb300.tree import HeteroTreeBuilder, TreeBuilder

N, K, GAMMA = 3, 4, 2
BUILDERS = [TreeBuilder, HeteroTreeBuilder]


class Drafting(Exception):
    pass


def _run(builder, key, ctx, pos):
    def drafter(*_):
        raise Drafting

    t = builder(N, K, GAMMA, device="cpu")
    with pytest.raises(Drafting):
        t.run(key, ctx, pos, drafter)
    return t


def _roots():
    return (torch.tensor([5, -6, 7]), torch.tensor([2 ** 40, 9, -(2 ** 50)]),
            torch.tensor([1, 2, 3], dtype=torch.int32))


@pytest.mark.parametrize("builder", BUILDERS)
def test_roots_reach_the_first_rows_and_the_root_nodes(builder):
    ids = _roots()
    t = _run(builder, *ids)
    per = 1 if builder is TreeBuilder else K
    for x, row, node in zip(ids, (t.row_key, t.row_ctx, t.row_pos), (t.node_key, t.node_ctx, t.node_pos)):
        assert torch.equal(row[:N * per], x.repeat_interleave(per))
        assert torch.equal(node[::1 + K * GAMMA], x)
        assert int(node.count_nonzero()) == N


@pytest.mark.parametrize("builder", BUILDERS)
@pytest.mark.parametrize("which", [0, 1, 2])
@pytest.mark.parametrize("change", ["dtype", "float", "short", "long"])
def test_roots_of_another_dtype_or_number_are_refused(builder, which, change):
    ids = list(_roots())
    x = ids[which]
    ids[which] = {"dtype": x.to(torch.int32 if which < 2 else torch.int64), "float": x.float(), "short": x[:2],
                  "long": torch.cat([x, x[:1]])}[change]
    with pytest.raises((RuntimeError, IndexError)):
        _run(builder, *ids)


def test_one_root_for_all_sequences():
    # the IID builder broadcasts a scalar or a single root; the proposal builder's rows are counted from the roots
    for one in (lambda x: x[:1], lambda x: x[0], lambda x: int(x[0])):
        key, ctx, pos = _roots()
        t = _run(TreeBuilder, one(key), ctx, one(pos))
        assert torch.equal(t.row_key[:N], key[:1].expand(N)) and torch.equal(t.row_pos[:N], pos[:1].expand(N))
        assert torch.equal(t.node_key[::1 + K * GAMMA], key[:1].expand(N))
        assert torch.equal(t.node_pos[::1 + K * GAMMA], pos[:1].expand(N))
    with pytest.raises(RuntimeError):
        _run(HeteroTreeBuilder, *(x[:1] for x in _roots()))
