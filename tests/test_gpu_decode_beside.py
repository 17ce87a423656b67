"""Decode calls with large tiles and narrow items beside them.  A narrow CTA
does not wait for the large launch before it; it is synchronised with what came
before both by a word that the large launch publishes behind its own wait and
that is moved on when the narrow launch is through.  Here every call follows
writes to the pages and the tables, on one stream without a wait between, and
the word's value after it says that both sides did their part."""
import pytest
import torch

from fg_harness import Run, compare
from workloads import Workload, queries

pytestmark = pytest.mark.gpu

WORD = 128  # byte offset of the word in the pool's workspace


def _word(pool):
    return int(pool.workspace[WORD:WORD + 4].view(torch.int32).item())


def _run(D, groups, L=2, prefix=700):
    n = sum(groups)
    w = Workload(name=f"beside_{D}_{n}", n_layers=L, n_q_heads=16, n_kv_heads=2, head_dim=D, n_blocks=2048, seed=81)
    run = Run(w, max_seqs=n + 2, max_decode_branches=n, max_splits=16)
    rids = []
    for g, size in enumerate(groups):
        m = run.create()
        run.append([m], prefix + 40 * g, ("prefix", g))
        rids += [m] + run.fork(m, size - 1)
    return w, run, rids


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("groups", [
    (9,), (16,),          # wide tiles: 72 and 128 stacked rows
    (17,), (32,),         # paired: 136 and 256
    (9, 17, 3),           # both, and a group on the narrow tile
    (9, 17, 12, 20, 16),  # a plan of more than 64 branches, read from device memory
])
def test_calls_in_a_row(stlib, D, groups):
    w, run, rids = _run(D, groups)
    steps = []
    for step in range(3):
        run.append(rids, 7, ("rows", step))          # the third crosses into new pages
        steps.append(run.decode(rids, ("q", step)))
        if step < 2:
            del steps[-1]                            # (the oracle below sees the last step's context)
    run.pool.sync()
    # every call has a tag of its own, two more than the last, and leaves it plus one
    assert _word(run.pool) == 2 * 3 + 1
    q, o, lse = steps[-1]
    for layer in range(w.n_layers):
        o_ref, l_ref = run.oracle_decode(rids, q, layer)
        compare(o[layer], lse[layer], o_ref, l_ref, f"layer {layer}")


def test_calls_without_a_large_tile_leave_the_word(stlib):
    _, run, rids = _run(64, (8, 3))
    run.append(rids, 7, ("rows",))
    run.decode(rids, ("q",))
    run.pool.sync()
    assert _word(run.pool) == 0


@pytest.mark.parametrize("groups", [(12,), (20, 9)])
def test_replayed_graph_reads_the_pages_as_they_are(stlib, groups):
    """A captured call carries one tag for all its replays."""
    w, run, rids = _run(128, groups)
    run.append(rids, 20, ("rows",))
    q, o, lse = run.decode(rids, ("q",))
    run.pool.sync()
    pool, handles = run.pool, [run.handle[r] for r in rids]
    o, lse = torch.empty_like(o), torch.empty_like(lse)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pool.decode_attn(handles, q, o, lse)
    for i in range(4):
        q.copy_(queries(w, ("replay", i), len(rids), device="cuda"))
        pool.k_pool.mul_(-0.75)
        pool.v_pool.mul_(1.5)
        graph.replay()
        again = pool.decode_attn(handles, q)
        pool.sync()
        assert torch.equal(o, again[0]) and torch.equal(lse, again[1])
