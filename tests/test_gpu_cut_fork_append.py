"""Appends of one call to a parent and to children forked from inside its last
page (fork_at): the parent copies its rows of that page away, and the last child
left writes its own in place, over rows that the parent copies.  The copy comes
first: what is in the pool, row by row, for every order of the sequences and
every call that appends."""
import pytest
import torch

from fg_harness import Run, compare
from workloads import Workload, kv_rows, queries

pytestmark = pytest.mark.gpu


def _rows_as_drawn(run, rids, layers):
    for r in rids:
        table, n = run.pool.block_table(run.handle[r])
        at = torch.tensor(table, device="cuda").repeat_interleave(16)[:n], torch.arange(n, device="cuda") % 16
        for layer in layers:
            k, v = run.context(r, layer)
            assert torch.equal(run.pool.k_pool[layer][at[0], :, at[1]].cpu(), k), (r, layer)
            assert torch.equal(run.pool.v_pool[layer][at[0], :, at[1]].cpu(), v), (r, layer)


def _append(run, w, rids, n_tok, how):
    """n_tok rows to each by one call of the kind `how`."""
    if how == "append":
        run.append(rids, n_tok, ("rows",))
    elif how == "prefill":
        run.prefill_batch(rids, [n_tok] * len(rids), ("rows",))
    else:
        k, v = kv_rows(w, ("rows",), len(rids), device="cuda")
        run.pool.decode_step([run.handle[r] for r in rids], k, v, queries(w, ("q",), len(rids), device="cuda"))
        run.ref.append(rids, 1)
        run.sizes[("rows",)] = len(rids)
        for i, r in enumerate(rids):
            run.hist[r].append((("rows",), i, 1))


# rows of the parent, where the children are cut, the children, the sequences of
# the call in order (0: the parent), and the append's kernels
@pytest.mark.parametrize("length,cut,kids,order,kernels", [
    (47, 35, 1, (0, 1), 2),          # the parent copies 15 rows, the child writes from row 3 on
    (47, 46, 1, (0, 1), 2),          # from its last one
    (47, 33, 3, (0, 1, 2, 3), 2),    # two children copy as well, the last one writes
    (47, 33, 3, (1, 0, 3, 2), 2),
    (47, 35, 1, (1, 0), 1),          # the child copies, the parent writes behind what it copied
    (47, 47, 2, (0, 1, 2), 1),       # all end on the same row
    (48, 35, 1, (0, 1), 1),          # the parent's page is full: it takes a new one, the child copies
    (47, 33, 36, tuple(range(37)), 2),   # a plan that is read from device memory
])
@pytest.mark.parametrize("how", ["append", "prefill", "step"])
def test_copies_come_before_rows(stlib, length, cut, kids, order, kernels, how):
    L = 12
    w = Workload(name="cut", n_layers=L, n_q_heads=8, n_kv_heads=8, head_dim=128, n_blocks=512, seed=101)
    for again in range(3):
        run = Run(w, max_seqs=kids + 2, max_decode_branches=kids + 1, max_splits=4, pool_seed=again)
        m = run.create()
        run.append([m], length, ("prefix",))
        seqs = [m] + run.fork_at(m, cut, kids)
        run.pool.profile_read()
        _append(run, w, [seqs[i] for i in order], 1 if how == "step" else 20, how)
        run.pool.sync()
        assert run.pool.profile_read()["append_kv"]["kernels"] == kernels
        run.check_tables()
        _rows_as_drawn(run, seqs, range(L))
        run.pool.close()


def test_decode_after_an_append_to_cut_forks(stlib):
    w = Workload(name="cut_decode", n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, n_blocks=256, seed=102)
    run = Run(w, max_seqs=8, max_decode_branches=6, max_splits=4)
    m = run.create()
    run.append([m], 300 + 13, ("prefix",))
    seqs = [m] + run.fork_at(m, 300 + 6, 2) + run.fork_at(m, 300 + 10, 2)
    run.append(seqs, 9, ("rows",))
    q, o, lse = run.decode(seqs, ("q",))
    run.pool.sync()
    for layer in range(2):
        o_ref, l_ref = run.oracle_decode(seqs, q, layer)
        compare(o[layer], lse[layer], o_ref, l_ref, f"layer {layer}")
