"""Appends that refresh the block tables in their own launch (small ones, their
rows' pages in the kernel parameters) and those that do not, at the sizes where
the form changes: the tables bit-exact against the reference pool, and a decode
over what was appended against the float64 oracle."""
import pytest

from fg_harness import Run, compare
from workloads import Workload

pytestmark = pytest.mark.gpu


def _run(n_blocks, max_seqs, seed, D=64):
    w = Workload(name=f"refresh_{seed}", n_layers=2, n_q_heads=4, n_kv_heads=2, head_dim=D, n_blocks=n_blocks, seed=seed)
    return Run(w, max_seqs=max_seqs, max_decode_branches=max_seqs, max_splits=8)


def _check(run, rids):
    run.check_tables()
    q, o, lse = run.decode(rids, ("q", len(rids)))
    run.pool.sync()
    for layer in range(2):
        o_ref, l_ref = run.oracle_decode(rids, q, layer)
        compare(o[layer], lse[layer], o_ref, l_ref, f"layer {layer}")


@pytest.mark.parametrize("before,rows", [
    (0, 1), (0, 16), (15, 1), (15, 2),     # one page, a full one, no new page, one
    (0, 3072), (0, 3073),                  # 192 pages: the inline list full; one more
    (5, 3067), (5, 3068),                  # the same with a partly filled first page
])
def test_one_sequence(stlib, before, rows):
    run = _run(512, 4, 71)
    m = run.create()
    if before:
        run.append([m], before, ("before",))
    run.append([m], rows, ("rows",))
    _check(run, [m])


@pytest.mark.parametrize("n_aux", [4, 31, 32, 33])   # 32: the most branches and copies in the parameters
@pytest.mark.parametrize("rows", [1, 20])
def test_forks_that_copy_and_grow(stlib, n_aux, rows):
    # the children's whole tables are new to the device when the append
    # refreshes them; all but the last holder copy the shared partial page
    run = _run(1024, 40, 72, D=128)
    m = run.create()
    run.append([m], 1000, ("prefix",))
    aux = run.fork(m, n_aux)
    run.append(aux, rows, ("rows",))
    _check(run, [m] + aux)
    run.append([m] + aux[:3], 17, ("more",))
    _check(run, [m] + aux)


def test_forks_not_appended_to_are_refreshed_too(stlib):
    run = _run(512, 12, 73)
    m, other = run.create(), run.create()
    run.append([m], 333, ("prefix",))
    run.append([other], 50, ("other",))
    aux = run.fork(m, 4)                    # their tables go up with the append below
    run.append([other], 30, ("rows",))
    _check(run, [other] + aux)


@pytest.mark.parametrize("pages,n_long,n_short,rows", [
    (1023, 1, 3, 1), (1024, 1, 3, 1), (1025, 1, 3, 1), (2050, 2, 40, 1),   # runs of 1024 entries at most
    (1025, 1, 3, 0), (5000, 1, 300, 0),                                    # the refresh as a launch of its own
    (1030, 520, 30, 0), (1030, 520, 30, 1),                                # more entries than a staging slot holds
    (4, 4200, 0, 1),                                                       # more runs than a staging slot's list
])
def test_device_tables_of_long_and_short_ranges(stlib, pages, n_long, n_short, rows):
    """Every live table on the device, entry by entry: ranges longer than a run
    beside short ones, refreshed by an append (rows > 0) or ahead of a decode."""
    import torch
    n = n_long + n_short + 8
    w = Workload(name="ranges", n_layers=1, n_q_heads=1, n_kv_heads=1, head_dim=64, n_blocks=pages + 64, seed=74)
    run = Run(w, max_seqs=n, max_decode_branches=2, max_splits=4, max_pages=pages + 8)
    long, short, x = run.create(), run.create(), run.create()
    run.append([long], 16 * pages - 3, ("long",))
    run.append([short], 20, ("short",))
    run.append([x], 5, ("x",))
    run.decode([x], ("q",))                               # every table so far is on the device
    live = [long, short, x] + run.fork(short, n_short // 2) + run.fork(long, n_long) + run.fork(short, n_short - n_short // 2)
    if rows:
        run.append([x], rows, ("rows",))
    else:
        run.decode([x], ("q",))
    run.pool.sync()
    tables = run.pool.workspace[256:256 + 4 * n * (pages + 8)].view(torch.int32).view(n, pages + 8).cpu()
    for r in live:
        h = run.handle[r]
        table, _ = run.pool.block_table(h)
        assert tables[h & 0xffffffff, :len(table)].tolist() == table, r
