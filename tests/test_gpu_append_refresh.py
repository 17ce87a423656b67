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
