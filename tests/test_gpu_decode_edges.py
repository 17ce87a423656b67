"""Decode at the sizes where its rings and its combine change form, against
the float64 oracle: contexts of one stage (64 keys) fewer and more than a ring
has slots, for both head dims and both tiles, and calls on either side of the
row count up to which the combine gives a row four warps."""
import pytest

from fg_harness import Run, compare
from workloads import Workload

pytestmark = pytest.mark.gpu


def _decode(D, Hq, Hkv, L, prefix, n_aux, suffix, max_splits=16, layers=None):
    w = Workload(name=f"edge_{D}_{Hq}_{Hkv}_{L}_{prefix}_{n_aux}", n_layers=L, n_q_heads=Hq, n_kv_heads=Hkv,
                 head_dim=D, n_blocks=prefix // 16 + (n_aux + 1) * (suffix // 16 + 3) + 8, seed=61)
    run = Run(w, max_seqs=n_aux + 2, max_decode_branches=n_aux + 1, max_splits=max_splits)
    m = run.create()
    run.append([m], prefix, ("prefix",))
    rids = [m] + run.fork(m, n_aux)
    if suffix:
        run.append(rids, suffix, ("suffix",))
    q, o, lse = run.decode(rids, ("q",))
    run.pool.sync()
    for layer in (layers or range(L)):
        o_ref, l_ref = run.oracle_decode(rids, q, layer)
        compare(o[layer], lse[layer], o_ref, l_ref, f"layer {layer}")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("stages", [1, 2, 3, 4, 5, 6, 7, 13])
@pytest.mark.parametrize("n_aux", [4, 8])    # 40 rows: narrow; 72 rows: wide
def test_stage_counts_around_the_ring(stlib, D, stages, n_aux):
    _decode(D, 16, 2, 1, 64 * stages, n_aux, 5)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("L", [19, 20])      # 2432 and 2560 rows: four warps a row, one warp a row
def test_combine_forms(stlib, D, L):
    _decode(D, 32, 8, L, 16 * 16 * 9, 3, 20, max_splits=32, layers=(0, L - 1))
