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


@pytest.mark.parametrize("D,Hq,Hkv", [(128, 32, 8), (64, 32, 8), (128, 64, 4)])
def test_items_of_many_shapes_taken_over(stlib, D, Hq, Hkv):
    """More than one wave of CTAs, so that each takes over further items: runs
    of one page to many, of one branch to a whole group (one to four softmax
    warps), short last pages, and groups on the wide tile."""
    L = 24 if D == 64 else 12
    w = Workload(name=f"taken_{D}_{Hq}_{Hkv}", n_layers=L, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D, n_blocks=2048,
                 seed=62)
    run = Run(w, max_seqs=64, max_decode_branches=48, max_splits=16)
    rids = []
    for g, (prefix, n_aux) in enumerate(((2000, 4), (640, 15), (5000, 1), (330, 12))):
        m = run.create()
        run.append([m], prefix, ("prefix", g))
        family = [m] + run.fork(m, n_aux)
        for i, r in enumerate(family):
            if (i + g) % 3:
                run.append([r], 1 + 13 * i, ("suffix", g, i))
        rids += family
    for i, n in enumerate((1, 15, 64, 65, 300, 1100)):
        rids.append(run.create())
        run.append([rids[-1]], n, ("single", i))
    assert len(run.pool.decode_plan([run.handle[r] for r in rids])[0]) * Hkv * L > 2 * 304
    for step in range(2):     # the rings and the slots start anew with every launch
        q, o, lse = run.decode(rids, ("q", step))
        run.pool.sync()
        for layer in (0, L - 1):
            o_ref, l_ref = run.oracle_decode(rids, q, layer)
            compare(o[layer], lse[layer], o_ref, l_ref, f"step {step} layer {layer}")
    # the rows of a step are stored by the items that are taken over
    from workloads import kv_rows, queries
    k, v = kv_rows(w, ("new",), len(rids), device="cuda")
    q = queries(w, ("newq",), len(rids), device="cuda")
    o, lse = run.pool.decode_step([run.handle[r] for r in rids], k, v, q)
    run.pool.sync()
    run.ref.append(rids, 1)
    run.sizes[("new",)] = len(rids)
    for i, r in enumerate(rids):
        run.hist[r].append((("new",), i, 1))
    o_ref, l_ref = run.oracle_decode(rids, q, L - 1)
    compare(o[L - 1], lse[L - 1], o_ref, l_ref, "step with new rows")


def test_many_short_items_beside_a_wide_tile(stlib):
    """Groups on the wide tile with more than four waves of one-page items
    beside them: those take over from one another and all wait for the tiles."""
    L = 16
    w = Workload(name="beside_many", n_layers=L, n_q_heads=32, n_kv_heads=8, head_dim=64, n_blocks=1024, seed=63)
    run = Run(w, max_seqs=64, max_decode_branches=40, max_splits=16)
    rids = []
    for g, n_aux in enumerate((19, 16)):      # 80 and 68 stacked rows
        m = run.create()
        run.append([m], 2600 + 16 * g, ("prefix", g))
        family = [m] + run.fork(m, n_aux)
        run.append(family, 3 + g, ("suffix", g))
        rids += family
    items, _, _ = run.pool.decode_plan([run.handle[r] for r in rids])
    assert sum(1 for it in items if not it["flags"]) * 8 * L > 4 * 304
    for step in range(2):
        q, o, lse = run.decode(rids, ("q", step))
        run.pool.sync()
        for layer in (0, L - 1):
            o_ref, l_ref = run.oracle_decode(rids, q, layer)
            compare(o[layer], lse[layer], o_ref, l_ref, f"step {step} layer {layer}")


@pytest.mark.parametrize("D", [64, 128])
def test_paired_items_taken_over(stlib, D):
    """More than one wave of CTAs on the paired tile, so that each takes over
    further items: runs of one page to many, short last stages, one row to all
    128 in the second tile, and a group split into two."""
    L = 12
    w = Workload(name=f"paired_taken_{D}", n_layers=L, n_q_heads=64, n_kv_heads=8, head_dim=D, n_blocks=2048, seed=64)
    run = Run(w, max_seqs=192, max_decode_branches=160, max_splits=16)
    rids = []
    for g, (prefix, n_aux) in enumerate(((2000, 16), (16, 31), (6016, 23), (130 * 16, 40), (144, 20))):
        m = run.create()
        run.append([m], prefix, ("prefix", g))
        family = [m] + run.fork(m, n_aux)
        run.append(family[::2], 3 + g, ("suffix", g))
        rids += family
    items, _, _ = run.pool.decode_plan([run.handle[r] for r in rids])
    paired = [it for it in items if it["n_members"] * 8 > 128]
    assert len(paired) * 8 * L > 2 * 152 and len({it["n_pages"] for it in paired}) > 2
    for step in range(2):     # the rings and the slots start anew with every launch
        q, o, lse = run.decode(rids, ("q", step))
        run.pool.sync()
        for layer in (0, L - 1):
            o_ref, l_ref = run.oracle_decode(rids, q, layer)
            compare(o[layer], lse[layer], o_ref, l_ref, f"step {step} layer {layer}")
