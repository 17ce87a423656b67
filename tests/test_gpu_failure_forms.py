"""Waits that run out in the forms of the attention kernels that launches of more
than one wave, of several tiles, or with few row tiles take: persistent decode
CTAs (narrow, wide, paired), narrow items beside large tiles, merges split over a
cluster, and merges in two launches.  With ST_FLAG_HOLD_LOADS the loaders issue
nothing; every CTA gives up after its limit (2 s) and winds down, a cluster's CTAs
through the cluster barriers, whose own wait has no limit and ends because each of
them gets there.  st_sync reports the timeout, the next one is clean, and the
device then works as before."""
import time

import pytest
import torch

import paper_2608_13667_gb300 as stpkg
from fg_harness import Run, compare
from oracle import attention as A
from workloads import Workload, kv_rows, queries

pytestmark = pytest.mark.gpu


def _pool(w, max_seqs, flags=0):
    return stpkg.Pool(n_layers=w.n_layers, n_q_heads=w.n_q_heads, n_kv_heads=w.n_kv_heads, head_dim=w.head_dim,
                      n_blocks=w.n_blocks, seed=w.seed, max_seqs=max_seqs, max_decode_branches=max_seqs,
                      max_splits=32, flags=flags)


def _append(pool, w, seqs, n, tag):
    k, v = kv_rows(w, tag, len(seqs) * n, device="cuda")
    shape = (w.n_layers, len(seqs), n, w.n_kv_heads, w.head_dim)
    pool.append_kv(seqs, k.view(shape), v.view(shape))


def _runs_out(pool, call):
    t0 = time.time()
    call()
    with pytest.raises(stpkg.STError) as e:
        pool.sync()
    assert e.value.status == stpkg.ST_ERR_TIMEOUT
    assert time.time() - t0 < 90
    pool.sync()                              # the status word was cleared


def _works_still():
    w = Workload(name="after", n_layers=1, n_q_heads=8, n_kv_heads=2, head_dim=128, n_blocks=64, seed=93)
    run = Run(w, max_seqs=2, max_decode_branches=1, max_splits=4)
    m = run.create()
    run.append([m], 300, ("ctx",))
    q, o, lse = run.decode([m], ("q",))
    run.pool.sync()
    o_ref, l_ref = run.oracle_decode([m], q, 0)
    compare(o[0], lse[0], o_ref, l_ref, "decode after the timeout")
    q, o, lse, L0 = run.merge(m, 20, ("rows",))
    run.pool.sync()
    o_ref, l_ref = A.merge_prefill(q[0].cpu(), *run.context(m, 0), L0)
    compare(o[0], lse[0], o_ref, l_ref, "merge after the timeout")


@pytest.mark.parametrize("groups,singles,prefix,form", [
    ((), 10, 500, "narrow"),
    ((9,), 0, 4000, "wide"),
    ((17,), 0, 4000, "paired"),
    ((9, 17), 14, 1100, "narrow beside"),   # more than four waves of narrow items
])
def test_decode_of_more_than_one_wave(stlib, groups, singles, prefix, form):
    L, Hkv, G = 4, 8, 8
    n = sum(groups) + singles
    w = Workload(name="hold_" + form, n_layers=L, n_q_heads=Hkv * G, n_kv_heads=Hkv, head_dim=128, n_blocks=4096, seed=91)
    pool = _pool(w, n, stpkg.ST_FLAG_HOLD_LOADS)
    seqs = []
    for g, size in enumerate(groups):
        m = pool.seq_create()
        _append(pool, w, [m], prefix, ("prefix", g))
        seqs += [m] + pool.fork(m, size - 1)
    for i in range(singles):
        seqs.append(pool.seq_create())
        _append(pool, w, [seqs[-1]], 500, ("single", i))
    items, _, _ = pool.decode_plan(seqs)
    ctas = {f: sum(1 for it in items if it["flags"] & 6 == f) * Hkv * L for f in (0, 2, 4)}
    assert {"narrow": ctas[0] > 304, "wide": ctas[2] > 304, "paired": ctas[4] > 152,
            "narrow beside": ctas[0] > 1216 and ctas[2] and ctas[4]}[form]
    # pages that do not stay in L2, as its half decides between the narrow tile's forms
    assert form in ("wide", "paired") or sum(it["n_pages"] for it in items) * 16 * Hkv * 128 * 4 * L > 68e6
    kn, vn = kv_rows(w, ("new",), n, device="cuda")
    q = queries(w, ("q",), n, device="cuda")
    _runs_out(pool, lambda: pool.decode_step(seqs, kn, vn, q))
    # every row of the step is stored all the same
    for i, h in enumerate(seqs):
        table, length = pool.block_table(h)
        page, row = table[(length - 1) // 16], (length - 1) % 16
        assert torch.equal(pool.k_pool[:, page, :, row], kn[:, i])
        assert torch.equal(pool.v_pool[:, page, :, row], vn[:, i])
    pool.close()
    _works_still()


@pytest.mark.parametrize("D,L,ctx,T,kernels", [
    (128, 1, 5000, 20, 1), (64, 1, 5000, 20, 1),   # one row tile per head, shared by both tiles, in a cluster
    (128, 1, 9000, 133, 1),                        # three
    (64, 32, 26000, 40, 2),                        # whole waves, and the other layers in a split launch
])
def test_split_merge(stlib, D, L, ctx, T, kernels):
    w = Workload(name=f"holds_{D}_{L}_{T}", n_layers=L, n_q_heads=32, n_kv_heads=8, head_dim=D,
                 n_blocks=(ctx + T) // 16 + 8, seed=92)
    pool = _pool(w, 1, stpkg.ST_FLAG_HOLD_LOADS)
    m = pool.seq_create()
    for i in range(0, ctx, 6500):
        _append(pool, w, [m], min(6500, ctx - i), ("ctx", i))
    k, v = kv_rows(w, ("rows",), T, device="cuda")
    q = queries(w, ("q",), T, device="cuda")
    pool.profile_read()
    _runs_out(pool, lambda: pool.merge(m, q, k, v))
    assert pool.profile_read()["merge_prefill"]["kernels"] == kernels
    pool.close()
    _works_still()


def test_batch_of_unequal_splits(stlib):
    # clusters for the long context; the short ones leave CTAs without a part
    w = Workload(name="holds_batch", n_layers=2, n_q_heads=32, n_kv_heads=8, head_dim=128, n_blocks=1024, seed=94)
    pool = _pool(w, 3, stpkg.ST_FLAG_HOLD_LOADS)
    lens, counts = (9000, 5, 1500), (9, 70, 33)
    seqs = [pool.seq_create() for _ in lens]
    for i, (s, n) in enumerate(zip(seqs, lens)):
        _append(pool, w, [s], n, ("ctx", i))
    R = sum(counts)
    k, v = kv_rows(w, ("rows",), R, device="cuda")
    q = queries(w, ("q",), R, device="cuda")
    _runs_out(pool, lambda: pool.prefill_batch(seqs, counts, q, k, v))
    pool.close()
    _works_still()
