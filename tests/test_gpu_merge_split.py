"""Merges whose row tiles are split over a cluster of CTAs, and tiles of at
most 128 rows, whose two halves of the tensor memory take the stages in turn:
against the float64 oracle at the sizes where a part, a stage or a tile begins
or ends.  A stage is 128 keys and a part at least 4 stages."""
import pytest
import torch

from fg_harness import Run, compare
from oracle import attention as A
from workloads import Workload, kv_rows, queries

pytestmark = pytest.mark.gpu


def _merge(D, Hq, Hkv, ctx, T, L=1):
    w = Workload(name=f"split_{D}_{Hq}_{Hkv}_{ctx}_{T}", n_layers=L, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D,
                 n_blocks=(ctx + T) // 16 + 8, seed=51)
    run = Run(w, max_seqs=2, max_decode_branches=1, max_splits=2)
    m = run.create()
    if ctx:
        run.append([m], ctx, ("ctx",))
    q, o, lse, L0 = run.merge(m, T, ("rows",))
    run.pool.sync()
    for layer in range(L):
        k, v = run.context(m, layer)
        o_ref, l_ref = A.merge_prefill(q[layer].cpu(), k, v, L0)
        compare(o[layer], lse[layer], o_ref, l_ref, f"layer {layer}")


@pytest.mark.parametrize("ctx,T", [
    (0, 1),                  # one key: one stage, tile B without any
    (127, 1), (128, 1),      # one stage full, a second one with one key
    (300, 32),               # 128 rows: the largest tile that takes the stages in turn
    (300, 33),               # 132 rows: the smallest of two tiles
    (1022, 2),               # 8 stages, 2 parts, the last key the last of its part
    (1023, 2),               # 9 stages: the last part's last stage holds one key
    (510, 130),              # causal limits on both sides of a part's first key
    (4096, 20), (6000, 45),  # parts of 4 and 5 stages
])
def test_merge_at_part_and_stage_edges(stlib, ctx, T):
    _merge(128, 32, 8, ctx, T)


@pytest.mark.parametrize("ctx,T", [(130, 3), (2050, 16), (9000, 40)])
def test_merge_split_head_dim_64(stlib, ctx, T):
    _merge(64, 8, 2, ctx, T)          # 2 row tiles or fewer: clusters of up to 16


def test_merge_split_over_many_stages(stlib):
    _merge(128, 8, 1, 20000, 5)       # one row tile: the largest cluster


def test_batch_of_short_and_long_tiles_in_one_cluster_size(stlib):
    # the launch's clusters suit the long context; the short ones have fewer
    # parts than a cluster has CTAs, or one
    w = Workload(name="split_batch", n_layers=2, n_q_heads=32, n_kv_heads=8, head_dim=128, n_blocks=1024, seed=52)
    run = Run(w, max_seqs=4, max_decode_branches=1, max_splits=2)
    lens, counts, rids = (9000, 5, 1500), (9, 70, 33), []
    for i, n in enumerate(lens):
        rids.append(run.create())
        run.append([rids[-1]], n, ("ctx", i))
    q, o, lse, L0 = run.prefill_batch(rids, counts, ("rows",))
    run.pool.sync()
    at = 0
    for r, n, l0 in zip(rids, counts, L0):
        for layer in range(2):
            k, v = run.context(r, layer)
            o_ref, l_ref = A.merge_prefill(q[layer, at:at + n].cpu(), k, v, l0)
            compare(o[layer, at:at + n], lse[layer, at:at + n], o_ref, l_ref, f"seq {r} layer {layer}")
        at += n


def test_layers_of_the_last_wave_in_a_launch_of_their_own(stlib):
    # 256 row tiles: 19 layers fill the SMs once, the other 13 are split
    L, ctx, T = 32, 26000, 40
    w = Workload(name="split_layers", n_layers=L, n_q_heads=32, n_kv_heads=8, head_dim=64, n_blocks=(ctx + T) // 16 + 8,
                 seed=53)
    run = Run(w, max_seqs=2, max_decode_branches=1, max_splits=2)
    m = run.create()
    for i in range(0, ctx, 6500):
        run.append([m], 6500, ("ctx", i))
    run.pool.profile_read()
    q, o, lse, L0 = run.merge(m, T, ("rows",))
    run.pool.sync()
    assert run.pool.profile_read()["merge_prefill"]["kernels"] == 2
    for layer in (0, 18, 19, L - 1):
        k, v = run.context(m, layer)
        o_ref, l_ref = A.merge_prefill(q[layer].cpu(), k, v, L0)
        compare(o[layer], lse[layer], o_ref, l_ref, f"layer {layer}")


@pytest.mark.parametrize("D,ctx,T", [(128, 300, 70), (64, 300, 70), (128, 40, 130), (128, 5000, 85), (64, 5000, 85)])
def test_short_last_tile_behind_the_others(stlib, D, ctx, T):
    # 280, 520 and 340 stacked rows in 3 layers of 8 heads: the last tile of 24, 8
    # and 84 rows comes behind the others of every head and layer, whole or split
    _merge(D, 32, 8, ctx, T, L=3)


def test_rows_merged_alone_and_among_others(stlib):
    """How a row tile's keys are split depends on what else is in the launch, so
    the same rows merged alone and in a batch may differ in their last bits, each
    within the tolerance.  The same call gives the same bits."""
    n, ctx, T = 16, 9000, 20
    w = Workload(name="split_among", n_layers=1, n_q_heads=32, n_kv_heads=8, head_dim=128,
                 n_blocks=n * ((ctx + T) // 16 + 2), seed=54)
    outs = []
    for batch, seed in ((True, 1), (True, 2), (False, 1)):
        run = Run(w, max_seqs=n, max_decode_branches=1, max_splits=2, pool_seed=seed)
        rids = [run.create() for _ in range(n)]
        for i, r in enumerate(rids):
            run.append([r], ctx, ("ctx", i))
        if batch:
            q, o, lse, L0 = run.prefill_batch(rids, [T] * n, ("rows",))
        else:                               # the last sequence's rows of the batch by themselves
            k, v = kv_rows(w, ("rows",), n * T, device="cuda")
            q = queries(w, ("prefill_q", "rows"), n * T, device="cuda")
            rows = slice((n - 1) * T, n * T)
            o, lse = run.pool.merge(run.handle[rids[-1]], q[:, rows].contiguous(), k[:, rows].contiguous(),
                                    v[:, rows].contiguous())
        run.pool.sync()
        outs.append((o.cpu(), lse.cpu()))
        if len(outs) == 1:
            ctx_k, ctx_v = run.context(rids[-1], 0)
            o_ref, l_ref = A.merge_prefill(q[0, (n - 1) * T:].cpu(), ctx_k, ctx_v, ctx)
        run.pool.close()
    (o1, l1), (o2, l2), (o3, l3) = outs
    assert torch.equal(o1, o2) and torch.equal(l1, l2)
    assert not torch.equal(o1[:, (n - 1) * T:], o3)      # other parts, another order of the sums
    compare(o1[0, (n - 1) * T:], l1[0, (n - 1) * T:], o_ref, l_ref, "among others")
    compare(o3[0], l3[0], o_ref, l_ref, "alone")
