"""Work tables of small plans: every block gets its work up front.

A plan with less than a 64 KiB item for every block cuts its items so that each
block has two; a small table's per-bucket units are fine enough for a range of
its buckets to give every block some, and the whole-sync pack's own units hold
every item (nothing is left to claim).  The tables reproduce the oracle's bytes
as any other's.
"""
import numpy as np
import pytest

import oracle
import paper_2512_22492_gb300 as rr
from tests import _util as U


@pytest.mark.parametrize("grid", [5, 152, 304])
@pytest.mark.parametrize("name", ["tiny", "tiny-tp4", "tiny-moe-tp2", "tiny-fsdp2"])
def test_small_plan_tables(name, grid):
    desc = U.workload_desc(name)
    L = U.to_oracle(desc)
    plan = rr.rr_plan_create(*U.to_product(desc), desc["bucket_bytes"],
                             rr.PlanOptions(host_only=True, grid_blocks=grid))
    total = sum(plan.stream_bytes_per_rank)
    items, _ = plan.export_pack()
    uitems, _ = plan.export_unpack()
    n = 2 * items["row_len"].astype(np.int64) * items["n_rows"]
    small = total < 64 * 1024 * grid
    share = max(4096, -(-(total // (2 * grid) + 1) // 1024) * 1024)
    assert n.max() <= (min(64 * 1024, share) if small else 64 * 1024)
    assert uitems["nbytes"].max() <= (min(64 * 1024, share) if small else 64 * 1024)
    U.check_units(plan, len(items), "pack")
    units, _ = U.check_units(plan, len(uitems))
    assert not small or len(units) - 1 >= min(len(uitems), grid)
    full, _ = plan.export_pack_full()
    whole, _ = U.check_units(plan, len(full), "pack_full")
    if small:
        assert whole[grid] == len(full), "a claimed unit holds items"
    shards = L.host_shards(desc["seed"], desc["specials"])
    want, _ = L.pack(oracle.Source(shards=shards))
    for table in (items, full):
        got = U.check_and_run_pack(table, shards, plan.n_buckets, plan.bucket_bytes,
                                   plan.shard_bytes)
        np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("mi", [8, 20, 22, 24, 25, 26, 28, 40])
def test_small_tables_are_told_by_their_traffic(mi):
    """Under 1 MiB of traffic a block every unit of the whole-sync pack is a
    block's own; from there on 15% of the table's weight is left to claim.  An
    item weighs 1 KiB beyond its bytes where this is decided, whatever it weighs
    in the split that follows."""
    n, grid = mi << 20, 152
    plan = rr.rr_plan_create([rr.Param("a", (n,), "f32")], rr.SrcLayout(1),
                             rr.DstLayout(1, [rr.DstTensor("t", 0, [rr.Block(0, 0, n, 0, 1)])]),
                             1 << 20, rr.PlanOptions(host_only=True, grid_blocks=grid))
    full, _ = plan.export_pack_full()
    whole, _ = U.check_units(plan, len(full), "pack_full")
    small = 6 * n + 1024 * len(full) < (grid << 20)
    assert small == (mi < 26)
    own = whole[grid] / len(full)
    assert own == 1 if small else 0.8 < own < 0.9


@pytest.mark.parametrize("mi,dtype", [(2, "f32"), (4, "bf16"), (12, "f32"), (16, "bf16")])
def test_ranges_of_small_tables_have_units_for_every_block(mi, dtype):
    """A range of a small table's buckets: a unit for every block of the grid, or
    one for every item where there are fewer items."""
    n, grid = mi << 20, 152
    plan = rr.rr_plan_create([rr.Param("a", (n,), dtype)], rr.SrcLayout(1),
                             rr.DstLayout(1, [rr.DstTensor("t", 0, [rr.Block(0, 0, n, 0, 1)])]),
                             1 << 18, rr.PlanOptions(host_only=True, grid_blocks=grid))
    for which, items in zip(("pack", "unpack"), (plan.export_pack()[0], plan.export_unpack()[0])):
        U.check_units(plan, len(items), which)
        first, bucket_unit = plan.work_units(which)
        for part in (2, 4, 8):
            b0 = plan.n_buckets // 4
            b1 = b0 + plan.n_buckets // part
            u0, u1 = int(bucket_unit[b0]), int(bucket_unit[b1])
            n_items = int(first[u1]) - int(first[u0])
            assert u1 - u0 >= min(n_items, grid), (which, part)


@pytest.mark.parametrize("k,n,mi,dtype,pack_most,unpack_most",
                         [(1000, 2048, 12, "f32", 24, 16), (1500, 2048, 12, "bf16", 24, 16),
                          (3000, 256, 4, "f32", 64, 8), (3900, 512, 4, "f32", 64, 8)])
def test_short_items_of_small_tables_are_spread(k, n, mi, dtype, pack_most, unpack_most):
    """Many short tensors beside a large one: no block gets a long run of short
    items, each of which costs it about as much as 32 KiB of traffic.  (Where
    short items make up the pack table several share a stage, and cost less.)"""
    sizes = [n] * k + [mi << 20]
    plan = rr.rr_plan_create([rr.Param(f"p{i}", (s,), dtype) for i, s in enumerate(sizes)],
                             rr.SrcLayout(1),
                             rr.DstLayout(1, [rr.DstTensor(f"t{i}", 0, [rr.Block(i, 0, s, 0, 1)])
                                              for i, s in enumerate(sizes)]),
                             1 << 20, rr.PlanOptions(host_only=True, grid_blocks=152))
    whole, _ = U.check_units(plan, len(plan.export_pack_full()[0]), "pack_full")
    assert np.diff(whole[:153]).max() <= pack_most
    units, _ = U.check_units(plan, len(plan.export_unpack()[0]))
    assert np.diff(units).max() <= unpack_most


@pytest.mark.parametrize("n", [100_000, 1 << 20, 3_000_001, 8 << 20])
@pytest.mark.parametrize("engine", ["auto", "registers"])
def test_items_per_block_of_either_engine(n, engine):
    """Two items a block, and for the register path's unpacks, which move one item
    after the other, one."""
    grid = 304
    plan = rr.rr_plan_create([rr.Param("a", (n,), "f32")], rr.SrcLayout(1),
                             rr.DstLayout(1, [rr.DstTensor("t", 0, [rr.Block(0, 0, n, 0, 1)])]),
                             1 << 20, rr.PlanOptions(host_only=True, grid_blocks=grid,
                                                     engine=engine))
    total = sum(plan.stream_bytes_per_rank)

    def share(blocks):
        return max(4096, min(65536, -(-(total // blocks + 1) // 1024) * 1024))

    assert 2 * int(plan.export_pack()[0]["row_len"].max()) == share(2 * grid)
    assert int(plan.export_unpack()[0]["nbytes"].max()) == \
        share(2 * grid if engine == "auto" else grid)
