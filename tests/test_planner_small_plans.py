"""Work tables of small plans: every block gets its work up front.

A plan with less than a 64 KiB item for every block cuts its items so that each
block has two; a small table's per-bucket units are no more than the grid has
blocks, and the whole-sync pack's own units hold every item (nothing is left to
claim).  The tables reproduce the oracle's bytes as any other's.
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
    full, _ = plan.export_pack_full()
    whole, _ = U.check_units(plan, len(full), "pack_full")
    if small:
        if len(uitems) < 8 * grid and plan.n_buckets <= grid // 2:
            assert len(units) - 1 <= grid
        assert whole[grid] == len(full), "a claimed unit holds items"
    shards = L.host_shards(desc["seed"], desc["specials"])
    want, _ = L.pack(oracle.Source(shards=shards))
    for table in (items, full):
        got = U.check_and_run_pack(table, shards, plan.n_buckets, plan.bucket_bytes,
                                   plan.shard_bytes)
        np.testing.assert_array_equal(got, want)
