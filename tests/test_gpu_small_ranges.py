"""Calls over ranges of a small plan's buckets, whose blocks take equal runs of
the range's units without claiming: fewer units than blocks, one more than some
multiple of them, and a single block for all; on both engines and against the
oracle, with everything outside the range untouched."""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_22492_gb300 as rr
from tests import _util as U
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


@pytest.mark.parametrize("engine", ["auto", "registers"])
@pytest.mark.parametrize("grid", [0, 1, 7, 1000])
@pytest.mark.parametrize("name", ["tiny-tp4", "tiny-moe-tp2"])
def test_ranges(name, grid, engine):
    desc = U.workload_desc(name)
    L = U.to_oracle(desc)
    plan = H.make_plan(*U.to_product(desc), desc["bucket_bytes"], grid_blocks=grid, engine=engine)
    shards = L.host_shards(desc["seed"], desc["specials"])
    want, want_cs = L.pack(oracle.Source(shards=shards))
    want_t = [L.unpack_tensor(want, t) for t in range(plan.n_tensors)]
    buf = H.alloc(plan)
    H.fill_from_host(buf, shards)
    n, B = plan.n_buckets, plan.bucket_bytes
    scratch = torch.zeros(n + 4, dtype=torch.int64, device="cuda")
    result = torch.full((2,), 7, dtype=torch.int64, device="cuda")
    pos = [plan.first_bucket_of_rank[plan.tensor_ranks[t]] * B + plan.tensor_stream_offset[t] +
           2 * np.arange(plan.tensor_numel[t], dtype=np.int64) for t in range(plan.n_tensors)]
    for b0, count in [(0, n), (0, 1), (n - 1, 1), (1, n - 2), (n // 2, n // 4)]:
        for b in H.bucket_list(buf):
            b.fill_(0xAB)
        buf.checksums.fill_(0x1234)
        for t in buf.dst:
            t.fill_(0x5A5A)
        rr.rr_pack_range(plan, b0, count, buf.shards, buf.buckets, buf.checksums)
        rr.rr_unpack_verify_async(plan, buf.buckets, buf.checksums, buf.dst, scratch, result,
                                  first_bucket=b0, n_buckets=count)
        got, cs = H.buckets_host(buf), buf.checksums.cpu().numpy().view(np.uint64)
        inside = np.zeros(n, bool)
        inside[b0:b0 + count] = True
        np.testing.assert_array_equal(got[inside], want[inside])
        np.testing.assert_array_equal(cs[inside], np.asarray(want_cs, np.uint64)[inside])
        assert np.all(got[~inside] == 0xAB) and np.all(cs[~inside] == 0x1234)
        assert result.cpu().tolist() == [0, -1]
        for again in range(2):   # the verifying unpack's tensors, then the plain unpack's
            for t in range(plan.n_tensors):
                mine = (pos[t] >= b0 * B) & (pos[t] < (b0 + count) * B)
                have = H.tensor_host(buf, t)
                np.testing.assert_array_equal(have[mine], want_t[t][mine])
                assert np.all(have[~mine] == 0x5A5A)
                buf.dst[t].fill_(0x5A5A)
            rr.rr_unpack_range(plan, b0, count, buf.buckets, buf.dst)
    rr.rr_plan_check(plan)
