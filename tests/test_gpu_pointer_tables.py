"""Launches at the limits of the pointer tables: separately allocated buckets, as
many as a launch's 64, 448 or 3968 pointers hold and one more, on both engines
and through the standalone verifies; bytes and checksums against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_22492_gb300 as rr
from tests import _util as U
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu

BUCKET = 4096


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


@pytest.mark.parametrize("engine", ["auto", "registers"])
@pytest.mark.parametrize("n", [63, 64, 65, 447, 448, 449, 3967, 3968])
def test_separate_buckets(n, engine):
    numel = n * BUCKET // 2 - 5
    desc = dict(params=[("a", (numel,), 4)], tensors=[("t", 0, [(0, 0, numel, 0, 1)])],
                n_shards=1, tp=1, bucket_bytes=BUCKET, align_bytes=16, tensor_align=256)
    L = U.to_oracle(desc)
    plan = H.make_plan(*U.to_product(desc), BUCKET, engine=engine)
    assert plan.n_buckets == n
    shards = L.host_shards(n)
    want, want_cs = L.pack(oracle.Source(shards=shards))
    buf = H.alloc(plan, separate_buckets=True)
    H.fill_from_host(buf, shards)
    H.pack(buf)
    np.testing.assert_array_equal(H.buckets_host(buf), want)
    np.testing.assert_array_equal(H.checksums_host(buf), want_cs)
    assert rr.rr_unpack_verify(plan, buf.buckets, buf.checksums, buf.dst) == (0, -1)
    np.testing.assert_array_equal(H.tensor_host(buf, 0), L.unpack_tensor(want, 0))
    buf.dst[0].fill_(0)
    H.unpack(buf)
    np.testing.assert_array_equal(H.tensor_host(buf, 0), L.unpack_tensor(want, 0))
    H.bucket_list(buf)[n - 2][40] ^= 4
    assert H.verify(buf) == (1, n - 2)
    assert rr.rr_verify_noalloc(buf.buckets, n, BUCKET, buf.checksums) == (1, n - 2)
