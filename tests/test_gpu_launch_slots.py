"""A plan's pooled launch slots: one per stream while they last, taken over by
another stream once idle, and none left when sixteen streams hold them.

The blocking verifies sum into a slot when there is one and into the plan's
scratch otherwise; both ways must name the damaged buckets.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_22492_gb300 as rr
from tests import _util as U
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu

SLEEP_CYCLES = 100_000_000   # about 50 ms: longer than enqueueing the calls below


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


def setup():
    desc = U.workload_desc("tiny-tp4")
    plan = H.make_plan(*U.to_product(desc), desc["bucket_bytes"])
    L = U.to_oracle(desc)
    shards = L.host_shards(desc["seed"], desc["specials"])
    buf = H.alloc(plan)
    H.fill_from_host(buf, shards)
    H.pack(buf)
    torch.cuda.synchronize()
    return plan, L, buf, L.pack(oracle.Source(shards=shards))


def damaged_copy(plan, buf, hit):
    other = H.alloc(plan, flat=buf.flat)
    other.bucket_store.copy_(buf.bucket_store)
    other.checksums.copy_(buf.checksums)
    for b in hit:
        H.bucket_list(other)[b][8] ^= 1
    torch.cuda.synchronize()
    return other


@pytest.mark.parametrize("held", [0, 15, 16, 20])
def test_blocking_verifies_while_other_streams_hold_slots(held):
    if not hasattr(torch.cuda, "_sleep"):
        pytest.skip("this PyTorch has no bounded sleep kernel to hold the streams")
    plan, L, buf, (want, want_cs) = setup()
    hit = [3, plan.n_buckets - 1]
    other = damaged_copy(plan, buf, hit)
    busy = [H.alloc(plan, flat=buf.flat) for _ in range(held)]
    streams = [torch.cuda.Stream() for _ in busy]
    mine = torch.cuda.Stream()
    torch.cuda.synchronize()
    for b, s in zip(busy, streams):
        with torch.cuda.stream(s):
            torch.cuda._sleep(SLEEP_CYCLES)
            rr.rr_pack(plan, b.shards, b.buckets, b.checksums, stream=s)
    bad = torch.full((plan.n_buckets,), 9, dtype=torch.uint8, device="cuda")
    mine.wait_stream(torch.cuda.current_stream())
    flags = np.zeros(plan.n_buckets, np.uint8)
    flags[hit] = 1
    for _ in range(2):
        assert rr.rr_verify_range(plan, 0, plan.n_buckets, other.buckets, other.checksums, bad,
                                  stream=mine) == (2, 3)
        np.testing.assert_array_equal(bad.cpu().numpy(), flags)
        assert rr.rr_verify_range(plan, 4, plan.n_buckets - 5, other.buckets, other.checksums,
                                  stream=mine) == (0, -1)
        assert rr.rr_unpack_verify(plan, other.buckets, other.checksums, other.dst, bad=bad,
                                   stream=mine) == (2, 3)
        np.testing.assert_array_equal(bad.cpu().numpy(), flags)
    torch.cuda.synchronize()
    for b in busy:
        np.testing.assert_array_equal(H.buckets_host(b), want)
        np.testing.assert_array_equal(H.checksums_host(b), want_cs)


def test_many_streams_one_after_another():
    """More streams than slots over a plan's life: each finds an idle slot."""
    plan, L, buf, (want, want_cs) = setup()
    for i in range(40):
        s = torch.cuda.Stream()
        b = H.alloc(plan, flat=buf.flat)
        s.wait_stream(torch.cuda.current_stream())
        rr.rr_pack(plan, b.shards, b.buckets, b.checksums, stream=s)
        assert rr.rr_unpack_verify(plan, b.buckets, b.checksums, b.dst, stream=s) == (0, -1)
        np.testing.assert_array_equal(H.buckets_host(b), want)
        np.testing.assert_array_equal(H.checksums_host(b), want_cs)
