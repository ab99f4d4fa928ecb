"""A plan's pooled launch slots: one per stream while they last, taken over by
another stream once idle, and none left when sixteen streams hold them.

The blocking verifies sum into a slot when there is one and into the plan's
scratch otherwise; both ways must name the damaged buckets.  The stream-ordered
verifying unpack leaves the caller's scratch alone when it holds a slot, and
zeroes and uses it otherwise: that tells which way a call went.
"""
import ctypes
import threading

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


MARK = 0x5EED


def checked_unpack(plan, buf, stream):
    """Enqueues a stream-ordered verifying unpack; its marked scratch, its result."""
    scratch = torch.full((plan.n_buckets + 4,), MARK, dtype=torch.int64, device="cuda")
    result = torch.full((2,), 7, dtype=torch.int64, device="cuda")
    torch.cuda.current_stream().synchronize()
    rr.rr_unpack_verify_async(plan, buf.buckets, buf.checksums, buf.dst, scratch, result,
                              stream=stream)
    return scratch, result


def held_slot(scratch, result):
    assert result.cpu().tolist() == [0, -1]
    return bool((scratch == MARK).all())


def test_many_streams_one_after_another():
    """More streams than slots over a plan's life: each finds an idle slot for its
    first launch."""
    plan, L, buf, (want, want_cs) = setup()
    for i in range(40):
        s = torch.cuda.Stream()
        scratch, result = checked_unpack(plan, buf, s)
        s.synchronize()
        assert held_slot(scratch, result), f"stream {i}"
        b = H.alloc(plan, flat=buf.flat)
        s.wait_stream(torch.cuda.current_stream())
        rr.rr_pack(plan, b.shards, b.buckets, b.checksums, stream=s)
        assert rr.rr_unpack_verify(plan, b.buckets, b.checksums, b.dst, stream=s) == (0, -1)
        np.testing.assert_array_equal(H.buckets_host(b), want)
        np.testing.assert_array_equal(H.checksums_host(b), want_cs)


@pytest.mark.parametrize("n", [16, 17, 24])
def test_streams_used_in_turn(n):
    """As many streams as slots and more (the set-up's stream holds one too), one
    after the other and round again: every call holds a slot, its own or one whose
    last launch has ended, however many launches came in between."""
    plan, L, buf, (want, want_cs) = setup()
    streams = [torch.cuda.Stream() for _ in range(n)]
    missed = []
    for turn in range(4):
        for i, s in enumerate(streams):
            scratch, result = checked_unpack(plan, buf, s)
            s.synchronize()
            if not held_slot(scratch, result):
                missed.append((turn, i))
    assert not missed
    for t in range(plan.n_tensors):
        np.testing.assert_array_equal(H.tensor_host(buf, t), L.unpack_tensor(want, t))


def test_no_slot_while_sixteen_streams_hold_them():
    """A seventeenth stream's calls fall back while the others' launches are in
    flight (every stream-ordered call, outputs as the oracle's), and hold a slot
    again once those have ended."""
    if not hasattr(torch.cuda, "_sleep"):
        pytest.skip("this PyTorch has no bounded sleep kernel to hold the streams")
    plan, L, buf, (want, want_cs) = setup()
    want_t = [L.unpack_tensor(want, t) for t in range(plan.n_tensors)]
    busy = [H.alloc(plan, flat=buf.flat) for _ in range(16)]
    streams = [torch.cuda.Stream() for _ in busy]
    mine = torch.cuda.Stream()
    whole, part, plain, fused = (H.alloc(plan, flat=buf.flat) for _ in range(4))
    n = plan.n_buckets
    torch.cuda.synchronize()
    for b, s in zip(busy, streams):
        with torch.cuda.stream(s):
            torch.cuda._sleep(SLEEP_CYCLES)
            rr.rr_pack(plan, b.shards, b.buckets, b.checksums, stream=s)
    rr.rr_pack(plan, whole.shards, whole.buckets, whole.checksums, stream=mine)
    rr.rr_pack_range(plan, 2, n - 5, part.shards, part.buckets, part.checksums, stream=mine)
    rr.rr_unpack(plan, buf.buckets, plain.dst, stream=mine)
    rr.rr_unpack_range(plan, 0, n, buf.buckets, part.dst, stream=mine)
    scratch = torch.full((n + 4,), MARK, dtype=torch.int64, device="cuda")
    result = torch.full((2,), 7, dtype=torch.int64, device="cuda")
    mine.wait_stream(torch.cuda.current_stream())
    rr.rr_unpack_verify_async(plan, buf.buckets, buf.checksums, fused.dst, scratch, result,
                              stream=mine)
    torch.cuda.synchronize()
    assert not held_slot(scratch, result), "a slot while all are held"
    np.testing.assert_array_equal(H.buckets_host(whole), want)
    np.testing.assert_array_equal(H.checksums_host(whole), want_cs)
    np.testing.assert_array_equal(H.buckets_host(part)[2:n - 3], want[2:n - 3])
    np.testing.assert_array_equal(H.checksums_host(part)[2:n - 3], want_cs[2:n - 3])
    for b in (plain, part, fused):
        for t in range(plan.n_tensors):
            np.testing.assert_array_equal(H.tensor_host(b, t), want_t[t])
    for b in busy:
        np.testing.assert_array_equal(H.buckets_host(b), want)
        np.testing.assert_array_equal(H.checksums_host(b), want_cs)
    scratch, result = checked_unpack(plan, buf, mine)
    mine.synchronize()
    assert held_slot(scratch, result), "no slot although all are idle"


def test_per_thread_default_stream():
    """cudaStreamPerThread is one handle for another stream in every thread: calls
    on it from several threads at once, each on buffers of its own."""
    plan, L, buf, (want, want_cs) = setup()
    want_t = [L.unpack_tensor(want, t) for t in range(plan.n_tensors)]
    per_thread = 2   # cudaStreamPerThread
    lib = ctypes.CDLL("libcudart.so.13")
    bufs = [H.alloc(plan, flat=buf.flat) for _ in range(6)]
    scratch = [torch.zeros(plan.n_buckets + 4, dtype=torch.int64, device="cuda") for _ in bufs]
    results = [torch.full((40, 2), 7, dtype=torch.int64, device="cuda") for _ in bufs]
    ids, errors = {}, []
    ready = threading.Barrier(len(bufs))
    torch.cuda.synchronize()

    def work(k):
        try:
            torch.cuda.set_device(0)
            sid = ctypes.c_ulonglong(0)
            assert lib.cudaStreamGetId(ctypes.c_void_p(per_thread), ctypes.byref(sid)) == 0
            ids[k] = sid.value
            ready.wait()
            b = bufs[k]
            for i in range(40):
                rr.rr_pack(plan, b.shards, b.buckets, b.checksums, stream=per_thread)
                rr.rr_unpack_verify_async(plan, b.buckets, b.checksums, b.dst, scratch[k],
                                          results[k][i], stream=per_thread)
            assert rr.rr_verify(plan, b.buckets, b.checksums, stream=per_thread) == (0, -1)
        except Exception as exc:   # reported by the main thread
            errors.append(exc)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(bufs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert len(set(ids.values())) == len(bufs), "one stream id for several threads' streams"
    for b, r in zip(bufs, results):
        assert (r == torch.tensor([0, -1], device="cuda")).all()
        np.testing.assert_array_equal(H.buckets_host(b), want)
        np.testing.assert_array_equal(H.checksums_host(b), want_cs)
        for t in range(plan.n_tensors):
            np.testing.assert_array_equal(H.tensor_host(b, t), want_t[t])
