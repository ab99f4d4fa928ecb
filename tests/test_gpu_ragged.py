"""Elements at any alignment through the bulk-copy engine, against the oracle.

The engine stages the 16-byte words around a run of misaligned elements (or
around each of several short rows) and re-cuts them at the destination's
16-byte boundaries.  The sizes here sit at the edges of that: every source and
destination phase, rows shorter than one word, rows at the limits between the
copy forms (16-byte gathers, one bulk copy per row, several stages per row),
source buffers and buckets that end in the middle of a 16-byte word.  Results
are bytes: every comparison is exact.
"""
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


def sync_and_check(desc):
    L = U.to_oracle(desc)
    plan = H.make_plan(*U.to_product(desc), desc["bucket_bytes"])
    shards = L.host_shards(desc["seed"], True)
    buf = H.alloc(plan)
    flat = np.zeros(buf.flat.numel(), np.uint8)
    for o, s in zip(H.source_offsets(plan), shards):
        flat[o:o + len(s)] = np.asarray(s, np.uint8)
    buf.flat.copy_(torch.from_numpy(flat))
    src = oracle.Source(shards=shards)
    want, want_cs = L.pack(src)
    want_t = [L.reshard_tensor(src, t) for t in range(len(L.tensors))]
    rng = plan.n_buckets // 3
    for call in ("full", "range"):
        if call == "full":
            H.pack(buf)
        else:   # the bucket-sorted table's own units
            for b in H.bucket_list(buf):
                b.fill_(0xAB)
            rr.rr_pack_range(plan, 0, rng, buf.shards, buf.buckets, buf.checksums)
            rr.rr_pack_range(plan, rng, plan.n_buckets - rng, buf.shards, buf.buckets,
                             buf.checksums)
        assert rr.rr_unpack_verify(plan, buf.buckets, buf.checksums, buf.dst) == (0, -1)
        np.testing.assert_array_equal(H.buckets_host(buf), want)
        np.testing.assert_array_equal(H.checksums_host(buf), want_cs)
        for t in range(plan.n_tensors):
            np.testing.assert_array_equal(H.tensor_host(buf, t), want_t[t])
        for d in buf.dst:
            d.fill_(0x5A5A)
    H.unpack(buf)
    torch.cuda.synchronize()
    for t in range(plan.n_tensors):
        np.testing.assert_array_equal(H.tensor_host(buf, t), want_t[t])
    rr.rr_plan_check(plan)


def layout(es, params, tensors, **kw):
    return dict(dict(params=[(f"p{i}", d, es) for i, d in enumerate(params)],
                     tensors=[(f"t{i}", r, b) for i, (r, b) in enumerate(tensors)],
                     tp=1 + max(r for r, _ in tensors), sharding="flat", n_shards=1,
                     bucket_bytes=1 << 20, align_bytes=es, tensor_align=256, seed=77,
                     specials=True), **kw)


@pytest.mark.parametrize("es", [4, 2])
@pytest.mark.parametrize("dst", ["bf16", "f16"])
def test_runs_at_every_phase(es, dst):
    """Contiguous runs: tensors back to back (every destination phase), each
    from its own source phase, of lengths around one vector, one stage of
    48 KiB and one 64 KiB item."""
    sizes = [1, 7, 8, 9, 15, 16, 17, 129, 12279, 12280, 12281, 24568, 24569, 32767, 32768, 70001]
    total = sum(sizes) + 16 * len(sizes)
    tensors, at = [], 0
    for i, n in enumerate(sizes):
        tensors.append((0, [(0, at + i % 9, n, 0, 1)]))
        at += n + 9
    sync_and_check(layout(es, [(total,)], tensors, tensor_align=2, n_shards=3,
                          bucket_bytes=(1 << 16) + 8, dst_dtype=dst))


@pytest.mark.parametrize("es", [4, 2])
@pytest.mark.parametrize("width", [1, 2, 3, 7, 8, 9, 15, 36, 101, 159, 161, 319, 321, 2757, 12283,
                                   12290, 24571, 24585])
def test_rows(es, width):
    """Column slices of odd widths for two ranks, and one that starts mid-row:
    around the limits between gathers, bulk copies per row and rows longer than
    a stage."""
    rows = max(3, min(400, 150000 // width))
    cols = 2 * width + 3
    tensors = [(r, [(0, 0, rows, r * width, width)]) for r in range(2)]
    tensors.append((1, [(0, 1, rows - 2, 2, width), (0, 0, rows, 0, cols)]))
    sync_and_check(layout(es, [(rows, cols)], tensors, n_shards=2, tensor_align=2,
                          bucket_bytes=(1 << 18) + 8))


@pytest.mark.parametrize("es", [4, 2])
@pytest.mark.parametrize("shape", [(1, 1), (3, 1), (13, 3), (7, 101), (5, 12289), (1, 50001)])
def test_buffers_that_end_mid_word(es, shape):
    """One buffer per parameter, of sizes that are not multiples of 16 bytes:
    the last word is read element by element."""
    rows, cols = shape
    tensors = [(0, [(0, 0, rows, cols // 2, cols - cols // 2)]), (0, [(0, 0, rows, 0, cols)]),
               (0, [(1, 1, rows, 0, cols)])]
    sync_and_check(layout(es, [shape, (rows + 1, cols)], tensors, sharding="tensors", n_shards=2,
                          tensor_align=2, bucket_bytes=(1 << 16) + 8))
