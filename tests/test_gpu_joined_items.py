"""One-row items that share a stage of the bulk-copy engine, against the oracle.

A relay puts row-parallel weights together from its ranks' pieces, row by row,
so its work table is long runs of short one-row items.  The sizes here put the
runs' ends on and around the edges: the 32-item window, one stage of 48 KiB, a
bucket's end, a change of element type, pieces that do not qualify (odd
widths) in between, and runs of one item.
"""
import pytest
import torch

from tests.test_gpu_ragged import layout, sync_and_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


def side_by_side(widths, rows):
    """Blocks that lay the rows of several parameters next to one another."""
    return [(p, r, 1, 0, w) for r in range(rows) for p, w in enumerate(widths)]


@pytest.mark.parametrize("es", [4, 2])
@pytest.mark.parametrize("widths", [(8, 8), (16, 24), (64,) * 8, (512, 1024), (1000, 1536, 8),
                                    (6144, 6144), (6152, 8), (40, 3, 40), (8, 12288, 8)])
def test_rows_side_by_side(es, widths):
    rows = max(2, min(97, 100000 // sum(widths)))
    params = [(rows, w) for w in widths]
    tensors = [(0, side_by_side(widths, rows)),
               (0, side_by_side(widths, rows)[1:-1] + [(0, 0, rows, 0, widths[0])])]
    for bucket in (1 << 16, (1 << 20) + 8):
        sync_and_check(layout(es, params, tensors, sharding="tensors", n_shards=len(widths),
                              bucket_bytes=bucket, dst_dtype="f16" if bucket == 1 << 16 else "bf16"))


def test_runs_break_where_the_type_changes():
    """fp32 and bf16 pieces side by side: no stage holds both."""
    desc = layout(4, [(50, 64), (50, 64), (50, 64)],
                  [(0, side_by_side((64, 64, 64), 50))], sharding="tensors", n_shards=3,
                  bucket_bytes=1 << 14)
    desc["params"][1] = ("p1", (50, 64), 2)
    sync_and_check(desc)
