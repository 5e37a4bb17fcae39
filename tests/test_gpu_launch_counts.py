"""kernel_launches of resident partition sorts: what their jobs enqueue.  Two
inputs with the same chunks and partitions differ by their jobs alone: keys that
differ in their upper four bytes are sorted by four passes and a repair (9
kernels and the publishing one less than a full sort's 10), keys that repeat by
eight passes; partitions of one key value are not sorted."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

N, CHUNK_KERNELS, CHUNK = 5_000_000, 4, (1 << 20)
PREFIX_JOB, FULL_JOB = 2 + 4 + 2 + 1, 2 + 8 + 1  # histogram and bases, passes, search and repair, publish


def _launches(keys, n_partitions):
    """The call's statistics, and how many partitions have pairs of more than one key value to sort."""
    c = vx.vx_open(512 << 20)
    try:
        kid = vx.vx_register_host_column(c, "key", keys)
        rows = np.arange(len(keys), dtype=np.uint32)
        rid = vx.vx_register_host_column(c, "row", rows)
        spl = np.zeros(2 * 128, np.uint64)
        o = vx.vx_sort_opts()
        o.n_partitions, o.splitters_out = n_partitions, spl.ctypes.data
        ok, orow = np.empty_like(keys), np.empty_like(rows)
        s = vx.vx_sort(c, kid, rid, ok, orow, o)
    finally:
        vx.vx_close(c)
    perm = np.argsort(keys, kind="stable")
    assert np.array_equal(ok, keys[perm]) and np.array_equal(orow, rows[perm])
    assert s["bytes_h2d"] == 12 * len(keys)  # the pairs stayed in the arena
    held = len(np.unique(np.searchsorted(spl[:s["n_partitions"] - 1], keys, side="right")))
    return s, held - s["passthrough_partitions"]


@pytest.mark.parametrize("P", [4, 11])
def test_resident_partition_sort(P):
    r = np.random.default_rng(P)
    chunks = -(-N // CHUNK) * CHUNK_KERNELS
    s, jobs = _launches(r.integers(0, 2**64 - 1, N, dtype=np.uint64), P)
    assert jobs == P and s["kernel_launches"] == chunks + jobs * PREFIX_JOB
    s, jobs = _launches(r.choice(r.integers(0, 2**64 - 1, N // 20, dtype=np.uint64), N), P)
    assert jobs == P and s["kernel_launches"] == chunks + jobs * FULL_JOB
    heavy = r.integers(0, 2**64 - 1, N, dtype=np.uint64)
    heavy[r.random(N) < 0.5] = 2**63
    s, jobs = _launches(heavy, P)
    assert s["passthrough_partitions"] == 1 and s["kernel_launches"] == chunks + jobs * FULL_JOB
