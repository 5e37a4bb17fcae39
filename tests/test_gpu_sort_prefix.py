"""The partition sorts that leave the low key bytes to a repair, against a
stable sort by the host (exact): keys whose upper bytes nearly all differ, with
planted groups that share them (pairs, groups at the repair's limit of 16 and
beyond, equal keys inside a group, groups at the ends of the key range), and
inputs that the sample takes for such keys although a partition is full of
shared prefixes (sorted in full after the check)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

N = 8_000_003


def _sort(k, budget_mib=160):
    n = len(k)
    v = np.arange(n, dtype=np.uint32)
    c = vx.vx_open(budget_mib << 20)
    try:
        kc, rc = vx.vx_register_host_column(c, "k", k), vx.vx_register_host_column(c, "r", v)
        ok, orr = np.empty(n, np.uint64), np.empty(n, np.uint32)
        st = vx.vx_sort(c, kc, rc, ok, orr, vx.vx_sort_opts())
    finally:
        vx.vx_close(c)
    perm = np.argsort(k, kind="stable")
    assert np.array_equal(ok, k[perm]) and np.array_equal(orr, v[perm])
    assert st["bytes_h2d"] == 12 * n
    return st["radix_pass_pairs"] / n


def _uniform(seed=1):
    return np.random.default_rng(seed).integers(0, 2**64 - 1, N, dtype=np.uint64)


@pytest.mark.parametrize("bits", [64, 60, 56])
def test_distinct_prefixes(bits):
    passes = _sort(_uniform() >> np.uint64(64 - bits))
    assert passes < 6  # four or five of the eight bytes


@pytest.mark.parametrize("size", [2, 3, 15, 16])
@pytest.mark.parametrize("equal", [False, True])
def test_groups_are_repaired(size, equal):
    r = np.random.default_rng(size)
    k = _uniform(2)
    heads = np.concatenate([r.integers(0, 2**32, 300, dtype=np.uint64), [0, 2**32 - 1]]).astype(np.uint64)
    at = r.permutation(N)[: len(heads) * size].reshape(len(heads), size)
    low = r.integers(0, 3 if equal else 2**32, at.shape, dtype=np.uint64)
    k[at] = (heads[:, None] << np.uint64(32)) | low
    passes = _sort(k)
    assert size == 16 or passes < 6  # one of the other keys may make a group of 16 one too large


@pytest.mark.parametrize("size", [17, 40, 100_000])
def test_larger_groups_sort_in_full(size):
    r = np.random.default_rng(size)
    k = _uniform(3)
    at = r.permutation(N)[:size]
    k[at] = (np.uint64(0x80000001) << np.uint64(32)) | r.integers(0, 2**32, size, dtype=np.uint64)
    k[at[0]] = (np.uint64(0x80000001) << np.uint64(32)) | np.uint64(2**32 - 1)
    _sort(k)


def test_repeating_keys_sort_in_full():
    k = _uniform(4)
    k[: N // 2] = k[N // 2 : N // 2 * 2]
    assert _sort(k) == 8
