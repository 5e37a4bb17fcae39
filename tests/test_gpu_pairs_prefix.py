"""vx_radix_sort_pairs where a sample of the keys decides whether the low key
bytes are left to a repair, against a stable sort by the host (exact): around
the size from which it samples, keys that repeat, all-ones keys, prefixes shared
by groups up to the repair's limit of 16, and larger groups and many groups that
lie between the sampled rows (sorted in full after the check)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")


@pytest.fixture(scope="module")
def ctx():
    c = vx.vx_open(256 << 20)
    yield c
    vx.vx_close(c)


def _hide(k, per, prefix_bits, r):
    """Every 100 rows, the rows between sampled ones: groups of `per` share their upper bits."""
    n = len(k)
    at = np.arange(n)
    at = at[(at % 100 >= 10) & (at % 100 < 90)]
    at = at[: len(at) // per * per].reshape(-1, per)
    k[at] = (k[at[:, :1]] >> np.uint64(64 - prefix_bits) << np.uint64(64 - prefix_bits)) | (
        k[at] & np.uint64((1 << (64 - prefix_bits)) - 1))


def _keys(kind, n):
    r = np.random.default_rng(n)
    k = r.integers(0, 2**64 - 1, n, dtype=np.uint64)
    if kind == "ones":
        k[r.random(n) < 0.5] = 2**64 - 1
    elif kind == "one_pair":
        k[:2] = 2**64 - 1
        k[n // 2:n // 2 + 2] = 0
    elif kind == "twice":
        k = r.choice(k[: n // 2 + 1], n)
    elif kind == "low32":
        k &= np.uint64(2**32 - 1)
    elif kind.startswith("hide"):
        _hide(k, int(kind[4:]), 40, r)
    elif kind.startswith("group"):  # 40 groups of neighbours, descending
        size = int(kind[5:])
        for j in range(40):
            at = 1 + j * (n // 41)
            k[at:at + size] = (k[at] >> np.uint64(8) << np.uint64(8)) | np.arange(size, dtype=np.uint64)[::-1]
    return k


@pytest.mark.parametrize("kind", ["random", "ones", "one_pair", "twice", "low32", "group2", "group16", "group17",
                                  "group200", "hide2", "hide16", "hide80"])
@pytest.mark.parametrize("n", [32_767, 32_768, 32_769, 100_003, 1_000_000, 3_000_017])
def test_against_a_stable_sort(ctx, kind, n):
    k, v = _keys(kind, n), np.arange(n, dtype=np.uint32)[::-1].copy()
    ok, ov = vx.vx_radix_sort_pairs(ctx, k, v)
    perm = np.argsort(k, kind="stable")
    assert np.array_equal(ok, k[perm]) and np.array_equal(ov, v[perm])
