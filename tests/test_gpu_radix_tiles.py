"""The radix sort's scatter at the edges of its 7,168-pair tile (3,584 for a
small sort), of a warp's pairs and of a round's 32, on keys whose digits are random, all equal but
one, few, or all ones (the pad of a last tile), against a stable sort by the
host (exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

TILE = 7168
SMALL = 3584


@pytest.fixture(scope="module")
def ctx():
    c = vx.vx_open(256 << 20)
    yield c
    vx.vx_close(c)


def _keys(kind, n):
    r = np.random.default_rng(n)
    k = r.integers(0, 2**64, n, dtype=np.uint64)
    if kind == "few":
        k = k % np.uint64(3) << np.uint64(40)
    elif kind == "one_off":
        k[:] = 2**64 - 1
        k[n // 2] = 0
    elif kind == "ones":
        k[r.random(n) < 0.5] = 2**64 - 1
    return k


@pytest.mark.parametrize("kind", ["random", "few", "one_off", "ones"])
@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, TILE - 1, TILE, TILE + 1, 2 * TILE, 300 * TILE + 17, 1_000_000,
                               SMALL - 1, SMALL, SMALL + 1, 152 * SMALL, 152 * SMALL + 1])
def test_tile_edges(ctx, kind, n):
    k, v = _keys(kind, n), np.arange(n, dtype=np.uint32)
    ok, ov = vx.vx_radix_sort_pairs(ctx, k, v)
    perm = np.argsort(k, kind="stable")
    assert np.array_equal(ok, k[perm]) and np.array_equal(ov, v[perm])
