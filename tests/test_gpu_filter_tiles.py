"""The single-pass device filter at the edges of its tiles and of its dispatch:
tile and look-back boundaries (4,096 rows, 32 tiles), the switch to large tiles
(2^24 rows), columns off a 16-byte boundary, every operator with empty and full
ranges, and a capacity below the count.  Row ids are compared with a plain mask
of the same predicates (exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")
torch = pytest.importorskip("torch")

I32MIN, I32MAX = -2**31, 2**31 - 1
OPS = {vx.VX_BETWEEN: lambda v, a, b: (v >= a) & (v <= b), vx.VX_EQ: lambda v, a, b: v == a,
       vx.VX_NE: lambda v, a, b: v != a, vx.VX_LT: lambda v, a, b: v < a, vx.VX_LE: lambda v, a, b: v <= a,
       vx.VX_GT: lambda v, a, b: v > a, vx.VX_GE: lambda v, a, b: v >= a}


def _check(cols, preds, row0=0, cap=None):
    n = len(cols[0])
    keep = np.ones(n, bool)
    for c, op, lo, hi in preds:
        keep &= OPS[op](cols[c].cpu().numpy(), lo, hi)
    want = np.nonzero(keep)[0] + row0
    cap = n if cap is None else cap
    out = torch.full((n + 8,), -1, dtype=torch.int64, device="cuda")
    st, cnt = vx.vx_filter_device_static([c.data_ptr() for c in cols], preds, n, row0, out.data_ptr(), cap)
    assert cnt == len(want) and st == (vx.VX_OK if cnt <= cap else vx.VX_E_CAPACITY)
    got = out.cpu().numpy()
    k = min(cnt, cap)
    assert np.array_equal(got[:k], want[:k]) and (got[k:] == -1).all()


def _cols(n, k, lo=-1000, hi=1000, shift=0, seed=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return [torch.randint(lo, hi, (n + shift,), dtype=torch.int32, device="cuda", generator=g)[shift:] for _ in range(k)]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [1, 3, 4095, 4096, 4097, 32 * 4096, 32 * 4096 + 1, 33 * 4096 + 5, 1 << 24, (1 << 24) + 1,
                               (1 << 26) - 3, 1 << 26])
def test_tile_edges(n, shift):
    _check(_cols(n, 2, shift=shift, seed=n), [(0, vx.VX_LT, 300, 0), (1, vx.VX_BETWEEN, -500, 900)], row0=1 << 40)


@pytest.mark.parametrize("op", list(OPS))
def test_operators_at_the_ends_of_the_range(op):
    v = torch.tensor([I32MIN, I32MIN + 1, -1, 0, 1, I32MAX - 1, I32MAX] * 1000, dtype=torch.int32, device="cuda")
    for a in (I32MIN, -1, 0, I32MAX):
        for b in (I32MIN, 0, I32MAX):
            _check([v], [(0, op, a, b)])


@pytest.mark.parametrize("n,thr", [(200_003, -1001), (200_003, 1001), (5_000_001, 1001), (20_000_001, 990)])
def test_none_all_and_capacity(n, thr):
    cols = _cols(n, 3, seed=7)
    preds = [(0, vx.VX_LT, thr, 0), (2, vx.VX_NE, 5, 0), (1, vx.VX_GE, -990, 0)]
    _check(cols, preds)
    _check(cols, preds, cap=n // 3)
    _check(cols, preds, cap=0)
