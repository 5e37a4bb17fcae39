"""Plans without group keys (one accumulator) through every kernel that adds to
it — fused, split and gather, bulk-copy, scalar, serving scan — over ragged row
ranges, with no, few and all rows surviving, against plain sums (exact,
wrapping)."""
import numpy as np
import pytest

import datagen as G

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

N = 400_003


@pytest.fixture(scope="module")
def tables():
    fact, dim = G.q1_fact(N, seed=3), G.date_dim()
    fact["price"][:7] = 2**31 - 1
    c = vx.vx_open(128 << 20)
    fid = {k: vx.vx_register_host_column(c, k, fact[k]) for k in fact}
    did = {k: vx.vx_register_host_column(c, "d." + k, dim[k]) for k in ("key", "year")}
    yield c, fact, dim, fid, did
    vx.vx_close(c)


@pytest.mark.parametrize("late", [vx.VX_LATE_FORCE_EARLY, vx.VX_LATE_FORCE_LATE])
@pytest.mark.parametrize("rows", [0, 2, 8, 16])
@pytest.mark.parametrize("agg", ["mul", "sub", "sum", "count"])
def test_one_group(tables, late, rows, agg):
    c, fact, dim, fid, did = tables
    year_of = np.zeros(len(dim["key"]), np.int64)
    year_of[dim["key"]] = dim["year"]
    cfg = vx.vx_get_config(c)
    cfg.kernel_rows, cfg.chunk_bytes = rows, 1 << 20
    vx.vx_set_config(c, cfg)
    for qty, (lo, hi) in ((0, (0, N)), (24, (0, N)), (50, (0, N)), (24, (1, 2)), (50, (1023, 1026)), (3, (5, N - 6))):
        t = {"dims": [{"dim": "date", "fk": "date_fk", "preds": [("year", 1993, 1996)]}],
             "fact_preds": [("quantity", vx.I32MIN, qty)], "group": [], "agg": (agg, "price", "discount")}
        if agg == "count":
            t["agg"] = (agg, None, None)
        plan = vx.make_plan(t, fid, {"date": did}, {"date": {"year": 1}}, late, lo, hi)
        st, gid, s, cnt, _ = vx.vx_run_plan(c, plan)
        y = year_of[fact["date_fk"][lo:hi]]
        k = (fact["quantity"][lo:hi] <= qty) & (y >= 1993) & (y <= 1996)
        a, b = (fact[x][lo:hi][k].astype(np.int64) for x in ("price", "discount"))
        want = {"mul": a * b, "sub": a - b, "sum": a, "count": 0 * a}[agg].sum()
        if k.sum():
            assert st == vx.VX_OK and gid.tolist() == [0] and cnt.tolist() == [k.sum()] and s.tolist() == [want]
        else:
            assert len(gid) == 0
