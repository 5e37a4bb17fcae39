"""The radix join's two layouts and its block-level join at their edges, against
the oracle (exact): tables that stay in device memory and tables whose
clustered chunks go through host memory; a run of groups with more build tuples
than a shared-memory table takes, with and without a key that repeats across
the table's pieces; a probe key hot enough to be split over work items; the
all-ones key; one-tuple tables; both schedules."""
import numpy as np
import pytest

import datagen as G
import oracle as O

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

ONES = np.array([-1], np.int64)


def _run(bk, bp, pk, budget_mib, bits=24, sched=0):
    c = vx.vx_open(budget_mib << 20)
    try:
        cfg = vx.vx_get_config(c)
        cfg.sched = sched
        vx.vx_set_config(c, cfg)
        ids = [vx.vx_register_host_column(c, n, a) for n, a in (("bk", bk), ("bp", bp), ("pk", pk))]
        o = vx.vx_join_opts()
        o.algorithm, o.radix_bits = vx.VX_JOIN_RADIX, bits
        return vx.vx_join(c, *ids, o)
    finally:
        vx.vx_close(c)


def _check(bk, bp, pk, *a, **kw):
    r = _run(bk, bp, pk, *a, **kw)
    assert (r["count"], r["payload_sum"], r["pair_fp"]) == O.join(bk, bp, pk, nthreads=8)
    return r


@pytest.mark.parametrize("bits", [8, 16, 24])
@pytest.mark.parametrize("nb,npr", [(1, 1), (1, 5000), (767, 4097), (1 << 18, (1 << 18) + 1), (800_001, 2_000_003)])
@pytest.mark.parametrize("sched", [0, 1])
def test_resident_sizes(nb, npr, bits, sched):
    bk, bp = G.build_side(nb)
    r = _check(bk, bp, G.probe_side(npr, nb, 0.5, 0.0, seed=nb), 512, bits, sched)
    assert r["bytes_d2h"] == 0


@pytest.mark.parametrize("bits,z", [(24, 0.0), (24, 1.0), (16, 1.0)])
def test_tables_beyond_the_budget(bits, z):
    nb, npr = 3_000_001, 21_000_003
    bk, bp = G.build_side(nb)
    r = _check(bk, bp, G.probe_side(npr, nb, 0.5, z), 256, bits)
    assert r["bytes_d2h"] > 12 * npr and r["ranges"] > 1


@pytest.mark.parametrize("budget", [512, 205])
def test_pieces_hot_key_and_ones(budget):
    base, _ = G.build_side(300_000)
    crowd = ((np.arange(5000, dtype=np.int64) + 1) << 24) | 5  # one group, five pieces of the table
    bk = np.unique(np.concatenate([base, crowd, ONES]))
    np.random.default_rng(1).shuffle(bk)
    bp = (bk * 5 + 3).astype(np.int64)
    pk = np.concatenate([np.full(200_000, crowd[4321]), bk[::3], np.full(70_000, bk[0]), ONES, ONES, crowd[::2],
                         crowd + 1, G.probe_side(20_000_000 if budget < 512 else 50_000, 300_000, 0.5, 1.0)])
    r = _check(bk, bp, pk, budget)
    assert (r["bytes_d2h"] > 0) == (budget < 512)
    for twin in (crowd[0], -1):  # the key's copies sit at the two ends of the build table
        k2 = np.concatenate([[twin], bk[bk != twin], [twin]]).astype(np.int64)
        with pytest.raises(vx.VxError) as e:
            _run(k2, k2, pk, budget)
        assert e.value.status == vx.VX_E_DUPKEY


@pytest.mark.parametrize("bits", [8, 16, 24])
@pytest.mark.parametrize("nb", [700, 768 * 200, 768 * 400])
def test_resident_clustering_by_upper_bytes(nb, bits):
    """Builds whose runs of groups need one to three clustered bytes; keys
    that share a byte (a pass left out) and keys that share all of them."""
    npr = 1_500_007
    base = np.random.default_rng(nb).permutation(nb).astype(np.int64)
    for shift in (0, 8, 16):
        bk = base << shift | 3 << 50
        bp = (base * 7 + 1).astype(np.int64)
        pk = np.random.default_rng(2).choice(bk, npr)
        pk[::5] += 1 << 55
        r = _check(bk, bp, pk, 4096, bits)
        assert r["bytes_d2h"] == 0
