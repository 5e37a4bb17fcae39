"""The merge plan with the pairs kept in the arena, against a stable sort by the
host (exact): the input's own runs (ties, run starts on and beside the loading
chunks' starts, one run, just as many as the merge takes and one more), chunks
sorted where they are (also with an odd number of radix passes, which leaves the
result in the other buffer), given partition counts, both schedules, and a
budget just too small."""
import numpy as np
import pytest

import datagen as G

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")


def _sort(k, budget_mib=200, sched=0, **opts):
    n = len(k)
    v = np.arange(n, dtype=np.uint32)
    c = vx.vx_open(budget_mib << 20)
    try:
        cfg = vx.vx_get_config(c)
        cfg.sched = sched
        vx.vx_set_config(c, cfg)
        kc, rc = vx.vx_register_host_column(c, "k", k), vx.vx_register_host_column(c, "r", v)
        ok, orr = np.empty(n, np.uint64), np.empty(n, np.uint32)
        o = vx.vx_sort_opts()
        o.plan = vx.VX_SORT_MERGE
        for name, x in opts.items():
            setattr(o, name, x)
        st = vx.vx_sort(c, kc, rc, ok, orr, o)
    finally:
        vx.vx_close(c)
    perm = np.argsort(k, kind="stable")
    assert np.array_equal(ok, k[perm]) and np.array_equal(orr, v[perm])
    assert st["max_partition"] - st["min_partition"] <= 1
    return st


def _runs(n, starts, hi=2**64 - 1, seed=0):
    k = np.random.default_rng(seed).integers(0, hi, n, dtype=np.uint64)
    for a, b in zip(starts, list(starts[1:]) + [n]):
        k[a:b].sort()
    return k


@pytest.mark.parametrize("hi", [5, 2**64 - 1])
@pytest.mark.parametrize("n,starts", [(1, [0]), (4097, [0, 4096]), (1 << 20, [0, 1, 2]), (2_500_001, [0]),
                                      (2_500_001, [0, (1 << 20) - 1, 1 << 20, (1 << 20) + 1, 2 << 20, 2_500_000])])
def test_own_runs(n, starts, hi):
    k = _runs(n, starts, hi, seed=n)
    st = _sort(k)
    assert st["natural_runs"] == 1 and st["n_runs"] == 1 + int(np.count_nonzero(k[1:] < k[:-1]))
    assert st["bytes_h2d"] == 12 * n == st["bytes_d2h"]


@pytest.mark.parametrize("n_runs", [2, 3, 255, 256, 257])
@pytest.mark.parametrize("sched", [0, 1])
def test_run_counts(n_runs, sched):
    n = 5_000_003
    k = _runs(n, [n * r // n_runs for r in range(n_runs)], seed=n_runs)
    st = _sort(k, sched=sched)
    assert st["natural_runs"] == (n_runs <= 256) and st["bytes_h2d"] == 12 * n


@pytest.mark.parametrize("dist", ["uniform", "zipf"])
@pytest.mark.parametrize("n,budget", [(300_001, 64), (4_000_037, 128), (9_000_001, 400)])
@pytest.mark.parametrize("mask", [2**64 - 1, 0xFFFFFF])  # eight radix passes, or three
def test_sorted_chunks(dist, n, budget, mask):
    k = G.sort_input(n, dist, seed=n)[0] & np.uint64(mask)
    st = _sort(k, budget)
    assert st["natural_runs"] == 0 and st["bytes_h2d"] == 12 * n


def test_runs_mode_and_partitions():
    n = 3_000_017
    k = _runs(n, [n * r // 64 for r in range(64)])
    assert _sort(k, runs_mode=1, n_partitions=37)["n_partitions"] == 37
    assert _sort(k, n_partitions=100)["n_partitions"] == 100


def test_budget_too_small_goes_through_host_memory():
    n = 3_000_017
    assert _sort(G.sort_input(n, "runs", seed=5)[0], 40)["bytes_h2d"] > 12 * n


@pytest.mark.parametrize("n_runs", [2, 5, 8, 9, 33, 63, 64, 65])
@pytest.mark.parametrize("kind", ["random", "equal", "disjoint", "backward", "few", "lopsided"])
def test_tiles(n_runs, kind):
    """Up to 64 runs merge by tiles of at most 4,096 pairs between sorted samples."""
    n = 1_200_007
    r = np.random.default_rng(n_runs)
    cuts = [n * i // n_runs for i in range(n_runs)]
    if kind == "lopsided":
        cuts = sorted({0, *(int(x) for x in (r.random(n_runs - 1) ** 4 * n))})
    k = r.integers(0, 2**64 - 1, n, dtype=np.uint64)
    if kind == "equal":
        k[:] = 11
    elif kind == "few":
        k %= np.uint64(7)
    elif kind in ("disjoint", "backward"):
        for i, (a, b) in enumerate(zip(cuts, cuts[1:] + [n])):
            k[a:b] = k[a:b] % np.uint64(1000) + np.uint64(1000 * (i if kind == "disjoint" else n_runs - i))
    for a, b in zip(cuts, cuts[1:] + [n]):
        k[a:b].sort()
    st = _sort(k, n_partitions=7)
    assert st["natural_runs"] == 1 and st["n_partitions"] == 7
