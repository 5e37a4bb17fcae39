"""The partition plan with partitions kept in the arena, against a stable sort
by the host (exact): budgets on both sides of what the pairs need, the three
partitioners, keys with heavy values (partitions of one key value pass through
unsorted), keys that repeat everywhere, and an input whose sampled rows say
nothing about the others, so that a region is too small and the call sorts
through host memory after all."""
import numpy as np
import pytest

import datagen as G

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

M64 = (1 << 64) - 1
PARTS = [vx.VX_PART_SAMPLE, vx.VX_PART_LEARNED_PL, vx.VX_PART_LEARNED_MLP]


def _sort(k, budget_mib, part=vx.VX_PART_SAMPLE, sample=0, n_part=0, sched=0):
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
        o.partitioner, o.sample_size, o.n_partitions, o.seed = part, sample, n_part, 3
        st = vx.vx_sort(c, kc, rc, ok, orr, o)
    finally:
        vx.vx_close(c)
    perm = np.argsort(k, kind="stable")
    assert np.array_equal(ok, k[perm]) and np.array_equal(orr, v[perm])
    return st


@pytest.mark.parametrize("part", PARTS)
@pytest.mark.parametrize("dist", ["uniform", "zipf", "runs"])
@pytest.mark.parametrize("n,budget", [(3_000_017, 64), (5_000_011, 96), (8_000_009, 200)])
def test_resident(part, dist, n, budget):
    st = _sort(G.sort_input(n, dist, seed=n)[0], budget, part)
    assert st["bytes_h2d"] == 12 * n == st["bytes_d2h"] and st["n_partitions"] >= 4


@pytest.mark.parametrize("sched", [0, 1])
def test_given_partition_count_and_schedules(sched):
    n = 4_000_003
    st = _sort(G.sort_input(n, "uniform", seed=1)[0], 96, n_part=23, sched=sched)
    assert st["n_partitions"] == 23 and st["bytes_h2d"] == 12 * n
    st = _sort(G.sort_input(n, "zipf", seed=1)[0], 96, n_part=40, sched=sched)  # the top key holds a tenth of the rows
    assert st["passthrough_partitions"] >= 1 and st["bytes_h2d"] == 12 * n


def test_beyond_the_budget_goes_through_host_memory():
    n = 6_000_005
    st = _sort(G.sort_input(n, "uniform", seed=2)[0], 64)
    assert st["bytes_h2d"] == 24 * n


@pytest.mark.parametrize("kind", ["constant", "two", "top"])
def test_repeating_keys(kind):
    n = 3_000_001
    r = np.random.default_rng(0)
    k = {"constant": np.full(n, 7, np.uint64), "two": r.integers(0, 2, n).astype(np.uint64) * np.uint64(M64),
         "top": np.where(r.random(n) < 0.7, np.uint64(M64), r.integers(0, 2**63, n).astype(np.uint64))}[kind]
    _sort(k, 64)


def _mix64(z):
    z &= M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def test_sample_that_misleads():
    n, m = 3_000_017, 2_000
    rows = [_mix64(3 * 0x9E3779B97F4A7C15 + i) % n for i in range(m)]  # the rows the library samples
    r = np.random.default_rng(5)
    k = r.integers(2**63, M64, n, dtype=np.uint64)
    k[rows] = r.integers(0, 2**63, m).astype(np.uint64)
    st = _sort(k, 80, sample=m)
    assert st["bytes_h2d"] > 12 * n
