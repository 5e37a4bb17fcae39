"""The radix join through host memory where the build keys crowd into a part of
the groups (dense small keys, a dense part beside a random one, one group with
most of the keys), so that runs of groups are cut shorter: against the oracle
(exact), with a key that repeats at the two ends of the table, and the time that
cutting them saves."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

NP = 21_000_003  # with 256 MiB, more than the arena holds


def _keys(kind, nb):
    r = np.random.default_rng(nb)
    k = r.permutation(nb).astype(np.int64)
    if kind == "half":
        k[::2] = (r.choice(1 << 30, len(k[::2]), replace=False).astype(np.int64) + 1) << 20
    elif kind == "crowd":
        k[: nb - nb // 8] <<= 24
        k[nb - nb // 8:] += 1 << 40
    return k


def _join(bk, bp, pk, bits):
    c = vx.vx_open(256 << 20)
    try:
        ids = [vx.vx_register_host_column(c, n, a) for n, a in (("bk", bk), ("bp", bp), ("pk", pk))]
        o = vx.vx_join_opts()
        o.algorithm, o.radix_bits = vx.VX_JOIN_RADIX, bits
        return vx.vx_join(c, *ids, o)
    finally:
        vx.vx_close(c)


def _probes(kind, bk):
    pk = np.random.default_rng(1).choice(bk, NP)
    if kind == "crowd":  # a group's tuples have to fit a staging slot: most probes go to the other keys
        pk[NP // 16:] = np.random.default_rng(2).choice(bk[len(bk) - len(bk) // 8:], NP - NP // 16)
    pk[::3] += 1 << 50
    return pk


@pytest.mark.parametrize("kind,nb,bits", [("dense", 769, 24), ("dense", 2049, 24), ("dense", 200_001, 24),
                                          ("dense", 200_001, 16), ("half", 100_000, 24), ("crowd", 6000, 24)])
def test_against_the_oracle(kind, nb, bits):
    bk = _keys(kind, nb)
    bp = (bk * 3 + 1).astype(np.int64)
    pk = _probes(kind, bk)
    r = _join(bk, bp, pk, bits)
    assert r["bytes_d2h"] > 12 * NP
    assert (r["count"], r["payload_sum"], r["pair_fp"]) == O.join(bk, bp, pk, nthreads=8)
    twin = np.concatenate([bk, bk[:1]])
    with pytest.raises(vx.VxError) as e:
        _join(twin, twin, pk, bits)
    assert e.value.status == vx.VX_E_DUPKEY


def test_one_key_for_all_probes_is_refused():
    bk = _keys("dense", 1)
    with pytest.raises(vx.VxError) as e:
        _join(bk, bk, _probes("dense", bk), 24)
    assert e.value.status == vx.VX_E_NOMEM  # one group beyond a staging slot


def test_dense_keys_are_probed_about_once():
    """200,001 dense keys filled few runs of 32,768 tuples, so that every probe
    was read for each of 32 tables: a join kernel of 18 ms, where random keys
    took 4."""
    nb = 200_001
    ms = {}
    for kind in ("dense", "random"):
        bk = _keys("dense", nb) if kind == "dense" else np.unique(np.random.default_rng(2).integers(0, 1 << 60, nb))
        pk = np.random.default_rng(1).choice(bk, NP)
        ms[kind] = min(_join(bk, bk, pk, 24)["ms_probe_kernel"] for _ in range(2))
    assert ms["dense"] < 2.5 * ms["random"] + 1.0
