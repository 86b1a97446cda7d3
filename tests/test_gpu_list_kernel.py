"""Pair lists of the list kernel at its edges, bit for bit against the oracle:
partly filled super-clusters, boxes of twice the list radius (every image,
two rounds of candidate columns, several passes of candidates), exclusion
groups and extra excluded partners across super-clusters, alchemical atoms."""
import numpy as np
import pytest

from paper_2307_08006_gb300 import synth

pytestmark = pytest.mark.gpu


def random_spec(n, r_cut, box, seed, n_alch):
    """n force-free atoms at random positions; runs of 1-5 atoms share an
    exclusion group (or none), random pairs are extra partners."""
    rng = np.random.default_rng(seed)
    group = np.repeat(np.arange(n), rng.integers(1, 6, n))[:n].astype(np.int32)
    group[rng.random(n) < 0.2] = -1
    extra = np.full((n, 4), -1, np.int32)
    for _ in range(n // 3):
        i, j = (int(v) for v in rng.integers(0, n, 2))
        a, b = (int((extra[k] >= 0).sum()) for k in (i, j))
        if i != j and a < 4 and b < 4:
            extra[i, a], extra[j, b] = j, i
    alch = np.zeros(n, np.uint8)
    alch[rng.choice(n, n_alch, replace=False)] = 1
    x = (rng.random((n, 3)) * box).astype(np.float32)
    return synth.SystemSpec(name="random", box=box, mass=np.ones(n), charge=np.zeros(n), sigma=np.zeros(n),
                            epsilon=np.zeros(n), alch=alch, excl_group=group, excl_extra=extra, x=x, r_cut=r_cut,
                            eps_rf=0.0, coul=0.0)


@pytest.mark.parametrize("n, r_cut, box, n_alch", [
    (1, 0.5, 2.0, 0),
    (63, 0.9, 2.0, 2),
    (64, 0.9, 2.0, 0),
    (65, 0.9, 2.0, 3),
    (257, 0.4, 2.0, 5),
    (1000, 0.9, 2.0, 8),
    (3001, 0.55, 2.0, 16),
    (6000, 0.9, 2.0, 3),   # 32 < candidate columns, > 512 candidates per super-cluster
    (6000, 0.15, 2.0, 3),
    (2500, 30.0, 100.0, 4),  # large box: list radius of few quantized units per nm
])
def test_pair_lists_match_oracle(n, r_cut, box, n_alch):
    import oracle
    from paper_2307_08006_gb300 import labf

    spec = random_spec(n, r_cut, box, 100 + n, n_alch)
    run = synth.harmonic_run(seed=5, n_walkers=2, n_bins=4)
    run.skin = 0.09 * box / 2.0
    eng = labf.engine_for(spec, run, options=dict(list_capacity_factor=4.0))
    osys = oracle.OracleSystem(spec)
    ref, kind = oracle.pair_set(osys, spec.x, spec.r_cut + run.skin)
    for w in range(2):
        got, gkind = eng.get_pairs(w)
        assert np.array_equal(got, ref) and np.array_equal(gkind, kind)
    eng.close()


def test_exclusion_group_ids_of_any_size():
    """Groups are told apart by their whole 32-bit id: ids that differ only
    above bit 29, and the largest ones, exclude their own atoms and no others."""
    import oracle
    from paper_2307_08006_gb300 import labf

    spec = random_spec(1000, 0.9, 2.0, 77, 6)
    ids = np.arange(spec.n, dtype=np.int64)
    ids[:40] = (0x3ffffffe, 0x3fffffff, 0x40000000, 0x7ffffffe, 0x7fffffff, *(0x40000000 + 300 + np.arange(35)))
    g = np.asarray(spec.excl_group)
    # (low ids that the large ones must not be taken for stay in use)
    order = np.unique(g[g >= 0])
    new = dict(zip(order, [*ids[:40], *range(300, 300 + len(order) - 40)]))
    spec.excl_group = np.array([new.get(k, -1) for k in g], np.int64).astype(np.int32)
    run = synth.harmonic_run(seed=5, n_walkers=1, n_bins=4)
    run.skin = 0.09
    eng = labf.engine_for(spec, run, options=dict(list_capacity_factor=4.0))
    ref, kind = oracle.pair_set(oracle.OracleSystem(spec), spec.x, spec.r_cut + run.skin)
    got, gkind = eng.get_pairs(0)
    assert np.array_equal(got, ref) and np.array_equal(gkind, kind)
    eng.close()
