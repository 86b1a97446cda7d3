"""The pair launches follow the lists of the state that runs, not those of the
state that an engine was created on: time and bits of a step after
`set_states`, against an engine created on that state."""
import numpy as np
import pytest

from paper_2307_08006_gb300 import synth

pytestmark = pytest.mark.gpu


def lattice(spacing, n, box, rng):
    """n points of a centred cubic lattice, jittered by up to 0.03."""
    edge = int(np.ceil(n ** (1.0 / 3.0)))
    p = np.stack(np.meshgrid(*[np.arange(edge)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    p = (p - 0.5 * (edge - 1)) * spacing + 0.5 * box + rng.uniform(-0.03, 0.03, (n, 3))
    return (p % box).astype(np.float32)


@pytest.mark.parametrize("condense", [True, False])
@pytest.mark.parametrize("plain", [False, True])
def test_state_of_another_density(condense, plain):
    """64 walkers of an LJ gas without a pair in reach, set to droplets of 30
    and more items per SM, and the other way round.  A launch sized by the gas's
    items took 200 times as long (one block); 1.25 leaves room for the timing."""
    import torch

    from paper_2307_08006_gb300 import labf

    rng = np.random.default_rng(5)
    base = synth.lj_fluid(seed=4, cells=7)
    box = 38.4
    gas, drop = (synth.with_changes(base, box=box, x=lattice(s, base.n, box, rng)) for s in (3.2, 1.12))
    first, second = (gas, drop) if condense else (drop, gas)
    walkers = 4 if plain else 64
    run = synth.lj_fluid_run(seed=9, n_walkers=walkers, n_bins=8)
    lam0 = list(np.linspace(0.1, 0.9, walkers))
    engines = []
    for spec in (first, second):
        eng = labf.engine_for(spec, run, synth.initial_state(spec, run, lam0=lam0),
                              options=dict(list_capacity_factor=8.0))
        engines.append(eng)
    s = synth.initial_state(second, run, lam0=lam0)
    for eng in engines:
        eng.set_states(x=s.x.reshape(-1, 3), v=s.v.reshape(-1, 3), lam=s.lam, plam=s.plam)
    best = [np.inf, np.inf]
    for _ in range(4):
        for k, eng in enumerate(engines):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            (eng.step_plain if plain else eng.step)(6 if plain else 60)
            b.record()
            torch.cuda.synchronize()
            best[k] = min(best[k], a.elapsed_time(b))
    out = [eng.get_states() for eng in engines]
    for k in ("x", "v", "lam", "plam"):
        assert np.array_equal(out[0][k], out[1][k]), k
    assert best[0] <= 1.25 * best[1], best
    for eng in engines:
        eng.close()


def test_tuning_in_the_latency_form():
    """The grid of the latency form is fixed: a tuning on few items that ends
    with the form's variant keeps the default grid for the common form, instead
    of one that noise picked."""
    from paper_2307_08006_gb300 import labf

    eng = labf.engine_for(synth.lj_fluid(seed=4), synth.lj_fluid_run(seed=9, n_walkers=2, n_bins=8))
    reports = [eng.autotune() for _ in range(6)]
    eng.close()
    assert any("pair_variant=0" in r for r in reports)
    assert all("pair_ctas_per_sm=4" in r for r in reports if "pair_variant=0" in r), reports


def test_close_waits_for_the_steps():
    """The steps write host memory that the engine owns: it is not given back
    before they are through."""
    import torch

    from paper_2307_08006_gb300 import labf

    eng = labf.engine_for(synth.lj_fluid(seed=4, cells=7), synth.lj_fluid_run(seed=9, n_walkers=16, n_bins=8))
    arena = eng.arena
    eng.step(2000)
    done = torch.cuda.Event()
    done.record()
    eng.step(1)
    eng.close()
    assert done.query()
    del arena
