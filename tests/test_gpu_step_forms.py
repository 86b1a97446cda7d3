"""The batched step's forms against the one-walker-per-launch step, bit for
bit: both sides of the line between the pair kernel's latency and common
forms, stages of more walkers than a warp has lanes, merged every step and
every few steps, with and without theta statistics."""
import numpy as np
import pytest

from paper_2307_08006_gb300 import synth

pytestmark = pytest.mark.gpu


def water(seed):
    sp = synth.water_box(137, 5, seed=seed, box=1.7, r_cut=0.7)
    rng = np.random.default_rng(seed)
    return synth.with_changes(sp, x=((sp.x + rng.normal(0.0, 0.01, sp.x.shape)) % sp.box).astype(np.float32))


def run_both(spec, run, steps, **options):
    from paper_2307_08006_gb300 import labf

    state = synth.initial_state(spec, run, lam0=list(np.linspace(0.02, 0.98, run.n_walkers)))
    out = []
    for plain in (False, True):
        eng = labf.engine_for(spec, run, state, options=options)
        (eng.step_plain if plain else eng.step)(steps)
        o = eng.get_states()
        o.update(eng.read_abf(0, 0))
        if run.theta_stats:
            o.update(eng.read_theta(0, 0))
        out.append(o)
        eng.close()
    for k in ("x", "v", "lam", "plam", "step", "sum", "sumsq", "count"):
        assert np.array_equal(out[0][k], out[1][k]), k
    if run.theta_stats:
        for k in ("sum_d2", "sum_d", "sum_sd"):
            assert np.array_equal(out[0][k], out[1][k]), k


@pytest.mark.parametrize("walkers, margin", [(1, 0.0), (4, 0.05), (10, 0.05), (40, 0.05), (40, 0.0)])
def test_pair_forms(walkers, margin):
    """1 to 40 walkers of 416 atoms: well below the line (latency form), near
    it and above it (common form), with and without pruned tiles."""
    run = synth.water_run(seed=3, walkers_per_stage=1, n_bins=8)
    run.stages = [synth.Stage(0.0, 1.0, 8, walkers)]
    run_both(water(31), run, 23, prune_margin=margin)


@pytest.mark.parametrize("walkers", [17, 24])
def test_pair_forms_near_the_line(walkers):
    """2049 LJ atoms per walker: 15 items per SM (latency form) and 21 (common
    form)."""
    run = synth.lj_fluid_run(seed=9, n_walkers=walkers, n_bins=7)
    run_both(synth.lj_fluid(seed=12, cells=8), run, 11)


@pytest.mark.parametrize("walkers, shared_freq, theta", [(1, 1, True), (3, 2, True), (33, 1, True), (70, 3, False),
                                                         (64, 1, False)])
def test_stage_sizes(walkers, shared_freq, theta):
    run = synth.lj_fluid_run(seed=9, n_walkers=walkers, n_bins=7)
    run.shared_freq, run.theta_stats = shared_freq, theta
    run_both(synth.lj_fluid(seed=12), run, 11)


@pytest.mark.parametrize("walkers", [2, 100])  # the gate in the integrator's launch, and in one of its own
def test_kernel_timer_runs_the_step(walkers):
    """The kernel timer issues the launches of the graph's step: as many, with
    the same bits."""
    from paper_2307_08006_gb300 import labf

    spec, out, launches = water(23), [], []
    run = synth.water_run(seed=8, walkers_per_stage=1, n_bins=8)
    run.stages = [synth.Stage(0.0, 1.0, 8, walkers)]
    state = synth.initial_state(spec, run, lam0=list(np.linspace(0.1, 0.9, walkers)))
    for timed in (False, True):
        eng = labf.engine_for(spec, run, state)
        before = int(eng.stats()[2])
        if timed:
            eng.time_kernels(25)
        else:
            eng.step(25)
        launches.append(int(eng.stats()[2]) - before)
        out.append(eng.get_states())
        eng.close()
    assert launches[0] == launches[1]
    for k in ("x", "v", "lam", "plam"):
        assert np.array_equal(out[0][k], out[1][k]), k


@pytest.mark.parametrize("chunk, margin", [(32, 0.05), (64, 0.0), (96, 0.05)])
def test_latency_form_items(chunk, margin):
    """The latency form (variant 0, few items) against the common form
    (variant 1 takes it at any size), items of one to three 32-entry passes."""
    from paper_2307_08006_gb300 import labf

    spec, out = water(17), []
    run = synth.water_run(seed=8, walkers_per_stage=1, n_bins=8)
    run.stages = [synth.Stage(0.0, 1.0, 8, 3)]
    state = synth.initial_state(spec, run, lam0=[0.1, 0.5, 0.9])
    for variant in (0, 1):
        eng = labf.engine_for(spec, run, state, options=dict(prune_margin=margin, chunk_entries=chunk,
                                                             pair_variant=variant))
        eng.step(23)
        out.append(eng.get_states())
        eng.close()
    for k in ("x", "v", "lam", "plam"):
        assert np.array_equal(out[0][k], out[1][k]), k


@pytest.mark.parametrize("walkers, n_bins", [(32, 3), (33, 1), (65, 3), (100, 2)])
def test_fold_of_large_stages(walkers, n_bins):
    """One step of a stage that merges every step, its walkers' lambdas in no
    order, so that a bin's first walker sits in another lane in each group of
    32: the shared statistics are the walkers' samples added in walker order."""
    from paper_2307_08006_gb300 import labf

    spec, run = synth.lj_fluid(seed=12), synth.lj_fluid_run(seed=9, n_walkers=walkers, n_bins=n_bins)
    run.shared_freq = 1
    lam0 = np.random.default_rng(walkers).uniform(0.05, 0.95, walkers)
    eng = labf.engine_for(spec, run, synth.initial_state(spec, run, lam0=list(lam0)))
    eng.step(1)
    got, lam = eng.read_abf(0, 0), eng.get_states()["lam"]
    ref = np.zeros((3, n_bins))
    st = run.stages[0]
    for w in range(walkers):
        k = min(max(int(np.floor((lam[w] - st.lo) / ((st.hi - st.lo) / n_bins))), 0), n_bins - 1)
        s = eng.energy_forces(w)["dUdl"]
        ref[:, k] += (s, s * s, 1.0)
    eng.close()
    assert np.array_equal(got["sum"], ref[0]) and np.array_equal(got["sumsq"], ref[1])
    assert np.array_equal(got["count"], ref[2])
