"""The time loop of small grids in one launch with the fields resident on the
SMs: blocks of at most 16 x 16 x 12 cells exchange halos step by step.  Its
arithmetic is that of the passes, rounding by rounding, so seismograms and
wavefields must equal those of the passes (which runs with per-launch
profiling take) bit for bit -- at block edges and remainders on every axis,
with one block and with the most, for every boundary and source kind, with a
free surface, with a coarse medium grid, over several launches, in chunks,
and with more receivers than one launch stages."""
import numpy as np
import pytest

from paper_2112_15071_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ews():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_15071_gb300 import ews as E
    E.load()
    yield E


def both(ews, p):
    """(seismograms, state) of a run in one launch and of the passes."""
    sim = ews.simulation_for(p)
    got, state = sim.run(p.nt, p.dt), sim.get_state()
    sim.set_tile_shape("32x8")
    sim.set_profiling(True)
    want = sim.run(p.nt, p.dt)
    return (got, state), (want, sim.get_state())


def same(a, b):
    assert np.abs(b[0]).max() > 0
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


# one block; 16 + 1 and 2 x 16 + 1 cells; 4, 5, 8 and 9..12 planes a block
# (the thread shapes); many small blocks; the largest grids that fit
SIZES = [(12, 11, 10), (17, 16, 9), (33, 18, 5), (16, 47, 33), (64, 60, 61), (31, 14, 150),
         (80, 75, 71)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("boundary", ["none", "sponge", "cpml"])
def test_equals_the_passes(ews, n, boundary):
    kind = "force" if n[0] % 2 else "moment"
    p = synth.small_problem(*n, nt=24, boundary=boundary, kind=kind, width=2, seed=301)
    same(*both(ews, p))


@pytest.mark.parametrize("at", [(15.6, 15.6, 7.6), (16.4, 15.4, 8.4), (1.2, 30.6, 22.6)])
@pytest.mark.parametrize("kind", ["moment", "force"])
def test_source_across_blocks(ews, at, kind):
    """Taps of the source and of receivers in several blocks, or at the edge."""
    p = synth.small_problem(33, 33, 25, nt=30, boundary="none", kind=kind, width=4, seed=303)
    p.src_pos = np.array(at) * np.array(p.spacing)
    p.rec_pos = np.array([[16.5, 16.5, 8.5], [15.5, 10.0, 7.5], [31.0, 31.0, 23.0]]) * np.array(p.spacing)
    same(*both(ews, p))


@pytest.mark.parametrize("boundary", ["sponge", "cpml"])
def test_surface_and_coarse_medium(ews, boundary):
    p = synth.small_problem(40, 36, 30, nt=30, boundary=boundary, kind="moment", width=5, seed=304)
    p.free_surface = (8, 1e-3)
    same(*both(ews, p))
    q = synth.small_problem(40, 36, 30, nt=30, boundary=boundary, kind="force", width=5, seed=305,
                            layered=False)
    synth.with_coarse_medium(q, (9, 7, 5), seed=305, layer_vp=(2400.0, 2700.0, 2950.0))
    same(*both(ews, q))


def test_chunks_and_staged_receivers(ews):
    """1500 receivers stage fewer steps than the run has (several launches);
    a run in uneven chunks continues the same state."""
    p = synth.small_problem(40, 36, 28, nt=70, boundary="sponge", kind="moment", width=5, seed=306,
                            nrec=1500)
    a, b = both(ews, p)
    same(a, b)
    sim = ews.simulation_for(p)
    seis = np.zeros_like(a[0])
    for n0, k in ((0, 1), (1, 32), (33, 37)):
        sim.advance(n0, k, p.dt, seis, p.nt)
    assert np.array_equal(seis, a[0]) and np.array_equal(sim.get_state(), a[1])


# 24 taps a receiver, all in one block (16 x 16 x 8 cells of a 64^3 grid): up
# to and beyond the lines of the reverse sweep (8192) and the forward loop (49152)
@pytest.mark.parametrize("nrec", [341, 342, 2048, 2049])
def test_crowded_receivers(ews, nrec):
    """Receivers that share a block beyond what its CTA serves faster: the
    passes take them, with equal bits forward; the gradient to the order in
    which the residuals of one cell add up (2049 terms of like sign: about
    sqrt(2049) roundings of 6e-8 either way) and the separately compiled
    products: 1e-5."""
    p = synth.small_problem(64, 64, 64, nt=45, boundary="sponge", kind="moment", width=4, seed=310)
    p.src_pos = np.array([24.6, 24.2, 29.7]) * np.array(p.spacing)
    rng = np.random.default_rng(8)
    p.rec_pos = (np.array([23.0, 23.0, 27.0]) + rng.uniform(0.2, 0.4, (nrec, 3))) * np.array(p.spacing)
    same(*both(ews, p))
    sim = ews.simulation_for(p)
    seis = sim.run(p.nt, p.dt)
    assert sim.tile_shape == ("resident" if nrec <= 2048 else "32x8")
    obs = (0.9 * seis).astype(np.float32)
    a = sim.gradient(p.nt, p.dt, obs, ckpt_every=20)
    sim.set_tile_shape("32x8")
    b = sim.gradient(p.nt, p.dt, obs, ckpt_every=20)
    assert a[0] == pytest.approx(b[0], rel=1e-6)
    for q in range(3):
        x, y = a[1][q].astype(np.float64), b[1][q].astype(np.float64)
        assert 0 < np.linalg.norm(y) and np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y), q


def test_launches_are_counted_as_they_are(ews):
    """One launch, and one of the receivers, for as many steps as the staging
    holds; none of the passes."""
    for nrec, calls in ((5, 1), (1500, 3)):            # 4 MiB hold 29 steps of 1500 receivers
        p = synth.small_problem(40, 36, 28, nt=70, boundary="sponge", kind="moment", width=5, seed=308,
                                nrec=nrec)
        sim = ews.simulation_for(p)
        sim.run(p.nt, p.dt)
        ms, n = sim.profile(reset=True)
        assert n[ews.EWS_KERNEL_LOOP] == calls and n[ews.EWS_KERNEL_RECORD] == calls
        assert n.sum() == 2 * calls
        sim.advance(0, 10, p.dt, None, 10)             # nothing recorded
        n = sim.profile(reset=True)[1]
        assert n[ews.EWS_KERNEL_LOOP] == 1 and n.sum() == 1
        sim.set_profiling(True)                        # the passes, one by one
        sim.run(p.nt, p.dt)
        n = sim.profile()[1]
        assert n[ews.EWS_KERNEL_VELOCITY] == p.nt and n[ews.EWS_KERNEL_LOOP] == 0


def test_the_route_is_reported_and_leaves_the_table_alone(ews):
    """Neither run nor table entry is one of the passes': nothing was timed."""
    p = synth.small_problem(40, 36, 28, nt=20, boundary="sponge", kind="moment", width=5, seed=309)
    key = (ews.ews_grid(p.nx, p.ny, p.nz, *p.spacing), "sponge", "f32")
    ews.ews_tile_tuning_clear()
    sim = ews.simulation_for(p)
    sim.run(p.nt, p.dt)
    assert sim.tile_shape == "resident" and ews.ews_tile_tuned(*key) == 0
    entry = {"nx": p.nx, "ny": p.ny, "nz": p.nz, "boundary": "sponge", "storage": "f32", "shape": "32x4"}
    ews.ews_tile_tuning_import([entry])                # of a run that took the passes
    try:
        sim.run(p.nt, p.dt)
        assert sim.tile_shape == "resident" and ews.ews_tile_tuning_export() == [entry]
        sim.set_profiling(True)
        sim.run(p.nt, p.dt)
        assert sim.tile_shape == "32x4"
        sim.set_profiling(False)
        sim.set_tile_shape("32x16")
        assert sim.tile_shape == "32x16"
        sim.run(p.nt, p.dt)
        assert sim.tile_shape == "32x16"
        with pytest.raises(ews.EwsError) as e:         # a report, not a request
            sim.set_tile_shape(ews.EWS_TILE_RESIDENT)
        assert e.value.status == ews.EWS_EINVAL
    finally:
        ews.ews_tile_tuning_clear()


@pytest.mark.parametrize("n,boundary", [((33, 18, 17), "sponge"), ((64, 64, 64), "sponge"),
                                        ((80, 75, 71), "none"), ((40, 36, 28), "cpml")])
def test_a_wait_that_runs_out_ends_the_run(ews, n, boundary):
    """One block leaves at once: its neighbours' bounded waits give up, all
    blocks leave, the call returns EWS_ETIMEOUT, and the next run is as usual;
    the reverse sweep too."""
    p = synth.small_problem(*n, nt=12, boundary=boundary, kind="moment", width=2, seed=311)
    sim = ews.simulation_for(p)
    want = sim.run(p.nt, p.dt)
    obs = np.ones_like(want) * 1e-9
    assert sim.tile_shape == "resident"
    for _ in range(2):
        ews.ews_test_resident_wait(sim.handle, 50)
        with pytest.raises(ews.EwsError) as e:
            sim.run(p.nt, p.dt)
        assert e.value.status == ews.EWS_ETIMEOUT
        if boundary != "cpml":
            with pytest.raises(ews.EwsError) as e:
                sim.gradient(p.nt, p.dt, obs)
            assert e.value.status == ews.EWS_ETIMEOUT
        ews.ews_test_resident_wait(sim.handle, 0)
        assert np.array_equal(sim.run(p.nt, p.dt), want)
    for bad in (-1, 2000):
        with pytest.raises(ews.EwsError) as e:
            ews.ews_test_resident_wait(sim.handle, bad)
        assert e.value.status == ews.EWS_EINVAL


# blocks of at most 4 planes (a thread per cell), of 5 to 8 (4 cells per thread)
@pytest.mark.parametrize("n", [(12, 11, 10), (33, 18, 17), (16, 47, 33), (64, 60, 61)])
@pytest.mark.parametrize("boundary", ["none", "sponge"])
@pytest.mark.parametrize("budget", [-1, 0])
def test_gradient_equals_the_passes(ews, n, boundary, budget):
    """The reverse sweep in one launch against the reverse passes: the same
    products, summed by kernels compiled apart (a few roundings of 6e-8 per
    step over 45 steps), and residual taps that share cells in either order:
    1e-5.  History resident (one launch, flushed every 20 steps) and
    recomputed (one launch per segment)."""
    p = synth.small_problem(*n, nt=45, boundary=boundary, kind="moment", width=2, seed=307, nrec=40)
    obs = np.random.default_rng(5).standard_normal((3, 40, p.nt)).astype(np.float32) * 1e-9
    got = []
    for shape in ("auto", "32x8"):
        sim = ews.simulation_for(p)
        sim.set_tile_shape(shape)
        sim.set_history_budget(budget)
        got.append(sim.gradient(p.nt, p.dt, obs, ckpt_every=20))
    assert got[0][0] == pytest.approx(got[1][0], rel=1e-6)
    for q in range(3):
        a, b = got[0][1][q].astype(np.float64), got[1][1][q].astype(np.float64)
        assert np.linalg.norm(b) > 0
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b), q
