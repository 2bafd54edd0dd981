"""The library's device-memory accounting and its optional cap
(ews_set_memory_limit): a call whose allocations would exceed the cap
returns EWS_ENOMEM without asking CUDA, releases what it had set up, and
leaves the other simulations and the CUDA context usable -- the same path a
full device takes, exercised here without a failing device allocation."""
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
    E.ews_set_memory_limit(-1)


def rel(a, b):
    a = np.asarray(a, np.float64)
    b = np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def test_accounting_follows_create_and_destroy(ews):
    base = ews.ews_memory_in_use()
    p = synth.small_problem(40, 36, 28, nt=20, boundary="cpml", width=5, seed=3)
    sim = ews.simulation_for(p)
    sim.run(p.nt, p.dt)
    held = ews.ews_memory_in_use()
    pitch = (p.nx + 31) // 32 * 32
    # at least the 9 wavefields, 3 medium arrays and 18 C-PML arrays
    assert held - base >= (9 + 3 + 18) * 4 * pitch * p.ny * p.nz
    sim.close()
    assert ews.ews_memory_in_use() == base


def test_capped_create_and_gradient_return_enomem(ews):
    p = synth.small_problem(40, 36, 28, nt=60, boundary="sponge", width=5, seed=4)
    sim = ews.simulation_for(p)
    want = sim.run(p.nt, p.dt)
    obs = (want * 1.1).astype(np.float32)
    held = ews.ews_memory_in_use()
    try:
        ews.ews_set_memory_limit(held + (1 << 20))
        assert ews.ews_memory_limit() == held + (1 << 20)
        with pytest.raises(ews.EwsError) as e:          # ~100 MB of wavefields and medium
            ews.Simulation(128, 128, 128, (10.0, 10.0, 10.0), boundary="sponge", width=8)
        assert e.value.status == ews.EWS_ENOMEM
        assert "memory limit" in str(e.value)
        assert ews.ews_memory_in_use() == held       # the partial set-up was released
        # the existing simulation still runs, with the same result
        assert np.array_equal(sim.run(p.nt, p.dt), want)
        # the gradient's adjoint state and checkpoints do not fit under the cap
        with pytest.raises(ews.EwsError) as e:
            sim.gradient(p.nt, p.dt, obs, ckpt_every=20)
        assert e.value.status == ews.EWS_ENOMEM
        assert np.array_equal(sim.run(p.nt, p.dt), want)
    finally:
        ews.ews_set_memory_limit(-1)
    # without the cap the same simulation computes the gradient a fresh one does
    m1, g1 = sim.gradient(p.nt, p.dt, obs, ckpt_every=20)
    fresh = ews.simulation_for(p)
    m2, g2 = fresh.gradient(p.nt, p.dt, obs, ckpt_every=20)
    assert m1 == pytest.approx(m2, rel=1e-6)
    for q in range(3):
        assert rel(g1[q], g2[q]) <= 1e-6


def test_history_budget_stays_under_the_cap(ews):
    """With the automatic history budget, a cap that leaves room for the
    checkpoints but not for the whole velocity history makes the gradient
    recompute segments instead of failing, and the result is unchanged."""
    p = synth.small_problem(40, 36, 28, nt=120, boundary="sponge", width=5, seed=6)
    obs = (ews.simulation_for(p).run(p.nt, p.dt) * 0.9).astype(np.float32)
    ref = ews.simulation_for(p)
    m0, g0 = ref.gradient(p.nt, p.dt, obs, ckpt_every=20)   # history resident
    sim = ews.simulation_for(p)
    sim.run(p.nt, p.dt)
    pitch = (p.nx + 31) // 32 * 32
    field = 4 * pitch * p.ny * p.nz
    # adjoint state (17 FP32 + 8 FP64 fields), 6 checkpoints of 9 fields,
    # 40 history slots of 3 fields (the full history needs 121), staging
    room = (17 + 16 + 6 * 9 + 40 * 3 + 3) * field + (1 << 20)
    try:
        ews.ews_set_memory_limit(ews.ews_memory_in_use() + room)
        m1, g1 = sim.gradient(p.nt, p.dt, obs, ckpt_every=20)
        assert ews.ews_memory_in_use() <= ews.ews_memory_limit()
    finally:
        ews.ews_set_memory_limit(-1)
    assert m1 == pytest.approx(m0, rel=1e-6)
    for q in range(3):
        assert rel(g1[q], g0[q]) <= 1e-5


def test_capped_batch_returns_enomem(ews):
    import torch
    probs = [synth.small_problem(40, 36, 28, nt=40, boundary="sponge", width=5, seed=7 + i)
             for i in range(2)]
    shots = []
    for p in probs:
        d = {"sim": ews.simulation_for(p), "nt": p.nt, "dt": p.dt,
             "seis": torch.zeros((3, p.rec_pos.shape[0], p.nt), device="cuda"),
             "observed": torch.zeros((3, p.rec_pos.shape[0], p.nt), device="cuda")}
        for k in ("g_lam", "g_mu", "g_rho"):
            d[k] = torch.zeros((p.nz, p.ny, p.nx), device="cuda")
        shots.append(d)
    try:
        ews.ews_set_memory_limit(ews.ews_memory_in_use())
        with pytest.raises(ews.EwsError) as e:
            ews.ews_batch(shots, ckpt_every=20)
        assert e.value.status == ews.EWS_ENOMEM
    finally:
        ews.ews_set_memory_limit(-1)
    ews.ews_batch(shots, ckpt_every=20)
    torch.cuda.synchronize()
    for p, d in zip(probs, shots):
        want = ews.simulation_for(p).run(p.nt, p.dt)
        assert rel(d["seis"].cpu().numpy(), want) <= 1e-6


def test_gradient_batch_runs_in_waves_under_the_limit(ews):
    """Three gradient shots whose gradient state fits the limit two at a time
    but not three at once: ews_batch splits them into waves (the forward shot
    rides with the first) and gives the results of the one-by-one path, which
    itself releases earlier shots' gradient state when it needs the room."""
    import torch
    probs = [synth.small_problem(40, 36, 28, nt=60, boundary="sponge", width=5, seed=20 + i,
                                 kind=("moment", "force")[i % 2]) for i in range(4)]
    rng = np.random.default_rng(3)

    def shots():
        out = []
        for i, p in enumerate(probs):
            sim = ews.simulation_for(p)
            sim.set_history_budget(0)                  # one segment of history per shot
            d = {"sim": sim, "nt": p.nt, "dt": p.dt,
                 "seis": torch.zeros((3, p.rec_pos.shape[0], p.nt), device="cuda")}
            if i < 3:
                obs = rng.standard_normal((3, p.rec_pos.shape[0], p.nt)).astype(np.float32) * 1e-9
                d["observed"] = torch.from_numpy(obs).cuda()
                for k in ("g_lam", "g_mu", "g_rho"):
                    d[k] = torch.zeros((p.nz, p.ny, p.nx), device="cuda")
            out.append(d)
        return out

    rng = np.random.default_rng(3)
    a = shots()
    rng = np.random.default_rng(3)
    b = shots()
    torch.cuda.synchronize()
    pitch = (probs[0].nx + 31) // 32 * 32
    field = 4 * pitch * probs[0].ny * probs[0].nz
    # per gradient shot: 17 FP32 + 8 FP64 adjoint fields, 2 checkpoints of 9
    # fields, 21 history slots of 3 fields, seismogram buffers: ~120 fields
    per_shot = (17 + 16 + 18 + 63 + 4) * field
    try:
        ews.ews_set_memory_limit(ews.ews_memory_in_use() + 2.5 * per_shot)
        ma = ews.ews_batch(a, ckpt_every=20, zchunk=12)      # the executor's waves
        torch.cuda.synchronize()
        for d in a:                                    # the last wave's state
            d["sim"].release_workspace()
        mb = ews.ews_batch(b, ckpt_every=20, mode=ews.EWS_BATCH_SEQUENTIAL)
        torch.cuda.synchronize()
    finally:
        ews.ews_set_memory_limit(-1)
    for i in range(4):
        assert rel(a[i]["seis"].cpu().numpy(), b[i]["seis"].cpu().numpy()) <= 1e-6, i
        if i < 3:
            assert ma[i] == pytest.approx(mb[i], rel=1e-6)
            for k in ("g_lam", "g_mu", "g_rho"):
                assert rel(a[i][k].cpu().numpy(), b[i][k].cpu().numpy()) <= 1e-5, (i, k)


def fused_problem(ews, seed):
    """A grid beyond the one-launch time loop whose tile-table entry is the
    fused step, and the bytes of one of its fields."""
    p = synth.small_problem(96, 72, 72, nt=30, boundary="sponge", width=6, seed=seed, kind="moment")
    ews.ews_tile_tuning_import([{"nx": 96, "ny": 72, "nz": 72, "boundary": "sponge", "storage": "f32",
                                 "shape": "fused"}])
    # receivers that the wave reaches within the run
    p.rec_pos = np.array([p.src_pos + np.array(o) * p.spacing for o in ([3.2, 1.1, 0.4], [-2.3, 2.6, 3.9])])
    return p, 4 * 96 * 72 * 72


def test_second_wavefield_sets_give_way(ews):
    """The set that a simulation keeps for the fused step makes no call fail:
    another simulation that does not fit beside it gets its memory, and a run
    that finds no room for one takes the two passes (to the rounding of the
    two kernels, 1e-6).  A shape asked for by name still fails."""
    import gc
    gc.collect()                                       # simulations of other tests
    p, field = fused_problem(ews, 11)
    a = ews.simulation_for(p)
    a.set_tile_shape("32x8")
    a.run(p.nt, p.dt)                                  # the seismogram buffer of host runs
    a.set_tile_shape("auto")
    before = ews.ews_memory_in_use()
    want = a.run(p.nt, p.dt)
    assert a.tile_shape == "fused" and ews.ews_memory_in_use() == before + 9 * field
    try:
        ews.ews_set_memory_limit(ews.ews_memory_in_use() + 4 * field)
        b = ews.simulation_for(p)                      # 12 fields: the set's 9 and 3 of the 4
        assert rel(b.run(p.nt, p.dt), want) <= 1e-6 and b.tile_shape == "32x8"
        assert rel(a.run(p.nt, p.dt), want) <= 1e-6 and a.tile_shape == "32x8"
        b.set_tile_shape("fused")
        with pytest.raises(ews.EwsError) as e:
            b.run(p.nt, p.dt)
        assert e.value.status == ews.EWS_ENOMEM
    finally:
        ews.ews_set_memory_limit(-1)
    assert np.array_equal(a.run(p.nt, p.dt), want) and a.tile_shape == "fused"
    a.release_workspace()                              # frees the set
    b.close()
    assert ews.ews_memory_in_use() <= before
    assert np.array_equal(a.run(p.nt, p.dt), want)
    # the gradient's working memory gets the set as well
    obs = np.zeros_like(want)
    try:
        ews.ews_set_memory_limit(before + 9 * field + (1 << 16))
        with pytest.raises(ews.EwsError) as e:         # more than the set
            a.gradient(p.nt, p.dt, obs, ckpt_every=10)
        assert e.value.status == ews.EWS_ENOMEM
        assert ews.ews_memory_in_use() < before + 9 * field
    finally:
        ews.ews_set_memory_limit(-1)
    assert np.array_equal(a.run(p.nt, p.dt), want)


def test_sets_are_taken_between_the_runs_of_another_thread(ews):
    """One thread runs the fused step while another creates simulations that
    take its set back whenever no run is using it: every run gives the same."""
    import gc
    import threading
    gc.collect()                                       # simulations of other tests
    p, field = fused_problem(ews, 12)
    a = ews.simulation_for(p)
    want = a.run(p.nt, p.dt)
    stop, bad, shapes = threading.Event(), [], set()

    def runs():
        while not stop.is_set() and not bad:
            try:
                got = a.run(p.nt, p.dt)
            except ews.EwsError as e:
                bad.append(e)
                return
            shapes.add(a.tile_shape)
            if rel(got, want) > 1e-6:
                bad.append(rel(got, want))

    t = threading.Thread(target=runs)
    try:
        ews.ews_set_memory_limit(ews.ews_memory_in_use() + 40 * field)   # a quarter holds a set
        t.start()
        for _ in range(30):
            held = []
            while len(held) < 40:                      # three or four fit
                try:
                    held.append(ews.Simulation(96, 72, 72, p.spacing, boundary="sponge", width=6))
                except ews.EwsError as e:
                    assert e.status == ews.EWS_ENOMEM
                    break
            assert 3 <= len(held) <= 4
            for s in held:
                s.close()
    finally:
        stop.set()
        t.join()
        ews.ews_set_memory_limit(-1)
        ews.ews_tile_tuning_clear()
    assert not bad and "fused" in shapes


def test_batch_without_room_for_second_sets(ews):
    """Shots that would run one by one with the fused step, where the memory
    limit leaves no room for its second wavefield sets: the batch runs all the
    same, and keeps none of the memory of its trial."""
    import torch
    import gc
    gc.collect()
    p, field = fused_problem(ews, 13)
    ews.ews_batch_tuning_clear()
    try:
        want = ews.simulation_for(p).run(p.nt, p.dt)
        for shape in ("fused", "auto"):                # by name (ENOMEM alone), from the table
            shots = [{"sim": ews.simulation_for(p), "nt": p.nt, "dt": p.dt,
                      "seis": torch.zeros((3, p.rec_pos.shape[0], p.nt), device="cuda")}
                     for _ in range(2)]
            for d in shots:
                d["sim"].set_tile_shape(shape)
            before = ews.ews_memory_in_use()
            ews.ews_set_memory_limit(before + 8 * field)
            ews.ews_batch(shots)
            ews.ews_set_memory_limit(-1)
            for d in shots:
                assert rel(d["seis"].cpu().numpy(), want) <= 1e-6
            assert ews.ews_memory_in_use() == before
            ews.ews_batch_tuning_clear()
    finally:
        ews.ews_set_memory_limit(-1)
        ews.ews_batch_tuning_clear()
        ews.ews_tile_tuning_clear()


@pytest.mark.parametrize("mode", ["default", "one_by_one"])
def test_batch_trial_keeps_no_set_where_the_executor_wins(ews, mode):
    """A batch leaves its simulations a second wavefield set only where it ran
    them with the fused step."""
    import torch
    p, field = fused_problem(ews, 14)
    ews.ews_batch_tuning_clear()
    shots = [{"sim": ews.simulation_for(p), "nt": p.nt, "dt": p.dt,
              "seis": torch.zeros((3, p.rec_pos.shape[0], p.nt), device="cuda")} for _ in range(3)]
    before = ews.ews_memory_in_use()
    try:
        kw = {} if mode == "default" else {"mode": ews.EWS_BATCH_ONE_BY_ONE}
        ews.ews_batch(shots, **kw)
        ran = [d["sim"].profile(reset=True)[1] for d in shots]
        ews.ews_batch(shots, **kw)                     # the cached choice
        alone = [d["sim"].profile(reset=True)[1].sum() > 0 for d in shots]
        assert len(set(alone)) == 1 and (mode == "default" or all(alone)), ran
        assert ews.ews_memory_in_use() == before + (27 * field if alone[0] else 0)
    finally:
        ews.ews_batch_tuning_clear()
        ews.ews_tile_tuning_clear()


def test_small_grids_run_the_passes_where_the_loop_lacks_memory(ews):
    """The one-launch time loop of small grids has inboxes beside the
    wavefields and staging beside the receivers; what fitted the limit without
    them still does, and runs the passes (equal bits)."""
    import gc
    gc.collect()
    p = synth.small_problem(40, 36, 28, nt=40, boundary="sponge", width=5, seed=15, nrec=1500)
    base = ews.ews_memory_in_use()
    ref = ews.simulation_for(p)
    took = ews.ews_memory_in_use() - base
    want = ref.run(p.nt, p.dt)
    assert np.abs(want).max() > 0 and ref.tile_shape == "resident"
    ref.close()
    base = ews.ews_memory_in_use()
    field = 4 * 64 * 36 * 28                           # pitched rows of 64
    seis = 4 * want.size
    try:
        # wavefields, medium, taps of 20 bytes and a little, but no inbox and no staging
        ews.ews_set_memory_limit(base + 12 * field + 24 * 1500 * 20 + seis + (1 << 15))
        assert took + seis > ews.ews_memory_limit() - base
        sim = ews.simulation_for(p)
        assert np.array_equal(sim.run(p.nt, p.dt), want) and sim.tile_shape != "resident"
        sim.close()
        ews.ews_set_memory_limit(-1)
        sim = ews.simulation_for(p)                    # inboxes, but no staging
        sim.set_receivers(p.rec_pos[:1])
        ews.ews_set_memory_limit(ews.ews_memory_in_use() + 24 * 1500 * 20 + seis + (1 << 12))
        sim.set_receivers(p.rec_pos)
        assert np.array_equal(sim.run(p.nt, p.dt), want) and sim.tile_shape != "resident"
        ews.ews_set_memory_limit(-1)
        sim.set_receivers(p.rec_pos)
        assert np.array_equal(sim.run(p.nt, p.dt), want) and sim.tile_shape == "resident"
    finally:
        ews.ews_set_memory_limit(-1)
