"""Simulations of several host threads: each thread's calls on its own
simulations, on their own streams, give what they give alone."""
import threading

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
    return E


def rel(a, b):
    a = np.asarray(a, np.float64)
    b = np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def test_loops_are_captured_while_others_come_and_go(ews):
    """A run captures its time loop (another dt: another loop) while another
    thread creates, uses and releases simulations on the default stream."""
    import torch
    p = synth.small_problem(48, 40, 36, nt=60, boundary="sponge", width=5, seed=401)
    a = ews.simulation_for(p)
    st = torch.cuda.Stream()
    a.set_stream(st.cuda_stream)
    a.set_tile_shape("32x8")
    dts = [p.dt * (1.0 - 0.01 * k) for k in range(20)]
    want = [a.run(p.nt, dt) for dt in dts]
    a.release_workspace()                              # the loops too
    stop, failed = threading.Event(), []

    def others():
        try:
            while not stop.is_set():
                s = ews.simulation_for(p)
                s.run(4, p.dt)
                s.release_workspace()
                s.close()
        except ews.EwsError as e:
            failed.append(e)

    t = threading.Thread(target=others)
    t.start()
    try:
        got = [a.run(p.nt, dt) for _ in range(3) for dt in dts]
    finally:
        stop.set()
        t.join()
    assert not failed
    for k, g in enumerate(got):
        assert np.array_equal(g, want[k % len(dts)]), k


@pytest.mark.parametrize("n,threads", [((24, 22, 20), 8), ((64, 60, 61), 3)])
def test_small_grids_in_several_threads(ews, n, threads):
    """One-launch loops, each with a CTA on most SMs, asked for on several
    streams at once: every run and gradient as alone."""
    import torch
    p = synth.small_problem(*n, nt=40, boundary="sponge", width=4, seed=402)
    ref = ews.simulation_for(p)
    want = ref.run(p.nt, p.dt)
    obs = (0.9 * want).astype(np.float32)
    gwant = ref.gradient(p.nt, p.dt, obs, ckpt_every=15)[1]
    sims = [ews.simulation_for(p) for _ in range(threads)]
    streams = [torch.cuda.Stream() for _ in sims]
    for s, st in zip(sims, streams):
        s.set_stream(st.cuda_stream)
    bad = []

    def work(s):
        try:
            for _ in range(12):
                if not np.array_equal(s.run(p.nt, p.dt), want):
                    bad.append("run")
                g = s.gradient(p.nt, p.dt, obs, ckpt_every=15)[1]
                # products and residuals in either order: 1e-5 as elsewhere
                bad.extend(q for q in range(3) if rel(g[q], gwant[q]) > 1e-5)
        except ews.EwsError as e:
            bad.append(e)

    pool = [threading.Thread(target=work, args=(s,)) for s in sims]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    assert not bad, bad
    assert all(s.tile_shape == "resident" for s in sims)
