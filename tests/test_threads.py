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
