"""Gaps advanced from several threads, each on a stream of its own.

Every push fills the device, so CTAs of one wait for the other's to leave and
start after some of their own launch have finished.  Each gap must still give
the integers it gives alone.
"""
import threading

import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return torch, native


def configs():
    large = W.scaled(W.gap_1d_fp32_large(5), n_pairs=400_000, beam_per_step=4000, see_scale=10.0, weight=4e9)
    small = W.scaled(W.gap_1d_fp64(6), n_pairs=60_000, beam_per_step=700, see_scale=10.0)
    return [large, W.scaled(large, seed=9, n_cells=1531, beam_mode=1), small, W.scaled(small, seed=8, n_cells=900)]


def make(native, cfg, stream):
    g = native.Gap(cfg, max_steps=400, stream=stream)
    xi, ue, ui = W.load_pairs(cfg)
    g.set_particles(native.ELECTRONS, xi, ue)
    g.set_particles(native.IONS, xi, ui)
    return g


def advance(native, g, calls):
    for n in calls:
        g.step(native.WEAK, n)


@pytest.mark.parametrize("calls", [[300], [1] * 60 + [140] + [3] * 33])
def test_threads_on_their_own_streams(env, calls):
    torch, native = env
    cfgs = configs()
    want = []
    for cfg in cfgs:
        g = make(native, cfg, None)
        advance(native, g, calls)
        want.append((g.history(), g.grid()["G"]))
        g.close()
    streams = [torch.cuda.Stream() for _ in cfgs]
    gaps = [make(native, cfg, st.cuda_stream) for cfg, st in zip(cfgs, streams)]
    ts = [threading.Thread(target=advance, args=(native, g, calls)) for g in gaps]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, (h, G) in zip(gaps, want):
        got = g.history()
        assert (got["absorbed"][:, 0, 1] > 0).any()
        for k in ("absorbed", "emitted", "injected", "n_live", "conv_count", "ion_energy_eV", "V_gap"):
            np.testing.assert_array_equal(got[k], h[k], err_msg=k)
        np.testing.assert_array_equal(g.grid()["G"], G)
        g.close()
