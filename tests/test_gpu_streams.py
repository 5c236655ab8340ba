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


def make_any(native, what, stream):
    if what == "2d":
        cfg = W.scaled(W.gap_2d(4, 128, 128, 150_000, beam_per_step=400), see_scale=8.0)
        g = native.Gap2D(cfg, max_steps=200, stream=stream)
        xi, eta, ue, we, ui, wi = W.load_pairs_2d(cfg)
        g.set_particles(native.ELECTRONS, xi, eta, ue, we)
        g.set_particles(native.IONS, xi, eta, ui, wi)
        return g
    if what == "ensemble":
        cfgs = W.ensemble(24, seed=3, steps=200, thin=20, n_cells_max=2048)
        b = native.Batch(cfgs, max_steps=200, stream=stream)
        for i, cfg in enumerate(cfgs):
            xi, ue, ui = W.load_pairs(cfg)
            b.set_particles(i, native.ELECTRONS, xi, ue)
            b.set_particles(i, native.IONS, xi, ui)
        return b
    return make(native, configs()[0], stream)


def outcome(what, g):
    if what == "2d":
        return [g.history()["V_gap"], g.history()["n_live"], g.fields()["G"]]
    if what == "ensemble":
        return [x for i in range(0, 24, 5) for x in (g.history(i)["V_gap"], g.history(i)["n_live"], g.grid(i)["G"])]
    return [g.history()["V_gap"], g.history()["n_live"], g.grid()["G"]]


def test_all_paths_beside_one_another(env):
    torch, native = env
    paths = ["2d", "ensemble", "1d", "2d"]
    want = {}
    for what in set(paths):
        g = make_any(native, what, None)
        advance(native, g, [130, 1, 1, 60])
        want[what] = outcome(what, g)
        g.close()
    streams = [torch.cuda.Stream() for _ in paths]
    gaps = [make_any(native, what, st.cuda_stream) for what, st in zip(paths, streams)]
    ts = [threading.Thread(target=advance, args=(native, g, [130, 1, 1, 60])) for g in gaps]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for what, g in zip(paths, gaps):
        for a, b in zip(outcome(what, g), want[what]):
            np.testing.assert_array_equal(a, b, err_msg=what)
        g.close()
