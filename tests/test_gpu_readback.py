"""Read-backs through page-locked memory and straight to the caller.

Small ones go through a buffer of 256 KiB, larger ones (a long history, the
grid of many cells) straight to the caller's memory; both give the stored
bits.  Refused calls write nothing, the level a step call starts from survives
them, and an ensemble's instances share one buffer between threads.
"""
import ctypes as C
import threading

import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return native


def filled(native, cfg, max_steps):
    g = native.Gap(cfg, max_steps=max_steps)
    xi, ue, ui = W.load_pairs(cfg)
    g.set_particles(native.ELECTRONS, xi, ue)
    g.set_particles(native.IONS, xi, ui)
    return g


def equal(a, b):
    assert a.keys() == b.keys()
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def test_long_history_and_large_grid(native):
    cfg = W.scaled(W.gap_1d_fp64(seed=2), n_cells=11_000, n_pairs=2000, precision=W.FP32)
    g = filled(native, cfg, 1500)
    assert g.step(native.WEAK, 1500) in (None, 0)
    whole = g.history(0, 1501)
    pieces = [g.history(k, min(100, 1501 - k)) for k in range(0, 1501, 100)]
    equal(whole, {k: np.concatenate([p[k] for p in pieces]) for k in whole})
    grid = g.grid()
    phi, G = np.zeros(11_001), np.zeros(11_001, dtype=np.int64)
    assert native.lib().cp_read_grid(g.ctx, phi.ctypes.data_as(C.POINTER(C.c_double)), None, None,
                                     G.ctypes.data_as(C.POINTER(C.c_int64)), 11_001) == native.OK
    np.testing.assert_array_equal(phi, grid["phi"])
    np.testing.assert_array_equal(G, grid["G"])
    g.close()


@pytest.mark.parametrize("rows", [3, 1500])
def test_refused_reads_write_nothing(native, rows):
    cfg = W.scaled(W.gap_1d_fp64(seed=3), n_pairs=500)
    g = filled(native, cfg, 2000)
    g.step(native.STRICT, rows - 1)
    out = (native.cp_diag * (rows + 1))()
    C.memset(out, 0x5A, C.sizeof(out))
    before = bytes(out)
    assert native.lib().cp_read_history(g.ctx, 0, rows + 1, out) == native.ERR_ARG
    assert native.lib().cp_read_history(g.ctx, 2001, 1, out) == native.ERR_ARG
    assert bytes(out) == before
    assert native.lib().cp_read_history(g.ctx, 0, rows, out) == native.OK
    g.close()


def test_steps_after_a_refused_call(native):
    cfg = W.scaled(W.gap_1d_fp64(seed=4), n_pairs=500)
    a, b = filled(native, cfg, 40), filled(native, cfg, 40)
    a.step(native.STRICT, 40)
    for n in (1, 7, 0, 20):
        b.step(native.STRICT, n)
        assert native.lib().cp_step_strict(b.ctx, 41, 1e-12) == native.ERR_ARG
    assert native.lib().cp_step_strict(b.ctx, 13, 1e-12) == native.ERR_ARG
    b.step(native.STRICT, 12)
    assert a.level == b.level == 40
    ha, hb = a.history(), b.history()
    equal({k: v for k, v in ha.items() if k != "residual"}, {k: v for k, v in hb.items() if k != "residual"})
    a.close()
    b.close()


def test_ensemble_instances_read_from_threads(native):
    cfgs = [W.scaled(W.gap_1d_fp64(seed=s), n_pairs=400, n_cells=64 + 16 * s, precision=W.FP32) for s in range(6)]
    b = native.Batch(cfgs, max_steps=300)
    for i, cfg in enumerate(cfgs):
        xi, ue, ui = W.load_pairs(cfg)
        b.set_particles(i, native.ELECTRONS, xi, ue)
        b.set_particles(i, native.IONS, xi, ui)
    assert b.step(native.STRICT, 300) == 0
    want = [(b.history(i), b.grid(i)) for i in range(6)]
    got = [None] * 6

    def read(i):
        for _ in range(20):
            got[i] = (b.history(i), b.grid(i))

    ts = [threading.Thread(target=read, args=(i,)) for i in range(6)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, w in zip(got, want):
        equal(g[0], w[0])
        equal(g[1], w[1])
    b.close()
