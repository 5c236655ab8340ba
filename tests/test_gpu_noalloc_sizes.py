"""The allocation-free ion push over the edges of its split.

A CTA takes at least 512 ions and requests 4096 at a time; its impacts come in
rounds of 1024, and a round's electrons go straight into the grid when they are
few.  Each call must give the context path's integers, survivors and electrons
exactly, with impacts in every CTA, at the smallest and the largest grid.
"""
import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W
from test_zz_no_alloc import ion_set, noalloc_step, same_multiset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return torch, native


@pytest.mark.parametrize("n,cells,scale", [
    (1, 4096, 20.0), (2, 16, 20.0), (511, 256, 8.0), (513, 4096, 8.0), (1024, 256, 0.0),
    (152 * 512 - 1, 4096, 8.0), (152 * 512 + 1, 256, 0.02), (152 * 1024 + 7, 600, 8.0),
    (1 << 19, 4096, 8.0), (1 << 19, 256, 0.02),
])
def test_matches_context_path(env, n, cells, scale):
    torch, native = env
    cfg = W.scaled(W.gap_1d_fp64(seed=7), beam_per_step=0, see_scale=scale, precision=W.FP32, n_cells=cells)
    xi, u, ids = ion_set(cfg, 23 + n % 97, n)
    g = native.Gap(cfg, max_steps=4, capacity=(64, n + 64, 15 * n + 64))
    g.set_particles(native.IONS, xi, u, ids)
    g.step(0, 0)
    E0 = g.grid()["E"].copy()
    g.step(0, 1)
    ref_G, ions, se, h = g.grid()["G"], g.particles(native.IONS)[:2], g.particles(native.SECONDARIES)[:2], g.history(1, 1)
    g.close()
    got = noalloc_step(torch, native, cfg, xi, u, ids, E0)
    c = got["counts"]
    assert list(c) == [h["absorbed"][0, 0, 1], h["absorbed"][0, 1, 1], h["emitted"][0, 0], h["emitted"][0, 1],
                       h["n_live"][0, 2], h["conv_count"][0]]
    if n > 1000:
        assert c[0] > n // 2 and (c[2] > 0 or scale == 0.0)
    np.testing.assert_array_equal(got["G"], ref_G)
    same_multiset(got["ions"], ions)
    same_multiset(got["se"], se)
