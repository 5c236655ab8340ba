"""Calls of the allocation-free ion push from several threads.

Each call has a stream and buffers of its own.  It must wait for its own
stream alone -- not for a call that another thread made earlier on a stream
that is still held up -- and calls that overlap on the GPU must not disturb
one another.
"""
import threading
import time

import numpy as np
import pytest

from paper_2603_24010_gb300 import workloads as W
from test_zz_no_alloc import ion_set, same_multiset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import native
    native.lib()
    return torch, native


class Call:
    """One ion set with its buffers; ``run`` makes the call on a stream of its own."""

    def __init__(self, torch, native, seed, n, cells, scale):
        self.torch, self.native, self.n = torch, native, n
        self.cfg = W.scaled(W.gap_1d_fp64(seed=seed), beam_per_step=0, see_scale=scale, precision=W.FP32, n_cells=cells)
        xi, u, ids = ion_set(self.cfg, seed, n)
        E = 1e6 * np.random.default_rng(seed).standard_normal(cells)

        def dev(a, dtype):
            return torch.tensor(a, dtype=dtype, device="cuda")

        self.start = dev(xi, torch.float32), dev(u, torch.float32)
        self.x, self.u = self.start[0].clone(), self.start[1].clone()
        self.ids, self.E = dev(ids.view(np.int32), torch.int32), dev(E, torch.float64)
        self.cap = 4 * n + 16
        self.G = dev(np.full(cells + 1, -7), torch.int64)
        self.sx, self.su = (torch.zeros(self.cap, dtype=torch.float32, device="cuda") for _ in range(2))
        self.counts = torch.full((6,), -3, dtype=torch.int64, device="cuda")
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()

    def run(self):
        gap, _, see, _ = self.native.structs_from_config(self.cfg)
        with self.torch.cuda.stream(self.stream):
            for a, b in zip((self.x, self.u), self.start):
                a.copy_(b)
        rc = self.native.cp_push_ions_noalloc(
            gap, see, self.cfg["dt"], self.cfg["seed"], 0, 1, self.E.data_ptr(), self.x.data_ptr(), self.u.data_ptr(),
            self.ids.data_ptr(), self.n, self.G.data_ptr(), self.sx.data_ptr(), self.su.data_ptr(), self.cap,
            self.counts.data_ptr(), self.stream.cuda_stream)
        assert rc == self.native.OK, rc

    def result(self):
        c = self.counts.cpu().numpy()
        m = int(c[4])
        return c, self.G.cpu().numpy(), self.x.cpu().numpy(), self.u.cpu().numpy(), (
            self.sx.cpu().numpy()[:m], self.su.cpu().numpy()[:m])


def check(got, want):
    for a, b in zip(got[:4], want[:4]):
        np.testing.assert_array_equal(a, b)
    same_multiset(got[4], want[4])


def test_a_call_waits_for_its_own_stream_alone(env):
    torch, native = env
    calls = [Call(torch, native, 31 + k, 3000, 256, 8.0) for k in range(2)]
    want = []
    for c in calls:
        c.run()
        want.append(c.result())
    assert want[0][0][2] > 0  # electrons were emitted
    held, done = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(held):
        torch.cuda._sleep(2_000_000_000)  # about a second
        done.record()
    calls[0].stream.wait_event(done)
    t = threading.Thread(target=calls[0].run)
    t.start()
    time.sleep(0.2)  # the first call is under way, behind `held`
    calls[1].run()
    early = not done.query()
    t.join()
    assert early, "a call on a free stream waited for one on a stream that was held up"
    for c, w in zip(calls, want):
        check(c.result(), w)


def test_calls_that_overlap(env):
    torch, native = env
    calls = [Call(torch, native, 41 + k, n, cells, 8.0)
             for k, (n, cells) in enumerate([(400_000, 4096), (1000, 16), (90_001, 600), (5000, 256)])]
    want = []
    for c in calls:
        c.run()
        want.append(c.result())
    bad = []

    def many(c, w):
        try:
            for _ in range(8):
                c.run()
                check(c.result(), w)
        except BaseException as e:  # reported by the main thread
            bad.append(e)

    ts = [threading.Thread(target=many, args=cw) for cw in zip(calls, want)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if bad:
        raise bad[0]
