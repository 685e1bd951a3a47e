"""me_unweight through one handle from several threads, and while another thread captures a
stream (GPU)."""
import ctypes
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def me():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2503_07439_gb300 as m
    return m


class Call:
    """One unweighting with its own buffers, through the C ABI."""

    def __init__(self, me, n, seed):
        x = synth.uniforms(seed, 0, n, 2)
        w = np.where(x[1] < 0.4, -1.0, 1.0) * np.exp(3.0 * x[0])
        self.me, self.n, self.seed = me, n, seed
        self.w = torch.from_numpy(w).cuda()
        self.kept = torch.zeros(n, dtype=torch.int32, device="cuda")
        self.kw = torch.zeros(n, dtype=torch.float64, device="cuda")

    def __call__(self, h, w_max=0.0):
        nk, wm, no = ctypes.c_int64(), ctypes.c_double(), ctypes.c_int64()
        rc = self.me.library().me_unweight(h.h, self.w.data_ptr(), self.n, w_max, self.seed, 1, 0, self.kept.data_ptr(),
                                           self.kw.data_ptr(), ctypes.byref(nk), ctypes.byref(wm), ctypes.byref(no))
        return rc, nk.value, wm.value, no.value

    def result(self, r):
        assert r[0] == self.me.ME_OK, self.me.library().me_last_error()
        return r[1:], self.kept[: r[1]].clone(), self.kw[: r[1]].clone()


def test_unweight_during_a_capture(me):
    """The first call of a handle sizes its workspace, also while a thread captures in global mode."""
    c = Call(me, 5000, 81)
    ref = c.result(c(me.Handle("gg_tt")))
    h = me.Handle("gg_tt")
    x, y = torch.ones(64, device="cuda"), torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    got = []
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        y.copy_(x)
        t = threading.Thread(target=lambda: got.append(c(h)))
        t.start()
        t.join()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, y)
    r = c.result(got[0])
    assert r[0] == ref[0] and torch.equal(r[1], ref[1]) and torch.equal(r[2], ref[2])


def test_unweight_of_a_stream_under_capture_is_refused(me):
    c = Call(me, 5000, 82)
    h = me.Handle("gg_tt")
    ref = c.result(c(h))
    s = torch.cuda.Stream()
    x, y = torch.ones(64, device="cuda"), torch.zeros(64, device="cuda")
    torch.cuda.synchronize()
    h.set_stream(s.cuda_stream)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        y.copy_(x)
        assert c(h)[0] == me.ME_ERR_CUDA
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, y)
    h.set_stream(None)
    r = c.result(c(h))
    assert r[0] == ref[0] and torch.equal(r[1], ref[1])


def test_unweight_from_several_threads(me):
    h = me.Handle("gg_tt")
    sizes = (300, 40000, 1 << 20, 4099, 2049, 70001)
    calls = [Call(me, n, 83 + i) for i, n in enumerate(sizes)]
    ref = [c.result(c(me.Handle("gg_tt"), 4.0 * (i % 2))) for i, c in enumerate(calls)]
    bad = []

    def work(i):
        for _ in range(30):
            rc = calls[i](h, 4.0 * (i % 2))
            if rc[0] != me.ME_OK or rc[1:] != ref[i][0]:
                bad.append((i, rc))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[:3]
    for c, r in zip(calls, ref):
        k = r[0][0]
        assert torch.equal(c.kept[:k], r[1]) and torch.equal(c.kw[:k], r[2])
