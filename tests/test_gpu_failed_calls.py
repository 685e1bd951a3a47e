"""A call that fails half way, or overlaps with another stream's, spoils no later call (GPU).

The failures are made on the host: me_internal_fail_stage lets the next evaluation report a launch
error at one of its stages, with the stages before it launched."""
import ctypes

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


def _fail(me, stage):
    f = me.library().me_internal_fail_stage
    f.argtypes, f.restype = [ctypes.c_int], None
    f(stage)


CALLS = [("gg_ttg", "real_subtracted", dict(term_queues=0)), ("gg_ttg", "real_subtracted", dict(term_queues=1)),
         ("uu_ttg", "real_subtracted", dict(term_queues=0, queued_rescue=1)),
         ("ee_uug", "real_subtracted", dict(term_queues=0, rescue=0)), ("gg_tt", "born", {}), ("gg_ttgg", "born", {}),
         ("uu_tt", "born", dict(term_queues=1, cut_pt_min=50.0))]


@pytest.mark.parametrize("stage", [1, 2, 3])
@pytest.mark.parametrize("name,entry,kw", CALLS)
def test_replay_and_call_after_a_failure(me, name, entry, kw, stage):
    b = synth.flat_points(name, 1500, 71)
    p, w = torch.from_numpy(b.p).cuda(), torch.from_numpy(b.wgt).cuda()
    h = me.Handle(name, precision=me.ME_PREC_MIXED, lanes_per_event=4 if name == "gg_ttgg" else 1, **kw)
    s = torch.cuda.Stream()
    h.set_stream(s.cuda_stream)
    out = torch.empty(b.n, dtype=torch.float64, device="cuda")
    f = getattr(h, entry)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        f(p, w, out)  # sizes the scratch
    torch.cuda.synchronize()
    ref, work = out.clone(), h.last_rescue_work()
    h.set_accumulators([0.0, 0.0, 0.0])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        f(p, w, out)

    def failing():
        _fail(me, stage)
        with pytest.raises(me.MEError):
            f(p, w, out)
        torch.cuda.synchronize()

    failing()
    out.zero_()
    torch.cuda.synchronize()
    g.replay()  # captured before the failure
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and h.last_rescue_work() == work
    failing()
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2, stream=s, capture_error_mode="relaxed"):  # captured after one
        f(p, w, out)
    for call in (lambda: f(p, w, out), g2.replay):
        out.zero_()
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        assert torch.equal(out, ref) and h.last_rescue_work() == work
    # the failed calls are not in the accumulators, the others are
    np.testing.assert_allclose(h.accumulators(), [3 * ref.sum().item(), 3 * (ref * ref).sum().item(), 3 * b.n], rtol=1e-12)


def test_tree_calls_overlapping_on_two_streams(me):
    """Born calls of one handle on two streams may overlap; what they leave behind is harmless."""
    n = (1 << 20, 1500, 1 << 18, 300)
    h = me.Handle("gg_ttg", precision=me.ME_PREC_MIXED, lanes_per_event=1, term_queues=0)
    p = [h.generate_flat(k, 73 + k, 1000.0)[0] for k in n]
    ref = [h.born(x) for x in p]
    sub = h.real_subtracted(p[1])
    work = h.last_rescue_work()
    out = [torch.empty_like(x) for x in ref]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for i in range(40):
        h.set_stream(streams[i % 2].cuda_stream)
        h.born(p[i % 4], out=out[i % 4])
    torch.cuda.synchronize()
    h.set_stream(None)
    assert all(torch.equal(a, b) for a, b in zip(out, ref))
    h.set_accumulators([0.0, 0.0, 0.0])
    assert torch.equal(h.real_subtracted(p[1]), sub) and h.last_rescue_work() == work
    assert torch.equal(h.born(p[2]), ref[2])
    x = torch.cat([sub, ref[2]])
    np.testing.assert_allclose(h.accumulators(), [x.sum().item(), (x * x).sum().item(), x.numel()], rtol=1e-12)
