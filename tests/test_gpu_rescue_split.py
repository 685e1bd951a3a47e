"""Rescue lists on both sides of the line at which a block's top spins are given to different
warps, and the queues that the automatic choice takes with cuts (GPU)."""
import numpy as np
import pytest

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


def test_short_and_long_rescue_lists_agree(me):
    """With tol 0 every point's four blocks are rescued: 65,536 points list 262,144 blocks, more than
    the lanes of the resident grid (two blocks of 128 threads on each SM), and one warp takes both
    spins of a block; 1024 points list 4096, fewer than half the lanes, and the spins go to
    different warps.  Both add the same sums in the same order."""
    n, m = 1 << 16, 1024
    lanes = 2 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    assert 4 * n > lanes and 2 * 4 * m <= lanes
    kw = dict(precision=me.ME_PREC_MIXED, lanes_per_event=1, term_queues=me.ME_TERMS_MASKED, tol=0.0)
    h = me.Handle("gg_ttg", **kw)
    p, w = h.generate_flat(n, 91, 1000.0)
    ref = h.real_subtracted(p, w)  # also sizes the lists, and the grid with them
    assert h.last_rescue_work()[:2] == (n, 4 * n)
    for i in range(0, n, 8 * m):
        got = h.real_subtracted(p[:, :, i:i + m].contiguous(), w[i:i + m].contiguous())
        assert h.last_rescue_work()[:2] == (m, 4 * m)
        assert torch.equal(got, ref[i:i + m])


@pytest.mark.parametrize("name,cuts", [("ee_uug", dict(cut_abs_cos_axis_max=0.8)), ("gg_ttg", dict(cut_pt_min=60.0)),
                                       ("uu_ttg", dict(cut_abs_y_max=1.5))])
def test_automatic_queues_with_cuts(me, name, cuts):
    """Only the queues count the flagged points' Born configurations."""
    n = 1 << 19
    p, w = me.Handle(name, precision=me.ME_PREC_MIXED).generate_flat(n, 93, 100.0 if name == "ee_uug" else 1000.0)
    kw = dict(precision=me.ME_PREC_MIXED, lanes_per_event=1, **cuts)
    auto = me.Handle(name, **kw)
    fixed = {m: me.Handle(name, term_queues=getattr(me, "ME_TERMS_" + m), **kw) for m in ("QUEUED", "MASKED")}
    out = auto.real_subtracted(p, w)
    x = {m: h.real_subtracted(p, w) for m, h in fixed.items()}
    assert torch.equal(out, x["QUEUED"])
    z = (out == 0.0).cpu().numpy()
    assert 0.0 < z.mean() < 1.0
    assert sum(auto.last_rescue_configs()) == sum(fixed["QUEUED"].last_rescue_configs()) > 0
    assert sum(fixed["MASKED"].last_rescue_configs()) == 0
    np.testing.assert_array_equal((x["MASKED"] == 0.0).cpu().numpy(), z)
