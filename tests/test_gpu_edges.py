"""Sizes at which the kernels' tiles, warps and blocks end (GPU).

A point's result does not depend on the batch it is in: batches cut at the edges of warps and
blocks are compared with the same points of a larger batch, exactly where the same arithmetic
runs, otherwise to the rounding of a sum of at most 16 positive terms (1e-13)."""
import numpy as np
import pytest

import synth
from oracle import matrix_element as ome
from oracle.unweight import unweight

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


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("name,lanes", [("ee_uu", 0), ("gg_tt", 0), ("uu_tt", 0), ("uu_ttg", 4), ("gg_ttg", 4),
                                        ("gg_ttgg", 1), ("gg_ttgg", 2), ("gg_ttgg", 4), ("gg_ttgg", 8)])
def test_tree_batch_ends(me, name, lanes):
    b = synth.flat_points(name, 300, 41)
    for prec in (me.ME_PREC_FP64, me.ME_PREC_MIXED):
        if prec == me.ME_PREC_MIXED and name == "gg_ttgg" and lanes != 4:
            continue
        ref = me.Handle(name, precision=prec, lanes_per_event=lanes).born(_dev(b.p)).cpu().numpy()
        for n in (1, 7, 9, 15, 17, 31, 33, 127, 129, 255, 257):
            got = me.Handle(name, precision=prec, lanes_per_event=lanes).born(_dev(b.p[:, :, :n])).cpu().numpy()
            np.testing.assert_array_equal(got, ref[:n])
        if prec == me.ME_PREC_FP64 and lanes > 1:
            one = me.Handle(name, precision=prec, lanes_per_event=1).born(_dev(b.p)).cpu().numpy()
            np.testing.assert_allclose(ref, one, rtol=1e-13)


@pytest.mark.parametrize("name", ["gg_ttg", "gg_ttgg"])
def test_beams_off_the_axis(me, name):
    """The blocks' general form: beams turned off the z axis, against the oracle."""
    p = synth.flat_points(name, 200, 43).p
    s = np.min([p[0, i] * p[0, j] - (p[1:, i] * p[1:, j]).sum(0) for i in range(p.shape[1]) for j in range(i)], axis=0)
    p = p[:, :, s > 5e-4 * 4 * p[0, 0] ** 2][:, :, :9]
    c, t = np.cos(0.7), np.sin(0.7)
    q = p.copy()
    q[1], q[3] = c * p[1] + t * p[3], c * p[3] - t * p[1]
    ref = ome.me2(name, ome.to_points(q[:, :, :3]))
    for lanes in (4, 8):
        got = me.Handle(name, precision=me.ME_PREC_FP64, lanes_per_event=lanes).born(_dev(q)).cpu().numpy()
        assert np.max(np.abs(got[:3] / ref - 1)) < 1e-10
    mix = me.Handle(name, precision=me.ME_PREC_MIXED).born(_dev(q)).cpu().numpy()
    assert np.max(np.abs(mix / got - 1)) < 2e-5


@pytest.mark.parametrize("n", [1, 31, 33, 129, 1000])
def test_rescue_list_ends(me, n):
    """Every point goes through the item rescue, whose last block recombines the weights."""
    p = synth.approach_points("gg_ttg", 256, 45)[0].p
    kw = dict(precision=me.ME_PREC_MIXED, lanes_per_event=4, term_queues=me.ME_TERMS_MASKED)
    ref = me.Handle("gg_ttg", **kw).real_subtracted(_dev(p)).cpu().numpy()
    h = me.Handle("gg_ttg", **kw)
    for _ in range(2):
        got = h.real_subtracted(_dev(p[:, :, :n])).cpu().numpy()
        np.testing.assert_allclose(got, ref[:n], rtol=1e-9)


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 304 * 1024 + 1])
def test_accumulators_of_ragged_batches(me, n):
    b = synth.flat_points("ee_uu", n, 47)
    h = me.Handle("ee_uu", precision=me.ME_PREC_FP64)
    w = h.born(_dev(b.p), _dev(b.wgt)).cpu().numpy()
    w = np.concatenate([w, h.born(_dev(b.p), _dev(b.wgt)).cpu().numpy()])
    a = h.accumulators()
    # a sum of m positive terms in any order: below m 2^-53 relative, in practice sqrt(m) 2^-53
    np.testing.assert_allclose([a[0], a[1], a[2]], [w.sum(), (w * w).sum(), w.size], rtol=1e-12)


@pytest.mark.parametrize("name", ["gg_ttg", "ee_uug"])
def test_fks_sampler_block_ends(me, name):
    s = {"gg_ttg": 1000.0, "ee_uug": 100.0}[name]
    h = me.Handle(name, precision=me.ME_PREC_MIXED)
    p, w = h.generate_fks(1025, 51, s, first_point=3)
    for n in (1, 255, 256, 257, 513):
        q, v = h.generate_fks(n, 51, s, first_point=3)
        assert torch.equal(q, p[:, :, :n]) and torch.equal(v, w[:n])


@pytest.mark.parametrize("n", [31, 32, 33, 2047, 2048, 2049, 16385])
@pytest.mark.parametrize("w_max", [0.0, 2.0])
def test_unweighting_tile_ends(me, n, w_max):
    x = synth.uniforms(53, 0, n, 2)
    w = np.where(x[1] < 0.4, -1.0, 1.0) * np.exp(3.0 * x[0])
    special = [0.0, -0.0, 5e-324, -1e-300, 1e-38, 2.0, -2.0, np.nextafter(2.0, 3.0), 3.4e38]
    w[:: max(1, n // 40)][: len(special)] = special[: len(w[:: max(1, n // 40)])]
    idx, ew, wm, nover = unweight(w, w_max, synth.uniforms(53, 5, n, 1, first_point=7)[0])
    h = me.Handle("gg_ttg", precision=me.ME_PREC_MIXED)
    kept, kw, wm_d, nover_d = h.unweight(_dev(w), w_max=w_max, seed=53, stream=5, first_point=7)
    np.testing.assert_array_equal(kept.cpu().numpy(), idx)
    np.testing.assert_array_equal(kw.cpu().numpy(), ew)
    assert wm_d == wm and nover_d == nover


@pytest.mark.parametrize("name,cuts,mode", [("ee_uug", {}, "MASKED"), ("ee_uug", {"cut_thrust_max": 0.9}, "QUEUED"),
                                            ("uu_ttg", {}, "QUEUED")])
def test_automatic_queues(me, name, cuts, mode):
    n = 1 << 19
    p, w = me.Handle(name, precision=me.ME_PREC_MIXED).generate_flat(n, 55, 100.0 if name == "ee_uug" else 1000.0)
    auto = me.Handle(name, precision=me.ME_PREC_MIXED, lanes_per_event=1, **cuts)
    fixed = me.Handle(name, precision=me.ME_PREC_MIXED, lanes_per_event=1, term_queues=getattr(me, "ME_TERMS_" + mode), **cuts)
    assert torch.equal(auto.real_subtracted(p, w), fixed.real_subtracted(p, w))
    assert auto.last_rescue_configs() == fixed.last_rescue_configs()
    assert (sum(auto.last_rescue_configs()) > 0) == (mode == "QUEUED" and not cuts)
