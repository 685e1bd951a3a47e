"""The stability test and the choice of the rescued blocks do not depend on the scale of the
weights (GPU)."""
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


@pytest.mark.parametrize("queues", [0, 1])
@pytest.mark.parametrize("shift", [-50, 50])
@pytest.mark.parametrize("name", ["ee_uug", "gg_ttg", "uu_ttg"])
def test_rescue_at_any_scale_of_the_weights(me, name, shift, queues):
    """Couplings scaled by a power of four scale every weight by a power of two, exactly, out of
    the range of float32 (2^-300, 2^300 with g^6): the same points and blocks are rescued."""
    p = torch.from_numpy(synth.flat_points(name, 2000, 63).p).cuda()
    kw = dict(precision=me.ME_PREC_MIXED, lanes_per_event=1, term_queues=queues)
    d = me.default_params()
    a, b = me.Handle(name, **kw), me.Handle(name, alpha=np.ldexp(d.alpha, 2 * shift),
                                            alpha_s=np.ldexp(d.alpha_s, 2 * shift), **kw)
    wa, wb = a.real_subtracted(p).cpu().numpy(), b.real_subtracted(p).cpu().numpy()
    assert a.last_rescued() > 100
    assert b.last_rescued() == a.last_rescued() and b.last_rescue_work() == a.last_rescue_work()
    np.testing.assert_array_equal(np.ldexp(wb, -6 * shift), wa)
