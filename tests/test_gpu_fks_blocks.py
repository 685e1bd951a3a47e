"""The FKS sampler's two block sizes give the same points (GPU)."""
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


@pytest.mark.parametrize("name", ["gg_ttg", "uu_ttg", "ee_uug"])
def test_block_sizes_agree(me, name):
    """Blocks of 128 threads up to 19,456 points, of 256 above: a point depends on its index alone."""
    line = 152 * 128
    h = me.Handle(name, precision=me.ME_PREC_MIXED)
    s = 100.0 if name == "ee_uug" else 1000.0
    p, w = h.generate_fks(2 * line, 101, s, first_point=5)
    for n in (1, 127, 128, 129, 4099, line - 1, line, line + 1, line + 257):
        q, v = h.generate_fks(n, 101, s, first_point=5)
        assert torch.equal(q, p[:, :, :n]) and torch.equal(v, w[:n])
