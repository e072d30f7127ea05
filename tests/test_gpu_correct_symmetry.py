"""The tensor-core correction's covariances depend on the offset of node and site alone, not on the
node's place in its tile: with one site on a node, nodes on opposite sides of it get the same
bits (mirrored in x and in y; under an anisotropic map, through the site).  The grid spacing is
a power of two, so that every offset in grid units is a whole number."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ce():
    from paper_2109_11044_gb300.build import build
    build()
    import paper_2109_11044_gb300 as mod
    mod.load_library()
    return mod


@pytest.mark.parametrize("prec", ["f16x3", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("nu", [0.5, 1.5])
@pytest.mark.parametrize("aniso", [None, (0.45, 0.7)])
@pytest.mark.parametrize("i0,j0", [(30, 33), (70, 61), (95, 130)])
def test_correction_is_symmetric_about_a_site(ce, prec, nu, aniso, i0, j0):
    m, h = 200, 2.0 ** -8
    ctx = ce.Context(m, 0.0, 0.0, h, 1.0, 0.1, nu, 0.05)
    if aniso:
        ctx.set_anisotropy(*aniso)
    ctx.krige_weights([[j0 * h, i0 * h]], "local", np_=2, prec=prec)
    B = torch.linspace(0.5, 2.0, 20, device="cuda").reshape(20, 1).contiguous()
    v = ctx.correct(B, torch.zeros((20, m, m), device="cuda"))
    a, b = min(i0, m - 1 - i0), min(j0, m - 1 - j0)
    w = v[:, i0 - a:i0 + a + 1, j0 - b:j0 + b + 1]
    if aniso:
        assert torch.equal(w, w.flip(1, 2))
    else:
        assert torch.equal(w, w.flip(2)) and torch.equal(w, w.flip(1))
    assert float(v.abs().max()) > 1.9
