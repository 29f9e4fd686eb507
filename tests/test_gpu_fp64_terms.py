"""The FP64 form's terms at double rounding: areas and gradients against the oracle, whose own error on
these inputs is 1e-13 A^2 and 3e-12 A (long double).

Bounds.  An area is a sum of about 60 terms of up to 120 A^2 that cancel: a rounding error of up to
0.7e-14 each, independent, adds up to 6e-14, four times that at the worst of some thousand atoms;
with the oracle's own error 4e-13.  A gradient entry contains the heights s of triple points over the
planes of their centres, R^2 - |z|^2 rounded to 2e-15 and divided by 2 s; the smallest s of these
inputs is 0.015 A, so 7e-14, times 2 pi R and some entries of such a triangle: 5e-12, and as much
again for the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,seed", [("globule", 1200, 3), ("globule", 5000, 0), ("rna", 13007, 1)])
def test_fp64_form_at_double_rounding(orc, gen, kind, n, seed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import api
    m = gen.make(kind, n, seed)
    x, r = torch.as_tensor(m.coords, device="cuda"), torch.as_tensor(m.radii, device="cuda")
    a, g = torch.empty_like(r), torch.empty_like(x)
    ctx = api.Context(precision="fp64")
    ctx.compute(x, r, a, g)
    ctx.status_sync()
    ctx.close()
    ra, _, rg = orc.sasa(m.coords, m.radii)
    assert np.abs(a.cpu().numpy() - ra).max() <= 4e-13
    assert np.abs(g.cpu().numpy() - rg).max() <= 1e-11
