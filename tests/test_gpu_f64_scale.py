"""The FP64 contraction in digits scales with its operands: radial functions multiplied by a power of two multiply the
elements by it, bit for bit, whatever the size of the products W A_P."""
import numpy as np
import pytest

import wpccc_inputs as wi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-40, 1, 6, 12, 40])
def test_elements_scale_with_the_radial_functions(power):
    import paper_2403_04252_gb300 as w
    zs = np.array([-6.0, 0.3, 9.0])

    def blocks(factor):
        basis = wi.make_basis(1.0, 2.0, 2, 1, 3, 2.0, True, Nr=600, Geta=24, Gtau=24)
        basis.P.f *= factor
        g = w.Basis(basis)
        S, H = g.matrix_elements(0.8, 1.2, zs)
        torch.cuda.synchronize()
        g.close()
        NT = basis.T.N
        return torch.stack([w.natural(x)[:, :NT, NT:] for x in (S, H)])

    one, scaled = blocks(1.0), blocks(2.0 ** power)
    assert torch.equal(scaled, one * 2.0 ** power)


@pytest.mark.parametrize("power", [-50, 20, 60])
def test_small_elements_scale_with_both_centres(power):
    import paper_2403_04252_gb300 as w
    zs = np.array([-6.0, 30.0, -80.0])

    def blocks(factor):
        basis = wi.make_basis(1.0, 1.0, 2, 1, 3, 2.0, True, Nr=600, Geta=24, Gtau=24)
        basis.T.f *= factor
        basis.P.f *= factor
        g = w.Basis(basis)
        S, H = g.matrix_elements(0.8, 1.2, zs)
        torch.cuda.synchronize()
        g.close()
        NT = basis.T.N
        return torch.stack([w.natural(x)[:, :NT, NT:] for x in (S, H)])

    one, scaled = blocks(1.0), blocks(2.0 ** power)
    assert torch.equal(scaled, one * 4.0 ** power)
