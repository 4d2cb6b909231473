"""The short-range direct elements of a model-potential target (k_direct_sr): four projectile radials per block, or one
where the nodes of four pass the shared memory, and the radials on the other side split over blocks by the number of
positions of the call."""
import numpy as np
import pytest

import wpccc_inputs as wi
from oracle import wpccc_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbins,Geta,Gtau", [(1, 12, 12), (5, 24, 16), (2, 77, 76)])   # 144, 384 and 5852 nodes
def test_short_range_direct_elements(nbins, Geta, Gtau):
    import paper_2403_04252_gb300 as w
    a, b = wi.li_parameters(0)
    basis = wi.li_basis(Z_p=1.0, a=a, b=b, nmax=3, lmax=2, nbins=nbins, kmax=2.0, Geta=Geta, Gtau=Gtau)
    g = w.Basis(basis)
    zs = np.linspace(-4.0, 4.0, 40)
    S, H = g.matrix_elements(0.9, 1.3, zs)
    S1, H1 = g.matrix_elements(0.9, 1.3, zs[7:8])
    torch.cuda.synchronize()
    assert torch.equal(S1[0], S[7]) and torch.equal(H1[0], H[7])
    So, Ho = O.assemble(basis, 0.9, 1.3, float(zs[7]))
    # the oracle's and the kernels' elements are the same sums in another order: the bar of the other element tests
    assert np.abs(w.natural(S)[7].cpu().numpy() - So).max() < 1e-12 * max(1.0, np.abs(So).max())
    assert np.abs(w.natural(H)[7].cpu().numpy() - Ho).max() < 1e-12 * max(1.0, np.abs(Ho).max())
    g.close()
