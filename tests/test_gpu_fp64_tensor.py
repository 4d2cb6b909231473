"""The FP64 form's contraction on the tensor cores (mol_fp64.cu) against the CUDA-core contraction, which the
no-allocation entry point runs, at node counts around its chunks (32 nodes) and windows (512 nodes), odd counts
(rows off 16-byte boundaries), uneven centres and row tiles of more than 56 states."""
import numpy as np
import pytest

import wpccc_inputs as wi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (nmax, lmax, nbins) per centre, Geta, Gtau
CASES = [
    ((1, 1), (0, 0), (1, 1), 5, 5),        # one chunk, mostly padding, odd rows
    ((2, 2), (1, 1), (2, 2), 31, 1),       # just below a chunk
    ((2, 3), (1, 2), (3, 2), 73, 7),       # 511 nodes: just below a window
    ((3, 2), (2, 1), (2, 3), 32, 16),      # 512: one window
    ((2, 2), (1, 1), (2, 2), 27, 19),      # 513: a window and one node
    ((4, 2), (0, 1), (56, 2), 36, 15),     # 60 target states of one projection: two row tiles
    ((6, 5), (5, 4), (2, 3), 37, 29),      # 1073 nodes, l = 5 and 4
]


@pytest.mark.parametrize("nmax,lmax,nbins,Geta,Gtau", CASES)
def test_tensor_contraction_matches_the_cuda_core_contraction(nmax, lmax, nbins, Geta, Gtau):
    import paper_2403_04252_gb300 as w
    basis = wi.make_basis(1.0, 2.0, nmax, lmax, nbins, 3.0, True, Nr=600, Geta=Geta, Gtau=Gtau)
    g = w.Basis(basis)
    zs = np.array([-9.5, -0.4, 0.0, 2.3])
    S, H = g.matrix_elements(0.7, 1.4, zs)
    S0, H0 = torch.full_like(S, float("nan")), torch.full_like(H, float("nan"))
    g.matrix_elements_noalloc(0.7, 1.4, zs, S0, H0)
    torch.cuda.synchronize()
    # both contractions round each of G terms' partial sums (or less) by 2^-53 of the sum of |terms|, which the
    # quadrature's Cauchy-Schwarz bound holds near 1 for the overlap of unit functions and near Z for the transfer;
    # the rotation adds up to (2l + 1)^2 such values with coefficients below 1
    bound = 2.0 * Geta * Gtau * 2.0 ** -53 * (2 * max(lmax) + 1) ** 2
    assert (S - S0).abs().max().item() <= bound
    assert (H - H0).abs().max().item() <= bound * max(2.0, H0.abs().max().item())
    # a position's elements do not depend on the others of the call
    S1, H1 = g.matrix_elements(0.7, 1.4, zs[2:3])
    torch.cuda.synchronize()
    assert torch.equal(S1[0], S[2]) and torch.equal(H1[0], H[2])
    g.close()


def test_a_non_finite_position_stays_non_finite_and_alone():
    import paper_2403_04252_gb300 as w
    basis = wi.make_basis(1.0, 1.0, 2, 1, 2, 2.0, True, Nr=600, Geta=16, Gtau=16)
    g = w.Basis(basis)
    S, H = g.matrix_elements(0.8, 1.2, np.array([0.5, np.nan, -1.0]))
    S0, H0 = g.matrix_elements(0.8, 1.2, np.array([0.5, -1.0]))
    torch.cuda.synchronize()
    NT = basis.T.N
    assert torch.equal(S[0], S0[0]) and torch.equal(H[0], H0[0])
    assert torch.equal(S[2], S0[1]) and torch.equal(H[2], H0[1])
    # column-major storage: the overlap block is rows < N_T of columns >= N_T
    assert not torch.isfinite(torch.view_as_real(S[1][NT:, :NT])).any()
    assert not torch.isfinite(torch.view_as_real(H[1][NT:, :NT])).any()
    g.close()


def test_a_wait_that_runs_out_reports_timeout_and_the_device_recovers():
    import paper_2403_04252_gb300 as w
    basis = wi.make_basis(1.0, 1.0, 2, 1, 2, 2.0, True, Nr=600, Geta=16, Gtau=16)
    g = w.Basis(basis)
    zs = np.array([-1.0, 0.0, 0.7])
    S0, H0 = g.matrix_elements(0.8, 1.2, zs)
    g.set_wait_limit(1)
    with pytest.raises(w.WpcccError) as e:
        g.matrix_elements(0.8, 1.2, zs)
    assert e.value.status == w.ETIMEOUT
    g.set_wait_limit(w.DEFAULT_WAIT_POLLS)
    S1, H1 = g.matrix_elements(0.8, 1.2, zs)
    torch.cuda.synchronize()
    assert torch.equal(S0, S1) and torch.equal(H0, H1)
    g.close()
