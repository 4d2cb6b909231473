"""Elements of the FP64 form far from the target, where overlaps fall to 1e-20, element by element: the contraction in digits
against the chain of FP64 multiply-adds, which the no-allocation entry point runs."""
import math

import numpy as np
import pytest

import oracle.wpccc_oracle as oc
import wpccc_inputs as wi
from scipy import special

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _terms(basis, b, v, z):
    """Sum of |terms| of every overlap and transfer element: the absolute values summed over the nodes and rotated."""
    T, P = basis.T, basis.P
    nd = oc._nodes(basis, b, v, z)
    AT = np.abs(oc._state_tables(T, T.f, nd["rT"], nd["cT"], basis.grid.r))
    AP = np.abs(oc._state_tables(P, P.f, nd["rP"], nd["cP"], basis.grid.r))
    th = math.acos(z / math.hypot(b, z))
    DT, DP = np.abs(oc.rotation_matrix(T, th)), np.abs(oc.rotation_matrix(P, th))
    out = []
    for u in (np.ones_like(nd["rT"]), np.abs(oc.target_potential(basis, nd["rT"]))):
        X = np.zeros((T.N, P.N))
        for d in range(int(T.st_l.max() + P.st_l.max()) + 1):
            w = np.abs(nd["base"]) * np.abs(special.jv(d, nd["x"])) * u
            on = np.abs(T.st_m[:, None] - P.st_m[None, :]) == d
            X[on] = ((AT * w) @ AP.T)[on]
        out.append(DT @ X @ DP.T)
    return out


@pytest.mark.parametrize("ZP,Geta,Gtau", [(1.0, 48, 48), (2.0, 50, 30)])
def test_small_elements_keep_their_relative_accuracy(ZP, Geta, Gtau):
    import paper_2403_04252_gb300 as w
    basis = wi.make_basis(1.0, ZP, (3, 3), (2, 1), (4, 3), 2.5, True, Geta=Geta, Gtau=Gtau)
    # window lengths of 512, 128, 64 and 32 nodes, and blocks of fewer tau nodes (the last two)
    zs, b, v = np.array([8.0, -16.0, 20.0, -30.0, 38.0, 50.0, 75.0, -110.0]), 1.0, 1.4
    g = w.Basis(basis)
    S, H = g.matrix_elements(b, v, zs)
    S0, H0 = torch.zeros_like(S), torch.zeros_like(H)
    g.matrix_elements_noalloc(b, v, zs, S0, H0)
    torch.cuda.synchronize()
    S, H, S0, H0 = (w.natural(x).cpu().numpy() for x in (S, H, S0, H0))
    NT = basis.T.N
    for k, z in enumerate(zs):
        for A, A0, terms in zip((S, H), (S0, H0), _terms(basis, b, v, z)):
            # the chain rounds a sum of G terms, the digits less (tests/test_f64_order.py); a factor of two for the
            # rotation's sums and the oracle's |terms|
            bound = 2 * Geta * Gtau * 2.0 ** -53 * terms
            assert (np.abs(A[k] - A0[k])[:NT, NT:] <= bound + 1e-300).all(), z
    g.close()
