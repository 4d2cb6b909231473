"""The FP64 Schur form with its rank-N_T update on the tensor cores (schur_fp64.cu) against the LU of the whole overlap
matrix, at sizes around its chunks (16 target states), windows (256 target states) and tiles (32 and 128 projectile
states), and just below the size from which the update runs there."""
import numpy as np
import pytest

import wpccc_inputs as wi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("NT,NP", [(15, 33), (16, 31), (17, 32), (33, 1), (16, 128), (31, 129), (255, 33), (256, 32), (257, 5)])
def test_schur_update_matches_the_lu_form(NT, NP):
    import paper_2403_04252_gb300 as w
    # s states only: one bound state and NT - 1, NP - 1 packets
    basis = wi.make_basis(1.0, 1.0, (1, 1), (0, 0), (NT - 1, NP - 1), 1.5, True, Nr=600, Geta=24, Gtau=16)
    assert (basis.T.N, basis.P.N) == (NT, NP)
    g = w.Basis(basis)
    steps = 2
    b, v, zg = np.array([1.5, 4.0]), 1.5, wi.uniform_zgrid(-0.1, 0.1, 0.1)[:steps + 1]
    c = {}
    for mode in ("SCHUR", "STAGE"):
        g.set_solve_mode(getattr(w, "SOLVE_" + mode))
        c[mode] = g.propagate(b, v, zg).cpu().numpy()
    cond = 0.0
    for bk in b:
        S, _ = g.matrix_elements(float(bk), v, zg)
        cond = max([cond] + [np.linalg.cond(s) for s in w.natural(S).cpu().numpy()])
    # each stage's solve errs by a few N 2^-53 cond(S) of its result in either form, and a step's four stages move the
    # amplitudes by less than their own size
    assert np.isfinite(cond)
    assert np.abs(c["SCHUR"] - c["STAGE"]).max() <= 8 * steps * basis.N * 2.0 ** -53 * cond * np.abs(c["STAGE"]).max()
    g.close()
