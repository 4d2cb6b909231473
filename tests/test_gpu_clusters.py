"""Systems and paths shared out over clusters of thread blocks: the cluster's size follows from the number of systems or
paths in a call, so the same system in calls of different sizes runs on clusters of different sizes.  Every element goes
through the same operations in the same order, so the results are the same bits; and they solve the system."""
import numpy as np
import pytest

import wpccc_inputs as wi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 31, 32, 33, 96, 131])
def test_lu_solve_does_not_depend_on_the_batch(N):
    import paper_2403_04252_gb300 as w
    rng = np.random.default_rng(N)
    A = rng.standard_normal((2, N, N)) + 1j * rng.standard_normal((2, N, N))
    B = rng.standard_normal((2, N, N)) + 1j * rng.standard_normal((2, N, N))

    def run(batch):
        S = w.colmajor(torch.from_numpy(np.resize(A, (batch, N, N)))).cuda()
        H = w.colmajor(torch.from_numpy(np.resize(B, (batch, N, N)))).cuda()
        piv, info = w.solve(S, H)
        torch.cuda.synchronize()
        assert int(info.abs().max()) == 0
        return S[:2], H[:2], piv[:2]

    S, H, piv = run(2)
    for batch in (20, 60, 170):     # from up to eight blocks per system down to one
        S1, H1, piv1 = run(batch)
        assert torch.equal(S, S1) and torch.equal(H, H1) and torch.equal(piv, piv1)
    X = w.natural(H).cpu().numpy()
    for k in range(2):
        # backward error of elimination with partial pivoting, growth allowed for
        bound = 64 * N * 2.0 ** -53 * np.linalg.cond(A[k]) * np.abs(X[k]).max()
        assert np.abs(X[k] - np.linalg.solve(A[k], B[k])).max() <= bound


def _bases():
    return {
        "one centre, 11 states": wi.make_basis(1.0, 1.0, 2, 1, 2, 2.0, False, Nr=400),
        "uneven centres": wi.make_basis(1.0, 1.0, (3, 2), (2, 1), (4, 5), 2.0, True, Nr=600, Geta=48, Gtau=16),
        "projectile part of three panels": wi.make_basis(1.0, 1.0, (2, 3), (1, 2), (3, 8), 2.0, True, Nr=600, Geta=48,
                                                         Gtau=16),
    }


@pytest.mark.parametrize("name", list(_bases()))
@pytest.mark.parametrize("solve", ["STAGE", "SCHUR", "MATRIX"])
@pytest.mark.parametrize("mode", [0, 2])
def test_a_path_does_not_depend_on_the_other_paths_of_the_call(name, solve, mode):
    import paper_2403_04252_gb300 as w
    basis = _bases()[name]
    if basis.n_centres == 1 and (solve != "STAGE" or mode != 0):
        pytest.skip("one form only")
    if solve == "MATRIX" and mode != 0:
        pytest.skip("the refined forms factorise S")
    g = w.Basis(basis)
    g.set_solve_mode(getattr(w, "SOLVE_" + solve))
    b = np.linspace(0.8, 6.0, 40)
    zg = [wi.uniform_zgrid(-0.5, 0.5, 0.1)[:k] for k in [4 + (p % 7) for p in range(40)]]   # uneven step counts
    c = g.propagate(b, 1.5, zg, precision_mode=mode)
    for sel in ([0], [3, 17], list(range(9, 21))):    # eight blocks per path at most, down to two or one
        c1 = g.propagate(b[sel], 1.5, [zg[p] for p in sel], precision_mode=mode)
        assert torch.equal(c1, c[sel])
    g.close()
