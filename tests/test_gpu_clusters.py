"""Systems and paths shared out over clusters of thread blocks: the cluster's size follows from the number of systems or
paths in a call, so the same system in calls of different sizes runs on clusters of different sizes.  Every element goes
through the same operations in the same order, so the results are the same bits; and they solve the system."""
import numpy as np
import pytest

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
