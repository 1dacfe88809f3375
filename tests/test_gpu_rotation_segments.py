"""The SCDM rotation beyond 512 orbitals, where the sum over the orbitals is taken
in two exact accumulations and the second is added to the stored first one.  The
localized orbitals are read at single grid points as M = Phi^T W dV with W the
points' indicators, against extended-precision sums with the call's own U."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [512, 513, 540])
def test_two_accumulations(n):
    from paper_2208_06097_gb300 import sea
    grid, L = (24, 25, 23), 9.0
    nx, ny, nz = grid
    N, dV = nx * ny * nz, L ** 3 / (nx * ny * nz)
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((N, n)))
    psi = np.ascontiguousarray(q.T / np.sqrt(dV))
    pts = np.sort(rng.choice(N, n, replace=False))
    pts[:3], pts[-1] = (0, 127, 128), N - 1  # edges of the 128-point tiles, the last point
    W = torch.zeros((n, N), dtype=torch.float64, device="cuda")
    W[torch.arange(n), torch.from_numpy(pts)] = 1.0 / dV
    with sea.Context((L,) * 3, grid) as ctx:
        U, _ = ctx.scdm(torch.from_numpy(psi.reshape(n, nz, ny, nx)).cuda())
        ctx.build_ace_from(W.reshape(n, nz, ny, nx))  # indefinite: the eigen form; M stands
        M, _ = ctx.ace_matrices()
    assert np.abs(U.T @ U - np.eye(n)).max() <= n * 2.0 ** -48
    col = list(range(0, n, 9)) + [1, 2, n - 1]  # of the points
    X = np.longdouble
    want = U.astype(X).T @ psi[:, pts[col]].astype(X)  # [orbital][point]
    # n terms: the digits' 2^-55 of the point's and of the column's largest value
    # (powers of two: 4) and as much for the dropped diagonals; two roundings; M's
    # own rounding
    scale = np.abs(U).max(0)[:, None] * np.abs(psi[:, pts[col]]).max(0)[None, :]
    bound = n * 8 * 2.0 ** -55 * scale + 4 * 2.0 ** -53 * np.abs(want).astype(float) + 2.0 ** -52
    assert np.all(np.abs(M[:, col] - want) <= bound)
