"""The plain form's contractions with W (seven-digit exact splitting) against
extended-precision sums of the same FP64 inputs: M = Phi^T W dV and
V^ACE psi for a caller-supplied W, at row counts around the block sizes, odd
and even row lengths, dense lists of up to 40 orbitals (blocks of 16, and the
expansion's long lists), values of very different size, and non-finite
vectors."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

L = 7.0


def _orthonormal(n, grid, seed, spread):
    rng = np.random.default_rng(seed)
    N = int(np.prod(grid))
    F = rng.standard_normal((n, N))
    F *= np.exp(spread * rng.standard_normal((1, N)))  # points of different size
    q, _ = np.linalg.qr(F.T)
    dV = L ** 3 / N
    return np.ascontiguousarray(q.T / np.sqrt(dV)), dV


def _gram_bound(A, W, dV):
    """Rounding of an FP64 sum of the products: N 2^-53 sum |a w|, and the
    splitting's 2^-52 of the largest product of each 128-point tile at most."""
    N = A.shape[1]
    return dV * (np.sqrt(N) * 2.0 ** -52 * (np.abs(A) @ np.abs(W).T)
                 + N * 2.0 ** -52 * np.abs(A).max(1)[:, None] * np.abs(W).max(1)[None, :])


@pytest.mark.parametrize("n,grid,spread", [(3, (16, 12, 8), 0.0), (16, (16, 9, 10), 1.0),
                                           (17, (15, 12, 9), 1.0), (40, (18, 17, 12), 2.0)])
def test_m_and_apply(n, grid, spread):
    from paper_2208_06097_gb300 import sea
    nx, ny, nz = grid
    F, dV = _orthonormal(n, grid, n, spread)
    rng = np.random.default_rng(n + 1)
    B = rng.standard_normal((n, n))
    G = B @ B.T / n + np.eye(n)
    W = -(G @ F)
    shape = (n, nz, ny, nx)
    X = np.longdouble
    M = (F.astype(X) @ W.astype(X).T) * X(dV)
    with sea.Context((L,) * 3, grid) as ctx:
        ctx.set_orbitals(torch.from_numpy(F.reshape(shape).copy()).cuda())
        ctx.build_ace_from(torch.from_numpy(W.reshape(shape).copy()).cuda())
        Mg, _ = ctx.ace_matrices()
        assert np.all(np.abs(Mg - M.astype(float)) <= _gram_bound(F, W, dV))
        K = np.linalg.inv(-0.5 * (M + M.T).astype(float))
        for m in (1, 5, 130):
            psi = rng.standard_normal((m, nz, ny, nx))
            y = torch.empty(psi.shape, dtype=torch.float64, device="cuda")
            ctx.apply_ace(torch.from_numpy(psi).cuda(), y)
            Gx = (W.astype(X) @ psi.reshape(m, -1).astype(X).T) * X(dV)
            want = -(K @ Gx.astype(float)).T @ W
            got = y.cpu().numpy().reshape(m, -1)
            # |H| rounding of the n x n products, then the n-term expansion
            scale = np.abs(W).max() * np.abs(K).sum(1).max() * np.abs(Gx).max().astype(float)
            assert np.abs(got - want).max() <= 64 * n * 2.0 ** -52 * scale


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("nx", [16, 15])
def test_non_finite_vectors_are_not_hidden(bad, nx):
    from paper_2208_06097_gb300 import sea
    grid = (nx, 12, 8)
    F, dV = _orthonormal(6, grid, 1, 0.5)
    shape = (6, 8, 12, nx)
    with sea.Context((L,) * 3, grid) as ctx:
        ctx.set_orbitals(torch.from_numpy(F.reshape(shape).copy()).cuda())
        ctx.build_ace_from(torch.from_numpy(-F.reshape(shape)).cuda())
        psi = torch.randn((3, 8, 12, nx), dtype=torch.float64, device="cuda")
        psi[1, 3, 5, 2] = bad
        y = torch.empty_like(psi)
        ctx.apply_ace(psi, y)
        assert torch.isnan(y[1]).all()
        assert torch.isfinite(y[0]).all() and torch.isfinite(y[2]).all()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx", [24, 23])
def test_vector_count_does_not_change_the_bits(precision, nx):
    # a few vectors go through warp-wide kernels, more through the 128-row
    # ones: the same digits and sums, hence the same bits
    from paper_2208_06097_gb300 import sea
    grid = (nx, 21, 22)
    F, dV = _orthonormal(19, grid, 2, 1.0)
    shape = (19, 22, 21, nx)
    W = -F - 0.3 * np.roll(F, 1, axis=0) - 0.3 * np.roll(F, -1, axis=0)
    with sea.Context((L,) * 3, grid, precision=precision) as ctx:
        ctx.set_orbitals(torch.from_numpy(F.reshape(shape).copy()).cuda())
        ctx.build_ace_from(torch.from_numpy(W.reshape(shape).copy()).cuda())
        psi = torch.randn((41, 22, 21, nx), dtype=torch.float64, device="cuda")
        whole = torch.empty_like(psi)
        ctx.apply_ace(psi, whole)
        for m in (1, 8, 9, 32, 33):
            y = torch.full((m,) + shape[1:], float("nan"), dtype=torch.float64, device="cuda")
            ctx.apply_ace(psi[:m].contiguous(), y)
            torch.cuda.synchronize()
            assert torch.equal(y, whole[:m]), m
