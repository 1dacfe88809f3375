"""What the plain form's exact splitting holds: M against the largest values of
each segment of 64 points (half a tile of 8 x 4 x 4), the expansion against each
point's own largest value, where the data's size varies by many powers of two
within a tile.  Against extended-precision sums of the same FP64 inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

L = 7.0
GRID = (24, 12, 12)
N = GRID[0] * GRID[1] * GRID[2]
DV = L ** 3 / N


def _segments():
    """Index of the half tile (8 x 4 x 2 points) of every grid point."""
    z, y, x = np.meshgrid(*(np.arange(g) for g in GRID[::-1]), indexing="ij")
    return ((z // 2 * (GRID[1] // 4) + y // 4) * (GRID[0] // 8) + x // 8).ravel()


def _profile(kind):
    x = np.arange(N) % GRID[0]
    rng = np.random.default_rng(3)
    return {"even": np.zeros(N), "rising": 1.0 * (x % 8), "steep": 3.0 * (x % 8),
            "ragged": 6.0 * rng.standard_normal(N)}[kind]


def _data(n, kind, anti):
    """Orthonormal F whose points follow 2^profile, and W = -G F 2^shift: with
    `anti` W falls by as much as F rises (M is then not a form of G any more)."""
    rng = np.random.default_rng(n)
    p = np.exp2(_profile(kind))
    q, _ = np.linalg.qr((rng.standard_normal((n, N)) * p).T)
    F = np.ascontiguousarray(q.T / np.sqrt(DV))
    B = rng.standard_normal((n, n))
    G = B @ B.T / n + np.eye(n)
    return F, np.ascontiguousarray(-(G @ F) / (p * p if anti else 1.0))


def _matrices(F, W, precision):
    from paper_2208_06097_gb300 import sea
    n = F.shape[0]
    shape = (n,) + GRID[::-1]
    xi = torch.empty(shape, dtype=torch.float64, device="cuda")
    with sea.Context((L,) * 3, GRID, precision=precision, ace_decomp=0) as ctx:
        ctx.set_orbitals(torch.from_numpy(F.reshape(shape)).cuda())
        ctx.build_ace_from(torch.from_numpy(W.reshape(shape)).cuda())
        M, Lc = ctx.ace_matrices()
        if ctx.stats()["ace_eigen"]:
            return M, None, None
        ctx.ace_vectors(xi)
    return M, Lc, xi.cpu().numpy().reshape(n, N)


@pytest.mark.parametrize("kind,anti", [("even", False), ("rising", False), ("rising", True),
                                       ("steep", True), ("ragged", False)])
def test_m_against_the_segments_maxima(kind, anti):
    F, W = _data(12, kind, anti)
    X = np.longdouble
    M = ((F.astype(X) @ W.astype(X).T) * X(DV)).astype(float)
    seg = _segments()
    nseg = seg.max() + 1
    fm, wm = np.zeros((12, nseg)), np.zeros((12, nseg))
    for s in range(nseg):
        fm[:, s], wm[:, s] = np.abs(F[:, seg == s]).max(1), np.abs(W[:, seg == s]).max(1)
    # a product errs by at most 2^-56 of the two segments' powers of two for either
    # factor (each power at most twice the maximum), with either sign: six standard
    # deviations of 64 of them a segment; then the sums of the partials
    split = 6.0 * 2.0 ** -55 * 4.0 * np.sqrt(64.0 * ((fm * fm) @ (wm * wm).T))
    part = np.zeros((12, 12))
    for s in range(nseg):
        part += np.abs(F[:, seg == s] @ W[:, seg == s].T)
    bound = DV * (split + 12 * 2.0 ** -53 * part) + 2.0 ** -52 * np.abs(M)
    plain, _, _ = _matrices(F, W, 0)
    assert np.all(np.abs(plain - M) <= bound)
    mixed, _, _ = _matrices(F, W, 1)  # six digits do not meet it
    assert np.any(np.abs(mixed - M) > bound)


@pytest.mark.parametrize("kind", ["even", "rising", "steep", "ragged"])
def test_expansion_against_the_points_own_values(kind):
    F, W = _data(12, kind, False)
    _, Lc, xi = _matrices(F, W, 0)
    X = np.longdouble
    Li = np.linalg.inv(Lc)  # and one correction step: far below the bound
    Li = Li.astype(X) @ (2 * np.eye(12, dtype=X) - Lc.astype(X) @ Li.astype(X))
    want = Li @ W.astype(X)
    size = np.abs(Li).max(1)[:, None] * np.abs(W).max(0)[None, :]
    # twelve terms within 2^-55 of the point's largest W and the vector's largest H
    # (powers of two: 2; the entries' scales on a tile differ by at most 2^8 here),
    # and L^-1 within 2^6 units of its largest entries
    assert np.all(np.abs(xi - want) <= (12 * 2 * 2.0 ** 8 * 2.0 ** -55 + 12 * 64 * 2.0 ** -53) * size)
