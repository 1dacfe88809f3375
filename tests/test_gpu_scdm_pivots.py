"""SCDM pivots where the candidate classes matter: orbitals of very
different widths (classes opened one after another), a flat density (too many
candidates: every grid point is downdated), one orbital, and sizes around the
tiles of the rotation.  Against the oracle's pivoted QR."""
import numpy as np
import pytest

from oracle import scdm as S
from paper_2208_06097_gb300.synth import loewdin_orthonormalize

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _gaussians(n, grid, L, widths, seed):
    """n Gaussians at random centres, exponents spread over `widths`."""
    rng = np.random.default_rng(seed)
    ax = [np.arange(g) * (L / g) for g in grid]
    Z, Y, X = np.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    phi = np.zeros((n, grid[2], grid[1], grid[0]))
    al = np.exp(np.linspace(np.log(widths[0]), np.log(widths[1]), n))
    for k in range(n):
        c = rng.uniform(0, L, 3)
        d = [(V - x + L / 2) % L - L / 2 for V, x in zip((X, Y, Z), c)]
        phi[k] = np.exp(-al[k] * (d[0] ** 2 + d[1] ** 2 + d[2] ** 2))
    dV = L ** 3 / (grid[0] * grid[1] * grid[2])
    return loewdin_orthonormalize(phi, dV)


def _noise(n, grid, L, seed):
    phi = np.random.default_rng(seed).standard_normal((n, grid[2], grid[1], grid[0]))
    dV = L ** 3 / (grid[0] * grid[1] * grid[2])
    return loewdin_orthonormalize(phi, dV)


CASES = {
    "widths": lambda: _gaussians(12, (20, 21, 23), 10.0, (0.08, 4.0), 3),
    "flat": lambda: _noise(5, (16, 17, 18), 8.0, 4),
    "one": lambda: _gaussians(1, (9, 8, 10), 6.0, (1.0, 1.0), 5),
    "n33": lambda: _gaussians(33, (24, 22, 26), 12.0, (0.6, 3.0), 6),
    "n65": lambda: _gaussians(65, (25, 24, 23), 12.0, (0.8, 3.0), 7),
}


@pytest.mark.parametrize("name", CASES)
def test_pivots_and_rotation(name):
    from paper_2208_06097_gb300 import sea
    phi = CASES[name]()
    n = phi.shape[0]
    R, _ = np.linalg.qr(np.random.default_rng(9).standard_normal((n, n)))
    can = np.ascontiguousarray((R.T @ phi.reshape(n, -1)).reshape(phi.shape))
    grid = can.shape[:0:-1]
    L = {"widths": 10.0, "flat": 8.0, "one": 6.0}.get(name, 12.0)
    C, U, pt = S.scdm(can)
    with sea.Context((L,) * 3, grid) as ctx:
        Ug, cols = ctx.scdm(torch.from_numpy(can).cuda())
        assert np.array_equal(cols, C)
        assert np.abs(Ug - U).max() <= 1e-9
        # the context's orbitals are Phi U: V_xx on them equals V_xx on the
        # oracle's localized orbitals up to the rounding of their values
        out = torch.empty(can.shape, dtype=torch.float64, device="cuda")
        e = ctx.apply_vxx(out)
    with sea.Context((L,) * 3, grid) as ref:
        ref.set_orbitals(torch.from_numpy(np.ascontiguousarray(pt)).cuda())
        want = torch.empty_like(out)
        er = ref.apply_vxx(want)
    assert abs(e - er) <= 1e-9 * abs(er)
    assert float((out - want).abs().max()) <= 1e-8 * float(want.abs().max())
