"""The plan's row and column sums formed as the orbitals are read: boxes equal to
the oracle's for row lengths at the edges of the kernel's forms (and beyond
them), from device and host buffers, again after a localization; non-finite
values and norms found wherever they lie."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _orbitals(grid, cell, seed, n=3):
    """Normalized Gaussians (with tails over the cell's edges) plus noise."""
    rng = np.random.default_rng(seed)
    ax = [np.arange(g) * c / g for g, c in zip(grid, cell)]
    phi = np.empty((n, grid[2], grid[1], grid[0]))
    for i in range(n):
        f = 1.0
        for a, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
            d = ax[a] - rng.uniform(0, cell[a])
            d -= cell[a] * np.round(d / cell[a])
            f = f * np.exp(-d * d / (0.02 * cell[a] ** 2)).reshape(shape)
        phi[i] = f + 1e-6 * rng.normal(size=f.shape)
    dV = np.prod(cell) / np.prod(grid)
    return phi / np.sqrt((phi ** 2).sum((1, 2, 3)) * dV)[:, None, None, None], dV


@pytest.mark.parametrize("grid", [(24, 26, 25), (64, 13, 12), (65, 12, 13), (96, 14, 15), (97, 17, 12),
                                  (128, 12, 19), (129, 12, 12), (192, 12, 12), (193, 13, 12),
                                  (256, 12, 12), (257, 12, 13)])
def test_boxes_equal_the_oracles(grid):
    from paper_2208_06097_gb300 import sea
    cell = [0.3 * g for g in grid]
    phi, dV = _orbitals(grid, cell, grid[0])
    want = O.boxes(phi, dV, 10.0 ** -3.5)
    for host in (False, True):
        with sea.Context(cell, grid) as ctx:
            ctx.set_orbitals(phi if host else torch.from_numpy(phi).cuda())
            out = torch.empty(phi.shape, dtype=torch.float64, device="cuda")
            ctx.apply_vxx(out)
            np.testing.assert_array_equal(ctx.plan()["box"], want)
            ctx.apply_vxx(out)  # the plan again, from the same sums
            np.testing.assert_array_equal(ctx.plan()["box"], want)


def test_sums_of_localized_orbitals():
    # the localization replaces the orbitals: their sums are formed anew
    from paper_2208_06097_gb300 import sea
    grid, cell = (40, 41, 42), (12.0, 12.3, 12.6)
    phi, dV = _orbitals(grid, cell, 2)
    q, r = np.linalg.qr(phi.reshape(3, -1).T)
    phi = (q.T / np.sqrt(dV)).reshape(phi.shape).copy()
    mix = np.linalg.qr(np.random.default_rng(3).normal(size=(3, 3)))[0]
    can = (mix @ phi.reshape(3, -1)).reshape(phi.shape)
    a, b = np.empty_like(phi), np.empty_like(phi)
    with sea.Context(cell, grid) as ctx, sea.Context(cell, grid) as ref:
        ctx.set_orbitals(phi)  # leaves sums of other orbitals
        U, _ = ctx.scdm(can)
        e = ctx.apply_vxx(a)
        U = np.asarray(U.cpu() if hasattr(U, "cpu") else U).reshape(3, 3)
        loc = (U.T @ can.reshape(3, -1)).reshape(phi.shape)
        ref.set_orbitals(loc)
        e2 = ref.apply_vxx(b)
        np.testing.assert_array_equal(ctx.plan()["box"], ref.plan()["box"])
    assert abs(e - e2) <= 1e-10 * abs(e2) and np.abs(a - b).max() <= 1e-9


@pytest.mark.parametrize("grid", [(24, 26, 25), (65, 13, 12), (129, 12, 12), (257, 12, 13)])
def test_bad_values_anywhere(grid):
    from paper_2208_06097_gb300 import sea
    cell = [0.3 * g for g in grid]
    phi, _ = _orbitals(grid, cell, 1)
    for at, value in ((( -1, -1, -1, -1), np.nan), ((0, 0, 0, 0), np.inf), ((1, 5, -1, 23), -np.inf),
                      ((2, 3, 2, -1), 50.0)):
        bad = phi.copy()
        bad[at] = value
        with sea.Context(cell, grid) as ctx:
            with pytest.raises(sea.SeaError):
                ctx.set_orbitals(torch.from_numpy(bad).cuda())
