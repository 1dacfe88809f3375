"""The accumulation of planes in slabs of rows (planes of which three do not fit an
SM): two and three slabs, odd rows and planes, windows across every edge of
the cell, device and host outputs, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("grid", [(100, 98, 24), (101, 97, 23), (128, 128, 24), (159, 157, 22)])
def test_slabs_match_the_oracle(grid):
    from paper_2208_06097_gb300 import sea
    h = 0.3
    cell = [h * g for g in grid]
    # two narrow orbitals, one across the cell's corner and one at a slab's edge
    phi = []
    for cen in ((0.2, 0.3, 0.1), (1.5, 0.5 * cell[1], 1.0), (0.4, 0.5 * cell[1] + 1.0, 0.6)):
        f = 1.0
        for a, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
            d = np.arange(grid[a]) * h - cen[a]
            d -= cell[a] * np.round(d / cell[a])
            f = f * np.exp(-1.5 * d * d).reshape(shape)
        phi.append(f / np.sqrt((f * f).sum() * h ** 3))
    phi = np.ascontiguousarray(np.stack(phi))
    ref = O.apply_vxx(phi, cell, O.Params(cg_tol=1e-12))
    host = np.empty_like(phi)
    with sea.Context(cell, grid, cg_tol=1e-12) as ctx:
        ctx.set_orbitals(torch.from_numpy(phi).cuda())
        out = torch.full(phi.shape, float("nan"), dtype=torch.float64, device="cuda")
        e = ctx.apply_vxx(out)
        # the bounds of the other parity tests at this CG tolerance
        assert np.abs(out.cpu().numpy() - ref["vxx"]).max() <= 1e-9
        assert abs(e - ref["exx"]) <= 1e-10 * abs(ref["exx"])
        ctx.apply_vxx(host)
        assert np.array_equal(host, out.cpu().numpy())
        ctx.build_ace()  # reads the context's own copy
        ace = torch.empty_like(out)
        ctx.apply_ace(torch.from_numpy(phi).cuda(), ace)
        W, F = ref["vxx"].reshape(3, -1), phi.reshape(3, -1)
        M = F @ W.T * h ** 3
        want = W.T @ np.linalg.solve(0.5 * (M + M.T), W @ F.T * h ** 3)
        # W within 1e-9 on both sides, |M^-1| and |W^T phi| of order 1
        assert np.abs(ace.cpu().numpy().reshape(3, -1) - want.T).max() <= 1e-7
