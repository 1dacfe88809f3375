"""ACE on a grid of more than 65,535 tiles of 8 x 4 x 4 points: the operator
applied to more vectors than the warp-wide kernels take, and the ACE vectors,
in both forms, against float64 products of the same W."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

L = 30.0
GRID = (208, 204, 204)  # 26 x 51 x 51 = 67,626 tiles


@pytest.mark.parametrize("precision", [0, 1])
def test_apply_and_vectors(precision):
    from paper_2208_06097_gb300 import sea
    n, m = 10, 9
    nx, ny, nz = GRID
    N, dV = nx * ny * nz, L ** 3 / (nx * ny * nz)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    q, _ = torch.linalg.qr(torch.randn((N, n), generator=g, dtype=torch.float64, device="cuda"))
    F = (q.T / dV ** 0.5).contiguous()
    B = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda")
    W = -((B @ B.T / n + torch.eye(n, dtype=torch.float64, device="cuda")) @ F)
    psi = torch.randn((m, N), generator=g, dtype=torch.float64, device="cuda")
    with sea.Context((L,) * 3, GRID, precision=precision) as ctx:
        ctx.set_orbitals(F.reshape(n, nz, ny, nx))
        ctx.build_ace_from(W.reshape(n, nz, ny, nx))
        _, Lc = ctx.ace_matrices()
        out = torch.empty_like(psi)
        ctx.apply_ace(psi.reshape(m, nz, ny, nx), out.reshape(m, nz, ny, nx))
        xi = torch.empty_like(F)
        ctx.ace_vectors(xi.reshape(n, nz, ny, nx))
    torch.cuda.synchronize()
    Li = torch.linalg.inv(torch.from_numpy(Lc).cuda())
    K = Li.T @ Li
    H = K @ (W @ psi.T) * dV
    # errors of the contraction: u of the largest product per point; of the n x n
    # products and the expansion: u of the sums of magnitudes, n terms each
    u = 2.0 ** -52 if precision == 0 else 2.0 ** -44
    wm = float(W.abs().max())
    dG = N * dV * u * wm * float(psi.abs().max())
    dH = float(K.abs().sum(1).max()) * (dG + 8 * n * u * float((W @ psi.T).abs().max()) * dV)
    bound = n * wm * (dH + 8 * u * float(H.abs().max()))
    assert float((out + H.T @ W).abs().max()) <= bound
    assert bound <= 1e-5 * float(out.abs().max())  # a wrong tile is far outside it
    want = Li @ W
    assert float((xi - want).abs().max()) <= 8 * n * u * float(Li.abs().sum(1).max()) * wm
