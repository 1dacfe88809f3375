"""Device memory of the ACE operator: the digit images of W follow its support,
not the grid, and where the device has no room for W's digits and images the
operator is built and applied in parts, with the same M and, through the
general expansion, the same result to rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("precision", [0, 1])
def test_images_follow_the_support(precision):
    # four narrow orbitals in a wide cell of 131,072 tiles: an image of every
    # tile would take 7.5 GB (6.4 GB mixed), those of the tiles in use 0.1 of it
    from paper_2208_06097_gb300 import sea
    n, g, L = 4, 256, 40.0
    x = torch.arange(g, dtype=torch.float64, device="cuda") * (L / g)
    phi = torch.empty((n, g, g, g), dtype=torch.float64, device="cuda")
    for k in range(n):
        e = torch.exp(-0.9 * (x - (8.0 + 8.0 * k)) ** 2)
        phi[k] = e[:, None, None] * e[None, :, None] * e[None, None, :]
        phi[k] /= torch.linalg.norm(phi[k].reshape(-1)) * (L / g) ** 1.5
    W = torch.empty_like(phi)
    with sea.Context((L,) * 3, (g,) * 3, precision=precision) as ctx:
        ctx.set_orbitals(phi)
        ctx.apply_vxx(W)
        before = _free()
        ctx.build_ace()
        assert before - _free() < 1.5e9
        # sum_i <phi_i|V^ACE phi_i> = E_xx^ACE, the images in use
        out = torch.empty_like(phi)
        ctx.apply_ace(phi, out)
        e = float((phi * out).sum()) * (L / g) ** 3
        assert abs(e - ctx.stats()["exx_ace"]) <= 1e-9 * abs(e)


@pytest.mark.parametrize("precision", [0, 1])
def test_little_memory(precision):
    from paper_2208_06097_gb300 import sea
    n, m, L = 16, 40, 20.0
    grid = (160, 160, 160)  # 32,000 tiles: digits 0.9 GB, images 0.9 GB in the plain form
    nx, ny, nz = grid
    N, dV = nx * ny * nz, L ** 3 / (nx * ny * nz)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    q, _ = torch.linalg.qr(torch.randn((N, n), generator=g, dtype=torch.float64, device="cuda"))
    F = (q.T / dV ** 0.5).contiguous()
    del q
    B = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda")
    W = -((B @ B.T / n + torch.eye(n, dtype=torch.float64, device="cuda")) @ F)
    psi = torch.randn((m, N), generator=g, dtype=torch.float64, device="cuda")

    def run(left):
        with sea.Context((L,) * 3, grid, precision=precision) as ctx:
            ctx.set_orbitals(F.reshape(n, nz, ny, nx))
            out = torch.empty_like(psi)
            fill = None
            if left:
                fill = torch.empty(_free() - left, dtype=torch.uint8, device="cuda")
            ctx.build_ace_from(W.reshape(n, nz, ny, nx))
            M, _ = ctx.ace_matrices()
            for v in (m, 5):  # the 128-row and the warp-wide kernels
                ctx.apply_ace(psi[:v].reshape(v, nz, ny, nx), out[:v].reshape(v, nz, ny, nx))
            torch.cuda.synchronize()
            del fill
        _free()
        return M, out

    M0, o0 = run(0)
    M1, o1 = run(900 * 1000 * 1000)  # lists and partial sums, half of the digits, no images
    assert np.array_equal(M0, M1)
    assert not torch.equal(o0, o1)  # the general expansion took part
    # n terms per point: units of rounding (2^-44 mixed) of the largest value, n of them
    u = 2.0 ** -52 if precision == 0 else 2.0 ** -43
    assert float((o0 - o1).abs().max()) <= 16 * n * u * float(o0.abs().max())
