"""SCDM of orbitals without any density (or one that underflows), the norm check
switched off: rank deficient, at grid sizes where every point is a candidate of
the pivots and where there are too many, and the context stays usable."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("value", [0.0, 1e-200])
@pytest.mark.parametrize("n,grid", [(4, (8, 8, 8)), (4, (12, 11, 10)), (1, (8, 8, 8))])
def test_no_density_is_rank_deficient(n, grid, value):
    from paper_2208_06097_gb300 import sea
    nx, ny, nz = grid
    phi = torch.full((n, nz, ny, nx), value, dtype=torch.float64, device="cuda")
    with sea.Context((6.0,) * 3, grid, orth_tol=0.0) as ctx:
        for _ in range(2):
            with pytest.raises(sea.SeaError) as e:
                ctx.scdm(phi)
            assert e.value.code == 8
        with pytest.raises(sea.SeaError) as e:
            ctx.apply_vxx(torch.empty_like(phi))  # no orbitals were set
        assert e.value.code == 2
        ctx.scdm(torch.randn(phi.shape, dtype=torch.float64, device="cuda"))
