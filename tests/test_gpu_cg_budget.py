"""The CG's time budget where the pairs are of both classes: (H2O)64 on 120^3 in
the FP64 form, whose large boxes hold the SMs first, so that CTAs of the other
class start when the large ones end.  The budget counts from the first start."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_budget_spans_both_classes():
    from paper_2208_06097_gb300 import sea, synth
    phi, cell, grid = synth.make_waters_device(64, 12.42, (120, 120, 120), 5, torch.device("cuda"))
    out = torch.empty_like(phi)

    def apply(timeout_ms, times=1):
        with sea.Context(cell, grid, timeout_ms=timeout_ms) as ctx:
            ctx.set_orbitals(phi)
            for _ in range(times):
                ctx.apply_vxx(out)
            return ctx.stats()["ms_cg"], ctx.plan()["ext"].astype(int).prod(1)

    ms, size = apply(0.0, times=3)
    assert 152 < (size > 4096).sum() < len(size) - 152
    # pairs are taken until close to the end of the stage, beyond 0.6 of it
    with pytest.raises(sea.SeaError) as e:
        apply(0.6 * ms)
    assert e.value.code == 7
    apply(4.0 * ms)
