"""The batched form's table of tuned workloads is bounded: a workload is known on its
second call, and tuned again (to the same result) after as many others as the table
holds."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(grid):
    from paper_2208_06097_gb300 import sea
    h = 0.4
    ax = [(torch.arange(g, dtype=torch.float64, device="cuda") - g // 2) * h for g in grid]
    e = [torch.exp(-1.1 * a * a) for a in ax]
    phi = (e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :])[None].contiguous()
    phi /= torch.linalg.norm(phi.reshape(-1)) * h ** 1.5
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with sea.Context([h * g for g in grid], grid, stream=st.cuda_stream) as ctx:
        ctx.set_orbitals(phi)
        out = torch.empty_like(phi)
        exx = sea.apply_vxx_batch([ctx], [out])[0]
        return ctx.stats()["batch_tune_ms"], exx, out


def test_table_of_workloads_is_bounded():
    first = (31, 30, 29)
    ms, exx, out = _run(first)
    assert ms > 0.0
    assert _run(first)[0] == 0.0  # known
    others = [(16 + k % 8, 16 + k // 8 % 8, 16 + k // 64) for k in range(256)]
    for grid in others:
        _run(grid)
    ms, exx2, out2 = _run(first)
    assert ms > 0.0  # given up and tuned again
    assert exx2 == exx and torch.equal(out2, out)
