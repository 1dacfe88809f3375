"""A bare box alone and in larger calls, where fewer CTAs share it: the sums then
add in another order, so the solutions agree to the tolerance and the iteration
counts to one, and each call gives the same bits every time."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

H = (0.21, 0.21, 0.24)
EXT = (14, 13, 15)


@pytest.mark.parametrize("noalloc", [False, True])
def test_alone_and_in_company(noalloc):
    from paper_2208_06097_gb300 import sea
    rng = np.random.default_rng(8)
    b = rng.normal(size=EXT[::-1])
    xr, kr, _ = O.cg(b, H, tol=1e-10)
    for others in (0, 30, 60, 140, 500):  # 8, 4, 4, 2 and 1 CTAs a box on 152 SMs
        exts = [EXT] + [(5, 6, 7)] * others
        rhs = torch.from_numpy(np.concatenate([b.ravel(), rng.normal(size=210 * others)])).cuda()
        got = []
        for _ in range(2):
            x = torch.full_like(rhs, float("nan"))
            it, rc = sea.poisson_batch(H, exts, rhs, x, tol=1e-10, noalloc=noalloc)
            assert rc == 0
            got.append((x, it))
        assert torch.equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
        xb = got[0][0][:b.size].cpu().numpy().reshape(b.shape)
        # both stop at 1e-10 of b: FP64 rounding moves the iterates by far less
        assert np.abs(xb - xr).max() <= 1e-9 * np.abs(xr).max()
        assert abs(int(got[0][1][0]) - kr) <= 1
