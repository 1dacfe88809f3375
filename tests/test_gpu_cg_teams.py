"""Bare boxes shared by clusters of CTAs: every team size (chosen by the number of
boxes), boxes whose shares end inside a plane, at the edges of a thread's 1, 2
and 4 points, with fewer planes than CTAs, and single points; equal and
different spacings; the same batch through the entry point without
allocations."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EXTS = [(16, 16, 16), (16, 17, 15), (64, 64, 1), (1, 1, 513), (8, 8, 8), (9, 8, 8), (16, 16, 9),
        (7, 5, 3), (1, 1, 1), (17, 16, 16), (3, 20, 20)]


@pytest.mark.parametrize("h", [(0.2, 0.2, 0.2), (0.2, 0.23, 0.18)])
@pytest.mark.parametrize("fill", [0, 40, 90, 330])  # teams of 8, 4, 2 and fewer on 152 SMs
def test_teams_match_the_oracle(h, fill):
    from paper_2208_06097_gb300 import sea
    exts = EXTS + [(4, 3, 2)] * fill
    rng = np.random.default_rng(fill)
    bs = [rng.normal(size=(e[2], e[1], e[0])) for e in exts]
    rhs = torch.from_numpy(np.concatenate([b.ravel() for b in bs])).cuda()
    x, y = torch.full_like(rhs, float("nan")), torch.empty_like(rhs)
    it, rc = sea.poisson_batch(h, exts, rhs, x, tol=1e-10)
    it2, rc2 = sea.poisson_batch(h, exts, rhs, y, tol=1e-10, noalloc=True)
    assert rc == 0 and rc2 == 0
    assert torch.equal(x, y) and np.array_equal(it, it2)
    off = 0
    for b, e, k in zip(bs, exts, it):
        n = e[0] * e[1] * e[2]
        xk = x[off:off + n].cpu().numpy().reshape(b.shape)
        off += n
        xr, kr, _ = O.cg(b, h, tol=1e-10)
        # both stop at 1e-10 of b: FP64 rounding moves the iterates by far less
        assert np.abs(xk - xr).max() <= 1e-9 * np.abs(xr).max()
        assert abs(int(k) - kr) <= 1


def test_one_box_that_fits_no_team():
    # 16,900 points are more than the threads of two CTAs of 1024 hold, and 152
    # boxes leave two CTAs each: the batch is then solved by single CTAs
    from paper_2208_06097_gb300 import sea
    exts = [(26, 26, 25), (5, 6, 7)] + [(4, 3, 2)] * 150
    h = (0.2,) * 3
    rng = np.random.default_rng(5)
    bs = [rng.normal(size=(e[2], e[1], e[0])) for e in exts]
    rhs = torch.from_numpy(np.concatenate([b.ravel() for b in bs])).cuda()
    x = torch.empty_like(rhs)
    it, rc = sea.poisson_batch(h, exts, rhs, x, tol=1e-10)
    assert rc == 0
    n = 26 * 26 * 25
    for b, xk, k in ((bs[0], x[:n], it[0]), (bs[1], x[n:n + 210], it[1])):
        xr, kr, _ = O.cg(b, h, tol=1e-10)
        assert np.abs(xk.cpu().numpy().reshape(b.shape) - xr).max() <= 1e-9 * np.abs(xr).max()
        assert abs(int(k) - kr) <= 1
