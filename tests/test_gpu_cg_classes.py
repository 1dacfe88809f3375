"""The CG's two classes of boxes (512- and 1024-thread CTAs, split at 4096
points) and the limits of their shared memory: FP64 boxes around the split,
beyond the fixed-point stencil's shared memory, elongated ones, equal and
different spacings, with right-hand sides far from 1 and non-finite ones;
and both forms on a system whose pair boxes lie on both sides."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2208_06097_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# at most 4096 points, 4096 < n within 28000 padded points, beyond those
EXTS = [(16, 16, 16), (17, 16, 16), (16, 17, 15), (1024, 2, 2), (1, 1, 513),
        (21, 20, 22), (25, 24, 23), (27, 28, 29), (2, 3, 1)]


def _solve(h, exts, seed, tol, scale=1.0):
    from paper_2208_06097_gb300 import sea
    rng = np.random.default_rng(seed)
    bs = [scale * rng.normal(size=(e[2], e[1], e[0])) for e in exts]
    rhs = torch.from_numpy(np.concatenate([b.ravel() for b in bs])).cuda()
    x = torch.empty_like(rhs)
    it, rc = sea.poisson_batch(h, exts, rhs, x, tol=tol)
    out, off = [], 0
    for e in exts:
        n = e[0] * e[1] * e[2]
        out.append(x[off:off + n].cpu().numpy().reshape(e[2], e[1], e[0]))
        off += n
    return bs, out, it, rc


@pytest.mark.parametrize("h", [(0.2, 0.2, 0.2), (0.2, 0.23, 0.18)])
@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e60])
def test_boxes_of_both_classes(h, scale):
    bs, xs, it, rc = _solve(h, EXTS, 3, 1e-10, scale)
    assert rc == 0
    for b, x, k in zip(bs, xs, it):
        xr, kr, _ = O.cg(b, h, tol=1e-10)
        # both stop at 1e-10 of b: FP64 rounding moves the iterates by far less
        assert np.abs(x - xr).max() <= 1e-9 * np.abs(xr).max()
        assert abs(int(k) - kr) <= 1


def test_values_outside_the_fixed_point_range():
    # outside 1e+-100 and for non-finite values the FP64 stencil decides: NaN
    # never converges, an infinite norm meets any relative tolerance at once,
    # and zero needs no step
    h = (0.25,) * 3
    assert _solve(h, [(5, 6, 7)], 1, 1e-8, float("nan"))[3] == 5
    for scale in (1e200, 0.0):
        bs, xs, it, rc = _solve(h, [(5, 6, 7)], 1, 1e-8, scale)
        assert rc == 0 and it[0] == 0 and not xs[0].any()


@pytest.mark.parametrize("precision,tol", [(0, 1e-9), (1, 2e-7)])
def test_system_with_boxes_of_both_classes(precision, tol):
    from paper_2208_06097_gb300 import sea
    s = synth.make_waters(2, 4.2, (44, 45, 44), seed=77)
    ref = O.apply_vxx(s.phi, s.cell, O.Params(cg_tol=1e-12 if precision == 0 else 1e-8))
    n = np.array([e.prod() for e in np.asarray(ref["ext"]).reshape(-1, 3)])
    assert (n > 4096).any() and (n <= 4096).any()
    with sea.Context(s.cell, s.grid, cg_tol=1e-12 if precision == 0 else 1e-8,
                     precision=precision) as ctx:
        phi = torch.from_numpy(s.phi).cuda()
        out = torch.empty_like(phi)
        ctx.set_orbitals(phi)
        e = ctx.apply_vxx(out)
    v = out.cpu().numpy()
    assert np.abs(v - ref["vxx"]).max() <= tol * max(1.0, np.abs(ref["vxx"]).max())
    assert abs(e - ref["exx"]) <= (1e-10 if precision == 0 else 1e-7) * abs(ref["exx"])
