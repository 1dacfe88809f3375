"""Two contexts whose kernels need different amounts of shared memory: the operator
of the larger one still applies after the smaller one was built, and
accumulations of different planes run from two threads at once."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [0, 1])
def test_long_lists_of_two_operators(precision):
    from paper_2208_06097_gb300 import sea
    grid, L = (16, 12, 8), 7.0
    N, dV = 16 * 12 * 8, 7.0 ** 3 / (16 * 12 * 8)
    ctxs, ops = [], []
    for n in (400, 250):  # lists of 400 and 250 entries on every tile: 102 and 64 KB
        rng = np.random.default_rng(n)
        q, _ = np.linalg.qr(rng.standard_normal((N, n)))
        F = torch.from_numpy(np.ascontiguousarray(q.T / np.sqrt(dV))).cuda()
        W = -F * torch.linspace(1.0, 2.0, n, dtype=torch.float64, device="cuda")[:, None]
        c = sea.Context((L,) * 3, grid, precision=precision)
        c.set_orbitals(F.reshape(n, 8, 12, 16))
        c.build_ace_from(W.reshape(n, 8, 12, 16).contiguous())
        ctxs.append(c)
        ops.append((F, W))
    psi = torch.randn((33, N), dtype=torch.float64, device="cuda")
    for c, (F, W) in zip(ctxs, ops):
        out = torch.empty_like(psi)
        c.apply_ace(psi.reshape(33, 8, 12, 16), out.reshape(33, 8, 12, 16))
        torch.cuda.synchronize()
        # -Mbar = diag(1..2): V psi = -sum_j |w_j> <w_j|psi> / a_j
        a = torch.linspace(1.0, 2.0, F.shape[0], dtype=torch.float64, device="cuda")
        want = -((W @ psi.T * dV) / a[:, None]).T @ W
        # N-term and n-term sums of numbers of size 1 (units of rounding, 2^-44 mixed)
        u = 2.0 ** -52 if precision == 0 else 2.0 ** -44
        assert float((out - want).abs().max()) <= 64 * F.shape[0] * u * float(want.abs().max())
        c.close()


def test_accumulations_from_two_threads():
    from paper_2208_06097_gb300 import sea, synth
    jobs = []
    for L, g in ((6.21, 40), (6.21, 104)):  # planes of 13 KB, and slabs of 87 KB planes
        phi, cell, grid = synth.make_waters_device(2, L, (g,) * 3, 7, torch.device("cuda"))
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        jobs.append((sea.Context(cell, grid, stream=st.cuda_stream), phi, torch.empty_like(phi)))
    want, bad = [], []
    for c, phi, out in jobs:
        c.set_orbitals(phi)
        want.append((c.apply_vxx(out), out.clone()))
    torch.cuda.synchronize()

    def work(k):
        c, phi, out = jobs[k]
        try:
            for _ in range(40):
                e = c.apply_vxx(out)
                torch.cuda.synchronize()
                if e != want[k][0] or not torch.equal(out, want[k][1]):
                    bad.append(k)
        except Exception as ex:  # noqa: BLE001
            bad.append(repr(ex))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for c, _, _ in jobs:
        c.close()
