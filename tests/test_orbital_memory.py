"""Where sea_set_orbitals and sea_scdm read the caller's array: memory of the
context's device by the kernels themselves, any other by a copy first (another
GPU's may have no peer access)."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_pointer_rule_host(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    exe = tmp_path / "pointer_check"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-o", str(exe), os.path.join(HERE, "host", "pointer_check.cu")],
                   check=True, capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


@pytest.mark.gpu
def test_page_locked_array_as_device_array():
    torch = pytest.importorskip("torch")
    from paper_2208_06097_gb300 import sea, synth
    s = synth.make_waters(2, 6.21, 32, seed=77)
    phi = torch.from_numpy(s.phi).cuda()
    pinned = torch.empty(phi.shape, dtype=phi.dtype, pin_memory=True).copy_(phi)
    got = []
    with sea.Context(s.cell, s.grid) as ctx:
        for p in (phi.data_ptr(), pinned.data_ptr()):
            rc = sea.lib().sea_set_orbitals(ctx.handle, ctypes.c_void_p(p), s.n_orb, 1)
            assert rc == 0
            ctx.n_orb = s.n_orb
            out = torch.empty_like(phi)
            got.append((ctx.apply_vxx(out), out))
    assert got[0][0] == got[1][0] and torch.equal(got[0][1], got[1][1])
