"""The entry point that allocates nothing on a GPU without room for the work space of its digit
products (512 MiB, loaded by the first call): the call runs the FP64 kernel and has the same values."""

import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1])
import afqmc_inputs as ai
from paper_2505_18519_gb300 import afqmc as lib
N, nu, nd, G, P, n = 50, 10, 9, 60, 8, 20
rng = np.random.default_rng(4)
s = ai.make_system(ai.SystemSpec(N, nu, nd, G, 3, True, 11))
Phi = np.linalg.qr(rng.standard_normal((n, N, nu)))[0]
phi = np.concatenate([Phi[::P], Phi[::P][:, :, :nd]], axis=2) + 0.05j * rng.standard_normal((3, N, nu + nd))
args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (s.h, s.L, Phi, phi.view(np.float64))]
out = [torch.zeros(2 * k, dtype=torch.float64).cuda() for k in (n, n, n * G)]
torch.cuda.synchronize()
if sys.argv[3] == "full":
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), dtype=torch.uint8, device="cuda")
for _ in range(2):
    lib.local_energy_noalloc(N, nu, nd, G, n, P, *args, *out)
np.savez(sys.argv[2], *[o.cpu().numpy() for o in out])
"""


def test_a_full_gpu_runs_the_fp64_kernel(tmp_path):
    """Tolerance 1e-11: both sides round in 64 bits (1.1e-16) sums over 50 orbitals and 60 matrices, of overlaps
    whose condition is near one."""
    from paper_2505_18519_gb300 import build
    build.build()
    torch.cuda.empty_cache()
    got = {}
    for mode in ("free", "full"):
        f = str(tmp_path / (mode + ".npz"))
        r = subprocess.run([sys.executable, "-c", PROGRAM, ROOT, f, mode], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        got[mode] = np.load(f)
    for k in got["free"].files:
        a, b = got["free"][k], got["full"][k]
        assert np.all(np.isfinite(a)) and np.max(np.abs(a - b)) < 1e-11 * max(1.0, np.max(np.abs(a)))
    assert any(not np.array_equal(got["free"][k], got["full"][k]) for k in got["free"].files)   # two kernels
