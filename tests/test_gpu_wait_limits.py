"""The bounded waits of the FP64 digit kernels run out without a GPU fault: with a limit
of one poll the first wait on a copy or an MMA still in flight gives up, the block
sets bit 4 of the status word and returns, and the device stays usable."""

import numpy as np
import pytest

import afqmc_inputs as ai
from oracle import afqmc as oa

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2505_18519_gb300 import afqmc as lib  # noqa: E402

AFQMC_ERR_TIMEOUT = 6


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2505_18519_gb300 import build
    build.build()
    lib.load_library()


@pytest.mark.parametrize("spec", [
    ai.SystemSpec(50, 10, 10, 250, 50, True, 1001),      # 8-bit digits
    ai.SystemSpec(70, 14, 13, 90, 10, True, 81),         # 7-bit digits, streamed past Y
])
def test_digit_kernels_report_a_timeout(spec):
    s = ai.make_system(spec)
    W, P, dtau, seed = 3, 8, 0.005, 97
    def context(**kw):
        cfg = lib.make_config(spec.N, spec.n_up, spec.n_dn, spec.n_chol, spec.K, W, P, dtau, seed, n_burn=1, **kw)
        assert lib.fp64_digits(cfg)
        return lib.Context(cfg, s.h, s.L, s.Phi0, s.U)
    ctx = context(wait_polls=1)
    with pytest.raises(lib.AfqmcError) as ei:
        ctx.energy()
    assert ei.value.status == AFQMC_ERR_TIMEOUT
    ctx.close()
    torch.cuda.synchronize()                             # the device is still usable
    ctx = context()
    ham = oa.prepare(s.h, s.L, s.Phi0, s.U, spec.n_up, spec.n_dn, dtau)
    ost = oa.init(ham, oa.OracleConfig(dtau=dtau, n_walkers=W, n_paths=P, seed=seed, n_burn=1))
    e = ctx.energy(walkers=True)
    ctx.close()
    assert np.max(np.abs(e["e_walker"] - oa.measure(ham, ost)["e_bar"])) < 1e-9


def test_entry_without_allocation_gives_nan_after_a_timeout():
    """... and not what an earlier call left in its work space; the next call has values again."""
    N, nu, nd, G, P, n = 50, 10, 9, 60, 8, 20
    rng = np.random.default_rng(4)
    dev = torch.device("cuda")
    s = ai.make_system(ai.SystemSpec(N, nu, nd, G, 3, True, 11))
    Phi = np.linalg.qr(rng.standard_normal((n, N, nu)))[0]
    phi = np.concatenate([Phi[::P], Phi[::P][:, :, :nd]], axis=2) + 0.05j * rng.standard_normal((3, N, nu + nd))
    args = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (s.h, s.L, Phi, phi.view(np.float64))]
    def values():
        out = [torch.zeros(2 * k, dtype=torch.float64, device=dev) for k in (n, n, n * G)]
        lib.local_energy_noalloc(N, nu, nd, G, n, P, *args, *out)
        return [o.cpu().numpy() for o in out]
    want = values()
    assert all(np.all(np.isfinite(o)) for o in want)
    lib.noalloc_wait_polls(1)
    try:
        got = values()
    finally:
        lib.noalloc_wait_polls(0)
    assert all(np.all(np.isnan(o)) for o in got)
    assert all(np.array_equal(a, b) for a, b in zip(values(), want))
    with pytest.raises(lib.AfqmcError):
        lib.noalloc_wait_polls(-1)
