"""Trial samples of the FP64 path whose Lanczos interval misses an eigenvalue of S:
the fixed-point series has to notice that its vectors outgrow their units and start
again, before a value that no longer fits is cut off."""

import numpy as np
import pytest

import afqmc_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2505_18519_gb300 import afqmc as lib  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2505_18519_gb300 import build
    build.build()
    lib.load_library()


def _lanczos_interval(S, steps=12):
    """The kernel's estimate in FP32: Lanczos from 1 + 0.5 sin(1.3 i + 0.7), Gershgorin's disks of the
    tridiagonal matrix, widened by 2 %."""
    f = np.float32
    S = S.astype(f)
    N = S.shape[0]
    v = (f(1) + f(0.5) * np.sin(f(1.3) * np.arange(N, dtype=f) + f(0.7))).astype(f)
    v /= np.linalg.norm(v)
    old, beta, a, b = np.zeros(N, f), f(0), [], []
    for _ in range(min(steps, N)):
        w = S @ v
        alpha = w @ v
        w = w - alpha * v - beta * old
        beta = np.linalg.norm(w)
        a.append(alpha)
        b.append(beta)
        if not beta > 1e-6 * abs(alpha):
            break
        old, v = v, w / beta
    r = [abs(b[j - 1]) * (j > 0) + abs(b[j]) for j in range(len(a))]
    lo, hi = min(x - y for x, y in zip(a, r)), max(x + y for x, y in zip(a, r))
    m = 0.02 * (hi - lo) + 1e-6
    return lo - m, hi + m


@pytest.mark.parametrize("rho,amp", [(0.002, 0.02), (0.002, 0.1), (0.01, 0.02), (0.01, 0.1), (0.1, 0.3)])
def test_growth_beyond_the_units_is_noticed(rho, amp):
    """S = 1 +- rho on two sets of orbitals, but for one vector of two orbitals (of nearly equal weight) whose
    eigenvalue lies 1.2 to 5.9 half-widths from the middle of the estimated interval.  The start vector lies in the span of
    two eigenvectors (the sets), so Lanczos stops after two steps, and the outlying vector is orthogonal to it.
    In some 6 to 10 terms its amplitude passes every multiple of the units somewhere in the range.

    Tolerance: 1e-13 e^||S|| times the norm of Phi0, as for every trial sample of the FP64 path."""
    N, n, K, i, j = 40, 1 << 16, 2, 3, 32
    low = (np.arange(N) < 10) | (np.arange(N) >= 30)
    half = np.where(low, -rho, rho)
    s = 1.0 + 0.5 * np.sin(1.3 * np.arange(N) + 0.7)
    e = np.zeros(N)
    e[i], e[j] = np.array([s[j], -s[i]]) / np.hypot(s[i], s[j])
    base, out = np.eye(N) + np.diag(half), np.outer(e, e)
    lo, hi = _lanczos_interval(base + 3.0 * rho * out)
    mid, wide = 0.5 * (lo + hi), 0.5 * (hi - lo)
    U = np.stack([base, out])
    x = np.ones((n, K))
    x[:, 1] = mid + wide * np.linspace(1.2, 5.9, n) - (1.0 - rho)         # base has the eigenvalue 1 - rho on e
    for q in (0, n // 2, n - 1):                          # the estimate misses the eigenvalue
        assert _lanczos_interval(U[0] + x[q, 1] * U[1])[1] < 1.0 - rho + x[q, 1] - 0.15 * wide
    sys = ai.make_system(ai.SystemSpec(N, 1, 0, 4, K, True, 5))
    rest = np.random.default_rng(3).standard_normal(N)
    rest -= e * (e @ rest)
    rest *= np.sqrt(0.79 ** 2 - amp ** 2) / np.linalg.norm(rest)          # the column's norm: 0.79 of its unit
    P0 = rest + amp * e
    ctx = lib.Context(lib.make_config(N, 1, 0, 4, K, n, 1, 0.005, 3, n_burn=0), sys.h, sys.L, P0[:, None], U)
    got = ctx.trial_orbitals(x)[:, :, 0]
    ctx.close()
    grow = np.exp(1.0 - rho + x[:, 1])[:, None]
    want = np.exp(1.0 + half) * rest + grow * amp * e
    assert np.all(np.abs(got - want) < 1e-13 * grow * np.linalg.norm(P0))
