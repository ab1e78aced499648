"""How far trial samples of the FP64 path are from exp(S) Phi0 in more than 64 bits
(numpy's long double): no further than the same Chebyshev series summed in FP64."""

import numpy as np
import pytest

import afqmc_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2505_18519_gb300 import afqmc as lib  # noqa: E402

WIDE = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2505_18519_gb300 import build
    build.build()
    lib.load_library()


def _taylor(S, Phi0):
    """exp(S) Phi0 in long double."""
    term = Phi0.astype(WIDE)
    want = term.copy()
    for k in range(1, 90):
        term = S @ term / WIDE(k)
        want = want + term
        if np.max(np.abs(term)) < 1e-23:
            break
    return want


def _chebyshev(S, Phi0):
    """The series on S's spectral interval in 64 bits, its coefficients from long double."""
    w = np.linalg.eigvalsh(S)
    c, rho = 0.5 * (w[0] + w[-1]), 0.505 * (w[-1] - w[0])
    ik = [WIDE(0), WIDE(1e-300)]                           # Miller's recurrence for I_k(rho), downwards
    for k in range(60, 0, -1):
        ik.append(ik[-2] + 2 * k / WIDE(rho) * ik[-1])
    ik = np.array(ik[:0:-1])
    coef = ik / (ik[0] + 2 * ik[1:].sum()) * np.exp(WIDE(c) + WIDE(rho))
    coef = np.concatenate([coef[:1], 2 * coef[1:]]).astype(float)
    t = (S - c * np.eye(len(S))) / rho

    def times(v):                                          # sums in the order of a kernel's loop
        out = np.zeros_like(v)
        for j in range(len(t)):
            out += t[:, j:j + 1] * v[j]
        return out

    old, v = Phi0, times(Phi0)
    out = coef[0] * old + coef[1] * v
    for a in coef[2:40]:
        old, v = v, 2 * times(v) - old
        out = out + a * v
    return out


@pytest.mark.parametrize("N,nu,K", [(24, 5, 24), (50, 10, 30), (120, 24, 20), (157, 1, 12)])
def test_trial_samples_round_like_fp64(N, nu, K):
    """Root mean square error over six random S of norm 2 to 3, relative to the result: at most 1.5 times that of
    the FP64 series.  Both round the interval's ends, t, the terms and the result in 64 bits or more; 1.5
    allows for the library's wider interval (estimated, not the spectrum) and the scatter of six samples."""
    s = ai.make_system(ai.SystemSpec(N, nu, nu, 4, K, True, 40 + N))
    rng = np.random.default_rng(N)
    n = 6
    x = rng.standard_normal((n, K)) * np.sqrt(50 / K)
    ctx = lib.Context(lib.make_config(N, nu, nu, 4, K, n, 1, 0.005, 3, n_burn=0), s.h, s.L, s.Phi0, s.U)
    got = ctx.trial_orbitals(x)
    ctx.close()
    S = np.tensordot(x.astype(WIDE), s.U.astype(WIDE), axes=(1, 0))
    ours = fp64 = size = 0.0
    for q in range(n):
        want = _taylor(S[q], s.Phi0)
        size += float((want ** 2).sum())
        ours += float(((got[q] - want) ** 2).sum())
        fp64 += float(((_chebyshev(np.tensordot(x[q], s.U, axes=(0, 0)), s.Phi0) - want) ** 2).sum())
    assert np.sqrt(ours) < 1.5 * np.sqrt(fp64), (np.sqrt(ours / size), np.sqrt(fp64 / size))
