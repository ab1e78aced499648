"""Trial samples of the FP64 path (the Chebyshev series in fixed point) against the
matrix exponential of PyTorch in 64 bits, over the sizes where the kernel's split
changes and over inputs at and beyond the limits of its units.

Tolerance: 1e-13 e^||S|| times the largest norm of a column of Phi0 (its own column's
where they differ).  Both sides round at 2^-53 of terms that sum to e^||S||, some
thirty of them here and the squarings of the reference, whose condition is the same.
"""

import numpy as np
import pytest

import afqmc_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2505_18519_gb300 import afqmc as lib  # noqa: E402

TOL = 1e-13


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2505_18519_gb300 import build
    build.build()
    lib.load_library()


def _check(N, nu, K, scale, seed, Phi0=None, U=None, n=6):
    s = ai.make_system(ai.SystemSpec(N, nu, nu, 4, K, True, seed))
    U = s.U if U is None else U
    Phi0 = s.Phi0 if Phi0 is None else Phi0
    ctx = lib.Context(lib.make_config(N, nu, nu, 4, K, n, 1, 0.005, 3, n_burn=0), s.h, s.L, s.Phi0, s.U)
    ctx.close()
    ctx = lib.Context(lib.make_config(N, nu, nu, 4, K, n, 1, 0.005, 3, n_burn=0), s.h, s.L, Phi0, U)
    x = scale * np.random.default_rng(seed).standard_normal((n, K))
    x[0] = 0.0                                             # S = 0
    got = ctx.trial_orbitals(x)
    ctx.close()
    S = np.tensordot(x, U, axes=(1, 0))
    want = (torch.linalg.matrix_exp(torch.from_numpy(S)) @ torch.from_numpy(np.ascontiguousarray(Phi0))).numpy()
    size = np.exp(np.linalg.norm(S, 2, axis=(1, 2)))[:, None, None] * np.linalg.norm(Phi0, axis=0)
    assert np.all(np.abs(got - want) <= TOL * size)


@pytest.mark.parametrize("N,nu", [
    (1, 1), (2, 1), (8, 4), (13, 7),
    (50, 10),                       # four problems or more to an SM
    (64, 33), (41, 37),             # columns past n_up in the last group of a thread's columns
    (96, 8), (100, 20),             # two problems
    (120, 24), (150, 5),            # one
    (157, 1),                       # the largest whose S fits shared memory
])
def test_fixed_point_series_matches_the_exponential(N, nu):
    _check(N, nu, 5, 1.0, 900 + N)


@pytest.mark.parametrize("scale", [1e-9, 4.0, 30.0])
def test_fixed_point_series_over_the_range_of_s(scale):
    _check(24, 5, 4, scale, 77)


def test_columns_of_any_size_keep_their_digits():
    """Columns of Phi0 from 1e-12 to 1e12, and one beyond the units (its
    problems take the FP64 recurrence)."""
    rng = np.random.default_rng(8)
    Phi0 = np.linalg.qr(rng.standard_normal((30, 6)))[0] * np.array([1.0, 1e-12, 1e12, 1e-8, 3.0, 1e-5])
    _check(30, 6, 4, 1.0, 78, Phi0=Phi0)
    Phi0[:, 3] *= 1e-32
    _check(30, 6, 4, 1.0, 78, Phi0=Phi0)


def test_an_interval_that_misses_the_spectrum_is_done_again():
    """S of two blocks, the second far outside the first and hardly in the Lanczos
    start vector's reach after few steps."""
    N, nu = 48, 6
    rng = np.random.default_rng(9)
    U = np.zeros((2, N, N))
    a = 0.05 * rng.standard_normal((2, N, N))
    U += a + a.transpose(0, 2, 1)
    U[:, N - 1, :] = U[:, :, N - 1] = 0.0
    U[0, N - 1, N - 1] = 3.0
    U[1, N - 1, N - 1] = -2.0
    _check(N, nu, 2, 1.0, 79, U=U)
