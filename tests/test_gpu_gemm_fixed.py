"""S = sum_k x_k U_k of the FP64 path in fixed point, through trial samples exp(S) Phi0
of small S, against the exponential's Taylor series in 64 bits.

Tolerance: 2^-43 on values of order one.  Both sides round at some 2^-50 of them; S, with
entries up to some 1e-2, is checked to about 1e-11 of itself, where a wrong tile, fold or exponent
shows in full.
"""

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


@pytest.mark.parametrize("N,K,n", [
    (10, 1, 9800),        # one term; 154 row tiles of two column tiles, the last ones ragged
    (10, 65, 4900),       # one term past the fold of the cross sums
    (33, 200, 530),       # several folds, odd sizes
    (8, 700, 9729),       # one column tile, many terms
    (8, 7, 640),          # too few tiles: the FP64 kernel
])
def test_fixed_point_s_matches_64_bits(N, K, n):
    s = ai.make_system(ai.SystemSpec(N, 1, 0, 4, K, True, 60 + N))
    rng = np.random.default_rng(N + K)
    U = rng.standard_normal((K, N, N)) * 10.0 ** rng.uniform(-3, 0, (K, 1, 1))
    U = 1e-3 / np.sqrt(K) * (U + U.transpose(0, 2, 1))
    ctx = lib.Context(lib.make_config(N, 1, 0, 4, K, n, 1, 0.005, 3, n_burn=0), s.h, s.L, s.Phi0, U)
    x = rng.standard_normal((n, K))
    x[n // 2] = 0.0
    x[n // 3] *= 1e-6
    got = ctx.trial_orbitals(x)[:, :, 0]
    ctx.close()
    S = np.tensordot(x, U, axes=(1, 0))
    V = np.ascontiguousarray(s.Phi0[:, 0])
    want, term = np.tile(V, (n, 1)), np.tile(V, (n, 1))
    for k in range(1, 9):
        term = np.einsum("pij,pj->pi", S, term) / k
        want = want + term
    assert np.max(np.abs(got - want)) < 2.0 ** -43
