"""The FP64 contraction as integer digit products against 64-bit values computed
here from their definition (Theta = phi (Phi^T phi)^-1, M_g = Phi^T X_g Theta), over
the sizes where its tiles and digits change and over walkers whose columns differ
in norm (Theta does not depend on the scale of a column of phi)."""

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


def _noalloc(h, L, Phi, phi, P, n_up):
    """Values of the pairs: Phi (pairs, N, n_up), phi (walkers, N, n_up + n_dn)."""
    dev = torch.device("cuda")
    pairs, N, _ = Phi.shape
    G, nt = L.shape[0], phi.shape[2]
    args = [torch.from_numpy(np.ascontiguousarray(a)).to(dev)
            for a in (h, L, Phi, np.ascontiguousarray(phi.astype(np.complex128)).view(np.float64))]
    out = [torch.empty(2 * k, dtype=torch.float64, device=dev) for k in (pairs, pairs, pairs * G)]
    lib.local_energy_noalloc(N, n_up, nt - n_up, G, pairs, P, *args, *out)
    logov, e, v = [o.cpu().numpy().view(np.complex128) for o in out]
    return logov, e, v.reshape(pairs, G)


def _values(h, L, Phi, phi, P, n_up):
    """The same from the definition, with the scale of every column of phi taken out first
    (powers of two: exact), and what the sums of the local energy add up to in absolute value."""
    nt = phi.shape[2]
    phi = phi / np.exp2(np.round(np.log2(np.linalg.norm(phi, axis=1, keepdims=True))))
    X = np.concatenate([h[None], L])
    e, v, size = [], [], []
    for p, F in enumerate(Phi):
        tr, ex, mag = 0.0, 0.0, 0.0
        for a, b in ((0, n_up), (n_up, nt)):
            if a == b:
                continue
            ph, f = phi[p // P][:, a:b], F[:, :b - a]
            M = f.T @ (X @ (ph @ np.linalg.inv(f.T @ ph)))
            t = np.trace(M, axis1=1, axis2=2)
            x = (M * M.transpose(0, 2, 1)).sum((1, 2))
            tr, ex, mag = tr + t, ex + x, mag + (np.abs(M) ** 2).sum((1, 2))
        v.append(tr[1:])
        e.append(tr[0] + 0.5 * (tr[1:] ** 2 - ex[1:]).sum())
        size.append(abs(tr[0]) + 0.5 * (np.abs(tr[1:]) ** 2 + mag[1:]).sum())
    return np.array(e), np.array(v), np.array(size)


def _orthonormal(rng, W, N, n):
    a = rng.standard_normal((W, N, n)) + 0.3j * rng.standard_normal((W, N, n))
    return np.linalg.qr(a)[0]


def _pairs_near(rng, phi, P, N, n_up):
    """Real trial orbitals near their walkers', so that the overlap matrices are well conditioned."""
    W = phi.shape[0]
    up = np.repeat(phi[:, :, :n_up].real, P, axis=0)
    return up + 0.15 / np.sqrt(N) * rng.standard_normal((W * P, N, n_up))


def _system(rng, N, G):
    a = 0.1 * rng.standard_normal((G + 1, N, N))
    X = a + a.transpose(0, 2, 1)
    return X[0] - np.diag(2.0 * rng.random(N)), X[1:]


SIZES = [
    (4, 1, 1, 70, 3, 65),        # 64 pairs to a row tile and one more; many matrices to a column tile
    (33, 11, 2, 9, 5, 1),        # a single path
    (50, 10, 10, 25, 3, 13),     # ragged last tiles of pairs and of matrices
    (64, 21, 20, 7, 2, 4),       # the last size of 8-bit digits
    (65, 22, 3, 7, 2, 4),        # the first of 7-bit digits
    (90, 33, 16, 6, 2, 3),       # one pair to a row tile
    (72, 48, 40, 4, 2, 2),       # the widest column tiles of 7-bit digits
    (224, 9, 1, 5, 2, 3),        # the largest size of the digits
]


def _check(N, nu, nd, G, W, P, scale, seed):
    """Tolerance 1e-13 of the sums of absolute values: both sides round at 2^-53 (the reference at
    every sum and in the inverse, whose condition is below 1e2 here)."""
    rng = np.random.default_rng(seed)
    h, L = _system(rng, N, G)
    phi = np.concatenate([_orthonormal(rng, W, N, nu)] + ([_orthonormal(rng, W, N, nd)] if nd else []), axis=2)
    if nd:
        phi[:, :, nu:] = 0.97 * phi[:, :, :nd] + 0.03 * phi[:, :, nu:]     # near the same trial orbitals
    Phi = _pairs_near(rng, phi, P, N, nu)
    for spin in (phi[:, :, :nu], phi[:, :, nu:]):
        n = spin.shape[2]
        if n:
            cond = np.linalg.cond(Phi[:, :, :n].transpose(0, 2, 1) @ np.repeat(spin, P, axis=0))
            assert np.max(cond) < 1e2
    assert N * G > 128                                                    # the digit products run
    phi = phi * scale(rng, phi.shape[2])[None, None, :]
    _, e, v = _noalloc(h, L, Phi, phi, P, nu)
    we, wv, size = _values(h, L, Phi, phi, P, nu)
    assert np.max(np.abs(e - we) / size) < 1e-13
    assert np.max(np.abs(v - wv)) < 1e-13 * max(1.0, np.max(np.abs(wv)))


@pytest.mark.parametrize("N,nu,nd,G,W,P", SIZES)
def test_digit_contraction_has_64_bit_accuracy(N, nu, nd, G, W, P):
    _check(N, nu, nd, G, W, P, lambda rng, n: np.ones(n), 100 + N)


@pytest.mark.parametrize("N,nu,nd,G,W,P", SIZES)
def test_columns_of_unequal_norm_keep_the_accuracy(N, nu, nd, G, W, P):
    """Norms from 1e-6 to 1 (and, in turn, one column far beyond), not powers of two."""
    _check(N, nu, nd, G, W, P, lambda rng, n: 10.0 ** -rng.uniform(0, 6, n), 200 + N)
    _check(N, nu, nd, G, W, P, lambda rng, n: np.where(np.arange(n) == n - 1, 3e-40, 1.0), 300 + N)


def test_context_of_unequal_columns_keeps_the_accuracy():
    """The same through a loaded state and the FP64 measurement."""
    N, nu, nd, G, W, P, K = 20, 5, 4, 30, 3, 6, 3
    rng = np.random.default_rng(9)
    s = ai.make_system(ai.SystemSpec(N, nu, nd, G, K, True, 77))
    phi = np.concatenate([_orthonormal(rng, W, N, nu), np.zeros((W, N, nd))], axis=2)
    phi[:, :, nu:] = phi[:, :, :nd]
    Phi = _pairs_near(rng, phi, P, N, nu)
    phi = phi * 10.0 ** -rng.uniform(0, 6, nu + nd)
    cfg = lib.make_config(N, nu, nd, G, K, W, P, 0.005, 3, n_burn=0)
    assert lib.fp64_digits(cfg)
    ctx = lib.Context(cfg, s.h, s.L, s.Phi0, s.U)
    ctx.load_state_arrays(dict(step=0, phi_up=phi[:, :, :nu], phi_dn=phi[:, :, nu:], weight=np.ones(W),
                               x=np.zeros((W, P, K)), Phi=Phi.reshape(W, P, N, nu)))
    ctx.energy()
    e = ctx.observables()["e_local"].reshape(-1)
    ctx.close()
    we, _, size = _values(s.h, s.L, Phi, phi, P, nu)
    assert np.max(np.abs(e - we) / size) < 1e-13


def test_trace_of_z_at_the_ends_of_its_low_half():
    """v_g = 2^-k (1 - 2^-28) for k = 0 .. 39, from one electron whose Phi^T L_g Theta is that one number:
    at one of the k the integer Z' is just below an odd multiple of 2^31, where its low half, rounding
    included, is at the end of 32 bits.  32 equal entries of Phi make the low half as wide as it gets.

    Every operand is a power of two but the number itself (28 bits), so v_g is exact to the units of Z'
    (2^-58 of the largest |L_g| entry)."""
    N, G = 40, 40
    Phi = np.zeros((1, N, 1))
    Phi[0, :32, 0] = 1.0
    phi = Phi.astype(np.complex128)
    h, L = np.zeros((N, N)), np.zeros((G, N, N))
    want = (1.0 - 2.0 ** -28) * 0.5 ** np.arange(G)
    L[:, 0, 0], L[:, 1, 1] = 32.0, -32.0                                  # cancel, and set the units
    L[:, 2, 2] = 32.0 * want
    _, _, v = _noalloc(h, L, Phi, phi, 1, 1)
    assert np.max(np.abs(v[0].real - want)) < 2.0 ** -50
    _, _, v = _noalloc(h, -L, Phi, phi, 1, 1)
    assert np.max(np.abs(v[0].real + want)) < 2.0 ** -50
    _, _, v = _noalloc(h, L, Phi, 1j * phi, 1, 1)                         # phi's phase cancels; the imaginary planes carry it
    assert np.max(np.abs(v[0].real - want)) < 2.0 ** -50
