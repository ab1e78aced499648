"""The FP64 contraction on the tensor cores (exact integer digit products)
against the general FP64 kernel of the entry point that allocates nothing, on the
same walker and path states, over the sizes where its tiles and digits change.

Tolerance: 1e-10 relative to the largest value.  Both sides round their sums in
64 bits (1.1e-16); a condition number of the overlap matrices up to 1e4 and the
growth of the sums (their terms' root, about 1e2) bound what they may differ by.
"""

import numpy as np
import pytest

import afqmc_inputs as ai

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2505_18519_gb300 import afqmc as lib  # noqa: E402

RTOL = 1e-10


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2505_18519_gb300 import build
    build.build()
    lib.load_library()


@pytest.mark.parametrize("N,nu,nd,G,W,P", [
    (1, 1, 0, 1, 1, 1),          # one orbital, one electron
    (4, 1, 1, 70, 3, 65),        # 64 pairs to a row tile and one more; many matrices to a column tile
    (8, 8, 8, 5, 2, 3),          # every orbital occupied
    (33, 11, 2, 9, 5, 1),        # a single path
    (50, 10, 10, 25, 3, 13),     # the medium molecule: ragged last tiles of pairs and of matrices
    (64, 21, 20, 7, 2, 4),       # the last size of 8-bit digits
    (65, 22, 3, 7, 2, 4),        # the first of 7-bit digits
    (90, 33, 16, 6, 2, 3),       # one pair to a row tile
    (72, 48, 40, 4, 2, 2),       # the widest column tiles of 7-bit digits
    (224, 9, 1, 5, 2, 3),        # the largest size of the digits
    (225, 3, 2, 5, 2, 9),        # beyond it: the general walker-side form
])
def test_digit_contraction_matches_the_general_form(N, nu, nd, G, W, P):
    s = ai.make_system(ai.SystemSpec(N, nu, nd, G, 3, True, 4000 + N))
    cfg = lib.make_config(N, nu, nd, G, 3, W, P, 0.005, 17, n_burn=1)
    ctx = lib.Context(cfg, s.h, s.L, s.Phi0, s.U)
    ctx.step(1)
    ctx.energy()
    got = ctx.observables()
    st = ctx.state_arrays()
    ctx.close()
    dev = torch.device("cuda")
    pairs = W * P
    phi = np.ascontiguousarray(np.concatenate([st["phi_up"], st["phi_dn"]], axis=2))
    args = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (s.h, s.L, st["Phi"], phi.view(np.float64))]
    out = [torch.empty(2 * k, dtype=torch.float64, device=dev) for k in (pairs, pairs, pairs * G)]
    lib.local_energy_noalloc(N, nu, nd, G, pairs, P, *args, *out)
    logov, e, v = [o.cpu().numpy().view(np.complex128) for o in out]
    e, v, S = e.reshape(W, P), v.reshape(W, P, G), np.exp(1j * logov.reshape(W, P).imag)
    assert np.max(np.abs(got["e_local"] - e)) < RTOL * max(1.0, np.max(np.abs(e)))
    sumS = S.sum(1)
    fb = (S[:, :, None] * v).sum(1) / sumS[:, None]
    grow = np.max(1.0 / np.abs(sumS)) * P                  # path signs that cancel magnify rounding
    assert np.max(np.abs(got["force_bias"] - fb)) < RTOL * grow * max(1.0, np.max(np.abs(v)))


@pytest.mark.parametrize("precision,N,nu,nd,G,W,P", [
    ("fp16x6", 140, 9, 7, 20, 5, 17),      # three row tiles of pairs a walker, walkers with few and with many
    ("fp16x3", 150, 24, 24, 12, 9, 6),     # two pairs to a row tile
    ("fp16x3", 129, 1, 0, 9, 70, 3),       # one spin, more walkers than a row tile of Y holds
    ("fp16x6", 200, 40, 33, 6, 4, 3),      # one pair to a row tile, the largest electron numbers
])
def test_refined_pairs_alone_are_replaced(precision, N, nu, nd, G, W, P):
    """Refinement at tolerances that list some pairs of some walkers: each pair's
    energy is the tensor cores' own, bit for bit, or that of the FP64 context, and
    the latter at least as often as the refinement counted.

    Tolerance of an FP64 energy: RTOL, as above."""
    s = ai.make_system(ai.SystemSpec(N, nu, nd, G, 3, True, 5000 + N))

    def energies(prec, tol, state, **kw):
        cfg = lib.make_config(N, nu, nd, G, 3, W, P, 0.005, 19, n_burn=2, precision=prec, refine_tol=tol, **kw)
        ctx = lib.Context(cfg, s.h, s.L, s.Phi0, s.U)
        ctx.load_state_arrays(state) if state is not None else ctx.step(1)
        ctx.energy()
        before = ctx.stats()["refined_pairs"]
        ctx.energy()                                       # the same state again: the same pairs
        out = ctx.observables()["e_local"], int(ctx.stats()["refined_pairs"] - before), ctx.state_arrays()
        ctx.close()
        return out

    e64, _, state = energies("fp64", 0.0, None)
    raw, none, _ = energies(precision, 0.0, state)
    assert none == 0
    counts = set()
    for tol in [1e-300] + [10.0 ** (-0.5 * k) for k in range(4, 25)]:
        e, n, _ = energies(precision, tol, state)
        changed = e != raw
        counts.add(n)
        assert np.count_nonzero(changed) <= n <= W * P
        assert np.count_nonzero(np.abs(e - e64) < RTOL * max(1.0, np.max(np.abs(e64)))) >= n
        assert np.all(np.abs(e - e64)[changed] < RTOL * max(1.0, np.max(np.abs(e64))))
    assert W * P in counts and len(counts) > 2             # some tolerance listed part of the pairs
