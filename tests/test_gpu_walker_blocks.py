"""Results that do not depend on how many rows, walkers or pairs a call holds: every
arithmetic is chosen by the sizes of the system, so that blocks of walkers (a sharded run), part
of a set of samples and part of a batch of pairs give the bits of the whole."""

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


def _blocks(spec, W, blocks, P, steps=2, **kw):
    s = ai.make_system(spec)
    def ctx(w, off):
        cfg = lib.make_config(spec.N, spec.n_up, spec.n_dn, spec.n_chol, spec.K, w, P, 0.005, 4321, n_burn=2,
                              walker_offset=off, **kw)
        return lib.Context(cfg, s.h, s.L, s.Phi0, s.U)
    cuts = np.cumsum([0] + blocks)
    assert cuts[-1] == W
    whole, parts = ctx(W, 0), [ctx(b, int(o)) for b, o in zip(blocks, cuts)]
    for c in [whole] + parts:
        c.step(steps)
        c.energy()
    a, b = whole.state_arrays(), [c.state_arrays() for c in parts]
    a["e_local"], refined = whole.observables()["e_local"], whole.stats()["refined_pairs"]
    for q, c in zip(b, parts):
        q["e_local"] = c.observables()["e_local"]
    for c in [whole] + parts:
        c.close()
    for key in ("phi_up", "phi_dn", "weight", "x", "Phi", "e_local"):
        assert np.array_equal(a[key], np.concatenate([q[key] for q in b])), key
    return refined


@pytest.mark.parametrize("spec,W,blocks,P,kw", [
    (ai.SystemSpec(50, 10, 10, 250, 50, True, 90), 128, [64, 64], 4, {}),             # field planes of 256 and 128 rows
    (ai.SystemSpec(50, 10, 10, 60, 50, True, 91), 40, [3, 37], 16, {}),               # S of 640, 48 and 592 rows
    (ai.SystemSpec(8, 4, 4, 32, 8, False, 92), 700, [1, 699], 16, {}),                # the smallest system
    (ai.SystemSpec(8, 2, 2, 32, 8, False, 93), 600, [10, 590], 16, dict(rcache=True)),  # ... with the cache allowed
    (ai.SystemSpec(5, 2, 2, 20, 5, False, 97), 900, [10, 890], 16, dict(rcache=True)),  # the cache read
])
def test_walker_blocks_of_the_fp64_path(spec, W, blocks, P, kw):
    _blocks(spec, W, blocks, P, **kw)


def test_walker_blocks_of_the_refined_mixed_path():
    """Refinement of every pair, of parts of them and of none: a refined pair's sum has one order,
    however many others are listed."""
    spec = ai.SystemSpec(70, 14, 13, 150, 10, True, 94)
    W, P = 24, 8
    counts = [_blocks(spec, W, [1, 5, 18], P, steps=1, precision="fp16x6", refine_tol=tol)
              for tol in [1e-300] + [10.0 ** (-0.15 * k) for k in range(42, 62)]]
    listed = 2 * W * P                                    # one measurement of the step and one after it
    assert counts[0] == listed and sum(0 < n < listed for n in counts) >= 3, counts


@pytest.mark.parametrize("N,K", [(50, 50), (8, 8), (24, 100)])
def test_part_of_the_samples(N, K):
    s = ai.make_system(ai.SystemSpec(N, 3, 2, 4, K, True, 95))
    x = np.random.default_rng(1).standard_normal((5000, K))
    ctx = lib.Context(lib.make_config(N, 3, 2, 4, K, 5000, 1, 0.005, 3, n_burn=0), s.h, s.L, s.Phi0, s.U)
    whole = ctx.trial_orbitals(x)
    for n in (1, 70, 1000):
        assert np.array_equal(ctx.trial_orbitals(x[:n]), whole[:n]), n
    ctx.close()


@pytest.mark.parametrize("N,nu,nd,G,P", [(8, 1, 1, 16, 16), (50, 10, 7, 40, 6), (20, 2, 2, 90, 24)])
def test_part_of_a_batch_of_pairs(N, nu, nd, G, P):
    rng = np.random.default_rng(2)
    W = 300 // P
    s = ai.make_system(ai.SystemSpec(N, nu, nd, G, 3, True, 96))
    phi = rng.standard_normal((W, N, nu + nd)) + 1j * rng.standard_normal((W, N, nu + nd))
    Phi = rng.standard_normal((W * P, N, nu))
    dev = torch.device("cuda")
    args = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (s.h, s.L, Phi, phi.view(np.float64))]
    def values(n):
        out = [torch.empty(2 * k, dtype=torch.float64, device=dev) for k in (n, n, n * G)]
        lib.local_energy_noalloc(N, nu, nd, G, n, P, *args, *out)
        return [o.cpu().numpy() for o in out]
    whole = values(W * P)
    for n in (1, P - 1, P, 2 * P + 1):
        for got, want in zip(values(n), whole):
            assert np.array_equal(got, want[:got.size]), n
