"""What a context asks for as workspace (host only)."""

import pytest

from paper_2505_18519_gb300 import afqmc as lib


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2505_18519_gb300 import build
    build.build()
    lib.load_library()


def test_no_digits_beside_a_cache_that_is_read():
    """5 orbitals with rcache = 1 read the cache: (n_chol + 1) N n_up doubles per pair, and in return no work
    space of the digit products (some 4 kB a pair here); 6 run the digits."""
    def config(**kw):
        return lib.make_config(5, 4, 4, 32, 8, 64, 16, 0.005, 1, **kw)
    assert lib.fp64_digits(config()) and not lib.fp64_digits(config(rcache=True))
    cache = 33 * 5 * 4 * 8 * 64 * 16
    assert lib.workspace_bytes(config(rcache=True)) - lib.workspace_bytes(config()) < cache - (1 << 20)
    assert lib.fp64_digits(lib.make_config(6, 4, 4, 32, 8, 64, 16, 0.005, 1, rcache=True))
