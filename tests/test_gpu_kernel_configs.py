"""Which kernel geometry a call runs: what the context has set, copied from one
context to another as it is, and the choice by call size where nothing is."""
import pytest

pytestmark = pytest.mark.gpu

NBITS, K = 2048, 2
SIZES = (1, 40, 403, 2056, 4113, 12000)


@pytest.fixture
def pair():
    import paper_2111_11924_gb300 as P

    a, b = P.Context(0), P.Context(0)
    ks = a.keygen(K, NBITS, 65537, 51)
    yield P, a, b, ks
    ks.free()
    a.close()
    b.close()


def _configs(ctx, ks):
    return [ctx.get_call_config(ks, crt, n) for crt in (False, True) for n in SIZES]


def test_call_config_follows_the_size_unless_set(pair):
    P, a, _, ks = pair
    by_size = _configs(a, ks)
    assert by_size[0][0] > by_size[5][0] and by_size[6][0] > by_size[11][0]  # more lanes for few chunks
    a.set_kernel_config(32, True, 4, 1)
    a.set_kernel_window(32, True, 4)
    assert [a.get_call_config(ks, True, n) for n in SIZES] == [(4, 1, 4)] * len(SIZES)
    a.set_kernel_config(32, True, 0)
    a.set_kernel_window(32, True, 0)
    assert _configs(a, ks) == by_size
    with pytest.raises(P.PMKError):
        a.get_call_config(ks, True, 0)


def test_copy_takes_a_geometry_equal_to_the_built_in_one(pair):
    """Tuned or set to the built-in throughput geometry is still set."""
    _, a, b, ks = pair
    for limbs, crt in ((64, False), (32, True)):
        a.set_kernel_config(limbs, crt, *a.get_kernel_config(limbs, crt))
    b.copy_kernel_configs_from(a, {NBITS: ks})
    assert _configs(b, ks) == _configs(a, ks)
    assert len(set(_configs(b, ks)[6:])) == 1


def test_copy_clears_what_the_source_has_not_set(pair):
    _, a, b, ks = pair
    by_size = _configs(a, ks)
    b.set_kernel_config(64, False, 16, 0)
    b.set_kernel_config(32, True, 8, 0)
    b.set_kernel_window(32, True, 4)
    b.copy_kernel_configs_from(a, {NBITS: ks})
    assert _configs(b, ks) == by_size
    b.set_kernel_config(32, True, 16, 1)
    b.copy_kernel_configs_from(b, {NBITS: ks})  # itself: nothing changes
    assert b.get_call_config(ks, True, 12000) == (16, 1, 5)
