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


def test_tuned_geometry_serves_its_size_only(pair):
    P, a, b, ks = pair
    by_size = {(crt, n): a.get_call_config(ks, crt, n) for crt in (False, True) for n in SIZES}
    for mode, crt, cfg in (("decrypt", False, (16, 1, 5)), ("crt", True, (8, 0, 4))):
        a.set_tuned_config(ks, 4113, mode, *cfg)
        for n in SIZES:
            same = by_size[crt, n][0] == by_size[crt, 4113][0]
            assert a.get_call_config(ks, crt, n) == (cfg if same else by_size[crt, n]), (mode, n)
        assert a.get_call_config(ks, crt, 4113) == cfg and a.get_call_config(ks, crt, 40) == by_size[crt, 40]
    b.copy_kernel_configs_from(a, {NBITS: ks})
    assert _configs(b, ks) == _configs(a, ks)
    a.set_kernel_config(64, False, 16, 1)  # by hand: every size
    assert {a.get_call_config(ks, False, n) for n in SIZES} == {(16, 1, 5)}
    a.set_kernel_window(32, True, 0)
    assert {a.get_call_config(ks, True, n) for n in SIZES} == {(8, 0, 5)}
    for args in ((4113, "crt", 5, 0, 5), (4113, "crt", 4, 0, 3), (0, "crt", 4, 0, 5)):
        with pytest.raises(P.PMKError):
            a.set_tuned_config(ks, *args)


def test_autotune_and_its_cache_leave_other_sizes_alone(pair, tmp_path):
    import numpy as np
    import torch

    P, a, b, ks = pair
    other = [(crt, n) for crt in (False, True) for n in SIZES]
    by_size = [a.get_call_config(ks, *c) for c in other]
    cache = P.TuneCache(str(tmp_path / "tune.json"))
    for ctx, cached in ((a, False), (b, True)):
        for mode, crt in (("decrypt", False), ("crt", True)):
            res = ctx.autotune(ks, 4113, mode, reps=1, cache=cache)
            assert bool(res.get("cached")) == cached
            assert ctx.get_call_config(ks, crt, 4113) == (res["tpi"], res["form"], res["window"])
        assert [c[0] for c in map(lambda c: ctx.get_call_config(ks, *c), other[:3] + other[6:9])] == \
            [c[0] for c in by_size[:3] + by_size[6:9]]
    m = np.random.default_rng(3).integers(0, 1 << 32, (40, NBITS // 32), dtype=np.uint64).astype(np.uint32)
    m[:, -1] = 0
    m = torch.from_numpy(m.view(np.int32)).cuda()
    c = a.encrypt_chunks(ks, m)
    jobs = [(ks, c, torch.empty_like(c), op) for op in (P.pmkrsa.OP_DECRYPT, P.pmkrsa.OP_DECRYPT_CRT)]
    batch = a.batch(jobs)
    batch.launch()
    a.check()
    for crt, job in zip((False, True), jobs):
        assert torch.equal(a.decrypt_chunks(ks, c, use_crt=crt), m) and torch.equal(job[2], m)
