"""A host encryption that fails at a later piece: earlier pieces have kernels
and copies to the caller's buffer queued on other streams by then, and none of
them may be in flight when the call returns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NBITS, SIZE = 2048, 48 << 20  # eight pieces


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2111_11924_gb300 as P

    ctx = P.Context(0)
    ks = ctx.keygen(8, NBITS, 65537, 41)
    msg = torch.from_numpy(np.random.default_rng(4).integers(0, 256, SIZE, dtype=np.uint8)).pin_memory()
    n = P.num_chunks(SIZE, NBITS)
    cipher = torch.zeros((n, NBITS // 32), dtype=torch.int32).pin_memory()
    want = ctx.encrypt_chunks(ks, ctx.split(NBITS, msg.cuda())).cpu()
    yield P, ctx, ks, msg, cipher, want
    ctx.close()


@pytest.mark.parametrize("piece", (1, 2, 3, 5, 7))
def test_failure_at_a_later_piece_leaves_no_copy_in_flight(env, monkeypatch, piece):
    import torch

    P, ctx, ks, msg, cipher, want = env
    stream = torch.cuda.Stream()
    monkeypatch.setenv("PMK_INJECT_FAULT", f"after_copy:{piece}")
    with pytest.raises(P.PMKError) as err:
        ctx.encrypt_message_host(ks, msg, cipher, stream=stream)
    cipher.fill_(0x5A5A5A5A)  # at once: a copy still in flight would write over it
    assert err.value.code == P.pmkrsa.PMK_ECUDA and stream.query()
    torch.cuda.synchronize()
    assert bool((cipher == 0x5A5A5A5A).all())
    monkeypatch.delenv("PMK_INJECT_FAULT")
    ctx.encrypt_message_host(ks, msg, cipher, stream=stream)
    assert torch.equal(cipher, want)


def test_a_piece_past_the_last_is_not_reached(env, monkeypatch):
    import torch

    P, ctx, ks, msg, cipher, want = env
    monkeypatch.setenv("PMK_INJECT_FAULT", "after_copy:8")
    cipher.zero_()
    ctx.encrypt_message_host(ks, msg, cipher)
    assert torch.equal(cipher, want)


def test_pageable_output_goes_in_one_piece(env, monkeypatch):
    """A copy to pageable memory holds the call up, so pieces would run one
    after another; a pageable input does not matter."""
    import torch

    P, ctx, ks, msg, cipher, want = env
    monkeypatch.setenv("PMK_INJECT_FAULT", "after_copy:1")
    pageable = torch.zeros_like(want)
    assert not pageable.is_pinned()
    for src in (msg, msg.clone()):
        pageable.zero_()
        ctx.encrypt_message_host(ks, src, pageable)
        assert torch.equal(pageable, want)
        with pytest.raises(P.PMKError):
            ctx.encrypt_message_host(ks, src, cipher)
