"""Host-buffer calls on messages long enough to go in pieces: the results are
those of the device calls, whatever the piece boundaries fall on."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pinned(shape, dtype):
    import torch

    return torch.zeros(shape, dtype=dtype).pin_memory()


# 6 MiB of message a piece, 8 pieces at most: one piece, two, and eight, with key counts that do and do not divide
# the piece starts, and last chunks of one byte, full and in between.
@pytest.mark.parametrize("nbits,K,size", [(1024, 3, (12 << 20) - 1), (1024, 3, 12 << 20), (1024, 16, 13_000_001),
                                          (2048, 7, 255 * 60_000), (512, 5, 63 * 900_000 + 1)])
def test_pieces_equal_the_device_calls(nbits, K, size):
    import torch

    import paper_2111_11924_gb300 as P

    ctx = P.Context(0)
    ks = ctx.keygen(K, nbits, 65537, 31)
    msg = torch.from_numpy(np.random.default_rng(size).integers(0, 256, size, dtype=np.uint8)).pin_memory()
    n = P.num_chunks(size, nbits)
    want = ctx.encrypt_chunks(ks, ctx.split(nbits, msg.cuda())).cpu()
    cipher, back = _pinned((n, nbits // 32), torch.int32), _pinned(size, torch.uint8)
    stream = torch.cuda.Stream()
    for s in (None, stream):
        cipher.zero_()
        ctx.encrypt_message_host(ks, msg, cipher, stream=s)
        assert torch.equal(cipher, want)
        back.zero_()
        ctx.decrypt_message_host(ks, cipher, back, use_crt=True, stream=s)
        assert torch.equal(back, msg)
    ctx.close()


def test_overlapping_host_buffers_read_all_input_first():
    # The output begins half way through the input: written piece by piece it would reach input not yet read.
    import torch

    import paper_2111_11924_gb300 as P

    nbits, size = 1024, 48 << 20
    ctx = P.Context(0)
    ks = ctx.keygen(3, nbits, 65537, 33)
    msg = torch.from_numpy(np.random.default_rng(2).integers(0, 256, size, dtype=np.uint8))
    n = P.num_chunks(size, nbits)
    total = n * nbits // 8
    want = ctx.encrypt_chunks(ks, ctx.split(nbits, msg.cuda())).cpu()
    buf = _pinned(2 * total, torch.uint8)
    buf[:size] = msg
    off = size // 2 // 16 * 16
    cipher = buf[off:off + total].view(torch.int32).view(n, nbits // 32)
    ctx.encrypt_message_host(ks, buf[:size], cipher)
    assert torch.equal(cipher, want)
    cipher = buf[:total].view(torch.int32).view(n, nbits // 32)
    cipher.copy_(want)
    back = buf[total // 2:total // 2 + size]
    ctx.decrypt_message_host(ks, cipher, back, use_crt=True)
    assert torch.equal(back, msg)
    ctx.close()


@pytest.mark.parametrize("K", [1, 64, 2000])
def test_pieces_by_key_count_and_priority(K):
    # 128 chunks a key and piece at least (2,000 keys: one piece), and a stream of another priority.
    import torch

    import paper_2111_11924_gb300 as P

    nbits, size = 512, 25_000_003
    ctx = P.Context(0)
    ks = ctx.keygen(K, nbits, 65537, 34)
    msg = torch.from_numpy(np.random.default_rng(3).integers(0, 256, size, dtype=np.uint8)).pin_memory()
    n = P.num_chunks(size, nbits)
    want = ctx.encrypt_chunks(ks, ctx.split(nbits, msg.cuda())).cpu()
    for s in (None, torch.cuda.Stream(priority=-1)):
        cipher = _pinned((n, nbits // 32), torch.int32)
        ctx.encrypt_message_host(ks, msg, cipher, stream=s)
        assert torch.equal(cipher, want)
    ctx.close()


def test_errors_in_pieces(monkeypatch):
    import torch

    import paper_2111_11924_gb300 as P
    from paper_2111_11924_gb300 import pmkrsa

    nbits, size = 512, 20 << 20
    ctx = P.Context(0)
    ks = ctx.keygen(4, nbits, 65537, 32)
    msg = torch.from_numpy(np.random.default_rng(1).integers(0, 256, size, dtype=np.uint8)).pin_memory()
    n = P.num_chunks(size, nbits)
    cipher, back = _pinned((n, nbits // 32), torch.int32), _pinned(size, torch.uint8)
    ctx.encrypt_message_host(ks, msg, cipher)
    keep = cipher[n - 2].clone()
    cipher[n - 2] = -1  # not below its modulus, in the last piece
    for use_crt in (False, True):
        with pytest.raises(P.PMKError) as err:
            ctx.decrypt_message_host(ks, cipher, back, use_crt=use_crt)
        assert err.value.code == pmkrsa.PMK_ERANGE
    cipher[n - 2] = keep
    s = torch.cuda.Stream()
    monkeypatch.setenv("PMK_INJECT_FAULT", "after_copy")
    for call in (lambda: ctx.encrypt_message_host(ks, msg, cipher, stream=s),
                 lambda: ctx.decrypt_message_host(ks, cipher, back, use_crt=True, stream=s)):
        with pytest.raises(P.PMKError) as err:
            call()
        assert err.value.code == pmkrsa.PMK_ECUDA and s.query()
    monkeypatch.delenv("PMK_INJECT_FAULT")
    ctx.decrypt_message_host(ks, cipher, back, use_crt=True, stream=s)
    assert torch.equal(back, msg) and ctx.status() == pmkrsa.PMK_OK
    ctx.close()
