"""The work a user of this library has it do, as timed cases.

A case names an operation of the message path (split -> exponentiation -> join,
through the public binding), the message length, the key set (K keys of nbits
bits with `primes` primes each) and how the call is made.  Messages are uniform
random bytes, as in the paper's experiments; the sizes are those of its tables
(100 KB plaintexts, 1 - 100 MB files) and of this repository's workloads.
Keys are what a program generates once and keeps, so they depend on the key
set's shape only; messages and blinding values depend on the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2111_11924_gb300 as P
from paper_2111_11924_gb300 import pmkrsa

E = 65537
KEY_SEED = 0x50444D4B00000700

# Operations:
#   encrypt        split, then c = m^e mod N
#   decrypt        m = c^d mod N with the full exponent, then join
#   crt            the same through the residues mod the primes
#   blind_encrypt  split, then (C*, C_R) of Algorithm 1 with the random matrix R
#   blind_decrypt  Algorithm 1 decryption in CRT form, then join
#   batch          a planned batch of messages of mixed widths and operations
# Options: "idx" binds chunks to keys by an explicit random index vector
# (serving coalesced requests does) instead of t mod K; "host" takes pinned
# host buffers through the whole call.


def _case(op, msg_bytes, nbits, K, primes=2, idx=False, host=False):
    return {"op": op, "msg_bytes": msg_bytes, "nbits": nbits, "K": K, "primes": primes, "idx": idx, "host": host}


def listed():
    def named(name, **kw):
        return {"name": name} | _case(**kw)

    return [
        # A short record with one pair of keys: five chunks, all launch latency.
        named("encrypt_1KiB_2048", op="encrypt", msg_bytes=1024, nbits=2048, K=2),
        # The small workload: 32 KiB under 1024-bit keys, decrypted with the full d.
        named("decrypt_32KiB_1024", op="decrypt", msg_bytes=32 << 10, nbits=1024, K=4),
        # The paper's Table 2 plaintext, full d: too few chunks to fill the GPU.
        named("decrypt_100KB_2048", op="decrypt", msg_bytes=102400, nbits=2048, K=16),
        # The headline: 1 MiB, 8 keys of 2048 bits, full d.
        named("decrypt_1MiB_2048", op="decrypt", msg_bytes=1 << 20, nbits=2048, K=8),
        # A file that fills the GPU several times over, full d.
        named("decrypt_10MiB_2048", op="decrypt", msg_bytes=10 << 20, nbits=2048, K=16),
        # The headline message decrypted the way a deployment does it, by CRT.
        named("crt_1MiB_2048", op="crt", msg_bytes=1 << 20, nbits=2048, K=8),
        # Table 3's 25 MB file by CRT, from pinned host buffers and back.
        named("crt_25MB_2048_host", op="crt", msg_bytes=25_000_000, nbits=2048, K=16, host=True),
        # Table 2's plaintext under 4096-bit keys by CRT: few, long exponentiations.
        named("crt_100KB_4096", op="crt", msg_bytes=102400, nbits=4096, K=4),
        # Coalesced serving requests of 3072-bit keys, chunks bound by key index.
        named("crt_256KiB_3072_idx", op="crt", msg_bytes=256 << 10, nbits=3072, K=8, idx=True),
        # The largest file of Table 3, encrypted.
        named("encrypt_100MiB_2048", op="encrypt", msg_bytes=100 << 20, nbits=2048, K=16),
        # Algorithm 1 proper: blinded decryption of the headline message.
        named("blind_decrypt_1MiB_2048", op="blind_decrypt", msg_bytes=1 << 20, nbits=2048, K=8),
        # Messages of 1024 - 3072 bits, mostly decryptions, in one planned batch.
        named("batch_24_mixed", op="batch", msg_bytes=600_000, nbits=0, K=0),
    ]


# Multiply-adds of the costliest listed case: no drawn one takes more.
_MAX_MACS = 6.4e11
_KEY_COUNTS = {1024: (2, 4, 8, 16), 2048: (2, 4, 8, 16), 3072: (2, 4, 8), 4096: (2, 4)}


def draw(rng):
    """One more case: any operation, width and option, sizes log-uniform from
    one chunk to the largest file of that operation."""
    op = rng.choice(("encrypt", "decrypt", "decrypt", "crt", "crt", "blind_encrypt", "blind_decrypt", "batch"))
    if op == "batch":
        return _case("batch", int(math.exp(rng.uniform(math.log(1e5), math.log(1.5e6)))), 0, 0)
    nbits = rng.choice((1024, 2048, 2048, 3072, 4096))
    primes = 4 if nbits == 4096 and rng.random() < 0.5 else 2
    case = _case(op, 0, nbits, rng.choice(_KEY_COUNTS[nbits]), primes)
    plain = op in ("encrypt", "decrypt", "crt")
    case["idx"] = plain and rng.random() < 0.3
    case["host"] = plain and not case["idx"] and rng.random() < 0.3
    per_byte = _macs_per_chunk(case) / (nbits // 8 - 1)
    top = min(100 << 20, _MAX_MACS / per_byte)
    case["msg_bytes"] = int(math.exp(rng.uniform(math.log(200), math.log(top))))
    return case


# ------------------------------------------------------------------ inputs


@functools.lru_cache(maxsize=None)
def _context():
    return P.Context(0)


@functools.lru_cache(maxsize=None)
def _keys(K, nbits, primes):
    return _context().keygen(K, nbits, E, KEY_SEED + nbits + primes, nprimes=primes)


@functools.lru_cache(maxsize=None)
def _moduli(K, nbits, primes):
    return [int.from_bytes(row.tobytes(), "little") for row in _keys(K, nbits, primes).export()["N"]]


def _chunks(case):
    return -(-case["msg_bytes"] // (case["nbits"] // 8 - 1))


def _message(case, seed):
    return np.random.default_rng([seed, 1]).integers(0, 256, case["msg_bytes"], dtype=np.uint8)


def _blinding(case, seed):
    """R of Algorithm 1: one value per chunk, below 2^(nbits - 8)."""
    raw = np.zeros((_chunks(case), case["nbits"] // 8), np.uint8)
    raw[:, :-1] = np.random.default_rng([seed, 2]).integers(0, 256, (raw.shape[0], raw.shape[1] - 1), dtype=np.uint8)
    return raw


def _index(case, seed):
    return np.random.default_rng([seed, 3]).integers(0, case["K"], _chunks(case), dtype=np.int32)


def _batch_jobs(case, seed):
    """24 messages whose lengths sum to about msg_bytes, log-uniform over a
    factor of 64, each with its own width, key count and operation."""
    rng = np.random.default_rng(case["msg_bytes"])  # the mix belongs to the case, the bytes to the seed
    share = np.exp(rng.uniform(0, math.log(64), 24))
    share *= case["msg_bytes"] / share.sum()
    jobs = []
    for i in range(24):
        op = str(rng.choice(("encrypt", "decrypt", "crt"), p=(0.2, 0.3, 0.5)))
        nbits = int(rng.choice((1024, 2048, 3072)))
        K = int(rng.choice((2, 4, 8)))
        jobs.append((_case(op, max(64, int(share[i])), nbits, K), seed * 64 + i))
    return jobs


def _device_message(case, seed):
    return torch.from_numpy(_message(case, seed)).cuda()


def _device_limbs(raw):
    return torch.from_numpy(raw.view(np.int32)).cuda()


def _prepare_one(case, seed):
    """The call's inputs and outputs: a message to encrypt, or ciphertext to decrypt."""
    ctx = _context()
    ks = _keys(case["K"], case["nbits"], case["primes"])
    st = {"case": case, "ctx": ctx, "ks": ks, "msg": _device_message(case, seed), "idx": None}
    if case["idx"]:
        st["idx"] = torch.from_numpy(_index(case, seed)).cuda()
    if case["op"] == "encrypt" and not case["host"]:
        return st
    m = ctx.split(case["nbits"], st["msg"])
    if case["op"].startswith("blind"):
        rnd = _device_limbs(_blinding(case, seed))
        if case["op"] == "blind_encrypt":
            st["rnd"] = rnd
        else:
            st["cstar"], st["cr"] = ctx.encrypt_blinded(ks, m, rnd)
    else:
        st["cipher"] = ctx.encrypt_chunks(ks, m, key_idx=st["idx"])
    if case["host"]:
        st["h_msg"] = torch.from_numpy(_message(case, seed)).pin_memory()
        st["h_cipher"] = st.pop("cipher").cpu().pin_memory()
        if case["op"] == "encrypt":
            st["h_cipher"].zero_()
        else:
            st["h_msg"].zero_()
    if case["op"] not in ("encrypt", "blind_encrypt"):
        del st["msg"]
    return st


def prepare(case, seed):
    if case["op"] != "batch":
        st = _prepare_one(case, seed)
        torch.cuda.synchronize()
        return st
    ctx = _context()
    jobs, outs = [], []
    ops = {"encrypt": pmkrsa.OP_ENCRYPT, "decrypt": pmkrsa.OP_DECRYPT, "crt": pmkrsa.OP_DECRYPT_CRT}
    for sub, sub_seed in _batch_jobs(case, seed):
        one = _prepare_one(sub, sub_seed)
        src = ctx.split(sub["nbits"], one["msg"]) if sub["op"] == "encrypt" else one["cipher"]
        out = torch.empty_like(src)
        jobs.append((one["ks"], src, out, ops[sub["op"]]))
        outs.append(out)
    torch.cuda.synchronize()
    return {"case": case, "batch": ctx.batch(jobs), "outs": outs}


# ------------------------------------------------------------------ one pass


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "batch":
        state["batch"].launch()
        return state["outs"]
    ctx, ks, nbits = state["ctx"], state["ks"], case["nbits"]
    if case["host"]:
        if op == "encrypt":
            ctx.encrypt_message_host(ks, state["h_msg"], state["h_cipher"])
            return state["h_cipher"]
        ctx.decrypt_message_host(ks, state["h_cipher"], state["h_msg"], use_crt=op == "crt")
        return state["h_msg"]
    if op == "encrypt":
        return ctx.encrypt_chunks(ks, ctx.split(nbits, state["msg"]), key_idx=state["idx"])
    if op == "blind_encrypt":
        return ctx.encrypt_blinded(ks, ctx.split(nbits, state["msg"]), state["rnd"])
    if op == "blind_decrypt":
        m = ctx.decrypt_blinded(ks, state["cstar"], state["cr"], use_crt=True)
    else:
        m = ctx.decrypt_chunks(ks, state["cipher"], use_crt=op == "crt", key_idx=state["idx"])
    return ctx.join(nbits, m, case["msg_bytes"])


# ------------------------------------------------------------------ work and exact values


def _exp_macs(limbs, bits, windows):
    """32x32 -> 64-bit multiply-adds of one windowed exponentiation mod a
    `limbs`-limb modulus: `bits` squarings (each cross product once) and
    `windows` products, every one with a Montgomery reduction."""
    reduce = limbs * limbs + limbs
    return bits * (limbs * (limbs + 1) // 2 + reduce) + windows * (limbs * limbs + reduce)


def _macs_per_chunk(case):
    s, b = case["nbits"] // 32, case["primes"]
    h, hb = s // b, case["nbits"] // b
    encrypt = _exp_macs(s, 16, 3)
    if case["op"] == "encrypt":
        return encrypt
    if case["op"] == "blind_encrypt":
        return 2 * encrypt + _exp_macs(s, 0, 2)
    if case["op"] == "decrypt":
        return _exp_macs(s, 32 * s, 32 * s / 6 + 18)
    recombine = _exp_macs(s, 0, b)
    if case["op"] == "crt":
        return b * _exp_macs(h, hb, hb / 6 + 18 + b) + recombine
    return b * _exp_macs(h, hb, 2 * (hb / 5 + 8 + b)) + recombine  # blind_decrypt: two exponents, one squaring chain


def work(case):
    if case["op"] == "batch":
        parts = [work(sub) for sub, _ in _batch_jobs(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n = _chunks(case)
    limbs = 4 * n * (case["nbits"] // 32)
    keys = 2 * case["K"] * case["nbits"] // 8
    moved = {"blind_encrypt": 3, "blind_decrypt": 2}.get(case["op"], 1) * limbs + case["msg_bytes"] + keys
    return {"bytes": moved + (4 * n if case["idx"] else 0), "flops": 2.0 * n * _macs_per_chunk(case)}


def _limb_rows(values, nbits):
    raw = b"".join(v.to_bytes(nbits // 8, "little") for v in values)
    return np.frombuffer(raw, np.int32).reshape(len(values), nbits // 32)


def _exact_chunks(case, seed):
    """The chunk values m_t and the modulus of each."""
    msg, p = _message(case, seed).tobytes(), case["nbits"] // 8 - 1
    vals = [int.from_bytes(msg[i:i + p], "little") for i in range(0, len(msg), p)]
    N = _moduli(case["K"], case["nbits"], case["primes"])
    idx = _index(case, seed) if case["idx"] else [t % case["K"] for t in range(len(vals))]
    return vals, [N[k] for k in idx]


def _exact_encrypt(case, seed):
    if _chunks(case) * (case["nbits"] / 2048) ** 2 > 1.2e5:
        return None  # m^e of this many chunks takes plain Python integers too long
    m, N = _exact_chunks(case, seed)
    return _limb_rows([pow(x, E, n) for x, n in zip(m, N)], case["nbits"])


def _exact_one(case, seed):
    op = case["op"]
    if op == "encrypt":
        return _exact_encrypt(case, seed)
    if op == "blind_encrypt":
        c = _exact_encrypt(case, seed)
        if c is None:
            return None
        r = [int.from_bytes(row.tobytes(), "little") for row in _blinding(case, seed)]
        m, N = _exact_chunks(case, seed)
        star = [pow(x * y, E, n) for x, y, n in zip(m, r, N)]
        return _limb_rows(star, case["nbits"]), _limb_rows([pow(y, E, n) for y, n in zip(r, N)], case["nbits"])
    return _message(case, seed)  # every decryption returns the message


def exact(case, seed):
    """What run returns, from plain integers: decryptions return the message
    they were made from, encryptions are recomputed with Python's pow."""
    if case["op"] != "batch":
        return _exact_one(case, seed)
    outs = []
    for sub, sub_seed in _batch_jobs(case, seed):
        if sub["op"] == "encrypt":
            outs.append(_exact_encrypt(sub, sub_seed))
        else:
            outs.append(_limb_rows(_exact_chunks(sub, sub_seed)[0], sub["nbits"]))
    return outs
