"""Workloads of the batch SHA-3 library, timed through its public Python entry points.

``listed()`` names the work a user of the library has it do; ``draw(rng)`` gives
further sizes of the same kinds.  Inputs are seeded random bytes made on the GPU
(host memory for the hash server, whose requests arrive there); sizes follow the
repository's benchmark, tests and smoke run.  Hash outputs are bytes, so they are
compared for equality; ``exact`` recomputes them with hashlib where that is quick.
"""
from __future__ import annotations

import hashlib
import math

import numpy as np
import torch

from paper_1902_05320_gb300 import binding, workloads
from paper_1902_05320_gb300.serve import Server

OPS_PER_PERMUTATION = 4163  # 32-bit integer operations of one Keccak-f[1600], leanest form
HASHES = (hashlib.sha3_224, hashlib.sha3_256, hashlib.sha3_384, hashlib.sha3_512, hashlib.shake_128, hashlib.shake_256)
EXACT_BYTES = 1 << 28  # hashlib is asked for at most this many message bytes


def listed():
    return [
        # A small latency-bound batch of short records (the smallest benchmark configuration).
        dict(name="uniform_4096x64", kind="uniform", n=4096, length=64, gap=0, variant=1, out_len=32),
        # The paper's largest batch: very short messages at no alignment.
        dict(name="uniform_119040x10", kind="uniform", n=119040, length=10, gap=0, variant=1, out_len=32),
        # The benchmark's headline: a large batch of 64-byte records.
        dict(name="uniform_2p24x64", kind="uniform", n=1 << 24, length=64, gap=0, variant=1, out_len=32),
        # Records of several blocks, of odd length and back to back, with the slowest function.
        dict(name="uniform_2p18x1023_512", kind="uniform", n=1 << 18, length=1023, gap=0, variant=3, out_len=64),
        # A handful of large objects hashed together (file checksums).
        dict(name="uniform_64x256KiB", kind="uniform", n=64, length=1 << 18, gap=0, variant=1, out_len=32),
        # A few hundred short byte strings of mixed functions (the smoke run's batch; what hash_many sends).
        dict(name="ragged_200x600", kind="ragged", n=200, max_len=600, gap=3),
        # The benchmark's ragged batch: a million messages from nothing to 64 KiB, six functions.
        dict(name="ragged_2p20x64KiB", kind="ragged", n=1 << 20, max_len=65536, gap=0),
        # The root of a small tree of odd-sized leaves (a block of records, a small file).
        dict(name="merkle_root_1000x1001", kind="merkle_root", leaves=1000, leaf_bytes=1001),
        # Every node of a 4 GiB tree of 8 KiB leaves, kept for proofs (the benchmark's tree).
        dict(name="merkle_levels_2p19x8KiB", kind="merkle_levels", leaves=1 << 19, leaf_bytes=8192),
        # Messages that arrive in pieces: many device sponge states, four pieces each.
        dict(name="stream_2p18x4x2KiB", kind="stream", n=1 << 18, piece=2048, pieces=4, variant=1, out_len=32),
        # The raw permutation on a large array of states.
        dict(name="keccak_p_1600_24_2p22", kind="keccak_p", n=1 << 22, b=1600, nr=24),
        # A burst of requests of the serving mix, 32 bytes to 1 MiB, through the hash server.
        dict(name="serve_burst_2000x1MiB", kind="serve", n=2000, max_len=1 << 20),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["uniform", "uniform", "uniform", "ragged", "ragged", "merkle_root", "merkle_levels", "stream",
                       "keccak_p", "serve"])
    if kind == "uniform":
        length = _log_int(rng, 8, 1 << 18) if rng.random() < 0.8 else rng.choice([32, 64, 65, 1024, 4096])
        variant = rng.randrange(6)
        out_len = workloads.DIGEST_BYTES[variant] or rng.randint(16, 512)
        n = _log_int(rng, 1, max(64, min(1 << 24, (1 << 31) // (length + 64))))
        return dict(kind=kind, n=n, length=length, gap=rng.choice([0, 0, 1, 8]), variant=variant, out_len=out_len)
    if kind == "ragged":
        return dict(kind=kind, n=_log_int(rng, 2, 1 << 19), max_len=rng.choice([600, 5000, 20000, 65536]),
                    gap=rng.choice([0, 3]))
    if kind.startswith("merkle"):
        leaf_bytes = _log_int(rng, 8, 8192)
        if rng.random() < 0.5:
            leaf_bytes = max(8, leaf_bytes // 8 * 8)
        return dict(kind=kind, leaves=_log_int(rng, 2, 1 << 18), leaf_bytes=leaf_bytes)
    if kind == "stream":
        variant = rng.randrange(6)
        out_len = workloads.DIGEST_BYTES[variant] or rng.randint(16, 512)
        return dict(kind=kind, n=_log_int(rng, 1, 1 << 17), piece=_log_int(rng, 16, 4096), pieces=rng.randint(2, 5),
                    variant=variant, out_len=out_len)
    if kind == "keccak_p":
        b = rng.choice([25, 50, 100, 200, 400, 800, 1600, 1600, 1600])
        full = 12 + 2 * int(math.log2(b // 25))
        return dict(kind=kind, n=_log_int(rng, 1, 1 << 21), b=b, nr=rng.choice([4, 12, full, full]))
    return dict(kind=kind, n=_log_int(rng, 16, 2000), max_len=_log_int(rng, 1 << 12, 1 << 20))


def _bytes(nbytes, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, 256, (max(int(nbytes), 1),), dtype=torch.uint8, device="cuda", generator=g)


def _dev(a):
    return torch.from_numpy(a.view({8: np.int64, 4: np.int32, 1: np.uint8}[a.itemsize])).cuda()


def _ragged_descriptors(case, seed):
    """(offsets, lens, variants, out_lens, total bytes): log-uniform lengths, six functions, SHAKE outputs 16..512.
    Functions and output sizes belong to the case, lengths and places to the seed."""
    n = case["n"]
    rng = np.random.default_rng(n)
    variants = rng.integers(0, 6, size=n).astype(np.uint8)
    out_lens = rng.integers(16, 513, size=n).astype(np.uint32)
    for v in range(4):
        out_lens[variants == v] = workloads.DIGEST_BYTES[v]
    rng = np.random.default_rng(seed)
    lens = workloads.log_uniform_lengths(rng, n, case["max_len"], 32 if case["kind"] == "serve" else 0)
    gaps = rng.integers(0, case.get("gap", 0) + 1, size=n).astype(np.uint64)
    ends = np.cumsum(lens + gaps, dtype=np.uint64)
    return ends - lens, lens, variants, out_lens, int(ends[-1])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "uniform":
        s["stride"] = case["length"] + case["gap"]
        s["msgs"] = _bytes(case["n"] * s["stride"], seed)
        s["out"] = torch.empty(case["n"] * case["out_len"], dtype=torch.uint8, device="cuda")
    elif kind == "ragged":
        offsets, lens, variants, out_lens, total = _ragged_descriptors(case, seed)
        s["msgs"] = _bytes(total, seed)
        s["offsets"], s["lens"], s["variants"], s["out_lens"] = (_dev(a) for a in (offsets, lens, variants, out_lens))
        s["out"] = torch.empty(int(out_lens.sum(dtype=np.uint64)), dtype=torch.uint8, device="cuda")
    elif kind in ("merkle_root", "merkle_levels"):
        s["buf"] = _bytes(case["leaves"] * case["leaf_bytes"], seed)
        s["nodes"] = torch.empty((binding.merkle_node_count(case["leaves"]), 32), dtype=torch.uint8, device="cuda")
    elif kind == "stream":
        n, piece = case["n"], case["piece"]
        s["states"] = torch.zeros(n * binding.KB_STATE_BYTES, dtype=torch.uint8, device="cuda")
        s["variants"] = torch.full((n,), case["variant"], dtype=torch.uint8, device="cuda")
        s["chunks"] = [_bytes(n * piece, seed * 31 + k) for k in range(case["pieces"])]
        s["offsets"] = torch.arange(n, dtype=torch.int64, device="cuda") * piece
        s["lens"] = torch.full((n,), piece, dtype=torch.int64, device="cuda")
        s["out_lens"] = torch.full((n,), case["out_len"], dtype=torch.int32, device="cuda")
        s["out"] = torch.empty(n * case["out_len"], dtype=torch.uint8, device="cuda")
    elif kind == "keccak_p":
        w = case["b"] // 25
        lanes = _bytes(case["n"] * 200, seed).view(torch.int64)
        s["states"] = lanes if w == 64 else lanes & ((1 << w) - 1)
    elif kind == "serve":
        offsets, lens, variants, out_lens, total = _ragged_descriptors(case, seed)
        s["offsets"], s["lens"], s["variants"], s["out_lens"] = offsets, lens, variants, out_lens
        s["arrival_ns"] = np.zeros(case["n"], dtype=np.int64)
        s["pool"] = Server.pinned(total)
        s["pool"].copy_(_bytes(total, seed))
        s["out"] = Server.pinned(int(out_lens.sum(dtype=np.uint64)))
        s["server"] = Server()
    return s


def run(s):
    kind = s["kind"]
    if kind == "uniform":
        binding.keccak_batch_uniform(s["msgs"], s["stride"], s["length"], s["variant"], s["out_len"], s["out"], s["n"])
        return s["out"]
    if kind == "ragged":
        binding.keccak_batch(s["msgs"], s["offsets"], s["lens"], s["variants"], s["out_lens"], s["out"], s["n"])
        return s["out"]
    if kind == "merkle_root":
        return np.frombuffer(binding.merkle_sha3_256(s["buf"], s["leaves"], s["leaf_bytes"]), dtype=np.uint8)
    if kind == "merkle_levels":
        binding.merkle_sha3_256_levels(s["buf"], s["leaves"], s["leaf_bytes"], s["nodes"])
        return s["nodes"]
    if kind == "stream":
        n, states, offsets, lens, chunks = s["n"], s["states"], s["offsets"], s["lens"], s["chunks"]
        binding.keccak_stream_init_absorb(states, s["variants"], chunks[0], offsets, lens, n)
        for c in chunks[1:-1]:
            binding.keccak_stream_absorb(states, c, offsets, lens, n)
        binding.keccak_stream_absorb_final(states, chunks[-1], offsets, lens, s["out_lens"], s["out"], n)
        return s["out"]
    if kind == "keccak_p":
        # In place: every pass permutes the states that the last one left.
        binding.keccak_p_batch(s["states"], s["b"], s["nr"], s["n"])
        return s["states"]
    s["server"].replay(s["pool"], s["offsets"], s["lens"], s["variants"], s["out_lens"], s["arrival_ns"], s["out"])
    return s["out"]


def _permutations(length, variant, out_len):
    rate = binding.RATE_BYTES[variant]
    return length // rate + 1 + (max(out_len, 1) - 1) // rate


def work(case):
    kind = case["kind"]
    if kind == "uniform":
        n = case["n"]
        nbytes = n * (case["length"] + case["out_len"])
        perms = n * _permutations(case["length"], case["variant"], case["out_len"])
    elif kind in ("ragged", "serve"):
        _, lens, variants, out_lens, _ = _ragged_descriptors(case, 1)
        rate = np.asarray(binding.RATE_BYTES, dtype=np.int64)[variants]
        nbytes = int(lens.sum()) + int(out_lens.sum(dtype=np.uint64)) + 21 * case["n"]
        perms = int((lens.astype(np.int64) // rate + 1 + (out_lens.astype(np.int64) - 1) // rate).sum())
    elif kind in ("merkle_root", "merkle_levels"):
        leaves = case["leaves"]
        nodes = leaves - 1
        nbytes = leaves * case["leaf_bytes"] + (32 * (leaves + nodes) if kind == "merkle_levels" else 32)
        perms = leaves * _permutations(case["leaf_bytes"] + 1, 1, 32) + nodes
    elif kind == "stream":
        n, length = case["n"], case["piece"] * case["pieces"]
        # The sponge states between the calls are read and written once a call, the pieces once.
        nbytes = n * (length + case["out_len"] + 2 * 216 * (case["pieces"] - 1))
        perms = n * _permutations(length, case["variant"], case["out_len"])
    else:  # keccak_p
        nbytes = case["n"] * 400
        perms = case["n"] * case["nr"] / 24 * min(1.0, max(case["b"], 800) / 1600)
    return {"bytes": nbytes, "flops": perms * OPS_PER_PERMUTATION}


def _hash(variant, data, out_len):
    h = HASHES[variant](data)
    return h.digest(out_len) if variant >= 4 else h.digest()


def _u8(parts):
    return np.frombuffer(b"".join(parts), dtype=np.uint8)


def _tree(digests):
    """Every node, leaves first: SHA3-256(0x01 || left || right), an odd last node carried up."""
    nodes, level = list(digests), list(digests)
    while len(level) > 1:
        up = [hashlib.sha3_256(b"\x01" + level[i] + level[i + 1]).digest() for i in range(0, len(level) - 1, 2)]
        level = up + level[len(level) & ~1:]
        nodes += level
    return nodes


def exact(case, seed):
    kind = case["kind"]
    calls = case.get("n", case.get("leaves", 0))
    if kind == "keccak_p" or calls > 1 << 18 or work(case)["bytes"] > EXACT_BYTES:
        return None
    if kind == "uniform":
        n, length, stride = case["n"], case["length"], case["length"] + case["gap"]
        data = _bytes(n * stride, seed).cpu().numpy().tobytes()
        return _u8([_hash(case["variant"], data[i * stride:i * stride + length], case["out_len"]) for i in range(n)])
    if kind in ("ragged", "serve"):
        offsets, lens, variants, out_lens, total = _ragged_descriptors(case, seed)
        data = _bytes(total, seed).cpu().numpy().tobytes()
        return _u8([_hash(int(v), data[int(o):int(o) + int(k)], int(d))
                    for o, k, v, d in zip(offsets, lens, variants, out_lens)])
    if kind in ("merkle_root", "merkle_levels"):
        leaves, size = case["leaves"], case["leaf_bytes"]
        data = _bytes(leaves * size, seed).cpu().numpy().tobytes()
        nodes = _tree([hashlib.sha3_256(b"\x00" + data[i * size:(i + 1) * size]).digest() for i in range(leaves)])
        return _u8(nodes[-1:]) if kind == "merkle_root" else _u8(nodes).reshape(-1, 32)
    n, piece = case["n"], case["piece"]
    data = [_bytes(n * piece, seed * 31 + k).cpu().numpy().tobytes() for k in range(case["pieces"])]
    return _u8([_hash(case["variant"], b"".join(c[i * piece:(i + 1) * piece] for c in data), case["out_len"])
                for i in range(n)])
