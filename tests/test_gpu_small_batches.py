"""Batches too small to fill the GPU with a thread per message: the forms with thirty and with two threads a
message, at the edges of their size ranges, of the rate and of the alignment, against hashlib."""
import hashlib

import numpy as np
import pytest

from paper_1902_05320_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HASHES = (hashlib.sha3_224, hashlib.sha3_256, hashlib.sha3_384, hashlib.sha3_512, hashlib.shake_128,
          hashlib.shake_256)
RATES = (144, 136, 104, 72, 168, 136)


def want(variant, data, out_len):
    h = HASHES[variant](data)
    return h.digest(out_len) if variant >= 4 else h.digest()


def run_uniform(cuda_lib, data, shift, stride, length, variant, out_len, n):
    """Digests of n messages whose first byte sits `shift` bytes into an allocation, with guard bytes around the
    output (one byte in, so no store is aligned by luck when shift is odd)."""
    import torch

    raw = torch.zeros(shift + data.size + 16, dtype=torch.uint8, device="cuda")
    raw[shift:shift + data.size] = torch.from_numpy(data).cuda()
    out = torch.full((n * out_len + 32,), 0xEE, dtype=torch.uint8, device="cuda")
    o = 16 + (shift & 1)
    cuda_lib.keccak_batch_uniform(raw.data_ptr() + shift, stride, length, variant, out_len, out.data_ptr() + o, n)
    got = out.cpu().numpy()
    assert (got[:o] == 0xEE).all() and (got[o + n * out_len:] == 0xEE).all(), "bytes outside the output were written"
    return got[o:o + n * out_len].reshape(n, out_len)


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 7])
@pytest.mark.parametrize("variant", range(6))
@pytest.mark.parametrize("per_sm", [0, 13, 70, 130])  # thirty threads a message; two; one, a warp or two a sub-partition
def test_lengths_and_alignments(cuda_lib, variant, shift, per_sm):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = max(3, per_sm * sms)
    rate = RATES[variant]
    rng = np.random.default_rng(1000 * variant + shift)
    for length in (0, 1, 6, 7, 8, rate - 1, rate, rate + 1, 2 * rate - 8, 2 * rate, 3 * rate - 1, 3 * rate, 4 * rate + 5):
        for out_len in ((W.DIGEST_BYTES[variant],) if variant < 4 else (1, 33, rate, rate + 1, 2 * rate + 3)):
            if variant >= 4 and length not in (0, rate, 3 * rate) and out_len != 33:
                continue
            stride = length + (shift % 3)
            data = rng.integers(0, 256, size=max(1, n * stride), dtype=np.uint8)
            got = run_uniform(cuda_lib, data, shift, stride, length, variant, out_len, n)
            blob = data.tobytes()
            for i in sorted({0, 1, 2, 31, 32, n // 2, n - 2, n - 1} & set(range(n))):
                assert got[i].tobytes() == want(variant, blob[i * stride:i * stride + length], out_len), (length, out_len, i)


@pytest.mark.parametrize("blocks", [1, 3])
@pytest.mark.parametrize("edge", [8, 12, 64, 128, 256])  # the lines between the forms, in messages per SM
def test_batch_sizes_around_the_lines(cuda_lib, edge, blocks):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    length = 136 * blocks - 9
    for n in (edge * sms - 1, edge * sms, edge * sms + 1):
        data = np.random.default_rng(n).integers(0, 256, size=n * length, dtype=np.uint8)
        got = run_uniform(cuda_lib, data, 0, length, length, 1, 32, n)
        blob = data.tobytes()
        for i in range(n):
            assert got[i].tobytes() == hashlib.sha3_256(blob[i * length:(i + 1) * length]).digest(), (n, i)


@pytest.mark.parametrize("variant,out_len", [(1, 32), (3, 64), (4, 337)])
@pytest.mark.parametrize("tiles,more", [(100, -1), (100, 0), (100, 1), (7 * 152, 1), (14 * 152 + 5, 127)])
def test_tiles_of_128_messages(cuda_lib, tiles, more, variant, out_len):
    """64-byte messages packed back to back, a block per tile: the last tile whole, one message short or with one."""
    n = 128 * tiles + more
    data = np.random.default_rng(n).integers(0, 256, size=n * 64, dtype=np.uint8)
    got = run_uniform(cuda_lib, data, 0, 64, 64, variant, out_len, n)
    blob = data.tobytes()
    for i in sorted({0, 1, 127, 128, 129, n // 2, n - 130, n - 129, n - 128, n - 127, n - 2, n - 1} |
                    set(range(77, n, 997))):
        assert got[i].tobytes() == want(variant, blob[64 * i:64 * i + 64], out_len), i


def run_ragged(cuda_lib, b, noalloc=False):
    """(output bytes with 0xEE where nothing was written, device status) of a RaggedBatch."""
    import torch

    view = {8: np.int64, 4: np.int32, 1: np.uint8}
    args = [torch.from_numpy(np.ascontiguousarray(a).view(view[a.itemsize])).cuda()
            for a in (b.msgs, b.offsets, b.lens, b.variants, b.out_lens)]
    out = torch.full((b.total_out() + 16,), 0xEE, dtype=torch.uint8, device="cuda")
    cuda_lib.keccak_last_error()
    (cuda_lib.keccak_batch_noalloc if noalloc else cuda_lib.keccak_batch)(*args, out, b.n)
    err = cuda_lib.keccak_last_error()
    got = out.cpu().numpy()
    assert (got[b.total_out():] == 0xEE).all()
    return got[:b.total_out()], err


def want_ragged(b):
    blob = b.msgs.tobytes()
    return b"".join(want(int(v), blob[int(o):int(o) + int(n)], int(d))
                    for o, n, v, d in zip(b.offsets, b.lens, b.variants, b.out_lens))


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("per_sm,more", [(0, 1), (0, 2), (0, 33), (20, 0), (20, 1), (40, 0)])
def test_ragged_sizes_around_the_line(cuda_lib, per_sm, more, noalloc):
    import torch

    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    b = W.ragged_batch(n, seed=n, max_len=1500, shake_out=(0, 400), gap=3)
    got, err = run_ragged(cuda_lib, b, noalloc)
    assert err == 0 and got.tobytes() == want_ragged(b)


def test_ragged_small_skips_bad_descriptors(cuda_lib):
    b = W.ragged_batch(300, seed=5, max_len=900, gap=2)
    bad = [3, 299] + [int(i) for i in np.flatnonzero(b.variants < 4)[5:8]]
    b.variants[bad[:2]] = 9
    b.out_lens[bad[2:]] += 1
    got, err = run_ragged(cuda_lib, b)
    assert err == cuda_lib.KB_DEV_BAD_VARIANT | cuda_lib.KB_DEV_BAD_OUTLEN
    blob, ends = b.msgs.tobytes(), np.cumsum(b.out_lens.astype(np.int64))
    for i in range(b.n):
        part = got[int(ends[i]) - int(b.out_lens[i]):int(ends[i])]
        if i in bad:
            assert (part == 0xEE).all(), i
        else:
            o, k = int(b.offsets[i]), int(b.lens[i])
            assert part.tobytes() == want(int(b.variants[i]), blob[o:o + k], int(b.out_lens[i])), i


@pytest.mark.parametrize("n,pad", [(3, 0), (3, 200), (2500, 200), (5000, 0), (20000, 0), (20000, 32)])
def test_chained_calls_see_each_other(cuda_lib, n, pad):
    """Launches overlap the set-up of the next one with the end of the last: each call here reads what the call
    before it wrote and overwrites what the one before that read, with a torch copy in between now and then."""
    import torch

    length = 32 + pad
    rng = np.random.default_rng(n + pad)
    start = rng.integers(0, 256, size=(n, length), dtype=np.uint8)
    a, b = torch.from_numpy(start).cuda(), torch.from_numpy(start).cuda()
    d, d2 = (torch.empty((n, 32), dtype=torch.uint8, device="cuda") for _ in range(2))
    ref = [start[i].tobytes() for i in range(min(n, 64))]
    for step in range(24):
        # The first 32 bytes of every message become its digest.
        cuda_lib.keccak_batch_uniform(a, length, length, 1, 32, d, n)
        if step % 3 == 0:
            b[:, :32].copy_(d)
        else:
            cuda_lib.keccak_batch_uniform(d, 32, 32, 1, 32, d2, n)
            b[:, :32].copy_(d2)
        a, b = b, a
        b.copy_(a)
        ref = [(hashlib.sha3_256(m).digest() if step % 3 == 0 else
                hashlib.sha3_256(hashlib.sha3_256(m).digest()).digest()) + m[32:] for m in ref]
    got = a.cpu().numpy()
    assert [got[i].tobytes() for i in range(len(ref))] == ref


@pytest.mark.parametrize("n,long_len,long_every", [(4000, 60000, 3), (9000, 60000, 40), (9000, 0, 1), (30000, 30000, 1000)])
def test_ragged_split_between_warps_and_threads(cuda_lib, n, long_len, long_every):
    """Batches whose plan gives a warp each to many, to a few or to all of the messages, beside the queue."""
    rng = np.random.default_rng(n + long_every)
    lens = rng.integers(0, 700, size=n)
    if long_len:
        lens[::long_every] = rng.integers(long_len // 2, long_len, size=lens[::long_every].size)
    b = W.ragged_batch(n, seed=n + 1, lens=lens, shake_out=(0, 200), gap=3)
    for noalloc in (False, True):
        got, err = run_ragged(cuda_lib, b, noalloc)
        assert err == 0 and got.tobytes() == want_ragged(b)


@pytest.mark.parametrize("k", [-1, 0, 33, "most", "all"])  # messages that take a warp each; the queue has the rest
@pytest.mark.parametrize("kind", ["equal", "empty", "one long", "one valid"])
def test_queue_parts(cuda_lib, kind, k):
    """The queue's costlier and cheaper part where costs tie, where one message is half of the work, and where most
    messages have no cost."""
    import torch

    n = 21 * torch.cuda.get_device_properties(0).multi_processor_count + 7
    lens = np.full(n, {"equal": 300, "one valid": 500}.get(kind, 0))
    if kind == "one long":
        lens[n // 3] = 50000
    b = W.ragged_batch(n, seed=11, lens=lens, shake_out=(1, 90), gap=1)
    if kind == "one valid":
        b.variants[np.arange(n) != 1000] = 77
    saved = cuda_lib.keccak_tune_get(cuda_lib.KB_TUNE_QUEUE_WARP_MESSAGES)
    cuda_lib.keccak_tune_set(cuda_lib.KB_TUNE_QUEUE_WARP_MESSAGES, {"most": n - 31, "all": n}.get(k, k))
    try:
        got, err = run_ragged(cuda_lib, b)
    finally:
        cuda_lib.keccak_tune_set(cuda_lib.KB_TUNE_QUEUE_WARP_MESSAGES, saved)
    if kind == "one valid":
        assert err == cuda_lib.KB_DEV_BAD_VARIANT
        at, size = int(b.out_offsets()[1000]), int(b.out_lens[1000])
        o = int(b.offsets[1000])
        assert got[at:at + size].tobytes() == want(int(b.variants[1000]), b.msgs.tobytes()[o:o + 500], size)
        got[at:at + size] = 0xEE
        assert (got == 0xEE).all()
    else:
        assert err == 0 and got.tobytes() == want_ragged(b)


def tree_nodes(leaves):
    nodes = level = [hashlib.sha3_256(b"\x00" + leaf).digest() for leaf in leaves]
    while len(level) > 1:
        up = [hashlib.sha3_256(b"\x01" + level[i] + level[i + 1]).digest() for i in range(0, len(level) - 1, 2)]
        level = up + level[len(level) & ~1:]
        nodes = nodes + level
    return b"".join(nodes)


@pytest.mark.parametrize("leaf_bytes", [1, 6, 7, 8, 127, 128, 134, 135, 136, 143, 144, 271, 272, 407, 1001])
@pytest.mark.parametrize("n", [1, 2, 3, 15, 16, 17, 33, 255, 257, 1303])
def test_merkle_small_trees_every_node(cuda_lib, n, leaf_bytes):
    import torch

    shift = (n + leaf_bytes) % 5
    data = np.random.default_rng(n * 2000 + leaf_bytes).integers(0, 256, size=n * leaf_bytes, dtype=np.uint8)
    raw = torch.zeros(data.size + 16, dtype=torch.uint8, device="cuda")
    raw[shift:shift + data.size] = torch.from_numpy(data).cuda()
    nodes = torch.empty(32 * cuda_lib.merkle_node_count(n), dtype=torch.uint8, device="cuda")
    cuda_lib.merkle_sha3_256_levels(raw.data_ptr() + shift, n, leaf_bytes, nodes)
    blob = data.tobytes()
    assert nodes.cpu().numpy().tobytes() == tree_nodes([blob[i * leaf_bytes:(i + 1) * leaf_bytes] for i in range(n)])


@pytest.mark.parametrize("per_sm", [12, 16, 32])  # the lines of the leaves and of the levels
@pytest.mark.parametrize("leaf_bytes", [137, 200])
def test_merkle_trees_around_the_lines(cuda_lib, per_sm, leaf_bytes):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (per_sm * sms, per_sm * sms + 1):
        data = np.random.default_rng(n).integers(0, 256, size=n * leaf_bytes, dtype=np.uint8)
        nodes = torch.empty(32 * cuda_lib.merkle_node_count(n), dtype=torch.uint8, device="cuda")
        cuda_lib.merkle_sha3_256_levels(torch.from_numpy(data).cuda(), n, leaf_bytes, nodes)
        blob = data.tobytes()
        want_nodes = tree_nodes([blob[i * leaf_bytes:(i + 1) * leaf_bytes] for i in range(n)])
        assert nodes.cpu().numpy().tobytes() == want_nodes


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("per_sm,more", [(0, 1), (3, 7), (12, 0), (12, 1)])  # the line between warps and threads
def test_stream_around_the_line(cuda_lib, per_sm, more, fused):
    """Pieces of 0, 1, a few and many bytes, opening blocks at every offset, through either form of every step."""
    import torch

    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    rng = np.random.default_rng(17 * n + fused)
    dev = lambda a: torch.from_numpy(a.view({8: np.int64, 4: np.int32, 1: np.uint8}[a.itemsize])).cuda()  # noqa: E731
    variants = rng.integers(0, 6, size=n).astype(np.uint8)
    out_lens = np.array([W.DIGEST_BYTES[v] or rng.integers(0, 400) for v in variants], dtype=np.uint32)
    d_var, d_out = dev(variants), dev(out_lens)
    states = torch.full((n * cuda_lib.KB_STATE_BYTES,), 0xA5, dtype=torch.uint8, device="cuda")
    out = torch.full((int(out_lens.sum()) + 16,), 0xEE, dtype=torch.uint8, device="cuda")
    messages = [b""] * n
    cuda_lib.keccak_last_error()
    steps = 5
    for step in range(steps):
        lens = np.where(rng.random(n) < 0.3, rng.integers(0, 9, size=n), rng.integers(0, 900, size=n)).astype(np.uint64)
        gaps = rng.integers(0, 4, size=n).astype(np.uint64)
        ends = np.cumsum(lens + gaps, dtype=np.uint64)
        data = rng.integers(0, 256, size=int(ends[-1]) + 1, dtype=np.uint8)
        blob = data.tobytes()
        messages = [m + blob[int(e - k):int(e)] for m, e, k in zip(messages, ends, lens)]
        args = (dev(data), dev(ends - lens), dev(lens))
        if step == 0 and fused:
            cuda_lib.keccak_stream_init_absorb(states, d_var, *args, n)
        elif step == steps - 1 and fused:
            cuda_lib.keccak_stream_absorb_final(states, *args, d_out, out, n)
        else:
            if step == 0:
                cuda_lib.keccak_stream_init(states, d_var, n)
            cuda_lib.keccak_stream_absorb(states, *args, n)
        torch.cuda.synchronize()
    if not fused:
        cuda_lib.keccak_stream_final(states, d_out, out, n)
    assert cuda_lib.keccak_last_error() == 0
    got = out.cpu().numpy()
    assert (got[int(out_lens.sum()):] == 0xEE).all()
    assert got[:int(out_lens.sum())].tobytes() == b"".join(want(int(v), m, int(d))
                                                           for v, m, d in zip(variants, messages, out_lens))


def test_stream_refusals_in_both_forms(cuda_lib):
    """An unknown function, a wrong digest size and a finalised state: the same status bits and untouched outputs
    from the warp form and the thread form."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    seen = []
    for n in (40, 12 * sms + 40):
        variants = torch.ones(n, dtype=torch.uint8, device="cuda")
        variants[5] = 9
        states = torch.zeros(n * cuda_lib.KB_STATE_BYTES, dtype=torch.uint8, device="cuda")
        data = torch.arange(100 * n, device="cuda").to(torch.uint8)
        offsets = torch.arange(n, device="cuda") * 100
        lens = torch.full((n,), 100, dtype=torch.int64, device="cuda")
        out_lens = torch.full((n,), 32, dtype=torch.int32, device="cuda")
        out_lens[7] = 31
        out = torch.full((32 * n,), 0xEE, dtype=torch.uint8, device="cuda")
        errs = []
        cuda_lib.keccak_last_error()
        cuda_lib.keccak_stream_init_absorb(states, variants, data, offsets, lens, n)
        errs.append(cuda_lib.keccak_last_error())
        cuda_lib.keccak_stream_absorb_final(states, data, offsets, lens, out_lens, out, n)
        errs.append(cuda_lib.keccak_last_error())
        mine = 32 * 40 - 1  # the outputs of the first 40 messages, one of them 31 bytes
        first = out.cpu().numpy()[:mine].copy()
        cuda_lib.keccak_stream_absorb(states, data, offsets, lens, n)  # finalised states refuse more
        errs.append(cuda_lib.keccak_last_error())
        cuda_lib.keccak_stream_absorb(states, data, offsets, torch.zeros_like(lens), n)
        errs.append(cuda_lib.keccak_last_error())
        cuda_lib.keccak_stream_final(states, out_lens, out, n)
        errs.append(cuda_lib.keccak_last_error())
        seen.append((errs, first.tobytes(), out.cpu().numpy()[:mine].tobytes()))
    assert seen[0] == seen[1] and seen[0][0][0] == cuda_lib.KB_DEV_BAD_VARIANT


@pytest.mark.parametrize("b,nr", [(25, 12), (200, 18), (800, 22), (1600, 3)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 129, 7 * 128 * 152 + 33])
def test_keccak_p_tiles(cuda_lib, b, nr, n):
    """The staged kernels at the edges of a warp's and a block's tile: the same results in reverse order (so every state
    at another place), the first and the last against the oracle, and the state past the last one untouched."""
    import torch

    import oracle

    w = b // 25
    given = np.random.default_rng(b + n).integers(0, 1 << 64, size=(n + 1, 25), dtype=np.uint64) >> np.uint64(64 - w)
    states = torch.from_numpy(given.view(np.int64)).cuda()
    turned = states[:n].flip(0).contiguous()
    cuda_lib.keccak_p_batch(states, b, nr, n)
    cuda_lib.keccak_p_batch(turned, b, nr, n)
    assert torch.equal(states[:n], turned.flip(0))
    got = states.cpu().numpy().view(np.uint64)
    assert (got[n] == given[n]).all()
    for i in {0, n - 1}:
        bits = np.array([(int(v) >> z) & 1 for v in given[i] for z in range(w)], dtype=np.uint8)
        lanes = oracle.keccak_p(b, nr, bits).reshape(25, w)
        assert [sum(int(x) << z for z, x in enumerate(lane)) for lane in lanes] == [int(v) for v in got[i]], i


@pytest.mark.parametrize("nr", [1, 2, 11, 12, 24, 25])
@pytest.mark.parametrize("per_sm,more", [(0, 1), (0, 5), (12, 0), (12, 1)])
def test_keccak_p_around_the_line(cuda_lib, per_sm, more, nr):
    """Few states (a warp each) against many (a thread each), and 24 rounds against hashlib."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = per_sm * sms + more
    states = np.random.default_rng(n + nr).integers(0, 2**63, size=(n, 25), dtype=np.int64)
    # Row 0 holds the padded one-block message of SHA3-256("abc").
    states[0] = 0
    states[0].view(np.uint8)[:4] = np.frombuffer(b"abc\x06", np.uint8)
    states[0].view(np.uint8)[135] = 0x80
    few = torch.from_numpy(states).cuda()
    cuda_lib.keccak_p_batch(few, 1600, nr, n)
    many = torch.from_numpy(np.tile(states, (12 * sms // n + 2, 1))).cuda()
    cuda_lib.keccak_p_batch(many, 1600, nr, many.shape[0])
    assert torch.equal(few, many[:n])
    if nr == 24:
        assert few[0].cpu().numpy().tobytes()[:32] == hashlib.sha3_256(b"abc").digest()
