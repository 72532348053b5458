"""Kernels that a dispatch by size takes only past the sizes of the other tests: the general fixed-stride kernels, the
64-byte kernels in either staging, the ragged queue with the plan's own split from a replayed graph, with a tuned
configuration and without allocation, its digest places past the tiles that one block adds up, and every overlapped
launch captured in a caller's graph."""
import hashlib

import numpy as np
import pytest

from paper_1902_05320_gb300 import workloads as W
from test_gpu_small_batches import RATES, run_ragged, run_uniform, want, want_ragged

pytestmark = pytest.mark.gpu


def sm_count():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a).view({8: np.int64, 4: np.int32, 1: np.uint8}[a.itemsize])).cuda()


@pytest.fixture
def restore_tuning(cuda_lib):
    saved = [cuda_lib.keccak_tune_get(k) for k in range(cuda_lib.KB_TUNE_KEYS)]
    yield
    for k, v in enumerate(saved):
        cuda_lib.keccak_tune_set(k, v)


@pytest.mark.parametrize("shift", [0, 1, 3, 4])
@pytest.mark.parametrize("variant", range(6))
def test_general_fixed_stride_kernel(cuda_lib, variant, shift):
    """More than two warps a sub-partition: messages and outputs of one block and of several, aligned and not."""
    n = 257 * sm_count() + 3
    rate = RATES[variant]
    rng = np.random.default_rng(50 * variant + shift)
    for length in (rate - 1, rate, 2 * rate - 8, 2 * rate + 5, 3 * rate):
        for out_len in ((W.DIGEST_BYTES[variant],) if variant < 4 else (33, rate, rate + 1, 2 * rate + 3)):
            stride = length + (8 - length % 8 if shift == 4 else shift % 3)
            data = rng.integers(0, 256, size=n * stride, dtype=np.uint8)
            got = run_uniform(cuda_lib, data, 2 * shift, stride, length, variant, out_len, n)
            blob = data.tobytes()
            for i in {0, 1, 31, 32, 127, 128, n // 2, n - 4, n - 3, n - 2, n - 1}:
                assert got[i].tobytes() == want(variant, blob[i * stride:i * stride + length], out_len), (length, out_len, i)


@pytest.mark.parametrize("out_len", [1, 31, 168, 169, 337])
@pytest.mark.parametrize("staging", [0, 1])
def test_64_byte_kernels_in_either_staging(cuda_lib, restore_tuning, staging, out_len):
    cuda_lib.keccak_tune_set(cuda_lib.KB_TUNE_STAGING, staging)
    n = 257 * sm_count() + 77
    for variant in (4,) if out_len != 31 else (0, 1, 2, 3, 4, 5):
        size = W.DIGEST_BYTES[variant] or out_len
        data = np.random.default_rng(out_len + variant).integers(0, 256, size=64 * n, dtype=np.uint8)
        got = run_uniform(cuda_lib, data, 0, 64, 64, variant, size, n)
        blob = data.tobytes()
        for i in {0, 1, 127, 128, n // 2, n - 78, n - 77, n - 1} | set(range(77, n, 1997)):
            assert got[i].tobytes() == want(variant, blob[64 * i:64 * i + 64], size), (variant, i)


def test_graph_replay_plans_the_split_anew(cuda_lib, restore_tuning):
    """The replayed launches read lengths and bytes as they are then: the plan gives none, a few or many messages a warp."""
    import torch

    cuda_lib.keccak_tune_set(cuda_lib.KB_TUNE_GRAPHS, 1)
    n, room = 21 * sm_count() + 7, 20000
    rng = np.random.default_rng(1)
    variants = rng.integers(0, 6, size=n).astype(np.uint8)
    out_lens = np.array([W.DIGEST_BYTES[v] or 100 for v in variants], dtype=np.uint32)
    offsets = np.arange(n, dtype=np.uint64) * room + 1
    msgs = torch.zeros(n * room + 16, dtype=torch.uint8, device="cuda")
    d = [msgs, dev(offsets), dev(np.zeros(n, np.uint64)), dev(variants), dev(out_lens)]
    out = torch.zeros(int(out_lens.sum()), dtype=torch.uint8, device="cuda")
    s = torch.cuda.Stream()
    for k, lens in enumerate((np.full(n, 300), np.where(np.arange(n) % 100 == 7, 15000, 20),
                              np.exp(rng.uniform(0, np.log(room - 1), size=n)).astype(np.int64), np.full(n, 300))):
        msgs.random_(0, 256, generator=torch.Generator(device="cuda").manual_seed(k))
        d[2].copy_(torch.from_numpy(lens.astype(np.int64)))
        out.zero_()
        torch.cuda.synchronize()
        cuda_lib.keccak_batch(*d, out, n, s)
        s.synchronize()
        host, got, at = msgs.cpu().numpy(), out.cpu().numpy().tobytes(), 0
        for i in range(n):
            o, size = int(offsets[i]), int(out_lens[i])
            assert got[at:at + size] == want(int(variants[i]), host[o:o + int(lens[i])].tobytes(), size), (k, i)
            at += size
    assert cuda_lib.keccak_last_error(s) == 0


def test_tuned_configuration_runs_past_the_single_launch(cuda_lib, restore_tuning):
    n = 21 * sm_count() + 7
    b = W.ragged_batch(n, seed=8, max_len=5000, gap=3)
    out = dev(np.zeros(b.total_out(), np.uint8))
    args = [dev(a) for a in (b.msgs, b.offsets, b.lens, b.variants, b.out_lens)]
    try:
        chosen = cuda_lib.keccak_batch_autotune(*args, out, n)
        assert out.cpu().numpy().tobytes() == want_ragged(b)
        tuned = cuda_lib.keccak_tuned_config(n)
        assert all(tuned[key] == chosen[key] for key in tuned)
        got, err = run_ragged(cuda_lib, b)
        assert err == 0 and got.tobytes() == want_ragged(b)
    finally:
        cuda_lib.keccak_release()  # forgets the tuned configuration


def test_noalloc_queue_skips_bad_descriptors(cuda_lib):
    b = W.ragged_batch(21 * sm_count() + 7, seed=6, max_len=900, gap=2)
    bad = [3, b.n - 1] + [int(i) for i in np.flatnonzero(b.variants < 4)[5:8]]
    b.variants[bad[:2]] = 9
    b.out_lens[bad[2:]] += 1
    got, err = run_ragged(cuda_lib, b, noalloc=True)
    assert err == 0  # that entry does not report them
    blob, ends = b.msgs.tobytes(), np.cumsum(b.out_lens.astype(np.int64))
    for i in range(b.n):
        part = got[int(ends[i]) - int(b.out_lens[i]):int(ends[i])]
        if i in bad:
            assert (part == 0xEE).all(), i
        else:
            o, k = int(b.offsets[i]), int(b.lens[i])
            assert part.tobytes() == want(int(b.variants[i]), blob[o:o + k], int(b.out_lens[i])), i


@pytest.mark.parametrize("tiles", [4096, 4097])  # 4096 messages each; from 4097 on a kernel of its own adds them up
def test_digest_places_of_many_tiles(cuda_lib, tiles):
    """Empty and one-byte messages, outputs of one byte but for some around the tiles' edges: every output byte."""
    n = tiles * 4096 - (3 if tiles % 2 else 0)
    rng = np.random.default_rng(tiles)
    offsets = rng.integers(0, 4, size=n).astype(np.uint64)  # which of four bytes, where there is one
    lens = rng.integers(0, 2, size=n).astype(np.uint64)
    variants = np.full(n, 4, dtype=np.uint8)
    out_lens = np.ones(n, dtype=np.uint32)
    special = np.unique(np.concatenate([rng.integers(0, n, size=3000), [0, 4095, 4096, 8191, n - 4097, n - 4096, n - 1]]))
    out_lens[special] = rng.integers(0, 200, size=special.size)
    four = np.array([7, 99, 0, 255], dtype=np.uint8)
    kinds = np.stack([np.frombuffer(hashlib.shake_128(m).digest(200), np.uint8)
                      for m in [b""] + [bytes([int(x)]) for x in four]])
    kind = np.where(lens == 0, 0, 1 + offsets.astype(np.int64))
    starts = np.cumsum(out_lens, dtype=np.int64) - out_lens
    expected = np.zeros(int(out_lens.sum()), dtype=np.uint8)
    one = out_lens == 1
    expected[starts[one]] = kinds[kind[one], 0]
    for i in special:
        expected[starts[i]:starts[i] + out_lens[i]] = kinds[kind[i], :out_lens[i]]
    out = dev(np.full(expected.size + 64, 0xEE, dtype=np.uint8))
    cuda_lib.keccak_batch(dev(four), dev(offsets), dev(lens), dev(variants), dev(out_lens), out, n)
    assert cuda_lib.keccak_last_error() == 0
    got = out.cpu().numpy()
    assert (got[expected.size:] == 0xEE).all()
    assert np.array_equal(got[:expected.size], expected)


def _calls(cuda_lib):
    """name -> (function of (buffers, stream) that enqueues a chain of calls, function that makes fresh buffers)."""
    import torch

    sms = sm_count()
    chains = {}

    def uniform(n, length, variant, out_len):
        def make(seed):
            g = torch.Generator(device="cuda").manual_seed(seed)
            return {"in": torch.randint(0, 256, (n, length), dtype=torch.uint8, device="cuda", generator=g),
                    "mid": torch.zeros(n * out_len, dtype=torch.uint8, device="cuda"),
                    "out": torch.zeros(n * out_len, dtype=torch.uint8, device="cuda")}

        def run(b, s):  # the second call reads what the first wrote
            cuda_lib.keccak_batch_uniform(b["in"], length, length, variant, out_len, b["mid"], n, s)
            cuda_lib.keccak_batch_uniform(b["mid"], out_len, out_len, variant, out_len, b["out"], n, s)
        return run, make

    for name, per_sm, length, variant, out_len in (("warp", 3, 300, 3, 64), ("two threads", 40, 300, 0, 28),
                                                   ("two threads, one block", 40, 50, 1, 32), ("thread", 130, 300, 4, 200),
                                                   ("block per 128", 300, 300, 5, 40), ("64 bytes", 300, 64, 3, 64)):
        chains["uniform, " + name] = uniform(per_sm * sms + 1, length, variant, out_len)

    def ragged(n, entry):
        b0 = W.ragged_batch(n, seed=n, max_len=700, gap=2)

        def make(seed):
            return {"args": [dev(a) for a in (W.random_bytes(b0.msgs.size, seed), b0.offsets, b0.lens, b0.variants, b0.out_lens)],
                    "out": torch.zeros(b0.total_out(), dtype=torch.uint8, device="cuda"),
                    "again": torch.zeros(32, dtype=torch.uint8, device="cuda")}

        def run(b, s):
            entry(*b["args"], b["out"], n, s)
            cuda_lib.keccak_batch_uniform(b["out"], 0, b0.total_out(), 1, 32, b["again"], 1, s)
        return run, make

    for per_sm in (5, 25):
        chains[f"ragged {per_sm}"] = ragged(per_sm * sms, cuda_lib.keccak_batch)
        chains[f"noalloc {per_sm}"] = ragged(per_sm * sms, cuda_lib.keccak_batch_noalloc)

    def merkle(leaves, leaf_bytes):
        def make(seed):
            g = torch.Generator(device="cuda").manual_seed(seed)
            return {"in": torch.randint(0, 256, (leaves * leaf_bytes,), dtype=torch.uint8, device="cuda", generator=g),
                    "out": torch.zeros(32 * cuda_lib.merkle_node_count(leaves), dtype=torch.uint8, device="cuda")}
        return (lambda b, s: cuda_lib.merkle_sha3_256_levels(b["in"], leaves, leaf_bytes, b["out"], s)), make

    chains["merkle, few leaves"] = merkle(3 * sms, 201)
    chains["merkle"] = merkle(50 * sms, 136)

    def stream(n):
        lens = np.random.default_rng(n).integers(0, 400, size=n).astype(np.uint64)
        ends = np.cumsum(lens, dtype=np.uint64)

        def make(seed):
            return {"in": dev(W.random_bytes(int(ends[-1]), seed)), "offsets": dev(ends - lens), "lens": dev(lens),
                    "variants": dev((np.arange(n) % 6).astype(np.uint8)),
                    "sizes": dev(np.array([W.DIGEST_BYTES[i % 6] or 70 for i in range(n)], dtype=np.uint32)),
                    "states": torch.zeros(n * cuda_lib.KB_STATE_BYTES, dtype=torch.uint8, device="cuda"),
                    "out": torch.zeros(70 * n, dtype=torch.uint8, device="cuda")}

        def run(b, s):
            piece = (b["in"], b["offsets"], b["lens"])
            cuda_lib.keccak_stream_init(b["states"], b["variants"], n, s)
            cuda_lib.keccak_stream_absorb(b["states"], *piece, n, s)
            cuda_lib.keccak_stream_absorb(b["states"], *piece, n, s)
            cuda_lib.keccak_stream_absorb_final(b["states"], *piece, b["sizes"], b["out"], n, s)
        return run, make

    chains["stream, few"] = stream(3 * sms)
    chains["stream"] = stream(20 * sms)

    def keccak_p(n, width, rounds):
        def make(seed):
            g = torch.Generator(device="cuda").manual_seed(seed)
            return {"states": torch.randint(0, 1 << min(width // 25, 62), (n, 25), device="cuda", generator=g)}

        def run(b, s):
            for nr in rounds:
                cuda_lib.keccak_p_batch(b["states"], width, nr, n, s)
        return run, make

    chains["keccak-p, few"] = keccak_p(500, 1600, (24, 3))
    chains["keccak-p"] = keccak_p(30 * sms, 1600, (24, 3, 16))
    chains["keccak-p, narrow"] = keccak_p(30 * sms, 200, (18, 5))
    return chains


def test_overlapped_launches_in_a_captured_graph(cuda_lib):
    """Each chain of calls captured into the caller's graph (the programmatic launches behind whatever node comes before),
    replayed on new contents of the same buffers, against the same calls made directly."""
    import torch

    s = torch.cuda.Stream()
    for name, (run, make) in _calls(cuda_lib).items():
        flat = lambda b: [t for v in b.values() for t in (v if isinstance(v, list) else [v])]  # noqa: E731
        held = make(1)
        torch.cuda.synchronize()
        run(held, s)  # allocates what the calls keep for the stream
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            run(held, s)
        for seed in (2, 3):
            direct = make(seed)
            for mine, fresh in zip(flat(held), flat(direct)):
                mine.copy_(fresh)
            torch.cuda.synchronize()
            run(direct, None)
            graph.replay()
            torch.cuda.synchronize()
            for mine, theirs in zip(flat(held), flat(direct)):
                assert torch.equal(mine, theirs), (name, seed)
    assert cuda_lib.keccak_last_error(s) == 0
