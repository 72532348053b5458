"""How a ragged batch is divided, judged by time where a wrong division costs a factor: between warps and threads, and
between the queue's two parts.  Bytes are checked against hashlib on a sample."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def restore_split(cuda_lib):
    saved = cuda_lib.keccak_tune_get(cuda_lib.KB_TUNE_QUEUE_WARP_MESSAGES)
    yield
    cuda_lib.keccak_tune_set(cuda_lib.KB_TUNE_QUEUE_WARP_MESSAGES, saved)


class Batch:
    """SHA3-256 messages of the given lengths back to back, in the given order."""

    def __init__(self, cuda_lib, lens):
        import torch

        self.lib, self.n = cuda_lib, len(lens)
        self.lens = np.asarray(lens, dtype=np.int64)
        self.offsets = np.cumsum(self.lens) - self.lens
        self.msgs = torch.randint(0, 256, (int(self.lens.sum()) + 16,), dtype=torch.uint8, device="cuda")
        dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
        self.out = torch.zeros(32 * self.n, dtype=torch.uint8, device="cuda")
        self.args = (self.msgs, dev(self.offsets), dev(self.lens), dev(np.ones(self.n, np.uint8)),
                     dev(np.full(self.n, 32, np.int32)), self.out, self.n)

    def ms(self, split=-1):
        """Median time of a call with `split` messages fixed to a warp each (-1: the plan's choice)."""
        import torch

        self.lib.keccak_tune_set(self.lib.KB_TUNE_QUEUE_WARP_MESSAGES, split)
        self.out.zero_()
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            self.lib.keccak_batch(*self.args)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        got, host = self.out.cpu().numpy().reshape(-1, 32), self.msgs.cpu().numpy()
        for i in {0, 1, self.n // 2, self.n - 1, int(self.lens.argmax()), int(self.lens.argmin())}:
            o, k = int(self.offsets[i]), int(self.lens[i])
            assert got[i].tobytes() == hashlib.sha3_256(host[o:o + k].tobytes()).digest(), i
        return float(np.median(times[2:]))


@pytest.mark.parametrize("many", [9, 14])  # fortieths of the sub-partitions that the long messages fill
def test_queue_long_chains_start_in_the_slots_that_issue_first(cuda_lib, restore_split, many):
    """Long messages that give fewer sub-partitions than there are a warp each last as long as one of them; short ones
    beside them, of less work in all than the GPU does meanwhile, add little.  (With half of the long chains left to the
    warps that issue second they took 1.8 times as long.)"""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_long = 4 * sms * 32 * many // 40
    rng = np.random.default_rng(many)
    both = np.concatenate([np.full(n_long, 30000), np.full(7 * n_long, 200)])
    rng.shuffle(both)
    alone = Batch(cuda_lib, np.full(n_long, 30000)).ms(0)
    assert Batch(cuda_lib, both).ms(0) < 1.3 * alone


@pytest.mark.parametrize("kind", ["equal", "below a block", "few long"])
@pytest.mark.parametrize("per_sm", [33, 66, 131])
def test_split_leaves_equal_costs_to_threads(cuda_lib, restore_split, per_sm, kind):
    """Where warps would take longer for the costliest class than threads do, the plan moves none of it: the time is
    that of a thread for every message, give or take the launch beside it (at most 0.01 ms) and a tenth."""
    import torch

    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(per_sm)
    lens = {"equal": np.full(n, 4096), "below a block": rng.integers(0, 136, size=n),
            "few long": np.where(rng.random(n) < 0.5, 30000, 100)}[kind]
    batch = Batch(cuda_lib, lens)
    threads = batch.ms(0)
    assert batch.ms() < 1.1 * threads + 0.01


@pytest.mark.parametrize("kind", ["log-uniform", "a hundred long"])
def test_split_gives_few_long_chains_a_warp_each(cuda_lib, restore_split, kind):
    """Where a thread's chain for the costliest messages is longer than all the rest takes, they get a warp each, which
    is a third of that chain; half of the gain is asked for."""
    import torch

    n = 66 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(7)
    lens = np.exp(rng.uniform(0, np.log(65536), size=n)).astype(np.int64) if kind == "log-uniform" else \
        np.where(np.arange(n) % (n // 100) == 0, 65536, 500)
    batch = Batch(cuda_lib, lens)
    assert batch.ms() < 0.67 * batch.ms(0)


@pytest.mark.parametrize("blocks", [2, 3])
def test_queue_beside_an_idle_warp_kernel_keeps_its_time(cuda_lib, restore_split, blocks):
    """Where the plan moves nothing, the queue takes what it takes alone, call after call: its warps are sorted into
    those that issue first and the others however the launch before them ends."""
    import torch

    rng = np.random.default_rng(3)
    n = 2000 * torch.cuda.get_device_properties(0).multi_processor_count
    batch = Batch(cuda_lib, np.exp(rng.uniform(0, np.log(16384), size=n)).astype(np.int64))
    keys = (cuda_lib.KB_TUNE_QUEUE_MIN_BLOCKS, cuda_lib.KB_TUNE_QUEUE_BLOCKS_PER_SM, cuda_lib.KB_TUNE_QUEUE_STAGING)
    saved = [cuda_lib.keccak_tune_get(k) for k in keys]
    for k, v in zip(keys, (blocks, blocks, 1)):
        cuda_lib.keccak_tune_set(k, v)
    try:
        alone = batch.ms(0)
        assert max(batch.ms() for _ in range(5)) < 1.06 * alone
    finally:
        for k, v in zip(keys, saved):
            cuda_lib.keccak_tune_set(k, v)
