"""What a queue configuration says about who decides the split between warps and threads (host only)."""
import pytest

from paper_1902_05320_gb300 import binding


@pytest.mark.parametrize("knob,warp_messages,split", [(-1, 0, "the plan of each batch"), (-1, 608, "fixed: 608"),
                                                      (0, 0, "fixed: 0"), (32, 32, "fixed: 32")])
def test_queue_config_tells_the_planned_split_from_a_fixed_one(knob, warp_messages, split):
    saved = binding.keccak_tune_get(binding.KB_TUNE_QUEUE_WARP_MESSAGES)
    binding.keccak_tune_set(binding.KB_TUNE_QUEUE_WARP_MESSAGES, knob)
    try:
        assert binding.QueueConfig(warp_messages=warp_messages).as_dict()["split"] == split
    finally:
        binding.keccak_tune_set(binding.KB_TUNE_QUEUE_WARP_MESSAGES, saved)
