"""The tests of the generation loop that small models run in one launch, once more with a launch per kernel (CS_SMALL=0): the greedy targets, the EOS rule, ragged batches,
sequences without room, and launches of consecutive steps that overlap, for heads that the mma.sync attention takes."""
import pytest

from test_gpu_loop import (pytestmark, test_a_sequence_without_room_does_not_stop_the_others, test_batch_of_sequences_with_eos_and_different_lengths,  # noqa: F401
                           test_loop_without_graph_capture_gives_the_same_result, test_tiny_config_real_mode_is_greedy_decoding,
                           test_tiny_config_scripted_mode)


@pytest.fixture(autouse=True)
def _a_launch_per_kernel(monkeypatch):
    monkeypatch.setenv("CS_SMALL", "0")
