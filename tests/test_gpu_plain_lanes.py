"""GPU parity of the plain form on both sides of the line between one env a
warp and full warps (32 envs for every SM), with a ragged last block."""
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_PLAIN

from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [-1, 0, 1])
def test_one_env_a_warp_and_full_warps_match_oracle(over):
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count + over
    roms = [synth.rom_sprite(4), synth.rom_playfield(2)]
    g, o = pair(roms, [0] * (n // 2) + [1] * (n - n // 2), form=FORM_PLAIN, startup_frames=3, max_noops=5)
    run_parity(g, o, synth.actions(94, 1, n))
