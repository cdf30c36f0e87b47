"""The launch shape that an env reports is the one that it launches: in the
plain form one env a warp while that is the faster, else full warps, in blocks
of two warps."""
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_PLAIN, OUT_PALETTE, AtariEnv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [-1, 0, 1])
def test_plain_form_reports_its_grid(over):
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count + over
    r = synth.rom_playfield(2)
    g = AtariEnv([r.data], [(r.score_addr, r.gameover_addr)], [0] * n, form=FORM_PLAIN, output_mode=OUT_PALETTE,
                 startup_frames=1, max_noops=1, n_cache=1, log_cap=256)
    lanes = 32 if over > 0 else 1
    assert g.launch_shape() == (lanes, 2 * lanes, 1, -(-n // (2 * lanes)), 1, 1)
