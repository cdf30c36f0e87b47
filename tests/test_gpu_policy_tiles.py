"""GPU parity of the policy kernel at the edges of its tiles: env counts
around a lane's four envs, a warp's 32 and a block's 128, and weights at an
address that is not 4-byte aligned.  Logits equal the
oracle's bit for bit, actions too."""
import numpy as np
import pytest
import torch

from oracle import OracleEnvs
from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, AtariEnv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(1, 0), (31, 0), (33, 1), (96, 0), (127, 0), (128, 1), (129, 0), (257, 0)])
def test_policy_tile_edges_bit_exact(n, shift):
    rom = synth.rom_sprite(1)
    g = AtariEnv([rom.data], [(rom.score_addr, rom.gameover_addr)], [0] * n, luma=synth.luma_table(), seed=9,
                 form=FORM_BATCHED, envs_per_warp=32, envs_per_block=64, tia_warps=2)
    o = OracleEnvs([rom.data], [rom.score_addr], [rom.gameover_addr], [0] * n, luma=synth.luma_table(), seed=9)
    W = synth.policy_weights(7)
    buf = torch.zeros(W.size + shift, dtype=torch.int16, device="cuda")
    buf[shift:] = torch.from_numpy(W.view(np.int16).reshape(-1)).cuda()   # shift 1: two bytes off a word
    obs = np.random.default_rng(n).integers(0, 256, (n, 4, 84, 84), dtype=np.uint8)
    logits = torch.empty((n, 18), dtype=torch.float32, device="cuda")
    act = g.policy(torch.from_numpy(obs).cuda(), buf[shift:], logits=logits)
    act_h, logit_h = o.policy(obs, W, n_threads=8)
    assert np.array_equal(logits.cpu().numpy().view(np.uint32), logit_h.view(np.uint32))
    assert np.array_equal(act.cpu().numpy(), act_h)
