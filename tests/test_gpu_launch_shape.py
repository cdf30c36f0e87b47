"""The launch shape that an env reports is the one that it launches, and can
be asked for: in the plain form one env a warp while that is the faster, else
full warps, in blocks of two warps; in the batched form blocks of up to eight
CPU warps (256 envs), the largest that the autotuner tries, with ragged last
items, checked against the oracle."""
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, FORM_PLAIN, OUT_PALETTE, AtariEnv, AtariError

from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [-1, 0, 1])
def test_plain_form_reports_its_grid(over):
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count + over
    r = synth.rom_playfield(2)
    g = AtariEnv([r.data], [(r.score_addr, r.gameover_addr)], [0] * n, form=FORM_PLAIN, output_mode=OUT_PALETTE,
                 startup_frames=1, max_noops=1, n_cache=1, log_cap=256)
    lanes = 32 if over > 0 else 1
    assert g.launch_shape() == (lanes, 2 * lanes, 1, -(-n // (2 * lanes)), 1, 1)


@pytest.mark.parametrize("kind,n,lanes,block,tia_warps", [
    ("4k", 257, 32, 256, 2),    # an item of one env after a full one
    ("f6", 513, 32, 256, 2),
    ("f6", 255, 32, 256, 2),    # a last lane without an env
    ("4k", 70, 5, 40, 2),
    ("f6", 300, 32, 256, 1),
    ("f4", 200, 32, 224, 2),    # cut: six warps and their eight banks' stage fill the shared memory
])
def test_blocks_of_eight_warps_match_oracle(kind, n, lanes, block, tia_warps):
    rom = synth.rom_banked(9, kind)
    g, o = pair([rom], [0] * n, form=FORM_BATCHED, sticky=True, startup_frames=3, max_noops=5, seed=4,
                envs_per_warp=lanes, envs_per_block=block, tia_warps=tia_warps)
    shape = g.launch_shape()
    assert shape[:2] == (lanes, 192 if kind == "f4" else block) and shape[4] == tia_warps
    run_parity(g, o, synth.actions(98, 2, n))


def test_reported_shapes_can_be_asked_for():
    n, rom = 4096, synth.rom_sprite(5)

    def make(**kw):
        g = AtariEnv([rom.data], [(rom.score_addr, rom.gameover_addr)], [0] * n, luma=synth.luma_table(),
                     form=FORM_BATCHED, startup_frames=1, max_noops=1, n_cache=1, **kw)
        return g.launch_shape()

    auto = make()
    assert make(envs_per_warp=auto[0], envs_per_block=auto[1], tia_warps=auto[4])[:5] == auto[:5]
    assert make(envs_per_warp=32, envs_per_block=256, tia_warps=2)[:2] == (32, 256)
    with pytest.raises(AtariError):
        make(envs_per_warp=32, envs_per_block=257)
