"""The issue rounds that atari_env_counters sums over the envs are those of an
env's warp, the same on each of its lanes, also where some lanes are in
decimal mode and others are not."""
import numpy as np
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, AtariEnv
from paper_1907_08467_gb300.synth.asm6502 import assemble

pytestmark = pytest.mark.gpu

# decimal arithmetic in the envs whose joystick points right, of a length that depends on the env's frame count
SRC = """
Reset:  CLD
        LDX #$FF
        TXS
Frame:  LDA #2
        STA VSYNC
        STA WSYNC
        LDA #0
        STA VSYNC
        INC $80
        LDA SWCHA
        BMI Plain
        SED
        LDY $80
Dec:    LDA $81
        ADC #7
        STA $81
        DEY
        BNE Dec
        CLD
Plain:  LDY #120
Line:   STA WSYNC
        DEY
        BNE Line
        JMP Frame
"""


@pytest.mark.parametrize("tia_warps", [1, 2])
def test_rounds_are_the_same_on_every_lane(tia_warps):
    img, _ = assemble(SRC + "\n        .org $FFFA\n        .word Reset, Reset, Reset\n")
    g = AtariEnv([bytes(img)], [(0x82, 0xF0)], [0] * 32, luma=synth.luma_table(), form=FORM_BATCHED, startup_frames=2,
                 max_noops=9, envs_per_warp=32, envs_per_block=32, tia_warps=tia_warps)
    right = np.zeros(32, np.uint8)
    right[[3, 4, 17]] = 3
    for a in (np.zeros(32, np.uint8), right):
        g.step(torch.from_numpy(a).cuda())
        ins, _, rounds = g.counters()
        assert rounds % 32 == 0 and 0 < ins <= rounds
