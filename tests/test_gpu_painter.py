"""GPU parity of the row painter where its spans and bands have edges: colour,
playfield, blanking and graphics writes that land at every column phase of a
row (first and last bytes of its eight-column groups, several spans in one
group), the HMOVE bar with and without a colour change in its columns, frames
shorter and longer than the 210-row window, and a log that overflows in the
middle of a frame.  Stacks and palette frames equal the oracle's."""
import numpy as np
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, FORM_PLAIN, OUT_PALETTE, OUT_STACK, AtariEnv
from paper_1907_08467_gb300.synth.asm6502 import assemble
from paper_1907_08467_gb300.synth.roms import Rom

from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu


def spans_rom(lines: int, writes: str) -> Rom:
    """`writes` run on every line after a delay that slides through the line by one cycle (three columns) per
    line and, through a three-step of RESP-like phases, by frame; `lines` lines between two VSYNCs."""
    src = f"""
Reset:  CLD
        LDX #$FF
        TXS
        LDA #$35
        STA NUSIZ0
        LDA #$13
        STA NUSIZ1
        LDA #$F0
        STA HMP0
        LDA #$70
        STA HMM1
Frame:  LDA #2
        STA VSYNC
        STA WSYNC
        LDA #0
        STA VSYNC
        INC $80
        LDY #0
Line:   STA WSYNC
        TYA
        AND #3
        BNE NoHm
        STA HMOVE
        STY COLUBK
NoHm:   TYA
        CLC
        ADC $80
        AND #15
        TAX
        LSR
        BCS Odd
Odd:    CPX #2
        BCC Go
        DEX
        BNE Odd
Go:     STX $81
{writes}
        INY
        CPY #{lines}
        BNE Line
        JMP Frame
        .org $FFFA
        .word Reset, Reset, Reset
"""
    img, _ = assemble(src)
    return Rom(f"spans-{lines}", bytes(img), 0x82, 0xFF)


COLOURS = "        STY COLUBK\n        STA COLUPF\n        STY PF1\n        STX COLUBK\n        STA PF2\n        STY VBLANK\n"
OBJECTS = ("        STY GRP0\n        STA GRP1\n        STY ENAM0\n        STY VDELP0\n        STA RESP1\n        STY CTRLPF\n"
           "        STY COLUP0\n        STA REFP1\n        STY RESMP0\n")


@pytest.mark.parametrize("mode", [OUT_STACK, OUT_PALETTE])
@pytest.mark.parametrize("lines,writes", [(230, "colours"), (120, "colours"), (236, "objects"), (250, "objects")])
def test_spans_and_short_frames_match_oracle(lines, writes, mode):
    rom = spans_rom(lines, COLOURS if writes == "colours" else OBJECTS)
    n = 5
    g, o = pair([rom], [0] * n, form=FORM_BATCHED, output_mode=mode, startup_frames=2, max_noops=3,
                envs_per_warp=4, envs_per_block=8, tia_warps=2)
    run_parity(g, o, synth.actions(95, 4, n))


def test_overflowing_log_keeps_state_and_status():
    """Records past log_cap are dropped in every form: the same machine states and the same status."""
    w = synth.workload(2, n_envs=8)
    a = AtariEnv.from_workload(w, form=FORM_PLAIN, log_cap=256)
    b = AtariEnv.from_workload(w, form=FORM_BATCHED, log_cap=256, envs_per_warp=8, envs_per_block=8, tia_warps=2)
    acts = synth.actions(96, 3, 8)
    for s in range(3):
        x = torch.from_numpy(acts[s]).cuda()
        a.step(x)
        obs, _, _ = b.step(x)
        assert torch.equal(a.status(), b.status()) and int(b.status().min()) != 0
        assert torch.equal(a.state(), b.state())
