"""A state may be loaded any number of cycles past its frame's first line; one
instruction then runs before the line cap ends the frame, and what it does at
that cycle (an object's position, the HMOVE bar, the collisions so far, a
frame end) is computed from the whole cycle count, not from its low half.
Cycle counts on both sides of multiples of 65536, and instructions whose
result depends on the cycle, in every form, against the oracle."""
import numpy as np
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, FORM_PLAIN
from paper_1907_08467_gb300.synth.asm6502 import assemble
from paper_1907_08467_gb300.synth.roms import Rom

from tests.test_gpu_parity import assert_same, pair

pytestmark = pytest.mark.gpu

SRC = """
Reset:  CLD
        LDX #$FF
        TXS
        STX GRP0
        STX PF1
        STX HMP0
        LDA #$42
        STA COLUP0
Frame:  LDA #2
        STA VSYNC
        STA WSYNC
        LDA #0
        STA VSYNC
        LDY #200
Line:   STA WSYNC
        STY COLUBK
        DEY
        BNE Line
        JMP Frame
At0:    STA RESP0
        JMP Frame
At1:    STA HMOVE
        JMP Frame
At2:    LDA CXP0FB
        STA $90
        JMP Frame
At3:    INC RESM1
        JMP Frame
At4:    STX VSYNC
        JMP Frame
At5:    STA CXCLR
        JMP Frame
At6:    STA WSYNC
        JMP Frame
At7:    INC $91
        JMP Frame
"""
LATE = [30399, 30400, 65529, 65530, 65531, 65532, 65533, 65534, 65535, 65536, 65537, 65600, 70001, 87381, 131067,
        131070, 131072, 200001, 1 << 20, (1 << 24) + 77]
FORMS = {
    "plain": dict(form=FORM_PLAIN),
    "batched-32": dict(form=FORM_BATCHED, envs_per_warp=32, envs_per_block=64, tia_warps=1),
    "batched-1": dict(form=FORM_BATCHED, envs_per_warp=1, envs_per_block=2, tia_warps=1),
    "split-32": dict(form=FORM_BATCHED, envs_per_warp=32, envs_per_block=64, tia_warps=2),
    "split-3": dict(form=FORM_BATCHED, envs_per_warp=3, envs_per_block=6, tia_warps=2),
}


@pytest.mark.parametrize("form", list(FORMS))
def test_cycles_past_sixteen_bits_match_oracle(form):
    img, sym = assemble(SRC + "\n        .org $FFFA\n        .word Reset, Reset, Reset\n")
    rom = Rom("late", bytes(img), 0x82, 0xF0)
    pcs = [sym[f"At{k}"] for k in range(8)]
    n = len(LATE) * len(pcs)
    g, o = pair([rom], [0] * n, startup_frames=3, max_noops=5, **FORMS[form])
    st = o.state()
    line = st[:, 0x50:0x58].copy().view(np.uint64)[:, 0]
    at = np.array([c for c in LATE for _ in pcs], np.uint64)
    st[:, 0x08:0x10].view(np.uint64)[:, 0] = 76 * line + at
    st[:, 0x06:0x08].view(np.uint16)[:, 0] = np.array(pcs * len(LATE), np.uint16)
    g.set_state(torch.from_numpy(st).cuda())
    o.set_state(st)
    acts = synth.actions(97, 2, n)
    for s in range(2):
        obs, rew, done = g.step(torch.from_numpy(acts[s]).cuda())
        oo, orw, od = o.step(acts[s])
        assert_same(f"step {s} rewards", rew.cpu().numpy(), orw)
        assert_same(f"step {s} dones", done.cpu().numpy(), od)
        assert_same("state", g.state().cpu().numpy(), o.state())
        assert_same(f"step {s} obs", obs.cpu().numpy(), oo)
