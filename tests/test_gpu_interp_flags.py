"""GPU parity of the hot loop's flag word, branch sums and address table: the
overflow flag through ADC, SBC, CLV, BVC and BVS, rotates and compares before
each kind of branch, taken and not, within and across pages; RAM, TIA and
cartridge addresses at the edges of what the loop takes (mirrors, zero-page
wrap, indexed stores below RAM); a branch whose target wraps past the end of
the address space.  Every output equals the oracle."""
import pytest

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED
from paper_1907_08467_gb300.synth.asm6502 import assemble
from paper_1907_08467_gb300.synth.roms import Rom

from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu

# every pair of operands from a walk through RAM, the outcome of each branch counted in a RAM byte of its own
FLAGS = """
Reset:  CLD
        LDX #$FF
        TXS
Frame:  LDA #2
        STA VSYNC
        STA WSYNC
        LDA #0
        STA VSYNC
        LDY #150
Line:   LDA $A0
        ADC $A1
        STA $A0
        BVC V1
        INC $90
V1:     BVS V2
        INC $91
V2:     SBC $A2
        STA $A1
        BVS V3
        INC $92
V3:     CLV
        BVS V4
        ROR $A2
V4:     BVC V5
        INC $93
V5:     CMP $A0
        BCC C1
        INC $94
C1:     BCS C2
        ROL $A1
C2:     EOR $A2
        BMI N1
        INC $95
N1:     BPL N2
        LSR
N2:     BEQ Z1
        INC $96
Z1:     BNE Z2
        INC $A0
Z2:     ADC SWCHA
        STA $A2
        STA COLUBK
        DEX
        DEY
        BEQ End
        JMP Line
End:    JMP Frame
"""
# page-crossing branches back and forth, mirrored RAM and TIA addresses, stores indexed across RAM's edges, and at
# $FFF0 a branch to $0071: the bus there reads zeros, so a BRK leads back through the vector
EDGES = """
Reset:  CLD
        LDX #$FF
        TXS
        LDA #2
        STA VSYNC
        STA WSYNC
        LDA #0
        STA VSYNC
        LDY #90
Line:   INC $80
        LDX $80
        LDA $F000,X
        STA $70,X
        STA $F0,X
        STA $0180,Y
        LDA $0080,Y
        STA $0109
        STA $49
        ROL $0180
        LDA $0580
        STA $8F
        JMP Up
        .org $F0F0
Up:     LDA $80
        BPL Over
        BMI Over
Back:   DEY
        STA WSYNC
        BEQ Out
        JMP Line
Out:    LDA $F1F8,X
        JMP Tail
        .org $F110
Over:   STA COLUPF
        CLC
        BCC Back
        .org $FFE0
Tail:   LDX #0
        LDA #1
        JMP Last
        .org $FFF0
Last:   .byte $D0, $7F
        JMP Reset
"""
SHAPES = {
    "split-32": dict(envs_per_warp=32, envs_per_block=64, tia_warps=2),
    "split-5": dict(envs_per_warp=5, envs_per_block=10, tia_warps=2),
    "batched-32": dict(envs_per_warp=32, envs_per_block=32, tia_warps=1),
    "batched-1": dict(envs_per_warp=1, envs_per_block=3, tia_warps=1),
}


def rom(src, name):
    img, _ = assemble(src + "\n        .org $FFFA\n        .word Reset, Reset, Reset\n")
    return Rom(name, bytes(img), 0x82, 0xFF)


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("which", ["flags", "edges"])
def test_flags_branches_and_addresses_match_oracle(which, shape):
    r = rom(FLAGS, "flags") if which == "flags" else rom(EDGES, "edges")
    n = 37
    g, o = pair([r], [0] * n, form=FORM_BATCHED, startup_frames=3, max_noops=5, **SHAPES[shape])
    run_parity(g, o, synth.actions(93, 3, n))
