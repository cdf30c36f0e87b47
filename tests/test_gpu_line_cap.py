"""GPU parity of frames that end at the line cap, in the middle of a program
that never starts one: zero-page wrap in reads and stores, page-crossing reads
and branches, accesses through pointers, stack instructions and a subroutine
between the hot loop's own instructions, in binary and in decimal mode.  The
oracle shows that the program stays on that path: the D flag as it was set,
no env done, every frame at the cap."""
import pytest

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, ST_FRAME_CAP
from paper_1907_08467_gb300.synth.asm6502 import assemble
from paper_1907_08467_gb300.synth.roms import Rom

from tests.test_gpu_interp_core import SHAPES
from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu

# X stays in $C0-$CF and $E0-$EF: stores wrap to TIA registers past WSYNC ($10-$1F, $30-$3F), INC to RAM
SRC = """
Reset:  {mode}
        LDX #$FF
        TXS
        LDA #$F8
        STA $9B
        LDA #$F0
        STA $9A
        LDX #$E5
Loop:   LDA ($9A),Y
        ADC $C0,X
        STA $50,X
        PHA
        PHP
        INC $C8,X
        JSR Sub
        PLP
        PLA
        SBC ($DA,X)
        STA $9C
        DEX
        TXA
        ORA #$C0
        AND #$EF
        TAX
        INY
        STA WSYNC
        STA COLUBK
        JMP Far
        .org $F0FA
Sub:    LDA $F0F0,Y
        BMI Back
        BPL Back
Far:    LDA SWCHA
        EOR $9C
        STA $9D
        CPX #$C7
        BCC Wrap
        BCS Wrap
Back:   ROL $9E
        RTS
Wrap:   JMP Loop
"""


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("mode", ["CLD", "SED"])
def test_frames_at_the_line_cap_match_oracle(mode, shape):
    img, _ = assemble(SRC.format(mode=mode) + "\n        .org $FFFA\n        .word Reset, Reset, Reset\n")
    n = 37
    g, o = pair([Rom("cap", bytes(img), 0x9C, 0xC0)], [0] * n, form=FORM_BATCHED, startup_frames=3, max_noops=5,
                **SHAPES[shape])
    run_parity(g, o, synth.actions(93, 3, n))
    st = o.state()
    assert ((st[:, 0x04] & 0x08 != 0) == (mode == "SED")).all()
    assert not st[:, 0x80 + 0x40].any() and (st[:, 0x6C] == ST_FRAME_CAP).all()
    assert (st[:, 0x58] > st[:, 0x60]).all()   # frames count on: no reset
