"""GPU parity of the branch-free interpreter at the places where its hot loop
hands over: event-queue pressure (a TIA write in every instruction for whole
lines), frames that end at the line cap, branches and indexed reads across
pages, zero-page wrap, code that runs into a bank's last bytes, instructions
of the general decoder between hot ones, and states loaded at a cycle count
past the line cap.  Batched (one warp) and split (paired warps) forms,
ragged lanes; every output equals the oracle."""
import numpy as np
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED
from paper_1907_08467_gb300.synth.asm6502 import assemble
from paper_1907_08467_gb300.synth.roms import Rom

from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu

# every visible line is one run of TIA stores, more than a queue's 32 entries between two reads
STORES = "".join(f"        STA ${r:02X}\n" for r in (0x06, 0x07, 0x08, 0x09, 0x0D, 0x0E, 0x0F, 0x1B, 0x1C, 0x1D,
                                                     0x1E, 0x1F, 0x10, 0x12, 0x14, 0x2A, 0x25, 0x28, 0x0A, 0x04))
FLOOD = f"""
Reset:  CLD
        LDX #$FF
        TXS
Frame:  LDA #2
        STA VSYNC
        STA WSYNC
        STA WSYNC
        STA WSYNC
        LDA #0
        STA VSYNC
        LDY #100
Line:   LDA $80,X
        EOR $81
        ROR
        STA $80
        INC $81
{STORES}{STORES}        LDA CXPPMM
        ORA CXBLPF
        EOR $82
        STA $82
        INX
        DEY
        BNE Line
        JMP Frame
"""
# no VSYNC: every frame ends at the line cap; stack and pointer instructions between hot ones, wrapping zero page,
# page-crossing branches and reads
CAPPED = """
Reset:  SED
        LDX #$FF
        TXS
        LDA #$F8
        STA $91
        LDA #$F0
        STA $90
Loop:   LDA ($90),Y
        ADC $80,X
        STA $7F,X
        PHA
        PHP
        INC $88,X
        JSR Sub
        PLP
        PLA
        SBC ($F0,X)
        DEX
        INY
        STA WSYNC
        STA COLUBK
        JMP Far
        .org $F0FA
Sub:    LDA $F0F0,Y
        BMI Back
        BNE Back
Far:    LDA SWCHA
        STA $95
        CPX #$81
        BCC Wrap
        BCS Wrap
Back:   ROL $96
        RTS
Wrap:   JMP Loop
"""


def _rom(src, name, size=4096):
    img, _ = assemble(src + "\n        .org $FFFA\n        .word Reset, Reset, Reset\n")
    return Rom(name, bytes(img), 0x82, 0xFF)


def _edge_rom():
    """F8 cartridge whose code runs through the bytes below the hotspots: the last hot fetch, then the general one."""
    bank = bytearray(b"\xEA" * 4096)                       # NOPs
    code = [0xA9, 0x02, 0x85, 0x00, 0x85, 0x02, 0xA9, 0x00, 0x85, 0x00, 0xE6, 0x80, 0xA5, 0x80, 0x85, 0x09,
            0x4C, 0x00, 0xFE]                              # frame start, INC $80, STA COLUBK, JMP $FE00
    bank[0:len(code)] = bytes(code)
    for a in (0xFE40, 0xFE80, 0xFF10):                     # WSYNC and colour on the way to the end of the bank
        bank[a & 0xFFF:(a & 0xFFF) + 4] = bytes([0x85, 0x02, 0x86, 0x06])
    bank[0xFF0:0xFF3] = bytes([0xE6, 0x81, 0xE8])          # INC $81, INX, then NOPs into $FF8/$FF9: bank switches
    bank[0xFF3:0xFFA] = bytes([0xEA, 0xA5, 0x81, 0x85, 0x08, 0xEA, 0xEA])
    bank[0xFFA:0x1000] = bytes([0x4C, 0x00, 0xF0, 0xF0, 0x00, 0xF0])  # JMP $F000; reset vector $F000
    bank[0xFFC:0xFFE] = bytes([0x00, 0xF0])
    return Rom("edge-f8", bytes(bank) * 2, 0x80, 0xFF)


SHAPES = {
    "split-32": dict(envs_per_warp=32, envs_per_block=64, tia_warps=2),
    "split-3": dict(envs_per_warp=3, envs_per_block=6, tia_warps=2),
    "batched-32": dict(envs_per_warp=32, envs_per_block=64, tia_warps=1),
    "batched-1": dict(envs_per_warp=1, envs_per_block=2, tia_warps=1),
}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("which", ["flood", "capped", "edge"])
def test_hot_loop_edges_match_oracle(which, shape):
    rom = {"flood": lambda: _rom(FLOOD, "flood"), "capped": lambda: _rom(CAPPED, "capped"), "edge": _edge_rom}[which]()
    n = 37
    g, o = pair([rom], [0] * n, form=FORM_BATCHED, startup_frames=3, max_noops=5, **SHAPES[shape])
    run_parity(g, o, synth.actions(91, 3, n))


@pytest.mark.parametrize("shape", ["split-32", "batched-32"])
def test_states_past_the_line_cap_match_oracle(shape):
    """A loaded state may stand past the 400-line cap: one instruction runs, then the frame ends."""
    rom = synth.rom_sprite(3)
    n = 33
    g, o = pair([rom], [0] * n, form=FORM_BATCHED, **SHAPES[shape])
    st = o.state()
    line = st[:, 0x50:0x58].copy().view(np.uint64)[:, 0]
    cyc = st[:, 0x08:0x10].view(np.uint64)
    cyc[:, 0] = 76 * (line + np.arange(n, dtype=np.uint64) * 20) + 5   # 0 .. 640 lines into the frame
    g.set_state(torch.from_numpy(st).cuda())
    o.set_state(st)
    acts = synth.actions(92, 2, n)
    for s in range(2):
        obs, rew, done = g.step(torch.from_numpy(acts[s]).cuda())
        oo, orw, od = o.step(acts[s])
        assert np.array_equal(rew.cpu().numpy(), orw) and np.array_equal(done.cpu().numpy(), od)
        assert np.array_equal(g.state().cpu().numpy(), o.state())
        assert np.array_equal(obs.cpu().numpy(), oo)
