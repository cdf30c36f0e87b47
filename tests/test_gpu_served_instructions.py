"""GPU parity of the instructions that the batched interpreter serves beside
its hot loop (accesses through pointers, the stack, BIT, RIOT and TIA
accesses, mirrors, hotspots, decimal arithmetic, undocumented opcodes), in
random order and at random addresses: cartridges of random instructions of
every size, whose lanes drift apart, against the oracle."""
import random

import numpy as np
import pytest

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED
from paper_1907_08467_gb300.synth.asm6502 import ALL_OPCODES
from paper_1907_08467_gb300.synth.roms import Rom

from tests.test_gpu_parity import pair, run_parity

pytestmark = pytest.mark.gpu

OPS = sorted({o for modes in ALL_OPCODES.values() for o in modes.values()} |
             {0x1A, 0x80, 0xC2, 0x04, 0x64, 0x14, 0xF4, 0x0C, 0x1C, 0xFC, 0xEB, 0x2B})
JUMPS = {0x10, 0x30, 0x50, 0x70, 0x90, 0xB0, 0xD0, 0xF0, 0x4C, 0x6C, 0x20, 0x60, 0x40, 0x00}
STRAIGHT, BRANCHES = [o for o in OPS if o not in JUMPS], sorted(JUMPS - {0x40, 0x00, 0x6C})
SHAPES = {
    "split-32": dict(envs_per_warp=32, envs_per_block=64, tia_warps=2),
    "split-3": dict(envs_per_warp=3, envs_per_block=6, tia_warps=2),
    "batched-32": dict(envs_per_warp=32, envs_per_block=64, tia_warps=1),
    "no-idle-skip": dict(envs_per_warp=8, envs_per_block=16, tia_warps=2, idle_skip=0),
}


def _length(o):
    if o == 0x20 or (o & 0x1F) in (0x0C, 0x0D, 0x0E, 0x0F, 0x19, 0x1B, 0x1C, 0x1D, 0x1E, 0x1F):
        return 3
    return 1 if (o & 0x0F) in (0x08, 0x0A) else 2


def random_rom(seed):
    """Random instructions; operands mostly in RAM and at the TIA, absolute ones at mirrors, RIOT and hotspots too."""
    rng = random.Random(seed)
    size = (4096, 4096, 8192, 16384, 32768)[seed % 5]
    b = bytearray()
    while len(b) < size:
        o = rng.choice(STRAIGHT if rng.random() < 0.97 else BRANCHES)
        r = rng.random()
        lo = rng.randrange(0x80, 0x100) if r < 0.5 else rng.randrange(0x80) if r < 0.8 else rng.randrange(256)
        hi = rng.choice([0, 0, 0, 1, 2, 2, 4, 8, 0x0F, 0xF0 + rng.randrange(16), 0xFF, 0x10 + rng.randrange(16), 0x42])
        if hi == 0xFF and rng.random() < 0.5:
            lo = rng.randrange(0xF0, 0x100)
        b += bytes([o, lo, hi][:_length(o)])
    b = b[:size]
    for e in range(0, size, 4096):  # reset and interrupt vectors
        b[e + 0xFFC:e + 0x1000] = bytes([rng.randrange(256), 0xF0 + rng.randrange(15)] * 2)
    return Rom(f"random-{seed}", bytes(b), 0x82, 0xF0)


# seeds whose programs neither halt nor write the game-over byte, and whose envs end up in different states
SEEDS = [(525, 595, 79, 3, 51, 421, 522, 456, 113, 486, 678, 562), (590, 336, 514, 243, 396, 121, 142, 220, 503, 520, 557, 494)]


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("group", [0, 1])
def test_random_instructions_match_oracle(group, shape):
    roms = [random_rom(k) for k in SEEDS[group]]
    per = 35
    n = per * len(roms)
    g, o = pair(roms, [i // per for i in range(n)], form=FORM_BATCHED, startup_frames=2, max_noops=6, **SHAPES[shape])
    run_parity(g, o, np.tile(synth.actions(99, 3, per), (1, len(roms))))
    st = o.state()
    assert not st[:, 0x1E].any() and not st[:, 0x80 + 0x70].any()   # no env has halted or ended
    assert len({x[:8].tobytes() + x[0x80:].tobytes() for x in st}) > n // 4
