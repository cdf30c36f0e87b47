"""An env's launches do not depend on which other envs or servers exist: a
block's shared memory differs from env to env (cartridge size, envs a block),
and the kernels are shared by all of them.  An env of the largest blocks is
stepped through every kind of launch (a graph captured for new buffers, the
host-buffer step, profiled launches) after envs of small blocks and an
autotuned one were made, and a server goes on ticking while an env is made.
Every output equals the oracle."""
import numpy as np
import pytest
import torch

from paper_1907_08467_gb300 import synth
from paper_1907_08467_gb300.env import FORM_BATCHED, AtariEnv
from paper_1907_08467_gb300.server import AtariServer

from tests.test_gpu_parity import assert_same, pair

pytestmark = pytest.mark.gpu


def _small(tia_warps):
    """Envs of one 4 KB cartridge in blocks of eight, and an autotuned one, which tries every shape."""
    r = synth.rom_playfield(3)
    made = []
    for shape in (dict(envs_per_warp=8, envs_per_block=8, tia_warps=tia_warps), dict(tia_warps=tia_warps)):
        made.append(AtariEnv([r.data], [(r.score_addr, r.gameover_addr)], [0] * 8, luma=synth.luma_table(),
                             form=FORM_BATCHED, startup_frames=3, max_noops=5, **shape))
    return made


@pytest.mark.parametrize("tia_warps", [1, 2])
def test_launches_after_smaller_envs_were_made(tia_warps):
    n = 130
    g, o = pair([synth.rom_banked(23, "f6")], [0] * n, form=FORM_BATCHED, startup_frames=3, max_noops=5,
                envs_per_warp=32, envs_per_block=128, tia_warps=tia_warps)
    acts = synth.actions(95, 4, n)

    def check(out, a):
        got = [x if isinstance(x, np.ndarray) else x.cpu().numpy() for x in out]
        for name, x, y in zip(("obs", "rewards", "dones"), got, o.step(a)):
            assert_same(name, x, y)
        assert_same("state", g.state().cpu().numpy(), o.state())

    check(g.step(torch.from_numpy(acts[0]).cuda()), acts[0])
    others = _small(tia_warps)
    check(g.step(torch.from_numpy(acts[1]).cuda()), acts[1])   # new buffers: a new capture
    check(g.step_host(acts[2]), acts[2])
    g.profile(True)
    check(g.step(torch.from_numpy(acts[3]).cuda()), acts[3])
    g.profile(False)
    for e in others:  # and the small ones go on
        e.step(torch.zeros(e.n, dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()


def test_server_ticks_after_a_smaller_env_was_made():
    n, key = 70, 5 << 11
    r = synth.rom_banked(23, "f6")
    srv = AtariServer.from_roms([r], budget_bytes=1 << 30, max_slots=128, sticky=True, seed=3)
    _, o = pair([r], [0] * n, env_key=[key + i for i in range(n)], form=FORM_BATCHED, sticky=True, seed=3)
    acts = synth.actions(96, 2, n)
    ses = srv.open(0, n, key)
    kept = None
    for a in acts:
        for name, x, y in zip(("obs", "rewards", "dones"), ses.step(a), o.step(a)):
            assert_same(name, np.asarray(x), y)
        kept = kept or _small(2)
    ses.close()
    srv.close()
