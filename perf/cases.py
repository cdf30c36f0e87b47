"""Performance cases: one pass each of the calls a user of this library makes,
over the sizes its configurations, tests and benchmark use.

A case is a dict of plain values.  `prepare` builds what a user's program has
in hand (an env or a server on seeded cartridges, a few steps into its
episodes, and the input buffers), `run` makes one pass through the public
entry points, `work` counts the bytes and operations a pass cannot do
without, and `exact` gives the 64-bit value of the computed (floating-point)
outputs.  Everything random comes from the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1907_08467_gb300.env import (FORM_BATCHED, FORM_PLAIN, OUT_PALETTE, OUT_STACK, AtariEnv, nstep_returns,
                                        vtrace)
from paper_1907_08467_gb300.server import AtariServer
from paper_1907_08467_gb300.synth import luma_table, policy_weights, rom_banked, rom_playfield, rom_sprite

STACK, PLANE, FRAME, STATE, A = 4 * 84 * 84, 84 * 84, 210 * 160, 256, 18
WARM_STEPS = 4   # steps before the first pass: episodes under way, stacks filled


def listed():
    return [
        # the smallest use: 16 envs of one playfield cartridge, raw palette frames out
        dict(name="step_tiny_palette", kind="step", family="playfield", roms=1, rom0=1, n=16, frameskip=4,
             sticky=False, palette=True, form="batched"),
        # an odd, small batch over many cartridges (evaluation: few envs of each game), F8/F6 banking, sticky actions
        dict(name="step_banked_333", kind="step", family="banked", roms=32, rom0=1, n=333, frameskip=4,
             sticky=True, palette=False, form="batched"),
        # the ordinary training batch: 4096 envs over 8 sprite cartridges, 84x84x4 stacks
        dict(name="step_sprite_4096", kind="step", family="sprite", roms=8, rom0=1, n=4096, frameskip=4,
             sticky=False, palette=False, form="batched"),
        # the largest: 32768 envs over 32 banked cartridges with sticky actions (the benchmark's default)
        dict(name="step_banked_32768", kind="step", family="banked", roms=32, rom0=1, n=32768, frameskip=4,
             sticky=True, palette=False, form="batched"),
        # the one-thread-per-env form (the constructor's default), rendered frames kept on the device
        dict(name="step_plain_sprite_1024", kind="step", family="sprite", roms=8, rom0=1, n=1024, frameskip=4,
             sticky=False, palette=False, form="plain"),
        # a learner on the host: actions from, stacks to page-locked host memory; a ragged env count
        dict(name="host_step_sprite_8195", kind="host", family="sprite", roms=8, rom0=1, n=8195, frameskip=4,
             sticky=False, palette=False, form="batched"),
        # the inference loop: policy, step and ring append, two steps, behaviour probabilities kept
        dict(name="rollout_sprite_16384", kind="rollout", family="sprite", roms=16, rom0=1, n=16384, steps=2),
        # the policy alone on full stacks
        dict(name="policy_16384", kind="policy", n=16384),
        # one client of the serving loop: a session's step, host buffers both ways
        dict(name="serve_banked_700", kind="serve", family="banked", roms=6, rom0=1, n=700),
        # learner-side targets over the ring of an N-step learner: a launch-bound call
        dict(name="nstep_5x16384", kind="nstep", T=5, n=16384),
        # off-policy targets over a long rollout of the largest batch
        dict(name="vtrace_60x32768", kind="vtrace", T=60, n=32768),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["host", "rollout", "policy", "serve", "nstep", "vtrace"])
    if kind in ("nstep", "vtrace"):
        n = _log_int(rng, 64, 32768)
        return dict(kind=kind, T=_log_int(rng, 1, 60), n=n)
    if kind == "policy":
        return dict(kind=kind, n=_log_int(rng, 16, 16384))
    family = rng.choice(["playfield", "sprite", "banked", "banked_f4"])
    rom0 = rng.randrange(1, 60)
    if kind == "serve":
        return dict(kind=kind, family=family, roms=rng.randrange(1, 7), rom0=rom0, n=_log_int(rng, 1, 2048))
    if kind == "rollout":
        n = _log_int(rng, 32, 16384)
        return dict(kind=kind, family=family, roms=rng.randrange(1, min(16, n) + 1), rom0=rom0, n=n,
                    steps=rng.randrange(1, 3))
    plain = kind == "step" and rng.random() < 0.15
    n = _log_int(rng, 1, 1024 if plain else 8195 if kind == "host" else 32768)
    return dict(kind=kind, family=family, roms=rng.randrange(1, min(32, n) + 1), rom0=rom0, n=n,
                frameskip=rng.choice([2, 3, 4, 4, 4]), sticky=rng.random() < 0.5,
                palette=kind == "step" and rng.random() < 0.25, form="plain" if plain else "batched")


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _rom(family, k):
    if family == "playfield":
        return rom_playfield(k)
    if family == "sprite":
        return rom_sprite(k)
    if family == "banked_f4":
        return rom_banked(k, "f4")
    return rom_banked(k, "4k" if k % 32 <= 12 and k % 32 else "f8" if k % 32 <= 22 and k % 32 else "f6")


def _roms(case):
    return [_rom(case["family"], case["rom0"] + j) for j in range(case["roms"])]


@functools.lru_cache(maxsize=None)
def _weights():
    return policy_weights(5).view(np.int16)


def _actions(seed, steps, n):
    return np.random.Generator(np.random.Philox(key=seed)).integers(0, A, size=(steps, n), dtype=np.uint8)


def _env(case, seed):
    roms = _roms(case)
    n, r = case["n"], len(roms)
    return AtariEnv([x.data for x in roms], [(x.score_addr, x.gameover_addr) for x in roms],
                    [i * r // n for i in range(n)], luma=luma_table(), seed=seed,
                    frameskip=case.get("frameskip", 4), sticky=case.get("sticky", False),
                    output_mode=OUT_PALETTE if case.get("palette") else OUT_STACK,
                    form=FORM_PLAIN if case.get("form") == "plain" else FORM_BATCHED)


def _warm(env, acts):
    out = env.alloc_outputs()
    for a in acts:
        env.step(torch.from_numpy(a).cuda(), *out)
    return out


def _obs(seed, n):
    """Stacks with a screen's values: luma levels, mostly the background's."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    lum = torch.tensor(list(luma_table()), dtype=torch.uint8, device="cuda")
    bg = torch.randint(0, 128, (n, 4, 84, 1), generator=g, device="cuda")
    px = torch.randint(0, 128, (n, 4, 84, 84), generator=g, device="cuda", dtype=torch.int16)
    px = torch.where(px < 96, bg.to(torch.int16), px)
    return lum[px.reshape(-1).int()].reshape(n, 4, 84, 84)


def _targets(case, seed):
    """Rewards, dones, behaviour and target probabilities, values of a rollout of T steps kept from ring slot 1 on."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    T, n = case["T"], case["n"]
    rew = torch.randint(-1, 5, (T, n), generator=g, device="cuda").float()
    done = (torch.rand((T, n), generator=g, device="cuda") < 0.02).to(torch.uint8)
    val = torch.randn((T + 1, n), generator=g, device="cuda")
    mu = torch.rand((T, n), generator=g, device="cuda") * 0.9 + 0.05
    pi = (mu * (torch.rand((T, n), generator=g, device="cuda") + 0.5)).clamp(max=1.0)
    return rew, done, val, mu, pi


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("nstep", "vtrace"):
        return dict(kind=kind, T=case["T"], x=_targets(case, seed))
    if kind == "policy":
        r = rom_sprite(1)
        # only the handle's keys and step counters are used: a fixed launch shape, nothing is stepped
        env = AtariEnv([r.data], [(r.score_addr, r.gameover_addr)], [0] * case["n"], luma=luma_table(), seed=seed,
                       form=FORM_BATCHED, envs_per_warp=32, envs_per_block=64, raster_warps_per_frame=4, tia_warps=2)
        return dict(kind=kind, env=env, obs=_obs(seed, case["n"]), w=torch.from_numpy(_weights()).cuda(),
                    act=torch.empty(case["n"], dtype=torch.uint8, device="cuda"),
                    logits=torch.empty((case["n"], A), dtype=torch.float32, device="cuda"))
    n = case["n"]
    acts = _actions(seed, WARM_STEPS + 1, n)
    if kind == "serve":
        srv = AtariServer.from_roms(_roms(case), budget_bytes=2 << 30, max_slots=2048, sticky=True, seed=seed)
        ses = srv.open(seed % case["roms"], n, (seed % 1000) << 11)
        out = (torch.empty((n, 4, 84, 84), dtype=torch.uint8).pin_memory(), np.empty(n, np.int32),
               np.empty(n, np.uint8))
        for a in acts[:-1]:
            ses.step(a, *out)
        return dict(kind=kind, srv=srv, ses=ses, act=acts[-1], out=out)
    env = _env(case, seed)
    if kind == "rollout":
        out = _warm(env, acts[:-1])
        k = case["steps"]
        cu = lambda *s, **kw: torch.zeros(s, device="cuda", **kw)  # noqa: E731
        return dict(kind=kind, env=env, steps=k, w=torch.from_numpy(_weights()).cuda(), out=out,
                    act=cu(n, dtype=torch.uint8),
                    ring=(cu(k, n, PLANE, dtype=torch.uint8), cu(k, n), cu(k, n, dtype=torch.uint8), cu(k, n)))
    if kind == "host":
        out = (torch.empty(env.obs_shape(), dtype=torch.uint8).pin_memory(), torch.empty(n, dtype=torch.int32).pin_memory(),
               torch.empty(n, dtype=torch.uint8).pin_memory())
        for a in acts[:-1]:
            env.step_host(a, *out)
        return dict(kind=kind, env=env, act=torch.from_numpy(acts[-1]).pin_memory(), out=out)
    out = _warm(env, acts[:-1])
    return dict(kind=kind, env=env, act=torch.from_numpy(acts[-1]).cuda(), out=out)


# ------------------------------------------------------------------ one pass

def run(s):
    kind = s["kind"]
    if kind == "nstep":
        rew, done, val, _, _ = s["x"]
        return nstep_returns(rew, done, val, s["T"], 0.99, ring_start=1)
    if kind == "vtrace":
        rew, done, val, mu, pi = s["x"]
        return vtrace(rew, done, mu, val, pi, s["T"], 0.99, ring_start=1)
    if kind == "policy":
        return s["env"].policy(s["obs"], s["w"], s["act"], s["logits"]), s["logits"]
    if kind == "serve":
        return s["ses"].step(s["act"], *s["out"])
    env = s["env"]
    if kind == "host":
        return env.step_host(s["act"], *s["out"])
    if kind == "rollout":
        env.rollout_ex(s["w"], s["steps"], s["out"][0], s["act"], s["out"][1], s["out"][2], *s["ring"])
        return s["out"], s["act"], s["ring"], env.state()
    return env.step(s["act"], *s["out"]), env.state()


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "nstep":   # rewards, dones, values in; returns out
        T = case["T"]
        return {"bytes": n * (T * (4 + 1 + 4) + 4 + T * 4), "flops": 2 * T * n}
    if kind == "vtrace":  # rewards, dones, mu, pi, values in; targets and advantages out
        T = case["T"]
        return {"bytes": n * (T * (4 + 1 + 4 + 4 + 4) + 4 + T * 8), "flops": 15 * T * n}
    policy = {"bytes": n * (STACK + STATE // 8 + 1) + STACK * A * 2, "flops": 2 * STACK * A * n}
    if kind == "policy":
        return {"bytes": policy["bytes"] + n * A * 4, "flops": policy["flops"]}
    # a step: action and machine state in, machine state, reward and done out; a palette frame, or the three kept
    # planes in, the new plane and the ordered stack out
    step = n * (1 + 2 * STATE + 4 + 1 + (FRAME if case.get("palette") else 3 * PLANE + PLANE + STACK))
    if kind == "rollout":  # per step the policy, the step, and the newest plane, reward, done and probability kept
        k = case["steps"]
        return {"bytes": k * (policy["bytes"] + step + n * (2 * PLANE + 9)), "flops": k * policy["flops"]}
    return {"bytes": step, "flops": 0}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("nstep", "vtrace"):
        T = case["T"]
        rew, done, val, mu, pi = _targets(case, seed)
        slot = [(1 + t) % T for t in range(T)]   # step t of the rollout is ring slot (start + t) mod depth
        r, m = rew.double()[slot], mu.double()[slot]
        # the discount is the fp32 number the call is given
        g = torch.where(done[slot] != 0, 0.0, float(np.float32(0.99))).double()
        V, p = val.double(), pi.double()
        if kind == "nstep":
            out, R = torch.empty_like(r), V[T]
            for t in reversed(range(T)):
                R = r[t] + g[t] * R
                out[t] = R
            return out
        vs, adv, v_next = torch.empty_like(r), torch.empty_like(r), V[T]
        for t in reversed(range(T)):
            rho = (p[t] / m[t]).clamp(max=1.0)
            adv[t] = rho * (r[t] + g[t] * v_next - V[t])
            v_next = V[t] + rho * (r[t] + g[t] * V[t + 1] - V[t]) + g[t] * rho * (v_next - V[t + 1])
            vs[t] = v_next
        return vs, adv
    if kind == "policy":
        obs = _obs(seed, case["n"]).reshape(case["n"], STACK)
        w = (torch.from_numpy(_weights()).cuda().to(torch.int32) << 16).view(torch.float32).double().reshape(STACK, A)
        return None, torch.cat([x.double() @ w for x in obs.split(2048)])
    return None
