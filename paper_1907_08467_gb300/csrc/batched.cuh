// Batched form: persistent ROM-grouped interpreter and fused replay +
// preprocessing.
//
// Interpreter: envs are grouped by cartridge into work items of E envs
// (E = warps per block x envs per warp; a warp may run fewer than 32 envs,
// which trades SIMT width for more independent instruction streams when the
// batch is small).  Each block takes work items from an atomic queue, stages
// the item's cartridge in shared memory when it differs from the one it
// holds, and runs every env of the item for the whole step.
//
// Fused replay + preprocessing (the paper's TIA kernel with the rows of a
// frame spread over several warps, followed by the agent's preprocessing):
// one block per env paints frame F over frame F-1 in shared memory, as the
// pixelwise maximum of their lumas, resamples to 84x84 and pushes the plane
// into the env's stack; frames never reach HBM.
#pragma once
#include <cstdint>

#include "device_machine.cuh"
#include "fast_console.cuh"
#include "paint.cuh"
#include "render.cuh"

namespace atari {

struct BatchArgs {
  uint8_t *state;
  const uint8_t *cache;
  const uint8_t *romb;       // [n_roms][ROMB_SLOT] cartridge bytes, banks of 4096
  const uint32_t *info;      // per ROM: scheme | score << 8 | gameover << 16 | banks << 24
  const uint8_t *dec_op;     // DEC_BYTES: op per opcode, mode/cycles/penalty per opcode, control words
  const uint8_t *actions;
  int32_t *rew_int;
  uint8_t *done_int;
  int32_t *rew_out;
  uint8_t *done_out;
  uint32_t *log;
  uint8_t *bsnap;            // [n][logged frames][BANDS][BAND_SNAP] band start snapshots
  uint32_t *meta;
  uint32_t *counters;
  const int32_t *grp_rom, *grp_start, *grp_count, *perm;
  const int32_t *opos;       // null, or the packed action/output position of each work-list entry
  int *queue;
  int n_groups, lanes, E, rom_stage;  // rom_stage: bytes of the largest cartridge
  int frameskip, sticky, n_cache, log_cap, first_slot;
  int tia_off;               // split form test mode: the TIA side takes no events
  int idle;                  // retire RIOT-timer wait-loop iterations at once
  int unit;                  // 1
  uint64_t seed;
};

__device__ __forceinline__ void fast_reset_from_cache(uint8_t *st, const uint8_t *cache, uint32_t score,
                                                      uint32_t rom, uint32_t n_cache, uint64_t seed,
                                                      uint32_t env_key, uint32_t episode) {
  uint32_t idx = scale32(philox_x0(seed, env_key, 0u, PURPOSE_RESET << 8, episode), n_cache);
  const uint8_t *src = cache + ((size_t)rom * n_cache + idx) * 256;
  const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
  uint4 *d4 = reinterpret_cast<uint4 *>(st);
#pragma unroll
  for (int i = 0; i < 6; ++i) d4[i] = s4[i];
#pragma unroll
  for (int i = 8; i < 16; ++i) d4[i] = s4[i];
  st[S::LAST_ACTION] = 0;
  st[S::SCORE_PREV] = src[S::RAM + score];
  *reinterpret_cast<uint32_t *>(st + S::EPISODE) = episode;
}

// Where the TIA side of env slot i leaves its logs and snapshots.
__device__ __forceinline__ TiaOut tia_out_of(const BatchArgs &a, int i) {
  const long long frame = (long long)i * (2 - a.first_slot) - a.first_slot;  // frames before this env's frame F-1
  return TiaOut{a.log + (size_t)i * 2 * a.log_cap, a.bsnap + frame * (long long)(BANDS * BAND_SNAP),
                a.meta + (size_t)i * 4, (uint32_t)a.log_cap};
}

// The frames of one env's step: the action of each frame (sticky draws), the
// logged frames' marks, and the reward.
template <bool SPLIT>
struct StepHook {
  const BatchArgs *a;
  uint32_t score;
  uint32_t env_key, step_no, episode, action, last, score_prev;
  int32_t reward;
  int f;

  __device__ void start_frame(FastConsoleT<SPLIT> &m) {
    uint32_t act = action;
    if (a->sticky) {
      const uint32_t u = philox_x0(a->seed, env_key, step_no, (uint32_t)f | PURPOSE_STICKY << 8, episode);
      if (u < 0x40000000u) act = last;
    }
    last = act;
    m.apply_action(act);
    const int slot = f - (a->frameskip - 1);
    if (slot >= a->first_slot) m.push(EV_BEGIN_LOG | (uint32_t)slot);
  }
  __device__ bool frame_done(FastConsoleT<SPLIT> &m) {
    const int slot = f - (a->frameskip - 1);
    if (slot >= a->first_slot) m.push(EV_END_LOG | (uint32_t)slot);
    const uint32_t s = m.ram(score);
    reward += (int32_t)(int8_t)(uint8_t)(s - score_prev);
    score_prev = s;
    if (f == a->frameskip) return false;
    ++f;
    start_frame(m);
    return true;
  }
};

// Env slot i; o = where its action is read and its reward and done written.
// Split form: the step ends once the TIA side has caught up.
template <bool SPLIT>
__device__ __forceinline__ void fast_step_env(FastConsoleT<SPLIT> &m, uint8_t *st, int i, int o, const BatchArgs &a, uint32_t rom, uint32_t score,
                                              uint32_t gameover) {
  const uint32_t *ew = reinterpret_cast<const uint32_t *>(st + S::EPISODE);
  uint32_t env_status = ew[3];
  uint32_t action = a.actions[o];
  if (action >= 18) { env_status |= ST_BAD_ACTION; action = 0; }
  StepHook<SPLIT> h{&a, score, ew[2], ew[1], ew[0], action, st[S::LAST_ACTION], st[S::SCORE_PREV], 0, 1};
  h.start_frame(m);
  m.run(h);
  if constexpr (SPLIT) {
    m.push(EV_STEP_END);
    if (!m.broken && !fc_q_wait_ack(m.io, m.nreq + 1)) m.stall();
  } else {
    m.drain();
  }
  env_status |= m.all_status();
  if (m.jam) env_status |= ST_ILLEGAL;
  const uint32_t done = (m.ram(gameover) != 0 || m.jam) ? 1u : 0u;
  a.rew_int[i] = h.reward;
  a.done_int[i] = (uint8_t)done;
  if (a.rew_out) a.rew_out[o] = h.reward;
  if (a.done_out) a.done_out[o] = (uint8_t)done;
  if (a.counters) {
    a.counters[3 * i] = m.instret;
    a.counters[3 * i + 2] = m.rounds;
    if constexpr (!SPLIT) a.counters[3 * i + 1] = m.ts.log_total;
  }
  uint32_t *ewo = reinterpret_cast<uint32_t *>(st + S::EPISODE);
  ewo[1] = h.step_no + 1;
  ewo[3] = env_status;
  if (done) {
    fast_reset_from_cache(st, a.cache, score, rom, (uint32_t)a.n_cache, a.seed, h.env_key, h.episode + 1);
  } else {
    m.store(st);
    st[S::LAST_ACTION] = (uint8_t)h.last;
    st[S::SCORE_PREV] = (uint8_t)h.score_prev;
  }
}

// TIA side of the split form for env slot i: applies the CPU side's events in
// order until the end of the step.  Every wait is bounded; running out sets
// ST_STALL and ends the loop.
__device__ void tia_worker(IoCtx c, uint32_t q, const uint8_t *st, int i, const BatchArgs &a) {
  if (a.tia_off) return;
  const TiaOut out = tia_out_of(a, i);
  const uint64_t l0 = *reinterpret_cast<const uint64_t *>(st + S::FRAME_LINE);
  const uint64_t cycles = *reinterpret_cast<const uint64_t *>(st + S::CYCLES);
  TiaSide s = tia_start(c, l0, (uint32_t)(cycles - 76ull * l0));
  uint64_t idle_since = 0;  // global-timer time the queue was first seen empty (0: not idle)
  for (;;) {
    const uint32_t ev = vsm32(q + 4 * (s.head & (QLEN - 1)));
    if ((ev ^ lap_bit(s.head)) & EV_LAP) {
      const uint64_t now = global_ns();
      if (!idle_since) idle_since = now;
      else if (now - idle_since >= WAIT_NS) {
        s.status |= ST_STALL;
        c.Sset(IO_STATUS, s.status);
        break;
      }
      __nanosleep(128);  // an idle TIA lane polls gently: the CPU warps share the SM's memory pipe
      continue;
    }
    idle_since = 0;
    ++s.head;
    __threadfence_block();  // the entry is read before its place is given back
    c.V(IO_QHEAD) = s.head;
    const uint32_t r = tia_event(c, ev, s, out);
    if (r) {
      c.Sset(IO_CX, s.cx);
      if (r & TIA_END) {
        c.Sset(IO_STATUS, s.status);
        if (a.counters) a.counters[3 * i + 1] = s.log_total;
      }
      __threadfence_block();
      c.V(IO_ACK) = ++s.ack;
      if (r & TIA_END) break;
    }
  }
}

// Shared memory of a block: the tables, the envs' RAM, the cartridge stage, then
// per env I/O words, TIA file and event queue.
__device__ __forceinline__ EnvOff env_off(uint32_t rom_stage, uint32_t envs, uint32_t j) {
  EnvOff o;
  o.rom = OFF_RAM + ram_part(envs);
  const uint32_t io = o.rom + 4 * rom_stage, tia = io + 4 * IO_STRIDE * envs, q = tia + TIA_STRIDE * envs;
  o.ram = OFF_RAM + j / 4 * RAM_GROUP + j % 4;
  o.io = io + 4 * IO_STRIDE * j;
  o.tia = tia + TIA_STRIDE * j;
  o.q = q + 4 * QSTRIDE * j;
  return o;
}
// Stage a cartridge (banks of 4096 bytes at src, 4-byte aligned) for a block of
// envs and its region table with the whole block.
__device__ __forceinline__ void stage_cartridge(const uint8_t *src, uint32_t banks, uint32_t scheme, uint32_t envs) {
  const uint32_t limit = scheme_fetch_limit(scheme);
  for (uint32_t g = threadIdx.x; g < banks * 1024u; g += blockDim.x)
    reinterpret_cast<uint4 *>(g_smem + OFF_RAM + ram_part(envs))[g] = stage_words(src + (g >> 10) * 4096u, 4u * (g & 1023u), limit);
  for (uint32_t p = threadIdx.x; p < REGION_BYTES / 4; p += blockDim.x) {
    uint32_t w = 0;
    for (uint32_t b = 0; b < 4; ++b) w |= region_byte(4 * p + b, scheme) << (8 * b);
    sm32(OFF_REG + 4 * p) = w;
  }
}
// blockDim = W warps (single-warp form) or 2 W (split form); warps [0, W) run
// the CPUs of the work item's envs, in the split form warp W + w the TIA side
// of CPU warp w's envs (lane for lane).
template <bool SPLIT>
__device__ __forceinline__ void interp_block(const BatchArgs &a) {
  __shared__ int s_group;
  for (uint32_t t = threadIdx.x; t < DEC_BYTES / 4; t += blockDim.x)
    sm32(OFF_DEC + 4 * t) = reinterpret_cast<const uint32_t *>(a.dec_op)[t];
  int cur_rom = -1;
  const int W = a.E / a.lanes;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool cpu = warp < W;
  const int cw = cpu ? warp : warp - W;
  for (;;) {
    __syncthreads();  // everyone is done with the previous item (cartridge, s_group)
    if (threadIdx.x == 0) s_group = atomicAdd(a.queue, 1);
    __syncthreads();
    const int g = s_group;
    if (g >= a.n_groups) break;
    const int rom = a.grp_rom[g];
    const uint32_t inf = a.info[rom];
    if (rom != cur_rom) {
      stage_cartridge(a.romb + (size_t)rom * ROMB_SLOT, inf >> 24, inf & 0xFF, (uint32_t)a.E);
      cur_rom = rom;
    }
    const int jj = cw * a.lanes + lane;
    const bool runs = lane < a.lanes && jj < a.grp_count[g];
    const uint32_t wmask = __ballot_sync(0xFFFFFFFFu, runs);
    const int p = a.grp_start[g] + jj;
    const int i = runs ? a.perm[p] : 0;
    const int o = runs ? (a.opos ? a.opos[p] : i) : 0;
    uint8_t *st = a.state + (size_t)i * 256;
    const EnvOff off = env_off((uint32_t)a.rom_stage, (uint32_t)a.E, (uint32_t)jj);
    FastConsoleT<SPLIT> m;
    if (cpu && runs) {
      m.attach(off);
      m.scheme = inf & 0xFF;
      m.wmask = wmask;
      m.idle = (uint32_t)a.idle;
      m.unit = (uint32_t)a.unit;
      m.to = tia_out_of(a, i);
      m.load(st);
    }
    __syncthreads();  // the cartridge and the envs' state are in shared memory
    if (runs) {
      if (cpu) fast_step_env<SPLIT>(m, st, i, o, a, (uint32_t)rom, (inf >> 8) & 0x7F, (inf >> 16) & 0x7F);
      else tia_worker(IoCtx{off.tia, off.io}, off.q, st, i, a);
    }
  }
}
__global__ void __launch_bounds__(256, 1) k_interp_batched(const __grid_constant__ BatchArgs a) { interp_block<false>(a); }
__global__ void __launch_bounds__(512, 1) k_interp_split(const __grid_constant__ BatchArgs a) { interp_block<true>(a); }

// Bank-aware grouping: within each cartridge's run [seg[r], seg[r+1]) of the
// env list, envs are ordered by the bank their canonical state holds at the
// start of the step (byte 5, reduced to the cartridge's bank bits), stable in
// env order, so the lanes of a warp start the step in one bank.  A counting
// sort with up to eight keys (F4); one block of 256 threads per cartridge.
// Cartridges with one bank keep the list as it is.
__global__ void __launch_bounds__(256) k_group_by_bank(const uint8_t *state, const int32_t *perm_in,
                                                        const int32_t *seg, const uint32_t *info, int32_t *perm_out) {
  constexpr uint32_t KEYS = 8;
  const int r = blockIdx.x;
  const int a = seg[r], b = seg[r + 1];
  const uint32_t banks = info[r] >> 24;
  if (banks <= 1) {
    for (int p = a + (int)threadIdx.x; p < b; p += blockDim.x) perm_out[p] = perm_in[p];
    return;
  }
  const uint32_t mask = banks - 1;  // 1 for F8, 3 for F6, 7 for F4
  __shared__ int cnt[KEYS], base[KEYS], wcnt[8][KEYS];
  if (threadIdx.x < KEYS) cnt[threadIdx.x] = 0;
  __syncthreads();
  for (int p = a + (int)threadIdx.x; p < b; p += blockDim.x)
    atomicAdd(&cnt[state[(size_t)perm_in[p] * 256 + 5] & mask], 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = a;
    for (uint32_t v = 0; v < KEYS; ++v) { base[v] = s; s += cnt[v]; }
  }
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int p0 = a; p0 < b; p0 += blockDim.x) {
    const int p = p0 + (int)threadIdx.x;
    const bool valid = p < b;
    const int env = valid ? perm_in[p] : 0;
    const uint32_t bk = valid ? (state[(size_t)env * 256 + 5] & mask) : 0u;
    uint32_t rank = 0;
#pragma unroll
    for (uint32_t v = 0; v < KEYS; ++v) {
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, valid && bk == v);
      if (lane == 0) wcnt[warp][v] = __popc(m);
      if (valid && bk == v) rank = __popc(m & ((1u << lane) - 1u));
    }
    __syncthreads();
    if (valid) {
      int off = 0;
      for (uint32_t w2 = 0; w2 < warp; ++w2) off += wcnt[w2][bk];
      perm_out[base[bk] + off + (int)rank] = env;
    }
    __syncthreads();
    if (threadIdx.x < KEYS) {
      int t = 0;
      for (int w2 = 0; w2 < 8; ++w2) t += wcnt[w2][threadIdx.x];
      base[threadIdx.x] += t;
    }
    __syncthreads();
  }
}

// Shared memory of the painting kernels: the frame, the threads' register
// files, the tables.  A warp paints 30 bands, 60 rows, which are 24 output rows
// of the resampling, so that warps need not wait for one another.
constexpr int PAINT_BANDS = 30, PAINT_WARPS = 4, PAINT_THREADS = 32 * PAINT_WARPS;
constexpr uint32_t PAINT_FILES = PAINT_FRAME, PAINT_LUT = PAINT_FILES + PAINT_THREADS * FILE_STRIDE;
constexpr uint32_t PAINT_SMEM = PAINT_LUT + PAINT_TABS;
static_assert(PAINT_BANDS * PAINT_WARPS >= (int)BANDS && PAINT_BANDS * BAND_ROWS % 5 == 0, "warps cover the frame in fives of rows");
__device__ __forceinline__ RowPainter painter() {
  RowPainter p;
  p.tabs = PaintTabs{PAINT_LUT + 1024, PAINT_LUT + 1152, PAINT_LUT, PAINT_LUT + 1280};
  p.file = PAINT_FILES + (threadIdx.x & (PAINT_THREADS - 1)) * FILE_STRIDE;
  return p;
}
// Frames first_slot .. 1 (0: F-1, 1: F) of env i, one over the other: this
// thread's band, into the frame in shared memory.
__device__ __forceinline__ void paint_frames(RowPainter &p, int i, int first_slot, const uint32_t *log,
                                             const uint8_t *bsnap, const uint32_t *meta, int log_cap) {
  const uint32_t lane = threadIdx.x & 31, band = (threadIdx.x >> 5) * PAINT_BANDS + lane;
  if (lane >= PAINT_BANDS || band >= BANDS) return;
  const uint32_t r0 = band * BAND_ROWS, r1 = min(r0 + BAND_ROWS, (uint32_t)FRAME_H);
  const uint8_t *snap = bsnap + ((size_t)i * (2 - first_slot) * BANDS + band) * BAND_SNAP;
  if (first_slot == 0) asm volatile("prefetch.global.L1 [%0];" ::"l"(snap + BANDS * BAND_SNAP));
#pragma unroll 1
  for (int slot = first_slot; slot < 2; ++slot) {
    const uint32_t *mt = meta + (size_t)i * 4 + slot * 2;
    const uint32_t *recs = log + ((size_t)i * 2 + slot) * log_cap;
    const uint32_t n_rec = min(mt[0], (uint32_t)log_cap);
    const uint32_t ri = min(p.start(snap), n_rec);
    p.paint(slot != first_slot, r0, r1, mt[1], recs, ri, n_rec, 0);
    snap += BANDS * BAND_SNAP;
  }
}

// One block per env: the rows of frames F-1 and F as luma, their pixelwise
// maximum, 84x84 area resampling, stack push.  Four warps paint; a thread
// paints its rows of frame F-1 and then frame F's over them, so one frame
// (36 KB) is kept and five blocks fit an SM, and a warp resamples its own
// rows.  The fifth warp copies the kept planes meanwhile.
__global__ void __launch_bounds__(PAINT_THREADS + 32, 5)
    k_raster_preprocess(const uint32_t *log, const uint8_t *bsnap, const uint32_t *meta, const uint8_t *luma_g,
                        uint8_t *ring, uint8_t *head, const uint8_t *done, uint8_t *obs, int n, int log_cap,
                        const int32_t *perm, const int32_t *opos, int base) {
  // block b (counted from base) serves env slot perm[b] and writes its stack
  // at position opos[b]
  const int blk = base + (int)blockIdx.x;
  if (blk >= n) return;
  const int i = perm ? perm[blk] : blk;
  const int o = opos ? opos[blk] : i;
  RowPainter p = painter();
  paint_tables(p.tabs, luma_g);
  // Resampling.  Output row i covers source rows [2.5 i, 2.5 i + 2.5), output
  // column j columns [160 j / 84, 160 (j + 1) / 84).  In units of 1/21 column
  // and 1/2 row the weights are whole numbers of at most 21 and 2, and the
  // area's weight is 40 x 5 = 200: out = (sum + 100) / 200, the same value as
  // with 1/84 units and 33600.
  for (uint32_t c = threadIdx.x; c < 84u; c += blockDim.x) {
    uint32_t x0, w0, w1, w2;
    col_weights(c, x0, w0, w1, w2);
    *reinterpret_cast<uint2 *>(&sm32(p.tabs.cols + 8u * c)) = make_uint2(x0, (w0 >> 2) | (w1 >> 2) << 8 | (w2 >> 2) << 16);
  }
  const uint32_t h = head[i];
  const bool finished = done[i] != 0;
  __syncthreads();  // the tables are built and the head is read
  uint8_t *rg = ring + (size_t)i * 4 * 7056;
  uint8_t *ob = obs ? obs + (size_t)o * 4 * 7056 : nullptr;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == PAINT_WARPS) {
    // the three kept planes, oldest first, to the stack; a finished env's ring is cleared
    if (ob) {
      for (int s = 0; s < 3; ++s) {
        const uint4 *src = reinterpret_cast<const uint4 *>(rg + ((h + 1 + s) & 3) * 7056);
        uint4 *dst = reinterpret_cast<uint4 *>(ob + s * 7056);
#pragma unroll 7
        for (uint32_t q = lane; q < 7056 / 16; q += 32) dst[q] = src[q];
      }
    }
    __syncwarp();
    if (finished) {
      uint4 *z = reinterpret_cast<uint4 *>(rg);
      for (uint32_t q = lane; q < 4 * 7056 / 16; q += 32) z[q] = make_uint4(0, 0, 0, 0);
    }
    if (lane == 0) head[i] = finished ? 0 : (uint8_t)((h + 1) & 3);
    return;
  }
  paint_frames(p, i, 0, log, bsnap, meta, log_cap);
  __syncwarp();
  // A lane takes four columns of a pair of output rows (five source rows): a
  // column's three pixels are one byte dot product per source row.
  const uint32_t pairs = PAINT_BANDS * BAND_ROWS / 5, k0 = warp * pairs, nk = min(pairs, 42u - k0);
  uint32_t *out0 = finished ? nullptr : reinterpret_cast<uint32_t *>(rg + h * 7056);
  uint32_t *out1 = ob ? reinterpret_cast<uint32_t *>(ob + 3 * 7056) : nullptr;
  for (uint32_t u = lane; u < 21u * nk; u += 32u) {
    const uint32_t k = k0 + u / 21u, m = u % 21u;
    uint32_t even = 0, odd = 0;
#pragma unroll
    for (uint32_t c = 0; c < 4; ++c) {
      const uint2 col = *reinterpret_cast<const uint2 *>(&sm32(p.tabs.cols + 8u * (4u * m + c)));
      const uint32_t at = col.x & ~3u, sh = col.x * 8u;  // the funnel shift takes it modulo 32
      uint32_t px[5];
#pragma unroll
      for (uint32_t r = 0; r < 5; ++r) {
        const uint32_t a = row_off(5u * k + r) + at;
        px[r] = __funnelshift_r(sm32(a), sm32(a + 4), sh);
      }
      const uint32_t mid = __dp4a(px[2], col.y, 100u), w2 = col.y * 2u;
      even |= __dp4a(px[0], w2, __dp4a(px[1], w2, mid)) / 200u << (8u * c);
      odd |= __dp4a(px[4], w2, __dp4a(px[3], w2, mid)) / 200u << (8u * c);
    }
    const uint32_t q = 42u * k + m;  // word of output row 2 k
    if (out1) { out1[q] = even; out1[q + 21] = odd; }
    if (out0) { out0[q] = even; out0[q + 21] = odd; }
  }
}

// Palette output: one block per env, frame F to the observation.
__global__ void __launch_bounds__(PAINT_THREADS, 5)
    k_raster_palette(const uint32_t *log, const uint8_t *bsnap, const uint32_t *meta, uint8_t *obs, int n, int log_cap) {
  const int i = (int)blockIdx.x;
  if (i >= n) return;
  RowPainter p = painter();
  paint_tables(p.tabs, nullptr);
  __syncthreads();
  paint_frames(p, i, 1, log, bsnap, meta, log_cap);
  __syncwarp();
  uint32_t *dst = reinterpret_cast<uint32_t *>(obs + (size_t)i * (FRAME_H * FRAME_W));
  const uint32_t rows = PAINT_BANDS * BAND_ROWS, q0 = (threadIdx.x >> 5) * rows * 40u;
  const uint32_t q1 = min(q0 + rows * 40u, (uint32_t)(FRAME_H * FRAME_W / 4));
  for (uint32_t q = q0 + (threadIdx.x & 31); q < q1; q += 32) dst[q] = sm32(row_off(q / 40u) + 4u * (q % 40u));
}

}  // namespace atari
