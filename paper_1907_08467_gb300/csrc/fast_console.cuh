// Console for the batched form, laid out for the issue rate of sm_103a.
//
// Same machine and canonical state as Console in device_machine.cuh:
//   - the hot loop is one branch-free sequence for every common instruction,
//     steered by control words per opcode (opcode_ctl.h);
//   - CPU registers, flags, the cycle counter and the bank in registers;
//   - RAM (bytes), the TIA register file (bytes) and the I/O state
//     (collision cursor and latches, RIOT timer and ports, inputs, log
//     cursor, frame base line) in shared memory, one block per env with odd
//     word strides, so lanes reading the same field never bank-conflict and
//     every access is a base offset plus a constant or one add;
//   - the block's cartridge staged in shared memory as bytes (16 KB for an
//     F6 cartridge); an instruction's bytes are fetched as two aligned words
//     joined by one funnel shift.
// Instructions the hot loop does not take (TIA and RIOT reads, RIOT, VSYNC
// and VBLANK writes, stack and pointer instructions, undocumented opcodes,
// decimal arithmetic, fetches outside the cartridge or next to a bank
// hotspot) run the general decoder out of line.
#pragma once
#include <cstdint>

#include "device_machine.cuh"
#include "opcode_ctl.h"

namespace atari {

enum TiaSlot : uint32_t {
  T_VSYNC = 0, T_VBLANK, T_NUSIZ0, T_NUSIZ1, T_COLUP0, T_COLUP1, T_COLUPF, T_COLUBK, T_CTRLPF, T_REFP0,
  T_REFP1, T_PF0, T_PF1, T_PF2, T_ENAM0, T_ENAM1, T_ENABL_N, T_ENABL_O, T_GRP0_N, T_GRP0_O, T_GRP1_N,
  T_GRP1_O, T_VDELP0, T_VDELP1, T_VDELBL, T_RESMP0, T_RESMP1, T_HMP0, T_HMP1, T_HMM0, T_HMM1, T_HMBL,
  T_P0, T_P1, T_M0, T_M1, T_BL
};
// I/O state words (shared memory, interleaved by env)
enum IoWord : uint32_t {
  IO_CEVAL = 0, IO_CX, IO_L0LO, IO_L0HI, IO_BARLO, IO_BARHI, IO_TCWLO, IO_TCWHI, IO_TV, IO_TSH, IO_PORTS,
  IO_JOY, IO_FIRE, IO_LATCH, IO_LOGLO, IO_LOGHI, IO_LOGN, IO_LOGCAP, IO_STATUS,
  IO_BANDN,      // next band whose start snapshot is due, BANDS: none
  IO_BSLO, IO_BSHI,  // where this frame's band snapshots go
  IO_QHEAD, IO_QTAIL, IO_ACK,  // split form: the TIA side's queue cursor and acknowledgements
  IO_WORDS
};
constexpr uint32_t IO_WSYNC = 1u;


// Per-env blocks of shared memory, env-major, with strides chosen so that a
// warp's lanes touching the same field hit 32 different banks: RAM 128 bytes
// padded to 132 (33 words), I/O state IO_WORDS words, TIA file 44 bytes (11
// words).  Every access is the lane's base plus a constant or one add.  Bytes
// rather than one word per RAM byte keep a 64-env work item small enough for
// four blocks per SM.
constexpr uint32_t RAM_BYTES = 132, IO_STRIDE = IO_WORDS, TIA_STRIDE = 44;
static_assert(IO_STRIDE % 2 == 1 && (TIA_STRIDE / 4) % 2 == 1 && (RAM_BYTES / 4) % 2 == 1 && RAM_BYTES % 4 == 0,
              "odd word strides");
constexpr uint32_t QLEN = 32;             // event queue entries per env (a power of two)
constexpr uint32_t QSTRIDE = QLEN + 1;    // shared-memory words per env queue (odd)
constexpr uint32_t ENV_SMEM = RAM_BYTES + 4 * IO_STRIDE + TIA_STRIDE + 4 * QSTRIDE;
// bytes per cartridge in the batched form's device copy (up to eight 4 KB banks, F4)
constexpr uint32_t ROMB_SLOT = 32768;

// The block's dynamic shared memory; every block of an env is a byte offset
// into it, so that out-of-line functions address it as shared memory too.
extern __shared__ __align__(16) uint8_t g_smem[];
__device__ __forceinline__ uint8_t &sm8(uint32_t off) { return g_smem[off]; }
__device__ __forceinline__ uint32_t &sm32(uint32_t off) { return *reinterpret_cast<uint32_t *>(g_smem + off); }
__device__ __forceinline__ volatile uint32_t &vsm32(uint32_t off) {
  return *reinterpret_cast<volatile uint32_t *>(g_smem + off);
}

// Views of one env's TIA file and I/O state.
struct IoCtx {
  uint32_t tia, io;
  __device__ __forceinline__ uint32_t T(uint32_t s) const { return sm8(tia + s); }
  __device__ __forceinline__ void Tset(uint32_t s, uint32_t v) const { sm8(tia + s) = (uint8_t)v; }
  __device__ __forceinline__ uint32_t G(uint32_t i) const { return sm32(io + 4 * i); }
  __device__ __forceinline__ void Sset(uint32_t i, uint32_t v) const { sm32(io + 4 * i) = v; }
  __device__ __forceinline__ volatile uint32_t &V(uint32_t i) const { return vsm32(io + 4 * i); }
  __device__ __forceinline__ uint64_t G64(uint32_t i) const { return (uint64_t)G(i) | (uint64_t)G(i + 1) << 32; }
  __device__ __forceinline__ void S64(uint32_t i, uint64_t v) const {
    Sset(i, (uint32_t)v);
    Sset(i + 1, (uint32_t)(v >> 32));
  }
};

// ---------------------------------------------------------------- collisions (cold)
__device__ __noinline__ uint32_t fc_collide_cols(IoCtx c, uint32_t live, uint32_t lo, uint32_t hi) {
  M160 r{range_word(0, lo, hi), range_word(1, lo, hi), range_word(2, lo, hi), range_word(3, lo, hi),
         range_word(4, lo, hi)};
  M160 z{0, 0, 0, 0, 0};
  const uint32_t nus0 = c.T(T_NUSIZ0), nus1 = c.T(T_NUSIZ1), ctrl = c.T(T_CTRLPF);
  M160 p0 = (live & 1) ? player_mask((c.T(T_VDELP0) & 1) ? c.T(T_GRP0_O) : c.T(T_GRP0_N), c.T(T_REFP0), nus0,
                                     c.T(T_P0))
                       : z;
  M160 p1 = (live & 2) ? player_mask((c.T(T_VDELP1) & 1) ? c.T(T_GRP1_O) : c.T(T_GRP1_N), c.T(T_REFP1), nus1,
                                     c.T(T_P1))
                       : z;
  M160 m0 = (live & 4) ? missile_mask(nus0, c.T(T_M0)) : z;
  M160 m1 = (live & 8) ? missile_mask(nus1, c.T(T_M1)) : z;
  M160 b = (live & 16) ? ball_mask(ctrl, c.T(T_BL)) : z;
  M160 f = (live & 32) ? pf_mask(c.T(T_PF0), c.T(T_PF1), c.T(T_PF2), ctrl) : z;
  uint32_t x = 0;
  x |= (uint32_t)meet(m0, p1, r) << 1 | (uint32_t)meet(m0, p0, r) << 0;
  x |= (uint32_t)meet(m1, p0, r) << 3 | (uint32_t)meet(m1, p1, r) << 2;
  x |= (uint32_t)meet(p0, f, r) << 5 | (uint32_t)meet(p0, b, r) << 4;
  x |= (uint32_t)meet(p1, f, r) << 7 | (uint32_t)meet(p1, b, r) << 6;
  x |= (uint32_t)meet(m0, f, r) << 9 | (uint32_t)meet(m0, b, r) << 8;
  x |= (uint32_t)meet(m1, f, r) << 11 | (uint32_t)meet(m1, b, r) << 10;
  x |= (uint32_t)meet(b, f, r) << 13;
  x |= (uint32_t)meet(p0, p1, r) << 15 | (uint32_t)meet(m0, m1, r) << 14;
  return x;
}

__device__ __forceinline__ uint32_t fc_live(IoCtx c) {
  const uint32_t g0 = (c.T(T_VDELP0) & 1) ? c.T(T_GRP0_O) : c.T(T_GRP0_N);
  const uint32_t g1 = (c.T(T_VDELP1) & 1) ? c.T(T_GRP1_O) : c.T(T_GRP1_N);
  const uint32_t eb = (c.T(T_VDELBL) & 1) ? c.T(T_ENABL_O) : c.T(T_ENABL_N);
  return (g0 ? 1u : 0u) | (g1 ? 2u : 0u) | (((c.T(T_ENAM0) & 2) && !(c.T(T_RESMP0) & 2)) ? 4u : 0u) |
         (((c.T(T_ENAM1) & 2) && !(c.T(T_RESMP1) & 2)) ? 8u : 0u) | ((eb & 2) ? 16u : 0u) |
         (((c.T(T_PF0) & 0xF0) | c.T(T_PF1) | c.T(T_PF2)) ? 32u : 0u);
}

// Account collisions for every color clock in [ceval, upto) (frame-relative).
__device__ __forceinline__ void fc_cx_eval(IoCtx c, uint32_t upto) {
  const uint32_t from = c.G(IO_CEVAL);
  if (upto <= from) return;
  c.Sset(IO_CEVAL, upto);
  if (c.T(T_VBLANK) & 2) return;
  const uint32_t la = from / 228u, xa = from - la * 228u;
  const uint32_t lb = upto / 228u, xb = upto - lb * 228u;
  if (la == lb && xb <= 68) return;  // the span lies in one line's horizontal blank
  const uint32_t live = fc_live(c);
  if (__popc(live) < 2) return;
  const uint64_t L0 = c.G64(IO_L0LO), bar = c.G64(IO_BARLO);
  uint32_t x = 0;
  auto seg = [&](uint32_t line, uint32_t x0, uint32_t x1) {
    if (x1 <= 68) return;
    uint32_t lo = x0 > 68 ? x0 - 68 : 0, hi = x1 - 68;
    if (L0 + line == bar && lo < 8) lo = 8;
    if (lo < hi) x |= fc_collide_cols(c, live, lo, hi);
  };
  if (la == lb) {
    seg(la, xa, xb);
  } else {
    seg(la, xa, 228);
    if (lb > la + 1) seg(la + 1, 0, 228);
    if (xb) seg(lb, 0, xb);
  }
  c.Sset(IO_CX, c.G(IO_CX) | x);
}

// ---------------------------------------------------------------- I/O (cold)
__device__ __forceinline__ uint32_t fc_res_pos(uint32_t eff, uint32_t add, uint32_t hb) {
  const uint32_t x = eff % 228u;
  if (x < 68) return hb;
  const uint32_t p = x - 68 + add;
  return p >= 160 ? p - 160 : p;
}
__device__ __forceinline__ uint32_t fc_hm_move(uint32_t pos, uint32_t hm) {
  int s = (int)((hm >> 4) & 0xF);
  if (s >= 8) s -= 16;
  int p = (int)pos - s;
  p += p < 0 ? 160 : 0;
  p -= p >= 160 ? 160 : 0;
  return (uint32_t)p;
}

// Read a TIA or RIOT address (13-bit, neither RAM nor cartridge) at cycle t.
// Read a RIOT address (ports, timer) at absolute CPU cycle `now`.
__device__ __forceinline__ uint32_t fc_riot_read(IoCtx c, uint32_t a, uint64_t now) {
  const uint32_t ports = c.G(IO_PORTS);
  if (!(a & 4)) {
    const uint32_t sh = 8 * (a & 2);             // SWCHA/SWACNT in bytes 0/1, SWCHB/SWBCNT in 2/3
    const uint32_t out = (ports >> sh) & 0xFF, ddr = (ports >> (sh + 8)) & 0xFF;
    if (a & 1) return ddr;
    const uint32_t pins = (a & 2) ? 0x0Bu : c.G(IO_JOY);
    return ((out & ddr) | (pins & ~ddr)) & 0xFF;
  }
  const uint64_t n = now - (c.G64(IO_TCWLO) + 1);
  const uint32_t tv = c.G(IO_TV), sh = c.G(IO_TSH);
  const uint64_t span = (uint64_t)(tv + 1) << sh;
  if (a & 1) return n >= span ? 0x80u : 0u;
  if (n < span) return tv - (uint32_t)(n >> sh);
  return (uint32_t)(0xFFull - (n - span)) & 0xFF;
}
// Collision-latch byte of TIA read register reg (0..7) from the CX word.
__device__ __forceinline__ uint32_t fc_cx_byte(uint32_t cx, uint32_t reg) {
  return (((cx >> (2 * reg + 1)) & 1u) << 7) | (((cx >> (2 * reg)) & 1u) << 6);
}
// Bands: groups of BAND_ROWS rows of the 210-row window.  While a frame is
// logged, the render state at the start of every band is kept (48 bytes), so
// that the painter's threads start their bands there instead of replaying the
// frame from its first record.
constexpr uint32_t BAND_ROWS = 2, BANDS = (FRAME_H + BAND_ROWS - 1) / BAND_ROWS, BAND_SNAP = 48;
// First color clock of band q.
__device__ __forceinline__ uint32_t fc_band_clk(uint32_t q) { return 228u * (WINDOW_Y0 + BAND_ROWS * q); }

// Snapshot the render state at the start of every band due by clock eff: the
// state after all records of earlier clocks.  Words 0..8: the TIA file's first
// 36 bytes; word 9: its last byte and, in the high half, the frame-relative
// line of the HMOVE bar or 0xFFFF; word 10: the log records before it.
__device__ __noinline__ void fc_band_snap(IoCtx c, uint32_t eff) {
  uint32_t bn = c.G(IO_BANDN);
  uint8_t *base = reinterpret_cast<uint8_t *>((uint64_t)c.G(IO_BSLO) | (uint64_t)c.G(IO_BSHI) << 32);
  const uint64_t bar = c.G64(IO_BARLO), l0 = c.G64(IO_L0LO);
  const uint32_t rel = bar != NO_LINE && bar >= l0 && bar - l0 < 1024 ? (uint32_t)(bar - l0) : 0xFFFFu;
  const uint32_t nrec = c.G(IO_LOGN);
  uint32_t v[10];
#pragma unroll
  for (int q = 0; q < 10; ++q) v[q] = sm32(c.tia + 4 * q);
  v[9] = (v[9] & 0xFFu) | rel << 16;
  uint4 *d = reinterpret_cast<uint4 *>(base) + 3 * bn;
  while (bn < BANDS && eff >= fc_band_clk(bn)) {
    d[0] = make_uint4(v[0], v[1], v[2], v[3]);
    d[1] = make_uint4(v[4], v[5], v[6], v[7]);
    d[2] = make_uint4(v[8], v[9], nrec, 0);
    d += 3;
    ++bn;
  }
  c.Sset(IO_BANDN, bn);
}

// Log the frame's TIA writes to p (cap records; p null: no log) and the band
// starts to bands.
__device__ __forceinline__ void fc_set_log(IoCtx c, uint32_t *p, uint32_t cap, uint8_t *bands) {
  c.Sset(IO_LOGLO, (uint32_t)(uint64_t)p);
  c.Sset(IO_LOGHI, (uint32_t)((uint64_t)p >> 32));
  c.Sset(IO_LOGN, 0);
  c.Sset(IO_LOGCAP, cap);
  c.Sset(IO_BANDN, bands ? 0u : BANDS);
  c.Sset(IO_BSLO, (uint32_t)(uint64_t)bands);
  c.Sset(IO_BSHI, (uint32_t)((uint64_t)bands >> 32));
}

// Append one TIA write record (effect clock, register, value) to the log of
// a rendered frame.
__device__ __forceinline__ void fc_log(IoCtx c, uint32_t eff, uint32_t reg, uint32_t v) {
  const uint32_t lo = c.G(IO_LOGLO), hi = c.G(IO_LOGHI);
  if (lo | hi) {
    if (c.G(IO_BANDN) < BANDS && eff >= fc_band_clk(c.G(IO_BANDN))) fc_band_snap(c, eff);
    uint32_t *lp = reinterpret_cast<uint32_t *>((uint64_t)lo | (uint64_t)hi << 32);
    const uint32_t nrec = c.G(IO_LOGN);
    if (nrec < c.G(IO_LOGCAP)) lp[nrec] = eff << 14 | reg << 8 | v;
    else c.Sset(IO_STATUS, c.G(IO_STATUS) | ST_LOG_OVERFLOW);
    c.Sset(IO_LOGN, nrec + 1);
  }
}

// Write a RIOT address at absolute CPU cycle `now`.
__device__ __forceinline__ void fc_riot_write(IoCtx c, uint32_t a, uint32_t v, uint64_t now) {
  if (!(a & 4)) {
    const uint32_t sh = 8 * (a & 3);
    c.Sset(IO_PORTS, (c.G(IO_PORTS) & ~(0xFFu << sh)) | (v & 0xFF) << sh);
  } else if (a & 0x10) {
    const uint32_t sel = a & 3;
    c.Sset(IO_TV, v & 0xFF);
    c.Sset(IO_TSH, sel == 0 ? 0 : sel == 1 ? 3 : sel == 2 ? 6 : 10);
    c.S64(IO_TCWLO, now);
  }
}
// Apply a TIA write (register reg at cycle t): collisions up to the write,
// log record, register update.
__device__ __forceinline__ void fc_tia_write(IoCtx c, uint32_t reg, uint32_t v, uint32_t t) {
  const uint32_t eff = 3u * (t + 1u);
  if ((COLL_REGS >> reg) & 1ull) fc_cx_eval(c, eff);
  if ((LOG_REGS >> reg) & 1ull) fc_log(c, eff, reg, v);
  switch (reg) {
    case 0x00: c.Tset(T_VSYNC, v); break;
    case 0x01: c.Tset(T_VBLANK, v); break;
    case 0x04: case 0x05: case 0x06: case 0x07: case 0x08: case 0x09: case 0x0A: case 0x0B: case 0x0C:
    case 0x0D: case 0x0E: case 0x0F:
      c.Tset(reg - 2, v); break;                 // NUSIZ0 .. PF2 are slots 2 .. 13
    case 0x10: c.Tset(T_P0, fc_res_pos(eff, 5, 3)); break;
    case 0x11: c.Tset(T_P1, fc_res_pos(eff, 5, 3)); break;
    case 0x12: c.Tset(T_M0, fc_res_pos(eff, 4, 2)); break;
    case 0x13: c.Tset(T_M1, fc_res_pos(eff, 4, 2)); break;
    case 0x14: c.Tset(T_BL, fc_res_pos(eff, 4, 2)); break;
    case 0x1B: c.Tset(T_GRP1_O, c.T(T_GRP1_N)); c.Tset(T_GRP0_N, v); break;
    case 0x1C:
      c.Tset(T_GRP0_O, c.T(T_GRP0_N)); c.Tset(T_ENABL_O, c.T(T_ENABL_N)); c.Tset(T_GRP1_N, v); break;
    case 0x1D: c.Tset(T_ENAM0, v); break;
    case 0x1E: c.Tset(T_ENAM1, v); break;
    case 0x1F: c.Tset(T_ENABL_N, v); break;
    case 0x20: case 0x21: case 0x22: case 0x23: case 0x24: c.Tset(T_HMP0 + (reg - 0x20), v); break;
    case 0x25: c.Tset(T_VDELP0, v); break;
    case 0x26: c.Tset(T_VDELP1, v); break;
    case 0x27: c.Tset(T_VDELBL, v); break;
    case 0x28: case 0x29: {
      const uint32_t i = reg - 0x28;
      if ((c.T(T_RESMP0 + i) & 2) && !(v & 2)) {
        const uint32_t nus = c.T(T_NUSIZ0 + i);
        const uint32_t sc = (nus & 7) == 5 ? 8u : (nus & 7) == 7 ? 16u : 4u;
        c.Tset(T_M0 + i, (c.T(T_P0 + i) + sc) % 160u);
      }
      c.Tset(T_RESMP0 + i, v);
      break;
    }
    case 0x2A:
      for (uint32_t o = 0; o < 5; ++o) c.Tset(T_P0 + o, fc_hm_move(c.T(T_P0 + o), c.T(T_HMP0 + o)));
      if (eff % 228u < 68u) c.S64(IO_BARLO, c.G64(IO_L0LO) + eff / 228u);
      break;
    case 0x2B:
      for (uint32_t o = 0; o < 5; ++o) c.Tset(T_HMP0 + o, 0);
      break;
    case 0x2C:
      if (eff > c.G(IO_CEVAL)) c.Sset(IO_CEVAL, eff);
      c.Sset(IO_CX, 0);
      break;
    default: break;  // RSYNC, audio, unused addresses
  }
}

// ---------------------------------------------------------------- event queue
// The CPU side pushes every TIA write into a per-env queue in shared memory;
// the TIA side applies the writes, logs them and evaluates collisions.  In
// the split form the TIA side is a second warp of the block (same lane, same
// env); in the single-warp form the warp drains its own queues between
// batches of instructions.  The CPU keeps its own copies of VSYNC, VBLANK,
// the fire latch and the frame base line; it waits for the TIA side only when
// it reads a collision register and at the end of the step.
// An event is one 32-bit word, written and read whole, so the word itself
// tells that it is there: bit 31 holds the parity of the queue's lap (1 in
// the first lap over the zeroed queue), and no fence orders data behind a
// cursor.  Bits 0-30:
//   write       0 | cycle:16 | register:6 | value:8
//   control     1 | kind:2 | argument:
//     mark      begin / end of a logged frame, end of the step
//     sync      evaluate collisions up to a cycle and acknowledge
//     frame end evaluate collisions up to the frame's last cycle
//     rebase    lines to the next frame's first line (follows the frame end)
constexpr uint32_t EV_CTRL = 1u << 30, EV_MARK = EV_CTRL, EV_SYNC = EV_CTRL | 1u << 28,
                   EV_FRAME_END = EV_CTRL | 2u << 28, EV_REBASE = EV_CTRL | 3u << 28;
constexpr uint32_t EV_BEGIN_LOG = EV_MARK, EV_END_LOG = EV_MARK | 1u << 26, EV_STEP_END = EV_MARK | 2u << 26;
// Lap parity of queue position k, in bit 31.
__device__ __forceinline__ uint32_t lap_bit(uint32_t k) { return (~k << 26) & 0x80000000u; }
// A wait between an env's CPU and TIA warps gives up after WAIT_NS of the
// GPU's global timer and the env is declared stalled.  The longest legitimate
// wait is about one frame of the slowest lane of the partner warp (a few
// milliseconds), so the limit is far above it and still short.
constexpr uint64_t WAIT_NS = 200000000ull;  // 200 ms
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Where the TIA side of one env leaves its logs and snapshots.
struct TiaOut {
  uint32_t *log;      // two logs of log_cap records
  uint8_t *bsnap;     // the band snapshots of frames F-1 and F (frame F-1's place is not used when it is not logged)
  uint32_t *meta;     // two times (records, lines)
  uint32_t log_cap;
};
struct TiaSide {
  uint32_t head, ack, lines, log_total;
};
constexpr uint32_t TIA_ACK = 1u, TIA_END = 2u;
// Apply one event; returns TIA_ACK when the CPU side waits for it, and
// TIA_END when it ends the step.
__device__ __forceinline__ uint32_t tia_event(IoCtx c, uint32_t ev, TiaSide &s, const TiaOut &o) {
  if (!(ev & EV_CTRL)) {
    fc_tia_write(c, (ev >> 8) & 0x3F, ev & 0xFF, (ev >> 14) & 0xFFFF);
    return 0;
  }
  const uint32_t kind = (ev >> 28) & 3;
  if (kind == 1) {
    fc_cx_eval(c, 3u * (ev & 0xFFFFu));
    return TIA_ACK;
  }
  if (kind == 2) {
    fc_cx_eval(c, 3u * (ev & 0xFFFFu));
    return 0;
  }
  if (kind == 3) {
    s.lines = ev & 0xFFFFFFFu;
    c.S64(IO_L0LO, c.G64(IO_L0LO) + s.lines);
    c.Sset(IO_CEVAL, c.G(IO_CEVAL) - 228u * s.lines);
    return 0;
  }
  const uint32_t sub = (ev >> 26) & 3, slot = ev & 1;
  if (sub == 0) {
    fc_set_log(c, o.log + (size_t)slot * o.log_cap, o.log_cap, o.bsnap + (size_t)slot * BANDS * BAND_SNAP);
    return 0;
  }
  if (sub == 1) {
    if (c.G(IO_BANDN) < BANDS) fc_band_snap(c, ~0u);  // band starts that the frame never reached take its last state
    const uint32_t nrec = c.G(IO_LOGN);
    o.meta[2 * slot] = nrec;
    o.meta[2 * slot + 1] = s.lines;
    s.log_total += nrec;
    fc_set_log(c, nullptr, 0, nullptr);
    return 0;
  }
  return TIA_ACK | TIA_END;
}
// Single-warp form: apply an env's queued events [s.head, tail).
__device__ __noinline__ void tia_drain(IoCtx c, uint32_t q, TiaSide &s, const TiaOut &o, uint32_t tail) {
  while (s.head != tail) {
    const uint32_t ev = sm32(q + 4 * (s.head & (QLEN - 1)));
    ++s.head;
    tia_event(c, ev, s, o);
  }
}

// ---------------------------------------------------------------- the console
// Split form, CPU side: bounded waits on the TIA side's cursors in this env's
// I/O block.  Wait until the queue has `room` free entries behind `qtail`
// (returns the last head read: still less room means the wait ran out), or
// until `n` events are acknowledged (false means the wait ran out).
__device__ __noinline__ uint32_t fc_q_wait_room(IoCtx c, uint32_t qtail, uint32_t room) {
  uint32_t head = c.V(IO_QHEAD);
  if (qtail - head > QLEN - room) {
    const uint64_t t0 = global_ns();
    while (qtail - head > QLEN - room && global_ns() - t0 < WAIT_NS) {
      __nanosleep(32);
      head = c.V(IO_QHEAD);
    }
  }
  __threadfence_block();  // the TIA side has read the entries that are overwritten next
  return head;
}
__device__ __noinline__ bool fc_q_wait_ack(IoCtx c, uint32_t n) {
  if ((int32_t)(c.V(IO_ACK) - n) < 0) {
    const uint64_t t0 = global_ns();
    while ((int32_t)(c.V(IO_ACK) - n) < 0) {
      if (global_ns() - t0 >= WAIT_NS) return false;
      __nanosleep(32);
    }
  }
  __threadfence_block();
  return true;
}

// Byte permutation with the sign-replicating selectors (selector bit 3).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}
// Predicated stores (addresses in the shared window), without a branch.
__device__ __forceinline__ void sts8_if(bool c, uint32_t a, uint32_t v) {
  asm volatile("{.reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.u8 [%1], %2;}" ::"r"((uint32_t)c), "r"(a), "r"(v)
               : "memory");
}
__device__ __forceinline__ void sts32_if(bool c, uint32_t a, uint32_t v) {
  asm volatile("{.reg .pred p; setp.ne.u32 p, %0, 0; @p st.volatile.shared.u32 [%1], %2;}" ::"r"((uint32_t)c), "r"(a),
               "r"(v)
               : "memory");
}
// Loads of the staged cartridge and the control words, which do not change
// while a work item runs: free to move past the stores of other lanes.
__device__ __forceinline__ uint32_t lds_const(uint32_t a) {
  uint32_t v;
  asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint4 lds_const4(uint32_t a) {
  uint4 v;
  asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}

// Byte offsets of an env's blocks in the block's dynamic shared memory.
struct EnvOff {
  uint32_t rom, dec, ram, io, tia, q;
};
// Rounds between two looks at the lanes that wait for service.  A look costs
// about 60 cycles beside rounds of about 270; a lane that waits loses half a
// batch.
constexpr uint32_t BATCH = 8;

template <bool SPLIT>
struct FastConsoleT {
  EnvOff off;              // this env's blocks of shared memory
  IoCtx io;
  uint32_t A, X, Y, SP, PC, fc, fv, fn, fz, fdi;  // fdi holds the D (0x08) and I (0x04) bits
  uint32_t bank, jam, scheme;
  uint32_t kf;             // CPU cycles since the first line of the frame
  uint32_t pend;           // I/O flags of the current instruction
  uint32_t vs_kf;          // cycle of a VSYNC rise in this frame, ~0 if none
  uint32_t status, instret, frame_no;
  uint32_t frame_inst;     // instret at the frame's start
  uint32_t rounds;         // issue rounds of this env's warp in the step (the same on every lane)
  uint32_t wmask;          // lanes of this warp running envs
  uint32_t idle;           // retire RIOT-timer wait-loop iterations at once
  uint32_t qtail, qhead_seen, nreq, vsync_c, vblank_c, broken;  // qhead_seen: the TIA side's cursor as last read
  uint64_t l0c;
  TiaSide ts;              // single-warp form: the TIA side
  TiaOut to;

  __device__ __forceinline__ uint32_t P() const {
    return (fn & 0x80) | fv | 0x20 | fdi | ((fz & 0xFF) ? 0u : 2u) | fc;
  }
  __device__ __forceinline__ void setP(uint32_t p) {
    fn = p & 0x80; fv = p & 0x40; fdi = p & 0x0C; fz = (p & 2) ? 0u : 1u; fc = p & 1;
  }

  __device__ __forceinline__ void attach(const EnvOff &o) {
    off = o;
    io = IoCtx{o.tia, o.io};
  }
  __device__ __forceinline__ uint8_t &ram(uint32_t i) const { return sm8(off.ram + i); }
  __device__ __forceinline__ uint32_t rom(uint32_t i) const { return sm8(off.rom + i); }

  // ---- canonical state I/O ----
  __device__ void load(const uint8_t *s) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(s);
    const uint32_t w0 = w[0], w1 = w[1];
    A = w0 & 0xFF; X = (w0 >> 8) & 0xFF; Y = (w0 >> 16) & 0xFF; SP = w0 >> 24;
    setP(w1 & 0xFF); PC = w1 >> 16;
    bank = (w1 >> 8) & (scheme == 3 ? 7u : scheme == 2 ? 3u : scheme == 1 ? 1u : 0u);  // scheme is set before load
    const uint64_t k = (uint64_t)w[2] | (uint64_t)w[3] << 32;
    io.Sset(IO_TCWLO, w[4]); io.Sset(IO_TCWHI, w[5]);
    const uint32_t w6 = w[6], w7 = w[7];
    io.Sset(IO_TV, w6 & 0xFF); io.Sset(IO_TSH, (w6 >> 8) & 0xFF);
    io.Sset(IO_PORTS, (w6 >> 16) | ((w7 & 0xFFFF) << 16));
    jam = (w7 >> 16) & 0xFF;
    io.Sset(IO_LATCH, w7 >> 24);
#pragma unroll
    for (int q_ = 0; q_ < 10; ++q_) {
      const uint32_t v = w[8 + q_];
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (q_ * 4 + b < 37) io.Tset(q_ * 4 + b, v >> (8 * b));
    }
    io.Sset(IO_CX, w[17] >> 16);
    io.Sset(IO_BARLO, w[18]); io.Sset(IO_BARHI, w[19]);
    io.Sset(IO_L0LO, w[20]); io.Sset(IO_L0HI, w[21]);
    frame_no = w[22];
    l0c = (uint64_t)w[20] | (uint64_t)w[21] << 32;
    kf = (uint32_t)(k - 76ull * l0c);
    io.Sset(IO_CEVAL, 3u * kf);
    io.Sset(IO_JOY, 0xFF); io.Sset(IO_FIRE, 0);
    io.Sset(IO_LOGLO, 0); io.Sset(IO_LOGHI, 0); io.Sset(IO_LOGN, 0); io.Sset(IO_LOGCAP, 0);
    io.Sset(IO_BANDN, BANDS);
    io.Sset(IO_STATUS, 0);
    const uint4 *r4 = reinterpret_cast<const uint4 *>(s + S::RAM);
    uint32_t *r32 = &sm32(off.ram);
#pragma unroll
    for (int q_ = 0; q_ < 8; ++q_) {
      const uint4 v = r4[q_];
      r32[4 * q_] = v.x; r32[4 * q_ + 1] = v.y; r32[4 * q_ + 2] = v.z; r32[4 * q_ + 3] = v.w;
    }
    for (uint32_t e = 0; e < QLEN; ++e) sm32(off.q + 4 * e) = 0;
    status = 0; instret = 0; frame_inst = 0; rounds = 0; pend = 0; vs_kf = ~0u;
    vsync_c = io.T(T_VSYNC);
    vblank_c = io.T(T_VBLANK);
    qtail = qhead_seen = nreq = broken = 0;
    io.Sset(IO_QHEAD, 0); io.Sset(IO_QTAIL, 0); io.Sset(IO_ACK, 0);
    ts = TiaSide{0, 0, 0, 0};
  }
  __device__ void store(uint8_t *s) const {
    uint32_t *w = reinterpret_cast<uint32_t *>(s);
    const uint64_t L0 = io.G64(IO_L0LO);
    w[0] = A | X << 8 | Y << 16 | SP << 24;
    w[1] = P() | bank << 8 | PC << 16;
    const uint64_t k = 76ull * L0 + kf;
    w[2] = (uint32_t)k; w[3] = (uint32_t)(k >> 32);
    w[4] = io.G(IO_TCWLO); w[5] = io.G(IO_TCWHI);
    const uint32_t ports = io.G(IO_PORTS);
    w[6] = io.G(IO_TV) | io.G(IO_TSH) << 8 | (ports & 0xFFFF) << 16;
    w[7] = (ports >> 16) | jam << 16 | io.G(IO_LATCH) << 24;
#pragma unroll
    for (int q_ = 0; q_ < 10; ++q_) {
      uint32_t v = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (q_ * 4 + b < 37) v |= io.T(q_ * 4 + b) << (8 * b);
      if (q_ == 9) v = (v & 0xFFFFu) | io.G(IO_CX) << 16;
      w[8 + q_] = v;
    }
    w[18] = io.G(IO_BARLO); w[19] = io.G(IO_BARHI);
    w[20] = (uint32_t)L0; w[21] = (uint32_t)(L0 >> 32);
    w[22] = frame_no; w[23] = 0;
    uint4 *r4 = reinterpret_cast<uint4 *>(s + S::RAM);
    const uint32_t *r32 = &sm32(off.ram);
#pragma unroll
    for (int q_ = 0; q_ < 8; ++q_)
      r4[q_] = make_uint4(r32[4 * q_], r32[4 * q_ + 1], r32[4 * q_ + 2], r32[4 * q_ + 3]);
  }
  __device__ uint32_t all_status() const { return status | io.G(IO_STATUS); }

  __device__ void apply_action(uint32_t a) {
    uint32_t d;
    switch (a) {
      case 2: case 10: d = 1; break;
      case 3: case 11: d = 2; break;
      case 4: case 12: d = 4; break;
      case 5: case 13: d = 8; break;
      case 6: case 14: d = 3; break;
      case 7: case 15: d = 5; break;
      case 8: case 16: d = 10; break;
      case 9: case 17: d = 12; break;
      default: d = 0; break;
    }
    io.Sset(IO_JOY, 0xFFu & ~(((d & 2) ? 0x80u : 0u) | ((d & 4) ? 0x40u : 0u) | ((d & 8) ? 0x20u : 0u) |
                              ((d & 1) ? 0x10u : 0u)));
    const uint32_t fire = (a == 1 || a >= 10) ? 1u : 0u;
    io.Sset(IO_FIRE, fire);
    if (fire && (vblank_c & 0x40)) io.Sset(IO_LATCH, 1);
  }

  // Cartridge bytes i .. i+3 of the stage, byte i lowest (i + 3 may run into
  // the padding after the last bank).
  __device__ __forceinline__ uint32_t fetch4(uint32_t i) const {
    const uint32_t a = off.rom + (i & ~3u);
    return __funnelshift_r(sm32(a), sm32(a + 4), (i & 3u) * 8u);
  }
  // Last offset in a bank whose instruction bytes are fetched from the stage:
  // no such fetch touches a hotspot (F8/F6 hotspots start at $FF6, F4's at $FF4).
  __device__ __forceinline__ uint32_t fetch_limit() const { return scheme == 3 ? 0xFF1u : scheme ? 0xFF3u : 0xFFCu; }

  // ---- bus ----
  __device__ __forceinline__ void hotspot(uint32_t at) {
    if (scheme == 1) { if (at == 0xFF8 || at == 0xFF9) bank = at - 0xFF8; }
    else if (scheme == 2) { if (at >= 0xFF6 && at <= 0xFF9) bank = at - 0xFF6; }
    else if (scheme == 3) { if (at >= 0xFF4 && at <= 0xFFB) bank = at - 0xFF4; }
  }
  __device__ __forceinline__ void stall() {
    broken = 1;
    status |= ST_STALL;
    jam = 1;
  }
  // Append an event; when the queue is full the split form waits (bounded)
  // for the TIA side, the single-warp form applies what is queued.
  __device__ void push(uint32_t ev) {
    if (broken) return;
    if (qtail - qhead_seen >= QLEN) {
      if constexpr (SPLIT) {
        qhead_seen = fc_q_wait_room(io, qtail, 1);
        if (qtail - qhead_seen >= QLEN) { stall(); return; }
      } else {
        drain();
      }
    }
    vsm32(off.q + 4 * (qtail & (QLEN - 1))) = ev | lap_bit(qtail);
    ++qtail;
  }
  __device__ __forceinline__ void drain() {
    tia_drain(io, off.q, ts, to, qtail);
    qhead_seen = ts.head;
  }
  // Collisions up to cycle t are in the latches when this returns.
  __device__ void sync_collisions(uint32_t t) {
    if constexpr (SPLIT) {
      if (broken) return;
      push(EV_SYNC | (t & 0xFFFFu));
      ++nreq;
      if (!broken && !fc_q_wait_ack(io, nreq)) stall();
      qhead_seen = qtail;  // acknowledged: the queue is empty
    } else {
      drain();
      fc_cx_eval(io, 3u * t);
    }
  }
  // Read / write a TIA or RIOT address (13-bit, neither RAM nor cartridge) at cycle t.
  __device__ uint32_t io_read(uint32_t a, uint32_t t) {
    if (a & 0x80) return fc_riot_read(io, a, 76ull * l0c + t);
    const uint32_t reg = a & 0x0F;
    if (reg < 8) {
      sync_collisions(t);
      return fc_cx_byte(io.V(IO_CX), reg);
    }
    if (reg == 0x0C) return (io.G(IO_FIRE) || io.G(IO_LATCH)) ? 0x00u : 0x80u;
    return reg == 0x0D ? 0x80u : 0u;
  }
  // WSYNC, the VSYNC rise and the VBLANK latch effects happen here, the
  // register itself on the TIA side.
  __device__ void io_write(uint32_t a, uint32_t v, uint32_t t) {
    if (a & 0x80) { fc_riot_write(io, a, v, 76ull * l0c + t); return; }
    const uint32_t reg = a & 0x3F;
    if (reg == 0x02) { pend |= IO_WSYNC; return; }
    if (reg == 0x00) {
      if (!(vsync_c & 2) && (v & 2) && vs_kf == ~0u) vs_kf = t;
      vsync_c = v;
    } else if (reg == 0x01) {
      vblank_c = v;
      if (!(v & 0x40)) io.Sset(IO_LATCH, 0);
      else if (io.G(IO_FIRE)) io.Sset(IO_LATCH, 1);
    }
    push((t & 0xFFFFu) << 14 | reg << 8 | v);
  }
  __device__ __forceinline__ uint32_t rd(uint32_t addr, uint32_t t) {
    const uint32_t a = addr & 0x1FFF;
    if ((a & 0x1280) == 0x0080) return ram(a & 0x7F);
    if (a & 0x1000) {
      if (scheme) hotspot(a & 0xFFF);
      return rom(bank * 4096u + (a & 0xFFF));
    }
    return io_read(a, t);
  }
  __device__ __forceinline__ void wr(uint32_t addr, uint32_t v, uint32_t t) {
    const uint32_t a = addr & 0x1FFF;
    if ((a & 0x1280) == 0x0080) { ram(a & 0x7F) = (uint8_t)v; return; }
    if (a & 0x1000) { if (scheme) hotspot(a & 0xFFF); return; }
    io_write(a, v & 0xFF, t);
  }

  // ---- ALU ----
  __device__ __forceinline__ void adc(uint32_t v) {
    const uint32_t c = fc;
    if (!(fdi & 0x08)) {
      const uint32_t s = A + v + c;
      const uint32_t r = s & 0xFF;
      fv = ((~(A ^ v) & (A ^ r)) & 0x80u) >> 1;
      fc = s >> 8;
      fn = fz = r;
      A = r;
      return;
    }
    const uint32_t zb = (A + v + c) & 0xFF;
    int lo = (int)(A & 0x0F) + (int)(v & 0x0F) + (int)c;
    if (lo > 9) lo = ((lo + 6) & 0x0F) + 0x10;
    const int hs = (int)(int8_t)(uint8_t)(A & 0xF0) + (int)(int8_t)(uint8_t)(v & 0xF0) + lo;
    int hu = (int)(A & 0xF0) + (int)(v & 0xF0) + lo;
    fn = (uint32_t)hs & 0x80;
    fv = (hs > 127 || hs < -128) ? 0x40u : 0u;
    if (hu >= 0xA0) hu += 0x60;
    fc = hu > 0xFF ? 1u : 0u;
    fz = zb;
    A = (uint32_t)hu & 0xFF;
  }
  __device__ __forceinline__ void sbc(uint32_t v) {
    const uint32_t c = fc;
    const uint32_t nv = v ^ 0xFF;
    const uint32_t s = A + nv + c;
    uint32_t r = s & 0xFF;
    fv = ((~(A ^ nv) & (A ^ r)) & 0x80u) >> 1;
    fc = s >> 8;
    fn = fz = r;
    if (fdi & 0x08) {
      int lo = (int)(A & 0x0F) - (int)(v & 0x0F) + (int)c - 1;
      if (lo < 0) lo = ((lo - 6) & 0x0F) - 0x10;
      int hi = (int)(A & 0xF0) - (int)(v & 0xF0) + lo;
      if (hi < 0) hi -= 0x60;
      r = (uint32_t)hi & 0xFF;
    }
    A = r;
  }
  __device__ __forceinline__ void cmp(uint32_t reg, uint32_t v) {
    fc = reg >= v ? 1u : 0u;
    fn = fz = (reg - v) & 0xFF;
  }
  __device__ __forceinline__ uint32_t asl(uint32_t v) { fc = v >> 7; const uint32_t r = (v << 1) & 0xFF; fn = fz = r; return r; }
  __device__ __forceinline__ uint32_t lsr(uint32_t v) { fc = v & 1; const uint32_t r = v >> 1; fn = fz = r; return r; }
  __device__ __forceinline__ uint32_t rol(uint32_t v) { const uint32_t r = ((v << 1) | fc) & 0xFF; fc = v >> 7; fn = fz = r; return r; }
  __device__ __forceinline__ uint32_t ror(uint32_t v) { const uint32_t r = (v >> 1) | (fc << 7); fc = v & 1; fn = fz = r; return r; }
  __device__ __forceinline__ uint32_t inc(uint32_t v) { const uint32_t r = (v + 1) & 0xFF; fn = fz = r; return r; }
  __device__ __forceinline__ uint32_t dec(uint32_t v) { const uint32_t r = (v - 1) & 0xFF; fn = fz = r; return r; }

  // ---- RIOT-timer wait loops ----
  // LDA INTIM at pc with BNE back to pc right after it: an iteration that
  // reads a nonzero timer value changes nothing but the cycle count (A and the
  // N, Z flags are overwritten by the read that exits), and the read has no
  // side effect.  With the timer counting in intervals of 2^sh >= 8 cycles, at
  // least the loop's period (7 cycles, 8 when the branch crosses a page), the
  // first read at or after the cycle where INTIM reaches 0 reads 0.  So the
  // iterations before that read retire at once: the cycle count advances
  // exactly as if they ran, and the returned cycle is where the exiting LDA
  // starts.  They are not counted in instret, which counts the instructions
  // the issue rounds execute.  Anything else (no such loop, a faster
  // timer, the timer already at 0 or past it, a frame that would reach the
  // line cap) returns k0 unchanged.
  __device__ __forceinline__ uint32_t idle_forward(uint32_t w, uint32_t pc, uint32_t k0) {
    const uint32_t a = (w >> 8) & 0xFFFF;
    if ((a & 0x1285u) != 0x0284u || (w >> 24) != 0xD0u) return k0;  // INTIM (any mirror), then BNE
    const uint32_t at = pc & 0xFFF;
    // BNE offset -5: back to pc, its bytes below the cartridge's hotspots
    if (at > (scheme == 3 ? 0xFEFu : scheme ? 0xFF1u : 0xFFBu) || rom(bank * 4096u + at + 4) != 0xFBu) return k0;
    const uint32_t sh = io.G(IO_TSH);
    if (sh < 3) return k0;
    const uint64_t n0 = 76ull * l0c + k0 + 3 - (io.G64(IO_TCWLO) + 1);  // the read's cycle, as the timer counts it
    const uint64_t zero = (uint64_t)io.G(IO_TV) << sh;                 // first cycle reading 0
    if (n0 >= zero) return k0;
    const uint32_t period = (((pc + 5) ^ pc) & 0xFF00) ? 8u : 7u;
    const uint64_t it = (zero - n0 + period - 1) / period;
    const uint64_t k1 = k0 + it * period;
    if (k1 + 6 >= 76ull * CAP_LINES) return k0;
    return (uint32_t)k1;
  }

  // ---- one instruction, general form (every case) ----
  __device__ void exec_general() {
    const uint32_t k0 = kf;
    pend = 0;
    const uint32_t pc = PC;
    const uint32_t opcode = rd(pc, k0);
    const uint32_t opb = sm8(off.dec + opcode);
    const uint32_t op = opb & 0x7F;
    const uint32_t info = sm8(off.dec + 256 + opcode);
    const uint32_t mode = info & 0xF;
    uint32_t n = info >> 4;
    if (op == O_JAM) { jam = 1; status |= ST_ILLEGAL; return; }
    uint32_t b1 = 0, b2 = 0, ea = 0, cross = 0;
    if (mode >= IMM) b1 = rd(pc + 1, k0);
    if (mode >= ABS && mode <= IND) b2 = rd(pc + 2, k0);
    switch (mode) {
      case IMP: case ACC: PC = (pc + 1) & 0xFFFF; break;
      case IMM: PC = (pc + 2) & 0xFFFF; break;
      case ZP: ea = b1; PC = (pc + 2) & 0xFFFF; break;
      case ZPX: ea = (b1 + X) & 0xFF; PC = (pc + 2) & 0xFFFF; break;
      case ZPY: ea = (b1 + Y) & 0xFF; PC = (pc + 2) & 0xFFFF; break;
      case ABS: ea = b1 | b2 << 8; PC = (pc + 3) & 0xFFFF; break;
      case ABX: { const uint32_t b = b1 | b2 << 8; ea = (b + X) & 0xFFFF; cross = (b ^ ea) >> 8; PC = (pc + 3) & 0xFFFF; break; }
      case ABY: { const uint32_t b = b1 | b2 << 8; ea = (b + Y) & 0xFFFF; cross = (b ^ ea) >> 8; PC = (pc + 3) & 0xFFFF; break; }
      case IND: { const uint32_t p = b1 | b2 << 8;
                  const uint32_t lo = rd(p, k0), hi = rd((p & 0xFF00) | ((p + 1) & 0xFF), k0);
                  ea = lo | hi << 8; PC = (pc + 3) & 0xFFFF; break; }
      case IZX: { const uint32_t z = (b1 + X) & 0xFF; const uint32_t lo = rd(z, k0), hi = rd((z + 1) & 0xFF, k0);
                  ea = lo | hi << 8; PC = (pc + 2) & 0xFFFF; break; }
      case IZY: { const uint32_t lo = rd(b1, k0), hi = rd((b1 + 1) & 0xFF, k0); const uint32_t b = lo | hi << 8;
                  ea = (b + Y) & 0xFFFF; cross = (b ^ ea) >> 8; PC = (pc + 2) & 0xFFFF; break; }
      default: PC = (pc + 2) & 0xFFFF; ea = (PC + (uint32_t)(int32_t)(int8_t)(uint8_t)b1) & 0xFFFF; break;
    }
    if (cross && (opb >> 7)) n++;
    instret++;
    if (mode == REL) {
      uint32_t take;
      switch (op) {
        case O_BCC: take = fc ^ 1u; break;
        case O_BCS: take = fc; break;
        case O_BNE: take = (fz & 0xFF) ? 1u : 0u; break;
        case O_BEQ: take = (fz & 0xFF) ? 0u : 1u; break;
        case O_BVC: take = fv ? 0u : 1u; break;
        case O_BVS: take = fv ? 1u : 0u; break;
        case O_BPL: take = (fn & 0x80) ? 0u : 1u; break;
        default: take = (fn & 0x80) ? 1u : 0u; break;
      }
      if (take) { n += ((PC ^ ea) & 0xFF00) ? 2u : 1u; PC = ea; }
      kf = k0 + n;
      return;
    }
    const uint32_t kA = k0 + n - 1;
    switch (op) {
      case O_LDA: A = mode == IMM ? b1 : rd(ea, kA); fn = fz = A; break;
      case O_LDX: X = mode == IMM ? b1 : rd(ea, kA); fn = fz = X; break;
      case O_LDY: Y = mode == IMM ? b1 : rd(ea, kA); fn = fz = Y; break;
      case O_STA: wr(ea, A, kA); break;
      case O_STX: wr(ea, X, kA); break;
      case O_STY: wr(ea, Y, kA); break;
      case O_ADC: adc(mode == IMM ? b1 : rd(ea, kA)); break;
      case O_SBC: sbc(mode == IMM ? b1 : rd(ea, kA)); break;
      case O_AND: A &= mode == IMM ? b1 : rd(ea, kA); fn = fz = A; break;
      case O_ORA: A |= mode == IMM ? b1 : rd(ea, kA); fn = fz = A; break;
      case O_EOR: A ^= mode == IMM ? b1 : rd(ea, kA); fn = fz = A; break;
      case O_CMP: cmp(A, mode == IMM ? b1 : rd(ea, kA)); break;
      case O_CPX: cmp(X, mode == IMM ? b1 : rd(ea, kA)); break;
      case O_CPY: cmp(Y, mode == IMM ? b1 : rd(ea, kA)); break;
      case O_BIT: { const uint32_t v = rd(ea, kA); fn = v; fv = v & 0x40; fz = A & v; break; }
      case O_ASL: case O_LSR: case O_ROL: case O_ROR: case O_INC: case O_DEC: {
        const uint32_t old = mode == ACC ? A : rd(ea, kA - 2);
        uint32_t r;
        switch (op) {
          case O_ASL: r = asl(old); break;
          case O_LSR: r = lsr(old); break;
          case O_ROL: r = rol(old); break;
          case O_ROR: r = ror(old); break;
          case O_INC: r = inc(old); break;
          default: r = dec(old); break;
        }
        if (mode == ACC) A = r;
        else { wr(ea, old, kA - 1); wr(ea, r, kA); }
        break;
      }
      case O_SLO: case O_RLA: case O_SRE: case O_RRA: case O_DCP: case O_ISC: {
        // read-modify-write of memory (both writes), then the accumulator operation
        const uint32_t old = rd(ea, kA - 2);
        uint32_t r, c = fc;
        switch (op) {
          case O_SLO: r = (old << 1) & 0xFF; c = old >> 7; break;
          case O_RLA: r = ((old << 1) | fc) & 0xFF; c = old >> 7; break;
          case O_SRE: r = old >> 1; c = old & 1; break;
          case O_RRA: r = (old >> 1) | (fc << 7); c = old & 1; break;
          case O_DCP: r = (old - 1) & 0xFF; break;
          default: r = (old + 1) & 0xFF; break;
        }
        wr(ea, old, kA - 1);
        wr(ea, r, kA);
        switch (op) {
          case O_SLO: A |= r; fc = c; fn = fz = A; break;
          case O_RLA: A &= r; fc = c; fn = fz = A; break;
          case O_SRE: A ^= r; fc = c; fn = fz = A; break;
          case O_RRA: fc = c; adc(r); break;
          case O_DCP: cmp(A, r); break;
          default: sbc(r); break;
        }
        break;
      }
      case O_SAX: wr(ea, A & X, kA); break;
      case O_LAX: A = rd(ea, kA); X = A; fn = fz = A; break;
      case O_ANC: A &= b1; fn = fz = A; fc = A >> 7; break;
      case O_ALR: A &= b1; fc = A & 1u; A >>= 1; fn = fz = A; break;
      case O_SBX: { const uint32_t ax = A & X; fc = ax >= b1 ? 1u : 0u; X = (ax - b1) & 0xFF; fn = fz = X; break; }
      case O_NOP: if (mode != IMP && mode != IMM) (void)rd(ea, kA); break;  // the operand read
      case O_INX: X = (X + 1) & 0xFF; fn = fz = X; break;
      case O_INY: Y = (Y + 1) & 0xFF; fn = fz = Y; break;
      case O_DEX: X = (X - 1) & 0xFF; fn = fz = X; break;
      case O_DEY: Y = (Y - 1) & 0xFF; fn = fz = Y; break;
      case O_TAX: X = A; fn = fz = X; break;
      case O_TAY: Y = A; fn = fz = Y; break;
      case O_TXA: A = X; fn = fz = A; break;
      case O_TYA: A = Y; fn = fz = A; break;
      case O_TSX: X = SP; fn = fz = X; break;
      case O_TXS: SP = X; break;
      case O_CLC: fc = 0; break;
      case O_SEC: fc = 1; break;
      case O_CLI: fdi &= ~0x04u; break;
      case O_SEI: fdi |= 0x04u; break;
      case O_CLV: fv = 0; break;
      case O_CLD: fdi &= ~0x08u; break;
      case O_SED: fdi |= 0x08u; break;
      case O_PHA: wr(0x100u | SP, A, kA); SP = (SP - 1) & 0xFF; break;
      case O_PHP: wr(0x100u | SP, P() | 0x10u, kA); SP = (SP - 1) & 0xFF; break;
      case O_PLA: SP = (SP + 1) & 0xFF; A = rd(0x100u | SP, kA); fn = fz = A; break;
      case O_PLP: SP = (SP + 1) & 0xFF; setP(rd(0x100u | SP, kA)); break;
      case O_JMP: PC = ea; break;
      case O_JSR: {
        const uint32_t ret = (pc + 2) & 0xFFFF;
        wr(0x100u | SP, ret >> 8, kA); SP = (SP - 1) & 0xFF;
        wr(0x100u | SP, ret & 0xFF, kA); SP = (SP - 1) & 0xFF;
        PC = ea;
        break;
      }
      case O_RTS: {
        SP = (SP + 1) & 0xFF; const uint32_t lo = rd(0x100u | SP, kA);
        SP = (SP + 1) & 0xFF; const uint32_t hi = rd(0x100u | SP, kA);
        PC = ((lo | hi << 8) + 1) & 0xFFFF;
        break;
      }
      case O_RTI: {
        SP = (SP + 1) & 0xFF; setP(rd(0x100u | SP, kA));
        SP = (SP + 1) & 0xFF; const uint32_t lo = rd(0x100u | SP, kA);
        SP = (SP + 1) & 0xFF; const uint32_t hi = rd(0x100u | SP, kA);
        PC = lo | hi << 8;
        break;
      }
      case O_BRK: {
        const uint32_t ret = (pc + 2) & 0xFFFF;
        wr(0x100u | SP, ret >> 8, kA); SP = (SP - 1) & 0xFF;
        wr(0x100u | SP, ret & 0xFF, kA); SP = (SP - 1) & 0xFF;
        wr(0x100u | SP, P() | 0x10u, kA); SP = (SP - 1) & 0xFF;
        fdi |= 0x04u;
        const uint32_t lo = rd(0x1FFE, kA), hi = rd(0x1FFF, kA);
        PC = lo | hi << 8;
        break;
      }
      default: break;
    }
    uint32_t k = k0 + n;
    if (pend & IO_WSYNC) k = ((k + 75u) / 76u) * 76u;
    kf = k;
  }

  // Append the end of the current frame and start counting the next.
  __device__ __forceinline__ void end_frame(uint32_t next_rel) {
    push(EV_FRAME_END | (kf & 0xFFFFu));
    push(EV_REBASE | (next_rel & 0xFFFFFFFu));
    l0c += next_rel;
    kf -= 76u * next_rel;
    frame_no++;
    vs_kf = ~0u;
    frame_inst = instret;
  }

  // Run this env (every lane of wmask its own) until hook.frame_done() says
  // that the step is over.
  //
  // The hot loop is one branch-free instruction sequence for every common
  // instruction, steered by the opcode's control words (opcode_ctl.h): one
  // adder with masks covers loads, transfers, arithmetic, logic, shifts left,
  // increments and compares, one sum covers the effective address, the branch
  // target and the immediate operand, and one load covers RAM and cartridge.
  // So lanes at different instructions still execute together: each lane
  // runs its own program at one instruction per round, with no leader, no
  // reconvergence and a loop that stays in the instruction cache's first
  // level.  What it does not take (RIOT accesses, collision reads, VSYNC and
  // VBLANK, stack and pointer instructions, bank hotspots, frame ends) stops
  // the lane in front of the instruction; every BATCH rounds the lanes that
  // wait are served together by the general decoder, at once when no lane is
  // left running, otherwise after at most one more batch, so that lanes a few
  // rounds apart share one call.
  template <class Hook> __device__ __forceinline__ void run(Hook &hook);
};

// One service of a waiting lane: the frame's end, or the instruction at PC by
// the general decoder (after a timer wait loop's idle iterations).  Returns
// false when the step is over.
template <bool SPLIT, class Hook>
__device__ __noinline__ bool fc_service(FastConsoleT<SPLIT> *c, Hook *h) {
  const uint32_t cap = 76u * CAP_LINES;
  // at least one instruction runs in every frame before the line cap ends it
  bool ended = c->jam || (c->kf >= cap && c->instret != c->frame_inst);
  if (!ended) {
    const uint32_t at = c->PC & 0xFFF;
    if (c->idle && (c->PC & 0x1000) && at <= c->fetch_limit()) {
      const uint32_t w = c->fetch4(c->bank * 4096u + at);
      if ((w & 0xFF) == 0xAD) c->kf = c->idle_forward(w, c->PC, c->kf);
    }
    c->exec_general();
    ended = c->jam || c->vs_kf != ~0u || c->kf >= cap;
  }
  while (ended) {
    uint32_t next_rel;
    if (c->jam) next_rel = c->kf / 76u;
    else if (c->vs_kf != ~0u) next_rel = c->vs_kf / 76u;
    else { c->status |= ST_FRAME_CAP; next_rel = c->kf / 76u; }
    c->end_frame(next_rel);
    if (!h->frame_done(*c)) return false;
    ended = c->jam != 0;
  }
  return true;
}

template <bool SPLIT>
template <class Hook>
__device__ __forceinline__ void FastConsoleT<SPLIT>::run(Hook &hook) {
  const EnvOff o = off;
  const uint32_t smb = (uint32_t)__cvta_generic_to_shared(g_smem);
  const uint32_t cap = 76u * CAP_LINES;
  const uint32_t ctl = o.dec + 512, romb = smb + o.rom;
  const uint32_t lim = fetch_limit();
  // cartridge reads below the first hotspot are plain loads
  const uint32_t hot = scheme == 3 ? 0xFF4u : scheme == 2 ? 0xFF6u : scheme == 1 ? 0xFF8u : 0x1000u;
  uint32_t R, Pf, pc, k, inst, qt, bk;
  uint32_t rec, cb;
  uint4 c;
  bool wait = false, active = true;
  // instruction bytes at p; the control words of opcode op
  auto bytes_at = [&](uint32_t p) {
    const uint32_t i = bk + (p & 0xFFFu);
    const uint32_t a = romb + (i & ~3u);
    return __funnelshift_r(lds_const(a), lds_const(a + 4), i * 8u);
  };
  auto control = [&](uint32_t op) {
    c = lds_const4(smb + ctl + op * 16u);
    cb = lds_const(smb + ctl + CTL_B_OFF + op * 4u);
  };
  // the console's fields to the loop's registers, and the next instruction
  auto enter = [&](bool stay) {
    R = A | X << 8 | Y << 16;
    Pf = P(); pc = PC; k = kf; inst = instret; qt = qtail; bk = bank * 4096u;
    rec = bytes_at(pc);
    wait = stay || ((pc & 0x1FFFu) - 0x1000u) > lim || k >= cap;
    control(wait ? CTL_HALT : rec & 0xFFu);
  };
  enter(jam != 0);
  uint32_t held = 0, act = wmask;
  for (;;) {
#pragma unroll 1
    for (uint32_t r = 0; r < BATCH; ++r) {
      // --- next instruction (branches and JMP abs: the sum is the target)
      const uint32_t pcn = pc + (c.w >> 28);
      const uint32_t base = prmt(rec, pcn, c.x);
      const uint32_t sum = base + prmt(R, rec, c.y);
      const bool tk = ((Pf ^ (c.y >> 24)) & (c.y >> 16) & 0xFFu) != 0;
      const uint32_t npc = tk ? sum & 0xFFFFu : pcn;
      const uint32_t nrec = bytes_at(npc);
      const bool nbad = ((npc & 0x1FFFu) - 0x1000u) > lim;
      // --- cycles
      const uint32_t tk1 = tk ? 1u : 0u;
      const uint32_t n = ((cb >> 8) & 0x7Fu) + tk1 + (((base ^ sum) >> 8) & (((cb >> 15) & 1u) | tk1));
      const uint32_t kn = k + n;
      // --- operand
      const uint32_t ea = sum & (c.x >> 16);
      const bool is_ram = (ea & 0x1280u) == 0x0080u;
      const bool is_cart = ea - 0x1000u < hot;
      const uint32_t tia = ea & 0x10BFu;                  // below $40: a TIA register
      const uint32_t at = is_ram ? o.ram + (ea & 0x7Fu) : o.rom + bk + (ea & 0xFFFu);
      const uint32_t ld = sm8(at);
      const uint32_t y = ((cb & CT_MEM) ? ld : sum) ^ (c.z >> 24);
      const uint32_t x = prmt(R, y | 0xFF00u, c.z);
      // --- what the general decoder takes
      const bool is_ld = (cb & CT_LD) != 0, is_st = (cb & CT_ST) != 0, is_rmw = (cb & CT_RMW) != 0;
      const bool ok = is_ram | (is_ld & is_cart) | (is_st & (tia - 2u < 0x3Eu));
      const bool slow = ((cb & CT_SLOW) != 0) | ((is_ld | is_st | is_rmw) & !ok) | ((Pf & (cb >> 24) & 0x08u) != 0);
      // --- result
      const uint32_t cin = (Pf & cb & 1u) | ((cb >> 1) & 1u);
      const uint32_t add = (x & y) * ((cb >> 24) & 3u) + ((x ^ y) & (c.z >> 16)) + cin;
      const uint32_t rot = (((y + (cin << 8)) * 513u) >> 1) & 0x1FFu;
      const uint32_t s = (cb & CT_SHR) ? rot : add;
      // --- flags
      uint32_t nf = (s & 0x80u) | ((s >> 8) & 1u) | ((((x ^ s) & ~(x ^ y)) & 0x80u) >> 1) | ((s & 0xFFu) ? 0u : 2u);
      const uint32_t bits = (cb >> 16) & 0xFFu, pm = slow ? 0u : (c.w >> 16) & 0xFFu;
      nf = (nf & ~bits) | (y & bits);
      // --- commit
      const uint32_t sv = (is_rmw ? s : x) & 0xFFu;
      sts8_if((is_st | is_rmw) & is_ram & !slow, smb + at, sv);
      const bool out = is_st & (tia - 3u < 0x3Du) & !slow;
      sts32_if(out, smb + o.q + (qt & (QLEN - 1)) * 4u, ((kn - 1u) << 14 | tia << 8 | sv) ^ lap_bit(qt));
      qt += out ? 1u : 0u;
      const uint32_t kw = (is_st & (tia == 2u)) ? (kn + 75u) / 76u * 76u : kn;
      R = prmt(R, s, slow ? 0x3210u : c.w);
      Pf = (Pf & ~pm) | (nf & pm);
      inst += slow ? 0u : (cb >> 28) & 1u;
      pc = slow ? pc : npc;
      k = slow ? k : kw;
      wait = wait | slow | nbad | (k >= cap);
      rec = nrec;
      control(wait ? CTL_HALT : nrec & 0xFFu);
    }
    // --- service: waiting lanes, and queues without room for another batch
    rounds += BATCH;
    const bool full = qt - qhead_seen > QLEN - BATCH;
    uint32_t m = __ballot_sync(wmask, (wait | full) & active);
    if (m == 0) continue;
    m = __ballot_sync(wmask, wait & active);
    if (m != 0 && (m == act || ++held > 1)) {
      held = 0;
      ++rounds;
      if (active && wait) {
        A = R & 0xFF; X = (R >> 8) & 0xFF; Y = (R >> 16) & 0xFF;
        setP(Pf); PC = pc; kf = k; instret = inst; qtail = qt;
        active = fc_service<SPLIT, Hook>(this, &hook);
        enter(!active);
      }
      act = __ballot_sync(wmask, active);
      if (act == 0) break;
    }
    // room for a batch of events
    if constexpr (SPLIT) {
      if (active & (qt - qhead_seen > QLEN - BATCH)) {
        qhead_seen = fc_q_wait_room(io, qt, BATCH);
        if (qt - qhead_seen > QLEN - BATCH) { stall(); wait = true; control(CTL_HALT); }
      }
    } else {
      if (__any_sync(wmask, qt - qhead_seen > QLEN - BATCH)) {
        qtail = qt;
        drain();
      }
    }
    __syncwarp(wmask);
  }
  A = R & 0xFF; X = (R >> 8) & 0xFF; Y = (R >> 16) & 0xFF;
  setP(Pf); PC = pc; kf = k; instret = inst; qtail = qt;
}

}  // namespace atari
