// Console for the batched form, laid out for the issue rate of sm_103a.
//
// Same machine and canonical state as Console in device_machine.cuh:
//   - the hot loop is one branch-free sequence for every common instruction,
//     steered by control words per opcode (opcode_ctl.h);
//   - CPU registers, flags, the cycle counter and the bank in registers;
//   - RAM (bytes), the TIA register file (bytes) and the I/O state
//     (collision latches, RIOT timer and ports, inputs) in shared memory with odd
//     word strides, so lanes reading the same field never bank-conflict and
//     every access is a base offset plus a constant or one add;
//   - a byte of RAM every four bytes, four envs interleaved, so that RAM and
//     cartridge addresses scale alike;
//   - the block's cartridge staged in shared memory as one word per byte (64 KB
//     for an F6 cartridge), the byte and the two after it: an instruction is
//     one load, and a data byte the first byte of its word.
// Instructions the hot loop does not take are served beside it, out of line:
// accesses through pointers, stack instructions, BIT, TIA and RIOT reads, RIOT
// and VBLANK writes, hotspots, decimal arithmetic and undocumented opcodes with
// the console in registers (fc_quick), what is left (frame ends, interrupts,
// JMP through a pointer, fetches outside the cartridge or next to a hotspot) by
// the general decoder.
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
  IO_CX = 0, IO_BARLO, IO_BARHI, IO_TCWLO, IO_TCWHI, IO_TV, IO_TSH, IO_PORTS, IO_JOY, IO_FIRE, IO_LATCH, IO_STATUS,
  IO_QHEAD, IO_ACK,  // split form: the TIA side's queue cursor and acknowledgements
  IO_PAD,            // an odd stride
  IO_WORDS
};
constexpr uint32_t IO_WSYNC = 1u;


// Blocks of shared memory per env, with strides chosen so that a warp's lanes
// touching the same field hit 32 different banks: I/O state IO_WORDS words, TIA
// file 44 bytes (11 words); RAM in groups of four envs of RAM_GROUP bytes, a
// word holding one byte of each.  Every access is the lane's base plus a
// constant or one add.
constexpr uint32_t RAM_GROUP = 516, IO_STRIDE = IO_WORDS, TIA_STRIDE = 44;
static_assert(IO_STRIDE % 2 == 1 && (TIA_STRIDE / 4) % 2 == 1 && (RAM_GROUP / 4) % 2 == 1 && RAM_GROUP % 4 == 0,
              "odd word strides");
constexpr uint32_t QLEN = 32;             // event queue entries per env (a power of two)
constexpr uint32_t QSTRIDE = QLEN + 1;    // shared-memory words per env queue (odd)
constexpr uint32_t ENV_SMEM = 4 * IO_STRIDE + TIA_STRIDE + 4 * QSTRIDE;  // beside the RAM
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

// ---------------------------------------------------------------- collisions
// Where the TIA side of one env leaves its logs and snapshots.
struct TiaOut {
  uint32_t *log;      // two logs of log_cap records
  uint8_t *bsnap;     // the band snapshots of frames F-1 and F (frame F-1's place is not used when it is not logged)
  uint32_t *meta;     // two times (records, lines)
  uint32_t log_cap;
};
// The TIA side's cursors, in registers while events are applied.
struct TiaSide {
  uint32_t head, ack, lines, log_total;
  uint32_t ceval;     // collisions are accounted for every color clock before it (frame-relative)
  uint32_t cx;        // collision latches
  uint32_t bar;       // frame-relative line of the HMOVE bar, ~0: none in this frame or later
  uint64_t l0;        // first line of the frame
  uint32_t hi;        // bits 16-31 of the cycles that the events carry
  uint32_t *log;      // next record of the logged frame, null: not logged
  uint32_t nrec;      // records so far
  uint8_t *bands;     // the frame's band snapshots
  uint32_t band, band_clk;  // next band whose start snapshot is due, and its first color clock
  uint32_t status;
};
constexpr uint32_t NO_BAR = ~0u;

// The n lowest bits of a word (all of them from 32 on).
__device__ __forceinline__ uint32_t low_bits(uint32_t n) {
  uint32_t m;
  asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(m) : "r"(n));
  return m;
}
// Bits below n of word w of a 160-bit mask.
__device__ __forceinline__ uint32_t below(uint32_t n, int w) {
  const int k = (int)n - 32 * w;
  return low_bits((uint32_t)(k < 0 ? 0 : k));
}

// Latch bits of each object (P0, P1, M0, M1, BL, PF): a pair's bit is in both its objects' sets.
constexpr uint32_t CXP_P0 = 0x8039u, CXP_P1 = 0x80C6u, CXP_M0 = 0x4303u, CXP_M1 = 0x4C0Cu, CXP_BL = 0x2550u,
                   CXP_PF = 0x2AA0u, CXP_ALL = 0xEFFFu;

// Collisions from (line la, clock xa) to (line lb, clock xb) under the current
// registers: the latch bits that are not in `cx` yet.  The registers do not
// change in between, so the visible columns of all the lines it covers count
// together: one evaluation whatever the number of lines.
__device__ __noinline__ uint32_t fc_collide(IoCtx c, uint32_t la, uint32_t xa, uint32_t lb, uint32_t xb, uint32_t bar,
                                            uint32_t cx) {
  const uint32_t w0 = sm32(c.tia), w2 = sm32(c.tia + 8), w3 = sm32(c.tia + 12), w4 = sm32(c.tia + 16),
                 w5 = sm32(c.tia + 20), w6 = sm32(c.tia + 24), w8 = sm32(c.tia + 32);
  // the registers as bytes of the file's words (TiaSlot order)
  const uint32_t g0 = (w5 & 0x10000u) ? w4 >> 24 : (w4 >> 16) & 0xFFu;         // VDELP0: GRP0 old or new
  const uint32_t g1 = (w5 & 0x1000000u) ? (w5 >> 8) & 0xFFu : w5 & 0xFFu;      // VDELP1
  const uint32_t bl = (w6 & 1u) ? w4 >> 8 : w4;                                // VDELBL
  uint32_t off = g0 ? 0u : CXP_P0;
  off |= g1 ? 0u : CXP_P1;
  off |= (w3 & 0x20000u) && !(w6 & 0x200u) ? 0u : CXP_M0;                      // ENAM0, RESMP0
  off |= (w3 & 0x2000000u) && !(w6 & 0x20000u) ? 0u : CXP_M1;
  off |= (bl & 2u) ? 0u : CXP_BL;
  off |= ((w2 & 0xF0000000u) | (w3 & 0xFFFFu)) ? 0u : CXP_PF;
  const uint32_t need = CXP_ALL & ~off & ~cx;
  if (need == 0) return 0;
  // visible columns: [a, 160) of line la, whole lines, [b0, b) of line lb; one line: [a, b)
  const bool one = la == lb;
  uint32_t a = xa > 68u ? xa - 68u : 0u;
  if (la == bar && a < 8u) a = 8u;
  const uint32_t b = xb > 68u ? xb - 68u : 0u;
  const uint32_t mid = lb > la + 1u && !one ? ~0u : 0u;
  M160 r;
  uint32_t *rw = &r.w0;
  const uint32_t bar8 = lb == bar ? ~0xFFu : ~0u;                              // line lb under the bar
  const uint32_t mid8 = la + 1u == bar && lb == la + 2u ? ~0xFFu : ~0u;        // the only whole line under it
#pragma unroll
  for (int w = 0; w < 5; ++w) {
    const uint32_t ge = ~below(a, w);
    uint32_t lt = below(b, w), md = mid;
    if (w == 0) { md &= mid8; lt &= one ? ~0u : bar8; }
    rw[w] = one ? ge & lt : ge | md | lt;
  }
  const M160 z{0, 0, 0, 0, 0};
  auto clip = [&](M160 m) { return M160{m.w0 & r.w0, m.w1 & r.w1, m.w2 & r.w2, m.w3 & r.w3, m.w4 & r.w4}; };
  const uint32_t nus0 = w0 >> 16, nus1 = w0 >> 24, ctrl = w2;
  const M160 p0 = (need & CXP_P0) ? clip(player_mask(g0, w2 >> 8, nus0, w8 & 0xFFu)) : z;
  const M160 p1 = (need & CXP_P1) ? clip(player_mask(g1, w2 >> 16, nus1, (w8 >> 8) & 0xFFu)) : z;
  const M160 m0 = (need & CXP_M0) ? clip(missile_mask(nus0, (w8 >> 16) & 0xFFu)) : z;
  const M160 m1 = (need & CXP_M1) ? clip(missile_mask(nus1, w8 >> 24)) : z;
  const M160 bm = (need & CXP_BL) ? clip(ball_mask(ctrl, sm8(c.tia + T_BL))) : z;
  const M160 f = (need & CXP_PF) ? pf_mask(w2 >> 24, w3 & 0xFFu, (w3 >> 8) & 0xFFu, ctrl) : z;
  auto pair = [](const M160 &u, const M160 &v, uint32_t bit) {
    return ((u.w0 & v.w0) | (u.w1 & v.w1) | (u.w2 & v.w2) | (u.w3 & v.w3) | (u.w4 & v.w4)) ? 1u << bit : 0u;
  };
  uint32_t x = pair(m0, p0, 0) | pair(m0, p1, 1) | pair(m1, p1, 2) | pair(m1, p0, 3) | pair(p0, p1, 15) |
               pair(m0, m1, 14);
  x |= pair(p0, bm, 4) | pair(p1, bm, 6) | pair(m0, bm, 8) | pair(m1, bm, 10);
  x |= pair(p0, f, 5) | pair(p1, f, 7) | pair(m0, f, 9) | pair(m1, f, 11) | pair(bm, f, 13);
  return x & need;
}

// Account collisions for every color clock before `upto` (frame-relative).
__device__ __forceinline__ void fc_cx_eval(IoCtx c, TiaSide &s, uint32_t upto) {
  const uint32_t from = s.ceval;
  if (upto <= from) return;
  s.ceval = upto;
  if (c.T(T_VBLANK) & 2) return;
  const uint32_t la = from / 228u, xa = from - la * 228u;
  const uint32_t lb = upto / 228u, xb = upto - lb * 228u;
  if (la == lb && xb <= 68) return;  // the span lies in one line's horizontal blank
  s.cx |= fc_collide(c, la, xa, lb, xb, s.bar, s.cx);
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
__device__ __noinline__ uint32_t fc_band_snap(IoCtx c, uint8_t *bands, uint32_t band, uint32_t bar, uint32_t nrec,
                                              uint32_t eff) {
  uint32_t v[10];
#pragma unroll
  for (int q = 0; q < 10; ++q) v[q] = sm32(c.tia + 4 * q);
  v[9] = (v[9] & 0xFFu) | (bar < 1024u ? bar : 0xFFFFu) << 16;
  uint4 *d = reinterpret_cast<uint4 *>(bands) + 3 * band;
  while (band < BANDS && eff >= fc_band_clk(band)) {
    d[0] = make_uint4(v[0], v[1], v[2], v[3]);
    d[1] = make_uint4(v[4], v[5], v[6], v[7]);
    d[2] = make_uint4(v[8], v[9], nrec, 0);
    d += 3;
    ++band;
  }
  return band;
}
__device__ __forceinline__ void fc_bands_due(IoCtx c, TiaSide &s, uint32_t eff) {
  s.band = fc_band_snap(c, s.bands, s.band, s.bar, s.nrec, eff);
  s.band_clk = s.band < BANDS ? fc_band_clk(s.band) : ~0u;
}

// Append one TIA write record (effect clock, register, value) to the log of
// a rendered frame.
__device__ __forceinline__ void fc_log(IoCtx c, TiaSide &s, uint32_t cap, uint32_t eff, uint32_t reg, uint32_t v) {
  if (!s.log) return;
  if (eff >= s.band_clk) fc_bands_due(c, s, eff);
  if (s.nrec < cap) s.log[s.nrec] = eff << 14 | reg << 8 | v;
  else s.status |= ST_LOG_OVERFLOW;
  ++s.nrec;
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
// Registers whose write only sets a slot of the file: all but the strobes, the
// graphics with their delayed copies and RESMPx.
constexpr uint64_t SET_REGS = 0xFFF0ull | (7ull << 0x1D) | (0x1Full << 0x20) | (7ull << 0x25);
// Apply a TIA write (register reg at cycle t): collisions up to the write,
// log record, register update.  A kernel writes most registers on every line
// with the value that they have; such a write leaves the span that the next
// evaluation covers open (the registers are the same on both sides of it), so
// the TIA warp evaluates a few spans a frame, not several a line.  Writes that
// only set a slot, nearly all of them, do not come to the switch: a level of
// its compare tree costs 30 cycles, and the TIA warp has to keep up with
// rounds of about 160.
__device__ __forceinline__ void fc_tia_write(IoCtx c, TiaSide &s, uint32_t cap, uint32_t reg, uint32_t v, uint32_t t) {
  const uint32_t eff = 3u * (t + 1u);
  const bool set = ((SET_REGS >> reg) & 1ull) != 0;
  // NUSIZ0 .. PF2 are slots 2 .. 13, HMP0 .. HMBL 27 .. 31, ENAM0 .. ENABL 14 .. 16, VDELP0 .. VDELBL 22 .. 24
  const uint32_t slot = reg - (reg < 0x10u ? 2u : reg - 0x20u < 5u ? 5u : 15u);
  bool change = true;
  if (set) change = c.T(slot) != v;
  else if (reg == 0x1B) change = (c.T(T_GRP0_N) != v) | (c.T(T_GRP1_O) != c.T(T_GRP1_N));
  else if (reg == 0x1C)
    change = (c.T(T_GRP1_N) != v) | (c.T(T_GRP0_O) != c.T(T_GRP0_N)) | (c.T(T_ENABL_O) != c.T(T_ENABL_N));
  if (change & (((COLL_REGS >> reg) & 1ull) != 0)) fc_cx_eval(c, s, eff);
  if ((LOG_REGS >> reg) & 1ull) fc_log(c, s, cap, eff, reg, v);
  if (set) {
    c.Tset(slot, v);
    return;
  }
  if (reg == 0x1B) {
    c.Tset(T_GRP1_O, c.T(T_GRP1_N));
    c.Tset(T_GRP0_N, v);
    return;
  }
  if (reg == 0x1C) {
    c.Tset(T_GRP0_O, c.T(T_GRP0_N));
    c.Tset(T_ENABL_O, c.T(T_ENABL_N));
    c.Tset(T_GRP1_N, v);
    return;
  }
  switch (reg) {
    case 0x00: c.Tset(T_VSYNC, v); break;
    case 0x01: c.Tset(T_VBLANK, v); break;
    case 0x10: case 0x11: c.Tset(T_P0 + reg - 0x10, fc_res_pos(eff, 5, 3)); break;
    case 0x12: case 0x13: case 0x14: c.Tset(T_P0 + reg - 0x10, fc_res_pos(eff, 4, 2)); break;
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
      if (eff % 228u < 68u) {
        s.bar = eff / 228u;
        c.S64(IO_BARLO, s.l0 + s.bar);
      }
      break;
    case 0x2B:
      for (uint32_t o = 0; o < 5; ++o) c.Tset(T_HMP0 + o, 0);
      break;
    case 0x2C:
      if (eff > s.ceval) s.ceval = eff;
      s.cx = 0;
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
// tells that it is there: bit 15 holds the parity of the queue's lap (1 in
// the first lap over the zeroed queue), and no fence orders data behind a
// cursor.  Bits 16-31 are a CPU cycle of the frame:
//   write       bit 14 = 0 | register << 8 | value; the cycle after the write's
//   control     bit 14 = 1 | kind << 8 | argument:
//     high      bits 16-31 are those bits of the cycles of all events up to the frame's end (0 at its start;
//               not 0 only where a state was loaded far past the line cap, for the one instruction that it runs)
//     begin / end of a logged frame (argument: 0 frame F-1, 1 frame F), end of the step
//     sync      evaluate collisions up to the cycle and acknowledge
//     frame end evaluate collisions up to the frame's last cycle
//     rebase    lines towards the next frame's first line (follow the frame
//               end; bits 16-31 and, above them, the argument)
constexpr uint32_t EV_CTRL = 1u << 14, EV_BEGIN_LOG = EV_CTRL, EV_END_LOG = EV_CTRL | 1u << 8,
                   EV_STEP_END = EV_CTRL | 2u << 8, EV_SYNC = EV_CTRL | 3u << 8, EV_FRAME_END = EV_CTRL | 4u << 8,
                   EV_REBASE = EV_CTRL | 5u << 8, EV_HIGH = EV_CTRL | 6u << 8;
// Lap parity of queue position k.
constexpr uint32_t EV_LAP = 1u << 15;
__device__ __forceinline__ uint32_t lap_bit(uint32_t k) { return (~k * (EV_LAP / QLEN)) & EV_LAP; }
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

constexpr uint32_t TIA_ACK = 1u, TIA_END = 2u;
// Apply one event; returns TIA_ACK when the CPU side waits for it, and
// TIA_END when it ends the step.
__device__ __forceinline__ uint32_t tia_event(IoCtx c, uint32_t ev, TiaSide &s, const TiaOut &o) {
  if (!(ev & EV_CTRL)) {
    fc_tia_write(c, s, o.log_cap, (ev >> 8) & 0x3F, ev & 0xFF, (ev >> 16 | s.hi) - 1u);
    return 0;
  }
  const uint32_t kind = (ev >> 8) & 0x3F, slot = ev & 1, cycle = ev >> 16;
  switch (kind) {
    case 3: fc_cx_eval(c, s, 3u * (cycle | s.hi)); return TIA_ACK;
    case 4:
      fc_cx_eval(c, s, 3u * (cycle | s.hi));
      s.hi = 0;
      s.lines = 0;
      return 0;
    case 5: {
      const uint32_t n = cycle | (ev & 0xFFu) << 16;
      s.lines += n;
      s.l0 += n;
      s.ceval -= 228u * n;
      s.bar = s.bar != NO_BAR && s.bar >= n ? s.bar - n : NO_BAR;
      return 0;
    }
    case 0:
      s.log = o.log + (size_t)slot * o.log_cap;
      s.nrec = 0;
      s.bands = o.bsnap + (size_t)slot * BANDS * BAND_SNAP;
      s.band = 0;
      s.band_clk = fc_band_clk(0);
      return 0;
    case 1:
      if (s.band < BANDS) fc_bands_due(c, s, ~0u);  // band starts that the frame never reached take its last state
      o.meta[2 * slot] = s.nrec;
      o.meta[2 * slot + 1] = s.lines;
      s.log_total += s.nrec;
      s.log = nullptr;
      return 0;
    case 6: s.hi = ev & 0xFFFF0000u; return 0;
    default: return TIA_ACK | TIA_END;
  }
}
// The TIA side at the start of a step: the latches, the HMOVE bar and the
// frame's first line l0 as loaded, collisions accounted up to CPU cycle kf.
__device__ __forceinline__ TiaSide tia_start(IoCtx c, uint64_t l0, uint32_t kf) {
  const uint64_t bar = c.G64(IO_BARLO);
  TiaSide s{};
  s.ceval = 3u * kf;
  s.cx = c.G(IO_CX);
  s.bar = bar != NO_LINE && bar >= l0 && bar - l0 < (1u << 30) ? (uint32_t)(bar - l0) : NO_BAR;
  s.l0 = l0;
  return s;
}
// Single-warp form: apply an env's queued events [s.head, tail).
__device__ __noinline__ void tia_drain(IoCtx c, uint32_t q, TiaSide &side, const TiaOut &out, uint32_t tail) {
  TiaSide s = side;
  const TiaOut o = out;
  while (s.head != tail) {
    const uint32_t ev = sm32(q + 4 * (s.head & (QLEN - 1)));
    ++s.head;
    tia_event(c, ev, s, o);
  }
  c.Sset(IO_CX, s.cx);
  side = s;
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
// a * b + c on the FMA pipe.  The interpreter's loop is bound by the integer
// ALU (two cycles a warp instruction), and adds, shifts left and address
// arithmetic would all go there; with a multiplier that is not a known
// constant they run beside it.
__device__ __forceinline__ uint32_t mad(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
// Loads of the staged cartridge and the control words, which do not change
// while a work item runs: free to move past the stores of other lanes.
__device__ __forceinline__ uint32_t lds_const(uint32_t a) {
  uint32_t v;
  asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
template <uint32_t OFF>
__device__ __forceinline__ uint4 lds_const4(uint32_t a) {
  uint4 v;
  asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4 + %5];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "r"(a), "n"(OFF));
  return v;
}
// Any function of three words, bit by bit: bit 4 a + 2 b + c of LUT.
template <uint32_t LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(LUT));
  return r;
}

// Byte offsets of an env's blocks in the block's dynamic shared memory.
struct EnvOff {
  uint32_t rom, ram, io, tia, q;
};
// The block's tables come first, at fixed offsets: region table, general
// decoder's bytes, control words.  The envs' RAM follows, then the cartridge,
// then the envs' other blocks.  The hot loop loads from RAM's base + 4 *
// (address - 0x80) for every address below the cartridge's and looks at the
// value only when the address is RAM's; the cartridge (16 KB at least) behind
// the RAM and the tables before it keep those loads inside the block's memory.
constexpr uint32_t OFF_REG = 0, OFF_DEC = OFF_REG + REGION_BYTES, OFF_CTL = OFF_DEC + DEC_CTL,
                   OFF_RAM = OFF_DEC + DEC_BYTES;
static_assert(OFF_RAM % 16 == 0 && OFF_RAM >= 0x4000u, "aligned; rom - 0x4000 and ram - 0x200 stay offsets");
__host__ __device__ inline uint32_t ram_part(uint32_t envs) { return ((envs + 3) / 4 * RAM_GROUP + 15) / 16 * 16; }
// Dynamic shared memory of a block of envs with rom_stage cartridge bytes.
__host__ __device__ inline uint32_t block_smem(uint32_t rom_stage, uint32_t envs) {
  return OFF_RAM + ram_part(envs) + 4 * rom_stage + envs * ENV_SMEM;
}
// Last offset in a bank whose instruction bytes are fetched from the stage: no
// such fetch touches a hotspot (F8/F6 hotspots start at $FF6, F4's at $FF4).
__device__ __forceinline__ uint32_t scheme_fetch_limit(uint32_t scheme) {
  return scheme == 3 ? 0xFF1u : scheme ? 0xFF3u : 0xFFCu;
}
// The cartridge is staged as one word per byte: the byte and the two after it
// (an instruction in one load), and in the top byte 0x80 where no instruction
// is fetched from the stage: past limit, and a branch whose target lies past
// the bank's end (the hot loop's sums would carry into the cycle count there).
// The operand of a zero-page or absolute access to RAM or the TIA is the
// address of the first mirror, which is the same to reads and writes and the
// one that the hot loop knows; data reads see a word's first byte only.
// Words i .. i+3 of a bank of 4096 bytes at src (4-byte aligned), i a multiple
// of 4.
constexpr uint32_t REC_BAD = 0x80000000u;
__host__ __device__ inline uint32_t stage_operand(uint32_t w) {
  const uint32_t op = w & 0xFFu, form = op & 0x1Cu, a = (w >> 8) & 0x1FFFu;
  if (form == 0x04u) return a & 0x80u ? w : w & ~0x4000u;                  // zero page
  if (form != 0x0Cu || op == 0x4Cu || op == 0x6Cu) return w;               // absolute, but for the jumps
  if ((a & 0x1280u) == 0x0080u) return op | (0x80u | (a & 0x7Fu)) << 8;    // RAM
  return (a & 0x1080u) == 0 ? op | (a & 0x3Fu) << 8 : w;                   // TIA
}
__device__ __forceinline__ uint32_t stage_bad(uint32_t w, uint32_t i, uint32_t limit) {
  const uint32_t off = (w >> 8) & 0xFFu;
  return i > limit || ((w & 0x1Fu) == 0x10u && off < 0x80u && i + 2u + off > 0xFFFu) ? REC_BAD : 0u;
}
__device__ __forceinline__ uint4 stage_words(const uint8_t *src, uint32_t i, uint32_t limit) {
  const uint32_t *b = reinterpret_cast<const uint32_t *>(src + i);
  const uint32_t lo = b[0], hi = i + 4u < 4096u ? b[1] : 0u, m = 0xFFFFFFu;
  uint4 r = make_uint4(stage_operand(lo & m), stage_operand(__funnelshift_r(lo, hi, 8) & m),
                       stage_operand(__funnelshift_r(lo, hi, 16) & m), stage_operand(__funnelshift_r(lo, hi, 24) & m));
  r.x |= stage_bad(r.x, i, limit);
  r.y |= stage_bad(r.y, i + 1u, limit);
  r.z |= stage_bad(r.z, i + 2u, limit);
  r.w |= stage_bad(r.w, i + 3u, limit);
  return r;
}
// Rounds between two looks at the lanes that wait for service, unrolled, so
// that a round's last instructions overlap the next one's loads (157 cycles a
// round, 173 as a loop).  Lanes that wait are served when every lane waits, or
// when the looks since the first of them add up to more than HOLD rounds: the
// lanes of a warp run much the same code, and served together they stay in step,
// which the TIA warp, whose lanes' events then take the same branches, needs
// more than the wait costs (served at every look, 4096 sprite envs took 2.5 ms a
// step instead of 1.8).  Of 4 .. 8 rounds a look, 7 is the fastest (sprite 1.70
// ms, 6: 1.79, 8: 1.74).  When the whole warp waited and was served, a batch of
// BRIEF rounds follows instead: code full of such instructions has them a few
// rounds apart (six accesses through pointers a line: 2.6 ms a step, 3.6 without
// the brief batches; 2 rounds 4.9, 4: 2.9).
constexpr uint32_t BATCH = 7, HOLD = 16, BRIEF = 3;
template <uint32_t N> struct Rounds { static constexpr uint32_t value = N; };

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
  uint32_t unit;           // 1, as a value that the compiler does not know (see mad)
  uint32_t qtail, qhead_seen, nreq, vsync_c, vblank_c, broken;  // qhead_seen: the TIA side's cursor as last read
  uint32_t ev_hi;          // bits 16-31 of the cycles of the events as the TIA side has them
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
  __device__ __forceinline__ uint8_t &ram(uint32_t i) const { return sm8(off.ram + 4 * i); }
  __device__ __forceinline__ uint32_t rom(uint32_t i) const { return sm8(off.rom + 4 * i); }

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
    frame_no = w[22];
    l0c = (uint64_t)w[20] | (uint64_t)w[21] << 32;
    kf = (uint32_t)(k - 76ull * l0c);
    io.Sset(IO_JOY, 0xFF); io.Sset(IO_FIRE, 0);
    io.Sset(IO_STATUS, 0);
    const uint32_t *r32 = reinterpret_cast<const uint32_t *>(s + S::RAM);
#pragma unroll 8
    for (uint32_t q_ = 0; q_ < 32; ++q_) {
      const uint32_t v = r32[q_];
      for (uint32_t b = 0; b < 4; ++b) ram(4 * q_ + b) = (uint8_t)(v >> (8 * b));
    }
    for (uint32_t e = 0; e < QLEN; ++e) sm32(off.q + 4 * e) = 0;
    status = 0; instret = 0; frame_inst = 0; rounds = 0; pend = 0; vs_kf = ~0u;
    vsync_c = io.T(T_VSYNC);
    vblank_c = io.T(T_VBLANK);
    qtail = qhead_seen = nreq = broken = ev_hi = 0;
    io.Sset(IO_QHEAD, 0); io.Sset(IO_ACK, 0);
    if constexpr (!SPLIT) ts = tia_start(io, l0c, kf);
  }
  __device__ void store(uint8_t *s) const {
    uint32_t *w = reinterpret_cast<uint32_t *>(s);
    const uint64_t L0 = l0c;
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
    uint32_t *r32 = reinterpret_cast<uint32_t *>(s + S::RAM);
#pragma unroll 8
    for (uint32_t q_ = 0; q_ < 32; ++q_)
      r32[q_] = ram(4 * q_) | ram(4 * q_ + 1) << 8 | ram(4 * q_ + 2) << 16 | (uint32_t)ram(4 * q_ + 3) << 24;
  }
  __device__ uint32_t all_status() const { return status | io.G(IO_STATUS) | (SPLIT ? 0u : ts.status); }

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
  // An event at a cycle of the frame, its upper half sent ahead where it
  // differs from the last event's.  The hot loop's events need none: its
  // cycles are below the line cap.
  __device__ __forceinline__ void push_at(uint32_t ev, uint32_t cycle) {
    if (cycle >> 16 != ev_hi) {
      ev_hi = cycle >> 16;
      push(EV_HIGH | ev_hi << 16);
    }
    push(ev | cycle << 16);
  }
  __device__ __forceinline__ void drain() {
    tia_drain(io, off.q, ts, to, qtail);
    qhead_seen = ts.head;
  }
  // Collisions up to cycle t are in the latches when this returns.
  __device__ void sync_collisions(uint32_t t) {
    if constexpr (SPLIT) {
      if (broken) return;
      push_at(EV_SYNC, t);
      ++nreq;
      if (!broken && !fc_q_wait_ack(io, nreq)) stall();
      qhead_seen = qtail;  // acknowledged: the queue is empty
    } else {
      drain();
      fc_cx_eval(io, ts, 3u * t);
      io.Sset(IO_CX, ts.cx);
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
  __device__ __forceinline__ void vblank_write(uint32_t v) {
    vblank_c = v;
    if (!(v & 0x40)) io.Sset(IO_LATCH, 0);
    else if (io.G(IO_FIRE)) io.Sset(IO_LATCH, 1);
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
      vblank_write(v);
    }
    push_at(reg << 8 | v, t + 1u);
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
  __device__ __forceinline__ uint32_t idle_forward(uint32_t w, uint32_t next_op, uint32_t pc, uint32_t k0) {
    const uint32_t a = (w >> 8) & 0xFFFF;
    if ((a & 0x1285u) != 0x0284u || next_op != 0xD0u) return k0;  // INTIM (any mirror), then BNE
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
    const uint32_t opb = sm8(OFF_DEC + opcode);
    const uint32_t op = opb & 0x7F;
    const uint32_t info = sm8(OFF_DEC + 256 + opcode);
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
    push_at(EV_FRAME_END, kf);
    ev_hi = 0;
    for (uint32_t left = next_rel; left;) {  // one event, but for loaded states far past the line cap
      const uint32_t n = left < 0xFFFFFFu ? left : 0xFFFFFFu;
      push(EV_REBASE | n << 16 | n >> 16);
      left -= n;
    }
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
  // runs its own program at one instruction per round, with no leader and no
  // reconvergence.  A lone warp is bound by the round's chain of dependent
  // loads (instruction word, control words, operand), which is why the next
  // instruction's words are loaded before this one's result is computed; eight
  // warps on an SM are bound by the integer pipe, two cycles an instruction,
  // which is why sums, shifts left and counters are multiply-adds.  One round:
  // 157 cycles with one warp on an SM, 284 with eight (with the control words
  // loaded at the round's end, V in a register of its own, the branch's
  // condition in three operations, RAM addressed apart from the cartridge and
  // regions of 32 bytes: 208 and 365).  What it does not take (fc_quick, and the
  // general decoder for the rest) stops the lane in front of the instruction;
  // after every BATCH rounds the lanes that wait are looked at, and served
  // together.
  template <class Hook> __device__ __forceinline__ void run(Hook &hook);
};

// One service of a waiting lane: the frame's end, or the instruction at PC by
// the general decoder.  Returns false when the step is over.
template <bool SPLIT, class Hook>
__device__ __noinline__ bool fc_service(FastConsoleT<SPLIT> *c, Hook *h) {
  const uint32_t cap = 76u * CAP_LINES;
  // at least one instruction runs in every frame before the line cap ends it
  bool ended = c->jam || (c->kf >= cap && c->instret != c->frame_inst);
  if (!ended) {
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

// Serve a waiting lane's instruction (word rec, kind QK_*) beside the loop: the
// console stays where it is, R, G and pk come and go in registers, and what can
// be put in a form that the loop takes (the pointer in the place of an absolute
// address, a value as an immediate operand) runs in the next round.  A call takes
// 400 to 900 cycles, the general decoder's, which has the whole console in local
// memory, 2,700 to 4,500; a program with six accesses through pointers a line
// steps 512 envs in 2.6 ms, 9.8 with the general decoder for each of them.
// The result's w: QS_NO (nothing is changed: the general decoder has to),
// QS_DONE (x, y, z: R, G, pk after the instruction) or QS_RUN (x, z: the
// instruction's word, and its length and cycles, as the loop is to run it with
// the control words of entry w >> 8; y: G).  QS_SYNC: the event queue's position
// is the console's, not qi's.
constexpr uint32_t QS_NO = 0, QS_DONE = 1, QS_RUN = 2, QS_SYNC = 4;
template <bool SPLIT>
__device__ __noinline__ uint4 fc_quick(FastConsoleT<SPLIT> *m, uint32_t R, uint32_t G, uint32_t pk, uint32_t rec,
                                       uint32_t kind, uint32_t qi) {
  const uint4 no = make_uint4(0, 0, 0, QS_NO);
  const uint32_t ramb = m->off.ram - 0x200u, fdi = m->fdi;
  const IoCtx io = m->io;
  if (m->jam) return no;
  auto ctl = [&](uint32_t entry, uint32_t t) {
    return *reinterpret_cast<const uint4 *>(&sm32(OFF_CTL + CTL_TABLE * t + 16u * entry));
  };
  const uint32_t opcode = rec & 0xFFu;
  const uint4 c = ctl(opcode, 0), d = ctl(opcode, 1), f = ctl(opcode, 3);
  uint32_t pn = pk + d.z;
  uint32_t base = prmt(rec, pn, c.x), sum = base + prmt(R, rec, c.y), ea = sum & d.y;
  const uint32_t live = fdi & 0x08u ? RG_DECIMAL : ~0u;
  auto ram = [&](uint32_t a) -> uint8_t & { return sm8(ramb + 4u * (0x80u | (a & 0x7Fu))); };  // mirrored or not
  auto is_ram = [](uint32_t a) { return (a & 0x1280u) == 0x0080u; };
  // the queue's position, from the loop's to the console's
  uint32_t sync = 0;
  auto queue = [&] {
    if (!sync) m->qtail += (qi & 0xFFFFu) - (m->qtail & 0xFFu);
    sync = QS_SYNC;
  };
  // the value at address a, read at cycle t
  auto value = [&](uint32_t a, uint32_t t) -> uint32_t {
    if (is_ram(a)) return ram(a);
    if (a & 0x1000u) {
      m->hotspot(a & 0xFFFu);
      return m->rom(m->bank * 4096u + (a & 0xFFFu));
    }
    if (a & 0x80u) return fc_riot_read(io, a, 76ull * m->l0c + t);
    const uint32_t reg = a & 0xFu;
    if (reg < 8u) {
      queue();
      m->sync_collisions(t);
      return fc_cx_byte(io.V(IO_CX), reg);
    }
    return reg == 0xCu ? (io.G(IO_FIRE) || io.G(IO_LATCH) ? 0u : 0x80u) : reg == 0xDu ? 0x80u : 0u;
  };
  auto nz = [&](uint32_t v) { G = (G & ~FL_NZ) | v | (v & 0x80u) << 16; };
  auto run = [&](uint32_t entry, uint32_t word, uint32_t len) {
    return make_uint4(word, G, len, sync | QS_RUN | entry << 8);
  };
  auto done = [&] { return make_uint4(R, G, pn, sync | QS_DONE); };
  // the operation of opcode o (not a store) on v
  auto operate = [&](uint32_t o, uint32_t v) -> uint4 {
    if (((o & 0xE3u) == 0x61u || (o & 0xE3u) == 0xE1u) && (fdi & 0x08u)) {  // decimal ADC, SBC
      m->A = R & 0xFFu;
      m->fc = (G >> 8) & 1u;
      if (o & 0x80u) m->sbc(v); else m->adc(v);
      R = prmt(R, m->A, 0x3214);
      G = ((m->fz & 0xFFu) ? 1u : 0u) | m->fc << 8 | (m->fn & 0x80u) << 16 | m->fv << 25;
      return done();
    }
    const uint32_t imm = (o & 3u) == 3u ? CTL_LAX : (o & 0xE0u) | ((o & 3u) == 1u ? 9u : o & 2u);  // the immediate form
    return run(imm, v << 8, pn - pk);
  };
  // whether v to TIA register reg is more than a write of it: WSYNC, a rise of VSYNC (which ends the frame)
  auto special = [&](uint32_t reg, uint32_t v) { return reg == 2u || (reg == 0u && (v & ~m->vsync_c & 2u)); };
  auto tia = [&](uint32_t reg, uint32_t v, uint32_t t) {
    if (reg == 0u) m->vsync_c = v;
    if (reg == 1u) m->vblank_write(v);
    queue();
    m->push_at(reg << 8 | v, t + 1u);
  };
  // v to address a at the instruction's last cycle
  auto store = [&](uint32_t a, uint32_t v) -> uint4 {
    const uint32_t t = (pn >> 16) - 1u;
    v &= 0xFFu;
    if (is_ram(a)) ram(a) = (uint8_t)v;
    else if (a & 0x1000u) m->hotspot(a & 0xFFFu);
    else if (a & 0x80u) fc_riot_write(io, a, v, 76ull * m->l0c + t);
    else if (special(a & 0x3Fu, v)) return no;
    else tia(a & 0x3Fu, v, t);
    return done();
  };
  // a read-modify-write of RAM or a TIA register (operation o >> 5: shifts, DEC, INC): the result to r
  auto modify = [&](uint32_t o, uint32_t a, uint32_t &r) -> bool {
    if (!is_ram(a) && (a & 0x1080u)) return false;
    const uint32_t t = (pn >> 16) - 1u, reg = a & 0x3Fu;
    if (!is_ram(a) && reg <= 2u) return false;
    const uint32_t v = value(a, t - 2u), cin = G >> 8 & 1u;
    uint32_t cout = cin;
    switch (o >> 5) {
      case 0: r = v << 1; cout = v >> 7; break;
      case 1: r = v << 1 | cin; cout = v >> 7; break;
      case 2: r = v >> 1; cout = v & 1u; break;
      case 3: r = v >> 1 | cin << 7; cout = v & 1u; break;
      case 6: r = v - 1u; break;
      default: r = v + 1u; break;
    }
    r &= 0xFFu;
    if (is_ram(a)) {
      ram(a) = (uint8_t)r;
    } else {
      tia(reg, v, t - 1u);
      tia(reg, r, t);
    }
    G = (G & ~FL_C) | cout << 8;
    return true;
  };
  // the pointer in RAM that ea is the address of, to sum (base: without the index)
  auto pointer = [&]() -> bool {
    if (ea < 0x80u || ea == 0xFFu) return false;
    base = ram(ea) | ram(ea + 1u) << 8;
    sum = base + ((opcode & 0x10u) ? R >> 16 & 0xFFu : 0u);
    return true;
  };
  uint32_t sp = m->SP;  // pulls, calls and returns outside RAM are the general decoder's
  switch (kind) {
    case QK_PTR: {
      if (!pointer()) return no;
      const uint32_t entry = CTL_N + (opcode >> 4);
      const uint4 g = ctl(entry, 3);
      ea = sum & 0x1FFFu;
      if (sm8(OFF_REG + ea) & g.x & live) return run(entry, opcode | base << 8, d.z);
      pn += ((base ^ sum) & g.z) << 8;
      return (g.x & RG_OUT) ? store(ea, R) : operate(opcode, value(ea, (pn >> 16) - 1u));
    }
    case QK_SUM:
      if (d.y == 0) return operate(opcode & ~2u, rec >> 8 & 0xFFu);  // immediate ($EB too)
      pn += ((base ^ sum) & f.z) << 8;
      return operate(opcode, value(ea, (pn >> 16) - 1u));
    case QK_MEM: {
      pn += ((base ^ sum) & f.z) << 8;
      if (f.x & RG_OUT) return store(ea, (opcode & 3u) == 1u ? R : (opcode & 2u) ? R >> 8 : R >> 16);
      if (f.x & RG_WRAM) {
        uint32_t r;
        if (!modify(opcode, ea, r)) return no;
        nz(r);
        return done();
      }
      // a timer wait loop: its idle iterations retire with the read that ends them
      if (opcode == 0xADu && m->idle) {
        const uint32_t then = m->rom(m->bank * 4096u + ((pk + 3u) & 0xFFFu));
        pn += (m->idle_forward(rec, then, pk & 0xFFFFu, pk >> 16) - (pk >> 16)) << 16;
      }
      const uint32_t v = value(ea, (pn >> 16) - 1u);
      if (pn - pk < 0x100000u) return operate(opcode, v);
      R = prmt(R, v, 0x3214);
      nz(v);
      return done();
    }
    case QK_BIT: {
      const uint32_t v = value(ea, (pn >> 16) - 1u);
      G = (G & FL_C) | ((R & v & 0xFFu) ? 1u : 0u) | (v & 0x80u) << 16 | (v & 0x40u) << 25;
      return done();
    }
    case QK_PUSH: {
      const uint32_t p = (G >> 16 & 0x80u) | (G >> 25 & 0x40u) | 0x30u | fdi | ((G & FL_Z) ? 0u : 2u) | (G >> 8 & 1u);
      const uint4 r = store(0x100u | sp, (opcode & 0x40u) ? R : p);
      if (r.w) m->SP = (sp - 1u) & 0xFFu;
      return r;
    }
    case QK_PULL: {
      if (sp < 0x7Fu || sp == 0xFFu) return no;
      m->SP = ++sp;
      const uint32_t v = ram(sp);
      if (opcode & 0x40u) {
        R = prmt(R, v, 0x3214);
        nz(v);
      } else {
        G = ((v & 2u) ? 0u : 1u) | (v & 1u) << 8 | (v & 0x80u) << 16 | (v & 0x40u) << 25;
        m->fdi = v & 0x0Cu;
      }
      return done();
    }
    case QK_JSR:
      if (sp < 0x81u) return no;
      ram(sp) = (uint8_t)((pk + 2u) >> 8);
      ram(sp - 1u) = (uint8_t)(pk + 2u);
      m->SP = sp - 2u;
      pn = prmt(rec, pn, 0x7621);
      return done();
    case QK_RTS:
      if (sp < 0x7Fu || sp >= 0xFEu) return no;
      m->SP = sp += 2u;
      pn = prmt((ram(sp - 1u) | ram(sp) << 8) + 1u, pn, 0x7610);
      return done();
    case QK_REG:
      switch (opcode) {
        case 0xBA: R = prmt(R, sp, 0x3240); nz(sp); break;
        case 0x9A: m->SP = R >> 8 & 0xFFu; break;
        case 0x58: m->fdi = fdi & ~0x04u; break;
        case 0x78: m->fdi = fdi | 0x04u; break;
        case 0xD8: m->fdi = fdi & ~0x08u; break;
        default: m->fdi = fdi | 0x08u; break;
      }
      return done();
    case QK_COMBO: {
      if ((opcode & 0x0Fu) == 3u && !pointer()) return no;
      const uint32_t a = sum & ((opcode & 0x0Fu) == 3u ? 0x1FFFu : d.y), op = opcode >> 5;
      if (op == 5u) {  // LAX
        pn += ((base ^ sum) & f.z) << 8;
        return operate(opcode, value(a, (pn >> 16) - 1u));
      }
      if (op == 4u) return store(a, R & (R >> 8));  // SAX
      // the memory operation, then the accumulator's with its result as an immediate operand
      uint32_t r;
      if (((op == 3u || op == 7u) && (fdi & 0x08u)) || !modify(opcode, a, r)) return no;
      return run((opcode & 0xE0u) | 9u, r << 8, d.z);
    }
    case QK_AND: {  // ANC, ALR, SBX: what they set from A and the operand
      const uint32_t b = rec >> 8 & 0xFFu;
      uint32_t r, cout;
      if (opcode == 0xCBu) {
        const uint32_t ax = R & (R >> 8) & 0xFFu;
        r = (ax - b) & 0xFFu;
        cout = ax >= b ? 1u : 0u;
        R = prmt(R, r, 0x3240);
      } else {
        r = R & b & 0xFFu;
        cout = opcode == 0x4Bu ? r & 1u : r >> 7;
        if (opcode == 0x4Bu) r >>= 1;
        R = prmt(R, r, 0x3214);
      }
      nz(r);
      G = (G & ~FL_C) | cout << 8;
      return done();
    }
    case QK_NOP:  // the operand's read changes nothing but at a hotspot
      if (ea & 0x1000u) m->hotspot(ea & 0xFFFu);
      pn += ((base ^ sum) & f.z) << 8;
      return done();
    default: return no;
  }
}

template <bool SPLIT>
template <class Hook>
__device__ __forceinline__ void FastConsoleT<SPLIT>::run(Hook &hook) {
  const EnvOff o = off;
  uint32_t smb;  // the shared window's address, taken here: no load of the stage moves above the block's barrier
  asm volatile("mov.u32 %0, %1;" : "=r"(smb) : "r"((uint32_t)__cvta_generic_to_shared(g_smem)) : "memory");
  const uint32_t cap = 76u * CAP_LINES;
  const uint32_t ctl = smb + OFF_CTL, ramb = o.ram - 0x200u;
  const uint32_t k1 = unit, k4 = unit * 4u, k256 = unit * 256u;
  // R: A, X, Y and FF as bytes.  G: flags (FL_*; D and I do not change here).
  // pk: PC, and the frame's CPU cycle in the high half.  nl: the first line
  // start at or after that cycle, in the high half, over FFFF.  qi: queue
  // position, and the instructions retired since the last service in the high
  // half.  bk, bf: the bank's words, for data at 4 * (bus address) and for the
  // fetch.  live: the accesses that the lane may make in the loop (RG_*).
  // run: live, or 0 while the lane waits.
  uint32_t R, G, pk, nl, qi, bk, bf, live, run;
  uint32_t rec;
  uint4 c, d, e, f;  // control words 0-3, 4-7, 8-11, 12-15
  bool active = true;
  auto word_at = [&](uint32_t p) { return lds_const(mad(p & 0xFFFu, k4, bf)); };
  auto control = [&](uint32_t entry, uint4 &c_, uint4 &d_, uint4 &e_, uint4 &f_) {
    const uint32_t a = mad(entry, unit * 16u, ctl);
    c_ = lds_const4<0>(a);
    d_ = lds_const4<CTL_TABLE>(a);
    e_ = lds_const4<2 * CTL_TABLE>(a);
    f_ = lds_const4<3 * CTL_TABLE>(a);
  };
  auto mode = [&] { live = fdi & 0x08u ? RG_DECIMAL : ~0u; };
  auto banked = [&] {
    bk = o.rom + bank * 16384u - 0x4000u;
    bf = smb + o.rom + bank * 16384u;
  };
  auto line = [&] { nl = (((pk >> 16) + 75u) / 76u * 76u) << 16 | 0xFFFFu; };
  // the instruction at pk, and whether the loop may run it
  auto next = [&] {
    rec = word_at(pk);
    run = ((pk & 0x1000u) == 0) | (rec >= REC_BAD) | ((pk >> 16) >= cap) ? 0u : live;
    control(rec & 0xFFu, c, d, e, f);
  };
  // the console's fields to the loop's registers, and the next instruction
  auto enter = [&](bool stay) {
    R = A | X << 8 | Y << 16 | 0xFF000000u;
    G = ((fz & 0xFFu) ? 1u : 0u) | fc << 8 | (fn & 0x80u) << 16 | fv << 25;
    pk = (PC & 0xFFFFu) | min(kf, 0xFFFFu) << 16;
    line();
    qi = qtail & 0xFFu;
    banked();
    mode();
    next();
    if (stay) run = 0;
  };
  auto leave = [&] {
    A = R & 0xFF; X = (R >> 8) & 0xFF; Y = (R >> 16) & 0xFF;
    fz = G & FL_Z; fc = (G >> 8) & 1u; fn = (G >> 16) & 0x80u; fv = (G >> 25) & 0x40u;
    PC = pk & 0xFFFFu;
    if ((pk >> 16) != 0xFFFFu) kf = pk >> 16;  // a loaded cycle count past 16 bits stays as it was
    qtail += (qi & 0xFFFFu) - (qtail & 0xFFu);
    instret += qi >> 16;
  };
  // n.value rounds of the hot loop, one block of code
  auto batch = [&](auto n) {
#pragma unroll
    for (uint32_t r = 0; r < n.value; ++r) {
      // --- next instruction (branches and JMP abs: the sum is the target and the cycle)
      const uint32_t pn = mad(pk, k1, d.z);
      const uint32_t base = prmt(rec, pn, c.x);
      const uint32_t sum = mad(base, k1, prmt(R, rec, c.y));
      const bool tk = mad(G & d.w, k1, f.w) > e.w;
      const uint32_t nx = tk ? sum : pn;
      const uint32_t nrec = word_at(nx);
      // a cycle for a taken branch, another one at a page crossing
      uint32_t pnext = mad((base ^ sum) & (tk ? 0x100u : f.z), k256, nx);
      if (tk) pnext = mad(k256, 256u, pnext);
      // --- operand
      const uint32_t ea = sum & d.y;
      const uint32_t put = sm8(OFF_REG + ea) & f.x & run;
      const uint32_t at = mad(ea, k4, ea >= 0x1000u ? bk : ramb);
      const uint32_t y = prmt(sm8(at), sum, d.x);
      const uint32_t x = prmt(R, y, c.z);
      uint4 cn, dn, en, fn;  // the next instruction's control words, on their way while this one is computed
      control(nrec & 0xFFu, cn, dn, en, fn);
      // --- result, of x and y ^ e.y
      const uint32_t xo = lop3<0x96>(x, y, e.y);
      const uint32_t raw = mad(lop3<0x60>(x, y, e.y), e.z, mad(xo, f.y, prmt(G, k1, e.w)));
      const uint32_t s = __funnelshift_r(raw, 0, f.w);
      // --- commit; nothing in put: the lane waits, or waits from here on for the general decoder
      const bool out = (put & RG_OUT) != 0;
      if (put & RG_WRAM) sm8(at) = (uint8_t)s;
      // events past another lap's bit: the lap's complement is bit 15 of -qi * 1024 - 1024
      const uint32_t ev = mad(ea, k256, s) | (mad(qi, unit * (0u - EV_LAP / QLEN), 0u - EV_LAP / QLEN) & EV_LAP);
      if (out) vsm32(mad(qi & (QLEN - 1), k4, o.q)) = prmt(ev, pnext, 0x7610);
      // one step: no instruction is longer than a line (a waiting lane's is set again when it is served)
      if (pnext > nl) nl = mad(k256, 76u << 8, nl);
      if (put & RG_WSYNC) pnext = prmt(pnext, nl, 0x7610);  // on to the next line's first cycle
      const bool done = put != 0;  // in single statements: a block of them would become a branch
      const uint32_t gn = (G & ~e.x) | (prmt(s, lop3<0x14>(x, s, xo), FL_SEL) & e.x);  // V: (x ^ s) & ~(x ^ y)
      if (done) R = prmt(R, s, c.w);
      if (done) G = gn;
      if (done) pk = pnext;
      if (done) qi = mad(k256, 256u, qi);
      if (out) qi = mad(k1, k1, qi);
      // bit 31: no instruction word there, the PC outside the cartridge, the line cap
      const uint32_t stop = nrec | mad(pnext, unit * 0xFFF80000u, 0xFFF80000u) | mad(pnext, 0u - unit, (cap << 16) - 1u);
      run = !done | ((int)stop < 0) ? 0u : live;
      rec = nrec; c = cn; d = dn; e = en; f = fn;
    }
  };
  enter(jam != 0);
  uint32_t held = 0, act = wmask;
  for (;;) {
    batch(Rounds<BATCH>{});
    // --- service: waiting lanes, and queues without room for another batch
    rounds += BATCH;
    const bool full = ((qi - qhead_seen) & 0xFFu) > QLEN - BATCH;
    uint32_t m = __ballot_sync(wmask, ((run == 0) | full) & active);
    if (m == 0) continue;
    m = __ballot_sync(wmask, (run == 0) & active);
    if (m != 0 && (m == act || (held += BATCH) > HOLD)) {
      held = 0;
      bool slow;
      for (;;) {
        ++rounds;  // in which each waiting lane's instruction is served
        slow = active & (run == 0);
        if (slow) {
          rec = word_at(pk);
          const uint32_t kind = sm8(OFF_DEC + DEC_QUICK + (rec & 0xFFu));
          const bool other = (kind == QK_NONE) | (rec >= REC_BAD) | ((pk & 0x1000u) == 0) | ((pk >> 16) >= cap);
          if (!other & (kind == QK_PTR)) {  // the common case, a third of a call's time
            const uint32_t z = (rec >> 8) + ((rec & 0x10u) ? 0u : R >> 8) & 0xFFu, za = ramb + 4u * z;
            const uint32_t w = (rec & 0xFFu) | sm8(za) << 8 | sm8(za + 4u) << 16;
            control(CTL_N + (rec >> 4 & 0xFu), c, d, e, f);
            const uint32_t at = ((w >> 8) + prmt(R, w, c.y)) & 0x1FFFu;
            if ((z >= 0x80u) & (z != 0xFFu) & ((sm8(OFF_REG + at) & f.x & live) != 0)) {
              rec = w;
              run = live;
              line();
              slow = false;
            }
          }
          if (!other & slow) {
            const uint4 r = fc_quick<SPLIT>(this, R, G, pk, rec, kind, qi);
            if (r.w & QS_SYNC) qi = (qi & 0xFFFF0000u) | (qtail & 0xFFu);
            banked();
            if (r.w & QS_DONE) {
              R = r.x; G = r.y; pk = r.z;
              line();
              qi += 1u << 16;
              mode();
              next();
              slow = false;
            } else if (r.w & QS_RUN) {
              rec = r.x; G = r.y;
              control(r.w >> 8, c, d, e, f);
              d.z = r.z;
              run = live;
              line();
              slow = false;
            }
            if ((r.w & QS_SYNC) && jam) run = 0;  // the TIA side stalled
          }
        }
        // lanes in step with one another, all served: most likely they soon wait together again.  The single-warp
        // form, whose rounds are not the longer part of a step, is 7 % slower with the second copy of the loop.
        if (!SPLIT || m != act) break;
        if (__any_sync(wmask, slow | (active & (((qi - qhead_seen) & 0xFFu) > QLEN - BRIEF)))) break;
        batch(Rounds<BRIEF>{});
        rounds += BRIEF;
        if (__any_sync(wmask, active & (run != 0))) break;
      }
      if (__any_sync(wmask, slow)) {
        if (slow) {
          leave();
          active = fc_service<SPLIT, Hook>(this, &hook);
          enter(!active);
        }
        act = __ballot_sync(wmask, active);
        if (act == 0) break;
      }
    }
    // room for a batch of events
    if constexpr (SPLIT) {
      if (active & (((qi - qhead_seen) & 0xFFu) > QLEN - BATCH)) {
        const uint32_t qt = qtail + (qi & 0xFFFFu) - (qtail & 0xFFu);
        qhead_seen = fc_q_wait_room(io, qt, BATCH);
        if (qt - qhead_seen > QLEN - BATCH) { stall(); run = 0; }
      }
    } else {
      if (__any_sync(wmask, ((qi - qhead_seen) & 0xFFu) > QLEN - BATCH)) {
        const uint32_t qt = qtail + (qi & 0xFFFFu) - (qtail & 0xFFu);
        tia_drain(io, off.q, ts, to, qt);
        qhead_seen = qt;
      }
    }
    __syncwarp(wmask);
  }
  leave();
}

}  // namespace atari
