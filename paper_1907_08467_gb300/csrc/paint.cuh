// Row painter: replays a frame's TIA writes with one thread per band of
// BAND_ROWS rows.
//
// Every thread holds its own register file (bytes in shared memory), starts
// from the band snapshot that the interpreter left and walks the records of
// its own rows only, so a record is applied once per frame.  A row is built
// as two 160-bit planes (five words each) holding the colour class of every
// column, 32 columns per operation; the planes turn into pixels eight columns
// at a time, with a byte permute that picks from the four class colours.
//
// Painting, maximum and resampling of 32768 banked envs take 1.94 ms, of 4096
// sprite envs 0.22 ms, 37,237 warp-instructions per env-step, at half of the
// issue slots.  With a lane per column instead (every lane applies every record
// to its own copy of the registers): 182,482 warp-instructions, 7.1 and 0.85 ms.
// With every object's mask rebuilt for every piece of a row: 2.4 and 0.27 ms;
// with the whole block resampling after a barrier and the kept planes copied by
// the painting warps: 2.17 and 0.24 ms.
#pragma once
#include <cstdint>

#include "device_machine.cuh"
#include "fast_console.cuh"

namespace atari {

constexpr uint32_t FILE_STRIDE = 44;          // bytes of a thread's register file (11 words: an odd stride)
constexpr uint32_t ROW_WORDS = 42;            // 40 words of pixels; with the skew below, threads BAND_ROWS rows
                                              // apart use different banks for 8-byte accesses
__device__ __forceinline__ uint32_t row_off(uint32_t r) { return 4u * (ROW_WORDS * r + 2u * (r / BAND_ROWS)); }
constexpr uint32_t PAINT_FRAME = 4 * (ROW_WORDS * FRAME_H + 2 * BANDS);  // bytes of a frame in shared memory

// Objects whose masks a register write can change.
constexpr uint32_t OB_A = 1u, OB_B = 2u, OB_BL = 4u, OB_PF = 8u, OB_ALL = 15u;  // player and missile 0, 1, ball, playfield
// What a register write does to the picture: its slot of the register file,
// 0x40 = it only sets that slot, 0x80 = the colours may change too, 0xC0 = it
// needs its own case; the objects it may change << 8.
__device__ __forceinline__ uint32_t paint_reg(uint32_t reg) {
  switch (reg) {
    case 0x01: return 0x80u | T_VBLANK;
    case 0x04: return 0x40u | T_NUSIZ0 | OB_A << 8;
    case 0x05: return 0x40u | T_NUSIZ1 | OB_B << 8;
    case 0x06: case 0x07: case 0x08: case 0x09: return 0x80u | (reg - 2);
    case 0x0A: return 0x40u | T_CTRLPF | (OB_BL | OB_PF) << 8;
    case 0x0B: return 0x40u | T_REFP0 | OB_A << 8;
    case 0x0C: return 0x40u | T_REFP1 | OB_B << 8;
    case 0x0D: case 0x0E: case 0x0F: return 0x40u | (reg - 2) | OB_PF << 8;
    case 0x1D: return 0x40u | T_ENAM0 | OB_A << 8;
    case 0x1E: return 0x40u | T_ENAM1 | OB_B << 8;
    case 0x10: case 0x12: case 0x25: case 0x28: return 0xC0u | OB_A << 8;
    case 0x11: case 0x13: case 0x26: case 0x29: return 0xC0u | OB_B << 8;
    case 0x14: case 0x1F: case 0x27: return 0xC0u | OB_BL << 8;
    case 0x1B: case 0x1C: return 0xC0u;  // the graphics shown depend on the vertical delays
    case 0x2A: return 0xC0u | (OB_A | OB_B | OB_BL) << 8;
    default: return reg >= 0x20 && reg <= 0x24 ? 0x40u | (T_HMP0 + reg - 0x20) : 0xC0u;
  }
}

// Offsets into shared memory of what the threads of a block share.
struct PaintTabs {
  uint32_t luma;    // 128 bytes: colour index -> output byte
  uint32_t regs;    // 64 half words: paint_reg()
  uint32_t spread;  // 256 words: bit i -> bit 4 i
  uint32_t cols;    // 84 pairs: source byte of an output column, its three weights in units of 1/21 column
};
constexpr uint32_t PAINT_TABS = 1024 + 128 + 128 + 672;
__device__ __forceinline__ uint32_t spread_nibbles(uint32_t b) {
  uint32_t x = (b | b << 12) & 0x000F000Fu;
  x = (x | x << 6) & 0x03030303u;
  return (x | x << 3) & 0x11111111u;
}

// Per-byte maximum of two words of four pixels.
__device__ __forceinline__ uint32_t max_u8x4(uint32_t a, uint32_t b) {
  // 16-bit maxima: the high bytes decide there whatever the low bytes are
  const uint32_t m = 0x00FF00FFu;
  return (__vmaxu2(a, b) & ~m) | __vmaxu2(a & m, b & m);
}

struct RowPainter {
  PaintTabs tabs;
  uint32_t file;       // offset of this thread's register file
  uint32_t bar;        // frame-relative line of the HMOVE bar, or 0xFFFF
  uint32_t a[5], b[5], l[5], f[5];  // masks: player and missile 0, player and missile 1, ball, playfield
  uint32_t c0[5], c1[5];  // class planes of the row being painted
  uint32_t stale;      // OB_*: the masks that the registers have left behind

  __device__ __forceinline__ uint32_t F(uint32_t s) const { return sm8(file + s); }
  __device__ __forceinline__ void Fset(uint32_t s, uint32_t v) const { sm8(file + s) = (uint8_t)v; }

  // Mask words of one object: pattern words u0..u2 at pixel 0, moved to pos.
  static __device__ __forceinline__ void place(uint32_t *m, const M160 &u, uint32_t pos) {
    const M160 r = rot160(u, pos);
    m[0] |= r.w0; m[1] |= r.w1; m[2] |= r.w2; m[3] |= r.w3; m[4] |= r.w4;
  }
  // Rebuild the stale masks.  A write stales one object as a rule, and the
  // rows of a warp's threads, two apart, stale the same one at the same time.
  __device__ __forceinline__ void refresh() {
    const uint32_t ctrl = F(T_CTRLPF);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (!(stale & (p ? OB_B : OB_A))) continue;
      uint32_t *m = p ? b : a;
#pragma unroll
      for (int w = 0; w < 5; ++w) m[w] = 0;
      const uint32_t nus = F(T_NUSIZ0 + p);
      const uint32_t g = p ? ((F(T_VDELP1) & 1) ? F(T_GRP1_O) : F(T_GRP1_N)) : ((F(T_VDELP0) & 1) ? F(T_GRP0_O) : F(T_GRP0_N));
      if (g) place(m, player_base(g, F(T_REFP0 + p), nus), F(T_P0 + p));
      if ((F(T_ENAM0 + p) & 2) && !(F(T_RESMP0 + p) & 2)) place(m, missile_base(nus), F(T_M0 + p));
    }
    if (stale & OB_BL) {
#pragma unroll
      for (int w = 0; w < 5; ++w) l[w] = 0;
      if (((F(T_VDELBL) & 1) ? F(T_ENABL_O) : F(T_ENABL_N)) & 2) place(l, ball_base(ctrl), F(T_BL));
    }
    if (stale & OB_PF) {
      const M160 pf = pf_mask(F(T_PF0), F(T_PF1), F(T_PF2), ctrl);
      f[0] = pf.w0; f[1] = pf.w1; f[2] = pf.w2; f[3] = pf.w3; f[4] = pf.w4;
    }
    stale = 0;
  }
  // Columns [x0, x1) of the row take the current registers' classes.  Normal
  // priority: player 0 and missile 0 (class 1), then player 1 and missile 1
  // (class 2), then playfield and ball (class 3), then background (class 0);
  // in score mode the playfield takes class 1 left of column 80 and 2 right of
  // it, and the ball shows where there is no playfield.  Playfield priority
  // (CTRLPF bit 2): playfield and ball first, score mode off.
  __device__ __forceinline__ void take(uint32_t x0, uint32_t x1) {
    if (stale) refresh();
    const uint32_t ctrl = F(T_CTRLPF);
    const uint32_t front = (ctrl & 4) ? ~0u : 0u;
    const uint32_t score = (ctrl & 6) == 2 ? ~0u : 0u;
#pragma unroll
    for (int w = 0; w < 5; ++w) {
      const uint32_t m = below(x1, w) & ~below(x0, w);
      const uint32_t right = score & (w < 2 ? 0u : w == 2 ? 0xFFFF0000u : ~0u), left = score & ~right;
      const uint32_t ab = (a[w] | b[w]) & ~front, both = l[w] & ~(f[w] & score);
      const uint32_t lo = (f[w] & ~right) | both, hi = (f[w] & ~left) | both;
      const uint32_t n0 = a[w] | (lo & ~ab), n1 = (b[w] & ~a[w]) | (hi & ~ab);
      c0[w] = (c0[w] & ~m) | (n0 & m);
      c1[w] = (c1[w] & ~m) | (n1 & m);
    }
  }
  // The four class colours as output bytes.
  __device__ __forceinline__ uint32_t palette() const {
    if (F(T_VBLANK) & 2) return sm8(tabs.luma) * 0x01010101u;
    return sm8(tabs.luma + (F(T_COLUBK) >> 1)) | sm8(tabs.luma + (F(T_COLUP0) >> 1)) << 8 |
           sm8(tabs.luma + (F(T_COLUP1) >> 1)) << 16 | sm8(tabs.luma + (F(T_COLUPF) >> 1)) << 24;
  }
  // Eight columns from their class bits: b0, b1 the planes' bytes, off the
  // columns to leave out (their pixels become 0).
  __device__ __forceinline__ uint2 pixels8(uint32_t pal, uint32_t b0, uint32_t b1, uint32_t off) const {
    uint32_t sel = sm32(tabs.spread + 4u * b0) | sm32(tabs.spread + 4u * b1) << 1;
    if (off) sel |= sm32(tabs.spread + 4u * (off & 0xFFu)) << 2;  // selector bit 2: the second operand, zero
    return make_uint2(__byte_perm(pal, 0, sel), __byte_perm(pal, 0, sel >> 16));
  }
  // Write columns [x0, x1) of the row at byte offset `row`, x0 = 0 or where
  // the last write of the row ended, as the maximum with what is there (over:
  // a frame painted over another one) or with nothing.  barred: the HMOVE bar
  // blanks columns 0..7.  Columns of a group that are left out are 0 until
  // the next write of the row.
  __device__ __forceinline__ void emit(bool over, uint32_t x0, uint32_t x1, uint32_t row, bool barred) {
    const uint32_t pal = palette();
    const uint32_t pal0 = barred ? sm8(tabs.luma) * 0x01010101u : pal;
    if (x0 == 0 && x1 == 160) {
#pragma unroll
      for (int g = 0; g < 20; ++g) {
        uint2 p = pixels8(g == 0 ? pal0 : pal, (c0[g >> 2] >> (8 * (g & 3))) & 0xFFu,
                          (c1[g >> 2] >> (8 * (g & 3))) & 0xFFu, 0);
        uint2 *d = reinterpret_cast<uint2 *>(&sm32(row + 8u * g));
        if (over) {
          const uint2 q = *d;
          p = make_uint2(max_u8x4(q.x, p.x), max_u8x4(q.y, p.y));
        }
        *d = p;
      }
      return;
    }
#pragma unroll 1
    for (uint32_t g = x0 >> 3; g < (x1 + 7u) >> 3; ++g) {
      const uint32_t w = g >> 2, sh = 8u * (g & 3u), xa = 8u * g;
      const uint32_t p0 = w == 0 ? c0[0] : w == 1 ? c0[1] : w == 2 ? c0[2] : w == 3 ? c0[3] : c0[4];
      const uint32_t p1 = w == 0 ? c1[0] : w == 1 ? c1[1] : w == 2 ? c1[2] : w == 3 ? c1[3] : c1[4];
      // columns of the group outside [x0, x1)
      const uint32_t off = (x0 > xa ? (1u << (x0 - xa)) - 1u : 0u) | (x1 < xa + 8u ? 0xFFu << (x1 - xa) & 0xFFu : 0u);
      const uint2 p = pixels8(g == 0 ? pal0 : pal, (p0 >> sh) & 0xFFu, (p1 >> sh) & 0xFFu, off | 0x100u);
      uint2 *d = reinterpret_cast<uint2 *>(&sm32(row + 8u * g));
      uint2 q = make_uint2(0, 0);
      if (over | (x0 > xa)) q = *d;
      *d = make_uint2(max_u8x4(q.x, p.x), max_u8x4(q.y, p.y));
    }
  }

  // Start from a band snapshot (48 bytes); returns the index of the band's first record.
  __device__ __forceinline__ uint32_t start(const uint8_t *snap) {
    const uint4 *s = reinterpret_cast<const uint4 *>(snap);
    const uint4 a = s[0], b = s[1], c = s[2];
    const uint32_t w[10] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y};
#pragma unroll
    for (int q = 0; q < 10; ++q) sm32(file + 4u * q) = w[q];
    bar = c.y >> 16;
    stale = OB_ALL;
    return c.z;
  }

  // Paint rows [r0, r1) of a frame of n_lines lines from its records
  // [ri, n_rec) (clock << 14 | register << 8 | value); over: as the maximum
  // with what is in the frame.
  __device__ __forceinline__ void paint(bool over, uint32_t r0, uint32_t r1, uint32_t n_lines, const uint32_t *recs, uint32_t ri,
                                        uint32_t n_rec, uint32_t frame) {
    // the record at ri and the next one; ~0: a clock beyond every line
    uint32_t rec = ri < n_rec ? recs[ri] : ~0u, ahead = ri + 1 < n_rec ? recs[ri + 1] : ~0u;
#pragma unroll 1
    for (uint32_t r = r0; r < r1; ++r) {
      const uint32_t line = WINDOW_Y0 + r, cl = 228u * line, row = frame + row_off(r);
      if (line >= n_lines) {
        const uint32_t black = sm8(tabs.luma) * 0x01010101u;
        for (uint32_t q = 0; q < 40; ++q) {
          uint32_t &d = sm32(row + 4u * q);
          d = over ? max_u8x4(d, black) : black;
        }
        continue;
      }
      uint32_t xs = 0, xe = 0;  // classes taken up to xs, pixels written up to xe
      for (;;) {
        // apply records up to one that changes the picture right of xs (classes) or xe (colours)
        uint32_t stop = 160u;
        bool colour = true;
        while ((rec >> 14) < cl + 228u) {
          const uint32_t clk = rec >> 14, reg = (rec >> 8) & 0x3Fu, v = rec & 0xFFu;
          const uint32_t x = clk > cl + 68u ? clk - cl - 68u : 0u;
          const uint32_t word = *reinterpret_cast<const uint16_t *>(&sm8(tabs.regs + 2u * reg));
          const uint32_t info = word & 0xFFu;
          uint32_t slot = info & 0x3Fu, val = v;
          uint32_t hit = word >> 8;  // the objects that change
          if (info < 0xC0u) {
            const bool change = F(slot) != v;
            if (change & ((info & 0x80u) != 0) & (x > xe)) { stop = x; break; }
            if (!change) hit = 0;
          } else {
            uint32_t from, to;  // the delayed copy that the write makes
            switch (reg) {
              // GRP0 sets P0's new graphic and copies P1's new graphic to its old one (shown when the vertical
              // delay is on); GRP1 likewise, and the ball's enable to its delayed copy
              case 0x1B:
                slot = T_GRP0_N; from = T_GRP1_N; to = T_GRP1_O;
                hit = (!(F(T_VDELP0) & 1) && v != F(slot) ? OB_A : 0u) | ((F(T_VDELP1) & 1) && F(from) != F(to) ? OB_B : 0u);
                break;
              case 0x1C:
                slot = T_GRP1_N; from = T_GRP0_N; to = T_GRP0_O;
                hit = (!(F(T_VDELP1) & 1) && v != F(slot) ? OB_B : 0u) | ((F(T_VDELP0) & 1) && F(from) != F(to) ? OB_A : 0u) |
                      ((F(T_VDELBL) & 1) && ((F(T_ENABL_O) ^ F(T_ENABL_N)) & 2) ? OB_BL : 0u);
                break;
              case 0x1F: slot = T_ENABL_N; hit = !(F(T_VDELBL) & 1) && ((F(slot) ^ v) & 2) ? hit : 0u; break;
              case 0x10: case 0x11: case 0x12: case 0x13: case 0x14:
                slot = T_P0 + reg - 0x10;
                val = reg < 0x12 ? fc_res_pos(clk, 5, 3) : fc_res_pos(clk, 4, 2);
                hit = F(slot) != val ? hit : 0u;
                break;
              case 0x25: case 0x26: case 0x27: slot = T_VDELP0 + reg - 0x25; hit = ((F(slot) ^ v) & 1) ? hit : 0u; break;
              case 0x28: case 0x29: slot = T_RESMP0 + reg - 0x28; break;
              default: slot = T_VSYNC; break;  // HMOVE, HMCLR
            }
          }
          if ((hit != 0) & (x > xs)) { stop = x; colour = false; break; }
          if (info >= 0xC0u) {
            if (reg == 0x1B || reg == 0x1C) {  // the delayed copies
              Fset(reg == 0x1B ? T_GRP1_O : T_GRP0_O, F(reg == 0x1B ? T_GRP1_N : T_GRP0_N));
            }
            if (reg == 0x1C) Fset(T_ENABL_O, F(T_ENABL_N));
            if (reg >= 0x28) {
              if (reg == 0x2A) {
                for (uint32_t q = 0; q < 5; ++q) Fset(T_P0 + q, fc_hm_move(F(T_P0 + q), F(T_HMP0 + q)));
                if (clk % 228u < 68u) bar = clk / 228u;
              } else if (reg == 0x2B) {
                for (uint32_t q = 0; q < 5; ++q) Fset(T_HMP0 + q, 0);
              } else if ((F(slot) & 2) && !(v & 2)) {  // the missile leaves the player it was locked to
                const uint32_t i = reg - 0x28, sz = F(T_NUSIZ0 + i) & 7u;
                Fset(T_M0 + i, (F(T_P0 + i) + (sz == 5 ? 8u : sz == 7 ? 16u : 4u)) % 160u);
              }
            }
          }
          stale |= hit;
          Fset(slot, val);
          ++ri;
          rec = ahead;
          ahead = ri + 1 < n_rec ? recs[ri + 1] : ~0u;
        }
        if (stop > xs) { take(xs, stop); xs = stop; }
        if (colour) {
          emit(over, xe, stop, row, line == bar);
          xe = stop;
          if (stop == 160u) break;
        }
      }
    }
  }
};

// The threads' register-effect and spread tables, and the colour table.
__device__ __forceinline__ void paint_tables(const PaintTabs &t, const uint8_t *luma) {
  for (uint32_t i = threadIdx.x; i < 128; i += blockDim.x) sm8(t.luma + i) = luma ? luma[i] : (uint8_t)(2 * i);
  for (uint32_t i = threadIdx.x; i < 64; i += blockDim.x) *reinterpret_cast<uint16_t *>(&sm8(t.regs + 2 * i)) = (uint16_t)paint_reg(i);
  for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) sm32(t.spread + 4 * i) = spread_nibbles(i);
}

}  // namespace atari
