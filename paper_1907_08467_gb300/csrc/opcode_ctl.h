// Control words and tables of the batched interpreter, built on the host from
// the decode table and copied to shared memory by every block.
//
// The interpreter runs every common instruction through one branch-free
// sequence (fast_console.cuh); an opcode's control words tell it which operand
// bytes, index, registers, adder inputs and flags the instruction uses.  On
// sm_103a a switch on the opcode costs about 30 cycles for each level of its
// compare tree (one warp, warp-uniform value: 49 cycles for 2 cases, 178 for
// 36, 241 for 150), and a jump table 100 cycles while its handlers fit the
// instruction cache's first level and 280-450 when they do not, so data beats
// code here.  The sequence is bound by the integer pipe (two cycles a warp
// instruction), so the words come in the form in which they are used, with as
// little unpacking as possible: 64 bytes an opcode, four 16-byte loads, each
// from a table of its own (lanes at different opcodes then fall into eight
// bank groups, not two).
#pragma once
#include <cstdint>
#include <cstring>

#include "device_machine.cuh"

namespace atari {

// What an access may fall on, a byte per address of the 13-bit bus: RAM (its
// zero-page addresses), RAM again for a result that is stored, the cartridge
// but for its hotspots, TIA registers whose writes are only passed on, WSYNC,
// and address 0 for an instruction without an access.  ADC and SBC look at
// bits of their own (RAM or cartridge, no access), which a lane in decimal mode
// masks out.  Every other address (mirrors too) is not the loop's.  A byte for
// each address costs 8 KB a block and saves the shift, the mirror masks and
// four compares a round that a table of 32-byte granules needs.
constexpr uint32_t RG_RAM = 1u, RG_WRAM = 2u, RG_CART = 4u, RG_OUT = 8u, RG_WSYNC = 16u, RG_NONE = 32u, RG_MSUM = 64u,
                   RG_ISUM = 128u, RG_DECIMAL = ~(RG_MSUM | RG_ISUM);

// Instructions that the loop does not take, or not at the address that they
// came with, but that need little: served beside the loop (fc_quick).
enum Quick : uint8_t {
  QK_NONE = 0,
  QK_PTR,    // (zp,X) and (zp),Y: the access runs in the loop once the pointer is read
  QK_BIT,
  QK_PUSH, QK_PULL, QK_JSR, QK_RTS,
  QK_REG,    // TSX, TXS, and the I and D flags
  QK_MEM,    // an access to RIOT, a TIA register that is read or does more than go into the queue, a hotspot
  QK_SUM,    // ADC, SBC: the same, or decimal
  QK_COMBO,  // undocumented: read-modify-write with an accumulator operation, SAX, LAX through a pointer
  QK_AND,    // undocumented: ANC, ALR, SBX
  QK_NOP     // undocumented: a NOP that reads memory
};

// Word by word (byte selectors are those of a 32-bit byte permute and use the
// low half):
//   0  selector of the address base from (instruction bytes, next PC)
//   1  selector of the index from (A X Y FF, instruction bytes)
//   2  selector of the adder's x from (A X Y FF, operand)
//   3  selector of the written registers from (A X Y FF, result)
//   4  selector of the operand from (memory byte, sum of base and index)
//   5  address mask
//   6  length | cycles << 16
//   7  branch: flag bits of which any takes it
//   8  flag bits that are written
//   9  operand invert
//  10  multiplier of (x & y): 0 eor, 1 and / or, 2 add, 513 shift right
//  11  selector of the carry-in from (flags, 1) (the flags' byte 1 is the carry, byte 5 a zero); a branch's
//      threshold
//  12  what the access may fall on (nothing: not the loop's instruction)
//  13  multiplier of (x ^ y): 0 and, 1 otherwise
//  14  page-cross penalty << 8
//  15  right shift of the sum (its low 5 bits); a branch is taken when word 15 + (flags & word 7) > word 11, unsigned
// Words 4 i .. 4 i + 3 of entry o are at CTL_TABLE i + 16 o.  Entries 0 .. 255
// are the opcodes'; entry CTL_N + i is opcode 16 i + 1's, an access through a
// pointer, with the pointer in the place of an absolute address; entry CTL_LAX
// is LAX with an immediate operand, which no opcode is.
constexpr uint32_t CTL_WORDS = 16, CTL_N = 256, CTL_LAX = CTL_N + 16, CTL_ENTRIES = CTL_N + 24, CTL_TABLE = 16 * CTL_ENTRIES;
static_assert(CTL_TABLE % 128 == 0, "the four tables start in the same bank");
constexpr uint32_t CTL_BYTES = 4 * CTL_WORDS * CTL_ENTRIES;
// General decoder's bytes, quick kinds, control words.
constexpr uint32_t DEC_QUICK = 512, DEC_CTL = 768, DEC_BYTES = DEC_CTL + CTL_BYTES;
constexpr uint32_t REGION_BYTES = 8192;          // what each address of the bus is

// Flags as the interpreter holds them: the 9-bit result that set them (bits 0-7
// zero when Z is set, bit 8 C), its low byte again (bit 23 is N: BIT and PLP can
// set N and Z both, so N has its own copy), and a byte whose bit 7 is V.  The
// bits that no FL_ names are not looked at; byte 1 holds C alone.
constexpr uint32_t FL_NZ = 0xFFu | 0xFFu << 16, FL_C = 0x100u, FL_Z = 0xFFu, FL_N = 0x80u << 16, FL_V = 0x80u << 24;
constexpr uint32_t FL_SEL = 0x4010u;           // selector of the flags from (result, overflow byte)

__host__ __device__ inline uint32_t region_byte(uint32_t at, uint32_t scheme) {
  if (at >= 0x1000u) return scheme && at >= 0x1FF4u && at <= 0x1FFBu ? 0u : RG_CART | RG_MSUM;
  if (at >= 0x80u) return at < 0x100u ? RG_RAM | RG_WRAM | RG_MSUM : 0u;
  return at == 0u ? RG_NONE | RG_ISUM : at == 2u ? RG_WSYNC : at > 2u && at < 0x40u ? RG_OUT : 0u;
}

inline Quick quick_kind(uint32_t op, uint32_t mode) {
  const bool ptr = mode == IZX || mode == IZY;
  switch (op) {
    case O_ADC: case O_SBC: return ptr ? QK_PTR : QK_SUM;
    case O_LDA: case O_STA: case O_AND: case O_ORA: case O_EOR: case O_CMP:
      if (ptr) return QK_PTR;
      break;
    case O_LDX: case O_LDY: case O_STX: case O_STY: case O_CPX: case O_CPY: case O_ASL: case O_ROL: case O_LSR:
    case O_ROR: case O_INC: case O_DEC: break;
    case O_LAX:
      if (ptr) return QK_COMBO;
      break;
    case O_SLO: case O_RLA: case O_SRE: case O_RRA: case O_DCP: case O_ISC: case O_SAX: return QK_COMBO;
    case O_ANC: case O_ALR: case O_SBX: return QK_AND;
    case O_NOP: return mode == IMP || mode == IMM ? QK_NONE : QK_NOP;
    case O_BIT: return QK_BIT;
    case O_PHA: case O_PHP: return QK_PUSH;
    case O_PLA: case O_PLP: return QK_PULL;
    case O_JSR: return QK_JSR;
    case O_RTS: return QK_RTS;
    case O_TSX: case O_TXS: case O_CLI: case O_SEI: case O_CLD: case O_SED: return QK_REG;
    default: return QK_NONE;
  }
  return mode >= ZP && mode <= ABY ? QK_MEM : QK_NONE;
}

// dec: per opcode, operation | mode << 8 | cycles << 12 | page-cross penalty << 16 (0: halts the CPU).
// out: DEC_BYTES, of which the quick kinds and the control words are written.
inline void build_ctl(const uint32_t *dec, uint8_t *out) {
  memset(out + DEC_CTL, 0, CTL_BYTES);
  for (uint32_t e = 0; e <= CTL_LAX; ++e) {
    const bool ptr = e >= CTL_N && e < CTL_LAX;  // the pointer read: the index comes after it
    const uint32_t o = ptr ? (e - CTL_N) * 16 + 1 : e == CTL_LAX ? 0xA7u : e;
    const uint32_t op = dec[o] & 0xFF, org = (dec[o] >> 8) & 0xF;
    const uint32_t mode = e == CTL_LAX ? (uint32_t)IMM : !ptr ? org : org == IZY ? ABY : ABS;
    if (e < CTL_N) out[DEC_QUICK + o] = quick_kind(op, mode);
    uint32_t cyc = (dec[o] >> 12) & 0xF;
    const uint32_t pen = (dec[o] >> 16) & 1;
    const uint32_t len = org <= ACC ? 1u : org >= ABS && org <= IND ? 3u : 2u;
    // zero bytes: byte 3 of the instruction bytes, byte 1 of the operand
    uint32_t selB = 0x3333, selI = 0x7777, selX = 0x5555, selD = 0x3210, selV = 0x7654, em = 0;
    uint32_t bm = 0, m2 = 1, inv = 0, gm = 0, k = 2, selC = 0x5555, one = 0, a = 0, regions = RG_NONE;
    bool mem = true, slow = op == O_JAM;
    switch (mode) {
      case IMM: selB = 0x3331; mem = false; break;
      case ZP: selB = 0x3331; em = 0xFF; break;
      case ZPX: selB = 0x3331; selI = 0x7771; em = 0xFF; break;
      case ZPY: selB = 0x3331; selI = 0x7772; em = 0xFF; break;
      case ABS: selB = 0x3321; em = 0x1FFF; break;
      case ABX: selB = 0x3321; selI = 0x7771; em = 0x1FFF; break;
      case ABY: selB = 0x3321; selI = 0x7772; em = 0x1FFF; break;
      case ACC: selI = 0x7770; mem = false; break;  // the operand is the sum of base and index: A
      // base and sum keep the cycle in their high halves: the sum is the next PC and cycle
      case REL: selB = 0x7654; selI = 0xDDD5; mem = false; break;
      case IMP: mem = false; break;
      case IZX: selB = 0x3331; selI = 0x7771; em = 0xFF; slow = true; break;  // the pointer's address
      case IZY: selB = 0x3331; em = 0xFF; slow = true; break;
      default: slow = true; break;
    }
    const uint32_t NZ = FL_NZ, NZC = FL_NZ | FL_C, C1 = 0x5551, A_ = 0x5550, X_ = 0x5551, Y_ = 0x5552, V_ = 0x5554, FF = 0x5553;
    const uint32_t dA = 0x3214, dX = 0x3240, dY = 0x3410;
    bool ld = false, st = false, rmw = false;
    switch (op) {
      case O_LDA: selD = dA; gm = NZ; ld = mem; break;
      case O_LAX: selD = 0x3244; gm = NZ; ld = mem; break;
      case O_LDX: selD = dX; gm = NZ; ld = mem; break;
      case O_LDY: selD = dY; gm = NZ; ld = mem; break;
      case O_ADC: selX = A_; selD = dA; gm = NZC | FL_V; selC = C1; ld = mem; break;
      case O_SBC: selX = A_; selD = dA; gm = NZC | FL_V; selC = C1; inv = 0xFF; ld = mem; break;
      case O_AND: selX = A_; selD = dA; gm = NZ; k = 1; m2 = 0; ld = mem; break;
      case O_ORA: selX = A_; selD = dA; gm = NZ; k = 1; ld = mem; break;
      case O_EOR: selX = A_; selD = dA; gm = NZ; k = 0; ld = mem; break;
      case O_CMP: selX = A_; gm = NZC; inv = 0xFF; one = 1; ld = mem; break;
      case O_CPX: selX = X_; gm = NZC; inv = 0xFF; one = 1; ld = mem; break;
      case O_CPY: selX = Y_; gm = NZC; inv = 0xFF; one = 1; ld = mem; break;
      case O_STA: selX = A_; st = true; break;
      case O_STX: selX = X_; st = true; break;
      case O_STY: selX = Y_; st = true; break;
      case O_ASL: selX = V_; gm = NZC; rmw = mem; break;
      case O_ROL: selX = V_; gm = NZC; selC = C1; rmw = mem; break;
      // y * 513 >> 1 holds y >> 1 in bits 0-6 and y's bit 0 in bit 8; the carry comes in at 256 >> 1
      case O_LSR: selX = V_; gm = NZC; k = 513; rmw = mem; break;
      case O_ROR: selX = V_; gm = NZC; k = 513; selC = 0x5515; rmw = mem; break;
      case O_INC: gm = NZ; one = 1; rmw = true; break;
      case O_DEC: selX = FF; gm = NZ; rmw = true; break;
      case O_INX: selX = X_; selD = dX; gm = NZ; one = 1; break;
      case O_INY: selX = Y_; selD = dY; gm = NZ; one = 1; break;
      case O_DEX: selX = X_; selD = dX; gm = NZ; inv = 0xFF; break;
      case O_DEY: selX = Y_; selD = dY; gm = NZ; inv = 0xFF; break;
      case O_TAX: selX = A_; selD = dX; gm = NZ; break;
      case O_TAY: selX = A_; selD = dY; gm = NZ; break;
      case O_TXA: selX = X_; selD = dA; gm = NZ; break;
      case O_TYA: selX = Y_; selD = dA; gm = NZ; break;
      case O_CLC: gm = FL_C; break;
      case O_SEC: gm = FL_C; inv = 0xFF; one = 1; break;  // 0 + FF + 1 carries
      case O_CLV: gm = FL_V; break;
      // taken when a flag bit is set: 0 + bits > 0; when none is: bits - 1 > FFFF0000
      case O_BCS: bm = FL_C; break;
      case O_BCC: bm = FL_C; a = ~0u; break;
      case O_BNE: bm = FL_Z; break;
      case O_BEQ: bm = FL_Z; a = ~0u; break;
      case O_BMI: bm = FL_N; break;
      case O_BPL: bm = FL_N; a = ~0u; break;
      case O_BVS: bm = FL_V; break;
      case O_BVC: bm = FL_V; a = ~0u; break;
      // a branch always taken: base = the operand over the cycle, the taken branch's cycle counted
      case O_JMP: if (mode == ABS) { a = ~0u; cyc = 2; selB = 0x7621; } else slow = true; break;
      case O_NOP: if (mode != IMP && mode != IMM) slow = true; break;  // its operand read may switch a bank
      default: slow = true; break;  // stack operations, BIT, other flag operations, undocumented opcodes
    }
    const bool sum = op == O_ADC || op == O_SBC;
    if (op == O_JMP) em = 0;
    if (mode == ACC) selD = dA;
    if (slow) {  // nothing happens here: the lane waits
      selD = 0x3210; gm = bm = a = regions = 0; ld = st = rmw = false;
    } else if (ld) {
      regions = sum ? RG_MSUM : RG_RAM | RG_CART; selV = 0x3210;
    } else if (st) {
      regions = RG_RAM | RG_WRAM | RG_OUT | RG_WSYNC; selV = 0x1111;  // operand 0: the result is x
    } else if (rmw) {
      regions = RG_RAM | RG_WRAM; selV = 0x3210;
    } else {
      em = 0;  // no access: address 0
      if (sum) regions = RG_ISUM;
    }
    if (one) selC = 0x5554;
    if (k == 513) a = 1;                               // the shift; no branch: 1 + 0 is below any selector
    const uint32_t thr = bm || a == ~0u ? a & 0xFFFF0000u : selC;
    const uint32_t w[CTL_WORDS] = {selB, selI, selX, selD, selV, em, len | cyc << 16, bm,
                                   gm, inv, k, thr, regions, m2, pen << 8, a};
    for (uint32_t i = 0; i < 4; ++i) memcpy(out + DEC_CTL + CTL_TABLE * i + 16 * e, w + 4 * i, 16);
  }
}

}  // namespace atari
