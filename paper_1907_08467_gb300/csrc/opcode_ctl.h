// Control words of the batched interpreter: one set per opcode, built on the
// host from the decode table and copied to shared memory by every block.
//
// The interpreter runs every common instruction through one branch-free
// sequence (fast_console.cuh); these words tell it which operand bytes, index,
// registers, adder inputs and flags the opcode uses.  On sm_103a a switch on
// the opcode costs about 30 cycles for each level of its compare tree (one
// warp, warp-uniform value: 49 cycles for 2 cases, 178 for 36, 241 for 150),
// and a jump table 100 cycles while its handlers fit the instruction cache's
// first level and 280-450 when they do not, so data beats code here.
#pragma once
#include <cstdint>
#include <cstring>

#include "device_machine.cuh"

namespace atari {

// words 0..3 (one 16-byte load per round):
//   0  byte selector of the address base from (instruction bytes, next PC)
//      | address mask << 16
//   1  byte selector of the index from (A X Y 0, instruction bytes)
//      | branch flag mask << 16 | branch flag invert << 24
//   2  byte selector of the adder's x from (A X Y 0, operand FF) | xor mask << 16 | operand invert << 24
//   3  byte selector of the written registers from (A X Y 0, result)
//      | flag write mask << 16 | length << 28
// word 4: the bits below, cycles << 8, page-cross penalty << 15, flags taken
//   from the operand (BIT) << 16, carries of (x & y) << 24, decimal check << 27
constexpr uint32_t CT_CIN = 1u, CT_ONE = 2u, CT_MEM = 4u, CT_LD = 8u, CT_ST = 16u, CT_RMW = 32u, CT_SHR = 64u,
                   CT_SLOW = 128u, CT_COUNT = 1u << 28;
constexpr uint32_t CTL_HALT = 256;             // entry that changes nothing: a lane waiting for service
constexpr uint32_t CTL_N = 257;
constexpr uint32_t CTL_B_OFF = 16 * CTL_N;     // word 4 of every entry follows the 16-byte entries
constexpr uint32_t CTL_BYTES = (CTL_B_OFF + 4 * CTL_N + 15) / 16 * 16;
constexpr uint32_t DEC_BYTES = 512 + CTL_BYTES;  // general decoder's bytes, then the control words

// dec: per opcode, operation | mode << 8 | cycles << 12 | page-cross penalty << 16 (0: halts the CPU).
inline void build_ctl(const uint32_t *dec, uint8_t *out) {
  memset(out, 0, CTL_BYTES);
  for (uint32_t o = 0; o < CTL_N; ++o) {
    const uint32_t op = o < 256 ? dec[o] & 0xFF : (uint32_t)O_NOP, mode = o < 256 ? (dec[o] >> 8) & 0xF : (uint32_t)IMP;
    uint32_t cyc = o < 256 ? (dec[o] >> 12) & 0xF : 0u;
    const uint32_t pen = o < 256 ? (dec[o] >> 16) & 1 : 0u;
    uint32_t len = o == CTL_HALT ? 0u : mode <= ACC ? 1u : mode >= ABS && mode <= IND ? 3u : 2u;
    uint32_t selB = 0x6666, selI = 0x3333, selX = 0x3333, selD = 0x3210, em = 0x1FFF;
    uint32_t bm = 0, binv = 0, m2 = 0xFF, inv = 0, pm = 0, cb = o == CTL_HALT ? 0u : CT_COUNT, k = 2;
    bool mem = true, slow = op == O_JAM;
    switch (mode) {
      case IMM: selB = 0x6661; mem = false; break;
      case ZP: selB = 0x6661; em = 0xFF; break;
      case ZPX: selB = 0x6661; selI = 0x3331; em = 0xFF; break;
      case ZPY: selB = 0x6661; selI = 0x3332; em = 0xFF; break;
      case ABS: selB = 0x6621; break;
      case ABX: selB = 0x6621; selI = 0x3331; break;
      case ABY: selB = 0x6621; selI = 0x3332; break;
      case ACC: selI = 0x3330; mem = false; break;  // the operand is the sum of base and index: A
      case REL: selB = 0x6654; selI = 0xDDD5; mem = false; break;
      case IMP: mem = false; break;
      default: slow = true; break;                  // pointers through RAM: the general decoder
    }
    const uint32_t NZ = 0x82, NZC = 0x83, A_ = 0x3330, X_ = 0x3331, Y_ = 0x3332, V_ = 0x3334, FF = 0x3335;
    const uint32_t dA = 0x3214, dX = 0x3240, dY = 0x3410;
    bool ld = false, st = false, rmw = false;
    switch (op) {
      case O_LDA: selD = dA; pm = NZ; ld = mem; break;
      case O_LDX: selD = dX; pm = NZ; ld = mem; break;
      case O_LDY: selD = dY; pm = NZ; ld = mem; break;
      case O_ADC: selX = A_; selD = dA; pm = 0xC3; cb |= CT_CIN | 1u << 27; ld = mem; break;
      case O_SBC: selX = A_; selD = dA; pm = 0xC3; inv = 0xFF; cb |= CT_CIN | 1u << 27; ld = mem; break;
      case O_AND: selX = A_; selD = dA; pm = NZ; k = 1; m2 = 0; ld = mem; break;
      case O_ORA: selX = A_; selD = dA; pm = NZ; k = 1; ld = mem; break;
      case O_EOR: selX = A_; selD = dA; pm = NZ; k = 0; ld = mem; break;
      case O_BIT: selX = A_; pm = 0xC2; k = 1; m2 = 0; cb |= 0xC0u << 16; ld = mem; break;
      case O_CMP: selX = A_; pm = NZC; inv = 0xFF; cb |= CT_ONE; ld = mem; break;
      case O_CPX: selX = X_; pm = NZC; inv = 0xFF; cb |= CT_ONE; ld = mem; break;
      case O_CPY: selX = Y_; pm = NZC; inv = 0xFF; cb |= CT_ONE; ld = mem; break;
      case O_STA: selX = A_; st = true; break;
      case O_STX: selX = X_; st = true; break;
      case O_STY: selX = Y_; st = true; break;
      case O_ASL: selX = V_; pm = NZC; rmw = mem; break;
      case O_ROL: selX = V_; pm = NZC; cb |= CT_CIN; rmw = mem; break;
      case O_LSR: pm = NZC; cb |= CT_SHR; rmw = mem; break;
      case O_ROR: pm = NZC; cb |= CT_SHR | CT_CIN; rmw = mem; break;
      case O_INC: pm = NZ; cb |= CT_ONE; rmw = true; break;
      case O_DEC: selX = FF; pm = NZ; rmw = true; break;
      case O_INX: selX = X_; selD = dX; pm = NZ; cb |= CT_ONE; break;
      case O_INY: selX = Y_; selD = dY; pm = NZ; cb |= CT_ONE; break;
      case O_DEX: selX = X_; selD = dX; pm = NZ; inv = 0xFF; break;
      case O_DEY: selX = Y_; selD = dY; pm = NZ; inv = 0xFF; break;
      case O_TAX: selX = A_; selD = dX; pm = NZ; break;
      case O_TAY: selX = A_; selD = dY; pm = NZ; break;
      case O_TXA: selX = X_; selD = dA; pm = NZ; break;
      case O_TYA: selX = Y_; selD = dA; pm = NZ; break;
      case O_CLC: pm = 0x01; break;
      case O_SEC: pm = 0x01; inv = 0xFF; cb |= CT_ONE; break;  // 0 + FF + 1 carries
      case O_CLI: pm = 0x04; break;
      case O_CLV: pm = 0x40; break;
      case O_CLD: pm = 0x08; break;
      case O_BCC: bm = binv = 0x01; break;
      case O_BCS: bm = 0x01; break;
      case O_BNE: bm = binv = 0x02; break;
      case O_BEQ: bm = 0x02; break;
      case O_BVC: bm = binv = 0x40; break;
      case O_BVS: bm = 0x40; break;
      case O_BPL: bm = binv = 0x80; break;
      case O_BMI: bm = 0x80; break;
      // a branch always taken (P bit 5 is always set): base = the operand, the taken branch's cycle counted
      case O_JMP: if (mode == ABS) { bm = 0x20; cyc = 2; } else slow = true; break;
      case O_NOP: if (mode != IMP && mode != IMM) slow = true; break;  // its operand read may switch a bank
      default: slow = true; break;  // stack operations, SEI, SED, undocumented opcodes
    }
    if (op == O_JMP) mem = false;
    if (mode == ACC) selD = dA;
    if (slow && o != CTL_HALT) {  // nothing happens here: the lane waits for the general decoder
      selD = 0x3210; pm = bm = binv = 0; ld = st = rmw = false;
      cb |= CT_SLOW;
    }
    cb |= (ld ? CT_MEM | CT_LD : 0u) | (st ? CT_ST : 0u) | (rmw ? CT_MEM | CT_RMW : 0u) | cyc << 8 | pen << 15 | k << 24;
    const uint32_t w[4] = {selB | em << 16, selI | bm << 16 | binv << 24, selX | m2 << 16 | inv << 24,
                           selD | pm << 16 | len << 28};
    memcpy(out + 16 * o, w, 16);
    memcpy(out + CTL_B_OFF + 4 * o, &cb, 4);
  }
}

}  // namespace atari
