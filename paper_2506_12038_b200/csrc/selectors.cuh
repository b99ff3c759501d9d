// Lookup selectors: packed weight indices -> PRMT selector words, written so that the integer pipe, which the lookups
// themselves need, does as little of it as possible.
//
// PRMT, shifts and logic operations share one pipe that issues a warp's instruction every 2 clocks (measured on B200);
// integer multiply-adds (2 clocks) and half-precision multiplies (1 clock) run on others at the same time.  A PRMT reads
// its four selector nibbles from the lower half of a register, so every selector word is used twice, as it is and moved
// down by 16 bits.  That move is done by the half-precision pipe here: a multiplication of the upper half by 1.0, exact
// for every pattern below 0x7c00 (infinities and NaNs; the selectors' nibbles are at most 7), subnormals included.
// Differences x - (x & mask) in place of x & ~mask are multiply-adds.  Integer-pipe instructions per 16 weights and two
// byte planes (lookups included): 2 bit 10 (13 with shifts and masks), 3 bit 11 (14.5), 4 bit 28 (34).
#ifndef LCD_SELECTORS_CUH_
#define LCD_SELECTORS_CUH_

#include <cstdint>

namespace lcd {

// x >> 16 in the lower half of the result (the upper half repeats it); halves below 0x7c00.
__device__ __forceinline__ uint32_t upper_half(uint32_t x) {
  uint32_t d;
  asm("{\n.reg .b16 l, h;\n.reg .b32 t;\nmov.b32 {l, h}, %1;\nmov.b32 t, {h, h};\nmul.rn.f16x2 %0, t, %2;\n}"
      : "=r"(d) : "r"(x), "r"(0x3c003c00u));
  return d;
}
// a + b and a - b on the multiply-add pipe
__device__ __forceinline__ uint32_t mad_add(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, 1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t mad_sub(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, 0xffffffff, %2;" : "=r"(d) : "r"(b), "r"(a));
  return d;
}

// 2 bit: 16 indices of a word; sel[0], sel[1]: the even ones, first and second eight columns; sel[2], sel[3]: the odd ones
__device__ __forceinline__ void selectors_2bit(uint32_t raw, uint32_t* sel) {
  const uint32_t even = raw & 0x33333333u, odd = mad_sub(raw, even) >> 2;
  sel[0] = even;
  sel[1] = upper_half(even);
  sel[2] = odd;
  sel[3] = upper_half(odd);
}
// 3 bit: 32 indices of a record's three words, eight selector words in column order (the last eight columns' bits are
// bit 3 of the nibbles of the three words)
__device__ __forceinline__ void selectors_3bit(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t* sel) {
  const uint32_t d0 = r0 & 0x77777777u, d1 = r1 & 0x77777777u, d2 = r2 & 0x77777777u;
  const uint32_t e0 = mad_sub(r0, d0), e1 = mad_sub(r1, d1), e2 = mad_sub(r2, d2);
  const uint32_t ex = mad_add(mad_add(e0 >> 1, e1) >> 1, e2) >> 1;
  sel[0] = d0; sel[1] = upper_half(d0);
  sel[2] = d1; sel[3] = upper_half(d1);
  sel[4] = d2; sel[5] = upper_half(d2);
  sel[6] = ex; sel[7] = upper_half(ex);
}
// 4 bit: eight indices of a word in column order; pick[i]: the byte choice 0x3210 + 4 * (bit 3 of each index) between the
// looked-up entries 0..7 and 8..15
__device__ __forceinline__ void selectors_4bit(uint32_t raw, uint32_t* sel, uint32_t* pick) {
  const uint32_t low = raw & 0x77777777u, choice = mad_add(mad_sub(raw, low) >> 1, 0x32103210u);
  sel[0] = low; sel[1] = upper_half(low);
  pick[0] = choice; pick[1] = upper_half(choice);
}

}  // namespace lcd
#endif
