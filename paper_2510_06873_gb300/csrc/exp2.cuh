// exp2_neg(y) = 2^-y in FP64 by integer arithmetic, for the Gaussian hills.
//
// A hill costs one exponential, and FP64 instructions are the scarce resource
// of this part (two lanes per clock and SM, 64 cycles each): the library's
// exp takes about 20 of them, this function none.  Table-driven reduction
// (P. T. P. Tang, "Table-driven implementation of the exponential function in
// IEEE floating-point arithmetic", ACM TOMS 15, 1989) in 64-bit fixed point:
//   y = n + i/64 + a/64,  n an integer, i = 0 .. 63, 0 <= a < 1,
//   2^-y = 2^-n 2^(-i/64) (1 - z + z^2/2 - ... - z^7/5040),  z = a ln2 / 64.
// y is split without rounding (bits below 2^-64 dropped), the series is
// summed to 2^-62 (terms from z^4 on in 32 bits: they start below 2^-30), and
// the product is rounded once to 53 bits: at most 0.502 units in the last
// place from the exact value, without bias (the library's bound is 1).
// Measured: the torsion walkers' step (256 x 10,000 hills), see hills.cuh.
//
// y >= 0.  From 1000 on (a factor below 1e-301, down to denormals and 0), and
// for infinities and NaN, the library function is called.
#pragma once

#include <stdint.h>

namespace metad {

// 2^(63 - i/64), rounded to integers.
static __device__ const unsigned long long kExp2Neg[64] = {
    0x8000000000000000ull, 0x7e9f06067a4360baull, 0x7d41d96db915019dull, 0x7be86fb985689ddcull,
    0x7a92be8a92436616ull, 0x7940bb9e2cffd89dull, 0x77f25ccdee6d7ae6ull, 0x76a7980f6cca15c2ull,
    0x75606373ee921c97ull, 0x741cb5281e25ee34ull, 0x72dc8373be41a454ull, 0x719fc4b95f452d29ull,
    0x70666f76154a7089ull, 0x6f307a412f074892ull, 0x6dfddbcbed791babull, 0x6cce8ae13c57ebdbull,
    0x6ba27e656b4eb57aull, 0x6a79ad55e7f6fd10ull, 0x69540ec8f895722dull, 0x683199ed779592caull,
    0x6712460a8fc24072ull, 0x65f60a7f79393e2eull, 0x64dcdec3371793d1ull, 0x63c6ba6455dcd8aeull,
    0x62b39508aa836d6full, 0x61a3666d124bb204ull, 0x6096266533384a2bull, 0x5f8bccdb3d398841ull,
    0x5e8451cfac061b5full, 0x5d7fad59099f22feull, 0x5c7dd7a3b17dcf75ull, 0x5b7ec8f19468bbc9ull,
    0x5a827999fcef3242ull, 0x5988e20954889245ull, 0x5891fac0e95612c8ull, 0x579dbc56b48521baull,
    0x56ac1f752150a563ull, 0x55bd1cdad49f699cull, 0x54d0ad5a753e077cull, 0x53e6c9da74b29ab5ull,
    0x52ff6b54d8a89c75ull, 0x521a8ad704f3404full, 0x513821818624b40cull, 0x50582887dcb8a7e1ull,
    0x4f7a993048d088d7ull, 0x4e9f6cd3967fdba8ull, 0x4dc69cdceaa72a9cull, 0x4cf022c9905bfd32ull,
    0x4c1bf828c6dc54b8ull, 0x4b4a169b900c2d00ull, 0x4a7a77d47f7b84b1ull, 0x49ad159789f37496ull,
    0x48e1e9b9d588e19bull, 0x4818ee218a3358eeull, 0x47521cc5a2e6a9e0ull, 0x468d6fadbf2dd4f3ull,
    0x45cae0f1f545eb73ull, 0x450a6abaa4b77ecdull, 0x444c0740496d4294ull, 0x438fb0cb4f468808ull,
    0x42d561b3e6243d8aull, 0x421d1461d66f2023ull, 0x4166c34c5615d0ecull, 0x40b268f9de0183baull};

static __device__ __forceinline__ double exp2_neg(double y)
{
    const unsigned hi = (unsigned)__double2hiint(y);
    if (hi >= 0x408f4000u) return exp2(-y);  // y >= 1000, infinity, NaN
    const int ex = (int)(hi >> 20) - 1023;
    const unsigned long long m = ((unsigned long long)__double_as_longlong(y) & 0xfffffffffffffull) | (1ull << 52);
    // n, and the fraction of y in units of 2^-64 (y = 0 leaves one unit)
    const int n = ex >= 0 ? (int)(m >> (52 - ex)) : 0;
    const unsigned long long fr = ex >= 0 ? m << (12 + ex) : (m << 11) >> min(-ex - 1, 63);
    const unsigned long long t = __ldg(kExp2Neg + (int)(fr >> 58));
    const unsigned long long a = fr << 6;
    const unsigned a32 = (unsigned)(a >> 32);
    // (ln2 / 64)^k / k!: k = 7 .. 4 in units of 2^-62, 3 .. 1 of 2^-70
    unsigned q = 0x2861u - __umulhi(a32, 0x10u);
    q = 0x576200u - __umulhi(a32, q);
    q = 0x9d955b7eu - __umulhi(a32, q);
    unsigned long long Q = 0xe35846b82506ull - (((unsigned long long)a32 * q) >> 24);
    Q = 0xf5fdeffc162c75ull - __umul64hi(a, Q);
    Q = 0xb17217f7d1cf79acull - __umul64hi(a, Q);
    // 1 - z + ... in units of 2^-63, times the table: in units of 2^-62
    const unsigned long long M = __umul64hi((1ull << 63) - (__umul64hi(a, Q) >> 7), t);
    const int one = (int)(M >> 62);  // 1 only for an integer y
    const unsigned long long mant = (M + (256ull << one)) >> (9 + one);  // bit 52 set (53 after a carry)
    return __longlong_as_double((long long)(((unsigned long long)(1021 + one - n) << 52) + mant));
}

}  // namespace metad
