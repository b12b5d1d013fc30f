// Block fixed point on the integer multiply-add pipe: a real number is two
// limbs h 2^29 + l with |l| <= 2^28 under an exponent shared by a group (a
// site, a row, a column of coefficients).  A product of two such numbers is
// h h 2^58 + (h l + l h) 2^29 (+ l l, below the last bit kept): three 32 x 32 ->
// 64 bit multiply-adds, at 64 per SM and clock against 2 FP64 FMA on GB300.
#pragma once

#include "common.cuh"

namespace dsbcg {

constexpr int FX_ZERO = -(1 << 20), FX_NAN = 1 << 20;
constexpr int FX_BASE = 29;                    // bits per limb
constexpr int FX_BITS = 57;                    // magnitude bits of a field value

__device__ __forceinline__ int2 fx_split(long long x) {
    const int h = (int)((x + (1ll << (FX_BASE - 1))) >> FX_BASE);
    return make_int2(h, (int)((unsigned)x - ((unsigned)h << FX_BASE)));
}
__device__ __forceinline__ long long fx_join(int h, int l) { return (long long)h * (1 << FX_BASE) + l; }
// x 2^-s rounded to nearest, s >= 0
__device__ __forceinline__ long long fx_shift(long long x, int s) {
    if (s > 62) return 0;
    return s > 0 ? (x + (1ll << (s - 1))) >> s : x;
}
// FP64 v in units of 2^(eb - 1079), eb >= v's biased exponent
__device__ __forceinline__ long long fx_of_double(double v, int eb) {
    const int hi = __double2hiint(v);
    const int e = (hi >> 20) & 0x7ff;
    const long long mant =
        ((long long)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32) | (unsigned)__double2loint(v);
    const long long x = fx_shift(mant << 4, eb - (e ? e : 1));
    return hi < 0 ? -x : x;
}
// v 2^e in FP64 (round to nearest; the slow path only outside the normal range)
__device__ __forceinline__ double fx_to_double(long long v, int e) {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d), x = ((hi >> 20) & 0x7ff) + e;
    if (v == 0) return 0.0;
    if (x > 0 && x < 2047) return __hiloint2double(hi + e * (1 << 20), __double2loint(d));
    return ldexp(d, e);
}
// x 2^s, rounded down for s < 0
__device__ __forceinline__ long long fx_align(long long x, int s) {
    return s >= 0 ? (s > 62 ? 0 : x << s) : x >> (s < -63 ? 63 : -s);
}
// high and middle limb sums of a complex product t u (limbs re.h, re.l, im.h, im.l)
__device__ __forceinline__ void fx_mac(int4 t, int4 u, long long& hr, long long& mr, long long& hi, long long& mi) {
    const int nz = -t.z, nw = -t.w;
    hr += (long long)t.x * u.x;
    hi += (long long)t.x * u.z;
    mr += (long long)t.x * u.y;
    mi += (long long)t.x * u.w;
    hr += (long long)nz * u.z;
    hi += (long long)t.z * u.x;
    mr += (long long)t.y * u.x;
    mi += (long long)t.y * u.z;
    mr += (long long)nz * u.w;
    mi += (long long)t.z * u.y;
    mr += (long long)nw * u.z;
    mi += (long long)t.w * u.x;
}

}  // namespace dsbcg
