// Fixed-point helpers of the FP64 paths: FP64 numbers as 64-bit integers, and load currents without the FP64 pipe.
#pragma once

#include <cstdint>

namespace tpf {

constexpr int kFx = 61;              // V, branch terms and path sums: 2^-kFx pu
__device__ __forceinline__ int order(double v) { return ((__double2hiint(v) >> 20) & 0x7ff) - 1023; }
// round(v * 2^s) by shifts of the significand; the caller keeps |v| * 2^s below 2^62.
__device__ __forceinline__ long long to_fx(double v, int s) {
    const int hi = __double2hiint(v), E = (hi >> 20) & 0x7ff, sh = E - 1075 + s;
    const unsigned long long m =
        ((unsigned long long)((hi & 0xfffff) | (E ? 0x100000 : 0)) << 32) | (unsigned)__double2loint(v);
    unsigned long long x;
    if (sh >= 0)
        x = m << (sh & 63);
    else
        x = sh > -55 ? ((m >> (-sh - 1)) + 1) >> 1 : 0ull;
    return hi < 0 ? -(long long)x : (long long)x;
}

// |v|^2 in FP32 of v in 2^-61 pu, from the high words.
__device__ __forceinline__ float abs2_fx(longlong2 v) {
    constexpr float k29 = 1.0f / 536870912.0f;
    const float x = (float)(int)(v.x >> 32) * k29, y = (float)(int)(v.y >> 32) * k29;
    return fmaf(x, x, y * y);
}
// Below half a pu the integers' last places, 2^-61 pu here and 2^-53 in current_fx, are no longer far enough
// below v: such a voltage's current is an FP64 division of an FP64 voltage.  (The quotients of current_fx lose
// bits in proportion to 1 / |v|, and wrap below 1e-4 pu; converged voltages of a feeder are above 0.5 pu.)
constexpr float kLowV2 = 0.25f;

// Demand current conj(s / v) of a constant-power bus in units of 2^cur, without the FP64 pipe: a quotient of
// 25 bits in FP32, its remainder exactly in integers, and twice the same again for the remainder.
//
// With w the quotient so far, conj(s) - w conj(v) is taken modulo 2^64: v in 2^-53 pu (54 bits) times an
// integer quotient of 26 bits would need 80, but the remainder is at most 2^5 quotient units times |v| and
// fits (|v| at least half a pu: the FP32 quotient's own error is 2^-29 / |v|, five bits of it in quotient units).
// Quotient units: 2^u = 2^(cur_e - 25), so that a current in range is below 2^25 of them; then 2^(u - 22);
// the last quotient is rounded to the sum's last place 2^cur, 37 - log2n bits below 2^u.
//   v: 2^-61 pu; s_mod: s in units of 2^(u - 53), modulo 2^64; s_f: s in units of 2^u.
// Returns false for a current out of range (or not a number) and for |v| below half a pu.
__device__ __forceinline__ bool current_fx(longlong2 v, longlong2 s_mod, float2 s_f, int log2n, longlong2 &out) {
    constexpr float k29 = 1.0f / 536870912.0f, k21 = 1.0f / 2097152.0f, k22 = 4194304.0f;
    const float vx = (float)(int)(v.x >> 32) * k29, vy = (float)(int)(v.y >> 32) * k29;
    const long long wx = (v.x + 128) >> 8, wy = (v.y + 128) >> 8;  // 2^-53 pu
    const float v2 = fmaf(vx, vx, vy * vy), inv = __fdividef(1.0f, v2);
    const float ix = fmaf(s_f.x, vx, s_f.y * vy) * inv, iy = fmaf(s_f.x, vy, -s_f.y * vx) * inv;
    const bool ok = fabsf(ix) < 33554432.0f && fabsf(iy) < 33554432.0f && v2 >= kLowV2;
    const int qx = __float2int_rn(ix), qy = __float2int_rn(iy);
    using u64 = unsigned long long;  // modulo 2^64
    auto mul = [](int q, long long w) { return (u64)(long long)q * (u64)w; };
    // r = conj(s) - q conj(v), units of 2^(u - 53)
    const u64 rx = (u64)s_mod.x - mul(qx, wx) - mul(qy, wy), ry = mul(qx, wy) - mul(qy, wx) - (u64)s_mod.y;
    float fx = (float)(int)(rx >> 32) * k21 * inv, fy = (float)(int)(ry >> 32) * k21 * inv;
    const int px = __float2int_rn(fmaf(fx, vx, -fy * vy) * k22), py = __float2int_rn(fmaf(fx, vy, fy * vx) * k22);
    // the remainder of that, units of 2^(u - 75)
    const u64 tx = (rx << 22) - mul(px, wx) - mul(py, wy), ty = (ry << 22) + mul(px, wy) - mul(py, wx);
    fx = (float)(int)(tx >> 32) * k21 * inv, fy = (float)(int)(ty >> 32) * k21 * inv;
    const int a = 37 - log2n, b = a - 22;
    const float last = (float)(1 << b);
    const int lx = __float2int_rn(fmaf(fx, vx, -fy * vy) * last), ly = __float2int_rn(fmaf(fx, vy, fy * vx) * last);
    out.x = (long long)(((u64)(long long)qx << a) + ((u64)(long long)px << b) + (u64)(long long)lx);
    out.y = (long long)(((u64)(long long)qy << a) + ((u64)(long long)py << b) + (u64)(long long)ly);
    return ok;
}

}  // namespace tpf
