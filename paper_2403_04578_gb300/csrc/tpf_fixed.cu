// FP64 dense sweeps on the tensor cores: V_{k+1} = K conj(S ./ V_k) + W (Eq. 2, Eq. 12) with the
// product evaluated in 55-bit fixed point from exact fp16 digit products.
//
// GB300 runs FP64 at 1/64 of its FP32 rate (1.2 TFLOP/s) and fp16 on the tensor cores at 1.9
// PFLOP/s, so the 8 n^2 FP64 operations of a column and sweep are replaced by integer arithmetic
// (the splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with digits of equal
// place instead of floating slices).  Bus j's column of K is divided by a power of two c_j, its largest
// component's order, and its current multiplied by it: J_j = c_j I_j is the largest voltage drop that the bus
// causes by itself, whatever the decades between impedances (an open switch modelled as one of 1e6 pu) or
// between loads.  Every component of K / c and of J (scaled per column of the tensor by that column's largest)
// becomes an integer of at most 2^55, so that the largest one keeps its whole FP64 significand, written as
// seven balanced base-256 digits d_0 .. d_6 in [-128, 128], each exact in fp16.  Then
//
//     K I = (K / c) J = sum over diagonals d of 256^-d  sum_{i + j = d} (K / c)_i J_j
//
// with the diagonals 0 .. 6 kept (28 digit products).  In units of the column's largest J, what is dropped
// is 2^-51 (root mean square, digits of no pattern) at 1,000 buses, 2^-42.4 at the very worst (12 n products
// of 2^14 two places below diagonal 6, all of one sign); J is below 2^-8 pu on the feeders of inputs.py.  With
// one scale for all of K and one for all currents, as this once was, an unloaded stub of 1e6 pu cost the other
// buses of a 200-bus feeder 1.3e-10 pu, and one load of 1,000 pu near the source 6.2e-14.
// A digit product's sum over 512 terms stays below 2^24, so the FP32 accumulators in TMEM hold it
// exactly whatever the order; the accumulated integers are then added in 64-bit integer arithmetic,
// down to a last place that the sum of all n terms cannot overflow (2^-53 of the largest J at 256 buses).  A column's result therefore does not depend on the tile it falls in.
//
// Measured against binary128 on one sweep from random starts, the largest error is 5.5e-17 to 7e-17 pu at
// 1 to 399 buses (half a last place of V: the only rounding left is that of the result), where the FP64
// sums have 5.5e-17 to 1.9e-16.
//
// Per sweep, over the columns that still iterate (a compacted list):
//   fx_slice   one block per column: I in FP64, its scale, the digit planes;
//   fx_gemm    persistent, warp-specialised: 128 buses x 64 columns per tile, both accumulators
//              (Re, Im) of two neighbouring diagonals per TMEM stage, the V update and the
//              column's largest step in the epilogue of the tile;
//   fx_column  the columns whose currents are not finite (or beyond 2^1000) in plain FP64;
//   fx_decide  the per-column stopping rule and the next list.
#include <cuda_fp16.h>
#include <math_constants.h>

#include <algorithm>
#include <cstring>

#include "tpf_fx.cuh"
#include "tpf_gemm.h"
#include "tpf_tc.cuh"

namespace tpf {

#define TPF_CK(call)                  \
    do {                              \
        if ((call) != cudaSuccess) {  \
            cudaGetLastError();       \
            return TPF_ECUDA;         \
        }                             \
    } while (0)

namespace {

using namespace tc;

constexpr int kDig = 7;       // base-256 digits of a 55-bit integer
constexpr int kBits = 55;
constexpr int kFxN = 64;      // columns per tile: 64 x 128 x 2 64-bit sums are what the registers hold
constexpr int kFxStages = 4;
constexpr uint32_t kABytes = kTileM * kChunkK * 2;                // 16 KB, one plane of K
constexpr uint32_t kBBytes = kFxN * kChunkK * 2;                  // 8 KB, one plane of I
constexpr uint32_t kFxStageBytes = 2 * kABytes + 3 * kBBytes;     // (Ar, Ai, Br, Bi, -Br)
constexpr size_t kFxBars = 128, kFxSmem = 1024 + kFxStages * kFxStageBytes + kFxBars + 16 * kFxN;
constexpr int kFxEpiWarps = 8;
constexpr int kFxEpiThreads = 32 * kFxEpiWarps;
constexpr int kFxThreads = 64 + kFxEpiThreads;
constexpr uint32_t kFxAcc = 4 * kFxN;  // TMEM columns of a stage: Re, Im of the upper and the lower diagonal
constexpr int kMinExp = -900, kMaxExp = 1000;  // binary orders of a column's largest J
constexpr int kFxMaxN = 8192;                  // fx_slice keeps a column's currents in shared memory

// Counters of the sweeps: columns left to fx_column, and the lengths of the two column lists (a sweep reads
// one and counts the other).
enum FxCounter : int { kFxPlain = 1, kFxCount = 6 };

struct FxArgs {
    int n, n_pad, m_tiles, n_chunks, ksteps;
    const int *count;     // device: columns that iterate
    int first, cap;       // this launch takes those from `first`, at most cap (the rows of a digit plane of I)
    const int *list;      // the columns, or null: 0, 1, ...
    double f1;            // 2^(drop - 62 + order of K / c): value of a last place for a column of order 0
    int drop;             // last place of the 64-bit sums, in bits above diagonal 6's
    const int *colexp;    // per column of this launch: binary order of the largest J; kMaxExp: skip
    const double2 *W;
    double2 *V;
    unsigned long long *delta;
    int *err;
};

__device__ __forceinline__ int64_t fx_col(const int *list, int c) { return list ? list[c] : c; }

__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// The seven balanced digits of x (|x| <= 2^55), most significant first.
__device__ __forceinline__ void digits(long long x, __half (&d)[kDig]) {
#pragma unroll
    for (int i = kDig - 1; i > 0; --i) {
        const int lo = (int)(signed char)(x & 0xff);
        d[i] = __int2half_rn(lo);
        x = (x - lo) >> 8;
    }
    d[0] = __int2half_rn((int)x);
}

// round(v * 2^(kBits - e)) for |v| < 2^e, from the bits of v (a scaling and a conversion would take two
// operations of the FP64 pipe, at a thirty-second of the integer rate).
__device__ __forceinline__ long long to_fixed(double v, int e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int E = (int)(b >> 52) & 0x7ff, k = e + 1022 - E;  // |v| = m 2^(E - 1075), so k >= 0
    const unsigned long long m = ((b & 0xfffffffffffffull) | (E ? 1ull << 52 : 0ull)) << 2;
    const unsigned long long x = k == 0 ? m : (k < 58 ? ((m >> (k - 1)) + 1) >> 1 : 0ull);
    return (long long)b < 0 ? -(long long)x : (long long)x;
}

// Digit planes [kDig][n_pad][n_pad] of K * 2^(shift - order of the column), zero padded.
__global__ void fx_k_digits(const double2 *__restrict__ K, const int *__restrict__ col_order, int n, int n_pad,
                            int shift, __half *Kr, __half *Ki) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, plane = (int64_t)n_pad * n_pad;
    if (idx >= plane) return;
    const int i = (int)(idx / n_pad), j = (int)(idx % n_pad);
    double2 k = make_double2(0.0, 0.0);
    const double scale = j < n ? ldexp(1.0, shift - col_order[j]) : 0.0;
    if (i < n && j < n) k = K[(size_t)i * n + j];
    __half dr[kDig], di[kDig];
    digits(__double2ll_rn(k.x * scale), dr);
    digits(__double2ll_rn(k.y * scale), di);
#pragma unroll
    for (int d = 0; d < kDig; ++d) {
        Kr[d * plane + idx] = dr[d];
        Ki[d * plane + idx] = di[d];
    }
}

__global__ void fx_init(int64_t T, int64_t cols, int n, int flat, double2 *V, int *flags, int *iters,
                        unsigned long long *delta) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx < cols) {
        flags[idx] = idx < T ? kActive : 0;
        iters[idx] = 0;
        delta[idx] = 0ull;
    }
    if (flat && idx < T * (int64_t)n) V[idx] = make_double2(1.0, 0.0);
}

// conj(s / v) = conj(s) v / |v|^2, or Eq. 3's alpha_P conj(s / v) + alpha_I conj(s) + alpha_Z conj(s) v.
__device__ __forceinline__ double2 demand(double2 s, double2 v, const double *__restrict__ zip, int n, int k) {
    const double inv = 1.0 / (v.x * v.x + v.y * v.y);
    const double2 csv = make_double2(s.x * v.x + s.y * v.y, s.x * v.y - s.y * v.x);
    double2 cur = make_double2(csv.x * inv, csv.y * inv);
    if (zip) {
        const double ap = zip[k], ai = zip[n + k], az = zip[2 * n + k];
        cur = make_double2(ap * cur.x + ai * s.x + az * csv.x, ap * cur.y - ai * s.y + az * csv.y);
    }
    return cur;
}

constexpr int kSliceThreads = 128;

// v * 2^-u in FP32, truncated; zero below the normal range.  |v| < 2^(u + 24).
__device__ __forceinline__ float scaled_f(double v, int u) {
    const int hi = __double2hiint(v), E = ((hi >> 20) & 0x7ff) - 1023 - u + 127;
    const int bits = (hi & 0x80000000) | E << 23 | (hi & 0xfffff) << 3 | (int)((unsigned)__double2loint(v) >> 29);
    return E > 0 ? __int_as_float(bits) : 0.0f;
}

// Injections J of one column per block and their digit planes [kDig][cap][n_pad] (re, im, -re).  The largest
// component's order comes from the high words (an ordered integer maximum; NaN is above infinity).  c_j is a
// power of two, so J is the current of a load c_j S.
// Constant-power currents of voltages from 0.5 to 2 pu come from integer remainders (current_fx), the others, ZIP loads
// and columns out of its range from FP64 divisions, which bound the kernel: 23.7 instead of 30.2 us for 4,800
// columns of 199 buses (the bytes of S, V and the planes take 13), 27.3 with the scales c_j; integer pipe 68 % active.
__global__ void __launch_bounds__(kSliceThreads)
    fx_slice(int n, int n_pad, const int *__restrict__ list, const int *count, int first,
             const double2 *__restrict__ S,
             const double2 *__restrict__ V, const double *__restrict__ zip, const int *__restrict__ col_order,
             __half *Dr, __half *Di, __half *Dn, int cap, int *colexp, int *plain, int *counters) {
    extern __shared__ double2 cur[];
    __shared__ unsigned s_max[3][kSliceThreads / 32];
    longlong2 *const cur_i = reinterpret_cast<longlong2 *>(cur);
    const int tid = threadIdx.x, c = blockIdx.x;
    if (first + c >= *count) return;
    const int64_t t = fx_col(list, first + c);
    auto top = [](double2 v) {
        return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
    };
    auto block_max = [&](unsigned m, int k) {
        m = __reduce_max_sync(0xffffffffu, m);
        if ((tid & 31) == 0) s_max[k][tid >> 5] = m;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kSliceThreads / 32; ++w) m = max(m, s_max[k][w]);
        return m;
    };
    unsigned m = 0;
    int e = kMaxExp;  // every component is below 2^e
    bool ints = false;
    int cut = 0;
    if (!zip) {
        // Constant power, |V| from 0.5 to 2 pu, J below four times the largest c_j S: in integers of 2^(e - 58)
        // at once (current_fx with four bits of headroom), cut to the 55 bits that the largest one needs.
        // Orders of the scaled loads; zeros and denormals count as none, infinities and NaN as the largest.
        for (int i = tid; i < n; i += kSliceThreads) {
            const int o = (int)(top(S[t * n + i]) >> 20);
            const int so = o == 0 ? 0 : (o == 0x7ff ? 4095 : max(o + col_order[i], 0));
            m = max(m, (unsigned)so);
        }
        m = block_max(m, 0);
        e = min(max((int)m - 1022, -800), 1024) + 2;
        if (e < 900) {
            const int u = e - 25;
            bool over = false;
            unsigned mx = 0;
            for (int i = tid; i < n; i += kSliceThreads) {
                const double2 s = S[t * n + i], v = V[t * n + i];
                const int c = col_order[i];
                over |= order(v.x) >= 1 || order(v.y) >= 1;
                over |= !current_fx(make_longlong2(to_fx(v.x, kFx), to_fx(v.y, kFx)),
                                    make_longlong2(to_fx(s.x, 53 - u + c), to_fx(s.y, 53 - u + c)),
                                    make_float2(scaled_f(s.x, u - c), scaled_f(s.y, u - c)), 4, cur_i[i]);
                const longlong2 x = cur_i[i];
                mx = max(mx, (unsigned)(max(llabs(x.x), llabs(x.y)) >> 32));
            }
            mx = block_max(over ? ~0u : mx, 1);
            if (mx != ~0u) {
                ints = true;
                cut = 9 - __clz(mx);  // every |x| is below 2^(64 - clz) = 2^(55 + cut)
                e += cut - 3;
            }
        }
    }
    if (!ints) {
        m = 0;
        for (int i = tid; i < n; i += kSliceThreads) {
            const double2 I = demand(S[t * n + i], V[t * n + i], zip, n, i);
            const double c = pow2d(col_order[i]);
            cur[i] = make_double2(I.x * c, I.y * c);
            m = max(m, top(cur[i]));
        }
        m = block_max(m, 2);
        e = (int)(m >> 20) - 1022;
        if (e >= kMaxExp) {
            if (tid == 0) {
                colexp[c] = kMaxExp;
                plain[atomicAdd(&counters[kFxPlain], 1)] = (int)t;
            }
            return;
        }
    }
    if (!ints) e = max(e, kMinExp);
    if (tid == 0) colexp[c] = e;
    const size_t plane = (size_t)cap * n_pad, row = (size_t)c * n_pad;
    for (int p = tid; p < n_pad / 2; p += kSliceThreads) {
        auto at = [&](int i) {
            if (i >= n) return make_longlong2(0, 0);
            if (!ints) return make_longlong2(to_fixed(cur[i].x, e), to_fixed(cur[i].y, e));
            const longlong2 x = cur_i[i];
            if (cut <= 0) return make_longlong2(x.x << -cut, x.y << -cut);
            const long long half = 1ll << (cut - 1);
            return make_longlong2((x.x + half) >> cut, (x.y + half) >> cut);
        };
        const longlong2 a = at(2 * p), b = at(2 * p + 1);
        __half x[kDig], y[kDig];
        digits(a.x, x);
        digits(b.x, y);
#pragma unroll
        for (int d = 0; d < kDig; ++d) {
            const __half2 xy = __halves2half2(x[d], y[d]);
            *reinterpret_cast<__half2 *>(Dr + d * plane + row + 2 * p) = xy;
            *reinterpret_cast<__half2 *>(Dn + d * plane + row + 2 * p) = __hneg2(xy);
        }
        digits(a.y, x);
        digits(b.y, y);
#pragma unroll
        for (int d = 0; d < kDig; ++d)
            *reinterpret_cast<__half2 *>(Di + d * plane + row + 2 * p) = __halves2half2(x[d], y[d]);
    }
}

// The columns whose currents have no fixed-point form: one block per column, FP64 throughout.
__global__ void __launch_bounds__(kSliceThreads)
    fx_column(const double2 *__restrict__ K, const double2 *__restrict__ W, const double2 *__restrict__ S, double2 *V,
              int n, const int *__restrict__ plain, int *counters, int next, unsigned long long *delta,
              const double *__restrict__ zip) {
    extern __shared__ double2 cur[];
    const int cnt = counters[kFxPlain];
    if (blockIdx.x == 0 && threadIdx.x == 0) counters[next] = 0;  // fx_decide counts the next list there
    for (int c = blockIdx.x; c < cnt; c += gridDim.x) {
        const int64_t t = plain[c];
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kSliceThreads) cur[i] = demand(S[t * n + i], V[t * n + i], zip, n, i);
        __syncthreads();
        double dmax = 0.0;
        for (int i = threadIdx.x; i < n; i += kSliceThreads) {
            double2 acc = make_double2(0.0, 0.0);
            for (int k = 0; k < n; ++k) {
                const double2 a = K[(size_t)i * n + k], b = cur[k];
                acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
                acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
            }
            const double2 vn = make_double2(acc.x + W[i].x, acc.y + W[i].y), vo = V[t * n + i];
            const double d = hypot(vn.x - vo.x, vn.y - vo.y);
            if (!(d <= dmax)) dmax = (d != d) ? CUDART_INF : d;  // a NaN step counts as infinite
            V[t * n + i] = vn;
        }
        if (dmax > 0.0) atomicMax(&delta[t], (unsigned long long)__double_as_longlong(dmax));
    }
}

// Per-column decision after a sweep, and the list of the columns that go on.
__global__ void fx_decide(int this_count, int next_count, const int *__restrict__ list, double tol, int max_iter,
                          int *flags, int *iters, unsigned long long *delta, int *counters, int *next) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31, count = counters[this_count];
    if (c == 0) counters[kFxPlain] = 0;
    int active = 0, conv = 0;
    int64_t t = 0;
    if (c < count) {
        t = fx_col(list, c);
        const int k = iters[t] + 1;
        iters[t] = k;
        const double d = __longlong_as_double((long long)delta[t]);
        delta[t] = 0ull;
        if (d <= tol) {
            flags[t] = kDone;
            conv = 1;
        } else if (k >= max_iter || !(d < 1e30)) {
            flags[t] = 0;
        } else {
            active = 1;
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, active), k = __ballot_sync(0xffffffffu, conv);
    int base = 0;
    if (lane == 0) {
        if (m) base = atomicAdd(&counters[next_count], __popc(m));
        if (k) atomicAdd(&counters[kCntConverged], __popc(k));
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    if (active) next[base + __popc(m & ((1u << lane) - 1))] = (int)t;
}

// acc += x * 2^sh for 32 accumulators of exact integers (|x| <= 2^24), rounding below the last place.
// sh is uniform; 31 does not occur (see fx_drop).
__device__ __forceinline__ void add_scaled(const uint32_t (&x)[32], long long (&acc)[32], int sh) {
    if (sh >= 32) {
        const unsigned m = 1u << (sh - 32);
#pragma unroll
        for (int q = 0; q < 32; ++q)
            acc[q] += (long long)((unsigned long long)((unsigned)__float2int_rn(__uint_as_float(x[q])) * m) << 32);
    } else if (sh >= 0) {
        const int m = 1 << sh;
#pragma unroll
        for (int q = 0; q < 32; ++q) acc[q] += (long long)__float2int_rn(__uint_as_float(x[q])) * m;
    } else {
        const int half = 1 << (-sh - 1);
#pragma unroll
        for (int q = 0; q < 32; ++q) acc[q] += (__float2int_rn(__uint_as_float(x[q])) + half) >> -sh;
    }
}

// Flush units.  Group g sums the diagonals 2g and (g > 0) 2g - 1: a step loads digit i of K and digit
// 2g - i of I and multiplies the latter with digit i (upper diagonal) and with digit i - 1, which is
// still in the ring from the step before (lower diagonal), so 16 loaded pairs serve 28 products.  After
// kFlush(g) chunks of 64 buses an accumulator may hold (2g + 1) * 64 * kFlush(g) <= 512 complex terms of
// at most 2^15, and is drained.  The longest group goes first: its units cover the epilogue of the tile before.
constexpr int kFxGroups = 4;
constexpr int kFxAhead = 4;  // columns of V loaded ahead of their update
__device__ __forceinline__ int fx_flush(int g) { return g == 0 ? 8 : (g == 1 ? 2 : 1); }

__device__ __forceinline__ void epi_sync_fx() { asm volatile("bar.sync 1, %0;" ::"n"(kFxEpiThreads) : "memory"); }

// What bounds it: the tensor pipe's operand reads and, for networks of a few hundred buses, the tile's
// epilogue.  With 64 columns an operand of one plane has N = 64, and the pipe, which reads 6 KB of shared
// memory for it, takes 73 cycles instead of the 32 of its arithmetic; with Re and Im side by side in one
// product (N = 128, hence the third plane -Ir) 110 cycles do the work of two.  Per 64 buses of K and tile:
// 26 us with descriptors built by a single divergent thread, 16.5 us with the loops run by the whole
// warp and an elected lane issuing, 12.6 us with N = 128 (28 x 64 x 128 x 64 complex terms: 41 % of the
// tensor peak).  In the epilogue, old values loaded four columns ahead instead of one at a time took a
// launch of 152 tiles at 199 buses from 131 to 68 us.
__global__ void __launch_bounds__(kFxThreads, 1)
    fx_gemm(const __grid_constant__ CUtensorMap tmAr, const __grid_constant__ CUtensorMap tmAi,
            const __grid_constant__ CUtensorMap tmBr, const __grid_constant__ CUtensorMap tmBi,
            const __grid_constant__ CUtensorMap tmBn, const __grid_constant__ FxArgs g) {
    extern __shared__ uint8_t smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + kFxStages * kFxStageBytes);  // [kFxStages] TMA -> MMA
    uint64_t *empty = full + kFxStages;                                // [kFxStages] MMA -> TMA
    uint64_t *tfull = empty + kFxStages;                               // [2] MMA -> epilogue
    uint64_t *tempty = tfull + 2;                                      // [2] epilogue -> MMA
    uint64_t *done = tempty + 2;                                       // [1] all MMAs retired
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *abort_flag = (int *)(tmem_slot + 1);
    double *col_scale = (double *)(abort_flag + 1);       // [kFxN] value of a column's last place, 0: skip
    long long *col_t = (long long *)(col_scale + kFxN);  // [kFxN] the column

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * kFxAcc)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < kFxStages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&tfull[a]), 1);
            mbar_init(smem_u32(&tempty[a]), kFxEpiWarps);
        }
        mbar_init(smem_u32(done), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int count = min(*g.count - g.first, g.cap), total = g.m_tiles * ((max(count, 0) + kFxN - 1) / kFxN);
    volatile int *vabort = abort_flag;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        const uint32_t sbase = smem_u32(smem);
        int64_t k = 0;  // steps issued by this CTA
        for (int tile = blockIdx.x; tile < total && !*vabort; tile += gridDim.x) {
            const int m0 = (tile % g.m_tiles) * kTileM, n0 = (tile / g.m_tiles) * kFxN;
            for (int gr = kFxGroups - 1; gr >= 0 && !*vabort; --gr)
                for (int c = 0; c < g.n_chunks && !*vabort; ++c)
                    for (int i = 0; i <= 2 * gr; ++i, ++k) {
                        const int slot = (int)(k % kFxStages);
                        if (!mbar_wait(smem_u32(&empty[slot]), ((uint32_t)(k / kFxStages) & 1) ^ 1)) {
                            *vabort = 1;
                            atomicExch(g.err, 1);
                            break;
                        }
                        const uint32_t st = sbase + slot * kFxStageBytes, bar = smem_u32(&full[slot]);
                        mbar_expect_tx(bar, kFxStageBytes);
                        const int ra = i * g.n_pad + m0, rb = (2 * gr - i) * g.cap + n0;
                        tma_load_2d(st, &tmAr, bar, c * kChunkK, ra);
                        tma_load_2d(st + kABytes, &tmAi, bar, c * kChunkK, ra);
                        tma_load_2d(st + 2 * kABytes, &tmBr, bar, c * kChunkK, rb);
                        tma_load_2d(st + 2 * kABytes + kBBytes, &tmBi, bar, c * kChunkK, rb);
                        tma_load_2d(st + 2 * kABytes + 2 * kBBytes, &tmBn, bar, c * kChunkK, rb);
                    }
        }
        if (*vabort) {  // let this CTA's copies in flight land before it leaves (bounded)
            for (int64_t q = k - 1; q >= 0 && q >= k - kFxStages; --q)
                mbar_wait(smem_u32(&full[q % kFxStages]), (uint32_t)(q / kFxStages) & 1);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // The whole warp walks the loops and one elected lane issues, so that addresses and descriptors
        // stay in uniform registers.
        const uint32_t sbase = smem_u32(smem);
        const uint32_t pos = idesc_f16(kTileM, 2 * kFxN, 0, 0), neg = idesc_f16(kTileM, 2 * kFxN, 1, 0);
        const bool lead = elect_one();
        uint32_t slot = 0, phase = 0, prev = 0;  // ring position of the next step, slot of the one before
        uint32_t j = 0;                          // flush units issued
        bool ok = true;
        for (int tile = blockIdx.x; tile < total && ok && !*vabort; tile += gridDim.x) {
            for (int gr = kFxGroups - 1; gr >= 0 && ok; --gr) {
                const int fl = fx_flush(gr);
                for (int c0 = 0; c0 < g.n_chunks && ok; c0 += fl, ++j) {
                    const uint32_t a = j & 1;
                    if (!mbar_wait(smem_u32(&tempty[a]), ((j >> 1) & 1) ^ 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t acc = tmem + a * kFxAcc;
                    const int c1 = min(c0 + fl, g.n_chunks);
                    for (int c = c0; c < c1 && ok; ++c) {
                        const int ks = min(kChunkK / 16, g.ksteps - c * (kChunkK / 16));
                        for (int i = 0; i <= 2 * gr; ++i) {
                            if (!mbar_wait(smem_u32(&full[slot]), phase)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const uint64_t dc = sw128_desc(sbase + slot * kFxStageBytes);
                            const uint64_t dp = sw128_desc(sbase + prev * kFxStageBytes);
                            if (lead) {
                                const uint32_t fresh = c == c0;
#pragma unroll
                                for (int kk = 0; kk < kChunkK / 16; ++kk) {
                                    if (kk >= ks) break;
                                    // 32 bytes a K step and the planes of a slot, in 16-byte units.  One
                                    // product serves Re and Im: Kr with (Ir | Ii), -Ki with (Ii | -Ir).
                                    const uint64_t ar = dc + kk * 2, ai = ar + kABytes / 16;
                                    const uint64_t b = ar + 2 * kABytes / 16, bx = b + kBBytes / 16;
                                    umma_f16(acc, ar, b, pos, !(fresh && i == 0 && kk == 0));
                                    umma_f16(acc, ai, bx, neg, 1u);
                                    if (i > 0) {
                                        const uint64_t pr = dp + kk * 2, pi = pr + kABytes / 16;
                                        umma_f16(acc + 2 * kFxN, pr, b, pos, !(fresh && i == 1 && kk == 0));
                                        umma_f16(acc + 2 * kFxN, pi, bx, neg, 1u);
                                    }
                                }
                                if (i > 0) umma_commit(smem_u32(&empty[prev]));
                                if (i == 2 * gr) umma_commit(smem_u32(&empty[slot]));
                            }
                            __syncwarp();
                            prev = slot;
                            if (++slot == kFxStages) slot = 0, phase ^= 1;
                        }
                    }
                    if (lead) umma_commit(smem_u32(&tfull[a]));
                    __syncwarp();
                }
            }
        }
        if (lead) {
            if (!ok) {
                *vabort = 1;
                atomicExch(g.err, 1);
            }
            umma_commit(smem_u32(done));
        }
        __syncwarp();
        mbar_wait(smem_u32(done), 0);  // every MMA of this CTA has retired (bounded)
    } else if (warp >= 2) {
        // ---------------- epilogue: one bus and 32 of the tile's columns per thread ----------------
        const int et = tid - 64;
        const int row = (warp & 3) * 32 + lane, half = (warp - 2) >> 2;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        __shared__ int s_fail;
        if (et == 0) s_fail = 0;
        epi_sync_fx();
        uint32_t j = 0;
        bool fail = false;
        for (int tile = blockIdx.x; tile < total && !fail; tile += gridDim.x) {
            const int n0 = (tile / g.m_tiles) * kFxN, m = (tile % g.m_tiles) * kTileM + row;
            if (et < kFxN) {
                const int c = n0 + et, e = c < count ? g.colexp[c] : kMaxExp;
                col_scale[et] = e < kMaxExp ? g.f1 * pow2d(e) : 0.0;
                col_t[et] = e < kMaxExp ? fx_col(g.list, g.first + c) : 0;
            }
            long long sr[32], si[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) sr[q] = si[q] = 0;
            for (int gr = kFxGroups - 1; gr >= 0; --gr) {
                const int fl = fx_flush(gr);
                const int up = 48 - 16 * gr - g.drop, lo = up + 8;  // places of the diagonals 2 gr and 2 gr - 1
                for (int c0 = 0; c0 < g.n_chunks; c0 += fl, ++j) {
                    const uint32_t a = j & 1;
                    if (!fail && !mbar_wait(smem_u32(&tfull[a]), (j >> 1) & 1)) fail = true;
                    if (fail) continue;
                    tc_fence_after();
                    const uint32_t ta = tmem + a * kFxAcc + lane_off + half * 32;
                    uint32_t x[32];
                    tmem_ld32(ta, x);
                    tmem_wait_ld();
                    add_scaled(x, sr, up);
                    tmem_ld32(ta + kFxN, x);
                    tmem_wait_ld();
                    add_scaled(x, si, up);
                    if (gr > 0) {
                        tmem_ld32(ta + 2 * kFxN, x);
                        tmem_wait_ld();
                        add_scaled(x, sr, lo);
                        tmem_ld32(ta + 3 * kFxN, x);
                        tmem_wait_ld();
                        add_scaled(x, si, lo);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tempty[a]));
                }
            }
            if (fail) atomicOr(&s_fail, 1);
            epi_sync_fx();  // the column information is complete
            if (s_fail) {
                *vabort = 1;
                atomicExch(g.err, 1);
                break;
            }
            const bool row_ok = m < g.n;
            const double2 w = row_ok ? g.W[m] : make_double2(0.0, 0.0);
            unsigned hi_mine = 0, lo_mine = 0;  // lane q: |step|^2 of column q over the warp's rows
            // The old values come kFxAhead columns ahead (the registers left beside the sums).
            double2 vo[kFxAhead];
#pragma unroll
            for (int q = 0; q < kFxAhead; ++q)
                vo[q] = row_ok ? g.V[col_t[half * 32 + q] * g.n + m] : make_double2(0.0, 0.0);
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                const double f = col_scale[half * 32 + q];
                const double2 old = vo[q % kFxAhead];
                if (q + kFxAhead < 32)
                    vo[q % kFxAhead] = row_ok ? g.V[col_t[half * 32 + q + kFxAhead] * g.n + m] : make_double2(0.0, 0.0);
                const double2 vn = make_double2(fma((double)sr[q], f, w.x), fma((double)si[q], f, w.y));
                const double dx = vn.x - old.x, dy = vn.y - old.y, d = fma(dx, dx, dy * dy);
                unsigned long long d2 = 0ull;
                if (f != 0.0 && row_ok) {
                    g.V[col_t[half * 32 + q] * g.n + m] = vn;
                    d2 = (unsigned long long)__double_as_longlong(d != d ? CUDART_INF : d);
                }
                // Non-negative doubles order like their bit patterns: the largest high word, then the
                // largest low word under it.
                const unsigned hi = (unsigned)(d2 >> 32), top = __reduce_max_sync(0xffffffffu, hi);
                const unsigned low = __reduce_max_sync(0xffffffffu, hi == top ? (unsigned)d2 : 0u);
                if (lane == q) hi_mine = top, lo_mine = low;
            }
            const double d = sqrt(__hiloint2double((int)hi_mine, (int)lo_mine));
            if (d > 0.0)
                atomicMax(&g.delta[col_t[half * 32 + lane]], (unsigned long long)__double_as_longlong(d));
            epi_sync_fx();  // the column information is rewritten by the next tile
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kFxAcc) : "memory");
    }
}

// Last place of the 64-bit sums in bits above diagonal 6's: n complex terms below 2^110 in units of
// 2^(48 + drop) stay below 2^62.  No diagonal's place falls on 31 (add_scaled).
int fx_drop(int n) {
    int r = 1;
    while ((1 << r) < 2 * n) ++r;
    for (int d = 0; d < kDig; ++d)
        if (48 - 8 * d - r == 31) ++r;
    return r;
}

struct FxEvents {
    cudaEvent_t e[2] = {nullptr, nullptr};
    bool ok;
    FxEvents() {
        ok = cudaEventCreateWithFlags(&e[0], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&e[1], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) cudaGetLastError();
    }
    ~FxEvents() {
        for (cudaEvent_t x : e)
            if (x) cudaEventDestroy(x);
    }
};

}  // namespace

// From 17 demand buses on: up to 16 the FP64 kernel takes a single chunk of K per tile and both sides wait
// for launches (3 to 10 buses: 260 to 390 us with FP64 FMAs, 276 to 410 here; 19 buses x 96 columns 573
// against 394, 33 x 1,440 905 against 514, 199 x 288 4,516 against 939, 199 x 8,760 26,540 against 1,950,
// 999 x 2,000 109.5 ms against 3.9).  Without room for the digit planes (28 n_pad^2 bytes of K, at most 104 MB of
// currents) solve_fixed returns TPF_ENOMEM before it touches V, and the FP64 kernel serves the call.  Past 8,192 a column's currents no longer fit fx_slice's shared memory.
bool use_fixed(int n, int64_t T) { return n > 16 && n <= kFxMaxN && T < ((int64_t)1 << 31) - kFxN; }

tpf_status solve_fixed(tpf_handle *h, int64_t T, const void *S, void *V, const tpf_opts &o, cudaStream_t st,
                       KernelTimer &timer, int *sweeps_out, int64_t *launches_out, int64_t *gemms_out,
                       int64_t *gemm_cols_out) {
    Workspace &w = h->ws;
    DeviceNet &d = h->dev;
    const int n = d.n, n_pad = d.n_pad;
    const size_t plane_k = (size_t)n_pad * n_pad;
    const int k_order = d.k_order;  // every component of K / c is below 2^k_order
    int64_t launches = 0, gemms = 0, gemm_cols = 0;
    if (!d.Kd16) {
        __half *planes = nullptr;
        if (cudaMalloc(&planes, sizeof(__half) * 2 * kDig * plane_k) != cudaSuccess) {
            cudaGetLastError();
            return TPF_ENOMEM;
        }
        fx_k_digits<<<(unsigned)((plane_k + 255) / 256), 256, 0, st>>>((const double2 *)d.K64, d.k_col_order, n, n_pad,
                                                                       kBits - k_order, planes, planes + kDig * plane_k);
        // The handle has them once they are written: its next solve may be on another stream.
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(planes);
            return TPF_ECUDA;
        }
        d.Kd16 = planes;
        ++launches;
    }
    int sms = 0;
    TPF_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    const int64_t per_col = (int64_t)sizeof(__half) * 3 * kDig * n_pad;
    // Columns per launch: two tiles per SM.  Their digit planes (104 MB) still pass from fx_slice to fx_gemm
    // mostly through the 129 MB L2, and the second tile's first products run under the first one's
    // epilogue: 8,760 columns of 199 buses take 1.92 ms, with one tile per SM and launch 2.02; 2,000 of 999
    // buses 3.85 and 3.99.
    const int64_t cap = std::min<int64_t>(round_up(T, kFxN), (int64_t)kFxN * std::max(1, 2 * sms / (n_pad / kTileM)));
    const size_t digit_bytes = (size_t)per_col * cap, exp_bytes = sizeof(int) * (size_t)round_up(cap, 64);
    const size_t need = digit_bytes + exp_bytes + 3 * sizeof(int) * (size_t)T;
    if (w.fx_bytes < need) {
        cudaFree(w.fx_buf);
        w.fx_buf = nullptr;
        w.fx_bytes = 0;
        if (cudaMalloc(&w.fx_buf, need) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(d.Kd16);  // leaves the room to the FP64 sweeps
            w.fx_buf = d.Kd16 = nullptr;
            return TPF_ENOMEM;
        }
        w.fx_bytes = need;
    }
    __half *const Dr = (__half *)w.fx_buf, *const Di = Dr + (size_t)kDig * cap * n_pad, *const Dn = Di + (size_t)kDig * cap * n_pad;
    int *const colexp = (int *)((char *)w.fx_buf + digit_bytes);
    int *const lists[2] = {(int *)((char *)colexp + exp_bytes), (int *)((char *)colexp + exp_bytes) + T};
    int *const plain = lists[1] + T;
    CUtensorMap ar, ai, br, bi, bn;
    if (!make_f16_map(&ar, d.Kd16, n_pad, (uint64_t)kDig * n_pad, kTileM) ||
        !make_f16_map(&ai, (__half *)d.Kd16 + kDig * plane_k, n_pad, (uint64_t)kDig * n_pad, kTileM) ||
        !make_f16_map(&br, Dr, n_pad, (uint64_t)kDig * cap, kFxN) ||
        !make_f16_map(&bi, Di, n_pad, (uint64_t)kDig * cap, kFxN) || !make_f16_map(&bn, Dn, n_pad, (uint64_t)kDig * cap, kFxN))
        return TPF_ECUDA;
    static std::atomic<uint64_t> attr{0};
    if (!once_per_device(attr, [] {
            return cudaFuncSetAttribute(fx_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFxSmem) == cudaSuccess &&
                   cudaFuncSetAttribute(fx_slice, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * kFxMaxN) == cudaSuccess &&
                   cudaFuncSetAttribute(fx_column, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * kFxMaxN) == cudaSuccess;
        }))
        return TPF_ECUDA;
    FxArgs g{};
    g.n = n;
    g.n_pad = n_pad;
    g.m_tiles = n_pad / kTileM;
    g.ksteps = (n + 15) / 16;
    g.n_chunks = (g.ksteps + kChunkK / 16 - 1) / (kChunkK / 16);
    g.cap = (int)cap;
    g.drop = fx_drop(n);
    g.f1 = ldexp(1.0, g.drop - 62 + k_order);
    g.colexp = colexp;
    g.W = (const double2 *)d.W64;
    g.V = (double2 *)V;
    g.delta = w.delta64;
    g.err = w.counters + kCntError;

    TPF_CK(cudaMemsetAsync(w.counters, 0, sizeof(int) * 8, st));
    const int64_t cols = round_up(T, kTileN), work = cols > T * n ? cols : T * n;
    fx_init<<<(unsigned)((work + 255) / 256), 256, 0, st>>>(T, cols, n, o.start == TPF_START_FLAT, (double2 *)V,
                                                            w.flags, w.iters, w.delta64);
    ++launches;
    const size_t smem = sizeof(double2) * (size_t)n;
    int *const host = w.counters_host;  // two blocks of 8, by sweep parity
    std::memset(host, 0, sizeof(int) * 16);
    host[0] = (int)T;
    TPF_CK(cudaMemcpyAsync(w.counters + kFxCount, host, sizeof(int), cudaMemcpyHostToDevice, st));
    FxEvents ev;
    if (!ev.ok) return TPF_ECUDA;
    // The lengths of the lists stay on the device, and sweep k + 1 is queued before the host has seen
    // whether sweep k left any column: the host's round trip is hidden at the price of one empty sweep.
    // `bound` is the last length seen.
    int bound = (int)T, sweeps = 0;
    for (int k = 0; k < o.max_iter; ++k) {
        const int *list = k ? lists[(k - 1) & 1] : nullptr;
        const int cur = kFxCount + (k & 1), next = kFxCount + ((k + 1) & 1);
        const int64_t gemms_before = gemms;
        g.list = list;
        g.count = w.counters + cur;
        for (int64_t c0 = 0; c0 < bound; c0 += cap) {
            const int cnt = (int)std::min<int64_t>(cap, bound - c0);
            g.first = (int)c0;
            timer.begin(KernelTimer::kResidual);
            fx_slice<<<(unsigned)cnt, kSliceThreads, smem, st>>>(n, n_pad, list, g.count, g.first, (const double2 *)S,
                                                                 (const double2 *)V, d.zip64, d.k_col_order, Dr, Di, Dn,
                                                                 (int)cap, colexp, plain, w.counters);
            timer.end();
            const int total = g.m_tiles * ((cnt + kFxN - 1) / kFxN);
            timer.begin(KernelTimer::kGemm);
            fx_gemm<<<(unsigned)std::min(total, sms), kFxThreads, kFxSmem, st>>>(ar, ai, br, bi, bn, g);
            timer.end();
            launches += 2;
            ++gemms;
        }
        timer.begin(KernelTimer::kResidual);
        fx_column<<<(unsigned)std::min(bound, sms), kSliceThreads, smem, st>>>(
            (const double2 *)d.K64, (const double2 *)d.W64, (const double2 *)S, (double2 *)V, n, plain, w.counters,
            next, w.delta64, d.zip64);
        fx_decide<<<(unsigned)((bound + 255) / 256), 256, 0, st>>>(cur, next, list, o.tol, o.max_iter, w.flags, w.iters,
                                                                   w.delta64, w.counters, lists[k & 1]);
        timer.end();
        launches += 2;
        TPF_CK(cudaGetLastError());
        TPF_CK(cudaMemcpyAsync(host + 8 * (k & 1), w.counters, sizeof(int) * 8, cudaMemcpyDeviceToHost, st));
        TPF_CK(cudaEventRecord(ev.e[k & 1], st));
        if (k == 0) {
            sweeps = 1;
            gemm_cols = T;
            continue;
        }
        // What sweep k - 1 left: the columns of sweep k.
        TPF_CK(cudaEventSynchronize(ev.e[(k - 1) & 1]));
        const int *seen = host + 8 * ((k - 1) & 1);
        if (seen[kCntError]) break;
        bound = seen[cur];
        if (bound == 0) {
            gemms = gemms_before;
            break;
        }
        ++sweeps;
        gemm_cols += bound;
    }
    TPF_CK(cudaStreamSynchronize(st));
    if (host[kCntError] | host[8 + kCntError]) return TPF_ETIMEOUT;
    *sweeps_out = sweeps;
    *launches_out = launches;
    *gemms_out = gemms;
    *gemm_cols_out = gemm_cols;
    return TPF_OK;
}

}  // namespace tpf
