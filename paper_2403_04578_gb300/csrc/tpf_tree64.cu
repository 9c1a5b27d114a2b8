// Sparse tensor formulation in plain double precision (Sec. IV-B, Eq. 13-14, Algorithm 2).
//
// The same iterate as the mixed tree kernel and as Algorithm 1, V_{k+1} = K conj(S ./ V_k) + W,
// evaluated without K: on a radial feeder Y_dd factors without fill-in, and with the demand buses
// in depth-first preorder the substitution is two prefix sums per sweep,
//
//     L_q      = P[end_q - 1] - P[q - 1],     P = inclusive prefix sum of I = conj(S ./ V)
//     V_new,q  = v_s - (prefix sum at q of E),  E_q = z_q L_q - sum of z_b L_b over the b whose
//                                                   subtree range [b, end_b) ends at q
//
// (the path sum of the branch drops from the slack to q).  This is the plain double-precision
// fixed-point iteration of the sparse form, with Algorithm 1's per-column stopping rule
// (max_i |V_{k+1,i} - V_{k,i}| <= tol, the first iterate that meets it is returned), so that it can stand
// beside the mixed-precision sparse path as a like-for-like FP64 reference.
//
// GB300 issues FP64 at 1/64 of its FP32 rate, and with every operation on that pipe it bounds this kernel
// (16,384 columns of 1,000 buses in 16.6 ms).  So the sums run in 64-bit fixed point, two integer
// instructions instead of an FP64 one that takes sixteen times as long, the load currents are integer
// quotients (tpf_fx.cuh) and the branch terms 128-bit integer products: 3.5 ms, bound by issue slots.  ZIP
// currents and the products of the balance at the end stay in FP64.  Currents are integers of a last place
// 2^cur that the sum over all buses cannot overflow (per column, from its largest load), branch terms,
// path sums and V integers of 2^-61 pu.  Integer sums are exact, so what an FP64 prefix sum loses at its
// own magnitude is not lost; V is rounded to FP64 where it enters a product and where it is returned.
// The block's largest step is taken in FP32 and repeated in FP64 when it lies within 1e-5 of tol.  A column
// that leaves the range of the integers (a voltage below half a pu, a current beyond four times the largest
// load, a drop of half a pu on one branch or of 1 pu in all, anything not finite), or whose last place is too coarse
// for the feeder's impedances (fixed_limits below), is solved in FP64 throughout.
//
// One block owns one column for its whole solve, with the slot layout of the mixed kernel
// (thread k owns depth-first positions k*bpt .. k*bpt + bpt - 1, position q at slot
// (q % bpt) * threads + q / bpt).  V and the thread's prefix values live in registers; shared
// memory holds S, z and one prefix array per slot (P in the first half of a sweep, the branch
// terms in ends-list order in the second), plus the range, ends-index and parent slots.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "tpf_fx.cuh"
#include "tpf_internal.h"

namespace tpf {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxWarps64 = kTreeMaxThreads / 32;
constexpr int kCntLeft = 6;

struct Tree64Args {
    int n, max_iter;
    double tol2;     // tol squared: a step is compared squared
    float tol2_lo, tol2_hi;  // tol2 in units of 2^-122 less and plus 1e-5 of itself
    int fixed;       // sums in fixed point
    int log2n;       // n <= 2^log2n
    int z_e;         // every component of z but the large ones is below 2^z_e
    int cur_max;     // the coarsest last place of a column's currents, and the finest with which the
    int cur_min;     // mismatch's branch currents still fit (DeviceNet)
    longlong2 vs_fx; // slack voltage in 2^-61 pu
    double2 vs;      // slack voltage
    const int *col, *end, *par, *ecnt, *kidx;
    const double2 *z;      // [slot] branch impedance to the parent
    const double2 *y;      // [slot] its inverse
    const double *zip;     // [3][n] (alpha_P, alpha_I, alpha_Z) by column, or null
    const double2 *S;      // [T][n]
    double2 *V;            // [T][n]; read first as V_0 when given
    int given;
    int32_t *iters_out;    // [T] or null
    double *mismatch_out;  // [T] or null
    int *counters;         // [kCntConverged] converged columns, [5] largest sweep count, [kCntLeft]
    const int *list;       // the columns of the launch, or null: 0, 1, ...
    int *left;             // not null: takes the columns that leave the integers, kCntLeft of them (tree64_bpt)
};

__device__ __forceinline__ double2 dadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 dsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 dmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double dabs2(double2 a) { return fma(a.x, a.x, a.y * a.y); }
// ---- fixed point ----
// x * 2^e, rounded once (the scale by the exponent field; the results are normal numbers).
__device__ __forceinline__ double from_fx(long long x, int e) {
    const double d = __ll2double_rn(x);
    return __hiloint2double(x ? __double2hiint(d) + (e << 20) : 0, __double2loint(d));
}
__device__ __forceinline__ longlong2 ladd(longlong2 a, longlong2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ longlong2 lsub(longlong2 a, longlong2 b) { return make_longlong2(a.x - b.x, a.y - b.y); }

// z L in 2^-61 pu from 128-bit products (|z| < 2^61 and |L| < 2^62 in their units), rounded once; false for
// half a pu and more.
__device__ __forceinline__ bool branch_fx(longlong2 z, longlong2 L, int sh, longlong2 &out) {
    const __int128 half = (__int128)1 << (sh - 1), lim = (__int128)1 << (kFx - 1);
    const __int128 x = ((__int128)z.x * L.x - (__int128)z.y * L.y + half) >> sh;
    const __int128 y = ((__int128)z.x * L.y + (__int128)z.y * L.x + half) >> sh;
    out = make_longlong2((long long)x, (long long)y);
    return x < lim && x >= -lim && y < lim && y >= -lim;
}

// max that returns NaN if either operand is NaN
__device__ __forceinline__ double dmax_nan(double m, double x) { return (m != m || x <= m) ? m : x; }

// Demand current of Eq. 3 in FP64: alpha_P conj(s / v) + alpha_I conj(s) + alpha_Z conj(s) v for
// the bus in column i (constant power, conj(s / v), without ZIP coefficients).
template <bool kZip>
__device__ __forceinline__ double2 demand64(double2 v, double2 s, const Tree64Args &g, int slot) {
    const double inv = 1.0 / dabs2(v);
    const double2 csv = make_double2(fma(s.x, v.x, s.y * v.y), fma(s.x, v.y, -s.y * v.x));  // conj(s) v
    const double2 c = make_double2(csv.x * inv, csv.y * inv);                             // conj(s / v)
    if (!kZip) return c;
    const int i = __ldg(g.col + slot), n = g.n;
    const double ap = __ldg(g.zip + i), ai = __ldg(g.zip + n + i), az = __ldg(g.zip + 2 * n + i);
    return make_double2(ap * c.x + ai * s.x + az * csv.x, ap * c.y - ai * s.y + az * csv.y);
}

// Exclusive scan over the block's threads (thread order) of one complex FP64 value; ends with all
// warp totals read, after one barrier.
__device__ __forceinline__ double2 block_scan64(double2 v, double2 *wt, int lane, int warp, int nw) {
    double2 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double ux = __shfl_up_sync(kFull, inc.x, o), uy = __shfl_up_sync(kFull, inc.y, o);
        if (lane >= o) inc = dadd(make_double2(ux, uy), inc);
    }
    const double ex = __shfl_up_sync(kFull, inc.x, 1), ey = __shfl_up_sync(kFull, inc.y, 1);
    if (lane == 31) wt[warp] = inc;
    __syncthreads();
    // Lane l scans the warp totals of warps 0..l; warp w takes lane w-1's sum.
    double2 t = lane < nw ? wt[lane] : make_double2(0.0, 0.0);
    for (int o = 1; o < nw; o <<= 1) {
        const double ux = __shfl_up_sync(kFull, t.x, o), uy = __shfl_up_sync(kFull, t.y, o);
        if (lane >= o) t = dadd(make_double2(ux, uy), t);
    }
    const int src = warp ? warp - 1 : 0;
    const double px = __shfl_sync(kFull, t.x, src), py = __shfl_sync(kFull, t.y, src);
    const double2 before = warp ? make_double2(px, py) : make_double2(0.0, 0.0);
    return dadd(before, lane ? make_double2(ex, ey) : make_double2(0.0, 0.0));
}

// The same of integers (a lane's exclusive value as its inclusive one less its own).
__device__ __forceinline__ longlong2 block_scan_fx(longlong2 v, longlong2 *wt, int lane, int warp, int nw) {
    longlong2 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long ux = __shfl_up_sync(kFull, inc.x, o), uy = __shfl_up_sync(kFull, inc.y, o);
        if (lane >= o) inc = ladd(make_longlong2(ux, uy), inc);
    }
    if (lane == 31) wt[warp] = inc;
    __syncthreads();
    longlong2 t = lane < nw ? wt[lane] : make_longlong2(0, 0);
    for (int o = 1; o < nw; o <<= 1) {
        const long long ux = __shfl_up_sync(kFull, t.x, o), uy = __shfl_up_sync(kFull, t.y, o);
        if (lane >= o) t = ladd(make_longlong2(ux, uy), t);
    }
    const int src = warp ? warp - 1 : 0;
    const long long px = __shfl_sync(kFull, t.x, src), py = __shfl_sync(kFull, t.y, src);
    const longlong2 off = lsub(inc, v);
    return warp ? ladd(make_longlong2(px, py), off) : off;
}

template <int kBPT>
__device__ __forceinline__ int next_slot64(int s, int th) {
    return s < (kBPT - 1) * th ? s + th : s - (kBPT - 1) * th + 1;
}

// Beside the slot of a subtree's last position (below 4,096): the position's impedance is 2^z_e and more.
constexpr int kLarge = 1 << 14;

// Currents in integers up to 2,048 buses (8 B more of shared memory a slot than 4,096 buses leave).
template <int kBPT>
constexpr bool kIntCurrents = kBPT < 8;

template <int kBPT, bool kZip>
__global__ void __launch_bounds__(kTreeMaxThreads) __maxnreg__(kBPT == 4 ? 80 : (kBPT == 2 ? 64 : 128)) f64_tree(const __grid_constant__ Tree64Args g) {
    extern __shared__ double2 dsm[];
    const int th = (int)blockDim.x, ns = th * kBPT, n = g.n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = th >> 5;
    double2 *const Ss = dsm;        // [ns] S of each position
    double2 *const Zs = dsm + ns;   // [ns] z of each position; branch currents J at the end
    double2 *const PX = dsm + 2 * ns;  // [ns] prefix sums P, then branch terms in ends-list order
    constexpr bool kInt = kIntCurrents<kBPT> && !kZip;
    float2 *const Sf = reinterpret_cast<float2 *>(dsm + 3 * ns);   // [ns] FP32 loads of current_fx (kIntCurrents)
    longlong2 *const Si = reinterpret_cast<longlong2 *>(Ss);       // its loads modulo 2^64, in place of Ss
    longlong2 *const Zi = reinterpret_cast<longlong2 *>(Zs);       // z in units of 2^(z_e - 61), in place of Zs
    short *const s_rng = reinterpret_cast<short *>(Sf + (kIntCurrents<kBPT> ? ns : 0));  // slot of the subtree's last position
    short *const s_kidx = s_rng + ns;  // where the position's branch term goes in ends-list order (-1: nowhere)
    short *const s_par = s_kidx + ns;  // parent slot, -1 = the slack
    longlong2 *const PXi = reinterpret_cast<longlong2 *>(PX);  // the same in fixed point
    __shared__ double2 wt[kMaxWarps64];
    longlong2 *const wti = reinterpret_cast<longlong2 *>(wt);
    __shared__ double wm[kMaxWarps64];
    __shared__ unsigned wu[kMaxWarps64];
    const int64_t t = g.list ? g.list[blockIdx.x] : (int)blockIdx.x;
    const int base = tid * kBPT;
    const double2 *S = g.S + t * n;
    double2 *Vc = g.V + t * n;

    double2 V[kBPT];  // in fixed point the bits of two integers of 2^-61 pu
    int ecnt[kBPT];
    unsigned smax = 0;  // largest high word of the thread's loads
    auto get_v = [&V](int j) { return make_longlong2(__double_as_longlong(V[j].x), __double_as_longlong(V[j].y)); };
    auto set_v = [&V](int j, longlong2 x) {
        V[j] = make_double2(__longlong_as_double(x.x), __longlong_as_double(x.y));
    };
#pragma unroll
    for (int j = 0; j < kBPT; ++j) {
        const int q = base + j, s = j * th + tid;
        double2 sv = make_double2(0.0, 0.0), zv = sv;
        V[j] = make_double2(1.0, 0.0);  // flat start (Algorithm 1)
        ecnt[j] = 0;
        int rng = s;
        if (q < n) {
            const int i = g.col[s];
            sv = S[i];
            zv = g.z[s];
            ecnt[j] = g.ecnt[s];
            const int e = g.end[s] - 1;  // last position of the subtree
            rng = (e % kBPT) * th + e / kBPT;
            if (g.given) V[j] = Vc[i];
        }
        smax = max(smax, max((unsigned)__double2hiint(sv.x) & 0x7fffffffu, (unsigned)__double2hiint(sv.y) & 0x7fffffffu));
        Ss[s] = sv;
        Zs[s] = zv;
        s_rng[s] = (short)rng;
        s_kidx[s] = (short)g.kidx[s];
        s_par[s] = (short)g.par[s];
    }
    smax = __reduce_max_sync(kFull, smax);
    if (lane == 0) wu[warp] = smax;
    __syncthreads();
    for (int w = 0; w < nw; ++w) smax = max(smax, wu[w]);
    // Currents below 2^cur_e each (four times the largest load), so sums below 2^(cur_e + log2n):
    // a last place of 2^cur keeps them within 62 bits.
    const int cur_e = min(max((int)(smax >> 20) - 1022, -800), 1024) + 2, cur = cur_e + g.log2n - 62;
    // Branch terms z L: products in units of 2^(cur + z_e - 61) for a result in 2^-61 pu.
    const int zsh = min(-(cur + g.z_e), 126);
    bool fixed = g.fixed && cur_e < 900 && zsh >= 1 && cur <= g.cur_max, over = false;
    if (fixed) {
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            over |= order(V[j].x) >= 1 || order(V[j].y) >= 1;
            set_v(j, make_longlong2(to_fx(V[j].x, kFx), to_fx(V[j].y, kFx)));
            const int s = j * th + tid;
            double2 zv = Zs[s];
            if (max(order(zv.x), order(zv.y)) >= g.z_e) {
                s_rng[s] |= kLarge;
                zv = make_double2(0.0, 0.0);
            }
            Zi[s] = make_longlong2(to_fx(zv.x, 61 - g.z_e), to_fx(zv.y, 61 - g.z_e));
            if (kInt) {
                const int u = cur_e - 25;
                const double2 sv = Ss[s];
                const double scale = __hiloint2double((1023 - u) << 20, 0);
                Sf[s] = make_float2(__double2float_rn(sv.x * scale), __double2float_rn(sv.y * scale));
                Si[s] = make_longlong2(to_fx(sv.x, 53 - u), to_fx(sv.y, 53 - u));
            }
        }
    }

    int it = 0;
    bool conv = false;
    auto leave = [&] {
        if (tid == 0) g.left[atomicAdd(&g.counters[kCntLeft], 1)] = (int)t;
    };
    if (kBPT == 2 && !fixed && g.left) {
        leave();
        return;
    }
    for (;;) {
        if (fixed) {
            longlong2 loc[kBPT], run = make_longlong2(0, 0);
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int q = base + j, s = j * th + tid;
                if (q < n) {
                    const longlong2 vi = get_v(j);
                    if (kInt) {
                        longlong2 I;
                        over |= !current_fx(vi, Si[s], Sf[s], g.log2n, I);
                        run = ladd(run, I);
                    } else {
                        const double2 I = demand64<kZip>(make_double2(from_fx(vi.x, -kFx), from_fx(vi.y, -kFx)), Ss[s], g, s);
                        over |= order(I.x) >= cur_e || order(I.y) >= cur_e || !(abs2_fx(vi) >= kLowV2);
                        run = ladd(run, make_longlong2(to_fx(I.x, -cur), to_fx(I.y, -cur)));
                    }
                }
                loc[j] = run;
            }
            longlong2 off = block_scan_fx(run, wti, lane, warp, nw);
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                loc[j] = ladd(off, loc[j]);
                PXi[j * th + tid] = loc[j];
            }
            __syncthreads();
#pragma unroll
            for (int j = kBPT - 1; j >= 0; --j) {
                const int q = base + j, s = j * th + tid;
                longlong2 x = make_longlong2(0, 0);
                if (q < n) {
                    const int rl = s_rng[s], ls = rl & (kLarge - 1);
                    longlong2 L = ls == s ? loc[j] : PXi[ls];
                    if (j) L = lsub(L, loc[j - 1]);
                    else if (q > 0) L = lsub(L, PXi[(kBPT - 1) * th + tid - 1]);
                    over |= !branch_fx(Zi[s], L, zsh, x);
                    if (rl & kLarge) over |= (L.x | L.y) != 0;
                }
                loc[j] = x;
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int k = s_kidx[j * th + tid];
                if (k >= 0) PXi[k] = loc[j];
            }
            __syncthreads();
            run = make_longlong2(0, 0);
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int st = ecnt[j] & 0xffff, cnt = (int)(((unsigned)ecnt[j] >> 16) & 0x3fffu);
                longlong2 e = loc[j];
                for (int k = 0; k < cnt; ++k) e = lsub(e, PXi[st + k]);
                run = ladd(run, e);
                loc[j] = run;
            }
            off = block_scan_fx(run, wti, lane, warp, nw);
            float m = 0.0f;
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int q = base + j;
                if (q < n) {
                    const longlong2 drop = ladd(off, loc[j]), vn = lsub(g.vs_fx, drop);
                    const longlong2 d = lsub(vn, get_v(j));
                    // |drop| < 1, |V_k+1| < 3, |V_k| < 3: a difference that wraps is still above 3.  (Where a
                    // path sum itself wraps, at 4, one above it on its path lies between 1 and 4.)
                    constexpr unsigned long long k1 = 1ull << kFx;
                    over |= (unsigned long long)drop.x + k1 >= 2 * k1 || (unsigned long long)drop.y + k1 >= 2 * k1;
                    const float dx = __ll2float_rn(d.x), dy = __ll2float_rn(d.y);
                    m = fmaxf(m, fmaf(dx, dx, dy * dy));
                    loc[j] = d;
                    set_v(j, vn);
                }
            }
            // Non-negative floats order like their bits; all ones stand for a column out of range.
            unsigned mu = __reduce_max_sync(kFull, over ? ~0u : __float_as_uint(m));
            if (lane == 0) wu[warp] = mu;
            __syncthreads();
            mu = wu[0];
            for (int w = 1; w < nw; ++w) mu = max(mu, wu[w]);
            if (mu == ~0u) {  // every thread alike: from the start again in FP64
                if (kBPT == 2 && g.left) {
                    leave();
                    return;
                }
                fixed = false;
                it = 0;
#pragma unroll
                for (int j = 0; j < kBPT; ++j) {
                    const int q = base + j, s = j * th + tid;
                    V[j] = q < n && g.given ? Vc[g.col[s]] : make_double2(1.0, 0.0);
                    if (kInt) Ss[s] = q < n ? S[g.col[s]] : make_double2(0.0, 0.0);
                    Zs[s] = q < n ? g.z[s] : make_double2(0.0, 0.0);
                    s_rng[s] &= kLarge - 1;
                }
                continue;
            }
            ++it;
            m = __uint_as_float(mu);
            if (m <= g.tol2_hi) {
                conv = m <= g.tol2_lo;
                if (!conv) {  // too close to tol for FP32
                    double md = 0.0;
#pragma unroll
                    for (int j = 0; j < kBPT; ++j)
                        if (base + j < n) md = fmax(md, dabs2(make_double2(from_fx(loc[j].x, -kFx), from_fx(loc[j].y, -kFx))));
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) md = fmax(md, __shfl_xor_sync(kFull, md, o));
                    if (lane == 0) wm[warp] = md;
                    __syncthreads();
                    md = wm[0];
                    for (int w = 1; w < nw; ++w) md = fmax(md, wm[w]);
                    conv = md <= g.tol2;
                }
                if (conv) break;
            }
            if (it >= g.max_iter) break;
            continue;
        }
        // Load currents and their inclusive prefix sums P.
        double2 loc[kBPT], run = make_double2(0.0, 0.0);
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int q = base + j, s = j * th + tid;
            if (q < n) run = dadd(run, demand64<kZip>(V[j], Ss[s], g, s));
            loc[j] = run;
        }
        double2 off = block_scan64(run, wt, lane, warp, nw);
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            loc[j] = dadd(off, loc[j]);
            PX[j * th + tid] = loc[j];
        }
        __syncthreads();
        // Branch terms x_q = z_q (P[end_q - 1] - P[q - 1]); descending j keeps loc[j - 1] = P[q - 1].
#pragma unroll
        for (int j = kBPT - 1; j >= 0; --j) {
            const int q = base + j, s = j * th + tid;
            double2 x = make_double2(0.0, 0.0);
            if (q < n) {
                const int ls = s_rng[s];
                double2 L = ls == s ? loc[j] : PX[ls];
                if (j) L = dsub(L, loc[j - 1]);
                else if (q > 0) L = dsub(L, PX[(kBPT - 1) * th + tid - 1]);
                x = dmul(Zs[s], L);
            }
            loc[j] = x;
        }
        __syncthreads();  // every read of P is done: PX takes the branch terms in ends-list order
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int k = s_kidx[j * th + tid];
            if (k >= 0) PX[k] = loc[j];
        }
        __syncthreads();
        // Path sums: prefix sums of E_q = x_q - (x_b of every b whose range ends at q).
        run = make_double2(0.0, 0.0);
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int st = ecnt[j] & 0xffff, cnt = (int)(((unsigned)ecnt[j] >> 16) & 0x3fffu);
            double2 e = loc[j];
            for (int k = 0; k < cnt; ++k) e = dsub(e, PX[st + k]);
            run = dadd(run, e);
            loc[j] = run;
        }
        off = block_scan64(run, wt, lane, warp, nw);
        double m = 0.0;
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int q = base + j;
            if (q < n) {
                const double2 vn = dsub(g.vs, dadd(off, loc[j]));
                m = dmax_nan(m, dabs2(dsub(vn, V[j])));
                V[j] = vn;
            }
        }
        // Block max of |step|^2 (a NaN stays NaN); every thread reads the same warp maxima and so
        // takes the same decision.
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = dmax_nan(m, __shfl_xor_sync(kFull, m, o));
        if (lane == 0) wm[warp] = m;
        __syncthreads();
        m = wm[0];
        for (int w = 1; w < nw; ++w) m = dmax_nan(m, wm[w]);
        ++it;
        if (m <= g.tol2) {
            conv = true;
            break;
        }
        if (it >= g.max_iter || !(m < 1e60)) break;
    }

    // Outputs: V, the iteration count, and the power mismatch max_i |V_i conj((Y v)_i) + S_i| at
    // the returned V (ZIP: |V_i| |(Y v)_i + i_d,i|).  On the tree (Y v)_q = -J_q + sum over the
    // children k of J_k with the branch currents J_k = y_k (V_parent(k) - V_k), y_k = 1 / z_k.
    // In fixed point the branch currents and their sums are integers of 2^cur like the load currents, and
    // the largest mismatch is compared as a square.  The last place of the returned V times a very large y can be
    // beyond those integers (cur_min): then FP64.
    double worst = 0.0;
    if (fixed) {
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const longlong2 v = get_v(j);
            V[j] = make_double2(from_fx(v.x, -kFx), from_fx(v.y, -kFx));
        }
    }
    if (fixed && g.mismatch_out && cur < g.cur_min) {
        fixed = false;
#pragma unroll 1
        for (int j = 0; j < kBPT; ++j) {
            const int q = base + j, s = j * th + tid;
            if (kInt) Ss[s] = q < n ? S[g.col[s]] : make_double2(0.0, 0.0);
            Zs[s] = q < n ? g.z[s] : make_double2(0.0, 0.0);
            s_rng[s] &= kLarge - 1;
        }
    }
    if (fixed) {
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int q = base + j, s = j * th + tid;
            if (q < n) Vc[g.col[s]] = V[j];
            PXi[s] = make_longlong2(to_fx(V[j].x, kFx), to_fx(V[j].y, kFx));  // the returned V, rounded to FP64
        }
        __syncthreads();
        longlong2 J[kBPT];
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int q = base + j, s = j * th + tid;
            J[j] = make_longlong2(0, 0);
            if (q < n && g.mismatch_out) {
                const int p = s_par[s];
                const longlong2 d = lsub(p >= 0 ? PXi[p] : g.vs_fx, PXi[s]);
                const double2 i = dmul(__ldg(g.y + s), make_double2(from_fx(d.x, -kFx), from_fx(d.y, -kFx)));
                J[j] = make_longlong2(to_fx(i.x, -cur), to_fx(i.y, -cur));
            }
        }
        if (g.mismatch_out) {
            __syncthreads();  // every parent has been read
#pragma unroll
            for (int j = 0; j < kBPT; ++j) PXi[j * th + tid] = J[j];
            __syncthreads();
            double worst2 = 0.0;
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int q = base + j, s = j * th + tid;
                if (q >= n) continue;
                longlong2 acc = make_longlong2(-J[j].x, -J[j].y);
                const int lq = s_rng[s] & (kLarge - 1);
                for (int ks = lq == s ? -1 : next_slot64<kBPT>(s, th); ks >= 0;) {
                    acc = ladd(acc, PXi[ks]);
                    const int lc = s_rng[ks] & (kLarge - 1);
                    ks = lc == lq ? -1 : next_slot64<kBPT>(lc, th);
                }
                const double2 a = make_double2(from_fx(acc.x, cur), from_fx(acc.y, cur)), v = V[j];
                const double2 sv = kInt ? S[g.col[s]] : Ss[s];
                double m2;
                if (kZip)
                    m2 = dabs2(v) * dabs2(dadd(a, demand64<kZip>(v, sv, g, s)));
                else
                    m2 = dabs2(make_double2(fma(v.x, a.x, fma(v.y, a.y, sv.x)), fma(v.y, a.x, fma(-v.x, a.y, sv.y))));
                worst2 = fmax(worst2, m2);
            }
            worst = sqrt(worst2);
        }
    } else {
#pragma unroll
        for (int j = 0; j < kBPT; ++j) {
            const int q = base + j, s = j * th + tid;
            if (q < n) Vc[g.col[s]] = V[j];
            PX[s] = V[j];
        }
        __syncthreads();
        if (g.mismatch_out) {
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int q = base + j, s = j * th + tid;
                if (q < n) {
                    const int p = s_par[s];
                    const double2 zq = Zs[s];
                    const double inv = 1.0 / dabs2(zq);
                    const double2 y = make_double2(zq.x * inv, -zq.y * inv);
                    Zs[s] = dmul(y, dsub(p >= 0 ? PX[p] : g.vs, V[j]));  // the slot's own z is read first
                }
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kBPT; ++j) {
                const int q = base + j, s = j * th + tid;
                if (q < n) {
                    double2 acc = make_double2(-Zs[s].x, -Zs[s].y);
                    // The first child is q + 1; each next one follows the previous one's last position;
                    // the child whose subtree ends where q's ends is the last.
                    const int lq = s_rng[s];
                    for (int ks = lq == s ? -1 : next_slot64<kBPT>(s, th); ks >= 0;) {
                        acc = dadd(acc, Zs[ks]);
                        const int lc = s_rng[ks];
                        ks = lc == lq ? -1 : next_slot64<kBPT>(lc, th);
                    }
                    const double2 v = V[j], sv = Ss[s];
                    double mm;
                    if (kZip) {
                        const double2 i_d = demand64<kZip>(v, sv, g, s);
                        mm = sqrt(dabs2(v) * dabs2(dadd(acc, i_d)));
                    } else {
                        // V conj(acc) + S
                        mm = sqrt(dabs2(make_double2(v.x * acc.x + v.y * acc.y + sv.x, v.y * acc.x - v.x * acc.y + sv.y)));
                    }
                    worst = dmax_nan(worst, mm);
                }
            }
        }
    }
    if (g.mismatch_out) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) worst = dmax_nan(worst, __shfl_xor_sync(kFull, worst, o));
        if (lane == 0) wm[warp] = worst;  // (the last sweep's maxima were read before two barriers)
        __syncthreads();
        if (tid == 0) {
            double r = wm[0];
            for (int w = 1; w < nw; ++w) r = dmax_nan(r, wm[w]);
            g.mismatch_out[t] = r != r ? __longlong_as_double(0x7ff0000000000000ll) : r;  // NaN reports as +inf
        }
    }
    if (tid == 0) {
        if (g.iters_out) g.iters_out[t] = conv ? it : -g.max_iter;
        if (conv) atomicAdd(&g.counters[kCntConverged], 1);
        atomicMax(&g.counters[5], it);
    }
}

template <int kBPT, bool kZip>
cudaError_t launch64_t(int threads, int64_t cols, size_t smem, const Tree64Args &g, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(f64_tree<kBPT, kZip>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && cols > 0) f64_tree<kBPT, kZip><<<(unsigned)cols, threads, smem, st>>>(g);
    return e;
}
template <int kBPT>
cudaError_t launch64(int threads, int64_t cols, size_t smem, const Tree64Args &g, cudaStream_t st) {
    return g.zip ? launch64_t<kBPT, true>(threads, cols, smem, g, st) : launch64_t<kBPT, false>(threads, cols, smem, g, st);
}

}  // namespace

size_t tree64_smem(int threads, int bpt) {
    const size_t ns = (size_t)threads * bpt;
    return 3 * ns * sizeof(double2) + (bpt < 8 ? ns * sizeof(float2) : 0) + 3 * ns * sizeof(short);
}

// Buses per thread: two up to 512 buses (256 threads), where a thread's chain of sums and products is what a
// column waits for; four up to 2,048, eight beyond (32 B of prefix sums and loads a slot).  In us, two against
// four: 33 buses x 16,384 columns 196 and 389, 64 buses 228 and 434, 129 x 8,000 333 and 497, 299 buses 572 and 699,
// 512 buses 865 and 872, 699 buses 1,487 and 1,287.  In FP64 throughout a thread's scans cost more than the chain,
// and two pay for the one warp of up to 64 buses only (us, two against four, behind a source of 12.66 kV): 64 buses
// x 16,384 columns 1,221 and 1,977, 96 x 8,192 1,344 and 1,127, 256 x 8,192 3,126 and 2,557, 512 x 4,096 3,589 and
// 2,776.  From 65 buses on a column that leaves the integers is therefore solved by a launch of its own at four.
int tree64_bpt(int n, bool fixed) {
    for (int b : {2, 4, 8})
        if ((b > 2 || n <= (fixed ? 512 : 64)) && tree_threads(n, b)) return b;
    return 0;
}

// Which columns take the integers.  A column's currents are rounded to 2^cur, an error of 0.29 2^cur (root mean
// square), and bus k's moves V_q by R_qk, the impedance that their paths share; impedances are rounded to
// 2^(z_e - 61), which moves V_q by 0.29 2^(z_e - 61) times the current of each branch on its path, at most
// 2^(cur + 62 - log2n) per bus below it.  Half a last place of V, 2^-54 pu, is allowed for both together, in root
// mean square; the sums of squares grow along a path.  The feeders of inputs.py are 21 times below that (1,000
// buses).  One load of thousands of times the others is not: such columns lost 3.3e-14 pu (1,000 pu beside 399
// ordinary loads) to 3.0e-11 (1e6 pu).
// Impedances above 2^8 times the upper quartile set neither z_e nor the limit, but a column with a current there goes
// to FP64 (the kernel looks).  Most are open switches, without a current: a stub of 1e6 pu cost the others 7.4e-13 pu
// when it set the place of all impedances, one of 1e12 pu 7.9e-7.  (Not the median: more than half of a feeder's
// branches may be couplers of next to no impedance, and its lines must not count as large.)
// cur_min is for the mismatch alone: a bus's branch currents are off by up to 2^-50 sum |y| (V is returned to 2^-52
// pu), and 2^61 integers hold that beside the currents.  Only branches of 1e-14 pu and less, or loads as small,
// come near (the sums wrapped there, and the mismatch was reported as 16 instead of 29).
// Returns false where no column of the feeder can take them: V is 61 bits below 2 pu, and none of it below 0.5.
bool fixed_limits(const Network &net, int &z_e, int &cur_max, int &cur_min) {
    const int n = net.n_pq;
    std::vector<int> e(n);
    for (int q = 0; q < n; ++q) frexp(std::max(std::fabs(net.dfs_z[2 * q]), std::fabs(net.dfs_z[2 * q + 1])), &e[q]);
    std::vector<int> by_size = e;
    std::nth_element(by_size.begin(), by_size.begin() + 3 * n / 4, by_size.end());
    const int cut = by_size[3 * n / 4] + 8;
    z_e = -2000;
    for (int v : e)
        if (v <= cut) z_e = std::max(z_e, v);
    int log2n = 0;
    while ((1 << log2n) < n) ++log2n;
    struct At {
        int end;              // of the subtree's positions
        double re, im, sum;  // path impedance; both sums of squares over 0.29^2 4^cur
        int q;
    };
    std::vector<double> y(n, 0.0);  // sum of |y| over the branches at a position
    std::vector<At> path;  // the ancestors of position q
    double worst = 0.0;
    for (int q = 0; q < n; ++q) {
        while (!path.empty() && path.back().end <= q) path.pop_back();
        const At up = path.empty() ? At{n, 0.0, 0.0, 0.0, -1} : path.back();
        At a = up;
        a.end = net.dfs_end[q];
        a.q = q;
        const double yq = 1.0 / std::hypot(net.dfs_z[2 * q], net.dfs_z[2 * q + 1]);
        y[q] += yq;
        if (up.q >= 0) y[up.q] += yq;
        if (e[q] <= cut) {
            const double size = a.end - q, zq = std::ldexp(size, z_e + 1 - log2n);
            a.re += net.dfs_z[2 * q];
            a.im += net.dfs_z[2 * q + 1];
            a.sum += size * ((a.re * a.re + a.im * a.im) - (up.re * up.re + up.im * up.im)) + zq * zq;
        }
        worst = std::max(worst, a.sum);
        path.push_back(a);
    }
    const double c = std::log2(std::ldexp(1.0, -54) / (0.29 * std::sqrt(worst)));
    cur_max = c >= 900.0 ? 900 : (c >= -900.0 ? (int)std::floor(c) : -10000);
    const double m = std::log2(*std::max_element(y.begin(), y.end())) - 111.0;
    cur_min = m <= 900.0 ? (int)std::ceil(std::max(m, -10000.0)) : 10000;
    return std::fabs(net.vs_re) < 2.0 && std::fabs(net.vs_im) < 2.0 && std::hypot(net.vs_re, net.vs_im) >= 0.5 &&
           cur_max > -10000;
}

tpf_status solve_tree64(tpf_handle *h, int64_t T, const void *S, void *V, int32_t *iters, double *mismatch,
                        const tpf_opts &o, cudaStream_t st) {
    const DeviceNet &d = h->dev;
    if (!d.radial || d.phases != 1 || d.t_threads == 0 || d.t_bpt == kTreeBigBPT || !d.t64.z) return TPF_EUNSUPPORTED;
    if (T > 0x7fffffff) return TPF_EUNSUPPORTED;  // one block per column
    if (tree64_smem(d.t64.threads, d.t64.bpt) > 227 * 1024) return TPF_EUNSUPPORTED;
    tpf_status rs = ensure_workspace(h, T, kWsState);  // counters
    if (rs != TPF_OK) return rs;
    Workspace &w = h->ws;
    if (cudaMemsetAsync(w.counters, 0, sizeof(int) * 8, st) != cudaSuccess) {
        cudaGetLastError();
        return TPF_ECUDA;
    }
    Tree64Args g{};
    g.n = d.n;
    g.max_iter = o.max_iter;
    g.tol2 = o.tol * o.tol;
    g.vs = make_double2(h->net.vs_re, h->net.vs_im);
    g.tol2_lo = (float)(ldexp(g.tol2, 2 * kFx) * (1.0 - 1e-5));
    g.tol2_hi = (float)(ldexp(g.tol2, 2 * kFx) * (1.0 + 1e-5));
    g.fixed = d.t64_fixed && o.tol < 1.0;
    while ((1 << g.log2n) < d.n) ++g.log2n;
    g.z_e = d.t64_z_e;
    g.cur_max = d.t64_cur_max;
    g.cur_min = d.t64_cur_min;
    if (g.fixed) g.vs_fx = make_longlong2(llrint(ldexp(g.vs.x, kFx)), llrint(ldexp(g.vs.y, kFx)));
    g.zip = d.zip64;
    g.S = static_cast<const double2 *>(S);
    g.V = static_cast<double2 *>(V);
    g.given = o.start != TPF_START_FLAT;
    g.iters_out = iters;
    g.mismatch_out = mismatch;
    g.counters = w.counters;
    KernelTimer timer(o.profile != 0, st);
    auto run = [&](const Tree64 &l, int64_t cols) {
        g.col = l.col;
        g.end = l.end;
        g.par = l.par;
        g.ecnt = l.ecnt;
        g.kidx = l.kidx;
        g.z = l.z;
        g.y = l.y;
        const size_t smem = tree64_smem(l.threads, l.bpt);
        timer.begin(KernelTimer::kGemm);
        cudaError_t e;
        switch (l.bpt) {
            case 2: e = launch64<2>(l.threads, cols, smem, g, st); break;
            case 4: e = launch64<4>(l.threads, cols, smem, g, st); break;
            case 8: e = launch64<8>(l.threads, cols, smem, g, st); break;
            default: return TPF_EUNSUPPORTED;
        }
        timer.end();
        if (e != cudaSuccess || cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(w.counters_host, w.counters, sizeof(int) * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            cudaGetLastError();
            return TPF_ECUDA;
        }
        return TPF_OK;
    };
    const bool leaves = d.t64.bpt < tree64_bpt(d.n, false);
    g.left = leaves ? w.flags : nullptr;
    auto plain = [&]() -> tpf_status {  // the layout of the columns that leave
        if (d.t64_plain.z) return TPF_OK;
        try {
            return layout_tree64(h->net, tree64_bpt(d.n, false), h->dev.t64_plain);
        } catch (const std::bad_alloc &) {
            return TPF_ENOMEM;
        }
    };
    int launches = 1;
    if (leaves && !g.fixed) {
        rs = plain();
        if (rs == TPF_OK) rs = run(d.t64_plain, T);
    } else {
        rs = run(d.t64, T);
        if (rs == TPF_OK && w.counters_host[kCntLeft] > 0) {
            rs = plain();
            g.list = w.flags;
            g.left = nullptr;
            g.fixed = 0;
            if (rs == TPF_OK) rs = run(d.t64_plain, w.counters_host[kCntLeft]);
            ++launches;
        }
    }
    if (rs != TPF_OK) return rs;
    const int64_t conv = w.counters_host[kCntConverged];
    h->stats.sweeps = w.counters_host[5];
    h->stats.kernel_launches = launches;
    h->stats.converged = conv;
    h->stats.gemm_ms = timer.total_ms(KernelTimer::kGemm);
    return conv == T ? TPF_OK : TPF_ENOCONV;
}

}  // namespace tpf
