// The per-sweep residual kernels of the mixed path (Eq. 1 residual, Algorithm 1 loop control), with
// their first-sweep and final-output variants.
//
// One block handles one column.  In a sweep it first takes the column's decision for the step the
// last sweep applied: stop at max |dV| <= tol (the per-column form of Algorithm 1's test), give up at
// max_iter or on a non-finite step, and anchor the column once its step is small.  It then forms rho_i:
//
//   before anchoring   rho = conj(S ./ V) + (Y v)         FP32, from the high words of V
//   anchoring sweep    V_ref <- fl(V), rho(V_ref) in double-float, stored
//   after anchoring    rho = rho(V_ref) + [rho(V_ref + d) - rho(V_ref)], the bracket in FP32
//
// with (Y v)_i = sum_j y_ij (V_i - V_j) over the branches at i (V_slack = v_s).  Finally rho is
// written as the fp16 B operand 2^e rho with the column's largest component in [2^13, 2^14) (e per
// column, exact to undo).
//
// The first sweep also splits S (and a given V_0) into the planes that later sweeps read; a flat start
// is not written anywhere (the product's epilogue knows it).  The final variant evaluates rho once
// more at the returned V (same formulas, no decision) and writes V as complex128, the iteration counts
// and the mismatch max_i |V_i| |rho_i| (= max_i |V_i conj((Y v)_i) + S_i|).
//
// mx_tree_residual serves radial feeders: rho_i = conj(S_i/V_i) - J_i + sum_{children c} J_c with the
// branch currents J_c = y_c (V_parent(c) - V_c); a bus leaves its admittance and voltage for its
// parent in shared memory, where the children of a bus are consecutive.  mx_residual takes any network
// over its neighbour lists.
#include "tpf_dd.cuh"

namespace tpf {

namespace {

struct FinalArgs {
    int64_t T;
    double2 *V_out;
    int32_t *iters_out;
    double *mismatch_out;
    int *tile_done;
};

enum Variant : int { kSweep = 0, kFirst = 1, kFinal = 2 };

// What a column does in this pass: its new flags, and whether it is anchored in it.
struct Decision {
    int f, it;
    bool anchor, blind, changed;  // blind: it was anchored at a given start before this pass
    float d;
};

// Every thread of a block decides alike from the column's state; commit() by one thread, once all have read.
template <int VAR>
__device__ __forceinline__ Decision decide(const PrologueArgs &a, const FinalArgs &fo, int64_t t) {
    Decision r{0, 0, false, false, false, 0.0f};
    if (VAR == kFinal) {
        // Every real column gets outputs; the residual uses the column's current mode.
        r.f = t < fo.T ? a.flags[t] | kActive : 0;
        return r;
    }
    if (VAR == kFirst) {
        r.f = t < a.T ? kActive : 0;
        if (r.f && a.given) {
            r.anchor = true;
            r.f |= kAnchored | kBlind;
        }
        return r;
    }
    r.f = a.flags[t];
    if (!(r.f & kActive)) return r;
    r.changed = true;
    r.blind = (r.f & kBlind) != 0;
    r.d = __uint_as_float(a.delta[t]);
    const float d = r.d, dp = __uint_as_float(a.dprev[t]);
    r.it = a.iters[t] + 1;
    // A column that stops keeps kAnchored: the final pass evaluates its residual at
    // V_ref + (V - V_ref) with the stored rho(V_ref).
    if (d <= a.tol) {
        r.f = kDone | (r.f & kAnchored);
    } else if (r.it >= a.max_iter || !(d < 1e30f)) {
        r.f &= kAnchored;
    } else if (!(r.f & kAnchored) || r.blind) {
        // Anchor once the step is small, or is predicted (geometric rate) to fall below
        // 3e-6 in the next sweep, while FP32 rounding (~1e-7) is still far below it.
        if (d < a.switch_tol || (dp > 0.0f && d * d < 3e-6f * dp)) {
            r.anchor = true;
            r.f = (r.f | kAnchored) & ~kBlind;
        }
    }
    return r;
}

template <int VAR>
__device__ __forceinline__ void commit(const PrologueArgs &a, int64_t t, const Decision &r) {
    if (VAR == kFirst) {
        a.flags[t] = r.f;
        a.iters[t] = 0;
        a.delta[t] = 0u;
        a.dprev[t] = 0u;
    } else if (VAR == kSweep && r.changed) {
        a.flags[t] = r.f;
        a.iters[t] = r.it;
        a.delta[t] = 0u;
        a.dprev[t] = __float_as_uint(r.d);
    }
}

__device__ __forceinline__ float2 hi_of(double2 s) { return make_float2(__double2float_rn(s.x), __double2float_rn(s.y)); }
__device__ __forceinline__ float2 lo_of(double2 s, float2 h) {
    return make_float2(__double2float_rn(s.x - (double)h.x), __double2float_rn(s.y - (double)h.y));
}
__device__ __forceinline__ c2 dd_of(double2 s) {
    const float2 h = hi_of(s), l = lo_of(s, h);
    return {{h.x, l.x}, {h.y, l.y}};
}

// Block maximum of non-negative values (a NaN is ignored, as fmaxf does); s_red holds one entry per warp.
__device__ __forceinline__ float block_max(float m, float *s_red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = m;
    __syncthreads();
    float mm = s_red[0];
    for (int w = 1; w < (int)blockDim.x / 32; ++w) mm = fmaxf(mm, s_red[w]);
    return mm;
}

// Exponent of a column's fp16 scale, and its bookkeeping.
__device__ __forceinline__ int scale_exp(float mm) {
    int e = 0;
    if (mm > 0.0f) {
        frexpf(mm, &e);
        e = 14 - e;
    }
    return e > 120 ? 120 : e;
}
__device__ __forceinline__ void publish_scale(const PrologueArgs &a, int64_t t, int e, bool anchor) {
    a.rexp[t] = e;
    atomicAdd(&a.tile_active[t / kTileN], 1);  // iterating columns of this 128-column tile
    if (anchor && a.counters[kCntPrecise] == 0) atomicExch(&a.counters[kCntPrecise], 1);
}
__device__ __forceinline__ void final_column(const PrologueArgs &a, const FinalArgs &fo, int64_t t, int f, float mm) {
    const bool done = (f & kDone) != 0;
    if (fo.mismatch_out) fo.mismatch_out[t] = (double)mm;
    if (fo.iters_out) fo.iters_out[t] = done ? a.iters[t] : -a.max_iter;
    if (done) atomicAdd(&fo.tile_done[t / kTileN], 1);
}
__device__ __forceinline__ float mismatch_of(float2 h, float2 l, float2 r) {
    const float vm = sqrtf((h.x + l.x) * (h.x + l.x) + (h.y + l.y) * (h.y + l.y));
    const float mv = vm * sqrtf(r.x * r.x + r.y * r.y);
    return mv != mv ? __int_as_float(0x7f800000) : mv;  // a NaN mismatch reports as +inf
}

// ------------------------------------------------------------------------------- radial feeders

// Per bus one 16-byte word: parent (0xffff: the slack) | place of the bus among all children << 16, 0, FP32
// admittance of the branch to the parent.  Per bus with children one 8-byte word, ordered by their number:
// bus | number of children << 16, place of the first child.  Half of the buses are leaves and a few have five
// children or more, so that with every bus looping over its own children a warp waits for its longest list
// five times as long as the average asks for.
//
// kP pairs of neighbouring buses per thread: 16-byte loads of the planes, half2 stores of the operand.
// Shared memory, per bus: V or d (8 B), rho (8 B), and what its parent needs of it (16 B).
//
// Bound by shared-memory and L1 wavefronts (1,900 a column of 999 buses) and the barriers between its
// phases; the bytes it must move take 48 us of an FP32 sweep of 16,384 such columns.  That sweep takes 167 us
// (203 with every bus looping over its own children, 196 before, with parents, admittances and child lists as
// five dependent loads a bus); an anchoring one, which is double-float arithmetic, 340 (420 before, over
// the neighbour lists of every bus); an anchored one 202.  Splitting S and writing the start used to be a pass
// of its own (32 B written a bus); the first sweep now does it in 179 us, and S's low words are taken from
// S again in the one sweep that needs them.  65,536 columns: 14.8 -> 12.1 ms for the whole solve.
template <int kP, int VAR>
__global__ void __launch_bounds__(kP >= 2 ? 512 : 64, kP >= 2 ? 2 : 1)
    mx_tree_residual(const __grid_constant__ PrologueArgs a, const __grid_constant__ FinalArgs fo) {
    extern __shared__ float4 rsm4[];
    float4 *const jdd = rsm4;                               // [n_pad] double-float branch currents (anchoring)
    float4 *const kid = rsm4;                               // [n_pad] admittance, V or d of every child
    float2 *const vb = reinterpret_cast<float2 *>(rsm4 + a.n_pad);  // [n_pad] V or d
    float2 *const rb = vb + a.n_pad;                                // [n_pad] rho
    __shared__ float s_red[16];
    const int tid = threadIdx.x, th = blockDim.x, n = a.n;
    const int64_t t = blockIdx.x, base = t * a.n_pad;
    const Decision dc = decide<VAR>(a, fo, t);
    const bool live = (dc.f & kActive) != 0, anchored = (dc.f & kAnchored) != 0;
    if (!live) {
        __syncthreads();
        if (tid == 0) commit<VAR>(a, t, dc);
        return;
    }
    // Buses i = 2 (tid + th k) + b, b = 0, 1.
    float4 v[kP], s[kP], d[kP];
    const double2 *const S64 = a.S64 + t * n;
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i = 2 * (tid + th * k);
        v[k] = make_float4(1.0f, 0.0f, 1.0f, 0.0f);
        s[k] = d[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (i >= n) continue;
        if (VAR == kFirst) {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                if (i + b >= n) continue;
                const float2 sh = hi_of(S64[i + b]);
                (b ? s[k].z : s[k].x) = sh.x;
                (b ? s[k].w : s[k].y) = sh.y;
                if (a.V0) {
                    const double2 v0 = a.V0[t * n + i + b];
                    const float2 vh = hi_of(v0), vl = a.given ? lo_of(v0, vh) : make_float2(0.0f, 0.0f);
                    (b ? v[k].z : v[k].x) = vh.x;
                    (b ? v[k].w : v[k].y) = vh.y;
                    (b ? d[k].z : d[k].x) = vl.x;
                    (b ? d[k].w : d[k].y) = vl.y;
                }
            }
            *reinterpret_cast<float4 *>(a.Shi + base + i) = s[k];
            if (a.V0) *reinterpret_cast<float4 *>(a.Vhi + base + i) = v[k];
        } else {
            v[k] = *reinterpret_cast<const float4 *>(a.Vhi + base + i);
            s[k] = *reinterpret_cast<const float4 *>(a.Shi + base + i);
            // Vlo exists from a column's first anchor on.
            if (anchored && (!dc.anchor || dc.blind)) d[k] = *reinterpret_cast<const float4 *>(a.Vlo + base + i);
        }
    }
    const bool rest = dc.anchor && (VAR == kFirst || dc.blind);
    if (dc.anchor) {
        // Re-base: V_ref <- fl(V), the remainder to d.
#pragma unroll
        for (int k = 0; k < kP; ++k) {
            const int i = 2 * (tid + th * k);
            const f2 x0 = two_sum(v[k].x, d[k].x), y0 = two_sum(v[k].y, d[k].y);
            const f2 x1 = two_sum(v[k].z, d[k].z), y1 = two_sum(v[k].w, d[k].w);
            v[k] = make_float4(x0.h, y0.h, x1.h, y1.h);
            d[k] = make_float4(x0.l, y0.l, x1.l, y1.l);
            if (i < n) {
                *reinterpret_cast<float4 *>(a.Vhi + base + i) = v[k];
                *reinterpret_cast<float4 *>(a.Vlo + base + i) = d[k];
                *reinterpret_cast<float4 *>(vb + i) = v[k];
            }
        }
        __syncthreads();
        // rho(V_ref) in double-float: the branch currents, then each bus.
#pragma unroll 1
        for (int i = tid; i < n; i += th) {
            const int4 w = a.topo[i];
            const int p = (short)(w.x & 0xffff), place = (short)((unsigned)w.x >> 16);
            if (place >= 0) {
                const float2 vi = vb[i], vp = vb[p];
                const float4 y = a.ypar4[i];
                const c2 j = c_mul(c2{{y.x, y.z}, {y.y, y.w}},
                                   c_sub(c2{{vp.x, 0.0f}, {vp.y, 0.0f}}, c2{{vi.x, 0.0f}, {vi.y, 0.0f}}));
                jdd[place] = make_float4(j.re.h, j.re.l, j.im.h, j.im.l);
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < n; i += th) {
            const int place = (short)((unsigned)a.topo[i].x >> 16);
            const float2 vi = vb[i];
            const c2 vd = {{vi.x, 0.0f}, {vi.y, 0.0f}};
            c2 j;
            if (place >= 0) {
                const float4 q = jdd[place];
                j = c2{{q.x, q.y}, {q.z, q.w}};
            } else {
                const float4 y = a.ypar4[i];
                j = c_mul(c2{{y.x, y.z}, {y.y, y.w}}, c_sub(a.vs_dd, vd));
            }
            const c2 acc = c_sub(load_current_dd(dd_of(S64[i]), vd), j);
            a.RefHi[base + i] = make_float2(acc.re.h, acc.im.h);
            a.RefLo[base + i] = make_float2(acc.re.l, acc.im.l);
        }
        __syncthreads();
#pragma unroll 1
        for (int k = tid; k < a.n_inner; k += th) {
            const int2 w = a.inner[k];
            const int i = w.x & 0xffff, cnt = (int)((unsigned)w.x >> 16);
            const float2 h = a.RefHi[base + i], l = a.RefLo[base + i];
            c2 acc = {{h.x, l.x}, {h.y, l.y}};
            for (int e = w.y; e < w.y + cnt; ++e) {
                const float4 q = jdd[e];
                acc = c_add(acc, c2{{q.x, q.y}, {q.z, q.w}});
            }
            a.RefHi[base + i] = make_float2(acc.re.h, acc.im.h);
            a.RefLo[base + i] = make_float2(acc.re.l, acc.im.l);
        }
        // A re-based column with a remainder: its correction over the neighbour lists.
        if (rest)
            for (int i = tid; i < n; i += th)
                rb[i] = residual_corr(i, a.Vhi + base, a.Vlo + base, a.Shi + base, a.row_ptr, a.nbr, a.y);
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i = 2 * (tid + th * k);
        if (i < n) *reinterpret_cast<float4 *>(vb + i) = anchored ? d[k] : v[k];
    }
    __syncthreads();
    if (tid == 0) commit<VAR>(a, t, dc);
    // Load currents (or their change) less the bus's own branch current, then its children's.
    if (!rest) {
#pragma unroll
        for (int k = 0; k < kP; ++k) {
            float4 r4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            const int i0 = 2 * (tid + th * k);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int i = i0 + b;
                if (i < n) {
                    const int4 w = a.topo[i];
                    const int p = (short)(w.x & 0xffff), place = (short)((unsigned)w.x >> 16);
                    const float2 y = make_float2(__int_as_float(w.z), __int_as_float(w.w));
                    const float2 vi = b ? make_float2(v[k].z, v[k].w) : make_float2(v[k].x, v[k].y);
                    const float2 di = b ? make_float2(d[k].z, d[k].w) : make_float2(d[k].x, d[k].y);
                    const float2 si = b ? make_float2(s[k].z, s[k].w) : make_float2(s[k].x, s[k].y);
                    const float2 x = anchored ? di : vi;
                    const float2 vp = p >= 0 ? vb[p] : (anchored ? make_float2(0.0f, 0.0f) : a.vs_f);
                    if (place >= 0) kid[place] = make_float4(y.x, y.y, x.x, x.y);
                    const float dr = vp.x - x.x, dm = vp.y - x.y;
                    const float2 c = anchored ? delta_current(vi, di, si) : load_current_f32(vi, si);
                    const float2 r = make_float2(c.x - (y.x * dr - y.y * dm), c.y - (y.x * dm + y.y * dr));  // - J_i
                    (b ? r4.z : r4.x) = r.x;
                    (b ? r4.w : r4.y) = r.y;
                }
            }
            if (i0 < a.n_pad) *reinterpret_cast<float4 *>(rb + i0) = r4;
        }
        __syncthreads();
        for (int k = tid; k < a.n_inner; k += th) {
            const int2 w = a.inner[k];
            const int i = w.x & 0xffff, cnt = (int)((unsigned)w.x >> 16);
            const float2 x = vb[i];
            float2 r = rb[i];
            for (int e = w.y; e < w.y + cnt; ++e) {  // + J_c = y_c (V_i - V_c) for the children c
                const float4 q = kid[e];
                const float dr = x.x - q.z, dm = x.y - q.w;
                r.x += q.x * dr - q.y * dm;
                r.y += q.x * dm + q.y * dr;
            }
            rb[i] = r;
        }
        __syncthreads();
    }
    float4 acc[kP];
    float m = 0.0f;
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i0 = 2 * (tid + th * k);
        float4 r4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (i0 < n) {
            r4 = *reinterpret_cast<const float4 *>(rb + i0);
            if (i0 + 1 >= n) r4.z = r4.w = 0.0f;
            if (anchored) {
                const float4 h = *reinterpret_cast<const float4 *>(a.RefHi + base + i0);
                const float4 l = *reinterpret_cast<const float4 *>(a.RefLo + base + i0);
                const f2 x0 = two_sum(h.x, r4.x), y0 = two_sum(h.y, r4.y);
                r4.x = x0.h + (x0.l + l.x);
                r4.y = y0.h + (y0.l + l.y);
                if (i0 + 1 < n) {
                    const f2 x1 = two_sum(h.z, r4.z), y1 = two_sum(h.w, r4.w);
                    r4.z = x1.h + (x1.l + l.z);
                    r4.w = y1.h + (y1.l + l.w);
                }
            }
        }
        acc[k] = r4;
        if (VAR == kFinal) {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                if (i0 + b >= n) continue;
                const float2 vh = b ? make_float2(v[k].z, v[k].w) : make_float2(v[k].x, v[k].y);
                const float2 vl = b ? make_float2(d[k].z, d[k].w) : make_float2(d[k].x, d[k].y);
                fo.V_out[t * n + i0 + b] = make_double2((double)vh.x + (double)vl.x, (double)vh.y + (double)vl.y);
                m = fmaxf(m, mismatch_of(vh, vl, b ? make_float2(r4.z, r4.w) : make_float2(r4.x, r4.y)));
            }
        } else {
            m = fmaxf(m, fmaxf(fmaxf(fabsf(r4.x), fabsf(r4.y)), fmaxf(fabsf(r4.z), fabsf(r4.w))));
        }
    }
    const float mm = block_max(m, s_red);
    if (VAR == kFinal) {
        if (tid == 0) final_column(a, fo, t, dc.f, mm);
        return;
    }
    const int e = scale_exp(mm);
    const float sc = pow2f(e);
#pragma unroll
    for (int k = 0; k < kP; ++k) {
        const int i = 2 * (tid + th * k);
        if (i < a.n_pad) {
            *reinterpret_cast<__half2 *>(a.Rr + base + i) = __floats2half2_rn(acc[k].x * sc, acc[k].z * sc);
            *reinterpret_cast<__half2 *>(a.Ri + base + i) = __floats2half2_rn(acc[k].y * sc, acc[k].w * sc);
        }
    }
    if (tid == 0) publish_scale(a, t, e, dc.anchor);
}

// ------------------------------------------------------------------------------- any network

constexpr int kResThreads = 128;

template <int VAR>
__global__ void __launch_bounds__(kResThreads)
    mx_residual(const __grid_constant__ PrologueArgs a, const __grid_constant__ FinalArgs fo) {
    extern __shared__ float4 rsm4[];
    float2 *const rb = reinterpret_cast<float2 *>(rsm4);  // [n_pad] rho
    __shared__ float s_red[kResThreads / 32];
    const int tid = threadIdx.x, n = a.n;
    const int64_t t = blockIdx.x, base = t * a.n_pad;
    const Decision dc = decide<VAR>(a, fo, t);
    __syncthreads();
    if (tid == 0) commit<VAR>(a, t, dc);
    if (!(dc.f & kActive)) return;
    const bool anchored = (dc.f & kAnchored) != 0;
    float2 *const vh = a.Vhi + base, *const vl = a.Vlo + base;
    float2 *const sh = a.Shi + base;
    const double2 *const S64 = a.S64 + t * n;
    if (VAR == kFirst) {
        for (int i = tid; i < n; i += kResThreads) {
            sh[i] = hi_of(S64[i]);
            float2 h = make_float2(1.0f, 0.0f);
            if (a.V0) {
                const double2 v0 = a.V0[t * n + i];
                h = hi_of(v0);
                if (a.given) vl[i] = lo_of(v0, h);
            }
            vh[i] = h;
        }
        __syncthreads();
    }
    if (dc.anchor) {
        // Re-base V, then rho(V_ref) in double-float.
        for (int i = tid; i < n; i += kResThreads) {
            const float2 h = vh[i], l = VAR == kFirst || dc.blind ? vl[i] : make_float2(0.0f, 0.0f);
            const f2 re = two_sum(h.x, l.x), im = two_sum(h.y, l.y);
            vh[i] = make_float2(re.h, im.h);
            vl[i] = make_float2(re.l, im.l);
        }
        __syncthreads();
        for (int i = tid; i < n; i += kResThreads) {
            const c2 ref = residual_dd(i, vh, dd_of(S64[i]), a.row_ptr, a.nbr, a.y, a.vs_dd);
            a.RefHi[base + i] = make_float2(ref.re.h, ref.im.h);
            a.RefLo[base + i] = make_float2(ref.re.l, ref.im.l);
        }
    }
    float m = 0.0f;
    for (int i = tid; i < n; i += kResThreads) {
        float2 r;
        if (anchored) {
            const float2 cr = residual_corr(i, vh, vl, sh, a.row_ptr, a.nbr, a.y);
            const float2 h = a.RefHi[base + i], l = a.RefLo[base + i];
            const f2 sr = two_sum(h.x, cr.x), si = two_sum(h.y, cr.y);
            r = make_float2(sr.h + (sr.l + l.x), si.h + (si.l + l.y));
        } else {
            r = residual_f32(i, vh, sh, a.row_ptr, a.nbr, a.y, a.vs_f);
        }
        if (VAR == kFinal) {
            const float2 h = vh[i], l = anchored ? vl[i] : make_float2(0.0f, 0.0f);
            fo.V_out[t * n + i] = make_double2((double)h.x + (double)l.x, (double)h.y + (double)l.y);
            m = fmaxf(m, mismatch_of(h, l, r));
        } else {
            rb[i] = r;
            m = fmaxf(m, fmaxf(fabsf(r.x), fabsf(r.y)));
        }
    }
    const float mm = block_max(m, s_red);
    if (VAR == kFinal) {
        if (tid == 0) final_column(a, fo, t, dc.f, mm);
        return;
    }
    const int e = scale_exp(mm);
    const float sc = pow2f(e);
    for (int i = tid; i < a.n_pad; i += kResThreads) {
        const float2 r = i < n ? rb[i] : make_float2(0.0f, 0.0f);
        a.Rr[base + i] = __float2half_rn(r.x * sc);
        a.Ri[base + i] = __float2half_rn(r.y * sc);
    }
    if (tid == 0) publish_scale(a, t, e, dc.anchor);
}

template <int VAR>
tpf_status launch(const PrologueArgs &a, const FinalArgs &fo, int64_t cols, cudaStream_t st) {
    if (cols <= 0) return TPF_OK;
    if (a.topo) {
        // Two pairs of buses per thread (64 registers, 32 warps per SM), one for up to 128 buses.
        const int th = a.n_pad <= 128 ? 64 : a.n_pad / 4;
        const size_t smem = (size_t)a.n_pad * (sizeof(float4) + 2 * sizeof(float2));  // at most 64 KB
        static std::atomic<uint64_t> attr{0};
        if (!once_per_device(attr, [] {
                return cudaFuncSetAttribute(mx_tree_residual<2, VAR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            2048 * (int)(sizeof(float4) + 2 * sizeof(float2))) == cudaSuccess;
            }))
            return TPF_ECUDA;
        if (a.n_pad <= 128)
            mx_tree_residual<1, VAR><<<(unsigned)cols, th, smem, st>>>(a, fo);
        else
            mx_tree_residual<2, VAR><<<(unsigned)cols, th, smem, st>>>(a, fo);
    } else {
        mx_residual<VAR><<<(unsigned)cols, kResThreads, (size_t)a.n_pad * sizeof(float2), st>>>(a, fo);
    }
    if (cudaGetLastError() != cudaSuccess) return TPF_ECUDA;
    return TPF_OK;
}

}  // namespace

tpf_status launch_residual(const PrologueArgs &a, cudaStream_t st) {
    return a.sweep == 0 ? launch<kFirst>(a, FinalArgs{}, a.cols, st) : launch<kSweep>(a, FinalArgs{}, a.cols, st);
}

tpf_status launch_final(const PrologueArgs &a, int64_t T, void *V_out, int32_t *iters_out, double *mismatch_out,
                        int *tile_done, cudaStream_t st) {
    FinalArgs fo{T, (double2 *)V_out, iters_out, mismatch_out, tile_done};
    return launch<kFinal>(a, fo, T, st);
}

}  // namespace tpf
