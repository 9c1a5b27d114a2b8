// Training kernels of the learned warm start: one step is features, a product per layer forward and
// backward whose epilogue does everything elementwise, all weight gradients in one launch, and Adam.
//
// A step of a 200-bus network (1,024 columns, 3 x 256 units) is 0.9 GFLOP, a microsecond of the tensor
// pipe: what it costs is launches, one after the other, and passes over activations that fit the L2.  So
//   - bias, GELU and its derivative, the loss gradient with its targets, the BF16 operands in both
//     layouts and the bias sums are formed in the product's epilogue, where the value is in a register;
//   - tiles are 128 units x 32 columns, so that 64 to 128 SMs share a layer's epilogue (the erf dominates
//     it) instead of 16 to 32;
//   - transposed copies are written 32 bytes a thread from the epilogue (a thread holds 16 consecutive
//     columns of its unit) or through shared memory, not 2 bytes apart by B;
//   - the layers' weight gradients need nothing from one another: one launch, which sums the bias gradients
//     beside them.  (Every sum keeps the order it would have in a launch of its own, so that weights do
//     not depend on how the work is cut; splitting the batch as well was no faster.);
//   - every kernel starts under its predecessor (programmatic dependent launch) and waits for it before it
//     touches memory.
// That step went from 31 launches and 202 us to 10 launches and 54 us, 5 to 7 us each and one after the other;
// a 34-bus network of one layer takes 32 us, 1,000 buses and 3 x 256 units 95.
#include <cuda_bf16.h>

#include <algorithm>

#include "tpf_gemm.h"
#include "tpf_mlp_train.h"
#include "tpf_tc.cuh"

using bf16 = __nv_bfloat16;

namespace tpf {

namespace {

using namespace tc;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// The launch before this one has finished and its results are visible; the next one may start.
__device__ __forceinline__ void after_predecessor() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
}

template <class K, class... A>
tpf_status launch_pdl(K kernel, dim3 grid, unsigned threads, size_t smem, cudaStream_t st, const A &...args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    if (cudaLaunchKernelEx(&c, kernel, args...) != cudaSuccess) {
        cudaGetLastError();
        return TPF_ECUDA;
    }
    return TPF_OK;
}

constexpr uint32_t kABytes = kTileM * kChunkK * 2;
constexpr int kEpiThreads = 256, kThreads = 64 + kEpiThreads;
constexpr int kWgrad = 3;  // beside LayerKind

template <int kN>
struct Ring {
    static constexpr uint32_t kStage = kABytes + kN * kChunkK * 2;
    static constexpr int kStages = 8;
    static constexpr size_t kSmem = 1024 + kStages * kStage + 256;
};

__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

__device__ __forceinline__ const CUtensorMap *map_a(const LayerArgs &g, int) { return &g.a; }
__device__ __forceinline__ const CUtensorMap *map_b(const LayerArgs &g, int) { return &g.b; }
__device__ __forceinline__ const CUtensorMap *map_a(const WgradArgs &g, int p) { return &g.a[p]; }
__device__ __forceinline__ const CUtensorMap *map_b(const WgradArgs &g, int p) { return &g.b[p]; }

// One 128 x kN tile of D = A B^T per CTA.  Warp 0 issues the TMA loads, warp 1 the MMAs, warps 2-9 the
// epilogue (two per TMEM lane quarter, half of the columns each).  Every wait is bounded; on expiry the
// error flag is set, nothing is written, and the CTA leaves once its copies and MMAs have ended.
template <int kN, int KIND, class Args>
__global__ void __launch_bounds__(kThreads, 1) mlp_gemm(const __grid_constant__ Args g) {
    using R = Ring<kN>;
    constexpr uint32_t kCols = kN < 32 ? 32 : kN;
    extern __shared__ uint8_t smem_raw[];
    __shared__ float s_loss[8];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + R::kStages * R::kStage);
    uint64_t *empty = full + R::kStages, *done = empty + R::kStages;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *abort_flag = (int *)(tmem_slot + 1);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < R::kStages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        mbar_init(smem_u32(done), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    after_predecessor();
    const uint32_t tmem = *tmem_slot;
    volatile int *vabort = abort_flag;

    const int chunks = g.chunks;
    int p = 0, m0, n0;
    if constexpr (KIND == kWgrad) {
        while (p + 1 < g.layers && (int)blockIdx.x >= g.first[p + 1]) ++p;
        const int tile = (int)blockIdx.x - g.first[p];
        m0 = (tile % g.m_tiles[p]) * kTileM;
        n0 = (tile / g.m_tiles[p]) * kN;
    } else {
        m0 = (int)blockIdx.y * kTileM;
        n0 = (int)blockIdx.x * kN;
    }

    if (warp == 0) {
        if (lane == 0) {
            const uint32_t sbase = smem_u32(smem);
            int k = 0;
            for (; k < chunks; ++k) {
                const int slot = k % R::kStages;
                if (!mbar_wait(smem_u32(&empty[slot]), ((uint32_t)(k / R::kStages) & 1) ^ 1)) {
                    *vabort = 1;
                    atomicExch(g.err, 1);
                    break;
                }
                const uint32_t st = sbase + slot * R::kStage, bar = smem_u32(&full[slot]);
                mbar_expect_tx(bar, R::kStage);
                tma_load_2d(st, map_a(g, p), bar, k * kChunkK, m0);
                tma_load_2d(st + kABytes, map_b(g, p), bar, k * kChunkK, n0);
            }
            if (*vabort)
                for (int q = k - 1; q >= 0 && q >= k - R::kStages; --q)
                    mbar_wait(smem_u32(&full[q % R::kStages]), (uint32_t)(q / R::kStages) & 1);
        }
    } else if (warp == 1) {
        const uint32_t sbase = smem_u32(smem), id = idesc_f16(kTileM, kN, 0, 1);
        const bool lead = elect_one();
        uint32_t slot = 0, phase = 0;
        for (int c = 0; c < chunks; ++c) {
            if (!mbar_wait(smem_u32(&full[slot]), phase)) {
                if (lead) {
                    *vabort = 1;
                    atomicExch(g.err, 1);
                }
                break;
            }
            tc_fence_after();
            const uint64_t da = sw128_desc(sbase + slot * R::kStage);
            if (lead) {
#pragma unroll
                for (int kk = 0; kk < kChunkK / 16; ++kk)
                    umma_f16(tmem, da + kk * 2, da + kABytes / 16 + kk * 2, id, c != 0 || kk != 0);
                umma_commit(smem_u32(&empty[slot]));
            }
            __syncwarp();
            if (++slot == R::kStages) slot = 0, phase ^= 1;
        }
        if (lead) umma_commit(smem_u32(done));
        __syncwarp();
        mbar_wait(smem_u32(done), 0);
    } else {
        const int quarter = warp & 3, half = (warp - 2) >> 2, row = quarter * 32 + lane, m = m0 + row;
        const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
        // What the epilogue reads of device memory comes while the product runs (after the first store the
        // compiler must keep loads and stores in order, one round trip per column: 6.5 us instead of 13.6 for
        // a backward launch, 9.9 instead of 17.5 for the output layer's).
        constexpr int kC = kN / 2;  // columns of this thread
        [[maybe_unused]] float pre[kC];
        [[maybe_unused]] float bm = 0.0f;
        if constexpr (KIND == kWgrad) {
            // The bias gradients of this tile's 128 units, shared out among the tiles beside it: one warp
            // per unit over the contiguous row of dZ^T.
            const int tiles = (g.first[p + 1] - g.first[p]) / g.m_tiles[p], B = g.chunks * kChunkK;
            for (int u = n0 / kN + tiles * (warp - 2); u < kTileM; u += tiles * (kEpiThreads / 32)) {
                const bf16 *const z = g.zT[p] + (int64_t)(m0 + u) * B;
                float s = 0.0f;
                for (int b = lane; b < B; b += 32) s += __bfloat162float(z[b]);
                for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
                if (lane == 0) g.gb[p][m0 + u] = s;
            }
        } else {
            const int b0 = n0 + half * kC;
            const bool live = m < g.real;
#pragma unroll
            for (int q = 0; q < kC; ++q) pre[q] = 0.0f;
            if (KIND != kBackward && live) bm = g.bias[m];
            if (KIND == kBackward && live)
#pragma unroll
                for (int q = 0; q < kC; ++q) pre[q] = g.Z[(int64_t)(b0 + q) * g.M + m];
            if (KIND == kOutput && live) {
                // Normalised target: (Re V - 1, Im V), z-scored.
                const float tm = g.mean[m], td = g.sd[m];
                const double *const tv = reinterpret_cast<const double *>(g.V + (int64_t)b0 * g.n) +
                                         (m < g.n ? 2 * m : 2 * (m - g.n) + 1);
                const double one = m < g.n ? 1.0 : 0.0;
                double raw[kC];
#pragma unroll
                for (int q = 0; q < kC; ++q) raw[q] = tv[(int64_t)q * 2 * g.n];
#pragma unroll
                for (int q = 0; q < kC; ++q) {
                    const float f = (float)(raw[q] - one);
                    pre[q] = td > 0.0f ? (f - tm) / td : 0.0f;
                }
            }
        }
        bool ok = mbar_wait(smem_u32(done), 0);
        if (!ok) atomicExch(g.err, 1);
        ok = ok && !*vabort;
        tc_fence_after();
        if constexpr (KIND == kWgrad) {
            float *const D = g.D[p];
            const int ld = g.ld[p];
            uint32_t x[kC];
            tmem_ld16(tmem + lane_off + half * kC, x);
            tmem_wait_ld();
            if (ok)
#pragma unroll
                for (int q = 0; q < kC; ++q) D[(int64_t)(n0 + half * kC + q) * ld + m] = __uint_as_float(x[q]);
        } else {
            static_assert(kC == 16, "a thread's columns fill two 16-byte stores of the transposed operand");
            uint32_t x[kC];
            tmem_ld16(tmem + lane_off + half * kC, x);
            tmem_wait_ld();
            const int b0 = n0 + half * kC;
            const bool live = m < g.real;
            float sq = 0.0f;
            uint32_t packed[kC / 2];
#pragma unroll
            for (int q = 0; q < kC; ++q) {
                const int64_t k = (int64_t)(b0 + q) * g.M + m;
                const float d = __uint_as_float(x[q]);
                float r = 0.0f;
                if (KIND == kHidden) {
                    const float z = live ? d + bm : 0.0f;
                    if (ok) g.Z[k] = z;
                    r = live ? gelu(z) : 0.0f;
                } else if (KIND == kOutput) {
                    if (live) {
                        const float e = (d + bm) - pre[q];
                        sq += e * e;
                        r = 2.0f * e / ((float)g.B * (float)g.real);
                    }
                } else if (live) {
                    r = d * gelu_grad(pre[q]);
                }
                const bf16 v = __float2bfloat16_rn(r);
                if (ok) g.o[k] = v;
                const uint32_t w = __bfloat16_as_ushort(v);
                packed[q / 2] = q & 1 ? packed[q / 2] | w << 16 : w;
            }
            if (ok) {
                uint4 *const t = reinterpret_cast<uint4 *>(g.oT + (int64_t)m * g.B + b0);
                t[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                t[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
            }
            if (KIND == kOutput) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                if (lane == 0) s_loss[warp - 2] = sq;
                epi_bar();
            }
            if (KIND == kOutput && tid == 64 && ok) {  // one atomic per tile: same-address atomics queue up
                sq = 0.0f;
                for (int k = 0; k < 8; ++k) sq += s_loss[k];
                atomicAdd(g.loss, (double)sq / ((double)g.B * (double)g.real));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

constexpr int kAdamThreads = 256;  // 32 x 8, for 32 x 32 tiles of a weight matrix

// A weight's step for gradient d, and its new moments.  The roundings are written out, so that every build
// takes the same steps (Adam turns a rounding of a near-zero gradient into one of full size).
__device__ __forceinline__ float adam_step(const AdamArgs &g, float d, float m, float v, float &mm, float &vv) {
    mm = __fmaf_rn(1.0f - g.b1, d, __fmul_rn(g.b1, m));
    vv = __fmaf_rn(__fmul_rn(1.0f - g.b2, d), d, __fmul_rn(g.b2, v));
    return g.lr * (mm / g.c1) / (sqrtf(vv / g.c2) + g.eps);
}

// One 32 x 32 tile of one layer's weights: the gradient comes [k][o], the weights are [o][k], and W^T leaves
// [k][o]; both turns go through shared memory.
__global__ void __launch_bounds__(kAdamThreads) mlp_adam(const __grid_constant__ AdamArgs g) {
    __shared__ float sg[32][33];
    __shared__ unsigned short sw[32][34];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    int i = 0;
    while (i + 1 < g.L && (int)blockIdx.x >= g.l[i + 1].tile0) ++i;
    const AdamLayer &a = g.l[i];
    const int tile = (int)blockIdx.x - a.tile0, kt = a.Pi / 32;
    const int o0 = tile / kt * 32, k0 = tile % kt * 32;
    after_predecessor();
    // All loads first: 4 weights per thread with their moments and gradients in flight together (loads
    // after the first store would wait behind it: 15.1 us per launch instead of 10.2 from a cold cache, a
    // 200-bus network of 3 x 256 units).
    float w[4], mo[4], ve[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t idx = (int64_t)(o0 + ty + 8 * r) * a.Pi + k0 + tx;
        w[r] = a.W[idx];
        mo[r] = ve[r] = 0.0f;
        if (g.update) {
            mo[r] = a.m[idx];
            ve[r] = a.v[idx];
        }
    }
    if (g.update) {
#pragma unroll
        for (int r = 0; r < 4; ++r) sg[ty + 8 * r][tx] = a.gWT[(int64_t)(k0 + ty + 8 * r) * a.Po + o0 + tx];
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int o = o0 + ty + 8 * r, k = k0 + tx;
        const int64_t idx = (int64_t)o * a.Pi + k;
        if (g.update && o < a.ro && k < a.ri) {
            const float d = sg[tx][ty + 8 * r];
            float mm, vv;
            w[r] -= adam_step(g, d, mo[r], ve[r], mm, vv);
            a.m[idx] = mm;
            a.v[idx] = vv;
            a.W[idx] = w[r];
        }
        const bf16 wb = __float2bfloat16_rn(w[r]);
        a.Wb[idx] = wb;
        sw[ty + 8 * r][tx] = __bfloat16_as_ushort(wb);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 32; r += 8)
        a.WTb[(int64_t)(k0 + ty + r) * a.Po + o0 + tx] = __ushort_as_bfloat16(sw[tx][ty + r]);
    const int o = o0 + tx;
    if (g.update && k0 == 0 && ty == 0 && o < a.ro) {
        const float d = a.gb[o];
        float mm, vv;
        a.b[o] -= adam_step(g, d, a.mb[o], a.vb[o], mm, vv);
        a.mb[o] = mm;
        a.vb[o] = vv;
    }
}

// Tiles of 32 buses (or padding features) x 32 columns.
__global__ void __launch_bounds__(256)
    mlp_features(const double2 *__restrict__ S, int B, int n, int P, int bus_tiles, const float *__restrict__ mean,
                 const float *__restrict__ sd, bf16 *X, bf16 *XT, int *err, double *loss) {
    __shared__ unsigned short s[2][32][34];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b0 = (int)blockIdx.x * 32, part = (int)blockIdx.y;
    after_predecessor();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        *err = 0;
        *loss = 0.0;
    }
    if (part >= bus_tiles) {  // padding features 2n .. P - 1
        const int j0 = (part - bus_tiles) * 32;
        for (int r = ty; r < 32; r += 8) {
            const bf16 z = __float2bfloat16_rn(0.0f);
            if (2 * n + j0 + tx < P) X[(int64_t)(b0 + r) * P + 2 * n + j0 + tx] = z;
            if (2 * n + j0 + r < P) XT[(int64_t)(2 * n + j0 + r) * B + b0 + tx] = z;
        }
        return;
    }
    const int j0 = part * 32, j = j0 + tx;
    if (j < n) {
        const float mr = mean[j], dr = sd[j], mi = mean[n + j], di = sd[n + j];
        double2 in[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) in[q] = S[(int64_t)(b0 + ty + 8 * q) * n + j];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = ty + 8 * q;
            const double2 v = in[q];
            const float xr = dr > 0.0f ? ((float)v.x - mr) / dr : 0.0f;
            const float xi = di > 0.0f ? ((float)v.y - mi) / di : 0.0f;
            const bf16 vr = __float2bfloat16_rn(xr), vi = __float2bfloat16_rn(xi);
            X[(int64_t)(b0 + r) * P + j] = vr;
            X[(int64_t)(b0 + r) * P + n + j] = vi;
            s[0][r][tx] = __bfloat16_as_ushort(vr);
            s[1][r][tx] = __bfloat16_as_ushort(vi);
        }
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8)
        if (j0 + r < n) {
            XT[(int64_t)(j0 + r) * B + b0 + tx] = __ushort_as_bfloat16(s[0][tx][r]);
            XT[(int64_t)(n + j0 + r) * B + b0 + tx] = __ushort_as_bfloat16(s[1][tx][r]);
        }
}

__global__ void mlp_flat(const __grid_constant__ FlatArgs g) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= g.total) return;
    int i = 0;
    while (i + 1 < g.L && idx >= g.l[i + 1].off) ++i;
    const FlatLayer &a = g.l[i];
    const int64_t e = idx - a.off, w = (int64_t)a.ro * a.ri;
    if (e < w) {
        const int o = (int)(e / a.ri), k = (int)(e % a.ri);
        float *const at = a.W + (int64_t)o * a.Pi + k;
        if (g.mode == 0) g.flat[idx] = *at;
        if (g.mode == 1) *at = g.flat[idx];
        if (g.mode == 2) g.flat[idx] = a.gWT[(int64_t)k * a.Po + o];
    } else {
        const int o = (int)(e - w);
        if (g.mode == 0) g.flat[idx] = a.b[o];
        if (g.mode == 1) a.b[o] = g.flat[idx];
        if (g.mode == 2) g.flat[idx] = a.gb[o];
    }
}

template <class K>
bool big_smem(K kernel, size_t bytes) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

}  // namespace

tpf_status launch_layer(int kind, const LayerArgs &g, cudaStream_t st) {
    using R = Ring<kTrainN>;
    static std::atomic<uint64_t> attr{0};
    if (!once_per_device(attr, [] {
            return big_smem(mlp_gemm<kTrainN, kHidden, LayerArgs>, R::kSmem) &&
                   big_smem(mlp_gemm<kTrainN, kOutput, LayerArgs>, R::kSmem) &&
                   big_smem(mlp_gemm<kTrainN, kBackward, LayerArgs>, R::kSmem);
        }))
        return TPF_ECUDA;
    const dim3 grid((unsigned)(g.B / kTrainN), (unsigned)(g.M / kTileM));  // y is limited to 65,535
    if (kind == kHidden) return launch_pdl(mlp_gemm<kTrainN, kHidden, LayerArgs>, grid, kThreads, R::kSmem, st, g);
    if (kind == kOutput) return launch_pdl(mlp_gemm<kTrainN, kOutput, LayerArgs>, grid, kThreads, R::kSmem, st, g);
    return launch_pdl(mlp_gemm<kTrainN, kBackward, LayerArgs>, grid, kThreads, R::kSmem, st, g);
}

tpf_status launch_wgrad(const WgradArgs &g, cudaStream_t st) {
    using R = Ring<kTrainN>;
    static std::atomic<uint64_t> attr{0};
    if (!once_per_device(attr, [] { return big_smem(mlp_gemm<kTrainN, kWgrad, WgradArgs>, R::kSmem); })) return TPF_ECUDA;
    return launch_pdl(mlp_gemm<kTrainN, kWgrad, WgradArgs>, dim3((unsigned)g.first[g.layers]), kThreads, R::kSmem, st, g);
}

tpf_status launch_adam(AdamArgs &g, cudaStream_t st) {
    int tiles = 0;
    for (int i = 0; i < g.L; ++i) {
        g.l[i].tile0 = tiles;
        tiles += g.l[i].Po / 32 * (g.l[i].Pi / 32);
    }
    return launch_pdl(mlp_adam, dim3((unsigned)tiles), kAdamThreads, 0, st, g);
}

tpf_status launch_train_features(const double2 *S, int B, int n, int P, const float *mean, const float *sd, bf16 *X,
                                 bf16 *XT, int *err, double *loss, cudaStream_t st) {
    const int bus_tiles = (n + 31) / 32, pad_tiles = (P - 2 * n + 31) / 32;
    return launch_pdl(mlp_features, dim3((unsigned)(B / 32), (unsigned)(bus_tiles + pad_tiles)), 256, 0, st, S, B, n, P,
                      bus_tiles, mean, sd, X, XT, err, loss);
}

tpf_status launch_flat(const FlatArgs &g, cudaStream_t st) {
    mlp_flat<<<(unsigned)((g.total + 255) / 256), 256, 0, st>>>(g);
    if (cudaGetLastError() != cudaSuccess) return TPF_ECUDA;
    return TPF_OK;
}

}  // namespace tpf
