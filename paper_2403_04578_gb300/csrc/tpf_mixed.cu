// Mixed-precision solve path: fp16 tensor-core sweeps (tcgen05, FP32 accumulation in TMEM) in
// residual form, with V and the residual carried in double-float.
//
// The fixed point of Eq. 2 / Eq. 12, V = K conj(S ./ V) + W with K = -Y_dd^{-1} and
// W = K Y_ds v_s, is the zero of the residual
//
//     rho(V) = (Y_dd V + Y_ds v_s) + conj(S ./ V)      (Eq. 1 with i_d = conj(S ./ V))
//
// and the fixed-point step is exactly  V_{k+1} = V_k + K rho(V_k)  (expand K rho with
// K Y_dd = -I).  Written this way the dense product only carries the correction: the fp16 error
// of K and rho scales with |rho| -> 0 instead of with |V|, so the iterates converge to the
// double-precision solution while the O(n^2) work per column runs on fp16 tensor cores.
// rho itself is O(n) per column: for a shunt-free network (Y V)_i = sum_j y_ij (V_i - V_j) over
// the branches at bus i (V_slack = v_s).
//
// Per sweep:  mx_tree_residual / mx_residual  (tpf_residual.cu, one block per column) decides
//                          convergence from the last step, forms rho (FP32 far from convergence,
//                          then against a double-float anchor), scales it by a per-column power of
//                          two and writes the fp16 B operand;
//             tc_gemm      (tpf_gemm.cu, persistent, warp-specialised) computes K rho with four
//                          real-plane MMAs per K step (Re = Kr rr - Ki ri, Im = Kr ri + Ki rr)
//                          over 128 x 128 tiles; its epilogue adds the update to V and folds
//                          max |dV| per column.
// This file holds the host loop of a solve.
#include <cuda_fp16.h>

#include <cstdlib>
#include <cstring>

#include "tpf_dd.cuh"
#include "tpf_gemm.h"

namespace tpf {

#define TPF_CK(call)                  \
    do {                              \
        if ((call) != cudaSuccess) {  \
            cudaGetLastError();       \
            return TPF_ECUDA;         \
        }                             \
    } while (0)

tpf_status selftest_gemm(int M, int N, int K, const void *Ar, const void *Ai, const void *Br, const void *Bi, float *Dr,
                         float *Di, cudaStream_t st, uint64_t wait_ns, int withhold_loads) {
    GemmMaps maps;
    if (!make_gemm_maps(&maps, Ar, Ai, M, K, Br, Bi, N)) return TPF_ECUDA;
    int *err = nullptr;
    TPF_CK(cudaMalloc(&err, sizeof(int)));
    TPF_CK(cudaMemsetAsync(err, 0, sizeof(int), st));
    GemmEpi ep{};
    ep.mode = 0;
    ep.cplx = 1;
    ep.err = err;
    ep.Dr = Dr;
    ep.Di = Di;
    ep.ldD = M;
    ep.wait_ns = wait_ns;
    ep.withhold_loads = withhold_loads;
    tpf_status rs = launch_gemm(maps, M / kTileM, N / kTileN, K / kChunkK, ep, st);
    int herr = 0;
    cudaError_t e = cudaSuccess;
    if (rs == TPF_OK) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (rs == TPF_OK && e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(err);
    if (rs != TPF_OK) return rs;
    if (e != cudaSuccess) {
        cudaGetLastError();
        return TPF_ECUDA;
    }
    return herr ? TPF_ETIMEOUT : TPF_OK;
}

namespace {
struct StreamEvent {
    cudaEvent_t e = nullptr;
    StreamEvent() {
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            e = nullptr;
        }
    }
    ~StreamEvent() {
        if (e) cudaEventDestroy(e);
    }
};
}  // namespace

tpf_status solve_mixed(tpf_handle *h, int64_t T, const void *S, void *V, int32_t *iters, double *mismatch,
                       const tpf_opts &o, cudaStream_t st) {
    const int n = h->dev.n, n_pad = h->dev.n_pad;
    if (n_pad > 2048) return TPF_EUNSUPPORTED;
    if (h->dev.zip64) return TPF_EUNSUPPORTED;    // ZIP loads: sparse formulation or FP64 path
    if (h->dev.phases > 1) return TPF_EUNSUPPORTED;  // polyphase: sparse formulation or FP64 path
    tpf_status rs = ensure_dense(h);
    if (rs != TPF_OK) return rs;
    rs = ensure_workspace(h, T, kWsMixed);
    if (rs != TPF_OK) return rs;
    Workspace &w = h->ws;
    const int64_t cols = round_up(T, kTileN);
    GemmMaps maps;
    if (!make_gemm_maps(&maps, h->dev.Kr16, h->dev.Ki16, n_pad, n_pad, w.Rr16, w.Ri16, cols)) return TPF_ECUDA;
    int64_t launches = 0, gemm_cols = 0;
    KernelTimer timer(o.profile != 0, st);
    TPF_CK(cudaMemsetAsync(w.counters, 0, sizeof(int) * 8, st));

    PrologueArgs pa{};
    pa.cols = cols;
    pa.T = T;
    pa.S64 = (const double2 *)S;
    pa.V0 = o.start != TPF_START_FLAT ? (const double2 *)V : nullptr;
    pa.n = n;
    pa.n_pad = n_pad;
    pa.max_iter = o.max_iter;
    pa.tol = (float)o.tol;
    pa.switch_tol = (float)o.switch_tol;
    pa.vs_f = make_float2((float)h->net.vs_re, (float)h->net.vs_im);
    {
        float rh = (float)h->net.vs_re, ih = (float)h->net.vs_im;
        pa.vs_dd = c2{{rh, (float)(h->net.vs_re - (double)rh)}, {ih, (float)(h->net.vs_im - (double)ih)}};
    }
    pa.Vhi = w.Vhi;
    pa.Vlo = w.Vlo;
    pa.Shi = w.Shi;
    pa.RefHi = w.RefHi;
    pa.RefLo = w.RefLo;
    pa.dprev = w.dprev;
    pa.given = o.start == TPF_START_GIVEN;
    pa.topo = h->dev.r_topo;
    pa.ypar4 = h->dev.r_ypar;
    pa.inner = h->dev.r_inner;
    pa.n_inner = h->dev.r_n_inner;
    pa.row_ptr = h->dev.row_ptr;
    pa.nbr = h->dev.nbr;
    pa.y = h->dev.y2f;
    pa.flags = w.flags;
    pa.iters = w.iters;
    pa.rexp = w.rexp;
    pa.tile_active = w.tile_active;
    pa.counters = w.counters;
    pa.delta = w.delta_bits;
    pa.Rr = (__half *)w.Rr16;
    pa.Ri = (__half *)w.Ri16;

    GemmEpi ep{};
    ep.mode = 1;
    ep.cplx = 1;
    ep.err = w.counters + kCntError;
    ep.n = n;
    ep.n_pad = n_pad;
    ep.k_exp = h->dev.k_exp;
    ep.flags = w.flags;
    ep.rexp = w.rexp;
    ep.tile_active = w.tile_active;
    ep.Vhi = w.Vhi;
    ep.Vlo = w.Vlo;
    ep.delta = w.delta_bits;

    int sweeps = 0, precise_sweeps = 0;
    const int64_t n_tiles = cols / kTileN;
    int *const tile_host = w.tile_host;
    StreamEvent seen;
    if (!seen.e) return TPF_ECUDA;
    for (int s = 0; s <= o.max_iter; ++s) {
        TPF_CK(cudaMemsetAsync(w.tile_active, 0, sizeof(int) * n_tiles, st));
        TPF_CK(cudaMemsetAsync(w.counters, 0, sizeof(int) * 2, st));  // active, precise
        pa.sweep = s;
        timer.begin(KernelTimer::kResidual);
        rs = launch_residual(pa, st);
        timer.end();
        if (rs != TPF_OK) return rs;
        ++launches;
        // The product is queued before the host has seen which tiles iterate (it skips the others), so that
        // the host's round trip runs beside it.
        TPF_CK(cudaMemcpyAsync(w.counters_host, w.counters, sizeof(int) * 8, cudaMemcpyDeviceToHost, st));
        TPF_CK(cudaMemcpyAsync(tile_host, w.tile_active, sizeof(int) * n_tiles, cudaMemcpyDeviceToHost, st));
        TPF_CK(cudaEventRecord(seen.e, st));
        ep.v_flat = s == 0 && !pa.V0;
        timer.begin(KernelTimer::kGemm);
        rs = launch_gemm(maps, n_pad / kTileM, cols / kTileN, n_pad / kChunkK, ep, st);
        timer.end();
        if (rs != TPF_OK) return rs;
        TPF_CK(cudaGetLastError());
        TPF_CK(cudaEventSynchronize(seen.e));
        if (w.counters_host[kCntError]) break;
        int64_t active = 0;
        for (int64_t k = 0; k < n_tiles; ++k) active += tile_host[k];
        if (active == 0) break;
        if (w.counters_host[kCntPrecise] > 0) ++precise_sweeps;
        gemm_cols += active;
        ++launches;
        ++sweeps;
    }
    TPF_CK(cudaMemsetAsync(w.tile_active, 0, sizeof(int) * n_tiles, st));  // reused: converged per tile
    timer.begin(KernelTimer::kOther);
    rs = launch_final(pa, T, V, iters, mismatch, w.tile_active, st);
    timer.end();
    if (rs != TPF_OK) return rs;
    ++launches;
    TPF_CK(cudaMemcpyAsync(w.counters_host, w.counters, sizeof(int) * 8, cudaMemcpyDeviceToHost, st));
    TPF_CK(cudaMemcpyAsync(tile_host, w.tile_active, sizeof(int) * n_tiles, cudaMemcpyDeviceToHost, st));
    TPF_CK(cudaStreamSynchronize(st));
    int64_t converged = 0;
    for (int64_t k = 0; k < n_tiles; ++k) converged += tile_host[k];
    h->stats.sweeps = sweeps;
    h->stats.precise_sweeps = precise_sweeps;
    h->stats.kernel_launches = launches;
    h->stats.converged = converged;
    h->stats.gemm_launches = sweeps;
    h->stats.gemm_columns = gemm_cols;
    h->stats.gemm_ms = timer.total_ms(KernelTimer::kGemm);
    h->stats.residual_ms = timer.total_ms(KernelTimer::kResidual);
    h->stats.other_ms = timer.total_ms(KernelTimer::kOther);
    if (w.counters_host[kCntError]) return TPF_ETIMEOUT;
    return h->stats.converged == T ? TPF_OK : TPF_ENOCONV;
}

}  // namespace tpf
