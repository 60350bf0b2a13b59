// ace_tables.cu — the offline expert tables of ACE on the GPU, from bf16
// weights in device memory.
//
// GSP (Algorithm 2; Eqs. gsp_up_path, gsp_gate_path, gsp_geometric_mean,
// gsp_layer_normalization). With G = Gamma W_gate, U = Gamma W_up (d x m) and
// W_down (m x d):
//   a_up = ||U||_F ||G W_down||_F,   a_gate = ||G||_F ||U W_down||_F,
//   a~_e = sqrt(a_up a_gate),        A^GSP(e) = a~_e / (mean_j a~_j + eps).
// ||Gamma W_p W_down||_F^2 = sum_i gamma_i^2 sum_j (sum_r W_p[i,r] W_down[r,j])^2
// is a d x d x m GEMM per expert and path whose d x d product never leaves
// the SM: k_gsp_frob runs it on the tensor cores (tcgen05.mma, bf16 operands
// exactly as stored, fp32 accumulators in TMEM) and its epilogue squares the
// accumulators, sums them per row, scales row i by gamma_i^2 (so Gamma is
// applied exactly, not rounded into a bf16 operand) and writes one fp64
// partial per (tile, warp). The nn.Linear layouts give W_p[i, r] =
// w_p[e][r][i] (the A operand, M-major: TMA loads 64 x 64 boxes of the weights
// as stored and the instruction descriptor says so) and W_down[r, j] =
// w_down[e][j][r] (the B operand, K-major as stored). The weights are read in
// place: repacking them into K-major tiles first took 0.53 ms of kernels and
// most of a 1.2 GB scratch allocation's 1 ms at d = 2048, N = 128, m = 768 (a
// call took 2.71 ms, 1.49 without, 1.25 with the RCR chain overlapped).
//
// RCR (Algorithm 3; Eqs. rcr_centered_router, rcr_direction_prototype,
// rcr_raw_amplification, rcr_layer_normalization): centred router rows
// w~_e = w_e - mean_j w_j, prototype q_e = w~_e / (RMS(w~_e) + eps) (rho = 1),
// a~_e = ||f_e(q_e)||_2 / (||q_e||_2 + eps), A^RCR(e) = a~_e / (mean a~ + eps),
// f_e(x) = (SiLU(x W_gate) * (x W_up)) W_down; q_e is scaled by gamma first
// when rcr_apply_gamma is set. One input row per expert makes this a GEMV
// over all expert weights: fp32 on the CUDA cores, bound by HBM.
//
// Every reduction is summed in a fixed order (per-thread, per-warp, per-tile
// partials combined by one thread per expert), so the tables are the same
// bits on every run.
#include <cuda.h>
#include <math.h>
#include <string.h>

#include <string>

#include "ace_device.cuh"
#include "ace_internal.h"
#include "ace_tc.cuh"

namespace ace {
namespace {

constexpr int kTabThreads = 192;
constexpr int kTabStages = 4;
constexpr int kTabA = 128 * kBK * 2;            // 16 KB: 128 rows i x 64 r
constexpr int kTabB = 256 * kBK * 2;            // 32 KB: 256 rows j x 64 r
constexpr int kTabStage = kTabA + kTabB;
constexpr int kTabSmem = kTabStages * kTabStage + 1024 + 256;

// Fixed-order block sum of one double per thread (blockDim.x = 256).
__device__ __forceinline__ double block_sum_256(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < 8; ++w) t += sh[w];
    __syncthreads();
    return t;   // valid in thread 0
}

// ---------------------------------------------------------------- GSP: Frobenius norms of the products

struct FrobParams {
    CUtensorMap tm_a[2];         // gate, up as [N * m rows r, d columns i]: boxes of 64 r x 64 i
    CUtensorMap tm_b;            // w_down as [N * d rows j, m columns r]: boxes of 256 j x 64 r
    const float* gamma2;         // [d] gamma_i^2 (exact in fp32 for bf16 gamma)
    double* partial;             // [N][2][d/128 * d/256][4]
    int n_e, d, m;
    int* err;
};

struct FrobItem {
    int el, path, tj, ti;
};

// Items in the order (expert, path, tj, ti): CTAs working at the same time
// share one expert's operands (L2-resident) and mostly the same B tile.
__device__ __forceinline__ FrobItem frob_item(const FrobParams& p, int item) {
    const int ti_n = p.d / 128, tj_n = p.d / 256;
    FrobItem it;
    it.ti = item % ti_n;
    item /= ti_n;
    it.tj = item % tj_n;
    item /= tj_n;
    it.path = item & 1;
    it.el = item >> 1;
    return it;
}

// Shared-memory descriptor of an M-major operand tile in the 128-byte swizzle:
// 64-element M blocks of 128-byte rows, one row per K index; 8 rows (1024
// bytes) to the next group of K indices, 64 rows (8 KB) to the next M block.
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);          // start address
    d |= (uint64_t)(8192 >> 4) << 16;               // leading byte offset: next 64-element M block
    d |= (uint64_t)(1024 >> 4) << 32;               // stride byte offset: next 8 K indices
    d |= (uint64_t)1 << 46;                         // descriptor version
    d |= (uint64_t)2 << 61;                         // 128-byte swizzle
    return d;
}

// 128 x 256 output tiles of C = A B^T, K = m, persistent over the items;
// warp 0 loads (TMA boxes of the weights as stored), warp 1 issues the MMAs,
// warps 2..5 reduce the accumulators. Two 256-column accumulator buffers.
// Bound by the tensor pipe under the power limit.
__global__ void __launch_bounds__(kTabThreads, 1) k_gsp_frob(const __grid_constant__ FrobParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kTabStages * kTabStage);
    uint64_t* empty = full + kTabStages;
    uint64_t* acc_full = empty + kTabStages;
    uint64_t* acc_empty = acc_full + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kTabStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&acc_full[a], 1);
            mbar_init(&acc_empty[a], 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int ti_n = p.d / 128, tj_n = p.d / 256, kblocks = p.m / kBK;
    const int n_items = p.n_e * 2 * ti_n * tj_n;

    if (warp == 0) {
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            long long issued = 0;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const FrobItem it = frob_item(p, item);
                const int a_row = it.el * p.m, b_row = it.el * p.d + it.tj * 256;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!mbar_wait(&empty[stage], phase ^ 1u, p.err) || *abort_flag) { ok = false; break; }
                    unsigned char* sa = smem + stage * kTabStage;
                    mbar_expect_tx(&full[stage], kTabStage);
                    tma_load_2d(sa, &p.tm_a[it.path], &full[stage], it.ti * 128, a_row + kb * kBK);
                    tma_load_2d(sa + kTabA / 2, &p.tm_a[it.path], &full[stage], it.ti * 128 + 64, a_row + kb * kBK);
                    tma_load_2d(sa + kTabA, &p.tm_b, &full[stage], kb * kBK, b_row);
                    ++issued;
                    if (++stage == kTabStages) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) {
                *abort_flag = 1;
                // let the copies already issued land before the CTA exits
                for (long long f = issued - 1; f >= 0 && f >= issued - kTabStages; --f)
                    if (!mbar_wait(&full[f % kTabStages], (uint32_t)((f / kTabStages) & 1), p.err)) break;
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(128, 256) | (1u << 15);   // A is M-major
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                if (!mbar_wait(&acc_empty[acc], acc_phase ^ 1u, p.err) || *abort_flag) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 256);
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!mbar_wait(&full[stage], phase, p.err) || *abort_flag) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a_addr = smem_u32(smem + stage * kTabStage);
                    const uint32_t b_addr = a_addr + kTabA;
                    // a K step of 16: 16 rows of A (2 KB), 32 bytes of B (addresses in units of 16 bytes)
                    const uint64_t ad = smem_desc_sw128_mn(a_addr), bd = smem_desc_sw128(b_addr);
#pragma unroll
                    for (int kk = 0; kk < kBK / kUmmaK; ++kk)
                        mma_bf16(d_tmem, ad + 128 * kk, bd + 2 * kk, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                    mma_commit(&empty[stage]);
                    if (++stage == kTabStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                mma_commit(&acc_full[acc]);
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            if (!ok) *abort_flag = 1;
        }
    } else {
        // warps 2..5: TMEM lanes 32 * (warp % 4) + lane hold rows i of the tile
        const int quad = warp & 3;
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
            if (!mbar_wait_warp(&acc_full[acc], acc_phase, p.err, abort_flag)) break;
            tc_fence_after();
            const FrobItem it = frob_item(p, item);
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 256);
            double row = 0.0;
#pragma unroll 1
            for (int c = 0; c < 16; c += 2) {
                uint32_t r0[16], r1[16];
                tmem_ld16(taddr + (uint32_t)(c * 16), r0);
                tmem_ld16(taddr + (uint32_t)(c * 16 + 16), r1);
                tmem_ld_wait();
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float v0 = __uint_as_float(r0[j]), v1 = __uint_as_float(r1[j]);
                    s0 = fmaf(v0, v0, s0);
                    s1 = fmaf(v1, v1, s1);
                }
                row += (double)s0;
                row += (double)s1;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[acc]);
            const int i = it.ti * 128 + quad * 32 + lane;
            row *= (double)p.gamma2[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) row += __shfl_xor_sync(0xffffffffu, row, o);
            if (lane == 0) {
                const size_t tile = (size_t)it.tj * ti_n + it.ti;
                p.partial[(((size_t)it.el * 2 + it.path) * ti_n * tj_n + tile) * 4 + quad] = row;
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u));
}

// ---------------------------------------------------------------- RCR

// Column means of the router weight: mean_i = (1/N) sum_e w_r[e, i].
__global__ void __launch_bounds__(256) k_rcr_colmean(const __nv_bfloat16* __restrict__ w_r, int n, int d,
                                                     double* __restrict__ mean) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= d) return;
    double s = 0.0;
    for (int e = 0; e < n; ++e) s += (double)__bfloat162float(w_r[(long long)e * d + i]);
    mean[i] = s / (double)n;
}

// Prototype of expert e (block e): x_e = q_e (* gamma), and ||q_e||_2.
__global__ void __launch_bounds__(256) k_rcr_proto(const __nv_bfloat16* __restrict__ w_r,
                                                   const double* __restrict__ mean,
                                                   const __nv_bfloat16* __restrict__ gamma, int apply_gamma, int d,
                                                   double eps, float* __restrict__ x, double* __restrict__ qnorm) {
    __shared__ double sh[8];
    __shared__ double s_inv;
    const long long e = blockIdx.x;
    const __nv_bfloat16* w = w_r + e * d;
    double ss = 0.0;
    for (int i = threadIdx.x; i < d; i += 256) {
        const double c = (double)__bfloat162float(w[i]) - mean[i];
        ss += c * c;
    }
    const double tot = block_sum_256(ss, sh);
    if (threadIdx.x == 0) s_inv = 1.0 / (sqrt(tot / (double)d) + eps);
    __syncthreads();
    const double inv = s_inv;
    double qq = 0.0;
    for (int i = threadIdx.x; i < d; i += 256) {
        const double q = ((double)__bfloat162float(w[i]) - mean[i]) * inv;
        qq += q * q;
        x[e * d + i] = (float)(apply_gamma ? q * (double)__bfloat162float(gamma[i]) : q);
    }
    const double qt = block_sum_256(qq, sh);
    if (threadIdx.x == 0) qnorm[e] = sqrt(qt);
}

// act_e[j] = SiLU(x_e . W_gate[e, j]) * (x_e . W_up[e, j]); grid (m / 64, N),
// each warp 8 rows j, the input row and gamma^2 in shared memory. The rows
// pass here anyway, so the block also sums its share of ||Gamma W_gate||_F^2
// and ||Gamma W_up||_F^2: gamma_i^2 w^2 over 8 elements in fp32, their sums in
// fp64 in a fixed order (a float pair would overflow where fp64 does not); one
// partial per block and path in norms[path][e][block].
__global__ void __launch_bounds__(256) k_rcr_gateup(const float* __restrict__ x, const float* __restrict__ gamma2,
                                                    const __nv_bfloat16* __restrict__ w_gate,
                                                    const __nv_bfloat16* __restrict__ w_up, int d, int m,
                                                    float* __restrict__ act, double* __restrict__ norms) {
    extern __shared__ __align__(16) float xs[];
    __shared__ double sh[8];
    float* gs = xs + d;
    const long long e = blockIdx.y;
    for (int i = threadIdx.x; i < d; i += 256) {
        xs[i] = x[e * d + i];
        gs[i] = gamma2[i];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cv = d / 8;
    double ng = 0.0, nu = 0.0;
    for (int t = 0; t < 8; ++t) {
        const int j = blockIdx.x * 64 + warp * 8 + t;
        const uint4* g = reinterpret_cast<const uint4*>(w_gate + (e * m + j) * (long long)d);
        const uint4* u = reinterpret_cast<const uint4*>(w_up + (e * m + j) * (long long)d);
        float sg = 0.f, su = 0.f;
#pragma unroll 4
        for (int q = lane; q < cv; q += 32) {
            float fg[8], fu[8];
            Vec16<__nv_bfloat16>::to_float(ld_stream(g + q), fg);
            Vec16<__nv_bfloat16>::to_float(ld_stream(u + q), fu);
            float qg = 0.f, qu = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                sg = fmaf(fg[k], xs[q * 8 + k], sg);
                su = fmaf(fu[k], xs[q * 8 + k], su);
                qg = fmaf(gs[q * 8 + k] * fg[k], fg[k], qg);
                qu = fmaf(gs[q * 8 + k] * fu[k], fu[k], qu);
            }
            ng += (double)qg;
            nu += (double)qu;
        }
        sg = warp_sum(sg);
        su = warp_sum(su);
        if (lane == 0) act[e * m + j] = sg / (1.0f + expf(-sg)) * su;
    }
    const double tg = block_sum_256(ng, sh), tu = block_sum_256(nu, sh);
    if (threadIdx.x == 0) {
        norms[e * gridDim.x + blockIdx.x] = tg;
        norms[((long long)gridDim.y + e) * gridDim.x + blockIdx.x] = tu;
    }
}

// y_e[c] = act_e . W_down[e, c]; grid (d / 64, N); each block writes the sum
// of its 64 y_c^2 (fixed order) to part[e][block].
__global__ void __launch_bounds__(256) k_rcr_down(const float* __restrict__ act, const __nv_bfloat16* __restrict__ w_down,
                                                  int d, int m, double* __restrict__ part) {
    extern __shared__ __align__(16) float as[];
    __shared__ double sh[8];
    const long long e = blockIdx.y;
    for (int j = threadIdx.x; j < m; j += 256) as[j] = act[e * m + j];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cv = m / 8;
    double y2 = 0.0;
    for (int t = 0; t < 8; ++t) {
        const int c = blockIdx.x * 64 + warp * 8 + t;
        const uint4* w = reinterpret_cast<const uint4*>(w_down + (e * d + c) * (long long)m);
        float s = 0.f;
        for (int q = lane; q < cv; q += 32) {
            float f[8];
            Vec16<__nv_bfloat16>::to_float(ld_stream(w + q), f);
#pragma unroll
            for (int k = 0; k < 8; ++k) s = fmaf(f[k], as[q * 8 + k], s);
        }
        s = warp_sum(s);
        y2 += (double)s * (double)s;   // identical in every lane
    }
    if (lane == 0) sh[warp] = y2;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += sh[w];
        part[e * gridDim.x + blockIdx.x] = t;
    }
}

// ---------------------------------------------------------------- final normalisation

// Block e sums expert e's partials, each list in a fixed order (strided
// per-thread sums, then block_sum_256): raw[e] = {||G W_down||^2,
// ||U W_down||^2, ||G||^2, ||U||^2, ||f_e(q_e)||^2}.
__global__ void __launch_bounds__(256) k_tables_reduce(const double* __restrict__ frob, int frob_per,
                                                       const double* __restrict__ norms, int norm_per,
                                                       const double* __restrict__ rcr_part, int rcr_per, int n,
                                                       double* __restrict__ raw) {
    __shared__ double sh[8];
    const size_t e = blockIdx.x;
    const double* lists[5] = {frob + (e * 2 + 0) * frob_per, frob + (e * 2 + 1) * frob_per, norms + e * norm_per,
                              norms + ((size_t)n + e) * norm_per, rcr_part + e * rcr_per};
    const int lens[5] = {frob_per, frob_per, norm_per, norm_per, rcr_per};
    for (int l = 0; l < 5; ++l) {
        double v = 0.0;
        for (int i = threadIdx.x; i < lens[l]; i += 256) v += lists[l][i];
        const double t = block_sum_256(v, sh);
        if (threadIdx.x == 0) raw[e * 5 + l] = t;
    }
}

// One block of 1024 threads: the per-expert scores and the layer normalisation.
__global__ void __launch_bounds__(1024) k_tables_final(const double* __restrict__ raw,
                                                       const double* __restrict__ qnorm, int n, double eps,
                                                       float* __restrict__ gsp_out, float* __restrict__ rcr_out) {
    __shared__ double sg[1024], sr[1024];
    const int e = threadIdx.x;
    double ag = 0.0, ar = 0.0;
    if (e < n) {
        const double* r = raw + (size_t)e * 5;
        const double a_up = sqrt(r[3]) * sqrt(r[0]);      // ||U||_F ||G W_down||_F   (Eq. gsp_up_path)
        const double a_gate = sqrt(r[2]) * sqrt(r[1]);    // ||G||_F ||U W_down||_F   (Eq. gsp_gate_path)
        ag = sqrt(a_up * a_gate);                         // Eq. gsp_geometric_mean
        ar = sqrt(r[4]) / (qnorm[e] + eps);               // Eq. rcr_raw_amplification
    }
    sg[e] = ag;
    sr[e] = ar;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (e < o) {
            sg[e] += sg[e + o];
            sr[e] += sr[e + o];
        }
        __syncthreads();
    }
    if (e < n) {
        gsp_out[e] = (float)(ag / (sg[0] / n + eps));   // Eq. gsp_layer_normalization
        rcr_out[e] = (float)(ar / (sr[0] / n + eps));   // Eq. rcr_layer_normalization
    }
}

__global__ void k_gamma2(const __nv_bfloat16* __restrict__ g, float* __restrict__ g2, int d) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < d) {
        const float v = __bfloat162float(g[i]);
        g2[i] = v * v;
    }
}

ace_status tab_fail(ace_status st, const std::string& m) {
    set_last_error(m.c_str());
    return st;
}

}  // namespace
}  // namespace ace

extern "C" ace_status ace_offline_tables_device(int d, int N, int m, const void* gamma, const void* router_w,
                                                const void* w_gate, const void* w_up, const void* w_down, double eps,
                                                int rcr_apply_gamma, size_t tile_budget, float* gsp_out,
                                                float* rcr_out, void* stream) {
    using namespace ace;
    if (!gamma || !router_w || !w_gate || !w_up || !w_down || !gsp_out || !rcr_out)
        return tab_fail(ACE_ERR_INVALID_ARG, "ace_offline_tables_device: NULL pointer");
    if (d <= 0 || N <= 0 || m <= 0) return tab_fail(ACE_ERR_INVALID_ARG, "ace_offline_tables_device: sizes must be > 0");
    if (N > kMaxExperts) return tab_fail(ACE_ERR_UNSUPPORTED, "ace_offline_tables_device: N > 1024");
    if (d % 256 || m % 64 || d > 16384)
        return tab_fail(ACE_ERR_UNSUPPORTED,
                        "ace_offline_tables_device: d must be a multiple of 256 (<= 16384), m a multiple of 64");
    if (!(eps >= 0.0)) return tab_fail(ACE_ERR_INVALID_ARG, "ace_offline_tables_device: eps must be >= 0");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return tab_fail(ACE_ERR_CUDA, std::string("ace_offline_tables_device: ") + cudaGetErrorString(e));

    (void)tile_budget;          // the weights are read in place
    const int ti_n = d / 128, tj_n = d / 256, frob_per = ti_n * tj_n * 4, rcr_per = d / 64;
    const int norm_per = m / 64;                 // k_rcr_gateup blocks per expert

    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
    const size_t o_frob = take((size_t)N * 2 * frob_per * 8), o_norm = take((size_t)N * 2 * norm_per * 8);
    const size_t o_raw = take((size_t)N * 5 * 8);
    const size_t o_mean = take((size_t)d * 8), o_x = take((size_t)N * d * 4), o_qn = take((size_t)N * 8);
    const size_t o_act = take((size_t)N * m * 4), o_rcr = take((size_t)N * rcr_per * 8);
    const size_t o_g2 = take((size_t)d * 4), o_out = take((size_t)(2 * N + 1) * 4);   // results, then the error word
    unsigned char* base = nullptr;
    e = cudaMalloc(&base, off);
    if (e != cudaSuccess) return tab_fail(ACE_ERR_OOM, "ace_offline_tables_device: scratch allocation failed");
    ace_status st = ACE_OK;
    const __nv_bfloat16* wg = static_cast<const __nv_bfloat16*>(w_gate);
    const __nv_bfloat16* wu = static_cast<const __nv_bfloat16*>(w_up);
    const __nv_bfloat16* wd = static_cast<const __nv_bfloat16*>(w_down);
    float* g2 = reinterpret_cast<float*>(base + o_g2);
    float* out = reinterpret_cast<float*>(base + o_out);
    int* err = reinterpret_cast<int*>(out + 2 * N);
    float host[2 * kMaxExperts + 1];
    int herr = 0;
    // the RCR chain (HBM-bound) runs beside the GSP GEMM (tensor-bound) on a stream of the call
    cudaStream_t s2 = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
#define TAB_CK(call)                                                                                      \
    do {                                                                                                  \
        cudaError_t e_ = (call);                                                                          \
        if (e_ != cudaSuccess) {                                                                          \
            st = tab_fail(ACE_ERR_CUDA, std::string("ace_offline_tables_device: ") + cudaGetErrorString(e_)); \
            goto done;                                                                                    \
        }                                                                                                 \
    } while (0)
    FrobParams p{};
    TAB_CK(cudaFuncSetAttribute(k_gsp_frob, cudaFuncAttributeMaxDynamicSharedMemorySize, kTabSmem));
    TAB_CK(ace::raise_smem_limit(k_rcr_gateup, d * 8));
    TAB_CK(ace::raise_smem_limit(k_rcr_down, m * 4));
    // one shared-memory split for all of them: blocks of the RCR chain fit beside the GEMM's CTAs
    TAB_CK(ace::prefer_shared(k_gsp_frob));
    TAB_CK(ace::prefer_shared(k_rcr_colmean));
    TAB_CK(ace::prefer_shared(k_rcr_proto));
    TAB_CK(ace::prefer_shared(k_rcr_gateup));
    TAB_CK(ace::prefer_shared(k_rcr_down));
    TAB_CK(cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking));
    TAB_CK(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
    TAB_CK(cudaEventCreateWithFlags(&join, cudaEventDisableTiming));
    TAB_CK(make_tensor_map(&p.tm_a[0], wg, (uint64_t)N * m, d, 64, true));
    TAB_CK(make_tensor_map(&p.tm_a[1], wu, (uint64_t)N * m, d, 64, true));
    TAB_CK(make_tensor_map(&p.tm_b, wd, (uint64_t)N * d, m, 256, true));
    TAB_CK(cudaMemsetAsync(err, 0, 4, s));
    k_gamma2<<<(d + 255) / 256, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(gamma), g2, d);
    TAB_CK(cudaGetLastError());
    TAB_CK(cudaEventRecord(fork, s));
    TAB_CK(cudaStreamWaitEvent(s2, fork, 0));
    p.gamma2 = g2;
    p.partial = reinterpret_cast<double*>(base + o_frob);
    p.n_e = N;
    p.d = d;
    p.m = m;
    p.err = err;
    {
        const long long items = (long long)N * 2 * ti_n * tj_n;
        k_gsp_frob<<<items < sms ? (int)items : sms, kTabThreads, kTabSmem, s>>>(p);
        TAB_CK(cudaGetLastError());
    }
    k_rcr_colmean<<<(d + 255) / 256, 256, 0, s2>>>(static_cast<const __nv_bfloat16*>(router_w), N, d,
                                                   reinterpret_cast<double*>(base + o_mean));
    TAB_CK(cudaGetLastError());
    k_rcr_proto<<<N, 256, 0, s2>>>(static_cast<const __nv_bfloat16*>(router_w), reinterpret_cast<double*>(base + o_mean),
                                   static_cast<const __nv_bfloat16*>(gamma), rcr_apply_gamma, d, eps,
                                   reinterpret_cast<float*>(base + o_x), reinterpret_cast<double*>(base + o_qn));
    TAB_CK(cudaGetLastError());
    k_rcr_gateup<<<dim3(m / 64, N), 256, d * 8, s2>>>(reinterpret_cast<const float*>(base + o_x), g2, wg, wu, d, m,
                                                      reinterpret_cast<float*>(base + o_act),
                                                      reinterpret_cast<double*>(base + o_norm));
    TAB_CK(cudaGetLastError());
    k_rcr_down<<<dim3(d / 64, N), 256, m * 4, s2>>>(reinterpret_cast<const float*>(base + o_act), wd, d, m,
                                                    reinterpret_cast<double*>(base + o_rcr));
    TAB_CK(cudaGetLastError());
    TAB_CK(cudaEventRecord(join, s2));
    TAB_CK(cudaStreamWaitEvent(s, join, 0));
    k_tables_reduce<<<N, 256, 0, s>>>(reinterpret_cast<const double*>(base + o_frob), frob_per,
                                      reinterpret_cast<const double*>(base + o_norm), norm_per,
                                      reinterpret_cast<const double*>(base + o_rcr), rcr_per, N,
                                      reinterpret_cast<double*>(base + o_raw));
    TAB_CK(cudaGetLastError());
    k_tables_final<<<1, 1024, 0, s>>>(reinterpret_cast<const double*>(base + o_raw),
                                      reinterpret_cast<const double*>(base + o_qn), N, eps, out, out + N);
    TAB_CK(cudaGetLastError());
    // one copy: each pageable one costs about 15 us
    TAB_CK(cudaMemcpyAsync(host, out, (size_t)(2 * N + 1) * 4, cudaMemcpyDeviceToHost, s));
    TAB_CK(cudaStreamSynchronize(s));
    memcpy(gsp_out, host, (size_t)N * 4);
    memcpy(rcr_out, host + N, (size_t)N * 4);
    memcpy(&herr, host + 2 * N, 4);
    if (herr & kErrTimeout) st = tab_fail(ACE_ERR_TIMEOUT, "ace_offline_tables_device: a bounded device wait ran out");
#undef TAB_CK
done:
    cudaStreamSynchronize(s);
    if (s2) {
        cudaStreamSynchronize(s2);
        cudaStreamDestroy(s2);
    }
    if (fork) cudaEventDestroy(fork);
    if (join) cudaEventDestroy(join);
    cudaFree(base);
    return st;
}
