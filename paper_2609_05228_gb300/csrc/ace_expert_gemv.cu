// ace_expert_gemv.cu — the SwiGLU experts (Eq. swiglu_expert) over the
// retained slots only, as weight-streaming GEMVs, and the gate-weighted
// combine (Eq. ace_sparse_output).
//
// Work items are (distinct retained expert, slice of weight rows); the blocks
// take equal shares of the weight rows. Each item streams its weight rows once
// per chunk of up to TC tokens routed to that expert, with 16-byte non-caching
// loads; the tokens' activations sit in shared memory, and a warp's first
// weights are on their way before it stages them. Small layers are bound by
// latency: the chain of dependent loads, the launches (PDL) and the sums over
// the warp (warp_sum_all). 64 tokens on the (256, 16 experts, top-4, 128) fp32
// layer: 42 us a call with 8-token chunks, one warp_sum per token and row and
// plain launches; 37.8 with 16-token chunks (run() says where) and dependent
// launches; 26.1 with the joint sums.
//   gate/up: act[r, j] = SiLU(h_t . W_gate[e, j]) * (h_t . W_up[e, j])
//   down:    y[r, c]   = g_hat(r) * (act[r] . W_down[e, c])
//   combine: out[t, c] = sum over t's kept slots, in rank order, of y[r, c]
#include <math.h>

#include "ace_device.cuh"
#include "ace_internal.h"

namespace ace {
namespace {

__device__ __forceinline__ float silu(float u) { return u / (1.0f + expf(-u)); }

// Rows [lo, hi) of the flattened (distinct expert, weight row) space owned by
// this block: every block streams the same number of weight rows.
__device__ __forceinline__ void block_range(long long total, long long& lo, long long& hi) {
    lo = total * blockIdx.x / gridDim.x;
    hi = total * (blockIdx.x + 1) / gridDim.x;
}

// Sums NV values over the warp at once: in each step of the butterfly a lane
// sends one half of its values and keeps the other, so 2 NV shuffles do what NV
// warp_sums do in 5 NV. Afterwards lane l holds the sums of values
// [l NV / 32, (l + 1) NV / 32) in v[0..] (NV >= 32), or of value l NV / 32 (NV
// < 32). The pairs added, and so the bits, are those of warp_sum.
template <int NV>
__device__ __forceinline__ void warp_sum_all(float (&v)[NV], int lane) {
    int n = NV;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < NV / 2; ++i) {
                if (i < n) {
                    const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
}

// gate/up: one warp per row pair (W_gate[e, j], W_up[e, j]); each lane issues
// up to kCh 16-byte loads of each row before the dot products.
template <typename T, int kTC>
__global__ void __launch_bounds__(256) k_gemv_gateup(const T* __restrict__ h, const T* __restrict__ w_gate,
                                                     const T* __restrict__ w_up,
                                                     const int32_t* __restrict__ offsets,
                                                     const int32_t* __restrict__ dlist,
                                                     const int32_t* __restrict__ perm,
                                                     const int32_t* __restrict__ meta,
                                                     float* __restrict__ act, int d, int m, int k) {
    constexpr int kCh = kTC <= 8 ? 8 : 4;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint4* hs = reinterpret_cast<uint4*>(smem_raw);     // [kTC][d / V] vectors
    constexpr int V = Vec16<T>::N;
    const int nvec = d / V;
    const int D = meta[kMetaDistinct];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    long long lo, hi;
    block_range((long long)D * m, lo, hi);
    while (lo < hi) {
        const int e = dlist[lo / m];
        const int rb = (int)(lo % m);
        const int re = (int)min((long long)m, rb + (hi - lo));
        const int r0 = offsets[e], ne = offsets[e + 1] - r0;
        for (int tc0 = 0; tc0 < ne; tc0 += kTC) {
            const int ntc = min(kTC, ne - tc0);
            // the first row pair's leading chunks load while the tokens are staged
            uint4 vg[kCh], vu[kCh];
            const auto load = [&](int j, int c0) {
                const uint4* wg = reinterpret_cast<const uint4*>(w_gate + ((size_t)e * m + j) * d);
                const uint4* wu = reinterpret_cast<const uint4*>(w_up + ((size_t)e * m + j) * d);
#pragma unroll
                for (int i = 0; i < kCh; ++i) {
                    const int c = c0 + lane + 32 * i;
                    const bool ok = c < nvec;
                    vg[i] = ok ? ld_stream(wg + c) : make_uint4(0, 0, 0, 0);
                    vu[i] = ok ? ld_stream(wu + c) : make_uint4(0, 0, 0, 0);
                }
            };
            if (rb + warp < re) load(rb + warp, 0);
            __syncthreads();
            for (int i = threadIdx.x; i < ntc * nvec; i += blockDim.x) {
                const int q = i / nvec, c = i % nvec;
                const int tok = perm[r0 + tc0 + q] / k;
                hs[i] = reinterpret_cast<const uint4*>(h + (size_t)tok * d)[c];
            }
            __syncthreads();
            for (int j = rb + warp; j < re; j += nwarps) {
                float acc[2 * kTC];                      // gate sums, then up sums
#pragma unroll
                for (int q = 0; q < 2 * kTC; ++q) acc[q] = 0.f;
                for (int c0 = 0; c0 < nvec; c0 += 32 * kCh) {
                    if (j != rb + warp || c0 != 0) load(j, c0);
#pragma unroll
                    for (int i = 0; i < kCh; ++i) {
                        const int c = c0 + lane + 32 * i;
                        if (c >= nvec) break;
                        float fg[V], fu[V];
                        Vec16<T>::to_float(vg[i], fg);
                        Vec16<T>::to_float(vu[i], fu);
#pragma unroll
                        for (int q = 0; q < kTC; ++q) {
                            if (q < ntc) {
                                float fh[V];
                                Vec16<T>::to_float(hs[q * nvec + c], fh);
#pragma unroll
                                for (int t = 0; t < V; ++t) {
                                    acc[q] = fmaf(fh[t], fg[t], acc[q]);
                                    acc[kTC + q] = fmaf(fh[t], fu[t], acc[kTC + q]);
                                }
                            }
                        }
                    }
                }
                // lanes below 16 hold gate sums, the others up sums of the same tokens
                warp_sum_all(acc, lane);
                const float u = __shfl_xor_sync(0xffffffffu, acc[0], 16);
                const int q = (lane & 15) * kTC / 16;
                if (lane < 16 && lane % (16 / kTC) == 0 && q < ntc)
                    act[(size_t)(r0 + tc0 + q) * m + j] = silu(acc[0]) * u;
            }
        }
        lo += re - rb;
    }
}

// down: one warp per 4 rows W_down[e, c..c+3] (each m long); up to kCh
// 16-byte loads per row and lane are in flight before the dot products.
template <typename T, int kTC>
__global__ void __launch_bounds__(256) k_gemv_down(const float* __restrict__ act, const T* __restrict__ w_down,
                                                   const float* __restrict__ ghat,
                                                   const int32_t* __restrict__ offsets,
                                                   const int32_t* __restrict__ dlist,
                                                   const int32_t* __restrict__ perm,
                                                   const int32_t* __restrict__ meta,
                                                   float* __restrict__ yslot, int d, int m) {
    constexpr int kCh = kTC <= 8 ? 4 : 2;
    constexpr int kRows = 4;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* as = reinterpret_cast<float*>(smem_raw);      // [kTC][m]
    __shared__ float gs[kTC];
    constexpr int V = Vec16<T>::N;
    const int nvec = m / V;
    const int D = meta[kMetaDistinct];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    long long lo, hi;
    block_range((long long)D * d, lo, hi);
    while (lo < hi) {
        const int e = dlist[lo / d];
        const int rb = (int)(lo % d);
        const int re = (int)min((long long)d, rb + (hi - lo));
        const int r0 = offsets[e], ne = offsets[e + 1] - r0;
        for (int tc0 = 0; tc0 < ne; tc0 += kTC) {
            const int ntc = min(kTC, ne - tc0);
            // the first rows' leading chunks load while the activations are staged
            uint4 wv[kRows][kCh];
            const auto load = [&](int c, int v0) {
#pragma unroll
                for (int r = 0; r < kRows; ++r) {
                    const uint4* wd = reinterpret_cast<const uint4*>(w_down + ((size_t)e * d + c + r) * m);
#pragma unroll
                    for (int i = 0; i < kCh; ++i) {
                        const int v = v0 + lane + 32 * i;
                        wv[r][i] = (c + r < re && v < nvec) ? ld_stream(wd + v) : make_uint4(0, 0, 0, 0);
                    }
                }
            };
            const int first = rb + warp * kRows;
            if (first < re) load(first, 0);
            __syncthreads();
            for (int i = threadIdx.x; i < ntc * (m / 4); i += blockDim.x) {
                const int q = i / (m / 4), c = i % (m / 4);
                reinterpret_cast<float4*>(as)[i] = reinterpret_cast<const float4*>(act + (size_t)(r0 + tc0 + q) * m)[c];
            }
            if (threadIdx.x < kTC) gs[threadIdx.x] = threadIdx.x < ntc ? ghat[perm[r0 + tc0 + threadIdx.x]] : 0.f;
            __syncthreads();
            for (int c = first; c < re; c += nwarps * kRows) {
                float acc[kTC * kRows];                  // value q * kRows + r: token q, row c + r
#pragma unroll
                for (int i = 0; i < kTC * kRows; ++i) acc[i] = 0.f;
                for (int v0 = 0; v0 < nvec; v0 += 32 * kCh) {
                    if (c != first || v0 != 0) load(c, v0);
#pragma unroll
                    for (int i = 0; i < kCh; ++i) {
                        const int v = v0 + lane + 32 * i;
                        if (v >= nvec) break;
#pragma unroll
                        for (int q = 0; q < kTC; ++q) {
                            if (q < ntc) {
                                float a[V];
                                const float4* ap = reinterpret_cast<const float4*>(as + q * m + v * V);
#pragma unroll
                                for (int t = 0; t < V / 4; ++t) {
                                    const float4 f = ap[t];
                                    a[4 * t] = f.x; a[4 * t + 1] = f.y; a[4 * t + 2] = f.z; a[4 * t + 3] = f.w;
                                }
#pragma unroll
                                for (int r = 0; r < kRows; ++r) {
                                    float fw[V];
                                    Vec16<T>::to_float(wv[r][i], fw);
#pragma unroll
                                    for (int t = 0; t < V; ++t) acc[q * kRows + r] = fmaf(a[t], fw[t], acc[q * kRows + r]);
                                }
                            }
                        }
                    }
                }
                warp_sum_all(acc, lane);
                constexpr int kPer = kTC * kRows / 32;   // sums per lane
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    const int q = (lane * kPer + i) / kRows, r = (lane * kPer + i) % kRows;
                    if (q < ntc && c + r < re) yslot[(size_t)(r0 + tc0 + q) * d + c + r] = gs[q] * acc[i];
                }
            }
        }
        lo += re - rb;
    }
}

// out[t, c] = (x[t, c] +) sum_{i kept, rank order} y[slot_pos[t*k+i], c]; a
// token's row indices are read together, then its rows, then the sum.
template <typename T, int KMAX>
__global__ void __launch_bounds__(256) k_combine(const float* __restrict__ yslot,
                                                 const int32_t* __restrict__ slot_pos, const T* __restrict__ resid,
                                                 T* __restrict__ out, int n_tokens, int d, int k) {
    pdl_wait();
    const int nq = d / 4;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)n_tokens * nq) return;
    const int t = (int)(idx / nq), c4 = (int)(idx % nq);
    int r[KMAX];
#pragma unroll
    for (int i = 0; i < KMAX; ++i) r[i] = i < k ? __ldg(slot_pos + (size_t)t * k + i) : -1;
    float4 y[KMAX];
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
        if (r[i] >= 0) y[i] = reinterpret_cast<const float4*>(yslot + (size_t)r[i] * d)[c4];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
        if (r[i] >= 0) {
            acc.x += y[i].x; acc.y += y[i].y; acc.z += y[i].z; acc.w += y[i].w;
        }
    if (resid) {
        const T* xr = resid + (size_t)t * d + c4 * 4;
        acc.x = to_f32(xr[0]) + acc.x;
        acc.y = to_f32(xr[1]) + acc.y;
        acc.z = to_f32(xr[2]) + acc.z;
        acc.w = to_f32(xr[3]) + acc.w;
    }
    T* o = out + (size_t)t * d + c4 * 4;
    o[0] = from_f32<T>(acc.x);
    o[1] = from_f32<T>(acc.y);
    o[2] = from_f32<T>(acc.z);
    o[3] = from_f32<T>(acc.w);
}

// Tokens per weight pass: 8, or 16 where experts hold more than 8 tokens, so that a second pass over
// the weights is saved, and two blocks' staged rows of either kernel fit an SM. 16 tokens halve the
// loads a lane has in flight and double the sums, so a layer whose experts hold few tokens loses by
// them (fp32 calls with 8 and 16: 1600 x 1600, 16 experts, 0.5 slots an expert 73.2 and 92.2 us, 4 slots
// 140.5 and 177.4; 1024 x 512, 64 experts, 1 slot 80.8 and 99.8). The line lies at 6 expected slots:
// the fullest experts, which the call waits for, then hold more than 8 (1024 x 512, 16 experts, 6 slots
// 66.0 and 60.8, 8 slots 77.7 and 69.0; 960 x 960 bf16, 64 experts, 6 slots 287 and 262). At 3 to 5 either is
// ahead, 16 by up to 10% and 8 by up to 23% of the time.
constexpr double kWideChunkSlots = 6.0;

template <typename T>
bool wide_chunk_fits(const ace_layer_desc& D) {
    constexpr size_t kMost = 100 << 10;
    return 16 * (size_t)D.hidden * sizeof(T) <= kMost && 16 * (size_t)D.ffn * sizeof(float) <= kMost;
}

template <typename T, int kTC>
cudaError_t run_chunk(const ace_layer* L, const void* x, void* out, int T_, cudaStream_t s, cudaEvent_t* ev) {
    const T* resid = L->desc.add_residual ? static_cast<const T*>(x) : nullptr;
    const ace_layer_desc& D = L->desc;
    const Workspace& W = L->ws;
    const int d = D.hidden, m = D.ffn, k = D.top_k;
    const dim3 grid(L->num_sms * 2);
    cudaError_t e = launch_pdl(k_gemv_gateup<T, kTC>, grid, dim3(256), (size_t)kTC * d * sizeof(T), s, (const T*)W.h,
                               (const T*)L->w_gate, (const T*)L->w_up, (const int32_t*)W.offsets,
                               (const int32_t*)W.dlist, (const int32_t*)W.perm, (const int32_t*)W.meta, W.act, d, m, k);
    if (e != cudaSuccess) return e;
    if (ev) ace::record_stage(ev[1], s);
    e = launch_pdl(k_gemv_down<T, kTC>, grid, dim3(256), (size_t)kTC * m * sizeof(float), s, (const float*)W.act,
                   (const T*)L->w_down, (const float*)W.ghat, (const int32_t*)W.offsets, (const int32_t*)W.dlist,
                   (const int32_t*)W.perm, (const int32_t*)W.meta, W.yslot, d, m);
    if (e != cudaSuccess) return e;
    const long long n = (long long)T_ * (d / 4);
    if (ev) ace::record_stage(ev[2], s);
    const dim3 cgrid((unsigned)((n + 255) / 256));
    e = k <= 8 ? launch_pdl(k_combine<T, 8>, cgrid, dim3(256), 0, s, (const float*)W.yslot, (const int32_t*)W.slot_pos,
                            resid, (T*)out, T_, d, k)
               : launch_pdl(k_combine<T, kMaxTopK>, cgrid, dim3(256), 0, s, (const float*)W.yslot,
                            (const int32_t*)W.slot_pos, resid, (T*)out, T_, d, k);
    if (ev) ace::record_stage(ev[3], s);
    return e;
}

template <typename T>
cudaError_t run(const ace_layer* L, const void* x, void* out, int T_, ace_skip_ctl ctl, cudaStream_t s,
                cudaEvent_t* ev) {
    const bool wide = wide_chunk_fits<T>(L->desc) && expected_expert_slots(L->desc, T_, ctl) >= kWideChunkSlots;
    return wide ? run_chunk<T, 16>(L, x, out, T_, s, ev) : run_chunk<T, 8>(L, x, out, T_, s, ev);
}

template <typename T>
cudaError_t init(const ace_layer_desc& D) {
    const int d = D.hidden, m = D.ffn;
    cudaError_t e;
    if (wide_chunk_fits<T>(D)) {
        if ((e = raise_smem_limit(k_gemv_gateup<T, 16>, (int)(16 * d * sizeof(T)))) != cudaSuccess) return e;
        if ((e = raise_smem_limit(k_gemv_down<T, 16>, (int)(16 * m * sizeof(float)))) != cudaSuccess) return e;
    }
    e = raise_smem_limit(k_gemv_gateup<T, 8>, (int)(8 * d * sizeof(T)));
    return e != cudaSuccess ? e : raise_smem_limit(k_gemv_down<T, 8>, (int)(8 * m * sizeof(float)));
}

}  // namespace

cudaError_t gemv_init(const ace_layer* L) {
    return L->desc.dtype == ACE_BF16 ? init<__nv_bfloat16>(L->desc) : init<float>(L->desc);
}

cudaError_t launch_experts_gemv(const ace_layer* L, const void* x, void* out, int T, ace_skip_ctl ctl, cudaStream_t s,
                                cudaEvent_t* ev) {
    if (L->desc.dtype == ACE_BF16) return run<__nv_bfloat16>(L, x, out, T, ctl, s, ev);
    return run<float>(L, x, out, T, ctl, s, ev);
}

}  // namespace ace
