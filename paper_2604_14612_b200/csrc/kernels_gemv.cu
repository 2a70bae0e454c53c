// Row-streaming matrix-vector kernels for T <= 9 activation rows on CUDA cores.
//
// y[t][r] = sum_c W[r][c] * x[t][c], W in its storage type (bf16 or fp32), x and the accumulation in fp32.
// Each warp owns pairs of consecutive weight rows and walks them with 16-byte coalesced, streaming
// (L1 no-allocate) loads; the T activation rows are re-read through L1.  The epilogue is one of:
//   STORE  plain store (QKV projection),
//   RESID  residual add in place (attention output and FFN down projections),
//   SILU   gate/up rows are interleaved in memory, so a row pair yields silu(gate) * up directly,
//   HEAD   LM head fused with the clamp, an online softmax / entropy reduction, top-1 probability and
//          argmax (Section 3.1, Eq. 1-4): logits are never written unless asked for.
// This is the general path (any T, fp32 or bf16 weights); it is bound by HBM weight streaming for T = 1.
#include <math.h>
#include <string.h>

#include <memory>
#include <algorithm>
#include <mutex>
#include <new>

#include "cl_internal.h"
#include "launch.cuh"

namespace {

__device__ __forceinline__ uint4 ld_stream16(const void *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

template <typename WT>
struct W8;
template <>
struct W8<__nv_bfloat16> {
    static __device__ __forceinline__ void load(const __nv_bfloat16 *p, float (&w)[8]) {
        uint4 v = ld_stream16(p);
        w[0] = __uint_as_float(v.x << 16); w[1] = __uint_as_float(v.x & 0xffff0000u);
        w[2] = __uint_as_float(v.y << 16); w[3] = __uint_as_float(v.y & 0xffff0000u);
        w[4] = __uint_as_float(v.z << 16); w[5] = __uint_as_float(v.z & 0xffff0000u);
        w[6] = __uint_as_float(v.w << 16); w[7] = __uint_as_float(v.w & 0xffff0000u);
    }
};
template <>
struct W8<__half> {
    static __device__ __forceinline__ void load(const __half *p, float (&w)[8]) {
        uint4 v = ld_stream16(p);
        ClPair16<__half>::get(v.x, w[0], w[1]);
        ClPair16<__half>::get(v.y, w[2], w[3]);
        ClPair16<__half>::get(v.z, w[4], w[5]);
        ClPair16<__half>::get(v.w, w[6], w[7]);
    }
};
template <>
struct W8<float> {
    static __device__ __forceinline__ void load(const float *p, float (&w)[8]) {
        uint4 a = ld_stream16(p), b = ld_stream16(p + 4);
        w[0] = __uint_as_float(a.x); w[1] = __uint_as_float(a.y); w[2] = __uint_as_float(a.z); w[3] = __uint_as_float(a.w);
        w[4] = __uint_as_float(b.x); w[5] = __uint_as_float(b.y); w[6] = __uint_as_float(b.z); w[7] = __uint_as_float(b.w);
    }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Merge two partial softmax statistics (see ClHeadPartial).  Empty partials have z == 0.
__device__ __forceinline__ ClHeadPartial head_merge(const ClHeadPartial &a, const ClHeadPartial &b) {
    if (b.z == 0.f) return a;
    if (a.z == 0.f) return b;
    ClHeadPartial r;
    r.m = fmaxf(a.m, b.m);
    float ea = expf(a.m - r.m), eb = expf(b.m - r.m);
    r.z = a.z * ea + b.z * eb;
    r.s = ea * (a.s + (a.m - r.m) * a.z) + eb * (b.s + (b.m - r.m) * b.z);
    r.idx = (a.m > b.m) ? a.idx : (b.m > a.m) ? b.idx : min(a.idx, b.idx);
    return r;
}

__device__ __forceinline__ float silu_f(float x) { return x / (1.f + expf(-x)); }

template <typename WT, int T, int EPI>
__global__ void __launch_bounds__(256) k_gemv(ClGemvArgs a) {
    pdl_launch_dependents();
    pdl_wait();
    if (a.st && a.st->done) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int gw = blockIdx.x * nw + warp, tw = gridDim.x * nw;
    const int ngroups = (a.rows + 1) >> 1;
    const int cols = a.cols;
    const WT *W = (const WT *)a.W;
    const float *xin = a.xin;
    if (a.g) {
        // RMSNorm of the rows into shared memory, a warp a row, by every CTA for itself: for several short rows that costs less than the launch
        // of a kernel that does it once (see cl_gemv_norm_max; 4 layers of width 256, fp32, cycle of 4 + 5 rows 491 -> 481 us)
        extern __shared__ __align__(16) float xs[];
        for (int t = warp; t < T; t += nw) {
            const float *xr = a.xin + (size_t)t * cols;
            // eight sums a lane: chains of four squares at most, as in k_rmsnorm
            float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f), t4 = s4;
            auto add = [&](float4 &s, int i) {
                const float4 v = *(const float4 *)(xr + i);
                s.x = fmaf(v.x, v.x, s.x); s.y = fmaf(v.y, v.y, s.y); s.z = fmaf(v.z, v.z, s.z); s.w = fmaf(v.w, v.w, s.w);
            };
            for (int i = lane * 4; i < cols; i += 256) {
                add(s4, i);
                if (i + 128 < cols) add(t4, i + 128);
            }
            const float ss = ((s4.x + s4.y) + (s4.z + s4.w)) + ((t4.x + t4.y) + (t4.z + t4.w));
            const float sc = 1.0f / sqrtf(warp_sum(ss) / (float)cols + a.eps);
            for (int i = lane * 4; i < cols; i += 128) {
                const float4 v = *(const float4 *)(xr + i), gv = *(const float4 *)(a.g + i);
                *(float4 *)(xs + t * cols + i) = make_float4(v.x * sc * gv.x, v.y * sc * gv.y, v.z * sc * gv.z, v.w * sc * gv.w);
            }
        }
        __syncthreads();
        xin = xs;
    }

    ClHeadPartial run[T];
    if (EPI == CL_EPI_HEAD) {
#pragma unroll
        for (int t = 0; t < T; ++t) run[t] = ClHeadPartial{0.f, 0.f, 0.f, 0x7fffffff};
    }

    for (int g = gw; g < ngroups; g += tw) {
        const int r0 = 2 * g;
        const bool has1 = (r0 + 1) < a.rows;
        const WT *w0 = W + (size_t)r0 * cols;
        const WT *w1 = W + (size_t)(has1 ? r0 + 1 : r0) * cols;
        float acc0[T], acc1[T];
#pragma unroll
        for (int t = 0; t < T; ++t) acc0[t] = acc1[t] = 0.f;
#pragma unroll 2
        for (int c = lane * 8; c < cols; c += 256) {
            float wa[8], wb[8];
            W8<WT>::load(w0 + c, wa);
            W8<WT>::load(w1 + c, wb);
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const float4 x0 = *(const float4 *)(xin + (size_t)t * cols + c);   // (plain: the predecessor wrote it while this kernel lived)
                const float4 x1 = *(const float4 *)(xin + (size_t)t * cols + c + 4);
                float s0 = acc0[t], s1 = acc1[t];
                s0 = fmaf(wa[0], x0.x, s0); s1 = fmaf(wb[0], x0.x, s1);
                s0 = fmaf(wa[1], x0.y, s0); s1 = fmaf(wb[1], x0.y, s1);
                s0 = fmaf(wa[2], x0.z, s0); s1 = fmaf(wb[2], x0.z, s1);
                s0 = fmaf(wa[3], x0.w, s0); s1 = fmaf(wb[3], x0.w, s1);
                s0 = fmaf(wa[4], x1.x, s0); s1 = fmaf(wb[4], x1.x, s1);
                s0 = fmaf(wa[5], x1.y, s0); s1 = fmaf(wb[5], x1.y, s1);
                s0 = fmaf(wa[6], x1.z, s0); s1 = fmaf(wb[6], x1.z, s1);
                s0 = fmaf(wa[7], x1.w, s0); s1 = fmaf(wb[7], x1.w, s1);
                acc0[t] = s0; acc1[t] = s1;
            }
        }
#pragma unroll
        for (int t = 0; t < T; ++t) {
            acc0[t] = warp_sum(acc0[t]);
            acc1[t] = warp_sum(acc1[t]);
        }
        if (lane == 0) {
#pragma unroll
            for (int t = 0; t < T; ++t) {
                if (EPI == CL_EPI_STORE) {
                    a.out[(size_t)t * a.ld + r0] = acc0[t];
                    if (has1) a.out[(size_t)t * a.ld + r0 + 1] = acc1[t];
                } else if (EPI == CL_EPI_RESID) {
                    a.out[(size_t)t * a.ld + r0] += acc0[t];
                    if (has1) a.out[(size_t)t * a.ld + r0 + 1] += acc1[t];
                } else if (EPI == CL_EPI_SILU) {
                    a.out[(size_t)t * a.ld + g] = silu_f(acc0[t]) * acc1[t];
                } else {
                    float l0 = fminf(fmaxf(acc0[t], -CL_LOGIT_CLAMP), CL_LOGIT_CLAMP);
                    if (a.logits) a.logits[(size_t)t * a.rows + r0] = l0;
                    run[t] = head_merge(run[t], ClHeadPartial{l0, 1.f, 0.f, r0});
                    if (has1) {
                        float l1 = fminf(fmaxf(acc1[t], -CL_LOGIT_CLAMP), CL_LOGIT_CLAMP);
                        if (a.logits) a.logits[(size_t)t * a.rows + r0 + 1] = l1;
                        run[t] = head_merge(run[t], ClHeadPartial{l1, 1.f, 0.f, r0 + 1});
                    }
                }
            }
        }
    }

    if (EPI == CL_EPI_HEAD) {
        __shared__ ClHeadPartial sm[256];
        __shared__ int is_last;
        if (lane == 0) {
#pragma unroll
            for (int t = 0; t < T; ++t) sm[warp * T + t] = run[t];   // nw * T <= 8 * 9 = 72 entries
        }
        __syncthreads();
        if (threadIdx.x < T) {
            ClHeadPartial r = sm[threadIdx.x];
            for (int w = 1; w < nw; ++w) r = head_merge(r, sm[w * T + threadIdx.x]);
            a.partials[(size_t)blockIdx.x * T + threadIdx.x] = r;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) is_last = (atomicAdd(a.ticket, 1u) == gridDim.x - 1);
        __syncthreads();
        if (!is_last) return;
        __threadfence();
        // The last block to finish reduces all blocks' partials in a fixed order (deterministic).
        for (int t = 0; t < T; ++t) {
            ClHeadPartial r{0.f, 0.f, 0.f, 0x7fffffff};
            for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
                const volatile ClHeadPartial *p = a.partials + (size_t)b * T + t;
                ClHeadPartial q;
                q.m = p->m; q.z = p->z; q.s = p->s; q.idx = p->idx;
                r = head_merge(r, q);
            }
            __syncthreads();
            sm[threadIdx.x] = r;
            __syncthreads();
            for (int o = blockDim.x >> 1; o > 0; o >>= 1) {
                if ((int)threadIdx.x < o) sm[threadIdx.x] = head_merge(sm[threadIdx.x], sm[threadIdx.x + o]);
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                ClHeadPartial f = sm[0];
                // H = log Z - S/Z (entropy of the softmax, from sums relative to the maximum);
                // confidence = 1 - H / log V (Eq. 3-4); top-1 probability = 1 / Z.
                float H = logf(f.z) - f.s / f.z;
                if (a.out_tok) a.out_tok[t] = f.idx;
                if (a.out_pmax) a.out_pmax[t] = 1.f / f.z;
                if (a.out_conf) a.out_conf[t] = 1.f - H * a.inv_log_v;
            }
        }
        if (threadIdx.x == 0) *a.ticket = 0u;
    }
}

template <typename WT, int T>
cudaError_t launch_t(int epi, const ClGemvArgs &a, int grid, cudaStream_t s) {
    if (a.g && a.cols > CL_GEMV_NORM_MAX) return cudaErrorInvalidValue;
    const size_t smem = a.g ? (size_t)T * a.cols * 4 : 0;
    switch (epi) {
        case CL_EPI_STORE: return launch_chained(k_gemv<WT, T, CL_EPI_STORE>, dim3(grid), 256, smem, 1, s, a);
        case CL_EPI_RESID: return launch_chained(k_gemv<WT, T, CL_EPI_RESID>, dim3(grid), 256, smem, 1, s, a);
        case CL_EPI_SILU: return launch_chained(k_gemv<WT, T, CL_EPI_SILU>, dim3(grid), 256, smem, 1, s, a);
        case CL_EPI_HEAD: return launch_chained(k_gemv<WT, T, CL_EPI_HEAD>, dim3(grid), 256, smem, 1, s, a);
        default: return cudaErrorInvalidValue;
    }
}

template <typename WT>
cudaError_t launch_w(int T, int epi, const ClGemvArgs &a, int grid, cudaStream_t s) {
    switch (T) {
        case 1: return launch_t<WT, 1>(epi, a, grid, s);
        case 2: return launch_t<WT, 2>(epi, a, grid, s);
        case 3: return launch_t<WT, 3>(epi, a, grid, s);
        case 4: return launch_t<WT, 4>(epi, a, grid, s);
        case 5: return launch_t<WT, 5>(epi, a, grid, s);
        case 6: return launch_t<WT, 6>(epi, a, grid, s);
        case 7: return launch_t<WT, 7>(epi, a, grid, s);
        case 8: return launch_t<WT, 8>(epi, a, grid, s);
        case 9: return launch_t<WT, 9>(epi, a, grid, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t cl_launch_gemv(int wdtype, int T, int epi, const ClGemvArgs &a, int grid, cudaStream_t s) {
    if (wdtype == 1) return launch_w<__nv_bfloat16>(T, epi, a, grid, s);
    if (wdtype == 2) return launch_w<__half>(T, epi, a, grid, s);
    return launch_w<float>(T, epi, a, grid, s);
}

// ---- confidence scoring without any allocation ------------------------------------------------------
// Scratch of cl_layer_confidences_static(): one file-scope array that every GPU loading this library holds until
// the process exits.  Layout (bytes): [0, 256) ticket counters; then the normalised rows
// xn [SC_CHUNK, CL_STATIC_MAX_D] fp32; the softmax partials of either path; the rows' normalisation factors
// [CL_STATIC_MAX_ROWS] fp64; the rows in three bf16 parts for the tensor cores (15 MB: 512 rows of 5120 elements); two flags and the three per-row results (confidence, top-1 probability, greedy token) [n_rows] each,
// side by side so that one copy fetches them.
// Few rows take passes of the streaming GEMV, eight rows each, more take the kernels of kernels_headrows.cu.
// fp32 heads, from 17 rows.  At 16 rows, two whole passes, it depends on how the tiles share the chip (16 rows, GEMV / tiled kernel, us: 32000 x 4096
// 604 / 481, 5003 x 768 132 / 96, but 5003 x 4096 222 / 285, 20480 x 4096 453 / 478); a third pass costs the GEMV more than that.
// bf16 heads: the tensor-core kernel costs much the same for 1 to 128 rows (32000 x 4096 with 100 rows 8 % more than with 6, 128256 x 4096 14 %) and waits for K
// block after K block, so that it needs a vocabulary that is long against the width.  Whole call from idle, GEMV with that many rows / tensor-core kernel, us (under load
// for some seconds both are up to 10 % faster and the lines hold within 2 %):
//   V < d         from 12 rows  1000 x 4096 105 / 101 (10 rows 95 / 99), 2000 x 8192 155 / 150 (10: 142 / 150), 200 x 4096 105 / 101 (10: 93 / 100)
//   d <= V < 3 d  from 9        4096 x 4096 104 / 101 (8: 88 / 100), 5003 x 4096 130 / 100 (8: 112 / 101, 7: 100 / 101), 8192 x 8192 205 / 152 (7: 138 / 151)
//   V >= 3 d      from 8        12288 x 4096 150 / 113, 40000 x 4096 274 / 226, 128256 x 4096 647 / 401; or from 7, 6 or 5 (few_rows_line)
namespace {

// Most rows for the GEMV where V >= 3 d.  Five to seven rows are a matter of the tensor-core kernel's last wave of tiles: both times in us, from fits of
// heads of 3000 x 512 to 128256 x 4096 (cost: of the fullest CTA, a K block).  Measured, GEMV / tensor cores:
// 5 rows  32000 x 4096 177 / 140, 32000 x 5120 187 / 164, 32000 x 768 88 / 76, 3000 x 512 61 / 51, but 12288 x 4096 112 / 113, 40000 x 4096 202 / 226,
//         50257 x 2560 163 / 166, 100000 x 4096 373 / 400
// 6 rows  50257 x 2560 177 / 166, 100000 x 4096 403 / 400, 128256 x 4096 498 / 400, but 12288 x 4096 112 / 112, 40000 x 4096 205 / 226
// 7 rows  12288 x 4096 125 / 114, 40000 x 4096 236 / 226
int few_rows_line(int V, int d, int n_sm) {
    const double tc = 60.0 + 7e-4 * (double)cl_head_tc_cost(V, n_sm) * ((d + 63) / 64), elems = (double)V * d;
    return tc <= 70.0 + 7.4e-7 * elems ? 4 : tc <= 70.0 + 8.2e-7 * elems ? 5 : tc <= 81.0 + 9.4e-7 * elems ? 6 : 7;
}

constexpr int SC_MAX_GRID = 1024;
constexpr int SC_CHUNK = 8;   // rows per LM-head pass of the GEMV
constexpr int SC_GEMV_ROWS = 2 * SC_CHUNK;   // most rows that take such passes, whatever the head
constexpr size_t SC_OFF_XN = 256;
constexpr size_t SC_OFF_PART = SC_OFF_XN + (size_t)SC_CHUNK * CL_STATIC_MAX_D * sizeof(float);
constexpr size_t SC_PARTIALS = std::max<size_t>(SC_MAX_GRID * SC_CHUNK, std::max(CL_HEAD_ROWS_PARTIALS, CL_HEAD_TC_PARTIALS));
constexpr size_t SC_OFF_SCALE = SC_OFF_PART + SC_PARTIALS * sizeof(ClHeadPartial);
constexpr size_t SC_OFF_SPLIT = SC_OFF_SCALE + (size_t)CL_STATIC_MAX_ROWS * sizeof(double);
constexpr size_t SC_SPLIT = (size_t)512 * 5120 * 6;   // (128 rows of 8192 elements take 6.3 MB)
constexpr size_t SC_OFF_RES = SC_OFF_SPLIT + SC_SPLIT;
static_assert(SC_OFF_SPLIT % 256 == 0 && SC_SPLIT >= (size_t)128 * CL_STATIC_MAX_D * 6, "a row tile's parts");
constexpr size_t SC_BYTES = SC_OFF_RES + (2 + 3 * (size_t)CL_STATIC_MAX_ROWS) * 4;

static __device__ __align__(256) unsigned char g_static_scratch[SC_BYTES];

constexpr int SC_MAX_DEVICES = 64;
std::mutex g_sc_mutex;
unsigned char *g_sc_addr[SC_MAX_DEVICES];   // device address of g_static_scratch on each device, once looked up
int g_sc_sms[SC_MAX_DEVICES];

// In host code `g_static_scratch` is only a handle for the runtime, not a device address: the address a kernel
// may use comes from cudaGetSymbolAddress, asked once per device with that device current.
int static_scratch(unsigned char **addr, int *n_sm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        cl_set_global_error("cl_layer_confidences_static: no CUDA device: %s", cudaGetErrorString(e));
        return CL_ECUDA;
    }
    if (dev < 0 || dev >= SC_MAX_DEVICES) {
        cl_set_global_error("cl_layer_confidences_static: device ordinal %d not supported (max %d)", dev, SC_MAX_DEVICES - 1);
        return CL_ERANGE;
    }
    std::lock_guard<std::mutex> lock(g_sc_mutex);
    if (!g_sc_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) {
            cl_set_global_error("cl_layer_confidences_static: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            return CL_ECUDA;
        }
        int sms = 0, major = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (major < 10 || sms <= 0) {
            cl_set_global_error("cl_layer_confidences_static: compute capability %d.x, built for sm_100a only", major);
            return CL_ECUDA;
        }
        g_sc_sms[dev] = sms;
        g_sc_addr[dev] = (unsigned char *)p;
    }
    *addr = g_sc_addr[dev];
    *n_sm = g_sc_sms[dev];
    return CL_OK;
}

}  // namespace

extern "C" int cl_layer_confidences_static(const void *lm_head, const float *final_norm, int vocab, int d_model,
                                           int weight_dtype, float rms_eps, const void *hidden, int n_rows,
                                           void *cuda_stream, float *conf, float *p_max, int32_t *argmax) {
    if (!lm_head || !final_norm || !hidden) {
        cl_set_global_error("cl_layer_confidences_static: null input pointer");
        return CL_EINVAL;
    }
    if (weight_dtype != 0 && weight_dtype != 1) {
        cl_set_global_error("cl_layer_confidences_static: weight_dtype must be 0 or 1");
        return CL_EINVAL;
    }
    if (vocab < 2 || d_model <= 0 || d_model % 8 || n_rows <= 0) {
        cl_set_global_error("cl_layer_confidences_static: need vocab >= 2, d_model a positive multiple of 8, n_rows > 0");
        return CL_EINVAL;
    }
    if (((uintptr_t)lm_head | (uintptr_t)final_norm | (uintptr_t)hidden) & 15u) {
        // the kernels read these with 16-byte vector loads; a misaligned pointer would trap on the device
        cl_set_global_error("cl_layer_confidences_static: lm_head, final_norm and hidden must be 16-byte aligned");
        return CL_EINVAL;
    }
    if (d_model > CL_STATIC_MAX_D || n_rows > CL_STATIC_MAX_ROWS) {
        cl_set_global_error("cl_layer_confidences_static: d_model %d / n_rows %d beyond the fixed scratch (max %d / %d)", d_model,
                            n_rows, CL_STATIC_MAX_D, CL_STATIC_MAX_ROWS);
        return CL_ERANGE;
    }
    unsigned char *sc = nullptr;
    int n_sm = 0;
    int rc = static_scratch(&sc, &n_sm);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    float *xn = (float *)(sc + SC_OFF_XN);
    unsigned *flags = (unsigned *)(sc + SC_OFF_RES);
    float *d_conf = (float *)(flags + 2), *d_pmax = d_conf + n_rows;
    int *d_arg = (int *)(d_pmax + n_rows);
    const size_t es = weight_dtype == 1 ? 2 : 4;
    auto many_rows = [&]() -> cudaError_t {
        return cl_launch_head_rows(weight_dtype, lm_head, hidden, final_norm, n_rows, vocab, d_model, rms_eps, n_sm, (double *)(sc + SC_OFF_SCALE),
                                   (ClHeadPartial *)(sc + SC_OFF_PART), d_conf, d_pmax, d_arg, s);
    };
    auto few_rows = [&]() -> cudaError_t {
        ClGemvArgs a;
        memset(&a, 0, sizeof(a));
        a.W = lm_head; a.rows = vocab; a.cols = d_model; a.xin = xn;
        a.partials = (ClHeadPartial *)(sc + SC_OFF_PART);
        a.ticket = (unsigned *)sc;
        a.inv_log_v = (float)(1.0 / log((double)vocab));
        int grid = ((vocab + 1) / 2 + 7) / 8;
        if (grid > n_sm * 4) grid = n_sm * 4;
        if (grid > SC_MAX_GRID) grid = SC_MAX_GRID;
        cudaError_t e = cudaSuccess;
        for (int r0 = 0; r0 < n_rows && e == cudaSuccess; r0 += SC_CHUNK) {
            const int T = n_rows - r0 < SC_CHUNK ? n_rows - r0 : SC_CHUNK;
            e = cl_launch_rmsnorm_rows(weight_dtype, (const char *)hidden + (size_t)r0 * d_model * es, final_norm, T, d_model, rms_eps, xn, s);
            if (e != cudaSuccess) break;
            a.out_tok = d_arg + r0; a.out_pmax = d_pmax + r0; a.out_conf = d_conf + r0;
            e = cl_launch_gemv(weight_dtype, T, CL_EPI_HEAD, a, grid, s);
        }
        return e;
    };
    // where the results come back to: on the stack for the usual calls (callers' threads may have little of it), else 49 KB at most from the heap
    unsigned few[2 + 3 * 256];
    std::unique_ptr<unsigned[]> many(n_rows > 256 ? new (std::nothrow) unsigned[2 + 3 * (size_t)n_rows] : nullptr);
    unsigned *res = n_rows > 256 ? many.get() : few;
    if (!res) {
        cl_set_global_error("cl_layer_confidences_static: no host memory for the results of %d rows", n_rows);
        return CL_ENOMEM;
    }
    auto fetch = [&]() -> cudaError_t {
        const cudaError_t e = cudaMemcpyAsync(res, flags, (2 + 3 * (size_t)n_rows) * 4, cudaMemcpyDeviceToHost, s);
        return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
    };
    cudaError_t e = cudaSuccess;
    const bool tc = weight_dtype == 1;
    const int gemv_rows = !tc ? SC_GEMV_ROWS : vocab < d_model ? 11 : vocab < 3LL * d_model ? 8 : few_rows_line(vocab, d_model, n_sm);   // most rows that take those passes
    if (tc && n_rows > gemv_rows) {
        e = cl_launch_head_tc(lm_head, hidden, final_norm, n_rows, vocab, d_model, rms_eps, n_sm, (double *)(sc + SC_OFF_SCALE), sc + SC_OFF_SPLIT, SC_SPLIT,
                              (ClHeadPartial *)(sc + SC_OFF_PART), flags, d_conf, d_pmax, d_arg, s);
        if (e == cudaSuccess) e = fetch();
        if (e == cudaSuccess && res[0] && !res[1]) {   // not a call for that kernel: once more on the others, whose tickets start at zero
            e = cudaMemsetAsync(sc, 0, SC_OFF_XN, s);
            if (e == cudaSuccess) e = n_rows > SC_GEMV_ROWS ? many_rows() : few_rows();
            if (e == cudaSuccess) e = fetch();
        }
    } else {
        // the tickets and flags must start at zero whatever the last call left
        e = cudaMemsetAsync(sc, 0, SC_OFF_XN, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(flags, 0, 8, s);
        if (e == cudaSuccess) e = n_rows > gemv_rows ? many_rows() : few_rows();
        if (e == cudaSuccess) e = fetch();
    }
    if (e != cudaSuccess) {
        cl_set_global_error("cl_layer_confidences_static: %s", cudaGetErrorString(e));
        return CL_ECUDA;
    }
    if (res[1]) {
        cl_set_global_error("cl_layer_confidences_static: a bounded device-side wait expired; results of this call are invalid");
        return CL_ETIMEOUT;
    }
    if (conf) memcpy(conf, res + 2, (size_t)n_rows * 4);
    if (p_max) memcpy(p_max, res + 2 + n_rows, (size_t)n_rows * 4);
    if (argmax) memcpy(argmax, res + 2 + 2 * (size_t)n_rows, (size_t)n_rows * 4);
    return CL_OK;
}
