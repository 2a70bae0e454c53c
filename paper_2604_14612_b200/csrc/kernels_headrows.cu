// LM head over many fp32-exact rows on the CUDA cores: the confidence statistics of up to 4096 hidden rows without a copy of
// the normalised rows and without logits in memory (the allocation-free scoring call).
//
//   logits[r, v] = sum_k (x[r, k] * scale[r] * gain[k]) * W[v, k]     x, W: bf16 or fp32; all arithmetic fp32
//
// Bound: fp32 multiply-adds (the activations stay fp32, so the 16-bit tensor pipe does not apply): 26 GFLOP for 100 rows of
// the 32000 x 4096 head are 0.35 ms at 74 TFLOP/s.  The eight-row GEMV passes it replaces re-read the head every eight rows and
// re-read the rows from L1 for every pair of weights, 266 us a pass (100 rows: 3.45 ms for the call, this kernel 1.04).  Shared-
// memory reads bound it next: 16 wavefronts per 28 packed multiply-adds of a warp at TM = 7.  A CTA takes a tile of 16 * TM rows
// by 128 weights, 32 elements of K at a time, a thread TM x 8 products as packed pairs (fma.rn.f32x2: two products an
// instruction, each rounded as fmaf rounds); two CTAs per SM cover each other's barriers.
// Sums are kept in chains of 64 elements of K, added up in shared memory; what such an addition rounds off opens the next chain.
// A row's scale and its confidence are worked out in 64 bits.  Error of the confidences against 64 bits, mean over 17 to 400 rows
// and five inputs, widths 768 / 4096 / 5120: GEMV 3.3e-7 / 3.8e-7 / 4.1e-7, here 2.7e-7 / 2.3e-7 / 2.5e-7 (with scale and confidence
// in 32 bits 3.5e-7 / 3.3e-7 / 3.3e-7).
// Rows are asked for in L2 eight lines ahead: a step of 32 elements is shorter than a trip to HBM.
// The rows of a tile are a matter of balance: R rows are ceil(R / 128) tiles of equal size, rounded up to 16 rows.
#include <math.h>

#include "cl_internal.h"

namespace {

constexpr int HN = 128, HK = 32, HT = 256, CHAIN = 64;

struct HeadRowsArgs {
    const void *W, *x;
    const float *gain, *scale;       // [d], [R]
    int R, V, d, MT, rows, NR, NT;   // rows, vocabulary, width, row tiles and their rows, vocabulary ranges, vocabulary tiles
    ClHeadPartial *part;             // [R, NR]
};

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ void fma2(unsigned long long &c, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Eight consecutive elements of a row as floats; zeros where k >= d (d is a multiple of 8).
template <typename T>
struct Raw8;
template <>
struct Raw8<__nv_bfloat16> {
    uint4 u;
    __device__ __forceinline__ void load(const __nv_bfloat16 *p, bool ok) { u = ok ? __ldg((const uint4 *)p) : make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void get(float (&v)[8]) const {
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) ClPair16<__nv_bfloat16>::get(w[i], v[2 * i], v[2 * i + 1]);
    }
};
template <>
struct Raw8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float *p, bool ok) {
        a = ok ? __ldg((const float4 *)p) : make_float4(0.f, 0.f, 0.f, 0.f);
        b = ok ? __ldg((const float4 *)p + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ void get(float (&v)[8]) const {
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
};

// Tiles in shared memory: [HK][128] floats, groups of four floats permuted by the octet of k so that the transposing stores
// (8 rows x 4 octets a warp) and the reads (groups of four) are free of bank conflicts.
__device__ __forceinline__ int tile_at(int k, int c) { return k * 128 + ((((c >> 2) ^ ((k >> 3) * 2)) << 2) | (c & 3)); }

template <typename T, int TM>
__global__ void __launch_bounds__(HT, 2) k_head_rows(HeadRowsArgs a) {
    extern __shared__ __align__(16) float sm[];
    float *As = sm, *Bs = As + HK * 128;
    unsigned long long *total = (unsigned long long *)(Bs + HK * HN);   // [TM * 4][HT] pairs, the sums of finished chains
    ClHeadPartial *run = (ClHeadPartial *)(total + TM * 4 * HT);        // [2][16 * TM], per half of a tile's columns
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mt = blockIdx.x % a.MT, rg = blockIdx.x / a.MT;
    const int row0 = mt * a.rows, nrows = min(a.rows, a.R - row0);
    const int nt0 = (int)((long long)a.NT * rg / a.NR), nt1 = (int)((long long)a.NT * (rg + 1) / a.NR);
    const int gr = (warp >> 1) * 4 + (lane >> 3), cw = warp & 1, gc = cw * 8 + (lane & 7);   // this thread's rows gr * TM .. and columns gc * 4 .. + 3, 64 + gc * 4 .. + 3
    const T *X = (const T *)a.x, *W = (const T *)a.W;

    for (int i = tid; i < 32 * TM; i += HT) run[i] = ClHeadPartial{0.f, 0.f, 0.f, 0x7fffffff};
    // what this thread stages: octet (tid & 3) of rows (tid >> 2) and (tid >> 2) + 64 of both tiles
    const int so = (tid & 3) * 8, sr = tid >> 2;
    float sc[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) sc[j] = sr + 64 * j < nrows ? a.scale[row0 + sr + 64 * j] : 0.f;

    for (int nt = nt0; nt < nt1; ++nt) {
        const int n0 = nt * HN;
#pragma unroll
        for (int i = 0; i < TM * 4; ++i) total[i * HT + tid] = 0ull;
        unsigned long long acc[TM][4];
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
        // one row of the row tile or of the weight tile per thread, asked for in L2 PF bytes ahead, a line at a time
        constexpr int LINE = 128 / (int)sizeof(T), PF = 8 * LINE;
        const int pr = tid & 127;
        const T *prow = tid < 128 ? X + (size_t)(row0 + min(pr, nrows - 1)) * a.d : W + (size_t)min(n0 + pr, a.V - 1) * a.d;
        auto ahead = [&](int k) {
            if (k < a.d) asm volatile("prefetch.global.L2 [%0];" ::"l"(prow + k));
        };
        for (int k = 0; k < PF; k += LINE) ahead(k);
        Raw8<T> ra[2], rb[2];
        Raw8<float> rg8;
        auto request = [&](int k0) {
            const bool kin = k0 + so < a.d;
            rg8.load(a.gain + k0 + so, kin);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                ra[j].load(X + (size_t)(row0 + sr + 64 * j) * a.d + k0 + so, kin && sr + 64 * j < nrows);
                rb[j].load(W + (size_t)(n0 + sr + 64 * j) * a.d + k0 + so, kin && n0 + sr + 64 * j < a.V);
            }
        };
        request(0);
        for (int k0 = 0; k0 < a.d; k0 += HK) {
            float g[8];
            rg8.get(g);
            if (k0 % LINE == 0) ahead(k0 + PF);
            __syncthreads();   // the previous tiles have been read
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float v[8];
                const int row = sr + 64 * j;
                ra[j].get(v);
                if (row < 16 * TM) {
                    const int col = (row / TM) * 8 + row % TM;
#pragma unroll
                    for (int e = 0; e < 8; ++e) As[tile_at(so + e, col)] = v[e] * sc[j] * g[e];
                }
                rb[j].get(v);
#pragma unroll
                for (int e = 0; e < 8; ++e) Bs[tile_at(so + e, row)] = v[e];
            }
            __syncthreads();
            if (k0 + HK < a.d) request(k0 + HK);
#pragma unroll 8
            for (int k = 0; k < HK; ++k) {
                float av[8];
                *(float4 *)&av[0] = *(const float4 *)&As[tile_at(k, gr * 8)];
                if (TM > 4) *(float4 *)&av[4] = *(const float4 *)&As[tile_at(k, gr * 8 + 4)];
                const ulonglong2 b0 = *(const ulonglong2 *)&Bs[tile_at(k, gc * 4)], b1 = *(const ulonglong2 *)&Bs[tile_at(k, 64 + gc * 4)];
#pragma unroll
                for (int r = 0; r < TM; ++r) {
                    const unsigned long long ar = pack2(av[r], av[r]);
                    fma2(acc[r][0], ar, b0.x);
                    fma2(acc[r][1], ar, b0.y);
                    fma2(acc[r][2], ar, b1.x);
                    fma2(acc[r][3], ar, b1.y);
                }
            }
            if ((k0 + HK) % CHAIN == 0 || k0 + HK >= a.d) {   // the chain ends: into the totals
#pragma unroll
                for (int r = 0; r < TM; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        unsigned long long &tot = total[(r * 4 + c) * HT + tid];
                        const unsigned long long t = tot, u = acc[r][c], sum = add2(t, u), b = sub2(sum, t);
                        float x, y;   // what the two sums lost opens the next chain; no number beside a sum that is not finite: that sum stays
                        unpack2(add2(sub2(t, sub2(sum, b)), sub2(u, b)), x, y);
                        tot = sum;
                        acc[r][c] = pack2(x == x ? x : 0.f, y == y ? y : 0.f);
                    }
            }
        }
        // softmax statistics of this tile's 128 logits per row: this thread's 8, then the 8 lanes of its row group
        const int c0 = n0 + gc * 4;
        auto col = [&](int c) { return c0 + (c & 3) + (c >> 2) * 64; };
#pragma unroll 1
        for (int r = 0; r < TM; ++r) {
            float l[8];
            ClHeadPartial p{-INFINITY, 0.f, 0.f, 0x7fffffff};
#pragma unroll
            for (int c = 0; c < 4; ++c) unpack2(total[(r * 4 + c) * HT + tid], l[2 * c], l[2 * c + 1]);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                l[c] = fminf(fmaxf(l[c], -CL_LOGIT_CLAMP), CL_LOGIT_CLAMP);   // clamp of Section 3.1
                if (col(c) < a.V && l[c] > p.m) { p.m = l[c]; p.idx = col(c); }
            }
            if (p.m == -INFINITY) p.m = 0.f;   // (no valid column: z stays 0 and the partial is ignored)
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (col(c) < a.V) {
                    const float d = l[c] - p.m, e = expf(d);
                    p.z += e;
                    p.s = fmaf(d, e, p.s);
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) p = cl_hp_merge(p, cl_hp_shfl_xor(p, o));
            if ((lane & 7) == 0) {
                ClHeadPartial &q = run[cw * 16 * TM + gr * TM + r];
                q = cl_hp_merge(q, p);
            }
        }
    }
    __syncthreads();
    for (int r = tid; r < nrows; r += HT) a.part[(size_t)(row0 + r) * a.NR + rg] = cl_hp_merge(run[r], run[16 * TM + r]);
}

// scale[r] = 1 / sqrt(mean x^2 + eps), one CTA per row.  In 64 bits up to the result: its error moves all logits of a row
// together, and fp32 sums, quotients and roots made it the largest part of a narrow row's error (see the head of this file).
template <typename T>
__global__ void __launch_bounds__(256) k_row_scale(const T *x, int d, float eps, float *scale) {
    __shared__ double red[8];
    double ss = 0.0;
    for (int i = threadIdx.x * 8; i < d; i += 2048) {
        Raw8<T> r;
        float v[8];
        r.load(x + (size_t)blockIdx.x * d + i, true);
        r.get(v);
#pragma unroll
        for (int e = 0; e < 8; ++e) ss = fma((double)v[e], (double)v[e], ss);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < 8; ++w) tot += red[w];
        scale[blockIdx.x] = (float)(1.0 / sqrt(tot / d + (double)eps));
    }
}

// One warp per row: the ranges' statistics in a fixed order, then Eq. 2-4.
__global__ void __launch_bounds__(128) k_head_rows_merge(const ClHeadPartial *part, int R, int NR, double inv_log_v, float *conf, float *pmax, int *arg) {
    const int r = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= R) return;
    ClHeadPartial f{0.f, 0.f, 0.f, 0x7fffffff};
    for (int g = lane; g < NR; g += 32) f = cl_hp_merge(f, part[(size_t)r * NR + g]);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const ClHeadPartial other = cl_hp_shfl_xor(f, o);
        f = (lane & o) == 0 ? cl_hp_merge(f, other) : cl_hp_merge(other, f);
    }
    if (lane == 0) {
        const double H = log((double)f.z) - (double)f.s / f.z;   // (64 bits: 1 - H / log V cancels most of a flat row's digits)
        conf[r] = (float)(1.0 - H * inv_log_v);
        pmax[r] = 1.f / f.z;
        arg[r] = f.idx;
    }
}

template <typename T, int TM>
cudaError_t launch(const HeadRowsArgs &a, cudaStream_t s) {
    const size_t smem = (size_t)(2 * HK * 128 + TM * 8 * HT) * 4 + 32 * TM * sizeof(ClHeadPartial);
    cudaError_t e = cudaFuncSetAttribute(k_head_rows<T, TM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_head_rows<T, TM><<<a.MT * a.NR, HT, smem, s>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_tm(const HeadRowsArgs &a, cudaStream_t s) {
    switch ((a.rows + 15) / 16) {
        case 1: return launch<T, 1>(a, s);
        case 2: return launch<T, 2>(a, s);
        case 3: return launch<T, 3>(a, s);
        case 4: return launch<T, 4>(a, s);
        case 5: return launch<T, 5>(a, s);
        case 6: return launch<T, 6>(a, s);
        case 7: return launch<T, 7>(a, s);
        default: return launch<T, 8>(a, s);
    }
}

}  // namespace

// Statistics of R rows; scale: scratch [R]; part: scratch [CL_HEAD_ROWS_PARTIALS].  wdtype 0 fp32, 1 bf16; 16-byte aligned inputs.
cudaError_t cl_launch_head_rows(int wdtype, const void *W, const void *x, const float *gain, int R, int V, int d, float eps, int n_sm,
                                float *scale, ClHeadPartial *part, float *conf, float *pmax, int *arg, cudaStream_t s) {
    HeadRowsArgs a;
    a.W = W; a.x = x; a.gain = gain; a.scale = scale; a.R = R; a.V = V; a.d = d; a.part = part;
    a.MT = (R + 127) / 128;
    a.rows = (R + a.MT - 1) / a.MT;
    a.MT = (R + a.rows - 1) / a.rows;
    a.NT = (V + HN - 1) / HN;
    a.NR = 2 * n_sm / a.MT;   // two CTAs per SM
    while (a.NR > 1 && (size_t)R * a.NR > CL_HEAD_ROWS_PARTIALS) --a.NR;
    if (a.NR > a.NT) a.NR = a.NT;
    if (a.NR < 1) a.NR = 1;
    if (wdtype == 1) k_row_scale<<<R, 256, 0, s>>>((const __nv_bfloat16 *)x, d, eps, scale);
    else k_row_scale<<<R, 256, 0, s>>>((const float *)x, d, eps, scale);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = wdtype == 1 ? launch_tm<__nv_bfloat16>(a, s) : launch_tm<float>(a, s);
    if (e != cudaSuccess) return e;
    k_head_rows_merge<<<(R + 3) / 4, 128, 0, s>>>(part, R, a.NR, 1.0 / log((double)V), conf, pmax, arg);
    return cudaGetLastError();
}
