// LM head over many fp32-exact rows: the confidence statistics of up to 4096 hidden rows without a copy of the normalised rows and
// without logits in memory (the allocation-free scoring call).  Two kernels: k_head_rows on the CUDA cores for fp32 heads (and the
// calls that k_head_tc hands over), k_head_tc on the tensor cores for bf16 heads (see there).
//
//   logits[r, v] = sum_k (x[r, k] * scale[r] * gain[k]) * W[v, k]     x, W: bf16 or fp32, activations and sums fp32 or better
//
// k_head_rows is bound by shared-memory reads (16 wavefronts per 28 packed multiply-adds of a warp at TM = 7; 100 rows of a bf16
// 32000 x 4096 head 0.99 ms, multiply-adds 0.35).  A CTA takes a tile of 16 * TM rows by 128 weights, 32 elements of K at a time, a
// thread TM x 8 products as packed pairs (fma.rn.f32x2: two products an instruction, each rounded as fmaf rounds); two CTAs per SM
// cover each other's barriers.
// Sums are kept in chains of 64 elements of K, added up in shared memory; what such an addition rounds off opens the next chain.
// A row's scale and its confidence are worked out in 64 bits.
// Rows are asked for in L2 eight lines ahead: a step of 32 elements is shorter than a trip to HBM.
// The rows of a tile are a matter of balance: R rows are ceil(R / 128) tiles of equal size, rounded up to 16 rows.
#include <math.h>

#include <type_traits>

#include "tc_common.cuh"

namespace {

constexpr int HN = 128, HK = 32, HT = 256, CHAIN = 64;
constexpr float HT_CUT = 0.268e-7f;   // what a cut takes of a sum in tensor memory, mean (see k_head_tc)

struct HeadRowsArgs {
    const void *W, *x;
    const float *gain;               // [d]
    const double *scale;             // [R]
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
    for (int j = 0; j < 2; ++j) sc[j] = sr + 64 * j < nrows ? (float)a.scale[row0 + sr + 64 * j] : 0.f;

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

__device__ __forceinline__ unsigned cvt_bf16x2(float a, float b) {   // a in the low half
    unsigned r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
    return r;
}
__device__ __forceinline__ void bf16x2_get(unsigned u, float &a, float &b) {
    a = __uint_as_float(u << 16);
    b = __uint_as_float(u & 0xffff0000u);
}

// scale[r] = 1 / sqrt(mean x^2 + eps), one CTA per row.  In 64 bits up to the result: its error moves all logits of a row
// together, and fp32 sums, quotients and roots made it the largest part of a narrow row's error (see the head of this file).
// With gain: more by what k_head_tc's sums of this row lose (see there).  A cut falls behind each of the four multiply-adds of a K block's highest part
// that adds anything, at the size of the block's sum so far.  That size is taken from the row's squares, as if the token's weights leaned towards the row,
// which those of a leading token do.  Eight lanes hold a K block, two of them the 16 elements of a multiply-add.
// split: the row's three parts for k_head_tc go there, [3][rows][d]; flags [2]: to be cleared.
template <typename T>
__global__ void __launch_bounds__(256) k_row_scale(const T *x, const float *gain, int d, float eps, double *scale, __nv_bfloat16 *split, unsigned *flags) {
    pdl_launch_dependents();
    if (blockIdx.x == 0 && threadIdx.x < 2 && flags) flags[threadIdx.x] = 0u;
    __shared__ double red[8];
    __shared__ float cuts[8], all[8];
    double ss = 0.0;
    float cut = 0.f, whole = 0.f;
    for (int i = threadIdx.x * 8; i < (d + 255) / 256 * 256; i += 2048) {   // (whole warps)
        Raw8<T> r;
        float v[8];
        r.load(x + (size_t)blockIdx.x * d + i, i < d);
        r.get(v);
#pragma unroll
        for (int e = 0; e < 8; ++e) ss = fma((double)v[e], (double)v[e], ss);
        if (gain) {
            Raw8<float> g8;
            float g[8], sq = 0.f;
            g8.load(gain + i, i < d);
            g8.get(g);
            if (split && i < d) {
                unsigned h[4], m[4], l[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float h0, h1, m0, m1;
                    h[e] = cvt_bf16x2(v[2 * e] * g[2 * e], v[2 * e + 1] * g[2 * e + 1]);
                    bf16x2_get(h[e], h0, h1);
                    const float q0 = fmaf(v[2 * e], g[2 * e], -h0), q1 = fmaf(v[2 * e + 1], g[2 * e + 1], -h1);   // exact: 32 bits less the leading eight
                    m[e] = cvt_bf16x2(q0, q1);
                    bf16x2_get(m[e], m0, m1);
                    l[e] = cvt_bf16x2(q0 - m0, q1 - m1);
                }
                __nv_bfloat16 *to = split + (size_t)blockIdx.x * d + i;
                const size_t part = (size_t)gridDim.x * d;
                *(uint4 *)to = make_uint4(h[0], h[1], h[2], h[3]);
                *(uint4 *)(to + part) = make_uint4(m[0], m[1], m[2], m[3]);
                *(uint4 *)(to + 2 * part) = make_uint4(l[0], l[1], l[2], l[3]);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) sq = fmaf(v[e] * g[e], v[e] * g[e], sq);
            sq += __shfl_xor_sync(0xffffffffu, sq, 1);   // a multiply-add's elements
            float sum = sq;                              // and with those before them in the K block
            const float b2 = __shfl_up_sync(0xffffffffu, sum, 2, 8);
            if ((threadIdx.x & 7) >= 2) sum += b2;
            const float b4 = __shfl_up_sync(0xffffffffu, sum, 4, 8);
            if ((threadIdx.x & 7) >= 4) sum += b4;
            cut += sq > 0.f ? sum : 0.f;   // (each multiply-add counted by both of its lanes, as in whole)
            whole += sq;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
        cut += __shfl_xor_sync(0xffffffffu, cut, o);
        whole += __shfl_xor_sync(0xffffffffu, whole, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = ss;
        cuts[threadIdx.x >> 5] = cut;
        all[threadIdx.x >> 5] = whole;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        ss = red[threadIdx.x];
        cut = cuts[threadIdx.x];
        whole = all[threadIdx.x];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            ss += __shfl_xor_sync(0xffu, ss, o);
            cut += __shfl_xor_sync(0xffu, cut, o);
            whole += __shfl_xor_sync(0xffu, whole, o);
        }
        if (threadIdx.x == 0) {
            const float n = gain ? cut / whole : 0.f;   // 1 .. 4 cuts at the size of the sum
            // (squares of very large or very small rows: no number, or none to speak of)
            scale[blockIdx.x] = 1.0 / sqrt(ss / d + (double)eps) * (1.0 + (double)HT_CUT * (n < 5.f ? n : 0.f));
        }
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

// ---- bf16 heads: the same products on the tensor cores --------------------------------------------------------------------
//
// A weight is one bf16 number, an activation x * gain three of them: hi + mid + lo hold 26 bits of the product, more than fp32.
// What is left to keep exact are the sums, and the accumulator in tensor memory cuts off where an fp32 addition rounds.  So:
//   - a chain is one K block: 4 multiply-adds (K 16) of lo, 4 of mid, 4 of hi, in this order, so that only the last four cut
//     off at the size of the sum; the finished chain is added to the row's fp32 total in registers, and what that addition
//     rounds off is put back into the accumulator, where the next but one chain starts from it (two accumulators alternate);
//   - what remains is a loss with a known mean, proportional to the sum: with a significand spread evenly over its logarithm a cut
//     takes 0.72 * 2^-25 of the value or a little more (HT_CUT, from the common shrinking of the logits of dense rows).  How many cuts a row's
//     sums meet, and at what size, k_row_scale reads off the row: 2.5 at full size where all of a K block adds up evenly, one where its
//     16 largest elements stand alone.  The row's scale makes up for it, by 1.07e-7 at most.  Mean error of a logit by kind of row (dense, one or four
//     elements, large channels at either end of the K blocks, widths 8 to 4096): -5e-8 .. +4e-8, and +6e-8 where sums come out exact; with nothing put
//     back -14e-8 .. -1e-8, with 6.7e-8 for every row -7e-8 .. +6e-8.  (Chains of 2 and 4 K blocks lose 2.5e-7 and 6.2e-7 and would be 10 us faster.)
// The scale is applied last, as a pair of floats.  Error of the confidences / of the top-1 probabilities against 64 bits, rows with
// leading logits of 10 to 14, three inputs: width 768 0.87e-7 .. 0.91e-7 / 1.78e-7 .. 1.83e-7 (k_head_rows 1.5e-7 / 2.1e-7), width 4096
// 0.78e-7 .. 0.84e-7 / 1.47e-7 .. 1.51e-7 (1.2e-7 / 1.7e-7).
//
// Bound: hand-overs between the multiplying thread and the chain warps, then shared memory.  A K block of 128 rows x 224 weights is 12 multiply-adds
// that read 11 KB each, 76 KB are written beside them: 1630 cycles at 128 bytes a cycle against 1344 of multiply-add; measured 2450, and 2000 where the
// chain warps only release (every CTA split the rows for itself before, 33 KB more in shared memory and a third of the issue slots: 2600).
// The parts are written once by k_row_scale.  100 rows of the 32000 x 4096 head: 102 us (137), of them 8 before the first K block and 5 of statistics
// (11, from two passes over the logits by eight warps); the rows' merge is a kernel of 5 us (13 on one SM by the last CTA).  The call 183 -> 146,
// 32000 x 768 95 -> 82, 128256 x 4096 513 -> 434, 400 rows of it 1836 -> 1570; 32000 x 4096, 4096 rows 3980 -> 3750.
// 224 weights a tile: 32000 of them are one tile per SM (143), and the totals of a tile are 80 registers a thread.
// 16 warps: 0 copies weights, 2 the rows' parts (TMA), 1 multiplies, 4-15 add up chains and keep the softmax statistics, a third of a tile's columns by
// four warps.  (The columns of a group are constants: with a bound at run time the loop over them took 2.7 us a K block instead of 1.3.)
// The head is asked for in L2 eight K blocks ahead.
// A logit that comes out as no finite number may have a sign all the same (an infinite weight times a part that is zero is NaN): the warp that
// holds it works its token out again for all its rows, from the weights that are not finite (see special_logit): one infinite weight costs 8 to 11
// us (6 rows of the 32000 x 4096 head 160 -> 168 us, of a second pass on other kernels 650), 300 tokens of infinities side by side 120.  Rows that are NaN throughout (a NaN or an infinity among the
// activations, or a row of zeros with eps = 0) need nothing: every logit counts as the lower clamp, as in the other kernels.
constexpr int HTC_THREADS = 512;
constexpr int HTC_A = 3 * 128 * 128,                // bytes of a K block's rows, split in three
              HTC_AST = 2, HTC_BST = 4, HTC_AHEAD = 8;   // stages of the rings (parts; K blocks of weights), K blocks asked for in L2

struct HeadTcArgs {
    const __nv_bfloat16 *x, *W, *split;  // [R, d], [V, d], [3][R, d]: x * gain in three parts
    const float *gain;
    const double *scale;                 // [R]
    int R, V, d, KB, MT, rows, NR, NT;   // rows, vocabulary, width, K blocks, row tiles and their rows, vocabulary ranges, vocabulary tiles
    ClHeadPartial *part;                 // [R, NR, groups of chain warps]
    unsigned *flags;                     // zero at launch: [0] results are to be had from the other kernels, [1] a wait ran out
};

struct HeadTcSmem {
    unsigned long long afull[HTC_AST], aempty[HTC_AST], bfull[HTC_BST], bempty[HTC_BST], tfull[2], tempty[2], done;
    unsigned tmem_base;
    int abort;
};

__device__ __forceinline__ void tmem_st16(unsigned taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"f"(v[0]), "f"(v[1]),
        "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]),
        "f"(v[13]), "f"(v[14]), "f"(v[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ float tmem_ld1(unsigned taddr) {
    float v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=f"(v) : "r"(taddr) : "memory");
    return v;
}
__device__ __forceinline__ void tmem_st1(unsigned taddr, float v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "f"(v) : "memory");
}
// The logits of 32 rows, a lane each, for one token some of whose weights are no finite numbers: these alone decide, in IEEE arithmetic on
// the operands that the other kernels have.  The warp looks through the token's weights; acc is set where there are such weights (any).
__device__ __noinline__ float special_logit(const __nv_bfloat16 *x, const __nv_bfloat16 *w, const float *gain, float scale, int d, bool want, bool *any) {
    const int lane = threadIdx.x & 31;
    float acc = 0.f;
    *any = false;
    for (int k0 = 0; k0 < d; k0 += 1024) {
        unsigned v[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = k0 + j * 256 + lane * 8;
            const uint4 u = k < d ? *(const uint4 *)(w + k) : make_uint4(0u, 0u, 0u, 0u);
            v[j][0] = u.x; v[j][1] = u.y; v[j][2] = u.z; v[j][3] = u.w;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            bool here = false;
#pragma unroll
            for (int e = 0; e < 4; ++e) here |= (v[j][e] & 0x7f80u) == 0x7f80u || (v[j][e] & 0x7f800000u) == 0x7f800000u;
            for (unsigned m = __ballot_sync(0xffffffffu, here); m; m &= m - 1u) {
                const int src = __ffs(m) - 1, k = k0 + j * 256 + src * 8;
                Raw8<__nv_bfloat16> xr, wr;
                float xv[8], wv[8];
                wr.u.x = __shfl_sync(0xffffffffu, v[j][0], src); wr.u.y = __shfl_sync(0xffffffffu, v[j][1], src);
                wr.u.z = __shfl_sync(0xffffffffu, v[j][2], src); wr.u.w = __shfl_sync(0xffffffffu, v[j][3], src);
                xr.u = want ? *(const uint4 *)(x + k) : make_uint4(0u, 0u, 0u, 0u);
                xr.get(xv);
                wr.get(wv);
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (!(fabsf(wv[e]) < INFINITY)) acc += xv[e] * scale * gain[k + e] * wv[e];
                *any = true;
                if (__all_sync(0xffffffffu, !want || acc != acc)) return acc;   // NaN for all: it stays NaN
            }
        }
    }
    return acc;
}
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap *map, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(map), "r"(c0), "r"(c1) : "memory");
}
template <int N>
__global__ void __launch_bounds__(HTC_THREADS, 1) k_head_tc(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW, HeadTcArgs a) {
    constexpr int B_BYTES = N * 128, NG = (N / 3 + 15) / 16 * 16, NG3 = N - 2 * NG, CHAIN_WARPS = NG3 > 0 ? 12 : 8;   // columns of a group of chain warps, of the third
    extern __shared__ unsigned char smem_dyn[];   // rings of swizzled tiles: 1 KB aligned
    unsigned char *ringA = (unsigned char *)(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023), *ringB = ringA + HTC_AST * HTC_A;
    HeadTcSmem *sm = (HeadTcSmem *)(ringB + HTC_BST * B_BYTES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = blockIdx.x % a.MT, rg = blockIdx.x / a.MT, KB = a.KB;
    const int row0 = mt * a.rows, nrows = min(a.rows, a.R - row0);
    const int nt0 = (int)((long long)a.NT * rg / a.NR), nt1 = (int)((long long)a.NT * (rg + 1) / a.NR), ntiles = nt1 - nt0;
    int *err = (int *)(a.flags + 1);

    if (tid == 0) {
        for (int i = 0; i < HTC_AST; ++i) {
            bar_init(&sm->afull[i], 1);
            bar_init(&sm->aempty[i], 1);
        }
        for (int i = 0; i < HTC_BST; ++i) {
            bar_init(&sm->bfull[i], 1);
            bar_init(&sm->bempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(&sm->tfull[i], 1);
            bar_init(&sm->tempty[i], CHAIN_WARPS);
        }
        bar_init(&sm->done, 1);
        sm->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s_u32(&sm->tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = *(volatile unsigned *)&sm->tmem_base;
    pdl_wait();   // the scales

    // ---------------- chains: a thread has a third of a row of the tile, columns [grp * NG, + NC) ----------------
    auto chains = [&](auto nc, int grp) {
        constexpr int NC = decltype(nc)::value;
        asm volatile("setmaxnreg.inc.sync.aligned.u32 144;");
        const int q = warp & 3, row = q * 32 + lane;
        const unsigned tl = tmem + ((unsigned)(q * 32) << 16) + (unsigned)(grp * NG);
        float s_hi = 0.f, s_lo = 0.f, scale = 0.f;
        bool ok = true, odd = false, redo = false;   // redo: a logit of this row that is not finite may be worked out again
        if (row < nrows) {
            const double raw = a.scale[row0 + row];
            const bool number = raw > 0.0 && raw < (double)INFINITY;   // else all logits of the row are NaN, here as in the other kernels
            odd = number && !(raw > 0x1p-100 && raw < 0x1p90);         // (the lowest parts of such a row, or its sums, could leave the range of a float)
            redo = number && !odd;
            scale = (float)raw;
            s_hi = scale;
            s_lo = (float)(raw - (double)s_hi);
        }
        const float zero[16] = {};
#pragma unroll 1
        for (int c = 0; c < NC; c += 16) {
            tmem_st16(tl + c, zero);
            tmem_st16(tl + 256u + c, zero);
        }
        auto release = [&](unsigned b) {
            if (lane == 0) bar_arrive(&sm->tempty[b]);
        };
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        release(0);
        release(1);
        ClHeadPartial run{0.f, 0.f, 0.f, 0x7fffffff};   // (a tile's sums by themselves first: added to a leading weight one by one they would lose more)
        unsigned g = 0;
        for (int t = 0; t < ntiles && ok; ++t) {
            float tot[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) tot[i] = 0.f;
            for (int ch = 0; ch < KB; ++ch, ++g) {
                const unsigned b = g & 1u, ta = tl + b * 256u, to = tl + (b ^ 1u) * 256u;
                ok = __all_sync(0xffffffffu, bar_wait(&sm->tfull[b], (g >> 1) & 1u, &sm->abort, err));
                if (!ok) break;
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (ch + 1 < KB) {
#pragma unroll
                    for (int c = 0; c < NC; c += 16) {
                        float v[16];
                        tmem_ld16(ta + c, v);
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {   // sum, and what it rounded off (in full where the total is the larger one)
                            const unsigned long long tt = pack2(tot[c + i], tot[c + i + 1]), uu = pack2(v[i], v[i + 1]), s = add2(tt, uu);
                            unpack2(sub2(uu, sub2(s, tt)), v[i], v[i + 1]);
                            unpack2(s, tot[c + i], tot[c + i + 1]);
                        }
                        tmem_st16(ta + c, v);
                    }
                } else {
                    // the row's last chain: the logits, with what both accumulators still owe; both start the next tile from zero
#pragma unroll
                    for (int c = 0; c < NC; c += 16) {
                        float u[16], o[16];
                        tmem_ld16(ta + c, u);
                        if (KB > 1) tmem_ld16(to + c, o);
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float s = tot[c + i] + u[i], r = (u[i] - (s - tot[c + i])) + (KB > 1 ? o[i] : 0.f);
                            tot[c + i] = fmaf(s, s_hi, fmaf(s, s_lo, r * s_hi));
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i) u[i] = tot[c + i];
                        tmem_st16(ta + c, u);
                    }
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                if (ch + 1 == KB) {
                    // softmax statistics of this third of the row, out of tensor memory again (in registers the logits unroll into
                    // code that takes longer to fetch than to run); then both accumulators start the next tile from zero
                    const int c0 = (nt0 + t) * N + grp * NG, nvalid = min(NC, a.V - c0);
                    ClHeadPartial p;
                    for (bool again = false;; again = true) {
                        p = ClHeadPartial{-INFINITY, 0.f, 0.f, 0x7fffffff};
                        bool bad = false;
#pragma unroll 1
                        for (int c = 0; c < nvalid; c += 16) {   // sums relative to the largest logit so far
                            float l[16];
                            tmem_ld16(ta + c, l);
                            float big = -INFINITY;
                            int at = 0;
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                            {   // (selections, not branches: a branch per logit costs ten times as much)
                                const bool in = c + i < nvalid;
                                bad |= in && !(fabsf(l[i]) < INFINITY);
                                l[i] = in ? fminf(fmaxf(l[i], -CL_LOGIT_CLAMP), CL_LOGIT_CLAMP) : -INFINITY;   // clamp of Section 3.1
                                at = l[i] > big ? i : at;
                                big = fmaxf(big, l[i]);
                            }
                            const float m = fmaxf(p.m, big), back = p.z > 0.f ? p.m - m : 0.f, f = expf(back);
                            p.idx = big > p.m ? c0 + c + at : p.idx;
                            p.m = m;
                            float z = 0.f, s = 0.f;
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const float d = c + i < nvalid ? l[i] - m : 0.f, e = c + i < nvalid ? expf(d) : 0.f;
                                z += e;
                                s = fmaf(d, e, s);
                            }
                            p.s = fmaf(f, fmaf(back, p.z, p.s), s);
                            p.z = fmaf(f, p.z, z);
                        }
                        if (again || !__any_sync(0xffffffffu, bad && redo)) break;
#pragma unroll 1
                        for (int c = 0; c < nvalid; ++c) {
                            const float l = tmem_ld1(ta + c);
                            const bool want = redo && !(fabsf(l) < INFINITY);
                            if (!__any_sync(0xffffffffu, want)) continue;
                            bool any;
                            const float v = special_logit(a.x + (size_t)(row0 + min(row, nrows - 1)) * a.d, a.W + (size_t)(c0 + c) * a.d, a.gain, scale, a.d, want, &any);
                            odd |= want && !any;   // a sum that overflowed
                            tmem_st1(ta + c, want && any ? v : l);
                        }
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    }
                    if (nvalid > 0) run = cl_hp_merge(run, p);
                    if (t + 1 < ntiles) {
#pragma unroll 1
                        for (int c = 0; c < NC; c += 16) {
                            tmem_st16(ta + c, zero);
                            if (KB > 1) tmem_st16(to + c, zero);
                        }
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (ch + 1 == KB && KB > 1) release(b ^ 1u);   // (held back so that it could be read once more)
                if (ch + 2 != KB) release(b);
            }
        }
        if (odd) a.flags[0] = 1u;
        // (each group's statistics go out by themselves: k_head_tc_merge adds them up in 64 bits)
        if (row < nrows) a.part[((size_t)(row0 + row) * a.NR + rg) * (CHAIN_WARPS / 4) + grp] = run;
    };
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        // ---------------- copies: warp 0 weights, warp 2 rows ----------------
        auto copies = [&](unsigned char *ring, unsigned bytes, int stages, unsigned long long *full, unsigned long long *empty, bool weights) {
            unsigned st = 0, par = 0, n = 0;
            bool ok = true;
            for (int t = 0; t < ntiles && ok; ++t)
                for (int kb = 0; kb < KB; ++kb, ++n) {
                    if (weights) {   // asked for in L2 ahead: a few K blocks in shared memory do not cover the trip to HBM
                        for (int k = kb ? kb + HTC_AHEAD : 0; k < min(kb + HTC_AHEAD + 1, KB); ++k) tma_prefetch_2d(&mapW, k * 64, (nt0 + t) * N);
                    }
                    ok = bar_wait(empty + st, par ^ 1u, &sm->abort, err);
                    if (!ok) break;
                    bar_expect(full + st, bytes);
                    if (weights) tma_load_2d(ring + st * bytes, &mapW, kb * 64, (nt0 + t) * N, full + st);
                    else
                        for (int p = 0; p < 3; ++p) tma_load_2d(ring + st * bytes + p * 16384, &mapX, kb * 64, p * a.R + row0, full + st);
                    if (++st == (unsigned)stages) { st = 0; par ^= 1u; }
                }
            // The CTA may not exit while a copy is in flight, and nobody else waits for it where another role gave up after the last one was
            // issued: wait (bounded) for the last `stages` of them, which in a pass that ends well is no wait at all.
            const unsigned long long t0 = gtime_ns();
            for (unsigned i = n > (unsigned)stages ? n - stages : 0; i < n; ++i)
                while (!bar_try(full + i % stages, (i / stages) & 1u) && gtime_ns() - t0 < WAIT_NS) {}
        };
        if (warp == 0) {
            if (lane == 0) copies(ringB, B_BYTES, HTC_BST, sm->bfull, sm->bempty, true);
        } else if (warp == 2) {
            if (lane == 0) copies(ringA, HTC_A, HTC_AST, sm->afull, sm->aempty, false);
        } else if (warp == 1 && lane == 0) {
            // ---------------- multiply-adds ----------------
            const unsigned idesc = umma_idesc(128, N);
            unsigned sa = 0, pa = 0, sb = 0, pb = 0, g = 0;
            bool ok = true;
            for (int t = 0; t < ntiles && ok; ++t)
                for (int kb = 0; kb < KB; ++kb, ++g) {
                    const unsigned b = g & 1u;
                    if (!bar_wait(&sm->tempty[b], (g >> 1) & 1u, &sm->abort, err) || !bar_wait(&sm->bfull[sb], pb, &sm->abort, err) ||
                        !bar_wait(&sm->afull[sa], pa, &sm->abort, err)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const unsigned a_addr = s_u32(ringA + sa * HTC_A), b_addr = s_u32(ringB + sb * B_BYTES), acc = tmem + b * 256u;
#pragma unroll
                    for (int p = 2; p >= 0; --p)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16(acc, umma_desc(a_addr + (unsigned)(p * 16384 + k * 32)), umma_desc(b_addr + (unsigned)(k * 32)), idesc, 1u);
                    umma_commit(&sm->aempty[sa]);
                    umma_commit(&sm->bempty[sb]);
                    umma_commit(&sm->tfull[b]);
                    if (++sa == HTC_AST) { sa = 0; pa ^= 1u; }
                    if (++sb == HTC_BST) { sb = 0; pb ^= 1u; }
                }
            // likewise the multiply-adds, before the tensor memory is given back
            umma_commit(&sm->done);
            const unsigned long long t0 = gtime_ns();
            while (!bar_try(&sm->done, 0u) && gtime_ns() - t0 < WAIT_NS) {}
        }
    } else if (warp < 8) {
        if constexpr (NG3 > 0) chains(std::integral_constant<int, NG3>(), 2);
    } else {
        chains(std::integral_constant<int, NG>(), (warp - 8) >> 2);
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// Behind k_head_tc: one warp per row, the ranges' statistics in a fixed order and in 64 bits, then Eq. 2-4.  (By the last CTA of a row tile it
// took 13 us at 100 rows, all of them on one SM.)
__global__ void __launch_bounds__(128) k_head_tc_merge(const ClHeadPartial *part, int R, int NR, double inv_log_v, float *conf, float *pmax, int *arg) {
    constexpr int PL = 7;   // partials a lane at a time: two turns of 32 * 7 cover three groups on 148 SMs
    pdl_wait();
    const int r = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= R) return;
    const float4 *pp = (const float4 *)(part + (size_t)r * NR);
    float m = -INFINITY;
    int idx = 0x7fffffff;
    double z = 0.0, t = 0.0;
    for (int g0 = lane; g0 < NR; g0 += 32 * PL) {
        float4 f[PL];
        float mn = m;
#pragma unroll
        for (int i = 0; i < PL; ++i) f[i] = g0 + 32 * i < NR ? __ldcg(pp + g0 + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < PL; ++i)
            if (f[i].y > 0.f && f[i].x > mn) { mn = f[i].x; idx = __float_as_int(f[i].w); }
        if (z > 0.0) {
            const double e = expf(m - mn);
            t = e * (t + (double)(m - mn) * z);
            z *= e;
        }
        m = mn;
#pragma unroll
        for (int i = 0; i < PL; ++i) {
            const float dm = f[i].y > 0.f ? f[i].x - m : 0.f, e = f[i].y > 0.f ? expf(dm) : 0.f;
            z += (double)(e * f[i].y);
            t += (double)(e * fmaf(dm, f[i].y, f[i].z));
        }
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, o), mm = fmaxf(m, om);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
        const double oz = __shfl_xor_sync(0xffffffffu, z, o), ot = __shfl_xor_sync(0xffffffffu, t, o);
        const double e = z > 0.0 ? expf(m - mm) : 0.f, oe = oz > 0.0 ? expf(om - mm) : 0.f;
        t = (z > 0.0 ? e * (t + (double)(m - mm) * z) : 0.0) + (oz > 0.0 ? oe * (ot + (double)(om - mm) * oz) : 0.0);
        z = e * z + oe * oz;
        idx = om > m || (om == m && oi < idx) ? oi : idx;
        m = mm;
    }
    if (lane == 0) {
        conf[r] = (float)(1.0 - (log(z) - t / z) * inv_log_v);   // H = log Z - S / Z (Eq. 2-4)
        pmax[r] = (float)(1.0 / z);
        arg[r] = idx;
    }
}

template <int N>
cudaError_t launch_tc(HeadTcArgs a, double inv_log_v, float *conf, float *pmax, int *arg, const void *W, cudaStream_t s) {
    CUtensorMap mapX, mapW;
    if (!make_map(&mapX, a.split, 3 * a.R, a.d, 128) || !make_map(&mapW, W, a.V, a.d, N)) return cudaErrorInvalidValue;
    a.NT = (a.V + N - 1) / N;
    a.NR = a.NR < a.NT ? a.NR : a.NT;
    const size_t smem = 1024 + HTC_AST * HTC_A + HTC_BST * N * 128 + sizeof(HeadTcSmem);
    cudaError_t e = cudaFuncSetAttribute(k_head_tc<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = launch_chained(k_head_tc<N>, dim3(a.MT * a.NR), HTC_THREADS, smem, 1, s, mapX, mapW, a);
    if (e != cudaSuccess) return e;
    return launch_chained(k_head_tc_merge, dim3((a.R + 3) / 4), 128, 0, 1, s, (const ClHeadPartial *)a.part, a.R, a.NR * ((N / 3 + 15) / 16 * 32 < N ? 3 : 2), inv_log_v, conf, pmax, arg);
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
        case 1:   // (fewer than 17 rows take the GEMV)
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

// Weights a tile of k_head_tc for V tokens in NR ranges: whichever lets the fullest CTA end first, a K block of N weights taken as 6 N + 500
// (by the work of the roles).  The cost is that CTA's, a K block.
static int head_tc_tile(int V, int NR, long long &cost) {
    int best = 0;
    for (int n : {224, 128, 64}) {
        const long long c = (long long)(((V + n - 1) / n + NR - 1) / NR) * (6 * n + 500);
        if (!best || c < cost) {
            best = n;
            cost = c;
        }
    }
    return best;
}

long long cl_head_tc_cost(int V, int n_sm) {
    long long cost = 0;
    head_tc_tile(V, n_sm, cost);
    return cost;
}

static void row_tiles(int R, int &MT, int &rows) {
    MT = (R + 127) / 128;
    rows = (R + MT - 1) / MT;
    MT = (R + rows - 1) / rows;
}

// Statistics of R rows on the CUDA cores.  scale: scratch [R]; part: scratch [CL_HEAD_ROWS_PARTIALS].  wdtype 0 fp32, 1 bf16; 16-byte
// aligned inputs.
cudaError_t cl_launch_head_rows(int wdtype, const void *W, const void *x, const float *gain, int R, int V, int d, float eps, int n_sm,
                                double *scale, ClHeadPartial *part, float *conf, float *pmax, int *arg, cudaStream_t s) {
    HeadRowsArgs a;
    a.W = W; a.x = x; a.gain = gain; a.scale = scale; a.R = R; a.V = V; a.d = d; a.part = part;
    row_tiles(R, a.MT, a.rows);
    a.NT = (V + HN - 1) / HN;
    a.NR = 2 * n_sm / a.MT;   // two CTAs per SM
    while (a.NR > 1 && (size_t)R * a.NR > CL_HEAD_ROWS_PARTIALS) --a.NR;
    if (a.NR > a.NT) a.NR = a.NT;
    if (a.NR < 1) a.NR = 1;
    if (wdtype == 1) k_row_scale<<<R, 256, 0, s>>>((const __nv_bfloat16 *)x, nullptr, d, eps, scale, nullptr, nullptr);
    else k_row_scale<<<R, 256, 0, s>>>((const float *)x, nullptr, d, eps, scale, nullptr, nullptr);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = wdtype == 1 ? launch_tm<__nv_bfloat16>(a, s) : launch_tm<float>(a, s);
    if (e != cudaSuccess) return e;
    k_head_rows_merge<<<(R + 3) / 4, 128, 0, s>>>(part, R, a.NR, 1.0 / log((double)V), conf, pmax, arg);
    return cudaGetLastError();
}

// The same of bf16 rows and a bf16 head on the tensor cores.  scale: scratch [R]; split: scratch of split_bytes (128 rows of d elements in
// three parts at least; calls of more rows than fit take several launches).  flags[0] != 0 after it: a sum of finite products overflowed, or
// a row's scale is beyond 2^-100 .. 2^90: the results are to be had from the other kernels; flags[1] != 0: a wait ran out.  They are
// cleared here.
cudaError_t cl_launch_head_tc(const void *W, const void *x, const float *gain, int R, int V, int d, float eps, int n_sm, double *scale, void *split, size_t split_bytes,
                              ClHeadPartial *part, unsigned *flags, float *conf, float *pmax, int *arg, cudaStream_t s) {
    const double inv_log_v = 1.0 / log((double)V);
    const int most = (int)(split_bytes / ((size_t)d * 6)) / 128 * 128;
    if (most < 128) return cudaErrorInvalidValue;
    const int chunks = (R + most - 1) / most, per = (R + chunks - 1) / chunks;
    for (int r0 = 0; r0 < R; r0 += per) {
        HeadTcArgs t;
        t.R = R - r0 < per ? R - r0 : per;
        t.x = (const __nv_bfloat16 *)x + (size_t)r0 * d; t.W = (const __nv_bfloat16 *)W; t.gain = gain; t.V = V; t.d = d; t.KB = (d + 63) / 64;
        t.split = (__nv_bfloat16 *)split;
        t.scale = scale;
        t.part = part; t.flags = flags;
        row_tiles(t.R, t.MT, t.rows);
        t.NR = n_sm / t.MT;
        while (t.NR > 1 && (size_t)t.R * t.NR * 3 > CL_HEAD_TC_PARTIALS) --t.NR;
        if (t.NR < 1) t.NR = 1;
        k_row_scale<<<t.R, 256, 0, s>>>(t.x, gain, d, eps, scale, (__nv_bfloat16 *)split, r0 ? nullptr : flags);   // (the flags are the whole call's)
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        long long cost;
        switch (head_tc_tile(V, t.NR, cost)) {
            case 224: e = launch_tc<224>(t, inv_log_v, conf + r0, pmax + r0, arg + r0, W, s); break;
            case 128: e = launch_tc<128>(t, inv_log_v, conf + r0, pmax + r0, arg + r0, W, s); break;
            default: e = launch_tc<64>(t, inv_log_v, conf + r0, pmax + r0, arg + r0, W, s);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
