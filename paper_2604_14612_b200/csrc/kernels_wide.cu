// Wide tensor-core GEMM for the prompt pass of a model stored in a 16-bit type (bf16 or fp16): the full-model pass of
// Section 3 over up to 512 prompt rows at a time, so that the weights stream from HBM once per 512 tokens instead
// of once per 8.
//
//   sum over parts of P[part, t, r] = sum_k a[t, k] * W[r, k]        a: M activation rows, W: [rows, K] 16-bit weights
//
// Activations are fp32 everywhere else; each row enters as hi = round16(v) and lo = round16(v - hi) in the weights' type
// and both products count, so the product keeps about 16 (bf16) or 22 (fp16) mantissa bits of the activation.
//   k_wide               the GEMM; its product parts are added in a fixed order by the kernel that consumes them:
//   k_wide_rope_append   q, k, v: rotary embedding at the row's position, cache append, q left in place
//   k_attn_wide          causal attention of the pass's rows over the cache -> hi/lo rows of the output projection
//   k_wide_norm          x += product (or x = E[token]); hidden tap; RMSNorm -> hi/lo rows of the next GEMM
//   k_wide_silu          h = silu(gate) * up on the interleaved gate/up product -> hi/lo rows of the down projection
// The launches of a pass are chained by programmatic dependent launch: a kernel lets its successor start at once and the
// successor waits (griddepcontrol.wait) before it touches anything another kernel writes; only weights are read earlier.
// Every wait is bounded in time.
#include <math.h>

#include <algorithm>

#include "tc_common.cuh"

namespace {

// ---- the GEMM ------------------------------------------------------------------------------------------------
// One CTA pair (cluster of 2, tcgen05 cta_group::2) computes tiles of 256 operand rows x 256 weight rows: each CTA holds
// 128 operand rows and half of the weight rows in its shared memory and the accumulator rows of its 128 operand rows
// (tensor-memory lanes) over all 256 columns.
// Bound: the tensor pipe for M > 128.  A single-CTA 128 x 256 tile has to fill 64 KB of shared memory per 64 elements of K
// and read 96 bytes of it per cycle for the multiply-adds, which held it at 1.06 PFLOP/s; the pair splits the weight rows,
// so a CTA fills 48 KB and reads 64 bytes per cycle.
//   full tile  256 token rows; per K block two products (hi, lo) into the same accumulator
//   half tile  128 token rows or fewer (the rest of M, if there is one of that size): their hi parts are the rows of CTA 0,
//              their lo parts those of CTA 1, one product per K block; the two halves of the sum are separate parts.  Half the
//              multiply-adds of a full tile, and with M <= 128, where the pass is bound by the weight stream, each SM fills
//              32 KB per K block, half of it weights.
// Work is cut evenly: the K blocks of all tiles, in tile order, are one sequence (cost 2 per block of a full tile, 1 of a
// half tile) of which every pair takes an equal contiguous share.  A share may end inside a tile: a tile's product comes in
// as many parts as pairs touched it, part = pair - first pair of the tile.  Equal shares matter: 4096 x 4096 outputs at
// M = 512 are 32 tiles for 74 pairs.
// The tensor-memory accumulator cuts off where an fp32 addition rounds: a sum loses about 2^-26 of itself per instruction, all in
// one direction.  So a chain is at most `chain` K blocks of one tile (a piece), and the pieces of a share are added in fp32 in
// the registers of the store warps.  Error of the sums against 64 bits, 512 rows x 4096 x 11008 fp16, chains of 32 / 16 / 8 / 4 blocks:
// 4.5e-6 / 2.4e-6 / 1.2e-6 / 6.6e-7; call of 512 tokens at 8 layers, chains of 16 / 8 / 4: 4.70 / 4.68 / 4.79 ms, of 61 tokens 2.10 / 2.11 / 2.17.
// (Later pieces were added in memory before, chains of 32: 4.83 ms.)  The accumulator is double-buffered (2 x 256 columns):
// reading one piece overlaps the multiply-adds of the next.
// Roles per CTA: warp 0 TMA producer (the weights of the first stages are requested before the wait for the previous
// kernel), warp 1 tensor memory and, in CTA 0, the multiply-adds, warps 2-9 add and store (thread = operand row x 128 columns,
// 32 bytes per store instruction).
constexpr int WN = 256, W_STORE_WARPS = 8, WTHREADS = 64 + 32 * W_STORE_WARPS, W_TILE = 128 * TC_BK * 2;   // 16 KB: 128 rows x 64 elements
constexpr int W_SMEM_TILES = 12;                                     // 192 KB ring: 4 stages of 3 tiles, or 6 of 2 (half tiles only)
constexpr int W_MAX_STAGES = 6;
constexpr int W_CHAIN = 8;    // K blocks (of 64 elements) per accumulation chain

struct WSmem {
    unsigned long long full[W_MAX_STAGES], empty[W_MAX_STAGES], tfull[2], tempty[2];
    unsigned tmem_base;
    int abort;
};

// The share of a pair, walked piece by piece.
struct WPiece {
    int nt, mt, kb0, kb1;   // tile and its K blocks
    bool half, last;        // last: the last piece of this share in the tile
};
struct WWalk {
    const ClWideParts &p;
    int chain, nt, mt, kb, c, c1;   // next K block; cost of all blocks before it; end of the share
    __device__ WWalk(const ClWideParts &parts, int pair, int chain_) : p(parts), chain(chain_) {
        const int T = cl_wide_cost(p), W = cl_wide_col_cost(p), c0 = (int)((long long)T * pair / p.G);
        c1 = (int)((long long)T * (pair + 1) / p.G);
        nt = c0 / W;
        const int rem = c0 - nt * W, full = 2 * p.KB * p.MT;
        if (rem < full) {
            mt = rem / (2 * p.KB);
            kb = (rem - mt * 2 * p.KB + 1) >> 1;   // a boundary inside a block of cost 2 belongs to the pair before it
        } else {
            mt = p.MT;
            kb = rem - full;
        }
        c = nt * W + (mt < p.MT ? 2 * (mt * p.KB + kb) : full + kb);
        if (kb == p.KB) step();
    }
    __device__ void step() {   // to the next tile
        kb = 0;
        if (++mt == p.MT + p.half) { mt = 0; ++nt; }
    }
    __device__ bool next(WPiece &o) {
        if (c >= c1) return false;
        o.nt = nt; o.mt = mt; o.half = mt == p.MT;
        o.kb0 = kb;
        const int left = o.half ? c1 - c : (c1 - c + 1) >> 1;
        o.kb1 = min(min(p.KB, kb + chain), kb + left);
        c += (o.kb1 - kb) * (o.half ? 1 : 2);
        kb = o.kb1;
        o.last = kb == p.KB || c >= c1;
        if (kb == p.KB) step();
        return true;
    }
};

__global__ void __launch_bounds__(WTHREADS, 1)
k_wide(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, const __grid_constant__ ClWideArgs a) {
    const int stage_tiles = a.p.MT ? 3 : 2, stages = W_SMEM_TILES / stage_tiles, stage_bytes = stage_tiles * W_TILE;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *tiles = (unsigned char *)(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    WSmem *sm = (WSmem *)(tiles + (size_t)W_SMEM_TILES * W_TILE);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank(), pair = blockIdx.x >> 1;

    if (tid == 0) {
        for (int i = 0; i < W_MAX_STAGES; ++i) {
            bar_init(&sm->full[i], 1);
            bar_init(&sm->empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(&sm->tfull[i], 1);
            bar_init(&sm->tempty[i], 2 * W_STORE_WARPS);   // the store warps of both CTAs
        }
        sm->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s_u32(&sm->tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();   // the peer's barriers exist before anything signals them
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    pdl_launch_dependents();
    const unsigned tmem = *(volatile unsigned *)&sm->tmem_base;

    WWalk walk(a.p, pair, a.chain);
    WPiece pc;
    if (warp == 0) {
        // ---------------- TMA producer: this CTA's operand rows and its half of the weight rows ----------------
        if (lane == 0) {
            auto load_b = [&](const WPiece &t, int kb, int s) {
                if (rank == 0) bar_expect(&sm->full[s], 2 * (t.half ? 2 : 3) * W_TILE);   // both CTAs' copies count on CTA 0's barrier
                tma_load_2d_pair(tiles + (size_t)s * stage_bytes + (stage_tiles - 1) * W_TILE, &mapB, kb * TC_BK,
                                 t.nt * WN + rank * 128, &sm->full[s]);
            };
            auto load_a = [&](const WPiece &t, int kb, int s) {
                unsigned char *dst = tiles + (size_t)s * stage_bytes;
                if (t.half) {
                    tma_load_2d_pair(dst, &mapA, kb * TC_BK, t.mt * 256 + rank * a.lo_row0, &sm->full[s]);
                } else {
                    tma_load_2d_pair(dst, &mapA, kb * TC_BK, t.mt * 256 + rank * 128, &sm->full[s]);
                    tma_load_2d_pair(dst + W_TILE, &mapA, kb * TC_BK, a.lo_row0 + t.mt * 256 + rank * 128, &sm->full[s]);
                }
            };
            // the weights of the first stages before the operand rows, which come from the previous kernel
            int n_pre = 0;
            {
                WWalk w(walk);
                while (n_pre < stages && w.next(pc))
                    for (int kb = pc.kb0; kb < pc.kb1 && n_pre < stages; ++kb) load_b(pc, kb, n_pre++);
            }
            pdl_wait();
            bool ok = true;
            int s = 0, i = 0;
            unsigned par = 1u;
            while (ok && walk.next(pc)) {
                for (int kb = pc.kb0; kb < pc.kb1; ++kb, ++i) {
                    if (i >= n_pre) {
                        if (!bar_wait(&sm->empty[s], par, &sm->abort, a.err)) { ok = false; break; }
                        load_b(pc, kb, s);
                    }
                    load_a(pc, kb, s);
                    if (++s == stages) { s = 0; par ^= 1u; }
                }
            }
            if (!ok) {   // gave up: let the copies in flight land (they signal CTA 0, so this CTA can only give them time)
                const unsigned long long t0 = gtime_ns();
                while (gtime_ns() - t0 < 2000000ull) {}
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (CTA 0, for both) ----------------
        if (lane == 0 && rank == 0) {
            const unsigned idesc = umma_idesc(256, WN, a.f16);
            int s = 0, n = 0;
            unsigned par = 0u;
            bool ok = true;
            pdl_wait();   // (operand rows cannot arrive earlier, and the time limits below are for this kernel's own work)
            while (ok && walk.next(pc)) {
                const unsigned b = (unsigned)n & 1u, acc = tmem + b * WN;
                if (!bar_wait(&sm->tempty[b], ((unsigned)(n >> 1) & 1u) ^ 1u, &sm->abort, a.err)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int kb = pc.kb0; kb < pc.kb1; ++kb) {
                    if (!bar_wait(&sm->full[s], par, &sm->abort, a.err)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const unsigned hi_addr = s_u32(tiles + (size_t)s * stage_bytes), b_addr = hi_addr + (stage_tiles - 1) * W_TILE;
#pragma unroll
                    for (int k = 0; k < TC_BK / 16; ++k) {
                        umma_pair(acc, umma_desc(hi_addr + k * 32), umma_desc(b_addr + k * 32), idesc, (unsigned)((kb - pc.kb0) | k));
                        if (!pc.half) umma_pair(acc, umma_desc(hi_addr + W_TILE + k * 32), umma_desc(b_addr + k * 32), idesc, 1u);
                    }
                    umma_commit_pair(&sm->empty[s]);   // free in both CTAs once these multiply-adds have read it
                    if (++s == stages) { s = 0; par ^= 1u; }
                }
                if (ok) umma_commit_pair(&sm->tfull[b]);
                ++n;
            }
        }
    } else {
        // ---------------- add and store: one thread per operand row and half of the columns ----------------
        constexpr int WC = WN * 4 / W_STORE_WARPS;   // columns of a warp
        const int q = warp & 3, colw = ((warp - 2) >> 2) * WC;   // q: the tensor-memory lane quadrant this warp may read
        float sum[WC];   // of the pieces so far of this share's tile
#pragma unroll
        for (int i = 0; i < WC; ++i) sum[i] = 0.f;
        pdl_wait();   // the previous kernel may still read the product buffer
        for (int n = 0; walk.next(pc); ++n) {
            const unsigned b = (unsigned)n & 1u;
            if (!bar_wait(&sm->tfull[b], (unsigned)(n >> 1) & 1u, &sm->abort, a.err)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int c = 0; c < WC; c += 16) {   // (16 at a time: 128 sums and 32 values loaded do not fit the 168 registers)
                float v[16];
                tmem_ld16(tmem + b * WN + ((unsigned)(q * 32) << 16) + (unsigned)(colw + c), v);
#pragma unroll
                for (int i = 0; i < 16; ++i) sum[c + i] += v[i];
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive_rank0(&sm->tempty[b]);
            if (!pc.last) continue;   // (uniform)
            const int t = pc.mt * 256 + q * 32 + lane + (pc.half ? 0 : rank * 128);
            if (t < a.p.M) {
                int part = pair - cl_wide_owner(a.p, pc.nt, pc.mt, 0);
                if (pc.half) part = 2 * part + rank;
                const int col0 = pc.nt * WN + colw;
                float *dst = a.p.P + ((size_t)part * a.p.M + (size_t)t) * a.p.rows + col0;
#pragma unroll
                for (int i = 0; i < WC; i += 8)
                    if (col0 + i + 8 <= a.p.rows) st_global_v8(dst + i, sum + i);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < WC; ++i) sum[i] = 0.f;
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();   // CTA 0's multiply-adds read CTA 1's shared memory, and both signal each other's barriers
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// Number of product parts at (row t, column col): the pairs that share the tile, twice in a half tile.
__device__ __forceinline__ int wide_parts(const ClWideParts &p, int t, int col) {
    const int nt = col >> 8, mt = t >> 8;
    return (cl_wide_owner(p, nt, mt, p.KB - 1) - cl_wide_owner(p, nt, mt, 0) + 1) << (mt == p.MT);
}

// One CTA per token row: x[t] = E[token] or x[t] += product parts (added in part order); the optional hidden tap;
// then the rows of the next GEMM: hi/lo(x * rsqrt(mean x^2 + eps) * g).  A thread's elements stay in registers between the two
// passes: KEEP chunks of 4, read side by side, part by part, before anything is written (a store between the loads would order
// them); of rows longer than KEEP * 4 * THREADS elements the rest is read again.
// Bound: L2 (parts and stream in, stream and two operand rows out).  Rows that do not all fit on the chip at once cost a second
// wave, few rows want many loads in flight each, so KEEP is the least of 1, 2, 4 that leaves one wave (cl_launch_wide_norm).
// us, within a pass, KEEP 1 / 2 / 4: width 4096, 61 rows 6.0 / 7.7 / 11.9, 200 rows 8.5 / 6.2 / 9.5, 512 rows 14.8 / 10.0 / 9.3; width
// 5120, 400 rows 16.5 / 12.0 / 8.8; width 768, 512 rows 4.7 / 6.5 / 9.0.
template <int KEEP, int THREADS, int AHEAD>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_wide_norm(ClWideNormArgs a) {
    __shared__ float red[32];
    pdl_launch_dependents();
    const int t = blockIdx.x, tid = threadIdx.x, d = a.d, span = 4 * blockDim.x;   // columns per round of the CTA
    float *xr = a.x + (size_t)t * d;
    float4 gain[KEEP];
    auto gains = [&]() {   // (weights: they may be read ahead of the wait)
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
            const int i = tid * 4 + k * span;
            gain[k] = a.g && i < d ? __ldg((const float4 *)(a.g + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    if (KEEP <= 2) gains();
    pdl_wait();
    const unsigned short *er = a.tok ? (const unsigned short *)a.embed + (size_t)a.tok[t] * d : nullptr;
    // only the last tap_P rows of the pass reach the ring: an earlier row of the same slot would be overwritten anyway
    unsigned short *tap = nullptr;
    if (a.tap && t >= a.M - a.tap_P) tap = (unsigned short *)a.tap + (size_t)((a.st->ctx + t) % a.tap_P) * d;
    const size_t plane = (size_t)a.M * d;
    float ss = 0.f;
    float4 keep[KEEP];
    auto read = [&](int i0, int n_chunks) {   // the updated stream at columns i0 + tid * 4 + k * span .. + 3 -> keep[k]
        int n[KEEP], nmax = 0;
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
            const int i = i0 + tid * 4 + k * span;
            const bool in = k < n_chunks && i < d;
            n[k] = 0;
            keep[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (in && er) {
                const uint2 u = *(const uint2 *)(er + i);
                pair16_to_f32(u.x, a.f16, keep[k].x, keep[k].y);
                pair16_to_f32(u.y, a.f16, keep[k].z, keep[k].w);
            } else if (in) {
                keep[k] = *(const float4 *)(xr + i);
                n[k] = wide_parts(a.parts, t, i);
                nmax = max(nmax, n[k]);
            }
        }
        const float *p0 = a.parts.P + (size_t)t * d + i0 + tid * 4;
#pragma unroll AHEAD
        for (int s = 0; s < nmax; ++s) {
            float4 p[KEEP];
#pragma unroll
            for (int k = 0; k < KEEP; ++k) p[k] = s < n[k] ? __ldcg((const float4 *)(p0 + (size_t)s * plane + k * span)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < KEEP; ++k) {
                keep[k].x += p[k].x; keep[k].y += p[k].y; keep[k].z += p[k].z; keep[k].w += p[k].w;
            }
        }
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
            const int i = i0 + tid * 4 + k * span;
            const float4 v = keep[k];
            ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss); ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss);
            if (k < n_chunks && i < d) {
                *(float4 *)(xr + i) = v;
                if (tap) {
                    const unsigned lo2 = (unsigned)f32_to_b16(v.x, a.f16) | ((unsigned)f32_to_b16(v.y, a.f16) << 16);
                    const unsigned hi2 = (unsigned)f32_to_b16(v.z, a.f16) | ((unsigned)f32_to_b16(v.w, a.f16) << 16);
                    *(uint2 *)(tap + i) = make_uint2(lo2, hi2);
                }
            }
        }
    };
    for (int i0 = KEEP * span; i0 < d; i0 += span) read(i0, 1);   // (what does not stay in registers first)
    read(0, KEEP);
    if (!a.g) return;   // uniform
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((tid & 31) == 0) red[tid >> 5] = ss;
    if (KEEP > 2) gains();
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];   // fixed order
    const float sc = 1.0f / sqrtf(tot / (float)d + a.eps);
    __nv_bfloat16 *hi = a.A + (size_t)t * d, *lo = a.A + (size_t)(a.lo_row0 + t) * d;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
        const int i = tid * 4 + k * span;
        if (i < d) store_split4(hi + i, lo + i, keep[k].x * sc * gain[k].x, keep[k].y * sc * gain[k].y, keep[k].z * sc * gain[k].z,
                                keep[k].w * sc * gain[k].w, a.f16);
    }
    for (int i = tid * 4 + KEEP * span; i < d; i += span) {
        const float4 v = *(const float4 *)(xr + i);   // this thread's own writes
        const float4 g = *(const float4 *)(a.g + i);
        store_split4(hi + i, lo + i, v.x * sc * g.x, v.y * sc * g.y, v.z * sc * g.z, v.w * sc * g.w, a.f16);
    }
}

// One item = the four rotary pairs (i .. i + 3, + hd / 2) of one head of one row: q heads first, then k heads, then the
// same shape over v (no rotation).  Rotary embedding at position ctx + t; q goes back in place (part 0), k and v go to the
// cache [kv head][position][hd].  grid (M, ceil(items / 256)).
__global__ void __launch_bounds__(256) k_wide_rope_append(ClWideParts p, int hd, int d, int Hkv, const float2 *rope_cs,
                                                          unsigned short *kcache, unsigned short *vcache, int max_seq,
                                                          const ClDevState *st, int f16) {
    pdl_launch_dependents();
    pdl_wait();
    const int t = blockIdx.x, half = hd >> 1, per_head = half >> 2, H = d / hd;
    const int item = blockIdx.y * 256 + threadIdx.x;
    const int head = item / per_head, i = (item - head * per_head) * 4;
    const int pos = st->ctx + t;
    if (head >= H + 2 * Hkv || pos >= max_seq) return;
    const int ld = p.rows, col = head * hd + i;   // [q heads | k heads | v heads]
    const size_t plane = (size_t)p.M * ld;
    float *row = p.P + (size_t)t * ld;
    auto total = [&](int c) {
        const int n = wide_parts(p, t, c);
        float4 v = __ldcg((const float4 *)(row + c));
#pragma unroll 2
        for (int s = 1; s < n; ++s) {
            const float4 w = __ldcg((const float4 *)(row + (size_t)s * plane + c));
            v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
        return v;
    };
    float4 x = total(col), y = total(col + half);
    if (head < H + Hkv) {
        const float4 c01 = *(const float4 *)(rope_cs + (size_t)pos * half + i), c23 = *(const float4 *)(rope_cs + (size_t)pos * half + i + 2);
        const float4 a = x, b = y;
        x = make_float4(a.x * c01.x - b.x * c01.y, a.y * c01.z - b.y * c01.w, a.z * c23.x - b.z * c23.y, a.w * c23.z - b.w * c23.w);
        y = make_float4(b.x * c01.x + a.x * c01.y, b.y * c01.z + a.y * c01.w, b.z * c23.x + a.z * c23.y, b.w * c23.z + a.w * c23.w);
    }
    if (head < H) {
        *(float4 *)(row + col) = x;
        *(float4 *)(row + col + half) = y;
        return;
    }
    unsigned short *dst = (head < H + Hkv ? kcache + ((size_t)(head - H) * max_seq + pos) * hd
                                          : vcache + ((size_t)(head - H - Hkv) * max_seq + pos) * hd) + i;
    auto pack = [&](const float4 &v) {
        return make_uint2((unsigned)f32_to_b16(v.x, f16) | ((unsigned)f32_to_b16(v.y, f16) << 16),
                          (unsigned)f32_to_b16(v.z, f16) | ((unsigned)f32_to_b16(v.w, f16) << 16));
    };
    *(uint2 *)dst = pack(x);
    *(uint2 *)(dst + half) = pack(y);
}

// ---- causal attention of the rows of the pass over the cache -------------------------------------------------
// grid (H, blocks of 64 rows), 4 warps of 16 rows each.  Row t sits at position ctx + t and attends to the keys 0 .. ctx + t
// (its own key is already in the cache).  Keys and values are walked 64 at a time through two shared-memory buffers
// (cp.async, 16-byte pieces permuted by row & 7), with the usual running maximum and sum per row.
// Both products run on the tensor cores although the queries and the probabilities are fp32: each enters as three parts
// of the storage type (keys and values are of that type already) that hold at least 24 bits of it.  fp16 has the exponents for
// that only with scaling: a query row is multiplied by a power of two that brings its largest element to [2^14, 2^15) (bf16: to
// [1, 2)), a probability by 2^14, and of a probability each part is 2^12 times what the parts before it left, so that weights
// down to 2^-38 of the row's largest keep 24 bits (ATT_STEP).
// The sums are as exact as fp32 multiply-adds (relative error against 64 bits at 512 rows after 512 / 64 rows after 4032 keys:
// 6.9e-7 / 1.4e-6 with those, 4.0e-7 / 7.4e-7 here, fp16): the accumulator of the instruction cuts off where an fp32 addition rounds, which
// over one chain for all keys of a row came to 2.2e-6 / 9.9e-6, so a chain is one tile of 64 keys, the parts have accumulators of their own,
// a score's chain is cut in two (one chain: 4.9e-7 / 8.0e-7) and everything else is added in fp32.
// Bound: multiply-add issue (384 instructions of 16 x 8 x 16 per warp and key tile, 8.4 cycles each at best) and the ALU work between them, which
// two warps per scheduler hardly overlap: at 512 rows after 512 of 32 heads 143000 cycles, 68000 of them multiply-adds.  So the
// instructions beside them count: chains start from a zero operand, masks are applied only where a key may lie ahead,
// fragment addresses flip bits of one base.  512 rows of 32 heads 53 -> 40 us, the pass after it 97 -> 78, 333 rows 38 -> 30.
// (A weight is expf of the exact difference.  ex2 of s * log2(e) less the rounded m * log2(e) takes 37, 73 and 28 us, but that rounding differs
// from tile to tile as the maximum rises, 2^-25 of the score, and at scores of 2^26 a weight could be 2^7: no number in fp16.)
// Key tiles dealt out evenly over the CTAs, jobs cut where shares end: 41 us (a cut costs more than the balance gains); eight warps of 32
// keys: 45.  Blocks of late rows see the most keys and are scheduled first.
constexpr int AQ = 64, AK = 64;   // rows per CTA, keys per tile

template <int HD>
constexpr size_t attn_wide_smem() { return (size_t)(3 * AQ + 4 * AK) * HD * 2 + AQ * 4; }

__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_t(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
template <int HD, int F16>
__global__ void __launch_bounds__(128, 2)
k_attn_wide(const float *q, int ld_q, const unsigned short *kcache, const unsigned short *vcache, __nv_bfloat16 *out_b,
            int lo_row0, int M, int d, int H, int Hkv, int max_seq, const ClDevState *st) {
    constexpr int RB = HD * 2, NC = HD / 8;           // bytes and 16-byte pieces per row
    constexpr unsigned TOP = F16 ? 14 : 0;            // exponent of the largest element of a scaled query row, and of a weight of 1
    constexpr int STEP = F16 ? ATT_STEP : 1;
    constexpr float PSCALE = F16 ? 16384.f : 1.f;
    extern __shared__ __align__(1024) unsigned char asm_[];   // (fragment addresses flip bits 4 .. 8)
    unsigned char *Qs = asm_;                          // [3][AQ][RB] parts of the scaled queries
    float *rs = (float *)(asm_ + (3 * AQ + 4 * AK) * RB);   // [AQ] what a row's scores are multiplied by
    const unsigned q_addr = s_u32(Qs), kv_addr = q_addr + 3 * AQ * RB;   // [2 buffers][keys | values][AK][RB]
    pdl_launch_dependents();
    pdl_wait();
    const int h = blockIdx.x, r0 = ((int)gridDim.y - 1 - (int)blockIdx.y) * AQ;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ctx = st->ctx;
    const int nkeys = min(ctx + min(r0 + AQ, M), max_seq), ntiles = (nkeys + AK - 1) / AK;
    const int kvh = h / (H / Hkv);
    const unsigned short *Kc = kcache + (size_t)kvh * max_seq * HD, *Vc = vcache + (size_t)kvh * max_seq * HD;

    auto load_tile = [&](int tile) {
        const unsigned base = kv_addr + (unsigned)(tile & 1) * 2 * AK * RB;
        for (int i = tid; i < AK * NC; i += 128) {
            const int key = i / NC, c = i % NC, src = min(tile * AK + key, nkeys - 1);
            const unsigned dst = base + key * RB + ((c ^ (key & 7)) << 4), n = tile * AK + key < nkeys ? 16u : 0u;   // (zeros past the end)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(Kc + (size_t)src * HD + c * 8), "r"(n) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + AK * RB), "l"(Vc + (size_t)src * HD + c * 8), "r"(n) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load_tile(0);

    // this warp's 16 query rows: scaled to [2^TOP, 2^(TOP + 1)) by a power of two, split, stored; nobody else reads them
    constexpr int EL = HD / 32;
#pragma unroll 1
    for (int r8 = 0; r8 < 16; r8 += 8) {
        float v[8][EL];
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {   // (eight rows' loads at once)
            const float *src = q + (size_t)min(r0 + warp * 16 + r8 + rr, M - 1) * ld_q + h * HD + lane * EL;
            if (EL == 4) {
                const float4 x = __ldcg((const float4 *)src);
                v[rr][0] = x.x; v[rr][1] = x.y; v[rr][2 % EL] = x.z; v[rr][3 % EL] = x.w;
            } else {
                const float2 x = __ldcg((const float2 *)src);
                v[rr][0] = x.x; v[rr][1] = x.y;
            }
        }
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
            const int row = warp * 16 + r8 + rr;
            float amax = 0.f;
#pragma unroll
            for (int e = 0; e < EL; ++e) {
                if (r0 + row >= M) v[rr][e] = 0.f;
                amax = fmaxf(amax, fabsf(v[rr][e]));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            const unsigned ex = min(max(__float_as_uint(amax) >> 23, 1u + TOP), 253u);
            const float inv = __uint_as_float((254u + TOP - ex) << 23);
#pragma unroll
            for (int e = 0; e < EL; e += 2) {
                unsigned s3[3];
                split3<F16, 1>(v[rr][e] * inv, v[rr][e + 1] * inv, s3);
                const int byte = (lane * EL + e) * 2;
#pragma unroll
                for (int p = 0; p < 3; ++p)
                    *(unsigned *)(Qs + (size_t)(p * AQ + row) * RB + (((byte >> 4) ^ (row & 7)) << 4) + (byte & 15)) = s3[p];
            }
            if (lane == 0) rs[row] = __uint_as_float((ex - TOP) << 23) * rsqrtf((float)HD);
        }
    }
    __syncwarp();

    const int lr = lane >> 2, lc = (lane & 3) * 2;     // accumulator: rows lr and lr + 8, columns lc and lc + 1 of a tile of 8
    const int mrow = lane & 7, mi = lane >> 3;         // ldmatrix: this lane's row and matrix
    const int row_a = r0 + warp * 16 + lr, pos_a = row_a < M ? ctx + row_a : -1, pos_b = row_a + 8 < M ? ctx + row_a + 8 : -1;
    const float rs_a = rs[warp * 16 + lr], rs_b = rs[warp * 16 + lr + 8];
    const int pos_first = r0 + warp * 16 + 15 < M ? ctx + r0 + warp * 16 : -1;   // every row of the warp sees the keys up to here
    float o[HD / 8][4], m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;

    for (int t = 0; t < ntiles; ++t) {
        if (t + 1 < ntiles) {
            load_tile(t + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const int k0 = t * AK;
        const unsigned ka = kv_addr + (unsigned)(t & 1) * 2 * AK * RB, va = ka + AK * RB;
        float s[AK / 8][4], u[AK / 8][4], w[AK / 8][4];   // products of the queries' first parts (in two chains) and of the two others
        const unsigned q_lane = q_addr + (warp * 16 + (mi & 1) * 8 + mrow) * RB + (((mi >> 1) ^ mrow) << 4);   // (piece ^ row & 7: ks only flips bits of it)
        const unsigned k_lane = ka + ((mi >> 1) * 8 + mrow) * RB + (((mi & 1) ^ mrow) << 4);
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
            unsigned qa[3][4];
#pragma unroll
            for (int p = 0; p < 3; ++p) ldsm4(qa[p], (q_lane ^ (ks << 5)) + p * AQ * RB);
#pragma unroll
            for (int np = 0; np < AK / 16; ++np) {
                unsigned kb[4];
                ldsm4(kb, (k_lane ^ (ks << 5)) + np * 16 * RB);
#pragma unroll
                for (int p = 2; p >= 0; --p)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        float(&acc)[4] = p != 0 ? u[2 * np + j] : ks < HD / 32 ? s[2 * np + j] : w[2 * np + j];
                        if ((ks == 0 && p != 1) || (ks == HD / 32 && p == 0)) mma16816_zero<F16>(acc, qa[p], kb[2 * j], kb[2 * j + 1]);
                        else mma16816<F16>(acc, qa[p], kb[2 * j], kb[2 * j + 1]);
                    }
            }
        }
        float odd = 0.f;
#pragma unroll
        for (int n = 0; n < AK / 8; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                s[n][e] = (s[n][e] + (w[n][e] + u[n][e])) * (e < 2 ? rs_a : rs_b);
                odd = fmaf(s[n][e], 0.f, odd);   // (not zero once a score is infinite or no number; 3 % of the kernel)
            }
        if (__any_sync(0xffffffffu, odd != 0.f)) {
            // An infinite key or query: parts of it are zeros and infinities of both signs, whose products add up to no number
            // where the score is infinite or finite.  This tile's scores anew, from whole queries.
            const float *qa = q + (size_t)min(row_a, M - 1) * ld_q + h * HD, *qb = q + (size_t)min(row_a + 8, M - 1) * ld_q + h * HD;
            const float scale = rsqrtf((float)HD);
#pragma unroll
            for (int n = 0; n < AK / 8; ++n) s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
#pragma unroll 1
            for (int i = 0; i < HD; ++i) {
                const float xa = __ldcg(qa + i) * scale, xb = __ldcg(qb + i) * scale;
#pragma unroll
                for (int n = 0; n < AK / 8; ++n)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int key = n * 8 + lc + e;
                        unsigned short raw;
                        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(raw) : "r"(ka + key * RB + (((i >> 3) ^ (key & 7)) << 4) + (i & 7) * 2) : "memory");
                        const float kv = b16_to_f32(raw, F16);
                        s[n][e] = fmaf(xa, kv, s[n][e]);
                        s[n][2 + e] = fmaf(xb, kv, s[n][2 + e]);
                    }
            }
#pragma unroll
            for (int n = 0; n < AK / 8; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[n][e] = s[n][e] > -INFINITY ? s[n][e] : -INFINITY;   // (no number: no weight)
        }
        float mx_a = m_a, mx_b = m_b;
        if (k0 + AK - 1 > pos_first) {   // (uniform over the warp; a row past M is behind all keys)
#pragma unroll
            for (int n = 0; n < AK / 8; ++n) {
                const int key = k0 + n * 8 + lc;
                s[n][0] = key <= pos_a ? s[n][0] : -INFINITY;
                s[n][1] = key + 1 <= pos_a ? s[n][1] : -INFINITY;
                s[n][2] = key <= pos_b ? s[n][2] : -INFINITY;
                s[n][3] = key + 1 <= pos_b ? s[n][3] : -INFINITY;
            }
        }
#pragma unroll
        for (int n = 0; n < AK / 8; ++n) {
            mx_a = fmaxf(mx_a, fmaxf(s[n][0], s[n][1]));
            mx_b = fmaxf(mx_b, fmaxf(s[n][2], s[n][3]));
        }
#pragma unroll
        for (int w = 1; w <= 2; w <<= 1) {
            mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, w));
            mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, w));
        }
        // (a row past M, or one whose scores are all -inf so far, keeps weights of 0)
        const float ba = mx_a > -INFINITY ? mx_a : 0.f, bb = mx_b > -INFINITY ? mx_b : 0.f;
        const float ra = expf(m_a - ba), rb = expf(m_b - bb);   // (0 while the maximum is -inf)
        m_a = mx_a;
        m_b = mx_b;
        float sa = 0.f, sb = 0.f;
#pragma unroll
        for (int n = 0; n < AK / 8; ++n) {
            s[n][0] = expf(s[n][0] - ba); s[n][1] = expf(s[n][1] - ba);
            s[n][2] = expf(s[n][2] - bb); s[n][3] = expf(s[n][3] - bb);
            sa += s[n][0] + s[n][1];
            sb += s[n][2] + s[n][3];
        }
        l_a = fmaf(l_a, ra, sa);   // (this lane's columns; added over the four lanes of a row at the end)
        l_b = fmaf(l_b, rb, sb);
        unsigned pa[AK / 16][3][4];
#pragma unroll
        for (int ks = 0; ks < AK / 16; ++ks) {
            unsigned s3[3];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float *w = &s[2 * ks + (e >> 1)][(e & 1) * 2];
                split3<F16, STEP>(w[0] * PSCALE, w[1] * PSCALE, s3);
                pa[ks][0][e] = s3[0]; pa[ks][1][e] = s3[1]; pa[ks][2][e] = s3[2];
            }
        }
        const unsigned v_lane = va + ((mi & 1) * 8 + mrow) * RB + (((mi >> 1) ^ mrow) << 4);
#pragma unroll
        for (int np = 0; np < HD / 16; ++np) {
            float c[3][2][4];   // this tile's sums, part by part (bf16: the two lower parts together, the lowest first)
            constexpr int LOW = F16 ? 2 : 1;
#pragma unroll
            for (int ks = 0; ks < AK / 16; ++ks) {
                unsigned vb[4];
                ldsm4_t(vb, (v_lane ^ (np << 5)) + ks * 16 * RB);
#pragma unroll
                for (int p = 2; p >= 0; --p)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        float(&acc)[4] = c[p == 2 ? LOW : p][j];
                        if (ks == 0 && (F16 || p != 1)) mma16816_zero<F16>(acc, pa[ks][p], vb[2 * j], vb[2 * j + 1]);
                        else mma16816<F16>(acc, pa[ks][p], vb[2 * j], vb[2 * j + 1]);
                    }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int j = i / 4, e = i % 4;
                const float low = F16 ? fmaf(c[2][j][e], 1.f / STEP, c[1][j][e]) : c[1][j][e], t = fmaf(low, 1.f / STEP, c[0][j][e]);
                o[2 * np + j][e] = fmaf(o[2 * np + j][e], e < 2 ? ra : rb, t);
            }
        }
        __syncthreads();   // everyone is done with this buffer: the load after next may overwrite it
    }
#pragma unroll
    for (int w = 1; w <= 2; w <<= 1) {
        l_a += __shfl_xor_sync(0xffffffffu, l_a, w);
        l_b += __shfl_xor_sync(0xffffffffu, l_b, w);
    }
    const float ia = 1.f / (l_a * PSCALE), ib = 1.f / (l_b * PSCALE);   // (exact: a power of two)
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) {
        const size_t col = (size_t)h * HD + n * 8 + lc;
        auto put = [&](int row, float x, float y) {
            unsigned short xh, xl, yh, yl;
            split_b16(x, F16, xh, xl);
            split_b16(y, F16, yh, yl);
            *(unsigned *)(out_b + (size_t)row * d + col) = (unsigned)xh | ((unsigned)yh << 16);
            *(unsigned *)(out_b + (size_t)(lo_row0 + row) * d + col) = (unsigned)xl | ((unsigned)yl << 16);
        };
        if (row_a < M) put(row_a, o[n][0] * ia, o[n][1] * ia);
        if (row_a + 8 < M) put(row_a + 8, o[n][2] * ib, o[n][3] * ib);
    }
}

// grid (M, ceil(F / 1024)): the gate/up product has rows interleaved (2 i = gate_i, 2 i + 1 = up_i); a thread takes four.
__global__ void __launch_bounds__(256) k_wide_silu(ClWideParts p, int F, __nv_bfloat16 *A, int lo_row0, int f16) {
    pdl_launch_dependents();
    pdl_wait();
    const int t = blockIdx.x, i = (blockIdx.y * 256 + threadIdx.x) * 4;
    if (i >= F) return;   // (F is a multiple of 8)
    const int n = wide_parts(p, t, 2 * i);   // (eight consecutive columns lie in one tile)
    const size_t plane = (size_t)p.M * 2 * F;
    const float *src = p.P + (size_t)t * 2 * F + 2 * i;
    float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
#pragma unroll 2
    for (int s = 0; s < n; ++s) {
        const float4 x = __ldcg((const float4 *)(src + (size_t)s * plane)), y = __ldcg((const float4 *)(src + (size_t)s * plane) + 1);
        u.x += x.x; u.y += x.y; u.z += x.z; u.w += x.w;
        v.x += y.x; v.y += y.y; v.z += y.z; v.w += y.w;
    }
    auto h = [](float g, float up) { return g / (1.f + expf(-g)) * up; };
    store_split4(A + (size_t)t * F + i, A + (size_t)(lo_row0 + t) * F + i, h(u.x, u.y), h(u.z, u.w), h(v.x, v.y), h(v.z, v.w), f16);
}

}  // namespace

// How a GEMM of M operand rows is cut: one CTA pair per two SMs, fewer when there is so little work that a pair's share would
// cost less than four (two K blocks of a full tile, four of a half tile), or when the product parts would not fit the workspace.
ClWideParts cl_wide_plan(int M, int rows, int KB, int n_sm, float *P, size_t ws_floats) {
    ClWideParts p;
    p.P = P; p.M = M; p.rows = rows; p.KB = KB;
    const int rest = M % 256;
    p.MT = M / 256 + (rest > 128);
    p.half = rest > 0 && rest <= 128;
    p.NT = (rows + WN - 1) / WN;
    p.G = std::max(1, std::min(n_sm / 2, cl_wide_cost(p) / 4));
    auto max_parts = [&]() {
        int m = 0;
        for (int nt = 0; nt < p.NT; ++nt)
            for (int mt = 0; mt < p.MT + p.half; ++mt)
                m = std::max(m, (cl_wide_owner(p, nt, mt, KB - 1) - cl_wide_owner(p, nt, mt, 0) + 1) << (mt == p.MT));
        return m;
    };
    while (p.G > 1 && (size_t)max_parts() * M * rows > ws_floats) --p.G;
    return p;
}

cudaError_t cl_launch_wide(const ClTensorMap &mapA, const ClTensorMap &mapB, const ClWideParts &p, int lo_row0, int *err, int f16,
                           cudaStream_t s) {
    const size_t smem = (size_t)W_SMEM_TILES * W_TILE + sizeof(WSmem) + 1024;
    ClWideArgs a;
    a.p = p; a.lo_row0 = lo_row0; a.err = err; a.f16 = f16; a.chain = W_CHAIN;
    if (p.rows % 8 || p.M < 1 || p.M > CL_WIDE_MAX_M) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_wide, dim3(2 * p.G), WTHREADS, smem, 2, s, *(const CUtensorMap *)mapA.bytes, *(const CUtensorMap *)mapB.bytes, a);
}

cudaError_t cl_launch_wide_norm(const ClWideNormArgs &a, int n_sm, cudaStream_t s) {
    if (a.d % 4) return cudaErrorInvalidValue;
    const int chunks = a.d / 4;
    auto launch = [&](void (*kern)(ClWideNormArgs), int keep, int most) {
        return launch_chained(kern, dim3(a.M), std::min(most, ((chunks + keep - 1) / keep + 31) / 32 * 32), 0, 1, s, a);
    };
    // as few chunks a thread as leave all rows on the chip at once (64 registers: 1024 threads an SM)
    auto fits = [&](int keep) { return chunks <= keep * 1024 && a.M <= n_sm * (1024 / ((chunks + keep - 1) / keep)); };
    if (fits(1)) return launch(k_wide_norm<1, 1024, 4>, 1, 1024);
    if (fits(2)) return launch(k_wide_norm<2, 1024, 2>, 2, 1024);
    return launch(k_wide_norm<4, 512, 2>, 4, 512);
}

cudaError_t cl_launch_wide_rope_append(const ClWideParts &p, int H, int Hkv, int hd, int d, const float2 *rope_cs, void *kcache,
                                       void *vcache, int max_seq, const ClDevState *st, int f16, cudaStream_t s) {
    const int items = (H + 2 * Hkv) * (hd / 8);
    return launch_chained(k_wide_rope_append, dim3(p.M, (items + 255) / 256), 256, 0, 1, s, p, hd, d, Hkv, rope_cs,
                          (unsigned short *)kcache, (unsigned short *)vcache, max_seq, st, f16);
}

cudaError_t cl_launch_wide_silu(const ClWideParts &p, int F, __nv_bfloat16 *A, int lo_row0, int f16, cudaStream_t s) {
    return launch_chained(k_wide_silu, dim3(p.M, (F + 1023) / 1024), 256, 0, 1, s, p, F, A, lo_row0, f16);
}

cudaError_t cl_launch_attn_wide(const float *q, int ld_q, const void *kcache, const void *vcache, __nv_bfloat16 *out_b,
                                int lo_row0, int M, int d, int H, int Hkv, int hd, int max_seq, const ClDevState *st,
                                int f16, cudaStream_t s) {
    if (hd != 128 && hd != 64) return cudaErrorInvalidValue;
    const size_t smem = hd == 128 ? attn_wide_smem<128>() : attn_wide_smem<64>();
    auto kern = hd == 128 ? (f16 ? k_attn_wide<128, 1> : k_attn_wide<128, 0>) : (f16 ? k_attn_wide<64, 1> : k_attn_wide<64, 0>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kern, dim3(H, (M + AQ - 1) / AQ), 128, smem, 1, s, q, ld_q, (const unsigned short *)kcache,
                          (const unsigned short *)vcache, out_b, lo_row0, M, d, H, Hkv, max_seq, st);
}

bool cl_make_tensor_map(ClTensorMap *m, const void *base, int rows, int cols, int box_rows, int f16) {
    static_assert(sizeof(ClTensorMap) >= sizeof(CUtensorMap), "tensor map storage");
    return make_map((CUtensorMap *)m->bytes, base, rows, cols, box_rows, f16);
}
