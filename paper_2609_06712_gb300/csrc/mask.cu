// Block mask: pooled block scores and per-query-block top-n_keep (kernel 1).
//
// The paper's sparse engine selects key blocks by a "topk ratio" (Alg. 1)
// without stating the score.  This library scores block pairs by the mean-
// pooled ROTATED vectors, s_ij = q_bar_i . k_bar_j / sqrt(d_h), keeps the
// n_keep largest per row (ties to the lower block id) and lists them
// ascending.  All score arithmetic is fp32.
#include <float.h>

#include "common.cuh"

namespace rola {

// ---------------------------------------------------------------------------
// scores[bh][i][j] = (q_bar_i . k_bar_j) / sqrt(128): fp32 SIMT GEMM, one 128 x 128
// tile per CTA, 256 threads with 8 x 8 register tiles, d staged through shared
// memory in chunks of 16, transposed and double-buffered: the next chunk's global
// loads are in flight while the current chunk is multiplied.  A warp owns a 32 x 64
// part of the tile (4 x 8 lanes, four wavefronts of shared loads per d), and a warp
// whose part lies outside the matrix skips the products: with 1182 blocks the
// padded tiles were 17 % of the work.  Bound by the fp32 FMA rate (1182 blocks, 40
// heads: 344 -> 322 us, 44 of the ~78 TFLOP/s of FMAs).  Two neighbouring columns go through one packed
// fma.rn.f32x2 (each element an IEEE fma), so every score is the same
// ascending-d fp32 FMA chain whatever the tiling.

constexpr int kSTile = 128, kSChunk = 16;

// (two CTAs per SM: the 128-register budget keeps both resident)
__global__ void __launch_bounds__(256, 2) block_scores_kernel(Shape s, const float* __restrict__ qbar,
                                                              const float* __restrict__ kbar,
                                                              float* __restrict__ scores)
{
    chain_begin();
    __shared__ __align__(16) float qs[2][kSChunk][kSTile + 4];
    __shared__ __align__(16) float ks[2][kSChunk][kSTile + 4];
    const int bh = blockIdx.z, i0 = blockIdx.y * kSTile, j0 = blockIdx.x * kSTile;
    const float* Q = qbar + (size_t)bh * s.nQ * kDh;
    const float* K = kbar + (size_t)bh * s.nB * kDh;
    // warp part (wr, wc): rows 32 wr .., columns 64 wc .. (the four warps of a column half and the two of
    // a row part sit on different schedulers, so an edge tile's work stays spread)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wc = warp >> 2, wr = ((warp & 3) + 2 * wc) & 3;
    const int ra0 = wr * 32 + (lane >> 3) * 4, ca0 = wc * 64 + (lane & 7) * 4;   // rows ra0 .., ra0 + 16 ..; columns ca0 .., ca0 + 32 ..
    const bool inside = i0 + wr * 32 < s.nQ && j0 + wc * 64 < s.nB;
    // loader: 128 rows x 16 d per operand = 512 float4, two per thread
    const int lrow = threadIdx.x >> 2, lq = threadIdx.x & 3;     // rows lrow, lrow + 64; d 4*lq .. 4*lq+3
    float4 ra[2], rb[2];
    auto fetch = [&](int d0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = lrow + 64 * h;
            const int gi = i0 + row, gj = j0 + row;
            ra[h] = gi < s.nQ ? __ldg(reinterpret_cast<const float4*>(Q + (size_t)gi * kDh + d0) + lq)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
            rb[h] = gj < s.nB ? __ldg(reinterpret_cast<const float4*>(K + (size_t)gj * kDh + d0) + lq)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto stash = [&](int buf) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = lrow + 64 * h;
            qs[buf][4 * lq][row] = ra[h].x; qs[buf][4 * lq + 1][row] = ra[h].y;
            qs[buf][4 * lq + 2][row] = ra[h].z; qs[buf][4 * lq + 3][row] = ra[h].w;
            ks[buf][4 * lq][row] = rb[h].x; ks[buf][4 * lq + 1][row] = rb[h].y;
            ks[buf][4 * lq + 2][row] = rb[h].z; ks[buf][4 * lq + 3][row] = rb[h].w;
        }
    };
    float acc[8][8] = {};
    fetch(0);
    stash(0);
    __syncthreads();
#pragma unroll 1
    for (int c = 0; c < kDh / kSChunk; ++c) {
        const int buf = c & 1;
        if (c + 1 < kDh / kSChunk) fetch((c + 1) * kSChunk);
        if (inside)
#pragma unroll
        for (int d = 0; d < kSChunk; ++d) {
            const float4 a0 = *reinterpret_cast<const float4*>(&qs[buf][d][ra0]);
            const float4 a1 = *reinterpret_cast<const float4*>(&qs[buf][d][ra0 + 16]);
            const float4 b0 = *reinterpret_cast<const float4*>(&ks[buf][d][ca0]);
            const float4 b1 = *reinterpret_cast<const float4*>(&ks[buf][d][ca0 + 32]);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int w = 0; w < 8; w += 2)
                    asm("{\n.reg .b64 ra, rb, rc;\n"
                        "mov.b64 ra, {%2, %2};\n"
                        "mov.b64 rb, {%3, %4};\n"
                        "mov.b64 rc, {%0, %1};\n"
                        "fma.rn.f32x2 rc, ra, rb, rc;\n"
                        "mov.b64 {%0, %1}, rc;\n}\n"
                        : "+f"(acc[u][w]), "+f"(acc[u][w + 1])
                        : "f"(av[u]), "f"(bv[w]), "f"(bv[w + 1]));
        }
        // the other buffer was last read in chunk c - 1, before the previous barrier
        if (c + 1 < kDh / kSChunk) stash(buf ^ 1);
        __syncthreads();
    }
    const float scale = 0.08838834764831845f;   // 1 / sqrt(128)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int gi = i0 + ra0 + (u < 4 ? u : 16 + u - 4);
        if (gi >= s.nQ) continue;
        float* out = scores + ((size_t)bh * s.nQ + gi) * s.nB;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int gj = j0 + ca0 + (w < 4 ? w : 32 + w - 4);
            if (gj < s.nB) out[gj] = acc[u][w] * scale;
        }
    }
}

// ---------------------------------------------------------------------------
// top-n_keep of each score row: one warp per row, 8 rows per CTA, lane l holding
// blocks l, l + 32, ... in K registers (in shared memory for the longest rows).  The
// row's n_keep-th largest score is found, then every block whose score is above it is
// taken, and the lowest-index blocks that equal it.
//
// The threshold: a 256-bin histogram that is linear between the row's least and
// largest score (a monotone map, so the counts give the bin of the n_keep-th
// largest), then the handful of scores in that bin are ranked against each other.
// Rows where that does not apply (a score that is not finite, all scores equal, a bin
// with over 128 scores) take a 4-pass 8-bit radix select on order-preserving keys.
// The map's shift is rounded, so where the scores differ by a few last bits only, the
// whole row may land far below bin 0 or above bin 255; the end bins take those in, both
// where scores are counted and where a bin's scores are listed.
//
// Bound by instruction issue: rows of 1182 took ~2600 instructions each with the
// radix select, or with a loop that tests every element's index; so the registers
// are filled up with -inf, and the blocks are written from one word per 32 of them:
// ~1770 now.  40 x 1182 rows of 1182: 182 -> 127 us.

__device__ __forceinline__ uint32_t order_key(float f)
{
    uint32_t u = __float_as_uint(f == 0.0f ? 0.0f : f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kTopkWarps = 8;

// The bin (of 256 counts) that holds the need-th largest, from the top down, and how many lie in
// higher bins; the same in all lanes.
__device__ __forceinline__ int find_bin(const uint32_t* hist, int need, int& above)
{
    const int lane = threadIdx.x & 31;
    // lane owns bins 8*(31-lane) .. 8*(31-lane)+7 so that lane 0 holds the top bins
    const int base = 8 * (31 - lane);
    uint32_t c[8];
    uint32_t tot = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) { c[t] = hist[base + t]; tot += c[t]; }
    // inclusive prefix over lanes (from the top bins down)
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    uint32_t excl = incl - tot;
    // the lane whose range holds the need-th key from the top
    const uint32_t ballot = __ballot_sync(0xffffffffu, excl < (uint32_t)need && incl >= (uint32_t)need);
    const int src = ballot ? __ffs(ballot) - 1 : 0;
    int bin = 0, ab = 0;
    if (lane == src) {
        uint32_t run = excl;
        for (int t = 7; t >= 0; --t) {
            if (run + c[t] >= (uint32_t)need) { bin = base + t; ab = (int)run; break; }
            run += c[t];
        }
    }
    above = __shfl_sync(0xffffffffu, ab, src);
    return __shfl_sync(0xffffffffu, bin, src);
}

// What the histogram map of a row needs: scale and shift, and whether it can be used.
struct LinearBins {
    float scale, shift;
    bool ok;
    __device__ LinearBins(float lo, float hi, bool finite)
    {
        scale = 255.0f / (hi - lo);
        shift = -lo * scale;
        ok = finite && hi > lo && hi - lo < INFINITY && fabsf(scale) < INFINITY && fabsf(shift) < INFINITY;
    }
    // (one rounding of a rising function of f: monotone)
    __device__ float at(float f) const { return fmaf(f, scale, shift); }
    __device__ static int bin(float t) { return max(0, min(255, __float2int_rz(t))); }
};

// The rank-th (from 0) of `count` <= 128 candidates in block order, ties in that order: its score and block.
__device__ __forceinline__ void pick(const float* cand, const int* cand_j, int count, int rank, float& thr, int& last)
{
    float mine = 0.0f;
    int mine_j = 0;
    bool hit = false;
    for (int i = threadIdx.x & 31; i < count; i += 32) {
        const float f = cand[i];
        int r = 0;
        for (int u = 0; u < count; ++u) r += cand[u] > f || (cand[u] == f && u < i);
        if (r == rank) {
            hit = true;
            mine = f;
            mine_j = cand_j[i];
        }
    }
    const uint32_t b = __ballot_sync(0xffffffffu, hit);
    const int src = b ? __ffs(b) - 1 : 0;
    thr = __shfl_sync(0xffffffffu, mine, src);
    last = __shfl_sync(0xffffffffu, mine_j, src);
}

// Rows of 32 (K - 8) + 1 .. 32 K blocks.
template <int K>
__global__ void __launch_bounds__(kTopkWarps * 32) block_topk_kernel(Shape s, const float* __restrict__ scores,
                                                                     int32_t* __restrict__ kv_idx)
{
    chain_begin();
    __shared__ uint32_t hist_s[kTopkWarps][256];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* hist = hist_s[warp];
    const int row = blockIdx.x * kTopkWarps + warp;
    const int bh = blockIdx.y, nB = s.nB;
    if (row >= s.nQ) return;
    const float* srow = scores + ((size_t)bh * s.nQ + row) * nB + lane;
    float v[K];
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = i < K - 8 || 32 * i + lane < nB ? __ldg(srow + 32 * i) : 0.0f;
    float nan = 0.0f, lo = INFINITY, hi = -INFINITY;      // nan: 0, or NaN once a score is not finite
#pragma unroll
    for (int i = 0; i < K; ++i) {
        nan = fmaf(v[i], 0.0f, nan);
        if (i < K - 8 || 32 * i + lane < nB) lo = fminf(lo, v[i]);
        else v[i] = -INFINITY;
        hi = fmaxf(hi, v[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const LinearBins lin(lo, hi, __all_sync(0xffffffffu, nan == 0.0f));

    // kept: scores above thr, and those equal to it up to block last
    float thr = hi;
    int last = -1;
    bool found = false;
    if (lin.ok) {
#pragma unroll
        for (int i = 0; i < 8; ++i) hist[32 * i + lane] = 0;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < K; ++i)
            if (i < K - 8 || 32 * i + lane < nB) atomicAdd(&hist[LinearBins::bin(lin.at(v[i]))], 1u);
        __syncwarp();
        int above;
        const int bin = find_bin(hist, s.n_keep, above);
        const int count = (int)hist[bin];
        __syncwarp();
        if (count <= 128) {
            // the bin's scores and blocks, in block order, where the counts were: t in [t0, t1) is the
            // bin that LinearBins::bin gives (t of a score is finite, of the fill -inf: outside)
            float* cand = reinterpret_cast<float*>(hist);
            int* cand_j = reinterpret_cast<int*>(hist + 128);
            const float t0 = bin == 0 ? -FLT_MAX : (float)bin, t1 = bin == 255 ? INFINITY : (float)(bin + 1);
            int n = 0;
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const float t = lin.at(v[i]);
                const bool in = t >= t0 && t < t1;
                const uint32_t m = __ballot_sync(0xffffffffu, in);
                if (m) {
                    if (in) {
                        const int at = n + __popc(m & ((1u << lane) - 1u));
                        cand[at] = v[i];
                        cand_j[at] = 32 * i + lane;
                    }
                    n += __popc(m);
                }
            }
            __syncwarp();
            found = n == count;
            if (found) pick(cand, cand_j, count, s.n_keep - above - 1, thr, last);
        }
    }
    // word w: the kept blocks 32 w .. 32 w + 31; lane l takes words l and 32 + l
    uint32_t w0 = 0, w1 = 0;
    if (found) {
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const uint32_t m = __ballot_sync(0xffffffffu, v[i] > thr || (v[i] == thr && 32 * i + lane <= last));
            if (i < 32) w0 = lane == i ? m : w0;
            else w1 = lane == i - 32 ? m : w1;
        }
    } else {
        uint32_t prefix = 0, pmask = 0;
        int need = s.n_keep, eq_taken = 0;
#pragma unroll 1
        for (int sh = 24; sh >= 0; sh -= 8) {
#pragma unroll
            for (int i = 0; i < 8; ++i) hist[32 * i + lane] = 0;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const uint32_t key = order_key(v[i]);
                if ((i < K - 8 || 32 * i + lane < nB) && (key & pmask) == prefix) atomicAdd(&hist[(key >> sh) & 255u], 1u);
            }
            __syncwarp();
            int above;
            const int bin = find_bin(hist, need, above);
            need -= above;
            prefix |= (uint32_t)bin << sh;
            pmask |= 255u << sh;
            __syncwarp();
        }
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const uint32_t key = order_key(v[i]);
            const bool in = i < K - 8 || 32 * i + lane < nB;
            const bool eq = in && key == prefix;
            const uint32_t eqb = __ballot_sync(0xffffffffu, eq);
            const uint32_t m = __ballot_sync(0xffffffffu, (in && key > prefix) ||
                                                              (eq && eq_taken + __popc(eqb & ((1u << lane) - 1u)) < need));
            eq_taken += __popc(eqb);
            if (i < 32) w0 = lane == i ? m : w0;
            else w1 = lane == i - 32 ? m : w1;
        }
    }
    int32_t* out = kv_idx + ((size_t)bh * s.nQ + row) * s.n_keep;
    int base = 0;                                     // blocks in the words before this round's
#pragma unroll
    for (int h = 0; h < (K > 32 ? 2 : 1); ++h) {
        uint32_t w = h ? w1 : w0;
        int pos = __popc(w);                          // inclusive count over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += y;
        }
        const int all = __shfl_sync(0xffffffffu, pos, 31);
        pos += base - __popc(w);
        for (; w; w &= w - 1, ++pos)
            if (pos < s.n_keep) out[pos] = 32 * (32 * h + lane) + __ffs(w) - 1;
        base += all;
    }
}

// Longer rows: the scores in shared memory, the same selection.
__global__ void __launch_bounds__(kTopkWarps * 32) block_topk_long_kernel(Shape s, const float* __restrict__ scores,
                                                                          int32_t* __restrict__ kv_idx)
{
    chain_begin();
    extern __shared__ uint32_t tk_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* hist = tk_smem + warp * 256;
    float* v = reinterpret_cast<float*>(tk_smem + kTopkWarps * 256) + (size_t)warp * s.nB;
    const int row = blockIdx.x * kTopkWarps + warp;
    const int bh = blockIdx.y, nB = s.nB;
    if (row >= s.nQ) return;
    const float* srow = scores + ((size_t)bh * s.nQ + row) * nB;
    float nan = 0.0f, lo = INFINITY, hi = -INFINITY;
#pragma unroll 8
    for (int j = lane; j < nB; j += 32) {
        const float f = __ldg(srow + j);
        v[j] = f;
        nan = fmaf(f, 0.0f, nan);
        lo = fminf(lo, f);
        hi = fmaxf(hi, f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const LinearBins lin(lo, hi, __all_sync(0xffffffffu, nan == 0.0f));
    float thr = hi;
    int last = -1;
    bool found = false;
    if (lin.ok) {
        for (int b = lane; b < 256; b += 32) hist[b] = 0;
        __syncwarp();
#pragma unroll 8
        for (int j = lane; j < nB; j += 32) atomicAdd(&hist[LinearBins::bin(lin.at(v[j]))], 1u);
        __syncwarp();
        int above;
        const int bin = find_bin(hist, s.n_keep, above);
        const int count = (int)hist[bin];
        __syncwarp();
        if (count <= 128) {
            float* cand = reinterpret_cast<float*>(hist);
            int* cand_j = reinterpret_cast<int*>(hist + 128);
            int n = 0;
            for (int j0 = 0; j0 < nB; j0 += 32) {
                const int j = j0 + lane;
                const bool in = j < nB && LinearBins::bin(lin.at(v[j])) == bin;
                const uint32_t m = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const int at = n + __popc(m & ((1u << lane) - 1u));
                    cand[at] = v[j];
                    cand_j[at] = j;
                }
                n += __popc(m);
            }
            __syncwarp();
            found = n == count;
            if (found) pick(cand, cand_j, count, s.n_keep - above - 1, thr, last);
        }
    }
    uint32_t prefix = 0, pmask = 0;
    int need = s.n_keep, eq_taken = 0;
    if (!found) {
#pragma unroll 1
        for (int sh = 24; sh >= 0; sh -= 8) {
            for (int b = lane; b < 256; b += 32) hist[b] = 0;
            __syncwarp();
            for (int j = lane; j < nB; j += 32) {
                const uint32_t key = order_key(v[j]);
                if ((key & pmask) == prefix) atomicAdd(&hist[(key >> sh) & 255u], 1u);
            }
            __syncwarp();
            int above;
            const int bin = find_bin(hist, need, above);
            need -= above;
            prefix |= (uint32_t)bin << sh;
            pmask |= 255u << sh;
            __syncwarp();
        }
    }
    int32_t* out = kv_idx + ((size_t)bh * s.nQ + row) * s.n_keep;
    int written = 0;
    for (int j0 = 0; j0 < nB; j0 += 32) {
        const int j = j0 + lane;
        const float f = j < nB ? v[j] : 0.0f;
        bool sel;
        if (found) {
            sel = j < nB && (f > thr || (f == thr && j <= last));
        } else {
            const uint32_t key = order_key(f);
            const bool eq = j < nB && key == prefix;
            const uint32_t eqb = __ballot_sync(0xffffffffu, eq);
            sel = (j < nB && key > prefix) || (eq && eq_taken + __popc(eqb & ((1u << lane) - 1u)) < need);
            eq_taken += __popc(eqb);
        }
        const uint32_t m = __ballot_sync(0xffffffffu, sel);
        const int pos = written + __popc(m & ((1u << lane) - 1u));
        if (sel && pos < s.n_keep) out[pos] = j;
        written += __popc(m);
    }
}

cudaError_t launch_block_topk(const Shape& s, const float* qbar, const float* kbar, float* scores,
                              int32_t* kv_idx, cudaStream_t st)
{
    const int tj = (s.nB + kSTile - 1) / kSTile, ti = (s.nQ + kSTile - 1) / kSTile;
    launch_kernel(block_scores_kernel, dim3(tj, ti, s.B * s.H), 256, 0, st, s, qbar, kbar, scores);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // registers per lane by the row's length; past 40 a lane too few warps would fit an SM
    const dim3 grid((s.nQ + kTopkWarps - 1) / kTopkWarps, s.B * s.H);
    if (s.nB <= 40 * 32) {
        auto kernel = s.nB <= 8 * 32    ? block_topk_kernel<8>
                      : s.nB <= 16 * 32 ? block_topk_kernel<16>
                      : s.nB <= 24 * 32 ? block_topk_kernel<24>
                      : s.nB <= 32 * 32 ? block_topk_kernel<32>
                                        : block_topk_kernel<40>;
        launch_kernel(kernel, grid, kTopkWarps * 32, 0, st, s, scores, kv_idx);
        return cudaGetLastError();
    }
    const size_t smem = (size_t)kTopkWarps * (256 + s.nB) * 4;
    if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(block_topk_long_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    launch_kernel(block_topk_long_kernel, grid, kTopkWarps * 32, smem, st, s, scores, kv_idx);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 128-token query means: the 64-token chunks' fp32 q sums S (each the pairwise
// tree over its 64 slots) give chunk c of 128 tokens the tree's top node
// S[2c] + S[2c+1] (an absent right half is the empty tree, +0), divided once by
// the chunk's token count -- the pairwise sum over 128 slots.
__global__ void qpool128_kernel(Shape s, const float* __restrict__ qsum, float* __restrict__ qbar)
{
    chain_begin();
    const int c = blockIdx.x, bh = blockIdx.y, d = threadIdx.x;
    const float* src = qsum + ((size_t)bh * s.nB + 2 * c) * kDh + d;
    const float right = 2 * c + 1 < s.nB ? src[kDh] : 0.0f;
    const int cnt = min(128, s.N - 128 * c);
    qbar[((size_t)bh * s.nQ + c) * kDh + d] = (src[0] + right) / (float)cnt;
}

cudaError_t launch_qpool128(const Shape& s, const float* qsum64, float* qbar128, cudaStream_t st)
{
    launch_kernel(qpool128_kernel, dim3(s.nQ, s.B * s.H), kDh, 0, st, s, qsum64, qbar128);
    return cudaGetLastError();
}

}  // namespace rola
