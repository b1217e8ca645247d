// Backward pass of the block-sparse softmax attention on the 5th-generation
// tensor cores (bf16, fp32 accumulation in TMEM):
//
//   P = exp(q^r k^r / sqrt d - lse),  dP = dO^s v^T,  dS = P (dP - D),
//   dq^r = dS k^r / sqrt d,  dk^r = dS^T q^r / sqrt d,  dv = P^T dO^s
//
// over the kept (query block, key block) pairs (Sec. 3 softmax form, its
// gradient).  Two kernels, both with the 64 rows of an item in the TMEM lanes
// (M = 64: lanes 0-15 of each quarter, row r at lane 32 (r / 16) + r mod 16) and
// the 128 rows of a tile, a pair of kept blocks, in the columns:
//
//   query side (item = a query block, tiles = pairs of its kept key blocks)
//     S  = Q K_pair^T,  dP = dO V_pair^T,  dQ += dS K_pair      (N = 128 each)
//   key side (item = a key block, tiles = pairs of the query blocks that kept it)
//     S^T = K Q_pair^T, dP^T = V dO_pair^T, dV += P^T dO_pair, dK += dS^T Q_pair
//
// P and dS go back to TMEM as packed bf16, the A operand of the accumulating
// products, so neither passes through shared memory.  The log-sum-exp of each
// query is known, so a tile needs no running maximum: eight warps share it, a
// thread 32 columns of one row (warpgroup w: block w of the pair; the two half
// warps 32 columns each).  Each result has one or two products' time (512 cycles
// each) until it is needed again, so S, dP and the accumulators are single-buffered.
//   query side: S, dP of a tile by one thread, dQ by another     dS double-buffered
//     (an issuer spends 75 cycles on every barrier it waits for even when that is
//     complete, and the pipe runs dry meanwhile: one thread for all took 18.1 ms
//     where this takes 16.0, 720p layer)
//   key side:   S(g+1) dK(g) dP(g+1) dV(g+1) by one thread       P written over S, dS over dP
//     (products are sure to run in the order they are issued in only where they share an
//     accumulator, so S(g+1) waits until dV(g) has read its P(g), dP(g+1) until dK(g) has
//     read its dS(g).  S and dP are a product per block of the pair, N = 64, so that the
//     first runs while the second block's dV or dK still does.  720p training step: 54.7
//     ms with no such wait, 58.3 waiting for whole products, 55.7 this way.
//     With the order S dP dV dK each wait has a product in between, but P and dS have one
//     product's time instead of two: 58.7.  With S, dV and dP, dK on two threads the
//     kernel took 25.7 ms instead of 21.6)
//
// What bounds it: an M = 64 product takes 64 cycles a K step of 16 with N = 128 (half
// the M = 128 rate) and 45 with N = 64, so 1536 (query side) and 2464 (key side) tensor
// cycles a tile; shared memory moves 192 / 256 KB a tile (1500 / 2000 cycles at 128
// B/cycle).  The transposed form used before (M = 128 x N = 64 products, 1152
// and 1536 tensor cycles, P and dS through shared memory) moved 224 and 288 KB,
// and its two-deep rings of 64 KB pairs were held through the whole tile.  At
// the 720p layer (40 heads, 75600 tokens, 118 of 1182 blocks kept): query side
// 27.3 -> 15.9 ms, key side 37.9 -> 22.5 ms (866 / 1226 ns a tile; the products
// alone take 750 / 1200 ns at the 2.05 GHz the SMs hold under this load); at
// the 12-head 480p layer 1.84 -> 0.99 and 2.52 -> 1.41 ms.
//
// Roles (384 threads, one persistent CTA per SM):
//   warps 0-7  P / dS and the epilogue; warp w owns TMEM lane quarter w mod 4
//   warps 8, 9 TMA producers (one elected thread each)
//   warp 10    issuer and TMEM owner
//   warp 11    query side: second issuer; key side: log-sum-exp and D of a tile's queries into shared memory
// Every mbarrier wait is bounded; a wait that gives up records ROLA_ERR_TIMEOUT
// and the CTA drains what it issued and frees TMEM.
#include <math_constants.h>
#include <stddef.h>

#include "common.cuh"
#include "tcgen05.cuh"
#include "tensor_map.cuh"

namespace rola {
namespace {

using namespace tc;

constexpr int kDsWarps = 8;
constexpr int kCols = 32;                        // tile columns of a dS thread
constexpr int kProdAWarp = 8, kProdBWarp = 9, kMmaWarp = 10, kMma2Warp = 11, kStatWarp = 11;
constexpr int kThreads = 32 * 12;
constexpr uint32_t kBlockBytes = 64 * 128 * 2;   // one block, [chunk][row][64]
constexpr uint32_t kPairBytes = 128 * 128 * 2;   // a pair of blocks, [chunk][block][row][64]
constexpr uint32_t kTmemCols = 512;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kScale = 0.08838834764831845f;   // 1 / sqrt(128)

struct Params {
    Shape s;
    const int32_t* kv_idx;              // query side: kept key blocks
    const int32_t* off;                 // key side: the transposed mask, [BH][nB + 1]
    const int32_t* list;                //   [BH][nB * n_keep]
    const float* lse;                   // block order, Np rows a head
    const float* Dv;
    const float* lr0;                   // fp32 low-rank part of dq (query side), of dk (key side)
    const float* lr1;                   //   of dv (key side)
    const float2* tab;
    __nv_bfloat16* out0;                // dq, or dk
    __nv_bfloat16* out1;                // dv (key side)
    DeviceStatus* status;
    int total_items;
};

__device__ __forceinline__ void record_timeout(const Params& p, int where)
{
    if (atomicCAS(&p.status->code, 0, (int)ROLA_ERR_TIMEOUT) == 0) p.status->where = where;
}

// The 32 columns of this thread: warpgroup wg's 64, split between the half warps
// (taddr: the warp's lanes, column 64 wg).
__device__ __forceinline__ void ld_cols(uint32_t taddr, float (&v)[kCols])
{
    tmem_ld16_half<32>(taddr, *reinterpret_cast<float(*)[16]>(&v[0]));
    tmem_ld16_half<32>(taddr + 16, *reinterpret_cast<float(*)[16]>(&v[16]));
    tmem_ld_wait(*reinterpret_cast<float(*)[16]>(&v[0]));
    reg_fence(*reinterpret_cast<float(*)[16]>(&v[16]));
}

// 32 values as packed bf16 into 16 TMEM columns per half warp (taddr: the warpgroup's first).
__device__ __forceinline__ void st_cols(uint32_t taddr, const float (&v)[kCols])
{
    uint32_t pk[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
    tmem_st16_half<16>(taddr, *reinterpret_cast<const float(*)[16]>(pk));
    tmem_st_wait();
}

// A pair of blocks (rows ra .. of the first, rb .. of the second when `two`) into
// the [chunk][block][row] layout at dst.
__device__ __forceinline__ void load_pair(uint32_t dst, const CUtensorMap* map, uint32_t full, int ra, int rb, bool two,
                                          int bh)
{
    tma_load_3d(dst, map, full, 0, ra, bh);
    tma_load_3d(dst + 16384, map, full, 64, ra, bh);
    if (two) {
        tma_load_3d(dst + 8192, map, full, 0, rb, bh);
        tma_load_3d(dst + 24576, map, full, 64, rb, bh);
    }
}

// d = A[smem, 64 rows, K-major] B[smem, the rows of a pair or of one of its blocks, K-major]^T (id: N columns)
__device__ __forceinline__ void mma_scores(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t id)
{
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
        mma_ss_split(d, a + (kk >> 2) * 512 + (kk & 3) * 2, a_hi, b + (kk >> 2) * 1024 + (kk & 3) * 2, b_hi, id,
                     kk > 0 ? 1u : 0u);
}

// d (+)= A[TMEM, 64 rows] B[smem, one block of a pair, MN-major]: K steps of 16 of its rows
__device__ __forceinline__ void mma_grad(uint32_t d, uint32_t a, uint32_t b, uint32_t b_hi, uint32_t id, bool first)
{
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) mma_ts_split(d, a + kk * 8, b + kk * 128, b_hi, id, !first || kk > 0 ? 1u : 0u);
}
constexpr uint32_t kSecond = (64 * 128) >> 4;     // descriptor offset from a pair's first block to its second

// The 128 bytes at p into L2 (the epilogue's rows, asked for when the item starts).
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p)); }

// The 32 outputs of a thread (columns d0 .. d0 + 31 of one row) at dst, as bf16.
__device__ __forceinline__ void store_row32(__nv_bfloat16* dst, const float (&v)[kCols])
{
#pragma unroll
    for (int c = 0; c < 4; ++c)
        reinterpret_cast<uint4*>(dst)[c] =
            make_uint4(pack_bf16(v[8 * c], v[8 * c + 1]), pack_bf16(v[8 * c + 2], v[8 * c + 3]),
                       pack_bf16(v[8 * c + 4], v[8 * c + 5]), pack_bf16(v[8 * c + 6], v[8 * c + 7]));
}
__device__ __forceinline__ void load_row32(const float* src, float (&v)[kCols])
{
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(src) + c);
        v[4 * c] = f.x;
        v[4 * c + 1] = f.y;
        v[4 * c + 2] = f.z;
        v[4 * c + 3] = f.w;
    }
}
// v = lr + R(n)^T (v / sqrt d) on the pairs of columns d0 .. d0 + 31
__device__ __forceinline__ void rotate_back32(float (&v)[kCols], const float (&lr)[kCols], const float2 (&cs)[16])
{
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float x0 = v[2 * i] * kScale, x1 = v[2 * i + 1] * kScale;
        v[2 * i] = lr[2 * i] + __fmaf_rn(x0, cs[i].x, __fmul_rn(x1, cs[i].y));
        v[2 * i + 1] = lr[2 * i + 1] + __fmaf_rn(x1, cs[i].x, -__fmul_rn(x0, cs[i].y));
    }
}
__device__ __forceinline__ void load_cs(const Params& p, int n, int d0, float2 (&cs)[16])
{
    const Shape& s = p.s;
    const int hw = s.Hh * s.Ww, t = n / hw, rem = n - t * hw, x = rem / s.Ww, y = rem - x * s.Ww;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int m = (d0 >> 1) + i;
        const int row = m < s.pt ? t : (m < s.pt + s.px ? s.T + x : s.T + s.Hh + y);
        cs[i] = __ldg(p.tab + row * kPairs + m);
    }
}

// =========================================================================== query side

namespace dq {

constexpr int KS = 3, VS = 2;                                   // K pairs (held until dQ), V pairs
constexpr uint32_t kSmQ = 0, kSmO = 2 * kBlockBytes, kSmK = 4 * kBlockBytes;   // Q and dO: two items
constexpr uint32_t kSmV = kSmK + KS * kPairBytes, kTiles = kSmV + VS * kPairBytes;   // 224 KB
constexpr uint32_t kS = 0, kDP = 128, kDQ = 256, kDS = 384;     // TMEM columns (dS: two buffers of 64)

enum Bar { Q_FULL = 0, Q_EMPTY = Q_FULL + 2, K_FULL = Q_EMPTY + 2, K_EMPTY = K_FULL + KS, V_FULL = K_EMPTY + KS,
           V_EMPTY = V_FULL + VS, S_FULL = V_EMPTY + VS, S_EMPTY, DP_FULL, DP_EMPTY, DS_FULL, DS_EMPTY = DS_FULL + 2,
           O_FULL = DS_EMPTY + 2, O_EMPTY, DRAIN, NUM_BARS = DRAIN + 2 };

struct Ctrl {
    uint64_t bar[NUM_BARS];
    ItemRing items;
    uint32_t tmem_base;
    int abort;
};
static_assert(kTiles % 1024 == 0 && kTiles + sizeof(Ctrl) <= 232448, "tiles and control block fit the 227 KB of a CTA");

}  // namespace dq

template <bool kCube>
__global__ void __launch_bounds__(kThreads, 1) sparse_bwd_dq_tc_kernel(const __grid_constant__ CUtensorMap map_q,
                                                                       const __grid_constant__ CUtensorMap map_o,
                                                                       const __grid_constant__ CUtensorMap map_k,
                                                                       const __grid_constant__ CUtensorMap map_v,
                                                                       const Params p)
{
    using namespace dq;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if (smem_u32(smem_raw) & 1023u) {
        if (threadIdx.x == 0) atomicCAS(&p.status->code, 0, (int)ROLA_ERR_UNSUPPORTED);
        return;
    }
    Ctrl& sm = *reinterpret_cast<Ctrl*>(smem_raw + kTiles);
    const uint32_t sbase = smem_u32(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar = [&](int i) { return smem_u32(&sm.bar[i]); };
    const Shape& s = p.s;
    const int nB = s.nB, T = (s.n_keep + 1) / 2;

    if (tid == 0) {
        sm.abort = 0;
        for (int i = 0; i < NUM_BARS; ++i) {
            const bool by_warps = i == S_EMPTY || i == DP_EMPTY || i == DS_FULL || i == DS_FULL + 1 || i == O_EMPTY;
            mbar_init(bar(i), by_warps ? kDsWarps : 1);
        }
        sm.items.init();
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
        tmem_relinquish();
    }
    if (warp == kProdAWarp && lane == 0) {
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_o);
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    chain_begin();
    volatile int* abort = &sm.abort;
    // the CTA's i-th item, for a single-thread role and for a warp
    auto item_at = [&](int i, bool& ok) { return sm.items.get<true>(i, ok, abort, s.wait_limit_ns); };
    auto item_at_warp = [&](int i, bool& ok) { return sm.items.get<false>(i, ok, abort, s.wait_limit_ns); };

    if (warp == kProdAWarp || warp == kProdBWarp) {
        // ------------------------------------------------------------ TMA: Q, dO and the K pairs / the V pairs
        const bool is_v = warp == kProdBWarp;
        const int NS = is_v ? VS : KS;
        const uint32_t ring = is_v ? kSmV : kSmK;
        const int full0 = is_v ? V_FULL : K_FULL, empty0 = is_v ? V_EMPTY : K_EMPTY;
        const CUtensorMap* map = is_v ? &map_v : &map_k;
        if (elect_one()) {
            int k = 0, issued_q = 0, issued = 0;
            bool ok = true;
            // (the K warp hands out the items: the next one is known, the one after asked for)
            int item = is_v ? item_at(0, ok) : (int)blockIdx.x, next = 0;
            int* counter = &p.status->next[kItemsDq];
            if (!is_v) {
                sm.items.post(0, item, abort, s.wait_limit_ns);
                next = gridDim.x + atomicAdd(counter, 1);
            }
            for (; item < p.total_items && ok; ++k) {
                const int bh = item / nB, qb = item - bh * nB;
                const int32_t* kept = p.kv_idx + (size_t)item * s.n_keep;
                int ja_n = __ldg(kept), jb_n = s.n_keep > 1 ? __ldg(kept + 1) : -1;     // block ids, one tile ahead
                if (!is_v) {
                    const int qs = k & 1;
                    if (k >= 2 && !(ok = mbar_wait(bar(Q_EMPTY + qs), ((k >> 1) - 1) & 1, abort, s.wait_limit_ns))) break;
                    mbar_expect_tx(bar(Q_FULL + qs), 2 * kBlockBytes);
                    tma_load_4d(sbase + kSmQ + qs * kBlockBytes, &map_q, bar(Q_FULL + qs), 0, qb * 64, 0, bh);
                    tma_load_4d(sbase + kSmO + qs * kBlockBytes, &map_o, bar(Q_FULL + qs), 0, qb * 64, 0, bh);
                    ++issued_q;
                }
                int after = 0;
                for (int t = 0; t < T; ++t) {
                    // (the first answer of the counter is given time: it is not needed before the second tile)
                    if (!is_v && t == (k == 0 && T > 1 ? 1 : 0)) {
                        if (!(ok = sm.items.post(k + 1, next, abort, s.wait_limit_ns))) break;
                        after = gridDim.x + atomicAdd(counter, 1);
                    }
                    const int g = issued, st = g % NS;
                    const int ra = ja_n * 64, rb = jb_n * 64;
                    const bool two = jb_n >= 0;
                    if (t + 1 < T) {
                        ja_n = __ldg(kept + 2 * t + 2);
                        jb_n = 2 * t + 3 < s.n_keep ? __ldg(kept + 2 * t + 3) : -1;
                    }
                    if (g >= NS && !(ok = mbar_wait(bar(empty0 + st), ((g / NS) - 1) & 1, abort, s.wait_limit_ns))) break;
                    ++issued;
                    // test hook: the CTA's first K pair is never loaded, so the waits on it run out
                    if (!is_v && (s.debug_flags & ROLA_DEBUG_SKIP_FIRST_K_COPY) && g == 0) continue;
                    mbar_expect_tx(bar(full0 + st), two ? 32768u : 16384u);
                    load_pair(sbase + ring + st * kPairBytes, map, bar(full0 + st), ra, rb, two, bh);
                }
                if (!ok) break;
                if (is_v) item = item_at(k + 1, ok);
                else item = next, next = after;
            }
            if (!ok) record_timeout(p, is_v ? 20 : 17);
            // every copy this thread issued lands before the CTA exits (bounded by time only)
            int never = 0;
            for (int u = issued_q > 2 ? issued_q - 2 : 0; u < issued_q; ++u)
                mbar_wait(bar(Q_FULL + (u & 1)), (u >> 1) & 1, &never, s.wait_limit_ns);
            for (int u = issued > NS ? issued - NS : 0; u < issued; ++u)
                mbar_wait(bar(full0 + u % NS), (u / NS) & 1, &never, s.wait_limit_ns);
        }
    } else if (warp == kMmaWarp || warp == kMma2Warp) {
        // ------------------------------------------------------------ issuers: S and dP / dQ
        if (elect_one()) {
            const bool grad = warp == kMma2Warp;
            const uint32_t id_s = idesc_bf16(64, 128, false, false), id_g = idesc_bf16(64, 128, false, true);
            const uint64_t dk = smem_desc(sbase, 16, 1024);          // K-major operands
            const uint64_t dm = smem_desc(sbase, 16384, 1024);       // a pair read MN-major (chunks 16 KB apart)
            const uint32_t lo = (uint32_t)dk, hi = (uint32_t)(dk >> 32), mlo = (uint32_t)dm, mhi = (uint32_t)(dm >> 32);
            bool ok = true;
            int k = 0, g = 0;
            for (int item = item_at(0, ok); item < p.total_items && ok; item = item_at(++k, ok)) {
                const int qs = k & 1;
                if (!grad && !(ok = mbar_wait(bar(Q_FULL + qs), (k >> 1) & 1, abort, s.wait_limit_ns))) break;
                const uint32_t q = lo + ((kSmQ + qs * kBlockBytes) >> 4), o = lo + ((kSmO + qs * kBlockBytes) >> 4);
                for (int t = 0; t < T; ++t, ++g) {
                    const int ks = g % KS, vs = g % VS, db = g & 1;
                    if (grad) {
                        if (!(ok = mbar_wait(bar(K_FULL + ks), (g / KS) & 1, abort, s.wait_limit_ns))) break;
                        if (t == 0 && k >= 1 && !(ok = mbar_wait(bar(O_EMPTY), (k - 1) & 1, abort, s.wait_limit_ns))) break;
                        if (!(ok = mbar_wait(bar(DS_FULL + db), (g >> 1) & 1, abort, s.wait_limit_ns))) break;
                        fence_after_sync();
                        const uint32_t b = mlo + ((kSmK + ks * kPairBytes) >> 4);
                        mma_grad(tmem + kDQ, tmem + kDS + db * 64, b, mhi, id_g, t == 0);
                        if (2 * t + 1 < s.n_keep)           // (a half tile has the first block only)
                            mma_grad(tmem + kDQ, tmem + kDS + db * 64 + 32, b + kSecond, mhi, id_g, false);
                        mma_commit(bar(DS_EMPTY + db));
                        mma_commit(bar(K_EMPTY + ks));
                        if (t == T - 1) mma_commit(bar(O_FULL));
                        continue;
                    }
                    if (!(ok = mbar_wait(bar(K_FULL + ks), (g / KS) & 1, abort, s.wait_limit_ns))) break;
                    if (g >= 1 && !(ok = mbar_wait(bar(S_EMPTY), (g - 1) & 1, abort, s.wait_limit_ns))) break;
                    fence_after_sync();
                    mma_scores(tmem + kS, q, hi, lo + ((kSmK + ks * kPairBytes) >> 4), hi, id_s);
                    mma_commit(bar(S_FULL));
                    if (!(ok = mbar_wait(bar(V_FULL + vs), (g / VS) & 1, abort, s.wait_limit_ns))) break;
                    if (g >= 1 && !(ok = mbar_wait(bar(DP_EMPTY), (g - 1) & 1, abort, s.wait_limit_ns))) break;
                    fence_after_sync();
                    mma_scores(tmem + kDP, o, hi, lo + ((kSmV + vs * kPairBytes) >> 4), hi, id_s);
                    mma_commit(bar(DP_FULL));
                    mma_commit(bar(V_EMPTY + vs));
                    if (t == T - 1) mma_commit(bar(Q_EMPTY + qs));
                }
            }
            if (!ok) record_timeout(p, grad ? 21 : 18);
            // every product this thread issued completes before TMEM is released
            int never = 0;
            mma_commit(bar(DRAIN + grad));
            mbar_wait(bar(DRAIN + grad), 0, &never, s.wait_limit_ns);
        }
    } else if (warp < kDsWarps) {
        // ------------------------------------------------------------ dS + epilogue
        const int wg = warp >> 2, quarter = warp & 3, hf = lane >> 4;
        const int row = 16 * quarter + (lane & 15), d0 = 64 * wg + 32 * hf;
        const float c_log2 = s.sm_scale_log2;
        const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16);
        bool ok = true;
        int k = 0, g = 0;
        for (int item = item_at_warp(0, ok); item < p.total_items && ok; item = item_at_warp(++k, ok)) {
            const int bh = item / nB, qb = item - bh * nB;
            const int32_t* kept = p.kv_idx + (size_t)item * s.n_keep;
            const int n = slot_token_g<kCube>(s, qb, row);             // this row's token, -1 for an empty slot
            const size_t r = (size_t)bh * s.Np + (size_t)qb * 64 + row;
            const float l2 = n >= 0 ? __ldg(p.lse + r) * kLog2e : CUDART_INF_F;
            const float Dn = n >= 0 ? -__ldg(p.Dv + r) : 0.0f;
            const size_t at = ((size_t)bh * s.N + (n >= 0 ? n : 0)) * kDh + d0;
            prefetch_l2(p.lr0 + at);                                    // this thread's row part of the epilogue
            int j_n = wg < s.n_keep ? __ldg(kept + wg) : -1;            // this group's block, one tile ahead
            for (int t = 0; t < T; ++t, ++g) {
                const int j = j_n;
                if (t + 1 < T) j_n = 2 * t + 2 + wg < s.n_keep ? __ldg(kept + 2 * t + 2 + wg) : -1;
                const uint32_t keys = block_mask32<kCube>(s, j, hf);       // columns that are tokens
                if (!(ok = mbar_wait(bar(S_FULL), g & 1, abort, s.wait_limit_ns))) break;
                fence_after_sync();
                float x[kCols], y[kCols];
                ld_cols(base + kS + 64 * wg, x);
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(S_EMPTY));
#pragma unroll
                for (int i = 0; i < kCols; i += 2) {
                    ffma2(x[i], x[i + 1], c_log2, -l2);
                    x[i] = fast_exp2(x[i]);
                    x[i + 1] = fast_exp2(x[i + 1]);
                }
                if (!(ok = mbar_wait(bar(DP_FULL), g & 1, abort, s.wait_limit_ns))) break;
                fence_after_sync();
                ld_cols(base + kDP + 64 * wg, y);
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(DP_EMPTY));
#pragma unroll
                for (int i = 0; i < kCols; i += 2) {
                    fadd2(y[i], y[i + 1], Dn, Dn);
                    fmul2(y[i], y[i + 1], x[i], x[i + 1]);
                }
                if (keys != 0xffffffffu) {
#pragma unroll
                    for (int i = 0; i < kCols; ++i)
                        if (!((keys >> i) & 1u)) y[i] = 0.0f;
                }
                if (g >= 2 && !(ok = mbar_wait(bar(DS_EMPTY + (g & 1)), ((g >> 1) - 1) & 1, abort, s.wait_limit_ns)))
                    break;
                st_cols(base + kDS + (g & 1) * 64 + 32 * wg, y);
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(DS_FULL + (g & 1)));
            }
            if (!ok) break;
            // ---- epilogue: dq = low-rank row + R(p)^T (dQ / sqrt d); this thread's 32 columns
            // of its row.  What does not depend on dQ is read before the wait for it.
            float lr[kCols], v[kCols];
            float2 cs[16];
            load_row32(p.lr0 + at, lr);
            load_cs(p, n >= 0 ? n : 0, d0, cs);
            if (!(ok = mbar_wait(bar(O_FULL), k & 1, abort, s.wait_limit_ns))) break;
            fence_after_sync();
            ld_cols(base + kDQ + 64 * wg, v);
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(O_EMPTY));
            rotate_back32(v, lr, cs);
            if (n >= 0) store_row32(p.out0 + at, v);
        }
        if (!ok) record_timeout(p, 19);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
}

// =========================================================================== key side

namespace kv {

constexpr int QS = 3, OS = 2;                                   // Q pairs (held until dK), dO pairs (until dV)
constexpr uint32_t kSmK = 0, kSmV = 2 * kBlockBytes, kSmQ = 4 * kBlockBytes;   // K and V: two items
constexpr uint32_t kSmO = kSmQ + QS * kPairBytes, kTiles = kSmO + OS * kPairBytes;   // 224 KB
constexpr uint32_t kS = 0, kDP = 128, kDV = 256, kDK = 384;     // TMEM columns (P over S, dS over dP)

enum Bar { KV_FULL = 0, KV_EMPTY = KV_FULL + 2, Q_FULL = KV_EMPTY + 2, Q_EMPTY = Q_FULL + QS, O_FULL = Q_EMPTY + QS,
           O_EMPTY = O_FULL + OS, S_FULL = O_EMPTY + OS, DP_FULL, P_FULL, DS_FULL, ACC_FULL, ACC_EMPTY,
           DV_HALF, DK_HALF, DRAIN, NUM_BARS };

struct Ctrl {
    float lse2[2][128];                  // log-sum-exp (log2 units) and -D of an even / odd tile's queries
    float nD[2][128];
    uint64_t bar[NUM_BARS];
    ItemRing items;
    uint32_t tmem_base;
    int abort;
};
static_assert(kTiles % 1024 == 0 && kTiles + sizeof(Ctrl) <= 232448, "tiles and control block fit the 227 KB of a CTA");

}  // namespace kv

template <bool kCube>
__global__ void __launch_bounds__(kThreads, 1) sparse_bwd_dkdv_tc_kernel(const __grid_constant__ CUtensorMap map_k,
                                                                         const __grid_constant__ CUtensorMap map_v,
                                                                         const __grid_constant__ CUtensorMap map_q,
                                                                         const __grid_constant__ CUtensorMap map_o,
                                                                         const Params p)
{
    using namespace kv;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if (smem_u32(smem_raw) & 1023u) {
        if (threadIdx.x == 0) atomicCAS(&p.status->code, 0, (int)ROLA_ERR_UNSUPPORTED);
        return;
    }
    Ctrl& sm = *reinterpret_cast<Ctrl*>(smem_raw + kTiles);
    const uint32_t sbase = smem_u32(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar = [&](int i) { return smem_u32(&sm.bar[i]); };
    const Shape& s = p.s;
    const int nB = s.nB;
    // the query blocks that kept key block kb of head bh: l[0 .. len)
    auto range = [&](int item, int& bh, int& kb, int& len) -> const int32_t* {
        bh = item / nB;
        kb = item - bh * nB;
        const int32_t* o = p.off + (size_t)bh * (nB + 1) + kb;
        const int e0 = __ldg(o);
        len = __ldg(o + 1) - e0;
        return p.list + (size_t)bh * nB * s.n_keep + e0;
    };

    if (tid == 0) {
        sm.abort = 0;
        for (int i = 0; i < NUM_BARS; ++i) {
            const bool by_warps = i == P_FULL || i == DS_FULL || i == ACC_EMPTY;
            const bool q_full = i >= Q_FULL && i < Q_FULL + QS;       // the Q pair and the tile's lse, D
            mbar_init(bar(i), by_warps ? kDsWarps : (q_full ? 2 : 1));
        }
        sm.items.init();
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
        tmem_relinquish();
    }
    if (warp == kProdAWarp && lane == 0) {
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_o);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    chain_begin();
    volatile int* abort = &sm.abort;
    // the CTA's i-th item, for a single-thread role and for a warp
    auto item_at = [&](int i, bool& ok) { return sm.items.get<true>(i, ok, abort, s.wait_limit_ns); };
    auto item_at_warp = [&](int i, bool& ok) { return sm.items.get<false>(i, ok, abort, s.wait_limit_ns); };

    if (warp == kProdAWarp || warp == kProdBWarp) {
        // ------------------------------------------------------------ TMA: K, V and the Q pairs / the dO pairs
        const bool is_o = warp == kProdBWarp;
        const int NS = is_o ? OS : QS;
        const uint32_t ring = is_o ? kSmO : kSmQ;
        const int full0 = is_o ? O_FULL : Q_FULL, empty0 = is_o ? O_EMPTY : Q_EMPTY;
        const CUtensorMap* map = is_o ? &map_o : &map_q;
        if (elect_one()) {
            int k = 0, issued_kv = 0, issued = 0;
            bool ok = true;
            // (the Q warp hands out the items: the next one is known, the one after asked for; i counts
            // them, k those that some query block kept)
            int next = 0, after = 0;
            int* counter = &p.status->next[kItemsDkDv];
            if (!is_o) {
                sm.items.post(0, blockIdx.x, abort, s.wait_limit_ns);
                next = gridDim.x + atomicAdd(counter, 1);
            }
            auto advance = [&](int i) {                       // the item after the i-th
                if (is_o) return item_at(i + 1, ok);
                const int x = next;
                next = after;
                return x;
            };
            int i = 0;
            for (int item = is_o ? item_at(0, ok) : (int)blockIdx.x; item < p.total_items && ok; item = advance(i), ++i) {
                if (!is_o) {
                    if (!(ok = sm.items.post(i + 1, next, abort, s.wait_limit_ns))) break;
                    after = gridDim.x + atomicAdd(counter, 1);
                }
                int bh, kb, len;
                const int32_t* l = range(item, bh, kb, len);
                if (len == 0) continue;
                if (!is_o) {
                    const int ks = k & 1;
                    if (k >= 2 && !(ok = mbar_wait(bar(KV_EMPTY + ks), ((k >> 1) - 1) & 1, abort, s.wait_limit_ns))) break;
                    mbar_expect_tx(bar(KV_FULL + ks), 2 * kBlockBytes);
                    tma_load_4d(sbase + kSmK + ks * kBlockBytes, &map_k, bar(KV_FULL + ks), 0, kb * 64, 0, bh);
                    tma_load_4d(sbase + kSmV + ks * kBlockBytes, &map_v, bar(KV_FULL + ks), 0, kb * 64, 0, bh);
                    ++issued_kv;
                }
                const int T = (len + 1) / 2;
                int qa_n = __ldg(l), qb_n = len > 1 ? __ldg(l + 1) : -1;      // block ids, one tile ahead
                for (int t = 0; t < T; ++t) {
                    const int g = issued, st = g % NS;
                    const int ra = qa_n * 64, rb = qb_n * 64;
                    const bool two = qb_n >= 0;
                    if (t + 1 < T) {
                        qa_n = __ldg(l + 2 * t + 2);
                        qb_n = 2 * t + 3 < len ? __ldg(l + 2 * t + 3) : -1;
                    }
                    if (g >= NS && !(ok = mbar_wait(bar(empty0 + st), ((g / NS) - 1) & 1, abort, s.wait_limit_ns))) break;
                    ++issued;
                    // test hook: the CTA's first Q / dO pair is never loaded, so the waits on it run out
                    if ((s.debug_flags & ROLA_DEBUG_SKIP_FIRST_K_COPY) && g == 0) continue;
                    mbar_expect_tx(bar(full0 + st), two ? 32768u : 16384u);
                    load_pair(sbase + ring + st * kPairBytes, map, bar(full0 + st), ra, rb, two, bh);
                }
                ++k;
            }
            if (!ok) record_timeout(p, is_o ? 36 : 33);
            // every copy this thread issued lands before the CTA exits (bounded by time only)
            int never = 0;
            for (int u = issued_kv > 2 ? issued_kv - 2 : 0; u < issued_kv; ++u)
                mbar_wait(bar(KV_FULL + (u & 1)), (u >> 1) & 1, &never, s.wait_limit_ns);
            for (int u = issued > NS ? issued - NS : 0; u < issued; ++u)
                mbar_wait(bar(full0 + u % NS), (u / NS) & 1, &never, s.wait_limit_ns);
        }
    } else if (warp == kStatWarp) {
        // ------------------------------------------------------------ log-sum-exp and -D of each tile's queries
        // lane i: queries i and i + 32 of either block (an empty slot or an absent
        // block: lse = +inf, so its P is 0); read one tile ahead
        int g = 0;
        bool ok = true;
        for (int it = 0, item = item_at_warp(0, ok); item < p.total_items && ok; item = item_at_warp(++it, ok)) {
            int bh, kb, len;
            const int32_t* l = range(item, bh, kb, len);
            const int T = (len + 1) / 2;
            float a[4], b[4];
            auto fetch = [&](int t) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = 2 * t + (i >> 1), slot = (i & 1) * 32 + lane;
                    const int blk = e < len ? __ldg(l + e) : -1;
                    const bool v = blk >= 0 && slot_token_g<kCube>(s, blk, slot) >= 0;
                    const size_t r = (size_t)bh * s.Np + (size_t)(v ? blk : 0) * 64 + (v ? slot : 0);
                    a[i] = v ? __ldg(p.lse + r) * kLog2e : CUDART_INF_F;
                    b[i] = v ? -__ldg(p.Dv + r) : 0.0f;
                }
            };
            if (len > 0) fetch(0);
            for (int t = 0; t < T; ++t, ++g) {
                // dK(g - 2) is done, so dS(g - 2) was evaluated and the buffer is free
                if (g >= 2 && !(ok = mbar_wait(bar(Q_EMPTY + (g - 2) % QS), ((g - 2) / QS) & 1, abort, s.wait_limit_ns)))
                    break;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sm.lse2[g & 1][i * 32 + lane] = a[i];
                    sm.nD[g & 1][i * 32 + lane] = b[i];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(Q_FULL + g % QS));
                if (t + 1 < T) fetch(t + 1);
            }
        }
        if (!ok && lane == 0) record_timeout(p, 37);
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ S(g), dK(g - 1), dP(g), dV(g), tile by tile
        if (elect_one()) {
            const uint32_t id_s = idesc_bf16(64, 64, false, false), id_g = idesc_bf16(64, 128, false, true);
            const uint64_t dk = smem_desc(sbase, 16, 1024);          // K-major operands
            const uint64_t dm = smem_desc(sbase, 16384, 1024);       // a pair read MN-major (chunks 16 KB apart)
            const uint32_t lo = (uint32_t)dk, hi = (uint32_t)(dk >> 32), mlo = (uint32_t)dm, mhi = (uint32_t)(dm >> 32);
            bool ok = true;
            int k = 0, g = 0;
            bool due = false, prev_half = false, prev_first = false, prev_last = false;
            // dK += dS^T Q of the tile before tile g, unless it was issued already
            auto grad_k = [&]() -> bool {
                if (!due) return true;
                const int u = g - 1;
                if (!mbar_wait(bar(DS_FULL), u & 1, abort, s.wait_limit_ns)) return false;
                fence_after_sync();
                const uint32_t b = mlo + ((kSmQ + (u % QS) * kPairBytes) >> 4);
                mma_grad(tmem + kDK, tmem + kDP, b, mhi, id_g, prev_first);
                mma_commit(bar(DK_HALF));
                if (!prev_half) mma_grad(tmem + kDK, tmem + kDP + 64, b + kSecond, mhi, id_g, false);
                mma_commit(bar(Q_EMPTY + u % QS));
                if (prev_last) mma_commit(bar(ACC_FULL));
                due = false;
                return true;
            };
            for (int i = 0, item = item_at(0, ok); item < p.total_items && ok; item = item_at(++i, ok)) {
                int bh, kb, len;
                range(item, bh, kb, len);
                if (len == 0) {
                    // the epilogue of the item before waits for this dK and reads no item until it has it, so
                    // the ring may end before the next item that has tiles
                    if (!(ok = grad_k())) break;
                    continue;
                }
                const int T = (len + 1) / 2, kbuf = k & 1;
                if (!(ok = mbar_wait(bar(KV_FULL + kbuf), (k >> 1) & 1, abort, s.wait_limit_ns))) break;
                const uint32_t ka = lo + ((kSmK + kbuf * kBlockBytes) >> 4), va = lo + ((kSmV + kbuf * kBlockBytes) >> 4);
                for (int t = 0; t < T; ++t, ++g) {
                    const int qs = g % QS, os = g % OS;
                    const bool half = 2 * t + 1 >= len;
                    const uint32_t q = lo + ((kSmQ + qs * kPairBytes) >> 4), o = lo + ((kSmO + os * kPairBytes) >> 4);
                    if (!(ok = mbar_wait(bar(Q_FULL + qs), (g / QS) & 1, abort, s.wait_limit_ns))) break;
                    // S goes where P of the tile before was, block by block once dV has read it
                    if (g >= 1 && !(ok = mbar_wait(bar(DV_HALF), (g - 1) & 1, abort, s.wait_limit_ns))) break;
                    fence_after_sync();
                    mma_scores(tmem + kS, ka, hi, q, hi, id_s);
                    if (g >= 1 && !(ok = mbar_wait(bar(O_EMPTY + (g - 1) % OS), ((g - 1) / OS) & 1, abort, s.wait_limit_ns)))
                        break;
                    fence_after_sync();
                    mma_scores(tmem + kS + 64, ka, hi, q + kSecond, hi, id_s);
                    mma_commit(bar(S_FULL));
                    if (!(ok = grad_k())) break;
                    if (!(ok = mbar_wait(bar(O_FULL + os), (g / OS) & 1, abort, s.wait_limit_ns))) break;
                    // dP goes where dS of the tile before was, once dK has read it
                    if (g >= 1 && !(ok = mbar_wait(bar(DK_HALF), (g - 1) & 1, abort, s.wait_limit_ns))) break;
                    fence_after_sync();
                    mma_scores(tmem + kDP, va, hi, o, hi, id_s);
                    if (g >= 1 && !(ok = mbar_wait(bar(Q_EMPTY + (g - 1) % QS), ((g - 1) / QS) & 1, abort, s.wait_limit_ns)))
                        break;
                    fence_after_sync();
                    mma_scores(tmem + kDP + 64, va, hi, o + kSecond, hi, id_s);
                    mma_commit(bar(DP_FULL));
                    if (t == T - 1) mma_commit(bar(KV_EMPTY + kbuf));
                    if (t == 0 && k >= 1 && !(ok = mbar_wait(bar(ACC_EMPTY), (k - 1) & 1, abort, s.wait_limit_ns))) break;
                    if (!(ok = mbar_wait(bar(P_FULL), g & 1, abort, s.wait_limit_ns))) break;
                    fence_after_sync();
                    const uint32_t om = mlo + ((kSmO + os * kPairBytes) >> 4);
                    mma_grad(tmem + kDV, tmem + kS, om, mhi, id_g, t == 0);
                    mma_commit(bar(DV_HALF));
                    if (!half) mma_grad(tmem + kDV, tmem + kS + 64, om + kSecond, mhi, id_g, false);
                    mma_commit(bar(O_EMPTY + os));
                    prev_half = half;
                    prev_first = t == 0;
                    prev_last = t == T - 1;
                    due = true;
                }
                if (!ok) break;
                ++k;
            }
            if (ok) ok = grad_k();
            if (!ok) record_timeout(p, 34);
            // every product this thread issued completes before TMEM is released
            int never = 0;
            mma_commit(bar(DRAIN));
            mbar_wait(bar(DRAIN), 0, &never, s.wait_limit_ns);
        }
    } else if (warp < kDsWarps) {
        // ------------------------------------------------------------ P, dS + epilogue
        const int wg = warp >> 2, quarter = warp & 3, hf = lane >> 4;
        const int row = 16 * quarter + (lane & 15), d0 = 64 * wg + 32 * hf;   // d0: this thread's tile columns too
        const float c_log2 = s.sm_scale_log2;
        const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16);
        bool ok = true;
        int k = 0, g = 0;
        for (int i = 0, item = item_at_warp(0, ok); item < p.total_items && ok; item = item_at_warp(++i, ok)) {
            int bh, kb, len;
            range(item, bh, kb, len);
            const int T = (len + 1) / 2;
            const int n = slot_token_g<kCube>(s, kb, row);            // this row's token, -1 for an empty slot
            const size_t at = ((size_t)bh * s.N + (n >= 0 ? n : 0)) * kDh + d0;
            prefetch_l2(p.lr0 + at);                                   // this thread's row parts of the epilogue
            prefetch_l2(p.lr1 + at);
            for (int t = 0; t < T; ++t, ++g) {
                float x[kCols], y[kCols];
                if (!(ok = mbar_wait(bar(Q_FULL + g % QS), (g / QS) & 1, abort, s.wait_limit_ns))) break;   // lse, D are there
                if (!(ok = mbar_wait(bar(S_FULL), g & 1, abort, s.wait_limit_ns))) break;
                fence_after_sync();
                ld_cols(base + kS + 64 * wg, x);
#pragma unroll
                for (int i = 0; i < kCols; i += 4) {
                    const float4 l = *reinterpret_cast<const float4*>(&sm.lse2[g & 1][d0 + i]);
                    x[i] = fast_exp2(fmaf(x[i], c_log2, -l.x));
                    x[i + 1] = fast_exp2(fmaf(x[i + 1], c_log2, -l.y));
                    x[i + 2] = fast_exp2(fmaf(x[i + 2], c_log2, -l.z));
                    x[i + 3] = fast_exp2(fmaf(x[i + 3], c_log2, -l.w));
                }
                st_cols(base + kS + 64 * wg, x);                      // P over this group's own columns of S
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(P_FULL));
                if (!(ok = mbar_wait(bar(DP_FULL), g & 1, abort, s.wait_limit_ns))) break;
                fence_after_sync();
                ld_cols(base + kDP + 64 * wg, y);
#pragma unroll
                for (int i = 0; i < kCols; i += 4) {
                    const float4 D = *reinterpret_cast<const float4*>(&sm.nD[g & 1][d0 + i]);
                    fadd2(y[i], y[i + 1], D.x, D.y);
                    fadd2(y[i + 2], y[i + 3], D.z, D.w);
                    fmul2(y[i], y[i + 1], x[i], x[i + 1]);
                    fmul2(y[i + 2], y[i + 3], x[i + 2], x[i + 3]);
                }
                st_cols(base + kDP + 64 * wg, y);                     // dS over dP
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(DS_FULL));
            }
            if (!ok) break;
            // ---- epilogue: dk = low-rank row + R(p)^T (dK / sqrt d), dv = low-rank row + dV; this
            // thread's 32 columns of its row.  A key block no query block kept has the low-rank
            // rows alone.
            float lr[kCols], v[kCols], w[kCols];
            float2 cs[16];
            load_row32(p.lr1 + at, lr);
            load_cs(p, n >= 0 ? n : 0, d0, cs);
            if (len > 0) {
                if (!(ok = mbar_wait(bar(ACC_FULL), k & 1, abort, s.wait_limit_ns))) break;
                fence_after_sync();
                ld_cols(base + kDV + 64 * wg, w);
                ld_cols(base + kDK + 64 * wg, v);
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(ACC_EMPTY));
                ++k;
            } else {
#pragma unroll
                for (int i = 0; i < kCols; ++i) v[i] = w[i] = 0.0f;
            }
            if (n >= 0) {
#pragma unroll
                for (int i = 0; i < kCols; ++i) lr[i] += w[i];
                store_row32(p.out1 + at, lr);
                load_row32(p.lr0 + at, lr);
                rotate_back32(v, lr, cs);
                store_row32(p.out0 + at, v);
            }
        }
        if (!ok) record_timeout(p, 35);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
}

// One persistent CTA per SM (fewer when there are fewer items).
template <typename Kernel>
cudaError_t launch(Kernel kernel, size_t smem, const CUtensorMap (&m)[4], const Params& p, cudaStream_t st)
{
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    launch_kernel(kernel, p.total_items < nsm ? p.total_items : nsm, kThreads, smem, st, m[0], m[1], m[2], m[3], p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sparse_bwd_dq_tc(const Shape& s, const void* qr, const void* kr, const void* v, const void* dOs,
                                    const int32_t* kv_idx, const float* lse, const float* Dv, const float2* tab,
                                    const float* dq_lr, void* dq, DeviceStatus* status, cudaStream_t st)
{
    // the maps span the block-ordered rows (the token order itself for contiguous chunks)
    Shape rows = s;
    rows.N = s.Np;
    CUtensorMap m[4];
    if (!make_block_map(&m[0], qr, rows) || !make_block_map(&m[1], dOs, rows) || !make_chunk_map(&m[2], kr, rows) ||
        !make_chunk_map(&m[3], v, rows))
        return cudaErrorInvalidValue;
    Params p = {};
    p.s = s;
    p.kv_idx = kv_idx;
    p.lse = lse;
    p.Dv = Dv;
    p.lr0 = dq_lr;
    p.tab = tab;
    p.out0 = static_cast<__nv_bfloat16*>(dq);
    p.status = status;
    p.total_items = s.B * s.H * s.nB;
    return launch(s.cube ? sparse_bwd_dq_tc_kernel<true> : sparse_bwd_dq_tc_kernel<false>, dq::kTiles + sizeof(dq::Ctrl),
                  m, p, st);
}

cudaError_t launch_sparse_bwd_dkdv_tc(const Shape& s, const void* qr, const void* kr, const void* v, const void* dOs,
                                      const int32_t* off, const int32_t* list, const float* lse, const float* Dv,
                                      const float2* tab, const float* dk_lr, const float* dv_lr, void* dk, void* dv,
                                      DeviceStatus* status, cudaStream_t st)
{
    Shape rows = s;
    rows.N = s.Np;
    CUtensorMap m[4];
    if (!make_block_map(&m[0], kr, rows) || !make_block_map(&m[1], v, rows) || !make_chunk_map(&m[2], qr, rows) ||
        !make_chunk_map(&m[3], dOs, rows))
        return cudaErrorInvalidValue;
    Params p = {};
    p.s = s;
    p.off = off;
    p.list = list;
    p.lse = lse;
    p.Dv = Dv;
    p.lr0 = dk_lr;
    p.lr1 = dv_lr;
    p.tab = tab;
    p.out0 = static_cast<__nv_bfloat16*>(dk);
    p.out1 = static_cast<__nv_bfloat16*>(dv);
    p.status = status;
    p.total_items = s.B * s.H * s.nB;
    return launch(s.cube ? sparse_bwd_dkdv_tc_kernel<true> : sparse_bwd_dkdv_tc_kernel<false>,
                  kv::kTiles + sizeof(kv::Ctrl), m, p, st);
}

}  // namespace rola
