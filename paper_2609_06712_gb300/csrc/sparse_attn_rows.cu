// Block-sparse softmax attention, one softmax thread (pair) per query row
// (kernel 2, bf16).
//
//   O^s_p = sum_{q in kept(i)} softmax_q(q^r_p . k^r_q / sqrt(d_h)) v_q,   p in query block i
//
// (Sec. 3 softmax form restricted to the kept key blocks, Alg. 1 sparse
// branch.)  Query blocks of QN = 64 tokens (the mask of Alg. 1) or QN = 128
// tokens (a mask chosen per 128-token chunk); key blocks are 64 tokens.  With
// cube blocks (kCube) q^r, k^r and v come in block order, 64 slots a cube, so a
// cube is one box like a chunk; empty slots are masked out of the softmax and
// each O^s row goes to its slot's token.
//
// An item (one query block of one head) is the M = QN rows of tcgen05 MMAs:
//   S    = Q (QN q x 128 d, smem, K-major)  x  K_pair^T (N = 128 keys, smem, K-major)
//   O   += P (QN q x 128 keys, TMEM, bf16)  x  V_pair (N = 128 d, smem, MN-major)
// S, P and O live in TMEM with one query row per TMEM lane (M = 128: lanes
// 0-127; M = 64: lanes 0-15 of each 32-lane quarter, row r at lane
// 32 (r / 16) + r mod 16).  The softmax reads its row of S, keeps the row
// maximum and the row sum in registers and writes P back to TMEM as packed
// bf16 (the lower key in the low half), the A operand of the P V product, so
// no P tile passes through shared memory.  For QN = 128 a thread owns a row
// (128 keys); for QN = 64 the two half-warps share the 16 rows of their
// quarter, threads 0-15 taking keys 0-63 and threads 16-31 keys 64-127 of
// the same rows (the 16x32bx2 TMEM access shape), and combine the row maximum
// and the row sum with one shuffle.
//
// Softmax (lazy rescaling, base 2): two warpgroups take the tiles of an item
// in turn, so a tile's softmax may last two tile periods.  -m, the running
// maximum that both use for a row, goes from one to the other through shared
// memory (sm.m): after its tile's row maximum a warp waits for -m of the tile
// before, raises m if the tile's largest t = s log2(e)/sqrt(d) - m exceeds 2^3
// (or on the first tile of the item), and passes it on before it evaluates the
// exponentials.  A raised m scales the O row by 2^(m_old - m_new), after the
// previous P V has finished and before this tile's P is handed over (a warp
// takes that path when any of its rows needs it).  Each group keeps the row
// sum of its own tiles; the group of the item's last tile adds the other's and
// writes O.  p = 2^t enters the row sum in fp32 and the product rounded to bf16.
//
// Warp roles (384 threads, one persistent CTA per SM):
//   warps 0-3, 4-7  softmax of the even / odd tiles of the CTA + epilogue: warp w owns TMEM lane quarter w mod 4
//   warp  8    TMA producer: Q (per item) and the K pairs
//   warp  9    TMA producer: the V blocks
//   warp 10    S = Q K^T issuer and TMEM owner
//   warp 11    O += P V issuer
// (QN = 128: the softmax groups hold 128 scores a thread, so they take 208
// registers and leave the last warpgroup 88.)
// Buffers (shared memory): Q (QN = 64: two 16 KB buffers, so the next item's
// Q arrives during this one; QN = 128: one of 32 KB), K pairs in a 3-deep
// ring (32 KB each), V blocks in a ring of single 16 KB blocks (6 for QN = 64,
// 5 for 128): 224 / 208 KB.  TMEM (512 columns): S double-buffered (2 x 128),
// O (128), P double-buffered (2 x 64 columns of bf16 pairs), so Q K^T of the
// next tile runs while the softmax of this one does.  Every mbarrier wait is
// bounded; a wait that gives up records ROLA_ERR_TIMEOUT in the status word
// and the CTA stops issuing, drains what it issued and releases its TMEM.
//
// What bounds it, measured at the 720p layer (40 heads, 75600 tokens, 118 of
// 1182 blocks kept; clock64 around every wait of one CTA):
//   - a producer warp that predicates each step on lanes spends ~640 cycles a
//     16 KB block on fixed latencies (mbarrier wait 110-170, expect_tx ~50, a TMA
//     instruction 80), whatever the ring's depth; one elected thread that keeps
//     the next block ids in registers needs ~350 for two boxes.  14.76 -> 11.85
//     ms (QN = 64); the L2 itself delivers a 16 KB block per 248 cycles and SM.
//   - two softmax groups in turn: 11.85 -> 11.5 ms (QN = 64), 8.2 -> 7.3 ms (QN = 128).
//   - cube blocks on this kernel instead of a transposed form of their own: 4.88 ->
//     3.43 ms (40 heads, 21 x 30 x 52 grid, 62 of 624 cubes kept).
//   - items off a counter instead of dealt out evenly: 11.5 -> 11.1 ms (QN = 64).
//   - QN = 64 takes ~1240 cycles a tile: 1024 of tensor work (an M = 64 product
//     runs at half the M = 128 rate) and 144 KB through the shared memory (1125 at
//     128 B/cycle).  QN = 128 takes ~1350 against the same 1024.  The 1400 W power
//     cap sets the clock: 1.95-2.03 GHz for QN = 64, 1.72-1.82 GHz for QN = 128,
//     whose 1650-1700 TFLOP/s (7.1-6.9 ms, by the clock) are 0.95-0.98 of the rate a
//     GEMM sustains under that cap.
//
// Per 64-query block and 128-key tile the shared memory sees 64 KB of TMA
// writes (K, V) and 80 KB of operand reads (Q 16, K 32, V 32) for 4.2 MFLOP,
// against 176 KB in a transposed form (S^T with M = 128 keys, P^T through
// shared memory); an M = 64 MMA runs at half the M = 128 rate.
#include <cudaTypedefs.h>
#include <stddef.h>

#include "common.cuh"
#include "tcgen05.cuh"
#include "tensor_map.cuh"

namespace rola {
namespace {

using namespace tc;

constexpr int kWarpsPerGroup = 4;                    // a softmax warpgroup
constexpr int kProducerKWarp = 8, kProducerVWarp = 9, kMmaWarp = 10, kPvWarp = 11;
constexpr int kThreads = 384;
constexpr uint32_t kKPairBytes = 128 * 128 * 2;      // a pair of key blocks [d-chunk][block][64 rows][64]
constexpr uint32_t kVBlockBytes = 64 * 128 * 2;      // one key block of v [d-chunk][64 rows][64]
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemS = 0;                       // S buffers at 0, 128
constexpr uint32_t kTmemO = 256;
constexpr uint32_t kTmemP = 384;                     // P buffers at 384, 448 (64 columns: 128 bf16 keys)
constexpr float kRescaleThreshold = 8.0f;            // log2 units

template <int QN>
struct Cfg {
    static_assert(QN == 64 || QN == 128, "query blocks of 64 or 128 rows");
    static constexpr int QB = QN == 64 ? 2 : 1;                  // Q buffers
    static constexpr int KS = 3;                                 // K ring (pairs)
    static constexpr int VB = QN == 64 ? 6 : 5;                  // V ring (single blocks)
    static constexpr int kCols = QN == 64 ? 64 : 128;            // keys of a tile per softmax thread
    static constexpr uint32_t kQBytes = QN * 128 * 2;            // [d-chunk][QN rows][64]
    static constexpr uint32_t kSmemQ = 0;
    static constexpr uint32_t kSmemK = kSmemQ + QB * kQBytes;
    static constexpr uint32_t kSmemV = kSmemK + KS * kKPairBytes;
    static constexpr uint32_t kSmemTiles = kSmemV + VB * kVBlockBytes;
    static constexpr int Q_FULL = 0, Q_EMPTY = Q_FULL + QB, K_FULL = Q_EMPTY + QB, K_EMPTY = K_FULL + KS,
                         V_FULL = K_EMPTY + KS, V_EMPTY = V_FULL + VB, S_FULL = V_EMPTY + VB, S_EMPTY = S_FULL + 2,
                         P_FULL = S_EMPTY + 2, PV_DONE = P_FULL + 2, O_FULL = PV_DONE + 4, O_EMPTY = O_FULL + 2,
                         M_READY = O_EMPTY + 1, L_READY = M_READY + 8, DRAIN = L_READY + 8, NUM_BARS = DRAIN + 2;
    static_assert(kSmemTiles % 1024 == 0, "the control block follows the 1024-aligned tiles");
};

template <int QN>
struct Ctrl {
    float m[2][QN];                      // -m of every row after an even / odd tile
    float2 l[2][QN];                     // (row sum, its -m) of the group that does not end item k, by k & 1
    uint64_t bar[Cfg<QN>::NUM_BARS];
    ItemRing items;
    uint32_t tmem_base;
    int abort;
};
static_assert(Cfg<64>::kSmemTiles + sizeof(Ctrl<64>) <= 232448 && Cfg<128>::kSmemTiles + sizeof(Ctrl<128>) <= 232448,
              "tiles and control block fit the 227 KB a CTA may have");

struct Params {
    Shape s;
    const int32_t* kv_idx;   // [B*H][nQ][n_keep]
    __nv_bfloat16* o;        // O^s [B*H][N][128]
    float* lse;              // nullable: log-sum-exp per query row (natural log)
    DeviceStatus* status;
    int items_per_head;      // query blocks per (batch, head) = rows of the mask
    int total_items;         // B*H*items_per_head
    int tiles;               // ceil(n_keep / 2)
};

__device__ __forceinline__ void record_timeout(const Params& p, int where)
{
    if (atomicCAS(&p.status->code, 0, (int)ROLA_ERR_TIMEOUT) == 0) p.status->where = where;
}

// A softmax thread's NC consecutive columns of its row starting at column c0:
// 32x32b for QN = 128 (the thread's own lane), 16x32bx2 with the half-warp
// split at column c0 + NC for QN = 64.
template <int QN, int NC>
__device__ __forceinline__ void row_load(uint32_t taddr, float (&v)[NC])
{
    static_assert(NC % 16 == 0, "loads of 16 columns");
#pragma unroll
    for (int c = 0; c < NC / 16; ++c) {
        float(&part)[16] = *reinterpret_cast<float(*)[16]>(&v[c * 16]);
        if constexpr (QN == 128) tmem_ld16(taddr + c * 16, part);
        else tmem_ld16_half<NC>(taddr + c * 16, part);
    }
    tmem_ld_wait(*reinterpret_cast<float(*)[16]>(&v[0]));
#pragma unroll
    for (int c = 1; c < NC / 16; ++c) reg_fence(*reinterpret_cast<float(*)[16]>(&v[c * 16]));
}
template <int QN, int NC>
__device__ __forceinline__ void row_store(uint32_t taddr, const float (&v)[NC])
{
#pragma unroll
    for (int c = 0; c < NC / 16; ++c) {
        const float(&part)[16] = *reinterpret_cast<const float(*)[16]>(&v[c * 16]);
        if constexpr (QN == 128) tmem_st16(taddr + c * 16, part);
        else tmem_st16_half<NC>(taddr + c * 16, part);
    }
}

// Moves registers between the warpgroups (executed by all warps of one).
template <int R>
__device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(R)); }
template <int R>
__device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(R)); }

template <int QN, bool kCube>
__global__ void __launch_bounds__(kThreads, 1) sparse_attn_rows_kernel(const __grid_constant__ CUtensorMap map_q,
                                                                       const __grid_constant__ CUtensorMap map_k,
                                                                       const __grid_constant__ CUtensorMap map_v,
                                                                       const Params p)
{
    using C = Cfg<QN>;
    constexpr int QB = C::QB, KS = C::KS, VB = C::VB, NC = C::kCols;
    constexpr uint32_t kQBytes = C::kQBytes, kSmemQ = C::kSmemQ, kSmemK = C::kSmemK, kSmemV = C::kSmemV;
    constexpr int Q_FULL = C::Q_FULL, Q_EMPTY = C::Q_EMPTY, K_FULL = C::K_FULL, K_EMPTY = C::K_EMPTY,
                  V_FULL = C::V_FULL, V_EMPTY = C::V_EMPTY, S_FULL = C::S_FULL, S_EMPTY = C::S_EMPTY,
                  P_FULL = C::P_FULL, PV_DONE = C::PV_DONE, O_FULL = C::O_FULL, O_EMPTY = C::O_EMPTY,
                  M_READY = C::M_READY, L_READY = C::L_READY, DRAIN = C::DRAIN;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // the 128-byte-swizzle atoms need a 1024-byte aligned base; the kernel has
    // no static shared memory, so the dynamic block starts on the window base
    if (smem_u32(smem_raw) & 1023u) {
        if (threadIdx.x == 0) atomicCAS(&p.status->code, 0, (int)ROLA_ERR_UNSUPPORTED);
        return;
    }
    Ctrl<QN>& sm = *reinterpret_cast<Ctrl<QN>*>(smem_raw + C::kSmemTiles);
    const uint32_t sbase = smem_u32(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar = [&](int i) { return smem_u32(&sm.bar[i]); };

    const Shape& s = p.s;
    const int T = p.tiles;
    const int nI = p.items_per_head;

    if (tid == 0) {
        sm.abort = 0;
        for (int i = 0; i < QB; ++i) {
            mbar_init(bar(Q_FULL + i), 1);
            mbar_init(bar(Q_EMPTY + i), 1);
        }
        for (int i = 0; i < KS; ++i) {
            mbar_init(bar(K_FULL + i), 1);
            mbar_init(bar(K_EMPTY + i), 1);
        }
        for (int i = 0; i < VB; ++i) {
            mbar_init(bar(V_FULL + i), 1);
            mbar_init(bar(V_EMPTY + i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(S_FULL + i), 1);
            mbar_init(bar(S_EMPTY + i), kWarpsPerGroup);
            mbar_init(bar(P_FULL + i), kWarpsPerGroup);
            mbar_init(bar(O_FULL + i), 1);
            mbar_init(bar(DRAIN + i), 1);
        }
        for (int i = 0; i < 4; ++i) mbar_init(bar(PV_DONE + i), 1);
        for (int i = 0; i < 8; ++i) {
            mbar_init(bar(M_READY + i), 1);
            mbar_init(bar(L_READY + i), 1);
        }
        mbar_init(bar(O_EMPTY), kWarpsPerGroup);
        sm.items.init();
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
        tmem_relinquish();
    }
    if (warp == kProducerKWarp && lane == 0) {
        tma_prefetch_desc(&map_q);
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

    if constexpr (QN == 128) {
        if (warp >= kProducerKWarp) regs_dec<88>();    // the softmax groups take 208: 208 + 208 + 88 = 3 x 168
    }
    if (warp == kProducerKWarp || warp == kProducerVWarp) {
        // ------------------------------------------------------------ TMA producers
        // One elected thread per warp.  K warp: Q (one box per item) and the K
        // pairs, 8 KB boxes in [chunk][block][row] order so that the pair is
        // one N = 128 operand.  V warp: a 16 KB box ([chunk][row]) per block
        // into its slot of the ring of single blocks.
        const bool is_v = warp == kProducerVWarp;
        if (elect_one()) {
            int k = 0, g = 0, issued_q = 0, issued = 0;
            bool ok = true;
            // (the K warp hands out the items: the next one is known, the one after asked for)
            int item = is_v ? item_at(0, ok) : (int)blockIdx.x, next = 0;
            int* counter = &p.status->next[kItemsForward];
            if (!is_v) {
                sm.items.post(0, item, abort, s.wait_limit_ns);
                next = gridDim.x + atomicAdd(counter, 1);
            }
            for (; item < p.total_items && ok; ++k) {
                const int bh = item / nI, qb = item - bh * nI;
                const int32_t* kept = p.kv_idx + (size_t)item * s.n_keep;
                int ja_n = __ldg(kept), jb_n = s.n_keep > 1 ? __ldg(kept + 1) : -1;     // block ids, one tile ahead
                if (!is_v) {
                    const int qs = k % QB;
                    if (k >= QB && !(ok = mbar_wait(bar(Q_EMPTY + qs), ((k / QB) - 1) & 1, abort, s.wait_limit_ns)))
                        break;
                    mbar_expect_tx(bar(Q_FULL + qs), kQBytes);
                    tma_load_4d(sbase + kSmemQ + qs * kQBytes, &map_q, bar(Q_FULL + qs), 0, qb * QN, 0, bh);
                    ++issued_q;
                }
                int after = 0;
                for (int t = 0; t < T; ++t, ++g) {
                    // (the first answer of the counter is given time: it is not needed before the second tile)
                    if (!is_v && t == (k == 0 && T > 1 ? 1 : 0)) {
                        if (!(ok = sm.items.post(k + 1, next, abort, s.wait_limit_ns))) break;
                        after = gridDim.x + atomicAdd(counter, 1);
                    }
                    const int ra = ja_n * 64, rb = jb_n * 64;
                    const bool two = jb_n >= 0;                 // the last tile of an odd n_keep holds one block
                    if (t + 1 < T) {
                        ja_n = __ldg(kept + 2 * t + 2);
                        jb_n = 2 * t + 3 < s.n_keep ? __ldg(kept + 2 * t + 3) : -1;
                    }
                    if (is_v) {
                        const int c = k * s.n_keep + 2 * t;     // cumulative block index of the tile's first block
                        const int sa = c % VB, sb = (c + 1) % VB;
                        if (c >= VB && !(ok = mbar_wait(bar(V_EMPTY + sa), ((c / VB) - 1) & 1, abort, s.wait_limit_ns)))
                            break;
                        mbar_expect_tx(bar(V_FULL + sa), kVBlockBytes);
                        tma_load_4d(sbase + kSmemV + sa * kVBlockBytes, &map_v, bar(V_FULL + sa), 0, ra, 0, bh);
                        issued = c + 1;
                        if (!two) continue;
                        if (c + 1 >= VB &&
                            !(ok = mbar_wait(bar(V_EMPTY + sb), (((c + 1) / VB) - 1) & 1, abort, s.wait_limit_ns)))
                            break;
                        mbar_expect_tx(bar(V_FULL + sb), kVBlockBytes);
                        tma_load_4d(sbase + kSmemV + sb * kVBlockBytes, &map_v, bar(V_FULL + sb), 0, rb, 0, bh);
                        issued = c + 2;
                    } else {
                        const int st = g % KS;
                        if (g >= KS && !(ok = mbar_wait(bar(K_EMPTY + st), ((g / KS) - 1) & 1, abort, s.wait_limit_ns)))
                            break;
                        issued = g + 1;
                        // test hook: the first K copy of the CTA is never issued, so the waits on it run out
                        if ((s.debug_flags & ROLA_DEBUG_SKIP_FIRST_K_COPY) && g == 0) continue;
                        const uint32_t dst = sbase + kSmemK + st * kKPairBytes, full = bar(K_FULL + st);
                        mbar_expect_tx(full, two ? 32768u : 16384u);
                        tma_load_3d(dst, &map_k, full, 0, ra, bh);
                        tma_load_3d(dst + 16384, &map_k, full, 64, ra, bh);
                        if (two) {
                            tma_load_3d(dst + 8192, &map_k, full, 0, rb, bh);
                            tma_load_3d(dst + 24576, &map_k, full, 64, rb, bh);
                        }
                    }
                }
                if (!ok) break;
                if (is_v) item = item_at(k + 1, ok);
                else item = next, next = after;
            }
            if (!ok) record_timeout(p, is_v ? 4 : 1);
            // every copy this thread issued lands before the CTA exits (bounded by time only)
            int never = 0;
            for (int u = issued_q > QB ? issued_q - QB : 0; u < issued_q; ++u)
                mbar_wait(bar(Q_FULL + u % QB), (u / QB) & 1, &never, s.wait_limit_ns);
            const int NS = is_v ? VB : KS;
            const int full0 = is_v ? V_FULL : K_FULL;
            for (int u = issued > NS ? issued - NS : 0; u < issued; ++u)
                mbar_wait(bar(full0 + u % NS), (u / NS) & 1, &never, s.wait_limit_ns);
        }
    } else if (warp == kMmaWarp || warp == kPvWarp) {
        // ------------------------------------------------------------ MMA issuers
        if (elect_one()) {
            const bool pv = warp == kPvWarp;
            const uint32_t id_qk = idesc_bf16(QN, 128, false, false);
            const uint32_t id_pv = idesc_bf16(QN, 128, false, true);
            const uint64_t dq = smem_desc(sbase + kSmemQ, 16, 1024);     // Q: A of Q K^T (K-major)
            const uint64_t dk = smem_desc(sbase + kSmemK, 16, 1024);     // K pair ring: B of Q K^T (K-major)
            const uint64_t dv = smem_desc(sbase + kSmemV, 8192, 1024);   // V block ring: B of P V (MN-major, d chunks 8 KB apart)
            const uint32_t q_lo = (uint32_t)dq, q_hi = (uint32_t)(dq >> 32);
            const uint32_t k_lo = (uint32_t)dk, k_hi = (uint32_t)(dk >> 32);
            const uint32_t v_lo = (uint32_t)dv, v_hi = (uint32_t)(dv >> 32);
            bool ok = true;
            int k = 0;
            for (int item = item_at(0, ok); item < p.total_items && ok; item = item_at(++k, ok)) {
                if (!pv) {
                    const int qs = k % QB;
                    if (!(ok = mbar_wait(bar(Q_FULL + qs), (k / QB) & 1, abort, s.wait_limit_ns))) break;
                    const uint32_t a = q_lo + qs * (kQBytes >> 4);
                    for (int t = 0; t < T; ++t) {
                        const int g = k * T + t, sb = g & 1, ks = g % KS;
                        if (!(ok = mbar_wait(bar(K_FULL + ks), (g / KS) & 1, abort, s.wait_limit_ns))) break;
                        if (g >= 2 && !(ok = mbar_wait(bar(S_EMPTY + sb), ((g >> 1) - 1) & 1, abort, s.wait_limit_ns)))
                            break;
                        fence_after_sync();
                        const uint32_t b = k_lo + ks * (kKPairBytes >> 4);
                        // K step kk: d-chunk kk / 4 (Q: QN rows of 128 B on, K pair: 16 KB on), 32 bytes per 16 d
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_ss_split(tmem + kTmemS + sb * 128, a + (kk >> 2) * (QN * 8) + (kk & 3) * 2, q_hi,
                                         b + (kk >> 2) * 1024 + (kk & 3) * 2, k_hi, id_qk, kk > 0 ? 1u : 0u);
                        mma_commit(bar(S_FULL + sb));
                        mma_commit(bar(K_EMPTY + ks));
                        if (t == T - 1) mma_commit(bar(Q_EMPTY + qs));
                    }
                } else {
                    for (int t = 0; t < T; ++t) {
                        const int g = k * T + t, pb = g & 1;
                        const bool half = 2 * t + 1 >= s.n_keep;
                        const int c0 = k * s.n_keep + 2 * t;
                        const int va = c0 % VB, vb = (c0 + 1) % VB;
                        // (V and O first: they are there long before P, whose wait is on the critical chain)
                        if (!(ok = mbar_wait(bar(V_FULL + va), (c0 / VB) & 1, abort, s.wait_limit_ns))) break;
                        if (!half && !(ok = mbar_wait(bar(V_FULL + vb), ((c0 + 1) / VB) & 1, abort, s.wait_limit_ns)))
                            break;
                        if (t == 0 && k >= 1 && !(ok = mbar_wait(bar(O_EMPTY), (k - 1) & 1, abort, s.wait_limit_ns)))
                            break;
                        if (!(ok = mbar_wait(bar(P_FULL + pb), (g >> 1) & 1, abort, s.wait_limit_ns))) break;
                        fence_after_sync();
                        // K step kk (16 keys): 8 TMEM columns of P, 2 KB of the V block
                        const uint32_t a = tmem + kTmemP + pb * 64;
                        const uint32_t b0 = v_lo + va * (kVBlockBytes >> 4), b1 = v_lo + vb * (kVBlockBytes >> 4);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_ts_split(tmem + kTmemO, a + kk * 8, b0 + kk * 128, v_hi, id_pv,
                                         (t > 0 || kk > 0) ? 1u : 0u);
                        if (!half) {
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                mma_ts_split(tmem + kTmemO, a + 32 + kk * 8, b1 + kk * 128, v_hi, id_pv, 1u);
                        }
                        mma_commit(bar(PV_DONE + (g & 3)));
                        mma_commit(bar(V_EMPTY + va));
                        if (!half) mma_commit(bar(V_EMPTY + vb));
                    }
                    if (!ok) break;
                    mma_commit(bar(O_FULL + (k & 1)));
                }
            }
            if (!ok) record_timeout(p, pv ? 5 : 2);
            // drain: every MMA this thread issued completes before TMEM is released
            int never = 0;
            const uint32_t drain = bar(pv ? DRAIN + 1 : DRAIN);
            mma_commit(drain);
            mbar_wait(drain, 0, &never, s.wait_limit_ns);
        }
    } else {
        // ------------------------------------------------------------ softmax + epilogue
        // QN = 128: thread wtid owns row wtid, keys 0-127 of a tile, d 0-127 of O.
        // QN = 64: thread (w, lane) owns row 16 w + lane mod 16, keys and d
        // [64 hf, 64 hf + 64) with hf = lane / 16 (its partner is lane ^ 16).
        if constexpr (QN == 128) regs_inc<208>();
        const int wg = warp >> 2, quarter = warp & 3, wtid = tid & 127;
        const int hf = QN == 64 ? lane >> 4 : 0;
        const int row = QN == 64 ? 16 * quarter + (lane & 15) : wtid;
        const float c_log2 = s.sm_scale_log2;
        const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
        const uint32_t s_addr = tmem + lane_off + kTmemS + wg * 128, p_addr = tmem + lane_off + kTmemP + wg * 64,
                       o_addr = tmem + lane_off + kTmemO;
        bool ok = true;
        int k = 0;
        for (int item = item_at_warp(0, ok); item < p.total_items && ok; item = item_at_warp(++k, ok)) {
            const int bh = item / nI, qb = item - bh * nI;
            const int32_t* kept = p.kv_idx + (size_t)item * s.n_keep;
            const int g0 = k * T;
            const int t0 = (g0 & 1) ^ wg;            // this group's first tile of the item (tiles t0, t0 + 2, ...)
            float neg_m = 0.0f;                      // -m (log2 units) of this row, as this group last used it
            float l0 = 0.0f, l1 = 0.0f, l2 = 0.0f, l3 = 0.0f;
            int ja_n = t0 < T ? __ldg(kept + 2 * t0) : 0;
            int jb_n = 2 * t0 + 1 < s.n_keep ? __ldg(kept + 2 * t0 + 1) : -1;
            for (int t = t0; t < T; t += 2) {
                const int g = g0 + t;
                const int ja = ja_n, jb = jb_n;
                if (t + 2 < T) {                     // kept ids of this group's next tile, one ahead
                    ja_n = __ldg(kept + 2 * t + 4);
                    jb_n = 2 * t + 5 < s.n_keep ? __ldg(kept + 2 * t + 5) : -1;
                }
                if (!(ok = mbar_wait(bar(S_FULL + wg), (g >> 1) & 1, abort, s.wait_limit_ns))) break;
                fence_after_sync();
                float x[NC];
                row_load<QN, NC>(s_addr, x);
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(S_EMPTY + wg));    // S buffer free for Q K^T(g + 2)
                // keys of the tile that are tokens; the others (a ragged block's end, an edge cube's empty
                // slots, the absent second block of a half tile) drop out of the maximum and the sum
                if constexpr (QN == 128) {
                    const int na = min(64, s.N - ja * 64), nb = jb >= 0 ? min(64, s.N - jb * 64) : 0;
                    if (na < 64 || nb < 64) {
#pragma unroll
                        for (int j = 0; j < 64; ++j) {
                            if (j >= na) x[j] = -INFINITY;
                            if (j >= nb) x[64 + j] = -INFINITY;
                        }
                    }
                } else {
                    const int blk = hf ? jb : ja;
                    const int left = blk >= 0 ? s.N - blk * 64 : 0;           // chunks: tokens from the block on
                    if (kCube || left < 64) {
                        const uint32_t m0 = block_mask32<kCube>(s, blk, 0), m1 = block_mask32<kCube>(s, blk, 1);
                        if (!kCube || (m0 & m1) != 0xffffffffu) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                if (!((m0 >> j) & 1u)) x[j] = -INFINITY;
                                if (!((m1 >> j) & 1u)) x[32 + j] = -INFINITY;
                            }
                        }
                    }
                }
                // the tile's row maximum (eight independent chains; the two halves of a row meet by shuffle)
                float mx[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) mx[i] = x[i];
#pragma unroll
                for (int j = 8; j < NC; ++j) mx[j & 7] = fmaxf(mx[j & 7], x[j]);
                float tile_max = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                                       fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
                if constexpr (QN == 64) tile_max = fmaxf(tile_max, __shfl_xor_sync(0xffffffffu, tile_max, 16));
                // the row's -m after tile g - 1, from the other group's warp of the same rows.  (The
                // wait is taken at an item's first tile too, where the value has no use: a group
                // publishes tile g + 1 only after the other has read tile g - 1.)
                if (g > 0 && !(ok = mbar_wait(bar(M_READY + 4 * (wg ^ 1) + quarter), ((g - 1) >> 1) & 1, abort,
                                              s.wait_limit_ns)))
                    break;
                const float neg_m_prev = t > 0 ? sm.m[wg ^ 1][row] : 0.0f;
                const bool need = t == 0 || fmaf(tile_max, c_log2, neg_m_prev) > kRescaleThreshold;
                const float neg_m_new = need ? -tile_max * c_log2 : neg_m_prev;
                if (hf == 0) sm.m[wg][row] = neg_m_new;
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(M_READY + 4 * wg + quarter));
                // this group's row sum follows m, whoever raised it
                if (t > 1 && __any_sync(0xffffffffu, neg_m_new != neg_m)) {
                    const float a = fast_exp2(neg_m_new - neg_m);
                    l0 *= a;
                    l1 *= a;
                    l2 *= a;
                    l3 *= a;
                }
                neg_m = neg_m_new;
                if (t > 0 && __any_sync(0xffffffffu, need)) {
                    // the O row must hold P V(g - 1) before it is scaled by 2^(m_old - m_new)
                    const float alpha = fast_exp2(neg_m_new - neg_m_prev);
                    if (!(ok = mbar_wait(bar(PV_DONE + ((g - 1) & 3)), ((g - 1) >> 2) & 1, abort, s.wait_limit_ns)))
                        break;
                    fence_after_sync();
                    // a thread holds as many d columns of its O row as it has keys of a tile
#pragma unroll
                    for (int c = 0; c < NC / 16; ++c) {
                        float ov[16];
                        if constexpr (QN == 128) tmem_ld16(o_addr + c * 16, ov);
                        else tmem_ld16_half<64>(o_addr + c * 16, ov);
                        tmem_ld_wait(ov);
#pragma unroll
                        for (int e = 0; e < 16; ++e) ov[e] *= alpha;
                        if constexpr (QN == 128) tmem_st16(o_addr + c * 16, ov);
                        else tmem_st16_half<64>(o_addr + c * 16, ov);
                    }
                    tmem_st_wait();
                }
                // p = 2^t, row sum in fp32, P packed to bf16 pairs (lower key in the low half)
                uint32_t pk[NC / 2];
#pragma unroll
                for (int j = 0; j < NC; j += 4) {
                    ffma2(x[j], x[j + 1], c_log2, neg_m);
                    ffma2(x[j + 2], x[j + 3], c_log2, neg_m);
                    const float p0 = fast_exp2(x[j]), p1 = fast_exp2(x[j + 1]);
                    const float p2 = fast_exp2(x[j + 2]), p3 = fast_exp2(x[j + 3]);
                    if ((j & 4) == 0) {
                        fadd2(l0, l1, p0, p1);
                        fadd2(l2, l3, p2, p3);
                    } else {
                        fadd2(l2, l3, p0, p1);
                        fadd2(l0, l1, p2, p3);
                    }
                    pk[j >> 1] = pack_bf16(p0, p1);
                    pk[(j >> 1) + 1] = pack_bf16(p2, p3);
                }
                // this group's P buffer is free once P V(g - 2) is done
                if (g >= 2 && !(ok = mbar_wait(bar(PV_DONE + ((g - 2) & 3)), ((g - 2) >> 2) & 1, abort,
                                               s.wait_limit_ns)))
                    break;
                row_store<QN, NC / 2>(p_addr, *reinterpret_cast<const float(*)[NC / 2]>(pk));
                tmem_st_wait();
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(P_FULL + wg));
            }
            if (!ok) break;
            float lsum = (l0 + l1) + (l2 + l3);
            if constexpr (QN == 64) lsum += __shfl_xor_sync(0xffffffffu, lsum, 16);
            if (((g0 + T - 1) & 1) != wg) {
                // the other group ends the item: it gets this group's share of the row sums
                if (T > 1) {
                    if (hf == 0) sm.l[k & 1][row] = make_float2(lsum, neg_m);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(L_READY + 4 * (k & 1) + quarter));
                }
                continue;
            }
            // ---- epilogue: O^s row = O / l
            if (T > 1) {
                if (!(ok = mbar_wait(bar(L_READY + 4 * (k & 1) + quarter), (k >> 1) & 1, abort, s.wait_limit_ns))) break;
                const float2 other = sm.l[k & 1][row];
                lsum = fmaf(other.x, fast_exp2(neg_m - other.y), lsum);
            }
            const int n = kCube ? slot_token_g<kCube>(s, qb, row) : (qb * QN + row < s.N ? qb * QN + row : -1);
            if (p.lse && hf == 0 && n >= 0) p.lse[(size_t)bh * s.N + n] = (log2f(lsum) - neg_m) * 0.6931471805599453f;
            const float inv_l = 1.0f / lsum;
            if (!(ok = mbar_wait(bar(O_FULL + (k & 1)), (k >> 1) & 1, abort, s.wait_limit_ns))) break;
            fence_after_sync();
            float ov[NC];                                     // this thread's d columns of the O row
            row_load<QN, NC>(o_addr, ov);
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(O_EMPTY));             // O free for the next item's P V
            if (n >= 0) {
                uint4* dst = reinterpret_cast<uint4*>(p.o + ((size_t)bh * s.N + n) * kDh + hf * 64);
#pragma unroll
                for (int c = 0; c < NC / 8; ++c) {
                    uint4 u;
                    u.x = pack_bf16(ov[8 * c] * inv_l, ov[8 * c + 1] * inv_l);
                    u.y = pack_bf16(ov[8 * c + 2] * inv_l, ov[8 * c + 3] * inv_l);
                    u.z = pack_bf16(ov[8 * c + 4] * inv_l, ov[8 * c + 5] * inv_l);
                    u.w = pack_bf16(ov[8 * c + 6] * inv_l, ov[8 * c + 7] * inv_l);
                    dst[c] = u;
                }
            }
        }
        if (!ok) record_timeout(p, 3);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
}

template <int QN, bool kCube>
cudaError_t launch_rows(const Shape& s, const void* qr, const void* kr, const void* v, const int32_t* kv_idx,
                        void* o_s, float* lse, DeviceStatus* status, cudaStream_t st)
{
    // the maps span the block-ordered rows (the token order itself for contiguous chunks)
    Shape rows = s;
    rows.N = s.Np;
    CUtensorMap mq, mk, mv;
    if (!make_block_map(&mq, qr, rows, QN) || !make_chunk_map(&mk, kr, rows) || !make_block_map(&mv, v, rows))
        return cudaErrorInvalidValue;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    Params p;
    p.s = s;
    p.kv_idx = kv_idx;
    p.o = static_cast<__nv_bfloat16*>(o_s);
    p.lse = lse;
    p.status = status;
    p.items_per_head = s.nQ;
    p.total_items = s.B * s.H * s.nQ;
    p.tiles = (s.n_keep + 1) / 2;
    const size_t smem = Cfg<QN>::kSmemTiles + sizeof(Ctrl<QN>);
    const int grid = p.total_items < nsm ? p.total_items : nsm;
    auto kernel = sparse_attn_rows_kernel<QN, kCube>;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    launch_kernel(kernel, grid, kThreads, smem, st, mq, mk, mv, p);
    return cudaGetLastError();
}

}  // namespace

// 64-token key blocks; query blocks of 64 slots (chunks or cubes; the mask has
// nQ = nB rows) or, with chunks, of 128 tokens (s.qb2 == 1).
cudaError_t launch_sparse_attn_rows(const Shape& s, const void* qr, const void* kr, const void* v,
                                    const int32_t* kv_idx, void* o_s, float* lse, DeviceStatus* status,
                                    cudaStream_t st)
{
    auto launch = s.cube ? launch_rows<64, true> : (s.qb2 ? launch_rows<128, false> : launch_rows<64, false>);
    return launch(s, qr, kr, v, kv_idx, o_s, lse, status, st);
}

}  // namespace rola
