// Low-rank readout and gated fusion of the bf16 path (kernel 4):
//   q~_p   = R_r(p) SiLU(P_q q^n_p)                     Eq. (qklr) (or the placement cfg selects)
//   O^lr_p = y_p / sqrt(mean_i y_{p,i}^2 + eps_lr),     y_p = q~_p^T C      Eq. (ctx)
//   r_p    = sqrt(mean_i (O^s_{p,i})^2 + eps_fuse)
//   O_p    = O^s_p + g_p r_p O^lr_p                     Eq. (gate), (O^s/r_p + g O^lr) r_p
//
// Work unit = (head, 16-token tile).  One persistent CTA per SM takes a contiguous
// range of tiles; P_q and C (bf16) are loaded once per head it meets, and within a
// head every warp works on tiles of its own with no barrier between warps:
//   U = Q P_q^T (mma.sync), q~ = R_r SiLU(U) in registers
//   (an accumulator pair is the A fragment of the next product), y += q~ C for all
//   128 d, the row sums of y^2 and (O^s)^2 over the four lanes of a row, and O
//   written over O^s in shared memory, from where a TMA store takes it (which also
//   clips the rows past N).
// A warp owns a q buffer (refilled as soon as its fragments are in registers) and
// two O^s buffers (one for r > 64), filled by its own TMA loads, so the warps of an
// SM are at different points of the chain and their loads, products and stores
// overlap.  Bound by HBM: 768 B per (head, token).  720p layer (40 heads, 75600
// tokens): r = 32 496 -> 350 us (6.6 TB/s), r = 64 1048 -> 552 us; the form before
// (64-token units over 8 warps with three CTA barriers each, one or two CTAs an SM)
// waited on its own chain most of the time.  From r = 64 the features' IEEE divides
// weigh (an approximate one, which loses features below -87: 464 us).
#include <cudaTypedefs.h>

#include "common.cuh"
#include "tcgen05.cuh"
#include "tensor_map.cuh"

namespace rola {
namespace {

using namespace tc;

constexpr int kTile = 16;                            // tokens of a tile
constexpr uint32_t kBox = kTile * 128 * 2;           // [chunk][16 rows][64]

template <int R>
struct Layout {
    static constexpr int warps = R <= 64 ? 16 : 12;  // (registers: 128 or 168 a thread)
    static constexpr int OB = R <= 64 ? 2 : 1;       // O^s buffers of a warp
    static constexpr uint32_t warp_bytes = (1 + OB) * kBox;     // q | O^s ...
    static constexpr uint32_t P = warps * warp_bytes;
    static constexpr uint32_t C = P + R * 256;
    static constexpr uint32_t bars = C + R * 256;    // full barriers of every warp: q, O^s ...
    static constexpr uint32_t abort = bars + warps * (1 + OB) * 8;
    static constexpr uint32_t total = abort + 16;
};

// Byte offset of 16-byte chunk c (0..15) of row r in a 16-row box (128-byte swizzle).
__device__ __forceinline__ uint32_t wsw(int r, int c)
{
    return (c >> 3) * (kTile * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4);
}

struct Params {
    Shape s;
    const __nv_bfloat16* Pq;
    const __nv_bfloat16* Cbf;
    const float* gate;
    const float2* tab;
    DeviceStatus* status;
    int tiles;                // 16-token tiles of a head
    int splits;               // > 0: CTAs per head, none of which meets two heads
};

template <int R, typename Feature>
__global__ void __launch_bounds__(32 * Layout<R>::warps, 1) readout_kernel(const __grid_constant__ CUtensorMap map_q,
                                                                          const __grid_constant__ CUtensorMap map_os,
                                                                          const __grid_constant__ CUtensorMap map_o,
                                                                          const Params p)
{
    using L = Layout<R>;
    constexpr int kWarps = L::warps, kThreads = 32 * kWarps, OB = L::OB;
    extern __shared__ __align__(1024) uint8_t smem[];
    if (smem_u32(smem) & 1023u) {
        if (threadIdx.x == 0) atomicCAS(&p.status->code, 0, (int)ROLA_ERR_UNSUPPORTED);
        return;
    }
    const Shape& s = p.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t4 = lane & 3, mi = lane >> 3;
    const uint32_t sbase = smem_u32(smem), sP = sbase + L::P, sC = sbase + L::C;
    const uint32_t qb = sbase + warp * L::warp_bytes;
    const uint32_t q_full = sbase + L::bars + warp * (1 + OB) * 8, o_full = q_full + 8;
    volatile int* abort = reinterpret_cast<volatile int*>(smem + L::abort);
    const long long total = (long long)s.B * s.H * p.tiles;
    long long u0 = (long long)blockIdx.x * total / gridDim.x, u1 = (long long)(blockIdx.x + 1) * total / gridDim.x;
    if (p.splits > 0) {
        const int bh = blockIdx.x / p.splits, i = blockIdx.x - bh * p.splits;
        u0 = (long long)bh * p.tiles + (long long)i * p.tiles / p.splits;
        u1 = (long long)bh * p.tiles + (long long)(i + 1) * p.tiles / p.splits;
    }
    const int hw = s.Hh * s.Ww;
    const Feature feature(s);
    const float2* tab = p.tab + t4;

    if (tid == 0) {
        *abort = 0;
        for (int i = 0; i < kWarps * (1 + OB); ++i) mbar_init(sbase + L::bars + 8 * i, 1);
        fence_mbar_init();
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_os);
        tma_prefetch_desc(&map_o);
    }
    chain_begin();
    bool ok = true;
    int i = 0;                                       // tiles of this warp so far (buffer and phase)
    int q_issued = 0, o_issued = 0;                  // loads of this warp so far
    for (long long u = u0; u < u1;) {
        const int bh = (int)(u / p.tiles), first = (int)(u - (long long)bh * p.tiles);
        const int end = (int)min((long long)p.tiles, first + (u1 - u));
        u += end - first;
        // (lane 0 issues all of a warp's copies, so that its bulk-group waits order a refill after the store)
        auto load_q = [&](int x) {
            if (lane == 0) {
                mbar_expect_tx(q_full, kBox);
                tma_load_4d(qb, &map_q, q_full, 0, x * kTile, 0, bh);
            }
            ++q_issued;
        };
        auto load_o = [&](int x, int buf) {
            if (lane == 0) {
                bulk_wait_read_all();                // the store that last read the buffer
                mbar_expect_tx(o_full + 8 * buf, kBox);
                tma_load_4d(qb + kBox + buf * kBox, &map_os, o_full + 8 * buf, 0, x * kTile, 0, bh);
            }
            ++o_issued;
        };
        __syncthreads();                             // the barriers are initialised; every reader of the last head is done
        if (ok && first + warp < end) {
            load_q(first + warp);
            load_o(first + warp, i % OB);
        }
        {
            const uint4* srcP = reinterpret_cast<const uint4*>(p.Pq + (size_t)(bh % s.H) * s.r * kDh);
            const uint4* srcC = reinterpret_cast<const uint4*>(p.Cbf + (size_t)bh * R * kDh);   // rp rows
            for (int e = tid; e < R * 16; e += kThreads) {
                const uint4 a = (e >> 4) < s.r ? __ldg(srcP + e) : make_uint4(0, 0, 0, 0), c = __ldg(srcC + e);
                const uint32_t off = sw128(e >> 4, e & 15);
                asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(sP + off), "r"(a.x), "r"(a.y), "r"(a.z),
                             "r"(a.w)
                             : "memory");
                asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(sC + off), "r"(c.x), "r"(c.y), "r"(c.z),
                             "r"(c.w)
                             : "memory");
            }
        }
        __syncthreads();
        // a warp whose wait gave up stays for the barriers of the heads to come and works no further tile
        for (int x = first + warp; ok && x < end; x += kWarps, ++i) {
            const int buf = i % OB;
            const bool more = x + kWarps < end;
            if (OB == 2 && more) load_o(x + kWarps, buf ^ 1);
            // grid positions and gates of this thread's two tokens
            const int n_lo = x * kTile + g;
            int tt[2], xx[2], yy[2];
            float gp[2];
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const int n = min(n_lo + 8 * hr, s.N - 1);
                tt[hr] = n / hw;
                const int rem = n - tt[hr] * hw;
                xx[hr] = rem / s.Ww;
                yy[hr] = rem - xx[hr] * s.Ww;
                gp[hr] = p.gate ? __ldg(p.gate + (size_t)(bh / s.H) * s.N + n) : s.default_gate;
            }
            ok = __all_sync(0xffffffffu, mbar_wait(q_full, i & 1, abort, s.wait_limit_ns));
            if (!ok) break;
            // ---- U = Q P_q^T, all r columns
            float u[R / 8][4];
#pragma unroll
            for (int j = 0; j < R / 8; ++j) u[j][0] = u[j][1] = u[j][2] = u[j][3] = 0.0f;
#pragma unroll
            for (int kc = 0; kc < 8; ++kc) {
                uint32_t a0, a1, a2, a3;
                ldsm_x4(qb + wsw((lane & 7) + (mi & 1) * 8, kc * 2 + (mi >> 1)), a0, a1, a2, a3);
#pragma unroll
                for (int j = 0; j < R / 16; ++j) {
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4(sP + sw128(j * 16 + (mi >> 1) * 8 + (lane & 7), kc * 2 + (mi & 1)), b0, b1, b2, b3);
                    mma_bf16(u[2 * j], a0, a1, a2, a3, b0, b1);
                    mma_bf16(u[2 * j + 1], a0, a1, a2, a3, b2, b3);
                }
            }
            __syncwarp();
            if (more) load_q(x + kWarps);
            // ---- q~: an accumulator's two rows and column pair are the A fragment of the next product
            // (rows of tokens past N are never stored)
            uint32_t af[R / 8][2];
            auto features = [&](auto row) {              // row(pair, token): the pair's table row
#pragma unroll
                for (int j = 0; j < R / 8; ++j)
#pragma unroll
                    for (int hr = 0; hr < 2; ++hr) {
                        const float2 f = feature(u[j][2 * hr], u[j][2 * hr + 1],
                                                 __ldg(tab + row(j * 4 + t4, hr) * kPairs + j * 4));
                        af[j][hr] = pack_bf16(f.x, f.y);
                    }
            };
            // (with every pair on the temporal axis, r <= 44 by default, a token has one table row)
            if (R / 2 <= s.pt) features([&](int, int hr) { return tt[hr]; });
            else
                features([&](int m, int hr) {
                    return m < s.pt ? tt[hr] : (m < s.pt + s.px ? s.T + xx[hr] : s.T + s.Hh + yy[hr]);
                });
            // ---- y = q~ C
            float y[16][4];
#pragma unroll
            for (int d = 0; d < 16; ++d) y[d][0] = y[d][1] = y[d][2] = y[d][3] = 0.0f;
#pragma unroll
            for (int j = 0; j < R / 16; ++j)
#pragma unroll
                for (int dp = 0; dp < 8; ++dp) {
                    uint32_t b0, b1, b2, b3;
                    ldsm_x4_t(sC + sw128(j * 16 + (mi & 1) * 8 + (lane & 7), dp * 2 + (mi >> 1)), b0, b1, b2, b3);
                    mma_bf16(y[2 * dp], af[2 * j][0], af[2 * j][1], af[2 * j + 1][0], af[2 * j + 1][1], b0, b1);
                    mma_bf16(y[2 * dp + 1], af[2 * j][0], af[2 * j][1], af[2 * j + 1][0], af[2 * j + 1][1], b2, b3);
                }
            // ---- row sums of y^2 and (O^s)^2, then O = O^s + g r_p O^lr over O^s
            ok = __all_sync(0xffffffffu, mbar_wait(o_full + 8 * buf, (i / OB) & 1, abort, s.wait_limit_ns));
            if (!ok) break;
            const uint32_t ob = qb + kBox + buf * kBox;
            // O^s in the accumulators' layout: the column pairs of two n-tiles, rows g and g + 8
            // (read twice: y leaves no registers to keep it)
            uint32_t w[2][2];
            const uint32_t oaddr = (lane & 7) + (mi & 1) * 8;            // row this lane addresses
            float ssy[2] = {0.0f, 0.0f}, sso[2] = {0.0f, 0.0f};
#pragma unroll
            for (int d = 0; d < 16; d += 2) {
                ldsm_x4(ob + wsw(oaddr, d + (mi >> 1)), w[0][0], w[0][1], w[1][0], w[1][1]);
#pragma unroll
                for (int e = d; e < d + 2; ++e)
#pragma unroll
                    for (int hr = 0; hr < 2; ++hr) {
                        const float2 f = unpack_bf16(w[e - d][hr]);
                        ssy[hr] += y[e][2 * hr] * y[e][2 * hr] + y[e][2 * hr + 1] * y[e][2 * hr + 1];
                        sso[hr] += f.x * f.x + f.y * f.y;
                    }
            }
            float coef[2];
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                ssy[hr] += __shfl_xor_sync(0xffffffffu, ssy[hr], 1);
                ssy[hr] += __shfl_xor_sync(0xffffffffu, ssy[hr], 2);
                sso[hr] += __shfl_xor_sync(0xffffffffu, sso[hr], 1);
                sso[hr] += __shfl_xor_sync(0xffffffffu, sso[hr], 2);
                coef[hr] = gp[hr] * sqrtf(sso[hr] * (1.0f / kDh) + s.eps_fuse) *
                           rsqrtf(ssy[hr] * (1.0f / kDh) + s.eps_lr);
            }
#pragma unroll
            for (int d = 0; d < 16; d += 2) {
                ldsm_x4(ob + wsw(oaddr, d + (mi >> 1)), w[0][0], w[0][1], w[1][0], w[1][1]);
#pragma unroll
                for (int e = d; e < d + 2; ++e)
#pragma unroll
                    for (int hr = 0; hr < 2; ++hr) {
                        const float2 f = unpack_bf16(w[e - d][hr]);
                        w[e - d][hr] = pack_bf16(f.x + coef[hr] * y[e][2 * hr], f.y + coef[hr] * y[e][2 * hr + 1]);
                    }
                stsm_x4(ob + wsw(oaddr, d + (mi >> 1)), w[0][0], w[0][1], w[1][0], w[1][1]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_store_4d(&map_o, ob, 0, x * kTile, 0, bh);
                bulk_commit();
            }
            if (OB == 1 && more) load_o(x + kWarps, 0);
        }
    }
    if (lane == 0) {
        if (!ok) {
            if (atomicCAS(&p.status->code, 0, (int)ROLA_ERR_TIMEOUT) == 0) p.status->where = 8;
            // loads issued and not yet waited for must land before the CTA exits
            int never = 0;
            if (q_issued > 0) mbar_wait(q_full, (q_issued - 1) & 1, &never, s.wait_limit_ns);
            for (int j = o_issued > OB ? o_issued - OB : 0; j < o_issued; ++j)
                mbar_wait(o_full + 8 * (j % OB), (j / OB) & 1, &never, s.wait_limit_ns);
        }
        bulk_wait_all();
    }
}

template <int R, typename Feature>
cudaError_t launch_ra(const CUtensorMap& mq, const CUtensorMap& mos, const CUtensorMap& mo, const Params& p, int ctas,
                      cudaStream_t st)
{
    using L = Layout<R>;
    static_assert(L::total <= 232448, "fits the shared memory of one SM");
    cudaError_t e =
        cudaFuncSetAttribute(readout_kernel<R, Feature>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::total);
    if (e != cudaSuccess) return e;
    launch_kernel(readout_kernel<R, Feature>, ctas, 32 * L::warps, L::total, st, mq, mos, mo, p);
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_r(const CUtensorMap& mq, const CUtensorMap& mos, const CUtensorMap& mo, const Params& p, int ctas,
                     cudaStream_t st)
{
    return default_feature(p.s) ? launch_ra<R, SiluOutside<SiluIeee>>(mq, mos, mo, p, ctas, st)
                                : launch_ra<R, AnyFeature<SiluIeee>>(mq, mos, mo, p, ctas, st);
}

}  // namespace

cudaError_t launch_readout(const Shape& s, const void* q, const void* P_q, const __nv_bfloat16* Cbf,
                           const float* gate, const void* o_s, void* o, const float2* tab, DeviceStatus* status,
                           cudaStream_t st)
{
    const int tiles = (s.N + kTile - 1) / kTile;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long total = (long long)s.B * s.H * tiles;
    // Small layers: a CTA that meets two heads loads two sets of weights one after the other, so where
    // whole CTAs per head leave every warp at most one tile, they are dealt out that way.
    const int heads = s.B * s.H, warps = s.rp <= 64 ? 16 : 12;                  // Layout<R>::warps
    const int splits = heads <= nsm ? (nsm / heads < tiles ? nsm / heads : tiles) : 0;
    const bool whole = splits > 0 && (tiles + splits - 1) / splits <= warps;
    const int ctas = whole ? heads * splits : (total < nsm ? (int)total : nsm);
    CUtensorMap mq, mos, mo;
    if (!make_block_map(&mq, q, s, kTile) || !make_block_map(&mos, o_s, s, kTile) || !make_block_map(&mo, o, s, kTile))
        return cudaErrorInvalidValue;
    Params p;
    p.s = s;
    p.Pq = static_cast<const __nv_bfloat16*>(P_q);
    p.Cbf = Cbf;
    p.gate = gate;
    p.tab = tab;
    p.status = status;
    p.tiles = tiles;
    p.splits = whole ? splits : 0;
    switch (s.rp) {
        case 16: return launch_r<16>(mq, mos, mo, p, ctas, st);
        case 32: return launch_r<32>(mq, mos, mo, p, ctas, st);
        case 48: return launch_r<48>(mq, mos, mo, p, ctas, st);
        case 64: return launch_r<64>(mq, mos, mo, p, ctas, st);
        case 80: return launch_r<80>(mq, mos, mo, p, ctas, st);
        case 96: return launch_r<96>(mq, mos, mo, p, ctas, st);
        case 112: return launch_r<112>(mq, mos, mo, p, ctas, st);
        case 128: return launch_r<128>(mq, mos, mo, p, ctas, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rola
