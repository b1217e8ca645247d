// 3D RoPE tables and the rotate + block-pool pass of the block mask.
//
// RoPE (Sec. 3, Eq. shiftinv; truncation Sec. 4.2): pair m acts on coordinates
// (2m, 2m+1); the first d_t/2 pairs turn with the temporal position, the next
// d_x/2 with the row, the rest with the column; within an axis the i-th pair
// turns by pos * theta^(-2i/d_axis).  The table holds (cos, sin) in fp32,
// evaluated in fp64 once per call (frequencies on the host, angles and (cos, sin) on the GPU).
#include <math.h>

#include "common.cuh"

namespace rola {

// theta^(-2i/d_axis) of every pair, in fp64.  Computed on the host: 64 of them
// serve a whole call, and a pow per table entry on the GPU's few fp64 lanes was most of
// the 11 us that the table used to take.
struct Frequencies {
    double f[kPairs];
};

// One CTA per table row; the row's axis owns pairs m0 .. m0 + count - 1, the others keep (1, 0).
__global__ void rope_table_kernel(float2* __restrict__ tab, int T, int Hh, int pt, int px, int off_t, int off_x,
                                  int off_y, const __grid_constant__ Frequencies freq, DeviceStatus* status)
{
    chain_begin();
    const int row = blockIdx.x, m = threadIdx.x;
    if (row == 0) reinterpret_cast<int*>(status)[m] = 0;
    static_assert(sizeof(DeviceStatus) == kPairs * sizeof(int), "one status word a thread");
    const int axis = row < T ? 0 : (row < T + Hh ? 1 : 2);
    const int m0 = axis == 0 ? 0 : (axis == 1 ? pt : pt + px);
    const int count = axis == 0 ? pt : (axis == 1 ? px : kPairs - pt - px);
    const int pos = axis == 0 ? row + off_t : (axis == 1 ? row - T + off_x : row - T - Hh + off_y);
    // thread i takes pair m0 + i (mod 64), so that the fp64 work of a row fills as few warps as it can
    const int pair = (m0 + m) & (kPairs - 1);
    float2 out = make_float2(1.0f, 0.0f);
    if (m < count) {
        double s, c;
        sincos((double)pos * freq.f[pair], &s, &c);
        out = make_float2((float)c, (float)s);
    }
    tab[row * kPairs + pair] = out;
}

cudaError_t launch_rope_table(const rola_config_t& cfg, float2* tab, DeviceStatus* status, cudaStream_t st)
{
    Frequencies freq;
    for (int axis = 0, m = 0; axis < 3; ++axis)
        for (int i = 0; i < cfg.rope_split[axis] / 2; ++i, ++m)
            freq.f[m] = pow(cfg.rope_theta, -2.0 * (double)i / (double)cfg.rope_split[axis]);
    launch_kernel(rope_table_kernel, cfg.T + cfg.Hh + cfg.Ww, kPairs, 0, st, tab, cfg.T, cfg.Hh, cfg.rope_split[0] / 2,
                  cfg.rope_split[1] / 2, cfg.pos_offset[0], cfg.pos_offset[1], cfg.pos_offset[2], freq, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// rotate + pool: one CTA per (64-slot block, head, q | k | v).  Eight warps: warp w
// takes slots 8 w .. 8 w + 7, a lane four coordinates (two pairs), so a token's grid
// position is the same for the whole warp.  Writes the rotated rows in the storage
// dtype (unless the caller only wants the mask) and the fp32 block mean of the
// fp32-rotated (unrounded) values.  The block mean is the pairwise sum of the
// block's 64 slots in slot order (empty slots hold +0), divided once by the token
// count: the evaluation order the block mask is defined with, so that every kernel
// computing it gives the same bits.  A lane adds its warp's eight slots (tree
// levels 1 to 3) in registers; the 8 nodes per coordinate pass through shared memory.
//
// Cube geometry: slots 8 w .. are two runs of four tokens along a grid row.  The
// rotated rows are written in block order (row 64 b + slot of the head's Np rows,
// zeros for slots outside the grid, so that the sparse kernels read finite values
// there); z = 2 copies v into the same order.
//
// HBM wants 512 B read (and 512 B written) per token of q and k at 16 bits.  With
// 16 lanes a token and each lane's position and table rows computed on its own, a
// thread took 550-670 instructions for its 32 values and issue was the bound.
// 720p layer (40 heads, 75600 tokens): means alone 380 us (4.1 TB/s read; they used
// to come with the rows, 771 us for both); 480p cubes of q, k and v 522 -> 348 us.

// Four coordinates of a row.
template <typename T>
struct Vec4;
template <>
struct Vec4<__nv_bfloat16> {
    using Raw = uint2;
    __device__ static void unpack(const Raw& r, float (&x)[4])
    {
        const float2 a = unpack_bf16(r.x), b = unpack_bf16(r.y);
        x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
    }
    __device__ static Raw pack(const float (&x)[4]) { return make_uint2(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3])); }
    __device__ static Raw zero() { return make_uint2(0u, 0u); }
};
template <>
struct Vec4<float> {
    using Raw = float4;
    __device__ static void unpack(const Raw& r, float (&x)[4]) { x[0] = r.x; x[1] = r.y; x[2] = r.z; x[3] = r.w; }
    __device__ static Raw pack(const float (&x)[4]) { return make_float4(x[0], x[1], x[2], x[3]); }
    __device__ static Raw zero() { return make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
};

template <typename T, bool kCube>
__global__ void __launch_bounds__(256) rope_pool_kernel(Shape s, const T* __restrict__ q, const T* __restrict__ k,
                                                        const T* __restrict__ v, const float2* __restrict__ tab,
                                                        T* __restrict__ qr, T* __restrict__ kr, T* __restrict__ vp,
                                                        float* __restrict__ qbar, float* __restrict__ kbar)
{
    chain_begin();
    using Raw = typename Vec4<T>::Raw;
    __shared__ __align__(16) float nodes[8][kDh];            // level-3 nodes of the pairwise sum, slot order
    const int blk = blockIdx.x, bh = blockIdx.y, z = blockIdx.z;
    const T* x = z == 0 ? q : (z == 1 ? k : v);
    T* xr = z == 0 ? qr : (z == 1 ? kr : vp);                // null: the rows are not wanted
    float* xbar = z == 0 ? qbar : (z == 1 ? kbar : nullptr);   // null: the means are not wanted
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp-uniform)
    // first token of each run (chunks: one run of eight, cubes: two of four) and how many tokens it holds
    constexpr int kRuns = kCube ? 2 : 1, kLen = 8 / kRuns;
    int n0[kRuns], cnt[kRuns], t, xx, yy, tokens;
    if constexpr (kCube) {
        const CubeOrigin o = cube_origin(s, blk);
        t = o.t + (warp >> 1);
        xx = o.x + 2 * (warp & 1);
        yy = o.y;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            n0[r] = (t * s.Hh + xx + r) * s.Ww + yy;
            cnt[r] = t < s.T && xx + r < s.Hh ? min(4, s.Ww - yy) : 0;
        }
        tokens = min(4, s.T - o.t) * min(4, s.Hh - o.x) * min(4, s.Ww - o.y);
    } else {
        n0[0] = blk * kBlock + 8 * warp;
        cnt[0] = min(8, max(0, s.N - n0[0]));
        const int hw = s.Hh * s.Ww;
        t = n0[0] / hw;
        const int rem = n0[0] - t * hw;
        xx = rem / s.Ww;
        yy = rem - xx * s.Ww;
        tokens = min(kBlock, s.N - blk * kBlock);
    }
    // all loads first: eight 8- or 16-byte vectors in flight per thread
    Raw raw[8];
    const Raw* src = reinterpret_cast<const Raw*>(x + (size_t)bh * s.N * kDh) + lane;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int r = j / kLen, i = j % kLen;
        raw[j] = i < cnt[r] ? __ldg(src + (size_t)(n0[r] + i) * 32) : Vec4<T>::zero();
    }
    // chunks: Np = N and a slot past the sequence has no row; cubes: every slot has one
    Raw* dst = xr ? reinterpret_cast<Raw*>(xr + ((size_t)bh * s.Np + (size_t)blk * kBlock + 8 * warp) * kDh) + lane : nullptr;
    if (z == 2) {
#pragma unroll
        for (int j = 0; j < 8; ++j) dst[j * 32] = raw[j];
        return;
    }
    // (cos, sin) of this lane's two pairs; from token to token along a grid row only the column's pairs change
    const int m = 2 * lane;
    const int ax0 = m < s.pt ? 0 : (m < s.pt + s.px ? 1 : 2), ax1 = m + 1 < s.pt ? 0 : (m + 1 < s.pt + s.px ? 1 : 2);
    const float2 *p0, *p1;
    float2 c0, c1;
    auto seek = [&]() {
        p0 = tab + (ax0 == 0 ? t : (ax0 == 1 ? s.T + xx : s.T + s.Hh + yy)) * kPairs + m;
        p1 = tab + (ax1 == 0 ? t : (ax1 == 1 ? s.T + xx : s.T + s.Hh + yy)) * kPairs + m + 1;
        c0 = __ldg(p0);
        c1 = __ldg(p1);
    };
    float sum[4];
    float y[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int r = j / kLen, i = j % kLen;
        if (i < cnt[r]) {
            if (i == 0) {
                if (r > 0) ++xx;
                seek();
            } else {
                if (++yy < s.Ww) {
                    if (ax0 == 2) c0 = __ldg(p0 += kPairs);
                    if (ax1 == 2) c1 = __ldg(p1 += kPairs);
                } else {
                    yy = 0;
                    if (++xx == s.Hh) {
                        xx = 0;
                        ++t;
                    }
                    seek();
                }
            }
            float w[4];
            Vec4<T>::unpack(raw[j], w);
            const float2 a = rope_rotate(w[0], w[1], c0), b = rope_rotate(w[2], w[3], c1);
            y[j][0] = a.x; y[j][1] = a.y; y[j][2] = b.x; y[j][3] = b.y;
        } else {
            y[j][0] = y[j][1] = y[j][2] = y[j][3] = 0.0f;    // an empty slot of the pairwise sum
        }
        if constexpr (kCube)
            if (i == kLen - 1 && r == 0 && cnt[0] > 0) yy -= cnt[0] - 1;   // back to the run's first column
        if (dst && (kCube || i < cnt[r])) dst[j * 32] = Vec4<T>::pack(y[j]);
    }
    if (!xbar) return;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        sum[i] = ((y[0][i] + y[1][i]) + (y[2][i] + y[3][i])) + ((y[4][i] + y[5][i]) + (y[6][i] + y[7][i]));
    *reinterpret_cast<float4*>(&nodes[warp][4 * lane]) = make_float4(sum[0], sum[1], sum[2], sum[3]);
    __syncthreads();
    if (threadIdx.x < kDh) {
        const int c = threadIdx.x;
        const float all = ((nodes[0][c] + nodes[1][c]) + (nodes[2][c] + nodes[3][c])) +
                          ((nodes[4][c] + nodes[5][c]) + (nodes[6][c] + nodes[7][c]));
        // with 128-token query blocks the query side keeps the sum (the 128-token tree's left or right half)
        xbar[((size_t)bh * s.nB + blk) * kDh + c] = z == 0 && s.qb2 ? all : all / (float)tokens;
    }
}

template <typename T>
cudaError_t launch_rope_pool_t(const Shape& s, const void* q, const void* k, const void* v, const float2* tab,
                               void* qr, void* kr, void* vp, float* qbar, float* kbar, cudaStream_t st)
{
    const dim3 grid(s.nB, s.B * s.H, s.cube && v ? 3 : 2);
    auto kernel = s.cube ? rope_pool_kernel<T, true> : rope_pool_kernel<T, false>;
    launch_kernel(kernel, grid, 256, 0, st, s, (const T*)q, (const T*)k, (const T*)v, tab, (T*)qr, (T*)kr, (T*)vp, qbar, kbar);
    return cudaGetLastError();
}

cudaError_t launch_rope_pool(const rola_config_t& cfg, const Shape& s, const void* q, const void* k, const void* v,
                             const float2* tab, void* qr, void* kr, void* vp, float* qbar, float* kbar,
                             cudaStream_t st)
{
    if (s.cube && v && !vp) return cudaErrorInvalidValue;
    return cfg.dtype == ROLA_BF16
               ? launch_rope_pool_t<__nv_bfloat16>(s, q, k, v, tab, qr, kr, vp, qbar, kbar, st)
               : launch_rope_pool_t<float>(s, q, k, v, tab, qr, kr, vp, qbar, kbar, st);
}

}  // namespace rola
