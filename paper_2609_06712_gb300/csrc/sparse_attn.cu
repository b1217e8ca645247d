// Block-sparse softmax attention over the kept key blocks (kernel 2).
//
//   O^s_p = sum_{q in kept(i)} softmax_q(q^r_p . k^r_q / sqrt(d_h)) v_q,   p in block i
//
// (Sec. 3 softmax form restricted to the kept blocks, Alg. 1 sparse branch).
// q^r, k^r are the rotated copies written by the rotate + pool pass.  The
// bf16 path is the tcgen05 kernel of sparse_attn_rows.cu; this file holds the
// fp32 validation-mode kernel (online softmax in fp32) and the dispatch.
#include "common.cuh"

namespace rola {

// ===========================================================================
// fp32 validation mode: SIMT, one CTA per (query block, head), 256 threads as 16
// row groups x 16.  Thread (ty, tx) owns rows ty + 16 i (i < 4) throughout: the
// scores of keys tx + 16 c (c < 4) and the outputs of d = 4 tx .. and 64 + 4 tx ..,
// so the row statistics stay in registers (the 16 threads of a row are half a warp).
// K and V tiles are double-buffered with cp.async; P goes through shared memory.
// Products run as packed fma.rn.f32x2, each element an IEEE fma: a score is the sum
// of an even-d and an odd-d chain.  q^r, k^r and v are read in block order (Np rows
// per head); O^s rows go to their tokens.
//
// Bound by the fp32 FMA rate at 3 shared-memory wavefronts a warp per 16 (scores)
// and 32 (P V) FMAs of a thread; with one score at a time from scalar shared loads
// (two per FMA) the kernel took 276 us for 4 heads, 2340 tokens, 7 of 37 blocks kept,
// in a layer of 427 us; it takes 54 now, the layer 131.

constexpr int kF32Threads = 256;
constexpr int kF32Row = kDh + 4;          // padded row of Q and K: 16 rows' 16-byte chunks fall on all banks
constexpr int kF32P = kBlock + 4;
struct F32Smem {
    float q[kBlock * kF32Row];
    float k[2][kBlock * kF32Row];
    float v[2][kBlock * kDh];
    float p[kBlock * kF32P];
};

// acc (even, odd chain) += x.xy * y.xy, then x.zw * y.zw
__device__ __forceinline__ void dot4(float2& acc, const float4& x, const float4& y)
{
    asm("{\n.reg .b64 a, b, c;\nmov.b64 c, {%0, %1};\n"
        "mov.b64 a, {%2, %3};\nmov.b64 b, {%6, %7};\nfma.rn.f32x2 c, a, b, c;\n"
        "mov.b64 a, {%4, %5};\nmov.b64 b, {%8, %9};\nfma.rn.f32x2 c, a, b, c;\n"
        "mov.b64 {%0, %1}, c;\n}\n"
        : "+f"(acc.x), "+f"(acc.y)
        : "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w), "f"(y.x), "f"(y.y), "f"(y.z), "f"(y.w));
}
// (a, b) += p * (x, y)
__device__ __forceinline__ void axpy2(float& a, float& b, float p, float x, float y)
{
    asm("{\n.reg .b64 c, s, v;\nmov.b64 c, {%0, %1};\nmov.b64 s, {%2, %2};\nmov.b64 v, {%3, %4};\n"
        "fma.rn.f32x2 c, s, v, c;\nmov.b64 {%0, %1}, c;\n}\n"
        : "+f"(a), "+f"(b)
        : "f"(p), "f"(x), "f"(y));
}

template <bool kCube>
__global__ void __launch_bounds__(kF32Threads, 1) sparse_attn_f32_kernel(Shape s, const float* __restrict__ qr,
                                                                         const float* __restrict__ kr,
                                                                         const float* __restrict__ v,
                                                                         const int32_t* __restrict__ kv_idx,
                                                                         float* __restrict__ o, float* __restrict__ lse)
{
    chain_begin();
    extern __shared__ __align__(16) uint8_t fsm[];
    F32Smem& sm = *reinterpret_cast<F32Smem*>(fsm);
    const int qb = blockIdx.x, bh = blockIdx.y, tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const size_t head = (size_t)bh * s.Np * kDh;
    const int32_t* kept = kv_idx + ((size_t)bh * s.nQ + (qb >> s.qb2)) * s.n_keep;   // the block's mask row
    // rows of block b (zeros past the end) into a tile with `stride` floats a row
    auto fetch = [&](float* dst, int stride, const float* src, int b) {
        for (int e = tid; e < kBlock * (kDh / 4); e += kF32Threads) {
            const int r = e >> 5, c = e & 31;
            const long long n = (long long)b * kBlock + r;
            const bool in = n >= 0 && n < s.Np;
            cp_async16(smem_u32(dst + r * stride + 4 * c), src + head + (in ? n : 0) * kDh + 4 * c, in ? 16 : 0);
        }
    };
    fetch(sm.q, kF32Row, qr, qb);
    fetch(sm.k[0], kF32Row, kr, kept[0]);
    fetch(sm.v[0], kDh, v, kept[0]);
    cp_async_commit();
    float acc[4][8];
    float m_run[4], l_run[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m_run[i] = -INFINITY;
        l_run[i] = 0.0f;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[i][e] = 0.0f;
    }
    const float scale = 0.08838834764831845f;   // 1/sqrt(128)
    for (int it = 0; it < s.n_keep; ++it) {
        const int j = kept[it], buf = it & 1;
        if (it + 1 < s.n_keep) {                 // (every thread has passed the barrier after the buffer's last use)
            fetch(sm.k[buf ^ 1], kF32Row, kr, kept[it + 1]);
            fetch(sm.v[buf ^ 1], kDh, v, kept[it + 1]);
        }
        cp_async_commit();
        cp_async_wait<1>();
        __syncthreads();
        // ---- scores of rows ty + 16 i and keys tx + 16 c
        float2 sc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) sc[i][c] = make_float2(0.0f, 0.0f);
        const float* kt = sm.k[buf];
#pragma unroll 4
        for (int d = 0; d < kDh; d += 4) {
            float4 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(sm.q + (ty + 16 * i) * kF32Row + d);
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = *reinterpret_cast<const float4*>(kt + (tx + 16 * c) * kF32Row + d);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) dot4(sc[i][c], a[i], b[c]);
        }
        // ---- online softmax
        const uint32_t m0 = block_mask32<kCube>(s, j, 0), m1 = block_mask32<kCube>(s, j, 1);
        const bool in[4] = {((m0 >> tx) & 1u) != 0, ((m0 >> (tx + 16)) & 1u) != 0, ((m1 >> tx) & 1u) != 0,
                            ((m1 >> (tx + 16)) & 1u) != 0};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float x[4], mx = m_run[i];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                x[c] = in[c] ? (sc[i][c].x + sc[i][c].y) * scale : -INFINITY;
                mx = fmaxf(mx, x[c]);
            }
#pragma unroll
            for (int w = 1; w < 16; w *= 2) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
            float sum = 0.0f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                x[c] = expf(x[c] - mx);
                sm.p[(ty + 16 * i) * kF32P + tx + 16 * c] = x[c];
                sum += x[c];
            }
#pragma unroll
            for (int w = 1; w < 16; w *= 2) sum += __shfl_xor_sync(0xffffffffu, sum, w);
            const float alpha = expf(m_run[i] - mx);
            l_run[i] = l_run[i] * alpha + sum;
            m_run[i] = mx;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[i][e] *= alpha;
        }
        __syncwarp();                            // a row's P is written and read by one half warp
        // ---- O += P V
        const float* vt = sm.v[buf];
#pragma unroll 2
        for (int c = 0; c < kBlock; c += 4) {
            float4 p4[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p4[i] = *reinterpret_cast<const float4*>(sm.p + (ty + 16 * i) * kF32P + c);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 v0 = *reinterpret_cast<const float4*>(vt + (c + u) * kDh + 4 * tx);
                const float4 v1 = *reinterpret_cast<const float4*>(vt + (c + u) * kDh + 64 + 4 * tx);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float p = u == 0 ? p4[i].x : (u == 1 ? p4[i].y : (u == 2 ? p4[i].z : p4[i].w));
                    axpy2(acc[i][0], acc[i][1], p, v0.x, v0.y);
                    axpy2(acc[i][2], acc[i][3], p, v0.z, v0.w);
                    axpy2(acc[i][4], acc[i][5], p, v1.x, v1.y);
                    axpy2(acc[i][6], acc[i][7], p, v1.z, v1.w);
                }
            }
        }
        __syncthreads();                         // the buffer's readers are done
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = ty + 16 * i, n = slot_token_g<kCube>(s, qb, row);
        if (n < 0) continue;
        const float inv = 1.0f / l_run[i];
        if (lse && tx == 0) lse[(size_t)bh * s.N + n] = m_run[i] + logf(l_run[i]);
        float* on = o + ((size_t)bh * s.N + n) * kDh;
        *reinterpret_cast<float4*>(on + 4 * tx) =
            make_float4(acc[i][0] * inv, acc[i][1] * inv, acc[i][2] * inv, acc[i][3] * inv);
        *reinterpret_cast<float4*>(on + 64 + 4 * tx) =
            make_float4(acc[i][4] * inv, acc[i][5] * inv, acc[i][6] * inv, acc[i][7] * inv);
    }
}

// bf16 (sparse_attn_rows.cu)
cudaError_t launch_sparse_attn_rows(const Shape& s, const void* qr, const void* kr, const void* v,
                                    const int32_t* kv_idx, void* o_s, float* lse, DeviceStatus* status,
                                    cudaStream_t st);

cudaError_t launch_sparse_attn(rola_dtype_t dt, const Shape& s, const void* qr, const void* kr, const void* v,
                               const int32_t* kv_idx, void* o_s, float* lse, DeviceStatus* status, cudaStream_t st)
{
    if (dt == ROLA_BF16) return launch_sparse_attn_rows(s, qr, kr, v, kv_idx, o_s, lse, status, st);
    auto kernel = s.cube ? sparse_attn_f32_kernel<true> : sparse_attn_f32_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(F32Smem));
    if (e != cudaSuccess) return e;
    launch_kernel(kernel, dim3(s.nB, s.B * s.H), kF32Threads, sizeof(F32Smem), st, s, (const float*)qr, (const float*)kr,
                                                                       (const float*)v, kv_idx, (float*)o_s, lse);
    return cudaGetLastError();
}

}  // namespace rola
