// fp32 rows as three bf16 parts for the tensor cores: x = h + m + l with h = bf16(x), m = bf16(x - h), l = x - h - m, 8 bits of
// the 24-bit significand each, so the sum is exact for every finite x, but for bits below 2^-133, the least that bf16 holds.  Keys of every
// layout land dense, part after part: row tok_off[u] + i of part p at k_split + (p * sumT + tok_off[u] + i) * d; the queries
// the same way.  The Euclidean norm of every key row, which the assignment needs, comes along.
//
// Bound by HBM: 10 bytes per element (16 units of 8,448 rows, d = 128: 173 MB).  One warp takes kRows rows side by side, so that
// their loads are in flight together.
#include "cask_internal.cuh"

namespace cask {

namespace {

constexpr int kRows = 4, kWarps = 8;

__global__ void __launch_bounds__(kWarps * 32) split_rows_kernel(const UnitDesc* __restrict__ desc, Shape sh, const float* __restrict__ K,
                                                                 const float* __restrict__ Q, int64_t sum_T, int key_blocks,
                                                                 __nv_bfloat16* __restrict__ k_split, __nv_bfloat16* __restrict__ q_split,
                                                                 float* __restrict__ k_norm) {
    pdl_wait();
    const int u = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const UnitDesc& ud = desc[u];
    const bool keys = (int)blockIdx.x < key_blocks;
    const int n = keys ? ud.T : sh.rows;
    const int r0 = (((int)blockIdx.x - (keys ? 0 : key_blocks)) * kWarps + w) * kRows;
    if (r0 >= n) return;
    const int64_t part = keys ? sum_T : (int64_t)sh.n_units * sh.rows;           // rows per part
    const int64_t row0 = keys ? ud.tok_off : (int64_t)u * sh.rows;
    __nv_bfloat16* dst = keys ? k_split : q_split;
    const bool on = 4 * lane < sh.d;                                             // d <= 128: four channels per lane
    const float* src[kRows];
    if (!keys || sh.page_size == 0) {
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            const int r = min(r0 + q, n - 1);
            src[q] = keys ? K + ud.k_off + (int64_t)r * sh.row_stride : Q + ud.q_off + (int64_t)r * sh.d;
        }
    } else {
#pragma unroll
        for (int q = 0; q < kRows; ++q) src[q] = K + row_elem_off(sh, ud, ud.k_off, min(r0 + q, n - 1));
    }
    float4 x[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) x[q] = on ? reinterpret_cast<const float4*>(src[q])[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
        const float v[4] = {x[q].x, x[q].y, x[q].z, x[q].w};
        float n2 = 0.f;
        struct alignas(8) Quad { __nv_bfloat16 e[4]; } p[3];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            split3(v[c], p[0].e[c], p[1].e[c], p[2].e[c]);
            n2 = fmaf(v[c], v[c], n2);
        }
        if (r0 + q < n && on) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
                reinterpret_cast<Quad*>(dst + (k * part + row0 + r0 + q) * sh.d)[lane] = p[k];
        }
        if (keys) {
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, off);
            if (lane == 0 && r0 + q < n) k_norm[row0 + r0 + q] = sqrtf(n2);
        }
    }
}

}  // namespace

SplitSizes split_sizes(int dtype, int d, int64_t sum_T, int64_t q_rows) {
    if (dtype != CASK_DTYPE_FP32 || d > 128) return SplitSizes{0, 0, 0};
    return SplitSizes{(size_t)(3 * sum_T * d * 2), (size_t)(3 * q_rows * d * 2), (size_t)(sum_T * 4)};
}

cudaError_t launch_split_rows(const Launch& L, Workspace& ws, bool queries) {
    const int per = kRows * kWarps;
    const int key_blocks = ws.split_ready ? 0 : (L.max_T + per - 1) / per;
    const int q_blocks = queries ? (L.sh.rows + per - 1) / per : 0;
    if (key_blocks + q_blocks == 0) return cudaSuccess;
    Timed t(L, KID_SPLIT);
    ws.split_ready = true;
    return launch_dependent(L.stream, split_rows_kernel, dim3(key_blocks + q_blocks, L.sh.n_units), kWarps * 32, 0, L.desc, L.sh,
                            (const float*)L.k, (const float*)L.q, L.sum_T, key_blocks, (__nv_bfloat16*)ws.k_split,
                            (__nv_bfloat16*)ws.q_split, ws.k_norm);
}

}  // namespace cask
