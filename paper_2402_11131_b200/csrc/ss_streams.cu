// Stream initialisation (Eq. 3 with the identity transformation) and the value-rotation stream variant
// (App. B, Eq. 7): element-wise, HBM-bound, 16 bytes per thread and step.  Compiled without fast-math: each
// product, difference and sum is one IEEE fp32 operation, so the results are defined bit by bit.
#include <cuda_bf16.h>
#include <math.h>

#include "ss_common.cuh"

namespace ss {

struct RotTable {
    float cs[SS_MAX_GAMMA], sn[SS_MAX_GAMMA];
};

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Both kernels: a thread owns 8 columns (16 bytes) of the width and walks down the rows, kRowBatch of them at a time, so
// that no index is divided and a thread has kRowBatch loads and gamma * kRowBatch stores in flight.  Bound by HBM, four
// fifths of it writes: both together take 15.7 us for 1024 rows of 4096 with four streams (84 MB; 17.0 us without the prefetch
// before the wait, behind a kernel that releases its successor early and with inputs in HBM; 21.4 us with one thread per output vector and its index
// divided into row, stream and column).
constexpr int kRowBatch = 2;

// A thread's first rows on their way to L2 (one thread asks for a line of 128 bytes): no data reaches the SM, so it may be asked
// for before the wait for the previous kernel, whoever writes them.  (Without / with it behind a kernel that does not release
// early 16.9 / 16.2 us; with inputs in L2 13.9 / 14.1.)
__device__ __forceinline__ void prefetch_rows(const uint4* in, long long first, int by, long long rows, int vec, int c) {
    if (c >= vec || (c & 7) != 0) return;
    #pragma unroll
    for (int i = 0; i < kRowBatch; ++i)
        if (first + i * by < rows) prefetch_l2(in + (first + i * by) * vec + c);
}

__device__ __forceinline__ uint4 add8(const uint4& a, const uint4& b) {
    uint4 r;
    r.x = pack2(__fadd_rn(bf16_lo(a.x), bf16_lo(b.x)), __fadd_rn(bf16_hi(a.x), bf16_hi(b.x)));
    r.y = pack2(__fadd_rn(bf16_lo(a.y), bf16_lo(b.y)), __fadd_rn(bf16_hi(a.y), bf16_hi(b.y)));
    r.z = pack2(__fadd_rn(bf16_lo(a.z), bf16_lo(b.z)), __fadd_rn(bf16_hi(a.z), bf16_hi(b.z)));
    r.w = pack2(__fadd_rn(bf16_lo(a.w), bf16_lo(b.w)), __fadd_rn(bf16_hi(a.w), bf16_hi(b.w)));
    return r;
}

// out[t][j][c] = m[t][c] + p[j][c]; the embeddings of the thread's columns stay in registers
template <bool kNarrow>
__global__ void __launch_bounds__(kNarrow ? 256 : 128)
stream_insert_kernel(const uint4* __restrict__ m, const uint4* __restrict__ p, uint4* __restrict__ out, long long rows, int gamma, int vec) {
    const int c = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x), by = kNarrow ? static_cast<int>(blockDim.y) : 1;
    const long long first = static_cast<long long>(blockIdx.y) * kRowBatch * by + (kNarrow ? threadIdx.y : 0u);
    prefetch_rows(m, first, by, rows, vec, c);
    wait_for_previous_kernel();
    release_next_kernel();
    if (c >= vec) return;
    uint4 emb[SS_MAX_GAMMA];
    #pragma unroll
    for (int j = 0; j < SS_MAX_GAMMA; ++j)
        if (j < gamma) emb[j] = __ldg(p + static_cast<long long>(j) * vec + c);
    const long long step = static_cast<long long>(gridDim.y) * kRowBatch * by;
    for (long long t = first; t < rows; t += step) {
        uint4 a[kRowBatch];
        #pragma unroll
        for (int i = 0; i < kRowBatch; ++i)
            if (t + i * by < rows) a[i] = m[(t + i * by) * vec + c];
        #pragma unroll
        for (int i = 0; i < kRowBatch; ++i) {
            #pragma unroll
            for (int j = 0; j < SS_MAX_GAMMA; ++j)
                if (j < gamma && t + i * by < rows) out[((t + i * by) * gamma + j) * vec + c] = add8(a[i], emb[j]);
        }
    }
}

// a 32-bit word holds one complex number (re in the low half, im in the high half)
__device__ __forceinline__ uint32_t rotate_word(uint32_t w, float cs, float sn) {
    const float re = bf16_lo(w), im = bf16_hi(w);
    return pack2(__fsub_rn(__fmul_rn(re, cs), __fmul_rn(im, sn)), __fadd_rn(__fmul_rn(re, sn), __fmul_rn(im, cs)));
}

// out[t][n][c] = v[t][c] rotated by eps * (n + 1)
template <bool kNarrow>
__global__ void __launch_bounds__(kNarrow ? 256 : 128)
value_rotate_kernel(const uint4* __restrict__ v, uint4* __restrict__ out, long long rows, int gamma, int vec, const __grid_constant__ RotTable tab) {
    const int c = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x), by = kNarrow ? static_cast<int>(blockDim.y) : 1;
    const long long first = static_cast<long long>(blockIdx.y) * kRowBatch * by + (kNarrow ? threadIdx.y : 0u);
    prefetch_rows(v, first, by, rows, vec, c);
    wait_for_previous_kernel();
    release_next_kernel();
    if (c >= vec) return;
    const long long step = static_cast<long long>(gridDim.y) * kRowBatch * by;
    for (long long t = first; t < rows; t += step) {
        uint4 a[kRowBatch];
        #pragma unroll
        for (int i = 0; i < kRowBatch; ++i)
            if (t + i * by < rows) a[i] = v[(t + i * by) * vec + c];
        #pragma unroll
        for (int i = 0; i < kRowBatch; ++i) {
            #pragma unroll
            for (int n = 0; n < SS_MAX_GAMMA; ++n) {
                if (n < gamma && t + i * by < rows) {
                    const float cs = tab.cs[n], sn = tab.sn[n];
                    uint4 r;
                    r.x = rotate_word(a[i].x, cs, sn); r.y = rotate_word(a[i].y, cs, sn);
                    r.z = rotate_word(a[i].z, cs, sn); r.w = rotate_word(a[i].w, cs, sn);
                    out[((t + i * by) * gamma + n) * vec + c] = r;
                }
            }
        }
    }
}

// 128 threads across the width.  A narrower one (kNarrow) has a thread for each of its vectors and as many rows as fit 256
// threads (262144 rows of 128, four streams, both calls 202 -> 108 us; 100000 of 8 55 -> 10 us).  Rows are dealt out
// until the SMs are full (16 such CTAs per SM).
static dim3 block_for(int vec) {
    return vec < 128 ? dim3(static_cast<unsigned>(vec), static_cast<unsigned>(256 / vec)) : dim3(128);
}
static dim3 grid_for(long long rows, int vec) {
    const int gx = (vec + 127) / 128;
    const long long per = static_cast<long long>(kRowBatch) * block_for(vec).y;
    long long gy = (rows + per - 1) / per;
    const long long cap = (static_cast<long long>(sm_count()) * 16 + gx - 1) / gx;
    if (gy > cap) gy = cap;
    if (gy > 65535) gy = 65535;
    return dim3(static_cast<unsigned>(gx), static_cast<unsigned>(gy < 1 ? 1 : gy));
}

}  // namespace ss

extern "C" int32_t ss_stream_insert(const void* main_hidden, const void* stream_emb, void* out, int64_t rows, int32_t gamma,
                                    int32_t hidden, void* stream) {
    if (rows < 0 || gamma < 1 || hidden < 8) return SS_ERR_INVALID_ARG;
    if (gamma > SS_MAX_GAMMA || (hidden & 7)) return SS_ERR_UNSUPPORTED;
    if (rows == 0) return SS_OK;                                   // nothing to do: the buffers may be empty
    if (!main_hidden || !stream_emb || !out) return SS_ERR_INVALID_ARG;
    if (!ss::aligned16(main_hidden) || !ss::aligned16(stream_emb) || !ss::aligned16(out)) return SS_ERR_INVALID_ARG;
    const int vec = hidden / 8;
    const cudaError_t err = ss::launch_after_previous(vec < 128 ? ss::stream_insert_kernel<true> : ss::stream_insert_kernel<false>, ss::grid_for(rows, vec), ss::block_for(vec),
                                                      static_cast<cudaStream_t>(stream), static_cast<const uint4*>(main_hidden),
                                                      static_cast<const uint4*>(stream_emb), static_cast<uint4*>(out),
                                                      static_cast<long long>(rows), gamma, vec);
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}

extern "C" int32_t ss_value_rotate(const void* v_main, void* v_streams, int64_t rows, int32_t gamma, int32_t width, float epsilon,
                                   void* stream) {
    if (rows < 0 || gamma < 1 || width < 8 || !(epsilon == epsilon)) return SS_ERR_INVALID_ARG;
    if (gamma > SS_MAX_GAMMA || (width & 7)) return SS_ERR_UNSUPPORTED;
    if (rows == 0) return SS_OK;                                   // nothing to do: the buffers may be empty
    if (!v_main || !v_streams) return SS_ERR_INVALID_ARG;
    if (!ss::aligned16(v_main) || !ss::aligned16(v_streams)) return SS_ERR_INVALID_ARG;
    ss::RotTable tab = {};
    for (int n = 0; n < gamma; ++n) {
        const double ang = static_cast<double>(epsilon) * (n + 1);
        tab.cs[n] = static_cast<float>(cos(ang));
        tab.sn[n] = static_cast<float>(sin(ang));
    }
    const int vec = width / 8;
    const cudaError_t err = ss::launch_after_previous(vec < 128 ? ss::value_rotate_kernel<true> : ss::value_rotate_kernel<false>, ss::grid_for(rows, vec), ss::block_for(vec),
                                                      static_cast<cudaStream_t>(stream), static_cast<const uint4*>(v_main),
                                                      static_cast<uint4*>(v_streams), static_cast<long long>(rows), gamma, vec, tab);
    return err == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}
