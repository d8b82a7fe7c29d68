// Rotary position encoding of bf16 rows, in place (an optional helper; the attention path rotates nothing).
// Paper, Sec. 3.2: positions are encoded as in the cited rotary embedding and every group keeps the positions it
// was computed with.  Formula as published (Su et al., "RoFormer"): pair j of a head is turned by pos * base^(-2j/D).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "../../include/enl.h"
#include "enl_internal.h"

namespace {

constexpr int kMaxPairs = ENL_ROPE_MAX_HEAD_DIM / 2;
constexpr int kThreads  = 256;
constexpr int kMaxRows  = 4;                  // rows per CTA of the wide kernel

struct RopeParams {
    double inv_freq[kMaxPairs];       // base^(-2j/D), formed on the host in double
    __nv_bfloat16 *rows;
    const int32_t *positions;
    long long n_pairs_total;          // n * n_heads * D / 2
    int32_t n, n_heads, D, first_pos, interleaved, rows_per_cta;
};

// the angle in double, brought into [-pi, pi] before it is rounded to fp32: positions reach 1e5 and more
__device__ __forceinline__ void turn_of(const RopeParams &p, long long row, int j, float &sn, float &cs)
{
    const int pos = p.positions ? p.positions[row] : p.first_pos + static_cast<int>(row);
    const double two_pi = 6.283185307179586476925286766559;
    double ang = static_cast<double>(pos) * p.inv_freq[j];
    ang -= two_pi * rint(ang / two_pi);
    sincosf(static_cast<float>(ang), &sn, &cs);
}
__device__ __forceinline__ void turn(float &x1, float &x2, float sn, float cs)
{
    const float a = x1, b = x2;
    x1 = a * cs - b * sn;
    x2 = b * cs + a * sn;
}

// A turn is the same for every head of a row: a CTA works the turns of its rows out once (the double-precision angle and the
// sine and cosine are most of the arithmetic) and its threads then take 16-byte pieces of the heads.  Bound by memory from there on.
// One thread per pair with 2-byte accesses, every turn worked out for every head, took 17.2 us for 820 rows of 32 heads, D 128
// (6.7 MB read and written); 5.5 us here, 5.8 -> 3.9 for 8 heads.
__global__ void __launch_bounds__(kThreads) rope_wide_kernel(const __grid_constant__ RopeParams p)
{
    __shared__ float2 turns[kMaxRows * kMaxPairs];
    const int half = p.D / 2;
    const long long row0 = static_cast<long long>(blockIdx.x) * p.rows_per_cta;
    const int n_rows = static_cast<int>(min(static_cast<long long>(p.rows_per_cta), p.n - row0));
    enl::pdl_trigger();
    enl::pdl_wait();                                   // the rows may come from the kernel before
    for (int i = threadIdx.x; i < n_rows * half; i += kThreads) {
        float sn, cs;
        turn_of(p, row0 + i / half, i % half, sn, cs);
        turns[i] = make_float2(sn, cs);
    }
    __syncthreads();
    // a piece: the 8 channels j .. j + 7 of the first half and their partners of the second, or 16 channels in a row
    const int per_head = p.D / 16, per_row = p.n_heads * per_head;
    for (int i = threadIdx.x; i < n_rows * per_row; i += kThreads) {
        const int r = i / per_row, hp = i % per_row, head = hp / per_head, c = hp % per_head;
        __nv_bfloat16 *base = p.rows + ((row0 + r) * p.n_heads + head) * p.D;
        uint4 *a = reinterpret_cast<uint4 *>(base + (p.interleaved ? c * 16 : c * 8));
        uint4 *b = reinterpret_cast<uint4 *>(base + (p.interleaved ? c * 16 + 8 : half + c * 8));
        uint4 va = *a, vb = *b;
        __nv_bfloat162 *xa = reinterpret_cast<__nv_bfloat162 *>(&va), *xb = reinterpret_cast<__nv_bfloat162 *>(&vb);
        const float2 *t = turns + r * half + c * 8;    // of the piece's eight pairs
        if (p.interleaved) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                __nv_bfloat162 &x = k < 4 ? xa[k] : xb[k - 4];
                float2 f = __bfloat1622float2(x);
                turn(f.x, f.y, t[k].x, t[k].y);
                x = __floats2bfloat162_rn(f.x, f.y);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float2 f = __bfloat1622float2(xa[k]), g = __bfloat1622float2(xb[k]);
                turn(f.x, g.x, t[2 * k].x, t[2 * k].y);
                turn(f.y, g.y, t[2 * k + 1].x, t[2 * k + 1].y);
                xa[k] = __floats2bfloat162_rn(f.x, f.y);
                xb[k] = __floats2bfloat162_rn(g.x, g.y);
            }
        }
        *a = va;
        *b = vb;
    }
}

// rows that the wide kernel cannot take 16 bytes at a time: one thread per (row, head, pair)
__global__ void rope_kernel(const __grid_constant__ RopeParams p)
{
    const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    enl::pdl_trigger();
    enl::pdl_wait();                                   // the rows may come from the kernel before
    if (idx >= p.n_pairs_total) return;
    const int half = p.D / 2;
    const int j = static_cast<int>(idx % half);
    const long long rh = idx / half;                   // (row, head)
    float sn, cs;
    turn_of(p, rh / p.n_heads, j, sn, cs);
    __nv_bfloat16 *base = p.rows + rh * p.D;
    const int i1 = p.interleaved ? 2 * j : j, i2 = p.interleaved ? 2 * j + 1 : j + half;
    float x1 = __bfloat162float(base[i1]), x2 = __bfloat162float(base[i2]);
    turn(x1, x2, sn, cs);
    base[i1] = __float2bfloat16_rn(x1);
    base[i2] = __float2bfloat16_rn(x2);
}

}  // namespace

extern "C" int enl_rope_rotate(void *rows, int32_t n, int32_t n_heads, int32_t head_dim, const int32_t *positions,
                               int32_t first_pos, double base, int32_t interleaved, void *cuda_stream)
{
    if (!rows || n < 0 || n_heads < 1 || head_dim < 2 || (head_dim & 1) || !(base > 0.0)) return ENL_E_INVAL;
    if (reinterpret_cast<uintptr_t>(rows) & 3) return ENL_E_INVAL;
    if (head_dim > ENL_ROPE_MAX_HEAD_DIM) return ENL_E_LIMIT;
    if (n == 0) return ENL_OK;
    // The frequencies depend on base and head_dim only: the last ones are kept (64 powers are 3 us of host time).
    static thread_local RopeParams p;
    static thread_local double have_base = 0.0;
    static thread_local int have_dim = 0;
    if (have_base != base || have_dim != head_dim) {
        for (int j = 0; j < kMaxPairs; ++j)
            p.inv_freq[j] = j < head_dim / 2 ? std::pow(base, -2.0 * j / head_dim) : 0.0;
        have_base = base;
        have_dim = head_dim;
    }
    p.rows = static_cast<__nv_bfloat16 *>(rows);
    p.positions = positions;
    p.n_pairs_total = static_cast<long long>(n) * n_heads * (head_dim / 2);
    p.n = n;
    p.n_heads = n_heads;
    p.D = head_dim;
    p.first_pos = first_pos;
    p.interleaved = interleaved ? 1 : 0;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e;
    if (head_dim % 16 == 0 && (reinterpret_cast<uintptr_t>(rows) & 15) == 0) {
        // few heads: several rows per CTA, so that every thread has a piece
        p.rows_per_cta = std::max(1, std::min(kMaxRows, kThreads / (n_heads * (head_dim / 16))));
        e = enl::launch_pdl(rope_wide_kernel, dim3(static_cast<unsigned>((n + p.rows_per_cta - 1) / p.rows_per_cta)), dim3(kThreads), 0, st, p);
    } else {
        const long long blocks = (p.n_pairs_total + kThreads - 1) / kThreads;
        if (blocks > 0x7fffffffll) return ENL_E_LIMIT;
        e = enl::launch_pdl(rope_kernel, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, st, p);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return ENL_E_CUDA;
    }
    return ENL_OK;
}
