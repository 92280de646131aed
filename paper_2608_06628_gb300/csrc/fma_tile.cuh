// fma_tile.cuh -- register-tiled float32 products of the CUDA-core kernels.
//
// C[rows][n] += A[rows][k] B[n][k], 256 threads, k in tiles of 32.  The B tile sits in
// shared memory as n rows of 128 bytes (32 k) with the 16-byte granules of row n
// permuted by XOR with (n mod 8): the layout of a state tile in global memory
// (hybrid.h), so a state tile is copied as it is and the other operands (W, K, V) are
// laid out the same way when they are staged.  A thread owns TM rows x 8 columns (8
// apart) and every KL-th granule of k: eight lanes side by side read eight neighbouring
// n of one granule (all banks, no conflict), and the KL lanes of an output are added by
// shuffles at the end.  Splitting k over lanes keeps the 8 x 8 thread tile for tiles of
// 16 and 32 rows: a granule then takes 16 shared-memory loads for 128 packed FMAs
// (fma.rn.f32x2 over pairs of neighbouring k), which is where the two pipes balance.
#pragma once

#include <stdint.h>

#include "hybrid_common.cuh"

namespace hyb {
namespace fma {

constexpr int kThreads = 256;

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 ffma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float sum2(f32x2 v)
{
    return __uint_as_float((uint32_t)v) + __uint_as_float((uint32_t)(v >> 32));
}

// Thread -> outputs of an RT x PN panel (PN = 64 or 128): rows row0 + RL i (i < TM),
// columns col0 + 8 c (c < 8), granules kl, kl + KL, .. of every tile.
template <int PN, int RT>
struct Map {
    static constexpr int KL = RT == 64 && PN == 128 ? 2 : 4;   // lanes along k
    static constexpr int RL = 4 / KL;                          // lanes along the rows
    static constexpr int TM = RT * PN * KL / (8 * kThreads);
    static constexpr int NO = TM * 8 / KL;                     // outputs per lane after the sum over k
    static_assert(TM >= 2, "row tile too small for the panel");
    int row0, col0, kl;
    __device__ __forceinline__ Map()
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        constexpr int wc = PN / 64;   // warps side by side over the panel's columns
        kl = (lane >> 3) & (KL - 1);
        col0 = (warp % wc) * 64 + (lane & 7);
        row0 = (warp / wc) * (TM * RL) + (lane >> 3) / KL;
    }
    // row and column of this lane's o-th output after finish()
    __device__ __forceinline__ int row(int o) const { return row0 + RL * ((kl * NO + o) >> 3); }
    __device__ __forceinline__ int col(int o) const { return col0 + 8 * ((kl * NO + o) & 7); }
};

// acc += A[rows][k0 .. k0 + 32) B[cols]; a points at A[0][k0], b at the tile.
template <class M>
__device__ __forceinline__ void tile32(const M &m, const float *a, int lda, const float *b, f32x2 (&acc)[M::TM * 8])
{
    const float *ar = a + m.row0 * lda;
    const float *br = b + m.col0 * 32;
    const int sw = m.col0 & 7;
#pragma unroll
    for (int jj = 0; jj < 8 / M::KL; ++jj) {
        const int j = m.kl + M::KL * jj;
        const int off = (j ^ sw) << 2;
        ulonglong2 bv[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) bv[c] = *reinterpret_cast<const ulonglong2 *>(br + c * 256 + off);
#pragma unroll
        for (int i = 0; i < M::TM; ++i) {
            const ulonglong2 av = *reinterpret_cast<const ulonglong2 *>(ar + i * M::RL * lda + 4 * j);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i * 8 + c] = ffma2(av.x, bv[c].x, acc[i * 8 + c]);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i * 8 + c] = ffma2(av.y, bv[c].y, acc[i * 8 + c]);
        }
    }
}

template <int N>
__device__ __forceinline__ void clear(f32x2 (&acc)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = 0ull;
}

// The sums over k: each of an output's KL lanes keeps NO of the TM x 8 outputs.
template <class M>
__device__ __forceinline__ void finish(const M &m, const f32x2 (&acc)[M::TM * 8], float (&out)[M::NO])
{
    constexpr int N = M::TM * 8;
    float v[N];
#pragma unroll
    for (int o = 0; o < N; ++o) v[o] = sum2(acc[o]);
    constexpr int H = N / 2;
    const bool up1 = m.kl & (M::KL / 2);
#pragma unroll
    for (int o = 0; o < H; ++o) {
        const float send = up1 ? v[o] : v[o + H], keep = up1 ? v[o + H] : v[o];
        v[o] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * M::KL);
    }
    if constexpr (M::KL == 4) {
        constexpr int H2 = H / 2;
        const bool up0 = m.kl & 1;
#pragma unroll
        for (int o = 0; o < H2; ++o) {
            const float send = up0 ? v[o] : v[o + H2], keep = up0 ? v[o + H2] : v[o];
            v[o] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
    }
#pragma unroll
    for (int o = 0; o < M::NO; ++o) out[o] = v[o];
}

// Four consecutive values of an I/O tensor at element offset i (a multiple of 4).
__device__ __forceinline__ float4 load4(const void *base, size_t i, bool bf16_io)
{
    if (bf16_io) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(static_cast<const __nv_bfloat16 *>(base) + i));
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16),
                           __uint_as_float(v.y & 0xFFFF0000u));
    }
    return __ldg(reinterpret_cast<const float4 *>(static_cast<const float *>(base) + i));
}

// A 4 x 4 block (rows k = 4 kq + i, columns n = 4 nq ..) into a tile, transposed.
__device__ __forceinline__ void store_block(float *tile, int kq, int nq, const float4 *x)
{
    float *t = tile + 4 * nq * 32;
    const int n0 = 4 * nq & 7;
    *reinterpret_cast<float4 *>(t + ((kq ^ n0) << 2)) = make_float4(x[0].x, x[1].x, x[2].x, x[3].x);
    *reinterpret_cast<float4 *>(t + 32 + ((kq ^ (n0 + 1)) << 2)) = make_float4(x[0].y, x[1].y, x[2].y, x[3].y);
    *reinterpret_cast<float4 *>(t + 64 + ((kq ^ (n0 + 2)) << 2)) = make_float4(x[0].z, x[1].z, x[2].z, x[3].z);
    *reinterpret_cast<float4 *>(t + 96 + ((kq ^ (n0 + 3)) << 2)) = make_float4(x[0].w, x[1].w, x[2].w, x[3].w);
}

// A tile on its way from global to shared memory: its loads are issued before the
// products of the tile in front of it and its stores after them.
struct Staged {
    static constexpr int R4 = 4;   // at most 128 rows of 32 k
    float4 r[R4];

    // Operand stored k-contiguous, B[n][k0 .. k0 + 32): row n at element base0 + n * stride.
    __device__ __forceinline__ void load_rows(const void *base, size_t base0, size_t stride, int n_rows, bool bf16_io)
    {
#pragma unroll
        for (int q = 0; q < R4; ++q) {
            const int p = threadIdx.x + q * kThreads;
            const int n = p >> 3, j = p & 7;
            if (n < n_rows) r[q] = load4(base, base0 + (size_t)n * stride + 4 * j, bf16_io);
        }
    }
    __device__ __forceinline__ void store_rows(float *tile, int n_rows) const
    {
#pragma unroll
        for (int q = 0; q < R4; ++q) {
            const int p = threadIdx.x + q * kThreads;
            const int n = p >> 3, j = p & 7;
            if (n < n_rows) *reinterpret_cast<float4 *>(tile + n * 32 + ((j ^ (n & 7)) << 2)) = r[q];
        }
    }
    // Operand stored n-contiguous, B[k0 + k][n] at element base0 + k * stride + n: 4 x 4
    // blocks, transposed in registers (rows k >= n_k are zero).  Eight lanes take the eight
    // k-groups of one n-group, so that their stores fall into different banks.
    __device__ __forceinline__ void load_cols(const void *base, size_t base0, size_t stride, int n_k, int n_cols,
                                              bool bf16_io)
    {
        const int kq = threadIdx.x & 7, nq = threadIdx.x >> 3;
        if (4 * nq >= n_cols) return;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = 4 * kq + i;
            r[i] = k < n_k ? load4(base, base0 + (size_t)k * stride + 4 * nq, bf16_io)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __device__ __forceinline__ void store_cols(float *tile, int n_cols) const
    {
        const int kq = threadIdx.x & 7, nq = threadIdx.x >> 3;
        if (4 * nq >= n_cols) return;
        store_block(tile, kq, nq, r);
    }
    // A state tile (n_rows rows of 128 bytes), already in the tile layout.  (Plain loads, as for z:
    // the kernel may start while the one in front still writes the state, so the state is not
    // read-only for its lifetime, as __ldg asks.)
    __device__ __forceinline__ void load_tile(const float *src, int n_rows)
    {
#pragma unroll
        for (int q = 0; q < R4; ++q) {
            const int p = threadIdx.x + q * kThreads;
            if (p < n_rows * 8) r[q] = reinterpret_cast<const float4 *>(src)[p];
        }
    }
    __device__ __forceinline__ void store_tile(float *tile, int n_rows) const
    {
#pragma unroll
        for (int q = 0; q < R4; ++q) {
            const int p = threadIdx.x + q * kThreads;
            if (p < n_rows * 8) reinterpret_cast<float4 *>(tile)[p] = r[q];
        }
    }
};

// Panels of U = X W (F columns): FP = 0 one of 64 (F <= 64), 1 one of 128, 2 two of 128.
template <int FP>
struct UPanels {
    static constexpr int PN = FP == 0 ? 64 : 128;
    static constexpr int N = FP == 2 ? 2 : 1;
};

// Row statistics over the outputs of a panel, in the registers finish() leaves them in:
// a lane holds RPL rows x CPL columns; a row's columns are spread over 8 lanes (16 when a
// lane has only half of them) and, for PN = 128, over two warps side by side.
template <int PN, int RT>
struct Rows {
    using M = Map<PN, RT>;
    static constexpr int RPL = M::NO >= 8 ? M::NO / 8 : 1, CPL = M::NO / RPL;
    static constexpr int kWarps = PN / 64;
    // op: 0 add, 1 max, 2 min
    template <int kOp>
    static __device__ __forceinline__ float comb(float a, float b)
    {
        return kOp == 0 ? a + b : kOp == 1 ? fmaxf(a, b) : fminf(a, b);
    }
    template <int kOp>
    static __device__ __forceinline__ float lanes(float v)
    {
        v = comb<kOp>(v, __shfl_xor_sync(0xffffffffu, v, 1));
        v = comb<kOp>(v, __shfl_xor_sync(0xffffffffu, v, 2));
        v = comb<kOp>(v, __shfl_xor_sync(0xffffffffu, v, 4));
        if (CPL < 8) v = comb<kOp>(v, __shfl_xor_sync(0xffffffffu, v, 8));
        return v;
    }
    // exchange between the two warps of a row through x[2][RT] per statistic: put, barrier, get
    static __device__ __forceinline__ void put(float *x, const M &m, int j, float v)
    {
        if constexpr (kWarps > 1) {
            if ((threadIdx.x & 7) == 0) x[((threadIdx.x >> 5) & 1) * RT + m.row(j * CPL)] = v;
        }
    }
    template <int kOp>
    static __device__ __forceinline__ float get(const float *x, const M &m, int j, float own)
    {
        if constexpr (kWarps > 1) return comb<kOp>(x[m.row(j * CPL)], x[RT + m.row(j * CPL)]);
        else return own;
    }
    static __device__ __forceinline__ void sync()
    {
        if constexpr (kWarps > 1) __syncthreads();
    }
};

// Hedgehog features of the panels' rows: u[p][o] (column p PN + col(o), valid below F)
// becomes the phi+ value and un the phi- value, both max-shifted and normalised.  With
// kDen, ld[j] = phi . z of the lane's j-th row.  x: xch_floats(RT) floats of shared memory.
template <int PN, int RT, int N, bool kDen>
__device__ __forceinline__ void phi_rows(const Map<PN, RT> &m, int F, float (&u)[N][Map<PN, RT>::NO],
                                         float (&un)[N][Map<PN, RT>::NO], const float *z,
                                         float (&ld)[Rows<PN, RT>::RPL], float *x)
{
    using R = Rows<PN, RT>;
    constexpr int RPL = R::RPL, CPL = R::CPL;
    float mx[RPL], mn[RPL];
#pragma unroll
    for (int j = 0; j < RPL; ++j) {
        mx[j] = -INFINITY;
        mn[j] = INFINITY;
#pragma unroll
        for (int p = 0; p < N; ++p)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const float v = u[p][j * CPL + c];
                const bool in = PN == 128 || m.col(j * CPL + c) < F;
                mx[j] = fmaxf(mx[j], in ? v : -INFINITY);
                mn[j] = fminf(mn[j], in ? v : INFINITY);
            }
        mx[j] = R::template lanes<1>(mx[j]);
        mn[j] = R::template lanes<2>(mn[j]);
        R::put(x, m, j, mx[j]);
        R::put(x + 2 * RT, m, j, mn[j]);
    }
    R::sync();
    float zp[N][CPL], zn[N][CPL];
    if constexpr (kDen) {
#pragma unroll
        for (int p = 0; p < N; ++p)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int f = p * PN + m.col(c);
                zp[p][c] = f < F ? z[f] : 0.f;
                zn[p][c] = f < F ? z[F + f] : 0.f;
            }
    }
    float sp[RPL], sn[RPL], lp[RPL], ln[RPL];
    float *xs = x + 4 * RT;
#pragma unroll
    for (int j = 0; j < RPL; ++j) {
        const float hi = R::template get<1>(x, m, j, mx[j]), lo = R::template get<2>(x + 2 * RT, m, j, mn[j]);
        sp[j] = sn[j] = lp[j] = ln[j] = 0.f;
#pragma unroll
        for (int p = 0; p < N; ++p)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const bool in = PN == 128 || m.col(j * CPL + c) < F;
                float &vp = u[p][j * CPL + c], &vn = un[p][j * CPL + c];
                vn = in ? expf(lo - vp) : 0.f;
                vp = in ? expf(vp - hi) : 0.f;
                sp[j] += vp;
                sn[j] += vn;
                if constexpr (kDen) {
                    lp[j] = fmaf(vp, zp[p][c], lp[j]);
                    ln[j] = fmaf(vn, zn[p][c], ln[j]);
                }
            }
        sp[j] = R::template lanes<0>(sp[j]);
        sn[j] = R::template lanes<0>(sn[j]);
        R::put(xs, m, j, sp[j]);
        R::put(xs + 2 * RT, m, j, sn[j]);
        if constexpr (kDen) {
            lp[j] = R::template lanes<0>(lp[j]);
            ln[j] = R::template lanes<0>(ln[j]);
            R::put(xs + 4 * RT, m, j, lp[j]);
            R::put(xs + 6 * RT, m, j, ln[j]);
        }
    }
    R::sync();
#pragma unroll
    for (int j = 0; j < RPL; ++j) {
        const float ip = 1.f / R::template get<0>(xs, m, j, sp[j]);
        const float in_ = 1.f / R::template get<0>(xs + 2 * RT, m, j, sn[j]);
        if constexpr (kDen)
            ld[j] = R::template get<0>(xs + 4 * RT, m, j, lp[j]) * ip + R::template get<0>(xs + 6 * RT, m, j, ln[j]) * in_;
#pragma unroll
        for (int p = 0; p < N; ++p)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                u[p][j * CPL + c] *= ip;
                un[p][j * CPL + c] *= in_;
            }
    }
}

// floats of shared memory that phi_rows and the score softmax exchange statistics in
__host__ __device__ constexpr int xch_floats(int RT) { return 12 * RT; }

}  // namespace fma
}  // namespace hyb
