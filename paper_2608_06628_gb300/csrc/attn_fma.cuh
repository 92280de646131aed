// attn_fma.cuh -- the block-hybrid step of Section 3.1 on the CUDA cores, float32
// throughout: float32 I/O, and the few bf16 shapes that the tensor-core kernels do not take
// (G not a divisor of 128).
//
// One CTA takes RT of the G B query rows (row t G + h) of a unit (request, state head),
// so that W, K, V and the state are read once per RT rows rather than once per query
// head and 16 rows.  All four products (U = Q W, Q K^T, phi(Q) S, P V) run through the
// register tiles of fma_tile.cuh over one stream of 32-deep operand tiles, each loaded
// to registers while the tile in front of it is multiplied.
//
// What bounds it: the shared-memory and FMA pipes (a row costs 2 d F + 4 F d + 4 B d
// operations; tensor cores cannot be used for float32 inputs without losing precision).
// One request, 2 heads, d = F = 64, B = 16, float32: 26.6 us with one CTA per query head and
// 16 rows, 8.8 us now (the host's launch time is 8 us).
#pragma once

#include <atomic>

#include "fma_tile.cuh"
#include "hybrid_kernels.h"
#include "tc_pipeline.cuh"

namespace hyb {
namespace fma {

struct AttnArgs {
    const void *Q, *K, *V, *W;
    const float *alpha;
    void *const *states;
    void *O;
    unsigned *err;
    int B, Hq, Hkv, G, F, tiles;   // tiles: row tiles per unit
    bool bf16_io;
};

__host__ __device__ constexpr int round_up(int x, int m) { return (x + m - 1) / m * m; }

// floats of an operand tile: 64 or 128 rows of 32
__host__ __device__ constexpr int attn_tile_floats(int d, int F, int B)
{
    return (d > 64 || F > 64 || B > 64 ? 128 : 64) * 32;
}
// Q rows, phi rows, score rows, two operand tiles, row results, exchanged statistics
inline size_t attn_smem_bytes(int d, int F, int B, int RT)
{
    return sizeof(float) * ((size_t)RT * (d + 4) + (size_t)RT * (2 * F + 4) + (size_t)RT * (round_up(B, 32) + 4) +
                            2 * (size_t)attn_tile_floats(d, F, B) + 5 * RT + xch_floats(RT));
}

template <int D, int RT, int FP>
__global__ void __launch_bounds__(kThreads) k_attn_fma(const AttnArgs a)
{
    extern __shared__ __align__(16) float smem[];
    using UP = UPanels<FP>;
    using MU = Map<UP::PN, RT>;
    using MD = Map<D, RT>;
    constexpr int ND = D / 32;                 // k-tiles of U and of the scores
    const int F = a.F, B = a.B, G = a.G, P2 = 2 * F;
    const int NF = (P2 + 31) / 32, NB = (B + 31) / 32;
    constexpr int LQ = D + 4;
    const int LP = P2 + 4, LB = NB * 32 + 4;
    const int tile_floats = attn_tile_floats(D, F, B);
    float *qs = smem;                          // [RT][LQ]
    float *ph = qs + RT * LQ;                  // [RT][LP] U, then phi
    float *ps = ph + RT * LP;                  // [RT][LB] scores, then e^(s - m)
    float *tb = ps + RT * LB;                  // two operand tiles
    float *wsm = tb + 2 * tile_floats;         // [RT] weight of the softmax numerator
    float *wlm = wsm + RT;                     // [RT] weight of the linear numerator
    float *rm = wlm + RT;                      // [RT] max score, [RT] sum e^(s - m), [RT] phi . z
    float *xch = rm + 3 * RT;                  // statistics on their way between warps

    const int tid = threadIdx.x;
    const int unit = blockIdx.x / a.tiles, i0 = (blockIdx.x % a.tiles) * RT;
    const int r = unit / a.Hkv, g = unit % a.Hkv;
    const int rows = min(RT, G * B - i0);

    ptx::griddep_launch_dependents();
    ptx::griddep_wait();
    const float *state = reinterpret_cast<const float *>(a.states[r]);
    if (!state_ptr_ok(state)) {
        if (tid == 0 && i0 == 0) raise_error(a.err, ERR_BAD_STATE_PTR);
        return;
    }
    const float *Sg = state + (size_t)g * head_floats(D, F);
    const float *zg = Sg + (size_t)P2 * D;
    const size_t w0 = (size_t)g * D * F;                               // W_g
    const size_t kv0 = ((size_t)r * B * a.Hkv + g) * D;                // token 0 of K, V
    const size_t kv_stride = (size_t)a.Hkv * D;

    // the tile stream: the next tile's loads, and its stores into buffer b
    Staged st;
    const int FC = FP == 2 ? 128 : F;          // columns of a W tile: tile k of panel p is the stream's p ND + k
    auto load_w = [&](int i) {
        st.load_cols(a.W, w0 + (size_t)(i % ND) * 32 * F + (i / ND) * UP::PN, F, 32, FC, a.bf16_io);
    };
    auto load_k = [&](int k) { st.load_rows(a.K, kv0 + k * 32, kv_stride, B, a.bf16_io); };
    auto load_s = [&](int t) { st.load_tile(Sg + (size_t)t * 32 * D, D); };
    auto load_v = [&](int t) {
        st.load_cols(a.V, kv0 + (size_t)t * 32 * kv_stride, kv_stride, B - 32 * t, D, a.bf16_io);
    };
    auto buf = [&](int b) { return tb + (b & 1) * tile_floats; };

    load_w(0);
    for (int p = tid; p < RT * (D / 4); p += kThreads) {
        const int i = p / (D / 4), e = (p % (D / 4)) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < rows) {
            const int t = (i0 + i) / G, h = (i0 + i) % G;
            v = load4(a.Q, (((size_t)r * B + t) * a.Hq + g * G + h) * D + e, a.bf16_io);
        }
        *reinterpret_cast<float4 *>(qs + i * LQ + e) = v;
    }
    st.store_cols(buf(0), FC);
    __syncthreads();

    int s = 0;   // tile in the stream
    // ---- U = Q W, then phi(q) and lin_den = phi(q) . z in registers
    {
        using R = Rows<UP::PN, RT>;
        const MU mu;
        float u[UP::N][MU::NO], un[UP::N][MU::NO], ld[R::RPL];
#pragma unroll
        for (int p = 0; p < UP::N; ++p) {
            f32x2 acc[MU::TM * 8];
            clear(acc);
#pragma unroll 1
            for (int k = 0; k < ND; ++k, ++s) {
                const bool more = s + 1 < UP::N * ND;
                if (more) load_w(s + 1);
                else load_k(0);
                tile32(mu, qs + 32 * k, LQ, buf(s), acc);
                if (more) st.store_cols(buf(s + 1), FC);
                else st.store_rows(buf(s + 1), B);
                __syncthreads();
            }
            finish(mu, acc, u[p]);
        }
        phi_rows<UP::PN, RT, UP::N, true>(mu, F, u, un, zg, ld, xch);
#pragma unroll
        for (int j = 0; j < R::RPL; ++j) {
            const int row = mu.row(j * R::CPL);
            float *out = ph + row * LP;
#pragma unroll
            for (int p = 0; p < UP::N; ++p)
#pragma unroll
                for (int c = 0; c < R::CPL; ++c) {
                    const int f = p * UP::PN + mu.col(j * R::CPL + c);
                    if (UP::PN == 128 || f < F) {
                        out[f] = u[p][j * R::CPL + c];
                        out[F + f] = un[p][j * R::CPL + c];
                    }
                }
            if (mu.col(0) == 0) rm[2 * RT + row] = ld[j];
        }
    }
    // ---- scores Q K^T / sqrt(d), every pair (no mask), and e^(s - m)
    const float inv_sqrt_d = rsqrtf((float)D);
    auto scores = [&](auto m, auto r) {
        using M = decltype(m);
        using R = decltype(r);
        f32x2 acc[M::TM * 8];
        clear(acc);
#pragma unroll 1
        for (int k = 0; k < ND; ++k, ++s) {
            if (k + 1 < ND) load_k(k + 1);
            else load_s(0);
            tile32(m, qs + 32 * k, LQ, buf(s), acc);
            if (k + 1 < ND) st.store_rows(buf(s + 1), B);
            else st.store_tile(buf(s + 1), D);
            __syncthreads();
        }
        float x[M::NO], mx[R::RPL], l[R::RPL];
        finish(m, acc, x);
#pragma unroll
        for (int j = 0; j < R::RPL; ++j) {
            mx[j] = -INFINITY;
#pragma unroll
            for (int c = 0; c < R::CPL; ++c) {
                float &v = x[j * R::CPL + c];
                v = m.col(j * R::CPL + c) < B ? v * inv_sqrt_d : -INFINITY;
                mx[j] = fmaxf(mx[j], v);
            }
            mx[j] = R::template lanes<1>(mx[j]);
            R::put(xch, m, j, mx[j]);
        }
        R::sync();
#pragma unroll
        for (int j = 0; j < R::RPL; ++j) {
            const int row = m.row(j * R::CPL);
            mx[j] = R::template get<1>(xch, m, j, mx[j]);
            l[j] = 0.f;
#pragma unroll
            for (int c = 0; c < R::CPL; ++c) {
                const int col = m.col(j * R::CPL + c);
                const float e = col < B ? expf(x[j * R::CPL + c] - mx[j]) : 0.f;
                l[j] += e;
                if (col < 32 * NB) ps[row * LB + col] = e;   // zero beyond B: the last V tile is 32 deep
            }
            l[j] = R::template lanes<0>(l[j]);
            R::put(xch + 2 * RT, m, j, l[j]);
        }
        R::sync();
#pragma unroll
        for (int j = 0; j < R::RPL; ++j) {
            l[j] = R::template get<0>(xch + 2 * RT, m, j, l[j]);
            if (m.col(0) == 0) {
                rm[m.row(j * R::CPL)] = mx[j];
                rm[RT + m.row(j * R::CPL)] = l[j];
            }
        }
    };
    if (B > 64) scores(Map<128, RT>(), Rows<128, RT>());
    else scores(Map<64, RT>(), Rows<64, RT>());
    __syncthreads();
    // merge weights of a row (read after the readout's barriers)
    if (tid < rows) {
        const MergeWeights mw =
            merge_weights(log_sigmoid(a.alpha[g * G + (i0 + tid) % G]), rm[tid], rm[RT + tid], rm[2 * RT + tid]);
        wsm[tid] = mw.ws;
        wlm[tid] = mw.wl;
    }

    // ---- lin_num = phi(q)^T S, then sm_num = P V
    const MD md;
    float lin[MD::NO], num[MD::NO];
    f32x2 acc[MD::TM * 8];
    clear(acc);
#pragma unroll 1
    for (int t = 0; t < NF; ++t, ++s) {
        if (t + 1 < NF) load_s(t + 1);
        else load_v(0);
        tile32(md, ph + 32 * t, LP, buf(s), acc);
        if (t + 1 < NF) st.store_tile(buf(s + 1), D);
        else st.store_cols(buf(s + 1), D);
        __syncthreads();
    }
    finish(md, acc, lin);
    clear(acc);
#pragma unroll 1
    for (int t = 0; t < NB; ++t, ++s) {
        if (t + 1 < NB) load_v(t + 1);
        tile32(md, ps + 32 * t, LB, buf(s), acc);
        if (t + 1 < NB) {
            st.store_cols(buf(s + 1), D);
            __syncthreads();
        }
    }
    finish(md, acc, num);
    // ---- gated shared-normaliser merge and store
    using R = Rows<D, RT>;
#pragma unroll
    for (int j = 0; j < R::RPL; ++j) {
        const int row = md.row(j * R::CPL);
        if (row >= rows) continue;
        const float ws = wsm[row], wl = wlm[row];
        const int t = (i0 + row) / G, h = (i0 + row) % G;
        const size_t o = (((size_t)r * B + t) * a.Hq + g * G + h) * D;
#pragma unroll
        for (int c = 0; c < R::CPL; ++c) {
            const int i = j * R::CPL + c;
            const float val = ws * num[i] + (wl == 0.f ? 0.f : wl * lin[i]);
            if (a.bf16_io) static_cast<__nv_bfloat16 *>(a.O)[o + md.col(i)] = __float2bfloat16_rn(val);
            else static_cast<float *>(a.O)[o + md.col(i)] = val;
        }
    }
}

// Launch with programmatic stream serialisation, the kernel's dynamic shared memory
// opted in once per device.
template <class Kern, class Args>
cudaError_t launch_opted(Kern kern, std::atomic<unsigned long long> &opted, unsigned grid, size_t smem,
                         cudaStream_t st, const Args &a, unsigned cluster = 1)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const unsigned long long bit = 1ull << dev;
    if (!(opted.load(std::memory_order_acquire) & bit)) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
        if (e != cudaSuccess) return e;
        opted.fetch_or(bit, std::memory_order_release);
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(kThreads);
    // up to a CTA per SM: ask for the SM's shared memory, or the block scheduler puts two on
    // one SM while others idle
    lc.dynamicSmemBytes = cluster == 1 && grid <= (unsigned)pipe::sm_count() && smem < 118 * 1024 ? 118 * 1024 : smem;
    lc.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&lc, kern, a);
}

template <int D, int RT, int FP>
cudaError_t launch_attn_rt(AttnArgs a, int n_req, cudaStream_t st)
{
    static std::atomic<unsigned long long> opted{0};
    a.tiles = (a.G * a.B + RT - 1) / RT;
    const unsigned grid = (unsigned)((long long)n_req * a.Hkv * a.tiles);
    return launch_opted(&k_attn_fma<D, RT, FP>, opted, grid, attn_smem_bytes(D, a.F, a.B, RT), st, a);
}

template <int D, int FP>
cudaError_t launch_attn_f(const AttnArgs &a, int n_req, int rt, cudaStream_t st)
{
    if (rt == 64) {
        if constexpr (FP < 2) return launch_attn_rt<D, 64, FP>(a, n_req, st);
    }
    return rt >= 32 ? launch_attn_rt<D, 32, FP>(a, n_req, st) : launch_attn_rt<D, 16, FP>(a, n_req, st);
}

template <int D>
cudaError_t launch_attn_d(const AttnArgs &a, int n_req, int rt, cudaStream_t st)
{
    if (a.F <= 64) return launch_attn_f<D, 0>(a, n_req, rt, st);
    if (a.F == 128) return launch_attn_f<D, 1>(a, n_req, rt, st);
    return launch_attn_f<D, 2>(a, n_req, rt, st);
}

cudaError_t launch_attn_d64(const AttnArgs &a, int n_req, int rt, cudaStream_t st);
cudaError_t launch_attn_d128(const AttnArgs &a, int n_req, int rt, cudaStream_t st);

}  // namespace fma
}  // namespace hyb
