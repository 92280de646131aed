// hybrid_attn_split.cu -- the block-hybrid step of Section 3.1 for the bf16 shapes that the
// streaming tensor-core kernels do not take (more than 128 query rows to a state, B not a
// multiple of 16, F < 64), on the tensor cores at float32 accuracy.
//
// These shapes ran float32 FMA kernels and keep that accuracy: bf16 products (U = Q W and
// the scores) are exact in float32, and every float32 operand of the other products goes in
// as a sum of parts,
//   phi S = phi_h S_h + phi_l S_h + phi_h S_l   tf32 parts x = x_h + x_l, x_h = x cut to 11
//                                               bits: what is left out is 2^-22 of a term
//   P V   = P_h V + P_l V                       bf16 parts of e^(s - m), 2^-17
// so the result differs from the FMA kernels' by less than its own bf16 rounding (2^-9).
// The merge weights of a row are known before the readout and are folded into phi and P, so
// one accumulator D takes both branches and holds the output.
//
// A work item is 128 of a unit's G B query rows (row t G + h, whole tokens).  256 threads, two
// per row; two CTAs per SM (F <= 128: 256 Tensor Memory columns and <= 110 KB of shared
// memory each), so that one's products run under the other's conversions.  Per 32-feature
// state tile the threads form phi's parts from U (kept in Tensor Memory) and the parts of
// the tile (through registers, loaded one tile ahead), and one thread issues 12 MMAs.
// Tensor Memory: [U (64, 128 or 256 columns) | D], the scores in D's columns until P V.
//
// What bounds it: per tile, forming the operands (0.4 us) and 12 MMAs (0.7 us), one after the
// other in a CTA; two CTAs on an SM overlap them.  32 requests, 16 : 4 heads, d = F = 128, B =
// 64: 29.7 us against 196 us on the CUDA cores (F = 256: 56 against 328); relative error
// against 64 bits 1.66e-3 on both, the rounding of a bf16 output.
#include <atomic>

#include "hybrid_common.cuh"
#include "hybrid_tc.h"
#include "tc_pipeline.cuh"

namespace hyb {

namespace {

using namespace pipe;

constexpr int kThreads = 256;
constexpr int kSmemLimit = 232448;
constexpr int kTwoCtas = 78 * 1024;    // at least this much shared memory: no third CTA on an SM

struct SplitArgs {
    // Q [panel][request][token][head][64], a box of G heads x 128 / G tokens; K, V the same
    // with one head x Bp tokens (token dimension B: rows beyond it are zero-filled); W
    // [Hkv*d][F], boxes of 64 columns (zero beyond F)
    CUtensorMap tmQ, tmK, tmV, tmW;
    const float *alpha;
    void *const *states;
    bf16 *O;
    unsigned *err;
    int B, Bp, Hq, Hkv, G, d, F, tiles;
    float inv_sqrt_d;
    uint32_t off_w, off_k, off_phi, off_s, off_v, off_z, off_x, off_bar;
    uint32_t tmem_cols, d_col;
};

struct SplitLayout {
    uint32_t off_w, off_k, off_phi, off_s, off_v, off_z, off_x, off_bar, bytes, tmem_cols, d_col;
};

// Shared memory: phase one [Q | W | K], then P's two parts, then [phi_h | phi_l | S_h | S_l]
// in the same space; V, z, statistics, barriers beside it.
SplitLayout make_split_layout(int d, int F, int Bp)
{
    SplitLayout L{};
    const uint32_t q = (uint32_t)(d / 64) * 128 * 128, w = (uint32_t)((F + 63) / 64) * d * 128;
    const uint32_t kv = (uint32_t)(d / 64) * Bp * 128;
    L.off_w = q;
    L.off_k = q + w;
    L.off_phi = 0;
    L.off_s = 2 * 128 * 128;
    const uint32_t ph1 = q + w + kv, pbytes = 2u * 128 * Bp * 2, ph2 = L.off_s + 2u * d * 128;
    uint32_t off = ph1 > ph2 ? ph1 : ph2;
    if (pbytes > off) off = pbytes;
    off = (off + 1023) & ~1023u;
    L.off_v = off; off += kv;
    L.off_z = off; off += (2u * F * 4 + 127) & ~127u;
    L.off_x = off; off += 8u * 256 * 4;
    L.off_bar = off; off += 64;
    L.bytes = off + 1024;
    if (L.bytes < (uint32_t)kTwoCtas) L.bytes = kTwoCtas;
    L.d_col = F <= 64 ? 64 : (uint32_t)F;
    L.tmem_cols = L.d_col + 128 <= 256 ? 256 : 512;
    return L;
}

// x cut to a tf32 value (the low 13 bits dropped), and the rest, itself cut by the MMA
__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

__global__ void __launch_bounds__(kThreads, 2) k_attn_split(const __grid_constant__ SplitArgs a)
{
    using namespace ptx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d, F = a.F, B = a.B, Bp = a.Bp, G = a.G;
    const int unit = blockIdx.x / a.tiles, tile = blockIdx.x % a.tiles;
    const int r = unit / a.Hkv, g = unit % a.Hkv;
    const int t0 = tile * (128 / G);                      // first token of the item
    const int rows = min(128, (B - t0) * G);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + a.off_bar);
    uint64_t *bar_ld = bars, *bar_v = bars + 1, *bar_u = bars + 2, *bar_m = bars + 3;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + 4);
    volatile int *fail = reinterpret_cast<volatile int *>(tmem_holder + 1);
    float *zs = reinterpret_cast<float *>(smem + a.off_z);
    float *ex = reinterpret_cast<float *>(smem + a.off_x);   // [8 statistics][2 parts][128]

    if (tid == 0) {
        prefetch_tensormap(&a.tmQ);
        prefetch_tensormap(&a.tmW);
        prefetch_tensormap(&a.tmK);
        prefetch_tensormap(&a.tmV);
        for (int i = 0; i < 4; ++i) mbar_init(&bars[i], 1);
        *fail = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(tmem_holder, a.tmem_cols);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    if (tid == 0) griddep_launch_dependents();
    griddep_wait();
    const uint32_t tmem = *tmem_holder;
    const float *state = reinterpret_cast<const float *>(a.states[r]);
    const bool usable = state_ptr_ok(state);
    if (!usable && tid == 0 && tile == 0) raise_error(a.err, ERR_BAD_STATE_PTR);
    bool bad = false;
    if (usable) {
        const float *Sg = state + (size_t)g * head_floats(d, F);
        const uint32_t kvb = (uint32_t)(d / 64) * Bp * 128;
        const int wp = (F + 63) / 64;
        if (tid == 0) {
            mbar_arrive_expect_tx(bar_ld, (uint32_t)(d / 64) * (128 * 128) + (uint32_t)wp * d * 128 + kvb);
            tma_load_5d(smem, &a.tmQ, 0, g * G, t0, r, 0, bar_ld);
            for (int p = 0; p < wp; ++p) tma_load_2d(smem + a.off_w + p * d * 128, &a.tmW, 64 * p, g * d, bar_ld);
            tma_load_5d(smem + a.off_k, &a.tmK, 0, g, 0, r, 0, bar_ld);
            mbar_arrive_expect_tx(bar_v, kvb);
            tma_load_5d(smem + a.off_v, &a.tmV, 0, g, 0, r, 0, bar_v);
        }
        for (int i = tid; i < 2 * F; i += kThreads) zs[i] = __ldg(Sg + (size_t)2 * F * d + i);
        // the first state tile, on its way while U is formed
        const int NS4 = d * 8 / kThreads;   // float4 of a state tile per thread (2 or 4)
        const float4 *sp4 = reinterpret_cast<const float4 *>(Sg);
        float4 sreg[4];
        auto load_s = [&](int t) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < NS4) sreg[i] = __ldg(sp4 + (size_t)t * 8 * d + i * kThreads + tid);
        };
        load_s(0);

        // ---- U = Q W and the scores
        const uint32_t s_u = smem_u32(smem);
        if (tid == 0) {
            bad = !wait_bar(bar_ld, 0, fail);
            if (!bad) {
                tc_fence_after();
                const uint32_t idU = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, F < 64 ? 64 : F);
                const uint32_t idS = instr_desc(FMT_BF16, FMT_BF16, false, false, 128, Bp);
                for (int k = 0; k < d / 16; ++k) {
                    const uint64_t aq = smem_desc(s_u + (k >> 2) * (128 * 128) + (k & 3) * 32, 16, 1024, SWZ_128B);
                    mma_bf16_ss(tmem, aq, smem_desc(s_u + a.off_w + 2 * k * 1024, d * 128, 1024, SWZ_128B), idU, k > 0);
                    mma_bf16_ss(tmem + a.d_col, aq,
                                smem_desc(s_u + a.off_k + (k >> 2) * (Bp * 128) + (k & 3) * 32, 16, 1024, SWZ_128B), idS,
                                k > 0);
                }
                mma_commit(bar_u);
            }
        }
        __syncwarp();
        bad = !wait_bar(bar_u, 0, fail) || bad;
        tc_fence_after();

        // ---- row statistics: two threads per row, every other 16-column chunk each
        const int q4 = warp & 3, part = warp >> 2;
        const int row = 32 * q4 + lane;
        const uint32_t lane_off = (uint32_t)(32 * q4) << 16;
        const uint32_t ucol = tmem + lane_off, dcol = tmem + a.d_col + lane_off;
        const bool valid = row < rows;
        const float alpha_row = valid ? a.alpha[g * G + row % G] : 0.f;
        const float scale_l2 = a.inv_sqrt_d * kLog2e;
        const int nu = F / 16, ns = Bp / 16;
        auto X = [&](int k, int p) -> float & { return ex[(k * 2 + p) * 128 + row]; };
        const uint32_t pair_bar = 1 + q4;
        float ms = -INFINITY, mx = -INFINITY, mn = INFINITY;
        for (int c = part; c < ns; c += 2) {
            float v[16];
            tmem_ld16(dcol + 16 * c, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) ms = fmaxf(ms, 16 * c + i < B ? v[i] : -INFINITY);
        }
        for (int c = part; c < nu; c += 2) {
            float v[16];
            tmem_ld16(ucol + 16 * c, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                mx = fmaxf(mx, v[i]);
                mn = fminf(mn, v[i]);
            }
        }
        X(0, part) = ms;
        X(1, part) = mx;
        X(2, part) = mn;
        bad = group_sync_failed(pair_bar, 64, bad);
        ms = fmaxf(X(0, 0), X(0, 1));
        mx = fmaxf(X(1, 0), X(1, 1));
        mn = fminf(X(2, 0), X(2, 1));
        __syncthreads();   // z is in place
        const float msl = ms * scale_l2, mxl = mx * kLog2e, mnl = mn * kLog2e;
        {
            float l = 0.f, sp = 0.f, sn = 0.f, lp = 0.f, ln = 0.f;
            for (int c = part; c < ns; c += 2) {
                float v[16];
                tmem_ld16(dcol + 16 * c, v);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) l += 16 * c + i < B ? ex2(fmaf(v[i], scale_l2, -msl)) : 0.f;
            }
            for (int c = part; c < nu; c += 2) {
                float v[16];
                tmem_ld16(ucol + 16 * c, v);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float ep = ex2(fmaf(v[i], kLog2e, -mxl)), en = ex2(fmaf(-v[i], kLog2e, mnl));
                    sp += ep;
                    sn += en;
                    lp = fmaf(ep, zs[16 * c + i], lp);
                    ln = fmaf(en, zs[F + 16 * c + i], ln);
                }
            }
            X(3, part) = l;
            X(4, part) = sp;
            X(5, part) = sn;
            X(6, part) = lp;
            X(7, part) = ln;
        }
        bad = group_sync_failed(pair_bar, 64, bad);
        const float isp = 1.f / (X(4, 0) + X(4, 1)), isn = 1.f / (X(5, 0) + X(5, 1));
        const float ld = (X(6, 0) + X(6, 1)) * isp + (X(7, 0) + X(7, 1)) * isn;
        MergeWeights mw{0.f, 0.f};
        if (valid) mw = merge_weights(log_sigmoid(alpha_row), ms * a.inv_sqrt_d, X(3, 0) + X(3, 1), ld);
        const float cp = isp * mw.wl, cn = isn * mw.wl;

        // ---- P (times its merge weight) as two bf16 parts, K-major without swizzle (core
        // matrices of 8 rows x 16 bytes), over Q and W, which the products have read
        {
            uint8_t *prow = smem + (row >> 3) * (Bp / 8) * 128 + (row & 7) * 16;
            const uint32_t pstride = 128u * Bp * 2;
            for (int c = part; c < ns; c += 2) {
                float v[16];
                tmem_ld16(dcol + 16 * c, v);
                tmem_wait_ld();
                uint32_t h[8], l[8];
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    const float p0 = 16 * c + i < B ? ex2(fmaf(v[i], scale_l2, -msl)) * mw.ws : 0.f;
                    const float p1 = 16 * c + i + 1 < B ? ex2(fmaf(v[i + 1], scale_l2, -msl)) * mw.ws : 0.f;
                    h[i / 2] = pack_bf16x2(p0, p1);
                    l[i / 2] = pack_bf16x2(p0 - __uint_as_float(h[i / 2] << 16), p1 - __uint_as_float(h[i / 2] & 0xFFFF0000u));
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    uint8_t *p = prow + (2 * c + j) * 128;
                    *reinterpret_cast<uint4 *>(p) = make_uint4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
                    *reinterpret_cast<uint4 *>(p + pstride) = make_uint4(l[4 * j], l[4 * j + 1], l[4 * j + 2], l[4 * j + 3]);
                }
            }
        }
        fence_proxy_async_smem();
        tc_fence_before();
        bad = __syncthreads_or(bad) != 0;
        if (tid == 0 && !bad) {
            bad = !wait_bar(bar_v, 0, fail);
            if (!bad) {
                tc_fence_after();
                const uint32_t idP = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, d);
                for (int h = 0; h < 2; ++h)
                    for (int k = 0; k < Bp / 16; ++k)
                        mma_bf16_ss(tmem + a.d_col,
                                    smem_desc(s_u + (uint32_t)h * 128 * Bp * 2 + k * 256, 128, (Bp / 8) * 128, SWZ_NONE),
                                    smem_desc(s_u + a.off_v + 2 * k * 1024, Bp * 128, 1024, SWZ_128B), idP, (h | k) != 0);
                mma_commit(bar_m);
            }
        }
        __syncwarp();

        // ---- readout, one 32-feature tile after the other
        const int NT = 2 * F / 32;
        uint32_t ph = 0;   // products committed on bar_m so far
        for (int t = 0; t < NT; ++t, ++ph) {
            // phi of 16 features: [32 t + 16 part, + 16), one sign throughout
            const int f = 32 * t + 16 * part;
            const bool neg = f >= F;
            float v[16];
            tmem_ld16(ucol + (neg ? f - F : f), v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i)
                v[i] = neg ? ex2(fmaf(-v[i], kLog2e, mnl)) * cn : ex2(fmaf(v[i], kLog2e, -mxl)) * cp;
            // the products in front have read the operands' space
            bad = !wait_bar(bar_m, ph & 1u, fail) || bad;
            uint8_t *prow = smem + a.off_phi + row * 128;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float4 h, l;
                h.x = tf32_hi(v[4 * j]);
                h.y = tf32_hi(v[4 * j + 1]);
                h.z = tf32_hi(v[4 * j + 2]);
                h.w = tf32_hi(v[4 * j + 3]);
                l = make_float4(v[4 * j] - h.x, v[4 * j + 1] - h.y, v[4 * j + 2] - h.z, v[4 * j + 3] - h.w);
                const uint32_t at = (uint32_t)(((4 * part + j) ^ (row & 7)) << 4);
                *reinterpret_cast<float4 *>(prow + at) = h;
                *reinterpret_cast<float4 *>(prow + 128 * 128 + at) = l;
            }
            float4 *sh = reinterpret_cast<float4 *>(smem + a.off_s);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < NS4) {
                    const float4 x = sreg[i];
                    const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
                    sh[i * kThreads + tid] = h;
                    sh[d * 8 + i * kThreads + tid] = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
                }
            if (t + 1 < NT) load_s(t + 1);
            fence_proxy_async_smem();
            bad = __syncthreads_or(bad) != 0;
            if (bad) break;
            if (tid == 0) {
                tc_fence_after();
                const uint32_t idR = instr_desc(FMT_TF32, FMT_TF32, false, false, 128, d);
                const uint32_t ph_u = s_u + a.off_phi, sh_u = s_u + a.off_s;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t ah = smem_desc(ph_u + 32 * kk, 16, 1024, SWZ_128B);
                    const uint64_t al = smem_desc(ph_u + 128 * 128 + 32 * kk, 16, 1024, SWZ_128B);
                    const uint64_t bh = smem_desc(sh_u + 32 * kk, 16, 1024, SWZ_128B);
                    const uint64_t bl = smem_desc(sh_u + d * 128 + 32 * kk, 16, 1024, SWZ_128B);
                    mma_tf32_ss(tmem + a.d_col, al, bh, idR, 1);
                    mma_tf32_ss(tmem + a.d_col, ah, bl, idR, 1);
                    mma_tf32_ss(tmem + a.d_col, ah, bh, idR, 1);
                }
                mma_commit(bar_m);
            }
            __syncwarp();
        }
        // ---- epilogue: D is the output row
        bad = bad || !wait_bar(bar_m, ph & 1u, fail);
        tc_fence_after();
        const int dh = d / 2;
        bf16 *orow = a.O + (((size_t)r * B + t0 + row / G) * a.Hq + g * G + row % G) * d + part * dh;
        for (int c = 0; c < dh; c += 32) {
            float v[32];
            tmem_ld32(dcol + part * dh + c, v);
            tmem_wait_ld();
            if (valid && !bad) {
                uint4 *dst = reinterpret_cast<uint4 *>(orow + c);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    dst[i] = make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                                        pack_bf16x2(v[8 * i + 4], v[8 * i + 5]), pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
            }
        }
        if (tid == 0 && *fail) {
            raise_error(a.err, ERR_WAIT_TIMEOUT);
            // copies and products in flight end before the CTA exits
            mbar_wait(bar_ld, 0, kWaitNs);
            mbar_wait(bar_v, 0, kWaitNs);
            mma_commit(bar_u);
            mbar_wait(bar_u, 1, kWaitNs);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, a.tmem_cols);
    }
}

}  // namespace

bool attn_split_supported(const hybrid_cfg &c)
{
    if (c.io_dtype != HYBRID_BF16) return false;
    const int G = c.n_q_heads / c.n_kv_heads;
    if (G > 128 || 128 % G != 0) return false;   // an item's Q is one box of 128 / G tokens x G heads
    return (int)make_split_layout(c.head_dim, c.feat_dim, (c.block_size + 15) / 16 * 16).bytes <= kSmemLimit;
}

cudaError_t launch_attn_split(const hybrid_cfg &c, const void *Q, const void *K, const void *V, const void *W,
                              const float *alpha, void *const *states, int n_req, void *O, unsigned *err,
                              cudaStream_t st)
{
    SplitArgs a{};
    const int d = c.head_dim, F = c.feat_dim, B = c.block_size, Hq = c.n_q_heads, Hkv = c.n_kv_heads, G = Hq / Hkv;
    const int Bp = (B + 15) / 16 * 16;
    const SplitLayout L = make_split_layout(d, F, Bp);
    {
        const cuuint64_t P = (cuuint64_t)d / 64;
        const cuuint64_t dq[5] = {64, (cuuint64_t)Hq, (cuuint64_t)B, (cuuint64_t)n_req, P};
        const cuuint64_t sq[4] = {(cuuint64_t)d * 2, (cuuint64_t)Hq * d * 2, (cuuint64_t)B * Hq * d * 2, 128};
        const cuuint32_t bq[5] = {64, (cuuint32_t)G, (cuuint32_t)(128 / G), 1, (cuuint32_t)P};
        const cuuint64_t dk[5] = {64, (cuuint64_t)Hkv, (cuuint64_t)B, (cuuint64_t)n_req, P};
        const cuuint64_t sk[4] = {(cuuint64_t)d * 2, (cuuint64_t)Hkv * d * 2, (cuuint64_t)B * Hkv * d * 2, 128};
        const cuuint32_t bk[5] = {64, 1, (cuuint32_t)Bp, 1, (cuuint32_t)P};
        const cuuint64_t dw[2] = {(cuuint64_t)F, (cuuint64_t)Hkv * d};
        const cuuint64_t sw[1] = {(cuuint64_t)F * 2};
        const cuuint32_t bw[2] = {64, (cuuint32_t)d};
        if (!encode_bf16(&a.tmQ, Q, 5, dq, sq, bq) || !encode_bf16(&a.tmK, K, 5, dk, sk, bk) ||
            !encode_bf16(&a.tmV, V, 5, dk, sk, bk) || !encode_bf16(&a.tmW, W, 2, dw, sw, bw))
            return cudaErrorInvalidValue;
    }
    a.alpha = alpha;
    a.states = states;
    a.O = static_cast<bf16 *>(O);
    a.err = err;
    a.B = B;
    a.Bp = Bp;
    a.Hq = Hq;
    a.Hkv = Hkv;
    a.G = G;
    a.d = d;
    a.F = F;
    a.tiles = (G * B + 127) / 128;
    a.inv_sqrt_d = 1.f / sqrtf((float)d);
    a.off_w = L.off_w;
    a.off_k = L.off_k;
    a.off_phi = L.off_phi;
    a.off_s = L.off_s;
    a.off_v = L.off_v;
    a.off_z = L.off_z;
    a.off_x = L.off_x;
    a.off_bar = L.off_bar;
    a.tmem_cols = L.tmem_cols;
    a.d_col = L.d_col;
    static std::atomic<unsigned long long> opted{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const unsigned long long bit = 1ull << dev;
    if (!(opted.load(std::memory_order_acquire) & bit)) {
        const cudaError_t e = cudaFuncSetAttribute(k_attn_split, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e != cudaSuccess) return e;
        opted.fetch_or(bit, std::memory_order_release);
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((long long)n_req * Hkv * a.tiles));
    lc.blockDim = dim3(kThreads);
    // up to a CTA per SM: ask for the SM's shared memory, or the block scheduler puts two on
    // one SM while others idle (8 requests, 16 heads, B = 24: 22.9 -> 15.9 us)
    const uint32_t one = 118 * 1024;
    lc.dynamicSmemBytes = (int)lc.gridDim.x <= sm_count() && L.bytes < one ? one : L.bytes;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, k_attn_split, a);
}

}  // namespace hyb
