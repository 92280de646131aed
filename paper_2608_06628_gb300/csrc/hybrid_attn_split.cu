// hybrid_attn_split.cu -- the block-hybrid step of Section 3.1 for the bf16 shapes that the
// streaming tensor-core kernels do not take (more than 128 query rows to a state, B not a
// multiple of 16, F < 64), on the tensor cores at float32 accuracy.
//
// These shapes ran float32 FMA kernels and keep that accuracy: bf16 products (U = Q W and
// the scores) are exact in float32, and every float32 operand of the other products goes in
// as a sum of parts,
//   phi S = phi_h S_h + phi_l S_h + phi_h S_l   tf32 parts, x_h = x rounded to 11 bits and
//                                               x_l the rest, itself cut: 2^-22 of a term
//   P V   = P_h V + P_m V + P_l V               bf16 parts of e^(s - m), 8 bits each: exact
// so the result differs from the FMA kernels' by less than its own bf16 rounding (2^-9).
// Infinities stay what the whole product makes of them, not inf - inf or 0 inf: an infinite
// state element is all in S_l, which only phi_h multiplies, and the parts of a P > 0 are cut,
// not rounded, and all positive.
//
// A work item is 128 of a unit's G B query rows (row t G + h, whole tokens).  One persistent
// CTA per SM walks a contiguous range of items; 18 warps:
//   warps 0-7    rows, two threads each: extrema, sums, merge weights, P; per 32-feature tile
//                phi's parts from U into Tensor Memory; the output rows
//   warps 8-15   the parts of the state tiles into shared memory, through registers, kAhead
//                tiles ahead (a load takes longer than a tile's products), and from the next
//                item on while the rows are still at this one
//   warp 16      MMA issuer.  S_h and S_l are neighbours and so are the accumulators D and D2,
//                so phi_h takes both in one product of N = 2 d: 8 MMAs per tile instead of 12
//                (F = 256 has no room for D2 and issues 12).  D2 takes every low product, so
//                that their additions round nothing off D
//   warp 17      TMA of an item's Q, W, K, V and z, the next item's during the readout
// Tensor Memory: [U (64, 128 or 256 columns) | D | D2 | two buffers of phi_h, phi_l], the
// scores in the phi buffers' columns until P is written.
//
// What bounds it: one item takes 12.5 us with d = F = 128, 1.2 for its loads, 3.3 from U to P
// (chains of Tensor Memory loads, exponentials and row exchanges), 0.65 per tile (tensor pipe
// 0.45) and 1.3 for the output.  16 : 4 heads, d = F = 128, B = 64: 14.4 us for one request,
// 29.9 for 32; 20.5 and 196 on the CUDA cores (F = 256: 22.6 and 47, against 31.6 and 328).
// Relative error against 64 bits 1.65751e-3 on both, the rounding of a bf16 output; outputs that
// are not the nearest bf16 value 0.037 % (F = 256, keys x 8: 0.031) against 0.021 (0.030) on the
// CUDA cores.  P as two rounded parts took 13.8 and 28.6 us, with 0.25 % and NaN for infinities.
// Two smaller CTAs per SM with single buffers took 2.4 and 1.9 us more (F = 256: 4.7 and 10).
#include <atomic>

#include "hybrid_common.cuh"
#include "hybrid_tc.h"
#include "tc_pipeline.cuh"

namespace hyb {

namespace {

using namespace pipe;

constexpr int kRowWarps = 8, kTileWarps = 8, kIssuer = kRowWarps + kTileWarps;
constexpr int kAhead = 3;              // state tiles loaded ahead
constexpr int kThreads = (kIssuer + 2) * 32;
constexpr int kSmemLimit = 232448;

struct SplitArgs {
    // Q [panel][request][token][head][64], a box of G heads x 128 / G tokens; K, V the same
    // with one head x Bp tokens (token dimension B: rows beyond it are zero-filled); W
    // [Hkv*d][F], boxes of 64 columns (zero beyond F)
    CUtensorMap tmQ, tmK, tmV, tmW;
    const float *alpha;
    void *const *states;
    bf16 *O;
    unsigned *err;
    int B, Bp, Hq, Hkv, G, d, F, tiles, n_items;
    int lbuf;                          // log2 of the buffers of a tile's operands
    float inv_sqrt_d;
    uint32_t off_w, off_k, off_s, off_v, off_z, off_x, off_bar;
    uint32_t d_col, a_col;             // Tensor Memory columns of D (then D2) and of the phi buffers
};

struct SplitLayout {
    uint32_t off_w, off_k, off_s, off_v, off_z, off_x, off_bar, bytes;
    int nbuf;
};

// Shared memory: [Q | W | K, then P's three parts][S_h | S_l x nbuf][V][z x 2][statistics]
// [barriers].  Only F = 256 with B > 112 and d = 128 has no room for a second tile buffer.
SplitLayout make_split_layout(int d, int F, int Bp)
{
    SplitLayout L{};
    const uint32_t q = (uint32_t)(d / 64) * 128 * 128, w = (uint32_t)((F + 63) / 64) * d * 128;
    const uint32_t kv = (uint32_t)(d / 64) * Bp * 128, pbytes = 3u * 128 * Bp * 2;
    for (L.nbuf = 2; L.nbuf >= 1; --L.nbuf) {
        uint32_t off = q + w + kv > pbytes ? q + w + kv : pbytes;
        L.off_w = q;
        L.off_k = q + w;
        L.off_s = off; off += (uint32_t)L.nbuf * 2 * d * 128;
        L.off_v = off; off += kv;
        L.off_z = off; off += 2 * ((2u * F * 4 + 127) & ~127u);
        L.off_x = off; off += 8u * 2 * 128 * 4;
        L.off_bar = off; off += 256;
        L.bytes = off + 1024;
        if (L.bytes <= (uint32_t)kSmemLimit) break;
    }
    if (L.bytes < 118 * 1024) L.bytes = 118 * 1024;   // one CTA per SM (Tensor Memory)
    return L;
}

// x rounded to a tf32 value (cvt.rna.tf32 issues at a fraction of the rate of the two)
__device__ __forceinline__ float tf32_rna(float x)
{
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}
// A thread's granules (stride apart, n of them) of a state tile's parts with an infinite high part
// among them: that one becomes 0 and the low part all of the element.
__device__ __noinline__ void split_infinities(float4 *hi, int low, int stride, int n)
{
    for (int j = 0; j < n; ++j) {
        float *h = reinterpret_cast<float *>(hi + j * stride), *l = reinterpret_cast<float *>(hi + low + j * stride);
        for (int k = 0; k < 4; ++k)
            if (fabsf(h[k]) == INFINITY) {
                // (rounded to an infinity, the element itself is finite)
                l[k] = isnan(l[k]) ? h[k] : copysignf(3.4e38f, h[k]);
                h[k] = 0.f;
            }
    }
}

// kTwo (F <= 128): two accumulators
template <bool kTwo>
__global__ void __launch_bounds__(kThreads, 1) k_attn_split(const __grid_constant__ SplitArgs a)
{
    using namespace ptx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d, F = a.F, B = a.B, Bp = a.Bp, G = a.G;
    const int NT = 2 * F / 32;                            // state tiles of an item
    const int per = a.n_items / (int)gridDim.x, rem = a.n_items % (int)gridDim.x;
    const int i_begin = (int)blockIdx.x * per + min((int)blockIdx.x, rem);
    const int i_end = i_begin + per + ((int)blockIdx.x < rem ? 1 : 0);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + a.off_bar);
    uint64_t *ldfull = bars;           // Q, W, K and z have landed
    uint64_t *vfull = bars + 1;
    uint64_t *uready = bars + 2;       // U and the scores are formed
    uint64_t *pready = bars + 3;       // rows -> issuer: P is written
    uint64_t *pvdone = bars + 4;       // P V is complete: Q, W, K, P and V space may be reloaded
    uint64_t *opr = bars + 5;          // [2] rows -> issuer: phi's and the state tile's parts
    uint64_t *rdone = bars + 7;        // [2] a tile's products are complete
    uint64_t *ddone = bars + 9;        // the item's products are complete
    uint64_t *dfree = bars + 10;       // rows -> issuer: D has been read
    uint64_t *mmadone = bars + 11;
    constexpr int n_bars = 12;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + n_bars);
    volatile int *fail = reinterpret_cast<volatile int *>(tmem_holder + 1);
    const int zstride = (int)((2u * F * 4 + 127) & ~127u) / 4;
    float *zbuf = reinterpret_cast<float *>(smem + a.off_z);

    if (tid == 0) {
        prefetch_tensormap(&a.tmQ);
        prefetch_tensormap(&a.tmW);
        prefetch_tensormap(&a.tmK);
        prefetch_tensormap(&a.tmV);
        mbar_init_n(ldfull, 3, 1);   // vfull, uready
        mbar_init_n(pready, 1, kRowWarps);
        mbar_init_n(pvdone, 1, 1);
        mbar_init_n(opr, 2, kRowWarps + kTileWarps);
        mbar_init_n(rdone, 3, 1);    // ddone
        mbar_init_n(dfree, 1, kRowWarps);
        mbar_init_n(mmadone, 1, 1);
        *fail = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(tmem_holder, 512);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    if (tid == 0) griddep_launch_dependents();
    griddep_wait();
    const uint32_t tmem = *tmem_holder;
    const uint32_t s_u = smem_u32(smem);
    // item i: rows of tile i % tiles of unit i / tiles
    auto item_state = [&](int i) -> const float * {
        const int u = i / a.tiles;
        const float *st = reinterpret_cast<const float *>(a.states[u / a.Hkv]);
        return state_ptr_ok(st) ? st + (size_t)(u % a.Hkv) * head_floats(d, F) : nullptr;
    };

    if (warp == kIssuer + 1) {
        // ------------------------------------------------------------- producer
        if (lane == 0) {
            const uint32_t kvb = (uint32_t)(d / 64) * Bp * 128;
            const int wp = (F + 63) / 64;
            uint32_t k = 0;
            for (int i = i_begin; i < i_end; ++i) {
                const float *Sg = item_state(i);
                if (!Sg) continue;
                const int u = i / a.tiles, r = u / a.Hkv, g = u % a.Hkv;
                if (k > 0 && !wait_bar(pvdone, (k - 1) & 1u, fail)) break;
                mbar_arrive_expect_tx(ldfull, (uint32_t)(d / 64) * (128 * 128) + (uint32_t)wp * d * 128 + kvb + 2 * F * 4);
                tma_load_5d(smem, &a.tmQ, 0, g * G, (i % a.tiles) * (128 / G), r, 0, ldfull);
                for (int p = 0; p < wp; ++p) tma_load_2d(smem + a.off_w + p * d * 128, &a.tmW, 64 * p, g * d, ldfull);
                tma_load_5d(smem + a.off_k, &a.tmK, 0, g, 0, r, 0, ldfull);
                bulk_g2s(zbuf + (k & 1) * zstride, Sg + (size_t)2 * F * d, 2 * F * 4, ldfull);
                mbar_arrive_expect_tx(vfull, kvb);
                tma_load_5d(smem + a.off_v, &a.tmV, 0, g, 0, r, 0, vfull);
                ++k;
            }
            if (*fail && k) {
                mbar_wait(ldfull, (k - 1) & 1u, kWaitNs);
                mbar_wait(vfull, (k - 1) & 1u, kWaitNs);
            }
        }
    } else if (warp == kIssuer) {
        // ------------------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint32_t idU = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, F < 64 ? 64 : F);
            const uint32_t idS = instr_desc(FMT_BF16, FMT_BF16, false, false, 128, Bp);
            const uint32_t idP = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, d);
            const uint32_t idR = instr_desc(FMT_TF32, FMT_TF32, false, false, 128, d);
            const uint32_t idR2 = instr_desc(FMT_TF32, FMT_TF32, false, false, 128, 2 * d);
            const uint32_t dcol = tmem + a.d_col, d2col = kTwo ? dcol + d : dcol;
            uint32_t k = 0, T = 0;
            bool ok = true;
            for (int i = i_begin; i < i_end && ok; ++i) {
                if (!item_state(i)) continue;
                if (!wait_bar(ldfull, k & 1u, fail)) break;
                // (the scores take the phi buffers, whose readers precede in issue order)
                tc_fence_after();
                for (int kk = 0; kk < d / 16; ++kk) {
                    const uint64_t aq = smem_desc(s_u + (kk >> 2) * (128 * 128) + (kk & 3) * 32, 16, 1024, SWZ_128B);
                    mma_bf16_ss(tmem, aq, smem_desc(s_u + a.off_w + 2 * kk * 1024, d * 128, 1024, SWZ_128B), idU, kk > 0);
                    mma_bf16_ss(tmem + a.a_col, aq,
                                smem_desc(s_u + a.off_k + (kk >> 2) * (Bp * 128) + (kk & 3) * 32, 16, 1024, SWZ_128B), idS,
                                kk > 0);
                }
                mma_commit(uready);
                if (!wait_bar(pready, k & 1u, fail) || !wait_bar(vfull, k & 1u, fail)) break;
                if (k > 0 && !wait_bar(dfree, (k - 1) & 1u, fail)) break;
                tc_fence_after();
                // P_h V initialises D, P_m V initialises D2
                for (int h = 0; h < 3; ++h)
                    for (int kk = 0; kk < Bp / 16; ++kk)
                        mma_bf16_ss(h ? d2col : dcol,
                                    smem_desc(s_u + (uint32_t)h * 128 * Bp * 2 + kk * 256, 128, (Bp / 8) * 128, SWZ_NONE),
                                    smem_desc(s_u + a.off_v + 2 * kk * 1024, Bp * 128, 1024, SWZ_128B), idP,
                                    kTwo ? h == 2 || kk != 0 : (h | kk) != 0);
                mma_commit(pvdone);
                for (int t = 0; t < NT; ++t, ++T) {
                    const uint32_t b = T & a.lbuf;
                    if (!wait_bar(&opr[b], (T >> a.lbuf) & 1u, fail)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t ah = tmem + a.a_col + b * 64, al = ah + 32;
                    const uint32_t sh_u = s_u + a.off_s + b * (uint32_t)(2 * d * 128);
                    // S_h and S_l are neighbours: with D2 beside D, phi_h takes both in one product
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint64_t bh = smem_desc(sh_u + 32 * kk, 16, 1024, SWZ_128B);
                        mma_tf32_ts(d2col, al + 8 * kk, bh, idR, 1);
                        if (kTwo) {
                            mma_tf32_ts(dcol, ah + 8 * kk, bh, idR2, 1);
                        } else {
                            mma_tf32_ts(dcol, ah + 8 * kk, smem_desc(sh_u + d * 128 + 32 * kk, 16, 1024, SWZ_128B), idR, 1);
                            mma_tf32_ts(dcol, ah + 8 * kk, bh, idR, 1);
                        }
                    }
                    mma_commit(&rdone[b]);
                }
                if (!ok) break;
                mma_commit(ddone);
                ++k;
            }
            mma_commit(mmadone);
            mbar_wait(mmadone, 0, kWaitNs);
        }
    } else if (warp >= kRowWarps) {
        // ------------------------------------------------------- state tiles
        const int st_tid = tid - kRowWarps * 32, NS4 = d * 8 / (kTileWarps * 32);
        // kAhead tiles on their way: a load takes longer than a tile's products.  (Plain loads: the
        // state may be a running kernel's output when this one starts, so it is not read-only
        // for the kernel's lifetime, as __ldg asks)
        float4 sreg[kAhead][4];
        auto load_s = [&](float4 (&x)[4], const float *Sg, int t) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < NS4)
                    x[i] = reinterpret_cast<const float4 *>(Sg)[(size_t)t * 8 * d + i * (kTileWarps * 32) + st_tid];
        };
        uint32_t T = 0;
        bool bad = false;
        for (int i = i_begin; i < i_end && !bad; ++i) {
            const float *Sg = item_state(i);
            if (!Sg) continue;
#pragma unroll
            for (int t = 0; t < kAhead; ++t)
                if (t < NT) load_s(sreg[t], Sg, t);
            for (int tb = 0; tb < NT; tb += kAhead) {
#pragma unroll
                for (int q = 0; q < kAhead; ++q) {
                    const int t = tb + q;
                    if (t >= NT) break;
                    const uint32_t b = (T + t) & a.lbuf, use = (T + t) >> a.lbuf;
                    if (use > 0) bad = !wait_bar(&rdone[b], (use - 1) & 1u, fail) || bad;
                    float4 *sh = reinterpret_cast<float4 *>(smem + a.off_s + (size_t)b * (2 * d * 128));
                    float top = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (j < NS4) {
                            const float4 x = sreg[q][j];
                            const float4 h = make_float4(tf32_rna(x.x), tf32_rna(x.y), tf32_rna(x.z), tf32_rna(x.w));
                            sh[j * (kTileWarps * 32) + st_tid] = h;
                            sh[d * 8 + j * (kTileWarps * 32) + st_tid] =
                                make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
                            // (fmaxf passes NaN by; the low part of one is NaN whatever the high part)
                            top = fmaxf(fmaxf(top, fmaxf(fabsf(h.x), fabsf(h.y))), fmaxf(fabsf(h.z), fabsf(h.w)));
                        }
                    if (top == INFINITY) split_infinities(sh + st_tid, d * 8, kTileWarps * 32, NS4);
                    if (t + kAhead < NT) load_s(sreg[q], Sg, t + kAhead);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && !bad) mbar_arrive(&opr[b]);
                }
            }
            T += NT;
        }
    } else {
        // ------------------------------------------------------------- rows
        const int q4 = warp & 3, part = warp >> 2;
        const int row = 32 * q4 + lane;
        const uint32_t lane_off = (uint32_t)(32 * q4) << 16;
        const uint32_t ucol = tmem + lane_off, scol = tmem + a.a_col + lane_off;
        const float scale_l2 = a.inv_sqrt_d * kLog2e;
        const int nu = F / 16, ns = Bp / 16;
        float *xrow = reinterpret_cast<float *>(smem + a.off_x) + row;   // [8 statistics][2 parts][128]
        auto X = [&](int k, int p) -> float & { return xrow[(k * 2 + p) * 128]; };
        auto pair_failed = [&](bool f) -> bool { return group_sync_failed(1 + q4, 64, f); };
        uint32_t k = 0, T = 0;
        for (int i = i_begin; i < i_end; ++i) {
            const float *Sg = item_state(i);
            if (!Sg) {
                if (tid == 0 && i % a.tiles == 0) raise_error(a.err, ERR_BAD_STATE_PTR);
                continue;
            }
            const int u = i / a.tiles, r = u / a.Hkv, g = u % a.Hkv, t0 = (i % a.tiles) * (128 / G);
            const bool valid = row < (B - t0) * G;
            // a quarter without rows leaves its lanes of the operands as they are: rows of a
            // product are independent, and these are not stored
            const bool active = 32 * q4 < (B - t0) * G;
            const int nsa = active ? ns : 0, nua = active ? nu : 0;
            // log w of the row's gate, formed while U is
            const float lw = valid ? log_sigmoid(a.alpha[g * G + row % G]) : 0.f;
            // ---- statistics: a part takes every other 16-column chunk
            bool bad = !wait_bar(ldfull, k & 1u, fail);
            bad = !wait_bar(uready, k & 1u, fail) || bad;
            tc_fence_after();
            const float *zs = zbuf + (k & 1) * zstride;
            float ms = -INFINITY, mx = -INFINITY, mn = INFINITY;
            for (int c = part; c < nsa; c += 2) {
                float v[16];
                tmem_ld16(scol + 16 * c, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) ms = fmaxf(ms, 16 * c + j < B ? v[j] : -INFINITY);
            }
            for (int c = part; c < nua; c += 2) {
                float v[16];
                tmem_ld16(ucol + 16 * c, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    mx = fmaxf(mx, v[j]);
                    mn = fminf(mn, v[j]);
                }
            }
            X(0, part) = ms;
            X(1, part) = mx;
            X(2, part) = mn;
            bad = pair_failed(bad);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                ms = fmaxf(ms, X(0, p));
                mx = fmaxf(mx, X(1, p));
                mn = fminf(mn, X(2, p));
            }
            const float msl = ms * scale_l2, mxl = mx * kLog2e, mnl = mn * kLog2e;
            {
                float l = 0.f, sp = 0.f, sn = 0.f, lp = 0.f, ln = 0.f;
                for (int c = part; c < nsa; c += 2) {
                    float v[16];
                    tmem_ld16(scol + 16 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) l += 16 * c + j < B ? ex2(fmaf(v[j], scale_l2, -msl)) : 0.f;
                }
                for (int c = part; c < nua; c += 2) {
                    float v[16];
                    tmem_ld16(ucol + 16 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 p4 = *reinterpret_cast<const float4 *>(zs + 16 * c + 4 * q);
                        const float4 n4 = *reinterpret_cast<const float4 *>(zs + F + 16 * c + 4 * q);
                        const float pz[4] = {p4.x, p4.y, p4.z, p4.w}, nz[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float x = v[4 * q + j];
                            const float ep = ex2(fmaf(x, kLog2e, -mxl)), en = ex2(fmaf(-x, kLog2e, mnl));
                            sp += ep;
                            sn += en;
                            lp = fmaf(ep, pz[j], lp);
                            ln = fmaf(en, nz[j], ln);
                        }
                    }
                }
                X(3, part) = l;
                X(4, part) = sp;
                X(5, part) = sn;
                X(6, part) = lp;
                X(7, part) = ln;
            }
            bad = pair_failed(bad);
            // the merge weights by one part, for both
            if (part == 0 && active) {
                auto total = [&](int q) { return X(q, 0) + X(q, 1); };
                const float isp = 1.f / total(4), isn = 1.f / total(5);
                const float ld = total(6) * isp + total(7) * isn, l = total(3);
                // the weights of merge_weights without its logarithms: e^t l and ld are the
                // branches' masses, both divided by the larger of e^t and 1
                float wsm = 0.f, wl = 0.f;
                if (valid && ld > 0.f) {
                    const float t = lw + ms * a.inv_sqrt_d, e = expf(-fabsf(t));
                    const float inv = 1.f / (t > 0.f ? fmaf(ld, e, l) : fmaf(l, e, ld));
                    wsm = t > 0.f ? inv : e * inv;
                    wl = t > 0.f ? e * inv : inv;
                } else if (valid) {
                    wsm = lw == -INFINITY ? __int_as_float(0x7fc00000) : 1.f / l;   // empty prefix
                }
                X(0, 0) = wsm;
                X(0, 1) = isp * wl;
                X(1, 0) = isn * wl;
            }
            bad = pair_failed(bad);
            const float wsm = X(0, 0), cp = X(0, 1), cn = X(1, 0);

            // ---- P (times its merge weight) as three bf16 parts, K-major without swizzle (core
            // matrices of 8 rows x 16 bytes), over Q, W and K, which the products have read
            {
                uint8_t *prow = smem + (row >> 3) * (Bp / 8) * 128 + (row & 7) * 16;
                const uint32_t pstride = 128u * Bp * 2;
                for (int c = part; c < nsa; c += 2) {
                    float v[16];
                    tmem_ld16(scol + 16 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        uint32_t q[3][4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float h[2], m[2], l[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const int k = 8 * j + 2 * i + e;
                                const float p = 16 * c + k < B ? ex2(fmaf(v[k], scale_l2, -msl)) * wsm : 0.f;
                                h[e] = bf16_hi(p);
                                const float rest = positive_rest(p, h[e], p);
                                m[e] = bf16_hi(rest);
                                l[e] = positive_rest(rest, m[e], rest);
                            }
                            q[0][i] = bf16_pair(h[0], h[1]);
                            q[1][i] = bf16_pair(m[0], m[1]);
                            q[2][i] = bf16_pair(l[0], l[1]);
                        }
#pragma unroll
                        for (int e = 0; e < 3; ++e)
                            *reinterpret_cast<uint4 *>(prow + e * pstride + (2 * c + j) * 128) =
                                make_uint4(q[e][0], q[e][1], q[e][2], q[e][3]);
                    }
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            // every part has read the row's scores: phi may take their columns
            bad = pair_failed(bad);
            tc_fence_after();
            if (lane == 0 && !bad) mbar_arrive(pready);

            // ---- operands of the readout, one 32-feature tile after the other
            for (int t = 0; t < NT; ++t) {
                const uint32_t b = (T + t) & a.lbuf, use = (T + t) >> a.lbuf;
                // phi of 16 features: [32 t + 16 part, + 16), one sign throughout
                const int f = 32 * t + 16 * part;
                const bool neg = f >= F;
                float v[16], l[16];
                if (active) {
                    tmem_ld16(ucol + (neg ? f - F : f), v);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float x = neg ? ex2(fmaf(-v[j], kLog2e, mnl)) * cn : ex2(fmaf(v[j], kLog2e, -mxl)) * cp;
                        v[j] = tf32_rna(x);
                        l[j] = x - v[j];
                    }
                }
                if (use > 0) bad = !wait_bar(&rdone[b], (use - 1) & 1u, fail) || bad;
                if (active) {
                    tc_fence_after();
                    tmem_st16(scol + b * 64 + 16 * part, v);
                    tmem_st16(scol + b * 64 + 32 + 16 * part, l);
                    tmem_wait_st();
                    tc_fence_before();
                }
                __syncwarp();
                if (lane == 0 && !bad) mbar_arrive(&opr[b]);
            }
            T += NT;
            // ---- epilogue: D (+ D2) is the output row, d / 2 columns per part
            bad = !wait_bar(ddone, k & 1u, fail) || bad;
            tc_fence_after();
            const int dq = d / 2;
            uint4 *dst = reinterpret_cast<uint4 *>(a.O + (((size_t)r * B + t0 + row / G) * a.Hq + g * G + row % G) * d + part * dq);
            if (!active) {
                if (lane == 0 && !bad) mbar_arrive(dfree);
            } else
            for (int c = 0; c < dq; c += 16) {
                float v[16], w[16];
                tmem_ld16(tmem + lane_off + a.d_col + part * dq + c, v);
                if constexpr (kTwo) tmem_ld16(tmem + lane_off + a.d_col + d + part * dq + c, w);
                tmem_wait_ld();
                if (c + 16 >= dq) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0 && !bad) mbar_arrive(dfree);
                }
                if constexpr (kTwo)
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] += w[j];
                if (valid && !bad)
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        dst[c / 8 + j] = make_uint4(pack_bf16x2(v[8 * j], v[8 * j + 1]), pack_bf16x2(v[8 * j + 2], v[8 * j + 3]),
                                                    pack_bf16x2(v[8 * j + 4], v[8 * j + 5]), pack_bf16x2(v[8 * j + 6], v[8 * j + 7]));
            }
            // (after a failure the item runs to its end without arrivals, so that the two
            // warps of a quarter leave together)
            if (pair_failed(bad)) break;
            ++k;
        }
        if (tid == 0 && *fail) raise_error(a.err, ERR_WAIT_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
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
    a.n_items = n_req * Hkv * a.tiles;
    a.lbuf = L.nbuf - 1;
    const bool two = F <= 128;
    a.inv_sqrt_d = 1.f / sqrtf((float)d);
    a.off_w = L.off_w;
    a.off_k = L.off_k;
    a.off_s = L.off_s;
    a.off_v = L.off_v;
    a.off_z = L.off_z;
    a.off_x = L.off_x;
    a.off_bar = L.off_bar;
    a.d_col = F <= 64 ? 64 : (uint32_t)F;
    a.a_col = a.d_col + (two ? 256 : 128);
    static std::atomic<unsigned long long> opted{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const unsigned long long bit = 1ull << dev;
    if (!(opted.load(std::memory_order_acquire) & bit)) {
        const cudaError_t e = cudaFuncSetAttribute(k_attn_split<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e != cudaSuccess) return e;
        const cudaError_t e1 = cudaFuncSetAttribute(k_attn_split<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e1 != cudaSuccess) return e1;
        opted.fetch_or(bit, std::memory_order_release);
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(a.n_items < sm_count() ? a.n_items : sm_count());
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = L.bytes;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return two ? cudaLaunchKernelEx(&lc, k_attn_split<true>, a) : cudaLaunchKernelEx(&lc, k_attn_split<false>, a);
}

}  // namespace hyb
