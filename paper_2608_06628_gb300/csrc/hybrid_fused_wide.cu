// hybrid_fused_wide.cu -- the block-hybrid step of Section 3.1 fused with the block commit
// for F = 256: every state tile is read once, used for the readout with the pre-commit
// state, updated with this block's phi(k) v^T and written back.
//
// Work unit = (request r, state head g) with G B <= 64 query rows and B <= 64 keys.  One CTA
// per SM walks a contiguous range of units.  Queries and keys share the feature map: their
// rows form one M = 128 operand (queries on Tensor Memory lanes 0-63, keys on 64-127), so one
// product U = [Q; K] W gives both, and every lane quarter of the math warps has rows to work
// on.  With F = 256, phi = [phi+, phi-] has 512 columns and dS^T as many, far beyond Tensor
// Memory, so the unit goes through it 32 columns of u at a time (a chunk: state tiles phi+ c
// and phi- c).  16 warps:
//   warp 0       ring producer: W of the unit (four ring slots), then the 16 state tiles in
//                chunk order (phi+ c, phi- c), z beside the ring
//   warp 1       MMA issuer (one thread); owns the Tensor Memory allocation
//   warp 2       Q and K, V (TMA)
//   warp 3       storer: bulk stores of the updated tiles and of z
//   warps 4-11   math, two threads per row: extrema and sums of both signs, the merge
//                weights, P; per chunk phi(q) (tf32, into Tensor Memory) and phi(k) (bf16
//                operand [token][32 phi+ | 32 phi-]); the output rows
//   warps 12-15  update: per chunk dS^T from Tensor Memory into the two tiles, in place in
//                their ring slots
// Tensor Memory: [0, 256) U, phi+(q) written over it chunk by chunk; [256, 384) D; [384, 448)
// phi-(q), two buffers; [448, 512) the scores, then dS^T of a chunk (phi+ | phi- columns).
// The merge weights of a row are known before the readout and are folded into phi and P (P as
// two bf16 parts), so D accumulates P V and the readout and is the output.  The parts are
// rounded (2^-18), unless V holds an infinity or NaN (the update warps look, while the math warps
// are at U): a low part that is zero or negative would make NaN of an infinity's product with
// P, so there the high part is cut and the low one positive (2^-17).  As three cut parts, always,
// the 256 requests below took 477 us.
//
// A ring slot holds one state tile (d rows x 128 bytes) or one 64-column panel of W.  W's four
// slots and the 16 tiles take 20 items of a 10-slot ring, so W always lands in slots 0-3, in
// one piece, and its space holds tiles for most of the unit.  P and phi(k) overlay Q and K
// once U and the scores are formed.
//
// What bounds it: HBM (the state in and out), and the start of a unit, whose feature map has
// to be complete before its first tile is done.  256 requests, 16 heads, d = 128, B = 64 (2.43
// GB, 359 us at the measured copy rate): 464 us; as two kernels, which read the state twice
// and update it by reductions at L2, 801 us.
#include <atomic>

#include "hybrid_common.cuh"
#include "hybrid_tc.h"
#include "tc_pipeline.cuh"

namespace hyb {

namespace {

using namespace pipe;

constexpr int kThreads = 512;
constexpr int F = 256, kChunks = F / 32;
constexpr int NS = 10, kW = F / 64;             // ring slots, slots of W
constexpr int kItems = kW + 2 * kChunks;        // ring items per unit
static_assert(kItems % NS == 0, "W stays in slots 0 .. kW - 1");
constexpr int kRows = 64;                       // query rows, and key rows, of a unit at most
constexpr int kSmemLimit = 232448;
constexpr uint32_t cU = 0, cD = 256, cM = 384, cS = 448;   // Tensor Memory columns
constexpr uint32_t kBarPair = 1, kBarKeys = 5;   // named barriers: 1..4 the two warps of a quarter; the key warps

struct WideArgs {
    // Q, K, V with a 64-element panel per copy: [n][B][H][d] boxes of G heads x 64 / G tokens
    // (Q) or one head x 64 tokens (K, V) over a token dimension of B (rows beyond zero-filled);
    // W [Hkv*d][F], all panels in one box
    CUtensorMap tmQ, tmK, tmV, tmW;
    const float *alpha;
    void *const *states;
    bf16 *O;
    unsigned *err;
    int n_units, B, Hq, Hkv, G, d;
    float inv_sqrt_d;
    uint32_t off_x, off_v, off_z, off_st, off_bar;
};

// Shared memory: [ring][X: Q and K rows, then P's parts | phi(k) x 2][V][z x 2 | dz][statistics]
// [barriers].  V always has two panels, so that V^T is an M = 128 operand for d = 64 too.
struct WLayout {
    uint32_t off_x, off_v, off_z, off_st, off_bar, bytes;
};
__host__ __device__ constexpr WLayout wide_layout(int d)
{
    WLayout L{};
    uint32_t off = NS * (uint32_t)d * 128;
    L.off_x = off; off += 2 * 128 * 128;
    L.off_v = off; off += 2 * kRows * 128;
    L.off_z = off; off += 4 * 2 * F * 4;
    L.off_st = off; off += 8 * 2 * 128 * 4;
    L.off_bar = off; off += 512;
    L.bytes = off + 1024;
    if (L.bytes < 118 * 1024) L.bytes = 118 * 1024;
    return L;
}

__device__ __forceinline__ float tf32_rna(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

__device__ __forceinline__ float *wide_state(const WideArgs &a, int u)
{
    float *st = reinterpret_cast<float *>(a.states[u / a.Hkv]);
    if (!state_ptr_ok(st)) return nullptr;
    return st + (size_t)(u % a.Hkv) * head_floats(a.d, F);
}

__global__ void __launch_bounds__(kThreads, 1) k_fused_wide(const __grid_constant__ WideArgs a)
{
    using namespace ptx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d, B = a.B, G = a.G;
    const uint32_t tile_bytes = (uint32_t)d * 128;
    const int per = a.n_units / (int)gridDim.x, rem = a.n_units % (int)gridDim.x;
    const int u_begin = (int)blockIdx.x * per + min((int)blockIdx.x, rem);
    const int u_end = u_begin + per + ((int)blockIdx.x < rem ? 1 : 0);

    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + a.off_bar);
    uint64_t *full = bars;             // [NS] a state tile has landed
    uint64_t *empty = full + NS;       // [NS] the slot may be refilled
    uint64_t *zfull = empty + NS;      // [2]
    uint64_t *zempty = zfull + 2;      // [2]
    uint64_t *phi = zempty + 2;        // [2] math -> issuer: a chunk's phi(q) and phi(k) are written
    uint64_t *rdone = phi + 2;         // [2] a chunk's dS^T and readout products are complete
    uint64_t *wfull = rdone + 2;       // W has landed
    uint64_t *qkfull = wfull + 1;      // Q and K have landed
    uint64_t *vfull = qkfull + 1;
    uint64_t *uready = vfull + 1;      // U and the scores are formed
    uint64_t *pready = uready + 1;     // math -> issuer: P is written
    uint64_t *vscan = pready + 1;      // update -> math: vbad tells whether V is finite
    uint64_t *dsready = vscan + 1;     // dS^T of a chunk is formed
    uint64_t *dsfree = dsready + 1;    // update -> issuer: dS^T has been read
    uint64_t *tready = dsfree + 1;     // [kChunks] update -> storer: a chunk's tiles are updated
    uint64_t *udone = tready + kChunks;   // every product of the unit is complete (D; Q, K and V space)
    uint64_t *dfree = udone + 1;       // math -> issuer: D has been read
    uint64_t *zdone = dfree + 1;       // math -> storer: z is updated
    uint64_t *mmadone = zdone + 1;
    constexpr int n_bars = 2 * NS + 8 + kChunks + 12;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + n_bars);
    volatile int *fail = reinterpret_cast<volatile int *>(tmem_holder + 1);
    int *vbad = reinterpret_cast<int *>(tmem_holder + 2);   // [4] an infinity or NaN in an update warp's part of V

    if (tid == 64) {
        prefetch_tensormap(&a.tmQ);
        prefetch_tensormap(&a.tmK);
        prefetch_tensormap(&a.tmV);
        prefetch_tensormap(&a.tmW);
    }
    if (tid == 0) {
        mbar_init_n(full, 2 * NS + 4, 1);     // empty, zfull, zempty
        mbar_init_n(phi, 2, 8);
        mbar_init_n(rdone, 6, 1);             // wfull, qkfull, vfull, uready
        mbar_init_n(pready, 1, 8);
        mbar_init_n(vscan, 1, 4);
        mbar_init_n(dsready, 1, 1);
        mbar_init_n(dsfree, 1 + kChunks, 4);  // tready
        mbar_init_n(udone, 1, 1);
        mbar_init_n(dfree, 2, 4);             // the query warps; zdone: the key warps
        mbar_init_n(mmadone, 1, 1);
        *fail = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_holder, 512);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    if (tid == 0) griddep_launch_dependents();
    griddep_wait();
    const uint32_t tmem = *tmem_holder;
    uint8_t *xs = smem + a.off_x;
    float *zbuf = reinterpret_cast<float *>(smem + a.off_z);    // [2][2F] z, [2][2F] token sums of phi(k)
    const uint32_t x_u = smem_u32(xs), v_u = smem_u32(smem + a.off_v), ring_u = smem_u32(smem);
    // P's two parts: 64 rows x 64 columns (K-major, no swizzle; the operand's rows 64-127 read
    // what follows and only reach the key lanes of D); then the two phi(k) panels
    constexpr uint32_t kPPart = kRows * kRows * 2, kPhi = 2 * kPPart, kPhiPanel = kRows * 128;
    // item i of a unit sits in slot i % NS; its fill's parity for the unit's index k
    auto full_par = [](int item, uint32_t k) -> uint32_t {
        return item % NS < kW ? (k & 1u) : (item >= NS ? 1u : 0u);
    };

    if (warp == 0) {
        // ------------------------------------------------------- ring producer
        if (lane == 0) {
            uint32_t k = 0;
            // copies issued per barrier, as the parity of their count (bits 0 .. NS - 1 the
            // slots, NS and NS + 1 the z buffers, NS + 2 W), for the drain after a failure
            uint32_t par = 0, any = 0;
            auto issued = [&](int i) {
                par ^= 1u << i;
                any |= 1u << i;
            };
            bool ok = true;
            for (int u = u_begin; u < u_end && ok; ++u) {
                float *Sg = wide_state(a, u);
                if (!Sg) continue;
                const int zb = k & 1;
                if (!wait_bar(&zempty[zb], ((k >> 1) & 1u) ^ 1u, fail)) break;
                mbar_arrive_expect_tx(&zfull[zb], 2 * F * 4);
                bulk_g2s(zbuf + zb * 2 * F, Sg + (size_t)2 * F * d, 2 * F * 4, &zfull[zb]);
                issued(NS + zb);
                // slot s is filled twice a unit: W (or an early tile), then a later tile
                for (int i = 0; i < kW && ok; ++i) ok = wait_bar(&empty[i], 1u, fail);
                if (!ok) break;
                mbar_arrive_expect_tx(wfull, kW * tile_bytes);
                tma_load_3d(smem, &a.tmW, 0, (u % a.Hkv) * d, 0, wfull);
                issued(NS + 2);
                for (int i = 0; i < 2 * kChunks; ++i) {
                    const int item = kW + i, slot = item % NS;
                    if (!wait_bar(&empty[slot], item >= NS ? 0u : 1u, fail)) { ok = false; break; }
                    mbar_arrive_expect_tx(&full[slot], tile_bytes);
                    // chunk i / 2: tile c of phi+, then tile c of phi-
                    bulk_g2s(smem + (size_t)slot * tile_bytes,
                             Sg + (size_t)((i & 1) * kChunks + (i >> 1)) * 32 * d, tile_bytes, &full[slot]);
                    issued(slot);
                }
                ++k;
            }
            if (*fail) {
                // copies in flight land before the CTA exits: the last one of every barrier
                for (int i = 0; i < NS + 3; ++i)
                    if (any >> i & 1u)
                        mbar_wait(i < NS ? &full[i] : i < NS + 2 ? &zfull[i - NS] : wfull, (par >> i & 1u) ^ 1u, kWaitNs);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint32_t idU = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, F);
            const uint32_t idS = instr_desc(FMT_BF16, FMT_BF16, false, false, 128, kRows);
            const uint32_t idP = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, d);
            const uint32_t idDS = instr_desc(FMT_BF16, FMT_BF16, true, true, 128, 64);
            const uint32_t idR = instr_desc(FMT_TF32, FMT_TF32, false, false, 128, d);
            uint32_t k = 0;
            bool ok = true;
            for (int u = u_begin; u < u_end && ok; ++u) {
                if (!wide_state(a, u)) continue;
                if (!wait_bar(qkfull, k & 1u, fail) || !wait_bar(wfull, k & 1u, fail)) break;
                // the scores take dS^T's columns: the previous unit's last chunk has been read
                if (k > 0 && !wait_bar(dsfree, 1u, fail)) break;
                tc_fence_after();
                for (int kk = 0; kk < d / 16; ++kk) {
                    const uint64_t ax = smem_desc(x_u + (kk >> 2) * (128 * 128) + (kk & 3) * 32, 16, 1024, SWZ_128B);
                    mma_bf16_ss(tmem + cU, ax, smem_desc(ring_u + 2 * kk * 1024, tile_bytes, 1024, SWZ_128B), idU, kk > 0);
                    // the keys: rows 64-127 of each panel
                    mma_bf16_ss(tmem + cS, ax,
                                smem_desc(x_u + (kk >> 2) * (128 * 128) + kRows * 128 + (kk & 3) * 32, 16, 1024, SWZ_128B),
                                idS, kk > 0);
                }
                mma_commit(uready);
                for (int i = 0; i < kW; ++i) mma_commit(&empty[i]);
                // P V initialises D once the previous unit's output has been read
                if (!wait_bar(pready, k & 1u, fail) || !wait_bar(vfull, k & 1u, fail)) break;
                if (k > 0 && !wait_bar(dfree, (k - 1) & 1u, fail)) break;
                tc_fence_after();
                for (int h = 0; h < 2; ++h)
                    for (int kk = 0; kk < B / 16; ++kk)
                        mma_bf16_ss(tmem + cD,
                                    smem_desc(x_u + h * kPPart + kk * 256, 128, (kRows / 8) * 128, SWZ_NONE),
                                    smem_desc(v_u + 2 * kk * 1024, kRows * 128, 1024, SWZ_128B), idP, (h | kk) != 0);
                for (int c = 0; c < kChunks; ++c) {
                    const uint32_t b = c & 1;
                    if (!wait_bar(&phi[b], (uint32_t)(c >> 1) & 1u, fail)) { ok = false; break; }
                    // (chunk 0 takes the scores' columns: P is written, so they have been read)
                    if (c > 0 && !wait_bar(dsfree, (uint32_t)(c - 1) & 1u, fail)) { ok = false; break; }
                    tc_fence_after();
                    for (int ks = 0; ks < B / 16; ++ks)
                        mma_bf16_ss(tmem + cS, smem_desc(v_u + ks * 2048, kRows * 128, 1024, SWZ_128B),
                                    smem_desc(x_u + kPhi + b * kPhiPanel + ks * 2048, kRows * 128, 1024, SWZ_128B), idDS,
                                    ks > 0);
                    mma_commit(dsready);
                    for (int h = 0; h < 2 && ok; ++h) {
                        const int item = kW + 2 * c + h, slot = item % NS;
                        if (!wait_bar(&full[slot], full_par(item, k), fail)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t acol = h == 0 ? cU + 32 * c : cM + 32 * b;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_tf32_ts(tmem + cD, tmem + acol + 8 * kk,
                                        smem_desc(ring_u + slot * tile_bytes + 32 * kk, 16, 1024, SWZ_128B), idR, 1);
                    }
                    if (!ok) break;
                    mma_commit(&rdone[b]);
                }
                if (!ok) break;
                mma_commit(udone);
                ++k;
            }
            mma_commit(mmadone);
            mbar_wait(mmadone, 0, kWaitNs);
        }
    } else if (warp == 2) {
        // ------------------------------------------------------- Q, K and V
        if (lane == 0) {
            uint32_t k = 0;
            const uint32_t qk = (uint32_t)(d / 64) * kRows * 128;
            for (int u = u_begin; u < u_end; ++u) {
                if (!wide_state(a, u)) continue;
                const int r = u / a.Hkv, g = u % a.Hkv;
                // their space holds P, phi(k) and V of the previous unit
                if (k > 0 && !wait_bar(udone, (k - 1) & 1u, fail)) break;
                mbar_arrive_expect_tx(qkfull, 2 * qk);
                for (int p = 0; p < d / 64; ++p) {
                    tma_load_4d(xs + p * (128 * 128), &a.tmQ, 64 * p, g * G, 0, r, qkfull);
                    tma_load_4d(xs + p * (128 * 128) + kRows * 128, &a.tmK, 64 * p, g, 0, r, qkfull);
                }
                mbar_arrive_expect_tx(vfull, qk);
                for (int p = 0; p < d / 64; ++p)
                    tma_load_4d(smem + a.off_v + p * kRows * 128, &a.tmV, 64 * p, g, 0, r, vfull);
                ++k;
                // the next unit's rows into L2 while this one runs
                if (u + 1 < u_end)
                    for (int p = 0; p < d / 64; ++p) {
                        const int r1 = (u + 1) / a.Hkv, g1 = (u + 1) % a.Hkv;
                        tma_prefetch_4d(&a.tmQ, 64 * p, g1 * G, 0, r1);
                        tma_prefetch_4d(&a.tmK, 64 * p, g1, 0, r1);
                        tma_prefetch_4d(&a.tmV, 64 * p, g1, 0, r1);
                    }
            }
            if (*fail) {
                if (k) {
                    mbar_wait(qkfull, (k - 1) & 1u, kWaitNs);
                    mbar_wait(vfull, (k - 1) & 1u, kWaitNs);
                }
            }
        }
    } else if (warp == 3) {
        // --------------------------------------------------------------- storer
        if (lane == 0) {
            uint32_t k = 0;
            bool ok = true;
            for (int u = u_begin; u < u_end && ok; ++u) {
                float *Sg = wide_state(a, u);
                if (!Sg) continue;
                for (int c = 0; c < kChunks; ++c) {
                    // (a barrier per chunk: the update warps may be chunks ahead)
                    if (!wait_bar(&tready[c], k & 1u, fail)) { ok = false; break; }
                    for (int h = 0; h < 2; ++h)
                        bulk_s2g(Sg + (size_t)(h * kChunks + c) * 32 * d,
                                 smem + (size_t)((kW + 2 * c + h) % NS) * tile_bytes, tile_bytes);
                    bulk_commit();
                    bulk_wait_read_all();
                    for (int h = 0; h < 2; ++h) mbar_arrive(&empty[(kW + 2 * c + h) % NS]);
                }
                if (!ok) break;
                const int zb = k & 1;
                if (!wait_bar(zdone, k & 1u, fail)) break;
                bulk_s2g(Sg + (size_t)2 * F * d, zbuf + zb * 2 * F, 2 * F * 4);
                bulk_commit();
                bulk_wait_read_all();
                mbar_arrive(&zempty[zb]);
                ++k;
            }
            bulk_wait_all();
        }
    } else if (warp >= 12) {
        // --------------------------------------------------------------- update
        const int e = 32 * (warp & 3) + lane;
        const uint32_t dscol = tmem + cS + ((uint32_t)(32 * (warp & 3)) << 16);
        uint32_t k = 0;
        for (int u = u_begin; u < u_end && !*fail; ++u) {
            if (!wide_state(a, u)) continue;
            bool bad = !wait_bar(vfull, k & 1u, fail);
            ++k;
            {
                // (0x7f80 + 0x80 reaches the sign's place: an exponent of all ones)
                uint32_t seen = 0;
                for (int i = e; i < (d / 64) * kRows * 8; i += 128) {
                    const uint4 x = reinterpret_cast<const uint4 *>(smem + a.off_v)[i];
                    seen |= ((x.x & 0x7F807F80u) + 0x00800080u) | ((x.y & 0x7F807F80u) + 0x00800080u) |
                            ((x.z & 0x7F807F80u) + 0x00800080u) | ((x.w & 0x7F807F80u) + 0x00800080u);
                }
                const bool any = __any_sync(0xffffffffu, (seen & 0x80008000u) != 0);
                if (lane == 0) {
                    vbad[warp & 3] = any;
                    if (!bad) mbar_arrive(vscan);
                }
            }
            for (int c = 0; c < kChunks; ++c) {
                bad = !wait_bar(dsready, (uint32_t)c & 1u, fail) || bad;
                tc_fence_after();
                float v[2][32];
                tmem_ld32(dscol, v[0]);
                tmem_ld32(dscol + 32, v[1]);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0 && !bad) mbar_arrive(dsfree);
                // the readout has consumed the tiles
                bad = !wait_bar(&rdone[c & 1], (uint32_t)(c >> 1) & 1u, fail) || bad;
                if (!bad && e < d) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint8_t *rowp = smem + (size_t)((kW + 2 * c + h) % NS) * tile_bytes + e * 128;
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            float4 *p4 = reinterpret_cast<float4 *>(rowp + ((q ^ (e & 7)) << 4));
                            const float4 s4 = *p4;
                            *p4 = make_float4(s4.x + v[h][4 * q], s4.y + v[h][4 * q + 1], s4.z + v[h][4 * q + 2],
                                              s4.w + v[h][4 * q + 3]);
                        }
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && !bad) mbar_arrive(&tready[c]);
            }
        }
    } else {
        // ------------------------------------------------------------- math
        const int q4 = warp & 3, part = (warp - 4) >> 2;
        const int row = 32 * q4 + lane;                 // Tensor Memory lane
        const bool is_q = q4 < 2;                       // queries on lanes 0-63, keys on 64-127
        const int kr = row - kRows;                     // token of a key row
        const uint32_t lane_off = (uint32_t)(32 * q4) << 16;
        const uint32_t ucol = tmem + cU + lane_off, scol = tmem + cS + lane_off, mcol = tmem + cM + lane_off,
                       dcol = tmem + cD + lane_off;
        const bool valid = is_q ? row < G * B : kr < B;
        const float scale_l2 = a.inv_sqrt_d * kLog2e;
        float *xrow = reinterpret_cast<float *>(smem + a.off_st) + row;
        auto X = [&](int k, int p) -> float & { return xrow[(k * 2 + p) * 128]; };
        auto pair_failed = [&](bool local_fail) -> bool { return group_sync_failed(kBarPair + q4, 64, local_fail); };
        uint32_t k = 0;
        for (int u = u_begin; u < u_end; ++u) {
            if (!wide_state(a, u)) {
                if (tid == 128) raise_error(a.err, ERR_BAD_STATE_PTR);
                continue;
            }
            const int r = u / a.Hkv, g = u % a.Hkv;
            const int zb = k & 1;
            float *zs = zbuf + zb * 2 * F, *dzs = zbuf + (2 + (q4 & 1)) * 2 * F;
            const float alpha_row = is_q && valid ? a.alpha[g * G + row % G] : 0.f;
            // (after a failure every wait returns at once and the unit runs to its end without
            // arrivals, so that all warps of a named barrier reach it and leave together)
            // ---- extrema; a part owns columns [32 c + 16 part, + 16) of every chunk c
            bool bad = !wait_bar(uready, k & 1u, fail);
            tc_fence_after();
            float ms = -INFINITY, mx = -INFINITY, mn = INFINITY;
#pragma unroll 2
            for (int c = 0; c < kChunks; ++c) {
                float v[16];
                tmem_ld16(ucol + 32 * c + 16 * part, v);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    mx = fmaxf(mx, v[i]);
                    mn = fminf(mn, v[i]);
                }
            }
            if (is_q)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float v[16];
                    tmem_ld16(scol + 32 * part + 16 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) ms = fmaxf(ms, 32 * part + 16 * c + i < B ? v[i] : -INFINITY);
                }
            X(0, part) = ms;
            X(1, part) = mx;
            X(2, part) = mn;
            bad = pair_failed(bad);
            ms = fmaxf(X(0, 0), X(0, 1));
            mx = fmaxf(X(1, 0), X(1, 1));
            mn = fminf(X(2, 0), X(2, 1));
            const float mxl = mx * kLog2e, mnl = mn * kLog2e, msl = ms * scale_l2;
            // ---- sums of both signs; the queries' products with z and score sums
            float sp = 0.f, sn = 0.f, lp = 0.f, ln = 0.f, l = 0.f;
            if (is_q) {
                bad = !wait_bar(&zfull[zb], (k >> 1) & 1u, fail) || bad;
#pragma unroll 1
                for (int c = 0; c < kChunks; ++c) {
                    float v[16];
                    tmem_ld16(ucol + 32 * c + 16 * part, v);
                    const float4 *zp = reinterpret_cast<const float4 *>(zs + 32 * c + 16 * part);
                    const float4 *zn = reinterpret_cast<const float4 *>(zs + F + 32 * c + 16 * part);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 p4 = zp[q], n4 = zn[q];
                        const float pz[4] = {p4.x, p4.y, p4.z, p4.w}, nz[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float ep = ex2(fmaf(v[4 * q + j], kLog2e, -mxl)), en = ex2(fmaf(-v[4 * q + j], kLog2e, mnl));
                            sp += ep;
                            sn += en;
                            lp = fmaf(ep, pz[j], lp);
                            ln = fmaf(en, nz[j], ln);
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float v[16];
                    tmem_ld16(scol + 32 * part + 16 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        l += 32 * part + 16 * c + i < B ? ex2(fmaf(v[i], scale_l2, -msl)) : 0.f;
                }
            } else {
                // keys: part 0 sums phi+, part 1 phi-, over all columns and in the order of the
                // block commit kernel (per 32 columns the halving tree of a warp, then quarters
                // and halves), so that both give the same bits of phi(k)
                const float sgn = part == 0 ? kLog2e : -kLog2e, off = part == 0 ? -mxl : mnl;
                auto chunk_sum = [&](int c) -> float {
                    float v[32];
                    tmem_ld32(ucol + 32 * c, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = ex2(fmaf(v[i], sgn, off));
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1)
#pragma unroll
                        for (int i = 0; i < w; ++i) v[i] += v[i + w];
                    return v[0];
                };
                float sum = 0.f;
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const float a0 = chunk_sum(4 * h), a1 = chunk_sum(4 * h + 1);
                    const float a2 = chunk_sum(4 * h + 2), a3 = chunk_sum(4 * h + 3);
                    const float q = (a0 + a1) + (a2 + a3);
                    sum = h == 0 ? q : sum + q;
                }
                if (part == 0) sp = sum;
                else sn = sum;
            }
            X(3, part) = sp;
            X(4, part) = sn;
            X(5, part) = lp;
            X(6, part) = ln;
            X(7, part) = l;
            bad = pair_failed(bad);
            float cp = 1.f / (X(3, 0) + X(3, 1)), cn = 1.f / (X(4, 0) + X(4, 1));
            if (is_q) {
                // merge weights into phi and P
                const float ld = (X(5, 0) + X(5, 1)) * cp + (X(6, 0) + X(6, 1)) * cn;
                MergeWeights mw{0.f, 0.f};
                if (valid) mw = merge_weights(log_sigmoid(alpha_row), ms * a.inv_sqrt_d, X(7, 0) + X(7, 1), ld);
                cp *= mw.wl;
                cn *= mw.wl;
                bad = !wait_bar(vscan, k & 1u, fail) || bad;
                const bool finite = (vbad[0] | vbad[1] | vbad[2] | vbad[3]) == 0;
                uint8_t *prow = xs + (row >> 3) * (kRows / 8) * 128 + (row & 7) * 16;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float v[16];
                    tmem_ld16(scol + 32 * part + 16 * c, v);
                    tmem_wait_ld();
                    uint32_t h[8], lo[8];
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const int j = 32 * part + 16 * c + i;
                        const float p0 = j < B ? ex2(fmaf(v[i], scale_l2, -msl)) * mw.ws : 0.f;
                        const float p1 = j + 1 < B ? ex2(fmaf(v[i + 1], scale_l2, -msl)) * mw.ws : 0.f;
                        h[i / 2] = finite ? pack_bf16x2(p0, p1) : bf16_pair(p0, p1);
                        const float h0 = __uint_as_float(h[i / 2] << 16), h1 = __uint_as_float(h[i / 2] & 0xFFFF0000u);
                        lo[i / 2] = finite ? pack_bf16x2(p0 - h0, p1 - h1)
                                           : pack_bf16x2(positive_rest(p0, h0, p0), positive_rest(p1, h1, p1));
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        uint8_t *p = prow + (4 * part + 2 * c + j) * 128;
                        *reinterpret_cast<uint4 *>(p) = make_uint4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
                        *reinterpret_cast<uint4 *>(p + kPPart) = make_uint4(lo[4 * j], lo[4 * j + 1], lo[4 * j + 2], lo[4 * j + 3]);
                    }
                }
            } else if (!valid) {
                cp = cn = 0.f;   // key rows beyond B
            }
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && !bad) mbar_arrive(pready);

            // ---- phi of every chunk
#pragma unroll 1
            for (int c = 0; c < kChunks; ++c) {
                const uint32_t b = c & 1;
                float v[16];
                tmem_ld16(ucol + 32 * c + 16 * part, v);
                // buffer b has been read (for c < 2 by the previous unit, complete before uready)
                if (c >= 2) bad = !wait_bar(&rdone[b], (uint32_t)((c >> 1) - 1) & 1u, fail) || bad;
                tmem_wait_ld();
                if (is_q) {
                    tc_fence_after();
                    float w[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        w[i] = tf32_rna(ex2(fmaf(-v[i], kLog2e, mnl)) * cn);
                        v[i] = tf32_rna(ex2(fmaf(v[i], kLog2e, -mxl)) * cp);
                    }
                    tmem_st16(ucol + 32 * c + 16 * part, v);
                    tmem_st16(mcol + 32 * b + 16 * part, w);
                    tmem_wait_st();
                    tc_fence_before();
                } else {
                    // row kr of [token][32 phi+ | 32 phi-], granules permuted by (kr mod 8)
                    float w[32];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        w[16 + i] = ex2(fmaf(v[i], -kLog2e, mnl)) * cn;
                        w[i] = ex2(fmaf(v[i], kLog2e, -mxl)) * cp;
                    }
                    uint8_t *rowp = xs + kPhi + b * kPhiPanel + kr * 128;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int gr = (j >> 1) * 4 + 2 * part + (j & 1);
                        *reinterpret_cast<uint4 *>(rowp + ((gr ^ (kr & 7)) << 4)) =
                            make_uint4(pack_bf16x2(w[8 * j], w[8 * j + 1]), pack_bf16x2(w[8 * j + 2], w[8 * j + 3]),
                                       pack_bf16x2(w[8 * j + 4], w[8 * j + 5]), pack_bf16x2(w[8 * j + 6], w[8 * j + 7]));
                    }
                    fence_proxy_async_smem();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0 && !bad) mbar_arrive(&phi[b]);
                    // token sums over this warp's 32 tokens: lane L < 16 phi+, L >= 16 phi-
                    const float sum = warp_reduce32<0>(w, lane);
                    dzs[(lane >> 4) * F + 32 * c + 16 * part + (lane & 15)] = sum;
                }
                if (is_q) {
                    __syncwarp();
                    if (lane == 0 && !bad) mbar_arrive(&phi[b]);
                }
            }
            if (is_q) {
                // ---- the output rows: D
                bad = !wait_bar(udone, k & 1u, fail) || bad;
                tc_fence_after();
                const int dh = d / 2;
                bf16 *orow = a.O + (((size_t)r * B + row / G) * a.Hq + g * G + row % G) * d + part * dh;
                for (int c0 = 0; c0 < dh; c0 += 32) {
                    float v[32];
                    tmem_ld32(dcol + part * dh + c0, v);
                    tmem_wait_ld();
                    if (c0 + 32 >= dh) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0 && !bad) mbar_arrive(dfree);
                    }
                    if (valid && !bad) {
                        uint4 *dst = reinterpret_cast<uint4 *>(orow + c0);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            dst[i] = make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                                                pack_bf16x2(v[8 * i + 4], v[8 * i + 5]), pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
                    }
                }
                bad = pair_failed(bad);
            } else {
                // ---- z += the two token halves' sums (the key warps; the queries have read z)
                bad = !wait_bar(&zfull[zb], (k >> 1) & 1u, fail) || bad;
                bad = group_sync_failed(kBarKeys, 128, bad);
                const int t = (q4 - 2) * 64 + part * 32 + lane;   // 0 .. 127
                const float *dz0 = zbuf + 2 * 2 * F, *dz1 = zbuf + 3 * 2 * F;
                for (int f = t; f < 2 * F; f += 128) zs[f] += dz0[f] + dz1[f];
                fence_proxy_async_smem();
                bad = group_sync_failed(kBarKeys, 128, bad);   // the sums have been read
                if (lane == 0 && !bad) mbar_arrive(zdone);
            }
            if (bad) break;
            ++k;
        }
        if (tid == 128 && *fail) raise_error(a.err, ERR_WAIT_TIMEOUT);
    }

    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace

bool fused_wide_supported(const hybrid_cfg &c)
{
    if (c.io_dtype != HYBRID_BF16 || c.feat_dim != F) return false;
    if (c.head_dim != 64 && c.head_dim != 128) return false;
    const int G = c.n_q_heads / c.n_kv_heads;
    return c.block_size % 16 == 0 && G * c.block_size <= kRows && kRows % G == 0;
}

cudaError_t launch_fused_wide(const hybrid_cfg &c, const void *Q, const void *K, const void *V, const void *W,
                              const float *alpha, void *const *states, int n_req, void *O, unsigned *err,
                              cudaStream_t st)
{
    const int d = c.head_dim, B = c.block_size, Hq = c.n_q_heads, Hkv = c.n_kv_heads, G = Hq / Hkv;
    const WLayout L = wide_layout(d);
    WideArgs a{};
    {
        const cuuint64_t dq[4] = {(cuuint64_t)d, (cuuint64_t)Hq, (cuuint64_t)B, (cuuint64_t)n_req};
        const cuuint64_t sq[3] = {(cuuint64_t)d * 2, (cuuint64_t)Hq * d * 2, (cuuint64_t)B * Hq * d * 2};
        const cuuint32_t bq[4] = {64, (cuuint32_t)G, (cuuint32_t)(kRows / G), 1};
        const cuuint64_t dk[4] = {(cuuint64_t)d, (cuuint64_t)Hkv, (cuuint64_t)B, (cuuint64_t)n_req};
        const cuuint64_t sk[3] = {(cuuint64_t)d * 2, (cuuint64_t)Hkv * d * 2, (cuuint64_t)B * Hkv * d * 2};
        const cuuint32_t bk[4] = {64, 1, (cuuint32_t)kRows, 1};
        const cuuint64_t dw[3] = {64, (cuuint64_t)Hkv * d, (cuuint64_t)kW};
        const cuuint64_t sw[2] = {(cuuint64_t)F * 2, 128};
        const cuuint32_t bw[3] = {64, (cuuint32_t)d, (cuuint32_t)kW};
        if (!encode_bf16(&a.tmQ, Q, 4, dq, sq, bq) || !encode_bf16(&a.tmK, K, 4, dk, sk, bk) ||
            !encode_bf16(&a.tmV, V, 4, dk, sk, bk) || !encode_bf16(&a.tmW, W, 3, dw, sw, bw))
            return cudaErrorInvalidValue;
    }
    a.alpha = alpha;
    a.states = states;
    a.O = static_cast<bf16 *>(O);
    a.err = err;
    a.n_units = n_req * Hkv;
    a.B = B;
    a.Hq = Hq;
    a.Hkv = Hkv;
    a.G = G;
    a.d = d;
    a.inv_sqrt_d = 1.f / sqrtf((float)d);
    a.off_x = L.off_x;
    a.off_v = L.off_v;
    a.off_z = L.off_z;
    a.off_st = L.off_st;
    a.off_bar = L.off_bar;
    static std::atomic<unsigned long long> opted{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const unsigned long long bit = 1ull << dev;
    if (!(opted.load(std::memory_order_acquire) & bit)) {
        const cudaError_t e = cudaFuncSetAttribute(k_fused_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e != cudaSuccess) return e;
        opted.fetch_or(bit, std::memory_order_release);
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(a.n_units < sm_count() ? a.n_units : sm_count());
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = L.bytes;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, k_fused_wide, a);
}

}  // namespace hyb
