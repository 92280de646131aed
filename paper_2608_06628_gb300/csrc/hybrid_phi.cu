// hybrid_phi.cu -- the feature map of Section 3.1, Phi = [softmax(X W_g), softmax(-X W_g)],
// for bf16 inputs on the tensor cores.  bf16 products are exact in float32, so U = X W is
// the float32 dot product of the same terms that the CUDA-core kernel adds; to keep its
// rounding no larger, d is split over two accumulators (added in float32 by the math warps)
// and everything after U is float32 as there (expf, max-shifted softmaxes).  Relative
// error against 64 bits, d = F = 128: 1.3e-7; a dot product added in one float32 chain, as
// one warp per row and head did, 1.5e-7; one accumulator (tried for F = 256) 2.1e-7.
//
// A tile is 128 (row, head) pairs of one state head's query group, so that W_g serves the
// whole tile.  One persistent CTA of 16 warps per SM, four threads per row with F / 4
// columns each; the row's extrema and sums meet in shared memory, and each warp turns its
// 32 rows x 32 columns through shared memory so that rows leave as whole 128-byte lines.
// Thread 0 also issues the MMAs of the next tile and the TMA of the one after it as soon as
// a tile's U is complete.  Tensor Memory: two buffers of kAcc accumulators x F columns, so
// that the next tile's products run under this tile's softmaxes (F = 256: one buffer).
//
// What bounds it: the output (2F float32 per row and head) is written once; 4096 rows x 16
// heads with d = F = 128: 24.4 us (84 MB, 3.4 TB/s) against 124 us on register tiles and 320
// us with one warp per row and head.
#include <atomic>

#include "hybrid_common.cuh"
#include "hybrid_tc.h"
#include "tc_pipeline.cuh"

namespace hyb {

namespace {

using namespace pipe;

constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kSmemLimit = 232448;
constexpr uint32_t kXBytes = 2 * 128 * 128;   // a tile of X: d / 64 panels of 128 rows, 16 KB apart

struct PhiTcArgs {
    CUtensorMap tmX, tmW;   // X [rows][nh][d] box {64, group, 128 / group, d / 64}; W box {64, d, F / 64}
    float *Phi;
    unsigned *err;
    long long rows;         // (row, head) pairs per state head
    int n_tiles, tiles_per_g, nh, log_group, d;
};

template <int F>
struct PhiCfg {
    static constexpr int kAcc = 2;                      // accumulators (the k range in as many parts)
    static constexpr int kCols = F / 4;                 // columns of a thread
    static constexpr uint32_t kBuf = (uint32_t)kAcc * F;   // Tensor Memory columns of a buffer
    static constexpr int kBufs = F <= 128 ? 2 : 1;      // F = 256: one buffer fills Tensor Memory
    static constexpr uint32_t kTmem = kBufs * kBuf;
};

inline uint32_t phi_smem(int d, int F) { return 2 * kXBytes + (uint32_t)(F / 64) * d * 128 + kWarps * 4096 + 16 * 512 + 256 + 1024; }

template <int F>
__global__ void __launch_bounds__(kThreads, 1) k_phi_tc(const __grid_constant__ PhiTcArgs a)
{
    using namespace ptx;
    using C = PhiCfg<F>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d;
    uint8_t *xs = smem;                                      // two tiles of X
    uint8_t *ws = smem + 2 * kXBytes;                        // W_g
    uint8_t *stage = ws + (F / 64) * d * 128;                // 4 KB per math warp
    float *stat = reinterpret_cast<float *>(stage + kWarps * 4096);   // [4 statistics][4 parts][128 rows]
    uint64_t *bars = reinterpret_cast<uint64_t *>(stat + 16 * 128);
    uint64_t *xfull = bars, *ufull = bars + 2, *ufree = bars + 4, *wfull = bars + 6;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + 7);
    volatile int *fail = reinterpret_cast<volatile int *>(tmem_holder + 1);

    const int per = a.n_tiles / (int)gridDim.x, rem = a.n_tiles % (int)gridDim.x;
    const int t_begin = (int)blockIdx.x * per + min((int)blockIdx.x, rem);
    const int n = per + ((int)blockIdx.x < rem ? 1 : 0);
    if (tid == 0) {
        prefetch_tensormap(&a.tmX);
        prefetch_tensormap(&a.tmW);
        mbar_init_n(xfull, 4, 1);   // ufull
        mbar_init_n(ufree, 2, kWarps);
        mbar_init_n(wfull, 1, 1);
        *fail = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(tmem_holder, C::kTmem);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    if (tid == 0) griddep_launch_dependents();
    griddep_wait();
    const uint32_t tmem = *tmem_holder;

    // thread 0: copies and MMAs of the CTA's tiles (bad: a wait of this thread ran out)
    int nx = 0, nw = 0, g_cur = -1;
    auto load_x = [&](int i) {
        const int t = t_begin + i, g = t / a.tiles_per_g, j = t % a.tiles_per_g;
        mbar_arrive_expect_tx(&xfull[i & 1], (uint32_t)(d / 64) * (128 * 128));
        tma_load_4d(xs + (i & 1) * kXBytes, &a.tmX, 0, g << a.log_group, (j * 128) >> a.log_group, 0, &xfull[i & 1]);
        ++nx;
    };
    // the products of tile i, once tile i - 1 is formed (so W may be replaced) and the math
    // warps have read the tile that held its Tensor Memory buffer
    auto form = [&](int i) -> bool {
        const int b = i & 1, ub = i % C::kBufs, g = (t_begin + i) / a.tiles_per_g;
        if (g != g_cur) {
            mbar_arrive_expect_tx(wfull, (uint32_t)(F / 64) * d * 128);
            tma_load_3d(ws, &a.tmW, 0, g * d, 0, wfull);
            ++nw;
            g_cur = g;
            if (!wait_bar(wfull, (uint32_t)(nw - 1) & 1u, fail)) return false;
        }
        if (!wait_bar(&xfull[b], (uint32_t)(i >> 1) & 1u, fail)) return false;
        if (i >= C::kBufs && !wait_bar(&ufree[ub], (uint32_t)(i / C::kBufs - 1) & 1u, fail)) return false;
        tc_fence_after();
        const uint32_t x_u = smem_u32(xs + b * kXBytes), w_u = smem_u32(ws);
        constexpr uint32_t idU = instr_desc(FMT_BF16, FMT_BF16, false, true, 128, F);
        const int part = d / 16 / C::kAcc;   // k-steps per accumulator
        for (int k = 0; k < d / 16; ++k)
            mma_bf16_ss(tmem + ub * C::kBuf + (uint32_t)(k / part) * F,
                        smem_desc(x_u + (k >> 2) * (128 * 128) + (k & 3) * 32, 16, 1024, SWZ_128B),
                        smem_desc(w_u + 2 * k * 1024, d * 128, 1024, SWZ_128B), idU, k % part > 0);
        mma_commit(&ufull[ub]);
        return true;
    };
    bool bad = false;
    int formed = 0;
    if (tid == 0 && n > 0) {
        load_x(0);
        if (n > 1) load_x(1);
        bad = !form(0);
        formed = bad ? 0 : 1;
    }
    {
        const int q4 = warp & 3, part = warp >> 2;
        const int row = 32 * q4 + lane;
        const uint32_t lane_off = (uint32_t)(32 * q4) << 16;
        uint8_t *sg = stage + warp * 4096;
        // statistics of the tile's rows, one [4 parts][128 rows] array each
        float *xmx = stat, *xmn = stat + 512, *xsp = stat + 1024, *xsn = stat + 1536;
        const uint32_t qbar = 1 + q4;
        constexpr int CW = C::kCols < 32 ? C::kCols : 32, NCH = C::kCols / CW;   // chunk width, chunks
        for (int i = 0; i < n; ++i) {
            const int ub = i % C::kBufs;
            const int t = t_begin + i, g = t / a.tiles_per_g;
            const long long r0 = (long long)(t % a.tiles_per_g) * 128;
            bad = !wait_bar(&ufull[ub], (uint32_t)(i / C::kBufs) & 1u, fail) || bad;
            tc_fence_after();
            auto next = [&]() {
                if (tid == 0 && !bad && i + 1 < n) {
                    if (i + 2 < n) load_x(i + 2);   // into the buffer this tile has read
                    bad = !form(i + 1);
                    if (!bad) ++formed;
                }
                __syncwarp();
            };
            if constexpr (C::kBufs > 1) next();
            const uint32_t ucol = tmem + lane_off + ub * C::kBuf + part * C::kCols;
            float u[NCH][CW];
            float mx = -INFINITY, mn = INFINITY;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                float v[CW];   // the second accumulator
                if constexpr (CW == 32) {
                    tmem_ld32(ucol + 32 * c, u[c]);
                    tmem_ld32(ucol + F + 32 * c, v);
                } else {
                    tmem_ld16(ucol, u[c]);
                    tmem_ld16(ucol + F, v);
                }
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < CW; ++k) {
                    u[c][k] += v[k];
                    mx = fmaxf(mx, u[c][k]);
                    mn = fminf(mn, u[c][k]);
                }
            }
            // U has been read: the products of a later tile may overwrite it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ufree[ub]);
            if constexpr (C::kBufs == 1) next();
            xmx[part * 128 + row] = mx;
            xmn[part * 128 + row] = mn;
            if (group_sync_failed(qbar, 128, bad)) break;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                mx = fmaxf(mx, xmx[p * 128 + row]);
                mn = fminf(mn, xmn[p * 128 + row]);
            }
            // one chunk: the exponentials stay in registers; two: they are formed again below
            float sp4[4] = {0.f, 0.f, 0.f, 0.f}, sn4[4] = {0.f, 0.f, 0.f, 0.f}, en[NCH == 1 ? CW : 1];
#pragma unroll
            for (int c = 0; c < NCH; ++c)
#pragma unroll
                for (int k = 0; k < CW; ++k) {
                    const float ep = expf(u[c][k] - mx), e = expf(mn - u[c][k]);
                    sp4[k & 3] += ep;   // four short chains: less rounding than one long one
                    sn4[k & 3] += e;
                    if constexpr (NCH == 1) {
                        u[c][k] = ep;
                        en[k] = e;
                    }
                }
            float sp = (sp4[0] + sp4[1]) + (sp4[2] + sp4[3]), sn = (sn4[0] + sn4[1]) + (sn4[2] + sn4[3]);
            xsp[part * 128 + row] = sp;
            xsn[part * 128 + row] = sn;
            if (group_sync_failed(qbar, 128, false)) break;
            sp = (xsp[row] + xsp[128 + row]) + (xsp[256 + row] + xsp[384 + row]);
            sn = (xsn[row] + xsn[128 + row]) + (xsn[256 + row] + xsn[384 + row]);
            const float ip = 1.f / sp, in = 1.f / sn;
            // a chunk of a sign through the warp's 4 KB: row = lane, granules permuted by the
            // row, then whole row pieces of CW values to global memory
            constexpr int GR = CW / 4;      // 16-byte granules of a row piece
            constexpr int RI = 32 / GR;     // rows written by one store instruction
            const long long rw = r0 + 32 * q4;
            auto put = [&](const float (&e)[CW], int col) {
                __syncwarp();
#pragma unroll
                for (int k = 0; k < GR; ++k)
                    *reinterpret_cast<float4 *>(sg + lane * (CW * 4) + ((k ^ (lane & (GR - 1))) << 4)) =
                        make_float4(e[4 * k], e[4 * k + 1], e[4 * k + 2], e[4 * k + 3]);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 32 / RI; ++k) {
                    const int rr = k * RI + lane / GR, gr = lane & (GR - 1);
                    const float4 v = *reinterpret_cast<const float4 *>(sg + rr * (CW * 4) + ((gr ^ (rr & (GR - 1))) << 4));
                    const long long ri = rw + rr;
                    if (ri < a.rows) {
                        const long long item = (ri >> a.log_group) * a.nh + (g << a.log_group) + (ri & ((1 << a.log_group) - 1));
                        *reinterpret_cast<float4 *>(a.Phi + item * (2 * F) + col + 4 * gr) = v;
                    }
                }
            };
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                float e[CW];
#pragma unroll
                for (int k = 0; k < CW; ++k) e[k] = (NCH == 1 ? u[c][k] : expf(u[c][k] - mx)) * ip;
                put(e, part * C::kCols + 32 * c);
#pragma unroll
                for (int k = 0; k < CW; ++k) e[k] = (NCH == 1 ? en[NCH == 1 ? k : 0] : expf(mn - u[c][k])) * in;
                put(e, F + part * C::kCols + 32 * c);
            }
        }
        if (tid == 0 && *fail) {
            raise_error(a.err, ERR_WAIT_TIMEOUT);
            // copies and products in flight end before the CTA exits
            for (int k = 0; k < 2 && k < nx; ++k)
                mbar_wait(&xfull[(nx - 1 - k) & 1], (uint32_t)((nx - 1 - k) >> 1) & 1u, kWaitNs);
            if (nw) mbar_wait(wfull, (uint32_t)(nw - 1) & 1u, kWaitNs);
            if (formed) mbar_wait(&ufull[(formed - 1) % C::kBufs], (uint32_t)((formed - 1) / C::kBufs) & 1u, kWaitNs);
        }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmem);
    }
}

template <int F>
cudaError_t launch_phi(const PhiTcArgs &a, cudaStream_t st)
{
    static std::atomic<unsigned long long> opted{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const unsigned long long bit = 1ull << dev;
    if (!(opted.load(std::memory_order_acquire) & bit)) {
        const cudaError_t e = cudaFuncSetAttribute(k_phi_tc<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e != cudaSuccess) return e;
        opted.fetch_or(bit, std::memory_order_release);
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(a.n_tiles < sm_count() ? a.n_tiles : sm_count());
    lc.blockDim = dim3(kThreads);
    const uint32_t smem = phi_smem(a.d, F);
    lc.dynamicSmemBytes = smem < 118 * 1024 ? 118 * 1024 : smem;   // one CTA per SM (Tensor Memory)
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, k_phi_tc<F>, a);
}

}  // namespace

// A tile's box is the group's heads of 128 / group rows.
bool phi_tc_supported(hybrid_dtype dt, long long n_rows, int group, int d, int F)
{
    if (dt != HYBRID_BF16 || (d != 64 && d != 128) || (F != 64 && F != 128 && F != 256)) return false;
    if (group > 128 || 128 % group != 0) return false;
    return n_rows * group <= (1ll << 30);
}

cudaError_t launch_phi_tc(const void *X, int n_rows, int nh, int Hkv, int d, int F, const void *W, float *Phi,
                          unsigned *err, cudaStream_t st)
{
    PhiTcArgs a{};
    const int group = nh / Hkv;
    const cuuint64_t dx[4] = {64, (cuuint64_t)nh, (cuuint64_t)n_rows, (cuuint64_t)d / 64};
    const cuuint64_t sx[3] = {(cuuint64_t)d * 2, (cuuint64_t)nh * d * 2, 128};
    const cuuint32_t bx[4] = {64, (cuuint32_t)group, (cuuint32_t)(128 / group), (cuuint32_t)d / 64};
    const cuuint64_t dw[3] = {64, (cuuint64_t)Hkv * d, (cuuint64_t)F / 64};
    const cuuint64_t sw[2] = {(cuuint64_t)F * 2, 128};
    const cuuint32_t bw[3] = {64, (cuuint32_t)d, (cuuint32_t)F / 64};
    if (!encode_bf16(&a.tmX, X, 4, dx, sx, bx) || !encode_bf16(&a.tmW, W, 3, dw, sw, bw)) return cudaErrorInvalidValue;
    a.Phi = Phi;
    a.err = err;
    a.rows = (long long)n_rows * group;
    a.tiles_per_g = (int)((a.rows + 127) / 128);
    a.n_tiles = a.tiles_per_g * Hkv;
    a.nh = nh;
    a.log_group = 0;
    while ((1 << a.log_group) < group) ++a.log_group;
    a.d = d;
    if (F == 64) return launch_phi<64>(a, st);
    if (F == 128) return launch_phi<128>(a, st);
    return launch_phi<256>(a, st);
}

}  // namespace hyb
