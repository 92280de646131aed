// hybrid_generic.cu -- CUDA-core kernels for every supported shape and dtype.
//
// These kernels do all arithmetic in float32 on the FMA pipes.  They are the
// exact path for float32 I/O and the path for shapes that the tensor-core
// kernels do not take.  Section 3.1 of "Retrofitting Linear Attention into
// Diffusion Language Models" defines every quantity computed here.  The step is
// in attn_fma.cuh; this file holds the feature map, the commit and the choice of
// tile sizes.
#include <cooperative_groups.h>

#include "attn_fma.cuh"

namespace hyb {

using namespace fma;

namespace {

// Rows per CTA: the fewest waves weighted by what a CTA costs.  One wave of the d = F =
// 128, B = 32 step takes 18 us with 16-row CTAs, 25 us with 32 and 41 us with 64 (one CTA
// per SM; the feature map 7.5, 10.3 and 15.8 us).
int pick_rows(long long units, long long rows, bool allow64)
{
    const int cand[3] = {16, 32, 64}, cost[3] = {18, 25, 41};
    const long long slots = pipe::sm_count();
    int best = 16;
    long long best_t = -1;
    for (int i = 0; i < (allow64 ? 3 : 2); ++i) {
        const long long ctas = units * ((rows + cand[i] - 1) / cand[i]);
        const long long t = (ctas + slots - 1) / slots * cost[i];
        if (best_t < 0 || t < best_t) {
            best_t = t;
            best = cand[i];
        }
    }
    return best;
}

// ---------------------------------------------------------------------------
// Feature map: Phi = [softmax(X W_g), softmax(-X W_g)] for RT rows of the heads of one
// state head (row i of group g is (i / group, g * group + i % group)), so that W_g is
// read once per RT rows (float32 rows, and bf16 ones with F < 64; the others run in
// hybrid_phi.cu).  4096 float32 rows x 16 heads, d = F = 128: 329 us with one warp per row and
// head (W_g read from L1 by every warp), 124 us now (bf16 rows, F = 32: 290 and 84); the FMA
// pipes' floor is 28 us, the rest is the staging of X and W and the exponentials, with 8 warps
// per SM to hide them.
// ---------------------------------------------------------------------------
struct PhiArgs {
    const void *X, *W;
    float *Phi;
    long long rows;          // rows per state head: n_rows * group
    int nh, group, d, F;
    long long tiles;         // row tiles per state head
    bool bf16_io;
};

size_t phi_smem_bytes(int d, int F, int RT)
{
    return sizeof(float) * ((size_t)RT * (d + 4) + 2 * (size_t)(F > 64 ? 128 : 64) * 32 + xch_floats(RT));
}

template <int RT, int FP>
__global__ void __launch_bounds__(kThreads) k_feature_map(const PhiArgs a)
{
    extern __shared__ __align__(16) float smem[];
    using UP = UPanels<FP>;
    using MU = Map<UP::PN, RT>;
    const int d = a.d, F = a.F, ND = d / 32, LQ = d + 4;
    float *xs = smem;                    // [RT][LQ]
    float *tb = xs + RT * LQ;            // two W tiles
    const int tile_floats = (F > 64 ? 128 : 64) * 32;
    float *xch = tb + 2 * tile_floats;   // statistics on their way between warps
    const int tid = threadIdx.x;
    const int g = (int)(blockIdx.x / a.tiles);
    const long long i0 = (blockIdx.x % a.tiles) * (long long)RT;
    const int rows = (int)min((long long)RT, a.rows - i0);
    const size_t w0 = (size_t)g * d * F;
    // element offset of row i's head vector, in units of d (X) or 2F (Phi)
    auto item = [&](int i) -> size_t {
        const long long ri = i0 + i;
        return (size_t)(ri / a.group) * a.nh + (size_t)(g * a.group) + (size_t)(ri % a.group);
    };
    ptx::griddep_launch_dependents();
    ptx::griddep_wait();
    const int FC = FP == 2 ? 128 : F;    // columns of a W tile: tile k of panel p is the stream's p ND + k
    Staged st;
    auto load_w = [&](int i) {
        st.load_cols(a.W, w0 + (size_t)(i % ND) * 32 * F + (i / ND) * UP::PN, F, 32, FC, a.bf16_io);
    };
    load_w(0);
    for (int p = tid; p < RT * (d / 4); p += kThreads) {
        const int i = p / (d / 4), e = (p % (d / 4)) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < rows) v = load4(a.X, item(i) * d + e, a.bf16_io);
        *reinterpret_cast<float4 *>(xs + i * LQ + e) = v;
    }
    st.store_cols(tb, FC);
    __syncthreads();
    using R = Rows<UP::PN, RT>;
    const MU mu;
    float u[UP::N][MU::NO], un[UP::N][MU::NO], ld[R::RPL];
    int s = 0;
#pragma unroll
    for (int p = 0; p < UP::N; ++p) {
        f32x2 acc[MU::TM * 8];
        clear(acc);
#pragma unroll 1
        for (int k = 0; k < ND; ++k, ++s) {
            const bool more = s + 1 < UP::N * ND;
            if (more) load_w(s + 1);
            tile32(mu, xs + 32 * k, LQ, tb + (s & 1) * tile_floats, acc);
            if (more) st.store_cols(tb + ((s + 1) & 1) * tile_floats, FC);
            __syncthreads();
        }
        finish(mu, acc, u[p]);
    }
    phi_rows<UP::PN, RT, UP::N, false>(mu, F, u, un, nullptr, ld, xch);
#pragma unroll
    for (int j = 0; j < R::RPL; ++j) {
        const int row = mu.row(j * R::CPL);
        if (row >= rows) continue;
        float *out = a.Phi + item(row) * 2 * F;
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
    }
}

template <int RT, int FP>
cudaError_t launch_phi_rt(PhiArgs a, int Hkv, cudaStream_t st)
{
    static std::atomic<unsigned long long> opted{0};
    a.tiles = (a.rows + RT - 1) / RT;
    return launch_opted(&k_feature_map<RT, FP>, opted, (unsigned)(a.tiles * Hkv), phi_smem_bytes(a.d, a.F, RT), st, a);
}
template <int FP>
cudaError_t launch_phi_f(const PhiArgs &a, int Hkv, cudaStream_t st)
{
    const int rt = pick_rows(Hkv, a.rows, FP < 2);
    if (rt == 64) {
        if constexpr (FP < 2) return launch_phi_rt<64, FP>(a, Hkv, st);
    }
    return rt >= 32 ? launch_phi_rt<32, FP>(a, Hkv, st) : launch_phi_rt<16, FP>(a, Hkv, st);
}

// ---------------------------------------------------------------------------
// Commit: S += sum_t phi(k_t) v_t^T, z += sum_t phi(k_t).  A cluster of F / FS CTAs takes
// one (request, state head); each CTA owns FS features of both signs (FS = 32 with d =
// 128, 64 with d = 64: the state slice is then 32 accumulators per thread).  U = K W is
// formed once per unit, a slice of columns per CTA; the softmaxes' extrema and sums over
// all F columns are exchanged through distributed shared memory, each CTA writing its own
// into every peer (one cluster barrier per chunk of 32 tokens).  The state slice is read
// at entry, accumulated in token order and written once.
//
// What bounds it at block size: latency (one pass of loads, one of products, one exchange).
// Step and commit of 8 requests, 16 : 4 heads, d = F = 128, B = 32, float32: 201 us with one
// CTA per query head and a commit that formed phi(K) again for every two state tiles; 37 us
// now, 25 of them the step.
// ---------------------------------------------------------------------------
constexpr int kTC = 32;

struct CommitFmaArgs {
    const void *K, *V, *W;
    void *const *states;
    unsigned *err;
    int n_tok, Hkv, F;
    bool bf16_io;
};

// statistics of a chunk, per (slice, token): max u, sum e^(u - max), min u, sum e^(min - u)
constexpr int kMaxSlices = 8;
constexpr int kStatFloats = kMaxSlices * kTC * 4;

template <int D, int FS>
constexpr size_t commit_smem_bytes()
{
    return sizeof(float) * ((size_t)FS * D + (size_t)kTC * 2 * FS * 2 + (size_t)kTC * (D + 4) + (size_t)kTC * D +
                            2 * kStatFloats + (kThreads / 32) * 2 * FS + (size_t)kTC * (FS + 1));
}

template <int D, int FS>
__global__ void __launch_bounds__(kThreads) k_commit_fma(const CommitFmaArgs a)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) float smem[];
    constexpr int P2s = 2 * FS, LK = D + 4, GQ = P2s / 4, WQ = GQ >= 8 ? GQ / 8 : 1;
    constexpr int NV = FS > 32 ? 2 : 1;      // features of a lane
    constexpr int NL = kTC * (D / 4) / kThreads;
    const int F = a.F, NS = F / FS;
    float *wt = smem;                     // D/32 tiles of FS rows x 32 (W^T slice)
    float *pd = wt + FS * D;              // [32][2 FS][2] phi, each value twice
    float *ks = pd + kTC * P2s * 2;       // [32][LK]
    float *vs = ks + kTC * LK;            // [32][D]
    float *stat = vs + kTC * D;           // [2][slice][token][4], written by every CTA of the cluster
    float *dzp = stat + 2 * kStatFloats;  // [warp][2 FS] token sums of phi
    float *us = dzp + (kThreads / 32) * P2s;   // [32][FS + 1]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    cg::cluster_group cluster = cg::this_cluster();
    const int slice = (int)(blockIdx.x % (unsigned)NS);
    const int unit = (int)(blockIdx.x / (unsigned)NS);
    const int r = unit / a.Hkv, g = unit % a.Hkv;

    ptx::griddep_launch_dependents();
    ptx::griddep_wait();
    float *state = reinterpret_cast<float *>(a.states[r]);
    if (!state_ptr_ok(state)) {           // the same for every CTA of the cluster
        if (tid == 0 && slice == 0 && g == 0) raise_error(a.err, ERR_BAD_STATE_PTR);
        return;
    }
    float *Sg = state + (size_t)g * head_floats(D, F);
    cluster.barrier_arrive();             // waited for before the first write into a peer

    // a chunk's K and V rows, loaded one chunk ahead
    float4 kv[NL], vv[NL];
    auto load_chunk = [&](int t0) {
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const int p = tid + i * kThreads;
            const int t = t0 + p / (D / 4), e = (p % (D / 4)) * 4;
            kv[i] = vv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (t < a.n_tok) {
                const size_t src = (((size_t)r * a.n_tok + t) * a.Hkv + g) * D + e;
                kv[i] = load4(a.K, src, a.bf16_io);
                vv[i] = load4(a.V, src, a.bf16_io);
            }
        }
    };
    load_chunk(0);
    // this thread's 4 features (granule q of the slice's 2 FS) x 8 columns e0 .. e0 + 7
    const int q = (tid & 7) + 8 * (warp % WQ);
    const int eg = ((tid >> 3) & 3) + 4 * (warp / WQ);
    const bool owner = q < GQ && eg < D / 8;
    const int e0 = 8 * eg;
    const int sgn = q >= FS / 4 ? 1 : 0;
    const int f = sgn * F + slice * FS + 4 * (q - sgn * (FS / 4));
    float4 s4[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        s4[j] = owner ? *reinterpret_cast<const float4 *>(Sg + s_offset(f, e0 + j, D)) : make_float4(0.f, 0.f, 0.f, 0.f);
    const int zf = tid < P2s ? (tid >= FS ? F + slice * FS + tid - FS : slice * FS + tid) : 0;
    float z = tid < P2s ? Sg[z_offset(zf, D, F)] : 0.f, dz = 0.f;

    // W^T slice: 4 x 4 blocks transposed in registers
#pragma unroll
    for (int i0 = 0; i0 < (D / 4) * (FS / 4); i0 += kThreads) {
        const int p = i0 + tid;
        if (p < (D / 4) * (FS / 4)) {
            const int kq = p & 7, nq = (p >> 3) % (FS / 4), kt = (p >> 3) / (FS / 4);
            float4 x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                x[i] = load4(a.W, ((size_t)g * D + 32 * kt + 4 * kq + i) * F + slice * FS + 4 * nq, a.bf16_io);
            store_block(wt + kt * FS * 32, kq, nq, x);
        }
    }

    // dS of 4 features x 8 columns as pairs of neighbouring columns
    f32x2 acc[16];
    clear(acc);
    for (int t0 = 0, b = 0; t0 < a.n_tok; t0 += kTC, b ^= 1) {
        const int tc = min(kTC, a.n_tok - t0);
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const int p = tid + i * kThreads;
            const int t = p / (D / 4), e = (p % (D / 4)) * 4;
            *reinterpret_cast<float4 *>(ks + t * LK + e) = kv[i];
            *reinterpret_cast<float4 *>(vs + t * D + e) = vv[i];
        }
        __syncthreads();
        if (t0 + kTC < a.n_tok) load_chunk(t0 + kTC);
        // U slice: token tid / 8, columns tid % 8 + 8 c
        {
            constexpr int NC = FS / 8;
            const int t = tid >> 3, n0 = tid & 7;
            f32x2 u[NC];
            clear(u);
#pragma unroll 4
            for (int j = 0; j < D / 4; ++j) {
                const ulonglong2 av = *reinterpret_cast<const ulonglong2 *>(ks + t * LK + 4 * j);
                const float *w = wt + (j >> 3) * FS * 32 + n0 * 32 + (((j & 7) ^ n0) << 2);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const ulonglong2 bv = *reinterpret_cast<const ulonglong2 *>(w + c * 256);
                    u[c] = ffma2(av.x, bv.x, u[c]);
                    u[c] = ffma2(av.y, bv.y, u[c]);
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) us[t * (FS + 1) + n0 + 8 * c] = sum2(u[c]);
        }
        __syncthreads();
        // softmaxes of +-u over all F columns: four tokens per warp.  Each slice's extrema and
        // sums go to every CTA of the cluster; the buffers alternate, so a CTA overwrites a
        // chunk's statistics only after the next chunk's barrier
        if (t0 == 0) cluster.barrier_wait();   // every CTA of the cluster has started
        float *sb = stat + b * kStatFloats;
        float x[4][NV];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 4 * warp + i;
            float mx = -INFINITY, mn = INFINITY;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const bool in = lane + 32 * k < FS;
                x[i][k] = in ? us[t * (FS + 1) + lane + 32 * k] : 0.f;
                mx = fmaxf(mx, in ? x[i][k] : -INFINITY);
                mn = fminf(mn, in ? x[i][k] : INFINITY);
            }
            mx = warp_max(mx);
            mn = warp_min(mn);
            float sp = 0.f, sn = 0.f;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const bool in = lane + 32 * k < FS;
                sp += in ? expf(x[i][k] - mx) : 0.f;
                sn += in ? expf(mn - x[i][k]) : 0.f;
            }
            sp = warp_sum(sp);
            sn = warp_sum(sn);
            if (lane < NS)
                *reinterpret_cast<float4 *>(cluster.map_shared_rank(sb, lane) + (slice * kTC + t) * 4) =
                    make_float4(mx, sp, mn, sn);
        }
        cluster.sync();
        float zp[NV], zn[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) zp[k] = zn[k] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 4 * warp + i;
            // lane p < NS holds slice p's statistics
            const float4 o = lane < NS ? *reinterpret_cast<const float4 *>(sb + (lane * kTC + t) * 4)
                                       : make_float4(-INFINITY, 0.f, INFINITY, 0.f);
            const float mx = warp_max(o.x), mn = warp_min(o.z);
            const float sp = warp_sum(lane < NS ? o.y * expf(o.x - mx) : 0.f);
            const float sn = warp_sum(lane < NS ? o.w * expf(mn - o.z) : 0.f);
            const float ip = t < tc ? 1.f / sp : 0.f, in_ = t < tc ? 1.f / sn : 0.f;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const int fl = lane + 32 * k;
                if (fl < FS) {
                    const float p = expf(x[i][k] - mx) * ip, n = expf(mn - x[i][k]) * in_;
                    zp[k] += p;
                    zn[k] += n;
                    *reinterpret_cast<float2 *>(pd + (t * P2s + fl) * 2) = make_float2(p, p);
                    *reinterpret_cast<float2 *>(pd + (t * P2s + FS + fl) * 2) = make_float2(n, n);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < NV; ++k)
            if (lane + 32 * k < FS) {
                dzp[warp * P2s + lane + 32 * k] = zp[k];
                dzp[warp * P2s + FS + lane + 32 * k] = zn[k];
            }
        __syncthreads();
        if (owner) {
            const float *pq = pd + 8 * q, *ve = vs + e0;
            auto fold = [&](int t) {
                const ulonglong2 p01 = *reinterpret_cast<const ulonglong2 *>(pq + t * P2s * 2);
                const ulonglong2 p23 = *reinterpret_cast<const ulonglong2 *>(pq + t * P2s * 2 + 4);
                const ulonglong2 v03 = *reinterpret_cast<const ulonglong2 *>(ve + t * D);
                const ulonglong2 v47 = *reinterpret_cast<const ulonglong2 *>(ve + t * D + 4);
                const f32x2 pv[4] = {p01.x, p01.y, p23.x, p23.y}, vv2[4] = {v03.x, v03.y, v47.x, v47.y};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[4 * i + j] = ffma2(pv[i], vv2[j], acc[4 * i + j]);
            };
#pragma unroll 4
            for (int t = 0; t < kTC; ++t) fold(t);   // tokens beyond tc hold zeros
        }
        if (tid < P2s)
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) dz += dzp[w * P2s + tid];
        __syncthreads();   // K, V and phi of this chunk have been read
    }
    if (owner) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int sh = (j & 1) * 32;
            s4[j].x += __uint_as_float((uint32_t)(acc[0 + (j >> 1)] >> sh));
            s4[j].y += __uint_as_float((uint32_t)(acc[4 + (j >> 1)] >> sh));
            s4[j].z += __uint_as_float((uint32_t)(acc[8 + (j >> 1)] >> sh));
            s4[j].w += __uint_as_float((uint32_t)(acc[12 + (j >> 1)] >> sh));
            *reinterpret_cast<float4 *>(Sg + s_offset(f, e0 + j, D)) = s4[j];
        }
    }
    if (tid < P2s) Sg[z_offset(zf, D, F)] = z + dz;
}

template <int D, int FS>
cudaError_t launch_commit_fs(const CommitFmaArgs &a, int n_req, cudaStream_t st)
{
    static std::atomic<unsigned long long> opted{0};
    const unsigned ns = (unsigned)(a.F / FS);
    return launch_opted(&k_commit_fma<D, FS>, opted, (unsigned)(n_req * a.Hkv) * ns, commit_smem_bytes<D, FS>(), st, a,
                        ns);
}

}  // namespace

// ---------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------
cudaError_t launch_feature_map(hybrid_dtype dt, const void *X, int n_rows, int nh, int Hkv, int d,
                               int F, const void *W, float *Phi, cudaStream_t st)
{
    PhiArgs a{};
    a.X = X;
    a.W = W;
    a.Phi = Phi;
    a.nh = nh;
    a.group = nh / Hkv;
    a.rows = (long long)n_rows * a.group;
    a.d = d;
    a.F = F;
    a.bf16_io = dt == HYBRID_BF16;
    if (F <= 64) return launch_phi_f<0>(a, Hkv, st);
    if (F == 128) return launch_phi_f<1>(a, Hkv, st);
    return launch_phi_f<2>(a, Hkv, st);
}

cudaError_t launch_attn_generic(const hybrid_cfg &c, const void *Q, const void *K, const void *V,
                                const void *W, const float *alpha, void *const *states, int n_req,
                                void *O, unsigned *err, cudaStream_t st)
{
    AttnArgs a{};
    a.Q = Q;
    a.K = K;
    a.V = V;
    a.W = W;
    a.alpha = alpha;
    a.states = states;
    a.O = O;
    a.err = err;
    a.B = c.block_size;
    a.Hq = c.n_q_heads;
    a.Hkv = c.n_kv_heads;
    a.G = c.n_q_heads / c.n_kv_heads;
    a.F = c.feat_dim;
    a.bf16_io = c.io_dtype == HYBRID_BF16;
    const int rt = pick_rows((long long)n_req * a.Hkv, (long long)a.G * a.B, a.F <= 128);
    return c.head_dim == 64 ? launch_attn_d64(a, n_req, rt, st) : launch_attn_d128(a, n_req, rt, st);
}

cudaError_t launch_commit_generic(const hybrid_cfg &c, const void *K, const void *V, int n_tok,
                                  const void *W, void *const *states, int n_req, unsigned *err,
                                  cudaStream_t st)
{
    CommitFmaArgs a{};
    a.K = K;
    a.V = V;
    a.W = W;
    a.states = states;
    a.err = err;
    a.n_tok = n_tok;
    a.Hkv = c.n_kv_heads;
    a.F = c.feat_dim;
    a.bf16_io = c.io_dtype == HYBRID_BF16;
    if (c.head_dim == 64) {
        if (a.F == 16) return launch_commit_fs<64, 16>(a, n_req, st);
        if (a.F == 32) return launch_commit_fs<64, 32>(a, n_req, st);
        return launch_commit_fs<64, 64>(a, n_req, st);
    }
    return a.F == 16 ? launch_commit_fs<128, 16>(a, n_req, st) : launch_commit_fs<128, 32>(a, n_req, st);
}

}  // namespace hyb
