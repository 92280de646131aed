// hybrid_state.cu -- zeroing and layout conversion of the per-request state.
//
// The state of one request is Hkv head blocks of S (2F x d) and z (2F),
// Section 3.1's S_n and Z_n, stored as documented in hybrid.h.
#include "hybrid_common.cuh"
#include "hybrid_kernels.h"
#include "tc_ptx.cuh"

namespace hyb {

// grid.x = n_req * chunks; zero 16-byte granules of each request's buffer
__global__ void k_state_init(void *const *__restrict__ states, int chunks, size_t n_gran)
{
    const int r = blockIdx.x / chunks;
    const size_t base = (size_t)(blockIdx.x % chunks) * blockDim.x * 8;
    float4 *p = reinterpret_cast<float4 *>(states[r]);
    if (!state_ptr_ok(p)) return;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const size_t i = base + (size_t)k * blockDim.x + threadIdx.x;
        if (i < n_gran) p[i] = zero;
    }
}

cudaError_t launch_state_init(const hybrid_cfg &c, void *const *states, int n_req, cudaStream_t st)
{
    const size_t n_gran = (size_t)c.n_kv_heads * head_floats(c.head_dim, c.feat_dim) / 4;
    const int threads = 256;
    const int chunks = (int)((n_gran + threads * 8 - 1) / (threads * 8));
    k_state_init<<<(unsigned)((long long)n_req * chunks), threads, 0, st>>>(states, chunks, n_gran);
    return cudaGetLastError();
}

// Pack and unpack: a thread turns one 4 x 4 block (4 features x 4 columns) in registers.
// Eight lanes take the eight 4-feature groups of a state tile and four the neighbouring
// column groups, so an image access is four whole 128-byte rows and a logical access eight
// pieces of 64 bytes.  One CTA per (request, state head, state tile).  What bounds it: the
// state is read and written once; 16 requests, 4 heads, d = F = 128 (8.4 MB in and out): the
// step and commit on logical states went from 46 us (an element per thread, its four-byte
// accesses scattered over the image) to 26 us.
//
// With a scratch base, request r's image is base + r * stride and the pointer array is
// written here too (hybrid_block_attn_commit_logical).  kVec: S is 16-byte
// aligned (4-byte accesses otherwise).
struct ConvertArgs {
    void *const *states;
    void **ptrs;               // written when base is set
    unsigned char *base;
    size_t stride;
    float *S, *z;
    unsigned *err;
    int Hkv, d, F, tiles;
};

template <bool kPack, bool kVec>
__global__ void __launch_bounds__(256) k_state_convert(const ConvertArgs a)
{
    const int d = a.d, F = a.F, P2 = 2 * F;
    const int tile = blockIdx.x % a.tiles, rh = blockIdx.x / a.tiles;
    const int r = rh / a.Hkv, g = rh % a.Hkv;
    ptx::griddep_launch_dependents();
    ptx::griddep_wait();
    float *st;
    if (a.base) {
        st = reinterpret_cast<float *>(a.base + (size_t)r * a.stride);
        if (kPack && threadIdx.x == 0 && tile == 0 && g == 0) a.ptrs[r] = st;
    } else {
        st = reinterpret_cast<float *>(a.states[r]);
        if (!state_ptr_ok(st)) {
            if (threadIdx.x == 0) raise_error(a.err, ERR_BAD_STATE_PTR);
            return;
        }
    }
    float *hb = st + (size_t)g * head_floats(d, F);
    float *Sl = a.S + (size_t)rh * P2 * d, *zl = a.z + (size_t)rh * P2;
    const int fq = threadIdx.x & 7, eq = threadIdx.x >> 3;
    if (4 * eq < d) {
        float *img = hb + (size_t)tile * 32 * d + (size_t)(4 * eq) * 32;
        float *lg = Sl + (size_t)(tile * 32 + 4 * fq) * d + 4 * eq;
        // granule fq of column 4 eq + i
        auto at = [&](int i) { return reinterpret_cast<float4 *>(img + i * 32 + ((fq ^ ((4 * eq + i) & 7)) << 2)); };
        auto ld = [&](const float *p) {
            if constexpr (kVec) return *reinterpret_cast<const float4 *>(p);
            else return make_float4(p[0], p[1], p[2], p[3]);
        };
        auto sto = [&](float *p, float x, float y, float z, float w) {
            if constexpr (kVec) {
                *reinterpret_cast<float4 *>(p) = make_float4(x, y, z, w);
            } else {
                p[0] = x;
                p[1] = y;
                p[2] = z;
                p[3] = w;
            }
        };
        if (kPack) {
            const float4 x0 = ld(lg), x1 = ld(lg + d), x2 = ld(lg + 2 * d), x3 = ld(lg + 3 * d);
            *at(0) = make_float4(x0.x, x1.x, x2.x, x3.x);
            *at(1) = make_float4(x0.y, x1.y, x2.y, x3.y);
            *at(2) = make_float4(x0.z, x1.z, x2.z, x3.z);
            *at(3) = make_float4(x0.w, x1.w, x2.w, x3.w);
        } else {
            const float4 x0 = *at(0), x1 = *at(1), x2 = *at(2), x3 = *at(3);
            sto(lg, x0.x, x1.x, x2.x, x3.x);
            sto(lg + d, x0.y, x1.y, x2.y, x3.y);
            sto(lg + 2 * d, x0.z, x1.z, x2.z, x3.z);
            sto(lg + 3 * d, x0.w, x1.w, x2.w, x3.w);
        }
    }
    if (tile == 0)
        for (int f = threadIdx.x; f < P2; f += 256) {
            if (kPack) hb[z_offset(f, d, F)] = zl[f];
            else zl[f] = hb[z_offset(f, d, F)];
        }
}

namespace {

template <bool kPack>
cudaError_t convert(const hybrid_cfg &c, void *const *states, unsigned char *base, void **ptrs, int n_req, float *S,
                    float *z, unsigned *err, cudaStream_t st)
{
    ConvertArgs a{};
    a.states = states;
    a.ptrs = ptrs;
    a.base = base;
    a.stride = (size_t)c.n_kv_heads * head_floats(c.head_dim, c.feat_dim) * sizeof(float);
    a.S = S;
    a.z = z;
    a.err = err;
    a.Hkv = c.n_kv_heads;
    a.d = c.head_dim;
    a.F = c.feat_dim;
    a.tiles = 2 * c.feat_dim / 32;
    const bool vec = (reinterpret_cast<uintptr_t>(S) & 15u) == 0;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((long long)n_req * a.Hkv * a.tiles));
    lc.blockDim = dim3(256);
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return vec ? cudaLaunchKernelEx(&lc, k_state_convert<kPack, true>, a)
               : cudaLaunchKernelEx(&lc, k_state_convert<kPack, false>, a);
}

}  // namespace

cudaError_t launch_state_unpack(const hybrid_cfg &c, void *const *states, int n_req, float *S,
                                float *z, unsigned *err, cudaStream_t st)
{
    return convert<false>(c, states, nullptr, nullptr, n_req, S, z, err, st);
}

cudaError_t launch_state_pack(const hybrid_cfg &c, const float *S, const float *z,
                              void *const *states, int n_req, unsigned *err, cudaStream_t st)
{
    return convert<true>(c, states, nullptr, nullptr, n_req, const_cast<float *>(S), const_cast<float *>(z), err, st);
}

cudaError_t launch_scratch_pack(const hybrid_cfg &c, const float *S, const float *z, unsigned char *base, void **ptrs,
                                int n_req, cudaStream_t st)
{
    return convert<true>(c, nullptr, base, ptrs, n_req, const_cast<float *>(S), const_cast<float *>(z), nullptr, st);
}

cudaError_t launch_scratch_unpack(const hybrid_cfg &c, unsigned char *base, int n_req, float *S, float *z,
                                  cudaStream_t st)
{
    return convert<false>(c, nullptr, base, nullptr, n_req, S, z, nullptr, st);
}

}  // namespace hyb
