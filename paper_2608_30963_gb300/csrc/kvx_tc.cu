// kvx_tc.cu -- the window kernel: tensor-core translation over windows of source rows (kvx_tc_window.cuh).
//
// It serves what the row-gather kernel (kvx_tc_rows.cu) does not take: units of several heads (the
// dense form), partial rotary heads, and input widths that are not one or several groups of 256.
#include "kvx_tc_window.cuh"

namespace kvx {
namespace {

using namespace window;

template <int DS, bool MULTI>
__global__ void __launch_bounds__(kThreads, 1)
translate_tc_kernel(const __grid_constant__ TranslateParams P, const __grid_constant__ TcLaunch L)
{
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned base, derived from smem_raw by pointer arithmetic so that the
    // compiler keeps every access in the shared address space
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    translate_body<DS, MULTI, true>(P, L, smem, 0);
}

// Span plan of the sub-tiles of target tokens [t_begin, t_end): one warp per
// 32-token sub-tile, one lane per token (layout: see the comment at the top).  Every
// sub-tile of the launch's 128-token tiles gets a header and 32 entries; those past
// the end get an empty window and entries marked past the end.
__global__ void __launch_bounds__(128) span_plan_kernel(const __grid_constant__ TranslateParams P, int t_begin,
                                                        int t_end, int cap_rows, int4* __restrict__ hdr,
                                                        int4* __restrict__ ent)
{
    // the previous launch in the stream may still read the plan buffer
    grid_dependency_wait();
    grid_launch_dependents();
    const int sub = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    const int nsub = (t_end - t_begin + kTileM - 1) / kTileM * kSubPerTile;
    if (sub >= nsub) return;
    const SeqView sv{P.seq_off, P.src_seq_len, P.batch};
    const int tp = t_begin + sub * kSub + lane;
    const bool valid = tp < t_end;
    int b = -1, lo = 0, hi = 0;
    if (valid) resolve_src(P, sv, tp, load_span(P, tp), b, lo, hi);
    write_window_plan(valid, b, lo, hi, sub, lane, cap_rows, hdr, ent);
}

// Weight images: for group g = ((j*Ht + h)*2 + kv)*n_split + nt, the B operand
// [n_tile rows = output columns][in] in K-major SW128 layout.  Image row n holds pair
// slot k = nt*hw + (n mod hw): its first channel for n < hw, its partner above
// (pair_channels: (k, k + d_t/2), or the partial rotary pairing), so an image holds
// whole RoPE pairs and the epilogue rotates columns n and n + hw together.
__global__ void tc_weight_relayout_kernel(const __nv_bfloat16* __restrict__ wk, const __nv_bfloat16* __restrict__ wv,
                                          uint8_t* __restrict__ img, int Lt, int Ht, int in_dim, int dt, int n_tile,
                                          int rhalf_t)
{
    const int n_split = dt / n_tile, hw = n_tile / 2;
    const long long chunks_per_img = (long long)n_tile * in_dim / 8;
    const long long total = (long long)Lt * Ht * 2 * n_split * chunks_per_img;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int gimg = (int)(idx / chunks_per_img);
    const int c = (int)(idx - (long long)gimg * chunks_per_img);   // chunk within image
    int rest = gimg;
    const int nt = rest % n_split; rest /= n_split;
    const int kv = rest & 1; rest >>= 1;
    const int h = rest % Ht;
    const int j = rest / Ht;
    // chunk c enumerates (n, k/8) with k fastest
    const int n = c / (in_dim / 8);
    const int k8 = c - n * (in_dim / 8);
    int c_lo, c_hi;
    pair_channels(nt * hw + (n < hw ? n : n - hw), dt / 2, rhalf_t, c_lo, c_hi);
    const int col = n < hw ? c_lo : c_hi;
    const __nv_bfloat16* w = (kv ? wv : wk) + ((size_t)j * Ht + h) * (size_t)in_dim * dt;
    uint32_t v[4];
    for (int e = 0; e < 4; ++e) {
        const int k = k8 * 8 + 2 * e;
        const __nv_bfloat16 lo = w[(size_t)k * dt + col];
        const __nv_bfloat16 hi = w[(size_t)(k + 1) * dt + col];
        v[e] = (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
    }
    const int k = k8 * 8;
    const size_t off = (size_t)gimg * ((size_t)n_tile * in_dim * 2) + (size_t)(k >> 6) * n_tile * 128 +
                       (size_t)(n >> 3) * 1024 + (n & 7) * 128 + ((((k >> 3) & 7) ^ (n & 7)) << 4);
    *reinterpret_cast<uint4*>(img + off) = make_uint4(v[0], v[1], v[2], v[3]);
}

// the B-loader warp (the last one) only when the weights stream
int tc_threads(const TcLaunch& L) { return L.n_b > 1 ? kThreads : kThreads - 32; }

}  // namespace

TcConfig tc_config(int in_dim, int dt, int ds, int share)
{
    TcLaunch L{};
    TcConfig c{0, 0, 0, kThreads, 0, 1};
    if (!tc_layout(in_dim, dt, ds, share, L)) return c;
    c.n_tile = L.n_tile;
    c.n_split = L.n_split;
    c.smem_bytes = kSmemMax;
    c.threads = tc_threads(L);
    c.hpu = L.hpu;
    c.ok = 1;
    return c;
}

size_t tc_weight_image_bytes(int in_dim, int dt, int Lt, int Ht)
{
    return (size_t)Lt * Ht * 2 * (size_t)in_dim * dt * 2;
}

cudaError_t launch_tc_weight_relayout(const void* w_k, const void* w_v, void* image, int Lt, int Ht, int in_dim,
                                      int dt, int n_tile, int rhalf_t, cudaStream_t stream)
{
    const long long total = (long long)Lt * Ht * 2 * dt * in_dim / 8;
    const int threads = 256;
    tc_weight_relayout_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, stream>>>(
        (const __nv_bfloat16*)w_k, (const __nv_bfloat16*)w_v, (uint8_t*)image, Lt, Ht, in_dim, dt, n_tile, rhalf_t);
    return cudaGetLastError();
}

template <int DS, bool MULTI>
static cudaError_t launch_span_ds(int grid, cudaStream_t stream, const TranslateParams& P, const TcLaunch& L)
{
    const cudaError_t e = smem_opt_in<translate_tc_kernel<DS, MULTI>>(kSmemMax);
    if (e != cudaSuccess) return e;
    return launch_pdl(translate_tc_kernel<DS, MULTI>, grid, tc_threads(L), kSmemMax, stream, P, L);
}
template <int DS>
static cudaError_t launch_span(int grid, cudaStream_t stream, const TranslateParams& P, const TcLaunch& L)
{
    return L.np > 1 ? launch_span_ds<DS, true>(grid, stream, P, L) : launch_span_ds<DS, false>(grid, stream, P, L);
}

size_t tc_plan_bytes(int tokens)
{
    const size_t nsub = (size_t)(tokens + kSub - 1) / kSub;
    return nsub * sizeof(int4) * (1 + kSub);
}

void tc_plan_layout(int T_total, int plan_tokens, int* nsub, int* ent_off)
{
    const int chunk = plan_tokens / kTileM * kTileM;
    *ent_off = (chunk + kSub - 1) / kSub;
    *nsub = 0;
    if (chunk <= 0 || T_total <= 0) return;
    const int last = (T_total - 1) / chunk * chunk;   // first token of the last chunk
    *nsub = (T_total - last + kTileM - 1) / kTileM * kSubPerTile;
}

cudaError_t launch_translate_tc(const TranslateParams& P, const TcConfig& cfg, int num_sms, void* plan,
                                int plan_tokens, cudaStream_t stream, int* launches)
{
    *launches = 0;
    TcLaunch L{};
    if (!tc_layout(P.in_dim, P.dt, P.ds, share_heads(P), L)) return cudaErrorNotSupported;
    if (P.ds != 64 && P.ds != 128 && P.ds != 256) return cudaErrorNotSupported;
    const int chunk = plan_tokens / kTileM * kTileM;
    if (chunk <= 0 || !plan) return cudaErrorInvalidValue;
    int4* hdr = reinterpret_cast<int4*>(plan);
    int4* ent = hdr + (chunk + kSub - 1) / kSub;
    // one plan + one translation launch per chunk of at most plan_tokens target tokens
    for (int t0 = 0; t0 < P.T_total; t0 += chunk) {
        const int t1 = P.T_total - t0 < chunk ? P.T_total : t0 + chunk;
        const int grid = tc_launch(P, t0, t1, hdr, ent, num_sms, L);
        const int nsub = L.m_tiles * kSubPerTile;
        cudaError_t e = launch_pdl(span_plan_kernel, (nsub + 3) / 4, 128, 0, stream, P, t0, t1, (int)L.cap_rows, hdr, ent);
        if (e != cudaSuccess) return e;
        ++*launches;
        switch (P.ds) {
        case 256: e = launch_span<256>(grid, stream, P, L); break;
        case 128: e = launch_span<128>(grid, stream, P, L); break;
        default: e = launch_span<64>(grid, stream, P, L); break;
        }
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    (void)cfg;
    return cudaSuccess;
}

}  // namespace kvx
