// kvx_simt.cu -- CUDA-core translation kernel.
//
// One CTA per (token tile, target head and 128 of its channels, target layer, K|V).  Three phases:
//   1. gather the span rows of the source heads feeding the target head (its GQA group, or every
//      head in the dense form, of one or several source layers), undo the source RoPE (K), take
//      the span mean -> A[tile][in] (fp32, shared memory);
//   2. projection A . W[j,h] with a register tile of TR tokens x 8 channels a thread; W passes
//      through shared memory 8 or 16 input rows at a time, the next ones on their way in registers;
//   3. the target RoPE (K) and the store, straight from the registers: a thread's 8 channels are 4
//      rotary pairs.
// It serves the float32 caches and any geometry the tensor-core kernel does not take.  Paper:
// Section 5 (T_theta per layer and KV head).
//
// Bound: shared-memory reads of W and A (70% of that pipe) and fp32 FMA issue (48% of the slots).  Each output is one accumulator in ascending input
// order.  1000 tokens of 7B -> 1.5B shapes (3.7 G FMA): 199 us; 608 us with a thread per output channel
// and scalar reads of A and W.
#include "kvx_common.cuh"
#include "kvx_kernels.h"
#include "kvx_schedule.h"

namespace kvx {

constexpr int kSimtPad = 4;         // floats between two rows of A: 16-byte reads of two rows miss each other's banks
constexpr int kSimtSmemMax = 200 * 1024;

// Register tile by slots per CTA (rotary pairs: 32 for d_t = 64, else 64): 4 slots (8 channels) a
// thread, so 8 or 16 threads across the channels and 16 or 8 groups of tokens.
constexpr int simt_groups(int slots) { return kSimtThreads / (slots / 4); }
// Input rows of W per shared-memory block: 8 under 32-token tiles, which leaves room for a fifth CTA an SM
// (199 us for the case above; 16 rows and four CTAs: 210), 16 under 16-token tiles, whose chain of blocks counts.
__host__ __device__ constexpr int simt_k(int tm) { return tm == 32 ? 8 : 16; }

// 4 consecutive elements; VEC: 16-byte aligned rows, else element by element.
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* p)
{
    if constexpr (VEC) return *reinterpret_cast<const float4*>(p);
    return make_float4(p[0], p[1], p[2], p[3]);
}
template <bool VEC>
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p)
{
    if constexpr (VEC) {
        const uint2 w = *reinterpret_cast<const uint2*>(p);
        return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                           __uint_as_float(w.y & 0xFFFF0000u));
    }
    return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
}
template <bool VEC>
__device__ __forceinline__ void store4(float* p, float4 x)
{
    if constexpr (VEC) *reinterpret_cast<float4*>(p) = x;
    else { p[0] = x.x; p[1] = x.y; p[2] = x.z; p[3] = x.w; }
}
template <bool VEC>
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 x)
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
    if constexpr (VEC) {
        *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    } else {
        p[0] = a.x; p[1] = a.y; p[2] = b.x; p[3] = b.y;
    }
}
// (c0, c1) += x (w0, w1): one packed instruction for two fp32 FMAs, each rounded as fmaf.  The packed
// form halves the issue slots of the projection (the case above with four CTAs an SM: 210 us, 236 with fmaf).
__device__ __forceinline__ void fma2(float& c0, float& c1, float x, float w0, float w1)
{
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b64 c, {%0, %1};\n\t"
        "fma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "+f"(c0), "+f"(c1)
        : "f"(x), "f"(w0), "f"(w1));
}
// R(-theta) of a pair (lo, hi): lo cos + hi sin, hi cos - lo sin
__device__ __forceinline__ void unrotate(float& lo, float& hi, float2 cs)
{
    const float a = lo, b = hi;
    lo = fmaf(a, cs.x, b * cs.y);
    hi = fmaf(b, cs.x, -a * cs.y);
}
// R(+theta)
__device__ __forceinline__ void rotate(float& lo, float& hi, float2 cs)
{
    const float a = lo, b = hi;
    lo = fmaf(a, cs.x, -b * cs.y);
    hi = fmaf(b, cs.x, a * cs.y);
}

template <typename T, int SLOTS, int TR, bool VEC>
__global__ void __launch_bounds__(kSimtThreads) translate_simt_kernel(const __grid_constant__ TranslateParams P)
{
    constexpr int CG = SLOTS / 4, RG = kSimtThreads / CG, TM = RG * TR, kSimtK = simt_k(TM);
    constexpr int WROW = 2 * SLOTS;                              // floats of one staged row of W
    constexpr int WPT = kSimtK * WROW / 4 / kSimtThreads;        // float4 of a staged block per thread
    extern __shared__ float smem[];
    __shared__ TokenInfo tinfo[TM];
    const int lda = P.in_dim + kSimtPad;
    float* A = smem;                     // [TM][lda]
    float* Ws = smem + TM * lda;         // [2][kSimtK][lo slots | hi slots]

    const int n_split = P.dt / WROW;
    const int h = blockIdx.y / n_split, a0 = (blockIdx.y - h * n_split) * SLOTS;   // first pair slot
    const int j = blockIdx.z >> 1;
    const int kv = blockIdx.z & 1;
    const int t0 = blockIdx.x * TM;
    const int ntok = min(TM, P.T_total - t0);
    const int tid = threadIdx.x;

    // W block b: rows [kSimtK b, kSimtK b + kSimtK), the CTA's channels, in registers until the block before is used
    const T* W = (const T*)P.w + ((size_t)(kv * P.Lt + j) * P.Ht + h) * (size_t)P.in_dim * P.dt;
    float4 wreg[WPT];
    int w_k[WPT], w_c[WPT], w_s[WPT];
#pragma unroll
    for (int i = 0; i < WPT; ++i) {
        const int it = tid + i * kSimtThreads, q = it % (WROW / 4) * 4;   // q: float of the staged row
        int c_lo, c_hi;
        pair_channels(a0 + q % SLOTS, P.dt >> 1, P.rhalf_t, c_lo, c_hi);
        w_k[i] = it / (WROW / 4);
        w_c[i] = q < SLOTS ? c_lo : c_hi;
        w_s[i] = w_k[i] * WROW + q;
    }
    auto load_w = [&](int b) {
#pragma unroll
        for (int i = 0; i < WPT; ++i) wreg[i] = load4<true>(W + (size_t)(b * kSimtK + w_k[i]) * P.dt + w_c[i]);
    };
    auto put_w = [&](int b) {
#pragma unroll
        for (int i = 0; i < WPT; ++i) *reinterpret_cast<float4*>(Ws + (b & 1) * kSimtK * WROW + w_s[i]) = wreg[i];
    };
    load_w(0);
    if (tid < ntok) tinfo[tid] = resolve_token(P, t0 + tid);
    __syncthreads();

    // ---- phase 1: un-rotate + span mean; one item = 4 pair slots of one token, all its head-blocks
    const bool rot_s = kv == 0 && P.rs.enabled;
    const int ncp = P.ds >> 3, heads = P.in_dim / P.ds;   // items per token; head-blocks of an input row
    for (int it = tid; it < TM * ncp; it += kSimtThreads) {
        const int tt = it / ncp, k = (it - tt * ncp) * 4;
        int c_lo, c_hi;
        pair_channels(k, P.ds >> 1, P.rhalf_s, c_lo, c_hi);
        float* row_a = A + tt * lda;
        if (tt >= ntok) {
            for (int q = 0; q < heads; ++q) {
                *reinterpret_cast<float4*>(row_a + q * P.ds + c_lo) = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4*>(row_a + q * P.ds + c_hi) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            continue;
        }
        const TokenInfo ti = tinfo[tt];
        const bool rot = rot_s && k < P.rhalf_s;
        const int n = ti.hi - ti.lo;
        const float nf = (float)n;
        float2 cs[4];
        if (rot && n == 1) {   // one (cos, sin) serves every head-block
            const int pos = src_pos_of(P, ti.b, ti.lo);
#pragma unroll
            for (int e = 0; e < 4; ++e) cs[e] = rope_cs(P.rs, pos, k + e);
        }
#pragma unroll 2
        for (int q = 0; q < heads; ++q) {
            int slot, g;
            head_block(P, j, h, q, slot, g);
            const T* base = (const T*)(kv ? P.src_v[slot] : P.src_k[slot]) + (long long)ti.b * P.sb + (long long)g * P.sh;
            float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
            for (int s = ti.lo; s < ti.hi; ++s) {
                const T* row = base + (long long)s * P.ss;
                float4 x = load4<VEC>(row + c_lo), y = load4<VEC>(row + c_hi);
                if (rot) {
                    if (n > 1) {
                        const int pos = src_pos_of(P, ti.b, s);
#pragma unroll
                        for (int e = 0; e < 4; ++e) cs[e] = rope_cs(P.rs, pos, k + e);
                    }
                    unrotate(x.x, y.x, cs[0]);
                    unrotate(x.y, y.y, cs[1]);
                    unrotate(x.z, y.z, cs[2]);
                    unrotate(x.w, y.w, cs[3]);
                }
                lo.x += x.x; lo.y += x.y; lo.z += x.z; lo.w += x.w;
                hi.x += y.x; hi.y += y.y; hi.z += y.z; hi.w += y.w;
            }
            if (n > 1) {
                lo.x /= nf; lo.y /= nf; lo.z /= nf; lo.w /= nf;
                hi.x /= nf; hi.y /= nf; hi.z /= nf; hi.w /= nf;
            }
            *reinterpret_cast<float4*>(row_a + q * P.ds + c_lo) = lo;
            *reinterpret_cast<float4*>(row_a + q * P.ds + c_hi) = hi;
        }
    }
    put_w(0);
    __syncthreads();

    // ---- phase 2: projection, fp32 accumulate in ascending input index
    const int cg = tid % CG, rg = tid / CG;
    float acc[TR][8];
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[u][e] = 0.f;
    const int nblk = P.in_dim / kSimtK;
    for (int b = 0; b < nblk; ++b) {
        if (b + 1 < nblk) load_w(b + 1);
        const float* ws = Ws + (b & 1) * kSimtK * WROW + cg * 4;
        const float* ar = A + rg * lda + b * kSimtK;
#pragma unroll
        for (int k0 = 0; k0 < kSimtK; k0 += 4) {
            float4 av[TR];
#pragma unroll
            for (int u = 0; u < TR; ++u) av[u] = *reinterpret_cast<const float4*>(ar + u * RG * lda + k0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 wl = *reinterpret_cast<const float4*>(ws + (k0 + k) * WROW);
                const float4 wh = *reinterpret_cast<const float4*>(ws + (k0 + k) * WROW + SLOTS);
#pragma unroll
                for (int u = 0; u < TR; ++u) {
                    const float x = k == 0 ? av[u].x : k == 1 ? av[u].y : k == 2 ? av[u].z : av[u].w;
                    fma2(acc[u][0], acc[u][1], x, wl.x, wl.y);
                    fma2(acc[u][2], acc[u][3], x, wl.z, wl.w);
                    fma2(acc[u][4], acc[u][5], x, wh.x, wh.y);
                    fma2(acc[u][6], acc[u][7], x, wh.z, wh.w);
                }
            }
        }
        if (b + 1 < nblk) put_w(b + 1);   // the other buffer: last read before the previous barrier
        __syncthreads();
    }

    // ---- phase 3: target RoPE + store
    T* dst = (T*)(kv ? P.dst_v[j] : P.dst_k[j]) + dst_head_off(P, h);
    const int k = a0 + cg * 4;
    const bool rot_t = kv == 0 && P.rt.enabled && k < P.rhalf_t;
    int c_lo, c_hi;
    pair_channels(k, P.dt >> 1, P.rhalf_t, c_lo, c_hi);
#pragma unroll
    for (int u = 0; u < TR; ++u) {
        const int tt = rg + u * RG;
        if (tt >= ntok || tinfo[tt].dst_off < 0) continue;
        if (rot_t) {
            const int pt = tinfo[tt].pt;
#pragma unroll
            for (int e = 0; e < 4; ++e) rotate(acc[u][e], acc[u][4 + e], rope_cs(P.rt, pt, k + e));
        }
        T* row = dst + tinfo[tt].dst_off;
        store4<VEC>(row + c_lo, make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]));
        store4<VEC>(row + c_hi, make_float4(acc[u][4], acc[u][5], acc[u][6], acc[u][7]));
    }
}

// Latent adapter product W = A . B per (target layer, head, K|V), once at translator creation:
// A [n][in][rank], B [n][rank][out] -> W [n][in][out], fp32 accumulation over rank in ascending
// order, rounded to T.  One thread per output element.
template <typename T>
__global__ void fold_low_rank_kernel(const T* __restrict__ a, const T* __restrict__ b, T* __restrict__ w, int n,
                                     int in_dim, int rank, int out)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per = (long long)in_dim * out;
    if (idx >= per * n) return;
    const int m = (int)(idx / per);
    const int rem = (int)(idx - (long long)m * per);
    const int i = rem / out, o = rem - i * out;
    const T* am = a + ((size_t)m * in_dim + i) * rank;
    const T* bm = b + (size_t)m * rank * out + o;
    float acc = 0.f;
    for (int c = 0; c < rank; ++c) acc = fmaf(to_f32<T>(am[c]), to_f32<T>(bm[(size_t)c * out]), acc);
    w[idx] = from_f32<T>(acc);
}

cudaError_t launch_fold_low_rank(const void* a, const void* b, void* w, int n, int in_dim, int rank, int out,
                                 int dtype, cudaStream_t stream)
{
    const long long total = (long long)n * in_dim * out;
    const unsigned blocks = (unsigned)((total + 255) / 256);
    if (dtype == KVX_BF16)
        fold_low_rank_kernel<__nv_bfloat16><<<blocks, 256, 0, stream>>>(
            (const __nv_bfloat16*)a, (const __nv_bfloat16*)b, (__nv_bfloat16*)w, n, in_dim, rank, out);
    else
        fold_low_rank_kernel<float><<<blocks, 256, 0, stream>>>((const float*)a, (const float*)b, (float*)w, n,
                                                                 in_dim, rank, out);
    return cudaGetLastError();
}

namespace {
size_t simt_smem(int in_dim, int slots, int tm)
{
    return ((size_t)tm * (in_dim + kSimtPad) + 2 * (size_t)simt_k(tm) * 2 * slots) * sizeof(float);
}
int simt_slots(int dt) { return dt == 64 ? 32 : 64; }

template <typename T, int SLOTS, int TR, bool VEC>
cudaError_t launch_simt_v(const TranslateParams& P, cudaStream_t stream)
{
    constexpr int TM = simt_groups(SLOTS) * TR;
    const size_t smem = simt_smem(P.in_dim, SLOTS, TM);
    // (also on every launch: the attribute is per device)
    const cudaError_t err = cudaFuncSetAttribute(translate_simt_kernel<T, SLOTS, TR, VEC>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kSimtSmemMax);
    if (err != cudaSuccess) return err;
    dim3 grid((P.T_total + TM - 1) / TM, P.Ht * (P.dt / (2 * SLOTS)), P.Lt * 2);
    translate_simt_kernel<T, SLOTS, TR, VEC><<<grid, kSimtThreads, smem, stream>>>(P);
    return cudaGetLastError();
}
template <typename T, int SLOTS, int TR>
cudaError_t launch_simt(const TranslateParams& P, bool vec, cudaStream_t stream)
{
    return vec ? launch_simt_v<T, SLOTS, TR, true>(P, stream) : launch_simt_v<T, SLOTS, TR, false>(P, stream);
}
template <typename T>
cudaError_t launch_simt_t(const TranslateParams& P, bool vec, bool big, cudaStream_t stream)
{
    if (simt_slots(P.dt) == 32)
        return big ? launch_simt<T, 32, 2>(P, vec, stream) : launch_simt<T, 32, 1>(P, vec, stream);
    return big ? launch_simt<T, 64, 4>(P, vec, stream) : launch_simt<T, 64, 2>(P, vec, stream);
}
}  // namespace

size_t simt_smem_bytes(int in_dim, int dt)
{
    const size_t big = simt_smem(in_dim, simt_slots(dt), 32);
    return big <= (size_t)kSimtSmemMax ? big : simt_smem(in_dim, simt_slots(dt), 16);
}

cudaError_t launch_translate_simt(const TranslateParams& P, int num_sms, int dtype, cudaStream_t stream)
{
    // 32 or 16 tokens a CTA: five CTAs of 32 tokens an SM overlap their phases (the case at the top: 199 us; two of 64
    // tokens and 128 threads 256, of 256 threads 227), and below two CTAs an SM the chain of one CTA counts
    const bool big = simt_tile_tokens(P.T_total, P.Ht, P.dt / (2 * simt_slots(P.dt)), P.Lt,
                                      simt_smem(P.in_dim, simt_slots(P.dt), 32) <= (size_t)kSimtSmemMax, num_sms) == 32;
    // the strides are whole 16-byte groups; the caches of the allocation-free entry may start anywhere
    uintptr_t a = 0;
    for (int i = 0; i < P.Lt * P.kl; ++i) a |= (uintptr_t)P.src_k[i] | (uintptr_t)P.src_v[i];
    for (int i = 0; i < P.Lt; ++i) a |= (uintptr_t)P.dst_k[i] | (uintptr_t)P.dst_v[i];
    const bool vec = (a & 15u) == 0;
    return dtype == KVX_BF16 ? launch_simt_t<__nv_bfloat16>(P, vec, big, stream)
                             : launch_simt_t<float>(P, vec, big, stream);
}

}  // namespace kvx
