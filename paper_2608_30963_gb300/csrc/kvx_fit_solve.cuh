// kvx_fit_solve.cuh -- blocked Cholesky solve of the fit's normal equations, in <= 256 (library-internal).
//
// Every group g is a system (X^T X + lambda I) W = X^T Y of `in` unknowns (a multiple of 32) and
// dt right-hand sides.  Two launches in 32 x 32 blocks:
//   fit_factor_kernel  one CTA per group: L L^T = X^T X + lambda I, right-looking.  Per block column the
//                      CTA factors the diagonal block in shared memory and inverts its factor in the
//                      same 32 steps; then one warp per 32 x 32 block multiplies the blocks below by the
//                      inverse and applies the rank-32 update (a 4 x 8 tile a lane).
//   fit_trsm_kernel    one warp per 8 right-hand sides of a group: L U = C, then L^T W = U, left-looking
//                      with the inverted diagonal blocks, so every step is a small matrix product.
// The blocks of L live in global scratch (352 KB a group at in = 256); the solves pass them through
// shared memory, three in flight, for the warps of a CTA together.
//
// Bound: the chain of block columns of one group (the factor) and FMA issue (the solves).  All loops
// are kept rolled and small: with the diagonal block and the rows below it unrolled in registers,
// instruction fetch was most of the factor's time.
// Measured, factor and solves: 112 systems of 256 x 128 in fp32 151 and 122 us (2.0 ms with an unblocked
// factor and one thread per right-hand side); 208 systems of 128 x 256 in pairs 220 and 464 us, the
// latter near the fp32 pipe's rate (its scaling included).
//
// Arithmetic is a parameter.  F32: fp32, for systems the pivots show to be well conditioned.  Pair:
// unevaluated sums h + l of two floats (about 48 bits), products exact by FMA (Dekker's two-product) and
// sums by Knuth's two-sum, for the others: GB300 runs 64 fp32 FMAs for one fp64 FMA, so the twelve
// fp32 operations of a pair multiply-add cost a fifth of one fp64 FMA.
//
// Pair systems are scaled first: S (X^T X + lambda I) S, S^-1 W and S X^T Y with powers of two that bring the
// diagonal into [1/2, 2), and every right-hand side to a largest element in [1, 2).  The scaling is exact, and a
// Cholesky solve's rounding errors do not depend on it, but the low words of a pair keep their bits only above 2^-102,
// so without it systems of small sums (channels of 1e-16 and below) would fall back to fp32.  It also makes the
// pivots show what the pairs have to resolve: channel scales do not count, nearly dependent channels do.
// Systems whose scaled pivots show a condition number above max_cond go to the double kernel: 48 bits begin to show
// in W there.
#pragma once

#include <climits>

#include "kvx_common.cuh"

namespace kvx {
namespace {

constexpr int kSolveBlk = 32;
constexpr int kFactorThreads = 256;
constexpr int kTrsmWarps = 4;   // 32 right-hand sides a CTA: 448 CTAs for 112 groups spread evenly over 152 SMs (122 us; 64 a CTA: 149)
constexpr int kTrsmStages = 3;  // blocks of L in shared memory
constexpr int kTrsmCols = 8;    // right-hand sides per warp

struct F32 {
    static constexpr int PL = 1;   // planes of a stored block
    float h;
    __device__ static F32 make(float x) { return F32{x}; }
    __device__ static F32 load(const float* p, int) { return F32{*p}; }
    __device__ void store(float* p, int) const { *p = h; }
    __device__ void sub_mul(F32 a, F32 b) { h = fmaf(-a.h, b.h, h); }   // *this -= a b
    __device__ void norm() {}
    __device__ F32 neg() const { return F32{-h}; }
    __device__ F32 add(float x) const { return F32{h + x}; }
    __device__ F32 root() const { return F32{sqrtf(h)}; }
    __device__ F32 inverse() const { return F32{1.f / h}; }
    __device__ F32 times(F32 x) const { return F32{h * x.h}; }
    __device__ float value() const { return h; }
};

// Twice-working-precision value h + l, |l| <= ulp(h)/2 after norm().
struct Pair {
    static constexpr int PL = 2;
    float h, l;
    __device__ static Pair make(float x) { return Pair{x, 0.f}; }
    __device__ static Pair load(const float* p, int plane) { return Pair{p[0], p[plane]}; }
    __device__ void store(float* p, int plane) const { p[0] = h; p[plane] = l; }
    __device__ void two_sum(float x)   // h + x exactly: the sum in h, its rounding error added to l
    {
        const float s = __fadd_rn(h, x), bb = __fsub_rn(s, h);
        l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
        h = s;
    }
    __device__ void sub_mul(Pair a, Pair b)
    {
        const float p = __fmul_rn(-a.h, b.h);
        float e = __fmaf_rn(-a.h, b.h, -p);
        e = __fmaf_rn(-a.h, b.l, e);
        e = __fmaf_rn(-a.l, b.h, e);
        two_sum(p);
        l = __fadd_rn(l, e);
    }
    __device__ void norm()
    {
        const float s = __fadd_rn(h, l);
        l = __fsub_rn(l, __fsub_rn(s, h));
        h = s;
    }
    __device__ Pair neg() const { return Pair{-h, -l}; }
    __device__ Pair add(float x) const
    {
        Pair r = *this;
        r.two_sum(x);
        r.norm();
        return r;
    }
    __device__ Pair root() const   // one Newton step on sqrtf
    {
        const float s = sqrtf(h);
        const float r = __fadd_rn(__fmaf_rn(-s, s, h), l);
        Pair y{s, r / (2.f * s)};
        y.norm();
        return y;
    }
    __device__ Pair inverse() const   // one Newton step on 1 / h
    {
        const float q = 1.f / h;
        const float r = __fmaf_rn(-q, l, __fmaf_rn(-q, h, 1.f));
        Pair y{q, __fmul_rn(q, r)};
        y.norm();
        return y;
    }
    __device__ Pair times(Pair x) const
    {
        const float p = __fmul_rn(h, x.h);
        float e = __fmaf_rn(h, x.h, -p);
        e = __fmaf_rn(h, x.l, e);
        e = __fmaf_rn(l, x.h, e);
        Pair y{p, e};
        y.norm();
        return y;
    }
    __device__ float value() const { return h + l; }
};

// Scratch of one group, blocks of S::PL planes of 32 x 32 floats:
//   F(I, J), I >= J   L's block, element (r, c) at c * 32 + r   (products with L)
//   B(I, J)           the same block, (r, c) at r * 32 + c      (products with L^T)
//   FI(k), BI(k)      the inverse of diagonal block k, both ways
__host__ __device__ inline size_t solve_blocks(int in)
{
    const size_t nb = in / kSolveBlk;
    return nb * (nb + 1) + 2 * nb;
}
template <class S>
struct Blocks {
    float* base;
    int nb;
    static constexpr int SZ = S::PL * kSolveBlk * kSolveBlk;
    __device__ float* F(int i, int j) const { return base + (size_t)(i * (i + 1) / 2 + j) * SZ; }
    __device__ float* B(int i, int j) const { return base + (size_t)(nb * (nb + 1) / 2 + i * (i + 1) / 2 + j) * SZ; }
    __device__ float* FI(int k) const { return base + (size_t)(nb * (nb + 1) + k) * SZ; }
    __device__ float* BI(int k) const { return base + (size_t)(nb * (nb + 1) + nb + k) * SZ; }
};
constexpr int kPlane = kSolveBlk * kSolveBlk;

// Exponent of unknown r's scaling factor, from the diagonal of its system (Pair).
__device__ __forceinline__ int scale_exponent(float g_rr, double lambda)
{
    const double d = (double)g_rr + lambda;
    if (!(d > 0.0) || isinf(d)) return 0;
    return -((ilogb(d) + 1) >> 1);   // d 2^(2e) in [1/2, 2)
}

// Four consecutive values of a block.
template <class S>
__device__ __forceinline__ void load4(const float* p, S (&x)[4])
{
    const float4 h = *reinterpret_cast<const float4*>(p);
    x[0].h = h.x; x[1].h = h.y; x[2].h = h.z; x[3].h = h.w;
    if constexpr (S::PL == 2) {
        const float4 l = *reinterpret_cast<const float4*>(p + kPlane);
        x[0].l = l.x; x[1].l = l.y; x[2].l = l.z; x[3].l = l.w;
    }
}
template <class S>
__device__ __forceinline__ void store4(float* p, const S (&x)[4])
{
    *reinterpret_cast<float4*>(p) = make_float4(x[0].h, x[1].h, x[2].h, x[3].h);
    if constexpr (S::PL == 2) *reinterpret_cast<float4*>(p + kPlane) = make_float4(x[0].l, x[1].l, x[2].l, x[3].l);
}

// flags[g]: 0 solved here, kSolveRedo ill-conditioned (left to the Pair kernels), kSolveDouble left to the
// double kernel, kSolveBroken too: a pivot was not positive.  The F32 pass writes every flag and counts the redo
// groups in counts[0]; the Pair pass works on those only.  What either leaves to the double kernel is counted in
// counts[1]; that kernel alone declares a system not positive definite.
constexpr int kSolveRedo = 1, kSolveDouble = 2, kSolveBroken = 3;

// acc -= A B^T over one 32 x 32 block pair; a, b: this lane's first row and column of blocks stored
// (r, p) at p * 32 + r.
template <class S>
__device__ __forceinline__ void block_product(S (&acc)[8][4], const float* a, const float* b)
{
#pragma unroll 2
    for (int p = 0; p < kSolveBlk; ++p) {
        S x[4], y[2][4];
        load4(a + p * kSolveBlk, x);
        load4(b + p * kSolveBlk, y[0]);
        load4(b + p * kSolveBlk + 4, y[1]);
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[c][r].sub_mul(x[r], y[c >> 2][c & 3]);
    }
}

template <class S>
__global__ void __launch_bounds__(kFactorThreads, 2) fit_factor_kernel(const float* G, float* scratch, int in, double lambda,
                                                                       float max_cond, int* counts, int* flags)
{
    constexpr bool kRedo = S::PL == 2;
    constexpr int kPitch = kSolveBlk + 1, kArea = kSolveBlk * kPitch, kWarps = kFactorThreads / 32;
    // Diagonal block (r, c) at c * kPitch + r, the rows of its factor's inverse (r, c) at r * kPitch + c
    // before their scaling, both in place; planes kArea apart.
    __shared__ float sh[2 * S::PL * kArea];
    __shared__ float sPiv[256];
    __shared__ int sExp[kRedo ? 256 : 1];
    __shared__ int sBad;
    float *sD = sh, *sE = sh + S::PL * kArea;
    const int g = blockIdx.x;
    if (kRedo && flags[g] != kSolveRedo) return;
    const int nb = in / kSolveBlk, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Blocks<S> L{scratch + (size_t)g * solve_blocks(in) * Blocks<S>::SZ, nb};
    const float* gg = G + (size_t)g * in * in;
    if (threadIdx.x == 0) sBad = 0;
    if (kRedo) {
        for (int r = threadIdx.x; r < in; r += kFactorThreads) sExp[r] = scale_exponent(gg[(size_t)r * in + r], lambda);
        __syncthreads();
    }
    // lower blocks of X^T X: element (r, c) of the sums is at c * in + r, as in the blocks
    for (int t = warp; t < nb * (nb + 1) / 2; t += kWarps) {
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= t) ++i;
        const int j = t - i * (i + 1) / 2;
        const float* from = gg + (size_t)j * kSolveBlk * in + i * kSolveBlk + lane;
        float* f = L.F(i, j) + lane;
        float x[kSolveBlk];   // all loads before the first store, which might alias them
#pragma unroll
        for (int c = 0; c < kSolveBlk; ++c) x[c] = from[(size_t)c * in];
#pragma unroll
        for (int c = 0; c < kSolveBlk; ++c) {
            if (kRedo) x[c] = ldexpf(x[c], sExp[i * kSolveBlk + lane] + sExp[j * kSolveBlk + c]);
            S::make(x[c]).store(f + c * kSolveBlk, kPlane);
        }
    }
    __syncthreads();

    const int dr = threadIdx.x >> 3, dc = threadIdx.x & 7;   // diagonal block: row, columns dc + 8 i
    const int r0 = (lane & 7) * 4, c0 = (lane >> 3) * 8;     // block products: 4 rows x 8 columns a lane
    for (int k = 0; k < nb; ++k) {
        {   // diagonal block with lambda, and the unit matrix
            const float* d = L.F(k, k);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = dc + 8 * i;
                S v = S::load(d + c * kSolveBlk + dr, kPlane);
                if (c == dr) {
                    const double l = kRedo ? ldexp(lambda, 2 * sExp[k * kSolveBlk + c]) : lambda;
                    v = v.add((float)l);
                    if (kRedo) v = v.add((float)(l - (double)(float)l));
                }
                v.store(sD + c * kPitch + dr, kArea);
                S::make(c == dr ? 1.f : 0.f).store(sE + dr * kPitch + c, kArea);
            }
        }
        __syncthreads();
        // step p: column p of L = column p / sqrt(pivot), row p of the inverse likewise; later rows lose
        // their multiples of both.  Column and row p are only read, the rest only written.
#pragma unroll 1
        for (int p = 0; p < kSolveBlk; ++p) {
            S piv = S::load(sD + p * kPitch + p, kArea);
            if (!(piv.value() > 0.f)) {
                piv = S::make(1.f);
                if (threadIdx.x == 0) sBad = 1;
            }
            const S root = piv.root(), inv = root.inverse();
            if (threadIdx.x == 0) sPiv[k * kSolveBlk + p] = root.value();
            if (dr > p) {
                const S lr = S::load(sD + p * kPitch + dr, kArea).times(inv);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int c = dc + 8 * i;
                    if (c > dr) continue;
                    float* at = c > p ? sD + c * kPitch + dr : sE + dr * kPitch + c;
                    const S other = S::load(c > p ? sD + p * kPitch + c : sE + p * kPitch + c, kArea).times(inv);
                    S v = S::load(at, kArea);
                    v.sub_mul(lr, other);
                    v.norm();
                    v.store(at, kArea);
                }
            }
            __syncthreads();
        }
        // the inverse, its rows scaled: (r, c) both ways
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = dc + 8 * i;
            S piv = S::load(sD + dr * kPitch + dr, kArea);
            if (!(piv.value() > 0.f)) piv = S::make(1.f);
            const S v = c <= dr ? S::load(sE + dr * kPitch + c, kArea).times(piv.root().inverse()) : S::make(0.f);
            v.store(L.FI(k) + c * kSolveBlk + dr, kPlane);
            v.store(L.BI(k) + dr * kSolveBlk + c, kPlane);
        }
        __syncthreads();
        // blocks below: L(i, k) = A(i, k) inverse^T
        for (int i = k + 1 + warp; i < nb; i += kWarps) {
            S acc[8][4];
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[c][r] = S::make(0.f);
            float *f = L.F(i, k), *bt = L.B(i, k);
            block_product(acc, f + r0, L.FI(k) + c0);
            __syncwarp();   // the block is overwritten
#pragma unroll
            for (int c = 0; c < 8; ++c) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    acc[c][r].norm();
                    acc[c][r] = acc[c][r].neg();
                    acc[c][r].store(bt + (r0 + r) * kSolveBlk + c0 + c, kPlane);
                }
                store4(f + (c0 + c) * kSolveBlk + r0, acc[c]);
            }
        }
        __syncthreads();
        // rank-32 update of the blocks to the right
        const int m = nb - 1 - k;
        for (int t = warp; t < m * (m + 1) / 2; t += kWarps) {
            int i = 0;
            while ((i + 1) * (i + 2) / 2 <= t) ++i;
            const int j = t - i * (i + 1) / 2;
            float* out = L.F(k + 1 + i, k + 1 + j) + c0 * kSolveBlk + r0;
            S acc[8][4];
#pragma unroll
            for (int c = 0; c < 8; ++c) load4(out + c * kSolveBlk, acc[c]);
            block_product(acc, L.F(k + 1 + i, k) + r0, L.F(k + 1 + j, k) + c0);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[c][r].norm();
                store4(out + c * kSolveBlk, acc[c]);
            }
        }
        __syncthreads();
    }
    if (warp == 0) {
        float dmin = sPiv[0], dmax = sPiv[0];
        for (int c = lane; c < in; c += 32) {
            dmin = fminf(dmin, sPiv[c]);
            dmax = fmaxf(dmax, sPiv[c]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
            dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        }
        if (lane == 0) {
            const float ratio = dmax / dmin;
            const bool ill = ratio * ratio > max_cond;
            const int to_double = sBad ? kSolveBroken : kRedo && ill ? kSolveDouble : 0;
            if (to_double) {
                flags[g] = to_double;
                atomicAdd(counts + 1, 1);
            } else if (!kRedo) {
                flags[g] = ill ? kSolveRedo : 0;
                if (ill) atomicAdd(counts, 1);
            }
        }
    }
}

// Two floats in one register pair, and the packed instructions on them: each half rounds as its scalar
// form does, at half the issue slots.
struct F2 {
    unsigned long long v;
    __device__ static F2 make(float x, float y)
    {
        F2 r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
        return r;
    }
    __device__ void get(float& x, float& y) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
};
__device__ __forceinline__ F2 add2(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// One row of a block row of the solutions, kTrsmCols columns: acc -= L[row][p] z[p], as F32 or Pair does it.
template <class S> struct TrsmRow;
template <> struct TrsmRow<F32> {
    F2 h[kTrsmCols / 2];
    __device__ void load(const float* z, int)
    {
#pragma unroll
        for (int q = 0; q < kTrsmCols / 4; ++q) {
            const float4 x = reinterpret_cast<const float4*>(z)[q];
            h[2 * q] = F2::make(x.x, x.y);
            h[2 * q + 1] = F2::make(x.z, x.w);
        }
    }
    __device__ void zero()
    {
#pragma unroll
        for (int c = 0; c < kTrsmCols / 2; ++c) h[c].v = 0;
    }
    __device__ void sub_mul(const float* l, const float* z, int)
    {
        const F2 a = F2::make(-*l, -*l);
#pragma unroll
        for (int c = 0; c < kTrsmCols / 4; ++c) {
            const float4 b = reinterpret_cast<const float4*>(z)[c];
            h[2 * c] = fma2(a, F2::make(b.x, b.y), h[2 * c]);
            h[2 * c + 1] = fma2(a, F2::make(b.z, b.w), h[2 * c + 1]);
        }
    }
    __device__ void store(float* z, int, bool neg) const
    {
        const float f = neg ? -1.f : 1.f;
#pragma unroll
        for (int q = 0; q < kTrsmCols / 4; ++q) {
            float4 x;
            h[2 * q].get(x.x, x.y);
            h[2 * q + 1].get(x.z, x.w);
            reinterpret_cast<float4*>(z)[q] = make_float4(f * x.x, f * x.y, f * x.z, f * x.w);
        }
    }
};
template <> struct TrsmRow<Pair> {
    F2 h[kTrsmCols / 2], l[kTrsmCols / 2];
    __device__ void load(const float* z, int plane)
    {
#pragma unroll
        for (int q = 0; q < kTrsmCols / 4; ++q) {
            const float4 x = reinterpret_cast<const float4*>(z)[q], y = reinterpret_cast<const float4*>(z + plane)[q];
            h[2 * q] = F2::make(x.x, x.y);
            h[2 * q + 1] = F2::make(x.z, x.w);
            l[2 * q] = F2::make(y.x, y.y);
            l[2 * q + 1] = F2::make(y.z, y.w);
        }
    }
    __device__ void zero()
    {
#pragma unroll
        for (int c = 0; c < kTrsmCols / 2; ++c) h[c].v = l[c].v = 0;
    }
    __device__ void sub_mul(const float* lp, const float* z, int plane)
    {
        const F2 lh = F2::make(lp[0], lp[0]), ah = F2::make(-lp[0], -lp[0]), al = F2::make(-lp[kPlane], -lp[kPlane]);
        const F2 minus = F2::make(-1.f, -1.f);
        auto sub2 = [&](F2 a, F2 b) { return fma2(b, minus, a); };   // a - b, rounded once
#pragma unroll
        for (int q = 0; q < kTrsmCols / 4; ++q) {
            const float4 zh = reinterpret_cast<const float4*>(z)[q], zl = reinterpret_cast<const float4*>(z + plane)[q];
            const F2 bh[2] = {F2::make(zh.x, zh.y), F2::make(zh.z, zh.w)}, bl[2] = {F2::make(zl.x, zl.y), F2::make(zl.z, zl.w)};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int c = 2 * q + u;
                // Pair::sub_mul: the product p and its error, the cross terms, Knuth's two-sum (np = -p)
                const F2 np = mul2(lh, bh[u]);
                const F2 e = fma2(al, bh[u], fma2(ah, bl[u], fma2(ah, bh[u], np)));
                const F2 s = sub2(h[c], np), bb = sub2(s, h[c]);
                const F2 t = sub2(sub2(h[c], sub2(s, bb)), add2(np, bb));
                h[c] = s;
                l[c] = add2(l[c], add2(t, e));
            }
        }
    }
    __device__ void store(float* z, int plane, bool neg) const
    {
        const float f = neg ? -1.f : 1.f;
#pragma unroll
        for (int q = 0; q < kTrsmCols / 4; ++q) {
            Pair x[4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                h[2 * q + u].get(x[2 * u].h, x[2 * u + 1].h);
                l[2 * q + u].get(x[2 * u].l, x[2 * u + 1].l);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u].norm();
            reinterpret_cast<float4*>(z)[q] = make_float4(f * x[0].h, f * x[1].h, f * x[2].h, f * x[3].h);
            reinterpret_cast<float4*>(z + plane)[q] = make_float4(f * x[0].l, f * x[1].l, f * x[2].l, f * x[3].l);
        }
    }
};

__device__ __forceinline__ void copy16(float* dst, const float* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// G, C: X^T X (its diagonal, for the scaling) and X^T Y, column-major [dt][in]; W out in the cache dtype, [in][dt] per
// group.  dt is a multiple of the CTA's kTrsmWarps * kTrsmCols columns.
template <class S, typename T>
__global__ void __launch_bounds__(kTrsmWarps * 32, 4) fit_trsm_kernel(const float* __restrict__ G, const float* __restrict__ C,
                                                                      const float* __restrict__ scratch, T* wk, T* wv,
                                                                      int in, int dt, double lambda,
                                                                      const int* __restrict__ flags)
{
    extern __shared__ float4 sm4[];   // [stage][block] | [warp][plane][in][kTrsmCols]
    constexpr bool kRedo = S::PL == 2;
    __shared__ int sExp[kRedo ? 256 : 1];
    constexpr int SZ = Blocks<S>::SZ;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x, o0 = (blockIdx.y * kTrsmWarps + warp) * kTrsmCols;
    T* w = ((g & 1) ? wv : wk) + (size_t)(g >> 1) * in * dt + o0;
    if (flags[g] != (kRedo ? kSolveRedo : 0)) return;
    const int nb = in / kSolveBlk, zplane = in * kTrsmCols;
    float* stage = reinterpret_cast<float*>(sm4);
    float* z = stage + kTrsmStages * SZ + (size_t)warp * S::PL * zplane;
    const Blocks<S> L{const_cast<float*>(scratch) + (size_t)g * solve_blocks(in) * SZ, nb};
    // The blocks in the order both solves take them: per step s the s blocks of the row, then the inverse.
    const int per_pass = nb * (nb + 1) / 2, total = 2 * per_pass;
    int f_i = 0, f_pass = 0, f_s = 0, f_t = 0;   // next block to fetch
    auto fetch = [&]() {
        if (f_i < total) {
            const int k = f_pass ? nb - 1 - f_s : f_s, j = f_pass ? nb - 1 - f_t : f_t;
            const float* from = f_t == f_s ? (f_pass ? L.BI(k) : L.FI(k)) : (f_pass ? L.B(j, k) : L.F(k, j));
            float* to = stage + (f_i % kTrsmStages) * SZ;
            for (int e = threadIdx.x * 4; e < SZ; e += kTrsmWarps * 32 * 4) copy16(to + e, from + e);
            ++f_i;
            if (++f_t > f_s) {
                f_t = 0;
                if (++f_s == nb) { f_s = 0; ++f_pass; }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");   // one group a call, empty ones at the end
    };
    for (int i = 0; i < kTrsmStages - 1; ++i) fetch();
    const float* cc = C + ((size_t)g * dt + o0) * in;
    int sc[kTrsmCols];   // exponents of the right-hand sides' scaling
    if constexpr (kRedo) {
        for (int r = threadIdx.x; r < in; r += kTrsmWarps * 32)
            sExp[r] = scale_exponent(G[(size_t)g * in * in + (size_t)r * in + r], lambda);
        for (int r = lane; r < in; r += 32) {   // all columns' loads in flight
            float x[kTrsmCols];
#pragma unroll
            for (int c = 0; c < kTrsmCols; ++c) x[c] = cc[(size_t)c * in + r];
#pragma unroll
            for (int c = 0; c < kTrsmCols; ++c) z[r * kTrsmCols + c] = x[c];
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kTrsmCols; ++c) sc[c] = INT_MIN;
        for (int r = lane; r < in; r += 32)
#pragma unroll
            for (int c = 0; c < kTrsmCols; ++c) {
                const int e = (int)(__float_as_uint(z[r * kTrsmCols + c]) >> 23 & 0xffu);   // (subnormals: 0)
                if (z[r * kTrsmCols + c] != 0.f && e != 255) sc[c] = max(sc[c], e - 127 + sExp[r]);
            }
#pragma unroll
        for (int c = 0; c < kTrsmCols; ++c) {
            sc[c] = __reduce_max_sync(0xffffffffu, sc[c]);
            sc[c] = sc[c] == INT_MIN ? 0 : -sc[c];
        }
        for (int r = lane; r < in; r += 32)
#pragma unroll
            for (int c = 0; c < kTrsmCols; ++c)
                S::make(ldexpf(z[r * kTrsmCols + c], sExp[r] + sc[c])).store(z + r * kTrsmCols + c, zplane);
    } else {
        for (int c = 0; c < kTrsmCols; ++c)
            for (int r = lane; r < in; r += 32) S::make(cc[(size_t)c * in + r]).store(z + r * kTrsmCols + c, zplane);
    }
    __syncwarp();
    int n = 0;
    // the next block: landed for every thread, the one before it free for the fetch after next
    auto next_block = [&]() -> const float* {
        asm volatile("cp.async.wait_group %0;" ::"n"(kTrsmStages - 2) : "memory");
        __syncthreads();
        fetch();
        return stage + (n++ % kTrsmStages) * SZ;
    };
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass)   // L U = C, then L^T W = U
#pragma unroll 1
        for (int s = 0; s < nb; ++s) {
            float* mine = z + ((pass ? nb - 1 - s : s) * kSolveBlk + lane) * kTrsmCols;   // lane = row
            TrsmRow<S> acc;
            acc.load(mine, zplane);
#pragma unroll 1
            for (int t = 0; t <= s; ++t) {
                if (t == s) {   // the diagonal block: the row so far, times its inverse
                    acc.store(mine, zplane, false);
                    acc.zero();
                }
                const float* zt = z + (pass ? nb - 1 - t : t) * kSolveBlk * kTrsmCols;
                const float* l = next_block() + lane;   // the barrier also orders the warp's stores
#pragma unroll 4
                for (int p = 0; p < kSolveBlk; ++p) acc.sub_mul(l + p * kSolveBlk, zt + p * kTrsmCols, zplane);
            }
            __syncwarp();   // every lane has read the row
            acc.store(mine, zplane, true);
            __syncwarp();
        }
    for (int r = lane; r < in; r += 32)
#pragma unroll
        for (int c = 0; c < kTrsmCols; ++c) {
            float x = S::load(z + r * kTrsmCols + c, zplane).value();
            if constexpr (kRedo) x = ldexpf(x, sExp[r] - sc[c]);
            w[(size_t)r * dt + c] = from_f32<T>(x);
        }
}

}  // namespace
}  // namespace kvx
