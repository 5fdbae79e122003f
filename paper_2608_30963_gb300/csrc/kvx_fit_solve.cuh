// kvx_fit_solve.cuh -- blocked Cholesky solve of the fit's normal equations, in <= 256 (library-internal).
//
// Every group g is a system (X^T X + lambda I) W = X^T Y of `in` unknowns (a multiple of 32) and
// dt right-hand sides.  Two launches in 32 x 32 blocks:
//   fit_factor_kernel  one CTA per group: L L^T = X^T X + lambda I, right-looking.  Per block column
//                      one warp factors the diagonal block in registers, then one thread per row
//                      below solves against it while one further warp runs the same recurrence on
//                      the unit rows (the inverse of the diagonal block), then one warp per 32 x 32
//                      block applies the rank-32 update (a 4 x 8 tile a lane).
//   fit_trsm_kernel    one warp per 8 right-hand sides of a group: L U = C, then L^T W = U, left-looking
//                      with the inverted diagonal blocks, so every step is a small matrix product.
// The blocks of L live in global scratch (352 KB a group at in = 256, read through L1/L2); the
// solutions of a warp live in shared memory.
//
// Bound: the chain of block columns of one group (the factor) and FMA issue (the solves).  One thread
// per matrix column of an unblocked factor, with three barriers a column, and one thread per right-hand
// side spent 2.0 ms on 112 systems of 256 x 128.
//
// Arithmetic is a parameter.  F32: fp32, for systems the pivots show to be well conditioned.  Pair:
// unevaluated sums h + l of two floats (about 48 bits), products exact by FMA (Dekker's two-product) and
// sums by Knuth's two-sum, for the others: GB300 runs 64 fp32 FMAs for one fp64 FMA, so the twelve
// fp32 operations of a pair multiply-add cost a fifth of one fp64 FMA.
#pragma once

#include "kvx_common.cuh"

namespace kvx {
namespace {

constexpr int kSolveBlk = 32;
constexpr int kFactorThreads = 256;
constexpr int kTrsmWarps = 4;
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
    __device__ F32 inverse() const { return *this; }                // div() takes what inverse() gives
    __device__ F32 div(F32 d) const { return F32{h / d.h}; }
    __device__ F32 shfl(int s) const { return F32{__shfl_sync(0xffffffffu, h, s)}; }
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
    __device__ Pair div(Pair inv) const   // *this times an inverse()
    {
        const float p = __fmul_rn(h, inv.h);
        float e = __fmaf_rn(h, inv.h, -p);
        e = __fmaf_rn(h, inv.l, e);
        e = __fmaf_rn(l, inv.h, e);
        Pair y{p, e};
        y.norm();
        return y;
    }
    __device__ Pair shfl(int s) const
    {
        return Pair{__shfl_sync(0xffffffffu, h, s), __shfl_sync(0xffffffffu, l, s)};
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

// flags[g]: 0 solved here, kSolveRedo ill-conditioned (left to the Pair kernels), kSolveBad not
// positive definite (W is zero).  The F32 pass writes every flag and counts the redo groups in
// *n_redo; the Pair pass (redo) works on the kSolveRedo groups only.
constexpr int kSolveRedo = 1, kSolveBad = 2;

template <class S>
__global__ void __launch_bounds__(kFactorThreads, 1) fit_factor_kernel(const float* G, float* scratch, int in, double lambda,
                                                                    float max_cond, unsigned bad_bit, unsigned* status,
                                                                    int* n_redo, int* flags)
{
    constexpr bool kRedo = S::PL == 2;
    __shared__ float sD[S::PL * kPlane];        // the diagonal block's factor, (r, c) at c * 32 + r
    __shared__ float sInv[S::PL * kSolveBlk];   // what div() by its diagonal takes
    __shared__ float sPiv[256];
    __shared__ int sBad;
    const int g = blockIdx.x;
    if (kRedo && flags[g] != kSolveRedo) return;
    const int nb = in / kSolveBlk, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Blocks<S> L{scratch + (size_t)g * solve_blocks(in) * Blocks<S>::SZ, nb};
    const float* gg = G + (size_t)g * in * in;
    if (threadIdx.x == 0) sBad = 0;
    // lower blocks of X^T X + lambda I (only the lower triangle of the sums is kept)
    for (int t = warp; t < nb * (nb + 1) / 2 * kSolveBlk; t += kFactorThreads / 32) {
        const int b = t / kSolveBlk, r = t - b * kSolveBlk;
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= b) ++i;
        const int j = b - i * (i + 1) / 2;
        const bool diag = i == j && r == lane;
        S v = S::make(gg[(size_t)(i * kSolveBlk + r) * in + j * kSolveBlk + lane]);
        if (diag) v = v.add((float)lambda);
        if (diag && kRedo) v = v.add((float)(lambda - (double)(float)lambda));
        v.store(L.F(i, j) + lane * kSolveBlk + r, kPlane);
    }
    __syncthreads();

    for (int k = 0; k < nb; ++k) {
        if (warp == 0) {   // diagonal block: lane = row, its 32 entries in registers
            S a[kSolveBlk];
            float* d = L.F(k, k);
#pragma unroll
            for (int c = 0; c < kSolveBlk; ++c) a[c] = S::load(d + c * kSolveBlk + lane, kPlane);
            int bad = 0;
#pragma unroll
            for (int c = 0; c < kSolveBlk; ++c) {
                S p = a[c].shfl(c);
                if (!(p.value() > 0.f)) { bad = 1; p = S::make(1.f); }
                const S l = p.root(), inv = l.inverse();
                const S v = lane == c ? l : a[c].div(inv);
                if (lane == 0) {
                    inv.store(sInv + c, kSolveBlk);
                    sPiv[k * kSolveBlk + c] = l.value();
                }
                v.store(sD + c * kSolveBlk + lane, kPlane);
#pragma unroll
                for (int q = c + 1; q < kSolveBlk; ++q) {
                    a[q].sub_mul(v, v.shfl(q));
                    if (q == c + 1) a[q].norm();
                }
            }
            if (bad && lane == 0) sBad = 1;
        }
        __syncthreads();
        // rows below, and the 32 unit rows whose solution is the inverse's columns
        const int below = in - (k + 1) * kSolveBlk;
        for (int t = threadIdx.x; t < below + kSolveBlk; t += kFactorThreads) {
            const bool unit = t >= below;
            const int row = unit ? t - below : t & 31, i = k + 1 + (t >> 5);
            S x[kSolveBlk];
            if (unit) {
#pragma unroll
                for (int c = 0; c < kSolveBlk; ++c) x[c] = S::make(c == row ? 1.f : 0.f);
            } else {
                const float* f = L.F(i, k) + row;
#pragma unroll
                for (int c = 0; c < kSolveBlk; ++c) x[c] = S::load(f + c * kSolveBlk, kPlane);
            }
#pragma unroll
            for (int c = 0; c < kSolveBlk; ++c) {
                x[c].norm();
                x[c] = x[c].div(S::load(sInv + c, kSolveBlk));
#pragma unroll
                for (int q0 = 0; q0 < kSolveBlk; q0 += 4) {
                    if (q0 + 3 <= c) continue;
                    S l[4];
                    load4(sD + c * kSolveBlk + q0, l);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (q0 + e > c) x[q0 + e].sub_mul(x[c], l[e]);
                }
            }
            float* by_col = unit ? L.BI(k) : L.F(i, k);   // element c of this row at c * 32 + row
            float* by_row = unit ? L.FI(k) : L.B(i, k);   // at row * 32 + c
#pragma unroll
            for (int c = 0; c < kSolveBlk; ++c) x[c].store(by_col + c * kSolveBlk + row, kPlane);
#pragma unroll
            for (int c0 = 0; c0 < kSolveBlk; c0 += 4) {
                const S v[4] = {x[c0], x[c0 + 1], x[c0 + 2], x[c0 + 3]};
                store4(by_row + row * kSolveBlk + c0, v);
            }
        }
        __syncthreads();
        // rank-32 update of the blocks to the right: lane = 4 rows x 8 columns
        const int m = nb - 1 - k, r0 = (lane & 7) * 4, c0 = (lane >> 3) * 8;
        for (int t = warp; t < m * (m + 1) / 2; t += kFactorThreads / 32) {
            int i = 0;
            while ((i + 1) * (i + 2) / 2 <= t) ++i;
            const int j = t - i * (i + 1) / 2;
            const float *fi = L.F(k + 1 + i, k) + r0, *fj = L.F(k + 1 + j, k) + c0;
            float* out = L.F(k + 1 + i, k + 1 + j) + c0 * kSolveBlk + r0;
            S acc[8][4];
#pragma unroll
            for (int c = 0; c < 8; ++c) load4(out + c * kSolveBlk, acc[c]);
#pragma unroll 4
            for (int p = 0; p < kSolveBlk; ++p) {
                S a[4], b[2][4];
                load4(fi + p * kSolveBlk, a);
                load4(fj + p * kSolveBlk, b[0]);
                load4(fj + p * kSolveBlk + 4, b[1]);
#pragma unroll
                for (int c = 0; c < 8; ++c)
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[c][r].sub_mul(a[r], b[c >> 2][c & 3]);
            }
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
            if (sBad) {
                flags[g] = kSolveBad;
                set_status(status, bad_bit);
            } else if (!kRedo) {
                const int ill = ratio * ratio > max_cond;
                flags[g] = ill ? kSolveRedo : 0;
                if (ill) atomicAdd(n_redo, 1);
            }
        }
    }
}

// acc (rows 4 (lane % 8).. of a block, two columns) -= block . z, z[32][kTrsmCols] of one block row.
template <class S>
__device__ __forceinline__ void trsm_step(S (&acc)[2][4], const float* block, const float* z, int zplane, int lane)
{
    const float* a0 = block + (lane & 7) * 4;
    const float* z0 = z + (lane >> 3) * 2;
#pragma unroll 8
    for (int p = 0; p < kSolveBlk; ++p) {
        S a[4];
        load4(a0 + p * kSolveBlk, a);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const S b = S::load(z0 + p * kTrsmCols + c, zplane);
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[c][r].sub_mul(a[r], b);
        }
    }
}

// C: X^T Y, column-major [dt][in]; W out in the cache dtype, [in][dt] per group.
template <class S, typename T>
__global__ void __launch_bounds__(kTrsmWarps * 32, 3) fit_trsm_kernel(const float* __restrict__ C,
                                                                   const float* __restrict__ scratch, T* wk, T* wv,
                                                                   int in, int dt, const int* __restrict__ flags)
{
    extern __shared__ float zs[];   // [warp][plane][in][kTrsmCols]
    constexpr bool kRedo = S::PL == 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x, o0 = (blockIdx.y * kTrsmWarps + warp) * kTrsmCols;
    const int flag = flags[g];
    if (o0 >= dt) return;
    T* w = ((g & 1) ? wv : wk) + (size_t)(g >> 1) * in * dt + o0;
    if (kRedo ? flag == 0 : flag == kSolveRedo) return;
    if (flag == kSolveBad) {
        for (int i = lane; i < in * kTrsmCols; i += 32)
            w[(size_t)(i / kTrsmCols) * dt + i % kTrsmCols] = from_f32<T>(0.f);
        return;
    }
    const int nb = in / kSolveBlk, zplane = in * kTrsmCols;
    float* z = zs + (size_t)warp * S::PL * zplane;
    const Blocks<S> L{const_cast<float*>(scratch) + (size_t)g * solve_blocks(in) * Blocks<S>::SZ, nb};
    const float* cc = C + ((size_t)g * dt + o0) * in;
    for (int c = 0; c < kTrsmCols; ++c)
        for (int r = lane; r < in; r += 32) S::make(cc[(size_t)c * in + r]).store(z + r * kTrsmCols + c, zplane);
    __syncwarp();
    const int mine = (lane & 7) * 4 * kTrsmCols + (lane >> 3) * 2;   // this lane's first value of a block row
    auto load_row = [&](int k, S (&acc)[2][4]) {
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int r = 0; r < 4; ++r)
                acc[c][r] = S::load(z + k * kSolveBlk * kTrsmCols + mine + r * kTrsmCols + c, zplane);
    };
    auto store_row = [&](int k, S (&acc)[2][4], bool neg) {
        __syncwarp();   // every lane has read block row k
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                acc[c][r].norm();
                (neg ? acc[c][r].neg() : acc[c][r]).store(z + k * kSolveBlk * kTrsmCols + mine + r * kTrsmCols + c, zplane);
            }
        __syncwarp();
    };
    auto row_of = [&](int k) { return z + k * kSolveBlk * kTrsmCols; };
    S acc[2][4];
    for (int pass = 0; pass < 2; ++pass) {   // L U = C, then L^T W = U
        for (int s = 0; s < nb; ++s) {
            const int k = pass ? nb - 1 - s : s;
            load_row(k, acc);
            for (int t = 0; t < s; ++t) {
                const int j = pass ? nb - 1 - t : t;
                trsm_step<S>(acc, pass ? L.B(j, k) : L.F(k, j), row_of(j), zplane, lane);
            }
            store_row(k, acc, false);
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[c][r] = S::make(0.f);
            trsm_step<S>(acc, pass ? L.BI(k) : L.FI(k), row_of(k), zplane, lane);
            store_row(k, acc, true);
        }
    }
    for (int r = lane; r < in; r += 32)
#pragma unroll
        for (int c = 0; c < kTrsmCols; ++c)
            w[(size_t)r * dt + c] = from_f32<T>(S::load(z + r * kTrsmCols + c, zplane).value());
}

}  // namespace
}  // namespace kvx
