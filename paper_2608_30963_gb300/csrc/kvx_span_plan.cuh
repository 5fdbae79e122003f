// kvx_span_plan.cuh -- span resolution and the window plan, shared by the span kernels (library-internal).
#pragma once

#include <climits>

#include "kvx_common.cuh"

namespace kvx {
namespace {

constexpr int kWindowRows = 48;   // source rows of a sub-tile's window

// Sequence metadata view: shared-memory copies of seq_off / src_seq_len when the
// batch is small enough, else the global arrays.
struct SeqView {
    const int* off;    // [batch+1]
    const int* slen;   // [batch]
    int batch;
    __device__ __forceinline__ int find(int tp) const
    {
        int lo = 0, hi = batch - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= tp) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
};

// Span bounds of target token tp as given (loaded ahead of use; identity: unused).
__device__ __forceinline__ int2 load_span(const TranslateParams& P, int tp)
{
    if (P.span_lo && tp < P.T_total) return make_int2(__ldg(&P.span_lo[tp]), __ldg(&P.span_hi[tp]));
    return make_int2(0, 0);
}

// Source-side resolution of one target token (sequence, clamped span) from its
// loaded span bounds; what was clamped is reported in the status word.
__device__ __forceinline__ void resolve_src(const TranslateParams& P, const SeqView& sv, int tp, int2 span, int& b,
                                            int& lo, int& hi)
{
    b = sv.find(tp);
    const int t = tp - sv.off[b];
    int S = sv.slen[b];
    if (S > P.src_max_seq || S < 0) {
        set_status(P.status, KVX_DEV_SEQ_CLAMPED);
        S = S < 0 ? 0 : P.src_max_seq;
    }
    if (P.span_lo) { lo = span.x; hi = span.y; }
    else { lo = t; hi = t + 1; }
    if (lo < 0 || hi > S || hi <= lo) {
        set_status(P.status, KVX_DEV_SPAN_CLAMPED);
        lo = lo < 0 ? 0 : (lo > S - 1 ? S - 1 : lo);
        hi = hi > S ? S : hi;
        if (hi <= lo) hi = lo + 1;
        if (S == 0) { lo = 0; hi = 0; }
    }
}

// Target-side resolution: output row offset (-1: not written) and RoPE position.
__device__ __forceinline__ void resolve_dst(const TranslateParams& P, const SeqView& sv, int tp, long long& dst_off,
                                            int& pt)
{
    const int b = sv.find(tp);
    const int t = tp - sv.off[b];
    const int p = P.tgt_pos ? __ldg(&P.tgt_pos[tp]) : t;
    pt = P.rt.enabled ? clamp_pos(p, P.max_position, P.status) : 0;
    if (!P.paged) {
        if (t >= P.dst_max_seq) { set_status(P.status, KVX_DEV_SEQ_CLAMPED); dst_off = -1; }
        else dst_off = (long long)b * P.db + (long long)t * P.dts;
    } else {
        const int pi = t / P.page_size;
        const int page = pi < P.max_pages ? __ldg(&P.page_table[(size_t)b * P.max_pages + pi]) : -1;
        if (page < 0 || page >= P.num_pages) { set_status(P.status, KVX_DEV_PAGE_INVALID); dst_off = -1; }
        else dst_off = ((long long)page * P.page_size + (t % P.page_size)) * (long long)P.Ht * P.dt;
    }
}

// Window plan of one 32-token sub-tile, read by every (layer, head, K|V) group of the window kernel
// (kvx_tc_window.cuh) and counted by kvx_span_plan_stats:
//   header  {b0, c0, rows, 0}: the window of source rows [c0, c0 + rows) of sequence b0
//   entries {w0, lo, hi, b} x 32, longest span first: w0 = window row of the span
//           start (low 16 bits, signed; -1: read from global memory) | A row within
//           the sub-tile << 16 (0xFFFF: token past the end); [lo, hi) the clamped
//           source span of sequence b.
// One warp writes the plan of sub-tile sub: lane = token (valid, its sequence and clamped span); returns whether
// the lane's token lies in the window.
__device__ __forceinline__ bool write_window_plan(bool valid, int b, int lo, int hi, int sub, int lane, int cap_rows,
                                                  int4* __restrict__ hdr, int4* __restrict__ ent)
{
    // valid tokens are a prefix of the sub-tile, so lane 0 opens the window
    const int b0 = __shfl_sync(0xffffffffu, b, 0);
    const int c0 = __shfl_sync(0xffffffffu, lo, 0);
    const bool same = valid && b == b0;
    const int hmax = __reduce_max_sync(0xffffffffu, same ? hi : INT_MIN);
    int R = hmax == INT_MIN ? 0 : max(hmax - c0, 0);
    R = min(R, cap_rows);
    const bool inwin = same && lo >= c0 && hi <= c0 + R;
    const int stage_row = inwin ? lo - c0 : -1;
    // rank: longest span first (lengths above 3 share a bucket), then lane order;
    // tokens past the end last
    const int key = valid ? min(max(hi - lo, 0), 3) : -1;
    int rank = 0;
#pragma unroll
    for (int k = 3; k >= -1; --k) {
        const unsigned bal = __ballot_sync(0xffffffffu, key == k);
        if (k > key) rank += __popc(bal);
        else if (k == key) rank += __popc(bal & ((1u << lane) - 1u));
    }
    const int w0 = (int)(((unsigned)stage_row & 0xFFFFu) | ((valid ? (unsigned)lane : 0xFFFFu) << 16));
    ent[(size_t)sub * 32 + rank] = make_int4(w0, lo, hi, b < 0 ? 0 : b);
    if (lane == 0) hdr[sub] = make_int4(b0 < 0 ? 0 : b0, c0, R, 0);
    return inwin;
}

// programmatic stream serialization: see the kernels' griddepcontrol.wait
template <typename K, typename... Args>
cudaError_t launch_pdl(K kernel, int grid, int threads, size_t smem, cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace
}  // namespace kvx
