// kvx_tc_rows.cu -- tensor-core translation kernel over gathered source rows (spans).
//
// A tile is 128 consecutive target tokens.  The first source row of each token's span goes from the
// cache straight into the K-major 128-byte-swizzled operand layout with 16-byte asynchronous copies, so
// a token of one source row (three in four) is in place when its copies land: for V nothing is left to
// do, for K the row is un-rotated where it lies.  Only tokens with more rows are averaged in registers,
// from A and from a side buffer that a warp of its own fills with the tile's further rows.  Building every
// row in registers from a staged window of source rows (kvx_tc_window.cuh) leaves the tensor core waiting for the
// chain of eight-lane steps that do it.
//
// Row plan (span_rows_kernel, once per translation, read by every (layer, head, K|V) group): per tile
// its tokens ordered by span length, longest first, so that the tokens with several rows are the first
// `multi` rows of A.  Any spans will do: overlapping, repeated, descending, empty (a zero row).
//
// Inputs wider than 256 channels (several source layers, wide groups) are gathered and un-rotated 256
// channels at a time (a K group) into the same accumulator; their weights do not stay but stream a K-block
// at a time through a ring, in the MMA's order.  Groups of two source layers, 70B -> 7B shapes, 8192
// tokens: 1092 us, 1339 in the window kernel.  Units of several heads (the dense form) stay there: with
// four heads' weights to stream per K-block the ring's 64 KB do not cover the L2's latency (1294 against
// 896 us).
//
// Persistent, one CTA per SM.  Work unit = (target layer j, target head h, K|V, output split nt, tile):
//   warp 0         MMA: TMEM allocation, the group's B image (kept across its tiles, or streamed),
//                  tcgen05.mma per K-block (64 channels), commits
//   warps 1-2      gather: 64 rows each, into a ring of K-block slots
//   warp 3         side buffer: the further rows of the tile's spans
//   warps 4-11     epilogue: TMEM -> target RoPE -> bf16 -> cache (bulk row stores); two warps per lane
//                  quadrant, each taking half of the rotary pairs
//   warps 12-19    prologue: source-RoPE undo of K rows in place, span means
// Every wait is bounded (~1 s, then KVX_DEV_WAIT_TIMEOUT and a drained exit).
//
// Dense spans.  Further rows that the side buffer has no room for are read from memory by the prologue, with their
// latency exposed; a window (kvx_tc_window.cuh) holds 48 rows of a 32-token sub-tile and is copied ahead.  The spans
// are known on the device only.  Where the source may hold 1.5 rows or more for each target token the kernel is
// launched in a form (kDense) that counts, over the plan's tiles, the further rows beyond the side buffer (o), the
// tokens of several rows (m) and the rows of the tokens outside their windows (w), and runs the window kernel's body
// where o + 2 m - w / 4 exceeds dense_sum a tile (rows_layout).  With fewer source rows the spans can only be dense
// where they overlap, and the plain form runs: the count and the second body cost it up to 2% (70B -> 7B shapes, 8192
// tokens: 513 us against 503; 1.5B -> Gemma-2B shapes, a ragged batch of 1574: 98.8 against 98.0).  4096
// tokens, 8 layers of 128 x 128 heads grouped by two, us here and in windows: spans of 1.3 rows 59 and 79, of 1.6 86 and 94, of 2 119 and 114, of two each 112 and 91, of 8 to 16 964 and 803.
#include "kvx_common.cuh"
#include "kvx_kernels.h"
#include "kvx_span_plan.cuh"
#include "kvx_tc_common.cuh"
#include "kvx_tc_window.cuh"

namespace kvx {
namespace {

constexpr int kTileM = 128;
constexpr int kBlockK = 64;
constexpr int kBlockBytes = kTileM * kBlockK * 2;   // 16 KB
constexpr int kMaxSlots = 12;
constexpr int kMmaWarp = 0;
constexpr int kGatherWarp0 = 1;
constexpr int kNumGatherWarps = 2;
constexpr int kSideWarp = kGatherWarp0 + kNumGatherWarps;
constexpr int kEpiWarp0 = kSideWarp + 1;
constexpr int kNumEpiWarps = 8;
constexpr int kEpiParts = kNumEpiWarps / 4;   // epilogue warps per TMEM lane quadrant
constexpr int kXfWarp0 = kEpiWarp0 + kNumEpiWarps;
constexpr int kNumXfWarps = 8;
constexpr int kThreads = (kXfWarp0 + kNumXfWarps) * 32;
static_assert(kThreads == kRowsThreads, "reported by kvx_get_info");

constexpr int kMaxB = 8;                            // weight ring slots (streamed)
constexpr int kBarBFull = 0, kBarBEmpty = kMaxB;    // +weight slot
constexpr int kBarDFull = 2 * kMaxB;                // +buf
constexpr int kBarDEmpty = kBarDFull + 2;           // +buf
constexpr int kBarFull = kBarDEmpty + 2;            // +slot: the gather's copies landed
constexpr int kBarEmpty = kBarFull + kMaxSlots;     // +slot: MMA done with it
// +(tile % nready): A is built (as many as tiles can lie between the prologue and the MMA)
constexpr int kBarKReady = kBarEmpty + kMaxSlots;
constexpr int kMaxKReady = kMaxSlots + 2;
// +(tile % kEntTabs): its row entries are in shared memory / the prologue is done with them
constexpr int kEntTabs = 4;
constexpr int kBarEntFull = kBarKReady + kMaxKReady;
constexpr int kBarEntEmpty = kBarEntFull + kEntTabs;
constexpr int kBarSideFull = kBarEntEmpty + kEntTabs, kBarSideEmpty = kBarSideFull + 1;
constexpr int kBarPair = kBarSideEmpty + 1;         // +quad*2 + {0,1}: the epilogue warps of a quadrant meet
constexpr int kBarMmaDone = kBarPair + 8;
constexpr int kNumBars = kBarMmaDone + 1;

// Plan entry of an A row.  src: {offset of the span's first row from its head's first row, in 16-byte
// units; rows of the span (0: zero row, -1: past the last token); position of the first row; the span's
// second row among the tile's further rows}.  dst: {target row offset (low, high word; -1: not written),
// target position, 0}.  where: {sequence, first row}.
struct RowEnt {
    int4 src, dst;
    int2 where, pad;
};
// Plan of a tile: rows with spans of other than one row, tokens, further rows, source rows of the tokens outside
// their sub-tile's window (both saturated at kRowsMax); the offsets of the first kSideMax further rows.
constexpr int kSideMax = 128;
constexpr int kRowsMax = 1 << 18;   // four times this over the 512 tiles of a launch fits an int
struct TilePlan {
    int4 count;
    unsigned side[kSideMax];
};

struct RowsLaunch {
    int n_tile, n_split, nslots, share;
    int nblk, kgs;         // K-blocks of a K group (at most 256 channels), K groups of an input row
    int nb;                // weight ring slots, each a K-block (several K groups); 0: the image stays resident
    int m_tiles;
    int side_rows;         // further rows the side buffer holds
    int dense_sum;         // dense spans: the sum a tile above which they are (see the top)
    const TilePlan* tiles; // [tile]
    const RowEnt* rows;    // [tile][128]
    unsigned b_bytes, stage_row_bytes;
    unsigned off_b, off_stage, off_bar, off_misc, off_turns, off_ent, off_ring, off_side;
    unsigned idesc, tmem_cols;
};

// The CTA's units: an equal share of the K units and of the V units, each group-major; every second
// CTA walks its V share first, so that K tiles (un-rotated) and V tiles (streamed) run side by side.
// share > 1: target heads that read the same source rows, walked by that many interleaved CTA sets,
// so that partners read a tile's rows at about the same time and all but one find them in L2.
// The walk, worked out once per CTA: units of the first share and in all, and where each share starts.
struct RWalkStart {
    int n1, count;
    int kv[2], j[2], h[2], nt[2], tile[2], h0[2];   // h0: this CTA's head among those that share rows
    __device__ void init(const TranslateParams& P, const RowsLaunch& L)
    {
        const int E = L.share;
        const long long UH = (long long)P.Lt * P.Ht * L.n_split * L.m_tiles / E;   // K (or V) units of one set
        const int G = gridDim.x / E, c = blockIdx.x / E, rev = (int)(gridDim.x - 1 - blockIdx.x), cv = rev / E;
        const int u0 = (int)((long long)c * UH / G), u1 = (int)((long long)(c + 1) * UH / G);
        const int v0 = (int)((long long)cv * UH / G), v1 = (int)((long long)(cv + 1) * UH / G);
        const bool v_first = (c & 1) == 0;
        n1 = v_first ? v1 - v0 : u1 - u0;
        count = (u1 - u0) + (v1 - v0);
        for (int i = 0; i < 2; ++i) {
            kv[i] = (i == 0) == v_first ? 1 : 0;
            const int idx = kv[i] ? v0 : u0, hg = idx / L.m_tiles, jq = hg / L.n_split, HtE = P.Ht / E;
            h0[i] = (kv[i] ? rev : (int)blockIdx.x) % E;
            tile[i] = idx - hg * L.m_tiles;
            nt[i] = hg % L.n_split;
            h[i] = (jq % HtE) * E + h0[i];
            j[i] = jq / HtE;
        }
    }
};
template <bool STREAM>
struct RWalker {
    const TranslateParams& P;
    const RowsLaunch& L;
    const RWalkStart& S;
    int it, kv, j, h, nt, tile;
    int kg;   // K group
    __device__ __forceinline__ RWalker(const TranslateParams& P_, const RowsLaunch& L_, const RWalkStart& S_) : P(P_), L(L_), S(S_)
    {
        it = 0;
        kg = 0;
        share(S.n1 > 0 ? 0 : 1);
    }
    __device__ __forceinline__ void share(int i)
    {
        kv = S.kv[i]; j = S.j[i]; h = S.h[i]; nt = S.nt[i]; tile = S.tile[i];
    }
    __device__ __forceinline__ int group() const { return ((j * P.Ht + h) * 2 + kv) * L.n_split + nt; }   // its B image
    __device__ __forceinline__ bool more() const { return it < S.count; }
    // the next K group (of the unit, then of the next)
    __device__ __forceinline__ void next()
    {
        if (STREAM) {
            if (++kg < L.kgs) return;
            kg = 0;
        }
        next_unit();
    }
    __device__ __forceinline__ void next_unit()
    {
        ++it;
        if (it == S.n1) { share(1); return; }
        if (++tile == L.m_tiles) {
            tile = 0;
            if (++nt == L.n_split) {
                nt = 0;
                if ((h += L.share) >= P.Ht) { h = S.h0[it < S.n1 ? 0 : 1]; ++j; }
            }
        }
    }
    // tile of the next K group
    __device__ __forceinline__ int next_tile() const { return STREAM && kg + 1 < L.kgs ? tile : next_unit_tile(); }
    // tile of the unit after this one (this one's after the last)
    __device__ __forceinline__ int next_unit_tile() const
    {
        if (it + 1 >= S.count) return tile;
        return it + 1 == S.n1 ? S.tile[1] : tile + 1 == L.m_tiles ? 0 : tile + 1;
    }
    __device__ __forceinline__ bool last_of_group() const
    {
        return it + 1 == S.count || it + 1 == S.n1 || tile + 1 == L.m_tiles;
    }
};

// Waiter with the slow path out of line: the kernel has some twenty waits, and its roles' code competes for
// the instruction cache (70B -> 7B shapes, 8192 tokens: 527 us with the path inline, 503 so).
__device__ __noinline__ bool wait_slow(volatile int* abort, unsigned* status, unsigned long long limit_ns, uint32_t bar,
                                       uint32_t parity)
{
    const unsigned long long t0 = globaltimer();
    while (true) {
        if (mbar_try_wait_sleep(bar, parity, 100000u)) return true;
        if (*abort) return false;
        if (globaltimer() - t0 > limit_ns) {
            *abort = 1;
            set_status(status, KVX_DEV_WAIT_TIMEOUT);
            return false;
        }
    }
}
struct RWaiter {
    volatile int* abort;
    unsigned* status;
    unsigned long long limit_ns;
    __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) const
    {
        return mbar_try_wait(bar, parity) || wait_slow(abort, status, limit_ns, bar, parity);
    }
};

struct Slot {
    uint32_t idx, phase;
    __device__ __forceinline__ void adv(uint32_t n)
    {
        if (++idx == n) { idx = 0; phase ^= 1; }
    }
};

// The calling thread's arrival on bar happens when its asynchronous copies so far have landed.
__device__ __forceinline__ void cp_async_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// acc += the 8 bf16 of w.
__device__ __forceinline__ void add8(float (&acc)[8], uint4 w)
{
    const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        acc[2 * k] += bf_lo(v[k]);
        acc[2 * k + 1] += bf_hi(v[k]);
    }
}
// (a0, a1) += the pairs of chunks w0, w1 un-rotated; unrotate8_first: set to them (for one row, as the
// identity-alignment kernel does it).
__device__ __forceinline__ void unrotate8(uint4 w0, uint4 w1, const float2 (&cs)[8], float (&a0)[8], float (&a1)[8])
{
    const uint32_t v0[4] = {w0.x, w0.y, w0.z, w0.w}, v1[4] = {w1.x, w1.y, w1.z, w1.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float x0 = k & 1 ? bf_hi(v0[k >> 1]) : bf_lo(v0[k >> 1]), x1 = k & 1 ? bf_hi(v1[k >> 1]) : bf_lo(v1[k >> 1]);
        a0[k] = fmaf(x0, cs[k].x, fmaf(x1, cs[k].y, a0[k]));
        a1[k] = fmaf(x1, cs[k].x, fmaf(-x0, cs[k].y, a1[k]));
    }
}
__device__ __forceinline__ void unrotate8_first(uint4 w0, uint4 w1, const float2 (&cs)[8], float (&a0)[8], float (&a1)[8])
{
    const uint32_t v0[4] = {w0.x, w0.y, w0.z, w0.w}, v1[4] = {w1.x, w1.y, w1.z, w1.w};
#pragma unroll
    for (int k = 0; k < 8; ++k)
        unrotate1(k & 1 ? bf_hi(v0[k >> 1]) : bf_lo(v0[k >> 1]), k & 1 ? bf_hi(v1[k >> 1]) : bf_lo(v1[k >> 1]), cs[k], a0[k], a1[k]);
}
__device__ __forceinline__ uint4 pack8(const float (&a)[8])
{
    return make_uint4(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(a[4], a[5]), pack_bf16(a[6], a[7]));
}
__device__ __forceinline__ uint4 pack8(const float (&a)[8], float f)
{
    return make_uint4(pack_bf16(a[0] * f, a[1] * f), pack_bf16(a[2] * f, a[3] * f), pack_bf16(a[4] * f, a[5] * f),
                      pack_bf16(a[6] * f, a[7] * f));
}
// HS: half head_dim of the source (32, 64 or 128); HEADS: source heads of a K group; STREAM: several K groups,
// weights streamed (else a resident image).  MODE: kDense, the spans may be dense (see the top), D is the window
// kernel's launch over the same tokens; kDiag, the diagnostics of the bounded waits.
constexpr int kPlain = 0, kDense = 1, kDiag = 2;
template <int HS, int HEADS, bool STREAM, int MODE>
__global__ void __launch_bounds__(kThreads, 1)
translate_rows_kernel(const __grid_constant__ TranslateParams P, const __grid_constant__ RowsLaunch L,
                      const __grid_constant__ window::TcLaunch D)
{
    constexpr bool DENSE = MODE == kDense;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* sB = smem + L.off_b;
    uint8_t* sRing = smem + L.off_ring;
    uint8_t* sStage = smem + L.off_stage;
    uint8_t* sSide = smem + L.off_side;
    int4* sEnt = reinterpret_cast<int4*>(smem + L.off_ent);   // [table][row]: RowEnt::src
    uint64_t* sBar = reinterpret_cast<uint64_t*>(smem + L.off_bar);
    volatile int* sAbort = reinterpret_cast<volatile int*>(smem + L.off_misc);
    uint32_t* sTmemBase = reinterpret_cast<uint32_t*>(smem + L.off_misc + 4);
    RWalkStart& sWalk = *reinterpret_cast<RWalkStart*>(smem + L.off_misc + 16);
    int* sDense = reinterpret_cast<int*>(smem + L.off_misc + 16 + sizeof(RWalkStart));
    unsigned long long* sTurnS = reinterpret_cast<unsigned long long*>(smem + L.off_turns);
    unsigned long long* sTurnT = sTurnS + HS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto bar = [&](int i) { return smem_u32(&sBar[i]); };
    const uint32_t NS = (uint32_t)L.nslots, NKR = NS / (uint32_t)L.nblk + 2;

    if (threadIdx.x == 32) sWalk.init(P, L);
    // f(index, arrivals) for every barrier
    auto barriers = [&](auto f) {
        for (int i = 0; i < kMaxB; ++i) {
            f(kBarBFull + i, 1);
            f(kBarBEmpty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            f(kBarDFull + i, 1);
            f(kBarDEmpty + i, kNumEpiWarps);
        }
        for (int i = 0; i < (int)NS; ++i) {
            f(kBarFull + i, kNumGatherWarps * 32);   // every gather lane's copies
            f(kBarEmpty + i, 1);
        }
        for (int i = 0; i < (int)NKR; ++i) f(kBarKReady + i, kNumXfWarps);
        for (int i = 0; i < kEntTabs; ++i) {
            f(kBarEntFull + i, kNumGatherWarps * 32);
            f(kBarEntEmpty + i, kNumXfWarps);
        }
        f(kBarSideFull, 32);
        f(kBarSideEmpty, kNumXfWarps);
        for (int i = 0; i < 8; ++i) f(kBarPair + i, kEpiParts);
        f(kBarMmaDone, 1);
    };
    if (threadIdx.x == 0) {
        *sAbort = 0;
        barriers([&](int i, int n) { mbar_init(bar(i), (uint32_t)n); });
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(sTmemBase), L.tmem_cols);
        tmem_relinquish();
    }
    // nothing above touched global memory
    grid_dependency_wait();
    grid_launch_dependents();
    // source turns transposed: pair 8 c + i at i * (HS / 8) + c
    for (int i = threadIdx.x; i < HS; i += blockDim.x)
        sTurnS[(i & 7) * (HS / 8) + (i >> 3)] = P.rs.enabled ? __ldg(&P.rs.turns[i]) : 0ull;
    for (int i = threadIdx.x; i < (P.dt >> 1); i += blockDim.x) sTurnT[i] = P.rt.enabled ? __ldg(&P.rt.turns[i]) : 0ull;
    if (DENSE && warp == kSideWarp) {
        int v = 0;
#pragma unroll 4
        for (int i = lane; i < L.m_tiles; i += 32) {
            const int4 c = __ldg(&L.tiles[i].count);
            v += 4 * (max(c.z - L.side_rows, 0) + 2 * min(c.x, c.z) - L.dense_sum) - c.w;
        }
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) *sDense = v;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *sTmemBase;
    const int dense = DENSE ? *sDense : 0;   // above 0: dense spans, in every CTA of the launch
    const RWaiter W{sAbort, P.status, P.wait_ns ? P.wait_ns : kWaitNs};
    const int hw = L.n_tile >> 1;

    if (DENSE && dense > 0) {
        // below
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            const uint64_t pol_keep = policy_evict_last();
            const uint32_t nb = STREAM ? (uint32_t)L.nb : 0u, kblock = (uint32_t)L.n_tile * 128;   // bytes of a K-block of weights
            int cur_g = -1;
            uint32_t b_cnt = 0, tcount = 0, kr_idx = 0, kr_phase = 0;   // b_cnt: images or weight K-blocks loaded
            Slot sp{0, 0};
            // streamed weights: the walk of the loads, nb - 1 K-blocks ahead of the MMAs
            RWalker<STREAM> y(P, L, sWalk);
            int y_kb = 0;
            auto load_next = [&]() -> bool {
                if (!y.more()) return true;
                const uint32_t slot = b_cnt % nb;
                if (!W.wait(bar(kBarBEmpty + slot), ((b_cnt / nb) & 1) ^ 1)) return false;
                mbar_arrive_expect_tx(bar(kBarBFull + slot), kblock);
                bulk_g2s(smem_u32(sB) + slot * kblock,
                         (const uint8_t*)P.w + (size_t)y.group() * L.b_bytes + (size_t)(y.kg * L.nblk + y_kb) * kblock, kblock,
                         bar(kBarBFull + slot), pol_keep);
                ++b_cnt;
                if (++y_kb == L.nblk) { y_kb = 0; y.next(); }
                return true;
            };
            uint32_t b_use = 0;   // weight K-blocks multiplied
            bool ok = true;
            if (STREAM)
                for (uint32_t i = 0; i + 1 < nb && ok; ++i) ok = load_next();
            RWalker<STREAM> x(P, L, sWalk);
            for (; x.more() && ok; x.next()) {
                if (!STREAM && x.group() != cur_g) {   // the group before has been multiplied when its last commit arrives
                    if (!W.wait(bar(kBarBEmpty), (b_cnt & 1) ^ 1)) break;
                    mbar_arrive_expect_tx(bar(kBarBFull), L.b_bytes);
                    const uint8_t* img = (const uint8_t*)P.w + (size_t)x.group() * L.b_bytes;
                    const uint32_t piece = L.b_bytes / 4;
                    for (int q = 0; q < 4; ++q)
                        bulk_g2s(smem_u32(sB) + q * piece, img + (size_t)q * piece, piece, bar(kBarBFull), pol_keep);
                    ++b_cnt;
                    if (!W.wait(bar(kBarBFull), (b_cnt - 1) & 1)) break;
                    cur_g = x.group();
                }
                const uint32_t buf = tcount & 1;
                if ((!STREAM || x.kg == 0) && !W.wait(bar(kBarDEmpty + buf), ((tcount >> 1) & 1) ^ 1)) break;
                if (!W.wait(bar(kBarKReady + kr_idx), kr_phase)) break;
                if (++kr_idx == NKR) { kr_idx = 0; kr_phase ^= 1; }
                tc_fence_after();
                const uint32_t d = tmem_base + buf * (uint32_t)L.n_tile;
                for (int kb = 0; kb < L.nblk; ++kb) {
                    const uint32_t a0 = smem_u32(sRing) + sp.idx * kBlockBytes;
                    const uint32_t slot = STREAM ? b_use % nb : 0;
                    const uint32_t b0 = smem_u32(sB) + (STREAM ? slot : (uint32_t)kb) * kblock;
                    if (STREAM) {
                        if (!W.wait(bar(kBarBFull + slot), (b_use / nb) & 1)) { ok = false; break; }
                        tc_fence_after();
                    }
#pragma unroll
                    for (int kk = 0; kk < kBlockK / 16; ++kk)
                        umma_bf16(d, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32), L.idesc,
                                  ((STREAM && x.kg > 0) || kb > 0 || kk > 0) ? 1u : 0u);
                    umma_commit(bar(kBarEmpty + sp.idx));
                    sp.adv(NS);
                    if (STREAM) {
                        umma_commit(bar(kBarBEmpty + slot));
                        ++b_use;
                        if (!load_next()) { ok = false; break; }
                    }
                }
                if (!ok) break;
                if (!STREAM || x.kg + 1 == L.kgs) {
                    umma_commit(bar(kBarDFull + buf));
                    ++tcount;
                }
                if (!STREAM && x.last_of_group()) umma_commit(bar(kBarBEmpty));
            }
            if (*sAbort) {   // MMAs whose results nobody waited for must finish before TMEM is freed, copies land
                umma_commit(bar(kBarMmaDone));
                const unsigned long long t0 = globaltimer();
                while (!mbar_try_wait(bar(kBarMmaDone), 0) && globaltimer() - t0 < W.limit_ns) {}
                const uint32_t n = STREAM ? nb : 1;
                for (uint32_t c = b_cnt > n ? b_cnt - n : 0; c < b_cnt; ++c)
                    while (!mbar_try_wait(bar(kBarBFull + c % n), (c / n) & 1) && globaltimer() - t0 < W.limit_ns) {}
            }
        }
        __syncwarp();
    } else if (warp >= kEpiWarp0 && warp < kXfWarp0) {
        // ------------------------------------------------------------ epilogue
        const int quad = warp & 3;
        const int part = (warp - kEpiWarp0) >> 2;
        const int m = quad * 32 + lane;
        const int pc_begin = part * (hw / kEpiParts), pc_end = pc_begin + hw / kEpiParts;
        uint8_t* srow = sStage + (size_t)m * L.stage_row_bytes;
        const uint32_t srow_u32 = smem_u32(srow);
        uint32_t tcount = 0;
        RWalker<STREAM> x(P, L, sWalk);
        int n_nxt = -1;                     // the next unit's plan words, loaded a unit ahead
        int4 d_nxt = make_int4(0, 0, 0, 0);
        auto fetch = [&](int tile) {
            const RowEnt* ent = L.rows + (size_t)tile * kTileM + m;
            n_nxt = __ldg(&ent->src.y);
            d_nxt = __ldg(&ent->dst);
        };
        if (x.more()) fetch(x.tile);
        for (; x.more(); x.next_unit()) {
            const int4 ed = d_nxt;
            const bool valid = n_nxt >= 0;
            fetch(x.next_unit_tile());
            const long long dst_off = (long long)(((unsigned long long)(unsigned)ed.y << 32) | (unsigned)ed.x);
            const int pt = ed.z;
            const bool rot = x.kv == 0 && P.rt.enabled;
            const uint32_t buf = tcount & 1;
            if (!W.wait(bar(kBarDFull + buf), (tcount >> 1) & 1)) break;
            tc_fence_after();
            // the staging row is shared by the warps of this quadrant; the row's previous store must have
            // read it
            bulk_wait_read0();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarPair + quad * 2));
            if (!W.wait(bar(kBarPair + quad * 2), tcount & 1)) break;
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + buf * (uint32_t)L.n_tile;
#pragma unroll 1
            for (int pc = pc_begin; pc < pc_end; pc += 8) {
                uint32_t r0[8], r1[8];
                tmem_ld8(taddr + pc, r0);
                tmem_ld8(taddr + hw + pc, r1);
                float2 cs[8];
                if (rot) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) cs[e] = turn_cs(sTurnT[x.nt * hw + pc + e], pt);
                }
                tmem_ld_wait();
                uint4 out0, out1;
                rotate8_to_bf16(r0, r1, cs, rot, out0, out1);
                *reinterpret_cast<uint4*>(srow + pc * 2) = out0;
                *reinterpret_cast<uint4*>(srow + (hw + pc) * 2) = out1;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarDEmpty + buf));
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarPair + quad * 2 + 1));
            if (!W.wait(bar(kBarPair + quad * 2 + 1), tcount & 1)) break;
            if ((lane & (kEpiParts - 1)) == part && valid && dst_off >= 0) {   // the quadrant's rows, split between its warps
                __nv_bfloat16* dst = (__nv_bfloat16*)(x.kv ? P.dst_v[x.j] : P.dst_k[x.j]) + dst_off + dst_head_off(P, x.h);
                if (P.plain_stores) {
                    store_row_slots_plain(dst, srow, x.nt * hw, hw, P.dt >> 1, P.dt >> 1);
                } else {
                    store_row_slots(dst, srow_u32, x.nt * hw, hw, P.dt >> 1, P.dt >> 1);
                    bulk_commit();
                }
            }
            ++tcount;
        }
        bulk_wait0();
    } else if (warp >= kXfWarp0) {
        // ------------------------------------------------------------ prologue
        // A pass gives every thread one (row, 16-byte chunk) of the rows with several source rows (V) or one
        // (row, chunk pair), every head (K), the chunk fastest: 8 lanes cover the 128 bytes of a row's
        // K-block.
        constexpr int CPH = HS / 8;                        // chunk pairs of a head
        constexpr int CPR = HEADS * 2 * CPH;               // chunks of a row
        constexpr int kXfThreads = kNumXfWarps * 32;
        constexpr int kRowsK = kXfThreads / CPH, kRowsV = kXfThreads / CPR;   // rows of a pass
        const int xt = threadIdx.x - kXfWarp0 * 32;
        const int cp = xt % CPH;                           // this thread's chunk pair (K)
        // turns of its pairs, the pair's index slowest: lanes of different chunks read different banks
        auto cs8 = [&](int pos, float2 (&cs)[8]) {
#pragma unroll
            for (int i = 0; i < 8; ++i) cs[i] = turn_cs(sTurnS[i * CPH + cp], pos);
        };
        Slot sp{0, 0};
        uint32_t kr_idx = 0, ent_cnt = 0;
        RWalker<STREAM> x(P, L, sWalk);
        int4 t_nxt = x.more() ? __ldg(&L.tiles[x.tile].count) : make_int4(0, 0, 0, 0);   // a unit ahead
        for (; x.more(); x.next()) {
            const bool rot = x.kv == 0 && P.rs.enabled;
            const int multi = t_nxt.x, tokens = t_nxt.y;
            t_nxt = __ldg(&L.tiles[x.next_tile()].count);
            const int4* ent = sEnt + (ent_cnt % kEntTabs) * kTileM;
            // ring slot of the tile's K-block kb
            auto a_block = [&](int kb) {
                const uint32_t si = sp.idx + (uint32_t)kb;
                return sRing + (si >= NS ? si - NS : si) * kBlockBytes;
            };
            // chunk ch of source row o >= 1 of a span: in the side buffer, or in the cache when that was full
            auto further = [&](const int4& s, int o, int ch) -> const uint4* {
                const int k = s.w + o - 1;
                if (k < L.side_rows) return reinterpret_cast<const uint4*>(sSide) + k * CPR + ch;
                int slot, gq;
                head_block(P, x.j, x.h, (STREAM ? x.kg * HEADS : 0) + ch / (2 * CPH), slot, gq);
                return reinterpret_cast<const uint4*>((const __nv_bfloat16*)(x.kv ? P.src_v[slot] : P.src_k[slot]) +
                                                      (long long)gq * P.sh + (long long)(unsigned)s.x * 8 + o * P.ss +
                                                      (ch % (2 * CPH)) * 8);
            };
            bool ok = W.wait(bar(kBarEntFull + ent_cnt % kEntTabs), (ent_cnt / kEntTabs) & 1) &&
                      W.wait(bar(kBarSideFull), ent_cnt & 1);
            for (int kb = 0; kb < L.nblk && ok; ++kb) {
                uint32_t si = sp.idx + kb, ph = sp.phase;
                if (si >= NS) { si -= NS; ph ^= 1; }
                ok = W.wait(bar(kBarFull + si), ph);
            }
            if (!ok) break;
            if (!rot) {
                // passes step by a multiple of 8 rows, so a thread's chunk keeps its place in the swizzled row
                static_assert(kRowsV % 8 == 0, "swizzle phase");
                const int ch = xt % CPR, r0 = xt / CPR;
                uint8_t* at0 = a_block(ch >> 3) + (((ch & 7) ^ (r0 & 7)) << 4);
#pragma unroll 1
                for (int row = r0; row < multi; row += kRowsV) {
                    const int4 s = ent[row];
                    uint4* at = reinterpret_cast<uint4*>(at0 + row * 128);
                    float acc[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) acc[k] = 0.f;
                    if (s.y > 0) add8(acc, *at);
#pragma unroll 1
                    for (int o = 1; o < s.y; ++o) add8(acc, *further(s, o, ch));
                    *at = pack8(acc, s.y == 2 ? 0.5f : s.y > 0 ? __frcp_rn((float)s.y) : 0.f);
                }
            } else {
                static_assert(kRowsK % 8 == 0, "swizzle phase");
                const int r0 = xt / CPH;
                // this thread's chunks of row 0: first and second of each head's pairs
                uint8_t *lo0[HEADS], *hi0[HEADS];
#pragma unroll
                for (int q = 0; q < HEADS; ++q) {
                    const int cl = q * 2 * CPH + cp, ch = cl + CPH;
                    lo0[q] = a_block(cl >> 3) + (((cl & 7) ^ (r0 & 7)) << 4);
                    hi0[q] = a_block(ch >> 3) + (((ch & 7) ^ (r0 & 7)) << 4);
                }
                int row = r0;
#pragma unroll 1
                for (; row < multi; row += kRowsK) {
                    const int4 s = ent[row];
                    constexpr int HP = HEADS < 2 ? 1 : 2;   // heads that share one (cos, sin)
#pragma unroll
                    for (int q = 0; q < HEADS; q += HP) {
                        float a0[HP][8], a1[HP][8];
#pragma unroll
                        for (int u = 0; u < HP; ++u)
#pragma unroll
                            for (int i = 0; i < 8; ++i) a0[u][i] = a1[u][i] = 0.f;
#pragma unroll 1
                        for (int o = 0; o < s.y; ++o) {
                            int pos = min(s.z + o, P.max_position - 1);   // the plan reports what is clamped
                            if (o > 0 && P.src_pos) {
                                const int2 at = __ldg(&L.rows[(size_t)x.tile * kTileM + row].where);
                                pos = src_pos_of(P, at.x, at.y + o);
                            }
                            float2 cs[8];
                            cs8(pos, cs);
#pragma unroll
                            for (int u = 0; u < HP; ++u) {
                                const uint4* lo = reinterpret_cast<const uint4*>(lo0[q + u] + row * 128);
                                const uint4* hi = reinterpret_cast<const uint4*>(hi0[q + u] + row * 128);
                                if (o > 0) {
                                    lo = further(s, o, (q + u) * 2 * CPH + cp);
                                    hi = lo + CPH;
                                }
                                unrotate8(*lo, *hi, cs, a0[u], a1[u]);
                            }
                        }
                        const float inv = s.y == 2 ? 0.5f : s.y > 0 ? __frcp_rn((float)s.y) : 0.f;
#pragma unroll
                        for (int u = 0; u < HP; ++u) {
                            *reinterpret_cast<uint4*>(lo0[q + u] + row * 128) = pack8(a0[u], inv);
                            *reinterpret_cast<uint4*>(hi0[q + u] + row * 128) = pack8(a1[u], inv);
                        }
                    }
                }
#pragma unroll 1
                for (; row < tokens; row += kRowsK) {   // one source row: one (cos, sin) for every head
                    float2 cs[8];
                    cs8(ent[row].z, cs);
#pragma unroll
                    for (int q = 0; q < HEADS; ++q) {
                        uint4 *lo = reinterpret_cast<uint4*>(lo0[q] + row * 128), *hi = reinterpret_cast<uint4*>(hi0[q] + row * 128);
                        float a0[8], a1[8];
                        unrotate8_first(*lo, *hi, cs, a0, a1);
                        *lo = pack8(a0);
                        *hi = pack8(a1);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(kBarSideEmpty));
                mbar_arrive(bar(kBarEntEmpty + ent_cnt % kEntTabs));
            }
            ++ent_cnt;
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarKReady + kr_idx));
            if (++kr_idx == NKR) kr_idx = 0;
            for (int kb = 0; kb < L.nblk; ++kb) sp.adv(NS);
        }
    } else if (warp < kSideWarp) {
        // ------------------------------------------------------------ gather
        // A lane holds the plan words of rows lane and lane + 32 of its warp's 64; 8 lanes copy the 128 bytes of
        // a row's K-block, the row's offset passed to them by a shuffle.
        constexpr int kRows = kTileM / kNumGatherWarps;
        static_assert(kRows == 64, "two plan words a lane");
        const int row0 = (warp - kGatherWarp0) * kRows, c = lane & 7, r0 = row0 + (lane >> 3);
        Slot sp{0, 0};
        uint32_t ent_cnt = 0;
        bool ok = true;
        int2 cur[2], nxt[2];   // {offset, rows}
        auto fetch = [&](int tile) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
                nxt[i] = __ldg(reinterpret_cast<const int2*>(&L.rows[(size_t)tile * kTileM + row0 + 32 * i + lane].src));
        };
        RWalker<STREAM> x(P, L, sWalk);
        if (x.more()) fetch(x.tile);
        for (; x.more() && ok; x.next()) {
            cur[0] = nxt[0];
            cur[1] = nxt[1];
            if (MODE == kDiag && blockIdx.x == 0 && x.it + 1 == P.stall_unit1) break;
            // the prologue's copy of the tile's row entries
            if (!W.wait(bar(kBarEntEmpty + ent_cnt % kEntTabs), ((ent_cnt / kEntTabs) & 1) ^ 1)) break;
#pragma unroll
            for (int i = 0; i < 2; ++i)
                cp_async16(smem_u32(sEnt + (ent_cnt % kEntTabs) * kTileM + row0 + 32 * i + lane),
                           &L.rows[(size_t)x.tile * kTileM + row0 + 32 * i + lane].src);
            cp_async_arrive(bar(kBarEntFull + ent_cnt % kEntTabs));
            ++ent_cnt;
            fetch(x.next_tile());
            const unsigned copy[2] = {__ballot_sync(0xffffffffu, cur[0].y > 0), __ballot_sync(0xffffffffu, cur[1].y > 0)};
            for (int kb = 0; kb < L.nblk; ++kb) {
                const int q = kb / (2 * HS / kBlockK), c0 = (kb - q * (2 * HS / kBlockK)) * kBlockK;
                int src_slot, gq;
                head_block(P, x.j, x.h, (STREAM ? x.kg * HEADS : 0) + q, src_slot, gq);
                const __nv_bfloat16* head = (const __nv_bfloat16*)(x.kv ? P.src_v[src_slot] : P.src_k[src_slot]) +
                                            (long long)gq * P.sh;
                if (!W.wait(bar(kBarEmpty + sp.idx), sp.phase ^ 1)) { ok = false; break; }
                uint8_t* block = sRing + sp.idx * kBlockBytes;
                // row r0 + 4 i: 16-byte chunk c, swizzled by the row's low bits (two values over i)
                const uint32_t dst = smem_u32(block) + r0 * 128;
                const uint32_t x0 = ((uint32_t)c ^ ((uint32_t)r0 & 7)) << 4, x1 = x0 ^ 64;
                const uint4* from = reinterpret_cast<const uint4*>(head + c0 + c * 8);
#pragma unroll
                for (int i = 0; i < kRows / 4; ++i) {
                    const int r = (i & 7) * 4 + (lane >> 3);
                    const uint32_t off = (uint32_t)__shfl_sync(0xffffffffu, cur[i >> 3].x, r);
                    if (copy[i >> 3] >> r & 1) cp_async16(dst + i * 512 + (i & 1 ? x1 : x0), from + off);
                }
                cp_async_arrive(bar(kBarFull + sp.idx));
                sp.adv(NS);
            }
        }
        cp_async_wait_all();
    } else {
        // ------------------------------------------------------------ side buffer: [further row][input row]
        constexpr int CPH2 = HS / 4, CPR = HEADS * CPH2, kAtOnce = 32 / CPR;   // chunks of a head, of a row; rows a copy
        const int ch = lane % CPR, sub = lane / CPR;
        const uint32_t dst = smem_u32(sSide) + lane * 16;
        uint32_t cnt = 0;
        int n_nxt = 0;
        unsigned off_nxt[kSideMax / 32];   // lane: offsets of further rows lane, lane + 32, ...
        auto fetch = [&](int tile) {
            n_nxt = __ldg(&L.tiles[tile].count.z);
#pragma unroll
            for (int i = 0; i < kSideMax / 32; ++i) off_nxt[i] = __ldg(&L.tiles[tile].side[32 * i + lane]);
        };
        RWalker<STREAM> x(P, L, sWalk);
        if (x.more()) fetch(x.tile);
        for (; x.more(); x.next(), ++cnt) {
            const int n = min(n_nxt, L.side_rows);
            unsigned off[kSideMax / 32];
#pragma unroll
            for (int i = 0; i < kSideMax / 32; ++i) off[i] = off_nxt[i];
            fetch(x.next_tile());
            int slot, gq;
            head_block(P, x.j, x.h, (STREAM ? x.kg * HEADS : 0) + ch / CPH2, slot, gq);
            const uint4* from = reinterpret_cast<const uint4*>(
                (const __nv_bfloat16*)(x.kv ? P.src_v[slot] : P.src_k[slot]) + (long long)gq * P.sh + (ch % CPH2) * 8);
            if (!W.wait(bar(kBarSideEmpty), (cnt & 1) ^ 1)) break;
#pragma unroll
            for (int i = 0; i < kSideMax / 32; ++i) {
                if (32 * i >= n) break;
#pragma unroll 8
                for (int k = 0; k < 32; k += kAtOnce) {
                    const unsigned o = __shfl_sync(0xffffffffu, off[i], k + sub);
                    if (32 * i + k + sub < n) cp_async16(dst + (32 * i + k) * CPR * 16, from + o);
                }
            }
            cp_async_arrive(bar(kBarSideFull));
        }
        cp_async_wait_all();
    }
    if (DENSE && dense > 0) {
        __syncthreads();   // everyone has read what the shared memory held
        if (threadIdx.x == 0)
            barriers([&](int i, int) { mbar_inval(bar(i)); });
        __syncthreads();
        window::translate_body<2 * HS, false, false>(P, D, smem, tmem_base);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, L.tmem_cols);
    }
}

// Row plan of target tokens [t_begin, t_end) (layout: see the top), one tile per CTA, one token per
// thread.  It also writes the window plan of the same tokens (kvx_span_plan.cuh).
__global__ void __launch_bounds__(kTileM) span_rows_kernel(const __grid_constant__ TranslateParams P, int t_begin, int t_end,
                                                           int cap_rows, int4* __restrict__ hdr, int4* __restrict__ win,
                                                           TilePlan* __restrict__ tiles, RowEnt* __restrict__ rows)
{
    constexpr int kClasses = 5;   // 0: four rows and more, 1: three, 2: two or none, 3: one, 4: past the last token
    __shared__ int cnt[kClasses][kTileM / 32];
    __shared__ int more[kTileM];   // [rank]: further rows
    __shared__ int out[kTileM / 32];
    // the previous launch in the stream may still read the plan
    grid_dependency_wait();
    grid_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SeqView sv{P.seq_off, P.src_seq_len, P.batch};
    const int tp = t_begin + (int)blockIdx.x * kTileM + (int)threadIdx.x;
    const bool valid = tp < t_end;
    int b = -1, lo = 0, hi = 0;
    if (valid) resolve_src(P, sv, tp, load_span(P, tp), b, lo, hi);
    const bool inwin = write_window_plan(valid, b, lo, hi, (int)blockIdx.x * (kTileM / 32) + warp, lane, cap_rows, hdr, win);
    const int n = valid ? hi - lo : -1;
    // (a tile's sums are at most 128 x 2048 = kRowsMax)
    const int out_rows = __reduce_add_sync(0xffffffffu, inwin || n < 0 ? 0 : min(n, kRowsMax / kTileM));
    if (lane == 0) out[warp] = out_rows;
    const int cls = n < 0 ? 4 : n == 1 ? 3 : n >= 4 ? 0 : n == 3 ? 1 : 2;
    int rank = 0;   // among the earlier lanes of the same class
#pragma unroll
    for (int k = 0; k < kClasses; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, cls == k);
        if (lane == 0) cnt[k][warp] = __popc(m);
        if (cls == k) rank = __popc(m & ((1u << lane) - 1u));
    }
    __syncthreads();
    int multi = 0, tokens = 0;
#pragma unroll
    for (int k = 0; k < kClasses; ++k)
#pragma unroll
        for (int w = 0; w < kTileM / 32; ++w) {
            const int c = cnt[k][w];
            if (k < cls || (k == cls && w < warp)) rank += c;
            if (k < 3) multi += c;
            if (k < 4) tokens += c;
        }
    more[rank] = n > 1 ? n - 1 : 0;
    __syncthreads();
    // further rows of the ranks before (only the first `multi` ranks have any)
    int side = 0;
    for (int r = 0; r < rank && r < multi; ++r) side += more[r];
    TilePlan& tile = tiles[blockIdx.x];
    if (rank == kTileM - 1)
        tile.count = make_int4(multi, tokens, min(side + more[rank], kRowsMax), out[0] + out[1] + out[2] + out[3]);
    RowEnt& row = rows[(size_t)blockIdx.x * kTileM + rank];
    if (!valid) {
        row.src = make_int4(0, -1, 0, 0);
        row.dst = make_int4(-1, -1, 0, 0);
        return;
    }
    long long dst_off;
    int pt;
    resolve_dst(P, sv, tp, dst_off, pt);
    const long long off = (long long)b * P.sb + (long long)lo * P.ss;
    int pos = 0;
    for (int o = 0; o < n; ++o) {
        const int p = P.rs.enabled ? src_pos_of(P, b, lo + o) : 0;
        if (o == 0) pos = p;
        else if (side + o - 1 < kSideMax) tile.side[side + o - 1] = (unsigned)((off + o * P.ss) >> 3);
    }
    row.src = make_int4((int)(unsigned)(off >> 3), n, pos, side);
    row.dst = make_int4((int)(unsigned)(dst_off & 0xffffffffll), (int)(dst_off >> 32), pt, 0);
    row.where = make_int2(b, lo);
}

// Shared-memory layout; false: this geometry takes the window kernel.
bool rows_layout(int in_dim, int dt, int ds, int share, RowsLaunch& L)
{
    const TcConfig c = tc_config(in_dim, dt, ds, share);
    const int width = in_dim < 256 ? in_dim : 256;   // channels of a K group
    if (!c.ok || c.hpu != 1 || in_dim % width || width == 3 * ds) return false;
    L.n_tile = c.n_tile;
    L.n_split = c.n_split;
    L.nblk = width / kBlockK;
    L.kgs = in_dim / width;
    L.b_bytes = (unsigned)(in_dim * L.n_tile * 2);
    // weights: the group's image with one K group, else a ring of K-blocks (also where the image of several K
    // groups would fit: 512 channels onto 64), since only the streaming form walks K groups
    constexpr unsigned kWeightBytes = 65536;
    L.nb = 0;
    if (L.kgs > 1) {
        L.nb = (int)(kWeightBytes / (unsigned)(L.n_tile * 128));
        if (L.nb > kMaxB) L.nb = kMaxB;
    }
    L.stage_row_bytes = (unsigned)(L.n_tile * 2 + 16);
    unsigned off = 0;
    auto take = [&](unsigned bytes, unsigned align) {
        off = (off + align - 1) / align * align;
        const unsigned o = off;
        off += bytes;
        return o;
    };
    L.off_b = take(L.nb ? (unsigned)(L.nb * L.n_tile * 128) : L.b_bytes, 1024);
    L.off_stage = take(kTileM * L.stage_row_bytes, 128);
    L.off_bar = take(kNumBars * 8, 8);
    L.off_misc = take(16 + sizeof(RWalkStart) + sizeof(int), 16);
    L.off_turns = take((unsigned)(ds / 2 + dt / 2) * 8, 16);
    L.off_ent = take(kEntTabs * kTileM * sizeof(int4), 16);
    L.off_ring = take(0, 1024);
    // K-block slots, of which a tile needs nblk, and the side buffer behind them: a tile of spans
    // averaging 1.3 rows has 38 further rows
    const int avail = kSmemMax - 1024 - (int)L.off_ring, row = width * 2;
    int slots = (avail - 40 * row) / kBlockBytes;
    if (avail < 0 || slots < L.nblk) return false;
    L.nslots = slots < kMaxSlots ? slots : kMaxSlots;
    L.off_side = L.off_ring + (unsigned)L.nslots * kBlockBytes;
    const int fit = (avail - L.nslots * kBlockBytes) / row;
    L.side_rows = fit < kSideMax ? fit : kSideMax;
    // Where the two sides meet: heads of 64 keep more lanes on a row.  Over 57 geometries and 21 laws of spans (1.3 to
    // 12 rows, disjoint and overlapping, even and uneven) the side taken is 0.8% above the faster one on average, and
    // at most 34% (128-channel heads, a tenth of the tokens with 16 rows).
    L.dense_sum = ds == 64 ? (L.kgs > 1 ? 240 : 300) : ds == 128 ? 220 : 165;
    L.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(L.n_tile >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
    unsigned cols = 32;
    while (cols < 2u * (unsigned)L.n_tile) cols <<= 1;
    L.tmem_cols = cols;
    return cols <= 512;
}

template <int HS, int HEADS, bool STREAM, int MODE>
cudaError_t launch_rows_v(int grid, cudaStream_t stream, const TranslateParams& P, const RowsLaunch& L,
                          const window::TcLaunch& D)
{
    const cudaError_t e = smem_opt_in<translate_rows_kernel<HS, HEADS, STREAM, MODE>>(kSmemMax);
    if (e != cudaSuccess) return e;
    return launch_pdl(translate_rows_kernel<HS, HEADS, STREAM, MODE>, grid, kThreads, kSmemMax, stream, P, L, D);
}
template <int HS, int HEADS, bool STREAM>
cudaError_t launch_rows_s(int grid, int mode, cudaStream_t stream, const TranslateParams& P, const RowsLaunch& L,
                          const window::TcLaunch& D)
{
    // (one shape is compiled for the diagnostics, to save the others' compile time)
    if constexpr (HS == 64 && HEADS == 2)
        if (mode == kDiag) return launch_rows_v<HS, HEADS, STREAM, kDiag>(grid, stream, P, L, D);
    return mode == kDense ? launch_rows_v<HS, HEADS, STREAM, kDense>(grid, stream, P, L, D)
                          : launch_rows_v<HS, HEADS, STREAM, kPlain>(grid, stream, P, L, D);
}
template <int HS, int HEADS>
cudaError_t launch_rows(int grid, int mode, cudaStream_t stream, const TranslateParams& P, const RowsLaunch& L,
                        const window::TcLaunch& D)
{
    return L.kgs > 1 ? launch_rows_s<HS, HEADS, true>(grid, mode, stream, P, L, D)
                     : launch_rows_s<HS, HEADS, false>(grid, mode, stream, P, L, D);
}

}  // namespace

bool rows_supported(int in_dim, int dt, int ds, int share)
{
    RowsLaunch L{};
    return rows_layout(in_dim, dt, ds, share, L);
}

bool rows_offsets_fit(const TranslateParams& P)
{
    return (long long)P.batch * P.sb + (long long)P.src_max_seq * P.ss < (1ll << 35);
}

size_t rows_plan_bytes(int tokens)
{
    const size_t tiles = (size_t)(tokens + kTileM - 1) / kTileM;
    return tiles * (kTileM * sizeof(RowEnt) + sizeof(TilePlan));
}

cudaError_t launch_translate_rows(const TranslateParams& P, int num_sms, void* window_plan, void* plan, int plan_tokens,
                                  cudaStream_t stream, int* launches)
{
    *launches = 0;
    RowsLaunch L{};
    window::TcLaunch D{};
    const int share = share_heads(P);
    if (!rows_layout(P.in_dim, P.dt, P.ds, share, L) || !window::tc_layout(P.in_dim, P.dt, P.ds, share, D) ||
        D.np != 1 || D.tmem_cols != L.tmem_cols)
        return cudaErrorNotSupported;
    const int chunk = plan_tokens / kTileM * kTileM;
    if (chunk <= 0 || !plan || !window_plan) return cudaErrorInvalidValue;
    int4* hdr = reinterpret_cast<int4*>(window_plan);
    int4* win = hdr + (chunk + 31) / 32;
    RowEnt* rows = reinterpret_cast<RowEnt*>(plan);
    TilePlan* tiles = reinterpret_cast<TilePlan*>(rows + chunk);
    L.tiles = tiles;
    L.rows = rows;
    // the source may hold 1.5 rows or more for each target token (what the host knows: the caches' capacity)
    const bool dense = P.span_lo && 2ll * P.batch * P.src_max_seq >= 3ll * P.T_total;
    const int mode = P.wait_ns != 0 || P.stall_unit1 != 0 ? kDiag : dense ? kDense : kPlain;
    L.share = share > 1 && P.Ht % share == 0 ? share : 1;
    for (int t0 = 0; t0 < P.T_total; t0 += chunk) {
        const int t1 = P.T_total - t0 < chunk ? P.T_total : t0 + chunk;
        L.m_tiles = (t1 - t0 + kTileM - 1) / kTileM;
        const long long UH = (long long)P.Lt * P.Ht * L.n_split * L.m_tiles;
        const int grid = (int)(UH < num_sms ? UH : num_sms);
        if (window::tc_launch(P, t0, t1, hdr, win, num_sms, D) != grid) return cudaErrorInvalidValue;
        if (grid % L.share) L.share = 1;
        cudaError_t e = launch_pdl(span_rows_kernel, L.m_tiles, kTileM, 0, stream, P, t0, t1, kWindowRows, hdr, win, tiles, rows);
        if (e != cudaSuccess) return e;
        ++*launches;
        switch (P.ds * 8 + L.nblk * kBlockK / P.ds) {   // source heads of a K group
        case 64 * 8 + 1: e = launch_rows<32, 1>(grid, mode, stream, P, L, D); break;
        case 64 * 8 + 2: e = launch_rows<32, 2>(grid, mode, stream, P, L, D); break;
        case 64 * 8 + 4: e = launch_rows<32, 4>(grid, mode, stream, P, L, D); break;
        case 128 * 8 + 1: e = launch_rows<64, 1>(grid, mode, stream, P, L, D); break;
        case 128 * 8 + 2: e = launch_rows<64, 2>(grid, mode, stream, P, L, D); break;
        case 256 * 8 + 1: e = launch_rows<128, 1>(grid, mode, stream, P, L, D); break;
        default: return cudaErrorNotSupported;
        }
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

}  // namespace kvx
