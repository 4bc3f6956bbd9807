// svt_kernels.cu -- sm_103a kernels of the SVT track-fitting chain.
//
// Stages (arXiv:1312.0917, Sec. II-A: unpack, combine, fit), followed by the
// chi-square cut and the hit-warrior:
//
//   P0  word spans (one per warp): count EE / EP words, check every word's fields
//   P1  word spans: decode the roads whose header lies in the span (header,
//       XFT track, hits ranked per layer), enforce the grammar and limits
//   P2  events: flag the hits a road shares with another road of the event
//       that holds its coordinates on >= 3 layers (the cross-road candidates)
//   P3  roads: combinations, fit, chi-square, cut and the road-local part of
//       the hit-warrior; publish cross-road group minima for flagged groups
//   P4  candidate roads: finish the hit-warrior across roads, count survivors
//   P5  road chunks: write the surviving tracks in (event, road, comb) order
//
// SVT_PLAIN runs P0, P1, P2, a combination scan, a fit kernel with one thread
// per combination that stores every key and track parameter in HBM, the
// warrior, P4 and P5 as separate kernels.  SVT_PERSISTENT runs all phases in
// one cooperative kernel separated by grid barriers whose waits are bounded,
// and evaluates each distinct fit once from per-hit partial sums kept in
// shared memory.  Both produce identical tracks.
//
// Integer exactness (the reason the fit runs in 32-bit): svt_load_constants
// admits only constant sets for which every partial and full sum of
// coefficient x input (+ 4096 x offset) stays below 2^31 in magnitude, so
// int32 accumulation equals the int64 sum; an arithmetic right shift by 12
// is floor division by 4096, and floor(s / 4096) + k == floor((s + 4096 k) /
// 4096).  chi2 < 2^38, so the track key (chi2 << 23 | road << 15 | comb)
// is a 61-bit integer ordered like (chi2, road, comb).
//
// The block size of every kernel is SVT_BLOCK (256 unless the including
// file sets it); each block size builds in a namespace of its own, and only
// the 256-thread build holds the plain pipeline.
#include <cstddef>

#include "svt_internal.h"

#ifndef SVT_BLOCK
#define SVT_BLOCK 256
#endif
#if SVT_BLOCK == 128
#define SVT_KNS b128
#elif SVT_BLOCK == 256
#define SVT_KNS b256
#elif SVT_BLOCK == 512
#define SVT_KNS b512
#else
#error "SVT_BLOCK must be 128, 256 or 512"
#endif

namespace svt {
namespace SVT_KNS {

constexpr int BLOCK = SVT_BLOCK;           // threads per CTA, every kernel of this build
constexpr int WARPS = BLOCK / 32;
constexpr int GRID_MAX = MAX_SPANS / WARPS < MAX_GRID ? MAX_SPANS / WARPS : MAX_GRID;

#define FULL_MASK 0xffffffffu

// ---------------------------------------------------------------------------
// small device helpers
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ unsigned warp_id() { return threadIdx.x >> 5; }

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// loads of data written earlier in the same launch by other CTAs: L2 only
template <class T>
__device__ __forceinline__ T ldcg(const T *p) { return __ldcg(p); }
template <>
__device__ __forceinline__ RoadRec ldcg(const RoadRec *p)
{
    static_assert(sizeof(RoadRec) == 16, "RoadRec is one 16-byte load");
    uint4 v = __ldcg(reinterpret_cast<const uint4 *>(p));
    RoadRec r;
    memcpy(&r, &v, sizeof r);
    return r;
}

__device__ __forceinline__ void raise_flag(const Dev &d, unsigned f)
{
    atomicOr(&d.ctrl->sync, (unsigned long long)f << 32);
}

// the flags raised before this kernel
__device__ __forceinline__ unsigned flags_of(const Dev &d) { return (unsigned)(ldcg(&d.ctrl->sync) >> 32); }

// a fault of the stream at word err >> 8 of rank err & 255
__device__ __forceinline__ void report(const Dev &d, unsigned long long err)
{
    atomicMax(&d.ctrl->err_inv, ~err);
    raise_flag(d, FLAG_FAULT);
}

// Survivor slot s of road g.  Slots are slot-major, so the first survivors
// of consecutive roads are adjacent (the output stage reads them in road
// order).
__device__ __forceinline__ size_t surv_at(const Dev &d, unsigned g, unsigned s)
{
    return (size_t)s * d.max_roads + g;
}

__device__ __forceinline__ bool word_ok(uint32_t w)
{
    uint32_t type = (w >> 27) & 7u, pl = w & 0x07FFFFFFu;
    if ((w >> 31) && !((w >> 30) & 1u))
        return false;                                   // EE without EP
    if (type <= 4)
        return (pl >> 12) == 0;
    if (type <= 6)
        return (pl >> 16) == 0;
    return (pl >> 10) == 0 && (pl & 15u) < 12 && ((pl >> 4) & 7u) < 6 && ((pl >> 7) & 7u) < 5;
}

// combinations of a road (product of its five hit counts) and its distinct
// fits (product over the four fitted layers: the excluded layer's hit does not
// enter the fit), from RoadRec::pk
// combinations N (at most 8^5) and distinct fits N4 of a road record
__device__ __forceinline__ void road_sizes(uint32_t pk, unsigned &N, unsigned &N4)
{
    const unsigned excl = (pk >> 20) & 7u;
    N = 1;
    N4 = 1;
    for (unsigned l = 0; l < N_LAYERS; ++l) {
        const unsigned n = (pk >> (4 * l)) & 15u;
        N *= n;
        if (l != excl)
            N4 *= n;
    }
}

// floor(x / m) for 1 <= m <= 8 and x < 2^16 with M = ceil(2^31 / m):
// (2x)(2^31 + e) / (m 2^32) = x / m + 2 x e / (m 2^32) with e < m, and
// 2 x e < 2^32, so the high word of 2x * M is the quotient (32-bit
// multiply-high, no 64-bit product).
__device__ __forceinline__ unsigned divm(unsigned x, unsigned M) { return __umulhi(x << 1, M); }
__host__ __device__ constexpr unsigned magic(unsigned m) { return (unsigned)(((1ull << 31) + m - 1) / m); }
// magic(m) for the hit counts m = 1..8 (entry 0 repeats m = 1)
__device__ __constant__ unsigned c_magic[MAX_HITS + 1] = {
    magic(1), magic(1), magic(2), magic(3), magic(4), magic(5), magic(6), magic(7), magic(8)};

template <class T>
__device__ __forceinline__ T warp_sum(T v)
{
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v)
{
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long u = __shfl_xor_sync(FULL_MASK, v, o);
        v = u < v ? u : v;
    }
    return v;
}

// block-wide exclusive scan of one unsigned long long per thread
__device__ unsigned long long block_excl_scan(unsigned long long v, unsigned long long *total)
{
    __shared__ unsigned long long s_w[WARPS + 1];
    unsigned long long inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long n = __shfl_up_sync(FULL_MASK, inc, o);
        if ((int)lane_id() >= o)
            inc += n;
    }
    if (lane_id() == 31)
        s_w[warp_id()] = inc;
    __syncthreads();
    if (warp_id() == 0) {
        unsigned long long x = lane_id() < WARPS ? s_w[lane_id()] : 0, xi = x;
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long n = __shfl_up_sync(FULL_MASK, xi, o);
            if ((int)lane_id() >= o)
                xi += n;
        }
        if (lane_id() < WARPS)
            s_w[lane_id()] = xi - x;
        if (lane_id() == WARPS - 1)
            s_w[WARPS] = xi;
    }
    __syncthreads();
    unsigned long long r = s_w[warp_id()] + inc - v;
    if (total)
        *total = s_w[WARPS];
    __syncthreads();
    return r;
}

// the same for one unsigned per thread (32-bit sums)
__device__ unsigned block_excl_scan32(unsigned v, unsigned *total)
{
    __shared__ unsigned s_w32[WARPS + 1];
    unsigned inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned n = __shfl_up_sync(FULL_MASK, inc, o);
        if ((int)lane_id() >= o)
            inc += n;
    }
    if (lane_id() == 31)
        s_w32[warp_id()] = inc;
    __syncthreads();
    if (warp_id() == 0) {
        const unsigned x = lane_id() < WARPS ? s_w32[lane_id()] : 0u;
        unsigned xi = x;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned n = __shfl_up_sync(FULL_MASK, xi, o);
            if ((int)lane_id() >= o)
                xi += n;
        }
        if (lane_id() < WARPS)
            s_w32[lane_id()] = xi - x;
        if (lane_id() == WARPS - 1)
            s_w32[WARPS] = xi;
    }
    __syncthreads();
    const unsigned r = s_w32[warp_id()] + inc - v;
    *total = s_w32[WARPS];
    __syncthreads();
    return r;
}

// block-wide sums of two unsigned long long per thread, one exchange
__device__ void block_sum2(unsigned long long &a, unsigned long long &b)
{
    __shared__ unsigned long long s_ab[2 * WARPS];   // a of each warp, then b
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane_id() == 0) {
        s_ab[warp_id()] = a;
        s_ab[WARPS + warp_id()] = b;
    }
    __syncthreads();
    a = 0;
    b = 0;
#pragma unroll
    for (unsigned w = 0; w < WARPS; ++w) {
        a += s_ab[w];
        b += s_ab[WARPS + w];
    }
    __syncthreads();
}

__device__ unsigned long long block_sum(unsigned long long v)
{
    unsigned long long t;
    block_excl_scan(v, &t);
    return t;
}

// Exclusive scan of in[0..n) into out[0..n) by one CTA; returns the total.
template <class TI, class TO>
__device__ unsigned long long block_scan_array(const TI *in, TO *out, unsigned n)
{
    unsigned long long carry = 0;
    for (unsigned base = 0; base < n; base += BLOCK) {
        unsigned i = base + threadIdx.x;
        unsigned long long v = i < n ? (unsigned long long)ldcg(in + i) : 0ull, tot;
        unsigned long long ex = block_excl_scan(v, &tot);
        if (i < n)
            out[i] = (TO)(carry + ex);
        carry += tot;
    }
    return carry;
}

// true in the CTA that arrives last at `counter` (all earlier CTAs' writes
// are visible to it)
__device__ bool last_block(unsigned *counter, unsigned nblocks)
{
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(counter, 1u) == nblocks - 1;
    }
    __syncthreads();
    if (s_last)
        __threadfence();
    return s_last;
}

// Every CTA of a batch's last kernel leaves through here, on every path.  The
// last one copies the control block out, to the host as well, and clears it
// for the next batch.  A memset in front of the kernel and a copy behind it
// did this before: two more commands in the stream, 4.0 us of a batch (35.8 ->
// 31.8 us around a kernel of 21 us).  wrote: thread 0 has, or may have, written the
// control block since the last barrier (a CTA that has not need not wait here for
// its tracks to land: 0.5 us).
__device__ void leave(const Dev &d, bool finished, bool wrote)
{
    __shared__ unsigned s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        if (wrote)
            __threadfence();
        s_last = atomicAdd(&d.ctrl->done[0], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last)
        return;
    __threadfence();
    static_assert(sizeof(Ctrl) % 8 == 0 && sizeof(Ctrl) / 8 <= BLOCK, "one word per thread");
    unsigned long long *c = reinterpret_cast<unsigned long long *>(d.ctrl);
    const unsigned i = threadIdx.x;
    if (i < sizeof(Ctrl) / 8) {
        unsigned long long v = ldcg(c + i);
        if (finished && i == offsetof(Ctrl, t_phase) / 8 + 6)
            v = globaltimer_ns();
        reinterpret_cast<unsigned long long *>(d.last)[i] = v;
        if (d.host)
            reinterpret_cast<unsigned long long *>(d.host)[i] = v;
        c[i] = 0;
    }
}

// next item of work queue q for the whole CTA
__device__ unsigned grab(const Dev &d, int q)
{
    __shared__ unsigned s_item;
    __syncthreads();
    if (threadIdx.x == 0)
        s_item = atomicAdd(&d.ctrl->q[q], 1u);
    __syncthreads();
    return s_item;
}

// Work queue q where every CTA's first item is its own index: the queue
// hands out items gridDim.x, gridDim.x + 1, ... (one claim per later item,
// none at the start, when every CTA would claim at once on one counter)
__device__ __forceinline__ unsigned grab_after_first(const Dev &d, int q)
{
    return gridDim.x + grab(d, q);
}

// A warp's items out of n for n_warps warps: `quarters` of four are dealt out in
// turn (warp wi: wi, wi + n_warps, ..), the rest, which evens the warps out, one
// by one from queue head q.  (All from the queue, 40,000 claims of one counter were
// 80 us: L2 takes about one atomic on an address in 2 ns.)  A half: items take
// unequal times where some roads are fitted twice.  The fit stage with a half / three
// quarters dealt out: 96,000 roads of skewed hit counts 38 / 40 us with hits
// anywhere, 55 / 74 within 64 strips, 63 / 86 within 16; 19,200 roads of one to
// eight hits within 16 strips 67 / 72; the uneven batch 85 / 84.
struct Share {
    unsigned n, n_warps, dealt;   // items dealt out
    unsigned *q;
    __device__ Share(unsigned n_, unsigned n_warps_, unsigned quarters, unsigned *q_)
        : n(n_), n_warps(n_warps_),
          dealt(n_ <= n_warps_ ? n_ : max(n_ / 4 * quarters / n_warps_, 1u) * n_warps_), q(q_)
    {
    }
    __device__ unsigned first(unsigned wi) const { return wi < dealt ? wi : ~0u; }   // (dealt is 0 or covers a turn)
    // the item after item i, or one past n
    __device__ unsigned next(unsigned i)
    {
        if (i + n_warps < dealt)
            return i + n_warps;
        if (dealt >= n)
            return ~0u;
        unsigned c = 0;
        if (lane_id() == 0)
            c = atomicAdd(q, 1u);
        return dealt + __shfl_sync(FULL_MASK, c, 0);
    }
};

// Grid barrier number k (1, 2, ..) of the persistent kernel; `flags` gets
// FLAG_* as they are once every CTA has arrived.  All CTAs are co-resident
// (cooperative launch).  The wait is bounded by d.wait_ns; on expiry the CTA
// raises FLAG_TIMEOUT and every CTA that sees the flag stops working.  Bound:
// L2 round trips.  The arrival returns nothing, and a poll reads the count and
// the flags as one word, so that a CTA leaves one trip after the last arrival
// (with the arrival's old value awaited and the flags loaded after the wait a
// barrier took 0.9 us more).
__device__ bool grid_sync(const Dev &d, unsigned k, unsigned &flags)
{
    __shared__ unsigned s_flags;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&d.ctrl->sync, 1ull);
        const unsigned target = k * gridDim.x;
        unsigned long long t0 = 0, v;
        // relaxed polls (the fence below orders what follows); the clock is
        // looked at every 16th poll
        for (unsigned it = 1; v = ld_relaxed(&d.ctrl->sync), (int)((unsigned)v - target) < 0; ++it) {
            if ((unsigned)(v >> 32) & FLAG_TIMEOUT)
                break;
            if ((it & 15u) == 0) {
                const unsigned long long t = globaltimer_ns();
                t0 = t0 ? t0 : t;
                if (t - t0 > d.wait_ns) {
                    raise_flag(d, FLAG_TIMEOUT);
                    v |= (unsigned long long)FLAG_TIMEOUT << 32;
                    break;
                }
            }
            __nanosleep(20);
        }
        __threadfence();
        s_flags = (unsigned)(v >> 32);
    }
    __syncthreads();
    flags = s_flags;
    return !(flags & FLAG_TIMEOUT);
}

// The batch's counts as every CTA knows them: events and EP words from the
// totals it sums in P1, the roads of complete events from the control block.
struct Batch {
    unsigned n_events, n_ep, n_roads;
};

// phase timestamp k of the persistent kernel (block 0, thread 0)
__device__ __forceinline__ void stamp(const Dev &d, unsigned k)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        d.ctrl->t_phase[k] = globaltimer_ns();
}

// work-queue indices (Ctrl::q)
enum { Q_P2 = 0, Q_BOX, Q_GROUP, Q_P4, Q_P5, Q_CNT, Q_CSC, Q_P2W };

// ---------------------------------------------------------------------------
// P0 / P1: the word stream, one warp per span.  The stream is cut into
// gridDim.x * WARPS spans of whole 32-word windows; warp w of CTA b owns span
// b * WARPS + w.  P0 counts each span's EE and EP words and the EP words after
// its last EE, and checks every word's fields.  P1 gives each warp the counts
// of the spans before its own (every CTA sums them itself, no CTA scans for
// the others) and decodes the roads whose header lies in the warp's span.
// P0 keeps the EP and EE masks of every window (bit i: word i); they give P1
// the roads that start in it, with their road index, event and place in the
// event; each road is then taken by one lane from its header to its EP word,
// which checks the grammar and ranks each hit in its layer.  A warp follows
// its last road past the end of its span.
// ---------------------------------------------------------------------------

constexpr unsigned WIN = 32;               // words per window: one per lane
constexpr unsigned SEG_EE = 0x80000000u;   // segment word: an EE was seen (low bits: EP words since)

// span i of the stream (0 <= i < gridDim.x * WARPS): words [a, e)
__device__ __forceinline__ void span_of(const Dev &d, unsigned i, unsigned long long &a, unsigned long long &e)
{
    const unsigned long long n = (unsigned long long)gridDim.x * WARPS;
    const unsigned long long per = ((d.n_words + n - 1) / n + WIN - 1) / WIN * WIN;
    a = min((unsigned long long)i * per, d.n_words);
    e = min(a + per, d.n_words);
}

// Join of the segment words of two stretches of words, x before y: the EP
// words since the last EE of both (SEG_EE when either holds an EE).  0 is the
// identity.  Counts stay below 2^31 (a batch holds fewer words).
__device__ __forceinline__ unsigned seg_join(unsigned x, unsigned y)
{
    return (y & SEG_EE) ? y : (x & SEG_EE) | ((x & ~SEG_EE) + y);
}

// segment word of one window from its EE and EP lane masks
__device__ __forceinline__ unsigned seg_window(unsigned em, unsigned pm)
{
    return em ? SEG_EE | (unsigned)__popc((pm >> (31 - __clz(em))) >> 1) : (unsigned)__popc(pm);
}

// In-order fold of one segment word per lane (lane i's stretch before lane
// i + 1's); the result in every lane.
__device__ __forceinline__ unsigned warp_seg_fold(unsigned v)
{
    for (unsigned o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_down_sync(FULL_MASK, v, o);
        if (lane_id() + o < 32)
            v = seg_join(v, u);
    }
    return __shfl_sync(FULL_MASK, v, 0);
}

// the same over the CTA (thread t's stretch before thread t + 1's)
__device__ unsigned block_seg_fold(unsigned v)
{
    __shared__ unsigned s_seg[WARPS];
    v = warp_seg_fold(v);
    if (lane_id() == 0)
        s_seg[warp_id()] = v;
    __syncthreads();
    unsigned r = 0;
#pragma unroll
    for (unsigned w = 0; w < WARPS; ++w)
        r = seg_join(r, s_seg[w]);
    __syncthreads();
    return r;
}

// Nonzero when !word_ok(w), without branches.
__device__ __forceinline__ uint32_t word_bad(uint32_t w)
{
    const uint32_t t = (w >> 27) & 7u;
    const uint32_t allowed = t == 7 ? 0x3FFu : t > 4 ? 0xFFFFu : 0xFFFu;
    const uint32_t pair = w & (w >> 1);   // wedge >= 12: bits 2 and 3; barrel >= 6: bits 5 and 6;
    const uint32_t head = (pair & 0x24u) | ((w | (w >> 1)) & (w >> 2) & 0x80u);   // excl >= 5: bit 9 and 8 or 7
    return (w & 0x07FFFFFFu & ~allowed) | (w & ~(w << 1) & 0x80000000u) | (t == 7 ? head : 0u);
}

// P0 of one warp's span.  A window's EP and EE masks (32 words each) are kept
// for P1, which then finds the roads without reading the words; the counts are
// taken from the masks, a window per lane.  Bound: the words' latency, then
// issue slots (22 instructions a window; 73 when every window was counted and
// checked by itself: 11.9 MB of words 10.8 -> 9.2 us, 16.5 MB 13.9 -> 11.9).
__device__ void scan_count(const Dev &d)
{
    const unsigned lane = lane_id(), sp = blockIdx.x * WARPS + warp_id();
    unsigned long long a, e;
    span_of(d, sp, a, e);
    unsigned ee = 0, ep = 0, seg = 0;
    uint32_t bad = 0;
    constexpr unsigned UNROLL = 8;   // windows whose loads are in flight together
    for (unsigned long long base = a; base < e; base += UNROLL * WIN) {
        uint32_t w[UNROLL];
#pragma unroll
        for (unsigned k = 0; k < UNROLL; ++k) {
            const unsigned long long i = base + k * WIN + lane;
            w[k] = i < e ? __ldg(d.words + i) : 0u;   // (0 is a valid word)
        }
        unsigned pm = 0, em = 0;   // lane k: window k's masks
#pragma unroll
        for (unsigned k = 0; k < UNROLL; ++k) {
            const unsigned m = __ballot_sync(FULL_MASK, (w[k] >> 30) & 1u), n = __ballot_sync(FULL_MASK, w[k] >> 31);
            pm = lane == k ? m : pm;
            em = lane == k ? n : em;
            bad |= word_bad(w[k]);
        }
        if (lane < UNROLL && base + lane * WIN < e)
            d.wmask[base / WIN + lane] = make_uint2(pm, em);
        const unsigned total = __reduce_add_sync(FULL_MASK, __popc(pm));
        ep += total;
        const unsigned last = __ballot_sync(FULL_MASK, em != 0u);
        if (last) {   // EP words after the last EE
            const unsigned lw = 31 - __clz(last);
            ee += __reduce_add_sync(FULL_MASK, __popc(em));
            seg = SEG_EE | __reduce_add_sync(FULL_MASK, lane == lw  ? seg_window(em, pm) & ~SEG_EE
                                                        : lane > lw ? __popc(pm)
                                                                    : 0u);
        } else {
            seg += total;   // (the flag in the top bit stays)
        }
    }
    if (__any_sync(FULL_MASK, bad != 0u)) {   // the first bad word, one window at a time
        unsigned long long first = ~0ull;
        for (unsigned long long i = a + lane; i < e && first == ~0ull; i += WIN)
            if (!word_ok(__ldg(d.words + i)))
                first = i;
        first = warp_min_u64(first);
        if (lane == 0)
            report(d, (first << 8) | RANK_BAD);
    }
    __shared__ unsigned s_cnt[3][WARPS];
    if (lane == 0) {
        d.span_ee[sp] = ee;
        d.span_ep[sp] = ep;
        d.span_seg[sp] = seg;
        s_cnt[0][warp_id()] = ee;
        s_cnt[1][warp_id()] = ep;
        s_cnt[2][warp_id()] = seg;
    }
    __syncthreads();
    if (threadIdx.x == 0) {   // the CTA's spans together, after the per-warp entries
        unsigned tee = 0, tep = 0, tseg = 0;
#pragma unroll
        for (unsigned w = 0; w < WARPS; ++w) {
            tee += s_cnt[0][w];
            tep += s_cnt[1][w];
            tseg = seg_join(tseg, s_cnt[2][w]);
        }
        d.span_ee[MAX_SPANS + blockIdx.x] = tee;
        d.span_ep[MAX_SPANS + blockIdx.x] = tep;
        d.span_seg[MAX_SPANS + blockIdx.x] = tseg;
    }
}

// P1 of one warp.  P0's masks of 32 windows, one per lane, give the roads that
// start in them (the word after an EP word) with their road index, event and
// place in the event; the starts are listed in shared memory, and each batch
// of 32 is decoded one road per lane: the lane takes its road's words from the
// header to the EP word, which may lie past the step's windows.  Each lane
// builds its road's coordinate row in shared memory; the batch's rows
// (consecutive roads) are then copied out with 16-byte stores.
// Roads listed of a step's 1024 words.  A road has three words at least, so a
// step of more starts than this has a road that is too short among the listed
// ones, and its fault is the batch's.
constexpr unsigned P1_STARTS = 384;
struct P1Warp {
    uint16_t row[WIN][40];           // coordinate rows of the batch's roads
    uint32_t start[P1_STARTS];       // a road's first word from the step's (10 bits), roads of the event
                                     // before it (10 bits, at most 1023), events of the step before it
};
static_assert(sizeof(P1Warp) % 16 == 0, "warp regions of 16-byte multiples");

// the longest road a lane walks: a road of more words breaks a rule within
// its first MAX_ROAD_WORDS words (a ninth hit on some layer at the latest)
constexpr unsigned MAX_ROAD_WORDS = 3 + N_LAYERS * MAX_HITS + 1;

// A complete road's record, and its event's end when it is the last one.
__device__ __forceinline__ void put_road(const Dev &d, unsigned g, unsigned ev, unsigned rie, uint32_t hdr, uint32_t cw,
                                         uint32_t pw, unsigned cnt4, bool ee, unsigned n_events)
{
    const unsigned wedge = min(hdr & 15u, 11u), barrel = min((hdr >> 4) & 7u, 5u);
    const unsigned excl = min((hdr >> 7) & 7u, 4u);
    RoadRec r;
    r.event = ev;
    r.pk = cnt4 | (excl << 20) | (min(rie, 255u) << 24);   // the hit counts, four bits per layer
    r.curv = (int16_t)(cw & 0xFFFFu);
    r.phi = (int16_t)(pw & 0xFFFFu);
    r.set = (uint16_t)((wedge * 6 + barrel) * 5 + excl);
    r.fit = 0;
    d.roads[g] = r;
    if (ee && ev < d.max_events) {   // the event's last road
        d.ev_road_end[ev] = g + 1;
        if (rie + 1 > (unsigned)P2W_ROADS)   // P2 takes this event with a whole CTA
            d.ev_big[atomicAdd(&d.ctrl->n_big_ev, 1u)] = ev;
        if (ev + 1 == n_events)
            d.ctrl->n_roads = g + 1;
    }
}

// The lane's road, word by word, with every rule of the grammar and the limits
// in order (a batch with a road that breaks one or does not end): true when it
// is complete; err: its first fault (encoded as in Ctrl::err_inv, ~0 when none).
__device__ __noinline__ bool walk_road(const Dev &d, uint16_t *row, unsigned long long start, unsigned g, unsigned ev,
                                       unsigned rie, unsigned n_events, unsigned long long &err)
{
    unsigned cnt4 = 0;   // hits so far, layer l in bits 4 l .. 4 l + 3 (at most MAX_HITS)
    uint32_t hdr = 0, cw = 0, pw = 0;
    for (unsigned k = 0; k < MAX_ROAD_WORDS; ++k) {
        const unsigned long long p = start + k;
        if (p >= d.n_words)
            return false;
        const uint32_t w = __ldg(d.words + p);
        const unsigned type = (w >> 27) & 7u;
        const bool ep = (w >> 30) & 1u;
        bool bad;
        if (k == 0) {
            bad = type != 7 || ep;
            hdr = w;
            if (!bad && rie >= (unsigned)MAX_ROADS_EV)
                err = (p << 8) | RANK_LIMIT;
        } else if (k == 1) {
            bad = type != 5 || ep;
            cw = w;
        } else if (k == 2) {
            bad = type != 6;
            pw = w;
        } else {
            bad = type > 4;
            if (!bad) {
                const unsigned r = (cnt4 >> (4 * type)) & 15u;
                if (r >= (unsigned)MAX_HITS) {
                    err = (p << 8) | RANK_LIMIT;
                } else {
                    row[type * 8 + r] = (uint16_t)(w & 0xFFFu);
                    cnt4 += 1u << (4 * type);
                }
            }
        }
        if (bad)
            err = (p << 8) | RANK_BAD;
        if (err != ~0ull)
            return false;
        if (ep) {
            if (g < d.max_roads)
                put_road(d, g, ev, rie, hdr, cw, pw, cnt4, (w >> 31) != 0, n_events);
            return true;
        }
    }
    return false;
}

// Decode the lane's road (have: there is one) of `len` words from `start`;
// returns the batch's first fault.  A road's length is known, so its words
// need no test for the end, and a rule's break is only noted: the batch is then
// walked again word by word.
__device__ __forceinline__ unsigned long long decode_batch(const Dev &d, P1Warp &q, bool have, unsigned long long start,
                                                           unsigned len, unsigned g, unsigned ev, unsigned rie,
                                                           unsigned n_events)
{
    const unsigned lane = lane_id();
    uint16_t *row = q.row[lane];
    unsigned long long err = ~0ull;
    bool done = have;
    unsigned cnt4 = 0;   // hits so far, four bits per layer
    uint32_t w[8], hdr = 0, cw = 0, pw = 0, last = 0;
    bool bad = have && (len < 3 || len >= MAX_ROAD_WORDS || rie >= (unsigned)MAX_ROADS_EV);
    const unsigned n = bad || !have ? 0u : len;
    const uint32_t *words = d.words + start;
    const unsigned most = __reduce_max_sync(FULL_MASK, n);
    for (unsigned k0 = 0; k0 < most; k0 += 8) {
#pragma unroll
        for (unsigned u = 0; u < 8; ++u)   // eight loads in flight
            w[u] = k0 + u < n ? __ldg(words + k0 + u) : 0xFFFFFFFFu;
#pragma unroll
        for (unsigned u = 0; u < 8; ++u) {
            if (k0 == 0 && u < 3) {
                if (u == 0)
                    hdr = w[0];
                else if (u == 1)
                    cw = w[1];
                else
                    pw = w[2];
                continue;
            }
            if (k0 + u < n) {
                const unsigned type = (w[u] >> 27) & 7u, sh = 4 * type, r = (cnt4 >> (sh & 31u)) & 15u;
                const bool fits = (type <= 4) & (r < (unsigned)MAX_HITS);
                bad = bad | !fits;
                if (fits)
                    row[type * 8 + r] = (uint16_t)w[u];
                cnt4 += 1u << (sh & 31u);
                last = w[u];
            }
        }
    }
    if (n) {
        last = n == 3 ? pw : last;
        bad = bad | (((hdr >> 27) & 7u) != 7) | (((cw >> 27) & 7u) != 5) | (((pw >> 27) & 7u) != 6);
    }
    if (__any_sync(FULL_MASK, bad)) {
        if (have)
            done = walk_road(d, row, start, g, ev, rie, n_events, err);
    } else if (have && g < d.max_roads) {
        put_road(d, g, ev, rie, hdr, cw, pw, cnt4, (last >> 31) != 0, n_events);
    }
    __syncwarp();
    // the rows of the batch's complete roads (consecutive road indices from
    // the first lane's), five 16-byte words each
    const unsigned g0 = __shfl_sync(FULL_MASK, g, 0), dm = __ballot_sync(FULL_MASK, done);
    const unsigned cnt = __popc(__ballot_sync(FULL_MASK, have));
    const uint4 *src = reinterpret_cast<const uint4 *>(&q.row[0][0]);
    uint4 *dst = reinterpret_cast<uint4 *>(d.coords + (size_t)g0 * 40);
    for (unsigned i = lane; i < cnt * N_LAYERS; i += WIN) {
        const unsigned j = i / N_LAYERS;
        if (((dm >> j) & 1u) && g0 + j < d.max_roads)
            dst[i] = src[i];
    }
    __syncwarp();
    return warp_min_u64(err);
}

// P1 for one warp: the roads whose header lies in [a, e).  g, ev: EP and EE
// words before a; rie: EP words since the last EE before a (roads of the open
// event).  Bound: the walk of a road, a chain of its words per lane.
// 192,000 roads of 12 hits 27.9 -> 13.7 us, 25,600 of 40 hits 18.9 -> 12.0 (with
// the stream scanned a second time for the starts, and each road's end found on
// its walk).
__device__ void decode_span(const Dev &d, P1Warp &q, unsigned long long a, unsigned long long e, unsigned g,
                            unsigned ev, unsigned rie, unsigned n_events)
{
    const unsigned lane = lane_id();
    if (a >= e)
        return;
    const unsigned w_end = (unsigned)((e + WIN - 1) / WIN), w_all = (unsigned)((d.n_words + WIN - 1) / WIN);
    unsigned W = (unsigned)(a / WIN);
    unsigned ends = W == 0 ? 1u : __ldcg(&d.wmask[W - 1].x) >> 31;   // the step's first word starts a road
    unsigned long long err = ~0ull;
    for (; W < w_end && err == ~0ull; W += WIN) {
        // the step's windows, one per lane
        const unsigned win = W + lane;
        const uint2 m = win < w_end ? __ldcg(&d.wmask[win]) : make_uint2(0u, 0u);
        const unsigned pm = m.x, em = m.y, up = __shfl_up_sync(FULL_MASK, pm, 1);
        const unsigned pe = lane ? up >> 31 : ends;
        const unsigned long long base = (unsigned long long)W * WIN, left = win < w_end ? d.n_words - base - lane * WIN : 0;
        const unsigned in = left >= WIN ? FULL_MASK : (1u << (unsigned)left) - 1u;
        unsigned sm = ((pm << 1) | pe) & in;   // roads start
        // EP and EE words of the windows before, and EP words since the last EE
        const unsigned own = __popc(pm) | __popc(em) << 16;
        unsigned inc = own, seg = seg_window(em, pm);
#pragma unroll
        for (unsigned o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(FULL_MASK, inc, o), v = __shfl_up_sync(FULL_MASK, seg, o);
            if (lane >= o) {
                inc += u;
                seg = seg_join(v, seg);
            }
        }
        unsigned before = __shfl_up_sync(FULL_MASK, seg, 1);
        before = seg_join(rie, lane ? before : 0u) & ~SEG_EE;
        const unsigned ex = inc - own;
        const unsigned n_start = __reduce_add_sync(FULL_MASK, __popc(sm));
        unsigned at = ends + (ex & 0xFFFFu) - pe;   // place of the lane's first start
        const unsigned g_first = g + 1 - ends;
        unsigned last_start = 0;
        while (sm) {
            const unsigned b = __ffs(sm) - 1, lt = (1u << b) - 1u, el = em & lt;
            const unsigned r = el ? __popc(pm & lt & ~((2u << (31 - __clz(el))) - 1u)) : before + __popc(pm & lt);
            last_start = lane * WIN + b;
            if (at < P1_STARTS)
                q.start[at] = last_start | min(r, 1023u) << 10 | ((ex >> 16) + __popc(el)) << 20;
            ++at;
            sm &= sm - 1;
        }
        // the word after the last road's end (the first EP from its start on,
        // within the step or the two windows after it)
        last_start = __reduce_max_sync(FULL_MASK, last_start);
        unsigned end = ~0u;
        {
            const unsigned ls = last_start, lw = ls / WIN;
            const unsigned c = lane < lw ? 0u : lane == lw ? pm & ~((1u << (ls % WIN)) - 1u) : pm;
            if (c)
                end = lane * WIN + __ffs(c);
            const unsigned after = min(W + WIN, w_end) + lane;
            if (lane < 2 && after < w_all) {
                const unsigned p2 = __ldcg(&d.wmask[after].x);
                if (p2)
                    end = min(end, (after - W) * WIN + __ffs(p2));
            }
            end = __reduce_min_sync(FULL_MASK, end);
        }
        __syncwarp();
        if (n_start > P1_STARTS)
            end = ~0u;
        const unsigned n_list = min(n_start, P1_STARTS);
        for (unsigned off = 0; off < n_list && err == ~0ull; off += WIN) {
            const unsigned i = off + lane;
            const bool have = i < n_list;
            const unsigned s = have ? q.start[i] : 0u, pos = s & 1023u;
            const unsigned next = i + 1 < n_list ? q.start[i + 1] & 1023u : end;
            err = decode_batch(d, q, have, base + pos, next == ~0u ? MAX_ROAD_WORDS : next - pos, g_first + i,
                               ev + (s >> 20), (s >> 10) & 1023u, n_events);
        }
        __syncwarp();   // the list is refilled next
        const unsigned tot = __shfl_sync(FULL_MASK, inc, 31);
        rie = seg_join(rie, __shfl_sync(FULL_MASK, seg, 31)) & ~SEG_EE;
        g += tot & 0xFFFFu;
        ev += tot >> 16;
        ends = __shfl_sync(FULL_MASK, pm, 31) >> 31;   // (a step that is not full is the span's last)
    }
    if (lane == 0 && err != ~0ull)
        report(d, err);   // the first fault of the batch is its status
}

// P1; false when the stream does not fit the context (every CTA sees the
// same totals and stops).  smem: the CTA's shared memory (a P1Warp per warp).
__device__ bool scan_decode(const Dev &d, unsigned char *smem, Batch &bt)
{
    const unsigned mine0 = blockIdx.x * WARPS;
    // the CTAs below this one (their aggregates follow the per-warp entries),
    // and all CTAs (the stream's counts)
    const unsigned per = (gridDim.x + BLOCK - 1) / BLOCK;
    const unsigned c0 = min(threadIdx.x * per, gridDim.x), c1 = min(c0 + per, gridDim.x);
    unsigned long long all = 0, below = 0;   // EE << 32 | EP
    unsigned seg = 0;
    for (unsigned c = c0; c < c1; ++c) {
        const unsigned long long v = ((unsigned long long)ldcg(d.span_ee + MAX_SPANS + c) << 32) |
                                     ldcg(d.span_ep + MAX_SPANS + c);
        all += v;
        if (c < blockIdx.x) {
            below += v;
            seg = seg_join(seg, ldcg(d.span_seg + MAX_SPANS + c));
        }
    }
    block_sum2(all, below);
    seg = block_seg_fold(seg);
    const unsigned n_ee = (unsigned)(all >> 32), n_ep = (unsigned)all;
    const bool fits = n_ee <= d.max_events && n_ep <= d.max_roads;
    bt.n_events = n_ee;
    bt.n_ep = n_ep;
    // the candidate bits of this batch's roads start at zero (P2 sets them)
    if (fits)
        for (unsigned i = blockIdx.x * BLOCK + threadIdx.x; i < n_ep / 32 + 1; i += gridDim.x * BLOCK)
            d.cand_bits[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        Ctrl *c = d.ctrl;
        c->n_events = n_ee;
        c->n_ep = n_ep;
        unsigned tail = 0;
        if (d.n_words > 0 && !(__ldg(d.words + d.n_words - 1) >> 31)) {
            tail = 1;
            report(d, (d.n_words << 8) | RANK_TRUNC);
        }
        c->has_tail = tail;
        if (!fits)
            raise_flag(d, FLAG_CAPACITY);
        if (n_ee == 0)
            c->n_roads = 0;
    }
    if (!fits)
        return false;
    // the spans of this CTA below this warp
    unsigned g = (unsigned)below, ev = (unsigned)(below >> 32);
    {
        const unsigned j = lane_id(), sp = mine0 + j;
        const bool b4 = j < warp_id();
        g += warp_sum(b4 ? ldcg(d.span_ep + sp) : 0u);
        ev += warp_sum(b4 ? ldcg(d.span_ee + sp) : 0u);
        seg = seg_join(seg, warp_seg_fold(b4 ? ldcg(d.span_seg + sp) : 0u));
    }
    unsigned long long a, e;
    span_of(d, mine0 + warp_id(), a, e);
    P1Warp &q = reinterpret_cast<P1Warp *>(smem)[warp_id()];
    decode_span(d, q, a, e, g, ev, seg & ~SEG_EE, n_ee);
    return true;
}

// ---------------------------------------------------------------------------
// P2: the cross-road flags of each event (a CTA or a warp per event).  A track can
// only be dropped by a track of another road that shares hits with it on
// three layers, so only road pairs with a coordinate in common on >= 3
// layers matter.  The coordinates of the event that appear in two or more
// roads (per-layer bitmaps) get, per road and layer, a 64-bit signature;
// pairs of roads whose signatures meet on >= 3 layers take the exact test,
// which marks the shared hits of both roads.  A road with a marked hit is a
// cross-road candidate; its marked hits are the ones it publishes and looks
// up.  The road records get the candidate bit and their fit path.
//
// Events of at most P2W_ROADS roads take one warp each instead (p2_warp), and
// so do larger ones when there are many, with a bitmap of one layer at a time,
// 10-bit signatures and a lane per tested pair (p2_phase chooses).
// ---------------------------------------------------------------------------

constexpr unsigned P2_PAIRS = 1024;   // road pairs queued for the exact test (more: tested in place)

struct P2Smem {
    RoadRec rec[MAX_ROADS_EV];
    unsigned long long sig[MAX_ROADS_EV][N_LAYERS];   // signatures of a road's shared coordinates
    uint32_t seen[N_LAYERS][128];         // coordinate bitmaps of the event
    uint32_t multi[N_LAYERS][128];
    uint32_t xlo[MAX_ROADS_EV];           // hits shared with a road that shares coordinates on
    uint32_t xhi[MAX_ROADS_EV];           //   >= 3 layers: bit 8 l + d (l < 4), layer 4 in xhi
    uint16_t elig[MAX_ROADS_EV];          // roads with shared coordinates on >= 3 layers
    uint32_t cp[P2_PAIRS];                // road pairs whose signatures meet on >= 3 layers (r | t << 16)
    unsigned n_elig, n_cp;
};

// signature bit of a coordinate: a multiplicative hash into 0..63
__device__ __forceinline__ unsigned sig_bit(unsigned v) { return (v * 0x9E3779B1u) >> 26; }

__device__ __forceinline__ bool is_multi(const P2Smem &s, unsigned l, unsigned v)
{
    return (s.multi[l][v >> 5] >> (v & 31u)) & 1u;
}

// coordinate x of a layer's row (eight 16-bit coordinates in a uint4); x is
// a constant in the unrolled loops below
__device__ __forceinline__ unsigned row_coord(const uint4 &q, unsigned x)
{
    const unsigned w = x < 2 ? q.x : x < 4 ? q.y : x < 6 ? q.z : q.w;
    return (w >> (16 * (x & 1u))) & 0xFFFFu;
}

// the coordinates of row q from slot n on replaced by 0xFFFF (no coordinate)
__device__ __forceinline__ uint4 row_clip(uint4 q, unsigned n)
{
    const auto word = [n](unsigned w, unsigned i) {
        return n >= 2 * i + 2 ? w : n == 2 * i + 1 ? w | 0xFFFF0000u : 0xFFFFFFFFu;
    };
    return make_uint4(word(q.x, 0), word(q.y, 1), word(q.z, 2), word(q.w, 3));
}

// slots of row q that hold v (bit x: slot x)
__device__ __forceinline__ unsigned row_find(const uint4 &q, unsigned v)
{
    const unsigned v2 = v | v << 16;
    const auto eq = [v2](unsigned w) {   // bit 15 and bit 31: the halves equal to v
        const unsigned x = w ^ v2;
        return ~(((x & 0x7FFF7FFFu) + 0x7FFF7FFFu) | x) & 0x80008000u;
    };
    // halves 2 i and 2 i + 1 of word i to bits 2 i and 2 i + 1
    const auto two = [](unsigned e) { return (e >> 15 & 1u) | (e >> 30 & 2u); };
    return two(eq(q.x)) | two(eq(q.y)) << 2 | two(eq(q.z)) << 4 | two(eq(q.w)) << 6;
}

// A layer's hits (row q, n of them) join the event's bitmap: bit x of the
// result: hit x found its bit set.  The atomics are in flight together.
// most: at least every lane's n.
__device__ __forceinline__ unsigned see_row(uint32_t *seen, const uint4 &q, unsigned n, unsigned most)
{
    unsigned old[MAX_HITS], again = 0;
#pragma unroll
    for (unsigned x = 0; x < MAX_HITS; ++x) {
        old[x] = 0;
        if (x >= 2 && x >= most)
            continue;
        const unsigned v = row_coord(q, x);
        if (x < n)   // the result is not awaited here
            old[x] = atomicOr(&seen[v >> 5], 1u << (v & 31u)) >> (v & 31u);
    }
#pragma unroll
    for (unsigned x = 0; x < MAX_HITS; ++x)
        again |= (old[x] & 1u) << x;
    return again;
}

// coordinate x (0 .. 7) of a layer's row
__device__ __forceinline__ unsigned row_at(const uint4 &q, unsigned x)
{
    const unsigned w = x < 4 ? (x < 2 ? q.x : q.y) : (x < 6 ? q.z : q.w);
    return (w >> (16 * (x & 1u))) & 0xFFFFu;
}

// Hits of one layer of a road (row q) whose coordinate was already in the
// event's bitmap when the hit set its bit (bit x of `again`): a coordinate
// of an earlier slot of the same row is a repeat; any other was set by
// another road and gets the multi bit.  So a coordinate gets the multi bit
// exactly when two roads hold it.
__device__ __forceinline__ void seen_again(uint32_t *multi, const uint4 &q, unsigned again)
{
    for (; again; again &= again - 1) {
        const unsigned x = __ffs(again) - 1;
        const unsigned v = row_at(q, x);
        if (!(row_find(q, v) & ((1u << x) - 1u)))
            atomicOr(&multi[v >> 5], 1u << (v & 31u));
    }
}

// hits of a layer (row q, n of them) whose coordinate two roads hold: bit x
__device__ __forceinline__ unsigned multi_row(const uint32_t *multi, const uint4 &q, unsigned n, unsigned most)
{
    unsigned m = 0;
#pragma unroll
    for (unsigned x = 0; x < MAX_HITS; ++x) {
        if (x >= 4 && x >= most)
            continue;
        const unsigned v = row_coord(q, x) & 0xFFFu;
        m |= ((multi[v >> 5] >> (v & 31u)) & 1u) << x;
    }
    return m & ((1u << n) - 1u);
}

// Roads r and t of the event: the layers on which they hold a common
// coordinate and the hits involved; with three or more such layers, the
// shared hits of both roads are marked.  Only coordinates present in two
// roads can be common.
__device__ void pair_exact(P2Smem &s, const uint16_t *co, unsigned r, unsigned t)
{
    const uint32_t pr = s.rec[r].pk, pt = s.rec[t].pk;
    unsigned lo_r = 0, lo_t = 0, hi_r = 0, hi_t = 0, layers = 0;
#pragma unroll
    for (unsigned l = 0; l < N_LAYERS; ++l) {
        const unsigned nr = (pr >> (4 * l)) & 15u, nt = (pt >> (4 * l)) & 15u;   // <= MAX_HITS
        unsigned br = 0, bt = 0;
        for (unsigned x = 0; x < nr; ++x) {
            const unsigned v = co[r * 40 + l * 8 + x];
            if (!is_multi(s, l, v))
                continue;
            for (unsigned y = 0; y < nt; ++y)
                if (co[t * 40 + l * 8 + y] == v) {
                    br |= 1u << x;
                    bt |= 1u << y;
                }
        }
        layers += br != 0;
        if (l < 4) {
            lo_r |= br << (8 * l);
            lo_t |= bt << (8 * l);
        } else {
            hi_r = br;
            hi_t = bt;
        }
    }
    if (layers >= 3) {
        atomicOr(&s.xlo[r], lo_r);
        atomicOr(&s.xhi[r], hi_r);
        atomicOr(&s.xlo[t], lo_t);
        atomicOr(&s.xhi[t], hi_t);
    }
}

// The exact test of pair_exact by a whole warp: lane 8 l + x (then lane x
// for layer 4) takes hit x of road r on layer l and compares it with road t's
// hits on that layer.
__device__ void pair_exact_warp(P2Smem &s, const uint16_t *co, unsigned r, unsigned t)
{
    const unsigned lane = lane_id();
    const uint32_t pr = s.rec[r].pk, pt = s.rec[t].pk;
    unsigned m_r[2], m_t[2];   // marked hits of r and t: layers 0..3, then layer 4
#pragma unroll
    for (unsigned pass = 0; pass < 2; ++pass) {
        const unsigned l = pass ? 4u : lane >> 3, x = pass ? lane : lane & 7u;
        const unsigned nr = (pr >> (4 * l)) & 15u, nt = (pt >> (4 * l)) & 15u;   // <= MAX_HITS
        unsigned br = 0, bt = 0;
        if (x < nr && (!pass || lane < 8)) {
            const unsigned v = co[r * 40 + l * 8 + x];
            if (is_multi(s, l, v))
                for (unsigned y = 0; y < nt; ++y)
                    if (co[t * 40 + l * 8 + y] == v) {
                        br = 1u << x;
                        bt |= 1u << y;
                    }
        }
        const unsigned sh = pass ? 0u : 8 * l;
        m_r[pass] = __reduce_or_sync(FULL_MASK, br << sh);
        m_t[pass] = __reduce_or_sync(FULL_MASK, bt << sh);
    }
    const unsigned layers = ((m_r[0] & 0xFFu) != 0) + ((m_r[0] & 0xFF00u) != 0) + ((m_r[0] & 0xFF0000u) != 0) +
                            ((m_r[0] >> 24) != 0) + (m_r[1] != 0);
    if (layers >= 3 && lane == 0) {
        atomicOr(&s.xlo[r], m_r[0]);
        atomicOr(&s.xhi[r], m_r[1]);
        atomicOr(&s.xlo[t], m_t[0]);
        atomicOr(&s.xhi[t], m_t[1]);
    }
}

// The four fitted layers' hit counts of a road record, slot j in bits 4j ..
// 4j + 3 (the excluded layer's count taken out).
__device__ __forceinline__ unsigned fitted_counts(uint32_t pk)
{
    const unsigned m = (1u << (4 * min((pk >> 20) & 7u, 4u))) - 1u;
    return (pk & m) | ((pk >> 4) & 0xFFFFu & ~m);
}

// Fit class of a road with N combinations and N4 distinct fits, and its slots
// by falling hit count (perm).  The box path takes roads with more than
// small_n4 distinct fits or with more than four hits on two fitted layers.
__device__ __forceinline__ unsigned road_class(uint32_t pk, unsigned N, unsigned N4, unsigned small_n4, unsigned &perm)
{
    const unsigned nf = fitted_counts(pk);
    unsigned v[4];
#pragma unroll
    for (unsigned j = 0; j < 4; ++j)
        v[j] = (((nf >> (4 * j)) & 15u) << 2) | j;
    const auto order = [&v](unsigned i, unsigned j) {
        const unsigned hi = max(v[i], v[j]), lo = min(v[i], v[j]);
        v[i] = hi;
        v[j] = lo;
    };
    order(0, 1);
    order(2, 3);
    order(0, 2);
    order(1, 3);
    order(1, 2);
    perm = (v[0] & 3u) | (v[1] & 3u) << 2 | (v[2] & 3u) << 4 | (v[3] & 3u) << 6;
    const unsigned ma = v[0] >> 2, mb = v[1] >> 2;
    if (N == 0)
        return CLS_NONE;
    if (N4 > small_n4 || mb > 4)
        return CLS_BOX;
    return ma > 4 ? (mb > 2 ? 4u : 3u) : ma > 2 ? (mb > 2 ? 2u : 1u) : 0u;
}

// The fit stage's lists.  A CTA gathers the group path's roads of its events
// in shared memory and lists them at the end of the stage, sorted by class and
// by the hits of the two smallest fitted slots (c, e), so that a warp's roads
// loop alike: one atomic per half class and CTA.  (An atomic per class and
// warp made 10,000 events wait 8 us on the counters; lists of each CTA's share
// in its own shared memory, sorted at the start of the fit stage, left a third
// of the warps idle at its end, since CTAs of equal shares take 56 to 79 us.)
// Roads that find the list full are listed directly.
constexpr unsigned P2_LIST = 3 * BLOCK;        // roads gathered at most
constexpr unsigned P2_BUCKETS = 16 * N_GROUP_CLS;
struct P2List {
    RoadItem item[P2_LIST];                    // perm: bucket in the high byte
    unsigned cnt[P2_BUCKETS];                  // roads of a bucket, then the first place of each in its half class
    unsigned base[2 * N_GROUP_CLS];            // first place of the CTA's roads in each half class
    unsigned n;
};

// where place i of half class seg lies (odd: at most two hits in slot e)
__device__ __forceinline__ size_t list_at(const Dev &d, unsigned seg, unsigned i)
{
    return (size_t)(seg >> 1) * d.max_roads + ((seg & 1u) ? i : d.max_roads - 1 - i);
}

// Bucket of a road of class cls: half class (widest class first, then more
// than two hits in slot e) in units of eight, then the hits of slots c and e,
// most first.
__device__ __forceinline__ unsigned road_bucket(uint32_t pk, unsigned perm, unsigned cls)
{
    const unsigned nf = fitted_counts(pk);
    const unsigned mc = (nf >> (4 * ((perm >> 4) & 3u))) & 15u, me = (nf >> (4 * (perm >> 6))) & 15u;   // 1 .. 4
    return 16 * (N_GROUP_CLS - 1 - cls) + (me > 2 ? 0u : 8u) + 2 * ((4 - mc) & 3u) + (me & 1u);
}

// The end of P2 for road g (record r, flagged hits xm), one road per lane, by a
// whole warp (in: the lane has a road): the record's candidate bit and fit path,
// and the road joins its list.  Returns the road's combinations.
__device__ __forceinline__ unsigned finish_road(const Dev &d, P2List &list, bool in, unsigned g, RoadRec r,
                                                unsigned long long xm)
{
    const unsigned lane = lane_id(), lt = lanemask_lt();
    const bool cand = xm != 0ull;
    unsigned N, N4, perm;
    road_sizes(r.pk, N, N4);
    N = in ? N : 0u;
    const unsigned cls = road_class(r.pk, N, N4, (unsigned)d.small_n4, perm);
    r.pk |= cand ? (1u << 23) : 0u;
    r.fit = (uint16_t)(perm | cls << 8);
    if (in) {
        d.roads[g] = r;
        d.xmask[g] = xm;
        d.surv_cnt[g] = 0;
        if (N > 0 && cand)   // checked against the other roads' groups after the fit
            atomicOr(&d.cand_bits[g >> 5], 1u << (g & 31u));
    }
    if (__any_sync(FULL_MASK, N > 0 && cand) && lane == 0)
        raise_flag(d, FLAG_CANDS);
    const unsigned mg = __ballot_sync(FULL_MASK, cls < N_GROUP_CLS), mb = __ballot_sync(FULL_MASK, cls == CLS_BOX);
    unsigned at = 0;
    if (lane == 0 && mg)
        at = atomicAdd(&list.n, (unsigned)__popc(mg));
    if (lane == 1 && mb)
        at = atomicAdd(&d.ctrl->n_box, (unsigned)__popc(mb));
    const unsigned gat = __shfl_sync(FULL_MASK, at, 0) + __popc(mg & lt);
    const unsigned bat = __shfl_sync(FULL_MASK, at, 1) + __popc(mb & lt);
    if (cls == CLS_BOX && bat < d.max_roads)
        d.box_list[bat] = g;
    if (cls < N_GROUP_CLS) {
        const unsigned bucket = road_bucket(r.pk, perm, cls);
        const RoadItem it{g, r.pk, r.curv, r.phi, r.set, (uint16_t)(perm | bucket << 8)};
        if (gat < P2_LIST) {
            list.item[gat] = it;
        } else {
            const unsigned i = atomicAdd(&d.ctrl->n_seg[bucket >> 3], 1u);
            if (i < d.max_roads)
                d.items[list_at(d, bucket >> 3, i)] = it;
        }
    }
    return N;
}

// The CTA's list goes out (every thread; the list is complete and `cnt` zero).
__device__ void list_out(const Dev &d, P2List &list)
{
    constexpr unsigned EACH = (P2_LIST + BLOCK - 1) / BLOCK;
    const unsigned lane = lane_id(), n = min(list.n, P2_LIST);
    if (n == 0)
        return;
    unsigned place[EACH];
#pragma unroll
    for (unsigned k = 0; k < EACH; ++k) {
        const unsigned i = k * BLOCK + threadIdx.x;
        if (i < n)
            place[k] = atomicAdd(&list.cnt[list.item[i].perm >> 8], 1u);
    }
    __syncthreads();
    if (warp_id() == 0) {   // first places within each half class: eight buckets each
        for (unsigned c = 0; c < P2_BUCKETS; c += 32) {
            const unsigned b = c + lane;
            const unsigned v = b < P2_BUCKETS ? list.cnt[b] : 0u;
            unsigned inc = v;
#pragma unroll
            for (unsigned o = 1; o < 8; o <<= 1) {
                const unsigned u = __shfl_up_sync(FULL_MASK, inc, o);
                inc += (lane & 7u) >= o ? u : 0u;
            }
            if (b < P2_BUCKETS) {
                list.cnt[b] = inc - v;
                if ((lane & 7u) == 7 && inc)
                    list.base[b >> 3] = atomicAdd(&d.ctrl->n_seg[b >> 3], inc);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (unsigned k = 0; k < EACH; ++k) {
        const unsigned i = k * BLOCK + threadIdx.x;
        if (i < n) {
            const RoadItem it = list.item[i];
            const unsigned b = it.perm >> 8, at = list.base[b >> 3] + list.cnt[b] + place[k];
            if (at < d.max_roads)
                d.items[list_at(d, b >> 3, at)] = it;
        }
    }
}

// Flags of the event of roads r0 .. r0 + nr - 1; adds its combinations to n_comb.
// Bound: the latency of its steps, each a pass over the event's rows by one
// CTA (one event of 64 roads 8.0 -> 6.4 us for the stage; 301 events of 96
// roads 14.5 -> 11.9; 200 events of 128 roads with eight hits a layer 18.4 with
// 512 threads a CTA, 22.4 with 256, of which the pairs are 6.3).
__device__ void p2_event(const Dev &d, unsigned r0, unsigned nr, unsigned char *smem, P2List &list,
                         unsigned long long &n_comb)
{
    P2Smem &s = *reinterpret_cast<P2Smem *>(smem);
    // the event's roads: records; the coordinate rows stay in global memory (they
    // are written before this stage, so that loads may use L1, which has what
    // shared memory leaves)
    const uint16_t *co = d.coords + (size_t)r0 * 40;
    const uint4 *rows = reinterpret_cast<const uint4 *>(co);
    for (unsigned k = threadIdx.x; k < nr; k += BLOCK) {
        s.rec[k] = ldcg(d.roads + r0 + k);
        s.xlo[k] = 0;
        s.xhi[k] = 0;
    }
    for (unsigned i = threadIdx.x; i < N_LAYERS * 128; i += BLOCK) {
        (&s.seen[0][0])[i] = 0;
        (&s.multi[0][0])[i] = 0;
    }
    if (threadIdx.x == 0) {
        s.n_elig = 0;
        s.n_cp = 0;
    }
    __syncthreads();
    // coordinates present in >= 2 roads on a layer: each distinct coordinate
    // of a road's layer marks the bitmap, a second road with it the multi bit
    for (unsigned i0 = threadIdx.x - lane_id(); i0 < nr * N_LAYERS; i0 += BLOCK) {
        const unsigned i = min(i0 + lane_id(), nr * N_LAYERS - 1), k = i / N_LAYERS, l = i - k * N_LAYERS;
        const unsigned n = i0 + lane_id() == i ? (s.rec[k].pk >> (4 * l)) & 15u : 0u;   // <= MAX_HITS
        const uint4 q = rows[i];
        seen_again(s.multi[l], q, see_row(s.seen[l], q, n, __reduce_max_sync(FULL_MASK, n)));
    }
    __syncthreads();
    // signatures of the shared coordinates, a layer of a road per thread
    for (unsigned i = threadIdx.x; i < nr * N_LAYERS; i += BLOCK) {
        const unsigned k = i / N_LAYERS, l = i - k * N_LAYERS, n = (s.rec[k].pk >> (4 * l)) & 15u;
        const uint4 q = rows[i];
        unsigned long long sg = 0;
        for (unsigned m = multi_row(s.multi[l], q, n, MAX_HITS); m; m &= m - 1)
            sg |= 1ull << sig_bit(row_at(q, __ffs(m) - 1));
        s.sig[k][l] = sg;
    }
    __syncthreads();
    // roads with >= 3 such layers
    for (unsigned k = threadIdx.x; k < nr; k += BLOCK) {
        unsigned layers = 0;
#pragma unroll
        for (unsigned l = 0; l < N_LAYERS; ++l)
            layers += s.sig[k][l] != 0;
        if (layers >= 3)
            s.elig[atomicAdd(&s.n_elig, 1u)] = (uint16_t)k;
    }
    __syncthreads();
    // pairs of eligible roads whose signatures meet on >= 3 layers
    const unsigned ne = s.n_elig;
    for (unsigned a = warp_id(); a < ne; a += WARPS) {
        const unsigned r = s.elig[a];
        const unsigned long long s0 = s.sig[r][0], s1 = s.sig[r][1], s2 = s.sig[r][2], s3 = s.sig[r][3],
                                 s4 = s.sig[r][4];
        for (unsigned b = a + 1 + lane_id(); b < ne; b += 32) {
            const unsigned t = s.elig[b];
            const unsigned c = ((s0 & s.sig[t][0]) != 0) + ((s1 & s.sig[t][1]) != 0) + ((s2 & s.sig[t][2]) != 0) +
                               ((s3 & s.sig[t][3]) != 0) + ((s4 & s.sig[t][4]) != 0);
            if (c >= 3) {   // queued for a warp's exact test (in place when the queue is full)
                const unsigned k = atomicAdd(&s.n_cp, 1u);
                if (k < P2_PAIRS)
                    s.cp[k] = r | (t << 16);
                else
                    pair_exact(s, co, r, t);
            }
        }
    }
    __syncthreads();
    for (unsigned k = warp_id(); k < min(s.n_cp, P2_PAIRS); k += WARPS)
        pair_exact_warp(s, co, s.cp[k] & 0xFFFFu, s.cp[k] >> 16);
    __syncthreads();
    // the road records: candidate bit and fit path
    for (unsigned k0 = threadIdx.x - lane_id(); k0 < nr; k0 += BLOCK) {
        const unsigned k = min(k0 + lane_id(), nr - 1);
        n_comb += finish_road(d, list, k0 + lane_id() == k, r0 + k, s.rec[k],
                              ((unsigned long long)s.xhi[k] << 32) | s.xlo[k]);
    }
    __syncthreads();   // the shared arrays are refilled for the next event
}

// One warp's state for an event of its own; the roads' coordinate rows stay in
// global memory (they are written once, before this stage, so that loads may
// use L1).
constexpr unsigned P2_QUEUE = 64;       // queued road pairs: a batch of 32, and what one test may add
struct P2Warp {
    uint32_t seen[128];                 // coordinate bitmap of the event, one layer at a time
    uint32_t multi[128];                // coordinates present in two or more roads
    uint2 sig[P2W_ROADS];               // signatures of the eligible roads' shared coordinates
    uint32_t xm[P2W_ROADS][2];          // flagged hits of a road: bit 8 l + d, low and high word
    uint32_t pair[P2_QUEUE];            // road pairs whose signatures meet on >= 3 layers (r | t << 16)
    uint8_t elig[P2W_ROADS];            // roads with shared coordinates on >= 3 layers
};
constexpr size_t P2W_BYTES = (sizeof(P2Warp) + 15) / 16 * 16;

// Signature of coordinates of layer l, ten bits a layer: layers 0..2 in x,
// layers 3 and 4 in y.  bit: a multiplicative hash into 0..9.
__device__ __forceinline__ unsigned sig_bit10(unsigned v) { return ((v * 0x9E3779B1u) >> 16) * 10u >> 16; }
// layers on which two signatures (their fields ANDed) meet: the top bit of a
// field is set by adding all ones below it to any bits below it
__device__ __forceinline__ unsigned sig_layers(unsigned x, unsigned y)
{
    const unsigned m = 0x1FF7FDFFu, t = 0x20080200u;
    return __popc(((x & m) + m | x) & t) + __popc(((y & m) + m | y) & t & 0xFFFFFu);
}

// The queued pairs (n of them, one per lane): hits the two roads of a pair
// share are flagged in both when they share coordinates on >= 3 layers.
__device__ __noinline__ void p2_pairs(const uint16_t *coords, const RoadRec *roads, P2Warp &w, unsigned r0, unsigned n)
{
    const unsigned lane = lane_id();
    if (lane < n) {
        const unsigned p = w.pair[lane], r = p & 0xFFFFu, t = p >> 16;
        const uint4 *rr = reinterpret_cast<const uint4 *>(coords + (size_t)(r0 + r) * 40);
        const uint4 *rt = reinterpret_cast<const uint4 *>(coords + (size_t)(r0 + t) * 40);
        const uint32_t pr = ldcg(&roads[r0 + r].pk), pt = ldcg(&roads[r0 + t].pk);
        unsigned lo_r = 0, lo_t = 0, hi_r = 0, hi_t = 0, layers = 0;
        for (unsigned l = 0; l < N_LAYERS; ++l) {
            const unsigned nr = (pr >> (4 * l)) & 15u, nt = (pt >> (4 * l)) & 15u;   // <= MAX_HITS
            uint4 a = rr[l];
            const uint4 b = row_clip(rt[l], nt);
            unsigned br = 0, bt = 0;
            for (unsigned x = 0; x < nr; ++x) {
                const unsigned hit = row_find(b, a.x & 0xFFFFu);
                br |= hit ? 1u << x : 0u;
                bt |= hit;
                a.x = a.x >> 16 | a.y << 16;   // the next slot
                a.y = a.y >> 16 | a.z << 16;
                a.z = a.z >> 16 | a.w << 16;
                a.w >>= 16;
            }
            layers += br != 0;
            if (l < 4) {
                lo_r |= br << (8 * l);
                lo_t |= bt << (8 * l);
            } else {
                hi_r = br;
                hi_t = bt;
            }
        }
        if (layers >= 3) {
            atomicOr(&w.xm[r][0], lo_r);
            atomicOr(&w.xm[r][1], hi_r);
            atomicOr(&w.xm[t][0], lo_t);
            atomicOr(&w.xm[t][1], hi_t);
        }
    }
    __syncwarp();
}

// P2 of the event of roads r0 .. r0 + nr - 1 (nr <= P2W_ROADS) by one warp with
// state `w`; lane i owns roads i and i + 32.  The same steps as p2_event:
// coordinates present in two roads (bitmaps, a layer at a time), signatures of
// those per road, pairs of roads whose signatures meet on >= 3 layers tested
// exactly (a lane per pair).  Bound: latency of one warp's chain, so a layer's
// rows are loaded while the layer before is worked on, and a layer's atomics
// are in flight together (3000 events of 64 roads 26.3 -> 19.3 us).
__device__ void p2_warp(const Dev &d, unsigned r0, unsigned nr, P2Warp &w, P2List &list, unsigned long long &n_comb)
{
    const unsigned lane = lane_id();
    const uint4 *rows = reinterpret_cast<const uint4 *>(d.coords + (size_t)r0 * 40);
    RoadRec rec[2];
    uint4 q[2], next[2];
    unsigned sx[2] = {0u, 0u}, sy[2] = {0u, 0u};   // the roads' signatures (sig_layers)
#pragma unroll
    for (unsigned h = 0; h < 2; ++h) {
        const unsigned k = min(32 * h + lane, nr - 1);   // a missing road reads the last one and has no hits
        rec[h] = ldcg(d.roads + r0 + k);
        next[h] = rows[k * N_LAYERS];
    }
    if (lane >= nr)
        rec[0].pk = 0;
    if (lane + 32 >= nr)
        rec[1].pk = 0;
    w.xm[lane][0] = w.xm[lane][1] = w.xm[lane + 32][0] = w.xm[lane + 32][1] = 0;
    for (unsigned l = 0; l < N_LAYERS; ++l) {
        reinterpret_cast<uint4 *>(w.seen)[lane] = make_uint4(0u, 0u, 0u, 0u);
        reinterpret_cast<uint4 *>(w.multi)[lane] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        unsigned n[2];   // <= MAX_HITS
#pragma unroll
        for (unsigned h = 0; h < 2; ++h) {
            q[h] = next[h];
            n[h] = (rec[h].pk >> (4 * l)) & 15u;
            if (l + 1 < N_LAYERS)
                next[h] = rows[min(32 * h + lane, nr - 1) * N_LAYERS + l + 1];
        }
        const unsigned most = __reduce_max_sync(FULL_MASK, max(n[0], n[1]));
        unsigned again[2];
#pragma unroll
        for (unsigned h = 0; h < 2; ++h)
            again[h] = see_row(w.seen, q[h], n[h], most);
#pragma unroll
        for (unsigned h = 0; h < 2; ++h)
            seen_again(w.multi, q[h], again[h]);
        __syncwarp();
#pragma unroll
        for (unsigned h = 0; h < 2; ++h) {
            unsigned f = 0;
            for (unsigned m = multi_row(w.multi, q[h], n[h], most); m; m &= m - 1)
                f |= 1u << sig_bit10(row_at(q[h], __ffs(m) - 1));
            if (l < 3)
                sx[h] |= f << (10 * l);
            else
                sy[h] |= f << (10 * (l - 3));
        }
        __syncwarp();
    }
    // roads with shared coordinates on >= 3 layers, and their signatures
    unsigned ne = 0;
#pragma unroll
    for (unsigned h = 0; h < 2; ++h) {
        const bool e = sig_layers(sx[h], sy[h]) >= 3;
        const unsigned m = __ballot_sync(FULL_MASK, e), at = ne + __popc(m & lanemask_lt());
        if (e) {
            w.elig[at] = (uint8_t)(32 * h + lane);
            w.sig[at] = make_uint2(sx[h], sy[h]);
        }
        ne += __popc(m);
    }
    __syncwarp();
    // pairs of them whose signatures meet on >= 3 layers
    unsigned qn = 0;
    for (unsigned b = 0; b + 1 < ne; b += 32) {
        const unsigned i = b + lane, r = i < ne ? w.elig[i] : 0u;
        const uint2 s = i < ne ? w.sig[i] : make_uint2(0u, 0u);
        for (unsigned j = b + 1; j < ne; ++j) {
            const unsigned t = w.elig[j];
            const uint2 u = w.sig[j];
            const bool hit = j > i && sig_layers(s.x & u.x, s.y & u.y) >= 3;
            const unsigned m = __ballot_sync(FULL_MASK, hit);
            if (!m)
                continue;
            if (hit)
                w.pair[qn + __popc(m & lanemask_lt())] = r | t << 16;
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32) {
                p2_pairs(d.coords, d.roads, w, r0, 32);
                const unsigned rest = qn - 32, p = lane < rest ? w.pair[32 + lane] : 0u;
                __syncwarp();
                if (lane < rest)
                    w.pair[lane] = p;
                qn = rest;
                __syncwarp();
            }
        }
    }
    if (qn)
        p2_pairs(d.coords, d.roads, w, r0, qn);
#pragma unroll
    for (unsigned h = 0; h < 2; ++h) {
        const unsigned k = 32 * h + lane;
        n_comb += finish_road(d, list, k < nr, r0 + k, rec[h], ((unsigned long long)w.xm[k][1] << 32) | w.xm[k][0]);
    }
    __syncwarp();   // the state is refilled for the next event
}

// P2 over the events.  At most P2_ROUNDS per CTA: a CTA each.  More: those of
// more than P2W_ROADS roads (listed in P1) a CTA each from a queue, then every
// warp takes the other events one at a time, its first by its own index
// (neighbouring indices on different SMs), the rest from a queue.  An event of
// 64 roads takes a warp some 18 us whether it is alone or not, a CTA 6 us, so
// the line is at three: a chain of 400 events of one to eight hits on 152 CTAs
// 103 us with a warp each, 99 us with a CTA each, 1100 events that share hits
// on 456 CTAs 89.9 -> 87.3 us, 170 events on 152 CTAs 48.1 -> 40.5 us.  One
// combination-count atomic per CTA.
constexpr unsigned P2_ROUNDS = 3;
constexpr size_t P2_LIST_AT = (sizeof(P2Smem) > WARPS * P2W_BYTES ? sizeof(P2Smem) : WARPS * P2W_BYTES) / 16 * 16 + 16;

// The end of P2 in a CTA: its list goes out, its combinations are counted.
__device__ void p2_finish(const Dev &d, P2List &list, unsigned long long n_comb)
{
    n_comb = block_sum(n_comb);   // and every road has joined the list
    if (threadIdx.x == 0 && n_comb)
        atomicAdd(&d.ctrl->n_comb, n_comb);
    list_out(d, list);
}

__device__ void p2_phase(const Dev &d, unsigned char *smem, Batch &bt)
{
    // what the stage reads first, in one trip
    const unsigned n_events = bt.n_events, e0 = blockIdx.x;
    const unsigned n_big_ev = min(ldcg(&d.ctrl->n_big_ev), n_events);
    bt.n_roads = min(ldcg(&d.ctrl->n_roads), d.max_roads);
    // survivor totals of the road chunks start at zero (the fit adds to them)
    const unsigned n_chunks = min((bt.n_ep + ROAD_CHUNK - 1) / ROAD_CHUNK, d.max_chunks_r);
    for (unsigned i = blockIdx.x * BLOCK + threadIdx.x; i < n_chunks; i += gridDim.x * BLOCK)
        d.rchunk_sum[i] = 0;
    unsigned long long n_comb = 0;
    P2List &list = *reinterpret_cast<P2List *>(smem + P2_LIST_AT);
    if (threadIdx.x == 0)
        list.n = 0;
    for (unsigned i = threadIdx.x; i < P2_BUCKETS; i += BLOCK)
        list.cnt[i] = 0;
    __syncthreads();
    // first road and roads of event e (an event of more than MAX_ROADS_EV
    // roads is a fault, reported in P1)
    const auto roads_of = [&d](unsigned e, unsigned &r0) {
        r0 = e == 0 ? 0u : min(ldcg(d.ev_road_end + e - 1), d.max_roads);
        const unsigned r1 = min(ldcg(d.ev_road_end + e), d.max_roads);
        return min(r1 - min(r0, r1), (unsigned)MAX_ROADS_EV);
    };
    if (n_events <= P2_ROUNDS * gridDim.x) {   // few: a CTA each is the shortest time per event
        for (unsigned e = e0; e < n_events; e += gridDim.x) {
            unsigned r0;
            const unsigned nr = roads_of(e, r0);
            p2_event(d, r0, nr, smem, list, n_comb);
        }
        p2_finish(d, list, n_comb);
        return;
    }
    if (n_big_ev) {
        for (unsigned i = e0; i < n_big_ev; i = grab_after_first(d, Q_P2)) {
            const unsigned e = min(ldcg(d.ev_big + i), n_events - 1);
            unsigned r0;
            const unsigned nr = roads_of(e, r0);
            p2_event(d, r0, nr, smem, list, n_comb);
        }
        __syncthreads();   // the shared memory becomes the warps' regions
    }
    {
        P2Warp &w = *reinterpret_cast<P2Warp *>(smem + warp_id() * P2W_BYTES);
        const unsigned n_warps = gridDim.x * WARPS;
        for (unsigned e = warp_id() * gridDim.x + blockIdx.x; e < n_events;) {
            unsigned r0;
            const unsigned nr = roads_of(e, r0);
            if (nr && nr <= (unsigned)P2W_ROADS)   // the others were listed
                p2_warp(d, r0, nr, w, list, n_comb);
            if (n_events <= n_warps)
                break;
            unsigned ne = 0;
            if (lane_id() == 0)
                ne = n_warps + atomicAdd(&d.ctrl->q[Q_P2W], 1u);
            e = __shfl_sync(FULL_MASK, ne, 0);
        }
    }
    p2_finish(d, list, n_comb);
}

// ---------------------------------------------------------------------------
// P3: fit + cut + road-local hit-warrior: roads of like shape several to a warp
// step (the group path), larger ones a warp each (the box path), then the groups
// of the cross-road candidates; all three by lists made in P2
// ---------------------------------------------------------------------------

// the same triples as constants the compiler folds in unrolled loops: layer
// k of triple t
__device__ __forceinline__ unsigned triple_l(unsigned t, unsigned k)
{
    return (unsigned)(((k == 0 ? 0x2111000000ull : k == 1 ? 0x3322322111ull : 0x4443443432ull) >> (4 * t)) & 15u);
}

__device__ __forceinline__ unsigned long long make_key(long long chi2, unsigned rie, unsigned comb)
{
    return ((unsigned long long)chi2 << 23) | ((unsigned long long)rie << 15) | comb;
}

__device__ __forceinline__ long long sq(int a) { return (long long)a * a; }

// hash of a group key (splitmix64 finaliser)
__device__ __forceinline__ unsigned hash_slot(unsigned long long k, unsigned mask)
{
    k ^= k >> 30;
    k *= 0xBF58476D1CE4E5B9ull;
    k ^= k >> 27;
    k *= 0x94D049BB133111EBull;
    k ^= k >> 31;
    return (unsigned)k & mask;
}

// The group table is probed linearly from a group's home slot, at most
// HASH_PROBES slots, and may be filled to three quarters of its slots: a
// batch that needs more raises FLAG_CAPACITY (SVT_E_CAPACITY, no tracks)
// instead of probing on.
constexpr unsigned HASH_PROBES = 64;

__device__ __forceinline__ unsigned hash_probes(const Dev &d) { return min(HASH_PROBES, d.hash_mask + 1); }

__device__ unsigned hash_min(const Dev &d, unsigned long long gk, unsigned long long key)
{
    unsigned h = hash_slot(gk, d.hash_mask);
    for (unsigned probe = 0; probe < hash_probes(d); ++probe) {
        unsigned long long prev = atomicCAS(&d.hash[h].key, 0ull, gk);
        if (prev == 0ull) {   // a new slot: marked for clearing (no value awaited)
            atomicOr(&d.hash_bits[h >> 5], 1u << (h & 31u));
        }
        if (prev == 0ull || prev == gk) {
            atomicMax(&d.hash[h].val_inv, ~key);
            return prev == 0ull;
        }
        h = (h + 1) & d.hash_mask;
    }
    raise_flag(d, FLAG_CAPACITY);
    return 0;
}

// The warp's new slots of the group table join the batch's count.
__device__ void hash_count(const Dev &d, unsigned n)
{
    n = __reduce_add_sync(FULL_MASK, n);
    if (lane_id() == 0 && n) {
        const unsigned used = atomicAdd(&d.ctrl->hash_used, n), slots = d.hash_mask + 1;
        if (used == 0)
            raise_flag(d, FLAG_GROUPS);
        if (used + n > slots - slots / 4)
            raise_flag(d, FLAG_CAPACITY);
    }
}

// lookup after the table is complete (no writer in flight): a slot's key and
// value are read by one 16-byte load
__device__ unsigned long long hash_get(const Dev &d, unsigned long long gk)
{
    static_assert(sizeof(HashSlot) == 16, "one 16-byte load per slot");
    unsigned h = hash_slot(gk, d.hash_mask);
    for (unsigned probe = 0; probe < hash_probes(d); ++probe) {
        const ulonglong2 sl = __ldcg(reinterpret_cast<const ulonglong2 *>(d.hash + h));
        if (sl.x == gk)
            return ~sl.y;
        if (sl.x == 0ull)
            return NO_KEY;
        h = (h + 1) & d.hash_mask;
    }
    return NO_KEY;
}

__device__ __forceinline__ unsigned long long group_key(unsigned event, unsigned t, unsigned v0,
                                                        unsigned v1, unsigned v2)
{
    return ((unsigned long long)(event + 1) << 40) | ((unsigned long long)t << 36) |
           ((unsigned long long)v0 << 24) | ((unsigned long long)v1 << 12) | v2;
}

__device__ __forceinline__ unsigned nth_bit(unsigned mask, unsigned n)
{
    for (unsigned i = 0; i < n; ++i)
        mask &= mask - 1;
    return __ffs(mask) - 1;
}

// ---------------------------------------------------------------------------
// P3, group path: a warp fits several small roads at once, a group of lanes
// per road.  The four fitted slots get roles by falling hit count, (a, b, c,
// e).  A road's class bounds the hits of a by A = 2^LA, those of b and c by B
// = YN 2^LY and those of e by W, and its group is A x 2^LY lanes: lane (x, yl)
// holds hit x of slot a and the YN hits y = yl + j 2^LY of slot b, and runs
// over the hits z and w of slots c and e.
//
// A distinct fit survives the road-local warrior iff no passing fit of the
// road with a lower key shares two of its four hits.  Fits are compared by a
// 32-bit word, the chi-square shifted right until the cut fits 31 bits.  Each
// of the lane's pairs (x, y) keeps its lowest fit; it survives iff its word is
// the minimum of the other five pair tables.  At each z the tables (a, c),
// (b, c) and (c, e) are complete after a shuffle minimum over the group's
// other y, other x, and all its lanes; (a, e) and (b, e) follow after the
// loop from the minima over z.  No table is kept in memory.  Without two
// passing fits of one word that meet in a minimum (a tie) the words order the
// fits as the keys do.  Hits a strip or two apart often give the same floors,
// so how many roads have a tie depends on how near their hits lie: 0.2 % with
// hits anywhere, 8 % within 64 strips, 24 % within 16, 44 % within 8.  The roads
// with a tie take the step once more, by the same lanes from the hits still in
// shared memory, with whole keys in place of words (EXACT).
//
// A coordinate repeated within a layer needs nothing of its own.  For the warrior
// its hits are one hit (hits are shared by value).  The fits of the later hit are
// the earlier one's with a higher comb: they tie with them, lose to them in whole
// keys, and what they drop or publish the earlier ones drop or publish too.
//
// Bound: issue slots.  Several hits of slot b per lane (YN = 2) share the
// road's set-up, the loads and the shuffles of (a, c) and (c, e); with one
// hit per lane a warp step took 700 instructions for half the roads.
// ---------------------------------------------------------------------------

// Key of a fit from its summed partials s: (chi2, road bits and comb), or
// NO_KEY when it fails the cut.  s.x, s.y, s.z are 4096 times the three
// chi-square components before the floor (exact in int32, see the header);
// s.w is road << 15 | comb.
__device__ __forceinline__ unsigned long long box_key(const int4 &s, long long cut, bool &pass)
{
    const long long chi2 = sq(s.x >> 12) + sq(s.y >> 12) + sq(s.z >> 12);
    pass = chi2 <= cut;
    return pass ? (((unsigned long long)chi2 << 23) | (unsigned)s.w) : NO_KEY;
}

__device__ __forceinline__ int4 add4(const int4 &a, const int4 &b)
{
    return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// the six pairs of fitted slots (a, b)
__device__ __forceinline__ unsigned pair_a(unsigned p) { return (0x211000u >> (4 * p)) & 15u; }
__device__ __forceinline__ unsigned pair_b(unsigned p) { return (0x332321u >> (4 * p)) & 15u; }

constexpr unsigned GROUP_HITS = 128;   // hits of a warp's roads at most (sixteen roads of class 0)
struct P3Group {
    int4 A[GROUP_HITS];   // a road's hits in role order: chi-square partial sums (x, y, z) and comb
                          // part (w); role a also carries curvature, phi, 4096 k and the road bits
};

// The shape of a class and one lane's view of its group's road.
template <unsigned LA_, unsigned LY_, unsigned YN_, unsigned W_>
struct GroupRoad {
    static constexpr unsigned A = 1u << LA_, YL = 1u << LY_, YN = YN_, B = YN * YL, W = W_;
    static constexpr unsigned G = A * YL, ROADS = 32 / G, HITS = A + 2 * B + W;   // W <= B
    static_assert(ROADS * HITS <= GROUP_HITS, "the warp's hits fit its table");
    RoadItem it;
    const int4 *hit;            // the road's hits
    unsigned nf, excl;          // hits per fitted slot (4 bits each), excluded layer
    unsigned mb, mc, me;        // hits of slots b, c, e
    unsigned x, yl;             // the lane's hits
    bool live;                  // hit x exists
    unsigned long long cb;      // plain mode: first combination of the road
    __device__ unsigned slot(unsigned role) const { return (it.perm >> (2 * role)) & 3u; }
    __device__ unsigned m(unsigned s) const { return (nf >> (4 * s)) & 15u; }
    __device__ unsigned y(unsigned j) const { return yl + j * YL; }
    template <bool PLAIN>
    __device__ unsigned long long key(const Dev &d, long long cut, const int4 &s) const
    {
        if (PLAIN)
            return ldcg(d.fit_key + cb + (unsigned)s.w);
        bool pass;
        return box_key(s, cut, pass);
    }
    // the lane's fit at its hit j of slot b and hits z, w of slots c and e
    template <bool PLAIN>
    __device__ unsigned long long key_at(const Dev &d, long long cut, unsigned j, unsigned z, unsigned w) const
    {
        return key<PLAIN>(d, cut, add4(add4(hit[x], hit[A + y(j)]), add4(hit[A + B + z], hit[A + 2 * B + w])));
    }
};

// How the group path compares fits: by word, or (EXACT) by whole key; FAIL: no
// passing fit is as high.
template <bool EXACT>
struct FitKey {
    using type = unsigned;
    static constexpr unsigned FAIL = 0x80000000u;
};
template <>
struct FitKey<true> {
    using type = unsigned long long;
    static constexpr unsigned long long FAIL = NO_KEY;
};

// What a lane has found of its road's survivors: those of its pairs (flag,
// key, place among the road's survivors by comb), and the road's number.
template <unsigned YN>
struct GroupFound {
    bool surv[YN];
    unsigned long long key[YN];
    unsigned rank[YN], cnt;
};

// The survivors' places by comb (whole warp).
template <unsigned YN>
__device__ __forceinline__ void group_rank(GroupFound<YN> &f, unsigned gmask)
{
    const unsigned lane = lane_id();
#pragma unroll
    for (unsigned j = 0; j < YN; ++j)
        f.rank[j] = 0;
#pragma unroll
    for (unsigned i = 0; i < YN; ++i) {
        unsigned rest = __ballot_sync(FULL_MASK, f.surv[i]) & gmask;
        while (__any_sync(FULL_MASK, rest != 0u)) {
            const unsigned other = __shfl_sync(FULL_MASK, (unsigned)f.key[i] & 0x7FFFu, rest ? __ffs(rest) - 1 : lane);
#pragma unroll
            for (unsigned j = 0; j < YN; ++j)
                f.rank[j] += rest && other < ((unsigned)f.key[j] & 0x7FFFu);
            rest &= rest - 1;
        }
    }
}

// ---------------------------------------------------------------------------
// P3, publish: the groups of the cross-road candidates.  A group is a layer
// triple and three coordinates whose three hits are flagged as shared with
// another road of the event; the table gets the lowest key of the road's
// passing fits in it.  (Hits that repeat a coordinate publish the same group
// with higher keys.)
//
// A candidate has few groups (1.7 on average where 60 % of the hits are
// shared, and one road in five is a candidate), so the candidates of 32 roads
// put theirs together, one group a lane, and the lane computes its fits anew
// from the road's coordinates and constants.  Publishing in the fit's own step
// (two lanes of 32 at work, nearly every step waiting for the mask, the
// coordinates and the table) took 30 of 68 us of the fit stage for 1501 events
// that share hits.
// ---------------------------------------------------------------------------

// flagged hits of layer l: byte l of the mask; groups of triple t
__device__ __forceinline__ unsigned flagged(unsigned long long xm, unsigned l)
{
    return (unsigned)(xm >> (8 * l)) & 0xFFu;
}
__device__ __forceinline__ unsigned groups_of(unsigned long long xm, unsigned t)
{
    return __popc(flagged(xm, triple_l(t, 0))) * __popc(flagged(xm, triple_l(t, 1))) *
           __popc(flagged(xm, triple_l(t, 2)));
}
__device__ __forceinline__ unsigned groups_of(unsigned long long xm)
{
    unsigned total = 0;
#pragma unroll
    for (unsigned t = 0; t < 10; ++t)
        total += groups_of(xm, t);
    return total;
}

__device__ __forceinline__ int4 mad4(const int4 &b, const int4 &c, int v, unsigned w)
{
    return make_int4(b.x + c.x * v, b.y + c.y * v, b.z + c.z * v, b.w + (int)w);
}

// Publish group gi of road g (record r, flagged hits xm); 1 if it claimed a slot.
__device__ __noinline__ unsigned publish_group(const Dev &d, unsigned g, const RoadRec &r, unsigned long long xm,
                                               unsigned gi)
{
    const uint32_t pk = r.pk;
    const unsigned excl = min((pk >> 20) & 7u, 4u);
    unsigned t = 0, rem = gi;
    bool found = false;
#pragma unroll
    for (unsigned tt = 0; tt < 10; ++tt) {   // the triple of group gi
        const unsigned c = groups_of(xm, tt);
        if (!found) {
            if (rem < c) {
                t = tt;
                found = true;
            } else {
                rem -= c;
            }
        }
    }
    const unsigned lt[3] = {triple_l(t, 0), triple_l(t, 1), triple_l(t, 2)};
    const unsigned f0 = flagged(xm, lt[0]), f1 = flagged(xm, lt[1]), f2 = flagged(xm, lt[2]);
    const unsigned p0 = __popc(f0), p1 = __popc(f1);   // at most 8 each: the quotients are divm's
    const unsigned r1 = divm(rem, c_magic[p0]), r2 = divm(r1, c_magic[p1]);
    const unsigned dsel[3] = {nth_bit(f0, rem - r1 * p0), nth_bit(f1, r1 - r2 * p1), nth_bit(f2, r2)};
    // every load in one trip
    const uint16_t *co = d.coords + (size_t)g * 40;
    const int4 *cc = d.fitc + SET_INT4 * min((unsigned)r.set, (unsigned)(N_SETS - 1)) + SET_C;
    unsigned v[3], rest = 0xFu;   // rest: the fitted slots outside the triple
    int4 ct[3];
#pragma unroll
    for (unsigned q = 0; q < 3; ++q) {
        v[q] = ldcg(co + lt[q] * 8 + dsel[q]);
        const unsigned sl = min(lt[q] - (lt[q] > excl), 3u);
        ct[q] = __ldg(cc + sl);
        rest &= lt[q] == excl ? ~0u : ~(1u << sl);
    }
    // one, or two when the triple has the excluded layer (one: u and v the same)
    const unsigned su = __ffs(rest) - 1, sv = 31 - __clz(rest), Lu = su + (su >= excl), Lv = sv + (sv >= excl);
    const uint4 hu = ldcg(reinterpret_cast<const uint4 *>(co + Lu * 8)),
                hv = ldcg(reinterpret_cast<const uint4 *>(co + Lv * 8));
    const int4 cu = __ldg(cc + su), cv = __ldg(cc + sv), c4 = __ldg(cc + 4), c5 = __ldg(cc + 5),
               kk = __ldg(cc + 6);
    const unsigned S1 = pk & 15u, S2 = S1 * ((pk >> 4) & 15u), S3 = S2 * ((pk >> 8) & 15u),
                   S4 = S3 * ((pk >> 12) & 15u);   // comb strides of the layers
    const auto stride = [&](unsigned L) { return L == 0 ? 1u : L == 1 ? S1 : L == 2 ? S2 : L == 3 ? S3 : S4; };
    int4 base = make_int4(c4.x * r.curv + c5.x * r.phi + 4096 * kk.x, c4.y * r.curv + c5.y * r.phi + 4096 * kk.y,
                          c4.z * r.curv + c5.z * r.phi + 4096 * kk.z, (int)((pk >> 24) << 15));
#pragma unroll
    for (unsigned q = 0; q < 3; ++q)   // the excluded layer's hit counts in the comb alone
        base = mad4(base, ct[q], lt[q] == excl ? 0 : (int)v[q], dsel[q] * stride(lt[q]));
    const unsigned mu = (pk >> (4 * Lu)) & 15u, mv = su == sv ? 1u : (pk >> (4 * Lv)) & 15u, Su = stride(Lu), Sv = stride(Lv);
    unsigned long long mn = NO_KEY;
    for (unsigned a = 0; a < mu; ++a) {
        const int4 bu = mad4(base, cu, (int)row_at(hu, a), a * Su);
        for (unsigned b = 0; b < mv; ++b) {
            bool pass;
            const unsigned long long k =
                box_key(su == sv ? bu : mad4(bu, cv, (int)row_at(hv, b), b * Sv), d.cut, pass);
            mn = k < mn ? k : mn;
        }
    }
    return mn == NO_KEY ? 0u : hash_min(d, group_key(r.event, t, v[0], v[1], v[2]), mn);
}

// The groups of one road by the whole warp (the box path's roads, which have
// the most).
__device__ __noinline__ void publish_road(const Dev &d, unsigned g, const RoadRec &r)
{
    const unsigned long long xm = ldcg(d.xmask + g);
    const unsigned total = groups_of(xm);
    unsigned fresh = 0;
    for (unsigned gi = lane_id(); gi < total; gi += 32)
        fresh += publish_group(d, g, r, xm, gi);
    __syncwarp();
    hash_count(d, fresh);
}

// Part `part` of `parts` of the groups of the candidates among roads
// 32 w .. 32 w + 31 that the group path fits.
__device__ __forceinline__ void publish_word(const Dev &d, unsigned w, unsigned part, unsigned parts, unsigned n_roads)
{
    const unsigned lane = lane_id(), g = w * 32 + lane;
    const bool cand = ((ldcg(d.cand_bits + w) >> lane) & 1u) && g < n_roads;
    RoadRec r{};
    unsigned long long xm = 0;
    if (cand) {
        r = ldcg(d.roads + g);
        xm = ldcg(d.xmask + g);
    }
    const unsigned total = cand && ((r.fit >> 8) & 7u) < N_GROUP_CLS ? groups_of(xm) : 0u;
    unsigned inc = total;   // groups up to and with the lane's road
#pragma unroll
    for (unsigned o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(FULL_MASK, inc, o);
        inc += lane >= o ? u : 0u;
    }
    const unsigned all = __shfl_sync(FULL_MASK, inc, 31);
    unsigned fresh = 0;
    for (unsigned i0 = 32 * part; i0 < all; i0 += 32 * parts) {
        const unsigned i = i0 + lane;
        unsigned src = 0;   // roads whose groups all lie below i
#pragma unroll
        for (unsigned o = 16; o; o >>= 1)
            src += __shfl_sync(FULL_MASK, inc, src + o - 1) <= i ? o : 0u;
        const unsigned gi = i - __shfl_sync(FULL_MASK, inc - total, src);
        uint4 v;
        memcpy(&v, &r, sizeof v);
        v.x = __shfl_sync(FULL_MASK, v.x, src);
        v.y = __shfl_sync(FULL_MASK, v.y, src);
        v.z = __shfl_sync(FULL_MASK, v.z, src);
        v.w = __shfl_sync(FULL_MASK, v.w, src);
        RoadRec rs;
        memcpy(&rs, &v, sizeof v);
        const unsigned long long xs = __shfl_sync(FULL_MASK, xm, src);
        if (i < all)
            fresh += publish_group(d, w * 32 + src, rs, xs, gi);
        __syncwarp();
    }
    hash_count(d, fresh);
}

// The groups of every word's candidates, a word in as many parts as there are
// warps for.
__device__ __noinline__ void publish_words(const Dev &d)
{
    const unsigned n_roads = min(ldcg(&d.ctrl->n_roads), d.max_roads), words = (n_roads + 31) / 32;
    const unsigned n_warps = gridDim.x * WARPS, parts = words ? max(n_warps / words, 1u) : 1u;
    for (unsigned i = warp_id() * gridDim.x + blockIdx.x; i < words * parts; i += n_warps)
        publish_word(d, i % words, i / words, parts, n_roads);
}

// ---------------------------------------------------------------------------
// P3, box path: one warp fits one listed road (more distinct fits than
// small_n4, or more than four hits in its second largest slot).  The four fitted
// slots get roles (a, b, c, e).  A fit survives the road-local warrior iff its
// key is the minimum of all six pair tables (minima over the fits with the same
// hits on two slots): two fitted hits and a hit of the excluded layer are a group,
// and a group of three fitted hits lies within the fits of two of them.  It is
// then the minimum of its pair (x, y) of slots a and b, so a pair has at most one
// candidate and a road at most 64 survivors.  box_warp is the fused form;
// box_plain reads the keys that the plain pipeline's fit kernel stored.
//
// box_plain: hits with one coordinate in one layer are one hit for the warrior
// (hits are shared by value), and among fits with the same coordinates the
// lowest hit index has the lowest comb.  So its tables and survivors take
// canonical hits only (the lowest index of each coordinate), and the warp works
// on the box of canonical fits; in pass p, lane t = 32 p + lane takes
// the pair (x, y) = (t mod m_a, t div m_a) and loops over (z, w) of slots c and
// e.  Of the six tables that loop makes three:
//   T_ab[x][y]  the lane's minimum over its own fits
//   T_ac, T_bc  the lane's minimum over w at each z, folded over the lanes
// A pair's minimum that holds T_ac and T_bc (about one per road) is then
// checked against the other three (T_ae, T_be, T_ce), taken on demand by a
// warp-wide minimum over the other two slots' hits (box_min2), as are the
// entries the publish step reads.
// The lane minima are folded by 32-bit shared-memory atomics without a
// return value, each pass into tables of its own: the high words first,
// then, after the warp has synchronised, the low words of the lanes whose
// high word is the minimum.  That is the exact minimum of the 64-bit keys
// over the pass (every lane of the pass takes part in the same steps); the
// survivor check takes the smaller of the two passes' entries.
// ---------------------------------------------------------------------------

enum { T_AB = 0, T_CE, T_AE, T_BE, T_AC, T_BC };
// table row stride: rows 9 entries apart put the entries [u][v] of
// different u in different banks
constexpr unsigned TS = 9;

// The float passes' partials by role (see box_warp): the components' / 4096, the
// first role's less 0.5.
struct P3Float {
    float4 hit[2][8];            // roles a and b
    ulonglong2 c[8][2];          // role c, each component as a pair of equals
    ulonglong2 e[2][3];          // role e, hits 4 i .. 4 i + 3 by component, in pairs
    float bias[8];               // what the floor pass adds to hit w's x component
};

struct P3Box {
    union {
        struct {
            unsigned long long T[4][8 * TS];   // T_ab, T_ce, T_ae, T_be: [u * TS + v] (u: the first
                                               // role's hit); the last three only where needed
            unsigned H[2][2][8 * TS];          // T_ac, T_bc of pass 0 and pass 1: high words
            unsigned L[2][2][8 * TS];          // and low words (of the keys with the minimum high word)
        };
        P3Float F;
    };
    int4 A[4][8];                      // slot j, canonical hit k: chi-square partial sums (x, y,
                                       // z) and comb part (w); slot 0 also carries curvature, phi,
                                       // 4096 k and the road bits of the key
    uint16_t co[40];                   // the road's coordinates, [layer * 8 + hit]
    uint8_t rank[4][8];                // canonical hit (class) of raw hit d of slot j
};
static_assert(offsetof(P3Box, A) % 16 == 0 && offsetof(P3Box, co) % 16 == 0 && sizeof(P3Float) % 16 == 0,
              "16-byte rows");

__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b)
{
    return b < a ? b : a;
}

// the warp's minimum key
__device__ __forceinline__ unsigned long long warp_min_key(unsigned long long key)
{
    const unsigned hi = (unsigned)(key >> 32);
    const unsigned mh = __reduce_min_sync(FULL_MASK, hi);
    const unsigned ml = __reduce_min_sync(FULL_MASK, hi == mh ? (unsigned)key : 0xFFFFFFFFu);
    return ((unsigned long long)mh << 32) | ml;
}

// entry idx of pair table tab: T_ab and T_ce as stored, the others the
// smaller of the two passes' (high, low) entries
__device__ __forceinline__ unsigned long long box_get(const P3Box &B, unsigned tab, unsigned idx)
{
    if (tab < T_AC)
        return B.T[tab][idx];
    const unsigned t = tab - T_AC;
    return umin64(((unsigned long long)B.H[0][t][idx] << 32) | B.L[0][t][idx],
                  ((unsigned long long)B.H[1][t][idx] << 32) | B.L[1][t][idx]);
}

// Fold v into entry idx of table t of pass q, stage 1 (high word); stage 2
// (low word) runs after the warp has synchronised: only lanes whose high
// word is then the minimum take part.
__device__ __forceinline__ void fold_hi(P3Box &B, unsigned q, unsigned t, unsigned idx, unsigned long long v)
{
    atomicMin(&B.H[q][t][idx], (unsigned)(v >> 32));
}
__device__ __forceinline__ void fold_lo(P3Box &B, unsigned q, unsigned t, unsigned idx, unsigned long long v)
{
    if ((unsigned)(v >> 32) == B.H[q][t][idx])
        atomicMin(&B.L[q][t][idx], (unsigned)v);
}

// hits of layer l of a road record (clamped to the format limit)
__device__ __forceinline__ unsigned hits_of(uint32_t pk, unsigned l)
{
    return min((pk >> (4 * l)) & 15u, (unsigned)MAX_HITS);
}

// Shape of a road in the box path, the same in every lane.
struct BoxShape {
    unsigned mpk;              // canonical hits of fitted slot j in bits 4j .. 4j + 3
    unsigned ra, rb, rc, re;   // the slots in roles a, b, c, e
    unsigned ma, mb, mc, me;   // their canonical hits
    unsigned ne;               // raw hits of the excluded layer
    unsigned long long cb;     // plain mode: first combination of the road
    __device__ unsigned m(unsigned s) const { return (mpk >> (4 * s)) & 15u; }
};

// The key of a fit without the cut: chi2 << 23 | cw (the cut is key < kb).
__device__ __forceinline__ unsigned long long box_key_raw(const int4 &s, unsigned cw)
{
    const long long chi2 = sq(s.x >> 12) + sq(s.y >> 12) + sq(s.z >> 12);
    const unsigned hi = (unsigned)((unsigned long long)chi2 >> 9);
    const unsigned lo = ((unsigned)chi2 << 23) + cw;
    return ((unsigned long long)hi << 32) | lo;
}

// One pass over the pairs (x, y) of slots a and b: lane t = 32 p + lane.
// The inner loop over the hits of slot e has ME (4 or 8, at least me) steps,
// unrolled and predicated, so a step has no branch.  FULLW: every lane has a
// pair and slot e eight hits.  T_ce is not made here (see box_tce).
template <unsigned ME, bool FULLW>
__device__ void box_pass(const Dev &d, P3Box &B, const BoxShape &sh, unsigned p)
{
    const unsigned lane = lane_id();
    const unsigned ma = sh.ma, mb = sh.mb, mc = sh.mc, me = sh.me;
    const unsigned t = p * 32 + lane;
    const bool act = t < ma * mb;
    const unsigned y = act ? divm(t, c_magic[ma]) : 0u, x = act ? t - y * ma : 0u;
    const int pab = B.A[sh.ra][x].w + B.A[sh.rb][y].w;
    unsigned long long qab = NO_KEY;
    for (unsigned z = 0; z < mc; ++z) {
        const int pz = pab + B.A[sh.rc][z].w;
        unsigned long long rz = NO_KEY;
#pragma unroll
        for (unsigned w = 0; w < ME; ++w)
            if (FULLW || (act && w < me))
                rz = umin64(rz, ldcg(d.fit_key + sh.cb + (unsigned)(pz + B.A[sh.re][w].w)));
        qab = umin64(qab, rz);
        const unsigned q = p & 1u;
        if (act) {
            fold_hi(B, q, T_AC - T_AC, x * TS + z, rz);
            fold_hi(B, q, T_BC - T_AC, y * TS + z, rz);
        }
        __syncwarp();
        if (act) {
            fold_lo(B, q, T_AC - T_AC, x * TS + z, rz);
            fold_lo(B, q, T_BC - T_AC, y * TS + z, rz);
        }
    }
    if (act)
        B.T[T_AB][x * TS + y] = qab;
    __syncwarp();
}

// The minimum key over the fits with canonical hit kp of slot sp and kq of
// slot sq (sp != sq), taken on demand by the warp: lanes over the canonical
// hits of the other two slots (every lane calls it with the same arguments;
// the result is the same in every lane).  Gives T_ae, T_be and T_ce, which
// the passes do not fold.
__device__ unsigned long long box_min2(const Dev &d, const P3Box &B, const BoxShape &sh, unsigned sp, unsigned kp,
                                       unsigned sq, unsigned kq)
{
    const unsigned lane = lane_id();
    const unsigned rest = 0xFu & ~(1u << sp) & ~(1u << sq);
    const unsigned su = __ffs(rest) - 1, sv = 31 - __clz(rest);
    const unsigned mu = sh.m(su), mv = sh.m(sv);
    const int pf = B.A[sp][kp].w + B.A[sq][kq].w;
    unsigned long long mn = NO_KEY;
    for (unsigned t = lane; t < mu * mv; t += 32) {
        const unsigned iv = divm(t, c_magic[mu]), iu = t - iv * mu;
        mn = umin64(mn, ldcg(d.fit_key + sh.cb + (unsigned)(pf + B.A[su][iu].w + B.A[sv][iv].w)));
    }
    return warp_min_key(mn);
}

// T_ce[z][w]: the minimum key over every pair (x, y) at hits z, w of slots c and e
__device__ __forceinline__ unsigned long long box_tce(const Dev &d, const P3Box &B, const BoxShape &sh, unsigned z,
                                                      unsigned w)
{
    return box_min2(d, B, sh, sh.rc, z, sh.re, w);
}

// the table holding the minima over slots p and q (p != q) and the index of
// canonical hits (kp, kq) in it
__device__ __forceinline__ unsigned box_tab(const BoxShape &sh, unsigned p, unsigned kp, unsigned q, unsigned kq,
                                            unsigned &idx)
{
    const auto role = [&sh](unsigned s) {
        return s == sh.ra ? 0u : s == sh.rb ? 1u : s == sh.rc ? 2u : 3u;
    };
    unsigned r1 = role(p), r2 = role(q), k1 = kp, k2 = kq;
    if (r1 > r2) {
        const unsigned tr = r1, tk = k1;
        r1 = r2;
        k1 = k2;
        r2 = tr;
        k2 = tk;
    }
    idx = k1 * TS + k2;
    // role pairs (0,1) ab, (2,3) ce, (0,2) ac, (1,2) bc, (0,3) ae, (1,3) be
    return r1 == 0 && r2 == 1 ? T_AB : r1 == 2 ? T_CE : r2 == 2 ? (r1 == 0 ? T_AC : T_BC) : (r1 == 0 ? T_AE : T_BE);
}

// ---------------------------------------------------------------------------
// P3, box path, fused: the road's chi-squares in float, two fits per
// instruction, with a bound on their error; whole numbers decide only where
// floats cannot.
//
// With v the float sums of the per-hit partials / 4096, less 0.5, each
// component differs from the floor a by at most 0.62: 0.5 from the floor, and
// 0.11 from the conversions (2^-5 in all), the 0.5 (2^-5) and three sums (2^-6
// each) of numbers below 2^19.  So | |v| - |a| | <= sqrt(3) 0.62 < 1.075, and
// the float c of |v|^2 is off by a relative 2.5e-7 at most.  Hence, for the
// chi-squares X of two fits with floats c:
//   X1 <= X2  =>  c1 <= c2 + 4.3 sqrt(c2) + 4.7 and a little  (near: not certainly larger)
//   X <= cut  =>  c <= float_hi,   X > cut  =>  c >= float_lo
//
// Lane (x, yl) holds hit x of slot a (eight) and hits yl, yl + 4 of slot b and
// runs over the hits z and w of slots c and e.  The passing fits are those
// below float_lo; a fit in [float_lo, float_hi] (one road in thirty) makes the
// warp count again in whole numbers.  A pair (x, y) is a candidate when its
// lowest row is near the minima of tables (a, c) and (b, c) there, which are
// shuffle minima.  A candidate's lowest fit is found in whole keys; it survives
// when none of the fits that share two hits with it (about 320) has a lower one.
//
// How many candidates there are depends on how near a road's hits lie: of 8^4
// roads 1 with hits anywhere, 3 within 64 strips, 12 within 16, 29 within 8.  The
// rows near at the first z say so (as many as there will be candidates): with more
// than FLOAT_CANDS of them the pass ends there and the floor pass takes its place,
// whose floats tell apart all but equal chi-squares (two candidates within 8
// strips); where many are equal (constants of zero), the key pass takes its.
//
// Bound: issue slots, nine instructions per fit (14 in the floor pass, 20 in
// the key pass, whose 64-bit minima have a seventh of the float rate).  The fit
// stage of 12,800 roads of 8^4 fits: 50 us with hits anywhere, 69 within 16 strips,
// 80 within 8, 105 with all chi-squares equal; in whole numbers with tables in
// shared memory alone 84, 85, 89 and 85.
// ---------------------------------------------------------------------------

constexpr long long FLOAT_CUT = 1ll << 24;   // a smaller cut's band [lo, hi] is a visible share of the fits: floor pass
constexpr float FLOAT_PAD = 1e18f;           // component of a missing hit: its fits are far above every cut
constexpr unsigned FLOAT_CANDS = 8;          // candidates a pass follows up (a candidate takes some 300 instructions)

// Two floats in one 64-bit register pair (kept packed from load to result:
// packing at every operation cost more moves than the operations), added and
// multiplied by one instruction each.
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_pack(float x, float y)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 f2_get(f2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// What the float of a fit not above one of float c2 stays below, without a root:
// 4.32 sqrt(c2) <= e c2 + 4.67 / e for every e; e = 5 / sqrt(cut) makes that equal
// near 0.2 cut (eps = 1.000002 + e, off = 4.8 + 0.94 sqrt(cut)).
#define float_thr(c2) fmaf((c2), eps, off)

// One lane's view of a road's fits: passing ones (below the band from `lo`),
// the lowest place in the band, and of each of its pairs the lowest row and
// the lowest row near the minima of tables (a, c) and (b, c).  hi: the band's end.
struct FloatPass {
    unsigned np, near_cut;
    float q[2], qok[2];
    bool many;   // the pass stopped after the first z: more than FLOAT_CANDS near rows
};

// TWO: slot b has more than four hits (the lane's second y); WIDE: slot e has.
template <bool TWO, bool WIDE>
__device__ __forceinline__ FloatPass float_pass(const P3Float &F, unsigned mc, unsigned lo, float hi, float eps, float off)
{
    constexpr unsigned NJ = TWO ? 2 : 1, NI = WIDE ? 2 : 1;
    const unsigned x = lane_id() & 7u, yl = lane_id() >> 3;
    FloatPass f{0u, ~0u, {3e38f, 3e38f}, {3e38f, 3e38f}, false};
    f2 px[NJ], py[NJ], pz[NJ];
#pragma unroll
    for (unsigned j = 0; j < NJ; ++j) {
        const float4 a = F.hit[0][x], b = F.hit[1][yl + 4 * j];
        px[j] = f2_pack(a.x + b.x, a.x + b.x);
        py[j] = f2_pack(a.y + b.y, a.y + b.y);
        pz[j] = f2_pack(a.z + b.z, a.z + b.z);
    }
#pragma unroll 1
    for (unsigned z = 0; z < mc; ++z) {
        const ulonglong2 cxy = F.c[z][0];
        const f2 cz = F.c[z][1].x;
        float rz[NJ];
#pragma unroll
        for (unsigned i = 0; i < NI; ++i) {
            const ulonglong2 ex = F.e[i][0], ey = F.e[i][1], ez = F.e[i][2];
#pragma unroll
            for (unsigned j = 0; j < NJ; ++j) {
                const f2 zx = f2_add(px[j], cxy.x), zy = f2_add(py[j], cxy.y), zz = f2_add(pz[j], cz);
#pragma unroll
                for (unsigned h = 0; h < 2; ++h) {
                    const f2 vx = f2_add(zx, h ? ex.y : ex.x), vy = f2_add(zy, h ? ey.y : ey.x),
                             vz = f2_add(zz, h ? ez.y : ez.x);
                    const float2 c = f2_get(f2_fma(vz, vz, f2_fma(vy, vy, f2_mul(vx, vx))));
                    const unsigned d0 = __float_as_uint(c.x) - lo, d1 = __float_as_uint(c.y) - lo;
                    f.np += d0 >> 31;
                    f.np += d1 >> 31;
                    f.near_cut = min(f.near_cut, min(d0, d1));
                    rz[j] = i + h ? fminf(rz[j], fminf(c.x, c.y)) : fminf(c.x, c.y);
                }
            }
        }
        float ac = TWO ? fminf(rz[0], rz[NJ - 1]) : rz[0];   // (a, c) at x, z
        ac = fminf(ac, __shfl_xor_sync(FULL_MASK, ac, 8));
        ac = fminf(ac, __shfl_xor_sync(FULL_MASK, ac, 16));
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j) {
            float bc = rz[j];   // (b, c) at y, z
            bc = fminf(bc, __shfl_xor_sync(FULL_MASK, bc, 1));
            bc = fminf(bc, __shfl_xor_sync(FULL_MASK, bc, 2));
            bc = fminf(bc, __shfl_xor_sync(FULL_MASK, bc, 4));
            f.q[j] = fminf(f.q[j], rz[j]);
            f.qok[j] = rz[j] <= float_thr(fminf(ac, bc)) ? fminf(f.qok[j], rz[j]) : f.qok[j];
        }
        if (z == 0) {
            unsigned n = 0;
#pragma unroll
            for (unsigned j = 0; j < NJ; ++j)
                n += __popc(__ballot_sync(FULL_MASK, f.qok[j] <= hi));
            f.many = n > FLOAT_CANDS;
            if (f.many)
                break;
        }
    }
    return f;
}

// The same with the components' floors, which floats hold exactly: a chi-square
// is then off by a relative 1.8e-7 at most, X1 <= X2 => c1 <= c2 FLOOR_EPS, and
// rows are near only where chi-squares are all but equal.  The floor a of a sum
// (|a| < 2^19) becomes a float by adding it to the bits of 1.5 2^23.  One loop over
// the pairs of hits of slot e, and one body of the key pass: roads of many shapes
// meet here (with a body for each, 19,200 roads of one to eight hits within 16
// strips took 87 us of the fit stage, 72 with these; 8^4 roads 70 and 69).
constexpr float FLOOR_EPS = 1.0000005f, FLOOR_BIAS = -12582912.f;

template <bool TWO>
__device__ __forceinline__ FloatPass floor_pass(const P3Box &B, const BoxShape &sh, unsigned lo, float hi)
{
    constexpr unsigned NJ = TWO ? 2 : 1;
    const unsigned x = lane_id() & 7u, yl = lane_id() >> 3;
    FloatPass f{0u, ~0u, {3e38f, 3e38f}, {3e38f, 3e38f}, false};
    const f2 bias = f2_pack(FLOOR_BIAS, FLOOR_BIAS);
    int4 pab[NJ];
    bool live[NJ];
    unsigned np[NJ];
#pragma unroll
    for (unsigned j = 0; j < NJ; ++j) {   // (a missing hit's row is unspecified)
        pab[j] = add4(B.A[0][x], B.A[1][yl + 4 * j]);
        live[j] = x < sh.ma && yl + 4 * j < sh.mb;
        np[j] = 0;
    }
#pragma unroll 1
    for (unsigned z = 0; z < sh.mc; ++z) {
        int4 pz[NJ];
        float rz[NJ];
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j)
            pz[j] = add4(pab[j], B.A[2][z]), rz[j] = 3e38f;
#pragma unroll 1
        for (unsigned i = 0; 2 * i < sh.me; ++i) {
            const int4 a0 = B.A[3][2 * i], a1 = B.A[3][2 * i + 1];
            const f2 bx = reinterpret_cast<const f2 *>(B.F.bias)[i];   // (a missing hit's: far above every cut)
            const auto part = [](int s, int t, f2 b) {
                return f2_add(f2_pack(__int_as_float((s >> 12) + 0x4B400000), __int_as_float((t >> 12) + 0x4B400000)), b);
            };
#pragma unroll
            for (unsigned j = 0; j < NJ; ++j) {
                const f2 vx = part(pz[j].x + a0.x, pz[j].x + a1.x, bx), vy = part(pz[j].y + a0.y, pz[j].y + a1.y, bias),
                         vz = part(pz[j].z + a0.z, pz[j].z + a1.z, bias);
                const float2 c = f2_get(f2_fma(vz, vz, f2_fma(vy, vy, f2_mul(vx, vx))));
                const unsigned d0 = __float_as_uint(c.x) - lo, d1 = __float_as_uint(c.y) - lo;
                np[j] += d0 >> 31;
                np[j] += d1 >> 31;
                f.near_cut = min(f.near_cut, min(d0, d1));
                rz[j] = fminf(rz[j], fminf(c.x, c.y));
            }
        }
        float ac = 3e38f;   // (a, c) at x, z
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j) {
            rz[j] = live[j] ? rz[j] : 3e38f;
            ac = fminf(ac, rz[j]);
        }
        ac = fminf(ac, __shfl_xor_sync(FULL_MASK, ac, 8));
        ac = fminf(ac, __shfl_xor_sync(FULL_MASK, ac, 16));
        unsigned n = 0;
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j) {
            float bc = rz[j];   // (b, c) at y, z
            bc = fminf(bc, __shfl_xor_sync(FULL_MASK, bc, 1));
            bc = fminf(bc, __shfl_xor_sync(FULL_MASK, bc, 2));
            bc = fminf(bc, __shfl_xor_sync(FULL_MASK, bc, 4));
            f.q[j] = fminf(f.q[j], rz[j]);
            f.qok[j] = rz[j] <= fminf(ac, bc) * FLOOR_EPS ? fminf(f.qok[j], rz[j]) : f.qok[j];
            if (z == 0)
                n += __popc(__ballot_sync(FULL_MASK, f.qok[j] <= hi));
        }
        f.many = n > FLOAT_CANDS;
        if (f.many)
            break;
    }
#pragma unroll
    for (unsigned j = 0; j < NJ; ++j)
        f.np += live[j] ? np[j] : 0u;
    return f;
}

// The same in whole keys: the lane's passing fits, and of each of its pairs the
// lowest one and whether tables (a, c) and (b, c) hold it too.  Keys differ by
// comb, so that a pair has one lowest fit and no two are near.
struct KeyPass {
    unsigned np;
    unsigned long long q[2];
    bool ok[2];
};

__device__ __forceinline__ KeyPass key_pass(const P3Box &B, const BoxShape &sh, long long cut)
{
    constexpr unsigned NJ = 2;
    const unsigned x = lane_id() & 7u, yl = lane_id() >> 3;
    // within a row (x, y, z) the order by (chi2, w) is that by key
    const unsigned long long rb = (unsigned long long)(min(cut, 1ll << 38) + 1) << 3;   // chi2 <= cut iff below
    KeyPass f{0u, {NO_KEY, NO_KEY}, {false, false}};
    int4 pab[NJ];
    unsigned np[NJ] = {0u, 0u};
#pragma unroll
    for (unsigned j = 0; j < NJ; ++j)
        pab[j] = add4(B.A[0][x], B.A[1][yl + 4 * j]);
#pragma unroll 1
    for (unsigned z = 0; z < sh.mc; ++z) {
        int4 pz[NJ];
        unsigned long long rz[NJ];
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j) {
            pz[j] = add4(pab[j], B.A[2][z]);
            rz[j] = NO_KEY;
        }
#pragma unroll 1
        for (unsigned w = 0; w < sh.me; ++w) {
            const int4 aw = B.A[3][w];
#pragma unroll
            for (unsigned j = 0; j < NJ; ++j) {
                const long long chi2 = sq((pz[j].x + aw.x) >> 12) + sq((pz[j].y + aw.y) >> 12) + sq((pz[j].z + aw.z) >> 12);
                const unsigned long long key = (unsigned long long)chi2 << 3 | w;
                np[j] += key < rb;
                rz[j] = umin64(rz[j], key);
            }
        }
        unsigned long long ac = NO_KEY;   // (a, c) at x, z
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j) {
            // (no passing fit, or a pair whose hits do not exist: its sums are unspecified)
            rz[j] = rz[j] < rb && x < sh.ma && yl + 4 * j < sh.mb
                        ? (rz[j] >> 3 << 23) + (unsigned)(pz[j].w + B.A[3][(unsigned)rz[j] & 7u].w)
                        : NO_KEY;
            ac = umin64(ac, rz[j]);
        }
        ac = umin64(ac, __shfl_xor_sync(FULL_MASK, ac, 8));
        ac = umin64(ac, __shfl_xor_sync(FULL_MASK, ac, 16));
#pragma unroll
        for (unsigned j = 0; j < NJ; ++j) {
            unsigned long long bc = rz[j];   // (b, c) at y, z
            bc = umin64(bc, __shfl_xor_sync(FULL_MASK, bc, 1));
            bc = umin64(bc, __shfl_xor_sync(FULL_MASK, bc, 2));
            bc = umin64(bc, __shfl_xor_sync(FULL_MASK, bc, 4));
            if (rz[j] < f.q[j]) {   // (keys differ by comb: no two are equal but NO_KEY)
                f.q[j] = rz[j];
                f.ok[j] = umin64(ac, bc) == rz[j];
            }
        }
    }
#pragma unroll
    for (unsigned j = 0; j < NJ; ++j)
        f.np += x < sh.ma && yl + 4 * j < sh.mb ? np[j] : 0u;
    return f;
}

// Fit road g with one warp.  The shape's slots are roles here, by falling hit
// count.  Hits that repeat a coordinate need nothing special (as in the group
// path).  Bound: issue slots (two fits an instruction).  The fit stage of 25,600
// roads of 8^4 distinct fits: 153.8 -> 80.5 us (whole keys with tables in shared
// memory before).
__device__ __noinline__ void box_warp(const Dev &d, unsigned char *region, unsigned g, unsigned long long &npass)
{
    P3Box &B = *reinterpret_cast<P3Box *>(region);
    P3Float &F = B.F;
    const unsigned lane = lane_id();
    const RoadRec rec = ldcg(d.roads + g);
    const uint32_t pk = rec.pk;
    const unsigned excl = min((pk >> 20) & 7u, 4u), nf = fitted_counts(pk);
    BoxShape sh;
    sh.ra = 0;
    sh.rb = 1;
    sh.rc = 2;
    sh.re = 3;
    sh.ma = (nf >> (4 * (rec.fit & 3u))) & 15u;
    sh.mb = (nf >> (4 * ((rec.fit >> 2) & 3u))) & 15u;
    sh.mc = (nf >> (4 * ((rec.fit >> 4) & 3u))) & 15u;
    sh.me = (nf >> (4 * ((rec.fit >> 6) & 3u))) & 15u;
    sh.mpk = sh.ma | sh.mb << 4 | sh.mc << 8 | sh.me << 12;
    sh.ne = hits_of(pk, excl);
    sh.cb = 0;
    __syncwarp();   // the region's previous user is done
    {   // lane 8 role + k: hit k
        const unsigned role = lane >> 3, k = lane & 7u, s = (rec.fit >> (2 * role)) & 3u;
        float4 v = make_float4(FLOAT_PAD, 0.f, 0.f, 0.f);
        if (k < sh.m(role)) {
            const unsigned L = s + (s >= excl);
            const int h = ldcg(d.coords + (size_t)g * 40 + L * 8 + k);
            const int4 *cc = d.fitc + SET_INT4 * min((unsigned)rec.set, (unsigned)(N_SETS - 1)) + SET_C;
            const int4 cj = __ldg(cc + s);
            unsigned S = 1;   // comb stride of layer L
            for (unsigned l = 0; l < L; ++l)
                S *= (pk >> (4 * l)) & 15u;
            int4 a = make_int4(cj.x * h, cj.y * h, cj.z * h, (int)(k * S));
            float o = 0.f;
            if (role == 0) {   // curvature, phi, 4096 * offset and the road bits
                const int4 c4 = __ldg(cc + 4), c5 = __ldg(cc + 5), kk = __ldg(cc + 6);
                a.x += c4.x * rec.curv + c5.x * rec.phi + 4096 * kk.x;
                a.y += c4.y * rec.curv + c5.y * rec.phi + 4096 * kk.y;
                a.z += c4.z * rec.curv + c5.z * rec.phi + 4096 * kk.z;
                a.w += (int)((pk >> 24) << 15);
                o = -0.5f;
            }
            B.A[role][k] = a;
            v = make_float4(fmaf((float)a.x, 1.f / 4096.f, o), fmaf((float)a.y, 1.f / 4096.f, o),
                            fmaf((float)a.z, 1.f / 4096.f, o), 0.f);
        }
        if (role < 2)
            F.hit[role][k] = v;
        if (role == 2) {
            F.c[k][0] = ulonglong2{f2_pack(v.x, v.x), f2_pack(v.y, v.y)};
            F.c[k][1].x = f2_pack(v.z, v.z);
        }
        if (role == 3) {
            float *e = reinterpret_cast<float *>(&F.e[k >> 2][0]) + (k & 3u);
            e[0] = v.x;
            e[4] = v.y;
            e[8] = v.z;
            F.bias[k] = k < sh.me ? FLOOR_BIAS : FLOAT_PAD;
        }
    }
    __syncwarp();
    unsigned cand[2];
    // what decides: 0 floats, 1 floats of the floors, 2 whole keys
    unsigned by = d.cut < FLOAT_CUT ? 1u : 0u, width = 0;
    const float cut = (float)min(d.cut, 1ll << 38);
    FloatPass f;
    // candidates of a float pass whose chi-squares are near within (eps, off)
    const auto candidates = [&](float eps, float off, float hi) {
#pragma unroll
        for (unsigned j = 0; j < 2; ++j)
            cand[j] = __ballot_sync(FULL_MASK, f.qok[j] <= float_thr(f.q[j]) && f.q[j] <= hi);
        return f.many || __popc(cand[0]) + __popc(cand[1]) > FLOAT_CANDS;   // too many
    };
    if (by == 0) {
        // the cut's band
        const float root = sqrt_approx(cut), band = fmaf(2.2f, root, 8.f);
        const float eps = 1.000002f + 5.f / root, off = fmaf(0.94f, root, 4.8f);   // of float_thr
        const float float_lo = cut * 0.999999f - band, float_hi = cut * 1.000001f + band;
        const unsigned lo = __float_as_uint(float_lo);
        width = __float_as_uint(float_hi) + 1 - lo;
        if (sh.mb > 4 && sh.me > 4)
            f = float_pass<true, true>(F, sh.mc, lo, float_hi, eps, off);
        else if (sh.mb > 4)
            f = float_pass<true, false>(F, sh.mc, lo, float_hi, eps, off);
        else if (sh.me > 4)
            f = float_pass<false, true>(F, sh.mc, lo, float_hi, eps, off);
        else
            f = float_pass<false, false>(F, sh.mc, lo, float_hi, eps, off);
        by = candidates(eps, off, float_hi);
    }
    if (by == 1) {
        const float floor_lo = cut * (2.f - FLOOR_EPS), floor_hi = cut * FLOOR_EPS;
        const unsigned lo = __float_as_uint(floor_lo);
        width = __float_as_uint(floor_hi) + 1 - lo;
        f = sh.mb > 4 ? floor_pass<true>(B, sh, lo, floor_hi) : floor_pass<false>(B, sh, lo, floor_hi);
        by += candidates(FLOOR_EPS, 0.f, floor_hi);
    }
    const unsigned x = lane & 7u, yl = lane >> 3;
    unsigned np = f.np;
    if (by == 2) {
        const KeyPass k = key_pass(B, sh, d.cut);
        np = k.np;
#pragma unroll
        for (unsigned j = 0; j < 2; ++j)
            cand[j] = __ballot_sync(FULL_MASK, k.ok[j]);
    } else if (__any_sync(FULL_MASK, f.near_cut < width)) {   // count in whole numbers
        np = 0;
        for (unsigned j = 0; j < 2; ++j) {
            const unsigned y = yl + 4 * j;
            if (x >= sh.ma || y >= sh.mb)
                continue;
            const int4 pab = add4(B.A[0][x], B.A[1][y]);
            for (unsigned z = 0; z < sh.mc; ++z) {
                const int4 p = add4(pab, B.A[2][z]);
                for (unsigned w = 0; w < sh.me; ++w) {
                    bool pass;
                    box_key(add4(p, B.A[3][w]), d.cut, pass);
                    np += pass;
                }
            }
        }
    }
    npass += (unsigned long long)np * sh.ne;

    // the candidates, one after the other; lane i keeps survivors i and i + 32
    unsigned n_surv = 0;
    unsigned long long mine[2] = {NO_KEY, NO_KEY};
    const unsigned u = lane >> 3, v = lane & 7u;   // the lane's two hits of a table: u, u + 4 and v
    const unsigned long long kb = (unsigned long long)(min(d.cut, 1ll << 38) + 1) << 23;   // chi2 <= cut iff key < kb
    for (unsigned j = 0; j < 2; ++j)
        for (unsigned bits = cand[j]; bits; bits &= bits - 1) {
            const unsigned src = __ffs(bits) - 1, cx = src & 7u, cy = (src >> 3) + 4 * j;
            const auto key_of = [](const int4 &p, const int4 &q) {   // without the cut
                const int4 s = add4(p, q);
                return box_key_raw(s, (unsigned)s.w);
            };
            const int4 a = B.A[0][cx], b = B.A[1][cy], ev = B.A[3][v];
            // the pair's lowest fit and its hits
            const unsigned long long k0 = key_of(add4(a, b), add4(B.A[2][u], ev)),
                                     k4 = key_of(add4(a, b), add4(B.A[2][u + 4], ev));
            const bool in = u < sh.mc & v < sh.me, in4 = u + 4 < sh.mc & v < sh.me;
            const unsigned long long kf = warp_min_key(umin64(in ? k0 : NO_KEY, in4 ? k4 : NO_KEY));
            if (kf >= kb)
                continue;   // it does not pass
            const unsigned at4 = __ballot_sync(FULL_MASK, in4 & (k4 == kf)),
                           at = at4 | __ballot_sync(FULL_MASK, in & (k0 == kf));   // (keys differ by comb: one lane)
            const unsigned cz = ((__ffs(at) - 1) >> 3) + (at4 ? 4u : 0u), cw = (__ffs(at) - 1) & 7u;
            // tables (a, c) and (b, c), two fits of each per lane, then the others
            const int4 c = B.A[2][cz], e = B.A[3][cw];
            bool kill = false;
#pragma unroll
            for (unsigned i = 0; i < 8; i += 4) {
                const unsigned w = u + i;
                kill |= w < sh.mb & v < sh.me & key_of(add4(a, c), add4(B.A[1][w], ev)) < kf;
                kill |= w < sh.ma & v < sh.me & key_of(add4(b, c), add4(B.A[0][w], ev)) < kf;
            }
            if (__any_sync(FULL_MASK, kill))
                continue;
            const int4 cv = B.A[2][v], av = B.A[0][v];
#pragma unroll
            for (unsigned i = 0; i < 8; i += 4) {
                const unsigned w = u + i;
                kill |= w < sh.mb & v < sh.mc & key_of(add4(a, e), add4(B.A[1][w], cv)) < kf;
                kill |= w < sh.ma & v < sh.mc & key_of(add4(b, e), add4(B.A[0][w], cv)) < kf;
                kill |= w < sh.mb & v < sh.ma & key_of(add4(c, e), add4(B.A[1][w], av)) < kf;
            }
            if (__any_sync(FULL_MASK, kill))
                continue;
            if (lane == (n_surv & 31u))
                mine[0] = n_surv < 32 ? kf : mine[0], mine[1] = n_surv < 32 ? mine[1] : kf;
            ++n_surv;
        }
    // in comb order
    unsigned rank[2] = {0u, 0u};
    for (unsigned i = 0; i < n_surv; ++i) {
        const unsigned other = (unsigned)__shfl_sync(FULL_MASK, i < 32 ? mine[0] : mine[1], i & 31u) & 0x7FFFu;
        rank[0] += other < ((unsigned)mine[0] & 0x7FFFu);
        rank[1] += other < ((unsigned)mine[1] & 0x7FFFu);
    }
#pragma unroll
    for (unsigned i = 0; i < 2; ++i)
        if (lane + 32 * i < n_surv)
            d.surv_pool[surv_at(d, g, rank[i])] = mine[i];
    if (lane == 0) {
        d.surv_cnt[g] = (uint8_t)n_surv;
        if (n_surv)
            atomicAdd(&d.rchunk_sum[g / ROAD_CHUNK], n_surv);
    }
    if ((pk >> 23) & 1u)   // a cross-road candidate
        publish_road(d, g, rec);
    __syncwarp();
}

// The road-local hit-warrior of the plain pipeline for a listed road, by one warp
// from the keys the fit kernel stored.
__device__ __noinline__ void box_plain(const Dev &d, unsigned char *region, unsigned g)
{
    P3Box &B = *reinterpret_cast<P3Box *>(region);
    const unsigned lane = lane_id();
    const RoadRec rec = ldcg(d.roads + g);
    const uint32_t pk = rec.pk;
    const unsigned excl = min((pk >> 20) & 7u, 4u);
    __syncwarp();   // the region's previous user is done
    if (lane < N_LAYERS)   // 80 bytes of coordinates, five 16-byte words
        reinterpret_cast<uint4 *>(B.co)[lane] = ldcg(reinterpret_cast<const uint4 *>(d.coords + (size_t)g * 40) + lane);
    __syncwarp();

    // lane 8 j + h: raw hit h of fitted slot j.  Canonical hits, their ranks
    // and comb parts.
    const unsigned j = lane >> 3, h = lane & 7u;
    const unsigned L = j + (j >= excl);
    const unsigned nj = hits_of(pk, L);
    const bool valid = h < nj;
    unsigned cls = h;   // the lowest index with the same coordinate
    if (valid) {
        const unsigned v = B.co[L * 8 + h];
        for (unsigned x = h; x-- > 0;)
            cls = B.co[L * 8 + x] == v ? x : cls;
    }
    const bool canon = valid && cls == h;
    const unsigned cm = __ballot_sync(FULL_MASK, canon);
    const unsigned mine = (cm >> (8 * j)) & 0xFFu;
    const unsigned k = __popc(mine & ((1u << h) - 1u));
    if (valid)
        B.rank[j][h] = (uint8_t)__popc(mine & ((1u << cls) - 1u));
    BoxShape sh;
    sh.mpk = 0;
#pragma unroll
    for (unsigned s = 0; s < 4; ++s)
        sh.mpk |= (unsigned)__popc((cm >> (8 * s)) & 0xFFu) << (4 * s);
    sh.ne = hits_of(pk, excl);
    sh.cb = ldcg(d.comb_off + g);
    if (canon) {
        unsigned SL = 1;   // comb stride of layer L
        for (unsigned l = 0; l < L; ++l)
            SL *= hits_of(pk, l);
        B.A[j][k] = make_int4(0, 0, 0, (int)(h * SL));
    }
    for (unsigned i = lane; i < 4 * 8 * TS; i += 32)
        (&B.T[0][0])[i] = NO_KEY;
    for (unsigned i = lane; i < 2 * 2 * 2 * 8 * TS; i += 32)   // H and L
        (&B.H[0][0][0])[i] = 0xFFFFFFFFu;
    // roles: the pair (a, b) that needs the fewest lane steps, then c before
    // e with e (the unrolled inner loop) the larger
    {
        const unsigned n4 = sh.m(0) * sh.m(1) * sh.m(2) * sh.m(3);
        unsigned best = ~0u, ba = 0, bb = 1;
#pragma unroll
        for (unsigned q = 0; q < 6; ++q) {
            const unsigned pa = pair_a(q), pb = pair_b(q);
            const unsigned prod = sh.m(pa) * sh.m(pb);
            const unsigned cost = (prod + 31) / 32 * (n4 / prod);
            if (cost < best) {
                best = cost;
                ba = pa;
                bb = pb;
            }
        }
        const unsigned rest = 0xFu & ~(1u << ba) & ~(1u << bb);
        const unsigned r0 = __ffs(rest) - 1, r1 = 31 - __clz(rest);
        const bool sw = sh.m(r0) > sh.m(r1);
        sh.ra = ba;
        sh.rb = bb;
        sh.rc = sw ? r1 : r0;
        sh.re = sw ? r0 : r1;
        sh.ma = sh.m(sh.ra);
        sh.mb = sh.m(sh.rb);
        sh.mc = sh.m(sh.rc);
        sh.me = sh.m(sh.re);
    }
    __syncwarp();

    // the loop over the box: every table but T_ce
    const unsigned ma = sh.ma, mb = sh.mb, me = sh.me;
    const unsigned passes = (ma * mb + 31) / 32;   // 1 or 2
    // full passes and all eight hits of slot e (every 8^4 road): no per-step predicate
    const bool fullw = (ma * mb) % 32 == 0 && me == 8;
    for (unsigned p = 0; p < passes; ++p) {
        if (fullw)
            box_pass<8, true>(d, B, sh, p);
        else if (me > 4)
            box_pass<8, false>(d, B, sh, p);
        else
            box_pass<4, false>(d, B, sh, p);
    }
    __syncwarp();

    // road-local survivors: the minimum of pair (x, y) survives iff it is
    // also the minimum of its other five tables; T_ce (the minimum over all
    // pairs at its hits of slots c and e) is taken last, for the pairs that
    // pass the other four, by the whole warp
    unsigned long long sk[2] = {NO_KEY, NO_KEY};
    bool sv[2] = {false, false};
    unsigned zw[2] = {0u, 0u};
#pragma unroll
    for (unsigned p = 0; p < 2; ++p) {
        const unsigned t = p * 32 + lane;
        if (p < passes && t < ma * mb) {
            const unsigned y = divm(t, c_magic[ma]), x = t - y * ma;
            const unsigned long long key = B.T[T_AB][x * TS + y];
            if (key != NO_KEY) {
                // raw hits of the layers of slots c and e from the comb
                unsigned rest = (unsigned)(key & 0x7FFFu), dc = 0, de = 0;
                const unsigned Lc = sh.rc + (sh.rc >= excl), Le = sh.re + (sh.re >= excl);
#pragma unroll
                for (unsigned l = 0; l < N_LAYERS; ++l) {
                    const unsigned n = max(hits_of(pk, l), 1u);
                    const unsigned q = divm(rest, c_magic[n]);
                    const unsigned dl = rest - q * n;
                    rest = q;
                    dc = l == Lc ? dl : dc;
                    de = l == Le ? dl : de;
                }
                const unsigned z = B.rank[sh.rc][dc], w = B.rank[sh.re][de];
                sv[p] = box_get(B, T_AC, x * TS + z) == key && box_get(B, T_BC, y * TS + z) == key;
                sk[p] = key;
                zw[p] = x | (y << 3) | (z << 6) | (w << 9);
            }
        }
    }
#pragma unroll
    for (unsigned p = 0; p < 2; ++p) {
        for (unsigned bits = __ballot_sync(FULL_MASK, sv[p]); bits; bits &= bits - 1) {
            const unsigned src = __ffs(bits) - 1;
            const unsigned e = __shfl_sync(FULL_MASK, zw[p], src);
            const unsigned long long key = __shfl_sync(FULL_MASK, sk[p], src);
            const unsigned x = e & 7u, y = (e >> 3) & 7u, z = (e >> 6) & 7u, w = e >> 9;
            // T_ae, T_be, T_ce of the candidate, on demand (each one only if
            // the ones before hold the key)
            bool ok = box_min2(d, B, sh, sh.ra, x, sh.re, w) == key;
            ok = ok && box_min2(d, B, sh, sh.rb, y, sh.re, w) == key;
            ok = ok && box_tce(d, B, sh, z, w) == key;
            if (lane == src)
                sv[p] = ok;
        }
    }
    // survivors in comb order: each finds its rank among the others
    const unsigned s0 = __ballot_sync(FULL_MASK, sv[0]), s1 = __ballot_sync(FULL_MASK, sv[1]);
    const unsigned n_surv = __popc(s0) + __popc(s1);
    unsigned rk[2] = {0u, 0u};
    const unsigned my0 = (unsigned)(sk[0] & 0x7FFFu), my1 = (unsigned)(sk[1] & 0x7FFFu);
    for (unsigned q = 0; q < 2; ++q) {
        for (unsigned bits = q ? s1 : s0; bits; bits &= bits - 1) {
            const unsigned src = __ffs(bits) - 1;
            const unsigned other = __shfl_sync(FULL_MASK, q ? my1 : my0, src);
            rk[0] += other < my0;
            rk[1] += other < my1;
        }
    }
#pragma unroll
    for (unsigned p = 0; p < 2; ++p)
        if (sv[p])
            d.surv_pool[surv_at(d, g, rk[p])] = sk[p];
    if (lane == 0) {
        d.surv_cnt[g] = (uint8_t)n_surv;
        if (n_surv)
            atomicAdd(&d.rchunk_sum[g / ROAD_CHUNK], n_surv);
    }

    // cross-road candidates: the minimum key of every group (layer triple,
    // three coordinates) whose three hits are canonical and flagged as
    // present in another road of the event
    if ((pk >> 23) & 1u) {
        // canonical hits of the excluded layer (lanes 0..7)
        unsigned xc = lane;
        const bool xv = lane < sh.ne;
        if (xv) {
            const unsigned v = B.co[excl * 8 + lane];
            for (unsigned x = lane; x-- > 0;)
                xc = B.co[excl * 8 + x] == v ? x : xc;
        }
        const unsigned cmx = __ballot_sync(FULL_MASK, xv && xc == lane) & 0xFFu;
        const unsigned long long xm = ldcg(d.xmask + g);
        const unsigned event = rec.event;
        unsigned fresh = 0;   // slots claimed
        unsigned long long flp = 0;
#pragma unroll
        for (unsigned l = 0; l < N_LAYERS; ++l) {
            const unsigned cl = l == excl ? cmx : (cm >> (8 * (l - (l > excl)))) & 0xFFu;
            flp |= (unsigned long long)((unsigned)(xm >> (8 * l)) & cl) << (8 * l);
        }
        const auto fl = [flp](unsigned l) { return (unsigned)(flp >> (8 * l)) & 0xFFu; };
        const auto groups = [&fl](unsigned t) {
            return __popc(fl(triple_l(t, 0))) * __popc(fl(triple_l(t, 1))) * __popc(fl(triple_l(t, 2)));
        };
        unsigned total = 0;
#pragma unroll
        for (unsigned t = 0; t < 10; ++t)
            total += groups(t);
        {   // the entries of the tables the passes do not fold (T_ae, T_be,
            // T_ce) that groups of (excluded layer, slot p, slot e) read
            if (fl(excl)) {
                const unsigned Le = sh.re + (sh.re >= excl), fe = fl(Le);
#pragma unroll
                for (unsigned q = 0; q < 3; ++q) {
                    const unsigned sp = q == 0 ? sh.ra : q == 1 ? sh.rb : sh.rc;
                    const unsigned Lp = sp + (sp >= excl);
                    for (unsigned bp = fl(Lp); bp; bp &= bp - 1)
                        for (unsigned be = fe; be; be &= be - 1) {
                            const unsigned kp = B.rank[sp][__ffs(bp) - 1], w = B.rank[sh.re][__ffs(be) - 1];
                            const unsigned long long m = box_min2(d, B, sh, sp, kp, sh.re, w);
                            if (lane == 0) {
                                B.T[q == 0 ? T_AE : q == 1 ? T_BE : T_CE][kp * TS + w] = m;
                            }
                        }
                }
            }
            __syncwarp();
        }
        unsigned Se = 1;   // comb stride of the excluded layer
        for (unsigned l = 0; l < excl; ++l)
            Se *= hits_of(pk, l);
        for (unsigned gi = lane; gi < total; gi += 32) {
            unsigned t = 0, rem = gi;
            bool found = false;
#pragma unroll
            for (unsigned tt = 0; tt < 10; ++tt) {
                const unsigned c = groups(tt);
                if (!found) {
                    if (rem < c) {
                        t = tt;
                        found = true;
                    } else {
                        rem -= c;
                    }
                }
            }
            const unsigned lt[3] = {triple_l(t, 0), triple_l(t, 1), triple_l(t, 2)};
            const unsigned f0 = fl(lt[0]), f1 = fl(lt[1]), f2 = fl(lt[2]);
            const unsigned p0 = __popc(f0), p1 = __popc(f1);
            const unsigned dsel[3] = {nth_bit(f0, rem % p0), nth_bit(f1, (rem / p0) % p1),
                                      nth_bit(f2, rem / (p0 * p1))};
            unsigned long long mn = NO_KEY;
            if (lt[0] != excl && lt[1] != excl && lt[2] != excl) {
                // three fitted slots fixed; the fourth runs over its canonical hits
                int base = 0;
                unsigned free_slot = 0 + 1 + 2 + 3;
#pragma unroll
                for (unsigned q = 0; q < 3; ++q) {
                    const unsigned s = lt[q] - (lt[q] > excl);
                    free_slot -= s;
                    base += B.A[s][B.rank[s][dsel[q]]].w;
                }
                for (unsigned z = 0; z < sh.m(free_slot); ++z) {
                    mn = umin64(mn, ldcg(d.fit_key + sh.cb + (unsigned)(base + B.A[free_slot][z].w)));
                }
            } else {
                // the excluded layer in the triple: the pair table of the two
                // fitted slots, then the excluded hit's comb
                unsigned de = 0, sa = 4, sb = 4, da = 0, db = 0;
#pragma unroll
                for (unsigned q = 0; q < 3; ++q) {
                    if (lt[q] == excl) {
                        de = dsel[q];
                    } else if (sa == 4) {
                        sa = lt[q] - (lt[q] > excl);
                        da = dsel[q];
                    } else {
                        sb = lt[q] - (lt[q] > excl);
                        db = dsel[q];
                    }
                }
                unsigned idx;
                const unsigned tab = box_tab(sh, sa, B.rank[sa][da], sb, B.rank[sb][db], idx);
                mn = box_get(B, tab, idx);
                if (mn != NO_KEY)
                    mn += (unsigned long long)de * Se;
            }
            if (mn != NO_KEY)
                fresh += hash_min(d, group_key(event, t, B.co[lt[0] * 8 + dsel[0]], B.co[lt[1] * 8 + dsel[1]],
                                      B.co[lt[2] * 8 + dsel[2]]),
                         mn);
        }
        hash_count(d, fresh);
    }
    __syncwarp();
}

template <bool PLAIN>
__device__ __forceinline__ void box_road(const Dev &d, unsigned char *region, unsigned g, unsigned long long &npass)
{
    if (PLAIN)
        box_plain(d, region, g);
    else
        box_warp(d, region, g, npass);
}

// Shared memory of P3: what every step reads of the kernel's argument (a load
// through the argument's address takes an L1 miss), then a region per warp, a
// group step's hits or a box road.
struct P3Shared {
    const uint16_t *coords;
    const int4 *fitc;
    unsigned long long *surv_pool;
    uint8_t *surv_cnt;
    uint32_t *rchunk_sum;
    long long cut;
    size_t max_roads;
    unsigned sh;                       // the shift of the 32-bit words
    unsigned n[2 * N_GROUP_CLS];       // roads of each half class
    unsigned end[2 * N_GROUP_CLS];     // steps up to and with each half class
};
constexpr size_t P3_SHARED_BYTES = (sizeof(P3Shared) + 15) / 16 * 16;
constexpr size_t P3_WARP_BYTES = ((sizeof(P3Box) > sizeof(P3Group) ? sizeof(P3Box) : sizeof(P3Group)) + 15) / 16 * 16;

// The classes' shapes (lanes of slot a, of slot b, hits of b per lane, hits of
// e).  Most roads of classes 2 and 4 have two hits at most in slot e: they
// take a loop of half the length.
using GroupCls0 = GroupRoad<1, 0, 2, 2>;    // (2, 2) hits: 16 roads a step
using GroupCls1 = GroupRoad<2, 0, 2, 2>;    // (4, 2): 8
using GroupCls2 = GroupRoad<2, 1, 2, 2>;    // (4, 4): 4
using GroupCls2e = GroupRoad<2, 1, 2, 4>;   // and more than two hits in slot e
using GroupCls3 = GroupRoad<3, 0, 2, 2>;    // (8, 2): 4
using GroupCls4 = GroupRoad<3, 1, 2, 2>;    // (8, 4): 2
using GroupCls4e = GroupRoad<3, 1, 2, 4>;

// Fit up to ROADS roads of a list (list[0], list[step], .., `left` of them) with
// one warp; adds the lane's passing combinations to np.  Returns the roads with
// a tie, bit by lane of their groups' first lanes.  EXACT: those roads (`tied`)
// again, in whole keys, straight after the call that found them.  Not inlined: a
// register allocation per class (in one function the five classes spilled 220
// bytes).  Bound: issue slots and the chain from the list to the hits.  The fit
// stage of 192,000 roads of one to four hits a layer, nearly all of them here:
// 124.4 -> 61.7 us (a lane per table entry, tables in shared memory, before).  At
// 80 registers the shapes with four hits of slot e spill 30 bytes (64 in whole
// keys), p3_phase and p3_boxes some 70 outside their items.
template <bool PLAIN, class Road, bool EXACT>
__device__ __noinline__ unsigned group_item(const Dev &d, unsigned char *smem, const RoadItem *list, int step,
                                            unsigned left, unsigned tied, unsigned &npass)
{
    using Key = typename FitKey<EXACT>::type;
    constexpr Key FAIL = FitKey<EXACT>::FAIL;
    const P3Shared &S = *reinterpret_cast<const P3Shared *>(smem);
    const unsigned sh = S.sh;
    constexpr unsigned A = Road::A, YN = Road::YN, B = Road::B, W = Road::W, G = Road::G, HITS = Road::HITS;
    const unsigned lane = lane_id(), gl = lane % G, gi = lane / G;
    const unsigned gmask = G == 32 ? FULL_MASK : ((1u << (G & 31u)) - 1u) << (gi * G);
    Road r;
    const bool on = EXACT ? (tied >> (gi * G)) & 1u : gi < left;
    r.it = RoadItem{};
    if (on) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(list + step * (int)gi));
        memcpy(&r.it, &v, sizeof v);
    }
    const uint32_t pk = r.it.pk;
    const size_t g = r.it.g;
    r.excl = min((pk >> 20) & 7u, 4u);
    r.nf = fitted_counts(pk);   // no road: no hits
    r.mb = r.m(r.slot(1));
    r.mc = r.m(r.slot(2));
    r.me = r.m(r.slot(3));
    r.x = gl % A;
    r.yl = gl / A;
    r.live = r.x < r.m(r.slot(0));
    r.cb = PLAIN && on ? ldcg(d.comb_off + g) : 0ull;
    int4 *hit = reinterpret_cast<P3Group *>(smem + P3_SHARED_BYTES + warp_id() * P3_WARP_BYTES)->A + gi * HITS;
    r.hit = hit;
    __syncwarp();   // the table's previous readers are done
    if (!EXACT) {
        // comb strides of the layers
        const unsigned S1 = pk & 15u, S2 = S1 * ((pk >> 4) & 15u), S3 = S2 * ((pk >> 8) & 15u),
                       S4 = S3 * ((pk >> 12) & 15u);
        // The road's hits, N per lane.  Every load is issued before the first
        // is used, without a branch (a missing hit reads its row's slot, whose
        // value is not used): one wait for L2 instead of one per round.
        constexpr unsigned N = (HITS + G - 1) / G;
        unsigned at[N];   // slot | k << 4, and bit 31: the hit exists
        int v[N];
        int4 cj[N];
        const int4 *cc = S.fitc + SET_INT4 * min((unsigned)r.it.set, (unsigned)(N_SETS - 1)) + SET_C;
        const uint16_t *row = S.coords + g * 40;
#pragma unroll
        for (unsigned i = 0; i < N; ++i) {
            const unsigned h = i * G + gl;
            const unsigned role = h < A ? 0u : h < A + B ? 1u : h < A + 2 * B ? 2u : 3u;
            const unsigned k = (h - (role == 0 ? 0u : A + (role - 1) * B)) & 7u, s = r.slot(role);
            at[i] = s | k << 4 | (k < r.m(s) && h < HITS ? 0x80000000u : 0u);
            v[i] = ldcg(row + (s + (s >= r.excl)) * 8 + k);
            if (!PLAIN)
                cj[i] = __ldg(cc + s);
        }
        int4 c4, c5, kk;
        if (!PLAIN) {
            c4 = __ldg(cc + 4);
            c5 = __ldg(cc + 5);
            kk = __ldg(cc + 6);
        }
#pragma unroll
        for (unsigned i = 0; i < N; ++i) {
            const unsigned s = at[i] & 15u, k = (at[i] >> 4) & 7u, L = s + (s >= r.excl);
            const unsigned S = L == 0 ? 1u : L == 1 ? S1 : L == 2 ? S2 : L == 3 ? S3 : S4;
            int4 a = make_int4(0, 0, 0, (int)(k * S));
            if (!PLAIN) {
                a.x = cj[i].x * v[i];
                a.y = cj[i].y * v[i];
                a.z = cj[i].z * v[i];
                if (i * G < A) {   // role a: curvature, phi, 4096 * offset and the road bits
                    const bool ra = i * G + gl < A;
                    const int curv = ra ? r.it.curv : 0, phi = ra ? r.it.phi : 0, off = ra ? 4096 : 0;
                    a.x += c4.x * curv + c5.x * phi + kk.x * off;
                    a.y += c4.y * curv + c5.y * phi + kk.y * off;
                    a.z += c4.z * curv + c5.z * phi + kk.z * off;
                    a.w += ra ? (int)((pk >> 24) << 15) : 0;
                }
            }
            if (at[i] >> 31)
                hit[i * G + gl] = a;
        }
    }
    __syncwarp();

    // The lane's fits.  A failing or missing fit's word is its own, above
    // every passing one's, so that two equal words are always two passing fits.
    // (Whole keys of passing fits differ by comb; the others are all NO_KEY.)
    const unsigned mcw = __reduce_max_sync(FULL_MASK, r.mc), mew = __reduce_max_sync(FULL_MASK, r.me);
    const long long cut = S.cut;
    int4 pab[YN];
    Key q[YN], cw[YN][W];   // a pair's lowest fit; minima over z
    unsigned code[YN], np = 0;   // the lowest fit's hits and state
    bool tie = false, tie2 = false, tie3 = false, tie4 = false;   // (several: no long chain of one flag)
    const auto meet = [](bool &tie, Key t, Key u) {
        if (!EXACT)
            tie = tie | (u == t);
        return u < t ? u : t;
    };
    // minimum of t over the lanes that differ in bits [o0, o1) of the lane
    const auto fold = [&meet](bool &tie, Key t, unsigned o0, unsigned o1) {
#pragma unroll
        for (unsigned o = o0; o < o1; o <<= 1)
            t = meet(tie, t, __shfl_xor_sync(FULL_MASK, t, o));
        return t;
    };
#pragma unroll
    for (unsigned j = 0; j < YN; ++j) {
        pab[j] = add4(hit[r.x], hit[A + r.y(j)]);   // unspecified unless the hits exist
        q[j] = EXACT ? FAIL : (Key)(0xE0000000u | (lane << 8) | j);
        code[j] = 0;
#pragma unroll
        for (unsigned w = 0; w < W; ++w)
            cw[j][w] = EXACT ? FAIL : (Key)(0xC0000000u | (lane << 8) | (j * W + w));
    }
    for (unsigned z = 0; z < mcw; ++z) {
        const int4 az = hit[A + B + z];
        const unsigned none = 0x80000000u | (lane << 8) | (z << 4);
        Key word[YN][W], rz[YN], ce[W];
#pragma unroll
        for (unsigned w = 0; w < W; ++w) {
            if (w >= 2 && w >= mew) {   // no road of the warp has hit w
                ce[w] = 0;
                continue;
            }
            const int4 aw = hit[A + 2 * B + w];
            const bool zw = r.live & (z < r.mc) & (w < r.me);
#pragma unroll
            for (unsigned j = 0; j < YN; ++j) {
                const bool in = zw & (r.y(j) < r.mb);
                if (EXACT) {
                    word[j][w] = in ? r.template key<PLAIN>(d, cut, add4(pab[j], add4(az, aw))) : FAIL;
                } else if (PLAIN) {
                    const unsigned long long k =
                        in ? ldcg(d.fit_key + r.cb + (unsigned)(pab[j].w + az.w + aw.w)) : NO_KEY;
                    word[j][w] = k == NO_KEY ? none + (j * W + w) : (unsigned)((k >> 23) >> sh);
                } else {
                    const long long chi2 = sq((pab[j].x + az.x + aw.x) >> 12) + sq((pab[j].y + az.y + aw.y) >> 12) +
                                           sq((pab[j].z + az.z + aw.z) >> 12);
                    const bool pass = in & (chi2 <= cut);
                    np += pass;
                    word[j][w] = pass ? (unsigned)((unsigned long long)chi2 >> sh) : none + (j * W + w);
                }
                cw[j][w] = meet(tie, cw[j][w], word[j][w]);
                rz[j] = w == 0 ? word[j][w] : meet(tie2, rz[j], word[j][w]);
            }
            // (c, e) at z, w
            ce[w] = word[0][w];
#pragma unroll
            for (unsigned j = 1; j < YN; ++j)
                ce[w] = meet(tie3, ce[w], word[j][w]);
            ce[w] = fold(tie3, ce[w], 1, G);
        }
        Key ac = rz[0];   // (a, c) at x, z
#pragma unroll
        for (unsigned j = 1; j < YN; ++j)
            ac = meet(tie4, ac, rz[j]);
        ac = fold(tie4, ac, A, G);
#pragma unroll
        for (unsigned j = 0; j < YN; ++j) {
            const Key t = min(ac, fold(tie4, rz[j], 1, A));   // and (b, c) at y, z
            bool ok = false;
            unsigned ws = 0;
#pragma unroll
            for (unsigned w = 0; w < W; ++w) {
                if (w >= 2 && w >= mew)
                    continue;
                const bool here = word[j][w] == rz[j];
                ws = here ? w : ws;
                ok = here ? ce[w] == rz[j] : ok;
            }
            if (!EXACT)
                tie2 = tie2 | (rz[j] == q[j]);
            if (rz[j] < q[j]) {
                q[j] = rz[j];
                code[j] = z << 2 | ws | (ok && t == rz[j] ? 0x80u : 0u);
            }
        }
    }

    // (a, e) and (b, e), then the survivors
    GroupFound<YN> f;
    Key te[YN];
#pragma unroll
    for (unsigned j = 0; j < YN; ++j)
        te[j] = 0;
#pragma unroll
    for (unsigned w = 0; w < W; ++w) {
        if (w >= 2 && w >= mew)
            continue;
        Key ae = cw[0][w];
#pragma unroll
        for (unsigned j = 1; j < YN; ++j)
            ae = meet(tie3, ae, cw[j][w]);
        ae = fold(tie3, ae, A, G);
#pragma unroll
        for (unsigned j = 0; j < YN; ++j) {
            const Key t = min(ae, fold(tie4, cw[j][w], 1, A));
            te[j] = (code[j] & 3u) == w ? t : te[j];
        }
    }
    const bool again = !EXACT && (__ballot_sync(FULL_MASK, tie | tie2 | tie3 | tie4) & gmask) != 0u;   // the road has a tie
    f.cnt = 0;
#pragma unroll
    for (unsigned j = 0; j < YN; ++j) {
        f.surv[j] = !again && code[j] >= 0x80u && te[j] == q[j] && q[j] < FAIL;
        f.key[j] = EXACT ? (unsigned long long)q[j] : NO_KEY;
        f.rank[j] = 0;
        f.cnt += __popc(__ballot_sync(FULL_MASK, f.surv[j]) & gmask);
    }
#pragma unroll
    for (unsigned j = 0; j < YN; ++j)
        if (!EXACT && f.surv[j])
            f.key[j] = r.template key_at<PLAIN>(d, cut, j, (code[j] >> 2) & 3u, code[j] & 3u);
    if (__any_sync(FULL_MASK, f.cnt > 1))
        group_rank(f, gmask);
#pragma unroll
    for (unsigned j = 0; j < YN; ++j)
        if (f.surv[j])
            S.surv_pool[f.rank[j] * S.max_roads + g] = f.key[j];
    if (on && gl == 0 && !again) {
        S.surv_cnt[g] = (uint8_t)f.cnt;
        if (f.cnt)
            atomicAdd(&S.rchunk_sum[g / ROAD_CHUNK], f.cnt);
    }
    if (EXACT)
        return 0;
    npass += np * ((pk >> (4 * r.excl)) & 15u);   // once per hit of the excluded layer
    return __ballot_sync(FULL_MASK, again && gl == 0);
}

// Step s (of the sequence over all half classes) if it is of half class SEG,
// and then its roads with ties.
template <bool PLAIN, class Road, unsigned SEG>
__device__ __forceinline__ void group_step(const Dev &d, unsigned char *smem, unsigned s, unsigned &np)
{
    const P3Shared &S = *reinterpret_cast<const P3Shared *>(smem);
    const unsigned first = (s - (SEG ? S.end[SEG - 1] : 0u)) * Road::ROADS, left = S.n[SEG] - first;
    const RoadItem *list = d.items + list_at(d, SEG, first);
    constexpr int dir = (SEG & 1u) ? 1 : -1;
    const unsigned tied = group_item<PLAIN, Road, false>(d, smem, list, dir, left, 0u, np);
    if (tied)
        group_item<PLAIN, Road, true>(d, smem, list, dir, left, tied, np);
}

// The roads of the box path (n_box of them), one warp each.
template <bool PLAIN>
__device__ __noinline__ void p3_boxes(const Dev &d, unsigned char *smem, unsigned n_box, int qbox,
                                      unsigned long long &npass)
{
    const unsigned n_warps = gridDim.x * WARPS, wi = warp_id() * gridDim.x + blockIdx.x;
    Share w(n_box, n_warps, 2, &d.ctrl->q[qbox]);
    unsigned i = w.first(wi), g = i < n_box ? ldcg(d.box_list + i) : 0u;
    while (i < n_box) {   // the next road is claimed and looked up ahead
        const unsigned ni = w.next(i), ng = ni < n_box ? ldcg(d.box_list + ni) : 0u;
        box_road<PLAIN>(d, smem + P3_SHARED_BYTES + warp_id() * P3_WARP_BYTES, min(g, d.max_roads - 1), npass);
        i = ni;
        g = ng;
    }
}

// P3: the roads listed in P2, the group path's first: a step is one warp's roads
// of one half class, widest first (neighbouring warp indices lie on different
// SMs); then those of the box path, one warp each, whose queue evens out the
// warps' first steps of a class (its code comes from L2 once per SM: 16 k
// cycles against 8 k later).  Each warp works in its own region of shared
// memory, so no part of P3 waits for the whole CTA.  Not inlined: the stages
// before and after it keep a register allocation of their own (inlined, the
// decode and the box path took 10 % and 3 % longer).
// cands: the batch has cross-road candidates
template <bool PLAIN>
__device__ __noinline__ void p3_phase(const Dev &d, unsigned char *smem, int qbox, int qgroup, bool cands)
{
    P3Shared &S = *reinterpret_cast<P3Shared *>(smem);
    unsigned long long npass = 0;
    const unsigned n_box = min(ldcg(&d.ctrl->n_box), d.max_roads);
    if (warp_id() == 0) {
        const unsigned lane = lane_id();
        // roads per step of the half classes: 2, 2, -, 4, 4, 4, -, 8, -, 16
        static_assert(GroupCls4e::ROADS == 2 && GroupCls4::ROADS == 2 && GroupCls3::ROADS == 4 &&
                          GroupCls2e::ROADS == 4 && GroupCls2::ROADS == 4 && GroupCls1::ROADS == 8 &&
                          GroupCls0::ROADS == 16, "roads per step");
        const unsigned per = lane < 2 ? 2u : lane < 6 ? 4u : lane < 8 ? 8u : 16u;
        const unsigned n = lane < 2 * N_GROUP_CLS ? min(ldcg(&d.ctrl->n_seg[lane]), d.max_roads) : 0u;
        unsigned inc = (n + per - 1) / per;
#pragma unroll
        for (unsigned o = 1; o < 16; o <<= 1) {
            const unsigned u = __shfl_up_sync(FULL_MASK, inc, o);
            inc += lane >= o ? u : 0u;
        }
        if (lane < 2 * N_GROUP_CLS) {
            S.n[lane] = n;
            S.end[lane] = inc;
        }
        if (lane == 0) {
            S.coords = d.coords;
            S.fitc = d.fitc;
            S.surv_pool = d.surv_pool;
            S.surv_cnt = d.surv_cnt;
            S.rchunk_sum = d.rchunk_sum;
            S.cut = d.cut;
            S.max_roads = d.max_roads;
            // the shift that brings the cut below 2^31 (a chi-square is below 2^38)
            const unsigned long long cut = min((unsigned long long)max(d.cut, 0ll), (1ull << 38) - 1);
            S.sh = cut >> 31 ? 33 - __clzll((long long)cut) : 0u;
        }
    }
    __syncthreads();
    const unsigned n_warps = gridDim.x * WARPS, wi = warp_id() * gridDim.x + blockIdx.x;
    const unsigned steps = S.end[2 * N_GROUP_CLS - 1];
    unsigned np = 0;
    // (svt_launch::run_roads)
    Share w(steps, n_warps, d.run_roads < 8 ? 1u : d.run_roads > 8 ? 3u : 2u, &d.ctrl->q[qgroup]);
    for (unsigned s = w.first(wi); s < steps; s = w.next(s)) {
        if (s < S.end[0])
            group_step<PLAIN, GroupCls4e, 0>(d, smem, s, np);
        else if (s < S.end[1])
            group_step<PLAIN, GroupCls4, 1>(d, smem, s, np);
        else if (s < S.end[3])
            group_step<PLAIN, GroupCls3, 3>(d, smem, s, np);
        else if (s < S.end[4])
            group_step<PLAIN, GroupCls2e, 4>(d, smem, s, np);
        else if (s < S.end[5])
            group_step<PLAIN, GroupCls2, 5>(d, smem, s, np);
        else if (s < S.end[7])
            group_step<PLAIN, GroupCls1, 7>(d, smem, s, np);
        else
            group_step<PLAIN, GroupCls0, 9>(d, smem, s, np);
    }
    __syncwarp();
    if (cands)
        publish_words(d);
    p3_boxes<PLAIN>(d, smem, n_box, qbox, npass);
    npass = block_sum(npass + np);
    if (!PLAIN && threadIdx.x == 0 && npass)
        atomicAdd(&d.ctrl->n_pass, npass);
}

// ---------------------------------------------------------------------------
// P4: cross-road hit-warrior and survivor counts, P5: output
// ---------------------------------------------------------------------------

__device__ unsigned cross_check(const Dev &d, unsigned g, unsigned &cnt)
{
    // everything about the road in one trip (the first survivor: unspecified
    // when there is none), then the lookups
    const RoadRec rec = ldcg(d.roads + g);
    const unsigned long long xm = ldcg(d.xmask + g);
    unsigned long long key = ldcg(d.surv_pool + surv_at(d, g, 0));
    uint4 rw[N_LAYERS];
#pragma unroll
    for (unsigned l = 0; l < N_LAYERS; ++l)
        rw[l] = ldcg(reinterpret_cast<const uint4 *>(d.coords + (size_t)g * 40) + l);
    cnt = ldcg(d.surv_cnt + g);
    if (!cnt || !((rec.pk >> 23) & 1u))
        return cnt;
    unsigned n[N_LAYERS];
#pragma unroll
    for (unsigned l = 0; l < N_LAYERS; ++l)
        n[l] = max(min((rec.pk >> (4 * l)) & 15u, (unsigned)MAX_HITS), 1u);
    unsigned kept = 0;
    for (unsigned i = 0; i < cnt; ++i) {
        if (i)
            key = ldcg(d.surv_pool + surv_at(d, g, i));
        unsigned t = (unsigned)(key & 0x7FFFu);
        unsigned dl[N_LAYERS], v[N_LAYERS];
#pragma unroll
        for (unsigned l = 0; l < N_LAYERS; ++l) {   // mixed-radix digits of comb
            const unsigned q = divm(t, c_magic[n[l]]);
            dl[l] = t - q * n[l];
            t = q;
            v[l] = row_at(rw[l], dl[l]);
        }
        bool dropped = false;
#pragma unroll
        for (unsigned t = 0; t < 10; ++t) {
            if (dropped)
                break;
            const unsigned l0 = triple_l(t, 0), l1 = triple_l(t, 1), l2 = triple_l(t, 2);
            bool flagged = ((xm >> (8 * l0 + dl[l0])) & 1ull) && ((xm >> (8 * l1 + dl[l1])) & 1ull) &&
                           ((xm >> (8 * l2 + dl[l2])) & 1ull);
            if (flagged && hash_get(d, group_key(rec.event, t, v[l0], v[l1], v[l2])) < key)
                dropped = true;
        }
        if (!dropped)
            d.surv_pool[surv_at(d, g, kept++)] = key;
    }
    return kept;
}

__device__ void p4_item(const Dev &d, unsigned c, unsigned n_roads)
{
    unsigned g = c * ROAD_CHUNK + threadIdx.x;
    unsigned cnt = 0;
    if (g < n_roads) {
        const unsigned kept = cross_check(d, g, cnt);
        if (kept != cnt)
            d.surv_cnt[g] = (uint8_t)(cnt = kept);
    }
    unsigned long long tot = block_sum(cnt);
    if (threadIdx.x == 0)
        d.rchunk_sum[c] = (uint32_t)tot;
}

__device__ void p4_finish(const Dev &d, unsigned n_chunks)
{
    unsigned long long total = block_scan_array(d.rchunk_sum, d.rchunk_off, n_chunks);
    if (threadIdx.x == 0) {
        d.ctrl->n_out = total;
        if (total > d.max_tracks)
            raise_flag(d, FLAG_CAPACITY);
        __threadfence();
    }
}

// The track of key `key` of road g (record rec, coordinate row rw: the
// road's 40 coordinates as five 16-byte words), written to *out.
// The loops are unrolled (registers, no local arrays).
template <bool PLAIN>
__device__ void build_track(const Dev &d, unsigned g, const RoadRec &rec, const uint4 (&rw)[N_LAYERS],
                            unsigned long long key, svt_track *out)
{
    int F[3][6], q[3];
    if (!PLAIN) {   // six 16-byte loads of the set's F and q
        const int4 *fc = d.fitc + SET_INT4 * min((unsigned)rec.set, (unsigned)(N_SETS - 1));
        int4 v[6];
#pragma unroll
        for (unsigned i = 0; i < 6; ++i)
            v[i] = __ldg(fc + i);
        const int f[24] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w,
                           v[2].x, v[2].y, v[2].z, v[2].w, v[3].x, v[3].y, v[3].z, v[3].w,
                           v[4].x, v[4].y, v[4].z, v[4].w, v[5].x, v[5].y, v[5].z, v[5].w};
#pragma unroll
        for (unsigned k = 0; k < 3; ++k) {
#pragma unroll
            for (unsigned jj = 0; jj < 6; ++jj)
                F[k][jj] = f[6 * k + jj];
            q[k] = f[18 + k];
        }
    }
    const unsigned excl = min((rec.pk >> 20) & 7u, 4u);
    const unsigned comb = (unsigned)(key & 0x7FFFu);
    unsigned v[N_LAYERS];
    unsigned rest = comb;
#pragma unroll
    for (unsigned l = 0; l < N_LAYERS; ++l) {   // mixed-radix digits of comb
        const unsigned n = max(min((rec.pk >> (4 * l)) & 15u, (unsigned)MAX_HITS), 1u);
        const unsigned qq = divm(rest, c_magic[n]);
        const unsigned dl = rest - qq * n;
        rest = qq;
        v[l] = row_at(rw[l], dl);
    }
    svt_track t;
    t.event = rec.event;
    t.road = (uint16_t)(rec.pk >> 24);
    t.comb = (uint16_t)comb;
    t.pad = 0;
    t.chi2 = (long long)(key >> 23);
    unsigned long long hits = 0;
#pragma unroll
    for (unsigned l = 0; l < N_LAYERS; ++l)
        hits |= (unsigned long long)v[l] << (12 * l);
    t.hits = hits;
    if (PLAIN) {
        const unsigned long long ci = ldcg(d.comb_off + g) + comb;
        t.p[0] = ldcg(d.fit_p + 3 * ci);
        t.p[1] = ldcg(d.fit_p + 3 * ci + 1);
        t.p[2] = ldcg(d.fit_p + 3 * ci + 2);
    } else {
        // the fit's inputs: the four layers other than excl, in order, then
        // curvature and phi
        const int x[6] = {(int)(excl == 0 ? v[1] : v[0]), (int)(excl <= 1 ? v[2] : v[1]),
                          (int)(excl <= 2 ? v[3] : v[2]), (int)(excl <= 3 ? v[4] : v[3]), rec.curv, rec.phi};
#pragma unroll
        for (unsigned k = 0; k < 3; ++k) {
            int acc = 0;
#pragma unroll
            for (unsigned jj = 0; jj < 6; ++jj)
                acc += F[k][jj] * x[jj];
            t.p[k] = (acc >> 12) + q[k];
        }
    }
    *out = t;
}

// Track of survivor idx of road g, written to output slot pos: the road's
// record, the key and the coordinate row go out together (none depends on
// another).
template <bool PLAIN>
__device__ void emit_track(const Dev &d, unsigned g, unsigned idx, unsigned long long pos)
{
    static_assert(sizeof(uint16_t) * 40 == N_LAYERS * sizeof(uint4), "a coordinate row is five 16-byte words");
    const RoadRec rec = ldcg(d.roads + g);
    const unsigned long long key = ldcg(d.surv_pool + surv_at(d, g, idx));
    const uint4 *row = reinterpret_cast<const uint4 *>(d.coords + (size_t)g * 40);
    uint4 rw[N_LAYERS];
#pragma unroll
    for (unsigned l = 0; l < N_LAYERS; ++l)
        rw[l] = ldcg(row + l);
    if (pos < d.max_tracks)
        build_track<PLAIN>(d, g, rec, rw, key, d.tracks + pos);
}

// road of survivor i of a chunk: the last r with s_first[r] <= i (a road
// with survivors; s_first holds the chunk's exclusive scan of counts)
__device__ __forceinline__ unsigned chunk_road(const unsigned *s_first, unsigned i)
{
    unsigned lo = 0, hi = ROAD_CHUNK;
    while (hi - lo > 1) {
        const unsigned mid = (lo + hi) >> 1;
        if (s_first[mid] <= i)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

#if SVT_BLOCK == 256   // the plain pipeline's output stage
// Output of one chunk of ROAD_CHUNK roads (plain kernels): a block scan of
// the survivor counts gives each road's first output slot; then each thread
// takes survivors (not roads), so roads with many survivors are spread out.
template <bool PLAIN>
__device__ void p5_item(const Dev &d, unsigned c, unsigned n_roads, unsigned *s_first)
{
    // s_first: ROAD_CHUNK + 1 shared words, the first survivor of each road
    static_assert(ROAD_CHUNK == BLOCK, "one thread per road of a chunk");
    const unsigned g_me = c * ROAD_CHUNK + threadIdx.x;
    const unsigned cnt_me = g_me < n_roads ? ldcg(d.surv_cnt + g_me) : 0u;
    unsigned long long total;
    const unsigned ex = (unsigned)block_excl_scan(cnt_me, &total);
    s_first[threadIdx.x] = ex;
    if (threadIdx.x == 0)
        s_first[ROAD_CHUNK] = (unsigned)total;
    const unsigned long long base = ldcg(d.rchunk_off + c);
    __syncthreads();
    for (unsigned i = threadIdx.x; i < (unsigned)total; i += BLOCK) {
        const unsigned r = chunk_road(s_first, i);
        emit_track<PLAIN>(d, c * ROAD_CHUNK + r, i - s_first[r], base + i);
    }
    __syncthreads();   // s_first is reused by the next chunk
}
#endif

// P4 of the persistent kernel: the cross-road hit-warrior over the
// candidate roads only (P2 sets their bits; the others keep their
// survivors).  One warp per word of candidate bits, one lane per road, so
// every candidate road checks its survivors at once; bit word w goes to CTA
// w % grid, so that a few candidates are spread out.  A road that loses
// survivors takes them off its chunk's total.
__device__ void p4_cand_phase(const Dev &d, unsigned n_roads)
{
    const unsigned n_words = (n_roads + 31) / 32;
    const unsigned lane = lane_id();
    for (unsigned w = warp_id() * gridDim.x + blockIdx.x; w < n_words; w += gridDim.x * WARPS) {
        const unsigned bits = ldcg(d.cand_bits + w);
        const unsigned g = w * 32 + lane;
        if (!((bits >> lane) & 1u) || g >= n_roads)
            continue;   // not a candidate, or a road of the truncated tail (not fitted)
        unsigned cnt;
        const unsigned kept = cross_check(d, g, cnt);
        if (kept != cnt) {
            d.surv_cnt[g] = (uint8_t)kept;
            atomicSub(&d.rchunk_sum[g / ROAD_CHUNK], cnt - kept);
        }
    }
}

// P5 of the persistent kernel: the tracks in road order.  Every CTA takes an
// equal share of the roads; the chunk totals and the counts before its share,
// which every CTA sums itself, give its first track's place.  A road's count,
// record, coordinate row and first key do not depend on each other: they are
// loaded together, a road per thread, and a scan of the counts places the
// tracks, which are gathered in shared memory and written out as one stretch.
// Bound: two trips to L2 and the writes (a search for the road of each of an
// equal share of the tracks took four trips and wrote each track's five words
// 40 bytes apart: 175,000 tracks 15.1 -> 10.2 us).
constexpr unsigned P5_TRACKS = 2 * BLOCK;   // tracks gathered at most (more: written by their thread)
struct P5Smem {
    svt_track track[P5_TRACKS];
};

// Thread 0 alone writes the control block here: `wrote`.
__device__ void p5_phase(const Dev &d, unsigned char *smem, unsigned n_roads, bool &wrote)
{
    wrote = false;
    P5Smem &s = *reinterpret_cast<P5Smem *>(smem);
    const unsigned n_chunks = min((n_roads + ROAD_CHUNK - 1) / ROAD_CHUNK, d.max_chunks_r);
    const unsigned lo = (unsigned)((unsigned long long)n_roads * blockIdx.x / gridDim.x);
    const unsigned hi = (unsigned)((unsigned long long)n_roads * (blockIdx.x + 1) / gridDim.x);
    const unsigned c_lo = lo / ROAD_CHUNK;
    unsigned long long all = 0, before = 0;   // survivors of the batch, and of the roads before lo
    for (unsigned c = threadIdx.x; c < n_chunks; c += BLOCK) {
        const unsigned t = ldcg(d.rchunk_sum + c);
        all += t;
        before += c < c_lo ? t : 0u;
    }
    for (unsigned g = c_lo * ROAD_CHUNK + threadIdx.x; g < lo; g += BLOCK)
        before += ldcg(d.surv_cnt + g);
    bool summed = false;
    for (unsigned r0 = lo; r0 < hi || !summed; r0 += BLOCK) {
        const unsigned g = r0 + threadIdx.x;
        unsigned cnt = 0;
        RoadRec rec{};
        unsigned long long key = 0;
        uint4 rw[N_LAYERS];
        if (g < hi) {
            cnt = ldcg(d.surv_cnt + g);
            rec = ldcg(d.roads + g);
            key = ldcg(d.surv_pool + surv_at(d, g, 0));   // (unspecified when there is none)
            const uint4 *row = reinterpret_cast<const uint4 *>(d.coords + (size_t)g * 40);
#pragma unroll
            for (unsigned l = 0; l < N_LAYERS; ++l)
                rw[l] = row[l];
        }
        if (!summed) {
            block_sum2(all, before);
            summed = true;
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                wrote = true;
                d.ctrl->n_out = all;
                if (all > d.max_tracks)
                    raise_flag(d, FLAG_CAPACITY);
            }
            if (all > d.max_tracks)
                return;
        }
        unsigned tot;
        const unsigned at = block_excl_scan32(cnt, &tot);
        const bool gather = tot <= P5_TRACKS;
        svt_track *out = gather ? s.track : d.tracks + before;
        for (unsigned i = 0; i < cnt; ++i) {
            if (i)
                key = ldcg(d.surv_pool + surv_at(d, g, i));
            if (gather || before + at + i < d.max_tracks)
                build_track<false>(d, g, rec, rw, key, out + at + i);
        }
        if (gather) {
            __syncthreads();
            static_assert(sizeof(svt_track) % 8 == 0, "whole words");
            const unsigned long long *src = reinterpret_cast<const unsigned long long *>(s.track);
            unsigned long long *dst = reinterpret_cast<unsigned long long *>(d.tracks + before);
            for (unsigned i = threadIdx.x; i < tot * (sizeof(svt_track) / 8); i += BLOCK)
                dst[i] = src[i];
            __syncthreads();
        }
        before += tot;
    }
    // the roads' counts and the chunk totals agree
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0 && before != all) {
        wrote = true;
        raise_flag(d, FLAG_INTERNAL);
    }
}

// Leave the group table empty: every claimed slot (its bit) is cleared, with
// its bit.  Run by the whole grid once every lookup is done.
__device__ void clear_hash(const Dev &d)
{
    if (ldcg(&d.ctrl->hash_used) == 0)
        return;
    const unsigned n_words = d.hash_mask / 32 + 1;
    for (unsigned w = blockIdx.x * BLOCK + threadIdx.x; w < n_words; w += gridDim.x * BLOCK) {
        unsigned bits = ldcg(d.hash_bits + w);
        if (!bits)
            continue;
        d.hash_bits[w] = 0;
        for (; bits; bits &= bits - 1) {
            const unsigned h = w * 32 + (unsigned)(__ffs(bits) - 1);
            d.hash[h].key = 0ull;
            d.hash[h].val_inv = 0ull;
        }
    }
}

// ---------------------------------------------------------------------------
// the persistent fused kernel
// ---------------------------------------------------------------------------


// The whole chain; false: it stopped early (a fault, a limit, a wait that ran out).
// wrote: as leave() takes it; true until the output stage says otherwise.
__device__ __forceinline__ bool chain(const Dev &d, bool &wrote)
{
    wrote = true;
    extern __shared__ __align__(16) unsigned char smem[];
    if (d.skip_arrival == 1 && blockIdx.x == 0)
        return false;   // test hook: this CTA never arrives at the first barrier
    stamp(d, 0);

    unsigned flags;
    Batch bt;
    scan_count(d);
    if (!grid_sync(d, 1, flags))
        return false;
    stamp(d, 1);
    if (!scan_decode(d, smem, bt))
        return false;
    if (!grid_sync(d, 2, flags))
        return false;
    stamp(d, 2);
    const bool fault = flags & FLAG_FAULT;   // a fault of the stream: no tracks
    if (!fault)
        p2_phase(d, smem, bt);
    if (!grid_sync(d, 3, flags))
        return false;
    stamp(d, 3);
    if (fault)
        return false;

    p3_phase<false>(d, smem, Q_BOX, Q_GROUP, flags & FLAG_CANDS);
    if (d.skip_arrival == 2 && blockIdx.x == 0)
        return false;   // test hook: this CTA leaves after publishing, the others' waits run out
    if (!grid_sync(d, 4, flags))
        return false;
    stamp(d, 4);

    const bool groups = flags & FLAG_GROUPS;   // no group published: nothing to look up or clear
    if (groups) {
        p4_cand_phase(d, bt.n_roads);
        if (!grid_sync(d, 5, flags))
            return false;
    }
    stamp(d, 5);
    p5_phase(d, smem, bt.n_roads, wrote);
    // every lookup is done (barrier above): leave the group table empty
    if (groups)
        clear_hash(d);
    return true;
}

__global__ void __launch_bounds__(BLOCK, BLOCK == 512 ? 2 : 768 / BLOCK) k_persistent(const __grid_constant__ Dev d)
{
    bool wrote;
    const bool finished = chain(d, wrote);
    leave(d, finished, wrote);
}

#if SVT_BLOCK == 256
// ---------------------------------------------------------------------------
// plain per-stage kernels
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(BLOCK) k_p0(Dev d) { scan_count(d); }

__global__ void __launch_bounds__(BLOCK) k_p1(Dev d)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Batch bt;
    scan_decode(d, smem, bt);
}

__global__ void __launch_bounds__(BLOCK) k_p2(Dev d)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (flags_of(d) & (FLAG_CAPACITY | FLAG_FAULT))
        return;
    Batch bt{ldcg(&d.ctrl->n_events), ldcg(&d.ctrl->n_ep), 0u};
    p2_phase(d, smem, bt);
}

__device__ __forceinline__ bool stop_after_unpack(const Dev &d)
{
    return flags_of(d) & (FLAG_CAPACITY | FLAG_FAULT);
}

// combinations per road -> exclusive offsets (the "combine" stage)
__global__ void __launch_bounds__(BLOCK) k_comb_count(Dev d)
{
    if (stop_after_unpack(d))
        return;
    const unsigned n_roads = ldcg(&d.ctrl->n_roads);
    const unsigned n_chunks = (n_roads + ROAD_CHUNK - 1) / ROAD_CHUNK;
    for (unsigned c = grab(d, Q_CNT); c < n_chunks; c = grab(d, Q_CNT)) {
        unsigned g = c * ROAD_CHUNK + threadIdx.x;
        unsigned long long N = 0;
        if (g < n_roads) {
            uint32_t pk = ldcg(&d.roads[g].pk);
            N = 1;
            for (unsigned l = 0; l < N_LAYERS; ++l)
                N *= (pk >> (4 * l)) & 15u;
        }
        unsigned long long t = block_sum(N);
        if (threadIdx.x == 0)
            d.cchunk_sum[c] = t;
    }
    if (last_block(&d.ctrl->done[2], gridDim.x)) {
        unsigned long long total = block_scan_array(d.cchunk_sum, d.cchunk_off, n_chunks);
        if (threadIdx.x == 0 && total > d.max_combs)
            raise_flag(d, FLAG_CAPACITY);
    }
}

__global__ void __launch_bounds__(BLOCK) k_comb_scatter(Dev d)
{
    if (stop_after_unpack(d))
        return;
    const unsigned n_roads = ldcg(&d.ctrl->n_roads);
    const unsigned n_chunks = (n_roads + ROAD_CHUNK - 1) / ROAD_CHUNK;
    for (unsigned c = grab(d, Q_CSC); c < n_chunks; c = grab(d, Q_CSC)) {
        unsigned g = c * ROAD_CHUNK + threadIdx.x;
        unsigned long long N = 0;
        if (g < n_roads) {
            uint32_t pk = ldcg(&d.roads[g].pk);
            N = 1;
            for (unsigned l = 0; l < N_LAYERS; ++l)
                N *= (pk >> (4 * l)) & 15u;
        }
        unsigned long long ex = block_excl_scan(N, nullptr);
        if (g < n_roads)
            d.comb_off[g] = ldcg(d.cchunk_off + c) + ex;
    }
}

// one thread per combination: the paper's fit kernel (Sec. II-A)
__global__ void __launch_bounds__(BLOCK) k_fit_plain(Dev d)
{
    if (stop_after_unpack(d))
        return;
    const unsigned n_roads = ldcg(&d.ctrl->n_roads);
    const unsigned long long n_comb = ldcg(&d.ctrl->n_comb);
    unsigned long long npass = 0;
    const unsigned long long stride = (unsigned long long)gridDim.x * BLOCK;
    for (unsigned long long base = (unsigned long long)blockIdx.x * BLOCK; base < n_comb; base += stride) {
        unsigned long long i = base + threadIdx.x;
        if (i < n_comb) {
            // road: last g with comb_off[g] <= i
            unsigned lo = 0, hi = n_roads;
            while (hi - lo > 1) {
                unsigned mid = (lo + hi) >> 1;
                if (ldcg(d.comb_off + mid) <= i)
                    lo = mid;
                else
                    hi = mid;
            }
            unsigned g = lo;
            RoadRec rec = ldcg(d.roads + g);
            unsigned comb = (unsigned)(i - ldcg(d.comb_off + g));
            const unsigned excl = min((rec.pk >> 20) & 7u, 4u);
            const uint16_t *co = d.coords + (size_t)g * 40;
            int x[6];
            unsigned t = comb, j = 0;
            for (unsigned l = 0; l < N_LAYERS; ++l) {
                unsigned nl = max(min((rec.pk >> (4 * l)) & 15u, (unsigned)MAX_HITS), 1u);
                unsigned q = divm(t, c_magic[nl]);
                unsigned dl = t - q * nl;
                t = q;
                if (l != excl)
                    x[j++] = ldcg(co + l * 8 + dl);
            }
            x[4] = rec.curv;
            x[5] = rec.phi;
            const svt_const_set *cs = d.consts + min((unsigned)rec.set, (unsigned)(N_SETS - 1));
            long long chi2 = 0;
            for (unsigned k = 0; k < 3; ++k) {
                int acc = 0;
                for (unsigned jj = 0; jj < 6; ++jj)
                    acc += (int)__ldg(&cs->C[k][jj]) * x[jj];
                chi2 += sq((acc >> 12) + __ldg(&cs->k[k]));
            }
            for (unsigned k = 0; k < 3; ++k) {
                int acc = 0;
                for (unsigned jj = 0; jj < 6; ++jj)
                    acc += (int)__ldg(&cs->F[k][jj]) * x[jj];
                d.fit_p[3 * i + k] = (acc >> 12) + __ldg(&cs->q[k]);
            }
            bool pass = chi2 <= d.cut;
            npass += pass;
            d.fit_key[i] = pass ? make_key(chi2, rec.pk >> 24, comb) : NO_KEY;
        }
    }
    npass = block_sum(npass);
    if (threadIdx.x == 0 && npass)
        atomicAdd(&d.ctrl->n_pass, npass);
}

__global__ void __launch_bounds__(BLOCK) k_warrior_plain(const __grid_constant__ Dev d)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (stop_after_unpack(d))
        return;
    p3_phase<true>(d, smem, Q_BOX, Q_GROUP, flags_of(d) & FLAG_CANDS);
}

__global__ void __launch_bounds__(BLOCK) k_p4(Dev d)
{
    if (stop_after_unpack(d))
        return;
    const unsigned n_roads = ldcg(&d.ctrl->n_roads);
    const unsigned n_chunks = (n_roads + ROAD_CHUNK - 1) / ROAD_CHUNK;
    for (unsigned c = grab(d, Q_P4); c < n_chunks; c = grab(d, Q_P4))
        p4_item(d, c, n_roads);
    if (last_block(&d.ctrl->done[1], gridDim.x))
        p4_finish(d, n_chunks);
}

__global__ void __launch_bounds__(BLOCK) k_p5(Dev d)
{
    __shared__ unsigned s_first[ROAD_CHUNK + 1];
    const unsigned n_roads = ldcg(&d.ctrl->n_roads);
    const unsigned n_chunks = (n_roads + ROAD_CHUNK - 1) / ROAD_CHUNK;
    if (!stop_after_unpack(d))
        for (unsigned c = grab(d, Q_P5); c < n_chunks; c = grab(d, Q_P5))
            p5_item<true>(d, c, n_roads, s_first);
    // the previous kernels' lookups are done: leave the group table empty
    clear_hash(d);
    leave(d, false, true);
}

__global__ void __launch_bounds__(BLOCK) k_export_roads(Dev d)
{
    const unsigned n_roads = min(ldcg(&d.last->n_roads), d.max_roads);
    for (unsigned g = blockIdx.x * BLOCK + threadIdx.x; g < n_roads; g += gridDim.x * BLOCK) {
        RoadRec rec = ldcg(d.roads + g);
        svt_road o;
        o.event = rec.event;
        o.road = (uint16_t)(rec.pk >> 24);
        unsigned set = rec.set, excl = set % 5, wb = set / 5;
        o.wedge = (uint8_t)(wb / 6);
        o.barrel = (uint8_t)(wb % 6);
        o.excl = (uint8_t)excl;
        for (unsigned l = 0; l < N_LAYERS; ++l)
            o.n[l] = (uint8_t)((rec.pk >> (4 * l)) & 15u);
        o.pad[0] = o.pad[1] = 0;
        o.curv = rec.curv;
        o.phi = rec.phi;
        for (unsigned j = 0; j < 40; ++j)   // slots beyond a layer's hits hold no coordinate
            o.coord[j >> 3][j & 7] = (j & 7u) < o.n[j >> 3] ? ldcg(d.coords + (size_t)g * 40 + j) : (uint16_t)0;
        d.road_out[g] = o;
    }
}

#endif   // the plain per-stage kernels

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

static size_t p1_smem() { return WARPS * sizeof(P1Warp); }
static size_t p2_smem() { return P2_LIST_AT + sizeof(P2List); }
static size_t p3_smem() { return P3_SHARED_BYTES + WARPS * P3_WARP_BYTES; }

size_t persistent_smem_bytes()
{
    size_t a = p2_smem(), b = p3_smem(), c = p1_smem(), e = sizeof(P5Smem);   // p2_smem: both P2 paths
    a = a > b ? a : b;
    a = a > c ? a : c;
    return a > e ? a : e;
}

static cudaError_t set_smem_attrs()
{
    static bool done = false;
    if (done)
        return cudaSuccess;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)persistent_smem_bytes())))
        return e;
#if SVT_BLOCK == 256
    if ((e = cudaFuncSetAttribute(k_p2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p2_smem())))
        return e;
    if ((e = cudaFuncSetAttribute(k_p1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p1_smem())))
        return e;
    if ((e = cudaFuncSetAttribute(k_warrior_plain, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)p3_smem())))
        return e;
#endif
    done = true;
    return cudaSuccess;
}

int persistent_max_blocks_per_sm(int device)
{
    (void)device;
    if (set_smem_attrs() != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_persistent, BLOCK,
                                                      persistent_smem_bytes()) != cudaSuccess)
        return 0;
    return nb;
}

cudaError_t launch_persistent(const Dev &d, cudaStream_t s, int blocks_per_sm, int max_ctas, int *n_launches)
{
    cudaError_t e = set_smem_attrs();
    if (e)
        return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int maxb = persistent_max_blocks_per_sm(dev);
    if (maxb <= 0)
        return cudaErrorInvalidConfiguration;
    Dev dd = d;
    void *args[] = {&dd};
    cudaLaunchConfig_t cfg = {};
    int grid = sms * ctas_per_sm(d.n_words, sms, BLOCK, maxb, blocks_per_sm);
    if (max_ctas > 0 && max_ctas < grid)
        grid = max_ctas;
    if (grid > GRID_MAX)   // the word spans (one per warp) and the per-CTA totals are sized for this
        grid = GRID_MAX;
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(BLOCK);
    cfg.dynamicSmemBytes = persistent_smem_bytes();
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelExC(&cfg, (const void *)k_persistent, args);
    *n_launches += 1;
    return e;
}

#if SVT_BLOCK == 256
static int plain_grid()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms * 4 < GRID_MAX ? sms * 4 : GRID_MAX;
}

cudaError_t launch_unpack_plain(const Dev &d, cudaStream_t s, int *n_launches)
{
    cudaError_t e = set_smem_attrs();
    if (e)
        return e;
    const int g = plain_grid();   // the same grid for P0 and P1: the word spans follow it
    k_p0<<<g, BLOCK, 0, s>>>(d);
    k_p1<<<g, BLOCK, p1_smem(), s>>>(d);
    k_p2<<<g, BLOCK, p2_smem(), s>>>(d);
    *n_launches += 3;
    return cudaGetLastError();
}

cudaError_t launch_fit_plain(const Dev &d, cudaStream_t s, int *n_launches)
{
    cudaError_t e = set_smem_attrs();
    if (e)
        return e;
    int g = plain_grid();
    k_comb_count<<<g, BLOCK, 0, s>>>(d);
    k_comb_scatter<<<g, BLOCK, 0, s>>>(d);
    k_fit_plain<<<g * 4, BLOCK, 0, s>>>(d);
    k_warrior_plain<<<g, BLOCK, p3_smem(), s>>>(d);
    k_p4<<<g, BLOCK, 0, s>>>(d);
    k_p5<<<g, BLOCK, 0, s>>>(d);
    *n_launches += 6;
    return cudaGetLastError();
}

cudaError_t launch_export_roads(const Dev &d, cudaStream_t s)
{
    k_export_roads<<<plain_grid(), BLOCK, 0, s>>>(d);
    return cudaGetLastError();
}
#endif

}  // namespace SVT_KNS
}  // namespace svt
