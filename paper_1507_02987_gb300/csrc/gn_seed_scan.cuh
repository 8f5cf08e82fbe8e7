// gn_seed_scan.cuh - seed lookup and hit chaining in one pass over the occurrence signatures
// (a6-a8 without storing hits); included by gn_search.cu.
//
// A chain of hits is worth an HSP only if it holds two or more (min_hsp_len > seed span), and
// its hits lie t, 2t .. D apart on one diagonal of one sequence (D < 4t here).  The signature
// word of an occurrence (SigKind) answers almost always whether such a hit can follow, so the
// scan reads 4 bytes a hit, once, and looks at nothing else for all but about 1 % of the hits.
// Those go to a candidate list and are checked against the packed bank: a hit with no
// predecessor within D starts its chain, walks it to the end and emits the HSP.  No other hit
// is stored, and none is sorted or grouped.
//
// Measured against the two-pass Bloom-filter fill and its bucket grouping (gn_search.cu), see
// the dispatch in search().
#pragma once

namespace gn {

// Per query offset: occurrence list [src, src + cnt), query signature (three fields as
// SIG_AHEAD, SIG_NEVER where no query window lies; or the bases around as SIG_FLANK).
// cnt = 0: no window here, none in the bank, or (SIG_FLANK) no chain can start here.
struct QueryRec {
    uint32_t src, cnt, sig, pad;
};
static_assert(sizeof(QueryRec) == 16, "QueryRec layout");

// One offset per thread.  qinfo = query << 16 | offset; units = 16-byte groups of four
// entries its list touches, at least one; hits[q] += the list's length.  The kernel waits on
// the list starts (random 8-byte reads, 33 MB for k = 11, mostly L2 hits); a warp finds its
// first query by one search and walks on from there.
template <int KIND>
__device__ __forceinline__ void query_rec(uint64_t x, const uint64_t *__restrict__ qstart, uint32_t nq, uint64_t M,
                                          const uint32_t *__restrict__ qpk, const uint32_t *__restrict__ qnb, const SeedShape &sh,
                                          int t, int ahead, int flank, const uint64_t *__restrict__ off,
                                          uint32_t *__restrict__ qinfo, QueryRec *__restrict__ rec, uint32_t *__restrict__ units,
                                          unsigned long long *__restrict__ hits) {
    const int lane = threadIdx.x & 31;
    uint32_t qi = 0;
    if (lane == 0) qi = dev_upper_index(qstart, nq + 1, x);
    qi = __shfl_sync(0xffffffffu, qi, 0);
    const bool in = x < M;
    uint32_t n = 0;
    if (in) {
        while (qstart[qi + 1] <= x) ++qi;
        const uint64_t qpos = x - qstart[qi], m = qstart[qi + 1] - qstart[qi];
        QueryRec r{0u, 0u, 0u, 0u};
        const bool window = qpos + (uint64_t)sh.span <= m && !dev_seed_has_nonbase(qnb, x, sh);
        if (window) {
            const uint32_t c = dev_seed_code(qpk, x, sh);
            const uint64_t o = off[c];
            n = (uint32_t)(off[c + 1] - o);
            if (n) { r.src = (uint32_t)o; r.cnt = n; }
        }
        if (KIND == SIG_FLANK) {
            r.sig = qpos > 0 ? dev_base(qpk, qnb, x - 1) : SIG_NO_BASE_QUERY;
            if (r.sig == SIG_NO_BASE) r.sig = SIG_NO_BASE_QUERY;
            // the next bases have to be there, or a chain from here ends before min_hsp_len
            const uint64_t y = qpos + (uint64_t)sh.span;
            if (r.cnt && y + flank <= m && !dev_has_nonbase(qnb, x + sh.span, flank))
                r.sig |= sig_flank(qpk, x + sh.span) & sig_flank_mask(flank);
            else
                r.cnt = 0;
            if (!r.cnt) r.src = 0;
        } else {
            for (int j = 0; j < SIG_FIELDS; ++j) {
                const uint64_t d = (uint64_t)t * (j + 1);
                uint32_t f = SIG_NEVER;
                if (window && j < ahead && qpos + d + (uint64_t)sh.span <= m && !dev_seed_has_nonbase(qnb, x + d, sh))
                    f = sig_hash(dev_seed_code(qpk, x + d, sh));
                r.sig |= f << (10 * j);
            }
            if (r.sig == (SIG_NEVER | SIG_NEVER << 10 | SIG_NEVER << 20)) r.src = r.cnt = 0;
        }
        qinfo[x] = (qi << 16) | (uint32_t)qpos;
        rec[x] = r;
        units[x] = r.cnt ? (uint32_t)(((uint64_t)r.src + r.cnt + 3u) >> 2) - (r.src >> 2) : 1u;
    }
    // hits per query: one atomic per warp where it lies in one query
    const uint32_t q0 = __shfl_sync(0xffffffffu, qi, 0);
    if (__all_sync(0xffffffffu, !in || qi == q0)) {
        const uint32_t top = __reduce_max_sync(0xffffffffu, n);
        unsigned long long sum = n;
        if (top < (1u << 27)) {
            sum = __reduce_add_sync(0xffffffffu, n);
        } else {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
        if (lane == 0 && sum) atomicAdd(&hits[q0], sum);
    } else if (n) {
        atomicAdd(&hits[qi], (unsigned long long)n);
    }
}

// unit_sums (null: none): the prefix sums of the units, by the block that finishes last, which saves
// a small search a launch (up to RECS_SUMS offsets; 6 of 205 us).
constexpr uint64_t RECS_SUMS = 4096;

template <int KIND>
__global__ void __launch_bounds__(256) k_query_recs(const uint64_t *__restrict__ qstart, uint32_t nq, uint64_t M,
                                                    const uint32_t *__restrict__ qpk, const uint32_t *__restrict__ qnb,
                                                    SeedShape sh, int t, int ahead, int flank,
                                                    const uint64_t *__restrict__ off, uint32_t *__restrict__ qinfo, QueryRec *__restrict__ rec,
                                                    uint32_t *__restrict__ units, unsigned long long *__restrict__ hits,
                                                    uint64_t *__restrict__ unit_sums, uint32_t *__restrict__ blocks_done) {
    const uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x - (threadIdx.x & 31) < M) query_rec<KIND>(x, qstart, nq, M, qpk, qnb, sh, t, ahead, flank, off, qinfo, rec, units, hits);
    if (!unit_sums) return;
    __shared__ uint64_t warp_sum[8];
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(blocks_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t per = (M + blockDim.x - 1) / blockDim.x, a = min(M, threadIdx.x * per), b = min(M, a + per);
    uint64_t sum = 0;
    for (uint64_t i = a; i < b; ++i) sum += __ldcg(&units[i]);
    uint64_t upto = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += y;
    }
    if (lane == 31) warp_sum[wid] = upto;
    __syncthreads();
    for (int w = 0; w < wid; ++w) upto += warp_sum[w];
    uint64_t at = upto - sum;
    for (uint64_t i = a; i < b; ++i) {
        unit_sums[i] = at;
        at += __ldcg(&units[i]);
    }
    if (threadIdx.x == blockDim.x - 1) unit_sums[M] = upto;
}

// What the checks of a hit need.
struct ScanCtx {
    const uint32_t *qinfo;
    const uint64_t *qstart;
    const uint32_t *post, *bpk, *bnb, *qpk, *qnb;
    SeedShape sh;
    int t, ahead, flank;
    uint32_t min_len;
    SeqMap sm;
    DevHsp *out;
    uint32_t *count, cap, *status;
    uint64_t n_post, n_bank, n_query;
};

// 64 packed bases from position p (any sign): word i holds bases 16 i .. 16 i + 15, first one
// in the top bits, bad the non-base bits.  Words outside [0, n] are clamped: the caller masks
// the positions they stand for.
struct Window64 {
    uint32_t w[4];
    uint64_t bad;
    __device__ __forceinline__ void load(const uint32_t *__restrict__ pk, const uint32_t *__restrict__ nb, int64_t p,
                                         uint64_t n) {
        const int64_t a = p >> 4, b = p >> 5, la = (int64_t)(n >> 4) + 1, lb = (int64_t)(n >> 5) + 1;  // last words (zero pad)
        uint32_t v[5], q[3];
#pragma unroll
        for (int i = 0; i < 5; ++i) v[i] = pk[max((int64_t)0, min(a + i, la))];
#pragma unroll
        for (int i = 0; i < 3; ++i) q[i] = nb[max((int64_t)0, min(b + i, lb))];
        const uint32_t sa = 2u * (uint32_t)(p & 15), sb = (uint32_t)(p & 31);
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = __funnelshift_l(v[i + 1], v[i], sa);
        bad = (uint64_t)__funnelshift_r(q[0], q[1], sb) | (uint64_t)__funnelshift_r(q[1], q[2], sb) << 32;
    }
};

// Bit i: the bases at distance o + i (i < 64) on the diagonal of (x, g) are equal bases, that
// is, codes agree and neither is a non-base.  lo, hi: distances that lie in the query and the
// sequence.
__device__ __forceinline__ uint64_t equal64_raw(const ScanCtx &c, uint64_t x, uint64_t g, int64_t o) {
    Window64 q, d;
    q.load(c.qpk, c.qnb, (int64_t)x + o, c.n_query);
    d.load(c.bpk, c.bnb, (int64_t)g + o, c.n_bank);
    uint64_t eq = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t y = ~(q.w[i] ^ d.w[i]);
        uint32_t v = __brev(y & (y >> 1) & 0x55555555u) >> 1;  // bit 2 k: base k of the word
        v = (v | v >> 1) & 0x33333333u;
        v = (v | v >> 2) & 0x0F0F0F0Fu;
        v = (v | v >> 4) & 0x00FF00FFu;
        v = (v | v >> 8) & 0x0000FFFFu;
        eq |= (uint64_t)v << (16 * i);
    }
    return eq & ~(q.bad | d.bad);
}
__device__ __forceinline__ uint64_t within(uint64_t eq, int64_t o, int64_t lo, int64_t hi) {
    if (o < lo) eq = lo - o < 64 ? eq >> (lo - o) << (lo - o) : 0ull;
    if (o + 64 > hi) eq = hi - o > 0 ? eq << (o + 64 - hi) >> (o + 64 - hi) : 0ull;
    return eq;
}
// The seed's kept bases all equal at distance o + s, from the 64 bits at o.  A hit's whole window lies
// in the query and the sequence, also the positions at its ends that a mask does not keep: with lo
// and hi drawn in by as many, the kept bases lie within exactly where the window does.
__device__ __forceinline__ bool seed_at(uint64_t eq, int s, uint32_t keep) { return ((uint32_t)(eq >> s) & keep) == keep; }

// Appends the HSPs of the lanes with `emit` set: one counter update per warp.
__device__ __forceinline__ void scan_emit(const ScanCtx &c, bool emit, uint32_t qi, uint32_t seq, uint32_t qs,
                                          uint32_t qe, uint32_t ds) {
    const int lane = threadIdx.x & 31;
    const uint32_t m = __ballot_sync(0xffffffffu, emit);
    if (!m) return;
    uint32_t at = 0;
    if (lane == __ffs(m) - 1) at = atomicAdd(c.count, (uint32_t)__popc(m));
    at = __shfl_sync(0xffffffffu, at, __ffs(m) - 1) + __popc(m & ((1u << lane) - 1u));
    if (!emit) return;
    if (at < c.cap) {
        DevHsp h;
        h.qi = qi; h.seq = seq; h.qs = qs; h.qe = qe; h.ds = ds; h.de = ds + (qe - qs); h.len = qe - qs;
        c.out[at] = h;
    } else {
        atomicOr(c.status, DEV_ERR_CAPACITY);
    }
}

// Checks up to 32 candidate hits, lane l the occurrence p of query offset x (valid lanes):
// chain heads walk their chains and emit HSPs.  A lane walks SCAN_LANE_STEPS links alone,
// then its warp goes on 32 grid positions (SIG_FLANK: 512 bases) at a time, so that a long
// chain does not hold 31 lanes up.
constexpr int SCAN_LANE_STEPS = 24;

// EDGES: the mask does not keep its first or its last position (a form of its own: taken from every
// mask, the two limits cost k_chain 710 instead of 692 us for 2,000 queries against 4 Gbp).
template <bool EDGES>
__device__ __forceinline__ void scan_check_ahead(const ScanCtx &c, bool valid, uint32_t p, uint32_t x) {
    const int lane = threadIdx.x & 31;
    // links 1 .. ahead of one hit lie in one 64-base window when (ahead - 1) t + span <= 64
    const bool near = (c.ahead - 1) * (int64_t)c.t + c.sh.span <= 64;
    const uint32_t keep = c.sh.keep;
    uint64_t g = 0, s0 = 0;
    int64_t lo = 0, hi = 0, d = 0;
    uint32_t qi = 0, sq = 0, qpos = 0;
    bool head = false, open = false;
    // distance from the hit at distance d to the next one on its diagonal, 0 if it is the last
    auto link = [&](uint64_t x, uint64_t g, int64_t d, int64_t lo, int64_t hi) -> int64_t {
        if (near) {
            const uint64_t e = within(equal64_raw(c, x, g, d + c.t), d + c.t, lo, hi);
            for (int j = 0; j < c.ahead; ++j)
                if (seed_at(e, j * c.t, keep)) return (int64_t)(j + 1) * c.t;
            return 0;
        }
        for (int j = 1; j <= c.ahead; ++j) {
            const int64_t o = d + (int64_t)j * c.t;
            if (seed_at(within(equal64_raw(c, x, g, o), o, lo, hi), 0, keep)) return (int64_t)j * c.t;
        }
        return 0;
    };
    if (valid) valid = GN_CHECK(p < c.n_post);
    if (valid) {
        g = c.post[p];
        const uint32_t qinf = c.qinfo[x];
        qi = qinf >> 16;
        qpos = qinf & 0xFFFFu;
        // bases on both sides first: they do not wait for the sequence lookup
        const int64_t back = -(int64_t)c.ahead * c.t;
        uint64_t ea = 0, eb = 0;
        if (near) {
            ea = equal64_raw(c, x, g, c.t);
            eb = equal64_raw(c, x, g, back);
        }
        sq = dev_seq_of(c.sm, g);
        s0 = c.sm.start[sq];
        lo = -(int64_t)min((uint64_t)qpos, g - s0);
        hi = (int64_t)min(c.qstart[qi + 1] - c.qstart[qi] - qpos, c.sm.start[sq + 1] - g);
        if (EDGES) {
            lo += __ffs(keep) - 1;
            hi -= c.sh.span - 32 + __clz(keep);
        }
        if (near) {
            ea = within(ea, c.t, lo, hi);
            eb = within(eb, back, lo, hi);
            for (int j = 0; j < c.ahead && !d; ++j)
                if (seed_at(ea, j * c.t, keep)) d = (int64_t)(j + 1) * c.t;
            head = d != 0;
            for (int j = 0; j < c.ahead; ++j) head = head && !seed_at(eb, j * c.t, keep);
        } else {
            d = link(x, g, 0, lo, hi);
            head = d != 0;
            for (int j = 1; j <= c.ahead && head; ++j) {
                const int64_t o = -(int64_t)j * c.t;
                head = !seed_at(within(equal64_raw(c, x, g, o), o, lo, hi), 0, keep);
            }
        }
        open = head;
        // d: distance of the chain's last hit.  A window holds the next `grid` positions; the walk
        // goes on in it while all positions in reach lie in it (a window a link: 18 instead of 12 us
        // for a chain of 30 links, 60 instead of 47 for 1,000 diverged copies on 400 Mbp).
        const int grid = near ? (64 - c.sh.span) / c.t + 1 : 0;
        for (int step = 0; step < SCAN_LANE_STEPS && open; ++step) {
            if (!near) {
                const int64_t l = link(x, g, d, lo, hi);
                d += l;
                open = l != 0;
                continue;
            }
            const uint64_t e = within(equal64_raw(c, x, g, d + c.t), d + c.t, lo, hi);
            uint32_t at = 0;  // positions past the last hit, from the window's first one
            for (int j = 0; j < grid && j < (int)at + c.ahead; ++j)
                if (seed_at(e, j * c.t, keep)) at = j + 1;
            d += (int64_t)at * c.t;
            open = (int)at + c.ahead > grid;
        }
    }
    uint32_t todo = __ballot_sync(0xffffffffu, open);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t wx = __shfl_sync(0xffffffffu, x, src);
        const uint64_t wg = __shfl_sync(0xffffffffu, g, src);
        const int64_t wlo = __shfl_sync(0xffffffffu, lo, src), whi = __shfl_sync(0xffffffffu, hi, src);
        int64_t wd = __shfl_sync(0xffffffffu, d, src);
        const uint32_t reach = (1u << c.ahead) - 1u;
        for (;;) {
            // bit i: a hit (i + 1) t past the last one; the chain goes on while a set bit lies in reach
            const int64_t o = wd + (int64_t)(lane + 1) * c.t;
            const bool hit = o < whi && seed_at(within(equal64_raw(c, wx, wg, o), o, wlo, whi), 0, keep);
            const uint32_t bits = __ballot_sync(0xffffffffu, hit);
            int last = 0;
            while (last < 32) {
                const uint32_t nx = (bits >> last) & reach;
                if (!nx) break;
                last += __ffs(nx);
            }
            wd += (int64_t)last * c.t;
            if (last + c.ahead <= 32) break;  // every position in reach of the last hit was looked at
        }
        if (lane == src) d = wd;
    }
    const uint32_t len = (uint32_t)(d + c.sh.span);
    scan_emit(c, head && len >= c.min_len, qi, sq, qpos, qpos + len, (uint32_t)(g - s0));
}

// SIG_FLANK (stride 1): a chain is a maximal run of equal bases, and its first hit the one
// whose preceding bases differ (the signature's first field, exact).
__device__ __forceinline__ void scan_check_flank(const ScanCtx &c, bool valid, uint32_t p, uint32_t x) {
    const int lane = threadIdx.x & 31;
    uint64_t g = 0, s0 = 0;
    uint32_t qi = 0, sq = 0, qpos = 0, run = 0, room = 0;
    bool open = false;
    if (valid) valid = GN_CHECK(p < c.n_post);
    if (valid) {
        g = c.post[p];
        const uint32_t qinf = c.qinfo[x];
        qi = qinf >> 16;
        qpos = qinf & 0xFFFFu;
        sq = dev_seq_of(c.sm, g);
        s0 = c.sm.start[sq];
        const uint64_t m = c.qstart[qi + 1] - c.qstart[qi];
        room = (uint32_t)min(m - qpos, c.sm.start[sq + 1] - g);  // bases left in both
        run = (uint32_t)c.sh.span;
        open = true;
    }
    // equal bases from offset r on, 16 at a time: their number, 16 if all are
    auto equal16 = [&](uint64_t q0, uint64_t d0) {
        uint32_t wq, bq, wd, bd;
        base_window16(c.qpk, c.qnb, (int64_t)q0, wq, bq);
        base_window16(c.bpk, c.bnb, (int64_t)d0, wd, bd);
        const uint32_t df = wq ^ wd, ne = (df | (df >> 1)) & 0x55555555u;  // bit 30 - 2k: bases k differ
        const uint32_t n_eq = ne ? (uint32_t)__clz(ne) >> 1 : 16u;
        const uint32_t bad = bq | bd;
        return bad ? min(n_eq, (uint32_t)__ffs(bad) - 1u) : n_eq;
    };
    for (int step = 0; step < SCAN_LANE_STEPS && open; ++step) {
        if (run >= room) { open = false; break; }
        const uint32_t e = min(equal16((uint64_t)x + run, g + run), room - run);
        run += e;
        if (e < 16) open = false;
    }
    uint32_t todo = __ballot_sync(0xffffffffu, open);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t wx = __shfl_sync(0xffffffffu, x, src), wroom = __shfl_sync(0xffffffffu, room, src);
        const uint64_t wg = __shfl_sync(0xffffffffu, g, src);
        uint32_t wr = __shfl_sync(0xffffffffu, run, src);
        for (;;) {
            const uint32_t r = wr + 16u * (uint32_t)lane;
            const uint32_t e = r < wroom ? min(equal16((uint64_t)wx + r, wg + r), wroom - r) : 0u;
            const uint32_t part = __ballot_sync(0xffffffffu, e < 16u);
            if (!part) { wr += 512u; continue; }
            const int first = __ffs(part) - 1;
            wr += 16u * (uint32_t)first + __shfl_sync(0xffffffffu, e, first);
            break;
        }
        if (lane == src) run = wr;
    }
    scan_emit(c, valid && run >= c.min_len, qi, sq, qpos, qpos + run, (uint32_t)(g - s0));
}

// The scan.  The lists of all query offsets form one index space of units (16-byte groups;
// uoff: their exclusive scan), cut into equal tiles that warps take from a counter, so a long
// list is shared and short ones do not cost a warp each.  Within a tile a warp holds the
// records of 32 offsets, one per lane, and steps through their units 32 at a time: the starts
// of lists inside a step, OR-ed into one word, give each lane its list by a bit count, and two
// shuffles its entries' address and signature.  Four steps' loads are in flight at a time
// (2 KB a warp).  Candidates gather in shared memory and leave 32 at a time to a list that
// k_chain works through: where a query meets a repeat family, half a tile's hits are
// candidates, and checked inside the scan they left most of the chip waiting for the warps
// that drew such tiles (2,000 queries against 4 Gbp: 4.3 ms; busiest SM 2.2 times the mean).
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_STEPS = 4;
constexpr int SCAN_QUEUE = 64;
// Units of one launch, at most (a call's limits are checked after the first; a tile's number has 32
// bits), and candidates of one list, at most: in low-complexity sequence every hit is a
// candidate, so they are counted in 64 bits, and listed, checked and made HSPs of in 32.
constexpr uint64_t SCAN_RANGE = 1ull << 32, CAND_MAX = 1ull << 31;

// A launch takes the units [u_from, u_to); n_all: where it leaves the number of all units.
template <int KIND>
__global__ void __launch_bounds__(SCAN_THREADS, 4) k_seed_scan(const QueryRec *__restrict__ rec,
                                                               const uint64_t *__restrict__ uoff, uint64_t M,
                                                               uint64_t u_from, uint64_t u_to,
                                                               unsigned long long *__restrict__ n_all,
                                                               const uint4 *__restrict__ sig4, uint64_t n_units,
                                                               int flank, uint2 *__restrict__ cand,
                                                               unsigned long long *__restrict__ cand_count, uint32_t cand_cap,
                                                               uint32_t *__restrict__ next_tile) {
    __shared__ uint2 queue_s[SCAN_THREADS / 32][SCAN_QUEUE];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u, le = lt | (1u << lane);
    uint2 *queue = queue_s[wib];
    uint32_t nqueue = 0;
    const uint64_t all = uoff[M], total = min(all, u_to);
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_all = all;
    const uint64_t warps = (uint64_t)gridDim.x * (SCAN_THREADS / 32);
    // tiles: eight or more a warp where there is work for that, 64 to 1,024 units
    const uint64_t R = min((uint64_t)1024, max((uint64_t)64, (uint64_t)(((total - u_from) / (warps * 8) + 31) & ~31ull)));
    const uint32_t next_mask = KIND == SIG_FLANK ? sig_flank_mask(flank) : 0u;
    auto flush = [&](uint32_t n) {  // the first n (<= 32) queued candidates
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(cand_count, (unsigned long long)n);
        at = __shfl_sync(0xffffffffu, at, 0) + lane;
        __syncwarp();
        if ((uint32_t)lane < n && at < cand_cap) cand[at] = queue[lane];
        uint2 rest = make_uint2(0u, 0u);
        if ((uint32_t)lane + n < nqueue) rest = queue[lane + n];
        __syncwarp();
        if ((uint32_t)lane + n < nqueue) queue[lane] = rest;
        nqueue -= n;
        __syncwarp();
    };
    for (;;) {
        uint32_t tile = 0;
        if (lane == 0) tile = atomicAdd(next_tile, 1u);
        tile = __shfl_sync(0xffffffffu, tile, 0);
        const uint64_t u0 = u_from + (uint64_t)tile * R;
        if (u0 >= total) break;
        const int64_t tile_end = (int64_t)min(R, total - u0);
        // last offset whose units start at or before u0: 32 probes a round
        uint64_t lo = 0, hi = M;
        while (hi - lo > 1) {
            const uint64_t step = (hi - lo + 31) / 32, at = lo + (uint64_t)lane * step;
            const uint32_t ok = __ballot_sync(0xffffffffu, at < hi && uoff[at] <= u0);
            const int top = 31 - __clz(ok);
            hi = min(hi, lo + (uint64_t)(top + 1) * step);
            lo += (uint64_t)top * step;
        }
        int32_t b = 0;
        for (uint64_t xw = lo; b < (int32_t)tile_end; xw += 32) {
            // the window's records; us: first unit of the lane's list, relative to the tile
            const uint64_t xi = xw + lane;
            int64_t us64 = INT32_MAX;
            QueryRec r{0u, 0u, 0u, 0u};
            if (xi < M) {
                us64 = (int64_t)(uoff[xi] - u0);
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(rec) + xi);
                r.src = v.x; r.cnt = v.y; r.sig = v.z;
            }
            const int64_t wend64 = (int64_t)(uoff[min(xw + 32, M)] - u0);
            const int32_t end = (int32_t)min(wend64, tile_end);
            const int32_t us = (int32_t)max(min(us64, (int64_t)INT32_MAX), (int64_t)INT32_MIN);
            const uint32_t dq = (r.src >> 2) - (uint32_t)(uint64_t)us64;  // unit u of the tile: group dq + u
            for (int32_t b0 = b; b0 < end; b0 += 32 * SCAN_STEPS) {
                uint4 e[SCAN_STEPS];
                uint32_t idx[SCAN_STEPS];
                uint32_t before = __popc(__ballot_sync(0xffffffffu, us < b0));
#pragma unroll
                for (int v = 0; v < SCAN_STEPS; ++v) {
                    const int32_t bv = b0 + 32 * v;
                    const uint32_t rel = (uint32_t)us - (uint32_t)bv;
                    const uint32_t starts = __reduce_or_sync(0xffffffffu, us >= bv && rel < 32u ? 1u << rel : 0u);
                    idx[v] = (before + __popc(starts & le) - 1u) & 31u;
                    before += __popc(starts);
                    const uint32_t grp = __shfl_sync(0xffffffffu, dq, idx[v]) + (uint32_t)(bv + lane);
                    bool ok = bv + lane < end;
                    if (ok) ok = GN_CHECK(grp < n_units);
                    e[v] = ok ? __ldg(&sig4[grp]) : make_uint4(0u, 0u, 0u, 0u);
                }
                uint32_t keep = 0;  // bit 4 v + u: entry u of step v may have a hit ahead
#pragma unroll
                for (int v = 0; v < SCAN_STEPS; ++v) {
                    const uint32_t qs = __shfl_sync(0xffffffffu, r.sig, idx[v]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t d = (u == 0 ? e[v].x : u == 1 ? e[v].y : u == 2 ? e[v].z : e[v].w) ^ qs;
                        bool k;
                        if (KIND == SIG_FLANK) k = (d & next_mask) == 0u && (d & 7u) != 0u;
                        else k = ((d - 0x00100401u) & ~d & 0x20080200u) != 0u;  // a 10-bit field of zeros
                        keep |= k ? 1u << (4 * v + u) : 0u;
                    }
                    if (b0 + 32 * v + lane >= end) keep &= ~(15u << (4 * v));
                }
                const uint32_t any = __reduce_or_sync(0xffffffffu, keep);
                if (!any) continue;
                const uint32_t packed = idx[0] | idx[1] << 8 | idx[2] << 16 | idx[3] << 24;
#pragma unroll 1
                for (uint32_t left = any; left; left &= left - 1) {
                    const int at = __ffs(left) - 1, v = at >> 2;
                    const uint32_t i = (packed >> (8 * v)) & 31u;
                    const uint32_t src = __shfl_sync(0xffffffffu, r.src, i);
                    const uint32_t cnt = __shfl_sync(0xffffffffu, r.cnt, i);
                    const uint32_t grp = __shfl_sync(0xffffffffu, dq, i) + (uint32_t)(b0 + 32 * v + lane);
                    const uint32_t p = grp * 4u + (uint32_t)(at & 3);
                    // entries of a neighbouring list that share the group do not count
                    const bool k = ((keep >> at) & 1u) && p - src < cnt;
                    const uint32_t mk = __ballot_sync(0xffffffffu, k);
                    if (!mk) continue;
                    if (k) queue[nqueue + __popc(mk & lt)] = make_uint2(p, (uint32_t)xw + i);
                    nqueue += __popc(mk);
                    if (nqueue >= 32u) flush(32u);
                }
            }
            b = end;
        }
    }
    if (nqueue) flush(nqueue);
}

// Checks the candidates of the scan, 32 to a warp from a counter.
template <int KIND, bool EDGES>
__global__ void __launch_bounds__(SCAN_THREADS) k_chain(const __grid_constant__ ScanCtx c, const uint2 *__restrict__ cand,
                                                        const unsigned long long *__restrict__ cand_count, uint32_t cand_cap,
                                                        uint32_t *__restrict__ next) {
    const int lane = threadIdx.x & 31;
    const uint32_t n = (uint32_t)min(*cand_count, (unsigned long long)cand_cap);
    for (;;) {
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(next, 32u);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (at >= n) break;
        const bool valid = at + lane < n;
        const uint2 e = valid ? cand[at + lane] : make_uint2(0u, 0u);
        if (KIND == SIG_FLANK) scan_check_flank(c, valid, e.x, e.y);
        else scan_check_ahead<EDGES>(c, valid, e.x, e.y);
    }
}

}  // namespace gn
