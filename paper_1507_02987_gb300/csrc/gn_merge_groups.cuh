// gn_merge_groups.cuh - overlap merging by groups (included by gn_search.cu).  The HSPs of one
// query and one range of bank sequences form a group; a group fits shared memory, where it is
// sorted, swept and compacted at once, so that no sort over the whole call's records is needed.
//   k_group_count    each HSP's group and its place in it
//   k_group_lists    groups by size: a warp's, a block's, a large block's, too large
//   k_group_scatter  indices of the HSPs, group by group
//   k_merge_groups*  one group each: order by (seq, qs, ds, qe), sweep, the N longest boxes
//   k_group_pack     boxes of all groups back to back, in (qi, seq, qs, ds, qe) order
// Sorting the call's records by (qi, seq, qs), sweeping and compacting them reads and writes the
// records and their keys once a pass, a launch each; the pieces of long queries' chains, joined
// in (qi, seq, diagonal, qs) order, the same with more passes.  By groups a record is read once
// and its box written twice.  Merge and selection, us: 2.1 M HSPs of 2,000 queries 730 -> 395;
// 103,000 of 1,000 queries 203 -> 105; 11,000 of 666 queries 163 -> 90.  The join of 177,000 pieces
// of 8 queries 241 -> 150, their merge and selection 425 -> 160.

namespace gn {

// HSPs a group has on average, at most, and the largest group of each kernel.  The merge phase in
// us at averages of 64 | 128 | 256: 2.1 M HSPs 277 | 308 | 380, 103,000 HSPs 58 | 62 | 105, 89,000 HSPs
// most of which lie in one sequence a query 66 | 113 | 110.  Warps taking up to 128 (256) instead of 64: 263 (271),
// 62 (78) and 70 (87); 128 threads of 8 records instead of 256 of 4: 320, 75 and 85.
constexpr uint32_t MG_TARGET = 64;
constexpr uint32_t MG_WARP = 64, MG_MID = 1024, MG_BIG = 8192;
constexpr int MG_BITS = 13;          // bits of an index into a group
static_assert(MG_BIG == 1u << MG_BITS, "an index fits its bits");

// Groups of the queries: first(q) .. first(q + 1), and in them the bank's sequences in equal ranges.
// Group order is (qi, seq) order.  A query has groups by its length (HSPs are about as many as
// bases), which needs no count, or, where that leaves a group too large (a short query of a
// frequent repeat), by its number of HSPs.
struct GroupMap {
    const uint64_t *qstart;
    uint64_t per_base;  // groups per base, 32 bits after the point
    uint32_t per_seq;   // 1 / sequences, 32 bits after the point, rounded down
    const uint64_t *by_count;  // first(q) - q, by the queries' HSPs (null: by length)
    __device__ __forceinline__ uint32_t first(uint32_t q) const {
        return q + (uint32_t)(by_count ? by_count[q] : (qstart[q] * per_base) >> 32);
    }
    __device__ __forceinline__ uint32_t of(uint32_t q, uint32_t seq) const {
        const uint32_t f = first(q), n = first(q + 1) - f;
        return f + (uint32_t)(((uint64_t)(seq * per_seq) * n) >> 32);
    }
};

// Groups of each query by its HSPs, but for its first: one more at every MG_TARGET-th HSP.
__global__ void __launch_bounds__(256) k_query_parts(const DevHsp *__restrict__ h, uint32_t n, uint32_t *__restrict__ seen,
                                                     uint32_t *__restrict__ more) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t q = i < n ? h[i].qi : 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xffffffffu, q);
    if (i >= n || (threadIdx.x & 31) != (uint32_t)(__ffs(peers) - 1)) return;
    const uint32_t c = __popc(peers), before = atomicAdd(&seen[q], c);
    const uint32_t n_more = (before + c) / MG_TARGET - before / MG_TARGET;
    if (n_more) atomicAdd(&more[q], n_more);
}

__global__ void __launch_bounds__(256) k_group_count(const DevHsp *__restrict__ h, uint32_t n, GroupMap gm,
                                                     uint32_t *__restrict__ cnt, uint2 *__restrict__ where) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const uint32_t g = i < n ? gm.of(h[i].qi, h[i].seq) : 0xFFFFFFFFu;
    // HSPs come in roughly by query: one atomic per group of a warp's 32
    const uint32_t peers = __match_any_sync(0xffffffffu, g);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (i < n && lane == leader) base = atomicAdd(&cnt[g], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (i < n) where[i] = make_uint2(g, base + __popc(peers & ((1u << lane) - 1u)));
}

// words: groups in list from its front (a block each), from its back (a large block each), and
// groups that no kernel holds
__global__ void k_group_lists(const uint32_t *__restrict__ cnt, uint32_t G, uint32_t *__restrict__ list,
                              uint32_t *__restrict__ words) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t c = g < G ? cnt[g] : 0u;
    if (c > MG_BIG) atomicAdd(&words[2], 1u);
    else if (c > MG_MID) list[G - 1 - atomicAdd(&words[1], 1u)] = g;
    else if (c > MG_WARP) list[atomicAdd(&words[0], 1u)] = g;
}

__global__ void __launch_bounds__(256) k_group_scatter(const uint2 *__restrict__ where, uint32_t n,
                                                       const uint64_t *__restrict__ off, uint32_t *__restrict__ perm) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint2 w = where[i];
    perm[off[w.x] + w.y] = i;
}

struct MergeGroups {
    const DevHsp *in;
    const uint32_t *perm;  // HSPs by group: group g's from off[g] on, cnt[g] of them (null: in lies so)
    const uint64_t *off;
    const uint32_t *cnt;
    int low_bits;          // of the sort key's second part: the query start (STITCH: the diagonal)
    int len_bytes;         // of the longest box
    uint32_t N;            // boxes kept of a group (0: all)
    uint32_t diag0, span, min_len;  // STITCH: added to the diagonal; the seed's span; shortest chain kept
    DevHsp *out;           // group g's boxes from off[g] on
    uint32_t *n_out;       // how many
};

template <int T, int E>
struct MergeSmem {  // of a team
    uint4 box[T * E];
    uint64_t key[T * E < 128 ? 128 : T * E];  // the sort's exchanges, then the lengths' histogram
    uint64_t tmp[33];
    uint32_t seq[T * E], heads[T * E / 32];
};

// One group of at most T * E HSPs: their overlap merging, or (STITCH) the join of the pieces of long
// queries' chains as k_stitch_sweep does it, on records whose len word is the diagonal.
//
// The sweep is the one of overlap_run, with two shortcuts.  Records of one qs are put in (ds, qe)
// order beforehand (few share one), and a record that begins at or after every end before it in
// its sequence opens a box whatever the open box is: a head bit there cuts the sequence's run
// into pieces that threads sweep side by side.  Boxes are written over the records of their piece
// already taken, never ahead of the reading.
template <int T, int E, bool STITCH>
__device__ __forceinline__ void merge_group(const MergeGroups &m, uint32_t g, MergeSmem<T, E> &S) {
    typedef Team<T, E> tm;
    const uint32_t t = tm::tid(), c = m.cnt[g];
    const uint64_t o = m.off[g];
    const uint32_t P = tm::padded(c);
    uint4 *box = S.box;
    // order of the records by (seq, qs) or (seq, diagonal): the records lie in shared memory as they come, then sorted
    {
        uint64_t r[E];
        const uint32_t A = P / E;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = e * A + t;
            r[e] = ~0ull;
            if (t < A && i < c) {
                const DevHsp h = m.in[m.perm ? m.perm[o + i] : o + i];
                r[e] = ((((uint64_t)h.seq << m.low_bits) | (STITCH ? h.len + m.diag0 : h.qs)) << MG_BITS) | i;
                box[i] = make_uint4(h.qs, h.qe, h.ds, h.de);
            }
        }
        tm::sort(r, S.key, P, KeyLess());
        tm::sync();
        uint4 b[E];
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (t * E + e < c) b[e] = box[(uint32_t)r[e] & ((1u << MG_BITS) - 1u)];
        tm::sync();
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = t * E + e;
            if (i < c) {
                box[i] = b[e];
                S.seq[i] = (uint32_t)(r[e] >> (m.low_bits + MG_BITS));
            }
        }
    }
    tm::sync();
    auto by_ds = [](const uint4 &b) { return ((uint64_t)b.z << 32) | b.y; };  // (ds, qe)
    auto order = [&](const uint4 &b) { return STITCH ? (uint64_t)b.x : by_ds(b); };  // of equal keys
    auto shares = [&](uint32_t i) {
        if (S.seq[i] != S.seq[i - 1]) return false;
        const uint4 a = box[i - 1], b = box[i];
        return STITCH ? a.z - a.x == b.z - b.x : a.x == b.x;
    };
    if (t < T * E / 32) S.heads[t] = 0;
    uint32_t tied = 0;  // of this thread's records: a bit for those with the key of the one before
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = t * E + e;
        if (i > 0 && i < c && shares(i)) tied |= 1u << e;
    }
    tm::sync();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = t * E + e;
        if (i < c && !((tied >> e) & 1u)) atomicOr(&S.heads[i >> 5], 1u << (i & 31));
    }
    tm::sync();
    auto is_head = [&](uint32_t i) { return (S.heads[i >> 5] >> (i & 31)) & 1u; };
    for (uint32_t i = t * E; i < min(c, t * E + E); ++i) {
        if (!is_head(i)) continue;
        for (uint32_t e = i + 1; e < c && !is_head(e); ++e) {
            const uint4 x = box[e];
            uint32_t j = e;
            for (; j > i && order(box[j - 1]) > order(x); --j) box[j] = box[j - 1];
            box[j] = x;
        }
    }
    tm::sync();
    if (!STITCH) {  // heads of equal keys so far, now of pieces
        if (t < T * E / 32) S.heads[t] = 0;
        uint64_t v[E], last = 0;  // (seq, end of the box) ; the largest one so far
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = t * E + e;
            v[e] = i < c ? ((uint64_t)S.seq[i] << 32) | box[i].y : 0ull;
            last = max(last, v[e]);
        }
        last = tm::excl_max(last, S.tmp);
        tm::sync();
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = t * E + e;
            if (i < c && (i == 0 || (uint32_t)(last >> 32) != (uint32_t)(v[e] >> 32) || (uint32_t)last <= box[i].x))
                atomicOr(&S.heads[i >> 5], 1u << (i & 31));
            last = max(last, v[e]);
        }
        tm::sync();
    }
    for (uint32_t i = t; i < c; i += T) {
        if (!is_head(i)) continue;
        uint32_t at = i, j = i + 1;  // next box slot, next record
        uint4 b = box[i];
        auto put = [&]() {  // boxes of one qs in (ds, qe, de) order, as they are selected
            if (STITCH) {
                b.w = b.z + (b.y - b.x);
                if (b.y - b.x >= m.min_len) box[at++] = b;
                return;
            }
            uint32_t p = at++;
            for (; p > i; --p) {
                const uint4 x = box[p - 1];
                if (x.x != b.x || by_ds(x) < by_ds(b) || (by_ds(x) == by_ds(b) && x.w <= b.w)) break;
                box[p] = x;
            }
            box[p] = b;
        };
        for (; j < c && !is_head(j); ++j) {
            const uint4 h = box[j];
            if (STITCH) {
                if (h.x + m.span <= b.y) {
                    b.y = max(b.y, h.y);
                } else {
                    put();
                    b = h;
                }
            } else if (h.x < b.y && b.x < h.y && h.z < b.w && b.z < h.w) {
                b = make_uint4(min(b.x, h.x), max(b.y, h.y), min(b.z, h.z), max(b.w, h.w));
            } else {
                put();
                b = h;
            }
        }
        put();
        for (; at < j; ++at) box[at].y = 0;  // no box ends at 0
    }
    tm::sync();
    // The boxes in order; of more than N only the N longest, the first ones of the shortest length
    // taken: no other box of the group can be among the query's N longest.  (A sort by length and
    // one back cost 27,000 to 42,000 cycles a block, as much as the first sort.)
    uint32_t len[E], n_box = 0, tot = 0;
    const uint32_t max_len = (1u << (8 * m.len_bytes)) - 1u;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = t * E + e;
        const uint4 b = i < c ? box[i] : make_uint4(0, 0, 0, 0);
        len[e] = min(min(b.y - b.x, b.w - b.z), max_len);
        if (!b.y) len[e] = 0;
        n_box += len[e] ? 1u : 0u;
    }
    uint32_t at = tm::excl_sum(n_box, S.tmp, tot), n = tot;
    uint32_t least = 1, ties = 0, tie = 0;  // boxes longer than `least` or among the first `ties` of it (none: all)
    if (m.N && tot > m.N) {
        uint32_t *hist = reinterpret_cast<uint32_t *>(S.key), *found = reinterpret_cast<uint32_t *>(S.tmp);
        uint32_t above = 0, top = 0;
        for (int shift = 8 * (m.len_bytes - 1); shift >= 0; shift -= 8) {
            for (int i = t; i < 256; i += T) hist[i] = 0;
            tm::sync();
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const bool in = len[e] && ((uint64_t)len[e] >> (shift + 8)) == top;
                const uint32_t bin = in ? (len[e] >> shift) & 0xFFu : 256u;
                const uint32_t peers = __match_any_sync(0xffffffffu, bin);
                if (in && (threadIdx.x & 31) == (uint32_t)(__ffs(peers) - 1)) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
            }
            tm::sync();
            if (t < 32) bin_of_nth(hist, m.N - above, found);
            tm::sync();
            top = (top << 8) | found[0];
            above += found[1];
            tm::sync();
        }
        least = top;
        ties = m.N - above;
        uint32_t n_eq = 0, n_gt = 0, all = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            n_eq += len[e] == least ? 1u : 0u;
            n_gt += len[e] > least ? 1u : 0u;
        }
        tie = tm::excl_sum(n_eq, S.tmp, all);
        at = tm::excl_sum(n_gt + min(n_eq, ties > tie ? ties - tie : 0u), S.tmp, all);
        n = m.N;
    } else {
        least = 0;
    }
    const uint32_t qi = m.in[m.perm ? m.perm[o] : o].qi;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (!len[e]) continue;
        const bool eq = len[e] == least;
        if (len[e] < least || (eq && tie++ >= ties)) continue;
        const uint32_t i = t * E + e;
        const uint4 b = box[i];
        m.out[o + at++] = DevHsp{qi, S.seq[i], b.x, b.y, b.z, b.w, min(b.y - b.x, b.w - b.z)};
    }
    if (t == 0) m.n_out[g] = n;
}

// groups of up to MG_WARP HSPs, a warp each (n_out of empty groups is 0 from the start)
template <bool STITCH>
__global__ void __launch_bounds__(256) k_merge_groups_warp(MergeGroups m, uint32_t G) {
    __shared__ MergeSmem<32, MG_WARP / 32> S[8];
    const uint32_t w = threadIdx.x >> 5, g = blockIdx.x * 8 + w;
    if (g >= G || m.cnt[g] == 0 || m.cnt[g] > MG_WARP) return;
    merge_group<32, MG_WARP / 32, STITCH>(m, g, S[w]);
}

// groups of list, a block each; dir: +1 from its front, -1 from its back
template <int T, int E, bool STITCH>
__global__ void __launch_bounds__(T) k_merge_groups(MergeGroups m, const uint32_t *__restrict__ list, int dir,
                                                    const uint32_t *__restrict__ n_list) {
    extern __shared__ unsigned char raw_smem[];
    MergeSmem<T, E> &S = *reinterpret_cast<MergeSmem<T, E> *>(raw_smem);
    const uint32_t n = *n_list;
    for (uint32_t x = blockIdx.x; x < n; x += gridDim.x) {
        merge_group<T, E, STITCH>(m, list[dir * (int64_t)x], S);
        __syncthreads();
    }
}

// Boxes of all groups back to back (pos: prefix sums of the groups' boxes), a warp a group; the
// first threads write each query's first box and the number that is selected of it (N = 0: qo;
// qfirst null: neither)
__global__ void __launch_bounds__(256) k_group_pack(const DevHsp *__restrict__ in, const uint64_t *__restrict__ off,
                                                    const uint64_t *__restrict__ pos, uint32_t G, GroupMap gm, uint32_t nq,
                                                    uint32_t N, DevHsp *__restrict__ out, uint32_t *__restrict__ qfirst,
                                                    uint32_t *__restrict__ cnt, uint64_t *__restrict__ qo) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, g = t >> 5;
    if (qfirst && t <= nq) {
        const uint64_t f = pos[gm.first(t)];
        qfirst[t] = (uint32_t)f;
        if (N == 0) qo[t] = f;
        else if (t < nq) cnt[t] = (uint32_t)min((uint64_t)N, pos[gm.first(t + 1)] - f);
    }
    if (g >= G) return;
    const uint64_t p = pos[g];
    const uint32_t words = (uint32_t)(pos[g + 1] - p) * HSP_WORDS;
    const uint32_t *from = reinterpret_cast<const uint32_t *>(in + off[g]);
    uint32_t *to = reinterpret_cast<uint32_t *>(out + p);
    for (uint32_t i = threadIdx.x & 31; i < words; i += 32) to[i] = from[i];
}

}  // namespace gn
