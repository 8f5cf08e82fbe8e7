// gn_search.cu - the search phases of the paper ("Searching process" section) on
// the device, for a batch of independent queries:
//   a5  input processing: rolling k-mer code of every query offset
//   a6  index lookup: gather of every occurrence of every code (hits)
//   a7  grouping: radix sort of hits by (diagonal key, query, query offset)
//   a8  merging of hits at most D apart on one (sequence, diagonal) into HSPs
//   a9  X-drop ungapped extension of both HSP ends
//   a10 merging of overlapped HSPs (single sweep per query and sequence)
//   a11 selection of the longest HSPs per query
//   a12 banded affine-gap Smith-Waterman of each selected HSP
//   a13 ranking by score, duplicate removal, e-value and bit score
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstddef>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <type_traits>

#include "gn_internal.cuh"

namespace gn {

// HSP record (7 words, same layout as gn_hsp)
struct DevHsp {
    uint32_t qi, seq, qs, qe, ds, de, len;
};
static_assert(sizeof(DevHsp) == 28, "DevHsp layout");
constexpr int HSP_WORDS = 7;
enum { W_QI = 0, W_SEQ = 1, W_QS = 2, W_QE = 3, W_DS = 4, W_DE = 5, W_LEN = 6 };

// alignment record (8 words)
struct DevAln {
    uint32_t qi, seq, qs, qe, ds, de;
    int32_t score;
    uint32_t pad;
};
static_assert(sizeof(DevAln) == 32, "DevAln layout");
constexpr int ALN_WORDS = 8;
enum { A_QI = 0, A_SEQ = 1, A_QS = 2, A_QE = 3, A_DS = 4, A_DE = 5, A_SCORE = 6 };

// ------------------------------------------------------ a5: query codes --
// Per global query offset x: query id and offset (qinfo = qi << 16 | qpos),
// k-mer code and the length of its occurrence list (0 for no window).
__global__ void k_query_codes(const uint64_t *__restrict__ qstart, uint32_t nq, uint64_t M,
                              const uint32_t *__restrict__ qpk, const uint32_t *__restrict__ qnb, SeedShape sh,
                              const uint64_t *__restrict__ off, uint32_t *__restrict__ codes,
                              uint32_t *__restrict__ qinfo, uint32_t *__restrict__ cnt,
                              uint32_t *__restrict__ src) {
    uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= M) return;
    uint32_t qi = dev_upper_index(qstart, nq + 1, x);
    uint64_t qpos = x - qstart[qi];
    uint64_t m = qstart[qi + 1] - qstart[qi];
    uint32_t c = 0, n = 0;
    uint64_t o = 0;
    if (qpos + (uint64_t)sh.span <= m && !dev_seed_has_nonbase(qnb, x, sh)) {
        c = dev_seed_code(qpk, x, sh);
        o = off[c];
        n = (uint32_t)(off[c + 1] - o);
    }
    codes[x] = c;
    qinfo[x] = (qi << 16) | (uint32_t)qpos;
    cnt[x] = n;
    src[x] = (uint32_t)o;  // occurrence indices fit 32 bits: the bank holds < 2^32 bases
}

// Seed hits of each query of a batch (request admission): one block per query sums the
// occurrence-list lengths of the seed codes of its offsets, read from ASCII bases.
__device__ __forceinline__ uint32_t ascii_base_code(uint8_t b) {
    const uint32_t c = b & 0xDFu;
    return c == 'A' ? 0u : c == 'C' ? 1u : c == 'G' ? 2u : (c == 'T' || c == 'U') ? 3u : 4u;
}

__global__ void __launch_bounds__(256) k_request_hits(const uint8_t *__restrict__ bases,
                                                      const uint64_t *__restrict__ start, uint32_t n, SeedShape sh,
                                                      const uint64_t *__restrict__ off,
                                                      unsigned long long *__restrict__ hits) {
    __shared__ unsigned long long part[8];
    for (uint32_t q = blockIdx.x; q < n; q += gridDim.x) {
        const uint64_t b0 = start[q], m = start[q + 1] - b0;
        unsigned long long sum = 0;
        for (uint64_t x = threadIdx.x; x + (uint64_t)sh.span <= m; x += blockDim.x) {
            uint32_t code = 0;
            bool ok = true;
            for (int p = 0; p < sh.span; ++p) {
                if (!((sh.keep >> p) & 1u)) continue;
                const uint32_t c = ascii_base_code(bases[b0 + x + p]);
                ok = ok && c < 4u;
                code = (code << 2) | (c & 3u);
            }
            if (ok) sum += off[code + 1] - off[code];
        }
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long t = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
            hits[q] = t;
        }
        __syncthreads();
    }
}

void count_request_hits(const gn_index *ix, const uint8_t *bases, const uint64_t *start, uint32_t n,
                        unsigned long long *hits, cudaStream_t s) {
    if (!n) return;
    GN_LAUNCH("k_request_hits", n, s,
              k_request_hits<<<(unsigned)std::min<uint32_t>(n, (uint32_t)num_sms() * 8), 256, 0, s>>>(
                  bases, start, n, seed_shape(ix), ix->off_d, hits));
}

__global__ void k_gather_u64(const uint64_t *__restrict__ src, const uint64_t *__restrict__ idx, uint32_t n,
                             uint64_t *__restrict__ out) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = src[idx[i]];
}

// ------------------------------------------------------- a6: seed gather --
// A warp takes 32 consecutive query offsets; their occurrence lists are
// copied one after another by the whole warp (coalesced reads of the list,
// coalesced writes of the hit keys).
// key = (gpos - qpos + QBIAS) << (16 + qbits) | (qi - qa) << 16 | qpos
__global__ void __launch_bounds__(256) k_seed_gather(const uint32_t *__restrict__ codes,
                                                     const uint32_t *__restrict__ qinfo,
                                                     const uint64_t *__restrict__ hoff, uint64_t xa, uint64_t xb,
                                                     uint64_t ha, const uint64_t *__restrict__ off,
                                                     const uint32_t *__restrict__ post, uint32_t qa, int qbits,
                                                     uint64_t *__restrict__ keys) {
    const int lane = threadIdx.x & 31;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (uint64_t x0 = xa + warp * 32; x0 < xb; x0 += nwarps * 32) {
        uint64_t x = x0 + lane;
        uint32_t my_cnt = 0;
        uint64_t my_src = 0, my_dst = 0, my_pref = 0;
        uint32_t my_qpos = 0;
        if (x < xb) {
            my_cnt = (uint32_t)(hoff[x + 1] - hoff[x]);
            if (my_cnt) {
                uint32_t qinf = qinfo[x];
                my_src = off[codes[x]];
                my_dst = hoff[x] - ha;
                my_qpos = qinf & 0xFFFFu;
                my_pref = ((uint64_t)((qinf >> 16) - qa) << 16) | my_qpos;
            }
        }
        uint32_t todo = __ballot_sync(0xffffffffu, my_cnt != 0);
        while (todo) {
            int src = __ffs(todo) - 1;
            todo &= todo - 1;
            uint32_t cnt = __shfl_sync(0xffffffffu, my_cnt, src);
            uint64_t sp = __shfl_sync(0xffffffffu, my_src, src);
            uint64_t dp = __shfl_sync(0xffffffffu, my_dst, src);
            uint64_t pref = __shfl_sync(0xffffffffu, my_pref, src);
            uint32_t qpos = __shfl_sync(0xffffffffu, my_qpos, src);
            for (uint32_t j = lane; j < cnt; j += 32) {
                uint64_t g = post[sp + j];
                uint64_t gkey = g + QBIAS - qpos;
                keys[dp + j] = (gkey << (16 + qbits)) | pref;
            }
        }
    }
}

// ------------------------------------------------------ a8: hit merging --
struct HitKey {
    uint64_t gkey;  // gpos - qpos + QBIAS
    uint32_t ql, qpos;
};

__device__ __forceinline__ HitKey dec_key(uint64_t key, int qbits) {
    HitKey h;
    h.qpos = (uint32_t)(key & 0xFFFFu);
    h.ql = (uint32_t)((key >> 16) & ((1ull << qbits) - 1ull));
    h.gkey = key >> (16 + qbits);
    return h;
}

// Chains of sorted hit keys: a hit starts a chain unless the previous key has the same
// diagonal and query, lies at most D query offsets before it and in the same bank
// sequence; the head walks its chain, whose hits must end before its sequence does.
__global__ void k_hit_merge(const uint64_t *__restrict__ keys, uint64_t n, int qbits, uint32_t qa, int k,
                            uint32_t D, uint32_t min_len, SeqMap sm, DevHsp *__restrict__ out,
                            uint32_t *__restrict__ count, uint32_t cap, uint32_t *__restrict__ status) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t key = keys[i];
        const HitKey a = dec_key(key, qbits);
        const uint64_t gpos = a.gkey - QBIAS + a.qpos;
        const uint32_t sq = dev_seq_of(sm, gpos);
        if (i > 0) {
            const uint64_t prev = keys[i - 1];
            const uint32_t qp = (uint32_t)(prev & 0xFFFFu);
            if ((prev >> 16) == (key >> 16) && a.qpos - qp <= D && sm.start[sq] <= gpos - (a.qpos - qp)) continue;
        }
        const uint64_t seq_end = sm.start[sq + 1];
        uint64_t j = i, kj = key;
        while (j + 1 < n) {
            const uint64_t kn = keys[j + 1];
            const uint32_t qn = (uint32_t)(kn & 0xFFFFu);
            if ((kn >> 16) != (key >> 16) || qn - (uint32_t)(kj & 0xFFFFu) > D || a.gkey - QBIAS + qn >= seq_end) break;
            kj = kn;
            ++j;
        }
        const uint32_t qs = a.qpos, qe = (uint32_t)(kj & 0xFFFFu) + (uint32_t)k;
        const uint32_t len = qe - qs;
        if (len < min_len) continue;
        const uint32_t ds = (uint32_t)(gpos - sm.start[sq]);
        const uint32_t slot = atomicAdd(count, 1u);
        if (slot < cap) {
            DevHsp h;
            h.qi = qa + a.ql; h.seq = sq; h.qs = qs; h.qe = qe; h.ds = ds; h.de = ds + len; h.len = len;
            out[slot] = h;
        } else {
            atomicOr(status, DEV_ERR_CAPACITY);
        }
    }
}

// ------------------------------------------ a6-a8: bucketed hit grouping --
// Hits of query i are partitioned into 2^b_i buckets by the high bits of their
// diagonal key G' = gpos - qpos + QBIAS (bucket = bbase[i] + (G' >> bshift[i])).
// Every (query, diagonal) lies in one bucket, so each bucket is grouped on its
// own.  A diagonal holding a single hit cannot form an HSP when min_hsp_len > k,
// so such hits are dropped before the (small) sort by (G', qpos) that the
// chaining needs.  Bucket entry: G' << 16 | qpos.

// Tile-level bucketing: a CTA takes tpos consecutive query offsets (the core).
// With the repeat filter on (min_hsp_len > k and D <= BT_MAX_D), every hit of the
// core and of the D offsets on either side (the halo) is first entered, by its
// (query, diagonal), into a shared-memory Bloom filter "seen" (three bits of one
// 32-bit word per key); a hit that finds all its bits set already enters its key
// into a second one, "seen twice" (two bits of one word).  A core hit can only be
// part of a chain of two or more hits if another hit lies on its diagonal within D
// query offsets, and all those offsets are inside core + halo; the later of two
// hits with one key always finds that key's "seen" bits set.  A Bloom filter has
// no false negatives, so a core hit whose "seen twice" bits are not all set cannot
// reach min_hsp_len and is dropped here; a false positive only keeps an extra hit.
constexpr int BT_MAX_D = 256;  // largest hit distance the tile filter supports

// The tile's occurrence lists are read in aligned quads of four entries (16-byte
// loads): the list of offset i, occurrences [beg_i, end_i), covers quads beg_i / 4
// to (end_i - 1) / 4 of the occurrence array, and the quads of all the tile's lists
// form one index space.  Warps take chunks of BF_QCHUNK quads from a shared counter
// (lane l holds quads c * BF_QCHUNK + 32 v + l, v < BF_QV), whatever lists they fall
// in, so every lane has work and a long list is shared by many warps.  A quad lies
// in one list; entries of a neighbouring list that share its 16 bytes are masked.
constexpr int BF_QV = 2;
constexpr int BF_QCHUNK = 32 * BF_QV;
constexpr int BF_CMAX = 512;  // chunks whose first list is tabulated (later ones are searched)
// Kept hits of a tile are staged in shared memory (stage_cap of them, the room the
// launch leaves) and placed in their buckets after the tile's placement pass, all
// threads at once, so that their global atomics overlap instead of stalling each warp's
// pass; hits past the stage's room are placed directly.
constexpr int BF_STAGE_BYTES = 14;  // per staged hit: key, bucket, query

// Key of a hit for the filters: the low 32 bits of its diagonal key G' mixed with its
// query (kadd = QBIAS - query offset, kx = query in chunk times an odd constant).
__device__ __forceinline__ uint32_t bf_key(uint32_t ent, uint32_t kadd, uint32_t kx) { return (ent + kadd) ^ kx; }
// Positions of a key in the two filters: the word of each from the top bits of one
// multiplicative (Fibonacci) hash, which spreads the keys of nearby diagonals over the
// words; the bits inside the word from 5-bit fields of the key itself, which differ
// between nearby diagonals.
__device__ __forceinline__ uint32_t bf_hash(uint32_t key) { return key * 0x9E3779B1u; }
// 1 << (x mod 32) in one funnel shift (the shift amount wraps modulo 32)
__device__ __forceinline__ uint32_t bit_of(uint32_t x) { return __funnelshift_l(0u, 1u, x); }
__device__ __forceinline__ uint32_t bf_mask(uint32_t key) {  // "seen": three bits
    return bit_of(key) | bit_of(key >> 5) | bit_of(key >> 10);
}
__device__ __forceinline__ uint32_t bf2_mask(uint32_t key) {  // "seen twice": two bits
    return bit_of(key >> 15) | bit_of(key >> 20);
}

// Shared-memory table of a tile's query offsets lo + i, i in [0, span): quad prefix
// relative to the tile's first quad (span + 1 entries), occurrence range [beg, end),
// (query in chunk << 16 | query offset), and the query's bucket base and shift;
// cs[c] is the offset holding quad c * BF_QCHUNK for the first BF_CMAX chunks.
// Tile-relative quad indices fit 32 bits: a query chunk holds < 2^32 hits.
struct TileTable {
    uint32_t *qp, *beg, *end, *qq, *bb, *cs;
    uint8_t *bs;
    uint32_t span, nchunks;
    uint64_t nquads;  // quads of the occurrence array (checked builds)
};

// Last table index i in [i_lo, i_hi] with qp[i] <= e: the offset whose list holds quad e.
__device__ __forceinline__ uint32_t tile_find(const uint32_t *qp, uint32_t i_lo, uint32_t i_hi, uint32_t e) {
    while (i_lo < i_hi) {
        const uint32_t mid = (i_lo + i_hi + 1) >> 1;
        if (qp[mid] <= e) i_lo = mid;
        else i_hi = mid - 1;
    }
    return i_lo;
}

__device__ __forceinline__ uint32_t tile_chunk_list(const TileTable &t, uint32_t c) {
    return c < BF_CMAX ? t.cs[c] : tile_find(t.qp, 0, t.span - 1, c * BF_QCHUNK);
}

// The BF_QV quads a lane holds of one chunk: entries (loads in flight until used),
// table index, occurrence index of the first entry, and whether the quad is inside
// the pass's quad range.
struct QuadLoad {
    uint4 ent[BF_QV];
    uint32_t idx[BF_QV], occ[BF_QV];
    bool ok[BF_QV];
};

// Issues the loads of chunk c, masked to the quad range [r0, r1): one search per lane
// for its first quad's list, then a boundary check per quad.
__device__ __forceinline__ void tile_quad_load(const TileTable &t, uint32_t c, uint32_t r0, uint32_t r1,
                                               const uint4 *__restrict__ post4, QuadLoad &L) {
    const int lane = threadIdx.x & 31;
    const uint32_t e0 = c * BF_QCHUNK + lane;
    const uint32_t i0 = tile_chunk_list(t, c);
    const uint32_t i1 = c + 1 < t.nchunks ? tile_chunk_list(t, c + 1) : t.span - 1;
    uint32_t i = tile_find(t.qp, i0, i1, e0);
    uint32_t nx = t.qp[i + 1];
#pragma unroll
    for (int v = 0; v < BF_QV; ++v) {
        const uint32_t e = e0 + 32u * v;
        while (e >= nx && i < i1) {  // the next non-empty list
            ++i;
            nx = t.qp[i + 1];
        }
        L.idx[v] = i;
        L.ok[v] = e >= r0 && e < r1;
        const uint32_t q = (t.beg[i] >> 2) + (e - t.qp[i]);
        L.occ[v] = q << 2;
        if (L.ok[v] && !GN_CHECK(q < t.nquads)) L.ok[v] = false;
        L.ent[v] = L.ok[v] ? __ldg(&post4[q]) : make_uint4(0u, 0u, 0u, 0u);
    }
}

// Calls f(L) for every chunk of quads meeting [r0, r1) (tile-relative quad indices);
// all lanes of a warp call f together.  A warp issues the loads of its next chunk
// before it processes the current one.
template <class F>
__device__ __forceinline__ void for_tile_quads(const TileTable &t, uint32_t r0, uint32_t r1, uint32_t *ctr,
                                               const uint4 *__restrict__ post4, F &&f) {
    const int lane = threadIdx.x & 31;
    if (r0 >= r1) return;
    const uint32_t c0 = r0 / BF_QCHUNK, nc = (r1 + BF_QCHUNK - 1) / BF_QCHUNK - c0;
    auto claim = [&]() {
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(ctr, 1u);
        return __shfl_sync(0xffffffffu, c, 0);
    };
    uint32_t c = claim();
    if (c >= nc) return;
    QuadLoad cur, nxt;
    tile_quad_load(t, c0 + c, r0, r1, post4, cur);
    for (;;) {
        const uint32_t cn = claim();
        const bool more = cn < nc;
        if (more) tile_quad_load(t, c0 + cn, r0, r1, post4, nxt);
        f(cur);
        if (!more) break;
        cur = nxt;
    }
}

__device__ __forceinline__ uint32_t quad_word(const uint4 &q, int u) {
    return u == 0 ? q.x : u == 1 ? q.y : u == 2 ? q.z : q.w;
}

// Exclusive scan of one value per thread over the block (blockDim.x a multiple of 32,
// at most 1,024); wtot holds 32 words of shared memory.
__device__ __forceinline__ uint32_t bf_block_scan(uint32_t v, uint32_t *wtot, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? wtot[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) wtot[lane] = w;
    }
    __syncthreads();
    total = wtot[nw - 1];
    const uint32_t before = warp ? wtot[warp - 1] : 0u;
    __syncthreads();  // wtot is reused by the next call
    return before + x - v;
}

// Places one kept hit (key = G' << 16 | query offset, ql = query in chunk) in bucket b:
// a global atomic reserves its slot; past the bucket's capacity it goes to the spill
// list in global hit-key format.
__device__ __forceinline__ void bucket_place(uint32_t b, uint64_t key, uint32_t ql, uint32_t *__restrict__ bcount,
                                             uint64_t *__restrict__ bkeys, uint32_t bcap, uint64_t *__restrict__ spill,
                                             unsigned long long *__restrict__ spill_count,
                                             unsigned long long spill_cap, int qbits, uint32_t NB) {
    if (!GN_CHECK(b < NB)) return;
    const uint32_t slot = atomicAdd(&bcount[b], 1u);
    if (slot < bcap) {
        bkeys[(uint64_t)b * bcap + slot] = key;
    } else {
        const unsigned long long at = atomicAdd(spill_count, 1ull);
        if (at < spill_cap) spill[at] = ((key >> 16) << (16 + qbits)) | ((uint64_t)ql << 16) | (key & 0xFFFFu);
    }
}

// Bucket fill: one kernel per query chunk.  Each tile (tpos core offsets) enters the
// hits of core + halo into the "seen" / "seen twice" filters (repeat filter), then
// places every kept core hit: one global atomic reserves its slot in its bucket.
// Buckets have a fixed capacity bcap; hits past it go to the spill list in global
// hit-key format, which the global sort path handles.  count_only: no placement,
// kept_total[0] counts the kept core hits and kept_total[1] all core hits of the
// tiles visited (tiles 0, tile_step, 2 tile_step, ...).  kept_total[2] hands out the
// tiles (zero at launch).
// FB, FB2: the filters' sizes in bits as constants (0: the run-time fbits, fbits2).
template <int FB, int FB2>
__global__ void __launch_bounds__(512, 2) k_bucket_fill(
    const uint32_t *__restrict__ qinfo, const uint32_t *__restrict__ src, const uint64_t *__restrict__ hoff,
    uint64_t xa, uint64_t xb, const uint32_t *__restrict__ post, uint32_t qa, const uint32_t *__restrict__ bbase,
    const uint32_t *__restrict__ bshift, uint32_t *__restrict__ bcount, uint64_t *__restrict__ bkeys, uint32_t bcap,
    uint64_t *__restrict__ spill, unsigned long long *__restrict__ spill_count, unsigned long long spill_cap,
    int qbits, int filter, uint32_t D, int tpos, int fbits, int fbits2, unsigned long long *__restrict__ kept_total,
    uint32_t tile_step, int count_only, uint32_t stage_cap, uint32_t NB, uint64_t post_quads) {
    extern __shared__ __align__(16) unsigned char bf_smem[];
    const uint32_t halo = filter ? D : 0u;
    const uint32_t span_max = (uint32_t)tpos + 2u * halo;
    const int wbits = (FB ? FB : fbits) - 5, wbits2 = (FB2 ? FB2 : fbits2) - 5;
    const uint32_t nwords = filter ? 1u << wbits : 0u, nwords2 = filter ? 1u << wbits2 : 0u;
    const uint4 *__restrict__ post4 = reinterpret_cast<const uint4 *>(post);
    uint64_t *stage_key = reinterpret_cast<uint64_t *>(bf_smem);  // G' << 16 | query offset
    uint32_t *seen = reinterpret_cast<uint32_t *>(stage_key + stage_cap);
    uint32_t *seen2 = seen + nwords;
    TileTable t;
    t.nquads = post_quads;
    t.qp = seen2 + nwords2;
    t.beg = t.qp + span_max + 1;
    t.end = t.beg + span_max;
    t.qq = t.end + span_max;
    t.bb = t.qq + span_max;
    t.cs = t.bb + span_max;
    uint32_t *stage_b = t.cs + BF_CMAX;                                 // bucket
    uint16_t *stage_q = reinterpret_cast<uint16_t *>(stage_b + stage_cap);  // query in chunk
    t.bs = reinterpret_cast<uint8_t *>(stage_q + stage_cap);
    __shared__ uint32_t ctr, nstage;
    __shared__ uint32_t wtot[32];
    uint32_t my_kept = 0;
    unsigned long long my_core = 0;  // core hits of the visited tiles (count-only runs)
    // tiles from a counter (kept_total[2]): blocks that drew small tiles take more
    __shared__ uint64_t s_t0;
    for (;;) {
        if (threadIdx.x == 0) s_t0 = xa + atomicAdd(kept_total + 2, 1ull) * tile_step * (uint64_t)tpos;
        __syncthreads();
        const uint64_t t0 = s_t0;
        if (t0 >= xb) break;
        const uint64_t t1 = min(xb, t0 + (uint64_t)tpos);
        const uint64_t lo = t0 - xa > halo ? t0 - halo : xa, hi = min(xb, t1 + halo);
        const uint32_t span = (uint32_t)(hi - lo);
        // per-offset table; quad counts first, then their exclusive scan in place
        for (uint32_t i = threadIdx.x; i < span; i += blockDim.x) {
            const uint64_t x = lo + i;
            const uint32_t b = src[x], n = (uint32_t)(hoff[x + 1] - hoff[x]);
            t.beg[i] = b;
            t.end[i] = b + n;
            t.qp[i] = n ? ((b + n + 3u) >> 2) - (b >> 2) : 0u;
            const uint32_t qinf = qinfo[x];
            const uint32_t ql = (qinf >> 16) - qa;
            t.qq[i] = (ql << 16) | (qinf & 0xFFFFu);
            t.bb[i] = bbase[ql];
            t.bs[i] = (uint8_t)bshift[ql];
        }
        for (uint32_t i = threadIdx.x; i < nwords + nwords2; i += blockDim.x) seen[i] = 0u;
        if (threadIdx.x == 0) ctr = nstage = 0;
        if (count_only && threadIdx.x == 0) my_core += hoff[t1] - hoff[t0];
        __syncthreads();
        {
            const uint32_t per = (span + blockDim.x - 1) / blockDim.x;
            const uint32_t a = min(span, threadIdx.x * per), b = min(span, a + per);
            uint32_t sum = 0;
            for (uint32_t i = a; i < b; ++i) sum += t.qp[i];
            uint32_t total = 0;
            uint32_t run = bf_block_scan(sum, wtot, total);
            for (uint32_t i = a; i < b; ++i) {
                const uint32_t nq = t.qp[i];
                t.qp[i] = run;
                run += nq;
            }
            if (threadIdx.x == 0) t.qp[span] = total;
        }
        __syncthreads();
        t.span = span;
        t.nchunks = (t.qp[span] + BF_QCHUNK - 1) / BF_QCHUNK;
        // chunk -> offset of its first quad
        for (uint32_t i = threadIdx.x; i < span; i += blockDim.x) {
            const uint32_t ca = (t.qp[i] + BF_QCHUNK - 1) / BF_QCHUNK;
            const uint32_t cb = min((t.qp[i + 1] + BF_QCHUNK - 1) / BF_QCHUNK, (uint32_t)BF_CMAX);
            for (uint32_t c = ca; c < cb; ++c) t.cs[c] = i;
        }
        __syncthreads();
        if (filter) {
            for_tile_quads(t, 0, t.qp[span], &ctr, post4, [&](const QuadLoad &L) {
#pragma unroll
                for (int v = 0; v < BF_QV; ++v) {
                    if (!L.ok[v]) continue;
                    const uint32_t qq = t.qq[L.idx[v]];
                    const uint32_t kadd = QBIAS - (qq & 0xFFFFu), kx = (qq >> 16) * 0x85EBCA77u;
                    // entries of a neighbouring list that share the quad are entered too: an
                    // extra key can only add false positives
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t key = bf_key(quad_word(L.ent[v], u), kadd, kx);
                        const uint32_t h = bf_hash(key), m = bf_mask(key);
                        const uint32_t old = atomicOr(&seen[h >> (32 - wbits)], m);
                        if ((old & m) == m) atomicOr(&seen2[h >> (32 - wbits2)], bf2_mask(key));
                    }
                }
            });
            __syncthreads();
            if (threadIdx.x == 0) ctr = 0;
            __syncthreads();
        }
        // place the kept core hits (count them only, when sampling the keep rate)
        for_tile_quads(t, t.qp[t0 - lo], t.qp[t1 - lo], &ctr, post4, [&](const QuadLoad &L) {
#pragma unroll
            for (int v = 0; v < BF_QV; ++v) {
                if (!L.ok[v]) continue;
                const uint32_t i = L.idx[v], qq = t.qq[i], beg = t.beg[i], end = t.end[i], occ = L.occ[v];
                // entries of this list in the quad: from beg - occ (first quad) to end - occ (last)
                const uint32_t first = occ < beg ? beg - occ : 0u, last = end - occ < 4u ? end - occ : 4u;
                uint32_t keep = (0xFu >> (4u - last)) & (0xFu << first);  // bit u: entry u is a kept hit
                if (filter) {
                    const uint32_t kadd = QBIAS - (qq & 0xFFFFu), kx = (qq >> 16) * 0x85EBCA77u;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t key = bf_key(quad_word(L.ent[v], u), kadd, kx);
                        const uint32_t m2 = bf2_mask(key);
                        if ((seen2[bf_hash(key) >> (32 - wbits2)] & m2) != m2) keep &= ~(1u << u);
                    }
                }
                if (!keep) continue;
                my_kept += __popc(keep);
                if (count_only) continue;
                const uint32_t bb = t.bb[i], bs = t.bs[i];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (!(keep >> u & 1u)) continue;
                    const uint64_t gk = (uint64_t)quad_word(L.ent[v], u) + QBIAS - (qq & 0xFFFFu);
                    const uint32_t b = bb + (uint32_t)(gk >> bs);
                    const uint64_t key = (gk << 16) | (qq & 0xFFFFu);
                    const uint32_t at = atomicAdd(&nstage, 1u);
                    if (at < stage_cap) {
                        stage_key[at] = key;
                        stage_b[at] = b;
                        stage_q[at] = (uint16_t)(qq >> 16);
                    } else {
                        bucket_place(b, key, qq >> 16, bcount, bkeys, bcap, spill, spill_count, spill_cap, qbits,
                                     NB);
                    }
                }
            }
        });
        if (!count_only) {
            __syncthreads();
            const uint32_t ns = min(nstage, stage_cap);
            for (uint32_t j = threadIdx.x; j < ns; j += blockDim.x)
                bucket_place(stage_b[j], stage_key[j], stage_q[j], bcount, bkeys, bcap, spill, spill_count, spill_cap,
                             qbits, NB);
        }
        __syncthreads();  // the table and filters are rebuilt for the next tile
    }
    if (my_kept) atomicAdd(kept_total, (unsigned long long)my_kept);
    if (my_core) atomicAdd(kept_total + 1, my_core);
}

// Dynamic shared memory of k_bucket_fill: staged kept hits, filters, offset table.
static size_t bucket_fill_smem(int tpos, uint32_t halo, int filter, int fbits, int fbits2, uint32_t stage_cap) {
    const size_t span_max = (size_t)tpos + 2 * halo;
    return (size_t)stage_cap * BF_STAGE_BYTES + (filter ? ((1u << fbits) + (1u << fbits2)) / 8 : 0) +
           (span_max + 1) * 4 + span_max * 17 + 4 * BF_CMAX;
}

__global__ void k_bucket_query(const uint32_t *__restrict__ bbase, uint32_t nqc, uint32_t NB,
                               uint16_t *__restrict__ bq) {
    uint32_t q = blockIdx.x;
    if (q >= nqc) return;
    for (uint32_t b = bbase[q] + threadIdx.x; b < bbase[q + 1]; b += blockDim.x) bq[b] = (uint16_t)q;
}

// Chains of candidates sorted by (G', qpos) within one bucket (one query): candidate i
// starts a chain unless candidate i - 1 has the same diagonal, lies at most D query
// offsets before it and in the same bank sequence.  The threads of a warp (NW = 1) or of
// a block mark the chain heads in a bitmask (words at heads[], one per 32 candidates);
// each head's chain ends before the next head, and an HSP is emitted for every chain of
// length >= min_len.  Threads are tid, tid + nthreads, ...; sync() orders the two steps.
template <class Sync>
__device__ __forceinline__ void chain_emit(const uint64_t *cand, uint32_t nc, uint32_t *heads, uint32_t tid,
                                           uint32_t nthreads, Sync sync, uint32_t ql, uint32_t qa, int k, uint32_t D,
                                           uint32_t min_len, const SeqMap &sm, DevHsp *__restrict__ out,
                                           uint32_t *__restrict__ count, uint32_t out_cap,
                                           uint32_t *__restrict__ status) {
    const uint32_t nw = (nc + 31) / 32;
    for (uint32_t i0 = tid & ~31u; i0 < nw * 32; i0 += nthreads) {
        const uint32_t i = i0 + (tid & 31);
        bool head = false;
        if (i < nc) {
            const uint64_t key = cand[i];
            const uint32_t qs = (uint32_t)(key & 0xFFFFu);
            const uint64_t gpos = (key >> 16) - QBIAS + qs;
            head = true;
            if (i > 0) {
                const uint64_t prev = cand[i - 1];
                const uint32_t qp = (uint32_t)(prev & 0xFFFFu);
                if ((prev >> 16) == (key >> 16) && qs - qp <= D) {
                    const uint32_t sq = dev_seq_of(sm, gpos);
                    head = sm.start[sq] > gpos - (qs - qp);  // a sequence starts between them
                }
            }
        }
        const uint32_t m = __ballot_sync(0xffffffffu, head);
        if ((tid & 31) == 0) heads[i0 / 32] = m;
    }
    sync();
    for (uint32_t i = tid; i < nc; i += nthreads) {
        if (!((heads[i / 32] >> (i & 31)) & 1u)) continue;
        // the next head after i
        uint32_t w = i / 32, rest = heads[w] & ~((2u << (i & 31)) - 1u);
        while (!rest && ++w < nw) rest = heads[w];
        const uint32_t end = (rest ? w * 32 + (uint32_t)(__ffs(rest) - 1) : nc) - 1;
        const uint64_t key = cand[i], kj = cand[end];
        const uint32_t qs = (uint32_t)(key & 0xFFFFu), qe = (uint32_t)(kj & 0xFFFFu) + (uint32_t)k;
        const uint32_t len = qe - qs;
        if (len < min_len) continue;
        const uint64_t gpos = (key >> 16) - QBIAS + qs;
        const uint32_t sq = dev_seq_of(sm, gpos);
        const uint32_t ds = (uint32_t)(gpos - sm.start[sq]);
        const uint32_t slot = atomicAdd(count, 1u);
        if (slot < out_cap) {
            DevHsp hh;
            hh.qi = qa + ql; hh.seq = sq; hh.qs = qs; hh.qe = qe; hh.ds = ds; hh.de = ds + len; hh.len = len;
            out[slot] = hh;
        } else {
            atomicOr(status, DEV_ERR_CAPACITY);
        }
    }
}
struct WarpSync {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};
struct BlockSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// One warp per bucket.  Two bitmaps per warp mark diagonal hashes seen once and
// seen twice; hits whose hash was seen twice are candidates (a hash collision
// only adds a candidate that the exact chaining below then drops).  Candidates
// are sorted by (G', qpos) with a warp bitonic sort and chained.  Buckets with
// more than BGW_CAND candidates go to the global sort path.
constexpr int BGW_WARPS = 8;
constexpr int BGW_BITS = 8192;
constexpr int BGW_CAND = 256;
constexpr int BGC_CAND = 1024;  // entries a block-level bucket group takes

__global__ void __launch_bounds__(BGW_WARPS * 32) k_bucket_group_warp(
    const uint64_t *__restrict__ bkeys, const uint32_t *__restrict__ bcount, uint32_t bcap, uint32_t NB,
    const uint16_t *__restrict__ bq, uint32_t qa, int qbits, int k, uint32_t D, uint32_t min_len, int singles,
    SeqMap sm, DevHsp *__restrict__ out, uint32_t *__restrict__ count,
    uint32_t out_cap, uint64_t *__restrict__ ovf, unsigned long long ovf_cap,
    unsigned long long *__restrict__ ovf_count, uint32_t *__restrict__ status, uint32_t *__restrict__ next_bucket,
    uint32_t *__restrict__ big, uint32_t *__restrict__ big_count) {
    extern __shared__ __align__(16) unsigned char gw_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t *seen = reinterpret_cast<uint32_t *>(gw_smem) + wib * (2 * BGW_BITS / 32);
    uint32_t *seen2 = seen + BGW_BITS / 32;
    uint64_t *cand = reinterpret_cast<uint64_t *>(gw_smem + BGW_WARPS * 2 * BGW_BITS / 8) + wib * BGW_CAND;
    uint32_t *heads = reinterpret_cast<uint32_t *>(gw_smem + BGW_WARPS * (2 * BGW_BITS / 8 + BGW_CAND * 8)) +
                      wib * (BGW_CAND / 32);
    const uint32_t lt = (1u << lane) - 1u;
    for (;;) {
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(next_bucket, 1u);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b >= NB) break;
        const uint64_t beg = (uint64_t)b * bcap;
        const uint32_t total = bcount[b];
        const uint32_t n = min(total, bcap);
        if (total <= bcap && (n == 0 || (n == 1 && !singles))) continue;
        const uint32_t ql = bq[b];
        // a bucket that overflowed its capacity has entries in the spill list already: send the
        // stored part there as well, so that every (query, diagonal) stays on one path
        bool spill = total > bcap;
        uint32_t nc = 0;
        if (!singles && !spill) {
            for (int i = lane; i < BGW_BITS / 32; i += 32) { seen[i] = 0u; seen2[i] = 0u; }
            __syncwarp();
            for (uint32_t i0 = 0; i0 < n; i0 += 128) {
                uint64_t e[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = i0 + u * 32 + lane;
                    e[u] = i < n ? bkeys[beg + i] : 0ull;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (i0 + u * 32 + lane >= n) break;
                    const uint32_t h = (uint32_t)(((e[u] >> 16) * 0x9E3779B97F4A7C15ull) >> 51);  // 13 bits
                    const uint32_t bit = 1u << (h & 31);
                    const uint32_t old = atomicOr(&seen[h >> 5], bit);
                    if (old & bit) atomicOr(&seen2[h >> 5], bit);
                }
            }
            __syncwarp();
        }
        for (uint32_t i0 = 0; i0 < n && !spill; i0 += 32) {
            const uint32_t i = i0 + lane;
            uint64_t key = 0;
            bool keep = false;
            if (i < n) {
                key = bkeys[beg + i];
                if (singles) {
                    keep = true;
                } else {
                    const uint32_t h = (uint32_t)(((key >> 16) * 0x9E3779B97F4A7C15ull) >> 51);  // 13 bits
                    keep = (seen2[h >> 5] >> (h & 31)) & 1u;
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (nc + __popc(m) > BGW_CAND) {
                if (n <= BGC_CAND) {  // the block kernel takes it
                    if (lane == 0) big[atomicAdd(big_count, 1u)] = b;
                    nc = 0;
                    break;
                }
                spill = true;
            } else {
                if (keep) cand[nc + __popc(m & lt)] = key;
                nc += __popc(m);
            }
        }
        if (spill) {
            // too many candidates: hand the bucket to the global sort path, in its key format
            unsigned long long p0 = 0;
            if (lane == 0) p0 = atomicAdd(ovf_count, (unsigned long long)n);
            p0 = __shfl_sync(0xffffffffu, p0, 0);
            if (p0 + n <= ovf_cap) {  // else: counted only; the host enlarges the buffer and reruns
                for (uint32_t i = lane; i < n; i += 32) {
                    const uint64_t e = bkeys[beg + i];
                    ovf[p0 + i] = ((e >> 16) << (16 + qbits)) | ((uint64_t)ql << 16) | (e & 0xFFFFu);
                }
            }
            __syncwarp();
            continue;
        }
        if (nc < 2 && !singles) { __syncwarp(); continue; }
        if (nc == 0) { __syncwarp(); continue; }
        uint32_t P = 1;
        while (P < nc) P <<= 1;
        for (uint32_t i = nc + lane; i < P; i += 32) cand[i] = ~0ull;
        __syncwarp();
        for (uint32_t k2 = 2; k2 <= P; k2 <<= 1) {
            for (uint32_t j = k2 >> 1; j > 0; j >>= 1) {
                for (uint32_t i = lane; i < P; i += 32) {
                    const uint32_t ixj = i ^ j;
                    if (ixj > i) {
                        const uint64_t a = cand[i], c = cand[ixj];
                        const bool up = (i & k2) == 0;
                        if ((a > c) == up) { cand[i] = c; cand[ixj] = a; }
                    }
                }
                __syncwarp();
            }
        }
        chain_emit(cand, nc, heads, lane, 32, WarpSync(), ql, qa, k, D, min_len, sm, out, count, out_cap, status);
        __syncwarp();
    }
}

// Exclusive prefix sum of v over the block (all threads call it); *total gets the sum.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *warp_tot, uint32_t &total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t t = lane < nw ? warp_tot[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) warp_tot[lane] = t;  // inclusive warp prefix
    }
    __syncthreads();
    total = warp_tot[nw - 1];
    const uint32_t before = wid ? warp_tot[wid - 1] : 0u;
    __syncthreads();  // warp_tot is reused by the next call
    return before + x - v;
}

// One block per bucket that has more candidates than a warp holds (at most BGC_CAND
// entries in all): the same filter, sort and chaining as k_bucket_group_warp, over
// the whole block.  Blocks take the listed buckets in turn.
__global__ void __launch_bounds__(256) k_bucket_group_block(
    const uint64_t *__restrict__ bkeys, const uint32_t *__restrict__ bcount, uint32_t bcap,
    const uint16_t *__restrict__ bq, const uint32_t *__restrict__ big, const uint32_t *__restrict__ big_count,
    uint32_t qa, int k, uint32_t D, uint32_t min_len, int singles, SeqMap sm, DevHsp *__restrict__ out,
    uint32_t *__restrict__ count, uint32_t out_cap, uint32_t *__restrict__ status) {
    __shared__ uint32_t seen[BGW_BITS / 32], seen2[BGW_BITS / 32];
    __shared__ uint64_t cand[BGC_CAND];
    __shared__ uint32_t heads[BGC_CAND / 32];
    __shared__ uint32_t warp_tot[8];
    const uint32_t nbig = *big_count;
    for (uint32_t j = blockIdx.x; j < nbig; j += gridDim.x) {
        const uint32_t b = big[j];
        const uint64_t beg = (uint64_t)b * bcap;
        const uint32_t n = min(bcount[b], bcap);
        const uint32_t ql = bq[b];
        for (uint32_t i = threadIdx.x; i < BGW_BITS / 32; i += blockDim.x) { seen[i] = 0u; seen2[i] = 0u; }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t h = (uint32_t)(((bkeys[beg + i] >> 16) * 0x9E3779B97F4A7C15ull) >> 51);  // 13 bits
            const uint32_t bit = 1u << (h & 31);
            const uint32_t old = atomicOr(&seen[h >> 5], bit);
            if (old & bit) atomicOr(&seen2[h >> 5], bit);
        }
        __syncthreads();
        uint32_t nc = 0;
        for (uint32_t i0 = 0; i0 < n; i0 += blockDim.x) {
            const uint32_t i = i0 + threadIdx.x;
            uint64_t key = 0;
            bool keep = false;
            if (i < n) {
                key = bkeys[beg + i];
                const uint32_t h = (uint32_t)(((key >> 16) * 0x9E3779B97F4A7C15ull) >> 51);
                keep = singles || ((seen2[h >> 5] >> (h & 31)) & 1u);
            }
            uint32_t tot = 0;
            const uint32_t pos = nc + block_excl_scan(keep ? 1u : 0u, warp_tot, tot);
            if (keep) cand[pos] = key;
            nc += tot;
        }
        uint32_t P = 1;
        while (P < nc) P <<= 1;
        for (uint32_t i = nc + threadIdx.x; i < P; i += blockDim.x) cand[i] = ~0ull;
        __syncthreads();
        for (uint32_t k2 = 2; k2 <= P; k2 <<= 1) {
            for (uint32_t jj = k2 >> 1; jj > 0; jj >>= 1) {
                for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) {
                    const uint32_t ixj = i ^ jj;
                    if (ixj > i) {
                        const uint64_t x = cand[i], y = cand[ixj];
                        if ((x > y) == ((i & k2) == 0)) { cand[i] = y; cand[ixj] = x; }
                    }
                }
                __syncthreads();
            }
        }
        chain_emit(cand, nc, heads, threadIdx.x, blockDim.x, BlockSync(), ql, qa, k, D, min_len, sm, out, count,
                   out_cap, status);
        __syncthreads();
    }
}

// quadruples (query, qpos, seq, pos) of sorted hits (tests)
__global__ void k_decode_hits(const uint64_t *__restrict__ keys, uint64_t n, int qbits, uint32_t qa,
                              const uint64_t *__restrict__ seq_start, uint32_t n_seqs, uint32_t *__restrict__ out) {
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    HitKey h = dec_key(keys[i], qbits);
    uint64_t gpos = h.gkey - QBIAS + h.qpos;
    uint32_t sq = dev_upper_index(seq_start, n_seqs + 1, gpos);
    out[4 * i + 0] = qa + h.ql;
    out[4 * i + 1] = h.qpos;
    out[4 * i + 2] = sq;
    out[4 * i + 3] = (uint32_t)(gpos - seq_start[sq]);
}

// --------------------------------------------------- a9: X-drop extension --
__device__ __forceinline__ int32_t dev_pair(uint32_t a, uint32_t b, int32_t match, int32_t mismatch) {
    return (a < 4u && a == b) ? match : mismatch;
}

// 16 bases from position p (p >= -16; bases before 0 read as code 0, non-base): 2-bit
// codes with base p in bits 31-30, and a mask with bit i set when base p + i is a non-base.
// The packed arrays carry two words past the last base, so p + 15 may pass the end.
__device__ __forceinline__ void base_window16(const uint32_t *__restrict__ pk, const uint32_t *__restrict__ nb,
                                             int64_t p, uint32_t &codes, uint32_t &bad) {
    const int64_t a = p >> 4, b = p >> 5;  // floor division
    const uint32_t w0 = a >= 0 ? pk[a] : 0u, w1 = pk[a + 1];
    const uint32_t off = (uint32_t)(p & 15);
    codes = (uint32_t)((((uint64_t)w0 << 32) | w1) >> (32 - 2 * off));
    const uint32_t n0 = b >= 0 ? nb[b] : 0xFFFFFFFFu, n1 = nb[b + 1];
    bad = (uint32_t)(((((uint64_t)n1) << 32) | n0) >> (uint32_t)(p & 31)) & 0xFFFFu;
}

// 32 bases from position p (any sign), first one on top, and their non-base bits from bit 0;
// words outside the array are clamped (the caller takes nothing from their positions).
__device__ __forceinline__ uint64_t window32(const uint32_t *__restrict__ pk, const uint32_t *__restrict__ nb, int64_t p,
                                             int64_t last_pk, int64_t last_nb, uint32_t &bad) {
    const int64_t a = p >> 4, b = p >> 5;
    const uint32_t w0 = pk[max((int64_t)0, min(a, last_pk))], w1 = pk[max((int64_t)0, min(a + 1, last_pk))];
    const uint32_t w2 = pk[max((int64_t)0, min(a + 2, last_pk))];
    const uint32_t n0 = nb[max((int64_t)0, min(b, last_nb))], n1 = nb[max((int64_t)0, min(b + 1, last_nb))];
    const uint32_t s = 2u * (uint32_t)(p & 15);
    bad = __funnelshift_r(n0, n1, (uint32_t)(p & 31));
    return (uint64_t)__funnelshift_l(w1, w0, s) << 32 | __funnelshift_l(w2, w1, s);
}

// Bit i of the low 16 bits of x to bits 31 - 2 i and 30 - 2 i.
__device__ __forceinline__ uint32_t spread16_down(uint32_t x) {
    x &= 0xFFFFu;
    x = (x | x << 8) & 0x00FF00FFu;
    x = (x | x << 4) & 0x0F0F0F0Fu;
    x = (x | x << 2) & 0x33333333u;
    x = (x | x << 1) & 0x55555555u;  // bit 2 i
    return __brev(x * 3u);
}
// Packed sequences of a search.
struct PackedPair {
    const uint32_t *qpk, *qnb, *bpk, *bnb;
    int64_t last_qpk, last_qnb, last_bpk, last_bnb;  // last words
};

// Bits 31 - 2 i and 30 - 2 i of w[j]: bases 16 j + i of the windows at q and d are equal bases
// (codes agree, no non-base); both windows start inside their arrays or, at the front, before
// them (base positions below 0 come out as anything).
__device__ __forceinline__ void equal32(const PackedPair &s, int64_t q, int64_t d, uint32_t w[2]) {
    uint32_t qb, db;
    uint64_t y;
    if (q >= 0 && d >= 0) {  // two words past the last base are there, so nothing needs a limit
        const uint32_t *a = s.qpk + (q >> 4), *b = s.bpk + (d >> 4), *m = s.qnb + (q >> 5), *n = s.bnb + (d >> 5);
        const uint32_t a0 = a[0], a1 = a[1], a2 = a[2], b0 = b[0], b1 = b[1], b2 = b[2];
        const uint32_t m0 = m[0], m1 = m[1], n0 = n[0], n1 = n[1];
        const uint32_t sq = 2u * (uint32_t)(q & 15), sd = 2u * (uint32_t)(d & 15);
        w[0] = __funnelshift_l(a1, a0, sq) ^ __funnelshift_l(b1, b0, sd);
        w[1] = __funnelshift_l(a2, a1, sq) ^ __funnelshift_l(b2, b1, sd);
        qb = __funnelshift_r(m0, m1, (uint32_t)(q & 31));
        db = __funnelshift_r(n0, n1, (uint32_t)(d & 31));
    } else {
        y = window32(s.qpk, s.qnb, q, s.last_qpk, s.last_qnb, qb) ^ window32(s.bpk, s.bnb, d, s.last_bpk, s.last_bnb, db);
        w[0] = (uint32_t)(y >> 32);
        w[1] = (uint32_t)y;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const uint32_t e = ~(w[j] | w[j] >> 1) & 0x55555555u;
        w[j] = e | e << 1;
    }
    if (qb | db) {
        w[0] &= ~spread16_down(qb | db);
        w[1] &= ~spread16_down((qb | db) >> 16);
    }
}

// X-drop extension.  The rule, step e = 1, 2, .. out from an HSP's end: score += s; if score >
// best: best = score, ext = e; else if best - score > X: stop.  Within a run of matches the
// best is at its end, and within a run of mismatches only the drop after the last one matters,
// so a walk takes one step per run, from 32 bases' equality bits at a time (left windows are
// mirrored).  A lane takes one end of an HSP.  Walks are mostly one window long and sometimes,
// inside a repeat, hundreds, so a lane whose walk has ended waits only until XD_REFILL lanes of its
// warp have, and then gets a new one from the counter.  Writes the end's two words; len is left
// to whoever needs it.  Bound by the latency of each end's first window, whose place is random.
// Measured against a step per base with 32 HSPs a warp, whose walks over 64 steps the warp
// continued one by one: 2.1 M HSPs on 4 Gbp 1.07 -> 0.35 ms, 103,000 on 400 Mbp 0.43 -> 0.08,
// 177,000 of chromosome-scale queries 0.49 -> 0.12.  Refill at 8, 16, 24 lanes: 0.43, 0.40, 0.35.
constexpr int XD_REFILL = 24;

__global__ void __launch_bounds__(256) k_xdrop(DevHsp *__restrict__ h, uint32_t n, PackedPair seq,
                                               const uint64_t *__restrict__ qstart,
                                               const uint64_t *__restrict__ seq_start, int32_t match, int32_t mismatch,
                                               int32_t X, uint32_t nq, uint32_t n_seqs,
                                               unsigned long long *__restrict__ next_end) {
    const int lane = threadIdx.x & 31;
    const uint64_t ends = 2ull * n;
    bool more = true;    // the counter has not run out
    bool open = false;   // the lane's walk goes on
    uint64_t item = 0;   // HSP << 1 | right end
    uint32_t e = 0, emax = 0, ext = 0;
    int64_t q = 0, d = 0;
    int32_t score = 0, best = 0;
    for (;;) {
        const uint32_t idle = __ballot_sync(0xffffffffu, !open);
        if (more && __popc(idle) >= XD_REFILL) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(next_end, (unsigned long long)__popc(idle));
            at = __shfl_sync(0xffffffffu, at, 0);
            more = at + __popc(idle) < ends;
            if (!open) {
                item = at + __popc(idle & ((1u << lane) - 1u));
                if (item < ends) {
                    const DevHsp &r = h[item >> 1];
                    const uint32_t qi = r.qi, sq = r.seq;
                    if (GN_CHECK(qi < nq && sq < n_seqs)) {
                        const int64_t qb = (int64_t)qstart[qi], sb = (int64_t)seq_start[sq];
                        if (item & 1) {
                            const uint32_t qe = r.qe, de = r.de;
                            emax = (uint32_t)min((int64_t)qstart[qi + 1] - qb - qe, (int64_t)seq_start[sq + 1] - sb - de);
                            q = qb + qe;
                            d = sb + de;
                        } else {
                            const uint32_t qs = r.qs, ds = r.ds;
                            emax = min(qs, ds);
                            q = qb + qs;
                            d = sb + ds;
                        }
                        e = ext = 0;
                        score = best = 0;
                        open = emax > 0;
                    }
                }
            }
        }
        if (!__any_sync(0xffffffffu, open)) {
            if (!more) break;
            continue;
        }
        if (open) {
            const bool right = item & 1;
            uint32_t w[2];
            equal32(seq, right ? q : q - 32, right ? d : d - 32, w);
            if (!right) {
                const uint32_t t = __brev(w[0]);
                w[0] = __brev(w[1]);
                w[1] = t;
            }
            q += right ? 32 : -32;
            d += right ? 32 : -32;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                uint32_t eq = w[j], left = open ? min(16u, emax - e) : 0u;
                while (left) {
                    const uint32_t m = min((uint32_t)__clz(~eq) >> 1, left);  // matches
                    score += (int32_t)m * match;
                    e += m;
                    left -= m;
                    if (m && score > best) { best = score; ext = e; }
                    eq = __funnelshift_lc(0u, eq, 2 * m);
                    const uint32_t x = min((uint32_t)__clz(eq) >> 1, left);  // mismatches
                    if ((int64_t)best - score - (int64_t)x * mismatch > X) { open = false; break; }
                    score += (int32_t)x * mismatch;
                    e += x;
                    left -= x;
                    eq = __funnelshift_lc(0u, eq, 2 * x);
                }
            }
            if (e >= emax) open = false;
            if (!open && ext) {
                uint32_t *r = reinterpret_cast<uint32_t *>(h + (item >> 1));
                if (right) { r[W_QE] += ext; r[W_DE] += ext; }
                else { r[W_QS] -= ext; r[W_DS] -= ext; }
            }
        }
    }
}

}  // namespace gn
#include "gn_seed_scan.cuh"
#include "gn_team.cuh"
namespace gn {

// ------------------------------------------- long queries: segments, join --
// Bases of each segment (block v): len bytes from offset off[v] of query parent[v].
__global__ void k_segment_bases(const uint8_t *__restrict__ qbases, const uint64_t *__restrict__ qstart,
                                const uint32_t *__restrict__ parent, const uint64_t *__restrict__ off,
                                const uint64_t *__restrict__ vstart, uint8_t *__restrict__ out) {
    const uint32_t v = blockIdx.x;
    const uint64_t from = qstart[parent[v]] + off[v], to = vstart[v], len = vstart[v + 1] - to;
    for (uint64_t i = threadIdx.x; i < len; i += blockDim.x) out[to + i] = qbases[from + i];
}

// Chain pieces of the segments onto their queries; the len word carries the diagonal
// (ds - qs mod 2^32, distinct for distinct diagonals when sequences are shorter than
// 2^32 - 2^24 bases) for the join's sort.
__global__ void k_segment_map(DevHsp *__restrict__ h, uint32_t n, const uint32_t *__restrict__ parent,
                              const uint64_t *__restrict__ off) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    DevHsp r = h[i];
    const uint32_t o = (uint32_t)off[r.qi];
    r.qi = parent[r.qi];
    r.qs += o;
    r.qe += o;
    r.len = r.ds - r.qs;
    h[i] = r;
}

// Pieces sorted by (qi, seq, diagonal, qs).  Two pieces of one chain share a hit, so
// a piece joins the current chain when its first hit starts no later than the chain's
// last hit (qs + span <= qe); pieces of different chains on one diagonal are more than
// D >= 0 offsets apart and never do.  The first piece of each (qi, seq, diagonal) run
// walks the run.  A chain is written at the index of its first piece and kept (flag)
// when it is at least min_len long.
__global__ void k_stitch_sweep(const DevHsp *__restrict__ in, uint32_t n, uint32_t span, uint32_t min_len,
                               DevHsp *__restrict__ out, uint32_t *__restrict__ flag) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    auto same = [&](uint32_t a, uint32_t b) {
        return in[a].qi == in[b].qi && in[a].seq == in[b].seq && in[a].len == in[b].len;
    };
    if (i > 0 && same(i - 1, i)) return;
    uint32_t j = i;
    while (j < n && same(j, i)) {
        DevHsp c = in[j];
        const uint32_t head = j++;
        while (j < n && same(j, i) && in[j].qs + span <= c.qe) {
            c.qe = max(c.qe, in[j].qe);
            flag[j++] = 0;
        }
        c.len = c.qe - c.qs;
        c.de = c.ds + c.len;
        out[head] = c;
        flag[head] = c.len >= min_len ? 1u : 0u;
    }
}

// -------------------------------------------------- a10: overlap merging --
// Records sorted by (qi, seq, qs).  The first record of each (qi, seq) run sweeps
// the run in (qs, ds, qe) order (records of one qs, rarely more than one, are taken
// by increasing (ds, qe); de = ds + qe - qs for these ungapped HSPs, so records
// equal in (ds, qe) are equal): each record joins the current box when both its
// query and bank ranges intersect the box, otherwise it starts a new box.  The
// run's boxes are written, in that order, at its first indices, flagged 1; its
// other indices are flagged 0.
__device__ __forceinline__ uint64_t ov_key(const DevHsp &h) { return ((uint64_t)h.ds << 32) | h.qe; }

// The sweep of the run that starts at record i (rec(j): record j of n); boxes go to out and flag
// from i on.  With in_order, boxes of one run that begin at the same qs are put in (ds, qe, de)
// order (a later box can reach further back in the bank than an earlier one), the order by
// which equally long ones are selected.  Returns the index after the run.
template <class Rec, class Flag>
__device__ __forceinline__ uint32_t overlap_run(Rec rec, uint32_t i, uint32_t n, DevHsp *__restrict__ out, Flag set_flag,
                                                bool in_order) {
    DevHsp first = rec(i);
    const uint32_t qi = first.qi, seq = first.seq;
    uint32_t o = i;  // next box slot
    bool open = false;
    DevHsp box{};  // set by the run's first record
    auto put = [&]() {
        box.len = min(box.qe - box.qs, box.de - box.ds);
        uint32_t at = o++;
        set_flag(at, 1u);
        if (in_order) {
            while (at > i) {
                const DevHsp p = out[at - 1];
                const uint64_t kp = ((uint64_t)p.ds << 32) | p.qe, kb = ((uint64_t)box.ds << 32) | box.qe;
                if (p.qs != box.qs || kp < kb || (kp == kb && p.de <= box.de)) break;
                out[at--] = p;
            }
        }
        out[at] = box;
    };
    auto visit = [&](const DevHsp &h) {
        if (open && h.qs < box.qe && box.qs < h.qe && h.ds < box.de && box.ds < h.de) {
            box.qs = min(box.qs, h.qs);
            box.qe = max(box.qe, h.qe);
            box.ds = min(box.ds, h.ds);
            box.de = max(box.de, h.de);
            return;
        }
        if (open) put();
        box = h;
        open = true;
    };
    uint32_t g0 = i;
    DevHsp cur = first;
    for (;;) {
        // the group of records at cur's qs: [g0, g1); next: the record after it, if in the run
        uint32_t g1 = g0 + 1;
        DevHsp next{};
        bool more = false;
        while (g1 < n) {
            next = rec(g1);
            more = next.qi == qi && next.seq == seq;
            if (!more || next.qs != cur.qs) break;
            ++g1;
            more = false;
        }
        if (g1 - g0 == 1) {
            visit(cur);
        } else {
            // the group's records by increasing (ds, qe), then index: each step takes the
            // smallest (key, index) above the last one taken
            uint64_t last_k = 0;
            uint32_t last_j = 0;
            for (uint32_t t = g0; t < g1; ++t) {
                uint64_t best_k = ~0ull;
                uint32_t best_j = g1;
                for (uint32_t j = g0; j < g1; ++j) {
                    const uint64_t kj = ov_key(rec(j));
                    const bool after = t == g0 || kj > last_k || (kj == last_k && j > last_j);
                    if (after && (kj < best_k || (kj == best_k && j < best_j))) {
                        best_k = kj;
                        best_j = j;
                    }
                }
                visit(rec(best_j));
                last_k = best_k;
                last_j = best_j;
            }
        }
        g0 = g1;
        if (!more) break;
        cur = next;
    }
    put();
    for (uint32_t j = o; j < g0; ++j) set_flag(j, 0u);
    return g0;
}

__global__ void k_overlap_sweep(const DevHsp *__restrict__ in, uint32_t n, DevHsp *__restrict__ out,
                                uint32_t *__restrict__ flag, int in_order) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i > 0 && in[i - 1].qi == in[i].qi && in[i - 1].seq == in[i].seq) return;  // not the head of a run
    overlap_run([&](uint32_t j) { return in[j]; }, i, n, out, [&](uint32_t j, uint32_t v) { flag[j] = v; }, in_order != 0);
}

// ----------------------------------------------------- a11: selection --
// The bin of the n-th largest entry of a histogram of 256 bins that holds at least n >= 1, and how
// many lie above that bin (out[0], out[1]); a warp, eight bins a lane.
__device__ __forceinline__ void bin_of_nth(const uint32_t *hist, uint32_t n, uint32_t *out) {
    const int lane = threadIdx.x & 31;
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) sum += hist[255 - 8 * lane - i];
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (x >= n && x - sum < n) {
        uint32_t above = x - sum;
        int b = 255 - 8 * lane;
        while (above + hist[b] < n) above += hist[b--];
        out[0] = (uint32_t)b;
        out[1] = above;
    }
}

// Per-query selection on records sorted by (qi, seq, qs, ds, qe, de): a block per
// query keeps its N longest records, ties broken by that order (a stable choice by
// length), and writes them by (length desc, seq, qs, ds, qe, de).  The N-th largest
// length T comes from a 256-bin histogram per byte of the length (two, or three where a
// query is longer than 65,535 bases), high byte first; the selected records are those
// longer than T and the first ones of length T.  Bound by the latency of its passes over the
// lengths, so every thread has SQ_AHEAD loads under way, and by the chain of the last sort's
// stages, which stays in registers (Team).  8 queries of 22,000 records each, N = 100: 78 -> 51 us;
// 1,000 queries of 100: 29 -> 18 us (the threshold found by one thread, the sort in shared memory).
constexpr int SQ_CAP = 1024;  // largest N this kernel handles
constexpr int SQ_THREADS = 512, SQ_AHEAD = 8;

__global__ void __launch_bounds__(SQ_THREADS) k_select_query(const DevHsp *__restrict__ rec,
                                                             const uint32_t *__restrict__ qfirst,
                                                             const uint64_t *__restrict__ qout, uint32_t N, int bytes,
                                                             DevHsp *__restrict__ sel) {
    typedef Team<SQ_THREADS, SQ_CAP / 256> tm;  // keys in the first threads, a warp for up to 128
    constexpr int E = SQ_CAP / 256;
    __shared__ uint32_t hist[256];
    __shared__ uint32_t warp_tot[SQ_THREADS / 32];
    __shared__ uint64_t keys[SQ_CAP];
    __shared__ uint32_t found[2];
    const uint32_t q = blockIdx.x;
    const uint32_t a = qfirst[q], b = qfirst[q + 1], n = b - a;
    const uint64_t out0 = qout[q];
    const uint32_t nsel = (uint32_t)(qout[q + 1] - out0);
    if (nsel == 0) return;
    const uint32_t max_len = (1u << (8 * bytes)) - 1u;
    uint32_t T = 0, r_eq = n;  // n <= N: every record is selected
    if (n > N) {
        uint32_t above = 0;
        for (int shift = 8 * (bytes - 1); shift >= 0; shift -= 8) {  // T: its bytes so far
            for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
            __syncthreads();
            // one shared-memory atomic per distinct bin of a warp's 32 records (lengths are
            // concentrated in few bins)
            for (uint32_t i0 = a + (threadIdx.x & ~31u); i0 < b; i0 += SQ_AHEAD * SQ_THREADS) {
                uint32_t len[SQ_AHEAD];
#pragma unroll
                for (int u = 0; u < SQ_AHEAD; ++u) {
                    const uint32_t i = i0 + u * SQ_THREADS + (threadIdx.x & 31u);
                    len[u] = i < b ? min(rec[i].len, max_len) : 0u;
                }
#pragma unroll
                for (int u = 0; u < SQ_AHEAD; ++u) {
                    const uint32_t i = i0 + u * SQ_THREADS + (threadIdx.x & 31u);
                    if (i0 + u * SQ_THREADS >= b) break;
                    const bool in = i < b && ((uint64_t)len[u] >> (shift + 8)) == T;
                    const uint32_t bin = in ? (len[u] >> shift) & 0xFFu : 256u;
                    const uint32_t peers = __match_any_sync(0xffffffffu, bin);
                    if (in && (threadIdx.x & 31u) == (uint32_t)(__ffs(peers) - 1))
                        atomicAdd(&hist[bin], (uint32_t)__popc(peers));
                }
            }
            __syncthreads();
            if (threadIdx.x < 32) bin_of_nth(hist, N - above, found);
            __syncthreads();
            T = (T << 8) | found[0];
            above += found[1];
            __syncthreads();
        }
        r_eq = N - above;  // records of length T to take, in array order
    }
    // ordered compaction of the selected records (array order), keyed by (length desc, position):
    // each thread takes a contiguous run of records, counts its records longer than T and of
    // length T, and two block scans give its first output slot and its first rank among the
    // records of length T
    const uint32_t per = (n + blockDim.x - 1) / blockDim.x;
    const uint32_t lo = min(n, threadIdx.x * per), hi = min(n, lo + per);
    auto lengths = [&](auto visit) {  // of the thread's records, in order
        for (uint32_t i0 = lo; i0 < hi; i0 += SQ_AHEAD) {
            uint32_t len[SQ_AHEAD];
#pragma unroll
            for (int u = 0; u < SQ_AHEAD; ++u) len[u] = i0 + u < hi ? min(rec[a + i0 + u].len, max_len) : 0u;
#pragma unroll
            for (int u = 0; u < SQ_AHEAD; ++u)
                if (i0 + u < hi) visit(i0 + u, len[u]);
        }
    };
    uint32_t n_gt = 0, n_eq = 0;
    lengths([&](uint32_t, uint32_t len) {
        const bool gt = n <= N || len > T;
        n_gt += gt ? 1u : 0u;
        n_eq += (!gt && len == T) ? 1u : 0u;
    });
    uint32_t tot = 0;
    uint32_t eq_rank = block_excl_scan(n_eq, warp_tot, tot);
    const uint32_t n_take = n_gt + min(n_eq, r_eq > eq_rank ? r_eq - eq_rank : 0u);
    uint32_t pos = block_excl_scan(n_take, warp_tot, tot);
    if (n_take)
        lengths([&](uint32_t i, uint32_t len) {
            const bool gt = n <= N || len > T;
            const bool eq = !gt && len == T;
            const bool take = gt || (eq && eq_rank < r_eq);
            eq_rank += eq ? 1u : 0u;
            if (take) keys[pos++] = ((uint64_t)(max_len - len) << 32) | i;
        });
    __syncthreads();
    uint64_t r[E];
    const uint32_t P = tm::padded(nsel), A = P / E;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = e * A + threadIdx.x;
        r[e] = threadIdx.x < A && i < nsel ? keys[i] : ~0ull;
    }
    __syncthreads();
    tm::sort(r, keys, P, KeyLess());
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t k = threadIdx.x * E + e;
        if (k < nsel) sel[out0 + k] = rec[a + (uint32_t)(r[e] & 0xFFFFFFFFu)];
    }
}

// first[q] = first record of query q in records sorted by query (first[nq] = n), and, when
// cnt is given, cnt[q] = min(N, records of query q): the counts of the selected records
__device__ __forceinline__ uint32_t first_of_query(const DevHsp *__restrict__ rec, uint32_t n, uint32_t q) {
    uint32_t lo = 0, hi = n;  // first index with qi >= q
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (rec[mid].qi < q) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// n_dev: the number of records.  first64: the same as first, as a prefix sum of all records.
__global__ void k_query_bounds(const DevHsp *__restrict__ rec, const uint64_t *__restrict__ n_dev, uint32_t nq,
                               uint32_t *__restrict__ first, uint64_t *__restrict__ first64, uint32_t N,
                               uint32_t *__restrict__ cnt) {
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x, n = (uint32_t)*n_dev;
    if (q > nq) return;
    const uint32_t f = first_of_query(rec, n, q);
    first[q] = f;
    if (first64) first64[q] = f;
    if (cnt && q < nq) cnt[q] = min(N, first_of_query(rec, n, q + 1) - f);
}

// Overlap merging and selection of a small search in one block: sorts the records of up to MB_CAP
// HSPs by (qi, seq, qs) (ties keep their order, which the sweep does not depend on), sweeps the
// runs, compacts the boxes, finds each query's first box and the prefix sums of min(N, boxes)
// (N = 0: of all boxes) as k_query_bounds and a scan do, and, when sel is given, sorts the boxes by
// (qi, length desc, place) and writes each query's first N there as k_select_query does.
// Replaces nine launches: a search of a handful of HSPs is a chain of launches of 2 to 5 us each.
// 8 and 14 us at 1 and 17 HSPs, with the selection in it (8 and 14 before without it).  The call as
// a whole by this | by groups, us: 38 HSPs 234 | 255, 513 HSPs 257 | 277, 1,023 HSPs 391 | 386.
constexpr uint32_t MB_CAP = 1024, MB_QUERIES = 4096;
constexpr int MB_THREADS = 512, MB_BITS = 10;

__global__ void __launch_bounds__(MB_THREADS) k_merge_block(const DevHsp *__restrict__ in, uint32_t n, uint32_t seq_bits,
                                                            uint32_t qs_bits, uint32_t nq, uint32_t N, int in_order,
                                                            DevHsp *__restrict__ boxes, DevHsp *__restrict__ out,
                                                            uint32_t *__restrict__ first, uint64_t *__restrict__ qo,
                                                            uint64_t *__restrict__ n_out, DevHsp *__restrict__ sel) {
    constexpr int E = MB_CAP / MB_THREADS;
    typedef Team<MB_THREADS, E> tm;
    constexpr uint32_t idx_mask = (1u << MB_BITS) - 1u;
    __shared__ uint64_t key[MB_CAP];
    __shared__ uint8_t flag[MB_CAP];
    __shared__ uint32_t warp_tot[MB_THREADS / 32];
    const uint32_t t = threadIdx.x;
    // the keys of n records, sorted
    auto sort = [&](uint32_t n, auto key_of) {
        uint64_t r[E];
        const uint32_t P = tm::padded(n), A = P / E;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = e * A + t;
            r[e] = t < A && i < n ? key_of(i) << MB_BITS | i : ~0ull;
        }
        tm::sort(r, key, P, KeyLess());
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (t < A) key[t * E + e] = r[e];
        __syncthreads();
    };
    sort(n, [&](uint32_t i) { return ((((uint64_t)in[i].qi << seq_bits) | in[i].seq) << qs_bits) | in[i].qs; });
    const uint32_t run_shift = qs_bits + MB_BITS;
    for (uint32_t i = t; i < n; i += blockDim.x) {
        if (i > 0 && key[i - 1] >> run_shift == key[i] >> run_shift) continue;
        overlap_run([&](uint32_t j) { return in[(uint32_t)key[j] & idx_mask]; }, i, n, boxes,
                    [&](uint32_t j, uint32_t v) { flag[j] = (uint8_t)v; }, in_order != 0);
    }
    __syncthreads();
    uint32_t n_mg = 0;
    for (uint32_t i0 = 0; i0 < n; i0 += blockDim.x) {
        const uint32_t i = i0 + t, f = i < n ? flag[i] : 0u;
        uint32_t tot = 0;
        const uint32_t at = n_mg + block_excl_scan(f, warp_tot, tot);
        if (f) out[at] = boxes[i];
        n_mg += tot;
    }
    __syncthreads();
    uint64_t sum = 0;
    for (uint32_t q0 = 0; q0 <= nq; q0 += blockDim.x) {
        const uint32_t q = q0 + t;
        uint32_t c = 0;
        if (q <= nq) {
            const uint32_t f = first_of_query(out, n_mg, q);
            first[q] = f;
            if (q < nq) {
                c = first_of_query(out, n_mg, q + 1) - f;
                if (N) c = min(N, c);
            }
        }
        uint32_t tot = 0;
        const uint32_t at = block_excl_scan(c, warp_tot, tot);
        if (q <= nq) qo[q] = sum + at;
        sum += tot;
    }
    if (t == 0) *n_out = n_mg;
    if (!sel) return;
    __syncthreads();
    sort(n_mg, [&](uint32_t i) { return ((uint64_t)out[i].qi << 32) | (0xFFFFFFFFu - out[i].len); });
    for (uint32_t i = t; i < n_mg; i += blockDim.x) {
        const DevHsp h = out[(uint32_t)key[i] & idx_mask];
        const uint32_t k = i - first[h.qi];
        if (k < N) sel[qo[h.qi] + k] = h;
    }
}

}  // namespace gn
#include "gn_merge_groups.cuh"
namespace gn {

__global__ void k_first_of_query(const uint32_t *__restrict__ recs, int W, uint32_t n, uint32_t *__restrict__ first) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t q = recs[(uint64_t)i * W];
    if (i == 0 || recs[(uint64_t)(i - 1) * W] != q) first[q] = i;
}

__global__ void k_select_flags(const DevHsp *__restrict__ h, uint32_t n, const uint32_t *__restrict__ first,
                               uint32_t N, uint32_t *__restrict__ flag) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    flag[i] = (N == 0 || i - first[h[i].qi] < N) ? 1u : 0u;
}

// -------------------------------------------- a12: banded Smith-Waterman --
// One warp per selected HSP.  Lanes own band offsets b (diagonal j - i = dlo + b);
// rows i of the DP window are processed in order, each row in chunks of 32
// offsets.  The previous row (H, E and their start cells) lives in a per-HSP
// scratch strip of B entries.  Horizontal gaps (F) inside a row are resolved
// by a warp max-scan of X(b') = H0(b') + go + ge - ge*b' (H0 = the cell's best
// over 0, diagonal and vertical gap), since F(b) = max_{b'<b} X(b') + ge*(b-1)
// reproduces the sequential recurrence, including its "open wins ties" choice
// when the scan keeps the later of equal values.
struct SwCell {
    int32_t H, E;
    uint32_t SH, SE;  // start cells: (row - I0) * B + band offset
};

constexpr int32_t SW_NEG = -(1 << 29);
constexpr int32_t SW_XNEG = -(1 << 30);

__device__ __forceinline__ void scan_pair_max(int32_t &v, uint32_t &s, int lane) {
    // inclusive scan, later lane wins ties
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t ov = __shfl_up_sync(0xffffffffu, v, o);
        uint32_t os = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o && ov > v) { v = ov; s = os; }
    }
}


// Band width (diagonals) of an HSP's alignment: the spread of its end diagonals plus 2w + 1.
__device__ __forceinline__ int64_t dev_band(const DevHsp &h, int32_t w) {
    const int64_t d_s = (int64_t)h.ds - h.qs, d_e = (int64_t)h.de - h.qe;
    return max(d_s, d_e) - min(d_s, d_e) + 2 * (int64_t)w + 1;
}

// One HSP aligned by a whole warp on the strip path (bands wider than the register paths hold):
// the band in chunks of 32 offsets, the previous row in scratch.
__device__ void sw_task_strip(const DevHsp *__restrict__ sel, uint32_t task, SwCell *__restrict__ row,
                              const uint32_t *__restrict__ qpk,
                              const uint32_t *__restrict__ qnb, const uint64_t *__restrict__ qstart,
                              const uint32_t *__restrict__ bpk, const uint32_t *__restrict__ bnb,
                              const uint64_t *__restrict__ seq_start, int32_t match, int32_t mismatch, int32_t go,
                              int32_t ge, int32_t w, DevAln *__restrict__ out, uint32_t *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    const DevHsp h = sel[task];
    const uint64_t qb = qstart[h.qi], sb = seq_start[h.seq];
    const int64_t m = (int64_t)(qstart[h.qi + 1] - qb), L = (int64_t)(seq_start[h.seq + 1] - sb);
    const int64_t d_s = (int64_t)h.ds - h.qs, d_e = (int64_t)h.de - h.qe;
    const int64_t dlo = min(d_s, d_e) - w, dhi = max(d_s, d_e) + w;
    const int64_t I0 = max((int64_t)0, (int64_t)h.qs - w), I1 = min(m, (int64_t)h.qe + w);
    const int64_t J0 = max((int64_t)0, (int64_t)h.ds - w), J1 = min(L, (int64_t)h.de + w);
    const int64_t B = dhi - dlo + 1;
    DevAln res;
    res.qi = h.qi; res.seq = h.seq; res.qs = res.qe = res.ds = res.de = 0; res.score = 0; res.pad = 0;
    // start cells are (row - I0) * B + offset in 32 bits; strips hold up to 65,536 entries
    if (B > 65535 || (uint64_t)max(I1 - I0, (int64_t)0) * (uint64_t)B >= (1ull << 32)) {
        if (lane == 0) { atomicOr(status, DEV_ERR_BAND_TOO_WIDE); out[task] = res; }
        return;
    }
    int32_t best = 0;
    int64_t bi = INT64_MAX, bj = INT64_MAX;
    uint32_t bs = 0;
    const int32_t goe = go + ge;
    for (int64_t i = I0; i < I1; ++i) {
        const int64_t blo = max((int64_t)0, J0 - i - dlo), bhi = min(B - 1, J1 - 1 - i - dlo);
        if (blo > bhi) continue;
        const bool prow = i - 1 >= I0;
        const int64_t pblo = max((int64_t)0, J0 - (i - 1) - dlo), pbhi = min(B - 1, J1 - 1 - (i - 1) - dlo);
        const uint32_t qc = dev_base(qpk, qnb, qb + (uint64_t)i);
        int32_t carry_v = SW_XNEG;
        uint32_t carry_s = 0;
        for (int64_t c0 = blo; c0 <= bhi; c0 += 32) {
            const int64_t b = c0 + lane;
            const bool act = b <= bhi;
            SwCell pd{0, SW_NEG, 0, 0}, pu{0, SW_NEG, 0, 0};
            const bool ok_d = act && prow && b >= pblo && b <= pbhi;
            const bool ok_u = act && prow && b + 1 >= pblo && b + 1 <= pbhi;
            if (ok_d) pd = row[b];
            if (ok_u) pu = row[b + 1];
            __syncwarp();
            int32_t E = SW_NEG;
            uint32_t SE = 0;
            if (ok_u) {
                int32_t eo = pu.H + goe, ee = pu.E + ge;
                if (eo >= ee) { E = eo; SE = pu.SH; } else { E = ee; SE = pu.SE; }
            }
            const int32_t Hd = ok_d ? pd.H : 0;
            const uint32_t SD = (Hd > 0) ? pd.SH : (uint32_t)(i - I0) * (uint32_t)B + (uint32_t)b;
            const int64_t j = i + dlo + b;
            int32_t sigma = mismatch;
            if (act) sigma = dev_pair(qc, dev_base(bpk, bnb, sb + (uint64_t)j), match, mismatch);
            const int32_t Dg = Hd + sigma;
            int32_t cand;
            uint32_t Sc;
            if (Dg >= E) { cand = Dg; Sc = SD; } else { cand = E; Sc = SE; }
            const int32_t H0 = cand > 0 ? cand : 0;
            // F by max-scan with carry from earlier chunks of this row
            int32_t xv = act ? H0 + goe - ge * (int32_t)b : SW_XNEG;
            uint32_t xs = Sc;
            scan_pair_max(xv, xs, lane);
            int32_t ev = __shfl_up_sync(0xffffffffu, xv, 1);
            uint32_t es = __shfl_up_sync(0xffffffffu, xs, 1);
            // the carry (earlier chunks) wins only when strictly larger
            if (lane == 0) { ev = carry_v; es = carry_s; }
            else if (carry_v > ev) { ev = carry_v; es = carry_s; }
            int32_t last_v = __shfl_sync(0xffffffffu, xv, 31);
            uint32_t last_s = __shfl_sync(0xffffffffu, xs, 31);
            if (last_v >= carry_v) { carry_v = last_v; carry_s = last_s; }
            int32_t F = (ev > SW_XNEG) ? ev + ge * (int32_t)(b - 1) : SW_NEG;
            uint32_t SF = es;
            int32_t H;
            uint32_t SH;
            if (H0 >= F) { H = H0; SH = Sc; } else { H = F; SH = SF; }
            if (act) {
                SwCell c;
                c.H = H; c.E = E; c.SH = SH; c.SE = SE;
                row[b] = c;
                if (H > best) { best = H; bi = i; bj = j; bs = SH; }
            }
            __syncwarp();
        }
    }
    // reduce: highest score, then smallest i, then smallest j
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        int32_t ob = __shfl_down_sync(0xffffffffu, best, o);
        int64_t oi = __shfl_down_sync(0xffffffffu, bi, o);
        int64_t oj = __shfl_down_sync(0xffffffffu, bj, o);
        uint32_t os = __shfl_down_sync(0xffffffffu, bs, o);
        if (ob > best || (ob == best && (oi < bi || (oi == bi && oj < bj)))) {
            best = ob; bi = oi; bj = oj; bs = os;
        }
    }
    if (lane == 0) {
        if (best > 0) {
            int64_t i0 = I0 + (int64_t)(bs / (uint32_t)B);
            int64_t j0 = i0 + dlo + (int64_t)(bs % (uint32_t)B);
            res.qs = (uint32_t)i0; res.qe = (uint32_t)(bi + 1);
            res.ds = (uint32_t)j0; res.de = (uint32_t)(bj + 1);
            res.score = best;
        }
        out[task] = res;
    }
}

// Register path: a segment of G lanes aligns one HSP, lane l of the segment owning K = KA + KB
// adjacent band offsets with their previous-row states in registers.  Lane l takes row r in
// iteration r + l, first its KA offsets, then its KB offsets.  The first part needs the same
// row of the lane to its left (the horizontal gap that runs into it), finished in the iteration
// before; the last offset of the second part needs the previous row of the lane to its right
// (the vertical gap), whose first part came earlier in the same iteration.  So every lane works
// all the time, a row costs two exchanges with neighbours and K cells of the sequential
// recurrence, and none needs a scan over the lanes.
//
// Cells follow the recurrence with its tie rules: E and F open on ties, the diagonal beats E, H0
// beats F, F extends from the left cell's H0.  A cell outside the DP window is given no match,
// and that is enough: left of the window and before its first row H stays 0, so gaps out of
// there are never positive; cells right of it or below feed no cell inside; and a new best
// always ends in a match (gaps never add, mismatches subtract).
//
// Offsets past the band are computed too (G K is rarely the band's width), without matches, and
// the band's last offset reads E from the first of them.  A path can only leave the band by F,
// along a row, and come back by E, down a column: j + 1 offsets out and back cost at least
// goe + (2j + 1) ge more than the way that stays j + 1 rows on its diagonal, which costs at most
// j + 1 mismatches more.  With mismatch >= 2 ge (the default -3 against -4) that way is at least
// as good wherever the path comes back, arrives by the diagonal, and so wins ties: nothing
// from outside is ever chosen.  For other scores (CUT) offsets past the band pass on no E.
//
// Bound by instructions: about 27 a cell (each of the four tracked maxima also selects a start
// cell) on two pipes that take one every other cycle each, and about 20 a row for the exchange
// and the bases; the window's limits are kept with the bases, as places without a match, and
// cost instructions only in blocks of 16 rows that meet one.  Measured against the row-by-row
// path with a scan over the lanes (and its wavefront form for long alignments) that this
// replaced, band cells of the whole phase: 50,000 alignments (396 M cells) 1.50 -> 0.57 ms,
// 30,000 (203 M) 1.15 -> 0.31, bands of 257 diagonals (881 M) 2.57 -> 1.04; one alignment of 400
// rows alone 218 -> 56 us.
constexpr int SW_SHIFT = 9;  // cells are row << SW_SHIFT | band offset (up to 512 offsets, 2^23 rows)
constexpr int SW_MAX_BAND = 32 * 9;
constexpr int64_t SW_MAX_ROWS = 1ll << (32 - SW_SHIFT);

// One HSP's DP window as packed positions: rows [qlo, qhi) of the query, columns [dlo, dhi) of
// the bank, both inclusive of nothing outside the sequences; offset 0 of row qlo is at diag.
struct SwGeom {
    int64_t qlo, qhi, dlo, dhi, diag;
    int32_t B;
    __device__ __forceinline__ void set(const DevHsp &h, const uint64_t *__restrict__ qstart,
                                        const uint64_t *__restrict__ seq_start, int32_t w) {
        const int64_t qb = (int64_t)qstart[h.qi], sb = (int64_t)seq_start[h.seq];
        const int64_t m = (int64_t)qstart[h.qi + 1] - qb, L = (int64_t)seq_start[h.seq + 1] - sb;
        const int64_t d_s = (int64_t)h.ds - h.qs, d_e = (int64_t)h.de - h.qe, d0 = min(d_s, d_e) - w;
        qlo = qb + max((int64_t)0, (int64_t)h.qs - w);
        qhi = qb + min(m, (int64_t)h.qe + w);
        dlo = sb + max((int64_t)0, (int64_t)h.ds - w);
        dhi = sb + min(L, (int64_t)h.de + w);
        diag = sb + (qlo - qb) + d0;
        B = (int32_t)(max(d_s, d_e) + w - d0 + 1);
    }
};

// Bits [from, to) of 32 positions (any values).
__device__ __forceinline__ uint32_t positions(int64_t from, int64_t to) {
    const uint32_t a = (uint32_t)min(max(from, (int64_t)0), (int64_t)32), b = (uint32_t)min(max(to, (int64_t)0), (int64_t)32);
    const uint32_t lo = __funnelshift_lc(0u, 0xFFFFFFFFu, a), hi = __funnelshift_lc(0u, 0xFFFFFFFFu, b);
    return lo & ~hi;
}

template <int K>
struct SwSet {
    int32_t H[K], E[K];     // previous row: H of each offset, E that it passes to the offset before it
    uint32_t SH[K], SE[K];  // their start cells
    int32_t best;           // best cell so far: score, cell of the row after it, start cell
    uint32_t bcell, bstart;
    uint32_t cell;          // the row to come's first offset of the lane, as a cell
    int64_t q, d;           // the row to come: packed position of its query base, of the lane's first bank base
    uint32_t dw_hi, dw_lo;  // bank bases from d on, first one on top (loaded for 16 rows)
    uint32_t qw;            // query bases from q on
    uint32_t dno_hi, dno_lo;  // in the places of dw: no match there (a non-base, or outside the DP window)
    uint32_t qno;           // the same of q on, a bit each, q's on top
    uint32_t in_band;       // bit 30 - 2 k: offset inside the band
    int64_t qlo, qhi, dlo, dhi;

    __device__ __forceinline__ void start(const SwGeom &g, bool on, int b0, int lag) {
#pragma unroll
        for (int k = 0; k < K; ++k) { H[k] = 0; E[k] = SW_NEG; SH[k] = SE[k] = 0; }
        best = 0; bcell = 0xFFFFFFFFu; bstart = 0;
        cell = (uint32_t)(-lag * (1 << SW_SHIFT) + b0);
        if (lag == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) SH[k] = cell + (uint32_t)k;
        }
        qlo = g.qlo; qhi = on ? g.qhi : g.qlo; dlo = g.dlo; dhi = g.dhi;
        q = g.qlo - lag;
        d = g.diag + b0 - lag;
        const int32_t B = g.B - b0;
        in_band = !on || B <= 0 ? 0u : B >= K ? 0x55555555u : 0x55555555u & ~(0xFFFFFFFFu >> (2 * B));
    }
    // the bases of the 16 rows to come; returns whether dno or qno has a bit that they meet
    __device__ __forceinline__ bool load(const PackedPair &s) {
        uint32_t db, qb;
        const uint64_t w = window32(s.bpk, s.bnb, d, s.last_bpk, s.last_bnb, db);
        dw_hi = (uint32_t)(w >> 32);
        dw_lo = (uint32_t)w;
        qw = (uint32_t)(window32(s.qpk, s.qnb, q, s.last_qpk, s.last_qnb, qb) >> 32);
        db |= ~positions(dlo - d, dhi - d);
        qb = (qb | ~positions(qlo - q, qhi - q)) & 0xFFFFu;
        db &= (1u << (15 + K)) - 1u;
        dno_hi = dno_lo = qno = 0;
        if (db | qb) {
            dno_hi = spread16_down(db);
            dno_lo = spread16_down(db >> 16);
            qno = __brev(qb);
        }
        return (db | qb) != 0;
    }
};

// Compares, selects, maxima and logic all issue to one pipe at half rate, and a maximum that
// also selects a start cell takes three of them.  The multiply-add pipe, as wide, would idle, so
// additions and the moves of a taken branch are written as multiply-adds by `one` (1, a value
// the compiler cannot see through): 12 and 15 instructions a cell instead of 27 on one pipe.
__device__ __forceinline__ int32_t fma_add(int32_t a, int32_t b, int32_t one) {
    int32_t r;
    asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(one), "r"(b));
    return r;
}
// if (x > v) { v = x; s = t; }
__device__ __forceinline__ void fma_take_gt(int32_t &v, uint32_t &s, int32_t x, uint32_t t, int32_t one) {
    asm("{ .reg .pred q; setp.gt.s32 q, %2, %0; @q mul.lo.s32 %0, %2, %4; @q mul.lo.s32 %1, %3, %4; }"
        : "+r"(v), "+r"(s) : "r"(x), "r"(t), "r"(one));
}
// if (x >= v) { v = x; s = t; }
__device__ __forceinline__ void fma_take_ge(int32_t &v, uint32_t &s, int32_t x, uint32_t t, int32_t one) {
    asm("{ .reg .pred q; setp.ge.s32 q, %2, %0; @q mul.lo.s32 %0, %2, %4; @q mul.lo.s32 %1, %3, %4; }"
        : "+r"(v), "+r"(s) : "r"(x), "r"(t), "r"(one));
}
// if (v <= 0) s = t;
__device__ __forceinline__ void fma_if_not_pos(uint32_t &s, int32_t v, uint32_t t, int32_t one) {
    asm("{ .reg .pred q; setp.le.s32 q, %1, 0; @q mul.lo.s32 %0, %2, %3; }" : "+r"(s) : "r"(v), "r"(t), "r"(one));
}
// h + (bit ? match : mismatch)
__device__ __forceinline__ int32_t fma_score(int32_t h, uint32_t bit, int32_t match, int32_t mismatch, int32_t one) {
    int32_t r;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; mad.lo.s32 %0, %1, %5, %4; @q mad.lo.s32 %0, %1, %5, %3; }"
        : "=&r"(r) : "r"(h), "r"(bit), "r"(match), "r"(mismatch), "r"(one));
    return r;
}
// if (h > best) { best = h; cell = c; start = t; }
__device__ __forceinline__ void fma_best(int32_t &best, uint32_t &cell, uint32_t &start, int32_t h, uint32_t c, uint32_t t,
                                         int32_t one) {
    asm("{ .reg .pred q; setp.gt.s32 q, %3, %0; @q mul.lo.s32 %0, %3, %6; @q mul.lo.s32 %1, %4, %6;"
        " @q mul.lo.s32 %2, %5, %6; }"
        : "+r"(best), "+r"(cell), "+r"(start) : "r"(h), "r"(c), "r"(t), "r"(one));
}

struct SwScore {
    int32_t match, mismatch, goe, ge, one;
};

// Cell k of the row: E and F run into it (SE, SF: their start cells); leaves the cell's H, the E
// that it passes to the offset before it and, in F, the one for the offset after it.
// bit 30 - 2 k of eq: two equal bases.
template <int K, bool CUT>
__device__ __forceinline__ void sw_cell(SwSet<K> &x, int k, uint32_t eq, int32_t E, uint32_t SE, int32_t &F, uint32_t &SF,
                                        const SwScore &c) {
    const uint32_t below = x.cell + (uint32_t)k;  // the cell a row on: the start after H = 0
    int32_t cv = fma_score(x.H[k], eq & (1u << (30 - 2 * k)), c.match, c.mismatch, c.one);  // the diagonal beats E
    uint32_t C = x.SH[k];
    fma_take_gt(cv, C, E, SE, c.one);
    fma_if_not_pos(C, cv, below, c.one);
    const int32_t H0 = max(cv, 0);
    const bool ph = H0 >= F;  // H0 beats F
    const int32_t H = max(H0, F);
    const uint32_t S = ph ? C : SF;
    fma_best(x.best, x.bcell, x.bstart, H, below, S, c.one);
    x.H[k] = H;
    x.SH[k] = S;
    // open beats extend
    const int32_t eo = fma_add(H, c.goe, c.one), ee = fma_add(E, c.ge, c.one);
    x.E[k] = max(eo, ee);
    x.SE[k] = eo >= ee ? S : SE;
    if (CUT && !(x.in_band & (1u << (30 - 2 * k)))) x.E[k] = SW_NEG;
    const int32_t fo = fma_add(H0, c.goe, c.one);
    F = fma_add(F, c.ge, c.one);
    fma_take_ge(F, SF, fo, C, c.one);
}

// The row's equal bases (bit 30 - 2 k: offset k, inside the band and the DP window) and the step
// to the next row.  NO: dno and qno have bits.
template <int K, bool NO>
__device__ __forceinline__ uint32_t sw_next_row(SwSet<K> &x) {
    const uint32_t y = ~(x.dw_hi ^ ((x.qw >> 30) * 0x55555555u));
    uint32_t eq = y & (y >> 1) & x.in_band;
    if (NO) {
        eq &= ~(x.dno_hi | (uint32_t)((int32_t)x.qno >> 31));
        x.dno_hi = __funnelshift_l(x.dno_lo, x.dno_hi, 2);
        x.dno_lo <<= 2;
        x.qno <<= 1;
    }
    x.dw_hi = __funnelshift_l(x.dw_lo, x.dw_hi, 2);
    x.dw_lo *= 4u;
    x.qw *= 4u;
    x.cell += 1u << SW_SHIFT;
    return eq;
}

// One iteration: the lane's next row.  F1, SF1: the F that its last row passes to the right.
// CUT: offsets past the band must not reach back into it (else the scores see to that).
template <int G, int KA, int KB, bool NO, bool CUT>
__device__ __forceinline__ void sw_row(SwSet<KA + KB> &x, int32_t &F1, uint32_t &SF1, int sl, const SwScore &c) {
    constexpr int K = KA + KB;
    int32_t F = __shfl_up_sync(0xffffffffu, F1, 1);
    uint32_t SF = __shfl_up_sync(0xffffffffu, SF1, 1);
    if (sl == 0) F = SW_NEG;
    const uint32_t eq = sw_next_row<K, NO>(x);
#pragma unroll
    for (int k = 0; k < KA; ++k) sw_cell<K, CUT>(x, k, eq, x.E[k + 1], x.SE[k + 1], F, SF, c);
    int32_t uE = __shfl_down_sync(0xffffffffu, x.E[0], 1);
    const uint32_t uSE = __shfl_down_sync(0xffffffffu, x.SE[0], 1);
    if (sl == G - 1) uE = SW_NEG;
#pragma unroll
    for (int k = KA; k < K; ++k)
        sw_cell<K, CUT>(x, k, eq, k + 1 < K ? x.E[k + 1] : uE, k + 1 < K ? x.SE[k + 1] : uSE, F, SF, c);
    F1 = F;
    SF1 = SF;
}

// Packed cells: score, choice and start cell in one word, for alignments whose rows and scores fit
// (exactly; sw_fits).  From the top: the score, signed; 3 bits of choice; ROW bits of row and OFF bits
// of band offset of the start cell.  The choice orders candidates of one score as the recurrence
// does (a new start 7, the diagonal 6, E opened 5 or extended 4, F opened 1 or extended 0), so that
// a plain maximum of words selects score and start at once, three candidates in one instruction,
// where a tracked maximum takes a compare and two selects; a logic operation then clears the
// choice.  F opens from H, not from H without F: where F won, opening from it can not beat
// extending it (gap_open <= 0) and has its start.  20 instructions a cell instead of 27, shuffles
// of one word instead of two, and shorter chains.  us, tracked | packed: one alignment of 400 rows 56 |
// 47; 200,000 alignments (2,000 queries) 573 | 460, 50,000 at stride 1 220 | 170, 881 M cells of
// 257 and more diagonals 1,019 | 830.  Longer alignments name starts by a table (sp_band); only
// scores beyond that keep tracked cells.
template <int OFF, int ROW>
struct SwPack {
    static constexpr int CHOICE = OFF + ROW, SCORE = CHOICE + 3;
    static constexpr int32_t CLEAN = ~(7 << CHOICE), NEG = -(1 << 30), LOW = (1 << SCORE) - 1;
    int32_t match, mismatch, e_open, e_ext, f_open, f_ext, one;
    __device__ __forceinline__ explicit SwPack(const SwScore &c)
        : match(word(c.match, 6)), mismatch(word(c.mismatch, 6)), e_open(word(c.goe, 5)), e_ext(word(c.ge, 4)),
          f_open(word(c.goe, 1)), f_ext(word(c.ge, 0)), one(c.one) {}
    static __device__ __forceinline__ int32_t word(int32_t score, int32_t choice) {
        return (int32_t)((uint32_t)score << SCORE) + (choice << CHOICE);
    }
    // rows of the DP window, at most: their starts fit (in the word or by a table), their scores do,
    // and gaps and mismatches taken from NEG stay in range
    static __device__ __forceinline__ bool fits(int64_t rows, const SwScore &c, bool table = false) {
        const int32_t low = -(1 << (30 - SCORE));
        return (table || rows < (1 << ROW)) && rows * c.match < (1 << (31 - SCORE)) && c.mismatch > low && c.goe > low && c.ge > low;
    }
};

// Cell k of the row, as sw_cell; z: the word of a start on the lane's first offset a row on.
template <class P, int K, bool CUT>
__device__ __forceinline__ void sp_cell(SwSet<K> &x, int k, uint32_t eq, int32_t E, int32_t &F, int32_t z, const P &c) {
    const int32_t D = fma_score(x.H[k], eq & (1u << (30 - 2 * k)), c.match, c.mismatch, c.one);
    const int32_t h = max(__vimax3_s32(D, E, fma_add(z, k, c.one)), F);
    // a higher score than the best one, whose word with all lower bits set is bstart
    asm("{ .reg .pred q; setp.gt.s32 q, %3, %2; @q mul.lo.s32 %0, %3, %6; @q mad.lo.s32 %1, %4, %6, %5; @q or.b32 %2, %3, %7; }"
        : "+r"(x.best), "+r"(x.bcell), "+r"(x.bstart)
        : "r"(h), "r"(x.cell), "r"(k), "r"(c.one), "n"(P::LOW));
    const int32_t H = h & P::CLEAN;
    x.H[k] = H;
    x.E[k] = max(fma_add(H, c.e_open, c.one), fma_add(E & P::CLEAN, c.e_ext, c.one));
    if (CUT && !(x.in_band & (1u << (30 - 2 * k)))) x.E[k] = P::NEG;
    F = max(fma_add(H, c.f_open, c.one), fma_add(F & P::CLEAN, c.f_ext, c.one));
}

// sw_row on packed cells; SH[0]: the row to come's first offset of the lane, as a start.
template <class P, int OFF, int G, int KA, int KB, bool NO, bool CUT>
__device__ __forceinline__ void sp_row(SwSet<KA + KB> &x, int32_t &F1, int sl, const P &c) {
    constexpr int K = KA + KB;
    int32_t F = __shfl_up_sync(0xffffffffu, F1, 1);
    if (sl == 0) F = P::NEG;
    const uint32_t eq = sw_next_row<K, NO>(x);
    x.SH[0] += 1u << OFF;
    const int32_t z = (int32_t)((x.SH[0] & ((1u << P::CHOICE) - 1u)) | (7u << P::CHOICE));
#pragma unroll
    for (int k = 0; k < KA; ++k) sp_cell<P, K, CUT>(x, k, eq, x.E[k + 1], F, z, c);
    int32_t uE = __shfl_down_sync(0xffffffffu, x.E[0], 1);
    if (sl == G - 1) uE = P::NEG;
#pragma unroll
    for (int k = KA; k < K; ++k) sp_cell<P, K, CUT>(x, k, eq, k + 1 < K ? x.E[k + 1] : uE, F, z, c);
    F1 = F;
}

// Highest score, then first cell, over the G lanes of a segment; the alignment it stands for.
template <int G>
__device__ __forceinline__ void sw_finish(int32_t best, uint32_t cell, uint32_t start, const DevHsp &h, bool on, int32_t w,
                                          DevAln &res) {
#pragma unroll
    for (int d = G / 2; d > 0; d >>= 1) {
        const int32_t ob = __shfl_xor_sync(0xffffffffu, best, d);
        const uint32_t oc = __shfl_xor_sync(0xffffffffu, cell, d), os = __shfl_xor_sync(0xffffffffu, start, d);
        if (ob > best || (ob == best && oc < cell)) { best = ob; cell = oc; start = os; }
    }
    res.qi = h.qi; res.seq = h.seq; res.qs = res.qe = res.ds = res.de = 0; res.score = 0; res.pad = 0;
    if (on && best > 0) {
        const uint32_t bm = (1u << SW_SHIFT) - 1u;
        const int64_t d_s = (int64_t)h.ds - h.qs, d_e = (int64_t)h.de - h.qe, dlo = min(d_s, d_e) - w;
        const int64_t I0 = max((int64_t)0, (int64_t)h.qs - w);
        const int64_t i1 = I0 + (cell >> SW_SHIFT) - 1, i0 = I0 + (start >> SW_SHIFT);  // cell: a row on
        res.qs = (uint32_t)i0; res.qe = (uint32_t)(i1 + 1);
        res.ds = (uint32_t)(i0 + dlo + (start & bm)); res.de = (uint32_t)(i1 + dlo + (cell & bm) + 1);
        res.score = best;
    }
}

// Aligns each segment's HSP h (where on; a band of at most G K offsets, at most SW_MAX_ROWS
// rows); every lane of the segment gets the alignment.
template <int G, int KA, int KB, bool CUT>
__device__ __forceinline__ void sw_band(const DevHsp &h, bool on, const PackedPair &q, const uint64_t *__restrict__ qstart,
                                        const uint64_t *__restrict__ seq_start, const SwScore &c, int32_t w, DevAln &res) {
    const int sl = (threadIdx.x & 31) % G;
    constexpr int K = KA + KB;
    SwSet<K> x;
    int32_t T = 0;
    {
        SwGeom g{};
        if (on) {
            g.set(h, qstart, seq_start, w);
            T = (int32_t)max(g.qhi - g.qlo, (int64_t)0) + (g.B - 1) / K;
        }
        x.start(g, on, K * sl, sl);
    }
    if (G < 32) T = (int32_t)__reduce_max_sync(0xffffffffu, (uint32_t)T);
    int32_t F1 = SW_NEG;
    uint32_t SF1 = 0;
    for (int32_t t0 = 0; t0 < T; t0 += 16) {
        const bool no = __any_sync(0xffffffffu, x.load(q));
        x.q += 16; x.d += 16;
        const int32_t t1 = min(t0 + 16, T);
        if (no) {
#pragma unroll 1
            for (int32_t t = t0; t < t1; ++t) sw_row<G, KA, KB, true, CUT>(x, F1, SF1, sl, c);
        } else {
#pragma unroll 1
            for (int32_t t = t0; t < t1; ++t) sw_row<G, KA, KB, false, CUT>(x, F1, SF1, sl, c);
        }
    }
    sw_finish<G>(x.best, x.bcell, x.bstart, h, on, w, res);
}

// sw_band on packed cells, for HSPs that fit them.  table (null: none; a word for each of the warp's
// 2 K + 1 cells a lane): the rows of start cells count from the 16 rows at hand, and a start before
// them is named by its place in the table, where the starts of all cells that still count are
// put after every 16 rows; with 5 bits of row and as many places a score of 18 (15) bits fits.  A
// tenth more instructions than without the table.  us, tracked | table, where the longest alignments
// have over 2,047 rows: 1,000 queries of up to 10,000 bases 291 | 265, 8 long queries 268 | 237.
template <int G, int KA, int KB, int OFF, int ROW, bool TABLE, bool CUT>
__device__ __forceinline__ void sp_band(const DevHsp &h, bool on, const PackedPair &q, const uint64_t *__restrict__ qstart,
                                        const uint64_t *__restrict__ seq_start, const SwScore &score, int32_t w,
                                        uint32_t *table, DevAln &res) {
    typedef SwPack<OFF, ROW> P;
    constexpr uint32_t CODE = (1u << P::CHOICE) - 1u, PLACES = TABLE ? 32 * (2 * (KA + KB) + 1) : 0;
    static_assert(!TABLE || PLACES + (17u << OFF) <= CODE + 1, "places and 17 rows of starts fit");
    static_assert(G * (KA + KB) <= 1 << OFF, "an offset fits its bits");
    const int sl = (threadIdx.x & 31) % G;
    constexpr int K = KA + KB;
    const P c(score);
    SwSet<K> x;
    int32_t T = 0;
    {
        SwGeom g{};
        if (on) {
            g.set(h, qstart, seq_start, w);
            T = (int32_t)max(g.qhi - g.qlo, (int64_t)0) + (g.B - 1) / K;
        }
        x.start(g, on, K * sl, sl);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) { x.H[k] = sl == 0 ? (int32_t)PLACES + k : 0; x.E[k] = P::NEG; }
    x.bstart = (uint32_t)P::LOW;
    x.SH[0] = (uint32_t)(-sl * (1 << OFF) + K * sl);
    if (G < 32) T = (int32_t)__reduce_max_sync(0xffffffffu, (uint32_t)T);
    int32_t F1 = P::NEG, best = 0;  // best: the word whose start is best_start
    uint32_t best_start = 0;
    for (int32_t t0 = 0; t0 < T; t0 += 16) {
        if (TABLE) x.SH[0] = PLACES + (uint32_t)(K * sl);
        const bool no = __any_sync(0xffffffffu, x.load(q));
        x.q += 16; x.d += 16;
        const int32_t t1 = min(t0 + 16, T);
        if (no) {
#pragma unroll 1
            for (int32_t t = t0; t < t1; ++t) sp_row<P, OFF, G, KA, KB, true, CUT>(x, F1, sl, c);
        } else {
#pragma unroll 1
            for (int32_t t = t0; t < t1; ++t) sp_row<P, OFF, G, KA, KB, false, CUT>(x, F1, sl, c);
        }
        if constexpr (TABLE) {
            auto cell_of = [&](int32_t word) {
                const uint32_t code = (uint32_t)word & CODE, n = code - PLACES;  // n: from PLACES on
                const uint32_t off = n & ((1u << OFF) - 1u), row = (uint32_t)t0 + (n >> OFF) - off / (uint32_t)K;
                return code < PLACES ? table[code] : row << SW_SHIFT | off;
            };
            uint32_t cell[2 * K + 1];
#pragma unroll
            for (int k = 0; k < K; ++k) { cell[2 * k] = cell_of(x.H[k]); cell[2 * k + 1] = cell_of(x.E[k]); }
            cell[2 * K] = cell_of(F1);
            if (x.best != best) { best = x.best; best_start = cell_of(best); }
            __syncwarp();
            const uint32_t place = (uint32_t)(threadIdx.x & 31) * (2 * K + 1);
#pragma unroll
            for (int i = 0; i < 2 * K + 1; ++i) table[place + i] = cell[i];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                x.H[k] = (x.H[k] & ~(int32_t)CODE) | (int32_t)(place + 2 * k);
                x.E[k] = (x.E[k] & ~(int32_t)CODE) | (int32_t)(place + 2 * k + 1);
            }
            F1 = (F1 & ~(int32_t)CODE) | (int32_t)(place + 2 * K);
            __syncwarp();
        }
    }
    if (!TABLE) {
        const uint32_t start = (uint32_t)x.best & CODE;
        best_start = (start >> OFF) << SW_SHIFT | (start & ((1u << OFF) - 1u));
    }
    sw_finish<G>(x.best >> P::SCORE, x.bcell, best_start, h, on, w, res);
}

// What the number of alignments, known on the device only, decides: see the alignment kernels'
// launch in search().
__device__ __forceinline__ bool sw_many(uint32_t n, uint32_t sms) { return n > sms * 64u; }
__device__ __forceinline__ uint32_t sw_long_rows(uint32_t n, uint32_t sms) {
    return n <= sms * 4u ? 1u : sw_many(n, sms) ? 1024u : 512u;
}

// Alignments of the selected HSPs, longest first (order): the first n_long tasks a warp each
// (32 lanes with two offsets: the shortest rows, for the alignments that would bound the
// kernel's time), the others 32 / G to a warp.  Bands over 64 diagonals (and windows of
// SW_MAX_ROWS rows) go to the list that k_banded_sw_wide takes.  <8, 3, 2> covers bands of up to
// 40 diagonals (33 and up at the default width), <16, 2, 1> 48; k_sw_prepare counts tasks with
// wider bands, up to 64, among the long ones.
template <int G, int KA, int KB, bool CUT>
__global__ void __launch_bounds__(128) k_banded_sw(const DevHsp *__restrict__ sel, const uint64_t *__restrict__ n_dev,
                                                   uint32_t sms, PackedPair q,
                                                   const uint64_t *__restrict__ qstart,
                                                   const uint64_t *__restrict__ seq_start, SwScore c, int32_t w,
                                                   uint32_t *__restrict__ next_task, const uint32_t *__restrict__ order,
                                                   uint32_t *__restrict__ wide, uint32_t *__restrict__ wide_count,
                                                   const uint32_t *__restrict__ n_long, uint32_t *__restrict__ next_long,
                                                   DevAln *__restrict__ out) {
    __shared__ uint32_t table[4][32 * 5];
    const int lane = threadIdx.x & 31, seg = lane / G;
    const uint32_t n = (uint32_t)*n_dev, nl = order ? *n_long : n;  // no order: a warp each
    if (!sw_many(n, sms) && blockIdx.x >= sms) return;  // four warps an SM (see the launch)
    // the task at place j of the order, if a register path of `cap` offsets takes it; wider ones
    // are listed by the lane `lists`
    auto take = [&](uint32_t j, uint32_t end, int cap, bool lists, uint32_t &task, DevHsp &h) {
        if (j >= end) return false;
        task = order ? order[j] : j;
        h = sel[task];
        const int64_t rows = (int64_t)h.qe - h.qs + 2 * (int64_t)w;
        if (dev_band(h, w) <= cap && rows <= SW_MAX_ROWS) return true;
        if (lists) wide[atomicAdd(wide_count, 1u)] = task;
        return false;
    };
    for (;;) {
        uint32_t j = 0;
        if (lane == 0) j = atomicAdd(next_long, 1u);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= nl) break;
        uint32_t task = 0;
        DevHsp h{};
        if (!take(j, nl, 64, lane == 0, task, h)) continue;
        DevAln res;
        if (SwPack<6, 11>::fits((int64_t)h.qe - h.qs + 2 * (int64_t)w, c))
            sp_band<32, 1, 1, 6, 11, false, CUT>(h, true, q, qstart, seq_start, c, w, nullptr, res);
        else if (SwPack<6, 5>::fits((int64_t)h.qe - h.qs + 2 * (int64_t)w, c, true))
            sp_band<32, 1, 1, 6, 5, true, CUT>(h, true, q, qstart, seq_start, c, w, table[threadIdx.x >> 5], res);
        else
            sw_band<32, 1, 1, CUT>(h, true, q, qstart, seq_start, c, w, res);
        if (lane == 0) out[task] = res;
    }
    constexpr uint32_t NT = 32 / G;
    for (;;) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(next_task, NT);
        base = __shfl_sync(0xffffffffu, base, 0) + nl;
        if (base >= n) return;
        uint32_t task = 0;
        DevHsp h{};
        const bool first = lane % G == 0, on = take(base + seg, n, G * (KA + KB), first, task, h);
        if (!__any_sync(0xffffffffu, on)) continue;
        DevAln res;
        if (__all_sync(0xffffffffu, !on || SwPack<6, 11>::fits((int64_t)h.qe - h.qs + 2 * (int64_t)w, c)))
            sp_band<G, KA, KB, 6, 11, false, CUT>(h, on, q, qstart, seq_start, c, w, nullptr, res);
        else
            sw_band<G, KA, KB, CUT>(h, on, q, qstart, seq_start, c, w, res);
        if (on && first) out[task] = res;
    }
}

// Bands wider than 64 diagonals, a warp each: up to SW_MAX_BAND offsets in registers; still
// wider ones are listed, with the widest band, for k_banded_sw_strip.  A kernel of its own, so
// that its registers do not limit the main alignment kernel.
template <bool CUT>
__global__ void __launch_bounds__(128) k_banded_sw_wide(const DevHsp *__restrict__ sel, const uint32_t *__restrict__ wide,
                                                        const uint32_t *__restrict__ wide_count,
                                                        uint32_t *__restrict__ next, PackedPair q,
                                                        const uint64_t *__restrict__ qstart,
                                                        const uint64_t *__restrict__ seq_start, SwScore c, int32_t w,
                                                        uint32_t *__restrict__ strip, uint32_t *__restrict__ strip_count,
                                                        uint32_t *__restrict__ strip_band, DevAln *__restrict__ out) {
    __shared__ uint32_t table[4][32 * 19];
    const int lane = threadIdx.x & 31;
    const uint32_t n = *wide_count;
    for (;;) {
        uint32_t j = 0;
        if (lane == 0) j = atomicAdd(next, 1u);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= n) return;
        const uint32_t task = wide[j];
        const DevHsp h = sel[task];
        const int64_t B = dev_band(h, w);
        if (B <= SW_MAX_BAND && (int64_t)h.qe - h.qs + 2 * (int64_t)w <= SW_MAX_ROWS) {
            DevAln res;
            if (SwPack<9, 9>::fits((int64_t)h.qe - h.qs + 2 * (int64_t)w, c))
                sp_band<32, 5, 4, 9, 9, false, CUT>(h, true, q, qstart, seq_start, c, w, nullptr, res);
            else if (SwPack<9, 5>::fits((int64_t)h.qe - h.qs + 2 * (int64_t)w, c, true))
                sp_band<32, 5, 4, 9, 5, true, CUT>(h, true, q, qstart, seq_start, c, w, table[threadIdx.x >> 5], res);
            else
                sw_band<32, 5, 4, CUT>(h, true, q, qstart, seq_start, c, w, res);
            if (lane == 0) out[task] = res;
        } else if (lane == 0) {
            strip[atomicAdd(strip_count, 1u)] = task;
            atomicMax(strip_band, (uint32_t)min(B, (int64_t)65536));
        }
        __syncwarp();
    }
}

// The listed alignments on the strip path, each warp with a strip of strip_cells cells.
__global__ void __launch_bounds__(128) k_banded_sw_strip(const DevHsp *__restrict__ sel, const uint32_t *__restrict__ strip,
                                                         uint32_t n, uint32_t *__restrict__ next,
                                                         SwCell *__restrict__ strips, uint64_t strip_cells, PackedPair q,
                                                         const uint64_t *__restrict__ qstart,
                                                         const uint64_t *__restrict__ seq_start, SwScore c, int32_t w,
                                                         DevAln *__restrict__ out, uint32_t *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    SwCell *row = strips + (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * strip_cells;
    for (;;) {
        uint32_t j = 0;
        if (lane == 0) j = atomicAdd(next, 1u);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= n) return;
        sw_task_strip(sel, strip[j], row, q.qpk, q.qnb, qstart, q.bpk, q.bnb, seq_start, c.match, c.mismatch, c.goe - c.ge,
                      c.ge, w, out, status);
        __syncwarp();
    }
}

// Alignment order: the longest first (they bound the phase's time), alignments of similar
// length together.  Each task falls in one of SWO_BINS bins by its DP-window rows, four a
// factor of two, falling; the first half of the bins takes the tasks that get a warp each: those
// of at least long_rows rows, and those whose bands are wider than the grouped path's `cap`
// offsets, up to 64.  k_sw_prepare counts the bins (hist) and, for the kernel times, the band
// area (rows x band, the cells the alignment kernels evaluate) of bands of at most 64 diagonals
// and of wider ones; k_sw_order places each task after the bins before its own.
constexpr int SWO_BINS = 128;

__device__ __forceinline__ uint32_t sw_bin(const DevHsp &x, int32_t w, int cap, const uint64_t *__restrict__ qstart,
                                           uint32_t long_rows, int64_t &rows) {
    const int64_t m = (int64_t)(qstart[x.qi + 1] - qstart[x.qi]), b = dev_band(x, w);
    rows = max(min(m, (int64_t)x.qe + w) - max((int64_t)0, (int64_t)x.qs - w), (int64_t)0);
    const uint32_t r = (uint32_t)min(rows, (int64_t)65535);
    const int e = 31 - __clz(r | 1u);  // 0 .. 15
    const uint32_t quarter = e >= 2 ? (r >> (e - 2)) & 3u : (r << (2 - e)) & 3u;
    const uint32_t bin = 63u - (uint32_t)(4 * e) - quarter;
    return (r >= long_rows || (b > cap && b <= 64)) ? bin : bin + 64u;
}

__global__ void __launch_bounds__(256) k_sw_prepare(const DevHsp *__restrict__ h, const uint64_t *__restrict__ n_dev,
                                                    int32_t w, int cap, const uint64_t *__restrict__ qstart,
                                                    uint32_t long_rows, uint32_t sms, uint32_t *__restrict__ hist,
                                                    unsigned long long *__restrict__ cells) {
    __shared__ uint32_t s_hist[SWO_BINS];
    const uint32_t n = (uint32_t)*n_dev, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x * blockDim.x >= n) return;
    if (!long_rows) long_rows = sw_long_rows(n, sms);
    for (int j = threadIdx.x; j < SWO_BINS; j += blockDim.x) s_hist[j] = 0u;
    __syncthreads();
    if (i < n) {
        const DevHsp x = h[i];
        int64_t rows;
        atomicAdd(&s_hist[sw_bin(x, w, cap, qstart, long_rows, rows)], 1u);
        if (cells && rows) {
            const int64_t b = dev_band(x, w);
            atomicAdd(cells + (b > 64 ? 1 : 0), (unsigned long long)(rows * b));
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < SWO_BINS; j += blockDim.x)
        if (s_hist[j]) atomicAdd(&hist[j], s_hist[j]);
}

__global__ void __launch_bounds__(256) k_sw_order(const DevHsp *__restrict__ h, const uint64_t *__restrict__ n_dev,
                                                  int32_t w, int cap, const uint64_t *__restrict__ qstart,
                                                  uint32_t long_rows, uint32_t sms, const uint32_t *__restrict__ hist,
                                                  uint32_t *__restrict__ placed, uint32_t *__restrict__ order,
                                                  uint32_t *__restrict__ n_long) {
    __shared__ uint32_t base[SWO_BINS], count[SWO_BINS], warp_tot[8];
    const uint32_t n = (uint32_t)*n_dev, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x * blockDim.x >= n) return;
    if (!long_rows) long_rows = sw_long_rows(n, sms);
    uint32_t tot = 0;
    const uint32_t before = block_excl_scan(threadIdx.x < SWO_BINS ? hist[threadIdx.x] : 0u, warp_tot, tot);
    if (threadIdx.x < SWO_BINS) {
        base[threadIdx.x] = before;
        count[threadIdx.x] = 0u;
    }
    if (blockIdx.x == 0 && threadIdx.x == SWO_BINS / 2) *n_long = before;
    __syncthreads();
    uint32_t bin = 0, rank = 0;
    if (i < n) {
        int64_t rows;
        bin = sw_bin(h[i], w, cap, qstart, long_rows, rows);
        rank = atomicAdd(&count[bin], 1u);
    }
    __syncthreads();
    if (threadIdx.x < SWO_BINS && count[threadIdx.x])
        base[threadIdx.x] += atomicAdd(&placed[threadIdx.x], count[threadIdx.x]);
    __syncthreads();
    if (i < n) order[base[bin] + rank] = i;
}

// ------------------------------------------------------ a13: ranking --
__global__ void k_dup_flags(const DevAln *__restrict__ a, uint32_t n, uint32_t *__restrict__ flag) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const DevAln x = a[i];
    bool keep = x.score > 0;
    if (keep && i > 0) {
        const DevAln y = a[i - 1];
        if (y.qi == x.qi && y.seq == x.seq && y.qs == x.qs && y.qe == x.qe && y.ds == x.ds && y.de == x.de)
            keep = false;
    }
    flag[i] = keep ? 1u : 0u;
}

__global__ void k_finalize(const DevAln *__restrict__ a, uint32_t n, const uint32_t *__restrict__ first,
                           const uint64_t *__restrict__ qstart, double n_bank, double lambda, double K,
                           double max_e, gn_hit *__restrict__ out, uint32_t *__restrict__ flag) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const DevAln x = a[i];
    double m = (double)(qstart[x.qi + 1] - qstart[x.qi]);
    gn_hit h;
    h.query = x.qi; h.seq = x.seq; h.q_start = x.qs; h.q_end = x.qe; h.db_start = x.ds; h.db_end = x.de;
    h.score = x.score;
    h.rank = i - first[x.qi];
    h.evalue = K * m * n_bank * exp(-lambda * (double)x.score);
    h.bits = (lambda * (double)x.score - log(K)) / log(2.0);
    out[i] = h;
    flag[i] = (h.evalue <= max_e) ? 1u : 0u;
}


// Per-query ranking (alignments of a query are contiguous and at most RQ_CAP): a block sorts a
// query's records by (score desc, seq, q_start, db_start, q_end, db_end), drops records that repeat
// an earlier one's sequence and ranges (and records with score <= 0), and writes the ranked hits
// with e-value and bit score at the query's input offset.  The sort moves keys of score, sequence
// and record in registers (Team) and compares the records only where score and sequence are
// equal; a table of the ranges, each with the first record that has them, finds the repeats.  Bound
// by the latency of the sort's stages.  Two sorts of record indices in shared memory, by ranges and
// by rank, took 123 us for 200 queries of up to 875 alignments (now 49), 61 for 4,096 queries of 22
// (35) and 55 for 2,000 of 100 (37).  Up to RQ_SMALL alignments a block of a thread each: a warp
// with four records a lane took 53 and 49 us (and 14 instead of 10 for a lone record: more code
// to fetch).
constexpr int RQ_CAP = 1024, RQ_SMALL = 128, RQ_BITS = 10;

__device__ __forceinline__ bool rq_less_rank(const DevAln &a, const DevAln &b) {
    if (a.score != b.score) return a.score > b.score;
    if (a.seq != b.seq) return a.seq < b.seq;
    if (a.qs != b.qs) return a.qs < b.qs;
    if (a.ds != b.ds) return a.ds < b.ds;
    if (a.qe != b.qe) return a.qe < b.qe;
    return a.de < b.de;
}

// E: records a thread sorts; the block's T threads take up to T E.  seq_bits: of a sequence number.
// qo: first alignment of each query, as a prefix sum.  A query of more alignments is left out and
// *too_many set: the caller then ranks the call by sorting.
template <int T, int E>
__global__ void __launch_bounds__(T) k_rank_query(const DevAln *__restrict__ aln, const uint64_t *__restrict__ qo,
                                                  uint32_t nq, const uint64_t *__restrict__ qstart, int seq_bits, double n_bank,
                                                  double lambda, double K, double max_e, gn_hit *__restrict__ out,
                                                  uint32_t *__restrict__ qcount, uint32_t *__restrict__ too_many) {
    typedef Team<T, E> tm;
    constexpr uint32_t CAP = T * E, SLOTS = 2 * CAP, EMPTY = 0xFFFFFFFFu, idx_mask = (1u << RQ_BITS) - 1u;
    static_assert(CAP <= 1u << RQ_BITS, "an index fits its bits");
    __shared__ DevAln rec[CAP];
    __shared__ uint64_t ex[CAP];  // the sort's exchanges, then the table
    __shared__ uint64_t tmp[33];
    __shared__ uint16_t order[CAP], slot[CAP];
    __shared__ uint32_t n_out;
    uint32_t *table = reinterpret_cast<uint32_t *>(ex);
    const uint32_t t = threadIdx.x;
    const int kept = min(seq_bits, 64 - 31 - RQ_BITS);  // bits of the sequence in the key, the high ones
    for (uint32_t q = blockIdx.x; q < nq; q += gridDim.x) {
        const uint64_t start = qo[q];
        const uint32_t n = (uint32_t)(qo[q + 1] - start);
        if (n == 0 || n > CAP) {
            if (t == 0) {
                qcount[q] = 0;
                if (n) *too_many = 1u;
            }
            continue;
        }
        for (uint32_t i = t; i < n; i += T) rec[i] = aln[start + i];
        if (t == 0) n_out = 0;
        __syncthreads();
        {
            uint64_t r[E];
            const uint32_t P = tm::padded(n), A = P / E;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t i = e * A + t;
                r[e] = ~0ull;
                if (t < A && i < n) {
                    const uint64_t score = 0x7FFFFFFFu - (uint32_t)max(rec[i].score, 0);
                    r[e] = ((score << kept | rec[i].seq >> (seq_bits - kept)) << RQ_BITS) | i;
                }
            }
            tm::sort(r, ex, P, [&](uint64_t a, uint64_t b) {
                if (a >> RQ_BITS != b >> RQ_BITS || a == ~0ull || b == ~0ull) return a < b;
                const DevAln &x = rec[(uint32_t)a & idx_mask], &y = rec[(uint32_t)b & idx_mask];
                if (rq_less_rank(x, y)) return true;
                return !rq_less_rank(y, x) && a < b;
            });
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e)  // (an alignment without a score may equal the padding: it is dropped)
                if (t * E + e < n) order[t * E + e] = r[e] == ~0ull ? 0xFFFFu : (uint16_t)((uint32_t)r[e] & idx_mask);
        }
        for (uint32_t i = t; i < SLOTS; i += T) table[i] = EMPTY;
        __syncthreads();
        // each range's entry: its first place in the order, and the record there
        for (uint32_t i = t; i < n; i += T) {
            const uint32_t x = order[i];
            slot[i] = 0xFFFFu;
            if (x == 0xFFFFu || rec[x].score <= 0) continue;
            const DevAln a = rec[x];
            const uint32_t entry = i << RQ_BITS | x;
            uint32_t h = a.seq * 0x9E3779B1u ^ a.qs * 0x85EBCA77u ^ a.qe * 0xC2B2AE3Du ^ a.ds * 0x27D4EB2Fu ^ a.de * 0x165667B1u;
            for (h = (h >> 16 ^ h) & (SLOTS - 1);; h = (h + 1) & (SLOTS - 1)) {  // half the slots stay empty
                const uint32_t old = atomicCAS(&table[h], EMPTY, entry);
                if (old == EMPTY) break;
                const DevAln &b = rec[old & idx_mask];
                if (a.seq == b.seq && a.qs == b.qs && a.qe == b.qe && a.ds == b.ds && a.de == b.de) {
                    atomicMin(&table[h], entry);
                    break;
                }
            }
            slot[i] = (uint16_t)h;
        }
        __syncthreads();
        const double m = (double)(qstart[q + 1] - qstart[q]);
        uint32_t placed = 0;
        for (uint32_t i0 = 0; i0 < n; i0 += T) {
            const uint32_t i = i0 + t;
            const bool keep = i < n && slot[i] != 0xFFFFu && table[slot[i]] >> RQ_BITS == i;
            uint32_t tot = 0;
            const uint32_t k = placed + tm::excl_sum(keep ? 1u : 0u, tmp, tot);
            placed += tot;
            if (!keep) continue;
            const DevAln &x = rec[order[i]];
            gn_hit h;
            h.query = x.qi; h.seq = x.seq; h.q_start = x.qs; h.q_end = x.qe; h.db_start = x.ds; h.db_end = x.de;
            h.score = x.score;
            h.rank = k;
            h.evalue = K * m * n_bank * exp(-lambda * (double)x.score);
            h.bits = (lambda * (double)x.score - log(K)) / log(2.0);
            // e-values rise as scores fall, so the cut keeps a prefix of the ranking
            if (h.evalue <= max_e) {
                out[start + k] = h;
                atomicAdd(&n_out, 1u);
            }
        }
        __syncthreads();
        if (t == 0) qcount[q] = n_out;
        __syncthreads();
    }
}

__global__ void k_gather_ranked(const gn_hit *__restrict__ in, const uint64_t *__restrict__ from,
                                const uint64_t *__restrict__ qoff, uint32_t nq, gn_hit *__restrict__ out) {
    for (uint32_t q = blockIdx.x; q < nq; q += gridDim.x) {
        const uint64_t start = from[q], o = qoff[q], c = qoff[q + 1] - o;
        for (uint32_t k = threadIdx.x; k < c; k += blockDim.x) out[o + k] = in[start + k];
    }
}

// ------------------------------------------------------------ compaction --
__global__ void k_scatter_flagged(const uint32_t *__restrict__ in, int W, const uint32_t *__restrict__ flags,
                                  const uint64_t *__restrict__ pos, uint32_t n, uint32_t *__restrict__ out) {
    uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (uint64_t)n * W) return;
    uint32_t i = (uint32_t)(t / W), w = (uint32_t)(t % W);
    if (flags[i]) out[pos[i] * W + w] = in[t];
}

const uint64_t *compact_records_async(const uint32_t *in, int W, const uint32_t *flags, uint32_t n, uint32_t *out,
                                      DeviceArena &arena, cudaStream_t s) {
    uint64_t *pos = arena.alloc_n<uint64_t>(n + 1ull);
    void *scr = arena.alloc(scan_scratch_bytes(n));
    exclusive_scan_u32(flags, pos, n, scr, s);
    const uint64_t tot = (uint64_t)n * W;
    if (n)
        GN_LAUNCH("k_scatter_flagged", n, s,
                  k_scatter_flagged<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(in, W, flags, pos, n, out));
    return pos + n;
}

uint32_t compact_records(const uint32_t *in, int W, const uint32_t *flags, uint32_t n, uint32_t *out,
                         DeviceArena &arena, cudaStream_t s) {
    if (n == 0) return 0;
    const uint64_t *count = compact_records_async(in, W, flags, n, out, arena, s);
    uint64_t cnt = 0;
    GN_CUDA(cudaMemcpyAsync(&cnt, count, sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    GN_CUDA(cudaStreamSynchronize(s));
    return (uint32_t)cnt;
}

// ---------------------------------------------------------------- driver --
namespace {
struct PhaseTimer {
    cudaStream_t s;
    HostPool &pool;
    std::vector<std::pair<const char *, cudaEvent_t>> marks;
    PhaseTimer(cudaStream_t st, HostPool &pl) : s(st), pool(pl) {}
    void mark(const char *name) {
        cudaEvent_t e = pool.take_event();
        if (!e) return;
        cudaEventRecord(e, s);
        marks.emplace_back(name, e);
    }
    void finish(std::vector<std::pair<const char *, float>> &out) {
        out.clear();
        for (size_t i = 1; i < marks.size(); ++i) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, marks[i - 1].second, marks[i].second);
            out.emplace_back(marks[i].first, ms);
        }
    }
    ~PhaseTimer() {
        for (auto &m : marks) pool.give_event(m.second);
    }
};

template <class T>
std::vector<T> to_host(const T *d, size_t n, cudaStream_t s) {
    std::vector<T> h(n);
    if (n) {
        GN_CUDA(cudaMemcpyAsync(h.data(), d, sizeof(T) * n, cudaMemcpyDeviceToHost, s));
        GN_CUDA(cudaStreamSynchronize(s));
    }
    return h;
}

// A few words from the device, fetched between two kernels and read while the second one runs.
struct GroupQuestion {
    HostPool &pool;
    cudaStream_t s;
    PinnedBlock pin;
    cudaEvent_t done = nullptr;
    GroupQuestion(HostPool &pl, cudaStream_t st) : pool(pl), s(st), pin(pl, 64, st) {}
    void ask(const uint32_t *dev) {
        pin.fetch(0, dev, 16);
        if (!done) done = pool.take_event();
        if (done) GN_CUDA(cudaEventRecord(done, s));
    }
    void answer(uint32_t *out) {
        if (done) {
            GN_CUDA(cudaEventSynchronize(done));
            pin.in_flight = false;
        } else {
            pin.wait();
        }
        memcpy(out, pin.p, 16);
    }
    ~GroupQuestion() {
        if (done) pool.give_event(done);
    }
};

// Resident blocks of a kernel without dynamic shared memory, asked of the driver once per kernel
// and device (a search asks for five).
int blocks_per_sm(const void *fn, int threads) {
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, int> known;
    int dev = 0;
    GN_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    int &n = known[{fn, dev}];
    if (!n) {
        int occ = 0;
        GN_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, 0));
        n = std::max(occ, 1);
    }
    return n;
}

unsigned blocks_for(uint64_t n, unsigned t = 256) { return (unsigned)std::max<uint64_t>(1, (n + t - 1) / t); }

// A hit-storing path is asked for: the path itself, or one of the settings that only the
// buckets have.
bool hit_path_forced() {
    for (const char *v : {"GN_HIT_GROUPING", "GN_TILE_FILTER", "GN_TILE_POS", "GN_TILE_FBITS", "GN_TILE_FBITS2",
                          "GN_FILL_THREADS", "GN_BUCKET_TARGET", "GN_BUCKET_CAP", "GN_SPILL_ROOM"})
        if (getenv(v)) return true;
    return false;
}

// Lets the kernels with a per-call dynamic shared-memory size use up to the device's opt-in
// maximum.  Set once per device: concurrent searches (serving threads) launch with different
// sizes, and a per-call attribute change by one thread could undercut another's launch.
void allow_max_smem(int device) {
    static std::mutex mu;
    static bool done[64] = {false};
    std::lock_guard<std::mutex> lk(mu);
    if (device < 0 || device >= 64 || done[device]) return;
    int optin = 0;
    GN_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    auto allow = [&](const void *fn) {  // the opt-in maximum less the kernel's static shared memory
        cudaFuncAttributes fa;
        GN_CUDA(cudaFuncGetAttributes(&fa, fn));
        GN_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes));
    };
    allow(reinterpret_cast<const void *>(k_bucket_fill<0, 0>));
    allow(reinterpret_cast<const void *>(k_bucket_fill<19, 17>));
    allow(reinterpret_cast<const void *>(k_bucket_group_warp));
    allow(reinterpret_cast<const void *>(k_merge_groups<1024, MG_BIG / 1024, false>));
    allow(reinterpret_cast<const void *>(k_merge_groups<1024, MG_BIG / 1024, true>));
    done[device] = true;
}
}  // namespace

// Both strands: query i of the input becomes query 2i (the bases as given) and query
// 2i + 1 (its reverse complement) of the output, back to back.  Complement: A <-> T,
// C <-> G in either case, U (read as T) -> A; any other byte is a non-base and stays.
__device__ __forceinline__ uint8_t dev_complement(uint8_t c) {
    switch (c) {
        case 'A': return 'T'; case 'T': return 'A'; case 'U': return 'A';
        case 'C': return 'G'; case 'G': return 'C';
        case 'a': return 't'; case 't': return 'a'; case 'u': return 'a';
        case 'c': return 'g'; case 'g': return 'c';
        default: return c;
    }
}
__global__ void k_both_strands(const uint8_t *__restrict__ in, const uint64_t *__restrict__ qstart, uint32_t nq,
                               uint64_t M, uint8_t *__restrict__ out) {
    const uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= M) return;
    const uint32_t i = dev_upper_index(qstart, nq + 1, x);
    const uint64_t s0 = qstart[i], m = qstart[i + 1] - s0, p = x - s0;
    const uint8_t c = in[x];
    out[2 * s0 + p] = c;
    out[2 * s0 + m + (m - 1 - p)] = dev_complement(c);
}

void both_strands(const uint8_t *qbases_dev, const std::vector<uint64_t> &qstart_h, DeviceArena &arena,
                  cudaStream_t s, const uint8_t **out_bases, std::vector<uint64_t> &out_start) {
    const uint32_t nq = (uint32_t)(qstart_h.size() - 1);
    const uint64_t M = qstart_h[nq];
    out_start.assign(2ull * nq + 1, 0);
    for (uint32_t i = 0; i < nq; ++i) {
        const uint64_t m = qstart_h[i + 1] - qstart_h[i];
        out_start[2 * i + 1] = 2 * qstart_h[i] + m;
        out_start[2 * i + 2] = 2 * qstart_h[i] + 2 * m;
    }
    uint8_t *d = arena.alloc_n<uint8_t>(2 * M);
    uint64_t *qs = arena.alloc_n<uint64_t>(nq + 1);
    GN_CUDA(cudaMemcpyAsync(qs, qstart_h.data(), 8ull * (nq + 1), cudaMemcpyHostToDevice, s));
    if (M) GN_LAUNCH("k_both_strands", M, s, k_both_strands<<<blocks_for(M), 256, 0, s>>>(qbases_dev, qs, nq, M, d));
    *out_bases = d;
}

// Words that a search's kernels write and its host code reads.
struct SearchWords {
    uint32_t wait_status, status;
    uint32_t n_hsp, next_cand;         // of the signature scan's range: HSPs, candidates,
    unsigned long long n_cand;         // and list units of all offsets
    uint32_t next_tile, scan_pad;
    unsigned long long n_units;
    uint32_t n_wide, next_wide, next_task, n_long, next_long;
    uint32_t n_strip, strip_band, next_strip;
    uint32_t too_many, recs_done;
    uint32_t groups[8];                // groups of a block, of a large block, of no kernel: of the join, of the merge
    unsigned long long next_end, cells[2];
    uint32_t bins[SWO_BINS], placed[SWO_BINS];
};
static_assert(sizeof(SearchWords) % 8 == 0, "SearchWords is followed by 64-bit words");

// Alignments that a search makes room for without asking how many there are (180 MB).
constexpr uint32_t SEL_ASK = 1u << 20;

// Seed lookup and chaining take one of two routes to the same HSPs.  The signature scan
// (gn_seed_scan.cuh) reads each occurrence's signature once and stores no hit; it serves
// searches in which a chain needs two hits (min_hsp_len > span) at most SIG_FIELDS windows
// apart (with SIG_FLANK: windows that overlap or touch), the distances a signature holds.
// Everything else, and a search for which a hit-storing path is forced, goes through the
// buckets or the global sort below.  Where both serve, the scan is faster at every size
// measured (scan and chains against fill, grouping and the sort of its spills): one query of
// 2,000 bases on 4 Gbp 29 against 36 us; 4,096 short queries on 400 Mbp 0.18 against 0.60 ms;
// 2,000 queries on 4 Gbp 1.46 against 3.70 ms; 500 queries at stride 1 0.13 against 3.2 ms.
bool takes_scan(const gn_index *ix, const gn_params &p) {
    const uint32_t links = p.max_hit_distance / (uint32_t)ix->t;  // windows from one hit to the next, at most
    return ix->sig_d && p.min_hsp_len > (uint32_t)ix->span && !(p.flags & GN_FLAG_KEEP_HITS) && !hit_path_forced() && links >= 1 &&
           links <= (uint32_t)(sig_kind(ix->k, ix->span, ix->t) == SIG_FLANK ? ix->k : SIG_FIELDS);
}

// Candidates that a list is enlarged to without asking for the free memory (256 MB).
constexpr uint64_t CAND_ASK = 1ull << 25;

// Segments of a query set: one per MAX_QUERY_LEN bases or part, SEG_STEP apart (see search).
uint64_t count_segments(const std::vector<uint64_t> &qstart) {
    uint64_t n = 0;
    for (size_t i = 0; i + 1 < qstart.size(); ++i) {
        const uint64_t m = qstart[i + 1] - qstart[i];
        n += m <= MAX_QUERY_LEN ? 1 : 1 + (m - MAX_QUERY_LEN + SEG_STEP - 1) / SEG_STEP;
    }
    return n;
}

void search(gn_index *ix, const uint8_t *qbases_dev, const std::vector<uint64_t> &qstart_h, const SearchOptions &o,
            cudaStream_t s, gn_results *res) {
    const uint32_t nq = (uint32_t)(qstart_h.size() - 1);
    const uint64_t M = qstart_h[nq];
    const int k = ix->span;  // HSPs end k bases after their last seed (the seed's span)
    const gn_params &p = o.p;
    const gn_scoring &sc = o.sc;
    const bool keep = (p.flags & GN_FLAG_KEEP_STAGES) != 0;
    const bool keep_hits = (p.flags & GN_FLAG_KEEP_HITS) != 0;
    res->n_queries = nq;
    res->has_stages = keep;
    PhaseTimer timer(s, ix->host_pool);
    timer.mark("start");
    KernelTimer ktimer;
    struct TimerScope {
        KernelTimer *prev;
        explicit TimerScope(KernelTimer *t) : prev(g_ktimer) { g_ktimer = t; }
        ~TimerScope() { g_ktimer = prev; }
    };
    TimerScope tscope((p.flags & GN_FLAG_TIME_KERNELS) ? &ktimer : nullptr);
    DeviceArena arena(s);
    // What the host reads back while a search runs, and the counters its kernels work with, in one
    // place that one memset clears: the words of SearchWords, the alignment order's bins, then the
    // hits per query (or segment).
    const uint64_t n_seg_max = count_segments(qstart_h);
    GN_REQUIRE(n_seg_max <= MAX_QUERIES, GN_ETOOBIG, "more than 65,536 query segments in one call");
    const size_t words_bytes = sizeof(SearchWords) + 8 * (n_seg_max + 1);
    SearchWords *words = static_cast<SearchWords *>(arena.alloc(words_bytes));
    GN_CUDA(cudaMemsetAsync(words, 0, words_bytes, s));
    uint64_t *hq_d = reinterpret_cast<uint64_t *>(words + 1);
    uint32_t *wait_status = &words->wait_status, *status = &words->status;
    WaitStatusScope wscope(wait_status);  // bounded device-side waits (the scans' look-back) record a timeout there
    PinnedBlock pin(ix->host_pool, std::max<size_t>(words_bytes, 1 << 16), s);
#ifdef GN_CHECKS
    uint32_t *check_bits = nullptr;  // the failed device-side checks of this search
    GN_CUDA(cudaGetSymbolAddress(reinterpret_cast<void **>(&check_bits), g_check_bits));
    GN_CUDA(cudaMemsetAsync(check_bits, 0, 4, s));
#endif

    // a5: pack queries, code every offset, list lengths
    Packed qp;
    qp.pk = arena.alloc_n<uint32_t>(Packed::pk_words(M));
    qp.nb = arena.alloc_n<uint32_t>(Packed::nb_words(M));
    pack_bases(qbases_dev, M, qp, s);
    uint64_t *qstart_d = arena.alloc_n<uint64_t>(nq + 1);
    GN_CUDA(cudaMemcpyAsync(qstart_d, qstart_h.data(), sizeof(uint64_t) * (nq + 1), cudaMemcpyHostToDevice, s));

    // The seed phases (a5-a8) run on the queries themselves, or, when a query is longer
    // than MAX_QUERY_LEN, on segments: every query of at most MAX_QUERY_LEN bases is one
    // segment, a longer one is cut into segments of MAX_QUERY_LEN bases SEG_STEP apart
    // (neighbours share SEG_OVERLAP bases; the last one ends with the query).  Every
    // chain of hits at most D offsets apart then has each pair of consecutive hits inside
    // one segment (D + span <= SEG_OVERLAP), so the chain is the union of its pieces in
    // the segments, and pieces of one chain share a hit.  The pieces are emitted whatever
    // their length, mapped back onto the query and joined after a8 (k_stitch_sweep),
    // which then applies min_hsp_len.
    std::vector<uint64_t> seg_start{0}, seg_off;  // per segment: start in the segment batch, offset in its query
    std::vector<uint32_t> seg_parent;
    bool segmented = false;
    uint64_t max_qlen = 0;
    for (uint32_t i = 0; i < nq; ++i) {
        const uint64_t m = qstart_h[i + 1] - qstart_h[i];
        max_qlen = std::max(max_qlen, m);
        for (uint64_t o = 0;; o += SEG_STEP) {
            const uint64_t len = std::min<uint64_t>(MAX_QUERY_LEN, m - o);
            seg_parent.push_back(i);
            seg_off.push_back(o);
            seg_start.push_back(seg_start.back() + len);
            if (o + MAX_QUERY_LEN >= m) break;
            segmented = true;
        }
    }
    if (segmented) {
        GN_REQUIRE(p.max_hit_distance + (uint32_t)k <= SEG_OVERLAP, GN_EINVAL,
                   "queries over 65,535 bases need max_hit_distance + seed span <= 8,192");
        GN_REQUIRE(!(p.flags & (GN_FLAG_KEEP_STAGES | GN_FLAG_KEEP_HITS)), GN_EINVAL,
                   "stage outputs are not kept for queries over 65,535 bases");
        GN_REQUIRE(ix->max_seq_len < (1ull << 32) - (1ull << 24), GN_ETOOBIG,
                   "queries over 65,535 bases need bank sequences shorter than 2^32 - 2^24 bases");
    }
    const uint32_t hnq = segmented ? (uint32_t)seg_parent.size() : nq;
    const std::vector<uint64_t> &hstart_h = segmented ? seg_start : qstart_h;
    const uint64_t HM = hstart_h[hnq];
    const uint32_t hit_min_len = segmented ? 1u : p.min_hsp_len;
    Packed hqp = qp;
    uint64_t *hstart_d = qstart_d;
    uint32_t *seg_parent_d = nullptr;
    uint64_t *seg_off_d = nullptr;
    if (segmented) {
        hstart_d = arena.alloc_n<uint64_t>(hnq + 1);
        seg_off_d = arena.alloc_n<uint64_t>(hnq);
        seg_parent_d = arena.alloc_n<uint32_t>(hnq);
        GN_CUDA(cudaMemcpyAsync(hstart_d, seg_start.data(), sizeof(uint64_t) * (hnq + 1), cudaMemcpyHostToDevice, s));
        GN_CUDA(cudaMemcpyAsync(seg_off_d, seg_off.data(), sizeof(uint64_t) * hnq, cudaMemcpyHostToDevice, s));
        GN_CUDA(cudaMemcpyAsync(seg_parent_d, seg_parent.data(), sizeof(uint32_t) * hnq, cudaMemcpyHostToDevice, s));
        uint8_t *sb = arena.alloc_n<uint8_t>(HM);
        GN_LAUNCH("k_segment_bases", HM, s,
                  k_segment_bases<<<hnq, 256, 0, s>>>(qbases_dev, qstart_d, seg_parent_d, seg_off_d, hstart_d, sb));
        hqp.pk = arena.alloc_n<uint32_t>(Packed::pk_words(HM));
        hqp.nb = arena.alloc_n<uint32_t>(Packed::nb_words(HM));
        pack_bases(sb, HM, hqp, s);
    }
    const int singles = p.min_hsp_len <= (uint32_t)k ? 1 : 0;
    const SigKind kind = sig_kind(ix->k, ix->span, ix->t);
    const uint32_t links = p.max_hit_distance / (uint32_t)ix->t;  // windows from one hit to the next, at most
    const bool scan = takes_scan(ix, p);
    uint32_t *codes = scan ? nullptr : arena.alloc_n<uint32_t>(HM);
    uint32_t *qinfo = arena.alloc_n<uint32_t>(HM);
    uint32_t *cnt = arena.alloc_n<uint32_t>(HM);  // list lengths; scan route: list units
    uint64_t *hoff = arena.alloc_n<uint64_t>(HM + 1);
    uint32_t *src = scan ? nullptr : arena.alloc_n<uint32_t>(HM);
    QueryRec *qrec = scan ? arena.alloc_n<QueryRec>(HM) : nullptr;
    const int flank = (int)std::min<uint32_t>(SIG_FLANK_BASES, p.min_hsp_len > (uint32_t)k ? p.min_hsp_len - (uint32_t)k : 0u);
    const bool recs_sum = scan && HM && HM <= RECS_SUMS;
    if (scan) {
        auto kernel = kind == SIG_FLANK ? k_query_recs<SIG_FLANK> : k_query_recs<SIG_AHEAD>;
        if (HM)
            GN_LAUNCH("k_query_recs", HM, s,
                      kernel<<<blocks_for(HM), 256, 0, s>>>(hstart_d, hnq, HM, hqp.pk, hqp.nb, seed_shape(ix), ix->t,
                                                            (int)links, flank, ix->off_d, qinfo, qrec, cnt,
                                                            reinterpret_cast<unsigned long long *>(hq_d),
                                                            recs_sum ? hoff : nullptr, &words->recs_done));
    } else if (HM) {
        GN_LAUNCH("k_query_codes", HM, s,
                  k_query_codes<<<blocks_for(HM), 256, 0, s>>>(hstart_d, hnq, HM, hqp.pk, hqp.nb, seed_shape(ix), ix->off_d, codes, qinfo,
                                                              cnt, src));
    }
    if (!recs_sum) {
        void *scr = arena.alloc(scan_scratch_bytes(HM));
        exclusive_scan_u32(cnt, hoff, HM, scr, s);
    }
    // per-query hit counts (limits; the chunk plan of the hit-storing paths), as prefix sums
    if (!scan)
        GN_LAUNCH("k_gather_u64", hnq + 1, s,
                  k_gather_u64<<<blocks_for(hnq + 1), 256, 0, s>>>(hoff, hstart_d, hnq + 1, hq_d));
    // hits per query as prefix sums; the scan route reads them with its HSP count
    std::vector<uint64_t> hq;
    auto read_hits = [&](const uint64_t *from) {
        hq.assign(from, from + hnq + 1);
        if (scan) {
            uint64_t at = 0;
            for (uint32_t i = 0; i <= hnq; ++i) {
                const uint64_t h = hq[i];
                GN_REQUIRE(i == hnq || h < (1ull << 32), GN_ETOOBIG, "a query has 2^32 seed hits or more");
                hq[i] = at;
                at += h;
            }
        }
        GN_REQUIRE(!o.max_hit_bytes || hq[hnq] * HIT_BYTES <= o.max_hit_bytes, GN_ETOOBIG,
                   "the query alone exceeds the server's memory budget");
    };
    if (!scan || g_ktimer) {
        pin.fetch(0, hq_d, 8 * (hnq + 1));
        pin.wait();
        read_hits(reinterpret_cast<const uint64_t *>(pin.p));
    }
    timer.mark("query_codes");

    // a6-a8 per chunk of queries whose hits fit the budget
    uint64_t hit_budget = 0, scan_range = SCAN_RANGE;
    auto free_bytes = []() {
        size_t free_b = 0, total_b = 0;
        GN_CUDA(cudaMemGetInfo(&free_b, &total_b));
        return free_b;
    };
    if (!scan) {
        // bytes per hit of a chunk: hit keys and their ping-pong buffer on the sort path, or the
        // fixed-capacity buckets (up to ~22 B per hit without the repeat filter) and spill lists
        uint64_t mem_for_hits = (uint64_t)(free_bytes() * 0.55);
        if (o.mem_cap) mem_for_hits = std::min(mem_for_hits, o.mem_cap);
        // (a query chunk holds < 2^32 hits: the fill kernel indexes a tile's hits in 32 bits)
        hit_budget = std::min<uint64_t>(0xFFFFFFFFull, std::max<uint64_t>(1ull << 20, mem_for_hits / HIT_BYTES));
    }
    if (const char *e = getenv("GN_MAX_CHUNK_HITS")) {  // smaller chunks, or ranges of the scan (exercises several of them)
        uint64_t v = strtoull(e, nullptr, 10);
        if (v) {
            hit_budget = std::min<uint64_t>(v, 0xFFFFFFFFull);
            scan_range = std::min(std::max<uint64_t>(v / 4, 1), SCAN_RANGE);
        }
    }
    const uint64_t gbits_max = (uint64_t)bits_for(ix->n_bases + QBIAS);
    const uint32_t max_chunk_q = (uint32_t)std::min<uint64_t>(MAX_QUERIES, 1ull << std::min<uint64_t>(48 - gbits_max, 31));

    // The scan route sizes its lists from the hits that the list lengths' mean promises (repeats
    // and skewed bases bring more): lists that turn out short are enlarged and their kernel rerun.
    const uint64_t hits_guess = scan ? (uint64_t)std::min((double)HM * (double)ix->n_postings / std::pow(4.0, ix->k), (double)CAND_MAX) : hq[hnq];
    uint32_t hsp_cap = (uint32_t)std::min<uint64_t>(0xFFFFFFFFull, std::max<uint64_t>(1u << 14, hits_guess / 64));
    DevHsp *hsp = arena.alloc_n<DevHsp>(hsp_cap);
    uint32_t n_hsp = 0;
    uint32_t *counter = &words->n_hsp;
    std::vector<uint32_t> hits_q;

    // appends HSPs through `launch(out, room)`, growing the HSP buffer and relaunching on overflow
    auto emit = [&](auto launch) {
        for (int attempt = 0; attempt < 3; ++attempt) {
            GN_CUDA(cudaMemsetAsync(counter, 0, 4, s));
            launch(hsp + n_hsp, hsp_cap - n_hsp);
            uint32_t got = 0;
            GN_CUDA(cudaMemcpyAsync(&got, counter, 4, cudaMemcpyDeviceToHost, s));
            GN_CUDA(cudaStreamSynchronize(s));
            if (n_hsp + (uint64_t)got <= hsp_cap) {
                n_hsp += got;
                return;
            }
            uint64_t need = (uint64_t)n_hsp + got;
            GN_REQUIRE(need < (1ull << 32), GN_ETOOBIG, "more than 2^32 HSPs in one call");
            uint32_t ncap = (uint32_t)std::min<uint64_t>(0xFFFFFFFFull,
                                                         std::max<uint64_t>(need + need / 4, 2ull * hsp_cap));
            DevHsp *nh = arena.alloc_n<DevHsp>(ncap);
            if (n_hsp) GN_CUDA(cudaMemcpyAsync(nh, hsp, sizeof(DevHsp) * n_hsp, cudaMemcpyDeviceToDevice, s));
            hsp = nh;
            hsp_cap = ncap;
            GN_CUDA(cudaMemsetAsync(status, 0, 4, s));
        }
        throw Error{GN_EINTERNAL, "HSP buffer growth did not converge"};
    };
    if (scan && HM) {
        auto kernel = kind == SIG_FLANK ? k_seed_scan<SIG_FLANK> : k_seed_scan<SIG_AHEAD>;
        const bool edges = !(ix->keep & 1u) || !(ix->keep >> (ix->span - 1));
        auto chain = kind == SIG_FLANK ? k_chain<SIG_FLANK, false> : edges ? k_chain<SIG_AHEAD, true> : k_chain<SIG_AHEAD, false>;
        const int occ = blocks_per_sm(reinterpret_cast<const void *>(kernel), SCAN_THREADS);
        const int cocc = blocks_per_sm(reinterpret_cast<const void *>(chain), SCAN_THREADS);
        // resident blocks; fewer when the units (four hits each, at least one an offset) do not fill them
        const uint64_t tiles = (hits_guess / 4 + 2 * HM) / 64 + 1;
        const unsigned grid = (unsigned)std::max<uint64_t>(
            1, std::min<uint64_t>((tiles + SCAN_THREADS / 32 - 1) / (SCAN_THREADS / 32), (uint64_t)num_sms() * occ));
        // The scan takes all units in one launch, or ranges of them, each scanned, checked and its HSPs
        // appended before the next: SCAN_RANGE units at a time, or as many as leave a list of
        // candidates that memory has room for (55 % of what is free, and no more than the caller grants).
        // A range costs a host wait and the ends of two kernels: 8.7 G hits at stride 1 took 7.60 ms in
        // five and 7.39 in one.  Room for candidates to begin with: about 1 % of the hits at stride 11 are.
        DeviceArena lists(s);  // enlarged candidate lists
        auto list_room = [&](uint64_t bytes) {  // candidates that `bytes` hold, within what the caller grants
            if (o.mem_cap) bytes = std::min(bytes, o.mem_cap);
            uint64_t room = std::max<uint64_t>(1u << 20, bytes / sizeof(uint2));
            if (const char *e = getenv("GN_CAND_ROOM")) room = std::max<uint64_t>(4, strtoull(e, nullptr, 10));  // (a unit's)
            return std::min(room, CAND_MAX);
        };
        uint64_t cand_cap = std::min(std::max<uint64_t>(1u << 14, hits_guess / 24), list_room(~0ull));
        uint2 *cand = arena.alloc_n<uint2>(cand_cap);
        uint64_t units = g_ktimer ? hq[hnq] : 0;
        const uint64_t max_range = scan_range;
        bool scanned = false;  // the range's candidates are listed
        int attempt = 0;       // of the range
        for (uint64_t done = 0, all = 1; done < all; ++attempt) {
            if (done || attempt)  // n_hsp and next_cand; n_cand and next_tile too if the scan runs again
                GN_CUDA(cudaMemsetAsync(&words->n_hsp, 0, scanned ? 8 : 20, s));
            if (!scanned)
                GN_LAUNCH("k_seed_scan", units, s,
                          kernel<<<grid, SCAN_THREADS, 0, s>>>(qrec, hoff, HM, done, done + scan_range, &words->n_units,
                                                               reinterpret_cast<const uint4 *>(ix->sig_d),
                                                               post_alloc_entries(ix->n_postings) / 4, flank, cand,
                                                               &words->n_cand, (uint32_t)cand_cap, &words->next_tile));
            const ScanCtx c{qinfo, hstart_d, ix->post_d, ix->bank.pk, ix->bank.nb, hqp.pk, hqp.nb, seed_shape(ix),
                            ix->t, (int)links, flank, hit_min_len, seq_map(ix), hsp + n_hsp, counter, hsp_cap - n_hsp, status,
                            ix->n_postings, ix->n_bases, HM};
            GN_LAUNCH("k_chain", units, s,
                      chain<<<(unsigned)std::min<uint64_t>((cand_cap + SCAN_THREADS - 1) / SCAN_THREADS, (uint64_t)num_sms() * cocc),
                              SCAN_THREADS, 0, s>>>(c, cand, &words->n_cand, (uint32_t)cand_cap, &words->next_cand));
            units = 0;  // of the first launch
            pin.fetch(0, words, words_bytes);
            pin.wait();
            const SearchWords *got = reinterpret_cast<const SearchWords *>(pin.p);
            if (hq.empty()) read_hits(reinterpret_cast<const uint64_t *>(pin.p + sizeof(SearchWords)));
            all = got->n_units;
            const uint64_t n_cand = got->n_cand, n_new = got->n_hsp;
            const uint64_t here = std::min(scan_range, all - done);
            scanned = n_cand <= cand_cap;
            if (scanned && n_hsp + n_new <= hsp_cap) {
                n_hsp += (uint32_t)n_new;
                done += here;
                if (n_cand < cand_cap / 4) scan_range = std::min(2 * scan_range, max_range);
                scanned = false;
                attempt = -1;
                continue;
            }
            GN_REQUIRE(attempt < 64, GN_EINTERNAL, "candidate and HSP list sizing did not converge");
            if (!scanned) {
                const uint64_t want = done + here < all ? n_cand + n_cand / 4 : n_cand,
                               room = list_room(want > CAND_ASK ? (uint64_t)(0.55 * free_bytes()) : ~0ull);
                if (n_cand > room) {  // fewer units, as their candidates go; a quarter of the list's length always fits it
                    cand_cap = std::max(cand_cap, room);
                    scan_range = std::max<uint64_t>({1, cand_cap / 4, (uint64_t)(0.75 * (double)here * (double)cand_cap / (double)n_cand)});
                } else {
                    cand_cap = std::min(want, room);
                }
                lists.release();
                cand = lists.alloc_n<uint2>(cand_cap);
            } else {
                const uint64_t need = n_hsp + n_new;
                GN_REQUIRE(need < (1ull << 32), GN_ETOOBIG, "more than 2^32 HSPs in one call");
                hsp_cap = (uint32_t)std::min<uint64_t>(0xFFFFFFFFull, need + need / 4);
                DevHsp *nh = arena.alloc_n<DevHsp>(hsp_cap);
                if (n_hsp) GN_CUDA(cudaMemcpyAsync(nh, hsp, sizeof(DevHsp) * n_hsp, cudaMemcpyDeviceToDevice, s));
                hsp = nh;
            }
            GN_CUDA(cudaMemsetAsync(status, 0, 4, s));
        }
        timer.mark("seed_scan");
    }
    if (hq.empty()) hq.assign(hnq + 1, 0);  // no offsets at all
    if (keep) {
        res->st_hit_counts.resize(hnq);
        for (uint32_t i = 0; i < hnq; ++i) res->st_hit_counts[i] = hq[i + 1] - hq[i];
    }

    uint32_t qa = scan ? hnq : 0;
    while (qa < hnq) {
        uint32_t qb = qa + 1;
        while (qb < hnq && qb - qa < max_chunk_q && hq[qb + 1] - hq[qa] <= hit_budget) ++qb;
        const uint64_t xa = hstart_h[qa], xb = hstart_h[qb];
        const uint64_t ha = hq[qa], Hc = hq[qb] - hq[qa];
        GN_REQUIRE(Hc < (1ull << 32), GN_ETOOBIG, "a query has 2^32 seed hits or more");
        if (Hc > 0) {
            const int qbits = bits_for(qb - qa - 1);
            const int gbits = (int)gbits_max;
            const uint32_t nqc = qb - qa;
            DeviceArena carena(s);
            // global path: gather every hit, LSD radix sort by diagonal key, merge sorted runs
            auto sort_path = [&](uint64_t *keys, uint64_t *keys_alt, uint64_t n, int lo_bit, const RadixTag &tag) {
                void *rs = carena.alloc(radix_scratch_bytes(n));
                bool fl = radix_sort(keys, keys_alt, nullptr, nullptr, n, lo_bit, 16 + qbits + gbits, rs, s, tag);
                uint64_t *sorted = fl ? keys_alt : keys;
                timer.mark("hit_sort");
                emit([&](DevHsp *o, uint32_t room) {
                    uint64_t threads = std::min<uint64_t>(n, (uint64_t)num_sms() * 2048);
                    GN_LAUNCH("k_hit_merge", n, s,
                              k_hit_merge<<<blocks_for(threads), 256, 0, s>>>(sorted, n, qbits, qa, k,
                                                                             p.max_hit_distance, hit_min_len,
                                                                             seq_map(ix), o, counter, room, status));
                });
                return sorted;
            };
            const char *grouping = getenv("GN_HIT_GROUPING");
            const bool bucketed = !keep_hits && !(grouping && strcmp(grouping, "sort") == 0);
            if (!bucketed) {
                uint64_t *keys = carena.alloc_n<uint64_t>(Hc);
                uint64_t *keys_alt = carena.alloc_n<uint64_t>(Hc);
                uint64_t gwarps = std::min<uint64_t>((xb - xa + 31) / 32, (uint64_t)num_sms() * 64);
                GN_LAUNCH("k_seed_gather", Hc, s,
                          k_seed_gather<<<blocks_for(gwarps * 32), 256, 0, s>>>(codes, qinfo, hoff, xa, xb, ha,
                                                                               ix->off_d, ix->post_d, qa, qbits,
                                                                               keys));
                timer.mark("seed_gather");
                uint64_t *sorted = sort_path(keys, keys_alt, Hc, 16 + qbits, TAG_HIT_SORT);
                if (keep_hits) {
                    uint32_t *quad = carena.alloc_n<uint32_t>(4 * Hc);
                    GN_LAUNCH("k_decode_hits", Hc, s,
                              k_decode_hits<<<blocks_for(Hc), 256, 0, s>>>(sorted, Hc, qbits, qa, ix->seq_start_d,
                                                                           ix->n_seqs, quad));
                    std::vector<uint32_t> hh = to_host(quad, 4 * Hc, s);
                    hits_q.insert(hits_q.end(), hh.begin(), hh.end());
                }
            } else {
                // bucket plan: 2^lg buckets per query, about `target` raw hits each
                const char *fenv = getenv("GN_TILE_FILTER");
                const int filter = (!singles && p.max_hit_distance <= (uint32_t)BT_MAX_D &&
                                    !(fenv && strcmp(fenv, "0") == 0)) ? 1 : 0;
                // 512-thread tiles of about 50,000 hits: 512 offsets at ~88 hits per offset (stride 11 on
                // a 4 Gbp bank), fewer where lists are long (small strides), up to 1,024 where they are
                // short; 2^19-bit "seen" and 2^17-bit "seen twice" bitmaps (two tiles per SM)
                const double per_offset = (double)Hc / (double)std::max<uint64_t>(1, xb - xa);
                const double tile_hits = ix->tuning.tile_hits ? (double)ix->tuning.tile_hits : 50000.0;
                int tpos = 32;
                while (tpos < 1024 && tpos * 2 * per_offset <= tile_hits * 1.5) tpos *= 2;
                // a small search (one query, a few) gets smaller tiles, so that its hits are spread
                // over the SMs instead of filling one or two tiles one after the other
                while (tpos > 32 && (xb - xa + tpos - 1) / tpos < 4ull * (uint64_t)num_sms()) tpos /= 2;
                int fthreads = ix->tuning.fill_threads == 256 ? 256 : 512;
                if (const char *e = getenv("GN_FILL_THREADS")) fthreads = atoi(e) >= 512 ? 512 : 256;
                // two 512-thread tiles or four 256-thread tiles per SM
                int fbits = fthreads == 512 ? 19 : 18, fbits2 = fthreads == 512 ? 17 : 16;
                if (const char *e = getenv("GN_TILE_POS")) tpos = std::max(32, std::min(4096, atoi(e)));
                if (const char *e = getenv("GN_TILE_FBITS")) fbits = std::max(12, std::min(19, atoi(e)));
                if (const char *e = getenv("GN_TILE_FBITS2")) fbits2 = std::max(12, std::min(19, atoi(e)));
                // the filter keeps about 2 % of the hits: buckets of about 4,096 raw hits hold about 80 kept
                // hits, most of them within the grouping warps' 256 candidates; capacity 1,024
                uint32_t target = filter ? (ix->tuning.bucket_target ? ix->tuning.bucket_target : 4096) : 512, bcap = 1024;
                if (const char *e = getenv("GN_BUCKET_TARGET")) target = std::max(64, std::min(65536, atoi(e)));
                if (const char *e = getenv("GN_BUCKET_CAP")) {  // small buckets (exercises the spill path)
                    bcap = (uint32_t)std::max(8ul, std::min(65536ul, strtoul(e, nullptr, 10)));
                    target = std::max<uint32_t>(2, bcap / 2);
                }
                const bool fixed_cap = getenv("GN_BUCKET_CAP") != nullptr;
                std::vector<uint32_t> bbase(nqc + 1), bshift(nqc);
                const int min_lg = std::max(0, gbits - 31);
                uint32_t NB = 0;
                uint32_t *d_bbase = carena.alloc_n<uint32_t>(nqc + 1);
                uint32_t *d_bshift = carena.alloc_n<uint32_t>(nqc);
                uint32_t *bcount = nullptr;
                uint64_t *bkeys = nullptr;
                uint16_t *bq = nullptr;
                // 2^lg buckets per query, about `target` raw hits each
                auto plan = [&](uint64_t target) {
                    uint64_t nb64 = 0;
                    for (uint32_t i = 0; i < nqc; ++i) {
                        const uint64_t hi = hq[qa + i + 1] - hq[qa + i];
                        const uint64_t want = (hi + target - 1) / target;
                        int lg = 0;
                        while ((1ull << lg) < want) ++lg;
                        lg = std::min(std::max(lg, min_lg), gbits);
                        bshift[i] = (uint32_t)(gbits - lg);
                        bbase[i] = (uint32_t)nb64;
                        nb64 += 1ull << lg;
                        GN_REQUIRE(nb64 < (1ull << 32), GN_ETOOBIG, "too many hit buckets in one chunk");
                    }
                    bbase[nqc] = (uint32_t)nb64;
                    NB = (uint32_t)nb64;
                    GN_CUDA(cudaMemcpyAsync(d_bbase, bbase.data(), 4 * (nqc + 1), cudaMemcpyHostToDevice, s));
                    GN_CUDA(cudaMemcpyAsync(d_bshift, bshift.data(), 4 * nqc, cudaMemcpyHostToDevice, s));
                };
                auto alloc_buckets = [&]() {
                    bcount = carena.alloc_n<uint32_t>(NB);
                    bkeys = carena.alloc_n<uint64_t>((uint64_t)NB * bcap);
                    bq = carena.alloc_n<uint16_t>(NB);
                };
                plan(target);
                unsigned long long *spill_count = reinterpret_cast<unsigned long long *>(carena.alloc_n<uint64_t>(1));
                uint64_t spill_room = std::max<uint64_t>(1u << 16, Hc / 32);
                uint64_t min_room = 0;  // GN_SPILL_ROOM: small first rooms (exercises the reruns)
                if (const char *e = getenv("GN_SPILL_ROOM")) min_room = std::max<uint64_t>(1, strtoull(e, nullptr, 10));
                if (min_room) spill_room = min_room;
                uint64_t *spill = carena.alloc_n<uint64_t>(spill_room);
                const uint64_t tiles = (xb - xa + tpos - 1) / tpos;
                // the kept-hit stage gets what the SM's shared memory leaves for two 512-thread (or four
                // 256-thread) tiles per SM after the filters and the table, at least 256 hits
                uint32_t stage_cap = 256;
                {
                    const uint32_t halo = filter ? p.max_hit_distance : 0u;
                    int per_sm = 0, reserved = 0;
                    GN_CUDA(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, ix->device));
                    GN_CUDA(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, ix->device));
                    const int64_t room = (int64_t)per_sm / (fthreads == 512 ? 2 : 4) - reserved - 512 -
                                         (int64_t)bucket_fill_smem(tpos, halo, filter, fbits, fbits2, 0);
                    if (room > 256 * BF_STAGE_BYTES)
                        stage_cap = (uint32_t)std::min<int64_t>(8192, room / BF_STAGE_BYTES) & ~31u;
                }
                const size_t bf_smem = bucket_fill_smem(tpos, filter ? p.max_hit_distance : 0u, filter, fbits, fbits2,
                                                        stage_cap);
                auto fill_kernel = (fbits == 19 && fbits2 == 17) ? k_bucket_fill<19, 17> : k_bucket_fill<0, 0>;
                allow_max_smem(ix->device);
                int focc = 0;
                GN_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&focc, fill_kernel, fthreads, bf_smem));
                const unsigned fgrid = (unsigned)std::max<uint64_t>(
                    1, std::min<uint64_t>(tiles, (uint64_t)num_sms() * std::max(focc, 1) * 4));
                unsigned long long n_spill = 0, n_kept = 0;
                // kept hits, core hits (sampling), tile counter
                unsigned long long *kept_total = reinterpret_cast<unsigned long long *>(carena.alloc_n<uint64_t>(3));
                // Keep rate of the repeat filter, measured on a sample of tiles (no placement): the plan
                // above assumes the stride-11 rate; where far more hits are kept (small strides, where
                // overlapping k-mers put most hits next to another on their diagonal) the buckets are
                // planned smaller.
                // With a keep rate above a quarter, 256-entry buckets of about 128 kept hits are planned:
                // the grouping warps take every such bucket whole.
                auto plan_for_keep = [&](double keep, uint32_t &t_new, uint32_t &cap_new) {
                    if (keep > 0.25) {
                        cap_new = 256;
                        t_new = (uint32_t)std::max(64.0, 128.0 / keep);
                    } else {
                        cap_new = bcap;
                        t_new = (uint32_t)std::max(64.0, std::min((double)target, bcap / 2.0 / keep));
                    }
                };
                if (filter && !fixed_cap && !getenv("GN_BUCKET_TARGET") && ix->t < 8) {
                    const uint32_t tile_step = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(256, tiles / 256));
                    const uint64_t stiles = (tiles + tile_step - 1) / tile_step;
                    unsigned long long got[2] = {0, 0};
                    GN_CUDA(cudaMemsetAsync(kept_total, 0, 24, s));
                    GN_LAUNCH("k_bucket_fill_sample", Hc / tile_step, s,
                              fill_kernel<<<(unsigned)std::max<uint64_t>(1, std::min<uint64_t>(stiles, fgrid)), fthreads,
                                            bf_smem, s>>>(
                                  qinfo, src, hoff, xa, xb, ix->post_d, qa, d_bbase, d_bshift, nullptr, nullptr, bcap,
                                  nullptr, nullptr, 0ull, qbits, filter, p.max_hit_distance, tpos, fbits, fbits2,
                                  kept_total, tile_step, 1, stage_cap, NB, post_alloc_entries(ix->n_postings) / 4));
                    GN_CUDA(cudaMemcpyAsync(got, kept_total, 16, cudaMemcpyDeviceToHost, s));
                    GN_CUDA(cudaStreamSynchronize(s));
                    if (got[1]) {
                        uint32_t t_new = target, cap_new = bcap;
                        plan_for_keep(std::max(1e-6, (double)got[0] / (double)got[1]), t_new, cap_new);
                        if (t_new != target || cap_new != bcap) {
                            target = t_new;
                            bcap = cap_new;
                            plan(target);
                        }
                    }
                }
                alloc_buckets();
                // Which of two colliding keys the filter keeps depends on arrival order, so the spill
                // count varies a little between runs: a rerun gets room with a margin, and the loop
                // ends on the run whose spills all fit.
                auto run_fill = [&]() {
                    for (int attempt = 0;; ++attempt) {
                        GN_CUDA(cudaMemsetAsync(bcount, 0, 4ull * NB, s));
                        GN_CUDA(cudaMemsetAsync(spill_count, 0, 8, s));
                        GN_CUDA(cudaMemsetAsync(kept_total, 0, 24, s));
                        GN_LAUNCH("k_bucket_fill", Hc, s,
                                  fill_kernel<<<fgrid, fthreads, bf_smem, s>>>(
                                      qinfo, src, hoff, xa, xb, ix->post_d, qa, d_bbase, d_bshift, bcount, bkeys, bcap,
                                      spill, spill_count, (unsigned long long)spill_room, qbits, filter,
                                      p.max_hit_distance, tpos, fbits, fbits2, kept_total, 1u, 0, stage_cap, NB,
                                      post_alloc_entries(ix->n_postings) / 4));
                        GN_CUDA(cudaMemcpyAsync(&n_spill, spill_count, 8, cudaMemcpyDeviceToHost, s));
                        GN_CUDA(cudaMemcpyAsync(&n_kept, kept_total, 8, cudaMemcpyDeviceToHost, s));
                        GN_CUDA(cudaStreamSynchronize(s));
                        if (n_spill <= spill_room) break;
                        GN_REQUIRE(attempt < 3, GN_EINTERNAL, "hit-bucket spill sizing did not converge");
                        spill_room = n_spill + n_spill / 8 + 1024;
                        spill = carena.alloc_n<uint64_t>(spill_room);
                    }
                };
                run_fill();
                // The plan assumes the stride-11 keep rate of the repeat filter.  Where far more hits
                // are kept (small strides: overlapping k-mers put most hits next to another on their
                // diagonal) the buckets overflow; plan again from the measured keep rate, once.
                if (!fixed_cap && n_kept && n_spill > std::max<unsigned long long>(1u << 16, n_kept / 32)) {
                    uint32_t t_new = target, cap_new = bcap;
                    plan_for_keep((double)n_kept / (double)Hc, t_new, cap_new);
                    if (t_new * 4 < target * 3 || cap_new != bcap) {
                        target = t_new;
                        bcap = cap_new;
                        plan(target);
                        alloc_buckets();
                        run_fill();
                    }
                }
                GN_LAUNCH("k_bucket_query", NB, s, k_bucket_query<<<nqc, 256, 0, s>>>(d_bbase, nqc, NB, bq));
                timer.mark("bucket_fill");
                // group each bucket; buckets with too many candidates are appended to the spill list too
                const size_t smem = (size_t)BGW_WARPS * (2 * BGW_BITS / 8 + BGW_CAND * 8 + BGW_CAND / 8);

                int occ = 0;
                GN_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bucket_group_warp, BGW_WARPS * 32, smem));
                const unsigned ggrid = (unsigned)std::max<uint64_t>(
                    1, std::min<uint64_t>((NB + BGW_WARPS - 1) / BGW_WARPS, (uint64_t)num_sms() * std::max(occ, 1)));
                const uint64_t spilled_fill = n_spill;
                uint64_t group_room = min_room ? min_room : std::max<uint64_t>(1u << 16, Hc / 16);
                uint64_t *gsp = carena.alloc_n<uint64_t>(spilled_fill + group_room);
                if (spilled_fill)
                    GN_CUDA(cudaMemcpyAsync(gsp, spill, 8 * spilled_fill, cudaMemcpyDeviceToDevice, s));
                unsigned long long n_ovf = 0;
                unsigned long long *ovf_count = spill_count;
                uint32_t *big = carena.alloc_n<uint32_t>(NB);  // buckets for the block-level grouping
                uint32_t *big_count = carena.alloc_n<uint32_t>(1), *next_bucket = carena.alloc_n<uint32_t>(1);
                uint32_t n_big = 0;
                for (int attempt = 0;; ++attempt) {
                    const uint32_t hsp_before = n_hsp;
                    emit([&](DevHsp *o, uint32_t room) {
                        GN_CUDA(cudaMemsetAsync(ovf_count, 0, 8, s));
                        GN_CUDA(cudaMemsetAsync(next_bucket, 0, 4, s));
                        GN_CUDA(cudaMemsetAsync(big_count, 0, 4, s));
                        GN_LAUNCH("k_bucket_group", n_kept, s,
                                  k_bucket_group_warp<<<ggrid, BGW_WARPS * 32, smem, s>>>(
                                      bkeys, bcount, bcap, NB, bq, qa, qbits, k, p.max_hit_distance, hit_min_len,
                                      singles, seq_map(ix), o, counter, room, gsp + spilled_fill,
                                      (unsigned long long)group_room, ovf_count, status, next_bucket, big,
                                      big_count));
                        // read back with the HSP count, in emit's one synchronisation
                        GN_CUDA(cudaMemcpyAsync(&n_ovf, ovf_count, 8, cudaMemcpyDeviceToHost, s));
                        GN_CUDA(cudaMemcpyAsync(&n_big, big_count, 4, cudaMemcpyDeviceToHost, s));
                    });
                    if (n_ovf <= group_room) break;
                    GN_REQUIRE(attempt < 3, GN_EINTERNAL, "hit-bucket overflow sizing did not converge");
                    n_hsp = hsp_before;  // the rerun emits this chunk's bucket HSPs again
                    group_room = n_ovf + n_ovf / 8 + 1024;
                    uint64_t *ng = carena.alloc_n<uint64_t>(spilled_fill + group_room);
                    if (spilled_fill)
                        GN_CUDA(cudaMemcpyAsync(ng, spill, 8 * spilled_fill, cudaMemcpyDeviceToDevice, s));
                    gsp = ng;
                    GN_CUDA(cudaMemsetAsync(status, 0, 4, s));
                }
                // buckets with more candidates than a warp holds: a block each
                int bocc = 0;
                if (n_big)
                    GN_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bocc, k_bucket_group_block, 256, 0));
                const unsigned bgrid =
                    (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(n_big, (uint64_t)num_sms() * std::max(bocc, 1)));
                if (n_big) emit([&](DevHsp *o, uint32_t room) {
                    GN_LAUNCH("k_bucket_group_block", n_big, s,
                              k_bucket_group_block<<<bgrid, 256, 0, s>>>(
                                  bkeys, bcount, bcap, bq, big, big_count, qa, k, p.max_hit_distance, hit_min_len,
                                  singles, seq_map(ix), o, counter, room, status));
                });
                timer.mark("bucket_group");
                const uint64_t n_sp = spilled_fill + n_ovf;
                if (n_sp) sort_path(gsp, carena.alloc_n<uint64_t>(n_sp), n_sp, 0, TAG_HIT_SORT);
            }
            timer.mark("hit_merge");
        }
        qa = qb;
    }
    const int qib = bits_for(nq ? nq - 1 : 0);
    const int seqb = bits_for(ix->n_seqs ? ix->n_seqs - 1 : 0);
    const int posb = bits_for(ix->max_seq_len);
    const int qposb = std::max(16, bits_for(max_qlen));
    // Groups of HSPs, their members counted and placed, for the join of long queries' pieces and for
    // the merge.
    struct {
        GroupMap map;
        uint32_t G = 0;
        uint32_t *cnt = nullptr, *list = nullptr, *perm = nullptr;
        uint2 *where = nullptr;
        uint64_t *off = nullptr;
        uint32_t words[4];
    } gr;
    GroupQuestion asked(ix->host_pool, s);
    auto count_groups = [&](bool by_count) {
        const uint64_t per_base = ((uint64_t)n_hsp << 32) / (std::max<uint64_t>(M, 1) * MG_TARGET);
        gr.map = GroupMap{qstart_d, per_base, 0xFFFFFFFFu / std::max(ix->n_seqs, 1u), nullptr};
        gr.G = nq + (uint32_t)((M * per_base) >> 32);
        if (by_count) {
            gr.G = nq + n_hsp / MG_TARGET;  // the last ones may stay empty
            uint32_t *seen = arena.alloc_n<uint32_t>(2ull * nq);
            uint64_t *first = arena.alloc_n<uint64_t>(nq + 1);
            GN_CUDA(cudaMemsetAsync(seen, 0, 8ull * nq, s));
            GN_LAUNCH("k_query_parts", n_hsp, s,
                      k_query_parts<<<blocks_for(n_hsp), 256, 0, s>>>(hsp, n_hsp, seen, seen + nq));
            void *scr = arena.alloc(scan_scratch_bytes(nq));
            exclusive_scan_u32(seen + nq, first, nq, scr, s);
            gr.map.by_count = first;
        }
        gr.cnt = arena.alloc_n<uint32_t>(gr.G);
        gr.where = arena.alloc_n<uint2>(n_hsp);
        GN_CUDA(cudaMemsetAsync(gr.cnt, 0, 4ull * gr.G, s));
        GN_LAUNCH("k_group_count", n_hsp, s,
                  k_group_count<<<blocks_for(n_hsp), 256, 0, s>>>(hsp, n_hsp, gr.map, gr.cnt, gr.where));
    };
    auto list_groups = [&](uint32_t *words) {  // by size, which the host learns
        gr.list = arena.alloc_n<uint32_t>(gr.G);
        GN_LAUNCH("k_group_lists", gr.G, s, k_group_lists<<<blocks_for(gr.G), 256, 0, s>>>(gr.cnt, gr.G, gr.list, words));
        asked.ask(words);
    };
    auto scan_groups = [&](const uint32_t *cnt) {
        uint64_t *off = arena.alloc_n<uint64_t>(gr.G + 1ull);
        void *scr = arena.alloc(scan_scratch_bytes(gr.G));
        exclusive_scan_u32(cnt, off, gr.G, scr, s);
        return off;
    };
    // The host's answer, and, where a group is too large, groups by the queries' HSPs; then the
    // members' order.  False: a group is still too large.
    auto place_groups = [&](uint32_t *words) {
        asked.answer(gr.words);
        if (gr.words[2]) {
            GN_CUDA(cudaMemsetAsync(words, 0, sizeof(gr.words), s));
            count_groups(true);
            list_groups(words);
            asked.answer(gr.words);
            if (gr.words[2]) return false;
        }
        gr.off = scan_groups(gr.cnt);
        gr.perm = arena.alloc_n<uint32_t>(n_hsp);
        GN_LAUNCH("k_group_scatter", n_hsp, s,
                  k_group_scatter<<<blocks_for(n_hsp), 256, 0, s>>>(gr.where, n_hsp, gr.off, gr.perm));
        return true;
    };
    auto run_groups = [&](const MergeGroups &m, const uint32_t *words, auto stitch) {
        constexpr bool ST = decltype(stitch)::value;
        constexpr int ME = MG_MID / 256, BE = MG_BIG / 1024;
        GN_CUDA(cudaMemsetAsync(m.n_out, 0, 4ull * gr.G, s));
        GN_LAUNCH("k_merge_groups_warp", n_hsp, s, k_merge_groups_warp<ST><<<(gr.G + 7) / 8, 256, 0, s>>>(m, gr.G));
        if (gr.words[0])
            GN_LAUNCH("k_merge_groups", n_hsp, s,
                      k_merge_groups<256, ME, ST><<<gr.words[0], 256, sizeof(MergeSmem<256, ME>), s>>>(m, gr.list, 1, words));
        if (gr.words[1]) {
            allow_max_smem(ix->device);
            GN_LAUNCH("k_merge_groups", n_hsp, s,
                      k_merge_groups<1024, BE, ST><<<gr.words[1], 1024, sizeof(MergeSmem<1024, BE>), s>>>(m, gr.list + (gr.G - 1), -1,
                                                                                                      words + 1));
        }
    };
    bool joined_groups = false;  // the HSPs lie by group
    if (segmented && n_hsp) {
        // pieces onto their queries, then one chain per run of pieces sharing seeds
        GN_LAUNCH("k_segment_map", n_hsp, s,
                  k_segment_map<<<blocks_for(n_hsp), 256, 0, s>>>(hsp, n_hsp, seg_parent_d, seg_off_d));
        const int diagb = bits_for((uint64_t)ix->max_seq_len + max_qlen);
        bool by_groups = seqb + diagb + MG_BITS <= 64;
        if (by_groups) {
            count_groups(false);
            list_groups(words->groups);
            by_groups = place_groups(words->groups);
        }
        DevHsp *joined = arena.alloc_n<DevHsp>(n_hsp);
        if (by_groups) {
            DevHsp *chains = arena.alloc_n<DevHsp>(n_hsp);
            uint32_t *n_chains = arena.alloc_n<uint32_t>(gr.G);
            run_groups(MergeGroups{hsp, gr.perm, gr.off, gr.cnt, diagb, 2, 0, (uint32_t)max_qlen, (uint32_t)k, p.min_hsp_len, chains, n_chains},
                       words->groups, std::true_type());
            uint64_t *to = scan_groups(n_chains);
            pin.fetch(0, to + gr.G, 8);
            GN_LAUNCH("k_group_pack", n_hsp, s,
                      k_group_pack<<<blocks_for(32ull * gr.G), 256, 0, s>>>(chains, gr.off, to, gr.G, gr.map, nq, 0, joined, nullptr, nullptr,
                                                                            nullptr));
            pin.wait();
            n_hsp = (uint32_t)*reinterpret_cast<const uint64_t *>(pin.p);
            gr.off = to;  // the chains lie by group
            gr.cnt = n_chains;
            gr.perm = nullptr;
            joined_groups = true;
        } else {
            uint32_t *perm = arena.alloc_n<uint32_t>(n_hsp);
            sort_records(reinterpret_cast<const uint32_t *>(hsp), HSP_WORDS, n_hsp,
                         {{W_QI, qib, false}, {W_SEQ, seqb, false}, {W_LEN, 32, false}, {W_QS, qposb, false}},
                         perm, arena, s);
            DevHsp *srt = arena.alloc_n<DevHsp>(n_hsp);
            gather_records(reinterpret_cast<const uint32_t *>(hsp), HSP_WORDS, perm, n_hsp,
                           reinterpret_cast<uint32_t *>(srt), s);
            DevHsp *chains = arena.alloc_n<DevHsp>(n_hsp);
            uint32_t *flag = arena.alloc_n<uint32_t>(n_hsp);
            GN_LAUNCH("k_stitch_sweep", n_hsp, s,
                      k_stitch_sweep<<<blocks_for(n_hsp), 256, 0, s>>>(srt, n_hsp, (uint32_t)k, p.min_hsp_len, chains,
                                                                      flag));
            n_hsp = compact_records(reinterpret_cast<const uint32_t *>(chains), HSP_WORDS, flag, n_hsp,
                                    reinterpret_cast<uint32_t *>(joined), arena, s);
        }
        hsp = joined;
        timer.mark("stitch");
    }
    if (keep_hits) res->st_hits.swap(hits_q);
    if (keep) {
        std::vector<DevHsp> v = to_host(hsp, n_hsp, s);
        res->st_hsp.resize(n_hsp);
        if (n_hsp) memcpy(res->st_hsp.data(), v.data(), sizeof(DevHsp) * n_hsp);
    }

    const PackedPair seqs{qp.pk, qp.nb, ix->bank.pk, ix->bank.nb, (int64_t)Packed::pk_words(M) - 1,
                          (int64_t)Packed::nb_words(M) - 1, (int64_t)Packed::pk_words(ix->n_bases) - 1,
                          (int64_t)Packed::nb_words(ix->n_bases) - 1};
    // From here on counts stay on the device (merged HSPs, selected ones, alignments kept): the
    // buffers are sized by what they can be at most, and the kernels read them there, so that the
    // phases follow each other without the host.  Only stage outputs and the paths that sort
    // records over the whole call read them in between.
    const uint32_t N = p.max_alignments;
    const char *senv = getenv("GN_SELECT_PATH"), *renv = getenv("GN_RANK_PATH");
    const bool sort_select = (N > (uint32_t)SQ_CAP) || (N == 0 && keep) || (senv && strcmp(senv, "sort") == 0);
    bool sort_rank = N > (uint32_t)RQ_CAP || sort_select || (renv && strcmp(renv, "sort") == 0);
    auto read_count = [&](const uint64_t *dev) {
        pin.fetch(0, dev, 8);
        pin.wait();
        return (uint32_t)*reinterpret_cast<const uint64_t *>(pin.p);
    };
    // How the HSPs are merged: in one block, by groups, or in order of the whole call.  Groups take
    // every call whose sort keys fit and in which no query has more HSPs in its range of sequences
    // than a block holds; otherwise, and for stage outputs and selections that sort the whole call
    // anyway, the records are sorted (figures: gn_merge_groups.cuh).  Which group an HSP is in does not
    // change when it is extended, so the groups are counted before, and the host learns whether all
    // of them fit while the extension runs.
    const bool merge_block = n_hsp <= MB_CAP && nq <= MB_QUERIES && qib + seqb + qposb + MB_BITS <= 64;
    bool merge_groups = n_hsp && !merge_block && !keep && !sort_select && seqb + qposb + MG_BITS <= 64;
    if (merge_groups) {
        if (!joined_groups) count_groups(false);
        list_groups(words->groups + 4);
    }
    // a9: extension
    if (n_hsp) {
        // resident warps only, taking HSP ends from a counter
        const uint64_t xwarps =
            std::min<uint64_t>((2ull * n_hsp + 31) / 32,
                               (uint64_t)num_sms() * blocks_per_sm(reinterpret_cast<const void *>(k_xdrop), 256) * 8);
        GN_LAUNCH("k_xdrop", n_hsp, s,
                  k_xdrop<<<blocks_for(xwarps * 32, 256), 256, 0, s>>>(hsp, n_hsp, seqs, qstart_d, ix->seq_start_d, sc.match,
                                                                      sc.mismatch, p.xdrop, nq, ix->n_seqs, &words->next_end));
    }
    timer.mark("xdrop_extend");
    if (keep) {
        std::vector<DevHsp> v = to_host(hsp, n_hsp, s);
        res->st_ext.resize(n_hsp);
        for (DevHsp &x : v) x.len = std::min(x.qe - x.qs, x.de - x.ds);  // the extension leaves len to its readers
        if (n_hsp) memcpy(res->st_ext.data(), v.data(), sizeof(DevHsp) * n_hsp);
    }

    // a10: merge overlapped HSPs; per query, its first box and the prefix sums of what is selected
    uint64_t *n_mg_d = arena.alloc_n<uint64_t>(2), *n_sel_own = n_mg_d + 1;
    DevHsp *merged = arena.alloc_n<DevHsp>(n_hsp);
    uint32_t *qfirst = arena.alloc_n<uint32_t>(nq + 1);
    uint64_t *qo = arena.alloc_n<uint64_t>(nq + 1);  // selected HSPs of the queries before each
    uint32_t n_mg = 0;                               // read only where it is needed
    // a11's room: longest first, at most max_alignments per query (all of them: the boxes as they are)
    uint32_t sel_cap = (uint32_t)std::min<uint64_t>(n_hsp, N ? (uint64_t)nq * N : ~0ull);
    const bool block_selects = merge_block && n_hsp && !sort_select && N;
    DevHsp *sel = block_selects ? arena.alloc_n<DevHsp>(sel_cap) : merged;
    // in_order: boxes of one query start in the order by which equally long ones are selected
    auto merge_boxes = [&](int in_order) {
        DevHsp *boxes = arena.alloc_n<DevHsp>(n_hsp);
        if (merge_groups) {
            if (joined_groups) asked.answer(gr.words);  // no larger than they were
            else merge_groups = place_groups(words->groups + 4);
        }
        if (merge_block) {
            GN_LAUNCH("k_merge_block", n_hsp, s,
                      k_merge_block<<<1, MB_THREADS, 0, s>>>(hsp, n_hsp, (uint32_t)seqb, (uint32_t)qposb, nq, N, in_order,
                                                             boxes, merged, qfirst, qo, n_mg_d, block_selects ? sel : nullptr));
        } else if (merge_groups) {
            uint32_t *n_boxes = arena.alloc_n<uint32_t>(gr.G), *cnt_sel = arena.alloc_n<uint32_t>(nq);
            run_groups(MergeGroups{hsp, gr.perm, gr.off, gr.cnt, qposb, max_qlen > 65535 ? 3 : 2, N, 0, 0, 0, boxes, n_boxes},
                       words->groups + 4, std::false_type());
            uint64_t *to = scan_groups(n_boxes);
            GN_LAUNCH("k_group_pack", n_hsp, s,
                      k_group_pack<<<blocks_for(32ull * gr.G), 256, 0, s>>>(boxes, gr.off, to, gr.G, gr.map, nq, N, merged, qfirst, cnt_sel,
                                                                            qo));
            void *scr = arena.alloc(scan_scratch_bytes(nq));
            if (N) exclusive_scan_u32(cnt_sel, qo, nq, scr, s);
        } else {
            uint32_t *perm = arena.alloc_n<uint32_t>(n_hsp);
            // (qi, seq, qs) order; the sweep takes the records of one qs by (ds, qe)
            sort_records(reinterpret_cast<const uint32_t *>(hsp), HSP_WORDS, n_hsp,
                         {{W_QI, qib, false}, {W_SEQ, seqb, false}, {W_QS, qposb, false}}, perm, arena, s);
            DevHsp *srt = arena.alloc_n<DevHsp>(n_hsp);
            gather_records(reinterpret_cast<const uint32_t *>(hsp), HSP_WORDS, perm, n_hsp,
                           reinterpret_cast<uint32_t *>(srt), s);
            uint32_t *flag = arena.alloc_n<uint32_t>(n_hsp);
            GN_LAUNCH("k_overlap_sweep", n_hsp, s,
                      k_overlap_sweep<<<blocks_for(n_hsp), 256, 0, s>>>(srt, n_hsp, boxes, flag, in_order));
            const uint64_t *count = compact_records_async(reinterpret_cast<const uint32_t *>(boxes), HSP_WORDS, flag, n_hsp,
                                                          reinterpret_cast<uint32_t *>(merged), arena, s);
            GN_CUDA(cudaMemcpyAsync(n_mg_d, count, 8, cudaMemcpyDeviceToDevice, s));
            uint32_t *cnt_sel = N && !sort_select ? arena.alloc_n<uint32_t>(nq) : nullptr;
            GN_LAUNCH("k_query_bounds", nq + 1, s,
                      k_query_bounds<<<blocks_for(nq + 1), 256, 0, s>>>(merged, n_mg_d, nq, qfirst, cnt_sel ? nullptr : qo, N, cnt_sel));
            if (cnt_sel) {
                void *scr = arena.alloc(scan_scratch_bytes(nq));
                exclusive_scan_u32(cnt_sel, qo, nq, scr, s);
            }
        }
    };
    if (n_hsp && keep) {  // the stage's boxes are in the sweep's order
        merge_boxes(0);
        n_mg = read_count(n_mg_d);
        std::vector<DevHsp> v = to_host(merged, n_mg, s);
        res->st_merged.resize(n_mg);
        if (n_mg) memcpy(res->st_merged.data(), v.data(), sizeof(DevHsp) * n_mg);
    }
    if (n_hsp) merge_boxes(1);
    timer.mark("overlap_merge");
    if (n_hsp && sort_select && !keep) n_mg = read_count(n_mg_d);

    // a11: selection
    uint32_t n_sel = 0;                      // read only where it is needed
    const uint64_t *n_sel_d = qo + nq;       // the same on the device
    // The buffers from here on take about 170 bytes an alignment: where they would take more than
    // SEL_ASK of them, many more perhaps than there are boxes, the host waits for the number
    // (20 us of a search that takes milliseconds).
    if (n_hsp && !sort_select && sel_cap > SEL_ASK) sel_cap = read_count(n_sel_d);
    if (n_hsp && !sort_select && N && !block_selects) {
        sel = arena.alloc_n<DevHsp>(sel_cap);
        GN_LAUNCH("k_select_query", n_hsp, s,
                  k_select_query<<<nq, SQ_THREADS, 0, s>>>(merged, qfirst, qo, N, max_qlen > 65535 ? 3 : 2, sel));
    } else if (n_mg && sort_select) {
        sel = arena.alloc_n<DevHsp>(n_mg);
        uint32_t *first = arena.alloc_n<uint32_t>(nq);
        uint32_t *perm = arena.alloc_n<uint32_t>(n_mg);
        sort_records(reinterpret_cast<const uint32_t *>(merged), HSP_WORDS, n_mg,
                     {{W_QI, qib, false}, {W_LEN, qposb, true}, {W_SEQ, seqb, false}, {W_QS, qposb, false},
                      {W_DS, posb, false}, {W_QE, qposb, false}, {W_DE, posb, false}},
                     perm, arena, s);
        DevHsp *srt = arena.alloc_n<DevHsp>(n_mg);
        gather_records(reinterpret_cast<const uint32_t *>(merged), HSP_WORDS, perm, n_mg,
                       reinterpret_cast<uint32_t *>(srt), s);
        GN_LAUNCH("k_first_of_query", 0, s,
                  k_first_of_query<<<blocks_for(n_mg), 256, 0, s>>>(reinterpret_cast<const uint32_t *>(srt), HSP_WORDS, n_mg, first));
        uint32_t *flag = arena.alloc_n<uint32_t>(n_mg);
        GN_LAUNCH("k_select_flags", n_mg, s,
                  k_select_flags<<<blocks_for(n_mg), 256, 0, s>>>(srt, n_mg, first, N, flag));
        const uint64_t *count = compact_records_async(reinterpret_cast<const uint32_t *>(srt), HSP_WORDS, flag, n_mg,
                                                      reinterpret_cast<uint32_t *>(sel), arena, s);
        GN_CUDA(cudaMemcpyAsync(n_sel_own, count, 8, cudaMemcpyDeviceToDevice, s));
        n_sel_d = n_sel_own;
    }
    timer.mark("select");
    if (n_hsp && (keep || sort_rank)) {
        n_sel = (n_mg || !sort_select) ? read_count(n_sel_d) : 0;
        sel_cap = n_sel;
    }
    if (keep) {
        std::vector<DevHsp> v = to_host(sel, n_sel, s);
        res->st_sel.resize(n_sel);
        if (n_sel) memcpy(res->st_sel.data(), v.data(), sizeof(DevHsp) * n_sel);
    }

    // a12: banded Smith-Waterman
    const bool any_sel = n_hsp && (!sort_select || n_mg);
    DevAln *aln = arena.alloc_n<DevAln>(any_sel ? sel_cap : 0);
    const SwScore score{sc.match, sc.mismatch, sc.gap_open + sc.gap_extend, sc.gap_extend, 1};
    const bool cut = sc.mismatch < 2 * sc.gap_extend;
    uint32_t *strip = nullptr, *wide = nullptr;
    uint64_t wide_area = 0;
    bool wide_done = true;
    auto align_wide = [&]() {
        auto kernel = cut ? k_banded_sw_wide<true> : k_banded_sw_wide<false>;
        GN_LAUNCH("k_banded_sw_wide", wide_area, s,
                  kernel<<<std::min<uint32_t>((sel_cap + 3) / 4, (uint32_t)num_sms() * 4), 128, 0, s>>>(
                      sel, wide, &words->n_wide, &words->next_wide, seqs, qstart_d, ix->seq_start_d, score, (int32_t)p.band_w, strip,
                      &words->n_strip, &words->strip_band, aln));
    };
    if (any_sel) {
        const uint32_t sms = (uint32_t)num_sms();
        // lanes per HSP of the grouped path (the index's tuning; GN_SW_LANES overrides)
        uint32_t sw_lanes = ix->tuning.sw_lanes ? ix->tuning.sw_lanes : 8;
        if (const char *e = getenv("GN_SW_LANES")) sw_lanes = (uint32_t)atoi(e);
        if (sw_lanes != 16 && sw_lanes != 32) sw_lanes = 8;
        // Alignments of at least sw_long rows get a warp each, and warps are few, one or two a
        // scheduler: a warp alone issues at nearly half the pipes' rate, and the longest alignments,
        // which bound the phase, slow down with every warp that shares theirs.  us at 4 | 8 | 16
        // warps an SM, rows from 512 | 1,024 (default band): 4,900 alignments 165 165 | 182 212 |
        // 223 257; 30,000 alignments 534 375 | 374 307 | 436 449; 50,000 1036 768 | 716 567 | 672
        // 613.  So rows from 512 at 4 warps an SM, from 1,024 at 8 with more than 64 alignments an
        // SM (sw_long_rows, sw_many: the device knows the number), and with no more alignments
        // than warps each gets its own, in any order (sw_lanes = 32 asks for that).
        uint32_t sw_long = ix->rows_by_count ? 0u : ix->tuning.sw_wave_rows;
        if (const char *e = getenv("GN_SW_LONG_ROWS")) sw_long = (uint32_t)std::max(1l, strtol(e, nullptr, 10));
        if (sw_lanes == 32) sw_long = 1;
        const bool ordered = sel_cap > sms * 4 || getenv("GN_SW_LONG_ROWS");
        uint32_t *order = ordered ? arena.alloc_n<uint32_t>(sel_cap) : nullptr;
        const int cap = sw_lanes == 16 ? 48 : 40;
        if (ordered || g_ktimer)
            GN_LAUNCH("k_sw_prepare", sel_cap, s,
                      k_sw_prepare<<<blocks_for(sel_cap), 256, 0, s>>>(sel, n_sel_d, (int32_t)p.band_w, cap, qstart_d, sw_long, sms,
                                                                       words->bins, g_ktimer ? words->cells : nullptr));
        if (ordered)
            GN_LAUNCH("k_sw_order", sel_cap, s,
                      k_sw_order<<<blocks_for(sel_cap), 256, 0, s>>>(sel, n_sel_d, (int32_t)p.band_w, cap, qstart_d, sw_long, sms,
                                                                     words->bins, words->placed, order, &words->n_long));
        uint64_t area[2] = {0, 0};
        if (g_ktimer) {
            pin.fetch(0, words->cells, 16);
            pin.wait();
            memcpy(area, pin.p, 16);
        }
        wide = arena.alloc_n<uint32_t>(sel_cap);
        strip = arena.alloc_n<uint32_t>(sel_cap);
        auto sw_kernel = sw_lanes == 16 ? (cut ? k_banded_sw<16, 2, 1, true> : k_banded_sw<16, 2, 1, false>)
                                        : (cut ? k_banded_sw<8, 3, 2, true> : k_banded_sw<8, 3, 2, false>);
        GN_LAUNCH("k_banded_sw", area[0], s,
                  sw_kernel<<<std::min<uint32_t>((sel_cap + 3) / 4, sms * 2), 128, 0, s>>>(
                      sel, n_sel_d, sms, seqs, qstart_d, ix->seq_start_d, score, (int32_t)p.band_w, &words->next_task, order, wide,
                      &words->n_wide, &words->n_long, &words->next_long, aln));
        wide_area = area[1];
        // Small calls at the default band rarely have an alignment for the wide kernel: they wait for
        // the count (3 of 200 us for an empty launch).
        wide_done = ordered || 2 * (int64_t)p.band_w + 1 > 64 || keep || sort_rank;
        if (wide_done) align_wide();
    }
    // bands that no register path holds, once the host knows of them: they are rare, and the rest of
    // the search does not wait for the question
    auto align_strips = [&](const SearchWords &got) {
        const uint64_t cells = (uint64_t)got.strip_band + 2;
        const uint64_t warps = std::min<uint64_t>({(uint64_t)got.n_strip, (uint64_t)num_sms() * 16,
                                                   std::max<uint64_t>(1, (1ull << 30) / (cells * sizeof(SwCell)))});
        const uint64_t blocks = (warps + 3) / 4;
        SwCell *strips = arena.alloc_n<SwCell>(blocks * 4 * cells);
        GN_LAUNCH("k_banded_sw_strip", got.n_strip, s,
                  k_banded_sw_strip<<<(unsigned)blocks, 128, 0, s>>>(sel, strip, got.n_strip, &words->next_strip, strips, cells, seqs,
                                                                     qstart_d, ix->seq_start_d, score, (int32_t)p.band_w, aln,
                                                                     status));
    };
    SearchWords got{};
    bool strips_done = false;
    if (any_sel && (keep || sort_rank)) {
        pin.fetch(0, words, sizeof(SearchWords));
        pin.wait();
        memcpy(&got, pin.p, sizeof(SearchWords));
        if (got.n_strip) align_strips(got);
        strips_done = true;
    }
    timer.mark("banded_sw");
    if (keep) {
        std::vector<DevAln> v = to_host(aln, n_sel, s);
        res->st_aln.resize(n_sel);
        for (uint32_t i = 0; i < n_sel; ++i) {
            gn_hit &h = res->st_aln[i];
            h.query = v[i].qi; h.seq = v[i].seq; h.q_start = v[i].qs; h.q_end = v[i].qe;
            h.db_start = v[i].ds; h.db_end = v[i].de; h.score = v[i].score; h.rank = 0; h.evalue = 0; h.bits = 0;
        }
    }

    // a13: duplicates (same query, sequence and ranges: keep the best score), rank by score, statistics
    uint32_t n_out = 0;
    gn_hit *fin = arena.alloc_n<gn_hit>(any_sel ? sel_cap : 0);
    bool hits_read = false;  // res->hits and res->qoff are filled
    if (any_sel && !sort_rank) {
        // a small call's hits come back as they lie (each query's at its selected HSPs' place)
        // with the counts, in one read; a larger one's are put together first
        const size_t hits_bytes = sizeof(gn_hit) * (size_t)sel_cap, qo_bytes = 8 * (nq + 1ull);
        const bool small = hits_bytes + qo_bytes + 4ull * nq <= (1u << 17);
        gn_hit *hits = arena.alloc_n<gn_hit>(sel_cap);
        uint32_t *qcount = arena.alloc_n<uint32_t>(nq);
        const bool few = N && N <= (uint32_t)RQ_SMALL;  // no query has more alignments
        const unsigned rgrid = (unsigned)std::min<uint64_t>(nq, (uint64_t)num_sms() * (few ? 16 : 5));
        auto rank_kernel = few ? k_rank_query<RQ_SMALL, 1> : k_rank_query<256, RQ_CAP / 256>;
        uint64_t *qoff = arena.alloc_n<uint64_t>(nq + 1);
        void *scr = arena.alloc(scan_scratch_bytes(nq));
        PinnedBlock back(ix->host_pool, sizeof(SearchWords) + qo_bytes + (small ? hits_bytes + 4ull * nq : 0), s);
        for (;;) {
            GN_LAUNCH("k_rank_query", sel_cap, s,
                      rank_kernel<<<rgrid, few ? RQ_SMALL : 256, 0, s>>>(
                          aln, qo, nq, qstart_d, seqb, (double)ix->n_bases, sc.lambda, sc.K, p.max_evalue, hits, qcount,
                          &words->too_many));
            size_t at = sizeof(SearchWords);
            if (small) {
                back.fetch(at, qo, qo_bytes);
                at += qo_bytes;
                back.fetch(at, hits, hits_bytes);
                at += hits_bytes;
                back.fetch(at, qcount, 4ull * nq);
            } else {
                exclusive_scan_u32(qcount, qoff, nq, scr, s);
                GN_LAUNCH("k_gather_ranked", sel_cap, s,
                          k_gather_ranked<<<(unsigned)std::min<uint64_t>(nq, (uint64_t)num_sms() * 8), 256, 0, s>>>(hits, qo, qoff, nq, fin));
                back.fetch(at, qoff, qo_bytes);
            }
            back.fetch(0, words, sizeof(SearchWords));
            back.wait();
            memcpy(&got, back.p, sizeof(SearchWords));
            if (!wide_done && got.n_wide) {
                align_wide();
                wide_done = true;
                continue;
            }
            if (strips_done || !got.n_strip) break;
            align_strips(got);
            strips_done = true;
        }
        if (got.too_many) {
            sort_rank = true;
            n_sel = read_count(n_sel_d);
        } else {
            res->qoff.resize(nq + 1);
            const uint64_t *q_at = reinterpret_cast<const uint64_t *>(back.p + sizeof(SearchWords));
            if (small) {
                const gn_hit *h = reinterpret_cast<const gn_hit *>(back.p + sizeof(SearchWords) + qo_bytes);
                const uint32_t *c = reinterpret_cast<const uint32_t *>(back.p + sizeof(SearchWords) + qo_bytes + hits_bytes);
                res->qoff[0] = 0;
                for (uint32_t q = 0; q < nq; ++q) {
                    res->hits.insert(res->hits.end(), h + q_at[q], h + q_at[q] + c[q]);
                    res->qoff[q + 1] = res->hits.size();
                }
            } else {
                memcpy(res->qoff.data(), q_at, qo_bytes);
                res->hits = to_host(fin, (size_t)res->qoff[nq], s);
            }
            hits_read = true;
        }
    }
    if (n_sel && sort_rank) {
        const int scb = std::min(31, bits_for(std::max<uint64_t>(65535, max_qlen) * (uint64_t)std::max(1, sc.match)));
        uint32_t *perm = arena.alloc_n<uint32_t>(n_sel);
        sort_records(reinterpret_cast<const uint32_t *>(aln), ALN_WORDS, n_sel,
                     {{A_QI, qib, false}, {A_SEQ, seqb, false}, {A_QS, qposb, false}, {A_QE, qposb, false},
                      {A_DS, posb, false}, {A_DE, posb, false}, {A_SCORE, scb, true}},
                     perm, arena, s);
        DevAln *srt = arena.alloc_n<DevAln>(n_sel);
        gather_records(reinterpret_cast<const uint32_t *>(aln), ALN_WORDS, perm, n_sel, reinterpret_cast<uint32_t *>(srt), s);
        uint32_t *flag = arena.alloc_n<uint32_t>(n_sel);
        GN_LAUNCH("k_dup_flags", n_sel, s,
                  k_dup_flags<<<blocks_for(n_sel), 256, 0, s>>>(srt, n_sel, flag));
        DevAln *uniq = arena.alloc_n<DevAln>(n_sel);
        uint32_t nu = compact_records(reinterpret_cast<const uint32_t *>(srt), ALN_WORDS, flag, n_sel,
                                      reinterpret_cast<uint32_t *>(uniq), arena, s);
        if (nu) {
            uint32_t *perm2 = arena.alloc_n<uint32_t>(nu);
            sort_records(reinterpret_cast<const uint32_t *>(uniq), ALN_WORDS, nu,
                         {{A_QI, qib, false}, {A_SCORE, scb, true}, {A_SEQ, seqb, false}, {A_QS, qposb, false},
                          {A_DS, posb, false}, {A_QE, qposb, false}, {A_DE, posb, false}},
                         perm2, arena, s);
            DevAln *ranked = arena.alloc_n<DevAln>(nu);
            gather_records(reinterpret_cast<const uint32_t *>(uniq), ALN_WORDS, perm2, nu,
                           reinterpret_cast<uint32_t *>(ranked), s);
            uint32_t *first = arena.alloc_n<uint32_t>(nq);
            GN_LAUNCH("k_first_of_query", 0, s,
                      k_first_of_query<<<blocks_for(nu), 256, 0, s>>>(reinterpret_cast<const uint32_t *>(ranked), ALN_WORDS, nu, first));
            gn_hit *hits = arena.alloc_n<gn_hit>(nu);
            uint32_t *f2 = arena.alloc_n<uint32_t>(nu);
            GN_LAUNCH("k_finalize", nu, s,
                      k_finalize<<<blocks_for(nu), 256, 0, s>>>(ranked, nu, first, qstart_d, (double)ix->n_bases, sc.lambda, sc.K,
                                                      p.max_evalue, hits, f2));
            static_assert(sizeof(gn_hit) % 4 == 0, "gn_hit words");
            n_out = compact_records(reinterpret_cast<const uint32_t *>(hits), (int)(sizeof(gn_hit) / 4), f2, nu,
                                    reinterpret_cast<uint32_t *>(fin), arena, s);
        }
    }
    timer.mark("rank");
    if (!hits_read) {
        res->hits = to_host(fin, n_out, s);
        pin.fetch(0, words, sizeof(SearchWords));
        pin.wait();
        memcpy(&got, pin.p, sizeof(SearchWords));
        res->qoff.assign(nq + 1, 0);
        for (uint32_t i = 0; i < n_out; ++i) res->qoff[res->hits[i].query + 1]++;
        for (uint32_t i = 0; i < nq; ++i) res->qoff[i + 1] += res->qoff[i];
    }
    GN_REQUIRE((got.wait_status & DEV_ERR_TIMEOUT) == 0, GN_ETIMEOUT, "a device-side wait ran out (scan look-back)");
#ifdef GN_CHECKS
    uint32_t cbits = 0;
    GN_CUDA(cudaMemcpyAsync(&cbits, check_bits, 4, cudaMemcpyDeviceToHost, s));
    GN_CUDA(cudaStreamSynchronize(s));
    GN_REQUIRE((cbits & DEV_ERR_BOUNDS) == 0, GN_EINTERNAL, "a device-side bounds check failed (checked build)");
#endif
    GN_REQUIRE((got.status & DEV_ERR_BOUNDS) == 0, GN_EINTERNAL, "a device-side bounds check failed");
    GN_REQUIRE((got.status & DEV_ERR_BAND_TOO_WIDE) == 0, GN_ETOOBIG,
               "an alignment band exceeded 65,535 diagonals or its window 2^32 cells");
    timer.mark("output");
    GN_CUDA(cudaStreamSynchronize(s));
    {
        std::lock_guard<std::mutex> lk(ix->phase_mu);
        timer.finish(ix->last_phases);
        ix->last_kernels.clear();
        for (auto &r : ktimer.recs) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, r.a, r.b);
            auto it = std::find_if(ix->last_kernels.begin(), ix->last_kernels.end(),
                                   [&](const gn_index::KernelStat &k) { return strcmp(k.name, r.name) == 0; });
            if (it == ix->last_kernels.end()) {
                ix->last_kernels.push_back({r.name, 0.0, 0u, 0ull});
                it = ix->last_kernels.end() - 1;
            }
            it->ms += ms;
            it->launches += 1;
            it->units += r.units;
        }
    }

    arena.release();
}

}  // namespace gn
