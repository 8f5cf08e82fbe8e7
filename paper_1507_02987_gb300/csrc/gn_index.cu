// gn_index.cu - device construction of the inverted index ("Inverted Indexes"
// section of the paper): the bank is packed to 2 bits per base, cut into
// non-overlapping windows at offsets 0, t, 2t, ... of every sequence, and each
// window's occurrence is filed under its k-mer code.  Buckets are a CSR
// structure: off[c] .. off[c+1] index the occurrences of code c, in ascending
// (sequence, position) order, stored as the window's global base offset.
#include <algorithm>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>

#include "gn_internal.cuh"

namespace gn {

// windows per sequence: len >= span ? (len - span) / t + 1 : 0 (span = k without a mask)
__global__ void k_window_counts(const uint64_t *__restrict__ seq_start, uint32_t n_seqs, int span, int t,
                                uint32_t *__restrict__ wcnt) {
    uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_seqs) return;
    uint64_t L = seq_start[s + 1] - seq_start[s];
    wcnt[s] = L >= (uint64_t)span ? (uint32_t)((L - span) / t + 1) : 0u;
}

constexpr int WIN_J = 8;  // windows per lane per warp chunk
constexpr int WIN_CHUNK = 32 * WIN_J;

// Windows of warp chunk c: [c * WIN_CHUNK, ...), lane by lane.  COUNT: the chunk's valid
// windows (no non-base at a kept position).  Otherwise: the key (code << 32 | global offset)
// of every valid window, in window order from the chunk's first slot, and the bucket
// histogram.  One count per chunk and a ballot rank give the slots, so that no flag or slot
// per window goes through memory (400 Mbp, 36.4 M windows: flags, their scan and the two
// window passes 0.9 GB, now 0.45 GB).  The number of windows, woff[n_seqs], is known to the device
// only: n_chunks is as many chunks as there can be.  prev (a key's bits above the code are
// free): the base before the window goes along there, so that its signature needs no look at it.
constexpr int PREV_SHIFT = 61;

template <bool COUNT>
__global__ void k_bank_windows(const uint64_t *__restrict__ seq_start, const uint64_t *__restrict__ woff,
                               uint32_t n_seqs, uint64_t n_chunks, const uint32_t *__restrict__ pk,
                               const uint32_t *__restrict__ nb, SeedShape sh, int t, bool prev,
                               uint32_t *__restrict__ count, uint32_t *__restrict__ hist,
                               const uint64_t *__restrict__ first, uint64_t *__restrict__ keys) {
    const int lane = threadIdx.x & 31;
    const uint64_t chunk = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t w0 = chunk * WIN_CHUNK, W = woff[n_seqs];
    if (chunk >= n_chunks) return;
    if (w0 >= W) {
        if (COUNT && lane == 0) count[chunk] = 0;
        return;
    }
    uint32_t s = 0;
    if (lane == 0) s = dev_upper_index(woff, n_seqs + 1, w0);
    s = __shfl_sync(0xffffffffu, s, 0);
    uint64_t slot = COUNT ? 0 : first[chunk];
    uint32_t total = 0;
#pragma unroll
    for (int it = 0; it < WIN_J; ++it) {
        const uint64_t w = w0 + (uint64_t)it * 32 + lane;
        uint64_t g = 0;
        bool ok = w < W;
        if (ok) {
            while (woff[s + 1] <= w) ++s;
            g = seq_start[s] + (w - woff[s]) * (uint64_t)t;
            ok = !dev_seed_has_nonbase(nb, g, sh);
        }
        const uint32_t m = __ballot_sync(0xffffffffu, ok);
        if (COUNT) {
            total += __popc(m);
        } else {
            if (ok) {
                const uint32_t code = dev_seed_code(pk, g, sh);
                atomicAdd(&hist[code], 1u);
                uint64_t key = ((uint64_t)code << 32) | g;
                if (prev) key |= (uint64_t)(g > seq_start[s] ? dev_base(pk, nb, g - 1) : SIG_NO_BASE) << PREV_SHIFT;
                keys[slot + __popc(m & ((1u << lane) - 1u))] = key;
            }
            slot += __popc(m);
        }
    }
    if (COUNT && lane == 0) count[chunk] = total;
}

// Signature of the occurrence at bank position g.  Fields ahead are taken from the packed
// bases whatever sequence they belong to and whether they are bases: a field that matches
// wrongly costs the search one check, none is missed.  Bound by the gather of the bases after
// g (one or two 32-byte sectors an occurrence).
__device__ __forceinline__ uint32_t occurrence_sig(uint64_t g, uint64_t n, const uint32_t *__restrict__ pk,
                                                   const uint32_t *__restrict__ nb, const SeqMap &sm,
                                                   const SeedShape &sh, int t, int kind) {
    uint32_t sig = 0;
    if (kind == SIG_FLANK) {
        sig = SIG_NO_BASE;
        if (g > 0 && g < n) {
            const uint32_t sq = sm.lut ? dev_seq_of(sm, g) : dev_upper_index(sm.start, sm.n_seqs + 1, g);
            if (sm.start[sq] != g) sig = dev_base(pk, nb, g - 1);
        }
        if (g + (uint64_t)sh.span <= n) sig |= sig_flank(pk, g + (uint64_t)sh.span);
    } else {
        for (int j = 0; j < SIG_FIELDS; ++j) {
            const uint64_t x = g + (uint64_t)t * (j + 1);
            sig |= (x + (uint64_t)sh.span <= n ? sig_hash(dev_seed_code(pk, x, sh)) : SIG_NONE) << (10 * j);
        }
    }
    return sig;
}

// Occurrences and their signatures from the sorted keys (keys null: signatures of the
// occurrences that post already holds).  post and sig: post_alloc_entries words.  prev: the keys
// hold the base before the window, and the signature costs the gather after it alone (build of
// 400 M occurrences at stride 1: 29.3 -> 23.0 ms).
__global__ void k_occurrences(const uint64_t *__restrict__ keys, uint64_t n_post, uint32_t *__restrict__ post,
                              uint32_t *__restrict__ sig, uint64_t n, const uint32_t *__restrict__ pk,
                              const uint32_t *__restrict__ nb, SeqMap sm, SeedShape sh, int t, int kind, bool prev) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_post) return;
    const uint64_t key = keys ? keys[i] : (uint64_t)post[i];
    const uint32_t g = (uint32_t)key;
    if (keys) post[i] = g;
    if (!sig) return;
    if (prev) {
        const uint64_t x = (uint64_t)g + (uint64_t)sh.span;
        sig[i] = (uint32_t)(key >> PREV_SHIFT) | (x <= n ? sig_flank(pk, x) : 0u);
    } else {
        sig[i] = occurrence_sig(g, n, pk, nb, sm, sh, t, kind);
    }
}

// Device memory of an index: two blocks, one of what the bank's size decides, one of what the
// number of occurrences decides.  An allocation or a release is 10 to 100 us of host time; with seven
// of each, build | release took 354 | 152 us at 1.25 Mbp and 2,954 | 507 us at 400 Mbp, now 281 | 111
// and 2,780 | 339.
static void alloc_fixed(gn_index *ix, uint64_t ns, uint64_t n, uint64_t nbk, uint64_t nlut) {
    size_t at = 0;
    auto place = [&](size_t bytes) {
        const size_t from = at;
        at += (bytes + 255) / 256 * 256;
        return from;
    };
    const size_t start = place(8 * (ns + 1)), pk = place(4 * Packed::pk_words(n)), nb = place(4 * Packed::nb_words(n)),
                 off = place(8 * (nbk + 1)), lut = place(4 * nlut);
    GN_CUDA(cudaMalloc(&ix->fixed_d, at));
    ix->seq_start_d = reinterpret_cast<uint64_t *>(ix->fixed_d + start);
    ix->bank.pk = reinterpret_cast<uint32_t *>(ix->fixed_d + pk);
    ix->bank.nb = reinterpret_cast<uint32_t *>(ix->fixed_d + nb);
    ix->off_d = reinterpret_cast<uint64_t *>(ix->fixed_d + off);
    ix->seq_lut_d = reinterpret_cast<uint32_t *>(ix->fixed_d + lut);
    ix->device_bytes = 8 * (ns + 1) + 4 * (Packed::pk_words(n) + Packed::nb_words(n)) + 8 * (nbk + 1) + 4 * nlut;
}

// Whether an index may take `bytes` for signatures: searches work without them, slower, so an eighth of
// the device stays free for the searches' own buffers (GN_SIGNATURE_RESERVE: as many bytes
// instead).  The pool's memory is theirs again after the build.  An index whose signatures are below
// SIG_SMALL does not ask.  400 Mbp build in 2.78 ms at stride 11 and 22.98 at 1, with the question or without.
constexpr size_t SIG_SMALL = 64 << 20;

static bool signatures_fit(const gn_index *ix, size_t bytes) {
    const char *env = getenv("GN_SIGNATURE_RESERVE");
    if (!env && bytes < SIG_SMALL) return true;
    size_t free_b = 0, total_b = 0;
    uint64_t pooled = 0;
    cudaMemPool_t pool;
    GN_CUDA(cudaMemGetInfo(&free_b, &total_b));
    GN_CUDA(cudaDeviceGetDefaultMemPool(&pool, ix->device));
    GN_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &pooled));
    const uint64_t reserve = env ? strtoull(env, nullptr, 10) : total_b / 8;
    return free_b + pooled >= bytes && free_b + pooled - bytes >= reserve;
}

// The occurrences and their signatures; without room for those searches take the path that does
// not read them.
static void alloc_occurrences(gn_index *ix) {
    const size_t want = (sizeof(uint32_t) * post_alloc_entries(ix->n_postings) + 255) / 256 * 256;
    if (signatures_fit(ix, 2 * want) && cudaMalloc(&ix->post_d, 2 * want) == cudaSuccess) {
        ix->sig_d = ix->post_d + want / sizeof(uint32_t);
        ix->device_bytes += 2 * sizeof(uint32_t) * ix->n_postings;
    } else {
        cudaGetLastError();
        GN_CUDA(cudaMalloc(&ix->post_d, want));
        ix->sig_d = nullptr;
        ix->device_bytes += sizeof(uint32_t) * ix->n_postings;
    }
}

// lut[j] = last sequence s with start[s] <= j << SEQ_LUT_SHIFT (positions past the bank
// map to the last sequence).
__global__ void k_seq_lut(const uint64_t *__restrict__ start, uint32_t ns, uint64_t n, uint64_t nlut,
                          uint32_t *__restrict__ lut) {
    const uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nlut) return;
    const uint64_t x = min(j << SEQ_LUT_SHIFT, n > 0 ? n - 1 : 0);
    lut[j] = dev_upper_index(start, ns, x);  // over the ns starts: the result is < ns
}

// Seeds of `span` bases keeping the positions set in `keep` (k of them).
static void index_build_shape(const gn_bank *db, int k, int span, uint32_t keep, int t, cudaStream_t s, gn_index *ix);

void index_build(const gn_bank *db, int k, int t, cudaStream_t s, gn_index *ix) {
    GN_REQUIRE(k >= 1 && k <= 16, GN_EINVAL, "k must be in 1..16");
    index_build_shape(db, k, k, (uint32_t)((1ull << k) - 1ull), t, s, ix);
}

// "Methods": a mask such as 111010010100110111 ('1' = base kept, '0' = removed) over
// windows of the mask's length.
void index_build_masked(const gn_bank *db, const char *mask, int t, cudaStream_t s, gn_index *ix) {
    GN_REQUIRE(mask, GN_EINVAL, "mask is required");
    const size_t span = strlen(mask);
    GN_REQUIRE(span >= 1 && span <= 32, GN_EINVAL, "a mask has 1..32 positions");
    uint32_t keep = 0;
    int k = 0;
    for (size_t i = 0; i < span; ++i) {
        GN_REQUIRE(mask[i] == '0' || mask[i] == '1', GN_EINVAL, "a mask holds only '0' and '1'");
        if (mask[i] == '1') { keep |= 1u << i; ++k; }
    }
    GN_REQUIRE(k >= 1 && k <= 16, GN_EINVAL, "a mask keeps 1..16 positions");
    index_build_shape(db, k, (int)span, keep, t, s, ix);
}

static void index_build_shape(const gn_bank *db, int k, int span, uint32_t keep, int t, cudaStream_t s,
                              gn_index *ix) {
    GN_REQUIRE(db && db->seq_start, GN_EINVAL, "bank and bank.seq_start are required");
    GN_REQUIRE(t >= 1, GN_EINVAL, "stride must be >= 1");
    const uint32_t ns = db->n_seqs;
    const uint64_t n = db->seq_start[ns] - db->seq_start[0];
    GN_REQUIRE(db->seq_start[0] == 0, GN_EINVAL, "bank.seq_start[0] must be 0");
    GN_REQUIRE(n < (1ull << 32), GN_ETOOBIG, "bank must hold fewer than 2^32 bases");
    GN_REQUIRE(n == 0 || db->bases, GN_EINVAL, "bank.bases is required");
    uint64_t maxlen = 0;
    for (uint32_t i = 0; i < ns; ++i) {
        GN_REQUIRE(db->seq_start[i + 1] >= db->seq_start[i], GN_EINVAL, "bank.seq_start must be non-decreasing");
        maxlen = std::max<uint64_t>(maxlen, db->seq_start[i + 1] - db->seq_start[i]);
    }
    GN_CUDA(cudaGetDevice(&ix->device));
    configure_mempool(ix->device);
    ix->k = k;
    ix->t = t;
    ix->span = span;
    ix->keep = keep;
    ix->n_seqs = ns;
    ix->n_bases = n;
    ix->max_seq_len = (uint32_t)maxlen;
    ix->seq_start_h.assign(db->seq_start, db->seq_start + ns + 1);
    const SeedShape sh{k, span, keep};

    const uint64_t nbk = 1ull << (2 * k);
    const uint64_t nlut = (n >> SEQ_LUT_SHIFT) + 1;
    alloc_fixed(ix, ns, n, nbk, nlut);
    GN_CUDA(cudaMemcpyAsync(ix->seq_start_d, ix->seq_start_h.data(), sizeof(uint64_t) * (ns + 1),
                            cudaMemcpyHostToDevice, s));
    // sequence lookup table: the sequence holding each block of 2^SEQ_LUT_SHIFT bases
    if (ns > 0)
        GN_LAUNCH("k_seq_lut", nlut, s,
                  k_seq_lut<<<(unsigned)((nlut + 255) / 256), 256, 0, s>>>(ix->seq_start_d, ns, n, nlut, ix->seq_lut_d));
    else
        GN_CUDA(cudaMemsetAsync(ix->seq_lut_d, 0, sizeof(uint32_t) * nlut, s));

    DeviceArena arena(s);
    uint32_t *wait_status = arena.alloc_n<uint32_t>(1);  // bounded waits of the scans
    GN_CUDA(cudaMemsetAsync(wait_status, 0, 4, s));
    WaitStatusScope wscope(wait_status);
    // K1: 2-bit packing of the bank
    const uint8_t *bases_d = reinterpret_cast<const uint8_t *>(db->bases);
    if (db->bases_mem == GN_MEM_HOST && n > 0) {
        uint8_t *tmp = arena.alloc_n<uint8_t>(n);
        GN_CUDA(cudaMemcpyAsync(tmp, db->bases, n, cudaMemcpyHostToDevice, s));
        bases_d = tmp;
    }
    pack_bases(bases_d, n, ix->bank, s);

    // windows per sequence and their exclusive scan
    uint32_t *wcnt = arena.alloc_n<uint32_t>(ns);
    uint64_t *woff = arena.alloc_n<uint64_t>(ns + 1);
    if (ns) {
        GN_LAUNCH("k_window_counts", ns, s,
                  k_window_counts<<<(ns + 255) / 256, 256, 0, s>>>(ix->seq_start_d, ns, span, t, wcnt));
    }
    void *scan_scr = arena.alloc(std::max(scan_scratch_bytes(ns), scan_scratch_bytes(nbk)));
    exclusive_scan_u32(wcnt, woff, ns, scan_scr, s);

    // K2: valid windows per chunk and their exclusive scan
    const uint64_t w_max = n / (uint64_t)t + ns;  // at most one window a sequence more than its share
    const uint64_t chunks = (w_max + WIN_CHUNK - 1) / WIN_CHUNK;
    const unsigned grid = (unsigned)std::max<uint64_t>(1, (chunks * 32 + 255) / 256);
    const SigKind kind = sig_kind(k, span, t);
    const bool prev = kind == SIG_FLANK && 32 + 2 * k <= PREV_SHIFT;
    uint32_t *ccnt = arena.alloc_n<uint32_t>(chunks);
    uint64_t *coff = arena.alloc_n<uint64_t>(chunks + 1);
    if (chunks) {
        GN_LAUNCH("k_bank_windows_count", w_max, s,
                  k_bank_windows<true><<<grid, 256, 0, s>>>(ix->seq_start_d, woff, ns, chunks, ix->bank.pk, ix->bank.nb, sh, t, prev,
                                                  ccnt, nullptr, nullptr, nullptr));
    }
    void *scan_scr2 = arena.alloc(scan_scratch_bytes(chunks));
    exclusive_scan_u32(ccnt, coff, chunks, scan_scr2, s);
    uint64_t P = 0;
    GN_CUDA(cudaMemcpyAsync(&P, coff + chunks, sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    GN_CUDA(cudaStreamSynchronize(s));
    ix->n_postings = P;

    // K3: keys of the valid windows and the bucket histogram, whose exclusive scan gives the
    // bucket starts
    uint32_t *hist = arena.alloc_n<uint32_t>(nbk);
    GN_CUDA(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * nbk, s));
    uint64_t *keys = arena.alloc_n<uint64_t>(P);
    uint64_t *keys_alt = arena.alloc_n<uint64_t>(P);
    if (P) {
        GN_LAUNCH("k_bank_windows_keys", w_max, s,
                  k_bank_windows<false><<<grid, 256, 0, s>>>(ix->seq_start_d, woff, ns, chunks, ix->bank.pk, ix->bank.nb, sh, t, prev,
                                                   nullptr, hist, coff, keys));
    }
    exclusive_scan_u32(hist, ix->off_d, nbk, scan_scr, s);

    // K4: stable scatter = stable radix sort of (code, global offset) keys by code
    void *rs = arena.alloc(radix_scratch_bytes(P));
    bool flipped = radix_sort(keys, keys_alt, nullptr, nullptr, P, 32, 32 + 2 * k, rs, s, TAG_INDEX_SORT);
    alloc_occurrences(ix);
    if (P) {
        GN_LAUNCH("k_occurrences", P, s,
                  k_occurrences<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(flipped ? keys_alt : keys, P, ix->post_d, ix->sig_d, n,
                                                                         ix->bank.pk, ix->bank.nb, seq_map(ix), sh, t, kind, prev));
    }
    uint32_t wst = 0;
    GN_CUDA(cudaMemcpyAsync(&wst, wait_status, 4, cudaMemcpyDeviceToHost, s));
    arena.release();
    GN_CUDA(cudaStreamSynchronize(s));
    GN_REQUIRE((wst & DEV_ERR_TIMEOUT) == 0, GN_ETIMEOUT, "a device-side wait ran out (scan look-back)");
}

void index_free(gn_index *ix) {
    if (!ix) return;
    cudaFree(ix->fixed_d);
    cudaFree(ix->post_d);
}

void index_export(const gn_index *ix, uint64_t *bucket_start, uint32_t *post_seq, uint32_t *post_pos) {
    const uint64_t nbk = 1ull << (2 * ix->k);
    if (bucket_start) GN_CUDA(cudaMemcpy(bucket_start, ix->off_d, sizeof(uint64_t) * (nbk + 1), cudaMemcpyDeviceToHost));
    if (!post_seq && !post_pos) return;
    std::vector<uint32_t> g(ix->n_postings);
    if (ix->n_postings)
        GN_CUDA(cudaMemcpy(g.data(), ix->post_d, sizeof(uint32_t) * ix->n_postings, cudaMemcpyDeviceToHost));
    // decode global offsets to (sequence, position) for the caller
    const std::vector<uint64_t> &st = ix->seq_start_h;
    for (uint64_t i = 0; i < ix->n_postings; ++i) {
        uint32_t sidx = (uint32_t)(std::upper_bound(st.begin(), st.end(), (uint64_t)g[i]) - st.begin()) - 1;
        if (post_seq) post_seq[i] = sidx;
        if (post_pos) post_pos[i] = (uint32_t)(g[i] - st[sidx]);
    }
}

// --------------------------------------------------------- persistence --
// File layout (little-endian): a header of 16 uint64 (magic, version, k, stride,
// n_seqs, n_bases, n_postings, max_seq_len, word counts of the sections that
// follow, seed span and kept-position mask), then the sections in order: sequence starts (n_seqs + 1 uint64), packed
// bank words, non-base words, bucket starts (4^k + 1 uint64), occurrences
// (n_postings uint32), sequence lookup table.  Device arrays move through a bounded
// host buffer, so an index of any size needs only that much host memory.
constexpr uint64_t IX_MAGIC = 0x31584449474F4E47ull;  // "GNOGIDX1"
constexpr uint64_t IX_VERSION = 2;
constexpr size_t IX_CHUNK = 64ull << 20;

namespace {
struct FileCloser {
    FILE *f;
    ~FileCloser() { if (f) fclose(f); }
};
void write_all(FILE *f, const void *p, size_t bytes) {
    GN_REQUIRE(bytes == 0 || fwrite(p, 1, bytes, f) == bytes, GN_EINVAL, "index file: write failed");
}
void read_all(FILE *f, void *p, size_t bytes) {
    GN_REQUIRE(bytes == 0 || fread(p, 1, bytes, f) == bytes, GN_EINVAL, "index file: truncated or unreadable");
}
void write_device(FILE *f, const void *d, size_t bytes, std::vector<uint8_t> &buf) {
    for (size_t o = 0; o < bytes; o += IX_CHUNK) {
        const size_t n = std::min(IX_CHUNK, bytes - o);
        GN_CUDA(cudaMemcpy(buf.data(), static_cast<const uint8_t *>(d) + o, n, cudaMemcpyDeviceToHost));
        write_all(f, buf.data(), n);
    }
}
void read_device(FILE *f, void *d, size_t bytes, std::vector<uint8_t> &buf) {
    for (size_t o = 0; o < bytes; o += IX_CHUNK) {
        const size_t n = std::min(IX_CHUNK, bytes - o);
        read_all(f, buf.data(), n);
        GN_CUDA(cudaMemcpy(static_cast<uint8_t *>(d) + o, buf.data(), n, cudaMemcpyHostToDevice));
    }
}
}  // namespace

void index_save(const gn_index *ix, const char *path) {
    GN_REQUIRE(path, GN_EINVAL, "path is required");
    FILE *f = fopen(path, "wb");
    GN_REQUIRE(f, GN_EINVAL, std::string("cannot create ") + path);
    FileCloser fc{f};
    GN_CUDA(cudaSetDevice(ix->device));
    const uint64_t npk = Packed::pk_words(ix->n_bases), nnb = Packed::nb_words(ix->n_bases);
    const uint64_t nbk = (1ull << (2 * ix->k)) + 1, nlut = (ix->n_bases >> SEQ_LUT_SHIFT) + 1;
    uint64_t hdr[16] = {IX_MAGIC, IX_VERSION, (uint64_t)ix->k, (uint64_t)ix->t, ix->n_seqs, ix->n_bases,
                        ix->n_postings, ix->max_seq_len, npk, nnb, nbk, nlut, (uint64_t)ix->span, ix->keep, 0, 0};
    write_all(f, hdr, sizeof(hdr));
    write_all(f, ix->seq_start_h.data(), sizeof(uint64_t) * (ix->n_seqs + 1));
    std::vector<uint8_t> buf(IX_CHUNK);
    write_device(f, ix->bank.pk, 4 * npk, buf);
    write_device(f, ix->bank.nb, 4 * nnb, buf);
    write_device(f, ix->off_d, 8 * nbk, buf);
    write_device(f, ix->post_d, 4 * ix->n_postings, buf);
    write_device(f, ix->seq_lut_d, 4 * nlut, buf);
    GN_REQUIRE(fflush(f) == 0, GN_EINVAL, "index file: write failed");
}

void index_load(const char *path, gn_index *ix) {
    GN_REQUIRE(path, GN_EINVAL, "path is required");
    FILE *f = fopen(path, "rb");
    GN_REQUIRE(f, GN_EINVAL, std::string("cannot open ") + path);
    FileCloser fc{f};
    uint64_t hdr[16];
    read_all(f, hdr, sizeof(hdr));
    GN_REQUIRE(hdr[0] == IX_MAGIC, GN_EINVAL, "not an index file");
    GN_REQUIRE(hdr[1] == IX_VERSION, GN_EINVAL, "unsupported index file version");
    const int k = (int)hdr[2], t = (int)hdr[3];
    GN_REQUIRE(k >= 1 && k <= 16 && t >= 1, GN_EINVAL, "index file: bad k or stride");
    const uint64_t ns = hdr[4], n = hdr[5], np = hdr[6];
    GN_REQUIRE(ns < (1ull << 32) && n < (1ull << 32) && np <= n, GN_EINVAL, "index file: bad sizes");
    const uint64_t npk = Packed::pk_words(n), nnb = Packed::nb_words(n);
    const uint64_t nbk = (1ull << (2 * k)) + 1, nlut = (n >> SEQ_LUT_SHIFT) + 1;
    GN_REQUIRE(hdr[8] == npk && hdr[9] == nnb && hdr[10] == nbk && hdr[11] == nlut, GN_EINVAL,
               "index file: section sizes do not match the header");
    GN_CUDA(cudaGetDevice(&ix->device));
    configure_mempool(ix->device);
    ix->k = k;
    ix->t = t;
    ix->span = (int)hdr[12];
    ix->keep = (uint32_t)hdr[13];
    GN_REQUIRE(ix->span >= k && ix->span <= 32 && __builtin_popcount(ix->keep) == k &&
                   (ix->span == 32 || (ix->keep >> ix->span) == 0),
               GN_EINVAL, "index file: bad seed shape");
    ix->n_seqs = (uint32_t)ns;
    ix->n_bases = n;
    ix->n_postings = np;
    ix->max_seq_len = (uint32_t)hdr[7];
    ix->seq_start_h.resize(ns + 1);
    read_all(f, ix->seq_start_h.data(), sizeof(uint64_t) * (ns + 1));
    GN_REQUIRE(ix->seq_start_h[0] == 0 && ix->seq_start_h[ns] == n, GN_EINVAL, "index file: bad sequence starts");
    for (uint64_t i = 0; i < ns; ++i)
        GN_REQUIRE(ix->seq_start_h[i + 1] >= ix->seq_start_h[i], GN_EINVAL, "index file: bad sequence starts");
    alloc_fixed(ix, ns, n, nbk - 1, nlut);
    alloc_occurrences(ix);
    ix->bank.n = n;
    GN_CUDA(cudaMemcpy(ix->seq_start_d, ix->seq_start_h.data(), 8 * (ns + 1), cudaMemcpyHostToDevice));
    std::vector<uint8_t> buf(IX_CHUNK);
    read_device(f, ix->bank.pk, 4 * npk, buf);
    read_device(f, ix->bank.nb, 4 * nnb, buf);
    read_device(f, ix->off_d, 8 * nbk, buf);
    read_device(f, ix->post_d, 4 * np, buf);
    read_device(f, ix->seq_lut_d, 4 * nlut, buf);
    uint64_t last = 0;
    GN_CUDA(cudaMemcpy(&last, ix->off_d + (nbk - 1), 8, cudaMemcpyDeviceToHost));
    GN_REQUIRE(last == np, GN_EINVAL, "index file: bucket starts do not end at the occurrence count");
    // the signatures are not in the file: they follow from the occurrences and the bank (the
    // lookup table, unchecked file content, is not walked here)
    if (np && ix->sig_d) {
        GN_LAUNCH("k_occurrences", np, 0,
                  k_occurrences<<<(unsigned)((np + 255) / 256), 256>>>(nullptr, np, ix->post_d, ix->sig_d, n, ix->bank.pk,
                                                                     ix->bank.nb, SeqMap{ix->seq_start_d, nullptr, ix->n_seqs},
                                                                     seed_shape(ix), ix->t,
                                                                     sig_kind(ix->k, ix->span, ix->t), false));
        GN_CUDA(cudaDeviceSynchronize());
    }
}

}  // namespace gn
