// gn_team.cuh - sums, maxima and sorts of a warp's or a block's threads (included by gn_search.cu)
namespace gn {

// T threads that work together, a warp or the block, on up to T * E things: thread t has the
// things t * E .. t * E + E - 1.
template <int T, int E>
struct Team {
    static constexpr bool WARP = T == 32;
    static __device__ __forceinline__ uint32_t tid() { return WARP ? threadIdx.x & 31 : threadIdx.x; }
    static __device__ __forceinline__ void sync() {
        if (WARP) __syncwarp();
        else __syncthreads();
    }
    // tmp: 32 words a team
    static __device__ __forceinline__ uint32_t excl_sum(uint32_t v, uint64_t *tmp, uint32_t &total) {
        if (!WARP) return block_excl_scan(v, reinterpret_cast<uint32_t *>(tmp), total);
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (tid() >= o) x += y;
        }
        total = __shfl_sync(0xffffffffu, x, 31);
        return x - v;
    }
    static __device__ __forceinline__ uint64_t warp_max_scan(uint64_t x) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x = max(x, y);
        }
        return x;
    }
    // largest of the values of the threads before this one (0: none)
    static __device__ __forceinline__ uint64_t excl_max(uint64_t v, uint64_t *tmp) {
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        const uint64_t x = warp_max_scan(v);
        uint64_t before = __shfl_up_sync(0xffffffffu, x, 1);
        if (lane == 0) before = 0;
        if (WARP) return before;
        if (lane == 31) tmp[wid] = x;
        __syncthreads();
        const uint64_t w = warp_max_scan(lane < T / 32 ? tmp[lane] : 0ull);
        const uint64_t pre = __shfl_sync(0xffffffffu, w, wid > 0 ? wid - 1 : 0);
        __syncthreads();  // tmp is reused by the next call
        return wid > 0 ? max(before, pre) : before;
    }
    // Bitonic sort of P keys, E a thread (P a multiple of 32 E, a power of two; threads from P / E
    // on only synchronise).  Exchanges within a thread cost no memory access, within a warp two
    // shuffles a key; only those between warps go through shared memory (ex: P keys): 6 of 55 stages
    // at 1,024 keys.  Sorted in shared memory alone, 2,048 keys took
    // 33,000 cycles a block, bound by shared-memory wavefronts (two-way bank conflicts, 8 wavefronts
    // for 32 keys and stage), and the merge of 103,000 HSPs 104 instead of 74 us.
    template <class Less>
    static __device__ __forceinline__ void sort(uint64_t (&r)[E], uint64_t *ex, uint32_t P, Less less) {
        const uint32_t t = tid(), A = P / E;
        const bool on = t < A;
        if (on) {
#pragma unroll
            for (int k = 2; k <= E; k <<= 1)
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if ((e & j) == 0) order(r[e], r[e + j], k < E ? (e & k) == 0 : (t & 1) == 0, less);
        }
        for (uint32_t k = 2; k <= A; k <<= 1) {  // sorted runs of k threads
            const bool up = (t & k) == 0 || k == A;
            uint32_t j = k >> 1;
            for (; j >= 32; j >>= 1) {
                if (on)
#pragma unroll
                    for (int e = 0; e < E; ++e) ex[e * A + t] = r[e];
                sync();
                if (on)
#pragma unroll
                    for (int e = 0; e < E; ++e) keep(r[e], ex[e * A + (t ^ j)], up == ((t & j) == 0), less);
                sync();
            }
            if (!on) continue;
            for (; j > 0; j >>= 1)
#pragma unroll
                for (int e = 0; e < E; ++e) keep(r[e], __shfl_xor_sync(0xffffffffu, r[e], j), up == ((t & j) == 0), less);
#pragma unroll
            for (int i = E >> 1; i > 0; i >>= 1)
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if ((e & i) == 0) order(r[e], r[e + i], up, less);
        }
    }
    // least power of two that sort takes, from n on
    static __device__ __forceinline__ uint32_t padded(uint32_t n) {
        uint32_t P = 32 * E;
        while (P < n) P <<= 1;
        return P;
    }

  private:
    template <class Less>
    static __device__ __forceinline__ void order(uint64_t &a, uint64_t &b, bool up, Less less) {
        const uint64_t x = a, y = b;
        const bool swap = less(y, x) == up;
        a = swap ? y : x;
        b = swap ? x : y;
    }
    template <class Less>
    static __device__ __forceinline__ void keep(uint64_t &a, uint64_t other, bool smaller, Less less) {
        if (less(other, a) == smaller) a = other;
    }
};

struct KeyLess {
    __device__ __forceinline__ bool operator()(uint64_t a, uint64_t b) const { return a < b; }
};

}  // namespace gn
