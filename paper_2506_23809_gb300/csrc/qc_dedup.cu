// qc_dedup.cu -- the sample table of Sec. IV-C-4 built on the device: a raw stream of
// sampled bitstrings (any order, repeats) becomes the ascending unique keys with their
// multiplicities, the input that qc_eloc_eval takes.  The paper names the construction of
// this lookup table as what limits scaling once the unique-sample count grows.
//
// A sampler's stream repeats its keys many times, so the keys are counted before they are
// sorted, and only the distinct ones are sorted:
//   KA count    one pass over the raw stream into a hash table of the distinct keys (a slot
//               holds the raw position of its key's first comer and a count).  Each CTA counts
//               what it sees in a table of its own in shared memory first, so a key that makes
//               up a sixth of the stream costs the chip 152 global atomics, not 10^6.
//   KL list     the distinct keys, unsorted
//   KT tiles    tiles of 2,048 keys sorted in shared memory
//   KM merge    runs merged in pairs until one is left (the run lengths and the number of
//               passes that do something follow the device's count of distinct keys)
//   KE emit     the sorted keys with their counts, looked up in the hash table
// A stream with too many distinct keys for the hash table (by a sample of it taken while the table is
// cleared, KS; or else a probe sequence longer than kProbeMax ends the counting), or a short one, is
// sorted whole instead by the same KT and KM,
// and its runs counted:
//   KH heads    heads of runs per tile; their prefix sum; KR runs: the head keys and their
//               positions; KC: multiplicities as differences of positions
// Every kernel of both ways is launched; the device's flag decides which of them do anything.  KA and KM
// are launched early (wait_previous): KA clears its shared memory while the global table is cleared,
// and the merge passes that a stream does not need follow each other closely, which pays for KS.
//
// Keys of up to 64 orbitals are sorted as one word.  Traffic: 16 B per raw key, then 16 (or 32)
// B per distinct key and merge pass, in place of 48 B per raw key and 8-bit digit of a radix sort of
// the whole stream.  10^7 raw keys at N=52: 1.02 ms with that sort (this stream), now 0.18 (counting
// 78 us, listing 10, tiles 16, six merges 48, the rest launches and the clearing); of 5*10^5 distinct
// 1.40 -> 0.36.  Sorted whole: 10^5 raw keys 0.42 -> 0.07 ms; 10^7 of 5*10^6 distinct 1.87 -> 0.96, and at
// N=28, four digits, 1.19 -> 0.96; 3*10^6 of 3*10^6 at N=28 0.41 -> 0.31 (0.49 when the counting had to
// fail first).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "qc_eloc.h"
#include "qc_internal.h"

namespace {

constexpr int kScanBlock = 1024;      // threads of a scan block
constexpr int kScanItems = 4;         // items per thread of a scan block
constexpr int kScanSeg = kScanBlock * kScanItems;

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kTile = kSortThreads * kSortItems;  // keys of a tile
// Shorter streams are sorted whole: the hash table's fixed cost (clearing and listing it) is more
// than the merge passes it saves (131,072 raw keys: 84 us whole, 108 us counted).
constexpr long long kCountMinRaw = 1 << 19;
constexpr unsigned kMaxSlots = 1u << 21;    // hash table: 24 MB, L2-resident
constexpr unsigned kProbeMax = 64;          // reached near 0.45 of the slots filled
constexpr int kCountThreads = 1024;

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

struct Ctrl {
    unsigned bad;    // a key had a bit >= n_orb
    unsigned full;   // the hash table is full (or not used): sort the whole stream
    unsigned m;      // distinct keys listed
    unsigned runs;   // distinct keys of the whole stream, sorted (0: it was not)
};

// bufA and bufB: the sort's two buffers when the whole stream is sorted.  When its distinct keys are
// counted, both are in bufA's space (its halves) and the hash table takes that of bufB and heads.
struct Layout {
    size_t bufA, bufB, heads, sums, ctrl, total;
    unsigned slots;  // hash slots (0: not used), 8 + 4 bytes each
};

Layout layout(long long n) {
    const size_t k = static_cast<size_t>(std::max<long long>(n, 1));
    Layout L{};
    size_t off = 0;
    L.bufA = off; off = align256(off + k * 16);
    L.bufB = off; off = align256(off + k * 16);
    L.heads = off; off = align256(off + (k + 1) * 8);
    L.sums = off; off = align256(off + (k / kTile + 2) * 4 + 4096);
    L.ctrl = off; off = align256(off + sizeof(Ctrl));
    L.total = off;
    if (n >= kCountMinRaw) {
        L.slots = kMaxSlots;
        while (L.slots > 2ULL * static_cast<unsigned long long>(n)) L.slots >>= 1;  // 12 B a slot, 24 B a raw key
    }
    return L;
}

// A sort key: one word for up to 64 orbitals, else two.
struct Key1 {
    unsigned long long v;
    __device__ static Key1 of(ulonglong2 k) { return Key1{k.x}; }
    __device__ static Key1 max() { return Key1{~0ULL}; }
    __device__ ulonglong2 wide() const { return make_ulonglong2(v, 0ULL); }
    __device__ bool less(const Key1& o) const { return v < o.v; }
    __device__ bool same(const Key1& o) const { return v == o.v; }
    __device__ unsigned long long mix() const { return v; }
};
struct alignas(16) Key2 {
    unsigned long long lo, hi;
    __device__ static Key2 of(ulonglong2 k) { return Key2{k.x, k.y}; }
    __device__ static Key2 max() { return Key2{~0ULL, ~0ULL}; }
    __device__ ulonglong2 wide() const { return make_ulonglong2(lo, hi); }
    __device__ bool less(const Key2& o) const { return hi < o.hi || (hi == o.hi && lo < o.lo); }
    __device__ bool same(const Key2& o) const { return lo == o.lo && hi == o.hi; }
    __device__ unsigned long long mix() const { return lo ^ (hi * 0x9E3779B97F4A7C15ULL); }
};

// Two multiply-xorshift rounds (the finalizer of splitmix64, Vigna).
template <typename K>
__device__ __forceinline__ unsigned long long key_hash(const K& k) {
    unsigned long long z = k.mix();
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

// ------------------------------------------------------------------------------------
// KA: counting
// ------------------------------------------------------------------------------------
// Add c to the count of key k (raw position i) in the global table.  A slot is written once, by
// compare-and-swap: the high half of its key's hash and the raw position (plus one) of the key.
// The raw stream does not change, so what a reader compares is always complete.
template <typename K>
__device__ __forceinline__ bool slot_holds(unsigned long long e, const ulonglong2* __restrict__ raw, const K& k,
                                           unsigned long long h) {
    return (e >> 32) == (h >> 32) && K::of(raw[static_cast<unsigned>(e) - 1u]).same(k);
}
// DIRECT: every key is its own slot number (no more orbitals than slot bits), so the table never fills.
template <bool DIRECT, typename K>
__device__ __forceinline__ unsigned first_slot(const K& k, unsigned long long h, unsigned mask) {
    return (DIRECT ? static_cast<unsigned>(k.wide().x) : static_cast<unsigned>(h >> 13)) & mask;
}
template <bool DIRECT, typename K>
__device__ __forceinline__ void count_global(const ulonglong2* __restrict__ raw, const K& k, unsigned i, unsigned c,
                                             unsigned long long h, unsigned long long* slot, unsigned* count,
                                             unsigned mask, Ctrl* ctrl) {
    unsigned s = first_slot<DIRECT>(k, h, mask);
    for (unsigned it = 0; it < kProbeMax; ++it) {
        unsigned long long e = __ldcg(slot + s);
        if (e == 0ULL) e = atomicCAS(slot + s, 0ULL, (h >> 32 << 32) | (i + 1u));
        if (e == 0ULL || slot_holds(e, raw, k, h)) {
            atomicAdd(count + s, c);
            return;
        }
        s = (s + 1u) & mask;
    }
    atomicOr(&ctrl->full, 1u);
}

// Shared-memory table of a CTA, in buckets of two slots: a slot's tag goes 0 (free) -> 1 (being
// written) -> hash | 2; its key and raw position are valid once the tag is a hash.  A key that finds
// neither slot its own goes to its warp's queue and is counted in the global table when 32 have
// come together: a step in which some lanes walk L2 and the others wait costs the whole warp two
// microseconds.  The bucket is read with one load and the common case (the key is there) has one
// branch; claiming a free slot is a second step that most warps skip.  10^7 raw keys of 10^5
// distinct: 206 us with four single-slot probes in a loop and no queue, 144 with the queue (269
// instructions per 32 keys), 78 us so (aggregating equal slots of a warp with __match_any_sync: 90).
template <typename K>
struct CountTable {
    static constexpr int slots = sizeof(K) == 8 ? 8192 : 4096;
    static constexpr int queue = 64;  // per warp: up to 31 waiting and 32 new
    static constexpr size_t bytes = slots * (sizeof(K) + 12) + kCountThreads / 32 * queue * 4;
};

template <bool DIRECT, typename K>
__global__ void __launch_bounds__(kCountThreads, 1) dedup_count_kernel(const ulonglong2* raw, long long n,
                                                                      ulonglong2 high, unsigned long long* slot,
                                                                      unsigned* count, unsigned mask, Ctrl* ctrl) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int S = CountTable<K>::slots;
    K* keys = reinterpret_cast<K*>(sm);
    unsigned* tag = reinterpret_cast<unsigned*>(sm + S * sizeof(K));
    unsigned* cnt = tag + S;
    unsigned* pos = cnt + S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned* queue = pos + S + warp * CountTable<K>::queue;
    for (int t = threadIdx.x; t < S; t += kCountThreads) tag[t] = cnt[t] = 0u;
    qc::wait_previous();
    if (__syncthreads_or(__ldcg(&ctrl->full) != 0u)) return;  // too many distinct keys
    bool bad = false;
    int qn = 0;
    auto flush = [&](int m) {  // the first m queued raw positions to the global table
        if (lane < m) {
            const unsigned i = queue[lane];
            const K k = K::of(raw[i]);
            count_global<DIRECT>(raw, k, i, 1u, key_hash(k), slot, count, mask, ctrl);
        }
        __syncwarp();
        const unsigned rest = lane < qn - m ? queue[m + lane] : 0u;
        __syncwarp();
        if (lane < qn - m) queue[lane] = rest;
        __syncwarp();
        qn -= m;
    };
    constexpr int kLoads = 4;  // raw keys in flight per thread
    const long long step = static_cast<long long>(gridDim.x) * kCountThreads * kLoads;
    for (long long b = (static_cast<long long>(blockIdx.x) * kCountThreads + 32 * warp) * kLoads; b < n; b += step) {
        ulonglong2 r[kLoads];
#pragma unroll
        for (int l = 0; l < kLoads; ++l)
            if (b + 32 * l + lane < n) r[l] = __ldg(raw + b + 32 * l + lane);
        if (__any_sync(0xffffffffu, *reinterpret_cast<volatile unsigned*>(&ctrl->full) != 0u)) break;
#pragma unroll
        for (int l = 0; l < kLoads; ++l) {
            const long long i = b + 32 * l + lane;
            bool miss = i < n;
            bad = bad || (miss && ((r[l].x & high.x) != 0ULL || (r[l].y & high.y) != 0ULL));
            const K k = K::of(r[l]);
            const unsigned long long h = key_hash(k);
            const unsigned mine = static_cast<unsigned>(h >> 32) | 2u;
            const unsigned s0 = static_cast<unsigned>(h) & (S - 2);
            const volatile unsigned* vt = tag + s0;
            const unsigned t0 = vt[0], t1 = vt[1];
            __threadfence_block();
            if (miss && (t0 == mine || t1 == mine)) {
                const unsigned s = t0 == mine ? s0 : s0 + 1u;
                if (keys[s].same(k)) {
                    atomicAdd(cnt + s, 1u);
                    miss = false;
                }
            }
            if (__any_sync(0xffffffffu, miss && (t0 == 0u || t1 == 0u))) {
                if (miss && (t0 == 0u || t1 == 0u)) {
                    const unsigned s = t0 == 0u ? s0 : s0 + 1u;
                    if (atomicCAS(tag + s, 0u, 1u) == 0u) {
                        keys[s] = k;
                        pos[s] = static_cast<unsigned>(i);
                        atomicAdd(cnt + s, 1u);
                        __threadfence_block();
                        *reinterpret_cast<volatile unsigned*>(tag + s) = mine;
                        miss = false;
                    }
                }
                __syncwarp();
            }
            const unsigned m = __ballot_sync(0xffffffffu, miss);
            if (miss) queue[qn + __popc(m & ((1u << lane) - 1u))] = static_cast<unsigned>(i);
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32) flush(32);
        }
    }
    if (qn > 0) flush(qn);
    if (bad) atomicOr(&ctrl->bad, 1u);
    __syncthreads();
    for (int t = threadIdx.x; t < S; t += kCountThreads)
        if (tag[t] >= 2u)
            count_global<DIRECT>(raw, keys[t], pos[t], cnt[t], key_hash(keys[t]), slot, count, mask, ctrl);
}

// KL: the distinct keys into `list`, in any order (they are sorted next and are distinct).  (Listing
// a key where it claims its slot costs the count an atomic on one address per distinct key: 158 ->
// 297 us at 4*10^5.)
constexpr int kListSlots = 4;  // slots a thread
template <typename K>
__global__ void __launch_bounds__(1024) dedup_list_kernel(const ulonglong2* __restrict__ raw,
                                                          const unsigned long long* __restrict__ slot,
                                                          K* __restrict__ list, Ctrl* ctrl) {
    __shared__ unsigned warp_n[32];
    __shared__ unsigned base;
    if (ctrl->full != 0u) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long e[kListSlots];
    unsigned have[kListSlots], before[kListSlots], n = 0;
#pragma unroll
    for (int t = 0; t < kListSlots; ++t) e[t] = __ldcg(slot + (blockIdx.x * kListSlots + t) * 1024u + threadIdx.x);
#pragma unroll
    for (int t = 0; t < kListSlots; ++t) {
        have[t] = __ballot_sync(0xffffffffu, e[t] != 0ULL);
        before[t] = n;
        n += __popc(have[t]);
    }
    if (lane == 0) warp_n[warp] = n;
    __syncthreads();
    if (warp == 0) {
        const unsigned v = warp_n[lane];
        unsigned x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        warp_n[lane] = x - v;
        if (lane == 31) base = x != 0u ? atomicAdd(&ctrl->m, x) : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kListSlots; ++t)
        if (e[t] != 0ULL)
            list[base + warp_n[warp] + before[t] + __popc(have[t] & ((1u << lane) - 1u))] =
                K::of(raw[static_cast<unsigned>(e[t]) - 1u]);
}

// Whether the whole stream is sorted: the hash table is not used or filled up, or holds more keys
// than half of bufA does.
template <typename K>
__device__ __forceinline__ bool sort_whole(const Ctrl* ctrl, long long n) {
    return ctrl->full != 0u || static_cast<long long>(ctrl->m) * static_cast<long long>(sizeof(K)) > 8 * n;
}

// ------------------------------------------------------------------------------------
// KT, KM: sort
// ------------------------------------------------------------------------------------
// A tile in shared memory: one key of padding after eight, so that threads reading or writing
// eight consecutive keys each hit different banks.
template <typename K>
struct Tile {
    K* sh;
    int at;
    __device__ K& operator[](int i) const { return sh[at + i + ((at + i) >> 3)]; }
};
constexpr int kTilePadded = kTile + kTile / 8;

// Keys a[0, na) before output position d of the merge of a and b (ties from a): the smallest i
// with a[i] > b[d - 1 - i], by bisection.
template <typename K>
__device__ __forceinline__ int merge_split(Tile<K> a, int na, Tile<K> b, int nb, int d) {
    int lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (b[d - 1 - mid].less(a[mid])) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// kSortItems outputs of the merge of a[i, na) and b[j, nb) into registers.
template <typename K>
__device__ __forceinline__ void merge_items(Tile<K> a, int i, int na, Tile<K> b, int j, int nb, K (&out)[kSortItems]) {
    K ka = i < na ? a[i] : K::max(), kb = j < nb ? b[j] : K::max();
#pragma unroll
    for (int t = 0; t < kSortItems; ++t) {
        const bool from_b = i >= na || (j < nb && kb.less(ka));
        out[t] = from_b ? kb : ka;
        if (from_b) {
            ++j;
            kb = j < nb ? b[j] : K::max();
        } else {
            ++i;
            ka = i < na ? a[i] : K::max();
        }
    }
}

// The block's keys from registers (8 consecutive ones a thread) to global memory, coalesced.
template <typename K>
__device__ __forceinline__ void store_tile(Tile<K> sh, const K (&v)[kSortItems], K* __restrict__ out, long long at, int n) {
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kSortItems; ++t) sh[threadIdx.x * kSortItems + t] = v[t];
    __syncthreads();
    for (int t = threadIdx.x; t < n; t += kSortThreads) out[at + t] = sh[t];
}

// KT: tiles of kTile keys of the list (or, whole, of the raw stream) sorted into `out`: eight
// keys a thread by an odd-even network, then merges of 8, 16, .. 1,024 keys in shared memory.
// `list` may be `out`: a tile is read whole before it is written.
template <typename K>
__global__ void __launch_bounds__(kSortThreads) dedup_tile_kernel(const ulonglong2* __restrict__ raw, long long n,
                                                                  const K* list, K* out, ulonglong2 high, Ctrl* ctrl) {
    __shared__ K tile[kTilePadded];
    const Tile<K> sh{tile, 0};
    const bool whole = sort_whole<K>(ctrl, n);
    const long long m = whole ? n : static_cast<long long>(ctrl->m);
    bool bad = false;
    for (long long at = static_cast<long long>(blockIdx.x) * kTile; at < m;
         at += static_cast<long long>(gridDim.x) * kTile) {
        const int have = m - at < kTile ? static_cast<int>(m - at) : kTile;
        __syncthreads();
        for (int t = threadIdx.x; t < kTile; t += kSortThreads) {
            K k = K::max();  // past the end: the largest key stays there
            if (t < have) {
                if (whole) {
                    const ulonglong2 r = raw[at + t];
                    bad = bad || (r.x & high.x) != 0ULL || (r.y & high.y) != 0ULL;
                    k = K::of(r);
                } else {
                    k = list[at + t];
                }
            }
            sh[t] = k;
        }
        __syncthreads();
        K v[kSortItems];
#pragma unroll
        for (int t = 0; t < kSortItems; ++t) v[t] = sh[threadIdx.x * kSortItems + t];
#pragma unroll
        for (int round = 0; round < kSortItems; ++round)
#pragma unroll
            for (int t = round & 1; t + 1 < kSortItems; t += 2)
                if (v[t + 1].less(v[t])) {
                    const K x = v[t];
                    v[t] = v[t + 1];
                    v[t + 1] = x;
                }
        for (int run = kSortItems; run < kTile; run *= 2) {
            __syncthreads();
#pragma unroll
            for (int t = 0; t < kSortItems; ++t) sh[threadIdx.x * kSortItems + t] = v[t];
            __syncthreads();
            const int p = threadIdx.x * kSortItems, a0 = p / (2 * run) * (2 * run), d = p - a0;
            const Tile<K> a{tile, a0}, b{tile, a0 + run};
            const int i = merge_split(a, run, b, run, d);
            merge_items(a, i, run, b, d - i, run, v);
        }
        store_tile(sh, v, out, at, have);
    }
    if (bad) atomicOr(&ctrl->bad, 1u);
}

// The split of output position d between the runs a[0, na) and b[0, nb) in global memory, by the
// 32 lanes of a warp: each step cuts the range to a 33rd, so a run of 10^6 keys takes four
// dependent loads instead of twenty.
template <typename K>
__device__ __forceinline__ long long merge_split_warp(const K* a, long long na, const K* b,
                                                      long long nb, long long d, int lane) {
    long long lo = d > nb ? d - nb : 0, hi = d < na ? d : na;  // the answer lies in [lo, hi]
    while (lo < hi) {
        const long long len = hi - lo;
        // lane's probe in [lo, hi): ascending with the lane
        const long long mid = lo + (len < 32 ? (lane < len ? lane : len - 1) : len * (lane + 1) / 33);
        const bool after = !b[d - 1 - mid].less(a[mid]);  // the answer is beyond mid
        const unsigned m = __ballot_sync(0xffffffffu, after);
        // probes are ascending and `after` is true up to the answer: count the leading ones
        const int c = m == 0xffffffffu ? 32 : __ffs(~m) - 1;
        const long long below = __shfl_sync(0xffffffffu, mid, c > 0 ? c - 1 : 0);
        const long long above = __shfl_sync(0xffffffffu, mid, c < 32 ? c : 31);
        if (c > 0) lo = below + 1;
        if (c < 32) hi = above;
    }
    return lo;
}

// KM: one merge pass: runs of `run` keys in pairs, from A to the other buffer (B, or for the listed
// keys half) or, odd, back; kTile outputs a block and step.  Nothing is left to do once a run
// holds every key.
template <typename K>
__global__ void __launch_bounds__(kSortThreads) dedup_merge_kernel(K* A, K* B, K* half, bool odd, long long n,
                                                                   long long run, const Ctrl* ctrl) {
    __shared__ K tile[kTilePadded];
    __shared__ long long split[2];
    const Tile<K> sh{tile, 0};
    qc::wait_previous();
    const bool whole = sort_whole<K>(ctrl, n);
    const long long m = whole ? n : static_cast<long long>(ctrl->m);
    if (run >= m) {  // (a pass that merges lets the next one start by ending: earlier, 10^7 keys take 14% longer)
        qc::let_next_start();
        return;
    }
    K* other = whole ? B : half;
    const K* in = odd ? other : A;
    K* out = odd ? A : other;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long at = static_cast<long long>(blockIdx.x) * kTile; at < m;
         at += static_cast<long long>(gridDim.x) * kTile) {
        const long long a0 = at / (2 * run) * (2 * run);
        const long long na = m - a0 < run ? m - a0 : run, nb = m - a0 - na < run ? m - a0 - na : run;
        const long long d0 = at - a0, d1 = d0 + kTile < na + nb ? d0 + kTile : na + nb;
        const K* a = in + a0;
        const K* b = a + na;
        if (warp < 2) {
            const long long i = merge_split_warp(a, na, b, nb, warp == 0 ? d0 : d1, lane);
            if (lane == 0) split[warp] = i;
        }
        __syncthreads();
        const long long i0 = split[0], i1 = split[1], j0 = d0 - i0;
        const int ca = static_cast<int>(i1 - i0), c = static_cast<int>(d1 - d0), cb = c - ca;
        for (int t = threadIdx.x; t < c; t += kSortThreads) sh[t] = t < ca ? a[i0 + t] : b[j0 + (t - ca)];
        __syncthreads();
        const int d = static_cast<int>(threadIdx.x) * kSortItems < c ? static_cast<int>(threadIdx.x) * kSortItems : c;
        const Tile<K> sb{tile, ca};
        const int i = merge_split(sh, ca, sb, cb, d);
        K v[kSortItems];
        merge_items(sh, i, ca, sb, d - i, cb, v);
        store_tile(sh, v, out, at, c);
        __syncthreads();
    }
}

// The buffer that holds the sorted keys: KT leaves them in A, every merge pass that did something
// swaps the two.
template <typename K>
__device__ __forceinline__ const K* sorted_in(const K* A, const K* B, long long m) {
    int passes = 0;
    for (long long run = kTile; run < m; run *= 2) ++passes;
    return (passes & 1) ? B : A;
}

// KE: the distinct keys with their counts.
template <bool DIRECT, typename K>
__global__ void __launch_bounds__(256) dedup_emit_kernel(const ulonglong2* __restrict__ raw, long long n,
                                                         const K* __restrict__ A, const K* __restrict__ half,
                                                         const unsigned long long* __restrict__ slot,
                                                         const unsigned* __restrict__ count, unsigned mask,
                                                         ulonglong2* __restrict__ keys_out,
                                                         long long* __restrict__ counts_out,
                                                         long long* __restrict__ n_unique, const Ctrl* ctrl) {
    if (sort_whole<K>(ctrl, n)) return;
    const long long m = ctrl->m;
    const K* sorted = sorted_in(A, half, m);
    for (long long j = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; j < m;
         j += static_cast<long long>(gridDim.x) * blockDim.x) {
        const K k = sorted[j];
        const unsigned long long h = key_hash(k);
        unsigned s = first_slot<DIRECT>(k, h, mask);
        for (unsigned it = 0; it < kProbeMax; ++it) {  // every listed key was placed within kProbeMax
            const unsigned long long e = slot[s];
            if (e == 0ULL || slot_holds(e, raw, k, h)) break;
            s = (s + 1u) & mask;
        }
        keys_out[j] = k.wide();
        counts_out[j] = count[s];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_unique = ctrl->bad != 0u ? -1 : m;
}

// KH: heads of runs per tile of the sorted stream.
template <typename K>
__device__ __forceinline__ bool run_head(const K* __restrict__ k, long long i) {
    return i == 0 || !k[i].same(k[i - 1]);
}
template <typename K>
__global__ void __launch_bounds__(kSortThreads) dedup_heads_kernel(const K* __restrict__ A, const K* __restrict__ B,
                                                                   long long n, unsigned* __restrict__ heads_of,
                                                                   const Ctrl* ctrl) {
    if (!sort_whole<K>(ctrl, n)) return;
    const K* k = sorted_in(A, B, n);
    __shared__ unsigned total;
    for (long long at = static_cast<long long>(blockIdx.x) * kTile; at < n;
         at += static_cast<long long>(gridDim.x) * kTile) {
        __syncthreads();
        if (threadIdx.x == 0) total = 0u;
        __syncthreads();
        unsigned c = 0;
        for (int t = threadIdx.x; t < kTile && at + t < n; t += kSortThreads) c += run_head(k, at + t) ? 1u : 0u;
        c = __reduce_add_sync(0xffffffffu, c);
        if ((threadIdx.x & 31) == 0) atomicAdd(&total, c);
        __syncthreads();
        if (threadIdx.x == 0) heads_of[at / kTile] = total;
    }
}

// exclusive scan of a u32 array in place: segment sums, a scan of the sums, segment scans
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned* sh, unsigned& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned s = lane < (blockDim.x >> 5) ? sh[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh[lane] = s;  // inclusive warp totals
    }
    __syncthreads();
    total = sh[(blockDim.x >> 5) - 1];
    const unsigned before = warp > 0 ? sh[warp - 1] : 0u;
    __syncthreads();
    return before + x - v;
}

__global__ void __launch_bounds__(kScanBlock) scan_sums_kernel(const unsigned* a, long long n,
                                                               unsigned* sums) {
    __shared__ unsigned sh[32];
    qc::let_next_start();
    qc::wait_previous();
    const long long base = static_cast<long long>(blockIdx.x) * kScanSeg + threadIdx.x * kScanItems;
    unsigned v = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) v += a[base + k];
    unsigned total;
    block_exclusive_scan(v, sh, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__device__ __forceinline__ void scan_top(unsigned* sums, long long m) {
    __shared__ unsigned sh[32];
    __shared__ unsigned carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (long long b = 0; b < m; b += kScanBlock) {
        const long long i = b + threadIdx.x;
        const unsigned v = i < m ? sums[i] : 0u;
        unsigned total;
        const unsigned ex = block_exclusive_scan(v, sh, total);
        if (i < m) sums[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[m] = carry;
}

__global__ void __launch_bounds__(kScanBlock) scan_top_kernel(unsigned* sums, long long m) {
    qc::let_next_start();
    qc::wait_previous();
    scan_top(sums, m);
}
template <typename K>
__global__ void __launch_bounds__(kScanBlock) dedup_scan_kernel(unsigned* __restrict__ sums, long long m, long long n,
                                                                const Ctrl* ctrl) {
    if (sort_whole<K>(ctrl, n)) scan_top(sums, m);
}

__global__ void __launch_bounds__(kScanBlock) scan_down_kernel(const unsigned* a, unsigned* out, long long n,
                                                               const unsigned* sums) {
    __shared__ unsigned sh[32];
    qc::let_next_start();
    qc::wait_previous();
    const long long base = static_cast<long long>(blockIdx.x) * kScanSeg + threadIdx.x * kScanItems;
    unsigned v[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < n ? a[base + k] : 0u;
        s += v[k];
    }
    unsigned total;
    unsigned run = sums[blockIdx.x] + block_exclusive_scan(s, sh, total);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) {
            out[base + k] = run;
            run += v[k];
        }
}



// KR: each head writes its key and its position at its rank.
template <typename K>
__global__ void __launch_bounds__(kSortThreads) dedup_runs_kernel(const K* __restrict__ A, const K* __restrict__ B,
                                                                  long long n, const unsigned* __restrict__ before,
                                                                  long long tiles, ulonglong2* __restrict__ keys_out,
                                                                  long long* __restrict__ heads,
                                                                  long long* __restrict__ n_unique, Ctrl* ctrl) {
    if (!sort_whole<K>(ctrl, n)) return;
    const K* k = sorted_in(A, B, n);
    __shared__ unsigned warp_n[kSortThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long at = static_cast<long long>(blockIdx.x) * kTile; at < n;
         at += static_cast<long long>(gridDim.x) * kTile) {
        unsigned base = before[at / kTile];
        for (int t0 = 0; t0 < kTile && at + t0 < n; t0 += kSortThreads) {
            const long long i = at + t0 + threadIdx.x;
            const bool head = i < n && run_head(k, i);
            const unsigned m = __ballot_sync(0xffffffffu, head);
            __syncthreads();
            if (lane == 0) warp_n[warp] = __popc(m);
            __syncthreads();
            unsigned mine = base;
            for (int w = 0; w < kSortThreads / 32; ++w) {
                if (w < warp) mine += warp_n[w];
                base += warp_n[w];
            }
            if (head) {
                const unsigned j = mine + __popc(m & ((1u << lane) - 1u));
                keys_out[j] = k[i].wide();
                heads[j] = i;
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned u = before[tiles];
        heads[u] = n;
        ctrl->runs = u;
        *n_unique = ctrl->bad != 0u ? -1 : static_cast<long long>(u);
    }
}

// KC: multiplicities = differences of consecutive head positions
__global__ void __launch_bounds__(256) dedup_counts_kernel(const long long* __restrict__ heads,
                                                           long long* __restrict__ counts_out, const Ctrl* ctrl) {
    const long long u = ctrl->runs;
    for (long long j = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; j < u;
         j += static_cast<long long>(gridDim.x) * blockDim.x)
        counts_out[j] = heads[j + 1] - heads[j];
}

// The stream is sorted whole from the start.
__global__ void dedup_whole_kernel(Ctrl* ctrl) { *ctrl = Ctrl{0u, 1u, 0u, 0u}; }

// KS: clears the hash table (all clusters but the first) and judges by a sample (the first) whether the
// stream has too many distinct keys for it.  kSample raw keys, one from each of as many equal parts
// of the stream, are put in a table of 32-bit hashes spread over the cluster; c of them find their
// hash there.  A stream in which two random places agree with probability 1/N2 has c near
// kSample^2 / (2 N2), and at least n N2 / (n + N2) distinct keys (Cauchy-Schwarz on the
// multiplicities).  With c taken two standard deviations high, too many by that bound are too many
// indeed, and the counting, which would end half-way after some 100 us, is left out (3*10^6 raw keys of
// 1.5*10^6 distinct at N=28: 444 -> 301 us; at N=20, of 8*10^5 and counted in slots of their own, 410 ->
// 223).  By one CTA the sample took 24 us, most of it waiting for 16,384 scattered sectors; a
// cluster's is done soon after the clearing.
constexpr int kSample = 1 << 14, kSampleCluster = 8, kSampleSlots = 4096;  // slots of one CTA
template <typename K>
__global__ void __cluster_dims__(kSampleCluster, 1, 1) __launch_bounds__(1024)
    dedup_start_kernel(const ulonglong2* __restrict__ raw, long long n, uint4* __restrict__ table, long long words,
                       unsigned slots, bool direct, Ctrl* ctrl) {
    __shared__ __align__(16) unsigned seen[kSampleSlots];
    __shared__ int found;
    qc::let_next_start();
    const bool sampler = blockIdx.x < kSampleCluster && !direct;
    if (!sampler) {
        const long long first = direct ? 0 : kSampleCluster;
        for (long long i = (blockIdx.x - first) * 1024 + threadIdx.x; i < words; i += (gridDim.x - first) * 1024)
            table[i] = make_uint4(0u, 0u, 0u, 0u);
        if (blockIdx.x == 0 && threadIdx.x == 0) *ctrl = Ctrl{0u, 0u, 0u, 0u};
        return;
    }
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    constexpr int kOwn = kSample / (1024 * kSampleCluster);
    const unsigned part = static_cast<unsigned>(n / kSample);
    ulonglong2 r[kOwn];
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
        const unsigned t = (blockIdx.x * kOwn + k) * 1024u + threadIdx.x;
        const unsigned in = __umulhi((t * 0x9E3779B1u) ^ (t << 19), part);  // any place of part t
        r[k] = raw[static_cast<long long>(t) * n / kSample + in];
    }
    reinterpret_cast<uint4*>(seen)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
    static_assert(kSampleSlots == 4 * 1024, "cleared by one store a thread");
    if (threadIdx.x == 0) found = 0;
    cl.sync();
    int c = 0;
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
        const unsigned long long h = key_hash(K::of(r[k]));
        const unsigned mine = static_cast<unsigned>(h >> 32) | 1u;
        unsigned* at = cl.map_shared_rank(seen, static_cast<unsigned>(h >> 16) % kSampleCluster);
        unsigned s = static_cast<unsigned>(h) % kSampleSlots;
        for (int it = 0; it < kSampleSlots; ++it) {
            const unsigned old = atomicCAS(at + s, 0u, mine);
            if (old == mine) ++c;
            if (old == 0u || old == mine) break;
            s = (s + 1u) % kSampleSlots;
        }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c != 0) atomicAdd(cl.map_shared_rank(&found, 0), c);
    cl.sync();  // (the CTAs' tables and rank 0's count are touched no more)
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const float all = static_cast<float>(found), high = all + 2.0f * sqrtf(all) + 2.0f;
        const float n2 = 0.5f * kSample * static_cast<float>(kSample) / high, fn = static_cast<float>(n);
        const bool many = fn * n2 / (fn + n2) > 0.45f * static_cast<float>(slots);
        *ctrl = Ctrl{0u, many ? 1u : 0u, 0u, 0u};
    }
}

template <bool DIRECT, typename K>
cudaError_t dedup(const ulonglong2* raw, long long n, ulonglong2 high, ulonglong2* keys_out, long long* counts_out,
                  long long* n_unique, unsigned char* W, const Layout& L, bool count, int sms, cudaStream_t s) {
    K* A = reinterpret_cast<K*>(W + L.bufA);
    K* B = reinterpret_cast<K*>(W + L.bufB);
    long long* heads = reinterpret_cast<long long*>(W + L.heads);
    // bufA's second half, on a 16-byte boundary (bufA's own rounding to 256 bytes covers the shift)
    K* half = reinterpret_cast<K*>(W + L.bufA + (static_cast<size_t>(n) * 8 + 15) / 16 * 16);
    unsigned long long* slot = reinterpret_cast<unsigned long long*>(W + L.bufB);
    unsigned* counts = reinterpret_cast<unsigned*>(slot + L.slots);
    unsigned* sums = reinterpret_cast<unsigned*>(W + L.sums);
    Ctrl* ctrl = reinterpret_cast<Ctrl*>(W + L.ctrl);
    const unsigned mask = L.slots - 1u;
    const long long tiles = (n + kTile - 1) / kTile;
    const unsigned grid = static_cast<unsigned>(std::min<long long>(tiles, 8LL * sms));
    cudaError_t e = cudaSuccess;
    if (!count) {
        dedup_whole_kernel<<<1, 1, 0, s>>>(ctrl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && count) {
        constexpr size_t smem = CountTable<K>::bytes;
        // a CTA an SM, in whole clusters: the count's CTAs start beside them
        const unsigned clusters = static_cast<unsigned>(std::max(2, sms / kSampleCluster));
        dedup_start_kernel<K><<<clusters * kSampleCluster, 1024, 0, s>>>(
            raw, n, reinterpret_cast<uint4*>(slot), static_cast<long long>(L.slots) * 12 / 16, L.slots, DIRECT, ctrl);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(dedup_count_kernel<DIRECT, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(smem));
        if (e == cudaSuccess) {
            e = qc::launch_early(dedup_count_kernel<DIRECT, K>, dim3(static_cast<unsigned>(sms)), dim3(kCountThreads), smem, s,
                                 true, raw, n, high, slot, counts, mask, ctrl);
        }
        if (e == cudaSuccess) {
            dedup_list_kernel<K><<<L.slots / (1024 * kListSlots), 1024, 0, s>>>(raw, slot, A, ctrl);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) {
        dedup_tile_kernel<K><<<grid, kSortThreads, 0, s>>>(raw, n, A, A, high, ctrl);
        e = cudaGetLastError();
    }
    bool odd = false;
    for (long long run = kTile; run < n && e == cudaSuccess; run *= 2) {
        e = qc::launch_early(dedup_merge_kernel<K>, dim3(grid), dim3(kSortThreads), 0, s, true, A, B, half, odd, n, run, ctrl);
        odd = !odd;
    }
    if (e == cudaSuccess && count) {
        dedup_emit_kernel<DIRECT, K><<<4 * sms, 256, 0, s>>>(raw, n, A, half, slot, counts, mask, keys_out, counts_out,
                                                    n_unique, ctrl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        dedup_heads_kernel<K><<<grid, kSortThreads, 0, s>>>(A, B, n, sums, ctrl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        dedup_scan_kernel<K><<<1, kScanBlock, 0, s>>>(sums, tiles, n, ctrl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        dedup_runs_kernel<K><<<grid, kSortThreads, 0, s>>>(A, B, n, sums, tiles, keys_out, heads, n_unique, ctrl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        dedup_counts_kernel<<<8 * sms, 256, 0, s>>>(heads, counts_out, ctrl);
        e = cudaGetLastError();
    }
    return e;
}

qc_status dfail(qc_status st, const char* msg) {
    qc::set_handleless_error(msg);
    return st;
}

}  // namespace

// Exclusive prefix sum of a u32 array, in place or into another (segment sums, a scan of the
// sums, segment scans): the join index's group starts and digit offsets (qc_join.cu).
cudaError_t qc::exclusive_scan_u32(const unsigned* in, unsigned* out, long long n, unsigned* sums, cudaStream_t s) {
    const long long segs = (n + kScanSeg - 1) / kScanSeg;
    if (segs == 0) return cudaSuccess;
    const dim3 grid(static_cast<unsigned>(segs)), block(kScanBlock);
    cudaError_t e = launch_early(scan_sums_kernel, grid, block, 0, s, true, in, n, sums);
    if (e == cudaSuccess) e = launch_early(scan_top_kernel, dim3(1), block, 0, s, true, sums, segs);
    if (e == cudaSuccess) e = launch_early(scan_down_kernel, grid, block, 0, s, true, in, out, n, sums);
    return e;
}

extern "C" int64_t qc_dedup_workspace_bytes(int64_t n_raw) {
    if (n_raw < 0) return -1;
    return static_cast<int64_t>(layout(n_raw).total);
}

extern "C" qc_status qc_dedup(const uint64_t* raw, int64_t n_raw, int n_orb, uint64_t* keys_out,
                              int64_t* counts_out, int64_t* n_unique, void* work, size_t work_bytes,
                              void* stream) {
    if (n_raw < 0 || n_raw > 0x7fffffffLL || n_orb < 1 || n_orb > 128 || !n_unique)
        return dfail(QC_ERR_ARG, "qc_dedup: bad size or NULL n_unique");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n_raw == 0) {
        const cudaError_t e = cudaMemsetAsync(n_unique, 0, sizeof(int64_t), s);
        return e == cudaSuccess ? QC_OK : dfail(QC_ERR_CUDA, cudaGetErrorString(e));
    }
    if (!raw || !keys_out || !counts_out || !work)
        return dfail(QC_ERR_ARG, "qc_dedup: NULL pointer");
    auto mis = [](const void* p, unsigned a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0; };
    if (mis(raw, 16) || mis(keys_out, 16) || mis(counts_out, 8) || mis(n_unique, 8) || mis(work, 256))
        return dfail(QC_ERR_ARG, "qc_dedup: alignment (keys 16, counts 8, work 256 bytes)");
    const long long n = n_raw;
    const Layout L = layout(n);
    if (work_bytes < L.total) return dfail(QC_ERR_CAPACITY, "qc_dedup: workspace too small");
    unsigned char* W = static_cast<unsigned char*>(work);
    ulonglong2 high{};
    high.x = n_orb >= 64 ? 0ULL : ~((1ULL << n_orb) - 1ULL);
    high.y = n_orb >= 128 ? 0ULL : (n_orb <= 64 ? ~0ULL : ~((1ULL << (n_orb - 64)) - 1ULL));
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return dfail(QC_ERR_CUDA, cudaGetErrorString(e));
    // counting reads the raw keys to the end, so outputs laid over them are written by the sort of
    // the whole stream, which has read them all before it writes
    auto over = [&](const void* p, size_t bytes) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(raw), b = reinterpret_cast<uintptr_t>(p);
        return b < a + static_cast<size_t>(n) * 16 && a < b + bytes;
    };
    const size_t un = static_cast<size_t>(n);
    const bool count = L.slots > 0 && !over(keys_out, un * 16) && !over(counts_out, un * 8) && !over(n_unique, 8);
    const ulonglong2* r = reinterpret_cast<const ulonglong2*>(raw);
    ulonglong2* ko = reinterpret_cast<ulonglong2*>(keys_out);
    long long* co = reinterpret_cast<long long*>(counts_out);
    long long* nu = reinterpret_cast<long long*>(n_unique);
    e = n_orb > 64 ? dedup<false, Key2>(r, n, high, ko, co, nu, W, L, count, sms, s)
        : n_orb <= 31 && (1u << n_orb) <= L.slots ? dedup<true, Key1>(r, n, high, ko, co, nu, W, L, count, sms, s)
                                                  : dedup<false, Key1>(r, n, high, ko, co, nu, W, L, count, sms, s);
    if (e != cudaSuccess) return dfail(QC_ERR_CUDA, cudaGetErrorString(e));
    return QC_OK;
}
