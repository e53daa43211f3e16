// The byte tries of a forest built on the device from the raw strings
// (Sec. 4.1; App. G.1 Step 1), for per-request sets that change every batch.
//
// Forests of small sets are sorted set by set (k_b_set_sort, k_b_set_nodes,
// below). The others: level by level over depth d, for all sets at once,
// without sorting the strings: every string of length > d ORs its byte d into the 256-bit
// child-label set of the node it has reached (its parent at depth d); the
// parents of a level, in order, give their children consecutive ids (first
// child = the level's end + an exclusive scan of the sets' popcounts), and a
// string moves to child first_child + popcount(labels below its byte). Level d
// is thus ordered by (set, parent, byte): breadth-first with sorted siblings
// within every set, the sets' nodes interleaved by depth. A final pass
// renumbers every node to base(set) + (its rank within the set's own
// breadth-first order), the layout of the host builder.
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include <cuda_runtime.h>

#include "tm_internal.h"

namespace tmk {

namespace {

constexpr int kBThreads = 256;
// Forests whose sets all hold at most this many strings are sorted, one CTA
// per set (42 B of shared memory a string). 256 sets of 300-2,000 names: 54 us
// to sort and 30 us to write the nodes, against 178 and 12 us by one CTA per
// set inserting level by level (seven barriers for each of ~32 levels), and
// 630 us by the level kernels over all sets.
constexpr int32_t kSetMaxStrings = 4096;
constexpr int kScanTile = 1024;  // parents per tile of the level scan

// Staging: copies the strings' offsets, the set offsets and the bytes into
// the scratch, checks the offsets (non-negative, non-decreasing) and finds
// the longest string. The sources are either the caller's host memory, read
// directly where the device accesses pageable memory coherently (Grace's
// NVLink-C2C), or device copies of it (src_off == off: checked in place;
// n_vec = 0: the bytes are in place). src_vec is the bytes' image in whole
// 16-byte blocks (the first and last block may hold bytes outside the
// strings; a 16-byte block never straddles a page).
__global__ void k_b_stage(const int64_t *src_off, int32_t K, const int32_t *src_soff, int32_t M,
                          const uint4 *src_vec, int64_t n_vec, int64_t *off, int32_t *soff, uint4 *vec,
                          int32_t *__restrict__ flags) {
    pdl_launch_dependents();
    pdl_wait();
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t i0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    int32_t longest = 0;
    int32_t bad = 0;
    for (int64_t i = i0; i <= K; i += stride) {
        const int64_t o = src_off[i];
        if (off != src_off) off[i] = o;
        if (o < 0) bad = 1;
        if (i < K) {
            const int64_t o2 = src_off[i + 1];
            if (o2 < o) bad = 1;
            else longest = max(longest, int32_t(min(o2 - o, int64_t(INT32_MAX))));
        }
    }
    if (soff != src_soff)
        for (int64_t i = i0; i <= M; i += stride) soff[i] = src_soff[i];
    for (int64_t k = i0; k < n_vec; k += stride) vec[k] = src_vec[k];
    longest = __reduce_max_sync(0xffffffffu, longest);
    bad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) {
        if (bad) atomicOr(flags, 1);
        if (longest) atomicMax(flags + 1, longest);
    }
}

// Strings: their set (from set_offsets), their node (the set's root), and the
// roots of sets with an empty string are terminal. Level 0 = the M roots;
// every non-empty string sets its first byte in its root's child-label set.
__global__ void k_b_init(const uint8_t *__restrict__ bytes, const int64_t *__restrict__ off,
                         const int32_t *__restrict__ set_off, int32_t M, int32_t K, int32_t *__restrict__ str_set,
                         int32_t *__restrict__ cur, int32_t *__restrict__ parent_g, uint8_t *__restrict__ label_g,
                         uint8_t *__restrict__ term_g, int32_t *__restrict__ set_g, int32_t *__restrict__ depth_g,
                         int32_t *__restrict__ ls, uint32_t *__restrict__ bits0) {
    pdl_launch_dependents();
    pdl_wait();
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M) {
        parent_g[i] = -1;
        label_g[i] = 0;
        set_g[i] = i;
        depth_g[i] = 0;
    }
    if (i == 0) {
        ls[0] = 0;
        ls[1] = M;
    }
    if (i >= K) return;
    int32_t lo = 0, hi = M;  // the set s with set_off[s] <= i < set_off[s + 1]
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (set_off[mid] <= i) lo = mid;
        else hi = mid;
    }
    str_set[i] = lo;
    cur[i] = lo;
    if (off[i + 1] == off[i]) {
        term_g[lo] = 1;  // the empty string: the root is terminal
    } else {
        const uint32_t b = bytes[off[i] - off[0]];
        atomicOr(bits0 + int64_t(lo) * 8 + (b >> 5), 1u << (b & 31u));
    }
}

__device__ __forceinline__ int32_t row_popc(const uint32_t *bits, int64_t row) {
    const uint4 *r = reinterpret_cast<const uint4 *>(bits + row * 8);
    const uint4 a = r[0], b = r[1];
    return __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w) + __popc(b.x) + __popc(b.y) + __popc(b.z) +
           __popc(b.w);
}

// Block-wide exclusive scan of one int per thread (kBThreads threads).
__device__ __forceinline__ int32_t block_excl_scan(int32_t v, int32_t *warp_sums, int32_t *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int32_t w = lane < kBThreads / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kBThreads / 32) warp_sums[lane] = w;
    }
    __syncthreads();
    const int32_t before = wid > 0 ? warp_sums[wid - 1] : 0;
    if (total) *total = warp_sums[kBThreads / 32 - 1];
    return before + x - v;
}

// Level d, pass 1: the children of every tile of kScanTile parents.
__global__ void __launch_bounds__(kBThreads) k_b_tile_sums(int32_t d, const int32_t *__restrict__ ls,
                                                           const uint32_t *__restrict__ bits,
                                                           int32_t *__restrict__ tile_sum) {
    __shared__ int32_t ws[kBThreads / 32];
    pdl_launch_dependents();
    pdl_wait();
    const int32_t width = ls[d + 1] - ls[d];
    const int32_t t0 = blockIdx.x * kScanTile;
    if (t0 >= width) {
        if (threadIdx.x == 0) tile_sum[blockIdx.x] = 0;
        return;
    }
    int32_t s = 0;
    for (int32_t j = threadIdx.x; j < kScanTile; j += kBThreads)
        if (t0 + j < width) s += row_popc(bits, t0 + j);
    int32_t tot;
    block_excl_scan(s, ws, &tot);
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}

// Level d, pass 2: first child of every parent of the level (the level's
// end + the children of the earlier tiles + an exclusive scan within the
// tile); block 0 also writes the end of level d + 1. Clears the other bits
// buffer (level d - 1's rows), into which the moves of level d set the
// child-label sets of level d + 1.
__global__ void __launch_bounds__(kBThreads) k_b_first(int32_t d, int32_t n_tiles, int32_t *__restrict__ ls,
                                                       const uint32_t *__restrict__ bits,
                                                       const int32_t *__restrict__ tile_sum,
                                                       int32_t *__restrict__ first, uint32_t *__restrict__ other) {
    __shared__ int32_t ws[kBThreads / 32];
    __shared__ int32_t carry;
    pdl_launch_dependents();
    pdl_wait();
    const int32_t width = ls[d + 1] - ls[d];
    const int32_t prev = d > 0 ? ls[d] - ls[d - 1] : 0;
    const int32_t t0 = blockIdx.x * kScanTile;
    for (int32_t j = threadIdx.x; j < kScanTile; j += kBThreads)
        if (t0 + j < prev) {
            uint4 *r = reinterpret_cast<uint4 *>(other + int64_t(t0 + j) * 8);
            r[0] = make_uint4(0u, 0u, 0u, 0u);
            r[1] = make_uint4(0u, 0u, 0u, 0u);
        }
    if (t0 >= width && blockIdx.x > 0) return;
    // children of the tiles before this one (all tiles for block 0's total)
    const int32_t upto = blockIdx.x > 0 ? int32_t(blockIdx.x) : n_tiles;
    int32_t part = 0;
    for (int32_t t = threadIdx.x; t < upto; t += kBThreads) part += tile_sum[t];
    int32_t sum;
    block_excl_scan(part, ws, &sum);
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) {
            ls[d + 2] = ls[d + 1] + sum;
            carry = ls[d + 1];
        } else {
            carry = ls[d + 1] + sum;
        }
    }
    __syncthreads();
    if (t0 >= width) return;
    for (int32_t j0 = 0; j0 < kScanTile; j0 += kBThreads) {
        const int32_t x = t0 + j0 + threadIdx.x;
        const int32_t c = x < width ? row_popc(bits, x) : 0;
        int32_t tot;
        const int32_t ex = block_excl_scan(c, ws, &tot);
        if (x < width) first[x] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

// Level d, pass 3: every string of length > d moves to its child at depth
// d + 1, writing the child's parent, label, set, depth and terminal flag
// (all strings through a child write the same values), and sets its byte
// d + 1, if any, in the child's child-label set (level d + 1's rows).
__global__ void k_b_move(const uint8_t *__restrict__ bytes, const int64_t *__restrict__ off, int32_t K, int32_t d,
                         const int32_t *__restrict__ ls, const uint32_t *__restrict__ bits,
                         const int32_t *__restrict__ first, const int32_t *__restrict__ str_set,
                         int32_t *__restrict__ cur, int32_t *__restrict__ parent_g, uint8_t *__restrict__ label_g,
                         uint8_t *__restrict__ term_g, int32_t *__restrict__ set_g, int32_t *__restrict__ depth_g,
                         uint32_t *__restrict__ bits_next) {
    pdl_launch_dependents();
    pdl_wait();
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= K) return;
    const int64_t len = off[i + 1] - off[i];
    if (len <= d) return;
    const int64_t a = off[i] - off[0];
    const uint32_t b = bytes[a + d];
    const int32_t x = cur[i];
    const int64_t row = x - ls[d];
    const uint32_t *r = bits + row * 8;
    int32_t below = 0;
#pragma unroll
    for (int w = 0; w < 8; w++) {
        const uint32_t v = r[w];
        const int32_t lo = w * 32;
        if (int32_t(b) >= lo + 32) below += __popc(v);
        else if (int32_t(b) >= lo) below += __popc(v & ((1u << (b - lo)) - 1u));
    }
    const int32_t c = first[row] + below;
    parent_g[c] = x;
    label_g[c] = uint8_t(b);
    set_g[c] = str_set[i];
    depth_g[c] = d + 1;
    cur[i] = c;
    if (len == d + 1) {
        term_g[c] = 1;
    } else {
        const uint32_t b1 = bytes[a + d + 1];
        atomicOr(bits_next + int64_t(c - ls[d + 1]) * 8 + (b1 >> 5), 1u << (b1 & 31u));
    }
}

// Renumbering, pass 1: the level-order range [first, end) of every (set,
// depth) group (level order sorts by depth, then set, so each group is one
// run), and the characters of the distinct strings (depths of terminals).
__global__ void k_b_count(const int32_t *__restrict__ ls, int32_t D, const int32_t *__restrict__ set_g,
                          const int32_t *__restrict__ depth_g, const uint8_t *__restrict__ term_g,
                          int32_t *__restrict__ first_sd, int32_t *__restrict__ end_sd,
                          unsigned long long *__restrict__ n_chars) {
    pdl_launch_dependents();
    pdl_wait();
    const int32_t n = ls[D + 1];
    unsigned long long chars = 0;
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const int32_t k = set_g[g] * (D + 1) + depth_g[g];
        if (g == 0 || set_g[g - 1] * (D + 1) + depth_g[g - 1] != k) first_sd[k] = g;
        if (g == n - 1 || set_g[g + 1] * (D + 1) + depth_g[g + 1] != k) end_sd[k] = g + 1;
        if (term_g[g]) chars += unsigned(depth_g[g]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) chars += __shfl_down_sync(0xffffffffu, chars, o);
    if ((threadIdx.x & 31) == 0 && chars) atomicAdd(n_chars, chars);
}

__device__ __forceinline__ int32_t group_size(const int32_t *first_sd, const int32_t *end_sd, int32_t k) {
    const int32_t e = end_sd[k];
    return e > 0 ? e - first_sd[k] : 0;  // end 0: no node of that set at that depth
}

// Renumbering, pass 2 (one CTA): the offset of every (set, depth) in the
// final layout (set after set, each in breadth-first order), and the roots.
__global__ void __launch_bounds__(kBThreads) k_b_offsets(int32_t M, int32_t D, const int32_t *__restrict__ first_sd,
                                                         const int32_t *__restrict__ end_sd,
                                                         int32_t *__restrict__ off_sd, int32_t *__restrict__ roots) {
    __shared__ int32_t ws[kBThreads / 32];
    __shared__ int32_t carry;
    pdl_launch_dependents();
    pdl_wait();
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int32_t s0 = 0; s0 < M; s0 += kBThreads) {
        const int32_t s = s0 + threadIdx.x;
        int32_t n_s = 0;
        if (s < M)
            for (int32_t d = 0; d <= D; d++) n_s += group_size(first_sd, end_sd, s * (D + 1) + d);
        int32_t tot;
        const int32_t base = carry + block_excl_scan(n_s, ws, &tot);
        if (s < M) {
            roots[s] = base;
            int32_t o = base;
            for (int32_t d = 0; d <= D; d++) {
                off_sd[s * (D + 1) + d] = o;
                o += group_size(first_sd, end_sd, s * (D + 1) + d);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

// Renumbering, pass 3: final id of every level-order id.
__global__ void k_b_map(const int32_t *__restrict__ ls, int32_t D, const int32_t *__restrict__ set_g,
                        const int32_t *__restrict__ depth_g, const int32_t *__restrict__ first_sd,
                        const int32_t *__restrict__ off_sd, int32_t *__restrict__ map) {
    pdl_launch_dependents();
    pdl_wait();
    const int32_t n = ls[D + 1];
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const int32_t k = set_g[g] * (D + 1) + depth_g[g];
        map[g] = off_sd[k] + (g - first_sd[k]);
    }
}

// Renumbering, pass 4: parent, label and terminal in the final layout.
__global__ void k_b_permute(const int32_t *__restrict__ ls, int32_t D, const int32_t *__restrict__ map,
                            const int32_t *__restrict__ parent_g, const uint8_t *__restrict__ label_g,
                            const uint8_t *__restrict__ term_g, int32_t *__restrict__ parent,
                            uint8_t *__restrict__ label, uint8_t *__restrict__ terminal) {
    pdl_launch_dependents();
    pdl_wait();
    const int32_t n = ls[D + 1];
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const int32_t f = map[g];
        const int32_t p = parent_g[g];
        parent[f] = p < 0 ? -1 : map[p];
        label[f] = label_g[g];
        terminal[f] = term_g[g];
    }
}

// ---- Forests of small sets: one CTA per set, without levels. The strings of
// the set are sorted in shared memory; string i of the sorted order then owns
// (is the first through) the nodes of depths lcp(i) + 1 .. len(i), lcp(i) the
// common prefix with string i - 1, so the node count is a sum, and within a
// depth the nodes in sorted order of their owners are the siblings-sorted
// breadth-first order: a node's rank is a count of owners before it, found by
// ballots, with no barrier per level.
constexpr int kSetThreads = 512;
constexpr int kSetKeyWords = 4;  // 8-byte words of a string kept in shared memory as its sort key
constexpr int kSetKeyBytes = 8 * kSetKeyWords;

// Exclusive scan of one int per thread over a block of kSetThreads.
__device__ __forceinline__ int32_t set_excl_scan(int32_t v, int32_t *ws, int32_t *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int32_t w = lane < kSetThreads / 32 ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kSetThreads / 32) ws[lane] = w;
    }
    __syncthreads();
    const int32_t before = wid > 0 ? ws[wid - 1] : 0;
    *total = ws[kSetThreads / 32 - 1];
    __syncthreads();  // ws is reused by the next scan
    return before + x - v;
}

// The first min(len, most) bytes at p as big-endian words (zeros after them),
// most <= kSetKeyBytes, by the aligned 8-byte words that hold them (all inside
// the staged image: only words with a byte of the string are read).
__device__ __forceinline__ void load_key(const uint8_t *p, int32_t len, int32_t most, uint64_t (&w)[kSetKeyWords]) {
    const int32_t n = len < most ? len : most;
    const uint32_t mis = uint32_t(reinterpret_cast<uintptr_t>(p)) & 7u;
    const uint64_t *q = reinterpret_cast<const uint64_t *>(p - mis);
    uint64_t raw[kSetKeyWords + 1];
#pragma unroll
    for (int k = 0; k <= kSetKeyWords; k++) raw[k] = 8 * k < n + int32_t(mis) && n > 0 ? q[k] : 0ull;
#pragma unroll
    for (int k = 0; k < kSetKeyWords; k++) {
        const uint64_t le = mis ? (raw[k] >> (8 * mis)) | (raw[k + 1] << (64 - 8 * mis)) : raw[k];
        const uint32_t lo = uint32_t(le), hi = uint32_t(le >> 32);
        uint64_t be = (uint64_t(__byte_perm(lo, 0, 0x0123)) << 32) | __byte_perm(hi, 0, 0x0123);
        const int32_t have = n - 8 * k;  // bytes of this word that belong to the string
        if (have <= 0) be = 0ull;
        else if (have < 8) be &= ~0ull << (64 - 8 * have);
        w[k] = be;
    }
}

// The strings of one set in shared memory: the key of string j in two halves
// of 16 bytes (key[j], key[cap + j]: one load compares 16 bytes, and names of
// one stem agree in their first 8) and its length. The key holds the string's
// bytes base .. limit - 1, at first the first kSetKeyBytes. Strings that agree
// in those and go on are sorted again by the bytes after them; their keys then
// begin with the number of the group of such neighbours (kGroupBytes of it).
constexpr int kGroupBytes = 2;

struct SetStrings {
    ulonglong2 *key;
    int32_t cap;
    uint16_t *len;
    int32_t base;
    int32_t limit;

    // What strings a and b of one group have in common from their start, or -1
    // where that is more than their keys show.
    __device__ __forceinline__ int32_t common(int32_t a, int32_t b) const {
        const int32_t n = min(int32_t(len[a]), int32_t(len[b]));
        const int32_t from = base ? base - kGroupBytes : 0;
#pragma unroll
        for (int h = 0; h < kSetKeyWords / 2; h++) {
            const ulonglong2 x = key[h * cap + a], y = key[h * cap + b];
            if (x.x != y.x) return min(n, from + 16 * h + (__clzll(static_cast<long long>(x.x ^ y.x)) >> 3));
            if (x.y != y.y) return min(n, from + 16 * h + 8 + (__clzll(static_cast<long long>(x.y ^ y.y)) >> 3));
        }
        return n <= limit ? n : -1;
    }

    // Whether a sorts before b by their keys; a0 and b0 are the first halves.
    __device__ __forceinline__ bool before(int32_t a, ulonglong2 a0, int32_t b, ulonglong2 b0) const {
        if (a0.x != b0.x) return a0.x < b0.x;
        if (a0.y != b0.y) return a0.y < b0.y;
        const ulonglong2 a1 = key[cap + a], b1 = key[cap + b];
        if (a1.x != b1.x) return a1.x < b1.x;
        if (a1.y != b1.y) return a1.y < b1.y;
        const int32_t la = len[a];
        return la <= limit && la < int32_t(len[b]);  // a prefix, then what it is a prefix of
    }
};

// Sorts the n strings listed in src by their keys, with dst for the rounds;
// the result is in src. Merge sort of 2-byte indices: every thread sorts
// kSortPer strings, then in each round finds by a search along its output's
// diagonal where its next kSortPer outputs begin in the two runs, and merges
// them. Ends with a barrier.
constexpr int kSortPer = 4;

__device__ __forceinline__ void sort_strings(const SetStrings &str, uint16_t *&src, uint16_t *&dst, int32_t n) {
    const int tid = threadIdx.x;
    const ulonglong2 *const key = str.key;
    for (int32_t o = kSortPer * tid; o < n; o += kSortPer * kSetThreads) {
        int32_t x[kSortPer];
        ulonglong2 x0[kSortPer];
        const int32_t m = min(kSortPer, n - o);
#pragma unroll
        for (int e = 0; e < kSortPer; e++) {
            x[e] = src[e < m ? o + e : o];
            x0[e] = key[x[e]];
        }
#pragma unroll
        for (int r = 1; r < kSortPer; r++)
#pragma unroll
            for (int e = r; e > 0; e--)
                if (r < m && str.before(x[e], x0[e], x[e - 1], x0[e - 1])) {
                    const int32_t y = x[e];
                    const ulonglong2 y0 = x0[e];
                    x[e] = x[e - 1], x0[e] = x0[e - 1];
                    x[e - 1] = y, x0[e - 1] = y0;
                }
#pragma unroll
        for (int e = 0; e < kSortPer; e++)
            if (e < m) src[o + e] = uint16_t(x[e]);
    }
    __syncthreads();
    for (int32_t w = kSortPer; w < n; w <<= 1) {
        for (int32_t o = kSortPer * tid; o < n; o += kSortPer * kSetThreads) {
            const int32_t first = o & ~(2 * w - 1), diag = o - first;
            const int32_t na = min(w, n - first), nb = max(0, min(w, n - first - w));
            const uint16_t *A = src + first, *B = A + w;
            int32_t lo = max(0, diag - nb), hi = min(diag, na);
            while (lo < hi) {  // the entries of A among the first diag outputs
                const int32_t mid = (lo + hi) >> 1;
                const int32_t x = A[mid], y = B[diag - 1 - mid];
                if (str.before(y, key[y], x, key[x])) hi = mid;
                else lo = mid + 1;
            }
            int32_t ia = lo, ib = diag - lo;
            int32_t x = ia < na ? int32_t(A[ia]) : 0, y = ib < nb ? int32_t(B[ib]) : 0;
            ulonglong2 x0 = key[x], y0 = key[y];
#pragma unroll
            for (int e = 0; e < kSortPer; e++) {
                if (o + e >= n) break;
                const bool from_b = ib < nb && (ia >= na || str.before(y, y0, x, x0));
                dst[o + e] = uint16_t(from_b ? y : x);
                if (from_b) {
                    ib++;
                    if (ib < nb) y = B[ib], y0 = key[y];
                } else {
                    ia++;
                    if (ia < na) x = A[ia], x0 = key[x];
                }
            }
        }
        __syncthreads();
        uint16_t *const t = src;
        src = dst;
        dst = t;
    }
}

// Sorts the strings of every set and gives their order: order[i] (i counted
// from the set's first string) = {lcp | len << 16, string within the set},
// the set's node count, and the characters of its distinct strings. The
// strings are sorted by their first kSetKeyBytes bytes; neighbours that agree
// in them and go on form groups, whose strings alone get the next bytes as
// keys, and are sorted again where those are not in order yet, until no two
// neighbours agree in all bytes looked at. So a root that all strings share is
// passed at a load and a comparison per kSetKeyBytes - kGroupBytes bytes (16
// sets of 1,200 strings of 24 bytes behind a root of 512: the build takes 0.27
// ms, 0.09 ms without the root; 29 ms where every comparison of the sort went
// through the root byte by byte). Three CTAs an SM, at 40 registers: at 64 a
// build of 2,000 sets of 100 strings takes 254 us, 231 us so.
// Bound by the chain of shared-memory loads of the merge sort's searches: about
// 3 us a round at 1,203 strings, 31 us in all. (Measured slower: every element
// searched for by itself in the neighbouring run, four side by side, 68 us for
// the 256 sets; 8-byte words of the key compared one load after the other, and
// keys of 32 contiguous bytes, whose first halves share half of the banks, 65
// us.) Does nothing when the staging found bad offsets or a string longer than
// the build takes (flags).
static_assert(kSetMaxStrings / kSetThreads <= 32, "a thread's places in the order have a bit each");

__global__ void __launch_bounds__(kSetThreads, 3) k_b_set_sort(const uint8_t *__restrict__ bytes,
                                                            const int64_t *__restrict__ off,
                                                            const int32_t *__restrict__ set_off, int32_t M,
                                                            int32_t cap, const int32_t *__restrict__ flags,
                                                            uint2 *__restrict__ order, int32_t *__restrict__ count,
                                                            unsigned long long *__restrict__ chars) {
    extern __shared__ uint4 dyn[];
    ulonglong2 *key = reinterpret_cast<ulonglong2 *>(dyn);
    uint16_t *len = reinterpret_cast<uint16_t *>(key + 2 * size_t(cap));
    uint16_t *pos = len + cap, *const lcp = pos + cap;  // the order, and what each string shares with the one before
    uint16_t *list = lcp + cap, *buf = list + cap;      // the strings to sort, and the sort's other side
    __shared__ int32_t ws[kSetThreads / 32];
    __shared__ int2 sums[kSetThreads / 32];
    __shared__ uint8_t edge[kSetThreads + 1];
    pdl_launch_dependents();
    pdl_wait();
    if (flags[0] != 0 || flags[1] > kDeviceBuildMaxDepth) return;
    const int tid = threadIdx.x;
    const int64_t off0 = off[0];
    for (int32_t s = blockIdx.x; s < M; s += gridDim.x) {
        const int32_t i0 = set_off[s], n = set_off[s + 1] - i0;
        for (int32_t j = tid; j < n; j += kSetThreads) {
            const int64_t a = off[i0 + j];
            const int32_t l = int32_t(off[i0 + j + 1] - a);
            uint64_t w[kSetKeyWords];
            load_key(bytes + (a - off0), l, kSetKeyBytes, w);
            key[j] = make_ulonglong2(w[0], w[1]);
            key[cap + j] = make_ulonglong2(w[2], w[3]);
            len[j] = uint16_t(l);
            list[j] = uint16_t(j);
        }
        __syncthreads();
        SetStrings str{key, cap, len, 0, kSetKeyBytes};
        // this thread's places in the order, r0 .. r1 - 1. Bit k of tied: the
        // string at place r0 + k is in the list; of joined: it agrees with the
        // one before it in all bytes looked at.
        const int32_t per = (n + kSetThreads - 1) / kSetThreads;
        const int32_t r0 = min(tid * per, n), r1 = min(r0 + per, n);
        uint32_t tied = (1u << (r1 - r0)) - 1u;
        uint32_t joined = r0 ? tied : tied & ~1u;
        int32_t listed = n, at0 = r0;  // strings in the list; this thread's first
        bool in_order = false;
        if (r0 == 0 && n > 0) lcp[0] = 0;
        while (true) {
            if (!in_order) {
                sort_strings(str, list, buf, listed);
                if (str.base == 0) {  // every string, so the list is the order
                    uint16_t *const t = pos;
                    pos = list;
                    list = t;
                } else {
                    for (int32_t k = 0, at = at0; k < r1 - r0; k++)
                        if ((tied >> k) & 1u) pos[r0 + k] = list[at++];
                    __syncthreads();
                }
            }
            for (int32_t k = 0; k < r1 - r0; k++) {
                if (!((joined >> k) & 1u)) continue;
                const int32_t c = str.common(pos[r0 + k - 1], pos[r0 + k]);
                if (c < 0) continue;
                lcp[r0 + k] = uint16_t(c);
                joined &= ~(1u << k);
            }
            if (tid == 0) edge[kSetThreads] = 0;
            edge[tid] = uint8_t(joined & 1u);
            if (!__syncthreads_or(joined != 0u)) break;
            tied = joined | (joined >> 1);  // joined, or the string after it is
            if (r1 < n && edge[tid + 1]) tied |= 1u << (r1 - r0 - 1);
            const uint32_t heads = tied & ~joined;
            str.base = str.limit;
            str.limit += kSetKeyBytes - kGroupBytes;
            const int32_t before = set_excl_scan(__popc(tied) | (__popc(heads) << 16), ws, &listed);
            listed &= 0xFFFF;
            at0 = before & 0xFFFF;
            int32_t group = before >> 16;
            for (int32_t k = 0, at = at0; k < r1 - r0; k++) {
                if (!((tied >> k) & 1u)) continue;
                group += int32_t((heads >> k) & 1u);
                const int32_t b = pos[r0 + k];
                uint64_t w[kSetKeyWords];
                load_key(bytes + (off[i0 + b] - off0) + str.base, int32_t(len[b]) - str.base,
                         kSetKeyBytes - kGroupBytes, w);
                key[b] = make_ulonglong2((w[0] >> 16) | (uint64_t(group) << 48), (w[1] >> 16) | (w[0] << 48));
                key[cap + b] = make_ulonglong2((w[2] >> 16) | (w[1] << 48), (w[3] >> 16) | (w[2] << 48));
                list[at++] = uint16_t(b);
            }
            __syncthreads();
            in_order = true;
            for (int32_t k = 0; k < r1 - r0; k++) {
                if (!((joined >> k) & 1u)) continue;
                const int32_t x = pos[r0 + k], y = pos[r0 + k - 1];
                in_order = in_order && !str.before(x, key[x], y, key[y]);
            }
            in_order = !__syncthreads_or(!in_order);
        }
        int32_t nodes = 0, my_chars = 0;
        for (int32_t i = tid; i < n; i += kSetThreads) {
            const int32_t b = pos[i], l = len[b], c = lcp[i];
            order[i0 + i] = make_uint2(uint32_t(c) | (uint32_t(l) << 16), uint32_t(b));
            nodes += l - c;
            if (i == 0 || c < l) my_chars += l;  // not a repetition of the string before it
        }
        nodes = __reduce_add_sync(0xffffffffu, nodes);
        my_chars = __reduce_add_sync(0xffffffffu, my_chars);
        if ((tid & 31) == 0) sums[tid >> 5] = make_int2(nodes, my_chars);
        __syncthreads();
        if (tid < 32) {
            const int2 v = tid < kSetThreads / 32 ? sums[tid] : make_int2(0, 0);
            nodes = __reduce_add_sync(0xffffffffu, v.x);
            my_chars = __reduce_add_sync(0xffffffffu, v.y);
            if (tid == 0) {
                count[s] = 1 + nodes;
                if (my_chars) atomicAdd(chars, static_cast<unsigned long long>(my_chars));
            }
        }
    }
}

// One CTA: every set's base (exclusive scan of the node counts) = its root,
// and the total.
__global__ void __launch_bounds__(kBThreads) k_b_set_scan(int32_t M, const int32_t *__restrict__ count,
                                                          int32_t *__restrict__ roots, int32_t *__restrict__ total) {
    __shared__ int32_t ws[kBThreads / 32];
    __shared__ int32_t carry;
    pdl_launch_dependents();
    pdl_wait();
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int32_t s0 = 0; s0 < M; s0 += kBThreads) {
        const int32_t s = s0 + threadIdx.x;
        int32_t tot;
        const int32_t ex = block_excl_scan(s < M ? count[s] : 0, ws, &tot);
        if (s < M) roots[s] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// The nodes of every set from its sorted strings, in their final place: a
// warp per depth goes through the strings in sorted order, 32 at a time; the
// owners at that depth take consecutive ids (their stores fall together), and
// a node's parent is the last owner at the depth above up to its string.
// kNodesBatch groups of 32 strings at a time, so that their label bytes (from
// L1 and L2) are waited for once. `parts` CTAs share a set, each taking every
// parts-th depth.
constexpr int kNodesBatch = 4;

__global__ void __launch_bounds__(kSetThreads) k_b_set_nodes(const uint8_t *__restrict__ bytes,
                                                             const int64_t *__restrict__ off,
                                                             const int32_t *__restrict__ set_off, int32_t M,
                                                             int32_t cap, int32_t D, int32_t parts,
                                                             const uint2 *__restrict__ order,
                                                             const int32_t *__restrict__ roots,
                                                             int32_t *__restrict__ parent, uint8_t *__restrict__ label,
                                                             uint8_t *__restrict__ terminal) {
    extern __shared__ uint4 dyn[];
    uint2 *str = reinterpret_cast<uint2 *>(dyn);            // sorted: {lcp | len << 16, place in the image}
    int32_t *start = reinterpret_cast<int32_t *>(str + cap);  // [D + 2] first id of each depth
    pdl_launch_dependents();
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t off0 = off[0];
    for (int64_t u = blockIdx.x; u < int64_t(M) * parts; u += gridDim.x) {
        const int32_t s = int32_t(u / parts), part = int32_t(u % parts);
        const int32_t i0 = set_off[s], n = set_off[s + 1] - i0, base = roots[s];
        __syncthreads();  // the set before this one is done with the shared arrays
        for (int32_t d = tid; d < D + 2; d += kSetThreads) start[d] = 0;
        __syncthreads();
        for (int32_t i = tid; i < n; i += kSetThreads) {
            const uint2 o = order[i0 + i];
            const int32_t lcp = int32_t(o.x & 0xFFFFu), l = int32_t(o.x >> 16);
            str[i] = make_uint2(o.x, uint32_t(off[i0 + int32_t(o.y)] - off0));
            if (lcp < l) {  // one more owner from depth lcp + 1, one fewer from l + 1
                atomicAdd(start + lcp + 1, 1);
                atomicAdd(start + l + 1, -1);
            }
        }
        __syncthreads();
        if (warp == 0) {  // changes of the owner count -> owners per depth -> first id of each depth
            int32_t owners = 0, ids = 1;
            for (int32_t d0 = 1; d0 <= D; d0 += 32) {
                int32_t x = d0 + lane <= D ? start[d0 + lane] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                const int32_t c = owners + x;  // owners at depth d0 + lane
                int32_t y = d0 + lane <= D ? c : 0;
                const int32_t mine = y;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t z = __shfl_up_sync(0xffffffffu, y, o);
                    if (lane >= o) y += z;
                }
                if (d0 + lane <= D) start[d0 + lane] = ids + y - mine;
                owners = __shfl_sync(0xffffffffu, c, 31);
                ids += __shfl_sync(0xffffffffu, y, 31);
            }
        }
        __syncthreads();
        if (part == 0 && tid == 0) {
            parent[base] = -1;
            label[base] = 0;
            terminal[base] = n > 0 && (str[0].x >> 16) == 0u;  // the empty string sorts first
        }
        for (int32_t d = 1 + warp * parts + part; d <= D; d += (kSetThreads / 32) * parts) {
            int32_t at = base + start[d];                                // next id at depth d
            int32_t above = base + (d > 1 ? start[d - 1] - 1 : 0);       // last node seen at depth d - 1
            for (int32_t c0 = 0; c0 < n; c0 += 32 * kNodesBatch) {
                int32_t id[kNodesBatch], up[kNodesBatch];
                uint32_t lab[kNodesBatch];
                bool ends[kNodesBatch];
#pragma unroll
                for (int k = 0; k < kNodesBatch; k++) {
                    const int32_t i = c0 + 32 * k + lane;
                    const uint2 sp = i < n ? str[i] : make_uint2(0xFFFFu, 0u);
                    const int32_t lcp = int32_t(sp.x & 0xFFFFu), l = int32_t(sp.x >> 16);
                    const bool own = lcp < d && d <= l;
                    const uint32_t here = __ballot_sync(0xffffffffu, own);
                    const uint32_t over = __ballot_sync(0xffffffffu, d > 1 && lcp < d - 1 && d - 1 <= l);
                    id[k] = own ? at + __popc(here & ((1u << lane) - 1u)) : -1;
                    up[k] = above + __popc(over & (0xFFFFFFFFu >> (31 - lane)));
                    lab[k] = own ? __ldg(bytes + sp.y + d - 1) : 0u;
                    ends[k] = d == l;
                    at += __popc(here);
                    above += __popc(over);
                }
#pragma unroll
                for (int k = 0; k < kNodesBatch; k++)
                    if (id[k] >= 0) {
                        parent[id[k]] = up[k];
                        label[id[k]] = uint8_t(lab[k]);
                        terminal[id[k]] = ends[k];
                    }
            }
        }
    }
}

}  // namespace

// Scratch of one device build. Staging part: the strings, the flags and
// counts read back, and the sorted order of a forest of small sets. Level part
// (once the longest string D is known): level-order node arrays (at most
// n_bytes + M nodes), two child-label buffers of max(K, M) rows, the level
// scans and ends, the (set, depth) tables.
struct DeviceBuild::Scratch {
    void *base = nullptr, *base2 = nullptr;
    size_t head_bytes;  // flags, total, characters and roots: one read-back
    uint8_t *bytes;
    uint4 *image;
    int64_t *off;
    int32_t *set_off, *str_set, *cur, *parent_g, *set_g, *depth_g, *first, *tile_sum, *ls, *flags;
    uint8_t *label_g, *term_g;
    uint32_t *bits[2];
    int32_t *end_sd, *first_sd, *off_sd, *roots, *map;
    int32_t *count, *total;  // small sets: nodes per set, all nodes
    uint2 *order;            // small sets: the sorted strings
    unsigned long long *n_chars;
};

DeviceBuild::~DeviceBuild() {
    if (s_) {
        if (s_->base) cudaFreeAsync(s_->base, stream_);
        if (s_->base2) cudaFreeAsync(s_->base2, stream_);
        delete s_;
    }
}

namespace {

struct Carver {
    size_t total = 0;
    size_t add(size_t b) {
        const size_t o = total;
        total += (b + 255) / 256 * 256;
        return o;
    }
};

// What the host reads back in one copy: {bad offsets, longest string, nodes,
// 0, characters (8 bytes)}, then the roots.
constexpr size_t kHeadRoots = 24;

size_t sort_smem(int32_t cap) { return size_t(cap) * (kSetKeyBytes + 5 * sizeof(uint16_t)); }
size_t nodes_smem(int32_t cap, int32_t D) {
    return size_t(cap) * sizeof(uint2) + sizeof(int32_t) * (size_t(D) + 2);
}

// Launches a kernel of one CTA per set, at most as many CTAs as are resident
// at once with `smem` bytes of dynamic shared memory (at most `smem_max`). The
// kernel's limit is state of the process that other threads' builds share, so
// it is always set to the same value, whatever this call needs.
template <typename... Params, typename... Args>
cudaError_t launch_sets(void (*kernel)(Params...), int64_t sets, size_t smem, size_t smem_max, int num_sms,
                        cudaStream_t st, Args... args) {
    int per_sm = 0;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_max))) !=
            cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kSetThreads, smem)) != cudaSuccess)
        return e;
    const int64_t grid = std::min<int64_t>(sets, int64_t(num_sms) * std::max(per_sm, 1));
    return launch_pdl_smem(kernel, grid, kSetThreads, smem, st, args...);
}

}  // namespace

cudaError_t DeviceBuild::stage(const uint8_t *h_bytes, const int64_t *h_off, const int32_t *h_set_off, int32_t M,
                               int32_t K, int64_t n_bytes, bool direct, int num_sms, cudaMemPool_t pool,
                               cudaStream_t st, int32_t *max_len, bool *offsets_ok) {
    stream_ = st;
    pool_ = pool;
    M_ = M;
    K_ = K;
    n_bytes_ = n_bytes;
    smax_ = 1;
    for (int32_t i = 0; i < M; i++) smax_ = std::max(smax_, h_set_off[i + 1] - h_set_off[i]);
    small_ = smax_ <= kSetMaxStrings;
    s_ = new Scratch();
    s_->head_bytes = kHeadRoots + 4 * size_t(M);
    Carver c;
    const size_t o_head = c.add(s_->head_bytes), o_img = c.add(size_t(n_bytes) + 32), o_off = c.add(8 * (size_t(K) + 1)),
                 o_soff = c.add(4 * (size_t(M) + 1)), o_cnt = c.add(4 * size_t(M)),
                 o_ord = c.add(small_ ? sizeof(uint2) * size_t(K) : 0);
    cudaError_t e = cudaMallocFromPoolAsync(&s_->base, c.total, pool, st);
    if (e != cudaSuccess) return e;
    char *b = static_cast<char *>(s_->base);
    const size_t mis = reinterpret_cast<uintptr_t>(h_bytes) & 15u;  // the image keeps the source's alignment
    s_->flags = reinterpret_cast<int32_t *>(b + o_head);
    s_->total = s_->flags + 2;
    s_->n_chars = reinterpret_cast<unsigned long long *>(b + o_head + 16);
    s_->roots = reinterpret_cast<int32_t *>(b + o_head + kHeadRoots);
    s_->image = reinterpret_cast<uint4 *>(b + o_img);
    s_->bytes = reinterpret_cast<uint8_t *>(b + o_img) + mis;
    s_->off = reinterpret_cast<int64_t *>(b + o_off);
    s_->set_off = reinterpret_cast<int32_t *>(b + o_soff);
    s_->count = reinterpret_cast<int32_t *>(b + o_cnt);
    s_->order = reinterpret_cast<uint2 *>(b + o_ord);
    if ((e = cudaMemsetAsync(s_->flags, 0, kHeadRoots, st)) != cudaSuccess) return e;
    const int64_t n_vec = n_bytes > 0 ? (int64_t(mis) + n_bytes + 15) / 16 : 0;
    const int64_t items = std::max<int64_t>(std::max<int64_t>(K, M) + 1, n_vec);
    const int64_t grid = std::min<int64_t>((items + kBThreads - 1) / kBThreads, int64_t(num_sms) * 16);
    if (direct) {
        e = launch_pdl(k_b_stage, grid, kBThreads, st, h_off, K, h_set_off, M,
                   reinterpret_cast<const uint4 *>(h_bytes - mis), n_vec, s_->off, s_->set_off, s_->image, s_->flags);
    } else {
        if ((n_bytes > 0 && (e = cudaMemcpyAsync(s_->bytes, h_bytes, size_t(n_bytes), cudaMemcpyHostToDevice, st)) !=
                                cudaSuccess) ||
            (e = cudaMemcpyAsync(s_->off, h_off, 8 * (size_t(K) + 1), cudaMemcpyHostToDevice, st)) != cudaSuccess ||
            (e = cudaMemcpyAsync(s_->set_off, h_set_off, 4 * (size_t(M) + 1), cudaMemcpyHostToDevice, st)) !=
                cudaSuccess)
            return e;
        e = launch_pdl(k_b_stage, grid, kBThreads, st, static_cast<const int64_t *>(s_->off), K,
                   static_cast<const int32_t *>(s_->set_off), M, static_cast<const uint4 *>(nullptr), int64_t(0),
                   s_->off, s_->set_off, s_->image, s_->flags);
    }
    if (e != cudaSuccess) return e;
    if (small_ &&
        ((e = launch_sets(k_b_set_sort, M, sort_smem(smax_), sort_smem(kSetMaxStrings), num_sms, st,
                          static_cast<const uint8_t *>(s_->bytes), static_cast<const int64_t *>(s_->off),
                          static_cast<const int32_t *>(s_->set_off), M, smax_, static_cast<const int32_t *>(s_->flags),
                          s_->order, s_->count, s_->n_chars)) != cudaSuccess ||
         (e = launch_pdl(k_b_set_scan, 1, kBThreads, st, M, static_cast<const int32_t *>(s_->count), s_->roots,
                         s_->total)) != cudaSuccess))
        return e;
    if ((e = read_head()) != cudaSuccess) return e;
    *offsets_ok = head_[0] == 0;
    *max_len = head_[1];
    return cudaSuccess;
}

// The flags, counts and roots, in one copy (host-synchronous).
cudaError_t DeviceBuild::read_head() {
    head_.resize(s_->head_bytes / 4);
    const cudaError_t e = cudaMemcpyAsync(head_.data(), s_->flags, s_->head_bytes, cudaMemcpyDeviceToHost, stream_);
    return e != cudaSuccess ? e : cudaStreamSynchronize(stream_);
}

void DeviceBuild::take_head(int32_t *n_nodes, std::vector<int32_t> *roots, int64_t *n_chars) {
    n_ = head_[2];
    *n_nodes = n_;
    memcpy(n_chars, head_.data() + 4, sizeof(int64_t));
    roots->assign(head_.begin() + kHeadRoots / 4, head_.end());
}

cudaError_t DeviceBuild::levels(int32_t D, int num_sms, int32_t *n_nodes, std::vector<int32_t> *roots,
                                int64_t *n_chars) {
    const cudaStream_t st = stream_;
    const int32_t M = M_, K = K_;
    D_ = D;
    if (small_) {  // sorted and counted behind the staging
        take_head(n_nodes, roots, n_chars);
        return cudaSuccess;
    }
    const int64_t U = n_bytes_ + M;             // nodes at most
    const int64_t W = std::max<int64_t>(K, M);  // parents of one level at most
    const int64_t tiles = (W + kScanTile - 1) / kScanTile + 1;
    const int64_t sd = int64_t(M) * (D + 1);
    Carver c;
    const size_t o_term = c.add(size_t(U)), o_b0 = c.add(32 * size_t(W) + 32), o_b1 = c.add(32 * size_t(W) + 32),
                 o_end = c.add(4 * size_t(sd)), zeroed = c.total, o_sset = c.add(4 * size_t(K)),
                 o_cur = c.add(4 * size_t(K)), o_par = c.add(4 * size_t(U)), o_set = c.add(4 * size_t(U)),
                 o_dep = c.add(4 * size_t(U)), o_first = c.add(4 * size_t(W)), o_ts = c.add(4 * size_t(tiles)),
                 o_lab = c.add(size_t(U)), o_map = c.add(4 * size_t(U)), o_ls = c.add(4 * (size_t(D) + 2)),
                 o_fsd = c.add(4 * size_t(sd)), o_osd = c.add(4 * size_t(sd));
    cudaError_t e = cudaMallocFromPoolAsync(&s_->base2, c.total, pool_, st);
    if (e != cudaSuccess) return e;
    char *b = static_cast<char *>(s_->base2);
    s_->term_g = reinterpret_cast<uint8_t *>(b + o_term);
    s_->bits[0] = reinterpret_cast<uint32_t *>(b + o_b0);
    s_->bits[1] = reinterpret_cast<uint32_t *>(b + o_b1);
    s_->end_sd = reinterpret_cast<int32_t *>(b + o_end);
    s_->str_set = reinterpret_cast<int32_t *>(b + o_sset);
    s_->cur = reinterpret_cast<int32_t *>(b + o_cur);
    s_->parent_g = reinterpret_cast<int32_t *>(b + o_par);
    s_->set_g = reinterpret_cast<int32_t *>(b + o_set);
    s_->depth_g = reinterpret_cast<int32_t *>(b + o_dep);
    s_->first = reinterpret_cast<int32_t *>(b + o_first);
    s_->tile_sum = reinterpret_cast<int32_t *>(b + o_ts);
    s_->label_g = reinterpret_cast<uint8_t *>(b + o_lab);
    s_->map = reinterpret_cast<int32_t *>(b + o_map);
    s_->ls = reinterpret_cast<int32_t *>(b + o_ls);
    s_->first_sd = reinterpret_cast<int32_t *>(b + o_fsd);
    s_->off_sd = reinterpret_cast<int32_t *>(b + o_osd);
    if ((e = cudaMemsetAsync(b, 0, zeroed, st)) != cudaSuccess) return e;
    const int64_t sgrid = (W + kBThreads - 1) / kBThreads;
    if ((e = launch_pdl(k_b_init, sgrid, kBThreads, st, static_cast<const uint8_t *>(s_->bytes),
                    static_cast<const int64_t *>(s_->off), static_cast<const int32_t *>(s_->set_off), M, K,
                    s_->str_set, s_->cur, s_->parent_g, s_->label_g, s_->term_g, s_->set_g, s_->depth_g, s_->ls,
                    s_->bits[0])) != cudaSuccess)
        return e;
    const int64_t kgrid = (int64_t(K) + kBThreads - 1) / kBThreads;
    const int32_t n_tiles = int32_t((W + kScanTile - 1) / kScanTile);
    for (int32_t d = 0; d < D; d++) {  // level d: bits[d & 1] holds its child-label sets
        uint32_t *bits = s_->bits[d & 1], *next = s_->bits[(d + 1) & 1];
        if ((e = launch_pdl(k_b_tile_sums, n_tiles, kBThreads, st, d, static_cast<const int32_t *>(s_->ls),
                        static_cast<const uint32_t *>(bits), s_->tile_sum)) != cudaSuccess ||
            (e = launch_pdl(k_b_first, n_tiles, kBThreads, st, d, n_tiles, s_->ls, static_cast<const uint32_t *>(bits),
                        static_cast<const int32_t *>(s_->tile_sum), s_->first, next)) != cudaSuccess ||
            (e = launch_pdl(k_b_move, kgrid, kBThreads, st, static_cast<const uint8_t *>(s_->bytes),
                        static_cast<const int64_t *>(s_->off), K, d, static_cast<const int32_t *>(s_->ls),
                        static_cast<const uint32_t *>(bits), static_cast<const int32_t *>(s_->first),
                        static_cast<const int32_t *>(s_->str_set), s_->cur, s_->parent_g, s_->label_g, s_->term_g,
                        s_->set_g, s_->depth_g, next)) != cudaSuccess)
            return e;
    }
    const int64_t ngrid = std::min<int64_t>((U + kBThreads - 1) / kBThreads, int64_t(num_sms) * 16);
    if ((e = launch_pdl(k_b_count, ngrid, kBThreads, st, static_cast<const int32_t *>(s_->ls), D,
                    static_cast<const int32_t *>(s_->set_g), static_cast<const int32_t *>(s_->depth_g),
                    static_cast<const uint8_t *>(s_->term_g), s_->first_sd, s_->end_sd, s_->n_chars)) != cudaSuccess ||
        (e = launch_pdl(k_b_offsets, 1, kBThreads, st, M, D, static_cast<const int32_t *>(s_->first_sd),
                    static_cast<const int32_t *>(s_->end_sd), s_->off_sd, s_->roots)) != cudaSuccess ||
        (e = launch_pdl(k_b_map, ngrid, kBThreads, st, static_cast<const int32_t *>(s_->ls), D,
                    static_cast<const int32_t *>(s_->set_g), static_cast<const int32_t *>(s_->depth_g),
                    static_cast<const int32_t *>(s_->first_sd), static_cast<const int32_t *>(s_->off_sd), s_->map)) !=
            cudaSuccess)
        return e;
    // the node count beside the roots and the characters
    if ((e = cudaMemcpyAsync(s_->total, s_->ls + D + 1, 4, cudaMemcpyDeviceToDevice, st)) != cudaSuccess ||
        (e = read_head()) != cudaSuccess)
        return e;
    take_head(n_nodes, roots, n_chars);
    return cudaSuccess;
}

cudaError_t DeviceBuild::emit(int32_t *parent, uint8_t *label, uint8_t *terminal, int num_sms) {
    if (small_) {
        // a few sets: their depths over several CTAs each, up to four CTAs an SM
        const int32_t parts = int32_t(std::min<int64_t>(8, std::max<int64_t>(1, 4 * int64_t(num_sms) / M_)));
        return launch_sets(k_b_set_nodes, int64_t(M_) * parts, nodes_smem(smax_, D_),
                           nodes_smem(kSetMaxStrings, kDeviceBuildMaxDepth), num_sms, stream_,
                           static_cast<const uint8_t *>(s_->bytes), static_cast<const int64_t *>(s_->off),
                           static_cast<const int32_t *>(s_->set_off), M_, smax_, D_, parts,
                           static_cast<const uint2 *>(s_->order), static_cast<const int32_t *>(s_->roots), parent,
                           label, terminal);
    }
    const int64_t ngrid = std::min<int64_t>((int64_t(n_) + kBThreads - 1) / kBThreads, int64_t(num_sms) * 16);
    return launch_pdl(k_b_permute, ngrid, kBThreads, stream_, static_cast<const int32_t *>(s_->ls), D_,
                  static_cast<const int32_t *>(s_->map), static_cast<const int32_t *>(s_->parent_g),
                  static_cast<const uint8_t *>(s_->label_g), static_cast<const uint8_t *>(s_->term_g), parent, label,
                  terminal);
}

}  // namespace tmk
