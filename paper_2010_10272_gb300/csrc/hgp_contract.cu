// libhgp: contraction of a vertex clustering into a coarse hypergraph (paper Sec. 3.2).
//
//   1. used cluster ids flagged and remapped to 0..n'-1 by an exclusive prefix sum;
//   2. coarse vertex weights by atomic adds (checked to fit int32);
//   3. every net's pins mapped to coarse ids, sorted and de-duplicated by size class: a thread
//      per net of at most 8 pins (sorting network in registers), a warp per net of 9..512 (bitonic
//      in registers, up to 16 values per lane), a CTA per net of up to 2048 (four such runs, merged
//      in shared memory), and for larger nets 2048-pin chunks sorted by separate CTAs and merged
//      pairwise by merge-path tiles spread over the whole grid; the net's fingerprint is taken
//      during the de-duplication;
//   4. nets with fewer than two pins dropped; identical nets found through a 64-bit
//      fingerprint table (key -> smallest net id) and an exact comparison with that net; a
//      net that only shares the fingerprint stays unresolved and takes part in the next round
//      (each round resolves the smallest net of every remaining fingerprint group);
//   5. the representatives (smallest id of each identical group) keep their original order;
//      their weights are the sums over the group; offsets by prefix sums.
// Everything is integer and the output is unique: pins sorted inside each net, nets ordered by
// their smallest original id.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <array>
#include <new>
#include <utility>

#include "hgp_host.cuh"

using namespace hgp;

struct hgp_coarse {
    int32_t fine_n = 0, n = 0, m = 0;
    int64_t P = 0;
    int64_t *net_off = nullptr;   // device [m+1]
    int32_t *pins = nullptr;      // device [P]
    int32_t *vw = nullptr;        // device [n]
    int32_t *nw = nullptr;        // device [m]
    int32_t *map = nullptr;       // device [fine_n]
    cudaStream_t stream = nullptr;
    int device = 0;
};

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kScanTile = 4096;
constexpr unsigned long long kKeyEmpty = ~0ull;
constexpr int32_t kUnresolved = -2, kDropped = -1;

int grid_of(int64_t work, int threads)
{
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 65535LL * 16) g = 65535LL * 16;
    return (int)g;
}

// ---------------------------------------------------------------- device-wide exclusive scan
// out[0..len] = exclusive prefix sums of in[0..len-1] (out[len] = total).  Reduce, then scan: a tile's
// sum first, so that the 8-byte output is written once (scanning the tiles and adding the offsets
// afterwards wrote and read it twice more; 10M entries 68 -> 35 us).
constexpr int kScanPer = 4;   // entries per thread

template <typename T>
__device__ __forceinline__ int64_t scan_load(const T *in, int64_t len, int64_t i0, int64_t (&v)[kScanPer])
{
    int64_t sum = 0;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        v[q] = i0 + q < len ? (int64_t)in[i0 + q] : 0;
        sum += v[q];
    }
    return sum;
}

// exclusive prefix of v over the CTA (kScanTile / kScanPer threads); total in *total
__device__ __forceinline__ int64_t scan_cta(int64_t v, int64_t *wt, int64_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wt[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const int64_t t = lane < kScanTile / kScanPer / 32 ? wt[lane] : 0;
        int64_t s = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(kFull, s, o);
            if (lane >= o) s += y;
        }
        wt[lane] = s - t;
        if (lane == 31) *total = s;
    }
    __syncthreads();
    return wt[wid] + x - v;
}

template <typename T>
__global__ void __launch_bounds__(kScanTile / kScanPer) k_scan_tile(const T *in, int64_t len, int64_t *sums)
{
    __shared__ int64_t wt[32], total;
    int64_t v[kScanPer];
    const int64_t s = scan_load(in, len, blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanPer, v);
    scan_cta(s, wt, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

template <typename T, typename O>
__global__ void __launch_bounds__(kScanTile / kScanPer) k_scan_out(const T *in, int64_t len, const int64_t *prefix,
                                                                   O *out)
{
    __shared__ int64_t wt[32], total;
    int64_t v[kScanPer];
    const int64_t i0 = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanPer;
    int64_t run = scan_cta(scan_load(in, len, i0, v), wt, &total) + (prefix ? prefix[blockIdx.x] : 0);
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        if (i0 + q <= len) out[i0 + q] = (O)run;
        run += v[q];
    }
}

// exclusive scan with the total at out[len]; out has len + 1 entries
template <typename T, typename O>
cudaError_t scan_excl(const T *in, int64_t len, O *out, cudaStream_t st)
{
    const int64_t tiles = len / kScanTile + 1;   // covers indices 0..len
    constexpr int threads = kScanTile / kScanPer;
    if (tiles == 1) {
        k_scan_out<T, O><<<1, threads, 0, st>>>(in, len, nullptr, out);
        return cudaGetLastError();
    }
    int64_t *sums = nullptr;
    cudaError_t e = dev_alloc(reinterpret_cast<void **>(&sums), sizeof(int64_t) * (size_t)(2 * tiles + 1), st);
    if (e != cudaSuccess) return e;
    int64_t *pref = sums + tiles;
    k_scan_tile<T><<<(unsigned)tiles, threads, 0, st>>>(in, len, sums);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = scan_excl(sums, tiles, pref, st);
    if (e == cudaSuccess) {
        k_scan_out<T, O><<<(unsigned)tiles, threads, 0, st>>>(in, len, pref, out);
        e = cudaGetLastError();
    }
    pool_free(sums, st);
    return e;
}

// ---------------------------------------------------------------- input checks
// offsets non-decreasing from 0 to P, pins in [0, n), weights >= 1
__global__ void k_ct_check(const int64_t *off, const int32_t *pins, const int32_t *vw, const int32_t *nw,
                           int32_t n, int32_t m, int64_t P, int32_t *err)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t e = t; e < m; e += stride) {
        if (off[e] < 0 || off[e] > off[e + 1] || off[e + 1] > P || (e == 0 && off[0] != 0)) atomicOr(err, ERR_INVALID);
        if (nw && nw[e] < 1) atomicOr(err, ERR_INVALID);
    }
    bool bad = false;
    for (int64_t j0 = t; j0 < P; j0 += 8 * stride) {   // eight pins per thread in flight
        int32_t v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = j0 + q * stride < P ? __ldcs(&pins[j0 + q * stride]) : 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) bad = bad || v[q] < 0 || v[q] >= n;
    }
    if (bad) atomicOr(err, ERR_INVALID);
    if (vw)
        for (int64_t u = t; u < n; u += stride)
            if (vw[u] < 1) atomicOr(err, ERR_INVALID);
}

// ---------------------------------------------------------------- clusters and weights
__global__ void k_ct_flag(const int32_t *cluster, int32_t n, int32_t *used, int32_t *err)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = cluster[u];
        if (c < 0 || c >= n) atomicOr(err, ERR_INVALID);
        else used[c] = 1;
    }
}

__global__ void k_ct_map(const int32_t *cluster, int32_t n, const int32_t *cid, const int32_t *vw,
                         int32_t *map, unsigned long long *w64)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = cid[cluster[u]];
        map[u] = c;
        atomicAdd(&w64[c], (unsigned long long)(vw ? vw[u] : 1));
    }
}

__global__ void k_ct_narrow(const unsigned long long *w64, int64_t len, int32_t *out, int32_t *err)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long w = w64[i];
        if (w >= (1ull << 31)) atomicOr(err, ERR_UNSUPPORTED);
        out[i] = (int32_t)w;
    }
}

// ---------------------------------------------------------------- per-net sort + dedupe
// Fingerprint of a sorted, de-duplicated pin list: the sum of a 64-bit mix of every pin
// (independent of how the pins are split over threads), mixed with the list's length.  Nets with equal
// fingerprints are compared, so the mix of a pin is a short one: two odd multipliers, the upper half
// folded into the lower after each.
__device__ __forceinline__ unsigned long long pin_mix(int32_t v)
{
    uint64_t x = (uint64_t)((uint32_t)v + 1u) * 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 32)) * 0xd1342543de82ef95ull;
    return x ^ (x >> 32);
}

__device__ __forceinline__ unsigned long long key_final(unsigned long long h, int32_t s)
{
    const unsigned long long k = splitmix64_output(h ^ ((uint64_t)(uint32_t)s << 32));
    return k == kKeyEmpty ? k - 1 : k;
}

// result of one net: its de-duplicated size, and its fingerprint (or dropped, < 2 pins)
__device__ __forceinline__ void net_done(int64_t e, int32_t kept, unsigned long long h, int32_t *size1,
                                         unsigned long long *key, int32_t *rep)
{
    size1[e] = kept;
    if (kept < 2) {
        rep[e] = kDropped;
    } else {
        key[e] = key_final(h, kept);
        rep[e] = kUnresolved;
    }
}

constexpr int kTiny = 8, kMid = 512, kMedium = 2048;
constexpr int kClasses = 4;   // listed classes: 9..32, 33..kMid, kMid+1..kMedium, larger

// thread per net: nets of at most kTiny pins are sorted in registers (an unrolled sorting
// network), de-duplicated and fingerprinted; larger nets go to the lists of the warp (9..32 pins,
// ..kMid), CTA (..kMedium) and chunked (larger) kernels.  A CTA reserves its places in a list with one
// atomic (one per warp: 800k returning atomics on one sector for 10M nets, and this kernel 464 us
// instead of 240).
__global__ void __launch_bounds__(256) k_ct_tiny(const int64_t *off, const int32_t *pins, int32_t m,
                                                 const int32_t *map, int32_t *a, int32_t *size1,
                                                 unsigned long long *key, int32_t *rep, int32_t *lists,
                                                 int32_t *counts)
{
    __shared__ int32_t n_of[kClasses][8], at[kClasses];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x; e0 < m; e0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = e0 + threadIdx.x;
        int cls = -1;
        if (e < m) {
            const int64_t b = off[e];
            const int32_t s = (int32_t)(off[e + 1] - b);
            if (s <= kTiny) {
                int32_t v[kTiny];
#pragma unroll
                for (int i = 0; i < kTiny; ++i) v[i] = i < s ? map[pins[b + i]] : 0x7fffffff;
#pragma unroll
                for (int i = 1; i < kTiny; ++i) {
#pragma unroll
                    for (int j = i; j > 0; --j) {
                        const int32_t lo = min(v[j - 1], v[j]), hi = max(v[j - 1], v[j]);
                        v[j - 1] = lo;
                        v[j] = hi;
                    }
                }
                int32_t kept = 0;
                unsigned long long h = 0;
#pragma unroll
                for (int i = 0; i < kTiny; ++i) {
                    if (i < s && (i == 0 || v[i] != v[i - 1])) {
                        a[b + kept] = v[i];
                        h += pin_mix(v[i]);
                        ++kept;
                    }
                }
                net_done(e, kept, h, size1, key, rep);
            } else {
                cls = s <= 32 ? 0 : (s <= kMid ? 1 : (s <= kMedium ? 2 : 3));
            }
        }
        // append of the larger nets to their class lists
        unsigned mine = 0;
#pragma unroll
        for (int c = 0; c < kClasses; ++c) {
            const unsigned mk = __ballot_sync(kFull, cls == c);
            if (cls == c) mine = mk;
            if (lane == 0) n_of[c][wid] = __popc(mk);
        }
        __syncthreads();
        if (threadIdx.x < kClasses) {
            int32_t total = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const int32_t x = n_of[threadIdx.x][w];
                n_of[threadIdx.x][w] = total;
                total += x;
            }
            at[threadIdx.x] = total ? atomicAdd(&counts[threadIdx.x], total) : 0;
        }
        __syncthreads();
        if (cls >= 0)
            lists[(int64_t)cls * m + at[cls] + n_of[cls][wid] + __popc(mine & ((1u << lane) - 1))] = (int32_t)e;
        __syncthreads();   // the counts are used again
    }
}

// Bitonic sort of 32 K values, K per lane in registers: ascending in the order lane * K + i.  Pairs
// closer than K are in the lane, the others come by shuffle; no shared memory and no barriers
// (sorting in shared memory, two accesses and a barrier per step, took 346 us for the nets of
// 33..256 pins and 584 us for those of 257..2048 of a 10M-net power-law instance; 244 us for 33..512
// and 135 for 513..2048 now).
template <int K>
__device__ __forceinline__ void warp_sort(int32_t (&v)[K])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32 * K; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= K) {
                const int dl = j / K;
                const bool keep_min = ((lane & dl) == 0) == (((lane * K) & k) == 0);
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const int32_t o = __shfl_xor_sync(kFull, v[i], dl);
                    v[i] = keep_min ? min(v[i], o) : max(v[i], o);
                }
            } else {
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    if (i & j) continue;
                    const bool up = ((lane * K + i) & k) == 0;
                    const int32_t x = v[i], y = v[i | j];
                    v[i] = up ? min(x, y) : max(x, y);
                    v[i | j] = up ? max(x, y) : min(x, y);
                }
            }
        }
    }
}

// mapped pins first .. of a run of s, 32 K of them into the lanes' registers (any order; absent ones sort
// last: coarse ids are below 2^31 - 1)
template <int K>
__device__ __forceinline__ void load_mapped(const int32_t *pins, const int32_t *map, int32_t first, int32_t s,
                                            int32_t (&v)[K])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = first + i * 32 + lane < s ? __ldcs(&pins[first + i * 32 + lane]) : -1;
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = v[i] >= 0 ? map[v[i]] : 0x7fffffff;
}

// one net of at most 32 K pins by a warp
template <int K>
__device__ __forceinline__ void warp_net(int64_t e, int64_t b, int32_t s, const int32_t *pins, const int32_t *map,
                                         int32_t *a, int32_t *size1, unsigned long long *key, int32_t *rep)
{
    const int lane = threadIdx.x & 31;
    int32_t v[K];
    load_mapped<K>(pins + b, map, 0, s, v);
    warp_sort<K>(v);
    int32_t prev = __shfl_up_sync(kFull, v[K - 1], 1);
    if (lane == 0) prev = -1;
    uint32_t keep = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        if (v[i] != prev && lane * K + i < s) keep |= 1u << i;
        prev = v[i];
    }
    int32_t incl = __popc(keep);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    int32_t *out = a + b + (incl - __popc(keep));
    unsigned long long h = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        if ((keep >> i) & 1) {
            *out++ = v[i];
            h += pin_mix(v[i]);
        }
    }
    for (int o = 16; o; o >>= 1) h += __shfl_xor_sync(kFull, h, o);
    if (lane == 31) net_done(e, incl, h, size1, key, rep);
}

// warp per listed net of 9..32 pins
__global__ void __launch_bounds__(256) k_ct_small(const int64_t *off, const int32_t *pins, const int32_t *map,
                                                  const int32_t *list, const int32_t *count, int32_t *a,
                                                  int32_t *size1, unsigned long long *key, int32_t *rep)
{
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int32_t cnt = *count;
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < cnt; i += warps) {
        const int64_t e = list[i], b = off[e];
        warp_net<1>(e, b, (int32_t)(off[e + 1] - b), pins, map, a, size1, key, rep);
    }
}

// warp per listed net of 33..kMid pins
__global__ void __launch_bounds__(256) k_ct_mid(const int64_t *off, const int32_t *pins, const int32_t *map,
                                                const int32_t *list, const int32_t *count, int32_t *a,
                                                int32_t *size1, unsigned long long *key, int32_t *rep)
{
    const int64_t warps = (int64_t)gridDim.x * 8;
    const int32_t cnt = *count;
    for (int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); i < cnt; i += warps) {
        const int64_t e = list[i], b = off[e];
        const int32_t s = (int32_t)(off[e + 1] - b);
        if (s <= 64) warp_net<2>(e, b, s, pins, map, a, size1, key, rep);
        else if (s <= 128) warp_net<4>(e, b, s, pins, map, a, size1, key, rep);
        else if (s <= 256) warp_net<8>(e, b, s, pins, map, a, size1, key, rep);
        else warp_net<16>(e, b, s, pins, map, a, size1, key, rep);
    }
}

// merge path: number of elements taken from A among the first d outputs of merge(A, B)
__device__ __forceinline__ int32_t merge_split(const int32_t *A, int32_t na, const int32_t *B, int32_t nb, int32_t d)
{
    int32_t lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {
        const int32_t i = (lo + hi) >> 1;          // candidate count from A
        if (A[i] <= B[d - 1 - i]) lo = i + 1;     // A[i] comes before B[d-1-i]: take more from A
        else hi = i;
    }
    return lo;
}

// A CTA of kCtaSort threads sorts up to kMedium mapped pins: a run of 512 per warp in registers, then two
// rounds of merges in shared memory, each thread 16 outputs of one merge.  Returns the buffer
// (x or y, kMedium values each) that holds the result.
constexpr int kCtaSort = 128;
constexpr int kRun = kMedium / (kCtaSort / 32);   // 512
constexpr int kOut = kMedium / kCtaSort;          // 16

__device__ __forceinline__ int32_t *cta_sort(const int32_t *pins, const int32_t *map, int32_t s, int32_t *x, int32_t *y)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    {
        int32_t v[kOut];
        load_mapped<kOut>(pins, map, wid * kRun, s, v);
        warp_sort<kOut>(v);
        int4 *dst = reinterpret_cast<int4 *>(x + wid * kRun + lane * kOut);
#pragma unroll
        for (int i = 0; i < kOut / 4; ++i) dst[i] = make_int4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
    __syncthreads();
#pragma unroll
    for (int w = kRun; w < kMedium; w *= 2) {
        const int o0 = tid * kOut, base = o0 / (2 * w) * (2 * w);
        const int32_t *A = x + base, *B = A + w;
        int i = merge_split(A, w, B, w, o0 - base), j = o0 - base - i;
        int32_t out[kOut];
        int32_t va = i < w ? A[i] : 0x7fffffff, vb = j < w ? B[j] : 0x7fffffff;
#pragma unroll
        for (int q = 0; q < kOut; ++q) {
            const bool take_a = j >= w || (i < w && va <= vb);
            out[q] = take_a ? va : vb;
            if (take_a) {
                ++i;
                va = i < w ? A[i] : 0x7fffffff;
            } else {
                ++j;
                vb = j < w ? B[j] : 0x7fffffff;
            }
        }
        int4 *dst = reinterpret_cast<int4 *>(y + o0);
#pragma unroll
        for (int q = 0; q < kOut / 4; ++q) dst[q] = make_int4(out[4 * q], out[4 * q + 1], out[4 * q + 2], out[4 * q + 3]);
        __syncthreads();
        int32_t *t = x;
        x = y;
        y = t;
    }
    return x;
}

// block-wide: order-preserving compaction of the first of every run of equal values of the
// sorted src[0..s) into dst (dst may equal src), fingerprint of the kept values
__device__ __forceinline__ void compact_runs(const int32_t *src, int32_t *dst, int32_t s, int32_t *wtot,
                                             unsigned long long *hsum, int32_t &kept_out, unsigned long long &h_out)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nw = blockDim.x >> 5;
    int32_t kept = 0;
    if (tid == 0) *hsum = 0;
    for (int32_t t0 = 0; t0 < s; t0 += blockDim.x) {
        const int32_t j = t0 + tid;
        const bool has = j < s;
        const int32_t v = has ? src[j] : 0;
        const bool keep = has && (j == 0 || v != src[j - 1]);
        const unsigned km = __ballot_sync(kFull, keep);
        if (lane == 0) wtot[wid] = __popc(km);
        __syncthreads();
        int32_t before = kept, tile_total = 0;
        for (int w = 0; w < nw; ++w) {
            if (w < wid) before += wtot[w];
            tile_total += wtot[w];
        }
        __syncthreads();   // every thread has read its input and the counts
        if (keep) dst[before + __popc(km & ((1u << lane) - 1))] = v;
        if (km) {
            unsigned long long h = keep ? pin_mix(v) : 0ull;
            for (int o = 16; o; o >>= 1) h += __shfl_xor_sync(kFull, h, o);
            if (lane == 0) atomicAdd(hsum, h);
        }
        kept += tile_total;
        __syncthreads();
    }
    kept_out = kept;
    h_out = *hsum;
}

// CTA per listed net of kMid+1..kMedium pins: sort, then compaction into a and the fingerprint
__global__ void __launch_bounds__(kCtaSort) k_ct_medium(const int64_t *off, const int32_t *pins, const int32_t *map,
                                                        const int32_t *list, const int32_t *count, int32_t *a,
                                                        int32_t *size1, unsigned long long *key, int32_t *rep)
{
    __shared__ __align__(16) int32_t x[kMedium], y[kMedium];
    __shared__ int32_t wtot[kCtaSort / 32];
    __shared__ unsigned long long hsum;
    const int32_t cnt = *count;
    for (int64_t i = blockIdx.x; i < cnt; i += gridDim.x) {
        const int64_t e = list[i], b = off[e];
        const int32_t s = (int32_t)(off[e + 1] - b);
        const int32_t *sorted = cta_sort(pins + b, map, s, x, y);
        int32_t kept;
        unsigned long long h;
        compact_runs(sorted, a + b, s, wtot, &hsum, kept, h);
        if (threadIdx.x == 0) net_done(e, kept, h, size1, key, rep);
        __syncthreads();
    }
}

// a representative's coarse id and offset, packed (see place_of)
__device__ __forceinline__ int64_t new_id(int64_t pos) { return pos >> 32; }
__device__ __forceinline__ int64_t new_off(int64_t pos) { return pos & 0xffffffff; }

// Nets of more than kMedium pins, load-balanced over the grid by tasks of kMedium pins: every chunk
// is sorted by one CTA (k_lg_chunk), then runs are merged pairwise, each CTA producing kMedium
// outputs of one merge found by a merge-path search (k_lg_merge); the distinct values of every chunk
// are counted and fingerprinted (k_lg_distinct), their places follow from a prefix sum, and each
// chunk is written there (k_lg_compact).  (One CTA per net for the last step took as long as the
// largest net: 543 us for nets of up to 100,000 pins.)
constexpr int kLgThreads = 256;

// The searches of a task are chains of dependent loads that its CTA waits for; a warp probes 32 places
// at a time (the six merge passes of a 10M-net power-law instance: 331 us with binary searches, 255 us).

// first index in [lo, hi) where `before` fails (it holds up to there); called by a whole warp
template <typename F>
__device__ __forceinline__ int32_t warp_search(int32_t lo, int32_t hi, F before)
{
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int32_t step = (hi - lo + 31) / 32;
        const int64_t i = lo + (int64_t)lane * step;
        const int c = __popc(__ballot_sync(kFull, i < hi && before((int32_t)i)));
        const int32_t from = lo;
        if (c) lo = from + (c - 1) * step + 1;
        if (c < 32) hi = (int32_t)min((int64_t)hi, from + (int64_t)c * step);
    }
    return lo;
}

// chunk task t -> (list index, chunk) through the exclusive prefix of the chunk counts
__device__ __forceinline__ int32_t find_task(const int64_t *cpre, int32_t nl, int64_t t)
{
    return warp_search(0, nl, [&](int32_t i) { return cpre[i] <= t; }) - 1;
}

// merge passes of a net of s pins.  Each net is merged as often as it needs and no more (with the
// finished ones copied along, the passes took 375 us instead of 331); its sorted pins end up in `b`,
// so its passes alternate from the buffer that makes it so.
__device__ __forceinline__ int merge_passes(int32_t s) { return 32 - __clz((s + kMedium - 1) / kMedium - 1); }

__global__ void k_lg_count(const int64_t *off, const int32_t *list, const int32_t *count, int32_t *chunks,
                           int32_t *max_size)
{
    const int32_t nl = *count;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nl; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = list[i];
        const int32_t sz = (int32_t)(off[e + 1] - off[e]);
        chunks[i] = (sz + kMedium - 1) / kMedium;
        atomicMax(max_size, sz);
    }
}

// task t: a representative's pins of the chunk to its coarse position (and with the first chunk its
// offset and summed weight)
__global__ void __launch_bounds__(kLgThreads) k_lg_emit(const int64_t *off, const int32_t *a, const int32_t *size1,
                                                        const int32_t *rep, const int64_t *pos,
                                                        const unsigned long long *w64, const int32_t *list,
                                                        const int32_t *count, const int64_t *cpre, int64_t tasks,
                                                        int32_t *pins2, int64_t *off2, int32_t *nw2, int32_t *err)
{
    const int32_t nl = *count;
    for (int64_t t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int32_t li = find_task(cpre, nl, t);
        const int64_t e = list[li];
        if (rep[e] != (int32_t)e) continue;
        const int64_t src = off[e], dst = new_off(pos[e]);
        const int32_t c0 = (int32_t)(t - cpre[li]) * kMedium, c1 = min(size1[e], c0 + kMedium);
#pragma unroll 4
        for (int32_t j = c0 + threadIdx.x; j < c1; j += kLgThreads) pins2[dst + j] = a[src + j];
        if (c0 == 0 && threadIdx.x == 0) {
            const int64_t id = new_id(pos[e]);
            off2[id] = dst;
            const unsigned long long w = w64[e];
            if (w >= (1ull << 31)) atomicOr(err, ERR_UNSUPPORTED);
            nw2[id] = (int32_t)w;
        }
    }
}

__global__ void __launch_bounds__(kCtaSort) k_lg_chunk(const int64_t *off, const int32_t *pins, const int32_t *map,
                                                       const int32_t *list, const int32_t *count, const int64_t *cpre,
                                                       int64_t tasks, int32_t *a, int32_t *bb)
{
    __shared__ __align__(16) int32_t x[kMedium], y[kMedium];
    const int32_t nl = *count;
    for (int64_t t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int32_t li = find_task(cpre, nl, t);
        const int64_t e = list[li], b = off[e];
        const int32_t s = (int32_t)(off[e + 1] - b);
        const int32_t c0 = (int32_t)(t - cpre[li]) * kMedium;
        const int32_t len = min(kMedium, s - c0);
        const int32_t *sorted = cta_sort(pins + b + c0, map, len, x, y);
        int32_t *dst = merge_passes(s) & 1 ? a : bb;
        for (int32_t j = threadIdx.x; j < len; j += kCtaSort) dst[b + c0 + j] = sorted[j];
        __syncthreads();
    }
}

// merge pass `pass` over the large nets that need it: sorted runs of kMedium << pass pins are merged
// pairwise; task t = output tile of kMedium elements of one net (same task numbering as the chunks).
// The tile's two input pieces are staged in shared memory.
__global__ void __launch_bounds__(kLgThreads) k_lg_merge(const int64_t *off, const int32_t *list, const int32_t *count,
                                                         const int64_t *cpre, int64_t tasks, int32_t *a, int32_t *bb,
                                                         int pass)
{
    const int32_t w = kMedium << pass;
    __shared__ int32_t in[kMedium], out[kMedium];
    __shared__ int32_t split[2];
    const int tid = threadIdx.x;
    const int32_t nl = *count;
    constexpr int kPer = kMedium / kLgThreads;
    for (int64_t t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int32_t li = find_task(cpre, nl, t);
        const int64_t e = list[li], b = off[e];
        const int32_t s = (int32_t)(off[e + 1] - b);
        const int left = merge_passes(s) - pass;
        if (left <= 0) continue;
        const int32_t *src = left & 1 ? a : bb;
        int32_t *dst = left & 1 ? bb : a;
        const int32_t o0 = (int32_t)(t - cpre[li]) * kMedium;   // the tile's outputs [o0, o0 + len)
        const int32_t len = min(kMedium, s - o0);
        const int32_t base = (o0 / (2 * w)) * (2 * w);           // w is a multiple of kMedium: one merge per tile
        const int32_t na = min(w, s - base), nb = max(0, min(w, s - base - w));
        const int32_t *A = src + b + base, *B = A + na;
        if (tid < 64) {   // as merge_split
            const int32_t d = o0 - base + (tid < 32 ? 0 : len);
            const int32_t x = warp_search(max(0, d - nb), min(d, na), [&](int32_t i) { return A[i] <= B[d - 1 - i]; });
            if ((tid & 31) == 0) split[tid >> 5] = x;
        }
        __syncthreads();
        const int32_t a0 = split[0], b0 = o0 - base - a0;
        const int32_t la = split[1] - a0, lb = len - la;
        for (int32_t j = tid; j < len; j += kLgThreads) in[j] = j < la ? A[a0 + j] : B[b0 + (j - la)];
        __syncthreads();
        const int32_t d0 = tid * kPer;
        if (d0 < len) {
            const int32_t *SA = in, *SB = in + la;
            int32_t i = merge_split(SA, la, SB, lb, d0), j = d0 - i;
            const int32_t n_out = min(kPer, len - d0);
            for (int q = 0; q < n_out; ++q) {
                const bool take_a = j >= lb || (i < la && SA[i] <= SB[j]);
                out[d0 + q] = take_a ? SA[i++] : SB[j++];
            }
        }
        __syncthreads();
        for (int32_t j = tid; j < len; j += kLgThreads) dst[b + o0 + j] = out[j];
        __syncthreads();
    }
}

// task t: number of values of its chunk that differ from the one before, and their fingerprint sum
__global__ void __launch_bounds__(kLgThreads) k_lg_distinct(const int64_t *off, const int32_t *list, const int32_t *count,
                                                            const int64_t *cpre, int64_t tasks, const int32_t *src,
                                                            int32_t *distinct, unsigned long long *hsum)
{
    const int tid = threadIdx.x;
    const int32_t nl = *count;
    for (int64_t t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int32_t li = find_task(cpre, nl, t);
        const int64_t e = list[li], b = off[e];
        const int32_t s = (int32_t)(off[e + 1] - b);
        const int32_t c0 = (int32_t)(t - cpre[li]) * kMedium, c1 = min(s, c0 + kMedium);
        int32_t kept = 0;
        unsigned long long h = 0;
        for (int32_t j = c0 + tid; j < c1; j += kLgThreads) {
            const int32_t v = src[b + j];
            if (j == 0 || v != src[b + j - 1]) {
                ++kept;
                h += pin_mix(v);
            }
        }
        kept = __reduce_add_sync(kFull, kept);
        for (int o = 16; o; o >>= 1) h += __shfl_xor_sync(kFull, h, o);
        if ((tid & 31) == 0 && kept) {
            atomicAdd(&distinct[t], kept);
            atomicAdd(&hsum[li], h);
        }
    }
}

// task t: its distinct values to their places (pre: exclusive prefix of the tasks' counts)
__global__ void __launch_bounds__(kLgThreads) k_lg_compact(const int64_t *off, const int32_t *list, const int32_t *count,
                                                           const int64_t *cpre, int64_t tasks, const int32_t *src,
                                                           const int64_t *pre, int32_t *a)
{
    __shared__ int32_t wtot[kLgThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int32_t nl = *count;
    for (int64_t t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int32_t li = find_task(cpre, nl, t);
        const int64_t e = list[li], b = off[e];
        const int32_t s = (int32_t)(off[e + 1] - b);
        const int32_t c0 = (int32_t)(t - cpre[li]) * kMedium, c1 = min(s, c0 + kMedium);
        int64_t at = b + (pre[t] - pre[cpre[li]]);
        for (int32_t j0 = c0; j0 < c1; j0 += kLgThreads) {
            const int32_t j = j0 + tid;
            const int32_t v = j < c1 ? src[b + j] : 0;
            const bool keep = j < c1 && (j == 0 || v != src[b + j - 1]);
            const unsigned km = __ballot_sync(kFull, keep);
            if (lane == 0) wtot[wid] = __popc(km);
            __syncthreads();
            int32_t before = 0, all = 0;
            for (int w = 0; w < kLgThreads / 32; ++w) {
                if (w < wid) before += wtot[w];
                all += wtot[w];
            }
            if (keep) a[at + before + __popc(km & ((1u << lane) - 1))] = v;
            at += all;
            __syncthreads();
        }
    }
}

// thread per large net: its size and fingerprint
__global__ void k_lg_done(const int32_t *list, const int32_t *count, const int64_t *cpre, const int64_t *pre,
                          const unsigned long long *hsum, int32_t *size1, unsigned long long *key, int32_t *rep)
{
    const int32_t nl = *count;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nl; i += (int64_t)gridDim.x * blockDim.x)
        net_done(list[i], (int32_t)(pre[cpre[i + 1]] - pre[cpre[i]]), hsum[i], size1, key, rep);
}

// ---------------------------------------------------------------- identical nets
// A slot holds a net's upper 32 fingerprint bits and its id, the smallest of the unresolved nets with
// those bits in their run of probes (which starts at the lower fingerprint bits).  All bytes 0xFF
// when free.  Nets that only share the bits are told apart by the comparison.
__device__ __forceinline__ uint64_t slot_value(unsigned long long key, int32_t e)
{
    return (key & 0xFFFFFFFF00000000ull) | (uint32_t)e;
}

// thread per unresolved net: its fingerprint's smallest unresolved net id
__global__ void k_ct_insert(const unsigned long long *key, const int32_t *rep, int32_t m, unsigned long long *tab,
                            uint64_t mask, int32_t *err)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        if (rep[e] != kUnresolved) continue;
        const unsigned long long val = slot_value(key[e], (int32_t)e);
        uint64_t p = key[e] & mask;
        bool placed = false;
        for (uint64_t probe = 0; probe <= mask; ++probe) {
            unsigned long long cur = __ldcg(&tab[p]);
            if (cur == kKeyEmpty) cur = atomicCAS(&tab[p], kKeyEmpty, val);
            if (cur == kKeyEmpty || (cur >> 32) == (val >> 32)) {
                if (cur != kKeyEmpty && val < cur) atomicMin(&tab[p], val);
                placed = true;
                break;
            }
            p = (p + 1) & mask;
        }
        if (!placed) atomicOr(err, ERR_INVALID);
    }
}

// the net in the slot of key's fingerprint bits, -1 if there is none
__device__ __forceinline__ int32_t smallest_net(const unsigned long long *tab, uint64_t mask, unsigned long long key)
{
    uint64_t p = key & mask;
    for (uint64_t probe = 0; probe <= mask; ++probe) {
        const unsigned long long cur = __ldcg(&tab[p]);
        if (cur == kKeyEmpty) return -1;
        if ((cur >> 32) == (key >> 32)) return (int32_t)(uint32_t)cur;
        p = (p + 1) & mask;
    }
    return -1;
}

// 32 nets per warp, one per lane: an unresolved net whose fingerprint's smallest net is itself
// is resolved to itself; the others compare their pin lists with that net, the whole warp on
// one net at a time, and are resolved to it if equal, else stay unresolved for the next round
__global__ void k_ct_resolve(const int64_t *off, const int32_t *a, const int32_t *size1,
                             const unsigned long long *key, int32_t *rep, int32_t m, const unsigned long long *tab,
                             uint64_t mask, int32_t *left)
{
    const int lane = threadIdx.x & 31;
    for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x; e0 < m; e0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = e0 + threadIdx.x;
        int32_t r = -1;
        bool todo = false;
        if (e < m && rep[e] == kUnresolved) {
            r = smallest_net(tab, mask, key[e]);
            if (r < 0) r = (int32_t)e;
            if (r == (int32_t)e) rep[e] = (int32_t)e;
            else todo = true;
        }
        unsigned tm = __ballot_sync(kFull, todo);
        int32_t nleft = 0;
        while (tm) {
            const int src = __ffs(tm) - 1;
            tm &= tm - 1;
            const int64_t ee = __shfl_sync(kFull, e, src);
            const int32_t rr = __shfl_sync(kFull, r, src);
            const int32_t se = size1[ee];
            bool eq = size1[rr] == se;
            if (eq) {
                const int32_t *pe = a + off[ee], *pr = a + off[rr];
                for (int32_t j = lane; j < se; j += 32) eq = eq && pe[j] == pr[j];
                eq = __all_sync(kFull, eq);
            }
            if (lane == src) {
                if (eq) rep[ee] = rr;
                else ++nleft;
            }
        }
        nleft = __reduce_add_sync(kFull, nleft);
        if (lane == 0 && nleft) atomicAdd(left, nleft);
    }
}

// Places of the representatives: one prefix sum over (1, pins) of each, packed as 1 << 32 | pins (both
// totals are below 2^31).  The first pass sums the tiles and sets every net's own weight, the second
// writes the places and adds the weights of the others to their representatives, which are few.
// (Separate flags, sizes and prefix sums, and an atomic on a zeroed weight for every net: 260 us for
// 10M nets, 130 now.)
__device__ __forceinline__ int64_t place_of(const int32_t *rep, const int32_t *size1, int64_t e)
{
    return rep[e] == (int32_t)e ? ((int64_t)1 << 32) + size1[e] : 0;
}

__global__ void __launch_bounds__(kScanTile / kScanPer) k_ct_groups(const int32_t *rep, const int32_t *size1,
                                                                    const int32_t *nw, int32_t m,
                                                                    unsigned long long *w64, int64_t *sums)
{
    __shared__ int64_t wt[32], total;
    const int64_t i0 = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanPer;
    int64_t s = 0;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        const int64_t e = i0 + q;
        if (e >= m) break;
        s += place_of(rep, size1, e);
        w64[e] = nw ? nw[e] : 1;
    }
    scan_cta(s, wt, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanTile / kScanPer) k_ct_places(const int32_t *rep, const int32_t *size1,
                                                                    const int32_t *nw, int32_t m,
                                                                    const int64_t *prefix, unsigned long long *w64,
                                                                    int64_t *pos)
{
    __shared__ int64_t wt[32], total;
    const int64_t i0 = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanPer;
    int64_t v[kScanPer], s = 0;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        v[q] = i0 + q < m ? place_of(rep, size1, i0 + q) : 0;
        s += v[q];
    }
    int64_t run = scan_cta(s, wt, &total) + prefix[blockIdx.x];
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        const int64_t e = i0 + q;
        if (e <= m) pos[e] = run;
        run += v[q];
        if (e < m && v[q] == 0) {
            const int32_t to = rep[e];
            if (to >= 0) atomicAdd(&w64[to], (unsigned long long)(nw ? nw[e] : 1));
        }
    }
}

__device__ __forceinline__ int slot_in(const int32_t *off33, int32_t i)
{
    int lo = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1)
        if (off33[lo + step] <= i) lo += step;
    return lo;
}

// 32 nets per warp, one per lane: the representatives' pins are copied to their coarse
// positions over the warp's flattened pin range (every lane copies a pin per step), and each
// representative's offset and summed weight are written by its lane
__global__ void k_ct_emit(const int64_t *off, const int32_t *a, const int32_t *size1, const int32_t *rep,
                          const int64_t *pos, const unsigned long long *w64, int32_t m, int32_t *pins2,
                          int64_t *off2, int32_t *nw2, int32_t *err)
{
    __shared__ int32_t off33_w[8][33];
    __shared__ int64_t src_w[8][32], dst_w[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *off33 = off33_w[wid];
    for (int64_t e0 = (blockIdx.x * (int64_t)blockDim.x) ; e0 < m; e0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = e0 + threadIdx.x;
        int32_t s = 0;
        if (e < m && rep[e] == (int32_t)e && off[e + 1] - off[e] <= kMedium) {   // larger: k_lg_emit
            s = size1[e];
            src_w[wid][lane] = off[e];
            const int64_t at = pos[e], id = new_id(at);
            dst_w[wid][lane] = new_off(at);
            off2[id] = new_off(at);
            const unsigned long long w = w64[e];
            if (w >= (1ull << 31)) atomicOr(err, ERR_UNSUPPORTED);
            nw2[id] = (int32_t)w;
        }
        int32_t incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        off33[lane] = incl - s;
        if (lane == 31) off33[32] = incl;
        __syncwarp();
        const int32_t total = off33[32];
        for (int32_t i0 = lane; i0 < total; i0 += 128) {   // four pins per lane in flight
            int32_t x[4];
            int64_t at[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t i = i0 + 32 * q;
                const int v = slot_in(off33, i < total ? i : 0);
                const int32_t k = i - off33[v];
                at[q] = dst_w[wid][v] + k;
                x[q] = i < total ? __ldcs(&a[src_w[wid][v] + k]) : 0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + 32 * q < total) pins2[at[q]] = x[q];
        }
        __syncwarp();
    }
}

__global__ void k_ct_project(const int32_t *map, int32_t n, const int32_t *coarse_part, int32_t *fine_part)
{
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
        fine_part[u] = coarse_part[map[u]];
}

std::array<void *, 5> coarse_arrays(const hgp_coarse *c) { return {c->net_off, c->pins, c->vw, c->nw, c->map}; }

}  // namespace

#define CT(x)                                   \
    do {                                        \
        e = (x);                                \
        if (e != cudaSuccess) goto done;        \
    } while (0)

extern "C" int hgp_contract(int32_t n, int32_t m, const int64_t *net_off, const int32_t *pins,
                            const int32_t *vertex_w, const int32_t *net_w, const int32_t *cluster,
                            void *cuda_stream, hgp_coarse **out)
{
    if (!out) return HGP_ERR_INVALID;
    *out = nullptr;
    if (n < 1 || m < 0 || !net_off || !cluster || (m > 0 && !pins)) return HGP_ERR_INVALID;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    hgp_coarse *c = new (std::nothrow) hgp_coarse;
    if (!c) return HGP_ERR_OOM;
    c->fine_n = n;
    c->stream = st;
    cudaGetDevice(&c->device);
    cudaError_t e = cudaSuccess;
    int rc = HGP_OK;
    int32_t *err = nullptr, *used = nullptr, *a = nullptr, *b = nullptr, *size1 = nullptr, *rep = nullptr;
    int32_t *left = nullptr, *lists = nullptr, *counts = nullptr;
    void *lg_scratch[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    int32_t n_large = 0;
    int64_t lg_tasks = 0;
    int sms = 1;
    int32_t *cid = nullptr, n2 = 0;
    int64_t *pos = nullptr;
    unsigned long long *w64 = nullptr, *key = nullptr, *nw64 = nullptr;
    unsigned long long *tab = nullptr;
    int64_t P = 0, m2 = 0, P2 = 0, end = 0;
    int32_t herr = 0;
    const int64_t mm = m > 0 ? m : 1;
    CT(cudaMemcpyAsync(&P, net_off + m, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CT(stream_wait(st));
    if (P < 0 || (m == 0 && P != 0)) { rc = HGP_ERR_INVALID; goto done; }
    if (P >= ((int64_t)1 << 31)) { rc = HGP_ERR_UNSUPPORTED; goto done; }
    CT(dev_alloc(reinterpret_cast<void **>(&err), sizeof(int32_t) * 2, st));
    CT(cudaMemsetAsync(err, 0, sizeof(int32_t) * 2, st));
    left = err + 1;
    k_ct_check<<<152 * 16, 256, 0, st>>>(net_off, pins, vertex_w, net_w, n, m, P, err);
    CT(cudaGetLastError());
    CT(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CT(stream_wait(st));
    if (herr) { rc = HGP_ERR_INVALID; goto done; }
    // (1) remap the used cluster ids
    CT(dev_alloc(reinterpret_cast<void **>(&used), sizeof(int32_t) * (size_t)n, st));
    CT(dev_alloc(reinterpret_cast<void **>(&cid), sizeof(int32_t) * ((size_t)n + 1), st));
    CT(cudaMemsetAsync(used, 0, sizeof(int32_t) * (size_t)n, st));
    k_ct_flag<<<grid_of(n, 256), 256, 0, st>>>(cluster, n, used, err);
    CT(cudaGetLastError());
    CT(scan_excl(used, n, cid, st));
    CT(cudaMemcpyAsync(&n2, cid + n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CT(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CT(stream_wait(st));
    if (herr) { rc = HGP_ERR_INVALID; goto done; }
    c->n = n2;
    // (2) map and cluster weights
    CT(dev_alloc(reinterpret_cast<void **>(&c->map), sizeof(int32_t) * (size_t)n, st));
    CT(dev_alloc(reinterpret_cast<void **>(&c->vw), sizeof(int32_t) * (size_t)n2, st));
    CT(dev_alloc(reinterpret_cast<void **>(&w64), sizeof(unsigned long long) * (size_t)n2, st));
    CT(cudaMemsetAsync(w64, 0, sizeof(unsigned long long) * (size_t)n2, st));
    k_ct_map<<<grid_of(n, 256), 256, 0, st>>>(cluster, n, cid, vertex_w, c->map, w64);
    k_ct_narrow<<<grid_of(n2, 256), 256, 0, st>>>(w64, n2, c->vw, err);
    CT(cudaGetLastError());
    // (3) per-net sort + dedupe
    CT(dev_alloc(reinterpret_cast<void **>(&a), sizeof(int32_t) * (size_t)(P > 0 ? P : 1), st));
    CT(dev_alloc(reinterpret_cast<void **>(&b), sizeof(int32_t) * (size_t)(P > 0 ? P : 1), st));
    CT(dev_alloc(reinterpret_cast<void **>(&size1), sizeof(int32_t) * (size_t)mm, st));
    CT(dev_alloc(reinterpret_cast<void **>(&key), sizeof(unsigned long long) * (size_t)mm, st));
    CT(dev_alloc(reinterpret_cast<void **>(&rep), sizeof(int32_t) * (size_t)mm, st));
    CT(dev_alloc(reinterpret_cast<void **>(&lists), sizeof(int32_t) * kClasses * (size_t)mm + 32, st));
    counts = lists + kClasses * mm;
    CT(cudaMemsetAsync(counts, 0, sizeof(int32_t) * (kClasses + 1), st));
    if (m > 0) {
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
        k_ct_tiny<<<grid_of(m, 256), 256, 0, st>>>(net_off, pins, m, c->map, a, size1, key, rep, lists, counts);
        k_ct_small<<<sms * 8, 256, 0, st>>>(net_off, pins, c->map, lists, counts, a, size1, key, rep);
        k_ct_mid<<<sms * 8, 256, 0, st>>>(net_off, pins, c->map, lists + mm, counts + 1, a, size1, key, rep);
        k_ct_medium<<<sms * 12, kCtaSort, 0, st>>>(net_off, pins, c->map, lists + 2 * mm, counts + 2, a, size1, key, rep);
        CT(cudaGetLastError());
        // nets of more than kMedium pins: chunk sorts, merge passes, de-duplication
        int32_t hcnt[kClasses] = {0, 0, 0, 0};
        CT(cudaMemcpyAsync(hcnt, counts, sizeof(int32_t) * kClasses, cudaMemcpyDeviceToHost, st));
        CT(stream_wait(st));
        n_large = hcnt[3];
        if (n_large > 0) {
            int32_t *chunks = nullptr;
            int64_t *cpre = nullptr;
            CT(dev_alloc(reinterpret_cast<void **>(&chunks), sizeof(int32_t) * ((size_t)n_large + 1), st));
            CT(dev_alloc(reinterpret_cast<void **>(&cpre), sizeof(int64_t) * ((size_t)n_large + 1), st));
            lg_scratch[0] = chunks;
            lg_scratch[1] = cpre;
            CT(cudaMemsetAsync(counts + kClasses, 0, sizeof(int32_t), st));
            k_lg_count<<<grid_of(n_large, 256), 256, 0, st>>>(net_off, lists + 3 * mm, counts + 3, chunks, counts + kClasses);
            CT(cudaGetLastError());
            CT(scan_excl(chunks, n_large, cpre, st));
            int64_t &tasks = lg_tasks;
            int32_t max_size = 0;
            CT(cudaMemcpyAsync(&tasks, cpre + n_large, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            CT(cudaMemcpyAsync(&max_size, counts + kClasses, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            CT(stream_wait(st));
            int32_t *distinct = nullptr;
            int64_t *pre = nullptr;
            unsigned long long *hsum = nullptr;
            CT(dev_alloc(reinterpret_cast<void **>(&distinct), sizeof(int32_t) * (size_t)tasks, st));
            lg_scratch[2] = distinct;
            CT(dev_alloc(reinterpret_cast<void **>(&pre), sizeof(int64_t) * ((size_t)tasks + 1), st));
            lg_scratch[3] = pre;
            CT(dev_alloc(reinterpret_cast<void **>(&hsum), sizeof(unsigned long long) * (size_t)n_large, st));
            lg_scratch[4] = hsum;
            CT(cudaMemsetAsync(distinct, 0, sizeof(int32_t) * (size_t)tasks, st));
            CT(cudaMemsetAsync(hsum, 0, sizeof(unsigned long long) * (size_t)n_large, st));
            const int32_t *list = lists + 3 * mm, *cnt = counts + 3;
            const int g = (int)std::min<int64_t>(tasks, (int64_t)sms * 12);
            // the sorted runs end up in b, the distinct values go to a
            k_lg_chunk<<<g, kCtaSort, 0, st>>>(net_off, pins, c->map, list, cnt, cpre, tasks, a, b);
            for (int pass = 0; ((int64_t)kMedium << pass) < max_size; ++pass)
                k_lg_merge<<<g, kLgThreads, 0, st>>>(net_off, list, cnt, cpre, tasks, a, b, pass);
            k_lg_distinct<<<g, kLgThreads, 0, st>>>(net_off, list, cnt, cpre, tasks, b, distinct, hsum);
            CT(cudaGetLastError());
            CT(scan_excl(distinct, tasks, pre, st));
            k_lg_compact<<<g, kLgThreads, 0, st>>>(net_off, list, cnt, cpre, tasks, b, pre, a);
            k_lg_done<<<grid_of(n_large, 256), 256, 0, st>>>(list, cnt, cpre, pre, hsum, size1, key, rep);
            CT(cudaGetLastError());
        }
    }
    // (4) identical nets
    if (m > 0) {
        uint64_t size = 1024;   // at most three quarters full
        while (3 * size < 4 * (uint64_t)m) size <<= 1;
        CT(dev_alloc(reinterpret_cast<void **>(&tab), sizeof(unsigned long long) * size, st));
        for (int round = 0;; ++round) {
            if (round >= 4096) { rc = HGP_ERR_INTERNAL; goto done; }
            int32_t hleft = 0;
            CT(cudaMemsetAsync(left, 0, sizeof(int32_t), st));
            CT(cudaMemsetAsync(tab, 0xFF, sizeof(unsigned long long) * size, st));
            k_ct_insert<<<grid_of(m, 256), 256, 0, st>>>(key, rep, m, tab, size - 1, err);
            k_ct_resolve<<<grid_of(m, 256), 256, 0, st>>>(net_off, a, size1, key, rep, m, tab, size - 1, left);
            CT(cudaGetLastError());
            CT(cudaMemcpyAsync(&hleft, left, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            CT(stream_wait(st));
            if (hleft == 0) break;
        }
    }
    // (5) representatives in original order, their weights and offsets
    if (m > 0) {
        const int64_t tiles = m / kScanTile + 1;   // covers indices 0..m
        CT(dev_alloc(reinterpret_cast<void **>(&pos), sizeof(int64_t) * ((size_t)m + 1 + 2 * (size_t)tiles + 1), st));
        CT(dev_alloc(reinterpret_cast<void **>(&nw64), sizeof(unsigned long long) * (size_t)m, st));
        int64_t *sums = pos + m + 1, *prefix = sums + tiles;
        k_ct_groups<<<(unsigned)tiles, kScanTile / kScanPer, 0, st>>>(rep, size1, net_w, m, nw64, sums);
        CT(cudaGetLastError());
        CT(scan_excl(sums, tiles, prefix, st));
        k_ct_places<<<(unsigned)tiles, kScanTile / kScanPer, 0, st>>>(rep, size1, net_w, m, prefix, nw64, pos);
        CT(cudaGetLastError());
        CT(cudaMemcpyAsync(&end, pos + m, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        CT(stream_wait(st));
        m2 = end >> 32;
        P2 = end & 0xffffffff;
    }
    c->m = (int32_t)m2;
    c->P = P2;
    CT(dev_alloc(reinterpret_cast<void **>(&c->net_off), sizeof(int64_t) * ((size_t)m2 + 1), st));
    CT(dev_alloc(reinterpret_cast<void **>(&c->pins), sizeof(int32_t) * (size_t)(P2 > 0 ? P2 : 1), st));
    CT(dev_alloc(reinterpret_cast<void **>(&c->nw), sizeof(int32_t) * (size_t)(m2 > 0 ? m2 : 1), st));
    CT(cudaMemcpyAsync(c->net_off + m2, &P2, sizeof(int64_t), cudaMemcpyHostToDevice, st));
    if (m > 0) {
        if (n_large > 0)
            k_lg_emit<<<(unsigned)std::min<int64_t>(lg_tasks, (int64_t)sms * 16), kLgThreads, 0, st>>>(
                net_off, a, size1, rep, pos, nw64, lists + 3 * mm, counts + 3, (const int64_t *)lg_scratch[1], lg_tasks,
                c->pins, c->net_off, c->nw, err);
        k_ct_emit<<<grid_of(m, 256), 256, 0, st>>>(net_off, a, size1, rep, pos, nw64, m, c->pins, c->net_off, c->nw, err);
        CT(cudaGetLastError());
    }
    CT(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CT(stream_wait(st));
    if (herr & ERR_UNSUPPORTED) rc = HGP_ERR_UNSUPPORTED;
    else if (herr) rc = HGP_ERR_INTERNAL;
done:
    if (err) pool_free(err, st);
    if (used) pool_free(used, st);
    if (cid) pool_free(cid, st);
    if (w64) pool_free(w64, st);
    if (a) pool_free(a, st);
    if (b) pool_free(b, st);
    if (size1) pool_free(size1, st);
    if (key) pool_free(key, st);
    if (rep) pool_free(rep, st);
    if (tab) pool_free(tab, st);
    if (lists) pool_free(lists, st);
    for (void *q : lg_scratch)
        if (q) pool_free(q, st);
    if (pos) pool_free(pos, st);
    if (nw64) pool_free(nw64, st);
    {
        const cudaError_t e2 = stream_wait(st);
        if (e == cudaSuccess) e = e2;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        rc = status_of(e);
    }
    if (rc != HGP_OK) {
        for (void *p : coarse_arrays(c)) dev_free(p, st);
        delete c;
        return rc;
    }
    *out = c;
    return HGP_OK;
}

extern "C" int hgp_coarse_get_sizes(const hgp_coarse *c, int32_t *n, int32_t *m, int64_t *num_pins)
{
    if (!c || !n || !m || !num_pins) return HGP_ERR_INVALID;
    *n = c->n;
    *m = c->m;
    *num_pins = c->P;
    return HGP_OK;
}

extern "C" int hgp_coarse_get_device_arrays(const hgp_coarse *c, const int64_t **net_off, const int32_t **pins,
                                            const int32_t **vertex_w, const int32_t **net_w, const int32_t **map)
{
    if (!c) return HGP_ERR_INVALID;
    if (net_off) *net_off = c->net_off;
    if (pins) *pins = c->pins;
    if (vertex_w) *vertex_w = c->vw;
    if (net_w) *net_w = c->nw;
    if (map) *map = c->map;
    return HGP_OK;
}

extern "C" int hgp_coarse_copy_to_host(const hgp_coarse *c, int64_t *net_off, int32_t *pins, int32_t *vertex_w,
                                       int32_t *net_w, int32_t *map)
{
    if (!c) return HGP_ERR_INVALID;
    cudaError_t e = cudaSuccess;
    if (net_off) e = cudaMemcpyAsync(net_off, c->net_off, sizeof(int64_t) * ((size_t)c->m + 1), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && pins && c->P > 0)
        e = cudaMemcpyAsync(pins, c->pins, sizeof(int32_t) * (size_t)c->P, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && vertex_w)
        e = cudaMemcpyAsync(vertex_w, c->vw, sizeof(int32_t) * (size_t)c->n, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && net_w && c->m > 0)
        e = cudaMemcpyAsync(net_w, c->nw, sizeof(int32_t) * (size_t)c->m, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && map)
        e = cudaMemcpyAsync(map, c->map, sizeof(int32_t) * (size_t)c->fine_n, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = stream_wait(c->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return HGP_OK;
}

extern "C" int hgp_coarse_project(const hgp_coarse *c, const int32_t *coarse_part, int32_t *fine_part)
{
    if (!c || !coarse_part || !fine_part) return HGP_ERR_INVALID;
    k_ct_project<<<grid_of(c->fine_n, 256), 256, 0, c->stream>>>(c->map, c->fine_n, coarse_part, fine_part);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = stream_wait(c->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return HGP_OK;
}

extern "C" void hgp_coarse_destroy(hgp_coarse *c)
{
    if (!c) return;
    // the arrays may be in use on any stream of their device: wait for that device, whichever is
    // current, and release them without the contraction's stream, which may be gone by now
    int now = 0;
    const bool other = cudaGetDevice(&now) == cudaSuccess && now != c->device;
    if (other) cudaSetDevice(c->device);
    // (a device that cannot be waited for, as during a stream capture, keeps them, as cudaFree would)
    if (cudaDeviceSynchronize() == cudaSuccess)
        for (void *p : coarse_arrays(c))   // on the default stream; cudaFree would not count them as given back
            if (p && cudaFreeAsync(p, nullptr) != cudaSuccess) cudaFree(p);
    if (other) cudaSetDevice(now);
    (void)cudaGetLastError();
    delete c;
}
