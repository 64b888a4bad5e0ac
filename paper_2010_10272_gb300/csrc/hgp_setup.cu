// libhgp: creation, validation, CSR transpose, state initialisation and getters.
//
// Setup builds, on the device, everything the refinement rounds read:
//   * the vertex -> incident nets CSR I(v) from the net -> pins CSR (Sec. 2; the paper
//     builds the same two adjacency arrays with prefix sums, Sec. 3.2);
//   * Phi(e, i) from the partition (Sec. 2 / Sec. 5.1), Lambda(e), S1(e) and omega(e) in the
//     per-net record, the block weights and the (lambda-1) objective (Sec. 2).
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <new>
#include <type_traits>

#include "hgp_host.cuh"

using namespace hgp;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kDefaultSmem = 32 << 10;   // dynamic shared memory beside the static arrays (48 KB in all)

// ------------------------------------------------------------------ prefix sums (int32)
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanChunk = kScanThreads * kScanItems;

__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t *warp_tot, int32_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int32_t t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
        int32_t s = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(kFull, s, o);
            if (lane >= o) s += y;
        }
        warp_tot[lane] = s - t;
        if (lane == 31) *total = s;
    }
    __syncthreads();
    const int32_t r = warp_tot[wid] + x - v;
    __syncthreads();
    return r;
}

__global__ void k_scan_reduce(const int32_t *in, int64_t count, int32_t *sums)
{
    __shared__ int32_t wt[32];
    __shared__ int32_t tot;
    const int64_t base = (int64_t)blockIdx.x * kScanChunk + (int64_t)threadIdx.x * kScanItems;
    int32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i < count) s += in[base + i];
    block_exclusive_scan(s, wt, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(int32_t *sums, int64_t nb)
{
    __shared__ int32_t wt[32];
    __shared__ int32_t tot;
    int32_t carry = 0;
    for (int64_t b = 0; b < nb; b += kScanThreads) {
        const int64_t i = b + threadIdx.x;
        const int32_t v = i < nb ? sums[i] : 0;
        const int32_t ex = block_exclusive_scan(v, wt, &tot);
        if (i < nb) sums[i] = carry + ex;
        carry += tot;
        __syncthreads();
    }
}

__global__ void k_scan_final(const int32_t *in, int32_t *out, int64_t count, const int32_t *sums)
{
    __shared__ int32_t wt[32];
    __shared__ int32_t tot;
    const int64_t base = (int64_t)blockIdx.x * kScanChunk + (int64_t)threadIdx.x * kScanItems;
    int32_t v[kScanItems];
    int32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = base + i < count ? in[base + i] : 0;
        s += v[i];
    }
    int32_t run = sums[blockIdx.x] + block_exclusive_scan(s, wt, &tot);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        if (base + i < count) out[base + i] = run;
        run += v[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[count] = sums[blockIdx.x] + tot;
}

// ------------------------------------------------------------------ validation
// Warp-wide: the pins of nets e0 .. e0 + 31 (clipped to e_hi) are contiguous; off33 receives
// their exclusive offsets inside that run (off33[32] = its length) and the run's first pin index
// is returned.  Lanes then walk the run flattened, one pin each, with pin_net to find the net.
__device__ __forceinline__ int32_t net_group(const int32_t *off, int64_t e0, int64_t e_hi, int32_t *off33,
                                             int32_t &sz_lane)
{
    const int lane = threadIdx.x & 31;
    const int64_t e = e0 + lane;
    sz_lane = e < e_hi ? off[e + 1] - off[e] : 0;
    int32_t incl = sz_lane;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    off33[lane] = incl - sz_lane;
    if (lane == 31) off33[32] = incl;
    __syncwarp();
    return off[e0];
}

// slot of the net holding run position i: the largest s with off33[s] <= i (empty nets skipped)
__device__ __forceinline__ int pin_net(const int32_t *off33, int32_t i)
{
    int lo = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1)
        if (off33[lo + step] <= i) lo += step;
    return lo;
}

// pins in [0, n) and strictly increasing inside every net; the largest net size.  Runs after
// k_check_inputs and does nothing if that found an error.  Whatever the nets' sizes, every thread
// walks pins and nets with one stride: the steps of the whole pin array that do not increase are
// counted, and so are those at the first pin of a net, which are allowed; the nets are increasing
// exactly if the two counts are equal.  (A warp per 32 nets spent the time of the longest net:
// power-law 5M, nets of up to 100,000 pins, 676 -> 50 us.)  The last CTA compares the counts.
__global__ void __launch_bounds__(256) k_check_pins(const int32_t *off, const int32_t *pins, int32_t m, int32_t n,
                                                    int64_t P, int32_t *err, int32_t *max_size,
                                                    unsigned long long *acc)
{
    __shared__ long long diff_s;
    __shared__ int32_t max_s;
    // the offsets may only be trusted when the checks before found nothing (they ran to
    // completion earlier on the same stream, so their flag is final)
    if (*reinterpret_cast<volatile int32_t *>(err) & ERR_INVALID) return;
    if (threadIdx.x == 0) {
        diff_s = 0;
        max_s = 0;
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool bad = false;
    int32_t diff = 0, local_max = 0;
    for (int64_t j0 = t0; j0 < P; j0 += 4 * stride) {   // four pins (and predecessors) per thread in flight
        int32_t v[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t j = j0 + i * stride;
            v[i] = j < P ? pins[j] : 0;
            q[i] = j < P && j > 0 ? pins[j - 1] : -1;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (j0 + i * stride >= P) continue;
            if (v[i] < 0 || v[i] >= n) bad = true;
            if (j0 + i * stride > 0) diff += q[i] >= v[i];
        }
    }
    for (int64_t e = t0; e < m; e += stride) {
        const int32_t b = off[e], sz = off[e + 1] - b;
        local_max = max(local_max, sz);
        if (sz > 0 && b > 0) diff -= pins[b - 1] >= pins[b];
    }
    if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(err, ERR_INVALID);
    diff = __reduce_add_sync(kFull, diff);
    local_max = (int32_t)__reduce_max_sync(kFull, (unsigned)local_max);
    if ((threadIdx.x & 31) == 0) {
        if (diff) atomicAdd(reinterpret_cast<unsigned long long *>(&diff_s), (unsigned long long)(long long)diff);
        atomicMax(&max_s, local_max);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (diff_s) atomicAdd(&acc[ACC_OBJ], (unsigned long long)diff_s);
        atomicMax(max_size, max_s);
        __threadfence();
        if (atomicAdd(&acc[ACC_DONE], 1ull) == gridDim.x - 1) {
            __threadfence();
            if (__ldcg(&acc[ACC_OBJ]) != 0) atomicOr(err, ERR_INVALID);
            acc[ACC_OBJ] = 0;
            acc[ACC_DONE] = 0;
        }
    }
}

// ------------------------------------------------------------------ internal net order
// Nets are relabelled by size class, the largest class first and by input id inside a class.
// On skewed instances a few large nets take most record gathers (each incidence reads its net's
// record); stored first, their records and Phi rows share L2 lines and stay resident there.
// Gains, objective and every move are sums over nets, so results do not depend on the order.
// Nets of at most 4 pins (Dev::tiny) come last, a class per size.
constexpr int kNrRanks = 34;        // rank 0: the largest size class (2^30 pins and up)
constexpr int kNrTiny = 30;         // rank of the nets of 4 pins
constexpr int kNrThreads = 256;

__device__ __forceinline__ int nr_rank(int32_t size)
{
    // sizes [2^c, 2^(c+1)) -> 31 - c; 5..7 -> 29; 4, 3, 2, at most 1 -> 30 .. 33
    return size > 4 ? __clz(size) : kNrTiny + 4 - max(size, 1);
}

// per CTA (a contiguous chunk of per_cta nets): nets per rank, written rank-major so that one
// exclusive scan yields every (rank, CTA) base position
__global__ void __launch_bounds__(kNrThreads) k_nr_count(const int32_t *off, int32_t m, int32_t per_cta,
                                                         int32_t *cnt)
{
    __shared__ int32_t c[kNrRanks];
    if (threadIdx.x < kNrRanks) c[threadIdx.x] = 0;
    __syncthreads();
    const int64_t lo = (int64_t)blockIdx.x * per_cta;
    const int64_t hi = min((int64_t)m, lo + per_cta);
    for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) atomicAdd(&c[nr_rank(off[e + 1] - off[e])], 1);
    __syncthreads();
    if (threadIdx.x < kNrRanks) cnt[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = c[threadIdx.x];
}

// same chunks: internal id of every net (stable inside a rank), the sizes in internal order, and where
// the pins of the large-net prefix [0, m_big) come from
__global__ void __launch_bounds__(kNrThreads) k_nr_place(const int32_t *off, int32_t m, int32_t per_cta,
                                                         const int32_t *base, int32_t *perm, int32_t *size_int,
                                                         int32_t m_big, int32_t *src_big)
{
    constexpr int W = kNrThreads / 32;
    __shared__ int32_t run[kNrRanks];
    __shared__ int32_t wc[W][kNrRanks];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x < kNrRanks) run[threadIdx.x] = base[(int64_t)threadIdx.x * gridDim.x + blockIdx.x];
    const int64_t lo = (int64_t)blockIdx.x * per_cta;
    const int64_t hi = min((int64_t)m, lo + per_cta);
    for (int64_t c0 = lo; c0 < hi; c0 += kNrThreads) {
        for (int i = threadIdx.x; i < W * kNrRanks; i += kNrThreads) (&wc[0][0])[i] = 0;
        __syncthreads();
        const int64_t e = c0 + threadIdx.x;
        const bool valid = e < hi;
        const int32_t size = valid ? off[e + 1] - off[e] : 0;
        const int rk = valid ? nr_rank(size) : kNrRanks;
        const unsigned peers = __match_any_sync(kFull, rk);
        const int below = __popc(peers & ((1u << lane) - 1));
        if (valid && below == 0) wc[wid][rk] = __popc(peers);
        __syncthreads();
        if (valid) {
            int32_t pos = run[rk] + below;
            for (int w = 0; w < wid; ++w) pos += wc[w][rk];
            perm[e] = pos;
            size_int[pos] = size;
            if (pos < m_big) src_big[pos] = off[e];
        }
        __syncthreads();
        if (threadIdx.x < kNrRanks) {
            int32_t t = 0;
            for (int w = 0; w < W; ++w) t += wc[w][threadIdx.x];
            run[threadIdx.x] += t;
        }
        __syncthreads();
    }
}

// pins (and net weights) into internal order; a warp copies the pins of 32 consecutive input
// nets, reading them as one coalesced run but for the nets of the large-net prefix, whose pins
// k_nr_pins_big copies (power-law 5M: 640 us with them -> 74 + 37 us)
__global__ void __launch_bounds__(256) k_nr_pins(const int32_t *off, const int32_t *pins, const int32_t *nw,
                                                 int32_t m, int32_t m_big, const int32_t *perm,
                                                 const int32_t *off_int, int32_t *pins_int, int32_t *nw_int)
{
    __shared__ int32_t off33_w[8][33];
    __shared__ int32_t dst_w[8][32], src_w[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *off33 = off33_w[wid];
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t e0 = ((int64_t)blockIdx.x * 8 + wid) * 32; e0 < m; e0 += warps * 32) {
        const int64_t e = e0 + lane;
        int32_t src = 0, sz = 0;
        if (e < m) {
            src = off[e];
            sz = off[e + 1] - src;
            const int32_t q = perm[e];
            dst_w[wid][lane] = off_int[q];
            if (nw) nw_int[q] = nw[e];
            if (q < m_big) sz = 0;
        }
        int32_t incl = sz;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        off33[lane] = incl - sz;
        src_w[wid][lane] = src;
        if (lane == 31) off33[32] = incl;
        __syncwarp();
        const int32_t total = off33[32];
        for (int32_t i0 = lane; i0 < total; i0 += 128) {   // four loads in flight per lane
            int32_t vq[4], at[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int32_t i = i0 + 32 * q;
                const int sl = i < total ? pin_net(off33, i) : 0;
                vq[q] = i < total ? __ldcs(&pins[src_w[wid][sl] + (i - off33[sl])]) : 0;
                at[q] = dst_w[wid][sl] + (i - off33[sl]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + 32 * q < total) pins_int[at[q]] = vq[q];
        }
        __syncwarp();
    }
}

// the pins of the large-net prefix into internal order: a CTA per kBigChunk of them, whose nets'
// offsets and sources sit in shared memory
constexpr int kBigChunk = 8192;
constexpr int32_t kBigNet = 256;                   // nets of the prefix have at least this many pins
constexpr int kBigWin = kBigChunk / kBigNet + 3;   // offsets of the nets a chunk overlaps, + 1

// the net of the prefix that holds pin p0: the largest e < m_big with off[e] <= p0
__device__ __forceinline__ int32_t net_of_pin(const int32_t *off, int32_t m_big, int32_t p0)
{
    int32_t lo = 0, hi = m_big - 1;
    while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (off[mid] <= p0) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int win_slot(const int32_t *win, int32_t j)
{
    int sl = 0;   // the largest slot with win[sl] <= j
#pragma unroll
    for (int step = 32; step; step >>= 1)
        if (sl + step < kBigWin && win[sl + step] <= j) sl += step;
    return sl;
}

__global__ void __launch_bounds__(1024) k_nr_pins_big(const int32_t *off_int, const int32_t *src_big, const int32_t *pins,
                                                      int32_t m_big, int32_t *pins_int)
{
    __shared__ int32_t win[kBigWin], src[kBigWin];
    __shared__ int32_t first;
    const int32_t p0 = blockIdx.x * kBigChunk;
    const int32_t len = chunk_length(p0, off_int[m_big], kBigChunk);
    if (threadIdx.x == 0) first = net_of_pin(off_int, m_big, p0);
    __syncthreads();
    if (threadIdx.x < kBigWin) {
        win[threadIdx.x] = off_int[min(m_big, first + (int32_t)threadIdx.x)];
        src[threadIdx.x] = src_big[min(m_big - 1, first + (int32_t)threadIdx.x)];
    }
    __syncthreads();
#pragma unroll 4
    for (int32_t i = threadIdx.x; i < len; i += blockDim.x) {
        const int32_t j = p0 + i;
        const int sl = win_slot(win, j);
        pins_int[j] = pins[src[sl] + (j - win[sl])];
    }
}

// Creation queues its kernels behind the input checks without waiting for their verdict (for
// instances whose net sizes the host reads itself, see create_impl): every kernel that indexes
// by a pin, a vertex id or a block then returns at once when the checks flagged the input, and
// the creation reports HGP_ERR_INVALID at its one read-back.  guard: the creation's error flag,
// or nullptr outside creation.
__device__ __forceinline__ bool input_invalid(const int32_t *guard)
{
    return guard && (*reinterpret_cast<const volatile int32_t *>(guard) & ERR_INVALID) != 0;
}

// Per-CTA block weights: counts of unit weights (32-bit, native shared atomics), or sums.
struct BlockSums {
    unsigned long long w[64];
    uint32_t c[64];
};
constexpr int kFewBlocks = 8;   // up to this k a warp's lanes share blocks: one update per distinct block

__device__ __forceinline__ void add_block_weights(BlockSums &b, bool ok, int blk, int32_t k, const int32_t *vw, int64_t v)
{
    if (!vw && k > kFewBlocks) {
        if (ok) atomicAdd(&b.c[blk], 1u);
        return;
    }
    const unsigned mask = __ballot_sync(kFull, ok);
    if (!ok) return;
    const unsigned peers = __match_any_sync(mask, blk);
    const bool lead = (int)(threadIdx.x & 31) == __ffs(peers) - 1;
    if (!vw) {
        if (lead) atomicAdd(&b.c[blk], (uint32_t)__popc(peers));
        return;
    }
    // two halves: 32 sums of either fit 32 bits
    const uint32_t x = (uint32_t)vw[v];
    const unsigned long long sum = (unsigned long long)__reduce_add_sync(peers, x & 0xFFFFu) +
                                   ((unsigned long long)__reduce_add_sync(peers, x >> 16) << 16);
    if (lead) atomicAdd(&b.w[blk], sum);
}

__device__ __forceinline__ void clear_block_weights(BlockSums &b)
{
    if (threadIdx.x < 64) {
        b.w[threadIdx.x] = 0;
        b.c[threadIdx.x] = 0;
    }
    __syncthreads();
}

__device__ __forceinline__ void flush_block_weights(const BlockSums &b, int32_t k, unsigned long long *acc)
{
    __syncthreads();
    if (threadIdx.x < k) {
        const unsigned long long v = b.w[threadIdx.x] + b.c[threadIdx.x];
        if (v) atomicAdd(&acc[ACC_BW + threadIdx.x], v);
    }
}

// Stores the valid entries of a partition as 1-byte Pi and adds their vertices' weights to w (shared,
// cleared); returns whether an entry was out of range.
__device__ __forceinline__ bool stage_partition(const int32_t *part_in, int32_t n, int32_t k, const int32_t *vw,
                                                uint8_t *part, BlockSums &w)
{
    bool bad = false;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); v0 < n; v0 += 4 * stride) {
        int32_t p[4];   // four entries per lane in flight
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t v = v0 + q * stride + (threadIdx.x & 31);
            p[q] = v < n ? __ldcs(&part_in[v]) : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t v = v0 + q * stride + (threadIdx.x & 31);
            const bool in = p[q] >= 0 && p[q] < k, ok = v < n && in;
            if (!in) bad = true;
            if (ok) part[v] = (uint8_t)p[q];
            add_block_weights(w, ok, p[q], k, vw, v);
        }
    }
    return bad;
}

// A new partition: range check, 1-byte Pi and block weights in one pass over it.
__global__ void __launch_bounds__(256) k_stage_partition(const int32_t *part_in, int32_t n, int32_t k, const int32_t *vw,
                                                         uint8_t *part, unsigned long long *acc, int32_t *err)
{
    __shared__ BlockSums w;
    clear_block_weights(w);
    const bool bad = stage_partition(part_in, n, k, vw, part, w);
    if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(err, ERR_INVALID);
    flush_block_weights(w, k, acc);
}

// The creation's checks of the offsets (converted to int32 on the way), the net and vertex
// weights and the partition in one launch; the partition is stored and weighed at the same time.
__global__ void __launch_bounds__(256) k_check_inputs(const int64_t *off64, int32_t *off32, int32_t m, int64_t P,
                                                      const int32_t *nw, const int32_t *vw, const int32_t *part_in,
                                                      int32_t n, int32_t k, uint8_t *part, unsigned long long *acc,
                                                      int32_t *err)
{
    __shared__ BlockSums w;
    clear_block_weights(w);
    bool bad = false;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t e = t0; e <= m; e += stride) {
        const int64_t a = off64[e];
        if ((e == 0 && a != 0) || (e == m && a != P) || a < 0 || a > P) bad = true;
        if (e < m && off64[e + 1] < a) bad = true;
        if (e < m && nw && nw[e] < 1) bad = true;
        off32[e] = (int32_t)(a < 0 ? 0 : (a > P ? P : a));
    }
    if (vw)
        for (int64_t v = t0; v < n; v += stride)
            if (vw[v] < 1) bad = true;
    if (stage_partition(part_in, n, k, vw, part, w)) bad = true;
    if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(err, ERR_INVALID);
    flush_block_weights(w, k, acc);
}

// ------------------------------------------------------------------ per-vertex net weight
// W(u) = sum of incident net weights must stay below 2^31 (int32 gain arithmetic); kept in vnw
// (weighted nets) for the gain step
__global__ void k_vertex_netweight(const int32_t *vtx_off, const int32_t *inc, const int32_t *nw,
                                   int32_t n, int32_t *vnw, int32_t *err, unsigned long long *max_w)
{
    if (input_invalid(err)) return;
    unsigned long long local = 0;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        int64_t s = 0;
        for (int32_t j = vtx_off[v]; j < vtx_off[v + 1]; ++j) s += nw ? nw[inc[j] & kNetMask] : 1;
        if (s >= (int64_t)1 << 31) atomicOr(err, ERR_UNSUPPORTED);
        if (vnw) vnw[v] = (int32_t)s;
        local = max(local, (unsigned long long)s);
    }
    for (int o = 16; o; o >>= 1) local = max(local, __shfl_xor_sync(kFull, local, o));
    if ((threadIdx.x & 31) == 0) atomicMax(max_w, local);
}

// ------------------------------------------------------------------ transpose (net -> vertex)
// Direct form, for instances whose vertex counters fit in L2: degrees by atomic increments,
// an exclusive scan into vtx_off, then every pin takes the next slot of its vertex (warp per
// net) and stores the net id with the wide flag.
constexpr int32_t kTpDirectMaxN = 1 << 21;
// nets are stored in internal (size class) order from this many nets on, when the largest net
// has at least kReorderSkew times the average size: below that count their records fit in L2
// whatever the order, and without large nets no small set of records takes most gathers (on
// near-uniform sizes the relabelling only adds creation time)
constexpr int32_t kReorderMinNets = 1 << 20;
constexpr int64_t kReorderSkew = 8;
// host inputs with fewer nets than this: the host reads the net sizes (see create_impl)
constexpr int32_t kHostSizesMaxNets = 1 << 20;
// device inputs with fewer nets than this carve their buffers from one allocation, too (about 30 pool
// calls at creation otherwise: 256 handles of 1k to 200k vertices 900 -> 55-154 ms)
constexpr int32_t kDeviceArenaMaxNets = 1 << 18;
// what such a handle may keep of its creation's scratch and as unused room in Phi.  Given back by all of
// 256 handles, the holes between them made every later call that waits 5 us longer (set_partition 29 ->
// 35 us); kept by handles of many vertices it was 8 bytes a vertex.
constexpr int64_t kKeptSpare = 8 << 20;
// in internal order, nets of at least kBigNet pins (a prefix) get their own CTAs at creation and
// initialisation (a power of two: size classes are powers of two)

__global__ void k_degrees(const int32_t *pins, int64_t P, int32_t *deg, const int32_t *guard)
{
    if (input_invalid(guard)) return;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P;
         j += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&deg[pins[j]], 1);
}

__global__ void k_scatter(const int32_t *off, const int32_t *pins, int32_t m, int32_t narrow_max, int32_t *fill,
                          int32_t *inc, const int32_t *guard)
{
    if (input_invalid(guard)) return;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; e < m; e += warps) {
        const int32_t b = off[e], end = off[e + 1];
        const int32_t ef = (int32_t)((uint32_t)e | (end - b > narrow_max ? kWideFlag : 0u));
        for (int64_t j = (int64_t)b + lane; j < end; j += 32) {
            const int32_t pos = atomicAdd(&fill[pins[j]], 1);
            inc[pos] = ef;
        }
    }
}

// Bucketed form, for large instances:
// vertices are grouped into buckets of 2^bshift consecutive ids (at most
// kTpMaxBuckets buckets).  k_tp_hist counts the pins per bucket; k_tp_scatter writes every pin
// as a (vertex, net | wide flag) pair into its bucket's region, reserving one range per (CTA,
// bucket) with a single global atomic; k_tp_place, a CTA per bucket, counts the degrees of its
// vertices, scans them into vtx_off and places the nets into inc.  Every step but the pair
// scatter stays inside one bucket's few hundred KB, so the random accesses hit L2.
constexpr int kTpMaxBuckets = 4096;
constexpr int kTpShift = 14;             // 16384 vertices per bucket, unless that gives too few
constexpr int kTpMinShift = 8;           // buckets for the GPU (small instances) or too many
constexpr int kTpSmemShift = 14;         // buckets up to this size count in shared memory
constexpr int kTpMinCtas = 608;          // target buckets and CTAs per launch (4 per SM)
constexpr int kTpThreads = 512;
// pins per scatter CTA, at most: every CTA reserves a range in every bucket.  Cut by pins, not by
// nets: in internal order 2048 nets are 6,000 pins or 400,000, and the launch took as long as
// the latter (power-law 5M 779 -> 351 us, 50M 5.85 -> 5.0 ms)
constexpr int kTpMaxPins = 32768, kTpMinPins = 4096;

__global__ void __launch_bounds__(256) k_tp_hist(const int32_t *pins, int64_t P, int bshift, int32_t nb,
                                                 int32_t *bucket_cnt, const int32_t *guard)
{
    if (input_invalid(guard)) return;
    __shared__ int32_t h[kTpMaxBuckets];
    for (int i = threadIdx.x; i < nb; i += blockDim.x) h[i] = 0;
    __syncthreads();
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < P; j += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&h[pins[j] >> bshift], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x)
        if (h[i]) atomicAdd(&bucket_cnt[i], h[i]);
}

// the first net e in [lo, hi] with off[e] >= p (hi if there is none before it)
__device__ __forceinline__ int32_t first_net_at(const int32_t *off, int32_t lo, int32_t hi, int32_t p)
{
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if (off[mid] >= p) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// CTA per per_cta pins: the nets from e_begin on that start there.  Pass 0 counts their pins per
// bucket, then one range per bucket is reserved, pass 1 writes the pairs.  A warp walks the pins of
// 32 nets at once (coalesced).
__global__ void __launch_bounds__(kTpThreads) k_tp_scatter(const int32_t *off, const int32_t *pins, int32_t m,
                                                    int32_t e_begin, int bshift, int32_t nb, int32_t narrow_max,
                                                    int32_t per_cta, int32_t *bucket_cur, unsigned long long *pairs,
                                                    const int32_t *guard)
{
    if (input_invalid(guard)) return;
    constexpr int kW = kTpThreads / 32;
    __shared__ int32_t cur[kTpMaxBuckets];
    __shared__ int32_t off33_w[kW][33];
    __shared__ int32_t bound[2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *off33 = off33_w[wid];
    if (threadIdx.x < 2) {
        const int64_t p = off[e_begin] + ((int64_t)blockIdx.x + threadIdx.x) * per_cta;
        bound[threadIdx.x] = p > off[m] ? m : first_net_at(off, e_begin, m, (int32_t)p);
    }
    for (int i = threadIdx.x; i < nb; i += blockDim.x) cur[i] = 0;
    __syncthreads();
    const int64_t e_lo = bound[0], e_hi = bound[1];
    auto walk = [&](auto each) {   // each(pin, net, whether wide)
        for (int64_t e0 = e_lo + 32 * wid; e0 < e_hi; e0 += 32 * kW) {
            int32_t sz;
            const int32_t base = net_group(off, e0, e_hi, off33, sz);
            const int32_t total = off33[32];
            // four pins per lane are loaded before any is used (their latencies overlap)
            for (int32_t i0 = lane; i0 < total; i0 += 128) {
                int32_t vq[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) vq[q] = i0 + 32 * q < total ? pins[base + i0 + 32 * q] : -1;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (vq[q] >= 0) each(vq[q], e0, i0 + 32 * q);
            }
            __syncwarp();
        }
    };
    walk([&](int32_t v, int64_t, int32_t) { atomicAdd(&cur[v >> bshift], 1); });   // no old value: a reduction
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const int32_t c = cur[i];
        cur[i] = c ? atomicAdd(&bucket_cur[i], c) : 0;
    }
    __syncthreads();
    walk([&](int32_t v, int64_t e0, int32_t i) {
        const int32_t pos = atomicAdd(&cur[v >> bshift], 1);
        const int sl = pin_net(off33, i);
        const uint32_t ef = (uint32_t)(e0 + sl) | (off33[sl + 1] - off33[sl] > narrow_max ? kWideFlag : 0u);
        pairs[pos] = ((unsigned long long)(uint32_t)v << 32) | ef;
    });
}

// The pins of the large-net prefix [0, m_big) of the internal order (nets of at least kBigNet
// pins), split into chunks of kBigChunk pins, one CTA each, so that no CTA takes many large
// nets.  Same two passes as k_tp_scatter.
__global__ void __launch_bounds__(kTpThreads) k_tp_scatter_big(const int32_t *off, const int32_t *pins, int32_t m_big,
                                                               int bshift, int32_t nb, int32_t narrow_max,
                                                               int32_t *bucket_cur, unsigned long long *pairs,
                                                               const int32_t *guard)
{
    if (input_invalid(guard)) return;
    __shared__ int32_t cur[kTpMaxBuckets];
    __shared__ int32_t win[kBigWin];
    __shared__ int32_t first;
    const int32_t p0 = blockIdx.x * kBigChunk;
    const int32_t len = chunk_length(p0, off[m_big], kBigChunk);
    if (threadIdx.x == 0) first = net_of_pin(off, m_big, p0);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) cur[i] = 0;
    __syncthreads();
    const int32_t e_f = first;
    if (threadIdx.x < kBigWin) win[threadIdx.x] = off[min(m_big, e_f + (int32_t)threadIdx.x)];
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
        for (int32_t i = threadIdx.x; i < len; i += blockDim.x) {
            const int32_t j = p0 + i;
            const int32_t v = pins[j];
            const int32_t pos = atomicAdd(&cur[v >> bshift], 1);
            if (pass == 1) {
                const int sl = win_slot(win, j);
                const uint32_t ef = (uint32_t)(e_f + sl) | (win[sl + 1] - win[sl] > narrow_max ? kWideFlag : 0u);
                pairs[pos] = ((unsigned long long)(uint32_t)v << 32) | ef;
            }
        }
        __syncthreads();
        if (pass == 0) {
            for (int i = threadIdx.x; i < nb; i += blockDim.x) {
                const int32_t c = cur[i];
                cur[i] = c ? atomicAdd(&bucket_cur[i], c) : 0;
            }
            __syncthreads();
        }
    }
}

// CTA per bucket: degrees, their exclusive prefix (from the bucket's first pair position) into
// vtx_off, then the nets of the bucket's pairs into inc.  SMEM: the bucket's counters live in
// shared memory (buckets of at most 2^kTpSmemShift vertices); otherwise in cursor (zeroed
// int32[n], global).
constexpr int kTpPlaceBatch = 8;

template <bool SMEM>
__global__ void __launch_bounds__(1024) k_tp_place(const unsigned long long *pairs, const int32_t *bucket_off,
                                                   int bshift, int32_t n, int32_t nb, int32_t *cursor,
                                                   int32_t *vtx_off, int32_t *inc, const int32_t *guard)
{
    if (input_invalid(guard)) return;
    __shared__ int32_t wt[32];
    __shared__ int32_t tot;
    extern __shared__ int32_t sc[];
    const int32_t bkt = blockIdx.x;
    const int64_t v0 = (int64_t)bkt << bshift;
    const int64_t v1 = min((int64_t)n, v0 + ((int64_t)1 << bshift));
    const int32_t p0 = bucket_off[bkt], p1 = bucket_off[bkt + 1];
    int32_t *cnt = SMEM ? sc : cursor + v0;          // indexed by v - v0
    if (SMEM)
        for (int64_t i = threadIdx.x; i < v1 - v0; i += blockDim.x) sc[i] = 0;
    __syncthreads();
    // kTpPlaceBatch pairs per thread are loaded before any is used (the loads' latencies overlap)
    const int32_t step = (int32_t)blockDim.x * kTpPlaceBatch;
    for (int64_t i0 = (int64_t)p0 + threadIdx.x; i0 < p1; i0 += step) {
        unsigned long long pr[kTpPlaceBatch];
#pragma unroll
        for (int q = 0; q < kTpPlaceBatch; ++q) {
            const int64_t i = i0 + q * (int32_t)blockDim.x;
            pr[q] = i < p1 ? pairs[i] : ~0ull;            // read again below: keep in L2
        }
#pragma unroll
        for (int q = 0; q < kTpPlaceBatch; ++q)
            if (pr[q] != ~0ull) atomicAdd(&cnt[(int32_t)(pr[q] >> 32) - v0], 1);
    }
    __syncthreads();
    int32_t carry = p0;
    for (int64_t base = v0; base < v1; base += blockDim.x) {
        const int64_t v = base + threadIdx.x;
        const int32_t dv = v < v1 ? (SMEM ? sc[v - v0] : __ldcg(&cnt[v - v0])) : 0;
        const int32_t ex = block_exclusive_scan(dv, wt, &tot);
        if (v < v1) {
            vtx_off[v] = carry + ex;
            cnt[v - v0] = carry + ex;
        }
        carry += tot;
    }
    if (bkt == nb - 1 && threadIdx.x == 0) vtx_off[n] = p1;
    __syncthreads();
    for (int64_t i0 = (int64_t)p0 + threadIdx.x; i0 < p1; i0 += step) {
        unsigned long long pr[kTpPlaceBatch];
#pragma unroll
        for (int q = 0; q < kTpPlaceBatch; ++q) {
            const int64_t i = i0 + q * (int32_t)blockDim.x;
            pr[q] = i < p1 ? __ldcs(&pairs[i]) : ~0ull;
        }
#pragma unroll
        for (int q = 0; q < kTpPlaceBatch; ++q) {
            if (pr[q] == ~0ull) continue;
            const int32_t pos = atomicAdd(&cnt[(int32_t)(pr[q] >> 32) - v0], 1);
            inc[pos] = (int32_t)(uint32_t)pr[q];
        }
    }
}

__global__ void k_wide_flags(const int32_t *off, int32_t m, int32_t narrow_max, int32_t *flags)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x)
        flags[e] = (off[e + 1] - off[e]) > narrow_max ? 1 : 0;
}

// ------------------------------------------------------------------ state initialisation
// Phi(e, .) counted from the partition, the Phi rows, the records (Lambda, S1, omega, stamp) and the
// objective sum (lambda(e) - 1) * omega(e).
constexpr int kInitWarps = 8;
constexpr int32_t kInitBig = 2048;   // larger nets (or beyond a narrow entry) take a whole CTA

// streaming stores: the table and the records exceed L2, where the partition has to stay
template <typename Rec>
__device__ __forceinline__ void write_record(const Dev &d, int64_t e, uint64_t lam, uint64_t s1, int32_t wf)
{
    uint4 *rec = reinterpret_cast<uint4 *>(reinterpret_cast<Rec *>(d.rec) + e);
    if constexpr (sizeof(Rec) == 16) {
        __stcs(rec, make_uint4((uint32_t)s1, (uint32_t)lam, (uint32_t)wf, (uint32_t)(kNever * 2)));
    } else {
        __stcs(rec, make_uint4((uint32_t)s1, (uint32_t)(s1 >> 32), (uint32_t)lam, (uint32_t)(lam >> 32)));
        __stcs(rec + 1, make_uint4((uint32_t)wf, (uint32_t)(kNever * 2), 0u, 0u));
    }
}

__device__ __forceinline__ int32_t narrow_max_of(const Dev &d)
{
    return d.phi_w == 1 ? 255 : (d.phi_w == 2 ? 65535 : 0x7fffffff);
}

// k_init_big: nets of at least kHugeNet pins take CTAs of 1024 threads (the largest net's walk is as
// long as the launch), the others of 256 (power-law 5M: 250 us with 256 for all -> 74 + 32)
constexpr int32_t kHugeNet = 4096;

// One net, by the whole CTA (at least 64 threads); cnt: 64 shared counters.  Returns the net's objective
// term in thread 0.
template <typename Rec>
__device__ __forceinline__ long long init_net_cta(const Dev &d, const uint8_t *part, int64_t e, int32_t *cnt)
{
    const int lane = threadIdx.x & 31;
    const int w = d.phi_w;
    long long obj = 0;
    if (threadIdx.x < 64) cnt[threadIdx.x] = 0;
    __syncthreads();
    const int32_t b = d.net_off[e], sz = d.net_off[e + 1] - b;
    for (int32_t j0 = 0; j0 < sz; j0 += 4 * (int32_t)blockDim.x) {
        int blk[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // four pins per thread in flight
            const int32_t j = j0 + q * (int32_t)blockDim.x + (int32_t)threadIdx.x;
            blk[q] = j < sz ? d.pins[b + j] : -1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) blk[q] = blk[q] >= 0 ? part[blk[q]] : -1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned peers = __match_any_sync(kFull, blk[q]);
            if (blk[q] >= 0 && lane == __ffs(peers) - 1) atomicAdd(&cnt[blk[q]], (int)__popc(peers));
        }
    }
    __syncthreads();
    const bool wide = d.widx != nullptr && sz > narrow_max_of(d);
    uint8_t *row = reinterpret_cast<uint8_t *>(d.phi) + e * (int64_t)(d.k * w);
    for (int i = threadIdx.x; i < d.k && e < d.tiny[0]; i += blockDim.x) {
        const int32_t v = wide ? 0 : cnt[i];
        if (w == 1) row[i] = (uint8_t)v;
        else if (w == 2) reinterpret_cast<uint16_t *>(row)[i] = (uint16_t)v;
        else reinterpret_cast<int32_t *>(row)[i] = v;
        if (wide) d.phi_wide[(int64_t)d.widx[e] * d.k + i] = cnt[i];
    }
    if (threadIdx.x < 32) {
        const unsigned lo_lam = __ballot_sync(kFull, lane < d.k && cnt[lane] > 0);
        const unsigned lo_s1 = __ballot_sync(kFull, lane < d.k && cnt[lane] == 1);
        const unsigned hi_lam = __ballot_sync(kFull, lane + 32 < d.k && cnt[lane + 32] > 0);
        const unsigned hi_s1 = __ballot_sync(kFull, lane + 32 < d.k && cnt[lane + 32] == 1);
        if (lane == 0) {
            const int32_t wv = d.nw ? d.nw[e] : 1;
            write_record<Rec>(d, e, (uint64_t)lo_lam | ((uint64_t)hi_lam << 32),
                              (uint64_t)lo_s1 | ((uint64_t)hi_s1 << 32), wv | (wide ? (int32_t)kWideFlag : 0));
            const int lambda = __popc(lo_lam) + __popc(hi_lam);
            if (lambda > 0) obj = (long long)(lambda - 1) * wv;
        }
    }
    __syncthreads();
    return obj;
}

// The nets of the large-net prefix of the internal order, one CTA per net: k_init_nets would give all
// of them to its first CTAs.
template <typename Rec>
__global__ void __launch_bounds__(1024) k_init_big(Dev d, const uint8_t *part, int32_t e0, int32_t e1, const int32_t *guard)
{
    if (input_invalid(guard)) return;
    __shared__ int32_t cnt[64];
    long long obj = 0;
    for (int64_t e = e0 + (int64_t)blockIdx.x; e < e1; e += gridDim.x) obj += init_net_cta<Rec>(d, part, e, cnt);
    if (threadIdx.x == 0 && obj) atomicAdd(&d.acc[ACC_OBJ], (unsigned long long)obj);
}

// entry i of the staged row block (rows of `wb` bytes per net, entries of `w` bytes)
__device__ __forceinline__ void stage_set(uint32_t *blk, int row, int i, int w, int wb, int32_t v)
{
    uint8_t *p = reinterpret_cast<uint8_t *>(blk) + row * wb + i * w;
    if (w == 1) *p = (uint8_t)v;
    else if (w == 2) *reinterpret_cast<uint16_t *>(p) = (uint16_t)v;
    else *reinterpret_cast<int32_t *>(p) = v;
}

// One lane's net of at most N pins, counted in registers: pin i stands for its block if no earlier
// pin is in it, with the number of pins that are.
template <int N>
struct LaneNet {
    int blk[N], c[N];   // c: 0 unless pin i stands for its block
    __device__ __forceinline__ void count(const int32_t *pins, const uint8_t *part, int32_t b, int32_t size)
    {
#pragma unroll
        for (int i = 0; i < N; ++i) blk[i] = i < size ? __ldcs(&pins[b + i]) : -1;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            blk[i] = i < size ? (int)part[blk[i]] : -1 - i;   // no two absent pins alike
            c[i] = i < size;
        }
#pragma unroll
        for (int i = 1; i < N; ++i) {
            bool merged = false;
#pragma unroll
            for (int j = 0; j < i; ++j) {
                const bool same = !merged && c[j] > 0 && blk[j] == blk[i];
                c[j] += same;
                merged = merged || same;
            }
            if (merged) c[i] = 0;
        }
    }
    __device__ __forceinline__ void sets(uint64_t &lam, uint64_t &s1) const
    {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (c[i] > 0) lam |= 1ull << blk[i];
            if (c[i] == 1) s1 |= 1ull << blk[i];
        }
    }
    template <bool CLEAR>
    __device__ __forceinline__ void stage(uint32_t *rows, int row, int w, int wb) const
    {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (c[i] > 0) stage_set(rows, row, blk[i], w, wb, CLEAR ? 0 : c[i]);
    }
};

// The nets from e_begin on, 32 consecutive ones per warp.  Where none of the 32 has more than 4
// pins, each lane counts its own in registers.  Else the lanes walk the 32 nets' pins, one run
// in memory, flattened, four each in flight: counts by shared-memory atomics, whose old values give
// the Lambda and S1 flips (a warp per net of more than 8 pins took the 32 nets one after another).
// The 32 Phi rows are written as one contiguous block (no separate zeroing of the table).  Nets
// beyond kInitBig pins or a narrow entry are left to the whole CTA.  Row-net 2M (20 M pins, k = 8):
// 325 -> 137 us; power-law 50M (345 M pins, k = 64, 2-byte entries): 4.2 -> 3.2 ms, of which the
// gathers of Pi take about 2.  4 CTAs per SM: with 5 (48 registers, spills) the power-law table took
// 6.7 ms, with 3 the row-net one 160 us.
// The last CTA to finish stores the block weights and the objective and resets the round state
// (and the sums), so no other launch does; part, when another buffer than d.part, is copied there.
template <typename Rec>
__global__ void __launch_bounds__(kInitWarps * 32, 4) k_init_nets(Dev d, const uint8_t *part, int32_t e_begin,
                                                               const int32_t *guard)
{
    if (input_invalid(guard)) return;
    typedef typename std::conditional<sizeof(Rec) == 16, uint32_t, uint64_t>::type Lam;
    constexpr int kHalves = sizeof(Lam) / 4;
    __shared__ int32_t off33_w[kInitWarps][33];
    __shared__ int32_t src_w[kInitWarps][32];
    __shared__ uint32_t lam_w[kInitWarps][32 * kHalves], s1_w[kInitWarps][32 * kHalves];
    __shared__ int32_t cnt[64];
    __shared__ int32_t big_list[kInitWarps * 32];
    __shared__ int32_t n_big;
    __shared__ unsigned long long obj_s;
    __shared__ bool last;
    extern __shared__ __align__(16) uint32_t stage_dyn[];   // kInitWarps blocks of 32 rows
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int w = d.phi_w, wb = d.k * d.phi_w;       // bytes per entry / per row
    const int blk_words = (32 * wb + 15) / 16 * 4;   // one warp's block, 16-byte multiple
    const int32_t big_from = min(kInitBig, narrow_max_of(d));
    const uint32_t fmask = w == 1 ? 0xFFu : (w == 2 ? 0xFFFFu : 0xFFFFFFFFu);
    uint32_t *stage = stage_dyn + wid * blk_words;
    int32_t *off33 = off33_w[wid];
    if (threadIdx.x == 0) {
        n_big = 0;
        obj_s = 0;
    }
    __syncthreads();
    long long obj = 0;
    constexpr int kPerCta = kInitWarps * 32;
    uint4 *s4 = reinterpret_cast<uint4 *>(stage);
    for (int i = lane; i < blk_words / 4; i += 32) s4[i] = make_uint4(0, 0, 0, 0);   // and zero after every group
    __syncwarp();
    auto store_rows = [&](int64_t e0, int32_t rows) {
        // the block of rows e0 .. e0 + rows - 1 starts at byte e0 * wb of the table
        const int64_t byte0 = e0 * (int64_t)wb;
        uint8_t *dst = reinterpret_cast<uint8_t *>(d.phi) + byte0;
        if ((byte0 & 15) == 0 && (rows * wb) % 16 == 0) {
            uint4 *d4 = reinterpret_cast<uint4 *>(dst);
            for (int i = lane; i < rows * wb / 16; i += 32) __stcs(&d4[i], s4[i]);
        } else {
            // byte-exact tail (the table's rows need not be 16-byte multiples for small k)
            const uint8_t *s8 = reinterpret_cast<const uint8_t *>(stage);
            for (int i = lane; i < rows * wb; i += 32) dst[i] = s8[i];
        }
    };
    for (int64_t c0 = e_begin + (int64_t)blockIdx.x * kPerCta; c0 < d.m; c0 += (int64_t)gridDim.x * kPerCta) {
        const int64_t e0 = c0 + wid * 32, e = e0 + lane;
        // rows of the table: none of tiny nets
        const int32_t rows = (int32_t)max((int64_t)0, min((int64_t)32, min((int64_t)d.m, (int64_t)d.tiny[0]) - e0));
        int32_t b = 0, size = 0;
        if (e < d.m) {
            b = d.net_off[e];
            size = d.net_off[e + 1] - b;
        }
        const bool big = size > big_from;
        const int32_t wv = e < d.m && d.nw ? d.nw[e] : 1;
        const int32_t most = (int32_t)__reduce_max_sync(kFull, (unsigned)size);
        uint64_t lam = 0, s1 = 0;
        auto in_registers = [&](auto net) {
            net.count(d.pins, part, b, size);
            net.sets(lam, s1);
            if (rows == 0) return;
            net.template stage<false>(stage, lane, w, wb);
            __syncwarp();
            store_rows(e0, rows);
            __syncwarp();
            net.template stage<true>(stage, lane, w, wb);
        };
        if (most <= 4) {
            in_registers(LaneNet<4>());
        } else {
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {
                lam_w[wid][h * 32 + lane] = 0;
                s1_w[wid][h * 32 + lane] = 0;
            }
            const int32_t sz = big ? 0 : size;
            int32_t incl = sz;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            off33[lane] = incl - sz;
            src_w[wid][lane] = b - (incl - sz);
            if (lane == 31) off33[32] = incl;
            if (big) big_list[atomicAdd(&n_big, 1)] = (int32_t)e;
            __syncwarp();
            const int32_t total = off33[32];
            for (int32_t i0 = 0; i0 < total; i0 += 128) {
                int v[4], blk[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int32_t i = i0 + q * 32 + lane;
                    v[q] = i < total ? pin_net(off33, i) : 0;
                    blk[q] = i < total ? __ldcs(&d.pins[src_w[wid][v[q]] + i]) : -1;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) blk[q] = blk[q] >= 0 ? part[blk[q]] : -1;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (blk[q] < 0) continue;
                    const int at = v[q] * wb + blk[q] * w;
                    const int sh = (at & 3) * 8;
                    const uint32_t old = (atomicAdd(&stage[at >> 2], 1u << sh) >> sh) & fmask;
                    const uint32_t bit = 1u << (blk[q] & 31);
                    const int word = (blk[q] >> 5) * 32 + v[q];
                    if (old == 0) atomicOr(&lam_w[wid][word], bit);
                    if (old <= 1) atomicXor(&s1_w[wid][word], bit);
                }
            }
            __syncwarp();
            lam = lam_w[wid][lane];
            s1 = s1_w[wid][lane];
            if (kHalves == 2) {
                lam |= (uint64_t)lam_w[wid][32 * (kHalves - 1) + lane] << 32;
                s1 |= (uint64_t)s1_w[wid][32 * (kHalves - 1) + lane] << 32;
            }
            store_rows(e0, rows);
            __syncwarp();
            for (int i = lane; i < blk_words / 4; i += 32) s4[i] = make_uint4(0, 0, 0, 0);
        }
        if (e < d.m && !big) {
            write_record<Rec>(d, e, lam, s1, wv);
            if (lam) obj += (long long)(__popcll(lam) - 1) * wv;
        }
        __syncwarp();
        // large nets of the CTA's 256; their rows were written as zeros above, before the barrier
        if (__syncthreads_or(big)) {
            const int32_t nb = n_big;
            for (int32_t i = 0; i < nb; ++i) obj += init_net_cta<Rec>(d, part, big_list[i], cnt);
            if (threadIdx.x == 0) n_big = 0;
            __syncthreads();
        }
    }
    if (part != d.part) {
        const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
        const int64_t n16 = d.n / 16;
        for (int64_t i = t0; i < n16; i += stride)
            reinterpret_cast<uint4 *>(d.part)[i] = reinterpret_cast<const uint4 *>(part)[i];
        for (int64_t i = n16 * 16 + t0; i < d.n; i += stride) d.part[i] = part[i];
    }
    for (int o = 16; o; o >>= 1) obj += __shfl_xor_sync(kFull, obj, o);
    if (lane == 0 && obj) atomicAdd(&obj_s, (unsigned long long)obj);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (obj_s) atomicAdd(&d.acc[ACC_OBJ], obj_s);
        __threadfence();
        last = atomicAdd(&d.acc[ACC_DONE], 1ull) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x < d.k) d.bw[threadIdx.x] = (int64_t)__ldcg(&d.acc[ACC_BW + threadIdx.x]);
    if (threadIdx.x == 64) *d.obj = (int64_t)__ldcg(&d.acc[ACC_OBJ]);
    if (threadIdx.x < 2) d.rs[threadIdx.x] = 0;   // round 0, every vertex eligible
    __syncthreads();
    if (threadIdx.x < kAccN) d.acc[threadIdx.x] = 0;
}

// ------------------------------------------------------------------ getters
__global__ void k_obj_from_phi(Dev d, unsigned long long *out)
{
    long long s = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < d.m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t size = d.net_off[e + 1] - d.net_off[e];
        const bool wide = d.widx != nullptr && size > (d.phi_w == 1 ? 255 : (d.phi_w == 2 ? 65535 : 0x7fffffff));
        const int32_t wrow = wide ? d.widx[e] : 0;
        int lambda = 0;
        if (e >= d.tiny[0])
            lambda = d.k <= 32 ? __popc(reinterpret_cast<const Rec16 *>(d.rec)[e].lam)
                               : __popcll((long long)reinterpret_cast<const Rec32 *>(d.rec)[e].lam);
        else
            for (int i = 0; i < d.k; ++i) lambda += phi_get(d, (int32_t)e, i, wide, wrow) > 0;
        if (lambda > 0) s += (long long)(lambda - 1) * (d.nw ? d.nw[e] : 1);
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, (unsigned long long)s);
}

// the per-net getters and the checkpoint take nets in input order
__device__ __forceinline__ int32_t internal_net(const Dev &d, int32_t e)
{
    return d.net_perm ? d.net_perm[e] : e;
}

__global__ void k_widen_phi(Dev d, int32_t *out)
{
    const int64_t total = (int64_t)d.m * d.k;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = internal_net(d, (int32_t)(x / d.k)), i = (int32_t)(x % d.k);
        const int32_t size = d.net_off[e + 1] - d.net_off[e];
        const bool wide = d.widx != nullptr && size > (d.phi_w == 1 ? 255 : (d.phi_w == 2 ? 65535 : 0x7fffffff));
        out[x] = phi_get(d, e, i, wide, wide ? d.widx[e] : 0);
    }
}

template <typename Rec>
__global__ void k_get_lambda(Dev d, uint64_t *out)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < d.m;
         e += (int64_t)gridDim.x * blockDim.x)
        out[e] = (uint64_t)reinterpret_cast<const Rec *>(d.rec)[internal_net(d, (int32_t)e)].lam;
}

// move stamps of the records
template <typename Rec>
__global__ void k_export_moved(Dev d, int32_t r, int32_t first, uint8_t *out)
{
    const Rec *recs = reinterpret_cast<const Rec *>(d.rec);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < d.m;
         e += (int64_t)gridDim.x * blockDim.x)
        out[e] = (!first && moved_in_prev_round(recs[internal_net(d, (int32_t)e)].mv, r)) ? 1 : 0;
}

template <typename Rec>
__global__ void k_import_moved(Dev d, int32_t r, const uint8_t *flags)
{
    Rec *recs = reinterpret_cast<Rec *>(d.rec);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < d.m;
         e += (int64_t)gridDim.x * blockDim.x)
        if (flags[e]) recs[internal_net(d, (int32_t)e)].mv = (r - 1) * 2;   // last move in round r-1
}

__global__ void k_set_round_state(int32_t *rs, int32_t r, int32_t started)
{
    if (threadIdx.x == 0) {
        rs[0] = r;
        rs[1] = started;
    }
}

__global__ void k_part_to_i32(const uint8_t *part, int32_t *out, int32_t n)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        out[v] = part[v];
}

// ------------------------------------------------------------------ host helpers
int grid_for(int64_t work, int threads, int cap = 152 * 32)
{
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

namespace hgp {

static constexpr int kMaxPoolDevices = 64;
static constexpr uint64_t kPoolKeepShare = 64;   // default retention: this fraction of the device's memory
static std::mutex g_pool_mu;
static cudaMemPool_t g_pool[kMaxPoolDevices];

static std::atomic<cudaMemPool_t> g_pool_ready[kMaxPoolDevices];   // set once created

// the library's pool on the current device, created on first use
cudaError_t library_pool(cudaMemPool_t *out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxPoolDevices) return cudaErrorInvalidDevice;
    if (cudaMemPool_t ready = g_pool_ready[dev].load(std::memory_order_acquire)) {
        *out = ready;
        return cudaSuccess;
    }
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps props;
        memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        e = cudaMemPoolCreate(&g_pool[dev], &props);
        if (e != cudaSuccess) {
            g_pool[dev] = nullptr;
            return e;
        }
        // keep freed memory between handles while the pool holds at most 1/64 of the device's (4.4 GB of
        // 284), in use and kept: mapping it afresh and unmapping it at the next
        // synchronisation took as long as the work itself
        // (creating and closing a 5M-vertex level 6.4 -> 3.6 ms, a 500k-pin request 457 -> 261
        // us, contraction of 10M vertices 10.4 -> 6.8 ms).  The reuse policies stay at their defaults:
        // when no more memory can be mapped, memory whose release is still queued on another stream
        // is taken, and the allocating stream waits for that release (a handle created on a nearly
        // full device while a destroyed one's rounds still run).
        size_t free_b = 0, total_b = 0;
        uint64_t keep = 0;
        if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess) keep = total_b / kPoolKeepShare;
        if (cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess)
            (void)cudaGetLastError();
        g_pool_ready[dev].store(g_pool[dev], std::memory_order_release);
    }
    *out = g_pool[dev];
    return cudaSuccess;
}

static std::atomic<int> g_blocking_waits{0};

// a blocking-sync event per thread and device, destroyed when the thread ends
struct WaitEvents {
    cudaEvent_t ev[kMaxPoolDevices] = {};
    ~WaitEvents()
    {
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        (void)cudaGetLastError();
    }
};
static thread_local WaitEvents t_wait;

cudaError_t stream_wait(cudaStream_t st)
{
    if (!g_blocking_waits.load(std::memory_order_relaxed)) return cudaStreamSynchronize(st);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxPoolDevices) return cudaErrorInvalidDevice;
    cudaEvent_t &ev = t_wait.ev[dev];
    if (!ev) {
        e = cudaEventCreateWithFlags(&ev, cudaEventBlockingSync | cudaEventDisableTiming);
        if (e != cudaSuccess) {
            ev = nullptr;
            return e;
        }
    }
    e = cudaEventRecord(ev, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(ev);
    return e;
}

cudaError_t dev_alloc(void **p, size_t bytes, cudaStream_t st)
{
    *p = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = library_pool(&pool);
    if (e == cudaSuccess) e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    if (e == cudaErrorMemoryAllocation) {
        // what the pool keeps may be what is missing: give it back and try once more
        (void)cudaGetLastError();
        if (cudaMemPoolTrimTo(pool, 0) == cudaSuccess) e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        *p = nullptr;
    }
    return e;
}

bool readable_in_place(const void *p, size_t bytes, int device)
{
    typedef CUresult (*Query)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static const Query query = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &found) != cudaSuccess) {
            (void)cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Query>(f);
    }();
    // one call for all of them; what an address does not have stays zero
    unsigned type = 0, managed = 0;
    int owner = -1;
    CUdeviceptr base = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL,
                                  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *to[] = {&type, &managed, &owner, &base, &size};
    return query && query(5, what, to, (CUdeviceptr)p) == CUDA_SUCCESS && type == CU_MEMORYTYPE_DEVICE && !managed &&
           owner == device && range_inside((uintptr_t)p, bytes, (uintptr_t)base, size);
}

void dev_free(void *p, cudaStream_t st)
{
    if (p && pool_free(p, st) != cudaSuccess) (void)cudaGetLastError();
}

}  // namespace hgp

namespace {

template <typename T>
cudaError_t dalloc(hgp_handle *h, T **p, int64_t count, bool in_arena = true)
{
    *p = nullptr;
    if (count < 1) count = 1;
    if (void *a = in_arena ? arena_take(h, (size_t)count * sizeof(T)) : nullptr) {
        *p = reinterpret_cast<T *>(a);
        return cudaSuccess;
    }
    if (h->n_allocs >= hgp_handle::kMaxAllocs) return cudaErrorMemoryAllocation;
    void *q = nullptr;
    cudaError_t e = dev_alloc(&q, (size_t)count * sizeof(T), h->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return e;
    }
    h->allocs[h->n_allocs++] = q;
    *p = reinterpret_cast<T *>(q);
    return cudaSuccess;
}

#define CK(call)                                   \
    do {                                           \
        cudaError_t _e = (call);                   \
        if (_e != cudaSuccess) {                   \
            (void)cudaGetLastError();              \
            return status_of(_e);                  \
        }                                          \
    } while (0)

// State of the partition in `part` (d.part, or a buffer that is copied there); its block weights are
// in d.acc.  guard: the creation's error flag while creating (kernels skip flagged input), else nullptr
int init_state(hgp_handle *h, const uint8_t *part, const int32_t *guard)
{
    Dev &d = h->d;
    cudaStream_t st = h->stream;
    const int32_t e_begin = h->m_big32;
    for (int huge = 1; huge >= 0; --huge) {
        const int32_t e0 = huge ? 0 : h->m_huge, e1 = huge ? h->m_huge : e_begin;
        if (e0 >= e1) continue;
        const int threads = huge ? 1024 : 256, gb = std::min(e1 - e0, 152 * (huge ? 2 : 16));
        if (d.k <= 32) k_init_big<Rec16><<<gb, threads, 0, st>>>(d, part, e0, e1, guard);
        else k_init_big<Rec32><<<gb, threads, 0, st>>>(d, part, e0, e1, guard);
        h->launches++;
    }
    const int g = grid_for(std::max<int64_t>((int64_t)d.m - e_begin, 1), kInitWarps * 32, 152 * 16);
    auto init_smem = [](int k, int w) { return kInitWarps * (32 * k * w + 15) / 16 * 16; };
    const int smem = init_smem(d.k, d.phi_w);
    // beyond the default limit the attribute is the kernel's largest need over every k and entry
    // width (the same value from every caller), so concurrent creations cannot lower it under
    // each other
    if (d.k <= 32) {
        if (smem > kDefaultSmem)
            CK(cudaFuncSetAttribute(k_init_nets<Rec16>, cudaFuncAttributeMaxDynamicSharedMemorySize, init_smem(32, 4)));
        k_init_nets<Rec16><<<g, kInitWarps * 32, smem, st>>>(d, part, e_begin, guard);
    } else {
        if (smem > kDefaultSmem)
            CK(cudaFuncSetAttribute(k_init_nets<Rec32>, cudaFuncAttributeMaxDynamicSharedMemorySize, init_smem(64, 4)));
        k_init_nets<Rec32><<<g, kInitWarps * 32, smem, st>>>(d, part, e_begin, guard);
    }
    h->launches++;
    CK(cudaGetLastError());
    h->next_round = 0;
    h->all_eligible = true;
    return HGP_OK;
}

constexpr int kSmallN = 72 + kAccN;   // int64 entries of a handle's small state (see create_impl)

size_t aligned_bytes(int64_t bytes) { return (size_t)((bytes < 1 ? 1 : bytes) + 255) / 256 * 256; }

// What a creation uses and the handle does not keep: the int64 offsets, the int32 partition, and the scan
// scratch (block sums, counts).
struct CreateScratch {
    int64_t off64, part_in, block_sums, tmp;   // entries
    CreateScratch(int32_t n, int32_t m)
    {
        const int64_t nm = n > m ? n : m;
        const int64_t nr_ctas = m > 0 ? std::min<int64_t>(((int64_t)m + 2047) / 2048, 1216) : 0;
        const int64_t scan_count = std::max<int64_t>(nm + 1, kNrRanks * nr_ctas + 1);
        off64 = (int64_t)m + 1;
        part_in = n;
        block_sums = (scan_count + kScanChunk - 1) / kScanChunk + 1;
        tmp = nm + 1;
    }
    size_t bytes() const
    {
        return aligned_bytes(8 * off64) + aligned_bytes(4 * part_in) + aligned_bytes(4 * block_sums) + aligned_bytes(4 * tmp);
    }
};

// Device bytes of every buffer a handle of few nets (see kHostSizesMaxNets, kDeviceArenaMaxNets) keeps,
// each rounded up to 256 bytes: the arena those buffers are carved from.  It covers the direct transpose
// in input net order without wide nets; buffers of any other path (or beyond a miscount) come from the
// pool instead.  max_size < 0: the largest net is not known yet, and Phi not part of the arena.
size_t small_handle_bytes(int32_t n, int32_t m, int64_t P, int32_t k, const hgp_options &o, int32_t max_size,
                          bool has_vw, bool has_nw)
{
    auto A = [](int64_t bytes) { return aligned_bytes(bytes); };
    const int64_t n_tiles = ((int64_t)n + kTile - 1) / kTile, nseg = segments_of(o.subrounds);
    const int64_t S = o.subrounds;
    const int w = o.phi_width ? o.phi_width : (max_size <= 255 ? 1 : 2);
    size_t b = 0;
    b += A(4 * ((int64_t)m + 1)) + A(4 * P);                                         // inputs
    if (has_vw) b += A(4 * (int64_t)n);
    if (has_nw) b += A(4 * (int64_t)m) + A(4 * (int64_t)n);                           // and W(u)
    b += A(4 * ((int64_t)n + 1)) + A(4 * P);                                         // vtx_off, inc
    if (max_size >= 0) b += A(4 * (((int64_t)m * k * w + 7) / 8 * 2));
    b += 2 * A(n) + A((int64_t)m * (k <= 32 ? 16 : 32)) + A(8 * kSmallN);
    b += A(2 * n_tiles * kTile) + A(2 * n_tiles * (S + 1)) + A(8 * n_tiles * kTile) + A(4 * n_tiles * nseg);
    b += A(8 * (int64_t)k * kBins) + A((int64_t)sizeof(Sel) * 64) + A(8 * (int64_t)k * n_tiles);
    if (o.revert_negative) {
        int64_t cap = 1024;
        while (cap < 2 * P) cap <<= 1;
        b += A(n_tiles * kTile) + A(16) + A(4 * (int64_t)m) + A(cap * kRvSlotBytes);
    }
    b += A(8 * ST_N * 16 + 4 * kWqPerRow * 16);                                      // statistics
    b += A(sizeof(Dev));                                                            // device Dev
    return b;
}

int create_impl(int32_t n, int32_t m, const int64_t *net_offsets, const int32_t *pins,
                const int32_t *vertex_w, const int32_t *net_w, int32_t k, double eps,
                const int32_t *initial_part, const hgp_options *opt, hgp_handle **out, bool on_device)
{
    if (!out) return HGP_ERR_INVALID;
    *out = nullptr;
    if (n < 1 || m < 0 || !net_offsets || !initial_part || (m > 0 && !pins)) return HGP_ERR_INVALID;
    if (k < 2 || !(eps > 0.0 && eps < 1.0)) return HGP_ERR_INVALID;
    if (k > 64) return HGP_ERR_UNSUPPORTED;
    hgp_options o;
    hgp_default_options(&o);
    if (opt) o = *opt;
    if (o.subrounds == 0) o.subrounds = 4;
    if (o.subrounds < 0) return HGP_ERR_INVALID;
    if (o.subrounds > 64) return HGP_ERR_UNSUPPORTED;
    if (o.phi_width != 0 && o.phi_width != 1 && o.phi_width != 2 && o.phi_width != 4) return HGP_ERR_INVALID;

    int64_t P = 0;
    if (on_device) {
        if (cudaMemcpy(&P, net_offsets + m, sizeof(int64_t), cudaMemcpyDeviceToHost) != cudaSuccess) {
            (void)cudaGetLastError();
            return HGP_ERR_INVALID;
        }
    } else {
        P = net_offsets[m];
    }
    if (P < 0) return HGP_ERR_INVALID;
    if (P >= ((int64_t)1 << 31)) return HGP_ERR_UNSUPPORTED;

    hgp_handle *h = new (std::nothrow) hgp_handle();
    if (!h) return HGP_ERR_OOM;
    int rc = HGP_OK;
    auto fail = [&](int code) {
        hgp_destroy(h);
        return code;
    };
    Dev &d = h->d;
    cudaGetDevice(&h->device);
    auto release = [&](void *ptr) {   // frees one of the handle's allocations before the end
        if (!ptr || in_arena(h, ptr)) return;
        for (int i = 0; i < h->n_allocs; ++i)
            if (h->allocs[i] == ptr) {
                dev_free(h->allocs[i], h->stream);
                h->allocs[i] = h->allocs[--h->n_allocs];
                return;
            }
    };
    // a temporary from the pool: the handle's until release(), so that a creation that fails frees it
    auto temporary = [&](auto **ptr, int64_t count) { return dalloc(h, ptr, count, false); };
    if (o.cuda_stream) {
        h->stream = (cudaStream_t)o.cuda_stream;
    } else {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
            (void)cudaGetLastError();
            return fail(HGP_ERR_CUDA);
        }
        h->own_stream = true;
    }
    cudaStream_t st = h->stream;
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    h->seed = o.seed;
    h->debug = o.debug;
    if (o.gain_ctas_per_sm < 0 || o.apply_ctas_per_sm < 0) return fail(HGP_ERR_INVALID);
    h->gain_ctas = o.gain_ctas_per_sm;
    h->apply_ctas = o.apply_ctas_per_sm;
    h->graph = o.graph;
    d.n = n;
    d.m = m;
    d.k = k;
    d.P = (int32_t)P;
    d.S = o.subrounds;
    for (int32_t &t : d.tiny) t = 0x7fffffff;
    d.n_tiles = (int32_t)(((int64_t)n + kTile - 1) / kTile);
    d.nseg = segments_of(d.S);

#define CKF(call)                                  \
    do {                                           \
        cudaError_t _e = (call);                   \
        if (_e != cudaSuccess) {                   \
            (void)cudaGetLastError();              \
            return fail(status_of(_e));            \
        }                                          \
    } while (0)

    // ---- small host inputs: the host checks the offsets and finds the largest net itself
    // (cheaper than a round trip to the device, which waits behind other work on a busy GPU), so
    // the creation is queued to its end without waiting for the device checks: the kernels after
    // them skip flagged input (guard) and the verdict comes with the final read-back.  Their
    // buffers are carved from one allocation (the arena), sized here.
    const bool host_sizes = !on_device && m < kHostSizesMaxNets;
    int32_t max_size = 0;
    if (host_sizes) {
        if (net_offsets[0] != 0) return fail(HGP_ERR_INVALID);
        // branch-free smallest and largest size (vectorisable); offsets checked afterwards
        int64_t lo = 0, hi = 0;
        for (int32_t e = 0; e < m; ++e) {
            const int64_t sz = net_offsets[e + 1] - net_offsets[e];
            lo = sz < lo ? sz : lo;
            hi = sz > hi ? sz : hi;
        }
        if (lo < 0) return fail(HGP_ERR_INVALID);   // then every size is at most P < 2^31
        max_size = (int32_t)hi;
    }
    const CreateScratch cs(n, m);
    int64_t *off64 = nullptr;
    int32_t *part_in = nullptr, *tmp = nullptr, *block_sums = nullptr;
    // device inputs: the largest net is not known yet, so Phi gets room for 2-byte entries.  That and the
    // scratch stay with the handle where they are little; else the scratch is an allocation of its own,
    // given back at the end, and Phi another one.
    const bool whole = host_sizes || (int64_t)cs.bytes() + (int64_t)m * k <= kKeptSpare;
    if (host_sizes || m < kDeviceArenaMaxNets) {
        const size_t keep = small_handle_bytes(n, m, P, k, o, host_sizes ? max_size : (whole ? 65535 : -1), vertex_w != nullptr,
                                               net_w != nullptr);
        const size_t bytes = keep + (whole ? cs.bytes() : 0);
        void *a = nullptr;
        if (dev_alloc(&a, bytes, st) == cudaSuccess) {   // else every buffer comes from the pool
            h->allocs[h->n_allocs++] = a;
            h->arena = static_cast<char *>(a);
            h->arena_size = bytes;
        }
        if (!whole && dev_alloc(&a, cs.bytes(), st) == cudaSuccess) {
            h->allocs[h->n_allocs++] = a;                // released as off64's
            char *at = static_cast<char *>(a);
            off64 = reinterpret_cast<int64_t *>(at);
            part_in = reinterpret_cast<int32_t *>(at += aligned_bytes(8 * cs.off64));
            block_sums = reinterpret_cast<int32_t *>(at += aligned_bytes(4 * cs.part_in));
            tmp = reinterpret_cast<int32_t *>(at += aligned_bytes(4 * cs.block_sums));
        }
    }
    if (!off64) {
        CKF(dalloc(h, &off64, cs.off64));
        CKF(dalloc(h, &part_in, cs.part_in));
        CKF(dalloc(h, &block_sums, cs.block_sums));
        CKF(dalloc(h, &tmp, cs.tmp));
    }

    // ---- inputs
    int32_t *net_off = nullptr, *pins_d = nullptr, *vw_d = nullptr, *nw_d = nullptr;
    CKF(dalloc(h, &net_off, (int64_t)m + 1));
    CKF(dalloc(h, &pins_d, P));
    // small state: block weights [64], objective, largest W(u), error flag and largest net (int32
    // each), round state (2 int32), then the sums of a state initialisation; zeroed once
    int64_t *small = nullptr;
    CKF(dalloc(h, &small, kSmallN));
    CKF(cudaMemsetAsync(small, 0, kSmallN * sizeof(int64_t), st));
    d.bw = small;
    d.obj = small + 64;
    unsigned long long *maxw_d = reinterpret_cast<unsigned long long *>(small + 65);
    d.err = reinterpret_cast<int32_t *>(small + 66);
    int32_t *max_size_d = d.err + 1;
    d.rs = reinterpret_cast<int32_t *>(small + 67);
    d.acc = reinterpret_cast<unsigned long long *>(small + 72);
    CKF(cudaMemcpyAsync(off64, net_offsets, sizeof(int64_t) * ((size_t)m + 1), kind, st));
    if (P) CKF(cudaMemcpyAsync(pins_d, pins, sizeof(int32_t) * (size_t)P, kind, st));
    CKF(cudaMemcpyAsync(part_in, initial_part, sizeof(int32_t) * (size_t)n, kind, st));
    if (vertex_w) {
        CKF(dalloc(h, &vw_d, n));
        CKF(cudaMemcpyAsync(vw_d, vertex_w, sizeof(int32_t) * (size_t)n, kind, st));
    }
    if (net_w) {
        CKF(dalloc(h, &nw_d, m));
        CKF(cudaMemcpyAsync(nw_d, net_w, sizeof(int32_t) * (size_t)m, kind, st));
    }
    d.net_off = net_off;
    d.pins = pins_d;
    d.vw = vw_d;
    d.nw = nw_d;

    // ---- validation
    uint8_t *part = nullptr;
    CKF(dalloc(h, &part, n));
    CKF(dalloc(h, &h->part_next, n));
    k_check_inputs<<<grid_for(std::max<int64_t>((int64_t)m + 1, n), 256, 152 * 8), 256, 0, st>>>(
        off64, net_off, m, P, nw_d, vw_d, part_in, n, k, part, d.acc, d.err); h->launches++;
    CKF(cudaGetLastError());
    int32_t host_err[2] = {0, 0};
    // one read-back for both checks: the pin check does nothing when the offsets were bad
    if (m > 0) {
        k_check_pins<<<grid_for(std::max<int64_t>(P / 4, m), 256, 152 * 8), 256, 0, st>>>(net_off, pins_d, m, n, P, d.err,
                                                                                    max_size_d, d.acc); h->launches++;
        CKF(cudaGetLastError());
    }
    const int32_t *guard = nullptr;
    if (host_sizes) {
        guard = d.err;
    } else {
        CKF(cudaMemcpyAsync(host_err, d.err, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        CKF(stream_wait(st));
        if (host_err[0] & ERR_INVALID) return fail(HGP_ERR_INVALID);
        max_size = host_err[1];
    }

    // ---- scans (in block_sums, shared by all of them)
    const int64_t nr_ctas = m > 0 ? std::min<int64_t>(((int64_t)m + 2047) / 2048, 1216) : 0;
    auto scan = [&](const int32_t *in, int32_t *outp, int64_t count) -> cudaError_t {
        const int64_t blocks = (count + kScanChunk - 1) / kScanChunk;
        const int64_t bl = blocks < 1 ? 1 : blocks;
        k_scan_reduce<<<(unsigned)bl, kScanThreads, 0, st>>>(in, count, block_sums); h->launches++;
        k_scan_sums<<<1, kScanThreads, 0, st>>>(block_sums, bl); h->launches++;
        k_scan_final<<<(unsigned)bl, kScanThreads, 0, st>>>(in, outp, count, block_sums); h->launches++;
        return cudaGetLastError();
    };

    // ---- internal net order (largest size class first); the input-order arrays are released
    const int64_t avg_size = m > 0 ? (P + m - 1) / m : 0;
    const bool reorder = m > 0 && !(o.debug & 8) &&
                         ((o.debug & 4) || (m >= kReorderMinNets && max_size >= kReorderSkew * avg_size));
    int32_t p_big = 0;   // pins of the large-net prefix
    if (reorder) {
        const int32_t per_cta = (int32_t)((m + nr_ctas - 1) / nr_ctas);
        const int32_t nslots = (int32_t)(kNrRanks * nr_ctas);
        int32_t *cnt = nullptr, *perm = nullptr, *off_int = nullptr, *pins_int = nullptr, *nw_int = nullptr;
        CKF(temporary(&cnt, 2 * (int64_t)nslots + 1));
        int32_t *base = cnt + nslots;
        CKF(dalloc(h, &perm, m));
        CKF(dalloc(h, &off_int, (int64_t)m + 1));
        if (P) CKF(dalloc(h, &pins_int, P));
        if (nw_d) CKF(dalloc(h, &nw_int, m));
        k_nr_count<<<(unsigned)nr_ctas, kNrThreads, 0, st>>>(net_off, m, per_cta, cnt); h->launches++;
        CKF(scan(cnt, base, nslots));
        // first internal id of every rank
        int32_t first[kNrRanks];
        CKF(cudaMemcpy2DAsync(first, sizeof(int32_t), base, sizeof(int32_t) * (size_t)nr_ctas, sizeof(int32_t), kNrRanks,
                              cudaMemcpyDeviceToHost, st));
        CKF(stream_wait(st));
        auto below = [&](int32_t size) {   // nets of at least `size` pins (a power of two)
            int rank = 0;
            while (((int64_t)1 << (31 - rank)) >= size) ++rank;
            return first[rank];
        };
        const int32_t mb = below(kBigNet);
        h->m_huge = below(kHugeNet);
        for (int i = 0; i < 4; ++i) d.tiny[i] = first[kNrTiny + i];
        int32_t *src_big = nullptr;   // where the pins of the large-net prefix come from
        if (mb > 0) CKF(temporary(&src_big, mb));
        k_nr_place<<<(unsigned)nr_ctas, kNrThreads, 0, st>>>(net_off, m, per_cta, base, perm, tmp, mb, src_big);
        h->launches++;
        CKF(scan(tmp, off_int, m));   // sizes in internal order -> offsets (off_int[m] = P)
        CKF(cudaMemcpyAsync(&p_big, off_int + mb, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        k_nr_pins<<<grid_for((int64_t)m, 256), 256, 0, st>>>(net_off, pins_d, nw_d, m, mb, perm, off_int, pins_int,
                                                             nw_int); h->launches++;
        CKF(cudaGetLastError());
        CKF(stream_wait(st));
        if (p_big > 0) {
            k_nr_pins_big<<<(unsigned)((p_big + kBigChunk - 1) / kBigChunk), 1024, 0, st>>>(off_int, src_big, pins_d, mb,
                                                                                            pins_int);
            h->launches++;
            CKF(cudaGetLastError());
        }
        release(cnt);
        release(src_big);
        h->m_big = mb;
        h->m_big32 = (int32_t)std::min((int64_t)m, ((int64_t)mb + 31) / 32 * 32);
        release(net_off);
        release(pins_d);
        if (nw_d) release(nw_d);
        net_off = off_int;
        pins_d = pins_int;
        nw_d = nw_int;
        d.net_off = net_off;
        d.pins = pins_d;
        d.nw = nw_d;
        d.net_perm = perm;
    }

    // ---- Phi width chosen by the largest net: 1 byte if every net fits, else 2 bytes; nets
    // beyond the entry's range keep int32 rows in the wide table
    int w = o.phi_width;
    if (w == 0) w = max_size <= 255 ? 1 : 2;
    d.phi_w = w;
    const int32_t narrow_max = w == 1 ? 255 : (w == 2 ? 65535 : 0x7fffffff);

    // ---- wide nets
    const int32_t phi_rows = std::min(m, d.tiny[0]);
    if (max_size > narrow_max) {
        int32_t *widx = nullptr;
        CKF(dalloc(h, &widx, (int64_t)m + 1));
        k_wide_flags<<<grid_for(m, 256), 256, 0, st>>>(net_off, m, narrow_max, tmp); h->launches++;
        CKF(scan(tmp, widx, m));
        int32_t nwide = 0;
        CKF(cudaMemcpyAsync(&nwide, widx + m, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        CKF(stream_wait(st));
        h->n_wide = nwide;
        d.widx = widx;
        int32_t *pw = nullptr;
        CKF(dalloc(h, &pw, (int64_t)nwide * k));
        d.phi_wide = pw;
    }

    // ---- vertex -> nets CSR (bucketed transpose; the wide flag goes into inc on the way)
    int32_t *vtx_off = nullptr, *inc = nullptr;
    CKF(dalloc(h, &vtx_off, (int64_t)n + 1));
    CKF(dalloc(h, &inc, P));
    CKF(cudaMemsetAsync(tmp, 0, sizeof(int32_t) * ((size_t)n + 1), st));
    if (P > 0 && n <= kTpDirectMaxN && !(o.debug & 2)) {
        k_degrees<<<grid_for(P, 256), 256, 0, st>>>(pins_d, P, tmp, guard); h->launches++;
        CKF(scan(tmp, vtx_off, n));
        CKF(cudaMemcpyAsync(tmp, vtx_off, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st));
        k_scatter<<<grid_for((int64_t)m * 32, 256), 256, 0, st>>>(net_off, pins_d, m, narrow_max, tmp, inc, guard);
        h->launches++;
        CKF(cudaGetLastError());
    } else if (P > 0) {
        auto buckets = [&](int sh) { return (((int64_t)n + ((int64_t)1 << sh) - 1) >> sh); };
        int bshift = kTpShift;
        while (bshift > kTpMinShift && buckets(bshift) < kTpMinCtas) --bshift;
        while (buckets(bshift) > kTpMaxBuckets) ++bshift;
        const int32_t nbk = (int32_t)buckets(bshift);
        const int32_t e_begin = h->m_big;   // the large-net prefix goes to k_tp_scatter_big
        const int64_t p_rest = P - p_big;
        const int64_t per_cta = std::min<int64_t>(kTpMaxPins, std::max<int64_t>(kTpMinPins, p_rest / kTpMinCtas));
        int32_t *bk = nullptr;           // counts [nbk + 1], offsets [nbk + 1], cursors [nbk]
        unsigned long long *pairs = nullptr;
        CKF(temporary(&bk, 3 * (int64_t)nbk + 2));
        CKF(temporary(&pairs, P));
        int32_t *bk_cnt = bk, *bk_off = bk + nbk + 1, *bk_cur = bk + 2 * nbk + 2;
        CKF(cudaMemsetAsync(bk_cnt, 0, sizeof(int32_t) * ((size_t)nbk + 1), st));
        k_tp_hist<<<grid_for(P, 256, 152 * 8), 256, 0, st>>>(pins_d, P, bshift, nbk, bk_cnt, guard); h->launches++;
        CKF(scan(bk_cnt, bk_off, nbk));
        CKF(cudaMemcpyAsync(bk_cur, bk_off, sizeof(int32_t) * (size_t)nbk, cudaMemcpyDeviceToDevice, st));
        const int64_t sc = (p_rest + per_cta - 1) / per_cta;
        if (e_begin > 0 && p_big > 0) {
            k_tp_scatter_big<<<(unsigned)((p_big + kBigChunk - 1) / kBigChunk), kTpThreads, 0, st>>>(
                net_off, pins_d, e_begin, bshift, nbk, narrow_max, bk_cur, pairs, guard); h->launches++;
        }
        if (sc > 0) {
            k_tp_scatter<<<(unsigned)sc, kTpThreads, 0, st>>>(net_off, pins_d, m, e_begin, bshift, nbk, narrow_max,
                                                       (int32_t)per_cta, bk_cur, pairs, guard); h->launches++;
        }
        if (bshift <= kTpSmemShift) {
            const int smem = (int)(sizeof(int32_t) << bshift);
            cudaFuncSetAttribute(k_tp_place<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(int32_t) << kTpSmemShift));   // largest need, as above
            k_tp_place<true><<<nbk, 1024, smem, st>>>(pairs, bk_off, bshift, n, nbk, tmp, vtx_off, inc, guard);
        } else {
            k_tp_place<false><<<nbk, 1024, 0, st>>>(pairs, bk_off, bshift, n, nbk, tmp, vtx_off, inc, guard);
        }
        h->launches++;
        CKF(cudaGetLastError());
        release(pairs);
        release(bk);
    } else {
        CKF(cudaMemsetAsync(vtx_off, 0, sizeof(int32_t) * ((size_t)n + 1), st));
    }
    d.vtx_off = vtx_off;
    d.inc = inc;

    int32_t *vnw = nullptr;
    if (nw_d) CKF(dalloc(h, &vnw, n));
    d.vnw = vnw;
    // the result of this check is read with the block weights at the end (nothing in between
    // depends on it)
    k_vertex_netweight<<<grid_for(n, 256), 256, 0, st>>>(vtx_off, inc, nw_d, n, vnw, d.err, maxw_d); h->launches++;
    CKF(cudaGetLastError());

    // ---- state (Pi was stored by the input check)
    d.part = part;
    const int64_t entries = (int64_t)phi_rows * k;
    const int64_t words = (entries * w + 7) / 8 * 2;
    uint32_t *phi = nullptr;
    CKF(dalloc(h, &phi, words, whole));
    d.phi = phi;   // written whole by init_state
    const size_t rec_bytes = k <= 32 ? sizeof(Rec16) : sizeof(Rec32);
    uint4 *rec = nullptr;
    CKF(dalloc(h, &rec, (int64_t)m * (int64_t)(rec_bytes / 16)));
    d.rec = rec;

    // ---- per-sub-round scratch
    uint16_t *sub_list = nullptr, *sub_start = nullptr;
    uint64_t *cand = nullptr;
    int32_t *cand_cnt = nullptr;
    int64_t *tie = nullptr;
    unsigned long long *hist = nullptr;
    Sel *sel = nullptr;
    CKF(dalloc(h, &sub_list, (int64_t)d.n_tiles * kTile));
    CKF(dalloc(h, &sub_start, (int64_t)d.n_tiles * (d.S + 1)));
    CKF(dalloc(h, &cand, (int64_t)d.n_tiles * kTile));
    CKF(dalloc(h, &cand_cnt, (int64_t)d.n_tiles * d.nseg));
    CKF(dalloc(h, &hist, (int64_t)k * kBins));
    CKF(dalloc(h, &sel, 64));
    CKF(dalloc(h, &tie, (int64_t)k * d.n_tiles));
    CKF(cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * (size_t)k * kBins, st));
    d.sub_list = sub_list;
    d.sub_start = sub_start;
    d.cand = cand;
    d.cand_cnt = cand_cnt;
    d.hist = hist;
    d.sel = sel;
    d.tie = tie;
    if (o.revert_negative) {
        // per candidate slot source blocks, and a table with room for the two (net, block)
        // keys of every incidence of a sub-round's movers (at most 2 P keys)
        uint8_t *rv_src = nullptr;
        unsigned long long *rv_cnt = nullptr;
        int64_t cap = 1024;
        while (cap < 2 * (int64_t)P) cap <<= 1;
        int32_t *rv_net = nullptr;
        CKF(dalloc(h, &rv_src, (int64_t)d.n_tiles * kTile));
        CKF(dalloc(h, &rv_cnt, 2));
        CKF(dalloc(h, &rv_net, m));
        CKF(dalloc(h, reinterpret_cast<uint4 **>(&d.rv_tab), cap * kRvSlotBytes / 16));
        CKF(cudaMemsetAsync(rv_cnt, 0, 2 * sizeof(unsigned long long), st));
        d.rv_net = rv_net;
        d.rv_src = rv_src;
        d.rv_cnt = rv_cnt;
        d.rv_cap = cap;
    }
    d.seed = o.seed;
    d.variant = (o.balance_moves ? 1 : 0) | (o.revert_negative ? 2 : 0);

    rc = init_state(h, part, guard);
    if (rc != HGP_OK) return fail(rc);

    // ---- L_max = floor((1 + eps) * ceil(c(V) / k))  (Sec. 2); the incident-weight check
    int64_t bw[67];
    CKF(cudaMemcpyAsync(bw, small, sizeof(bw), cudaMemcpyDeviceToHost, st));
    CKF(stream_wait(st));
    const int64_t maxw = bw[65];
    memcpy(host_err, &bw[66], sizeof(int32_t));
    if (host_err[0] & ERR_INVALID) return fail(HGP_ERR_INVALID);
    if (host_err[0] & ERR_UNSUPPORTED) return fail(HGP_ERR_UNSUPPORTED);
    h->max_vertex_netweight = maxw;
    d.bins = (int32_t)std::min<int64_t>(kBins, (maxw + kThreads) / kThreads * kThreads);   // > maxw
    int64_t total = 0;
    for (int i = 0; i < k; ++i) total += bw[i];
    h->total_weight = total;
    const int64_t avg = (total + k - 1) / k;
    d.lmax = (int64_t)floor((1.0 + eps) * (double)avg);

    // the int64 offsets and the int32 partition copy are no longer needed
    for (int i = 0; i < h->n_allocs; ++i) {
        if (h->allocs[i] && !in_arena(h, h->allocs[i]) &&
            (h->allocs[i] == off64 || h->allocs[i] == part_in || h->allocs[i] == block_sums ||
             h->allocs[i] == tmp)) {
            dev_free(h->allocs[i], st);
            h->allocs[i] = nullptr;
        }
    }
    if (in_arena(h, tmp)) h->scratch_n = tmp;   // max(n, m) + 1 entries, free from here on
    rc = ensure_stats(h, 16);
    if (rc != HGP_OK) return fail(rc);
    // the event a batch records its end on (see settle); made here, on the creating thread
    CKF(cudaEventCreateWithFlags(&h->ev_batch, cudaEventDisableTiming));
    *out = h;
    return HGP_OK;
#undef CKF
}

}  // namespace

// ================================================================== C ABI
extern "C" {

void hgp_default_options(hgp_options *opt)
{
    if (!opt) return;
    memset(opt, 0, sizeof(*opt));
    opt->subrounds = 4;
}

int hgp_set_blocking_waits(int32_t on)
{
    hgp::g_blocking_waits.store(on ? 1 : 0, std::memory_order_relaxed);
    return HGP_OK;
}

int hgp_set_pool_retention(int64_t bytes)
{
    if (bytes < 0) return HGP_ERR_INVALID;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = hgp::library_pool(&pool);
    uint64_t v = (uint64_t)bytes;
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &v);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return HGP_OK;
}

int hgp_get_pool_usage(int64_t *used, int64_t *kept)
{
    cudaMemPool_t pool = nullptr;
    uint64_t in_use = 0, reserved = 0;
    cudaError_t e = hgp::library_pool(&pool);
    if (e == cudaSuccess) e = cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &in_use);
    if (e == cudaSuccess) e = cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    if (used) *used = (int64_t)in_use;
    if (kept) *kept = (int64_t)(reserved > in_use ? reserved - in_use : 0);
    return HGP_OK;
}

const char *hgp_strerror(int code)
{
    switch (code) {
    case HGP_OK: return "ok";
    case HGP_ERR_INVALID: return "invalid argument";
    case HGP_ERR_OOM: return "out of memory";
    case HGP_ERR_UNSUPPORTED: return "unsupported size or parameter";
    case HGP_ERR_CUDA: return "CUDA error";
    case HGP_ERR_TIMEOUT: return "device wait timed out";
    case HGP_ERR_INTERNAL: return "internal consistency check failed";
    default: return "unknown status";
    }
}

int hgp_create(int32_t n, int32_t m, const int64_t *net_offsets, const int32_t *pins,
               const int32_t *vertex_w, const int32_t *net_w, int32_t k, double eps,
               const int32_t *initial_part, const hgp_options *opt, hgp_handle **out)
{
    return create_impl(n, m, net_offsets, pins, vertex_w, net_w, k, eps, initial_part, opt, out, false);
}

int hgp_create_device(int32_t n, int32_t m, const int64_t *net_offsets, const int32_t *pins,
                      const int32_t *vertex_w, const int32_t *net_w, int32_t k, double eps,
                      const int32_t *initial_part, const hgp_options *opt, hgp_handle **out)
{
    return create_impl(n, m, net_offsets, pins, vertex_w, net_w, k, eps, initial_part, opt, out, true);
}

// Releases are queued on the handle's stream behind its pending work (and behind the batch
// work that hgp_batch_refine ordered before it), so the call does not wait for the device.
void hgp_destroy(hgp_handle *h)
{
    if (!h) return;
    settle(h);
    if (h->graph_exec) cudaGraphExecDestroy(h->graph_exec);
    for (int i = 0; i < h->n_allocs; ++i)
        if (h->allocs[i]) dev_free(h->allocs[i], h->stream);
    for (int32_t i = 0; i < h->n_events; ++i) cudaEventDestroy(h->events[i]);
    if (h->ev_batch) cudaEventDestroy(h->ev_batch);
    delete[] h->events;
    delete[] h->event_phase;
    delete[] h->event_count;
    if (h->d.stats && !in_arena(h, h->d.stats)) dev_free(h->d.stats, h->stream);
    if (h->d_dev && !in_arena(h, h->d_dev)) dev_free(h->d_dev, h->stream);
    free(h->h_stats);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    (void)cudaGetLastError();
    delete h;
}

int hgp_set_partition(hgp_handle *h, const int32_t *part, int32_t on_device)
{
    if (!h || !part) return HGP_ERR_INVALID;
    settle(h);
    Dev &d = h->d;
    cudaStream_t st = h->stream;
    // two launches and one read-back: the check stages the 1-byte partition and its block weights, and
    // once it is known to be valid (else the handle keeps its state) k_init_nets does the rest.  A
    // device partition is read where it is, if it is in this device's memory.  10k vertices: 110 ->
    // 28 us a call.
    const int32_t *src = part;
    int32_t *tmp = nullptr;
    cudaError_t e = cudaSuccess;
    if (!on_device || (reinterpret_cast<uintptr_t>(part) & 3) ||
        !readable_in_place(part, sizeof(int32_t) * (size_t)d.n, h->device)) {
        tmp = h->scratch_n;
        if (!tmp) CK(dev_alloc(reinterpret_cast<void **>(&tmp), sizeof(int32_t) * (size_t)d.n, st));
        src = tmp;
        e = cudaMemcpyAsync(tmp, part, sizeof(int32_t) * (size_t)d.n,
                            on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st);
    }
    int32_t err = 0;
    if (e == cudaSuccess) {
        k_stage_partition<<<grid_for(d.n, 256, 152 * 8), 256, 0, st>>>(src, d.n, d.k, d.vw, h->part_next, d.acc, d.err);
        h->launches++;
        e = cudaGetLastError();
    }
    if (tmp && tmp != h->scratch_n) pool_free(tmp, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, d.err, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = stream_wait(st);
    if (e == cudaSuccess && (err & ERR_INVALID)) {
        e = cudaMemsetAsync(d.err, 0, sizeof(int32_t), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(d.acc, 0, sizeof(unsigned long long) * kAccN, st);
        if (e == cudaSuccess) return HGP_ERR_INVALID;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return init_state(h, h->part_next, nullptr);
}

int hgp_export_state(hgp_handle *h, int32_t *part, uint8_t *moved_nets, int64_t *next_round,
                     int32_t *first_round)
{
    if (!h) return HGP_ERR_INVALID;
    settle(h);
    if (part) {
        const int rc = hgp_get_partition(h, part, 0);
        if (rc != HGP_OK) return rc;
    }
    if (moved_nets && h->d.m > 0) {
        Dev &d = h->d;
        uint8_t *tmp = nullptr;
        CK(dev_alloc(reinterpret_cast<void **>(&tmp), (size_t)d.m, h->stream));
        if (d.k <= 32)
            k_export_moved<Rec16><<<grid_for(d.m, 256), 256, 0, h->stream>>>(d, (int32_t)h->next_round,
                                                                             h->all_eligible ? 1 : 0, tmp);
        else
            k_export_moved<Rec32><<<grid_for(d.m, 256), 256, 0, h->stream>>>(d, (int32_t)h->next_round,
                                                                             h->all_eligible ? 1 : 0, tmp);
        h->launches++;
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(moved_nets, tmp, (size_t)d.m, cudaMemcpyDeviceToHost, h->stream);
        pool_free(tmp, h->stream);
        if (e == cudaSuccess) e = stream_wait(h->stream);
        CK(e);
    }
    if (next_round) *next_round = h->next_round;
    if (first_round) *first_round = h->all_eligible ? 1 : 0;
    return HGP_OK;
}

int hgp_import_state(hgp_handle *h, const int32_t *part, const uint8_t *moved_nets,
                     int64_t next_round, int32_t first_round)
{
    if (!h || !part || next_round < 0 || next_round >= ((int64_t)1 << 30)) return HGP_ERR_INVALID;
    settle(h);
    if (!first_round && !moved_nets && h->d.m > 0) return HGP_ERR_INVALID;
    int rc = hgp_set_partition(h, part, 0);
    if (rc != HGP_OK) return rc;
    Dev &d = h->d;
    const int32_t r = (int32_t)next_round;
    if (!first_round && d.m > 0) {
        uint8_t *tmp = nullptr;
        CK(dev_alloc(reinterpret_cast<void **>(&tmp), (size_t)d.m, h->stream));
        cudaError_t e = cudaMemcpyAsync(tmp, moved_nets, (size_t)d.m, cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess) {
            if (d.k <= 32) k_import_moved<Rec16><<<grid_for(d.m, 256), 256, 0, h->stream>>>(d, r, tmp);
            else k_import_moved<Rec32><<<grid_for(d.m, 256), 256, 0, h->stream>>>(d, r, tmp);
            h->launches++;
            e = cudaGetLastError();
        }
        pool_free(tmp, h->stream);
        if (e == cudaSuccess) e = stream_wait(h->stream);
        CK(e);
    }
    k_set_round_state<<<1, 32, 0, h->stream>>>(d.rs, r, first_round ? 0 : 1);
    h->launches++;
    CK(cudaGetLastError());
    CK(stream_wait(h->stream));
    h->next_round = next_round;
    h->all_eligible = first_round != 0;
    return HGP_OK;
}

int hgp_objective(hgp_handle *h, int64_t *out)
{
    if (!h || !out) return HGP_ERR_INVALID;
    settle(h);
    CK(cudaMemcpyAsync(out, h->d.obj, sizeof(int64_t), cudaMemcpyDeviceToHost, h->stream));
    CK(stream_wait(h->stream));
    return HGP_OK;
}

int hgp_objective_from_phi(hgp_handle *h, int64_t *out)
{
    if (!h || !out) return HGP_ERR_INVALID;
    settle(h);
    unsigned long long *tmp = nullptr;
    CK(dev_alloc(reinterpret_cast<void **>(&tmp), sizeof(*tmp), h->stream));
    cudaError_t e = objective_from_phi(h, reinterpret_cast<int64_t *>(tmp));
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, tmp, sizeof(int64_t), cudaMemcpyDeviceToHost, h->stream);
    pool_free(tmp, h->stream);
    if (e == cudaSuccess) e = stream_wait(h->stream);
    CK(e);
    return HGP_OK;
}

int hgp_get_partition(hgp_handle *h, int32_t *part, int32_t on_device)
{
    if (!h || !part) return HGP_ERR_INVALID;
    settle(h);
    Dev &d = h->d;
    cudaStream_t st = h->stream;
    if (on_device) {
        k_part_to_i32<<<grid_for(d.n, 256), 256, 0, st>>>(d.part, part, d.n); h->launches++;
        CK(cudaGetLastError());
        CK(stream_wait(st));
        return HGP_OK;
    }
    int32_t *tmp = h->scratch_n;
    if (!tmp) CK(dev_alloc(reinterpret_cast<void **>(&tmp), sizeof(int32_t) * (size_t)d.n, st));
    k_part_to_i32<<<grid_for(d.n, 256), 256, 0, st>>>(d.part, tmp, d.n); h->launches++;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(part, tmp, sizeof(int32_t) * (size_t)d.n, cudaMemcpyDeviceToHost, st);
    if (tmp != h->scratch_n) pool_free(tmp, st);
    if (e == cudaSuccess) e = stream_wait(st);
    CK(e);
    return HGP_OK;
}

int hgp_get_block_weights(hgp_handle *h, int64_t *w)
{
    if (!h || !w) return HGP_ERR_INVALID;
    settle(h);
    CK(cudaMemcpyAsync(w, h->d.bw, sizeof(int64_t) * h->d.k, cudaMemcpyDeviceToHost, h->stream));
    CK(stream_wait(h->stream));
    return HGP_OK;
}

int hgp_get_phi(hgp_handle *h, int32_t *phi)
{
    if (!h || !phi) return HGP_ERR_INVALID;
    settle(h);
    Dev &d = h->d;
    const int64_t total = (int64_t)d.m * d.k;
    if (total == 0) return HGP_OK;
    int32_t *tmp = nullptr;
    CK(dev_alloc(reinterpret_cast<void **>(&tmp), sizeof(int32_t) * (size_t)total, h->stream));
    k_widen_phi<<<grid_for(total, 256), 256, 0, h->stream>>>(d, tmp); h->launches++;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(phi, tmp, sizeof(int32_t) * (size_t)total, cudaMemcpyDeviceToHost, h->stream);
    pool_free(tmp, h->stream);
    if (e == cudaSuccess) e = stream_wait(h->stream);
    CK(e);
    return HGP_OK;
}

int hgp_get_lambda(hgp_handle *h, uint64_t *lam)
{
    if (!h || !lam) return HGP_ERR_INVALID;
    settle(h);
    Dev &d = h->d;
    if (d.m == 0) return HGP_OK;
    uint64_t *tmp = nullptr;
    CK(dev_alloc(reinterpret_cast<void **>(&tmp), sizeof(uint64_t) * (size_t)d.m, h->stream));
    if (d.k <= 32) { k_get_lambda<Rec16><<<grid_for(d.m, 256), 256, 0, h->stream>>>(d, tmp); h->launches++; }
    else { k_get_lambda<Rec32><<<grid_for(d.m, 256), 256, 0, h->stream>>>(d, tmp); h->launches++; }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(lam, tmp, sizeof(uint64_t) * (size_t)d.m, cudaMemcpyDeviceToHost, h->stream);
    pool_free(tmp, h->stream);
    if (e == cudaSuccess) e = stream_wait(h->stream);
    CK(e);
    return HGP_OK;
}

int hgp_get_info(hgp_handle *h, int32_t *n, int32_t *m, int32_t *k, int64_t *pins, int64_t *lmax,
                 int32_t *phi_width, int32_t *wide_nets, int64_t *next_round)
{
    if (!h) return HGP_ERR_INVALID;
    if (n) *n = h->d.n;
    if (m) *m = h->d.m;
    if (k) *k = h->d.k;
    if (pins) *pins = h->d.P;
    if (lmax) *lmax = h->d.lmax;
    if (phi_width) *phi_width = h->d.phi_w;
    if (wide_nets) *wide_nets = h->n_wide;
    if (next_round) *next_round = h->next_round;
    return HGP_OK;
}

int hgp_refine(hgp_handle *h, int32_t rounds, hgp_round_stats *stats)
{
    if (!h || rounds < 0) return HGP_ERR_INVALID;
    settle(h);
    return refine_rounds(h, rounds, stats);
}

int hgp_debug_candidates(hgp_handle *h, int32_t s, int32_t *target, int64_t *gain)
{
    if (!h || !target || !gain || s < 0 || s >= h->d.S) return HGP_ERR_INVALID;
    settle(h);
    return debug_candidates(h, s, target, gain);
}

}  // extern "C"

namespace hgp {

cudaError_t objective_from_phi(hgp_handle *h, int64_t *d_out)
{
    cudaError_t e = cudaMemsetAsync(d_out, 0, sizeof(int64_t), h->stream);
    if (e != cudaSuccess) return e;
    k_obj_from_phi<<<grid_for(h->d.m, 256), 256, 0, h->stream>>>(h->d, reinterpret_cast<unsigned long long *>(d_out)); h->launches++;
    return cudaGetLastError();
}

}  // namespace hgp
