// libhgp: the gain step (best target and gain per vertex) without any device allocation.
//
// Some callers cannot allocate device memory at the point where they need this computation:
// code that runs while the application's own allocator owns the whole device (frameworks that
// reserve HBM up front and forbid other allocations), code inside host callbacks or other
// contexts where cudaMalloc is not permitted, and latency-critical paths that must not block
// on the allocator.  hgp_candidates_noalloc serves them: it takes every input and output as a
// caller-owned device buffer and keeps its only scratch (per-net records and block weights)
// in a fixed file-scope device array.
//
// The scratch array has room for kNoAllocMaxNets nets.  Every GPU that loads the library holds
// it until the process exits.  Its device address is looked up once per device, on the first
// call made with that device current; that first call should therefore come before any
// stream capture.  No call may be made while its stream is being captured (it reads the
// validation result back and synchronises the stream); such a call returns HGP_ERR_INVALID.
// All calls share the array and it keeps the last call's contents, so calls whose work
// overlaps on the GPU (on different streams, or from several host threads) race.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "hgp_host.cuh"

using namespace hgp;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int32_t kNoAllocMaxNets = 1 << 18;
constexpr int kMaxDevices = 64;

// scratch layout (bytes): [0, 512) block weights int64[64]; [512, 516) error flag; [520, 528)
// falling steps of the lists (see k_na_prepare); [1024, ...) one 32-byte record per net
struct __align__(16) NaRec {
    uint64_t s1;     // bit i: Phi(e,i) == 1
    uint64_t lam;    // bit i: Phi(e,i) > 0
    int32_t w;       // omega(e)
    int32_t pad[3];
};
constexpr size_t kRecOffset = 1024;
constexpr size_t kScratchBytes = kRecOffset + (size_t)kNoAllocMaxNets * sizeof(NaRec);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_mu;
void *g_addr[kMaxDevices];

int scratch_address(void **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return HGP_ERR_CUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) return HGP_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[dev]) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            (void)cudaGetLastError();
            return HGP_ERR_CUDA;
        }
        g_addr[dev] = p;
    }
    *out = g_addr[dev];
    return HGP_OK;
}

constexpr int kLaneNet = 16;   // nets of up to this many pins are read by one lane

__global__ void k_na_clear(int64_t *bw, int32_t *err)
{
    if (threadIdx.x < 64) bw[threadIdx.x] = 0;
    if (threadIdx.x < 4) err[threadIdx.x] = 0;   // and the falling steps
}

// input checks (every index the later kernels use must be in range)
__global__ void k_na_check(int32_t n, int32_t m, const int32_t *net_off, const int32_t *pins,
                           const int32_t *vtx_off, const int32_t *inc, const int32_t *vw,
                           const int32_t *nw, const int32_t *part, int32_t k, int32_t *err)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t P = net_off[m];
    bool bad = P < 0;
    for (int64_t e = i0; e <= m; e += stride) {
        const int32_t a = net_off[e];
        if ((e == 0 && a != 0) || (e == m && a != P) || (e < m && net_off[e + 1] < a)) bad = true;
        if (e < m && nw && nw[e] < 1) bad = true;
    }
    for (int64_t v = i0; v <= n; v += stride) {
        const int32_t a = vtx_off[v];
        if ((v == 0 && a != 0) || (v == n && a != P) || (v < n && vtx_off[v + 1] < a)) bad = true;
        if (v < n) {
            if (part[v] < 0 || part[v] >= k) bad = true;
            if (vw && vw[v] < 1) bad = true;
        }
    }
    for (int64_t j = i0; j < P; j += stride)
        if (pins[j] < 0 || pins[j] >= n || inc[j] < 0 || inc[j] >= m) bad = true;
    if (bad) atomicOr(err, 1);
}

// After k_na_check (does nothing if that found an error), in one launch:
//   * order: pins strictly increasing inside each net (this also excludes a pin listed twice) and
//     net ids strictly increasing inside each vertex's list.  The steps of both arrays that do not
//     increase are counted, those at the first entry of a list, which are allowed, are taken off:
//     zero is left exactly if every list increases (whatever the lists' lengths, every thread reads
//     with one stride);
//   * transpose: vertex v's list may name net e only if v is a pin of e (binary search in the sorted
//     pin list; a list out of order is reported by the first check).  With distinct entries per list
//     and P entries in total, the two CSRs then describe exactly the same incidences;
//   * block weights;
//   * records: Lambda(e) and S1(e) need no pin counts: a block seen again is no longer in S1.  A lane
//     per net of up to kLaneNet pins, else the warp.
// 250k nets, 1M pins: 140 us as four launches -> 28.
__global__ void __launch_bounds__(256) k_na_prepare(int32_t n, int32_t m, const int32_t *net_off, const int32_t *pins,
                                                    const int32_t *vtx_off, const int32_t *inc, const int32_t *part,
                                                    const int32_t *vw, const int32_t *nw, NaRec *recs, int64_t *bw,
                                                    int32_t *err)
{
    if (*reinterpret_cast<volatile int32_t *>(err)) return;
    __shared__ unsigned long long w[64];
    __shared__ int falls_s;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 64) w[threadIdx.x] = 0;
    if (threadIdx.x == 0) falls_s = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t P = net_off[m];
    bool bad = false;
    int falls = 0;
    for (int64_t j = i0 + 1; j < P; j += stride) falls += (pins[j - 1] >= pins[j]) + (inc[j - 1] >= inc[j]);
    for (int64_t v = i0; v < n; v += stride) {
        const int32_t b = vtx_off[v], end = vtx_off[v + 1];
        if (b > 0 && b < end) falls -= inc[b - 1] >= inc[b];
        for (int32_t j = b; j < end; ++j) {
            const int32_t e = inc[j];
            int32_t lo = net_off[e];
            const int32_t hi0 = net_off[e + 1];
            int32_t hi = hi0;
            while (lo < hi) {
                const int32_t mid = lo + ((hi - lo) >> 1);
                if (pins[mid] < v) lo = mid + 1;
                else hi = mid;
            }
            if (lo >= hi0 || pins[lo] != (int32_t)v) bad = true;
        }
        atomicAdd(&w[part[v]], (unsigned long long)(vw ? vw[v] : 1));
    }
    for (int64_t e0 = i0 - lane; e0 < m; e0 += stride) {
        const int64_t e = e0 + lane;
        int32_t b = 0, end = 0;
        if (e < m) {
            b = net_off[e];
            end = net_off[e + 1];
            if (b > 0 && b < end) falls -= pins[b - 1] >= pins[b];
        }
        uint64_t lam = 0, again = 0;
        if (end - b <= kLaneNet) {
            for (int32_t j = b; j < end; ++j) {
                const uint64_t bit = 1ull << part[pins[j]];
                again |= lam & bit;
                lam |= bit;
            }
        }
        unsigned big = __ballot_sync(kFull, end - b > kLaneNet);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int32_t bb = __shfl_sync(kFull, b, src), be = __shfl_sync(kFull, end, src);
            uint64_t l = 0, a = 0;
            for (int32_t j = bb + lane; j < be; j += 32) {
                const uint64_t bit = 1ull << part[pins[j]];
                a |= l & bit;
                l |= bit;
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {   // a block of both halves is a block seen again
                const uint64_t l2 = __shfl_xor_sync(kFull, l, o), a2 = __shfl_xor_sync(kFull, a, o);
                a |= a2 | (l & l2);
                l |= l2;
            }
            if (lane == src) {
                lam = l;
                again = a;
            }
        }
        if (e < m) {
            NaRec r;
            r.s1 = lam & ~again;
            r.lam = lam;
            r.w = nw ? nw[e] : 1;
            r.pad[0] = r.pad[1] = r.pad[2] = 0;
            recs[e] = r;
        }
    }
    if (__any_sync(kFull, bad) && lane == 0) atomicOr(err, 1);
    falls = __reduce_add_sync(kFull, falls);
    if (lane == 0 && falls) atomicAdd(&falls_s, falls);
    __syncthreads();
    if (threadIdx.x < 64 && w[threadIdx.x])
        atomicAdd(reinterpret_cast<unsigned long long *>(&bw[threadIdx.x]), w[threadIdx.x]);
    if (threadIdx.x == 0 && falls_s)   // next to the error flag, read with it
        atomicAdd(reinterpret_cast<unsigned long long *>(err + 2), (unsigned long long)(long long)falls_s);
}

// conn_t for every block at once in NP bit planes (bit t of plane p is bit p of conn_t; W < 2^NP), then
// the block of T with the largest, smallest id among equals
template <int NP>
__device__ __forceinline__ void na_planes(const NaRec *recs, const int32_t *inc, int32_t jb, int32_t je, uint64_t T,
                                          int &t_out, int32_t &conn_out)
{
    uint64_t c[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) c[p] = 0;
    for (int32_t j = jb; j < je; ++j) {
        const NaRec &r = recs[inc[j]];
        const uint64_t x = r.lam & T;
        const int32_t w = r.w;
        uint64_t carry = 0;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const uint64_t ad = ((w >> p) & 1) ? x : 0ull;
            const uint64_t cp = c[p];
            c[p] = cp ^ ad ^ carry;
            carry = (cp & ad) | (carry & (cp ^ ad));
        }
    }
    uint64_t C = T;
#pragma unroll
    for (int p = NP - 1; p >= 0; --p) C = (C & c[p]) ? C & c[p] : C;
    t_out = __ffsll((long long)C) - 1;
    conn_out = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) conn_out |= (int32_t)((c[p] >> t_out) & 1) << p;
}

__device__ __forceinline__ void take_net(const NaRec &r, int a, int64_t &W, int64_t &b, uint64_t &T)
{
    W += r.w;
    if ((r.s1 >> a) & 1) {
        b += r.w;
        T |= r.lam;
    }
}

// blocks of T with room for weight cu
__device__ __forceinline__ uint64_t na_room(uint64_t T, const long long *slack, int32_t cu)
{
    for (uint64_t x = T; x; x &= x - 1) {
        const int t = __ffsll((long long)x) - 1;
        if (slack[t] < cu) T &= ~(1ull << t);
    }
    return T;
}

// A vertex of many nets by the whole warp: the lanes stride over its nets, then each keeps the sums of
// two blocks.  By one lane, which the 31 others of its warp wait for, 30k vertices with Zipf degrees up to
// 1,378 took 2.02 ms a call; 0.89 so, of which 0.76 are the transpose check.
constexpr int32_t kNaLaneDeg = 96;   // as kLaneDeg of the refinement rounds

__device__ __forceinline__ int64_t warp_sum(int64_t v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ void na_hub(const NaRec *recs, const int32_t *inc, int32_t jb, int32_t je, int a, int32_t cu,
                                       const long long *slack, int &t_best, int64_t &g_best)
{
    const int lane = threadIdx.x & 31;
    const int32_t deg = je - jb;
    int64_t W = 0, b = 0;
    uint64_t T = 0;
    for (int32_t i = lane; i < deg; i += 32) take_net(recs[inc[jb + i]], a, W, b, T);
    W = warp_sum(W);
    b = warp_sum(b);
    T = (uint64_t)__reduce_or_sync(kFull, (uint32_t)T) | ((uint64_t)__reduce_or_sync(kFull, (uint32_t)(T >> 32)) << 32);
    T = na_room(T & ~(1ull << a), slack, cu);
    t_best = -1;
    g_best = 0;
    if (T == 0) return;
    int64_t conn0 = 0, conn1 = 0;   // of blocks lane and lane + 32
    for (int32_t i0 = 0; i0 < deg; i0 += 32) {
        uint64_t lam = 0;
        int32_t w = 0;
        if (i0 + lane < deg) {
            const NaRec &r = recs[inc[jb + i0 + lane]];
            lam = r.lam & T;
            w = r.w;
        }
        const int nn = min(32, deg - i0);
        for (int q = 0; q < nn; ++q) {
            const uint32_t lo = __shfl_sync(kFull, (uint32_t)lam, q), hi = __shfl_sync(kFull, (uint32_t)(lam >> 32), q);
            const int32_t wq = __shfl_sync(kFull, w, q);
            conn0 += ((lo >> lane) & 1) ? wq : 0;
            conn1 += ((hi >> lane) & 1) ? wq : 0;
        }
    }
    // the larger gain, then the smaller block
    int64_t g = 0;
    int t = -1;
    if (((T >> lane) & 1) && b - W + conn0 > 0) {
        g = b - W + conn0;
        t = lane;
    }
    if (((T >> (lane + 32)) & 1) && b - W + conn1 > g) {
        g = b - W + conn1;
        t = lane + 32;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const int64_t g2 = __shfl_xor_sync(kFull, g, o);
        const int t2 = __shfl_xor_sync(kFull, t, o);
        if (g2 > g || (g2 == g && t2 >= 0 && t2 < t)) {
            g = g2;
            t = t2;
        }
    }
    t_best = t;
    g_best = g;
}

// The gain step of round 0 (every vertex eligible) for sub-round s, as in the refinement rounds:
// T = blocks of Lambda(e) over nets with Phi(e,a) = 1, minus a and the blocks without room; best t in
// T by g_t = b(u) - W + omega({e : t in Lambda(e)}), smallest block on ties; no candidate unless the
// gain is positive.  A warp takes kNaRange vertices, whose active ones it gathers to full lanes.
// 250k vertices, 1M pins: 34 -> 17 us.
constexpr int kNaRange = 128;

__global__ void __launch_bounds__(256) k_na_candidates(int32_t n, int32_t k, double eps, const int32_t *vtx_off,
                                                       const int32_t *inc, const NaRec *recs, const int32_t *part,
                                                       const int32_t *vw, const int64_t *bw, int32_t S, uint64_t seed,
                                                       int32_t s, int32_t *target, int64_t *gain)
{
    __shared__ long long slack[64];
    __shared__ uint8_t list_w[8][kNaRange];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint8_t *list = list_w[wid];
    if (threadIdx.x < 32) {
        long long total = 0;
        for (int i = lane; i < k; i += 32) total += bw[i];
        for (int o = 16; o; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
        const long long avg = (total + k - 1) / k;
        const long long lmax = (long long)floor((1.0 + eps) * (double)avg);
        for (int i = lane; i < 64; i += 32) slack[i] = i < k ? lmax - bw[i] : -1;
    }
    __syncthreads();
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t base = ((int64_t)blockIdx.x * 8 + wid) * kNaRange; base < n; base += warps * kNaRange) {
        int cnt = 0;
#pragma unroll
        for (int c = 0; c < kNaRange; c += 32) {
            const int64_t u = base + c + lane;
            const uint64_t z = splitmix64_output(seed ^ (uint64_t)(uint32_t)u);
            const bool on = u < n && (int32_t)(z % (uint64_t)S) == s;
            const unsigned om = __ballot_sync(kFull, on);
            if (on) list[cnt + __popc(om & ((1u << lane) - 1))] = (uint8_t)(c + lane);
            cnt += __popc(om);
            if (u < n && !on) {
                target[u] = -1;
                gain[u] = 0;
            }
        }
        __syncwarp();
        for (int i0 = 0; i0 < cnt; i0 += 32) {
            const bool on = i0 + lane < cnt;
            int64_t u = 0;
            int t_best = -1, a = 0;
            int64_t g_best = 0;
            int32_t cu = 1, jb = 0, je = 0;
            if (on) {
                u = base + list[i0 + lane];
                a = part[u];
                cu = vw ? vw[u] : 1;
                jb = vtx_off[u];
                je = vtx_off[u + 1];
            }
            const bool hub = je - jb > kNaLaneDeg;
            int64_t W = 0, b = 0;
            uint64_t T = 0;
            if (!hub) {
                for (int32_t j = jb; j < je; ++j) take_net(recs[inc[j]], a, W, b, T);
                T = na_room(T & ~(1ull << a), slack, cu);
            }
            const bool planes = T != 0 && W < 2048;
            const bool wide = __any_sync(kFull, planes && W >= 64);   // the warp takes one path
            if (planes) {
                int t;
                int32_t conn;
                if (wide) na_planes<11>(recs, inc, jb, je, T, t, conn);
                else na_planes<6>(recs, inc, jb, je, T, t, conn);
                const int64_t g = b - W + conn;
                if (g > 0) {
                    g_best = g;
                    t_best = t;
                }
            } else {
                // one pass over the nets per candidate block (registers only)
                for (uint64_t x = T; x; x &= x - 1) {
                    const int t = __ffsll((long long)x) - 1;
                    int64_t conn = 0;
                    for (int32_t j = jb; j < je; ++j) {
                        const NaRec &r = recs[inc[j]];
                        if ((r.lam >> t) & 1) conn += r.w;
                    }
                    const int64_t g = b - W + conn;
                    if (g > g_best) {
                        g_best = g;
                        t_best = t;
                    }
                }
            }
            for (unsigned hm = __ballot_sync(kFull, hub); hm; hm &= hm - 1) {
                const int src = __ffs(hm) - 1;
                int t;
                int64_t g;
                na_hub(recs, inc, __shfl_sync(kFull, jb, src), __shfl_sync(kFull, je, src), __shfl_sync(kFull, a, src),
                       __shfl_sync(kFull, cu, src), slack, t, g);
                if (lane == src) {
                    t_best = t;
                    g_best = g;
                }
            }
            if (on) {
                target[u] = t_best;
                gain[u] = g_best;
            }
        }
        __syncwarp();
    }
}

}  // namespace

extern "C" int hgp_candidates_noalloc(int32_t n, int32_t m, const int32_t *net_offsets,
                                      const int32_t *pins, const int32_t *vtx_offsets,
                                      const int32_t *inc_nets, const int32_t *vertex_w,
                                      const int32_t *net_w, int32_t k, double eps,
                                      const int32_t *part, int32_t subrounds, uint64_t seed,
                                      int32_t s, int32_t *target, int64_t *gain, void *cuda_stream)
{
    if (n < 1 || m < 0 || !net_offsets || !vtx_offsets || !part || !target || !gain)
        return HGP_ERR_INVALID;
    if (k < 2 || !(eps > 0.0 && eps < 1.0) || subrounds < 1 || s < 0 || s >= subrounds)
        return HGP_ERR_INVALID;
    if (k > 64 || subrounds > 64 || m > kNoAllocMaxNets) return HGP_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // the call reads sizes and the validation result back to the host and synchronises its
    // stream, which a stream capture forbids
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
        (void)cudaGetLastError();
        return HGP_ERR_INVALID;
    }
    if (cap != cudaStreamCaptureStatusNone) return HGP_ERR_INVALID;
    void *base = nullptr;
    int rc = scratch_address(&base);
    if (rc != HGP_OK) return rc;
    unsigned char *sc = reinterpret_cast<unsigned char *>(base);
    int64_t *bw = reinterpret_cast<int64_t *>(sc);
    int32_t *err = reinterpret_cast<int32_t *>(sc + 512);
    NaRec *recs = reinterpret_cast<NaRec *>(sc + kRecOffset);

    cudaError_t e = cudaSuccess;
    int dev = 0;
    cudaGetDevice(&dev);
    // offsets that are not plainly this device's are read by a copy first, which refuses what is no
    // device array; pins and lists may only be missing where there are no pins
    if (!pins || !inc_nets || !readable_in_place(net_offsets, sizeof(int32_t) * ((size_t)m + 1), dev)) {
        int32_t P = 0;
        e = cudaMemcpyAsync(&P, net_offsets + m, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return HGP_ERR_CUDA;
        }
        if (P < 0 || (P > 0 && (!pins || !inc_nets))) return HGP_ERR_INVALID;
    }

    // block weights start from zero and the error flag is cleared on every call
    k_na_clear<<<1, 64, 0, st>>>(bw, err);
    k_na_check<<<152 * 4, 256, 0, st>>>(n, m, net_offsets, pins, vtx_offsets, inc_nets, vertex_w,
                                        net_w, part, k, err);
    // the order and transpose checks, weights and records follow if every index is in range
    k_na_prepare<<<152 * 8, 256, 0, st>>>(n, m, net_offsets, pins, vtx_offsets, inc_nets, part, vertex_w, net_w, recs,
                                          bw, err);
    // one read-back: the error flag, and the falling steps that are not at the start of a list
    int64_t bad[2] = {0, 0};
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(bad, err, sizeof(bad), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return HGP_ERR_CUDA;
    }
    if ((int32_t)(bad[0] & 0xffffffff) != 0 || bad[1] != 0) return HGP_ERR_INVALID;

    const int64_t blocks = ((int64_t)n + 8 * kNaRange - 1) / (8 * kNaRange);
    k_na_candidates<<<(unsigned)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, st>>>(
        n, k, eps, vtx_offsets, inc_nets, recs, part, vertex_w, bw, subrounds, seed, s, target, gain);
    e = cudaGetLastError();
    if (e != cudaSuccess) return HGP_ERR_CUDA;
    return HGP_OK;
}
