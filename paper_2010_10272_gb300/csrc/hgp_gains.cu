// libhgp: exact gains of a move sequence in parallel (paper Sec. 5.4, Lemma 1).
//
// For moves m_1..m_t (vertex u_j from block a_j to b_j, every vertex at most once), the gain of
// m_j if m_1..m_{j-1} were performed first is
//     omega({e in I(u_j) : Phi_j(e, a_j) = 1}) - omega({e in I(u_j) : Phi_j(e, b_j) = 0}),
// with Phi_j the pin counts before m_j.  Lemma 1 turns both conditions into order statistics
// of the moves touching (e, i):
//     Phi_j(e, a) = 1  <=>  Psi(e, a) = 0, j = max out(e, a), min in(e, a) > j
//     Phi_j(e, b) = 0  <=>  Psi(e, b) = 0, j = min in(e, b),  max out(e, b) < j
// where out / in are the moves of a pin of e out of / into the block and
// Psi(e, i) = Phi_1(e, i) - |out(e, i)|.  Pass 1 records, per touched (e, i), max out, min in
// and |out| with atomics; pass 2 evaluates the conditions per move.  The (e, i) entries live in
// an open-addressing hash table sized to the moves (the paper's dense table is O(|E| k)).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "hgp_host.cuh"

using namespace hgp;

namespace {

constexpr unsigned long long kEmpty = ~0ull;
constexpr unsigned kFull = 0xffffffffu;

// order statistics of one (net, block), one 32-byte sector; all bytes 0xFF when free, so a memset
// clears the table
struct __align__(32) Slot {
    unsigned long long key;   // e * 64 + i, kEmpty when free
    int32_t max_out;          // largest index of a move out of block i with a pin of e, -1 if none
    uint32_t min_in;          // smallest index of a move into block i, 0xFFFFFFFF if none
    int32_t n_out;            // |out(e, i)| - 1
    int32_t pad[3];
};

__device__ __forceinline__ uint64_t slot_hash(uint64_t key) { return splitmix64_output(key); }

// find or insert (linear probing; the table is at most two thirds full, so a free slot exists).
// cur: the key at the first position, already loaded.
// Keys are read through L1: one that is there never changes, and a free slot read too late is settled by
// the compare-and-swap (the slots of a large net are read by every move of its pins).
__device__ __forceinline__ Slot *find_slot(Slot *table, uint64_t mask, uint64_t p, unsigned long long cur,
                                           unsigned long long key, bool insert)
{
    for (uint64_t probe = 0; probe <= mask; ++probe) {
        Slot *s = table + p;
        if (cur == key) return s;
        if (cur == kEmpty) {
            if (!insert) return nullptr;
            cur = atomicCAS(&s->key, kEmpty, key);
            if (cur == kEmpty || cur == key) return s;
        }
        p = (p + 1) & mask;
        cur = table[p].key;
    }
    return nullptr;
}

// the slots of (e, a) and (e, b); the first probes of both are in flight together
__device__ __forceinline__ void find_both(Slot *table, uint64_t mask, unsigned long long e, int a, int b, bool insert,
                                          Slot *&sa, Slot *&sb)
{
    const unsigned long long ka = e * 64 + a, kb = e * 64 + b;
    const uint64_t pa = slot_hash(ka) & mask, pb = slot_hash(kb) & mask;
    const unsigned long long ca = table[pa].key, cb = table[pb].key;
    sa = find_slot(table, mask, pa, ca, ka, insert);
    sb = find_slot(table, mask, pb, cb, kb, insert);
}

// validation: vertex in range, moved once, from = Pi(u), to in range and different; and the sum of
// the degrees of the moved vertices (each contributes 2 keys per incident net).  out: error, sum, largest
// degree
__global__ void k_eg_check(Dev d, const int32_t *moves, int32_t count, int32_t *seen, unsigned long long *out)
{
    unsigned long long s = 0;
    int32_t most = 0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < count;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = moves[3 * j], a = moves[3 * j + 1], b = moves[3 * j + 2];
        bool bad = u < 0 || u >= d.n || b < 0 || b >= d.k || a == b;
        if (!bad) {
            bad = d.part[u] != a || atomicExch(&seen[u], 1) != 0;
            const int32_t deg = d.vtx_off[u + 1] - d.vtx_off[u];
            s += (unsigned long long)deg;
            most = max(most, deg);
        }
        if (bad) atomicOr(&out[0], 1ull);
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    most = (int32_t)__reduce_max_sync(kFull, (unsigned)most);
    if ((threadIdx.x & 31) == 0 && s) {
        atomicAdd(&out[1], s);
        atomicMax(&out[2], (unsigned long long)most);
    }
}

// Up to this many moves (all of whose warps run at once) a warp takes one each: the chain of dependent
// accesses per 32 incidences is what a short sequence waits for (5k moves of 4 nets, 8 per warp: 144
// us, one: 119 us).
constexpr int kEgWarps = 152 * 32;
constexpr uint64_t kEgDense = 1 << 20;   // slots (32 MB) from which a table may be two thirds full,
constexpr uint64_t kEgHub = 128;         // unless a move has more nets than this

// `per` (at most 32) moves of a warp, about 32 incidences in all, one run that the lanes walk
// flattened (a warp per move left most lanes idle, 6 nets of 32; 32 moves per warp were as slow, too
// few warps for the chains of dependent accesses).  100k moves of 6 nets each, the whole call: 295 ->
// 253 us, of which the host copies and waits are about 100; 218 us with keys read through L1.
struct MoveWarp {
    int32_t off[33];
    int32_t jb[32];
    int32_t a[32], b[32];
    unsigned long long g[32];
    __device__ __forceinline__ int32_t load(const Dev &d, const int32_t *moves, int64_t j0, int32_t count, int per)
    {
        const int lane = threadIdx.x & 31;
        const int64_t j = j0 + lane;
        int32_t deg = 0, first = 0, ma = 0, mb = 0;
        if (j < count && lane < per) {
            const int32_t u = moves[3 * j];
            ma = moves[3 * j + 1];
            mb = moves[3 * j + 2];
            first = d.vtx_off[u];
            deg = d.vtx_off[u + 1] - first;
        }
        int32_t incl = deg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        __syncwarp();
        off[lane] = incl - deg;
        jb[lane] = first;
        a[lane] = ma;
        b[lane] = mb;
        g[lane] = 0;
        if (lane == 31) off[32] = incl;
        __syncwarp();
        return off[32];
    }
    __device__ __forceinline__ int slot(int32_t i) const
    {
        int v = 0;
#pragma unroll
        for (int st = 16; st; st >>= 1)
            if (off[v + st] <= i) v += st;
        return v;
    }
};

// order statistics of every (net, block) the moves touch
__global__ void __launch_bounds__(256) k_eg_pass1(Dev d, const int32_t *moves, int32_t count, int per, Slot *table,
                                                  uint64_t mask, unsigned long long *out)
{
    __shared__ MoveWarp mw[8];
    MoveWarp &w = mw[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t j0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * per; j0 < count; j0 += warps * per) {
        const int32_t total = w.load(d, moves, j0, count, per);
        for (int32_t i = lane; i < total; i += 32) {
            const int v = w.slot(i);
            const int32_t j = (int32_t)j0 + v;
            const unsigned long long e = (unsigned long long)(d.inc[w.jb[v] + (i - w.off[v])] & kNetMask);
            Slot *sa, *sb;
            find_both(table, mask, e, w.a[v], w.b[v], true, sa, sb);
            if (!sa || !sb) {
                atomicOr(&out[0], 2ull);
                continue;
            }
            atomicMax(&sa->max_out, j);
            atomicAdd(&sa->n_out, 1);
            atomicMin(&sb->min_in, (uint32_t)j);
        }
    }
}

// exact gain of every move from Lemma 1; Phi is only read where the order statistics leave it to decide
__global__ void __launch_bounds__(256) k_eg_pass2(Dev d, const int32_t *moves, int32_t count, int per, Slot *table,
                                                  uint64_t mask, int64_t *gains)
{
    __shared__ MoveWarp mw[8];
    MoveWarp &w = mw[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * 8;
    const Rec16 *r16 = reinterpret_cast<const Rec16 *>(d.rec);
    const Rec32 *r32 = reinterpret_cast<const Rec32 *>(d.rec);
    for (int64_t j0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * per; j0 < count; j0 += warps * per) {
        const int32_t total = w.load(d, moves, j0, count, per);
        // a lane's sum over the incidences of one move, added to the move's when the lane leaves it (32
        // lanes adding to one hub's sum at every step: 15.3 instead of 14.5 ms in the case below)
        long long g = 0;
        int at = 0;
        for (int32_t i = lane; i < total; i += 32) {
            const int v = w.slot(i);
            if (v != at) {
                if (g) atomicAdd(&w.g[at], (unsigned long long)g);
                g = 0;
                at = v;
            }
            const int32_t j = (int32_t)j0 + v, a = w.a[v], b = w.b[v];
            const int32_t eraw = d.inc[w.jb[v] + (i - w.off[v])];
            const int32_t e = eraw & kNetMask;
            const bool wide = eraw < 0;
            const int32_t wrow = wide ? d.widx[e] : 0;
            const int32_t we = (d.k <= 32 ? r16[e].w : r32[e].w) & 0x7fffffff;
            Slot *sa, *sb;
            find_both(table, mask, (unsigned long long)e, a, b, false, sa, sb);
            if (sa && sa->max_out == j && sa->min_in > (uint32_t)j && sa->n_out + 1 == phi_get(d, e, a, wide, wrow)) g += we;
            if (sb && sb->min_in == (uint32_t)j && sb->max_out < j && sb->n_out + 1 == phi_get(d, e, b, wide, wrow)) g -= we;
        }
        if (g) atomicAdd(&w.g[at], (unsigned long long)g);
        __syncwarp();
        if (lane < per && j0 + lane < count) gains[j0 + lane] = (int64_t)w.g[lane];
        __syncwarp();
    }
}

int grid_of(int64_t work, int threads)
{
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 152 * 32) g = 152 * 32;
    return (int)g;
}

}  // namespace

extern "C" int hgp_exact_gains(hgp_handle *h, int32_t count, const int32_t *moves, int64_t *gains)
{
    if (!h || count < 0 || (count > 0 && (!moves || !gains))) return HGP_ERR_INVALID;
    settle(h);
    if (count == 0) return HGP_OK;
    Dev &d = h->d;
    cudaStream_t st = h->stream;
    Slot *table = nullptr;
    char *buf = nullptr;
    unsigned long long host[3] = {0, 0, 0};
    int rc = HGP_OK;
    // one buffer (five took 10 us more): error, degree sum and maximum, seen flags (both zeroed), gains, moves
    const size_t zero_bytes = (sizeof(host) + sizeof(int32_t) * (size_t)d.n + 15) / 16 * 16;
    const size_t g_bytes = sizeof(int64_t) * (size_t)count;
    cudaError_t e = dev_alloc(reinterpret_cast<void **>(&buf), zero_bytes + g_bytes + sizeof(int32_t) * 3 * (size_t)count, st);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(buf);
    int32_t *seen = reinterpret_cast<int32_t *>(buf + sizeof(host));
    int64_t *g_d = reinterpret_cast<int64_t *>(buf + zero_bytes);
    int32_t *mv = reinterpret_cast<int32_t *>(buf + zero_bytes + g_bytes);
    if (e == cudaSuccess) e = cudaMemcpyAsync(mv, moves, sizeof(int32_t) * 3 * (size_t)count, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(buf, 0, zero_bytes, st);
    if (e == cudaSuccess) {
        k_eg_check<<<grid_of(count, 256), 256, 0, st>>>(d, mv, count, seen, out);
        h->launches += 1;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(host, out, sizeof(host), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = stream_wait(st);
    if (e == cudaSuccess && host[0]) rc = HGP_ERR_INVALID;
    // at most 2 keys per incident net of a moved vertex.  The table is at most half full while it is small
    // or a move has many nets, two thirds above: a chain of accesses waits for the longest run of probes of
    // every 32, and few moves (5.4k: 114 -> 96 us) or one of a hub wait for a chain (50k moves of 1M
    // vertices with Zipf degrees, one of 21,185 nets: 14.5 ms two thirds full, 8.1 half full)
    uint64_t size = 64;
    while (size < (size < kEgDense || host[2] > kEgHub ? 4 : 3) * (uint64_t)host[1]) size <<= 1;
    if (e == cudaSuccess && rc == HGP_OK) {
        e = dev_alloc(reinterpret_cast<void **>(&table), sizeof(Slot) * size, st);
        // on a nearly full device, half the slots if those still hold every key
        if (e == cudaErrorMemoryAllocation && size / 2 >= 2 * (uint64_t)host[1]) {
            size /= 2;
            e = dev_alloc(reinterpret_cast<void **>(&table), sizeof(Slot) * size, st);
        }
    }
    if (e == cudaSuccess && rc == HGP_OK) e = cudaMemsetAsync(table, 0xFF, sizeof(Slot) * size, st);
    if (e == cudaSuccess && rc == HGP_OK) {
        const uint64_t fit = 32 * (uint64_t)count / std::max<uint64_t>(1, host[1]);   // moves of 32 incidences
        const int per = (int)std::max<uint64_t>(1, std::min<uint64_t>({32, fit, (uint64_t)count / kEgWarps}));
        const int grid = grid_of(((int64_t)count + per - 1) / per * 32, 256);
        k_eg_pass1<<<grid, 256, 0, st>>>(d, mv, count, per, table, size - 1, out);
        k_eg_pass2<<<grid, 256, 0, st>>>(d, mv, count, per, table, size - 1, g_d);
        h->launches += 2;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && rc == HGP_OK) e = cudaMemcpyAsync(host, out, sizeof(host), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && rc == HGP_OK) e = cudaMemcpyAsync(gains, g_d, g_bytes, cudaMemcpyDeviceToHost, st);
    if (buf) pool_free(buf, st);
    if (table) pool_free(table, st);
    const cudaError_t e2 = stream_wait(st);
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    if (rc == HGP_OK && host[0]) rc = HGP_ERR_INTERNAL;
    return rc;
}
