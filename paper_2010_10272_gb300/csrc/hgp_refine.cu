// libhgp: synchronous label-propagation rounds (Sec. 6) on the device.
//
// One round r = round_prep, then for each sub-round s: gain -> approval -> apply, then
// round_end.  Kernels and what they compute:
//
//   k_round_prep   splitmix64(seed ^ (r << 32 | u)) mod S for every vertex, and per tile of 2048
//                  vertices a list of its vertices grouped by sub-round (id order kept); the
//                  sub-round kernels take such a list in segments of 32.
//   k_gain         for each active vertex u (a = Pi(u)), against the frozen state:
//                  W = omega(I(u)), b(u) = omega({e : Phi(e,a) = 1}) (Sec. 5), eligibility
//                  (a net of u moved in round r-1, Sec. 6), and the best target
//                  t = argmax_{i != a, feasible} g_i(u), g_i(u) = b(u) - p_i(u)
//                    = b(u) + omega({e in I(u) : i in Lambda(e)}) - W,
//                  ties to the smaller block; only blocks in the union of Lambda(e) over the
//                  nets with Phi(e,a) = 1 can have positive gain (g_i <= omega of those nets
//                  that contain i), so only those are evaluated.
//   k_select       per target block t whose candidates do not all fit (w(t) + sum c > L_max): the
//                  histogram of candidate weight by gain, filled by k_gain, scanned from the
//                  highest gain to find the threshold gain G_t and the budget left for
//                  candidates with gain == G_t (approval order (gain desc, id asc), inclusive
//                  prefix sums); k_hist refines gains beyond the histogram.
//   k_tie_sum/k_tie_cut   per tile weight of the gain == G_t candidates, then the vertex id up to
//                  which they fit the remaining budget (ties are approved in id order).
//   k_apply        applies every approved move: Pi(u) = t, block weights, Phi(e,a)--,
//                  Phi(e,t)++ with integer atomics, and Lambda(e), S1(e) and the objective
//                  from the atomics' old values (each step of a pin count across 0/1/2 toggles
//                  the matching bit, so the final bits are right whatever the order).
//   k_round_end    per-round objective and heaviest block; advances the device round state.
//
// A small instance runs all of this as one thread-block cluster in one launch (hgp_small.cuh).
//
// Every kernel takes the instance state as `const Dev *devs` in device memory and a list of
// work items (k_gain and k_apply of one handle take the state as a parameter).  A single-handle
// launch passes items == nullptr: item i is the handle's own tile / block i.  A batch launch passes
// (instance, local index) pairs covering many handles at once, so one launch per phase refines a
// whole batch.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <vector>

#include "hgp_host.cuh"

using namespace hgp;

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// instance and local index of work item i
__device__ __forceinline__ const Dev &item_of(const Dev *devs, const int2 *items, int32_t i, int32_t &local)
{
    if (items) {
        const int2 it = items[i];
        local = it.y;
        return devs[it.x];
    }
    local = i;
    return devs[0];
}

// The kernels of a round are launched with programmatic stream serialisation: the next one's CTAs are
// set up while the last CTAs of this one still run, and start with this wait for its end.  Every
// thread calls it before anything else (also those that then return), so the end of a kernel
// implies the end of all before it.  Row-net 2M, 10 rounds: 4.23 -> 3.83 ms; rebalancing 5M, 3 passes: 2.93 -> 2.57 ms.
__device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
}

enum { ITEM_TILE = 1, ITEM_BLOCK = 2 };
__device__ __forceinline__ int32_t item_count(const Dev *devs, const int2 *items, int32_t n_items, int kind)
{
    if (items) return n_items;
    return kind == ITEM_TILE ? devs[0].n_tiles : devs[0].k;
}

// A run of segments of one tile's candidates, spread over the lanes of a warp: candidate i of the
// run is in slot at(i).  At most 32 segments.
struct SegRun {
    int32_t off[33];    // exclusive prefix of the segments' counts
    int32_t slot0;      // first slot of the run (in Dev::cand / rv_src)
    __device__ __forceinline__ int32_t load(const Dev &d, int32_t tile, int32_t s0, int32_t s1)
    {
        const int lane = threadIdx.x & 31;
        const int32_t c = s0 + lane < s1 ? d.cand_cnt[(int64_t)tile * d.nseg + s0 + lane] : 0;
        int32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        __syncwarp();
        off[lane] = incl - c;
        if (lane == 31) off[32] = incl;
        if (lane == 0) slot0 = tile * kTile + s0 * kSeg;
        __syncwarp();
        return off[32];
    }
    __device__ __forceinline__ int32_t at(int32_t i) const
    {
        int v = 0;
#pragma unroll
        for (int st = 16; st; st >>= 1)
            if (off[v + st] <= i) v += st;
        return slot0 + v * kSeg + (i - off[v]);
    }
};

// the segments of a tile that warp wid of a CTA of kWarps takes: [s0, s1)
__device__ __forceinline__ void warp_segments(const Dev &d, int wid, int32_t &s0, int32_t &s1)
{
    const int32_t per = (d.nseg + kWarps - 1) / kWarps;
    s0 = min(d.nseg, wid * per);
    s1 = min(d.nseg, s0 + per);
}

// vertex of a candidate: its slot's tile and the offset in it
__device__ __forceinline__ int32_t cand_vertex(int32_t slot, int ul) { return slot / kTile * kTile + ul; }

// ------------------------------------------------------------------ round preparation
// CTA per tile item; warp w hashes the tile's vertices [256 w, 256 w + 256), 8 per lane
// r_ovr >= 0: hash with that round number instead of the device round state (rebalancing)
__global__ void __launch_bounds__(kThreads) k_round_prep(const Dev *devs, const int2 *items, int32_t n_items,
                                                         int32_t r_ovr = -1)
{
    after_previous();
    __shared__ int32_t cnt[64][kWarps];   // then the first list position of (sub-round, warp)
    __shared__ int32_t tot[64];
    constexpr int kPer = kTile / kThreads;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if ((int32_t)blockIdx.x >= item_count(devs, items, n_items, ITEM_TILE)) return;
    int32_t tile;
    const Dev &d = item_of(devs, items, blockIdx.x, tile);
    const int32_t r = r_ovr >= 0 ? r_ovr : d.rs[0];
    const uint64_t seed = d.seed;
    const int32_t S = d.S;
    const int32_t nv = min(kTile, d.n - tile * kTile);
    const bool pow2 = (S & (S - 1)) == 0;
    for (int i = tid; i < S * kWarps; i += kThreads) (&cnt[0][0])[i] = 0;
    __syncthreads();
    int sv[kPer];
    const int first = wid * (kTile / kWarps) + lane;
#pragma unroll
    for (int c = 0; c < kPer; ++c) {
        const int idx = first + c * 32;
        const uint32_t u = (uint32_t)(tile * kTile + idx);
        const uint64_t z = splitmix64_output(seed ^ (((uint64_t)(uint32_t)r << 32) | u));
        sv[c] = idx < nv ? (pow2 ? (int)(z & (uint64_t)(S - 1)) : (int)(z % (uint64_t)S)) : -1;
        const unsigned peers = __match_any_sync(kFull, sv[c]);
        if (sv[c] >= 0 && lane == __ffs(peers) - 1) cnt[sv[c]][wid] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    if (tid < S) {
        int32_t t = 0;
        for (int w = 0; w < kWarps; ++w) t += cnt[tid][w];
        tot[tid] = t;
    }
    __syncthreads();
    uint16_t *ss = d.sub_start + (int64_t)tile * (S + 1);
    if (tid <= S) {
        int32_t run = 0;
        for (int i = 0; i < tid; ++i) run += tot[i];
        ss[tid] = (uint16_t)run;
        if (tid < S)
            for (int w = 0; w < kWarps; ++w) {
                const int32_t c = cnt[tid][w];
                cnt[tid][w] = run;
                run += c;
            }
    }
    __syncthreads();
    uint16_t *list = d.sub_list + (int64_t)tile * kTile;
#pragma unroll
    for (int c = 0; c < kPer; ++c) {
        const unsigned peers = __match_any_sync(kFull, sv[c]);
        if (sv[c] >= 0) list[cnt[sv[c]][wid] + __popc(peers & lanemask_lt())] = (uint16_t)(first + c * 32);
        __syncwarp();
        if (sv[c] >= 0 && lane == __ffs(peers) - 1) cnt[sv[c]][wid] += __popc(peers);
        __syncwarp();
    }
}

// ------------------------------------------------------------------ gain + best target
template <typename Rec> struct RecIO;

// COH: the record may have been changed by another SM earlier in the same launch (hgp_small.cuh), so
// it is read from L2; else through the read-only path.
template <> struct RecIO<Rec16> {
    typedef uint32_t Lam;
    template <bool COH>
    __device__ static void load_full(const Rec16 *r, Lam &s1, int32_t &w, int32_t &mv, Lam &lam)
    {
        const uint4 *p = reinterpret_cast<const uint4 *>(r);
        const uint4 q = COH ? __ldcg(p) : __ldg(p);
        s1 = q.x; lam = q.y; w = (int32_t)q.z; mv = (int32_t)q.w;
    }
    template <bool COH>
    __device__ static void load_b(const Rec16 *r, Lam &lam, int32_t &w)
    {
        const uint4 *p = reinterpret_cast<const uint4 *>(r);
        const uint4 q = COH ? __ldcg(p) : __ldg(p);
        lam = q.y; w = (int32_t)q.z;
    }
};

template <> struct RecIO<Rec32> {
    typedef uint64_t Lam;
    // the whole record is one 32-byte load (records are 32-byte aligned)
    template <bool COH>
    __device__ static void load_full(const Rec32 *r, Lam &s1, int32_t &w, int32_t &mv, Lam &lam)
    {
        if (COH) {
            const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(r));
            const int2 l = __ldcg(reinterpret_cast<const int2 *>(&r->w));
            s1 = (uint64_t)q.x | ((uint64_t)q.y << 32); lam = (uint64_t)q.z | ((uint64_t)q.w << 32);
            w = l.x; mv = l.y;
            return;
        }
        uint64_t wm;
        [[maybe_unused]] uint64_t tail;
        asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(s1), "=l"(lam), "=l"(wm), "=l"(tail) : "l"(r));
        w = (int32_t)(uint32_t)wm; mv = (int32_t)(uint32_t)(wm >> 32);
    }
    template <bool COH>
    __device__ static void load_b(const Rec32 *r, Lam &lam, int32_t &w)
    {
        const unsigned long long *p = reinterpret_cast<const unsigned long long *>(&r->lam);
        lam = COH ? __ldcg(p) : __ldg(p);
        w = __ldg(&r->w);
    }
};

template <typename Lam> __device__ __forceinline__ uint32_t lo32(Lam x) { return (uint32_t)x; }
template <typename Lam> __device__ __forceinline__ uint32_t hi32(Lam x)
{
    return sizeof(Lam) == 8 ? (uint32_t)((uint64_t)x >> 32) : 0u;
}

__device__ __forceinline__ int slot_of(const int32_t *off, int32_t i)
{
    int v = 0;
#pragma unroll
    for (int st = 16; st; st >>= 1)
        if (off[v + st] <= i) v += st;
    return v;
}

// COH: the list may be a copy in shared memory
template <bool COH>
__device__ __forceinline__ int32_t load_inc(const int32_t *inc, int32_t j)
{
    return COH ? inc[j] : __ldg(&inc[j]);
}

constexpr int32_t kPlaneMaxW = 2047;   // W(u) up to this uses bit planes (NP <= 11)
// degrees above this are walked by the whole warp: its two passes cost about as many issue slots
// as a lane's walk of this length with the other lanes idle
constexpr int32_t kLaneDeg = 96;
constexpr int kHubPlanes = 13;         // bit planes of such a walk (with 16, kernels that keep within their
constexpr int32_t kHubMaxW = (1 << kHubPlanes) - 1;   // registers spill: row-net 2M 3.57 -> 3.66 ms)
// Segments of a rebalancing item, of the gain and of the apply step alike, with S sub-rounds: the active
// vertices of 256, 384 or 512 consecutive ids, as `share`, the vertices per warp of the apply step, grows.
// Its candidates lie together, so a larger item fills more lanes but also gives more of a run of hubs to
// one warp.  S = 4, ms a call with 2 / 3 / 4 segments (and with 6 in the gain and up to 9 in the apply step):
// planted 2M (share 411) 0.40 / 0.44 / 0.45 (0.48); power-law 5M (1,028) 1.79 / 1.67 / 1.71 (1.88) and
// numbered by falling Zipf degree 7.9 / 9.0 / 10.2 (15.2); 10M 2.93 / 2.68 / 2.60 (2.84); 50M (10,280)
// 13.3 / 12.0 / 11.2 (11.3), falling 32 / 35 / 37 (51).  S = 16, 5M falling, 1 / 2 / 6: 12.0 / 15.2 / 20.3.
inline int32_t rb_segments(int32_t S, int64_t share)
{
    const int32_t ids = share < 640 ? 256 : (share < 3200 ? 384 : 512);
    return std::min(6, std::max(1, ids / (kSeg * S)));
}
constexpr int kFeasW = 8;              // vertex weights up to this have a mask of blocks with room

// Per-warp state of the gain step that depends on the instance.
struct GainInst {
    int32_t r;           // round number
    int32_t all_elig;    // first round: every vertex eligible
};

// per-warp tables of the instance: room left per block, and the blocks with room for weight c
struct alignas(16) GainWarp {
    long long slack[64];
    unsigned long long feas[kFeasW + 1];
};

// Rebalancing pass settings (RB instances of the gain step).
struct RbArgs {
    int32_t r;       // round number of the sub-round hash for this pass
    int32_t phase;   // 1: gain >= 0 only; 2: any gain
    int32_t off;     // added to the gain to make the approval priority non-negative
    int32_t segs;    // segments of an item
};

// What one pass over a vertex's nets gives.
template <typename Lam>
struct Nets {
    Lam T;        // union of Lambda(e) over the nets with Phi(e,a) = 1
    Lam A2;       // intersection over the others (balance moves)
    int32_t b;    // omega of the nets with Phi(e,a) = 1
    int32_t elig; // a net moved in round r - 1
};

template <typename Lam>
__device__ __forceinline__ void take_net(Nets<Lam> &x, Lam s1, Lam lam, int32_t w, int32_t mv, int a, int32_t r)
{
    const bool alone = (s1 >> a) & 1;
    if (alone) {
        x.b += w;
        x.T |= lam;
    } else {
        x.A2 &= lam;
    }
    if (moved_in_prev_round(mv, r)) x.elig = 1;
}

// blocks of T with room for weight cu
template <typename Lam>
__device__ __forceinline__ Lam with_room(Lam T, const GainWarp &g, int32_t cu)
{
    if (cu <= kFeasW) return T & (Lam)g.feas[cu];
    for (Lam x = T; x; x &= x - 1) {
        const int t = lam_bits_ctz(x);
        if (g.slack[t] < cu) T &= ~((Lam)1 << t);
    }
    return T;
}

// One lane's vertex: a single walk over its nets that gathers each record once and accumulates
// b(u), T, eligibility and, for all blocks at once, conn_t = omega({e in I(u) : t in Lambda(e)})
// in NP bit planes held in registers (bit t of plane p is bit p of conn_t): adding omega(e) to
// every block of Lambda(e) is a ripple-carry addition on whole bitsets, O(NP) word operations
// whatever the number of blocks.  W(u) is known from creation, so NP is too (conn_t <= W(u) <
// 2^NP).  kAhead records are in flight per lane, and the net ids of the next ones (32-byte records, 3
// ahead on 3 CTAs per SM: 30.2 ms per power-law step, 2 on 4: 31.8, 4 on 3: 32.0, 1 on 4: 34.0).
// Then the block of T with room with the largest conn_t (smallest id among equals).  Against incidences spread over the lanes (a binary search
// and three shared-memory atomics each, (Lambda, omega) kept for a second pass over the nets):
// row-net 2M, k = 8, records in L2: 93 -> 56 us per launch of 5 M gathers (47 with full segments and
// overlapped launches); power-law 50M, k = 64, bound by random sectors from DRAM: 1.77 -> 1.65 ms per
// launch of 86 M (1.53 with the net ids loaded ahead).
template <typename Lam, typename Rec, int NP, bool UNIT, bool RB, bool COH>
__device__ __forceinline__ void lane_best(const Rec *recs, const int32_t *inc, int32_t jb, int32_t je, int a, int32_t r,
                                          const GainWarp &g, int32_t cu, Lam kall, int32_t eq_value, Nets<Lam> &x,
                                          Lam &T_all, Lam &T, int &t_out, int32_t &conn_out, Lam &eq_out)
{
    constexpr int kAhead = RB || (COH && sizeof(Lam) == 8) ? 2 : 3;   // by registers
    Lam c[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) c[p] = 0;
    int32_t e[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) e[q] = jb + q < je ? (load_inc<COH>(inc, jb + q) & kNetMask) : -1;
    for (int32_t j = jb; j < je; j += kAhead) {
        Lam s1[kAhead], lam[kAhead];
        int32_t w[kAhead], mv[kAhead];
        bool on[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            s1[q] = 0; lam[q] = 0; w[q] = 0; mv[q] = 0;
            on[q] = e[q] >= 0;
            if (on[q]) RecIO<Rec>::template load_full<COH>(recs + e[q], s1[q], w[q], mv[q], lam[q]);
        }
        // the next records' net ids, while these are on their way
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            const int32_t jn = j + kAhead + q;
            e[q] = jn < je ? (load_inc<COH>(inc, jn) & kNetMask) : -1;
        }
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            if (!on[q]) continue;
            const int32_t we = UNIT ? 1 : w[q] & 0x7fffffff;
            take_net(x, s1[q], lam[q], we, mv[q], a, r);
            if (UNIT) {
                Lam carry = lam[q];
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const Lam t = c[p] & carry;
                    c[p] ^= carry;
                    carry = t;
                }
            } else {
                Lam carry = 0;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const Lam ad = ((we >> p) & 1) ? lam[q] : (Lam)0;
                    const Lam cp = c[p];
                    c[p] = cp ^ ad ^ carry;
                    carry = (cp & ad) | (carry & (cp ^ ad));
                }
            }
        }
    }
    T_all = x.elig ? (RB ? kall : x.T) & ~((Lam)1 << a) : (Lam)0;
    T = with_room(T_all, g, cu);
    Lam C = T;
#pragma unroll
    for (int p = NP - 1; p >= 0; --p) {
        const Lam m = C & c[p];
        C = m ? m : C;
    }
    t_out = -1;
    conn_out = 0;
    eq_out = 0;
    if (T) {
        const int t = lam_bits_ctz(C);
#pragma unroll
        for (int p = 0; p < NP; ++p) conn_out |= (int32_t)((c[p] >> t) & 1) << p;
        t_out = t;
    }
    // balance moves: blocks of T with gain 0, conn_t = W - b (eq_value = W; < 0: not asked for)
    if (eq_value >= 0) {
        const int32_t v = eq_value - x.b;
        Lam eq = T;
#pragma unroll
        for (int p = 0; p < NP; ++p) eq &= ((v >> p) & 1) ? c[p] : ~c[p];
        eq_out = eq;
    }
}

// Level-0 histogram of an approval stage: each lane's weight cu (ok lanes) by key block and gain (or
// priority) bin, a reduction in L2.  Gains are small numbers, so a warp's candidates share bins: one
// reduction per distinct (block, bin).  The warp calls it together.
__device__ __forceinline__ void count_gain(const Dev &d, bool ok, int key, int32_t g, int32_t cu)
{
    const unsigned mask = __ballot_sync(kFull, ok);
    if (!ok) return;
    const int bin = g < kBins - 1 ? g : kBins - 1;
    const unsigned peers = __match_any_sync(mask, key * kBins + bin);
    // two halves: 32 sums of either fit 32 bits
    const unsigned long long sum = (unsigned long long)__reduce_add_sync(peers, (uint32_t)cu & 0xFFFFu) +
                                   ((unsigned long long)__reduce_add_sync(peers, (uint32_t)cu >> 16) << 16);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&d.hist[(int64_t)key * kBins + bin], sum);
}

// The sums conn_t of a vertex of many nets, those of blocks lane and lane + 32 in each lane: every lane
// adds its nets' weights into bit planes over the blocks of T (as lane_best; with 64 blocks a net has two
// lanes, one for either half, so that the planes are 32-bit words), and the lanes' planes are added
// pairwise.  Every net's bits passed around the warp instead (32 steps per 32 nets): 2M vertices, k = 8,
// numbered by falling degree (3,030 nets at most), gain step of 5 rounds 15.7 -> 9.7 ms with 4 sub-rounds,
// 57.9 -> 41.1 with 64; 5M power-law, k = 64, 64 sub-rounds 124 -> 107.
template <typename Lam, typename Rec, bool COH>
__device__ __forceinline__ void hub_planes(const Rec *recs, const int32_t *inc, int32_t jb, int32_t je, Lam T, int32_t &acc0,
                                           int32_t &acc1)
{
    constexpr bool kWide = sizeof(Lam) == 8;
    constexpr int NP = kHubPlanes, kNets = kWide ? 16 : 32;   // nets of a step
    const int lane = threadIdx.x & 31;
    const uint32_t mine = kWide && lane >= 16 ? hi32(T) : lo32(T);
    uint32_t c[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) c[p] = 0;
    for (int32_t j = jb + lane % kNets; j < je; j += kNets) {
        Lam lam;
        int32_t w;
        RecIO<Rec>::template load_b<COH>(recs + (load_inc<COH>(inc, j) & kNetMask), lam, w);
        const uint32_t x = (kWide && lane >= 16 ? hi32(lam) : lo32(lam)) & mine;
        uint32_t carry = 0;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const uint32_t ad = ((w >> p) & 1) ? x : 0u, cp = c[p];
            c[p] = cp ^ ad ^ carry;
            carry = (cp & ad) | (carry & (cp ^ ad));
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int o = kNets / 2; o; o >>= 1) {
        uint32_t carry = 0;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const uint32_t ad = __shfl_xor_sync(kFull, c[p], o), cp = c[p];
            c[p] = cp ^ ad ^ carry;
            carry = (cp & ad) | (carry & (cp ^ ad));
        }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        acc0 |= (int32_t)((__shfl_sync(kFull, c[p], 0) >> lane) & 1) << p;
        if (kWide) acc1 |= (int32_t)((__shfl_sync(kFull, c[p], 16) >> lane) & 1) << p;
    }
}

// The best target of the vertex in this lane (a = its block, cu its weight, [jb, je) its nets, W their
// weight, inc the incidence lists): block t_best (-1: none) and its gain; returns eligibility.  The
// warp calls it together.
template <typename Rec, bool RB, bool COH>
__device__ __forceinline__ bool gain_vertex(const Dev &d, const int32_t *inc, const GainWarp &g,
                                            const GainInst &gi, const RbArgs &rb, bool valid, int32_t a, int32_t cu, int32_t jb, int32_t je,
                                            int32_t W, int &t_best, int32_t &g_best)
{
    typedef typename RecIO<Rec>::Lam Lam;
    constexpr bool kWide = sizeof(Lam) == 8;
    const int lane = threadIdx.x & 31;
    const int32_t r = gi.r;
    const bool balance = !RB && (d.variant & 1) != 0;
    const Rec *recs = reinterpret_cast<const Rec *>(d.rec);
    const bool unit = d.nw == nullptr;
    const Lam kall = d.k >= (int)(8 * sizeof(Lam)) ? ~(Lam)0 : (((Lam)1 << d.k) - 1);
    Nets<Lam> x;
    x.T = 0; x.A2 = ~(Lam)0; x.b = 0;
    x.elig = valid && (RB || gi.all_elig);
    Lam T_all = 0, T = 0, zero_in = 0;
    t_best = -1;
    int32_t conn = 0;
    const bool heavy = valid && (W > kPlaneMaxW || je - jb > kLaneDeg);
    const bool light = valid && !heavy;
    const unsigned wmax = __reduce_max_sync(kFull, light ? (unsigned)W : 0u);
    if (light) {
        const int np = 32 - __clz((int)wmax);   // 2^np > wmax >= conn_t
        const int32_t eqv = balance ? W : -1;
#define HGP_LANE(NP, U) lane_best<Lam, Rec, NP, U, RB, COH>(recs, inc, jb, je, a, r, g, cu, kall, eqv, x, T_all, T, t_best, conn, zero_in)
        if (unit) {
            if (np <= 4) HGP_LANE(4, true);
            else HGP_LANE(7, true);             // at most kLaneDeg nets
        } else {
            if (np <= 6) HGP_LANE(6, false);
            else if (np <= 8) HGP_LANE(8, false);
            else HGP_LANE(11, false);
        }
#undef HGP_LANE
    }
    __syncwarp();
    const int32_t bw_ = x.b - W;
    g_best = bw_ + conn;
    if (!(light && t_best >= 0 && (RB ? (rb.phase == 2 || g_best >= 0) : g_best > 0))) {
        t_best = -1;
        g_best = 0;
    }
    // ---- vertices with many nets or large W: the whole warp on one vertex at a time
    unsigned hm = __ballot_sync(kFull, heavy);
    while (hm) {
        const int src = __ffs(hm) - 1;
        hm &= hm - 1;
        const int32_t hjb = __shfl_sync(kFull, jb, src), hje = __shfl_sync(kFull, je, src);
        const int32_t ha = __shfl_sync(kFull, a, src), hcu = __shfl_sync(kFull, cu, src);
        const int32_t hW = __shfl_sync(kFull, W, src);
        Nets<Lam> y;
        y.T = 0; y.A2 = ~(Lam)0; y.b = 0; y.elig = RB || gi.all_elig;
        for (int32_t j = hjb + lane; j < hje; j += 32) {
            Lam s1, lam;
            int32_t w, mv;
            RecIO<Rec>::template load_full<COH>(recs + (load_inc<COH>(inc, j) & kNetMask), s1, w, mv, lam);
            take_net(y, s1, lam, w & 0x7fffffff, mv, ha, r);
        }
        y.b = __reduce_add_sync(kFull, y.b);
        y.elig = __any_sync(kFull, y.elig);
        uint32_t tl = __reduce_or_sync(kFull, lo32(y.T)), al = __reduce_and_sync(kFull, lo32(y.A2));
        uint32_t th = kWide ? __reduce_or_sync(kFull, hi32(y.T)) : 0u;
        uint32_t ah = kWide ? __reduce_and_sync(kFull, hi32(y.A2)) : 0u;
        y.T = (Lam)((uint64_t)tl | ((uint64_t)th << 32));
        y.A2 = (Lam)((uint64_t)al | ((uint64_t)ah << 32));
        const Lam hTa = y.elig ? (RB ? kall : y.T) & ~((Lam)1 << ha) : (Lam)0;
        const Lam hT = with_room(hTa, g, hcu);
        if (lane == src) {
            x = y;
            T_all = hTa;
            T = hT;
        }
        if (hT == 0) continue;
        const uint32_t Tlo = lo32(hT), Thi = hi32(hT);
        const int32_t hbw = y.b - hW;
        int32_t acc0 = 0, acc1 = 0;
        if (hW <= kHubMaxW) hub_planes<Lam, Rec, COH>(recs, inc, hjb, hje, hT, acc0, acc1);
        else for (int32_t j0 = hjb; j0 < hje; j0 += 32) {
            const int32_t j = j0 + lane;
            Lam lam = 0;
            int32_t w = 0;
            if (j < hje) {
                RecIO<Rec>::template load_b<COH>(recs + (load_inc<COH>(inc, j) & kNetMask), lam, w);
                w &= 0x7fffffff;
            }
            const int nn = min(32, hje - j0);
            const uint32_t llo = lo32(lam), lhi = hi32(lam);
            for (int q = 0; q < nn; ++q) {
                const uint32_t bl = __shfl_sync(kFull, llo, q);
                const int32_t wi = __shfl_sync(kFull, w, q);
                acc0 += ((bl >> lane) & 1) ? wi : 0;
                if (kWide) {
                    const uint32_t bh = __shfl_sync(kFull, lhi, q);
                    acc1 += ((bh >> lane) & 1) ? wi : 0;
                }
            }
        }
        // key = gain << 8 | (255 - block): the larger key is the higher gain, then the
        // smaller block (RB: the gain's sign bit flipped, so negative gains order too)
        unsigned long long key = 0;
        if ((Tlo >> lane) & 1) {
            const int32_t gg = hbw + acc0;
            if (RB ? (rb.phase == 2 || gg >= 0) : gg > 0)
                key = ((unsigned long long)((uint32_t)gg ^ (RB ? 0x80000000u : 0u)) << 8) | (unsigned long long)(255 - lane);
        }
        if (kWide && ((Thi >> lane) & 1)) {
            const int32_t gg = hbw + acc1;
            if (RB ? (rb.phase == 2 || gg >= 0) : gg > 0) {
                const unsigned long long k2 = ((unsigned long long)((uint32_t)gg ^ (RB ? 0x80000000u : 0u)) << 8) | (unsigned long long)(255 - (lane + 32));
                key = k2 > key ? k2 : key;
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long y2 = __shfl_xor_sync(kFull, key, o);
            key = y2 > key ? y2 : key;
        }
        if (lane == src && key) {
            t_best = 255 - (int)(key & 0xFF);
            g_best = (int32_t)((uint32_t)(key >> 8) ^ (RB ? 0x80000000u : 0u));
        }
        if (balance) {
            // zero-gain blocks of T among the ones this lane owns
            const unsigned zlo = __ballot_sync(kFull, ((Tlo >> lane) & 1) && hbw + acc0 == 0);
            const unsigned zhi = __ballot_sync(kFull, kWide && ((Thi >> lane) & 1) && hbw + acc1 == 0);
            if (lane == src) zero_in = kWide ? (Lam)((uint64_t)zlo | ((uint64_t)zhi << 32)) : (Lam)zlo;
        }
    }
    if (balance && valid && x.elig && t_best < 0) {
        // zero-gain moves that improve the balance (Sec. 6): blocks of T with gain 0, and
        // blocks outside T that lie in every net where u is not alone (their gain is
        // b - p_t = 0 exactly then); room and w(t) + c(u) < w(a); lightest block first
        Lam z = (zero_in | (x.A2 & ~T_all & ~((Lam)1 << a))) & kall;
        const long long wa = d.lmax - g.slack[a];
        long long best_w = 0;
        for (Lam y = z; y; y &= y - 1) {
            const int t = lam_bits_ctz(y);
            const long long wt = d.lmax - g.slack[t];
            if (g.slack[t] < cu || wt + cu >= wa) continue;
            if (t_best < 0 || wt < best_w) {
                t_best = t;
                best_w = wt;
            }
        }
        g_best = 0;
    }
    return valid && x.elig;
}

// Segments [seg, seg_end) of one tile's list of sub-round s (see k_gain); returns the number of
// candidates written, to the slots of segment seg.
// RB: a rebalancing pass (Sec. 8): only vertices of overloaded blocks take part, their target
// is the block with room of highest gain (any sign), and the candidate records its source
// block (bits 19..24) and the priority gain + off, by which it is counted.
template <typename Rec, bool RB>
__device__ __forceinline__ int32_t gain_seg(const Dev &d, int32_t tile, int32_t seg, int32_t seg_end, int32_t s,
                                            const GainWarp &g, uint16_t *picked,
                                            const GainInst &gi, int32_t &nel, const RbArgs &rb)
{
    const int lane = threadIdx.x & 31;
    const bool unit = d.nw == nullptr;
    const int32_t rbase = tile * kTile;
    nel = 0;
    if (s >= d.S) return 0;
    const uint16_t *ss = d.sub_start + (int64_t)tile * (d.S + 1);
    const int32_t beg = ss[s] + seg * kSeg, end = ss[s + 1];
    int32_t cnt = (seg_end == d.nseg ? end : min(end, (int32_t)ss[s] + seg_end * kSeg)) - beg;
    if (cnt <= 0) return 0;
    const uint16_t *list = d.sub_list + (int64_t)tile * kTile + beg;
    uint64_t *out = d.cand + (int64_t)tile * kTile + seg * kSeg;
    int32_t nout = 0;
    if (RB) {
        // the vertices of overloaded blocks, few of a list, moved together first so that the
        // lanes are full
        int32_t kept = 0;
        for (int32_t c0 = 0; c0 < cnt; c0 += 32) {
            const int32_t ul = c0 + lane < cnt ? list[c0 + lane] : 0;
            const bool over = c0 + lane < cnt && g.slack[d.part[rbase + ul]] < 0;
            const unsigned om = __ballot_sync(kFull, over);
            if (over) picked[kept + __popc(om & lanemask_lt())] = (uint16_t)ul;
            kept += __popc(om);
        }
        __syncwarp();
        list = picked;
        cnt = kept;
    }
    for (int32_t c0 = 0; c0 < cnt; c0 += 32) {
        const int32_t idx = c0 + lane;
        const bool valid = idx < cnt;
        int32_t ul = 0, cu = 1, jb = 0, je = 0, a = 0, W = 0;
        if (valid) {
            ul = list[idx];
            const int32_t u = rbase + ul;
            a = d.part[u];
            cu = d.vw ? d.vw[u] : 1;
            jb = d.vtx_off[u];
            je = d.vtx_off[u + 1];
            W = unit ? je - jb : d.vnw[u];
        }
        int t_best;
        int32_t g_best;
        const bool elig = gain_vertex<Rec, RB, false>(d, d.inc, g, gi, rb, valid, a, cu, jb, je, W, t_best, g_best);
        nel += __popc(__ballot_sync(kFull, elig));
        const unsigned cm = __ballot_sync(kFull, t_best >= 0);
        if (t_best >= 0) {
            const int pos = nout + __popc(cm & lanemask_lt());
            if (RB)
                out[pos] = ((uint64_t)(uint32_t)(g_best + rb.off) << 32) | ((uint32_t)a << 19) |
                           ((uint32_t)ul << 8) | (uint32_t)t_best;
            else
                out[pos] = ((uint64_t)(uint32_t)g_best << 32) | ((uint32_t)ul << 8) | (uint32_t)t_best;
        }
        count_gain(d, t_best >= 0, RB ? a : t_best, RB ? g_best + rb.off : g_best, cu);
        nout += __popc(cm);
        __syncwarp();
    }
    return nout;
}

__device__ __forceinline__ void room_tables(const Dev &d, const int64_t *bw, GainWarp &g)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const long long s0 = lane < d.k ? d.lmax - bw[lane] : -1, s1 = lane + 32 < d.k ? d.lmax - bw[lane + 32] : -1;
    g.slack[lane] = s0;
    g.slack[lane + 32] = s1;
    for (int c = 1; c <= kFeasW; ++c) {
        const unsigned lo = __ballot_sync(kFull, s0 >= c), hi = __ballot_sync(kFull, s1 >= c);
        if (lane == 0) g.feas[c] = (unsigned long long)lo | ((unsigned long long)hi << 32);
    }
    __syncwarp();
}

template <typename Rec>
__device__ __forceinline__ void gain_refresh(const Dev &d, GainWarp &g, GainInst &gi)
{
    room_tables(d, d.bw, g);
    gi.r = d.rs[0];
    gi.all_elig = d.rs[1] == 0;
}

// copies devs[inst] into a warp's shared slot
__device__ __forceinline__ void load_dev(Dev &dst, const Dev *src)
{
    const int lane = threadIdx.x & 31;
    const uint32_t *a = reinterpret_cast<const uint32_t *>(src);
    uint32_t *b = reinterpret_cast<uint32_t *>(&dst);
    for (int i = lane; i < (int)(sizeof(Dev) / 4); i += 32) b[i] = a[i];
    __syncwarp();
}

// Persistent: each warp walks work items, a segment of one tile's sub-round list each (a
// rebalancing item is RbArgs::segs segments, few of whose vertices take part), one vertex per lane
// (lane_best).  Only blocks in T can have a positive gain, since g_t <= omega({e : Phi(e,a) = 1,
// t in Lambda(e)}); the best of them has the largest g_t = b(u) - W + conn_t.  Vertices with more
// than kLaneDeg nets or W > kPlaneMaxW are walked by the whole warp.
// B = false: one instance, d0 (parameter space); B = true: a batch, items name (instance, tile)
// and each warp copies its item's instance into shared memory.  per_tile: items per tile (batches:
// the members' largest number of segments).  Work is handed out dynamically: a warp's first item is its index, the next
// ones come from a per-launch device counter, `take` of them at a time (so that a large
// instance's 10^5 items do not queue at one address), fetched while the items before are worked on.
template <typename Rec, bool B, bool RB = false>
__global__ void __launch_bounds__(kThreads, sizeof(Rec) == 16 || RB ? 4 : 3) k_gain(const Dev d0, const Dev *devs, const int2 *items,
                                                      int32_t n_items, int32_t per_tile, int32_t take, int32_t s,
                                                      int32_t rr, RbArgs rb = RbArgs{0, 0, 0, 1})
{
    after_previous();
    typedef typename RecIO<Rec>::Lam Lam;
    __shared__ GainWarp ws[kWarps];
    __shared__ uint16_t picked[RB ? kWarps : 1][RB ? kTile : 1];
    __shared__ Dev dsm[B ? kWarps : 1];
    __shared__ unsigned long long cnt_s[2];
    __shared__ int warps_done;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) { cnt_s[0] = 0; cnt_s[1] = 0; warps_done = 0; }
    __syncthreads();   // before any warp adds into them
    GainInst gi;
    int32_t nelig = 0, ncand = 0;
    int inst_prev = -1;
    const int32_t n_it = (B ? n_items : d0.n_tiles) * per_tile;
    const int32_t warps = gridDim.x * kWarps;
    int32_t *wq = d0.wq + (int64_t)rr * kWqPerRow + s;
    int32_t group = blockIdx.x * kWarps + wid;
    while ((int64_t)group * take < n_it) {
        // issued by lane 0 now, read (broadcast) when the items are done
        int32_t next = 0;
        if (lane == 0 && (int64_t)warps * take < n_it) next = atomicAdd(wq, 1);
        const int32_t it1 = min(n_it, (group + 1) * take);
        for (int32_t it = group * take; it < it1; ++it) {
            int32_t tile = it / per_tile;
            const int32_t seg = (it - tile * per_tile) * (RB ? rb.segs : 1);
            int32_t nel = 0;
            if (B) {
                const int2 im = items[tile];
                tile = im.y;
                if (im.x != inst_prev) {
                    __syncwarp();
                    load_dev(dsm[wid], devs + im.x);
                    gain_refresh<Rec>(dsm[wid], ws[wid], gi);
                    inst_prev = im.x;
                }
                const Dev &d = dsm[wid];
                if (seg >= d.nseg) continue;
                const int32_t nout = gain_seg<Rec, false>(d, tile, seg, seg + 1, s, ws[wid], nullptr, gi, nel, rb);
                if (lane == 0) {
                    d.cand_cnt[(int64_t)tile * d.nseg + seg] = nout;
                    unsigned long long *row = reinterpret_cast<unsigned long long *>(d.stats + (int64_t)rr * ST_N);
                    if (nel) atomicAdd(row + ST_ELIG, (unsigned long long)nel);
                    if (nout) atomicAdd(row + ST_CAND, (unsigned long long)nout);
                }
                __syncwarp();
            } else {
                if (inst_prev < 0) {
                    gain_refresh<Rec>(d0, ws[wid], gi);
                    if (RB) gi.r = rb.r;
                    inst_prev = 0;
                }
                const int32_t seg_end = RB ? min(d0.nseg, seg + rb.segs) : seg + 1;
                const int32_t nout = gain_seg<Rec, RB>(d0, tile, seg, seg_end, s, ws[wid], picked[RB ? wid : 0], gi, nel,
                                                       rb);
                int32_t *cnt = d0.cand_cnt + (int64_t)tile * d0.nseg + seg;
                if (RB) {
                    // the item's candidates lie together, filled segments first
                    const int32_t q = lane, left = max(0, nout - q * kSeg);
                    if (q < seg_end - seg) cnt[q] = seg + q == d0.nseg - 1 ? left : min(kSeg, left);
                } else if (lane == 0) {
                    *cnt = nout;
                }
                nelig += nel;
                ncand += nout;
            }
        }
        group = warps + __shfl_sync(kFull, next, 0);
        if ((int64_t)warps * take >= n_it) break;
    }
    if (!B) {
        // one instance: the warps' partial sums meet in shared memory and the last warp of the CTA
        // flushes them (no barrier, so warps that finish early do not wait for the slowest one)
        if (lane == 0) {
            if (nelig) atomicAdd(&cnt_s[0], (unsigned long long)nelig);
            if (ncand) atomicAdd(&cnt_s[1], (unsigned long long)ncand);
        }
        __threadfence_block();
        __syncwarp();
        int last = 0;
        if (lane == 0) last = atomicAdd(&warps_done, 1) == kWarps - 1;
        last = __shfl_sync(kFull, last, 0);
        if (last) {
            __threadfence_block();
            if (lane == 0) {
                unsigned long long *row = reinterpret_cast<unsigned long long *>(d0.stats + (int64_t)rr * ST_N);
                const unsigned long long c0 = atomicAdd(&cnt_s[0], 0ull), c1 = atomicAdd(&cnt_s[1], 0ull);
                if (c0) atomicAdd(row + ST_ELIG, c0);
                if (c1) atomicAdd(row + ST_CAND, c1);
            }
        }
    }
}

// ------------------------------------------------------------------ approval
__device__ __forceinline__ void decode(uint64_t c, int &t, int32_t &g, int &ul)
{
    t = (int)(c & 0xFF);
    ul = (int)((c >> 8) & (kTile - 1));
    g = (int32_t)(c >> 32);
}

// Which block an approval stage groups a candidate by, and which candidates take part:
//   KEY_T   LP: by target block, all candidates, inclusive prefix <= L_max - w(t);
//   KEY_A   rebalancing, source side: by source block (bits 19..24), all candidates, a
//           candidate passes while the weight before it is <= w(a) - L_max - 1 (exclusive);
//   KEY_TS  rebalancing, target side: by target block, only candidates marked by KEY_A
//           (bit 25), inclusive prefix <= L_max - w(t).
enum { KEY_T = 0, KEY_A = 1, KEY_TS = 2 };
constexpr uint64_t kSelBit = 1ull << 25;

template <int KEY>
__device__ __forceinline__ bool decode_key(uint64_t c, int &key, int &t, int32_t &g, int &ul)
{
    decode(c, t, g, ul);
    key = KEY == KEY_A ? (int)((c >> 19) & 0x3F) : t;
    return KEY != KEY_TS || (c & kSelBit) != 0;
}

// capacity of a key block for the stage (the weight its passing candidates may add up to)
template <int KEY>
__device__ __forceinline__ long long stage_cap(const Dev &d, int key)
{
    return KEY == KEY_A ? (long long)d.bw[key] - d.lmax - 1 : (long long)d.lmax - d.bw[key];
}

// digit of the overflow-bin refinement at `level` (1..3) for value v = g - (kBins - 1),
// and whether v matches the prefix resolved so far
__device__ __forceinline__ int refine_digit(int32_t v, int level, int64_t prefix, bool &match)
{
    if (level == 1) { match = true; return v >> 20; }
    if (level == 2) { match = (v >> 20) == prefix; return (v >> 10) & 1023; }
    match = (v >> 10) == prefix;
    return v & 1023;
}

// CTA per tile item: histogram of candidate weight by digit (level 1..3) for the key blocks whose
// threshold lies in the overflow bin
template <int KEY = KEY_T>
__global__ void __launch_bounds__(kThreads) k_hist(const Dev *devs, const int2 *items, int32_t n_items, int level)
{
    after_previous();
    __shared__ int active[64];
    __shared__ long long prefix[64];
    __shared__ SegRun run_w[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if ((int32_t)blockIdx.x >= item_count(devs, items, n_items, ITEM_TILE)) return;
    int32_t tile;
    const Dev &d = item_of(devs, items, blockIdx.x, tile);
    int a = 0;
    if (tid < d.k) {
        const Sel sl = d.sel[tid];
        a = sl.mode == SEL_REFINE && sl.level == level;
        prefix[tid] = sl.g;
    }
    if (tid < 64) active[tid] = a;
    if (!__syncthreads_or(a)) return;
    int32_t s0, s1;
    warp_segments(d, wid, s0, s1);
    if (s0 >= s1) return;
    SegRun &run = run_w[wid];
    const int32_t n = run.load(d, tile, s0, s1);
    for (int32_t i = lane; i < n; i += 32) {
        const int32_t slot = run.at(i);
        int t, ul, key;
        int32_t g;
        if (!decode_key<KEY>(d.cand[slot], key, t, g, ul) || !active[key]) continue;
        t = key;
        const unsigned long long c = d.vw ? (unsigned long long)d.vw[cand_vertex(slot, ul)] : 1ull;
        if (g < kBins - 1) continue;
        bool match;
        const int bin = refine_digit(g - (kBins - 1), level, prefix[t], match);
        if (!match) continue;
        atomicAdd(&d.hist[(int64_t)t * kBins + bin], c);
    }
}

// block-wide exclusive scan of 64-bit values (kThreads threads)
__device__ __forceinline__ unsigned long long block_scan_u64(unsigned long long v, unsigned long long *wt)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wt[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long t = lane < (int)(blockDim.x >> 5) ? wt[lane] : 0;
        unsigned long long s = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, s, o);
            if (lane >= o) s += y;
        }
        wt[lane] = s - t;
    }
    __syncthreads();
    const unsigned long long r = wt[wid] + x - v;
    __syncthreads();
    return r;
}

// one CTA per block item (instance, t): threshold of the (gain desc, id asc) prefix that fits
// (the level-0 histogram was filled by the gain step, or by k_rb_mark for the target side; bins: how
// many of its bins are in use, 0: Dev::bins)
template <int KEY = KEY_T>
__global__ void __launch_bounds__(kThreads) k_select(const Dev *devs, const int2 *items, int32_t n_items, int level,
                                                     int32_t bins)
{
    after_previous();
    __shared__ unsigned long long wt[32];
    __shared__ int found_bin;
    __shared__ long long found_before;
    __shared__ unsigned long long tot_s;
    const int tid = threadIdx.x;
    if ((int32_t)blockIdx.x >= item_count(devs, items, n_items, ITEM_BLOCK)) return;
    int32_t t;
    const Dev &d = item_of(devs, items, blockIdx.x, t);
    const Sel sl = d.sel[t];
    if (level > 0 && (sl.mode != SEL_REFINE || sl.level != level)) return;
    const int nbins = level == 0 ? (bins ? bins : d.bins) : (level == 1 ? 2048 : 1024);
    const long long cap = level == 0 ? stage_cap<KEY>(d, t) : (long long)sl.rem;
    unsigned long long *row = d.hist + (int64_t)t * kBins;
    // thread i owns bins [nbins - per*(i+1), nbins - per*i), visited from high to low
    const int per = nbins / kThreads;
    const int hi = nbins - per * tid;
    unsigned long long sum = 0;
    for (int b = hi - 1; b >= hi - per; --b) sum += row[b];
    if (tid == 0) { found_bin = -1; found_before = 0; }
    const unsigned long long before = block_scan_u64(sum, wt);
    if (level == 0) {
        if (tid == kThreads - 1) tot_s = before + sum;
        __syncthreads();
        const long long tot = (long long)tot_s;
        if (tot == 0 || tot <= cap) {   // every candidate passes
            if (sum)
                for (int b = hi - 1; b >= hi - per; --b) row[b] = 0;
            if (tid == 0) {
                Sel o;
                o.mode = SEL_ALL; o.level = 0; o.g = 0; o.rem = 0; o.cut = 0;
                d.sel[t] = o;
            }
            return;
        }
    }
    if ((long long)before <= cap && (long long)(before + sum) > cap) {
        unsigned long long c = before;
        for (int b = hi - 1; b >= hi - per; --b) {
            if ((long long)(c + row[b]) > cap) {
                found_bin = b;
                found_before = (long long)c;
                break;
            }
            c += row[b];
        }
    }
    __syncthreads();
    for (int b = tid; b < nbins; b += kThreads) row[b] = 0;
    if (tid == 0) {
        const int fb = found_bin;
        const long long rem = cap - found_before;
        Sel o;
        o.cut = 0;
        if (level == 0) {
            if (fb < kBins - 1) {
                o.mode = SEL_THRESH; o.level = 0; o.g = fb; o.rem = rem;
            } else {
                o.mode = SEL_REFINE; o.level = 1; o.g = 0; o.rem = rem;
            }
        } else {
            const long long p = level == 1 ? fb : (sl.g << 10) | fb;
            if (level == 3) {
                o.mode = SEL_THRESH; o.level = 0; o.g = (kBins - 1) + p; o.rem = rem;
            } else {
                o.mode = SEL_REFINE; o.level = level + 1; o.g = p; o.rem = rem;
            }
        }
        d.sel[t] = o;
    }
}

// Weight of the candidates at their block's threshold gain, per tile and block: CTAs walk the tile
// items with a grid stride and read an instance's thresholds once (a CTA per tile read them 24,400
// times on the power-law instance; approval 1.88 -> 1.44 ms per step).
template <int KEY = KEY_T>
__global__ void __launch_bounds__(kThreads) k_tie_sum(const Dev *devs, const int2 *items, int32_t n_items)
{
    after_previous();
    __shared__ int thr[64];
    __shared__ int32_t gthr[64];
    __shared__ unsigned long long ts[64];
    __shared__ SegRun run_w[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int32_t total = item_count(devs, items, n_items, ITEM_TILE);
    const Dev *prev = nullptr;
    bool any = false;
    for (int32_t item = blockIdx.x; item < total; item += gridDim.x) {
        int32_t tile;
        const Dev &d = item_of(devs, items, item, tile);
        if (&d != prev) {
            prev = &d;
            int a = 0;
            __syncthreads();
            if (tid < 64) {
                if (tid < d.k) {
                    const Sel sl = d.sel[tid];
                    a = sl.mode == SEL_THRESH;
                    gthr[tid] = (int32_t)sl.g;
                }
                thr[tid] = a;
                ts[tid] = 0;
            }
            any = __syncthreads_or(a) != 0;
        }
        if (!any) continue;
        int32_t s0, s1;
        warp_segments(d, wid, s0, s1);
        if (s0 < s1) {
            const int32_t n = run_w[wid].load(d, tile, s0, s1);
            for (int32_t i = lane; i < n; i += 32) {
                const int32_t slot = run_w[wid].at(i);
                int t, ul, key;
                int32_t g;
                if (decode_key<KEY>(d.cand[slot], key, t, g, ul) && thr[key] && g == gthr[key])
                    atomicAdd(&ts[key], d.vw ? (unsigned long long)d.vw[cand_vertex(slot, ul)] : 1ull);
            }
        }
        __syncthreads();
        if (tid < 64) {
            if (thr[tid]) d.tie[(int64_t)tid * d.n_tiles + tile] = (int64_t)ts[tid];
            ts[tid] = 0;
        }
        __syncthreads();
    }
}

// one CTA per block item with a threshold gain: the vertex id up to which the candidates at that
// gain pass.  Their inclusive (KEY_A: exclusive) weight prefix in id order only grows, so the
// passing ones are those up to one id: the tile where the prefix crosses the budget is found from
// the tile sums (tiles are in id order), the id inside it from the tile's candidates.  The apply
// step then only compares ids; rebuilding the prefix of every 256 vertices that held a tie there
// (the earlier ones of the tile read again, one candidate at a time) took 2.0 ms of the power-law
// instance's 67.3 ms (50 M vertices, k = 64, 5 rounds) and 0.06 of the row-net one's 6.56 ms.
template <int KEY = KEY_T>
__global__ void __launch_bounds__(1024) k_tie_cut(const Dev *devs, const int2 *items, int32_t n_items)
{
    after_previous();
    __shared__ unsigned long long wt[32];
    __shared__ unsigned long long carry_s, cross_before;
    __shared__ int32_t cross_tile;
    __shared__ int32_t cut_s;
    if ((int32_t)blockIdx.x >= item_count(devs, items, n_items, ITEM_BLOCK)) return;
    int32_t t;
    const Dev &d = item_of(devs, items, blockIdx.x, t);
    const Sel sl = d.sel[t];
    if (sl.mode != SEL_THRESH) return;
    const int tid = threadIdx.x;
    const unsigned long long rem = (unsigned long long)sl.rem;
    const int64_t *row = d.tie + (int64_t)t * d.n_tiles;
    if (tid == 0) {
        carry_s = 0;
        cross_tile = -1;
    }
    __syncthreads();
    constexpr int kPer = 8;   // consecutive tiles per thread
    for (int32_t b = 0; b < d.n_tiles; b += (int32_t)blockDim.x * kPer) {
        unsigned long long part[kPer], v = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int32_t i = b + tid * kPer + q;
            part[q] = i < d.n_tiles ? (unsigned long long)row[i] : 0;
            v += part[q];
        }
        const unsigned long long ex = carry_s + block_scan_u64(v, wt);
        // the tile of the candidate that first exceeds the budget: all of the earlier tiles'
        // candidates pass, none of the later tiles' (under either rule)
        if (ex <= rem && ex + v > rem) {
            unsigned long long before = ex;
            int q = 0;
            while (before + part[q] <= rem) before += part[q++];   // ends: the sum exceeds rem
            cross_tile = b + tid * kPer + q;
            cross_before = before;
        }
        __syncthreads();
        if (cross_tile >= 0) break;
        if (tid == (int)blockDim.x - 1) carry_s = ex + v;
        __syncthreads();
    }
    const int32_t tile = cross_tile;
    if (tile < 0) {   // everything fits
        if (tid == 0) d.sel[t].cut = 0x7fffffff;
        return;
    }
    // the crossing tile's candidates in id order, kTile slots
    if (tid == 0) {
        cut_s = tile * kTile - 1;
        carry_s = cross_before;
    }
    __syncthreads();
    for (int b = 0; b < kTile; b += (int)blockDim.x) {
        const int slot = b + tid;
        const int32_t seg = min(slot / kSeg, d.nseg - 1);
        unsigned long long v = 0;
        int32_t u = -1;
        if (slot - seg * kSeg < d.cand_cnt[(int64_t)tile * d.nseg + seg]) {
            int key, tt, ul;
            int32_t g;
            if (decode_key<KEY>(d.cand[(int64_t)tile * kTile + slot], key, tt, g, ul) && key == t && g == (int32_t)sl.g) {
                u = tile * kTile + ul;
                v = d.vw ? (unsigned long long)d.vw[u] : 1ull;
            }
        }
        const unsigned long long ex = carry_s + block_scan_u64(v, wt);
        if (u >= 0 && (KEY == KEY_A ? ex : ex + v) <= rem) atomicMax(&cut_s, u);
        __syncthreads();
        if (tid == (int)blockDim.x - 1) carry_s = ex + v;
        __syncthreads();
    }
    if (tid == 0) d.sel[t].cut = cut_s;
}

// ------------------------------------------------------------------ apply
constexpr uint8_t kRvNone = 0xFF, kRvBack = 0x80;   // revert variant: per candidate slot marks

struct alignas(16) ApplyWarp {
    int32_t off[33];
    int32_t jb[32];
    int32_t a[32];
    int32_t t[32];
};

// Approved moves of a warp that wait until 32 of them fill its lanes.
constexpr int kDecide = 4;            // candidates a lane decides at a time
constexpr int kQueue = 32 * (kDecide + 1);
struct alignas(16) MoveQueue {
    int32_t u[kQueue];
    uint16_t at[kQueue];    // source block | target block << 8
};

// Applies up to kPins moved pins per lane (vertex moved a -> t, incident net e): Phi(e,a)--,
// Phi(e,t)++, and from the old values the Lambda / S1 bit flips and the objective change
// (Sec. 2: a pin count that steps 1 -> 0 removes the block from Lambda(e), 0 -> 1 adds it,
// each changing (lambda-1) by one; a step into or out of the value 1 flips the S1 bit), then
// stamps e as moved in round r.  Every load and atomic of the kPins pins is issued before any
// result is used, so their latencies overlap.
constexpr int kPins = 4;

// Lambda and S1 of a tiny net (Dev::tiny) after one pin went a -> t, by compare-and-swap (at most
// three other movers can come between); whether a left Lambda and whether t entered it.
__device__ __forceinline__ void tiny_step(uint64_t &s1, uint64_t &lam, int a, int t, int size, bool &left, bool &entered)
{
    const int ca = tiny_count<uint64_t>(s1, lam, size, a), ct = tiny_count<uint64_t>(s1, lam, size, t);
    const uint64_t ba = 1ull << a, bt = 1ull << t;
    left = ca == 1;
    entered = ct == 0;
    lam = (lam & ~(left ? ba : 0ull)) | bt;
    s1 = (s1 & ~(ba | bt)) | (ca == 2 ? ba : 0ull) | (entered ? bt : 0ull);
}

__device__ __forceinline__ void tiny_move(Rec16 *rc, int a, int t, int size, bool &left, bool &entered)
{
    unsigned long long *p = reinterpret_cast<unsigned long long *>(rc);   // s1 | lam << 32
    unsigned long long cur = __ldcg(p);
    while (true) {
        uint64_t s1 = (uint32_t)cur, lam = cur >> 32;
        tiny_step(s1, lam, a, t, size, left, entered);
        const unsigned long long old = atomicCAS(p, cur, s1 | (lam << 32));
        if (old == cur) return;
        cur = old;
    }
}

__device__ __forceinline__ void tiny_move(Rec32 *rc, int a, int t, int size, bool &left, bool &entered)
{
    ulonglong2 cur = __ldcg(reinterpret_cast<const ulonglong2 *>(rc));
    while (true) {
        uint64_t s1 = cur.x, lam = cur.y;
        tiny_step(s1, lam, a, t, size, left, entered);
        ulonglong2 old;
        asm volatile(
            "{\n\t.reg .b128 c, n, o;\n\t"
            "mov.b128 c, {%2, %3};\n\t"
            "mov.b128 n, {%4, %5};\n\t"
            "atom.relaxed.gpu.global.cas.b128 o, [%6], c, n;\n\t"
            "mov.b128 {%0, %1}, o;\n\t}"
            : "=l"(old.x), "=l"(old.y)
            : "l"(cur.x), "l"(cur.y), "l"(s1), "l"(lam), "l"(rc)
            : "memory");
        if (old.x == cur.x && old.y == cur.y) return;
        cur = old;
    }
}

// RVC (LP apply with the revert variant on): also counts the movers of every net (d.rv_net)
// and, in `shared`, the moved incidences on nets with several movers (a second mover adds its
// own incidence and the first one's, later movers their own).
template <typename Rec, bool STAMP = true, bool RVC = false>
__device__ __forceinline__ long long apply_pins(const Dev &d, const int32_t *inc, Rec *recs, const ApplyWarp &w_,
                                                int32_t i0, int32_t total, int32_t r, int32_t *shared = nullptr)
{
    typedef typename RecIO<Rec>::Lam Lam;
    int32_t e[kPins], a[kPins], t[kPins], oa[kPins], ot[kPins], w[kPins], mv[kPins];
    bool ok[kPins];
#pragma unroll
    for (int q = 0; q < kPins; ++q) {
        const int32_t i = i0 + q * 32;
        ok[q] = i < total;
        e[q] = 0; a[q] = 0; t[q] = 0;
        if (ok[q]) {
            const int v = slot_of(w_.off, i);
            a[q] = w_.a[v];
            t[q] = w_.t[v];
            e[q] = inc[w_.jb[v] + (i - w_.off[v])];
        }
    }
#pragma unroll
    for (int q = 0; q < kPins; ++q) {
        if (!ok[q]) continue;
        const bool wide = e[q] < 0;
        const int32_t ee = e[q] & kNetMask;
        const int32_t wrow = wide ? d.widx[ee] : 0;
        Rec *rc = recs + ee;
        const int2 wm = __ldcg(reinterpret_cast<const int2 *>(&rc->w));   // omega and stamp
        mv[q] = STAMP ? wm.y : 0;
        w[q] = wm.x & 0x7fffffff;
        if (ee < d.tiny[0]) phi_move(d, ee, a[q], t[q], wide, wrow, oa[q], ot[q]);
        if (RVC && d.rv_net) {
            const int32_t before = atomicAdd(&d.rv_net[ee], 1);
            *shared += before == 1 ? 2 : (before >= 2 ? 1 : 0);
        }
    }
    long long dobj = 0;
#pragma unroll
    for (int q = 0; q < kPins; ++q) {
        if (!ok[q]) continue;
        Rec *rc = recs + (e[q] & kNetMask);
        const int32_t ee = e[q] & kNetMask;
        bool left, entered;
        if (ee >= d.tiny[0]) {
            tiny_move(rc, a[q], t[q], tiny_size(d, ee), left, entered);
        } else {
            const Lam ba = (Lam)1 << a[q], bt = (Lam)1 << t[q];
            left = oa[q] == 1;
            entered = ot[q] == 0;
            const Lam lx = (left ? ba : (Lam)0) | (entered ? bt : (Lam)0);
            const Lam sx = ((oa[q] == 1 || oa[q] == 2) ? ba : (Lam)0) | ((ot[q] == 0 || ot[q] == 1) ? bt : (Lam)0);
            if (sizeof(Lam) == 8) {
                if (lx) atomicXor(reinterpret_cast<unsigned long long *>(&rc->lam), (unsigned long long)lx);
                if (sx) atomicXor(reinterpret_cast<unsigned long long *>(&rc->s1), (unsigned long long)sx);
            } else if (sx) {   // a Lambda flip is an S1 flip, too
                atomicXor(reinterpret_cast<unsigned long long *>(rc), (unsigned long long)sx | ((unsigned long long)lx << 32));
            }
        }
        // stamp: every writer of round r derives the same, larger value from the pre-round stamp, so
        // the order does not matter.  A reduction, not a store: in a round's first sub-round all
        // pins of a large net find it unstamped at once, and stores to one address queue up (power-law
        // 3M, k = 32: 519 us in a round's first sub-round, 127 in the others; now 135)
        if (STAMP) {
            const int32_t last = mv[q] >> 1;
            if (last != r) atomicMax(&rc->mv, (r << 1) | (last == r - 1 ? 1 : 0));
        }
        dobj += (long long)(entered ? w[q] : 0) - (long long)(left ? w[q] : 0);
    }
    return dobj;
}

// Per-warp approval state of one instance.
struct ApplyInst {
    int32_t gthr[64];    // a candidate of the block passes above this gain,
    int32_t cut[64];     // or at it up to this vertex id
};

__device__ __forceinline__ void apply_refresh(const Dev &d, ApplyInst &ai, int32_t &r)
{
    const int lane = threadIdx.x & 31;
    for (int t = lane; t < 64; t += 32) {
        int32_t g = -1, cut = -1;   // every candidate passes (gains and priorities are >= 0)
        if (t < d.k) {
            const Sel sl = d.sel[t];
            if (sl.mode == SEL_THRESH) {
                g = (int32_t)sl.g;
                cut = (int32_t)sl.cut;
            }
        }
        ai.gthr[t] = g;
        ai.cut[t] = cut;
    }
    r = d.rs[0];
    __syncwarp();
}

// Approval of candidate i of a run: above its key block's threshold gain, or at it up to the
// block's last id.
template <int KEY>
__device__ __forceinline__ bool approve(uint64_t c, int32_t slot, const ApplyInst &ai, int &t, int32_t &u)
{
    int key, ul;
    int32_t g;
    if (!decode_key<KEY>(c, key, t, g, ul)) return false;
    u = cand_vertex(slot, ul);
    return g > ai.gthr[key] || (g == ai.gthr[key] && u <= ai.cut[key]);
}

// Applies the queued moves [first, first + 32) (at most `queued` in all) over their incidences,
// flattened across the lanes.
template <typename Rec, int KEY>
__device__ __forceinline__ void apply_queue(const Dev &d, const int32_t *vtx_off, const int32_t *inc, const int32_t *qu, const uint16_t *qat, int32_t first,
                                            int32_t queued, int32_t r, ApplyWarp &w_,
                                            long long &dobj, int32_t &npins, int32_t &nshared)
{
    const int lane = threadIdx.x & 31;
    Rec *recs = reinterpret_cast<Rec *>(d.rec);
    int32_t deg = 0, jb = 0, a = 0, t = 0;
    if (first + lane < queued) {
        const int32_t u = qu[first + lane], at = qat[first + lane];
        a = at & 0xFF;
        t = at >> 8;
        jb = vtx_off[u];
        deg = vtx_off[u + 1] - jb;
        npins += deg;
    }
    int32_t incl = deg;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int32_t total = __shfl_sync(kFull, incl, 31);
    w_.off[lane] = incl - deg;
    w_.jb[lane] = jb;
    w_.a[lane] = a;
    w_.t[lane] = t;
    if (lane == 31) w_.off[32] = total;
    __syncwarp();
    for (int32_t i0 = 0; i0 < total; i0 += 32 * kPins)
        dobj += apply_pins<Rec, KEY == KEY_T, KEY == KEY_T>(d, inc, recs, w_, i0 + lane, total, r, &nshared);
    __syncwarp();
}

// Segments [s0, s1) of one tile in the apply step (see k_apply).  KEY_T: LP (stamps the nets,
// records the revert variant's source blocks); KEY_TS: rebalancing (no stamps).
template <typename Rec, int KEY>
__device__ __forceinline__ void apply_segs(const Dev &d, int32_t tile, int32_t s0, int32_t s1, int32_t r,
                                           const ApplyInst &ai, unsigned long long *bwd, SegRun &run, ApplyWarp &w_,
                                           MoveQueue &mq, int32_t &queued, long long &dobj, int32_t &nappr,
                                           int32_t &npins, int32_t &nshared)
{
    const int lane = threadIdx.x & 31;
    const int32_t ncand = run.load(d, tile, s0, s1);
    for (int32_t c0 = 0; c0 < ncand; c0 += 32 * kDecide) {
        // kDecide candidates per lane, their loads in flight together
        int32_t slot[kDecide], u[kDecide];
        int t[kDecide], a[kDecide];
        uint64_t c[kDecide];
        bool appr[kDecide];
#pragma unroll
        for (int q = 0; q < kDecide; ++q) {
            const int32_t i = c0 + q * 32 + lane;
            slot[q] = i < ncand ? run.at(i) : -1;
            c[q] = slot[q] >= 0 ? d.cand[slot[q]] : 0;
        }
#pragma unroll
        for (int q = 0; q < kDecide; ++q) {
            t[q] = 0; a[q] = 0; u[q] = 0;
            appr[q] = slot[q] >= 0 && approve<KEY>(c[q], slot[q], ai, t[q], u[q]);
            if (appr[q]) a[q] = d.part[u[q]];
        }
#pragma unroll
        for (int q = 0; q < kDecide; ++q) {
            if (KEY == KEY_T && d.rv_src && slot[q] >= 0) d.rv_src[slot[q]] = appr[q] ? (uint8_t)a[q] : kRvNone;
            const unsigned am = __ballot_sync(kFull, appr[q]);
            if (am == 0) continue;
            if (appr[q]) {
                const unsigned long long cw = d.vw ? (unsigned long long)d.vw[u[q]] : 1ull;
                d.part[u[q]] = (uint8_t)t[q];
                if (!d.vw) {
                    // unit weights: one update per distinct block
                    const unsigned pa = __match_any_sync(am, a[q]), pt = __match_any_sync(am, t[q]);
                    if (lane == __ffs(pa) - 1) atomicAdd(&bwd[a[q]], (unsigned long long)(-(long long)__popc(pa)));
                    if (lane == __ffs(pt) - 1) atomicAdd(&bwd[t[q]], (unsigned long long)__popc(pt));
                } else {
                    atomicAdd(&bwd[a[q]], (unsigned long long)(-(long long)cw));
                    atomicAdd(&bwd[t[q]], cw);
                }
                ++nappr;
                const int pos = queued + __popc(am & lanemask_lt());
                mq.u[pos] = u[q];
                mq.at[pos] = (uint16_t)(a[q] | (t[q] << 8));
            }
            queued += __popc(am);
        }
        __syncwarp();
        int32_t first = 0;
        for (; queued - first >= 32; first += 32)
            apply_queue<Rec, KEY>(d, d.vtx_off, d.inc, mq.u, mq.at, first, queued, r, w_, dobj, npins, nshared);
        if (first && queued - first > 0) {   // the rest moves to the front
            int32_t u2 = 0;
            uint16_t at2 = 0;
            if (first + lane < queued) {
                u2 = mq.u[first + lane];
                at2 = mq.at[first + lane];
            }
            __syncwarp();
            mq.u[lane] = u2;
            mq.at[lane] = at2;
        }
        queued -= first;
        __syncwarp();
    }
}

// Persistent: each warp walks work items with a grid stride, `per` consecutive segments of a tile
// each.  For each 32 candidates it decides approval (threshold gain and last tied id of the target
// block, see k_tie_cut) and queues the approved ones; whenever 32 are queued, from whichever items,
// it applies them over their incidences flattened across the lanes, so all atomics are in flight
// at once.  (In a saturated sub-round a fifth of the candidates is approved: without the queue a
// chunk had 6 moves and 40 of the 128 pins it can have in flight.  Row-net 2M 35 -> 32 us per
// launch, power-law 50M 1.05 -> 0.98 ms, and 26 us and 0.73 ms since tiny nets, phi_move and stamps
// by reductions; the queue with one candidate decided per lane at a time, a chain of loads for every
// 32, was slower than no queue, 42 us and 1.19 ms.)
// B as for k_gain.
template <typename Rec, bool B, int KEY = KEY_T>
__global__ void __launch_bounds__(kThreads, B ? 3 : 4) k_apply(const Dev d0, const Dev *devs, const int2 *items,
                                                       int32_t n_items, int32_t nseg, int32_t per, int32_t rr)
{
    after_previous();
    __shared__ ApplyInst ai_w[kWarps];
    __shared__ SegRun run_w[kWarps];
    __shared__ MoveQueue mq_w[kWarps];
    __shared__ unsigned long long bwd_w[kWarps][64];
    __shared__ ApplyWarp aw[kWarps];
    __shared__ Dev dsm[B ? kWarps : 1];
    __shared__ unsigned long long objd, napp, mpins;
    __shared__ int warps_done;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    bwd_w[wid][lane] = 0;
    bwd_w[wid][lane + 32] = 0;
    if (tid == 0) { objd = 0; napp = 0; mpins = 0; warps_done = 0; }
    __syncthreads();   // before any warp can add into another warp's slots (at its end)
    long long dobj = 0;
    int32_t nappr = 0, npins = 0, r = 0, nshared = 0, queued = 0;
    int inst_prev = -1;
    const int32_t groups = (nseg + per - 1) / per;
    const int32_t n_it = (B ? n_items : d0.n_tiles) * groups;
    // a batch instance's queue, block weights and counters, before the warp turns to another one
    auto leave = [&](const Dev &d) {
        if (queued) apply_queue<Rec, KEY>(d, d.vtx_off, d.inc, mq_w[wid].u, mq_w[wid].at, 0, queued, r, aw[wid], dobj, npins, nshared);
        queued = 0;
        for (int o = 16; o; o >>= 1) {
            dobj += __shfl_xor_sync(kFull, dobj, o);
            nappr += __shfl_xor_sync(kFull, nappr, o);
            npins += __shfl_xor_sync(kFull, npins, o);
        }
        __syncwarp();
        for (int t = lane; t < 64; t += 32) {
            const unsigned long long v = bwd_w[wid][t];
            if (v) {
                atomicAdd(reinterpret_cast<unsigned long long *>(&d.bw[t]), v);
                bwd_w[wid][t] = 0;
            }
        }
        if (lane == 0) {
            unsigned long long *row = reinterpret_cast<unsigned long long *>(d.stats + (int64_t)rr * ST_N);
            if (dobj) atomicAdd(reinterpret_cast<unsigned long long *>(d.obj), (unsigned long long)dobj);
            if (nappr) atomicAdd(row + ST_APPR, (unsigned long long)nappr);
            if (npins) atomicAdd(row + ST_MOVED, (unsigned long long)npins);
        }
        dobj = 0;
        nappr = 0;
        npins = 0;
        __syncwarp();
    };
    // static assignment (measured faster here than the gain step's dynamic distribution)
    for (int32_t item = blockIdx.x * kWarps + wid; item < n_it; item += gridDim.x * kWarps) {
        int32_t tile = item / groups;
        const int32_t s0 = (item - tile * groups) * per;
        if (B) {
            const int2 it = items[tile];
            tile = it.y;
            if (it.x != inst_prev) {
                if (inst_prev >= 0) leave(dsm[wid]);
                load_dev(dsm[wid], devs + it.x);
                apply_refresh(dsm[wid], ai_w[wid], r);
                inst_prev = it.x;
            }
            const Dev &d = dsm[wid];
            if (s0 >= d.nseg) continue;
            apply_segs<Rec, KEY>(d, tile, s0, min(d.nseg, s0 + per), r, ai_w[wid], bwd_w[wid], run_w[wid], aw[wid],
                                 mq_w[wid], queued, dobj, nappr, npins, nshared);
        } else {
            if (inst_prev < 0) {
                apply_refresh(d0, ai_w[wid], r);
                inst_prev = 0;
            }
            apply_segs<Rec, KEY>(d0, tile, s0, min(d0.nseg, s0 + per), r, ai_w[wid], bwd_w[wid], run_w[wid], aw[wid],
                                 mq_w[wid], queued, dobj, nappr, npins, nshared);
        }
    }
    if (B) {
        if (inst_prev >= 0) leave(dsm[wid]);
        return;
    }
    if (queued) apply_queue<Rec, KEY>(d0, d0.vtx_off, d0.inc, mq_w[wid].u, mq_w[wid].at, 0, queued, r, aw[wid], dobj, npins, nshared);
    if (!B && KEY == KEY_T && d0.rv_cnt) {
        // revert variant: moved incidences on nets with several movers (sizes the order-statistics table)
        nshared = __reduce_add_sync(kFull, nshared);
        if (lane == 0 && nshared) atomicAdd(d0.rv_cnt + 1, (unsigned long long)nshared);
    }
    if (!B) {
        // as in k_gain: partial sums into warp 0's slots, the last warp to finish flushes
        for (int o = 16; o; o >>= 1) {
            dobj += __shfl_xor_sync(kFull, dobj, o);
            nappr += __shfl_xor_sync(kFull, nappr, o);
            npins += __shfl_xor_sync(kFull, npins, o);
        }
        if (wid != 0) {
            for (int t = lane; t < 64; t += 32)
                if (bwd_w[wid][t]) atomicAdd(&bwd_w[0][t], bwd_w[wid][t]);
        }
        if (lane == 0) {
            if (dobj) atomicAdd(&objd, (unsigned long long)dobj);
            if (nappr) atomicAdd(&napp, (unsigned long long)nappr);
            if (npins) atomicAdd(&mpins, (unsigned long long)npins);
        }
        __threadfence_block();
        __syncwarp();
        int last = 0;
        if (lane == 0) last = atomicAdd(&warps_done, 1) == kWarps - 1;
        last = __shfl_sync(kFull, last, 0);
        if (last) {
            __threadfence_block();
            for (int t = lane; t < 64 && t < d0.k; t += 32) {
                const unsigned long long v = atomicAdd(&bwd_w[0][t], 0ull);
                if (v) atomicAdd(reinterpret_cast<unsigned long long *>(&d0.bw[t]), v);
            }
            if (lane == 0) {
                unsigned long long *row = reinterpret_cast<unsigned long long *>(d0.stats + (int64_t)rr * ST_N);
                const unsigned long long o1 = atomicAdd(&objd, 0ull), a1 = atomicAdd(&napp, 0ull),
                                         p1 = atomicAdd(&mpins, 0ull);
                if (o1) atomicAdd(reinterpret_cast<unsigned long long *>(d0.obj), o1);
                if (a1) atomicAdd(row + ST_APPR, a1);
                if (p1) atomicAdd(row + ST_MOVED, p1);
                if (KEY == KEY_T && p1 && d0.rv_cnt) atomicAdd(d0.rv_cnt, p1);
            }
        }
    }
}

#include "hgp_small.cuh"

// ------------------------------------------------------------------ revert variant
// Attributed gains (Sec. 5.2) of a sub-round's approved moves, with every net seeing its moves
// in ascending vertex id: the gain of u (a -> b) if the moves of smaller ids had been made
// first.  Lemma 1 (Sec. 5.4) gives it from order statistics of the moves that touch (e, i),
// with the vertex id as the position in the sequence:
//     +omega(e)  iff  Psi(e, a) = 0, u = max out(e, a), min in(e, a) > u
//     -omega(e)  iff  Psi(e, b) = 0, u = min in(e, b),  max out(e, b) < u
// where Psi(e, i) is the number of pins of e that were in block i at the start of the sub-round
// and stayed: Phi(e, i) after the moves minus |in(e, i)|.  Most touched nets have one mover in
// a sub-round; for them the two conditions reduce to Phi(e, a) = 0 and Phi(e, b) = 1 after the
// move.  The apply step counts the movers of every net and the moved incidences of nets with
// several movers; INSERT records max out, min in and |in| of those nets' (e, i) in an
// open-addressing table sized to that count, EVAL sums the terms per move and marks the moves
// whose sum is negative, and the revert step moves those back (Sec. 6).  Balance holds after it: each
// block's approval was checked against its weight at the start of the sub-round, without credit for
// departures.
struct alignas(16) RvSlot {
    unsigned long long key;   // e * 64 + i, kRvEmpty when free
    int32_t max_out;          // largest id of a mover that left block i (a pin of e), -1 if none
    int32_t min_in;           // smallest id of a mover that entered block i, INT32_MAX if none
    int32_t n_in;             // number of movers that entered block i
    int32_t pad[3];
};
static_assert(sizeof(RvSlot) == kRvSlotBytes, "revert table slot size");
constexpr unsigned long long kRvEmpty = ~0ull;

// slots in use this sub-round: a power of two >= 4 x moved incidences of shared nets (>= 2 x
// keys), at most the capacity (>= 2 P >= keys, so a free slot always exists)
__device__ __forceinline__ uint64_t rv_slots(const Dev &d)
{
    const uint64_t need = 4ull * __ldcg(d.rv_cnt + 1);
    uint64_t c = 1024;
    while (c < need && c < (uint64_t)d.rv_cap) c <<= 1;
    return c;
}

// find (or insert) key by linear probing from p, whose key is cur; at most `mask + 1` probes.  Keys are
// read through L1: one that is there stays, and a free slot read too late is settled by the
// compare-and-swap (the slots of a large net are read by all its movers).
__device__ __forceinline__ RvSlot *rv_find(RvSlot *tab, uint64_t mask, uint64_t p, unsigned long long cur,
                                           unsigned long long key, bool insert)
{
    for (uint64_t probe = 0; probe <= mask; ++probe) {
        RvSlot *sl = tab + p;
        if (cur == key) return sl;
        if (cur == kRvEmpty) {
            if (!insert) return nullptr;
            cur = atomicCAS(&sl->key, kRvEmpty, key);
            if (cur == kRvEmpty || cur == key) return sl;
        }
        p = (p + 1) & mask;
        cur = tab[p].key;
    }
    return nullptr;
}

// the slots of (e, a) and (e, b); the first probes of both are in flight together
__device__ __forceinline__ void rv_find_both(RvSlot *tab, uint64_t mask, int32_t e, int a, int b, bool insert,
                                             RvSlot *&sa, RvSlot *&sb)
{
    const unsigned long long ka = (unsigned long long)e * 64 + a, kb = (unsigned long long)e * 64 + b;
    const uint64_t pa = splitmix64_output(ka) & mask, pb = splitmix64_output(kb) & mask;
    const unsigned long long ca = tab[pa].key, cb = tab[pb].key;
    sa = rv_find(tab, mask, pa, ca, ka, insert);
    sb = rv_find(tab, mask, pb, cb, kb, insert);
}

// half a slot per thread, so that a warp's store is one run and not every second 16 bytes of two.  With
// this and the two changes above the revert launches of 5 rounds take 2.33 instead of 2.59 ms (power-law
// 3M, k = 32), 27.8 instead of 30.5 (50M, k = 64).
__global__ void k_rv_clear(const Dev d)
{
    after_previous();
    const uint64_t n = 2 * rv_slots(d);
    int4 *tab = reinterpret_cast<int4 *>(d.rv_tab);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        tab[i] = i & 1 ? make_int4(0, 0, 0, 0) : make_int4(-1, -1, -1, 0x7fffffff);   // n_in; key, max_out, min_in
}

struct alignas(16) RvWarp {
    ApplyWarp w;
    int32_t u[32];
    int32_t g[32];
};

enum { RV_INSERT = 0, RV_EVAL = 1 };

// CTA per tile, a run of its segments per warp: the approved movers of each 32 candidates, their
// incidences flattened over the lanes, one of the passes above per launch.
template <typename Rec, int PASS>
__global__ void __launch_bounds__(kThreads) k_rv_pass(const Dev d)
{
    after_previous();
    __shared__ RvWarp rw_[kWarps];
    __shared__ SegRun run_w[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t s0, s1;
    warp_segments(d, wid, s0, s1);
    if (s0 >= s1) return;
    SegRun &run = run_w[wid];
    const int32_t ncand = run.load(d, blockIdx.x, s0, s1);
    if (ncand == 0) return;
    RvWarp &rw = rw_[wid];
    const uint64_t mask = (PASS == RV_INSERT || PASS == RV_EVAL) ? rv_slots(d) - 1 : 0;
    RvSlot *tab = reinterpret_cast<RvSlot *>(d.rv_tab);
    const Rec *recs = reinterpret_cast<const Rec *>(d.rec);
    uint8_t *src = d.rv_src;
    bool lost = false;
    for (int32_t c0 = 0; c0 < ncand; c0 += 32) {
        const int32_t idx = c0 + lane < ncand ? run.at(c0 + lane) : 0;
        int32_t deg = 0, jb = 0, u = 0;
        int t = 0, a = 0;
        const uint8_t sa = c0 + lane < ncand ? src[idx] : kRvNone;
        if (sa != kRvNone) {
            int ul;
            int32_t g;
            decode(d.cand[idx], t, g, ul);
            u = cand_vertex(idx, ul);
            a = sa;
            jb = d.vtx_off[u];
            deg = d.vtx_off[u + 1] - jb;
        }
        int32_t incl = deg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int32_t total = __shfl_sync(kFull, incl, 31);
        rw.w.off[lane] = incl - deg;
        rw.w.jb[lane] = jb;
        rw.w.a[lane] = a;
        rw.w.t[lane] = t;
        rw.u[lane] = u;
        rw.g[lane] = 0;
        if (lane == 31) rw.w.off[32] = total;
        __syncwarp();
        for (int32_t i = lane; i < total; i += 32) {
            const int v = slot_of(rw.w.off, i);
            const int32_t e = d.inc[rw.w.jb[v] + (i - rw.w.off[v])];
            const int32_t ee = e & kNetMask;
            const int32_t movers = __ldcg(&d.rv_net[ee]);
            const int32_t av = rw.w.a[v], bv = rw.w.t[v], uv = rw.u[v];
            if (PASS == RV_INSERT) {
                if (movers < 2) continue;
                RvSlot *s_a, *s_b;
                rv_find_both(tab, mask, ee, av, bv, true, s_a, s_b);
                if (!s_a || !s_b) {
                    lost = true;
                    continue;
                }
                atomicMax(&s_a->max_out, uv);
                atomicMin(&s_b->min_in, uv);
                atomicAdd(&s_b->n_in, 1);
            } else {
                const bool wide = e < 0;
                const int32_t wrow = wide ? d.widx[ee] : 0;
                const int32_t pa = phi_get(d, ee, av, wide, wrow), pb = phi_get(d, ee, bv, wide, wrow);
                const int32_t w = __ldg(&recs[ee].w) & 0x7fffffff;
                int32_t g = 0;
                if (movers < 2) {
                    // the only mover of e: Phi(e, a) went 1 -> 0, or Phi(e, b) went 0 -> 1
                    if (pa == 0) g += w;
                    if (pb == 1) g -= w;
                } else {
                    RvSlot *s_a, *s_b;
                    rv_find_both(tab, mask, ee, av, bv, false, s_a, s_b);
                    if (!s_a || !s_b) {
                        lost = true;
                        continue;
                    }
                    if (pa == s_a->n_in && s_a->max_out == uv && s_a->min_in > uv) g += w;
                    if (pb == s_b->n_in && s_b->min_in == uv && s_b->max_out < uv) g -= w;
                }
                if (g) atomicAdd(&rw.g[v], g);
            }
        }
        __syncwarp();
        if (PASS == RV_EVAL && sa != kRvNone && rw.g[lane] < 0) src[idx] = (uint8_t)(sa | kRvBack);
        __syncwarp();
    }
    if (lost) atomicOr(d.err, ERR_TABLE);
}

// CTA per tile, a run of its segments per warp: the marked moves go back to their source blocks (Phi,
// Lambda, S1, block weights, objective as in the apply step; the nets keep their round-r stamps).  Resets the
// sub-round's moved-incidence count for the next sub-round.
template <typename Rec>
__global__ void __launch_bounds__(kThreads) k_rv_revert(const Dev d, int32_t rr)
{
    after_previous();
    __shared__ ApplyWarp aw[kWarps];
    __shared__ SegRun run_w[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        d.rv_cnt[0] = 0;
        d.rv_cnt[1] = 0;
    }
    int32_t s0, s1;
    warp_segments(d, wid, s0, s1);
    if (s0 >= s1) return;
    SegRun &run = run_w[wid];
    const int32_t ncand = run.load(d, blockIdx.x, s0, s1);
    if (ncand == 0) return;
    Rec *recs = reinterpret_cast<Rec *>(d.rec);
    const int32_t r = d.rs[0];
    long long dobj = 0;
    int32_t nrev = 0;
    for (int32_t c0 = 0; c0 < ncand; c0 += 32) {
        const int32_t idx = c0 + lane < ncand ? run.at(c0 + lane) : 0;
        const uint8_t sa = c0 + lane < ncand ? d.rv_src[idx] : kRvNone;
        const bool back = sa != kRvNone && (sa & kRvBack);
        if (!__any_sync(kFull, back)) continue;
        int32_t deg = 0, jb = 0;
        int t = 0, a = 0;
        if (back) {
            int ul;
            int32_t g;
            decode(d.cand[idx], t, g, ul);
            const int32_t u = cand_vertex(idx, ul);
            a = sa & 0x3F;
            d.part[u] = (uint8_t)a;
            const long long cw = d.vw ? d.vw[u] : 1;
            atomicAdd(reinterpret_cast<unsigned long long *>(&d.bw[t]), (unsigned long long)(-cw));
            atomicAdd(reinterpret_cast<unsigned long long *>(&d.bw[a]), (unsigned long long)cw);
            jb = d.vtx_off[u];
            deg = d.vtx_off[u + 1] - jb;
            ++nrev;
        }
        int32_t incl = deg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int32_t total = __shfl_sync(kFull, incl, 31);
        aw[wid].off[lane] = incl - deg;
        aw[wid].jb[lane] = jb;
        aw[wid].a[lane] = t;     // the move back leaves the target block ...
        aw[wid].t[lane] = a;     // ... for the source block
        if (lane == 31) aw[wid].off[32] = total;
        __syncwarp();
        for (int32_t i0 = 0; i0 < total; i0 += 32 * kPins)
            dobj += apply_pins<Rec>(d, d.inc, recs, aw[wid], i0 + lane, total, r);
        __syncwarp();
    }
    for (int o = 16; o; o >>= 1) {
        dobj += __shfl_xor_sync(kFull, dobj, o);
        nrev += __shfl_xor_sync(kFull, nrev, o);
    }
    if (lane == 0) {
        if (dobj) atomicAdd(reinterpret_cast<unsigned long long *>(d.obj), (unsigned long long)dobj);
        if (nrev) atomicAdd(reinterpret_cast<unsigned long long *>(d.stats + (int64_t)rr * ST_N + ST_REV),
                            (unsigned long long)nrev);
    }
}

// The 1-byte partitions of up to kGather members one after another (batch read-back): grid row i
// copies member i.  One launch for 120 of them; a launch each cost the host 1 ms for 256.
constexpr int kGather = 120;
struct GatherArgs {
    const uint8_t *part[kGather];
    int64_t off[kGather + 1];
};
__global__ void __launch_bounds__(256) k_part_gather(const GatherArgs g, uint8_t *out)
{
    const int i = blockIdx.y;
    const uint8_t *src = g.part[i];
    const int64_t n = g.off[i + 1] - g.off[i];
    uint8_t *dst = out + g.off[i];
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        dst[v] = src[v];
}

// thread per instance: per-round objective and heaviest block; advance the round state
__global__ void k_round_end(const Dev *devs, int32_t n_inst, int32_t rr, int32_t advance = 1)
{
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_inst) return;
    const Dev d = devs[i];
    unsigned long long *row = reinterpret_cast<unsigned long long *>(d.stats + (int64_t)rr * ST_N);
    long long mx = 0;
    for (int t = 0; t < d.k; ++t) mx = d.bw[t] > mx ? d.bw[t] : mx;
    row[ST_OBJ] = (unsigned long long)*d.obj;
    row[ST_MAXW] = (unsigned long long)mx;
    if (advance) {
        d.rs[0] += 1;
        d.rs[1] = 1;
    }
}

// Rebalancing, source side (KEY_A): persistent, a CTA per tile with a grid stride (the
// per-block thresholds are read once per warp); marks the candidates that may leave their block
// (bit 25) and counts them by target block and priority for the target-side stage.
__global__ void __launch_bounds__(kThreads) k_rb_mark(const Dev d)
{
    after_previous();
    __shared__ ApplyInst ai_w[kWarps];
    __shared__ SegRun run_w[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t r;
    apply_refresh(d, ai_w[wid], r);
    int32_t s0, s1;
    warp_segments(d, wid, s0, s1);
    for (int32_t tile = blockIdx.x; tile < d.n_tiles && s0 < s1; tile += gridDim.x) {
        const int32_t ncand = run_w[wid].load(d, tile, s0, s1);
        for (int32_t i0 = 0; i0 < ncand; i0 += 32) {
            int t = 0;
            int32_t u = 0, g = 0, cu = 1;
            bool pass = false;
            if (i0 + lane < ncand) {
                const int32_t slot = run_w[wid].at(i0 + lane);
                const uint64_t c = d.cand[slot];
                pass = approve<KEY_A>(c, slot, ai_w[wid], t, u);
                g = (int32_t)(c >> 32);
                if (pass) {
                    d.cand[slot] = c | kSelBit;
                    if (d.vw) cu = d.vw[u];
                }
            }
            count_gain(d, pass, t, g, cu);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_expand_candidates(const Dev *devs, int32_t *target, int64_t *gain)
{
    __shared__ SegRun run_w[kWarps];
    const Dev &d = devs[0];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t s0, s1;
    warp_segments(d, wid, s0, s1);
    if (s0 >= s1) return;
    const int32_t n = run_w[wid].load(d, blockIdx.x, s0, s1);
    for (int32_t i = lane; i < n; i += 32) {
        const int32_t slot = run_w[wid].at(i);
        int t, ul;
        int32_t g;
        decode(d.cand[slot], t, g, ul);
        target[cand_vertex(slot, ul)] = t;
        gain[cand_vertex(slot, ul)] = g;
    }
}

// ------------------------------------------------------------------ launch plans (host)
// A set of instances with one record type, launched together: one instance with its own
// tiles (items == nullptr), or a batch group with explicit (instance, local index) items.
struct Plan {
    Dev d0{};                     // single instance: its state by value (kernel parameter)
    const Dev *devs = nullptr;
    const int2 *tiles = nullptr, *blocks = nullptr;
    int32_t n_tiles = 0, n_blocks = 0, n_inst = 0;
    int32_t S_max = 0;
    int32_t nseg = 1;      // segments per tile (batches: the members' largest)
    int32_t take = 1;      // gain items a warp takes at a time
    int32_t per = 1;       // segments per apply item
    bool levels = false;   // some instance can have gains >= kBins - 1
    bool rec32 = false;
    bool revert = false;   // revert variant (single instance only)
    int grid_gain = 0, grid_apply = 0;
    cudaStream_t st = nullptr;
    int64_t *launches = nullptr;
    hgp_handle *prof = nullptr;   // per-phase event timing (single-instance launches only)
};

// persistent grid of ctas_per_sm CTAs per SM (0: as many as fit), at most one warp per work item
template <typename K>
int persistent_grid(int device, K kernel, int ctas_per_sm, int64_t n_items)
{
    int sms = 0, per_sm = ctas_per_sm;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (per_sm <= 0) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, 0);
    (void)cudaGetLastError();
    int64_t g = (int64_t)(sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
    const int64_t need = (n_items + kWarps - 1) / kWarps;
    if (g > need) g = need;
    return (int)(g < 1 ? 1 : g);
}

// Grids and work granularity of the gain and apply kernels.  A gain item is one segment; a warp
// takes several at a time once it has 32 or more of them (the counter is one address).  An apply
// item is as many segments as leave a warp one item (its candidates are decided together), at
// most half a tile.
void set_grids(Plan &p, int device, int gain_ctas, int apply_ctas)
{
    const bool b = p.tiles != nullptr;
    const int64_t segs = (int64_t)p.n_tiles * p.nseg;
    if (p.rec32) {
        p.grid_gain = persistent_grid(device, b ? k_gain<Rec32, true> : k_gain<Rec32, false>, gain_ctas, segs);
        p.grid_apply = persistent_grid(device, b ? k_apply<Rec32, true> : k_apply<Rec32, false>, apply_ctas, segs);
    } else {
        p.grid_gain = persistent_grid(device, b ? k_gain<Rec16, true> : k_gain<Rec16, false>, gain_ctas, segs);
        p.grid_apply = persistent_grid(device, b ? k_apply<Rec16, true> : k_apply<Rec16, false>, apply_ctas, segs);
    }
    p.take = (int32_t)std::min<int64_t>(4, std::max<int64_t>(1, segs / ((int64_t)p.grid_gain * kWarps * 8)));
    int64_t per = (segs + (int64_t)p.grid_apply * kWarps - 1) / ((int64_t)p.grid_apply * kWarps);
    per = std::min<int64_t>(std::max<int64_t>(per, 1), std::min<int64_t>(32, (p.nseg + 1) / 2));
    const int64_t groups = (p.nseg + per - 1) / per;
    p.per = (int32_t)((p.nseg + groups - 1) / groups);
}

// Per-phase event timing (profiling mode): a pair of events around each phase instance.
enum { PH_PREP = 0, PH_GAIN = 1, PH_APPROVE = 2, PH_APPLY = 3, PH_END = 4, PH_REVERT = 5 };

cudaError_t phase_begin(hgp_handle *h)
{
    if (!h || !h->profiling) return cudaSuccess;
    if (h->events_used + 2 > h->n_events) {
        // grow the pool (existing events stay valid; pending pairs are kept)
        const int32_t cap = h->n_events ? h->n_events * 2 : 256;
        cudaEvent_t *ev = new (std::nothrow) cudaEvent_t[cap];
        int32_t *ph = new (std::nothrow) int32_t[cap / 2];
        int32_t *ct = new (std::nothrow) int32_t[cap / 2];
        if (!ev || !ph || !ct) {
            delete[] ev; delete[] ph; delete[] ct;
            return cudaErrorMemoryAllocation;
        }
        for (int32_t i = 0; i < h->n_events; ++i) ev[i] = h->events[i];
        for (int32_t i = 0; i < h->n_events / 2; ++i) { ph[i] = h->event_phase[i]; ct[i] = h->event_count[i]; }
        for (int32_t i = h->n_events; i < cap; ++i) {
            cudaError_t e = cudaEventCreate(&ev[i]);
            if (e != cudaSuccess) {
                for (int32_t j = h->n_events; j < i; ++j) cudaEventDestroy(ev[j]);
                delete[] ev; delete[] ph; delete[] ct;
                return e;
            }
        }
        delete[] h->events; delete[] h->event_phase; delete[] h->event_count;
        h->events = ev; h->event_phase = ph; h->event_count = ct;
        h->n_events = cap;
    }
    return cudaEventRecord(h->events[h->events_used], h->stream);
}

cudaError_t phase_end(hgp_handle *h, int phase, int32_t launches)
{
    if (!h || !h->profiling) return cudaSuccess;
    cudaError_t e = cudaEventRecord(h->events[h->events_used + 1], h->stream);
    h->event_phase[h->events_used / 2] = phase;
    h->event_count[h->events_used / 2] = launches;
    h->events_used += 2;
    return e;
}

cudaError_t collect_profile(hgp_handle *h)
{
    if (!h->profiling || h->events_used == 0) return cudaSuccess;
    cudaError_t e = stream_wait(h->stream);
    for (int32_t i = 0; i + 1 < h->events_used && e == cudaSuccess; i += 2) {
        float ms = 0.f;
        e = cudaEventElapsedTime(&ms, h->events[i], h->events[i + 1]);
        h->prof_ms[h->event_phase[i / 2]] += ms;
        h->prof_launches[h->event_phase[i / 2]] += h->event_count[i / 2];
    }
    h->events_used = 0;
    return e;
}

constexpr int32_t kTieCtas = 152 * 8;   // k_tie_sum: as many as are resident

// a kernel of a round (see after_previous); errors are read by cudaGetLastError at the call site
template <typename... KA, typename... A>
void launch(void (*kernel)(KA...), int64_t grid, unsigned block, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

cudaError_t launch_gain(const Plan &p, int32_t s, int32_t rr)
{
    const bool b = p.tiles != nullptr;
    if (p.rec32 && b) launch(k_gain<Rec32, true>, p.grid_gain, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.take, s, rr, RbArgs{0, 0, 0, 1});
    else if (p.rec32) launch(k_gain<Rec32, false>, p.grid_gain, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.take, s, rr, RbArgs{0, 0, 0, 1});
    else if (b) launch(k_gain<Rec16, true>, p.grid_gain, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.take, s, rr, RbArgs{0, 0, 0, 1});
    else launch(k_gain<Rec16, false>, p.grid_gain, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.take, s, rr, RbArgs{0, 0, 0, 1});
    *p.launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_prep(const Plan &p)
{
    launch(k_round_prep, p.n_tiles, kThreads, p.st, p.devs, p.tiles, p.n_tiles, -1);
    *p.launches += 1;
    return cudaGetLastError();
}

// one round: sub-round lists, then per sub-round gain -> approval -> apply, then round end
cudaError_t launch_round(const Plan &p, int32_t rr)
{
    cudaError_t e = phase_begin(p.prof);
    if (e == cudaSuccess) e = launch_prep(p);
    if (e == cudaSuccess) e = phase_end(p.prof, PH_PREP, 1);
    for (int32_t s = 0; s < p.S_max && e == cudaSuccess; ++s) {
        e = phase_begin(p.prof);
        if (e == cudaSuccess) e = launch_gain(p, s, rr);
        if (e == cudaSuccess) e = phase_end(p.prof, PH_GAIN, 1);
        if (e == cudaSuccess) e = phase_begin(p.prof);
        if (e != cudaSuccess) break;
        int32_t n = 0;
        // the level-0 histogram was filled by the gain step
        launch(k_select<KEY_T>, p.n_blocks, kThreads, p.st, p.devs, p.blocks, p.n_blocks, 0, 0);
        n += 1;
        if (p.levels) {
            for (int level = 1; level <= 3; ++level) {
                launch(k_hist<KEY_T>, p.n_tiles, kThreads, p.st, p.devs, p.tiles, p.n_tiles, level);
                launch(k_select<KEY_T>, p.n_blocks, kThreads, p.st, p.devs, p.blocks, p.n_blocks, level, 0);
                n += 2;
            }
        }
        launch(k_tie_sum<KEY_T>, std::min(p.n_tiles, kTieCtas), kThreads, p.st, p.devs, p.tiles, p.n_tiles);
        launch(k_tie_cut<KEY_T>, p.n_blocks, 1024, p.st, p.devs, p.blocks, p.n_blocks);
        n += 2;
        *p.launches += n;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = phase_end(p.prof, PH_APPROVE, n);
        if (e == cudaSuccess) e = phase_begin(p.prof);
        if (e != cudaSuccess) break;
        const bool b = p.tiles != nullptr;
        if (p.revert) e = cudaMemsetAsync(p.d0.rv_net, 0, sizeof(int32_t) * (size_t)p.d0.m, p.st);
        if (e != cudaSuccess) break;
        if (p.rec32 && b) launch(k_apply<Rec32, true>, p.grid_apply, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.per, rr);
        else if (p.rec32) launch(k_apply<Rec32, false>, p.grid_apply, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.per, rr);
        else if (b) launch(k_apply<Rec16, true>, p.grid_apply, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.per, rr);
        else launch(k_apply<Rec16, false>, p.grid_apply, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, p.per, rr);
        *p.launches += 1;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = phase_end(p.prof, PH_APPLY, 1);
        if (p.revert && e == cudaSuccess) e = phase_begin(p.prof);
        if (e == cudaSuccess && p.revert) {
            const unsigned g = p.n_tiles;
            // the apply step counted the movers of every net and the shared incidences
            launch(k_rv_clear, p.grid_apply * 4, kThreads, p.st, p.d0);
            if (p.rec32) {
                launch(k_rv_pass<Rec32, RV_INSERT>, g, kThreads, p.st, p.d0);
                launch(k_rv_pass<Rec32, RV_EVAL>, g, kThreads, p.st, p.d0);
                launch(k_rv_revert<Rec32>, g, kThreads, p.st, p.d0, rr);
            } else {
                launch(k_rv_pass<Rec16, RV_INSERT>, g, kThreads, p.st, p.d0);
                launch(k_rv_pass<Rec16, RV_EVAL>, g, kThreads, p.st, p.d0);
                launch(k_rv_revert<Rec16>, g, kThreads, p.st, p.d0, rr);
            }
            *p.launches += 4;
            e = cudaGetLastError();
            if (e == cudaSuccess) e = phase_end(p.prof, PH_REVERT, 4);
        }
    }
    if (e == cudaSuccess) e = phase_begin(p.prof);
    if (e == cudaSuccess) {
        launch(k_round_end, (p.n_inst + 127) / 128, 128, p.st, p.devs, p.n_inst, rr, 1);
        *p.launches += 1;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = phase_end(p.prof, PH_END, 1);
    return e;
}

// the handle's instance state as a device-resident Dev (re-uploaded when it changed)
cudaError_t sync_dev(hgp_handle *h)
{
    if (!h->d_dev) {
        h->d_dev = static_cast<Dev *>(arena_take(h, sizeof(Dev)));
        if (!h->d_dev) {
            cudaError_t e = dev_alloc(reinterpret_cast<void **>(&h->d_dev), sizeof(Dev), h->stream);
            if (e != cudaSuccess) return e;
        }
        h->dev_dirty = true;
    }
    if (!h->dev_dirty) return cudaSuccess;
    cudaError_t e = cudaMemcpyAsync(h->d_dev, &h->d, sizeof(Dev), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = stream_wait(h->stream);
    if (e == cudaSuccess) h->dev_dirty = false;
    return e;
}

Plan single_plan(hgp_handle *h)
{
    Plan p;
    p.d0 = h->d;
    p.devs = h->d_dev;
    p.n_tiles = h->d.n_tiles;
    p.nseg = h->d.nseg;
    p.n_blocks = h->d.k;
    p.n_inst = 1;
    p.S_max = h->d.S;
    p.levels = h->max_vertex_netweight >= kBins - 1;
    p.rec32 = h->d.k > 32;
    p.revert = h->d.rv_src != nullptr;
    if (!h->grid_gain) {
        set_grids(p, h->device, h->gain_ctas, h->apply_ctas);
        h->grid_gain = p.grid_gain;
        h->grid_apply = p.grid_apply;
        h->gain_take = p.take;
        h->apply_per = p.per;
    }
    p.grid_gain = h->grid_gain;
    p.grid_apply = h->grid_apply;
    p.take = h->gain_take;
    p.per = h->apply_per;
    p.st = h->stream;
    p.launches = &h->launches;
    p.prof = h->profiling ? h : nullptr;
    return p;
}

// Whether a handle's rounds run as one cluster (hgp_small.cuh): instances of up to kSmallVertices
// vertices and kSmallPins pins on a device that can hold the cluster.  Per-phase profiling and the
// revert variant take the launches of the general path.
bool small_plan(const Plan &p, int device, int32_t debug)
{
    if (p.prof || p.revert || p.tiles || p.d0.n > kSmallVertices || (debug & 32)) return false;
    if (p.d0.P > (p.rec32 ? kSmallPinsWide : kSmallPins)) return false;
    static std::mutex mu;
    static int8_t ready[64][2];   // per device and record type: 0 not asked yet, 1 yes, 2 no
    if (device < 0 || device >= 64) return false;
    std::lock_guard<std::mutex> lk(mu);
    int8_t &r = ready[device][p.rec32];
    if (r == 0) {
        auto kernel = p.rec32 ? k_small<Rec32> : k_small<Rec16>;
        cudaLaunchAttribute at;
        bool cached;
        int32_t inc_room;
        cudaLaunchConfig_t cfg = small_config(p.d0, nullptr, &at, cached, inc_room);
        cfg.dynamicSmemBytes = kSmMaxBytes;   // the largest of any handle
        int clusters = 0;
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
        if (e != cudaSuccess) (void)cudaGetLastError();
        r = e == cudaSuccess && clusters > 0 ? 1 : 2;
    }
    return r == 1;
}

cudaError_t launch_small(const Plan &p, int32_t rounds, int64_t max_netweight)
{
    int nd = 1;
    while (nd < 4 && (max_netweight >> (kSmDigit * nd)) > 0) ++nd;
    cudaLaunchAttribute at;
    bool cached;
    int32_t inc_room;
    const cudaLaunchConfig_t cfg = small_config(p.d0, p.st, &at, cached, inc_room);
    *p.launches += 1;
    return p.rec32 ? cudaLaunchKernelEx(&cfg, k_small<Rec32>, p.d0, rounds, (int32_t)nd, cached, inc_room)
                   : cudaLaunchKernelEx(&cfg, k_small<Rec16>, p.d0, rounds, (int32_t)nd, cached, inc_room);
}

cudaError_t enqueue_rounds(const Plan &p, int64_t *stats, int32_t rounds, bool small, int64_t max_netweight)
{
    if (small) return launch_small(p, rounds, max_netweight);
    cudaError_t e = cudaMemsetAsync(stats, 0, sizeof(int64_t) * ST_N * (size_t)rounds, p.st);
    if (e == cudaSuccess && p.d0.wq) e = cudaMemsetAsync(p.d0.wq, 0, sizeof(int32_t) * kWqPerRow * (size_t)rounds, p.st);
    for (int32_t rr = 0; rr < rounds && e == cudaSuccess; ++rr) e = launch_round(p, rr);
    return e;
}

}  // namespace

namespace hgp {

int ensure_stats(hgp_handle *h, int32_t rounds)
{
    if (rounds <= h->stats_cap) return HGP_OK;
    int32_t cap = h->stats_cap ? h->stats_cap : 16;
    while (cap < rounds) cap *= 2;
    int64_t *dev = nullptr, *host = nullptr;
    // stats rows, then the gain step's work counters
    const size_t bytes = sizeof(int64_t) * ST_N * (size_t)cap + sizeof(int32_t) * kWqPerRow * (size_t)cap;
    cudaError_t e = cudaSuccess;
    dev = static_cast<int64_t *>(arena_take(h, bytes));
    if (!dev) e = dev_alloc(reinterpret_cast<void **>(&dev), bytes, h->stream);
    if (e == cudaSuccess) {
        host = static_cast<int64_t *>(malloc(sizeof(int64_t) * ST_N * (size_t)cap));
        if (!host) e = cudaErrorMemoryAllocation;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        if (!in_arena(h, dev)) dev_free(dev, h->stream);
        return status_of(e);
    }
    if (h->d.stats && !in_arena(h, h->d.stats)) dev_free(h->d.stats, h->stream);
    free(h->h_stats);
    h->d.stats = dev;
    h->d.wq = reinterpret_cast<int32_t *>(dev + (size_t)ST_N * cap);
    h->h_stats = host;
    h->stats_cap = cap;
    h->dev_dirty = true;
    if (h->graph_exec) {
        cudaGraphExecDestroy(h->graph_exec);
        h->graph_exec = nullptr;
        h->graph_rounds = 0;
    }
    return HGP_OK;
}

static int copy_stats_out(hgp_handle *h, int32_t rounds, hgp_round_stats *stats)
{
    cudaError_t e = cudaMemcpyAsync(h->h_stats, h->d.stats, sizeof(int64_t) * ST_N * (size_t)rounds,
                                    cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = stream_wait(h->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    if (stats) {
        for (int32_t rr = 0; rr < rounds; ++rr) {
            const int64_t *row = h->h_stats + (int64_t)rr * ST_N;
            stats[rr].objective = row[ST_OBJ];
            stats[rr].candidates = row[ST_CAND];
            stats[rr].approved = row[ST_APPR];
            stats[rr].eligible = row[ST_ELIG];
            stats[rr].max_block_weight = row[ST_MAXW];
            stats[rr].moved_pins = row[ST_MOVED];
            stats[rr].reverted = row[ST_REV];
        }
    }
    return HGP_OK;
}

int refine_rounds(hgp_handle *h, int32_t rounds, hgp_round_stats *stats)
{
    if (rounds == 0) return HGP_OK;
    if (h->next_round + rounds >= ((int64_t)1 << 30)) return HGP_ERR_UNSUPPORTED;
    int rc = ensure_stats(h, rounds);
    if (rc != HGP_OK) return rc;
    cudaError_t e = sync_dev(h);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    Plan p = single_plan(h);
    const bool use_graph = h->graph && !h->profiling;
    const bool small = small_plan(p, h->device, h->debug);
    if (use_graph) {
        if (!h->graph_exec || h->graph_rounds != rounds) {
            if (h->graph_exec) {
                cudaGraphExecDestroy(h->graph_exec);
                h->graph_exec = nullptr;
            }
            // the captured launches are counted at replay, not at capture
            int64_t scratch = 0;
            Plan q = p;
            q.launches = &scratch;
            cudaGraph_t graph = nullptr;
            e = cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                const cudaError_t e2 = enqueue_rounds(q, h->d.stats, rounds, small, h->max_vertex_netweight);
                e = cudaStreamEndCapture(h->stream, &graph);
                if (e2 != cudaSuccess) e = e2;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&h->graph_exec, graph, 0);
            if (graph) cudaGraphDestroy(graph);
            if (e == cudaSuccess) {
                h->graph_rounds = rounds;
                h->graph_launches = scratch;
            }
        }
        if (e == cudaSuccess) e = cudaGraphLaunch(h->graph_exec, h->stream);
        if (e == cudaSuccess) h->launches += h->graph_launches;
    } else {
        e = enqueue_rounds(p, h->d.stats, rounds, small, h->max_vertex_netweight);
        if (e == cudaSuccess) e = collect_profile(h);
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    h->next_round += rounds;
    h->all_eligible = false;
    if (h->debug & 16) {
        // fault injection (tests): the maintained objective loses one unit, as if an update
        // had been dropped; written from the host after the rounds, so no kernel is involved
        int64_t obj = 0;
        e = cudaMemcpyAsync(&obj, h->d.obj, sizeof(int64_t), cudaMemcpyDeviceToHost, h->stream);
        if (e == cudaSuccess) e = stream_wait(h->stream);
        obj -= 1;
        if (e == cudaSuccess) e = cudaMemcpyAsync(h->d.obj, &obj, sizeof(int64_t), cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess) e = stream_wait(h->stream);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return status_of(e);
        }
    }
    if (stats || (h->debug & 1)) {
        rc = copy_stats_out(h, rounds, stats);
        if (rc != HGP_OK) return rc;
    }
    if (h->debug & 1) {
        int64_t *tmp = nullptr;
        int64_t from_phi = 0, maintained = 0;
        e = dev_alloc(reinterpret_cast<void **>(&tmp), sizeof(int64_t), h->stream);
        if (e == cudaSuccess) e = objective_from_phi(h, tmp);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&from_phi, tmp, sizeof(int64_t), cudaMemcpyDeviceToHost, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&maintained, h->d.obj, sizeof(int64_t), cudaMemcpyDeviceToHost, h->stream);
        if (tmp) pool_free(tmp, h->stream);
        if (e == cudaSuccess) e = stream_wait(h->stream);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return status_of(e);
        }
        if (from_phi != maintained) return HGP_ERR_INTERNAL;
    }
    return HGP_OK;
}

int debug_candidates(hgp_handle *h, int32_t s, int32_t *target, int64_t *gain)
{
    const int rc = ensure_stats(h, 1);
    if (rc != HGP_OK) return rc;
    Dev &d = h->d;
    cudaStream_t st = h->stream;
    cudaError_t e = sync_dev(h);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    Plan p = single_plan(h);
    int32_t *t_d = nullptr;
    int64_t *g_d = nullptr;
    e = dev_alloc(reinterpret_cast<void **>(&t_d), sizeof(int32_t) * (size_t)d.n, st);
    if (e == cudaSuccess) e = dev_alloc(reinterpret_cast<void **>(&g_d), sizeof(int64_t) * (size_t)d.n, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(t_d, 0xFF, sizeof(int32_t) * (size_t)d.n, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(g_d, 0, sizeof(int64_t) * (size_t)d.n, st);
    // the stats row written here is scratch: refine() clears the stats before use
    if (e == cudaSuccess) e = launch_prep(p);
    if (e == cudaSuccess) e = cudaMemsetAsync(d.wq, 0, sizeof(int32_t) * kWqPerRow, st);
    if (e == cudaSuccess) e = launch_gain(p, s, 0);
    if (e == cudaSuccess) e = cudaMemsetAsync(d.hist, 0, sizeof(unsigned long long) * (size_t)d.k * kBins, st);
    if (e == cudaSuccess) {
        k_expand_candidates<<<d.n_tiles, kThreads, 0, st>>>(h->d_dev, t_d, g_d);
        h->launches++;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(target, t_d, sizeof(int32_t) * (size_t)d.n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(gain, g_d, sizeof(int64_t) * (size_t)d.n, cudaMemcpyDeviceToHost, st);
    if (t_d) pool_free(t_d, st);
    if (g_d) pool_free(g_d, st);
    if (e == cudaSuccess) e = stream_wait(st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return HGP_OK;
}

}  // namespace hgp

// ================================================================== launch shape
extern "C" int hgp_set_launch_shape(hgp_handle *h, int32_t gain_ctas_per_sm, int32_t apply_ctas_per_sm)
{
    if (!h || gain_ctas_per_sm < 0 || apply_ctas_per_sm < 0) return HGP_ERR_INVALID;
    settle(h);
    const cudaError_t e = stream_wait(h->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    h->gain_ctas = gain_ctas_per_sm;
    h->apply_ctas = apply_ctas_per_sm;
    h->grid_gain = 0;   // recomputed at the next launch
    h->grid_apply = 0;
    if (h->graph_exec) {
        cudaGraphExecDestroy(h->graph_exec);
        h->graph_exec = nullptr;
        h->graph_rounds = 0;
    }
    return HGP_OK;
}

// ================================================================== rebalancing (Sec. 8)
namespace {

// one approval stage over all candidates of the sub-round, grouped by KEY
template <int KEY>
int64_t launch_stage(const Plan &p, bool levels, int32_t bins)
{
    int64_t n = 0;
    launch(k_select<KEY>, p.n_blocks, kThreads, p.st, p.devs, p.blocks, p.n_blocks, 0, bins);
    n += 1;
    if (levels) {
        for (int level = 1; level <= 3; ++level) {
            launch(k_hist<KEY>, p.n_tiles, kThreads, p.st, p.devs, p.tiles, p.n_tiles, level);
            launch(k_select<KEY>, p.n_blocks, kThreads, p.st, p.devs, p.blocks, p.n_blocks, level, 0);
            n += 2;
        }
    }
    launch(k_tie_sum<KEY>, std::min(p.n_tiles, kTieCtas), kThreads, p.st, p.devs, p.tiles, p.n_tiles);
    launch(k_tie_cut<KEY>, p.n_blocks, 1024, p.st, p.devs, p.blocks, p.n_blocks);
    return n + 2;
}

// one rebalancing pass: S sub-rounds of gain (vertices of overloaded blocks), source-side
// selection, target-side approval and apply, then the pass's objective and heaviest block
template <typename Rec>
cudaError_t launch_rebalance_pass(const Plan &p, int32_t pass, RbArgs rb, bool levels, int32_t bins)
{
    launch(k_round_prep, p.n_tiles, kThreads, p.st, p.devs, p.tiles, p.n_tiles, rb.r);
    *p.launches += 1;
    for (int32_t s = 0; s < p.S_max; ++s) {
        launch(k_gain<Rec, false, true>, p.grid_gain, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, (p.nseg + rb.segs - 1) / rb.segs, 1, s,
                                                                    pass, rb);
        *p.launches += 1;
        *p.launches += launch_stage<KEY_A>(p, levels, bins);
        launch(k_rb_mark, p.grid_apply, kThreads, p.st, p.d0);
        *p.launches += 1;
        *p.launches += launch_stage<KEY_TS>(p, levels, bins);
        launch(k_apply<Rec, false, KEY_TS>, p.grid_apply, kThreads, p.st, p.d0, p.devs, p.tiles, p.n_tiles, p.nseg, std::min(p.per, rb.segs), pass);
        *p.launches += 1;
    }
    launch(k_round_end, 1, 128, p.st, p.devs, 1, pass, 0);
    *p.launches += 1;
    return cudaGetLastError();
}

}  // namespace

extern "C" int hgp_rebalance(hgp_handle *h, int32_t max_passes, hgp_round_stats *stats, int32_t *phases,
                             int32_t *num_passes)
{
    if (!h || max_passes < 0) return HGP_ERR_INVALID;
    settle(h);
    if (num_passes) *num_passes = 0;
    if (max_passes == 0) return HGP_OK;
    // phase-2 priorities are gain + W_max in [0, 2 W_max]; they must fit the 31-bit gain field
    const int64_t off = h->max_vertex_netweight;
    if (2 * off >= ((int64_t)1 << 31)) return HGP_ERR_UNSUPPORTED;
    int rc = ensure_stats(h, max_passes);
    if (rc != HGP_OK) return rc;
    cudaError_t e = sync_dev(h);
    const cudaStream_t st = h->stream;
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d.stats, 0, sizeof(int64_t) * ST_N * (size_t)max_passes, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d.wq, 0, sizeof(int32_t) * kWqPerRow * (size_t)max_passes, st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    Plan p = single_plan(h);
    p.prof = nullptr;
    std::vector<int32_t> ph;
    int32_t phase = 1, pass = 0;
    while (pass < max_passes && e == cudaSuccess) {
        int64_t bw[64];
        e = cudaMemcpyAsync(bw, h->d.bw, sizeof(int64_t) * (size_t)h->d.k, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = stream_wait(st);
        if (e != cudaSuccess) break;
        int64_t heaviest = 0;
        for (int i = 0; i < h->d.k; ++i) heaviest = bw[i] > heaviest ? bw[i] : heaviest;
        if (heaviest <= h->d.lmax) break;
        RbArgs rb;
        rb.r = (1 << 30) + pass;
        rb.phase = phase;
        rb.off = phase == 2 ? (int32_t)off : 0;
        rb.segs = rb_segments(h->d.S, h->d.n / ((int64_t)p.grid_apply * kWarps));
        const int64_t top = phase == 2 ? 2 * off : off;   // largest priority
        const bool levels = top >= kBins - 1;
        const int32_t bins = (int32_t)std::min<int64_t>(kBins, (top + kThreads) / kThreads * kThreads);
        e = p.rec32 ? launch_rebalance_pass<Rec32>(p, pass, rb, levels, bins)
                    : launch_rebalance_pass<Rec16>(p, pass, rb, levels, bins);
        int64_t appr = 0;
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&appr, h->d.stats + (int64_t)pass * ST_N + ST_APPR, sizeof(int64_t),
                                cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = stream_wait(st);
        if (e != cudaSuccess) break;
        ph.push_back(phase);
        ++pass;
        if (phase == 1) phase = 2;
        else if (appr == 0) break;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    if (pass > 0 && stats) {
        rc = copy_stats_out(h, pass, stats);
        if (rc != HGP_OK) return rc;
    }
    if (phases)
        for (int32_t i = 0; i < pass; ++i) phases[i] = ph[i];
    if (num_passes) *num_passes = pass;
    return HGP_OK;
}

// ================================================================== batch of handles
struct hgp_batch {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int32_t use_graph = 1;
    int32_t gain_ctas = 0, apply_ctas = 0;     // per-SM CTA overrides (0 = occupancy)
    std::vector<hgp_handle *> hs;
    // the members' streams other than the batch's: a call waits (on the device) for their
    // pending work through events[i], and records its end on each such member's own event
    std::vector<cudaStream_t> member_streams;
    std::vector<cudaEvent_t> events;
    int32_t last_rounds = 0;                    // round count of the last hgp_batch_refine
    cudaEvent_t ev_end = nullptr;               // recorded at the end of each hgp_batch_refine
    cudaStream_t aux = nullptr;                 // statistics read-back of a call, after ev_end only
    struct Group {
        Plan plan;
        std::vector<int32_t> members;           // indices into hs
        Dev *d_devs = nullptr;
        int2 *d_items = nullptr;                // tiles, then blocks
        int32_t *d_wq = nullptr;                // gain-step work counters [stats_cap * kWqPerRow]
    } g[2];
    int64_t *d_stats = nullptr;
    int64_t *h_stats = nullptr;
    int32_t stats_cap = 0;
    cudaGraphExec_t exec = nullptr;
    int32_t graph_rounds = 0;
    int64_t graph_launches = 0;
    int64_t launches = 0;
};

namespace {

void free_groups(hgp_batch *b)
{
    for (auto &gr : b->g) {
        dev_free(gr.d_devs, b->stream);
        dev_free(gr.d_items, b->stream);
        dev_free(gr.d_wq, b->stream);
        gr.d_devs = nullptr;
        gr.d_items = nullptr;
        gr.d_wq = nullptr;
    }
    if (b->exec) cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
    b->graph_rounds = 0;
}

// (re)builds the per-group device arrays for a stats capacity of `cap` rounds
int build_groups(hgp_batch *b, int32_t cap)
{
    free_groups(b);
    const int32_t count = (int32_t)b->hs.size();
    dev_free(b->d_stats, b->stream);
    free(b->h_stats);
    b->d_stats = nullptr;
    b->h_stats = nullptr;
    cudaError_t e = dev_alloc(reinterpret_cast<void **>(&b->d_stats), sizeof(int64_t) * ST_N * (size_t)cap * count,
                              b->stream);
    if (e == cudaSuccess) {
        b->h_stats = static_cast<int64_t *>(malloc(sizeof(int64_t) * ST_N * (size_t)cap * count));
        if (!b->h_stats) e = cudaErrorMemoryAllocation;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    b->stats_cap = cap;
    for (int gi = 0; gi < 2; ++gi) {
        auto &gr = b->g[gi];
        gr.members.clear();
        for (int32_t i = 0; i < count; ++i)
            if ((b->hs[i]->d.k > 32) == (gi == 1)) gr.members.push_back(i);
        gr.plan = Plan();
        if (gr.members.empty()) continue;
        std::vector<Dev> devs;
        std::vector<int2> tiles, blocks;
        int32_t S_max = 0, nseg = 1;
        bool levels = false;
        for (size_t j = 0; j < gr.members.size(); ++j) {
            const hgp_handle *h = b->hs[gr.members[j]];
            Dev d = h->d;
            d.stats = b->d_stats + (int64_t)gr.members[j] * cap * ST_N;
            devs.push_back(d);
            for (int32_t t = 0; t < d.n_tiles; ++t) tiles.push_back(make_int2((int)j, t));
            for (int32_t t = 0; t < d.k; ++t) blocks.push_back(make_int2((int)j, t));
            S_max = d.S > S_max ? d.S : S_max;
            nseg = d.nseg > nseg ? d.nseg : nseg;
            levels = levels || h->max_vertex_netweight >= kBins - 1;
        }
        const size_t n_items = tiles.size() + blocks.size();
        e = dev_alloc(reinterpret_cast<void **>(&gr.d_devs), sizeof(Dev) * devs.size(), b->stream);
        if (e == cudaSuccess) e = dev_alloc(reinterpret_cast<void **>(&gr.d_items), sizeof(int2) * n_items, b->stream);
        if (e == cudaSuccess)
            e = dev_alloc(reinterpret_cast<void **>(&gr.d_wq), sizeof(int32_t) * kWqPerRow * (size_t)cap, b->stream);
        std::vector<int2> all;
        all.reserve(n_items);
        all.insert(all.end(), tiles.begin(), tiles.end());
        all.insert(all.end(), blocks.begin(), blocks.end());
        // pageable sources: each call returns once its source has been staged
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(gr.d_devs, devs.data(), sizeof(Dev) * devs.size(), cudaMemcpyHostToDevice, b->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(gr.d_items, all.data(), sizeof(int2) * n_items, cudaMemcpyHostToDevice, b->stream);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return status_of(e);
        }
        Plan &p = gr.plan;
        p.d0.wq = gr.d_wq;   // the batch kernels read only the work counters from d0
        p.devs = gr.d_devs;
        p.tiles = gr.d_items;
        p.blocks = gr.d_items + tiles.size();
        p.nseg = nseg;
        p.n_tiles = (int32_t)tiles.size();
        p.n_blocks = (int32_t)blocks.size();
        p.n_inst = (int32_t)devs.size();
        p.S_max = S_max;
        p.levels = levels;
        p.rec32 = gi == 1;
        set_grids(p, b->device, b->gain_ctas, b->apply_ctas);
        p.st = b->stream;
        p.launches = &b->launches;
    }
    return HGP_OK;
}

cudaError_t enqueue_batch(hgp_batch *b, int32_t rounds, int64_t *launch_counter)
{
    const int32_t count = (int32_t)b->hs.size();
    cudaError_t e = cudaMemsetAsync(b->d_stats, 0, sizeof(int64_t) * ST_N * (size_t)b->stats_cap * count, b->stream);
    for (int32_t rr = 0; rr < rounds && e == cudaSuccess; ++rr)
        for (auto &gr : b->g) {
            if (gr.members.empty() || e != cudaSuccess) continue;
            Plan p = gr.plan;
            p.launches = launch_counter;
            if (rr == 0) e = cudaMemsetAsync(p.d0.wq, 0, sizeof(int32_t) * kWqPerRow * (size_t)rounds, b->stream);
            if (e == cudaSuccess) e = launch_round(p, rr);
        }
    return e;
}

}  // namespace

// waits for the batch's stream and unpacks the per-member statistics of its last call
static int batch_stats_unpack(hgp_batch *b, int32_t rounds, hgp_round_stats *stats)
{
    const int32_t count = (int32_t)b->hs.size();
    for (int32_t i = 0; i < count; ++i)
        for (int32_t rr = 0; rr < rounds; ++rr) {
            const int64_t *row = b->h_stats + ((int64_t)i * b->stats_cap + rr) * ST_N;
            hgp_round_stats &o = stats[(int64_t)i * rounds + rr];
            o.objective = row[ST_OBJ];
            o.candidates = row[ST_CAND];
            o.approved = row[ST_APPR];
            o.eligible = row[ST_ELIG];
            o.max_block_weight = row[ST_MAXW];
            o.moved_pins = row[ST_MOVED];
            o.reverted = row[ST_REV];
        }
    return HGP_OK;
}

static int batch_stats_out(hgp_batch *b, int32_t rounds, hgp_round_stats *stats)
{
    const int32_t count = (int32_t)b->hs.size();
    cudaError_t e = cudaMemcpyAsync(b->h_stats, b->d_stats, sizeof(int64_t) * ST_N * (size_t)b->stats_cap * count,
                                    cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = stream_wait(b->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return batch_stats_unpack(b, rounds, stats);
}

extern "C" {

void hgp_batch_default_options(hgp_batch_options *opt)
{
    if (!opt) return;
    memset(opt, 0, sizeof(*opt));
    opt->graph = 1;
}

int hgp_batch_create(hgp_handle *const *handles, int32_t count, const hgp_batch_options *opt, hgp_batch **out)
{
    if (!out) return HGP_ERR_INVALID;
    *out = nullptr;
    if (!handles || count < 1) return HGP_ERR_INVALID;
    hgp_batch_options o;
    hgp_batch_default_options(&o);
    if (opt) o = *opt;
    int dev = 0;
    cudaGetDevice(&dev);
    for (int32_t i = 0; i < count; ++i) {
        if (!handles[i] || handles[i]->device != dev) return HGP_ERR_INVALID;
        if (handles[i]->d.rv_src) return HGP_ERR_UNSUPPORTED;   // revert variant: single instances only
        for (int32_t j = 0; j < i; ++j)
            if (handles[j] == handles[i]) return HGP_ERR_INVALID;
    }
    hgp_batch *b = new (std::nothrow) hgp_batch();
    if (!b) return HGP_ERR_OOM;
    b->device = dev;
    b->use_graph = o.graph;
    b->gain_ctas = o.gain_ctas_per_sm;
    b->apply_ctas = o.apply_ctas_per_sm;
    b->hs.assign(handles, handles + count);
    if (o.cuda_stream) {
        b->stream = (cudaStream_t)o.cuda_stream;
    } else if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
        (void)cudaGetLastError();
        delete b;
        return HGP_ERR_CUDA;
    } else {
        b->own_stream = true;
    }
    for (hgp_handle *h : b->hs) {
        if (h->stream == b->stream) continue;
        bool seen = false;
        for (cudaStream_t s2 : b->member_streams) seen = seen || s2 == h->stream;
        if (!seen) b->member_streams.push_back(h->stream);
    }
    for (size_t i = 0; i < b->member_streams.size(); ++i) {
        cudaEvent_t ev = nullptr;
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
            (void)cudaGetLastError();
            hgp_batch_destroy(b);
            return HGP_ERR_CUDA;
        }
        b->events.push_back(ev);
    }
    for (hgp_handle *h : b->hs)
        if (h->stream != b->stream && !h->ev_batch &&
            cudaEventCreateWithFlags(&h->ev_batch, cudaEventDisableTiming) != cudaSuccess) {
            (void)cudaGetLastError();
            h->ev_batch = nullptr;
            hgp_batch_destroy(b);
            return HGP_ERR_CUDA;
        }
    if (cudaEventCreateWithFlags(&b->ev_end, cudaEventDisableTiming) != cudaSuccess) {
        (void)cudaGetLastError();
        b->ev_end = nullptr;
        hgp_batch_destroy(b);
        return HGP_ERR_CUDA;
    }
    const int rc = build_groups(b, 8);
    if (rc != HGP_OK) {
        hgp_batch_destroy(b);
        return rc;
    }
    *out = b;
    return HGP_OK;
}

int hgp_batch_refine(hgp_batch *b, int32_t rounds, hgp_round_stats *stats)
{
    if (!b || rounds < 0) return HGP_ERR_INVALID;
    if (rounds == 0) return HGP_OK;
    for (hgp_handle *h : b->hs)
        if (h->next_round + rounds >= ((int64_t)1 << 30)) return HGP_ERR_UNSUPPORTED;
    // the batch reads the handles' state on its own stream: after their streams' pending work,
    // and after the last call of another batch that refined them (on another stream)
    for (size_t i = 0; i < b->member_streams.size(); ++i) {
        cudaError_t e = cudaEventRecord(b->events[i], b->member_streams[i]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->events[i], 0);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return status_of(e);
        }
    }
    for (hgp_handle *h : b->hs) {
        if (!h->after_batch) continue;
        const cudaError_t e = cudaStreamWaitEvent(b->stream, h->ev_batch, 0);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return status_of(e);
        }
    }
    if (rounds > b->stats_cap) {
        int32_t cap = b->stats_cap;
        while (cap < rounds) cap *= 2;
        const int rc = build_groups(b, cap);
        if (rc != HGP_OK) return rc;
    }
    cudaError_t e = cudaSuccess;
    if (b->use_graph) {
        if (!b->exec || b->graph_rounds != rounds) {
            if (b->exec) {
                cudaGraphExecDestroy(b->exec);
                b->exec = nullptr;
            }
            int64_t scratch = 0;
            cudaGraph_t graph = nullptr;
            e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                const cudaError_t e2 = enqueue_batch(b, rounds, &scratch);
                e = cudaStreamEndCapture(b->stream, &graph);
                if (e2 != cudaSuccess) e = e2;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, graph, 0);
            if (graph) cudaGraphDestroy(graph);
            if (e == cudaSuccess) {
                b->graph_rounds = rounds;
                b->graph_launches = scratch;
            }
        }
        if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, b->stream);
        if (e == cudaSuccess) b->launches += b->graph_launches;
    } else {
        e = enqueue_batch(b, rounds, &b->launches);
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    for (hgp_handle *h : b->hs) {
        h->next_round += rounds;
        h->all_eligible = false;
    }
    b->last_rounds = rounds;
    e = cudaEventRecord(b->ev_end, b->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    // later work on the members' own streams (read-backs, releases) must come after this call:
    // the call's end is recorded on each such member's event, which its next entry point waits on
    for (hgp_handle *h : b->hs) {
        if (h->stream == b->stream) continue;
        e = cudaEventRecord(h->ev_batch, b->stream);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return status_of(e);
        }
        h->after_batch = true;
    }
    if (stats) return batch_stats_out(b, rounds, stats);
    return HGP_OK;
}

int hgp_batch_get_stats(hgp_batch *b, int32_t rounds, hgp_round_stats *stats)
{
    if (!b || !stats || rounds < 1 || rounds != b->last_rounds) return HGP_ERR_INVALID;
    // waits for the last call only, not for work queued on the batch's stream after it (the
    // next tick of a pipelined caller): the copy runs on a private stream after ev_end
    cudaError_t e = cudaSuccess;
    if (!b->aux) {
        e = cudaStreamCreateWithFlags(&b->aux, cudaStreamNonBlocking);
        if (e != cudaSuccess) b->aux = nullptr;
    }
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->aux, b->ev_end, 0);
    if (e == cudaSuccess) {
        const int32_t count = (int32_t)b->hs.size();
        e = cudaMemcpyAsync(b->h_stats, b->d_stats, sizeof(int64_t) * ST_N * (size_t)b->stats_cap * count,
                            cudaMemcpyDeviceToHost, b->aux);
    }
    if (e == cudaSuccess) e = stream_wait(b->aux);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return batch_stats_unpack(b, rounds, stats);
}

static std::mutex g_stage_mu;       // page-locked staging of hgp_batch_get_partitions
static void *g_stage = nullptr;
static size_t g_stage_cap = 0;

int hgp_batch_get_partitions(hgp_batch *b, const int32_t *members, int32_t count, int32_t *out)
{
    if (!b || count < 0 || (count > 0 && (!members || !out))) return HGP_ERR_INVALID;
    int64_t total = 0;
    for (int32_t i = 0; i < count; ++i) {
        if (members[i] < 0 || members[i] >= (int32_t)b->hs.size()) return HGP_ERR_INVALID;
        total += b->hs[members[i]]->d.n;
    }
    if (total == 0) return HGP_OK;
    // after the batch's last call only (work queued on its stream later is not waited for)
    cudaError_t e = cudaSuccess;
    if (!b->aux) {
        e = cudaStreamCreateWithFlags(&b->aux, cudaStreamNonBlocking);
        if (e != cudaSuccess) b->aux = nullptr;
    }
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->aux, b->ev_end, 0);
    uint8_t *stage = nullptr;
    if (e == cudaSuccess) e = dev_alloc(reinterpret_cast<void **>(&stage), (size_t)total, b->aux);
    int64_t off = 0;
    for (int32_t i = 0; i < count && e == cudaSuccess;) {
        GatherArgs g;
        int64_t most = 0;
        int32_t rows = 0;
        for (; rows < kGather && i < count; ++rows, ++i) {
            const Dev &d = b->hs[members[i]]->d;
            g.part[rows] = d.part;
            g.off[rows] = off;
            off += d.n;
            most = std::max<int64_t>(most, d.n);
        }
        g.off[rows] = off;
        const dim3 grid((unsigned)std::min<int64_t>((most + 1023) / 1024, 152), (unsigned)rows);
        k_part_gather<<<grid, 256, 0, b->aux>>>(g, stage);
        e = cudaGetLastError();
        b->launches++;
    }
    // through a page-locked staging buffer of the library (grown when needed), so the copy runs
    // at the link's rate whatever memory `out` is; the bytes are widened on the way out of it
    const size_t bytes = (size_t)total;
    std::lock_guard<std::mutex> lk(g_stage_mu);
    if (e == cudaSuccess && g_stage_cap < bytes) {
        if (g_stage) cudaFreeHost(g_stage);
        g_stage = nullptr;
        g_stage_cap = 0;
        const size_t cap = std::max(bytes, (size_t)16 << 20);
        e = cudaMallocHost(&g_stage, cap);
        if (e == cudaSuccess) g_stage_cap = cap;
        else g_stage = nullptr;
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(g_stage, stage, bytes, cudaMemcpyDeviceToHost, b->aux);
    if (stage) dev_free(stage, b->aux);
    if (e == cudaSuccess) e = stream_wait(b->aux);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    const uint8_t *from = static_cast<const uint8_t *>(g_stage);
    for (int64_t v = 0; v < total; ++v) out[v] = from[v];
    return HGP_OK;
}

int hgp_batch_query(hgp_batch *b, int32_t *done)
{
    if (!b || !done) return HGP_ERR_INVALID;
    const cudaError_t e = cudaEventQuery(b->ev_end);
    if (e == cudaErrorNotReady) {
        (void)cudaGetLastError();
        *done = 0;
        return HGP_OK;
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    *done = 1;
    return HGP_OK;
}

int hgp_batch_synchronize(hgp_batch *b)
{
    if (!b) return HGP_ERR_INVALID;
    const cudaError_t e = stream_wait(b->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return status_of(e);
    }
    return HGP_OK;
}

int hgp_batch_get_launch_count(hgp_batch *b, int64_t *out)
{
    if (!b || !out) return HGP_ERR_INVALID;
    *out = b->launches;
    return HGP_OK;
}

void hgp_batch_destroy(hgp_batch *b)
{
    if (!b) return;
    free_groups(b);   // touches no member handle: members may already be destroyed
    dev_free(b->d_stats, b->stream);
    free(b->h_stats);
    for (cudaEvent_t ev : b->events) cudaEventDestroy(ev);
    if (b->ev_end) cudaEventDestroy(b->ev_end);
    if (b->aux) cudaStreamDestroy(b->aux);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    (void)cudaGetLastError();
    delete b;
}

int hgp_set_profiling(hgp_handle *h, int32_t enable)
{
    if (!h) return HGP_ERR_INVALID;
    h->profiling = enable != 0;
    h->events_used = 0;
    for (int i = 0; i < HGP_PHASES; ++i) {
        h->prof_ms[i] = 0.0;
        h->prof_launches[i] = 0;
    }
    return HGP_OK;
}

int hgp_get_profile(hgp_handle *h, hgp_profile *out)
{
    if (!h || !out) return HGP_ERR_INVALID;
    for (int i = 0; i < HGP_PHASES; ++i) {
        out->ms[i] = h->prof_ms[i];
        out->launches[i] = h->prof_launches[i];
    }
    return HGP_OK;
}

int hgp_get_launch_count(hgp_handle *h, int64_t *out)
{
    if (!h || !out) return HGP_ERR_INVALID;
    *out = h->launches;
    return HGP_OK;
}

}  // extern "C"
