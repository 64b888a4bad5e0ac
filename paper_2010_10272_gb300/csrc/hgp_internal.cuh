// Internal device-side layout of libhgp.  Not part of the public ABI (include/hgp.h).
//
// HBM layout of one handle (n vertices, m nets, P pins, k blocks):
//   net_off[m+1], pins[P]        net -> pins CSR, int32 (Sec. 2 / Sec. 3.2 adjacency arrays)
//   vtx_off[n+1], inc[P]         vertex -> incident nets CSR I(v), int32 (bit 31: wide net)
//   vw[n]                        vertex weights c(v) (absent for unit weights)
//   part[n]                      Pi as uint8 (k <= 64)
//   phi                          Phi(e, i), row-major [m][k], entries of 1, 2 or 4 bytes packed
//                                into 32-bit words (in internal net order without the tiny
//                                nets, see Dev::tiny); nets larger than the entry can count keep
//                                int32 rows in phi_wide[n_wide][k] (Sec. 5.1 pin-count table)
//   rec[m]                       per-net hot record read by the gain step: Lambda(e) bitset,
//                                S1(e) = {i : Phi(e,i) = 1} bitset, omega(e), move stamp
//   bw[k], obj                   block weights c(V_i) and the (lambda-1) objective, int64
// plus per-sub-round scratch (candidate slots, approval histograms, tie prefix sums).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "hgp.h"

namespace hgp {

constexpr int kSeg = 32;                 // list entries of a segment: one per lane
constexpr int kWarps = 8;                // warps per tile CTA
constexpr int kRvSlotBytes = 32;         // one slot of the revert variant's hash table
constexpr int kWqPerRow = 64;            // work counters per stats row: the gain step's, one per sub-round
constexpr int kThreads = 32 * kWarps;
// consecutive vertices whose sub-round lists are built together.  A warp takes a list 32 entries
// (a segment) at a time: the longer the list, the fewer of its segments are partly empty (with
// S = 4, 512 +- 20 entries of 2048 vertices; of 256 vertices it was 64 +- 7, so that every second
// list had a third segment of a few entries)
constexpr int kTile = 2048;
constexpr int kMaxSeg = kTile / kSeg;
constexpr int kBins = 4096;              // approval histogram bins (gains 1..4094 exact)
constexpr int kNever = -2;               // move-stamp round meaning "never moved"
constexpr uint32_t kWideFlag = 0x80000000u;
// inc[] entries carry the net id in bits 0..30 and, in bit 31, whether the net's Phi row lives
// in the wide table (so the apply step knows it without reading the net's record first)
constexpr int32_t kNetMask = 0x7fffffff;

// Per-net record for k <= 32, 16 bytes (two per 32-byte sector).  S1 and Lambda are neighbours, so
// that one atomic changes both.
struct __align__(16) Rec16 {
    uint32_t s1;    // bit i set iff Phi(e,i) == 1
    uint32_t lam;   // Lambda(e): bit i set iff Phi(e,i) > 0
    int32_t w;      // omega(e) in bits 0..30, bit 31 = row lives in the wide table
    int32_t mv;     // move stamp: (last round with a pin move) * 2 + (moved in the round before)
};

// Per-net record for k <= 64, 32 bytes (one sector).
struct __align__(32) Rec32 {
    uint64_t s1;
    uint64_t lam;
    int32_t w;
    int32_t mv;
    int32_t pad[2];
};

// Approval state of one target block for the current sub-round.
struct Sel {
    int32_t mode;   // 0: approve every candidate; 1: threshold; 2: threshold inside the
                    //    overflow bin, being resolved digit by digit
    int32_t level;  // next refinement level for mode 2
    int64_t g;      // threshold gain (mode 1) / digit prefix (mode 2)
    int64_t rem;    // weight budget left for candidates with gain == g (mode 1) or with the
                    // current digit prefix (mode 2)
    int64_t cut;    // mode 1: candidates with gain == g are approved up to this vertex id
};

enum { SEL_ALL = 0, SEL_THRESH = 1, SEL_REFINE = 2 };
enum { ST_OBJ = 0, ST_CAND = 1, ST_APPR = 2, ST_ELIG = 3, ST_MAXW = 4, ST_MOVED = 5, ST_REV = 6, ST_N = 7 };
// Dev::acc: block weights, objective, CTAs done
enum { ACC_BW = 0, ACC_OBJ = 64, ACC_DONE = 65, kAccN = 66 };
enum { ERR_INVALID = 1, ERR_UNSUPPORTED = 2, ERR_TABLE = 4 };

// segments per tile: two standard deviations above the mean length of a sub-round's list
inline int32_t segments_of(int32_t S)
{
    const double mean = (double)kTile / S;
    const double len = mean + 2.0 * sqrt(mean * (1.0 - 1.0 / S));
    const int32_t s = (int32_t)((len + kSeg - 1) / kSeg);
    return s < 1 ? 1 : (s > kMaxSeg ? kMaxSeg : s);
}

struct Dev {
    int32_t n, m, k, P;
    int32_t S;
    int32_t phi_w;          // 1, 2 or 4
    int32_t n_tiles;
    int32_t nseg;           // segments per tile and sub-round; the last one takes the list's rest
    int64_t lmax;
    const int32_t *net_off;
    const int32_t *pins;
    const int32_t *vtx_off;
    const int32_t *inc;
    const int32_t *vw;      // nullptr: unit weights
    const int32_t *nw;      // net weights as given (nullptr: unit)
    const int32_t *vnw;     // [n] W(u), the weight of u's nets (nullptr with unit nets: the degree)
    int32_t bins;           // gains lie below this (a multiple of kThreads), or it is kBins
    int32_t pad1;
    uint8_t *part;
    uint32_t *phi;          // a whole number of 8-byte words
    int32_t *phi_wide;
    const int32_t *widx;    // [m] row index in phi_wide (valid where the wide flag is set)
    const int32_t *net_perm;  // [m] internal id of input net e (nullptr: input order kept);
                              // every per-net array above is in internal order
    // Internal order: first net of at most 4, 3, 2, 1 pins (m at least where there are none; input
    // order: INT32_MAX).  Such a net has no Phi row: Lambda, S1 and the size give its pin counts (a
    // block outside S1 has what is left, or 2 when there are two of them), and a move changes
    // Lambda and S1 by one compare-and-swap.  79% of the power-law instance's nets and 35% of its
    // incidences are tiny: their moves touch one sector instead of three (apply 19.5 -> 16.5 ms per
    // step, initialisation 3.7 -> 2.3 ms), and the handle takes 5 GB less.
    int32_t tiny[4];
    void *rec;              // Rec16[m] (k <= 32) or Rec32[m]
    int64_t *bw;
    int64_t *obj;
    // scratch
    uint16_t *sub_list;     // [n_tiles * kTile] vertex offsets in the tile grouped by sub-round
    uint16_t *sub_start;    // [n_tiles * (S + 1)]
    uint64_t *cand;         // [n_tiles * kTile] (gain << 32 | offset << 8 | target); a segment's
                            // candidates start at slot kSeg * segment of its tile
    int32_t *cand_cnt;      // [n_tiles * nseg]
    unsigned long long *hist;  // [k * kBins]
    Sel *sel;               // [k]
    int64_t *tie;           // [k * n_tiles] weight of the candidates at the threshold gain
    int64_t *stats;         // [rounds * ST_N]
    int32_t *wq;            // [rounds * kWqPerRow] work counters of the gain step (a batch's launches
                            // share one set, passed beside the members' states)
    int32_t *err;
    unsigned long long *acc;  // [kAccN] sums of a state initialisation, zero between them
    uint64_t seed;          // sub-round hash seed
    int32_t variant;        // bit 0: zero-gain balance moves; bit 1: revert negative moves
    int32_t pad0;
    int32_t *rs;            // round state on the device: rs[0] = next round r, rs[1] = 0 while
                            // every vertex is eligible (first round), 1 afterwards
    // revert variant only (nullptr otherwise)
    uint8_t *rv_src;        // [n_tiles * kTile] per candidate slot: block an approved move left,
                            // | 0x80 when it is to be undone; 0xFF when not approved
    void *rv_tab;           // hash table of (net, block) order statistics of the sub-round's moves
    int64_t rv_cap;         // its capacity in slots (a power of two >= 2 P)
    unsigned long long *rv_cnt;  // [2] incidences of the vertices moved in the current sub-round,
                                 // and those of them on nets with several movers
    int32_t *rv_net;        // [m] movers of each net in the current sub-round
};

__device__ __forceinline__ int lam_bits_ctz(uint32_t x) { return __ffs(x) - 1; }
__device__ __forceinline__ int lam_bits_ctz(uint64_t x) { return __ffsll((long long)x) - 1; }
__device__ __forceinline__ int lam_popc(uint32_t x) { return __popc(x); }
__device__ __forceinline__ int lam_popc(uint64_t x) { return __popcll(x); }

// Adds delta (+1 or -1) to Phi(e, i) and returns the value before the update.  Narrow
// entries are updated with one 32-bit atomic on the word that holds them; this is exact
// because every intermediate value of an entry stays in [0, |e|] (decrements of Phi(e,i)
// in one sub-round come from distinct pins that were in block i at its start), so no
// borrow or carry crosses into a neighbouring entry.
__device__ __forceinline__ int32_t phi_add(const Dev &d, int32_t e, int32_t i, int32_t delta,
                                           bool wide, int32_t wrow)
{
    if (wide) return atomicAdd(&d.phi_wide[(int64_t)wrow * d.k + i], delta);
    const int64_t x = (int64_t)e * d.k + i;
    if (d.phi_w == 4) return atomicAdd(reinterpret_cast<int *>(d.phi) + x, delta);
    if (d.phi_w == 2) {
        const uint32_t sh = (uint32_t)(x & 1) * 16u;
        const uint32_t old = atomicAdd(&d.phi[x >> 1], (uint32_t)delta << sh);
        return (int32_t)((old >> sh) & 0xFFFFu);
    }
    const uint32_t sh = (uint32_t)(x & 3) * 8u;
    const uint32_t old = atomicAdd(&d.phi[x >> 2], (uint32_t)delta << sh);
    return (int32_t)((old >> sh) & 0xFFu);
}

// One pin of net e from block a to block t: Phi(e, a)--, Phi(e, t)++, and the values before.  With few
// blocks both entries mostly share an aligned 8-byte word (always up to k = 8 with 1-byte
// entries), which one 64-bit atomic changes; exact for the same reason as above.
__device__ __forceinline__ void phi_move(const Dev &d, int32_t e, int32_t a, int32_t t, bool wide, int32_t wrow,
                                         int32_t &old_a, int32_t &old_t)
{
    if (!wide) {
        const int64_t ba = ((int64_t)e * d.k + a) * d.phi_w, bt = ((int64_t)e * d.k + t) * d.phi_w;
        if ((ba >> 3) == (bt >> 3)) {
            const int sa = (int)(ba & 7) * 8, st = (int)(bt & 7) * 8;
            const unsigned long long old = atomicAdd(reinterpret_cast<unsigned long long *>(d.phi) + (ba >> 3),
                                                     (1ull << st) - (1ull << sa));
            const uint32_t mask = d.phi_w == 1 ? 0xFFu : (d.phi_w == 2 ? 0xFFFFu : 0xFFFFFFFFu);
            old_a = (int32_t)((uint32_t)(old >> sa) & mask);
            old_t = (int32_t)((uint32_t)(old >> st) & mask);
            return;
        }
    }
    old_a = phi_add(d, e, a, -1, wide, wrow);
    old_t = phi_add(d, e, t, +1, wide, wrow);
}

// pins of a tiny net
__device__ __forceinline__ int tiny_size(const Dev &d, int32_t e)
{
    return 4 - (e >= d.tiny[1]) - (e >= d.tiny[2]) - (e >= d.tiny[3]);
}

// pin count of block i of a tiny net of `size` pins
template <typename Lam>
__device__ __forceinline__ int tiny_count(Lam s1, Lam lam, int size, int i)
{
    if (!((lam >> i) & 1)) return 0;
    if ((s1 >> i) & 1) return 1;
    return lam_popc((Lam)(lam & ~s1)) == 2 ? 2 : size - lam_popc(s1);
}

__device__ __forceinline__ int32_t phi_get(const Dev &d, int32_t e, int32_t i, bool wide,
                                           int32_t wrow)
{
    if (e >= d.tiny[0]) {
        if (d.k <= 32) {
            const Rec16 *r = reinterpret_cast<const Rec16 *>(d.rec) + e;
            return tiny_count<uint32_t>(r->s1, r->lam, tiny_size(d, e), i);
        }
        const Rec32 *r = reinterpret_cast<const Rec32 *>(d.rec) + e;
        return tiny_count<uint64_t>(r->s1, r->lam, tiny_size(d, e), i);
    }
    if (wide) return d.phi_wide[(int64_t)wrow * d.k + i];
    const int64_t x = (int64_t)e * d.k + i;
    if (d.phi_w == 4) return reinterpret_cast<const int *>(d.phi)[x];
    if (d.phi_w == 2) return reinterpret_cast<const uint16_t *>(d.phi)[x];
    return reinterpret_cast<const uint8_t *>(d.phi)[x];
}

// Eligibility test of Sec. 6 ("u and its neighbours"): did net e have a pin moved in
// round r-1?  The stamp keeps the last round with a move and whether the round before it
// had one too, so writes during round r do not hide round r-1.
__device__ __forceinline__ bool moved_in_prev_round(int32_t mv, int32_t r)
{
    const int32_t last = mv >> 1;
    return last == r - 1 || (last == r && (mv & 1));
}

__device__ __forceinline__ uint64_t splitmix64_output(uint64_t z)
{
    // SplitMix64 output function (Steele, Lea, Flood, OOPSLA 2014)
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

// ---------------------------------------------------------------- host-side helpers
struct Handle;
cudaError_t launch_scan_i32(const int32_t *in, int32_t *out, int64_t count, int32_t *block_sums,
                            cudaStream_t st);
int64_t scan_scratch_elems(int64_t count);

}  // namespace hgp
