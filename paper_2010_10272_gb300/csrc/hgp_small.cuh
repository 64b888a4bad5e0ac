// A whole refine call of a small instance in one launch (included by hgp_refine.cu, inside its
// anonymous namespace).
//
// A round of a few ten thousand vertices is bound by the latency of its launches and of the
// dependent loads in each: 22 launches of 5-11 us for 2,500 moves.  Here one thread-block cluster
// (16 CTAs of 16 warps) runs all rounds, with cluster barriers between the phases, and what passes
// between the launches of the general path stays on the chip:
//   * a warp owns a contiguous range of vertices, hashes its sub-rounds once per round, and keeps
//     its candidates in shared memory between the gain and the apply step;
//   * the vertices' blocks, weights and list offsets are kept in shared memory, and the lists
//     where they fit: a cluster barrier drops the L1 lines, so each of them would cost an L2 round
//     trip in every phase (10k vertices 255 -> 239 us a call, 30k 381 -> 373 us);
//   * block weights are a copy per CTA, updated through distributed shared memory;
//   * the approval is a radix select on the key (gain desc, id asc): the candidates' weights are
//     summed per target block and key digit in the shared memory of the block's home CTA, and the
//     first key whose inclusive weight prefix exceeds the block's room is found digit by digit.
//     Only the first digit (summed by the gain step) is needed while every candidate fits.
// The records and pin counts live in global memory as in the general path; another SM's updates
// are read from L2 (RecIO<..>::load_full<true>, atomics), ordered by the cluster barriers.
//
// 10k vertices (k = 2, 60k pins, 5 rounds), new partition and read-back included: 777 -> 239 us a call.

constexpr int kSmWarps = 16;
constexpr int kSmThreads = 32 * kSmWarps;
constexpr int kSmCtas = 16;                          // cluster size (above 8: opt-in)
constexpr int kSmDigit = 9;                          // key bits per digit
constexpr int kSmBins = 1 << kSmDigit;
constexpr int kSmRow = kSmBins + kSmBins / 16;       // padded: a lane sums 16 consecutive bins
constexpr int kSmIdBits = 2 * kSmDigit;
constexpr int32_t kSmMaxN = 1 << kSmIdBits;
// Instances that run this way.  Its time grows with the pins (16 SMs), that of the launches hardly
// does at this size.  5 rounds, planted, k = 4: 264 / 344 / 469 us at 90 / 180 / 360 thousand pins
// against 522-526 us; power-law, k = 16: 360 / 470 / 632 us at 91 / 185 / 369 thousand against
// 659-686 us; k = 64, 64-bit masks: 412 / 520 / 704 us at 87 / 178 / 358 thousand against 706-736 us.
constexpr int32_t kSmallVertices = 1 << 17;
constexpr int32_t kSmallPins = 7 << 16, kSmallPinsWide = 11 << 15;   // 459k for k <= 32, 360k for k > 32
constexpr int kSmPerHome = (64 + kSmCtas - 1) / kSmCtas;
static_assert(kSmallVertices <= kSmMaxN, "ids of two digits");

// dynamic shared memory: per warp the vertices' sub-rounds, a sub-round's list and its candidates
__host__ __device__ inline int small_per_warp(int32_t n)
{
    const int32_t v = (n + kSmCtas * kSmWarps - 1) / (kSmCtas * kSmWarps);
    return (v + 7) / 8 * 8;
}
// and, with `cached`, their list offsets, blocks, and weights c and W where they are not one
__host__ __device__ inline int small_warp_bytes(int per_warp, bool cached, bool vw, bool nw)
{
    return per_warp * (8 + 2 + 1) + (cached ? (per_warp + 2) * 4 + per_warp * (1 + 4 * vw + 4 * nw) : 0) + 7 & ~7;
}
constexpr int kSmMaxBytes = 226 << 10;   // dynamic shared memory of a CTA
// lists are copied only where all fit and this leaves enough L1 for the rest (with the copy filling
// all of it, 60k vertices and k = 64 took 843 us instead of 704)
constexpr int kSmListBytes = 150 << 10;

struct SmallShared {
    unsigned long long row[kSmPerHome][kSmRow];   // home CTA: weight per key digit of a block
    long long rem[kSmPerHome];                    // home CTA: budget left at the digit
    unsigned long long key[64];                   // per block: first key not approved (pass done), or
                                                  // the key prefix found so far
    int32_t open[64];                             // per block: 1 while its key is being resolved
    int64_t bw[64];                               // block weights
    unsigned long long dbw[64];                   // this CTA's changes to them
    unsigned long long sum[6];                    // CTA 0: the round's counters (ST_* order)
    GainWarp g[kSmWarps];
    ApplyWarp aw[kSmWarps];
    int32_t qu[kSmWarps][64];                     // moves that wait for a full warp, as MoveQueue
    uint16_t qat[kSmWarps][64];
};

// a lane's share of a candidate: gain, and the vertex's offset in the warp's range, source and
// target block
struct SmallCand {
    int32_t g;
    uint32_t uat;   // offset << 12 | source << 6 | target
};

// A candidate's key: the gain's nd digits, inverted so that larger gains come first, then the id's two.  Pass
// p of the approval takes its p-th digit from the top.
__device__ __forceinline__ unsigned long long small_key(int32_t g, int32_t u, int nd)
{
    const unsigned long long inv = ((1ull << (kSmDigit * nd)) - 1) - (unsigned long long)(uint32_t)g;
    return (inv << kSmIdBits) | (unsigned long long)(uint32_t)u;
}

template <typename T>
__device__ __forceinline__ T *in_cta(T *p, unsigned rank)
{
    uint64_t out;
    asm("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
    return reinterpret_cast<T *>(out);
}

// every thread of the cluster; orders their shared and global accesses before and after it
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Adds each lane's weight (ok lanes) to bin `digit` of its block's row in the home CTA, one update per
// distinct bin of the warp.
__device__ __forceinline__ void small_count(SmallShared &sh, bool ok, int t, int digit, int32_t cu)
{
    const unsigned mask = __ballot_sync(kFull, ok);
    if (!ok) return;
    const unsigned peers = __match_any_sync(mask, t * kSmBins + digit);
    const unsigned long long sum = (unsigned long long)__reduce_add_sync(peers, (uint32_t)cu & 0xFFFFu) +
                                   ((unsigned long long)__reduce_add_sync(peers, (uint32_t)cu >> 16) << 16);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1)
        atomicAdd(in_cta(&sh.row[t / kSmCtas][digit + digit / 16], t % kSmCtas), sum);
}

// Home CTA, a warp per block: pass 0 decides whether every candidate fits; otherwise, and in the later
// passes of an open block, the digit at which the prefix first exceeds the budget.  The outcome
// goes to every CTA; the row is cleared.
__device__ __forceinline__ void small_select(SmallShared &sh, const Dev &d, unsigned rank, int pass, int passes)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int q = wid, t = q * kSmCtas + (int)rank;
    if (q >= kSmPerHome || t >= d.k) return;
    if (pass > 0 && !sh.open[t]) return;
    unsigned long long *row = sh.row[q] + lane * 17;
    unsigned long long v[16], part = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        v[i] = row[i];
        part += v[i];
    }
    unsigned long long incl = part;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const long long budget = pass == 0 ? (long long)d.lmax - sh.bw[t] : sh.rem[q];
    const unsigned over = __ballot_sync(kFull, (long long)incl > budget);
    const unsigned any = __ballot_sync(kFull, part != 0);
    unsigned long long key = ~0ull;
    int open = 0;
    // an overloaded block has no candidates (no room), so a budget below zero never meets a weight
    if (any && over) {
        const int src = __ffs(over) - 1;
        int digit = 0;
        unsigned long long before = incl - part;
        if (lane == src) {
            bool found = false;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (!found && (long long)(before + v[i]) > budget) {
                    digit = lane * 16 + i;
                    found = true;
                }
                if (!found) before += v[i];
            }
        }
        digit = __shfl_sync(kFull, digit, src);
        before = __shfl_sync(kFull, before, src);
        key = ((pass == 0 ? 0ull : sh.key[t]) << kSmDigit) | (unsigned long long)digit;
        open = pass < passes - 1;
        __syncwarp();
        if (lane == 0) sh.rem[q] = budget - (long long)before;
    }
    if (any) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (v[i]) row[i] = 0;
    }
    if (lane < kSmCtas) {
        *in_cta(&sh.key[t], lane) = key;
        *in_cta(&sh.open[t], lane) = open;
    }
}

template <typename Rec>
__global__ void __launch_bounds__(kSmThreads, 1) k_small(const Dev d, int32_t rounds, int32_t nd, bool cached, int32_t inc_room)
{
    extern __shared__ __align__(16) unsigned char small_dyn[];
    SmallShared &sh = *reinterpret_cast<SmallShared *>(small_dyn);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned rank = blockIdx.x;   // one cluster: the CTA's rank in it
    const int per_warp = small_per_warp(d.n);
    const int warp_bytes = small_warp_bytes(per_warp, cached, d.vw != nullptr, d.nw != nullptr);
    unsigned char *mine = small_dyn + sizeof(SmallShared) + wid * warp_bytes;
    SmallCand *cand = reinterpret_cast<SmallCand *>(mine);
    // per_warp is a multiple of 8, so every array is aligned
    int32_t *offs = reinterpret_cast<int32_t *>(mine + per_warp * 8);            // [per_warp + 2] if cached
    unsigned char *rest = mine + per_warp * 8 + (cached ? (per_warp + 2) * 4 : 0);
    int32_t *vws = reinterpret_cast<int32_t *>(rest);                            // [per_warp] if cached, weighted
    rest += cached && d.vw ? per_warp * 4 : 0;
    int32_t *vnws = reinterpret_cast<int32_t *>(rest);                           // the same
    rest += cached && d.nw ? per_warp * 4 : 0;
    uint16_t *list = reinterpret_cast<uint16_t *>(rest);
    uint8_t *sub = rest + per_warp * 2;
    uint8_t *blocks = rest + per_warp * 3;                                       // [per_warp] if cached
    int32_t *incs = reinterpret_cast<int32_t *>(small_dyn + sizeof(SmallShared) + kSmWarps * warp_bytes);   // [inc_room]
    int32_t *qu = sh.qu[wid];
    uint16_t *qat = sh.qat[wid];
    const int32_t v0 = ((int32_t)rank * kSmWarps + wid) * per_warp;
    const int32_t nv = max(0, min(per_warp, d.n - v0));
    const int32_t c0 = min(d.n, (int32_t)rank * kSmWarps * per_warp), c1 = min(d.n, c0 + kSmWarps * per_warp);
    const int passes = nd + 2;
    const bool unit = d.nw == nullptr;
    const int32_t S = d.S;
    const bool pow2 = (S & (S - 1)) == 0;
    GainInst gi;
    const int32_t r0 = d.rs[0], started = d.rs[1];
    for (int i = tid; i < kSmPerHome * kSmRow; i += kSmThreads) (&sh.row[0][0])[i] = 0;
    if (tid < 64) {
        sh.bw[tid] = tid < d.k ? d.bw[tid] : 0;
        sh.dbw[tid] = 0;
        sh.key[tid] = ~0ull;
        sh.open[tid] = 0;
    }
    if (tid < 6) sh.sum[tid] = 0;
    // the CTA's lists from the first on, and the warp's vertices
    const int32_t inc0 = d.vtx_off[c0], inc_n = min(inc_room, d.vtx_off[c1] - inc0);
    for (int32_t i = tid; i < inc_n; i += kSmThreads) incs[i] = __ldg(&d.inc[inc0 + i]);
    const int32_t *vtx = d.vtx_off, *inc = d.inc;   // indexed by vertex / incidence, wherever they are
    if (cached) {
        for (int32_t i = lane; i < nv; i += 32) {
            blocks[i] = d.part[v0 + i];
            if (d.vw) vws[i] = d.vw[v0 + i];
            if (!unit) vnws[i] = d.vnw[v0 + i];
        }
        for (int32_t i = lane; i <= nv; i += 32) offs[i] = nv ? d.vtx_off[v0 + i] : 0;
        __syncwarp();
        vtx = offs - v0;
        if (nv && offs[nv] - inc0 <= inc_n) inc = incs - inc0;
    }
    long long obj = rank == 0 && tid == 0 ? *d.obj : 0;
    cluster_sync();
    for (int32_t rr = 0; rr < rounds; ++rr) {
        const int32_t r = r0 + rr;
        gi.r = r;
        gi.all_elig = started == 0 && rr == 0;
        for (int32_t i = lane; i < nv; i += 32) {
            const uint64_t z = splitmix64_output(d.seed ^ (((uint64_t)(uint32_t)r << 32) | (uint32_t)(v0 + i)));
            sub[i] = (uint8_t)(pow2 ? (int)(z & (uint64_t)(S - 1)) : (int)(z % (uint64_t)S));
        }
        __syncwarp();
        long long dobj = 0;
        int32_t nelig = 0, ncand_r = 0, nappr = 0, npins = 0, nshared = 0;
        for (int32_t s = 0; s < S; ++s) {
            // ---- gain: this warp's vertices of the sub-round, 32 at a time
            int32_t cnt = 0;
            for (int32_t i0 = 0; i0 < nv; i0 += 32) {
                const bool on = i0 + lane < nv && sub[i0 + lane] == (uint8_t)s;
                const unsigned m = __ballot_sync(kFull, on);
                if (on) list[cnt + __popc(m & lanemask_lt())] = (uint16_t)(i0 + lane);
                cnt += __popc(m);
            }
            room_tables(d, sh.bw, sh.g[wid]);
            int32_t ncand = 0;
            for (int32_t c0 = 0; c0 < cnt; c0 += 32) {
                const bool valid = c0 + lane < cnt;
                int32_t ul = 0, cu = 1, jb = 0, je = 0, a = 0, W = 0;
                if (valid) {
                    ul = list[c0 + lane];
                    const int32_t u = v0 + ul;
                    a = cached ? blocks[ul] : d.part[u];   // only this warp reads or changes it here
                    cu = d.vw ? (cached ? vws[ul] : d.vw[u]) : 1;
                    jb = vtx[u];
                    je = vtx[u + 1];
                    W = unit ? je - jb : (cached ? vnws[ul] : d.vnw[u]);
                }
                int t_best;
                int32_t g_best;
                const bool elig = gain_vertex<Rec, false, true>(d, inc, sh.g[wid], gi, RbArgs{0, 0, 0, 1}, valid, a, cu, jb, je, W,
                                                                t_best, g_best);
                nelig += elig;
                const unsigned cm = __ballot_sync(kFull, t_best >= 0);
                if (t_best >= 0) {
                    SmallCand &c = cand[ncand + __popc(cm & lanemask_lt())];
                    c.g = g_best;
                    c.uat = ((uint32_t)ul << 12) | ((uint32_t)a << 6) | (uint32_t)t_best;
                }
                ncand += __popc(cm);
                const int digit = (int)(small_key(g_best, 0, nd) >> (kSmDigit * (passes - 1))) & (kSmBins - 1);
                small_count(sh, t_best >= 0, t_best, digit, cu);
            }
            __syncwarp();
            ncand_r += ncand;
            cluster_sync();
            // ---- approval
            small_select(sh, d, rank, 0, passes);
            cluster_sync();
            for (int pass = 1; pass < passes; ++pass) {
                if (!__any_sync(kFull, sh.open[lane] | sh.open[lane + 32])) break;   // the same in every warp
                const int shift = kSmDigit * (passes - 1 - pass);
                for (int32_t c0 = 0; c0 < ncand; c0 += 32) {
                    bool in = false;
                    int t = 0, digit = 0;
                    int32_t cu = 1;
                    if (c0 + lane < ncand) {
                        const SmallCand c = cand[c0 + lane];
                        t = c.uat & 63;
                        const int32_t u = v0 + (int32_t)(c.uat >> 12);
                        const unsigned long long key = small_key(c.g, u, nd);
                        in = sh.open[t] && (key >> (shift + kSmDigit)) == sh.key[t];
                        digit = (int)(key >> shift) & (kSmBins - 1);
                        if (in && d.vw) cu = cached ? vws[c.uat >> 12] : d.vw[u];
                    }
                    small_count(sh, in, t, digit, cu);
                }
                cluster_sync();
                small_select(sh, d, rank, pass, passes);
                cluster_sync();
            }
            // ---- apply: this warp's approved candidates
            int32_t queued = 0;
            for (int32_t c0 = 0; c0 < ncand; c0 += 32) {
                bool appr = false;
                int a = 0, t = 0;
                int32_t u = 0;
                if (c0 + lane < ncand) {
                    const SmallCand c = cand[c0 + lane];
                    t = c.uat & 63;
                    a = (c.uat >> 6) & 63;
                    u = v0 + (int32_t)(c.uat >> 12);
                    appr = small_key(c.g, u, nd) < sh.key[t];
                }
                const unsigned am = __ballot_sync(kFull, appr);
                if (appr) {
                    d.part[u] = (uint8_t)t;
                    if (cached) blocks[u - v0] = (uint8_t)t;
                    const unsigned long long cw = d.vw ? (unsigned long long)(cached ? vws[u - v0] : d.vw[u]) : 1ull;
                    atomicAdd(&sh.dbw[a], (unsigned long long)(-(long long)cw));
                    atomicAdd(&sh.dbw[t], cw);
                    ++nappr;
                    const int pos = queued + __popc(am & lanemask_lt());
                    qu[pos] = u;
                    qat[pos] = (uint16_t)(a | (t << 8));
                }
                queued += __popc(am);
                __syncwarp();
                if (queued >= 32) {
                    apply_queue<Rec, KEY_T>(d, vtx, inc, qu, qat, 0, queued, r, sh.aw[wid], dobj, npins, nshared);
                    int32_t u2 = 0;
                    uint16_t at2 = 0;
                    if (32 + lane < queued) {
                        u2 = qu[32 + lane];
                        at2 = qat[32 + lane];
                    }
                    __syncwarp();
                    qu[lane] = u2;
                    qat[lane] = at2;
                    queued -= 32;
                    __syncwarp();
                }
            }
            if (queued) apply_queue<Rec, KEY_T>(d, vtx, inc, qu, qat, 0, queued, r, sh.aw[wid], dobj, npins, nshared);
            __syncthreads();
            // this CTA's block weight changes into every CTA's copy
            for (int i = tid; i < 64 * kSmCtas; i += kSmThreads) {
                const unsigned long long v = sh.dbw[i & 63];
                if (v) atomicAdd(reinterpret_cast<unsigned long long *>(in_cta(&sh.bw[i & 63], i >> 6)), v);
            }
            if (s + 1 == S) {   // the round's counters to CTA 0
                for (int o = 16; o; o >>= 1) {
                    dobj += __shfl_xor_sync(kFull, dobj, o);
                    nelig += __shfl_xor_sync(kFull, nelig, o);
                    nappr += __shfl_xor_sync(kFull, nappr, o);
                    npins += __shfl_xor_sync(kFull, npins, o);
                }
                if (lane < 5) {
                    const unsigned long long v = lane == ST_OBJ    ? (unsigned long long)dobj
                                                 : lane == ST_CAND ? (unsigned long long)ncand_r
                                                 : lane == ST_APPR ? (unsigned long long)nappr
                                                 : lane == ST_ELIG ? (unsigned long long)nelig
                                                                   : (unsigned long long)npins;
                    if (v) atomicAdd(in_cta(&sh.sum[lane], 0), v);
                }
            }
            cluster_sync();
            if (tid < 64) sh.dbw[tid] = 0;   // used again after the next sub-round's barriers
        }
        if (rank == 0 && wid == 0) {
            long long mx = max((long long)sh.bw[lane], (long long)sh.bw[lane + 32]);
            for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(kFull, mx, o));
            if (lane == 0) {
                int64_t *row = d.stats + (int64_t)rr * ST_N;
                obj += (long long)sh.sum[ST_OBJ];
                row[ST_OBJ] = obj;
                row[ST_CAND] = (int64_t)sh.sum[ST_CAND];
                row[ST_APPR] = (int64_t)sh.sum[ST_APPR];
                row[ST_ELIG] = (int64_t)sh.sum[ST_ELIG];
                row[ST_MAXW] = mx;
                row[ST_MOVED] = (int64_t)sh.sum[4];
                row[ST_REV] = 0;
                for (int i = 0; i < 6; ++i) sh.sum[i] = 0;   // added to again after later barriers
            }
        }
    }
    if (rank == 0) {
        if (tid < d.k) d.bw[tid] = sh.bw[tid];
        if (tid == 0) {
            *d.obj = obj;
            d.rs[0] = r0 + rounds;
            d.rs[1] = 1;
        }
    }
    cluster_sync();   // no CTA leaves while others may still reach into its shared memory
}

// launch of k_small: one cluster.  cached / inc_room: what its shared memory has room for.
inline cudaLaunchConfig_t small_config(const Dev &d, cudaStream_t st, cudaLaunchAttribute *at, bool &cached, int32_t &inc_room)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kSmCtas);
    cfg.blockDim = dim3(kSmThreads);
    const int per_warp = small_per_warp(d.n);
    auto bytes = [&](bool c) {
        return (int)sizeof(SmallShared) + kSmWarps * small_warp_bytes(per_warp, c, d.vw != nullptr, d.nw != nullptr);
    };
    cached = bytes(true) <= kSmMaxBytes;
    // the lists of a CTA's vertices, twice their average
    const int64_t want = 2 * ((int64_t)d.P / kSmCtas + 256);
    inc_room = cached && bytes(true) + 4 * want <= kSmListBytes ? (int32_t)want : 0;
    cfg.dynamicSmemBytes = (size_t)bytes(cached) + 4 * (size_t)inc_room;
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = kSmCtas;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}
