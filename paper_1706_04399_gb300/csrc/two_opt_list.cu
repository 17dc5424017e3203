// Edge exchange of Sec. 3.2.3 (best-improvement 2-opt to 2-optimality) on a
// short list of the best candidate pairs.
//
// Same mathematics and tie order as two_opt_tiled.cu: over the pairs of tour
// positions i, j (i + 2 <= j, not (0, n-1)),
//   delta(i, j) = C[x_i][x_j] + C[x_i+1][x_j+1] - C[x_i][x_i+1] - C[x_j][x_j+1],
// the applied move is the smallest (delta, i, j) with delta < 0.
//
// Why a list.  A pair of tour edges {u, w}, {v, z} can be reconnected in two
// ways, {u,v},{w,z} or {u,z},{w,v}; which one keeps a single tour depends only
// on whether the tour runs through the two edges in the same direction.  A
// move replaces two edges and turns the direction of the edges between them,
// so it changes *which* of the two a pair offers for a large share of all
// pairs, but the two deltas themselves only for the pairs that hold one of
// the two new edges: 2n of n^2/2.  The kernel therefore keeps both
// reconnections of a pair as candidates, whatever the direction now:
//  * Edges live in slots; a move's new edges take over the slots of the two
//    it removes.  pos[slot] holds the edge's tour position and direction,
//    at[position] the slot and direction, so a reversal is a pass over these
//    two uint16 arrays and touches nothing else.
//  * The list holds every candidate with delta < T (packed delta, slots,
//    reconnection).  A pass drops the candidates of the two removed edges,
//    adds those of the two new ones and takes the smallest (delta, i, j)
//    among the candidates whose reconnection fits the present directions.
//    While there is one, it is the best move of the plain scan.
//  * A pair belongs to its longer edge (ties: the larger slot).  low[slot] is
//    a lower bound on the deltas of the slot's own pairs that are not in the
//    list; before anything is known it is -2 C[u][w], since a pair's delta is
//    no smaller than minus its edges (with neighbour lists, below, the cheapest
//    neighbours of u and w are added).  When no candidate fits, T is raised to
//    T' and the slots with low < T' scan their row: candidates in [T, T') go
//    to the list, the smallest delta past T' becomes the slot's low.
//  * T' is the largest, over groups of threads, of the group's smallest low:
//    about G ln G rows for G groups, a few scans per move in all.  From the
//    fifth raise in a row on, every one that brings no move is made with twice
//    as many groups: a tour that is 2-optimal already needs all its rows, and
//    would take some 20 of them at a time (1200 viewpoints, 48 such tours, whole
//    call: 72 raises and 600 us, now 255, of which 190 were an allocation; with
//    doubling from the second raise the first moves of random tours scan too
//    much, 150 tours, one move: 137 -> 766 us).
// Longer tours (kLists) also save on those scans:
//  * Every city has a list of its 32 cheapest neighbours.  A pair that shows in
//    neither list of an edge's two ends costs at least the lists' radii there,
//    so where those keep its delta at or past T' the row's scan reads the two
//    lists (a "short" row: four fifths of them) instead of all n slots.
//  * A new edge's pair costs at least the cheapest neighbours of its two ends.
//    A first pass over len and low picks the slots where that bound lies below
//    T, or below the low of a longer slot; only those pairs are evaluated.
// With T = 0 and no candidate that fits, the tour is 2-optimal.
//
// A list that runs full folds its upper part back into low (T falls).  Where
// more candidates than it holds tie on one delta, so that T cannot rise, passes
// take the best move directly: they look at the edges in tour order, each
// against the later ones, and end with the first that attains the smallest low,
// since of equal deltas the smallest position counts.  The edges before it stay
// without such a pair but for the edges that the move turns round, so the next
// pass looks at those alone there.  T is tried again once such passes have
// looked at eight times the edges that a trial scans.  Costs of 1 and 2, whole
// call: 300 viewpoints, 1024 tours 12.4 ms when every pass scanned every row,
// 2.6 so; 700 viewpoints, 300 tours 69 and 9.0; 1500 viewpoints, 48 tours 303
// and 45.
//
// What bounds it: for long tours the gathers of the rows that are scanned in
// full (the cost rows of the edge's two ends, staged interleaved in shared
// memory, so that one 8-byte gather brings both ends' costs to a city) and of
// the new edges' pairs; for short ones the issue slots and the chain of a
// pass, about 9000 cycles at n = 400.  Against scanning every row and every
// pair of the new edges, on GB300: 600 tours at n = 1992 39 -> 26 ms, 150 at
// n = 2999 28 -> 18, 600 at n = 1000 10.1 -> 6.2.
#include <climits>

#include "tiled_common.cuh"

namespace dpso {
namespace {

using namespace tiled;

constexpr int kThreadsPerSm = 640;  // the register budget's resident threads
constexpr int kBig = 1 << 30;  // on a staged row's own city: a pair that shares it never improves
constexpr unsigned long long kDead = ~0ull;  // a dropped list entry

// Entry: delta (32 bits), reconnection (bit 26), slots (13 bits each).
__device__ __forceinline__ unsigned long long pack_entry(int delta, int e, int f, int type) {
    return (static_cast<unsigned long long>(static_cast<uint32_t>(delta)) << 32) |
           static_cast<uint32_t>((type << 26) | (e << 13) | f);
}

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr(smem)), "l"(gmem)
                 : "memory");
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// At most `Pending` of this thread's latest copy groups are still in flight.
template <int Pending>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(Pending) : "memory");
}

// The staged matrix's pitch (FULL; odd, so that a column's cities fall on
// different banks).
__host__ __device__ constexpr int full_ld(int n) { return n | 1; }

// Shared bytes for tours of up to n viewpoints.
__host__ __device__ constexpr size_t list_smem(int n, int bufs, bool full, int cap) {
    const size_t m = (n + 7) / 8 * 8;
    const size_t staged =
        full ? (static_cast<size_t>(n) * full_ld(n) + 3) / 4 * 16 : m * bufs * sizeof(int2);
    return staged + m * (2 * sizeof(unsigned) + 2 * sizeof(int) + 3 * sizeof(uint16_t)) +
           static_cast<size_t>(cap) * sizeof(unsigned long long);
}

// One warp per city: its kNear cheapest neighbours, one per lane in increasing
// (cost, city) order.  A chunk of 32 cities that holds none cheaper than the
// dearest so far is passed over; else it is sorted and merged by a bitonic
// network over the lanes.
__device__ __forceinline__ unsigned long long bitonic_step(unsigned long long v, int xor_lane,
                                                           bool up) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, xor_lane);
    const bool low_lane = (threadIdx.x & xor_lane) == 0;
    return (v < o) == (low_lane == up) ? v : o;
}

__global__ void __launch_bounds__(128) near_kernel(const int* __restrict__ C, int ldc, int n,
                                                   int2* __restrict__ near) {
    const int lane = threadIdx.x & 31, u = (blockIdx.x * 128 + threadIdx.x) >> 5;
    if (u >= n) return;
    const int* row = C + static_cast<size_t>(u) * ldc;
    unsigned long long kept = ~0ull;
    for (int c0 = 0; c0 < n; c0 += 32) {
        const int c = c0 + lane;
        unsigned long long v =
            c < n && c != u ? (static_cast<unsigned long long>(row[c]) << 16) | c : ~0ull;
        if (!__any_sync(0xffffffffu, v < __shfl_sync(0xffffffffu, kept, 31))) continue;
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) v = bitonic_step(v, j, (lane & k) == 0);
        v = min(kept, __shfl_sync(0xffffffffu, v, 31 - lane));  // the 32 smallest, bitonic
#pragma unroll
        for (int j = 16; j > 0; j >>= 1) v = bitonic_step(v, j, true);
        kept = v;
    }
    near[u * kNear + lane] =
        kept == ~0ull ? make_int2(INT_MAX / 2, u == 0 ? 1 : 0)
                      : make_int2(static_cast<int>(kept >> 16), static_cast<int>(kept & 0xffff));
}

// How a launch stages cost rows and shares out the rows of a scan round.
//   kMatrix    the whole matrix in shared memory (few tours per SM: no wait for
//              L2 after the first); every warp scans its own rows
//   kWarpRows  each warp stages and scans its own rows (two buffers per warp)
//   kCtaRows   the CTA scans one row at a time while the next one arrives
//   kGlobal    every warp scans its own rows from C (few tours per SM, where
//              more threads serve a tour than could stage; the longest tours)
enum Staging { kMatrix, kWarpRows, kCtaRows, kGlobal };

__host__ __device__ constexpr int staged_bufs(int threads, Staging st) {
    return st == kWarpRows ? 2 * (threads / 32) : (st == kCtaRows ? 2 : 0);
}

// NT threads solve one tour.
template <int NT, Staging ST>
__global__ void __launch_bounds__(NT, (NT >= 512 ? 1 : kThreadsPerSm / NT))
    two_opt_list_kernel(TwoOptBatch b, int cap) {
    constexpr int kW = NT / 32;                     // warps
    constexpr int kBufs = staged_bufs(NT, ST);      // staged row pairs
    constexpr bool kFull = ST == kMatrix;
    constexpr bool kStages = ST == kWarpRows || ST == kCtaRows;
    constexpr bool kWarpScan = ST != kCtaRows;
    // Neighbour lists and bounds on the new edges' pairs; short tours, whose rows
    // are read in a few steps, are faster without (n = 400, 1024 tours: a swarm's
    // generations 8 % slower with them).
    constexpr bool kLists = ST == kCtaRows || ST == kGlobal;
    // partners a thread has in flight (whole calls, one, two and four of them: 1024
    // tours of 400 3.29, 3.27 and 3.34 ms, 150 of 2999 19.0, 18.0 and 18.2)
    constexpr int kBatch = 2;
    // threads per group of the choice of T' (see the head of the file): eight
    // groups (four, eight and sixteen: 1024 tours of 400 3.22, 3.27 and 3.43 ms,
    // 600 of 1000 6.42, 6.12 and 6.83)
    constexpr int kGroup = NT >= 256 ? 32 : (NT >= 128 ? 16 : 8);
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned long long s_key[2][kW];  // the warps' best, by pass parity
    __shared__ int s_lo[kW], s_hi[kW];
    __shared__ int s_item, s_cnt, s_rows, s_wide, s_drop;
    __shared__ long long s_pf;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m8 = (b.max_n + 7) / 8 * 8;
    int2* const buf0 = reinterpret_cast<int2*>(smraw);
    int* const mat = reinterpret_cast<int*>(smraw);
    unsigned long long* const list = reinterpret_cast<unsigned long long*>(
        smraw + (kFull ? (static_cast<size_t>(b.max_n) * full_ld(b.max_n) + 3) / 4 * 16
                       : kBufs * m8 * sizeof(int2)));
    unsigned* const ends = reinterpret_cast<unsigned*>(list + cap);  // u | w << 16
    int* const len = reinterpret_cast<int*>(ends + m8);              // C[u][w]
    int* const low = len + m8;
    unsigned* const inc = reinterpret_cast<unsigned*>(low + m8);  // city -> its two slots
    uint16_t* const pos = reinterpret_cast<uint16_t*>(inc + m8);  // slot -> position | dir << 15
    uint16_t* const at = pos + m8;                                // position -> slot | dir << 15
    uint16_t* const rows = at + m8;  // slots to scan: short rows from the front, wide from the back

    for (;;) {
        if (tid == 0) s_item = static_cast<int>(atomicAdd(b.queue, 1u));
        __syncthreads();
        const int g = s_item;
        if (g >= b.total) break;
        const int prob = find_inst(b.off, b.nprob, g);
        const TwoOptTask& a = b.tasks[prob];
        const int p = a.order ? a.order[g - b.off[prob]] : g - b.off[prob];
        if (a.gate && *a.gate == 0) {  // this problem does not exchange edges now
            __syncthreads();
            continue;
        }
        const int n = a.n;
        const int* __restrict__ const C = a.C;
        const int ldc = a.ldc;
        const int2* __restrict__ const near = kLists ? a.near : nullptr;
        const int max_moves = a.max_moves;
        const int mld = full_ld(n);
        uint16_t* const tour = a.tours + static_cast<size_t>(p) * a.ldt;

        if (kFull) {
            for (int r = warp; r < n; r += kW)
                for (int c = lane; c < n; c += 32) {
                    if (r == c) mat[r * mld + c] = kBig;
                    else cp_async4(&mat[r * mld + c], C + static_cast<size_t>(r) * ldc + c);
                }
            cp_commit();
        }
        for (int i = tid; i < n; i += NT) {
            const unsigned u = tour[i], w = tour[i + 1 == n ? 0 : i + 1];
            const int d = C[static_cast<size_t>(u) * ldc + w];
            ends[i] = u | (w << 16);
            len[i] = d;
            low[i] = -2 * d + (near ? near[u * kNear].x + near[w * kNear].x : 0);
            inc[u] = i | ((i == 0 ? n - 1 : i - 1) << 16);
            pos[i] = static_cast<uint16_t>(i);
            at[i] = static_cast<uint16_t>(i);
        }
        if (tid == 0) {
            s_cnt = 0;
            s_rows = 0;
            s_drop = INT_MAX;
        }
        long long f = a.cost[p];
        long long scans = 0;  // rows decided: new edges, and rows scanned
        int moves = 0, passes = 0;
        int T = INT_MIN;      // the list holds every candidate with delta < T
        int clean = 0, clean_lo = 0, clean_moves = -2, last_bi = 0, last_bj = 0;  // direct passes
        int direct = 0;       // edges that direct passes may still look at (ties overflow the list)
        int level = 0;        // doublings of the groups that choose T' (after a full list)
        int par = 0;
        const int guard = 1000 + 100 * n;
        if (kFull) cp_wait_all();
        __syncthreads();

        // Stages the cost rows of edge (u, w) interleaved into buffer k, by
        // threads t0, t0 + step, ..: one copy group.
        auto load_rows = [&](int k, int u, int w, int t0, int step) {
            if constexpr (kStages) {
                int2* const buf = buf0 + k * m8;
                const int* ru = C + static_cast<size_t>(u) * ldc;
                const int* rw = C + static_cast<size_t>(w) * ldc;
#pragma unroll 4
                for (int c = t0; c < n; c += step) {
                    cp_async4(&buf[c].x, ru + c);
                    cp_async4(&buf[c].y, rw + c);
                }
                cp_commit();
            }
        };
        // After the thread's copies of the row landed: its own cities' costs
        // are such that a pair sharing a city never improves.
        auto seal_rows = [&](int k, int u, int w, int t0, int step) {
            if constexpr (kStages) {
                if (u % step == t0) buf0[k * m8 + u].x = kBig;
                if (w % step == t0) buf0[k * m8 + w].y = kBig;
            }
        };
        // Costs of city c to the two ends (u, w) of the edge staged in buffer k.
        auto costs = [&](int k, int u, int w, int c) {
            if constexpr (kFull) return make_int2(mat[u * mld + c], mat[w * mld + c]);
            else if constexpr (kStages) return buf0[k * m8 + c];
            else return make_int2(c == u ? kBig : C[static_cast<size_t>(u) * ldc + c],
                                  c == w ? kBig : C[static_cast<size_t>(w) * ldc + c]);
        };
        // C between two cities; a city's cheapest and dearest listed neighbour
        // (0 without the table: no bound, no short rows).
        auto cost = [&](int u, int w) {
            if constexpr (kFull) return mat[u * mld + w];
            else return C[static_cast<size_t>(u) * ldc + w];
        };
        auto nearest = [&](int u) { return near ? near[u * kNear].x : 0; };
        auto farthest = [&](int u) { return near ? near[u * kNear + kNear - 1].x : 0; };
        // The key (delta, i, j) of a candidate whose reconnection fits, else ~0.
        auto key_of = [&](int d, int e, int h, int type) {
            const unsigned pe = pos[e], ph = pos[h];
            const int i = pe & 0x7fff, j = ph & 0x7fff;
            return static_cast<int>((pe ^ ph) >> 15) == type ? pack_key(d, min(i, j), max(i, j))
                                                              : ~0ull;
        };
        // The smallest key among list entries first.. of this thread's share.
        auto list_best = [&](int first, int cnt) {
            unsigned long long best = ~0ull;
            for (int k = first + tid; k < cnt; k += NT) {
                const unsigned long long v = list[k];
                const unsigned lo = static_cast<unsigned>(v);
                if (v != kDead)
                    best = min(best, key_of(static_cast<int>(v >> 32), (lo >> 13) & 0x1fff,
                                            lo & 0x1fff, (lo >> 26) & 1));
            }
            return best;
        };
        // The block's smallest key; one barrier.
        auto block_best = [&](unsigned long long mine) {
            const unsigned hi = static_cast<unsigned>(mine >> 32);
            const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
            const unsigned ml =
                __reduce_min_sync(0xffffffffu, hi == mh ? static_cast<unsigned>(mine) : ~0u);
            if (lane == 0) s_key[par][warp] = (static_cast<unsigned long long>(mh) << 32) | ml;
            __syncthreads();
            unsigned long long best = s_key[par][0];
#pragma unroll
            for (int w = 1; w < kW; ++w) best = min(best, s_key[par][w]);
            par ^= 1;
            return best;
        };
        auto owner = [&](int e, int h) {
            const int de = len[e], dh = len[h];
            return de > dh || (de == dh && e > h) ? e : h;
        };
        auto insert = [&](int d, int e, int h, int type) {
            const int k = atomicAdd(&s_cnt, 1);
            if (k < cap) list[k] = pack_entry(d, e, h, type);
            return k < cap;
        };
        // Warp 0 squeezes dropped entries out of the list's first cnt.
        auto compact = [&](int cnt) {
            if (warp != 0) return;
            int o = 0;
            for (int k0 = 0; k0 < cnt; k0 += 32) {
                const unsigned long long v = k0 + lane < cnt ? list[k0 + lane] : kDead;
                const unsigned keep = __ballot_sync(0xffffffffu, v != kDead);
                if (v != kDead) list[o + __popc(keep & ((1u << lane) - 1))] = v;
                o += __popc(keep);
                __syncwarp();
            }
            __syncwarp();
            if (lane == 0) s_cnt = o;
        };
        // Drops candidates with delta >= te and puts those at or above t back
        // into low.  Called by all threads with the list at rest; ends with a
        // barrier.
        auto fold = [&](int t, int te) {
            const int cnt = min(s_cnt, cap);
            for (int k = tid; k < cnt; k += NT) {
                const unsigned long long v = list[k];
                const int d = static_cast<int>(v >> 32);
                if (v == kDead || (d < t && d < te)) continue;
                const unsigned lo = static_cast<unsigned>(v);
                if (d < te) atomicMin(&low[owner((lo >> 13) & 0x1fff, lo & 0x1fff)], d);
                list[k] = kDead;
            }
            __syncthreads();
            compact(cnt);
            if (tid == 0) s_drop = INT_MAX;
            __syncthreads();
        };

        // The best move over all pairs, which is known to be no better than lo: a
        // warp per tour position i against the later ones, in order, until one
        // attains lo.  Of the positions below `clean` only pairs with a j in
        // [seg_lo, seg_hi] may.  Adds the positions looked at to `looked`.
        auto direct_best = [&](int lo, int clean, int seg_lo, int seg_hi, int& looked) {
            const unsigned bound = static_cast<unsigned>(lo) ^ 0x80000000u;
            unsigned long long found = ~0ull;
            for (int i0 = 0; i0 < n - 2 && static_cast<unsigned>(found >> 32) > bound;) {
                const bool part = i0 < clean;  // (a block's share of these is taken at once)
                const int i1 = part ? min(i0 + 4 * kW, clean) : min(i0 + kW, n - 2);
                unsigned long long mine = ~0ull;
                for (int i = i0 + warp; i < i1; i += kW) {
                    const unsigned ai = at[i], vi = ends[ai & 0x7fff];
                    const int de = len[ai & 0x7fff];
                    const int u = ai >> 15 ? vi >> 16 : vi & 0xffff, w = ai >> 15 ? vi & 0xffff : vi >> 16;
                    const int* const ru = kFull ? mat + u * mld : C + static_cast<size_t>(u) * ldc;
                    const int* const rw = kFull ? mat + w * mld : C + static_cast<size_t>(w) * ldc;
                    const int j0 = part ? max(i + 2, seg_lo) : i + 2;
                    const int j1 = part ? seg_hi + 1 : n;
#pragma unroll 4
                    for (int j = j0 + lane; j < j1; j += 32) {
                        const unsigned aj = at[j], vj = ends[aj & 0x7fff];
                        const int c0 = aj >> 15 ? vj >> 16 : vj & 0xffff;
                        const int c1 = aj >> 15 ? vj & 0xffff : vj >> 16;
                        const int d = ru[c0] + rw[c1] - de - len[aj & 0x7fff];
                        if (d < 0 && (i > 0 || j < n - 1)) mine = min(mine, pack_key(d, i, j));
                    }
                }
                looked += i1 - i0;
                i0 = i1;
                found = min(found, block_best(mine));
            }
            return found;
        };

        unsigned long long best = ~0ull;  // the pass's best move
        for (;;) {
            if (max_moves > 0 && moves >= max_moves) break;
            if (moves >= guard) {
                if (tid == 0 && a.status) atomicExch(a.status, DPSO_ERR_INTERNAL);
                break;
            }
            // No candidate fits: raise T until one does or none is left.
            for (int rounds = 0; best == ~0ull && T < 0; ++rounds) {
                // (a round raises T by at least one; far more rounds than rows
                // would mean one tie after another: look directly)
                if (rounds > 1000 + n) direct = max(direct, 1);
                if (tid == 0) {
                    s_rows = 0;
                    s_wide = 0;
                }
                compact(min(s_cnt, cap));
                int mn = INT_MAX;
#pragma unroll 4
                for (int s = tid; s < n; s += NT) mn = min(mn, low[s]);
                int gm = mn;
                const int group = (kGroup << level) >> min(max(rounds - 3, 0), 5);
                for (int o = 1; o < min(group, 32); o <<= 1)
                    gm = min(gm, __shfl_xor_sync(0xffffffffu, gm, o));
                mn = __reduce_min_sync(0xffffffffu, mn);
                gm = __reduce_max_sync(0xffffffffu, gm == INT_MAX ? INT_MIN : gm);
                if (lane == 0) {
                    s_lo[warp] = mn;
                    s_hi[warp] = gm;
                }
                __syncthreads();
                int lo = s_lo[0], hi = s_hi[0];
#pragma unroll
                for (int w = 1; w < kW; ++w) {
                    lo = min(lo, s_lo[w]);
                    hi = max(hi, s_hi[w]);
                }
                if (lo >= 0) {
                    T = 0;
                    break;
                }
                if (direct > 0) {
                    // (after one move since the last direct pass at this lo, the
                    // positions below that pass's and the move's hold no pair of
                    // lo but with an edge that the move turned or brought in; where
                    // none is found at all, what else those hold counts as well)
                    int looked = 0;
                    for (int c = clean_lo == lo && moves == clean_moves + 1 ? clean : 0;; c = 0) {
                        best = direct_best(lo, c, last_bi, last_bj, looked);
                        if (c == 0 || static_cast<int>(static_cast<uint32_t>(best >> 32) ^ 0x80000000u) == lo)
                            break;
                    }
                    direct -= looked;
                    scans += looked;
                    if (best == ~0ull) T = 0;  // every pair was looked at
                    clean_lo = lo;
                    clean_moves = moves;
                    clean = static_cast<int>(best >> 16) & 0xffff;
                    break;
                }
                const int c0 = s_cnt;
                if (group > (kW > 1 ? 32 : 16)) hi = lo;
                int Tn = min(0, max(hi, lo + 1));
                // Rows to scan.  A short row's pairs all show in the neighbour
                // lists of its two ends: a pair that is in neither costs at
                // least the two radii, so its delta is no less than
                // reach - 2 len.
                auto reach = [&](unsigned ends_e, int len_e) {
                    return min(farthest(ends_e & 0xffff), len_e) + min(farthest(ends_e >> 16), len_e);
                };
                unsigned take = 0;  // bit k: this thread's k-th slot (at most 32)
#pragma unroll 4
                for (int s = tid, k = 0; s < n; s += NT, ++k)
                    take |= static_cast<unsigned>(low[s] < Tn) << k;
                for (; take; take &= take - 1) {
                    const int s = tid + (__ffs(take) - 1) * NT;
                    const bool wide = reach(ends[s], len[s]) - 2 * len[s] < Tn;
                    const int k = atomicAdd(wide ? &s_wide : &s_rows, 1);
                    rows[wide ? n - 1 - k : k] = static_cast<uint16_t>(s);
                    low[s] = INT_MAX;
                }
                __syncthreads();
                const int ns = s_rows, nr = s_wide;
                const uint16_t* const wrows = rows + n - nr;  // (in whatever order)
                // Scans the pairs that edge e (staged in buffer k) owns, over
                // slots t0, t0 + step, ..: candidates in [T, Tn) go to the list,
                // the smallest delta past Tn is returned.
                auto scan = [&](int k, int e, int t0, int step) {
                    const unsigned ve = ends[e];
                    const int eu = ve & 0xffff, ew = ve >> 16, de = len[e];
                    int lbe = INT_MAX;
                    for (int s0 = t0; s0 < n; s0 += kBatch * step) {
                        int d0[kBatch], d1[kBatch], m = INT_MAX;
#pragma unroll
                        for (int q = 0; q < kBatch; ++q) {
                            const int s = min(s0 + q * step, n - 1);
                            const unsigned v = ends[s];
                            const int ds = len[s];
                            const int2 A = costs(k, eu, ew, v & 0xffff);
                            const int2 B = costs(k, eu, ew, v >> 16);
                            // (a longer edge, or an equal one of a larger slot, owns
                            // the pair; past the last slot: nothing)
                            const bool own =
                                ds <= de - (s >= e ? 1 : 0) && s0 + q * step < n;
                            d0[q] = own ? A.x + B.y - de - ds : INT_MAX;
                            d1[q] = own ? B.x + A.y - de - ds : INT_MAX;
                            m = min(m, min(d0[q], d1[q]));
                        }
                        if (m < Tn) {
                            m = INT_MAX;
#pragma unroll
                            for (int q = 0; q < kBatch; ++q) {
                                const int s = s0 + q * step;
                                if (d0[q] >= T && d0[q] < Tn) insert(d0[q], e, s, 0);
                                if (d1[q] >= T && d1[q] < Tn) insert(d1[q], e, s, 1);
                                if (d0[q] >= Tn) m = min(m, d0[q]);
                                if (d1[q] >= Tn) m = min(m, d1[q]);
                            }
                        }
                        lbe = min(lbe, m);
                    }
                    return __reduce_min_sync(0xffffffffu, lbe);
                };
                auto load_row = [&](int k, int r, int t0, int step) {
                    if (r < nr) {
                        const unsigned v = ends[wrows[r]];
                        load_rows(k, v & 0xffff, v >> 16, t0, step);
                    } else {
                        cp_commit();
                    }
                };
                auto seal_row = [&](int k, int r, int t0, int step) {
                    const unsigned v = ends[wrows[r]];
                    seal_rows(k, v & 0xffff, v >> 16, t0, step);
                };
                // Scans the short rows, eight lanes for each end of an edge, four
                // neighbours per lane: their costs are read together, then those
                // of the pairs they leave open (two waits for L2 per row).
                auto scan_short = [&]() {
                    constexpr int kPer = kNear / 8;
                    for (int i0 = 4 * warp; i0 < 2 * ns; i0 += 4 * kW) {
                        const int item = min(i0 + (lane >> 3), 2 * ns - 1);
                        const bool on = i0 + (lane >> 3) < 2 * ns;
                        const int e = rows[item >> 1], side = item & 1;
                        const unsigned ve = ends[e];
                        const int u = side ? ve >> 16 : ve & 0xffff, w = side ? ve & 0xffff : ve >> 16;
                        const int de = len[e];
                        int2 nb[kPer];
#pragma unroll
                        for (int k = 0; k < kPer; ++k) nb[k] = near[u * kNear + (lane & 7) + 8 * k];
                        const int rw = min(farthest(w), de);
                        const int ru =
                            min(__shfl_sync(0xffffffffu, nb[kPer - 1].x, (lane & 24) + 7), de);
                        int lbe = ru + rw - 2 * de;  // what the lists leave out
                        int c2[2 * kPer], slot[2 * kPer];
#pragma unroll
                        for (int k = 0; k < kPer; ++k) {
                            const int v = nb[k].y;
                            const bool listed = on && nb[k].x < ru && v != w;
                            const unsigned two = inc[v];
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const int s = q ? two >> 16 : two & 0xffff, ds = len[s];
                                const unsigned vs = ends[s];
                                const bool first = static_cast<int>(vs & 0xffff) == v;
                                const int z = first ? vs >> 16 : vs & 0xffff;
                                const bool open = listed && ds <= de - (s >= e ? 1 : 0) && z != u &&
                                                  z != w && nb[k].x - de - ds < 0;
                                slot[2 * k + q] = open ? s | (first ? 0x2000 : 0) : -1;
                                if (open) c2[2 * k + q] = cost(w, z);
                            }
                        }
#pragma unroll
                        for (int k = 0; k < 2 * kPer; ++k) {
                            if (slot[k] < 0 || (side && c2[k] < rw)) continue;  // (the other end lists it)
                            const int s = slot[k] & 0x1fff, d = nb[k / 2].x + c2[k] - de - len[s];
                            const int type = (slot[k] >> 13) == (side == 0 ? 1 : 0) ? 0 : 1;
                            if (d >= Tn) lbe = min(lbe, d);
                            else if (d >= T) insert(d, e, s, type);
                        }
#pragma unroll
                        for (int o = 1; o < 8; o <<= 1)
                            lbe = min(lbe, __shfl_xor_sync(0xffffffffu, lbe, o));
                        if (on && (lane & 7) == 0 && lbe < 0) atomicMin(&low[e], lbe);
                    }
                };
                bool shrunk = false;
                for (;;) {
                    scans += nr + ns;
                    scan_short();
                    if constexpr (kWarpScan) {
                        if (kStages) load_row(2 * warp, warp, lane, 32);
                        for (int r = warp, q = 0; r < nr; r += kW, q ^= 1) {
                            const int k = 2 * warp + q;
                            if (kStages) {
                                load_row(2 * warp + (q ^ 1), r + kW, lane, 32);
                                cp_wait<1>();
                                seal_row(k, r, lane, 32);
                            }
                            __syncwarp();
                            const int e = wrows[r];
                            const int lbe = scan(k, e, lane, 32);
                            if (lane == 0) atomicMin(&low[e], lbe);
                            __syncwarp();  // the buffer is no longer read
                        }
                        if (kStages) cp_wait_all();
                    } else {
                        if (nr > 0) load_row(0, 0, tid, NT);
                        for (int r = 0; r < nr; ++r) {
                            const int k = r & 1;
                            cp_wait_all();
                            seal_row(k, r, tid, NT);
                            __syncthreads();
                            if (r + 1 < nr) load_row(k ^ 1, r + 1, tid, NT);
                            const int e = wrows[r];
                            const int lbe = scan(k, e, tid, NT);
                            if (lane == 0) atomicMin(&low[e], lbe);
                        }
                    }
                    __syncthreads();
                    if (s_cnt <= cap) break;
                    // The list ran full: T' falls to the largest, over 32 groups of
                    // threads, of the group's smallest delta, what this round
                    // added is dropped and its rows are scanned again.  Where T'
                    // cannot stay above T (ties), T falls too, which bounds those
                    // rows as well, and the next passes are direct.
                    int mk = INT_MAX;
                    for (int k = tid; k < cap; k += NT)
                        if (list[k] != kDead) mk = min(mk, static_cast<int>(list[k] >> 32));
#pragma unroll
                    for (int o = 1; o < kW; o <<= 1)  // 32 groups of threads
                        mk = min(mk, __shfl_xor_sync(0xffffffffu, mk, o));
                    mk = __reduce_max_sync(0xffffffffu, mk == INT_MAX ? INT_MIN : mk);
                    if (lane == 0) s_hi[warp] = mk;
                    __syncthreads();
                    int t = s_hi[0];
#pragma unroll
                    for (int w = 1; w < kW; ++w) t = max(t, s_hi[w]);
                    Tn = min(Tn, t);
                    fold(Tn, T);
                    shrunk = true;
                    if (Tn <= T) {
                        T = Tn;
                        direct = 8 * n;
                        for (int k = tid; k < ns + nr; k += NT)
                            low[k < ns ? rows[k] : wrows[k - ns]] = T;
                        __syncthreads();
                        break;
                    }
                }
                const int cnt = s_cnt;
                best = block_best(list_best(min(c0, cnt), cnt));
                T = Tn;
                if (shrunk) level = min(level + 1, 6);
                else if (level > 0 && cnt < cap / 4) --level;
            }
            ++passes;
            if (best == ~0ull) break;

            // Apply it: positions bi < bj, slots e and h.
            const int bi = static_cast<int>((best >> 16) & 0xffffu);
            const int bj = static_cast<int>(best & 0xffffu);
            f += static_cast<int>(static_cast<uint32_t>(best >> 32) ^ 0x80000000u);
            last_bi = bi;
            last_bj = bj;
            const unsigned ae = at[bi], ah = at[bj];
            const int e = ae & 0x7fff, h = ah & 0x7fff;
            const unsigned ve = ends[e], vh = ends[h];
            const int xa = ae >> 15 ? ve >> 16 : ve & 0xffff, xa1 = ae >> 15 ? ve & 0xffff : ve >> 16;
            const int xb = ah >> 15 ? vh >> 16 : vh & 0xffff, xb1 = ah >> 15 ? vh & 0xffff : vh >> 16;
            if (!kLists) {
                load_rows(0, xa, xb, tid, NT);
                load_rows(1, xa1, xb1, tid, NT);
            }
            const int cnt0 = s_cnt;
            // the new edges, and the least a pair can cost at their ends
            const int de = cost(xa, xb), dh = cost(xa1, xb1);
            const int least_e = nearest(xa) + nearest(xb), least_h = nearest(xa1) + nearest(xb1);
            // candidates of the removed edges go
            for (int k = tid; k < cnt0; k += NT) {
                const unsigned lo = static_cast<unsigned>(list[k]);
                const int s0 = (lo >> 13) & 0x1fff, s1 = lo & 0x1fff;
                if (s0 == e || s0 == h || s1 == e || s1 == h) list[k] = kDead;
            }
            // the edges strictly between turn round
            for (int q = tid; q < (bj - bi) / 2; q += NT) {
                const int p0 = bi + 1 + q, p1 = bj - 1 - q;
                const unsigned a0 = at[p0] ^ 0x8000u, a1 = at[p1] ^ 0x8000u;
                at[p0] = static_cast<uint16_t>(a1);
                at[p1] = static_cast<uint16_t>(a0);
                pos[a1 & 0x7fff] = static_cast<uint16_t>(p0 | (a1 & 0x8000u));
                pos[a0 & 0x7fff] = static_cast<uint16_t>(p1 | (a0 & 0x8000u));
            }
            __syncthreads();  // every thread has read at[bi], at[bj] and their ends
            if (tid == 0) {
                ends[e] = xa | (xb << 16);
                ends[h] = xa1 | (xb1 << 16);
                len[e] = de;
                len[h] = dh;
                low[e] = kLists ? max(T, least_e - 2 * de) : INT_MAX;
                low[h] = kLists ? max(T, least_h - 2 * dh) : INT_MAX;
                // xb changes from h to e, xa1 from e to h
                const unsigned ib = inc[xb], ia = inc[xa1];
                inc[xb] = static_cast<int>(ib & 0xffff) == h ? (ib & 0xffff0000u) | e
                                                             : (ib & 0xffff) | (e << 16);
                inc[xa1] = static_cast<int>(ia & 0xffff) == e ? (ia & 0xffff0000u) | h
                                                              : (ia & 0xffff) | (h << 16);
                at[bi] = static_cast<uint16_t>(e);
                at[bj] = static_cast<uint16_t>(h);
                pos[e] = static_cast<uint16_t>(bi);
                pos[h] = static_cast<uint16_t>(bj);
                s_rows = 0;
            }
            if (!kLists && !kFull) {
                cp_wait_all();
                seal_rows(0, xa, xb, tid, NT);
                seal_rows(1, xa1, xb1, tid, NT);
            }
            __syncthreads();

            if constexpr (kLists) {
                // The pairs of the two new edges.  Their deltas are no less than
                // least - (both edges), so only slots where that is below T, or
                // below the low of a longer slot, are looked at: their own lows
                // start at that bound.
                {
                    unsigned fe = 0, fh = 0;  // bit k: this thread's k-th slot (at most 32)
#pragma unroll 4
                    for (int s = tid, k = 0; s < n; s += NT, ++k) {
                        const int ds = len[s], over = min(max(low[s], T), 0);
                        const bool le = least_e - de - ds < (ds > de - (s >= e ? 1 : 0) ? over : T);
                        const bool lh = least_h - dh - ds < (ds > dh - (s >= h ? 1 : 0) ? over : T);
                        fe |= static_cast<unsigned>(le && s != e) << k;
                        fh |= static_cast<unsigned>(lh && s != h && s != e) << k;
                    }
                    const int mine = __popc(fe | fh);
                    int upto = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, upto, o);
                        if (lane >= o) upto += y;
                    }
                    int k = lane == 31 ? atomicAdd(&s_rows, upto) : 0;
                    k = __shfl_sync(0xffffffffu, k, 31) + upto - mine;
                    for (unsigned f = fe | fh; f; f &= f - 1) {
                        const int bit = __ffs(f) - 1;
                        rows[k++] = static_cast<uint16_t>((tid + bit * NT) | (fe >> bit & 1) << 13 |
                                                          (fh >> bit & 1) << 14);
                    }
                }
                __syncthreads();
                {
                    // (a thread's entries' costs are read together)
                    constexpr int kHits = 4;
                    const int hits = 2 * s_rows;
                    for (int k0 = tid; k0 < hits; k0 += kHits * NT) {
                        int d0[kHits], d1[kHits], slot[kHits];
#pragma unroll
                        for (int q = 0; q < kHits; ++q) {
                            const int k = k0 + q * NT;
                            const int v = k < hits ? rows[k >> 1] : 0, s = v & 0x1fff;
                            const bool second = k & 1;
                            const int u = second ? xa1 : xa, w = second ? xb1 : xb;
                            const unsigned vs = ends[s];
                            const int c0 = vs & 0xffff, c1 = vs >> 16;
                            // (a shared city: one reconnection changes nothing, the
                            // other is none)
                            const bool on = (v & (second ? 0x4000 : 0x2000)) && c0 != u && c0 != w &&
                                            c1 != u && c1 != w;
                            slot[q] = on ? s : -1;
                            if (on) {
                                const int both = (second ? dh : de) + len[s];
                                d0[q] = cost(u, c0) + cost(w, c1) - both;
                                d1[q] = cost(u, c1) + cost(w, c0) - both;
                            }
                        }
#pragma unroll
                        for (int q = 0; q < kHits; ++q) {
                            const int s = slot[q];
                            if (s < 0) continue;
                            const bool second = (k0 + q * NT) & 1;
                            const int x = second ? h : e, dx = second ? dh : de;
                            const int own = len[s] <= dx - (s >= x ? 1 : 0) ? x : s;
                            if (min(d0[q], d1[q]) >= low[own]) continue;  // (T <= low)
                            int keep = INT_MAX;  // the smallest not in the list
#pragma unroll
                            for (int type = 0; type < 2; ++type) {
                                const int d = type ? d1[q] : d0[q];
                                if (d < T) {
                                    if (insert(d, x, s, type)) continue;
                                    atomicMin(&s_drop, d);  // T falls to it after the pass
                                }
                                keep = min(keep, d);
                            }
                            if (keep < low[own]) atomicMin(&low[own], keep);
                        }
                    }
                }
            } else {
                // The new edge x (staged in buffer k) against every other but
                // `skip`: candidates below T go to the list, the smallest delta past
                // T to the low of the pair's owner.
                auto against = [&](int k, int x, int u, int w, int skip) {
                    const int dx = len[x];
                    int lbx = INT_MAX;
                    for (int s0 = tid; s0 < n; s0 += kBatch * NT) {
                        int d0[kBatch], d1[kBatch], ml[kBatch], m = INT_MAX;
                        bool lower = false;
#pragma unroll
                        for (int q = 0; q < kBatch; ++q) {
                            const int s = min(s0 + q * NT, n - 1);
                            const unsigned v = ends[s];
                            const int ds = len[s];
                            const int2 A = costs(k, u, w, v & 0xffff);
                            const int2 B = costs(k, u, w, v >> 16);
                            const bool ok = s0 + q * NT < n && s != x && s != skip;
                            d0[q] = ok ? A.x + B.y - dx - ds : INT_MAX;
                            d1[q] = ok ? B.x + A.y - dx - ds : INT_MAX;
                            const int mq = min(d0[q], d1[q]);
                            const bool own = ds <= dx - (s >= x ? 1 : 0);
                            m = min(m, mq);
                            lbx = min(lbx, own && mq >= T ? mq : INT_MAX);
                            ml[q] = own ? INT_MAX : mq;
                            lower = lower || ml[q] < low[s];
                        }
                        if (m < T || lower) {
#pragma unroll
                            for (int q = 0; q < kBatch; ++q) {
                                const int s = s0 + q * NT;
                                int keep = INT_MAX;  // the smallest not in the list
#pragma unroll
                                for (int type = 0; type < 2; ++type) {
                                    const int d = type ? d1[q] : d0[q];
                                    if (d < T) {
                                        if (insert(d, x, s, type)) continue;
                                        atomicMin(&s_drop, d);  // T falls to it after the pass
                                    }
                                    keep = min(keep, d);
                                }
                                if (ml[q] == INT_MAX) lbx = min(lbx, keep);
                                else if (keep < low[s]) atomicMin(&low[s], keep);
                            }
                        }
                    }
                    lbx = __reduce_min_sync(0xffffffffu, lbx);
                    if (lane == 0) atomicMin(&low[x], lbx);
                };
                against(0, e, xa, xb, -1);
                against(1, h, xa1, xb1, e);
            }
            scans += 2;
            ++moves;
            __syncthreads();
            if (s_cnt > cap) {
                T = min(T, s_drop);
                __syncthreads();
                fold(T, INT_MAX);
            }
            best = block_best(list_best(0, s_cnt));
        }

        __syncthreads();
        for (int i = tid; i < n; i += NT) {
            const unsigned v = ends[at[i] & 0x7fff];
            tour[i] = static_cast<uint16_t>(at[i] >> 15 ? v >> 16 : v & 0xffff);
        }
        if (tid == 0) {
            const long long npairs = static_cast<long long>(n) * (n - 3) / 2;
            a.cost[p] = f;
            if (a.tour_passes) {
                a.tour_passes[p] = static_cast<unsigned int>(passes);
                a.tour_moves[p] = static_cast<unsigned int>(moves);
            } else {
                atomicAdd(a.pairs, static_cast<unsigned long long>(passes * npairs));
                atomicAdd(a.moves, static_cast<unsigned long long>(moves));
            }
            if (a.evals)
                atomicAdd(a.evals, static_cast<unsigned long long>(
                                       min(scans * (n - 3), static_cast<long long>(passes) * npairs)));
            s_pf = a.pbest ? a.pcost[p] : LLONG_MIN;
        }
        __syncthreads();
        if (a.pbest && f < s_pf) {
            uint16_t* pb = a.pbest + static_cast<size_t>(p) * a.ldt;
            for (int i = tid; i < n; i += NT) {
                const unsigned v = ends[at[i] & 0x7fff];
                pb[i] = static_cast<uint16_t>(at[i] >> 15 ? v >> 16 : v & 0xffff);
            }
            if (tid == 0) a.pcost[p] = f;
        }
        __syncthreads();
    }
}

constexpr size_t kMaxSmem = 224 * 1024;

template <int NT, Staging ST>
cudaError_t launch_cfg(const TwoOptBatch& b, int cap, int num_sms, cudaStream_t st) {
    auto* kern = two_opt_list_kernel<NT, ST>;
    const size_t smem = list_smem(b.max_n, staged_bufs(NT, ST), ST == kMatrix, cap);
    cudaError_t e = raise_smem_limit(kern, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int grid = max(1, min(b.total, per_sm * num_sms));
    kern<<<grid, NT, smem, st>>>(b, cap);
    return cudaGetLastError();
}

// Launch configurations: for tours of up to max_n viewpoints (and, with
// `few`, launches of at most that many tours per SM): threads per tour,
// staging, list entries.  Measured on GB300 (random tours of a grid, at 1992 of
// the bridge, to 2-optimality, whole call, ms; warp = each warp stages its rows;
// CTA and C with neighbour lists):
//   n     tours  matrix 256  warp 64 / 128  CTA 128 / 256  C 128 / 256
//   157   256    0.42        0.58 / 0.47    -              0.52 / 0.51
//   157   1024   1.27        0.74 / 0.95    -              0.95 / 1.60
//   200   128    0.48        -    / 0.58    -              0.66 / 0.59
//   220   128    0.49        -    / 0.68    -              0.78 / 0.64
//   200   304    -           0.80 / 0.64    -              0.72 / 0.67
//   200   450    -           0.86 / 0.68    -              0.76 / 1.15
//   400   150    -           1.90 / 1.34    -              1.48 / 1.27
//   400   304    -           1.91 / 1.56    -              1.64 / 1.43
//   400   330    -           2.04 / 1.65    -              1.64 / 2.29
//   400   608    -           2.23 / 2.02    -              1.85 / 2.67
//   400   1024   -           2.82 / 3.38    -              3.18 / 4.74
//   512   450    -           2.80 / 2.17    -              2.20 / 3.38
//   512   1024   -           5.68 / 4.67    -              4.17 / 6.37
//   700   150    -           -              2.95 / 2.46    2.87 / 2.42
//   1000  150    -           -              4.63 / 3.81    4.74 / 3.87
//   1000  304    -           -              4.99 / 4.48    5.22 / 4.56
//   1000  600    -           -              6.28 / 8.70    6.67 / 8.81
//   1200  150    -           -              5.89 / 4.98    6.22 / 5.13
//   1200  600    -           -              8.17 / 11.4    9.29 / 11.8
//   1992  600    -           -              30.6 / 26.2    -    / 31.6
//   2999  150    -           -              -    / 18.1    -    / 24.9
// (512 viewpoints and 64 threads: six tours an SM, so 1024 take two waves.)
struct ListConfig {
    int max_n, few, threads;
    Staging staging;
    int cap;
};
constexpr int kAny = INT_MAX;
constexpr ListConfig kConfigs[] = {
    {160, 2, 256, kMatrix, 512},        {220, 1, 256, kMatrix, 512},
    {512, 2, 256, kGlobal, 512},        {512, 4, 128, kWarpRows, 512},
    {512, kAny, 64, kWarpRows, 1024},    {1200, 1, 256, kGlobal, 1024},
    {1200, kAny, 128, kCtaRows, 1024},  {5000, kAny, 256, kCtaRows, 2048},
    {DPSO_MAX_N, kAny, 512, kGlobal, 1024},
};
constexpr int kNumConfigs = sizeof(kConfigs) / sizeof(kConfigs[0]);

constexpr size_t config_smem(const ListConfig& c, int n) {
    return list_smem(n, staged_bufs(c.threads, c.staging), c.staging == kMatrix, c.cap);
}

int find_config(int n, int total, int num_sms) {
    int k = 0;
    while (k + 1 < kNumConfigs &&
           (n > kConfigs[k].max_n ||
            (kConfigs[k].few != kAny && total > kConfigs[k].few * num_sms)))
        ++k;
    return k;
}

template <int K>
cudaError_t launch_k(const TwoOptBatch& b, int k, int num_sms, cudaStream_t st) {
    constexpr ListConfig c = kConfigs[K];
    static_assert(config_smem(c, c.max_n) <= kMaxSmem, "does not fit");
    if (k == K) return launch_cfg<c.threads, c.staging>(b, c.cap, num_sms, st);
    if constexpr (K + 1 < kNumConfigs) return launch_k<K + 1>(b, k, num_sms, st);
    else return cudaErrorInvalidValue;
}

// Tours that go to the kernel that scans every pair (two_opt_small.cu).
// Measured as above, us, against the best list configuration: n = 30, 256
// tours 2 and 66, 1024 tours 45 and 109; n = 65, 256 tours 72 and 130, 1024
// tours 189 and 233; n = 80, 256 tours 151 and 177, 1024 tours 487 and 311.
constexpr int kSmallAlways = 65, kSmallFew = 2;
bool takes_small(int n, int total, int num_sms) {
    return two_opt_small_threads(n) > 0 && (n <= kSmallAlways || total <= kSmallFew * num_sms);
}

}  // namespace

int two_opt_class(int n, int* ctas) {
    constexpr int kMany = 1 << 24;
    *ctas = 0;
    if (takes_small(n, kMany, 1)) return -1;
    const int k = find_config(n, kMany, 1);
    const ListConfig& c = kConfigs[k];
    // 228 KB of shared memory per SM, 1 KB of it reserved per CTA
    *ctas = min(static_cast<int>((228 * 1024) / (config_smem(c, n) + 1280)),
                kThreadsPerSm / c.threads);
    return k;
}

bool near_used(int n, int total, int num_sms) {
    if (takes_small(n, total, num_sms)) return false;
    const Staging st = kConfigs[find_config(n, total, num_sms)].staging;
    return st == kCtaRows || st == kGlobal;
}

cudaError_t build_near(const int* C, int ldc, int n, int2* near, cudaStream_t st) {
    near_kernel<<<(n + 3) / 4, 128, 0, st>>>(C, ldc, n, near);
    return cudaGetLastError();
}

cudaError_t launch_two_opt(const TwoOptBatch& b, int num_sms, cudaStream_t st) {
    if (b.total <= 0) return cudaSuccess;
    if (b.kind == 1) return launch_node_swap(b, num_sms, st);
    if (b.rows > 0 && b.shifted) {  // a pinned shape of the tiled kernel
        const int tpc = b.tpc > 0 ? b.tpc : two_opt_tiled_tpc(b.max_n, b.rows);
        const int tg = b.tg > 0 ? b.tg : two_opt_tiled_tg(b.max_n, b.rows, tpc);
        return launch_two_opt_tiled(b, b.rows, tpc, tg, num_sms, st);
    }
    if (b.max_n < 3 || b.max_n > DPSO_MAX_N) return cudaErrorInvalidValue;
    if (takes_small(b.max_n, b.total, num_sms)) return launch_two_opt_small(b, num_sms, st);
    return launch_k<0>(b, find_config(b.max_n, b.total, num_sms), num_sms, st);
}

}  // namespace dpso
