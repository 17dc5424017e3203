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
//    no smaller than minus its edges.  When no candidate fits, T is raised to
//    T' and the slots with low < T' scan their row: candidates in [T, T') go
//    to the list, the smallest delta past T' becomes the slot's low.
//  * T' is the largest, over groups of threads, of the group's smallest low:
//    about G ln G rows for G groups, a few scans per move in all.
// With T = 0 and no candidate that fits, the tour is 2-optimal.
//
// A list that runs full folds its upper part back into low (T falls).  Where
// more candidates than it holds tie on one delta, so that T cannot rise, a
// pass scans every row with low < 0 and takes the best directly.
//
// What bounds it: a row scan reads the cost rows of the edge's two ends from
// L2 (staged interleaved in shared memory, so that one 8-byte gather brings
// both ends' costs to a city) and gathers them at both ends of every other
// edge: shared-memory gathers with random bank conflicts, then issue slots.
// Short tours wait for L2 and barriers; several tours per SM hide that.
#include <climits>

#include "tiled_common.cuh"

namespace dpso {
namespace {

using namespace tiled;

constexpr int kThreadsPerSm = 768;  // the register budget's resident threads
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
    return staged + m * (sizeof(unsigned) + 2 * sizeof(int) + 3 * sizeof(uint16_t)) +
           static_cast<size_t>(cap) * sizeof(unsigned long long);
}

// How a launch stages cost rows and shares out the rows of a scan round.
//   kMatrix    the whole matrix in shared memory (few tours per SM: no wait for
//              L2 after the first); every warp scans its own rows
//   kWarpRows  each warp stages and scans its own rows (two buffers per warp)
//   kCtaRows2  the CTA scans one row at a time while the next one arrives
//   kCtaRows1  the same with one buffer (the longest tours)
enum Staging { kMatrix, kWarpRows, kCtaRows2, kCtaRows1 };

__host__ __device__ constexpr int staged_bufs(int threads, Staging st) {
    return st == kWarpRows ? 2 * (threads / 32) : (st == kCtaRows1 ? 1 : 2);
}

// NT threads solve one tour.
template <int NT, Staging ST>
__global__ void __launch_bounds__(NT, (NT >= 512 ? 1 : kThreadsPerSm / NT))
    two_opt_list_kernel(TwoOptBatch b, int cap) {
    constexpr int kW = NT / 32;                     // warps
    constexpr int kBufs = staged_bufs(NT, ST);      // staged row pairs
    constexpr bool kFull = ST == kMatrix;
    constexpr bool kWarpScan = ST == kMatrix || ST == kWarpRows;
    constexpr int kBatch = 4;                       // partners a thread has in flight
    // threads per group of the choice of T' (see the head of the file)
    constexpr int kGroup = NT / 16;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned long long s_key[2][kW];  // the warps' best, by pass parity
    __shared__ int s_lo[kW], s_hi[kW];
    __shared__ int s_item, s_cnt, s_rows, s_drop;
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
    uint16_t* const pos = reinterpret_cast<uint16_t*>(low + m8);  // slot -> position | dir << 15
    uint16_t* const at = pos + m8;                                // position -> slot | dir << 15
    uint16_t* const rows = at + m8;                               // slots to scan

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
            low[i] = -2 * d;
            pos[i] = static_cast<uint16_t>(i);
            at[i] = static_cast<uint16_t>(i);
        }
        if (tid == 0) {
            s_cnt = 0;
            s_drop = INT_MAX;
        }
        long long f = a.cost[p];
        long long scans = 0;  // rows scanned
        int moves = 0, passes = 0;
        int T = INT_MIN;      // the list holds every candidate with delta < T
        int direct = 0;       // passes to take directly (ties overflow the list)
        int level = 0;        // doublings of the groups that choose T' (after a full list)
        int par = 0;
        const int guard = 1000 + 100 * n;
        if (kFull) cp_wait_all();
        __syncthreads();

        // Stages the cost rows of edge (u, w) interleaved into buffer k, by
        // threads t0, t0 + step, ..: one copy group.
        auto load_rows = [&](int k, int u, int w, int t0, int step) {
            if constexpr (!kFull) {
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
            if constexpr (!kFull) {
                if (u % step == t0) buf0[k * m8 + u].x = kBig;
                if (w % step == t0) buf0[k * m8 + w].y = kBig;
            }
        };
        // Costs of city c to the two ends (u, w) of the edge staged in buffer k.
        auto costs = [&](int k, int u, int w, int c) {
            if constexpr (kFull) return make_int2(mat[u * mld + c], mat[w * mld + c]);
            else return buf0[k * m8 + c];
        };
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
                if (tid == 0) s_rows = 0;
                compact(min(s_cnt, cap));
                int mn = INT_MAX;
                for (int s = tid; s < n; s += NT) mn = min(mn, low[s]);
                int gm = mn;
                for (int o = 1; o < min(kGroup << level, 32); o <<= 1)
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
                const int c0 = s_cnt;
                const bool dir = direct > 0;
                if ((kGroup << level) > (kW > 1 ? 32 : 16)) hi = lo;
                int Tn = dir ? 0 : min(0, max(hi, lo + 1));
                for (int s0 = 0; s0 < n; s0 += NT) {
                    const int s = s0 + tid;
                    const bool take = s < n && low[s] < Tn;
                    const unsigned mask = __ballot_sync(0xffffffffu, take);
                    if (mask == 0) continue;
                    int k = lane == 0 ? atomicAdd(&s_rows, __popc(mask)) : 0;
                    k = __shfl_sync(0xffffffffu, k, 0) + __popc(mask & ((1u << lane) - 1));
                    if (take) {
                        rows[k] = static_cast<uint16_t>(s);
                        if (!dir) low[s] = INT_MAX;
                    }
                }
                __syncthreads();
                const int nr = s_rows;  // at least the row whose low is lo
                unsigned long long mine = ~0ull;
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
                                if (dir) {
                                    if (d0[q] < 0) mine = min(mine, key_of(d0[q], e, s, 0));
                                    if (d1[q] < 0) mine = min(mine, key_of(d1[q], e, s, 1));
                                } else {
                                    if (d0[q] >= T && d0[q] < Tn) insert(d0[q], e, s, 0);
                                    if (d1[q] >= T && d1[q] < Tn) insert(d1[q], e, s, 1);
                                    if (d0[q] >= Tn) m = min(m, d0[q]);
                                    if (d1[q] >= Tn) m = min(m, d1[q]);
                                }
                            }
                        }
                        lbe = min(lbe, m);
                    }
                    return __reduce_min_sync(0xffffffffu, lbe);
                };
                auto load_row = [&](int k, int r, int t0, int step) {
                    if (r < nr) {
                        const unsigned v = ends[rows[r]];
                        load_rows(k, v & 0xffff, v >> 16, t0, step);
                    } else {
                        cp_commit();
                    }
                };
                auto seal_row = [&](int k, int r, int t0, int step) {
                    const unsigned v = ends[rows[r]];
                    seal_rows(k, v & 0xffff, v >> 16, t0, step);
                };
                bool shrunk = false;
                for (;;) {
                    scans += nr;
                    if constexpr (kWarpScan) {
                        if (!kFull) load_row(2 * warp, warp, lane, 32);
                        for (int r = warp, q = 0; r < nr; r += kW, q ^= 1) {
                            const int k = 2 * warp + q;
                            if (!kFull) {
                                load_row(2 * warp + (q ^ 1), r + kW, lane, 32);
                                cp_wait<1>();
                                seal_row(k, r, lane, 32);
                            }
                            __syncwarp();
                            const int e = rows[r];
                            const int lbe = scan(k, e, lane, 32);
                            if (!dir && lane == 0) low[e] = lbe;
                            __syncwarp();  // the buffer is no longer read
                        }
                        if (!kFull) cp_wait_all();
                    } else {
                        load_row(0, 0, tid, NT);
                        for (int r = 0; r < nr; ++r) {
                            const int k = ST == kCtaRows2 ? r & 1 : 0;
                            cp_wait_all();
                            seal_row(k, r, tid, NT);
                            __syncthreads();
                            if (ST == kCtaRows2 && r + 1 < nr) load_row(k ^ 1, r + 1, tid, NT);
                            const int e = rows[r];
                            const int lbe = scan(k, e, tid, NT);
                            if (!dir && lane == 0) atomicMin(&low[e], lbe);
                            if (ST == kCtaRows1 && r + 1 < nr) {
                                __syncthreads();  // the buffer is no longer read
                                load_row(0, r + 1, tid, NT);
                            }
                        }
                    }
                    __syncthreads();
                    if (s_cnt <= cap) break;
                    // The list ran full: T' falls to the largest, over 32
                    // groups of threads, of the group's smallest delta, what this round added is dropped and its
                    // rows are scanned again.  Where T' cannot stay above T
                    // (ties), T falls too and the next passes are direct.
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
                    if (Tn <= T) {
                        T = Tn;
                        direct = 16;
                    }
                    shrunk = true;
                }
                const int cnt = s_cnt;
                if (!dir) mine = list_best(min(c0, cnt), cnt);
                best = block_best(mine);
                if (dir) {
                    --direct;
                    if (best == ~0ull) T = 0;  // every row was looked at
                } else {
                    T = Tn;
                    if (shrunk) level = min(level + 1, 6);
                    else if (level > 0 && cnt < cap / 4) --level;
                }
            }
            ++passes;
            if (best == ~0ull) break;

            // Apply it: positions bi < bj, slots e and h.
            const int bi = static_cast<int>((best >> 16) & 0xffffu);
            const int bj = static_cast<int>(best & 0xffffu);
            f += static_cast<int>(static_cast<uint32_t>(best >> 32) ^ 0x80000000u);
            const unsigned ae = at[bi], ah = at[bj];
            const int e = ae & 0x7fff, h = ah & 0x7fff;
            const unsigned ve = ends[e], vh = ends[h];
            const int xa = ae >> 15 ? ve >> 16 : ve & 0xffff, xa1 = ae >> 15 ? ve & 0xffff : ve >> 16;
            const int xb = ah >> 15 ? vh >> 16 : vh & 0xffff, xb1 = ah >> 15 ? vh & 0xffff : vh >> 16;
            load_rows(0, xa, xb, tid, NT);
            if (kBufs > 1) load_rows(1, xa1, xb1, tid, NT);
            const int cnt0 = s_cnt;
            int de = 0, dh = 0;
            if (tid == 0) {
                de = kFull ? mat[xa * mld + xb] : C[static_cast<size_t>(xa) * ldc + xb];
                dh = kFull ? mat[xa1 * mld + xb1] : C[static_cast<size_t>(xa1) * ldc + xb1];
            }
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
                low[e] = INT_MAX;
                low[h] = INT_MAX;
                at[bi] = static_cast<uint16_t>(e);
                at[bj] = static_cast<uint16_t>(h);
                pos[e] = static_cast<uint16_t>(bi);
                pos[h] = static_cast<uint16_t>(bj);
            }
            if (!kFull) cp_wait_all();
            seal_rows(0, xa, xb, tid, NT);
            if (kBufs > 1) seal_rows(1, xa1, xb1, tid, NT);
            __syncthreads();

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
            if (kBufs == 1) {
                __syncthreads();
                load_rows(0, xa1, xb1, tid, NT);
                cp_wait_all();
                seal_rows(0, xa1, xb1, tid, NT);
                __syncthreads();
            }
            against(kBufs > 1 ? 1 : 0, h, xa1, xb1, e);
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
// staging, list entries.  Measured on GB300 (random grid and facade tours to
// 2-optimality, us; calls of one move taken off up to n = 220):
//   n     tours  matrix, 256 thr.  warp rows, 64 thr.  warp rows, 128 thr.
//   90    32     178               305                 256
//   90    1024   578               483                 559
//   157   256    389               719                 529
//   157   1024   1307              884                 1112
//   220   128    496               980                 691
//   220   304    907               1013                767
//   400   256    -                 2815                2116
//   400   1024   -                 4080                4550
// and with the CTA's rows: n = 1000, 600 tours 10.1 ms with 128 threads, 13.9
// with 256; n = 1992, 600 tours 45 and 39; n = 2999, 150 tours 35 and 28, 512
// threads 29.
struct ListConfig {
    int max_n, few, threads;
    Staging staging;
    int cap;
};
constexpr int kAny = INT_MAX;
constexpr ListConfig kConfigs[] = {
    {160, 2, 256, kMatrix, 512},        {220, 1, 256, kMatrix, 512},
    {512, 3, 128, kWarpRows, 512},      {512, kAny, 64, kWarpRows, 512},
    {1200, kAny, 128, kCtaRows2, 1024}, {5000, kAny, 256, kCtaRows2, 1024},
    {DPSO_MAX_N, kAny, 512, kCtaRows1, 1024},
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
