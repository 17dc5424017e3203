// Node-swap exchange: the "swap nodes(i,j) and evaluate fitness" reading of
// the edge exchange in the paper's GPU listing (Sec. 3.2.3, Fig. "pseudocode"
// GPU kernels).  The swap of x_i and x_j (every pair of positions i < j of the
// cyclic tour) with the most improvement is applied, repeatedly, until none
// improves (ties: smallest (delta, i, j)).
//
// With d_k = C[x_k][x_k+1] and s_k = d_k-1 + d_k (indices mod n):
//   delta(i, j) = C[x_i-1][x_j] + C[x_i+1][x_j] + C[x_j-1][x_i] + C[x_j+1][x_i]
//                 - s_i - s_j,
//   plus 2 d_i when j = i + 1 (that edge stays), 2 d_j when i = j + 1 (mod n).
//
// A swap changes the neighbourhood of six positions at most (p and q and the
// ones beside them), so only their pairs change: 6n of n^2/2.  The kernel
// keeps, for every position, the best of the pairs it owns (the position with
// the larger s owns a pair; ties: the larger position) and after a swap
//  * evaluates the pairs of the six positions: those they own give their new
//    best, the others may improve the best of their owners;
//  * marks a position whose best was with one of the six as stale: its value
//    is then a lower bound on the pairs it owns;
//  * takes the smallest best; stale positions below the best that is not stale
//    scan the pairs they own first.
// Owning by the larger s keeps stale positions few: the ones that many others
// would pair with own those pairs themselves.
//
// The first pass looks at every pair.  With M_i(j) = C[x_i][x_j] the four costs
// above are M_i-1(j), M_i+1(j), M_i(j-1) and M_i(j+1): a thread that holds
// neighbouring positions j and walks all i gathers one cost per pair, from the
// row of x_i+1 that the block staged meanwhile, and has the others from the
// steps before and from its neighbour lane.  Against
// a scan of every position's row, one swap per tour, whole call: 999 viewpoints,
// 30 tours 1143 -> 395 us; 1500 viewpoints, 700 tours 8.9 -> 1.8 ms; 2000
// viewpoints, 304 tours 8.3 -> 1.5 ms.  What bounds it: issue, six instructions
// a pair and the gather; with one tour per SM, the chain of n steps of some 500
// cycles each.
//
// The costs of a scanned position's pairs lie in three rows of C, those of the
// six positions in ten; they are staged in shared memory (short tours: the
// whole matrix).  What bounds it: the gathers from those rows (random bank
// conflicts) and, with few tours per SM, the chain of a pass.
#include <climits>

#include "tiled_common.cuh"

namespace dpso {
namespace {

using namespace tiled;

// A position's best: (delta, i, j), with bit 15 set once it is exact.  A stale
// value sorts before every exact one of the same (delta, i), so a tie with a
// stale position is looked at.  ~0: no improving pair.
constexpr unsigned long long kExact = 0x8000;
constexpr unsigned long long kNone = ~0ull;
constexpr int kNodeSwapMaxN = 4497;  // longer tours are refused (as the header says)
constexpr int kRowsStaged = 10;  // two swapped positions, two on each side

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// At most `Pending` of this thread's latest copy groups are still in flight.
template <int Pending>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(Pending) : "memory");
}

__host__ __device__ constexpr int mat_ld(int n) { return n | 1; }

// Where costs are read: the whole matrix in shared memory, staged rows (three
// per warp, ten at least), or C itself (the longest tours; the first pass's rows
// lie in the room of bestof, which it fills at its end, and in up to four rows
// more, as many as leave two blocks their room on an SM).
enum Costs { kMatrix, kStaged, kGlobal };

__host__ __device__ constexpr int rows_beside(int n, int warps, Costs costs) {
    if (costs == kStaged) return 3 * warps > kRowsStaged ? 3 * warps : kRowsStaged;
    const int room = (112 * 1024 - 20 * n) / (4 * n);
    return room > 4 ? 4 : (room < 2 ? 2 : room);
}
// Rows the first pass stages: pairs of them, at most four.
__host__ __device__ constexpr int ring_rows(int n, int warps, Costs costs) {
    const int rows = rows_beside(n, warps, costs) + (costs == kGlobal ? 2 : 0);
    return rows > 8 ? 8 : rows / 2 * 2;
}

__host__ __device__ constexpr size_t staged_words(int n, int warps, Costs costs) {
    return (costs == kMatrix ? static_cast<size_t>(n) * mat_ld(n)
                             : static_cast<size_t>(rows_beside(n, warps, costs)) * n) + 3;
}

constexpr size_t swap_smem(int n, int warps, Costs costs) {
    return staged_words(n, warps, costs) / 4 * 16 +
           static_cast<size_t>((n + 7) / 8 * 8) *
               (sizeof(unsigned long long) + 2 * sizeof(int) + 2 * sizeof(uint16_t));
}

// NT threads solve one tour; COLS: positions a thread holds in the first pass;
// CTAS: blocks that an SM is to hold, which sets the registers of one (128
// threads, 321 viewpoints, 127 tours: 2.43 ms with room for three blocks, 2.67
// with room for five; 760 tours of 700 need the five).
template <int NT, Costs COSTS, int COLS, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) node_swap_kernel(TwoOptBatch b) {
    constexpr int kW = NT / 32;
    constexpr bool kFull = COSTS == kMatrix, kRows = COSTS == kStaged;
    constexpr int kCols = COLS;
    constexpr int kNobody = 0xffff;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned long long s_exact[2][kW], s_stale[2][kW], s_six[2][kW][6];
    __shared__ int s_item, s_rows;
    __shared__ long long s_pf;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m8 = (b.max_n + 7) / 8 * 8;
    int* const mat = reinterpret_cast<int*>(smraw);  // the matrix, or staged rows
    unsigned long long* const bestof = reinterpret_cast<unsigned long long*>(
        smraw + staged_words(b.max_n, kW, COSTS) / 4 * 16);
    int* const dd = reinterpret_cast<int*>(bestof + m8);  // d_k
    int* const ss = dd + m8;                              // s_k
    uint16_t* const X = reinterpret_cast<uint16_t*>(ss + m8);
    uint16_t* const rows = X + m8;  // positions to scan

    for (;;) {
        if (tid == 0) s_item = static_cast<int>(atomicAdd(b.queue, 1u));
        __syncthreads();
        const int g = s_item;
        if (g >= b.total) break;
        const int prob = find_inst(b.off, b.nprob, g);
        const TwoOptTask& a = b.tasks[prob];
        const int p = a.order ? a.order[g - b.off[prob]] : g - b.off[prob];
        if (a.gate && *a.gate == 0) {  // this problem does not exchange now
            __syncthreads();
            continue;
        }
        const int n = a.n, ld = mat_ld(n);
        const int* __restrict__ const C = a.C;
        const int ldc = a.ldc, max_moves = a.max_moves;
        uint16_t* const tour = a.tours + static_cast<size_t>(p) * a.ldt;
        auto next = [&](int k) { return k + 1 == n ? 0 : k + 1; };
        auto prev = [&](int k) { return k == 0 ? n - 1 : k - 1; };

        if (kFull)
            for (int r = warp; r < n; r += kW)
                for (int c = lane; c < n; c += 32)
                    cp_async4(&mat[r * ld + c], C + static_cast<size_t>(r) * ldc + c);
        for (int i = tid; i < n; i += NT) {
            const int u = tour[i], w = tour[next(i)];
            X[i] = static_cast<uint16_t>(u);
            dd[i] = C[static_cast<size_t>(u) * ldc + w];
        }
        if (tid == 0) s_rows = 0;
        __syncthreads();
        for (int i = tid; i < n; i += NT) {
            ss[i] = dd[prev(i)] + dd[i];
        }
        long long f = a.cost[p];
        int moves = 0, passes = 0, par = 0;
        const int guard = 1000 + 100 * n;
        if (kFull) cp_wait_all();
        __syncthreads();

        // Costs of city c in staged row k, which holds C[city].
        auto cost = [&](int k, int city, int c) {
            if constexpr (kFull) return mat[city * ld + c];
            else if constexpr (kRows) return mat[k * n + c];
            else return C[static_cast<size_t>(city) * ldc + c];
        };
        // Stages C[city] as row k, by threads t0, t0 + step, ..
        auto load_row = [&](int k, int city, int t0, int step) {
            if constexpr (kRows) {
                const int* r = C + static_cast<size_t>(city) * ldc;
#pragma unroll 4
                for (int c = t0; c < n; c += step) cp_async4(&mat[k * n + c], r + c);
            }
        };
        // What the pair's shared edge gives back when i and j are neighbours.
        auto adjacent = [&](int i, int j) {
            return (next(i) == j ? 2 * dd[i] : 0) + (next(j) == i ? 2 * dd[j] : 0);
        };
        auto key_of = [&](int d, int i, int j) {
            return d < 0 ? pack_key(d, min(i, j), max(i, j)) | kExact : kNone;
        };
        auto owns = [&](int si, int i, int sj, int j) { return si > sj || (si == sj && i > j); };
        auto warp_min = [&](unsigned long long v) {
            const unsigned hi = static_cast<unsigned>(v >> 32);
            const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
            const unsigned ml =
                __reduce_min_sync(0xffffffffu, hi == mh ? static_cast<unsigned>(v) : ~0u);
            return (static_cast<unsigned long long>(mh) << 32) | ml;
        };

        unsigned long long exact, stale;  // the smallest of each kind
        auto smallest = [&]() {  // over all positions; one barrier
            exact = kNone;
            stale = kNone;
            for (int i = tid; i < n; i += NT) {
                const unsigned long long v = bestof[i];
                if (v & kExact) exact = min(exact, v);
                else stale = min(stale, v);
            }
            exact = warp_min(exact);
            stale = warp_min(stale);
            if (lane == 0) {
                s_exact[par][warp] = exact;
                s_stale[par][warp] = stale;
            }
            __syncthreads();
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                exact = min(exact, s_exact[par][w]);
                stale = min(stale, s_stale[par][w]);
            }
            par ^= 1;
        };

        // The first pass, NT * kCols positions j at a time.  Of the pairs with
        // an s_i no larger than s_j (those that j owns, and ties) the best one's i
        // goes to rows[j], except where i and j are neighbours: kApart in the place
        // of C's diagonal keeps those from improving.  Two rows are taken per
        // barrier, the next ones meanwhile on their way.
        constexpr int kApart = 1 << 29;  // twice it: no less than any s_i + s_j
        // The q-th row that a walk over i = 0 .. n-1 needs, q = i + 2 for x_i+1.
        auto walk_city = [&](int q) { return static_cast<int>(X[q == 0 ? n - 1 : (q > n ? 0 : q - 1)]); };
        const int steps = (n + 3) / 2, ahead = kFull ? 0 : ring_rows(b.max_n, kW, COSTS) / 2;
        const bool wide = ((reinterpret_cast<size_t>(C) | (4 * static_cast<size_t>(ldc))) & 15) == 0 &&
                          (n & 3) == 0;  // rows (and the staged ones) start on 16 bytes
        auto stage = [&](int t, int slot) {
            if constexpr (!kFull) {
                if (t < steps) {
                    const int* r0 = C + static_cast<size_t>(walk_city(2 * t)) * ldc;
                    const int* r1 = C + static_cast<size_t>(walk_city(2 * t + 1)) * ldc;
                    int* const to = mat + 2 * slot * n;
                    if (wide) {
                        for (int c = 4 * tid; c < n; c += 4 * NT) {
                            cp_async16(&to[c], r0 + c);
                            cp_async16(&to[n + c], r1 + c);
                        }
                    } else {
#pragma unroll 4
                        for (int c = tid; c < n; c += NT) {
                            cp_async4(&to[c], r0 + c);
                            cp_async4(&to[n + c], r1 + c);
                        }
                    }
                }
                cp_commit();
            }
        };
        for (int c0 = 0; c0 < n; c0 += NT * kCols) {
            const int j0 = c0 + tid * kCols;
            // (best: s_j + the best delta so far; past n: nothing is owned)
            int xj[kCols], sj[kCols], up[kCols], mid[kCols], best[kCols], bi[kCols];
#pragma unroll
            for (int k = 0; k < kCols; ++k) {
                const int j = j0 + k;
                xj[k] = X[j < n ? j : 0];  // (position n - 1 is followed by 0)
                sj[k] = j < n ? ss[j] : -1;
                best[k] = sj[k];
                bi[k] = kNobody;
                up[k] = mid[k] = 0;
            }
            // the neighbours of the warp's first and last position
            const int xe = X[lane == 0 ? (j0 == 0 ? n - 1 : min(j0, n) - 1)
                                       : (j0 + kCols < n ? j0 + kCols : 0)];
            int mid_e = 0;
            auto look = [&](int i, const int (&u)[kCols], const int (&m)[kCols], int m_e,
                            const int (&w)[kCols]) {
                const int si = ss[i];
                int left = __shfl_up_sync(0xffffffffu, m[kCols - 1], 1);
                int right = __shfl_down_sync(0xffffffffu, m[0], 1);
                if (lane == 0) left = m_e;
                if (lane == 31) right = m_e;
#pragma unroll
                for (int k = 0; k < kCols; ++k) {
                    const int d = u[k] + w[k] + (k > 0 ? m[k - 1] : left) +
                                  (k + 1 < kCols ? m[k + 1] : right) - si;
                    // (of equal deltas the smaller i has the smaller key)
                    const bool better = sj[k] >= si && d < best[k];
                    best[k] = better ? d : best[k];
                    bi[k] = better ? i : bi[k];
                }
            };
            for (int t = 0; t + 1 < ahead; ++t) stage(t, t);
            for (int t = 0, slot = 0; t < steps; ++t) {
                const int u0 = walk_city(2 * t), u1 = walk_city(2 * t + 1);
                const int* const r0 = kFull ? mat + u0 * ld : mat + 2 * slot * n;
                const int* const r1 = kFull ? mat + u1 * ld : r0 + n;
                if constexpr (!kFull) {
                    if (ahead > 3) cp_wait<2>();
                    else if (ahead > 2) cp_wait<1>();
                    else cp_wait<0>();
                    // (by the thread that copied the word)
                    if ((wide ? u0 / 4 : u0) % NT == tid) mat[2 * slot * n + u0] = kApart;
                    if ((wide ? u1 / 4 : u1) % NT == tid) mat[2 * slot * n + n + u1] = kApart;
                    __syncthreads();  // rows 2t, 2t + 1 are there, those before no longer read
                    stage(t + ahead - 1, slot == 0 ? ahead - 1 : slot - 1);
                }
                auto read = [&](const int* row, int u, int x) {
                    const int v = row[x];
                    return kFull && x == u ? kApart : v;
                };
                int a0[kCols], a1[kCols], e0 = 0, e1 = 0;
#pragma unroll
                for (int k = 0; k < kCols; ++k) {
                    a0[k] = read(r0, u0, xj[k]);
                    a1[k] = read(r1, u1, xj[k]);
                }
                if (lane == 0 || lane == 31) {
                    e0 = read(r0, u0, xe);
                    e1 = read(r1, u1, xe);
                }
                if (t > 0) {
                    look(2 * t - 2, up, mid, mid_e, a0);
                    if (2 * t - 1 < n) look(2 * t - 1, mid, a0, e0, a1);
                }
#pragma unroll
                for (int k = 0; k < kCols; ++k) {
                    up[k] = a0[k];
                    mid[k] = a1[k];
                }
                mid_e = e1;
                if (++slot == ahead) slot = 0;
            }
#pragma unroll
            for (int k = 0; k < kCols; ++k)
                if (j0 + k < n) rows[j0 + k] = static_cast<uint16_t>(bi[k]);
            if (!kFull) cp_wait_all();
            __syncthreads();  // the staged rows are no longer read
        }
        // ... and with the pairs of neighbours that j owns, its best.
        for (int j = tid; j < n; j += NT) {
            auto at = [&](int p0, int q0) {
                const int u = X[p0], w = X[q0];
                return kFull ? mat[u * ld + w] : C[static_cast<size_t>(u) * ldc + w];
            };
            const int from[3] = {rows[j], prev(j), next(j)};
            unsigned long long v = kNone;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int i = from[q];
                if (i == kNobody || (q > 0 && !owns(ss[j], j, ss[i], i))) continue;
                v = min(v, key_of(at(prev(i), j) + at(next(i), j) + at(i, prev(j)) + at(i, next(j)) -
                                      ss[i] - ss[j] + adjacent(i, j), i, j));
            }
            bestof[j] = v;
        }
        smallest();  // (a thread reads what it wrote; the barrier is for the others)
        for (;;) {
            if (max_moves > 0 && moves >= max_moves) break;
            if (moves >= guard) {
                if (tid == 0 && a.status) atomicExch(a.status, DPSO_ERR_INTERNAL);
                break;
            }
            // Positions that are stale below the best exact value scan their
            // pairs, one warp each; then no stale value is below it.
            while (stale < exact) {
                for (int i0 = 0; i0 < n; i0 += NT) {
                    const int i = i0 + tid;
                    const unsigned long long v = i < n ? bestof[i] : kNone;
                    const bool take = v < exact && !(v & kExact);
                    const unsigned mask = __ballot_sync(0xffffffffu, take);
                    if (mask == 0) continue;
                    int k = lane == 0 ? atomicAdd(&s_rows, __popc(mask)) : 0;
                    k = __shfl_sync(0xffffffffu, k, 0) + __popc(mask & ((1u << lane) - 1));
                    if (take) rows[k] = static_cast<uint16_t>(i);
                }
                __syncthreads();
                const int nr = s_rows;
                for (int r = warp; r < nr; r += kW) {
                    const int i = rows[r], si = ss[i], k = 3 * warp;
                    const int xa = X[prev(i)], xi = X[i], xc = X[next(i)];
                    load_row(k, xa, lane, 32);
                    load_row(k + 1, xi, lane, 32);
                    load_row(k + 2, xc, lane, 32);
                    if (kRows) cp_wait_all();
                    __syncwarp();
                    unsigned long long best = kNone;
#pragma unroll 4
                    for (int j = lane; j < n; j += 32) {
                        const int xj = X[j], xm = X[prev(j)], xp = X[next(j)], sj = ss[j];
                        const int d = cost(k, xa, xj) + cost(k + 2, xc, xj) + cost(k + 1, xi, xm) +
                                      cost(k + 1, xi, xp) - si - sj;
                        if (d < 0 && owns(si, i, sj, j))
                            best = min(best, key_of(d + adjacent(i, j), i, j));
                    }
                    best = warp_min(best);
                    if (lane == 0) bestof[i] = best;
                    __syncwarp();  // the rows are no longer read
                }
                __syncthreads();
                if (tid == 0) s_rows = 0;
                smallest();
            }
            ++passes;
            if (exact == kNone) break;

            // Swap positions p0 < q0.  The six positions and the ten cities
            // around them, as they stand after the swap:
            const int p0 = static_cast<int>((exact >> 16) & 0x7fffu);
            const int q0 = static_cast<int>(exact & 0x7fffu);
            f += static_cast<int>(static_cast<uint32_t>(exact >> 32) ^ 0x80000000u);
            ++moves;
            const int xp0 = X[p0], xq0 = X[q0];
            auto after = [&](int k) { return k == p0 ? xq0 : (k == q0 ? xp0 : X[k]); };
            int six[6], city[kRowsStaged];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = h ? q0 : p0;
                six[3 * h] = prev(c);
                six[3 * h + 1] = c;
                six[3 * h + 2] = next(c);
                city[5 * h] = after(prev(prev(c)));
                city[5 * h + 4] = after(next(next(c)));
#pragma unroll
                for (int k = 0; k < 3; ++k) city[5 * h + 1 + k] = after(six[3 * h + k]);
            }
#pragma unroll
            for (int k = 0; k < kRowsStaged; ++k) load_row(k, city[k], tid, NT);
            __syncthreads();  // every thread has read X
            if (warp == 0) {
                if (lane == 0) {
                    X[p0] = static_cast<uint16_t>(xq0);
                    X[q0] = static_cast<uint16_t>(xp0);
                }
                __syncwarp();
                if (lane < 4) {  // the edges from p-1, p, q-1, q
                    const int c = lane < 2 ? p0 : q0, k = lane & 1 ? c : prev(c);
                    const int u = X[k], w = X[next(k)];
                    dd[k] = kFull ? mat[u * ld + w] : C[static_cast<size_t>(u) * ldc + w];
                }
                __syncwarp();
                if (lane < 6) {
                    const int c = lane < 3 ? p0 : q0;
                    const int k = lane % 3 == 0 ? prev(c) : (lane % 3 == 1 ? c : next(c));
                    ss[k] = dd[prev(k)] + dd[k];
                }
            }
            if (kRows) cp_wait_all();
            __syncthreads();

            // The pairs of the six positions.
            unsigned long long sixbest[6];
            int sd[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                sixbest[k] = kNone;
                sd[k] = ss[six[k]];
            }
            exact = kNone;
            stale = kNone;
            for (int j = tid; j < n; j += NT) {
                const int xj = X[j], xm = X[prev(j)], xp = X[next(j)], sj = ss[j];
                int d[6];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    int at[5], beside[3];
#pragma unroll
                    for (int k = 0; k < 5; ++k) at[k] = cost(5 * h + k, city[5 * h + k], xj);
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        beside[k] = cost(5 * h + k + 1, city[5 * h + k + 1], xm) +
                                    cost(5 * h + k + 1, city[5 * h + k + 1], xp);
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        d[3 * h + k] = at[k] + at[k + 2] + beside[k] - sd[3 * h + k] - sj;
                }
                bool in_six = false;
                unsigned long long mine = kNone;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const int c = six[k];
                    in_six = in_six || j == c;
                    if (d[k] < 0 && j != c) {
                        const unsigned long long key = key_of(d[k] + adjacent(c, j), c, j);
                        if (owns(sd[k], c, sj, j)) sixbest[k] = min(sixbest[k], key);
                        else mine = min(mine, key);
                    }
                }
                if (!in_six) {
                    unsigned long long v = bestof[j];
                    if (v != kNone) {
                        // its best was with one of the six: a lower bound now
                        const int i0 = static_cast<int>((v >> 16) & 0x7fffu);
                        const int j0 = static_cast<int>(v & 0x7fffu), c = i0 == j ? j0 : i0;
                        bool touched = false;
#pragma unroll
                        for (int k = 0; k < 6; ++k) touched = touched || c == six[k];
                        if (touched) v &= ~kExact;
                    }
                    v = min(v, mine);
                    bestof[j] = v;
                    if (v & kExact) exact = min(exact, v);
                    else stale = min(stale, v);
                }
            }
            exact = warp_min(exact);
            stale = warp_min(stale);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const unsigned long long v = warp_min(sixbest[k]);
                if (lane == 0) s_six[par][warp][k] = v;
            }
            if (lane == 0) {
                s_exact[par][warp] = exact;
                s_stale[par][warp] = stale;
            }
            __syncthreads();
            if (tid < 6) {
                unsigned long long v = kNone;
                for (int w = 0; w < kW; ++w) v = min(v, s_six[par][w][tid]);
                const int c = tid < 3 ? p0 : q0;
                bestof[tid % 3 == 0 ? prev(c) : (tid % 3 == 1 ? c : next(c))] = v;
            }
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                exact = min(exact, s_exact[par][w]);
                stale = min(stale, s_stale[par][w]);
#pragma unroll
                for (int k = 0; k < 6; ++k) exact = min(exact, s_six[par][w][k]);
            }
            par ^= 1;
            __syncthreads();
        }

        __syncthreads();
        for (int i = tid; i < n; i += NT) tour[i] = X[i];
        if (tid == 0) {
            const long long npairs = static_cast<long long>(n) * (n - 1) / 2;
            a.cost[p] = f;
            if (a.tour_passes) {
                a.tour_passes[p] = static_cast<unsigned int>(passes);
                a.tour_moves[p] = static_cast<unsigned int>(moves);
            } else {
                atomicAdd(a.pairs, static_cast<unsigned long long>(passes * npairs));
                atomicAdd(a.moves, static_cast<unsigned long long>(moves));
            }
            // (the node swap reports the plain scan's count)
            if (a.evals) atomicAdd(a.evals, static_cast<unsigned long long>(passes * npairs));
            s_pf = a.pbest ? a.pcost[p] : LLONG_MIN;
        }
        __syncthreads();
        if (a.pbest && f < s_pf) {
            uint16_t* pb = a.pbest + static_cast<size_t>(p) * a.ldt;
            for (int i = tid; i < n; i += NT) pb[i] = X[i];
            if (tid == 0) a.pcost[p] = f;
        }
        __syncthreads();
    }
}

template <int NT, Costs COSTS, int COLS, int CTAS>
cudaError_t launch_nt(const TwoOptBatch& b, int num_sms, cudaStream_t st) {
    auto* kern = node_swap_kernel<NT, COSTS, COLS, CTAS>;
    const size_t smem = swap_smem(b.max_n, NT / 32, COSTS);
    cudaError_t e = raise_smem_limit(kern, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int grid = max(1, min(b.total, per_sm * num_sms));
    kern<<<grid, NT, smem, st>>>(b);
    return cudaGetLastError();
}

}  // namespace

bool node_swap_fits(int n) { return n >= 3 && n <= kNodeSwapMaxN; }

namespace {

// Launch configurations: for tours of up to max_n viewpoints in launches of at
// most `few` tours per SM.  Measured on GB300 (whole call, random grid tours
// to local optimality, us; matrix = the whole matrix in shared memory):
//   n     tours  matrix 64 / 128 thr.  staged 64 / 96 / 128 thr.  from C, 256
//   64    1024   504 / 617             588 / 693 / 690            -
//   100   1024   1006 / 938            963 / 1206 / 1185          -
//   157   256    1009 / 948            1257 / 1162 / 1172         -
//   157   1024   2600 / 2444           1572 / 1952 / 2012         -
//   220   48     1584 / 1290           2095 / 1788 / 1620         -
//   400   256    -                     5367 / 4496 / 4448         -
//   400   512    -                     5883 / 4993 / 5495         -
//   400   1024   -                     7648 / 9351 / 9645         -
// and with the first pass by column blocks (one swap only in brackets; a block
// is NT * cols positions; 128 threads with 8, past 1024 viewpoints 12 of them):
//   620   600    -                     - / 8586 (345) / 8785 (402)      -
//   800   600    -                     - / 13586 (732) / 13703 (521)    -
//   999   150    -                     - / - / 14257 (390)        12451 (426)
//   999   300    -                     - / - / 16364 (486)        16612 (648)
//   999   600    -                     - / 36213 (1379) / 32533 (869)   32756 (1225)
//   1200  150    -                     - / - / 19800 (726, cols 8) 17786 (502)
//   1200  300    -                     - / - / 21406 (616)        24647 (768)
//   1200  600    -                     - / 50215 (1764) / 41118 (1150)  47664 (1452)
//   1500  150    -                     - / - / 29363 (905, cols 8) 27310 (623)
//   1500  300    -                     - / - / 32566 (799)        40545 (982)
//   1500  760    -                     - / - / 92768 (1841)       111130 (2235)
//   2000  300    -                     - / - / 175774 (cols 8)    153964
// From 800 to 1024 viewpoints, one tour per SM at most, C is the faster for whole
// descents and the staged rows for few swaps; the line lies where both agree.
// (The tiled kernel that scanned every pair took 46 ms for 512 tours at 400.)
struct SwapConfig {
    int max_n, few, threads;
    Costs costs;
    int cols, ctas;
};
constexpr int kAny = INT_MAX;
constexpr SwapConfig kConfigs[] = {
    {64, kAny, 64, kMatrix, 2, 10},     {100, kAny, 128, kMatrix, 2, 5},
    {160, 2, 128, kMatrix, 2, 5},       {220, 1, 128, kMatrix, 2, 5},
    {1024, 2, 128, kStaged, 8, 3},      {1500, 1, 256, kGlobal, 8, 2},
    {1500, 2, 128, kStaged, 12, 3},     {768, 5, 96, kStaged, 8, 5},
    {600, kAny, 64, kStaged, 8, 9},    {1024, kAny, 128, kStaged, 8, 5},
    {1500, kAny, 128, kStaged, 12, 3},  {kNodeSwapMaxN, kAny, 256, kGlobal, 8, 2},
};
constexpr int kNumConfigs = sizeof(kConfigs) / sizeof(kConfigs[0]);

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
    constexpr SwapConfig c = kConfigs[K];
    static_assert(swap_smem(c.max_n, c.threads / 32, c.costs) <= 224 * 1024, "does not fit");
    if (k == K) return launch_nt<c.threads, c.costs, c.cols, c.ctas>(b, num_sms, st);
    if constexpr (K + 1 < kNumConfigs) return launch_k<K + 1>(b, k, num_sms, st);
    else return cudaErrorInvalidValue;
}

}  // namespace

int node_swap_class(int n) { return find_config(n, 1 << 24, 1); }

cudaError_t launch_node_swap(const TwoOptBatch& b, int num_sms, cudaStream_t st) {
    if (!node_swap_fits(b.max_n)) return cudaErrorInvalidValue;
    return launch_k<0>(b, find_config(b.max_n, b.total, num_sms), num_sms, st);
}

}  // namespace dpso
