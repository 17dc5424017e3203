// Particle kernels of the enhanced DPSO (Phung et al., arXiv:1706.04399):
// tour fitness (Eq. min), initialisation (Sec. 3.2.1 and Fig. "pseudocode"),
// the velocity / position update (Eqs. velocity, position with the Sec. 3.1
// operators), random mutation (Sec. 3.2.2) and the pbest / gbest reduction.
//
// Velocities are stored as the label permutation their transposition list
// induces (x + v only depends on it).  With w = 1 the list is never truncated,
// so this is exact; with w < 1 the list is taken to be the canonical one of
// that permutation, (identity + v) - identity.
#include "common.cuh"

namespace dpso {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ unsigned long long warp_sum_u(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Warp-cooperative Eq. (min) for the tour x (closing edge included).
__device__ __forceinline__ long long tour_cost_warp(const int* __restrict__ C, int ldc, int n,
                                                    const uint16_t* x, int lane) {
    long long f = 0;
    // eight positions per lane per round, their gathers issued together
    for (int base = 0; base < n; base += 256) {
        int a[8], b[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = base + lane + 32 * k;
            a[k] = i < n ? x[i] : 0;
            b[k] = i < n ? x[i + 1 == n ? 0 : i + 1] : 0;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (base + lane + 32 * k < n) f += C[(size_t)a[k] * ldc + b[k]];
    }
    return warp_sum(f);
}

// ------------------------------------------------------------------ fitness
// Public entry: labels outside [0, n) contribute nothing (never read C).
// Bound by one L2 sector per gather (26 us for 4096 tours of 1992 at the rate
// of independent gathers).  `split` warps share a tour, as many as keep all
// tours resident and still have a round each, in blocks of one tour: few long
// tours are a chain of rounds otherwise, and blocks of eight tours leave the
// SMs uneven (4096 tours: four blocks on some, three on the others).  One warp
// per tour in blocks of eight, then now, random tours: 4096 x 1992 39.2 -> 35.0
// us, 512 x 1992 18.6 -> 10.4, 64 x 2999 26.0 -> 8.5, 1 x 2999 11.2 -> 6.2.
template <bool SPLIT>
__global__ void fitness_kernel(const int* __restrict__ C, int ldc, int n,
                               const uint16_t* __restrict__ tours, int ldt, int count,
                               long long* __restrict__ out, int split) {
    __shared__ long long part[8];
    if (!SPLIT) split = 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = (blockIdx.x * (blockDim.x >> 5) + warp) / split, sub = warp % split;
    long long f = 0;
    if (w < count) {
        const uint16_t* x = tours + (size_t)w * ldt;
        // A round covers 256 positions, eight per lane (lane, lane + 32, ...): the
        // labels of all eight edges are read first, then the eight gathers from C
        // are issued together, so every lane keeps eight L2 requests in flight.
        for (int base = 256 * sub; base < n; base += 256 * split) {
            int a[8], b[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = base + lane + 32 * k;
                a[k] = i < n ? x[i] : n;
                b[k] = i < n ? x[i + 1 == n ? 0 : i + 1] : n;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (a[k] < n && b[k] < n) f += C[(size_t)a[k] * ldc + b[k]];
        }
    }
    f = warp_sum(f);
    if (SPLIT) {
        if (lane == 0) part[warp] = f;
        __syncthreads();
        for (int q = 1; sub == 0 && q < split; ++q) f += part[warp + q];
    }
    if (w < count && sub == 0 && lane == 0) out[w] = f;
}

// ----------------------------------------------------- deterministic orders
// Back-and-forth order of variant v (Sec. 3.2.1): bit0 walks lines along
// columns instead of rows, bit1 visits lines in descending order, bit2 flips
// the direction of even lines; line L runs forward iff (L odd) == bit2.  The
// key of a viewpoint is (face, line', pos'); its rank among all keys is its
// place in the order.  Duplicate keys (duplicate tags) set *err.

struct Key {
    int face, line, pos;
};

__device__ __forceinline__ Key det_key(const int* tags, int i, int v) {
    const int face = tags[3 * i], row = tags[3 * i + 1], col = tags[3 * i + 2];
    const int line = (v & 1) ? col : row;
    const int pos = (v & 1) ? row : col;
    const bool backward = ((line & 1) != 0) != ((v & 4) != 0);
    return Key{face, (v & 2) ? -line : line, backward ? -pos : pos};
}

__device__ __forceinline__ bool key_less(const Key& a, const Key& b) {
    if (a.face != b.face) return a.face < b.face;
    if (a.line != b.line) return a.line < b.line;
    return a.pos < b.pos;
}

// Eight lanes count one viewpoint's rank, each over every eighth viewpoint: 38
// us at n = 1992 (243 with one thread per viewpoint).
__global__ void __launch_bounds__(256) det_orders_kernel(const int* __restrict__ tags, int n,
                                                         uint16_t* orders, int ldn, int* err) {
    const int v = blockIdx.y, part = threadIdx.x & 7;
    const int i = blockIdx.x * 32 + (threadIdx.x >> 3);
    __shared__ int st[3 * 512];
    Key mine{0, 0, 0};
    if (i < n) mine = det_key(tags, i, v);
    int rank = 0, same = 0;
    for (int j0 = 0; j0 < n; j0 += 512) {
        const int cnt = min(512, n - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < 3 * cnt; e += blockDim.x) st[e] = tags[3 * j0 + e];
        __syncthreads();
#pragma unroll 4
        for (int j = part; j < cnt; j += 8) {
            const Key o = det_key(st, j, v);
            rank += key_less(o, mine);
            same += o.face == mine.face && o.line == mine.line && o.pos == mine.pos;
        }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        rank += __shfl_xor_sync(kFull, rank, o);
        same += __shfl_xor_sync(kFull, same, o);
    }
    if (i < n && part == 0) {
        if (same != 1) atomicOr(err, 1);
        else orders[(size_t)v * ldn + rank] = static_cast<uint16_t>(i);
    }
}

// ----------------------------------------------------------- initialisation
// Particle p < n_det takes variant p%8 rotated left by floor(p/8); the others
// are Fisher-Yates shuffles of the identity: for i = n-1 .. 1, j = draw
// (n-1-i) of phase 1 bounded to [0, i], swap x[i], x[j].  v = identity,
// pbest = x.

// One warp per particle.  The draws are taken by all lanes; the swaps are one
// chain, run by lane 0 in shared memory: 43 us for 512 particles at n = 1992
// (1085 with one thread per particle on global memory).
__global__ void __launch_bounds__(32) init_particles_kernel(Consts k, SwarmDev d,
                                                            const uint16_t* __restrict__ orders,
                                                            int n_det) {
    extern __shared__ __align__(16) uint16_t sm[];
    const int p = blockIdx.x, lane = threadIdx.x, n = k.n;
    uint16_t* x = d.X + (size_t)p * k.ldn;
    uint16_t* pb = d.P + (size_t)p * k.ldn;
    uint16_t* v = d.V + (size_t)p * k.ldn;
    uint16_t* y = sm;            // the permutation
    uint16_t* with = sm + k.ldn;  // swap partner of position i
    if (lane == 0) d.order[p] = p;  // until the first generation ranks the particles
    if (p < n_det) {
        const uint16_t* ord = orders + (size_t)(p % 8) * k.ldn;
        const int rot = (p / 8) % n;
        for (int i = lane; i < n; i += 32) {
            const int at = i + rot;
            y[i] = ord[at < n ? at : at - n];
        }
    } else {
        for (int i = lane; i < n; i += 32) y[i] = static_cast<uint16_t>(i);
        for (int b0 = lane; 4 * b0 < n - 1; b0 += 32) {
            const Block4 b = philox(static_cast<uint32_t>(b0), p, 0, kPhaseInit, k.seed);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = n - 1 - (4 * b0 + q);
                if (i > 0)
                    with[i] = static_cast<uint16_t>(bounded(b.v[q], static_cast<uint32_t>(i + 1)));
            }
        }
        __syncwarp();
        if (lane == 0) {
            int j = with[n - 1];
            for (int i = n - 1; i > 0; --i) {
                const int nxt = with[i - 1];
                const uint16_t a = y[i], b = y[j];
                y[i] = b;
                y[j] = a;
                j = nxt;
            }
        }
    }
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
        const uint16_t yi = y[i];
        x[i] = yi;
        pb[i] = yi;
        v[i] = static_cast<uint16_t>(i);
    }
}

// ------------------------------------------------------------ gbest (init)

__device__ __forceinline__ unsigned long long fit_key(long long f, int p) {
    return (static_cast<unsigned long long>(f) << 16) | static_cast<unsigned long long>(p);
}

// Block-wide minimum of (fitness, index) keys; result valid in every thread.
__device__ unsigned long long block_min_key(const long long* __restrict__ f, int S) {
    __shared__ unsigned long long red[32];
    unsigned long long best = ~0ull;
    for (int p = threadIdx.x; p < S; p += blockDim.x) best = min(best, fit_key(f[p], p));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(kFull, best, o));
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[w] = best;
    __syncthreads();
    if (w == 0) {
        best = lane < (int)(blockDim.x >> 5) ? red[lane] : ~0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(kFull, best, o));
        if (lane == 0) red[0] = best;
    }
    __syncthreads();
    best = red[0];
    __syncthreads();
    return best;
}

__global__ void gbest_init_kernel(Consts k, SwarmDev d) {
    const unsigned long long key = block_min_key(d.F, k.S);
    const int bp = static_cast<int>(key & 0xffffu);
    for (int i = threadIdx.x; i < k.n; i += blockDim.x) d.G[i] = d.X[(size_t)bp * k.ldn + i];
    if (threadIdx.x == 0) {
        Ctl* c = d.ctl;
        c->gf = d.F[bp];
        c->gf_start = d.F[bp];
        c->t = 0;
        c->stall = 0;
        c->done = 0;
        c->run_two_opt = 0;
        c->queue = 0;
    }
}

// ---------------------------------------------------------------- the move
// Sec. 3.1 subtraction tgt - base read as the greedy left-to-right list: scan
// positions; where the running copy y differs from the target, swap the labels
// y[k] and tgt[k].  Written out, the list is a chain of n dependent steps; its
// effect is not.  With next(c) the place in the target of the label at
// position c of the base, the cycles of `next` are what the list sorts:
//  * Step k swaps unless k is the last place of its cycle that the scan
//    reaches, its largest; so the list has n - cycles transpositions, and the
//    first `cnt` of them end at the place K - 1 of the cnt-th k that is not
//    the largest of its cycle.
//  * After them y[k] = tgt[k] below K; at and past K, y[k] is the label at the
//    end of the chain k, next(k), next(next(k)), .. that runs through places
//    below K, i.e. the first c whose next(c) is not below K.
// Both are found by doubling: each round every place joins the stretch of its
// path it knows with the stretch that starts where its own ends (a place's
// end and largest member share a word, so a round may run in place).

// |tgt - base| and, with `next` left in `nxt`, what truncation needs: low half
// of big[c] unused afterwards, high half the largest place of c's cycle.
__device__ int subtract_cycles(const uint16_t* ix, const uint16_t* tgt, uint16_t* nxt,
                               uint32_t* big, int n, int lane) {
    for (int k = lane; k < n; k += 32) nxt[ix ? ix[tgt[k]] : tgt[k]] = static_cast<uint16_t>(k);
    __syncwarp();
    for (int c = lane; c < n; c += 32) big[c] = (static_cast<uint32_t>(c) << 16) | nxt[c];
    __syncwarp();
    for (int known = 1; known < n; known *= 2) {
        for (int c = lane; c < n; c += 32) {
            const uint32_t a = big[c], b = big[a & 0xffffu];
            big[c] = (max(a >> 16, b >> 16) << 16) | (b & 0xffffu);
        }
        __syncwarp();
    }
    int cnt = 0;
    for (int c = lane; c < n; c += 32) cnt += (big[c] >> 16) != static_cast<uint32_t>(c);
    return __reduce_add_sync(kFull, cnt);
}

// y = base after the first `cnt` of the `len` transpositions of tgt - base
// (base: x, or the identity when x is null); uses and overwrites nxt.
__device__ void subtract_apply(const uint16_t* x, const uint16_t* tgt, uint16_t* nxt,
                               const uint32_t* big, int cnt, int len, uint16_t* y, int n,
                               int lane) {
    int K = cnt >= len ? n : 0;
    if (cnt < len && cnt > 0) {
        int seen = 0;
        for (int c0 = 0; c0 < n; c0 += 32) {
            const int c = c0 + lane;
            const unsigned mask =
                __ballot_sync(kFull, c < n && (big[c] >> 16) != static_cast<uint32_t>(c));
            const int here = __popc(mask);
            if (seen + here >= cnt) {
                K = c0 + __fns(mask, 0, cnt - seen) + 1;
                break;
            }
            seen += here;
        }
    }
    if (K > 0 && K < n) {
        // (a cycle that lies wholly below K has no end and is not asked for)
        for (int c = lane; c < n; c += 32) {
            const int t = nxt[c], top = static_cast<int>(big[c] >> 16);
            nxt[c] = static_cast<uint16_t>(t >= K || top < K ? c : t);
        }
        __syncwarp();
        bool moved = true;  // a chain has fewer than n places: log2 n rounds at most
        for (int known = 1; known < n && moved; known *= 2) {
            bool mine = false;
            for (int c = lane; c < n; c += 32) {
                const uint16_t t = nxt[c], u = nxt[t];
                mine = mine || t != u;
                nxt[c] = u;
            }
            __syncwarp();
            moved = __any_sync(kFull, mine);
        }
    }
    for (int k = lane; k < n; k += 32) {
        if (k < K) {
            y[k] = tgt[k];
        } else {
            const uint16_t c = K > 0 ? nxt[k] : static_cast<uint16_t>(k);
            y[k] = x ? x[c] : c;
        }
    }
    __syncwarp();
}

// floor(c |v|) with c = phi * u / 2^32 in Q32 fixed point.
__device__ __forceinline__ int scaled_count(unsigned long long phi_q, uint32_t u, int len) {
    const unsigned long long cq = (phi_q * static_cast<unsigned long long>(u)) >> 32;
    return static_cast<int>((cq * static_cast<unsigned long long>(len)) >> 32);
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// One warp per particle of any instance in the batch: the truncated
// subtractions toward P and G (and of the velocity from the identity when the
// instance has w < 1) in shared memory, then v <- sigma_b o sigma_a o
// sigma_wv, x <- v o x, fitness, pbest, and in mutation generations the hash
// of the new tour.  Shared memory per warp: xs (x), ix (its inverse), nxt, ya,
// yb (x moved toward P and G) and big; with w < 1 also yw.  What bounds it:
// the log2 n rounds of the cycle search, shared-memory loads in random order:
// 167 us for 512 particles at n = 1992, 39 us for 1024 at n = 400 (the list
// run step by step by one lane: 343 and 78).
__global__ void move_kernel(BatchView b) {
    extern __shared__ __align__(16) uint16_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * (blockDim.x >> 5) + warp;
    if (g >= b.total) return;
    const int inst = find_inst(b.off, b.ninst, g);
    const int p = g - b.off[inst];
    const Consts k = b.desc[inst].k;
    const SwarmDev d = b.desc[inst].d;
    const Ctl* ctl = d.ctl;
    if (ctl->done) return;
    const int t = ctl->t + 1;
    const int n = k.n, ldn = k.ldn;
    const bool partial = k.w_q < (1ull << 32);
    uint16_t* xs = sm + static_cast<size_t>(warp) * b.arrays * b.max_ldn;
    uint32_t* big = reinterpret_cast<uint32_t*>(xs);  // two arrays wide
    xs += 2 * ldn;
    uint16_t* ix = xs + ldn;
    uint16_t* nxt = ix + ldn;
    uint16_t* ya = nxt + ldn;
    uint16_t* yb = ya + ldn;
    uint16_t* yw = yb + ldn;
    uint16_t* x = d.X + static_cast<size_t>(p) * ldn;
    uint16_t* v = d.V + static_cast<size_t>(p) * ldn;
    uint16_t* P = d.P + static_cast<size_t>(p) * ldn;

    for (int i = lane; i < n; i += 32) {
        const uint16_t xi = x[i];
        xs[i] = xi;
        ix[xi] = static_cast<uint16_t>(i);
    }
    __syncwarp();
    const Block4 r = philox(0, p, t, kPhaseVelocity, k.seed);
    {
        const int len = subtract_cycles(ix, P, nxt, big, n, lane);
        subtract_apply(xs, P, nxt, big, scaled_count(k.phi1_q, r.v[0], len), len, ya, n, lane);
    }
    {
        const int len = subtract_cycles(ix, d.G, nxt, big, n, lane);
        subtract_apply(xs, d.G, nxt, big, scaled_count(k.phi2_q, r.v[1], len), len, yb, n, lane);
    }
    if (partial) {
        if (k.w_q == 0) {
            for (int l = lane; l < n; l += 32) yw[l] = static_cast<uint16_t>(l);
        } else {
            const int len = subtract_cycles(nullptr, v, nxt, big, n, lane);
            const int kw = static_cast<int>((k.w_q * static_cast<unsigned long long>(len)) >> 32);
            subtract_apply(nullptr, v, nxt, big, kw, len, yw, n, lane);
        }
        __syncwarp();
    }

    // sigma_a(m) = ya[ix[m]], sigma_b(m) = yb[ix[m]]; new velocity into nxt.
    for (int l = lane; l < n; l += 32) {
        uint16_t m = partial ? yw[l] : v[l];
        m = ya[ix[m]];
        m = yb[ix[m]];
        nxt[l] = m;
        v[l] = m;
    }
    __syncwarp();
    const bool hashed = mutation_due(k, ctl);
    unsigned long long h = 0;
    for (int i = lane; i < n; i += 32) {
        const uint16_t xn = nxt[xs[i]];
        ya[i] = xn;
        x[i] = xn;
        if (hashed) h += mix64((static_cast<unsigned long long>(i) << 16) | xn);
    }
    __syncwarp();
    const long long f = tour_cost_warp(d.C, k.ldc, n, ya, lane);
    if (hashed) {
        h = warp_sum_u(h);
        if (lane == 0) d.hash[p] = h;
    }
    const long long pf = d.PF[p];  // read by every lane before lane 0 may write it
    __syncwarp();
    if (lane == 0) d.F[p] = f;
    if (f < pf) {
        for (int i = lane; i < n; i += 32) P[i] = ya[i];
        if (lane == 0) d.PF[p] = f;
    }
}

// ---------------------------------------------------------------- mutation
// Sec. 3.2.2: order the particles by (fitness, index); a particle equal (as a
// tour array) to an earlier one in that order is a duplicate; the first
// ceil(S/3) non-duplicates are kept; every other particle gets mut_swaps
// swaps of two distinct positions (phase-3 draws 2q, 2q+1), an empty
// velocity, a new fitness and a pbest update.  Equal tours have equal
// fitness, so "earlier" means equal fitness and a smaller index; a 64-bit
// hash (the move kernel's) screens the candidates and full compares decide.

// Global particle g of the batch -> (instance, particle); false when g is past
// the batch or the instance does not mutate in its running generation.
__device__ __forceinline__ bool mut_item(const BatchView& b, int g, Consts& k, SwarmDev& d,
                                         int& p) {
    if (g >= b.total) return false;
    const int inst = find_inst(b.off, b.ninst, g);
    p = g - b.off[inst];
    k = b.desc[inst].k;
    d = b.desc[inst].d;
    return mutation_due(k, d.ctl);
}

__device__ bool tours_equal(const uint16_t* a, const uint16_t* b, int ldn) {
    const uint4* va = reinterpret_cast<const uint4*>(a);
    const uint4* vb = reinterpret_cast<const uint4*>(b);
    for (int i = 0; i < ldn / 8; ++i) {
        const uint4 u = va[i], w = vb[i];
        if (u.x != w.x || u.y != w.y || u.z != w.z || u.w != w.w) return false;
    }
    return true;
}

// One warp per particle, the lanes over the others: 12 and 15 us for 1024
// particles in this kernel and the next (83 and 91 with one thread each).
__global__ void mut_dup_kernel(BatchView b) {
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    Consts k;
    SwarmDev d;
    int p;
    if (!mut_item(b, g, k, d, p)) return;
    const long long fp = d.F[p];
    const unsigned long long hp = d.hash[p];
    bool dup = false;
#pragma unroll 4
    for (int q = lane; q < p; q += 32)
        if (d.F[q] == fp && d.hash[q] == hp)
            dup = dup || tours_equal(d.X + static_cast<size_t>(q) * k.ldn,
                                     d.X + static_cast<size_t>(p) * k.ldn, k.ldn);
    dup = __any_sync(kFull, dup);
    if (lane == 0) d.dup[p] = dup;
}

__global__ void mut_kept_kernel(BatchView b) {
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    Consts k;
    SwarmDev d;
    int p;
    if (!mut_item(b, g, k, d, p)) return;
    const long long fp = d.F[p];
    int rank = 0;
#pragma unroll 4
    for (int q = lane; q < k.S; q += 32)
        rank += !d.dup[q] && (d.F[q] < fp || (d.F[q] == fp && q < p));
    rank = __reduce_add_sync(kFull, rank);
    if (lane == 0) d.kept[p] = !d.dup[p] && rank < (k.S + 2) / 3;
}

__global__ void mut_apply_kernel(BatchView b) {
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    Consts k;
    SwarmDev d;
    int p;
    if (!mut_item(b, g, k, d, p) || d.kept[p]) return;
    const int t = d.ctl->t + 1, n = k.n;
    uint16_t* x = d.X + static_cast<size_t>(p) * k.ldn;
    if (lane == 0) {
        for (int q = 0; q < k.mut_swaps; ++q) {
            const uint32_t di = 2u * q, dj = 2u * q + 1u;
            const Block4 bi = philox(di >> 2, p, t, kPhaseMutation, k.seed);
            const Block4 bj = philox(dj >> 2, p, t, kPhaseMutation, k.seed);
            const int i = static_cast<int>(bounded(bi.v[di & 3u], static_cast<uint32_t>(n)));
            int j = static_cast<int>(bounded(bj.v[dj & 3u], static_cast<uint32_t>(n - 1)));
            j += (j >= i);
            const uint16_t tmp = x[i];
            x[i] = x[j];
            x[j] = tmp;
        }
    }
    __syncwarp();
    uint16_t* v = d.V + static_cast<size_t>(p) * k.ldn;
    for (int i = lane; i < n; i += 32) v[i] = static_cast<uint16_t>(i);
    const long long f = tour_cost_warp(d.C, k.ldc, n, x, lane);
    const long long pf = d.PF[p];
    __syncwarp();
    if (lane == 0) d.F[p] = f;
    if (f < pf) {
        uint16_t* P = d.P + static_cast<size_t>(p) * k.ldn;
        for (int i = lane; i < n; i += 32) P[i] = x[i];
        if (lane == 0) d.PF[p] = f;
    }
}

// ------------------------------------------------------------------ gbest
// Fig. "pseudocode": the particle with the smallest (pbest fitness, index)
// replaces the gbest only on strict improvement.  Pass 0 runs after the
// particle loop (and mutation) and schedules the edge exchange; pass 1 runs
// after the exchange.  The generation is closed (history, stall counter,
// generation counter, stop flag) by the last pass that runs.  One block per
// instance of the batch.

__global__ void gbest_kernel(BatchView b, int second, unsigned int* queue, int queues) {
    if (blockIdx.x == 0)
        for (int q = threadIdx.x; q < queues; q += blockDim.x) queue[q] = 0;
    const Consts k = b.desc[blockIdx.x].k;
    const SwarmDev d = b.desc[blockIdx.x].d;
    Ctl* c = d.ctl;
    if (c->done) return;
    if (second && !c->run_two_opt) return;
    const bool mut_iter = mutation_due(k, c);
    const unsigned long long key = block_min_key(d.PF, k.S);
    const long long best = static_cast<long long>(key >> 16);
    const int bp = static_cast<int>(key & 0xffffu);
    const long long gf_old = c->gf;
    __syncthreads();
    if (best < gf_old)
        for (int i = threadIdx.x; i < k.n; i += blockDim.x)
            d.G[i] = d.P[static_cast<size_t>(bp) * k.ldn + i];
    if (threadIdx.x != 0) return;
    const int t = c->t + 1;
    if (!second) c->gf_start = gf_old;
    if (best < gf_old) c->gf = best;
    if (t <= c->hist_cap) c->hist[t - 1] = c->gf;
    else c->status = DPSO_ERR_INTERNAL;
    const bool improved = c->gf < c->gf_start;
    if (!second) {
        const bool run = (k.flags & DPSO_FLAG_TWO_OPT) && !improved && (k.trigger == 0 || mut_iter);
        c->run_two_opt = run ? 1 : 0;
        if (run) {
            c->runs += 1;
            return;
        }
    } else {
        c->run_two_opt = 0;
    }
    c->stall = improved ? 0 : c->stall + 1;
    c->t = t;
    if (k.stall_limit > 0 && c->stall >= k.stall_limit) c->done = 1;
}

// ------------------------------------------------------ exchange order
// order[r] = the particle of rank r by (fitness descending, index ascending)
// within each instance, so the edge exchange starts the tours expected to
// need the most passes first (longest-processing-time-first list
// scheduling; the post-move fitness is the estimate).  One warp per particle:
// 6 us for 1024 (17 with one thread each).
__global__ void rank_cost_kernel(BatchView b) {
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (g >= b.total) return;
    const int inst = find_inst(b.off, b.ninst, g);
    const SwarmDesc& ds = b.desc[inst];
    const int p = g - b.off[inst], S = ds.k.S;
    const long long* __restrict__ F = ds.d.F;
    const long long mine = F[p];
    int rank = 0;
#pragma unroll 4
    for (int q = lane; q < S; q += 32) {
        const long long o = F[q];
        rank += (o > mine) | ((o == mine) & (q < p));
    }
    rank = __reduce_add_sync(kFull, rank);
    if (lane == 0) ds.d.order[rank] = p;
}

__global__ void philox_draws_kernel(unsigned long long seed, uint32_t phase, uint32_t iter,
                                    uint32_t particle, int count, uint32_t* out) {
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d < count) out[d] = draw(seed, phase, iter, particle, static_cast<uint32_t>(d));
}

// Warps per block of the move kernel: up to 8, within 200 KB of shared memory.
int move_warps(const BatchView& b) {
    const size_t per = static_cast<size_t>(b.arrays) * b.max_ldn * sizeof(uint16_t);
    int w = 8;
    while (w > 1 && per * w > 200 * 1024) --w;
    return w;
}

}  // namespace

cudaError_t launch_fitness(const int* C, int ldc, int n, const uint16_t* tours, int ldt, int count,
                           long long* out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    int split = 1;
    // A tour of one round is not split, and eight of them share a block (4096
    // tours of 64: 5.5 us, in blocks of two 5.8); so do tours of two rounds, and
    // tours enough for eight blocks of eight per SM, where the number of blocks
    // counts more than uneven SMs (60000 tours of 257: 45.7 us in blocks of two,
    // 37.2 in blocks of eight).  Where C does not fit L2 and there are tours
    // enough to fill the chip, splitting loses a little (1000 tours of 8192: 110
    // us whole, 117 split; 300 tours 72 and 40).
    int threads = 256;
    if (n > 256) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        while (split < 8 && 256 * split < n && 2ll * split * count <= 64 * sms) split *= 2;
        if (split > 1 || (n > 512 && count < 64 * sms)) threads = max(64, 32 * split);
    }
    const int per = threads / (32 * split);
    auto* kern = split > 1 ? fitness_kernel<true> : fitness_kernel<false>;
    kern<<<(count + per - 1) / per, threads, 0, st>>>(C, ldc, n, tours, ldt, count, out, split);
    return cudaGetLastError();
}

cudaError_t launch_det_orders(const int* tags, int n, uint16_t* orders, int ldn, int* err,
                              cudaStream_t st) {
    dim3 grid((n + 31) / 32, 8);
    det_orders_kernel<<<grid, 256, 0, st>>>(tags, n, orders, ldn, err);
    return cudaGetLastError();
}

cudaError_t launch_init_particles(const Consts& k, const SwarmDev& d, const uint16_t* orders,
                                  int n_det, cudaStream_t st) {
    const size_t smem = 2 * static_cast<size_t>(k.ldn) * sizeof(uint16_t);  // at most 32 KB
    init_particles_kernel<<<k.S, 32, smem, st>>>(k, d, orders, n_det);
    return cudaGetLastError();
}

cudaError_t launch_gbest_init(const Consts& k, const SwarmDev& d, cudaStream_t st) {
    gbest_init_kernel<<<1, 1024, 0, st>>>(k, d);
    return cudaGetLastError();
}

cudaError_t launch_move(const BatchView& b, cudaStream_t st) {
    if (b.total <= 0) return cudaSuccess;
    const int w = move_warps(b);
    const size_t smem = static_cast<size_t>(b.arrays) * b.max_ldn * sizeof(uint16_t) * w;
    const cudaError_t e = raise_smem_limit(move_kernel, smem);
    if (e != cudaSuccess) return e;
    move_kernel<<<(b.total + w - 1) / w, 32 * w, smem, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_mutation(const BatchView& b, cudaStream_t st) {
    if (b.total <= 0) return cudaSuccess;
    const int wb = (b.total * 32 + 255) / 256;
    mut_dup_kernel<<<wb, 256, 0, st>>>(b);
    mut_kept_kernel<<<wb, 256, 0, st>>>(b);
    mut_apply_kernel<<<wb, 256, 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_rank_cost(const BatchView& b, cudaStream_t st) {
    if (b.total <= 0) return cudaSuccess;
    rank_cost_kernel<<<(b.total * 32 + 255) / 256, 256, 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_gbest(const BatchView& b, int second, unsigned int* queue, int queues,
                         cudaStream_t st) {
    if (b.ninst <= 0) return cudaSuccess;
    const int threads = min(1024, max(128, round_up(b.max_S, 32)));
    gbest_kernel<<<b.ninst, threads, 0, st>>>(b, second, queue, queues);
    return cudaGetLastError();
}

cudaError_t launch_philox_draws(unsigned long long seed, uint32_t phase, uint32_t iter,
                                uint32_t particle, int count, uint32_t* out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    philox_draws_kernel<<<(count + 255) / 256, 256, 0, st>>>(seed, phase, iter, particle, count,
                                                             out);
    return cudaGetLastError();
}

}  // namespace dpso
