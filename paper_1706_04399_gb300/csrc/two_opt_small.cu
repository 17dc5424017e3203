// Edge exchange of Sec. 3.2.3 (best-improvement 2-opt to 2-optimality) for
// short tours: every pass scans every pair, with the whole cost matrix in
// shared memory.
//
// Same mathematics and tie order as two_opt_list.cu.  A short tour's passes
// are bound by latency, not by the pairs they evaluate: a pass here is one
// scan, one reduction and one reversal with two block barriers between them
// and no access to L2, where the list kernel takes several dependent steps.
//
// The rows i = 0..n-3 hold n-2-i pairs each; row r and row n-3-r together hold
// n-1, so the pairs are numbered along such folded rows and dealt out evenly:
// a thread has the same at most kPairs pairs in every pass and keeps their
// positions in registers.  It gathers for half of them at once, and for the
// other half only where the pair's two edges together could gain more than its
// best so far (costs are not negative).  Records rec[p] =
// {x_p | x_p+1 << 16, C[x_p][x_p+1]} bring both labels and the edge of a
// position in one 8-byte load.  What bounds it: the chain of a pass when few
// tours share an SM, else the two random shared-memory gathers per pair.
#include <climits>

#include "tiled_common.cuh"

namespace dpso {
namespace {

using namespace tiled;

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr(smem)), "l"(gmem)
                 : "memory");
}

// Odd pitch: the cities of a column fall on different banks.
__host__ __device__ constexpr int small_ld(int n) { return n | 1; }

constexpr size_t small_smem(int n) {
    return (static_cast<size_t>(n) * sizeof(int2) + static_cast<size_t>(n) * small_ld(n) * 4 + 15) /
           16 * 16;
}

constexpr int kPairs = 8;  // pairs a thread scans

// Folded rows of n - 1 columns: (n - 1) / 2 of them.
constexpr bool small_fits(int n, int threads) {
    return n >= 3 && ((n - 1) / 2) * (n - 1) <= threads * kPairs;
}

template <int NT>
__global__ void __launch_bounds__(NT) two_opt_small_kernel(TwoOptBatch b) {
    constexpr int kW = NT / 32;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned long long s_key[2][kW];
    __shared__ unsigned s_evals[kW];
    __shared__ int s_item;
    __shared__ long long s_pf;
    int2* const rec = reinterpret_cast<int2*>(smraw);
    int* const mat = reinterpret_cast<int*>(rec + b.max_n);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

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
        const int n = a.n, ld = small_ld(n);
        const int* __restrict__ const C = a.C;
        const int ldc = a.ldc, max_moves = a.max_moves;
        uint16_t* const tour = a.tours + static_cast<size_t>(p) * a.ldt;
        for (int r = warp; r < n; r += kW)
            for (int c = lane; c < n; c += 32)
                cp_async4(&mat[r * ld + c], C + static_cast<size_t>(r) * ldc + c);
        for (int i = tid; i < n; i += NT) {
            const int u = tour[i], w = tour[i + 1 == n ? 0 : i + 1];
            rec[i] = make_int2(u | (w << 16), C[static_cast<size_t>(u) * ldc + w]);
        }
        // this thread's pairs, i << 16 | j (~0: none; (0, n-1) is no pair)
        unsigned ij[kPairs];
#pragma unroll
        for (int q = 0; q < kPairs; ++q) {
            const int k = tid + q * NT, r = k / (n - 1), c = k - r * (n - 1);
            const bool lo = c < n - 2 - r;
            const int i = lo ? r : n - 3 - r, j = lo ? r + 2 + c : c + 1;
            const bool in = 2 * r < n - 3 || (2 * r == n - 3 && lo);
            ij[q] = in && (i != 0 || j != n - 1) ? (i << 16) | j : 0xffffffffu;
        }
        long long f = a.cost[p];
        int moves = 0, passes = 0, par = 0;
        unsigned evals = 0;
        const int guard = 1000 + 100 * n;
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();

        for (;;) {
            if (max_moves > 0 && moves >= max_moves) break;
            if (moves >= guard) {
                if (tid == 0 && a.status) atomicExch(a.status, DPSO_ERR_INTERNAL);
                break;
            }
            int bd = 0;  // only improving moves count
            unsigned bij = 0xffffffffu;
#pragma unroll
            for (int h = 0; h < kPairs; h += kPairs / 2) {
                int d[kPairs / 2];
                bool ok[kPairs / 2];
#pragma unroll
                for (int q = 0; q < kPairs / 2; ++q) {
                    const unsigned v = ij[h + q];
                    ok[q] = v != 0xffffffffu;
                    const int2 ri = rec[ok[q] ? v >> 16 : 0], rj = rec[ok[q] ? v & 0xffff : 0];
                    const int gain = ri.y + rj.y;
                    ok[q] = ok[q] && gain >= -bd;  // (an equal delta still meets the tie order)
                    if (ok[q])
                        d[q] = mat[(ri.x & 0xffff) * ld + (rj.x & 0xffff)] +
                               mat[(ri.x >> 16) * ld + (rj.x >> 16)] - gain;
                }
#pragma unroll
                for (int q = 0; q < kPairs / 2; ++q) {
                    evals += ok[q];
                    if (ok[q] && (d[q] < bd || (d[q] == bd && ij[h + q] < bij && bd < 0))) {
                        bd = d[q];
                        bij = ij[h + q];
                    }
                }
            }
            const int md = __reduce_min_sync(0xffffffffu, bd);
            const unsigned mij = __reduce_min_sync(0xffffffffu, bd == md ? bij : 0xffffffffu);
            if (lane == 0)
                s_key[par][warp] =
                    (static_cast<unsigned long long>(static_cast<uint32_t>(md) ^ 0x80000000u) << 32) |
                    mij;
            __syncthreads();
            unsigned long long best = s_key[par][0];
#pragma unroll
            for (int w = 1; w < kW; ++w) best = min(best, s_key[par][w]);
            par ^= 1;
            ++passes;
            const int d = static_cast<int>(static_cast<uint32_t>(best >> 32) ^ 0x80000000u);
            if (d >= 0) break;
            const int bi = static_cast<int>((best >> 16) & 0xffffu);
            const int bj = static_cast<int>(best & 0xffffu);
            f += d;
            ++moves;
            // the edges strictly between turn round; the two new ones join
            for (int q = tid; q < (bj - bi) / 2; q += NT) {
                const int p0 = bi + 1 + q, p1 = bj - 1 - q;
                const int2 a0 = rec[p0], a1 = rec[p1];
                rec[p0] = make_int2(static_cast<int>(__byte_perm(a1.x, 0, 0x1032)), a1.y);
                rec[p1] = make_int2(static_cast<int>(__byte_perm(a0.x, 0, 0x1032)), a0.y);
            }
            if (tid == NT - 1) {
                const int2 ri = rec[bi], rj = rec[bj];
                const int xa = ri.x & 0xffff, xa1 = ri.x >> 16, xb = rj.x & 0xffff, xb1 = rj.x >> 16;
                rec[bi] = make_int2(xa | (xb << 16), mat[xa * ld + xb]);
                rec[bj] = make_int2(xa1 | (xb1 << 16), mat[xa1 * ld + xb1]);
            }
            __syncthreads();
        }

        __syncthreads();
        for (int i = tid; i < n; i += NT) tour[i] = static_cast<uint16_t>(rec[i].x & 0xffff);
        evals = __reduce_add_sync(0xffffffffu, evals);
        if (lane == 0) s_evals[warp] = evals;
        if (tid == 0) s_pf = a.pbest ? a.pcost[p] : LLONG_MIN;
        __syncthreads();
        if (a.pbest && f < s_pf) {
            uint16_t* pb = a.pbest + static_cast<size_t>(p) * a.ldt;
            for (int i = tid; i < n; i += NT) pb[i] = static_cast<uint16_t>(rec[i].x & 0xffff);
            if (tid == 0) a.pcost[p] = f;
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
            if (a.evals) {
                unsigned long long e = 0;
                for (int w = 0; w < kW; ++w) e += s_evals[w];
                atomicAdd(a.evals, e);
            }
        }
        __syncthreads();
    }
}

template <int NT>
cudaError_t launch_nt(const TwoOptBatch& b, int num_sms, cudaStream_t st) {
    auto* kern = two_opt_small_kernel<NT>;
    const size_t smem = small_smem(b.max_n);
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

// Threads per tour for tours of up to n viewpoints; 0: too long for this kernel.
int two_opt_small_threads(int n) {
    for (int threads : {128, 256, 512})
        if (small_fits(n, threads)) return threads;
    return 0;
}

cudaError_t launch_two_opt_small(const TwoOptBatch& b, int num_sms, cudaStream_t st) {
    switch (two_opt_small_threads(b.max_n)) {
        case 128: return launch_nt<128>(b, num_sms, st);
        case 256: return launch_nt<256>(b, num_sms, st);
        case 512: return launch_nt<512>(b, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace dpso
