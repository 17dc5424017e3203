// Edge-cost matrix of the extended TSP (Sec. 2.3): straight-segment Euclidean
// length in millimetres, rounded to nearest in FP64, plus a penalty when the
// closed segment meets an obstacle box grown by the UAV radius.
//
// Every FP64 step is an explicit round-to-nearest intrinsic, so nothing is
// contracted into an FMA and sqrt / divide are the correctly rounded IEEE
// operations; the file is also built with -fmad=false.
//
// FP64 is scarce here (about one multiply-add per SM and clock for each 32 in
// FP32), and the slab test divides six times per pair and box.  A filter in
// FP32 with an error bound decides nearly every (pair, box); the FP64 test runs
// on what it leaves open, so the matrix is that of the FP64 test alone.  At
// n = 1992 with 20 boxes the kernel took 3.32 ms without the filter, 0.18 with
// it and FP64 lengths, and 0.13 with lengths in pairs of FP32 numbers (below),
// FP64 only next to a rounding tie.  Boxes that lie beside all of a tile's
// points are dropped per tile (whole call 153 -> 128 us); what is left is the
// filter on the others.
#include <math.h>

#include "common.cuh"

namespace dpso {
namespace {

// Closed segment p + t (q - p), t in [0, 1], against the closed box
// [lo - r, hi + r] (slab test, axes x, y, z in order).
__device__ bool segment_blocked(const double p[3], const double q[3], const double* box,
                                double r) {
    double tmin = 0.0, tmax = 1.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double lo = __dsub_rn(box[k], r);
        const double hi = __dadd_rn(box[3 + k], r);
        const double d = __dsub_rn(q[k], p[k]);
        if (d == 0.0) {
            if (p[k] < lo || p[k] > hi) return false;
        } else {
            double t1 = __ddiv_rn(__dsub_rn(lo, p[k]), d);
            double t2 = __ddiv_rn(__dsub_rn(hi, p[k]), d);
            if (t1 > t2) {
                const double tt = t1;
                t1 = t2;
                t2 = tt;
            }
            if (t1 > tmin) tmin = t1;
            if (t2 < tmax) tmax = t2;
        }
    }
    return tmin <= tmax;
}

constexpr int kTile = 32;
constexpr int kBoxes = 256;  // boxes staged at once

// FP32 view of a pair on one axis: p, 1 / (q - p), and the smaller and larger
// of p and q.
struct Axis {
    float p, inv, a, b;
};

// The FP32 filter for one box: 0 free, 1 blocked, 2 open.
//
// With M the largest magnitude of the pair's and the box's coordinates, every
// difference of two of them is off by at most 2^-22 M (both rounded to FP32,
// and the difference rounded); E is twice that and more.
//  * An axis on which both ends lie E beyond the box: free.  (The FP64 test
//    finds t > 1 or t < 0 there, by at least E / |d| >= 2^-22.)
//  * An axis with |d| < 64 E, d = 0 among them: no constraint when both ends
//    lie E inside, else open.
//  * The other axes: t = (side - p) / d is off by at most E / |d| where it is
//    near [0, 1], plus its own rounding; when the ends of the common interval
//    are further apart than twice the largest such error, their order is that
//    of the FP64 values, whose error is some 2^-52.
// Infinities and NaN (coordinates past FP32) leave every comparison false: open.
__device__ __forceinline__ int filter_box(const Axis (&ax)[3], const float (&lo)[3],
                                          const float (&hi)[3], float E) {
    bool out = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) out = out || ax[k].b < lo[k] - E || ax[k].a > hi[k] + E;
    if (out) return 0;
    float tmin = 0.f, tmax = 1.f, worst_inv = 0.f;
    bool open = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (ax[k].b - ax[k].a >= 64.f * E) {
            const float t1 = (lo[k] - ax[k].p) * ax[k].inv, t2 = (hi[k] - ax[k].p) * ax[k].inv;
            tmin = fmaxf(tmin, fminf(t1, t2));
            tmax = fminf(tmax, fmaxf(t1, t2));
            worst_inv = fmaxf(worst_inv, fabsf(ax[k].inv));
        } else {
            open = open || !(ax[k].a > lo[k] + E && ax[k].b < hi[k] - E);
        }
    }
    const float gap = tmax - tmin, w = 2.f * (E * worst_inv + 0x1p-19f);
    if (gap < -w) return 0;
    return !open && gap > w ? 1 : 2;
}

// A coordinate as the sum of two FP32 numbers (off by at most 2^-48 of it).
struct Split {
    float hi, lo;
};

__device__ __forceinline__ Split split(double v) {
    const float hi = static_cast<float>(v);
    return Split{hi, static_cast<float>(__dsub_rn(v, static_cast<double>(hi)))};
}

// 1000 |q - p| rounded to the nearest integer, in pairs of FP32 numbers (sums
// with their rounding error after Knuth and, for ordered terms, Dekker, products
// with theirs by FMA, the root by one Newton correction of the reciprocal square
// root), where the result is not near a tie; -1: not decided.  With M the largest coordinate magnitude,
// the differences are off by some 2^-46 M and everything after by some 2^-44
// of itself, so the length r in mm by less than (r + 1000 M) 2^-40; a tie
// closer than 2^8 times that (and 2^-20) is left to FP64, whose own error is
// far below.  Lengths past 2^22 mm, and anything not finite, are left too.
__device__ __forceinline__ int length_mm(const Split (&p)[3], const Split (&q)[3], float mag) {
    float sh = 0.f, sl = 0.f;  // the sum of squares
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = __fsub_rn(q[k].hi, p[k].hi);  // d = a + e, normalised to h + l
        const float bb = __fsub_rn(a, q[k].hi);
        const float e = __fadd_rn(
            __fsub_rn(__fsub_rn(q[k].hi, __fsub_rn(a, bb)), __fadd_rn(p[k].hi, bb)),
            __fsub_rn(q[k].lo, p[k].lo));
        const float h = __fadd_rn(a, e), l = __fsub_rn(e, __fsub_rn(h, a));
        const float m = __fmul_rn(h, h);
        const float ml = __fmaf_rn(2.f * h, l, __fmaf_rn(h, h, -m));
        const float t = __fadd_rn(sh, m);  // sh + m and its error
        const float tb = __fsub_rn(t, sh);
        const float te = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, tb)), __fsub_rn(m, tb));
        sl = __fadd_rn(sl, __fadd_rn(te, ml));
        sh = t;
    }
    if (!(sh < 1.76e7f)) return -1;  // 4.19 km squared, as (2^22 mm)^2
    if (sh < 1e-20f) return sh == 0.f && sl == 0.f ? 0 : -1;
    const float y = rsqrtf(sh);
    const float r0 = __fmul_rn(sh, y);
    const float res = __fadd_rn(__fmaf_rn(-r0, r0, sh), sl);  // (s - r0^2), r0 within 2^-21
    const float r1 = __fmul_rn(res, __fmul_rn(0.5f, y));
    // one more step for the remainder's own square
    const float r2 = __fmaf_rn(-__fmul_rn(r1, r1), __fmul_rn(0.5f, y), r1);
    const float vh = __fmul_rn(r0, 1000.f);
    const float vl = __fadd_rn(__fmaf_rn(r0, 1000.f, -vh), __fmul_rn(r2, 1000.f));
    const float n = rintf(vh);
    const float f = __fadd_rn(__fsub_rn(vh, n), vl);  // the distance from n, small
    const float g = rintf(f);
    const float away = fabsf(__fsub_rn(fabsf(__fsub_rn(f, g)), 0.5f));
    if (!(away > 0x1p-20f + (vh + 1000.f * mag) * 0x1p-32f)) return -1;
    return static_cast<int>(n) + static_cast<int>(g);
}

// One thread per (i, j) with i < j inside 32 x 32 tiles of the upper triangle,
// four pairs per thread; boxes are staged in shared memory in chunks.  The
// tile is mirrored through shared memory, so both halves are written in rows.
// Flags non-finite coordinates and inverted boxes (bit 0 of *err) and entries
// above DPSO_COST_MAX (bit 1).
__global__ void __launch_bounds__(kTile * 8, 2) cost_matrix_kernel(
    const double* __restrict__ xyz, int n, const double* __restrict__ boxes, int m, double r,
    int penalty, int* __restrict__ C, int ldc, int* err) {
    const int bi = blockIdx.y * kTile, bj = blockIdx.x * kTile;
    if (bj + kTile <= bi) return;  // strictly below the diagonal
    __shared__ double sbox[kBoxes * 6];
    __shared__ float slo[kBoxes][3], shi[kBoxes][3], smag[kBoxes];
    __shared__ unsigned char sidx[kBoxes];  // the kept boxes' places in sbox
    __shared__ int tile[kTile][kTile + 1];
    __shared__ Split rows[kTile][3];  // the tile's row points
    __shared__ float hull[2][2][3];   // of the row and the column points: lowest, highest
    // Boxes of the chunk that meet the hull of both, by the chunk's parity: a
    // warp may clear the next chunk's count while another has yet to read this
    // chunk's; this one's is cleared again two chunks on, after the barriers of
    // the one between.
    __shared__ int kept[2];
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    const int tid = ty * kTile + tx;
    const int j = bj + tx;
    double q[3] = {0, 0, 0};
    float qf[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (j < n) q[k] = xyz[3 * (size_t)j + k];
        qf[k] = static_cast<float>(q[k]);
    }
    bool bad = false;
    if (tid < 3 * kTile && bi + tid / 3 < n) {
        const double v = xyz[3 * (size_t)bi + tid];
        bad = !isfinite(v);  // (every point is a row of its diagonal tile)
        rows[tid / 3][tid % 3] = split(v);
    }
    if (m > 0 && ty < 2) {  // warp 0: the rows' hull, warp 1: the columns'
        const int i = ty == 0 ? bi + tx : j;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            // (a point past n repeats one; NaN coordinates are reported, not used)
            float lo = static_cast<float>(xyz[3 * (size_t)min(i, n - 1) + k]), hi = lo;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            }
            if (tx == 0) {
                hull[ty][0][k] = lo;
                hull[ty][1][k] = hi;
            }
        }
    }
    unsigned blocked = 0;  // bit s: pair s
    for (int b0 = 0, par = 0; b0 < m; b0 += kBoxes, par ^= 1) {
        int cnt = min(kBoxes, m - b0);
        if (tid == 0) kept[par] = 0;
        __syncthreads();
        for (int e = tid; e < cnt * 6; e += kTile * 8) {
            const double v = boxes[6 * (size_t)b0 + e];
            sbox[e] = v;
            bad = bad || !isfinite(v);
        }
        __syncthreads();
        // Boxes that no segment between the tile's points can meet are dropped:
        // both hulls lie on one side of the box on some axis, by the filter's E.
        if (tid < cnt) {
            float mg = 0.f, lo[3], hi[3];
            for (int k = 0; k < 3; ++k) {
                bad = bad || sbox[6 * tid + k] > sbox[6 * tid + 3 + k];
                lo[k] = static_cast<float>(__dsub_rn(sbox[6 * tid + k], r));
                hi[k] = static_cast<float>(__dadd_rn(sbox[6 * tid + 3 + k], r));
                mg = fmaxf(mg, fmaxf(fabsf(lo[k]), fabsf(hi[k])));
            }
            bool out = false;
            float hm = mg;
            for (int k = 0; k < 3; ++k)
                for (int h = 0; h < 2; ++h)
                    hm = fmaxf(hm, fmaxf(fabsf(hull[h][0][k]), fabsf(hull[h][1][k])));
            const float E = 2.f * hm * 0x1p-20f + 1e-30f;
            for (int k = 0; k < 3; ++k)
                out = out || fmaxf(hull[0][1][k], hull[1][1][k]) < lo[k] - E ||
                      fminf(hull[0][0][k], hull[1][0][k]) > hi[k] + E;
            if (!out) {
                const int at = atomicAdd(&kept[par], 1);
                for (int k = 0; k < 3; ++k) {
                    slo[at][k] = lo[k];
                    shi[at][k] = hi[k];
                }
                smag[at] = mg;
                sidx[at] = static_cast<unsigned char>(tid);
            }
        }
        __syncthreads();
        cnt = kept[par];
#pragma unroll 1
        for (int s = 0; s < 4; ++s) {
            const int i = bi + ty + 8 * s;
            if (i >= n || j >= n || i >= j || (blocked >> s & 1)) continue;
            double p[3];
            Axis ax[3];
            float mag = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                p[k] = xyz[3 * (size_t)i + k];
                const float pf = static_cast<float>(p[k]);
                ax[k] = Axis{pf, 1.f / static_cast<float>(__dsub_rn(q[k], p[k])), fminf(pf, qf[k]),
                             fmaxf(pf, qf[k])};
                mag = fmaxf(mag, fmaxf(fabsf(pf), fabsf(qf[k])));
            }
            bool hit = false;
            for (int g0 = 0; g0 < cnt && !hit; g0 += 32) {
                unsigned open = 0;
                const int g1 = min(cnt, g0 + 32);
#pragma unroll 2
                for (int b = g0; b < g1; ++b) {
                    const float lo[3] = {slo[b][0], slo[b][1], slo[b][2]};
                    const float hi[3] = {shi[b][0], shi[b][1], shi[b][2]};
                    const int v = filter_box(ax, lo, hi, (mag + smag[b]) * 0x1p-20f + 1e-30f);
                    hit = hit || v == 1;
                    open |= static_cast<unsigned>(v == 2) << (b - g0);
                }
                for (; open && !hit; open &= open - 1)
                    hit = segment_blocked(p, q, sbox + 6 * sidx[g0 + __ffs(open) - 1], r);
            }
            blocked |= static_cast<unsigned>(hit) << s;
        }
    }
    __syncthreads();
    Split qs[3];
    float qmag = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        qs[k] = split(q[k]);
        qmag = fmaxf(qmag, fabsf(qf[k]));
    }
#pragma unroll 2
    for (int s = 0; s < 4; ++s) {
        const int r0 = ty + 8 * s, i = bi + r0;
        int v = 0;
        if (i < n && j < n && i < j) {
            const Split ps[3] = {rows[r0][0], rows[r0][1], rows[r0][2]};
            const float mag =
                fmaxf(fmaxf(qmag, fabsf(ps[0].hi)), fmaxf(fabsf(ps[1].hi), fabsf(ps[2].hi)));
            long long c = length_mm(ps, qs, mag);
            if (c < 0) {
                const double* p = xyz + 3 * (size_t)i;
                const double dx = __dsub_rn(q[0], p[0]);
                const double dy = __dsub_rn(q[1], p[1]);
                const double dz = __dsub_rn(q[2], p[2]);
                double acc = __dmul_rn(dx, dx);
                acc = __dadd_rn(acc, __dmul_rn(dy, dy));
                acc = __dadd_rn(acc, __dmul_rn(dz, dz));
                c = __double2ll_rn(__dmul_rn(1000.0, __dsqrt_rn(acc)));
            }
            if (blocked >> s & 1) c += penalty;
            if (c > DPSO_COST_MAX) {
                atomicOr(err, 2);
                c = DPSO_COST_MAX;
            }
            v = static_cast<int>(c);
        }
        if (i < n && j < n && i <= j) C[(size_t)i * ldc + j] = v;  // (0 on the diagonal)
        tile[r0][tx] = v;
    }
    if (bad) atomicOr(err, 1);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 4; ++s) {  // row bj + r of the lower half, columns bi ..
        const int rr = ty + 8 * s, row = bj + rr, col = bi + tx;
        if (row < n && col < n && col < row) C[(size_t)row * ldc + col] = tile[tx][rr];
    }
}

// Flags an asymmetric matrix or a non-zero diagonal (bit 0) and entries outside
// [0, limit] (bit 1).  A block compares a 32 x 32 tile on or above the diagonal
// with its mirror image, read in rows and turned in shared memory: bound by the
// one read of the matrix (read down columns instead, it took 20 us at
// n = 1992).
__global__ void __launch_bounds__(kTile * 8) check_cost_kernel(const int* __restrict__ C, int n,
                                                               int ldc, int limit, int* err) {
    const int bi = blockIdx.y * kTile, bj = blockIdx.x * kTile;
    if (bj < bi) return;
    __shared__ int tile[kTile][kTile + 1];
    const int tx = threadIdx.x, ty = threadIdx.y;
    int bits = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {  // the mirror tile
        const int i = bj + ty + 8 * s, j = bi + tx;
        const int v = i < n && j < n ? C[(size_t)i * ldc + j] : 0;
        if (v < 0 || v > limit) bits |= 2;
        tile[ty + 8 * s][tx] = v;
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int i = bi + ty + 8 * s, j = bj + tx;
        if (i >= n || j >= n) continue;
        const int v = C[(size_t)i * ldc + j];
        if (v < 0 || v > limit) bits |= 2;
        if (i == j ? v != 0 : v != tile[tx][ty + 8 * s]) bits |= 1;
    }
    if (bits) atomicOr(err, bits);
}

}  // namespace

cudaError_t launch_cost_matrix(const double* xyz, int n, const double* boxes, int m, double radius,
                               int penalty, int* C, int ldc, int* err, cudaStream_t st) {
    const int tiles = (n + kTile - 1) / kTile;
    dim3 grid(tiles, tiles), block(kTile, 8);
    cost_matrix_kernel<<<grid, block, 0, st>>>(xyz, n, boxes, m, radius, penalty, C, ldc, err);
    return cudaGetLastError();
}

cudaError_t launch_check_cost(const int* C, int n, int ldc, int* err, cudaStream_t st) {
    return launch_check_cost_limit(C, n, ldc, DPSO_COST_MAX, err, st);
}

cudaError_t launch_check_cost_limit(const int* C, int n, int ldc, int limit, int* err,
                                    cudaStream_t st) {
    const int tiles = (n + kTile - 1) / kTile;
    check_cost_kernel<<<dim3(tiles, tiles), dim3(kTile, 8), 0, st>>>(C, n, ldc, limit, err);
    return cudaGetLastError();
}

}  // namespace dpso

using namespace dpso;

extern "C" int dpso_cost_matrix(const double* xyz_dev, int32_t n, const double* boxes_dev,
                                int32_t m, const dpso_cost_params* cp, int32_t* C_dev,
                                void* stream) {
    if (!xyz_dev || !C_dev || !cp || n < 1 || m < 0 || (m > 0 && !boxes_dev)) return DPSO_ERR_ARG;
    if (n > DPSO_MAX_N) return DPSO_ERR_RANGE;
    if (!(cp->uav_radius_m >= 0.0) || !isfinite(cp->uav_radius_m) || cp->blocked_penalty_mm < 0 ||
        cp->reserved != 0)
        return DPSO_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Scratch scratch;
    if (scratch.acquire(sizeof(int), st) != cudaSuccess) return DPSO_ERR_NO_MEMORY;
    int* err = static_cast<int*>(scratch.p);
    int herr = 0;
    cudaError_t e = cudaMemsetAsync(err, 0, sizeof(int), st);
    if (e == cudaSuccess)
        e = launch_cost_matrix(xyz_dev, n, boxes_dev, m, cp->uav_radius_m, cp->blocked_penalty_mm,
                               C_dev, n, err, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return DPSO_ERR_CUDA;
    scratch.release();  // (the stream was waited for)
    if (herr & 1) return DPSO_ERR_ARG;
    if (herr & 2) return DPSO_ERR_RANGE;
    return DPSO_OK;
}
