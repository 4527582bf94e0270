// Sign of the grid points beyond the band (the fill the paper names as the step after the narrow
// band, Section 11.3): every point outside the band gets -inf inside the surface and +inf outside,
// so the whole grid carries the inside/outside sign.
//
// The band half-width w exceeds the grid step h, so the surface never passes between two
// neighbouring grid points that are both outside the band: if it crossed the segment between
// them, both would lie within h < w of it.  Hence
//   (1) along an x-row, every run of points outside the band has the sign of the band point next
//       to it (left or right);
//   (2) a row with no band point at all has one sign along its whole length, and it is the sign
//       of the point next to it in a neighbouring row (y or z), whichever row that is;
//   (3) a grid without any band point is taken as outside.
// Kernels: k_fill_rows applies (1) and records per row the sign at x = 0 (0 for a row without band
// points); k_fill_lines_y and _z resolve (2) by nearest-known propagation along y, then along z;
// k_fill_empty writes the rows of (2) that lie inside.  Points start at +inf (written by the tile
// kernel), so only inside points are written.
#include <math.h>
#include <stdint.h>

#include "sdf_internal.cuh"

namespace sdf {
namespace {

constexpr unsigned FULL_MASK = 0xffffffffu;

__device__ __forceinline__ int find_row_prob(const long long *rbase, int n, long long r) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (rbase[mid] <= r) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// negative in the sense of the field: d < 0, or -0
__device__ __forceinline__ bool is_neg(float v) { return signbit(v); }

// What is known along a stretch of at most 32 x 32 entries, for the warp that holds it: lane c has the
// known entries of chunk c (known: a bit each) and which of them are negative.  `carry` is the sign of
// the last known entry before the stretch (+-1, or 0: none yet); on return the sign after it.  Lane c
// gets the sign that holds before the first known entry of its chunk, the one of the first known
// entry of the stretch where nothing is known before.  0 everywhere when nothing is known at all.
__device__ __forceinline__ int chunk_signs(unsigned known, unsigned neg, int &carry) {
    const int lane = threadIdx.x & 31;
    const unsigned any = __ballot_sync(FULL_MASK, known != 0);
    if (!any) return carry;
    const int fc = __ffs(any) - 1, lc = 31 - __clz(any);
    const unsigned fk = __shfl_sync(FULL_MASK, known, fc), fn = __shfl_sync(FULL_MASK, neg, fc);
    const unsigned lk = __shfl_sync(FULL_MASK, known, lc), ln = __shfl_sync(FULL_MASK, neg, lc);
    const int lead = carry ? carry : (((fn >> (__ffs(fk) - 1)) & 1u) ? -1 : 1);
    const unsigned before = any & ((1u << lane) - 1u);
    const int src = before ? 31 - __clz(before) : 0;
    const unsigned sk = __shfl_sync(FULL_MASK, known, src), sn = __shfl_sync(FULL_MASK, neg, src);
    carry = ((ln >> (31 - __clz(lk))) & 1u) ? -1 : 1;
    return before ? (((sn >> (31 - __clz(sk))) & 1u) ? -1 : 1) : lead;
}
// the sign at this lane's entry of a chunk: of the nearest known entry up to it, else `in`
__device__ __forceinline__ int sign_at(unsigned known, unsigned neg, int in) {
    const unsigned left = known & (0xffffffffu >> (31 - (threadIdx.x & 31)));
    return left ? (((neg >> (31 - __clz(left))) & 1u) ? -1 : 1) : in;
}

// One warp per x-row, 1024 points of it at a time.  rowsign[r] = sign at x = 0 (+1 / -1), or 0 if the
// row has no band point.  Bound by the read of the field (4 B per point, once, eight loads in flight
// per lane); what the points are stays in two bit masks per lane, from which the inside points are
// written.  Reading the row up to its first band point and then again from the start, one load at a
// time, took 63 us on a 333 x 331 x 257 grid; now 37 us.
__global__ void __launch_bounds__(256) k_fill_rows(const FillProb *P, const long long *rbase, int n, long long r_tot,
                                                   int8_t *rowsign) {
    dep_wait();
    dep_next();
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < r_tot; r += warps) {
        const int p = find_row_prob(rbase, n, r);
        const FillProb pr = P[p];
        float *row = pr.dist + (r - rbase[p]) * (long long)pr.nx;
        int first = 0, carry = 0;
        // (unsigned: the ends of steps of 1024 and of eight chunks may lie beyond the largest int)
        const unsigned nx = (unsigned)pr.nx;
        for (unsigned s0 = 0; s0 < nx; s0 += 1024) {
            const int chunks = (int)min(32u, (nx - s0 + 31) >> 5);
            unsigned known = 0, neg = 0;
            for (int c0 = 0; c0 < chunks; c0 += 8) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    const unsigned x = s0 + (c0 + u) * 32 + lane;
                    v[u] = x < nx ? row[x] : INFINITY;
                }
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    const bool band = isfinite(v[u]);
                    const unsigned bm = __ballot_sync(FULL_MASK, band), nm = __ballot_sync(FULL_MASK, band && is_neg(v[u]));
                    if (lane == c0 + u) {
                        known = bm;
                        neg = nm;
                    }
                }
            }
            const int had = carry;
            const int in = chunk_signs(known, neg, carry);
            if (had == 0 && carry != 0) {  // the first band point of the row: it decides all before it
                first = __shfl_sync(FULL_MASK, in, 0);
                if (first < 0)
                    for (unsigned x = lane; x < s0; x += 32) row[x] = -INFINITY;
            }
            // the chunks that can hold inside points
            for (unsigned todo = __ballot_sync(FULL_MASK, lane < chunks && (in < 0 || neg != 0)); todo; todo &= todo - 1) {
                const int c = __ffs(todo) - 1;
                const unsigned ck = __shfl_sync(FULL_MASK, known, c), cn = __shfl_sync(FULL_MASK, neg, c);
                const int s = sign_at(ck, cn, __shfl_sync(FULL_MASK, in, c));
                const unsigned x = s0 + c * 32 + lane;
                if (x < nx && !((ck >> lane) & 1u) && s < 0) row[x] = -INFINITY;
            }
        }
        if (lane == 0) rowsign[r] = (int8_t)first;  // 0: resolved by the line passes
    }
}

// Nearest-known propagation of the row signs along y for every (problem, z), one warp per line: rows
// without band points (0) take the sign of the nearest row before them that has some, else after them.
// Resolved rows are marked +-2 so that k_fill_empty can tell them from rows with band points.
__global__ void __launch_bounds__(256) k_fill_lines_y(const FillProb *P, const long long *zbase, int n, long long l_tot,
                                                      const long long *rbase, int8_t *rowsign) {
    dep_wait();
    dep_next();
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long L = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); L < l_tot; L += warps) {
        const int p = find_row_prob(zbase, n, L);
        const unsigned len = (unsigned)P[p].ny;
        int8_t *e = rowsign + rbase[p] + (L - zbase[p]) * (long long)len;
        int carry = 0;
        for (unsigned s0 = 0; s0 < len; s0 += 1024) {
            const int chunks = (int)min(32u, (len - s0 + 31) >> 5);
            unsigned known = 0, neg = 0;
            for (int c0 = 0; c0 < chunks; c0 += 8) {
                int v[8];
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    const unsigned i = s0 + (c0 + u) * 32 + lane;
                    v[u] = i < len ? (int)e[i] : 0;
                }
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    const unsigned km = __ballot_sync(FULL_MASK, v[u] != 0), nm = __ballot_sync(FULL_MASK, v[u] < 0);
                    if (lane == c0 + u) {
                        known = km;
                        neg = nm;
                    }
                }
            }
            const int had = carry;
            const int in = chunk_signs(known, neg, carry);
            if (carry == 0) continue;  // nothing known so far
            if (had == 0) {
                const int8_t m = (int8_t)(2 * __shfl_sync(FULL_MASK, in, 0));
                for (unsigned i = lane; i < s0; i += 32) e[i] = m;
            }
            for (int c = 0; c < chunks; c++) {
                const unsigned ck = __shfl_sync(FULL_MASK, known, c), cn = __shfl_sync(FULL_MASK, neg, c);
                const int s = sign_at(ck, cn, __shfl_sync(FULL_MASK, in, c));
                const unsigned i = s0 + c * 32 + lane;
                if (i < len && !((ck >> lane) & 1u)) e[i] = (int8_t)(2 * s);
            }
        }
    }
}

// The same along z for every (problem, y), after which the rows still unknown (a problem without band
// points) become outside.  A line's entries are ny bytes apart, so a block takes 32 neighbouring
// lines, one per lane, and its warps an eighth of their length each: first what is known in each part,
// then the entries.  (A warp per line, its lanes along the stride, took 9 us
// for 331 lines of 257 and 13.8 us for 128 of 96; now 5.5 and 4.5.)
__global__ void __launch_bounds__(256) k_fill_lines_z(const FillProb *P, const long long *ybase, int n, long long l_tot,
                                                      const long long *rbase, int8_t *rowsign) {
    dep_wait();
    dep_next();
    __shared__ int8_t s_first[8][32], s_last[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long L0 = (long long)blockIdx.x * 32; L0 < l_tot; L0 += (long long)gridDim.x * 32) {
        const long long L = L0 + lane;
        int8_t *e = nullptr;
        int k0 = 0, k1 = 0;
        long long stride = 0;
        if (L < l_tot) {
            const int p = find_row_prob(ybase, n, L);
            const int len = P[p].nz, part = (len + 7) / 8;
            stride = P[p].ny;
            e = rowsign + rbase[p] + (L - ybase[p]);
            k0 = min(warp * part, len);
            k1 = min(k0 + part, len);
        }
        int first = 0, last = 0;
#pragma unroll 8
        for (int k = k0; k < k1; k++) {
            const int v = e[k * stride];
            if (v != 0) {
                last = v < 0 ? -1 : 1;
                if (first == 0) first = last;
            }
        }
        s_first[warp][lane] = (int8_t)first;
        s_last[warp][lane] = (int8_t)last;
        __syncthreads();
        int carry = 0, lead = 0;
        for (int w = 7; w >= 0; w--) lead = s_first[w][lane] ? s_first[w][lane] : lead;
        for (int w = 0; w < warp; w++) carry = s_last[w][lane] ? s_last[w][lane] : carry;
        if (carry == 0) carry = lead ? lead : 1;  // no band point in the whole problem: outside
        for (int kk = k0; kk < k1; kk += 8) {  // (eight loads, then the stores: they would wait for each other)
            int v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = kk + u < k1 ? (int)e[(kk + u) * stride] : 1;
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (v[u] == 0) e[(kk + u) * stride] = (int8_t)(2 * carry);
                else if (kk + u < k1) carry = v[u] < 0 ? -1 : 1;
            }
        }
        __syncthreads();  // the shared signs are written again for the next lines
    }
}

// rows without band points that lie inside: the whole row becomes -inf
__global__ void k_fill_empty(const FillProb *P, const long long *rbase, int n, long long r_tot,
                             const int8_t *rowsign) {
    dep_wait();
    dep_next();
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < r_tot; r += warps) {
        if (rowsign[r] != -2) continue;
        const int p = find_row_prob(rbase, n, r);
        const FillProb pr = P[p];
        float *row = pr.dist + (r - rbase[p]) * (long long)pr.nx;
        for (int x = lane; x < pr.nx; x += 32) row[x] = -INFINITY;
    }
}

}  // namespace

cudaError_t fill_sign(const FillProb *P, const long long *rbase, const long long *zbase, const long long *ybase, int n,
                      long long r_tot, long long z_tot, long long y_tot, int8_t *rowsign, int n_sm, cudaStream_t s) {
    const dim3 blocks(8 * n_sm), bt(256);  // 8 warps per block, grid-stride over rows / lines
    cudaError_t e = launch_dep(k_fill_rows, blocks, bt, 0, s, P, rbase, n, r_tot, rowsign);
    if (e == cudaSuccess) e = launch_dep(k_fill_lines_y, blocks, bt, 0, s, P, zbase, n, z_tot, rbase, rowsign);
    if (e == cudaSuccess) e = launch_dep(k_fill_lines_z, blocks, bt, 0, s, P, ybase, n, y_tot, rbase, rowsign);
    if (e == cudaSuccess) e = launch_dep(k_fill_empty, blocks, bt, 0, s, P, rbase, n, r_tot, (const int8_t *)rowsign);
    return e;
}

}  // namespace sdf
