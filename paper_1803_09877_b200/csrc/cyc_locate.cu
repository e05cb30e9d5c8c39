// Cyclic-code adversary locator phi(R) (Section 3, "Cyclic Code"; correctness: Lemmas 4, 6-8).
//
//   cyc_project_kernel   e_j = sum_i f_i R[j][i]: the one O(d P) step, a single pass over R; beside it
//                        q_j = sum_i |R[j][i]|^2, the yardstick of the rank cutoff below.
//   cyc_reduce_partials_kernel   the blocks' partial sums of e and q added up in a fixed order.
//   cyc_solve_kernel     [h_{n-2s} .. h_{n-1}] = e C_R^dagger, the s x s Toeplitz system for
//                        beta (pseudo-inverse by a Jacobi SVD: its rank = the number of
//                        adversaries seen), the recurrence h_l = sum_u beta_u h_{l+u-s}, t = C h,
//                        V = the `rank` nodes with the largest |t_j|.
//   cyc_decode_vector_kernel   b with support in U = [n] \ V and [C_L]_{.,U} b_U = (0,..,0,1)^T
//                        (equivalent to W_{.,U} b = 1_P, proof of Lemma 3), minimum 2-norm.
//
// The small solves run in fp64 in a single thread block; only the projection touches HBM:
// 8 n len + 4 len bytes read.
#include <math.h>

#include <mutex>

#include "draco_internal.cuh"

namespace draco {

namespace {

constexpr int kThreads = kProjectWarps * 32;
constexpr int kSolveThreads = 512;
constexpr int kProjectChunk = 512;    // coordinates per warp and step of the few-rows projection

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {   // a * conj(b)
    return make_double2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    const double den = b.x * b.x + b.y * b.y;
    const double2 q = cmulc(a, b);
    return make_double2(q.x / den, q.y / den);
}
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }

// ------------------------------------------------------------------ projection
// Arithmetic.  f_i and R[j][i] are fp32, so their product has at most 48 significant bits and is exact in fp64:
// every term enters an fp64 running sum through one fused multiply-add on the converted operands, and the only
// rounding left is that of fp64 addition (2^-53 per term).  The device's e_j therefore carries the rounding of the
// complex64 vectors themselves and nothing of its own; products or short runs in fp32 would add about as much
// again per term (a 16-term fp32 run: three times as much), which the s x s syndrome system amplifies by about
// sqrt(s): at s = 20 that noise alone reached the rank cutoff and flagged an honest node.
//
// q_j = sum_i |R[j][i]|^2 travels with e_j: it is the yardstick of the locator's rank cutoff (rounding R to
// complex64 perturbs e_j by about 2^-25 (E f^2 q_j)^(1/2), whatever e_j itself cancels to).  It is summed in fp64
// from the converted values as well: squares of fp32 values overflow fp32 from 1.8e19 on, which a node may well
// send (W itself reaches 1e17 at n = 128, s = 20).  Layout of the block partials: [grid][n] double2 (e), then
// [grid][n] double (q).
__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    return a;
}
// Block partials: [cap][n] double2 (e) followed by [cap][n] double (q); cap = the capacity of the buffer in blocks,
// of which a launch fills the first gridDim.x.
__device__ __forceinline__ double* q_partials(double2* partial, int cap, int n) {
    return reinterpret_cast<double*>(partial + (int64_t)cap * n);
}
// Block = 8 warps over one tile of coordinates; warp w owns rows row0 + w, row0 + w + 8, ... of the
// launch's nrows <= 8 RPW rows; f for the tile sits in shared memory as fp64 (converted once per tile, used by every row).
// `every` > 1: only each `every`-th tile is read (a sample).  More than 64 rows take two launches of half the rows each (rows are
// independent; f is read twice, 1 % more traffic): 16 rows per warp in registers halve the blocks per SM
// (0.79 of the copy bandwidth at n = 105), and per-lane sums in shared memory left the compiler too few
// registers to keep its loads in flight once the squared norms were added (0.98 -> 0.68).
template <int RPW, bool VEC2, int TILE>
__global__ void __launch_bounds__(kThreads, 4)
cyc_project_kernel(const float2* __restrict__ R, const float* __restrict__ f, int64_t len, int64_t ld, int n,
                   int row0, int nrows, double2* __restrict__ partial, int cap, int accumulate, int every) {
    pdl_begin();
    __shared__ __align__(16) double fs[TILE];
    // Running sums of row warp + r * 8 over this block's tiles, kept by lane 0 of the row's warp: after every tile
    // the warp adds its lanes' sums up (fixed butterfly order) and lane 0 adds the result here.  Keeping them in
    // registers instead (2 RPW doubles per lane) left too few of the 64 registers for eight 128-bit loads in flight.
    __shared__ double2 es[kProjectWarps * RPW];
    __shared__ double qs[kProjectWarps * RPW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Short vectors have fewer tiles than the device has SMs; the launch then splits the rows over gridDim.y as well
    // (whole multiples of the 8 warps' rows), every (tile, node) partial still being written by exactly one block.
    if (gridDim.y > 1) {
        const int per = (((nrows + (int)gridDim.y - 1) / (int)gridDim.y + kProjectWarps - 1) / kProjectWarps) * kProjectWarps;
        const int skip = (int)blockIdx.y * per;
        if (skip >= nrows) return;
        row0 += skip;
        nrows = (nrows - skip) < per ? (nrows - skip) : per;
    }
    if (lane == 0) {
#pragma unroll
        for (int r = 0; r < RPW; ++r) {
            es[r * kProjectWarps + warp] = make_double2(0.0, 0.0);
            qs[r * kProjectWarps + warp] = 0.0;
        }
    }

    const int64_t ntiles = (len + TILE - 1) / TILE;
    for (int64_t tile = (int64_t)blockIdx.x * every; tile < ntiles; tile += (int64_t)gridDim.x * every) {
        const int64_t c0 = tile * TILE;
        const int cnt = (int)((len - c0) < TILE ? (len - c0) : TILE);
        for (int i = threadIdx.x; i < TILE; i += kThreads) fs[i] = (i < cnt) ? (double)__ldcs(f + c0 + i) : 0.0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RPW; ++r) {
            const int j = row0 + warp + r * kProjectWarps;
            if (j < row0 + nrows) {
                const float2* row = R + (int64_t)j * ld + c0;
                double eq = 0.0;
                double ar = 0.0, ai = 0.0;
                if (VEC2 && cnt == TILE) {
                    const float4* row4 = reinterpret_cast<const float4*>(row);
#pragma unroll 1
                    for (int step0 = 0; step0 < TILE / 64; step0 += 8) {
                        float4 v[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) v[q] = __ldcs(row4 + (step0 + q) * 32 + lane);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const double2 ff = *reinterpret_cast<const double2*>(&fs[((step0 + q) * 32 + lane) * 2]);
                            const double x0 = (double)v[q].x, y0 = (double)v[q].y, x1 = (double)v[q].z, y1 = (double)v[q].w;
                            ar = fma(ff.x, x0, ar); ai = fma(ff.x, y0, ai);
                            ar = fma(ff.y, x1, ar); ai = fma(ff.y, y1, ai);
                            eq = fma(x0, x0, eq); eq = fma(y0, y0, eq);
                            eq = fma(x1, x1, eq); eq = fma(y1, y1, eq);
                        }
                    }
                } else if (RPW == 4 && TILE == kProjectTile) {
                    // Up to four rows per warp, full tiles, rows off the 16-byte grid: left to the compiler's order of loads.  Sixteen at
                    // a time, as below, cost 12 % (n = 17, d = 12,000,001 327 us, 280 so; n = 32 505 and 461), eight or four no less;
                    // with more rows per warp they gain (n = 45 757 us so, 707).
                    for (int i = lane; i < cnt; i += 32) {
                        const float2 v = __ldcs(row + i);
                        const double ff = fs[i], x0 = (double)v.x, y0 = (double)v.y;
                        ar = fma(ff, x0, ar);
                        ai = fma(ff, y0, ai);
                        eq = fma(y0, y0, fma(x0, x0, eq));
                    }
                } else {
                    // 8-byte loads, which any row start allows; entries beyond the vector count as zero (and fs is zero there)
#pragma unroll 1
                    for (int step0 = 0; step0 * 32 < cnt; step0 += 16) {
                        float2 v[16];
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            const int i = (step0 + q) * 32 + lane;
                            v[q] = i < cnt ? __ldcs(row + i) : make_float2(0.f, 0.f);
                        }
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            const double ff = fs[(step0 + q) * 32 + lane], x0 = (double)v[q].x, y0 = (double)v[q].y;
                            ar = fma(ff, x0, ar);
                            ai = fma(ff, y0, ai);
                            eq = fma(y0, y0, fma(x0, x0, eq));
                        }
                    }
                }
                ar = warp_sum(ar);
                ai = warp_sum(ai);
                eq = warp_sum(eq);
                if (lane == 0) {
                    double2 acc = es[r * kProjectWarps + warp];
                    acc.x += ar;
                    acc.y += ai;
                    es[r * kProjectWarps + warp] = acc;
                    qs[r * kProjectWarps + warp] += eq;
                }
            }
        }
        __syncthreads();
    }
    double* qpartial = q_partials(partial, cap, n);
    if (lane == 0) {
#pragma unroll
        for (int r = 0; r < RPW; ++r) {
            const int j = row0 + warp + r * kProjectWarps;
            if (j < row0 + nrows) {
                double2* dst = partial + (int64_t)blockIdx.x * n + j;
                double* qdst = qpartial + (int64_t)blockIdx.x * n + j;
                double2 a = es[r * kProjectWarps + warp];
                double c = qs[r * kProjectWarps + warp];
                if (accumulate) { a.x += dst->x; a.y += dst->y; c += *qdst; }
                *dst = a;
                *qdst = c;
            }
        }
    }
}

// The same projection for few rows (n <= 16): with one or two rows per warp the block-wide tile
// barriers of the kernel above dominate, so here every warp works alone on 512-coordinate chunks of all n rows, row by row,
// with f for its chunk in registers (16 values per lane), eight 128-bit loads per lane in flight and no barrier in the loop.
// The three sums of a row live in registers for that row only; the lanes' sums are added by a butterfly and kept by lane 0 in
// shared memory, so that three blocks fit on an SM.  With per-lane sums of all rows (32 doubles, and 16 more did not fit) it
// was two blocks and ten shuffles per row and 256 coordinates for q alone (n = 15, reduction included: d = 30 M 602 us, now
// 524 = 7.1 TB/s; d = 1 M 44 us, now 30; d = 30 M + 1, whose rows went 32 coordinates at a time, 3750 us, now 630).
constexpr int kFewRows = 16;
template <bool VEC2, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 3)
cyc_project_fewrows_kernel(const float2* __restrict__ R, const float* __restrict__ f, int64_t len, int64_t ld, int n,
                           double2* __restrict__ partial, int cap, int accumulate, int every) {
    pdl_begin();
    constexpr int CH = kProjectChunk;
    __shared__ double2 es[kProjectWarps][kFewRows];
    __shared__ double qs[kProjectWarps][kFewRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < kFewRows) {
        es[warp][lane] = make_double2(0.0, 0.0);
        qs[warp][lane] = 0.0;
    }
    __syncwarp();
    auto keep = [&](int j, double ar, double ai, double eq) {
        ar = warp_sum(ar);
        ai = warp_sum(ai);
        eq = warp_sum(eq);
        if (lane == 0) {
            double2 acc = es[warp][j];
            acc.x += ar;
            acc.y += ai;
            es[warp][j] = acc;
            qs[warp][j] += eq;
        }
    };
    int row0 = 0, nrows = n;                             // rows of this block
    if (SPLIT) {
        const int per = (n + (int)gridDim.y - 1) / (int)gridDim.y;
        row0 = (int)blockIdx.y * per;
        nrows = (n - row0) < per ? (n - row0) : per;
    }
    const int64_t nchunks = (len + CH - 1) / CH;
    const int64_t nwarps = (int64_t)gridDim.x * kProjectWarps * every;
    for (int64_t chunk = ((int64_t)blockIdx.x * kProjectWarps + warp) * every; chunk < nchunks; chunk += nwarps) {
        const int64_t c0 = chunk * CH;
        const int cnt = (int)((len - c0) < CH ? (len - c0) : CH);
        if (VEC2 && cnt == CH) {
            float2 ff[CH / 64];
#pragma unroll
            for (int q = 0; q < CH / 64; ++q) ff[q] = __ldcs(reinterpret_cast<const float2*>(f + c0) + q * 32 + lane);
#pragma unroll 1
            for (int j = row0; j < row0 + nrows; ++j) {
                const float4* row = reinterpret_cast<const float4*>(R + (int64_t)j * ld + c0) + lane;
                float4 v[CH / 64];
#pragma unroll
                for (int q = 0; q < CH / 64; ++q) v[q] = __ldcs(row + q * 32);
                double ar = 0.0, ai = 0.0, eq = 0.0;
#pragma unroll
                for (int q = 0; q < CH / 64; ++q) {
                    const double fx = (double)ff[q].x, fy = (double)ff[q].y;
                    const double x0 = (double)v[q].x, y0 = (double)v[q].y, x1 = (double)v[q].z, y1 = (double)v[q].w;
                    ar = fma(fx, x0, ar); ai = fma(fx, y0, ai);
                    ar = fma(fy, x1, ar); ai = fma(fy, y1, ai);
                    eq = fma(x0, x0, eq); eq = fma(y0, y0, eq);
                    eq = fma(x1, x1, eq); eq = fma(y1, y1, eq);
                }
                keep(j, ar, ai, eq);
            }
        } else {                                             // any row start, ragged chunk: 8-byte loads, zero beyond the vector
            float ff[CH / 32];
#pragma unroll
            for (int q = 0; q < CH / 32; ++q) ff[q] = q * 32 + lane < cnt ? __ldcs(f + c0 + q * 32 + lane) : 0.0f;
#pragma unroll 1
            for (int j = row0; j < row0 + nrows; ++j) {
                const float2* row = R + (int64_t)j * ld + c0 + lane;
                float2 v[CH / 32];
#pragma unroll
                for (int q = 0; q < CH / 32; ++q) v[q] = q * 32 + lane < cnt ? __ldcs(row + q * 32) : make_float2(0.f, 0.f);
                double ar = 0.0, ai = 0.0, eq = 0.0;
#pragma unroll
                for (int q = 0; q < CH / 32; ++q) {
                    const double fx = (double)ff[q], x0 = (double)v[q].x, y0 = (double)v[q].y;
                    ar = fma(fx, x0, ar); ai = fma(fx, y0, ai);
                    eq = fma(y0, y0, fma(x0, x0, eq));
                }
                keep(j, ar, ai, eq);
            }
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < nrows) {
        const int j = row0 + threadIdx.x;
        double a = 0.0, b = 0.0, c = 0.0;
        for (int w = 0; w < kProjectWarps; ++w) {            // fixed order: reproducible
            a += es[w][j].x;
            b += es[w][j].y;
            c += qs[w][j];
        }
        double2* dst = partial + (int64_t)blockIdx.x * n + j;
        double* qdst = q_partials(partial, cap, n) + (int64_t)blockIdx.x * n + j;
        if (accumulate) { a += dst->x; b += dst->y; c += *qdst; }
        *dst = make_double2(a, b);
        *qdst = c;
    }
}

// e_j and q_j = sums over the blocks' partials: one block of 128 threads per node j.  Thread t adds the partials
// of blocks t, t + 128, .. in ascending order, the 128 thread sums are then added by a butterfly inside each warp
// and the four warp sums in ascending order.  The order is fixed, so the sums are reproducible bit for bit.
// record: n (re, im) pairs, then n values q_j (3 n doubles).  (A single block doing this for all nodes took
// 20-40 us: one SM's load latency, serialised.)
constexpr int kReduceThreads = 128;
__global__ void __launch_bounds__(kReduceThreads)
cyc_reduce_partials_kernel(const double2* __restrict__ partial, int grid, int cap, int n, double* __restrict__ record) {
    pdl_begin();
    constexpr int kBatch = 8;
    __shared__ double wsum[3][kReduceThreads / 32];
    const int j = blockIdx.x, tid = threadIdx.x;
    const double* __restrict__ qpartial = reinterpret_cast<const double*>(partial + (int64_t)cap * n);
    double a = 0.0, b = 0.0, c = 0.0;
    for (int base = 0; base < grid; base += kBatch * kReduceThreads) {
        double2 pe[kBatch];
        double pq[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {               // all loads first (beyond the grid: block 0 again, not added)
            const int blk = base + u * kReduceThreads + tid;
            const int64_t at = (int64_t)(blk < grid ? blk : 0) * n + j;
            pe[u] = __ldcg(partial + at);
            pq[u] = __ldcg(qpartial + at);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (base + u * kReduceThreads + tid < grid) {
                a += pe[u].x;
                b += pe[u].y;
                c += pq[u];
            }
        }
    }
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_sum(c);
    if ((tid & 31) == 0) { wsum[0][tid >> 5] = a; wsum[1][tid >> 5] = b; wsum[2][tid >> 5] = c; }
    __syncthreads();
    if (tid == 0) {
        double x = 0.0, y = 0.0, z = 0.0;
        for (int w = 0; w < kReduceThreads / 32; ++w) { x += wsum[0][w]; y += wsum[1][w]; z += wsum[2][w]; }
        record[2 * j] = x;
        record[2 * j + 1] = y;
        record[2 * n + j] = z;
    }
}

// The small solves below run either on the whole block (WARP = false: block-wide barriers, any size) or on its
// first warp alone (WARP = true: warp barriers only; the matrices then sit in shared memory).  The arithmetic and
// its order are the same in both.
template <bool WARP>
__device__ __forceinline__ void small_sync() {
    if (WARP) __syncwarp(); else __syncthreads();
}

// ------------------------------------------------------------------ small dense solve
// Gauss-Jordan elimination with complete pivoting on the dim x (dim+1) augmented matrix A
// (row stride dim+1).  Pivots with |pivot| <= tol end the elimination (numerical rank); the
// free unknowns are set to zero.  x receives the solution.  WARP: called by warp 0 only, dim <= 32.
template <bool WARP>
__device__ int block_gauss_jordan(double2* A, int dim, double tol, double2* x, int* perm, double* rowbest,
                                  int* rowbestc, int* sh) {
    const int tid = threadIdx.x, ldA = dim + 1;
    const int nthr = WARP ? 32 : blockDim.x;
    for (int i = tid; i < dim; i += nthr) perm[i] = i;
    small_sync<WARP>();
    int rank = 0;
    for (int p = 0; p < dim; ++p) {
        for (int i = p + tid; i < dim; i += nthr) {
            double best = -1.0;
            int bc = p;
            for (int c = p; c < dim; ++c) {
                const double m = cabs2(A[i * ldA + c]);
                if (m > best) { best = m; bc = c; }
            }
            rowbest[i] = best;
            rowbestc[i] = bc;
        }
        small_sync<WARP>();
        if (tid == 0) {
            double best = -1.0;
            int br = p;
            for (int i = p; i < dim; ++i)
                if (rowbest[i] > best) { best = rowbest[i]; br = i; }
            sh[0] = br;
            sh[1] = rowbestc[br];
            sh[2] = (best > tol * tol) ? 1 : 0;
        }
        small_sync<WARP>();
        const int pr = sh[0], pc = sh[1], ok = sh[2];
        if (!ok) break;
        if (pr != p)
            for (int c = tid; c <= dim; c += nthr) {
                const double2 tmp = A[p * ldA + c];
                A[p * ldA + c] = A[pr * ldA + c];
                A[pr * ldA + c] = tmp;
            }
        small_sync<WARP>();
        if (pc != p) {
            for (int i = tid; i < dim; i += nthr) {
                const double2 tmp = A[i * ldA + p];
                A[i * ldA + p] = A[i * ldA + pc];
                A[i * ldA + pc] = tmp;
            }
            if (tid == 0) { const int tmp = perm[p]; perm[p] = perm[pc]; perm[pc] = tmp; }
        }
        small_sync<WARP>();
        const double2 piv = A[p * ldA + p];
        for (int i = tid; i < dim; i += nthr) {
            if (i == p) continue;
            const double2 factor = cdiv(A[i * ldA + p], piv);
            for (int c = p + 1; c <= dim; ++c) {
                const double2 q = cmul(factor, A[p * ldA + c]);
                A[i * ldA + c].x -= q.x;
                A[i * ldA + c].y -= q.y;
            }
            A[i * ldA + p] = make_double2(0.0, 0.0);
        }
        small_sync<WARP>();
        rank = p + 1;
    }
    small_sync<WARP>();
    for (int i = tid; i < dim; i += nthr) x[i] = make_double2(0.0, 0.0);
    small_sync<WARP>();
    for (int k = tid; k < rank; k += nthr) x[perm[k]] = cdiv(A[k * ldA + dim], A[k * ldA + k]);
    small_sync<WARP>();
    return rank;
}

// Rotation of one Jacobi pair from alpha = |a_p|^2, beta = |a_q|^2 and gamma = a_p^H a_q (g2 = |gamma|^2 > 0): the
// unitary [[c, st], [-conj(st), c]] (c real, st complex) that makes the new columns a_p' = c a_p - conj(st) a_q and
// a_q' = st a_p + c a_q orthogonal, the smaller of the two angles.  With delta = beta - alpha, h = (delta^2 +
// 4 |gamma|^2)^(1/2) and x = |delta| / h:  c^2 = (1 + x) / 2,  st = sign(delta) gamma / (h c).  (The textbook form
// first turns a_q by exp(-i arg gamma) and then rotates by a real angle; the result differs by a unit factor on the
// second column, which one-sided Jacobi does not care about.)  Two reciprocal square roots and no division or square
// root: the chain of long-latency operations is serial and is most of a Jacobi step.
__device__ __forceinline__ void jacobi_rotation(double alpha, double bet, double gr, double gi, double g2, double& c,
                                                double2& st) {
    const double delta = bet - alpha;
    const double rh = rsqrt(fma(delta, delta, 4.0 * g2));
    const double c2 = fma(0.5 * fabs(delta), rh, 0.5);
    const double rc = rsqrt(c2);
    c = c2 * rc;
    const double k = copysign(rh * rc, delta);
    st = make_double2(gr * k, gi * k);
}

// (xo, yo) = (c x - conj(st) y, st x + c y)
__device__ __forceinline__ void rotate(double2 x, double2 y, double c, double2 st, double2& xo, double2& yo) {
    xo = make_double2(c * x.x - (st.x * y.x + st.y * y.y), c * x.y - (st.x * y.y - st.y * y.x));
    yo = make_double2(st.x * x.x - st.y * x.y + c * y.x, st.x * x.y + st.y * x.x + c * y.y);
}
// one column pair, rows i0, i0 + step, ..
__device__ __forceinline__ void rotate_pair(double2* xp, double2* yp, int i0, int step, int rows, double c, double2 st) {
    for (int i = i0; i < rows; i += step) rotate(xp[i], yp[i], c, st, xp[i], yp[i]);
}

// ------------------------------------------------------------------ small SVD solve
// Pseudo-inverse solution of the s x s complex system A beta = rhs by one-sided (Hestenes)
// Jacobi: columns of [A; V] are rotated in pairs until the columns of A are orthogonal; then
// A = U Sigma, sigma_k = |a_k|, and beta = sum_{sigma_k > tol} v_k (a_k^H rhs) / sigma_k^2.
// Singular values come out to high relative accuracy, so the rank decision (sigma_k > tol)
// matches a LAPACK SVD except on a knife edge.  A, V: column-major with column stride ld
// (ld = s rounded up to even; a zero pad column never rotates).  One thread per column pair,
// pairs of a step disjoint (round-robin schedule).  Returns the rank.
__device__ int block_jacobi_pinv(double2* A, double2* V, const double2* rhs, int s, double tol, double2* beta,
                                 double2* coef, int* sh) {
    const int tid = threadIdx.x;
    const int nthr = blockDim.x;
    const int sp = s + (s & 1);
    for (int idx = tid; idx < sp * sp; idx += nthr) {
        const int c = idx / sp, i = idx % sp;
        V[idx] = make_double2(c == i ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    int sweeps = 0;
    bool converged = false;
    for (int sweep = 0; sweep < kJacobiSweepLimit; ++sweep) {
        if (tid == 0) sh[0] = 0;
        __syncthreads();
        for (int step = 0; step < sp - 1; ++step) {
            if (tid < sp / 2) {
                int a, b;
                if (tid == 0) { a = sp - 1; b = step; }
                else {                                    // (step +- tid) mod (sp - 1); both step and tid are below sp - 1
                    a = step + tid;
                    if (a >= sp - 1) a -= sp - 1;
                    b = step - tid;
                    if (b < 0) b += sp - 1;
                }
                const int p = a < b ? a : b, q = a < b ? b : a;
                double2* ap = A + p * sp;
                double2* aq = A + q * sp;
                double alpha = 0.0, bet = 0.0, gr = 0.0, gi = 0.0;
                for (int i = 0; i < s; ++i) {
                    const double2 x = ap[i], y = aq[i];
                    alpha += x.x * x.x + x.y * x.y;
                    bet += y.x * y.x + y.y * y.y;
                    gr += x.x * y.x + x.y * y.y;          // conj(x) * y
                    gi += x.x * y.y - x.y * y.x;
                }
                const double g2 = gr * gr + gi * gi;
                if (g2 > 1e-30 * alpha * bet && g2 > 0.0) {
                    double c;
                    double2 st;
                    jacobi_rotation(alpha, bet, gr, gi, g2, c, st);
                    rotate_pair(ap, aq, 0, 1, s, c, st);
                    rotate_pair(V + p * sp, V + q * sp, 0, 1, sp, c, st);
                    sh[0] = 1;
                }
            }
            __syncthreads();
        }
        const int rotated = sh[0];
        __syncthreads();
        ++sweeps;
        if (!rotated) { converged = true; break; }
    }
    if (tid == 0) { sh[1] = 0; sh[3] = converged ? sweeps : -sweeps; }
    __syncthreads();
    if (tid < sp) {
        const double2* ak = A + tid * sp;
        double sig2 = 0.0, pr = 0.0, pi = 0.0;
        for (int i = 0; i < s; ++i) {
            const double2 x = ak[i], r = rhs[i];
            sig2 += x.x * x.x + x.y * x.y;
            pr += x.x * r.x + x.y * r.y;                  // conj(x) * r
            pi += x.x * r.y - x.y * r.x;
        }
        const bool keep = sqrt(sig2) > tol;
        coef[tid] = keep ? make_double2(pr / sig2, pi / sig2) : make_double2(0.0, 0.0);
        if (keep) atomicAdd(&sh[1], 1);
    }
    __syncthreads();
    if (tid < s) {
        double re = 0.0, im = 0.0;
        for (int k = 0; k < sp; ++k) {
            const double2 q = cmul(V[k * sp + tid], coef[k]);
            re += q.x;
            im += q.y;
        }
        beta[tid] = make_double2(re, im);
    }
    __syncthreads();
    return sh[1];
}


// The same solve by one warp for s <= 16 (A, V in shared memory): the pairs of a step sit side by side in the
// warp, LP lanes per pair (a power of two), each lane holding the rows sub, sub + LP, .. of its pair's columns;
// the three inner products of a pair are reduced with shuffles inside its LP lanes, every lane of the pair then
// forms the same rotation and applies it to its own rows.  Only warp barriers.  Called by all 32 lanes of warp 0.
__device__ int warp_jacobi_pinv(double2* A, double2* V, const double2* rhs, int s, double tol, double2* beta,
                                double2* coef, int* sh) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int sp = s + (s & 1), npairs = sp / 2;
    for (int idx = lane; idx < sp * sp; idx += 32) {
        const int c = idx / sp, i = idx % sp;
        V[idx] = make_double2(c == i ? 1.0 : 0.0, 0.0);
    }
    __syncwarp();
    int sweeps = 0;
    bool converged = false;
    // the columns of a pair at a step
    auto columns = [&](int pair, int step, int& p, int& q) {
        int a, b;
        if (pair == 0) { a = sp - 1; b = step; }
        else {                                            // (step +- pair) mod (sp - 1); both are below sp - 1
            a = step + pair;
            if (a >= sp - 1) a -= sp - 1;
            b = step - pair;
            if (b < 0) b += sp - 1;
        }
        p = a < b ? a : b;
        q = a < b ? b : a;
    };
    if (sp <= 8) {
        // Eight lanes per pair, a row of A and of V per lane: everything of a step sits in registers between one round of loads
        // and one of stores.  s = 5: an iteration of about 35 steps takes 12 us instead of 18 with loops over the rows.
        const int pair = lane >> 3, sub = lane & 7;
        const bool act = pair < npairs, ra = act && sub < s, rv = act && sub < sp;
#pragma unroll 1
        for (int sweep = 0; sweep < kJacobiSweepLimit; ++sweep) {
            bool rotated = false;
#pragma unroll 1
            for (int step = 0; step < sp - 1; ++step) {
                int p = 0, q = 1;
                if (act) columns(pair, step, p, q);
                double2* const at[4] = {A + p * sp + sub, A + q * sp + sub, V + p * sp + sub, V + q * sp + sub};
                const double2 zero = make_double2(0.0, 0.0);
                const double2 x = ra ? *at[0] : zero, y = ra ? *at[1] : zero;
                const double2 vx = rv ? *at[2] : zero, vy = rv ? *at[3] : zero;
                double alpha = x.x * x.x + x.y * x.y, bet = y.x * y.x + y.y * y.y;
                double gr = x.x * y.x + x.y * y.y, gi = x.x * y.y - x.y * y.x;      // conj(x) * y
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) {
                    alpha += __shfl_xor_sync(full, alpha, off);
                    bet += __shfl_xor_sync(full, bet, off);
                    gr += __shfl_xor_sync(full, gr, off);
                    gi += __shfl_xor_sync(full, gi, off);
                }
                const double g2 = gr * gr + gi * gi;
                if (act && g2 > 1e-30 * alpha * bet && g2 > 0.0) {
                    double c;
                    double2 st;
                    jacobi_rotation(alpha, bet, gr, gi, g2, c, st);
                    if (ra) rotate(x, y, c, st, *at[0], *at[1]);
                    if (rv) rotate(vx, vy, c, st, *at[2], *at[3]);
                    rotated = true;
                }
                __syncwarp();
            }
            ++sweeps;
            if (!__any_sync(full, rotated)) { converged = true; break; }
        }
    } else {
        int lp = 1;
        while (lp * 2 * npairs <= 32) lp *= 2;
        const int pair = lane / lp, sub = lane % lp;
        const bool act = pair < npairs;
        for (int sweep = 0; sweep < kJacobiSweepLimit; ++sweep) {
            bool rotated = false;
            for (int step = 0; step < sp - 1; ++step) {
                int p = 0, q = 1;
                if (act) columns(pair, step, p, q);
                double2* ap = A + p * sp;
                double2* aq = A + q * sp;
                double alpha = 0.0, bet = 0.0, gr = 0.0, gi = 0.0;
                if (act)
                    for (int i = sub; i < s; i += lp) {
                        const double2 x = ap[i], y = aq[i];
                        alpha += x.x * x.x + x.y * x.y;
                        bet += y.x * y.x + y.y * y.y;
                        gr += x.x * y.x + x.y * y.y;          // conj(x) * y
                        gi += x.x * y.y - x.y * y.x;
                    }
                for (int off = lp >> 1; off > 0; off >>= 1) {
                    alpha += __shfl_xor_sync(full, alpha, off);
                    bet += __shfl_xor_sync(full, bet, off);
                    gr += __shfl_xor_sync(full, gr, off);
                    gi += __shfl_xor_sync(full, gi, off);
                }
                const double g2 = gr * gr + gi * gi;
                if (act && g2 > 1e-30 * alpha * bet && g2 > 0.0) {
                    double c;
                    double2 st;
                    jacobi_rotation(alpha, bet, gr, gi, g2, c, st);
                    rotate_pair(ap, aq, sub, lp, s, c, st);
                    rotate_pair(V + p * sp, V + q * sp, sub, lp, sp, c, st);
                    rotated = true;
                }
                __syncwarp();
            }
            ++sweeps;
            if (!__any_sync(full, rotated)) { converged = true; break; }
        }
    }
    bool keep = false;
    if (lane < sp) {
        const double2* ak = A + lane * sp;
        double sig2 = 0.0, pr = 0.0, pi = 0.0;
        for (int i = 0; i < s; ++i) {
            const double2 x = ak[i], r = rhs[i];
            sig2 += x.x * x.x + x.y * x.y;
            pr += x.x * r.x + x.y * r.y;                  // conj(x) * r
            pi += x.x * r.y - x.y * r.x;
        }
        keep = sqrt(sig2) > tol;
        coef[lane] = keep ? make_double2(pr / sig2, pi / sig2) : make_double2(0.0, 0.0);
    }
    const int rank = __popc(__ballot_sync(full, keep));
    __syncwarp();
    if (lane < s) {
        double re = 0.0, im = 0.0;
        for (int k = 0; k < sp; ++k) {
            const double2 q = cmul(V[k * sp + lane], coef[k]);
            re += q.x;
            im += q.y;
        }
        beta[lane] = make_double2(re, im);
    }
    if (lane == 0) { sh[1] = rank; sh[3] = converged ? sweeps : -sweeps; }
    __syncwarp();
    return rank;
}

constexpr int kSmallDim = 16;         // systems up to this size are solved in shared memory by one warp
constexpr int kFusedReduceMax = 16 * kSolveThreads;   // up to this many block partials (3 per block and node) are added up by the
                                                      // locator kernel itself: 16 loads per thread, about the 4 us of the reduction kernel

// ------------------------------------------------------------------ small systems, one warp
// What follows runs once per call, in one warp or one block, so its time is the chain of dependent operations and the
// instructions fetched for it (with the compiler's own unrolling 774 requests went past the instruction cache in 37,000
// cycles, n = 45, s = 5, five adversaries): loops are kept rolled, the elements of a system are spread over the lanes, and nothing divides by
// a run-time number (x mod n and the lanes of a sum are shifts and one multiplication).
constexpr int kRegSystem = 8;                              // unknowns of the systems below
struct ModN {                                              // x mod n for x < 2^16; magic = ceil(2^32 / n)
    uint32_t n, magic;
    __device__ __forceinline__ int operator()(int x) const { return x - (int)(__umulhi((uint32_t)x, magic) * n); }
};

// Gauss-Jordan elimination of the S x W matrix M (row-major, W <= 2 S + 1; its first S columns the system, the others right-hand
// sides), S <= 8.  PIVOT: rows are searched (never moved); otherwise the system is Hermitian positive definite.  Lane k gets the
// row and the reciprocal of pivot k: unknown k of right-hand side c is M[row][c] * inv.  False on a zero or non-finite pivot.
// QN: elements per lane, 32 QN >= S W.
template <bool PIVOT, int QN>
__device__ __forceinline__ bool warp_eliminate(double2* M, int S, int W, int& row, double2& inv) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int ei[QN], ci[QN];                                    // row and column of this lane's elements; others: element 0, not stored
    bool live[QN];
#pragma unroll
    for (int q = 0; q < QN; ++q) {
        const int e = lane + 32 * q;
        live[q] = e < S * W;
        ei[q] = live[q] ? (int)((float)e * __frcp_rn((float)W) + 1e-3f) : 0;        // e / W, e < 136
        ci[q] = live[q] ? e - ei[q] * W : 0;
    }
    unsigned used = 0;
    row = 0;
    inv = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int k = 0; k < S; ++k) {
        int pr = k;
        if (PIVOT) {                                       // largest |.|^2 to 20 bits
            const bool open = lane < S && !((used >> lane) & 1u);
            const double size = cabs2(M[(open ? lane : 0) * W + k]);
            const unsigned key = open ? (unsigned)__double2hiint(size) + 1u : 0u;
            const unsigned best = __reduce_max_sync(full, key);
            pr = __ffs(__ballot_sync(full, open && key == best)) - 1;
            used |= 1u << pr;
        }
        const double2 p = M[pr * W + k];
        double2 f[QN], m[QN], v[QN];
#pragma unroll
        for (int q = 0; q < QN; ++q) {
            f[q] = M[ei[q] * W + k];
            m[q] = M[pr * W + ci[q]];
            v[q] = M[ei[q] * W + ci[q]];
        }
        const double den = cabs2(p);
        if (!(den > 0.0 && den < 1e300)) return false;     // the same in every lane
        const double r = 1.0 / den;
        const double2 ip = make_double2(p.x * r, -p.y * r);
        if (lane == k) { row = pr; inv = ip; }
#pragma unroll
        for (int q = 0; q < QN; ++q) {
            const double2 g = cmul(m[q], ip), t = cmul(f[q], g);
            v[q].x -= t.x;
            v[q].y -= t.y;
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < QN; ++q)
            if (live[q] && ei[q] != pr) M[ei[q] * W + ci[q]] = v[q];
        __syncwarp();
    }
    return true;
}

// beta = A^{-1} rhs for the S x S syndrome system (row i: [h_{n-S-1-i} .. h_{n-2-i}] beta = h_{n-1-i}) when it certainly has
// full rank: sigma_min >= 1 / |A^{-1}|_F, so |A^{-1}|_F cut < 0.9 leaves every singular value above the cutoff and the
// pseudo-inverse solution is the solution.  The usual case, s adversaries at work, then needs no singular-value iteration
// (n = 45, s = 5: 24 us, the elimination about 2 us).  The bound on |A|_F |A^{-1}|_F keeps the computed inverse good to
// three digits.  Returns false, with beta untouched, when there is any doubt.  M: S (2 S + 1) elements of work space.
__device__ __forceinline__ bool warp_full_rank_solve(double2* M, const double2* h, int n, int S, double cut, double fro2,
                                                     double2* beta) {
    const int lane = threadIdx.x & 31, W = 2 * S + 1;
#pragma unroll 4
    for (int i = 0; i < S; ++i)
        if (lane < W) M[i * W + lane] = lane <= S ? h[n - S - 1 - i + lane] : make_double2(lane == S + 1 + i ? 1.0 : 0.0, 0.0);
    __syncwarp();
    int row;
    double2 inv;
    if (!(S * W <= 64 ? warp_eliminate<true, 2>(M, S, W, row, inv) : warp_eliminate<true, 5>(M, S, W, row, inv))) return false;
    double inv2 = 0.0;
    if (lane < S) {
#pragma unroll 1
        for (int c = S + 1; c < W; ++c) inv2 += cabs2(M[row * W + c]);
        inv2 *= cabs2(inv);
    }
    inv2 = warp_sum(inv2);
    if (!(inv2 * cut * cut < 0.81 && inv2 * fro2 < 1e24)) return false;
    if (lane < S) beta[lane] = cmul(M[row * W + S], inv);
    __syncwarp();
    return true;
}

// h_l = sum_u beta_u h_{l+u-S}, l = 0 .. count - 1, from h_{n-S} .. h_{n-1}: one thread, the last S values in registers.  The
// terms of the older values are summed in two chains while the newest value is still on its way, so that a step waits for
// two multiply-adds.
template <int S>
__device__ __noinline__ void run_recurrence(double2* h, int n, int count, const double2* beta) {
    double2 b[S], w[S];
#pragma unroll
    for (int u = 0; u < S; ++u) {
        b[u] = beta[u];
        w[u] = h[n - S + u];
    }
#pragma unroll 1
    for (int l0 = 0; l0 < count; l0 += S) {
#pragma unroll
        for (int k = 0; k < S; ++k) {                              // w[(k + u) mod S] = h_{l+u-S}
            double2 a = make_double2(0.0, 0.0), c = make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < S - 1; ++u) {
                const double2 v = w[(k + u) % S];
                a.x = fma(b[u].x, v.x, a.x);
                c.x = fma(-b[u].y, v.y, c.x);
                a.y = fma(b[u].x, v.y, a.y);
                c.y = fma(b[u].y, v.x, c.y);
            }
            const double2 v = w[(k + S - 1) % S];
            const double2 o = make_double2(a.x + c.x, a.y + c.y);
            w[k] = make_double2(fma(-b[S - 1].y, v.y, fma(b[S - 1].x, v.x, o.x)), fma(b[S - 1].y, v.x, fma(b[S - 1].x, v.y, o.y)));
            h[l0 + k < count ? l0 + k : kMaxN] = w[k];             // beyond the end: the spare entry
        }
    }
}

// The same for more than kRegSystem unknowns, the terms left to the compiler's unrolling: their loads are most of a step (n = 128,
// s = 20, locate 1295 us rolled, 1231 so).  A function of its own, so that its instructions do not lie between those of the small
// systems (in their midst: n = 15, s = 2, d = 4096, locate and decode 16.4 us, 15.9 so).
__device__ __noinline__ void run_recurrence_any(double2* h, int n, int count, int S, const double2* beta) {
#pragma unroll 1
    for (int l = 0; l < count; ++l) {
        double a = 0.0, b = 0.0;
        for (int u = 0; u < S; ++u) {
            int idx = l + u - S;
            if (idx < 0) idx += n;
            const double2 q = cmul(beta[u], h[idx]);
            a += q.x;
            b += q.y;
        }
        h[l] = make_double2(a, b);
    }
}

#define DRACO_BY_SIZE(size, CALL)                                                                            \
    switch (size) {                                                                                          \
        case 1: CALL(1); break;                                                                              \
        case 2: CALL(2); break;                                                                              \
        case 3: CALL(3); break;                                                                              \
        case 4: CALL(4); break;                                                                              \
        case 5: CALL(5); break;                                                                              \
        case 6: CALL(6); break;                                                                              \
        case 7: CALL(7); break;                                                                              \
        case 8: CALL(8); break;                                                                              \
        default: break;                                                                                      \
    }
static_assert(kRegSystem == 8, "the sizes of DRACO_BY_SIZE");

// Lanes that share one of `items` sums, as a shift: the largest power of two that the block has threads for, 32 at most.  The
// groups do not straddle warps, and every thread of the block takes part in the butterfly.
__device__ __forceinline__ int lanes_shift(int items) {
    const int shift = 9 - (32 - __clz(items - 1));
    return shift > 5 ? 5 : shift < 0 ? 0 : shift;
}
static_assert(kSolveThreads == 512, "2^9 in lanes_shift");
__device__ __forceinline__ double lane_sum(double a, int shift) {
#pragma unroll 1
    for (int off = (1 << shift) >> 1; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    return a;
}

// The nodes with fl != 0 in ascending order; returns how many.  bits: kMaxN / 32 words.  Called by the whole block.
__device__ __forceinline__ int list_flagged(const uint8_t* fl, int n, int* list, uint32_t* bits) {
    const int tid = threadIdx.x;
    const bool set = tid < n && fl[tid] != 0;
    const uint32_t w = __ballot_sync(0xffffffffu, set);
    if (tid < kMaxN && (tid & 31) == 0) bits[tid >> 5] = w;
    __syncthreads();
    int total = 0, before = 0;
#pragma unroll
    for (int k = 0; k < kMaxN / 32; ++k) {
        if (k == (tid >> 5)) before = total + __popc(bits[k] & ((1u << (tid & 31)) - 1u));
        total += __popc(bits[k]);
    }
    if (set) list[before] = tid;
    __syncthreads();
    return total;
}

// ------------------------------------------------------------------ decode vector
// With B = [C_L]_{.,V} and A = [C_L]_{.,U}: A A^H = I - B B^H, so the minimum-norm solution of
// A b_U = e_last is b_U = A^H y, y = e_last + B (I - B^H B)^{-1} B^H e_last, and
// I - B^H B = [C_R]_{.,V}^H [C_R]_{.,V} is only |V| x |V| (|V| <= 2 s).
// Called by every thread of a block of kSolveThreads threads; fl (the flags) and tw (w^k) in shared memory.
__device__ void decode_vector_body(CycDevice* cd, const uint8_t* fl, const double2* tw, int n, int s, ModN mod, double rsn,
                                   DeviceInfo* info) {
    __shared__ int vlist[kMaxN], rowbestc[kMaxN], perm_s[kMaxN], sh[4];
    __shared__ uint32_t bits[kMaxN / 32];
    __shared__ double rowbest[kMaxN];
    __shared__ double2 y[kMaxN], x_s[kMaxN];
    __shared__ double2 As[kSmallDim * (kSmallDim + 1)];
    const int tid = threadIdx.x;
    const int rows = n - 2 * s, L = rows - 1;
    const int a = list_flagged(fl, n, vlist, bits);
    if (a > 2 * s) {                                       // fewer than n - 2 s rows left: no b exists
        if (tid < n) cd->b[tid] = make_double2(0.0, 0.0);
        if (tid == 0) {
            info->n_active = 0; info->n_flagged = a; info->status = DRACO_ETOOMANY;
            info->im_residual_bits = 0ull; info->re_max_bits = 0ull;
        }
        return;
    }
    double2* x = x_s;
    if (a > 0) {
        const bool small = a <= kSmallDim;
        double2* A = small ? As : cd->work;
#pragma unroll 1
        for (int p = tid >> 5; p < a; p += kSolveThreads / 32)                  // a row per warp
#pragma unroll 1
            for (int q = tid & 31; q <= a; q += 32) {
                double2 val;
                if (q < a) {                               // (1/n) sum_{m >= n-2s} w^(m (v_q - v_p))
                    int dv = vlist[q] - vlist[p];
                    if (dv < 0) dv += n;
                    double re = 0.0, im = 0.0;
                    int k = mod((n - 2 * s) * dv);
#pragma unroll 1
                    for (int m = n - 2 * s; m < n; ++m) {
                        const double2 w = tw[k];
                        re += w.x;
                        im += w.y;
                        k += dv;
                        if (k >= n) k -= n;
                    }
                    val = make_double2(re * (rsn * rsn), im * (rsn * rsn));
                } else {                                   // conj(C[L][v_p])
                    const double2 w = tw[mod(L * vlist[p])];
                    val = make_double2(w.x * rsn, -w.y * rsn);
                }
                A[p * (a + 1) + q] = val;
            }
        __syncthreads();
        if (small) {
            if (tid < 32) {
                if (a <= kRegSystem) {                     // [C_R]_{.,V} has full column rank: positive definite
                    int row;
                    double2 inv;
                    warp_eliminate<false, 3>(As, a, a + 1, row, inv);
                    if (tid < a) x_s[tid] = cmul(As[row * (a + 1) + a], inv);
                } else {
                    block_gauss_jordan<true>(As, a, 0.0, x, perm_s, rowbest, rowbestc, sh);
                }
            }
            __syncthreads();
        } else {
            block_gauss_jordan<false>(A, a, 0.0, x, perm_s, rowbest, rowbestc, sh);
        }
    }
    if (tid < rows) {
        double re = (tid == L) ? 1.0 : 0.0, im = 0.0;
#pragma unroll 1
        for (int p = 0; p < a; ++p) {
            const double2 w = tw[mod(tid * vlist[p])];
            const double2 q = cmul(w, x[p]);
            re += q.x * rsn;
            im += q.y * rsn;
        }
        y[tid] = make_double2(re, im);
    }
    __syncthreads();
    const int shift = lanes_shift(n), per = 1 << shift, node = tid >> shift, sub = tid & (per - 1);
    double re = 0.0, im = 0.0;
    if (node < n) {
        int k = mod(sub * node);                           // (m node) mod n
        const int step = mod(per * node);
#pragma unroll 1
        for (int m = sub; m < rows; m += per) {
            const double2 q = cmulc(y[m], tw[k]);
            re += q.x;
            im += q.y;
            k += step;
            if (k >= n) k -= n;
        }
    }
    re = lane_sum(re, shift);
    im = lane_sum(im, shift);
    if (node < n && sub == 0) {
        const bool flagged = fl[node] != 0;
        const double2 b = flagged ? make_double2(0.0, 0.0) : make_double2(re * rsn, im * rsn);
        cd->b[node] = b;
        if (!flagged) {                                    // the active rows in ascending order
            int before = 0;
            for (int k = 0; k <= node >> 5; ++k)
                before += __popc(k < node >> 5 ? bits[k] : bits[k] & ((1u << (node & 31)) - 1u));
            cd->active[node - before] = node;
            cd->b_active[node - before] = b;
        }
    }
    if (tid == kSolveThreads - 1) {
        info->n_active = n - a;
        info->n_flagged = a;
        info->im_residual_bits = 0ull;                     // the recovery kernel's blocks merge their maxima into these
        info->re_max_bits = 0ull;
        if (info->status == DRACO_ETOOMANY) info->status = DRACO_OK;
    }
}


__global__ void __launch_bounds__(kSolveThreads)
cyc_decode_vector_kernel(CycDevice* cd, const uint8_t* __restrict__ flags, int n, int s, ModN mod, double rsn,
                         DeviceInfo* info) {
    pdl_begin();
    __shared__ double2 tw[kMaxN];
    __shared__ uint8_t fl[kMaxN];
    const int tid = threadIdx.x;
    if (tid < n) {
        tw[tid] = cd->twiddle[tid];
        fl[tid] = flags[tid];
    }
    __syncthreads();
    decode_vector_body(cd, fl, tw, n, s, mod, rsn, info);
}

// ------------------------------------------------------------------ locator after the projection
// One block; what bounds it is the length of the chain of dependent fp64 operations (9 cycles each), shuffles (46 a double)
// and barriers (59), not their number.  Sums over the nodes are therefore spread over as many lanes as the block has, lists
// come from ballots, and the systems of up to 8 unknowns are solved in one warp's registers.  n = 45, s = 5, five adversaries,
// decode vector included: 47 us with a thread per sum, one-thread list building and the singular-value iteration.
__global__ void __launch_bounds__(kSolveThreads)
cyc_solve_kernel(CycDevice* cd, const double2* __restrict__ e_in, const double2* __restrict__ partial, int used, int cap,
                 int n, int s, double theta, ModN mod, double rsn, uint8_t* flags, uint8_t* flags2, DeviceInfo* info, int with_b,
                 const uint8_t* sample_flags, const DeviceInfo* sample) {
    __shared__ double2 e[kMaxN], h[kMaxN + 1], tw[kMaxN];
    __shared__ double2 As[kSmallDim * kSmallDim], Vs[kSmallDim * kSmallDim];
    __shared__ double2 rhs_s[kMaxN / 2], beta_s[kMaxN / 2], coef_s[kMaxN / 2];
    __shared__ double mag[kMaxN], sorted[kMaxN], qv[kMaxN];
    __shared__ int sh[4], rank_s;
    __shared__ double maxsyn_s;
    const int tid = threadIdx.x;
    // lanes of one node, for the sums over the nodes
    const int shift = lanes_shift(n), per = 1 << shift, node = tid >> shift, sub = tid & (per - 1);

    if (tid < n) tw[tid] = cd->twiddle[tid];              // written when the plan was made: no need to wait
    pdl_begin();
    if (e_in != nullptr) {                                 // the projection record: n (re, im) pairs, then n values q_j
        if (tid < n) {
            e[tid] = e_in[tid];
            qv[tid] = reinterpret_cast<const double*>(e_in + n)[tid];
        }
    } else {
        // the projection's block partials, few enough to add up here: `lanes` lanes take one of the three sums of a node,
        // lane l the blocks l, l + lanes, .. in ascending order, eight loads in flight; then a butterfly: reproducible
        const double* __restrict__ qpartial = reinterpret_cast<const double*>(partial + (int64_t)cap * n);
        const int lshift = lanes_shift(3 * n), lanes = 1 << lshift, first = tid & (lanes - 1), groups = kSolveThreads >> lshift;
#pragma unroll 1
        for (int base = 0; base < 3 * n; base += groups) {
            const int idx = base + (tid >> lshift);
            const bool on = idx < 3 * n;
            const int part = idx < n || !on ? 0 : idx < 2 * n ? 1 : 2, j = on ? idx - part * n : 0;
            double acc = 0.0;
#pragma unroll 1
            for (int b0 = first; b0 < used; b0 += 8 * lanes) {
                double v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int b = b0 + k * lanes;
                    const int64_t at = (int64_t)(b < used ? b : b0) * n + j;
                    v[k] = part == 2 ? __ldcg(qpartial + at) : (part == 0 ? __ldcg(&partial[at].x) : __ldcg(&partial[at].y));
                }
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (b0 + k * lanes < used) acc += v[k];
            }
            acc = lane_sum(acc, lshift);
            if (on && first == 0) {
                if (part == 0) e[j].x = acc;
                else if (part == 1) e[j].y = acc;
                else qv[j] = acc;
            }
        }
    }
    __syncthreads();
    // A node whose record is not finite sent NaN or infinities: no honest vector does.  It is flagged outright and
    // its record taken as zero, which keeps the arithmetic below finite (the node then looks to the locator as if it
    // had sent a vector with f R_j = 0: one of the at most s errors it locates anyway).
    __shared__ uint8_t fl_s[kMaxN];                        // V so far
    if (tid < n) {
        const bool bad = !(isfinite(e[tid].x) && isfinite(e[tid].y) && isfinite(qv[tid]));
        fl_s[tid] = bad ? 1 : 0;
        if (bad) {
            e[tid] = make_double2(0.0, 0.0);
            qv[tid] = 0.0;
        }
        mag[tid] = sqrt(qv[tid]);
        h[tid] = make_double2(0.0, 0.0);
    }
    if (tid == 0) sh[3] = 0;
    __syncthreads();
    __shared__ double2 syn[kMaxN];                         // h_{n-2s+i}: every pass rewrites h
    {
        // scale = median of q_j^(1/2) by rank counting
        int rank = 0;
        if (node < n)
#pragma unroll 1
            for (int k = sub; k < n; k += per) rank += (mag[k] < mag[node]) || (mag[k] == mag[node] && k < node);
#pragma unroll 1
        for (int off = per >> 1; off > 0; off >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, off);
        if (node < n && sub == 0) sorted[rank] = mag[node];
        // syndromes h_m = n^(-1/2) sum_j e_j w^(-m j), m = n-2s .. n-1
        const int lshift = lanes_shift(2 * s), lanes = 1 << lshift, i = tid >> lshift, first = tid & (lanes - 1);
        double a = 0.0, b = 0.0;
        if (i < 2 * s) {
            const int m = n - 2 * s + i;
            int idx = mod(first * m);                      // (m j) mod n
            const int step = mod(lanes * m);
#pragma unroll 1
            for (int j = first; j < n; j += lanes) {
                const double2 q = cmulc(e[j], tw[idx]);
                a += q.x;
                b += q.y;
                idx += step;
                if (idx >= n) idx -= n;
            }
        }
        a = lane_sum(a, lshift);
        b = lane_sum(b, lshift);
        if (i < 2 * s && first == 0) syn[i] = make_double2(a * rsn, b * rsn);
    }
    __syncthreads();
    const double scale = (n & 1) ? sorted[n / 2] : 0.5 * (sorted[n / 2 - 1] + sorted[n / 2]);
    if (tid >= kSolveThreads - 32) {                       // the last warp, which the passes below leave idle
        const int lane = tid & 31;
        double mx = 0.0;
#pragma unroll 1
        for (int i = lane; i < 2 * s; i += 32) mx = fmax(mx, cabs2(syn[i]));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        if (lane == 0) maxsyn_s = sqrt(mx);
    }
    const double tol = theta * scale;
    // The locator runs in passes.  The first is the paper's phi.  Each further pass treats the set E of nodes flagged
    // so far (nodes with a non-finite record from the start) as erasures: with lambda(x) = prod_{v in E} (x - w^v) =
    // sum_k lambda_k x^k the sequence T_m = sum_k lambda_k h_{m-k} no longer contains the nodes of E and is again a sum
    // of exponentials, one per adversary not yet flagged, so its last 2 s2 values, s2 = floor((2 s - |E|) / 2), go
    // through the same Toeplitz system, recurrence and IDFT with s2 in place of s.  A pass that finds nothing (the
    // usual second pass: rounding noise) ends the search.  Adversaries that sit side by side make one pass miss some of
    // them with complex64 vectors; the passes then still end with a set that contains them all.
    __shared__ double2 lam[kMaxN + 2];
    __shared__ int elist[kMaxN];
    __shared__ uint32_t bits[kMaxN / 32];
    __shared__ double lam1_s, weakest_s, strongest_s;
    int rank_total = 0, sweeps = 0;                        // the same in every thread
    bool first = true, has_margin = false;
#pragma unroll 1
    for (int pass = 0; pass <= 2 * s && s > 0; ++pass) {
        const int eps = __syncthreads_count(tid < n && fl_s[tid] != 0);
        const int s2 = (2 * s - eps) / 2;
        if (s2 < 1) break;
        if (eps == 0) {                                    // T = h
            if (tid < 2 * s) h[n - 2 * s + tid] = syn[tid];
            if (tid == 0) lam1_s = 1.0;
        } else {
            // lambda: one factor (x - w^v) at a time, new_k = old_{k-1} - w^v old_k
            list_flagged(fl_s, n, elist, bits);
            if (eps < 32) {                                // lambda_k in lane k of the first warp
                if (tid < 32) {
                    double2 l = make_double2(tid == 0 ? 1.0 : 0.0, 0.0);
#pragma unroll 1
                    for (int a = 0; a < eps; ++a) {
                        const double2 q = cmul(tw[elist[a]], l);
                        const double px = __shfl_up_sync(0xffffffffu, l.x, 1), py = __shfl_up_sync(0xffffffffu, l.y, 1);
                        l = make_double2((tid > 0 ? px : 0.0) - q.x, (tid > 0 ? py : 0.0) - q.y);
                    }
                    lam[tid] = l;
                }
            } else {
                if (tid <= eps) lam[tid] = make_double2(tid == 0 ? 1.0 : 0.0, 0.0);
                __syncthreads();
#pragma unroll 1
                for (int a = 0; a < eps; ++a) {
                    double2 nv = make_double2(0.0, 0.0);
                    if (tid <= a + 1) {
                        const double2 wv = tw[elist[a]];
                        const double2 prev = tid > 0 ? lam[tid - 1] : make_double2(0.0, 0.0);
                        const double2 cur = tid <= a ? lam[tid] : make_double2(0.0, 0.0);
                        const double2 q = cmul(wv, cur);
                        nv = make_double2(prev.x - q.x, prev.y - q.y);
                    }
                    __syncthreads();
                    if (tid <= a + 1) lam[tid] = nv;
                    __syncthreads();
                }
            }
            __syncthreads();
            if (tid < n) {                                 // T_m on its window m = n - 2 s2 .. n - 1, zero before it
                double a = 0.0, b = 0.0;
                if (tid >= n - 2 * s2)
#pragma unroll 1
                    for (int k = 0; k <= eps; ++k) {
                        const double2 q = cmul(lam[k], syn[tid - k - (n - 2 * s)]);
                        a += q.x;
                        b += q.y;
                    }
                h[tid] = make_double2(a, b);
            } else if (tid >= kSolveThreads - 32) {
                double acc = 0.0;
#pragma unroll 1
                for (int k = tid & 31; k <= eps; k += 32) acc += sqrt(cabs2(lam[k]));
                acc = warp_sum(acc);
                if ((tid & 31) == 0) lam1_s = acc;
            }
        }
        __syncthreads();
        const double cut = tol * lam1_s;                   // the rounding noise of h enters T through |lambda_k|
        // row i of the system: [h_{n-s2-1-i} .. h_{n-2-i}] beta = h_{n-1-i}.  No singular value exceeds the Frobenius norm:
        // when that is within the cutoff (the usual step without any adversary, and the usual last pass: rounding noise) the
        // rank is 0 and nothing is solved.
        const int sp = s2 + (s2 & 1);
        if (sp <= kSmallDim) {
            if (tid < 32) {
                double fro2 = 0.0;
                if (tid < 2 * s2 - 1) {                    // h_{n-2 s2+i} stands in the matrix once per anti-diagonal entry
                    const int times = tid < s2 ? tid + 1 : 2 * s2 - 1 - tid;
                    fro2 = times * cabs2(h[n - 2 * s2 + tid]);
                }
                fro2 = warp_sum(fro2);
                int rank = 0, swept = 0;
                if (fro2 > cut * cut) {
                    const bool done = s2 <= kRegSystem && warp_full_rank_solve(As, h, n, s2, cut, fro2, beta_s);
                    if (done) {
                        rank = s2;
                    } else {                               // stored by columns
#pragma unroll 1
                        for (int idx = tid; idx < sp * sp; idx += 32) {
                            const int c = idx / sp, i = idx % sp;
                            As[idx] = (c < s2 && i < s2) ? h[n - s2 - 1 - i + c] : make_double2(0.0, 0.0);
                        }
                        if (tid < s2) rhs_s[tid] = h[n - 1 - tid];
                        __syncwarp();
                        rank = warp_jacobi_pinv(As, Vs, rhs_s, s2, cut, beta_s, coef_s, sh);
                        swept = sh[3];
                    }
                }
                if (tid == 0) { rank_s = rank; sh[3] = swept; }
            }
            __syncthreads();
        } else {
            double2* A = cd->work;
#pragma unroll 1
            for (int idx = tid; idx < sp * sp; idx += blockDim.x) {
                const int c = idx / sp, i = idx % sp;
                A[idx] = (c < s2 && i < s2) ? h[n - s2 - 1 - i + c] : make_double2(0.0, 0.0);
            }
            if (tid < s2) rhs_s[tid] = h[n - 1 - tid];
            if (tid == 0) sh[3] = 0;
            __syncthreads();
            if (tid < 32) {
                double fro2 = 0.0;
#pragma unroll 1
                for (int idx = tid; idx < sp * sp; idx += 32) fro2 += cabs2(A[idx]);
                fro2 = warp_sum(fro2);
                if (tid == 0) sh[2] = (fro2 > cut * cut) ? 1 : 0;
            }
            __syncthreads();
            int rank = 0;
            if (sh[2]) rank = block_jacobi_pinv(A, cd->work + sp * sp, rhs_s, s2, cut, beta_s, coef_s, sh);
            if (tid == 0) rank_s = rank;
            __syncthreads();
        }
        const int rank = rank_s;
        // sweeps of the longest iteration; negative once one hit the limit
        if (sh[3] < 0) sweeps = sh[3];
        else if (sweeps >= 0 && sh[3] > sweeps) sweeps = sh[3];
        if (rank == 0) break;
        if (tid == 0) {
            const int count = n - 2 * s2;
            if (s2 <= kRegSystem) {
#define DRACO_RECUR(S) run_recurrence<S>(h, n, count, beta_s)
                DRACO_BY_SIZE(s2, DRACO_RECUR)
#undef DRACO_RECUR
            } else {
                run_recurrence_any(h, n, count, s2, beta_s);
            }
        }
        __syncthreads();
        {
            double a = 0.0, b = 0.0;
            if (node < n) {
                int idx = mod(sub * node);                 // (node m) mod n
                const int step = mod(per * node);
#pragma unroll 1
                for (int m = sub; m < n; m += per) {
                    const double2 q = cmul(h[m], tw[idx]);
                    a += q.x;
                    b += q.y;
                    idx += step;
                    if (idx >= n) idx -= n;
                }
            }
            a = lane_sum(a, shift);
            b = lane_sum(b, shift);
            // |t_j|^2; nodes already in V are not candidates
            if (node < n && sub == 0) mag[node] = fl_s[node] ? -1.0 : cabs2(make_double2(a * rsn, b * rsn));
        }
        __syncthreads();
        // exactly `rank` entries of t are non-zero in exact arithmetic: the rank largest |t_j| join V
        int pos = 0;
        if (node < n)
#pragma unroll 1
            for (int k = sub; k < n; k += per) pos += (mag[k] > mag[node]) || (mag[k] == mag[node] && k < node);
#pragma unroll 1
        for (int off = per >> 1; off > 0; off >>= 1) pos += __shfl_xor_sync(0xffffffffu, pos, off);
        if (node < n && sub == 0) {
            if (first && pos == rank - 1) weakest_s = mag[node];    // |t|^2 of the weakest flagged node ..
            if (first && pos == rank) strongest_s = mag[node];      // .. and of the strongest unflagged one
            if (pos < rank) fl_s[node] = 1;
        }
        rank_total += rank;
        if (first) has_margin = rank < n - eps;
        first = false;
        __syncthreads();
    }
    __syncthreads();
    if (tid < n) {
        if (flags) flags[tid] = fl_s[tid];
        if (flags2) flags2[tid] = fl_s[tid];
    }
    const int count = __syncthreads_count(tid < n && fl_s[tid] != 0);
    if (tid == kSolveThreads - 1) {
        info->n_flagged = count;
        info->locator_rank = rank_total;
        info->scale = scale;
        info->max_syndrome = maxsyn_s;
        const double margin = has_margin ? sqrt(weakest_s / fmax(strongest_s, 1e-300)) : 1e300;
        // exactly `rank` entries of t are non-zero in exact arithmetic: where the weakest flagged and the strongest
        // unflagged |t_j| of the first pass are less than a decade apart the choice of V is not to be trusted, nor is a
        // rank that comes from an iteration that was stopped at its sweep limit
        info->status = (margin >= kMarginBar && sweeps >= 0) ? DRACO_OK : DRACO_EUNSURE;
        info->no_majority = 0;
        info->locator_margin = margin;
        info->svd_sweeps = sweeps;
        info->im_residual_bits = 0ull;                     // a decode's self-check belongs to the locate before it
        info->re_max_bits = 0ull;
    }
    if (with_b) {                                          // the decode vector for the V just found, same launch
        __syncthreads();
        decode_vector_body(cd, fl_s, tw, n, s, mod, rsn, info);
        if (sample != nullptr) {                           // u has been written for the sample's V, if there was a decode vector
            const int differ = __syncthreads_count(tid < n && fl_s[tid] != sample_flags[tid]);
            if (tid == kSolveThreads - 1) {
                info->combine = info->n_active;
                if (differ == 0 && sample->status != DRACO_ETOOMANY) {
                    info->im_residual_bits = sample->im_residual_bits;
                    info->re_max_bits = sample->re_max_bits;
                    info->combine = -1;
                }
            }
        }
    }
}

}  // namespace

// Capacity in blocks of the projection's partials: four per SM.
int project_grid_size(int sm_count) { return sm_count * 4; }

// Blocks along x of a projection, cap at most, each leaving one partial per node: no more than have work, so that short
// vectors leave a handful of partials.  n <= 16: a chunk per warp; as many blocks as are resident at once (three per SM) with
// the chunks dealt out evenly.  Otherwise a tile per block.  Short vectors take smaller tiles, whose warps are through after one
// round of loads (d = 4096, n = 45: four rounds one after the other with the full tile), and so do those whose full tiles
// would not occupy the device twice over, once the locator kernel would not add their few partials up itself (n = 45,
// reduction included: d = 200 k 42 -> 26 us, 600 k 65 -> 50 us; n = 105, d = 100 k 42 -> 34 us; but 1 M, where small tiles are
// four rounds of blocks, 62 -> 69 us, and n = 45, d = 60 k, where they cost the reduction a kernel, 32 -> 37 us with the decode).
struct ProjectShape {
    int grid, gridy, tile;
};
static ProjectShape project_shape(int cap, int sm_count, int64_t len, int n) {
    ProjectShape g = {1, 1, kProjectTile};
    if (n <= kFewRows) {
        const int64_t work = (len + (int64_t)kProjectChunk * kProjectWarps - 1) / ((int64_t)kProjectChunk * kProjectWarps);
        int64_t room = 3 * (int64_t)sm_count;
        if (room > cap) room = cap;
        const int64_t rounds = (work + room - 1) / room;
        g.grid = (int)((work + rounds - 1) / rounds);
        g.gridy = (int)(3 * (int64_t)sm_count / g.grid);     // what is left over divides the rows
        if (g.gridy > n) g.gridy = n;
        if (g.gridy < 1) g.gridy = 1;
        return g;
    }
    int64_t work = (len + kProjectTile - 1) / kProjectTile;
    const int64_t work_short = (len + kProjectTileShort - 1) / kProjectTileShort;
    if (work_short <= 64 || (3 * n * work > kFusedReduceMax && work_short <= 2 * (int64_t)cap)) {
        g.tile = kProjectTileShort;
        work = work_short;
    }
    g.grid = (int)(work < cap ? work : cap);
    return g;
}

// All launches of one projection: n <= 16 the few-rows kernel, n <= 64 one launch of the tile kernel, otherwise two
// launches of it over half the rows each.  partial: [cap][n] double2 followed by [cap][n] double.
static cudaError_t launch_project_kernels(int cap, const ProjectShape& shape, cudaStream_t st, const float2* R, const float* f,
                                          int64_t len, int64_t ld, int n, double2* partial, int accumulate, int every = 1) {
    const bool vec2 = (ld % 2 == 0);
    const int grid = shape.grid, tile = shape.tile;
    if (n <= kFewRows) {
        const dim3 grid2(grid, shape.gridy);
#define DRACO_FEW(VV, SS) launch_dependent(cyc_project_fewrows_kernel<VV, SS>, grid2, kThreads, 0, st, R, f, len, ld, n, partial, cap, accumulate, every)
        if (shape.gridy > 1) {
            if (vec2) DRACO_FEW(true, true); else DRACO_FEW(false, true);
        } else {
            if (vec2) DRACO_FEW(true, false); else DRACO_FEW(false, false);
        }
#undef DRACO_FEW
        return cudaGetLastError();
    }
    const int parts = n <= 64 ? 1 : 2;
    const int per = (n + parts - 1) / parts;
    // fewer tiles than an eighth of the blocks the device takes: spread the rows over gridDim.y too (latency of short vectors)
    int ysplit = 1;
    if (grid * 8 <= cap) {
        ysplit = (per + kProjectWarps - 1) / kProjectWarps;
        const int room = cap / (2 * grid);
        if (ysplit > room) ysplit = room;
        if (ysplit < 1) ysplit = 1;
    }
    const dim3 grid2(grid, ysplit);
#define DRACO_PROJECT(RR, VV, TT) \
    launch_dependent(cyc_project_kernel<RR, VV, TT>, grid2, kThreads, 0, st, R, f, len, ld, n, row0, nrows, partial, cap, accumulate, every)
#define DRACO_PROJECT_TILE(RR, VV)                                           \
    do {                                                                     \
        if (tile == kProjectTile) DRACO_PROJECT(RR, VV, kProjectTile);       \
        else DRACO_PROJECT(RR, VV, kProjectTileShort);                       \
    } while (0)
    for (int row0 = 0; row0 < n; row0 += per) {
        const int nrows = (n - row0) < per ? (n - row0) : per;
        if (nrows <= 32) {
            if (vec2) DRACO_PROJECT_TILE(4, true);
            else DRACO_PROJECT_TILE(4, false);
        } else {
            if (vec2) DRACO_PROJECT_TILE(8, true);
            else DRACO_PROJECT_TILE(8, false);
        }
#undef DRACO_PROJECT_TILE
#undef DRACO_PROJECT
        const cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

// accumulate: add to the partials of the plan's earlier launches (column chunks of one vector).  A chunk that needs
// more blocks than any before it finds the extra slots cleared first.
int launch_cyc_project(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, bool accumulate,
                       cudaStream_t st) {
    const int cap = p->project_grid;
    const ProjectShape shape = project_shape(cap, p->sm_count, len, p->n);
    const int want = shape.grid;
    if (!accumulate) p->project_used = 0;
    if (accumulate && want > p->project_used) {
        const size_t n = (size_t)p->n;
        DRACO_CUDA(cudaMemsetAsync(p->partial_dev + (size_t)p->project_used * n, 0,
                                   sizeof(double2) * n * (size_t)(want - p->project_used), st));
        double* q = reinterpret_cast<double*>(p->partial_dev + (size_t)cap * n);
        DRACO_CUDA(cudaMemsetAsync(q + (size_t)p->project_used * n, 0, sizeof(double) * n * (size_t)(want - p->project_used), st));
    }
    DRACO_CUDA(launch_project_kernels(cap, shape, st, R, f, len, ld, p->n, p->partial_dev, accumulate ? 1 : 0));
    if (want > p->project_used) p->project_used = want;
    return DRACO_OK;
}

static ModN mod_n(int n) { return ModN{(uint32_t)n, (uint32_t)(((1ull << 32) + (uint64_t)n - 1) / (uint64_t)n)}; }

// The locator and the decode vector from a sample of R's columns, tiles spread over the whole length: the flags to the second half
// of flags_dev, the status to info_dev[1].  As many tiles as the locator kernel adds up itself, 48 at most (24,576 coordinates),
// n <= 16: sixteen blocks (65,536); the sums over them are as telling as those of a vector of that length.
int launch_cyc_sample(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, cudaStream_t st) {
    const int n = p->n, cap = p->project_grid;
    const bool few = n <= kFewRows;
    int blocks = few ? 16 : kFusedReduceMax / (3 * n);
    if (blocks > 48) blocks = 48;
    const int64_t sample = (int64_t)blocks * (few ? kProjectChunk * kProjectWarps : kProjectTileShort);
    const int64_t every = len < sample ? 1 : len / sample;
    const ProjectShape shape = {blocks, few ? n : 1, kProjectTileShort};
    DRACO_CUDA(launch_project_kernels(cap, shape, st, R, f, len, ld, n, p->partial_dev, 0, (int)every));
    launch_dependent(cyc_solve_kernel, 1, kSolveThreads, 0, st, p->cyc_dev, nullptr, p->partial_dev, blocks, cap, n, p->s, p->theta,
                     mod_n(n), 1.0 / sqrt((double)n), nullptr, p->flags_dev + kMaxN, p->info_dev + 1, 1, nullptr, nullptr);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

int launch_cyc_project_finish(draco_plan* p, double2* e_out, cudaStream_t st) {
    launch_dependent(cyc_reduce_partials_kernel, p->n, kReduceThreads, 0, st, p->partial_dev, p->project_used,
                     p->project_grid, p->n, reinterpret_cast<double*>(e_out));
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

// e == nullptr: the record of the plan's own projection (launch_cyc_project) is formed first: by the locator kernel
// itself when the projection left few block partials (short vectors, where every launch counts), by the reduction
// kernel otherwise.  with_b: the decode vector for the set V just found is formed in the same launch.
int launch_cyc_solve(draco_plan* p, const double2* e, uint8_t* flags, bool with_b, cudaStream_t st, bool sampled) {
    const double2* partial = nullptr;
    int used = 0;
    if (!e) {
        if (3 * p->n * p->project_used <= kFusedReduceMax) {
            partial = p->partial_dev;
            used = p->project_used;
        } else {
            double2* own = reinterpret_cast<double2*>(p->cyc_dev->record);  // address arithmetic only: cyc_dev is a device pointer
            const int rc = launch_cyc_project_finish(p, own, st);
            if (rc != DRACO_OK) return rc;
            e = own;
        }
    }
    launch_dependent(cyc_solve_kernel, 1, kSolveThreads, 0, st, p->cyc_dev, e, partial, used, p->project_grid, p->n, p->s,
                     p->theta, mod_n(p->n), 1.0 / sqrt((double)p->n), flags, p->flags_dev, p->info_dev, with_b ? 1 : 0,
                     sampled ? p->flags_dev + kMaxN : nullptr, sampled ? p->info_dev + 1 : nullptr);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

int launch_cyc_decode_vector(draco_plan* p, const uint8_t* flags, cudaStream_t st) {
    launch_dependent(cyc_decode_vector_kernel, 1, kSolveThreads, 0, st, p->cyc_dev, flags, p->n, p->s, mod_n(p->n),
                     1.0 / sqrt((double)p->n), p->info_dev);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

}  // namespace draco

// ------------------------------------------------------------------ projection without any allocation
// Some callers must not allocate device memory at all: a parameter server embedded in a host
// process whose memory pool owner has handed out the whole device up front (a later cudaMalloc
// fails or fragments the pool), or a step loop that cannot afford the implicit device-wide
// synchronisation an allocation or a free may cause.  For them the block partials of the
// projection live in this fixed array instead of in a plan.  Every GPU that loads the library
// carries its 888 KB until the process exits.
namespace draco {
namespace {
constexpr int kStaticGridMax = 296;                                   // blocks whose partials fit
// per block and node one double2 (partial of e_j) and, after all of those, one double (partial of q_j)
static __device__ __align__(256) double2 g_static_partial[kStaticGridMax * kMaxN * 3 / 2];
constexpr int kMaxDevices = 64;
double2* g_static_partial_ptr[kMaxDevices] = {};                      // device address per device, set once
int g_static_sm_count[kMaxDevices] = {};
std::mutex g_static_mutex;
}  // namespace
}  // namespace draco

extern "C" int draco_cyc_project_noalloc(int n, int64_t d, const void* R, const float* f, double* e, void* stream) {
    using namespace draco;
    if (n < 1 || d < 1 || !R || !f || !e) return DRACO_EINVAL;
    if (n > kMaxN) return DRACO_ELIMIT;                               // the static array holds at most kMaxN rows per block
    if ((reinterpret_cast<uintptr_t>(R) & 15u) || (reinterpret_cast<uintptr_t>(f) & 15u) ||
        (reinterpret_cast<uintptr_t>(e) & 15u))
        return DRACO_EINVAL;
    int dev = 0;
    DRACO_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return DRACO_ELIMIT;
    double2* partial = nullptr;
    int sms = 0;
    {
        // Set-up, once per device, with that device current.  In host code the array's name is only a
        // stand-in for the symbol; the kernel needs the device address, which the runtime looks up here.
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_partial_ptr[dev]) {
            double2* ptr = nullptr;
            DRACO_CUDA(cudaGetSymbolAddress((void**)&ptr, g_static_partial));
            int count = 0;
            DRACO_CUDA(cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev));
            g_static_sm_count[dev] = count;
            g_static_partial_ptr[dev] = ptr;
        }
        partial = g_static_partial_ptr[dev];
        sms = g_static_sm_count[dev];
    }
    int grid = project_grid_size(sms);
    if (grid > kStaticGridMax) grid = kStaticGridMax;
    if (grid < 1) grid = 1;
    cudaStream_t st = (cudaStream_t)stream;
    const float2* Rc = static_cast<const float2*>(R);
    // Every block that is launched writes its n partials and only those are read back, so nothing has
    // to be cleared between calls even though the array keeps the previous call's contents.
    const ProjectShape shape = project_shape(grid, sms, d, n);
    DRACO_CUDA(launch_project_kernels(grid, shape, st, Rc, f, d, d, n, partial, 0));
    launch_dependent(cyc_reduce_partials_kernel, n, kReduceThreads, 0, st, partial, shape.grid, grid, n, e);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}
