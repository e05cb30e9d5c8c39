// Cyclic-code recovery, Algorithm 1 step 4: u = Re(R_{.,U} b) for the decode vector b left
// in the plan's device state by the decode-vector kernel.
//
// One pass over the rows with b_j != 0.  The code cancels entries of W as large as 1e5 back
// to 1, so the running sums are kept in fp64 (fp32 would lose about kappa * 2^-24 of the
// result); R stays fp32 in memory.  HBM traffic: 8 |U| len bytes read + 4 len written.
//
// Self-check (unpacked plans).  u-hat = G 1_P is real, so Im(u-hat) is rounding residue as long as every
// row of U is honest, and of the size of the result when an adversary is left in U.  The kernel forms
// Im(u-hat_i) on one coordinate run in eight (floor(i / 64) mod 8 = 0, uniform in a warp) and leaves max |Im| and
// max |Re| over those coordinates in the plan's info block.  (The compiler predicates the extra multiply-adds
// instead of branching, so the fp64 pipe is 19 % busy instead of 10 %; the kernel stays memory-bound, and two
// specialised copies of the loop behind a real branch cost 118 registers instead of 80.)
#include "draco_internal.cuh"

namespace draco {

namespace {

constexpr int kThreads = 256;
constexpr int kUnroll = 8;
constexpr int kShortCoordinates = 300;   // per SM: up to this length the short kernel is the faster one ..
constexpr int kShortFewRows = 140;       // .. and with at most 16 rows

// PACKED: the vectors carry two gradient coordinates per complex entry (Section 3, last
// paragraph): u[i] = Re(u-hat_i), u[len + i] = Im(u-hat_i) for len + i < d_packed.
// VEC2: a thread owns two neighbouring coordinates, one 16-byte load per row.  Otherwise (odd row starts) two coordinates
// kThreads apart and two 8-byte loads per row, so that a warp's loads are contiguous and as many bytes are in flight (one
// coordinate per thread and no batch of rows: n = 45, d = 20,000,001 1589 us with the decode vector, now 1107).
// ONCE: u may have been written already, beside the projection; the others do without the look (1 % of 1 M coordinates).
template <bool VEC2, bool PACKED, bool ONCE>
__global__ void __launch_bounds__(kThreads)
cyc_recover_kernel(const float2* __restrict__ R, int64_t len, int64_t ld, const CycDevice* __restrict__ cd,
                   DeviceInfo* info, float* __restrict__ u, int64_t d_packed, float* __restrict__ w, float scale) {
    pdl_begin();
    __shared__ double2 bs[kMaxN];
    __shared__ int rows[kMaxN];
    const int count = ONCE ? info->combine : info->n_active;
    if (ONCE && count < 0) return;
    double im_max = 0.0, re_max = 0.0;                    // over this thread's sampled coordinates
    for (int k = threadIdx.x; k < count; k += kThreads) {
        bs[k] = cd->b_active[k];
        rows[k] = cd->active[k];
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    // Two loops and not one with its addresses chosen by VEC2: that form was 0.5 - 1.5 % slower on long vectors (n = 45, s = 3,
    // d = 60.2 M, update 3396 us, 3331 so; n = 15, s = 2 1194 and 1166).
    if constexpr (VEC2) {
        const int64_t nvec = len / 2;
        for (int64_t v = (int64_t)blockIdx.x * kThreads + threadIdx.x; v < nvec; v += stride) {
            const float2* col = R + v * 2;
            const bool sampled = !PACKED && ((v >> 5) & 7) == 0;       // coordinates 2 v, 2 v + 1: floor(i / 64) mod 8 == 0
            double a0 = 0.0, a1 = 0.0, i0 = 0.0, i1 = 0.0;
            for (int k0 = 0; k0 < count; k0 += kUnroll) {
                float4 x[kUnroll];
#pragma unroll
                for (int q = 0; q < kUnroll; ++q)
                    if (k0 + q < count) x[q] = __ldcs(reinterpret_cast<const float4*>(col + (int64_t)rows[k0 + q] * ld));
#pragma unroll
                for (int q = 0; q < kUnroll; ++q)
                    if (k0 + q < count) {
                        const double2 b = bs[k0 + q];
                        const double xr0 = (double)x[q].x, xi0 = (double)x[q].y, xr1 = (double)x[q].z, xi1 = (double)x[q].w;
                        a0 = fma(b.x, xr0, a0);
                        a0 = fma(-b.y, xi0, a0);
                        a1 = fma(b.x, xr1, a1);
                        a1 = fma(-b.y, xi1, a1);
                        if (PACKED || sampled) {
                            i0 = fma(b.x, xi0, i0);
                            i0 = fma(b.y, xr0, i0);
                            i1 = fma(b.x, xi1, i1);
                            i1 = fma(b.y, xr1, i1);
                        }
                    }
            }
            if (sampled) {
                im_max = fmax(im_max, fmax(magnitude(i0), magnitude(i1)));
                re_max = fmax(re_max, fmax(magnitude(a0), magnitude(a1)));
            }
            if (u != nullptr) {
                __stcs(reinterpret_cast<float2*>(u + v * 2), make_float2((float)a0, (float)a1));
                if (PACKED) __stcs(reinterpret_cast<float2*>(u + len + v * 2), make_float2((float)i0, (float)i1));
            }
            if (w != nullptr) {                          // w <- w - scale * u, u rounded to fp32 first as when stored
                float2* wp = reinterpret_cast<float2*>(w + v * 2);
                float2 wv = *wp;
                wv.x = fmaf(-scale, (float)a0, wv.x);
                wv.y = fmaf(-scale, (float)a1, wv.y);
                *wp = wv;
                if (PACKED) {
                    wp = reinterpret_cast<float2*>(w + len + v * 2);
                    wv = *wp;
                    wv.x = fmaf(-scale, (float)i0, wv.x);
                    wv.y = fmaf(-scale, (float)i1, wv.y);
                    *wp = wv;
                }
            }
        }
    } else {
        for (int64_t c0 = (int64_t)blockIdx.x * 2 * kThreads; c0 < len; c0 += 2 * stride) {
            const int64_t i = c0 + threadIdx.x;
            if (i >= len) continue;
            const bool two = i + kThreads < len;
            const int step = two ? kThreads : 0;         // beyond the vector: the first coordinate again
            const bool sampled = !PACKED && ((i >> 6) & 7) == 0;       // the second coordinate is four runs of 64 on, never sampled
            const bool im0 = PACKED && len + i < d_packed, im1 = PACKED && two && len + i + step < d_packed;
            float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f;
            if (w != nullptr) {                          // under way beside the rows
                w0 = w[i];
                w1 = w[i + step];
                if (im0) w2 = w[len + i];
                if (im1) w3 = w[len + i + step];
            }
            const float2* col = R + i;
            double a0 = 0.0, a1 = 0.0, i0 = 0.0, i1 = 0.0;
            for (int k0 = 0; k0 < count; k0 += kUnroll) {
                float4 x[kUnroll];
#pragma unroll
                for (int q = 0; q < kUnroll; ++q)
                    if (k0 + q < count) {
                        const float2* row = col + (int64_t)rows[k0 + q] * ld;
                        const float2 y0 = __ldcs(row), y1 = __ldcs(row + step);
                        x[q] = make_float4(y0.x, y0.y, y1.x, y1.y);
                    }
#pragma unroll
                for (int q = 0; q < kUnroll; ++q)
                    if (k0 + q < count) {
                        const double2 b = bs[k0 + q];
                        const double xr0 = (double)x[q].x, xi0 = (double)x[q].y, xr1 = (double)x[q].z, xi1 = (double)x[q].w;
                        a0 = fma(b.x, xr0, a0);
                        a0 = fma(-b.y, xi0, a0);
                        a1 = fma(b.x, xr1, a1);
                        a1 = fma(-b.y, xi1, a1);
                        if (PACKED || sampled) {
                            i0 = fma(b.x, xi0, i0);
                            i0 = fma(b.y, xr0, i0);
                            if (PACKED) {
                                i1 = fma(b.x, xi1, i1);
                                i1 = fma(b.y, xr1, i1);
                            }
                        }
                    }
            }
            if (sampled) {
                im_max = fmax(im_max, magnitude(i0));
                re_max = fmax(re_max, magnitude(a0));
            }
            if (u != nullptr) {
                u[i] = (float)a0;
                if (two) u[i + step] = (float)a1;
                if (im0) u[len + i] = (float)i0;
                if (im1) u[len + i + step] = (float)i1;
            }
            if (w != nullptr) {
                w[i] = fmaf(-scale, (float)a0, w0);
                if (two) w[i + step] = fmaf(-scale, (float)a1, w1);
                if (im0) w[len + i] = fmaf(-scale, (float)i0, w2);
                if (im1) w[len + i + step] = fmaf(-scale, (float)i1, w3);
            }
        }
    }
    if (!PACKED) {
        // non-negative doubles order like their bit patterns
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            im_max = fmax(im_max, __shfl_xor_sync(0xffffffffu, im_max, off));
            re_max = fmax(re_max, __shfl_xor_sync(0xffffffffu, re_max, off));
        }
        if ((threadIdx.x & 31) == 0) {
            if (im_max > 0.0) atomicMax(&info->im_residual_bits, (unsigned long long)__double_as_longlong(im_max));
            if (re_max > 0.0) atomicMax(&info->re_max_bits, (unsigned long long)__double_as_longlong(re_max));
        }
    }
}

// The same for short vectors, whose time is a chain of load latencies (five batches of eight rows one after the other at
// n = 45): a block takes 64 coordinates, its warps the rows w, w + 8, .., all loads of a warp in flight together; the
// warps' sums are added in ascending order.  Where the lines lie, locate and decode, the other kernel / this one in us: n = 45,
// s = 5, d = 10,000 22.0 / 21.6, 20,000 26.9 / 24.3, 40,000 34.5 / 31.6, but 50,000 34.4 / 37.0, 94,000 46 / 58; n = 105, s = 2,
// 31,000 53 / 50, 60,000 73 / 88, 94,000 96 / 125; n = 15, s = 2, 20,000 17.0 / 17.2, 31,000 17.4 / 19.7, 94,000 21.5 / 27.5.
constexpr int kShortBatch = 8;
template <bool VEC2, bool PACKED>
__global__ void __launch_bounds__(kThreads)
cyc_recover_short_kernel(const float2* __restrict__ R, int64_t len, int64_t ld, const CycDevice* __restrict__ cd,
                         DeviceInfo* info, float* __restrict__ u, int64_t d_packed, float* __restrict__ w, float scale) {
    pdl_begin();
    constexpr int kWarps = kThreads / 32;
    __shared__ double sums[kWarps][4][32];                // a0, a1, i0, i1 of every lane
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int count = info->n_active;
    const int64_t c0 = (int64_t)blockIdx.x * 64;
    const int64_t i = c0 + (VEC2 ? 2 * lane : lane);
    const bool in0 = i < len, in1 = VEC2 ? in0 : i + 32 < len;
    const bool sampled = !PACKED && (blockIdx.x & 7) == 0;             // floor(i / 64) mod 8 == 0
    double a0 = 0.0, a1 = 0.0, i0 = 0.0, i1 = 0.0;
    for (int k0 = warp; k0 < count; k0 += kWarps * kShortBatch) {
        float4 x[kShortBatch];
        double2 b[kShortBatch];
#pragma unroll
        for (int q = 0; q < kShortBatch; ++q) {
            const int k = k0 + q * kWarps;
            x[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int slot = k < kMaxN ? k : 0;            // read beside `count`, not after it
            const int node = cd->active[slot];
            b[q] = cd->b_active[slot];
            if (k < count) {
                const float2* row = R + (int64_t)node * ld + i;
                if (VEC2) {
                    if (in0) x[q] = __ldcs(reinterpret_cast<const float4*>(row));
                } else {
                    const float2 y0 = in0 ? __ldcs(row) : make_float2(0.f, 0.f), y1 = in1 ? __ldcs(row + 32) : make_float2(0.f, 0.f);
                    x[q] = make_float4(y0.x, y0.y, y1.x, y1.y);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kShortBatch; ++q)
            if (k0 + q * kWarps < count) {
                const double xr0 = (double)x[q].x, xi0 = (double)x[q].y, xr1 = (double)x[q].z, xi1 = (double)x[q].w;
                a0 = fma(-b[q].y, xi0, fma(b[q].x, xr0, a0));
                a1 = fma(-b[q].y, xi1, fma(b[q].x, xr1, a1));
                if (PACKED || sampled) {
                    i0 = fma(b[q].y, xr0, fma(b[q].x, xi0, i0));
                    i1 = fma(b[q].y, xr1, fma(b[q].x, xi1, i1));
                }
            }
    }
    sums[warp][0][lane] = a0;
    sums[warp][1][lane] = a1;
    sums[warp][2][lane] = i0;
    sums[warp][3][lane] = i1;
    __syncthreads();
    // warp 0, 1: real parts of the first and second coordinates; 2, 3: imaginary parts
    if (warp >= (PACKED || sampled ? 4 : 2)) return;
    double a = 0.0;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) a += sums[q][warp][lane];
    const bool second = warp & 1, imag = warp >= 2;
    const bool in = second ? in1 : in0;
    const int64_t at = (imag ? len : 0) + i + (second ? (VEC2 ? 1 : 32) : 0);
    if (in && (PACKED ? (!imag || at < d_packed) : !imag)) {
        if (u != nullptr) u[at] = (float)a;
        if (w != nullptr) w[at] = fmaf(-scale, (float)a, w[at]);
    }
    if (sampled) {
        double m = in ? magnitude(a) : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
        if (lane == 0 && m > 0.0) atomicMax(imag ? &info->im_residual_bits : &info->re_max_bits, (unsigned long long)__double_as_longlong(m));
    }
}

}  // namespace

int launch_cyc_recover(draco_plan* p, const float2* R, int64_t len, int64_t ld, float* u, int64_t d_packed,
                       cudaStream_t st, float* w, float scale, bool once) {
    const bool packed = d_packed > 0;
    // 64-bit stores of u need len even; in packed mode the second half starts at u + len and must cover it fully
    const bool vec2 = (len % 2 == 0) && (ld % 2 == 0) && (!packed || d_packed == 2 * len);
    const int64_t nvec = (len + 1) / 2;
    int64_t want = (nvec + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)p->sm_count * 16;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
#define DRACO_REC_ONCE(V2, PK, ONCE) \
    launch_dependent(cyc_recover_kernel<V2, PK, ONCE>, (int)want, kThreads, 0, st, R, len, ld, p->cyc_dev, p->info_dev, u, d_packed, w, scale)
#define DRACO_REC(V2, PK)                                                                    \
    do {                                                                                     \
        if (once) DRACO_REC_ONCE(V2, PK, true); else DRACO_REC_ONCE(V2, PK, false);          \
    } while (0)
#define DRACO_REC_SHORT(V2, PK)                                                                                                    \
    launch_dependent(cyc_recover_short_kernel<V2, PK>, (int)((len + 63) / 64), kThreads, 0, st, R, len, ld, p->cyc_dev, p->info_dev, u, d_packed, w, \
                                                                                  scale)
    if (!once && len <= (int64_t)p->sm_count * (p->n <= 16 ? kShortFewRows : kShortCoordinates)) {
        if (vec2) {
            if (packed) DRACO_REC_SHORT(true, true); else DRACO_REC_SHORT(true, false);
        } else {
            if (packed) DRACO_REC_SHORT(false, true); else DRACO_REC_SHORT(false, false);
        }
    } else if (vec2) {
        if (packed) DRACO_REC(true, true); else DRACO_REC(true, false);
    } else {
        if (packed) DRACO_REC(false, true); else DRACO_REC(false, false);
    }
#undef DRACO_REC_ONCE
#undef DRACO_REC
#undef DRACO_REC_SHORT
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

}  // namespace draco
