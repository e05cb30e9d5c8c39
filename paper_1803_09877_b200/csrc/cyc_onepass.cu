// Cyclic code, locate and decode of long vectors with one read of R.
//
// The decode vector b depends on V = phi(R), and phi needs the projection of every coordinate: taken one after the other, the
// projection and the recovery read R twice.  The adversaries of a vector show in any sizeable part of it, though.  A long vector is
// therefore located on a sample of its columns first; the kernel below then reads R once and forms, from the same registers, the
// whole projection (e, q) and the sum that the sample's decode vector gives.  The locator runs again on the whole projection: V
// comes from all coordinates, as ever.  Where it is the sample's V, the sum is the one that the recovery would have formed and the
// recovery kernel returns at once; where it is not (an adversary that leaves the sampled columns alone), the recovery overwrites it
// with the sum for the right V, at the cost of the second read that was to be saved.  A sample in doubt (DRACO_EUNSURE: adversaries
// side by side from s = 5 on) is acted on like any other: only the comparison of V with V' says whether the sum stands.  Where the
// sample has more than 2 s nodes flagged there is no decode vector and the kernel only projects.
//
// Bound by HBM: 8 n + 4 bytes read and 4 written per coordinate (packed: per complex coordinate, 8 written).  Locate and decode, two
// reads / one: n = 45, s = 5, d = 60.2 M 6150 -> 3490 us (6.3 TB/s; with back-to-back passes 6300 -> 3640), packed 3180 -> 2150; d =
// 20,000,001, off the 16-byte grid, 2360 -> 1350; n = 15, s = 2, 30 M 1067 -> 651; n = 105, s = 2, 11.7 M 2970 -> 1635.  Tried and slower: one
// block per SM with twice the ring 3940, half the chunk per warp 4140 (each row's additions over the lanes are shared by half
// as many coordinates), half the ring 3580; warps that share a tile of 512 coordinates by rows, without additions over the
// lanes but with a barrier per tile, 3850.
#include "draco_internal.cuh"

namespace draco {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kBlocksPerSM = 2;
constexpr int kBatch = 8;             // rows whose lane sums are added up together

// K 16-byte items per lane and row: a warp takes 64 K coordinates.  kRing bytes of rows are on their way per warp.
template <bool PACKED>
struct OneCfg {
    static constexpr int K = PACKED ? 2 : 4;
    static constexpr int kChunk = 64 * K;
    static constexpr int kRowBytes = 512 * K;
    static constexpr int kRing = 8192;
    static constexpr int kDepth = kRing / kRowBytes;
};

// K items of a lane, 512 bytes apart on either side, or twice as many 8-byte pieces.  `after` is the sign and exponent word of a sum
// of squares that the values read from `dst` before went into: no such sum has kNever (a tiny negative number), so the copies are
// always made, and never before those reads are complete.
constexpr int kNever = (int)0x80001234;
template <int K, bool VEC2>
__device__ __forceinline__ void copy_row(uint32_t dst, const float2* src, int after) {
    if constexpr (VEC2 && K == 4) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, %3;\n\t"
            "@p cp.async.cg.shared.global [%0], [%1], 16;\n\t@p cp.async.cg.shared.global [%0 + 512], [%1 + 512], 16;\n\t"
            "@p cp.async.cg.shared.global [%0 + 1024], [%1 + 1024], 16;\n\t@p cp.async.cg.shared.global [%0 + 1536], [%1 + 1536], 16;\n\t}"
            ::"r"(dst), "l"(src), "r"(after), "n"(kNever) : "memory");
    } else if constexpr (VEC2) {
        static_assert(K == 2 || K == 4, "items of a lane");
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, %3;\n\t"
            "@p cp.async.cg.shared.global [%0], [%1], 16;\n\t@p cp.async.cg.shared.global [%0 + 512], [%1 + 512], 16;\n\t}"
            ::"r"(dst), "l"(src), "r"(after), "n"(kNever) : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q)
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, %3;\n\t"
                "@p cp.async.ca.shared.global [%0], [%1], 8;\n\t@p cp.async.ca.shared.global [%0 + 8], [%1 + 256], 8;\n\t}"
                ::"r"(dst + q * 512), "l"(src + q * 64), "r"(after), "n"(kNever) : "memory");
    }
}
// as cp_async8_if
__device__ __forceinline__ void cp_async16_if(uint32_t dst, const void* src, bool on) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %2, 0;\n\tcp.async.cg.shared.global [%0], [%1], 16, p;\n\t}" ::"r"(dst), "l"(src), "r"((uint32_t)on) : "memory");
}

struct Sums {
    double er, ei, q;
};
// Adds two rows' lane sums: lanes with bit `off` clear end with the first row's sums over the lane pair, the others with the second's.
__device__ __forceinline__ Sums merge(const Sums& x, const Sums& y, int off) {
    const bool hi = threadIdx.x & off;
    auto one = [&](double a, double b) { return (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, off); };
    return Sums{one(x.er, y.er), one(x.ei, y.ei), one(x.q, y.q)};
}

// Every warp walks chunks of 64 K coordinates on its own and visits the n rows of a chunk once.  Rows come through a private
// shared-memory column of asynchronous copies (kRing bytes per warp in flight, running on into the next chunk; lanes outside the
// vector have their source switched off and read zeros), so there is no barrier.  A lane owns its coordinates: the sum over the rows
// stays in its registers.  The sums over the coordinates, three per row, are added up over the lanes eight rows at a time, the
// rows spread over the lanes as the partial sums shrink (27 exchanges for eight rows instead of 120), and collected per warp.
// VEC2: a lane's item is two neighbouring coordinates (16 bytes); otherwise two coordinates 32 apart (rows off the 16-byte grid).
template <bool VEC2, bool PACKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
cyc_onepass_kernel(const float2* __restrict__ R, const float* __restrict__ f, int64_t len, int64_t ld, int n,
                   double2* __restrict__ partial, int cap, const CycDevice* __restrict__ cd, const uint8_t* __restrict__ flags,
                   DeviceInfo* sample, float* __restrict__ u, int64_t d_packed) {
    using Cfg = OneCfg<PACKED>;
    constexpr int K = Cfg::K, kRing = Cfg::kRing;
    extern __shared__ __align__(16) unsigned char smem[];             // ring[kWarps][kRing], sums[kWarps][n]
    __shared__ double2 bs[kMaxN];
    __shared__ uint8_t use[kMaxN];
    pdl_begin();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Sums* const acc_all = reinterpret_cast<Sums*>(smem + kWarps * kRing);
    Sums* const acc = acc_all + warp * n;
    const bool go = sample->status != DRACO_ETOOMANY;
    for (int j = threadIdx.x; j < n; j += kThreads) {
        bs[j] = cd->b[j];
        use[j] = go && !flags[j];
    }
    for (int j = lane; j < n; j += 32) acc[j] = Sums{0.0, 0.0, 0.0};
    __syncthreads();

    const int64_t nchunks = (len + Cfg::kChunk - 1) / Cfg::kChunk;
    const int64_t chunk0 = (int64_t)blockIdx.x * kWarps + warp, step = (int64_t)gridDim.x * kWarps;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem) + warp * kRing + lane * 16;
    // first coordinate of this lane's item q of a chunk
    auto coord = [&](int64_t chunk, int q) { return chunk * Cfg::kChunk + q * 64 + (VEC2 ? 2 * lane : lane); };

    // The fetch side: kDepth rows ahead of the row being consumed.
    int64_t fchunk = chunk0;
    const float2* fp = R;                                             // this lane's first coordinate in the next row
    int frow = 0, inside = 0;                                         // 2: the whole chunk lies in the vector, 0: past the last chunk
    uint32_t fslot = 0;
    auto open = [&]() {
        frow = 0;
        inside = fchunk >= nchunks ? 0 : (fchunk + 1) * Cfg::kChunk <= len ? 2 : 1;
        fp = R + (inside == 2 ? coord(fchunk, 0) : 0);
    };
    auto fetch = [&](int after) {
        const uint32_t dst = ring + fslot;
        if (inside == 2) {
            copy_row<K, VEC2>(dst, fp, after);
        } else if (inside == 1 && after != kNever) {                  // coordinates beyond the vector read zeros
#pragma unroll
            for (int q = 0; q < K; ++q) {
                const int64_t c = coord(fchunk, q);
                if constexpr (VEC2) {
                    cp_async16_if(dst + q * 512, fp + (c < len ? c : 0), c < len);
                } else {
                    cp_async8_if(dst + q * 512, fp + (c < len ? c : 0), c < len);
                    cp_async8_if(dst + q * 512 + 8, fp + (c + 32 < len ? c + 32 : 0), c + 32 < len);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        fslot = (fslot + Cfg::kRowBytes) & (kRing - 1);
        fp += ld;
        if (++frow == n) {
            fchunk += step;
            open();
        }
    };
    open();
#pragma unroll 1
    for (int k = 0; k < Cfg::kDepth; ++k) fetch(0);

    uint32_t slot = 0;
    double im_max = 0.0, re_max = 0.0;
    for (int64_t chunk = chunk0; chunk < nchunks; chunk += step) {
        double ff[K][2], a[K][2], b[K][2];                            // f; Re and Im of the sum over the rows
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const int64_t c = coord(chunk, q);
            if constexpr (VEC2) {
                const float2 v = c < len ? __ldcs(reinterpret_cast<const float2*>(f + c)) : make_float2(0.f, 0.f);
                ff[q][0] = (double)v.x;
                ff[q][1] = (double)v.y;
            } else {
                ff[q][0] = c < len ? (double)__ldcs(f + c) : 0.0;
                ff[q][1] = c + 32 < len ? (double)__ldcs(f + c + 32) : 0.0;
            }
            a[q][0] = a[q][1] = b[q][0] = b[q][1] = 0.0;
        }
        // the self-check's coordinates, floor(i / 64) mod 8 = 0: the first item of every other chunk
        const bool sampled = !PACKED && (chunk * K) % 8 == 0;
#pragma unroll 1
        for (int j0 = 0; j0 < n; j0 += kBatch) {
            Sums part[3], cur;
#pragma unroll
            for (int r = 0; r < kBatch; ++r) {
                cur = Sums{0.0, 0.0, 0.0};
                if (j0 + r < n) {
                    const bool used = use[j0 + r];
                    const double2 w = bs[j0 + r];
                    asm volatile("cp.async.wait_group %0;" ::"n"(Cfg::kDepth - 1) : "memory");
                    float4 x[K];
#pragma unroll
                    for (int q = 0; q < K; ++q) x[q] = lds128(ring + slot + q * 512);
                    slot = (slot + Cfg::kRowBytes) & (kRing - 1);
#pragma unroll
                    for (int q = 0; q < K; ++q) {
                        const double x0 = (double)x[q].x, y0 = (double)x[q].y, x1 = (double)x[q].z, y1 = (double)x[q].w;
                        cur.er = fma(ff[q][0], x0, cur.er); cur.ei = fma(ff[q][0], y0, cur.ei);
                        cur.er = fma(ff[q][1], x1, cur.er); cur.ei = fma(ff[q][1], y1, cur.ei);
                        cur.q = fma(x0, x0, cur.q); cur.q = fma(y0, y0, cur.q);
                        cur.q = fma(x1, x1, cur.q); cur.q = fma(y1, y1, cur.q);
                        if (used) {
                            a[q][0] = fma(w.x, x0, a[q][0]); a[q][0] = fma(-w.y, y0, a[q][0]);
                            a[q][1] = fma(w.x, x1, a[q][1]); a[q][1] = fma(-w.y, y1, a[q][1]);
                            if (PACKED || (q == 0 && sampled)) {
                                b[q][0] = fma(w.x, y0, b[q][0]); b[q][0] = fma(w.y, x0, b[q][0]);
                                b[q][1] = fma(w.x, y1, b[q][1]); b[q][1] = fma(w.y, x1, b[q][1]);
                            }
                        }
                    }
                    fetch(__double2hiint(cur.q));                     // refill the slot
                }
                if (r & 1) {
                    cur = merge(part[0], cur, 16);
                    if (r & 2) {
                        cur = merge(part[1], cur, 8);
                        if (r & 4) cur = merge(part[2], cur, 4);
                        else part[2] = cur;
                    } else {
                        part[1] = cur;
                    }
                } else {
                    part[0] = cur;
                }
            }
#pragma unroll
            for (int off = 2; off > 0; off >>= 1) {
                cur.er += __shfl_xor_sync(0xffffffffu, cur.er, off);
                cur.ei += __shfl_xor_sync(0xffffffffu, cur.ei, off);
                cur.q += __shfl_xor_sync(0xffffffffu, cur.q, off);
            }
            // lane bits 4, 3, 2: row bits 0, 1, 2
            const int j = j0 + ((lane >> 4) & 1) + ((lane >> 2) & 2) + (lane & 4);
            if ((lane & 3) == 0 && j < n) {
                Sums s = acc[j];
                s.er += cur.er; s.ei += cur.ei; s.q += cur.q;
                acc[j] = s;
            }
        }
        if (go) {
            if (sampled) {
                const int64_t c = coord(chunk, 0);
                const bool in0 = c < len, in1 = VEC2 ? in0 : c + 32 < len;
                im_max = fmax(im_max, fmax(in0 ? magnitude(b[0][0]) : 0.0, in1 ? magnitude(b[0][1]) : 0.0));
                re_max = fmax(re_max, fmax(in0 ? magnitude(a[0][0]) : 0.0, in1 ? magnitude(a[0][1]) : 0.0));
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                const int64_t c = coord(chunk, q);
                if constexpr (VEC2) {
                    if (c < len) {
                        __stcs(reinterpret_cast<float2*>(u + c), make_float2((float)a[q][0], (float)a[q][1]));
                        if (PACKED) __stcs(reinterpret_cast<float2*>(u + len + c), make_float2((float)b[q][0], (float)b[q][1]));
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int64_t i = c + 32 * k;
                        if (i < len) {
                            u[i] = (float)a[q][k];
                            if (PACKED && len + i < d_packed) u[len + i] = (float)b[q][k];
                        }
                    }
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (!PACKED) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            im_max = fmax(im_max, __shfl_xor_sync(0xffffffffu, im_max, off));
            re_max = fmax(re_max, __shfl_xor_sync(0xffffffffu, re_max, off));
        }
        if (lane == 0) {                                              // non-negative doubles order like their bit patterns
            if (im_max > 0.0) atomicMax(&sample->im_residual_bits, (unsigned long long)__double_as_longlong(im_max));
            if (re_max > 0.0) atomicMax(&sample->re_max_bits, (unsigned long long)__double_as_longlong(re_max));
        }
    }
    __syncthreads();
    double* const qpartial = reinterpret_cast<double*>(partial + (int64_t)cap * n);
    for (int j = threadIdx.x; j < n; j += kThreads) {
        Sums s = Sums{0.0, 0.0, 0.0};
        for (int w = 0; w < kWarps; ++w) {                            // fixed order: reproducible
            const Sums t = acc_all[w * n + j];
            s.er += t.er; s.ei += t.ei; s.q += t.q;
        }
        partial[(int64_t)blockIdx.x * n + j] = make_double2(s.er, s.ei);
        qpartial[(int64_t)blockIdx.x * n + j] = s.q;
    }
}

template <bool VEC2, bool PACKED>
int launch_onepass(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, float* u, int64_t d_packed, cudaStream_t st) {
    using Cfg = OneCfg<PACKED>;
    const int64_t nblocks = ((len + Cfg::kChunk - 1) / Cfg::kChunk + kWarps - 1) / kWarps;
    int64_t grid = (int64_t)p->sm_count * kBlocksPerSM;
    if (grid > p->project_grid) grid = p->project_grid;
    if (grid > nblocks) grid = nblocks;
    auto smem = [](int n) { return (size_t)kWarps * (Cfg::kRing + sizeof(Sums) * (size_t)n); };
    DRACO_CUDA(cudaFuncSetAttribute(cyc_onepass_kernel<VEC2, PACKED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(kMaxN)));
    launch_dependent(cyc_onepass_kernel<VEC2, PACKED>, (int)grid, kThreads, smem(p->n), st, R, f, len, ld, p->n, p->partial_dev,
                     p->project_grid, p->cyc_dev, p->flags_dev + kMaxN, p->info_dev + 1, u, d_packed);
    DRACO_CUDA(cudaGetLastError());
    p->project_used = (int)grid;
    return DRACO_OK;
}

}  // namespace

// The projection of all of R into the plan's partials, and u for the decode vector and flags that the plan's sample left.
int launch_cyc_onepass(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, float* u, int64_t d_packed,
                       cudaStream_t st) {
    const bool packed = d_packed > 0;
    const bool vec2 = (len % 2 == 0) && (ld % 2 == 0) && (!packed || d_packed == 2 * len);
    if (vec2) return packed ? launch_onepass<true, true>(p, R, f, len, ld, u, d_packed, st) : launch_onepass<true, false>(p, R, f, len, ld, u, d_packed, st);
    return packed ? launch_onepass<false, true>(p, R, f, len, ld, u, d_packed, st) : launch_onepass<false, false>(p, R, f, len, ld, u, d_packed, st);
}

}  // namespace draco
