// Repetition code (Section 3, "Fractional Repetition Code"): the encoder
// E^Rep_j(Y_j) = Y_j 1_P and the decoder D^Rep(R) = sum over groups of the
// element-wise majority of the group's received vectors, found with the
// streaming majority vote of Algorithm 2 on 32-bit patterns.
//
// Both kernels are single passes over an [n][len] fp32 matrix: a thread owns
// four coordinates, walks the groups, and keeps one group's replicas in registers.  HBM-bound: encode moves
// 8 n len bytes, vote 4 n len + 4 len bytes.
#include "draco_internal.cuh"

namespace draco {

namespace {

constexpr int kThreads = 256;

// Four columns of one row, as bit patterns.
struct Pack {
    uint4 v;
    __device__ __forceinline__ uint32_t get(int c) const { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }
};

// The four columns of a thread.  ADJ: neighbours, one 128-bit access (every row starts on a 16-byte boundary and holds whole
// vectors).  Otherwise blockDim.x apart, four 32-bit accesses, so that a warp's accesses are contiguous wherever a row starts;
// `in` has bit c set for the columns inside the vector, the others read the first column again.  As many bytes in flight per
// thread as with one 128-bit access; with one column per thread the vote ran at 2.6 - 3.9 TB/s on such rows (n = 45, s = 5,
// d = 5,000,011: 348 us, now 150; n = 45, s = 3: 236, now 154; s = 1: 277, now 166; encode, s = 5: 427, now 344).
template <bool ADJ>
struct Columns {
    int64_t col;
    uint32_t in;
    int o1, o2, o3;
    __device__ __forceinline__ void open(int64_t c, int64_t len) {
        col = c;
        if constexpr (ADJ) {
            in = 15u;
        } else {
            const int step = (int)blockDim.x;
            in = 1u | (c + step < len ? 2u : 0u) | (c + 2 * step < len ? 4u : 0u) | (c + 3 * step < len ? 8u : 0u);
            o1 = (in & 2u) ? step : 0;
            o2 = (in & 4u) ? 2 * step : 0;
            o3 = (in & 8u) ? 3 * step : 0;
        }
    }
    __device__ __forceinline__ bool has(int c) const { return ADJ || ((in >> c) & 1u); }
    __device__ __forceinline__ void load(Pack& p, const uint32_t* row) const {
        const uint32_t* ptr = row + col;
        if constexpr (ADJ) p.v = __ldcs(reinterpret_cast<const uint4*>(ptr));
        else p.v = make_uint4(__ldcs(ptr), __ldcs(ptr + o1), __ldcs(ptr + o2), __ldcs(ptr + o3));
    }
    __device__ __forceinline__ void store(float* row, const float (&x)[4]) const {
        float* ptr = row + col;
        if constexpr (ADJ) {
            __stcs(reinterpret_cast<float4*>(ptr), make_float4(x[0], x[1], x[2], x[3]));
        } else {
            const int off[4] = {0, o1, o2, o3};
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (has(c)) __stcs(ptr + off[c], x[c]);
        }
    }
    // w <- w - scale * x (the SGD step of Section 2 fused into the decoder's epilogue)
    __device__ __forceinline__ void update(float* row, const float (&x)[4], float scale) const {
        float* ptr = row + col;
        if constexpr (ADJ) {
            float4 w = *reinterpret_cast<const float4*>(ptr);
            w.x = fmaf(-scale, x[0], w.x); w.y = fmaf(-scale, x[1], w.y); w.z = fmaf(-scale, x[2], w.z); w.w = fmaf(-scale, x[3], w.w);
            *reinterpret_cast<float4*>(ptr) = w;
        } else {
            const int off[4] = {0, o1, o2, o3};
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (has(c)) ptr[off[c]] = fmaf(-scale, x[c], ptr[off[c]]);
        }
    }
};

// ---------------------------------------------------------------- encode
// MMAX > 0: groups of at most MMAX members, GB groups fetched together so that about 16 rows are in flight per
// thread whatever the group size (as in the vote kernel); MMAX == 0: larger groups, members streamed, eight at a time (off the
// 16-byte grid four: eight at n = 128, s = 20, d = 12,000,001 3802 us, four 3135).
// Groups do not depend on one another: where the columns alone give few blocks, gridDim.y blocks share the groups of a column
// range.  A thread that walks all of them is a chain of latencies (n = 45, s = 3, d = 100,000: 15.6 us so, 4.7 us shared; with
// rows off the grid, d = 100,003, 19.1 and 8.9; streamed groups, n = 42, s = 10, d = 100,003, 41 and 10.7).
// Rows off the 16-byte grid (ADJ false): a block reads kSector columns more than it writes and writes of each row the run that
// starts on a 32-byte sector, so that no sector is shared between blocks (a shared one may go to memory half filled).  Aligned
// rows keep a loop of their own: in the other's the loads of a batch are issued a few at a time (n = 15, s = 2, d = 30 M 617 us,
// 586 so; n = 45, s = 5 1789 and 1763).
constexpr int kSector = 8;                              // fp32 values
constexpr int kStreamBatch = 8;
template <int MMAX, bool ADJ, int GB>
__global__ void __launch_bounds__(kThreads)
rep_encode_kernel(const float* __restrict__ G, float* __restrict__ Z, int64_t len, int64_t ldg, int64_t ldz,
                  GroupTable gt) {
    // Streamed groups let the kernel after them be set up only at their end (n = 42, s = 10, d = 30,000,001: 3107 us with the
    // others' early start, 2823 so; d = 100,000: 9.1 and 7.2).
    if constexpr (MMAX > 0) pdl_begin();
    else cudaGridDependencySynchronize();
    const uint32_t* Gb = reinterpret_cast<const uint32_t*>(G);
    // this block's groups, for the columns of one thread; emit(row, sums) writes them to one row
    auto encode_columns = [&](const Columns<ADJ>& cols, auto emit) {
        if constexpr (MMAX > 0) {
            for (int g0 = (int)blockIdx.y * GB; g0 < gt.num_groups; g0 += GB * (int)gridDim.y) {
                Pack val[GB][MMAX];
#pragma unroll
                for (int b = 0; b < GB; ++b)
                    if (g0 + b < gt.num_groups) {
                        const int first = gt.first[g0 + b], m = gt.size[g0 + b];
#pragma unroll
                        for (int k = 0; k < MMAX; ++k)
                            if (k < m) cols.load(val[b][k], Gb + (int64_t)(first + k) * ldg);
                    }
#pragma unroll
                for (int b = 0; b < GB; ++b)
                    if (g0 + b < gt.num_groups) {
                        const int first = gt.first[g0 + b], m = gt.size[g0 + b];
                        float acc[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[c] = __uint_as_float(val[b][0].get(c));
#pragma unroll
                        for (int k = 1; k < MMAX; ++k)
                            if (k < m) {
#pragma unroll
                                for (int c = 0; c < 4; ++c) acc[c] = __fadd_rn(acc[c], __uint_as_float(val[b][k].get(c)));
                            }
                        for (int k = 0; k < m; ++k) emit(first + k, acc);
                    }
            }
        } else {
            for (int g = (int)blockIdx.y; g < gt.num_groups; g += (int)gridDim.y) {
                const int first = gt.first[g], m = gt.size[g];
                float acc[4];
                constexpr int kBatch = ADJ ? kStreamBatch : kStreamBatch / 2;
                for (int k0 = 0; k0 < m; k0 += kBatch) {
                    Pack x[kBatch];
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (k0 + q < m) cols.load(x[q], Gb + (int64_t)(first + k0 + q) * ldg);
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (k0 + q < m) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const float v = __uint_as_float(x[q].get(c));
                                acc[c] = k0 + q == 0 ? v : __fadd_rn(acc[c], v);
                            }
                        }
                }
                for (int k = 0; k < m; ++k) emit(first + k, acc);
            }
        }
    };
    if constexpr (ADJ) {
        const int64_t stride = (int64_t)gridDim.x * blockDim.x;
        for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < len / 4; v += stride) {
            Columns<ADJ> cols;
            cols.open(4 * v, len);
            encode_columns(cols, [&](int row, const float(&acc)[4]) { cols.store(Z + (int64_t)row * ldz, acc); });
        }
    } else {
        const int tile = 4 * (int)blockDim.x - kSector;
        const int64_t ntiles = (len + tile - 1) / tile;
        for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
            const int64_t c0 = t * tile;
            const int64_t first_col = c0 + threadIdx.x;
            if (first_col >= len) continue;
            Columns<ADJ> cols;
            cols.open(first_col, len);
            uint32_t mask = 0;                          // byte c, bit k: column c is written in rows whose run starts k columns in
            const int shift0 = (int)(-((int64_t)(reinterpret_cast<uintptr_t>(Z) >> 2) + c0)) & (kSector - 1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int i = (int)threadIdx.x + c * (int)blockDim.x;
#pragma unroll
                for (int k = 0; k < kSector; ++k)
                    if (cols.has(c) && (i >= k || t == 0) && i < k + tile) mask |= 1u << (c * kSector + k);
            }
            encode_columns(cols, [&](int row, const float(&acc)[4]) {
                const uint32_t m = mask >> ((shift0 - (int)((row * ldz) & (kSector - 1))) & (kSector - 1));
                float* z = Z + (int64_t)row * ldz + cols.col;
                if (m & 1u) __stcs(z, acc[0]);
                if (m & 0x100u) __stcs(z + cols.o1, acc[1]);
                if (m & 0x10000u) __stcs(z + cols.o2, acc[2]);
                if (m & 0x1000000u) __stcs(z + cols.o3, acc[3]);
            });
        }
    }
    if constexpr (MMAX == 0) cudaTriggerProgrammaticLaunchCompletion();
}

// ---------------------------------------------------------------- vote
struct RepScratch {
    uint32_t mask[kMaxN];             // per group: bit k set <=> member k disagreed somewhere
    unsigned long long no_majority;
    unsigned int done;                // blocks that have added their part
};

// mask words -> flag bytes and the info block, by the block that comes last, which leaves the scratch cleared for the next
// call on the plan: a memset before and a one-block kernel after the vote were two thirds of a short vote's time
// (n = 15, s = 2, d = 100,000: 11.3 - 12.8 us with them, 7.6 - 8.2 without;
// 7.15 against 7.43 us a call with one thread's fence instead of every thread's and the two exchanges under way together).
__device__ __forceinline__ void finish_vote(const GroupTable& gt, RepScratch* scratch, uint8_t* flags, uint8_t* flags2,
                                            DeviceInfo* info) {
    __shared__ int count;
    unsigned long long no_majority = 0;
    if (threadIdx.x == 0) {
        count = 0;
        no_majority = atomicExch(&scratch->no_majority, 0ull);     // under way while the masks are fetched
    }
    __syncthreads();
    for (int g = threadIdx.x; g < gt.num_groups; g += blockDim.x) {
        const int first = gt.first[g], m = gt.size[g];
        int c = 0;
        uint32_t word = 0;
        for (int k = 0; k < m; ++k) {
            if (k % 32 == 0) word = atomicExch(&scratch->mask[first + k / 32], 0u);
            const uint8_t bit = (word >> (k & 31)) & 1u;
            if (flags) flags[first + k] = bit;
            flags2[first + k] = bit;
            c += bit;
        }
        if (c) atomicAdd(&count, c);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        info->n_flagged = count;
        info->no_majority = no_majority;
        info->status = no_majority ? DRACO_ENOMAJ : DRACO_OK;
        info->locator_rank = 0;
        info->n_active = 0;
        info->scale = 0.0;
        info->max_syndrome = 0.0;
    }
}

// One step of Algorithm 2 for item x.
__device__ __forceinline__ void vote_step(uint32_t x, uint32_t& ma, int& counter) {
    const bool empty = counter == 0;
    const bool same = ma == x;
    ma = empty ? x : ma;
    counter = empty ? 1 : (same ? counter + 1 : counter - 1);
}

// Majority of one group whose m <= MMAX replicas sit in registers.  Returns the selected bit
// patterns in sel[], adds the members that disagree somewhere to `dis` and the coordinates (of those in `in`)
// without a strict majority to `nomaj`.
template <int MMAX>
__device__ __forceinline__ void vote_group(const Pack (&val)[MMAX], int m, uint32_t in, uint32_t (&sel)[4], uint32_t& dis,
                                           unsigned int& nomaj) {
    // A value held by strictly more than half of the group IS what Algorithm 2 returns.  So count first the members that equal
    // member 0 in all four columns (five logic operations each), then those that equal member 1 (member 0 may be the
    // adversary); only if neither has a strict majority is the streaming vote itself run, column by column.  Counting column by
    // column at once took about twice the instructions and left large groups bound by them (n = 45, d = 5 M: s = 7 244 us, now
    // 188; s = 5 162 us, now 141).
    // Nearly all groups agree bit for bit: up to eight members the differences from member 0 are looked at together before they are
    // counted (n = 45, s = 1, d = 20 M 617 us without, 560 so; n = 64, s = 2 873 and 788; every group with an adversary, n = 10, s = 2
    // 145 and 144).  Larger groups have no registers to keep them (n = 9, s = 4, 20 M 251 us, 282 so).
    bool settled = false;
#pragma unroll
    for (int ref = 0; ref < 2 && ref < MMAX; ++ref) {
        if (!settled && ref < m) {
            const uint4 r = val[ref].v;
            auto apart = [&](int k) {                      // non-zero where member k differs from `ref`
                const uint4 x = val[k].v;
                return (x.x ^ r.x) | (x.y ^ r.y) | (x.z ^ r.z) | (x.w ^ r.w);
            };
            uint32_t ne = 0;
            if constexpr (MMAX <= 8) {
                uint32_t diff[MMAX], any = 0;
#pragma unroll
                for (int k = 0; k < MMAX; ++k)
                    if (k != ref && k < m) {
                        diff[k] = apart(k);
                        any |= diff[k];
                    }
                if (ref == 0 && any == 0u) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) sel[c] = val[0].get(c);
                    return;
                }
#pragma unroll
                for (int k = 0; k < MMAX; ++k)
                    if (k != ref && k < m) ne |= (diff[k] != 0u ? 1u : 0u) << k;
            } else {
#pragma unroll
                for (int k = 0; k < MMAX; ++k)
                    if (k != ref && k < m) ne |= (apart(k) != 0u ? 1u : 0u) << k;
            }
            if (2 * (m - __popc(ne)) > m) {
#pragma unroll
                for (int c = 0; c < 4; ++c) sel[c] = val[ref].get(c);
                dis |= ne;
                settled = true;
            }
        }
    }
    if (!settled) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t ma = val[0].get(c);
            int counter = 0;
#pragma unroll
            for (int k = 0; k < MMAX; ++k)
                if (k < m) vote_step(val[k].get(c), ma, counter);
            uint32_t ne = 0;
#pragma unroll
            for (int k = 0; k < MMAX; ++k)
                if (k < m) ne |= (val[k].get(c) != ma ? 1u : 0u) << k;
            nomaj += (2 * (m - __popc(ne)) <= m) && ((in >> c) & 1u);
            dis |= ne;
            sel[c] = ma;
        }
    }
}

// MMAX > 0: groups of at most MMAX members, GB groups fetched together so that about 16 rows
// (128-bit or 64-bit loads) are in flight per thread whatever the group size.
// MMAX == 0: groups larger than the register budget, members streamed twice (GB ignored).
template <int MMAX, bool ADJ, int GB, int TPB>
__global__ void __launch_bounds__(TPB)
rep_vote_kernel(const uint32_t* __restrict__ R, int64_t len, int64_t ld, GroupTable gt, float* __restrict__ u,
                float* __restrict__ maj, RepScratch* scratch, float* __restrict__ w, float scale, uint8_t* flags, uint8_t* flags2,
                DeviceInfo* info) {
    pdl_begin();
    __shared__ uint32_t smask[kMaxN][MMAX > 0 ? 1 : 4];   // generic path: up to 128 members = 4 words
    for (int i = threadIdx.x; i < kMaxN * (MMAX > 0 ? 1 : 4); i += blockDim.x) (&smask[0][0])[i] = 0;
    __syncthreads();

    unsigned int nomaj = 0;
    auto vote_columns = [&](const Columns<ADJ>& cols) {
        float acc[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] = 0.0f;
        if constexpr (MMAX > 0) {
            for (int g0 = 0; g0 < gt.num_groups; g0 += GB) {
                Pack val[GB][MMAX];
#pragma unroll
                for (int b = 0; b < GB; ++b)
                    if (g0 + b < gt.num_groups) {
                        const int first = gt.first[g0 + b], m = gt.size[g0 + b];
                        const uint32_t* base = R + (int64_t)first * ld;
#pragma unroll
                        for (int k = 0; k < MMAX; ++k)
                            if (k < m) cols.load(val[b][k], base + (int64_t)k * ld);
                    }
#pragma unroll
                for (int b = 0; b < GB; ++b)
                    if (g0 + b < gt.num_groups) {
                        const int g = g0 + b, m = gt.size[g];
                        uint32_t sel[4];
                        uint32_t dis = 0;
                        vote_group<MMAX>(val[b], m, cols.in, sel, dis, nomaj);
                        if (dis & ~smask[g][0]) atomicOr(&smask[g][0], dis);
                        float selv[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            selv[c] = __uint_as_float(sel[c]);
                            acc[c] = __fadd_rn(acc[c], selv[c]);
                        }
                        if (maj != nullptr) cols.store(maj + (int64_t)g * len, selv);
                    }
            }
        } else {
            // Off the 16-byte grid eight members' loads at a time (n = 42, s = 10, d = 100,003: 29.5 us one by one, 21.0 so; n = 128,
            // s = 31, 1 M + 3: 320 and 242); aligned rows four, left to the compiler: with eight the second pass finds fewer of them
            // cached (n = 42, s = 10, 11.7 M: 561 us, 682 with batches of eight).
            constexpr int kBatch = ADJ ? 1 : kStreamBatch;
            for (int g = 0; g < gt.num_groups; ++g) {
                const int first = gt.first[g], m = gt.size[g];
                const uint32_t* base = R + (int64_t)first * ld;
                uint32_t ma[4];
                int counter[4], votes[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) { ma[c] = 0u; counter[c] = 0; votes[c] = 0; }
#pragma unroll (ADJ ? 4 : 1)
                for (int k0 = 0; k0 < m; k0 += kBatch) {
                    Pack x[kBatch];
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (k0 + q < m) cols.load(x[q], base + (int64_t)(k0 + q) * ld);
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (k0 + q < m) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) vote_step(x[q].get(c), ma[c], counter[c]);
                        }
                }
#pragma unroll (ADJ ? 4 : 1)
                for (int k0 = 0; k0 < m; k0 += kBatch) {
                    Pack x[kBatch];
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (k0 + q < m) cols.load(x[q], base + (int64_t)(k0 + q) * ld);
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (k0 + q < m) {
                            const int k = k0 + q;
                            bool any_diff = false;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const bool same = x[q].get(c) == ma[c];
                                votes[c] += same;
                                any_diff |= !same;
                            }
                            if (any_diff && !(smask[g][k >> 5] & (1u << (k & 31)))) atomicOr(&smask[g][k >> 5], 1u << (k & 31));
                        }
                }
                float selv[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    nomaj += (2 * votes[c] <= m) && cols.has(c);
                    selv[c] = __uint_as_float(ma[c]);
                    acc[c] = __fadd_rn(acc[c], selv[c]);
                }
                if (maj != nullptr) cols.store(maj + (int64_t)g * len, selv);
            }
        }
        if (u != nullptr) cols.store(u, acc);
        if (w != nullptr) cols.update(w, acc, scale);
    };
    // Aligned rows, groups of up to eight: a loop without the block's tiles, whose loads the compiler issues together (n = 15,
    // s = 1, d = 4 M 52.8 -> 45.5 us); from nine on the loop over tiles is as good or better (n = 45, s = 5, 1 M 33.3 us, 35.0 so).
    if constexpr (ADJ && MMAX > 0 && MMAX <= 8) {
        const int64_t stride = (int64_t)gridDim.x * blockDim.x;
        for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < len / 4; v += stride) {
            Columns<ADJ> cols;
            cols.open(4 * v, len);
            vote_columns(cols);
        }
    } else {
        const int64_t tile = 4 * (int64_t)blockDim.x;
        for (int64_t c0 = blockIdx.x * tile; c0 < len; c0 += gridDim.x * tile) {
            const int64_t first_col = c0 + (ADJ ? 4 : 1) * (int)threadIdx.x;
            if (first_col >= len) continue;
            Columns<ADJ> cols;
            cols.open(first_col, len);
            vote_columns(cols);
        }
    }

    // block totals -> global scratch (integer OR / add: order-independent, hence deterministic)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) nomaj += __shfl_xor_sync(0xffffffffu, nomaj, off);
    if ((threadIdx.x & 31) == 0 && nomaj) atomicAdd(&scratch->no_majority, (unsigned long long)nomaj);
    __syncthreads();
    if constexpr (MMAX > 0) {
        for (int g = threadIdx.x; g < gt.num_groups; g += blockDim.x)
            if (smask[g][0]) atomicOr(&scratch->mask[gt.first[g]], smask[g][0]);
    } else {
        // generic path keeps one word per 32 members; spread them over the members' own slots
        for (int g = threadIdx.x; g < gt.num_groups; g += blockDim.x)
            for (int w = 0; w < 4; ++w)
                if (smask[g][w]) atomicOr(&scratch->mask[gt.first[g] + w], smask[g][w]);
    }
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();                       // the block's parts come before its count: the barrier, then one thread's fence
        last = atomicInc(&scratch->done, gridDim.x - 1) == gridDim.x - 1;     // wraps to 0
    }
    __syncthreads();
    if (last) {
        __threadfence();
        finish_vote(gt, scratch, flags, flags2, info);
    }
}

// Threads per block: the kernel's limit, fewer for vectors too short to give every SM two such blocks.
int block_for(int64_t quads, int sm_count, int limit) {
    int threads = limit;
    while (threads > 64 && quads < 2 * (int64_t)sm_count * threads) threads /= 2;
    return threads;
}

int grid_for(int64_t quads, int threads, int64_t cap) {
    const int64_t want = (quads + threads - 1) / threads;
    return (int)(want < cap ? want : cap);
}

template <typename Kernel>
int resident_blocks(Kernel kernel, int threads) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1) per_sm = 1;
    return per_sm;
}

}  // namespace

int launch_rep_encode(const draco_plan* p, const float* G, float* Z, int64_t len, int64_t ldg, int64_t ldz,
                      cudaStream_t st) {
    const GroupTable& gt = p->groups;
    const bool adj = (len % 4 == 0) && (ldg % 4 == 0) && (ldz % 4 == 0);
    struct Shape {
        dim3 grid;
        int threads;
    };
    auto shape = [&](int gb) {
        const int64_t steps = (gt.num_groups + gb - 1) / gb, sms = p->sm_count;
        auto tiles = [&](int threads) {                    // column ranges of that many threads
            const int64_t tile = 4 * threads - (adj ? 0 : kSector);
            return (len + tile - 1) / tile;
        };
        // the kernel's limit, fewer where that would not give every SM two blocks (n = 15, s = 5, d = 48,827: 256 threads 7.0 us,
        // 64 3.9); the grid counts ranges and not coordinates per thread, so that no block has a second one (100,003: 7.6 and 3.9)
        int threads = kThreads;
        while (threads > 64 && tiles(threads) * steps < 2 * sms) threads /= 2;
        const int64_t cap = sms * 8 * (kThreads / threads), x = tiles(threads) < cap ? tiles(threads) : cap;
        // blocks that share the groups of a column range: as many as make sixteen blocks per SM (aligned rows) or eight.  More for
        // the others costs where the shares are unequal: n = 15, s = 2, d = 1,000,003, two shares of three groups, 21.9 -> 24.4 us.
        const int64_t room = sms * (adj ? 16 : 8) * (kThreads / threads) / x, share = room < steps ? room : steps;
        return Shape{dim3((unsigned)x, share < 1 ? 1 : (unsigned)share), threads};
    };
#define DRACO_ENC(MM, AA, GG)                                                                                     \
    do {                                                                                                          \
        const Shape sh = shape(GG);                                                                               \
        launch_dependent(rep_encode_kernel<MM, AA, GG>, sh.grid, sh.threads, 0, st, G, Z, len, ldg, ldz, gt);     \
    } while (0)
#define DRACO_ENC_BY_SIZE(AA)                                      \
    do {                                                           \
        if (gt.max_size <= 3) DRACO_ENC(3, AA, 5);                 \
        else if (gt.max_size <= 4) DRACO_ENC(4, AA, 4);            \
        else if (gt.max_size <= 5) DRACO_ENC(5, AA, 2);            \
        else if (gt.max_size <= 8) DRACO_ENC(8, AA, 1);            \
        else if (gt.max_size <= 16) DRACO_ENC(16, AA, 1);          \
        else DRACO_ENC(0, AA, 1);                                  \
    } while (0)
    if (adj) DRACO_ENC_BY_SIZE(true);
    else DRACO_ENC_BY_SIZE(false);
#undef DRACO_ENC_BY_SIZE
#undef DRACO_ENC
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

int launch_rep_vote(draco_plan* p, const float* R, int64_t len, int64_t ld, float* u, float* maj, uint8_t* flags,
                    cudaStream_t st, float* w, float scale) {
    const GroupTable& gt = p->groups;
    RepScratch* scratch = reinterpret_cast<RepScratch*>(p->mask_dev);
    const bool adj = (len % 4 == 0) && (ld % 4 == 0);
    const int64_t quads = (len + 3) / 4;
    const uint32_t* Rb = reinterpret_cast<const uint32_t*>(R);
    // no more blocks than are resident at once: a block's end (its part of the masks, the fence, the count) costs a microsecond
    // or two, which rounds of blocks one after the other pay each (eight blocks per SM and this: n = 15, s = 1, d = 1 M 20.1 and
    // 17.0 us, 4 M 57.2 and 52.8; n = 45, s = 3, 11.7 M 321 and 317; s = 5, 60.2 M 1814 and 1665)
#define DRACO_VOTE(MM, AA, GG, TT)                                                                                \
    do {                                                                                                          \
        static const int per_sm = resident_blocks(rep_vote_kernel<MM, AA, GG, TT>, TT);                           \
        const int threads = block_for(quads, p->sm_count, TT);                                                    \
        const int grid = grid_for(quads, threads, p->sm_count * per_sm * (TT / threads));                         \
        launch_dependent(rep_vote_kernel<MM, AA, GG, TT>, grid, threads, 0, st, Rb, len, ld, gt, u, maj, scratch, w, scale, flags,  \
                                                                  p->flags_dev, p->info_dev);                      \
    } while (0)
#define DRACO_VOTE_BY_SIZE(AA)                                                                                    \
    do {                                                                                                          \
        if (gt.max_size <= 3) DRACO_VOTE(3, AA, 5, 256);             /* s = 1: five groups of three, 15 rows in flight */ \
        else if (gt.max_size <= 4) DRACO_VOTE(4, AA, 4, 256);                                                     \
        else if (gt.max_size <= 5) DRACO_VOTE(5, AA, 3, 256);        /* s = 2: three groups of five */             \
        else if (gt.max_size <= 8) DRACO_VOTE(8, AA, 2, 256);                                                     \
        else if (gt.max_size <= 12) DRACO_VOTE(12, AA, 1, 128);                                                   \
        else if (gt.max_size <= 16) DRACO_VOTE(16, AA, 1, 128);      /* 16 rows of 4 words per thread: small blocks keep 3 per SM */ \
        else DRACO_VOTE(0, AA, 1, 256);                                                                           \
    } while (0)
    if (adj) DRACO_VOTE_BY_SIZE(true);
    else DRACO_VOTE_BY_SIZE(false);
#undef DRACO_VOTE_BY_SIZE
#undef DRACO_VOTE
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

size_t rep_scratch_bytes() { return sizeof(RepScratch); }

}  // namespace draco
