// Cyclic-code encoder (Section 3, "Cyclic Code"): Z = G W, z_j = G W_{.,j}.
//
// W = [Q 1_P] C_L has the closed form W[j][k] = n^(-1/2) prod_{m in alpha_j} (w^k - w^m),
// w = exp(2 pi i / n), alpha_j = {j+2s+1 .. j+n-1} mod n, so its rows are shifted copies of
// row 0 up to a unit phase: W[j][k] = w^(j M) W[0][(k - j) mod n], M = n - 2 s - 1.  Hence
//
//     z_j = phase[j] * sum_{t=0..2s} tap[t] * g_{(j - t) mod n},
//     tap[t] = w^(-t M) W[0][t],   phase[j] = w^(j M)
//
// (with a unit factor moved from the taps to the phases that makes the centre tap real):
// one fixed (2 s + 1)-tap complex filter run around the circle of gradients, then one unit
// rotation per output.  The taps do not depend on j, so they sit in the kernel's constant
// parameter bank and every multiply-add takes its coefficient from there.
//
// Data movement.  Every warp walks strips of 128 coordinates (64 complex coordinates in packed mode)
// on its own, a lane owning 4 of them, and visits the n rows of a strip once.  Each lane streams its
// 16 bytes of every row from global memory into a private column of a shared-memory ring with
// asynchronous copies (cp.async, one group per row, 12 rows in flight, running on into the next strip),
// and takes them from there into a register window of the last 2 s + 1 rows.  No thread reads what
// another thread copied, so the kernel has no barrier, no flag and no wait other than
// cp.async.wait_group.  The first 2 s rows of a strip are also kept in shared memory, because the
// circle closes on them at the end of the walk; nothing is read twice.
// HBM traffic is the algorithmic minimum: 4 n len bytes read + 8 n len bytes written.
//
// Arithmetic.  |tap| peaks in the middle of the filter (1.8e5 at n = 45, s = 5) and decoding
// cancels the sum back to O(1), so rounding in the encoder is amplified by that factor.  The
// outer taps are accumulated in fp32, smallest first; the three centre taps, the rotation
// and the final sum run in fp64, and each output is rounded to fp32 once.  That keeps the
// encoder at the accuracy floor of complex64 transport (2 n (2 s + 1) FMA per coordinate,
// of which 5 n + 4 n in fp64).
//
// Packed mode filters complex inputs: the two halves' sums are combined before the rotation (s = 0, where there is nothing
// to sum, after it: n = 15, d = 11.7 M 286 us, 238 so), which halves its cost and the conversions of the results, and up to
// s = 4 everything runs in fp64 (each fp32 partial sum costs a conversion of 8 cycles, a fp64 multiply-add 2).  Against the sums
// kept apart, both timed in turn: n = 45, d = 60.2 M: s = 5 5.79 -> 5.17 ms, s = 3 5.30 -> 4.44 ms, s = 7 6.52 -> 5.91 ms; n = 15,
// s = 2 1.45 -> 1.20 ms; error against fp64 at s <= 4 2.7e-8 -> 2.53e-8, elsewhere unchanged.  All of s = 5 in fp64 measured
// 5.79 ms, five fp64 taps 6.02 ms.  The real centre tap (one fp64 operation per coordinate less) took the unpacked encoder from
// 6.21 to 6.13 ms at s = 5 and from 7.39 to 7.27 ms at s = 7.  In a loop of launches the power cap lowers the clock: unpacked,
// s = 5, 5.6 ms at 1965 MHz, 6.3 at 1665; packed 5.0 and 5.4 at 1820.
#include <math.h>

#include "draco_internal.cuh"

namespace draco {

namespace {

constexpr int kVec = 4;                         // coordinates per thread
constexpr int kRing = 12;                       // rows in flight per thread
constexpr int kGenericThreads = 256;

// Shapes per s.  The window of the s >= 3 kernels needs 140-168 registers, which a scheduler's 16 K
// registers allow for 3 warps: 12 warps per block, one block per SM.  The s <= 2 kernels fit in 128
// registers and run 16 warps.
template <int S, bool PACKED>
struct StreamCfg {
    static constexpr int R = 2 * S + 1;                            // taps
    static constexpr int NBIG = R < 3 || (PACKED && S <= 4) ? R : 3;   // centre taps in fp64
    static constexpr int H = (NBIG - 1) / 2;
    static constexpr int SL = ((R + NBIG - 1) / NBIG) * NBIG;      // register slots: a multiple of NBIG
    static constexpr int kThreads = S <= 2 ? 512 : 384;
    static constexpr int NSTASH = S > 0 ? 2 * S : 1;
    static constexpr uint32_t kRowBytes = kThreads * 16;           // one ring / stash row: 16 bytes per thread
    static constexpr size_t kSmem = (size_t)kRowBytes * (kRing + NSTASH);
};

// ---------------------------------------------------------------- asynchronous-copy and shared-memory wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {          // at most N of this thread's groups still pending
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t a, float4 v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// ---------------------------------------------------------------- per-thread state
template <int S, bool PACKED>
struct Window {
    float4 win[StreamCfg<S, PACKED>::SL];                 // rows (vv - t), slot = vv mod SL
    double cw[StreamCfg<S, PACKED>::NBIG][4];              // fp64 copies of the rows under the centre taps
};

// One output z_j of a thread's coordinates, rotated and stored: win[(P - t) mod SL] = row (j - t) mod n, cw its fp64 copies.
template <int S, int P, bool PACKED, bool REALC>
__device__ __forceinline__ void encode_output(const Window<S, PACKED>& w, const double2 rot, float2* dst, bool act0, bool act1,
                                              const EncodeTaps& taps, const EncodeTaps64& taps64) {
    using Cfg = StreamCfg<S, PACKED>;
    constexpr int R = Cfg::R, NBIG = Cfg::NBIG, H = Cfg::H, SL = Cfg::SL;
    float ar[4] = {0.f, 0.f, 0.f, 0.f}, ai[4] = {0.f, 0.f, 0.f, 0.f};
    // taps grow towards the middle of the filter: add the outer (small) terms first so the
    // running sums stay small while most of the fp32 roundings happen
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int t = (k & 1) ? 2 * S - (k >> 1) : (k >> 1);
        if (t >= S - H && t <= S + H) continue;
        const float4 g = w.win[(P - t + 2 * SL) % SL];
        const float cr = taps.tap[t].x, ci = taps.tap[t].y;
        ar[0] = fmaf(cr, g.x, ar[0]); ai[0] = fmaf(ci, g.x, ai[0]);
        ar[1] = fmaf(cr, g.y, ar[1]); ai[1] = fmaf(ci, g.y, ai[1]);
        ar[2] = fmaf(cr, g.z, ar[2]); ai[2] = fmaf(ci, g.z, ai[2]);
        ar[3] = fmaf(cr, g.w, ar[3]); ai[3] = fmaf(ci, g.w, ai[3]);
    }
    constexpr bool kJoin = PACKED && S > 0;          // the two halves' sums are joined before the rotation
    constexpr int NOUT = kJoin ? 2 : 4;              // rotations of this thread
    double dr[NOUT], di[NOUT];
    if constexpr (kJoin) {
        // components 0, 1 of a row are the real parts of two complex coordinates, 2, 3 their imaginary parts
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            dr[c] = S > H ? (double)ar[c] - (double)ai[c + 2] : 0.0;
            di[c] = S > H ? (double)ai[c] + (double)ar[c + 2] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < NBIG; ++k) {
            const int t = (k & 1) ? S + H - (k >> 1) : S - H + (k >> 1);
            const double cr = taps64.tap[t].x, ci = taps64.tap[t].y;
            const double(&g)[4] = w.cw[((P - t + 2 * SL) % SL) % NBIG];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                dr[c] = fma(cr, g[c], dr[c]);
                di[c] = fma(cr, g[c + 2], di[c]);
                if (t != S) {                        // the centre tap is real
                    dr[c] = fma(-ci, g[c + 2], dr[c]);
                    di[c] = fma(ci, g[c], di[c]);
                }
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) { dr[c] = (double)ar[c]; di[c] = (double)ai[c]; }
#pragma unroll
        for (int t = S - H; t <= S + H; ++t) {
            const int q = ((P - t + 2 * SL) % SL) % NBIG;
            const double cr = taps64.tap[t].x, ci = taps64.tap[t].y;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                dr[c] = fma(cr, w.cw[q][c], dr[c]);
                if (!REALC || t != S) di[c] = fma(ci, w.cw[q][c], di[c]);
            }
        }
    }
    double xr[NOUT], xi[NOUT];
#pragma unroll
    for (int c = 0; c < NOUT; ++c) {
        xr[c] = fma(dr[c], rot.x, -di[c] * rot.y);
        xi[c] = fma(dr[c], rot.y, di[c] * rot.x);
    }
    if constexpr (kJoin) {
        if (act0) __stcs(reinterpret_cast<float4*>(dst), make_float4((float)xr[0], (float)xi[0], (float)xr[1], (float)xi[1]));
    } else if constexpr (PACKED) {
        // components 0, 1 filtered the real parts (X), 2, 3 the imaginary parts (Y): z = X + i Y
        if (act0)
            __stcs(reinterpret_cast<float4*>(dst), make_float4((float)(xr[0] - xi[2]), (float)(xi[0] + xr[2]),
                                                               (float)(xr[1] - xi[3]), (float)(xi[1] + xr[3])));
    } else {
        // A lane's two 16-byte stores are 512 bytes apart, so that each store instruction of the warp
        // covers 512 contiguous bytes (whole 32-byte sectors).  With the 4 coordinates of a lane adjacent,
        // every instruction wrote half of 32 sectors and the kernel stopped at 4.9 TB/s.
        if (act0) __stcs(reinterpret_cast<float4*>(dst), make_float4((float)xr[0], (float)xi[0], (float)xr[1], (float)xi[1]));
        if (act1) __stcs(reinterpret_cast<float4*>(dst + 64), make_float4((float)xr[2], (float)xi[2], (float)xr[3], (float)xi[3]));
    }
}

// The fetch side: the rows of this warp's strips, one after the other, kRing rows ahead of the row being
// consumed.  A lane copies coordinates 2l, 2l+1 and 64+2l, 64+2l+1 of the strip (packed: complex
// coordinates 2l, 2l+1, real parts from G[r][c], imaginary parts from G[r][half + c]).
template <bool PACKED>
struct Fetcher {
    const float* G;
    const float* ga;            // this lane's first pair in the next row to fetch
    int64_t boff;               // from there to its second pair: 64, or `half` when PACKED
    int64_t boff_now;           // the same, 0 while the second pair is switched off
    int64_t strip, nstrips, strip_step, len, ldg;
    int row, n, lane;
    bool act0, act1;            // the pairs lie inside the vector (and the strip exists)
    __device__ __forceinline__ void open_strip() {
        constexpr int kStrip = PACKED ? 64 : 128;
        const int64_t c = strip * kStrip + 2 * lane;
        act0 = strip < nstrips && c < len;
        act1 = PACKED ? act0 : (strip < nstrips && c + 64 < len);
        // switched-off copies still carry an address: keep it inside the matrix (this lane's first pair of strip 0, and
        // the first pair again for a second pair beyond the row's end)
        ga = G + (act0 ? c : (int64_t)(2 * lane < len ? 2 * lane : 0));
        boff_now = act1 ? boff : 0;
        row = 0;
    }
    // copy this lane's 16 bytes of the next row to shared address dst and close the group (copies of a lane
    // outside the vector are switched off; every thread counts the same groups)
    __device__ __forceinline__ void fetch(uint32_t dst) {
        cp_async8_if(dst, ga, act0);
        cp_async8_if(dst + 8, ga + boff_now, act1);
        cp_async_commit();
        ga += ldg;
        if (++row == n) {
            strip += strip_step;
            open_strip();
        }
    }
};

struct Cursor {
    uint32_t ring0, rd;         // this thread's column of the ring, and the byte offset of the next row to consume
    float2* zout;               // next output row (modes 0 and 1)
};

// One step of the walk: bring row vv of the strip into window slot P (from the ring, or from the stash once
// the circle has closed), emit z_{vv mod n} when the window is full, and refill the ring slot.
// REALC: the centre tap's imaginary part, which is zero, is left out.
// MODE 0: first SL steps of a strip (all rows from the ring; outputs from step 2 S on);
// MODE 1: steady state (ring row + output);  MODE 2: anything (run-time guards).
template <int S, int P, int MODE, bool PACKED, bool REALC>
__device__ __forceinline__ void encode_step(Window<S, PACKED>& w, Cursor& cur, Fetcher<PACKED>& f, int vv, int n, int64_t ldz,
                                            uint32_t stash0, float2* zcol, bool act0, bool act1,
                                            const EncodeTaps& taps, const EncodeTaps64& taps64,
                                            const EncodePhase64& ph64) {
    using Cfg = StreamCfg<S, PACKED>;
    constexpr int NBIG = Cfg::NBIG, H = Cfg::H, SL = Cfg::SL;
    constexpr uint32_t kRowBytes = Cfg::kRowBytes;
    const int total = n + 2 * S;
    if (MODE == 2 && vv >= total) return;
    const bool from_ring = (MODE != 2) || (vv < n);
    float4 x;
    if (from_ring) {
        cp_async_wait<kRing - 1>();          // kRing groups were committed after the one that carries this row
        x = lds128(cur.ring0 + cur.rd);
        if ((MODE == 0 && P < 2 * S) || (MODE == 2 && vv < 2 * S)) sts128(stash0 + (uint32_t)vv * kRowBytes, x);
    } else {
        x = lds128(stash0 + (uint32_t)(vv - n) * kRowBytes);
    }
    w.win[P] = x;
    if (MODE != 2 || vv >= S - H) {          // the row now under tap S-H enters the fp64 window
        constexpr int Q = (P - (S - H) + 2 * SL) % SL;
        w.cw[Q % NBIG][0] = (double)w.win[Q].x;
        w.cw[Q % NBIG][1] = (double)w.win[Q].y;
        w.cw[Q % NBIG][2] = (double)w.win[Q].z;
        w.cw[Q % NBIG][3] = (double)w.win[Q].w;
    }
    const bool emit = (MODE == 1) || (MODE == 0 && P >= 2 * S) || (MODE == 2 && vv >= 2 * S);
    if (emit) {
        // win[(P - t) mod SL] = row (vv - t) mod n: this output is z_j, j = vv mod n
        const int j = (MODE == 2 && vv >= n) ? vv - n : vv;
        float2* dst;
        if (MODE == 2) {
            dst = zcol + (int64_t)j * ldz;
        } else {
            dst = cur.zout;
            cur.zout += ldz;
        }
        encode_output<S, P, PACKED, REALC>(w, ph64.phase[j], dst, act0, act1, taps, taps64);
    }
    if (from_ring) {
        // The slot just consumed is refilled with the row kRing ahead.  Its read has completed by then: the stash
        // store or the global stores above need the value read and come before the copy in program order (a lane
        // without stores issues no copy either).
        f.fetch(cur.ring0 + cur.rd);
        cur.rd += kRowBytes;
        if (cur.rd == kRing * kRowBytes) cur.rd = 0;
    }
}

template <int S, int MODE, bool PACKED, bool REALC, int P = 0>
__device__ __forceinline__ void encode_chunk(Window<S, PACKED>& w, Cursor& cur, Fetcher<PACKED>& f, int v0, int n, int64_t ldz,
                                             uint32_t stash0, float2* zcol, bool act0, bool act1,
                                             const EncodeTaps& taps, const EncodeTaps64& taps64,
                                             const EncodePhase64& ph64) {
    if constexpr (P < StreamCfg<S, PACKED>::SL) {
        encode_step<S, P, MODE, PACKED, REALC>(w, cur, f, v0 + P, n, ldz, stash0, zcol, act0, act1, taps, taps64, ph64);
        encode_chunk<S, MODE, PACKED, REALC, P + 1>(w, cur, f, v0, n, ldz, stash0, zcol, act0, act1, taps, taps64, ph64);
    }
}

// PACKED: the real -> complex packing of Section 3's last paragraph.  `len` then counts complex
// coordinates, a strip holds 64 of them, and a lane receives two pairs of each row:
// G[r][c], G[r][c + 1] (real parts) and G[r][half + c], G[r][half + c + 1] (imaginary parts).
template <int S, bool PACKED, bool REALC>
__global__ void __launch_bounds__(StreamCfg<S, PACKED>::kThreads, 1)
cyc_encode_stream_kernel(const float* __restrict__ G, float2* __restrict__ Z, int64_t len, int64_t ldg, int64_t ldz,
                         int64_t half, int n,
                         const __grid_constant__ EncodeTaps taps, const __grid_constant__ EncodeTaps64 taps64,
                         const __grid_constant__ EncodePhase64 ph64) {
    pdl_begin();
    using Cfg = StreamCfg<S, PACKED>;
    constexpr int SL = Cfg::SL, kWarps = Cfg::kThreads / 32;
    constexpr int kStrip = PACKED ? 64 : 128;
    extern __shared__ __align__(16) unsigned char smem_raw[];        // ring[kRing][kThreads], stash[2 S][kThreads], 16 bytes each
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nstrips = (len + kStrip - 1) / kStrip;
    const int64_t strip0 = (int64_t)blockIdx.x * kWarps + warp, strip_step = (int64_t)gridDim.x * kWarps;
    Cursor cur;
    cur.ring0 = smem_u32(smem_raw) + threadIdx.x * 16;
    cur.rd = 0;
    const uint32_t stash0 = cur.ring0 + kRing * Cfg::kRowBytes;
    Fetcher<PACKED> f;
    f.G = G; f.boff = PACKED ? half : 64; f.nstrips = nstrips; f.len = len; f.ldg = ldg; f.n = n; f.lane = lane;
    f.strip = strip0; f.strip_step = strip_step;
    f.open_strip();
#pragma unroll 1
    for (int q = 0; q < kRing; ++q) f.fetch(cur.ring0 + q * Cfg::kRowBytes);
    Window<S, PACKED> w;
#pragma unroll
    for (int q = 0; q < SL; ++q) w.win[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int total = n + 2 * S;
    for (int64_t strip = strip0; strip < nstrips; strip += strip_step) {
        const int64_t c = strip * kStrip + 2 * lane;
        const bool act0 = c < len;
        const bool act1 = PACKED ? act0 : (c + 64 < len);
        float2* zcol = Z + c;
        cur.zout = zcol + (int64_t)(2 * S) * ldz;
        int v0 = 0;
        if (n >= SL && S > 0) {
            encode_chunk<S, 0, PACKED, REALC>(w, cur, f, 0, n, ldz, stash0, zcol, act0, act1, taps, taps64, ph64);
            for (v0 = SL; v0 + SL <= n; v0 += SL)
                encode_chunk<S, 1, PACKED, REALC>(w, cur, f, v0, n, ldz, stash0, zcol, act0, act1, taps, taps64, ph64);
        }
        for (; v0 < total; v0 += SL)
            encode_chunk<S, 2, PACKED, REALC>(w, cur, f, v0, n, ldz, stash0, zcol, act0, act1, taps, taps64, ph64);
    }
    cp_async_wait<0>();
}

// The same for short vectors, where a warp's walk over all rows is a chain of latencies: a warp computes J outputs of its strip and
// loads their 2 s + J rows at once; the others' rows are re-read through L2.  The same operations on every entry, hence the same bits.
constexpr int kShortWarps = 4;
template <int S, bool PACKED, bool REALC, int J>
__global__ void __launch_bounds__(32 * kShortWarps)
cyc_encode_short_kernel(const float* __restrict__ G, float2* __restrict__ Z, int64_t len, int64_t ldg, int64_t ldz, int64_t half,
                        int n, const __grid_constant__ EncodeTaps taps, const __grid_constant__ EncodeTaps64 taps64,
                        const __grid_constant__ EncodePhase64 ph64) {
    pdl_begin();
    using Cfg = StreamCfg<S, PACKED>;
    constexpr int NBIG = Cfg::NBIG, H = Cfg::H, SL = Cfg::SL, kStrip = PACKED ? 64 : 128;
    const int64_t c = ((int64_t)blockIdx.x * kShortWarps + (threadIdx.x >> 5)) * kStrip + 2 * (threadIdx.x & 31);
    const bool act0 = c < len, act1 = PACKED ? act0 : c + 64 < len;
    if (!act0) return;
    const int j0 = (int)blockIdx.y * J;
    const float* g = G + c;
    const int64_t second = PACKED ? half : act1 ? 64 : 0;
    float4 x[2 * S + J];
#pragma unroll
    for (int q = 0; q < 2 * S + J; ++q) {
        int r = j0 + q - 2 * S;
        r = r < 0 ? r + n : r < n ? r : n - 1;             // rows past the last output's are not used
        const float2 a = *reinterpret_cast<const float2*>(g + (int64_t)r * ldg), b = *reinterpret_cast<const float2*>(g + (int64_t)r * ldg + second);
        x[q] = make_float4(a.x, a.y, b.x, b.y);
    }
#pragma unroll
    for (int k = 0; k < J; ++k) {
        if (j0 + k < n) {
            constexpr int P = 2 * S;
            Window<S, PACKED> w;
#pragma unroll
            for (int q = 0; q < SL; ++q) w.win[q] = x[k + (q < 2 * S ? q : 2 * S)];
#pragma unroll
            for (int q = S - H; q <= S + H; ++q) {
                w.cw[q % NBIG][0] = (double)x[k + q].x;
                w.cw[q % NBIG][1] = (double)x[k + q].y;
                w.cw[q % NBIG][2] = (double)x[k + q].z;
                w.cw[q % NBIG][3] = (double)x[k + q].w;
            }
            encode_output<S, P, PACKED, REALC>(w, ph64.phase[j0 + k], Z + (int64_t)(j0 + k) * ldz + c, act0, act1, taps, taps64);
        }
    }
}

// Rows of any alignment and length, 1 <= s <= 7: the same walk with two coordinates kThreads apart (packed: one complex
// coordinate) per thread, so that a warp's 4-byte loads and 8-byte stores are contiguous wherever a row starts, and everything
// in fp64.  A thread keeps the last 2 s + 1 rows as fp64 in a register window and fetches each row 2 s + 1 steps ahead, into
// the register that the step just freed; the first 2 s rows stay in shared memory for the end of the walk.
//
// Row j of Z starts anywhere relative to a 32-byte sector.  A block computes kAlign coordinates more than it writes and writes
// of each row the run that starts on a sector, so that no sector is shared between blocks: shared ones left L2 half written
// (n = 45, s = 1, d = 60.2 M + 1: 12.1 ms with plain strips, 8.3 ms so).  Two coordinates per thread instead of one take the
// instructions per output from 61 to about 46 (s = 5: 8.3 -> 7.5 ms; s = 1: 8.3 -> 6.9 ms), and a barrier per 2 s + 1 rows
// keeps a block's warps on neighbouring addresses (s = 5: 7.8 -> 7.5 ms).  What is left is latency: 16 to 24 warps per SM, fp64
// pipe half busy.  Against the one-coordinate-per-thread kernel below, which re-reads every row 2 s + 1 times through the
// caches: n = 45, s = 3, d = 3,000,017: 1130 -> 347 us (4.7 TB/s).
template <int S, bool PACKED>
struct FirCfg {
    static constexpr int R = 2 * S + 1;
    static constexpr int C = PACKED ? 1 : 2;                       // output coordinates per thread, kThreads apart
    static constexpr int NI = 2;                                   // real inputs per thread and row
    static constexpr int kThreads = 128;
    static constexpr int kAlign = 4;                               // complex entries per 32-byte sector
    static constexpr int kTile = kThreads * C - kAlign;            // coordinates that a block writes of every row
    static constexpr int kBlocks = S <= 2 ? 6 : S <= 5 ? 4 : 3;    // per SM, what the registers allow
};

template <int S, bool PACKED>
struct FirState {
    float raw[FirCfg<S, PACKED>::R][FirCfg<S, PACKED>::NI];        // rows on their way
    double win[FirCfg<S, PACKED>::R][FirCfg<S, PACKED>::NI];       // rows vv .. vv - 2 S, slot = vv mod R
    const float* gp;                                               // next row to fetch
    float2* zp;                                                    // next output row
    int64_t off1;                                                  // from the first to the second input
    int shift, dshift;                                             // entries of the next output row before its first sector
    uint32_t mask[FirCfg<S, PACKED>::C];                           // bit k: this coordinate is written when shift = k
    bool on1;
};

template <int S, bool PACKED>
__device__ __forceinline__ void fir_fetch(FirState<S, PACKED>& w, int p, int64_t ldg) {
    w.raw[p][0] = __ldcs(w.gp);
    w.raw[p][1] = w.on1 ? __ldcs(w.gp + w.off1) : 0.0f;
    w.gp += ldg;
}

// The filter's sums for one output of a thread's coordinates: win[(P - t) mod R] = row (j - t) mod n of output j.
template <int S, int P, bool PACKED>
__device__ __forceinline__ void fir_sums(const double (&win)[FirCfg<S, PACKED>::R][FirCfg<S, PACKED>::NI], const EncodeTaps64& taps,
                                         double (&ar)[FirCfg<S, PACKED>::C], double (&ai)[FirCfg<S, PACKED>::C]) {
    using Cfg = FirCfg<S, PACKED>;
    constexpr int R = Cfg::R, NI = Cfg::NI, C = Cfg::C;
#pragma unroll
    for (int c = 0; c < C; ++c) ar[c] = ai[c] = 0.0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int t = (k & 1) ? 2 * S - (k >> 1) : (k >> 1);       // small taps first
        const double cr = taps.tap[t].x, ci = taps.tap[t].y;
        const double(&x)[NI] = win[(P - t + 2 * R) % R];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            ar[c] = fma(cr, x[c], ar[c]);
            if (t != S) ai[c] = fma(ci, x[c], ai[c]);              // the centre tap is real
        }
        if constexpr (PACKED) {
            if (t != S) ar[0] = fma(-ci, x[1], ar[0]);
            ai[0] = fma(cr, x[1], ai[0]);
        }
    }
}
// Rotated and rounded, where the output is stored: formed for every thread, whether it stores or not, the packed walk at n = 45, s = 5, d =
// 2,000,003 took 242 us, 218 so.
__device__ __forceinline__ float2 fir_rotated(double ar, double ai, const double2 rot) {
    return make_float2((float)fma(ar, rot.x, -ai * rot.y), (float)fma(ar, rot.y, ai * rot.x));
}

// Step vv of the walk, slot P = vv mod R.  HEAD: the first R steps; TAIL: run-time guards.
template <int S, int P, bool PACKED, bool HEAD, bool TAIL>
__device__ __forceinline__ void fir_step(FirState<S, PACKED>& w, int vv, int n, int64_t ldg, int64_t ldz, float* stash,
                                         const EncodeTaps64& taps, const EncodePhase64& ph) {
    using Cfg = FirCfg<S, PACKED>;
    constexpr int R = Cfg::R, NI = Cfg::NI, C = Cfg::C, kT = Cfg::kThreads;
    if (TAIL && vv >= n + 2 * S) return;
    if (TAIL && vv >= n) {
#pragma unroll
        for (int c = 0; c < NI; ++c) w.win[P][c] = (double)stash[((vv - n) * NI + c) * kT];
    } else {
#pragma unroll
        for (int c = 0; c < NI; ++c) {
            w.win[P][c] = (double)w.raw[P][c];
            if (HEAD && P < 2 * S) stash[(P * NI + c) * kT] = w.raw[P][c];
        }
        if (vv + R < n) fir_fetch<S, PACKED>(w, P, ldg);
    }
    if (HEAD && P < 2 * S) return;
    double ar[C], ai[C];
    fir_sums<S, P, PACKED>(w.win, taps, ar, ai);
    const double2 rot = ph.phase[TAIL && vv >= n ? vv - n : vv];
#pragma unroll
    for (int c = 0; c < C; ++c)
        if ((w.mask[c] >> w.shift) & 1u) __stcs(w.zp + c * kT, fir_rotated(ar[c], ai[c], rot));
    w.zp += ldz;
    w.shift = (w.shift - w.dshift) & (Cfg::kAlign - 1);
    if (TAIL && vv == n - 1) {
        w.zp -= (int64_t)n * ldz;
        w.shift = (w.shift + n * w.dshift) & (Cfg::kAlign - 1);
    }
}

template <int S, bool PACKED, bool HEAD, bool TAIL, int P = 0>
__device__ __forceinline__ void fir_chunk(FirState<S, PACKED>& w, int v0, int n, int64_t ldg, int64_t ldz, float* stash,
                                          const EncodeTaps64& taps, const EncodePhase64& ph) {
    if constexpr (P < FirCfg<S, PACKED>::R) {
        fir_step<S, P, PACKED, HEAD, TAIL>(w, v0 + P, n, ldg, ldz, stash, taps, ph);
        fir_chunk<S, PACKED, HEAD, TAIL, P + 1>(w, v0, n, ldg, ldz, stash, taps, ph);
    }
}

template <int S, bool PACKED>
__global__ void __launch_bounds__(FirCfg<S, PACKED>::kThreads, FirCfg<S, PACKED>::kBlocks)
cyc_encode_fir_kernel(const float* __restrict__ G, float2* __restrict__ Z, int64_t len, int64_t ldg, int64_t ldz,
                      int64_t half, int64_t d_real, int n, const __grid_constant__ EncodeTaps64 taps,
                      const __grid_constant__ EncodePhase64 ph) {
    pdl_begin();
    using Cfg = FirCfg<S, PACKED>;
    constexpr int R = Cfg::R, C = Cfg::C, kT = Cfg::kThreads, kTile = Cfg::kTile, kAlign = Cfg::kAlign;
    __shared__ float stash_all[2 * S * Cfg::NI * kT];
    float* stash = stash_all + threadIdx.x;                        // this thread's column
    const int64_t nstrips = (len + kTile - 1) / kTile;
    for (int64_t strip = blockIdx.x; strip < nstrips; strip += gridDim.x) {
        FirState<S, PACKED> w;
        const int64_t c0 = strip * kTile, c = c0 + threadIdx.x;
        w.gp = G + (c < len ? c : c0);                             // threads beyond the vector read their strip's first entry
        w.off1 = PACKED ? half : kT;
        w.on1 = PACKED ? (c < len && half + c < d_real) : (c + kT < len);
        w.zp = Z + c + (int64_t)(2 * S) * ldz;
        w.dshift = (int)(ldz & (kAlign - 1));
        w.shift = (int)(-((int64_t)(reinterpret_cast<uintptr_t>(Z) >> 3) + c0 + (int64_t)(2 * S) * ldz)) & (kAlign - 1);
#pragma unroll
        for (int q = 0; q < C; ++q) {
            const int i = threadIdx.x + q * kT;
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < kAlign; ++k)
                if ((i >= k || strip == 0) && i < k + kTile && c0 + i < len) m |= 1u << k;
            w.mask[q] = m;
        }
#pragma unroll
        for (int p = 0; p < R; ++p) fir_fetch<S, PACKED>(w, p, ldg);       // n >= R
        fir_chunk<S, PACKED, true, false>(w, 0, n, ldg, ldz, stash, taps, ph);
        if (n == R) {                                              // the head ended at row n - 1: the next output is row 0
            w.zp -= (int64_t)n * ldz;
            w.shift = (w.shift + n * w.dshift) & (kAlign - 1);
        }
        int v0 = R;
        for (; v0 + R < n; v0 += R) {
            __syncthreads();
            fir_chunk<S, PACKED, false, false>(w, v0, n, ldg, ldz, stash, taps, ph);
        }
        for (; v0 < n + 2 * S; v0 += R) {
            __syncthreads();
            fir_chunk<S, PACKED, false, true>(w, v0, n, ldg, ldz, stash, taps, ph);
        }
    }
}

// The same for short vectors: a thread computes J outputs of its coordinates from rows that it loads at once (the same bits).
template <int S, bool PACKED, int J>
__global__ void __launch_bounds__(FirCfg<S, PACKED>::kThreads)
cyc_encode_fir_short_kernel(const float* __restrict__ G, float2* __restrict__ Z, int64_t len, int64_t ldg, int64_t ldz, int64_t half,
                            int64_t d_real, int n, const __grid_constant__ EncodeTaps64 taps, const __grid_constant__ EncodePhase64 ph) {
    pdl_begin();
    using Cfg = FirCfg<S, PACKED>;
    constexpr int C = Cfg::C, NI = Cfg::NI, kT = Cfg::kThreads;
    const int64_t c = (int64_t)blockIdx.x * (kT * C) + threadIdx.x;
    if (c >= len) return;
    const bool on1 = PACKED ? half + c < d_real : c + kT < len;
    const int64_t off1 = !on1 ? 0 : PACKED ? half : kT;
    const int j0 = (int)blockIdx.y * J;
    float x[2 * S + J][NI];
#pragma unroll
    for (int q = 0; q < 2 * S + J; ++q) {
        int r = j0 + q - 2 * S;
        r = r < 0 ? r + n : r < n ? r : n - 1;             // rows past the last output's are not used
        x[q][0] = G[(int64_t)r * ldg + c];
        x[q][1] = G[(int64_t)r * ldg + c + off1];
        if (!on1) x[q][1] = 0.0f;
    }
#pragma unroll
    for (int k = 0; k < J; ++k) {
        if (j0 + k < n) {
            double win[Cfg::R][NI];
#pragma unroll
            for (int q = 0; q < Cfg::R; ++q) {
                win[q][0] = (double)x[k + q][0];
                win[q][1] = (double)x[k + q][1];
            }
            double ar[C], ai[C];
            fir_sums<S, 2 * S, PACKED>(win, taps, ar, ai);
            const double2 rot = ph.phase[j0 + k];
#pragma unroll
            for (int q = 0; q < C; ++q)
                if (q == 0 || on1) Z[(int64_t)(j0 + k) * ldz + c + q * kT] = fir_rotated(ar[q], ai[q], rot);
        }
    }
}

// s = 0 off the streaming kernel's alignment, s > 7: one coordinate per thread, rows re-read through the caches,
// fp64 taps and fp64 accumulation throughout (a tap rounded to fp32 is a fixed error of 2^-24 |tap| that
// the decoder's cancellation amplifies like any other).  half > 0: packed mode (len complex coordinates; the imaginary
// parts come from G[r][half + i], zero beyond d_real).
__global__ void __launch_bounds__(kGenericThreads)
cyc_encode_generic_kernel(const float* __restrict__ G, float2* __restrict__ Z, int64_t len, int64_t ldg, int64_t ldz,
                          int64_t half, int64_t d_real, int n, int s, const double2* __restrict__ taps,
                          const __grid_constant__ EncodePhase64 ph) {
    pdl_begin();
    const int64_t stride = (int64_t)gridDim.x * kGenericThreads;
    for (int64_t i = (int64_t)blockIdx.x * kGenericThreads + threadIdx.x; i < len; i += stride) {
        const bool has_b = half > 0 && half + i < d_real;
        for (int j = 0; j < n; ++j) {
            double ar = 0.0, ai = 0.0, br = 0.0, bi = 0.0;
            for (int t = 0; t <= 2 * s; ++t) {
                int r = j - t;
                if (r < 0) r += n;
                const double2 c = taps[t];
                const double g = (double)G[(int64_t)r * ldg + i];
                ar = fma(c.x, g, ar);
                ai = fma(c.y, g, ai);
                if (has_b) {
                    const double gb = (double)G[(int64_t)r * ldg + half + i];
                    br = fma(c.x, gb, br);
                    bi = fma(c.y, gb, bi);
                }
            }
            const double2 rot = ph.phase[j];
            const double xr = fma(ar, rot.x, -ai * rot.y), xi = fma(ar, rot.y, ai * rot.x);
            const double yr = fma(br, rot.x, -bi * rot.y), yi = fma(br, rot.y, bi * rot.x);
            Z[(int64_t)j * ldz + i] = make_float2((float)(xr - yi), (float)(xi + yr));
        }
    }
}

// Outputs per thread of the short kernels, 0: the walking kernels.  warps: what one output row takes.  The short kernels' time grows
// with the warps of outputs per SM and with s, whatever n is; a walk takes its n + 2 s steps, however short the vector.  One output each
// while that gives an SM no more than 110 - 10 s warps, then four, which read and convert a third to half as often, but few at a time.
// Walking / one / four outputs, us of GPU time in a captured chain: n = 45, s = 5, 34 warps 22 / 3.5 / 3.6, 68 22 / 5.5 / 5.9, 120 22 / 8.6 / 6.7,
// 203 22 / 13 / 10; n = 5, s = 1, 68 4.5 / 3.8 / 5.0, 300 10.1 / 12.3 / 9.6; n = 9, s = 3, 68 6.0 / 4.7 / 6.2, 160 9.8 / 8.5 / 7.5.  (s = 0: four from 16 warps on,
// n = 9, 50 6.2 / 2.7 / 3.3, 203 9.2 / 8.5 / 5.8.)  Up to 600 warps (n = 45, s = 5: as many strips as the walk has under way at once), but the walk where
//   * it has only one row, and nothing is read twice (n = 1, 160 7.5 / 6.8 / 6.8, 300 10.5 / 12.3 / 12.2);
//   * packed vectors with s = 3, 4 (all fp64: every output repeats its rows' conversions) have few rows (n = 9, s = 3, 300 12.7 / 14.6 / 13.1,
//     581 22.9 / 27 / 24.5, n = 17, s = 4, 405 18.2 / 24 / 21; but n = 45, s = 3, 581 33 / 28 / 24);
//   * all its strips are under way at once (12 an SM) and the outputs are many beside its steps (s >= 3, from 9 (n + 2 s) on).
int short_outputs(const draco_plan* p, int64_t warps, bool packed) {
    const int64_t sms = p->sm_count, n = p->n, s = p->s, all = warps * n;
    const auto each_up_to = [&](int64_t most) { return all <= most * sms; };
    if (each_up_to(16)) return 1;
    if (!each_up_to(600)) return 0;
    if (n == 1) return each_up_to(180) ? 1 : 0;
    if (s == 0) return 4;
    if (each_up_to(110 - 10 * s)) return 1;
    if (packed && (s == 3 || s == 4) && n <= 20 && !each_up_to(300)) return 0;
    if (s >= 3 && warps <= 12 * sms && !each_up_to(9 * (n + 2 * s))) return 0;
    return 4;
}
// The same off the 16-byte grid, up to 300 warps of outputs per SM.  blocks, resident: the walk's blocks, and how many an SM holds.  Up to 60
// warps (s = 1: 100) the short kernels are ahead, one output each from s = 4 on (n = 45, s = 5, 51 warps 7.7 / 4.0 / 4.9; s = 1 7.0 / 2.4 / 2.7).
// Beyond, four outputs are compared with the walk by the time that either was measured to take, in us: n = 9, s = 4, 90 warps 4.3 / 5.3 / 5.8, 291
// 8.0 / 14 / 10.2; n = 21, s = 5, 160 8.4 / 9.7 / 7.1, 291 9.2 / 16 / 11.5; n = 45, s = 5, 291 13.9 / 16 / 11.3.
int short_outputs_fir(const draco_plan* p, int64_t warps, int64_t blocks, int resident, bool packed) {
    const double sms = p->sm_count, s = p->s, each = (double)(warps * p->n) / sms;
    if (each <= 16.0) return 1;
    if (each > 300.0) return 0;
    if (each <= 60.0) return p->s >= 4 ? 1 : 4;
    if (p->s == 1 && each <= 100.0) return 4;
    const double rounds = fmax(1.0, (double)blocks / (sms * resident));
    const double walk = rounds * fmax(packed ? 4.7 : 3.5, 0.3 + (p->s <= 2 ? 0.33 : 0.25) * (p->n + 2 * p->s));
    const double four = packed ? fmax(4.2 + 0.4 * s, each * (0.011 + 0.0034 * s)) : fmax(3.7 + 0.55 * s, each * (0.0167 + 0.0045 * s));
    return walk < four ? 0 : 4;
}

template <int S, bool PACKED, bool REALC = true>
int launch_stream(const draco_plan* p, const float* G, float2* Z, int64_t len, int64_t ldg, int64_t ldz, int64_t half,
                  cudaStream_t st) {
    using Cfg = StreamCfg<S, PACKED>;
    constexpr int kThreads = Cfg::kThreads;
    constexpr int kStrip = PACKED ? 64 : 128;
    const int64_t nstrips = (len + kStrip - 1) / kStrip;
    const int outputs = short_outputs(p, nstrips, PACKED);
    if (outputs > 0) {
#define DRACO_SHORT(J) launch_dependent(cyc_encode_short_kernel<S, PACKED, REALC, J>, dim3((unsigned)((nstrips + kShortWarps - 1) / kShortWarps), (unsigned)((p->n + J - 1) / J)), \
                                        32 * kShortWarps, 0, st, G, Z, len, ldg, ldz, half, p->n, p->taps, p->taps64, p->phase64)
        if (outputs == 1) DRACO_SHORT(1); else DRACO_SHORT(4);
#undef DRACO_SHORT
        DRACO_CUDA(cudaGetLastError());
        return DRACO_OK;
    }
    auto kern = cyc_encode_stream_kernel<S, PACKED, REALC>;
    static bool configured[64] = {};
    int dev = p->device;
    if (dev < 0 || dev >= 64) dev = 0;
    if (!configured[dev]) {
        DRACO_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem));
        configured[dev] = true;
    }
    int per_sm = 1;
    DRACO_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, Cfg::kSmem));
    if (per_sm < 1) per_sm = 1;
    const int64_t nblocks = (nstrips + kThreads / 32 - 1) / (kThreads / 32);
    int64_t grid = (int64_t)p->sm_count * per_sm;
    if (grid > nblocks) grid = nblocks;
    if (grid < 1) grid = 1;
    launch_dependent(kern, (int)grid, kThreads, Cfg::kSmem, st, G, Z, len, ldg, ldz, half, p->n, p->taps, p->taps64, p->phase64);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

template <bool PACKED>
int launch_stream_any(const draco_plan* p, const float* G, float2* Z, int64_t len, int64_t ldg, int64_t ldz, int64_t half,
                      cudaStream_t st) {
    switch (p->s) {
        case 0: return launch_stream<0, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        case 1: return launch_stream<1, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        case 2: return launch_stream<2, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        case 3: return launch_stream<3, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        case 4: return launch_stream<4, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        case 5: return launch_stream<5, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        case 6: return launch_stream<6, PACKED>(p, G, Z, len, ldg, ldz, half, st);
        default:
            // a walk of fewer than 2 R rows is all head and tail, whose code is the slower one without the zero term (n = 15,
            // s = 7, d = 1 M 52.3 us, 49.2 with it, 30 M 1196 and 1172; n = 29 2298 and 2247; but n = 30 2358 and 2365, n = 45
            // 7195 and 7313 at 60.2 M)
            if (!PACKED && p->n < 2 * StreamCfg<7, PACKED>::R) return launch_stream<7, PACKED, PACKED>(p, G, Z, len, ldg, ldz, half, st);
            return launch_stream<7, PACKED>(p, G, Z, len, ldg, ldz, half, st);
    }
}

template <int S, bool PACKED>
int launch_fir(const draco_plan* p, const float* G, float2* Z, int64_t len, int64_t ldg, int64_t ldz, int64_t half,
               int64_t d_real, cudaStream_t st) {
    using Cfg = FirCfg<S, PACKED>;
    constexpr int kPer = Cfg::kThreads * Cfg::C;
    const int64_t nshort = (len + kPer - 1) / kPer;
    const int64_t nstrips = (len + Cfg::kTile - 1) / Cfg::kTile;
    const int outputs = short_outputs_fir(p, nshort * (Cfg::kThreads / 32), nstrips, Cfg::kBlocks, PACKED);
    if (outputs > 0) {
#define DRACO_SHORT(J) launch_dependent(cyc_encode_fir_short_kernel<S, PACKED, J>, dim3((unsigned)nshort, (unsigned)((p->n + J - 1) / J)), Cfg::kThreads, 0, st, G, Z, len, ldg, ldz, \
                                        half, d_real, p->n, p->taps64, p->phase64)
        if (outputs == 1) DRACO_SHORT(1); else DRACO_SHORT(4);
#undef DRACO_SHORT
        DRACO_CUDA(cudaGetLastError());
        return DRACO_OK;
    }
    int64_t grid = (int64_t)p->sm_count * Cfg::kBlocks;
    if (grid > nstrips) grid = nstrips;
    launch_dependent(cyc_encode_fir_kernel<S, PACKED>, (int)grid, Cfg::kThreads, 0, st, G, Z, len, ldg, ldz, half, d_real,
                     p->n, p->taps64, p->phase64);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

template <bool PACKED>
int launch_fir_any(const draco_plan* p, const float* G, float2* Z, int64_t len, int64_t ldg, int64_t ldz, int64_t half,
                   int64_t d_real, cudaStream_t st) {
    switch (p->s) {
        case 1: return launch_fir<1, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
        case 2: return launch_fir<2, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
        case 3: return launch_fir<3, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
        case 4: return launch_fir<4, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
        case 5: return launch_fir<5, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
        case 6: return launch_fir<6, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
        default: return launch_fir<7, PACKED>(p, G, Z, len, ldg, ldz, half, d_real, st);
    }
}

}  // namespace

// half == 0: Z[j][i], i < len, from G[.][i].  half > 0 (packed): Z[j][i], i < len complex coordinates,
// from G[.][i] (real parts) and G[.][half + i] (imaginary parts, zero for half + i >= d_real).
int launch_cyc_encode(const draco_plan* p, const float* G, float2* Z, int64_t len, int64_t ldg, int64_t ldz,
                      int64_t half, int64_t d_real, cudaStream_t st) {
    // the streaming kernel copies 8 bytes and stores 16 bytes at a time: row starts, strip starts and the half offset
    // are multiples of 4 floats
    const bool packed = half > 0;
    bool fast = (ldg % 4 == 0) && (ldz % 2 == 0) && p->s <= 7;
    // (and, for a column chunk of a longer vector, what the whole vector's call would need: all of it goes the same way)
    if (packed) fast = fast && (len % 4 == 0) && (half % 4 == 0) && (half + len <= d_real) && (ldz % 4 == 0) && (p->d % 2 == 0);
    else fast = fast && (len % 4 == 0) && (ldz % 4 == 0);
    if (fast) return packed ? launch_stream_any<true>(p, G, Z, len, ldg, ldz, half, st)
                            : launch_stream_any<false>(p, G, Z, len, ldg, ldz, 0, st);
    if (p->s >= 1 && p->s <= 7)                            // the register window's sizes
        return packed ? launch_fir_any<true>(p, G, Z, len, ldg, ldz, half, d_real, st)
                      : launch_fir_any<false>(p, G, Z, len, ldg, ldz, 0, d_real, st);
    int64_t want = (len + kGenericThreads - 1) / kGenericThreads;
    const int64_t cap = (int64_t)p->sm_count * 16;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    // Launched in the ordinary way, after everything before it: set up early, repeated encodes of a matrix that stays in L2 take
    // up to twice as long (n = 20, s = 8, d = 65,539 60 us so, 90 early; packed 200,003 57 and 95; no difference elsewhere).
    cyc_encode_generic_kernel<<<(int)want, kGenericThreads, 0, st>>>(G, Z, len, ldg, ldz, half, d_real, p->n, p->s,
                                                                    p->taps_full_dev, p->phase64);
    DRACO_CUDA(cudaGetLastError());
    return DRACO_OK;
}

}  // namespace draco
