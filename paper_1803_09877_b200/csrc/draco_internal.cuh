// Internal declarations shared by the translation units of libdraco.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "draco.h"

namespace draco {

constexpr int kMaxN = DRACO_MAX_N;
constexpr int kMaxTaps = 15;          // 2 s + 1 for the register-window encoder (s <= 7)
constexpr int kProjectTile = 2048;    // coordinates per tile of the projection kernel
constexpr int kProjectTileShort = 512;   // the same for short vectors
constexpr int kProjectWarps = 8;
constexpr double kMarginBar = 10.0;        // locator_margin below this, or ..
constexpr double kImResidualBar = 1e-2;    // .. im_residual above this fraction of re_max: status DRACO_EUNSURE
constexpr int kJacobiSweepLimit = 60;

struct GroupTable {                   // repetition code: consecutive groups
    int num_groups;
    int max_size;
    uint8_t first[kMaxN];
    uint8_t size[kMaxN];
};

struct EncodeTaps {                   // cyclic encoder: z_j = phase[j] * sum_t tap[t] * g_{(j-t) mod n}
    float2 tap[kMaxTaps];
};

struct EncodeTaps64 {                 // the same taps / phases in fp64 (centre taps and the final rotation)
    double2 tap[kMaxTaps];
};

struct EncodePhase64 {
    double2 phase[kMaxN];
};

// Device-resident state of the cyclic decoder (lives in the plan's scratch).
struct CycDevice {
    double2 twiddle[kMaxN];           // w^k, w = exp(2 pi i / n)
    double2 b[kMaxN];                 // decode vector (zero on flagged nodes)
    double2 b_active[kMaxN];          // b_j of the active rows, packed
    int32_t active[kMaxN];            // their node indices
    double2 work[kMaxN * (kMaxN + 1)];  // elimination work space
    double record[3 * kMaxN];         // the plan's own projection record: n (re, im) pairs, then n values q_j
};

struct DeviceInfo {                   // mirrors draco_info
    int32_t status;
    int32_t n_flagged;
    int32_t locator_rank;
    int32_t n_active;
    unsigned long long no_majority;
    double scale;
    double max_syndrome;
    int32_t internal_error;
    int32_t svd_sweeps;
    double locator_margin;
    unsigned long long im_residual_bits;   // bit patterns of non-negative doubles: they order like integers, so the
    unsigned long long re_max_bits;        // blocks of the recovery kernel merge their maxima with atomicMax
    int32_t combine;                  // not in draco_info, set after a sample: n_active, or -1: u has been written already
};

}  // namespace draco

struct draco_plan {
    int n, s, code;
    int64_t d;
    int device;
    int sm_count;
    double theta;
    // repetition
    draco::GroupTable groups;
    // cyclic (host copies)
    double* W_host;                   // [n][n][2]
    draco::EncodeTaps taps;
    draco::EncodeTaps64 taps64;
    draco::EncodePhase64 phase64;
    double2* taps_full_dev;           // generic encoder: fp64 taps for any s, device [2s+1]
    // device scratch
    draco::CycDevice* cyc_dev;
    draco::DeviceInfo* info_dev;      // [2]: the plan's, and that of the locator's run on a sample
    double2* partial_dev;             // [project_grid][n]
    int project_grid;                 // capacity of partial_dev in blocks
    int project_used;                 // blocks whose partials the plan's last projection (all its chunks) filled
    int reads;                        // of R by the last draco_locate_decode: 0 none yet, 2, or 1: one, if `combine` is negative
    uint8_t* flags_dev;               // [2 kMaxN] internal flags, and those of the sample
    uint32_t* mask_dev;               // repetition: the vote's scratch, zero between calls
    // host-buffer pipeline (allocated on its first call)
    float* stage_dev;                 // two [n][stage_chunk] slices of G (double buffer)
    cudaStream_t copy_stream, work_stream;
    cudaEvent_t ev_copied[2], ev_consumed[2];
    int64_t stage_chunk;
    float* f_dev;                     // [d]
    float* u_dev;                     // [d]
};

namespace draco {

// Set the thread's last CUDA error text; returns DRACO_ECUDA.
int cuda_fail(cudaError_t err, const char* what);

#define DRACO_CUDA(call)                                              \
    do {                                                              \
        cudaError_t err__ = (call);                                   \
        if (err__ != cudaSuccess) return draco::cuda_fail(err__, #call); \
    } while (0)

// Launch whose blocks may be set up while the kernel before it in the stream is still running (programmatic dependent launch).
// Every kernel launched so begins with pdl_begin(): it lets the kernel after it be set up in turn (one of them does so at its
// end), and waits until everything before it in the stream is complete and visible, before it touches global memory that another
// kernel writes.  Saves the launch gap, 1 - 2 us a kernel: n = 45, s = 5, d = 4096, locate and decode (three kernels) 37.8 -> 31.8
// us; n = 15, s = 2, d = 1 M 68.7 -> 63.5 us; a repetition encode of 100,000 coordinates costs the caller 3.8 instead of 4.4 us.
template <typename... Params, typename... Args>
void launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);    // an error is left for cudaGetLastError, as by <<< >>>
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_begin() {
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
}
// |a| for the decoder's self-check maxima; NaN, which a node may send and fmax would drop, counts as infinity
__device__ __forceinline__ double magnitude(double a) { return a == a ? fabs(a) : __longlong_as_double(0x7ff0000000000000ll); }
// 8 bytes to shared memory, asynchronously, with the source switched off by a predicate (ignore-src: zeros are written, src is not
// read), so that a lane outside the vector needs no branch around its copies.
__device__ __forceinline__ void cp_async8_if(uint32_t dst, const void* src, bool on) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %2, 0;\n\tcp.async.ca.shared.global [%0], [%1], 8, p;\n\t}" ::"r"(dst), "l"(src), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ float4 lds128(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
#endif

// kernels / launchers (one per translation unit)
int launch_rep_encode(const draco_plan* p, const float* G, float* Z, int64_t len, int64_t ldg, int64_t ldz,
                      cudaStream_t st);
int launch_rep_vote(draco_plan* p, const float* R, int64_t len, int64_t ld, float* u, float* maj, uint8_t* flags,
                    cudaStream_t st, float* w = nullptr, float scale = 0.0f);
int launch_cyc_encode(const draco_plan* p, const float* G, float2* Z, int64_t len, int64_t ldg, int64_t ldz,
                      int64_t half, int64_t d_real, cudaStream_t st);
int launch_cyc_project(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, bool accumulate,
                       cudaStream_t st);
int launch_cyc_project_finish(draco_plan* p, double2* e_out, cudaStream_t st);
int launch_cyc_sample(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, cudaStream_t st);
int launch_cyc_onepass(draco_plan* p, const float2* R, const float* f, int64_t len, int64_t ld, float* u, int64_t d_packed,
                       cudaStream_t st);
// with_b: the decode vector too; sampled: the flags are compared with those that launch_cyc_sample found
int launch_cyc_solve(draco_plan* p, const double2* e, uint8_t* flags, bool with_b, cudaStream_t st, bool sampled = false);
int launch_cyc_decode_vector(draco_plan* p, const uint8_t* flags, cudaStream_t st);
// once: after launch_cyc_onepass, whose sum stands where the sample's V was the right one
int launch_cyc_recover(draco_plan* p, const float2* R, int64_t len, int64_t ld, float* u, int64_t d_packed,
                       cudaStream_t st, float* w = nullptr, float scale = 0.0f, bool once = false);
int launch_generate(float* out, int rows, int64_t len, int64_t ld, int64_t i0, int row0, float mean, float std,
                    uint64_t seed, cudaStream_t st);
int launch_corrupt(float* R, int64_t row_pitch, int64_t nvals, int64_t v0, const int* node, const int* model,
                   const float* param, int n_adv, uint64_t seed, bool is_complex, int sm_count, cudaStream_t st);
int project_grid_size(int sm_count);

}  // namespace draco
