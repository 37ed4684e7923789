// Shared device-side declarations of the MONA step library (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mona {

// A chunk is the unit that goes through prologue -> Newton-Schulz -> update together: up to MAXC
// same-shape matrices whose bf16 iterates fit the chunk budget (sized for full machine occupancy, not for cache).
constexpr int MAXC = 512;   // per-matrix pointers travel as kernel arguments (at most 10 KiB of the 32 KiB CUDA 12 allows)
// The Frobenius norm is the sum, in a fixed order, of at most MAX_UNITS partial sums of squares per matrix.  A unit's length follows
// from the matrix size alone, so the norm's bits do not depend on how many matrices share a launch.
constexpr int MAX_UNITS = 256;
inline long long norm_unit(long long e) {
    const long long least = (e + MAX_UNITS - 1) / MAX_UNITS;
    return (least + 1023) / 1024 * 1024;                 // a multiple of the prologue's loop trip
}

// Slab decomposition of `count` matrices of e elements that go through one elementwise launch.  A slab is one block's work: a
// multiple of `unit` elements (the prologue: norm units; otherwise one trip of the loop), 16 K of them at most where a unit is not
// longer (longer slabs leave fewer blocks than the device holds at once), as short as it takes to give every SM its eleven
// blocks - with 16 K always, a 256 x 512 matrix ran on 8 blocks and its prologue took 10.6 us, 128 blocks take 4.1 - and long
// enough for at most MAX_UNITS per matrix.
inline void slab_plan(long long e, long long count, long long unit, long long* slab_len, int* slabs) {
    const long long resident = 148 * 11, longest = 16384;
    long long slab = (e * count + resident - 1) / resident;
    slab = slab < longest ? slab : longest;
    if ((e + slab - 1) / slab > MAX_UNITS) slab = (e + MAX_UNITS - 1) / MAX_UNITS;
    const bool shorter = slab <= longest;
    slab = (slab + unit - 1) / unit * unit;
    if (shorter && slab > longest && slab > unit) slab -= unit;
    *slab_len = slab;
    *slabs = (int)((e + slab - 1) / slab);
}

// Per-chunk pointers, filled on the host; the elementwise kernels take the parts they need in tables of their own size.
struct ChunkPtrs {
    const void* g[MAXC];   // gradient of matrix c (fp32 or bf16)
    float* w[MAXC];        // parameter of matrix c
    float* o[MAXC];        // optional fp32 copy of O_k (may be null)
    int gid[MAXC];         // global matrix index (descriptor order), for error reports
};

// Device status word, latched by kernels and read by mona_poll_status().
struct DeviceStatus {
    unsigned int flags;        // bit 0: non-finite norm, bit 1: a bounded wait ran out
    int first_bad;             // lowest global matrix index that reported (or INT_MAX)
    unsigned int timeout_site; // which wait gave up (diagnostic)
    unsigned int pad;
};
constexpr unsigned STATUS_NONFINITE = 1u;
constexpr unsigned STATUS_TIMEOUT = 2u;
constexpr unsigned STATUS_BOUNDS = 4u;       // debug build only: an index check failed (site in timeout_site)

// Index checks of the debug build (-DMONA_DEBUG).  compute-sanitizer is not available everywhere this library is
// developed, so the kernels can check their own indices: a failed check latches STATUS_BOUNDS with a site number in the
// status word - it never traps - and the guarded access is skipped.  In the normal build the macro is `true`.
#ifdef MONA_DEBUG
#define MONA_IN_BOUNDS(cond, status, site) \
    ((cond) ? true : (atomicOr(&(status)->flags, ::mona::STATUS_BOUNDS), (status)->timeout_site = (site), false))
#else
#define MONA_IN_BOUNDS(cond, status, site) true
#endif

// Programmatic dependent launch: a kernel launched with `early` may be set up, and its blocks placed, while the kernel before it in
// the stream still runs.  It calls wait_for_stream() before it touches global memory; a kernel that others follow early calls
// let_next_start() when its own work is all placed.  Without the attribute both are free.  Where a chain of launches is the time
// this takes the launch gaps out (one 256 x 512 matrix 83.4 -> 79.5 us per step, a mixed small set 108.3 -> 104.0, a dense block of 1024 and
// 2816 370 -> 362, fp32: one 501 x 303 269 -> 239, one 1001 x 1500 945 -> 922).
__device__ __forceinline__ void wait_for_stream() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... Q>
cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, bool early, Q&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// A scalar hyper-parameter carried as an unevaluated sum of two floats, hi + lo, so that products with
// it are accurate to ~2^-45 instead of 2^-24: rounding beta_a = 0.99 to one float would by itself
// cost 3e-8 per step in the EMA, which accumulates over its ~1/(1-beta_a) step memory.
struct F2 {
    float hi, lo;
};

struct PrologueScalars {
    F2 beta;            // beta_a
    F2 one_minus_beta;  // 1 - beta_a, formed in double
    F2 alpha;           // alpha
    F2 mu;              // mu
    float eps;          // norm_eps
};

}  // namespace mona
