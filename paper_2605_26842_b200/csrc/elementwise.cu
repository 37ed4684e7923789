// Elementwise passes of the MONA step: the fused prologue (Algorithm 1 lines 4-7 and 10 plus the
// Frobenius norm that Eq. newton_schulz starts from) and the parameter update (line 9).
// Both are single HBM passes over contiguous slabs with 128-bit accesses.
#include "elementwise.cuh"

#include <math.h>

namespace mona {

namespace {

// 128-thread blocks of ~46 registers: small enough to run on an SM beside a resident CTA of the Newton-Schulz kernel
// (which leaves 7168 registers free), so the elementwise passes of one chunk overlap the GEMMs of another.
constexpr int EW_THREADS = 128;

__device__ __forceinline__ float mul_add2(F2 k, float x, float addend) {
    // (k.hi + k.lo) * x + addend with a single rounding on the dominant term
    return fmaf(k.hi, x, fmaf(k.lo, x, addend));
}

template <typename GT>
struct GradLoad;
template <>
struct GradLoad<float> {
    static __device__ __forceinline__ float4 load4(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
    static __device__ __forceinline__ float load1(const float* p) { return __ldcs(p); }
};
template <>
struct GradLoad<__nv_bfloat16> {
    static __device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
        uint2 raw = __ldcs(reinterpret_cast<const uint2*>(p));
        float4 r;
        r.x = __uint_as_float(raw.x << 16);
        r.y = __uint_as_float(raw.x & 0xffff0000u);
        r.z = __uint_as_float(raw.y << 16);
        r.w = __uint_as_float(raw.y & 0xffff0000u);
        return r;
    }
    static __device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
};

// Storage format of the two auxiliary buffers A_k and G_{k-1}: fp32, or bfloat16 (MONA-Lite: the value is
// rounded once, to nearest even, when it is stored, and the stored value is what the step goes on with).
template <typename ST>
struct StateIO;
template <>
struct StateIO<float> {
    using elem = float;
    static constexpr bool has_gp = true;
    static __device__ __forceinline__ float4 load4(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
    static __device__ __forceinline__ void store4(float* p, float4 v) { __stcs(reinterpret_cast<float4*>(p), v); }
    static __device__ __forceinline__ float load1(const float* p) { return *p; }
    static __device__ __forceinline__ void store1(float* p, float v) { *p = v; }
    static __device__ __forceinline__ float round(float v) { return v; }
};
template <>
struct StateIO<__nv_bfloat16> {
    using elem = __nv_bfloat16;
    static constexpr bool has_gp = true;
    static __device__ __forceinline__ float4 load4(const __nv_bfloat16* p) { return GradLoad<__nv_bfloat16>::load4(p); }
    static __device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {     // v holds already-rounded values
        __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        __stcs(reinterpret_cast<uint2*>(p), make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi)));
    }
    static __device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store1(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
    static __device__ __forceinline__ float round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
};

// Tag for the single-buffer ("streaming") form of the acceleration state.  A_k and G_{k-1} enter step k+1 only
// through Z_k = beta_a A_k - (1 - beta_a) G_k:  A_{k+1} = beta_a A_k + (1 - beta_a)(G_{k+1} - G_k) = Z_k + (1 - beta_a) G_{k+1}.
// So one fp32 buffer Z replaces the two of Algorithm 1 (Z_0 = 0), and the pass moves 22 bytes per element, not 30.
// The buffer travels through the kernel in the `A` slot; the `G_prev` slot is unused.
struct Combined {};
template <>
struct StateIO<Combined> : StateIO<float> {
    static constexpr bool has_gp = false;
};

// Tag for the plain Muon step (Eq. muon_momentum): there is no acceleration state to read or write.
struct NoAux {};
template <>
struct StateIO<NoAux> {
    using elem = float;
    static constexpr bool has_gp = false;
    static __device__ __forceinline__ float4 load4(const float*) { return make_float4(0.f, 0.f, 0.f, 0.f); }
    static __device__ __forceinline__ void store4(float*, float4) {}
    static __device__ __forceinline__ float load1(const float*) { return 0.f; }
    static __device__ __forceinline__ void store1(float*, float) {}
    static __device__ __forceinline__ float round(float v) { return v; }
};
// The G_{k-1} slot only exists in the two-buffer formats.
template <typename ST>
__device__ __forceinline__ float4 gp_load4(const typename StateIO<ST>::elem* p) {
    if constexpr (StateIO<ST>::has_gp) return StateIO<ST>::load4(p); else return make_float4(0.f, 0.f, 0.f, 0.f);
}
template <typename ST>
__device__ __forceinline__ void gp_store4(typename StateIO<ST>::elem* p, float4 v) {
    if constexpr (StateIO<ST>::has_gp) StateIO<ST>::store4(p, v);
}
template <typename ST>
__device__ __forceinline__ float gp_load1(const typename StateIO<ST>::elem* p) {
    if constexpr (StateIO<ST>::has_gp) return StateIO<ST>::load1(p); else return 0.f;
}
template <typename ST>
__device__ __forceinline__ void gp_store1(typename StateIO<ST>::elem* p, float v) {
    if constexpr (StateIO<ST>::has_gp) StateIO<ST>::store1(p, v);
}

template <typename ST>
__device__ __forceinline__ void mona_elem(float g, float& gp, float& a, float& m, const PrologueScalars& k) {

    float d = g - gp;                                              // D_k = G_k - G_{k-1}
    a = StateIO<ST>::round(mul_add2(k.beta, a, fmaf(k.one_minus_beta.hi, d, k.one_minus_beta.lo * d)));  // A_k as stored
    float gt = mul_add2(k.alpha, a, g);                             // G~_k = G_k + alpha A_k
    m = mul_add2(k.mu, m, gt);                                      // M_k = mu M_{k-1} + G~_k
    gp = StateIO<ST>::round(g);                                     // G_{k-1} <- G_k
}
template <>
__device__ __forceinline__ void mona_elem<Combined>(float g, float&, float& z, float& m, const PrologueScalars& k) {
    const float w = fmaf(k.one_minus_beta.hi, g, k.one_minus_beta.lo * g);   // (1 - beta_a) G_k
    const float a = z + w;                                          // A_k = Z_{k-1} + (1 - beta_a) G_k
    float gt = mul_add2(k.alpha, a, g);                             // G~_k = G_k + alpha A_k
    m = mul_add2(k.mu, m, gt);                                      // M_k = mu M_{k-1} + G~_k
    // Z_k = beta_a A_k - (1 - beta_a) G_k = beta_a Z_{k-1} - (1 - beta_a)^2 G_k; the second form does not cancel
    z = mul_add2(k.beta, z, -fmaf(k.one_minus_beta.hi, w, k.one_minus_beta.lo * w));
}
template <>
__device__ __forceinline__ void mona_elem<NoAux>(float g, float&, float&, float& m, const PrologueScalars& k) {
    m = mul_add2(k.mu, m, g);                                       // Eq. muon_momentum: M_k = mu M_{k-1} + G_k
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Pointers of up to CAP matrices as the kernels take them.  The driver copies a launch's arguments on the host, and a table
// sized for the largest chunk (14 KiB with all pointers of 512 matrices) cost about 10 us per launch (19 -> 10 us of host time
// for one call that launches the prologue), more than the kernel of a small set runs: chunks of up to SMALL_TABLE matrices
// travel in a small table, larger ones in a full one.
constexpr int SMALL_TABLE = 32;
template <int CAP>
struct GradTable {
    const void* g[CAP];
    float* w[CAP];
    int gid[CAP];
};
template <int CAP>
struct ParamTable {
    float* w[CAP];
    float* o[CAP];
};

// grid = (slabs, C).  Block (p, c) owns elements [p*slab_len, min(e, (p+1)*slab_len)) of matrix c: one or more units of the norm,
// each with a partial sum of its own (thread sums in the order of the trips, added over the warp and then over the block's
// warps).  The last block of a matrix to finish adds the partials in index order, so ||M||_F depends neither on scheduling nor
// on the length of the slabs; it then resets the arrival counter for the next call.
// A unit's sum is added over the warp while the next unit's loads are under way, so that short units cost the pass nothing (512 matrices of
// 256 x 768, units of one trip: 503 us with one sum per 16 K slab, 505 so; 93 of 768 x 2048 736 -> 720).
template <typename GT, typename ST, int VEC, int CAP>
__global__ void __launch_bounds__(EW_THREADS, 9)      // 56 registers at most: what is free beside a Newton-Schulz CTA
prologue_kernel(const __grid_constant__ GradTable<CAP> ptrs, float* __restrict__ Mst, void* __restrict__ Ast, void* __restrict__ Gpst,
                __nv_bfloat16* __restrict__ xhat, float* __restrict__ partials, unsigned int* __restrict__ counters,
                float* __restrict__ inv_norm, DeviceStatus* __restrict__ status, long long e, long long slab_len,
                int unit_len, int slab_units, int units, PrologueScalars k, unsigned int* __restrict__ zero, int zero_words,
                float** __restrict__ params) {
    let_next_start();
    if (params && blockIdx.x == 0 && threadIdx.x == 0) params[blockIdx.y] = ptrs.w[blockIdx.y];
    for (unsigned i = (blockIdx.y * gridDim.x + blockIdx.x) * EW_THREADS + threadIdx.x; i < (unsigned)zero_words; i += gridDim.x * gridDim.y * EW_THREADS) zero[i] = 0u;
    constexpr int WARPS = EW_THREADS / 32, MAX_SLAB_UNITS = 16;      // (a slab of several units is at most 16 K elements long)
    __shared__ float red[MAX_SLAB_UNITS * WARPS];
    __shared__ int is_last;
    const int c = blockIdx.y, p = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long lo = (long long)p * slab_len;
    const long long hi = (lo + slab_len < e) ? lo + slab_len : e;
    if (!MONA_IN_BOUNDS(c < MAXC && lo < e && slab_len == slab_units * (long long)unit_len && slab_units <= MAX_SLAB_UNITS && units <= MAX_UNITS && e <= units * (long long)unit_len && (VEC == 1 || (lo % 4 == 0 && e % 4 == 0)), status, 201)) return;
    const long long at = (long long)c * e + lo;             // the block's elements of the state; below, positions are within the slab
    const int n = (int)(hi - lo);
    const GT* __restrict__ g = reinterpret_cast<const GT*>(ptrs.g[c]) + lo;
    float* __restrict__ M = Mst + at;
    using AuxT = typename StateIO<ST>::elem;
    AuxT* __restrict__ A = reinterpret_cast<AuxT*>(Ast) + at;      // never dereferenced by formats without it
    AuxT* __restrict__ Gp = reinterpret_cast<AuxT*>(Gpst) + at;
    __nv_bfloat16* __restrict__ X = xhat ? xhat + at : nullptr;

    float acc = 0.f, full = 0.f;          // sums of the present unit, and of one that is complete
    int units_done = 0;
    int unit_end = unit_len;
    auto unit_boundary = [&](int trip) -> bool {            // (the same for all threads)
        if (trip != unit_end) return false;
        full = acc; acc = 0.f; unit_end += unit_len;
        return true;
    };
    auto keep_sum = [&](float v) {
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[units_done * WARPS + warp] = v;
        ++units_done;
    };
    if (VEC == 4) {
        constexpr int STEP = EW_THREADS * 4;
        static_assert(2 * STEP == PROLOGUE_UNIT, "a unit is a whole number of trips");
        for (int trip = 0; trip < n; trip += 2 * STEP) {
            const int i = trip + (int)threadIdx.x * 4;
            const bool boundary = unit_boundary(trip);
            if (trip + 2 * STEP <= n) {
                // two independent vectors per trip keep ~128 B per thread in flight
                float4 g0 = GradLoad<GT>::load4(g + i), g1 = GradLoad<GT>::load4(g + i + STEP);
                float4 p0 = gp_load4<ST>(Gp + i), p1 = gp_load4<ST>(Gp + i + STEP);
                float4 a0 = StateIO<ST>::load4(A + i), a1 = StateIO<ST>::load4(A + i + STEP);
                float4 m0 = __ldcs(reinterpret_cast<const float4*>(M + i)), m1 = __ldcs(reinterpret_cast<const float4*>(M + i + STEP));
                if (boundary) keep_sum(full);
                mona_elem<ST>(g0.x, p0.x, a0.x, m0.x, k); mona_elem<ST>(g0.y, p0.y, a0.y, m0.y, k);
                mona_elem<ST>(g0.z, p0.z, a0.z, m0.z, k); mona_elem<ST>(g0.w, p0.w, a0.w, m0.w, k);
                mona_elem<ST>(g1.x, p1.x, a1.x, m1.x, k); mona_elem<ST>(g1.y, p1.y, a1.y, m1.y, k);
                mona_elem<ST>(g1.z, p1.z, a1.z, m1.z, k); mona_elem<ST>(g1.w, p1.w, a1.w, m1.w, k);
                gp_store4<ST>(Gp + i, p0); gp_store4<ST>(Gp + i + STEP, p1);
                StateIO<ST>::store4(A + i, a0);  StateIO<ST>::store4(A + i + STEP, a1);
                __stcs(reinterpret_cast<float4*>(M + i), m0);  __stcs(reinterpret_cast<float4*>(M + i + STEP), m1);
                if (X) {
                    *reinterpret_cast<uint2*>(X + i) = make_uint2(pack_bf16x2(m0.x, m0.y), pack_bf16x2(m0.z, m0.w));
                    *reinterpret_cast<uint2*>(X + i + STEP) = make_uint2(pack_bf16x2(m1.x, m1.y), pack_bf16x2(m1.z, m1.w));
                }
                acc = fmaf(m0.x, m0.x, acc); acc = fmaf(m0.y, m0.y, acc); acc = fmaf(m0.z, m0.z, acc); acc = fmaf(m0.w, m0.w, acc);
                acc = fmaf(m1.x, m1.x, acc); acc = fmaf(m1.y, m1.y, acc); acc = fmaf(m1.z, m1.z, acc); acc = fmaf(m1.w, m1.w, acc);
            } else {                       // the last trip of a matrix
                if (boundary) keep_sum(full);
                for (int j = i; j < n; j += STEP) {
                    float4 g0 = GradLoad<GT>::load4(g + j);
                    float4 p0 = gp_load4<ST>(Gp + j);
                    float4 a0 = StateIO<ST>::load4(A + j);
                    float4 m0 = __ldcs(reinterpret_cast<const float4*>(M + j));
                    mona_elem<ST>(g0.x, p0.x, a0.x, m0.x, k); mona_elem<ST>(g0.y, p0.y, a0.y, m0.y, k);
                    mona_elem<ST>(g0.z, p0.z, a0.z, m0.z, k); mona_elem<ST>(g0.w, p0.w, a0.w, m0.w, k);
                    gp_store4<ST>(Gp + j, p0);
                    StateIO<ST>::store4(A + j, a0);
                    __stcs(reinterpret_cast<float4*>(M + j), m0);
                    if (X) *reinterpret_cast<uint2*>(X + j) = make_uint2(pack_bf16x2(m0.x, m0.y), pack_bf16x2(m0.z, m0.w));
                    acc = fmaf(m0.x, m0.x, acc); acc = fmaf(m0.y, m0.y, acc); acc = fmaf(m0.z, m0.z, acc); acc = fmaf(m0.w, m0.w, acc);
                }
            }
        }
    } else {
        // single elements (an odd matrix size leaves the matrices of a stack unaligned): eight per thread and trip, all loads
        // first, or the pass is one dependent round trip after the other (five odd matrices, 1023 x 511 the largest bucket:
        // the whole step 3.15 -> 2.91 ms with this, the update's unrolling and the shorter slabs)
        constexpr int UNROLL = PROLOGUE_UNIT / EW_THREADS;
        for (int trip = 0; trip < n; trip += PROLOGUE_UNIT) {
            const int i = trip + (int)threadIdx.x;
            const bool boundary = unit_boundary(trip);
            float gv[UNROLL], pv[UNROLL], av[UNROLL], mv[UNROLL];
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const int j = i + u * EW_THREADS;
                gv[u] = pv[u] = av[u] = mv[u] = 0.f;
                if (j < n) { gv[u] = GradLoad<GT>::load1(g + j); pv[u] = gp_load1<ST>(Gp + j); av[u] = StateIO<ST>::load1(A + j); mv[u] = M[j]; }
            }
            if (boundary) keep_sum(full);
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const int j = i + u * EW_THREADS;
                if (j < n) {
                    mona_elem<ST>(gv[u], pv[u], av[u], mv[u], k);
                    gp_store1<ST>(Gp + j, pv[u]); StateIO<ST>::store1(A + j, av[u]); M[j] = mv[u];
                    if (X) X[j] = __float2bfloat16_rn(mv[u]);
                    acc = fmaf(mv[u], mv[u], acc);
                }
            }
        }
    }
    keep_sum(acc);

    __syncthreads();
    if (warp == 0) {
        if (lane < units_done) {
            float total = red[lane * WARPS];
            #pragma unroll
            for (int w = 1; w < WARPS; ++w) total += red[lane * WARPS + w];
            __stcg(partials + (long long)c * MAX_UNITS + p * slab_units + lane, total);
        }
        __syncwarp();
        if (lane == 0) {
            __threadfence();               // the block's partials, all written by this warp, precede its arrival
            unsigned int prev = atomicAdd(counters + c, 1u);
            is_last = (prev == gridDim.x - 1);
        }
    }
    __syncthreads();
    if (is_last && threadIdx.x < 32) {
        __threadfence();
        double s = 0.0;
        float part[MAX_UNITS / 32];        // all loads first: one round trip (in a loop they were eight, 2 us of a small launch)
        #pragma unroll
        for (int q = 0; q < MAX_UNITS / 32; ++q) part[q] = lane + 32 * q < units ? __ldcg(partials + (long long)c * MAX_UNITS + lane + 32 * q) : 0.f;
        #pragma unroll
        for (int q = 0; q < MAX_UNITS / 32; ++q) s += (double)part[q];
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) {
            float nrm = (float)sqrt(s);
            inv_norm[c] = 1.0f / (nrm + k.eps);        // X_0 = M / (||M||_F + eps)
            if (!isfinite(nrm)) {
                atomicOr(&status->flags, STATUS_NONFINITE);
                atomicMin(&status->first_bad, ptrs.gid[c]);
            }
            counters[c] = 0u;
        }
    }
}

__global__ void __launch_bounds__(EW_THREADS) param_table_kernel(const __grid_constant__ ParamTable<MAXC> ptrs, float** __restrict__ params, int C) {
    for (int c = threadIdx.x; c < C; c += EW_THREADS) params[c] = ptrs.w[c];
}

// W <- W - eta (gamma O + lambda W), evaluated as (W - (eta lambda) W) - (eta gamma) O.
template <typename OT, int VEC, int CAP>
__global__ void __launch_bounds__(EW_THREADS)
update_kernel(const __grid_constant__ ParamTable<CAP> ptrs, const OT* __restrict__ O, long long e, long long slab_len, float eta_lambda,
              float eta_gamma) {
    wait_for_stream();
    const int c = blockIdx.y, p = blockIdx.x;
    const long long lo = (long long)p * slab_len;
    const long long hi = (lo + slab_len < e) ? lo + slab_len : e;
    float* __restrict__ W = ptrs.w[c];
    float* __restrict__ Oout = ptrs.o[c];
    const OT* __restrict__ Oc = O + (long long)c * e;
    if (VEC == 4) {
        // Four independent vectors per thread and trip, all loads first: when the block runs squeezed beside a resident
        // GEMM CTA (one 128-thread block per SM), the bytes it keeps in flight are all the bandwidth it gets.
        constexpr int UNROLL = 4;
        constexpr long long STEP = (long long)EW_THREADS * 4;
        long long i = lo + (long long)threadIdx.x * 4;
        for (; i + (UNROLL - 1) * STEP < hi; i += UNROLL * STEP) {
            float4 w[UNROLL], o[UNROLL];
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) w[u] = __ldcs(reinterpret_cast<const float4*>(W + i + u * STEP));
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) o[u] = GradLoad<OT>::load4(Oc + i + u * STEP);
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                w[u].x = fmaf(-eta_gamma, o[u].x, fmaf(-eta_lambda, w[u].x, w[u].x));
                w[u].y = fmaf(-eta_gamma, o[u].y, fmaf(-eta_lambda, w[u].y, w[u].y));
                w[u].z = fmaf(-eta_gamma, o[u].z, fmaf(-eta_lambda, w[u].z, w[u].z));
                w[u].w = fmaf(-eta_gamma, o[u].w, fmaf(-eta_lambda, w[u].w, w[u].w));
                __stcs(reinterpret_cast<float4*>(W + i + u * STEP), w[u]);
                if (Oout) *reinterpret_cast<float4*>(Oout + i + u * STEP) = o[u];
            }
        }
        for (; i < hi; i += STEP) {
            float4 w = __ldcs(reinterpret_cast<const float4*>(W + i));
            float4 o = GradLoad<OT>::load4(Oc + i);
            w.x = fmaf(-eta_gamma, o.x, fmaf(-eta_lambda, w.x, w.x));
            w.y = fmaf(-eta_gamma, o.y, fmaf(-eta_lambda, w.y, w.y));
            w.z = fmaf(-eta_gamma, o.z, fmaf(-eta_lambda, w.z, w.z));
            w.w = fmaf(-eta_gamma, o.w, fmaf(-eta_lambda, w.w, w.w));
            __stcs(reinterpret_cast<float4*>(W + i), w);
            if (Oout) *reinterpret_cast<float4*>(Oout + i) = o;
        }
    } else {
        constexpr int UNROLL = 8;            // as in the prologue
        for (long long i = lo + threadIdx.x; i < hi; i += UNROLL * EW_THREADS) {
            float w[UNROLL], o[UNROLL];
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const long long j = i + u * EW_THREADS;
                w[u] = o[u] = 0.f;
                if (j < hi) { w[u] = W[j]; o[u] = GradLoad<OT>::load1(Oc + j); }
            }
            #pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
                const long long j = i + u * EW_THREADS;
                if (j < hi) {
                    W[j] = fmaf(-eta_gamma, o[u], fmaf(-eta_lambda, w[u], w[u]));
                    if (Oout) Oout[j] = o[u];
                }
            }
        }
    }
}

// X_0 = M * inv_norm (fp32 validation path only).
__global__ void __launch_bounds__(EW_THREADS)
scale_kernel(const float* __restrict__ M, float* __restrict__ X, const float* __restrict__ inv_norm, long long e,
             long long slab_len) {
    let_next_start();
    wait_for_stream();
    const int c = blockIdx.y;
    const long long lo = (long long)blockIdx.x * slab_len;
    const long long hi = (lo + slab_len < e) ? lo + slab_len : e;
    const float s = inv_norm[c];
    for (long long i = lo + threadIdx.x; i < hi; i += EW_THREADS) X[(long long)c * e + i] = M[(long long)c * e + i] * s;
}

}  // namespace

namespace {
template <typename GT, typename ST, int CAP>
void launch_prologue_cap(dim3 grid, dim3 block, cudaStream_t stream, bool vec4, const ChunkPtrs& ptrs, float* M, void* A, void* Gp,
                         __nv_bfloat16* xhat, float* partials, unsigned int* counters, float* inv_norm, DeviceStatus* status,
                         long long e, long long slab_len, const PrologueScalars& k, unsigned int* zero, int zero_words, float** params) {
    GradTable<CAP> t;
    for (unsigned c = 0; c < grid.y; ++c) { t.g[c] = ptrs.g[c]; t.w[c] = ptrs.w[c]; t.gid[c] = ptrs.gid[c]; }
    if (vec4) prologue_kernel<GT, ST, 4, CAP><<<grid, block, 0, stream>>>(t, M, A, Gp, xhat, partials, counters, inv_norm, status, e, slab_len, (int)norm_unit(e), (int)(slab_len / norm_unit(e)), (int)((e + norm_unit(e) - 1) / norm_unit(e)), k, zero, zero_words, params);
    else      prologue_kernel<GT, ST, 1, CAP><<<grid, block, 0, stream>>>(t, M, A, Gp, xhat, partials, counters, inv_norm, status, e, slab_len, (int)norm_unit(e), (int)(slab_len / norm_unit(e)), (int)((e + norm_unit(e) - 1) / norm_unit(e)), k, zero, zero_words, params);
}
template <typename GT, typename ST>
void launch_prologue_t(dim3 grid, dim3 block, cudaStream_t stream, bool vec4, const ChunkPtrs& ptrs, float* M, void* A, void* Gp,
                       __nv_bfloat16* xhat, float* partials, unsigned int* counters, float* inv_norm, DeviceStatus* status,
                       long long e, long long slab_len, const PrologueScalars& k, unsigned int* zero, int zero_words, float** params) {
    if (grid.y <= SMALL_TABLE) launch_prologue_cap<GT, ST, SMALL_TABLE>(grid, block, stream, vec4, ptrs, M, A, Gp, xhat, partials, counters, inv_norm, status, e, slab_len, k, zero, zero_words, params);
    else                       launch_prologue_cap<GT, ST, MAXC>(grid, block, stream, vec4, ptrs, M, A, Gp, xhat, partials, counters, inv_norm, status, e, slab_len, k, zero, zero_words, params);
}
template <typename OT, int CAP>
cudaError_t launch_update_cap(dim3 grid, dim3 block, cudaStream_t stream, bool vec4, const ChunkPtrs& ptrs, const void* O, long long e,
                              long long slab_len, float eta_lambda, float eta_gamma, bool early) {
    ParamTable<CAP> t;
    for (unsigned c = 0; c < grid.y; ++c) { t.w[c] = ptrs.w[c]; t.o[c] = ptrs.o[c]; }
    return launch_kernel(vec4 ? update_kernel<OT, 4, CAP> : update_kernel<OT, 1, CAP>, grid, block, 0, stream, early, t, (const OT*)O, e, slab_len, eta_lambda, eta_gamma);
}
}  // namespace

cudaError_t launch_prologue(const ChunkPtrs& ptrs, int C, bool grad_bf16, int state_kind, bool vec4, float* M, void* A, void* Gp,
                            __nv_bfloat16* xhat, float* partials, unsigned int* counters, float* inv_norm,
                            DeviceStatus* status, long long e, long long slab_len, int slabs,
                            const PrologueScalars& k, unsigned int* zero, int zero_words, float** params, cudaStream_t stream) {
    dim3 grid(slabs, C), block(EW_THREADS);
#define MONA_PROLOGUE_CASE(GT, ST) launch_prologue_t<GT, ST>(grid, block, stream, vec4, ptrs, M, A, Gp, xhat, partials, counters, inv_norm, status, e, slab_len, k, zero, zero_words, params)
    if (grad_bf16) {
        if (state_kind == PROLOGUE_NO_AUX) MONA_PROLOGUE_CASE(__nv_bfloat16, NoAux);
        else if (state_kind == PROLOGUE_AUX_COMBINED) MONA_PROLOGUE_CASE(__nv_bfloat16, Combined);
        else if (state_kind == PROLOGUE_AUX_BF16) MONA_PROLOGUE_CASE(__nv_bfloat16, __nv_bfloat16);
        else MONA_PROLOGUE_CASE(__nv_bfloat16, float);
    } else {
        if (state_kind == PROLOGUE_NO_AUX) MONA_PROLOGUE_CASE(float, NoAux);
        else if (state_kind == PROLOGUE_AUX_COMBINED) MONA_PROLOGUE_CASE(float, Combined);
        else if (state_kind == PROLOGUE_AUX_BF16) MONA_PROLOGUE_CASE(float, __nv_bfloat16);
        else MONA_PROLOGUE_CASE(float, float);
    }
#undef MONA_PROLOGUE_CASE
    return cudaGetLastError();
}

cudaError_t launch_param_table(const ChunkPtrs& ptrs, int C, float** params, cudaStream_t stream) {
    ParamTable<MAXC> t = {};
    for (int c = 0; c < C; ++c) t.w[c] = ptrs.w[c];
    return launch_kernel(param_table_kernel, dim3(1), dim3(EW_THREADS), 0, stream, false, t, params, C);
}

cudaError_t launch_update(const ChunkPtrs& ptrs, int C, bool o_is_bf16, bool vec4, const void* O, long long e,
                          long long slab_len, int slabs, float eta_lambda, float eta_gamma, bool early, cudaStream_t stream) {
    dim3 grid(slabs, C), block(EW_THREADS);
    const bool small = C <= SMALL_TABLE;
#define MONA_UPDATE_CASE(OT, CAP) return launch_update_cap<OT, CAP>(grid, block, stream, vec4, ptrs, O, e, slab_len, eta_lambda, eta_gamma, early)
    if (o_is_bf16) { if (small) MONA_UPDATE_CASE(__nv_bfloat16, SMALL_TABLE); else MONA_UPDATE_CASE(__nv_bfloat16, MAXC); }
    else           { if (small) MONA_UPDATE_CASE(float, SMALL_TABLE); else MONA_UPDATE_CASE(float, MAXC); }
#undef MONA_UPDATE_CASE
}

cudaError_t launch_scale(const float* M, float* X, const float* inv_norm, int C, long long e, long long slab_len,
                         int slabs, cudaStream_t stream) {
    return launch_kernel(scale_kernel, dim3(slabs, C), dim3(EW_THREADS), 0, stream, true, M, X, inv_norm, e, slab_len);
}

}  // namespace mona

// ---------------------------------------------------------------------------------------------------
// Allocation-free single-matrix prologue (mona_prologue_noalloc, declared in include/mona.h).
//
// The fused prologue needs a little global scratch: a partial sum of squares per unit of the norm and a counter
// that tells the last slab to finish that it must add them up.  The handle-based path keeps that
// scratch in the caller's workspace.  Some callers have no workspace to give and cannot create one:
// a process whose framework allocator has already claimed the whole device, or a hook that must not
// trigger the device-wide synchronisation that cudaMalloc/cudaFree imply.  For them the scratch below
// lives in the library image itself; every GPU that loads the library carries these 2 KiB until the
// process exits.
#include <mutex>

#include "../../include/mona.h"

namespace mona {
namespace {

constexpr long long NOALLOC_MAX_ELEMS = 1ll << 24;      // one 4096 x 4096 matrix
constexpr int NOALLOC_MAX_DEVICES = 64;

struct NoAllocScratch {
    float partials[MAX_UNITS];     // partial sums of squares (fully rewritten by every call)
    unsigned int counter;          // slab arrival counter; must be 0 when a call starts
    unsigned int pad[3];
    DeviceStatus status;           // sink of the kernel's non-finite flag; the caller reads inv_norm_out instead
};
static_assert(sizeof(NoAllocScratch) <= 2048, "scratch layout");

// In host code this name is only a handle for cudaGetSymbolAddress, never an address to hand to a kernel.
static __device__ __align__(256) unsigned char g_noalloc_scratch[2048];

std::mutex g_noalloc_mutex;
NoAllocScratch* g_noalloc_dev_ptr[NOALLOC_MAX_DEVICES] = {nullptr};
int g_noalloc_dev_major[NOALLOC_MAX_DEVICES] = {0};

void set_msg(char* buf, size_t len, const char* msg) {
    if (buf && len) {
        size_t i = 0;
        for (; msg[i] && i + 1 < len; ++i) buf[i] = msg[i];
        buf[i] = 0;
    }
}

F2 split_double(double v) {
    F2 r;
    r.hi = (float)v;
    r.lo = (float)(v - (double)r.hi);
    return r;
}

}  // namespace
}  // namespace mona

extern "C" mona_status mona_prologue_noalloc(const void* grad, int32_t grad_dtype, float* M, float* A, float* G_prev,
                                             void* xhat_bf16, float* inv_norm_out, int64_t rows, int64_t cols,
                                             const mona_hparams* hp, void* stream_v, char* err, size_t err_len) {
    using namespace mona;
    if (!grad || !M || !A || !G_prev || !inv_norm_out || !hp) { set_msg(err, err_len, "null pointer argument"); return MONA_ERR_INVALID_ARG; }
    if (rows <= 0 || cols <= 0) { set_msg(err, err_len, "rows and cols must be positive"); return MONA_ERR_INVALID_ARG; }
    if (grad_dtype != MONA_F32 && grad_dtype != MONA_BF16) { set_msg(err, err_len, "unknown grad_dtype"); return MONA_ERR_INVALID_ARG; }
    if (hp->algorithm != 0) { set_msg(err, err_len, "this entry point runs the MONA prologue only (hp->algorithm must be 0)"); return MONA_ERR_INVALID_ARG; }
    if (rows > NOALLOC_MAX_ELEMS || cols > NOALLOC_MAX_ELEMS || rows * cols > NOALLOC_MAX_ELEMS) {
        set_msg(err, err_len, "matrix larger than the built-in scratch supports: rows*cols must be <= 16777216 (4096 x 4096)");
        return MONA_ERR_UNSUPPORTED_SHAPE;
    }
    if (((uintptr_t)grad | (uintptr_t)M | (uintptr_t)A | (uintptr_t)G_prev | (uintptr_t)xhat_bf16) & 15) {
        set_msg(err, err_len, "matrix pointers must be 16-byte aligned");
        return MONA_ERR_ALIGNMENT;
    }
    int dev = -1;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) { set_msg(err, err_len, "no current CUDA device"); return MONA_ERR_CUDA; }
    NoAllocScratch* scratch = nullptr;
    {
        // once per device, with that device current: resolve the device address of the static array
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_dev_ptr[dev]) {
            void* p = nullptr;
            ce = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (ce != cudaSuccess || !p) { set_msg(err, err_len, cudaGetErrorString(ce)); return MONA_ERR_CUDA; }
            int major = 0;
            ce = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
            if (ce != cudaSuccess) { set_msg(err, err_len, cudaGetErrorString(ce)); return MONA_ERR_CUDA; }
            g_noalloc_dev_major[dev] = major;
            g_noalloc_dev_ptr[dev] = reinterpret_cast<NoAllocScratch*>(p);
        }
        if (g_noalloc_dev_major[dev] != 10) { set_msg(err, err_len, "the current device is not compute capability 10.x"); return MONA_ERR_ARCH; }
        scratch = g_noalloc_dev_ptr[dev];
    }
    cudaStream_t stream = (cudaStream_t)stream_v;
    const long long e = rows * cols;
    long long slab = 0;
    int slabs = 0;
    slab_plan(e, 1, norm_unit(e), &slab, &slabs);
    // the array keeps whatever the previous call left: the counter has to start from zero
    ce = cudaMemsetAsync(&scratch->counter, 0, sizeof(unsigned int), stream);
    if (ce != cudaSuccess) { set_msg(err, err_len, cudaGetErrorString(ce)); return MONA_ERR_CUDA; }
    ChunkPtrs ptrs;
    ptrs.g[0] = grad; ptrs.w[0] = nullptr; ptrs.o[0] = nullptr; ptrs.gid[0] = 0;
    PrologueScalars k;
    k.beta = split_double(hp->accel_beta);
    k.one_minus_beta = split_double(1.0 - hp->accel_beta);
    k.alpha = split_double(hp->accel_alpha);
    k.mu = split_double(hp->momentum);
    k.eps = (float)hp->norm_eps;
    ce = launch_prologue(ptrs, 1, grad_dtype == MONA_BF16, PROLOGUE_AUX_F32, e % 4 == 0, M, A, G_prev, (__nv_bfloat16*)xhat_bf16, scratch->partials,
                         &scratch->counter, inv_norm_out, &scratch->status, e, slab, slabs, k, nullptr, 0, nullptr, stream);
    if (ce != cudaSuccess) { set_msg(err, err_len, cudaGetErrorString(ce)); return MONA_ERR_CUDA; }
    set_msg(err, err_len, "");
    return MONA_OK;
}
