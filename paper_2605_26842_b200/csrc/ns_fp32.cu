// fp32 validation path of Eq. newton_schulz: a plain shared-memory tiled SGEMM with generic operand
// strides, so that X X^T, X^T X, A A and B X / X B all go through the same kernel without any
// transposed copy.  Products and sums are fp32 FMA throughout; this path exists to separate algorithmic
// errors from bf16 rounding, and to serve shapes the tensor-core path does not take.
#include "ns_fp32.cuh"

namespace mona {

namespace {

// A block computes a 64 x 64 tile of D with four groups of 64 threads.  Each group takes a quarter of every k-slab (16 of 64) and
// each thread 8 x 8 elements of the whole tile, so that 64 FMAs cost four 16-byte shared-memory reads (4 x 4 per thread cost
// eight 4-byte reads per 16); the groups' sums are added through shared memory at the end, in group order.  The k split, not
// a larger tile, fills the block: these matrices have few tiles (1001 x 1001: 136 of 64 x 64 in the lower triangle, 36 of
// 128 x 128), so the tile stays small and eight warps share it.  Slabs are fetched with 4-byte asynchronous copies - odd row
// lengths leave no wider alignment - two slabs ahead of the arithmetic.
// Bound: fp32 FMA issue while there is a tile for every SM, the chain of dependent products below that.  Symmetric products
// compute the tiles on and below the diagonal and write each twice.
// Measured (T = 5 products of one 1001 x 1500 matrix, X X^T / A A / B' X): 154 / 100 / 122 us with the 4 x 4 kernel and both halves
// of the symmetric products, 83 / 59 / 158 with these tiles, 54 / 38 / 101 with packed FMAs, unchecked copies of interior slabs
// and no register cap (an SM holds one block then, but a capped one spilled), slabs of 64 instead of 32 another 7 %; five odd
// matrices, 1001 x 1500 the largest: 2.91 -> 1.21 ms per step.
constexpr int TS = 64;                   // tile of D per block
constexpr int TK = 64;                   // k-slab
constexpr int SG_GROUPS = 4;             // thread groups, TK / SG_GROUPS k each
constexpr int SG_THREADS = 64 * SG_GROUPS;
constexpr int PITCH = TS + 4;            // 4 mod 32: see copy_slab
constexpr int SLAB = TK * PITCH;         // floats of one operand's slab
constexpr int SG_STAGES = 3;             // slabs in flight or in use
constexpr size_t SG_SMEM = sizeof(float) * (2 * SG_STAGES * SLAB > SG_GROUPS * TS * PITCH ? 2 * SG_STAGES * SLAB : SG_GROUPS * TS * PITCH);

__device__ __forceinline__ void cp_async4(uint32_t d, const float* src, bool valid) {
    const int bytes = valid ? 4 : 0;                       // 0: the word is zero-filled and nothing is read
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
// One thread's share of fetching an operand: slab n becomes dst[k][r] (pitch PITCH) = src(r0 + r, n TK + k) for r < 64, k < TK, zero
// outside rows x K, src(r, k) = src[r * s_r + k * s_k].  When k is contiguous, a warp's lanes cover 8 k of 4 rows: whole 32-byte
// sectors, and with PITCH = 4 mod 32 the 32 words fall into different banks; otherwise they cover 32 consecutive rows.  Either way a
// thread's elements differ in one coordinate only, so that each costs an addition and a comparison.
struct SlabCopy {
    static constexpr int ROWS = 4 * (SG_THREADS / 32) / (TK / 8);    // rows all warps cover at once when k is contiguous
    const float* src;           // this thread's first element of slab 0
    long long step, slab_step;  // in elements: to its next element, to the next slab
    int first, limit, stride;   // row of its first element, bound, change per element
    int k, k_stride;            // k of its first element in slab 0, change per element
    int dst, dst_step;          // position in the slab, change per element
    __device__ __forceinline__ SlabCopy(const float* base, long long s_r, long long s_k, int r0, int rows) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const bool k_fast = s_k == 1;
        constexpr int KW = TK / 8;       // warps side by side along k when k is contiguous
        const int r = k_fast ? (warp / KW) * 4 + (lane >> 3) : (warp & 1) * 32 + lane;
        k = k_fast ? (warp % KW) * 8 + (lane & 7) : warp >> 1;
        src = base + (long long)(r0 + r) * s_r + (long long)k * s_k;
        step = k_fast ? ROWS * s_r : 4 * s_k;
        slab_step = (long long)TK * s_k;
        dst = k * PITCH + r;
        dst_step = k_fast ? ROWS : 4 * PITCH;
        first = r0 + r; limit = rows; stride = k_fast ? ROWS : 0;
        k_stride = k_fast ? 0 : 4;
    }
    // `inside`: the whole slab lies inside rows x K (the same for all threads of the block)
    __device__ __forceinline__ void fetch(float* buf, const float* safe, int n, int K, bool inside) const {
        const float* p = src + (long long)n * slab_step;
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(buf + dst);
        if (inside) {
            #pragma unroll
            for (int q = 0; q < TS * TK / SG_THREADS; ++q) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + (uint32_t)(q * dst_step * 4)), "l"(p) : "memory");
                p += step;
            }
            return;
        }
        int r = first, kk = n * TK + k;
        #pragma unroll
        for (int q = 0; q < TS * TK / SG_THREADS; ++q) {
            const bool valid = r < limit && kk < K;
            cp_async4(d + (uint32_t)(q * dst_step * 4), valid ? p : safe, valid);
            p += step; r += stride; kk += k_stride;
        }
    }
};

// Two independent fp32 FMAs (round to nearest) in one instruction: half the issue slots of the scalar form.
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__global__ void __launch_bounds__(SG_THREADS, 1) sgemm_kernel(const __grid_constant__ SgemmArgs g) {
    extern __shared__ __align__(16) float sg[];
    wait_for_stream();
    const int z = blockIdx.z;
    const float* __restrict__ A = g.a + (long long)z * g.a_batch;
    const float* __restrict__ B = g.b + (long long)z * g.b_batch;
    int ti = blockIdx.y, tj = blockIdx.x;
    if (g.symmetric) {                                     // lower triangle, row by row
        ti = 0;
        while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.x) ++ti;
        tj = blockIdx.x - ti * (ti + 1) / 2;
    }
    const int i0 = ti * TS, j0 = tj * TS;
    const int group = threadIdx.x >> 6, tx = threadIdx.x & 7, ty = (threadIdx.x >> 3) & 7;
    const int slabs = (g.K + TK - 1) / TK;
    const SlabCopy copy_a(A, g.a_si, g.a_sk, i0, g.M), copy_b(B, g.b_sj, g.b_sk, j0, g.N);
    auto fetch = [&](int n, int stage) {
        float* buf = sg + stage * 2 * SLAB;
        const bool k_inside = (n + 1) * TK <= g.K;
        if (n < slabs) { copy_a.fetch(buf, A, n, g.K, k_inside && i0 + TS <= g.M); copy_b.fetch(buf + SLAB, B, n, g.K, k_inside && j0 + TS <= g.N); }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    unsigned long long acc[8][4];                          // 8 x 8 sums, two neighbouring columns per register pair
    #pragma unroll
    for (int r = 0; r < 8; ++r)
        #pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
    #pragma unroll
    for (int n = 0; n < SG_STAGES - 1; ++n) fetch(n, n);
    int stage = 0;
    for (int n = 0; n < slabs; ++n) {
        asm volatile("cp.async.wait_group %0;" ::"n"(SG_STAGES - 2) : "memory");
        __syncthreads();                                   // the slab is here, and everyone is done with the one before it
        fetch(n + SG_STAGES - 1, stage == 0 ? SG_STAGES - 1 : stage - 1);
        const float* as = sg + stage * 2 * SLAB + group * (TK / SG_GROUPS) * PITCH;
        const float* bs = as + SLAB;
        #pragma unroll
        for (int kk = 0; kk < TK / SG_GROUPS; ++kk) {
            float a[8];
            ulonglong2 b[2];
            *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(as + kk * PITCH + 4 * ty);
            *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(as + kk * PITCH + 32 + 4 * ty);
            b[0] = *reinterpret_cast<const ulonglong2*>(bs + kk * PITCH + 4 * tx);
            b[1] = *reinterpret_cast<const ulonglong2*>(bs + kk * PITCH + 32 + 4 * tx);
            #pragma unroll
            for (int r = 0; r < 8; ++r) {
                unsigned long long aa;
                asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(a[r]));
                fma2(acc[r][0], aa, b[0].x); fma2(acc[r][1], aa, b[0].y);
                fma2(acc[r][2], aa, b[1].x); fma2(acc[r][3], aa, b[1].y);
            }
        }
        stage = stage + 1 == SG_STAGES ? 0 : stage + 1;
    }
    let_next_start();                                      // not earlier: waiting blocks would hold SMs that other streams' products need
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();                                       // the slabs' memory becomes the groups' partial tiles
    float* part = sg + group * TS * PITCH;
    #pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int row = (r >> 2) * 32 + 4 * ty + (r & 3);
        #pragma unroll
        for (int h = 0; h < 2; ++h)
            *reinterpret_cast<ulonglong2*>(part + row * PITCH + 32 * h + 4 * tx) = make_ulonglong2(acc[r][2 * h], acc[r][2 * h + 1]);
    }
    __syncthreads();
    float* __restrict__ D = g.d + (long long)z * g.d_batch;
    const float* __restrict__ Cin = g.cin ? g.cin + (long long)z * g.d_batch : nullptr;
    const bool mirror = g.symmetric && ti != tj;
    #pragma unroll 4
    for (int idx = threadIdx.x; idx < TS * TS; idx += SG_THREADS) {
        const int r = idx >> 6, c = idx & 63, gi = i0 + r, gj = j0 + c;
        float v = sg[r * PITCH + c];
        #pragma unroll
        for (int q = 1; q < SG_GROUPS; ++q) v += sg[q * TS * PITCH + r * PITCH + c];
        v *= g.c2;
        if (gi < g.M && gj < g.N) {
            const long long off = (long long)gi * g.ldd + gj;
            if (Cin) v = fmaf(g.c1, Cin[off], v);
            if (gi == gj) v += g.diag_add;
            D[off] = v;
        }
        if (mirror) sg[r * PITCH + c] = v;                 // (each thread rewrites only words it alone has read)
    }
    if (mirror) {
        __syncthreads();
        #pragma unroll 4
        for (int idx = threadIdx.x; idx < TS * TS; idx += SG_THREADS) {
            const int c = idx >> 6, r = idx & 63, gi = i0 + r, gj = j0 + c;
            if (gi < g.M && gj < g.N) D[(long long)gj * g.ldd + gi] = sg[r * PITCH + c];
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Small matrices (shorter side <= 64, e.g. a 32 x 1024 router): the whole Newton-Schulz iteration of one matrix in ONE
// cluster of 1 to 8 blocks.  The matrix lives in shared memory in its wide orientation Y (s x l, tall inputs are transposed
// while loading).  Its columns are cut into 1, 2, 4 or 8 parts by the shape alone; every block holds one or several neighbouring
// parts.  An iteration forms the share of A = Y Y^T of each part, adds the shares as a binary tree over the parts - inside the
// block first, then over the blocks through distributed shared memory, the same tree whatever the number of blocks, so that a
// matrix's result does not depend on how many are in the launch - forms B' = b A + c A^2 + a I in every block and overwrites the
// block's columns with B' Y, in plain fp32 FMA throughout.
//
// Bound: latency - a few thousand FMAs per thread and iteration, one cluster barrier each.  A matrix has 4 s^2 l FMAs' worth of work
// per iteration, too much for one block; split by columns the only exchange is the s x s sum.  The two products read shared
// memory 16 bytes at a time: Y Y^T as 4 x 4 register tiles whose k range is dealt to four neighbouring lanes (20 wavefronts
// per 64 FMAs and lane), B' Y with a column of Y in registers and the rows of B' as broadcasts.
// Measured against one block per matrix with scalar shared-memory reads, five iterations: one 32 x 512 matrix 180 -> 31 us, 512 of
// 32 x 1024 1247 -> 664, one 63 x 1000 459 -> 111.
constexpr int SMALL_THREADS = 256, SMALL_THREADS64 = 384;    // s up to 32, up to 64 (512 leave a thread too few registers for its column)
constexpr int SMALL_KGROUPS = 4;             // lanes that share a 4 x 4 block of A
constexpr int SMALL_MAX_CLUSTER = 8;         // the largest portable cluster
constexpr int SMALL_MIN_COLS = 64;           // a part with fewer columns spends its time in barriers
constexpr size_t SMALL_MAX_SMEM = 200 * 1024;

struct SmallLayout {                         // of one block's shared memory, in floats
    int s4, part, cols, lp, sp;              // padded rows, columns per part and per block, pitch of Y, pitch of the s x s matrices
    __host__ __device__ SmallLayout(int s, int l, int parts, int cluster) {
        s4 = (s + 3) & ~3;
        part = ((l + parts - 1) / parts + 4 * SMALL_KGROUPS - 1) / (4 * SMALL_KGROUPS) * (4 * SMALL_KGROUPS);
        cols = parts / cluster * part;
        lp = cols + 4;                       // 4 mod 16: rows 4 apart start 16 banks apart, two rows of four lanes per wavefront
        sp = s4 + 4;
    }
    __host__ __device__ size_t bytes() const { return ((size_t)s4 * lp + 4 * (size_t)s4 * sp) * sizeof(float); }   // Y, two shares of A, A, B'
};

__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void small_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ float4 add4(const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

template <int SMAX, int THREADS>   // SMAX: upper bound of the padded shorter side, 32 or 64 (a thread holds a column of Y in registers)
__global__ void __launch_bounds__(THREADS, SMAX <= 32 ? 2 : 1)
small_ns_kernel(const float* __restrict__ M, float* __restrict__ O, const float* __restrict__ inv_norm, int rows, int cols,
                int parts, int T, float ca, float cb, float cc) {
    extern __shared__ __align__(16) float sm[];
    wait_for_stream();
    uint32_t rank, n;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    const bool tall = rows > cols;
    const int s = tall ? cols : rows, l = tall ? rows : cols;
    const SmallLayout L(s, l, parts, (int)n);
    const int s4 = L.s4, lp = L.lp, sp = L.sp, nc = L.cols;
    float* Y = sm;
    float* share[2] = {Y + (size_t)s4 * lp, Y + (size_t)s4 * lp + s4 * sp};
    float* A = share[1] + s4 * sp;
    float* B = A + s4 * sp;
    const int mat = blockIdx.x / n;
    const float* Mz = M + (long long)mat * rows * cols;
    float* Oz = O + (long long)mat * rows * cols;
    const float scale = inv_norm[mat];
    const int tid = threadIdx.x;
    const int c_lo = (int)rank * nc;                              // this block's columns of the wide orientation
    const int c_n = max(0, min(nc, l - c_lo));

    // X_0 = M / (||M||_F + eps); rows and columns of the padding are zero and stay zero
    for (int idx = tid; idx < s4 * lp; idx += THREADS) Y[idx] = 0.f;
    __syncthreads();
    for (int idx = tid; idx < s * c_n; idx += THREADS) {
        if (!tall) { const int r = idx / c_n, q = idx - r * c_n; Y[r * lp + q] = Mz[(long long)r * cols + c_lo + q] * scale; }
        else       { const int q = idx / s, r = idx - q * s;     Y[r * lp + q] = Mz[(long long)c_lo * cols + idx] * scale; }
    }
    __syncthreads();

    const int nb = s4 >> 2;               // 4 x 4 blocks of A per side
    const int nblocks = nb * (nb + 1) / 2;
    const int kg = tid % SMALL_KGROUPS;
    for (int t = 0; t < T; ++t) {
        float* mine = share[t & 1];       // two, so that one cluster barrier per iteration is enough
        // (the loop bound is the same for all threads of a warp's group of four; the shuffles stay inside the group)
        for (int blk0 = 0; blk0 < nblocks; blk0 += THREADS / SMALL_KGROUPS) {
            const int blk = blk0 + tid / SMALL_KGROUPS;
            int bi = 0;
            while ((bi + 1) * (bi + 2) / 2 <= blk) ++bi;
            const int bj = blk - bi * (bi + 1) / 2;
            float4 sum, level0, level1, level2;       // of the parts so far: complete groups of 1, 2 and 4
            const int block_parts = parts / (int)n;
            for (int pt = 0; pt < block_parts; ++pt) {
                float acc[4][4];
                #pragma unroll
                for (int r = 0; r < 4; ++r)
                    #pragma unroll
                    for (int q = 0; q < 4; ++q) acc[r][q] = 0.f;
                if (blk < nblocks) {
                    const float* ya = Y + (size_t)4 * bi * lp + pt * L.part + 4 * kg;
                    const float* yb = Y + (size_t)4 * bj * lp + pt * L.part + 4 * kg;
                    for (int k = 0; k < L.part; k += 4 * SMALL_KGROUPS) {
                        float4 a[4], b[4];
                        #pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            a[r] = *reinterpret_cast<const float4*>(ya + r * lp + k);
                            b[r] = *reinterpret_cast<const float4*>(yb + r * lp + k);
                        }
                        #pragma unroll
                        for (int r = 0; r < 4; ++r)
                            #pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                acc[r][q] = fmaf(a[r].x, b[q].x, acc[r][q]);
                                acc[r][q] = fmaf(a[r].y, b[q].y, acc[r][q]);
                                acc[r][q] = fmaf(a[r].z, b[q].z, acc[r][q]);
                                acc[r][q] = fmaf(a[r].w, b[q].w, acc[r][q]);
                            }
                    }
                }
                // added over the four lanes so that lane kg is left with row kg of the block
                const bool up2 = kg & 2, up1 = kg & 1;
                float half[2][4], v[4];
                #pragma unroll
                for (int r = 0; r < 2; ++r)
                    #pragma unroll
                    for (int q = 0; q < 4; ++q)
                        half[r][q] = (up2 ? acc[2 + r][q] : acc[r][q]) + __shfl_xor_sync(0xffffffffu, up2 ? acc[r][q] : acc[2 + r][q], 2);
                #pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = (up1 ? half[1][q] : half[0][q]) + __shfl_xor_sync(0xffffffffu, up1 ? half[0][q] : half[1][q], 1);
                sum = make_float4(v[0], v[1], v[2], v[3]);
                if (!(pt & 1)) level0 = sum;
                else {
                    sum = add4(level0, sum);
                    if (!(pt & 2)) level1 = sum;
                    else {
                        sum = add4(level1, sum);
                        if (!(pt & 4)) level2 = sum; else sum = add4(level2, sum);
                    }
                }
            }
            if (blk < nblocks) {                     // row kg of the block and its mirror image
                *reinterpret_cast<float4*>(mine + (4 * bi + kg) * sp + 4 * bj) = sum;
                mine[(4 * bj) * sp + 4 * bi + kg] = sum.x; mine[(4 * bj + 1) * sp + 4 * bi + kg] = sum.y;
                mine[(4 * bj + 2) * sp + 4 * bi + kg] = sum.z; mine[(4 * bj + 3) * sp + 4 * bi + kg] = sum.w;
            }
        }
        // A = the sum of all blocks' shares, the tree over the parts carried on
        if (n > 1) small_cluster_sync(); else __syncthreads();
        const uint32_t mine_addr = (uint32_t)__cvta_generic_to_shared(mine);
        for (int idx = tid; idx < s4 * nb; idx += THREADS) {
            const int off = (idx / nb) * sp + 4 * (idx % nb);
            float4 v[SMALL_MAX_CLUSTER];
            #pragma unroll
            for (uint32_t r = 0; r < SMALL_MAX_CLUSTER; ++r) {
                if (r < n) {
                    uint32_t addr;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(mine_addr + 4u * off), "r"(r));
                    v[r] = ld_cluster4(addr);
                }
            }
            #pragma unroll
            for (uint32_t w = 1; w < SMALL_MAX_CLUSTER; w *= 2)
                #pragma unroll
                for (uint32_t r = 0; r < SMALL_MAX_CLUSTER; r += 2 * w)
                    if (r + w < n) v[r] = add4(v[r], v[r + w]);
            *reinterpret_cast<float4*>(A + off) = v[0];
        }
        __syncthreads();
        // B' = b A + c A A + a I
        for (int idx = tid; idx < s4 * nb; idx += THREADS) {
            const int i = idx / nb, j = 4 * (idx - i * nb);
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
            #pragma unroll 8
            for (int k = 0; k < s4; ++k) {
                const float a = A[i * sp + k];
                const float4 v = *reinterpret_cast<const float4*>(A + k * sp + j);
                sum.x = fmaf(a, v.x, sum.x); sum.y = fmaf(a, v.y, sum.y); sum.z = fmaf(a, v.z, sum.z); sum.w = fmaf(a, v.w, sum.w);
            }
            const float4 v = *reinterpret_cast<const float4*>(A + i * sp + j);
            float4 o;
            o.x = fmaf(cb, v.x, cc * sum.x) + (i == j ? ca : 0.f);
            o.y = fmaf(cb, v.y, cc * sum.y) + (i == j + 1 ? ca : 0.f);
            o.z = fmaf(cb, v.z, cc * sum.z) + (i == j + 2 ? ca : 0.f);
            o.w = fmaf(cb, v.w, cc * sum.w) + (i == j + 3 ? ca : 0.f);
            *reinterpret_cast<float4*>(B + i * sp + j) = o;
        }
        __syncthreads();
        // Y <- B' Y: THREADS / 128 threads own a column, each a range of its rows; all hold the old column in registers
        constexpr int COLS = 128, ROW_GROUPS = THREADS / COLS;
        const int row0 = nb * (tid / COLS) / ROW_GROUPS * 4, row1 = nb * (tid / COLS + 1) / ROW_GROUPS * 4;
        for (int c0 = 0; c0 < nc; c0 += COLS) {
            const int q = c0 + tid % COLS;
            float y[SMAX];
            #pragma unroll
            for (int k = 0; k < SMAX; ++k) y[k] = (k < s4 && q < nc) ? Y[k * lp + q] : 0.f;
            __syncthreads();
            if (q < nc) {
                for (int i = row0; i < row1; ++i) {
                    float o[4] = {0.f, 0.f, 0.f, 0.f};
                    #pragma unroll
                    for (int k = 0; k < SMAX; k += 4) {
                        // s > 32: the load is predicated and zeros are added, since behind branches a row's loads wait for one
                        // another (a 63 x 1000 matrix 137 -> 117 us); below that the additions saved weigh more
                        if (SMAX <= 32 && k >= s4) continue;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (k < s4) v = *reinterpret_cast<const float4*>(B + i * sp + k);
                        o[0] = fmaf(v.x, y[k], o[0]); o[1] = fmaf(v.y, y[k + 1], o[1]);
                        o[2] = fmaf(v.z, y[k + 2], o[2]); o[3] = fmaf(v.w, y[k + 3], o[3]);
                    }
                    Y[i * lp + q] = (o[0] + o[1]) + (o[2] + o[3]);
                }
            }
        }
        __syncthreads();
    }
    let_next_start();
    for (int idx = tid; idx < s * c_n; idx += THREADS) {          // O = X_T, back in the input's orientation
        if (!tall) { const int r = idx / c_n, q = idx - r * c_n; Oz[(long long)r * cols + c_lo + q] = Y[r * lp + q]; }
        else       { const int q = idx / s, r = idx - q * s;     Oz[(long long)c_lo * cols + idx] = Y[r * lp + q]; }
    }
    if (n > 1) small_cluster_sync();      // no block leaves while another may still read its share
}

// Parts of a matrix, by its shape alone: as many as leave each SMALL_MIN_COLS columns.
int small_ns_parts(int l) {
    int n = 1;
    while (n < SMALL_MAX_CLUSTER && l >= 2 * n * SMALL_MIN_COLS) n *= 2;
    return n;
}
// Blocks per matrix: as many as there are parts while all matrices together have about one block per SM, and at least as many as
// the matrix needs to fit.
int small_ns_cluster(int s, int l, int parts, int batch) {
    int n = 1;
    while (n < parts && (SmallLayout(s, l, parts, n).bytes() > SMALL_MAX_SMEM || 2 * n * batch <= 148)) n *= 2;
    return n;
}

}  // namespace

// Every shape whose parts fit takes this path, however many there are: from a few hundred long matrices of s > 32 on the tiled
// products would be faster (512 of 63 x 2500: 4.8 ms against 7.3; 48: 1.24 against 0.82; one: 0.98 against 0.20), but they add in
// another order, and which path a matrix takes must not depend on its neighbours.
bool small_ns_eligible(long long rows, long long cols) {
    const long long s = rows < cols ? rows : cols, l = rows < cols ? cols : rows;
    if (s > 64 || l > (1 << 16)) return false;
    const int parts = small_ns_parts((int)l);
    return SmallLayout((int)s, (int)l, parts, parts).bytes() <= SMALL_MAX_SMEM;
}

cudaError_t small_ns_configure() {
    cudaError_t e = cudaFuncSetAttribute(small_ns_kernel<32, SMALL_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_MAX_SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(small_ns_kernel<64, SMALL_THREADS64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_MAX_SMEM);
}

cudaError_t launch_small_ns(const float* M, float* O, const float* inv_norm, int batch, int rows, int cols, int T,
                            float a, float b, float c, cudaStream_t stream) {
    const int s = rows < cols ? rows : cols, l = rows < cols ? cols : rows;
    const int parts = small_ns_parts(l), n = small_ns_cluster(s, l, parts, batch);
    const size_t smem = SmallLayout(s, l, parts, n).bytes();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(batch * n));
    cfg.blockDim = dim3(s > 32 ? SMALL_THREADS64 : SMALL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)n; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return s <= 32 ? cudaLaunchKernelEx(&cfg, small_ns_kernel<32, SMALL_THREADS>, M, O, inv_norm, rows, cols, parts, T, a, b, c)
                   : cudaLaunchKernelEx(&cfg, small_ns_kernel<64, SMALL_THREADS64>, M, O, inv_norm, rows, cols, parts, T, a, b, c);
}

cudaError_t sgemm_configure() { return cudaFuncSetAttribute(sgemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SG_SMEM); }

cudaError_t launch_sgemm(const SgemmArgs& g, cudaStream_t stream) {
    const int tm = (g.M + TS - 1) / TS, tn = (g.N + TS - 1) / TS;
    dim3 grid(g.symmetric ? tm * (tm + 1) / 2 : tn, g.symmetric ? 1 : tm, g.batch);
    return launch_kernel(sgemm_kernel, grid, dim3(SG_THREADS), SG_SMEM, stream, true, g);
}

}  // namespace mona
