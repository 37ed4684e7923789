// fp32 validation path of Eq. newton_schulz: a plain shared-memory tiled SGEMM with generic operand
// strides, so that X X^T, X^T X, A A and B X / X B all go through the same kernel without any
// transposed copy.  Accumulation is sequential fp32 FMA; this path exists to separate algorithmic
// errors from bf16 rounding, and to serve shapes the tensor-core path does not take.
#include "ns_fp32.cuh"

namespace mona {

namespace {

constexpr int TS = 64;   // tile of D per block
constexpr int TK = 16;   // k-slice
// 256 threads, each owns a 4x4 patch of the 64x64 tile.
__global__ void __launch_bounds__(256) sgemm_kernel(SgemmArgs g) {
    __shared__ float As[TK][TS + 4];
    __shared__ float Bs[TK][TS + 4];
    const int z = blockIdx.z;
    const float* __restrict__ A = g.a + (long long)z * g.a_batch;
    const float* __restrict__ B = g.b + (long long)z * g.b_batch;
    const int i0 = blockIdx.y * TS, j0 = blockIdx.x * TS;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[4][4];
    #pragma unroll
    for (int r = 0; r < 4; ++r)
        #pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;

    for (int k0 = 0; k0 < g.K; k0 += TK) {
        // each thread brings 4 elements of each operand slice
        #pragma unroll
        for (int q = 0; q < 4; ++q) {
            int idx = threadIdx.x + q * 256;          // 0..1023 = TK*TS
            int kk, mm;
            if (g.a_sk == 1) { kk = idx % TK; mm = idx / TK; } else { mm = idx % TS; kk = idx / TS; }
            int gi = i0 + mm, gk = k0 + kk;
            As[kk][mm] = (gi < g.M && gk < g.K) ? A[(long long)gi * g.a_si + (long long)gk * g.a_sk] : 0.f;
            int kb, nn;
            if (g.b_sk == 1) { kb = idx % TK; nn = idx / TK; } else { nn = idx % TS; kb = idx / TS; }
            int gj = j0 + nn, gk2 = k0 + kb;
            Bs[kb][nn] = (gj < g.N && gk2 < g.K) ? B[(long long)gk2 * g.b_sk + (long long)gj * g.b_sj] : 0.f;
        }
        __syncthreads();
        #pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            float a[4], b[4];
            #pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[kk][ty * 4 + r];
            #pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = Bs[kk][tx * 4 + c];
            #pragma unroll
            for (int r = 0; r < 4; ++r)
                #pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(a[r], b[c], acc[r][c]);
        }
        __syncthreads();
    }
    float* __restrict__ D = g.d + (long long)z * g.d_batch;
    const float* __restrict__ Cin = g.cin ? g.cin + (long long)z * g.d_batch : nullptr;
    #pragma unroll
    for (int r = 0; r < 4; ++r) {
        int gi = i0 + ty * 4 + r;
        if (gi >= g.M) continue;
        #pragma unroll
        for (int c = 0; c < 4; ++c) {
            int gj = j0 + tx * 4 + c;
            if (gj >= g.N) continue;
            long long off = (long long)gi * g.ldd + gj;
            float v = g.c2 * acc[r][c];
            if (Cin) v = fmaf(g.c1, Cin[off], v);
            D[off] = v;
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Small matrices (shorter side <= 64, e.g. a 32 x 1024 router): the whole Newton-Schulz iteration of one matrix in ONE
// cluster of 1 to 8 blocks.  The matrix lives in shared memory in its wide orientation Y (s x l, tall inputs are transposed
// while loading), every block holding a contiguous range of its columns.  An iteration forms the block's share of A = Y Y^T,
// adds the shares of all blocks through distributed shared memory (in rank order, so that all blocks hold the same bits), forms
// B' = b A + c A^2 + a I in every block and overwrites the block's columns with B' Y, in plain fp32 FMA throughout.
//
// Bound: latency - a few thousand FMAs per thread and iteration, one cluster barrier each.  A matrix has 4 s^2 l FMAs' worth of work
// per iteration, too much for one block; split by columns the only exchange is the s x s sum.  The two products read shared
// memory 16 bytes at a time: Y Y^T as 4 x 4 register tiles whose k range is dealt to four neighbouring lanes (20 wavefronts
// per 64 FMAs and lane), B' Y with a column of Y in registers and the rows of B' as broadcasts.
// Measured against one block per matrix with scalar shared-memory reads: a 32 x 512 matrix 182 -> 39 us (five iterations, 4
// blocks); the step of four layers of 512 x 1024 experts with their 32 x 1024 routers 4.26 -> 3.87 ms.
constexpr int SMALL_THREADS = 256;
constexpr int SMALL_KGROUPS = 4;             // lanes that share a 4 x 4 block of A
constexpr int SMALL_MAX_CLUSTER = 8;         // the largest portable cluster
constexpr int SMALL_MIN_COLS = 64;           // a block with fewer columns spends its time in barriers
constexpr size_t SMALL_MAX_SMEM = 200 * 1024;

struct SmallLayout {                         // of one block's shared memory, in floats
    int s4, cols, lp, sp;                    // padded rows, columns per block, pitch of Y, pitch of the s x s matrices
    __host__ __device__ SmallLayout(int s, int l, int cluster) {
        s4 = (s + 3) & ~3;
        cols = ((l + cluster - 1) / cluster + 4 * SMALL_KGROUPS - 1) / (4 * SMALL_KGROUPS) * (4 * SMALL_KGROUPS);
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

template <int SMAX>   // upper bound of the padded shorter side: 32 or 64 (a thread holds a column of Y in registers)
__global__ void __launch_bounds__(SMALL_THREADS)
small_ns_kernel(const float* __restrict__ M, float* __restrict__ O, const float* __restrict__ inv_norm, int rows, int cols,
                int T, float ca, float cb, float cc) {
    extern __shared__ __align__(16) float sm[];
    uint32_t rank, n;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    const bool tall = rows > cols;
    const int s = tall ? cols : rows, l = tall ? rows : cols;
    const SmallLayout L(s, l, (int)n);
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
    for (int idx = tid; idx < s4 * lp; idx += SMALL_THREADS) Y[idx] = 0.f;
    __syncthreads();
    for (int idx = tid; idx < s * c_n; idx += SMALL_THREADS) {
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
        for (int blk0 = 0; blk0 < nblocks; blk0 += SMALL_THREADS / SMALL_KGROUPS) {
            const int blk = blk0 + tid / SMALL_KGROUPS;
            int bi = 0;
            while ((bi + 1) * (bi + 2) / 2 <= blk) ++bi;
            const int bj = blk - bi * (bi + 1) / 2;
            float acc[4][4];
            #pragma unroll
            for (int r = 0; r < 4; ++r)
                #pragma unroll
                for (int q = 0; q < 4; ++q) acc[r][q] = 0.f;
            if (blk < nblocks) {
                const float* ya = Y + (size_t)4 * bi * lp + 4 * kg;
                const float* yb = Y + (size_t)4 * bj * lp + 4 * kg;
                for (int k = 0; k < nc; k += 4 * SMALL_KGROUPS) {
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
            #pragma unroll
            for (int r = 0; r < 4; ++r)
                #pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float v = acc[r][q];
                    #pragma unroll
                    for (int o = SMALL_KGROUPS / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    if (kg == r && blk < nblocks) {      // lane kg of the four writes row kg of the block and its mirror image
                        mine[(4 * bi + r) * sp + 4 * bj + q] = v;
                        mine[(4 * bj + q) * sp + 4 * bi + r] = v;
                    }
                }
        }
        // A = the sum of all blocks' shares
        if (n > 1) small_cluster_sync(); else __syncthreads();
        const uint32_t mine_addr = (uint32_t)__cvta_generic_to_shared(mine);
        for (int idx = tid; idx < s4 * nb; idx += SMALL_THREADS) {
            const int off = (idx / nb) * sp + 4 * (idx % nb);
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
            for (uint32_t r = 0; r < n; ++r) {
                uint32_t addr;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(mine_addr + 4u * off), "r"(r));
                const float4 v = ld_cluster4(addr);
                sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
            }
            *reinterpret_cast<float4*>(A + off) = sum;
        }
        __syncthreads();
        // B' = b A + c A A + a I
        for (int idx = tid; idx < s4 * nb; idx += SMALL_THREADS) {
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
        // Y <- B' Y: two threads own a column, each half of its rows; both hold the old column in registers
        constexpr int COLS = SMALL_THREADS / 2;
        const int row0 = (tid / COLS) * (nb + 1) / 2 * 4, row1 = tid / COLS ? s4 : (nb + 1) / 2 * 4;
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
                        if (k < s4) {
                            const float4 v = *reinterpret_cast<const float4*>(B + i * sp + k);
                            o[0] = fmaf(v.x, y[k], o[0]); o[1] = fmaf(v.y, y[k + 1], o[1]);
                            o[2] = fmaf(v.z, y[k + 2], o[2]); o[3] = fmaf(v.w, y[k + 3], o[3]);
                        }
                    }
                    Y[i * lp + q] = (o[0] + o[1]) + (o[2] + o[3]);
                }
            }
        }
        __syncthreads();
    }
    for (int idx = tid; idx < s * c_n; idx += SMALL_THREADS) {          // O = X_T, back in the input's orientation
        if (!tall) { const int r = idx / c_n, q = idx - r * c_n; Oz[(long long)r * cols + c_lo + q] = Y[r * lp + q]; }
        else       { const int q = idx / s, r = idx - q * s;     Oz[(long long)c_lo * cols + idx] = Y[r * lp + q]; }
    }
    if (n > 1) small_cluster_sync();      // no block leaves while another may still read its share
}

// Blocks per matrix: as many as leave each SMALL_MIN_COLS columns and all matrices together about one block per SM, and at
// least as many as the matrix needs to fit.
int small_ns_cluster(int s, int l, int batch) {
    int n = 1;
    while (n < SMALL_MAX_CLUSTER && (SmallLayout(s, l, n).bytes() > SMALL_MAX_SMEM || (l >= 2 * n * SMALL_MIN_COLS && 2 * n * batch <= 148))) n *= 2;
    return n;
}

}  // namespace

bool small_ns_eligible(long long rows, long long cols) {
    const long long s = rows < cols ? rows : cols, l = rows < cols ? cols : rows;
    return s <= 64 && l <= (1 << 16) && SmallLayout((int)s, (int)l, SMALL_MAX_CLUSTER).bytes() <= SMALL_MAX_SMEM;
}

cudaError_t small_ns_configure() {
    cudaError_t e = cudaFuncSetAttribute(small_ns_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_MAX_SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(small_ns_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_MAX_SMEM);
}

cudaError_t launch_small_ns(const float* M, float* O, const float* inv_norm, int batch, int rows, int cols, int T,
                            float a, float b, float c, cudaStream_t stream) {
    const int s = rows < cols ? rows : cols, l = rows < cols ? cols : rows;
    const int n = small_ns_cluster(s, l, batch);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(batch * n));
    cfg.blockDim = dim3(SMALL_THREADS);
    cfg.dynamicSmemBytes = SmallLayout(s, l, n).bytes();
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)n; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return s <= 32 ? cudaLaunchKernelEx(&cfg, small_ns_kernel<32>, M, O, inv_norm, rows, cols, T, a, b, c)
                   : cudaLaunchKernelEx(&cfg, small_ns_kernel<64>, M, O, inv_norm, rows, cols, T, a, b, c);
}

cudaError_t launch_sgemm(const SgemmArgs& g, cudaStream_t stream) {
    dim3 grid((g.N + TS - 1) / TS, (g.M + TS - 1) / TS, g.batch);
    sgemm_kernel<<<grid, 256, 0, stream>>>(g);
    return cudaGetLastError();
}

}  // namespace mona
