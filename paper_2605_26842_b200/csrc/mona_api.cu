// C ABI of the MONA step library: plan (shape buckets, chunking, state/workspace layout, TMA descriptors)
// and the per-step launch sequence.  See include/mona.h for the contract of every entry point.
#include <cuda.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <numeric>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/mona.h"
#include "common.cuh"
#include "elementwise.cuh"
#include "ns_fp32.cuh"
#include "ns_tc.cuh"

using namespace mona;

namespace {

// ---- workspace layout -------------------------------------------------------------------------------
// [status word | control blocks of the slots | iterates of slot 0 | 1 | 2 | 3]
// Consecutive large chunks alternate between slots 0 and 1 (and two streams), so that the last wave of each GEMM
// launch is filled by the other chunk's tiles and launch gaps of one chunk are covered by the other.  Small chunks, whose
// products have too few tiles for the machine, go to slots 2 and 3 beside them, or to all four when there is nothing else.
constexpr int NSLOTS = 4;
constexpr int BIG_SLOTS = 2;
constexpr size_t WS_STATUS_OFF = 0;
constexpr size_t WS_CTRL_OFF = 4096;                 // first control block
constexpr size_t WS_CTRL_BYTES = 1024 * 1024;        // per slot
constexpr size_t CTRL_COUNTERS_OFF = 0;
constexpr size_t CTRL_INVNORM_OFF = 4096;
constexpr size_t CTRL_PARTIALS_OFF = 8192;
constexpr size_t CTRL_SCHED_OFF = CTRL_PARTIALS_OFF + sizeof(float) * MAXC * MAX_UNITS;   // work counter + done counters of the NS kernel
constexpr size_t CTRL_PARAMS_OFF = (CTRL_SCHED_OFF + sizeof(unsigned int) * (64 + (size_t)MAXC * NS_MAX_PHASES) + 255) / 256 * 256;   // parameter pointers of the chunk
constexpr size_t WS_DATA_OFF = WS_CTRL_OFF + NSLOTS * WS_CTRL_BYTES;
static_assert(CTRL_PARAMS_OFF + sizeof(float*) * MAXC <= WS_CTRL_BYTES, "control block overflow");
static_assert(sizeof(unsigned int) * MAXC <= CTRL_INVNORM_OFF && sizeof(float) * MAXC <= CTRL_PARTIALS_OFF - CTRL_INVNORM_OFF, "control block overflow");

// Process-wide defaults behind mona_set_chunk_budget() / mona_set_chunk_overlap().  They only seed
// mona_default_options(); a handle keeps the options it was created with, so changing a default later
// never reaches an existing handle.
//   overlap: 1 = consecutive chunks are pipelined over two streams; 0 = everything on the caller's stream.
//   budget : bytes of bf16 iterates (X_t, X_{t+1}, A_t, B'_t) one chunk may hold.  Chunks are sized to keep every
//            SM pair busy, not for cache residency: chunks small enough to stay in L2 hold fewer tiles than the
//            device has CTA pairs.
constexpr size_t DEFAULT_CHUNK_BUDGET = 768ull << 20;
std::atomic<int> g_chunk_overlap{1};
std::atomic<size_t> g_chunk_budget_bytes{DEFAULT_CHUNK_BUDGET};

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// NVTX range over the host-side enqueue of a phase (shows up in timeline tools; costs nothing without one attached).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

struct MatRef {
    int desc;
    int64_t b;
};

struct Bucket {
    int64_t rows = 0, cols = 0, s = 0, l = 0, e = 0;
    int grad_dtype = 0, state_dtype = 0;
    bool tall = false, tc_ok = false;
    double chain_us = 0.0;      // rough time of a small bucket's step, for ordering and slots only
    int slot = 0;               // of a small bucket: where it always runs (large ones alternate between slots 0 and 1)
    bool small = false;         // its products do not fill the machine: runs beside other chunks (see bucket_is_small)
    bool paired = false;        // takes its first two iterations together on the s x s side (see ns_pair_pays)
    std::vector<MatRef> mats;
    // bytes from the state base of the three blocks: M (fp32), A and G_prev (fp32, or bf16 with MONA-Lite storage)
    size_t off_M = 0, off_A = 0, off_G = 0;
    int Cb = 1, Cf = 1;         // chunk capacity: bf16 tensor-core mode / fp32 mode
    int slabs = 1, up_slabs = 1;                // of the prologue; of the update and scale passes
    int64_t slab_len = 0, up_slab_len = 0;
    size_t off_x[2] = {0, 0}, off_a = 0, off_b = 0, off_delta = 0;   // bf16 mode, bytes from the slot's iterate base
    size_t off32_x[2] = {0, 0}, off32_a = 0, off32_b = 0;    // fp32 mode
    size_t data_bytes = 0;
    NsMaps maps[NSLOTS] = {};      // per workspace slot: X ping, X pong, A, B', C of a chunk of this bucket
};
constexpr int MAP_X0 = 0, MAP_A = 2, MAP_B = 3, MAP_C = 4;

// The first two iterations can be taken on the s x s side without forming the iterate between them:
//     A = X X^T, P = b A + c A^2 + a I, A' = P (P A), P' = b A' + c A'^2 + a I, Q = P' P, X'' = Q X
// (A, P and their products are polynomials in A: they commute and are symmetric, lower-triangle tiles all).  Against two plain
// iterations this saves one X X^T and one B' X and costs three s x s products.  It pays where that is clearly less tensor work
// (tile-k-slices of the pair against two plain iterations, one step before -> after: 1024 x 4096 0.68, 21.7 -> 20.1 ms; 768 x 2048
// 0.76, 20.2 -> 19.6 ms; 256 x 768 0.79, 3.87 -> 3.79 ms; but 512 x 1024 0.85, 4.05 -> 4.12 ms; 1024 x 1536 0.91, 6.93 -> 6.95 ms).
// By the shape alone: the pair rounds elsewhere than two plain iterations, and what a matrix gets must not depend on how many others
// of its shape there are.  On a few tiles, where the launch is bound by its chain of dependent products, the chain gets one longer
// (16 instead of 15) and its links shorter: one 256 x 768 97.9 -> 99.0 us per step, eight 107.7 -> 110.1, one 1024 x 2816 234 -> 236,
// 256 x 4096 171 -> 157, eight 1024 x 4096 716 -> 677, a block of 2048 and 8192 2498 -> 2250, sixteen of 1160 x 3096 and four of
// its square 2023 -> 1976.
bool ns_pair_pays(int64_t s, int64_t l) {
    const int64_t ts = (s + TC_BM - 1) / TC_BM, tl = (l + TC_BM - 1) / TC_BM, ks = (s + TC_BK - 1) / TC_BK, kl = (l + TC_BK - 1) / TC_BK;
    const int64_t sym = ts * (ts + 1) / 2;
    const int64_t plain = 2 * (sym * kl + sym * ks + ts * tl * ks), paired = sym * kl + 5 * sym * ks + ts * tl * ks;
    return paired * 100 <= plain * 80;
}
// The quintic of Eq. newton_schulz as the paper gives it.
constexpr double NS_A = 3.4445, NS_B = -4.7750, NS_C = 2.0315;
// Whether a run takes its first two iterations together: the paper's coefficients and at least four iterations only.  Rounding A
// to bf16 perturbs A' by up to a^2 |A| 2^-9 in the directions of small singular values, so only the first two are, where |A| is
// small (the iterate has Frobenius norm 1).  Relative error of O_5 against fp64 at 256 x 768 (bf16 emulation, mean of twelve
// draws; plain iterations -> every iteration apart with the diagonal correction -> first two together with it): Gaussian 0.0088 ->
// 0.0081 -> 0.0082, rows scaled over a factor of ten 0.0093 -> 0.0085 -> 0.0089, training-like 0.0091 -> 0.0085 -> 0.0084,
// condition number 100 0.0279 -> 0.0278 -> 0.0228; with all singular values equal, or all but one, it goes either way (0.0046 ->
// 0.0066, 0.0079 -> 0.0056).  Other coefficients can lose: (4.0848, -6.8946, 2.9270) 0.0304 -> 0.0301 -> 0.0457 on Gaussian and
// 0.0532 -> 0.0474 -> 0.0700 on scaled rows, (1.5, -0.5, 0) 0.0048 -> 0.0048 -> 0.0050; none but the paper's were found to be safe
// by a bound, so every other set iterates plainly.  With the last two together as well the ill-conditioned ones get worse
// (0.030), and for T < 4 an error of the first two has no iterations left to shrink in.
bool ns_first_two_together(bool pair_pays, const mona_hparams& hp) {
    return pair_pays && hp.ns_steps >= 4 && hp.ns_a == NS_A && hp.ns_b == NS_B && hp.ns_c == NS_C;
}

// A bucket whose symmetric products are at most four waves of tiles over the machine's 74 CTA pairs, and whose iterates are
// few enough to hold once more, does not get the machine to itself: a launch of it is a chain of dependent products with many
// pairs idle at the end of each, so such buckets run side by side on streams and SM pairs of their own.  Measured: buckets of four
// 1024 x 1024, two 2816 x 1024 and one 1024 x 2816 928 -> 372 us per step; sixteen, eight and four of 1160 and 3096 (240, 120 and 60
// tiles; with the line at two waves 2.03 ms) -> 1.75 ms; from five waves on (six tried) nothing changes.  Everything on the
// fp32 path that takes one block cluster per matrix is small too.  The line in bytes: with 64 MiB the set of 1160 and 3096 takes
// 2121 us instead of 1911 and a block of 2048 and 8192 2987 instead of 2250; with 400 instead of 200 nothing changes but the
// workspace (twelve blocks of 1024 and 2816, whose tall bucket has 360 MiB: 3470 us with 200, 3450 with 400, 952 and 1313 MiB).
constexpr size_t SMALL_BUCKET_BYTES = 200ull << 20;
bool bucket_is_small(int64_t s, int64_t e, int64_t count, bool tc_ok, bool one_cluster) {
    const int64_t tile = tc_ok ? TC_BM : 64, ts = (s + tile - 1) / tile;       // the fp32 GEMM: 64 x 64 tiles, one block per SM
    return (one_cluster || ts * (ts + 1) / 2 * count <= 4 * (tc_ok ? 74 : 148)) && (size_t)(2 * e + 2 * s * s) * (tc_ok ? 2 : 4) * count <= SMALL_BUCKET_BYTES;
}
// NARROW_ROUNDS: a launch on a share of the pairs looks at other tile widths for phases of at most this many rounds of items (with 1
// instead of 4 a dense block of 1024 and 2816 takes 407 us instead of 373, but one of 768 and 3072 254 instead of 276; the other sets
// tried are the same).  GATE_ROUNDS: the claim gate (NsProgram::gate) pays while a phase leaves pairs idle (mixed small set 151 ->
// 124 us) and costs a round trip per item where every pair has several (12 dense blocks, a bucket at 1.6 rounds: 1-2 %).
constexpr double NARROW_ROUNDS = 4.0, GATE_ROUNDS = 1.5;

struct Plan {
    std::vector<mona_matrix_desc> descs;
    std::vector<Bucket> buckets;
    // Buckets in the order in which a step takes them: small ones first, so that they run beside the first big prologue and the
    // large chunks (last, routers alone were a 400 us tail with the machine idle), the longest chain of them first.
    std::vector<int> order;
    std::vector<int> desc_bucket;          // bucket of descriptor i
    std::vector<int64_t> desc_pos;         // position of descriptor i's matrix 0 inside its bucket
    std::vector<int64_t> desc_first_gid;   // global matrix index (descriptor order) of matrix 0
    bool all_small = true;                 // no large bucket: small ones use all slots
    int n_slots = 1;                       // slots that hold something
    size_t state_bytes = 0, workspace_bytes = 0;
    size_t slot_off[NSLOTS] = {};          // bytes from the workspace base
};

mona_status build_plan(const mona_matrix_desc* descs, int64_t n_desc, size_t chunk_budget, Plan& plan, std::string& err) {
    if (!descs || n_desc <= 0) { err = "descs is null or n_desc <= 0"; return MONA_ERR_INVALID_ARG; }
    plan.descs.assign(descs, descs + n_desc);
    std::map<std::tuple<int64_t, int64_t, int, int>, int> index;
    int64_t gid = 0;
    for (int64_t i = 0; i < n_desc; ++i) {
        mona_matrix_desc& d = plan.descs[i];
        if (d.rows <= 0 || d.cols <= 0 || d.batch <= 0) { err = "descriptor with non-positive rows/cols/batch"; return MONA_ERR_INVALID_ARG; }
        if (d.grad_dtype != MONA_F32 && d.grad_dtype != MONA_BF16) { err = "descriptor with unknown grad_dtype"; return MONA_ERR_INVALID_ARG; }
        if (d.state_dtype != MONA_F32 && d.state_dtype != MONA_BF16 && d.state_dtype != MONA_STATE_COMBINED) { err = "descriptor with unknown state_dtype"; return MONA_ERR_INVALID_ARG; }
        if (d.rows > (1 << 20) || d.cols > (1 << 20) || d.rows * d.cols > (1ll << 31)) { err = "matrix too large"; return MONA_ERR_UNSUPPORTED_SHAPE; }
        if (d.batch_stride == 0) d.batch_stride = d.rows * d.cols;
        if (d.batch_stride < d.rows * d.cols) { err = "batch_stride smaller than rows*cols"; return MONA_ERR_INVALID_ARG; }
        auto key = std::make_tuple(d.rows, d.cols, (int)d.grad_dtype, (int)d.state_dtype);
        auto it = index.find(key);
        int bi;
        if (it == index.end()) {
            bi = (int)plan.buckets.size();
            index[key] = bi;
            Bucket b;
            b.rows = d.rows; b.cols = d.cols; b.grad_dtype = d.grad_dtype; b.state_dtype = d.state_dtype;
            b.tall = d.rows > d.cols;
            b.s = std::min(d.rows, d.cols); b.l = std::max(d.rows, d.cols); b.e = d.rows * d.cols;
            // below 64 rows bf16 iterates of very wide matrices drift past the 2e-2 bound (measured 2.0-2.4e-2 at 32 x 1024),
            // so such matrices keep the fp32 path
            b.tc_ok = (b.s % 8 == 0) && (b.l % 8 == 0) && b.s >= 64;
            plan.buckets.push_back(b);
        } else {
            bi = it->second;
        }
        plan.desc_bucket.push_back(bi);
        plan.desc_pos.push_back((int64_t)plan.buckets[bi].mats.size());
        plan.desc_first_gid.push_back(gid);
        for (int64_t b = 0; b < d.batch; ++b) plan.buckets[bi].mats.push_back({(int)i, b});
        gid += d.batch;
    }
    size_t state_bytes = 0;
    for (Bucket& b : plan.buckets) {
        const int64_t count = (int64_t)b.mats.size();
        const size_t aux = b.state_dtype == MONA_BF16 ? 2 : 4;              // every block starts 256-byte aligned
        b.off_M = state_bytes; state_bytes += align_up((size_t)count * b.e * 4, 256);
        b.off_A = state_bytes; state_bytes += align_up((size_t)count * b.e * aux, 256);
        b.off_G = state_bytes;                                              // the single-buffer form has no G_prev block
        if (b.state_dtype != MONA_STATE_COMBINED) state_bytes += align_up((size_t)count * b.e * aux, 256);
        // chunk capacity
        const size_t per_mat_bf16 = (size_t)(2 * b.e + 2 * b.s * b.s) * 2;
        int64_t cb = (int64_t)(chunk_budget / per_mat_bf16);
        cb = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(cb, MAXC), count));
        b.Cb = (int)cb;
        // fp32 iterates take twice the bytes.  A bucket that has no other path gets whole chunks; in validation mode one that
        // also has the bf16 path must not make a large workspace larger than that path needs.
        const int64_t cf = b.tc_ok && per_mat_bf16 * cb > (32u << 20) ? cb / 2 : std::min<int64_t>(cb, (int64_t)(chunk_budget / (2 * per_mat_bf16)));
        b.Cf = (int)std::max<int64_t>(1, cf);
        long long slab = 0;
        slab_plan(b.e, cb, norm_unit(b.e), &slab, &b.slabs);
        b.slab_len = slab;
        slab_plan(b.e, cb, UPDATE_UNIT, &slab, &b.up_slabs);
        b.up_slab_len = slab;
        b.paired = b.tc_ok && ns_pair_pays(b.s, b.l);
        size_t off = 0;
        for (int i = 0; i < 2; ++i) { b.off_x[i] = off; off += align_up((size_t)b.Cb * b.e * 2, 1024); }
        b.off_a = off; off += align_up((size_t)b.Cb * b.s * b.s * 2, 1024);
        b.off_b = off; off += align_up((size_t)b.Cb * b.s * b.s * 2, 1024);
        b.off_delta = off; off += align_up((size_t)b.Cb * b.s * sizeof(float), 1024);
        size_t off32 = 0;
        for (int i = 0; i < 2; ++i) { b.off32_x[i] = off32; off32 += align_up((size_t)b.Cf * b.e * 4, 1024); }
        b.off32_a = off32; off32 += align_up((size_t)b.Cf * b.s * b.s * 4, 1024);
        b.off32_b = off32; off32 += align_up((size_t)b.Cf * b.s * b.s * 4, 1024);
        b.data_bytes = std::max(off, off32);
        b.small = bucket_is_small(b.s, b.e, count, b.tc_ok, !b.tc_ok && small_ns_eligible(b.rows, b.cols)) && (b.tc_ok ? b.Cb : b.Cf) == count;
        {   // a five-step chain: about 100 us on the tensor cores, 25 in one block cluster, three products per iteration in fp32
            const double ts = (double)((b.s + 63) / 64), tl = (double)((b.l + 63) / 64), waves = (double)count / 148.0;
            const double product = std::max(1.0, ts * (ts + 1) / 2 * waves) * (double)(b.l + b.s) / 32 + std::max(1.0, ts * tl * waves) * (double)b.s / 32;
            b.chain_us = b.tc_ok ? 100.0 : small_ns_eligible(b.rows, b.cols) ? 25.0 : 5.0 * (1.2 * product + 20.0);
        }
    }
    for (int i = 0; i < (int)plan.buckets.size(); ++i) plan.order.push_back(i);
    plan.state_bytes = state_bytes;
    // Every small bucket gets the slot with the least in it so far, and a slot is as large as the largest bucket it ever holds.  All
    // slots together hold no more than two chunks (of the budget, or of the largest matrix) and an eighth of that: where they
    // would, the largest small bucket runs as a large one, until they do.  The eighth is for sets whose large buckets fill two
    // chunks: four layers of 512 x 1024 experts with their sixteen 1024 x 1024 beside them 3.79 ms per step, behind them 3.83, with
    // chunks shortened by as much 3 % more.
    size_t slot_bytes[NSLOTS], limit = chunk_budget;
    for (const Bucket& b : plan.buckets) limit = std::max(limit, b.data_bytes);
    limit = 2 * limit + limit / 4;
    while (true) {
        plan.all_small = std::all_of(plan.buckets.begin(), plan.buckets.end(), [](const Bucket& b) { return b.small; });
        std::stable_sort(plan.order.begin(), plan.order.end(), [&](int x, int y) {
            const Bucket &a = plan.buckets[x], &b = plan.buckets[y];
            return a.small != b.small ? a.small : a.small && a.chain_us > b.chain_us;
        });
        double slot_load[NSLOTS] = {};
        const int first_small = plan.all_small ? 0 : BIG_SLOTS;
        Bucket* largest = nullptr;
        std::fill_n(slot_bytes, NSLOTS, (size_t)0);
        for (int i : plan.order) {
            Bucket& b = plan.buckets[i];
            if (!b.small) {
                for (int sl = 0; sl < BIG_SLOTS; ++sl) slot_bytes[sl] = std::max(slot_bytes[sl], b.data_bytes);
                continue;
            }
            b.slot = first_small;
            for (int sl = first_small; sl < NSLOTS; ++sl) if (slot_load[sl] < slot_load[b.slot]) b.slot = sl;
            slot_load[b.slot] += b.chain_us;
            slot_bytes[b.slot] = std::max(slot_bytes[b.slot], b.data_bytes);
            if (!largest || b.data_bytes > largest->data_bytes) largest = &b;
        }
        if (!largest || std::accumulate(slot_bytes, slot_bytes + NSLOTS, (size_t)0) <= limit) break;
        largest->small = false;
    }
    plan.workspace_bytes = WS_DATA_OFF;
    for (int sl = 0; sl < NSLOTS; ++sl) {
        plan.slot_off[sl] = plan.workspace_bytes;
        plan.workspace_bytes += align_up(slot_bytes[sl], 1024);
        if (slot_bytes[sl]) plan.n_slots = sl + 1;
    }
    return MONA_OK;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// bf16 tensor [C][outer][inner] (inner contiguous, matrices `mat_stride` elements apart) cut into boxes of 64 x box_rows with the
// 128-byte swizzle.
bool encode_map(EncodeTiledFn fn, CUtensorMap* map, void* base, int64_t inner, int64_t outer, int64_t C, int box_rows, int64_t mat_stride) {
    cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)outer, (cuuint64_t)C};
    cuuint64_t strides[2] = {(cuuint64_t)inner * 2, (cuuint64_t)mat_stride * 2};
    cuuint32_t box[3] = {(cuuint32_t)TC_BOX, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

F2 split(double v) {
    F2 r;
    r.hi = (float)v;
    r.lo = (float)(v - (double)r.hi);
    return r;
}

}  // namespace

struct mona_handle {
    Plan plan;
    mona_options opt = {};      // as resolved at creation; later changes of the process-wide defaults do not reach the handle
    int device = 0, max_pairs = 0;
    std::vector<int> pairs_beside;   // per bucket: SM pairs of a small one beside others
    uint8_t* state = nullptr;
    uint8_t* ws = nullptr;
    cudaStream_t side[NSLOTS] = {};        // stream of slot 1 .. NSLOTS - 1 (slot 0 uses the caller's)
    cudaEvent_t ev_fork = nullptr, ev_join[NSLOTS] = {};
    // host-to-host pipeline of mona_step_host(): copy streams and per-chunk events, created on first use
    cudaStream_t h2d = nullptr, d2h = nullptr;
    cudaEvent_t ev_hfork = nullptr, ev_hjoin = nullptr;
    std::vector<cudaEvent_t> ev_in;     // the gradients of chunk i have arrived on the device
    std::vector<cudaEvent_t> ev_out;    // chunk i has been updated
    DeviceStatus* host_status = nullptr;   // pinned
    std::string last_error;
    int64_t launches = 0;
    double flops_exec = 0.0, flops_dense = 0.0, flops_useful = 0.0;

    mona_status fail(mona_status st, const char* fmt, ...) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        last_error = buf;
        return st;
    }
};

static std::vector<int> share_pairs(const Plan& plan, int max_pairs);

#define MONA_CUDA(h, call)                                                                                 \
    do {                                                                                                   \
        cudaError_t e_ = (call);                                                                           \
        if (e_ != cudaSuccess) return (h)->fail(MONA_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

extern "C" {

mona_status mona_default_hparams(mona_hparams* hp) {
    if (!hp) return MONA_ERR_INVALID_ARG;
    memset(hp, 0, sizeof *hp);
    hp->lr = 1e-3; hp->momentum = 0.95; hp->accel_beta = 0.99; hp->accel_alpha = -1.0 / (2.0 * (1.0 - 0.99));
    hp->weight_decay = 0.1; hp->ns_a = NS_A; hp->ns_b = NS_B; hp->ns_c = NS_C; hp->norm_eps = 1e-7;
    hp->scale_value = 0.2; hp->ns_steps = 5; hp->scale_mode = 0; hp->ns_precision = 0;
    return MONA_OK;
}

mona_status mona_set_chunk_budget(size_t bytes) {
    if (bytes < (1u << 20)) return MONA_ERR_INVALID_ARG;
    g_chunk_budget_bytes.store(bytes);
    return MONA_OK;
}

mona_status mona_set_chunk_overlap(int enabled) {
    g_chunk_overlap.store(enabled ? 1 : 0);
    return MONA_OK;
}

mona_status mona_default_options(mona_options* opt) {
    if (!opt) return MONA_ERR_INVALID_ARG;
    memset(opt, 0, sizeof *opt);
    opt->chunk_budget_bytes = g_chunk_budget_bytes.load();
    opt->chunk_overlap = g_chunk_overlap.load();
    opt->fuse_update = 0;
    opt->ns_delay = 20;
    opt->macro_tile_min_k = 1;
    return MONA_OK;
}

}  // extern "C"

namespace {
// Options as the plan uses them: NULL means the defaults; a zero budget or delay means the default value.
mona_status resolve_options(const mona_options* in, mona_options& out) {
    mona_default_options(&out);
    if (!in) return MONA_OK;
    if (in->chunk_budget_bytes != 0) {
        if (in->chunk_budget_bytes < (1u << 20)) return MONA_ERR_INVALID_ARG;
        out.chunk_budget_bytes = in->chunk_budget_bytes;
    }
    out.chunk_overlap = in->chunk_overlap ? 1 : 0;
    out.fuse_update = in->fuse_update ? 1 : 0;
    if (in->ns_delay < 0 || in->ns_delay > 1024) return MONA_ERR_INVALID_ARG;
    if (in->ns_delay > 0) out.ns_delay = in->ns_delay;
    if (in->macro_tile_min_k < 0) return MONA_ERR_INVALID_ARG;
    if (in->macro_tile_min_k > 0) out.macro_tile_min_k = in->macro_tile_min_k;
    return MONA_OK;
}
}  // namespace

extern "C" {

mona_status mona_query_sizes_opt(const mona_matrix_desc* descs, int64_t n_desc, const mona_options* options,
                                 size_t* state_bytes, size_t* workspace_bytes) {
    mona_options opt;
    if (resolve_options(options, opt) != MONA_OK) return MONA_ERR_INVALID_ARG;
    Plan plan;
    std::string err;
    mona_status st = build_plan(descs, n_desc, opt.chunk_budget_bytes, plan, err);
    if (st != MONA_OK) return st;
    if (state_bytes) *state_bytes = plan.state_bytes;
    if (workspace_bytes) *workspace_bytes = plan.workspace_bytes;
    return MONA_OK;
}

mona_status mona_query_sizes(const mona_matrix_desc* descs, int64_t n_desc, size_t* state_bytes, size_t* workspace_bytes) {
    return mona_query_sizes_opt(descs, n_desc, nullptr, state_bytes, workspace_bytes);
}

mona_status mona_create(mona_handle** out, const mona_matrix_desc* descs, int64_t n_desc, void* state, size_t state_bytes,
                        void* workspace, size_t workspace_bytes, int device) {
    return mona_create_opt(out, descs, n_desc, nullptr, state, state_bytes, workspace, workspace_bytes, device);
}

mona_status mona_create_opt(mona_handle** out, const mona_matrix_desc* descs, int64_t n_desc, const mona_options* options,
                            void* state, size_t state_bytes, void* workspace, size_t workspace_bytes, int device) {
    if (!out) return MONA_ERR_INVALID_ARG;
    *out = nullptr;
    mona_handle* h = new mona_handle();
    *out = h;     // returned even on failure so that mona_last_error() can be read; destroy it either way
    if (resolve_options(options, h->opt) != MONA_OK)
        return h->fail(MONA_ERR_INVALID_ARG, "options: chunk_budget_bytes must be 0 or at least 1 MiB, ns_delay within 0..1024");
    mona_status st = build_plan(descs, n_desc, h->opt.chunk_budget_bytes, h->plan, h->last_error);
    if (st != MONA_OK) return st;
    if (!state || !workspace) return h->fail(MONA_ERR_INVALID_ARG, "state or workspace is null");
    if (((uintptr_t)state & 255) || ((uintptr_t)workspace & 255)) return h->fail(MONA_ERR_ALIGNMENT, "state/workspace must be 256-byte aligned");
    if (state_bytes < h->plan.state_bytes || workspace_bytes < h->plan.workspace_bytes)
        return h->fail(MONA_ERR_BUFFER_TOO_SMALL, "need state %zu B, workspace %zu B", h->plan.state_bytes, h->plan.workspace_bytes);
    int ndev = 0;
    cudaError_t ce = cudaGetDeviceCount(&ndev);
    if (ce != cudaSuccess || device < 0 || device >= ndev)
        return h->fail(MONA_ERR_CUDA, "no usable CUDA device %d (%s)", device, cudaGetErrorString(ce));
    MONA_CUDA(h, cudaSetDevice(device));
    cudaDeviceProp prop;
    MONA_CUDA(h, cudaGetDeviceProperties(&prop, device));
    if (prop.major != 10) return h->fail(MONA_ERR_ARCH, "device %d is sm_%d%d; this library is built for sm_100a only", device, prop.major, prop.minor);
    h->device = device;
    h->state = (uint8_t*)state;
    h->ws = (uint8_t*)workspace;

    EncodeTiledFn encode = nullptr;
    cudaDriverEntryPointQueryResult qres;
    MONA_CUDA(h, cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", (void**)&encode, cudaEnableDefault, &qres));
    if (!encode || qres != cudaDriverEntryPointSuccess) return h->fail(MONA_ERR_CUDA, "cuTensorMapEncodeTiled not available");
    for (Bucket& b : h->plan.buckets) {
        if (!b.tc_ok) continue;
        bool ok = true;
        for (int sl = 0; sl < NSLOTS; ++sl) {
            if (b.small ? sl != b.slot : sl >= BIG_SLOTS) continue;
            uint8_t* data = h->ws + h->plan.slot_off[sl];
            for (int big = 0; big < 2; ++big) {     // 64-row boxes, then 128-row boxes
                const int rows = big ? 2 * TC_BOX : TC_BOX, at = big * NS_TENSORS;
                for (int i = 0; i < 2; ++i) ok = ok && encode_map(encode, &b.maps[sl].m[at + MAP_X0 + i], data + b.off_x[i], b.cols, b.rows, b.Cb, rows, b.e);
                ok = ok && encode_map(encode, &b.maps[sl].m[at + MAP_A], data + b.off_a, b.s, b.s, b.Cb, rows, b.s * b.s);
                ok = ok && encode_map(encode, &b.maps[sl].m[at + MAP_B], data + b.off_b, b.s, b.s, b.Cb, rows, b.s * b.s);
                // C of a matrix lives in the second iterate of the SAME matrix, which nothing holds until the first pair's Q X is
                // stored there - after the last read of C, by the order of the matrix's own phases
                ok = ok && encode_map(encode, &b.maps[sl].m[at + MAP_C], data + b.off_x[1], b.s, b.s, b.Cb, rows, b.e);
            }
        }
        if (!ok) return h->fail(MONA_ERR_CUDA, "cuTensorMapEncodeTiled failed for bucket %lldx%lld", (long long)b.rows, (long long)b.cols);
    }
    MONA_CUDA(h, ns_configure(&h->max_pairs));
    h->pairs_beside = share_pairs(h->plan, h->max_pairs);
    MONA_CUDA(h, small_ns_configure());
    MONA_CUDA(h, sgemm_configure());
    MONA_CUDA(h, cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
    for (int sl = 1; sl < h->plan.n_slots; ++sl) {
        MONA_CUDA(h, cudaStreamCreateWithFlags(&h->side[sl], cudaStreamNonBlocking));
        MONA_CUDA(h, cudaEventCreateWithFlags(&h->ev_join[sl], cudaEventDisableTiming));
    }
    MONA_CUDA(h, cudaMallocHost((void**)&h->host_status, sizeof(DeviceStatus)));
    // M_0 = A_0 = G_0 = 0; control block cleared
    MONA_CUDA(h, cudaMemset(h->state, 0, h->plan.state_bytes));
    MONA_CUDA(h, cudaMemset(h->ws, 0, WS_DATA_OFF));
    DeviceStatus init = {0u, INT_MAX, 0u, 0u};
    MONA_CUDA(h, cudaMemcpy(h->ws + WS_STATUS_OFF, &init, sizeof init, cudaMemcpyHostToDevice));
    MONA_CUDA(h, cudaDeviceSynchronize());
    return MONA_OK;
}

}  // extern "C"

// Appends to `g` the phases of one iteration (or of two taken together) of a chunk of bucket `b`.  X is read from tensor
// MAP_X0 + x_cur and written to the other one, or over itself with `in_place`; `first`: X is still un-normalised.
static void ns_plan_group(NsProgram& g, const Bucket& b, bool together, bool first, int x_cur, uint8_t* data, float* delta,
                          float ns_a, float ns_b, float ns_c, int macro_tile_min_k, bool fuse_update, bool update, bool in_place) {
    const int s = (int)b.s, l = (int)b.l;
    const size_t offset[NS_TENSORS] = {b.off_x[0], b.off_x[1], b.off_a, b.off_b, b.off_x[1]};
    auto output = [&](NsPhase& p, int d_map, int64_t ld) {
        p.d_map = d_map; p.d = (__nv_bfloat16*)(data + offset[d_map]); p.ld = ld;
        p.mat_stride = d_map == MAP_A || d_map == MAP_B ? (int64_t)s * s : b.e;
    };
    // D = product of two symmetric s x s matrices, operands and result lower-block-stored
    auto small = [&](int a_map, int b_map, int d_map) -> NsPhase& {
        NsPhase& p = g.ph[g.P++];
        p.M = p.N = p.K = s; p.a_map = a_map; p.b_map = b_map; p.a_sym = p.b_sym = 1; p.symmetric = p.small_sym = 1; p.ab_same = a_map == b_map;
        output(p, d_map, s); p.c2 = 1.f;
        ns_phase_plan(p);
        return p;
    };
    // D = b A + c A A + a I
    auto poly = [&](int d_map) {
        NsPhase& p = small(MAP_A, MAP_A, d_map);
        p.cin = (const __nv_bfloat16*)(data + b.off_a); p.cin_stride = (long long)s * s; p.c1 = ns_b; p.c2 = ns_c; p.diag_add = ns_a; p.delta_in = delta;
    };
    NsPhase& g1 = g.ph[g.P++];      // A = X X^T (wide) or X^T X (tall): lower-triangle tiles only
    g1.M = g1.N = s; g1.K = l; g1.a_map = g1.b_map = MAP_X0 + x_cur; g1.a_mn = g1.b_mn = b.tall ? 1 : 0;
    g1.symmetric = 1; g1.ab_same = 1; output(g1, MAP_A, s);
    g1.c2 = 1.f; g1.post_mode = first ? 2 : 0; g1.delta_out = delta;
    ns_phase_plan(g1);
    poly(MAP_B);                                        // P
    if (together) {
        small(MAP_B, MAP_A, MAP_C);                     // P A
        small(MAP_B, MAP_C, MAP_A).delta_out = delta;   // A' = P (P A)
        poly(MAP_C);                                    // P'
        small(MAP_C, MAP_B, MAP_A);                     // Q = P' P
    }
    const int q_map = together ? MAP_A : MAP_B;
    NsPhase& g3 = g.ph[g.P++];      // X' = Q X (wide) or X Q (tall); 256 x 512 macro-tiles when the inner dimension is long
    g3.K = s; g3.wide = s >= macro_tile_min_k ? 1 : 0; output(g3, MAP_X0 + (in_place ? x_cur : x_cur ^ 1), b.cols);
    g3.c2 = 1.f; g3.post_mode = first ? 1 : 0; g3.fuse_update = fuse_update ? 1 : 0; g3.update = update ? 1 : 0;
    if (!b.tall) {   // Q is the symmetric "A" operand, X the MN-major "B" operand
        g3.M = s; g3.N = l; g3.a_map = q_map; g3.a_sym = 1; g3.b_map = MAP_X0 + x_cur; g3.b_mn = 1;
    } else {         // X is K-major, the symmetric Q serves as its own transpose
        g3.M = l; g3.N = s; g3.a_map = MAP_X0 + x_cur; g3.a_mn = 0; g3.b_map = q_map; g3.b_sym = 1;
    }
    if (fuse_update || update) g3.d = nullptr;
    ns_phase_plan(g3);
}

// Tile work of a bucket's iteration, in k-slices of 256 x 256 tiles.
static double bucket_work(const Bucket& b) {
    const double ts = (double)((b.s + TC_BM - 1) / TC_BM), tl = (double)((b.l + TC_BM - 1) / TC_BM);
    const double ks = (double)((b.s + TC_BK - 1) / TC_BK), kl = (double)((b.l + TC_BK - 1) / TC_BK);
    return (double)b.mats.size() * (ts * (ts + 1) / 2 * (kl + ks) + ts * tl * ks);
}
// SM pairs of every bucket's launches when they run beside others: its share of the work when only small buckets run; beside large ones
// four times that, and eight at least, so that it is through long before they are.  (Pairs that a launch does not find free
// simply come later: items are handed out to whichever pairs run.)  Twelve blocks of 1024 and 2816: 3433 us per step, 3599 with
// the share alone, 3472 with all pairs; four layers of 512 x 1024 experts the same with all three; a drawn set of experts 2571, 2421 and 2630.
static std::vector<int> share_pairs(const Plan& plan, int max_pairs) {
    double work_total = 0.0;
    for (const Bucket& b : plan.buckets) if (b.tc_ok) work_total += bucket_work(b);
    std::vector<int> pairs;
    for (const Bucket& b : plan.buckets) {
        const double share = b.tc_ok ? max_pairs * bucket_work(b) / work_total : 0.0;
        pairs.push_back(std::max(1, std::min(max_pairs, (int)(plan.all_small ? share + 0.5 : std::max(8.0, 4.0 * share)))));
    }
    // Where only small buckets run, what can run at once fits the device.  Launches are placed as they come, some before their prologue
    // has ended: with shares rounded up beyond the device, one of five 2048 x 2048 took all pairs and a chain of 13 of 128 x 128 with
    // a share of one began when it was through (1040 instead of 880 us per step).
    while (plan.all_small) {
        int widest[NSLOTS] = {}, of_slot[NSLOTS] = {}, total = 0, most = 0;
        for (int i = 0; i < (int)pairs.size(); ++i) {
            const Bucket& b = plan.buckets[i];
            if (b.tc_ok && pairs[i] > widest[b.slot]) { widest[b.slot] = pairs[i]; of_slot[b.slot] = i; }
        }
        for (int sl = 0; sl < NSLOTS; ++sl) { total += widest[sl]; if (widest[sl] > widest[most]) most = sl; }
        if (total <= max_pairs || widest[most] <= 1) break;
        --pairs[of_slot[most]];
    }
    return pairs;
}
// Whether a launch over C matrices deals them whole to its SM pairs (NsForm::Whole) or spreads every product over the pairs.  Only where the
// shorter side is one tile.  Time per step, whole against spread, us, on 74 pairs unless said otherwise:
//  - one round, two matrices per pair at most: one-tile matrices (l <= 256) from nine on, 8 of 256 x 256 92 against 90, 12 93 against 101,
//    74 121-133 against 172, 148 183 against 230 (up to 128 x 128 from eight, 8 of 64 x 64 60 against 74); up to l = 512 once every pair
//    has one, 74 of 256 x 512 176-197 against 219; up to l = 1024 with one and a half, 90 of 256 x 768 296 against 287, 111 326 against 339,
//    148 406 against 439, 148 of 1024 x 256 505 against 530; beyond that not, 111 of 256 x 1280 490 against 483, 148 656 against 640,
//    74 of 192 x 2048 434 against 415;
//  - more: a last round without second matrices counts half, a full one leaves a ragged end, and spread over all pairs as many matrices
//    take 1.1 times a full round's share: 185, 222, 296, 370 and 512 of 256 x 768 550, 624, 861, 990 and 1377 against 532, 643, 820, 1037
//    and 1425, of 256 x 256 277, 291, 418, 468 and 640 against 271, 312, 412, 500 and 690.  Not where one CTA of the pair has no rows
//    and l > 512: 512 of 96 x 1024 950 against 917.  Always up to 128 x 128: 160, 300 and 512 167, 269 and 386 against 169, 284 and 446;
//  - on a share of the pairs the iterates stay in L2 either way and spreading is quicker as soon as a pair needs a second matrix: 40 of 256 x
//    256 on 32, 16 and 8 pairs 125, 206 and 313 against 162, 160 and 275; 42 beside two small buckets 187 against 162.  Longer ones never:
//    40 of 1088 x 256 on 32 pairs 307 against 264.
static bool whole_matrices(const Bucket& b, int C, int pairs, bool shared) {
    const bool tiny = b.l <= TC_BN / 2, one_tile = b.l <= TC_BN;
    if (b.s > TC_BM || C < (tiny ? 8 : 9)) return false;
    if (shared) return one_tile && C <= pairs;
    if (tiny) return true;
    if (C <= 2 * pairs) return one_tile || (b.l <= 2 * TC_BN ? C >= pairs : b.l <= 4 * TC_BN && 2 * C >= 3 * pairs);
    if (b.l > (b.s > TC_BM / 2 ? 3 : 2) * TC_BN) return false;
    const int rest = C % (2 * pairs);
    return C / (2 * pairs) + (rest == 0 ? 0.2 : rest <= pairs ? 0.5 : 1.0) < 1.1 * C / (2.0 * pairs);
}
// Whether the last X' = B' X updates the parameters, or a pass of its own does: by estimated time.  Inside it lengthens the epilogue of every
// 256 x 256 tile by some 3.5 us (8 x 64 KiB of parameters in and out of a pair), of half a tile's columns by half of that, however few
// rows it has, and only the pairs of the launch work at it; apart it is a launch, 6 us, and 10 bytes per element at the bandwidth of the whole device.  One bucket on
// 1, 8, 16 and 32 pairs, inside against apart, us per step: 40 of 256 x 256 2012 / 275 / 160 / 162 against 1868 / 262 / 158 / 165, 24 of
// 512 x 512 4248 / 592 / 332 / 226 against 3928 / 567 / 325 / 227, 13 of 128 x 128 on 8 and 32 94 / 93 against 97 / 96; on all 74, 300 of
// 72 x 648 439 against 428, but of 648 x 72 430 against 447.
static bool update_pays_inside(const Bucket& b, int C, int pairs) {
    const double tiles = 0.5 * (double)C * (double)((b.rows + TC_BM - 1) / TC_BM) * (double)((b.cols + TC_BN / 2 - 1) / (TC_BN / 2));
    return 3.5 * std::max(1.0, tiles / pairs) <= 6.0 + (double)C * (double)b.e * 10.0 / 6.2e6;
}
// The product that updates the parameters takes plain tiles where it has at least two rounds of macro-tiles.  Its epilogue is the
// longest, 8 bytes per element in and out of the SM: behind a macro-tile nothing hides it, with plain tiles the next one's
// products run beside it (12 dense blocks 3480 -> 3414 us per step, 1024 x 1536 experts 6778 -> 6650, three layers of 768 x 2048
// 18.78 -> 18.48 ms; 512 x 1024 and 256 x 768 experts within the noise).  With fewer rounds it goes either way, by how well the last round fills:
// rounds of macro-tiles and us with macro-tiles -> plain ones, 0.9: 8 of 1024 x 1024 260 -> 268, 2 of 2048 x 2048 388 -> 427; 1.5: 9 of
// 768 x 2048 311 -> 322; 1.7: 4 of 1024 x 4096 424 -> 414, 16 of 1024 x 1024 460 -> 453, 4 of 2048 x 2048 702 -> 690; 2.2: 5 of 2048 x 2048
// 874 -> 869; 2.6: 24 of 768 x 2048 708 -> 690.
static void ns_plain_update_tiles(NsProgram& g, int pairs) {
    for (int q = 0; q < g.P; ++q) {
        NsPhase& p = g.ph[q];
        if (p.update && p.wide && (long long)g.C * p.items_per_mat >= 2ll * pairs) { p.wide = 0; ns_phase_plan(p); }
    }
}
// Fits a launch to `pairs` SM pairs: tile widths by estimated time, the claim gate, no more pairs than a phase has items.
// (`shared`: beside other launches on a part of the pairs.)  A launch that has all pairs looks at other tile widths only for phases
// that do not fill them once; macro-tiles move the fewest bytes per flop.
static void ns_fit_launch(NsProgram& g, int pairs, bool shared) {
    int most = 0;
    bool fused = false;
    for (int q = 0; q < g.P; ++q) fused = fused || g.ph[q].fuse_update;
    for (int q = 0; q < g.P; ++q) {
        NsPhase& p = g.ph[q];
        NsPhase best = p;
        double best_cycles = ns_phase_cycles(p, std::ceil((double)g.C * p.items_per_mat / pairs));
        if (!fused && (double)g.C * p.items_per_mat <= (shared ? NARROW_ROUNDS : 1.0) * pairs) {
            for (int narrow = 0; narrow < 2; ++narrow) {
                NsPhase alt = p;
                alt.wide = 0; alt.narrow = narrow;
                ns_phase_plan(alt);
                const double cycles = ns_phase_cycles(alt, std::ceil((double)g.C * alt.items_per_mat / pairs));
                if (cycles < best_cycles) { best_cycles = cycles; best = alt; }
            }
        }
        p = best;
        most = std::max(most, p.items_per_mat * g.C);
    }
    g.gate = !fused && most < GATE_ROUNDS * pairs ? 1 : 0;
    if (g.gate) g.form = NsForm::Few;
    for (int q = 0; q < g.P; ++q) if (g.ph[q].narrow) g.form = NsForm::Few;
    g.max_pairs = std::min(pairs, most);
}

// How the launches of a chunk on the tensor-core path are made: what a step, the self-test and mona_describe_step() go by.
struct NsChoice {
    int pairs;              // SM pairs the launches may use
    bool shared;            // beside other chunks, on a share of the pairs
    bool whole;             // NsForm::Whole
    bool together;          // the first two iterations on the s x s side
    bool update_inside;     // the last X' = B' X updates the parameters
    int groups;             // iterations, the first two counted as one when taken together
};
static NsChoice ns_choose(const mona_options& opt, int max_pairs, int pairs_beside, const Bucket& b, int C, bool beside, bool may_update, const mona_hparams& hp) {
    NsChoice k;
    k.shared = beside;
    k.pairs = beside ? pairs_beside : max_pairs;
    k.whole = !opt.fuse_update && whole_matrices(b, C, k.pairs, beside);
    k.together = ns_first_two_together(b.paired, hp);
    k.groups = k.together ? hp.ns_steps - 1 : hp.ns_steps;
    k.update_inside = may_update && !opt.fuse_update && update_pays_inside(b, C, k.pairs);
    return k;
}
// The next launch of a chunk: the phases of group `gi` and of as many after it as one launch holds; moves `gi` behind them.
static NsProgram ns_next_launch(const mona_options& opt, const Bucket& b, int C, const NsChoice& k, const mona_hparams& hp, bool update_fused, uint8_t* data, int& gi) {
    NsProgram g{};
    g.C = C; g.delay = std::min(opt.ns_delay, C);       // beyond C matrices the order is the same
    for (; gi < k.groups && g.P + (gi == 0 && k.together ? 7 : 3) <= NS_MAX_PHASES; ++gi) {
        const bool last = gi + 1 == k.groups;
        ns_plan_group(g, b, gi == 0 && k.together, gi == 0, k.whole ? 0 : gi & 1, data, (float*)(data + b.off_delta), (float)hp.ns_a, (float)hp.ns_b,
                      (float)hp.ns_c, opt.macro_tile_min_k, update_fused && last, k.update_inside && last, k.whole);
    }
    ns_plain_update_tiles(g, k.pairs);
    if (k.whole) { g.form = NsForm::Whole; g.max_pairs = k.pairs; g.lane_tensors = C >= 2 * k.pairs; }
    else ns_fit_launch(g, k.pairs, k.shared);
    ns_program_plan(g);
    return g;
}

// Matrices per chunk of a step (`host_bytes`: the bytes of parameters a chunk may hold in mona_step_host(), else 0).
static int chunk_capacity(const Bucket& b, const mona_hparams& hp, size_t host_bytes) {
    const int cap = hp.ns_precision == 0 && b.tc_ok && hp.ns_steps >= 1 ? b.Cb : b.Cf;
    return host_bytes ? (int)std::min<size_t>(cap, std::max<size_t>(1, host_bytes / ((size_t)b.e * 4))) : cap;
}
// Whether a step's chunks run on several streams.
static bool chunks_overlap(const Plan& plan, const mona_options& opt, const mona_hparams& hp, size_t host_bytes) {
    int64_t chunks = 0;
    for (const Bucket& b : plan.buckets) {
        const int cap = chunk_capacity(b, hp, host_bytes);
        chunks += ((int64_t)b.mats.size() + cap - 1) / cap;
    }
    return opt.chunk_overlap && chunks > 1;
}
// Whether the matrices [start, start + C) of a bucket can be accessed 16 bytes at a time (base pointers are aligned).
static bool strides_aligned(const Plan& plan, const Bucket& b, int64_t start, int C) {
    const int64_t gsz = b.grad_dtype == MONA_BF16 ? 2 : 4;
    for (int c = 0; c < C; ++c) {
        const int64_t stride = plan.descs[b.mats[start + c].desc].batch_stride;
        if (stride * gsz % 16 != 0 || stride * 4 % 16 != 0) return false;
    }
    return b.e % 4 == 0;
}

// Bytes of parameters per chunk in mona_step_host(): a sixteenth of the set, so that the copy back starts early and little of either
// direction is left alone at the ends, but not so few that a chunk is all launch latency (8 MiB are 150 us of the link).
// One layer of 512 x 1024 experts, 218 MB each way: with chunks as large as the workspace holds the copy back started when two thirds
// of the gradients had arrived, 7.2 ms per step; with sixteenths 5.7
// (eighths 5.7, thirty-seconds 5.9, sixty-fourths 8.9).
static size_t host_chunk_bytes(const Plan& plan) {
    size_t total = 0;
    for (const Bucket& b : plan.buckets) total += b.mats.size() * (size_t)b.e * 4;
    return std::max<size_t>(8u << 20, total / 16);
}

// One optimizer step.  With `params_host` set (mona_step_host) every chunk's gradients are copied in on the handle's host-to-device
// stream before it runs, and its parameters are copied back on the device-to-host stream as soon as it is updated, so
// transfers in both directions overlap the remaining chunks.
static mona_status step_impl(mona_handle* h, const mona_hparams* hp, void* const* params, const void* const* grads,
                             void* const* o_out, uint32_t phase_mask, void* stream_v, void* const* params_host,
                             const void* const* grads_host) {
    if (!h) return MONA_ERR_INVALID_ARG;
    if (!hp || !params || !grads) return h->fail(MONA_ERR_INVALID_ARG, "hp, params or grads is null");
    if (hp->ns_steps < 0 || hp->ns_steps > 64) return h->fail(MONA_ERR_INVALID_ARG, "ns_steps out of range");
    if (hp->ns_precision != 0 && hp->ns_precision != 1) return h->fail(MONA_ERR_INVALID_ARG, "ns_precision must be 0 or 1");
    if (hp->scale_mode != 0 && hp->scale_mode != 1) return h->fail(MONA_ERR_INVALID_ARG, "scale_mode must be 0 or 1");
    if (hp->algorithm != 0 && hp->algorithm != 1) return h->fail(MONA_ERR_INVALID_ARG, "algorithm must be 0 (MONA) or 1 (Muon)");
    const Plan& plan = h->plan;
    const int64_t n_desc = (int64_t)plan.descs.size();
    for (int64_t i = 0; i < n_desc; ++i) {
        if (!params[i] || !grads[i]) return h->fail(MONA_ERR_INVALID_ARG, "params[%lld] or grads[%lld] is null", (long long)i, (long long)i);
        if (((uintptr_t)params[i] & 15) || ((uintptr_t)grads[i] & 15) || (o_out && o_out[i] && ((uintptr_t)o_out[i] & 15)))
            return h->fail(MONA_ERR_ALIGNMENT, "descriptor %lld: pointers must be 16-byte aligned", (long long)i);
    }
    MONA_CUDA(h, cudaSetDevice(h->device));
    NvtxRange step_range("mona_step");

    PrologueScalars ps;
    ps.beta = split(hp->accel_beta);
    ps.one_minus_beta = split(1.0 - hp->accel_beta);
    ps.alpha = split(hp->accel_alpha);
    ps.mu = split(hp->momentum);
    ps.eps = (float)hp->norm_eps;
    const float eta_lambda = (float)(hp->lr * hp->weight_decay);
    const int T = hp->ns_steps;
    const float ns_a = (float)hp->ns_a, ns_b = (float)hp->ns_b, ns_c = (float)hp->ns_c;     // fp32 path

    DeviceStatus* dstatus = (DeviceStatus*)(h->ws + WS_STATUS_OFF);
    // chunks alternate between the caller's stream (slot 0) and the handle's own stream (slot 1)
    const size_t host_bytes = params_host ? host_chunk_bytes(plan) : 0;
    const bool overlap = chunks_overlap(plan, h->opt, *hp, host_bytes);
    cudaStream_t slot_stream[NSLOTS] = {(cudaStream_t)stream_v};
    bool slot_used[NSLOTS] = {true};
    for (int sl = 1; sl < NSLOTS; ++sl) slot_stream[sl] = overlap && h->side[sl] ? h->side[sl] : (cudaStream_t)stream_v;
    if (overlap) MONA_CUDA(h, cudaEventRecord(h->ev_fork, slot_stream[0]));
    int64_t big_index = 0;
    struct DescRange { int desc; int64_t b0, b1; };      // matrices [b0, b1) of a descriptor
    std::vector<DescRange> ranges;                       // of the chunk (host pipeline only)
    size_t host_chunk = 0;
    h->launches = 0;
    h->flops_exec = 0.0;
    h->flops_dense = 0.0;
    h->flops_useful = 0.0;

    for (int bucket_index : plan.order) {
        const Bucket& b = plan.buckets[bucket_index];
        const bool tc = (hp->ns_precision == 0) && b.tc_ok && T >= 1;
        const int cap = chunk_capacity(b, *hp, host_bytes);
        const int64_t count = (int64_t)b.mats.size();
        const bool small = b.small && cap >= count;       // one chunk: the extra slots are made for whole buckets
        const double gamma = hp->scale_mode == 0 ? hp->scale_value * std::sqrt((double)b.l) : hp->scale_value;
        const float eta_gamma = (float)(hp->lr * gamma);
        const size_t gsz = b.grad_dtype == MONA_BF16 ? 2 : 4;
        const size_t aux = b.state_dtype == MONA_BF16 ? 2 : 4;
        float* Mst = (float*)(h->state + b.off_M);

        for (int64_t start = 0; start < count; start += cap) {
            const int C = (int)std::min<int64_t>(cap, count - start);
            ChunkPtrs ptrs;
            const bool vec4 = strides_aligned(plan, b, start, C);
            ranges.clear();
            for (int c = 0; c < C; ++c) {
                const MatRef& mr = b.mats[start + c];
                const mona_matrix_desc& d = plan.descs[mr.desc];
                if (params_host) {
                    if (ranges.empty() || ranges.back().desc != mr.desc) ranges.push_back({mr.desc, mr.b, mr.b});
                    ranges.back().b1 = mr.b + 1;
                }
                ptrs.g[c] = (const uint8_t*)grads[mr.desc] + (size_t)mr.b * d.batch_stride * gsz;
                ptrs.w[c] = (float*)params[mr.desc] + mr.b * d.batch_stride;
                ptrs.o[c] = (o_out && o_out[mr.desc]) ? (float*)o_out[mr.desc] + mr.b * d.batch_stride : nullptr;
                ptrs.gid[c] = (int)(plan.desc_first_gid[mr.desc] + mr.b);
            }
            const int slot = b.small ? b.slot : overlap ? (int)(big_index++ % BIG_SLOTS) : 0;
            if (overlap) {
                if (!slot_used[slot]) MONA_CUDA(h, cudaStreamWaitEvent(slot_stream[slot], h->ev_fork, 0));
                slot_used[slot] = true;
            }
            cudaStream_t stream = slot_stream[slot];
            uint8_t* ctrl = h->ws + WS_CTRL_OFF + slot * WS_CTRL_BYTES;
            uint8_t* data = h->ws + plan.slot_off[slot];
            unsigned int* sched = (unsigned int*)(ctrl + CTRL_SCHED_OFF);
            unsigned int* counters = (unsigned int*)(ctrl + CTRL_COUNTERS_OFF);
            float* inv_norm = (float*)(ctrl + CTRL_INVNORM_OFF);
            float* partials = (float*)(ctrl + CTRL_PARTIALS_OFF);
            float* Mc = Mst + start * b.e;
            void* Ac = h->state + b.off_A + (size_t)start * b.e * aux;
            void* Gc = h->state + b.off_G + (size_t)start * b.e * aux;
            __nv_bfloat16* xb[2] = {(__nv_bfloat16*)(data + b.off_x[0]), (__nv_bfloat16*)(data + b.off_x[1])};
            float* xf[2] = {(float*)(data + b.off32_x[0]), (float*)(data + b.off32_x[1])};
            float* af = (float*)(data + b.off32_a);
            float* bf = (float*)(data + b.off32_b);

            // elements [first, last) of a descriptor's buffer that belong to a range (padding up to the next matrix included)
            auto span = [&](const DescRange& r, int64_t& first, int64_t& last) {
                const mona_matrix_desc& d = plan.descs[r.desc];
                first = r.b0 * d.batch_stride;
                last = r.b1 == d.batch ? (d.batch - 1) * d.batch_stride + d.rows * d.cols : r.b1 * d.batch_stride;
            };
            if (params_host) {
                if (host_chunk == h->ev_in.size()) {
                    cudaEvent_t in = nullptr, out = nullptr;
                    MONA_CUDA(h, cudaEventCreateWithFlags(&in, cudaEventDisableTiming));
                    h->ev_in.push_back(in);
                    MONA_CUDA(h, cudaEventCreateWithFlags(&out, cudaEventDisableTiming));
                    h->ev_out.push_back(out);
                }
                for (const DescRange& r : ranges) {
                    int64_t first, last;
                    span(r, first, last);
                    MONA_CUDA(h, cudaMemcpyAsync((uint8_t*)const_cast<void*>(grads[r.desc]) + first * gsz, (const uint8_t*)grads_host[r.desc] + first * gsz,
                                                 (size_t)(last - first) * gsz, cudaMemcpyHostToDevice, h->h2d));
                }
                MONA_CUDA(h, cudaEventRecord(h->ev_in[host_chunk], h->h2d));
                MONA_CUDA(h, cudaStreamWaitEvent(stream, h->ev_in[host_chunk], 0));
            }
            const bool cleared_by_prologue = tc && small;
            // The last X' = B' X updates the parameters, from O rounded to bf16 as the separate pass would read it: O is neither written
            // nor read back, 4 of 12 bytes per element.  (Not host to host, where the step waits for the link and the update inside goes either
            // way: us apart -> inside, one 256 x 512 123 -> 115, 7 of 1024 x 2816 and 4 of its square 2455 -> 2411, 64 of 256 x 768 1357 -> 1402,
            // 16 each of 384 x 768 and 768 x 384 1160 -> 1174, one layer of 512 x 1024 experts 5650 -> 5660.)
            bool asked_for_o = false;
            for (int c = 0; c < C; ++c) asked_for_o = asked_for_o || ptrs.o[c];
            const NsChoice k = ns_choose(h->opt, h->max_pairs, h->pairs_beside[bucket_index], b, C, overlap && small, (phase_mask & 6u) == 6u && !params_host && vec4 && !asked_for_o, *hp);
            const bool update_inside = tc && k.update_inside;
            float** param_table = (float**)(ctrl + CTRL_PARAMS_OFF);
            if (phase_mask & 1u) {
                NvtxRange range("mona.prologue");
                MONA_CUDA(h, launch_prologue(ptrs, C, b.grad_dtype == MONA_BF16,
                                             hp->algorithm == 1 ? PROLOGUE_NO_AUX : (b.state_dtype == MONA_BF16 ? PROLOGUE_AUX_BF16 :
                                                 b.state_dtype == MONA_STATE_COMBINED ? PROLOGUE_AUX_COMBINED : PROLOGUE_AUX_F32), vec4, Mc, Ac, Gc, tc ? xb[0] : nullptr, partials,
                                             counters, inv_norm, dstatus, b.e, b.slab_len, b.slabs, ps, sched, cleared_by_prologue ? (int)ns_sched_words(C, NS_MAX_PHASES) : 0, update_inside ? param_table : nullptr, stream));
                ++h->launches;
            }
            else if (update_inside) {
                MONA_CUDA(h, launch_param_table(ptrs, C, param_table, stream));
                ++h->launches;
            }
            const void* o_final = nullptr;
            bool update_fused = false;
            if (tc) {
                if (phase_mask & 2u) {
                    NvtxRange range("mona.newton_schulz");
                    // the last X' = B' X applies the parameter update in its epilogue when this call runs both phases and the
                    // fp32 rows can be accessed 32 bytes at a time
                    update_fused = h->opt.fuse_update && (phase_mask & 4u) != 0u;
                    for (int c = 0; c < C && update_fused; ++c)
                        if (((uintptr_t)ptrs.w[c] & 31) || ((uintptr_t)ptrs.o[c] & 31)) update_fused = false;
                    bool launched = false;
                    for (int gi = 0; gi < k.groups;) {
                        NsProgram g = ns_next_launch(h->opt, b, C, k, *hp, update_fused, data, gi);
                        g.inv_norm = inv_norm; g.work_counter = sched; g.done = sched + 64;
                        g.eta_lambda = eta_lambda; g.eta_gamma = eta_gamma; g.params = param_table;
                        for (int q = 0; q < g.P; ++q) h->flops_exec += (double)C * ns_phase_executed_flops(g.ph[q]);
                        // For a small chunk the prologue of this call has cleared the scheduler words of the first launch: one
                        // operation less in a short chain (one 256 x 512 matrix 102 -> 100 us, a mixed small set 126 -> 124).
                        // Between a large prologue and its launch the memset stays: without it the launch takes the SMs
                        // before the other stream's prologue has started on them (12 dense blocks 3.20 -> 3.36 ms).
                        if (!(cleared_by_prologue && (phase_mask & 1u)) || launched) MONA_CUDA(h, cudaMemsetAsync(sched, 0, sizeof(unsigned int) * ns_sched_words(C, g.P), stream));
                        // Nothing stands between a small chunk's prologue and its first launch: launch and set-up overlap the prologue.
                        g.early = cleared_by_prologue && (phase_mask & 1u) && !launched;
                        launched = true;
                        NsUpdatePtrs up{};
                        if (update_fused && gi == k.groups) { up.w = ptrs.w; up.o = ptrs.o; }
                        MONA_CUDA(h, launch_ns_program(b.maps[slot], g, up, h->max_pairs, dstatus, stream));
                        ++h->launches;
                    }
                    h->flops_dense += (double)T * C * (4.0 * b.s * b.s * b.l + 2.0 * (double)b.s * b.s * b.s);
                    h->flops_useful += (double)T * C * (3.0 * b.s * b.s * b.l + (double)b.s * b.s * b.s);
                }
                o_final = xb[k.whole ? 0 : k.groups & 1];
            } else if (small_ns_eligible(b.rows, b.cols)) {
                // short side <= 64 (routers): the whole iteration in one launch, one block cluster per matrix
                if (phase_mask & 2u) {
                    NvtxRange range("mona.newton_schulz.small");
                    MONA_CUDA(h, launch_small_ns(Mc, xf[0], inv_norm, C, (int)b.rows, (int)b.cols, T, ns_a, ns_b, ns_c, stream));
                    ++h->launches;
                    h->flops_dense += (double)T * C * (4.0 * b.s * b.s * b.l + 2.0 * (double)b.s * b.s * b.s);
                }
                o_final = xf[0];
            } else {
                if (phase_mask & 2u) {
                    NvtxRange range("mona.newton_schulz.fp32");
                    MONA_CUDA(h, launch_scale(Mc, xf[0], inv_norm, C, b.e, b.up_slab_len, b.up_slabs, stream));
                    ++h->launches;
                    for (int t = 0; t < T; ++t) {
                        const int cur = t & 1, nxt = cur ^ 1;
                        SgemmArgs g1{};   // A = X X^T (wide) or X^T X (tall), s x s
                        g1.a = xf[cur]; g1.b = xf[cur]; g1.a_batch = g1.b_batch = b.e;
                        if (!b.tall) { g1.a_si = b.cols; g1.a_sk = 1; g1.b_sk = 1; g1.b_sj = b.cols; }
                        else         { g1.a_si = 1; g1.a_sk = b.cols; g1.b_sk = b.cols; g1.b_sj = 1; }
                        g1.cin = nullptr; g1.d = af; g1.ldd = b.s; g1.d_batch = b.s * b.s;
                        g1.M = g1.N = (int)b.s; g1.K = (int)b.l; g1.batch = C; g1.c1 = 0.f; g1.c2 = 1.f; g1.symmetric = 1;
                        MONA_CUDA(h, launch_sgemm(g1, stream));
                        SgemmArgs g2{};   // B' = b A + c A A + a I
                        g2.a = af; g2.b = af; g2.a_batch = g2.b_batch = b.s * b.s;
                        g2.a_si = b.s; g2.a_sk = 1; g2.b_sk = b.s; g2.b_sj = 1;
                        g2.cin = af; g2.d = bf; g2.ldd = b.s; g2.d_batch = b.s * b.s;
                        g2.M = g2.N = g2.K = (int)b.s; g2.batch = C; g2.c1 = ns_b; g2.c2 = ns_c; g2.diag_add = ns_a; g2.symmetric = 1;
                        MONA_CUDA(h, launch_sgemm(g2, stream));
                        SgemmArgs g3{};   // X' = B' X (wide) or X B' (tall)
                        if (!b.tall) {
                            g3.a = bf; g3.a_si = b.s; g3.a_sk = 1; g3.a_batch = b.s * b.s;
                            g3.b = xf[cur]; g3.b_sk = b.cols; g3.b_sj = 1; g3.b_batch = b.e;
                            g3.M = (int)b.s; g3.N = (int)b.l;
                        } else {
                            g3.a = xf[cur]; g3.a_si = b.cols; g3.a_sk = 1; g3.a_batch = b.e;
                            g3.b = bf; g3.b_sk = b.s; g3.b_sj = 1; g3.b_batch = b.s * b.s;
                            g3.M = (int)b.l; g3.N = (int)b.s;
                        }
                        g3.K = (int)b.s; g3.cin = nullptr; g3.d = xf[nxt]; g3.ldd = b.cols; g3.d_batch = b.e;
                        g3.batch = C; g3.c1 = 0.f; g3.c2 = 1.f;
                        MONA_CUDA(h, launch_sgemm(g3, stream));
                        h->launches += 3;
                        h->flops_dense += (double)C * (4.0 * b.s * b.s * b.l + 2.0 * (double)b.s * b.s * b.s);
                    }
                }
                o_final = xf[T & 1];
            }
            if ((phase_mask & 4u) && !update_fused && !update_inside) {
                NvtxRange range("mona.update");
                MONA_CUDA(h, launch_update(ptrs, C, tc, vec4, o_final, b.e, b.up_slab_len, b.up_slabs, eta_lambda, eta_gamma, !tc, stream));
                ++h->launches;
            }
            if (params_host) {
                MONA_CUDA(h, cudaEventRecord(h->ev_out[host_chunk], stream));
                MONA_CUDA(h, cudaStreamWaitEvent(h->d2h, h->ev_out[host_chunk], 0));
                for (const DescRange& r : ranges) {
                    int64_t first, last;
                    span(r, first, last);
                    MONA_CUDA(h, cudaMemcpyAsync((float*)params_host[r.desc] + first, (const float*)params[r.desc] + first, (size_t)(last - first) * 4,
                                                 cudaMemcpyDeviceToHost, h->d2h));
                }
                ++host_chunk;
            }
        }
    }
    for (int sl = 1; sl < NSLOTS; ++sl) {
        if (!overlap || !slot_used[sl]) continue;
        MONA_CUDA(h, cudaEventRecord(h->ev_join[sl], slot_stream[sl]));
        MONA_CUDA(h, cudaStreamWaitEvent(slot_stream[0], h->ev_join[sl], 0));
    }
    return MONA_OK;
}

extern "C" {

mona_status mona_step_ex(mona_handle* h, const mona_hparams* hp, void* const* params, const void* const* grads,
                         void* const* o_out, uint32_t phase_mask, void* stream_v) {
    return step_impl(h, hp, params, grads, o_out, phase_mask, stream_v, nullptr, nullptr);
}

mona_status mona_step(mona_handle* h, const mona_hparams* hp, void* const* params, const void* const* grads, void* stream) {
    return step_impl(h, hp, params, grads, nullptr, 7u, stream, nullptr, nullptr);
}

mona_status mona_step_host(mona_handle* h, const mona_hparams* hp, void* const* params, void* const* grads,
                           const void* const* grads_host, void* const* params_host, void* stream_v) {
    if (!h) return MONA_ERR_INVALID_ARG;
    if (!params || !grads || !grads_host || !params_host) return h->fail(MONA_ERR_INVALID_ARG, "null pointer array");
    cudaStream_t stream = (cudaStream_t)stream_v;
    MONA_CUDA(h, cudaSetDevice(h->device));
    const int64_t n_desc = (int64_t)h->plan.descs.size();
    for (int64_t i = 0; i < n_desc; ++i)
        if (!grads_host[i] || !grads[i] || !params_host[i] || !params[i])
            return h->fail(MONA_ERR_INVALID_ARG, "descriptor %lld: a gradient or parameter pointer (host or device) is null", (long long)i);
    if (!h->h2d) {
        MONA_CUDA(h, cudaStreamCreateWithFlags(&h->h2d, cudaStreamNonBlocking));
        MONA_CUDA(h, cudaStreamCreateWithFlags(&h->d2h, cudaStreamNonBlocking));
        MONA_CUDA(h, cudaEventCreateWithFlags(&h->ev_hfork, cudaEventDisableTiming));
        MONA_CUDA(h, cudaEventCreateWithFlags(&h->ev_hjoin, cudaEventDisableTiming));
    }
    // both copy streams start after whatever the caller's stream holds so far
    MONA_CUDA(h, cudaEventRecord(h->ev_hfork, stream));
    MONA_CUDA(h, cudaStreamWaitEvent(h->h2d, h->ev_hfork, 0));
    MONA_CUDA(h, cudaStreamWaitEvent(h->d2h, h->ev_hfork, 0));
    mona_status st = step_impl(h, hp, params, (const void* const*)grads, nullptr, 7u, stream_v, params_host, grads_host);
    // join the copy streams back into the caller's stream whether or not the step was enqueued completely
    const std::string step_error = h->last_error;
    MONA_CUDA(h, cudaEventRecord(h->ev_hjoin, h->h2d));
    MONA_CUDA(h, cudaStreamWaitEvent(stream, h->ev_hjoin, 0));
    MONA_CUDA(h, cudaEventRecord(h->ev_hjoin, h->d2h));
    MONA_CUDA(h, cudaStreamWaitEvent(stream, h->ev_hjoin, 0));
    if (st != MONA_OK) h->last_error = step_error;
    return st;
}

mona_status mona_selftest_timeout(mona_handle* h, void* stream_v) {
    if (!h) return MONA_ERR_INVALID_ARG;
    MONA_CUDA(h, cudaSetDevice(h->device));
    for (const Bucket& b : h->plan.buckets) {
        if (!b.tc_ok) continue;
        // the first matrix of the workspace slot, in the launch that a step with the default hyper-parameters makes over the bucket's first
        // chunk (O is stored instead of updating parameters), with stages that expect 16 bytes too many: the first product
        // never gets its operands, the others never get the first
        mona_hparams hp;
        mona_default_hparams(&hp);
        const int64_t i = &b - h->plan.buckets.data();
        const int C = (int)std::min<int64_t>(b.Cb, (int64_t)b.mats.size());
        uint8_t* ctrl = h->ws + WS_CTRL_OFF;
        uint8_t* data = h->ws + h->plan.slot_off[b.small ? b.slot : 0];
        unsigned int* sched = (unsigned int*)(ctrl + CTRL_SCHED_OFF);
        int gi = 0;
        NsProgram g = ns_next_launch(h->opt, b, C, ns_choose(h->opt, h->max_pairs, h->pairs_beside[i], b, C, b.small && chunks_overlap(h->plan, h->opt, hp, 0), false, hp),
                                     hp, false, data, gi);
        g.C = 1; g.delay = 1;
        g.inv_norm = (const float*)(ctrl + CTRL_INVNORM_OFF); g.work_counter = sched; g.done = sched + 64;
        g.selftest_extra_tx = 16;
        ns_program_plan(g);
        MONA_CUDA(h, cudaMemsetAsync(sched, 0, sizeof(unsigned int) * ns_sched_words(g.C, g.P), (cudaStream_t)stream_v));
        MONA_CUDA(h, launch_ns_program(b.maps[b.small ? b.slot : 0], g, NsUpdatePtrs{}, h->max_pairs, (DeviceStatus*)(h->ws + WS_STATUS_OFF), (cudaStream_t)stream_v));
        return MONA_OK;
    }
    return h->fail(MONA_ERR_UNSUPPORTED_SHAPE, "no descriptor of this handle takes the tensor-core path");
}

mona_status mona_describe_step(const mona_matrix_desc* descs, int64_t n_desc, const mona_options* options, const mona_hparams* hp, int32_t sm_pairs,
                               mona_launch_info* out, size_t capacity, size_t* n_launches) {
    if (!hp || !n_launches || sm_pairs < 1 || (capacity && !out) || hp->ns_steps < 0 || hp->ns_steps > 64) return MONA_ERR_INVALID_ARG;
    mona_options opt;
    if (resolve_options(options, opt) != MONA_OK) return MONA_ERR_INVALID_ARG;
    Plan plan;
    std::string err;
    const mona_status st = build_plan(descs, n_desc, opt.chunk_budget_bytes, plan, err);
    if (st != MONA_OK) return st;
    const std::vector<int> pairs_beside = share_pairs(plan, sm_pairs);
    const bool overlap = chunks_overlap(plan, opt, *hp, 0);
    int64_t big_index = 0;
    *n_launches = 0;
    for (int bucket_index : plan.order) {
        const Bucket& b = plan.buckets[bucket_index];
        const int64_t count = (int64_t)b.mats.size();
        const int cap = chunk_capacity(b, *hp, 0);
        for (int64_t start = 0; start < count; start += cap) {
            const int C = (int)std::min<int64_t>(cap, count - start);
            const int slot = b.small ? b.slot : overlap ? (int)(big_index++ % BIG_SLOTS) : 0;
            if (hp->ns_precision != 0 || !b.tc_ok) continue;
            const NsChoice k = ns_choose(opt, sm_pairs, pairs_beside[bucket_index], b, C, overlap && b.small && cap >= count, strides_aligned(plan, b, start, C), *hp);
            for (int gi = 0; gi < k.groups;) {
                const NsProgram g = ns_next_launch(opt, b, C, k, *hp, opt.fuse_update != 0, nullptr, gi);
                const NsPhase& p = g.ph[g.P - 1];
                if (*n_launches < capacity)
                    out[*n_launches] = {b.rows, b.cols, C, g.max_pairs, slot, p.fuse_update ? 0 : (int32_t)g.form, g.P, p.update || p.fuse_update ? (p.wide ? 2 * TC_BN : ns_tile_cols(p)) : 0};
                ++*n_launches;
            }
        }
    }
    return MONA_OK;
}

mona_status mona_poll_status(mona_handle* h, void* stream_v, int64_t* first_bad_matrix) {
    if (!h) return MONA_ERR_INVALID_ARG;
    cudaStream_t stream = (cudaStream_t)stream_v;
    MONA_CUDA(h, cudaSetDevice(h->device));
    MONA_CUDA(h, cudaMemcpyAsync(h->host_status, h->ws + WS_STATUS_OFF, sizeof(DeviceStatus), cudaMemcpyDeviceToHost, stream));
    static const DeviceStatus cleared = {0u, INT_MAX, 0u, 0u};
    MONA_CUDA(h, cudaMemcpyAsync(h->ws + WS_STATUS_OFF, &cleared, sizeof cleared, cudaMemcpyHostToDevice, stream));
    MONA_CUDA(h, cudaStreamSynchronize(stream));
    const DeviceStatus s = *h->host_status;
    if (first_bad_matrix) *first_bad_matrix = (s.first_bad == INT_MAX) ? -1 : s.first_bad;
    if (s.flags & STATUS_BOUNDS) return h->fail(MONA_ERR_BOUNDS, "an index check of the debug build failed (site %u)", s.timeout_site);
    if (s.flags & STATUS_TIMEOUT) return h->fail(MONA_ERR_TIMEOUT, "a device-side wait ran out (site %u)", s.timeout_site);
    if (s.flags & STATUS_NONFINITE) return h->fail(MONA_ERR_NONFINITE, "non-finite ||M||_F, first at matrix %d", s.first_bad);
    return MONA_OK;
}

mona_status mona_state_layout(const mona_handle* h, int64_t desc, size_t* off_M, size_t* off_A, size_t* off_Gprev) {
    if (!h || desc < 0 || desc >= (int64_t)h->plan.descs.size()) return MONA_ERR_INVALID_ARG;
    const Bucket& b = h->plan.buckets[h->plan.desc_bucket[desc]];
    const size_t aux = b.state_dtype == MONA_BF16 ? 2 : 4;
    const size_t pos = (size_t)h->plan.desc_pos[desc] * (size_t)b.e;
    if (off_M) *off_M = b.off_M + pos * 4;
    if (off_A) *off_A = b.off_A + pos * aux;
    if (off_Gprev) *off_Gprev = b.state_dtype == MONA_STATE_COMBINED ? (size_t)-1 : b.off_G + pos * aux;
    return MONA_OK;
}

int64_t mona_last_launch_count(const mona_handle* h) { return h ? h->launches : 0; }

mona_status mona_last_ns_flops(const mona_handle* h, double* executed, double* dense_equivalent) {
    if (!h) return MONA_ERR_INVALID_ARG;
    if (executed) *executed = h->flops_exec;
    if (dense_equivalent) *dense_equivalent = h->flops_dense;
    return MONA_OK;
}

mona_status mona_last_ns_useful_flops(const mona_handle* h, double* useful) {
    if (!h || !useful) return MONA_ERR_INVALID_ARG;
    *useful = h->flops_useful;
    return MONA_OK;
}

static_assert(MONA_TRACE_ROWS == mona::NS_TRACE_ROWS && MONA_TRACE_SLOTS == mona::NS_TRACE_SLOTS &&
              (int)MONA_TRACE_TILE0 == (int)mona::NS_TRACE_TILE0 && (int)MONA_TRACE_EPI_TILE0 == (int)mona::NS_TRACE_EPI_TILE0 && (int)MONA_TRACE_ITEMS == (int)mona::NS_TRACE_ITEMS &&
              (int)MONA_TRACE_EPI_ROLE == (int)mona::NS_TRACE_EPI_ROLE && (int)MONA_TRACE_SCHED_ROLE == (int)mona::NS_TRACE_SCHED_ROLE,
              "the public description of the profiling table follows the kernel's");

static_assert(mona::NS_MAX_PHASES == 16, "the range of n_phases that include/mona.h gives");
mona_status mona_work_order(int32_t n_matrices, int32_t n_phases, int32_t delay, const uint32_t* items_per_phase,
                            uint32_t start, uint32_t stride, int32_t* out_cqt, size_t capacity, size_t* n_written) {
    if (!n_written) return MONA_ERR_INVALID_ARG;
    const int n = mona::ns_work_order(n_matrices, n_phases, delay, items_per_phase, start, stride, out_cqt, capacity);
    if (n < 0) return MONA_ERR_INVALID_ARG;
    *n_written = (size_t)n;
    return MONA_OK;
}

mona_status mona_trace_read(unsigned long long* out, size_t rows, int reset) {
    if (rows && !out) return MONA_ERR_INVALID_ARG;
    int available = 0;
    const cudaError_t e = mona::ns_trace_read(out, rows, reset, &available);
    if (!available) return MONA_ERR_NOT_BUILT;
    return e == cudaSuccess ? MONA_OK : MONA_ERR_CUDA;
}

const char* mona_last_error(const mona_handle* h) { return h ? h->last_error.c_str() : "null handle"; }

void mona_destroy(mona_handle* h) {
    if (!h) return;
    for (cudaStream_t s : h->side) if (s) cudaStreamDestroy(s);
    if (h->ev_fork) cudaEventDestroy(h->ev_fork);
    if (h->h2d) cudaStreamDestroy(h->h2d);
    if (h->d2h) cudaStreamDestroy(h->d2h);
    if (h->ev_hfork) cudaEventDestroy(h->ev_hfork);
    if (h->ev_hjoin) cudaEventDestroy(h->ev_hjoin);
    for (cudaEvent_t e : h->ev_in) if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : h->ev_out) if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : h->ev_join) if (e) cudaEventDestroy(e);
    if (h->host_status) cudaFreeHost(h->host_status);
    delete h;
}

}  // extern "C"
