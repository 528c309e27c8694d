// Batched BEM products on the 5th-generation tensor cores (tcgen05, kind::tf32,
// "3xTF32": A_hi X_hi + A_hi X_lo + A_lo X_hi with FP32 accumulation in TMEM).
//
// The same-mesh batch turns u2_S = B u1_S (forward chain) and c_S = B^T t_S
// (adjoint chain) of the hybrid FEM/BEM open boundary (Sec. 3.1) into two dense
// GEMMs with the batch as the N dimension.  Both are computed as
//     Y[m][n] = sum_k A[m][k] X[n][k]        (A = B or B^T, both K-major)
// from padded FP32 copies of B and B^T and a transposed, hi/lo-split copy of the
// surface vectors.  One CTA computes a 128 x 64 tile over a K range (split-K,
// partials summed in a fixed order by a second kernel).
//
// Both products are one launch.  Warp roles (192 threads): warp 0 issues TMA loads (one
// elected lane), warp 1 owns the TMEM and issues the MMAs (one elected lane), warps 2-5
// split each A tile into its TF32 head (low mantissa bits cleared) and tail (A - head),
// a row per thread, and store both to TMEM, from where the MMAs take A; finally they read
// the accumulator back (each warp its lane quadrant).  Every wait on an mbarrier gives up
// after one second, sets the context's error word and leaves the CTA through the common
// exit that frees the TMEM columns.
//
// With head and tail in shared memory, its bandwidth bound the kernel: 150 KB a stage (16
// KB of A written by TMA, read, written twice by the split and read by twelve MMAs, with X)
// took 1200 clocks where HBM needs 680 for the 16 KB.  With A in TMEM a stage moves 72 KB,
// and 52 with 32 instances or fewer (tiles of 32 columns).
// Both products of 64 / 32 instances at n = 30, with split and sum: 113 / 99 -> 93 / 84 us.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <cuda.h>
#include <stdint.h>

#include "lbm_host.h"

namespace lbm {

namespace tc {

constexpr int BM = 128, BN = 64, BK = 32, STAGES = 6, THREADS = 192;
constexpr int A_BYTES = BM * BK * 4;   // 16 KB
template <int NT> constexpr int X_BYTES = NT * BK * 4;   // NT = 32 or BN columns: 4 or 8 KB
template <int NT> constexpr int STAGE_BYTES = A_BYTES + 2 * X_BYTES<NT>;
template <int NT> constexpr int SMEM_BYTES = STAGES * STAGE_BYTES<NT> + 1024 + 256;
// TMEM columns: the accumulator, then head and tail of A per stage (32 words each)
constexpr uint32_t TMEM_A = BN, TMEM_COLS = 512;
static_assert(TMEM_A + STAGES * 2 * BK <= TMEM_COLS, "one CTA's accumulator and stages of A");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Wait for the phase with the given parity; false after 1 s (error word set).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err) {
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t spin = 0;; ++spin) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((spin & 63u) == 63u) {
            if (*(volatile int*)err) return false;
            if (globaltimer_ns() - t0 > 1000000000ull) {
                atomicOr(err, DEV_ERR_TIMEOUT);
                return false;
            }
        }
    }
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor: K-major tile written by TMA with 128-byte
// swizzling (rows of 128 B, 8-row groups 1024 B apart).
__device__ __forceinline__ uint64_t sw128_desc(const void* tile) {
    const uint32_t addr = smem_u32(tile);
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);    // start address
    d |= (uint64_t)1 << 16;                     // leading byte offset (unused here)
    d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;                     // descriptor version
    d |= (uint64_t)2 << 61;                     // 128-byte swizzle
    return d;
}

// Instruction descriptor, kind::tf32: D FP32, A and B TF32, both K-major.
template <int NT>
constexpr uint32_t IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(NT >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);

// D += A X^T, A (128 rows = lanes, 8 words along K = columns) in TMEM
template <int NT>
__device__ __forceinline__ void mma_tf32(uint32_t dtmem, uint32_t atmem, uint64_t bdesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(dtmem),
        "r"(atmem), "l"(bdesc), "r"(IDESC<NT>), "r"(acc));
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};" ::"r"(r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
        "r"(r[29]), "r"(r[30]), "r"(r[31]), "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Ypart[product][split][m][n] = sum_{k in split} A[m][k] X[product ncols + n][k], m < nb,
// n < ncols; A = B for product 0 and B^T for product 1 (the second half of blockIdx.x)
template <int NT>
__global__ void __launch_bounds__(THREADS, 1)
    k_bem_tc(const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBT,
             const __grid_constant__ CUtensorMap mapXhi, const __grid_constant__ CUtensorMap mapXlo, int nb, int ncols,
             int kblocks_per_split, float* __restrict__ Ypart, int* err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = (uint64_t*)(smem + STAGES * STAGE_BYTES<NT>);
    uint64_t* full = bars;                 // [STAGES] TMA landed
    uint64_t* conv = bars + STAGES;        // [STAGES] head and tail of A in TMEM
    uint64_t* empty = bars + 2 * STAGES;   // [STAGES] MMAs of the stage done
    uint64_t* done = bars + 3 * STAGES;    // accumulator complete
    uint32_t* s_taddr = (uint32_t*)(bars + 3 * STAGES + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = gridDim.x / 2, second = (int)blockIdx.x >= mt;
    const int m0 = ((int)blockIdx.x - second * mt) * BM, xrow0 = second * ncols;
    const CUtensorMap* mapA = second ? &mapBT : &mapB;
    const int kb0 = blockIdx.y * kblocks_per_split;
    const int nkb_total = (nb + BK - 1) / BK;
    const int nkb = max(0, min(kblocks_per_split, nkb_total - kb0));

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&conv[s], 128);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_taddr)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *s_taddr;

    if (nkb > 0) {
        if (warp == 0 && lane == 0) {
            // ---- producer: TMA loads of A, X_hi, X_lo per stage -----------------
            for (int kb = 0; kb < nkb; ++kb) {
                const int s = kb % STAGES;
                if (kb >= STAGES && !mbar_wait(&empty[s], ((kb / STAGES) - 1) & 1, err)) break;
                uint8_t* st = smem + s * STAGE_BYTES<NT>;
                mbar_expect_tx(&full[s], A_BYTES + 2 * X_BYTES<NT>);
                const int k = (kb0 + kb) * BK;
                tma_load_2d(st, mapA, &full[s], k, m0);
                tma_load_2d(st + A_BYTES, &mapXhi, &full[s], k, xrow0);
                tma_load_2d(st + A_BYTES + X_BYTES<NT>, &mapXlo, &full[s], k, xrow0);
            }
        } else if (warp == 1 && lane == 0) {
            // ---- MMA issuer ----------------------------------------------------------
            for (int kb = 0; kb < nkb; ++kb) {
                const int s = kb % STAGES;
                if (!mbar_wait(&conv[s], (kb / STAGES) & 1, err)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint8_t* st = smem + s * STAGE_BYTES<NT>;
                const uint32_t ah = tmem + TMEM_A + s * 2 * BK, al = ah + BK;
                const uint64_t dXh = sw128_desc(st + A_BYTES), dXl = sw128_desc(st + A_BYTES + X_BYTES<NT>);
#pragma unroll
                for (int kk = 0; kk < BK / 8; ++kk) {
                    const uint64_t o = (uint64_t)(kk * 32) >> 4;   // 8 TF32 = 32 B along K
                    mma_tf32<NT>(tmem, ah + kk * 8, dXh + o, (kb > 0 || kk > 0) ? 1u : 0u);
                    mma_tf32<NT>(tmem, ah + kk * 8, dXl + o, 1u);
                    mma_tf32<NT>(tmem, al + kk * 8, dXh + o, 1u);
                }
                mma_commit(&empty[s]);
            }
            mma_commit(done);
        } else if (warp >= 2) {
            // ---- converters: row of A -> TF32 head and tail (A - head) in TMEM ----------
            // (a warp reaches the TMEM lanes of its quadrant: the same rows as its epilogue)
            const int row = (warp & 3) * 32 + lane;
            const uint32_t quadrant = (uint32_t)((warp & 3) * 32) << 16;
            bool ok = true;
            for (int kb = 0; kb < nkb && ok; ++kb) {
                const int s = kb % STAGES;
                // the stage's MMAs of the round before have finished: the producer waited for them
                ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (kb / STAGES) & 1, err));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint8_t* a = smem + s * STAGE_BYTES<NT> + row * (BK * 4);
                uint32_t h[32], l[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {   // 16-byte chunks, 128-byte swizzle
                    const uint4 v = *reinterpret_cast<const uint4*>(a + ((c ^ (row & 7)) << 4));
                    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        h[4 * c + q] = w[q] & 0xFFFFE000u;
                        l[4 * c + q] = __float_as_uint(__uint_as_float(w[q]) - __uint_as_float(h[4 * c + q]));
                    }
                }
                const uint32_t at = tmem + quadrant + TMEM_A + s * 2 * BK;
                tmem_st32(at, h);
                tmem_st32(at + BK, l);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive(&conv[s]);
            }
            // ---- epilogue: accumulator rows of this warp's lane quadrant -----------------
            if (ok && __all_sync(0xffffffffu, mbar_wait(done, 0, err))) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int quad = warp & 3;
                const int m = m0 + quad * 32 + lane;
                float* yrow = Ypart + (((size_t)second * gridDim.y + blockIdx.y) * nb + (m < nb ? m : 0)) * NT;
#pragma unroll
                for (int half = 0; half < NT / 32; ++half) {
                    float v[32];
                    tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 32), v);
                    if (m < nb)
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (half * 32 + j < ncols) yrow[half * 32 + j] = v[j];
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Y[m][product ncols + n] = sum_s Ypart[product][s][m][n] (fixed order)
template <typename T>
__global__ void k_tc_sum(const float* __restrict__ Ypart, int splits, int nb, int ncols, int nt, T* __restrict__ Y) {
    const int C = 2 * ncols, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nb * C) return;
    const int m = t / C, c = t - m * C, second = c >= ncols, n = c - second * ncols;
    const float* y = Ypart + ((size_t)second * splits * nb + m) * nt + n;
    float acc = 0.f;
#pragma unroll 4
    for (int s = 0; s < splits; ++s) acc += y[(size_t)s * nb * nt];
    Y[t] = T(acc);
}

// XT_hi / XT_lo [2B][ldp]: the surface vectors, transposed (column c of the
// [nb][2B] array becomes row c) and split into TF32 head and tail.
template <typename T>
__global__ void k_tc_split(const T* __restrict__ X, int nb, int C, int ldp, float* __restrict__ hi,
                           float* __restrict__ lo) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nb * C) return;
    const int k = t / C, c = t % C;
    const float v = (float)X[t];
    const float h = __uint_as_float(__float_as_uint(v) & 0xFFFFE000u);
    hi[(size_t)c * ldp + k] = h;
    lo[(size_t)c * ldp + k] = v - h;
}

}  // namespace tc

// ---- host side --------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The tensor-map encoder is a driver-API function; it is looked up through the
// runtime so that the library itself does not link against libcuda.
static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

static int make_map(CUtensorMap* map, const float* base, int inner, int outer, int ld, int box_inner, int box_outer) {
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_outer};
    const cuuint32_t estr[2] = {1, 1};
    EncodeTiledFn enc = encode_fn();
    if (!enc) return -3;
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)base, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : (int)r;
}

int tc_ld(int nb) { return (nb + 31) & ~31; }

constexpr int TC_MAX_SPLITS = 8;   // largest split-K count the autotuner tries

size_t tc_scratch_floats(int nb, int B, int num_sms) {
    (void)num_sms;
    const int ldp = tc_ld(nb);
    return (size_t)2 * (2 * B) * ldp + (size_t)2 * TC_MAX_SPLITS * nb * (B <= 32 ? 32 : tc::BN) + 64;
}

// ---- autotuner: split-K count of the tensor-core product ----------------------------
// At the first product of a (nb, B, SM count) the kernel is timed with every
// candidate split count (K blocks per split rounded so that every split has
// work) on the operands in scratch, with CUDA events on the launching stream;
// the fastest is kept for the process.  Only scratch is written while tuning.
namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int>, int> g_tc_splits;

int splits_for(int nkb, int want, int* kps_out) {
    int splits = want < 1 ? 1 : (want > nkb ? nkb : want);
    const int kps = (nkb + splits - 1) / splits;
    *kps_out = kps;
    return (nkb + kps - 1) / kps;   // every split has at least one K block
}
}  // namespace

template <typename F>
static int tc_tuned_splits(const Launch& L, int nb, int B, F&& launch_with) {
    const auto key = std::make_tuple(nb, B, L.num_sms);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tc_splits.find(key);
        if (it != g_tc_splits.end()) return it->second;
    }
    const int mt = (nb + tc::BM - 1) / tc::BM, nkb = (nb + tc::BK - 1) / tc::BK;
    // at least as many as fill the chip with one product: the tensor cores' FP32 sums lose
    // accuracy with their length (twice the error at twice the K range)
    const int least = std::min(std::min(TC_MAX_SPLITS, nkb), (L.num_sms + mt - 1) / mt);
    if (!L.tune) return least;
    int best = 0;
    float best_ms = 0.f;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    for (int want = least; want <= TC_MAX_SPLITS; ++want) {
        int kps;
        const int splits = splits_for(nkb, want, &kps);
        if (splits != want) continue;
        float t[3];
        for (int rep = 0; rep < 3; ++rep) {
            cudaEventRecord(e0, L.stream);
            launch_with(splits, kps);
            cudaEventRecord(e1, L.stream);
            cudaEventSynchronize(e1);
            cudaEventElapsedTime(&t[rep], e0, e1);
            *L.launches += 1;
        }
        const float med = std::max(std::min(t[0], t[1]), std::min(std::max(t[0], t[1]), t[2]));
        if (best == 0 || med < best_ms) {
            best = splits;
            best_ms = med;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (best == 0) best = least;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tc_splits[key] = best;
    return best;
}

int tc_splits_chosen(int nb, int B, int num_sms) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tc_splits.find(std::make_tuple(nb, B, num_sms));
    return it == g_tc_splits.end() ? 0 : it->second;
}

// Both BEM products of the batch on the tensor cores.  A32 / A32T: padded FP32
// copies of B and B^T (ld = tc_ld(nb)); scratch: tc_scratch_floats(...) floats.
template <typename T>
int bem_product_tc(const Launch& L, int nb, const float* A32, const float* A32T, const T* ub_in, T* ub_out, int B,
                   float* scratch) {
    if (B > tc::BN) return -1;
    const int C = 2 * B, ldp = tc_ld(nb);
    float* xhi = scratch;
    float* xlo = scratch + (size_t)C * ldp;
    float* ypart = scratch + (size_t)2 * C * ldp;
    const int total = nb * C, nt = B <= 32 ? 32 : tc::BN;
    tc::k_tc_split<T><<<(total + 255) / 256, 256, 0, L.stream>>>(ub_in, nb, C, ldp, xhi, xlo);
    const int mt = (nb + tc::BM - 1) / tc::BM, nkb = (nb + tc::BK - 1) / tc::BK;
    CUtensorMap mA, mAT, mXh, mXl;
    int e = make_map(&mA, A32, nb, nb, ldp, tc::BK, tc::BM);
    if (!e) e = make_map(&mAT, A32T, nb, nb, ldp, tc::BK, tc::BM);
    if (!e) e = make_map(&mXh, xhi, nb, C, ldp, tc::BK, nt);
    if (!e) e = make_map(&mXl, xlo, nb, C, ldp, tc::BK, nt);
    if (e) return e;
    // forward: rows 0..B-1 of X; adjoint: rows B..2B-1 with B^T
    auto run = [&](auto fn, int smem) -> int {
        if (kernel_smem_attr((const void*)fn, smem) != cudaSuccess) return -3;
        auto launch = [&](int splits, int kps) {
            fn<<<dim3(2 * mt, splits), tc::THREADS, smem, L.stream>>>(mA, mAT, mXh, mXl, nb, B, kps, ypart, L.err);
        };
        int kps;
        const int splits = splits_for(nkb, tc_tuned_splits(L, nb, B, launch), &kps);
        launch(splits, kps);
        tc::k_tc_sum<T><<<(total + 255) / 256, 256, 0, L.stream>>>(ypart, splits, nb, B, nt, ub_out);
        return 0;
    };
    e = nt == 32 ? run(tc::k_bem_tc<32>, tc::SMEM_BYTES<32>) : run(tc::k_bem_tc<tc::BN>, tc::SMEM_BYTES<tc::BN>);
    if (e) return e;
    *L.launches += 3;
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

// padded FP32 copies of B and B^T for the tensor-core path
__global__ void k_tc_pad(const float* __restrict__ B32, int nb, int ldp, float* __restrict__ A, float* __restrict__ AT) {
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t >= (size_t)nb * nb) return;
    const int i = (int)(t / nb), j = (int)(t % nb);
    const float v = B32[t];
    A[(size_t)i * ldp + j] = v;
    AT[(size_t)j * ldp + i] = v;
}

void tc_prepare(const Launch& L, const float* B32, int nb, float* A, float* AT) {
    const int ldp = tc_ld(nb);
    cudaMemsetAsync(A, 0, sizeof(float) * (size_t)nb * ldp, L.stream);
    cudaMemsetAsync(AT, 0, sizeof(float) * (size_t)nb * ldp, L.stream);
    const size_t total = (size_t)nb * nb;
    k_tc_pad<<<(unsigned)((total + 255) / 256), 256, 0, L.stream>>>(B32, nb, ldp, A, AT);
    *L.launches += 1;
}

template int bem_product_tc<float>(const Launch&, int, const float*, const float*, const float*, float*, int, float*);
template int bem_product_tc<double>(const Launch&, int, const float*, const float*, const double*, double*, int,
                                    float*);

}  // namespace lbm
