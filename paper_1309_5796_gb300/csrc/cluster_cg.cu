// CG with a Chebyshev polynomial of the Jacobi-scaled matrix as preconditioner, one
// thread-block cluster per group of VEC systems, the iteration's vectors in the
// cluster's shared memory: the potential solves of general meshes (two-stage
// FEM/BEM chains, as k_pcg in solver.cu).
//
// CTA r of a cluster owns the contiguous rows [r rpc, (r+1) rpc).  z (and the copy
// its polynomial steps alternate with) of its rows is in its shared memory, where
// the other CTAs' products read it (distributed shared memory); the step dd, r, p, q
// and the correction d of x follow as far as they fit, the rest stay in global
// memory.  The CTA's matrix entries are there too when they fit, each with the
// cluster address of its z.  Per iteration:
//   B  alpha = rho / p.q, d += alpha p, r -= alpha q, z = dd = D^-1 r / theta, sums r.r, r
//   C  DEG - 1 steps dd = c1 dd + c2 D^-1 (r - K z), z += dd; sum r.z with the last
//   A  p = z + beta p, q = K z + beta q (= K p), sum p.q
// The polynomial is Chebyshev's on [b / ratio, b], b a bound of the eigenvalues of
// D^-1 K (Gershgorin, at most 4 for linear tetrahedra), its degree by size (cc_degree):
// on a ball of 19 683 nodes 15 iterations of 16 products do the work of 187 CG
// iterations, with one plain cluster barrier a product in place of two reductions.
// A sum goes from the warps (W) to a total per CTA that is pushed to every CTA's
// shared memory before the barrier, and is added there over the CTAs (FP64) in a
// fixed order.  The launch shape depends on the sizes and the batch only, so a
// solve gives the same bits every time.
//
// Measured (both stages of both chains): one instance on 19 683 nodes in FP32 1.83 ms,
// 7.2 with the grid-wide kernel; 16 on 3 375 nodes in FP64 4.0 ms, before 8.5.
// What bounds it: latency, in FP64 also the FP64 units.  A cluster barrier costs 400 to 650
// clocks, a reduction with its barrier about 1700, a product of 15 entries a row about 2000
// at two rows a thread (distributed shared memory serves 19 bytes a clock to an SM).
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "solver_common.cuh"

namespace lbm {
namespace {

constexpr size_t CC_SMEM_MAX = 225 * 1024;
// A CTA whose matrix entries are in global memory: the products read them a row a thread,
// so a line has to stay in the L1 (what the shared memory leaves of 256 KB) until its next
// entries are used.  Less shared memory, and vectors that go to global memory instead, are
// faster then (ms an evaluation with all of it -> with this much): FP32, 4 / 8 instances on
// 59 319 nodes 23.1 -> 11.5 / 32.6 -> 15.7, one on 117 649 64 -> 25, 5 iterated in FP32 on
// 74 088 128 -> 43.  In FP64, where the units bind too, 4 on 46 656 39.4 -> 35.4 and one on
// 59 319 41.8 -> 36.7 at 200 KB; less than that takes vectors of small shapes (12 on 24 389
// 30 -> 43 ms at 130 KB).
template <typename W> constexpr size_t CC_SMEM_BARE = (sizeof(W) == 8 ? 200 : 130) * 1024;
constexpr int CC_MAX_CL = 16;
constexpr int CC_NQ = 4;            // most quantities of one reduction
constexpr int CC_VECS = 7;          // z, z', dd, r, p, q, d (dd from z and z' instead: 2 to 4 % slower)

// Products of an iteration and the ratio of the polynomial's interval.  A higher degree
// saves reductions, but the last iteration's surplus weighs more where few are needed.
// ms an evaluation at 4 on [b / 60, b], 6 on [b / 120, b], 8, 12 and 16 on [b / 240, b]:
// FP64, one instance on 27 nodes 0.59, 0.73 (2 on [b / 15, b]: 0.38), on 729 1.12, 1.23, 1.48,
// 1.42, 1.36, on 2 197 1.65, 1.61, 1.86, 1.78, 1.67, on 4 913 2.89, 2.64, 2.78, 2.67, 2.58, on
// 9 261 4.76, 4.37, 4.35, 4.17, 4.21, on 19 683 11.3, 10.7, 10.3, 10.5, 10.6, 32 on 3 375 9.2,
// 9.8, 12.0, 11.4, 11.5; FP32, one on 1 331 0.50, 0.45, 0.48, 0.47, 0.43, on 4 913 0.83, 0.74,
// 0.73, 0.70, 0.69, on 9 261 1.27, 1.15, 1.07, 1.05, 1.08, on 19 683 2.19, 2.03, 1.94, 1.94,
// 1.92, 32 on 2 197 1.15, 1.13, 1.21, 1.19, 1.22; FP64 iterated in FP32 as FP32.  Within 8 %
// of the best of these in FP64, within 12 % for one FP32 instance between the lines (up to
// 20 % on 1 331 to 2 197 nodes) and 3 % for thirty-two.
void cc_degree(int rows, int& deg, double& ratio) {
    deg = rows >= 8192 ? 16 : rows >= 3000 ? 6 : rows >= 90 ? 4 : 2;
    ratio = rows >= 8192 ? 240.0 : rows >= 3000 ? 120.0 : rows >= 90 ? 60.0 : 15.0;
}

extern __shared__ __align__(16) unsigned char cc_sm[];

__device__ __forceinline__ unsigned cc_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cc_index() {
    unsigned r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cc_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cc_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cc_peer(uint32_t a, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cc_ld(uint32_t a, float (&v)[1]) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[0]) : "r"(a));
}
__device__ __forceinline__ void cc_ld(uint32_t a, float (&v)[2]) {
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(a));
}
__device__ __forceinline__ void cc_ld(uint32_t a, float (&v)[4]) {
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(a));
}
__device__ __forceinline__ void cc_ld(uint32_t a, double (&v)[1]) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[0]) : "r"(a));
}
__device__ __forceinline__ void cc_ld(uint32_t a, double (&v)[2]) {
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
}
__device__ __forceinline__ void cc_st(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ float cc_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double cc_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
// VEC consecutive values; CG: through L2 (values other CTAs write)
template <int VEC, bool CG, typename X>
__device__ __forceinline__ void cc_get(X (&d)[VEC], const X* p) {
    if constexpr (VEC == 1) d[0] = CG ? __ldcg(p) : *p;
    else vload<X, VEC, CG>(d, p);
}
template <int VEC, typename X>
__device__ __forceinline__ void cc_put(X* p, const X (&d)[VEC]) {
    if constexpr (VEC == 1) *p = d[0];
    else vstore<X, VEC>(p, d);
}

struct CcGeo {
    int rows, rpc, cl;                 // rows of a system, rows per CTA, CTAs per cluster
    int nvec;                          // vectors in shared memory: z, z', then dd, r, p, q, d
    int fit;                           // as many as would fit it
    int deg;                           // products of an iteration
    double ratio;                      // the polynomial's interval: [b / ratio, b]
    double th, de;                     // its centre and half-width
    int ent;                           // general meshes: most entries of a CTA when they are in shared memory, else 0
    unsigned mul, shift;               // j / rpc = umulhi(j, mul) >> shift
    unsigned o_dinv, o_ent, o_ptr, o_scr, o_slot, o_col, smem;
};

template <typename T, typename W>
struct CcArgs {
    PcgArgs<T> P;
    CcGeo g;
    W *v[5];                           // global room of dd, r, p, q, d: [group][rows][VEC]
};

// T: type of the potential x and of the residual f - K x; W: type of the CG
// vectors and of an iteration's sums inside a CTA (the residual's and its reference's are
// SumOf's, the gauge's FP64).  T = W: CG to the tolerance.  T = double,
// W = float: cycles of the FP64 residual and FP32 CG until it has reduced that
// residual by MP_INNER; the solve ends on the FP64 residual test.
template <typename T, typename W, int VEC>
__global__ void __launch_bounds__(sizeof(W) == 8 ? 512 : 1024, 1) k_cluster_cg(const __grid_constant__ CcArgs<T, W> A) {
    constexpr bool MP = sizeof(T) != sizeof(W);
    const CcGeo& g = A.g;
    const PcgArgs<T>& P = A.P;
    W* const z0s = reinterpret_cast<W*>(cc_sm);                       // [2][rpc][VEC]: z and the copy the steps alternate with
    W* const dtab = reinterpret_cast<W*>(cc_sm + g.o_dinv);           // [rpc] 1 / K_ii, 0 where z stays zero
    uint32_t* eaddr = reinterpret_cast<uint32_t*>(cc_sm + g.o_ent + (size_t)g.ent * sizeof(W));
    W* eval = reinterpret_cast<W*>(cc_sm + g.o_ent);
    int* eptr = reinterpret_cast<int*>(cc_sm + g.o_ptr);              // [rpc + 1]
    W* scr = reinterpret_cast<W*>(cc_sm + g.o_scr);                   // [32 warps][CC_NQ * VEC]
    double* slots = reinterpret_cast<double*>(cc_sm + g.o_slot);      // [2][CC_NQ * VEC][CC_MAX_CL]
    double* out = reinterpret_cast<double*>(cc_sm + g.o_col);         // [CC_NQ * VEC]
    double* s_rho = out + CC_NQ * VEC;
    double* s_rhop = s_rho + VEC;
    double* s_tol = s_rhop + VEC;
    double* s_tin = s_tol + VEC;
    double* s_mean = s_tin + VEC;
    W* s_ab = reinterpret_cast<W*>(s_mean + VEC);
    int* s_flag = reinterpret_cast<int*>(reinterpret_cast<double*>(s_ab) + VEC);
    int* s_it = s_flag + VEC;
    int* s_done = s_it + VEC;
    uint32_t* s_base = reinterpret_cast<uint32_t*>(s_done + VEC);     // [CC_MAX_CL] cluster address of every CTA's z
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const unsigned rank = cc_rank();
    const int B = P.V.B, C = 2 * B, mode = P.mode, R = g.rows, rpc = g.rpc;
    const int grp = (int)cc_index(), c0 = grp * VEC, b0 = c0 % B;
    const bool neu = mode == c0 / B;   // B % VEC == 0: one kind per cluster
    const int lo = (int)rank * rpc, hi = min(R, lo + rpc), cnt = max(0, hi - lo);
    bool act[VEC], any = false;
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        act[k] = P.V.st[b0 + k].phase != PH_DONE;
        any |= act[k];
    }
    int itmax = 0;
    if (any) {
        W* vec[5];   // of the own rows, indexed by local row
#pragma unroll
        for (int v = 0; v < 5; ++v)
            vec[v] = v + 3 <= g.nvec ? z0s + (size_t)(v + 2) * rpc * VEC : A.v[v] + ((size_t)grp * R + lo) * VEC;
        W* __restrict__ dd = vec[0];
        W* __restrict__ r = vec[1];
        W* __restrict__ p = vec[2];
        W* __restrict__ q = vec[3];
        W* __restrict__ d = vec[4];
        const uint32_t zflip = (uint32_t)((size_t)rpc * VEC * sizeof(W));
        T* __restrict__ x = mode ? P.V.U2 : P.V.U1;
        for (int o = tid; o < g.cl; o += nt) s_base[o] = cc_peer(cc_addr(z0s), (unsigned)o);
        if (tid < VEC) {
            s_it[tid] = 0;
            s_done[tid] = 0;
            s_tin[tid] = 0.0;
            s_mean[tid] = 0.0;
        }
        __syncthreads();
        auto owner = [&](int j) { return (int)(__umulhi((unsigned)j, g.mul) >> g.shift); };
        auto zaddr = [&](int j) {
            const int o = owner(j);
            return s_base[o] + (uint32_t)((j - o * rpc) * VEC * (int)sizeof(W));
        };
        if (g.ent) {   // the CTA's matrix entries with the places of their z
            const W* kv = GenTab<W>::k(P.M);
            const int e0 = P.M.kptr[lo], e1 = P.M.kptr[hi];
            for (int e = e0 + tid; e < e1; e += nt) {
                eaddr[e - e0] = zaddr((int)((unsigned)P.M.kent[e] >> 8));
                eval[e - e0] = kv[e];
            }
            for (int i = tid; i <= cnt; i += nt) eptr[i] = P.M.kptr[lo + i] - e0;
        }
        int par = 0;
        // Totals over the cluster of NQ quantities of VEC columns into out[(q0 + q) * VEC + k];
        // of W, or of what keeps more (SumOf, FP64; two FP32 words of scr hold one: at most
        // CC_NQ / 2 quantities then).
        auto reduce = [&](auto& v, int q0) {
            constexpr int NQ = sizeof(v) / sizeof(v[0]), NV = NQ * VEC;
            using X = typename std::remove_reference<decltype(v[0][0])>::type;
            static_assert(NQ * sizeof(X) <= CC_NQ * sizeof(W), "scr holds them");
            X* const sc = reinterpret_cast<X*>(scr);   // [32 warps][NV]
#pragma unroll
            for (int a = 0; a < NQ; ++a)
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v[a][k] = plus(v[a][k], shfl_x(v[a][k], o));
                    if (lane == 0) sc[warp * NV + a * VEC + k] = v[a][k];
                }
            __syncthreads();
            const uint32_t sl = cc_addr(slots + par * CC_NQ * VEC * CC_MAX_CL);
            for (int w = warp; w < NV; w += nw) {
                X t{};
                if (lane < nw) t = sc[lane * NV + w];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) t = plus(t, shfl_x(t, o));
                if (lane < g.cl) cc_st(cc_peer(sl + (uint32_t)(w * CC_MAX_CL + (int)rank) * 8u, (unsigned)lane), total(t));
            }
            cc_sync();
            for (int w = warp; w < NV; w += nw) {
                double t = lane < g.cl ? slots[(par * CC_NQ * VEC + w) * CC_MAX_CL + lane] : 0.0;
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (lane == 0) out[q0 * VEC + w] = t;
            }
            par ^= 1;   // rewritten only after a further barrier, when every CTA has read it
            __syncthreads();
        };
        int cur = 0;   // which of the two copies holds z
        // (K z) of the own local row l
        auto apply = [&](int l, W (&w)[VEC]) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) w[k] = W(0);
            // BATCH entries at a time: their places and values, then every z, then the sums
            constexpr int BATCH = VEC == 4 ? 4 : 8;
            int e0, e1;
            if (g.ent) {
                e0 = eptr[l];
                e1 = eptr[l + 1];
            } else {
                e0 = P.M.kptr[lo + l];
                e1 = P.M.kptr[lo + l + 1];
            }
            const W* kv = GenTab<W>::k(P.M);
            for (int e = e0; e < e1; e += BATCH) {
                uint32_t ad[BATCH];
                W a[BATCH], z[BATCH][VEC];
                if (g.ent) {
#pragma unroll
                    for (int t = 0; t < BATCH; ++t) {
                        const int m = min(e + t, e1 - 1);
                        ad[t] = eaddr[m] + (cur ? zflip : 0u);
                        a[t] = e + t < e1 ? eval[m] : W(0);
                    }
                } else {
#pragma unroll
                    for (int t = 0; t < BATCH; ++t) {
                        const int m = min(e + t, e1 - 1);
                        ad[t] = zaddr((int)((unsigned)__ldg(&P.M.kent[m]) >> 8)) + (cur ? zflip : 0u);
                        a[t] = e + t < e1 ? __ldg(&kv[m]) : W(0);
                    }
                }
#pragma unroll
                for (int t = 0; t < BATCH; ++t) cc_ld(ad[t], z[t]);
#pragma unroll
                for (int t = 0; t < BATCH; ++t)
#pragma unroll
                    for (int k = 0; k < VEC; ++k) w[k] = cc_fma(a[t], z[t][k], w[k]);
            }
        };
        // 1 / K_ii; 0 on frozen rows
        for (int l = tid; l < cnt; l += nt) {
            const int row = lo + l;
            const bool frozen = !neu && ((unsigned)__ldg(&P.M.node[row]) >> 16) != 0;
            dtab[l] = frozen ? W(0) : W(1) / __ldg(&GenTab<W>::d(P.M)[row]);
        }

        // Dirichlet systems: surface values (stage 1 adjoint: zero; stage 2 forward: B u1_S)
        if (!neu)
            for (int row = lo + tid; row < hi; row += nt) {
                const int bp = (int)((unsigned)P.M.node[row] >> 16);
                if (!bp) continue;
#pragma unroll
                for (int k = 0; k < VEC; ++k)
                    if (act[k]) x[(size_t)row * C + c0 + k] = mode ? P.V.ub_out[(size_t)(bp - 1) * C + b0 + k] : T(0);
            }
        cc_sync();
        for (int cycle = 0;; ++cycle) {
            {   // residual of the current x into r; sums r.r, r and f.f, f (f: the norm reference)
                typename SumOf<W>::type v[2][VEC], vf[2][VEC];
                for (int l = tid; l < cnt; l += nt) {
                    const int row = lo + l;
                    W rv[VEC];
                    const int bp = (int)((unsigned)P.M.node[row] >> 16);
                    if (!neu && bp) {
#pragma unroll
                        for (int k = 0; k < VEC; ++k) rv[k] = W(0);
                    } else {
                        const T* kvT = GenTab<T>::k(P.M);
                        T xi[VEC], kx[VEC];
                        double f[VEC];
                        typename SumOf<T>::type ks[VEC];
                        cc_get<VEC, true>(xi, x + (size_t)row * C + c0);
#pragma unroll
                        for (int k = 0; k < VEC; ++k) {
                            kx[k] = T(0);
                            f[k] = 0.0;
                        }
                        const int e0 = P.M.kptr[row], e1 = P.M.kptr[row + 1];
                        // entries in flight; with four, wider FP32 vectors spill in every product
                        constexpr int RU = sizeof(W) == 8 || (VEC == 1 && !MP) ? 4 : 2;
#pragma unroll RU
                        for (int e = e0; e < e1; ++e) {
                            const int j = (int)((unsigned)__ldg(&P.M.kent[e]) >> 8);
                            const T kv = __ldg(&kvT[e]);
                            T xj[VEC];
                            cc_get<VEC, true>(xj, x + (size_t)j * C + c0);
                            const bool s = !neu && mode && ((unsigned)__ldg(&P.M.node[j]) >> 16);
#pragma unroll
                            for (int k = 0; k < VEC; ++k) {
                                kx[k] = cc_fma(kv, xj[k] - xi[k], kx[k]);
                                if (s) ks[k].fma(kv, xj[k]);   // K_IS x_S
                            }
                        }
                        if (!(mode == 1 && !neu)) {
                            cc_get<VEC, false>(f, P.V.bvec + (size_t)row * B + b0);
#pragma unroll
                            for (int k = 0; k < VEC; ++k) {
                                if (!act[k]) f[k] = 0.0;
                                if (mode == 1 && bp) f[k] += (double)P.V.ub_out[(size_t)(bp - 1) * C + c0 + k];
                            }
                        }
#pragma unroll
                        for (int k = 0; k < VEC; ++k) {
                            rv[k] = W(T(f[k]) - kx[k]);
                            const W ref = W(T(f[k]) - scaled(T(1), ks[k]));
                            v[0][k].fma(rv[k], rv[k]);
                            v[1][k].add(rv[k]);
                            vf[0][k].fma(ref, ref);
                            vf[1][k].add(ref);
                        }
                    }
                    cc_put<VEC>(r + (size_t)l * VEC, rv);
                }
                reduce(v, 0);
                reduce(vf, 2);
                if (tid < VEC) {
                    const double sf = out[3 * VEC + tid], ff = out[2 * VEC + tid];
                    if (cycle == 0) s_tol[tid] = P.tol2 * (neu ? fmax(ff - sf * sf / (double)R, 0.0) : ff);
                    s_rhop[tid] = 1.0;
                }
                __syncthreads();
            }
            int it = 0;
            for (;; ++it) {
                // out: r.r, sum r (first pass: of the residual with its mean)
                if (tid < VEC) {
                    if (it > 0) {   // bookkeeping of the iteration just finished
                        s_rhop[tid] = s_rho[tid];
                        if (!s_flag[tid]) s_it[tid] += 1;
                    }
                    const double sr = out[VEC + tid];
                    // Neumann: the residual without its null-space (mean) component
                    const double rr = neu ? fmax(out[tid] - sr * sr / (double)R, 0.0) : out[tid];
                    const bool a = P.V.st[b0 + tid].phase != PH_DONE;
                    int conv;
                    if constexpr (MP) {
                        if (it == 0) {   // rr is the true (FP64) residual of this cycle
                            s_done[tid] = !a || !(rr > s_tol[tid]) || s_it[tid] >= P.max_iter;
                            s_tin[tid] = fmax(s_tol[tid], MP_INNER * MP_INNER * rr);
                        }
                        conv = s_done[tid] || !(rr > s_tin[tid]) || s_it[tid] >= P.max_iter;
                    } else {
                        conv = !a || !(rr > s_tol[tid]) || it >= P.max_iter;
                    }
                    s_flag[tid] = conv;
                    s_mean[tid] = neu && it == 0 ? sr / (double)R : 0.0;   // a consistent residual (sum zero)
                }
                // the same totals in every CTA of the cluster: every CTA leaves together
                if (__syncthreads_and(tid < VEC ? s_flag[tid] : 1)) break;
                // ---- C: z = p(D^-1 K) D^-1 r -----------------------------------------
                const W th = W(g.th), de = W(g.de);
                W ab[VEC], v1[1][VEC];
                if (it == 0) {   // later iterations: done with the update of r
#pragma unroll
                    for (int k = 0; k < VEC; ++k) ab[k] = W(s_mean[k]);
                    for (int l = tid; l < cnt; l += nt) {
                        W rv[VEC], zv[VEC];
                        const W di = dtab[l], dt = di / th;
                        cc_get<VEC, false>(rv, r + (size_t)l * VEC);
#pragma unroll
                        for (int k = 0; k < VEC; ++k) {
                            if (di != W(0)) rv[k] -= ab[k];
                            zv[k] = rv[k] * dt;
                        }
                        cc_put<VEC>(r + (size_t)l * VEC, rv);
                        cc_put<VEC>(z0s + (size_t)(cur * rpc + l) * VEC, zv);
                        cc_put<VEC>(dd + (size_t)l * VEC, zv);
                    }
                    cc_sync();
                }
                W rho_c = de / th;
                for (int st = 1; st < g.deg; ++st) {
                    const W rn = W(1) / (W(2) * th / de - rho_c), c1 = rn * rho_c, c2 = W(2) * rn / de;
                    rho_c = rn;
                    const bool last = st + 1 == g.deg;
#pragma unroll
                    for (int k = 0; k < VEC; ++k) v1[0][k] = W(0);
                    for (int l = tid; l < cnt; l += nt) {
                        W wv[VEC], rv[VEC], zv[VEC], tv[VEC];
                        cc_get<VEC, false>(rv, r + (size_t)l * VEC);
                        cc_get<VEC, false>(tv, dd + (size_t)l * VEC);
                        cc_get<VEC, false>(zv, z0s + (size_t)(cur * rpc + l) * VEC);
                        const W di = c2 * dtab[l];
                        apply(l, wv);
#pragma unroll
                        for (int k = 0; k < VEC; ++k) {
                            tv[k] = cc_fma(di, rv[k] - wv[k], c1 * tv[k]);
                            zv[k] += tv[k];
                            v1[0][k] = cc_fma(rv[k], zv[k], v1[0][k]);
                        }
                        cc_put<VEC>(dd + (size_t)l * VEC, tv);
                        cc_put<VEC>(z0s + (size_t)((cur ^ 1) * rpc + l) * VEC, zv);
                    }
                    if (!last) cc_sync();
                    cur ^= 1;
                }
                reduce(v1, 0);   // r.z
                if (tid < VEC) {
                    const double rho = out[tid];
                    s_ab[tid] = (it == 0 || s_flag[tid]) ? W(0) : W(rho) / W(s_rhop[tid]);
                    s_rho[tid] = rho;
                }
                __syncthreads();
                // ---- A ---------------------------------------------------------------
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    ab[k] = s_ab[k];
                    v1[0][k] = W(0);
                }
                for (int l = tid; l < cnt; l += nt) {
                    W zv[VEC], wv[VEC], pv[VEC], qv[VEC];
                    cc_get<VEC, false>(zv, z0s + (size_t)(cur * rpc + l) * VEC);
                    if (it) {
                        cc_get<VEC, false>(pv, p + (size_t)l * VEC);
                        cc_get<VEC, false>(qv, q + (size_t)l * VEC);
                    } else {
#pragma unroll
                        for (int k = 0; k < VEC; ++k) pv[k] = qv[k] = W(0);
                    }
                    const bool frozen = dtab[l] == W(0);
                    apply(l, wv);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        pv[k] = cc_fma(ab[k], pv[k], zv[k]);
                        qv[k] = frozen ? W(0) : cc_fma(ab[k], qv[k], wv[k]);
                        v1[0][k] = cc_fma(pv[k], qv[k], v1[0][k]);
                    }
                    cc_put<VEC>(p + (size_t)l * VEC, pv);
                    cc_put<VEC>(q + (size_t)l * VEC, qv);
                }
                reduce(v1, 0);   // p.q
                if (tid < VEC) s_ab[tid] = s_flag[tid] ? W(0) : W(s_rho[tid]) / W(out[tid]);
                __syncthreads();
                // ---- B, and the first step of the next polynomial -------------------------
                W u[2][VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    ab[k] = s_ab[k];
                    u[0][k] = u[1][k] = W(0);
                }
                for (int l = tid; l < cnt; l += nt) {
                    W rv[VEC], dv[VEC], pv[VEC], qv[VEC], zv[VEC];
                    if (it) cc_get<VEC, false>(dv, d + (size_t)l * VEC);
                    else
#pragma unroll
                        for (int k = 0; k < VEC; ++k) dv[k] = W(0);
                    cc_get<VEC, false>(pv, p + (size_t)l * VEC);
                    cc_get<VEC, false>(rv, r + (size_t)l * VEC);
                    cc_get<VEC, false>(qv, q + (size_t)l * VEC);
                    const W dt = dtab[l] / th;
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        dv[k] = cc_fma(ab[k], pv[k], dv[k]);
                        rv[k] = cc_fma(-ab[k], qv[k], rv[k]);
                        zv[k] = rv[k] * dt;
                        u[0][k] = cc_fma(rv[k], rv[k], u[0][k]);
                        u[1][k] += rv[k];
                    }
                    cc_put<VEC>(d + (size_t)l * VEC, dv);
                    cc_put<VEC>(r + (size_t)l * VEC, rv);
                    // the other copy: this one may still be read by the neighbours' products
                    cc_put<VEC>(z0s + (size_t)((cur ^ 1) * rpc + l) * VEC, zv);
                    cc_put<VEC>(dd + (size_t)l * VEC, zv);
                }
                cur ^= 1;
                reduce(u, 0);
            }
            // fold the cycle's correction into x before anything reads x
            for (int l = tid; it > 0 && l < cnt; l += nt) {
                W dv[VEC];
                cc_get<VEC, false>(dv, d + (size_t)l * VEC);
                T xv[VEC];
                T* xp = x + (size_t)(lo + l) * C + c0;
                cc_get<VEC, true>(xv, xp);
#pragma unroll
                for (int k = 0; k < VEC; ++k) xv[k] += T(dv[k]);
                cc_put<VEC>(xp, xv);
            }
            cc_sync();
            if constexpr (!MP) {
                break;
            } else {
                // done when every system met the tolerance on its true residual at the
                // start of this cycle (or ran out of iterations or cycles)
                if (__syncthreads_and(tid < VEC ? s_done[tid] : 1) || cycle + 1 >= MP_MAX_CYCLES) break;
            }
        }
        // epilogue: Neumann systems are gauged to zero V-weighted mean and (stage 1)
        // hand u1_S to the BEM product; stage-1 Dirichlet (adjoint) systems hand
        // t = b_S - K_SI w (w vanishes on the surface, so K_SI w = (K w)_S)
        if (neu) {
            double pv[1][VEC];
#pragma unroll
            for (int k = 0; k < VEC; ++k) pv[0][k] = 0.0;
            for (int row = lo + tid; row < hi; row += nt) {
                const double vi = P.M.gV[row];
                T xv[VEC];
                cc_get<VEC, true>(xv, x + (size_t)row * C + c0);
#pragma unroll
                for (int k = 0; k < VEC; ++k) pv[0][k] = fma(vi, (double)xv[k], pv[0][k]);
            }
            reduce(pv, 0);
            T mean[VEC];
#pragma unroll
            for (int k = 0; k < VEC; ++k) mean[k] = T(out[k] / P.M.vsum);
            for (int row = lo + tid; row < hi; row += nt) {
                const int bp = (int)((unsigned)P.M.node[row] >> 16);
                T xv[VEC];
                cc_get<VEC, true>(xv, x + (size_t)row * C + c0);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    if (!act[k]) continue;
                    xv[k] -= mean[k];
                    if (mode == 0 && bp) P.V.ub_in[(size_t)(bp - 1) * C + c0 + k] = xv[k];
                }
                cc_put<VEC>(x + (size_t)row * C + c0, xv);
            }
        } else if (mode == 0) {
            const T* kvT = GenTab<T>::k(P.M);
            for (int row = lo + tid; row < hi; row += nt) {
                const int bp = (int)((unsigned)P.M.node[row] >> 16);
                if (!bp) continue;
                T kw[VEC];
                double f[VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) kw[k] = T(0);
                for (int e = P.M.kptr[row]; e < P.M.kptr[row + 1]; ++e) {
                    T xj[VEC];
                    cc_get<VEC, true>(xj, x + (size_t)((unsigned)__ldg(&P.M.kent[e]) >> 8) * C + c0);
                    const T kv = __ldg(&kvT[e]);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) kw[k] = cc_fma(kv, xj[k], kw[k]);
                }
                cc_get<VEC, false>(f, P.V.bvec + (size_t)row * B + b0);
#pragma unroll
                for (int k = 0; k < VEC; ++k)
                    if (act[k]) P.V.ub_in[(size_t)(bp - 1) * C + c0 + k] = T(f[k]) - kw[k];
            }
        }
        if (rank == 0 && tid < VEC)
            atomicAdd((unsigned long long*)(neu ? &P.V.st[b0 + tid].cg1 : &P.V.st[b0 + tid].cg2),
                      (unsigned long long)s_it[tid]);
        for (int k = 0; k < VEC; ++k) itmax = max(itmax, s_it[k]);
    }
    // sweep counter: the largest iteration count of the launch (the last cluster
    // to finish adds it and clears the two counter words)
    if (rank == 0 && tid == 0) {
        atomicMax(&P.bar[2], (unsigned)itmax);
        __threadfence();
        if (atomicAdd(&P.bar[3], 1u) == gridDim.x / g.cl - 1) {
            __threadfence();
            const unsigned km = atomicExch(&P.bar[2], 0u);
            atomicExch(&P.bar[3], 0u);
            if (P.sweeps) P.sweeps[mode + (sizeof(T) == 8 ? 2 : 0)] += (unsigned long long)km;
        }
    }
    cc_sync();   // no CTA leaves while another may still read its shared memory
}

struct CcChoice {
    CcGeo g;
    int vec = 0, threads = 0, waves = 0;
};

// Shared memory of a shape; false when not even z fits.
bool cc_fit(CcGeo& g, int vec, size_t word, int entries, size_t bare) {
    auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
    const size_t scr = up(std::max(word * 32 * CC_NQ * vec, sizeof(double) * 32 * vec));
    const size_t slot = up(sizeof(double) * 2 * CC_NQ * vec * CC_MAX_CL);
    const size_t col = up(sizeof(double) * (CC_NQ + 6) * vec + sizeof(int) * 3 * vec + 4 * CC_MAX_CL);
    const size_t one = word * vec * (size_t)g.rpc, di = up(word * (size_t)g.rpc), fixed = scr + slot + col + di;
    if (up(2 * one) + fixed > CC_SMEM_MAX) return false;
    g.nvec = g.fit = (int)std::min<size_t>(CC_VECS, (CC_SMEM_MAX - fixed - 16) / one);
    size_t o = up(one * g.nvec);
    g.o_dinv = (unsigned)o;
    o += di;
    g.ent = 0;
    g.o_ent = g.o_ptr = (unsigned)o;
    if (entries > 0 && g.nvec >= 4) {
        const size_t e = up((4 + word) * (size_t)entries), pt = up(4 * ((size_t)g.rpc + 1));
        if (o + e + pt + fixed - di <= CC_SMEM_MAX) {
            g.ent = entries;
            o += e;
            g.o_ptr = (unsigned)o;
            o += pt;
        }
    }
    if (!g.ent) {
        while (g.nvec > 3 && up(one * g.nvec) + fixed + 16 > bare) --g.nvec;
        o = up(one * g.nvec);
        g.o_dinv = (unsigned)o;
        o += di;
        g.o_ent = g.o_ptr = (unsigned)o;
    }
    g.o_scr = (unsigned)o;
    o += scr;
    g.o_slot = (unsigned)o;
    o += slot;
    g.o_col = (unsigned)o;
    o += col;
    g.smem = (unsigned)o;
    // j / rpc for 0 <= j < 2^31 by a multiplication: mul = ceil(2^(32 + s) / rpc) with 2^s < rpc <= 2^(s + 1)
    int s = 0;
    while ((1u << (s + 1)) < (unsigned)g.rpc) ++s;
    g.shift = (unsigned)s;
    if (g.rpc < 2) return false;
    g.mul = (unsigned)((((uint64_t)1 << (32 + s)) + g.rpc - 1) / g.rpc);
    return o <= CC_SMEM_MAX;
}

template <typename T, typename W, int VEC>
int cc_resident(const CcGeo& g, int threads) {
    auto fn = k_cluster_cg<T, W, VEC>;
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, unsigned>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_tuple(dev, g.cl, threads, g.smem);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int ncl = 0;
    if (kernel_smem_attr((const void*)fn, (int)CC_SMEM_MAX) == cudaSuccess &&
        cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)g.cl);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = g.smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)g.cl;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&ncl, (const void*)fn, &cfg) != cudaSuccess) ncl = 0;
    }
    cudaGetLastError();
    cache.emplace(key, ncl);
    return ncl;
}

// rows: of a system; cols: systems; emax[cl]: most matrix entries of a CTA when the
// rows are dealt to cl CTAs
template <typename T, typename W, int VEC>
void cc_try(int rows, int cols, const int* emax, CcChoice& best, double& best_cost) {
    if ((cols / 2) % VEC) return;
    for (int cl = CC_MAX_CL; cl >= 1; cl = cl > 8 ? cl - 2 : cl / 2) {
        CcGeo g = {};
        g.rows = rows;
        g.cl = cl;
        g.rpc = (rows + cl - 1) / cl;
        if (g.rpc < 32 && cl > 1) continue;
        g.cl = (rows + g.rpc - 1) / g.rpc;   // every CTA has rows
        if (!cc_fit(g, VEC, sizeof(W), emax[cl], CC_SMEM_BARE<W>)) continue;
        const int most = sizeof(W) == 8 ? 512 : 1024, per = (g.rpc + most - 1) / most;
        const int threads = std::min(most, std::max(128, ((g.rpc + per - 1) / per + 31) & ~31));
        if (g.nvec < 3) continue;   // dd has no global room
        cc_degree(rows, g.deg, g.ratio);
        const int r = cc_resident<T, W, VEC>(g, threads);
        if (r < 1) continue;
        const int waves = (cols / VEC + r - 1) / r;
        // an iteration's time in rows of a thread block: the rows' vectors (twice as
        // dear in global memory, unless they went there for the L1's sake), their matrix
        // entries, and barriers and latencies worth about 3000 rows
        const double mat = g.ent ? 2.0 : 6.0;
        const double cost = waves * (g.rpc * (VEC * (1.0 + 0.25 * (CC_VECS - g.fit)) * (sizeof(W) == 8 ? 24.0 : 1.0) + mat) + 3000.0);
        if (best.vec == 0 || cost < best_cost) {
            best_cost = cost;
            best.g = g;
            best.vec = VEC;
            best.threads = threads;
            best.waves = waves;
        }
    }
}

// Where the Jacobi-CG kernels, which spread a product over the whole chip, are faster: many
// systems in plain FP64, whose clusters run in waves (the polynomial takes about a quarter
// more products, and FP64 units are what bounds both), and the largest meshes (a system has
// sixteen SMs and its entries come from global memory).  ms an evaluation here / there, plain
// FP64, systems a cluster by waves: 2 by 5, 64 instances on 3 375 nodes 17.4 / 12.6; 2 by 3,
// 96 on 1 331 8.6 / 7.5, 40 on 12 167 44.0 / 38.0, 20 on 29 791 71 / 62, but 20 on 12 167 23.7 /
// 27.3, 40 on 4 913 14.6 / 15.6; 2 by 4, 48 on 3 375 13.9 / 13.3 (as its instances finish, a
// minimisation is faster here); 1 by 3, 9 on 19 683 25.5 / 28.4, on 29 791 39.6 / 39.5, 8 on
// 46 656 62 / 55, on 50 653 70 / 64; 1 by 4, 25 on 9 261 20.3 / 24.4, 24 on 24 389 59.9 /
// 57.3; one or two waves 1.0 to 2.3 times faster here over 60 such shapes of 343 to 42 875
// nodes; one on 74 088 46.7 / 37.5, on 59 319 36.7 / 34.5.  Iterated in FP32: one on 74 088 26.5
// / 25.8, on 91 125 33.5 / 31.8, five 61 / 44, one on 166 375 99 / 44.  FP32 solves stay here at
// any size: there Jacobi-CG of one reduction a product does not always come to its tolerance
// (fields off by 1.4e-6 here and up to 2e-5 there for one instance on 117 649 nodes, 1e-2 for
// five, after 5000 iterations; on 166 375 45 ms here, 23 there, both within 2e-6).
bool cc_slower(int rows, int cols, int vec, int waves, bool fp32, bool fp64_vectors) {
    if (fp32) return false;
    if (!fp64_vectors) return rows > 80000;
    const bool wide = cols >= 100 || rows >= 14000 || (cols >= 80 && rows >= 10000);
    return rows > 65000 || waves >= 5 || (wide && waves >= (vec == 2 ? 3 : 4)) || (rows >= 45000 && waves >= 3);
}

template <typename T, typename W>
CcChoice cc_choose(int rows, int cols, const int* emax) {
    CcChoice c;
    double cost = 0.0;
    if constexpr (sizeof(W) == 4) cc_try<T, W, 4>(rows, cols, emax, c, cost);
    cc_try<T, W, 2>(rows, cols, emax, c, cost);
    cc_try<T, W, 1>(rows, cols, emax, c, cost);
    if (cc_slower(rows, cols, c.vec, c.waves, sizeof(T) == 4, sizeof(W) == 8)) c.vec = 0;
    return c;
}

template <typename T, typename W, int VEC>
cudaError_t cc_launch(const Launch& L, const CcArgs<T, W>& a, const CcChoice& c, int cols) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cols / VEC * c.g.cl));
    cfg.blockDim = dim3((unsigned)c.threads);
    cfg.dynamicSmemBytes = c.g.smem;
    cfg.stream = L.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)c.g.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_cluster_cg<T, W, VEC>, a);
}

template <typename T, typename W>
cudaError_t cc_launch_vec(const Launch& L, const CcArgs<T, W>& a, const CcChoice& c, int cols) {
    if constexpr (sizeof(W) == 4)
        if (c.vec == 4) return cc_launch<T, W, 4>(L, a, c, cols);
    if (c.vec == 2) return cc_launch<T, W, 2>(L, a, c, cols);
    return cc_launch<T, W, 1>(L, a, c, cols);
}

template <typename T, typename W>
cudaError_t cc_fem(const Launch& L, const MeshView& M, const BatchView<T>& V, const PcgArgs<T>& P, bool* ok) {
    const int cols = 2 * V.B;
    const CcChoice c = cc_choose<T, W>(M.N, cols, M.emax);
    *ok = c.vec != 0;
    if (!c.vec) return cudaSuccess;
    CcArgs<T, W> a = {};
    a.P = P;
    a.g = c.g;
    // b: a bound of the eigenvalues of D^-1 K
    a.g.th = 0.5 * (1.0 + 1.0 / c.g.ratio) * M.jac_bound;
    a.g.de = 0.5 * (1.0 - 1.0 / c.g.ratio) * M.jac_bound;
    // z, z' and dd are in shared memory (cc_try); r, p, q, d have the batch's work vectors
    a.v[1] = reinterpret_cast<W*>(V.r);
    a.v[2] = reinterpret_cast<W*>(V.p);
    a.v[3] = reinterpret_cast<W*>(V.q);
    a.v[4] = reinterpret_cast<W*>(V.z);
    return cc_launch_vec<T, W>(L, a, c, cols);
}

}  // namespace

bool cluster_cg_takes(const Launch& L, const MeshView& M, int B, bool fp64, bool mixed_iter) {
    // (a cap on the blocks, L.max_blocks, comes with served cubes only; the other kernels keep to it)
    if (!M.gen || L.pcg_kernel != 0 || L.wait_test || L.max_blocks > 0) return false;
    if (!fp64) return cc_choose<float, float>(M.N, 2 * B, M.emax).vec != 0;
    return (mixed_iter ? cc_choose<double, float>(M.N, 2 * B, M.emax) : cc_choose<double, double>(M.N, 2 * B, M.emax)).vec != 0;
}

// General meshes: 1 when launched (*err its status), 0 when the cluster shapes do
// not take it (z of a system exceeds a cluster's shared memory).
template <typename T>
int cluster_cg_fem(const Launch& L, const MeshView& M, const BatchView<T>& V, int mode, double tol, int max_iter,
                   bool mixed_iter, cudaError_t* err) {
    *err = cudaSuccess;
    if (!M.gen || L.pcg_kernel != 0 || L.wait_test || L.max_blocks > 0) return 0;
    PcgArgs<T> P{M, V, mode, tol * tol, max_iter, L.bar, L.err, L.sweeps, L.fin};
    bool ok = false;
    if constexpr (sizeof(T) == 4) *err = cc_fem<T, float>(L, M, V, P, &ok);
    else if (mixed_iter) *err = cc_fem<T, float>(L, M, V, P, &ok);
    else *err = cc_fem<T, double>(L, M, V, P, &ok);
    if (!ok && *err == cudaSuccess) return 0;
    *L.launches += 1;
    return 1;
}

template int cluster_cg_fem<float>(const Launch&, const MeshView&, const BatchView<float>&, int, double, int, bool,
                                   cudaError_t*);
template int cluster_cg_fem<double>(const Launch&, const MeshView&, const BatchView<double>&, int, double, int, bool,
                                    cudaError_t*);

}  // namespace lbm
