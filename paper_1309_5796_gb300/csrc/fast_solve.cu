// Potential solves (Table 2 "solve linear system"; Sec. 3.1 "magnetic scalar
// potential") on Kuhn cubes: fast diagonalisation with iterative refinement.
//
// On the Kuhn cube the P1 stiffness couples a node only to its six axis
// neighbours.  Inside the cube every coupling is -6 (units h/6) and on a face
// -3, as for the tensor product of 1-D operators
//     K_T = 6 (L x W x W + W x L x W + W x W x L),
// L the 1-D second difference, W = diag(1/2, 1, ..., 1, 1/2); only along the
// cube's twelve edges is it -2 or -1 where K_T has -1.5: K = K_T + E, E on the
// 12n - 4 edge nodes only.  With zero boundary values (interior rows) E = 0.
// K_T is inverted exactly by three small dense transforms (cosines, or sines
// with zero boundary values), a scaling, and the three transforms back:
//     K_T^+ r = (Q x Q x Q) diag(1 / 6(l_a + l_b + l_c)) (Q x Q x Q)^T r,
// L q = l W q, Q^T W Q = 1 (Lynch, Rice, Thomas 1964).  Every eigenvector is
// even or odd about the cube's centre, so a transform of n+1 values is one of
// half that length on v[k] + v[n-k] and one on v[k] - v[n-k].
//
// Refinement: z = K_T^+ rhs, x += z, r -= K z.  Dirichlet systems: rhs = r, one
// step reaches rounding.  Neumann systems take steps in pairs: rhs = r, then
// rhs = r + H z on the edge nodes with z of the step before, where
//     H = E - G,  G = E (1 + R E)^-1,  R = K_T^+ restricted to the edge nodes:
// by the Woodbury identity K^+ = K_T^+ - K_T^+ G K_T^+, so a pair reaches rounding.
// A solve thus takes 1 (Dirichlet) or 2 (Neumann) steps at any size and
// tolerance, and more only when rounding calls for it (FP32 far below 1e-6);
// diagonally preconditioned CG takes 100 to 700.
//
// Measured on GB300 (two stages of both chains, FP64 n = 10 / FP32 n = 20, 80, one
// instance / FP32 n = 30, 64 instances, before: diagonally preconditioned CG):
// 0.11 / 0.14 / 1.57 / 0.77 ms, before 6.1 / 5.6 / 36 / 12 ms.
//
// One thread-block cluster solves VEC systems (columns of the [N][2B] layout)
// of one kind; CTA r owns the z-planes [r ppc, (r+1) ppc).  Per step:
//   P1  fold the right-hand side, x and y transforms of the own planes
//   P2  z transform, scaling, z transform back, for the CTA's share of the
//       (y', x') positions, gathered from and scattered to all CTAs
//   P3  y and x transforms back, unfold: z on the own planes
//   P4  x += z, r -= K z (stencil); Neumann: H z after the first of a pair
// with a hardware cluster barrier after each.  The transformed planes stay in
// the CTAs' shared memory (TS; the z transform reads the other CTAs' by
// distributed shared memory) and, for cubes too large for that, in global
// memory.
//
// A result does not depend on how many systems share a cluster, how many CTAs
// it has or how many threads they run: every sum is taken per chunk of 32
// quadruples of mirrored nodes of one plane (small cubes in FP64: of 8, a lane
// per node), then over
// the chunks of a plane, then over the planes, each in a fixed order.
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "solver_common.cuh"

namespace lbm {
namespace {

constexpr size_t FS_SMEM_MAX = 226 * 1024;   // dynamic; the rest of the 227 KB is static
constexpr int FS_MAX_N1 = 97;       // largest cube: 96 cells
constexpr int FS_NQ = 5;            // most quantities of one reduction
constexpr int FS_NODE_H = 9;        // FP64: largest half side with a lane per node (n <= 17)
constexpr int FS_MAX_CL = 16;
constexpr int FS_SPLIT = 8;         // parts of a row of H

extern __shared__ __align__(16) unsigned char fs_sm[];

__device__ __forceinline__ unsigned cl_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_index() {
    unsigned r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
// All threads of all CTAs of the cluster, release/acquire at cluster scope.
__device__ __forceinline__ void cl_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t sm_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// generic address of p in the CTA `rank` of the cluster
template <typename X>
__device__ __forceinline__ X* peer_ptr(X* p, unsigned rank) {
    X* r;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(p), "r"(rank));
    return r;
}
__device__ __forceinline__ double ld_peer1(uint32_t a, double) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_peer1(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_peer1(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// four consecutive values (16-byte aligned)
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double* p, const double (&v)[4]) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }

// VEC consecutive columns of one row; CG: through L2 (values other CTAs write)
template <int VEC, bool CG, typename X>
__device__ __forceinline__ void ldc(X (&d)[VEC], const X* p) {
    if constexpr (VEC == 1) d[0] = CG ? __ldcg(p) : *p;
    else vload<X, VEC, CG>(d, p);
}
template <int VEC, typename X>
__device__ __forceinline__ void stc(X* p, const X (&d)[VEC]) {
    if constexpr (VEC == 1) *p = d[0];
    else vstore<X, VEC>(p, d);
}

// Stiffness weight (units h/6) of the axis edges whose other two coordinates
// are (a, b): 2 from a cell that has the edge at its (low, low) or (high, high)
// corner, 1 otherwise; 6 inside, 3 on a face, 2 or 1 on the cube's edges.
__device__ __forceinline__ int edge_weight(int a, int b, int n) {
    const int la = a > 0, ha = a < n, lb = b > 0, hb = b < n;
    return 2 * ((ha & hb) + (la & lb)) + (ha & lb) + (la & hb);
}

// Sizes of a launch (see choose()).
struct FsGeo {
    // n+1 = s2; even/odd halves h, ho, padded to multiples of 4 (hp, hop); a sheet
    // is one plane of one system, s2 rows of ldx = hp + hop: x < h at column x, x >= h
    // at column x + hp - h (zeros in the gap).  Folded, the even part of a mirrored
    // pair (k, n-k) stands at k, the odd one at n-k, so folding is in place
    int n, s2, h, ho, hp, hop, ldx, ss;
    int cl, ppc;                          // CTAs per cluster, planes per CTA
    int nch;                              // chunks of a plane's sums: 32 quadruples, small cubes in FP64 8
    int zc, pr;                           // positions per CTA in P2, and per round of them
    int spl;                              // TS = false: planes per round of P1 and P3
    int matw;                             // words of one kind's transform matrices
    int ne, er;                           // edge nodes, rows of H per CTA
    int vs;                               // 1: r and d in shared memory
    unsigned o_z, o_mat, o_part, o_slot, o_edge, o_vec, o_col, smem;   // shared-memory offsets (bytes)
};

template <typename T, typename W>
struct FsArgs {
    PcgArgs<T> P;
    FsGeo g;
    const W* mat;      // [2 kinds][F_e | G_e | F_o | G_o], F[point][mode], G = F^T, rows padded to 4
    const W* inv;      // [2 kinds][s2 modes][ss] 1 / 6(l_a + l_b + l_c) (0: no such mode, or the constant)
    const W* edge;     // [ne][ne] H (symmetric)
    W* gt;             // TS = false: [group][s2][VEC][ss]
    int first, clusters;   // this launch's first cluster, and those of all launches of the solve
};

// Register tile of the transforms: rows x columns per thread.  FP32: 4 x 4, so
// that two 16-byte shared loads feed sixteen FMAs.  FP64 issues at 1/64 of the
// FP32 rate, so loads never bound it; 1 x 2 spreads a small plane's products
// over more warps (n = 10: one warp held all of a 4 x 4 tiling).
template <typename W> struct FsTile;
template <> struct FsTile<float> { static constexpr int R = 4, C = 4; };
template <> struct FsTile<double> { static constexpr int R = 1, C = 2; };
template <int K> __device__ __forceinline__ void ldk(const float* p, float (&v)[K]) {
    static_assert(K == 4, "");
    ld4(p, v);
}
template <int K> __device__ __forceinline__ void ldk(const double* p, double (&v)[K]) {
    static_assert(K == 1 || K == 2, "");
    if constexpr (K == 1) v[0] = *p;
    else {
        const double2 a = *reinterpret_cast<const double2*>(p);
        v[0] = a.x; v[1] = a.y;
    }
}
template <int K> __device__ __forceinline__ void stk(float* p, const float (&v)[K]) { st4(p, v); }
template <int K> __device__ __forceinline__ void stk(double* p, const double (&v)[K]) {
    if constexpr (K == 1) *p = v[0];
    else *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}

// In place, on `nsheets` sheets at shared offset o: every row times the
// block-diagonal matrix (Me, Mo), out[row][m'] = sum_m v[row][m] M[m][m'].  A
// thread holds one tile of a round of lines (a line: TR rows, all column tiles)
// in registers until every thread has read its operands.
template <typename W>
__device__ __noinline__ void pass_right(unsigned o, int nsheets, unsigned oe, unsigned oo, int s2, int hp, int hop) {
    constexpr int TR = FsTile<W>::R, TC = FsTile<W>::C;
    W* sh = reinterpret_cast<W*>(fs_sm + o);
    const int ldx = hp + hop, ss = s2 * ldx;
    const int te = hp / TC, ct = te + hop / TC, rt = (s2 + TR - 1) / TR;
    const int lines = nsheets * rt, lr = (int)blockDim.x / ct;
    const int dl = (int)threadIdx.x / ct, t = (int)threadIdx.x - dl * ct;
    const bool even = t < te;
    const int c0 = even ? 0 : hp, K = even ? hp : hop, tt = (even ? t : t - te) * TC;
    const W* M = reinterpret_cast<const W*>(fs_sm + (even ? oe : oo)) + tt;
    for (int l0 = 0; l0 < lines; l0 += lr) {
        const int line = l0 + dl;
        const bool on = dl < lr && line < lines;
        W acc[TR][TC];
        W* dst = nullptr;
        int r0 = 0;
        if (on) {
            const int sheet = line / rt;
            r0 = (line - sheet * rt) * TR;
            W* base = sh + sheet * ss + c0;
            const W* row[TR];
#pragma unroll
            for (int r = 0; r < TR; ++r) row[r] = base + min(r0 + r, s2 - 1) * ldx;
#pragma unroll
            for (int r = 0; r < TR; ++r)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[r][j] = W(0);
            for (int m = 0; m < K; m += 4) {
                W a[TR][4];
#pragma unroll
                for (int r = 0; r < TR; ++r) ld4(row[r] + m, a[r]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    W b[TC];
                    ldk<TC>(M + (m + q) * K, b);
#pragma unroll
                    for (int r = 0; r < TR; ++r)
#pragma unroll
                        for (int j = 0; j < TC; ++j) acc[r][j] = fma_(a[r][q], b[j], acc[r][j]);
                }
            }
            dst = base + tt;
        }
        __syncthreads();
        if (on)
#pragma unroll
            for (int r = 0; r < TR; ++r)
                if (r0 + r < s2) stk<TC>(dst + (r0 + r) * ldx, acc[r]);
        __syncthreads();
    }
}

// In place: the block-diagonal (Me, Mo) applied along the rows' index,
// out[m'][x] = sum_m M[m][m'] v[m][x], rows [0, h) the even part, [h, s2) the
// odd one; ld columns a row (a multiple of 4), nsheets sheets of s2 rows.
// inv (or null): out[m'][x] *= inv[m' ss + x % pc].
template <typename W>
__device__ __noinline__ void pass_left(unsigned o, int nsheets, int ld, unsigned oe, unsigned oo, int s2, int hp, int hop,
                                       const W* __restrict__ inv, int pc) {
    constexpr int TR = FsTile<W>::R, TC = FsTile<W>::C;
    W* sh = reinterpret_cast<W*>(fs_sm + o);
    const int h = (s2 + 1) >> 1, ho = s2 >> 1, ssl = s2 * ld, ss = s2 * (hp + hop);
    const int te = (h + TR - 1) / TR, rt = te + (ho + TR - 1) / TR, ct = ld / TC;
    const int lines = nsheets * ct, lr = min((int)blockDim.x / rt, lines);
    const int rr = (int)threadIdx.x / lr, dl = (int)threadIdx.x - rr * lr;
    const bool even = rr < te;
    const int K = even ? h : ho, ldm = even ? hp : hop, tt = (even ? rr : rr - te) * TR, row0 = (even ? 0 : h);
    const W* M = reinterpret_cast<const W*>(fs_sm + (even ? oe : oo)) + tt;
    for (int l0 = 0; l0 < lines; l0 += lr) {
        const int line = l0 + dl;
        const bool on = rr < rt && line < lines;
        W acc[TR][TC];
        W* dst = nullptr;
        int x0 = 0;
        if (on) {
            const int sheet = line / ct;
            x0 = (line - sheet * ct) * TC;
            dst = sh + sheet * ssl + row0 * ld + x0;
            const W* v = dst;
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = W(0);
#pragma unroll 4
            for (int m = 0; m < K; ++m) {
                W a[TR], b[TC];
                ldk<TR>(M + m * ldm, a);
                ldk<TC>(v + m * ld, b);
#pragma unroll
                for (int i = 0; i < TR; ++i)
#pragma unroll
                    for (int j = 0; j < TC; ++j) acc[i][j] = fma_(a[i], b[j], acc[i][j]);
            }
        }
        __syncthreads();
        if (on)
#pragma unroll
            for (int i = 0; i < TR; ++i)
                if (tt + i < K) {
                    if (inv) {
                        W w[TC];
                        ldk<TC>(inv + (size_t)(row0 + tt + i) * ss + x0 % pc, w);
#pragma unroll
                        for (int j = 0; j < TC; ++j) acc[i][j] *= w[j];
                    }
                    stk<TC>(dst + (tt + i) * ld, acc[i]);
                }
        __syncthreads();
    }
}

// The edge nodes: the four lines along x with their ends, then the four along y
// and the four along z without.
__device__ __forceinline__ int edge_index(int i, int j, int k, int n) {   // -1: not on an edge
    const bool bi = i == 0 || i == n, bj = j == 0 || j == n, bk = k == 0 || k == n;
    if (bj && bk) return ((j != 0) + 2 * (k != 0)) * (n + 1) + i;
    if (bi && bk) return 4 * (n + 1) + ((i != 0) + 2 * (k != 0)) * (n - 1) + j - 1;
    if (bi && bj) return 4 * (n + 1) + 4 * (n - 1) + ((i != 0) + 2 * (j != 0)) * (n - 1) + k - 1;
    return -1;
}
__device__ __forceinline__ void edge_node(int e, int n, int& i, int& j, int& k) {
    if (e < 4 * (n + 1)) {
        const int l = e / (n + 1);
        i = e - l * (n + 1);
        j = (l & 1) ? n : 0;
        k = (l & 2) ? n : 0;
        return;
    }
    e -= 4 * (n + 1);
    const bool y = e < 4 * (n - 1);
    if (!y) e -= 4 * (n - 1);
    const int l = e / (n - 1), t = e - l * (n - 1) + 1, b0 = (l & 1) ? n : 0, b1 = (l & 2) ? n : 0;
    i = b0;
    j = y ? t : b1;
    k = y ? b1 : t;
}

// T: type of the potential x and of the residual f - K x; W: type of the
// refinement (transforms, r, the sum of the steps) and of a step's dot products inside
// a chunk (sums over chunks, planes and CTAs in FP64; those of the first residual, of its
// reference and of the gauge in FP64 or pairs (SumOf) from the node on).  T = W: d starts as x and
// collects the steps; the first residual's stencil runs on a copy of x in the
// planes' place, so x is read once and written once (a system's values lie 2B words
// apart in it).  T = double, W = float (solves iterated in FP32): cycles of the FP64
// residual and FP32 refinement until it has reduced that residual by MP_INNER; the
// solve ends on the FP64 residual test.  Neumann systems (forward in mode 0,
// adjoint in mode 1): residual taken without its mean (consistent right-hand
// side), solution gauged to zero V-weighted mean.  Dirichlet systems: surface
// values frozen.
template <typename T, typename W, int VEC, bool TS>
__global__ void __launch_bounds__(sizeof(W) == 8 ? 512 : 1024, 1) k_fast_solve(const __grid_constant__ FsArgs<T, W> A) {
    constexpr bool MP = sizeof(T) != sizeof(W), ND = sizeof(W) == 8;
    const FsGeo& g = A.g;
    W* buf = reinterpret_cast<W*>(fs_sm);                       // TS: own planes [ppc][VEC][ss]; else a round of planes
    W* zb = reinterpret_cast<W*>(fs_sm + g.o_z);                // P2: [s2][VEC * pr] (TS = false: in buf's room)
    double* part = reinterpret_cast<double*>(fs_sm + g.o_part);   // [ppc][nch][FS_NQ][VEC]
    double* slots = reinterpret_cast<double*>(fs_sm + g.o_slot);  // [2][ppc][FS_NQ][VEC]
    W* ec = reinterpret_cast<W*>(fs_sm + g.o_edge);             // [ne][VEC] H z at the edge nodes (own planes' valid)
    W* ev = ec + g.ne * VEC;                                    // [ne][VEC] z at the edge nodes
    W* ep = ev + g.ne * VEC;                                    // [er][FS_SPLIT][VEC] partial products
    double* out = reinterpret_cast<double*>(fs_sm + g.o_col);     // [FS_NQ][VEC]
    double* s_tol = out + FS_NQ * VEC;
    double* s_tin = s_tol + VEC;
    double* s_mean = s_tin + VEC;
    W** s_plane = reinterpret_cast<W**>(s_mean + VEC);            // [s2] every plane's sheets (peers' shared memory, or gt)
    uint32_t* s_slot = reinterpret_cast<uint32_t*>(s_plane + FS_MAX_N1);   // [s2] its partial sums (slot 0)
    int* s_flag = reinterpret_cast<int*>(s_slot + FS_MAX_N1);
    int* s_it = s_flag + VEC;
    int* s_done = s_it + VEC;
    __shared__ int s_grp;

    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const unsigned rank = cl_rank();
    const int B = A.P.V.B, C = 2 * B, n = g.n, s2 = g.s2, N = A.P.M.N, mode = A.P.mode;
    const int ss = g.ss, ldx = g.ldx, h = g.h, ho = g.ho, hp = g.hp, hop = g.hop;
    const int gap = hp - h, pn = s2 * s2;

    // the cluster's group of VEC systems: the k-th one with an active instance
    if (warp == 0) {
        const int ng = C / VEC, want = A.first + (int)cl_index();
        int found = -1, cnt = 0;
        for (int base = 0; base < ng; base += 32) {
            bool a = false;
            if (base + lane < ng)
                for (int i = 0; i < VEC; ++i) a |= A.P.V.st[((base + lane) * VEC + i) % B].phase != PH_DONE;
            unsigned bal = __ballot_sync(0xffffffffu, a);
            const int pc = __popc(bal);
            if (found < 0 && want < cnt + pc) {
                for (int k = cnt; k < want; ++k) bal &= bal - 1u;
                found = base + __ffs(bal) - 1;
            }
            cnt += pc;
        }
        if (lane == 0) {
            s_grp = found;
            if (rank == 0 && want == 0 && cnt > A.clusters) atomicOr(A.P.err, DEV_ERR_SHAPE);
        }
    }
    __syncthreads();
    const int grp = s_grp;
    const int c0 = (grp < 0 ? 0 : grp) * VEC, b0 = c0 % B;
    const bool neu = (mode == c0 / B);   // B % VEC == 0: one kind per cluster
    const int k0 = (int)rank * g.ppc, k1 = min(s2, k0 + g.ppc), np = max(0, k1 - k0);
    const int lo = k0 * pn, hi = max(lo, k1 * pn);
    int itmax = 0;
    if (grp >= 0) {
        const PcgArgs<T>& P = A.P;
        bool act[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) act[k] = P.V.st[b0 + k].phase != PH_DONE;
        // r and d of the own planes, [rows][VEC], and x at the first own row and column
        W *r, *d;
        if (g.vs) {
            r = reinterpret_cast<W*>(fs_sm + g.o_vec);
            d = r + (ptrdiff_t)g.ppc * pn * VEC;
        } else {
            const size_t gb = ((size_t)grp * N + lo) * VEC;
            r = reinterpret_cast<W*>(P.V.r) + gb;
            d = reinterpret_cast<W*>(P.V.z) + gb;
        }
        W* gt = TS ? nullptr : A.gt + (size_t)grp * s2 * VEC * ss;
        T* const x = (mode ? P.V.U2 : P.V.U1) + (size_t)lo * C + c0;
        const double* const bv = P.V.bvec + (size_t)lo * B + b0;
        const int* const nodes = P.M.node + lo;
        const int kind = neu ? 0 : 1;
        // transforms: forward F, back G
        const unsigned oFe = g.o_mat, oGe = oFe + (unsigned)(hp * hp * sizeof(W)), oFo = oGe + (unsigned)(hp * hp * sizeof(W)),
                       oGo = oFo + (unsigned)(hop * hop * sizeof(W));
        const W* inv = A.inv + (size_t)kind * s2 * ss;
        {
            W* mats = reinterpret_cast<W*>(fs_sm + g.o_mat);
            for (int i = tid; i < g.matw; i += nt) mats[i] = A.mat[(size_t)kind * g.matw + i];
        }
        for (int k = tid; k < s2; k += nt) {
            const int o = k / g.ppc, lp = k - o * g.ppc;
            s_plane[k] = TS ? peer_ptr(buf, (unsigned)o) + (size_t)lp * VEC * ss : gt + (size_t)k * VEC * ss;
            s_slot[k] = peer_addr(sm_addr(slots), (unsigned)o) + (uint32_t)(lp * FS_NQ * VEC * sizeof(double));
        }
        if constexpr (TS)   // the gap columns stay zero
            for (int i = tid; i < np * VEC * ss; i += nt) buf[i] = W(0);
        if (tid < VEC) {
            s_it[tid] = 0;
            s_done[tid] = 0;
            s_tin[tid] = 0.0;
        }
        __syncthreads();
        int par = 0;
        // Totals over the cluster of the nq quantities whose chunk sums the CTA has
        // written to part: chunks of a plane, then planes (lanes stride, then a fixed
        // butterfly); the same bits in every CTA.  The slots alternate: one is
        // rewritten only after a further barrier, when every CTA has read it.
        auto reduce = [&](int nq) {
            __syncthreads();
            double* slot = slots + par * g.ppc * FS_NQ * VEC;
            for (int it = warp; it < np * nq * VEC; it += nw) {
                const int pl = it / (nq * VEC), v = it - pl * nq * VEC;
                double acc = 0.0;
                for (int c = lane; c < g.nch; c += 32) acc += part[(pl * g.nch + c) * FS_NQ * VEC + v];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) slot[pl * FS_NQ * VEC + v] = acc;
            }
            cl_sync();
            const uint32_t so = (uint32_t)(par * g.ppc * FS_NQ * VEC * (int)sizeof(double));
            for (int v = warp; v < nq * VEC; v += nw) {
                double acc = 0.0;
                for (int k = lane; k < s2; k += 32) acc += ld_peer1(s_slot[k] + so + (uint32_t)v * 8u, 0.0);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) out[v] = acc;
            }
            par ^= 1;
            __syncthreads();
        };
        // chunk sums of the quantities a0, a0 + 1, ... in v into part (whole warp): halves of
        // the values change sides at every step while there are several, so that each step
        // adds half as many; the sum of a value is the same butterfly's in any case
        auto put = [&](auto& v, int a0, int pl, int ch) {
            constexpr int NV = sizeof(v) / sizeof(v[0][0]);
            using X = typename std::remove_reference<decltype(v[0][0])>::type;
            X f[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) f[i] = v[i / VEC][i % VEC];
            int at = 0;
#pragma unroll
            for (int o = 16, n2 = NV; o > 0; o >>= 1) {
                if (n2 % 2 == 0) {
                    n2 >>= 1;
                    const bool up = lane & o;
                    if (up) at += n2;
#pragma unroll
                    for (int i = 0; i < n2; ++i) {
                        const X send = up ? f[i] : f[i + n2], keep = up ? f[i + n2] : f[i];
                        f[i] = plus(keep, shfl_x(send, o));
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < n2; ++i) f[i] = plus(f[i], shfl_x(f[i], o));
                }
            }
            static_assert((NV & (NV - 1)) == 0 && NV <= 16, "one value a lane is left");
            if ((lane & (32 / NV - 1)) == 0) part[((pl * g.nch + ch) * FS_NQ + a0) * VEC + at] = total(f[0]);
        };
        // f(pl, ch, q) for every chunk ch of the CTA's planes [pa, pb), a warp per chunk, a
        // lane per quadruple of mirrored nodes: u = 0 (y, x), 1 (y, n-x), 2 (n-y, x),
        // 3 (n-y, n-x), x, y < h.  A warp keeps its chunk from plane to plane where the
        // CTA has as many warps as a plane has chunks, so q is computed once.
        struct Quad {
            int y, x;
            bool on, has[4];
            int row[4];    // in a plane of rows
            int at[4];     // in a sheet
        };
        auto quads = [&](int pa, int pb, auto&& f) {
            const int nc = (h * h + 31) / 32;
            const bool wide = nw >= nc;
            const int ps = wide ? nw / nc : 1, pf = wide ? warp / nc : 0, cf = wide ? warp - pf * nc : warp;
            if (pf >= ps) return;
            for (int ch = cf; ch < nc; ch += wide ? nc : nw) {
                Quad q;
                const int e = ch * 32 + lane;
                q.y = e / h;
                q.x = e - q.y * h;
                q.on = q.y < h;
                if (!q.on) q.y = 0;
                const bool mx = q.x < ho, my = q.y < ho;
                q.has[0] = q.on;
                q.has[1] = q.on && mx;
                q.has[2] = q.on && my;
                q.has[3] = q.on && mx && my;
                const int xm = mx ? n - q.x : q.x, ym = my ? n - q.y : q.y, cm = mx ? xm + gap : q.x;
                q.row[0] = q.y * s2 + q.x;
                q.row[1] = q.y * s2 + xm;
                q.row[2] = ym * s2 + q.x;
                q.row[3] = ym * s2 + xm;
                q.at[0] = q.y * ldx + q.x;
                q.at[1] = q.y * ldx + cm;
                q.at[2] = ym * ldx + q.x;
                q.at[3] = ym * ldx + cm;
                for (int pl = pa + pf; pl < pb; pl += ps) f(pl, ch, q);
            }
        };
        // The stencil: f(u, value) of (K v) at the quadruple's nodes for column k of the
        // plane kk's sheets s (own plane), with the planes below and above.  Weights in
        // units h/6: an axis edge counts 6 times 1/2 per other coordinate on the boundary,
        // +-1/2 on the cube's edges (same end of both other axes: +).
        auto stencil = [&](const Quad& q, int kk, const W* s, const W* sm, const W* sp, auto&& f) {
            const bool ex = q.x == 0, ey = q.y == 0, ek = kk == 0 || kk == n;
            const W ax = ex ? W(0.5) : W(1), ay = ey ? W(0.5) : W(1), ak = ek ? W(0.5) : W(1);
            const W wx = W(6) * ay * ak, wy = W(6) * ax * ak, wz = W(6) * ax * ay;
            const W cx = ey && ek ? (kk == 0 ? W(0.5) : W(-0.5)) : W(0), cy = ex && ek ? (kk == 0 ? W(0.5) : W(-0.5)) : W(0),
                    cz = ex && ey ? W(0.5) : W(0);
            const int xo = ex ? 0 : -1, xi = q.x + 1 < h ? 1 : 1 + gap, xim = n - q.x - 1 >= h ? -1 : -1 - gap;
            const int yo = ey ? 0 : -ldx;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!q.has[u]) continue;
                const W* z = s + q.at[u];
                const W z0 = z[0];
                const W vx = wx + ((u & 2) ? -cx : cx), vy = wy + ((u & 1) ? -cy : cy), vz = wz + (u == 0 || u == 3 ? cz : -cz);
                // towards the boundary (none there: the difference vanishes) and away from it
                W a = vx * (z0 - z[(u & 1) ? -xo : xo]);
                a = fma_(vx, z0 - z[(u & 1) ? xim : xi], a);
                a = fma_(vy, z0 - z[(u & 2) ? -yo : yo], a);
                a = fma_(vy, z0 - z[(u & 2) ? -ldx : ldx], a);
                a = fma_(vz, z0 - sm[q.at[u]], a);
                a = fma_(vz, z0 - sp[q.at[u]], a);
                f(u, z0, a);
            }
        };
        // Small cubes in FP64: the same with a lane per node, a warp per chunk of 8
        // quadruples.  A warp's FP64 instruction takes its scheduler 64 clocks, and a plane of
        // 11 x 11 nodes is one warp of quadruples: four nodes one after the other on one of an
        // SM's four schedulers.  One instance at n = 10: 57 -> 51 us a stage; at n = 25, whose
        // planes are six warps of quadruples, the lanes' index work costs 3 %.
        bool nodewise = false;
        if constexpr (ND) nodewise = h <= FS_NODE_H;
        struct Node {
            int y, x;      // of the quadruple
            bool mx, my, on;
            int row, at;
        };
        auto each = [&](int pa, int pb, auto&& f) {
            const int nc = g.nch;
            const bool wide = nw >= nc;
            const int ps = wide ? nw / nc : 1, pf = wide ? warp / nc : 0, cf = wide ? warp - pf * nc : warp;
            if (pf >= ps) return;
            for (int ch = cf; ch < nc; ch += wide ? nc : nw) {
                Node q;
                const int e = ch * 8 + (lane >> 2);
                q.y = e / h;
                q.x = e - q.y * h;
                q.mx = lane & 1;
                q.my = lane & 2;
                q.on = q.y < h && (!q.mx || q.x < ho) && (!q.my || q.y < ho);
                if (!q.on) q.y = q.x = 0, q.mx = q.my = false;
                const int xm = q.mx ? n - q.x : q.x, ym = q.my ? n - q.y : q.y;
                q.row = ym * s2 + xm;
                q.at = ym * ldx + xm + (q.mx ? gap : 0);
                for (int pl = pa + pf; pl < pb; pl += ps) f(pl, ch, q);
            }
        };
        // (K v) at a node: the arithmetic of stencil, the weights (1, 2, 3 or 6) by selection
        auto stencil1 = [&](const Node& q, int kk, const W* s, const W* sm, const W* sp, W& z0) -> W {
            const bool ex = q.x == 0, ey = q.y == 0, ek = kk == 0 || kk == n, lo_end = kk == 0;
            const W vx = ey && ek ? (lo_end != q.my ? W(2) : W(1)) : ey || ek ? W(3) : W(6);
            const W vy = ex && ek ? (lo_end != q.mx ? W(2) : W(1)) : ex || ek ? W(3) : W(6);
            const W vz = ex && ey ? (q.mx == q.my ? W(2) : W(1)) : ex || ey ? W(3) : W(6);
            const int xo = ex ? 0 : -1, xi = q.x + 1 < h ? 1 : 1 + gap, xim = n - q.x - 1 >= h ? -1 : -1 - gap;
            const int yo = ey ? 0 : -ldx;
            const W* z = s + q.at;
            z0 = z[0];
            W a = vx * (z0 - z[q.mx ? -xo : xo]);
            a = fma_(vx, z0 - z[q.mx ? xim : xi], a);
            a = fma_(vy, z0 - z[q.my ? -yo : yo], a);
            a = fma_(vy, z0 - z[q.my ? -ldx : ldx], a);
            a = fma_(vz, z0 - sm[q.at], a);
            return fma_(vz, z0 - sp[q.at], a);
        };
        // the sheets of the planes below and above plane kk (its own where there is none)
        auto below = [&](int kk, int pl) -> const W* { return kk == 0 ? s_plane[0] : (TS && pl > 0 ? buf + (pl - 1) * VEC * ss : s_plane[kk - 1]); };
        auto above = [&](int kk, int pl) -> const W* { return kk == n ? s_plane[n] : (TS && pl + 1 < np ? buf + (pl + 1) * VEC * ss : s_plane[kk + 1]); };
        auto own = [&](int kk, int pl) -> const W* { return TS ? buf + pl * VEC * ss : s_plane[kk]; };

        // Surface values of the Dirichlet systems (stage 1 adjoint: zero; stage 2 forward:
        // B u1_S).  T = W: x with them into d and into the planes' place.
        if constexpr (!MP) {
            quads(0, np, [&](int pl, int, const Quad& q) {
                const int kk = k0 + pl;
                const bool surf = q.x == 0 || q.y == 0 || kk == 0 || kk == n;
                T xv[4][VEC];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (q.has[u]) ldc<VEC, false>(xv[u], x + (ptrdiff_t)(pl * pn + q.row[u]) * C);
                W* s = const_cast<W*>(own(kk, pl));
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (!q.has[u]) continue;
                    if (!neu && surf) {
                        const int bp = (int)((unsigned)nodes[pl * pn + q.row[u]] >> 16);
#pragma unroll
                        for (int k = 0; k < VEC; ++k)
                            if (act[k]) xv[u][k] = mode ? P.V.ub_out[(size_t)(bp - 1) * C + b0 + k] : T(0);
                    }
                    W wv[VEC];
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        wv[k] = W(xv[u][k]);
                        s[k * ss + q.at[u]] = wv[k];
                    }
                    stc<VEC>(d + (ptrdiff_t)(pl * pn + q.row[u]) * VEC, wv);
                }
            });
        } else if (!neu) {
            for (int l = tid; l < hi - lo; l += nt) {
                const int bp = (int)((unsigned)nodes[l] >> 16);
                if (!bp) continue;
#pragma unroll
                for (int k = 0; k < VEC; ++k)
                    if (act[k]) x[(ptrdiff_t)l * C + k] = mode ? P.V.ub_out[(size_t)(bp - 1) * C + b0 + k] : T(0);
            }
        }
        cl_sync();
        const int step = TS ? max(np, 1) : g.spl;
        bool ended = false;
        for (int cycle = 0;; ++cycle) {
            // residual of the current x into r; sums r.r, f.f (f: the norm reference,
            // Dirichlet: f - K_IS x_S) and, Neumann, r, f and (MP) V x for the gauge
            if constexpr (ND) if (nodewise) each(0, np, [&](int pl, int ch, const Node& q) {
                const int kk = k0 + pl;
                const bool surf = q.x == 0 || q.y == 0 || kk == 0 || kk == n, froz = !neu && surf;
                W v[4][VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) v[0][k] = v[1][k] = v[2][k] = v[3][k] = W(0);
                if (q.on) {
                    const int l = pl * pn + q.row;
                    double fb[VEC];
#pragma unroll
                    for (int k = 0; k < VEC; ++k) fb[k] = 0.0;
                    if (!froz && (neu || !mode)) {
                        ldc<VEC, false>(fb, bv + (ptrdiff_t)l * B);
                        if (mode && surf) {   // the BEM term of the adjoint Neumann system
                            const int bp = (int)((unsigned)nodes[l] >> 16);
#pragma unroll
                            for (int k = 0; k < VEC; ++k) fb[k] += (double)P.V.ub_out[(size_t)(bp - 1) * C + c0 + k];
                        }
                    }
                    const W *s = own(kk, pl), *sm = below(kk, pl), *sp = above(kk, pl);
                    const bool nx = q.x == 1, nx2 = q.x + 1 == n, ny = q.y == 1, ny2 = q.y + 1 == n, nk = kk == 1, nk2 = kk + 1 == n;
                    const bool ref_differs = !froz && !neu && mode && (nx || nx2 || ny || ny2 || nk || nk2);
                    W rv[VEC];
#pragma unroll
                    for (int k = 0; k < VEC; ++k, s += ss, sm += ss, sp += ss) {
                        W kx = W(0), z0, ref = act[k] ? W(fb[k]) : W(0);
                        rv[k] = ref;
                        if (!froz) kx = stencil1(q, kk, s, sm, sp, z0), rv[k] -= kx;
                        if (ref_differs) {   // neighbours on the surface
                            const int xi = q.x + 1 < h ? 1 : 1 + gap, xim = n - q.x - 1 >= h ? -1 : -1 - gap;
                            const W* z = s + q.at;
                            W t = W(0);
                            if (nx) t += z[q.mx ? 1 : -1];
                            if (nx2) t += z[q.mx ? xim : xi];
                            if (ny) t += z[q.my ? ldx : -ldx];
                            if (ny2) t += z[q.my ? -ldx : ldx];
                            if (nk) t += sm[q.at];
                            if (nk2) t += sp[q.at];
                            ref = fma_(W(6), t, ref);
                        }
                        v[0][k] = rv[k] * rv[k];
                        v[1][k] = ref * ref;
                        v[2][k] = rv[k];
                        v[3][k] = ref;
                    }
                    stc<VEC>(r + (ptrdiff_t)l * VEC, rv);
                }
                put(v, 0, pl, ch);
            });
            if (!nodewise) quads(0, np, [&](int pl, int ch, const Quad& q) {
                const int kk = k0 + pl;
                const bool surf = q.x == 0 || q.y == 0 || kk == 0 || kk == n;
                typename SumOf<W>::type v[4][VEC];
                double vx[1][VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) vx[0][k] = 0.0;
                const bool froz = !neu && surf;
                // node: r = f - kx stored; sums of r.r and of the square of the reference f - ks (f:
                // none in the stage-2 forward system), of Neumann systems also of r and f
                auto node = [&](int l, const T (&kx)[VEC], const T (&ks)[VEC], bool differs) {
                    double f[VEC];
                    const bool rhs = !froz && (neu || !mode);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) f[k] = 0.0;
                    if (rhs) {
                        ldc<VEC, false>(f, bv + (ptrdiff_t)l * B);
                        if (mode && surf) {   // the BEM term of the adjoint Neumann system
                            const int bp = (int)((unsigned)nodes[l] >> 16);
#pragma unroll
                            for (int k = 0; k < VEC; ++k) f[k] += (double)P.V.ub_out[(size_t)(bp - 1) * C + c0 + k];
                        }
                    }
                    W rv[VEC];
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        const T ft = act[k] ? T(f[k]) : T(0);
                        rv[k] = W(ft - kx[k]);
                        if (froz) continue;
                        v[0][k].fma(rv[k], rv[k]);
                        if (neu) v[2][k].add(rv[k]);
                        if (!rhs && !differs) continue;
                        const W ref = W(ft - ks[k]);
                        v[1][k].fma(ref, ref);
                        if (neu) v[3][k].add(ref);
                    }
                    stc<VEC>(r + (ptrdiff_t)l * VEC, rv);
                };
                if constexpr (!MP) {
                    T kx[4][VEC];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int k = 0; k < VEC; ++k) kx[u][k] = T(0);
                    const W *s = own(kk, pl), *sm = below(kk, pl), *sp = above(kk, pl);
                    if (!froz)
#pragma unroll
                        for (int k = 0; k < VEC; ++k)
                            stencil(q, kk, s + k * ss, sm + k * ss, sp + k * ss, [&](int u, W, W a) { kx[u][k] = a; });
                    // neighbours on the surface (K_IS x_S of the stage-2 forward system)
                    const bool nx = q.x == 1, nx2 = q.x + 1 == n, ny = q.y == 1, ny2 = q.y + 1 == n;
                    const bool differs = !froz && !neu && mode && (nx || nx2 || ny || ny2 || kk == 1 || kk + 1 == n);
                    const int xi = q.x + 1 < h ? 1 : 1 + gap, xim = n - q.x - 1 >= h ? -1 : -1 - gap;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (!q.has[u]) continue;
                        T ks[VEC];
#pragma unroll
                        for (int k = 0; k < VEC; ++k) {
                            ks[k] = T(0);
                            if (!differs) continue;
                            const W* z = s + k * ss + q.at[u];
                            typename SumOf<W>::type t;
                            if (nx) t.add(z[(u & 1) ? 1 : -1]);
                            if (nx2) t.add(z[(u & 1) ? xim : xi]);
                            if (ny) t.add(z[(u & 2) ? ldx : -ldx]);
                            if (ny2) t.add(z[(u & 2) ? -ldx : ldx]);
                            if (kk == 1) t.add(sm[k * ss + q.at[u]]);
                            if (kk + 1 == n) t.add(sp[k * ss + q.at[u]]);
                            ks[k] = scaled(W(-6), t);
                        }
                        node(pl * pn + q.row[u], kx[u], ks, differs);
                    }
                } else {
                    const int co[3] = {q.x, q.y, kk};
                    const ptrdiff_t st[3] = {(ptrdiff_t)C, (ptrdiff_t)s2 * C, (ptrdiff_t)pn * C};
#pragma unroll 1
                    for (int u = 0; u < 4; ++u) {
                        const bool mx = u & 1, my = u & 2;
                        if (!(mx ? (my ? q.has[3] : q.has[1]) : (my ? q.has[2] : q.has[0]))) continue;
                        const int j = my ? n - q.y : q.y, i = mx ? n - q.x : q.x, l = pl * pn + j * s2 + i;
                        T kx[VEC], ks[VEC];
                        bool differs = false;
#pragma unroll
                        for (int k = 0; k < VEC; ++k) kx[k] = ks[k] = T(0);
                        if (!froz) {
                            const T* xp = x + (ptrdiff_t)l * C;
                            T xi[VEC];
                            ldc<VEC, false>(xi, xp);
                            const int wt[3] = {surf ? edge_weight(j, kk, n) : 6, surf ? edge_weight(i, kk, n) : 6,
                                               surf ? edge_weight(i, j, n) : 6};
#pragma unroll
                            for (int a = 0; a < 3; ++a)
#pragma unroll
                                for (int sg = -1; sg <= 1; sg += 2) {
                                    // x and y: sg < 0 towards the boundary; z: down
                                    const int ca = co[a] + sg;
                                    if (ca < 0 || ca > n) continue;
                                    const bool flip = (a == 0 && mx) || (a == 1 && my);
                                    T xj[VEC];
                                    ldc<VEC, false>(xj, xp + ((sg < 0) != flip ? -st[a] : st[a]));
                                    const T w = T(wt[a]);
#pragma unroll
                                    for (int k = 0; k < VEC; ++k) kx[k] = fma_(w, xi[k] - xj[k], kx[k]);
                                    if (!neu && mode && (ca == 0 || ca == n)) {   // the neighbour lies on the surface
                                        differs = true;
#pragma unroll
                                        for (int k = 0; k < VEC; ++k) ks[k] -= T(6) * xj[k];
                                    }
                                }
                            if (neu) {
                                const double vi = (double)(nodes[l] & 0xff);
#pragma unroll
                                for (int k = 0; k < VEC; ++k) vx[0][k] = fma_(vi, (double)xi[k], vx[0][k]);
                            }
                        }
                        node(l, kx, ks, differs);
                    }
                }
                if (neu) {
                    put(v, 0, pl, ch);
                    if constexpr (MP) put(vx, 4, pl, ch);
                } else {
                    put(reinterpret_cast<typename SumOf<W>::type(&)[2][VEC]>(v), 0, pl, ch);
                }
            });
            reduce(!neu ? 2 : MP ? 5 : 4);
            int it = 0;
            for (;; ++it) {
                const bool first = it == 0;
                if (tid < VEC) {
                    // Neumann: residual (and first of all the reference) without their means
                    const double sr = neu ? out[(first ? 2 : 1) * VEC + tid] : 0.0;
                    const double rr = neu ? fmax(out[tid] - sr * sr / (double)N, 0.0) : out[tid];
                    const bool a = P.V.st[b0 + tid].phase != PH_DONE;
                    if (first) {
                        const double ff = out[VEC + tid], sf = neu ? out[3 * VEC + tid] : 0.0;
                        s_tol[tid] = P.tol2 * (neu ? fmax(ff - sf * sf / (double)N, 0.0) : ff);
                    } else if (!s_flag[tid]) {
                        s_it[tid] += 1;
                    }
                    // every solve takes a step (Neumann: a pair): it costs little, and the
                    // error is then rounding's, not the tolerance's; a pair is completed.
                    // A system that has met the test waits for the others of its cluster: the
                    // second step of a pair belongs to the first one, which it has not taken.
                    const bool stays = !first && s_flag[tid];
                    const bool must = (first && cycle == 0) || (neu && (it & 1));
                    int conv;
                    if constexpr (MP) {
                        if (first) {   // rr is the true (FP64) residual of this cycle
                            s_done[tid] = !a || (!must && !(rr > s_tol[tid])) || s_it[tid] >= P.max_iter;
                            s_tin[tid] = fmax(s_tol[tid], MP_INNER * MP_INNER * rr);
                        }
                        conv = stays || s_done[tid] || (!must && !(rr > s_tin[tid])) || s_it[tid] >= P.max_iter;
                    } else {
                        conv = stays || !a || (!must && !(rr > s_tol[tid])) || it >= P.max_iter;
                    }
                    s_flag[tid] = conv;
                    s_mean[tid] = neu ? sr / (double)N : 0.0;
                }
                // the same totals in every CTA of the cluster: every CTA leaves together
                if (__syncthreads_and(tid < VEC ? s_flag[tid] : 1)) break;
                W mean[VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) mean[k] = W(s_mean[k]);
                const bool second = neu && (it & 1);   // of a Neumann pair
                // ---- P1 ------------------------------------------------------------
                for (int pa = 0; pa < np; pa += step) {
                    const int pb = min(np, pa + step), nsh = (pb - pa) * VEC;
                    quads(pa, pb, [&](int pl, int, const Quad& q) {
                        W f[4][VEC];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
#pragma unroll
                            for (int k = 0; k < VEC; ++k) f[u][k] = mean[k];
                            if (q.has[u]) ldc<VEC, false>(f[u], r + (ptrdiff_t)(pl * pn + q.row[u]) * VEC);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int k = 0; k < VEC; ++k) f[u][k] -= mean[k];
                        if (second) {
                            const int kk = k0 + pl, bnd = (q.x == 0) + (q.y == 0) + (kk == 0 || kk == n);
                            if (bnd >= 2)
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    if (!q.has[u]) continue;
                                    const int e = edge_index((u & 1) ? n - q.x : q.x, (u & 2) ? n - q.y : q.y, kk, n);
#pragma unroll
                                    for (int k = 0; k < VEC; ++k) f[u][k] += ec[e * VEC + k];
                                }
                        }
                        if (!q.on) return;
                        // fold about the centre in x, then in y
                        W* s = buf + (pl - pa) * VEC * ss;
#pragma unroll
                        for (int k = 0; k < VEC; ++k, s += ss) {
                            const W e0 = f[0][k] + f[1][k], e1 = f[2][k] + f[3][k];
                            const W o0 = f[0][k] - f[1][k], o1 = f[2][k] - f[3][k];
                            s[q.at[0]] = e0 + e1;
                            if (q.has[1]) s[q.at[1]] = o0 + o1;
                            if (q.has[2]) s[q.at[2]] = e0 - e1;
                            if (q.has[3]) s[q.at[3]] = o0 - o1;
                            if (!TS && q.x == h - 1)   // the gap columns (TS: zero from the start)
                                for (int c = 0; c < gap + (hop - ho); ++c) {
                                    const int cc = c < gap ? h + c : hp + ho + c - gap;
                                    s[q.y * ldx + cc] = W(0);
                                    if (q.has[2]) s[(n - q.y) * ldx + cc] = W(0);
                                }
                        }
                    });
                    __syncthreads();
                    pass_right<W>(0, nsh, oFe, oFo, s2, hp, hop);
                    pass_left<W>(0, nsh, ldx, oFe, oFo, s2, hp, hop, nullptr, 1);
                    if constexpr (!TS) {
                        for (int i = tid * 4; i < nsh * ss; i += nt * 4) {
                            W v[4];
                            ld4(buf + i, v);
                            st4(gt + (size_t)(k0 + pa) * VEC * ss + i, v);
                        }
                        __syncthreads();
                    }
                }
                cl_sync();
                // ---- P2 ------------------------------------------------------------
                const int z0 = (int)rank * g.zc, z1 = min(ss, z0 + g.zc);
                for (int za = z0; za < z1; za += g.pr) {
                    const int pc = min(g.pr, z1 - za), ld = VEC * pc, q4 = pc >> 2, per = VEC * q4;
                    for (int e = tid; e < h * per; e += nt) {
                        const int k = e / per, rem = e - k * per, c = VEC == 1 ? 0 : rem / q4, p4 = 4 * (rem - c * q4);
                        const int off = c * ss + za + p4;
                        W a[4], b[4] = {W(0), W(0), W(0), W(0)}, s[4];
                        ld4(s_plane[k] + off, a);
                        if (k < ho) ld4(s_plane[n - k] + off, b);
                        W* zp = zb + k * ld + c * pc + p4;
#pragma unroll
                        for (int j = 0; j < 4; ++j) s[j] = a[j] + b[j];
                        st4(zp, s);
                        if (k < ho) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) s[j] = a[j] - b[j];
                            st4(zp + (n - 2 * k) * ld, s);   // row n - k
                        }
                    }
                    __syncthreads();
                    pass_left<W>(g.o_z, 1, ld, oFe, oFo, s2, hp, hop, inv + za, pc);
                    pass_left<W>(g.o_z, 1, ld, oGe, oGo, s2, hp, hop, nullptr, 1);
                    for (int e = tid; e < h * per; e += nt) {
                        const int k = e / per, rem = e - k * per, c = VEC == 1 ? 0 : rem / q4, p4 = 4 * (rem - c * q4);
                        const int off = c * ss + za + p4;
                        const W* zp = zb + k * ld + c * pc + p4;
                        W a[4], b[4] = {W(0), W(0), W(0), W(0)}, s[4], t[4];
                        ld4(zp, a);
                        if (k < ho) ld4(zp + (n - 2 * k) * ld, b);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            s[j] = a[j] + b[j];
                            t[j] = a[j] - b[j];
                        }
                        st4(s_plane[k] + off, s);
                        if (k < ho) st4(s_plane[n - k] + off, t);
                    }
                    __syncthreads();
                }
                cl_sync();
                // ---- P3 ------------------------------------------------------------
                for (int pa = 0; pa < np; pa += step) {
                    const int pb = min(np, pa + step), nsh = (pb - pa) * VEC;
                    if constexpr (!TS) {
                        for (int i = tid * 4; i < nsh * ss; i += nt * 4) {
                            W v[4];
                            ldc<4, true>(v, gt + (size_t)(k0 + pa) * VEC * ss + i);
                            st4(buf + i, v);
                        }
                        __syncthreads();
                    }
                    pass_left<W>(0, nsh, ldx, oGe, oGo, s2, hp, hop, nullptr, 1);
                    pass_right<W>(0, nsh, oGe, oGo, s2, hp, hop);
                    quads(pa, pb, [&](int pl, int, const Quad& q) {
                        if (!q.on) return;   // unfold, in place
                        W* s = buf + (pl - pa) * VEC * ss;
#pragma unroll
                        for (int k = 0; k < VEC; ++k, s += ss) {
                            const W ee = s[q.at[0]], eo = q.has[1] ? s[q.at[1]] : W(0), oe = q.has[2] ? s[q.at[2]] : W(0);
                            const W oo = q.has[3] ? s[q.at[3]] : W(0);
                            s[q.at[0]] = (ee + eo) + (oe + oo);
                            if (q.has[1]) s[q.at[1]] = (ee - eo) + (oe - oo);
                            if (q.has[2]) s[q.at[2]] = (ee + eo) - (oe + oo);
                            if (q.has[3]) s[q.at[3]] = (ee - eo) - (oe - oo);
                        }
                    });
                    if constexpr (!TS) {
                        __syncthreads();
                        for (int i = tid * 4; i < nsh * ss; i += nt * 4) {
                            W v[4];
                            ld4(buf + i, v);
                            st4(gt + (size_t)(k0 + pa) * VEC * ss + i, v);
                        }
                        __syncthreads();
                    }
                }
                cl_sync();
                // ---- P4 ------------------------------------------------------------
                W keep[VEC];   // 0: the system has converged and stays as it is
#pragma unroll
                for (int k = 0; k < VEC; ++k) keep[k] = s_flag[k] ? W(0) : W(1);
                if constexpr (ND) if (nodewise) each(0, np, [&](int pl, int ch, const Node& q) {
                    W v[2][VEC];   // r.r, sum r
                    const int kk = k0 + pl;
                    const bool froz = !neu && (q.x == 0 || q.y == 0 || kk == 0 || kk == n);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) v[0][k] = v[1][k] = W(0);
                    if (q.on) {
                        W rv[VEC], dv[VEC];
                        const ptrdiff_t o = (ptrdiff_t)(pl * pn + q.row) * VEC;
                        ldc<VEC, false>(rv, r + o);
                        ldc<VEC, false>(dv, d + o);
                        const W *s = own(kk, pl), *sm = below(kk, pl), *sp = above(kk, pl);
#pragma unroll
                        for (int k = 0; k < VEC; ++k, s += ss, sm += ss, sp += ss) {
                            W z0, a = stencil1(q, kk, s, sm, sp, z0);
                            if (froz) a = W(0);
                            rv[k] = fma_(-keep[k], a, rv[k] - mean[k]);
                            dv[k] = fma_(keep[k], z0, dv[k]);
                            v[0][k] = rv[k] * rv[k];
                            v[1][k] = rv[k];
                        }
                        stc<VEC>(r + o, rv);
                        stc<VEC>(d + o, dv);
                    }
                    put(v, 0, pl, ch);
                });
                if (!nodewise) quads(0, np, [&](int pl, int ch, const Quad& q) {
                    W v[2][VEC];   // r.r, sum r
#pragma unroll
                    for (int k = 0; k < VEC; ++k) v[0][k] = v[1][k] = W(0);
                    const int kk = k0 + pl;
                    const bool froz = !neu && (q.x == 0 || q.y == 0 || kk == 0 || kk == n);
                    W rv[4][VEC], dv[4][VEC];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (!q.has[u]) continue;
                        const ptrdiff_t o = (ptrdiff_t)(pl * pn + q.row[u]) * VEC;
                        ldc<VEC, false>(rv[u], r + o);
                        if (!MP || !first) ldc<VEC, false>(dv[u], d + o);
                        else
#pragma unroll
                            for (int k = 0; k < VEC; ++k) dv[u][k] = W(0);
                    }
                    const W *s = own(kk, pl), *sm = below(kk, pl), *sp = above(kk, pl);
#pragma unroll
                    for (int k = 0; k < VEC; ++k)
                        stencil(q, kk, s + k * ss, sm + k * ss, sp + k * ss, [&](int u, W zc, W a) {
                            if (froz) a = W(0);
                            rv[u][k] = fma_(-keep[k], a, rv[u][k] - mean[k]);
                            dv[u][k] = fma_(keep[k], zc, dv[u][k]);
                            v[0][k] = fma_(rv[u][k], rv[u][k], v[0][k]);
                            v[1][k] += rv[u][k];
                        });
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (!q.has[u]) continue;
                        const ptrdiff_t o = (ptrdiff_t)(pl * pn + q.row[u]) * VEC;
                        stc<VEC>(r + o, rv[u]);
                        stc<VEC>(d + o, dv[u]);
                    }
                    put(v, 0, pl, ch);
                });
                if (neu && !second) {
                    // H z on the edge nodes for the second step of the pair: this CTA's
                    // rows, each in FS_SPLIT parts, to the CTAs that own the nodes
                    for (int t = tid; t < g.ne * VEC; t += nt) {
                        const int k = VEC == 1 ? 0 : t / g.ne, e = t - k * g.ne;
                        int i, j, l;
                        edge_node(e, n, i, j, l);
                        ev[e * VEC + k] = s_plane[l][k * ss + j * ldx + i + (i < h ? 0 : gap)];
                    }
                    __syncthreads();
                    const int e0 = (int)rank * g.er, er = max(0, min(g.er, g.ne - e0)), sl = (g.ne + FS_SPLIT - 1) / FS_SPLIT;
                    for (int t = tid; t < er * FS_SPLIT; t += nt) {
                        const int sq = t / er, e = t - sq * er;
                        W acc[VEC];
#pragma unroll
                        for (int k = 0; k < VEC; ++k) acc[k] = W(0);
                        const W* Hp = A.edge + e0 + e;   // column e0 + e of the symmetric matrix
                        const int fb = min(g.ne, (sq + 1) * sl);
#pragma unroll 8
                        for (int f = sq * sl; f < fb; ++f) {
                            const W hv = __ldg(Hp + f * g.ne);
#pragma unroll
                            for (int k = 0; k < VEC; ++k) acc[k] = fma_(hv, ev[f * VEC + k], acc[k]);
                        }
#pragma unroll
                        for (int k = 0; k < VEC; ++k) ep[t * VEC + k] = acc[k];
                    }
                    __syncthreads();
                    for (int t = tid; t < er * VEC; t += nt) {
                        const int e = t / VEC, k = t - e * VEC;
                        W acc = W(0);
#pragma unroll
                        for (int sq = 0; sq < FS_SPLIT; ++sq) acc += ep[(sq * er + e) * VEC + k];
                        int i, j, l;
                        edge_node(e0 + e, n, i, j, l);
                        st_peer1(peer_addr(sm_addr(ec + (e0 + e) * VEC + k), (unsigned)(l / g.ppc)), acc);
                    }
                }
                reduce(2);
            }
            if constexpr (!MP) {
                break;
            } else {
                // done when every system met the tolerance on its true residual at the
                // start of this cycle (or ran out of iterations)
                if (__syncthreads_and(tid < VEC ? s_done[tid] : 1)) {
                    ended = true;
                    break;
                }
                if (it > 0)   // the cycle's steps into x before anything reads x
                    for (int l = tid; l < hi - lo; l += nt) {
                        T xv[VEC];
                        W dv[VEC];
                        ldc<VEC, false>(xv, x + (ptrdiff_t)l * C);
                        ldc<VEC, false>(dv, d + (ptrdiff_t)l * VEC);
#pragma unroll
                        for (int k = 0; k < VEC; ++k) xv[k] += T(dv[k]);
                        stc<VEC>(x + (ptrdiff_t)l * C, xv);
                    }
                cl_sync();
                if (cycle + 1 >= MP_MAX_CYCLES) break;
            }
        }
        // Neumann systems are gauged to zero V-weighted mean and (stage 1) hand u1_S to
        // the BEM product; stage-1 Dirichlet (adjoint) systems hand t = b_S - K_SI w (w
        // vanishes on the surface, so K_SI w = (K w)_S)
        double mean[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) mean[k] = 0.0;
        if (neu) {
            if (!ended) {   // MP: the residual pass that ended the solve has summed V x
                if constexpr (ND) if (nodewise) each(0, np, [&](int pl, int ch, const Node& q) {
                    W v[1][VEC], xv[VEC];
#pragma unroll
                    for (int k = 0; k < VEC; ++k) xv[k] = W(0);
                    const int l = pl * pn + q.row;
                    if (q.on) ldc<VEC, false>(xv, d + (ptrdiff_t)l * VEC);
                    const W vi = W(nodes[l] & 0xff);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) v[0][k] = vi * xv[k];
                    put(v, 4, pl, ch);
                });
                if (!nodewise) quads(0, np, [&](int pl, int ch, const Quad& q) {
                    typename SumOf<T>::type v[1][VEC];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (!q.has[u]) continue;
                        const int l = pl * pn + q.row[u];
                        const T vi = T(nodes[l] & 0xff);
                        T xv[VEC];
                        if constexpr (MP) {
                            ldc<VEC, false>(xv, x + (ptrdiff_t)l * C);
                        } else {
                            ldc<VEC, false>(xv, d + (ptrdiff_t)l * VEC);
                        }
#pragma unroll
                        for (int k = 0; k < VEC; ++k) v[0][k].fma(vi, xv[k]);
                    }
                    put(v, 4, pl, ch);
                });
                reduce(5);
            }
#pragma unroll
            for (int k = 0; k < VEC; ++k) mean[k] = out[4 * VEC + k] / P.M.vsum;
        }
        if (!MP || neu)
            for (int l = tid; l < hi - lo; l += nt) {
                T xv[VEC];
                if constexpr (MP) {
                    ldc<VEC, false>(xv, x + (ptrdiff_t)l * C);
                } else {
                    W dv[VEC];
                    ldc<VEC, false>(dv, d + (ptrdiff_t)l * VEC);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) xv[k] = T(dv[k]);
                }
                const int bp = neu && mode == 0 ? (int)((unsigned)nodes[l] >> 16) : 0;
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    if (!act[k]) continue;
                    xv[k] -= T(mean[k]);
                    if (bp) P.V.ub_in[(size_t)(bp - 1) * C + c0 + k] = xv[k];
                }
                stc<VEC>(x + (ptrdiff_t)l * C, xv);
            }
        if (!neu && mode == 0) {
            cl_sync();   // x of the neighbouring planes
            for (int l = tid; l < hi - lo; l += nt) {
                const int bp = (int)((unsigned)nodes[l] >> 16);
                if (!bp) continue;
                // at most one of the six neighbours of a surface node lies inside
                const int row = lo + l, i = row % s2, j = (row / s2) % s2, k3 = row / pn;
                const T* xp = x + (ptrdiff_t)l * C;
                const ptrdiff_t st[3] = {(ptrdiff_t)C, (ptrdiff_t)s2 * C, (ptrdiff_t)pn * C};
                const int co[3] = {i, j, k3};
                T kw[VEC];
                double f[VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) kw[k] = T(0);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (co[a] != 0 && co[a] != n) continue;
                    const int u = co[(a + 1) % 3], w = co[(a + 2) % 3];
                    if (u == 0 || u == n || w == 0 || w == n) continue;   // never when n = 1
                    T xj[VEC];
                    ldc<VEC, true>(xj, xp + (co[a] == 0 ? st[a] : -st[a]));
#pragma unroll
                    for (int k = 0; k < VEC; ++k) kw[k] = T(-6) * xj[k];
                }
                ldc<VEC, false>(f, bv + (ptrdiff_t)l * B);
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
    // sweep counter: the largest step count of the solve (its last cluster to
    // finish adds it and clears the two counter words)
    if (rank == 0 && tid == 0) {
        atomicMax(&A.P.bar[2], (unsigned)itmax);
        __threadfence();
        if (atomicAdd(&A.P.bar[3], 1u) == (unsigned)A.clusters - 1u) {
            __threadfence();
            const unsigned km = atomicExch(&A.P.bar[2], 0u);
            atomicExch(&A.P.bar[3], 0u);
            if (A.P.sweeps) A.P.sweeps[mode + (sizeof(T) == 8 ? 2 : 0)] += (unsigned long long)km;
        }
    }
    cl_sync();   // no CTA leaves while another may still read its shared memory
}

// inv[mode][position of a sheet] = 1 / 6(l_z + l_y + l_x), lam_row[s2] and
// lam_col[ldx] the 1-D eigenvalues in the transforms' order (negative: no such mode)
__global__ void k_fast_inv(int s2, int ldx, const double* __restrict__ lam_row, const double* __restrict__ lam_col,
                           double* __restrict__ inv64, float* __restrict__ inv32) {
    const size_t total = (size_t)s2 * s2 * ldx;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const double a = lam_col[i % ldx], b = lam_row[(i / ldx) % s2], c = lam_row[i / ((size_t)ldx * s2)];
        const double l = 6.0 * (a + b + c);
        const double v = (a < 0.0 || b < 0.0 || c < 0.0 || !(l > 1e-9)) ? 0.0 : 1.0 / l;
        inv64[i] = v;
        inv32[i] = (float)v;
    }
}

FsGeo base_geo(int n) {
    FsGeo g = {};
    g.n = n;
    g.s2 = n + 1;
    g.h = (g.s2 + 1) / 2;
    g.ho = g.s2 / 2;
    g.hp = (g.h + 3) & ~3;
    g.hop = (g.ho + 3) & ~3;
    g.ldx = g.hp + g.hop;
    g.ss = g.s2 * g.ldx;
    g.matw = 2 * (g.hp * g.hp + g.hop * g.hop);
    g.ne = 12 * n - 4;
    return g;
}

// Geometry of clusters of `vec` systems with `ppc` planes per CTA; false when it
// does not fit the shared memory (ts: transformed planes there, else in global memory).
bool fit_geo(FsGeo& g, int vec, int ppc, size_t word, int threads, bool ts) {
    g.ppc = ppc;
    g.cl = (g.s2 + ppc - 1) / ppc;
    if (g.cl > FS_MAX_CL) return false;
    g.er = (g.ne + g.cl - 1) / g.cl;
    g.nch = word == 8 && g.h <= FS_NODE_H ? (g.h * g.h + 7) / 8 : (g.h * g.h + 31) / 32;
    auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
    const size_t mat = up(g.matw * word), part = up(sizeof(double) * (size_t)ppc * g.nch * FS_NQ * vec);
    const size_t slot = up(sizeof(double) * 2 * (size_t)ppc * FS_NQ * vec);
    const size_t edge = up(word * vec * (2 * (size_t)g.ne + (size_t)g.er * FS_SPLIT));
    const size_t col = up(sizeof(double) * (FS_NQ + 3) * vec + sizeof(int) * 3 * vec + (8 + 4) * FS_MAX_N1);
    const size_t vecs = up(word * vec * 2 * (size_t)ppc * g.s2 * g.s2);
    const size_t fixed = mat + part + slot + edge + col;
    const size_t sheet = (size_t)g.ss * word * vec;
    const int tr = word == 8 ? 1 : 4, tc = word == 8 ? 2 : 4;
    const int rt = (g.h + tr - 1) / tr + (g.ho + tr - 1) / tr;
    g.zc = ((g.ss + g.cl - 1) / g.cl + 3) & ~3;
    // positions per round of P2: what one round of pass_left holds, and what fits
    size_t pr = std::min(g.zc, std::max(4, (tc * ((threads / rt) / vec)) & ~3));
    size_t room, buf;
    if (ts) {
        buf = up(sheet * ppc);
        if (fixed + buf >= FS_SMEM_MAX) return false;
        room = FS_SMEM_MAX - fixed - buf;
    } else {
        if (fixed + sheet > FS_SMEM_MAX) return false;
        room = FS_SMEM_MAX - fixed;
        g.spl = std::max(1, std::min(ppc, (int)(room / sheet)));
        buf = up(sheet * g.spl);
    }
    pr = std::min(pr, room / (word * g.s2 * vec) / 4 * 4);
    if (pr < 4 || (ts && pr < (size_t)std::min(16, g.zc))) return false;
    g.pr = (int)pr;
    const size_t z = up((size_t)g.s2 * vec * pr * word);
    size_t o = ts ? buf : std::max(buf, z);
    g.o_z = ts ? (unsigned)o : 0;
    if (ts) o += z;
    auto take = [&o](size_t b) { const size_t at = o; o += b; return (unsigned)at; };
    g.o_mat = take(mat);
    g.o_part = take(part);
    g.o_slot = take(slot);
    g.o_edge = take(edge);
    g.o_col = take(col);
    g.vs = ts && o + vecs <= FS_SMEM_MAX;
    g.o_vec = g.vs ? take(vecs) : 0;
    g.smem = (unsigned)o;
    return o <= FS_SMEM_MAX;
}

template <typename T, typename W, int VEC, bool TS>
int resident(const FsGeo& g, int threads) {
    auto fn = k_fast_solve<T, W, VEC, TS>;
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, unsigned>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_tuple(dev, g.cl, threads, g.smem);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int ncl = 0;
    if (kernel_smem_attr((const void*)fn, (int)FS_SMEM_MAX) == cudaSuccess &&
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

struct FsChoice {
    FsGeo g;
    int vec = 0, threads = 0, clusters = 0;
    int per = 0;   // clusters of one launch (all of them without a cap on the blocks)
    bool ts = true;
};

template <typename T, typename W, int VEC, bool TS>
void try_shapes(const Launch& L, int n, int B, int groups, FsChoice& best, double& best_cost) {
    if (B % VEC) return;
    const int most = sizeof(W) == 8 ? 512 : 1024;
    for (int ppc = 1, last = 0; ppc <= n + 1; ++ppc) {
        const int cl = (n + ppc) / ppc;
        if (cl > FS_MAX_CL || cl == last) continue;   // more planes, no fewer CTAs
        last = cl;
        for (int threads = 256; threads <= most; threads *= 2) {
            FsGeo g = base_geo(n);
            if (!fit_geo(g, VEC, ppc, sizeof(W), threads, TS)) continue;
            int r = resident<T, W, VEC, TS>(g, threads);
            if (L.max_blocks > 0) r = std::min(r, L.max_blocks / cl);
            if (r < 1) continue;
            const int waves = (groups + r - 1) / r;
            // CTAs that share an SM share its issue slots; a CTA's own rows take their
            // latencies whatever the others do (us of two stages)
            const double rows = (double)ppc * VEC * g.s2 * g.s2 * (sizeof(W) == 8 ? 3.9 : 1.0);
            const double load = std::max(1.0, std::min(groups, r) * (double)cl / L.num_sms);
            double cost = waves * (TS ? 1.0 : 1.5) *
                          (5.8 + 1.1 * threads / 256 +
                           rows * std::max(0.83e-3 * load, 3.1e-3 * 256 / threads) * (1.0 + 0.14 * (VEC - 1)));
            if (sizeof(T) != sizeof(W))   // FP64 residuals: latencies weigh more, waves overlap
                cost = std::max(1.0, (double)groups / r) * (TS ? 1.0 : 1.5) * (1.0 + 0.04 * ppc) *
                       (3.0 + 0.3 * threads / 256 + rows * std::max(1.9e-3 * load, 2.5e-3 * 256 / threads));
            if (best.vec == 0 || cost < best_cost) {
                best_cost = cost;
                best.g = g;
                best.vec = VEC;
                best.threads = threads;
                best.ts = TS;
                best.clusters = waves > 1 ? 2 * B / VEC : std::min(r, 2 * B / VEC);
                best.per = best.clusters;
                if (L.max_blocks > 0) {   // waves as launches one after the other, none for idle groups only
                    best.clusters = std::min(waves * r, 2 * B / VEC);
                    best.per = r;
                }
            }
        }
    }
}

// The launch for a batch: VEC systems per cluster, planes per CTA, threads.  Clusters
// are independent, so more of them than can be resident at once run in waves; a cap on
// the blocks (L.max_blocks: size groups that share the chip) makes the waves launches.  The
// constants are fitted to some 400 measured shapes of 25 sizes and batches (n = 10 to
// 80, 1 to 64 instances), on which the rule's shape is within 5 % of the fastest (1 % on
// average): 64 instances at n = 30 run one system on two CTAs of 16 planes and 512
// threads (0.36 ms a stage in that measurement; 0.46 on sixteen CTAs of two planes, 0.80 on one CTA), one
// instance at n = 20 on eleven CTAs of two planes (62 us; 120 on two CTAs).
template <typename T, typename W>
FsChoice choose(const Launch& L, const MeshView& M, int B) {
    // groups of 1, 2 and 4 systems with an active instance
    int groups[3];
    for (int v = 0; v < 3; ++v) {
        const int vec = 1 << v;
        groups[v] = 0;
        for (int gi = 0; B % vec == 0 && gi < B / vec; ++gi) {
            bool a = L.active == nullptr;
            for (int i = 0; i < vec && !a; ++i) a = L.active[gi * vec + i] != 0;
            groups[v] += 2 * a;   // forward and adjoint systems
        }
        groups[v] = std::max(1, groups[v]);
    }
    // the search takes some 10 us: its results are kept (a bounded number of them)
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, int, int, int, int>, FsChoice> known;
    int dev = 0;
    cudaGetDevice(&dev);
    const auto key = std::make_tuple(dev, M.n, B, groups[0], groups[1], groups[2], L.max_blocks);
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = known.find(key);
        if (it != known.end()) return it->second;
    }
    FsChoice c;
    double cost = 0.0;
    // mixed iterations run one system per cluster: their FP64 residual gathers gain
    // nothing from vectors of instances (32 at n = 30: 1.9 ms for two stages, 2.2 with
    // two systems, 3.9 with four; the best shape of all eleven measured sizes has one)
    if constexpr (sizeof(T) == 4) try_shapes<T, W, 4, true>(L, M.n, B, groups[2], c, cost);
    if constexpr (sizeof(T) == sizeof(W)) try_shapes<T, W, 2, true>(L, M.n, B, groups[1], c, cost);
    try_shapes<T, W, 1, true>(L, M.n, B, groups[0], c, cost);
    // (where batches have room for the planes in global memory)
    if (!c.vec && fast_scratch_words(M.n, sizeof(W))) try_shapes<T, W, 1, false>(L, M.n, B, groups[0], c, cost);
    std::lock_guard<std::mutex> lk(mu);
    if (known.size() >= 4096) known.clear();
    known.emplace(key, c);
    return c;
}

template <typename T, typename W, int VEC, bool TS>
cudaError_t launch_fast(const Launch& L, FsArgs<T, W>& a, const FsChoice& c) {
    cudaLaunchConfig_t cfg = {};
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
    cudaError_t e = cudaSuccess;
    a.clusters = c.clusters;
    for (a.first = 0; a.first < c.clusters && e == cudaSuccess; a.first += c.per) {
        cfg.gridDim = dim3((unsigned)(std::min(c.per, c.clusters - a.first) * c.g.cl));
        e = cudaLaunchKernelEx(&cfg, k_fast_solve<T, W, VEC, TS>, a);
        *L.launches += 1;
    }
    return e;
}

template <typename T, typename W>
cudaError_t solve_as(const Launch& L, const MeshView& M, const BatchView<T>& V, const PcgArgs<T>& P, bool* ok) {
    const FsChoice c = choose<T, W>(L, M, V.B);
    *ok = c.vec != 0;
    if (!c.vec) return cudaSuccess;
    FsArgs<T, W> a;
    a.P = P;
    a.g = c.g;
    if constexpr (sizeof(W) == 4) {
        a.mat = M.fast->mat32;
        a.inv = M.fast->inv32;
        a.edge = M.fast->edge32;
    } else {
        a.mat = M.fast->mat64;
        a.inv = M.fast->inv64;
        a.edge = M.fast->edge64;
    }
    a.gt = reinterpret_cast<W*>(V.fs);
    if (!c.ts && !a.gt) {
        *ok = false;
        return cudaSuccess;
    }
    switch (c.vec * 2 + (c.ts ? 1 : 0)) {
        case 9:
            if constexpr (sizeof(T) == 4) return launch_fast<T, W, 4, true>(L, a, c);
            return cudaErrorInvalidValue;
        case 5:
            if constexpr (sizeof(T) == sizeof(W)) return launch_fast<T, W, 2, true>(L, a, c);
            return cudaErrorInvalidValue;
        case 3: return launch_fast<T, W, 1, true>(L, a, c);
        default: return launch_fast<T, W, 1, false>(L, a, c);
    }
}

template <typename T, typename W>
int64_t shape_as(const Launch& L, const MeshView& M, int B) {
    const FsChoice c = choose<T, W>(L, M, B);
    if (!c.vec) return 0;
    return ((((int64_t)c.vec * 32 + c.g.cl) * 2 + c.ts) * 1024 + c.clusters) * 2048 + c.threads;
}

}  // namespace

bool fast_qualifies(const Launch& L, const MeshView& M, int B) {
    return M.fast && !M.gen && L.pcg_kernel == 0 && !L.wait_test && B >= 1 && B <= 256 && M.n + 1 <= FS_MAX_N1;
}

int64_t fast_shape(const Launch& L, const MeshView& M, int B, bool fp64, bool mixed_iter) {
    if (!fast_qualifies(L, M, B)) return 0;
    if (!fp64) return shape_as<float, float>(L, M, B);
    return mixed_iter ? shape_as<double, float>(L, M, B) : shape_as<double, double>(L, M, B);
}

template <typename T>
int fast_solve(const Launch& L, const MeshView& M, const BatchView<T>& V, int mode, double tol, int max_iter,
               bool mixed_iter, cudaError_t* err) {
    *err = cudaSuccess;
    if (!fast_qualifies(L, M, V.B)) return 0;
    PcgArgs<T> P{M, V, mode, tol * tol, max_iter, L.bar, L.err, L.sweeps, L.fin};
    bool ok = false;
    if constexpr (sizeof(T) == 4) *err = solve_as<T, float>(L, M, V, P, &ok);
    else if (mixed_iter) *err = solve_as<T, float>(L, M, V, P, &ok);
    else *err = solve_as<T, double>(L, M, V, P, &ok);
    return ok || *err != cudaSuccess;
}

template int fast_solve<float>(const Launch&, const MeshView&, const BatchView<float>&, int, double, int, bool, cudaError_t*);
template int fast_solve<double>(const Launch&, const MeshView&, const BatchView<double>&, int, double, int, bool, cudaError_t*);

// Words of one system's transformed planes in global memory (0: they fit the
// shared memory of a cluster).
size_t fast_scratch_words(int n, size_t word) {
    for (int ppc = 1; ppc <= n + 1; ++ppc) {
        FsGeo g = base_geo(n);
        if (fit_geo(g, 1, ppc, word, word == 8 ? 512 : 1024, true)) return 0;
    }
    return (size_t)(n + 1) * base_geo(n).ss;
}

void fast_sizes(int n, FastTables& t) {
    const FsGeo g = base_geo(n);
    t.words = g.matw;
    t.inv = (size_t)g.s2 * g.ss;
    t.ldx = g.ldx;
}

void fast_tables(int n, FastTables& t) {
    const FsGeo g = base_geo(n);
    fast_sizes(n, t);
    t.mat.assign((size_t)2 * g.matw, 0.0);
    t.lam_row.assign((size_t)2 * g.s2, -1.0);
    t.lam_col.assign((size_t)2 * g.ldx, -1.0);
    const double pi = 3.14159265358979323846;
    for (int kind = 0; kind < 2; ++kind)
        for (int odd = 0; odd < 2; ++odd) {
            const int len = odd ? g.ho : g.h, pad = odd ? g.hop : g.hp;
            double* F = t.mat.data() + (size_t)kind * g.matw + (odd ? 2 * (size_t)g.hp * g.hp : 0);
            double* G = F + (size_t)pad * pad;
            int c = 0;   // modes of this parity so far
            for (int m = kind; m <= (kind ? n - 1 : n); ++m) {
                // cos(pi m k / n) is even about the centre for even m, sin for odd m
                if (((m + kind) & 1) != odd) continue;
                const double s = sin(0.5 * pi * m / n), l = 4.0 * s * s;
                for (int k = 0; k < len; ++k) {
                    const int pt = odd ? g.ho - 1 - k : k;   // the odd part of (k, n-k) stands at n-k
                    const double ang = pi * (double)(((long long)m * pt) % (2 * n)) / n;
                    const double v = kind ? sqrt(2.0 / n) * sin(ang)
                                          : sqrt((m == 0 || m == n ? 1.0 : 2.0) / n) * cos(ang);
                    F[(size_t)k * pad + c] = v;
                    G[(size_t)c * pad + k] = v;
                }
                t.lam_row[(size_t)kind * g.s2 + (odd ? g.h : 0) + c] = l;
                t.lam_col[(size_t)kind * g.ldx + (odd ? g.hp : 0) + c] = l;
                ++c;
            }
        }
}

// X = A^-1 by Newton's iteration X <- X (2 - A X) from X = 2 - A: the residual
// 1 - A X squares at every step, (1 - A)^32 after four (spectral radius of 1 - A at
// most 1/3: 5e-16).  Set-up work of a mesh; one output per thread in 16 x 16 tiles
// keeps the FP64 units of all SMs busy from n = 20 on (20 us a product there, where
// 64 x 64 tiles on a few SMs took 250 us).
template <bool FIRST>
__global__ void __launch_bounds__(256) k_newton_mm(int n, const double* __restrict__ A, const double* __restrict__ Bm,
                                                   const double* __restrict__ X, double* __restrict__ Y) {
    // Y = A B, or (X given) Y = 2 X - A B
    __shared__ double As[16][17], Bs[16][17];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, i = blockIdx.y * 16 + ty, j = blockIdx.x * 16 + tx;
    double acc = 0.0;
    for (int k = 0; k < n; k += 16) {
        As[ty][tx] = i < n && k + tx < n ? A[(size_t)i * n + k + tx] : 0.0;
        Bs[ty][tx] = k + ty < n && j < n ? Bm[(size_t)(k + ty) * n + j] : 0.0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16; ++q) acc = fma(As[ty][q], Bs[q][tx], acc);
        __syncthreads();
    }
    if (i < n && j < n) Y[(size_t)i * n + j] = FIRST ? acc : 2.0 * X[(size_t)i * n + j] - acc;
}
__global__ void k_newton_start(int n, const double* __restrict__ A, double* __restrict__ X) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)n * n; i += (size_t)gridDim.x * blockDim.x)
        X[i] = (i / n == i % n ? 2.0 : 0.0) - A[i];
}
void launch_inverse_newton(int n, const double* A, double* X, double* T1, double* T2, cudaStream_t st) {
    const dim3 grid((n + 15) / 16, (n + 15) / 16);
    k_newton_start<<<256, 256, 0, st>>>(n, A, T2);
    double *cur = T2, *nxt = X;
    for (int k = 0; k < 4; ++k) {
        k_newton_mm<true><<<grid, 256, 0, st>>>(n, A, cur, nullptr, T1);
        k_newton_mm<false><<<grid, 256, 0, st>>>(n, cur, T1, cur, nxt);
        std::swap(cur, nxt);
    }
    if (cur != X) cudaMemcpyAsync(X, cur, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, st);
}

// E of the edge nodes: sum of delta (e_i - e_j)(e_i - e_j)^T over the edges along
// the cube's twelve lines, delta = -1/2 where the stiffness has -1, +1/2 where -2
// (K_T: -3/2); as a list of neighbours per node.
namespace {
struct EdgeNb {
    int e;
    double d;
};
int edge_id(int i, int j, int k, int n) {
    const bool bi = i == 0 || i == n, bj = j == 0 || j == n, bk = k == 0 || k == n;
    if (bj && bk) return ((j != 0) + 2 * (k != 0)) * (n + 1) + i;
    if (bi && bk) return 4 * (n + 1) + ((i != 0) + 2 * (k != 0)) * (n - 1) + j - 1;
    return 4 * (n + 1) + 4 * (n - 1) + ((i != 0) + 2 * (j != 0)) * (n - 1) + k - 1;
}
}  // namespace

// A = 1 + R E (ne x ne, row-major), R = K_T^+ between edge nodes.  Every node is
// taken on one line: (axis, position t along it, ends b, c of the two other axes in
// axis order).  With q0[m] = Q[0][m], Q[n][m] = (-1)^m q0[m]:
//   lines of one axis: sum_m Q[t][m] Q[t'][m] W_s(m), W the sum over the two other
//     modes of q0^2 q0^2 / 6(l + l + l), with a sign (-1)^m' where the ends differ;
//   lines of two axes: sum Q[t*][m] q0[m] V_s(m, m') q0[m'] Q[t'*][m'], V the sum over
//     the third mode of q0^2 / 6(l + l + l), t* = t or n - t by the other line's end.
void fast_edge_system(int n, std::vector<double>& A) {
    const int s = n + 1, ne = 12 * n - 4;
    const double pi = 3.14159265358979323846;
    std::vector<double> Q((size_t)s * s), lam(s), q0(s);
    for (int m = 0; m < s; ++m) {
        const double sn = sin(0.5 * pi * m / n);
        lam[m] = 4.0 * sn * sn;
        for (int t = 0; t < s; ++t)
            Q[(size_t)t * s + m] = sqrt((m == 0 || m == n ? 1.0 : 2.0) / n) * cos(pi * (double)(((long long)m * t) % (2 * n)) / n);
        q0[m] = Q[m];
    }
    auto inv = [&](int a, int b, int c) { return a + b + c == 0 ? 0.0 : 1.0 / (6.0 * (lam[a] + lam[b] + lam[c])); };
    std::vector<double> V[2], Wp[2][2], Pm[2][2], Cm[2];
    for (int sg = 0; sg < 2; ++sg) {
        V[sg].assign((size_t)s * s, 0.0);
        for (int a = 0; a < s; ++a)
            for (int b = 0; b < s; ++b) {
                double acc = 0.0;
                for (int c = 0; c < s; ++c) acc += q0[c] * q0[c] * inv(a, b, c) * (sg && (c & 1) ? -1.0 : 1.0);
                V[sg][(size_t)a * s + b] = acc;
            }
    }
    for (int s1 = 0; s1 < 2; ++s1)
        for (int s2 = 0; s2 < 2; ++s2) {
            Wp[s1][s2].assign(s, 0.0);
            for (int a = 0; a < s; ++a)
                for (int b = 0; b < s; ++b)
                    Wp[s1][s2][a] += q0[b] * q0[b] * V[s2][(size_t)a * s + b] * (s1 && (b & 1) ? -1.0 : 1.0);
            Pm[s1][s2].assign((size_t)s * s, 0.0);
            for (int t = 0; t < s; ++t)
                for (int u = 0; u < s; ++u) {
                    double acc = 0.0;
                    for (int m = 0; m < s; ++m) acc += Q[(size_t)t * s + m] * Q[(size_t)u * s + m] * Wp[s1][s2][m];
                    Pm[s1][s2][(size_t)t * s + u] = acc;
                }
        }
    for (int sg = 0; sg < 2; ++sg) {
        std::vector<double> t1((size_t)s * s, 0.0);   // (Q q0) V
        for (int t = 0; t < s; ++t)
            for (int a = 0; a < s; ++a) {
                const double f = Q[(size_t)t * s + a] * q0[a];
                for (int b = 0; b < s; ++b) t1[(size_t)t * s + b] += f * V[sg][(size_t)a * s + b];
            }
        Cm[sg].assign((size_t)s * s, 0.0);
        for (int t = 0; t < s; ++t)
            for (int u = 0; u < s; ++u) {
                double acc = 0.0;
                for (int b = 0; b < s; ++b) acc += t1[(size_t)t * s + b] * q0[b] * Q[(size_t)u * s + b];
                Cm[sg][(size_t)t * s + u] = acc;
            }
    }
    struct Node {
        int ax, t, end[3];   // end[a]: 0 or 1 on the other axes
    };
    std::vector<Node> nd(ne);
    std::vector<std::vector<EdgeNb>> nb(ne);
    for (int ax = 0; ax < 3; ++ax)
        for (int b = 0; b < 2; ++b)
            for (int c = 0; c < 2; ++c) {
                const int a1 = ax == 0 ? 1 : 0, a2 = ax == 2 ? 1 : 2;
                int prev = -1;
                for (int t = 0; t <= n; ++t) {
                    int x[3];
                    x[ax] = t;
                    x[a1] = b ? n : 0;
                    x[a2] = c ? n : 0;
                    const int e = edge_id(x[0], x[1], x[2], n);
                    if (ax == 0 || (t > 0 && t < n)) {
                        nd[e].ax = ax;
                        nd[e].t = t;
                        nd[e].end[ax] = 0;
                        nd[e].end[a1] = b;
                        nd[e].end[a2] = c;
                    }
                    if (t) {
                        const double dl = b == c ? 0.5 : -0.5;
                        nb[e].push_back({prev, dl});
                        nb[prev].push_back({e, dl});
                    }
                    prev = e;
                }
            }
    auto Rv = [&](const Node& e, const Node& f) {
        if (e.ax == f.ax) {
            const int a1 = e.ax == 0 ? 1 : 0, a2 = e.ax == 2 ? 1 : 2;
            return Pm[e.end[a1] != f.end[a1]][e.end[a2] != f.end[a2]][(size_t)e.t * s + f.t];
        }
        const int third = 3 - e.ax - f.ax;
        const int te = f.end[e.ax] ? n - e.t : e.t, tf = e.end[f.ax] ? n - f.t : f.t;
        return Cm[e.end[third] != f.end[third]][(size_t)te * s + tf];
    };
    A.assign((size_t)ne * ne, 0.0);
    for (int e = 0; e < ne; ++e) {
        double* row = A.data() + (size_t)e * ne;
        row[e] = 1.0;
        for (int f = 0; f < ne; ++f) {
            const double r = Rv(nd[e], nd[f]);
            for (const EdgeNb& v : nb[f]) {   // (R E)[e][.] += R[e][f] E[f][.]
                row[f] += r * v.d;
                row[v.e] -= r * v.d;
            }
        }
    }
}

// H = E - E X with X = (1 + R E)^-1 (ne x ne, row-major).
void fast_edge_matrix(int n, const std::vector<double>& X, std::vector<double>& H) {
    const int ne = 12 * n - 4;
    H.assign((size_t)ne * ne, 0.0);
    auto line = [&](int ax, int b, int c, int t) {
        int x[3];
        x[ax] = t;
        x[ax == 0 ? 1 : 0] = b ? n : 0;
        x[ax == 2 ? 1 : 2] = c ? n : 0;
        return edge_id(x[0], x[1], x[2], n);
    };
    for (int ax = 0; ax < 3; ++ax)
        for (int b = 0; b < 2; ++b)
            for (int c = 0; c < 2; ++c)
                for (int t = 0; t < n; ++t) {
                    const int e = line(ax, b, c, t), f = line(ax, b, c, t + 1);
                    const double dl = b == c ? 0.5 : -0.5;
                    double *he = H.data() + (size_t)e * ne, *hf = H.data() + (size_t)f * ne;
                    const double *xe = X.data() + (size_t)e * ne, *xf = X.data() + (size_t)f * ne;
                    for (int g = 0; g < ne; ++g) {
                        const double v = dl * ((g == e) - (g == f) - xe[g] + xf[g]);
                        he[g] += v;
                        hf[g] -= v;
                    }
                }
    for (int e = 0; e < ne; ++e)   // H is symmetric: rounding aside
        for (int f = 0; f < e; ++f) {
            const double v = 0.5 * (H[(size_t)e * ne + f] + H[(size_t)f * ne + e]);
            H[(size_t)e * ne + f] = H[(size_t)f * ne + e] = v;
        }
}

void launch_fast_inv(int n, const double* lam_row, const double* lam_col, double* inv64, float* inv32, cudaStream_t st) {
    const FsGeo g = base_geo(n);
    for (int kind = 0; kind < 2; ++kind)
        k_fast_inv<<<256, 256, 0, st>>>(g.s2, g.ldx, lam_row + (size_t)kind * g.s2, lam_col + (size_t)kind * g.ldx,
                                        inv64 + (size_t)kind * g.s2 * g.ss, inv32 + (size_t)kind * g.s2 * g.ss);
}

}  // namespace lbm
