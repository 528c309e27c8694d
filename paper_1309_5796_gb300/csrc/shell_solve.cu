// Scalar potential with the open boundary by space transformation (Sec. 3.1:
// the scheme of the paper's own steepest-descent solver): the magnet, an air
// box and a shell mapped onto the rest of space share one Kuhn grid; the
// shell's tetrahedra carry the tensor M = |det J| J^-1 J^-T of the map, the
// outer face (the image of infinity) has u = 0, and one symmetric solve
//     K_grid u = b      (b = (1/4) Gint m at the magnet's nodes, 0 elsewhere)
// gives the total potential, whose lumped gradient at the magnet's nodes is
// exactly the gradient field of the stray-field energy (no boundary matrix, no
// adjoint chain).  The host set-up (csrc/shell.cu) builds the grid and its
// stiffness; here the solve runs on the device for all instances of a batch
// at once: CG with a Chebyshev polynomial of the Jacobi-scaled matrix as
// preconditioner, one persistent cooperative kernel per solve (grid barriers with
// the context's time limit), the grid potential warm-started from the instance's
// previous solve.
//
// Every row that is not on the outer face is an interior node of the grid, and
// the Kuhn split couples a node only to the 14 neighbours along +-x, +-y, +-z,
// +-(x+y), +-(x+z), +-(y+z), +-(x+y+z).  The operator is therefore applied as a
// stencil with per-row coefficients (no column indices): a 16-value record per
// row (diagonal, the 14 couplings in that order, 1/K_ii).  Where M = I (the
// magnet and the air) the diagonal couplings vanish and the row takes the
// 7-point form.
#include <type_traits>

#include "solver_common.cuh"

namespace lbm {
namespace {

template <typename W>
struct ShellArgs {
    ShellDev S;
    int B;
    const InstState* st;
    const double* bvec;           // [N][B] divergence right-hand side of the magnet
    double* x;                    // [Ng][B] FP64 grid potential
    W *r, *z, *z2, *p, *q, *d;   // [Ng][B] work vectors (d: this solve's correction of x)
    double th, de;                // centre and half-width of the polynomial's interval
    int deg;                      // products of a CG iteration
    int deal;                     // rows dealt round all blocks instead of a run for each
    double tol2;
    int max_iter;
    unsigned* bar;
    int* err;
    double* part;
    double* fin;
    unsigned long long* sweeps;
};

template <typename C> struct CoefLoad;
template <> struct CoefLoad<float> {
    __device__ static void row(const float* p, float (&c)[16]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(p) + k);
            c[4 * k] = v.x; c[4 * k + 1] = v.y; c[4 * k + 2] = v.z; c[4 * k + 3] = v.w;
        }
    }
};
template <> struct CoefLoad<double> {
    __device__ static void row(const double* p, double (&c)[16]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double2 v = __ldg(reinterpret_cast<const double2*>(p) + k);
            c[2 * k] = v.x; c[2 * k + 1] = v.y;
        }
    }
};

// VEC consecutive values (instances c0 .. c0+VEC-1 of one row).  Values that other
// blocks wrote are read after a grid barrier, whose acquire makes plain loads (and so
// the L1, which serves a product's neighbours) see them; CG: past the L1.
template <int VEC, bool CG, typename W>
__device__ __forceinline__ void ldv(W (&d)[VEC], const W* p) {
    if constexpr (VEC == 1) {
        d[0] = CG ? __ldcg(p) : *p;
    } else if constexpr (std::is_same<W, float>::value && VEC == 4) {
        const float4 v = CG ? __ldcg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(p);
        d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    } else if constexpr (std::is_same<W, float>::value && VEC == 2) {
        const float2 v = CG ? __ldcg(reinterpret_cast<const float2*>(p)) : *reinterpret_cast<const float2*>(p);
        d[0] = v.x; d[1] = v.y;
    } else {   // doubles, VEC = 2 or 4: 16-byte loads
#pragma unroll
        for (int k = 0; k < VEC; k += 2) {
            const double2 v = CG ? __ldcg(reinterpret_cast<const double2*>(p + k)) : *reinterpret_cast<const double2*>(p + k);
            d[k] = v.x; d[k + 1] = v.y;
        }
    }
}
template <int VEC, typename W>
__device__ __forceinline__ void stv(W* p, const W (&d)[VEC]) {
    if constexpr (VEC == 1) {
        *p = d[0];
    } else if constexpr (std::is_same<W, float>::value && VEC == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(d[0], d[1], d[2], d[3]);
    } else if constexpr (std::is_same<W, float>::value && VEC == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(d[0], d[1]);
    } else {
#pragma unroll
        for (int k = 0; k < VEC; k += 2) *reinterpret_cast<double2*>(p + k) = make_double2(d[k], d[k + 1]);
    }
}

// (K v)_row for VEC instances (ADD: plus w): v points at the row's first value; sx, sy, sz
// are the strides of one grid step along x, y, z in v.
template <int VEC, bool ADD = false, typename R, typename C, typename V>
__device__ __forceinline__ void kuhn_apply(const C (&c)[16], const V* v, ptrdiff_t sx, ptrdiff_t sy, ptrdiff_t sz,
                                           bool full, R (&w)[VEC]) {
    const ptrdiff_t off[15] = {0, sx, -sx, sy, -sy, sz, -sz, sx + sy, -sx - sy, sx + sz, -sx - sz, sy + sz, -sy - sz,
                               sx + sy + sz, -sx - sy - sz};
    if (!ADD) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) w[k] = R(0);
    }
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        V t[VEC];
        ldv<VEC, false>(t, v + off[j]);
#pragma unroll
        for (int k = 0; k < VEC; ++k) w[k] += R(c[j]) * R(t[k]);
    }
    if (full) {
#pragma unroll
        for (int j = 7; j < 15; ++j) {
            V t[VEC];
            ldv<VEC, false>(t, v + off[j]);
#pragma unroll
            for (int k = 0; k < VEC; ++k) w[k] += R(c[j]) * R(t[k]);
        }
    }
}

// Products of a CG iteration and the ratio of the polynomial's interval.  A higher degree
// saves reductions and their barriers; but an iteration is a whole number of polynomials,
// and a small grid needs few: 11^3 nodes 97 plain CG iterations in FP64, twenty of degree
// 16.  ms an evaluation at degree, ratio (first plain CG, last what every grid had):
//   6^3, 64 instances in FP64    0.95 | 3, 8: 0.84   4, 15: 0.91   8, 60: 1.28
//   7^3, 64 in FP64              1.13 | 3, 8: 1.06   4, 15: 1.04   6, 30: 1.13   8, 60: 1.35
//   9^3, 64 in FP64                   | 4, 15: 1.40   6, 30: 1.38   8, 60: 1.51   16, 400: 3.06
//   11^3, 256 in FP64            3.71 | 6, 30: 3.06   8, 60: 3.31   12, 220: 4.60   16, 400: 6.05
//   11^3, 64 in FP32             1.03 | 6, 30: 0.72   8, 60: 0.72   12, 220: 0.82   16, 400: 1.03
//   17^3, 64 in FP64                  | 8, 60: 4.21   8, 100: 4.08   12, 220: 4.49   16, 400: 5.24
//   21^3, 128 in FP64            13.3 | 8, 100: 11.7   12, 220: 11.7   16, 400: 13.4
//   27^3, 16 in FP32                  | 8, 100: 1.62   12, 220: 1.48   16, 400: 1.39
//   39^3, 32 in FP64                  | 8, 100: 39.1   12, 220: 38.0   16, 400: 37.1
// The lines lie between these sizes.
constexpr int SH_DEG_MAX = 16;
void sh_degree(int rows, int& deg, double& ratio) {
    struct Step {
        int rows, deg;
        double ratio;
    };
    static constexpr Step steps[] = {{280, 3, 8.0},     {600, 4, 15.0},     {1000, 6, 30.0},
                                     {2500, 8, 60.0},   {6500, 8, 100.0},   {14000, 12, 220.0}};
    deg = SH_DEG_MAX;
    ratio = 400.0;
    for (const Step& t : steps)
        if (rows <= t.rows) {
            deg = t.deg;
            ratio = t.ratio;
            return;
        }
}
// rows times instances from which on FP64 batches deal their rows round all blocks: odd
// batches, one instance a thread, and even ones, two
constexpr double SH_DEAL1 = 3e5, SH_DEAL2 = 8e5;

// Threads hold VEC consecutive instances of one row: thread tid works on
// instances c0 = (tid % G) VEC .. c0 + VEC - 1 (G = B / VEC) of row lane tid / G.
// W is the type of the CG work vectors and of the per-thread and per-block
// dot-product sums (grid totals in FP64):
//   W = double: plain FP64 CG on K d = f - K x, then x += d;
//   W = float, RES64 = false (the FP32 phase of a mixed run): the residual of
//     the warm start in FP32 arithmetic, FP32 CG to the tolerance, x += d;
//   W = float, RES64 = true (FP64 solves with mixed iterations): cycles of the
//     FP64 residual f - K x, FP32 CG until it has reduced that residual by
//     MP_INNER (or met the tolerance), x += d; the solve ends on the FP64
//     residual test (restarted CG, as the magnet's mixed-iteration solves).
// Per CG iteration:
//   B: alpha = rho / p.q, d += alpha p, r -= alpha q, z = D^-1 r / theta, r.r
//   C: deg - 1 steps z'' = z' + c1 (z' - z) + c2 D^-1 (r - K z'), z'' in z's place (no
//      vector for the steps themselves); r.z with the last
//   A: w = K z, p = z + beta p, q = w + beta q (= K p), p.q
// The polynomial is Chebyshev's on [b / ratio, b], b a bound of the eigenvalues of
// D^-1 K, its degree by size (sh_degree): on the 54^3-cell grid 29 iterations of 16
// products where Jacobi-CG takes 358 of one, and a product with its step moves 4 vector
// words and one barrier where a CG iteration moves 12 and four.  (20 on [b / 800, b] gives
// 3 % more on that grid.  Multigrid and fast diagonalisation stall on the shell's growing
// tangential stiffness.)
// Measured on that grid: 0.36 ms an iteration of 32 instances, 0.083 of one; an evaluation of
// smooth states (34 iterations) 12.5 and 2.9 ms, with Jacobi-CG 28.6 and 6.8.
// Every block has one run of consecutive rows, so that the L1 serves a product's
// neighbours along x and y and about three of its fifteen reads go to L2 (with
// rows dealt round all blocks and loads past the L1, all fifteen did).
// Outer-face rows keep zero in every vector (and 1/K_ii = 0 there), so they
// drop out of every product.
template <typename W, bool RES64, int THREADS, int VEC>
__global__ void __launch_bounds__(THREADS, 1) k_shell_pcg(ShellArgs<W> A) {
    using R0 = typename std::conditional<RES64 || std::is_same<W, double>::value, double, float>::type;
    extern __shared__ double sm[];
    const int B = A.B, tid = threadIdx.x, bd = blockDim.x;
    const int G = B / VEC, RB = bd / G;
    const bool lane = tid < RB * G;
    const int g = tid % G, c0 = g * VEC, rl = tid / G;
    const int nrow = (G <= 32 && (32 % G) == 0) ? (bd >> 5) : RB;
    double* scratch = sm;                          // [2][nrow][B] doubles (or floats in the same room)
    double* out = scratch + 2 * (size_t)nrow * B;  // [2][B]
    double* s_rho = out + 2 * B;
    double* s_rhop = s_rho + B;
    double* s_ab = s_rhop + B;
    double* s_tol = s_ab + B;
    double* s_tin = s_tol + B;
    int* s_flag = (int*)(s_tin + B);
    int* s_act = s_flag + B;
    int* s_it = s_act + B;
    int* s_done = s_it + B;
    // alpha or beta of the current step in W for the row loops (a conversion from
    // FP64 per thread would issue at GB300's FP64 rate)
    W* s_abw = reinterpret_cast<W*>(s_done + B);   // 8-byte aligned: four int arrays of B
    for (int i = tid; i < B; i += bd) {
        s_act[i] = A.st[i].phase != PH_DONE;
        s_it[i] = 0;
        s_done[i] = 0;
    }
    __syncthreads();
    bool act[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) act[k] = lane && s_act[c0 + k];
    const int Ng = A.S.Ng, n1 = A.S.n1;
    const ptrdiff_t sx = B, sy = (ptrdiff_t)n1 * B, sz = (ptrdiff_t)n1 * n1 * B;
    const W* coefW;
    if constexpr (std::is_same<W, double>::value) coefW = A.S.coef64;
    else coefW = A.S.coef32;
    // a run of consecutive rows for each block (the header says why), or, where the FP64
    // units bind, rows dealt round all blocks, so that each has its share of the 7- and of
    // the 15-point rows (ms an evaluation, runs -> dealt.  Odd batches above the line: 13
    // instances on 29 791 nodes 9.90 -> 9.12, 33 20.3 -> 18.2, 3 on 117 649 15.7 -> 15.9,
    // 25 94.3 -> 84.1, 17 on 166 375 104 -> 90; below it 9 on 29 791 7.46 -> 7.67, 7 6.26 ->
    // 6.55.  Even ones above: 32 on 29 791 17.3 -> 15.3, 8 on 117 649 30.2 -> 28.4, 32 104 ->
    // 91.5, 16 on 166 375 86.4 -> 76.5; below 8 on 29 791 6.25 -> 7.01, 4 on 166 375 25.3 ->
    // 26.8, 2 16.0 -> 18.5, though 16 on 29 791 10.5 -> 9.2, 4 on 117 649 17.5 -> 16.1)
    const int rpb = (Ng + (int)gridDim.x - 1) / (int)gridDim.x, rstep = A.deal ? (int)gridDim.x * RB : RB;
    const int rlo = (int)blockIdx.x * (A.deal ? RB : rpb);
    const int rhi = !lane ? 0 : A.deal ? Ng : min(Ng, rlo + rpb);   // idle lanes have no rows
    const int row0 = rlo + rl;
    const W th = W(A.th), de = W(A.de);
    unsigned epoch = 0;
    // totals of v over the grid into out (NQ quantities of B instances)
    auto publish = [&](auto& v) -> bool {
        constexpr int NQ = sizeof(v) / sizeof(v[0]);
        using R = typename std::remove_reference<decltype(v[0][0])>::type;
        block_reduce_cols<NQ, VEC, R>(v, reinterpret_cast<R*>(scratch), out, B, G, RB);
        if (tid < B)
            for (int k = 0; k < NQ; ++k) A.part[((size_t)blockIdx.x * B + tid) * 4 + k] = out[k * B + tid];
        return grid_reduce<NQ>(A.part, 0, B, A.fin, out, A.bar, epoch, A.err);
    };
    W* z = A.z;
    W* zo = A.z2;   // the steps alternate between the two
    for (int cycle = 0;; ++cycle) {
        // residual of the current x: r = f - K x, z = D^-1 r / theta, zero outer faces
        {
            R0 v[2][VEC];   // r.r, f.f
#pragma unroll
            for (int k = 0; k < VEC; ++k) v[0][k] = v[1][k] = R0(0);
            const W zero[VEC] = {};
            for (int row = row0; row < rhi; row += rstep) {
                const size_t i = (size_t)row * B + c0;
                const int kind = __ldg(&A.S.kind[row]);
                if (kind == 0) {   // outer face: u = 0
                    stv<VEC>(A.r + i, zero);
                    stv<VEC>(z + i, zero);
                    stv<VEC>(zo + i, zero);
                    stv<VEC>(A.p + i, zero);
                    stv<VEC>(A.q + i, zero);
                    stv<VEC>(A.d + i, zero);
                    continue;
                }
                const int gn = __ldg(&A.S.gnode[row]);
                double f[VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) f[k] = 0.0;
                if (gn >= 0) ldv<VEC, false>(f, A.bvec + (size_t)gn * B + c0);
                R0 kx[VEC];
                W dinv;
                if constexpr (std::is_same<R0, double>::value) {
                    double c[16];
                    CoefLoad<double>::row(A.S.coef64 + (size_t)row * 16, c);
                    kuhn_apply<VEC>(c, A.x + i, sx, sy, sz, kind == 2, kx);
                    dinv = W(c[15]);
                } else {
                    float c[16];
                    CoefLoad<float>::row(A.S.coef32 + (size_t)row * 16, c);
                    kuhn_apply<VEC>(c, A.x + i, sx, sy, sz, kind == 2, kx);
                    dinv = c[15];
                }
                W rw[VEC], zw[VEC];
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    if (!act[k]) f[k] = 0.0;
                    const R0 rv = R0(f[k]) - kx[k];
                    rw[k] = W(rv);
                    zw[k] = rw[k] * (dinv / th);
                    if (act[k]) {
                        v[0][k] += rv * rv;
                        v[1][k] += R0(f[k]) * R0(f[k]);
                    }
                }
                stv<VEC>(A.r + i, rw);
                stv<VEC>(z + i, zw);
            }
            if (!publish(v)) return;
        }
        if (tid < B) {
            const double rr = out[tid];
            if (cycle == 0) s_tol[tid] = A.tol2 * out[B + tid];
            // (a residual that is no number ends the solve: no step mends it)
            s_done[tid] = !s_act[tid] || !(rr > s_tol[tid]) || s_it[tid] >= A.max_iter;
            s_tin[tid] = RES64 ? fmax(s_tol[tid], MP_INNER * MP_INNER * rr) : s_tol[tid];
            s_rhop[tid] = 1.0;
        }
        if (__syncthreads_and(tid < B ? s_done[tid] : 1)) break;
        int it = 0;
        for (;; ++it) {
            if (tid < B) {   // out: r.r
                if (it > 0) {
                    s_rhop[tid] = s_rho[tid];
                    if (!s_flag[tid]) s_it[tid] += 1;
                }
                s_flag[tid] = s_done[tid] || !(out[tid] > s_tin[tid]) || s_it[tid] >= A.max_iter;
            }
            if (__syncthreads_and(tid < B ? s_flag[tid] : 1)) break;
            bool run[VEC];
#pragma unroll
            for (int k = 0; k < VEC; ++k) run[k] = act[k] && !s_flag[c0 + k];
            // ---- C: outer-face rows (kind 0) keep zero ----
            W v1[1][VEC];
            W rho_c = de / th;
            // counted up to a constant: to A.deg the loop takes 2 % longer
            for (int st = SH_DEG_MAX - A.deg + 1, st1 = st; st < SH_DEG_MAX; ++st) {
                const bool last = st + 1 == SH_DEG_MAX;
                const W rn = W(1) / (W(2) * th / de - rho_c), c1 = rn * rho_c, c2 = W(2) * rn / de, c3 = W(1) + c1;
                rho_c = rn;
#pragma unroll
                for (int k = 0; k < VEC; ++k) v1[0][k] = W(0);
                for (int row = row0; row < rhi; row += rstep) {
                    const int kind = __ldg(&A.S.kind[row]);
                    if (kind == 0) continue;
                    const size_t i = (size_t)row * B + c0;
                    W c[16];
                    CoefLoad<W>::row(coefW + (size_t)row * 16, c);
                    W w[VEC], rv[VEC], tv[VEC], zv[VEC];
                    ldv<VEC, false>(rv, A.r + i);
                    ldv<VEC, false>(zv, z + i);
                    // z'' = (1 + c1) z' - c1 z - c2 D^-1 (K z' - r), in the place of z (none at first)
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        tv[k] = W(0);
                        w[k] = -rv[k];
                    }
                    if (st > st1) ldv<VEC, false>(tv, zo + i);
                    kuhn_apply<VEC, true>(c, z + i, sx, sy, sz, kind == 2, w);
                    const W di = c2 * c[15];
#pragma unroll
                    for (int k = 0; k < VEC; ++k) {
                        zv[k] = c3 * zv[k] - c1 * tv[k] - di * w[k];
                        if (last && run[k]) v1[0][k] += rv[k] * zv[k];
                    }
                    stv<VEC>(zo + i, zv);
                }
                W* t = z;
                z = zo;
                zo = t;
                if (!last && !grid_sync(A.bar, gridDim.x, epoch, A.err)) return;
            }
            if (!publish(v1)) return;   // r.z
            if (tid < B) {
                const double rho = out[tid];
                s_ab[tid] = (it == 0 || s_flag[tid]) ? 0.0 : rho / s_rhop[tid];
                s_abw[tid] = W(s_ab[tid]);
                s_rho[tid] = rho;
            }
            __syncthreads();
            // ---- A ----
            W ab[VEC];
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                ab[k] = s_abw[c0 < B ? c0 + k : 0];
                v1[0][k] = W(0);
            }
            for (int row = row0; row < rhi; row += rstep) {
                const int kind = __ldg(&A.S.kind[row]);
                if (kind == 0) continue;
                const size_t i = (size_t)row * B + c0;
                W c[16];
                CoefLoad<W>::row(coefW + (size_t)row * 16, c);
                W w[VEC], zi[VEC], pv[VEC], qv[VEC];
                ldv<VEC, false>(zi, z + i);
                if (it) {
                    ldv<VEC, false>(pv, A.p + i);
                    ldv<VEC, false>(qv, A.q + i);
                } else {
#pragma unroll
                    for (int k = 0; k < VEC; ++k) pv[k] = qv[k] = W(0);
                }
                kuhn_apply<VEC>(c, z + i, sx, sy, sz, kind == 2, w);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    pv[k] = zi[k] + ab[k] * pv[k];
                    qv[k] = w[k] + ab[k] * qv[k];
                    if (run[k]) v1[0][k] += pv[k] * qv[k];
                }
                stv<VEC>(A.p + i, pv);
                stv<VEC>(A.q + i, qv);
            }
            if (!publish(v1)) return;   // p.q
            if (tid < B) {
                s_ab[tid] = s_flag[tid] ? 0.0 : s_rho[tid] / out[tid];
                s_abw[tid] = W(s_ab[tid]);
            }
            __syncthreads();
            // ---- B, and the first step of the next polynomial, into the copy of z that no
            // block's products still read; outer-face rows need no test: their vectors
            // and 1/K_ii are zero, and stay so ----
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                ab[k] = s_abw[c0 < B ? c0 + k : 0];
                v1[0][k] = W(0);
            }
            for (int row = row0; row < rhi; row += rstep) {
                const size_t i = (size_t)row * B + c0;
                const W dt = __ldg(coefW + (size_t)row * 16 + 15) / th;
                W xa[VEC], pa[VEC], ra[VEC], qa[VEC];
                if (it) ldv<VEC, false>(xa, A.d + i);
                else
#pragma unroll
                    for (int k = 0; k < VEC; ++k) xa[k] = W(0);
                ldv<VEC, false>(pa, A.p + i);
                ldv<VEC, false>(ra, A.r + i);
                ldv<VEC, false>(qa, A.q + i);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    xa[k] += ab[k] * pa[k];
                    ra[k] -= ab[k] * qa[k];
                    pa[k] = ra[k] * dt;   // z
                    if (run[k]) v1[0][k] += ra[k] * ra[k];
                }
                stv<VEC>(A.d + i, xa);
                stv<VEC>(A.r + i, ra);
                stv<VEC>(zo + i, pa);
            }
            W* t = z;
            z = zo;
            zo = t;
            if (!publish(v1)) return;   // r.r
        }
        // fold the cycle's correction into x before anything reads x
        if (it > 0)
            for (int row = row0; row < rhi; row += rstep) {
                const size_t i = (size_t)row * B + c0;
                double xv[VEC];
                W dv[VEC];
                ldv<VEC, false>(xv, A.x + i);
                ldv<VEC, false>(dv, A.d + i);
#pragma unroll
                for (int k = 0; k < VEC; ++k) xv[k] += (double)dv[k];
                stv<VEC>(A.x + i, xv);
            }
        if (!RES64 || cycle + 1 >= MP_MAX_CYCLES) break;
        if (!grid_sync(A.bar, gridDim.x, epoch, A.err)) return;
    }
    if (blockIdx.x == 0) {
        for (int i = tid; i < B; i += bd)
            atomicAdd((unsigned long long*)&((InstState*)A.st)[i].cg1, (unsigned long long)s_it[i]);
        if (tid == 0 && A.sweeps) {
            int kmax = 0;
            for (int i = 0; i < B; ++i) kmax = max(kmax, s_it[i]);
            A.sweeps[std::is_same<W, float>::value && !RES64 ? 0 : 2] += (unsigned long long)kmax;
        }
    }
}

// The magnet's potential for the field kernel, which reads (U1 + U2 + U2adj)/2:
// U1 = u, U2 = 0 (forward columns), U2adj = u (the operator is symmetric).
template <typename T>
__global__ void k_shell_scatter(ShellDev S, int N, int B, const double* __restrict__ x, T* U1, T* U2) {
    const size_t total = (size_t)N * B;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int b = (int)(t % B);
        const size_t i = t / B;
        const T u = T(x[(size_t)S.magnet[i] * B + b]);
        U1[i * 2 * B + b] = u;
        U2[i * 2 * B + b] = T(0);
        U2[i * 2 * B + B + b] = u;
    }
}

template <typename W, bool RES64, int THREADS, int VEC>
int launch_shell(const Launch& L, const ShellDev& S, const double* bvec, double* shx, double* part, int B,
                 const InstState* st, double tol, int max_iter) {
    const int G = B / VEC, RB = THREADS / G;
    const int nrow = (G <= 32 && (32 % G) == 0) ? (THREADS >> 5) : RB;
    const size_t smem = sizeof(double) * (2 * (size_t)nrow * B + 7 * (size_t)B) + sizeof(int) * 4 * B + sizeof(W) * B;
    const void* fn = (const void*)k_shell_pcg<W, RES64, THREADS, VEC>;
    int occ = 1;
    cudaError_t e = kernel_smem_attr(fn, 160 * 1024, THREADS, smem, &occ);
    if (e != cudaSuccess) return (int)e;
    if (occ < 1) return (int)cudaErrorInvalidConfiguration;
    int nblk = (S.Ng + RB - 1) / RB;
    if (nblk > L.num_sms) nblk = L.num_sms;   // one block per SM (the partials hold one block per SM)
    const size_t Gv = (size_t)S.Ng * B;
    ShellArgs<W> a;
    a.S = S;
    a.B = B;
    a.st = st;
    a.bvec = bvec;
    a.x = shx;
    W* w = reinterpret_cast<W*>(shx + Gv);   // six work vectors after x
    a.r = w;
    a.z = w + Gv;
    a.p = w + 2 * Gv;
    a.q = w + 3 * Gv;
    a.d = w + 4 * Gv;
    a.z2 = w + 5 * Gv;
    double ratio;
    sh_degree(S.Ng, a.deg, ratio);
    a.th = 0.5 * (1.0 + 1.0 / ratio) * S.jac_bound;
    a.de = 0.5 * (1.0 - 1.0 / ratio) * S.jac_bound;
    a.deal = sizeof(W) == 8 && (double)S.Ng * B >= (VEC == 1 && B > 1 ? SH_DEAL1 : SH_DEAL2);
    a.tol2 = tol * tol;
    a.max_iter = max_iter;
    a.bar = L.bar;
    a.err = L.err;
    a.part = part;
    a.fin = L.fin;
    a.sweeps = L.sweeps;
    void* args[] = {&a};
    e = cudaMemsetAsync(L.bar, 0, sizeof(unsigned), L.stream);
    if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(fn, dim3(nblk), dim3(THREADS), args, smem, L.stream);
    return (int)e;
}

template <typename W, bool RES64, int THREADS>
int launch_shell_vec(const Launch& L, const ShellDev& S, const double* bvec, double* shx, double* part, int B,
                     const InstState* st, double tol, int max_iter) {
    // the widest vectors the batch allows (FP64 work vectors at most two wide)
    if constexpr (sizeof(W) == 4)
        if (B % 4 == 0) return launch_shell<W, RES64, THREADS, 4>(L, S, bvec, shx, part, B, st, tol, max_iter);
    if (B % 2 == 0) return launch_shell<W, RES64, THREADS, 2>(L, S, bvec, shx, part, B, st, tol, max_iter);
    return launch_shell<W, RES64, THREADS, 1>(L, S, bvec, shx, part, B, st, tol, max_iter);
}

}  // namespace

template <typename T>
int shell_solve(const Launch& L, const MeshView& M, const BatchView<T>& V, double tol, int max_iter, bool mixed_iter) {
    const ShellDev& S = *M.shell;
    const int B = V.B;
    if (B < 1 || B > 512) return (int)cudaErrorInvalidValue;
    int e;
    // FP32 iterations for FP32 batches and for FP64 solves with mixed iterations
    if (sizeof(T) == 4) e = launch_shell_vec<float, false, 1024>(L, S, V.bvec, V.shx, V.part, B, V.st, tol, max_iter);
    else if (mixed_iter) e = launch_shell_vec<float, true, 1024>(L, S, V.bvec, V.shx, V.part, B, V.st, tol, max_iter);
    else e = launch_shell_vec<double, false, 512>(L, S, V.bvec, V.shx, V.part, B, V.st, tol, max_iter);
    if (e) return e;
    size_t blocks = ((size_t)M.N * B + 255) / 256;
    if (blocks > (size_t)8 * L.num_sms) blocks = (size_t)8 * L.num_sms;
    k_shell_scatter<T><<<(unsigned)blocks, 256, 0, L.stream>>>(S, M.N, B, V.shx, V.U1, V.U2);
    *L.launches += 2;
    return 0;
}

template int shell_solve<float>(const Launch&, const MeshView&, const BatchView<float>&, double, int, bool);
template int shell_solve<double>(const Launch&, const MeshView&, const BatchView<double>&, double, int, bool);

}  // namespace lbm
