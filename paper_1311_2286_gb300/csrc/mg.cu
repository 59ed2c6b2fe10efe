// Row a9: the logical-space Poisson solve (Sec. II.B.3; eq. (poiscurv)), device resident.
//
// Discretisation (conservative finite volume with ghost cells): the flux through a face
// normal to axis a is a^{aa} (phi_R - phi_L) + sum_{b != a} a^{ab} / 4 [(phi_R(+b) + phi_L(+b))
// - (phi_R(-b) + phi_L(-b))], a^{ab} = Omega J g^{ab} from the geometry; Dirichlet ghosts
// 2 phi_b - phi_in (a Dirichlet face carries a^{aa} 2 (phi_in - phi_b)), Neumann ghosts
// phi_in (a Neumann face carries no flux), periodic wrap. The assembled row of cell c is
// M phi = Omega_c Q_c + (Dirichlet terms), M = -(divergence), stored as a 9-point (2D) or
// 19-point (3D) stencil of which only the 5/7 face entries are used when the map is
// orthogonal.
//
// Solver: multigrid, the method class the paper uses (Sec. II.B.3: coarse-grid correction
// plus Gauss-Seidel smoothing on each level), arranged for GB300, whose FP64 rate is ~1/64
// of its FP32 rate: the solution phi, the right-hand side and the residual are FP64, and
// each iteration solves for the correction with one FP32 V-cycle (mixed-precision
// iterative refinement):
//     r = b - M phi (FP64);  stop if ||r||_2 / ||b||_2 <= rtol;
//     e = V-cycle_FP32(M, float(r)) from e = 0;  phi += e (FP64).
// The FP32 cycle only has to reduce the error by its multigrid factor, so the iteration
// converges to FP64 accuracy at the rate of an FP64 multigrid.
// V-cycle: coarse levels rediscretised from the map sampled at every other vertex (BoxMG's
// variational coarse operators and operator-induced interpolation are not reproduced),
// restriction by summing the 2^D fine residuals (finite-volume conservation), (bi/tri)linear
// prolongation with homogeneous ghost rules, colour-ordered Gauss-Seidel (2 colours for
// 5/7-point stencils, 2^D colours with cross terms), levels of at most COARSE_CELLS cells
// inside one CTA, and a dense inverse on the coarsest level (bordered with the constant
// null vector when the problem is singular). A singular problem (no Dirichlet face) has its
// right-hand side projected by subtracting a uniform physical charge density and its
// solution gauged to sum_c J_c phi_c = 0.
//
// Optional outer Krylov iteration (cpic_set_solver): BiCGStab (van der Vorst 1992) on
// M phi = b, right-preconditioned by the same FP32 V-cycle, on the kernel-chain path. One
// iteration: p = r + beta (p - omega v); p^ = V(p); v = M p^, alpha = rho / (r^, v);
// s = r - alpha v; s^ = V(s); t = M s^, omega = (t, s) / (t, t); phi += alpha p^ + omega s^;
// then r = b - M phi is recomputed in FP64 (not updated), so the stopping test sees the true
// residual, and rho' = (r^, r), beta = (rho' / rho)(alpha / omega). A vanishing rho, alpha
// or omega restarts the recurrence with r^ = p = r. The direction vectors p, v, s and the
// products M p^ and M s^ only choose the search space and the step lengths alpha and omega:
// they are FP32 (the products with the FP32 copy of the full operator; FP64 on GB300 runs at
// 1/64 of the FP32 rate), while phi is only ever changed by FP64 additions of FP32 steps
// and the stopping test reads the FP64 residual, so the result's accuracy does not depend
// on them; the dot products accumulate in FP64.
//
// The residual kernel ends with a last-block reduction that decides whether to continue;
// it writes the decision into a CUDA graph conditional handle, so inside a captured step
// the cycle loop is a conditional WHILE node that runs on the device with no host round
// trip and no idle launches.
#include <cooperative_groups.h>
#include <stdlib.h>
#include <math.h>
#include <string.h>

#include <type_traits>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace cpic {
namespace {

constexpr int RED_BLOCKS = 256;
// The V-cycle drops the cross entries of the stencil (face entries only: 2D+1 points, two
// colours) when no finest-level row's cross entries sum to more than this fraction of its
// diagonal, e.g. the shell map, orthogonal up to O(h^2) terms of a few 1e-3; the residual
// and the Krylov products keep the full operator, so only the preconditioner changes.
constexpr float PC_CROSS_DROP = 0.02f;

__constant__ int c_off2[9][2] = {{0, 0}, {-1, 0}, {1, 0}, {0, -1}, {0, 1}, {-1, -1}, {1, -1}, {-1, 1}, {1, 1}};
// 3D slots: 19-point stencil, then the 8 corners that Galerkin coarse operators add
__constant__ int c_off3[27][3] = {{0, 0, 0},  {-1, 0, 0},  {1, 0, 0},  {0, -1, 0}, {0, 1, 0},
                                  {0, 0, -1}, {0, 0, 1},   {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0},
                                  {1, 1, 0},  {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1}, {1, 0, 1},
                                  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}, {0, 1, 1},
                                  {-1, -1, -1}, {1, -1, -1}, {-1, 1, -1}, {1, 1, -1},
                                  {-1, -1, 1}, {1, -1, 1}, {-1, 1, 1}, {1, 1, 1}};

template <typename R>
struct LV {
    int D;
    int n[3];
    int ncell;
    int S;      // stored stencil entries (9 / 27)
    int used;   // entries used (5/7 without cross terms, else 9 / 19, or 27 with Galerkin levels)
    int ncol;   // Gauss-Seidel colours (2 or 2^D)
    int per[3];
    int bc[6];
    const R* A;
    R* x;
    R* b;
    float* lw;  // 2D line relaxation: work [2][ncell] in global memory (FP32 levels)
    const R* dinv;  // inverse diagonal (FP32 levels)
    const R* pw;  // 2D operator-induced prolongation: own-parent weight per axis [2][ncell], or null
};

struct LVSet {
    int nl;
    int first_cta;  // first level solved inside one CTA
    int line;       // 1: alternating zebra line relaxation (2D) instead of point smoothing
    LV<float> l[MAX_LEVELS];
    int* status;    // DevCounters::mg_converged, for a wait that ran out
    const float* dense_inv;  // transposed
    int dense_m;   // unknowns of the coarsest level
    int singular;
};

template <typename R>
__device__ __forceinline__ void cell_coords(const LV<R>& L, int c, int* q) {
    q[0] = c % L.n[0];
    int r = c / L.n[0];
    q[1] = r % L.n[1];
    q[2] = r / L.n[1];
}

template <typename R>
__device__ __forceinline__ int lin(const LV<R>& L, const int* q) {
    return q[0] + L.n[0] * (q[1] + L.n[1] * q[2]);
}

__device__ __forceinline__ void offsets(int D, int k, int* o) {
    if (D == 2) {
        o[0] = c_off2[k][0];
        o[1] = c_off2[k][1];
        o[2] = 0;
    } else {
        o[0] = c_off3[k][0];
        o[1] = c_off3[k][1];
        o[2] = c_off3[k][2];
    }
}

// neighbour index with periodic wrap; non-periodic out-of-range entries have zero
// coefficients after assembly, their index is clamped (setup kernels only)
template <typename R>
__device__ __forceinline__ int nbr(const LV<R>& L, const int* q, const int* o) {
    int c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int v = q[a] + o[a];
        if (a < L.D) {
            if (v < 0) v = L.per[a] ? v + L.n[a] : 0;
            else if (v >= L.n[a]) v = L.per[a] ? v - L.n[a] : L.n[a] - 1;
        }
        c[a] = v;
    }
    return lin(L, c);
}

// stencil offset of slot k along axis a (2D: 9 slots, 3D: 27 slots); called with
// unrolled constant arguments, so it folds away
__host__ __device__ constexpr int koff(int D, int k, int a) {
    constexpr int t2[9][3] = {{0, 0, 0}, {-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0},
                              {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0}, {1, 1, 0}};
    constexpr int t3[27][3] = {{0, 0, 0},  {-1, 0, 0},  {1, 0, 0},  {0, -1, 0}, {0, 1, 0},  {0, 0, -1}, {0, 0, 1},
                               {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0}, {1, 1, 0},  {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                               {1, 0, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}, {0, 1, 1},
                               {-1, -1, -1}, {1, -1, -1}, {-1, 1, -1}, {1, 1, -1},
                               {-1, -1, 1}, {1, -1, 1}, {-1, 1, 1}, {1, 1, 1}};
    return D == 2 ? t2[k][a] : t3[k][a];
}

// sum_{k >= K0} A_k x_{nb_k} for cell q with compile-time stencil shape <D, NPT>: the
// wrapped/clamped neighbour coordinates are computed once per axis, slot offsets fold to
// constants
template <int D, int NPT, int K0, typename R>
__device__ __forceinline__ R stencil_sum(const LV<R>& L, int c, const int* q) {
    int lo[3], hi[3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        lo[a] = q[a] > 0 ? q[a] - 1 : (L.per[a] ? L.n[a] - 1 : 0);
        hi[a] = q[a] + 1 < L.n[a] ? q[a] + 1 : (L.per[a] ? 0 : L.n[a] - 1);
    }
    const int ix[3] = {lo[0], q[0], hi[0]};
    const int jy[3] = {L.n[0] * lo[1], L.n[0] * q[1], L.n[0] * hi[1]};
    int kz[3] = {0, 0, 0};
    if (D == 3) {
        const int pl = L.n[0] * L.n[1];
        kz[0] = pl * lo[2];
        kz[1] = pl * q[2];
        kz[2] = pl * hi[2];
    }
    R s = R(0);
#pragma unroll
    for (int k = K0; k < NPT; ++k) {
        const int idx = ix[koff(D, k, 0) + 1] + jy[koff(D, k, 1) + 1] + (D == 3 ? kz[koff(D, k, 2) + 1] : 0);
        s += L.A[k * L.ncell + c] * L.x[idx];
    }
    return s;
}

// sum_k A_k y_{nb_k} with the level's coefficients (type R) and values y of type TX,
// accumulated in R
template <int D, int NPT, typename R, typename TX>
__device__ __forceinline__ R stencil_apply(const LV<R>& L, const TX* __restrict__ y, int c, const int* q) {
    int lo[3], hi[3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        lo[a] = q[a] > 0 ? q[a] - 1 : (L.per[a] ? L.n[a] - 1 : 0);
        hi[a] = q[a] + 1 < L.n[a] ? q[a] + 1 : (L.per[a] ? 0 : L.n[a] - 1);
    }
    const int ix[3] = {lo[0], q[0], hi[0]};
    const int jy[3] = {L.n[0] * lo[1], L.n[0] * q[1], L.n[0] * hi[1]};
    int kz[3] = {0, 0, 0};
    if (D == 3) {
        const int pl = L.n[0] * L.n[1];
        kz[0] = pl * lo[2];
        kz[1] = pl * q[2];
        kz[2] = pl * hi[2];
    }
    R acc = R(0);
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int idx = ix[koff(D, k, 0) + 1] + jy[koff(D, k, 1) + 1] + (D == 3 ? kz[koff(D, k, 2) + 1] : 0);
        acc += L.A[k * L.ncell + c] * (R)y[idx];
    }
    return acc;
}

// cells of one colour: parity colouring (i + j + k) % 2 when ncol == 2 (n[0] even), one
// bit per axis otherwise (NPT > 2D + 1). The colour-local index space (m, j, k) has a
// half-length first axis.
template <int D, int NPT>
struct Col {
    static constexpr bool parity = NPT == 2 * D + 1;
    template <typename R>
    static __device__ __forceinline__ void dims(const LV<R>& L, int* d) {
        d[0] = L.n[0] / 2;
        d[1] = parity ? L.n[1] : L.n[1] / 2;
        d[2] = D == 3 ? (parity ? L.n[2] : L.n[2] / 2) : 1;
    }
    static __device__ __forceinline__ void cell(int colour, int m, int j, int k, int* q) {
        if (parity) {
            q[0] = 2 * m + ((j + k + colour) & 1);
            q[1] = j;
            q[2] = k;
        } else {
            q[0] = 2 * m + (colour & 1);
            q[1] = 2 * j + ((colour >> 1) & 1);
            q[2] = D == 3 ? 2 * k + ((colour >> 2) & 1) : 0;
        }
    }
};

template <int D, int NPT, typename R>
__device__ __forceinline__ void smooth_at(const LV<R>& L, const R* dinv, const int* q) {
    const int c = q[0] + L.n[0] * (q[1] + L.n[1] * q[2]);
    L.x[c] = (L.b[c] - stencil_sum<D, NPT, 1>(L, c, q)) * dinv[c];
}

// Prolongation x_f += sum over the 2^D parents of w * x_parent: per axis the fine cell's own
// parent (weight own, 3/4 when bilinear) and the parent on the fine cell's side (1 - own,
// with the correction's ghost rules: periodic wrap, or else the boundary parent itself, its
// sign flipped at a Dirichlet face). The per-axis offsets, signs
// and weights are set up once and combined per parent: w = ((1 w_0) w_1) w_2 and the signed
// parent value, accumulated over the parents in order.
template <int D, typename R>
__device__ __forceinline__ R prolonged_at(const LV<R>& F, const LV<R>& Cl, const int* q) {
    const int f = q[0] + F.n[0] * (q[1] + F.n[1] * q[2]);
    R own[3] = {R(0.75), R(0.75), R(0.75)};  // weight of the own parent per axis (bilinear: 3/4)
    if (F.pw)
#pragma unroll
        for (int a = 0; a < D; ++a) own[a] = F.pw[a * F.ncell + f];
    int off[3][2];
    R sg[3][2], wt[3][2];
    int stride = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int pa = q[a] >> 1;
        int nb = pa + ((q[a] & 1) ? 1 : -1);
        R sign = R(1);
        if (nb < 0 || nb >= Cl.n[a]) {
            const int side = nb < 0 ? 0 : 1;
            if (Cl.per[a]) {
                nb = nb < 0 ? nb + Cl.n[a] : nb - Cl.n[a];
            } else {
                nb = side == 0 ? 0 : Cl.n[a] - 1;
                if (Cl.bc[2 * a + side] == CPIC_BC_DIRICHLET) sign = -sign;
            }
        }
        off[a][0] = pa * stride;
        off[a][1] = nb * stride;
        sg[a][0] = R(1);
        sg[a][1] = sign;
        wt[a][0] = own[a];
        wt[a][1] = R(1) - own[a];
        stride *= Cl.n[a];
    }
    R acc = R(0);
#pragma unroll
    for (int o = 0; o < (D == 2 ? 4 : 8); ++o) {
        R w = R(1), sign = R(1);
        int idx = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int bit = (o >> a) & 1;
            w *= wt[a][bit];
            sign *= sg[a][bit];
            idx += off[a][bit];
        }
        acc += w * (sign * Cl.x[idx]);
    }
    return F.x[f] + acc;
}
template <int D, typename R>
__device__ __forceinline__ void prolong_at(const LV<R>& F, const LV<R>& Cl, const int* q) {
    F.x[q[0] + F.n[0] * (q[1] + F.n[1] * q[2])] = prolonged_at<D>(F, Cl, q);
}

// ------------------------------------------------------------------ line relaxation
// Zebra line Gauss-Seidel (robust for anisotropic cells, Sec. II.B.3): every line of cells
// along `axis` is solved exactly (a tridiagonal system, cyclic on a periodic axis) with the
// cells of the neighbouring lines at their current values. Lines are coloured by the parity
// of their transverse coordinates (a periodic transverse axis with an odd count gives its
// last index a third colour), so lines of one colour share no stencil entry and are
// independent. One sweep relaxes the lines along axis 0, then axis 1 (then axis 2).
template <int D, int NPT>
__device__ void line_solve(const LV<float>& L, int axis, int base) {
    const int n = L.n[axis];
    const int stride = axis == 0 ? 1 : (axis == 1 ? L.n[0] : L.n[0] * L.n[1]);
    const int km = 1 + 2 * axis, kp = 2 + 2 * axis;  // in-line -1 / +1 slots
    const bool per = L.per[axis] != 0;
    float* cp = L.lw;            // eliminated upper diagonal (cells of this line only)
    float* z = L.lw + L.ncell;   // second solve of the cyclic case
    const int nc = L.ncell;
    auto coeff = [&](int k, int c) { return L.A[k * nc + c]; };
    // right-hand side of cell c: b - (off-line stencil terms), neighbours as in stencil_sum
    auto rhs = [&](int c) {
        int q[3];
        cell_coords(L, c, q);
        int lo[3], hi[3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            lo[a] = q[a] > 0 ? q[a] - 1 : (L.per[a] ? L.n[a] - 1 : 0);
            hi[a] = q[a] + 1 < L.n[a] ? q[a] + 1 : (L.per[a] ? 0 : L.n[a] - 1);
        }
        const int ix[3] = {lo[0], q[0], hi[0]};
        const int jy[3] = {L.n[0] * lo[1], L.n[0] * q[1], L.n[0] * hi[1]};
        int kz[3] = {0, 0, 0};
        if (D == 3) {
            const int pl = L.n[0] * L.n[1];
            kz[0] = pl * lo[2];
            kz[1] = pl * q[2];
            kz[2] = pl * hi[2];
        }
        float sacc = L.b[c];
#pragma unroll
        for (int k = 1; k < NPT; ++k) {
            if (k == km || k == kp) continue;
            sacc -= coeff(k, c) * L.x[ix[koff(D, k, 0) + 1] + jy[koff(D, k, 1) + 1] + (D == 3 ? kz[koff(D, k, 2) + 1] : 0)];
        }
        return sacc;
    };
    if (n == 1) {
        const int c = base;
        const float d = coeff(0, c) + (per ? coeff(km, c) + coeff(kp, c) : 0.0f);
        L.x[c] = rhs(c) / d;
        return;
    }
    if (n == 2 && per) {  // both in-line neighbours are the other cell
        const int c0 = base, c1 = base + stride;
        const float a00 = coeff(0, c0), a01 = coeff(km, c0) + coeff(kp, c0);
        const float a10 = coeff(km, c1) + coeff(kp, c1), a11 = coeff(0, c1);
        const float r0 = rhs(c0), r1 = rhs(c1);
        const float det = a00 * a11 - a01 * a10;
        L.x[c0] = (r0 * a11 - a01 * r1) / det;
        L.x[c1] = (a00 * r1 - a10 * r0) / det;
        return;
    }
    // cyclic system: corners beta = A[0][n-1] (slot km of cell 0), alpha = A[n-1][0] (slot kp
    // of the last cell); Sherman-Morrison with gamma = -d_0: T' = A - v w^T, v = (gamma, 0, ..,
    // 0, alpha), w = (1, 0, .., 0, beta / gamma); x = y - z (w . y) / (1 + w . z) with T' y = r,
    // T' z = v
    const int cl = base + (n - 1) * stride;
    const float beta = per ? coeff(km, base) : 0.0f, alpha = per ? coeff(kp, cl) : 0.0f;
    const float gamma = -coeff(0, base);
    float prev_cp = 0.0f, prev_y = 0.0f, prev_z = 0.0f;
    for (int i = 0; i < n; ++i) {
        const int c = base + i * stride;
        float d = coeff(0, c);
        const float l = i == 0 ? 0.0f : coeff(km, c);
        const float u = i == n - 1 ? 0.0f : coeff(kp, c);
        if (per && i == 0) d -= gamma;
        if (per && i == n - 1) d -= alpha * beta / gamma;
        const float den = d - l * prev_cp;
        const float ci = u / den;
        const float yi = (rhs(c) - l * prev_y) / den;
        cp[c] = ci;
        L.x[c] = yi;
        prev_cp = ci;
        prev_y = yi;
        if (per) {
            const float v = i == 0 ? gamma : (i == n - 1 ? alpha : 0.0f);
            const float zi = (v - l * prev_z) / den;
            z[c] = zi;
            prev_z = zi;
        }
    }
    for (int i = n - 2; i >= 0; --i) {
        const int c = base + i * stride, cn = c + stride;
        L.x[c] -= cp[c] * L.x[cn];
        if (per) z[c] -= cp[c] * z[cn];
    }
    if (per) {
        const float fact = (L.x[base] + beta * L.x[cl] / gamma) / (1.0f + z[base] + beta * z[cl] / gamma);
        for (int i = 0; i < n; ++i) {
            const int c = base + i * stride;
            L.x[c] -= fact * z[c];
        }
    }
}

// colours per transverse axis (2, or 3 for a periodic axis of odd size) and of an index
__host__ __device__ inline int tcolours(int n, int per) { return per && (n & 1) ? 3 : 2; }
__host__ __device__ inline int tcolour(int x, int n, int per) { return tcolours(n, per) == 3 && x == n - 1 ? 2 : (x & 1); }

// the transverse axes of lines along `axis`, and the number of line colours
template <typename R>
__host__ __device__ inline void line_axes(const LV<R>& L, int D, int axis, int& b, int& c, int& ncol) {
    b = axis == 0 ? 1 : 0;
    c = D == 3 ? (axis == 2 ? 1 : 2) : -1;
    ncol = tcolours(L.n[b], L.per[b]) * (c >= 0 ? tcolours(L.n[c], L.per[c]) : 1);
}

// does line `idx` (transverse index, b fastest) have colour `col`? returns its first cell
template <typename R>
__host__ __device__ inline int line_start(const LV<R>& L, int D, int axis, int idx, int col) {
    int b, c, ncol;
    line_axes(L, D, axis, b, c, ncol);
    const int xb = idx % L.n[b], xc = c >= 0 ? idx / L.n[b] : 0;
    const int cb = tcolour(xb, L.n[b], L.per[b]);
    const int cc = c >= 0 ? tcolour(xc, L.n[c], L.per[c]) : 0;
    if (cb + tcolours(L.n[b], L.per[b]) * cc != col) return -1;
    int q[3] = {0, 0, 0};
    q[b] = xb;
    if (c >= 0) q[c] = xc;
    return q[0] + L.n[0] * (q[1] + L.n[1] * q[2]);
}

template <int D, int NPT>
__global__ void line_kernel(LV<float> L, int axis, int col, int lines) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= lines) return;
    const int start = line_start(L, D, axis, idx, col);
    if (start >= 0) line_solve<D, NPT>(L, axis, start);
}

// ------------------------------------------------------------------ Galerkin coarse operators
// A_C = R A P (BoxMG's variational coarse operator, Sec. II.B.3) with the V-cycle's own
// transfers: R sums the 2^D fine children, P is the prolongation of prolong_at (bilinear or
// operator-induced weights) with its homogeneous ghost rules (an out-of-range coarse source
// is the boundary cell, negated at a Dirichlet face; periodic axes wrap). Every source of
// P e_C' reached from a child of C lies within one coarse cell of C, so the coarse operator
// has the 3^D-point shape (9 in 2D, 27 in 3D). FP64, one thread per coarse cell, entries in
// stencil-slot order.
template <int D>
__global__ void galerkin_kernel(LV<double> F, LV<double> C, double* Ac) {
    constexpr int NS = D == 2 ? 9 : 27, NCH = 1 << D;
    for (int cc = blockIdx.x * blockDim.x + threadIdx.x; cc < C.ncell; cc += gridDim.x * blockDim.x) {
        int Q[3];
        cell_coords(C, cc, Q);
        double acc[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) acc[k] = 0.0;
        for (int ch = 0; ch < NCH; ++ch) {
            int fq[3] = {2 * Q[0] + (ch & 1), 2 * Q[1] + ((ch >> 1) & 1), D == 3 ? 2 * Q[2] + ((ch >> 2) & 1) : 0};
            const int f = fq[0] + F.n[0] * (fq[1] + F.n[1] * fq[2]);
            for (int k = 0; k < NS; ++k) {
                const double a = F.A[k * F.ncell + f];
                if (a == 0.0) continue;
                int g[3], p[3], sdir[3];
                for (int ax = 0; ax < D; ++ax) {
                    g[ax] = fq[ax] + koff(D, k, ax);  // unwrapped
                    p[ax] = g[ax] >> 1;               // floor(g / 2), also for g = -1
                    sdir[ax] = (g[ax] & 1) ? 1 : -1;
                }
                double own[3] = {0.75, 0.75, 0.75};  // the prolongation row of fine cell g
                if (F.pw) {
                    int gw[3] = {0, 0, 0};
                    for (int ax = 0; ax < D; ++ax) gw[ax] = (g[ax] % F.n[ax] + F.n[ax]) % F.n[ax];
                    const int gi = gw[0] + F.n[0] * (gw[1] + F.n[1] * gw[2]);
                    for (int ax = 0; ax < D; ++ax) own[ax] = F.pw[ax * F.ncell + gi];
                }
                for (int o = 0; o < NCH; ++o) {
                    double w = 1.0;
                    int off[3] = {0, 0, 0};
                    for (int ax = 0; ax < D; ++ax) {
                        const int src = p[ax] + (((o >> ax) & 1) ? sdir[ax] : 0);
                        w *= ((o >> ax) & 1) ? 1.0 - own[ax] : own[ax];
                        off[ax] = src - Q[ax];
                        if (!C.per[ax] && (src < 0 || src >= C.n[ax])) {
                            off[ax] = 0;  // the ghost maps onto this boundary cell
                            const int side = src < 0 ? 0 : 1;
                            if (C.bc[2 * ax + side] == CPIC_BC_DIRICHLET) w = -w;
                        }
                    }
                    int slot = 0;
                    for (int k2 = 0; k2 < NS; ++k2)
                        if (koff(D, k2, 0) == off[0] && koff(D, k2, 1) == off[1] && (D == 2 || koff(D, k2, 2) == off[2]))
                            slot = k2;
                    acc[slot] += w * a;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) Ac[k * C.ncell + cc] = acc[k];
    }
}

// ------------------------------------------------------------------ operator-induced prolongation
// BoxMG takes its interpolation weights from the operator (Sec. II.B.3). Reading for this
// cell-centred 2:1 hierarchy: along each axis a fine cell is interpolated from its own
// coarse parent C and the parent's neighbour N on the fine cell's side, with the weights of
// the flux-continuous 1D solution between the two coarse centres: resistances from the fine
// operator's couplings across faces, collapsed over the transverse directions (the sum of
// the entries linking the two layers of cells, as BoxMG collapses its stencils),
//   R1 = 1 / (2 g(f_other -> f))   (C's centre is the face between its two children),
//   R2 = 1 / g(f -> n) + 1 / (2 g(n -> n_other))   (n, n_other: N's children, n next to f),
// own-parent weight R2 / (R1 + R2); uniform couplings give bilinear's 3/4. The weights of a
// cell are the product of its axes' weights. Cells whose neighbour parent is outside a
// non-periodic boundary, or whose couplings are not all positive, keep 3/4 (the ghost rule
// of prolong_at then applies).
template <int D>
__global__ void interp_weights_kernel(LV<double> F, double* pw, float* pw32) {
    constexpr int NS = D == 2 ? 9 : 27;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < F.ncell; f += gridDim.x * blockDim.x) {
        int q[3];
        cell_coords(F, f, q);
        for (int ax = 0; ax < D; ++ax) {
            double w = 0.75;
            const int s = (q[ax] & 1) ? 1 : -1;  // side of the neighbour parent
            const int nc = F.n[ax] / 2;
            const int pn = (q[ax] >> 1) + s;      // neighbour parent (coarse index)
            const bool inside = F.per[ax] || (pn >= 0 && pn < nc);
            if (inside) {
                // fine cells along the axis: f_other, f, n, n_other at offsets -s, 0, s, 2s
                auto cell = [&](int d) {
                    int c[3] = {q[0], q[1], q[2]};
                    c[ax] = ((c[ax] + d) % F.n[ax] + F.n[ax]) % F.n[ax];
                    return c[0] + F.n[0] * (c[1] + F.n[1] * c[2]);
                };
                // collapsed coupling from cell c towards dir (+-1) along ax
                auto coupling = [&](int c, int dir) {
                    double gsum = 0.0;
                    for (int k = 1; k < NS; ++k)
                        if (koff(D, k, ax) == dir) gsum -= F.A[k * F.ncell + c];
                    return gsum;
                };
                const double g1 = coupling(cell(-s), s);  // f_other -> f
                const double g2 = coupling(f, s);          // f -> n
                const double g3 = coupling(cell(s), s);    // n -> n_other
                if (g1 > 0.0 && g2 > 0.0 && g3 > 0.0) {
                    const double R1 = 0.5 / g1, R2 = 1.0 / g2 + 0.5 / g3;
                    w = R2 / (R1 + R2);
                }
            }
            pw[ax * F.ncell + f] = w;
            pw32[ax * F.ncell + f] = (float)w;
        }
    }
}

// ------------------------------------------------------------------ FP32 cycle kernels
// 3D launch geometry: x covers the first (index) dimension, y the second, z the third.
template <int D, int NPT>
__global__ void smooth_kernel(LV<float> L, const float* __restrict__ dinv, int colour) {
    int d[3];
    Col<D, NPT>::dims(L, d);
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    int k = blockIdx.z;
    if (m >= d[0] || j >= d[1] || k >= d[2]) return;
    int q[3];
    Col<D, NPT>::cell(colour, m, j, k, q);
    smooth_at<D, NPT>(L, dinv, q);
}

// The first two colour sweeps of a 3D two-colour level, from x = 0, in one pass: the first colour
// is b / diag, so the second reads its neighbours' b and 1 / diag in place of their x (the same
// products in the same order). A thread takes the two cells of a pair along axis 0 (n[0] is even
// on a level that coarsens). Bound by L2: a colour's sweep touches every sector of the operator
// and uses half of it, so two sweeps in one pass read it once. 128^3 and the 64^3 level below:
// 16.1 us a V-cycle, 21 us as a memset and two sweeps each.
__global__ void __launch_bounds__(256) first_sweeps3_kernel(const __grid_constant__ LV<float> L) {
    const int m = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z;
    const int n0 = L.n[0], n1 = L.n[1], pl = n0 * n1, nc = L.ncell;
    if (2 * m >= n0 || j >= n1) return;
    const int c = 2 * m + n0 * (j + n1 * k), odd = (j + k) & 1;  // the first colour is cell c + odd
    const float2 b = *reinterpret_cast<const float2*>(L.b + c), d = __ldg(reinterpret_cast<const float2*>(L.dinv + c));
    const float x0 = (odd ? b.y : b.x) * (odd ? d.y : d.x);
    const int e = c + 1 - odd, i = 2 * m + 1 - odd;  // the second colour's cell
    auto first = [&](int q) { return L.b[q] * __ldg(L.dinv + q); };
    // beyond a closed face the stencil entry is zero: any neighbour will do
    float s = 0.0f;
    s += __ldg(L.A + nc + e) * (odd ? first(e + (i > 0 ? -1 : n0 - 1)) : x0);
    s += __ldg(L.A + 2 * nc + e) * (odd ? x0 : first(e + (i < n0 - 1 ? 1 : 1 - n0)));
    s += __ldg(L.A + 3 * nc + e) * first(e + (j > 0 ? -1 : n1 - 1) * n0);
    s += __ldg(L.A + 4 * nc + e) * first(e + (j < n1 - 1 ? 1 : 1 - n1) * n0);
    s += __ldg(L.A + 5 * nc + e) * first(e + (k > 0 ? -1 : L.n[2] - 1) * pl);
    s += __ldg(L.A + 6 * nc + e) * first(e + (k < L.n[2] - 1 ? 1 : 1 - L.n[2]) * pl);
    const float x1 = ((odd ? b.x : b.y) - s) * (odd ? d.x : d.y);
    *reinterpret_cast<float2*>(L.x + c) = odd ? make_float2(x1, x0) : make_float2(x0, x1);
}

template <int D, int NPT>
__global__ void __launch_bounds__(256) restrict_kernel(LV<float> F, LV<float> Cl) {
    // one thread per fine cell (block RB_X x RB_Y x RB_Z fine cells): its residual goes to
    // shared memory, then one thread per coarse cell of the block sums its 2^D children in
    // the children's order: ch = 0 .. 2^D - 1, axis 0 fastest
    constexpr int BX = 32, BY = D == 3 ? 4 : 8, BZ = D == 3 ? 2 : 1;
    __shared__ float rs[BX * BY * BZ];
    const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z;
    const int t = tx + BX * (ty + BY * tz);
    int q[3] = {(int)blockIdx.x * BX + tx, (int)blockIdx.y * BY + ty, D == 3 ? (int)blockIdx.z * BZ + tz : 0};
    float r = 0.0f;
    if (q[0] < F.n[0] && q[1] < F.n[1] && q[2] < F.n[2]) {
        const int f = q[0] + F.n[0] * (q[1] + F.n[1] * q[2]);
        r = F.b[f] - stencil_sum<D, NPT, 0>(F, f, q);
    }
    rs[t] = r;
    __syncthreads();
    constexpr int CX = BX / 2, CY = BY / 2, CZ = D == 3 ? BZ / 2 : 1;
    if (t < CX * CY * CZ) {
        const int ci = t % CX, cj = (t / CX) % CY, ck = t / (CX * CY);
        const int qc[3] = {(int)blockIdx.x * CX + ci, (int)blockIdx.y * CY + cj, D == 3 ? (int)blockIdx.z * CZ + ck : 0};
        if (qc[0] < Cl.n[0] && qc[1] < Cl.n[1] && qc[2] < Cl.n[2]) {
            float acc = 0.0f;
#pragma unroll
            for (int ch = 0; ch < (D == 2 ? 4 : 8); ++ch)
                acc += rs[(2 * ci + (ch & 1)) + BX * ((2 * cj + ((ch >> 1) & 1)) + BY * (D == 3 ? 2 * ck + ((ch >> 2) & 1) : 0))];
            const int C = qc[0] + Cl.n[0] * (qc[1] + Cl.n[1] * qc[2]);
            Cl.b[C] = acc;
            Cl.x[C] = 0.0f;
        }
    }
}

template <int D>
__global__ void prolong_kernel(LV<float> F, LV<float> Cl) {
    int q[3] = {(int)(blockIdx.x * blockDim.x + threadIdx.x), (int)(blockIdx.y * blockDim.y + threadIdx.y), (int)blockIdx.z};
    if (q[0] >= F.n[0] || q[1] >= F.n[1] || q[2] >= F.n[2]) return;
    prolong_at<D>(F, Cl, q);
}

// ---- one level's half of a V-cycle in one launch (2D, two colours)
//
// A block relaxes its tile of TL_X x TL_Y cells with TL_H cells of its surroundings: the four colour
// sweeps of a V(2,2) half need no other block's values then, each leaving one ring of the
// surroundings behind. So a level costs one launch on the way down (four sweeps from x = 0,
// residual, restriction) and one on the way up (prolongation, four sweeps) in place of five
// each, and its stencil is read once a launch and not once a sweep. A thread holds two pairs of
// neighbouring cells (one cell of each colour) with their couplings in registers; x is in shared
// memory with the colours of a row apart, so that a sweep's reads do not conflict. The tile: a
// taller or wider one relaxes less twice (1.9 cells a cell here), a smaller one fills more of
// the chip on the small levels, where the time is latency. On a 512 x 1024 V-cycle (levels
// down to 64 x 128) a launch takes 3.9 us down and 4.7 us up on average, 82 us of sweeps,
// transfers and memsets before.
constexpr int TL_X = 32, TL_Y = 16, TL_H = 4, TL_THREADS = 256;
constexpr int TL_W = TL_X + 2 * TL_H, TL_R = TL_Y + 2 * TL_H;  // cells of the extended tile
constexpr int TL_HALF = TL_W / 2, TL_PAIRS = TL_HALF * TL_R;
constexpr int TL_ITEMS = (TL_PAIRS + TL_THREADS - 1) / TL_THREADS;

struct TilePair {
    int at;            // shared offset of index m of the row's first colour (one row and word of margin)
    int i, j;          // global cell of the pair's first cell (wrapped); i < 0: outside the domain
    int ring;          // rings of the surroundings the pair lies in (0: own tile)
    int odd;           // 1: its even cell is of the second colour
    float a[2][4];     // couplings W, E, S, N per colour (the stencil's slots 1 .. 4)
    float b[2], d[2];
};

// pair p of the extended tile of block (bx, by): its cells, couplings, right-hand side
__device__ __forceinline__ void tile_pair(const LV<float>& L, int p, TilePair& t) {
    const int r = p / TL_HALF, m = p - r * TL_HALF;
    t.at = (r + 1) * TL_W + m + 1;
    int i = (int)blockIdx.x * TL_X - TL_H + 2 * m, j = (int)blockIdx.y * TL_Y - TL_H + r;
    const int x = 2 * m, rx = max(max(TL_H - x - 1, x - TL_H - TL_X + 1), 0), ry = max(max(TL_H - r, r - TL_H - TL_Y + 1), 0);
    t.ring = max(rx, ry);  // of the pair's cell nearer to the tile
    t.odd = j & 1;
    bool in = p < TL_PAIRS;
    if (L.per[0]) {
        while (i < 0) i += L.n[0];
        while (i >= L.n[0]) i -= L.n[0];
    } else {
        in = in && i >= 0 && i < L.n[0];
    }
    if (L.per[1]) {
        while (j < 0) j += L.n[1];
        while (j >= L.n[1]) j -= L.n[1];
    } else {
        in = in && j >= 0 && j < L.n[1];
    }
    t.i = in ? i : -1;
    t.j = j;
    const int c = in ? i + L.n[0] * j : 0, nc = L.ncell;
    float2 z = make_float2(0.f, 0.f);
    float2 w[4], bb, dd;
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = in ? __ldg(reinterpret_cast<const float2*>(L.A + (k + 1) * nc + c)) : z;
    bb = in ? *reinterpret_cast<const float2*>(L.b + c) : z;
    dd = in ? __ldg(reinterpret_cast<const float2*>(L.dinv + c)) : z;
    const bool o = t.odd != 0;  // colour 0 is the odd cell (2 m + 1) then
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        t.a[0][k] = o ? w[k].y : w[k].x;
        t.a[1][k] = o ? w[k].x : w[k].y;
    }
    t.b[0] = o ? bb.y : bb.x;
    t.b[1] = o ? bb.x : bb.y;
    t.d[0] = o ? dd.y : dd.x;
    t.d[1] = o ? dd.x : dd.y;
}

// s + couplings times neighbours of the pair's cell of colour C, in the order of stencil_sum
template <int C>
__device__ __forceinline__ float tile_sum(const TilePair& t, const float* x, float s) {
    const float* o = x + t.at + (1 - C) * TL_HALF;
    const bool even = (C == 0) != (t.odd != 0);  // the cell is 2 m: its pair neighbour is to the east
    s += t.a[C][0] * o[even ? -1 : 0];
    s += t.a[C][1] * o[even ? 0 : 1];
    s += t.a[C][2] * o[-TL_W];
    s += t.a[C][3] * o[TL_W];
    return s;
}
template <int C>
__device__ __forceinline__ float tile_relaxed(const TilePair& t, const float* x) {
    return (t.b[C] - tile_sum<C>(t, x, 0.0f)) * t.d[C];
}

// the ring of the pair's cell of colour C (a pair astride a column of rings: its outer cell is one
// further out)
template <int C>
__device__ __forceinline__ int ring_of(const TilePair& t, int p) {
    const int r = p / TL_HALF, m = p - r * TL_HALF;
    const int x = 2 * m + (((C == 0) != (t.odd != 0)) ? 0 : 1);
    return max(max(TL_H - x, x - TL_H - TL_X + 1), max(max(TL_H - r, r - TL_H - TL_Y + 1), 0));
}

// Down: x = 0, sweeps of colours 0, 1, 0, 1, then Cl.b = sums of the residuals, in
// restrict_kernel's order. x keeps the first colour only: the way up prolongs onto it and relaxes the
// second from it.
__global__ void __launch_bounds__(TL_THREADS) level_down2_kernel(const __grid_constant__ LV<float> L, float* bc, int cn0) {
    __shared__ float x[(TL_R + 2) * TL_W + 2];
    __shared__ float rs[TL_Y][TL_X];
    const int tid = threadIdx.x;
    for (int e = tid; e < (TL_R + 2) * TL_W + 2; e += TL_THREADS) x[e] = 0.0f;
    TilePair t[TL_ITEMS];
#pragma unroll
    for (int u = 0; u < TL_ITEMS; ++u) tile_pair(L, tid + u * TL_THREADS, t[u]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int u = 0; u < TL_ITEMS; ++u) {
            const int p = tid + u * TL_THREADS;
            if (p >= TL_PAIRS) continue;
            if (k & 1) {
                if (ring_of<1>(t[u], p) <= TL_H - k) x[t[u].at + TL_HALF] = tile_relaxed<1>(t[u], x);
            } else if (ring_of<0>(t[u], p) <= TL_H - k) {
                x[t[u].at] = k ? tile_relaxed<0>(t[u], x) : t[u].b[0] * t[u].d[0];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < TL_ITEMS; ++u) {
        const int p = tid + u * TL_THREADS;
        if (p >= TL_PAIRS || t[u].ring) continue;
        const int r = p / TL_HALF - TL_H, m = p % TL_HALF - TL_H / 2;
        const int gi = (int)blockIdx.x * TL_X + 2 * m, gj = (int)blockIdx.y * TL_Y + r;
        if (gi >= L.n[0] || gj >= L.n[1]) continue;
        const float2 dg = __ldg(reinterpret_cast<const float2*>(L.A + gi + L.n[0] * gj));
        const float x0 = x[t[u].at], x1 = x[t[u].at + TL_HALF];
        const int o = t[u].odd;
        rs[r][2 * m + o] = t[u].b[0] - tile_sum<0>(t[u], x, __fmul_rn(o ? dg.y : dg.x, x0));
        rs[r][2 * m + 1 - o] = t[u].b[1] - tile_sum<1>(t[u], x, __fmul_rn(o ? dg.x : dg.y, x1));
        L.x[gi + o + L.n[0] * gj] = x0;
    }
    __syncthreads();
    if (tid < TL_X / 2 * (TL_Y / 2)) {
        const int ic = tid % (TL_X / 2), jc = tid / (TL_X / 2);
        const int I = (int)blockIdx.x * (TL_X / 2) + ic, J = (int)blockIdx.y * (TL_Y / 2) + jc;
        if (2 * I < L.n[0] && 2 * J < L.n[1])
            bc[I + cn0 * J] = ((rs[2 * jc][2 * ic] + rs[2 * jc][2 * ic + 1]) + rs[2 * jc + 1][2 * ic]) + rs[2 * jc + 1][2 * ic + 1];
    }
}

// Up: prolongation onto the first colour, sweeps of colours 1, 0, 1, 0, result into xo (other
// blocks read this level's x meanwhile)
__global__ void __launch_bounds__(TL_THREADS) level_up2_kernel(const __grid_constant__ LV<float> L, const __grid_constant__ LV<float> Cl,
                                                               float* xo) {
    __shared__ float x[(TL_R + 2) * TL_W + 2];
    const int tid = threadIdx.x;
    for (int e = tid; e < (TL_R + 2) * TL_W + 2; e += TL_THREADS) x[e] = 0.0f;
    TilePair t[TL_ITEMS];
    float v[TL_ITEMS];
#pragma unroll
    for (int u = 0; u < TL_ITEMS; ++u) {
        tile_pair(L, tid + u * TL_THREADS, t[u]);
        v[u] = 0.0f;
        if (t[u].i >= 0) {
            const int q[3] = {t[u].i + t[u].odd, t[u].j, 0};
            v[u] = prolonged_at<2>(L, Cl, q);
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < TL_ITEMS; ++u)
        if (tid + u * TL_THREADS < TL_PAIRS) x[t[u].at] = v[u];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int u = 0; u < TL_ITEMS; ++u) {
            const int p = tid + u * TL_THREADS;
            if (p >= TL_PAIRS) continue;
            if (k & 1) {
                if (ring_of<0>(t[u], p) < TL_H - k) x[t[u].at] = tile_relaxed<0>(t[u], x);
            } else if (ring_of<1>(t[u], p) < TL_H - k) {
                x[t[u].at + TL_HALF] = tile_relaxed<1>(t[u], x);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < TL_ITEMS; ++u) {
        const int p = tid + u * TL_THREADS;
        if (p >= TL_PAIRS || t[u].ring) continue;
        const int r = p / TL_HALF - TL_H, m = p % TL_HALF - TL_H / 2;
        const int gi = (int)blockIdx.x * TL_X + 2 * m, gj = (int)blockIdx.y * TL_Y + r;
        if (gi >= L.n[0] || gj >= L.n[1]) continue;
        const float c0 = x[t[u].at], c1 = x[t[u].at + TL_HALF];
        *reinterpret_cast<float2*>(xo + gi + L.n[0] * gj) = t[u].odd ? make_float2(c1, c0) : make_float2(c0, c1);
    }
}

// ---- the lower part of the V-cycle (levels first_cta .. nl-1) inside one CTA

// sizes of a level in the one-CTA part, with multipliers for its index divisions
struct CtaLevel {
    int n0, n1, n2, half, ncell;
    unsigned mh, m1;  // idx / half, idx / n1 as __umulhi (0: the divisor is 1)
    float *A, *dinv, *x, *b;
};

__device__ __forceinline__ unsigned div_magic(int d) { return d > 1 ? 0xffffffffu / (unsigned)d + 1u : 0u; }
__device__ __forceinline__ int div_by(int idx, unsigned magic) { return magic ? (int)__umulhi((unsigned)idx, magic) : idx; }

// steps from a cell to its neighbours along each axis. They wrap on every axis: where an axis
// is not periodic the stencil entry of a neighbour beyond the face is zero.
template <int D>
struct Steps {
    int lo[3], hi[3];
    __device__ __forceinline__ Steps(const CtaLevel& L, int i, int j, int k) {
        lo[0] = i > 0 ? -1 : L.n0 - 1;
        hi[0] = i < L.n0 - 1 ? 1 : 1 - L.n0;
        lo[1] = (j > 0 ? -1 : L.n1 - 1) * L.n0;
        hi[1] = (j < L.n1 - 1 ? 1 : 1 - L.n1) * L.n0;
        if (D == 3) {
            const int pl = L.n0 * L.n1;
            lo[2] = (k > 0 ? -1 : L.n2 - 1) * pl;
            hi[2] = (k < L.n2 - 1 ? 1 : 1 - L.n2) * pl;
        }
    }
    __device__ __forceinline__ int operator()(int slot) const {  // constant arguments: folds away
        int o = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) o += koff(D, slot, a) < 0 ? lo[a] : (koff(D, slot, a) > 0 ? hi[a] : 0);
        return o;
    }
};

// sum of the stencil's entries from K0 on times their cells, in the order of stencil_sum (the
// Krylov iteration amplifies a rounding to the size of its stopping error, so every form of
// the V-cycle keeps to one order of operations)
template <int D, int NPT, int K0>
__device__ __forceinline__ float cta_sum(const CtaLevel& L, int c, const Steps<D>& st) {
    float acc = 0.0f;
#pragma unroll
    for (int k = K0; k < NPT; ++k) acc += L.A[k * L.ncell + c] * L.x[c + st(k)];
    return acc;
}

// One colour of a level. The cells of a colour are (m, j, k) with a half-length first axis (and
// half-length other axes when the stencil has 2^D colours); first: x = 0 everywhere else.
template <int D, int NPT>
__device__ __forceinline__ void cta_sweep(const CtaLevel& L, int colour, bool first) {
    constexpr bool parity = Col<D, NPT>::parity;
    const int d1 = parity ? L.n1 : L.n1 / 2, d2 = D == 3 ? (parity ? L.n2 : L.n2 / 2) : 1;
    const unsigned m1 = parity ? L.m1 : div_magic(d1);
    const int count = L.half * d1 * d2;
    for (int idx = threadIdx.x; idx < count; idx += blockDim.x) {
        const int row = div_by(idx, L.mh), m = idx - row * L.half;
        const int k = D == 3 ? div_by(row, m1) : 0, j = row - k * d1;
        int q[3];
        Col<D, NPT>::cell(colour, m, j, k, q);
        const int c = q[0] + L.n0 * (q[1] + L.n1 * q[2]);
        const float s = first ? 0.0f : cta_sum<D, NPT, 1>(L, c, Steps<D>(L, q[0], q[1], q[2]));
        L.x[c] = (L.b[c] - s) * L.dinv[c];
    }
    __syncthreads();
}

// Cl.b = sum of the children's residuals, in restrict_kernel's order
template <int D, int NPT>
__device__ __forceinline__ void cta_restrict(const CtaLevel& F, const CtaLevel& Cl) {
    for (int C = threadIdx.x; C < Cl.ncell; C += blockDim.x) {
        const int row = div_by(C, F.mh), ic = C - row * Cl.n0;  // Cl.n0 = F.half
        const int kc = D == 3 ? row / Cl.n1 : 0, jc = row - kc * Cl.n1;
        float acc = 0.0f;
#pragma unroll
        for (int ch = 0; ch < (D == 2 ? 4 : 8); ++ch) {
            const int i = 2 * ic + (ch & 1), j = 2 * jc + ((ch >> 1) & 1), k = D == 3 ? 2 * kc + ((ch >> 2) & 1) : 0;
            const int c = i + F.n0 * (j + F.n1 * k);
            acc += F.b[c] - cta_sum<D, NPT, 0>(F, c, Steps<D>(F, i, j, k));
        }
        Cl.b[C] = acc;
        Cl.x[C] = 0.0f;
    }
    __syncthreads();
}

// mbarrier with one arrival, and bulk copies from global memory that complete on it
struct BulkLoad {
    unsigned bar;
    unsigned bytes;
    __device__ __forceinline__ void init(unsigned long long* b) {
        bar = (unsigned)__cvta_generic_to_shared(b);
        bytes = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __device__ __forceinline__ void copy(float* dst, const float* src, unsigned n) {
        bytes += n;
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         (unsigned)__cvta_generic_to_shared(dst)),
                     "l"(src), "r"(n), "r"(bar)
                     : "memory");
    }
    __device__ __forceinline__ void arrive() const {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    }
};
// Waits for the copies, a microsecond or so: every thread of the block calls it, and all get the same
// answer. False after BULK_WAIT cycles (about a second): the data is not there and may still be on
// its way. The kernel then sets MG_WAIT_RAN_OUT, which ends the solve and reaches the host
// (CPIC_ERR_TIMEOUT), and waits once more before it leaves, as the copies write its memory.
constexpr long long BULK_WAIT = 1ll << 31;
__device__ __forceinline__ bool bulk_wait(unsigned long long* b) {
    const unsigned bar = (unsigned)__cvta_generic_to_shared(b);
    const long long start = clock64();
    unsigned done = 0;
    do {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar)
            : "memory");
    } while (!done && clock64() - start < BULK_WAIT);
    return !__syncthreads_or(!done);
}

// Lays the one-CTA levels out in shared memory from word off on (per smoothed level A [NPT], dinv,
// x, b, a multiple of four words each since its axes are even; of the dense level x and b) and
// starts the copies of their stencils and inverse diagonals. One thread.
template <int NPT>
__device__ void cta_levels(const LVSet& S, float* sm, int off, LV<float>* V, CtaLevel* T, BulkLoad& load) {
    for (int l = S.first_cta; l < S.nl; ++l) {
        const LV<float>& G = S.l[l];
        const int nc = (G.ncell + 3) & ~3;
        V[l] = G;
        CtaLevel& L = T[l];
        L.n0 = G.n[0], L.n1 = G.n[1], L.n2 = G.n[2], L.half = G.n[0] / 2, L.ncell = G.ncell;
        L.mh = div_magic(L.half);
        L.m1 = div_magic(L.n1);
        if (l < S.nl - 1) {
            L.A = sm + off;
            L.dinv = L.A + NPT * nc;
            L.x = L.dinv + nc;
            off += (NPT + 2) * nc;
            load.copy(L.A, G.A, NPT * nc * 4);
            load.copy(L.dinv, G.dinv, nc * 4);
        } else {
            L.A = L.dinv = nullptr;
            L.x = sm + off;
            off += nc;
        }
        L.b = sm + off;
        off += nc;
        V[l].A = L.A;
        V[l].x = L.x;
        V[l].b = L.b;
    }
}

// The V-cycle over the one-CTA levels, x = 0 before it, once their copies are in: every thread
// of the block. dense: the dense inverse in shared memory, or null.
template <int D, int NPT>
__device__ __forceinline__ void cta_cycle(const LVSet& S, const LV<float>* V, const CtaLevel* T, const float* dense, int nu1,
                                          int nu2) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int m = S.dense_m, mm = m + (S.singular ? 1 : 0);
    // alternating zebra line relaxation: lines along each axis in turn, each colour in turn
    // (reverse order after the coarse-grid correction)
    auto line_sweep = [&](int l, bool reverse) {
        const LV<float>& L = V[l];
        for (int st = 0; st < D; ++st) {
            const int axis = reverse ? D - 1 - st : st;
            int b, c, ncol;
            line_axes(L, D, axis, b, c, ncol);
            const int lines = L.ncell / L.n[axis];
            for (int cc = 0; cc < ncol; ++cc) {
                const int col = reverse ? ncol - 1 - cc : cc;
                for (int idx = tid; idx < lines; idx += nt) {
                    const int start = line_start(L, D, axis, idx, col);
                    if (start >= 0) line_solve<D, NPT>(L, axis, start);
                }
                __syncthreads();
            }
        }
    };
    constexpr int NCOL = Col<D, NPT>::parity ? 2 : 1 << D;
    for (int l = S.first_cta; l < S.nl - 1; ++l) {
        const CtaLevel L = T[l];
        for (int it = 0; it < nu1; ++it) {
            if (S.line) line_sweep(l, false);
            else
                for (int col = 0; col < NCOL; ++col) cta_sweep<D, NPT>(L, col, it == 0 && col == 0);
        }
        cta_restrict<D, NPT>(L, T[l + 1]);
    }
    {
        // dense solve, one unknown a thread (the inverse is stored transposed, so that
        // neighbouring threads read neighbours)
        const float* bs = T[S.nl - 1].b;
        for (int i = tid; i < m; i += nt) {
            float acc = 0.0f;
            if (dense) {
#pragma unroll 8
                for (int k = 0; k < m; ++k) acc += dense[k * mm + i] * bs[k];
            } else {
#pragma unroll 16
                for (int k = 0; k < m; ++k) acc += __ldg(S.dense_inv + k * mm + i) * bs[k];
            }
            T[S.nl - 1].x[i] = acc;
        }
        __syncthreads();
    }
    for (int l = S.nl - 2; l >= S.first_cta; --l) {
        const LV<float>& L = V[l];
        const CtaLevel F = T[l];
        for (int idx = tid; idx < F.ncell; idx += nt) {
            const int row = div_by(idx >> 1, F.mh), i = idx - row * F.n0;
            const int k = D == 3 ? div_by(row, F.m1) : 0, j = row - k * F.n1;
            // with two colours the next sweep overwrites the second
            if (!S.line && Col<D, NPT>::parity && ((i + j + k) & 1)) continue;
            const int q[3] = {i, j, k};
            prolong_at<D>(L, V[l + 1], q);
        }
        __syncthreads();
        for (int it = 0; it < nu2; ++it) {
            if (S.line) line_sweep(l, true);
            else
                for (int col = NCOL - 1; col >= 0; --col) cta_sweep<D, NPT>(F, col, false);
        }
    }
}

// All of these levels' stencils, inverse diagonals and right-hand sides come in by bulk copies
// (one a level and array, so the load is one latency and not a chain of them); with the dense
// inverse beside them when it fits; the first sweep from x = 0 reads no neighbours, and of two
// colours the second is not prolonged onto (the next sweep overwrites it). The CTA part of a
// 512 x 1024 V-cycle (levels of 32 x 64 cells and below) takes 16 us (33 with per-cell index
// divisions, element-wise staging and the dense inverse read a row per thread), that of
// a 24 x 20 x 16 one (12 x 10 x 8 and below) 10.5 us (18.8).
template <int D, int NPT>
__global__ void __launch_bounds__(512, 1) coarse_cycle_kernel(const __grid_constant__ LVSet S, int nu1, int nu2, int dense_smem) {
    extern __shared__ __align__(16) float sm[];
    __shared__ LV<float> V[MAX_LEVELS];
    __shared__ CtaLevel T[MAX_LEVELS];
    __shared__ __align__(8) unsigned long long bar;
    const int tid = threadIdx.x, nt = blockDim.x;
    const bool smoothed = S.first_cta < S.nl - 1;
    const LV<float>& G = S.l[S.first_cta];
    if (tid == 0) {
        BulkLoad load;
        load.init(&bar);
        cta_levels<NPT>(S, sm, 0, V, T, load);
        if (smoothed) load.copy(T[S.first_cta].b, G.b, G.ncell * 4);
        const int mm = S.dense_m + (S.singular ? 1 : 0);
        if (dense_smem) load.copy(sm + dense_smem, S.dense_inv, (unsigned)((mm * mm * 4 + 15) & ~15));
        load.arrive();
    }
    __syncthreads();
    for (int c = tid; c < G.ncell; c += nt) {
        T[S.first_cta].x[c] = 0.0f;
        if (!smoothed) T[S.first_cta].b[c] = G.b[c];
    }
    if (!bulk_wait(&bar)) {
        if (tid == 0) *S.status = MG_WAIT_RAN_OUT;
        (void)bulk_wait(&bar);
        return;
    }
    cta_cycle<D, NPT>(S, V, T, dense_smem ? sm + dense_smem : nullptr, nu1, nu2);
    for (int c = tid; c < G.ncell; c += nt) G.x[c] = T[S.first_cta].x[c];
}

// ---- the lower part of a 3D two-colour V-cycle on a thread-block cluster
//
// Levels too large for one CTA but far too small for the chip (a colour sweep of 32^3 cells has
// 4 us of launch and ramp for 0.5 us of work) are split by planes over the cluster's CTAs, in
// shared memory: a sweep hands the new values of its first and last plane to the neighbours'
// halo planes and ends with a cluster barrier (0.4 us). The one-CTA levels below are solved by
// every CTA redundantly. Same operations in the same order as the kernels per level. Measured:
// 40 us for the levels from 32^3 down of a 128^3 V-cycle on 8 CTAs (55 us as 23 launches), 20
// us for a whole 24 x 20 x 16 V-cycle (30 us). 64^3 stays on its launches: 15 planes of 4096
// cells a CTA do not fit, and its sweeps fill the chip.
constexpr int SL_MAX = 2;           // split levels
constexpr int SL_CELLS = 40960;     // a level joins from this many cells down
constexpr size_t SL_SMEM_MAX = 216 * 1024;

struct SlabPlan {
    int cs;          // CTAs
    int first, ns;   // split levels first .. first + ns - 1; the one-CTA levels follow
    int oa[SL_MAX], od[SL_MAX], ob[SL_MAX], ox[SL_MAX];  // shared offsets (words)
    int ocoarse;     // of the one-CTA levels
    int odense;      // of the dense inverse (0: global)
};

// first plane of CTA `rank` on the level below the split ones (whose restriction must not cross
// CTAs); each finer level doubles it
__host__ __device__ inline int slab_start(int rank, int cs, int planes) { return rank * planes / cs; }

struct Slab {
    int n0, n1, n2, half, plane, z0, R;
    unsigned mh, m1;
    const float *A, *d;
    float *b, *x;        // x: one halo plane below and above
    float *lower, *upper;  // the neighbours' halo planes that mirror this CTA's first and last
};

// one colour; first: x = 0 before it
__device__ __forceinline__ void slab_sweep(const Slab& L, int colour, bool first) {
    const int count = L.R * L.n1 * L.half, nc = L.R * L.plane;
    for (int idx = threadIdx.x; idx < count; idx += 512) {
        const int row = div_by(idx, L.mh), m = idx - row * L.half, kk = div_by(row, L.m1), j = row - kk * L.n1;
        const int i = 2 * m + ((j + L.z0 + kk + colour) & 1);
        const int in = j * L.n0 + i, c = kk * L.plane + in;
        float* x = L.x + c + L.plane;
        float s = 0.0f;
        if (!first) {
            s += L.A[nc + c] * x[i > 0 ? -1 : L.n0 - 1];
            s += L.A[2 * nc + c] * x[i < L.n0 - 1 ? 1 : 1 - L.n0];
            s += L.A[3 * nc + c] * x[(j > 0 ? -1 : L.n1 - 1) * L.n0];
            s += L.A[4 * nc + c] * x[(j < L.n1 - 1 ? 1 : 1 - L.n1) * L.n0];
            s += L.A[5 * nc + c] * x[-L.plane];
            s += L.A[6 * nc + c] * x[L.plane];
        }
        const float v = (L.b[c] - s) * L.d[c];
        *x = v;
        if (kk == 0 && L.lower) L.lower[in] = v;
        if (kk == L.R - 1 && L.upper) L.upper[in] = v;
    }
}

__global__ void __launch_bounds__(512, 1) coarse_cluster_kernel(const __grid_constant__ LVSet S, const __grid_constant__ SlabPlan P,
                                                                int nu1, int nu2) {
    extern __shared__ __align__(16) float sm[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), cs = P.cs, tid = threadIdx.x;
    __shared__ LV<float> V[MAX_LEVELS];
    __shared__ CtaLevel T[MAX_LEVELS];
    __shared__ Slab W[SL_MAX];
    __shared__ __align__(8) unsigned long long bar;
    const int zc = S.l[S.first_cta].n[2];  // planes of the level below the split ones
    if (tid == 0) {
        BulkLoad load;
        load.init(&bar);
        for (int t = 0; t < P.ns; ++t) {
            const LV<float>& G = S.l[P.first + t];
            const int up = P.ns - t;
            auto start = [&](int q) { return slab_start(q, cs, zc) << up; };
            Slab& L = W[t];
            L.n0 = G.n[0], L.n1 = G.n[1], L.n2 = G.n[2], L.half = L.n0 / 2, L.plane = L.n0 * L.n1;
            L.mh = div_magic(L.half);
            L.m1 = div_magic(L.n1);
            L.z0 = start(rank);
            L.R = start(rank + 1) - L.z0;
            L.A = sm + P.oa[t];
            L.d = sm + P.od[t];
            L.b = sm + P.ob[t];
            L.x = sm + P.ox[t];
            const int lo = rank > 0 ? rank - 1 : (G.per[2] ? cs - 1 : -1), hi = rank < cs - 1 ? rank + 1 : (G.per[2] ? 0 : -1);
            L.lower = lo >= 0 ? cl.map_shared_rank(L.x, lo) + (start(lo + 1) - start(lo) + 1) * L.plane : nullptr;
            L.upper = hi >= 0 ? cl.map_shared_rank(L.x, hi) : nullptr;
            const int nc = L.R * L.plane;
            for (int k = 1; k < 7; ++k) load.copy(sm + P.oa[t] + k * nc, G.A + (size_t)k * G.ncell + L.z0 * L.plane, nc * 4);
            load.copy(sm + P.oa[t], G.A + L.z0 * L.plane, nc * 4);
            load.copy(sm + P.od[t], G.dinv + L.z0 * L.plane, nc * 4);
            if (t == 0) load.copy(L.b, G.b + L.z0 * L.plane, nc * 4);
        }
        cta_levels<7>(S, sm, P.ocoarse, V, T, load);
        const int mm = S.dense_m + (S.singular ? 1 : 0);
        if (P.odense) load.copy(sm + P.odense, S.dense_inv, (unsigned)((mm * mm * 4 + 15) & ~15));
        load.arrive();
    }
    __syncthreads();
    for (int t = 0; t < P.ns; ++t)
        for (int c = tid; c < (W[t].R + 2) * W[t].plane; c += 512) W[t].x[c] = 0.0f;
    for (int c = tid; c < T[S.first_cta].ncell; c += 512) T[S.first_cta].x[c] = 0.0f;
    const bool loaded = bulk_wait(&bar);
    // (a CTA whose wait ran out keeps to the barriers, on values that nobody uses)
    if (!loaded && tid == 0) *S.status = MG_WAIT_RAN_OUT;
    cl.sync();  // every CTA's x is set before a neighbour writes into it
    for (int t = 0; t < P.ns; ++t) {
        const Slab L = W[t];
        for (int it = 0; it < nu1; ++it)
            for (int col = 0; col < 2; ++col) {
                slab_sweep(L, col, it == 0 && col == 0);
                cl.sync();
            }
        // restriction, in restrict_kernel's order: to this CTA's planes of a split level, or to every
        // CTA's copy of the first level held whole
        const bool whole = t == P.ns - 1;
        const int cn0 = L.half, cn1 = L.n1 / 2, cplane = cn0 * cn1, cells = L.R / 2 * cplane, nc = L.R * L.plane;
        float* cb = whole ? T[S.first_cta].b : W[t + 1].b;
        for (int idx = tid; idx < cells; idx += 512) {
            const int row = div_by(idx, L.mh), ic = idx - row * cn0, kc = row / cn1, jc = row - kc * cn1;
            float acc = 0.0f;
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                const int i = 2 * ic + (ch & 1), j = 2 * jc + ((ch >> 1) & 1), kk = 2 * kc + (ch >> 2);
                const int c = kk * L.plane + j * L.n0 + i;
                const float* x = L.x + c + L.plane;
                float s = 0.0f;
                s += L.A[c] * x[0];
                s += L.A[nc + c] * x[i > 0 ? -1 : L.n0 - 1];
                s += L.A[2 * nc + c] * x[i < L.n0 - 1 ? 1 : 1 - L.n0];
                s += L.A[3 * nc + c] * x[(j > 0 ? -1 : L.n1 - 1) * L.n0];
                s += L.A[4 * nc + c] * x[(j < L.n1 - 1 ? 1 : 1 - L.n1) * L.n0];
                s += L.A[5 * nc + c] * x[-L.plane];
                s += L.A[6 * nc + c] * x[L.plane];
                acc += L.b[c] - s;
            }
            if (whole) {
                const int off = L.z0 / 2 * cplane + idx;
                for (int q = 0; q < cs; ++q) cl.map_shared_rank(cb, q)[off] = acc;
            } else {
                cb[idx] = acc;
            }
        }
        if (whole) cl.sync();
        else __syncthreads();
    }
    cta_cycle<3, 7>(S, V, T, P.odense ? sm + P.odense : nullptr, nu1, nu2);
    for (int t = P.ns - 1; t >= 0; --t) {
        const Slab L = W[t];
        const LV<float>& Cl = S.l[P.first + t + 1];
        const bool whole = t == P.ns - 1;
        const int cplane = Cl.n[0] * Cl.n[1];
        // plane K of the coarse correction is at xc + K cplane (a split level's planes are local)
        const float* xc = whole ? T[S.first_cta].x : W[t + 1].x + (1 - W[t + 1].z0) * cplane;
        for (int idx = tid; idx < L.R * L.n1 * L.half; idx += 512) {
            // prolongation onto the first colour (the next sweep overwrites the second), as prolong_at
            const int row = div_by(idx, L.mh), m = idx - row * L.half, kk = div_by(row, L.m1), j = row - kk * L.n1;
            const int q[3] = {2 * m + ((j + L.z0 + kk) & 1), j, L.z0 + kk};
            int off[3][2];
            float sg[3];
            int stride = 1;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int pa = q[a] >> 1;
                int nb = pa + ((q[a] & 1) ? 1 : -1);
                sg[a] = 1.0f;
                if (nb < 0 || nb >= Cl.n[a]) {
                    const int side = nb < 0 ? 0 : 1;
                    if (Cl.per[a]) {
                        if (a < 2 || whole) nb = nb < 0 ? nb + Cl.n[a] : nb - Cl.n[a];  // else: the halo plane
                    } else {
                        nb = side == 0 ? 0 : Cl.n[a] - 1;
                        if (Cl.bc[2 * a + side] == CPIC_BC_DIRICHLET) sg[a] = -1.0f;
                    }
                }
                off[a][0] = pa * stride;
                off[a][1] = nb * stride;
                stride *= Cl.n[a];
            }
            float acc = 0.0f;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                float w = 1.0f, sign = 1.0f;
                int at = 0;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int bit = (o >> a) & 1;
                    w *= bit ? 0.25f : 0.75f;
                    if (bit) sign *= sg[a];
                    at += off[a][bit];
                }
                acc += w * (sign * xc[at]);
            }
            const int in = j * L.n0 + q[0];
            float* x = L.x + (kk + 1) * L.plane + in;
            const float v = *x + acc;
            *x = v;
            if (kk == 0 && L.lower) L.lower[in] = v;
            if (kk == L.R - 1 && L.upper) L.upper[in] = v;
        }
        cl.sync();
        for (int it = 0; it < nu2; ++it)
            for (int col = 1; col >= 0; --col) {
                slab_sweep(L, col, false);
                cl.sync();  // the last one also keeps every CTA's memory until its neighbours are done
            }
    }
    const Slab L = W[0];
    float* out = S.l[P.first].x + L.z0 * L.plane;
    for (int c = tid; c < L.R * L.plane; c += 512) out[c] = L.x[L.plane + c];
    if (!loaded) (void)bulk_wait(&bar);
}

// ------------------------------------------------------------------ FP64 outer iteration
__device__ __forceinline__ void block_sum2(double& a, double& b, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    int w = tid >> 5, l = tid & 31;
    if (l == 0) {
        sh[2 * w] = a;
        sh[2 * w + 1] = b;
    }
    __syncthreads();
    if (w == 0) {
        int nw = (blockDim.x * blockDim.y) >> 5;
        a = l < nw ? sh[2 * l] : 0.0;
        b = l < nw ? sh[2 * l + 1] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
    }
    __syncthreads();
}

// Sums of N doubles a thread over a block of 256 threads, in a fixed order, given to every thread.
// The first step goes through shared memory so that one warp a sum does the additions: FP64 runs
// at under two operations per SM and clock here, and a shuffle tree in all eight warps costs
// 15 N x 256 / 1.7 cycles of it (3 us a block for three sums) against N x 400.
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N], double (*sh)[256]) {
    const int tid = threadIdx.x + blockDim.x * threadIdx.y, w = tid >> 5, l = tid & 31;
#pragma unroll
    for (int n = 0; n < N; ++n) sh[n][tid] = v[n];
    __syncthreads();
#pragma unroll
    for (int n = 0; n < N; ++n)
        if (w == n) {
            double a = sh[n][l];
#pragma unroll
            for (int i = 1; i < 8; ++i) a += sh[n][l + 32 * i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (l == 0) sh[n][0] = a;
        }
    __syncthreads();
#pragma unroll
    for (int n = 0; n < N; ++n) v[n] = sh[n][0];
    __syncthreads();
}

struct ResidualParams {
    LV<double> L;       // finest level, FP64 (x = phi, b = right-hand side)
    float* r32;         // FP32 residual (right-hand side of the correction cycle), or null
    double* r64;        // FP64 residual (Krylov iteration), or null
    const double* rh;   // shadow residual r^: (r^, r) is reduced when ks is set and !init
    KrylovState* ks;    // Krylov scalars to update, or null
    int init;           // first residual of a Krylov solve: start the recurrence
    double* part;       // [3 * gridDim.x]
    unsigned* ticket;
    DevCounters* ctr;
    int* done;
    int* told;          // page-locked host memory that gets *done too, or null
    double rtol;
    int max_cycles;
    int count_cycle;    // V-cycles since the previous residual
    int use_handle;
    cudaGraphConditionalHandle handle;
};

// r = b - M phi in FP64, its FP32 copy, and ||r|| (and ||b|| with the first residual of a solve);
// the last block to finish sums the block partials in a fixed order, updates the counters and
// decides whether to continue. A warp takes a row's segments of 32 cells.
// Bound by the FP64 rate: 19 operations a cell for the 3D operator.
template <int D, int NPT>
__global__ void __launch_bounds__(256) residual_kernel(const __grid_constant__ ResidualParams P) {
    __shared__ double sh[3][256];
    __shared__ bool last;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    if (!P.use_handle && *P.done) {  // a cycle enqueued before the host knew that the solve was done
        if (P.told && blockIdx.x == 0 && tid == 0) *P.told = 1;
        return;
    }
    const LV<double>& L = P.L;
    const bool dot_rh = P.ks && !P.init, with_b = P.count_cycle == 0;
    double v[3] = {0.0, 0.0, 0.0};  // (r, r), (r^, r), (b, b)
    const int spr = (L.n[0] + 31) / 32, nseg = L.n[1] * L.n[2] * spr;
    for (int w = blockIdx.x * blockDim.y + threadIdx.y; w < nseg; w += gridDim.x * blockDim.y) {
        const int row = w / spr, i = (w - row * spr) * 32 + threadIdx.x;
        if (i >= L.n[0]) continue;
        const int k = row / L.n[1], q[3] = {i, row - k * L.n[1], k};
        const int c = i + L.n[0] * row;
        const double b = L.b[c], r = b - stencil_sum<D, NPT, 0>(L, c, q);
        if (P.r32) P.r32[c] = (float)r;
        if (P.r64) P.r64[c] = r;
        v[0] += r * r;
        if (dot_rh) v[1] += P.rh[c] * r;
        if (with_b) v[2] += b * b;
    }
    block_sums<3>(v, sh);
    if (tid == 0) {
#pragma unroll
        for (int n = 0; n < 3; ++n) P.part[3 * blockIdx.x + n] = v[n];
        __threadfence();
        unsigned t = atomicAdd(P.ticket, 1u);
        last = t == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int n = 0; n < 3; ++n) v[n] = 0.0;
    for (int i = tid; i < (int)gridDim.x; i += 256)
#pragma unroll
        for (int n = 0; n < 3; ++n) v[n] += __ldcg(P.part + 3 * i + n);
    block_sums<3>(v, sh);
    if (tid == 0) {
        const double a = v[0], h = v[1];
        *P.ticket = 0;
        DevCounters* ctr = P.ctr;
        ctr->mg_cycles += P.count_cycle;
        if (with_b) ctr->mg_bnorm = sqrt(v[2]);
        if (KrylovState* ks = P.ks) {
            // (r^, r) of the new residual; a vanishing rho, alpha or omega restarts the
            // recurrence from r^ = p = r, whose rho is (r, r)
            const bool restart = P.init || !(ks->omega != 0.0) || !(ks->rho != 0.0) || !(ks->alpha != 0.0) ||
                                 !(fabs(h) > 1e-300) || !isfinite(h);
            if (restart) {
                ks->restart = 1;
                ks->rho = a;
                ks->beta = 0.0;
            } else {
                ks->restart = 0;
                ks->beta = (h / ks->rho) * (ks->alpha / ks->omega);
                ks->rho = h;
            }
        }
        const double res = relative_residual(a, ctr->mg_bnorm);
        ctr->mg_residual = res;
        bool converged = res <= P.rtol;
        const bool lost = ctr->mg_converged == MG_WAIT_RAN_OUT;  // a V-cycle's data did not arrive
        if (converged) set_converged(ctr);
        bool cont = !converged && !lost && ctr->mg_cycles < P.max_cycles;
        *P.done = cont ? 0 : 1;
        if (P.told) *P.told = cont ? 0 : 1;
        if (P.use_handle) cudaGraphSetConditional(P.handle, cont ? 1u : 0u);
    }
}

// phi += e (FP64 update with the FP32 correction), unless the solve is done (see mg_solve)
__global__ void update_kernel(double* phi, const float* e, int n, const int* done) {
    if (*done) return;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) phi[c] += (double)e[c];
}

// ---- BiCGStab steps (the scalars live in KrylovState; see the header comment)

// p = r + beta (p - omega v), or p = r^ = r on a restart; p is also the V-cycle's right-hand
// side. The direction vectors p, v and s are FP32 (they only shape the Krylov space: the
// residual and phi stay FP64), which keeps these passes off GB300's FP64 units.
__global__ void bicg_direction_kernel(int n, const double* __restrict__ r, double* rh, float* p, const float* v,
                                      float* b32, const KrylovState* ks) {
    const float beta = (float)ks->beta, omega = (float)ks->omega;
    const bool restart = ks->restart != 0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        float pc;
        if (restart) {
            rh[c] = r[c];
            pc = (float)r[c];
        } else {
            pc = (float)r[c] + beta * (p[c] - omega * v[c]);
        }
        p[c] = pc;
        b32[c] = pc;
    }
}

// y = M x32 over the finest level with the FP32 copy of the full operator (every stencil
// entry; on GB300 an FP64 product is bound by the FP64 rate, at about a third of the memory
// rate), reduced in FP64; mode 0: v = y, p^ = x32 kept, reduce (r^, v) ->
// alpha = rho / (r^, v); mode 1: reduce (y, s), (y, y) -> omega = (t, s) / (t, t)
template <int D, int NPT>
__global__ void __launch_bounds__(256) bicg_matvec_kernel(const __grid_constant__ LV<float> L, const float* __restrict__ x32, int mode,
                                                           float* v, float* ph32, const double* __restrict__ wr,
                                                           const float* __restrict__ ws, KrylovState* ks) {
    __shared__ double sh[2][256];
    __shared__ bool last;
    double d0 = 0.0, d1 = 0.0;
    const int nrows = L.n[1] * L.n[2];
    // one cell's product and its contributions to the reductions
    auto emit = [&](int c, float yf) {
        const double y = (double)yf;
        if (mode == 0) {
            v[c] = yf;
            ph32[c] = x32[c];
            d0 += wr[c] * y;  // r^
        } else {
            d0 += y * (double)ws[c];  // s
            d1 += y * y;
        }
    };
    if (L.n[0] % 4 == 0) {
        // four consecutive cells along axis 0 per thread: each stencil entry of the four is one
        // 16-byte load, and a neighbour row's four values one 16-byte load plus the value
        // beyond the end the shifted entries need; the per-cell sums are stencil_apply's
        const int n0 = L.n[0], spr = (n0 + 127) / 128, nseg = nrows * spr;
        for (int w = blockIdx.x * blockDim.y + threadIdx.y; w < nseg; w += gridDim.x * blockDim.y) {
            const int row = w / spr, i0 = ((w - row * spr) * 32 + threadIdx.x) * 4;
            if (i0 >= n0) continue;
            const int k = row / L.n[1], j = row - k * L.n[1];
            int lo[3], hi[3];
            const int qq[3] = {0, j, k};
#pragma unroll
            for (int a = 1; a < D; ++a) {
                lo[a] = qq[a] > 0 ? qq[a] - 1 : (L.per[a] ? L.n[a] - 1 : 0);
                hi[a] = qq[a] + 1 < L.n[a] ? qq[a] + 1 : (L.per[a] ? 0 : L.n[a] - 1);
            }
            const int jy[3] = {n0 * lo[1], n0 * j, n0 * hi[1]};
            int kz[3] = {0, 0, 0};
            if (D == 3) {
                const int pl = n0 * L.n[1];
                kz[0] = pl * lo[2];
                kz[1] = pl * k;
                kz[2] = pl * hi[2];
            }
            {
                const int il = i0 > 0 ? i0 - 1 : (L.per[0] ? n0 - 1 : 0);
                const int ir = i0 + 4 < n0 ? i0 + 4 : (L.per[0] ? 0 : n0 - 1);
                const int c = i0 + n0 * row;
                float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int e = 0; e < NPT; ++e) {
                    const int dx = koff(D, e, 0);
                    const int rb = jy[koff(D, e, 1) + 1] + (D == 3 ? kz[koff(D, e, 2) + 1] : 0);
                    const float4 xm = *reinterpret_cast<const float4*>(x32 + rb + i0);
                    float xs[4];
                    if (dx == 0) {
                        xs[0] = xm.x, xs[1] = xm.y, xs[2] = xm.z, xs[3] = xm.w;
                    } else if (dx < 0) {
                        // cell i0's left neighbour: wrapped, or i0 itself at a closed face
                        xs[0] = i0 > 0 || L.per[0] ? x32[rb + il] : xm.x;
                        xs[1] = xm.x, xs[2] = xm.y, xs[3] = xm.z;
                    } else {
                        xs[0] = xm.y, xs[1] = xm.z, xs[2] = xm.w;
                        xs[3] = i0 + 4 < n0 || L.per[0] ? x32[rb + ir] : xm.w;
                    }
                    const float4 a4 = *reinterpret_cast<const float4*>(L.A + (size_t)e * L.ncell + c);
                    acc[0] += a4.x * xs[0];
                    acc[1] += a4.y * xs[1];
                    acc[2] += a4.z * xs[2];
                    acc[3] += a4.w * xs[3];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) emit(c + u, acc[u]);
            }
        }
    } else {
        for (int row = blockIdx.x * blockDim.y + threadIdx.y; row < nrows; row += gridDim.x * blockDim.y) {
            int j = row % L.n[1], k = row / L.n[1];
            for (int i = threadIdx.x; i < L.n[0]; i += blockDim.x) {
                int q[3] = {i, j, k};
                int c = i + L.n[0] * row;
                emit(c, stencil_apply<D, NPT>(L, x32, c, q));
            }
        }
    }
    double d[2] = {d0, d1};
    block_sums<2>(d, sh);
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    if (tid == 0) {
        ks->part[3 * blockIdx.x] = d[0];
        ks->part[3 * blockIdx.x + 1] = d[1];
        __threadfence();
        unsigned t = atomicAdd(&ks->ticket, 1u);
        last = t == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    d[0] = d[1] = 0.0;
    for (int i = tid; i < (int)gridDim.x; i += 256) {
        d[0] += __ldcg(&ks->part[3 * i]);
        d[1] += __ldcg(&ks->part[3 * i + 1]);
    }
    block_sums<2>(d, sh);
    const double a = d[0], b = d[1];
    if (tid == 0) {
        ks->ticket = 0;
        if (mode == 0) {
            const double al = ks->rho / a;
            ks->alpha = (a != 0.0 && isfinite(al)) ? al : 0.0;
            ks->restart = 0;
        } else {
            const double om = a / b;
            ks->omega = (b > 0.0 && isfinite(om)) ? om : 0.0;
        }
    }
}

// s = r - alpha v (FP32), also the V-cycle's right-hand side
__global__ void bicg_s_kernel(int n, const double* __restrict__ r, const float* __restrict__ v, float* s,
                              float* b32, const KrylovState* ks) {
    const float alpha = (float)ks->alpha;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const float sc = (float)r[c] - alpha * v[c];
        s[c] = sc;
        b32[c] = sc;
    }
}

// phi += alpha p^ + omega s^: the step formed in FP32, added to phi in FP64
__global__ void bicg_update_kernel(int n, double* phi, const float* __restrict__ ph32, const float* __restrict__ sh32,
                                   const KrylovState* ks) {
    const float alpha = (float)ks->alpha, omega = (float)ks->omega;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x)
        phi[c] += (double)(alpha * ph32[c] + omega * sh32[c]);
}

// ------------------------------------------------------------------ small grids: the solve in one CTA
// A grid whose whole V-cycle runs in one CTA (COARSE_CELLS cells and fewer) is solved by BiCGStab in
// one launch, with every vector beside the levels in shared memory: as launches, an iteration
// on such a grid is eight kernels of two to ten microseconds each, most of it launch, ramp and
// the levels' staging. The same operations in the same order as those kernels (only the FP64
// sums are added up differently). A 32 x 32 cycle (9-point, 6
// iterations): 455 us with launches, 349 us so.
constexpr int CS_THREADS = 512;
constexpr size_t CS_SMEM_MAX = 208 * 1024;

struct CtaSolve {
    const double* A64;   // finest level, FP64 [NPF][ncell]
    const double* b64;
    double* phi;
    const float* A32;    // its FP32 copy
    int ovec;            // shared-memory offset (words) of the vectors
    int odense;          // of the dense inverse (0: global)
    double rtol;
    int max_cycles;
    DevCounters* ctr;
};

// sums of N doubles a thread over the block, in a fixed order, given to every thread
template <int N>
__device__ __forceinline__ void cta_sums(double (&v)[N], double (*sh)[CS_THREADS]) {
    const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
#pragma unroll
    for (int n = 0; n < N; ++n) sh[n][tid] = v[n];
    __syncthreads();
#pragma unroll
    for (int n = 0; n < N; ++n)
        if (w == n) {
            double a = sh[n][l];
#pragma unroll
            for (int i = 1; i < CS_THREADS / 32; ++i) a += sh[n][l + 32 * i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (l == 0) sh[n][0] = a;
        }
    __syncthreads();
#pragma unroll
    for (int n = 0; n < N; ++n) v[n] = sh[n][0];
    __syncthreads();
}

// NPT: stencil of the V-cycle, NPF: of the operator
template <int D, int NPT, int NPF>
__global__ void __launch_bounds__(CS_THREADS, 1) cta_solve_kernel(const __grid_constant__ LVSet S, const __grid_constant__ CtaSolve P,
                                                                  int nu1, int nu2) {
    extern __shared__ __align__(16) float sm[];
    __shared__ LV<float> V[MAX_LEVELS];
    __shared__ CtaLevel T[MAX_LEVELS];
    __shared__ double sh[3][CS_THREADS];
    __shared__ __align__(8) unsigned long long bar;
    const int tid = threadIdx.x, n = S.l[0].ncell;
    double* phi = reinterpret_cast<double*>(sm + P.ovec);
    double *r = phi + n, *rh = r + n;
    float *p = reinterpret_cast<float*>(rh + n), *v = p + n, *s = v + n, *ph = s + n;
    if (tid == 0) {
        BulkLoad load;
        load.init(&bar);
        cta_levels<NPT>(S, sm, 0, V, T, load);
        const int mm = S.dense_m + (S.singular ? 1 : 0);
        if (P.odense) load.copy(sm + P.odense, S.dense_inv, (unsigned)((mm * mm * 4 + 15) & ~15));
        load.arrive();
    }
    __syncthreads();  // the barrier is initialised before any other thread waits on it
    for (int c = tid; c < n; c += CS_THREADS) phi[c] = P.phi[c];
    if (!bulk_wait(&bar)) {
        if (tid == 0) *S.status = MG_WAIT_RAN_OUT;
        (void)bulk_wait(&bar);
        return;
    }
    const CtaLevel L = T[0];
    const float* dense = P.odense ? sm + P.odense : nullptr;
    auto steps = [&](int c) {
        const int row = div_by(c >> 1, L.mh), i = c - row * L.n0;  // an even first axis
        const int k = D == 3 ? div_by(row, L.m1) : 0;
        return Steps<D>(L, i, row - k * L.n1, k);
    };
    // r = b - M phi; (r, r), (r^, r) and, at the start, (b, b)
    auto residual = [&](bool init, double (&sum)[3]) {
        sum[0] = sum[1] = sum[2] = 0.0;
        for (int c = tid; c < n; c += CS_THREADS) {
            const Steps<D> st = steps(c);
            double acc = 0.0;
#pragma unroll
            for (int k = 0; k < NPF; ++k) acc += P.A64[k * n + c] * phi[c + st(k)];
            const double b = P.b64[c], x = b - acc;
            r[c] = x;
            sum[0] += x * x;
            if (init) sum[2] += b * b;
            else sum[1] += rh[c] * x;
        }
        cta_sums<3>(sum, sh);
    };
    // y = M x over the finest level
    auto product = [&](int c) {
        const Steps<D> st = steps(c);
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < NPF; ++k) acc += (NPF == NPT ? L.A[k * n + c] : __ldg(P.A32 + k * n + c)) * L.x[c + st(k)];
        return acc;
    };
    double sum[3], rho = 0.0, alpha = 0.0, omega = 0.0, beta = 0.0;
    bool restart = true;
    residual(true, sum);
    const double bnorm = sqrt(sum[2]);
    rho = sum[0];
    int cycles = 0;
    for (;;) {
        const double res = relative_residual(sum[0], bnorm);
        if (tid == 0) {
            P.ctr->mg_cycles = cycles;
            P.ctr->mg_residual = res;
            P.ctr->mg_bnorm = bnorm;
            if (res <= P.rtol) set_converged(P.ctr);
        }
        if (res <= P.rtol || cycles >= P.max_cycles) break;
        // p, and the V-cycle on it
        {
            const float bt = (float)beta, om = (float)omega;
            for (int c = tid; c < n; c += CS_THREADS) {
                float pc;
                if (restart) {
                    rh[c] = r[c];
                    pc = (float)r[c];
                } else {
                    pc = (float)r[c] + bt * (p[c] - om * v[c]);
                }
                p[c] = pc;
                L.b[c] = pc;
                L.x[c] = 0.0f;
            }
        }
        __syncthreads();
        cta_cycle<D, NPT>(S, V, T, dense, nu1, nu2);
        double d[2] = {0.0, 0.0};
        for (int c = tid; c < n; c += CS_THREADS) {
            const float y = product(c);
            v[c] = y;
            ph[c] = L.x[c];
            d[0] += rh[c] * (double)y;
        }
        cta_sums<2>(d, sh);
        {
            const double al = rho / d[0];
            alpha = (d[0] != 0.0 && isfinite(al)) ? al : 0.0;
        }
        // s, and the V-cycle on it
        {
            const float al = (float)alpha;
            for (int c = tid; c < n; c += CS_THREADS) {
                const float sc = (float)r[c] - al * v[c];
                s[c] = sc;
                L.b[c] = sc;
                L.x[c] = 0.0f;
            }
        }
        __syncthreads();
        cta_cycle<D, NPT>(S, V, T, dense, nu1, nu2);
        d[0] = d[1] = 0.0;
        for (int c = tid; c < n; c += CS_THREADS) {
            const double y = (double)product(c);
            d[0] += y * (double)s[c];
            d[1] += y * y;
        }
        cta_sums<2>(d, sh);
        {
            const double om = d[0] / d[1];
            omega = (d[1] > 0.0 && isfinite(om)) ? om : 0.0;
        }
        {
            const float al = (float)alpha, om = (float)omega;
            for (int c = tid; c < n; c += CS_THREADS) phi[c] += (double)(al * ph[c] + om * L.x[c]);
        }
        __syncthreads();
        cycles += 2;
        residual(false, sum);
        // as the residual kernel: a vanishing rho, alpha or omega restarts the recurrence
        const double h = sum[1];
        restart = !(omega != 0.0) || !(rho != 0.0) || !(alpha != 0.0) || !(fabs(h) > 1e-300) || !isfinite(h);
        beta = restart ? 0.0 : (h / rho) * (alpha / omega);
        rho = restart ? sum[0] : h;
    }
    for (int c = tid; c < n; c += CS_THREADS) P.phi[c] = phi[c];
}

// mode 1: (sum b, -); mode 2: (sum J phi, -)
__global__ void sum_kernel(LV<double> L, int mode, const double* Jc, double* part) {
    __shared__ double sh[64];
    double a = 0.0, b = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < L.ncell; c += gridDim.x * blockDim.x)
        a += mode == 1 ? L.b[c] : Jc[c] * L.x[c];
    block_sum2(a, b, sh);
    if (threadIdx.x == 0) part[2 * blockIdx.x] = a;
}

__device__ __forceinline__ double sum_parts(const double* part, int nb, double* sh) {
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) a += part[2 * i];
    block_sum2(a, b, sh);
    return a;  // valid in warp 0
}

// b -= (sum b / sum J) J  (singular problems)
__global__ void project_kernel(LV<double> L, const double* part, int nb, double sumJ, const double* Jc) {
    __shared__ double sh[64];
    __shared__ double shift;
    double s = sum_parts(part, nb, sh);
    if (threadIdx.x == 0) shift = s / sumJ;
    __syncthreads();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < L.ncell; c += gridDim.x * blockDim.x) L.b[c] -= shift * Jc[c];
}

// phi -= (sum J phi / sum J)  (gauge of singular problems)
__global__ void gauge_kernel(LV<double> L, const double* part, int nb, double sumJ) {
    __shared__ double sh[64];
    __shared__ double shift;
    double s = sum_parts(part, nb, sh);
    if (threadIdx.x == 0) shift = s / sumJ;
    __syncthreads();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < L.ncell; c += gridDim.x * blockDim.x) L.x[c] -= shift;
}

// ------------------------------------------------------------------ setup kernels
struct AsmParams {
    LV<double> L;
    const double* face[3];
    int bc[6];
    double bcv[6];
    double* A;
    double* bbc;  // may be null (coarse levels: homogeneous)
    int* cross_flag;
    unsigned* cross_max;  // largest (sum of |cross entries|) / diagonal of a row, as float bits
};

__device__ __forceinline__ int slot_of(int D, const int* o) {
    if (D == 2) {
        const int tab[9] = {5, 3, 6, 1, 0, 2, 7, 4, 8};
        return tab[(o[0] + 1) + 3 * (o[1] + 1)];
    }
    for (int k = 0; k < 27; ++k)
        if (c_off3[k][0] == o[0] && c_off3[k][1] == o[1] && c_off3[k][2] == o[2]) return k;
    return -1;
}

__global__ void assemble_kernel(AsmParams P) {
    const LV<double>& L = P.L;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < L.ncell; c += gridDim.x * blockDim.x) {
        int q[3];
        cell_coords(L, c, q);
        double a[27];
        for (int k = 0; k < 27; ++k) a[k] = 0.0;
        double rb = 0.0;
        auto add = [&](int* o, double val) {
            // fold ghost targets on non-periodic axes (Dirichlet: -phi_in + 2 phi_b)
            for (int ax = 0; ax < L.D; ++ax) {
                int tgt = q[ax] + o[ax];
                if (o[ax] != 0 && !L.per[ax] && (tgt < 0 || tgt >= L.n[ax])) {
                    int side = tgt < 0 ? 0 : 1;
                    o[ax] = 0;
                    if (P.bc[2 * ax + side] == CPIC_BC_DIRICHLET) {
                        rb -= 2.0 * val * P.bcv[2 * ax + side];
                        val = -val;
                    }
                }
            }
            int k = slot_of(L.D, o);
            a[k] += val;
        };
        for (int ax = 0; ax < L.D; ++ax) {
            int fn[3] = {L.n[0], L.n[1], L.D == 3 ? L.n[2] : 1};
            fn[ax] += 1;
            long long nf = (long long)fn[0] * fn[1] * fn[2];
            for (int side = 0; side < 2; ++side) {
                int fq[3] = {q[0], q[1], q[2]};
                fq[ax] += side;
                long long f = fq[0] + (long long)fn[0] * (fq[1] + (long long)fn[1] * fq[2]);
                double cf[3] = {0, 0, 0};
                for (int b = 0; b < L.D; ++b) cf[b] = P.face[ax][(long long)b * nf + f];
                bool boundary = !L.per[ax] && (fq[ax] == 0 || fq[ax] == L.n[ax]);
                if (boundary) {
                    if (P.bc[2 * ax + side] == CPIC_BC_DIRICHLET) {
                        a[0] += 2.0 * cf[ax];
                        rb += 2.0 * cf[ax] * P.bcv[2 * ax + side];
                    }
                    continue;
                }
                double sgn = side == 0 ? 1.0 : -1.0;
                int oR = side == 0 ? 0 : 1, oL = side == 0 ? -1 : 0;
                int o[3] = {0, 0, 0};
                o[ax] = oR;
                add(o, sgn * cf[ax]);
                o[0] = o[1] = o[2] = 0;
                o[ax] = oL;
                add(o, -sgn * cf[ax]);
                for (int b = 0; b < L.D; ++b) {
                    if (b == ax || cf[b] == 0.0) continue;
                    for (int sb = -1; sb <= 1; sb += 2) {
                        double val = sgn * sb * cf[b] * 0.25;
                        int o1[3] = {0, 0, 0};
                        o1[ax] = oR;
                        o1[b] = sb;
                        add(o1, val);
                        int o2[3] = {0, 0, 0};
                        o2[ax] = oL;
                        o2[b] = sb;
                        add(o2, val);
                    }
                }
            }
        }
        int faces = 2 * L.D + 1;
        bool cross = false;
        for (int k = 0; k < L.S; ++k) {
            P.A[(size_t)k * L.ncell + c] = a[k];
            if (k >= faces && a[k] != 0.0) cross = true;
        }
        if (cross) {
            atomicOr(P.cross_flag, 1);
            double off = 0.0;
            for (int k = faces; k < L.S; ++k) off += fabs(a[k]);
            const float ratio = a[0] != 0.0 ? (float)(off / fabs(a[0])) : 3.0e38f;
            atomicMax(P.cross_max, __float_as_uint(ratio));  // non-negative floats order as their bits
        }
        if (P.bbc) P.bbc[c] = rb;
    }
}

__global__ void inv_diag_kernel(const float* A, float* dinv, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dinv[i] = 1.0f / A[i];
}

__global__ void to_float_kernel(const double* src, float* dst, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (float)src[i];
}

// dst = src^T, rounded to FP32 (the dense inverse, as the coarse solves read it)
__global__ void to_float_transposed_kernel(const double* src, float* dst, int n) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
        const int i = e / n, k = e - i * n;
        dst[k * n + i] = (float)src[e];
    }
}

// dense matrix of the coarsest level (bordered with ones when singular), row-major mm x mm
__global__ void dense_matrix_kernel(LV<double> L, int singular, double* M) {
    int m = (int)L.ncell, mm = m + (singular ? 1 : 0);
    for (long long e = threadIdx.x; e < (long long)mm * mm; e += blockDim.x) M[e] = 0.0;
    __syncthreads();
    for (int c = threadIdx.x; c < m; c += blockDim.x) {
        int q[3];
        cell_coords(L, c, q);
        for (int k = 0; k < L.used; ++k) {
            int o[3];
            offsets(L.D, k, o);
            long long nb = nbr(L, q, o);
            double v = L.A[(size_t)k * L.ncell + c];
            if (v != 0.0) M[(long long)c * mm + nb] += v;
        }
        if (singular) {
            M[(long long)c * mm + m] = 1.0;
            M[(long long)m * mm + c] = 1.0;
        }
    }
}

// Gauss-Jordan inverse with partial pivoting, one block (setup only)
__global__ void gauss_jordan_kernel(double* M, double* Inv, int n, int* fail) {
    __shared__ int piv;
    for (long long e = threadIdx.x; e < (long long)n * n; e += blockDim.x) Inv[e] = (e / n == e % n) ? 1.0 : 0.0;
    __syncthreads();
    for (int col = 0; col < n; ++col) {
        if (threadIdx.x == 0) {
            int best = col;
            double bv = fabs(M[(long long)col * n + col]);
            for (int r = col + 1; r < n; ++r) {
                double v = fabs(M[(long long)r * n + col]);
                if (v > bv) {
                    bv = v;
                    best = r;
                }
            }
            piv = best;
            if (bv == 0.0) *fail = 1;
        }
        __syncthreads();
        int p = piv;
        if (p != col)
            for (int k = threadIdx.x; k < n; k += blockDim.x) {
                double t = M[(long long)col * n + k];
                M[(long long)col * n + k] = M[(long long)p * n + k];
                M[(long long)p * n + k] = t;
                t = Inv[(long long)col * n + k];
                Inv[(long long)col * n + k] = Inv[(long long)p * n + k];
                Inv[(long long)p * n + k] = t;
            }
        __syncthreads();
        double d = M[(long long)col * n + col];
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            M[(long long)col * n + k] /= d;
            Inv[(long long)col * n + k] /= d;
        }
        __syncthreads();
        for (long long e = threadIdx.x; e < (long long)n * n; e += blockDim.x) {
            int r = (int)(e / n), k = (int)(e % n);
            if (r == col || k == col) continue;
            double f = M[(long long)r * n + col];
            M[e] -= f * M[(long long)col * n + k];
            Inv[e] -= f * Inv[(long long)col * n + k];
        }
        __syncthreads();
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            if (r == col) continue;
            double f = M[(long long)r * n + col];
            Inv[(long long)r * n + col] -= f * Inv[(long long)col * n + col];
            M[(long long)r * n + col] = 0.0;
        }
        __syncthreads();
    }
}

template <typename R>
LV<R> make_lv(const cpic_run* r, int l, bool fp32) {
    const Level& Lv = r->lev[l];
    LV<R> L;
    L.D = r->D;
    for (int a = 0; a < 3; ++a) {
        L.n[a] = a < r->D ? Lv.n[a] : 1;
        L.per[a] = a < r->D ? (r->cfg.field_bc[2 * a] == CPIC_BC_PERIODIC) : 0;
    }
    for (int f = 0; f < 6; ++f) L.bc[f] = r->cfg.field_bc[f];
    L.ncell = (int)Lv.ncell;
    L.S = Lv.S;
    const bool cross = Lv.cross && !(fp32 && r->pc_face_only);
    const int full = r->D == 2 ? 9 : (r->mg_coarse == CPIC_MG_COARSE_GALERKIN ? 27 : 19);
    L.used = cross ? full : 2 * r->D + 1;
    L.ncol = cross ? (1 << r->D) : 2;
    L.lw = Lv.lw;
    L.pw = nullptr;
    if (r->mg_interp == CPIC_MG_INTERP_OPERATOR && l + 1 < r->nlevels)
        L.pw = fp32 ? (const R*)(const void*)Lv.pw32 : (const R*)(const void*)Lv.pw;
    if (fp32) {
        L.A = (const R*)Lv.A32;
        L.x = (R*)Lv.x32;
        L.b = (R*)Lv.b32;
        L.dinv = (const R*)Lv.dinv32;
    } else {
        L.dinv = nullptr;
        L.A = (const R*)Lv.A;
        L.x = (R*)Lv.x;
        L.b = (R*)Lv.b;
    }
    return L;
}

int grid_blocks(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 8LL * device_sm_count()) b = 8LL * device_sm_count();
    if (b < 1) b = 1;
    return (int)b;
}

constexpr size_t CTA_SMEM_MAX = 200 * 1024;  // shared memory of the one-CTA coarse cycle

// words of the one-CTA part from level l on: stencil (of the finest level's shape on every
// level), inverse diagonal, x, b of every smoothed level, x and b of the dense one
size_t cta_words(const LVSet& S, int l) {
    size_t f = 0;
    for (int k = l; k < S.nl; ++k) f += (size_t)(k < S.nl - 1 ? S.l[0].used + 3 : 2) * ((S.l[k].ncell + 3) & ~3);
    return f;
}

LVSet make_set(const cpic_run* r) {
    LVSet S;
    S.nl = r->nlevels;
    S.line = r->mg_smoother == CPIC_MG_SMOOTH_LINE ? 1 : 0;
    for (int l = 0; l < r->nlevels; ++l) S.l[l] = make_lv<float>(r, l, true);
    S.status = &r->ctr->mg_converged;
    S.dense_inv = r->dense_inv32;
    S.dense_m = (int)r->lev[r->nlevels - 1].ncell;
    S.singular = r->singular ? 1 : 0;
    // the one-CTA part starts at the first level of at most COARSE_CELLS cells from which
    // every coarser level fits the CTA's shared memory
    S.first_cta = r->nlevels - 1;
    for (int l = r->nlevels - 1; l >= 0; --l) {
        if (r->lev[l].ncell > COARSE_CELLS) break;
        if (cta_words(S, l) * sizeof(float) > CTA_SMEM_MAX) break;
        S.first_cta = l;
    }
    return S;
}

// shared memory of the one-CTA part; dense: the offset (words) of the dense inverse in it, 0 when it
// does not fit
size_t cta_smem_bytes(const LVSet& S, int* dense) {
    size_t f = cta_words(S, S.first_cta);
    const size_t mm = S.dense_m + S.singular, with = f + ((mm * mm + 3) & ~size_t(3));
    *dense = 0;
    if (with * sizeof(float) <= CTA_SMEM_MAX) {
        *dense = (int)f;
        f = with;
    }
    return f * sizeof(float);
}

int* done_flag(cpic_run* r) { return reinterpret_cast<int*>(r->red + 3 * KRY_BLOCKS + 2); }

// blocks of a pass over the finest level in segments of rows, eight warps a block: one segment a
// warp up to some three blocks an SM, four a warp beyond (each block ends with FP64 sums, 0.4 us)
int row_blocks(const cpic_run* r, int segment) {
    const long long rows = (long long)r->lev[0].n[1] * (r->D == 3 ? r->lev[0].n[2] : 1);
    const long long b = (rows * ((r->lev[0].n[0] + segment - 1) / segment) + 7) / 8;
    const long long few = b < 512 ? b : (b / 4 > 512 ? b / 4 : 512);
    return (int)(few > KRY_BLOCKS ? KRY_BLOCKS : few);
}

const dim3 kCellBlock(32, 8, 1);

dim3 cell_grid(int n0, int n1, int n2) {
    return dim3((unsigned)((n0 + 31) / 32), (unsigned)((n1 + 7) / 8), (unsigned)n2);
}

// calls f(std::integral_constant<int, D>, std::integral_constant<int, NPT>) for the run's
// stencil shape (all levels share it: the finest level's cross-term flag decides)
template <class F>
int dispatch_shape(const cpic_run* r, F f) {
    const bool cross = r->lev[0].cross != 0;
    if (r->D == 2) return cross ? f(std::integral_constant<int, 2>(), std::integral_constant<int, 9>())
                                : f(std::integral_constant<int, 2>(), std::integral_constant<int, 5>());
    if (r->mg_coarse == CPIC_MG_COARSE_GALERKIN)  // 27-point coarse levels
        return f(std::integral_constant<int, 3>(), std::integral_constant<int, 27>());
    return cross ? f(std::integral_constant<int, 3>(), std::integral_constant<int, 19>())
                 : f(std::integral_constant<int, 3>(), std::integral_constant<int, 7>());
}

// stencil shape of the FP32 V-cycle: the operator's, or its face entries alone when the
// cross entries are small enough to leave to the outer iteration (pc_face_only)
template <class F>
int dispatch_vshape(const cpic_run* r, F f) {
    const bool cross = r->lev[0].cross != 0 && !r->pc_face_only;
    if (r->D == 2) return cross ? f(std::integral_constant<int, 2>(), std::integral_constant<int, 9>())
                                : f(std::integral_constant<int, 2>(), std::integral_constant<int, 5>());
    if (r->mg_coarse == CPIC_MG_COARSE_GALERKIN)
        return f(std::integral_constant<int, 3>(), std::integral_constant<int, 27>());
    return cross ? f(std::integral_constant<int, 3>(), std::integral_constant<int, 19>())
                 : f(std::integral_constant<int, 3>(), std::integral_constant<int, 7>());
}

// The cluster part's levels, sizes and layout; false: the V-cycle has none (see SlabPlan). The
// CTAs are as many as the level below the split ones has planes, 16 at most (cs_max where the
// device co-schedules fewer).
bool plan_slabs(const LVSet& S, int cs_max, SlabPlan* P, size_t* smem) {
    const LV<float>& F = S.l[0];
    if (F.D != 3 || F.used != 7 || S.line || F.pw || cs_max < 2 || S.first_cta < 1 || S.first_cta >= S.nl - 1) return false;
    for (int ns = SL_MAX; ns > 0; --ns) {
        const int first = S.first_cta - ns;
        if (first < 0 || S.l[first].ncell > SL_CELLS) continue;
        const int planes = S.l[S.first_cta].n[2];
        const int cs = planes < cs_max ? planes : cs_max;
        if (cs < 2) continue;
        P->cs = cs;
        P->first = first;
        P->ns = ns;
        size_t off = 0;
        for (int t = 0; t < ns; ++t) {
            const LV<float>& L = S.l[first + t];
            const size_t plane = (size_t)L.n[0] * L.n[1], R = (size_t)((planes + cs - 1) / cs) << (ns - t);
            P->oa[t] = (int)off, off += 7 * R * plane;
            P->od[t] = (int)off, off += R * plane;
            P->ob[t] = (int)off, off += R * plane;
            P->ox[t] = (int)off, off += (R + 2) * plane;
        }
        P->ocoarse = (int)off;
        off += cta_words(S, S.first_cta);
        const size_t mm = S.dense_m + S.singular, dense = (mm * mm + 3) & ~size_t(3);
        P->odense = 0;
        if ((off + dense) * sizeof(float) <= SL_SMEM_MAX) {
            P->odense = (int)off;
            off += dense;
        }
        *smem = off * sizeof(float);
        if (*smem <= SL_SMEM_MAX) return true;
    }
    return false;
}

void slab_config(const SlabPlan& P, size_t smem, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
    cfg->gridDim = dim3(P.cs, 1, 1);
    cfg->blockDim = dim3(512, 1, 1);
    cfg->dynamicSmemBytes = smem;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = P.cs;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
}

// the largest cluster the device co-schedules for this run's cluster part (0: none)
int prepare_slabs(const cpic_run* r, int* cs_max) {
    *cs_max = 0;
    const LVSet S = make_set(r);
    for (int cs : {16, 8}) {
        SlabPlan P;
        size_t smem = 0;
        if (!plan_slabs(S, cs, &P, &smem)) return CPIC_OK;
        CPIC_CUDA(cudaFuncSetAttribute(coarse_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SL_SMEM_MAX));
        if (cudaFuncSetAttribute(coarse_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            cudaGetLastError();
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr;
        slab_config(P, smem, &cfg, &attr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, coarse_cluster_kernel, &cfg) == cudaSuccess && n > 0) {
            *cs_max = cs;
            return CPIC_OK;
        }
        cudaGetLastError();
    }
    return CPIC_OK;
}

// the levels of the one-CTA part
template <int D, int NPT>
int enqueue_coarse(cpic_run* r, const LVSet& S, int nu1, int nu2) {
    int dense = 0;
    const size_t smem = cta_smem_bytes(S, &dense);
    if (smem > CTA_SMEM_MAX) {
        set_error("multigrid: coarse levels need %zu bytes of shared memory", smem);
        return CPIC_ERR_INVALID;
    }
    // per-function attribute shared by every run (and by graphs captured earlier): set it
    // to the bound checked above, not to this run's need
    CPIC_CUDA(cudaFuncSetAttribute(coarse_cycle_kernel<D, NPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)CTA_SMEM_MAX));
    coarse_cycle_kernel<D, NPT><<<1, 512, smem, r->stream>>>(S, nu1, nu2, dense);
    CPIC_CHECK_LAUNCH();
    return CPIC_OK;
}

// whether the V-cycle takes one launch per level and direction (2D, two colours, point smoothing)
bool fused_levels(const LVSet& S) { return S.l[0].D == 2 && S.l[0].used == 5 && !S.line; }
// where the V-cycle leaves level l's correction
float* vcycle_result(const LVSet& S, int l) { return fused_levels(S) && l < S.first_cta ? S.l[l].lw : S.l[l].x; }

// one FP32 V-cycle on the correction equation (e = 0 first): vcycle_result(S, 0) = V(lev[0].b32)
int enqueue_vcycle(cpic_run* r, const LVSet& S) {
    return dispatch_vshape(r, [&](auto Dc, auto Nc) -> int {
        constexpr int D = decltype(Dc)::value, NPT = decltype(Nc)::value;
        cudaStream_t st = r->stream;
        const int nu1 = 2, nu2 = 2;
        int top = S.first_cta;  // levels above take a launch per pass
        SlabPlan slabs;
        size_t slab_smem = 0;
        const bool cluster = plan_slabs(S, r->slab_cs, &slabs, &slab_smem);
        if (cluster) top = slabs.first;
        // 2D two-colour levels: one launch down and one up each, the results in the levels' second
        // buffers (the line-relaxation work, free with point smoothing)
        if (D == 2 && NPT == 5 && fused_levels(S)) {
            auto tiles = [&](int l) {
                return dim3((unsigned)((S.l[l].n[0] + TL_X - 1) / TL_X), (unsigned)((S.l[l].n[1] + TL_Y - 1) / TL_Y));
            };
            for (int l = 0; l < top; ++l) {
                level_down2_kernel<<<tiles(l), TL_THREADS, 0, st>>>(S.l[l], S.l[l + 1].b, S.l[l + 1].n[0]);
                CPIC_CHECK_LAUNCH();
            }
            if (int e = enqueue_coarse<D, NPT>(r, S, nu1, nu2)) return e;
            for (int l = top - 1; l >= 0; --l) {
                LV<float> C = S.l[l + 1];
                C.x = vcycle_result(S, l + 1);
                level_up2_kernel<<<tiles(l), TL_THREADS, 0, st>>>(S.l[l], C, vcycle_result(S, l));
                CPIC_CHECK_LAUNCH();
            }
            return CPIC_OK;
        }
        const bool first = D == 3 && NPT == 7 && !S.line && nu1 > 0;  // the first two sweeps in one pass
        if (top > 0 && !first) CPIC_CUDA(cudaMemsetAsync(r->lev[0].x32, 0, sizeof(float) * r->lev[0].ncell, st));
        auto smooth = [&](int l, int col) -> int {
            const LV<float>& L = S.l[l];
            int d[3] = {L.n[0] / 2, Col<D, NPT>::parity ? L.n[1] : L.n[1] / 2,
                        D == 3 ? (Col<D, NPT>::parity ? L.n[2] : L.n[2] / 2) : 1};
            smooth_kernel<D, NPT><<<cell_grid(d[0], d[1], d[2]), kCellBlock, 0, st>>>(L, r->lev[l].dinv32, col);
            CPIC_CHECK_LAUNCH();
            return CPIC_OK;
        };
        // alternating zebra line relaxation: one thread per line (those of other colours
        // return at once)
        auto line_smooth = [&](int l, bool reverse) -> int {
            const LV<float>& L = S.l[l];
            for (int stp = 0; stp < D; ++stp) {
                const int axis = reverse ? D - 1 - stp : stp;
                int b, c, ncol;
                line_axes(L, D, axis, b, c, ncol);
                const int lines = L.ncell / L.n[axis];
                for (int cc = 0; cc < ncol; ++cc) {
                    const int col = reverse ? ncol - 1 - cc : cc;
                    line_kernel<D, NPT><<<(lines + 63) / 64, 64, 0, st>>>(L, axis, col, lines);
                    CPIC_CHECK_LAUNCH();
                }
            }
            return CPIC_OK;
        };
        for (int l = 0; l < top; ++l) {
            for (int it = 0; it < nu1; ++it) {
                if (S.line) {
                    if (int e = line_smooth(l, false)) return e;
                    continue;
                }
                if (first && it == 0) {
                    const LV<float>& L = S.l[l];
                    first_sweeps3_kernel<<<cell_grid(L.n[0] / 2, L.n[1], L.n[2]), kCellBlock, 0, st>>>(L);
                    CPIC_CHECK_LAUNCH();
                    continue;
                }
                for (int col = 0; col < S.l[l].ncol; ++col)
                    if (int e = smooth(l, col)) return e;
            }
            const LV<float>& C = S.l[l + 1];
            const LV<float>& Fl = S.l[l];
            const dim3 rb(32, D == 3 ? 4 : 8, D == 3 ? 2 : 1);
            const dim3 rg((unsigned)((Fl.n[0] + 31) / 32), (unsigned)((Fl.n[1] + rb.y - 1) / rb.y),
                          (unsigned)(D == 3 ? (Fl.n[2] + 1) / 2 : 1));
            restrict_kernel<D, NPT><<<rg, rb, 0, st>>>(Fl, C);
            CPIC_CHECK_LAUNCH();
        }
        if (cluster) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr;
            slab_config(slabs, slab_smem, &cfg, &attr);
            cfg.stream = st;
            CPIC_CUDA(cudaLaunchKernelEx(&cfg, coarse_cluster_kernel, S, slabs, nu1, nu2));
            CPIC_CHECK_LAUNCH();
        } else if (int e = enqueue_coarse<D, NPT>(r, S, nu1, nu2)) {
            return e;
        }
        for (int l = top - 1; l >= 0; --l) {
            const LV<float>& L = S.l[l];
            prolong_kernel<D><<<cell_grid(L.n[0], L.n[1], L.n[2]), kCellBlock, 0, st>>>(L, S.l[l + 1]);
            CPIC_CHECK_LAUNCH();
            for (int it = 0; it < nu2; ++it) {
                if (S.line) {
                    if (int e = line_smooth(l, true)) return e;
                    continue;
                }
                for (int col = L.ncol - 1; col >= 0; --col)
                    if (int e = smooth(l, col)) return e;
            }
        }
        return CPIC_OK;
    });
}

// one V-cycle on the residual, then phi += e
int enqueue_correction(cpic_run* r, const LVSet& S) {
    int st = enqueue_vcycle(r, S);
    if (st) return st;
    update_kernel<<<grid_blocks(r->lev[0].ncell, 256), 256, 0, r->stream>>>(r->lev[0].x, vcycle_result(S, 0),
                                                                            (int)r->lev[0].ncell, done_flag(r));
    CPIC_CHECK_LAUNCH();
    return CPIC_OK;
}

// krylov: 0 plain iteration (FP32 residual for the next V-cycle); 1 first residual of a
// BiCGStab solve; 2 residual after a BiCGStab iteration
int enqueue_residual(cpic_run* r, double rtol, int max_cycles, int count_cycle, bool use_handle,
                     cudaGraphConditionalHandle h, int krylov = 0, int* told = nullptr) {
    ResidualParams P;
    P.L = make_lv<double>(r, 0, false);
    P.r32 = krylov ? nullptr : r->lev[0].b32;
    P.r64 = krylov ? r->kv : nullptr;
    P.rh = krylov ? r->kv + r->ncell : nullptr;
    P.ks = krylov ? r->kry : nullptr;
    P.init = krylov == 1 ? 1 : 0;
    P.part = r->red;
    P.ticket = r->ticket;
    P.ctr = r->ctr;
    P.done = done_flag(r);
    P.told = told;
    P.rtol = rtol;
    P.max_cycles = max_cycles;
    P.count_cycle = count_cycle;
    P.use_handle = use_handle ? 1 : 0;
    P.handle = h;
    return dispatch_shape(r, [&](auto Dc, auto Nc) -> int {
        residual_kernel<decltype(Dc)::value, decltype(Nc)::value><<<row_blocks(r, 32), kCellBlock, 0, r->stream>>>(P);
        CPIC_CHECK_LAUNCH();
        return CPIC_OK;
    });
}

// one BiCGStab iteration (two V-cycles) ending with the residual that decides whether to go on
int enqueue_bicg_iteration(cpic_run* r, const LVSet& S, double rtol, int max_cycles, bool use_handle,
                           cudaGraphConditionalHandle h) {
    const int n = (int)r->ncell;
    double* rv = r->kv;
    double* rh = r->kv + r->ncell;
    float* p = reinterpret_cast<float*>(r->kv + 2 * r->ncell);  // FP32 p, v, s after r, r^
    float* v = p + r->ncell;
    float* s = v + r->ncell;
    float* b32 = r->lev[0].b32;
    const float* x32 = vcycle_result(S, 0);
    cudaStream_t st = r->stream;
    const int gb = grid_blocks(n, 256);
    bicg_direction_kernel<<<gb, 256, 0, st>>>(n, rv, rh, p, v, b32, r->kry);
    CPIC_CHECK_LAUNCH();
    int e = enqueue_vcycle(r, S);
    if (e) return e;
    LV<float> L0 = make_lv<float>(r, 0, true);  // A32 holds every entry of the operator
    e = dispatch_shape(r, [&](auto Dc, auto Nc) -> int {
        bicg_matvec_kernel<decltype(Dc)::value, decltype(Nc)::value>
            <<<row_blocks(r, r->n[0] % 4 ? 32 : 128), kCellBlock, 0, st>>>(L0, x32, 0, v, r->ph32, rh, nullptr, r->kry);
        CPIC_CHECK_LAUNCH();
        return CPIC_OK;
    });
    if (e) return e;
    bicg_s_kernel<<<gb, 256, 0, st>>>(n, rv, v, s, b32, r->kry);
    CPIC_CHECK_LAUNCH();
    e = enqueue_vcycle(r, S);
    if (e) return e;
    e = dispatch_shape(r, [&](auto Dc, auto Nc) -> int {
        bicg_matvec_kernel<decltype(Dc)::value, decltype(Nc)::value>
            <<<row_blocks(r, r->n[0] % 4 ? 32 : 128), kCellBlock, 0, st>>>(L0, x32, 1, nullptr, nullptr, nullptr, s, r->kry);
        CPIC_CHECK_LAUNCH();
        return CPIC_OK;
    });
    if (e) return e;
    bicg_update_kernel<<<gb, 256, 0, st>>>(n, r->lev[0].x, r->ph32, x32, r->kry);
    CPIC_CHECK_LAUNCH();
    return enqueue_residual(r, rtol, max_cycles, 2, use_handle, h, 2);
}

// the one-CTA solve's shared memory, or 0 where it does not apply
size_t cta_solve_bytes(const cpic_run* r, const LVSet& S, CtaSolve* P) {
    if (r->solver != CPIC_SOLVER_BICGSTAB || r->cluster_class || S.first_cta != 0 || S.nl < 2 || S.line || S.l[0].pw ||
        r->mg_coarse == CPIC_MG_COARSE_GALERKIN)
        return 0;
    size_t f = (cta_words(S, 0) + 3) & ~size_t(3);
    P->ovec = (int)f;
    f += (size_t)10 * S.l[0].ncell;  // three FP64 and four FP32 vectors
    const size_t mm = S.dense_m + S.singular, dense = (mm * mm + 3) & ~size_t(3);
    P->odense = 0;
    if ((f + dense) * sizeof(float) <= CS_SMEM_MAX) {
        P->odense = (int)f;
        f += dense;
    }
    return f * sizeof(float) <= CS_SMEM_MAX ? f * sizeof(float) : 0;
}

template <int D, int NPT, int NPF>
int launch_cta_solve(cpic_run* r, const LVSet& S, const CtaSolve& P, size_t smem) {
    auto kernel = cta_solve_kernel<D, NPT, NPF>;
    CPIC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CS_SMEM_MAX));
    kernel<<<1, CS_THREADS, smem, r->stream>>>(S, P, 2, 2);
    CPIC_CHECK_LAUNCH();
    return CPIC_OK;
}

int enqueue_cta_solve(cpic_run* r, const LVSet& S, CtaSolve P, size_t smem, double rtol, int max_cycles) {
    P.A64 = r->lev[0].A;
    P.b64 = r->lev[0].b;
    P.phi = r->lev[0].x;
    P.A32 = r->lev[0].A32;
    P.rtol = rtol;
    P.max_cycles = max_cycles;
    P.ctr = r->ctr;
    const bool cross = r->lev[0].cross != 0, face = !cross || r->pc_face_only;
    if (r->D == 2)
        return !cross ? launch_cta_solve<2, 5, 5>(r, S, P, smem)
                      : (face ? launch_cta_solve<2, 5, 9>(r, S, P, smem) : launch_cta_solve<2, 9, 9>(r, S, P, smem));
    return !cross ? launch_cta_solve<3, 7, 7>(r, S, P, smem)
                  : (face ? launch_cta_solve<3, 7, 19>(r, S, P, smem) : launch_cta_solve<3, 19, 19>(r, S, P, smem));
}

bool use_krylov(const cpic_run* r) { return r->solver == CPIC_SOLVER_BICGSTAB && !r->cluster_class; }

// right-hand side (and its projection); resets the solve counters
int enqueue_prologue(cpic_run* r, bool fold) {
    int st = launch_rhs(r, r->lev[0].b, fold, done_flag(r), r->ticket);
    if (st) return st;
    if (r->singular) {
        LV<double> L0 = make_lv<double>(r, 0, false);
        sum_kernel<<<RED_BLOCKS, 256, 0, r->stream>>>(L0, 1, r->lev[0].Jc, r->red);
        CPIC_CHECK_LAUNCH();
        project_kernel<<<grid_blocks(L0.ncell, 256), 256, 0, r->stream>>>(L0, r->red, RED_BLOCKS, r->sumJ, r->lev[0].Jc);
        CPIC_CHECK_LAUNCH();
    }
    return CPIC_OK;
}

int enqueue_epilogue(cpic_run* r) {
    if (r->singular) {
        LV<double> L0 = make_lv<double>(r, 0, false);
        sum_kernel<<<RED_BLOCKS, 256, 0, r->stream>>>(L0, 2, r->lev[0].Jc, r->red);
        CPIC_CHECK_LAUNCH();
        gauge_kernel<<<grid_blocks(L0.ncell, 256), 256, 0, r->stream>>>(L0, r->red, RED_BLOCKS, r->sumJ);
        CPIC_CHECK_LAUNCH();
    }
    int st = launch_floating(r);  // a floating conductor's potential from its charge
    if (st) return st;
    return launch_field_energy(r);
}

}  // namespace

int mg_setup(cpic_run* r) {
    int* flag = reinterpret_cast<int*>(r->red + 3 * KRY_BLOCKS + 4);
    unsigned* cmax = reinterpret_cast<unsigned*>(r->red + 3 * KRY_BLOCKS + 6);
    r->pc_face_only = 0;
    for (int l = 0; l < r->nlevels; ++l) {
        Level& Lv = r->lev[l];
        CPIC_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), r->stream));
        CPIC_CUDA(cudaMemsetAsync(cmax, 0, sizeof(unsigned), r->stream));
        AsmParams P;
        Lv.cross = 1;  // all entries while assembling
        P.L = make_lv<double>(r, l, false);
        for (int a = 0; a < 3; ++a) P.face[a] = Lv.face[a];
        for (int f = 0; f < 6; ++f) {
            P.bc[f] = r->cfg.field_bc[f];
            P.bcv[f] = l == 0 ? r->cfg.field_bc_value[f] : 0.0;
        }
        P.A = Lv.A;
        P.bbc = l == 0 ? r->rhs_bc : nullptr;
        P.cross_flag = flag;
        P.cross_max = cmax;
        const bool galerkin = r->mg_coarse == CPIC_MG_COARSE_GALERKIN;
        if (l > 0 && r->mg_interp == CPIC_MG_INTERP_OPERATOR) {
            // the prolongation weights of the level above, from its (finished) operator
            LV<double> F = make_lv<double>(r, l - 1, false);
            if (r->D == 2)
                interp_weights_kernel<2><<<grid_blocks(F.ncell, 256), 256, 0, r->stream>>>(F, r->lev[l - 1].pw,
                                                                                           r->lev[l - 1].pw32);
            else
                interp_weights_kernel<3><<<grid_blocks(F.ncell, 256), 256, 0, r->stream>>>(F, r->lev[l - 1].pw,
                                                                                           r->lev[l - 1].pw32);
            CPIC_CHECK_LAUNCH();
        }
        if (galerkin && l > 0) {
            // variational coarse operator from the level above (its full stencil)
            LV<double> F = make_lv<double>(r, l - 1, false);
            if (r->D == 2)
                galerkin_kernel<2><<<grid_blocks(Lv.ncell, 256), 256, 0, r->stream>>>(F, P.L, Lv.A);
            else
                galerkin_kernel<3><<<grid_blocks(Lv.ncell, 256), 256, 0, r->stream>>>(F, P.L, Lv.A);
        } else {
            assemble_kernel<<<grid_blocks(Lv.ncell, 256), 256, 0, r->stream>>>(P);
        }
        CPIC_CHECK_LAUNCH();
        to_float_kernel<<<grid_blocks((long long)Lv.S * Lv.ncell, 256), 256, 0, r->stream>>>(Lv.A, Lv.A32,
                                                                                              (long long)Lv.S * Lv.ncell);
        CPIC_CHECK_LAUNCH();
        inv_diag_kernel<<<grid_blocks(Lv.ncell, 256), 256, 0, r->stream>>>(Lv.A32, Lv.dinv32, (int)Lv.ncell);
        CPIC_CHECK_LAUNCH();
        int hflag = 0;
        unsigned hmax = 0;
        CPIC_CUDA(cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, r->stream));
        CPIC_CUDA(cudaMemcpyAsync(&hmax, cmax, sizeof(unsigned), cudaMemcpyDeviceToHost, r->stream));
        CPIC_CUDA(cudaStreamSynchronize(r->stream));
        Lv.cross = hflag;
        // Galerkin coarse operators are 9/27-point: the V-cycle keeps every entry on every level
        if (r->mg_coarse == CPIC_MG_COARSE_GALERKIN) Lv.cross = 1;
        if (l == 0) {
            float ratio;
            memcpy(&ratio, &hmax, sizeof(ratio));
            // CPIC_PC_FULL_STENCIL in the environment keeps the full stencil in the V-cycle
            // (the face-only form is a cost choice; both meet the same stopping test)
            r->pc_face_only = hflag && ratio <= PC_CROSS_DROP && !getenv("CPIC_PC_FULL_STENCIL") &&
                                      r->mg_coarse != CPIC_MG_COARSE_GALERKIN
                                  ? 1
                                  : 0;
        }
    }
    const Level& Lc = r->lev[r->nlevels - 1];
    int m = (int)Lc.ncell;
    int mm = m + (r->singular ? 1 : 0);
    r->dense_m = mm;
    LV<double> L = make_lv<double>(r, r->nlevels - 1, false);
    if (r->pc_face_only) L.used = 2 * r->D + 1;  // the coarsest solve of the V-cycle's operator
    dense_matrix_kernel<<<1, 256, 0, r->stream>>>(L, r->singular ? 1 : 0, r->dense_tmp);
    CPIC_CHECK_LAUNCH();
    int* fail = flag;
    CPIC_CUDA(cudaMemsetAsync(fail, 0, sizeof(int), r->stream));
    gauss_jordan_kernel<<<1, 1024, 0, r->stream>>>(r->dense_tmp, r->dense_inv, mm, fail);
    CPIC_CHECK_LAUNCH();
    to_float_transposed_kernel<<<grid_blocks((long long)mm * mm, 256), 256, 0, r->stream>>>(r->dense_inv, r->dense_inv32, mm);
    CPIC_CHECK_LAUNCH();
    CPIC_CUDA(cudaMemsetAsync(r->ticket, 0, sizeof(unsigned) * 4, r->stream));
    CPIC_CUDA(cudaMemsetAsync(r->kry, 0, sizeof(KrylovState), r->stream));
    int hfail = 0;
    CPIC_CUDA(cudaMemcpyAsync(&hfail, fail, sizeof(int), cudaMemcpyDeviceToHost, r->stream));
    CPIC_CUDA(cudaStreamSynchronize(r->stream));
    if (hfail) {
        set_error("coarsest multigrid operator is singular");
        return CPIC_ERR_INVALID;
    }
    return prepare_slabs(r, &r->slab_cs);
}

// Stream-ordered solve (cpic_solve_field and the steps of an uncaptured cpic_step); where no single
// kernel holds the loop, the host reads the device's decision after every cycle.
int mg_solve(cpic_run* r, double rtol, int max_cycles, bool fold, int* cycles, double* res) {
    LVSet S = make_set(r);
    CtaSolve one;
    // The grids of the cluster solver's class that no layout fits (see cluster_takes) have cycles of
    // some 40 us, and a host that waits for each adds half as much: they are kept one cycle ahead,
    // with the decision written straight to host memory, and what is enqueued beyond the last one
    // leaves phi and the counters alone. (Larger grids lose more by that cycle than by the waits.)
    // 192 x 128, 15 cycles: 850 to 903 us, 1009 with a copy and a wait a cycle; 256 x 64, 90: 4229 to
    // 4454 and 5583.
    const bool ahead = max_cycles > 0 && r->cluster_class && !r->cluster_cs;
    auto told = [&](int cyc) { return ahead ? r->done_host + (cyc & 1) : nullptr; };
    auto mark = [&](int cyc) -> int {
        CPIC_CUDA(cudaEventRecord(r->done_event[cyc & 1], r->stream));
        return CPIC_OK;
    };
    int st = enqueue_prologue(r, fold);
    if (st) return st;
    if (r->cluster_cs) {
        st = mg_cluster_solve(r, rtol, max_cycles);
        if (st) return st;
        max_cycles = 0;  // the loop ran inside the cluster kernel
    } else if (const size_t smem = cta_solve_bytes(r, S, &one)) {
        st = enqueue_cta_solve(r, S, one, smem, rtol, max_cycles);
        if (st) return st;
        max_cycles = 0;
    } else {
        st = enqueue_residual(r, rtol, max_cycles, 0, false, 0, use_krylov(r) ? 1 : 0, told(0));
        if (!st && ahead) st = mark(0);
        if (st) return st;
    }
    for (int cyc = 0; cyc < max_cycles; ++cyc) {
        if (!ahead) {
            int hd = 0;
            CPIC_CUDA(cudaMemcpyAsync(&hd, done_flag(r), sizeof(int), cudaMemcpyDeviceToHost, r->stream));
            CPIC_CUDA(cudaStreamSynchronize(r->stream));
            if (hd) break;
        }
        if (use_krylov(r)) {
            st = enqueue_bicg_iteration(r, S, rtol, max_cycles, false, 0);
        } else {
            st = enqueue_correction(r, S);
            if (!st) st = enqueue_residual(r, rtol, max_cycles, 1, false, 0, 0, told(cyc + 1));
        }
        if (!st && ahead) st = mark(cyc + 1);
        if (st) return st;
        if (ahead) {
            CPIC_CUDA(cudaEventSynchronize(r->done_event[cyc & 1]));
            if (r->done_host[cyc & 1]) break;
        }
    }
    st = enqueue_epilogue(r);
    if (st) return st;
    if (cycles || res) {
        DevCounters h;
        CPIC_CUDA(cudaMemcpyAsync(&h, r->ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost, r->stream));
        CPIC_CUDA(cudaStreamSynchronize(r->stream));
        if (cycles) *cycles = h.mg_cycles;
        if (res) *res = h.mg_residual;
        if (h.mg_converged == MG_WAIT_RAN_OUT) return wait_ran_out();
        if (!h.mg_converged) {
            set_error("multigrid: relative residual %.3e > %.3e after %d cycles", h.mg_residual, rtol, h.mg_cycles);
            return CPIC_ERR_NOT_CONVERGED;
        }
    }
    return CPIC_OK;
}

// The solve as part of a graph being captured on r->stream (capture target `g`): the
// prologue and first residual are captured in place, the cycles go into the body of a
// conditional WHILE node the residual kernel drives, the epilogue follows the node.
int mg_capture_solve(cpic_run* r, cudaGraph_t g, double rtol, int max_cycles) {
    LVSet S = make_set(r);
    if (r->cluster_cs) {
        int st = enqueue_prologue(r, true);
        if (st) return st;
        st = mg_cluster_solve(r, rtol, max_cycles);
        if (st) return st;
        return enqueue_epilogue(r);
    }
    CtaSolve one;
    if (const size_t smem = cta_solve_bytes(r, S, &one)) {
        int st = enqueue_prologue(r, true);
        if (!st) st = enqueue_cta_solve(r, S, one, smem, rtol, max_cycles);
        return st ? st : enqueue_epilogue(r);
    }
    cudaGraphConditionalHandle h;
    CPIC_CUDA(cudaGraphConditionalHandleCreate(&h, g, 0, 0));
    int st = enqueue_prologue(r, true);
    if (st) return st;
    st = enqueue_residual(r, rtol, max_cycles, 0, true, h, use_krylov(r) ? 1 : 0);
    if (st) return st;
    // splice the WHILE node after the current capture frontier
    cudaStreamCaptureStatus cs;
    const cudaGraphNode_t* deps = nullptr;
    size_t ndeps = 0;
    CPIC_CUDA(cudaStreamGetCaptureInfo(r->stream, &cs, nullptr, nullptr, &deps, nullptr, &ndeps));
    // the parameter struct has a union member without a default constructor: zeroed storage
    alignas(cudaGraphNodeParams) unsigned char npbuf[sizeof(cudaGraphNodeParams)];
    memset(npbuf, 0, sizeof(npbuf));
    cudaGraphNodeParams* np = reinterpret_cast<cudaGraphNodeParams*>(npbuf);
    np->type = cudaGraphNodeTypeConditional;
    np->conditional.handle = h;
    np->conditional.type = cudaGraphCondTypeWhile;
    np->conditional.size = 1;
    cudaGraphNode_t wnode;
    CPIC_CUDA(cudaGraphAddNode(&wnode, g, deps, nullptr, ndeps, np));
    cudaGraph_t body = np->conditional.phGraph_out[0];
    // the rest of the outer capture depends on the WHILE node
    CPIC_CUDA(cudaStreamUpdateCaptureDependencies(r->stream, &wnode, nullptr, 1, cudaStreamSetCaptureDependencies));
    // body: capture on a side stream into the body graph
    cudaStream_t side;
    CPIC_CUDA(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    cudaStream_t saved = r->stream;
    r->stream = side;
    st = CPIC_OK;
    cudaError_t e = cudaStreamBeginCaptureToGraph(side, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
    if (e == cudaSuccess) {
        if (use_krylov(r)) {
            st = enqueue_bicg_iteration(r, S, rtol, max_cycles, true, h);
        } else {
            st = enqueue_correction(r, S);
            if (!st) st = enqueue_residual(r, rtol, max_cycles, 1, true, h);
        }
        cudaGraph_t out = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(side, &out);
        if (!st && e2 != cudaSuccess) st = cuda_fail(e2, "cudaStreamEndCapture(body)", __FILE__, __LINE__);
    } else {
        st = cuda_fail(e, "cudaStreamBeginCaptureToGraph(body)", __FILE__, __LINE__);
    }
    r->stream = saved;
    cudaStreamDestroy(side);
    if (st) return st;
    return enqueue_epilogue(r);
}

}  // namespace cpic
