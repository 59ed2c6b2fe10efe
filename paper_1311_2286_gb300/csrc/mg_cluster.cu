// Row a9 on a thread-block cluster: the whole mixed-precision multigrid solve of a 2D
// 5-point problem in one kernel launch.
//
// Same method as mg.cu (FP64 solution and stopping test, FP32 V(2,2)-cycles on the
// correction, two-colour Gauss-Seidel, residual-sum restriction, bilinear prolongation, dense
// coarsest solve, stop at ||r||/||b|| <= rtol), laid out so that a V-cycle is a short chain:
//   - Levels 0 .. nd-1 are split by rows over the cluster's CTAs, the levels below are held
//     whole and solved redundantly by every CTA, all in shared memory. A CTA also holds HALO
//     rows of its neighbours' slabs and relaxes them redundantly: one exchange of halo rows
//     (written straight into the neighbours' shared memory) and one cluster barrier carry
//     four colour sweeps, so a split level costs two cluster barriers a V-cycle. A cluster
//     barrier with its exchange takes about 700 cycles here, a block barrier 45.
//   - Each row stores its two colours apart, so a sweep reads shared memory without bank
//     conflicts; the symmetric operator is kept as two couplings a cell.
//   - Work whose result the cycle does not use is left out: the first sweep from x = 0 is
//     x = b / diag; after the last sweep the cells of its colour have no residual, so only the
//     other colour is restricted, and only that colour takes the prolonged correction (the
//     sweep after it overwrites the rest).
//   - FP64 runs at 1.7 FMA per SM and clock here (128 in FP32), so the residual of a cycle is
//     carried in pairs of floats (about 48 bits): r -= M e with the FP64 operator split
//     likewise. The pair's error is of order 2^-46 |A| |e|, some 1e-10 of the residual it
//     starts from, so it is used once that residual is below DF_FROM |b|; before that, and
//     whenever the iteration is about to stop, r = b - M phi is evaluated in FP64, and only
//     such a residual ends the solve.
// A V-cycle on 128 x 256 cells takes 34 k cycles (18 us): the sweeps of the finest level 9 k, bound
// by shared memory, the rest latency (a colour sweep of a small level some 230 cycles). With one
// cluster barrier per sweep, the neighbours' rows read remotely and every residual in FP64 it
// took 60 us. Offsets wrap on every axis (the coupling over a closed face is zero), and the
// couplings are re-read every sweep: kept in registers they spill, and what a kernel spills
// that takes all of an SM's shared memory goes to L2.
//
// Used for 2D runs without cross terms (mg_cluster_prepare); other runs use mg.cu's kernels.
#include <cooperative_groups.h>
#include <math.h>
#include <stdlib.h>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace cpic {
namespace {

constexpr int CL_MAX_LEVELS = 16;
constexpr int CL_THREADS = 512;
constexpr int HALO = 5;        // rows of the neighbours held above and below a slab
constexpr float DF_FROM = 0.1f;
constexpr int DENSE_REGS = 8;

struct ClLevel {
    int n0, n1, half;    // global cells; half = n0 / 2
    unsigned magic;      // idx / half == __umulhi(idx, magic) for half > 1
    unsigned magic_r;    // the same for the coarse cells below this level's rows of a CTA
    int R;               // rows per CTA (split levels)
    const float* A;      // global FP32 stencil [5][ncell]
    const float* dinv;   // global FP32 inverse diagonal
    // shared-memory offsets (floats): correction, right-hand side, inverse diagonal, couplings to
    // the next cell along axis 0 and axis 1
    int ox, ob, od, oe, on;
};

struct ClParams {
    int nl;              // levels
    int nd;              // split levels (0 .. nd-1)
    int cs;              // cluster size
    int per0, per1;      // periodic axes
    int bc[4];           // field bc kinds per face (ghost rules of the prolongation)
    ClLevel L[CL_MAX_LEVELS];
    const double* A64;   // finest FP64 stencil [5][ncell]
    const double* b64;   // finest right-hand side
    double* phi;         // finest solution (in/out)
    const float* split;  // [6][ncell], colours of a row apart: FP32 diagonal, then the low words
                         // of the diagonal and of the couplings W, E, S, N
    const float* dense_inv;
    int dense_m;         // coarsest unknowns
    int singular;
    int ob1;             // second right-hand side of the finest level (ping-pong)
    int orl;             // low words of the residual [R][n0]
    int oeh, oel;        // correction since the last FP64 update of phi, as pairs [R][n0] each
    int opart;           // partial norms (doubles): [2][16][2]
    int odense;          // partial sums of the dense solve
    int ors;             // residuals of a level's first colour, own rows
    double rtol;
    float rtol2;         // its square
    int max_cycles;
    DevCounters* ctr;
};

__device__ __forceinline__ int div_half(const ClLevel& L, int idx) {
    return L.half == 1 ? idx : (int)__umulhi((unsigned)idx, L.magic);
}

// pairs of floats: s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}
// (h, l) -= (ah + al) x
__device__ __forceinline__ void pair_sub(float& h, float& l, float ah, float al, float x) {
    const float p = __fmul_rn(ah, x);
    const float pe = __fmaf_rn(al, x, __fmaf_rn(ah, x, -p));
    float e;
    two_sum(h, -p, h, e);
    l = __fadd_rn(l, __fsub_rn(e, pe));
}

// the shared memory of the CTAs whose slabs lie below and above (null outside the domain)
struct Neighbours {
    float *lower, *upper;
};

// a value at offset off of slab row rr into the halo rows of the neighbours, h rows deep (h <= R)
__device__ __forceinline__ void send(const Neighbours& X, int off, int rr, int R, int n0, int h, float v) {
    if (rr < h && X.lower) X.lower[off + R * n0] = v;
    if (rr >= R - h && X.upper) X.upper[off - R * n0] = v;
}

// Two cells next to each other along axis 0, one of each colour (cells 2 m and 2 m + 1 of a
// row): what a thread relaxes. Every neighbour of a cell is of the other colour: at index m in the
// rows below and above, and at index m (the pair's other cell) and one beside it in its own row.
// Offsets wrap on every axis: where an axis is not periodic the coupling found there is zero.
struct Pair {
    int base;            // offset of index m of the row's first colour
    int west[2], east[2];  // per colour, from index m of the other colour
    int south, north;
    unsigned sweeps;     // bit k: sweep k relaxes it; bit 4: of this CTA's own rows
};

// Rows of a leg: pairs of rows [lo, hi), of which [0, own) are this CTA's; j0: global row of row 0.
struct Leg {
    int lo, hi, own, j0;
};

template <bool SPLIT>
__device__ __forceinline__ Pair make_pair_at(const ClLevel& L, const Leg& g, int idx) {
    Pair p;
    const int r = div_half(L, idx), m = idx - r * L.half, row = g.lo + r;
    p.base = (SPLIT ? row + HALO : row) * L.n0 + m;
    p.south = !SPLIT && row == 0 ? (L.n1 - 1) * L.n0 : -L.n0;
    p.north = !SPLIT && row == L.n1 - 1 ? -(L.n1 - 1) * L.n0 : L.n0;
    const int dw = m == 0 ? L.half - 1 : -1, de = m == L.half - 1 ? 1 - L.half : 1;
    const bool odd = (g.j0 + row) & 1;  // the pair's even cell is of the second colour
    p.west[0] = odd ? 0 : dw;
    p.west[1] = odd ? dw : 0;
    p.east[0] = odd ? de : 0;
    p.east[1] = odd ? 0 : de;
    p.sweeps = 15u;
    if (SPLIT) {  // a sweep relaxes one halo row less than the one before
        const int out = row < 0 ? -row : row - g.own + 1;
        p.sweeps = out >= 4 ? 1u : out == 3 ? 3u : out == 2 ? 7u : 15u;
    }
    if (row >= 0 && row < g.own) p.sweeps = 31u;
    return p;
}

// the right-hand side minus the couplings times the neighbours, for the pair's cell of colour C
template <int C, bool SPLIT>
__device__ __forceinline__ float gather_pair(const ClLevel& L, const float* sm, int ob, const Pair& p) {
    const int own = p.base + C * L.half, oth = p.base + (1 - C) * L.half;
    const int w = oth + p.west[C], e = oth + p.east[C];
    const int s = SPLIT ? oth - L.n0 : oth + p.south, n = SPLIT ? oth + L.n0 : oth + p.north;
    float acc = sm[ob + own];
    acc -= sm[L.oe + w] * sm[L.ox + w];
    acc -= sm[L.oe + own] * sm[L.ox + e];
    acc -= sm[L.on + s] * sm[L.ox + s];
    acc -= sm[L.on + own] * sm[L.ox + n];
    return acc;
}

// The four colour sweeps of one side of a V-cycle. Down: from x = 0, then the residual of the own
// rows' first colour into rs[row * half + m] (the value the last sweep of that colour solved for
// is what its neighbours contributed then, so the residual is what they have changed by since).
// Up: colours in reverse order. NI pairs a thread.
template <int NI, bool SPLIT, bool DOWN>
__device__ __forceinline__ void leg(const ClLevel& L, float* sm, const Leg& g, int ob, float* rs) {
    const int count = (g.hi - g.lo) * L.half, h = L.half;
    Pair p[NI];
    float solved[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int idx = (int)threadIdx.x + i * CL_THREADS;
        p[i] = make_pair_at<SPLIT>(L, g, idx);
        if (idx >= count) p[i].sweeps = 0u;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int i = 0; i < NI; ++i)
            if (p[i].sweeps >> k & 1u) {
                const bool second = DOWN ? k & 1 : !(k & 1);
                const int own = p[i].base + (second ? h : 0);
                float acc;
                if (DOWN && k == 0) acc = sm[ob + own];
                else acc = second ? gather_pair<1, SPLIT>(L, sm, ob, p[i]) : gather_pair<0, SPLIT>(L, sm, ob, p[i]);
                if (DOWN && k == 2) solved[i] = acc;
                sm[L.ox + own] = acc * sm[L.od + own];
            }
        __syncthreads();
    }
    if (!DOWN) return;
#pragma unroll
    for (int i = 0; i < NI; ++i)
        if (p[i].sweeps & 16u) rs[(int)threadIdx.x + i * CL_THREADS + g.lo * h] = gather_pair<0, SPLIT>(L, sm, ob, p[i]) - solved[i];
    __syncthreads();
}

// the same for levels with more pairs than NI = 4 covers
template <bool SPLIT>
__device__ __forceinline__ void leg_large(const ClLevel& L, float* sm, const Leg& g, int ob, float* rs, bool down) {
    const int count = (g.hi - g.lo) * L.half, h = L.half;
    for (int k = 0; k < (down ? 5 : 4); ++k) {
        const bool second = down ? k & 1 : !(k & 1);
        for (int idx = threadIdx.x; idx < count; idx += CL_THREADS) {
            const Pair p = make_pair_at<SPLIT>(L, g, idx);
            if (!(p.sweeps >> k & 1u)) continue;
            const int own = p.base + (second ? h : 0);
            float acc;
            if (down && k == 0) acc = sm[ob + own];
            else acc = second ? gather_pair<1, SPLIT>(L, sm, ob, p) : gather_pair<0, SPLIT>(L, sm, ob, p);
            if (k == 4) rs[idx + g.lo * h] = acc - __fdiv_rn(sm[L.ox + own], sm[L.od + own]);
            else sm[L.ox + own] = acc * sm[L.od + own];
        }
        __syncthreads();
    }
}

template <bool SPLIT, bool DOWN>
__device__ __forceinline__ void run_leg(const ClLevel& L, float* sm, const Leg& g, int ob, float* rs) {
    const int ni = ((g.hi - g.lo) * L.half + CL_THREADS - 1) / CL_THREADS;
    if (ni <= 1) leg<1, SPLIT, DOWN>(L, sm, g, ob, rs);
    else if (ni == 2) leg<2, SPLIT, DOWN>(L, sm, g, ob, rs);
    else if (ni == 3) leg<3, SPLIT, DOWN>(L, sm, g, ob, rs);
    else if (ni == 4) leg<4, SPLIT, DOWN>(L, sm, g, ob, rs);
    else leg_large<SPLIT>(L, sm, g, ob, rs, DOWN);
}

// the offset of cell (J, I) in a level held whole: natural order on the dense level
__device__ __forceinline__ int at_whole(const ClLevel& L, bool natural, int J, int I) {
    return natural ? J * L.n0 + I : J * L.n0 + ((I + J) & 1) * L.half + (I >> 1);
}

__global__ void __launch_bounds__(CL_THREADS, 1) mg_cluster_kernel(const __grid_constant__ ClParams P) {
    extern __shared__ __align__(16) float sm[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), cs = P.cs;
    const int tid = threadIdx.x;
    __shared__ double red64[CL_THREADS];
    __shared__ float redf[CL_THREADS / 32];
    __shared__ double s_bn, s_res;  // ||b||, ||r|| / ||b||
    __shared__ float s_scale;  // 1 / ||b||
    __shared__ int s_next;  // 0: within the tolerance, 1: cycle, residual in FP64, 2: cycle, in pairs
    const ClLevel L0 = P.L[0];
    const int R0 = L0.R, j00 = rank * R0, nc0 = R0 * L0.n0, gn0 = L0.n0 * L0.n1;
    int ob_cur = L0.ob, ob_nxt = P.ob1;
    float *rl = sm + P.orl, *eh = sm + P.oeh, *el = sm + P.oel, *rs = sm + P.ors;
    double* part = reinterpret_cast<double*>(sm + P.opart);  // [2][16][2]
    float* partf = sm + P.opart + 128;                       // [2][16]
    Neighbours X;
    X.lower = rank > 0 ? cl.map_shared_rank(sm, rank - 1) : (P.per1 ? cl.map_shared_rank(sm, cs - 1) : nullptr);
    X.upper = rank < cs - 1 ? cl.map_shared_rank(sm, rank + 1) : (P.per1 ? cl.map_shared_rank(sm, 0) : nullptr);

    // ---- stage the couplings and inverse diagonals; what a sweep may read outside the domain
    // has zero couplings and a finite value
    for (int l = 0; l < P.nl - 1; ++l) {  // the dense level keeps its right-hand side and solution only
        const ClLevel L = P.L[l];
        const bool split = l < P.nd;
        const int rows = split ? L.R + 2 * HALO : L.n1, gn = L.n0 * L.n1, jb = split ? rank * L.R - HALO : 0;
#pragma unroll 4
        for (int idx = tid; idx < rows * L.n0; idx += CL_THREADS) {
            const int row = div_half(L, idx >> 1), i = idx - row * L.n0;
            int j = jb + row;
            bool inside = true;
            if (j < 0 || j >= L.n1) {
                inside = P.per1 != 0;
                j += j < 0 ? L.n1 : -L.n1;
            }
            const int at = row * L.n0 + ((i + j) & 1) * L.half + (i >> 1), g = j * L.n0 + i;
            sm[L.oe + at] = inside ? __ldg(L.A + 2 * gn + g) : 0.0f;
            sm[L.on + at] = inside ? __ldg(L.A + 4 * gn + g) : 0.0f;
            sm[L.od + at] = inside ? __ldg(L.dinv + g) : 0.0f;
            sm[L.ox + at] = 0.0f;
            sm[L.ob + at] = 0.0f;
            if (l == 0) sm[P.ob1 + at] = 0.0f;
        }
    }
    for (int e = tid; e < nc0; e += CL_THREADS) eh[e] = el[e] = 0.0f;
    // dense solve: thread w takes unknown w % m and every parts-th entry of its row from w / m on;
    // up to DENSE_REGS of them stay in registers
    const int dm = P.dense_m, dmm = dm + (P.singular ? 1 : 0);
    const int dparts = dm < CL_THREADS ? CL_THREADS / dm : 1;
    const int dp = tid / dm, di = tid - dp * dm;
    const bool dense_regs = dm <= DENSE_REGS * dparts;
    float drow[DENSE_REGS];
#pragma unroll
    for (int k = 0; k < DENSE_REGS; ++k) {
        const int c = dp + k * dparts;
        drow[k] = dense_regs && dp < dparts && c < dm ? __ldg(P.dense_inv + c * dmm + di) : 0.0f;
    }
    cl.sync();

    auto block_sum64 = [&](double v) {  // in thread 0; fixed order
        red64[tid] = v;
        __syncthreads();
        double a = 0.0;
        if (tid < 32) {
#pragma unroll 4
            for (int w = 0; w < CL_THREADS / 32; ++w) a += red64[tid + 32 * w];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        }
        __syncthreads();
        return a;
    };
    // FP64 residual of the slab's rows into the next right-hand side (and the neighbours' halos), its
    // low words, and the block's part of its norm (and of b's) into slot q of every CTA
    auto residual64 = [&](bool with_b, int q) {
        double rr = 0.0, bb = 0.0;
#pragma unroll 2
        for (int idx = tid; idx < nc0; idx += CL_THREADS) {
            const int row = div_half(L0, idx >> 1), i = idx - row * L0.n0, j = j00 + row;
            const int im = i > 0 ? i - 1 : (P.per0 ? L0.n0 - 1 : 0), ip = i + 1 < L0.n0 ? i + 1 : (P.per0 ? 0 : L0.n0 - 1);
            const int jm = j > 0 ? j - 1 : (P.per1 ? L0.n1 - 1 : 0), jp = j + 1 < L0.n1 ? j + 1 : (P.per1 ? 0 : L0.n1 - 1);
            const int g = j * L0.n0 + i;
            const double b = P.b64[g];
            double r = b - P.A64[g] * __ldcg(P.phi + g);
            r -= P.A64[gn0 + g] * __ldcg(P.phi + j * L0.n0 + im);
            r -= P.A64[2 * gn0 + g] * __ldcg(P.phi + j * L0.n0 + ip);
            r -= P.A64[3 * gn0 + g] * __ldcg(P.phi + jm * L0.n0 + i);
            r -= P.A64[4 * gn0 + g] * __ldcg(P.phi + jp * L0.n0 + i);
            const float h = (float)r;
            const int at = ((i + j) & 1) * L0.half + (i >> 1), off = ob_nxt + (row + HALO) * L0.n0 + at;
            sm[off] = h;
            send(X, off, row, R0, L0.n0, HALO - 1, h);
            rl[row * L0.n0 + at] = (float)(r - (double)h);
            rr += r * r;
            if (with_b) bb += b * b;
        }
        rr = block_sum64(rr);
        if (with_b) bb = block_sum64(bb);
        if (tid < cs) {
            double* to = cl.map_shared_rank(part, tid) + 32 * q + 2 * rank;
            to[0] = rr;
            to[1] = bb;
        }
    };

    int q = 0, cycles = 0;
    bool exact = true, pending = false;  // pending: corrections held in (eh, el)
    residual64(true, q);
    for (bool start = true;; start = false) {
        // a residual has just been written: every CTA takes the same decision from the norms
        cl.sync();
        if (tid < 32) {
            if (exact) {
                double a = tid < cs ? part[32 * q + 2 * tid] : 0.0, b = start && tid < cs ? part[32 * q + 2 * tid + 1] : 0.0;
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) {
                    a += __shfl_xor_sync(0xffffffffu, a, o);
                    if (start) b += __shfl_xor_sync(0xffffffffu, b, o);
                }
                if (tid == 0) {
                    if (start) {
                        s_bn = sqrt(b);
                        s_scale = (float)(1.0 / s_bn);
                    }
                    s_res = relative_residual(a, s_bn);
                    s_next = s_res <= P.rtol ? 0 : (s_res < (double)DF_FROM ? 2 : 1);
                }
            } else {
                float a = tid < cs ? partf[16 * q + tid] : 0.0f;
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                // (one that is not a number goes to the FP64 residual, which decides)
                if (tid == 0) s_next = !(a > P.rtol2) ? 0 : (a < DF_FROM * DF_FROM ? 2 : 1);
            }
        }
        __syncthreads();
        const int next = s_next;
        q ^= 1;
        const int swap = ob_cur;
        ob_cur = ob_nxt;
        ob_nxt = swap;
        const bool stop = next == 0 || cycles >= P.max_cycles;
        if (stop && exact) break;
        const bool cycled = !stop;
        bool to64 = true;
        if (cycled) {
            ++cycles;
            to64 = next == 1 || cycles >= P.max_cycles;
            // ---- FP32 V(2,2) cycle on the correction
            for (int l = 0; l < P.nl - 1; ++l) {
                const ClLevel L = P.L[l];
                const bool split = l < P.nd;
                Leg g;
                g.own = L.R;
                if (split) {
                    g.j0 = rank * L.R;
                    g.lo = P.per1 ? -4 : max(-4, -g.j0);
                    g.hi = P.per1 ? L.R + 4 : min(L.R + 4, L.n1 - g.j0);
                    run_leg<true, true>(L, sm, g, l == 0 ? ob_cur : L.ob, rs);
                } else {
                    g.j0 = g.lo = 0;
                    g.hi = L.R;
                    run_leg<false, true>(L, sm, g, L.ob, rs);
                }
                // restriction: the second colour was relaxed last, so only the first has a residual
                const bool csplit = l + 1 < P.nd, natural = l + 1 == P.nl - 1;
                const int cn0 = L.half, ch = cn0 / 2, ocb = P.L[l + 1].ob, CR = L.R / 2, cells = CR * cn0;
                // a level held whole below a split one goes to every CTA: the threads share that out
                const int every = split && !csplit ? cs : 1;
                const int groups = every > 1 && cells < CL_THREADS ? CL_THREADS / cells : 1;
                const int part_ = groups > 1 ? (int)__umulhi((unsigned)tid, L.magic_r) : 0;
                for (int idx = tid - part_ * cells; idx < cells && part_ < groups; idx += groups > 1 ? cells : CL_THREADS) {
                    const int jc = div_half(L, idx), ic = idx - jc * cn0;
                    const float acc = rs[2 * jc * cn0 + ic] + rs[(2 * jc + 1) * cn0 + ic];
                    const int J = g.j0 / 2 + jc;
                    const int in = natural ? ic : ((ic + J) & 1) * ch + (ic >> 1);
                    if (csplit) {
                        const int off = ocb + (jc + HALO) * cn0 + in;
                        sm[off] = acc;
                        send(X, off, jc, CR, cn0, HALO - 1, acc);
                    } else if (split) {
                        for (int c = part_; c < cs; c += groups) cl.map_shared_rank(sm, c)[ocb + J * cn0 + in] = acc;
                    } else {
                        sm[ocb + J * cn0 + in] = acc;
                    }
                }
                if (split) cl.sync();
                else __syncthreads();
            }
            {
                // dense solve (the inverse is stored transposed)
                const int ob = P.L[P.nl - 1].ob, ox = P.L[P.nl - 1].ox;
                float* ps = sm + P.odense;
                if (dense_regs) {
                    float acc = 0.0f;
#pragma unroll
                    for (int k = 0; k < DENSE_REGS; ++k) {
                        const int c = dp + k * dparts;
                        if (c < dm) acc += drow[k] * sm[ob + c];
                    }
                    if (dp < dparts) ps[tid] = acc;
                } else {
                    for (int w = tid; w < dparts * dm; w += CL_THREADS) {
                        float acc = 0.0f;
#pragma unroll 8
                        for (int k = dp; k < dm; k += dparts) acc += __ldg(P.dense_inv + k * dmm + w - dp * dm) * sm[ob + k];
                        ps[w] = acc;
                    }
                }
                __syncthreads();
                for (int i = tid; i < dm; i += CL_THREADS) {
                    float acc = ps[i];
                    for (int p = 1; p < dparts; ++p) acc += ps[p * dm + i];
                    sm[ox + i] = acc;
                }
                __syncthreads();
            }
            for (int l = P.nl - 2; l >= 0; --l) {
                const ClLevel L = P.L[l];
                const bool split = l < P.nd, csplit = l + 1 < P.nd, natural = l + 1 == P.nl - 1;
                const int j0 = split ? rank * L.R : 0, J0 = csplit ? j0 / 2 : 0;
                const int cn0 = L.half, ch = cn0 / 2, cn1 = P.L[l + 1].n1;
                // row J of the coarse correction is at xc + J * cn0 (a split level's rows are local)
                const float* xc = sm + P.L[l + 1].ox + (csplit ? (HALO - J0) * cn0 : 0);
                // prolongation onto the first colour (the next sweep overwrites the second)
#pragma unroll 2
                for (int idx = tid; idx < L.R * cn0; idx += CL_THREADS) {
                    const int rr = div_half(L, idx), m = idx - rr * cn0;
                    const int j = j0 + rr, s = 2 * (j & 1) - 1;
                    int I2 = m + s, J = j >> 1, J2 = J + s;
                    float wi = 0.1875f, wj = 0.1875f, wij = 0.0625f;  // signs: Dirichlet ghosts
                    if (I2 < 0 || I2 >= cn0) {
                        if (P.per0) I2 = I2 < 0 ? cn0 - 1 : 0;
                        else {
                            if (P.bc[I2 < 0 ? 0 : 1] == CPIC_BC_DIRICHLET) wi = -wi, wij = -wij;
                            I2 = m;
                        }
                    }
                    if (J2 < 0 || J2 >= cn1) {
                        if (!P.per1) {
                            if (P.bc[J2 < 0 ? 2 : 3] == CPIC_BC_DIRICHLET) wj = -wj, wij = -wij;
                            J2 = J;
                        } else if (!csplit) {
                            J2 = J2 < 0 ? cn1 - 1 : 0;
                        }
                    }
                    // index m or I2 of a coarse row: plain, or by the row's colours
                    const float *r1 = xc + J * cn0, *r2 = xc + J2 * cn0;
                    auto col = [&](int JJ, int I) { return natural ? I : ((I + JJ) & 1) * ch + (I >> 1); };
                    const float v = 0.5625f * r1[col(J, m)] + wi * r1[col(J, I2)] + wj * r2[col(J2, m)] + wij * r2[col(J2, I2)];
                    const int off = L.ox + (split ? rr + HALO : rr) * L.n0 + m;
                    const float xn = sm[off] + v;
                    sm[off] = xn;
                    if (split) send(X, off, rr, L.R, L.n0, HALO, xn);
                }
                Leg g;
                g.own = L.R;
                g.j0 = j0;
                if (split) {
                    cl.sync();
                    g.lo = P.per1 ? -4 : max(-4, -j0);
                    g.hi = P.per1 ? L.R + 4 : min(L.R + 4, L.n1 - j0);
                    run_leg<true, false>(L, sm, g, l == 0 ? ob_cur : L.ob, rs);
                } else {
                    __syncthreads();
                    g.lo = 0;
                    g.hi = L.R;
                    run_leg<false, false>(L, sm, g, L.ob, rs);
                }
            }
        }
        if (!to64) {
            // the correction joins those not yet in phi; the residual in pairs
            pending = true;
            float norm = 0.0f;
            const float scale = s_scale;
            const int half_rows = R0 * L0.half;
            const float *x = sm + L0.ox, *E = sm + L0.oe, *N = sm + L0.on;
#pragma unroll 2
            for (int idx = tid; idx < nc0; idx += CL_THREADS) {
                const int col = idx >= half_rows ? 1 : 0, id = idx - col * half_rows;
                const int rr = div_half(L0, id), m = id - rr * L0.half;
                const int j = j00 + rr, s = (j + col) & 1;
                const int at = rr * L0.n0 + col * L0.half + m;
                const int own = at + HALO * L0.n0, oth = (rr + HALO) * L0.n0 + (1 - col) * L0.half;
                const float* S = P.split + j * L0.n0 + col * L0.half + m;
                const float s0 = __ldg(S), s1 = __ldg(S + gn0), s2 = __ldg(S + 2 * gn0), s3 = __ldg(S + 3 * gn0),
                            s4 = __ldg(S + 4 * gn0), s5 = __ldg(S + 5 * gn0);
                const float e = x[own];
                float sh, se;
                two_sum(eh[at], e, sh, se);
                eh[at] = sh;
                el[at] += se;
                int mw = m - 1 + s, me = m + s;
                const bool west = mw >= 0 || P.per0;
                if (mw < 0) mw = P.per0 ? L0.half - 1 : 0;
                if (me == L0.half) me = P.per0 ? 0 : L0.half - 1;
                float h = sm[ob_cur + own], lo = rl[at];
                pair_sub(h, lo, s0, s1, e);
                pair_sub(h, lo, west ? E[oth + mw] : 0.0f, s2, x[oth + mw]);
                pair_sub(h, lo, E[own], s3, x[oth + me]);
                pair_sub(h, lo, N[oth - L0.n0 + m], s4, x[oth - L0.n0 + m]);
                pair_sub(h, lo, N[own], s5, x[oth + L0.n0 + m]);
                float hn, ln;
                two_sum(h, lo, hn, ln);
                sm[ob_nxt + own] = hn;
                rl[at] = ln;
                send(X, ob_nxt + own, rr, R0, L0.n0, HALO - 1, hn);
                const float u = hn * scale;
                norm = fmaf(u, u, norm);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
            if ((tid & 31) == 0) redf[tid >> 5] = norm;
            __syncthreads();
            if (tid < 32) {
                norm = tid < CL_THREADS / 32 ? redf[tid] : 0.0f;
#pragma unroll
                for (int o = CL_THREADS / 64; o > 0; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
                if (tid < cs) cl.map_shared_rank(partf, tid)[16 * q + rank] = norm;
            }
        } else {
            // phi takes the corrections, then the true residual
#pragma unroll 2
            for (int idx = tid; idx < nc0; idx += CL_THREADS) {
                const int row = div_half(L0, idx >> 1), i = idx - row * L0.n0, j = j00 + row;
                const int at = row * L0.n0 + ((i + j) & 1) * L0.half + (i >> 1), g = j * L0.n0 + i;
                double f = __ldcg(P.phi + g);
                if (cycled) f += (double)sm[L0.ox + at + HALO * L0.n0];
                if (pending) {
                    f += (double)eh[at] + (double)el[at];
                    eh[at] = el[at] = 0.0f;
                }
                P.phi[g] = f;
            }
            pending = false;
            cl.sync();
            residual64(false, q);
        }
        exact = to64;
    }
    if (rank == 0 && tid == 0) {
        P.ctr->mg_cycles = cycles;
        P.ctr->mg_residual = s_res;
        P.ctr->mg_bnorm = s_bn;
        if (s_next == 0) set_converged(P.ctr);
    }
    cl.sync();  // no CTA leaves while another may still write to its shared memory
}

// The finest level's operator for the pairs' residual, colours of a row apart: the FP32
// diagonal, and what FP32 leaves out of the diagonal and of the couplings the kernel holds (the
// coupling to the west is the western cell's own eastern one, likewise south)
__global__ void split_operator_kernel(const double* A, float* out, int n0, int n1, int per0, int per1) {
    const int n = n0 * n1;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const int j = g / n0, i = g - j * n0;
        const int at = j * n0 + ((i + j) & 1) * (n0 / 2) + (i >> 1);
        const int w = i > 0 ? g - 1 : (per0 ? g + n0 - 1 : -1), s = j > 0 ? g - n0 : (per1 ? g + (n1 - 1) * n0 : -1);
        const float d = (float)A[g];
        const float cw = w >= 0 ? (float)A[2 * n + w] : 0.0f, csn = s >= 0 ? (float)A[4 * n + s] : 0.0f;
        const float ce = (float)A[2 * n + g], cn = (float)A[4 * n + g];
        out[at] = d;
        out[n + at] = (float)(A[g] - (double)d);
        out[2 * n + at] = (float)(A[n + g] - (double)cw);
        out[3 * n + at] = (float)(A[2 * n + g] - (double)ce);
        out[4 * n + at] = (float)(A[3 * n + g] - (double)csn);
        out[5 * n + at] = (float)(A[4 * n + g] - (double)cn);
    }
}

// Which runs iterate V-cycles: 2D, no cross terms, the default multigrid components, an even
// first axis on every level, and a finest level that 16 or 8 CTAs can split into even slabs of
// at least four rows within 200 KB of eight words a cell. (Other runs take the kernel chain's
// outer iteration; the two stop at the same tolerance, but at different points below it.) Nearly
// all of them run on the cluster; where no layout of the halo slabs fits (192 x 128, 256 x 64
// and other grids long in axis 0: the halo rows outweigh the slab) the same iteration runs on
// the kernels per level: a 256 x 128 cylinder step takes 1276 us for its 30 V-cycles (1900 us in
// one cluster with slabs without halos, which fit).
bool cluster_takes(const cpic_run* r) {
    if (r->D != 2 || r->lev[0].cross || r->nlevels < 2 || r->nlevels > CL_MAX_LEVELS) return false;
    if (r->mg_coarse != CPIC_MG_COARSE_REDISCRETIZED || r->mg_smoother != CPIC_MG_SMOOTH_POINT ||
        r->mg_interp != CPIC_MG_INTERP_BILINEAR)
        return false;
    for (int l = 0; l < r->nlevels; ++l)
        if (r->lev[l].n[0] % 2) return false;
    for (int cs : {16, 8}) {
        size_t words = 0;
        int nd = 0;
        for (int l = 0; l < r->nlevels; ++l) {
            const int n0 = r->lev[l].n[0], n1 = r->lev[l].n[1];
            const bool split = l < r->nlevels - 1 && nd == l && n1 % cs == 0 && n1 / cs >= 4 && (n1 / cs) % 2 == 0;
            nd += split;
            words += 8 * (size_t)n0 * (split ? n1 / cs : n1);
        }
        words += 2 * (size_t)r->lev[0].n[0] * (r->lev[0].n[1] / cs);
        if (nd > 0 && words * sizeof(float) + 32 <= 200 * 1024) return true;
    }
    return false;
}

// Layout and launch data of the cluster solver.
struct ClusterPlan {
    size_t smem;
    double cost;
    ClParams P;
};

// an upper bound, of the 227 KB a CTA may have; mg_cluster_prepare asks the device what the kernel's
// static memory leaves
constexpr size_t CL_SMEM_MAX = 225 * 1024;

// cs CTAs with nd split levels; false where the slabs do not come out even or do not fit
bool plan_cluster(const cpic_run* r, int cs, int nd, ClusterPlan* out) {
    ClParams& P = out->P;
    P.nl = r->nlevels;
    P.nd = nd;
    P.cs = cs;
    P.per0 = r->cfg.field_bc[0] == CPIC_BC_PERIODIC;
    P.per1 = r->cfg.field_bc[2] == CPIC_BC_PERIODIC;
    for (int f = 0; f < 4; ++f) P.bc[f] = r->cfg.field_bc[f];
    size_t off = 0;  // floats
    // cycles of a V-cycle, roughly: a sweep is bound by shared memory (ten words a cell of one
    // colour) or by its latency and barrier (180), an exchange with its cluster barrier takes 850
    double cost = 0.0;
    auto take = [&](size_t words) {
        const size_t at = off;
        off += (words + 3) & ~size_t(3);
        return (int)at;
    };
    for (int l = 0; l < P.nl; ++l) {
        ClLevel& L = P.L[l];
        L.n0 = r->lev[l].n[0];
        L.n1 = r->lev[l].n[1];
        L.half = L.n0 / 2;
        L.magic = L.half > 1 ? (unsigned)(0x100000000ull / (unsigned)L.half + 1) : 0u;
        L.A = r->lev[l].A32;
        L.dinv = r->lev[l].dinv32;
        const bool split = l < nd;
        // even slabs, at least as deep as the halo so that it is the next CTA's
        if (split && (L.n1 % cs || (L.n1 / cs) % 2 || L.n1 / cs < HALO)) return false;
        L.R = split ? L.n1 / cs : L.n1;
        const unsigned below = (unsigned)(L.R / 2 * L.half);
        L.magic_r = below > 1 ? (unsigned)(0x100000000ull / below + 1) : 0u;
        if (l == P.nl - 1) {
            L.ox = take((size_t)L.n0 * L.n1);
            L.ob = take((size_t)L.n0 * L.n1);
            L.od = L.oe = L.on = 0;
            break;
        }
        const size_t nc = (size_t)L.n0 * (split ? L.R + 2 * HALO : L.n1);
        L.ox = take(nc);
        L.ob = take(nc);
        L.od = take(nc);
        L.oe = take(nc);
        L.on = take(nc);
        if (l == 0) P.ob1 = take(nc);
        const double upd = 10.0 / 32 * L.half * (split ? L.R + 4 : L.n1);
        cost += 8 * (upd > 180 ? upd : 180) + (split ? 2 * 850 : 0);
    }
    const size_t own = (size_t)P.L[0].n0 * P.L[0].R;
    cost += 0.5 * (double)own;
    P.orl = take(own);
    P.oeh = take(own);
    P.oel = take(own);
    P.opart = take(128 + 32);
    P.odense = take(CL_THREADS + r->lev[r->nlevels - 1].ncell);
    size_t most = 0;  // own pairs of a level
    for (int l = 0; l + 1 < P.nl; ++l) {
        const size_t pairs = (size_t)P.L[l].half * P.L[l].R;
        most = pairs > most ? pairs : most;
    }
    P.ors = take(most);
    out->smem = off * sizeof(float);
    out->cost = cost;
    if (out->smem > CL_SMEM_MAX) return false;
    P.A64 = r->lev[0].A;
    P.b64 = r->lev[0].b;
    P.phi = r->lev[0].x;
    P.split = reinterpret_cast<const float*>(r->kv);
    P.dense_inv = r->dense_inv32;
    P.dense_m = (int)r->lev[r->nlevels - 1].ncell;
    P.singular = r->singular ? 1 : 0;
    P.ctr = r->ctr;
    return true;
}

void cluster_config(const ClusterPlan& plan, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
    cfg->gridDim = dim3(plan.P.cs, 1, 1);
    cfg->blockDim = dim3(CL_THREADS, 1, 1);
    cfg->dynamicSmemBytes = plan.smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.P.cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
}

}  // namespace

// Decide once per run whether the cluster solver applies, and with which cluster size and
// number of split levels (the cheapest that the device can co-schedule).
int mg_cluster_prepare(cpic_run* r) {
    r->cluster_cs = 0;
    r->cluster_class = !getenv("CPIC_NO_CLUSTER_SOLVER") && cluster_takes(r);
    if (!r->cluster_class) return CPIC_OK;
    // the attributes are per function, shared by every run of the process: raise them to the
    // device's maximum once (they bound launches, they do not change occupancy)
    int dev = 0, optin = 0;
    CPIC_CUDA(cudaGetDevice(&dev));
    CPIC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    cudaFuncAttributes fa;
    CPIC_CUDA(cudaFuncGetAttributes(&fa, mg_cluster_kernel));
    const int dyn_max = optin - (int)fa.sharedSizeBytes;
    CPIC_CUDA(cudaFuncSetAttribute(mg_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max));
    if (cudaFuncSetAttribute(mg_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        cudaGetLastError();
    double best = 0.0;
    for (int cs : {1, 2, 4, 8, 16})
        for (int nd = 1; nd < r->nlevels; ++nd) {
            ClusterPlan plan;
            if (!plan_cluster(r, cs, nd, &plan)) continue;
            // (a larger cluster or another split level for less than the model can tell, 3 %, is not taken)
            if ((int)plan.smem > dyn_max || (r->cluster_cs && plan.cost >= 0.97 * best)) continue;
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[1];
            cluster_config(plan, &cfg, attr);
            int nclusters = 0;
            cudaError_t e = cudaOccupancyMaxActiveClusters(&nclusters, mg_cluster_kernel, &cfg);
            if (e != cudaSuccess || nclusters < 1) {
                cudaGetLastError();
                continue;
            }
            r->cluster_cs = cs;
            r->cluster_nd = nd;
            best = plan.cost;
        }
    if (!r->cluster_cs) {
        if (!r->done_host) {  // (set up with the map: a solve allocates nothing)
            CPIC_CUDA(cudaHostAlloc((void**)&r->done_host, 2 * sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped));
            for (int k = 0; k < 2; ++k) CPIC_CUDA(cudaEventCreateWithFlags(&r->done_event[k], cudaEventDisableTiming));
        }
        return CPIC_OK;
    }
    const long long nb = (r->ncell + 255) / 256;
    split_operator_kernel<<<(int)(nb < 1024 ? nb : 1024), 256, 0, r->stream>>>(
        r->lev[0].A, reinterpret_cast<float*>(r->kv), r->n[0], r->n[1], r->cfg.field_bc[0] == CPIC_BC_PERIODIC,
        r->cfg.field_bc[2] == CPIC_BC_PERIODIC);
    CPIC_CHECK_LAUNCH();
    return CPIC_OK;
}

// The solve loop on the cluster (right-hand side already assembled and projected).
int mg_cluster_solve(cpic_run* r, double rtol, int max_cycles) {
    ClusterPlan plan;
    if (!r->cluster_cs || !plan_cluster(r, r->cluster_cs, r->cluster_nd, &plan)) {
        set_error("cluster solver not applicable");
        return CPIC_ERR_STATE;
    }
    plan.P.rtol = rtol;
    plan.P.rtol2 = (float)(rtol * rtol);
    plan.P.max_cycles = max_cycles;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cluster_config(plan, &cfg, attr);
    cfg.stream = r->stream;
    CPIC_CUDA(cudaLaunchKernelEx(&cfg, mg_cluster_kernel, plan.P));
    CPIC_CHECK_LAUNCH();
    return CPIC_OK;
}

}  // namespace cpic
