// cvx_grid.cu -- the global-grid form of the method (Secs. 4.1-4.3, 5.1-5.3,
// 6.1, 6.8): Eq. (4.3) iterated on the cuboid deformation-gradient grid of
// Sec. 5.2 for F in R^{2x2} or R^{3x3} (four or nine components) with a set
// of grid-index directions (the reduced set R^1_1 of Eq. 5.1), the
// one-dimensional convexification of Algorithm 1 on every rank-one line of
// the grid, the lamination forest, and Algorithm 2's trees (with the
// multilinear-interpolation branching of Sec. 5.3) evaluated by Algorithm 3
// at arbitrary points.  Energies: Eq. (2.9) over Eq. (2.3) (Neo-Hooke) or
// Eq. (2.2) (St. Venant-Kirchhoff), and the double-well test energy.
//
// Design.  For a direction R every grid point lies on exactly one maximal
// line {F + l R} of the grid, and all points of one line share the line's
// lower hull: the value of Eq. (4.3) at a point is the hull read at that
// point.  So one thread builds Algorithm 1's hull of one (direction, line)
// pair once (a stack in shared memory) and then walks the line again: a
// point strictly inside a hull edge records the edge's ends and an FP32 lower
// bound of its chord value.  The per-point minimum over the directions (lowest
// direction index on equal values, a strict decrease required) is a second
// kernel over the points; it evaluates in FP64 only the directions whose bound
// says that they can win.  Predicates and chord values are the FP64
// expressions of the hull at the point with every operation rounded on its
// own (no contraction into FMA): the hull's vertex set does not depend on
// where the line is read, so each step is reproducible bit for bit.
// The global iteration stops on the device: a one-thread kernel after each
// step sets a flag once the largest decrease is at most tol, and the kernels
// of the later steps return at once, so the host enqueues kmax steps without
// waiting on the device.
#include <cuda_runtime.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "cvx_handle.h"

namespace cvx {
namespace {

constexpr int kGridMaxDirs = 4096;   // directions per call
constexpr int kGridMaxIters = 64;    // global iterations (lamination orders) per call
constexpr int kGridMaxLine = 512;    // grid points per component (longest line)
constexpr size_t kGridChunkBytes = (size_t)1 << 30;  // per-direction line results per chunk

// Bytes of line results per chunk of directions: kGridChunkBytes, or the
// environment variable CVX_GRID_CHUNK_BYTES (smaller chunks, for tests).
size_t grid_chunk_bytes() {
    const char *e = getenv("CVX_GRID_CHUNK_BYTES");
    if (e && *e) {
        const long long v = atoll(e);
        if (v > 0) return (size_t)v;
    }
    return kGridChunkBytes;
}

template <int D>
struct GridT {
    int n[D];
    int s[D];  // flat-index strides (last component fastest)
    double lo[D], delta[D];
    int N;
};

template <int D>
struct GridDirT {
    int o[D];  // grid-index offset of one step along the line
    int step;  // its flat-index step
    unsigned pos, neg;  // bit c: o[c] > 0, o[c] < 0
};

__device__ __forceinline__ bool finite_bits(double x) {
    return ((__double_as_longlong(x) >> 52) & 0x7ff) != 0x7ff;
}

// Key of a non-NaN double whose signed-integer order is the order of the
// values (-0 and +0 share the key 0): the comparisons of the hull run on the
// integer pipe and leave the FP64 pipe to the arithmetic.
__device__ __forceinline__ long long order_key(double x) {
    long long b = __double_as_longlong(x);
    if (b == (long long)0x8000000000000000ULL) b = 0;
    return b < 0 ? (b ^ 0x7fffffffffffffffLL) : b;
}

// Exact double of a nonzero integer with |v| < 2^20, assembled on the integer
// pipe from the IEEE-754 binary64 layout (sign, biased exponent, fraction).
__device__ __forceinline__ double exact_double(int v) {
    const unsigned a = (unsigned)(v < 0 ? -v : v);
    const int e = 31 - __clz(a);  // a in [2^e, 2^(e+1))
    const unsigned long long frac = ((unsigned long long)a << (52 - e)) & ((1ull << 52) - 1);
    unsigned long long bits = ((unsigned long long)(1023 + e) << 52) | frac;
    if (v < 0) bits |= 1ull << 63;
    return __longlong_as_double((long long)bits);
}

// A double truncated to FP32 on the integer pipe (relative error below
// 2^-23; magnitudes below 2^-126 give 0, above 2^127 infinity).
__device__ __forceinline__ float trunc32(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int m = (hi & 0x7fffffff) - (896 << 20);  // exponent rebiased, top 20 fraction bits
    int b = (m << 3) | (int)((unsigned)lo >> 29);
    b = m < (1 << 20) ? 0 : (m >= (254 << 20) ? 0x7f800000 : b);
    return __int_as_float(b | (hi & 0x80000000));
}

// fl(1 / v), v = 1 .. 2 kGridMaxLine (the chord denominators; the compiler's
// constant division is correctly rounded).
struct RcpTable {
    double y[2 * kGridMaxLine + 1];
    constexpr RcpTable() : y() {
        for (int v = 1; v <= 2 * kGridMaxLine; ++v) y[v] = 1.0 / v;
    }
};
__device__ const RcpTable kRcp = RcpTable();

// num / den for a positive integer den, y = fl(1 / den): the correctly rounded
// quotient in five operations.  fl(num y) is within two units in the last
// place, the first correction (residual exact by FMA) makes it faithful, and
// Markstein's theorem (a faithful quotient corrected with the correctly
// rounded reciprocal rounds correctly) the second exact.  Outside the exponent
// range where no intermediate over- or underflows: the division.
__device__ __forceinline__ double quotient(double num, int den, double y) {
    const int e = (__double2hiint(num) >> 20) & 0x7ff;
    const double b = exact_double(den);
    if (e < 128 || e > 1900) return __ddiv_rn(num, b);
    double q = __dmul_rn(num, y);
    q = __fma_rn(__fma_rn(-q, b, num), y, q);
    return __fma_rn(__fma_rn(-q, b, num), y, q);
}

template <int D>
__device__ __forceinline__ void grid_index(const GridT<D> &g, int idx, int *i) {
#pragma unroll
    for (int c = D - 1; c >= 0; --c) {
        i[c] = idx % g.n[c];
        idx /= g.n[c];
    }
}

// Grid point F_c = lo_c + i_c delta_c, each operation rounded on its own.
template <int D>
__device__ __forceinline__ void grid_point(const GridT<D> &g, int idx, double *F) {
    int i[D];
    grid_index<D>(g, idx, i);
#pragma unroll
    for (int c = 0; c < D; ++c) F[c] = __dadd_rn(g.lo[c], __dmul_rn((double)i[c], g.delta[c]));
}

// Eq. (2.9) in s = psi0: s <= beta: (1 - D(beta)) (s - beta); otherwise
// (1 - D_inf)(s - beta) + D_inf D_0 (e^{-beta/D_0} - e^{-s/D_0}); ek = e^{-beta/D_0}.
__device__ __forceinline__ double w_of_psi0(double s, double beta, double ek, const Material &m) {
    if (s <= beta) return (1.0 - m.Dinf * (1.0 - ek)) * (s - beta);
    return (1.0 - m.Dinf) * (s - beta) + m.Dinf * m.D0 * (ek - exp(-s / m.D0));
}

// Invariants of C = F^T F (Sec. 2) for F in R^{dxd}, D = d^2, row-major:
// I1 = tr C, I2 = the sum of the principal 2x2 minors of C, J = det F; d = 2
// is plane strain (C33 = 1: I1 gains 1, I2 gains C11 + C22).
// kAll false: I1 and J only.
template <int D, bool kAll>
__device__ void invariants(const double *F, double &I1, double &I2, double &J, double *C) {
    if (D == 4) {
        C[0] = F[0] * F[0] + F[2] * F[2];
        C[1] = F[0] * F[1] + F[2] * F[3];
        C[2] = C[1];
        C[3] = F[1] * F[1] + F[3] * F[3];
        I1 = C[0] + C[3] + 1.0;
        if (kAll) I2 = (C[0] * C[3] - C[1] * C[1]) + C[0] + C[3];
        J = __dsub_rn(__dmul_rn(F[0], F[3]), __dmul_rn(F[1], F[2]));
    } else {
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                C[3 * a + b] = F[a] * F[b] + F[3 + a] * F[3 + b] + F[6 + a] * F[6 + b];
        I1 = C[0] + C[4] + C[8];
        if (kAll)
            I2 = (C[0] * C[4] - C[1] * C[3]) + (C[0] * C[8] - C[2] * C[6]) +
                 (C[4] * C[8] - C[5] * C[7]);
        // each operation rounded on its own, in the oracle's order: which
        // points count as det F <= 0 must not depend on FMA contraction
        const double m0 = __dsub_rn(__dmul_rn(F[4], F[8]), __dmul_rn(F[5], F[7]));
        const double m1 = __dsub_rn(__dmul_rn(F[3], F[8]), __dmul_rn(F[5], F[6]));
        const double m2 = __dsub_rn(__dmul_rn(F[3], F[7]), __dmul_rn(F[4], F[6]));
        J = __dadd_rn(__dsub_rn(__dmul_rn(F[0], m0), __dmul_rn(F[1], m1)), __dmul_rn(F[2], m2));
    }
}

// psi0 (Eq. 2.3 with ln|J|, or Eq. 2.2) and whether det F <= 0 excludes F
// under the rule: 0 excludes det F <= 0; 1 keeps det F < 0 for Eq. (2.3)
// (ln|det F|) and every F for Eq. (2.2) (a polynomial).
template <int D>
__device__ bool psi0_grid(const double *F, const Material &m, int rule, double &s, double &J,
                          double &I1, double *C) {
    if (m.energy == CVX_ENERGY_STVK_DAMAGE) {
        double I2;
        invariants<D, true>(F, I1, I2, J, C);
        s = m.lam / 8.0 * (I1 - 3.0) * (I1 - 3.0) + m.mu / 4.0 * (I1 * I1 - 2.0 * I1 - 2.0 * I2 + 3.0);
        return rule == 0 && !(J > 0.0);
    }
    double I2;
    invariants<D, false>(F, I1, I2, J, C);
    const double aj = fabs(J);
    const double lj = log(aj);
    s = 0.5 * m.mu * (I1 - 3.0) - m.mu * lj + 0.5 * m.lam * lj * lj;
    return rule == 0 ? !(J > 0.0) : !(aj > 0.0);
}

// W, P = dW/dF and (kA) the tangent d^2W/dFdF at one F, sharing the invariants,
// one logarithm and one exponential (ek = e^{-beta/D_0}):
//   P = g dpsi0/dF, g = 1 - D(max(s, beta)), with
//   Eq. (2.3): dpsi0/dF = mu F - mu F^-T + lambda ln|J| F^-T (F^-T = cof F / J);
//   Eq. (2.2): dpsi0/dF = F S, S = lambda/2 (I1 - 3) 1 + mu (C - 1);
//   A = g d^2psi0 + g' dpsi0 (x) dpsi0, on loading (s > beta)
//   g' = -(D_inf / D_0) e^{-s / D_0}, else 0, with
//   Eq. (2.3), G = F^-T:
//     d^2psi0/dF_iJ dF_kL = mu d_ik d_JL + lambda G_iJ G_kL + (mu - lambda ln|J|) G_iL G_kJ;
//   Eq. (2.2): d_ik S_LJ + lambda F_iJ F_kL + mu F_iL F_kJ + mu (F F^T)_ik d_JL.
// A is symmetric: its upper triangle, row by row (D (D + 1) / 2 values).
template <int D, bool kA>
__device__ void grid_wpa64(const double *F, double beta, double ek, const Material &m, int rule,
                           double &W, double *P, double *A) {
    constexpr int d = D == 4 ? 2 : 3;
    if (m.energy == CVX_ENERGY_DOUBLE_WELL) {
        if (D == 4) {
            W = energy64(F, beta, m);
            stress64(F, beta, m, P);
            if (kA) {
                double T[16];
                tangent64(F, beta, m, T);
                int k = 0;
                for (int r = 0; r < 4; ++r)
                    for (int c = r; c < 4; ++c) A[k++] = T[4 * r + c];
            }
        }
        return;  // the call refuses it for D = 9
    }
    double s, J, I1, C[D];
    if (psi0_grid<D>(F, m, rule, s, J, I1, C)) {
        W = nan("");
        for (int c = 0; c < D; ++c) P[c] = nan("");
        if (kA)
            for (int c = 0; c < D * (D + 1) / 2; ++c) A[c] = nan("");
        return;
    }
    const bool load = s > beta;
    const double es = load ? exp(-s / m.D0) : ek;
    W = s <= beta ? (1.0 - m.Dinf * (1.0 - ek)) * (s - beta)
                  : (1.0 - m.Dinf) * (s - beta) + m.Dinf * m.D0 * (ek - es);
    const double g = 1.0 - m.Dinf * (1.0 - es);
    const double gp = load ? -(m.Dinf / m.D0) * es : 0.0;
    double dp[D];  // dpsi0/dF
    if (m.energy == CVX_ENERGY_STVK_DAMAGE) {
        double S[D];
        for (int a = 0; a < d; ++a)
            for (int c = 0; c < d; ++c)
                S[d * a + c] = m.mu * (C[d * a + c] - (a == c ? 1.0 : 0.0)) +
                               (a == c ? 0.5 * m.lam * (I1 - 3.0) : 0.0);
        for (int a = 0; a < d; ++a)
            for (int c = 0; c < d; ++c) {
                double v = 0.0;
                for (int k = 0; k < d; ++k) v += F[d * a + k] * S[d * k + c];
                dp[d * a + c] = v;
            }
        if (kA) {
            double FF[D];
            for (int a = 0; a < d; ++a)
                for (int c = 0; c < d; ++c) {
                    double v = 0.0;
                    for (int k = 0; k < d; ++k) v += F[d * a + k] * F[d * c + k];
                    FF[d * a + c] = v;
                }
            int n = 0;
#pragma unroll
            for (int r = 0; r < D; ++r)
#pragma unroll
                for (int q = r; q < D; ++q) {
                    const int i = r / d, jj = r % d, k = q / d, l = q % d;
                    const double d2 = (i == k ? S[d * l + jj] : 0.0) + m.lam * F[r] * F[q] +
                                      m.mu * F[d * i + l] * F[d * k + jj] +
                                      (jj == l ? m.mu * FF[d * i + k] : 0.0);
                    A[n++] = g * d2 + gp * dp[r] * dp[q];
                }
        }
    } else {
        double G[D];
        if (D == 4) {
            G[0] = F[3] / J;
            G[1] = -F[2] / J;
            G[2] = -F[1] / J;
            G[3] = F[0] / J;
        } else {
            G[0] = (F[4] * F[8] - F[5] * F[7]) / J;
            G[1] = (F[5] * F[6] - F[3] * F[8]) / J;
            G[2] = (F[3] * F[7] - F[4] * F[6]) / J;
            G[3] = (F[2] * F[7] - F[1] * F[8]) / J;
            G[4] = (F[0] * F[8] - F[2] * F[6]) / J;
            G[5] = (F[1] * F[6] - F[0] * F[7]) / J;
            G[6] = (F[1] * F[5] - F[2] * F[4]) / J;
            G[7] = (F[2] * F[3] - F[0] * F[5]) / J;
            G[8] = (F[0] * F[4] - F[1] * F[3]) / J;
        }
        const double lj = log(fabs(J));
        for (int c = 0; c < D; ++c) dp[c] = m.mu * F[c] - m.mu * G[c] + m.lam * lj * G[c];
        if (kA) {
            const double cc = m.mu - m.lam * lj;
            int n = 0;
#pragma unroll
            for (int r = 0; r < D; ++r)
#pragma unroll
                for (int q = r; q < D; ++q) {
                    const int i = r / d, jj = r % d, k = q / d, l = q % d;
                    const double d2 = (r == q ? m.mu : 0.0) + m.lam * G[r] * G[q] +
                                      cc * G[d * i + l] * G[d * k + jj];
                    A[n++] = g * d2 + gp * dp[r] * dp[q];
                }
        }
    }
    for (int c = 0; c < D; ++c) P[c] = g * dp[c];
}

// Number of grid points on the line that starts at index i along offset o.
template <int D>
__device__ __forceinline__ int line_length(const GridT<D> &g, const int *i, const int *o) {
    int len = 1 << 30;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        if (o[c] > 0) len = min(len, (g.n[c] - 1 - i[c]) / o[c]);
        else if (o[c] < 0) len = min(len, i[c] / (-o[c]));
    }
    return len + 1;
}

// W^0 on the grid.
template <int D>
__global__ void __launch_bounds__(256) k_grid_energy(GridT<D> g, Material m, double beta, int rule,
                                                     double *W) {
    __shared__ double s_ek;
    if (threadIdx.x < 32) s_ek = exp(-beta / m.D0);  // once per block: FP64 work
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.N) return;
    double F[D];
    grid_point<D>(g, p, F);
    double w = nan("");
    if (m.energy == CVX_ENERGY_DOUBLE_WELL) {
        if (D == 4) w = energy64(F, beta, m);
    } else {
        double s, J, I1, C[D];
        if (!psi0_grid<D>(F, m, rule, s, J, I1, C)) w = w_of_psi0(s, beta, s_ek, m);
    }
    W[p] = w;
}

// Lines.  The ends of a line are vertices of its hull, so a point can split
// along a direction only if both its neighbours along it lie in the grid
// ("interior" below).  In nine dimensions with three values per off-diagonal
// component that leaves 15 of the 169 directions per point on average, nearly
// all of them lines of three points, whose one chord k_grid_reduce takes
// itself there; the lines listed and walked are those of kMinLine points or
// more.
//
// The number of lines of m or more points of a direction o is
// C(m) - C(m + 1), C(m) = prod_c max(0, n_c - (m - 1) |o_c|) (the points whose
// (m - 1)-fold successor lies in the grid).
// Points of the shortest line that is listed.
template <int D>
constexpr int kMinLine = D == 4 ? 3 : 4;

template <int D>
__host__ __device__ inline long long lines_of(const GridT<D> &g, const GridDirT<D> &d, int m) {
    long long a = 1, b = 1;
    for (int c = 0; c < D; ++c) {
        const long long o = d.o[c] < 0 ? -d.o[c] : d.o[c];
        const long long x = g.n[c] - (m - 1) * o, y = x - o;
        a *= x > 0 ? x : 0;
        b *= y > 0 ? y : 0;
    }
    return a - b;
}

// cur[j][len]: where the next line of that length goes in direction j's region
// of the starts, longest lines first, so that a warp of the line kernel takes
// lines of one length.  Once k_grid_starts has placed the lines, cur[j][len]
// is the number of lines of len or more points.
template <int D>
__global__ void k_grid_cursors(GridT<D> g, const GridDirT<D> *dirs, int nd, int cap, unsigned *cur) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nd * (cap + 1)) return;
    cur[t] = (unsigned)lines_of<D>(g, dirs[t / (cap + 1)], t % (cap + 1) + 1);
}

// Line starts: per point (one index decomposition) and direction j, the point
// starts a line of kMinLine or more points if its predecessor along j lies
// outside the grid and its (kMinLine - 1)-th successor inside.  Lanes of a warp with the
// same (direction, length) share one atomic; the order among lines of one
// length is arbitrary and changes no result.  kUnit: all offsets in {-1, 0,
// 1}, where both tests are masks of the components at or next to an end of
// their axis.  The directions are staged in shared memory.
template <int D, bool kUnit>
__global__ void k_grid_starts(GridT<D> g, const GridDirT<D> *dirs, int nd,
                              const long long *line_off, unsigned *cur, int cap, int *starts) {
    extern __shared__ int soff[];  // kUnit: masks (pos, neg); else nd x D offsets
    constexpr int kPer = kUnit ? 2 : D;
    for (int k = threadIdx.x; k < nd * kPer; k += blockDim.x) {
        const GridDirT<D> &d = dirs[k / kPer];
        soff[k] = kUnit ? (int)(k & 1 ? d.neg : d.pos) : d.o[k % kPer];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (long long b = (long long)blockIdx.x * blockDim.x; b < g.N;
         b += (long long)gridDim.x * blockDim.x) {
        const long long p = b + threadIdx.x;
        const bool valid = p < g.N;
        int i[D];
        unsigned lo1 = 0, hi1 = 0, lom = 0, him = 0;  // components at / too near an end
        if (valid) {
            grid_index<D>(g, (int)p, i);
#pragma unroll
            for (int c = 0; c < D; ++c) {
                lo1 |= i[c] < 1 ? 1u << c : 0u;
                lom |= i[c] < kMinLine<D> - 1 ? 1u << c : 0u;
                hi1 |= i[c] > g.n[c] - 2 ? 1u << c : 0u;
                him |= i[c] > g.n[c] - kMinLine<D> ? 1u << c : 0u;
            }
        }
        for (int j = 0; j < nd; ++j) {
            bool st = false;
            int len = 0;
            if (kUnit) {
                const unsigned pos = (unsigned)soff[2 * j], neg = (unsigned)soff[2 * j + 1];
                st = valid && ((lo1 & pos) | (hi1 & neg)) && !((him & pos) | (lom & neg));
                if (st) {
                    len = 1 << 30;
#pragma unroll
                    for (int c = 0; c < D; ++c) {
                        if ((pos >> c) & 1) len = min(len, g.n[c] - i[c]);
                        if ((neg >> c) & 1) len = min(len, i[c] + 1);
                    }
                }
            } else if (valid) {
#pragma unroll
                for (int c = 0; c < D; ++c) {
                    const int q = i[c] - soff[j * D + c];
                    st |= (q < 0) || (q >= g.n[c]);
                }
                if (st) len = line_length<D>(g, i, soff + j * D);
                st = len >= kMinLine<D>;
            }
            const unsigned act = __ballot_sync(0xffffffffu, st);
            if (!st) continue;
            const unsigned grp = __match_any_sync(act, len);
            const int leader = __ffs(grp) - 1;
            unsigned base = 0;
            if (lane == leader)
                base = atomicAdd(cur + (size_t)j * (cap + 1) + len, (unsigned)__popc(grp));
            base = __shfl_sync(grp, base, leader);
            starts[line_off[j] + base + __popc(grp & ((1u << lane) - 1))] = (int)p;
        }
    }
}

// One thread per (direction, line of kMinLine or more points) of directions
// [j0, j1): Algorithm 1 on the finite values of W_in along the line (stack in
// shared memory, layout [slot][thread]), then every interior point of the
// line reads the hull there:
//   a hull vertex keeps its own value (no split): H = inf;
//   a point strictly between vertices a < x < b, with x_a, x_b taken relative
//   to the point (x_a < 0 < x_b), records the pair (x_a, x_b) as two 16-bit
//   fields in S and in H a lower bound, in FP32, of its chord value
//   h = (x_b w_a - x_a w_b) / (x_b - x_a); k_grid_reduce evaluates h in FP64
//   where it can win.
// Non-finite points keep their value.  H and S are chunk-major: entry
// (j - j0) N + point.
//
// The FP64 pipe has 2 lanes per SM and clock, so FP64 is left to what decides:
// a comparison takes FP32 values (truncated from the bits on the integer
// pipe), and FP64 where those are within their error.  Each predicate has the
// value of the FP64 one with every operation rounded on its own.  The stack
// holds abscissae only; its values are read again from W_in.
// (All lines of one or more points, both differences and products in FP64,
// FP64 chord numerators of every point and direction read back by the
// reduction: the 648,025-point study took 167 us per step here and 68 us in
// the reduction, the nine-dimensional one 13.7 and 2.0 ms; now 103 and 42 us,
// 0.10 and 0.90 ms.  A loop that pops or pushes once per turn took 121 us, and
// values kept in the stack 113 us at a third of the resident warps.)
template <int D>
__global__ void __launch_bounds__(128) k_grid_lines(GridT<D> g, const GridDirT<D> *dirs,
                                                    const long long *line_off, int j0, int j1,
                                                    const int *starts, const unsigned *cur,
                                                    const double *Win, float *H, unsigned *S,
                                                    int cap, const int *done) {
    if (done && *done) return;
    extern __shared__ short gsm[];
    const int T = blockDim.x, lane = threadIdx.x & 31;
    const long long end = line_off[j1];
    const long long t0 = line_off[j0] + (long long)blockIdx.x * T + (threadIdx.x & ~31), t = t0 + lane;
    if (t0 >= end) return;  // whole warps only: the search below is warp-wide
    // the direction of the warp's first line, and that line's length: the
    // largest with more than its rank of lines
    int j = j0;
    for (int b = j0 + 1; b < j1; b += 32)
        j += __popc(__ballot_sync(0xffffffffu, b + lane < j1 && line_off[b + lane] <= t0));
    const unsigned rank0 = (unsigned)(t0 - line_off[j]);
    int len = kMinLine<D> - 1;
    for (int b = kMinLine<D>; b <= cap; b += 32) {
        const unsigned m = __ballot_sync(0xffffffffu, b + lane <= cap &&
                                                          cur[(size_t)j * (cap + 1) + b + lane] > rank0);
        len += __popc(m);
        if (m != 0xffffffffu) break;
    }
    if (t >= end) return;
    while (t >= line_off[j + 1]) {  // later lines of the warp: next directions ...
        ++j;
        len = cap;
    }
    {  // ... and shorter lines
        const unsigned *cj = cur + (size_t)j * (cap + 1), rank = (unsigned)(t - line_off[j]);
        while (cj[len] <= rank) --len;
    }
    const int step = dirs[j].step;
    const int p0 = starts[t];
    const double *src = Win + p0;
    const long long base = (long long)(j - j0) * g.N + p0;
    short *sx = gsm + threadIdx.x;

    // Algorithm 1: monotone chain over the finite values, pops while the top
    // of the stack is not strictly below the chord to the new point.  The two
    // top vertices p, q are kept in registers, their values also in FP32 (P, Q).
    int k = 0, xp = 0, xq = 0;
    double wp = 0.0, wq = 0.0;
    float P = 0.0f, Q = 0.0f;
    bool holes = false;
    double wn = src[0];
    for (int l = 0; l < len; ++l) {
        const double w = wn;
        if (l + 1 < len) wn = src[(long long)(l + 1) * step];
        if (!finite_bits(w)) {
            holes = true;
            continue;
        }
        const float V = trunc32(w);
        while (k >= 2) {
            // (w_q - w_p)(x - x_q) >= (w - w_q)(x_q - x_p)?  The FP32 values
            // decide where their error (2^-23 of each value) allows
            const int di = l - xq, dp = xq - xp;
            const float fi = (float)di, fp = (float)dp;
            const float d = (Q - P) * fi - (V - Q) * fp;
            const float mag = fabsf(P) + fabsf(Q) + fabsf(V);
            bool pop;
            if (fabsf(d) > 4e-7f * mag * (fi + fp) && mag < 1e30f && mag > 1e-20f) {
                pop = d > 0.0f;
            } else {
                const double A = __dsub_rn(wq, wp), B = __dsub_rn(w, wq);
                // multiplying by 1 is exact
                const double lhs = di == 1 ? A : __dmul_rn(A, exact_double(di));
                const double rhs = dp == 1 ? B : __dmul_rn(B, exact_double(dp));
                pop = order_key(lhs) >= order_key(rhs);
            }
            if (!pop) break;
            --k;
            wq = wp;
            xq = xp;
            Q = P;
            if (k >= 2) {
                xp = sx[(k - 2) * T];
                wp = src[(long long)xp * step];
                P = trunc32(wp);
            }
        }
        wp = wq;
        xp = xq;
        P = Q;
        wq = w;
        xq = l;
        Q = V;
        sx[k * T] = (short)l;
        ++k;
    }
    // every finite point lies between the first and the last vertex
    int e = -1, xa = 0, xb = -1;  // the current edge
    float fa = 0.0f, slope = 0.0f, off = 0.0f;
    for (int l = 1; l < len - 1; ++l) {
        while (l >= xb && e + 2 < k) {
            ++e;
            xa = sx[e * T];
            xb = sx[(e + 1) * T];
            fa = trunc32(src[(long long)xa * step]);
            const float fb = trunc32(src[(long long)xb * step]);
            // the bound covers the truncation of both ends and the rounding of
            // the chord; ends outside FP32's range leave it to the FP64 value
            off = 1e-6f * (fabsf(fa) + fabsf(fb)) + 1e-36f;
            slope = __fdividef(fb - fa, (float)(xb - xa));
            if (!(off < 1e30f)) {
                fa = -INFINITY;
                slope = off = 0.0f;
            }
        }
        const long long at = base + (long long)l * step;
        float h = INFINITY;
        // strictly inside the edge (and finite: a non-finite point is no
        // vertex, but a hole can lie inside an edge)
        if (xa < l && l < xb && (!holes || finite_bits(src[(long long)l * step]))) {
            h = __fmaf_rn(slope, (float)(l - xa), fa) - off;
            S[at] = ((unsigned)(xa - l) & 0xffffu) | ((unsigned)(xb - l) << 16);
        }
        H[at] = h;
    }
}

constexpr int kGridChunkDirs = 64;  // directions per chunk at most (a mask word in the reduction)

// For offsets in {-1, 0, 1}: the directions of a chunk along which a point is
// interior depend only on which components lie at an end of their axis; per
// chunk and pattern of components, their mask (nine dimensions: most points
// are interior along few directions, and testing each cost more than the
// rest).
template <int D>
__global__ void k_grid_patterns(const GridDirT<D> *dirs, int nd, int chunk, unsigned long long *pat) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, j0 = (t >> D) * chunk;
    if (j0 >= nd) return;
    unsigned long long m = 0;
    for (int q = 0; q < chunk && j0 + q < nd; ++q)
        if (!((t & ((1 << D) - 1)) & (dirs[j0 + q].pos | dirs[j0 + q].neg))) m |= 1ull << q;
    pat[t] = m;
}

// Per point, directions [j0, j1): the smallest chord value h below the best so
// far wins, the lowest direction on equal values (first chunk: the best so far
// is W_in itself, no split).  The FP32 lower bounds of the interior
// directions are read, the direction with the smallest one is evaluated in
// FP64, then those whose bound does not exceed its value: every lane its own
// next one, so that a warp evaluates as often as its busiest lane needs (once
// or twice), not once per direction.  lam = (dir, l-, l+) per point (dir =
// -1: no split).  The last chunk adds the point's decrease W_in - W_out to
// the step's maximum (dec, as the bits of a non-negative double).
template <int D, bool kUnit>
__global__ void __launch_bounds__(256) k_grid_reduce(GridT<D> g, const GridDirT<D> *dirs, int j0,
                                                     int j1, int first, int last, const double *Win,
                                                     const float *H, const unsigned *S,
                                                     const unsigned long long *pat, double *Wout,
                                                     int *lam, unsigned long long *dec,
                                                     const int *done) {
    if (done && *done) return;
    constexpr bool kPat = kUnit && D == 9;
    __shared__ GridDirT<D> s_d[kGridChunkDirs];
    __shared__ unsigned s_nz[kGridChunkDirs];  // components that the direction moves
    const int n = j1 - j0;
    for (int k = threadIdx.x; k < n * (int)(sizeof(GridDirT<D>) / 4); k += blockDim.x)
        reinterpret_cast<int *>(s_d)[k] = reinterpret_cast<const int *>(dirs + j0)[k];
    if (threadIdx.x < n) s_nz[threadIdx.x] = dirs[j0 + threadIdx.x].pos | dirs[j0 + threadIdx.x].neg;
    __syncthreads();
    const long long N = g.N, p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long dbits = 0;
    if (p < N) {
        const double w0 = Win[p];
        double best = w0;
        int bd = -1, bm = 0, bp = 0;
        if (!first) {
            best = Wout[p];
            bd = lam[3 * p];
            bm = lam[3 * p + 1];
            bp = lam[3 * p + 2];
        }
        int i[D], mg[D];  // grid points between the point and the nearer end of each axis
        unsigned edge = 0, lo2 = 0, hi2 = 0;  // components at an end, within one of an end
        grid_index<D>(g, (int)p, i);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            mg[c] = min(i[c], g.n[c] - 1 - i[c]);
            edge |= mg[c] < 1 ? 1u << c : 0u;
            lo2 |= i[c] < 2 ? 1u << c : 0u;
            hi2 |= i[c] > g.n[c] - 3 ? 1u << c : 0u;
        }
        auto interior = [&](int q) {
            if (kUnit) return !(edge & s_nz[q]);
            bool in = true;
#pragma unroll
            for (int c = 0; c < D; ++c) in = in && mg[c] >= abs(s_d[q].o[c]);
            return in;
        };
        // an interior point's line has three points: neither second neighbour
        // lies in the grid
        auto three = [&](int q) {
            if (kMinLine<D> == 3) return false;  // listed
            const GridDirT<D> &d = s_d[q];
            if (kUnit) return ((hi2 & d.pos) | (lo2 & d.neg)) && ((lo2 & d.pos) | (hi2 & d.neg));
            bool fwd = true, back = true;
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const int a = i[c] + 2 * d.o[c], b = i[c] - 2 * d.o[c];
                fwd = fwd && a >= 0 && a < g.n[c];
                back = back && b >= 0 && b < g.n[c];
            }
            return !fwd && !back;
        };
        // FP32 lower bound of the chord value of interior direction j0 + q, inf
        // if the point is a vertex of the line's hull
        const float f0 = trunc32(w0);
        auto lower = [&](int q) {
            if (!three(q)) return H[q * N + p];
            // Algorithm 1 on three points: the centre is popped unless it lies
            // strictly below the chord of its neighbours
            const int st = s_d[q].step;
            const double wa = Win[p - st], wb = Win[p + st];
            if (!finite_bits(wa) || !finite_bits(wb)) return INFINITY;
            const float fa = trunc32(wa), fb = trunc32(wb), a = fabsf(fa) + fabsf(fb);
            const float d = (f0 - fa) - (fb - f0), mag = a + fabsf(f0);
            bool in;
            if (fabsf(d) > 1e-6f * mag && mag < 1e30f && mag > 1e-20f) in = d > 0.0f;
            else in = order_key(__dsub_rn(w0, wa)) >= order_key(__dsub_rn(wb, w0));
            if (!in) return INFINITY;
            return a < 1e30f ? 0.5f * (fa + fb) - (1e-6f * a + 1e-36f) : -INFINITY;
        };
        // the exact chord value of direction j0 + q
        auto exact = [&](int q) {
            int ra = -1, rb = 1;
            const int st = s_d[q].step;
            double h;
            if (three(q)) {
                h = __dmul_rn(0.5, __dadd_rn(Win[p + st], Win[p - st]));
            } else {
                const unsigned sp = S[q * N + p];
                ra = (int)(short)(sp & 0xffffu);
                rb = (int)(sp >> 16);
                const double wa = Win[p + (long long)ra * st], wb = Win[p + (long long)rb * st];
                const double num = __dsub_rn(__dmul_rn(exact_double(rb), wa),
                                             __dmul_rn(exact_double(ra), wb));
                h = quotient(num, rb - ra, kRcp.y[rb - ra]);
            }
            const long long kh = order_key(h), kb = order_key(best);
            if (kh < kb || (kh == kb && j0 + q < bd)) {
                best = h;
                bd = j0 + q;
                bm = ra;
                bp = rb;
            }
        };
        if (finite_bits(w0)) {
            float m1 = INFINITY, m2 = INFINITY;  // the two smallest bounds
            int q1 = 0;
            auto see = [&](int q) {
                const float h = lower(q);
                m2 = fminf(m2, fmaxf(m1, h));
                if (h < m1) {
                    m1 = h;
                    q1 = q;
                }
            };
            unsigned long long in = 0;
            if (kPat) {
                in = pat[edge];
                for (unsigned long long m = in; m; m &= m - 1) see(__ffsll((long long)m) - 1);
            } else {
#pragma unroll 4
                for (int q = 0; q < n; ++q)
                    if (interior(q)) see(q);
            }
            if (m1 < INFINITY && m1 <= __double2float_ru(best)) exact(q1);
            float lim = __double2float_ru(best);
            unsigned long long more = 0;
            if (m2 < INFINITY && m2 <= lim) {
                auto again = [&](int q) {
                    const float h = lower(q);
                    if (q != q1 && h < INFINITY && h <= lim) more |= 1ull << q;
                };
                if (kPat) {
                    for (unsigned long long m = in; m; m &= m - 1) again(__ffsll((long long)m) - 1);
                } else {
                    for (int q = 0; q < n; ++q)
                        if (interior(q)) again(q);
                }
            }
            for (; more; more &= more - 1) exact(__ffsll((long long)more) - 1);
        }
        Wout[p] = best;
        lam[3 * p] = bd;
        lam[3 * p + 1] = bm;
        lam[3 * p + 2] = bp;
        if (last && finite_bits(w0) && finite_bits(best))
            dbits = (unsigned long long)__double_as_longlong(__dsub_rn(w0, best));
    }
    if (!last || !dec) return;
    // non-negative doubles order like their bit patterns: reduce on the integer pipe
    for (int o = 16; o; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, dbits, o);
        dbits = v > dbits ? v : dbits;
    }
    if ((threadIdx.x & 31) == 0 && dbits) atomicMax(dec, dbits);
}

// After step k: the step count so far, and the stop flag once the step's
// largest decrease is at most tol (Sec. 4.1's stopping rule).
__global__ void k_grid_check(const unsigned long long *dec_k, double tol, int *done, int *iters,
                             int k) {
    if (*done) return;
    *iters = k + 1;
    if (__longlong_as_double((long long)*dec_k) <= tol) *done = 1;
}

// W^K ends in the ping buffer when K is odd: copy it to the output.
__global__ void k_grid_final(int N, const int *iters, const double *pong, double *W) {
    if ((*iters & 1) == 0) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) W[p] = pong[p];
}

// Trees of Algorithm 2 tabulated per grid point and order (Algorithm 3 by
// dynamic programming over the orders).  T_d(p) = (W, P, A, leaves) of the
// tree below grid point p at order d: at d = 0 (or where no iteration up to d
// split p) the leaf values W(p), P(p) (Eq. 2.12), A(p) and one leaf; where
// iteration d split p with record (dir, l-, l+), xi = -l- / (l+ - l-),
//   T_d(p) = (1 - xi) T_{d-1}(p + l- R) + xi T_{d-1}(p + l+ R);
// elsewhere T_d(p) = T_{d-1}(p) (the latest split below d decides).  A record
// this library did not write makes p a leaf at that order.
//
// Layout: one record per point, W, P, the upper triangle of A, leaves (int64)
// -- 16 words of 8 bytes for D = 4 with the tangent -- in two buffers; a flag
// per point says which buffer holds its latest record.  An order writes the
// records of the points it split into their other buffer, so that the old
// ones stay readable, and only copies the flags of the rest.  A group of
// lanes takes a point or a query, a lane per word, so that a record is read
// and written in whole sectors.  (Values in separate arrays, copied whole per
// order, and A accumulated in global memory by one thread per query: 648,025
// points, 15 orders, 1,048,576 queries with the tangent took 0.85 + 1.43 +
// 6.46 ms; this takes 0.33 + 0.53 + 0.95 ms.)
template <int D, bool kA>
struct TreeRec {
    static constexpr int kTri = D * (D + 1) / 2;
    static constexpr int kLeaf = 1 + D + (kA ? kTri : 0);  // the word of the leaf count
    static constexpr int kWords = D == 4 ? (kA ? 16 : 8) : (kA ? 56 : 12);
    static constexpr int kLanes = D == 4 ? kWords : (kA ? 32 : 16);
    static_assert(kLeaf < kWords, "record layout");
};

template <int D, bool kA>
__device__ void leaf_record(const GridT<D> &g, int p, const Material &m, double beta, double ek,
                            int rule, double *r) {
    using R = TreeRec<D, kA>;
    double F[D], P[D], A[kA ? R::kTri : 1], W;
    grid_point<D>(g, p, F);
    grid_wpa64<D, kA>(F, beta, ek, m, rule, W, P, A);
    r[0] = W;
#pragma unroll
    for (int c = 0; c < D; ++c) r[1 + c] = P[c];
    if (kA)
#pragma unroll
        for (int c = 0; c < R::kTri; ++c) r[1 + D + c] = A[c];
    r[R::kLeaf] = __longlong_as_double(1ll);
#pragma unroll
    for (int c = R::kLeaf + 1; c < R::kWords; ++c) r[c] = 0.0;
}

constexpr int kTreeThreads = 64;

template <int D, bool kA>
__global__ void __launch_bounds__(kTreeThreads) k_grid_tree0(GridT<D> g, Material m, double beta,
                                                             int rule, double *T,
                                                             unsigned char *flag) {
    using R = TreeRec<D, kA>;
    constexpr int kPitch = R::kWords + 1;  // odd: no bank conflicts in the transposition
    __shared__ double s_r[kTreeThreads * kPitch];
    const int p0 = blockIdx.x * kTreeThreads, p = p0 + threadIdx.x;
    const double ek = exp(-beta / m.D0);
    if (p < g.N) {
        leaf_record<D, kA>(g, p, m, beta, ek, rule, s_r + threadIdx.x * kPitch);
        flag[p] = 0;
    }
    __syncthreads();
    const int n = min(kTreeThreads, g.N - p0) * R::kWords;
    double *out = T + (size_t)p0 * R::kWords;
    for (int i = threadIdx.x; i < n; i += kTreeThreads)
        out[i] = s_r[i / R::kWords * kPitch + i % R::kWords];
}

constexpr int kStepThreads = 256;

// One order: a thread per point reads the iteration's record (and divides),
// then groups of lanes, a lane per word, combine the records of the points it
// split.
template <int D, bool kA>
__global__ void __launch_bounds__(kStepThreads)
    k_grid_tree_step(GridT<D> g, const GridDirT<D> *dirs, int nd, const int *rec, Material m,
                     double beta, int rule, double *T0, double *T1, const unsigned char *flag,
                     unsigned char *flag_out) {
    using R = TreeRec<D, kA>;
    __shared__ double s_xi[kStepThreads];
    __shared__ int s_c[kStepThreads][2];            // the children's points
    __shared__ unsigned short s_p[kStepThreads];    // thread | buffers of F-, F+ and the output << 8
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int p0 = blockIdx.x * kStepThreads;
    const long long p = (long long)p0 + threadIdx.x;
    if (p < g.N) {
        const int dj = rec[3 * p];
        int f = flag[p];
        if (dj >= 0) {
            const int lm = rec[3 * p + 1], lp = rec[3 * p + 2];
            const int step = dj < nd ? dirs[dj].step : 0;
            const long long cm = p + (long long)lm * step, cp = p + (long long)lp * step;
            if (dj >= nd || !(lm < 0 && lp > 0) || cm < 0 || cm >= g.N || cp < 0 || cp >= g.N) {
                leaf_record<D, kA>(g, (int)p, m, beta, exp(-beta / m.D0), rule,
                                   (f ? T0 : T1) + (size_t)p * R::kWords);
            } else {
                const int i = atomicAdd(&s_n, 1);
                s_xi[i] = __ddiv_rn((double)(-lm), (double)(lp - lm));
                s_c[i][0] = (int)cm;
                s_c[i][1] = (int)cp;
                s_p[i] = (unsigned short)(threadIdx.x | (flag[cm] << 8) | (flag[cp] << 9) |
                                          ((1 - f) << 10));
            }
            f = 1 - f;
        }
        flag_out[p] = (unsigned char)f;  // not split: the tree of the order below
    }
    __syncthreads();
    const int v = threadIdx.x % R::kLanes;
    for (int i = threadIdx.x / R::kLanes; i < s_n; i += kStepThreads / R::kLanes) {
        const double xi = s_xi[i], xm = __dsub_rn(1.0, xi);
        const unsigned sp = s_p[i];
        const double *Tm = (sp & 0x100 ? T1 : T0) + (size_t)s_c[i][0] * R::kWords;
        const double *Tp = (sp & 0x200 ? T1 : T0) + (size_t)s_c[i][1] * R::kWords;
        double *out = (sp & 0x400 ? T1 : T0) + (size_t)(p0 + (int)(sp & 0xff)) * R::kWords;
#pragma unroll
        for (int w = v; w < R::kWords; w += R::kLanes) {
            const double a = Tm[w], b = Tp[w];
            double r = __dadd_rn(__dmul_rn(xm, a), __dmul_rn(xi, b));
            if (w == R::kLeaf) {
                const long long la = __double_as_longlong(a), l = la + __double_as_longlong(b);
                r = __longlong_as_double(l < la ? 0x7fffffffffffffffLL : l);  // saturates
            }
            out[w] = r;
        }
    }
}

// Algorithm 2's tree at n points evaluated by Algorithm 3: the corners of the
// grid cell holding F (multilinear weights prod_c (1 - t_c or t_c); a
// coordinate within 1e-12 grid steps of a grid value counts as on it; corners
// of weight 0 left out; corner bit c counted from the first component) at
// order K, each contributing its weight times the tabulated tree T_K.
// W_interp is the multilinear interpolation of W^K.  A thread per query finds
// the cell and W_interp, then a group of lanes per query sums the records, a
// lane per word, each lane having computed the weight of one corner per turn.
// What bounds it at many queries is the FP64 pipe (2 lanes per SM and clock): a
// sum per corner, word and query, the weights, and the division and tests of
// the cell.  In nine dimensions (512 corners) the weights' products are shared:
// those of the first five components by 16 corners for W_interp, those of a
// turn by its lanes; the order of the factors is the same everywhere.
// 300,000 queries on 46,656 points, d = 3: 11.2 -> 8.3 ms, with the tangent
// 24.4 -> 21.8 ms.
constexpr int kQueryThreads = 128;

template <int D, bool kA>
__global__ void __launch_bounds__(kQueryThreads)
    k_grid_query(GridT<D> g, const double *WK, const double *T0, const double *T1,
                 const unsigned char *flag, long long n, int per, const double *F, double *Wi,
                 double *Wt, double *P, double *A, long long *leaves) {
    using R = TreeRec<D, kA>;
    constexpr int kG = R::kLanes, kC = 1 << D, kPer = (R::kWords + kG - 1) / kG;
    // a group takes kG corners per turn: the turn's number holds the bits of the
    // first kHead components, the lane's place those of the others
    constexpr int kTurns = kC / kG, kHead = __builtin_ctz(kTurns);
    constexpr int kHeads = (kTurns + kG - 1) / kG;  // turns whose head products a lane computes
    __shared__ double s_t[kQueryThreads][2 * D];  // 1 - t_c and t_c
    __shared__ int s_flat[kQueryThreads];  // flat index of the cell's first corner, -1 outside
    __shared__ int s_in[kQueryThreads];    // bit c: the cell has an upper corner in component c
    const long long q0 = (long long)blockIdx.x * per;
    if (threadIdx.x < per) {
        const long long q = q0 + threadIdx.x;
        bool inside = q < n;
        double t[D];
        int flat0 = 0, in = 0;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const double u =
                inside ? __ddiv_rn(__dsub_rn(F[D * q + c], g.lo[c]), g.delta[c]) : -1.0;
            if (u < -1e-12 || u > (double)(g.n[c] - 1) + 1e-12) inside = false;
            double f = floor(u);
            double r = __dsub_rn(u, f);
            if (r > 1.0 - 1e-12) {
                f = __dadd_rn(f, 1.0);
                r = 0.0;
            } else if (r < 1e-12) {
                r = 0.0;
            }
            int ii = (int)f;
            ii = ii > g.n[c] - 1 ? g.n[c] - 1 : ii;
            ii = ii < 0 ? 0 : ii;
            flat0 += ii * g.s[c];
            in |= (ii < g.n[c] - 1 ? 1 : 0) << c;
            t[c] = r;
            s_t[threadIdx.x][2 * c] = __dsub_rn(1.0, r);
            s_t[threadIdx.x][2 * c + 1] = r;
        }
        s_flat[threadIdx.x] = inside ? flat0 : -1;
        s_in[threadIdx.x] = in;
        if (q < n) {
            double wi = inside ? 0.0 : nan("");
            if (inside) {
                // corners in order; the products of the first D - 4 components
                // are shared by 16 corners
#pragma unroll 1
                for (int head = 0; head < 1 << (D - 4); ++head) {
                    double p = 1.0;
                    int off = flat0;
#pragma unroll
                    for (int c = 0; c < D - 4; ++c) {
                        const int up = (head >> (D - 5 - c)) & 1;
                        const double x = s_t[threadIdx.x][2 * c + up];
                        p = c == 0 ? x : __dmul_rn(p, x);
                        off += (up & (in >> c)) * g.s[c];
                    }
#pragma unroll
                    for (int corner = 0; corner < 16; ++corner) {
                        double w = p;
                        int flat = off;
#pragma unroll
                        for (int c = D - 4; c < D; ++c) {
                            const int up = (corner >> (D - 1 - c)) & 1;
                            const double x = up ? t[c] : __dsub_rn(1.0, t[c]);
                            w = c == 0 ? x : __dmul_rn(w, x);
                            flat += (up & (in >> c)) * g.s[c];
                        }
                        if (w == 0.0) continue;
                        wi = __dadd_rn(wi, __dmul_rn(w, WK[flat]));
                    }
                }
            }
            Wi[q] = wi;
        }
    }
    __syncthreads();
    const int v = threadIdx.x % kG, grp = threadIdx.x / kG;
    const unsigned lane0 = (threadIdx.x & 31) / kG * kG;  // the group's first lane
    const unsigned gm = (kG == 32 ? 0xffffffffu : ((1u << (kG & 31)) - 1u) << lane0);
    int at0[kPer], at1[kPer];  // places of the lane's words of A in a query's 4 x 4 or 9 x 9
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        int e = v + j * kG - 1 - D, r = 0;  // upper triangle, row r from (r, r)
        while (r < D && e >= D - r) {
            e -= D - r;
            ++r;
        }
        at0[j] = D * r + r + e;
        at1[j] = D * (r + e) + r;
    }
    for (int i = grp; i < per && q0 + i < n; i += kQueryThreads / kG) {
        const long long q = q0 + i;
        const int flat0 = s_flat[i], in = s_in[i];
        double acc[kPer];
        long long nl = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) acc[k] = 0.0;
        if (flat0 >= 0) {
            // head products of turns v, v + kG, ... and this lane's own factors
            double hw[kHeads], x[D];
            int ho[kHeads], lo = flat0;
#pragma unroll
            for (int h = 0; h < kHeads; ++h) {
                hw[h] = 1.0;
                ho[h] = 0;
#pragma unroll
                for (int c = 0; c < kHead; ++c) {
                    const int up = ((h * kG + v) >> (kHead - 1 - c)) & 1;
                    const double y = s_t[i][2 * c + up];
                    hw[h] = c == 0 ? y : __dmul_rn(hw[h], y);
                    ho[h] += (up & (in >> c)) * g.s[c];
                }
            }
#pragma unroll
            for (int c = kHead; c < D; ++c) {
                const int up = (v >> (D - 1 - c)) & 1;
                x[c] = s_t[i][2 * c + up];
                lo += (up & (in >> c)) * g.s[c];
            }
#pragma unroll
            for (int h = 0; h < kHeads; ++h)
#pragma unroll 1
                for (int t = 0; t < kG && h * kG + t < kTurns; ++t) {
                    // this lane's corner: weight and record
                    double w = kHead ? __shfl_sync(gm, hw[h], t, kG) : 1.0;
#pragma unroll
                    for (int c = kHead; c < D; ++c) w = c == 0 ? x[0] : __dmul_rn(w, x[c]);
                    const int flat = lo + (kHead ? __shfl_sync(gm, ho[h], t, kG) : 0);
                    // the record's place, its buffer (bit 62), and -1 for a corner of
                    // weight 0, which is not read (tested on the bits: comparing in
                    // FP64 would cost as much as the sums)
                    long long at = -1;
                    if ((__double_as_longlong(w) << 1) != 0)
                        at = (long long)flat * R::kWords | (flag[flat] ? 1ll << 62 : 0);
#pragma unroll(D == 4 ? kG : 4)
                    for (int k = 0; k < kG; ++k) {
                        const double wk = __shfl_sync(gm, w, k, kG);
                        const long long ak = __shfl_sync(gm, at, k, kG);
                        const double *r = ((ak >> 62) ? T1 : T0) + (ak & ((1ll << 62) - 1));
#pragma unroll
                        for (int j = 0; j < kPer; ++j) {
                            const int e = v + j * kG;
                            double val = 0.0;  // (a corner of weight 0 is not read)
                            if (ak >= 0 && e < R::kWords) val = r[e];
                            acc[j] = __fma_rn(wk, val, acc[j]);
                            if (e == R::kLeaf) nl += __double_as_longlong(val);
                        }
                    }
                }
        } else {
#pragma unroll
            for (int k = 0; k < kPer; ++k) acc[k] = nan("");
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int x = v + j * kG;
            if (x == 0) Wt[q] = acc[j];
            else if (x <= D) P[D * q + x - 1] = acc[j];
            else if (x == R::kLeaf) {
                if (leaves) leaves[q] = nl;
            } else if (kA && x < R::kLeaf) {
                A[(long long)D * D * q + at0[j]] = acc[j];
                A[(long long)D * D * q + at1[j]] = acc[j];
            }
        }
    }
}

// ------------------------------------------------------------------ host

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

template <int D>
int check_grid(const cvx_grid *g, GridT<D> &gd) {
    long long N = 1;
    for (int c = 0; c < D; ++c) {
        if (g->n[c] < 1 || g->n[c] > kGridMaxLine)
            return fail(CVX_ERR_INVALID_ARG, "grid points per component must be in [1, %d]",
                        kGridMaxLine);
        if (!(g->delta[c] > 0.0) || !isfinite(g->delta[c]) || !isfinite(g->lo[c]))
            return fail(CVX_ERR_INVALID_ARG, "grid spacing must be positive and bounds finite");
        N *= g->n[c];
        if (N > 0x7fffffffLL)
            return fail(CVX_ERR_INVALID_ARG, "grid has more than 2^31 - 1 points");
    }
    for (int c = 0; c < D; ++c) {
        gd.n[c] = g->n[c];
        gd.lo[c] = g->lo[c];
        gd.delta[c] = g->delta[c];
    }
    gd.s[D - 1] = 1;
    for (int c = D - 2; c >= 0; --c) gd.s[c] = gd.s[c + 1] * g->n[c + 1];
    gd.N = (int)N;
    return CVX_OK;
}

template <int D>
int check_dirs(int nd, const int32_t *off, const GridT<D> &gd, std::vector<GridDirT<D>> &dirs,
               std::vector<long long> &line_off) {
    if (nd < 1 || nd > kGridMaxDirs)
        return fail(CVX_ERR_INVALID_ARG, "direction count must be in [1, %d]", kGridMaxDirs);
    if (!off) return fail(CVX_ERR_INVALID_ARG, "direction offsets are NULL");
    constexpr int d = D == 4 ? 2 : 3;
    dirs.resize(nd);
    line_off.assign(nd + 1, 0);
    for (int j = 0; j < nd; ++j) {
        GridDirT<D> g{};
        bool nz = false;
        for (int c = 0; c < D; ++c) {
            const int o = off[D * j + c];
            if (o < -kGridMaxLine || o > kGridMaxLine)
                return fail(CVX_ERR_INVALID_ARG, "direction %d: offset out of range", j);
            g.o[c] = o;
            nz |= o != 0;
            if (o > 0) g.pos |= 1u << c;
            if (o < 0) g.neg |= 1u << c;
        }
        if (!nz) return fail(CVX_ERR_INVALID_ARG, "direction %d is zero", j);
        // rank one: every 2x2 minor of the d x d offset matrix vanishes
        for (int a = 0; a < d; ++a)
            for (int b = a + 1; b < d; ++b)
                for (int c = 0; c < d; ++c)
                    for (int e = c + 1; e < d; ++e)
                        if ((long long)g.o[d * a + c] * g.o[d * b + e] !=
                            (long long)g.o[d * a + e] * g.o[d * b + c])
                            return fail(CVX_ERR_INVALID_ARG, "direction %d is not rank-one", j);
        long long step = 0;
        for (int c = 0; c < D; ++c) step += (long long)g.o[c] * gd.s[c];
        g.step = (int)step;
        dirs[j] = g;
        line_off[j + 1] = line_off[j] + lines_of<D>(gd, g, kMinLine<D>);
    }
    return CVX_OK;
}

// Device buffers shared by cvx_grid_step and cvx_grid_convexify.
template <int D>
struct GridWork {
    GridDirT<D> *dirs;
    long long *line_off;
    unsigned *cur;  // nd x (longest line + 1): line counts by length (k_grid_cursors)
    int *starts;
    float *H;
    unsigned *S;
    unsigned long long *pat;  // k_grid_patterns
    int chunk;  // directions per chunk
    bool unit;  // all offsets in {-1, 0, 1}
};

template <int D>
size_t grid_patterns(int nd, int chunk) {
    return (size_t)((nd + chunk - 1) / chunk) << D;
}

template <int D>
size_t grid_work_bytes(int nd, const GridT<D> &gd, long long lines, int &chunk) {
    const size_t per_dir = (size_t)gd.N * (sizeof(float) + sizeof(unsigned));
    chunk = (int)std::max<size_t>(
        1, std::min<size_t>(std::min(nd, kGridChunkDirs), grid_chunk_bytes() / per_dir));
    return up256(sizeof(GridDirT<D>) * nd) + up256(sizeof(long long) * (nd + 1)) +
           up256(sizeof(unsigned) * nd * (size_t)(kGridMaxLine + 1)) +
           up256(sizeof(int) * (size_t)lines) + up256(sizeof(unsigned long long) * grid_patterns<D>(nd, chunk)) +
           up256(sizeof(float) * (size_t)chunk * gd.N) +
           up256(sizeof(unsigned) * (size_t)chunk * gd.N);
}

template <int D>
void carve_grid_work(char *ws, const std::vector<GridDirT<D>> &dirs, const GridT<D> &gd,
                     long long lines, int chunk, GridWork<D> &w) {
    const int nd = (int)dirs.size();
    w.dirs = (GridDirT<D> *)ws;
    ws += up256(sizeof(GridDirT<D>) * nd);
    w.line_off = (long long *)ws;
    ws += up256(sizeof(long long) * (nd + 1));
    w.cur = (unsigned *)ws;
    ws += up256(sizeof(unsigned) * nd * (size_t)(kGridMaxLine + 1));
    w.starts = (int *)ws;
    ws += up256(sizeof(int) * (size_t)lines);
    w.pat = (unsigned long long *)ws;
    ws += up256(sizeof(unsigned long long) * grid_patterns<D>(nd, chunk));
    w.H = (float *)ws;
    ws += up256(sizeof(float) * (size_t)chunk * gd.N);
    w.S = (unsigned *)ws;
    w.chunk = chunk;
    w.unit = true;
    for (const GridDirT<D> &d : dirs)
        for (int c = 0; c < D; ++c) w.unit = w.unit && std::abs(d.o[c]) <= 1;
}

template <int D>
int grid_line_cap(const GridT<D> &gd) {
    int cap = 1;
    for (int c = 0; c < D; ++c) cap = std::max(cap, gd.n[c]);
    return cap;
}

// Threads per line-kernel CTA so that the stacks fit in shared memory.
int grid_line_threads(int cap) { return cap <= 128 ? 128 : (cap <= 256 ? 64 : 32); }

// Direction table, line regions and line starts.
template <int D>
int grid_setup(const GridT<D> &gd, const std::vector<GridDirT<D>> &dirs,
               const std::vector<long long> &line_off, const GridWork<D> &w, cudaStream_t s) {
    const int nd = (int)dirs.size();
    CK(cudaMemcpyAsync(w.dirs, dirs.data(), sizeof(GridDirT<D>) * nd, cudaMemcpyHostToDevice, s),
       "grid setup");
    CK(cudaMemcpyAsync(w.line_off, line_off.data(), sizeof(long long) * (nd + 1),
                       cudaMemcpyHostToDevice, s),
       "grid setup");
    if (w.unit && D == 9) {
        const size_t np = grid_patterns<D>(nd, w.chunk);
        k_grid_patterns<D><<<(unsigned)((np + 127) / 128), 128, 0, s>>>(w.dirs, nd, w.chunk, w.pat);
        CK(cudaGetLastError(), "grid patterns");
    }
    if (line_off[nd] == 0) return CVX_OK;
    const int cap = grid_line_cap<D>(gd);
    k_grid_cursors<D><<<(nd * (cap + 1) + 127) / 128, 128, 0, s>>>(gd, w.dirs, nd, cap, w.cur);
    CK(cudaGetLastError(), "grid line counts");
    auto ks = w.unit ? k_grid_starts<D, true> : k_grid_starts<D, false>;
    const size_t smem = sizeof(int) * (size_t)nd * (w.unit ? 2 : D);
    CK(cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
       "grid line starts shared memory");
    const int bx = (int)std::min<long long>((gd.N + 255) / 256, 4096);
    ks<<<bx, 256, smem, s>>>(gd, w.dirs, nd, w.line_off, w.cur, cap, w.starts);
    CK(cudaGetLastError(), "grid line starts");
    return CVX_OK;
}

// One step (all chunks) from Win to Wout.
template <int D>
int grid_enqueue_step(const GridT<D> &gd, int nd, const std::vector<long long> &line_off,
                      const GridWork<D> &w, int cap, const double *Win, double *Wout, int *lam,
                      unsigned long long *dec, const int *done, cudaStream_t s,
                      cvx_handle *h) {
    const int T = grid_line_threads(cap);
    const size_t smem = (size_t)cap * T * sizeof(short);
    for (int j0 = 0; j0 < nd; j0 += w.chunk) {
        const int j1 = std::min(nd, j0 + w.chunk);
        const long long lines = line_off[j1] - line_off[j0];
        if (lines > 0) {
            std::vector<cudaEvent_t> ev;
            int rc = scan_events(h, 1, ev);
            if (rc) return rc;
            if (!ev.empty()) CK(cudaEventRecord(ev[0], s), "grid profiling");
            k_grid_lines<D><<<(unsigned)((lines + T - 1) / T), T, smem, s>>>(
                gd, w.dirs, w.line_off, j0, j1, w.starts, w.cur, Win, w.H, w.S, cap, done);
            CK(cudaGetLastError(), "grid line kernel");
            if (!ev.empty()) CK(cudaEventRecord(ev[1], s), "grid profiling");
        }
        auto kr = w.unit ? k_grid_reduce<D, true> : k_grid_reduce<D, false>;
        kr<<<(unsigned)((gd.N + 255LL) / 256), 256, 0, s>>>(gd, w.dirs, j0, j1, j0 == 0, j1 == nd,
                                                            Win, w.H, w.S,
                                                            w.pat + ((size_t)(j0 / w.chunk) << D),
                                                            Wout, lam, dec, done);
        CK(cudaGetLastError(), "grid reduce kernel");
    }
    return CVX_OK;
}

template <int D>
int set_line_smem(int cap) {
    const int T = grid_line_threads(cap);
    const size_t smem = (size_t)cap * T * sizeof(short);
    CK(cudaFuncSetAttribute(k_grid_lines<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)smem),
       "grid line kernel shared memory");
    return CVX_OK;
}

int check_grid_call(const cvx_params *p, const cvx_grid *g, int32_t det_rule, double beta_k) {
    if (p) {
        int rc = check_params(p, false, true);
        if (rc) return rc;
    }
    if (!g) return fail(CVX_ERR_INVALID_ARG, "grid is NULL");
    if (g->dim != 2 && g->dim != 3) return fail(CVX_ERR_INVALID_ARG, "grid dim must be 2 or 3");
    if (p && g->dim == 3 && p->energy == CVX_ENERGY_DOUBLE_WELL)
        return fail(CVX_ERR_INVALID_ARG, "the double-well energy is two-dimensional");
    if (det_rule != 0 && det_rule != 1) return fail(CVX_ERR_INVALID_ARG, "det_rule must be 0 or 1");
    if (!isfinite(beta_k)) return fail(CVX_ERR_INVALID_ARG, "beta_k must be finite");
    return CVX_OK;
}

template <int D>
int grid_energy_t(cvx_handle *h, const cvx_params *p, const cvx_grid *g, double beta_k,
                  int32_t rule, double *W, cudaStream_t s) {
    GridT<D> gd;
    int rc = check_grid<D>(g, gd);
    if (rc) return rc;
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (!W) return fail(CVX_ERR_INVALID_ARG, "W is NULL");
    DeviceGuard dg(h->device);
    k_grid_energy<D><<<(gd.N + 255) / 256, 256, 0, s>>>(gd, material_of(p), beta_k, rule, W);
    CK(cudaGetLastError(), "cvx_grid_energy");
    return CVX_OK;
}

template <int D>
int grid_step_t(cvx_handle *h, const cvx_grid *g, int32_t nd, const int32_t *off,
                const double *W_in, double *W_out, int32_t *lam, double *dec, cudaStream_t s) {
    GridT<D> gd;
    int rc = check_grid<D>(g, gd);
    if (rc) return rc;
    std::vector<GridDirT<D>> dirs;
    std::vector<long long> line_off;
    rc = check_dirs<D>(nd, off, gd, dirs, line_off);
    if (rc) return rc;
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (!W_in || !W_out) return fail(CVX_ERR_INVALID_ARG, "W_in and W_out are required");
    if (W_in == W_out) return fail(CVX_ERR_INVALID_ARG, "W_out must not alias W_in");
    DeviceGuard dg(h->device);
    const long long lines = line_off[nd];
    int chunk = 0;
    size_t bytes = grid_work_bytes<D>(nd, gd, lines, chunk);
    const size_t lam_off = bytes;
    if (!lam) bytes += up256(sizeof(int) * 3 * (size_t)gd.N);
    rc = ensure_ws(h, bytes, s);
    if (rc) return rc;
    GridWork<D> w;
    carve_grid_work<D>(h->ws, dirs, gd, lines, chunk, w);
    int *lam_w = lam ? lam : (int *)(h->ws + lam_off);
    const int cap = grid_line_cap<D>(gd);
    rc = set_line_smem<D>(cap);
    if (rc) return rc;
    rc = grid_setup<D>(gd, dirs, line_off, w, s);
    if (rc) return rc;
    if (dec) CK(cudaMemsetAsync(dec, 0, sizeof(double), s), "cvx_grid_step");
    return grid_enqueue_step<D>(gd, nd, line_off, w, cap, W_in, W_out, lam_w,
                                reinterpret_cast<unsigned long long *>(dec), nullptr, s, h);
}

template <int D>
int grid_convexify_t(cvx_handle *h, const cvx_params *p, const cvx_grid *g, double beta_k,
                     int32_t rule, int32_t nd, const int32_t *off, int32_t kmax, double tol,
                     double *W, int32_t *forest, double *decs, int32_t *iters, cudaStream_t s) {
    GridT<D> gd;
    int rc = check_grid<D>(g, gd);
    if (rc) return rc;
    std::vector<GridDirT<D>> dirs;
    std::vector<long long> line_off;
    rc = check_dirs<D>(nd, off, gd, dirs, line_off);
    if (rc) return rc;
    if (kmax < 1 || kmax > kGridMaxIters)
        return fail(CVX_ERR_INVALID_ARG, "kmax must be in [1, %d]", kGridMaxIters);
    if (!(tol >= 0.0)) return fail(CVX_ERR_INVALID_ARG, "tol must be >= 0");
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (!W || !iters) return fail(CVX_ERR_INVALID_ARG, "W and iters are required");
    DeviceGuard dg(h->device);
    const long long lines = line_off[nd];
    int chunk = 0;
    size_t bytes = grid_work_bytes<D>(nd, gd, lines, chunk);
    const size_t o_pong = bytes;
    bytes += up256(sizeof(double) * (size_t)gd.N);
    const size_t o_lam = bytes;
    if (!forest) bytes += up256(sizeof(int) * 3 * (size_t)gd.N);
    const size_t o_dec = bytes;
    if (!decs) bytes += up256(sizeof(double) * kmax);
    const size_t o_done = bytes;
    bytes += 256;
    rc = ensure_ws(h, bytes, s);
    if (rc) return rc;
    GridWork<D> w;
    carve_grid_work<D>(h->ws, dirs, gd, lines, chunk, w);
    double *pong = (double *)(h->ws + o_pong);
    unsigned long long *dk =
        reinterpret_cast<unsigned long long *>(decs ? decs : (double *)(h->ws + o_dec));
    int *done = (int *)(h->ws + o_done);
    const int cap = grid_line_cap<D>(gd);
    rc = set_line_smem<D>(cap);
    if (rc) return rc;
    rc = grid_setup<D>(gd, dirs, line_off, w, s);
    if (rc) return rc;
    CK(cudaMemsetAsync(dk, 0, sizeof(double) * kmax, s), "cvx_grid_convexify");
    CK(cudaMemsetAsync(done, 0, sizeof(int), s), "cvx_grid_convexify");
    CK(cudaMemsetAsync(iters, 0, sizeof(int32_t), s), "cvx_grid_convexify");
    const unsigned pb = (unsigned)((gd.N + 255) / 256);
    k_grid_energy<D><<<pb, 256, 0, s>>>(gd, material_of(p), beta_k, rule, W);
    CK(cudaGetLastError(), "cvx_grid_convexify energy");
    for (int k = 0; k < kmax; ++k) {
        const double *in = (k & 1) ? pong : W;
        double *out = (k & 1) ? W : pong;
        int *lam = forest ? forest + 3 * (size_t)k * gd.N : (int *)(h->ws + o_lam);
        rc = grid_enqueue_step<D>(gd, nd, line_off, w, cap, in, out, lam, dk + k, done, s, h);
        if (rc) return rc;
        k_grid_check<<<1, 1, 0, s>>>(dk + k, tol, done, iters, k);
        CK(cudaGetLastError(), "cvx_grid_convexify check");
    }
    k_grid_final<<<pb, 256, 0, s>>>(gd.N, iters, pong, W);
    CK(cudaGetLastError(), "cvx_grid_convexify final");
    return CVX_OK;
}

template <int D, bool kA>
int grid_query_run(cvx_handle *h, const GridT<D> &gd, const std::vector<GridDirT<D>> &dirs,
                   const cvx_params *p, double beta_k, int32_t rule, int32_t K, const double *WK,
                   const int32_t *forest, int64_t n, const double *F, double *W_interp,
                   double *W_tree, double *P, double *A, int64_t *leaves, cudaStream_t s) {
    using R = TreeRec<D, kA>;
    const int nd = (int)dirs.size();
    // two buffers of records, two arrays of flags
    const size_t tab = up256(sizeof(double) * R::kWords * (size_t)gd.N), fl = up256(gd.N);
    const size_t o_t = up256(sizeof(GridDirT<D>) * nd);
    int rc = ensure_ws(h, o_t + 2 * tab + 2 * fl, s);
    if (rc) return rc;
    GridDirT<D> *dd = (GridDirT<D> *)h->ws;
    double *T0 = (double *)(h->ws + o_t), *T1 = (double *)(h->ws + o_t + tab);
    unsigned char *f0 = (unsigned char *)(h->ws + o_t + 2 * tab), *f1 = f0 + fl;
    CK(cudaMemcpyAsync(dd, dirs.data(), sizeof(GridDirT<D>) * nd, cudaMemcpyHostToDevice, s),
       "cvx_grid_query");
    const Material mat = material_of(p);
    k_grid_tree0<D, kA><<<(unsigned)((gd.N + (long long)kTreeThreads - 1) / kTreeThreads), kTreeThreads, 0, s>>>(
        gd, mat, beta_k, rule, T0, f0);
    CK(cudaGetLastError(), "cvx_grid_query leaves");
    const unsigned nb = (unsigned)((gd.N + (long long)kStepThreads - 1) / kStepThreads);
    for (int d = 1; d <= K; ++d) {
        k_grid_tree_step<D, kA><<<nb, kStepThreads, 0, s>>>(gd, dd, nd, forest + 3 * (size_t)(d - 1) * gd.N, mat,
                                                   beta_k, rule, T0, T1, f0, f1);
        CK(cudaGetLastError(), "cvx_grid_query tree order");
        std::swap(f0, f1);
    }
    // queries per block: fewer where there are not enough for eight blocks per
    // SM, and fewer than a warp's lanes (whose cells a block finds first) only
    // where there is not one block per SM.  1,000 queries, d = 3: 1.66 ms in
    // blocks of 128, 0.36 ms so; 10,000, d = 2 with the tangent: 0.27 and 0.23 ms
    int per = kQueryThreads;
    while (per > 32 && n < (long long)per * 8 * h->sm_count) per /= 2;
    while (per > kQueryThreads / R::kLanes && n < (long long)per * h->sm_count) per /= 2;
    k_grid_query<D, kA><<<(unsigned)((n + per - 1) / per), kQueryThreads, 0, s>>>(
        gd, WK, T0, T1, f0, n, per, F, W_interp, W_tree, P, A, reinterpret_cast<long long *>(leaves));
    CK(cudaGetLastError(), "cvx_grid_query");
    return CVX_OK;
}

template <int D>
int grid_query_t(cvx_handle *h, const cvx_params *p, const cvx_grid *g, double beta_k,
                 int32_t rule, int32_t nd, const int32_t *off, int32_t K, const double *WK,
                 const int32_t *forest, int64_t n, const double *F, double *W_interp,
                 double *W_tree, double *P, double *A, int64_t *leaves, cudaStream_t s) {
    GridT<D> gd;
    int rc = check_grid<D>(g, gd);
    if (rc) return rc;
    std::vector<GridDirT<D>> dirs;
    std::vector<long long> line_off;
    rc = check_dirs<D>(nd, off, gd, dirs, line_off);
    if (rc) return rc;
    if (K < 0 || K > kGridMaxIters)
        return fail(CVX_ERR_INVALID_ARG, "K must be in [0, %d]", kGridMaxIters);
    if (!h) return fail(CVX_ERR_INVALID_ARG, "handle is NULL");
    if (n < 0) return fail(CVX_ERR_INVALID_ARG, "n < 0");
    if (n > 0 && (!WK || !F || !W_interp || !W_tree || !P || (K > 0 && !forest)))
        return fail(CVX_ERR_INVALID_ARG, "NULL array (WK, F, W_interp, W_tree, P; forest if K > 0)");
    if (n == 0) return CVX_OK;
    DeviceGuard dg(h->device);
    return A ? grid_query_run<D, true>(h, gd, dirs, p, beta_k, rule, K, WK, forest, n, F, W_interp,
                                       W_tree, P, A, leaves, s)
             : grid_query_run<D, false>(h, gd, dirs, p, beta_k, rule, K, WK, forest, n, F, W_interp,
                                        W_tree, P, A, leaves, s);
}

}  // namespace
}  // namespace cvx

using namespace cvx;

extern "C" {

int cvx_grid_r11(int32_t dim, int32_t *off) {
    if (!off) return fail(CVX_ERR_INVALID_ARG, "off is NULL");
    if (dim == 2) {
        // a, b over (1,0), (0,1), (1,1), (1,-1): one of each pair +-v (the
        // sign of a (x) b gives the same line); direction 4 ia + ib
        static const int v[4][2] = {{1, 0}, {0, 1}, {1, 1}, {1, -1}};
        for (int ia = 0; ia < 4; ++ia)
            for (int ib = 0; ib < 4; ++ib)
                for (int i = 0; i < 2; ++i)
                    for (int j = 0; j < 2; ++j)
                        off[4 * (4 * ia + ib) + 2 * i + j] = v[ia][i] * v[ib][j];
        return CVX_OK;
    }
    if (dim == 3) {
        // the 13 vectors of {-1,0,1}^3 with first nonzero entry +1: axes,
        // face diagonals, body diagonals; direction 13 ia + ib
        static const int v[13][3] = {{1, 0, 0},  {0, 1, 0},  {0, 0, 1},  {1, 1, 0}, {1, -1, 0},
                                     {1, 0, 1},  {1, 0, -1}, {0, 1, 1},  {0, 1, -1}, {1, 1, 1},
                                     {1, 1, -1}, {1, -1, 1}, {1, -1, -1}};
        for (int ia = 0; ia < 13; ++ia)
            for (int ib = 0; ib < 13; ++ib)
                for (int i = 0; i < 3; ++i)
                    for (int j = 0; j < 3; ++j)
                        off[9 * (13 * ia + ib) + 3 * i + j] = v[ia][i] * v[ib][j];
        return CVX_OK;
    }
    return fail(CVX_ERR_INVALID_ARG, "dim must be 2 or 3");
}

int cvx_grid_energy(cvx_handle *h, const cvx_params *p, const cvx_grid *g, double beta_k,
                    int32_t det_rule, double *W, cvx_stream sv) {
    if (!p) return fail(CVX_ERR_INVALID_ARG, "params is NULL");
    int rc = check_grid_call(p, g, det_rule, beta_k);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)sv;
    return g->dim == 2 ? grid_energy_t<4>(h, p, g, beta_k, det_rule, W, s)
                       : grid_energy_t<9>(h, p, g, beta_k, det_rule, W, s);
}

int cvx_grid_step(cvx_handle *h, const cvx_grid *g, int32_t nd, const int32_t *off,
                  const double *W_in, double *W_out, int32_t *lam, double *dec, cvx_stream sv) {
    int rc = check_grid_call(nullptr, g, 0, 0.0);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)sv;
    return g->dim == 2 ? grid_step_t<4>(h, g, nd, off, W_in, W_out, lam, dec, s)
                       : grid_step_t<9>(h, g, nd, off, W_in, W_out, lam, dec, s);
}

int cvx_grid_convexify(cvx_handle *h, const cvx_params *p, const cvx_grid *g, double beta_k,
                       int32_t det_rule, int32_t nd, const int32_t *off, int32_t kmax, double tol,
                       double *W, int32_t *forest, double *decs, int32_t *iters,
                       cvx_stream sv) {
    if (!p) return fail(CVX_ERR_INVALID_ARG, "params is NULL");
    int rc = check_grid_call(p, g, det_rule, beta_k);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)sv;
    return g->dim == 2 ? grid_convexify_t<4>(h, p, g, beta_k, det_rule, nd, off, kmax, tol, W,
                                             forest, decs, iters, s)
                       : grid_convexify_t<9>(h, p, g, beta_k, det_rule, nd, off, kmax, tol, W,
                                             forest, decs, iters, s);
}

int cvx_grid_query(cvx_handle *h, const cvx_params *p, const cvx_grid *g, double beta_k,
                   int32_t det_rule, int32_t nd, const int32_t *off, int32_t K, const double *WK,
                   const int32_t *forest, int64_t n, const double *F, double *W_interp,
                   double *W_tree, double *P, double *A, int64_t *leaves, cvx_stream sv) {
    if (!p) return fail(CVX_ERR_INVALID_ARG, "params is NULL");
    int rc = check_grid_call(p, g, det_rule, beta_k);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)sv;
    return g->dim == 2 ? grid_query_t<4>(h, p, g, beta_k, det_rule, nd, off, K, WK, forest, n, F,
                                         W_interp, W_tree, P, A, leaves, s)
                       : grid_query_t<9>(h, p, g, beta_k, det_rule, nd, off, K, WK, forest, n, F,
                                         W_interp, W_tree, P, A, leaves, s);
}

}  // extern "C"
