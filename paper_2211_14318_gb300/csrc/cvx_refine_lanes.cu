// cvx_refine_lanes.cu -- the FP64 refinement of the damage energy's candidates
// after the lane-per-line scan, one candidate per lane.
//
// A candidate is a line with the scan's FP32 bridge pair (a, b).  Its FP64
// bridge is the pair whose chord lies strictly below every other sample of
// the left and right sets.  Per round a lane takes the chord of its pair in
// FP64 (two samples), asks which parts of its line can hold a sample at or
// below the chord (the interval bounds of cvx_intervals.cuh on FP32 samples,
// with their error bound), and has only the samples in question taken in
// FP64:
//  - a run of such intervals around an end of the pair on which v is convex
//    (a bound of v'' from below) needs the end's two neighbours only: a convex
//    function that vanishes at the end and is positive next to it is positive
//    beyond;
//  - a run from an end on the line's edge on which v is concave (and whose
//    far end lies above the chord) needs none;
//  - elsewhere every sample whose FP32 value is inconclusive is taken.
// A sample below an end of the pair (v - s x at the chord's slope s; on equal
// values the outer one) moves that end to the lowest one of its side: the
// supporting-slope iteration, ties as in Algorithm 1.  A pair is done when all
// other samples lie strictly above its chord, or when both ends are the lowest
// of a search in full; samples within rounding of the chord need no more than
// that.  The scan's pair is that of FP32 samples, on nearly affine
// lines up to 64 samples off: an end in a convex run first goes to where v has
// the chord's slope (a Newton step in FP32, twice at most), and a neighbour
// found on or below the chord is moved to (three times at most) before its
// side is searched in full.  None of these decides anything: the pair is done
// when the intervals and samples above say so for its own chord.  A candidate
// that needs too many FP64 samples has its whole line taken by the warp, each
// sample once (ref_full).
//
// The samples to be taken in FP64 queue in shared memory over the warp's 32
// candidates and are taken 32 at a time, one per lane.  What bounds the
// refinement is the FP64 pipe (2 lanes per SM and clock: a sample, one
// logarithm and one exponential, costs a warp about 1,400 cycles of it
// whether 1 or 32 lanes take part), so a full queue is what counts.
#include <cuda_runtime.h>
#include <limits.h>

#include "cvx_bridge.cuh"
#include "cvx_intervals.cuh"
#include "cvx_refine.cuh"

namespace cvx {

namespace {

constexpr int kRefWarps = 4;
// Newton steps and neighbour moves per candidate.  Without them a candidate of
// a load step's proposal windows took 29 FP64 samples beside its chords' ends,
// with them 2 (k_refine_lanes 15.9 -> 5.2 ms of a step).
constexpr int kRefJumps = 2, kRefWalks = 3;
// Candidates per warp at least: eight, but four where lines are longer than
// kRefLongL in a window narrower than kRefNarrow: lines are nearly affine there,
// and their searches in full a serial chain in their warp.  2,000 points, 16^2
// directions, L = 2049, t_half = 0.01: 10.7 ms with eight, 8.4 with four; in
// windows of 0.5 the FP64 pipe counts, which a half-filled warp loads as much: a
// mesh of 676 points, 30^2 directions, L = 987: 96 us of refinement with eight,
// 125 with four.
constexpr int kRefLongL = 512;
constexpr float kRefNarrow = 0.03f;
// Half as many FP64 samples, or half the line, and the candidate has its whole
// line taken.  2,000 points, 16^2 directions, L = 201, t_half = 1e-6 (nearly all
// samples within rounding of the chord): 58 ms without this limit and with pairs
// that move on to samples within rounding above their chord, 10 ms so; at half
// the line alone, L = 33, t_half = 1e-4: 2.8 ms, with 128 at least 2.1.
constexpr int kRefMany = 128;
constexpr int kRefRounds = 24;  // chords per candidate before the whole line is taken in FP64

// A lane's candidate as the queue's other lanes need it.
struct RefLane {
    double F[4], R[4], beta, ek, h, wa, s;
    const ProbDesc *pd;
    long long key[2];  // lowest v - s x (dkey) on or below the chord, left and right
    int k[2];          // its sample
    int a, m0, L;
};

__device__ __noinline__ double ref_sample(const RefLane &r, int k) {
    return sample_w64_ek(r.F, r.R, k, r.m0, r.h, r.beta, r.ek, r.pd->mat);
}

// Key of v - s x at sample k of value v, rounded once everywhere, so that keys
// of one slope compare.
__device__ __forceinline__ long long ref_key(double v, double s, int k, int m0) {
    return dkey(__fma_rn(-s, (double)(k - m0), v));
}

// Takes queued samples (owner lane << 12 | sample) in FP64, 32 at a time, and
// records those on or below their owner's chord; with `all` the rest too.
// Returns the number of entries left in the queue.
__device__ __noinline__ int ref_spots(RefLane *rl, int *q, int nq, bool all, int lane,
                                      unsigned &n_spot) {
    while (nq >= 32 || (all && nq > 0)) {
        const int n = min(nq, 32);
        bool low = false;
        long long e = kKeyInf;
        int side = 0, k = 0;
        RefLane *r = rl;
        if (lane < n) {
            const int ent = q[lane];
            r = rl + (ent >> 12);
            k = ent & 0xfff;
            side = k > r->m0;
            const double v = ref_sample(*r, k);
            const double line = r->wa + r->s * (double)(k - r->a);
            low = v == v && !(v > line + 1e-14 * fabs(line));  // NaN: det <= 0, excluded
            if (low) e = ref_key(v, r->s, k, r->m0);
            ++n_spot;
        }
        const long long old = r->key[side];
        __syncwarp();
        if (low) atomicMin(&r->key[side], e);
        __syncwarp();
        const long long now = r->key[side];
        const bool win = low && e == now;
        if (win && now < old) r->k[side] = side ? -1 : INT_MAX;
        __syncwarp();
        if (win) {
            if (side) atomicMax(&r->k[1], k);
            else atomicMin(&r->k[0], k);
        }
        __syncwarp();
        const int rest = nq - n;
        const int m0 = lane < rest ? q[n + lane] : 0, m1 = 32 + lane < rest ? q[n + 32 + lane] : 0;
        __syncwarp();
        if (lane < rest) q[lane] = m0;
        if (32 + lane < rest) q[32 + lane] = m1;
        __syncwarp();
        nq = rest;
    }
    return nq;
}

// The whole line in FP64 (warp-wide, for the candidate of one lane): the
// supporting-slope iteration of bridge64.  Sample k is lane k % 32's k / 32-th,
// taken once (in local memory: the passes that follow cost two FP64 operations
// per sample, a sample some forty).
constexpr int kFullPer = (2079 + 31) / 32;

__device__ __noinline__ void ref_full(const RefLane &r, int L, int lane, int &a, int &b, double &wa,
                                      double &wb) {
    double s = 0.0, v[kFullPer];
    for (int k = lane, i = 0; k < L; k += 32, ++i) {
        const double x = k == r.m0 ? INFINITY : ref_sample(r, k);
        v[i] = x == x ? x : INFINITY;
    }
    __syncwarp();
    a = b = -1;
    for (int it = 0; it < 128; ++it) {
        long long bl = kKeyInf, br = kKeyInf;
        int kl = INT_MAX, kr = -1;
        for (int k = lane, i = 0; k < L; k += 32, ++i) {
            if (!(v[i] < INFINITY)) continue;
            const long long e = ref_key(v[i], s, k, r.m0);
            if (k < r.m0) {
                if (e < bl || (e == bl && k < kl)) {
                    bl = e;
                    kl = k;
                }
            } else if (e < br || (e == br && k > kr)) {
                br = e;
                kr = k;
            }
        }
        __syncwarp();
        warp_min_key(bl, kl, true);
        warp_min_key(br, kr, false);
        if (kl == INT_MAX || kr < 0) {
            a = b = -1;
            return;
        }
        if (kl == a && kr == b) return;
        a = kl;
        b = kr;
        wa = __shfl_sync(kFull, v[a >> 5], a & 31);
        wb = __shfl_sync(kFull, v[b >> 5], b & 31);
        s = (wb - wa) / (double)(b - a);
    }
}

// Samples from t to where v has slope ls per sample, by one Newton step in FP32
// (v' and v'' from the line's constants, so their error is relative to them and
// not to v).  Only a guess: the samples decide.
__device__ __forceinline__ float tangent_step(const IvLine &l, float t, float h, float ls) {
    float A0, A1, B1, B2, u;
    upk2(l.c.A0, A0, u);
    upk2(l.c.A1, A1, u);
    upk2(l.c.B1, B1, u);
    upk2(l.c.B2, B2, u);
    const float J = __fmaf_rn(t, l.cJ, l.J0), lg = lg2_approx(J), r = __fdividef(l.cJ, J);
    const float d = __fmaf_rn(lg, __fmaf_rn(lg, B2, B1), __fmaf_rn(t, __fmaf_rn(t, l.A2, A1), A0));
    const float d1 = __fmaf_rn(r * (1.0f / kLn2), __fmaf_rn(2.0f * B2, lg, B1), __fmaf_rn(2.0f * l.A2, t, A1));
    const float d2 = __fmaf_rn(r * r, __fmaf_rn(-l.c1, lg, l.c0), 2.0f * l.A2);
    const float E = l.K2 * ex2_approx(-fmaxf(d, 0.0f));
    const float v1 = h * __fmaf_rn(E, d1, d1);
    const float v2 = h * h * (d > 0.0f ? __fmaf_rn(E, d2 - kLn2 * d1 * d1, d2) : __fmaf_rn(E, d2, d2));
    return __fdividef(ls - v1, v2);
}

}  // namespace

// One warp takes 32 candidates at a time: phase 0 each node's first candidate,
// phase 1 the others whose lower bound does not exceed the node's first value
// (see k_refine).  With fewer candidates than lanes the warps take fewer each,
// but some at least (kRefLongL): a chord's two FP64 samples cost a warp the same
// for 1 and 32 lanes (an FE step of 20,011 points: 10.80 ms with one, 10.60 with
// 8, 10.58 with 16, 10.64 with 32).
// Measured per call, all launches together, against one warp per candidate
// with 32 or 64 FP64 samples in two windows and the certificate over every
// FP32 sample: 1,706,177 candidates at L = 201: 22.3 -> 1.25 ms (one spot
// sample each); 1,809,226 candidates of a load
// step's proposal windows at L = 2049, nearly affine lines: 47.5 -> 5.2 ms (2
// each); 110 candidates: 474 -> 48 us over four launches.
__global__ void __launch_bounds__(32 * kRefWarps) k_refine_lanes(const Pipe P, int level, int phase) {
    __shared__ RefLane s_rl[kRefWarps][32];
    __shared__ int s_q[kRefWarps][96];
    __shared__ int2 s_w[kRefWarps][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    RefLane *rl = s_rl[warp];
    RefLane &my = rl[lane];
    int *q = s_q[warp];
    int2 *sw = s_w[warp];
    const unsigned below = (1u << lane) - 1u;
    const int nwarps = gridDim.x * kRefWarps, gw = blockIdx.x * kRefWarps + warp;
    const int nwork = P.cnt[(P.K + 1) + level];
    const int least = P.stride32 > kRefLongL && P.t_half < kRefNarrow ? 4 : 8;
    const int bs = min(32, max(least, (nwork + nwarps - 1) / nwarps));
    const int32_t *qp = P.qp[level], *qh = P.qh[level];
    unsigned n_ref = 0, n_full = 0, n_spot = 0;
    long long blk = gw;
    int nbuf = 0;
    for (;;) {
        // ---- the warp's next candidates
        while (nbuf < 32 && blk * bs < nwork) {
            const long long i = blk * bs + lane;
            bool ok = lane < bs && i < nwork;
            int2 wk = make_int2(0, 0);
            if (ok) {
                wk = P.work[i];
                if (phase == 0) {
                    ok = wk.y == 0;
                } else if (wk.y == 0) {
                    ok = false;
                } else {
                    const RefineOut *ro = P.refined + (long long)wk.x * kNodeCand;
                    const ProbDesc &pd = P.probs[P.pid[qp[wk.x]]];
                    const double w_node = node_ptr(pd, qp[wk.x], qh[wk.x])->w;
                    const double V0 = ro[0].ok && ro[0].q < w_node ? ro[0].q : w_node;
                    ok = !(ro[wk.y].q > V0);  // else screened out by the stored lower bound
                }
            }
            const unsigned bal = __ballot_sync(kFull, ok);
            if (ok) sw[nbuf + __popc(bal & below)] = wk;
            nbuf += __popc(bal);
            blk += nwarps;
            __syncwarp();
        }
        if (nbuf == 0) break;
        const int nb = min(nbuf, 32);
        const bool act = lane < nb;
        const int2 wk = sw[act ? lane : 0];
        const int2 nxt = 32 + lane < nbuf ? sw[32 + lane] : make_int2(0, 0);
        __syncwarp();
        if (32 + lane < nbuf) sw[lane] = nxt;
        nbuf -= nb;
        n_ref += nb;

        // ---- the lane's candidate
        const int qi = wk.x, c = wk.y, p = qp[qi];
        const ProbDesc &pd = P.probs[P.pid[p]];
        const cvx_node *nd = node_ptr(pd, p, qh[qi]);
        const NodeCands &nc = P.cands[qi];
        const LineSpec ln = scaled_line(pd.line, nd->window_exp);
        const int m0 = ln.m0, L = ln.L, np = m0 >> 1;
        const int dir = nc.dir[c], hab = nc.ab[c];
        {
            const double *d = P.dir64 + 4 * ((long long)pd.dir_off + dir);
            my.R[0] = __dmul_rn(d[0], d[2]);
            my.R[1] = __dmul_rn(d[0], d[3]);
            my.R[2] = __dmul_rn(d[1], d[2]);
            my.R[3] = __dmul_rn(d[1], d[3]);
            for (int k = 0; k < 4; ++k) my.F[k] = nd->F[k];
            my.beta = pd.beta[p - pd.point_off];
            my.ek = nc.ek;
            my.h = ln.h64;
            my.pd = &pd;
            my.m0 = m0;
            my.L = L;
        }
        const DirLine dl =
            make_dir_line<CVX_ENERGY_NH_DAMAGE>(nc.nl, P.dir32[pd.dir_off + dir]);
        const IvLine l = iv_line(nc.nl, dl.A1, dl.A2, dl.cJ);
        const IvGeom G = iv_geom(ln.h32, m0);
        const f32x2 H = pk2(ln.h32, ln.h32);
        const double kap = pd.kappa, C = nc.shift;
        const float kapf = pd.kappa_f, Cf = (float)C;
        int a = hab & 0xffff, b = hab >> 16;
        bool slow = act && !(hab >= 0 && a < m0 && b > m0 && b < L);
        bool done = !act || slow;
        bool newA = true, newB = true, fullL = false, fullR = false;
        int jumps = 0, walks = 0;  // tangent steps and neighbour moves taken
        int taken = 0;             // FP64 samples taken beside the chords' ends
        double wa = 0.0, wb = 0.0;
        __syncwarp();

        for (int round = 0; round < kRefRounds; ++round) {
            if (__all_sync(kFull, done)) break;
            // ---- the chord
            if (!done && newA) wa = ref_sample(my, a);
            __syncwarp();
            if (!done && newB) wb = ref_sample(my, b);
            __syncwarp();
            if (!done && !(wa < INFINITY && wb < INFINITY)) slow = done = true;
            newA = newB = false;
            const double s = (wb - wa) / (double)(b - a);
            const float la = (float)(kap * wa - C), ls = (float)(kap * s);
            my.wa = wa;
            my.s = s;
            my.a = a;
            my.key[0] = my.key[1] = kKeyInf;
            // ---- intervals that can hold a sample on or below it
            unsigned todo[2] = {0u, 0u};
            int spot[4] = {-1, -1, -1, -1};
            bool moved = false;
            if (!done) {
                const float base = iv_base(kapf, Cf, ls, m0);
                float lev = __fmaf_rn(-ls, (float)(a - m0), la);  // the chord in v - s x
                const f32x2 NS = pk2(-ls, -ls);
#pragma unroll 1
                for (int side = 0; side < 2; ++side) {
                    const int xb = side ? 1 : -m0, xl = side ? m0 : -1;
                    const int NI = iv_count(G, np);
                    float ga, g1, Ea, E1;
                    iv_eval(l.c, H, NS, pk2((float)xb, (float)xl), ga, g1, Ea, E1);
                    unsigned m = iv_sweep<false>(l, G, H, NS, base, xb, (float)xl, NI, ga, Ea, lev);
                    if (NI == 0) continue;  // one sample: the end of the pair
                    const int k = side ? b : a;
                    const int j = min((int)(((float)((side ? k - m0 - 1 : k) >> 1) + 0.5f) * G.rPP), NI - 1);
                    m |= 1u << j;
                    // the run of intervals around the pair's end
                    const unsigned lo = ~m & ((1u << j) - 1u), hi = ~m >> j;
                    const int j0 = lo ? 32 - __clz(lo) : 0;
                    const int j1 = hi ? j + __ffs(hi) - 2 : 31;
                    unsigned run = (j1 >= 31 ? kFull : (1u << (j1 + 1)) - 1u) & ~((1u << j0) - 1u);
                    const int x0 = xb + 2 * G.PP * j0, x1 = min(xb + 2 * G.PP * (j1 + 1), xl);
                    bool full = side ? fullR : fullL;
                    if (!full) {
                        float low;
                        const int sh = line_shape(l, (float)x0 * G.h, (float)x1 * G.h, low);
                        const bool edge = side ? (b == L - 1 && j0 > 0) : (a == 0 && j1 < NI - 1);
                        if (sh > 0) {
                            const int k0 = side ? m0 + 1 : 0, k1 = side ? L - 1 : m0 - 1;
                            spot[2 * side] = k > k0 ? k - 1 : -1;
                            spot[2 * side + 1] = k < k1 ? k + 1 : -1;
                            if (jumps < kRefJumps && k > k0 && k < k1) {
                                // to where the chord's slope is the tangent's, if
                                // that is another sample of the run
                                const float st = tangent_step(l, (float)(k - m0) * G.h, G.h, ls);
                                const int kt = max(max(k0, x0 + m0), min(min(k1, x1 + m0),
                                                   k + (int)rintf(fmaxf(fminf(st, 4096.0f), -4096.0f))));
                                if (kt != k) {
                                    moved = true;
                                    if (side) {
                                        b = kt;
                                        newB = true;
                                    } else {
                                        a = kt;
                                        newA = true;
                                    }
                                }
                            }
                        } else if (!(sh < 0 && edge)) {
                            full = true;
                        }
                    }
                    if (full) run = 0;
                    todo[side] = m & ~run;
                    if (side) fullR = full;
                    else fullL = full;
                }
            }
            if (moved) {  // nothing to check against this chord
                ++jumps;
                fullL = fullR = false;
                todo[0] = todo[1] = 0u;
                for (int i = 0; i < 4; ++i) spot[i] = -1;
            }
            // ---- the neighbours of the pair's ends
            int nq = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const unsigned bal = __ballot_sync(kFull, spot[i] >= 0);
                taken += spot[i] >= 0 ? 1 : 0;
                if (spot[i] >= 0) q[nq + __popc(bal & below)] = (lane << 12) | spot[i];
                nq += __popc(bal);
                __syncwarp();
                if (nq >= 32) nq = ref_spots(rl, q, nq, false, lane, n_spot);
            }
            // ---- the samples of the remaining intervals whose FP32 value is
            // inconclusive
            const int PPmax = __reduce_max_sync(kFull, act ? G.PP : 0);
            while (__any_sync(kFull, (todo[0] | todo[1]) != 0u)) {
                const int side = todo[0] ? 0 : 1;
                const unsigned m = todo[side];
                const int j = __ffs(m) - 1;
                todo[side] = m & (m - 1u);
                const int xb = side ? 1 : -m0;
                const bool tail = m != 0 && (m0 & 1) && j == iv_count(G, np) - 1;
                for (int t = 0; t <= PPmax; ++t) {
                    // pair t of the interval; after its pairs the side's last
                    // sample, if that is a pair of its own
                    const int k = j * G.PP + t;
                    const bool pair = m != 0 && t < G.PP && k < np;
                    const bool last = tail && t == PPmax;
                    const float x = last ? (side ? (float)m0 : -1.0f) : (float)(xb + 2 * k);
                    const f32x2 X = pk2(x, x + 1.0f);
                    float v[2];
                    upk2(sample_nh2(l.c, mul2(X, H)), v[0], v[1]);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int ks = (int)x + i + m0;
                        bool need = (pair || (last && i == 0)) && ks != a && ks != b;
                        if (need && v[i] < INFINITY && v[i] > -INFINITY) {
                            const float xs = (float)(ks - a);
                            const float Lv = __fmaf_rn(ls, xs, la);
                            const float err = 2.0f * kU32 * (fabsf(la) + fabsf(ls * xs) + fabsf(Lv)) +
                                              kEps32 * fmaxf(kapf, fabsf(v[i]) + Cf) + 1e-30f;
                            need = !(__fsub_rn(v[i], Lv) > 1.001f * err);  // else above the chord
                        }
                        const unsigned bal = __ballot_sync(kFull, need);
                        taken += need ? 1 : 0;
                        if (need) q[nq + __popc(bal & below)] = (lane << 12) | ks;
                        nq += __popc(bal);
                    }
                    __syncwarp();
                    if (nq >= 32) nq = ref_spots(rl, q, nq, false, lane, n_spot);
                }
            }
            ref_spots(rl, q, nq, true, lane, n_spot);
            __syncwarp();
            // ---- certified, or on to the next chord
            if (!done && !moved) {
                const bool lowL = my.key[0] < kKeyInf, lowR = my.key[1] < kKeyInf;
                // of the samples on or below the chord, and those within rounding
                // above it, only one below the pair's end moves it (on equal values
                // the outermost, as in bridge64)
                bool betL = false, betR = false;
                if (lowL) {
                    const long long e = ref_key(wa, s, a, m0);
                    betL = my.key[0] < e || (my.key[0] == e && my.k[0] < a);
                }
                if (lowR) {
                    const long long e = ref_key(wb, s, b, m0);
                    betR = my.key[1] < e || (my.key[1] == e && my.k[1] > b);
                }
                if (!betL && !betR && (fullL || !lowL) && (fullR || !lowR)) {
                    done = true;
                } else if (2 * taken > max(my.L, kRefMany)) {
                    // most of the line is within rounding of its chord: one pass over
                    // it costs less than further chords
                    slow = done = true;
                } else {
                    // a side searched in full moves to its lowest sample; where only
                    // neighbours were taken, to the lower neighbour a few times, then
                    // the side is searched in full
                    const bool step = walks++ < kRefWalks;
                    newA = betL && (fullL || step);
                    newB = betR && (fullR || step);
                    if (newA) a = my.k[0];
                    if (newB) b = my.k[1];
                    // where the chord changed, start from the neighbours again
                    const bool same = !newA && !newB;
                    fullL = lowL ? !newA : fullL && same;
                    fullR = lowR ? !newB : fullR && same;
                }
            }
            __syncwarp();
        }
        if (!done) slow = true;
        for (unsigned sl = __ballot_sync(kFull, slow); sl; sl &= sl - 1) {
            const int o = __ffs(sl) - 1;
            int fa, fb;
            double fwa = 0.0, fwb = 0.0;
            ref_full(rl[o], rl[o].L, lane, fa, fb, fwa, fwb);
            if (lane == o) {
                a = fa;
                b = fb;
                wa = fwa;
                wb = fwb;
            }
            ++n_full;
        }
        if (act) {
            RefineOut o;
            o.a = a;
            o.b = b;
            o.pad = 0;
            if (a >= 0) {
                const double xa = (double)(a - m0), xb = (double)(b - m0);
                o.q = (xb * wa - xa * wb) / (xb - xa);
                o.ok = 1;
            } else {
                o.q = INFINITY;
                o.ok = 0;
            }
            P.refined[(long long)qi * kNodeCand + c] = o;
        }
        __syncwarp();
    }
    n_spot = __reduce_add_sync(kFull, n_spot);
    if (lane == 0) {
        if (n_ref) atomicAdd(P.counters + C_REFINED, (unsigned long long)n_ref);
        if (n_full) atomicAdd(P.counters + C_REFFULL, (unsigned long long)n_full);
        if (n_spot) atomicAdd(P.counters + C_FP64, (unsigned long long)n_spot);
    }
}

cudaError_t launch_refine_lanes(const Pipe &p, int level, int phase, int sms, long long max_work,
                                cudaStream_t s) {
    const long long want = (max_work + kRefWarps - 1) / kRefWarps, most = (long long)sms * 8;
    k_refine_lanes<<<(unsigned)(want < most ? want : most), 32 * kRefWarps, 0, s>>>(p, level, phase);
    return cudaGetLastError();
}

}  // namespace cvx
