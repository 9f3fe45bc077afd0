// Primal-dual interior-point AC optimal power flow, one scenario per CTA
// (Section II-B-1: a contingency is severe when the OPF does not converge or
// its solution violates an operational limit).
//
// Algorithm: the MIPS primal-dual interior-point method (Wang, Murillo-Sanchez,
// Zimmerman, Thomas 2007) in polar coordinates, x = [Va, Vm, Pg, Qg], cost
// sum c2 (B Pg)^2 + c1 B Pg + c0, equalities = bus power balance and the
// reference angle, inequalities = |S|^2 flow limits at both branch ends and
// box bounds on Vm, Pg, Qg.  Start Va = 0, Vm = 1, Pg = (Pmin + Pmax)/2,
// Qg = 0, z = max(-h, 1), mu = 1/z, lam = 0; step factor 0.99995, centring
// sigma = 0.1; stop when the feasibility, gradient, complementarity and cost
// conditions are all below tol, at most max_it iterations.
//
// GB300 design:
//  * persistent grid: each CTA pulls scenarios from an atomic counter, so
//    scenarios with uneven iteration counts never idle a CTA;
//  * outaged elements are masked, the network pattern is kept: an outaged
//    branch contributes numeric zeros and its flow rows are inactive, an
//    outaged generator's variables are decoupled and its bound rows inactive;
//  * the Newton system is reduced exactly before factorisation: the generator
//    variables (diagonal in the Hessian) are eliminated into the multiplier
//    diagonal, and the reference-angle row is replaced by dVa_ref = 0 (its
//    multiplier step is recovered from its own Newton row afterwards).  What
//    remains has one 4x4 block [dVa, dVm, dlamP, dlamQ] per bus and the bus
//    graph as block pattern;
//  * that matrix is factorised as a block LDL^T on ONE symbolic analysis per
//    network (minimum-degree order, elimination tree, fill pattern and
//    left-looking update lists, built on the host at load time), with the
//    4x4 pivot blocks inverted by LU with partial pivoting.  Columns
//    of one elimination-tree level are independent, so a level is one
//    parallel step of the CTA: its block updates are cut into equal shares
//    for eight groups of 16 threads, an entry of the target per thread.  The
//    narrow upper levels leave most threads at barriers, so CTAs are small
//    (128 threads) and four are resident per SM to overlap one another's waits;
//  * every branch quantity (flows, first and second derivatives of both end
//    powers, the weighted 4x4 Hessian) is computed once per iteration by one
//    thread from the branch's own four voltage variables and gathered by
//    buses and blocks, deterministically (no atomics);
//  * main-island form (an extension after Sections II-A, V-A and VI): an
//    islanded scenario gets the OPF of the component whose in-service
//    generators have the largest total Pmax.  Buses outside it are masked like
//    outaged elements (identity blocks, no rows, no constraints, their load
//    shed), so the pattern and the symbolic analysis stay those of the
//    network; the reference moves to the island's largest unit when the
//    original one lies outside.  A generator bus carries the generator's
//    multiplier diagonal, so its reference block stays a regular pivot
//    wherever it falls in the elimination order.
#include <cmath>

#include "cs_internal.h"

namespace {

#ifndef CS_OPF_THREADS
#define CS_OPF_THREADS 128
#endif
#ifndef CS_OPF_CTAS
#define CS_OPF_CTAS 4
#endif
constexpr int kThreads = CS_OPF_THREADS;   // threads per scenario CTA
constexpr int kCtasPerSm = CS_OPF_CTAS;    // resident CTAs per SM the register budget is sized for
constexpr int kWarps = kThreads / 32;
constexpr int kGroups = kThreads / 16;     // groups of 16 threads, one thread per entry of a 4x4 block
constexpr int kBatch = 4;                  // block updates whose loads are in flight together
constexpr int kRec = 34;     // doubles per branch record
constexpr double kXi = 0.99995;
constexpr double kSigma = 0.1;
constexpr double kLimitTol = 1e-6;
constexpr int kRefineSteps = 3;              // FP64 iterative refinement steps per Newton solve (at most)
constexpr double kRefineTol = 4.0 * 2.220446049250313e-16;   // refinement done: backward error at rounding level
constexpr double kBackwardTol = 1e-15;       // componentwise backward error accepted from the block solve + GMRES
constexpr int kDenseMax = 1024;              // dense fallback for reduced systems up to this order
constexpr int kLossBits = 30;                // most that z . mu can shrink in one iteration, bits (rounded up)
constexpr int kStateBits = 100;              // largest |x| of a point that could still converge, bits (see sc.lost)
constexpr int kPanel = 8;                    // panel width of the dense fallback's blocked LU
constexpr int kGmresM = 8;                   // GMRES iterations per Newton solve (at most)
constexpr int kRedMax = kGmresM + 1 > 10 ? kGmresM + 1 : 10;   // values per block reduction (at most)

// Branch record.  Every branch quantity depends on the two end angles through theta = Va_f -
// Va_t alone, so derivatives are kept by (theta, Vm_f, Vm_t); those by Va_t are those by theta with
// the sign changed.  R_H: second derivatives (theta theta, theta f, theta t, f f, f t, t t);
// R_DF, R_DT: complex derivatives of the powers at the f and t ends; R_G: gradients of the two
// |S|^2; R_L, R_N: contributions to the Lagrangian gradient and to N; R_S: S_f, S_t.
constexpr int R_H = 0, R_DF = 6, R_DT = 12, R_G = 18, R_L = 24, R_N = 27, R_S = 30;

// x with its sign changed (on the integer pipe)
__device__ __forceinline__ double neg(double x) {
    return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}
__device__ __forceinline__ bool non_finite(double x) { return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000; }

// Maxima of non-negative doubles run on the integer pipe: as 64-bit integers they have the same
// order, +0 below everything, NaN above everything (a NaN in one of the maxima makes the
// iteration fail, as it should).  An FP64 comparison would hold the sub-partition's FP64 pipe for
// as long as a multiply-add does.
typedef unsigned long long key_t64;
__device__ __forceinline__ key_t64 abs_key(double x) {
    return (key_t64)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ key_t64 pos_key(double x) {      // negative values count as 0
    const long long v = __double_as_longlong(x);
    return v < 0 ? 0ull : (key_t64)v;
}
__device__ __forceinline__ double key_value(key_t64 k) { return __longlong_as_double((long long)k); }
__device__ __forceinline__ key_t64 warp_max_key(key_t64 k) {
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    return ((key_t64)mh << 32) | ml;
}

struct Lay {
    // bus
    int Va, Vm, lP, lQ, zu, zl, rzu, rzl, muu, mul, gP, gQ, NVa, NVm, DP, DQ, rP, rQ, dzu, dzl, dmuu, dmul;
    // gen
    int Pg, Qg, gz, gmu, gdz, gdmu, grz, MP, MQ, NP, NQ, dPg, dQg;   // MP, MQ: reciprocals of the pivots
    // branch
    int zf, zt, muf, mut, hf, ht, rzf, rzt, dzf, dzt, dmuf, dmut, rec;   // rz..: 1 / z
    // KKT: assembled blocks (Kb, Kd) kept for refinement, factor (Ub, Lb, Db, Di), vectors
    int Kb, Kd, Ub, Lb, Db, Di, x, bv, rv, cs, drs, dpiv;   // drs, dpiv: dense backstop's row scales, pivots
    int kv, kz, gx0, gxb, gr;   // GMRES: Krylov basis, preconditioned basis, start, best iterate, work
    int uf, cap, dead;          // main island: union-find parents (int), capacity per root, bus flags (bytes)
    long dense;                 // dense fallback matrix (4nb)^2, -1 if the network is too large
    long total;
};

Lay make_layout(const DevNet& n) {
    Lay L{};
    int o = 0;
    auto take = [&](int cnt) { int r = o; o += cnt; return r; };
    int nb = n.nb, ng = n.ng, nbr = n.nbr;
    L.Va = take(nb); L.Vm = take(nb); L.lP = take(nb); L.lQ = take(nb); L.zu = take(nb); L.zl = take(nb);
    L.muu = take(nb); L.mul = take(nb); L.gP = take(nb); L.gQ = take(nb); L.rzu = take(nb); L.rzl = take(nb);
    L.NVa = take(nb); L.NVm = take(nb); L.DP = take(nb); L.DQ = take(nb); L.rP = take(nb); L.rQ = take(nb);
    L.dzu = take(nb); L.dzl = take(nb); L.dmuu = take(nb); L.dmul = take(nb);
    L.Pg = take(ng); L.Qg = take(ng); L.gz = take(4 * ng); L.gmu = take(4 * ng); L.gdz = take(4 * ng);
    L.gdmu = take(4 * ng); L.MP = take(ng); L.MQ = take(ng); L.NP = take(ng); L.NQ = take(ng);
    L.grz = take(4 * ng); L.dPg = take(ng); L.dQg = take(ng);
    L.zf = take(nbr); L.zt = take(nbr); L.muf = take(nbr); L.mut = take(nbr); L.hf = take(nbr); L.ht = take(nbr);
    L.dzf = take(nbr); L.dzt = take(nbr); L.dmuf = take(nbr); L.dmut = take(nbr);
    L.rzf = take(nbr); L.rzt = take(nbr);
    o = (o + 15) & ~15;
    L.rec = take(kRec * nbr);
    o = (o + 15) & ~15;
    L.Kb = take(16 * n.nL); L.Kd = take(16 * nb);
    L.Ub = take(16 * n.nL); L.Lb = take(16 * n.nL); L.Db = take(16 * nb); L.Di = take(16 * nb);
    L.x = take(4 * nb); L.bv = take(4 * nb); L.rv = take(4 * nb); L.cs = take(4 * nb);
    L.drs = take(4 * nb); L.dpiv = take(2 * nb);
    L.kv = take(4 * nb * (kGmresM + 1)); L.kz = take(4 * nb * kGmresM);
    L.gx0 = take(4 * nb); L.gxb = take(4 * nb); L.gr = take(4 * nb);
    L.uf = take((nb + 1) / 2); L.cap = take(nb); L.dead = take((nb + 7) / 8);
    o = (o + 31) & ~31;
    if (4 * nb <= kDenseMax) {
        L.dense = o;
        L.total = (long)o + (long)16 * nb * nb;
    } else {
        L.dense = -1;
        L.total = o;
    }
    L.total = (L.total + 31) & ~31L;
    return L;
}

// ------------------------------------------------------------------ helpers --
struct RedBuf {
    double v[kRedMax][kWarps];
};

__device__ __forceinline__ double red_op(int op, double a, double b) {
    return op == 1 ? a + b : (op == 0 ? fmax(a, b) : fmin(a, b));
}

// reduce K values per thread: ops[k] = 0 max, 1 sum, 2 min.  Result broadcast in out[]
// (shared).  Warp shuffles, then one pass over the per-warp results.
template <int K>
__device__ void block_reduce(RedBuf& rb, double (&val)[K], const int (&ops)[K], double* out) {
    static_assert(K <= kRedMax, "block_reduce: more values than RedBuf and Scal::red hold");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = 0; k < K; ++k) {
        double v = val[k];
        for (int off = 16; off; off >>= 1) v = red_op(ops[k], v, __shfl_xor_sync(0xffffffffu, v, off));
        val[k] = v;
    }
    if (kWarps == 1) {
        if (tid == 0)
            for (int k = 0; k < K; ++k) out[k] = val[k];
        __syncthreads();
        return;
    }
    if (lane == 0)
        for (int k = 0; k < K; ++k) rb.v[k][warp] = val[k];
    __syncthreads();
    if (tid == 0) {
        for (int k = 0; k < K; ++k) {
            double v = rb.v[k][0];
            for (int w = 1; w < kWarps; ++w) v = red_op(ops[k], v, rb.v[k][w]);
            out[k] = v;
        }
    }
    __syncthreads();
}

// Inverse of the symmetric part of a 4x4 pivot block: LU factorisation with
// partial pivoting, forward/back substitution for each column of the identity,
// then symmetrisation of the result.  (Near the end of the interior-point
// iteration some pivot blocks are nearly singular; the LU-based inverse keeps
// the error low-rank, which the iterative refinement removes, where a
// Gauss-Jordan inverse did not.)  Two forms of the same steps:
//  * inv4_wide, four lanes a pivot, for levels with many columns: each lane repeats the
//    factorisation and solves for column q; ~77 FP64 instructions for eight pivots per warp;
//  * inv4, sixteen lanes a pivot, one entry each (lane e = 4 r + c: a = A(r, c), the result
//    Ainv(r, c)), for the top of the tree, where every level waits for one pivot's chain of
//    dependent FP64 instructions: ~41 of them.
// ok becomes false, on all lanes of the group (mask grp), if a pivot is exactly zero or not finite.
__device__ void inv4_wide(const double* A, double* Ainv, int q, unsigned grp, bool& ok) {
    double a[4][4], dinv[4];
    int piv[4] = {0, 1, 2, 3};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        a[r][r] = A[5 * r];
#pragma unroll
        for (int c = 0; c < r; ++c) a[c][r] = a[r][c] = 0.5 * (A[4 * r + c] + A[4 * c + r]);
    }
    ok = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int p = k;
        key_t64 best = abs_key(a[k][k]);
        if (best > 0x7ff0000000000000ull) ok = false;   // NaN on the diagonal
#pragma unroll
        for (int r = k + 1; r < 4; ++r) {
            const key_t64 v = abs_key(a[r][k]);
            if (v > best && v <= 0x7ff0000000000000ull) { best = v; p = r; }
        }
        if (best == 0ull || best >= 0x7ff0000000000000ull) ok = false;
#pragma unroll
        for (int r = k + 1; r < 4; ++r)
            if (p == r) {                               // rows k and p trade places
#pragma unroll
                for (int c = 0; c < 4; ++c) { const double t = a[k][c]; a[k][c] = a[r][c]; a[r][c] = t; }
                const int t = piv[k]; piv[k] = piv[r]; piv[r] = t;
            }
        dinv[k] = 1.0 / a[k][k];
#pragma unroll
        for (int r = k + 1; r < 4; ++r) {
            a[r][k] *= dinv[k];
#pragma unroll
            for (int c = k + 1; c < 4; ++c) a[r][c] -= a[r][k] * a[k][c];
        }
    }
    double y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        double v = (piv[i] == q) ? 1.0 : 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) v -= a[i][k] * y[k];
        y[i] = v;
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        double v = y[i];
#pragma unroll
        for (int k = i + 1; k < 4; ++k) v -= a[i][k] * y[k];
        y[i] = v * dinv[i];
    }
    // symmetrised below (see inv4): entry (i, q) meets entry (q, i), which lane i holds as its y[q]
    const int base = threadIdx.x & 28;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        double t = 0.0;
#pragma unroll
        for (int s = 0; s < 4; ++s) {                   // lane q sends y[s] to the lane that wants it
            const double v = __shfl_sync(grp, y[s], base + i);
            if (s == q) t = v;
        }
        Ainv[4 * i + q] = 0.5 * (y[i] + t);
    }
}

__device__ double inv4(double a, unsigned grp, bool& ok) {
    const int lane = threadIdx.x & 31, e = lane & 15, base = lane & 16, r = e >> 2, c = e & 3;
    a = 0.5 * (a + __shfl_sync(grp, a, base + 4 * c + r));
    double dinv[4];
    int perm = 0x3210;                                  // original row of row i in bits 4 i .. 4 i + 3
    ok = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        double col[4];
#pragma unroll
        for (int i = k; i < 4; ++i) col[i] = __shfl_sync(grp, a, base + 4 * i + k);
        int p = k;
        key_t64 best = abs_key(col[k]);
        if (best > 0x7ff0000000000000ull) ok = false;   // NaN on the diagonal
#pragma unroll
        for (int i = k + 1; i < 4; ++i) {
            const key_t64 v = abs_key(col[i]);
            if (v > best && v <= 0x7ff0000000000000ull) { best = v; p = i; }
        }
        if (best == 0ull || best >= 0x7ff0000000000000ull) ok = false;
        const double piv = p == k ? col[k] : p == k + 1 ? col[k < 3 ? k + 1 : 3] : p == 2 ? col[2] : col[3];
        const int src = r == k ? p : r == p ? k : r;    // rows k and p trade places
        a = __shfl_sync(grp, a, base + 4 * src + c);
        const int pk = (perm >> (4 * k)) & 15, pp = (perm >> (4 * p)) & 15;
        perm = (perm & ~(15 << (4 * k)) & ~(15 << (4 * p))) | (pp << (4 * k));
        if (p != k) perm |= pk << (4 * p);
        dinv[k] = 1.0 / piv;
        double mine = col[k];                           // column k of this lane's row after the exchange
#pragma unroll
        for (int i = k; i < 4; ++i)
            if (src == i) mine = col[i];
        const double m = mine * dinv[k];
        const double u = __shfl_sync(grp, a, base + 4 * k + c);
        if (r > k) a = (c == k) ? m : (c > k ? a - m * u : a);
    }
    double y = ((perm >> (4 * r)) & 15) == c ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double yk = __shfl_sync(grp, y, base + 4 * k + c), l = __shfl_sync(grp, a, base + 4 * r + k);
        if (r > k) y -= l * yk;
    }
#pragma unroll
    for (int k = 3; k >= 0; --k) {
        const double xk = __shfl_sync(grp, y, base + 4 * k + c) * dinv[k], u = __shfl_sync(grp, a, base + 4 * r + k);
        if (r == k) y = xk;
        if (r < k) y -= u * xk;
    }
    // Symmetrise.  Only the lower blocks are stored and updated with L(i,k) U(j,k)^T,
    // which assumes a symmetric pivot inverse; an LU-based inverse of a nearly singular
    // symmetric block is far from symmetric in rounding, and the factorisation would
    // then not be a consistent L D L^T (refinement stalls).
    return 0.5 * (y + __shfl_sync(grp, y, base + 4 * c + r));
}

// One branch at the current iterate: flows, derivatives, weighted Hessian,
// Lagrangian-gradient and N contributions.  If init, also sets z, mu of the
// two flow rows from h (z = max(-h, 1), mu = gamma / z).
//
// With theta = Va_f - Va_t, a = conj(yft) e^{j theta} and c = conj(ytf) e^{-j theta}:
//   S_f = Vf^2 conj(yff) + Vf Vt a,   S_t = Vt^2 conj(ytt) + Vf Vt c,
// and every derivative is one of a few products of these.  The FP64 pipe is the OPF's bound
// (one warp instruction per 16 cycles and SM, whatever its lanes), so what counts here is the
// number of FP64 instructions: ~200 with one sincos and two reciprocals, where the product rule
// over four complex variables took ~1,400.  With it, the reductions' comparisons on the integer
// pipe and stored reciprocals, 10,000 pairs (118 buses) went from 1,329 to 1,198 ms, one
// scenario's OPF from 21.6 to 18.7 ms.
__device__ __forceinline__ void eval_branch(const DevNet& net, int b, double* W, const Lay& L, double gamma,
                                            bool init) {
    const int f = net.f[b], t = net.t[b];
    const double vf = W[L.Vm + f], vt = W[L.Vm + t];
    double sn, cs;
    sincos(W[L.Va + f] - W[L.Va + t], &sn, &cs);
    const cplx yff = net.yff[b], yft = net.yft[b], ytf = net.ytf[b], ytt = net.ytt[b];
    const cplx a = cm(yft.re * cs + yft.im * sn, yft.re * sn - yft.im * cs);
    const cplx c = cm(ytf.re * cs - ytf.im * sn, neg(ytf.re * sn + ytf.im * cs));
    const double p = vf * vt;
    const cplx A = p * a, C = p * c;
    const cplx Sf = cm(vf * vf * yff.re + A.re, A.im - vf * vf * yff.im);
    const cplx St = cm(vt * vt * ytt.re + C.re, C.im - vt * vt * ytt.im);
    // derivatives by (theta, Vm_f, Vm_t); those of S_f by theta are j A, of S_t -j C
    const double df[6] = {neg(A.im), A.re, 2.0 * vf * yff.re + vt * a.re, vt * a.im - 2.0 * vf * yff.im,
                          vf * a.re, vf * a.im};
    const double dt[6] = {C.im, neg(C.re), vt * c.re, vt * c.im,
                          2.0 * vt * ytt.re + vf * c.re, vf * c.im - 2.0 * vt * ytt.im};
    const double smax2 = net.smax2[b];
    const double hf = abs2(Sf) - smax2, ht = abs2(St) - smax2;
    double muf, mut, rzf, rzt;
    if (init) {
        const double zf = fmax(-hf, 1.0), zt = fmax(-ht, 1.0);
        rzf = 1.0 / zf;
        rzt = 1.0 / zt;
        muf = gamma * rzf;
        mut = gamma * rzt;
        W[L.zf + b] = zf; W[L.zt + b] = zt; W[L.muf + b] = muf; W[L.mut + b] = mut;
    } else {
        rzf = 1.0 / W[L.zf + b];
        rzt = 1.0 / W[L.zt + b];
        muf = W[L.muf + b]; mut = W[L.mut + b];
    }
    W[L.rzf + b] = rzf;
    W[L.rzt + b] = rzt;
    W[L.hf + b] = hf;
    W[L.ht + b] = ht;
    const double lPf = W[L.lP + f], lQf = W[L.lQ + f], lPt = W[L.lP + t], lQt = W[L.lQ + t];
    double gf[3], gt[3], lg[3], ng[3];
    const double nf = (muf * hf + gamma) * rzf, nt = (mut * ht + gamma) * rzt;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        gf[q] = 2.0 * (Sf.re * df[2 * q] + Sf.im * df[2 * q + 1]);
        gt[q] = 2.0 * (St.re * dt[2 * q] + St.im * dt[2 * q + 1]);
        lg[q] = lPf * df[2 * q] + lQf * df[2 * q + 1] + lPt * dt[2 * q] + lQt * dt[2 * q + 1] + muf * gf[q] +
                mut * gt[q];
        ng[q] = nf * gf[q] + nt * gt[q];
    }
    // weights: lamP Re d2S + lamQ Im d2S + 2 mu Re(conj(S) d2S) = wr Re d2S + wi Im d2S
    const double m2f = 2.0 * muf, m2t = 2.0 * mut;
    const double wfr = lPf + m2f * Sf.re, wfi = lQf + m2f * Sf.im;
    const double wtr = lPt + m2t * St.re, wti = lQt + m2t * St.im;
    const double qf = wfr * a.re + wfi * a.im, rf = wfi * a.re - wfr * a.im;      // of a and j a
    const double qt = wtr * c.re + wti * c.im, rt = wti * c.re - wtr * c.im;      // of c and j c
    double H[6] = {neg(p * (qf + qt)), vt * (rf - rt), vf * (rf - rt), 2.0 * (wfr * yff.re - wfi * yff.im), qf + qt,
                   2.0 * (wtr * ytt.re - wti * ytt.im)};
    const double bf = muf * rzf, bt = mut * rzt;
#pragma unroll
    for (int x = 0, e = 0; x < 3; ++x) {
        const double fr = m2f * df[2 * x], fi = m2f * df[2 * x + 1], fg = bf * gf[x];
        const double tr = m2t * dt[2 * x], ti = m2t * dt[2 * x + 1], tg = bt * gt[x];
#pragma unroll
        for (int y = x; y < 3; ++y, ++e)
            H[e] += fr * df[2 * y] + fi * df[2 * y + 1] + fg * gf[y] + tr * dt[2 * y] + ti * dt[2 * y + 1] +
                    tg * gt[y];
    }
    double2* rec = reinterpret_cast<double2*>(W + L.rec + (size_t)kRec * b);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        rec[R_H / 2 + q] = make_double2(H[2 * q], H[2 * q + 1]);
        rec[R_DF / 2 + q] = make_double2(df[2 * q], df[2 * q + 1]);
        rec[R_DT / 2 + q] = make_double2(dt[2 * q], dt[2 * q + 1]);
    }
    rec[R_G / 2] = make_double2(gf[0], gf[1]);
    rec[R_G / 2 + 1] = make_double2(gf[2], gt[0]);
    rec[R_G / 2 + 2] = make_double2(gt[1], gt[2]);
    rec[R_L / 2] = make_double2(lg[0], lg[1]);
    rec[R_L / 2 + 1] = make_double2(lg[2], ng[0]);
    rec[R_L / 2 + 2] = make_double2(ng[1], ng[2]);
    rec[R_S / 2] = make_double2(Sf.re, Sf.im);
    rec[R_S / 2 + 1] = make_double2(St.re, St.im);
}

// Sum of the block updates u0 .. u1 - 1 for entry (r, c) of their target: sum of L(i,k) U(j,k)^T.
// The blocks come from the L2 as often as from the L1, so kBatch updates' loads are issued before
// the first multiply-add.
__device__ __forceinline__ double run_sum(const DevNet& net, const double* W, const Lay& L, int u0, int u1, int r,
                                          int c) {
    double acc = 0.0;
    const double* Lr = W + L.Lb + 4 * r;
    const double* Uc = W + L.Ub + 4 * c;
    int u = u0;
    for (; u + kBatch <= u1; u += kBatch) {
        double2 l[kBatch][2], w[kBatch][2];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            const double2* la = reinterpret_cast<const double2*>(Lr + 16 * __ldg(net.sh_a + u + q));
            const double2* ub = reinterpret_cast<const double2*>(Uc + 16 * __ldg(net.sh_b + u + q));
            l[q][0] = la[0]; l[q][1] = la[1]; w[q][0] = ub[0]; w[q][1] = ub[1];
        }
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
            acc += l[q][0].x * w[q][0].x + l[q][0].y * w[q][0].y + l[q][1].x * w[q][1].x + l[q][1].y * w[q][1].y;
    }
    for (; u < u1; ++u) {
        const double2* la = reinterpret_cast<const double2*>(Lr + 16 * __ldg(net.sh_a + u));
        const double2* ub = reinterpret_cast<const double2*>(Uc + 16 * __ldg(net.sh_b + u));
        const double2 l0 = la[0], l1 = la[1], w0 = ub[0], w1 = ub[1];
        acc += l0.x * w0.x + l0.y * w0.y + l1.x * w1.x + l1.y * w1.y;
    }
    return acc;
}

// Solve (L D L^T) v = v in place for the 4-vector-per-bus array v (new order):
// forward by elimination-tree levels, block diagonal, backward by levels.
//
// A narrow level (the top of the tree: 21 of the 118-bus network's 26 levels hold one column)
// takes a warp per column with eight groups of four lanes: a group takes every eighth block of
// the column, a lane one of its four rows, and three shuffle additions sum the groups.  An FP64
// instruction costs its sub-partition 64 cycles with one lane or with 32, so a column of up to
// eight blocks costs 4 + 3 of them; with a lane per block and the four row sums reduced one after
// another it was 16 + 20.
__device__ void ldl_solve(const DevNet& net, const double* W, const Lay& L, double* v) {
    const int tid = threadIdx.x, nb = net.nb, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, r = lane & 3;
    for (int lev = 0; lev < net.nlevels; ++lev) {
        const int c0 = __ldg(net.lev_ptr + lev), c1 = __ldg(net.lev_ptr + lev + 1);
        if (c1 - c0 <= kWarps) {
            if (warp < c1 - c0) {
                const int j = __ldg(net.lev_col + c0 + warp);
                double acc = 0.0;
                for (int e = __ldg(net.Lrowptr + j) + g; e < __ldg(net.Lrowptr + j + 1); e += 8) {
                    const double2* Lq = reinterpret_cast<const double2*>(W + L.Lb + 16 * __ldg(net.Lrowblk + e) + 4 * r);
                    const double2* y = reinterpret_cast<const double2*>(v + 4 * __ldg(net.Lrowcol + e));
                    const double2 l0 = Lq[0], l1 = Lq[1], y0 = y[0], y1 = y[1];
                    acc += l0.x * y0.x + l0.y * y0.y + l1.x * y1.x + l1.y * y1.y;
                }
                for (int off = 16; off >= 4; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                if (lane < 4) v[4 * j + lane] -= acc;
            }
        } else {
            for (int w = tid; w < 4 * (c1 - c0); w += kThreads) {
                const int j = __ldg(net.lev_col + c0 + (w >> 2)), q = w & 3;
                double acc = v[4 * j + q];
                for (int e = __ldg(net.Lrowptr + j); e < __ldg(net.Lrowptr + j + 1); ++e) {
                    const double* Lq = W + L.Lb + 16 * __ldg(net.Lrowblk + e) + 4 * q;
                    const double* y = v + 4 * __ldg(net.Lrowcol + e);
                    acc -= Lq[0] * y[0] + Lq[1] * y[1] + Lq[2] * y[2] + Lq[3] * y[3];
                }
                v[4 * j + q] = acc;
            }
        }
        __syncthreads();
    }
    for (int w0 = 0; w0 < 4 * nb; w0 += kThreads) {          // four lanes per bus
        const int w = w0 + tid, j = w >> 2;
        double t = 0.0;
        if (w < 4 * nb) {
            const double* Di = W + L.Di + 4 * w;             // row w & 3 of block j
            const double* y = v + 4 * j;
            t = Di[0] * y[0] + Di[1] * y[1] + Di[2] * y[2] + Di[3] * y[3];
        }
        __syncwarp();
        if (w < 4 * nb) v[w] = t;
    }
    __syncthreads();
    for (int lev = net.nlevels - 1; lev >= 0; --lev) {
        const int c0 = __ldg(net.lev_ptr + lev), c1 = __ldg(net.lev_ptr + lev + 1);
        if (c1 - c0 <= kWarps) {
            if (warp < c1 - c0) {
                const int j = __ldg(net.lev_col + c0 + warp);
                double acc = 0.0;
                for (int e = __ldg(net.Lcolptr + j) + g; e < __ldg(net.Lcolptr + j + 1); e += 8) {
                    const double* Lq = W + L.Lb + 16 * e + r;
                    const double* xi = v + 4 * __ldg(net.Lrow + e);
                    acc += Lq[0] * xi[0] + Lq[4] * xi[1] + Lq[8] * xi[2] + Lq[12] * xi[3];
                }
                for (int off = 16; off >= 4; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                if (lane < 4) v[4 * j + lane] -= acc;
            }
        } else {
            for (int w = tid; w < 4 * (c1 - c0); w += kThreads) {
                const int j = __ldg(net.lev_col + c0 + (w >> 2)), q = w & 3;
                double acc = v[4 * j + q];
                for (int e = __ldg(net.Lcolptr + j); e < __ldg(net.Lcolptr + j + 1); ++e) {
                    const double* Lq = W + L.Lb + 16 * e + q;
                    const double* xi = v + 4 * __ldg(net.Lrow + e);
                    acc -= Lq[0] * xi[0] + Lq[4] * xi[1] + Lq[8] * xi[2] + Lq[12] * xi[3];
                }
                v[4 * j + q] = acc;
            }
        }
        __syncthreads();
    }
}

// r = b - K x with the assembled (unfactored) blocks, one thread per (bus, row),
// and the componentwise backward error of x, max_i |r_i| / (|K| |x| + |b|)_i
// (on every thread).  Only the blocks that hold a branch are read: two in three of the
// factor's blocks are fill, zero in K.
__device__ double kkt_residual(const DevNet& net, const double* W, const Lay& L, RedBuf& rb, const double* x,
                               double* r) {
    const int tid = threadIdx.x, nb = net.nb;
    key_t64 worst = 0;
    for (int w = tid; w < 4 * nb; w += kThreads) {
        const int i = w >> 2, rr = w & 3;
        const double* Kd = W + L.Kd + 4 * w;
        const double* xi = x + 4 * i;
        double acc = W[L.bv + w], sc = fabs(acc);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            acc = fma(-Kd[c], xi[c], acc);
            sc = fma(fabs(Kd[c]), fabs(xi[c]), sc);
        }
        for (int e = __ldg(net.adj_ptr + i); e < __ldg(net.adj_ptr + i + 1); ++e) {
            const int code = __ldg(net.adj_blk + e);
            const double* Kq = W + L.Kb + 16 * (code >> 1) + ((code & 1) ? rr : 4 * rr);
            const int st = (code & 1) ? 4 : 1;
            const double* xk = x + 4 * __ldg(net.adj_col + e);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double k = Kq[c * st], xc = xk[c];
                acc = fma(-k, xc, acc);
                sc = fma(fabs(k), fabs(xc), sc);
            }
        }
        r[w] = acc;
        // |acc| / sc; 0 / 0 counts as 0, a non-finite quotient as infinite
        key_t64 be = abs_key(sc) > 0 ? abs_key(acc / sc) : (abs_key(acc) ? 0x7ff0000000000000ull : 0ull);
        if (be > 0x7ff0000000000000ull) be = 0x7ff0000000000000ull;
        worst = max(worst, be);
    }
    worst = warp_max_key(worst);
    if ((tid & 31) == 0) rb.v[0][tid >> 5] = key_value(worst);
    __syncthreads();
    worst = 0;
    for (int w = 0; w < kWarps; ++w) worst = max(worst, abs_key(rb.v[0][w]));
    __syncthreads();
    return key_value(worst);
}

// y = K x with the assembled blocks (x, y: 4-vectors per bus, new order).
__device__ void kkt_matvec(const DevNet& net, const double* W, const Lay& L, const double* x, double* y) {
    const int tid = threadIdx.x, nb = net.nb;
    for (int w = tid; w < 4 * nb; w += kThreads) {
        const int i = w >> 2, rr = w & 3;
        const double* Kd = W + L.Kd + 4 * w;
        const double* xi = x + 4 * i;
        double acc = Kd[0] * xi[0] + Kd[1] * xi[1] + Kd[2] * xi[2] + Kd[3] * xi[3];
        for (int e = __ldg(net.adj_ptr + i); e < __ldg(net.adj_ptr + i + 1); ++e) {
            const int code = __ldg(net.adj_blk + e);
            const double* Kq = W + L.Kb + 16 * (code >> 1) + ((code & 1) ? rr : 4 * rr);
            const int st = (code & 1) ? 4 : 1;
            const double* xk = x + 4 * __ldg(net.adj_col + e);
            acc += Kq[0] * xk[0] + Kq[st] * xk[1] + Kq[2 * st] * xk[2] + Kq[3 * st] * xk[3];
        }
        y[w] = acc;
    }
    __syncthreads();
}

struct GmresShared {
    double H[kGmresM + 1][kGmresM];
    double g[kGmresM + 1], c[kGmresM], s[kGmresM], y[kGmresM];
};

// GMRES on K d = r, right-preconditioned by the block LDL^T factors, starting
// from the current solution x (r = b - K x in rv, omega0 its backward error).
// When the pivot blocks are nearly singular, the factors are exact except in
// a subspace of small dimension, so a few Krylov steps remove what plain
// refinement cannot.  Arnoldi with classical Gram-Schmidt applied twice; the
// candidate solution is formed and its componentwise backward error checked
// after every step; x ends as the best candidate.  Returns its backward error.
__device__ __noinline__ double kkt_gmres(const DevNet& net, double* W, const Lay& L, RedBuf& rb, double* red, GmresShared& gs,
                            double omega0) {
    const int tid = threadIdx.x, N = 4 * net.nb;
    double* x = W + L.x;
    double* x0 = W + L.gx0;
    double* xb = W + L.gxb;
    double* V = W + L.kv;
    double* Z = W + L.kz;
    double* t = W + L.gr;
    const int ops_sum[1] = {1};
    int ops_h[kGmresM + 1];
    for (int i = 0; i <= kGmresM; ++i) ops_h[i] = 1;
    {
        double ss = 0.0;
        for (int w = tid; w < N; w += kThreads) {
            x0[w] = x[w];
            xb[w] = x[w];
            const double rw = W[L.rv + w];
            ss += rw * rw;
        }
        double v1[1] = {ss};
        block_reduce<1>(rb, v1, ops_sum, red);
    }
    const double beta = sqrt(red[0]);
    if (!(beta > 0.0) || !isfinite(beta)) return omega0;
    for (int w = tid; w < N; w += kThreads) V[w] = W[L.rv + w] / beta;
    if (tid == 0) {
        for (int i = 0; i <= kGmresM; ++i) gs.g[i] = 0.0;
        gs.g[0] = beta;
    }
    __syncthreads();
    double best = omega0;
    for (int j = 0; j < kGmresM; ++j) {
        double* zj = Z + (size_t)j * N;
        for (int w = tid; w < N; w += kThreads) zj[w] = V[(size_t)j * N + w];
        __syncthreads();
        ldl_solve(net, W, L, zj);
        kkt_matvec(net, W, L, zj, t);
        for (int pass = 0; pass < 2; ++pass) {              // classical Gram-Schmidt, twice
            double h[kGmresM + 1];
            for (int i = 0; i <= kGmresM; ++i) h[i] = 0.0;
            for (int w = tid; w < N; w += kThreads) {
                const double tw = t[w];
#pragma unroll
                for (int i = 0; i <= kGmresM; ++i)
                    if (i <= j) h[i] += V[(size_t)i * N + w] * tw;
            }
            block_reduce<kGmresM + 1>(rb, h, ops_h, red);
            for (int w = tid; w < N; w += kThreads) {
                double tw = t[w];
#pragma unroll
                for (int i = 0; i <= kGmresM; ++i)
                    if (i <= j) tw -= red[i] * V[(size_t)i * N + w];
                t[w] = tw;
            }
            if (tid == 0)
                for (int i = 0; i <= j; ++i) gs.H[i][j] = (pass == 0 ? 0.0 : gs.H[i][j]) + red[i];
            __syncthreads();
        }
        double hn;
        {
            double ss = 0.0;
            for (int w = tid; w < N; w += kThreads) ss += t[w] * t[w];
            double v1[1] = {ss};
            block_reduce<1>(rb, v1, ops_sum, red);
            hn = sqrt(red[0]);
        }
        if (tid == 0) {                                     // Givens rotations, least-squares solve
            gs.H[j + 1][j] = hn;
            for (int i = 0; i < j; ++i) {
                const double a0 = gs.H[i][j], a1 = gs.H[i + 1][j];
                gs.H[i][j] = gs.c[i] * a0 + gs.s[i] * a1;
                gs.H[i + 1][j] = -gs.s[i] * a0 + gs.c[i] * a1;
            }
            const double d = hypot(gs.H[j][j], gs.H[j + 1][j]);
            gs.c[j] = (d > 0.0) ? gs.H[j][j] / d : 1.0;
            gs.s[j] = (d > 0.0) ? gs.H[j + 1][j] / d : 0.0;
            gs.H[j][j] = d;
            gs.H[j + 1][j] = 0.0;
            gs.g[j + 1] = -gs.s[j] * gs.g[j];
            gs.g[j] = gs.c[j] * gs.g[j];
            for (int i = j; i >= 0; --i) {
                double acc = gs.g[i];
                for (int k = i + 1; k <= j; ++k) acc -= gs.H[i][k] * gs.y[k];
                gs.y[i] = (gs.H[i][i] != 0.0) ? acc / gs.H[i][i] : 0.0;
            }
        }
        __syncthreads();
        if (hn > 0.0)
            for (int w = tid; w < N; w += kThreads) V[(size_t)(j + 1) * N + w] = t[w] / hn;
        for (int w = tid; w < N; w += kThreads) {
            double xw = x0[w];
            for (int i = 0; i <= j; ++i) xw += gs.y[i] * Z[(size_t)i * N + w];
            x[w] = xw;
        }
        __syncthreads();
        const double om = kkt_residual(net, W, L, rb, x, t);
        if (om < best) {
            best = om;
            for (int w = tid; w < N; w += kThreads) xb[w] = x[w];
        }
        if (om <= kBackwardTol || !(hn > 0.0)) break;
        __syncthreads();
    }
    __syncthreads();
    for (int w = tid; w < N; w += kThreads) x[w] = xb[w];
    __syncthreads();
    return best;
}

struct DenseShared {
    unsigned long long val[kWarps];
    int idx[kWarps];
    int piv;
    int nr, nc;                       // rows and columns the current panel's trailing update touches
    double pv;
    unsigned short rows[kDenseMax], cols[kDenseMax];
};

// |a| as an integer of the same order (NaN below everything), so that a pivot search does not
// occupy the FP64 pipe with comparisons
__device__ __forceinline__ unsigned long long abs_bits(double a) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
    return u <= 0x7ff0000000000000ull ? u : 0ull;
}

// append w to a list in shared memory for the lanes with on (any order: the list's entries are
// independent pieces of work)
__device__ __forceinline__ void list_add(unsigned short* list, int* cnt, bool on, int w) {
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (m == 0u) return;
    const int lane = threadIdx.x & 31;
    int at = 0;
    if (lane == 0) at = atomicAdd(cnt, __popc(m));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (on) list[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)w;
}

constexpr int kTri = 32;              // block of the dense triangular solves

// v <- U^{-1} v with the upper triangle of the row-major N x N matrix A (kUpper), or v <- L^{-1} v
// with its unit lower one: blocks of kTri unknowns, one warp per diagonal block (a lane per
// unknown), then every row takes the block's contribution.
template <bool kUpper>
__device__ void dense_tri(const double* A, int N, double* v) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nblk = (N + kTri - 1) / kTri;
    for (int q = 0; q < nblk; ++q) {
        const int b0 = (kUpper ? nblk - 1 - q : q) * kTri, b1 = min(b0 + kTri, N), nb = b1 - b0;
        if (warp == 0) {
            double y = (lane < nb) ? v[b0 + lane] : 0.0;
            const double* row = A + (long)(b0 + lane) * N + b0;
            if (kUpper) {
                const double dinv = (lane < nb) ? 1.0 / row[lane] : 0.0;
                for (int k = nb - 1; k >= 0; --k) {
                    const double yk = __shfl_sync(0xffffffffu, y * dinv, k);
                    if (lane == k) y = yk;
                    if (lane < k) y -= row[k] * yk;
                }
            } else {
                for (int k = 0; k < nb - 1; ++k) {
                    const double yk = __shfl_sync(0xffffffffu, y, k);
                    if (lane > k && lane < nb) y -= row[k] * yk;
                }
            }
            if (lane < nb) v[b0 + lane] = y;
        }
        __syncthreads();
        const int r0 = kUpper ? 0 : b1, r1 = kUpper ? b0 : N;
        for (int i = r0 + tid; i < r1; i += kThreads) {
            const double* row = A + (long)i * N + b0;
            double acc = v[i];
            for (int k = 0; k < nb; ++k) acc -= row[k] * v[b0 + k];
            v[i] = acc;
        }
        __syncthreads();
    }
}

// Dense LU with partial pivoting of the equilibrated assembled reduced system
// (order 4 nb, row-major in scratch), solving for b into x.  Backstop for the Newton steps
// whose block solve did not reach the backward-error target.  The factors, the
// scales and the pivot sequence stay in the scratch for dense_resolve (the
// refinement of the backstop's solution).  Returns false when a pivot column is
// exactly zero.
//
// The matrix is stored dense but is sparse (118 buses: 2 % of its entries), and in elimination
// order partial pivoting keeps most multipliers and most of U zero until the last panels.  Each
// panel's trailing update therefore runs over the rows with a nonzero multiplier and the columns
// with a nonzero in the panel's block row of U only (lists in shared memory); the updates left
// out subtract exact zeros, so the factors are those of the full update.  One CTA factorises
// alone, while the rest of the launch may have run out of scenarios, so this is the tail of small
// and middle-sized batches: 240 single outages at 90 % load take 79.5 ms instead of 173.6 (mixed
// form), 501 pairs 93 instead of 147, 10,000 pairs 1,329 instead of 1,369.
__device__ __noinline__ bool dense_solve(const DevNet& net, double* W, const Lay& L, DenseShared& ds) {
    const int tid = threadIdx.x, nb = net.nb, N = 4 * nb;
    const int warp = tid >> 5, lane = tid & 31;
    double* A = W + L.dense;
    double* x = W + L.x;
    for (long w = tid; w < (long)N * N; w += kThreads) A[w] = 0.0;
    // Equilibrate rows then columns by powers of two (exact): the reduced system's
    // rows span ~1e-5..1e12 near convergence, and partial pivoting is only normwise
    // stable, so without scaling the balance rows lose all accuracy.
    double* rs = W + L.drs;         // row scales
    double* cs = W + L.cs;          // column scales
    int* piv = reinterpret_cast<int*>(W + L.dpiv);   // row exchanged with row k at step k
    // largest entry of row w of the symmetric K, entry (w, c) scaled by sc[c] if given
    auto row_scale = [&](int w, const double* sc) {
        const int i = w >> 2, rr = w & 3;
        unsigned long long m = 0ull;
        auto look = [&](double a, int c) { m = max(m, abs_bits(sc ? a * sc[c] : a)); };
        for (int c = 0; c < 4; ++c) look(W[L.Kd + 16 * i + 4 * (sc ? c : rr) + (sc ? rr : c)], 4 * i + c);
        for (int e = net.adj_ptr[i]; e < net.adj_ptr[i + 1]; ++e) {
            const int code = net.adj_blk[e];
            const double* Kq = W + L.Kb + 16 * (code >> 1) + ((code & 1) ? rr : 4 * rr);
            for (int c = 0; c < 4; ++c) look(Kq[(code & 1) ? 4 * c : c], 4 * net.adj_col[e] + c);
        }
        if (m == 0ull) return 1.0;
        int e;
        frexp(__longlong_as_double((long long)m), &e);
        return ldexp(1.0, -e);
    };
    for (int w = tid; w < N; w += kThreads) {
        rs[w] = row_scale(w, nullptr);
        x[w] = W[L.bv + w] * rs[w];
    }
    __syncthreads();
    for (int w = tid; w < N; w += kThreads) cs[w] = row_scale(w, rs);
    __syncthreads();
    for (int w = tid; w < 16 * nb; w += kThreads) {
        const int i = w >> 4, r = 4 * i + ((w >> 2) & 3), c = 4 * i + (w & 3);
        A[(long)r * N + c] = W[L.Kd + w] * rs[r] * cs[c];
    }
    for (int w = tid; w < 16 * net.nL; w += kThreads) {
        const int q = w >> 4, i = 4 * net.Lrow[q] + ((w >> 2) & 3), j = 4 * net.Lcol[q] + (w & 3);
        if (net.blk_br_ptr[q] == net.blk_br_ptr[q + 1]) continue;      // fill: zero in K
        const double v = W[L.Kb + w];
        A[(long)i * N + j] = v * rs[i] * cs[j];
        A[(long)j * N + i] = v * rs[j] * cs[i];
    }
    __syncthreads();
    // Right-looking LU with partial pivoting in panels of kPanel columns: the panel is
    // factorised column by column (whole rows are swapped), then the block row of U
    // is solved with the panel's unit lower triangle and the trailing matrix takes
    // one rank-kPanel update, so it is read and written once per panel.  The right-
    // hand side is eliminated along the way.
    for (int k0 = 0; k0 < N; k0 += kPanel) {
        const int ke = min(k0 + kPanel, N);
        for (int k = k0; k < ke; ++k) {
            unsigned long long best = 0ull;
            int bi = k;
            for (int i = k + tid; i < N; i += kThreads) {
                const unsigned long long a = abs_bits(A[(long)i * N + k]);
                if (a > best) { best = a; bi = i; }
            }
            for (int off = 16; off; off >>= 1) {
                const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, off);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (lane == 0) { ds.val[warp] = best; ds.idx[warp] = bi; }
            __syncthreads();
            if (tid == 0) {
                unsigned long long b0 = ds.val[0];
                int i0 = ds.idx[0];
                for (int q = 1; q < kWarps; ++q)
                    if (ds.val[q] > b0 || (ds.val[q] == b0 && ds.idx[q] < i0)) { b0 = ds.val[q]; i0 = ds.idx[q]; }
                ds.piv = i0;
                ds.pv = __longlong_as_double((long long)b0);
                ds.nr = 0;
                ds.nc = 0;
                piv[k] = i0;
            }
            __syncthreads();
            if (!(ds.pv > 0.0) || !isfinite(ds.pv)) return false;
            const int p = ds.piv;
            if (p != k) {
                for (int c = tid; c < N; c += kThreads) {
                    const double t = A[(long)k * N + c];
                    A[(long)k * N + c] = A[(long)p * N + c];
                    A[(long)p * N + c] = t;
                }
                if (tid == 0) { const double t = x[k]; x[k] = x[p]; x[p] = t; }
                __syncthreads();
            }
            const double* pk = A + (long)k * N;
            const double inv = 1.0 / pk[k];
            const double xk = x[k];
            for (int i = k + 1 + tid; i < N; i += kThreads) {       // column k and the rest of the panel
                double* ri = A + (long)i * N;
                const double a = ri[k];
                if (a == 0.0) continue;
                const double l = a * inv;
                ri[k] = l;
                for (int j = k + 1; j < ke; ++j) ri[j] -= l * pk[j];
                x[i] -= l * xk;
            }
            __syncthreads();
        }
        if (ke == N) break;
        const int kb = ke - k0;
        for (int j0 = ke; j0 < N; j0 += kThreads) {                  // U block row: unit lower solve
            const int j = j0 + tid;
            bool on = false;
            if (j < N) {
                double u[kPanel];
#pragma unroll
                for (int t = 0; t < kPanel; ++t) {
                    u[t] = (t < kb) ? A[(long)(k0 + t) * N + j] : 0.0;
                    on = on || u[t] != 0.0;
                }
                if (on) {
#pragma unroll
                    for (int r = 1; r < kPanel; ++r) {
                        if (r < kb) {
#pragma unroll
                            for (int t = 0; t < r; ++t) u[r] -= A[(long)(k0 + r) * N + k0 + t] * u[t];
                            A[(long)(k0 + r) * N + j] = u[r];
                        }
                    }
                }
            }
            list_add(ds.cols, &ds.nc, on, j);
        }
        for (int i0 = ke; i0 < N; i0 += kThreads) {                  // rows with a nonzero multiplier
            const int i = i0 + tid;
            bool on = false;
            if (i < N)
                for (int t = 0; t < kb; ++t) on = on || A[(long)i * N + k0 + t] != 0.0;
            list_add(ds.rows, &ds.nr, on, i);
        }
        __syncthreads();
        const int nr = ds.nr, nc = ds.nc;
        for (int q = warp; q < nr; q += kWarps) {                    // trailing rank-kb update
            double* ri = A + (long)ds.rows[q] * N;
            double l[kPanel];
#pragma unroll
            for (int t = 0; t < kPanel; ++t) l[t] = (t < kb) ? ri[k0 + t] : 0.0;
            for (int c = lane; c < nc; c += 32) {
                const int j = ds.cols[c];
                double acc = ri[j];
#pragma unroll
                for (int t = 0; t < kPanel; ++t)
                    if (t < kb) acc -= l[t] * A[(long)(k0 + t) * N + j];
                ri[j] = acc;
            }
        }
        __syncthreads();
    }
    dense_tri<true>(A, N, x);
    for (int w = tid; w < N; w += kThreads) x[w] *= cs[w];     // undo the column scaling
    __syncthreads();
    return true;
}

// v <- K^{-1} v with the factors dense_solve left (row scaling, the recorded row
// exchanges, unit lower and upper triangular solves, column scaling).
__device__ __noinline__ void dense_resolve(const DevNet& net, double* W, const Lay& L, double* v) {
    const int tid = threadIdx.x, N = 4 * net.nb;
    const double* A = W + L.dense;
    const double* rs = W + L.drs;
    const double* cs = W + L.cs;
    const int* piv = reinterpret_cast<const int*>(W + L.dpiv);
    for (int w = tid; w < N; w += kThreads) v[w] *= rs[w];
    __syncthreads();
    if (tid == 0)
        for (int k = 0; k < N; ++k) {
            const int p = piv[k];
            if (p != k) { const double t = v[k]; v[k] = v[p]; v[p] = t; }
        }
    __syncthreads();
    dense_tri<false>(A, N, v);
    dense_tri<true>(A, N, v);
    for (int w = tid; w < N; w += kThreads) v[w] *= cs[w];
    __syncthreads();
}

struct Scal {          // per-scenario scalars in shared memory
    double gamma, f, f_prev, lref, dlref, ap, ad;
    double red[kRedMax];
    double niq, shed;  // number of inequality rows; load outside the main island (p.u.)
    int fail;
    int conv;
    int lost;          // 1: too far from converging for the iterations left
    int scen;
    int ref;           // reference bus of this scenario (-1: no main island)
    int isl;           // 1: main-island form of an islanded scenario
};

// In service in this scenario: not outaged and, in the main-island form of an
// islanded scenario (isl), inside the main island (per-bus flags in the scratch).
struct Live {
    const DevNet& net;
    const Outage& out;
    const double* W;
    const Lay& L;
    const int& isl;        // shared per-scenario flag: the main-island form is on
    __device__ bool bus(int i) const {
        return !isl || reinterpret_cast<const unsigned char*>(W + L.dead)[i] == 0;
    }
    __device__ bool br(int b) const { return !br_out(out, b) && bus(net.f[b]); }
    __device__ bool gen(int k) const { return !gen_out(out, k) && bus(net.gbus[k]); }
};

__device__ int uf_root(int* p, int u) {
    while (p[u] != u) {
        p[u] = p[p[u]];
        u = p[u];
    }
    return u;
}

// Main island of an islanded scenario (one thread; the components are the
// islanding kernel's, rebuilt here).  Union by the smaller index makes every
// root its component's lowest bus, so scanning roots in bus order with a
// strict comparison gives equal totals to the component of the lowest bus.
// Capacities are summed in per unit in generator order.  Sets the bus flags,
// sc.ref (-1 if no component has generation), sc.shed and sc.niq.
__device__ __noinline__ void main_island_setup(const DevNet& net, const Outage& out, const double* Pd, double* W,
                                  const Lay& L, Scal& sc) {
    const int nb = net.nb;
    int* par = reinterpret_cast<int*>(W + L.uf);
    double* cap = W + L.cap;
    unsigned char* dead = reinterpret_cast<unsigned char*>(W + L.dead);
    for (int i = 0; i < nb; ++i) { par[i] = i; cap[i] = 0.0; }
    for (int b = 0; b < net.nbr; ++b) {
        if (br_out(out, b)) continue;
        const int x = uf_root(par, net.f[b]), y = uf_root(par, net.t[b]);
        if (x != y) {
            if (x < y) par[y] = x; else par[x] = y;
        }
    }
    for (int k = 0; k < net.ng; ++k)
        if (!gen_out(out, k)) cap[uf_root(par, net.gbus[k])] += net.pmax[k];
    int main = -1;
    double best = 0.0;
    for (int i = 0; i < nb; ++i)
        if (par[i] == i && cap[i] > best) { main = i; best = cap[i]; }
    double shed = 0.0;
    int nb_live = 0;
    for (int i = 0; i < nb; ++i) {
        const bool d = (main < 0) || uf_root(par, i) != main;
        dead[i] = d ? 1 : 0;
        if (d) shed += Pd[i]; else ++nb_live;
    }
    int ref = -1;
    if (main >= 0) {
        if (!dead[net.ref]) {
            ref = net.ref;
        } else {
            double pb = -INFINITY;
            for (int k = 0; k < net.ng; ++k)
                if (!gen_out(out, k) && !dead[net.gbus[k]] && net.pmax[k] > pb) { pb = net.pmax[k]; ref = net.gbus[k]; }
        }
    }
    int nbr_live = 0, ng_live = 0;
    for (int b = 0; b < net.nbr; ++b) nbr_live += (!br_out(out, b) && !dead[net.f[b]]) ? 1 : 0;
    for (int k = 0; k < net.ng; ++k) ng_live += (!gen_out(out, k) && !dead[net.gbus[k]]) ? 1 : 0;
    sc.ref = ref;
    sc.shed = shed;
    sc.niq = 2.0 * nbr_live + 2.0 * nb_live + 4.0 * ng_live;
}

__global__ void __launch_bounds__(kThreads, kCtasPerSm)
opf_kernel(DevNet net, EvalArgs a, const int* islanded, OpfOut o, double tol, int max_it,
           double* scratch, size_t per_cta, Lay L, int* counter) {
    __shared__ RedBuf rb;
    __shared__ double fsum[2 * kThreads];  // sums of the targets cut between groups (at most 2 per group)
    __shared__ Scal sc;
    const int tid = threadIdx.x;
    double* W = scratch + per_cta * blockIdx.x;
    const int nb = net.nb, ng = net.ng, nbr = net.nbr;
    const double B = net.base;
    const double* Pd = net.Pd + (size_t)a.level * nb;
    const double* Qd = net.Qd + (size_t)a.level * nb;
    const int nx = 2 * nb + 2 * ng;

    for (;;) {
        if (tid == 0) sc.scen = atomicAdd(counter, 1);
        __syncthreads();
        const int s = sc.scen;
        if (s >= a.n) break;
        const bool isl = islanded[s] == 1 && a.main_island;
        if (islanded[s] != 0 && !isl) {        // islanded or invalid: nothing to do here
            if (tid == 0) o.status[s] = 3;
            __syncthreads();
            continue;
        }
        const Outage out = decode_outage(nbr, ng, a.ei[s], a.ej[s], a.ek ? a.ek[s] : -1);
        if (tid == 0) {
            sc.isl = isl ? 1 : 0;
            if (isl) {
                main_island_setup(net, out, Pd, W, L, sc);
            } else {
                sc.ref = net.ref;
                sc.niq = 2.0 * (nbr - n_br_out(out)) + 2.0 * nb + 4.0 * (ng - n_gen_out(out));
            }
        }
        __syncthreads();
        if (sc.ref < 0) {                      // no component has generation: nothing to run
            if (tid == 0) {
                const double nan = __longlong_as_double(0x7ff8000000000000ll);
                o.status[s] = 3;
                a.out.opf_iters[s] = 0;
                if (a.out.shed_mw) a.out.shed_mw[s] = B * sc.shed;
                if (a.out.main_klass) a.out.main_klass[s] = CS_OPF_NONCONV;
                if (a.out.max_loading) a.out.max_loading[s] = nan;
                if (a.out.v_margin) a.out.v_margin[s] = nan;
            }
            for (int i = tid; i < nb; i += kThreads) {
                if (a.out.Va) a.out.Va[(size_t)s * nb + i] = 0.0;
                if (a.out.Vm) a.out.Vm[(size_t)s * nb + i] = 0.0;
            }
            __syncthreads();
            continue;
        }
        const Live lv{net, out, W, L, sc.isl};
        const double niq = sc.niq;

        // ---------------- initial point ----------------
        if (tid == 0) {
            sc.gamma = 1.0;
            sc.lref = 0.0;
            sc.fail = 0;
            sc.conv = 0;
            sc.lost = 0;
        }
        for (int i = tid; i < nb; i += kThreads) {
            W[L.Va + i] = 0.0;
            W[L.Vm + i] = 1.0;
            W[L.lP + i] = 0.0;
            W[L.lQ + i] = 0.0;
        }
        for (int k = tid; k < ng; k += kThreads) {
            const bool off = !lv.gen(k);
            W[L.Pg + k] = off ? 0.0 : 0.5 * (net.pmin[k] + net.pmax[k]);
            W[L.Qg + k] = 0.0;
        }
        __syncthreads();
        int it = 0;
        // evaluate(x) then the convergence quantities; init = first call
        auto evaluate = [&](bool init) {
            const double gamma = init ? 1.0 : sc.gamma;
            for (int b = tid; b < nbr; b += kThreads) {
                if (!lv.br(b)) {
                    double* rec = W + L.rec + (size_t)kRec * b;
                    for (int q = 0; q < kRec; ++q) rec[q] = 0.0;
                    W[L.zf + b] = 1.0; W[L.zt + b] = 1.0; W[L.muf + b] = 0.0; W[L.mut + b] = 0.0;
                    W[L.hf + b] = -1.0; W[L.ht + b] = -1.0;
                    continue;
                }
                eval_branch(net, b, W, L, gamma, init);
            }
            __syncthreads();
            // per-thread partial reductions: max |g|, h, |x|, z, mu, |Lx|, |lam|; sum z mu, cost
            key_t64 kx[7] = {0, 0, 0, 0, 0, 0, 0};
            double zmu = 0.0, cost = 0.0;
            auto top = [&](int q, key_t64 k) { kx[q] = max(kx[q], k); };
            for (int b = tid; b < nbr; b += kThreads) {
                if (!lv.br(b)) continue;
                const double zf = W[L.zf + b], zt = W[L.zt + b], mf = W[L.muf + b], mt = W[L.mut + b];
                top(1, max(pos_key(W[L.hf + b]), pos_key(W[L.ht + b])));
                top(3, max(abs_key(zf), abs_key(zt)));
                top(4, max(abs_key(mf), abs_key(mt)));
                zmu += zf * mf + zt * mt;
            }
            for (int i = tid; i < nb; i += kThreads) {
                if (!lv.bus(i)) {              // outside the main island: no rows, no bounds, load shed
                    if (init) { W[L.zu + i] = 1.0; W[L.zl + i] = 1.0; W[L.muu + i] = 0.0; W[L.mul + i] = 0.0; }
                    W[L.rzu + i] = 1.0; W[L.rzl + i] = 1.0;
                    W[L.gP + i] = 0.0; W[L.gQ + i] = 0.0;
                    W[L.NVa + i] = 0.0; W[L.NVm + i] = 0.0; W[L.DP + i] = 0.0; W[L.DQ + i] = 0.0;
                    W[L.rP + i] = 0.0; W[L.rQ + i] = 0.0;
                    continue;
                }
                const double Vm = W[L.Vm + i], Va = W[L.Va + i];
                const double hu = Vm - net.vmax[i], hl = net.vmin[i] - Vm;
                double zu, zl, muu, mul, rzu, rzl;
                if (init) {
                    zu = fmax(-hu, 1.0); zl = fmax(-hl, 1.0);
                    rzu = 1.0 / zu; rzl = 1.0 / zl;
                    muu = gamma * rzu; mul = gamma * rzl;
                    W[L.zu + i] = zu; W[L.zl + i] = zl; W[L.muu + i] = muu; W[L.mul + i] = mul;
                } else {
                    zu = W[L.zu + i]; zl = W[L.zl + i]; muu = W[L.muu + i]; mul = W[L.mul + i];
                    rzu = 1.0 / zu; rzl = 1.0 / zl;
                }
                W[L.rzu + i] = rzu; W[L.rzl + i] = rzl;
                const double lP = W[L.lP + i], lQ = W[L.lQ + i];
                double Sre = Vm * Vm * net.gsh[i], Sim = -Vm * Vm * net.bsh[i];
                double LxVa = 0.0, LxVm = 2.0 * Vm * (lP * net.gsh[i] - lQ * net.bsh[i]) + muu - mul;
                double NVa = 0.0, NVm = (muu * hu + gamma) * rzu - (mul * hl + gamma) * rzl;
                for (int e = net.bus_br_ptr[i]; e < net.bus_br_ptr[i + 1]; ++e) {
                    const int code = net.bus_br[e];
                    const int b = code >> 1, side = code & 1;
                    if (!lv.br(b)) continue;
                    const double* rec = W + L.rec + (size_t)kRec * b;
                    const double sg = side ? -1.0 : 1.0;
                    Sre += rec[R_S + 2 * side];
                    Sim += rec[R_S + 2 * side + 1];
                    LxVa += sg * rec[R_L];
                    LxVm += rec[R_L + 1 + side];
                    NVa += sg * rec[R_N];
                    NVm += rec[R_N + 1 + side];
                }
                if (i == sc.ref) LxVa += sc.lref;
                double Pgen = 0.0, Qgen = 0.0, DP = 0.0, DQ = 0.0, rP = 0.0, rQ = 0.0;
                for (int e = net.bus_gen_ptr[i]; e < net.bus_gen_ptr[i + 1]; ++e) {
                    const int k = net.bus_gen[e];
                    if (!lv.gen(k)) continue;
                    const double Pg = W[L.Pg + k], Qg = W[L.Qg + k];
                    const double h4[4] = {Pg - net.pmax[k], net.pmin[k] - Pg, Qg - net.qmax[k], net.qmin[k] - Qg};
                    double m4[4], r4[4];
                    for (int q = 0; q < 4; ++q) {
                        double z;
                        if (init) {
                            z = fmax(-h4[q], 1.0);
                            r4[q] = 1.0 / z;
                            m4[q] = gamma * r4[q];
                            W[L.gz + 4 * k + q] = z;
                            W[L.gmu + 4 * k + q] = m4[q];
                        } else {
                            z = W[L.gz + 4 * k + q];
                            m4[q] = W[L.gmu + 4 * k + q];
                            r4[q] = 1.0 / z;
                        }
                        W[L.grz + 4 * k + q] = r4[q];
                        top(1, pos_key(h4[q]));
                        top(3, abs_key(z));
                        top(4, abs_key(m4[q]));
                        zmu += z * m4[q];
                    }
                    const double PgMW = B * Pg;
                    const double LxP = B * (2.0 * net.c2[k] * PgMW + net.c1[k]) - lP + m4[0] - m4[1];
                    const double LxQ = -lQ + m4[2] - m4[3];
                    const double NP = LxP + (m4[0] * h4[0] + gamma) * r4[0] - (m4[1] * h4[1] + gamma) * r4[1];
                    const double NQ = LxQ + (m4[2] * h4[2] + gamma) * r4[2] - (m4[3] * h4[3] + gamma) * r4[3];
                    const double rMP = 1.0 / (2.0 * net.c2[k] * B * B + m4[0] * r4[0] + m4[1] * r4[1]);
                    const double rMQ = 1.0 / (m4[2] * r4[2] + m4[3] * r4[3]);
                    W[L.NP + k] = NP; W[L.NQ + k] = NQ;
                    W[L.MP + k] = rMP; W[L.MQ + k] = rMQ;
                    DP += rMP;
                    DQ += rMQ;
                    rP += NP * rMP;
                    rQ += NQ * rMQ;
                    Pgen += Pg;
                    Qgen += Qg;
                    top(2, max(abs_key(Pg), abs_key(Qg)));
                    top(5, max(abs_key(LxP), abs_key(LxQ)));
                    cost += net.c2[k] * PgMW * PgMW + net.c1[k] * PgMW + net.c0[k];
                }
                NVa += LxVa;
                NVm += LxVm;
                const double gP = Sre - Pgen + Pd[i], gQ = Sim - Qgen + Qd[i];
                W[L.gP + i] = gP; W[L.gQ + i] = gQ;
                W[L.NVa + i] = NVa; W[L.NVm + i] = NVm;
                W[L.DP + i] = DP; W[L.DQ + i] = DQ; W[L.rP + i] = rP; W[L.rQ + i] = rQ;
                top(0, max(abs_key(gP), abs_key(gQ)));
                if (non_finite(NVa) || non_finite(NVm)) top(0, 0x7ff0000000000000ull);
                top(1, max(pos_key(hu), pos_key(hl)));
                top(2, max(abs_key(Va), abs_key(Vm)));
                top(3, max(abs_key(zu), abs_key(zl)));
                top(4, max(abs_key(muu), abs_key(mul)));
                top(5, max(abs_key(LxVa), abs_key(LxVm)));
                top(6, max(abs_key(lP), abs_key(lQ)));
                zmu += zu * muu + zl * mul;
            }
            if (tid == 0) top(6, abs_key(sc.lref));
#pragma unroll
            for (int q = 0; q < 7; ++q) kx[q] = warp_max_key(kx[q]);
            for (int off = 16; off; off >>= 1) {
                zmu += __shfl_xor_sync(0xffffffffu, zmu, off);
                cost += __shfl_xor_sync(0xffffffffu, cost, off);
            }
            if ((tid & 31) == 0) {
#pragma unroll
                for (int q = 0; q < 7; ++q) rb.v[q][tid >> 5] = key_value(kx[q]);
                rb.v[7][tid >> 5] = zmu;
                rb.v[8][tid >> 5] = cost;
            }
            __syncthreads();
            if (tid < 32) {
                // every lane takes the totals; lanes 0..3 divide for one stopping condition each
                key_t64 mx[7];
#pragma unroll
                for (int q = 0; q < 7; ++q) {
                    mx[q] = 0;
                    for (int w = 0; w < kWarps; ++w) mx[q] = max(mx[q], abs_key(rb.v[q][w]));
                }
                double zm = rb.v[7][0], f = rb.v[8][0];
                for (int w = 1; w < kWarps; ++w) {
                    zm += rb.v[7][w];
                    f += rb.v[8][w];
                }
                const double fp = init ? f : sc.f_prev;
                // feasibility (the largest |g| is at least 0, so only a positive h can decide it),
                // gradient, complementarity, cost
                const double num = tid == 0 ? key_value(max(mx[0], mx[1])) : tid == 1 ? key_value(mx[5])
                                 : tid == 2 ? zm : fabs(f - fp);
                const double den = 1.0 + (tid == 0 ? key_value(max(mx[2], mx[3]))
                                        : tid == 1 ? key_value(max(mx[6], mx[4]))
                                        : tid == 2 ? key_value(mx[2]) : fabs(fp));
                const double cnd = num / den;
                const unsigned wild = __ballot_sync(0xffffffffu, non_finite(cnd) || non_finite(f)) & 0xfu;
                const unsigned met = __ballot_sync(0xffffffffu, cnd < tol) & 0xfu;
                if (tid == 2) {
                    sc.f = f;
                    if (init) sc.f_prev = f;
                    if (wild) sc.fail = 1;
                    sc.conv = met == 0xfu ? 1 : 0;
                    // Stop on a scenario that is too far from converging.  One step keeps at least the fraction
                    // 1 - xi = 5e-5 of every z and of every mu, so z . mu loses less than 2^29 an iteration, and
                    // to converge it has to come below tol (1 + max |x|).  A z . mu that all iterations left
                    // would take to 2^100 tol at best can only do so with max |x| above 2^100.  Vm, Pg and
                    // Qg cannot get there: h + z of their bounds is linear and shrinks by 1 - alpha a step, so they
                    // stay within their limits, the start's violation of them and 1.  A bus angle has no such
                    // bound, so this is no proof for angles of 2^100 rad, which FP64 does not resolve to a
                    // turn.  On an infeasible scenario the multipliers grow by decades per iteration, and the
                    // iterations saved are those whose Newton systems need the dense backstop (14 buses, 300
                    // pairs: 13.2 -> 10.9 ms).  The record states the cap.  Run to the end, such iterates are
                    // rounding, and a singular or non-finite system ends some of them sooner: over 1,945 runs
                    // of infeasible scenarios of 6 and 14 buses the count equals the oracle's in 1,917 with the stop
                    // and in 1,865 without it.
                    if (zm > 0.0 && !non_finite(zm))
                        sc.lost = ilogb(zm) > ilogb(tol) + kStateBits + kLossBits * (max_it - it) ? 1 : 0;
                }
            }
            __syncthreads();
        };

        evaluate(true);

        while (!sc.conv && !sc.fail && !sc.lost && it < max_it) {
            ++it;
            const double gamma = sc.gamma;
            // ---------------- assemble the reduced KKT blocks ----------------
            for (int tg = tid; tg < nb + net.nL; tg += kThreads) {
                double blk[16];
                for (int q = 0; q < 16; ++q) blk[q] = 0.0;
                if (tg < nb) {
                    const int j = tg, i = net.perm[j];
                    const double Vm = W[L.Vm + i];
                    double J[2][2] = {{0.0, 2.0 * net.gsh[i] * Vm}, {0.0, -2.0 * net.bsh[i] * Vm}};
                    blk[5] = 2.0 * (W[L.lP + i] * net.gsh[i] - W[L.lQ + i] * net.bsh[i]) +
                             W[L.muu + i] * W[L.rzu + i] + W[L.mul + i] * W[L.rzl + i];
                    for (int e = net.bus_br_ptr[i]; e < net.bus_br_ptr[i + 1]; ++e) {
                        const int code = net.bus_br[e];
                        const int b = code >> 1, side = code & 1;
                        if (!lv.br(b)) continue;
                        const double* rec = W + L.rec + (size_t)kRec * b;
                        const double sg = side ? -1.0 : 1.0;
                        const double* dS = rec + (side ? R_DT : R_DF);
                        blk[0] += rec[R_H];
                        blk[1] += sg * rec[R_H + 1 + side];
                        blk[5] += rec[side ? R_H + 5 : R_H + 3];
                        J[0][0] += sg * dS[0];
                        J[1][0] += sg * dS[1];
                        J[0][1] += dS[2 + 2 * side];
                        J[1][1] += dS[3 + 2 * side];
                    }
                    blk[4] = blk[1];
                    for (int q = 0; q < 2; ++q)
                        for (int r = 0; r < 2; ++r) {
                            blk[4 * r + 2 + q] = J[q][r];
                            blk[4 * (2 + q) + r] = J[q][r];
                        }
                    blk[10] = -W[L.DP + i];
                    blk[15] = -W[L.DQ + i];
                    if (i == sc.ref) {
                        for (int q = 0; q < 4; ++q) { blk[q] = 0.0; blk[4 * q] = 0.0; }
                        blk[0] = 1.0;
                    }
                    const bool on = lv.bus(i);
                    if (!on)                   // outside the main island: identity block, zero step
                        for (int q = 0; q < 16; ++q) blk[q] = (q % 5 == 0) ? 1.0 : 0.0;
                    double* D = W + L.Kd + 16 * j;
                    double* Dc = W + L.Db + 16 * j;
                    for (int q = 0; q < 16; ++q) { D[q] = blk[q]; Dc[q] = blk[q]; }
                    double bq[4] = {0.0, 0.0, 0.0, 0.0};
                    if (on) {
                        bq[0] = (i == sc.ref) ? 0.0 : -W[L.NVa + i];
                        bq[1] = -W[L.NVm + i];
                        bq[2] = -W[L.gP + i] - W[L.rP + i];
                        bq[3] = -W[L.gQ + i] - W[L.rQ + i];
                    }
                    for (int q = 0; q < 4; ++q) { W[L.bv + 4 * j + q] = bq[q]; W[L.x + 4 * j + q] = bq[q]; }
                } else {
                    const int q = tg - nb;
                    const int Rn = net.Lrow[q], Cn = net.Lcol[q];
                    const int Rb = net.perm[Rn], Cb = net.perm[Cn];
                    for (int e = net.blk_br_ptr[q]; e < net.blk_br_ptr[q + 1]; ++e) {
                        const int b = net.blk_br[e];
                        if (!lv.br(b)) continue;
                        const double* rec = W + L.rec + (size_t)kRec * b;
                        const bool flip = (net.f[b] != Rb);     // stored block is (t row, f col)
                        const double* H = rec + R_H;
                        const double* DF = rec + R_DF;
                        const double* DT = rec + R_DT;
                        // rows (theta_f, Vm_f, lamP_f, lamQ_f), columns the same of t
                        const double K[16] = {neg(H[0]), H[2], DT[0], DT[1],
                                              neg(H[1]), H[4], DT[2], DT[3],
                                              neg(DF[0]), DF[4], 0.0, 0.0,
                                              neg(DF[1]), DF[5], 0.0, 0.0};
                        for (int r = 0; r < 4; ++r)
                            for (int c = 0; c < 4; ++c) blk[4 * r + c] += flip ? K[4 * c + r] : K[4 * r + c];
                    }
                    if (Rb == sc.ref) for (int c = 0; c < 4; ++c) blk[c] = 0.0;
                    if (Cb == sc.ref) for (int r = 0; r < 4; ++r) blk[4 * r] = 0.0;
                    double* U = W + L.Ub + 16 * q;
                    for (int c = 0; c < 16; ++c) U[c] = blk[c];
                    if (net.blk_br_ptr[q] < net.blk_br_ptr[q + 1]) {     // not fill: kept for the residual
                        double* Kq = W + L.Kb + 16 * q;
                        for (int c = 0; c < 16; ++c) Kq[c] = blk[c];
                    }
                }
            }
            __syncthreads();
            // ---------------- block LDL^T, level by level ----------------
            for (int lev = 0; lev < net.nlevels; ++lev) {
                // A thread per block entry, groups of 16 threads per block.  The level's block updates are
                // dealt out to the groups in equal shares; a target whose list is cut between groups
                // collects their sums in shared memory.  On a level with one column (the top of the
                // tree) the first warp sums and inverts the pivot while the others sum the off-
                // diagonal blocks.  What bounds it is latency, per level on one scenario: ~5k cycles
                // for the pivot's updates, ~6k for its inverse, ~3k for the blocks' L; the iteration's
                // factorisation takes 462k cycles alone (551k with a target per group and four lanes
                // per pivot), one scenario's OPF 13.1 ms (18.7 with the solves of the same change).
                const int c0 = net.lev_ptr[lev], nc = net.lev_ptr[lev + 1] - c0;
                const int e = tid & 15, r = e >> 2, c = e & 3, grp = tid >> 4;
                const int* rp = net.rn_ptr + lev * kGroups + grp;
                const bool one = nc == 1 && kGroups > 2;
                if (one && grp < 2) {
                    const int j = net.lev_col[c0];
                    double acc = 0.0;
                    if (rp[0] < rp[1]) acc = run_sum(net, W, L, net.rn_first[rp[0]], net.rn_first[rp[0] + 1], r, c);
                    __syncwarp();
                    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
                    bool ok;
                    const double inv = inv4(W[L.Db + 16 * j + e] - acc, 0xffffu << (tid & 16), ok);
                    if (grp == 0) W[L.Di + 16 * j + e] = inv;
                    if (!ok) sc.fail = 1;
                } else {
                    for (int q = rp[0]; q < rp[1]; ++q) {
                        const int to = __ldg(net.rn_end + q);
                        const double acc = run_sum(net, W, L, __ldg(net.rn_first + q), __ldg(net.rn_first + q + 1), r, c);
                        if (to >= nb) W[L.Ub + 16 * (to - nb) + e] -= acc;
                        else if (to >= 0) W[L.Db + 16 * to + e] -= acc;
                        else fsum[16 * (-1 - to) + e] = acc;
                    }
                }
                __syncthreads();
                if (!one) {
                    for (int w = tid; w < 4 * nc; w += kThreads) {
                        const int j = __ldg(net.lev_col + c0 + (w >> 2));
                        bool ok;
                        inv4_wide(W + L.Db + 16 * j, W + L.Di + 16 * j, w & 3, 0xfu << (tid & 28), ok);
                        if (!ok) sc.fail = 1;
                    }
                    __syncthreads();
                }
                {                                      // L = U D^-1, two blocks of a group at a time
                    const unsigned m = 0xffffu << (tid & 16);
                    const int b = (tid & 16) + 4 * r;  // the four lanes of row r
                    const int o1 = __ldg(net.off_ptr + lev + 1);
                    for (int o = __ldg(net.off_ptr + lev) + grp; o < o1; o += 2 * kGroups) {
                        const bool two = o + kGroups < o1;
                        int4 of[2] = {__ldg(net.off + o), make_int4(0, 0, 0, 0)};
                        if (two) of[1] = __ldg(net.off + o + kGroups);
                        double u[2], d[2][4];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const double* Di = W + L.Di + 16 * of[q].y + c;
                            u[q] = W[L.Ub + 16 * of[q].x + e];
                            d[q][0] = Di[0]; d[q][1] = Di[4]; d[q][2] = Di[8]; d[q][3] = Di[12];
                        }
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            if (q == 1 && !two) break;
                            for (int p = 0; p < of[q].w; ++p) u[q] -= fsum[16 * (of[q].z + p) + e];
                            if (of[q].w) W[L.Ub + 16 * of[q].x + e] = u[q];
                            const double u0 = __shfl_sync(m, u[q], b), u1 = __shfl_sync(m, u[q], b + 1),
                                         u2 = __shfl_sync(m, u[q], b + 2), u3 = __shfl_sync(m, u[q], b + 3);
                            W[L.Lb + 16 * of[q].x + e] = u0 * d[q][0] + u1 * d[q][1] + u2 * d[q][2] + u3 * d[q][3];
                        }
                    }
                }
                __syncthreads();
            }
            if (sc.fail) break;
            // ---------------- solve, then FP64 iterative refinement against the assembled K ----------------
            // The blocks are eliminated in a fixed order without pivoting between blocks;
            // near convergence some pivot blocks become nearly singular (a load bus whose
            // voltage sits at a bound has one free local variable for two balance rows),
            // which leaves a low-rank error in the first solve that refinement removes.
            // Refinement stops once the componentwise backward error is at rounding level.
            ldl_solve(net, W, L, W + L.x);
            double om;
            for (int ref_step = 0;; ++ref_step) {
                om = kkt_residual(net, W, L, rb, W + L.x, W + L.rv);
                if (om <= kRefineTol || ref_step == kRefineSteps) break;
                ldl_solve(net, W, L, W + L.rv);
                for (int w = tid; w < 4 * nb; w += kThreads) W[L.x + w] += W[L.rv + w];
                __syncthreads();
            }
            if (!(om <= kBackwardTol)) {
                // Krylov steps on the factors, then, if those stall, the dense backstop
                __shared__ GmresShared gs;
                om = kkt_gmres(net, W, L, rb, sc.red, gs, om);
                if (L.dense >= 0 && !(om <= kBackwardTol)) {
                    __shared__ DenseShared ds;
                    if (!dense_solve(net, W, L, ds)) sc.fail = 1;
                    __syncthreads();
                    if (sc.fail) break;
                    // FP64 refinement of the backstop's solution with its own factors; the
                    // best iterate is kept (refinement diverges on a system too ill-conditioned
                    // for FP64, and then the backstop's first solution is the best there is)
                    double best = INFINITY;
                    for (int ref_step = 0;; ++ref_step) {
                        const double om_now = kkt_residual(net, W, L, rb, W + L.x, W + L.rv);
                        if (ref_step > 0 && !(om_now < best)) {          // no progress: back to the best
                            for (int w = tid; w < 4 * nb; w += kThreads) W[L.x + w] = W[L.gxb + w];
                            __syncthreads();
                            break;
                        }
                        best = om_now;
                        if (om_now <= kRefineTol || ref_step == kRefineSteps) break;
                        for (int w = tid; w < 4 * nb; w += kThreads) W[L.gxb + w] = W[L.x + w];
                        dense_resolve(net, W, L, W + L.rv);
                        for (int w = tid; w < 4 * nb; w += kThreads) W[L.x + w] += W[L.rv + w];
                        __syncthreads();
                    }
                }
            }
            // ---------------- recover the eliminated steps, dz, dmu, ratios ----------------
            // Step lengths: xi over the largest -dz / z and -dmu / mu of all rows; the first is a
            // product with the stored 1 / z.
            key_t64 kp = 0, kd = 0;
            bool bad = false;
            auto row = [&](double rz, double m, double dz, int odz, int odm) {
                const double dm = (gamma - m * dz) * rz - m;
                W[odz] = dz;
                W[odm] = dm;
                kp = max(kp, pos_key(neg(dz) * rz));
                if (__double2hiint(dm) < 0) kd = max(kd, pos_key(neg(dm) / m));
                bad = bad || non_finite(dz) || non_finite(dm);
            };
            for (int k = tid; k < ng; k += kThreads) {
                if (!lv.gen(k)) continue;
                const int jn = net.iperm[net.gbus[k]];
                const double dPg = (W[L.x + 4 * jn + 2] - W[L.NP + k]) * W[L.MP + k];
                const double dQg = (W[L.x + 4 * jn + 3] - W[L.NQ + k]) * W[L.MQ + k];
                W[L.dPg + k] = dPg;
                W[L.dQg + k] = dQg;
                const double Pg = W[L.Pg + k], Qg = W[L.Qg + k];
                const double h4[4] = {Pg - net.pmax[k], net.pmin[k] - Pg, Qg - net.qmax[k], net.qmin[k] - Qg};
                const double dh4[4] = {dPg, neg(dPg), dQg, neg(dQg)};
                for (int q = 0; q < 4; ++q)
                    row(W[L.grz + 4 * k + q], W[L.gmu + 4 * k + q], -h4[q] - W[L.gz + 4 * k + q] - dh4[q],
                        L.gdz + 4 * k + q, L.gdmu + 4 * k + q);
            }
            for (int b = tid; b < nbr; b += kThreads) {
                if (!lv.br(b)) continue;
                const double* G = W + L.rec + (size_t)kRec * b + R_G;
                const double* xf = W + L.x + 4 * net.iperm[net.f[b]];
                const double* xt = W + L.x + 4 * net.iperm[net.t[b]];
                const double dth = xf[0] - xt[0], df = xf[1], dt = xt[1];
                row(W[L.rzf + b], W[L.muf + b], -W[L.hf + b] - W[L.zf + b] - (G[0] * dth + G[1] * df + G[2] * dt),
                    L.dzf + b, L.dmuf + b);
                row(W[L.rzt + b], W[L.mut + b], -W[L.ht + b] - W[L.zt + b] - (G[3] * dth + G[4] * df + G[5] * dt),
                    L.dzt + b, L.dmut + b);
            }
            for (int i = tid; i < nb; i += kThreads) {
                if (!lv.bus(i)) continue;
                const int jn = net.iperm[i];
                const double dVm = W[L.x + 4 * jn + 1];
                const double Vm = W[L.Vm + i];
                const double hu = Vm - net.vmax[i], hl = net.vmin[i] - Vm;
                row(W[L.rzu + i], W[L.muu + i], -hu - W[L.zu + i] - dVm, L.dzu + i, L.dmuu + i);
                row(W[L.rzl + i], W[L.mul + i], -hl - W[L.zl + i] + dVm, L.dzl + i, L.dmul + i);
                for (int r = 0; r < 4; ++r) bad = bad || non_finite(W[L.x + 4 * jn + r]);
            }
            if (tid == kThreads - 1) {         // a warp with few rows of its own above
                // multiplier step of the reference-angle row from its Newton row
                const int i = sc.ref;
                double sum = 0.0;
                for (int e = net.bus_br_ptr[i]; e < net.bus_br_ptr[i + 1]; ++e) {
                    const int code = net.bus_br[e];
                    const int b = code >> 1, side = code & 1;
                    if (!lv.br(b)) continue;
                    const double* rec = W + L.rec + (size_t)kRec * b;
                    const double* xf = W + L.x + 4 * net.iperm[net.f[b]];
                    const double* xt = W + L.x + 4 * net.iperm[net.t[b]];
                    const double th = rec[R_H] * (xf[0] - xt[0]) + rec[R_H + 1] * xf[1] + rec[R_H + 2] * xt[1] +
                                      rec[R_DF] * xf[2] + rec[R_DF + 1] * xf[3] + rec[R_DT] * xt[2] +
                                      rec[R_DT + 1] * xt[3];
                    sum += side ? neg(th) : th;
                }
                sc.dlref = -W[L.NVa + i] - sum;
                bad = bad || non_finite(sc.dlref);
            }
            kp = warp_max_key(kp);
            kd = warp_max_key(kd);
            bad = __any_sync(0xffffffffu, bad);
            if ((tid & 31) == 0) {
                rb.v[0][tid >> 5] = key_value(kp);
                rb.v[1][tid >> 5] = key_value(kd);
                rb.v[2][tid >> 5] = bad ? 1.0 : 0.0;
            }
            __syncthreads();
            if (tid < 2) {
                key_t64 k = 0;
                for (int w = 0; w < kWarps; ++w) {
                    k = max(k, abs_key(rb.v[tid][w]));
                    if (rb.v[2][w] != 0.0) sc.fail = 1;
                }
                const double al = fmin(kXi / key_value(k), 1.0);   // no row decreases: 1
                if (tid == 0) sc.ap = al;
                else sc.ad = al;
            }
            __syncthreads();
            if (sc.fail) break;
            // ---------------- update ----------------
            const double ap = sc.ap, ad = sc.ad;
            double zmu = 0.0;
            for (int i = tid; i < nb; i += kThreads) {
                if (!lv.bus(i)) continue;
                const int jn = net.iperm[i];
                W[L.Va + i] += ap * W[L.x + 4 * jn];
                W[L.Vm + i] += ap * W[L.x + 4 * jn + 1];
                W[L.lP + i] += ad * W[L.x + 4 * jn + 2];
                W[L.lQ + i] += ad * W[L.x + 4 * jn + 3];
                const double zu = W[L.zu + i] + ap * W[L.dzu + i], zl = W[L.zl + i] + ap * W[L.dzl + i];
                const double mu_ = W[L.muu + i] + ad * W[L.dmuu + i], ml = W[L.mul + i] + ad * W[L.dmul + i];
                W[L.zu + i] = zu; W[L.zl + i] = zl; W[L.muu + i] = mu_; W[L.mul + i] = ml;
                zmu += zu * mu_ + zl * ml;
            }
            for (int k = tid; k < ng; k += kThreads) {
                if (!lv.gen(k)) continue;
                W[L.Pg + k] += ap * W[L.dPg + k];
                W[L.Qg + k] += ap * W[L.dQg + k];
                for (int q = 0; q < 4; ++q) {
                    const double z = W[L.gz + 4 * k + q] + ap * W[L.gdz + 4 * k + q];
                    const double m = W[L.gmu + 4 * k + q] + ad * W[L.gdmu + 4 * k + q];
                    W[L.gz + 4 * k + q] = z;
                    W[L.gmu + 4 * k + q] = m;
                    zmu += z * m;
                }
            }
            for (int b = tid; b < nbr; b += kThreads) {
                if (!lv.br(b)) continue;
                const double zf = W[L.zf + b] + ap * W[L.dzf + b], zt = W[L.zt + b] + ap * W[L.dzt + b];
                const double mf = W[L.muf + b] + ad * W[L.dmuf + b], mt = W[L.mut + b] + ad * W[L.dmut + b];
                W[L.zf + b] = zf; W[L.zt + b] = zt; W[L.muf + b] = mf; W[L.mut + b] = mt;
                zmu += zf * mf + zt * mt;
            }
            {
                double v1[1] = {zmu};
                const int ops1[1] = {1};
                block_reduce<1>(rb, v1, ops1, sc.red);
            }
            if (tid == 0) {
                sc.lref += ad * sc.dlref;
                sc.gamma = kSigma * sc.red[0] / niq;
                sc.f_prev = sc.f;
            }
            __syncthreads();
            evaluate(false);
        }
        if (sc.lost && !sc.conv && !sc.fail) it = max_it;     // stopped early: the record states the cap
        // ---------------- outputs ----------------
        double viol = 0.0, load_max = 0.0, vmarg = INFINITY;
        const bool converged = sc.conv && !sc.fail;
        if (converged) {
            for (int b = tid; b < nbr; b += kThreads) {
                if (!lv.br(b)) continue;
                const double sm = sqrt(net.smax2[b]);
                const double sf = sqrt(fmax(W[L.hf + b] + net.smax2[b], 0.0));
                const double st = sqrt(fmax(W[L.ht + b] + net.smax2[b], 0.0));
                if (sf - sm > kLimitTol || st - sm > kLimitTol) viol = 1.0;
                load_max = fmax(load_max, fmax(sf, st) / sm);
            }
            for (int i = tid; i < nb; i += kThreads) {
                if (!lv.bus(i)) continue;
                const double Vm = W[L.Vm + i];
                if (Vm - net.vmax[i] > kLimitTol || net.vmin[i] - Vm > kLimitTol) viol = 1.0;
                vmarg = fmin(vmarg, fmin(Vm - net.vmin[i], net.vmax[i] - Vm));
            }
            for (int k = tid; k < ng; k += kThreads) {
                if (!lv.gen(k)) continue;
                const double Pg = W[L.Pg + k], Qg = W[L.Qg + k];
                if (Pg - net.pmax[k] > kLimitTol || net.pmin[k] - Pg > kLimitTol ||
                    Qg - net.qmax[k] > kLimitTol || net.qmin[k] - Qg > kLimitTol) viol = 1.0;
            }
        }
        {
            double v3[3] = {viol, load_max, vmarg};   // non-binary severity: loading, voltage margin
            const int ops3[3] = {0, 0, 2};
            block_reduce<3>(rb, v3, ops3, sc.red);
        }
        double* xs = o.x + (size_t)s * nx;
        for (int i = tid; i < nb; i += kThreads) {
            // a bus outside the main island is de-energised: Vm = 0 also tells the
            // small-signal kernels which buses are out
            const bool on = lv.bus(i);
            xs[i] = on ? W[L.Va + i] : 0.0;
            xs[nb + i] = on ? W[L.Vm + i] : 0.0;
            if (a.out.Va) a.out.Va[(size_t)s * nb + i] = xs[i];
            if (a.out.Vm) a.out.Vm[(size_t)s * nb + i] = xs[nb + i];
        }
        for (int k = tid; k < ng; k += kThreads) {
            xs[2 * nb + k] = W[L.Pg + k];
            xs[2 * nb + ng + k] = W[L.Qg + k];
        }
        if (tid == 0) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            a.out.opf_iters[s] = (int16_t)it;
            a.out.cost[s] = converged ? sc.f : nan;
            if (a.out.max_loading) a.out.max_loading[s] = converged ? sc.red[1] : nan;
            if (a.out.v_margin) a.out.v_margin[s] = converged ? sc.red[2] : nan;
            if (isl) {                         // main island of an islanded scenario: class unchanged
                const bool ok = converged && sc.red[0] == 0.0;
                o.status[s] = ok ? 1 : 3;      // within limits: on to the small-signal screen, which sets main_klass
                if (a.out.shed_mw) a.out.shed_mw[s] = B * sc.shed;
                if (a.out.main_klass && !ok) a.out.main_klass[s] = converged ? CS_LIMIT : CS_OPF_NONCONV;
            } else if (!converged || sc.red[0] != 0.0) {
                o.status[s] = 2;
                a.out.klass[s] = converged ? CS_LIMIT : CS_OPF_NONCONV;
                a.out.severe[s] = 1;
                a.out.max_re[s] = nan;
                a.out.min_zeta[s] = nan;
            } else {
                o.status[s] = 1;
            }
        }
        __syncthreads();
    }
}

}  // namespace

int opf_groups() { return kGroups; }

int opf_ctas_per_sm() { return kCtasPerSm; }

size_t opf_scratch_doubles(const DevNet& net) { return (size_t)make_layout(net).total; }

cudaError_t launch_opf(const DevNet& net, const EvalArgs& a, const int* islanded, OpfOut o, double tol,
                       int max_it, double* scratch, size_t scratch_per_cta, int grid, int* counter,
                       cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    const Lay L = make_layout(net);
    if ((size_t)L.total > scratch_per_cta) return cudaErrorInvalidValue;
    opf_kernel<<<grid, kThreads, 0, s>>>(net, a, islanded, o, tol, max_it, scratch, scratch_per_cta, L, counter);
    return cudaGetLastError();
}
