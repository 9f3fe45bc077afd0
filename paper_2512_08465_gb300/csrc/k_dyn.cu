// Small-signal screen of converged OPF points, one scenario per CTA
// (Section II-B-2: the system model is linearised at the OPF operating point
// and a scenario is unstable when an eigenvalue has a non-negative real part;
// the configuration adds a minimum damping ratio).
//
// Model (per in-service generator, machine data converted to the system base):
// states delta, omega, e'q, e'd, Efd (index 5k + s); E' = (e'q - j e'd) e^{j delta}
// behind j x' (x'd = x'q, Ra = 0); I = Y_red E' with Y_red the Kron reduction of
// the network (loads as constant admittances at the OPF voltage, machines as
// 1/(j x') to their internal nodes); i_d + j i_q = j I e^{-j delta};
//   d delta/dt = ws (omega - 1)
//   2H d omega/dt = Pm - (e'd i_d + e'q i_q) - D (omega - 1)
//   T'd0 d e'q/dt = -e'q - (x_d - x') i_d + Efd
//   T'q0 d e'd/dt = -e'd + (x_q - x') i_q
//   T_A d Efd/dt = -Efd + K_A (V_ref - |E' - j x' I|)
// The state matrix is written from hand-derived partial derivatives of these
// equations (the CPU oracle differentiates them automatically instead).
//
// Steps inside one CTA:
//  1. Y_bb = Ybus(outages masked) + loads + machine admittances, factorised as
//     a complex symmetric LDL^T on the network's shared symbolic analysis
//     (scalar complex blocks, same elimination-tree levels as the OPF kernel);
//  2. one thread per in-service machine solves Y_bb x = e_{bus} to get the
//     machine-bus entries of Y_bb^{-1}, hence Y_red;
//  3. equilibrium from the OPF point; one thread per machine pair writes the
//     5x5 block of A;
//  4. balancing by powers of two, Householder Hessenberg reduction, Francis
//     double-shift QR (eigenvalues only), with the same steps and thresholds
//     as the textbook algorithm, the Hessenberg reduction in one pass over A
//     per column and the QR sweeps in windows of several steps; A lives in
//     the CTA's global scratch;
//  5. max Re and min damping ratio over all eigenvalues, classify.
// Angle reference: every rotor angle is referred to the first in-service
// machine (delta'_k = delta_k - delta_0, d delta'_k/dt = ws (omega_k - omega_0),
// delta_0 dropped).  The absolute-angle matrix has an exact zero eigenvalue
// (common rotation) to which the slow common-frequency mode is nearly parallel;
// the referred matrix (5m - 1 states) has the same eigenvalues less that zero
// and a well-conditioned slow mode.
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "cs_internal.h"

namespace {

constexpr int kMaxThreads = 512;     // threads of a dyn_kernel block: 128, 256 or 512 (see launch_mode)
constexpr int kCtasPerSm = 4;        // resident blocks per SM, of 128 threads
constexpr double kEps = 2.220446049250313e-16;
// FP32 QR deflates a subdiagonal entry below kDeflTol times its two diagonal neighbours
// (not the FP32 unit roundoff): the screen's eigenvalues need only be within kEigDelta of
// the exact ones where the decisive ones are refined in FP64 (within the 5e-3 guard band
// where a network's screen has no refinement), and the sweeps that take a converged entry
// from ~1e-6 relative down to rounding level are most of the QR's work.
// On 118-bus state matrices (order 264-269, FP32 emulation) it cuts the sweeps per matrix
// from 785 to 322 on average, the largest eigenvalue error staying at 8e-5 either way.
constexpr float kDeflTol = 3e-6f;
// FP32 screen in global memory (no refinement): a decision this close to a threshold is
// taken by the FP64 screen instead
constexpr double kGuardRe = 5e-3;      // |max Re| within this of 0
constexpr double kGuardZeta = 5e-3;    // |min zeta - threshold| within this

struct DLay {
    int Yu, Yl, Yd, Ydi;      // complex arrays (2 doubles per entry)
    int Z;                    // [ng*ng] complex
    int rhs;                  // [ng*nb] complex
    int gen;                  // [ng * kGen]
    int A;                    // [(5ng)^2]
    int A32;                  // [(5ng)^2] floats (mixed precision screen)
    int wr, wi, v;            // [5ng]
    int hp;                   // [kHsSlices * 5ng] partial sums of the Hessenberg reduction
    int total;
};
constexpr int kGen = 16;      // per-generator doubles: E(2) I(2) e^{jd}(2) Vt(2) |Vt| id iq eq ed ym(2)
enum { G_E = 0, G_I = 2, G_ED = 4, G_VT = 6, G_VTM = 8, G_ID = 9, G_IQ = 10, G_EQ = 11, G_EDD = 12, G_YM = 13 };

DLay make_dlayout(const DevNet& n) {
    DLay L{};
    int o = 0;
    auto take = [&](long cnt) { int r = o; o += (int)cnt; return r; };
    L.Yu = take(2L * n.nL); L.Yl = take(2L * n.nL); L.Yd = take(2L * n.nb); L.Ydi = take(2L * n.nb);
    L.Z = take(2L * n.ng * n.ng);
    L.rhs = take(2L * n.ng * n.nb);
    L.gen = take((long)kGen * n.ng);
    o = (o + 31) & ~31;
    L.A = take(25L * n.ng * n.ng);
    L.A32 = take((25L * n.ng * n.ng + 1) / 2);
    o = (o + 31) & ~31;
    L.wr = take(5L * n.ng); L.wi = take(5L * n.ng); L.v = take(5L * n.ng);
    // partial sums of the Hessenberg slices: on the reduction's right-hand sides, which nothing reads once
    // the state matrix is formed, where they fit
    L.hp = 2L * n.nb >= 40 ? L.rhs : take(8L * 5 * n.ng);
    L.total = (o + 31) & ~31;
    return L;
}

__device__ __forceinline__ cplx ld(const double* p) { return cplx{p[0], p[1]}; }
__device__ __forceinline__ void st(double* p, cplx v) { p[0] = v.re; p[1] = v.im; }

struct DShared {
    double red[kMaxThreads / 32];
    int ired[kMaxThreads / 32];
    double hs[3];                    // Hessenberg reduction: tail, alpha, beta of the current column
    int fail, scen, m, nn;
};

// block reductions ---------------------------------------------------------
__device__ int bmax_int(DShared& sh, int v) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int off = 16; off; off >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, off));
    if ((tid & 31) == 0) sh.ired[tid >> 5] = v;
    __syncthreads();
    int r = sh.ired[0];
    for (int w = 1; w < nthr / 32; ++w) r = max(r, sh.ired[w]);
    __syncthreads();
    return r;
}
__device__ double bmax(DShared& sh, double v) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int off = 16; off; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if ((tid & 31) == 0) sh.red[tid >> 5] = v;
    __syncthreads();
    double r = sh.red[0];
    for (int w = 1; w < nthr / 32; ++w) r = fmax(r, sh.red[w]);
    __syncthreads();
    return r;
}

// eigenvalues of [[p, q], [r, s]] (same formulas as the textbook closed form)
__device__ void eig2(double p, double q, double r, double s, double* re, double* im) {
    const double hm = 0.5 * (p - s);
    const double disc = hm * hm + q * r;
    const double mean = 0.5 * (p + s);
    if (disc >= 0.0) {
        const double root = sqrt(disc);
        const double big = mean + (hm >= 0.0 ? root : -root);
        const double det = p * s - q * r;
        const double other = (big != 0.0) ? det / big : mean - (hm >= 0.0 ? root : -root);
        re[0] = big; im[0] = 0.0;
        re[1] = other; im[1] = 0.0;
    } else {
        const double root = sqrt(-disc);
        re[0] = mean; im[0] = root;
        re[1] = mean; im[1] = -root;
    }
}


// ---------------------------------------------------------------------------
// Eigenvalues of a real matrix: balancing by powers of two, Householder
// reduction to upper Hessenberg form, Francis double-shift QR with deflation
// (eigenvalues only), as in the textbook algorithm.  A is row-major n x n in
// global memory; cs, rs, v are n-entry shared arrays of T.

// Balancing (radix 2).  Each sweep starts from exact off-diagonal column and
// row 1-norms; within the sweep the norms are updated as rows and columns are
// scaled (a scaling by a power of two changes the other norms by a known
// amount), so the scan over the indices needs no reduction: all threads look at
// their indices' norms at once, and the first one that wants a factor is scaled.
// The sequential sweeps end it as they always did (until no index improves by
// 5 %), but most factors come from kBalJoint sweeps before them that scale all
// indices at once, each by the root of its best factor: an entry joins two
// indices, and with both moved the whole way it would overshoot.  (A factor of
// 2 has no root here: the two halves of the indices take those in turn.)  One
// index at a time costs two barriers and two strided passes; a joint sweep two
// passes over the matrix.
// (118 buses, front kernel: one scenario 2.0 -> 1.3 ms, 417 of them 5.2 -> 4.8.)
// The scale search stops at 2^+-kBalExp (T = float) or
// 2^+-(4 kBalExp) (T = double), so a row or column norm that is tiny next to
// the other cannot drive the factor to overflow or zero; an index whose best
// factor lies beyond that is scaled by the bound.  dsc[i]
// receives the product of the factors of index i: the balanced matrix is
// diag(dsc)^-1 A diag(dsc), exactly (every factor is a power of two).
constexpr int kBalExp = 30;
constexpr int kBalJoint = 12;

// exponent of the factor of an index with column norm c and row norm r; 0: leave it
template <typename T>
__device__ __forceinline__ int bal_exponent(T c, const T r) {
    if (c == 0 || r == 0 || !isfinite(c) || !isfinite(r)) return 0;
    constexpr int top = sizeof(T) == 8 ? 4 * kBalExp : kBalExp;
    const T ssum = c + r;
    T g = r / 2, f = 1;
    int e = 0;
    while (c < g && e < top) { f *= 2; c *= 4; ++e; }
    g = r * 2;
    while (c > g && e > -top) { f /= 2; c /= 4; --e; }
    return ((c + r) / f < (T)0.95 * ssum) ? e : 0;
}

template <typename T>
__device__ void balance(T* A, const int n, T* cs, T* rs, T* dsc, DShared& sh) {
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
    for (int j = tid; j < n; j += nthr) dsc[j] = (T)1;
    for (int sweep = 0; sweep < kBalJoint + 100; ++sweep) {
        for (int j = tid; j < n; j += nthr) {
            T c = 0;
#pragma unroll 8
            for (int i = 0; i < n; ++i) {
                const T a = fabs(A[(size_t)i * n + j]);
                c += (i != j) ? a : (T)0;
            }
            cs[j] = c;
        }
        for (int i = warp; i < n; i += nthr / 32) {
            T r = 0;
            for (int j = lane; j < n; j += 32)
                if (j != i) r += fabs(A[(size_t)i * n + j]);
            for (int off = 16; off; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
            if (lane == 0) rs[i] = r;
        }
        __syncthreads();
        if (sweep < kBalJoint) {
            int any = 0;
            for (int i = tid; i < n; i += nthr) {
                int e = bal_exponent(cs[i], rs[i]);
                if (e == 1 || e == -1) e = ((i ^ sweep) & 1) ? 0 : e;
                else e /= 2;
                any |= e;
                cs[i] = ldexp((T)1, e);                        // the norms have been read: now the factors
                dsc[i] *= cs[i];
            }
            any = __syncthreads_or(any);
            if (any == 0) {
                sweep = kBalJoint - 1;
                continue;
            }
            for (int i = warp; i < n; i += nthr / 32) {
                const T fi = (T)1 / cs[i];
                for (int j = lane; j < n; j += 32) A[(size_t)i * n + j] *= fi * cs[j];
            }
            __syncthreads();
            continue;
        }
        bool changed = false;
        int i0 = 0;
        for (;;) {
            int pick = n;
            for (int i = i0 + tid; i < n && pick == n; i += nthr)
                if (bal_exponent(cs[i], rs[i]) != 0) pick = i;
            const int i = -bmax_int(sh, -pick);
            if (i >= n) break;
            const int e = bal_exponent(cs[i], rs[i]);
            const T f = ldexp((T)1, e), finv = ldexp((T)1, -e);
            __syncthreads();                                   // cs[i], rs[i] read by all
            for (int j = tid; j < n; j += nthr) {
                if (j == i) {
                    cs[i] *= f;
                    rs[i] *= finv;
                    dsc[i] *= f;
                    continue;
                }
                const T a = A[(size_t)i * n + j], b = A[(size_t)j * n + i];
                A[(size_t)i * n + j] = a * finv;
                A[(size_t)j * n + i] = b * f;
                cs[j] += fabs(a) * (finv - 1);
                rs[j] += fabs(b) * (f - 1);
            }
            changed = true;
            i0 = i + 1;
            __syncthreads();
        }
        if (!changed) break;
    }
}

// Householder reduction to upper Hessenberg form, in place, A row-major n x n in global memory.
// Column k: reflector v of its rows k+1.., w = beta v^T A, then every row once: left update
// x = row - v_i w, dot x . v, right update x - beta (x . v) v.  So the matrix is read twice and
// written once per column (the two updates one after the other read it four times and wrote it
// twice), the four multiply-adds per entry are the floor, and the row reductions (FP64 additions
// that fill a warp instruction with one useful lane in the end) go two rows at a time.
//  * w: the rows in kHsSlices slices, a warp per slice with a lane's columns in registers; the
//    slices' sums meet in `part` (kHsSlices x n, global).  The slices are fixed, so the sums do not
//    depend on the number of threads.
//  * rows: a warp per pair of rows, up to kHsReg * 32 columns in registers; longer rows make the
//    second pass over memory.
// The next column is picked up while its rows are written (vn).  v, w, vn: n entries of shared memory.
constexpr int kHsSlices = 8;
constexpr int kHsReg = 12;
template <typename T>
__device__ __forceinline__ void sum2(T& a, T& b) {            // both over the warp, to all lanes
    const bool up = (threadIdx.x & 16) != 0;
    T mine = up ? b : a, other = up ? a : b;
    mine += __shfl_xor_sync(0xffffffffu, other, 16);
    for (int off = 8; off; off >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, off);
    other = __shfl_xor_sync(0xffffffffu, mine, 16);
    a = up ? other : mine;
    b = up ? mine : other;
}

template <typename T>
__device__ __noinline__ void hessenberg(T* A, const int n, T* v, T* w, T* vn, T* part, DShared& sh) {
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nthr >> 5;
    for (int i = tid; i + 1 < n; i += nthr) v[i] = A[(size_t)(i + 1) * n];
    __syncthreads();
    for (int k = 0; k + 2 < n; ++k) {
        const int m = n - k - 1;
        if (warp == 0) {
            T t = 0;
            for (int i = 1 + lane; i < m; i += 32) t += v[i] * v[i];
            for (int off = 16; off; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
            if (lane == 0) {
                sh.hs[0] = (double)t;
                if (t != (T)0) {
                    const T x0 = v[0], nrm = sqrt(x0 * x0 + t), al = (x0 >= (T)0) ? -nrm : nrm, v0 = x0 - al;
                    v[0] = v0;
                    sh.hs[1] = (double)al;
                    sh.hs[2] = (double)((T)2 / (v0 * v0 + t));
                }
            }
        }
        __syncthreads();
        T* A1 = A + (size_t)(k + 1) * n + k + 1;               // rows and columns k + 1 ..
        if (sh.hs[0] == 0.0) {                                 // column already reduced (uniform)
            for (int i = tid; i + 1 < m; i += nthr) vn[i] = A1[(size_t)(i + 1) * n];
            __syncthreads();
            T* q = v; v = vn; vn = q;
            continue;
        }
        const T alpha = (T)sh.hs[1], beta = (T)sh.hs[2];
        for (int j0 = 0; j0 < m; j0 += 32 * kHsReg) {
            for (int sl = warp; sl < kHsSlices; sl += nw) {
                const int i1 = m * (sl + 1) / kHsSlices;
                T acc[kHsReg];
#pragma unroll
                for (int c = 0; c < kHsReg; ++c) acc[c] = (T)0;
#pragma unroll 2
                for (int i = m * sl / kHsSlices; i < i1; ++i) {
                    const T vi = v[i];
                    const T* row = A1 + (size_t)i * n + j0 + lane;
#pragma unroll
                    for (int c = 0; c < kHsReg; ++c)
                        if (j0 + 32 * c + lane < m) acc[c] += vi * row[32 * c];
                }
#pragma unroll
                for (int c = 0; c < kHsReg; ++c) {
                    const int j = j0 + 32 * c + lane;
                    if (j < m) part[(size_t)sl * n + j] = acc[c];
                }
            }
        }
        __syncthreads();
        for (int j = tid; j < m; j += nthr) {
            T t = part[j];
#pragma unroll
            for (int sl = 1; sl < kHsSlices; ++sl) t += part[(size_t)sl * n + j];
            w[j] = beta * t;
        }
        __syncthreads();
        for (int i0 = 2 * warp; i0 < n; i0 += 2 * nw) {
            T* row[2] = {A + (size_t)i0 * n + k + 1, A + (size_t)min(i0 + 1, n - 1) * n + k + 1};
            const bool two = i0 + 1 < n;
            const T vi[2] = {i0 > k ? v[i0 - k - 1] : (T)0, (two && i0 + 1 > k) ? v[i0 - k] : (T)0};
            T x[2][kHsReg], acc[2] = {(T)0, (T)0};
            const bool fits = m <= 32 * kHsReg;
            for (int j0 = 0; j0 < m; j0 += 32 * kHsReg) {
#pragma unroll
                for (int c = 0; c < kHsReg; ++c) {
                    const int j = j0 + 32 * c + lane;
                    x[0][c] = x[1][c] = (T)0;
                    if (j < m) {
                        const T wj = w[j], vj = v[j];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            x[q][c] = row[q][j];
                            if (i0 + q > k) x[q][c] -= vi[q] * wj;
                            acc[q] += x[q][c] * vj;
                        }
                        if (!fits) {
                            row[0][j] = x[0][c];
                            if (two) row[1][j] = x[1][c];
                        }
                    }
                }
            }
            sum2(acc[0], acc[1]);
            acc[0] *= beta;
            acc[1] *= beta;
            for (int j0 = 0; j0 < m; j0 += 32 * kHsReg) {
#pragma unroll
                for (int c = 0; c < kHsReg; ++c) {
                    const int j = j0 + 32 * c + lane;
                    if (j < m) {
                        const T vj = v[j];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            if (q == 1 && !two) break;
                            const T y = (fits ? x[q][c] : row[q][j]) - acc[q] * vj;
                            row[q][j] = y;
                            if (j == 0 && i0 + q >= k + 2) vn[i0 + q - k - 2] = y;
                        }
                    }
                }
            }
            if (lane < (two ? 2 : 1) && i0 + lane > k)
                A[(size_t)(i0 + lane) * n + k] = (i0 + lane == k + 1) ? alpha : (T)0;
        }
        __syncthreads();
        T* q = v; v = vn; vn = q;
    }
}

// One Francis double-shift sweep on rows and columns lo..hi, eigenvalues only, in windows of kQrNB
// bulge steps:
//  * chase: one warp carries the bulge through the window with the window's rows in registers, a
//    lane per column: left reflectors act within a lane, right reflectors act as far as the next
//    reflector needs them.
//  * strips: the other warps apply the window's kQrNB reflectors to the rest, a thread per row (right
//    reflectors) and per column to the right (left reflectors), with the row's or column's kQrNB + 2
//    entries in registers.
// So a window costs two barriers where a step cost two, and an entry is loaded and stored once per
// window.  A reflector is kept with tau v1 and tau v2, so a row or a column takes five multiply-adds
// of it (seven operations before: 2,000 pairs in FP64 591 -> 576 ms).  What bounds it is the chase, a
// chain of dependent instructions of one warp (FP32 ~350 cycles a step, FP64 ~2,900; the strips take
// 100 and 1,000, beside it).  118 buses: FP32 QR of one scenario from shared memory 8.2 -> 5.4 ms with
// windows, 4.3 with two sweeps at a time and the strips beside the chase (qr_sweep).
//
// Reflector of (x0, x1, x2): I - tau v v^T with v = (1, v1, v2), tau = 1 + |x0| / |x|.
template <typename T>
constexpr int kQrNB = sizeof(T) == 8 ? 8 : 12;   // measured: FP32 8 / 12 / 16, FP64 8 / 12 steps
constexpr int kQrCols = 32;                      // columns of a window kept in the chasing warp

template <typename T>
struct alignas(16) QrStep {                      // reflector of one step; t1 = tau v1, t2 = tau v2
    T v1, v2, tau, t1, t2;
};
template <typename T>
struct QrSpace {                                 // in shared memory
    QrStep<T> st[kQrNB<T>];
};

// 1 / sqrt(x) and 1 / x.  FP32: the hardware approximation and one Newton step, to rounding level: a
// reflector that is orthogonal to 2^-22 only, with the approximation's bias, moves the eigenvalues by
// more than the refinement allows for after the few hundred sweeps (one to three scenarios of 24,000
// went to the FP64 screen for it).  FP64: the FP32 approximation and one step of Halley's
// iteration (third order: 2^-22 -> 2^-66 relative before rounding), five and three FP64
// instructions.  Arguments within 1e-30 .. 1e30.
__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float qr_rsqrt(float x) {
    const float y = rsqrt_approx(x), e = fmaf(-(x * y), y, 1.0f);
    return fmaf(0.5f * y, e, y);
}
__device__ __forceinline__ float qr_rcp(float x) {
    const float y = rcp_approx(x);
    return fmaf(y, fmaf(-x, y, 1.0f), y);
}
// (The seeds' conversions run on the integer pipe: an FP64 conversion costs an FP64 instruction.)
__device__ __forceinline__ float qr_seed(double x) {        // x truncated to FP32
    const int hi = __double2hiint(x), lo = __double2loint(x);
    return __int_as_float(((hi - (896 << 20)) << 3) | ((unsigned)lo >> 29));
}
__device__ __forceinline__ double qr_wide(float y) {
    const int b = __float_as_int(y);
    return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}
__device__ __forceinline__ double qr_rsqrt(double x) {
    const double y = qr_wide(rsqrt_approx(qr_seed(x))), e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double qr_rcp(double x) {
    const double y = qr_wide(rcp_approx(qr_seed(x))), e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// x within about 1e-30 .. 1e30 (x a sum of squares: not negative; NaN and infinity are not)
__device__ __forceinline__ bool qr_safe(float x) { return x > 1e-30f && x < 1e30f; }
__device__ __forceinline__ bool qr_safe(double x) {
    return (unsigned)((__double2hiint(x) >> 20) - (1023 - 99)) <= 2u * 99u;
}

// matrices: row-major in global memory, packed Hessenberg rows in shared memory.  Wide: the type in which
// a sweep's shifts, its first column and its reflectors are formed before they are rounded to T.  FP64 for
// a matrix in global memory in both forms: the FP32 eigenvalues of a large network are its record (there is no
// refinement behind them).  600 pairs of 300 buses against their FP64 form: 3.0e-6 at most and 6.5e-7 on
// average, with all of it in FP32 3.3e-6 and 7.1e-7; one scenario takes 123 ms instead of 83, 600 pairs 264
// instead of 255.
template <typename T>
struct DenseMat {
    using Wide = double;
    T* a;
    int n;
    __device__ T* at(int i, int j) const { return a + (size_t)i * n + j; }
};
template <typename T>
struct PackedMat {
    using Wide = T;
    T* a;
    const int* rb;
    __device__ T* at(int i, int j) const { return a + rb[i] + j; }
};

// (x0, x1, x2): the bulge column's entries (x2 = 0 where the row does not exist); its reflector and the
// column's new first entry.  (x1 = x2 = 0 gives v = 0, tau = 2: a change of sign.)
template <typename T>
struct QrRefl {
    T v1, v2, tau, alpha;
};

template <typename T>
__device__ __forceinline__ QrRefl<T> qr_reflector_of(T x0, T x1, T x2, T s) {
    QrRefl<T> h;
    const T r = qr_rsqrt(s);
    h.tau = fabs(x0) * r + (T)1;
    const T f = copysign(r, x0) * qr_rcp(h.tau);
    h.v1 = x1 * f;
    h.v2 = x2 * f;
    h.alpha = -copysign(s * r, x0);
    return h;
}

// out of the range where the squares are safe
template <typename T>
__device__ __noinline__ QrRefl<T> qr_reflector_scaled(T x0, T x1, T x2) {
    const T m = fmax(fabs(x0), fmax(fabs(x1), fabs(x2)));
    if (!(m > (T)0) || !isfinite(m)) return QrRefl<T>{(T)0, (T)0, (T)0, x0};   // nothing to reflect (or to save)
    x0 /= m; x1 /= m; x2 /= m;
    QrRefl<T> h = qr_reflector_of(x0, x1, x2, x0 * x0 + (x1 * x1 + x2 * x2));
    h.alpha *= m;
    return h;
}

template <typename T>
__device__ __forceinline__ QrRefl<T> qr_reflector(T x0, T x1, T x2) {
    const T s = x0 * x0 + (x1 * x1 + x2 * x2);
    if (!qr_safe(s)) return qr_reflector_scaled(x0, x1, x2);
    return qr_reflector_of(x0, x1, x2, s);
}

// The bulge between two steps: the entries of its column k - 1 (x, rows k .. k + 2) and the one it
// fills in column k (b, row k + 2).  They live in registers, never in the matrix.
template <typename T, typename R>
struct QrBulge {
    R x0, x1, x2;
    T b;
};

// Reflectors first .. cnt - 1 on the entries y of one row or column.
template <bool kFull, typename T>
__device__ __forceinline__ void qr_apply(T (&y)[kQrNB<T> + 2], const QrSpace<T>& sp, int first, int cnt) {
#pragma unroll
    for (int t = 0; t < kQrNB<T>; ++t) {
        if (!kFull && (t >= cnt || t < first)) continue;
        const QrStep<T> st = sp.st[t];
        const T d = y[t] + st.v1 * y[t + 1] + st.v2 * y[t + 2];
        y[t] -= st.tau * d;
        y[t + 1] -= st.t1 * d;
        y[t + 2] -= st.t2 * d;
    }
}

// Steps kw .. kw + cnt - 1 of the sweep, one warp, the bulge in and out.  The right reflectors are
// applied to the three rows below the bulge at once, as the next reflector needs; the window's rows
// take the rest of them in the strips, each from its own step on.  So every entry takes its
// reflections in the order of the step-by-step sweep.  (All left reflectors first and the right ones
// after them is the same product and a shorter step, but the entries below the bulge then come
// from cancellation within the window: in FP32 one to three scenarios of 24,000 did not converge.)
//
// In FP32 the chain from one reflector to the next runs on copies of its few entries that every
// lane keeps: rows k .. k + 2 of columns k and k + 1, and column k + 2, fetched before the reflector
// is known.  An FP64 instruction takes longer than a shuffle, so there the entries are fetched.
template <typename T, typename M>
__device__ __forceinline__ void qr_chase_full(const M& A, int lo, int hi, int kw, QrBulge<T, typename M::Wide>& bu,
                                              QrSpace<T>& sp) {
    using R = typename M::Wide;
    constexpr int NB = kQrNB<T>;
    constexpr bool kCopies = sizeof(T) == 4;
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31, col = kw + lane;
    T w[NB + 3];
#pragma unroll
    for (int r = 0; r < NB + 3; ++r)
        w[r] = (col <= hi && lane + 1 >= r) ? *A.at(kw + r, col) : (T)0;
    if (lane == 0) w[2] = bu.b;
    R x0 = bu.x0, x1 = bu.x1, x2 = bu.x2;
    T sub = 0;                                            // subdiagonal entry (kw + lane, kw + lane - 1)
    T m00 = 0, m01 = 0, m10 = 0, m11 = 0, m20 = 0, m21 = 0;
    if (kCopies) {
        m00 = __shfl_sync(all, w[0], 0); m01 = __shfl_sync(all, w[0], 1);
        m10 = __shfl_sync(all, w[1], 0); m11 = __shfl_sync(all, w[1], 1);
        m20 = bu.b;                      m21 = __shfl_sync(all, w[2], 1);
    }
#pragma unroll
    for (int t = 0; t < NB; ++t) {
        T c0 = 0, c1 = 0, c2 = 0, s3 = 0;
        if (kCopies) {
            c0 = __shfl_sync(all, w[t], t + 2);
            c1 = __shfl_sync(all, w[t + 1], t + 2);
            c2 = __shfl_sync(all, w[t + 2], t + 2);
            s3 = __shfl_sync(all, w[t + 3], t + 2);
        }
        const QrRefl<R> h = qr_reflector(x0, x1, x2);
        const T v1 = (T)h.v1, v2 = (T)h.v2, tau = (T)h.tau, t1 = (T)(h.tau * h.v1), t2 = (T)(h.tau * h.v2);
        sp.st[t] = {v1, v2, tau, t1, t2};                         // the same from every lane
        if (lane == t) sub = (T)h.alpha;
        T da, db, dc;
        if (kCopies) {
            const T d0 = m00 + v1 * m10 + v2 * m20, d1 = m01 + v1 * m11 + v2 * m21, d2 = c0 + v1 * c1 + v2 * c2;
            const T n10 = m10 - t1 * d0, n20 = m20 - t2 * d0, n11 = m11 - t1 * d1, n21 = m21 - t2 * d1,
                    n12 = c1 - t1 * d2, n22 = c2 - t2 * d2;
            da = n10 + v1 * n11 + v2 * n12;
            db = n20 + v1 * n21 + v2 * n22;
            dc = v2 * s3;
            x0 = n10 - tau * da;
            x1 = n20 - tau * db;
            x2 = -(tau * dc);
            m00 = n11 - t1 * da; m01 = n12 - t2 * da;
            m10 = n21 - t1 * db; m11 = n22 - t2 * db;
            m20 = -(t1 * dc);    m21 = s3 - t2 * dc;
        }
        const T d = w[t] + v1 * w[t + 1] + v2 * w[t + 2]; // left, rows kw + t ..
        w[t] -= tau * d;
        w[t + 1] -= t1 * d;
        w[t + 2] -= t2 * d;
        if (!kCopies) {                                   // right, the three rows below
            const T a0 = __shfl_sync(all, w[t + 1], t), a1 = __shfl_sync(all, w[t + 1], t + 1),
                    a2 = __shfl_sync(all, w[t + 1], t + 2);
            const T b0 = __shfl_sync(all, w[t + 2], t), b1 = __shfl_sync(all, w[t + 2], t + 1),
                    b2 = __shfl_sync(all, w[t + 2], t + 2);
            da = a0 + v1 * a1 + v2 * a2;
            db = b0 + v1 * b1 + v2 * b2;
            dc = v2 * __shfl_sync(all, w[t + 3], t + 2);
        }
        // (column kw + t itself is the next bulge column: only needed as x)
        const T co = lane == t + 1 ? t1 : lane == t + 2 ? t2 : kCopies ? (T)0 : lane == t ? tau : (T)0;
        w[t + 1] -= co * da;
        w[t + 2] -= co * db;
        w[t + 3] -= co * dc;
        if (!kCopies) {
            x0 = __shfl_sync(all, w[t + 1], t);
            x1 = __shfl_sync(all, w[t + 2], t);
            x2 = __shfl_sync(all, w[t + 3], t);
        }
    }
    bu = QrBulge<T, R>{x0, x1, x2, kCopies ? m20 : __shfl_sync(all, w[NB + 2], NB)};
    // a column of the window is final on and above its diagonal; its subdiagonal entry is the next
    // step's alpha (the last one's, the next window's, or x0 at the end of the sweep)
#pragma unroll
    for (int r = 0; r < NB + 3; ++r)
        if (col <= hi && (lane >= r || (lane + 1 == r && lane >= NB)))
            *A.at(kw + r, col) = w[r];
    if (lane < NB && col > lo) *A.at(col, col - 1) = sub;
}

// qr_chase_full takes a window that ends three rows above the block's end or higher, unrolled; qr_chase any, in a
// loop of kQrUnroll steps with the rows in a rolling buffer.  The size of the code counts: with all SMs at
// it a warp waits for its instructions (118 buses, three scenarios on each SM: 15.0 ms with both kinds
// of windows unrolled and the strips inlined four times, 13.4 like this; one scenario alone took 4.1 and
// 4.4 ms.  Everything rolled: 15.0 and 4.9).
constexpr int kQrUnroll = 4;
template <typename T, typename M>
__device__ __forceinline__ void qr_chase(const M& A, int lo, int hi, int kw, int cnt, QrBulge<T, typename M::Wide>& bu,
                                         QrSpace<T>& sp) {
    using R = typename M::Wide;
    constexpr int NB = kQrNB<T>, U = kQrUnroll;
    static_assert(NB % U == 0 && U >= 3, "");
    constexpr bool kCopies = sizeof(T) == 4;
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31, col = kw + lane;
    auto load = [&](int r) -> T {
        return (kw + r <= hi && col <= hi && lane + 1 >= r) ? *A.at(kw + r, col) : (T)0;
    };
    // a column of the window is final on and above its diagonal; its subdiagonal entry is the next
    // step's alpha (the last one's, the next window's, or x0 at the end of the sweep)
    auto store = [&](int r, T x) {
        if (kw + r <= hi && col <= hi && (lane >= r || (lane + 1 == r && lane >= cnt))) *A.at(kw + r, col) = x;
    };
    T w[U + 3];                                           // rows t0 ..
#pragma unroll
    for (int r = 0; r < U + 3; ++r) w[r] = load(r);
    if (lane == 0) w[2] = bu.b;
    R x0 = bu.x0, x1 = bu.x1, x2 = bu.x2;
    T sub = 0;                                            // subdiagonal entry (kw + lane, kw + lane - 1)
    T m00 = 0, m01 = 0, m10 = 0, m11 = 0, m20 = 0, m21 = 0;
    if (kCopies) {
        m00 = __shfl_sync(all, w[0], 0); m01 = __shfl_sync(all, w[0], 1);
        m10 = __shfl_sync(all, w[1], 0); m11 = __shfl_sync(all, w[1], 1);
        m20 = bu.b;                      m21 = __shfl_sync(all, w[2], 1);
    }
#pragma unroll 1
    for (int t0 = 0; t0 < cnt; t0 += U) {
        T next[U];                                        // rows of the steps after these
#pragma unroll
        for (int u = 0; u < U; ++u) next[u] = t0 + U < NB ? load(t0 + U + 3 + u) : (T)0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = t0 + u;
            if (t >= cnt) break;
            T c0 = 0, c1 = 0, c2 = 0, s3 = 0;
            if (kCopies) {
                c0 = __shfl_sync(all, w[u], t + 2);
                c1 = __shfl_sync(all, w[u + 1], t + 2);
                c2 = __shfl_sync(all, w[u + 2], t + 2);
                s3 = __shfl_sync(all, w[u + 3], t + 2);
            }
            const QrRefl<R> h = qr_reflector(x0, x1, x2);
            const T v1 = (T)h.v1, v2 = (T)h.v2, tau = (T)h.tau, t1 = (T)(h.tau * h.v1), t2 = (T)(h.tau * h.v2);
            sp.st[t] = {v1, v2, tau, t1, t2};             // the same from every lane
            if (lane == t) sub = (T)h.alpha;
            T da, db, dc;
            if (kCopies) {
                const T d0 = m00 + v1 * m10 + v2 * m20, d1 = m01 + v1 * m11 + v2 * m21, d2 = c0 + v1 * c1 + v2 * c2;
                const T n10 = m10 - t1 * d0, n20 = m20 - t2 * d0, n11 = m11 - t1 * d1, n21 = m21 - t2 * d1,
                        n12 = c1 - t1 * d2, n22 = c2 - t2 * d2;
                da = n10 + v1 * n11 + v2 * n12;
                db = n20 + v1 * n21 + v2 * n22;
                dc = v2 * s3;
                x0 = n10 - tau * da;
                x1 = n20 - tau * db;
                x2 = -(tau * dc);
                m00 = n11 - t1 * da; m01 = n12 - t2 * da;
                m10 = n21 - t1 * db; m11 = n22 - t2 * db;
                m20 = -(t1 * dc);    m21 = s3 - t2 * dc;
            }
            const T d = w[u] + v1 * w[u + 1] + v2 * w[u + 2]; // left, rows kw + t ..
            w[u] -= tau * d;
            w[u + 1] -= t1 * d;
            w[u + 2] -= t2 * d;
            if (!kCopies) {                               // right, the three rows below
                const T a0 = __shfl_sync(all, w[u + 1], t), a1 = __shfl_sync(all, w[u + 1], t + 1),
                        a2 = __shfl_sync(all, w[u + 1], t + 2);
                const T b0 = __shfl_sync(all, w[u + 2], t), b1 = __shfl_sync(all, w[u + 2], t + 1),
                        b2 = __shfl_sync(all, w[u + 2], t + 2);
                da = a0 + v1 * a1 + v2 * a2;
                db = b0 + v1 * b1 + v2 * b2;
                dc = v2 * __shfl_sync(all, w[u + 3], t + 2);
            }
            // (column kw + t itself is the next bulge column: only needed as x)
            const T co = lane == t + 1 ? t1 : lane == t + 2 ? t2 : kCopies ? (T)0 : lane == t ? tau : (T)0;
            w[u + 1] -= co * da;
            w[u + 2] -= co * db;
            w[u + 3] -= co * dc;
            if (!kCopies) {
                x0 = __shfl_sync(all, w[u + 1], t);
                x1 = __shfl_sync(all, w[u + 2], t);
                x2 = __shfl_sync(all, w[u + 3], t);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) store(t0 + u, w[u]);
#pragma unroll
        for (int r = 0; r < 3; ++r) w[r] = w[r + U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u + 3] = next[u];
    }
    const int end = (cnt + U - 1) / U * U;
    bu = QrBulge<T, R>{x0, x1, x2, kCopies ? m20 : __shfl_sync(all, w[2], NB)};   // (the last window's is not used)
#pragma unroll
    for (int r = 0; r < 3; ++r) store(end + r, w[r]);
    if (lane < cnt && col > lo) *A.at(col, col - 1) = sub;
    if (kw + cnt == hi && lane == 0) *A.at(hi, hi - 1) = (T)x0;
}

// One window's strips: its reflectors on 32 of the rows above it and its own (each from its own step
// on), task < rows(), or on 32 of the columns right of it, task - rows() < cols().
template <typename T, typename M>
struct QrStrips {
    static constexpr int NB = kQrNB<T>;
    const M& A;
    const QrSpace<T>& sp;
    int lo, hi, kw, cnt;
    __device__ QrStrips(const M& A_, const QrSpace<T>& sp_, int lo_, int hi_, int kw_)
        : A(A_), sp(sp_), lo(lo_), hi(hi_), kw(kw_), cnt(min(NB, hi_ - kw_)) {}
    __device__ bool live() const { return kw >= lo && kw < hi; }
    __device__ int rows() const { return (kw + cnt - lo + 31) >> 5; }
    __device__ int cols() const { return (max(0, hi + 1 - kw - kQrCols) + 31) >> 5; }
    __device__ int far() const { return live() ? rows() + max(0, cols() - 1) : 0; }   // all but the nearest columns
    __device__ __forceinline__ void run(int task) const {
        const int lane = threadIdx.x & 31;
        T y[NB + 2];
        if (task < rows()) {
            const int i = lo + 32 * task + lane, first = max(0, i - kw);
            if (i >= kw + cnt) return;
            T* row = A.at(i, kw);
            if (cnt == NB && kw + NB + 1 <= hi && lo + 32 * task + 31 < kw) {
#pragma unroll
                for (int c = 0; c < NB + 2; ++c) y[c] = row[c];
                qr_apply<true>(y, sp, 0, NB);
#pragma unroll
                for (int c = 0; c < NB + 2; ++c) row[c] = y[c];
            } else {
#pragma unroll
                for (int c = 0; c < NB + 2; ++c) y[c] = (c >= first && c <= cnt + 1 && kw + c <= hi) ? row[c] : (T)0;
                qr_apply<false>(y, sp, first, cnt);
#pragma unroll
                for (int c = 0; c < NB + 2; ++c)
                    if (c >= first && c <= cnt + 1 && kw + c <= hi) row[c] = y[c];
            }
        } else {                                                 // (columns right of a window: it is full)
            const int j = kw + kQrCols + 32 * (task - rows()) + lane;
            if (j > hi) return;
#pragma unroll
            for (int r = 0; r < NB + 2; ++r) y[r] = *A.at(kw + r, j);
            qr_apply<true>(y, sp, 0, NB);
#pragma unroll
            for (int r = 0; r < NB + 2; ++r) *A.at(kw + r, j) = y[r];
        }
    }
};

// First column of the double-shift step, (H - a I)(H - b I) e1 / h10 of the block lo..hi, a and b the
// eigenvalues of its trailing 2x2 block (or, if exceptional, a pair off its last entry by the size of
// the last subdiagonals), in differences to the leading diagonal entry: formed from the shifts' sum
// and product, a block whose eigenvalues differ by little (the exciters' cluster near -1/T_A) loses
// the differences to cancellation in FP32 and its sweeps go nowhere (118 buses: 331 -> 276 sweeps a
// scenario, and the scenario in 20,000 that ran to the sweep limit converges).
template <typename R>
struct QrShift {
    R a11, a22, w;                               // trailing 2x2 block: diagonal, product of the off-diagonal
};
template <typename R, typename M>
__device__ __forceinline__ QrShift<R> qr_shift(const M& A, int hi, bool exceptional) {
    QrShift<R> q{(R)*A.at(hi - 1, hi - 1), (R)*A.at(hi, hi), (R)*A.at(hi - 1, hi) * (R)*A.at(hi, hi - 1)};
    if (exceptional) {
        const R ww = fabs((R)*A.at(hi, hi - 1)) + fabs((R)*A.at(hi - 1, hi - 2));
        q.a11 = q.a22 = q.a22 + (R)0.75 * ww;
        q.w = (R)-0.4375 * ww * ww;
    }
    return q;
}
template <typename T, typename R, typename M>
__device__ __forceinline__ void qr_start(const M& A, int lo, const QrShift<R>& q, QrBulge<T, R>& bu) {
    const R h00 = *A.at(lo, lo), h01 = *A.at(lo, lo + 1), h10 = *A.at(lo + 1, lo), h11 = *A.at(lo + 1, lo + 1);
    const R r = q.a22 - h00, s = q.a11 - h00;
    bu.x0 = (r * s - q.w) / h10 + h01;
    bu.x1 = h11 - h00 - r - s;
    bu.x2 = *A.at(lo + 2, lo + 1);
    bu.b = (T)0;
}

// Whole sweep by the block, or (two) two sweeps, the second one kQrLag steps behind the first with the
// same shifts.  What bounds a sweep is the chase, a serial chain of one warp, so everything else runs
// beside it: warp 0 (and warp 1, the second sweep) chases a window while the other warps apply the strips
// of the window before; only the 32 columns nearest to a window, which the next one starts in, wait for
// the chase and are waited for.
//
// Where the two sweeps meet: the second one's chase ends left of the columns that the first one's
// right reflectors mix (kQrLag - kQrNB >= kQrCols), and its near columns hold all or none of them, so no
// right reflector mixes columns with and without the second one's left reflectors.
//
// The shifts of the second sweep are a sweep old: 118 buses, orders 259 .. 269: 306 sweeps a matrix
// instead of 274, in little more than half the chases.  (Eigenvalues of the trailing 4x4 block as shifts:
// 303 sweeps, and a serial eigenvalue problem for each pair.  In FP64, whose sweeps at two or more blocks
// per SM are bound by the pipe and not by the chase, two at a time are not used.)  From blocks of kQrPair
// on the lag is worth it; 44, 60 and 90 measure the same.
// 118 buses, FP32 QR of one scenario 5.4 -> 4.3 ms, 10,000 pairs mixed 883 -> 817 ms; FP64, 240 single
// outages 133 -> 129 ms, 2,000 pairs 576 -> 565 ms.
template <typename T>
constexpr int kQrLag = (kQrCols + 2 * kQrNB<T> - 1) / kQrNB<T> * kQrNB<T>;
static_assert(kQrLag<float> + kQrNB<float> + 2 <= 2 * kQrCols && kQrLag<double> + kQrNB<double> + 2 <= 2 * kQrCols,
              "the second sweep's near columns hold the first one's window");
constexpr int kQrPair = 60;
template <bool kTwo, typename T, typename M>
__device__ __forceinline__ void qr_sweep(const M& A, int lo, int hi, bool exceptional, bool two,
                                         QrSpace<T> (&sp)[2][2], int nthreads) {
    using R = typename M::Wide;
    constexpr int NB = kQrNB<T>;
    const int sweeps = kTwo && two ? 2 : 1;
    const int warp = threadIdx.x >> 5, nworkers = (nthreads >> 5) - sweeps;
    const int last = hi + (sweeps - 1) * kQrLag<T>;
    QrBulge<T, R> bu{};
    QrShift<R> q{};
    if (warp < sweeps) q = qr_shift<R>(A, hi, exceptional);
    int par = 0;
    for (int ka = lo;; ka += NB, par ^= 1) {                      // (the last round: strips only)
        const int kw = ka - warp * kQrLag<T>;                     // of a chasing warp
        if (warp < sweeps && kw >= lo && kw < hi) {
            if (kw == lo) qr_start<T>(A, lo, q, bu);
            if (kw + NB + 2 <= hi) qr_chase_full(A, lo, hi, kw, bu, sp[warp][par]);
            else qr_chase(A, lo, hi, kw, min(NB, hi - kw), bu, sp[warp][par]);
        }
        // One loop (one copy of the strips' code) for both kinds: the windows' before, but for their nearest
        // columns, by the other warps, then, after a barrier, the nearest of these by the chasing warps.
#pragma unroll 1
        for (int near = 0; near < 2; ++near) {
            int task = 0, n = 0, na = 0;
            if (near) {
                n = warp < sweeps && kw >= lo && kw + kQrCols <= hi;
            } else if (warp >= sweeps) {
                na = n = QrStrips<T, M>(A, sp[0][0], lo, hi, ka - NB).far();
                if (sweeps == 2) n += QrStrips<T, M>(A, sp[0][0], lo, hi, ka - NB - kQrLag<T>).far();
                task = warp - sweeps;
            }
            for (; task < n; task += nworkers) {                  // (near: one)
                const int second = !kTwo ? 0 : near ? warp : task >= na;
                const QrStrips<T, M> st(A, sp[second][near ? par : par ^ 1], lo, hi,
                                        near ? kw : ka - NB - second * kQrLag<T>);
                const int t = task - second * na, rows = st.rows();
                st.run(near ? rows : t < rows ? t : t + 1);
            }
            __syncthreads();
            if (ka >= last) return;
        }
    }
}

// Francis double-shift QR on the Hessenberg matrix in global memory,
// eigenvalues only (updates restricted to the active block lo..hi).
// sh.fail = 2 if it does not converge in 30 n sweeps.
template <typename T>
__device__ __noinline__ void hqr_global(T* Ag, const int n, double* wr, double* wi, DShared& sh) {
    static_assert(sizeof(typename DenseMat<T>::Wide) == 8, "no refinement follows: shifts and reflectors in FP64");
    __shared__ QrSpace<T> sp[2][2];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const DenseMat<T> A{Ag, n};
    const double eps = (sizeof(T) == 8) ? kEps : (double)kDeflTol;       // deflation tolerance
    double hmax;
    {
        double hm = 0.0;
        for (int i = tid >> 5; i < n; i += nthr / 32)
            for (int j = max(0, i - 1) + (tid & 31); j < n; j += 32) hm = fmax(hm, fabs((double)*A.at(i, j)));
        hmax = bmax(sh, hm);
    }
    int hi = n - 1, its = 0;
    while (hi >= 0) {
        // top of the unreduced block ending at hi: largest l <= hi with a negligible A[l][l-1]
        int cand = 0;
        for (int l = 1 + tid; l <= hi; l += nthr) {
            double sd = fabs((double)*A.at(l - 1, l - 1)) + fabs((double)*A.at(l, l));
            if (sd == 0.0) sd = hmax;
            if (fabs((double)*A.at(l, l - 1)) <= eps * sd) cand = max(cand, l);
        }
        const int lo = bmax_int(sh, cand);
        if (lo == hi) {
            if (tid == 0) {
                wr[hi] = *A.at(hi, hi);
                wi[hi] = 0.0;
            }
            hi -= 1;
            its = 0;
            continue;
        }
        if (lo == hi - 1) {
            if (tid == 0) {
                double re[2], im[2];
                eig2(*A.at(hi - 1, hi - 1), *A.at(hi - 1, hi), *A.at(hi, hi - 1), *A.at(hi, hi), re, im);
                wr[hi - 1] = re[0]; wi[hi - 1] = im[0];
                wr[hi] = re[1]; wi[hi] = im[1];
            }
            hi -= 2;
            its = 0;
            continue;
        }
        if (its >= 30 * n) {
            if (tid == 0) sh.fail = 2;
            break;
        }
        ++its;
        qr_sweep<false, T>(A, lo, hi, its == 10 || its == 20, false, sp, nthr);
    }
    __syncthreads();                               // eigenvalues and sh.fail written by thread 0
}

template <typename T>
__device__ void eigen_screen(T* A, const int n, T* cs, T* rs, T* v, T* part, double* wr, double* wi, DShared& sh) {
    balance<T>(A, n, cs, rs, v, sh);             // (the factors are not needed: eigenvalues only)
    hessenberg<T>(A, n, v, cs, rs, part, sh);
    hqr_global<T>(A, n, wr, wi, sh);
}

// ---------------------------------------------------------------------------
// Packed Hessenberg storage for the shared-memory QR: row i keeps columns
// max(i-3, 0)..n-1: the Hessenberg part, and two sub-diagonals more that stay zero (a
// sweep's bulge is in registers; the rows' offsets are those of a bulge in the matrix).  hq_off(n, i) is the offset of row i; hq_off(n, n) the size.
__host__ __device__ inline int hq_start(int i) { return i > 3 ? i - 3 : 0; }
__host__ __device__ inline int hq_off(int n, int i) {
    if (i <= 3) return n * i;
    return 3 * n + (i - 3) * (n + 3) - (i * (i - 1) / 2 - 3);
}
constexpr int kHqHead = 4;          // floats before the packed matrix: the order n (int bits), padding

// Slot of one scenario in the balanced-matrix buffer (front kernel -> cluster
// Hessenberg kernel -> refinement kernel), floats: the head, the balanced
// matrix (row-major n x n), then the balancing factors D (the balanced matrix is
// D^-1 A D) and the Householder factors beta_k.  The cluster kernel overwrites
// the matrix area with the Householder vectors once it has loaded the matrix:
// vector k (entries for rows k+1..n-1, the first one the reflector's head) at
// refl_off(n, k).
__host__ __device__ inline size_t ab_mat_floats(int nmax) { return ((size_t)nmax * nmax + 3) & ~(size_t)3; }
__host__ __device__ inline size_t ab_d_off(int nmax) { return kHqHead + ab_mat_floats(nmax); }
__host__ __device__ inline size_t ab_beta_off(int nmax) { return ab_d_off(nmax) + (((size_t)nmax + 3) & ~(size_t)3); }
__host__ __device__ inline size_t ab_stride(int nmax) { return ab_beta_off(nmax) + (((size_t)nmax + 3) & ~(size_t)3); }
__host__ __device__ inline int refl_off(int n, int k) { return k * (n - 1) - (k * (k - 1)) / 2; }

// Candidates of the FP64 refinement per scenario (shared-memory QR -> refinement
// kernel), floats: [0] count (int bits), [1] flags (int bits; bit 2c: candidate c
// may carry the largest real part, bit 2c+1: the smallest damping ratio), then
// the FP32 eigenvalue (re, im >= 0) of each candidate.
constexpr int kRefK = 4;                     // candidates per scenario at most (more: FP64 re-run)
constexpr int kCandStride = 4 + 2 * kRefK;
// Bound on the distance of an FP32 eigenvalue of the 118-bus state matrix from the
// exact one (measured differences are below 3e-5): an eigenvalue can decide max Re
// or min zeta only if its FP32 value is within this bound of deciding it.
constexpr float kEigDelta = 1e-3f;
// Refined statistics within this distance of a threshold (max Re = 0, min zeta =
// damping_min) are decided by the FP64 screen instead (the refined values are within
// ~1e-9 of the FP64 screen's).
constexpr double kRefinedGuard = 1e-7;

// max Re and min damping ratio over the n eigenvalues (block-wide, result on all threads)
__device__ void eig_stats(DShared& sh, int n, const double* wr, const double* wi, double& maxre, double& minz) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    double mr = -INFINITY, mz = INFINITY;
    if (!sh.fail) {
        for (int i = tid; i < n; i += nthr) {
            mr = fmax(mr, wr[i]);
            const double mg = sqrt(wr[i] * wr[i] + wi[i] * wi[i]);
            mz = fmin(mz, mg > 0.0 ? -wr[i] / mg : 1.0);
        }
    }
    maxre = bmax(sh, mr);
    minz = -bmax(sh, -mz);
}

// Kernel modes.  FULL64: FP64 screen of every converged OPF point (the FP64
// form).  MIXED_INLINE: FP32 screen in global memory with the FP64 re-run
// inline (mixed form, kept for networks the tensor-core path does not take).
// FRONT: model and FP32 balancing; the balanced matrix goes to a per-scenario
// buffer for hess_cluster_kernel.  RERUN: FP64 screen of the scenarios that
// the FP32 screen could not decide (status 6).  FRONT_LARGE / QR_LARGE: the
// mixed form of networks whose Hessenberg matrix exceeds shared memory: the
// balanced FP32 matrix, padded to the network's largest state order with a
// decoupled -1 diagonal (so one batch has one order), goes to the tensor-core
// blocked Hessenberg reduction (k_tc.cu), then FP32 QR in global memory over the
// padded order with statistics over the first n eigenvalues (the padding's -1
// eigenvalues deflate first, into the last positions), guard band to RERUN.
enum { DYN_FULL64 = 0, DYN_MIXED_INLINE = 1, DYN_FRONT = 2, DYN_RERUN = 3, DYN_FRONT_LARGE = 4, DYN_QR_LARGE = 5 };

template <int kMode>
__global__ void __launch_bounds__(kMaxThreads, 1)
dyn_kernel(DevNet net, EvalArgs a, OpfOut o, double damping_min, double* scratch, size_t per_cta, DLay L,
           float* hbuf, size_t hstride, double* a64, size_t a64stride, int* counter) {
    __shared__ DShared sh;
    extern __shared__ double dsm[];   // [ng] ints (compact -> generator id), then cs, rs, v [5 ng] each
    int* gidx = reinterpret_cast<int*>(dsm);
    double* cs_d = dsm + ((net.ng + 1) >> 1);
    double* rs_d = cs_d + 5 * net.ng;
    double* v_d = rs_d + 5 * net.ng;
    const int tid = threadIdx.x, nthr = blockDim.x;
    double* W = scratch + per_cta * blockIdx.x;
    const int nb = net.nb, ng = net.ng, nbr = net.nbr;
    const int nx = 2 * nb + 2 * ng;
    const double* Pd = net.Pd + (size_t)a.level * nb;
    const double* Qd = net.Qd + (size_t)a.level * nb;

    for (;;) {
        if (tid == 0) sh.scen = atomicAdd(counter, 1);
        __syncthreads();
        const int s = sh.scen;
        if (s >= a.n) break;
        if (o.status[s] != (kMode == DYN_RERUN ? 6 : 1)) {
            __syncthreads();
            continue;
        }
        if (kMode == DYN_QR_LARGE) {                  // QR of the padded Hessenberg matrix (tensor-core reduction)
            float* slot = hbuf + (size_t)s * hstride;
            const int n = __float_as_int(slot[0]), nmax = 5 * ng - 1;
            double* wr = W + L.wr;
            double* wi = W + L.wi;
            if (tid == 0) sh.fail = 0;
            __syncthreads();
            hqr_global<float>(slot + kHqHead, nmax, wr, wi, sh);
            double maxre = 0.0, minz = 0.0;
            eig_stats(sh, n, wr, wi, maxre, minz);
            if (tid == 0) {
                const bool near = sh.fail || !(fabs(maxre) > kGuardRe) || !(fabs(minz - damping_min) > kGuardZeta);
                if (near) {                           // decision too close to call in FP32: FP64 screen
                    o.status[s] = 6;
                    atomicAdd(a.reruns, 1);
                } else {
                    uint8_t k;
                    if (maxre >= 0.0) k = CS_SS_UNSTABLE;
                    else if (minz < damping_min) k = CS_SS_POORLY_DAMPED;
                    else k = CS_SECURE;
                    if (a.out.n_islands[s] > 1) {     // main island: the scenario's class stays ISLANDED
                        if (a.out.main_klass) a.out.main_klass[s] = k;
                    } else {
                        a.out.klass[s] = k;
                        a.out.severe[s] = (k != CS_SECURE);
                    }
                    a.out.max_re[s] = maxre;
                    a.out.min_zeta[s] = minz;
                }
            }
            __syncthreads();
            continue;
        }
        const Outage out = decode_outage(nbr, ng, a.ei[s], a.ej[s], a.ek ? a.ek[s] : -1);
        const double* xs = o.x + (size_t)s * nx;
        // main island of an islanded scenario: the OPF point has Vm = 0 at the buses
        // outside it; those buses, their branches and their machines are out of the model
        const bool isl = a.out.n_islands[s] > 1;
        auto live = [&](int i) { return !isl || xs[nb + i] != 0.0; };
        if (tid == 0) {
            int m = 0;
            for (int k = 0; k < ng; ++k)
                if (!gen_out(out, k) && live(net.gbus[k])) gidx[m++] = k;
            sh.m = m;
            sh.nn = 5 * m - 1;           // angles referred to the first in-service machine
            sh.fail = 0;
        }
        __syncthreads();
        const int m = sh.m, n = sh.nn;

        // ---- 1. assemble Y_bb on the symbolic pattern ----
        for (int tg = tid; tg < nb + net.nL; tg += nthr) {
            if (tg < nb) {
                const int j = tg, i = net.perm[j];
                if (!live(i)) {                       // de-energised bus: identity row
                    st(W + L.Yd + 2 * j, cm(1.0, 0.0));
                    continue;
                }
                const double Vm = xs[nb + i];
                cplx y = cm(net.gsh[i], net.bsh[i]);
                y = y + (1.0 / (Vm * Vm)) * cm(Pd[i], -Qd[i]);
                for (int e = net.bus_br_ptr[i]; e < net.bus_br_ptr[i + 1]; ++e) {
                    const int code = net.bus_br[e];
                    const int b = code >> 1, side = code & 1;
                    if (br_out(out, b)) continue;
                    y = y + (side ? net.ytt[b] : net.yff[b]);
                }
                for (int e = net.bus_gen_ptr[i]; e < net.bus_gen_ptr[i + 1]; ++e) {
                    const int k = net.bus_gen[e];
                    if (gen_out(out, k)) continue;
                    y = y + cm(0.0, -1.0 / net.xp[k]);
                }
                st(W + L.Yd + 2 * j, y);
            } else {
                const int q = tg - nb;
                const int Rb = net.perm[net.Lrow[q]];
                cplx y = cm(0.0, 0.0);
                for (int e = net.blk_br_ptr[q]; e < net.blk_br_ptr[q + 1]; ++e) {
                    const int b = net.blk_br[e];
                    if (br_out(out, b) || !live(net.f[b])) continue;
                    y = y + ((net.f[b] == Rb) ? net.yft[b] : net.ytf[b]);
                }
                st(W + L.Yu + 2 * q, y);
            }
        }
        __syncthreads();
        // ---- complex LDL^T, level by level ----
        for (int lev = 0; lev < net.nlevels; ++lev) {
            const int t0 = net.tgt_ptr[lev], t1 = net.tgt_ptr[lev + 1];
            for (int w = tid; w < t1 - t0; w += nthr) {
                const int tg = net.tgt[t0 + w];
                double* A = (tg < nb) ? (W + L.Yd + 2 * tg) : (W + L.Yu + 2 * (tg - nb));
                cplx acc = ld(A);
                for (int u = net.upd_ptr[tg]; u < net.upd_ptr[tg + 1]; ++u)
                    acc = acc - ld(W + L.Yl + 2 * net.upd_a[u]) * ld(W + L.Yu + 2 * net.upd_b[u]);
                st(A, acc);
            }
            __syncthreads();
            for (int w = net.lev_ptr[lev] + tid; w < net.lev_ptr[lev + 1]; w += nthr) {
                const int j = net.lev_col[w];
                const cplx d = ld(W + L.Yd + 2 * j);
                if (!(abs2(d) > 0.0) || !isfinite(abs2(d))) sh.fail = 1;
                st(W + L.Ydi + 2 * j, cdiv(cm(1.0, 0.0), d));
            }
            __syncthreads();
            for (int w = tid; w < t1 - t0; w += nthr) {
                const int tg = net.tgt[t0 + w];
                if (tg < nb) continue;
                const int q = tg - nb;
                st(W + L.Yl + 2 * q, ld(W + L.Yu + 2 * q) * ld(W + L.Ydi + 2 * net.Lcol[q]));
            }
            __syncthreads();
        }
        // ---- 2. machine-bus entries of Y_bb^{-1}: one sparse solve per machine ----
        for (int kk = tid; kk < m; kk += nthr) {
            double* y = W + L.rhs + (size_t)2 * nb * kk;
            for (int j = 0; j < nb; ++j) { y[2 * j] = 0.0; y[2 * j + 1] = 0.0; }
            const int jb = net.iperm[net.gbus[gidx[kk]]];
            y[2 * jb] = 1.0;
            for (int j = 0; j < nb; ++j) {           // forward, elimination order
                cplx acc = ld(y + 2 * j);
                for (int e = net.Lrowptr[j]; e < net.Lrowptr[j + 1]; ++e)
                    acc = acc - ld(W + L.Yl + 2 * net.Lrowblk[e]) * ld(y + 2 * net.Lrowcol[e]);
                st(y + 2 * j, acc);
            }
            for (int j = 0; j < nb; ++j) st(y + 2 * j, ld(y + 2 * j) * ld(W + L.Ydi + 2 * j));
            for (int j = nb - 1; j >= 0; --j) {       // backward
                cplx acc = ld(y + 2 * j);
                for (int e = net.Lcolptr[j]; e < net.Lcolptr[j + 1]; ++e)
                    acc = acc - ld(W + L.Yl + 2 * e) * ld(y + 2 * net.Lrow[e]);
                st(y + 2 * j, acc);
            }
        }
        __syncthreads();
        // Y_red[k][l] = ym_k delta_kl - ym_k ym_l (Ybb^-1)[b_k][b_l]
        for (int w = tid; w < m * m; w += nthr) {
            const int k = w / m, l = w % m;
            const cplx ymk = cm(0.0, -1.0 / net.xp[gidx[k]]), yml = cm(0.0, -1.0 / net.xp[gidx[l]]);
            const int jl = net.iperm[net.gbus[gidx[l]]];
            cplx z = ld(W + L.rhs + (size_t)2 * nb * k + 2 * jl);
            cplx v = cm(0.0, 0.0) - ymk * yml * z;
            if (k == l) v = v + ymk;
            st(W + L.Z + 2 * (size_t)(k * m + l), v);
        }
        // ---- 3. equilibrium per machine ----
        for (int kk = tid; kk < m; kk += nthr) {
            const int k = gidx[kk], i = net.gbus[k];
            double sa, ca;
            sincos(xs[i], &sa, &ca);
            const cplx V = xs[nb + i] * cm(ca, sa);
            const cplx S = cm(xs[2 * nb + k], xs[2 * nb + ng + k]);
            const cplx I = conj(cdiv(S, V));
            const cplx EQ = V + mulj(net.xq[k] * I);
            const double delta = atan2(EQ.im, EQ.re);
            double sd, cd;
            sincos(delta, &sd, &cd);
            const cplx ejd = cm(cd, sd);
            const cplx rot = mulj(conj(ejd));            // j e^{-j delta}
            const cplx Idq = I * rot, Vdq = V * rot;   // OPF current, used for the equilibrium only
            const double xp = net.xp[k];
            const double eq = Vdq.im + xp * Idq.re;
            const double ed = Vdq.re - xp * Idq.im;
            const cplx E = cm(eq, -ed) * ejd;
            double* g = W + L.gen + kGen * kk;
            st(g + G_E, E);
            st(g + G_ED, ejd);
            g[G_EQ] = eq;
            g[G_EDD] = ed;
        }
        __syncthreads();
        // network currents at the equilibrium state: I = Y_red E' (the OPF injection up
        // to the OPF residual), and the dq currents and terminal voltage from them
        for (int kk = tid; kk < m; kk += nthr) {
            double* g = W + L.gen + kGen * kk;
            cplx I = cm(0.0, 0.0);
            for (int ll = 0; ll < m; ++ll)
                I = I + ld(W + L.Z + 2 * (size_t)(kk * m + ll)) * ld(W + L.gen + kGen * ll + G_E);
            const cplx rot = mulj(conj(ld(g + G_ED)));
            const cplx Idq = I * rot;
            const cplx Vt = ld(g + G_E) - mulj(net.xp[gidx[kk]] * I);
            st(g + G_I, I);
            st(g + G_VT, Vt);
            g[G_VTM] = sqrt(abs2(Vt));
            g[G_ID] = Idq.re;
            g[G_IQ] = Idq.im;
        }
        __syncthreads();
        // ---- state matrix: one thread per 5x5 block (k, l) ----
        // (the front kernel keeps it per scenario for the FP64 refinement)
        double* A = (kMode == DYN_FRONT && a64) ? a64 + (size_t)s * a64stride : W + L.A;
        for (int w = tid; w < m * m; w += nthr) {
            const int kk = w / m, ll = w % m;
            const int k = gidx[kk];
            const double* gk = W + L.gen + kGen * kk;
            const double* gl = W + L.gen + kGen * ll;
            const cplx Y = ld(W + L.Z + 2 * (size_t)(kk * m + ll));
            const cplx El = ld(gl + G_E), ejl = ld(gl + G_ED);
            const cplx dE[3] = {mulj(El), ejl, cm(0.0, -1.0) * ejl};   // d E'_l / d(delta, e'q, e'd)
            const cplx rotk = mulj(conj(ld(gk + G_ED)));
            const cplx Ik = ld(gk + G_I), Vt = ld(gk + G_VT);
            const double idk = gk[G_ID], iqk = gk[G_IQ], eqk = gk[G_EQ], edk = gk[G_EDD], Vtm = gk[G_VTM];
            const double xp = net.xp[k];
            double blk[5][5];
            for (int r = 0; r < 5; ++r)
                for (int c = 0; c < 5; ++c) blk[r][c] = 0.0;
            const int colmap[3] = {0, 2, 3};
            for (int th = 0; th < 3; ++th) {
                const cplx dI = Y * dE[th];
                cplx didq = rotk * dI;
                if (kk == ll && th == 0) didq = didq + cm(0.0, -1.0) * cplx{idk, iqk};
                double dPe = edk * didq.re + eqk * didq.im;
                if (kk == ll && th == 1) dPe += iqk;
                if (kk == ll && th == 2) dPe += idk;
                cplx dVt = cm(0.0, -xp) * dI;
                if (kk == ll) dVt = dVt + dE[th];
                const double dVm = (Vt.re * dVt.re + Vt.im * dVt.im) / Vtm;
                const int c = colmap[th];
                blk[1][c] = -dPe / net.H2[k];
                blk[2][c] = -(net.xd[k] - xp) * didq.re / net.Td0[k];
                blk[3][c] = (net.xq[k] - xp) * didq.im / net.Tq0[k];
                blk[4][c] = -net.KA[k] * dVm / net.TA[k];
            }
            // angle rows: d delta'_k/dt = ws (omega_k - omega_0) for k != 0 (row of delta_0 dropped)
            if (kk == ll && kk != 0) blk[0][1] = net.ws;
            if (ll == 0 && kk != 0) blk[0][1] = -net.ws;
            if (kk == ll) {
                blk[1][1] = -net.Dm[k] / net.H2[k];
                blk[2][2] += -1.0 / net.Td0[k];
                blk[2][4] = 1.0 / net.Td0[k];
                blk[3][3] += -1.0 / net.Tq0[k];
                blk[4][4] = -1.0 / net.TA[k];
            }
            // reduced indexing: full index 5k + s -> 5k + s - 1, the angle of machine 0 dropped
            for (int r = 0; r < 5; ++r) {
                if (kk == 0 && r == 0) continue;
                for (int c = 0; c < 5; ++c) {
                    if (ll == 0 && c == 0) continue;
                    A[(size_t)(5 * kk + r - 1) * n + 5 * ll + c - 1] = blk[r][c];
                }
            }
        }
        __syncthreads();
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        if (sh.fail) {                                // Y_bb singular: no model at this point
            if (tid == 0) {
                if (isl) {                            // the main island's class; the scenario's stays ISLANDED
                    if (a.out.main_klass) a.out.main_klass[s] = CS_EIG_FAIL;
                } else {
                    a.out.klass[s] = CS_EIG_FAIL;
                    a.out.severe[s] = 1;
                }
                a.out.max_re[s] = nan;
                a.out.min_zeta[s] = nan;
                if (kMode == DYN_FRONT || kMode == DYN_FRONT_LARGE) o.status[s] = 7;
            }
            __syncthreads();
            continue;
        }
        // ---- 4. eigenvalues: FP64, or an FP32 screen with an FP64 re-run in the guard band ----
        double* wr = W + L.wr;
        double* wi = W + L.wi;
        double maxre = 0.0, minz = 0.0;
        if (kMode == DYN_FRONT) {                     // balanced FP32 matrix for the cluster kernel
            float* dst = hbuf + (size_t)s * hstride;
            float* A32 = dst + kHqHead;
            for (int w = tid; w < n * n; w += nthr) A32[w] = (float)A[w];
            if (tid == 0) dst[0] = __int_as_float(n);
            __syncthreads();
            balance<float>(A32, n, reinterpret_cast<float*>(cs_d), reinterpret_cast<float*>(rs_d),
                           dst + ab_d_off(5 * ng - 1), sh);
            __syncthreads();
            continue;
        }
        if (kMode == DYN_FRONT_LARGE) {               // balanced FP32 matrix, padded, for the tensor-core reduction
            float* A32 = reinterpret_cast<float*>(W + L.A32);
            for (int w = tid; w < n * n; w += nthr) A32[w] = (float)A[w];
            __syncthreads();
            balance<float>(A32, n, reinterpret_cast<float*>(cs_d), reinterpret_cast<float*>(rs_d),
                           reinterpret_cast<float*>(v_d), sh);
            __syncthreads();
            float* slot = hbuf + (size_t)s * hstride;
            const int nmax = 5 * ng - 1;
            float* M = slot + kHqHead;
            for (int w = tid; w < nmax * nmax; w += nthr) {
                const int i = w / nmax, j = w % nmax;
                M[w] = (i < n && j < n) ? A32[i * n + j] : (i == j ? -1.0f : 0.0f);
            }
            if (tid == 0) slot[0] = __int_as_float(n);
            __syncthreads();
            continue;
        }
        if (kMode == DYN_MIXED_INLINE) {
            float* A32 = reinterpret_cast<float*>(W + L.A32);
            for (int w = tid; w < n * n; w += nthr) A32[w] = (float)A[w];
            __syncthreads();
            eigen_screen<float>(A32, n, reinterpret_cast<float*>(cs_d), reinterpret_cast<float*>(rs_d),
                                reinterpret_cast<float*>(v_d), reinterpret_cast<float*>(W + L.hp), wr, wi, sh);
            eig_stats(sh, n, wr, wi, maxre, minz);
            const bool near = sh.fail || !(fabs(maxre) > kGuardRe) || !(fabs(minz - damping_min) > kGuardZeta);
            if (near) {                               // decision too close to call in FP32
                if (tid == 0) {
                    sh.fail = 0;
                    atomicAdd(a.reruns, 1);
                }
                __syncthreads();
                eigen_screen<double>(A, n, cs_d, rs_d, v_d, W + L.hp, wr, wi, sh);
                eig_stats(sh, n, wr, wi, maxre, minz);
            }
        } else {
            eigen_screen<double>(A, n, cs_d, rs_d, v_d, W + L.hp, wr, wi, sh);
            eig_stats(sh, n, wr, wi, maxre, minz);
        }
        // ---- 5. class ----
        {
            if (tid == 0) {
                uint8_t k;
                if (sh.fail) k = CS_EIG_FAIL;
                else if (maxre >= 0.0) k = CS_SS_UNSTABLE;
                else if (minz < damping_min) k = CS_SS_POORLY_DAMPED;
                else k = CS_SECURE;
                if (isl) {
                    if (a.out.main_klass) a.out.main_klass[s] = k;
                } else {
                    a.out.klass[s] = k;
                    a.out.severe[s] = (k != CS_SECURE);
                }
                a.out.max_re[s] = sh.fail ? nan : maxre;
                a.out.min_zeta[s] = sh.fail ? nan : minz;
            }
            __syncthreads();
        }
    }
}

__global__ void record_kernel(int nbr, int nE, EvalArgs a) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < a.n; s += gridDim.x * blockDim.x) {
        const int ei = a.ei[s], ej = a.ej[s];
        if (ei < 0 || ei >= nE || ej >= nE || ej < -1) continue;
        if (a.ek && a.ek[s] >= 0 && a.ek[s] != ei && a.ek[s] != ej) continue;   // N-3: not in the N-2 tables
        const uint8_t S = a.out.severe[s] ? 1 : 0;
        if (ej < 0 || ej == ei) {
            a.sev_n1[ei] = S;
        } else {
            const long long i = min(ei, ej), j = max(ei, ej);
            const long long k = i * nE - (i * (i + 1)) / 2 + (j - i - 1);
            a.sev_pairs[k] = S;
        }
    }
}



// ---------------------------------------------------------------------------
// FP32 screen, middle part: Householder reduction to Hessenberg form of the
// balanced matrix, held on chip by a cluster of two CTAs (each keeps half of
// the rows in its shared memory; the 269 x 269 matrix of the 118-bus network
// is 289 KB, more than one CTA may hold).  Per column, each CTA writes its
// rows' part of the reflector and of the squared norm into both CTAs' shared
// memory (distributed shared memory), then the partial sums v^T A of the left
// update; two cluster barriers per column.  Exchange buffers alternate with the
// column parity, so a CTA that runs ahead never overwrites what its peer still
// reads.  The packed Hessenberg matrix goes to hbuf for hqr_smem_kernel.
//
// The reflector and w = beta v^T A are indexed by absolute rows and columns, zero up to the column
// being reduced, so a row's two updates need no masks: a lane takes two adjacent columns of each
// group of 64, and groups left of the column are skipped.  (With a lane per column counted from
// the reduced one, and twelve masked columns per lane whatever was left, most of the
// instructions were masks.  118 buses, one scenario 1.69 -> 1.24 ms, 417 of them 10.1 -> 7.4 ms.)
constexpr int kHsThreads = 512;
constexpr int kHsWarps = kHsThreads / 32;
constexpr int kHsCols = 12;         // columns per lane in the row pass: orders up to 32 * 12
constexpr int kHsGroups = kHsCols / 2;

// row stride in shared memory: even (pairs of columns), not a multiple of 32 banks
__host__ __device__ inline int hs_ld(int n) {
    const int ld = (n + 1) & ~1;
    return (ld & 31) == 0 ? ld + 2 : ld;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kHsThreads, 1)
hess_cluster_kernel(EvalArgs a, OpfOut o, float* __restrict__ abuf, size_t astride, float* __restrict__ hbuf,
                    size_t hstride, int nmax, int* counter) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) float csm[];
    const int hmax = (nmax + 1) / 2, ldm = hs_ld(nmax);
    float* As = csm;                                  // own rows, row stride ld
    float* vb = As + (size_t)hmax * ldm;              // [2 parity][ldm] reflector, by absolute row
    float* wb = vb + 2 * ldm;                         // [2 parity][2 rank][ldm] partial v^T A, by absolute column
    float* ws = wb + 4 * ldm;                         // [kHsSlices][ldm] this CTA's partial sums by row slices
    float* np = ws + kHsSlices * ldm;                 // [2 parity][2 rank] partial squared norms
    __shared__ float red[kHsWarps];
    __shared__ int scen;
    float* peer_vb = cl.map_shared_rank(vb, rank ^ 1);
    float* peer_wb = cl.map_shared_rank(wb, rank ^ 1);
    float* peer_np = cl.map_shared_rank(np, rank ^ 1);
    int* peer_scen = cl.map_shared_rank(&scen, rank ^ 1);

    for (;;) {
        if (rank == 0 && tid == 0) {
            const int s0 = atomicAdd(counter, 1);
            scen = s0;
            *peer_scen = s0;
        }
        cl.sync();
        const int s = scen;
        cl.sync();                                    // both have read scen
        if (s >= a.n) break;
        if (o.status[s] != 1) continue;
        float* src = abuf + (size_t)s * astride;
        const int n = __float_as_int(src[0]), ld = hs_ld(n);
        const float* Ag = src + kHqHead;
        // Householder vectors and factors for the refinement kernel: rank 0 writes them
        // over the slot's matrix, after both CTAs have loaded their rows (the first
        // cluster barrier of column 0)
        float* refl = src + kHqHead;
        float* betas = src + ab_beta_off(nmax);
        const int h = (n + 1) / 2, r0 = rank * h, r1 = min(n, r0 + h), nr = max(0, r1 - r0);
        for (int i = warp; i < nr; i += kHsWarps)
            for (int j = lane; j < ld; j += 32) As[(size_t)i * ld + j] = (j < n) ? Ag[(size_t)(r0 + i) * n + j] : 0.0f;
        for (int w = tid; w < 2 * ldm; w += kHsThreads) vb[w] = 0.0f;
        // the peer writes its part of the reflector into vb: not before it is cleared
        cl.sync();
        for (int k = 0; k + 2 < n; ++k) {
            const int par = k & 1;
            float* v = vb + par * ldm;
            float* pv = peer_vb + par * ldm;
            const int i0 = max(r0, k + 1);
            float t = 0.0f;
            for (int i = i0 + tid; i < r1; i += kHsThreads) {
                const float q = As[(size_t)(i - r0) * ld + k];
                v[i] = q;
                pv[i] = q;
                if (i >= k + 2) t += q * q;
            }
            if (tid < 2 && k - tid >= 0) v[k - tid] = 0.0f;   // left from two columns ago
            for (int off = 16; off; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
            if (lane == 0) red[warp] = t;
            __syncthreads();
            if (tid == 0) {
                float tt = 0.0f;
                for (int q = 0; q < kHsWarps; ++q) tt += red[q];
                np[par * 2 + rank] = tt;
                peer_np[par * 2 + rank] = tt;
            }
            cl.sync();                                // reflector and norm partials in place
            const float tail = np[par * 2] + np[par * 2 + 1];
            if (tail == 0.0f) {                       // column already reduced (same in both CTAs)
                if (rank == 0 && tid == 0) betas[k] = 0.0f;
                continue;
            }
            const float x0 = v[k + 1];
            const float nrm = sqrtf(x0 * x0 + tail);
            const float alpha = (x0 >= 0.0f) ? -nrm : nrm;
            const float v0 = x0 - alpha;
            const float beta = 2.0f / (v0 * v0 + tail);
            // this CTA's copy of the reflector takes v0 in place of x0 (the peer writes only the
            // other parity's copy during this column)
            __syncthreads();
            if (tid == 0) v[k + 1] = v0;
            __syncthreads();
            if (rank == 0) {
                float* rk = refl + refl_off(n, k);
                for (int i = tid; i < n - k - 1; i += kHsThreads) rk[i] = v[k + 1 + i];
                if (tid == 0) betas[k] = beta;
            }
            // partial v^T A over own rows: pairs of columns, the rows in kHsSlices slices
            const int p0 = (k + 1) >> 1, np2 = (ld >> 1) - p0;
            for (int w = tid; w < kHsSlices * np2; w += kHsThreads) {
                const int sl = w / np2, j = 2 * (p0 + w - sl * np2);
                const int m0 = i0 + (r1 - i0) * sl / kHsSlices, m1 = i0 + (r1 - i0) * (sl + 1) / kHsSlices;
                float ax = 0.0f, ay = 0.0f, bx = 0.0f, by = 0.0f;
                const float* col = As + (size_t)(m0 - r0) * ld + j;
                int i = m0;
                for (; i + 2 <= m1; i += 2, col += 2 * ld) {
                    const float2 q = *reinterpret_cast<const float2*>(col), u = *reinterpret_cast<const float2*>(col + ld);
                    const float v1 = v[i], v2 = v[i + 1];
                    ax += v1 * q.x; ay += v1 * q.y;
                    bx += v2 * u.x; by += v2 * u.y;
                }
                if (i < m1) {
                    const float2 q = *reinterpret_cast<const float2*>(col);
                    ax += v[i] * q.x; ay += v[i] * q.y;
                }
                *reinterpret_cast<float2*>(ws + sl * ldm + j) = make_float2(ax + bx, ay + by);
            }
            __syncthreads();
            float* w_own = wb + (par * 2 + rank) * ldm;
            float* w_peer = peer_wb + (par * 2 + rank) * ldm;
            for (int j = 2 * p0 + tid; j < ld; j += kHsThreads) {
                float q = 0.0f;
#pragma unroll
                for (int sl = 0; sl < kHsSlices; ++sl) q += ws[sl * ldm + j];
                if (j == k) q = 0.0f;                 // the reduced column is written below
                w_own[j] = q;
                w_peer[j] = q;
            }
            cl.sync();                                // partial sums exchanged
            // One pass per own row, a warp per two rows: the left update (rows k+1..), the right
            // update, then column k; a lane keeps w and v of its columns in registers.
            const float* w0 = wb + (par * 2) * ldm;
            const int g0 = (k + 1) >> 6, g1 = (ld + 63) >> 6;
            float2 wv[kHsGroups], vv[kHsGroups];
#pragma unroll
            for (int g = 0; g < kHsGroups; ++g) {
                const int j = 64 * g + 2 * lane;
                wv[g] = vv[g] = make_float2(0.0f, 0.0f);
                if (g >= g0 && g < g1 && j >= 2 * p0 && j < ld) {
                    const float2 q = *reinterpret_cast<const float2*>(w0 + j), u = *reinterpret_cast<const float2*>(w0 + ldm + j);
                    wv[g] = make_float2(beta * (q.x + u.x), beta * (q.y + u.y));
                    vv[g] = *reinterpret_cast<const float2*>(v + j);
                }
            }
            for (int i = 2 * warp; i < nr; i += 2 * kHsWarps) {
                const bool two = i + 1 < nr;
                float* row[2] = {As + (size_t)i * ld + 2 * lane, As + (size_t)(two ? i + 1 : i) * ld + 2 * lane};
                const float vi[2] = {v[r0 + i], two ? v[r0 + i + 1] : 0.0f};
                float2 x[2][kHsGroups];
                float acc[2] = {0.0f, 0.0f};
#pragma unroll
                for (int g = 0; g < kHsGroups; ++g) {
                    if (g < g0 || g >= g1) continue;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        float2 y = make_float2(0.0f, 0.0f);
                        if (64 * g + 2 * lane < ld) y = *reinterpret_cast<const float2*>(row[q] + 64 * g);
                        y.x -= vi[q] * wv[g].x;
                        y.y -= vi[q] * wv[g].y;
                        acc[q] += y.x * vv[g].x + y.y * vv[g].y;
                        x[q][g] = y;
                    }
                }
                for (int off = 16; off; off >>= 1) {
                    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
                    acc[1] += __shfl_xor_sync(0xffffffffu, acc[1], off);
                }
                acc[0] *= beta;
                acc[1] *= beta;
#pragma unroll
                for (int g = 0; g < kHsGroups; ++g) {
                    if (g < g0 || g >= g1) continue;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (64 * g + 2 * lane < ld && (q == 0 || two))
                            *reinterpret_cast<float2*>(row[q] + 64 * g) =
                                make_float2(x[q][g].x - acc[q] * vv[g].x, x[q][g].y - acc[q] * vv[g].y);
                    }
                }
                __syncwarp();
                if (lane < (two ? 2 : 1) && r0 + i + lane > k)
                    As[(size_t)(i + lane) * ld + k] = (r0 + i + lane == k + 1) ? alpha : 0.0f;
            }
            __syncthreads();
        }
        float* dst = hbuf + (size_t)s * hstride;      // packed rows for the shared-memory QR
        if (rank == 0 && tid == 0) dst[0] = __int_as_float(n);
        for (int i = r0 + warp; i < r1; i += kHsWarps) {
            const int j0 = hq_start(i);
            float* drow = dst + kHqHead + hq_off(n, i) - j0;
            for (int j = j0 + lane; j < n; j += 32) drow[j] = As[(size_t)(i - r0) * ld + j];
        }
        cl.sync();                                    // the peer has read this CTA's exchange buffers
    }
}

// ---------------------------------------------------------------------------
// FP32 screen, last part: Francis double-shift QR of the packed Hessenberg
// matrix held in shared memory (one scenario per CTA, one CTA per SM), the
// sweeps in windows (qr_sweep).  Every thread carries the same loop state
// (lo, hi, sweep count), computed redundantly from shared memory.
// Exceptional shifts come every tenth sweep without a deflation, and a stalled
// window also deflates at the normwise FP32 level (kStallIts).  A scenario whose
// QR does not converge is marked for the FP64 re-run; the others get their
// refinement candidates and go on to eig_refine_kernel, which classifies them.
#ifndef CS_QR_THREADS
#define CS_QR_THREADS 256
#endif
constexpr int kQrThreads = CS_QR_THREADS;
// FP32 QR without a deflation for this many sweeps (the double-shift iteration can
// stall at FP32 rounding level): from then on a subdiagonal entry below eps_32 times
// the largest entry of the matrix counts as negligible too.  The screen's eigenvalues
// only need to be within kEigDelta of the exact ones (the decisive ones are refined in
// FP64), which that normwise perturbation respects.
constexpr int kStallIts = 40;

__device__ __forceinline__ void eig2f(float p, float q, float r, float s, float* re, float* im) {
    const float hm = 0.5f * (p - s);
    const float disc = hm * hm + q * r;
    const float mean = 0.5f * (p + s);
    if (disc >= 0.0f) {
        const float root = sqrtf(disc);
        const float big = mean + (hm >= 0.0f ? root : -root);
        const float det = p * s - q * r;
        const float other = (big != 0.0f) ? det / big : mean - (hm >= 0.0f ? root : -root);
        re[0] = big; im[0] = 0.0f;
        re[1] = other; im[1] = 0.0f;
    } else {
        const float root = sqrtf(-disc);
        re[0] = mean; im[0] = root;
        re[1] = mean; im[1] = -root;
    }
}

__global__ void __launch_bounds__(kQrThreads, 1)
hqr_smem_kernel(EvalArgs a, OpfOut o, const float* __restrict__ hbuf, size_t hstride, int nmax,
                double damping_min, float* __restrict__ cand, int* counter) {
    extern __shared__ float qsm[];
    __shared__ float red[2][kQrThreads / 32];
    __shared__ QrSpace<float> sp[2][2];
    __shared__ int scen;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float* H = qsm;                                           // hq_off(nmax, nmax) floats
    int* rb = reinterpret_cast<int*>(qsm + ((hq_off(nmax, nmax) + 3) & ~3));   // row i at H[rb[i] + j]
    float* wr = reinterpret_cast<float*>(rb + nmax);
    float* wi = wr + nmax;
    const PackedMat<float> A{H, rb};
    const float eps = 1.1920928955078125e-07f;

    for (;;) {
        if (tid == 0) scen = atomicAdd(counter, 1);
        __syncthreads();
        const int s = scen;
        if (s >= a.n) break;
        if (o.status[s] != 1) {
            __syncthreads();
            continue;
        }
        const float* src = hbuf + (size_t)s * hstride;
        const int n = __float_as_int(src[0]);
        const int hs = hq_off(n, n);
        {
            const float4* s4 = reinterpret_cast<const float4*>(src + kHqHead);
            float4* d4 = reinterpret_cast<float4*>(H);
            for (int w = tid; w < (hs >> 2); w += kQrThreads) d4[w] = s4[w];
            for (int w = (hs & ~3) + tid; w < hs; w += kQrThreads) H[w] = src[kHqHead + w];
        }
        for (int i = tid; i < n; i += kQrThreads) rb[i] = hq_off(n, i) - hq_start(i);
        __syncthreads();
        float hmax;
        {
            float hm = 0.0f;
            for (int w = tid; w < hs; w += kQrThreads) hm = fmaxf(hm, fabsf(H[w]));
            for (int off = 16; off; off >>= 1) hm = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, off));
            if (lane == 0) red[0][warp] = hm;
            __syncthreads();
            hmax = red[0][0];
            for (int w = 1; w < kQrThreads / 32; ++w) hmax = fmaxf(hmax, red[0][w]);
        }
        int hi = n - 1, its = 0;
        bool fail = false;
        while (hi >= 0) {
            // top of the unreduced block ending at hi (every warp scans; all agree)
            int lo = 0;
            for (int base = hi; base >= 1; base -= 32) {
                const int l = base - lane;
                bool neg = false;
                if (l >= 1) {
                    float sd = fabsf(H[rb[l - 1] + l - 1]) + fabsf(H[rb[l] + l]);
                    if (sd == 0.0f) sd = hmax;
                    const float h = fabsf(H[rb[l] + l - 1]);
                    // after kStallIts sweeps without a deflation, a subdiagonal entry at FP32
                    // rounding level of the whole matrix also counts as negligible
                    neg = h <= kDeflTol * sd || (its >= kStallIts && h <= eps * hmax);
                }
                const unsigned m = __ballot_sync(0xffffffffu, neg);
                if (m) {
                    lo = base - (__ffs(m) - 1);
                    break;
                }
            }
            if (lo == hi) {
                if (tid == 0) {
                    wr[hi] = H[rb[hi] + hi];
                    wi[hi] = 0.0f;
                }
                hi -= 1;
                its = 0;
                continue;
            }
            if (lo == hi - 1) {
                if (tid == 0) {
                    float re[2], im[2];
                    eig2f(H[rb[hi - 1] + hi - 1], H[rb[hi - 1] + hi], H[rb[hi] + hi - 1], H[rb[hi] + hi], re, im);
                    wr[hi - 1] = re[0]; wi[hi - 1] = im[0];
                    wr[hi] = re[1]; wi[hi] = im[1];
                }
                hi -= 2;
                its = 0;
                continue;
            }
            if (its >= 30 * n) {
                fail = true;
                break;
            }
            ++its;
            __syncthreads();              // every warp has read the block before the sweep writes
            const bool exceptional = its % 10 == 0;               // every tenth time without a deflation
            qr_sweep<true, float>(A, lo, hi, exceptional, !exceptional && hi - lo >= kQrPair, sp, kQrThreads);
        }
        __syncthreads();                                   // wr, wi written by thread 0
        // statistics over all eigenvalues: max Re, min damping ratio
        float mr = -INFINITY, mz = INFINITY;
        if (!fail) {
            for (int i = tid; i < n; i += kQrThreads) {
                mr = fmaxf(mr, wr[i]);
                const float mg = sqrtf(wr[i] * wr[i] + wi[i] * wi[i]);
                mz = fminf(mz, mg > 0.0f ? -wr[i] / mg : 1.0f);
            }
        }
        for (int off = 16; off; off >>= 1) {
            mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, off));
            mz = fminf(mz, __shfl_xor_sync(0xffffffffu, mz, off));
        }
        if (lane == 0) {
            red[0][warp] = mr;
            red[1][warp] = mz;
        }
        __syncthreads();
        if (warp == 0) {
            float maxre = red[0][0];
            for (int w = 1; w < kQrThreads / 32; ++w) maxre = fmaxf(maxre, red[0][w]);
            // The class is decided after the FP64 refinement (eig_refine_kernel), from
            // values within ~1e-9 of the FP64 screen's, so no FP32 guard band applies here;
            // a QR that did not converge goes to the FP64 screen.
            // Candidates of the FP64 refinement, in index order: every eigenvalue
            // (im >= 0 of a pair) whose exact value may carry the largest real part
            // or the smallest damping ratio, given |FP32 - exact| <= kEigDelta.
            // Damping ratio of lambda with |delta lambda| <= d moves by at most 2 d / |lambda|.
            auto modulus = [&](int i) { return sqrtf(wr[i] * wr[i] + wi[i] * wi[i]); };
            float zu = INFINITY;
            if (!fail)
                for (int i = lane; i < n; i += 32) {
                    const float mg = modulus(i);
                    if (!(wi[i] < 0.0f) && mg > 0.0f) zu = fminf(zu, -wr[i] / mg + 2.0f * kEigDelta / mg);
                }
            for (int off = 16; off; off >>= 1) zu = fminf(zu, __shfl_xor_sync(0xffffffffu, zu, off));
            float* cs = cand + (size_t)s * kCandStride;
            int cnt = 0, flags = 0;
            for (int i0 = 0; i0 < n && !fail; i0 += 32) {
                const int i = i0 + lane;
                bool cre = false, cz = false;
                if (i < n && !(wi[i] < 0.0f)) {
                    const float mg = modulus(i);
                    const float z = mg > 0.0f ? -wr[i] / mg : 1.0f;
                    cre = wr[i] >= maxre - 2.0f * kEigDelta;
                    cz = !(mg > 0.0f) || z - 2.0f * kEigDelta / mg <= zu;
                }
                for (unsigned m = __ballot_sync(0xffffffffu, cre || cz); m; m &= m - 1, ++cnt) {
                    const int src = __ffs(m) - 1;
                    const int f = __shfl_sync(0xffffffffu, (cre ? 1 : 0) | (cz ? 2 : 0), src);
                    if (cnt >= kRefK) continue;
                    flags |= f << (2 * cnt);
                    if (lane == src) {
                        cs[4 + 2 * cnt] = wr[i];
                        cs[5 + 2 * cnt] = wi[i];
                    }
                }
            }
            if (lane == 0) {
                if (fail || cnt > kRefK) {                 // not converged, or too many to refine: FP64 screen
                    o.status[s] = 6;
                    atomicAdd(a.reruns, 1);
                } else {
                    cs[0] = __int_as_float(cnt);
                    cs[1] = __int_as_float(flags);
                    o.status[s] = 8;
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// FP64 refinement of the FP32 screen's decisive eigenvalues.  For each candidate
// (an FP32 eigenvalue sigma that may carry max Re or min zeta), one warp computes
// the right and another the left eigenvector of the packed FP32 Hessenberg matrix
// H by two passes of inverse iteration with shift sigma, and takes each back to
// the balanced matrix through the Householder vectors of the cluster kernel.  The
// eigenvalue is then the two-sided Rayleigh quotient w^H A v / w^H v with the
// scenario's FP64 state matrix A (v, w scaled by the balancing factors), whose
// error is second order in the vectors' FP32 error.  The statistics over the
// refined candidates decide the class.  A candidate whose quotient is
// ill-conditioned or lands away from sigma sends the scenario to the FP64 screen.
//
// Inverse iteration on an upper Hessenberg G - sigma I, one warp: Gaussian
// elimination with partial pivoting between each carried row and the next row of
// G (the only one with an entry below the diagonal), U^{-X} b (X = H or T) formed
// row by row as U's rows appear, so U is never stored; the row operations E_k
// (swap flag and multiplier) are kept and applied as E_0^X ... E_{n-2}^X at the
// end.  The left vector solves (H - sigma I)^H z = b with G = H; the right one
// solves (H - sigma I) x = b as (G - sigma I)^T (J x) = J b with G = J H^T J
// (J reverses the order), which is upper Hessenberg again.
//
// What bounds it is latency: two passes of 269 dependent steps and 267 reflectors a vector, one warp each.  So a step
// takes one complex reciprocal (two divisions with scaling before), its columns are loaded three at a time
// ahead of the stores, the row operations carry their one dependent entry in registers, and the next
// reflector is loaded while one is applied.  118 buses, 10,000 pairs mixed 817 -> 795 ms.
constexpr int kRfThreads = 256;
constexpr int kRfWarps = kRfThreads / 32;
constexpr int kRfBatch = 3;           // columns per lane and trip of the inverse iteration's inner loop
static_assert(2 * kRefK <= kRfWarps, "one warp per eigenvector");

__device__ __forceinline__ float2 cmul2(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 cconj2(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 crcp2(float2 b) {
    const float sc = 1.0f / fmaxf(fabsf(b.x), fabsf(b.y));
    const float bx = b.x * sc, by = b.y * sc;
    const float d = sc / (bx * bx + by * by);
    return make_float2(bx * d, -by * d);
}

template <bool kRight>
__device__ __forceinline__ float hess_g(const float* Hs, const int* rb, int n, int i, int j) {
    return kRight ? Hs[rb[n - 1 - j] + n - 1 - i] : Hs[rb[i] + j];
}

// y <- (G - sig I)^{-X} y (X = H for the left vector, T for the right one), one warp.
template <bool kRight>
__device__ void hess_inverse_pass(const float* Hs, const int* rb, int n, float2 sig, float tiny, float2* y, float2* c,
                                  float2* mul, unsigned* swp, int lane) {
    const bool cj = !kRight;
    for (int j = lane; j < n; j += 32)
        c[j] = make_float2(hess_g<kRight>(Hs, rb, n, 0, j) - (j == 0 ? sig.x : 0.0f), j == 0 ? -sig.y : 0.0f);
    for (int w = lane; w < (n + 31) / 32; w += 32) swp[w] = 0u;
    __syncwarp();
    for (int k = 0; k < n; ++k) {
        const bool last = (k == n - 1);
        const float2 ck = c[k];
        const float2 bk = y[k];
        const float rk = last ? 0.0f : hess_g<kRight>(Hs, rb, n, k + 1, k);
        const bool sw = !last && fabsf(rk) > fabsf(ck.x) + fabsf(ck.y);
        float2 pk = sw ? make_float2(rk, 0.0f) : ck;
        if (pk.x == 0.0f && pk.y == 0.0f) pk.x = tiny;             // exactly singular: perturb the pivot
        const float2 ok = sw ? ck : make_float2(rk, 0.0f);
        const float2 ik = crcp2(pk);                                // one reciprocal for the multiplier and y_k
        const float2 mk = last ? make_float2(0.0f, 0.0f) : cmul2(ok, ik);
        const float2 yk = cmul2(bk, cj ? cconj2(ik) : ik);
        __syncwarp();                                               // every lane has read c[k], y[k]
        for (int j0 = k + 1 + lane; j0 < n; j0 += 32 * kRfBatch) {
            float g[kRfBatch];                                      // a batch's loads before its stores
            float2 cb[kRfBatch], yb[kRfBatch];
#pragma unroll
            for (int q = 0; q < kRfBatch; ++q) {
                const int j = min(j0 + 32 * q, n - 1);
                g[q] = hess_g<kRight>(Hs, rb, n, k + 1, j);
                cb[q] = c[j];
                yb[q] = y[j];
            }
#pragma unroll
            for (int q = 0; q < kRfBatch; ++q) {
                const int j = j0 + 32 * q;
                if (j >= n) break;
                float2 rj = make_float2(g[q], 0.0f);
                if (j == k + 1) {
                    rj.x -= sig.x;
                    rj.y -= sig.y;
                }
                const float2 cv = cb[q];
                const float2 pj = sw ? rj : cv, oj = sw ? cv : rj;
                const float2 t = cmul2(cj ? cconj2(pj) : pj, yk);
                y[j] = make_float2(yb[q].x - t.x, yb[q].y - t.y);
                const float2 u = cmul2(mk, pj);
                c[j] = make_float2(oj.x - u.x, oj.y - u.y);
            }
        }
        if (lane == 0) {
            y[k] = yk;
            mul[k] = mk;
            if (sw) swp[k >> 5] |= 1u << (k & 31);
        }
        __syncwarp();
    }
    if (lane == 0) {
        float2 up = y[n - 1];                                       // y[k + 1] so far
        float2 m = mul[max(n - 2, 0)], v = y[max(n - 2, 0)];        // of step k, loaded a step ahead
        for (int k = n - 2; k >= 0; --k) {
            const float2 mn = mul[max(k - 1, 0)], vn = y[max(k - 1, 0)];
            const float2 t = cmul2(cj ? cconj2(m) : m, up);
            const float2 d = make_float2(v.x - t.x, v.y - t.y);
            const bool sw = (swp[k >> 5] >> (k & 31)) & 1u;
            y[k + 1] = sw ? d : up;
            up = sw ? up : d;
            m = mn;
            v = vn;
        }
        y[0] = up;
    }
    __syncwarp();
}

// scale y to a largest component of modulus 1; false if it has none (zero or not finite)
__device__ bool warp_normalise(float2* y, int n, int lane) {
    float mx = 0.0f;
    for (int j = lane; j < n; j += 32) mx = fmaxf(mx, fmaxf(fabsf(y[j].x), fabsf(y[j].y)));
    for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (!(mx > 0.0f) || !isfinite(mx)) return false;
    const float inv = 1.0f / mx;
    for (int j = lane; j < n; j += 32) y[j] = make_float2(y[j].x * inv, y[j].y * inv);
    __syncwarp();
    return true;
}

struct RfShared {
    int scen, cnt, flags;
    float tiny;
    int bad[2 * kRefK];
    float hred[kRfWarps];
    double acc[kRfWarps][kRefK][6];   // per warp: num (re, im), den (re, im), |v|^2, |w|^2
};

__global__ void __launch_bounds__(kRfThreads, 1)
eig_refine_kernel(EvalArgs a, OpfOut o, const float* __restrict__ hbuf, size_t hstride, const float* __restrict__ abuf,
                  size_t astride, const double* __restrict__ a64, size_t a64stride, const float* __restrict__ cand,
                  int nmax, double damping_min, int* counter) {
    extern __shared__ float4 rsm4[];
    float* rsm = reinterpret_cast<float*>(rsm4);
    __shared__ RfShared sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t hsz = ((size_t)hq_off(nmax, nmax) + 3) & ~(size_t)3;
    const size_t vsz = (size_t)4 * kRefK * nmax * 2;                 // FP64 vectors (doubles as float pairs)
    float* Hs = rsm;                                                  // packed H, later the FP64 vectors
    double2* vA = reinterpret_cast<double2*>(rsm);                    // [kRefK][nmax]
    double2* wA = vA + (size_t)kRefK * nmax;                          // [kRefK][nmax]
    int* rb = reinterpret_cast<int*>(rsm + (hsz > vsz ? hsz : vsz));
    float2* wk = reinterpret_cast<float2*>(rb + ((nmax + 3) & ~3));   // per warp: c, mul [nmax] each
    float2* vec = wk + (size_t)kRfWarps * 2 * nmax;                   // [2 kRefK][nmax] vectors
    unsigned* swp = reinterpret_cast<unsigned*>(vec + (size_t)2 * kRefK * nmax);   // per warp: bits
    const int swords = (nmax + 31) / 32;

    for (;;) {
        if (tid == 0) sh.scen = atomicAdd(counter, 1);
        __syncthreads();
        const int s = sh.scen;
        if (s >= a.n) break;
        if (o.status[s] != 8) {
            __syncthreads();
            continue;
        }
        const float* src = hbuf + (size_t)s * hstride;
        const int n = __float_as_int(src[0]);
        const int hs = hq_off(n, n);
        const float* slot = abuf + (size_t)s * astride;
        const float* cs = cand + (size_t)s * kCandStride;
        {
            const float4* s4 = reinterpret_cast<const float4*>(src + kHqHead);
            float4* d4 = reinterpret_cast<float4*>(Hs);
            for (int w = tid; w < (hs >> 2); w += kRfThreads) d4[w] = s4[w];
            for (int w = (hs & ~3) + tid; w < hs; w += kRfThreads) Hs[w] = src[kHqHead + w];
        }
        for (int i = tid; i < n; i += kRfThreads) rb[i] = hq_off(n, i) - hq_start(i);
        if (tid == 0) {
            sh.cnt = __float_as_int(cs[0]);
            sh.flags = __float_as_int(cs[1]);
        }
        if (tid < 2 * kRefK) sh.bad[tid] = 0;
        __syncthreads();
        {
            float hm = 0.0f;
            for (int w = tid; w < hs; w += kRfThreads) hm = fmaxf(hm, fabsf(Hs[w]));
            for (int off = 16; off; off >>= 1) hm = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, off));
            if (lane == 0) sh.hred[warp] = hm;
            __syncthreads();
            if (tid == 0) {
                float m = sh.hred[0];
                for (int w = 1; w < kRfWarps; ++w) m = fmaxf(m, sh.hred[w]);
                sh.tiny = 1.1920928955078125e-07f * (m > 0.0f ? m : 1.0f);
            }
            __syncthreads();
        }
        const int cnt = sh.cnt;
        // ---- eigenvectors of H, one warp each: task 2c = right vector of candidate c, 2c+1 = left ----
        if (warp < 2 * cnt) {
            const int c = warp >> 1;
            const bool right = (warp & 1) == 0;
            const float2 sig = make_float2(cs[4 + 2 * c], cs[5 + 2 * c]);
            float2* y = vec + (size_t)warp * nmax;
            float2* cw = wk + (size_t)warp * 2 * nmax;
            float2* mw = cw + nmax;
            unsigned* sb = swp + warp * swords;
            for (int j = lane; j < n; j += 32) y[j] = make_float2(1.0f, 0.0f);
            __syncwarp();
            bool ok = true;
            for (int pass = 0; pass < 2 && ok; ++pass) {
                if (right) hess_inverse_pass<true>(Hs, rb, n, sig, sh.tiny, y, cw, mw, sb, lane);
                else hess_inverse_pass<false>(Hs, rb, n, sig, sh.tiny, y, cw, mw, sb, lane);
                ok = warp_normalise(y, n, lane);
            }
            if (ok && right) {                                   // J x -> x
                for (int j = lane; j < n / 2; j += 32) {
                    const float2 q = y[j];
                    y[j] = y[n - 1 - j];
                    y[n - 1 - j] = q;
                }
                __syncwarp();
            }
            if (ok) {                                            // Q x: reflectors n-3 .. 0
                // (the next reflector's loads are on their way while this one is applied)
                const float* betas = slot + ab_beta_off(nmax);
                float un[kHsCols], btn = 0.0f;
                auto fetch = [&](int k) {
                    const float* u = slot + kHqHead + refl_off(n, max(k, 0));
                    btn = betas[max(k, 0)];
#pragma unroll
                    for (int q = 0; q < kHsCols; ++q)
                        if (32 * q < n - k - 1) un[q] = u[min(lane + 32 * q, n - max(k, 0) - 2)];
                };
                fetch(n - 3);
                for (int k = n - 3; k >= 0; --k) {
                    const float bt = btn;
                    float u[kHsCols];
#pragma unroll
                    for (int q = 0; q < kHsCols; ++q) u[q] = un[q];
                    fetch(k - 1);
                    if (bt == 0.0f) continue;
                    const int mm = n - k - 1;
                    float2* yk = y + k + 1 + lane;
                    float2 w[kHsCols];
                    float sr = 0.0f, si = 0.0f;
#pragma unroll
                    for (int q = 0; q < kHsCols; ++q) {
                        if (lane + 32 * q < mm) {
                            w[q] = yk[32 * q];
                            sr += u[q] * w[q].x;
                            si += u[q] * w[q].y;
                        }
                    }
                    for (int off = 16; off; off >>= 1) {
                        sr += __shfl_xor_sync(0xffffffffu, sr, off);
                        si += __shfl_xor_sync(0xffffffffu, si, off);
                    }
                    sr *= bt;
                    si *= bt;
#pragma unroll
                    for (int q = 0; q < kHsCols; ++q)
                        if (lane + 32 * q < mm) yk[32 * q] = make_float2(w[q].x - sr * u[q], w[q].y - si * u[q]);
                    __syncwarp();
                }
                ok = warp_normalise(y, n, lane);
            }
            if (lane == 0 && !ok) sh.bad[warp] = 1;
        }
        __syncthreads();
        // ---- FP64: v_A = D v_B, w_A = D^-1 w_B; two-sided Rayleigh quotient with A ----
        const float* D = slot + ab_d_off(nmax);
        for (int w = tid; w < cnt * n; w += kRfThreads) {
            const int c = w / n, j = w % n;
            const double d = (double)D[j];
            const float2 v = vec[(size_t)(2 * c) * nmax + j], u = vec[(size_t)(2 * c + 1) * nmax + j];
            vA[(size_t)c * nmax + j] = make_double2(d * v.x, d * v.y);
            wA[(size_t)c * nmax + j] = make_double2(u.x / d, u.y / d);
        }
        __syncthreads();
        {
            double acc[kRefK][6];
#pragma unroll
            for (int c = 0; c < kRefK; ++c)
#pragma unroll
                for (int q = 0; q < 6; ++q) acc[c][q] = 0.0;
            const double* A = a64 + (size_t)s * a64stride;
            for (int i = warp; i < n; i += kRfWarps) {
                const double* Ar = A + (size_t)i * n;
                double pr[kRefK], pi[kRefK];
#pragma unroll
                for (int c = 0; c < kRefK; ++c) pr[c] = pi[c] = 0.0;
                for (int j = lane; j < n; j += 32) {
                    const double aij = Ar[j];
#pragma unroll
                    for (int c = 0; c < kRefK; ++c) {
                        if (c < cnt) {
                            const double2 v = vA[(size_t)c * nmax + j];
                            pr[c] = fma(aij, v.x, pr[c]);
                            pi[c] = fma(aij, v.y, pi[c]);
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < kRefK; ++c) {
                    if (c >= cnt) continue;
                    for (int off = 16; off; off >>= 1) {
                        pr[c] += __shfl_xor_sync(0xffffffffu, pr[c], off);
                        pi[c] += __shfl_xor_sync(0xffffffffu, pi[c], off);
                    }
                    const double2 w = wA[(size_t)c * nmax + i], v = vA[(size_t)c * nmax + i];
                    // conj(w_i) (A v)_i and conj(w_i) v_i
                    acc[c][0] += w.x * pr[c] + w.y * pi[c];
                    acc[c][1] += w.x * pi[c] - w.y * pr[c];
                    acc[c][2] += w.x * v.x + w.y * v.y;
                    acc[c][3] += w.x * v.y - w.y * v.x;
                    acc[c][4] += v.x * v.x + v.y * v.y;
                    acc[c][5] += w.x * w.x + w.y * w.y;
                }
            }
            if (lane == 0)
#pragma unroll
                for (int c = 0; c < kRefK; ++c)
#pragma unroll
                    for (int q = 0; q < 6; ++q) sh.acc[warp][c][q] = acc[c][q];
        }
        __syncthreads();
        if (tid == 0) {
            bool good = true;
            double maxre = -INFINITY, minz = INFINITY;
            for (int c = 0; c < cnt; ++c) {
                double t[6] = {0, 0, 0, 0, 0, 0};
                for (int w = 0; w < kRfWarps; ++w)
                    for (int q = 0; q < 6; ++q) t[q] += sh.acc[w][c][q];
                const cplx lam = cdiv(cm(t[0], t[1]), cm(t[2], t[3]));
                const double sx = cs[4 + 2 * c], sy = cs[5 + 2 * c];
                const bool ok = !sh.bad[2 * c] && !sh.bad[2 * c + 1] && isfinite(lam.re) && isfinite(lam.im) &&
                                t[2] * t[2] + t[3] * t[3] >= 1e-10 * t[4] * t[5] &&
                                fabs(lam.re - sx) <= 2.0 * kEigDelta && fabs(fabs(lam.im) - sy) <= 2.0 * kEigDelta;
                if (!ok) {
                    good = false;
                    break;
                }
                const double mg = sqrt(lam.re * lam.re + lam.im * lam.im);
                if ((sh.flags >> (2 * c)) & 1) maxre = fmax(maxre, lam.re);
                if ((sh.flags >> (2 * c)) & 2) minz = fmin(minz, mg > 0.0 ? -lam.re / mg : 1.0);
            }
            if (!good || !(maxre > -INFINITY) || !(minz < INFINITY) || !(fabs(maxre) > kRefinedGuard) ||
                !(fabs(minz - damping_min) > kRefinedGuard)) {
                o.status[s] = 6;                                // FP64 screen instead
                atomicAdd(a.reruns, 1);
            } else {
                uint8_t k;
                if (maxre >= 0.0) k = CS_SS_UNSTABLE;
                else if (minz < damping_min) k = CS_SS_POORLY_DAMPED;
                else k = CS_SECURE;
                if (a.out.n_islands[s] > 1) {                   // main island: the scenario's class stays ISLANDED
                    if (a.out.main_klass) a.out.main_klass[s] = k;
                } else {
                    a.out.klass[s] = k;
                    a.out.severe[s] = (k != CS_SECURE);
                }
                a.out.max_re[s] = maxre;
                a.out.min_zeta[s] = minz;
                o.status[s] = 1;
            }
        }
        __syncthreads();
    }
}

}  // namespace

int dyn_ctas_per_sm() { return kCtasPerSm; }

size_t dyn_scratch_doubles(const DevNet& net) { return (size_t)make_dlayout(net).total; }

size_t dyn_hbuf_stride(const DevNet& net) {
    const int nmax = 5 * net.ng - 1;
    return (size_t)kHqHead + (size_t)((hq_off(nmax, nmax) + 3) & ~3);
}

size_t dyn_abuf_stride(const DevNet& net) { return ab_stride(5 * net.ng - 1); }

size_t dyn_a64_stride(const DevNet& net) {
    const size_t nmax = 5 * (size_t)net.ng - 1;
    return nmax * nmax;
}

size_t dyn_cand_stride() { return kCandStride; }

static size_t qr_smem_bytes(int nmax) {
    return sizeof(float) * ((size_t)((hq_off(nmax, nmax) + 3) & ~3) + 3 * (size_t)nmax);
}

static size_t refine_smem_bytes(int nmax) {
    const size_t hsz = ((size_t)hq_off(nmax, nmax) + 3) & ~(size_t)3;
    const size_t vsz = (size_t)8 * kRefK * nmax;
    return sizeof(float) * (std::max(hsz, vsz) + (((size_t)nmax + 3) & ~(size_t)3) + (size_t)kRfWarps * 4 * nmax +
                            (size_t)4 * kRefK * nmax + (size_t)kRfWarps * ((nmax + 31) / 32));
}

static size_t hess_smem_bytes(int nmax) {
    return sizeof(float) * ((size_t)((nmax + 1) / 2 + 6 + kHsSlices) * hs_ld(nmax) + 4);
}

bool dyn_split_fits(const DevNet& net, int device) {
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) return false;
    const int nmax = 5 * net.ng - 1;
    if (nmax > 32 * kHsCols) return false;
    return qr_smem_bytes(nmax) + 1024 <= (size_t)optin && hess_smem_bytes(nmax) + 1024 <= (size_t)optin &&
           refine_smem_bytes(nmax) + sizeof(RfShared) + 1024 <= (size_t)optin;
}

template <int kMode>
static cudaError_t launch_mode(const DevNet& net, const EvalArgs& a, OpfOut o, double damping_min, double* scratch,
                               size_t per_cta, const DLay& L, float* hbuf, size_t hstride, double* a64, int grid,
                               int sms, int* counter, cudaStream_t s) {
    const size_t smem = sizeof(double) * ((size_t)((net.ng + 1) >> 1) + 15 * (size_t)net.ng);
    if (smem > 48 * 1024) {
        cudaError_t e = open_shared((const void*)dyn_kernel<kMode>);
        if (e != cudaSuccess) return e;
    }
    // One block has a chain of dependent FP64 steps (the QR bulge, one warp) between wide phases: with
    // few scenarios a block of many threads shortens the wide phases, with many scenarios small blocks,
    // four per SM, fill one another's chains.  Results do not depend on the number of threads.
    // 118 buses, FP64 screen: 2,000 pairs 572 ms with four blocks of 128 threads per SM, 713 with two of 256
    // (485 now, with the one-pass Hessenberg reduction); 240 single outages 144 and 124 (112 now).
    // The front kernels have no such chain and move more memory per block: two blocks of 256.
    const bool front = kMode == DYN_FRONT || kMode == DYN_FRONT_LARGE;
    const int threads = grid <= sms ? 512 : (front || grid <= 2 * sms) ? 256 : 128;
    dyn_kernel<kMode><<<grid, threads, smem, s>>>(net, a, o, damping_min, scratch, per_cta, L, hbuf, hstride, a64,
                                                  dyn_a64_stride(net), counter);
    return cudaGetLastError();
}

cudaError_t launch_dyn(const DevNet& net, const EvalArgs& a, OpfOut o, double damping_min, int precision,
                       double* scratch, size_t scratch_per_cta, int grid, float* abuf, float* hbuf, double* a64,
                       float* cand, float* hws, int sms, int* counters, int* launches, cudaStream_t s) {
    *launches = 0;
    if (a.n <= 0) return cudaSuccess;
    const DLay L = make_dlayout(net);
    if ((size_t)L.total > scratch_per_cta) return cudaErrorInvalidValue;
    cudaError_t e;
    if (precision == CS_PREC_MIXED && hbuf && abuf && a64 && cand) {
        // FP32 screen in five kernels: front (model, balancing) at several CTAs per SM,
        // Hessenberg reduction on a two-CTA cluster, QR from shared memory at one CTA per
        // SM, FP64 refinement of the decisive eigenvalues, and the FP64 re-run of the
        // scenarios the FP32 screen cannot decide.
        const size_t hstride = dyn_hbuf_stride(net), astride = dyn_abuf_stride(net);
        e = launch_mode<DYN_FRONT>(net, a, o, damping_min, scratch, scratch_per_cta, L, abuf, astride, a64, grid, sms,
                                   counters, s);
        if (e != cudaSuccess) return e;
        const int nmax = 5 * net.ng - 1;
        const size_t hsm = hess_smem_bytes(nmax);
        e = open_shared((const void*)hess_cluster_kernel);
        if (e != cudaSuccess) return e;
        const int gh = 2 * (int)std::min<int64_t>((int64_t)std::max(1, sms / 2), a.n);
        hess_cluster_kernel<<<gh, kHsThreads, hsm, s>>>(a, o, abuf, astride, hbuf, hstride, nmax, counters + 3);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const size_t qsm = qr_smem_bytes(nmax);
        e = open_shared((const void*)hqr_smem_kernel);
        if (e != cudaSuccess) return e;
        const int gq = (int)std::min<int64_t>((int64_t)sms, a.n);
        hqr_smem_kernel<<<gq, kQrThreads, qsm, s>>>(a, o, hbuf, hstride, nmax, damping_min, cand, counters + 1);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const size_t rsm = refine_smem_bytes(nmax);
        e = open_shared((const void*)eig_refine_kernel);
        if (e != cudaSuccess) return e;
        eig_refine_kernel<<<gq, kRfThreads, rsm, s>>>(a, o, hbuf, hstride, abuf, astride, a64, dyn_a64_stride(net),
                                                       cand, nmax, damping_min, counters + 4);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        e = launch_mode<DYN_RERUN>(net, a, o, damping_min, scratch, scratch_per_cta, L, nullptr, 0, nullptr, grid, sms,
                                   counters + 2, s);
        if (e != cudaSuccess) return e;
        *launches = 5;
    } else if (precision == CS_PREC_MIXED && abuf && hws) {
        // networks whose Hessenberg matrix exceeds one block's shared memory: model and
        // balancing, the blocked Hessenberg reduction of the whole chunk on the tensor
        // cores, FP32 QR per scenario, FP64 re-run of the undecided ones
        const int nmax = 5 * net.ng - 1;
        const size_t astride = dyn_abuf_stride(net);
        e = launch_mode<DYN_FRONT_LARGE>(net, a, o, damping_min, scratch, scratch_per_cta, L, abuf, astride, nullptr, grid, sms, counters, s);
        if (e != cudaSuccess) return e;
        e = launch_hess_tc(a.n, nmax, abuf + kHqHead, (long long)astride, hws, a.err, s);
        if (e != cudaSuccess) return e;
        e = launch_mode<DYN_QR_LARGE>(net, a, o, damping_min, scratch, scratch_per_cta, L, abuf, astride, nullptr, grid, sms,
                                      counters + 1, s);
        if (e != cudaSuccess) return e;
        e = launch_mode<DYN_RERUN>(net, a, o, damping_min, scratch, scratch_per_cta, L, nullptr, 0, nullptr, grid, sms,
                                   counters + 2, s);
        if (e != cudaSuccess) return e;
        *launches = 4;
    } else if (precision == CS_PREC_MIXED) {
        e = launch_mode<DYN_MIXED_INLINE>(net, a, o, damping_min, scratch, scratch_per_cta, L, nullptr, 0, nullptr, grid, sms, counters, s);
        if (e != cudaSuccess) return e;
        *launches = 1;
    } else {
        e = launch_mode<DYN_FULL64>(net, a, o, damping_min, scratch, scratch_per_cta, L, nullptr, 0, nullptr, grid, sms,
                                    counters, s);
        if (e != cudaSuccess) return e;
        *launches = 1;
    }
    if (a.sev_n1 && a.sev_pairs) {
        int blocks = (a.n + 255) / 256;
        if (blocks > 4096) blocks = 4096;
        record_kernel<<<blocks, 256, 0, s>>>(net.nbr, net.nE, a);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        *launches += 1;
    }
    return cudaSuccess;
}
