// Fast per-instance solve for supports up to 128 tokens and n = 2 .. 32: one CTA per instance.
//
// Same mathematics as the general kernel (gr_solve.cu): the gradient of the convex functions
// of the inner system / of an outer block (Thm "Inner Convex Solver", Thm "Outer Convex Solver")
// is the one-dimensional integral
//   g_i = w_i int e^{-t slack} x_i(t) n! [lambda^n] P(lambda; t) h_i(lambda; t) dt,   x_i = e^{-t w_i},
// and Newton's method on alpha = log w uses its exact Hessian.  How the work is laid out:
//   - the power series are scaled, lambda -> sigma lambda with sigma^n = n!, so that n! disappears and every
//     coefficient is of order one (fp32 can hold them);
//   - h(mu; x) = (e^mu - 1) / (1 + x (e^mu - 1)) obeys h' = 1 + (1 - 2x) h - x (1 - x) h^2 (the logistic curve's
//     Riccati equation), which gives its coefficients stably at every x; up to eight of them come from the closed
//     polynomials in x (1 - x) that the equation generates (the cumulants of a Bernoulli variable);
//   - the product P = e^{lambda h} prod_j f_j is not multiplied out: d/dlambda log f_j = x_j d_j (1 + (1 - x_j) h_j), so
//     the log-derivative S of P is a SUM over the tokens and P follows from P' = S P;
//   - S: one thread per (quadrature node, share of the tokens), no reduction across lanes but the shares' sums;
//     P: one thread per node;  g: one thread per token, walking the nodes (no reduction at all);
//   - the Hessian's off-diagonal part  - sum_q c_q t_q (w x)_i (w x)_l n! [lambda^n] P h_i h_l  is a dense contraction over
//     (node, series index): operands staged in shared memory in fp16, MMAs, fp32 accumulators in registers from the first node to
//     the end of the factorisation.  The tokens are ordered by draft mass, so that the lower triangle pairs the series
//     P h of the heavier token (all terms positive) with the h of the lighter one, and nothing cancels;
//   - above 16 drafts the series give way to samples on a circle (eval_contour): the factors f_j are entire functions of
//     lambda, so [lambda^n] is a mean over a few points of |lambda| = 0.8 n (conjugate pairs, 16 to 24 of them), exact to
//     1e-11 and free of the cancellation that a dominant token brings into the division e / f as series;
//   - the iteration runs in fp32 as long as the residual is far above fp32's noise; the last evaluations, the only ones
//     that can end it at a tolerance below 1e-4, are fp64 and reuse the last Hessian (a Newton step with a Hessian from a point at a
//     distance of d in alpha leaves 0.02 + d of the residual at most: 0.004 away, the median, as little as one with a fresh one).
#pragma once
#include "gr_prep.cuh"
#include "gr_verify.cuh"
#include "gr_quad.cuh"

namespace gr {
namespace fast {

constexpr double kFTEnd = 25.0;       // quadrature range constants, identical to the general kernel's
constexpr double kFDrop = 1.0;
constexpr double kFTail = 3.0;
constexpr int kFMaxNodes = 128;
constexpr double kFAlphaClamp = 80.0;
constexpr double kFStepClamp = 3.0;
constexpr double kFCoarse = 1.0e-2;        // above this residual the trapezoid step is doubled
constexpr double kFPredictStep = 1.0;      // largest |delta alpha| after which the stop on a predicted residual is allowed
constexpr double kFPredictSafety = 10.0;   // the prediction s2 must be this many times below the tolerance
constexpr double kFRatioSafety = 3.0;      // the residual predicted by the last step's contraction must be this many times below the tolerance
constexpr double kFBaseSafety = 1.5;       // and what the Hessian leaves of it this many times
constexpr double kFTrustPivot = 0.02;      // smallest relative pivot at which a predicted stop is allowed
constexpr double kFPredictBound = 3.0;     // reported norm after such a stop: kFPredictBound * s2
constexpr double kFLowLeave = 3.0e-3;      // bound on the next residual (kFPredictBound * s2; it is mostly a fiftieth of that) at which the iteration goes over to fp64
constexpr double kFLowFloor = 1.0e-4;      // below this residual a failure to improve is taken for fp32's noise
constexpr double kFChordBase = 0.02;       // contraction assumed of a step by conjugate gradients (a third of what the stop allows for; 0.008 seen)
constexpr int kFCgMax = 16;                // conjugate-gradient iterations before the factorisation takes over
constexpr float kFCgTol = 2.0e-4f;         // and their relative residual; in fp32 kFCgLow times the gradient norm, up to kFCgLoose (at
                                           // 2e-4 throughout no instance of 16 shapes takes an evaluation less; 1 to 3 % more time at 128 tokens)
constexpr float kFCgLow = 0.1f, kFCgLoose = 5.0e-3f;
constexpr float kFScaleJump = 0.02f, kFScaleJumpLow = 1.0e-3f;    // distance of the common scale from which its curve is inverted exactly, in fp64 and in fp32
                                           // evaluations (a difference of logarithms: good to 1e-7, which has to be far below the distance, and near the solution below the tolerance)
constexpr float kFScaleJumpFar = 0.5f;     // the same where it is known roughly, and under a cap of one or two evaluations
constexpr float kFSmallSlack = 1.0e-4f;     // share of the mass below which Tn - sum g is mostly rounding in fp32
constexpr float kFLeastSlack = 1.0e-9f;     // and the least share aimed at (the quadrature's floor)
constexpr double kFLowEnds = 1.0e-4;       // tolerance from which on an fp32 evaluation may end the iteration
constexpr float kFNone = 1.0e30f;          // no residual or ratio yet

// Compile-time geometry.  NT: series length (>= n), MP: padded support size, T: threads, JC: Hessian nodes staged
// together, CTAS: CTAs per SM the registers are held to, QC: quadrature nodes handled together.
template <int NT_, int MP_, int T_, int JC_, int CTAS_, int QC_ = 32>
struct Cfg {
    static constexpr int NT = NT_, MP = MP_, T = T_, JC = JC_, kCtas = CTAS_, kQC = QC_;
    static constexpr bool kContour = NT > 16;     // samples on a circle instead of series (NT: largest number of them)
    // Fixed-point sweeps of the starting point: five where an evaluation weighs more than the sweeps, three elsewhere.  Whole calls, us, three / five sweeps:
    // one headline row 50.8 / 48.7, 256 rows of n = 4, k = 8 52.0 / 51.5, 64 whole rows of 16 ids 60.8 / 59.1 (evaluations 3.96 / 3.81); full SMs 1024
    // headline rows 280.6 / 283.0 (3.04 / 3.01), 600 rows of n = 12, k = 50 138.4 / 139.2; up to 128 tokens, 4096 rows of n = 16, k = 100 1431 / 1460, 600 of n = 8
    // 223.5 / 221.9.  On the circle 512 rows of n = 32, k = 20 107.1 / 102.8 (2.74 / 2.31); solve calls up to 64 tokens, 700 rows of n = 17, k = 50 195.8 / 188.4, of
    // n = 20, k = 40 182.9 / 173.6, of n = 32, k = 50 218.5 / 205.5, 256 rows of these 84.7 / 89.9, 78.3 / 75.9, 97.2 / 95.9 (evaluations 2.98 / 2.69, 2.94 / 2.42,
    // 2.97 / 2.55); up to 128 tokens 700 rows of n = 24, k = 128 480 / 492, 64 of n = 20, k = 100 131 / 112 (one evaluation more in the slowest instance).
    static constexpr int kSweeps = kContour || (MP <= 64 && (NT == 16 || kCtas <= 2)) ? 5 : 3;
    static constexpr int kNG = T / MP;            // copies of the token threads (they share the nodes out among them)
    static constexpr int kW = T / 32, kTW = MP / 32;
    static constexpr int kRow = NT + 4;           // row stride of the product series (16-byte aligned rows in fp32 and fp64)
    static constexpr int kTS = MP + 4;            // token stride of the staged operands: conflict-free fragment loads
    static constexpr int kPanels = MP / 8;
    static constexpr int kPr = MP / 32;           // pairs of 16-row tiles (a, MP / 16 - 1 - a): equal work per pair
    static constexpr int kS = kW / kPr;           // warps that share a pair's column tiles
    static constexpr int kNA = (MP / 16 + kS - 1) / kS, kNB = (MP / 8 + kS - 1) / kS;
    static constexpr int kPack = NT >= 16 ? 1 : 16 / NT;   // Hessian nodes that fill one MMA depth of 16
    static constexpr int kKS = kContour ? (JC * NT + 7) / 8 : JC / kPack;   // MMA steps per staged chunk
    static_assert(T % MP == 0 && kW % kPr == 0 && kS * kNB <= MP / 8 && T >= kQC && JC % kPack == 0, "geometry");
    // shared memory, byte offsets
    static constexpr int oD = 0, oRhs = oD + MP * 8, oDr = oRhs + MP * 8, oWd = oDr + (MP + 4) * 8, oDsd = oWd + MP * 8;
    static constexpr int oRed = oDsd + MP * 8, oScal = oRed + 64 * 8, oTq = oScal + 16 * 8, oCq = oTq + kQC * 8, oKq = oCq + kQC * 8;
    // (contour: x of every token and node in SP, samples of the product in PP, their square roots behind them (only the fp32
    // evaluation, which leaves half of PP free, has them), tables of e^(lambda d) - 1
    // in fp64 and fp32, and the samples' weights)
    static constexpr int kXS = kQC + 1;
    static constexpr int kPPBytes = kContour ? NT * kQC * 16 : kQC * kRow * 8;
    static constexpr int kSPMin = T * 16 > MP * 16 ? T * 16 : MP * 16;
    static constexpr int kSPShares = kW * kQC * (NT + 2) * 8, kSPVec = T * 16 + 12 * (MP + 4 * kNG);
    static constexpr int kSPBytes = !kContour ? (kSPShares > kSPVec ? kSPShares : kSPVec) : (MP * kXS * 8 > kSPMin ? MP * kXS * 8 : kSPMin);
    static constexpr int oPP = oKq + kQC * 4, oSP = oPP + kPPBytes, oSQ = oPP + NT * kQC * 8;
    static constexpr int oEd = oSP + kSPBytes, oEs = oEd + (kContour ? NT * MP * 16 : 0);
    static constexpr int oCd = oEs + (kContour ? NT * MP * 8 : 0);
    static constexpr int oWf = oCd + (kContour ? NT * 16 : 0), oDsf = oWf + MP * 4, oE = oDsf + MP * 4;
    static constexpr int oDg = oE + (NT <= 8 ? MP * 32 : 0), oYv = oDg + MP * 4, oDl = oYv + MP * 4;
    static constexpr int oLd = oDl + MP * 4;                     // factored 8 x 8 diagonal blocks
    static constexpr int oBlk = oLd + kPanels * 64 * 4, oOrd = oBlk + MP * 4, oTr = oOrd + MP * 4;
    static constexpr int oU = (oTr + MP * 4 + 15) & ~15;           // union: staging / factor / start table / preparation
    static constexpr int kStage = kKS * 4 * kTS * 8;               // bytes of one staged operand (contour: the only one)
    static constexpr int kLFloats = 8 * (MP * kPanels - 4 * kPanels * (kPanels - 1));
    static constexpr int kNS = MP + 8;                             // row stride of the scaled Hessian (halves): conflict-free rows
    static constexpr int kPi = MP * kNS * 2;
    static constexpr int kPrep = MP * 8 * 3 + (MP + 4) * 8 + MP * 8;
    static constexpr int kOps = kContour ? 1 : 2;
    static constexpr int kU0 = kOps * kStage > kLFloats * 4 ? kOps * kStage : kLFloats * 4;
    static constexpr int kU1 = kPi > kPrep ? kPi : kPrep;
    static constexpr int kU2 = kU0 > kU1 ? kU0 : kU1;
    static constexpr int kU = kU2 > kVerifyScratchBytes ? kU2 : kVerifyScratchBytes;
    static constexpr int kBytes = oU + kU;
};

extern __shared__ __align__(16) unsigned char smem_raw[];

// four (fp32) or two (fp64) consecutive elements; the other type's version is never called
template <class P> __device__ __forceinline__ void ld_vec(const P& p, float* o) { const float4 v = ld_f4(p); o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
template <class P> __device__ __forceinline__ void ld_vec(const P& p, double* o) { const double2 v = ld_d2(p); o[0] = v.x; o[1] = v.y; }
template <class P> __device__ __forceinline__ void st_vec(const P& p, const float* o) { st_f4(p, make_float4(o[0], o[1], o[2], o[3])); }
template <class P> __device__ __forceinline__ void st_vec(const P& p, const double* o) { st_d2(p, make_double2(o[0], o[1])); }

// Every array of the layout.  The base is the kernel's dynamic shared memory, so the addresses are constants wherever this
// is constructed (functions that are kept out of line build it for themselves).
template <class C>
struct FSm {
    GR_PTR(double) d, rhs, Dr, wd, dsd, red, scal;
    GR_PTR(float) wf, E, dg, yv, dl, Ld, Lp;
    GR_PTR(uint32_t) AS, HS;       // staged operands: half2 elements [step][4][token][2]
    GR_PTR(float) kq;
    GR_PTR(__half) pi;              // start: presence probabilities; later the scaled Hessian (row stride kNS)
    GR_PTR(int) blk, ord, trunc;
    char* base;
    int* flag;
    __device__ __forceinline__ explicit FSm(int* ck) {
        char* const sb = reinterpret_cast<char*>(smem_raw);
        base = sb; flag = ck;
        d = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oD), C::MP, ck);
        rhs = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oRhs), C::MP, ck);
        Dr = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oDr), C::MP + 4, ck);
        wd = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oWd), C::MP, ck);
        dsd = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oDsd), C::MP, ck);
        red = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oRed), 64, ck);
        scal = GR_MKPTR(double, reinterpret_cast<double*>(sb + C::oScal), 16, ck);
        wf = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oWf), C::MP, ck);
        E = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oE), C::MP * 8, ck);
        dg = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oDg), C::MP, ck);
        yv = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oYv), C::MP, ck);
        dl = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oDl), C::MP, ck);
        Ld = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oLd), C::kPanels * 64, ck);
        blk = GR_MKPTR(int, reinterpret_cast<int*>(sb + C::oBlk), C::MP, ck);
        ord = GR_MKPTR(int, reinterpret_cast<int*>(sb + C::oOrd), C::MP, ck);
        trunc = GR_MKPTR(int, reinterpret_cast<int*>(sb + C::oTr), C::MP, ck);
        AS = GR_MKPTR(uint32_t, reinterpret_cast<uint32_t*>(sb + C::oU), C::kStage / 4, ck);
        HS = GR_MKPTR(uint32_t, reinterpret_cast<uint32_t*>(sb + C::oU + (C::kOps - 1) * C::kStage), C::kStage / 4, ck);
        kq = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oKq), C::kQC, ck);
        Lp = GR_MKPTR(float, reinterpret_cast<float*>(sb + C::oU), C::kLFloats, ck);
        pi = GR_MKPTR(__half, reinterpret_cast<__half*>(sb + C::oU), C::MP * C::kNS, ck);
    }
};
// (what stays the same during a system is read from here: kept in registers it was spilled around every call)
enum { SC_FAIL = 0, SC_PIVOT = 1, SC_NP = 2, SC_RANGE = 3, SC_OUT = 4, SC_TOL = 8, SC_QSTEP = 9, SC_SIGMA = 10, SC_HS = 11, SC_TN = 12, SC_GNORM = 13, SC_ITERS = 14, SC_RATIO = 15 };

// The circle of the contour kernels: `np` conjugate pairs of points r e^(i theta), angles theta and n theta (mod 2 pi),
// factor 2 n! / (N r^n) of the mean.
constexpr int kMaxPoints = 24;
struct Circle { int np; double r, factor; double ct[kMaxPoints], st[kMaxPoints], nth[kMaxPoints]; };
struct NoCircle {};
template <bool> struct CircleOf { typedef NoCircle type; };
template <> struct CircleOf<true> { typedef Circle type; };

// Arrays whose element type is the precision of the evaluation.
template <class C, typename R>
struct RSm {
    GR_PTR(R) tq, cq, PP, SP, w, ds;
    __device__ explicit RSm(const FSm<C>& sm) {
        tq = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oTq), C::kQC, sm.flag);
        cq = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oCq), C::kQC, sm.flag);
        PP = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oPP), C::kPPBytes / (int)sizeof(R), sm.flag);
        SP = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oSP), C::kSPBytes / (int)sizeof(R), sm.flag);
        const int ow = sizeof(R) == 4 ? C::oWf : C::oWd, od = sizeof(R) == 4 ? C::oDsf : C::oDsd;
        w = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + ow), C::MP, sm.flag);
        ds = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + od), C::MP, sm.flag);
    }
};

__device__ __forceinline__ double ipow(double x, int n) {
    double r = 1.0;
#pragma unroll 1
    while (n > 0) { if (n & 1) r *= x; x *= x; n >>= 1; }
    return r;
}

__device__ __forceinline__ float ex2_approx(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
template <typename R> struct Rx;
template <> struct Rx<double> {
    static __device__ __forceinline__ double expneg(double y) { return exp_neg(y); }
    static __device__ __forceinline__ double ex(double x) { return m_exp(x); }
    static __device__ __forceinline__ double lg(double x) { return m_log(x); }
};
template <> struct Rx<float> {
    static __device__ __forceinline__ float expneg(float y) { return ex2_approx(y * -1.4426950408889634f); }
    static __device__ __forceinline__ float ex(float x) { return ex2_approx(x * 1.4426950408889634f); }
    static __device__ __forceinline__ float lg(float x) { return __logf(x); }
};

// Two fp32 numbers (of two tokens or of two quadrature nodes) as one operand of the formulas below.
struct F2 {
    unsigned long long v;
    __device__ __forceinline__ F2() {}
    __device__ __forceinline__ explicit F2(unsigned long long x) : v(x) {}
    __device__ __forceinline__ explicit F2(double c) : v(f_pack((float)c, (float)c)) {}
    __device__ __forceinline__ explicit F2(float c) : v(f_pack(c, c)) {}
    __device__ __forceinline__ explicit F2(int c) : F2((float)c) {}
    __device__ __forceinline__ F2(float lo, float hi) : v(f_pack(lo, hi)) {}
    __device__ __forceinline__ float lo() const { return f_lo(v); }
    __device__ __forceinline__ float hi() const { return f_hi(v); }
};
using ::fma;
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return F2(fma2(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(mul2(a.v, b.v)); }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(add2(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return fma(b, F2(-1.f), a); }

// h[c], c = 1 .. N (N <= 8): coefficients of h(mu; x), from u = 1 - 2x and p = x (1 - x)
// (closed forms of the Riccati recurrence below).
template <int N, typename R>
__device__ __forceinline__ void unit_series(R u, R p, R* h)
{
    h[1] = R(1);
    if (N >= 2) h[2] = u * R(0.5);
    if (N >= 3) h[3] = R(1.0 / 6) - p;
    if (N >= 4) h[4] = u * fma(p, R(-0.5), R(1.0 / 24));
    if (N >= 5) h[5] = fma(p, p - R(0.25), R(1.0 / 120));
    if (N >= 6) h[6] = u * fma(p, fma(p, R(0.5), R(-1.0 / 12)), R(1.0 / 720));
    if (N >= 7) h[7] = fma(p, fma(p, R(1.0 / 3) - p, R(-1.0 / 40)), R(1.0 / 5040));
    if (N >= 8) h[8] = u * fma(p, fma(p, fma(p, R(-0.5), R(1.0 / 8)), R(-1.0 / 160)), R(1.0 / 40320));
}
// h[c], c = 1 .. N: coefficients of h(ds lambda; x) in lambda by the Riccati recurrence
//   (c + 1) h_{c+1} = ds (1 - 2x) h_c - ds x (1 - x) sum_{a=1}^{c-1} h_a h_{c-a},   h_1 = ds.
template <int N, typename R>
__device__ __forceinline__ void riccati_series(R ds, R du, R dp, R* h)
{
    h[1] = ds;
    const R m2 = R(-2) * dp;
#pragma unroll
    for (int c = 1; c < N; c++) {
        // (the term with the newest coefficient last: the others do not wait for it)
        R a = R(0);
        if (c % 2 == 0) a = (R(0.5) * h[c / 2]) * h[c / 2];
#pragma unroll
        for (int k = (c - 1) / 2; k >= 1; k--) a = c % 2 != 0 && k == (c - 1) / 2 ? h[k] * h[c - k] : fma(h[k], h[c - k], a);
        h[c + 1] = fma(m2, a, du * h[c]) * R(1.0 / (c + 1));
    }
}

__device__ __forceinline__ void mma_tf32(float* c, const float* a, const float* b)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])),
                   "r"(__float_as_uint(a[3])), "r"(__float_as_uint(b[0])), "r"(__float_as_uint(b[1])));
}

__device__ __forceinline__ void mma_f16(float* c, const uint32_t* a, const uint32_t* b)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ uint32_t pack_half(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Sums (fp64 and fp32) and maxima (unsigned) over the token threads, every thread gets them: the first kTW warps hold the
// tokens (the other copies hold the same values, and no barrier is needed where a warp holds them all).  Two scratch areas
// in turn (`par`), one barrier for all values of a call: what an iteration needs is asked for together, since a call costs
// about 400 cycles whatever it carries.
template <class C, int ND, int NF, int NU>
__device__ __forceinline__ void tok_reduce(const FSm<C>& sm, double* d, float* f, unsigned* u, int& par)
{
    static_assert(ND <= 2 && NF <= 4 && NU <= 4 && C::kTW <= 4, "a warp's slot is eight doubles");
    __syncwarp();
    const int w = threadIdx.x >> 5;
    if (C::kTW == 1 || w < C::kTW) {
#pragma unroll
        for (int k = 0; k < NU; k++) u[k] = __reduce_max_sync(0xffffffffu, u[k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < ND; k++) d[k] += __shfl_xor_sync(0xffffffffu, d[k], o);
#pragma unroll
            for (int k = 0; k < NF; k++) f[k] += __shfl_xor_sync(0xffffffffu, f[k], o);
        }
    }
    if (C::kTW == 1) return;
    GR_PTR(double) area = sm.red + 32 * par;
    par ^= 1;
    if ((threadIdx.x & 31) == 0 && w < C::kTW) {
        GR_PTR(double) r = area + 8 * w;
        if (ND > 0) st_d2(r, make_double2(d[0], ND > 1 ? d[ND > 1 ? 1 : 0] : 0.0));
        if (NF > 0) st_f4(GR_PCAST(float, r + 2), make_float4(f[0], NF > 1 ? f[NF > 1 ? 1 : 0] : 0.f, NF > 2 ? f[NF > 2 ? 2 : 0] : 0.f, NF > 3 ? f[NF > 3 ? 3 : 0] : 0.f));
        if (NU > 0) st_f4(GR_PCAST(float, r + 4), make_float4(__uint_as_float(u[0]), __uint_as_float(u[NU > 1 ? 1 : 0]), __uint_as_float(u[NU > 2 ? 2 : 0]), __uint_as_float(u[NU > 3 ? 3 : 0])));
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < C::kTW; i++) {
        GR_PTR(double) r = area + 8 * i;
        if (ND > 0) {
            const double2 t = ld_d2(r);
            d[0] = i == 0 ? t.x : d[0] + t.x;
            if (ND > 1) d[ND > 1 ? 1 : 0] = i == 0 ? t.y : d[ND > 1 ? 1 : 0] + t.y;
        }
        if (NF > 0) {
            const float4 t = ld_f4(GR_PCAST(float, r + 2));
            const float tv[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int k = 0; k < NF; k++) f[k] = i == 0 ? tv[k] : f[k] + tv[k];
        }
        if (NU > 0) {
            const float4 t = ld_f4(GR_PCAST(float, r + 4));
            const float tv[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int k = 0; k < NU; k++) u[k] = i == 0 ? __float_as_uint(tv[k]) : max(u[k], __float_as_uint(tv[k]));
        }
    }
}
template <class C>
__device__ __forceinline__ double tok_sum(const FSm<C>& sm, double v, int& par)
{
    tok_reduce<C, 1, 0, 0>(sm, &v, nullptr, nullptr, par);
    return v;
}

// Accumulator fragments of the tiles a warp owns: row tiles a and b of its pair, column tiles cs, cs + kS, ...
template <class C>
struct Frags { float A[C::kNA][4], B[C::kNB][4]; };

// Adds the staged operands (ksteps MMA depths of 16) to the fragments.  Straight-line: every tile of the pair, those above
// the diagonal included, so that the loads of a step go out together.  (An m16n8k16 fp16 MMA takes the tensor pipe as long
// as an m16n8k8 tf32 one, 8 cycles, and carries the same mantissa.)
template <class C>
__device__ __forceinline__ void hess_mma(const FSm<C>& sm, Frags<C>& fr, int ksteps)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gid = lane >> 2, tig = lane & 3;
    const int ra = warp % C::kPr, rb = C::MP / 16 - 1 - ra, cs = warp / C::kPr;
#pragma unroll 1
    for (int ks = 0; ks < ksteps; ks++) {
        GR_PTR(const uint32_t) Ap = sm.AS + 2 * ((ks * 4 + tig) * C::kTS + gid);
        GR_PTR(const uint32_t) Hp = sm.HS + 2 * ((ks * 4 + tig) * C::kTS + gid);
        uint2 hv[C::kNB];
#pragma unroll
        for (int s = 0; s < C::kNB; s++) hv[s] = ld_u2(Hp + 16 * (cs + s * C::kS));
        if (C::kContour) {
            // Re(a b) = Re a Re b - Im a Im b
#pragma unroll
            for (int s = 0; s < C::kNB; s++) { hv[s].x ^= 0x80000000u; hv[s].y ^= 0x80000000u; }
        }
        const uint2 a0 = ld_u2(Ap + 32 * ra), a1 = ld_u2(Ap + 32 * ra + 16), b0 = ld_u2(Ap + 32 * rb), b1 = ld_u2(Ap + 32 * rb + 16);
        const uint32_t fa[4] = {a0.x, a1.x, a0.y, a1.y}, fb[4] = {b0.x, b1.x, b0.y, b1.y};
#pragma unroll
        for (int s = 0; s < C::kNB; s++) {
            const uint32_t bb[2] = {hv[s].x, hv[s].y};
            if (s < C::kNA) mma_f16(fr.A[s < C::kNA ? s : 0], fa, bb);
            mma_f16(fr.B[s], fb, bb);
        }
    }
}

// Extent of a point's weights: the extreme log-weights, and the largest over the smallest total W of a tuple's weights (slack +
// sum over its distinct tokens), infinite where the caller's quadrature step asks for more than the tables hold.
// Beside it which sum an fp32 evaluation takes: its nodes (0: the trapezoid rule) and first entry.  In shared memory, written by one thread (a
// barrier before it is read is the caller's): five registers of every thread across the evaluations were spilled around them, and every thread looked for the
// level (512 rows of n = 16, k = 20 86.1 -> 84.4 us a solve call, 1024 headline rows 270.6 -> 269.1, 4096 of n = 16, k = 100 1387 -> 1378; on the circle 700 of n = 24, k = 64
// 209.5 -> 212.4).
struct Extent { float amax, amin, ratio; int nodes, at; };
template <class C>
__device__ __forceinline__ void put_extent(const FSm<C>& sm, float amax, float amin, float wsum, int n, int slack)
{
    const float s = slack ? 1.f : 0.f;
    // (rounded up: exponentials of fp32 log-weights are good to 1e-5, the quotient to 2 ulp, its divisor within e^80 + 1.  One thread's chain: with a
    // correctly rounded quotient, us a call, 64 whole rows of 16 ids 68.3 for 67.7, 256 rows of n = 4, k = 8 52.1 for 51.7, one headline row 53.1 for 52.8)
    const float ratio = sm.scal[SC_QSTEP] >= kTableStep ? __fdividef(1.0001f * (s + fminf(wsum, (float)n * Rx<float>::ex(amax))), s + Rx<float>::ex(amin)) : INFINITY;
    const bool fine = sm.scal[SC_TOL] >= kFLowEnds;
    const int level = fine ? quad_level<double>(ratio) : quad_level<float>(ratio);
    const int nodes = level < (fine ? kLevels64 : kLevels32) ? 2 * (level + 1) : 0;
    GR_PTR(float) e = GR_PCAST(float, sm.scal);
    e[2 * SC_RANGE] = amax; e[2 * SC_RANGE + 1] = amin; e[2 * SC_RATIO] = ratio;
    e[2 * SC_RATIO + 1] = __int_as_float(nodes | (level * (level + 1) + (fine ? kFine : 0)) << 8);
}
template <class C>
__device__ __forceinline__ Extent get_extent(const FSm<C>& sm)
{
    GR_PTR(const float) e = GR_PCAST(const float, sm.scal);
    const int low = __float_as_int(e[2 * SC_RATIO + 1]);
    return Extent{e[2 * SC_RANGE], e[2 * SC_RANGE + 1], e[2 * SC_RATIO], low & 255, low >> 8};
}

// Quadrature nodes for one evaluation, of R's accuracy.  Where 1 / W is wanted for W in a known interval, the fewest nodes are those of the
// best exponential sum on it (gr_quad.cuh): 4 to 16 where the trapezoid rule in the log-time variable, with its lower tail
// compressed below s0, takes 20 to 30 for the same accuracy.  The trapezoid rule serves the rest: wider intervals and steps below kTableStep.
// (Where a grid lies does not matter to its accuracy: fp32.)
template <typename R>
struct Grid {
    int Q;
    bool table;
    R unit;                         // table: 1 / smallest W; else the step
    int at;                         // table: first entry
    float s_hi, s0;
    __device__ __forceinline__ Grid(const Extent& e, int slack, R qstep)
    {
        const float wmin = Rx<float>::ex(e.amin), s = slack ? 1.f : 0.f;
        int level = 0;
        if (sizeof(R) == 8) { level = quad_level<double>(e.ratio); table = level < kLevels64; }
        else table = e.nodes > 0;
        if (table) {
            Q = sizeof(R) == 8 ? 2 * (level + 1) : e.nodes; at = sizeof(R) == 8 ? level * (level + 1) : e.at;
            unit = (R)__fdividef(1.00005f, s + wmin);              // (any number not below 1 / lo)
            s_hi = s0 = 0.f;
        } else {
            s_hi = Rx<float>::lg((float)kFTEnd / (s + wmin));
            s0 = -Rx<float>::lg(s + Rx<float>::ex(e.amax)) - (float)kFDrop;
            Q = min((int)ceilf((s_hi - (s0 - (float)kFTail)) / (float)qstep) + 1, kFMaxNodes);
            unit = qstep; at = 0;
        }
    }
    // node q (any q; beyond the last one of a table: the last) and its weight, e^(-t slack) included
    __device__ __forceinline__ void node(int q, int slack, R& t, R& c) const
    {
        if (table) {
            R tc, cc;
            QuadTable<R>::load(at + min(q, Q - 1), tc, cc);
            t = tc * unit; c = cc * unit;
        } else {
            const R s = (R)s_hi - unit * (R)q, e = Rx<R>::expneg(s - (R)s0);
            t = Rx<R>::expneg(e - s);
            c = unit * (R(1) + e) * t;
        }
        if (slack) c *= Rx<R>::expneg(t);
    }
};
// Node slots of an evaluation's first phase (a power of two; the threads beyond one set share out the tokens).
__device__ __forceinline__ int slot_bits(int nq) { return nq <= 8 ? 3 : nq <= 16 ? 4 : 5; }
// Sums over the shares that a warp holds of the same nodes (32 >> bits lanes each), left in `row`: lanes that meet each go on with half
// of the series, so two steps take 3/4 of NT shuffles.
template <int N, typename R, class P>
__device__ __forceinline__ void st_row(const P& row, const R* v)
{
    constexpr int kVec = 16 / (int)sizeof(R);
#pragma unroll
    for (int c = 0; c < N; c += N % kVec ? 1 : kVec) { if constexpr (N % kVec) row[c] = v[c]; else st_vec(row + c, v + c); }
}
template <int NT, typename R, class P>
__device__ __forceinline__ void put_shares(R* S, int bits, bool on, const P& row)
{
    const int lane = threadIdx.x & 31;
    if (bits == 5) {
        if (on) st_row<NT>(row, S);
        return;
    }
    __syncwarp();
    auto meet = [&](int half, int o) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int c = 0; c < NT / 2; c++) {
            if (c < half) {
                const R send = up ? S[c] : S[c + half], keep = up ? S[c + half] : S[c];
                S[c] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
    };
    meet(NT / 2, 16);
    const int c0 = lane & 16 ? NT / 2 : 0;
    if (bits == 3) {
        meet(NT / 4, 8);
        if (on) st_row<NT / 4>(row + c0 + (lane & 8 ? NT / 4 : 0), S);
    } else if (on) {
        st_row<NT / 2>(row + c0, S);
    }
}

// Sum of (g, g2) over the copies of the token threads, in the same order everywhere.  (A barrier before the array is written
// again is the caller's.)
template <class C>
__device__ __forceinline__ void sum_copies(const FSm<C>& sm, double& g, double& g2)
{
    if (C::kNG > 1) {
        const int tid = threadIdx.x, i = tid % C::MP;
        GR_PTR(double) gs = GR_MKPTR(double, reinterpret_cast<double*>(sm.base + C::oSP), C::kSPBytes / 8, sm.flag);
        st_d2(gs + 2 * tid, make_double2(g, g2));
        __syncthreads();
        g = 0.0; g2 = 0.0;
#pragma unroll
        for (int k = 0; k < C::kNG; k++) { const double2 t = ld_d2(gs + 2 * (k * C::MP + i)); g += t.x; g2 += t.y; }
    }
}

// Arrays of the contour kernels; complex numbers are pairs of R.
template <class C, typename R>
struct CSm {
    GR_PTR(R) tq, cq, X, P, E, c, w;
    GR_PTR(float) sq;
    __device__ explicit CSm(const FSm<C>& sm) {
        constexpr int k = (int)sizeof(R);
        tq = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oTq), C::kQC, sm.flag);
        cq = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oCq), C::kQC, sm.flag);
        X = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oSP), C::MP * C::kXS, sm.flag);
        P = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + C::oPP), 2 * C::NT * C::kQC, sm.flag);
        E = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + (k == 4 ? C::oEs : C::oEd)), 2 * C::NT * C::MP, sm.flag);
        w = GR_MKPTR(R, reinterpret_cast<R*>(sm.base + (k == 4 ? C::oWf : C::oWd)), C::MP, sm.flag);
        sq = GR_MKPTR(float, reinterpret_cast<float*>(sm.base + C::oSQ), 2 * C::NT * C::kQC, sm.flag);
    }
};
template <class P> __device__ __forceinline__ void ld_c(const P& p, float& a, float& b) { const float2 v = ld_f2(p); a = v.x; b = v.y; }
template <class P> __device__ __forceinline__ void ld_c(const P& p, double& a, double& b) { const double2 v = ld_d2(p); a = v.x; b = v.y; }
template <class P> __device__ __forceinline__ void st_c(const P& p, float a, float b) { st_f2(p, make_float2(a, b)); }
template <class P> __device__ __forceinline__ void st_c(const P& p, double a, double b) { st_d2(p, make_double2(a, b)); }

// Tables of a system for the contour: e^(lambda_p d_j) - 1 for every point and token, and the points' weights
// 2 n! / (N r^n) e^(-i n theta_p) e^(lambda_p h) T^n, with the masses relative to the system's total T.
template <class C>
__device__ __noinline__ void contour_tables(const Circle& ci, int m, double rel, double hrel, double Tn, int* flag)
{
    const FSm<C> sm(flag);
    const CSm<C, double> cd(sm);
    const CSm<C, float> cf(sm);
    GR_PTR(double) cw = GR_MKPTR(double, reinterpret_cast<double*>(sm.base + C::oCd), 2 * C::NT, flag);
    const int tid = threadIdx.x, i = tid % C::MP;
    // (points p and np - 1 - p lie on either side of the imaginary axis, angles theta and pi - theta: one sine and cosine for both, and the reciprocal
    // of the exponential.  np is a multiple of four.)
    for (int p = tid / C::MP; p < ci.np / 2; p += C::kNG) {
        double sn = 0.0, cs = 1.0, e = 1.0;
        if (i < m) { sincos(ci.r * ci.st[p] * rel, &sn, &cs); e = m_exp(ci.r * ci.ct[p] * rel); }
#pragma unroll
        for (int z = 0; z < 2; z++) {
            const int at = z == 0 ? p : ci.np - 1 - p;
            const double re = e * cs - 1.0, im = e * sn;
            st_d2(cd.E + 2 * (at * C::MP + i), make_double2(re, im));
            st_f2(cf.E + 2 * (at * C::MP + i), make_float2((float)re, (float)im));
            if (z == 0) e = __drcp_rn(e);
        }
    }
    if (tid < ci.np) {
        double sn, cs;
        sincos(ci.r * ci.st[tid] * hrel - ci.nth[tid], &sn, &cs);
        const double e = m_exp(ci.r * ci.ct[tid] * hrel) * ci.factor * Tn;
        st_d2(cw + 2 * tid, make_double2(e * cs, e * sn));
    }
    if (tid == 0) sm.scal[SC_NP] = (double)ci.np;
}

__device__ __forceinline__ float recip(float x) { return __fdividef(1.f, x); }
__device__ __forceinline__ double recip(double x) { return __drcp_rn(x); }

// As eval_system (same arguments and results), with [lambda^n] taken as a mean over points of a circle:
//   M = sum_p c_p prod_j f_pj,  dM/dx_i = sum_p Re(P_p h_pi),  d2M/dx_i dx_l = sum_p Re(P_p h_pi h_pl),
//   f_pj = 1 + x_j E_pj,  h = E / f,  E_pj = e^(lambda_p d_j) - 1 (tables).
// The rounded f that went into the product is the one that is divided out again, so a factor close to zero does no harm.
// For the Hessian sqrt(P_p) h_pi is staged, once, as (Re, Im) half pairs: products of two such are of order one, whatever
// the token's mass.  Errors against 96 points and fp64 throughout, n = 17 to 32, largest mass 0.12 to 0.6: flows 1e-11 in
// fp64, 1e-7 in fp32; scaled Hessian 2e-5 from 11-bit operands.
template <class C, typename R, bool kJac>
__device__ __forceinline__ void eval_contour(const FSm<C>& sm, int m, int slack, double qstep_d, int jstride,
                                             double w_own, float z_own, double& g_out, double& g2_out, Frags<C>& fr)
{
    constexpr int T = C::T;
    const CSm<C, R> cs(sm);
    GR_PTR(double) cw = GR_MKPTR(double, reinterpret_cast<double*>(sm.base + C::oCd), 2 * C::NT, sm.flag);
    const int tid = threadIdx.x, i = tid % C::MP, ng = tid / C::MP;
    const int np = (int)sm.scal[SC_NP];
    const R wi = (R)w_own;
    const Grid<R> grid(get_extent(sm), slack, (R)qstep_d);
    const int Q = grid.Q;
    R g = R(0), g2 = R(0);
    if (kJac) {
#pragma unroll
        for (int s = 0; s < C::kNA; s++) { fr.A[s][0] = fr.A[s][1] = fr.A[s][2] = fr.A[s][3] = 0.f; }
#pragma unroll
        for (int s = 0; s < C::kNB; s++) { fr.B[s][0] = fr.B[s][1] = fr.B[s][2] = fr.B[s][3] = 0.f; }
    }
    const bool live = kJac || (i & ~31) < m;
#pragma unroll 1
    for (int q0 = 0; q0 < Q; q0 += C::kQC) {
        const int nq = min(C::kQC, Q - q0);
        // ---- x of every token at this thread's node
        // (threads are dealt to nodes evenly: 5 nodes of 24 points are one round of 128 threads)
        const int grp = tid / nq, q = tid - grp * nq, G = T / nq;
        if (grp < G) {
            R t, c0;
            grid.node(q0 + q, slack, t, c0);
            if (grp == 0) {
                cs.tq[q] = t; cs.cq[q] = c0;
                if (kJac) sm.kq[q] = sqrtf((float)((R)jstride * c0 * t));
            }
#pragma unroll 2
            for (int j = grp; j < m; j += G) cs.X[j * C::kXS + q] = Rx<R>::expneg(t * cs.w[j]);
        }
        __syncthreads();
        // ---- product of the factors, one thread per (node, point)
        if (grp < G) {
#pragma unroll 1
            for (int p = grp; p < np; p += G) {
                R a = (R)cw[2 * p], b = (R)cw[2 * p + 1];
#pragma unroll 4
                for (int j = 0; j < m; j++) {
                    const R x = cs.X[j * C::kXS + q];
                    R er, ei;
                    ld_c(cs.E + 2 * (p * C::MP + j), er, ei);
                    const R fx = fma(x, er, R(1)), fy = x * ei;
                    const R a2 = fma(a, fx, -(b * fy));
                    b = fma(a, fy, b * fx);
                    a = a2;
                }
                st_c(cs.P + 2 * (p * C::kQC + q), a, b);
                if (kJac) {
                    // square root, either branch: only products of two of them are used
                    const float af = (float)a, bf = (float)b, mag = sqrtf(fmaf(af, af, bf * bf));
                    const float u = sqrtf(0.5f * (mag + fabsf(af))), v = u > 0.f ? __fdividef(0.5f * bf, u) : 0.f;
                    st_c(cs.sq + 2 * (p * C::kQC + q), af >= 0.f ? u : fabsf(v), af >= 0.f ? v : copysignf(u, bf));
                }
            }
        }
        __syncthreads();
        // ---- g: one thread per token, its copies share out the points; with kJac the operands of the contraction for every jstride-th node
        const int span = kJac ? jstride * C::JC : nq, pw = np / C::kNG;
#pragma unroll 1
        for (int qa = 0; qa < nq; qa += span) {
            const int qb = min(nq, qa + span);
            const int nst = kJac ? (qb - qa + jstride - 1) / jstride : 0;
            if (live) {
#pragma unroll 1
                for (int q2 = qa; q2 < qb; q2++) {
                    const R t2 = cs.tq[q2], c0 = cs.cq[q2];
                    const R x = i < m ? cs.X[i * C::kXS + q2] : R(0);
                    const R ux = wi * x;
                    const bool stage = kJac && (jstride == 1 || ((q2 - qa) & 1) == 0);
                    const float uz = stage ? sm.kq[q2] * (float)ux * z_own : 0.f;
                    const int f0 = stage ? (q2 - qa) / jstride * np : 0;
                    R v0 = R(0), v1 = R(0);
#pragma unroll 4
                    for (int p = ng * pw; p < (ng + 1) * pw; p++) {
                        R er, ei, pr, pi;
                        ld_c(cs.E + 2 * (p * C::MP + i), er, ei);
                        ld_c(cs.P + 2 * (p * C::kQC + q2), pr, pi);
                        const R fx = fma(x, er, R(1)), fy = x * ei;
                        const R inv = recip(fma(fx, fx, fy * fy));
                        // h = E conj(f) / |f|^2
                        const R ix = fx * inv, iy = fy * inv;
                        const R hr = fma(er, ix, ei * iy), hi = fma(ei, ix, -(er * iy));
                        v0 = fma(pr, hr, v0); v1 = fma(-pi, hi, v1);
                        if (kJac && stage) {
                            float sr, si;
                            ld_c(cs.sq + 2 * (p * C::kQC + q2), sr, si);
                            const float a = uz * (float)hr, b = uz * (float)hi;
                            const int f = f0 + p;
                            sm.AS[((f >> 3) * 4 + (f & 3)) * 2 * C::kTS + 2 * i + ((f >> 2) & 1)] =
                                pack_half(fmaf(sr, a, -(si * b)), fmaf(sr, b, si * a));
                        }
                    }
                    const R gi = c0 * ux * (v0 + v1);
                    g += gi;
                    g2 = fma(gi * t2, wi, g2);
                }
            }
            if (kJac) {
                // unused slots of the last MMA depth
                const int tot = nst * np;
                for (int f = tot + ng; f < ((tot + 7) & ~7); f += C::kNG)
                    sm.AS[((f >> 3) * 4 + (f & 3)) * 2 * C::kTS + 2 * i + ((f >> 2) & 1)] = 0u;
                __syncthreads();
                hess_mma<C>(sm, fr, (tot + 7) >> 3);
                __syncthreads();
            }
        }
        if (!kJac) __syncthreads();
    }
    g_out = (double)g; g2_out = (double)g2;
    sum_copies<C>(sm, g_out, g2_out);
}

// Series S of d/dlambda log P -> product series P[0 .. n-1] of one node, handed to put(e, P[e]) (zeros at and beyond n).
template <int NT, typename R, class F>
__device__ __forceinline__ void product_series(const R* S, int n, F put)
{
    R P[NT + 1], acc[NT + 1];
    P[0] = R(1);
#pragma unroll
    for (int c = 1; c <= NT; c++) acc[c] = R(0);
#pragma unroll
    for (int k = 0; k < NT - 1; k++) {
#pragma unroll
        for (int c = k + 1; c < NT; c++) acc[c] = fma(S[c - 1 - k], P[k], acc[c]);
        P[k + 1] = acc[k + 1] * R(1.0 / (k + 1));
    }
#pragma unroll
    for (int e = 0; e < NT; e++) put(e, P[e]);
}

// Gradient g and the Hessian's diagonal part g2 at the weights in shared memory (this thread's in w_own), in fp64.
//   hs = sigma * (draft mass above the block)
// Every token thread (all copies) gets g and g2.
template <class C>
__device__ __forceinline__ void eval_system(const FSm<C>& sm, int m, int n, double hs, int slack, double qstep,
                                            double w_own, double ds_own, double& g_out, double& g2_out)
{
    constexpr int NT = C::NT, T = C::T;
    typedef double R;
    const RSm<C, R> rs(sm);
    const int tid = threadIdx.x, i = tid % C::MP, ng = tid / C::MP;
    const Grid<R> grid(get_extent(sm), slack, qstep);
    const int Q = grid.Q;
    const R wi = w_own, dsi = ds_own;
    R dp[NT <= 8 ? NT + 1 : 1];
    if (NT <= 8) {
        dp[0] = R(1);
#pragma unroll
        for (int c = 1; c <= (NT <= 8 ? NT : 0); c++) dp[c] = dp[c - 1] * dsi;
    }
    R g = R(0), g2 = R(0);
    const bool live = (i & ~31) < m;
#pragma unroll 1
    for (int q0 = 0; q0 < Q; q0 += C::kQC) {
        const int nq = min(C::kQC, Q - q0);
        // ---- S: this thread's share of the tokens at its node
        const int bits = slot_bits(nq), q = tid & ((1 << bits) - 1), G = T >> bits, grp = tid >> bits;
        constexpr int kSS = NT + 2;                                // row stride of the shares: conflict-free vector access
        {
            R t, c0;
            grid.node(q0 + q, slack, t, c0);
            if (tid < nq) { rs.tq[q] = t; rs.cq[q] = c0; }
            R S[NT];
#pragma unroll
            for (int c = 0; c < NT; c++) S[c] = R(0);
            if (q < nq) {
#pragma unroll 2
                for (int j = grp; j < m; j += G) {
                    const R x = Rx<R>::expneg(t * rs.w[j]);
                    const R d = rs.ds[j];
                    const R u = fma(R(-2), x, R(1)), p = fma(-x, x, x);
                    S[0] = fma(x, d, S[0]);
                    R h[NT + 1];
                    if (NT <= 8) {
                        unit_series<NT - 1, R>(u, p, h);
                        R pe[8];                           // p ds^(c+1)
                        const R d2 = d * d, d4 = d2 * d2, pd = p * d;
                        pe[1] = p * d2; pe[2] = pd * d2; pe[3] = p * d4; pe[4] = pd * d4;
                        pe[5] = pe[1] * d4; pe[6] = pe[2] * d4; pe[7] = pe[3] * d4;
#pragma unroll
                        for (int c = 1; c < NT; c++) S[c] = fma(pe[c & 7], h[c], S[c]);
                    } else {
                        const R pd = p * d;
                        riccati_series<NT - 1, R>(d, d * u, pd, h);
#pragma unroll
                        for (int c = 1; c < NT; c++) S[c] = fma(pd, h[c], S[c]);
                    }
                }
            }
            put_shares<NT, R>(S, bits, q < nq, rs.SP + ((tid >> 5) * C::kQC + q) * kSS);
        }
        __syncthreads();
        // ---- P: one thread per node.  PP[j] = P[n - 1 - j], so that PP[c - 1] pairs with h[c] in [lambda^n] P h
        if (tid < nq) {
            R S[NT];
#pragma unroll
            for (int c = 0; c < NT; c++) S[c] = R(0);
#pragma unroll 2
            for (int k = 0; k < C::kW; k++) {
                GR_PTR(const R) row = rs.SP + (k * C::kQC + tid) * kSS;
#pragma unroll
                for (int c = 0; c < NT; c += 2) {
                    R v[2];
                    ld_vec(row + c, v);
                    S[c] += v[0]; S[c + 1] += v[1];
                }
            }
            S[0] += hs;
            GR_PTR(R) row = rs.PP + tid * C::kRow;
            product_series<NT, R>(S, n, [&](int e, R v) { if (e < n) row[n - 1 - e] = v; else row[e] = R(0); });
        }
        __syncthreads();
        // ---- g: one thread per token
        if (live) {
#pragma unroll 2
            for (int q2 = ng; q2 < nq; q2 += C::kNG) {
                const R t = rs.tq[q2], c0 = rs.cq[q2];
                const R x = Rx<R>::expneg(t * wi);
                const R u = fma(R(-2), x, R(1)), p = fma(-x, x, x);
                R h[NT + 1];
                if (NT <= 8) {
                    unit_series<NT, R>(u, p, h);
#pragma unroll
                    for (int c = 1; c <= NT; c++) h[c] *= dp[NT <= 8 ? c : 0];
                } else {
                    riccati_series<NT, R>(dsi, dsi * u, dsi * p, h);
                }
                R pr[NT];
                R v0 = R(0), v1 = R(0);
#pragma unroll
                for (int c = 0; c < NT; c += 2) ld_vec(rs.PP + q2 * C::kRow + c, pr + c);
#pragma unroll
                for (int c = 0; c < NT; c += 2) { v0 = fma(pr[c], h[c + 1], v0); v1 = fma(pr[c + 1], h[c + 2], v1); }
                const R gi = c0 * (wi * x) * (v0 + v1);
                g += gi;
                g2 = fma(gi * t, wi, g2);
            }
        }
        __syncthreads();
    }
    g_out = g; g2_out = g2;
    sum_copies<C>(sm, g_out, g2_out);
}

// The same in fp32, and the Hessian's contraction (fragments fr) from every jstride-th node: the off-diagonal entries
// times z_i z_l, z = rhs^(-1/2) (z_own is this thread's), which keeps the fp16 operands of order one.
// Packed arithmetic: two tokens at a time where a node's series are summed, two nodes (of which both or neither give the
// contraction operands: jstride apart) where a token walks them.  The kernel runs a few warps per scheduler and waits for
// its own results; packed, a wait serves two.  (4096 rows of n = 16, k = 100: 1552 to 1480 us, 64 whole rows of
// 16 ids 70 to 63, headline 163 to 159.)
template <class C>
__device__ __forceinline__ void eval_low(const FSm<C>& sm, int m, int n, float hs, int slack, float qstep, int jstride,
                                         float wi, float dsi, float z_own, double& g_out, double& g2_out, Frags<C>& fr)
{
    constexpr int NT = C::NT, T = C::T, kRow2 = 2 * C::kRow;
    static_assert(C::JC % 2 == 0, "whole pairs of nodes");
    typedef float R;
    const RSm<C, R> rs(sm);
    const int tid = threadIdx.x, i = tid % C::MP, ng = tid / C::MP;
    const Grid<R> grid(get_extent(sm), slack, qstep);
    const int Q = grid.Q;
    F2 dp[NT <= 8 ? NT + 1 : 1];
    if (NT <= 8) {
        float pw = 1.f;
#pragma unroll
        for (int c = 1; c <= (NT <= 8 ? NT : 0); c++) { pw *= dsi; dp[c] = F2(pw); }
    }
    F2 g(0.f), g2(0.f);
#pragma unroll
    for (int s = 0; s < C::kNA; s++) { fr.A[s][0] = fr.A[s][1] = fr.A[s][2] = fr.A[s][3] = 0.f; }
#pragma unroll
    for (int s = 0; s < C::kNB; s++) { fr.B[s][0] = fr.B[s][1] = fr.B[s][2] = fr.B[s][3] = 0.f; }
    // place of a node among the pairs: node 2 p + h of a coarse grid, nodes 4 p + {0, 2} and 4 p + {1, 3} of a full one
    auto place = [&](int q) { return jstride == 1 ? q : (q & ~3) | ((q & 1) << 1) | ((q >> 1) & 1); };
#pragma unroll 1
    for (int q0 = 0; q0 < Q; q0 += C::kQC) {
        const int nq = min(C::kQC, Q - q0), nqp = (nq + 3) & ~3;
        // ---- S: this thread's share of the pairs of tokens at its node
        const int bits = slot_bits(nq), q = tid & ((1 << bits) - 1), G = T >> bits, grp = tid >> bits;
        constexpr int kSS = NT + 4;                                // row stride of the shares: conflict-free vector access
        {
            R t, c0;
            grid.node(q0 + q, slack, t, c0);
            if (tid < nqp) {
                // (places beyond the last node: weight zero)
                const int at = place(tid);
                c0 = tid < nq ? c0 : 0.f;
                rs.tq[at] = tid < nq ? t : 0.f; rs.cq[at] = c0;
                sm.kq[at] = sqrtf((float)jstride * c0 * t);
            }
            F2 S2[NT];
#pragma unroll
            for (int c = 0; c < NT; c++) S2[c] = F2(0.f);
            if (q < nq) {
                // (behind the last token draft masses and weights are zero)
#pragma unroll 2
                for (int j = grp; j < (m + 1) >> 1; j += G) {
                    const float2 wv = ld_f2(rs.w + 2 * j), dv = ld_f2(rs.ds + 2 * j);
                    const F2 x(Rx<R>::expneg(t * wv.x), Rx<R>::expneg(t * wv.y)), d(dv.x, dv.y);
                    const F2 u = fma(F2(-2.f), x, F2(1.f)), p = fma(x * F2(-1.f), x, x);
                    S2[0] = fma(x, d, S2[0]);
                    F2 h[NT + 1];
                    if (NT <= 8) {
                        unit_series<NT - 1, F2>(u, p, h);
                        GR_PTR(const float) ep = sm.E + 16 * j;       // ds^(c+1) of both
#pragma unroll
                        for (int c = 0; c < NT; c += 2) {
                            const float4 ev = ld_f4(ep + 2 * c);
                            if (c > 0) S2[c] = fma(p * F2(ev.x, ev.y), h[c], S2[c]);
                            S2[c + 1] = fma(p * F2(ev.z, ev.w), h[c + 1], S2[c + 1]);
                        }
                    } else {
                        const F2 pd = p * d;
                        riccati_series<NT - 1, F2>(d, d * u, pd, h);
#pragma unroll
                        for (int c = 1; c < NT; c++) S2[c] = fma(pd, h[c], S2[c]);
                    }
                }
            }
            R S[NT];
#pragma unroll
            for (int c = 0; c < NT; c++) S[c] = S2[c].lo() + S2[c].hi();
            put_shares<NT, R>(S, bits, q < nq, rs.SP + ((tid >> 5) * C::kQC + q) * kSS);
        }
        __syncthreads();
        // ---- P: one thread per node.  PP[j] = P[n - 1 - j], so that PP[c - 1] pairs with h[c] in [lambda^n] P h
        if (tid < nqp) {
            const int at = place(tid);
            GR_PTR(R) row = rs.PP + (at >> 1) * kRow2 + (at & 1);
            if (tid < nq) {
                R S[NT];
#pragma unroll
                for (int c = 0; c < NT; c++) S[c] = R(0);
#pragma unroll 2
                for (int k = 0; k < C::kW; k++) {
                    GR_PTR(const R) part = rs.SP + (k * C::kQC + tid) * kSS;
#pragma unroll
                    for (int c = 0; c < NT; c += 4) {
                        R v[4];
                        ld_vec(part + c, v);
#pragma unroll
                        for (int z = 0; z < 4; z++) S[c + z] += v[z];
                    }
                }
                S[0] += hs;
                product_series<NT, R>(S, n, [&](int e, R v) { if (e < n) row[2 * (n - 1 - e)] = v; else row[2 * e] = R(0); });
            } else {
#pragma unroll
                for (int e = 0; e < NT; e++) row[2 * e] = R(0);
            }
        }
        __syncthreads();
        // ---- g: one thread per token; pairs of nodes, those that stage the operands of the contraction first
        auto pair = [&](int at, bool stage, int slot) {
            const float2 tv = ld_f2(rs.tq + 2 * at), cv = ld_f2(rs.cq + 2 * at);
            const F2 x(Rx<R>::expneg(tv.x * wi), Rx<R>::expneg(tv.y * wi));
            const F2 u = fma(F2(-2.f), x, F2(1.f)), p = fma(x * F2(-1.f), x, x);
            F2 h[NT + 1];
            if (NT <= 8) {
                unit_series<NT, F2>(u, p, h);
#pragma unroll
                for (int c = 1; c <= NT; c++) h[c] = h[c] * dp[NT <= 8 ? c : 0];
            } else {
                const F2 ds2(dsi);
                riccati_series<NT, F2>(ds2, ds2 * u, ds2 * p, h);
            }
            F2 pr[NT];
            F2 v0(0.f), v1(0.f);
#pragma unroll
            for (int c = 0; c < NT; c += 2) {
                const float4 v = ld_f4(rs.PP + at * kRow2 + 2 * c);
                pr[c] = F2(v.x, v.y); pr[c + 1] = F2(v.z, v.w);
            }
#pragma unroll
            for (int c = 0; c < NT; c += 2) { v0 = fma(pr[c], h[c + 1], v0); v1 = fma(pr[c + 1], h[c + 2], v1); }
            const F2 ux = x * F2(wi);
            const F2 gi = F2(cv.x, cv.y) * ux * (v0 + v1);
            g = g + gi;
            g2 = fma(gi * F2(tv.x, tv.y), F2(wi), g2);
            if (stage) {
                // A = P h (series), paired as sum_kappa A[n - kappa] h_l[kappa], kappa = 1 .. n - 1; both sides carry the
                // square root of the node's weight and of the token's scale
                const float2 kv = ld_f2(sm.kq + 2 * at);
                const F2 uz = F2(kv.x, kv.y) * ux * F2(z_own);
                // (pair z of a node's series indices: element (z & 3) of its MMA depth, half (z >> 2) of the fragment)
                const int oa = (slot / C::kPack) * 8 * C::kTS + 2 * i, ob = ((slot + 1) / C::kPack) * 8 * C::kTS + 2 * i;
                const int sa = (slot % C::kPack) * (NT / 2), sb = ((slot + 1) % C::kPack) * (NT / 2);
#pragma unroll
                for (int z = 0; z < NT / 2; z++) {
                    F2 a[2];
#pragma unroll
                    for (int y = 0; y < 2; y++) {
                        const int kap = 2 * z + y + 1;
                        F2 v(0.f);
#pragma unroll
                        for (int c = 1; c <= NT - kap; c++) v = fma(h[c], pr[kap + c - 1], v);
                        a[y] = uz * v;
                    }
                    const F2 h0 = uz * h[2 * z + 1], h1 = z == NT / 2 - 1 ? F2(0.f) : uz * h[2 * z + 2];
                    const int fa = sa + z, fb = sb + z;
                    const int ata = oa + (fa & 3) * 2 * C::kTS + (fa >> 2), atb = ob + (fb & 3) * 2 * C::kTS + (fb >> 2);
                    sm.AS[ata] = pack_half(a[0].lo(), a[1].lo()); sm.HS[ata] = pack_half(h0.lo(), h1.lo());
                    sm.AS[atb] = pack_half(a[0].hi(), a[1].hi()); sm.HS[atb] = pack_half(h0.hi(), h1.hi());
                }
            }
        };
        const int staged = ((nq + jstride - 1) / jstride + 1) >> 1;         // pairs of nodes that stage
        if (jstride == 2 && (i & ~31) < m) {
            // (the copies that have one pair less to stage begin)
#pragma unroll 1
            for (int z = C::kNG - 1 - ng; z < nqp >> 2; z += C::kNG) pair(2 * z + 1, false, 0);
        }
#pragma unroll 1
        for (int pa = 0; pa < staged; pa += C::JC / 2) {
            const int np = min(staged - pa, C::JC / 2), nst = 2 * np;
#pragma unroll 1
            for (int z = ng; z < np; z += C::kNG) pair((pa + z) * jstride, true, 2 * z);
            // unused slots of the last MMA depth
            if (C::kPack > 2 && nst % C::kPack != 0) {
                for (int e = nst * (NT / 2) + tid / C::MP; e < (nst + C::kPack - 1) / C::kPack * 8; e += C::kNG) {
                    const int at = (e >> 3) * 8 * C::kTS + 2 * i + (e & 3) * 2 * C::kTS + ((e & 7) >> 2);
                    sm.AS[at] = 0u; sm.HS[at] = 0u;
                }
            }
            __syncthreads();
            hess_mma<C>(sm, fr, (nst + C::kPack - 1) / C::kPack);
            __syncthreads();
        }
    }
    g_out = (double)g.lo() + (double)g.hi(); g2_out = (double)g2.lo() + (double)g2.hi();
    sum_copies<C>(sm, g_out, g2_out);
}

// The fp64 evaluation, kept out of line (it is called once or twice per system, and its registers stay its own).
template <class C>
__device__ __noinline__ double2 eval_fp64(int m, int n, int slack, bool coarse, int* flag)
{
    const FSm<C> sm(flag);
    const int i = threadIdx.x % C::MP;
    const double qstep = sm.scal[SC_QSTEP] * (coarse ? 2.0 : 1.0);
    double2 r;
    if constexpr (C::kContour) { Frags<C> none; eval_contour<C, double, false>(sm, m, slack, qstep, 1, sm.wd[i], 0.f, r.x, r.y, none); }
    else eval_system<C>(sm, m, n, sm.scal[SC_HS], slack, qstep, sm.wd[i], i < m ? sm.dsd[i] : 0.0, r.x, r.y);
    return r;
}

// Float index of row r (>= 8 j) of the j-th 8-column panel.  Within a factored row column c sits at panel_pos(c), so that
// the columns t and t + 4 an MMA fragment needs are adjacent.
template <class C>
__device__ __forceinline__ int panel_row(int j, int r) { return 8 * (C::MP * j - 4 * j * (j - 1)) + (r - 8 * j) * 8; }
__device__ __forceinline__ int panel_pos(int c) { return c < 4 ? 2 * c : 2 * c - 7; }
__device__ __forceinline__ float fast_rsqrt(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
// fp32 value as two tf32 parts (the tensor core drops the low bits of the second)
__device__ __forceinline__ void split_tf32(float x, float& hi, float& lo) {
    hi = __uint_as_float(__float_as_uint(x) & 0xffffe000u);
    lo = x - hi;
}

// Factorisation H = L L^T (fp32) out of the fragments, which hold the contraction: off-diagonal add - fr times sm.wf of row and
// column, diagonal in sm.dg; the forward substitution of sm.yv is carried along (result in sm.dl).  L stays in shared memory for later
// right-hand sides.  The matrix never leaves the fragments as a whole: each 8-column panel is written to shared memory,
// every thread factors the 8 x 8 diagonal block in registers (redundantly: no exchange), one thread per row solves the
// panel below it, and the fragments take the rank-8 update (operands split into two tf32 parts, ~fp32 products).  The
// eight threads of the block's own rows solve for unit vectors instead: they get the inverse of the block's factor,
// which turns the substitutions' 8 x 8 solves into independent dot products (sm.Ld: row i holds column i of the inverse).
// SC_FAIL / SC_PIVOT receive whether a pivot was not positive and the smallest relative pivot.
template <class C>
__device__ __forceinline__ void factor(const FSm<C>& sm, Frags<C>& fr, int m, float add)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const int ra = warp % C::kPr, rb = C::MP / 16 - 1 - ra, cs = warp / C::kPr;
    const int m16 = (m + 15) & ~15;
    // matrix out of the contraction (identity beyond m)
    auto entry = [&](float f, int row, int col) {
        return row == col ? sm.dg[row] : (row < m && col < m ? add - f * sm.wf[row] * sm.wf[col] : 0.f);
    };
#pragma unroll
    for (int s = 0; s < C::kNB; s++) {
        const int ni = cs + s * C::kS;
#pragma unroll
        for (int z = 0; z < 4; z++) {
            const int col = 8 * ni + 2 * tig + (z & 1), r = gid + 8 * (z >> 1);
            if (s < C::kNA) fr.A[s < C::kNA ? s : 0][z] = entry(fr.A[s < C::kNA ? s : 0][z], 16 * ra + r, col);
            fr.B[s][z] = entry(fr.B[s][z], 16 * rb + r, col);
        }
    }
    bool bad = false;
    float pmin = 1.f;
    const int npan = (m + 7) >> 3;
#pragma unroll 1
    for (int j = 0; j < npan; j++) {
        // the panel's columns out of the fragments
        auto put = [&](int rt, const float* v) {
            GR_PTR(float) p = sm.Lp + panel_row<C>(j, 16 * rt + gid) + 2 * tig;
            if (2 * rt >= j) st_f2(p, make_float2(v[0], v[1]));
            st_f2(p + 64, make_float2(v[2], v[3]));               // (eight rows further)
        };
#pragma unroll
        for (int s = 0; s < C::kNB; s++) {
            if (cs + s * C::kS == j) {
                if (s < C::kNA && 2 * ra + 1 >= j) put(ra, fr.A[s < C::kNA ? s : 0]);
                if (2 * rb + 1 >= j && 16 * rb < m16) put(rb, fr.B[s]);
            }
        }
        __syncthreads();
        const int r = 8 * j + tid;
        if (r < m16) {
            float Lb[8][8], yb[8], v[8];
            {
                GR_PTR(const float) p = sm.Lp + panel_row<C>(j, 8 * j);
                GR_PTR(const float) yp = sm.yv + 8 * j;
                GR_PTR(const float) q = sm.Lp + panel_row<C>(j, r);
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const float4 lo = ld_f4(p + 8 * c);
                    Lb[c][0] = lo.x; Lb[c][1] = lo.y; Lb[c][2] = lo.z; Lb[c][3] = lo.w;
                    if (c >= 4) { const float4 hi = ld_f4(p + 8 * c + 4); Lb[c][4] = hi.x; Lb[c][5] = hi.y; Lb[c][6] = hi.z; Lb[c][7] = hi.w; }
                }
                const float4 y0 = ld_f4(yp), y1 = ld_f4(yp + 4), q0 = ld_f4(q), q1 = ld_f4(q + 4);
                yb[0] = y0.x; yb[1] = y0.y; yb[2] = y0.z; yb[3] = y0.w; yb[4] = y1.x; yb[5] = y1.y; yb[6] = y1.z; yb[7] = y1.w;
                v[0] = q0.x; v[1] = q0.y; v[2] = q0.z; v[3] = q0.w; v[4] = q1.x; v[5] = q1.y; v[6] = q1.z; v[7] = q1.w;
            }
            float yi = sm.yv[r];
            if (tid < 8) {
#pragma unroll
                for (int c = 0; c < 8; c++) v[c] = tid == c ? 1.f : 0.f;
                yi = 0.f;
            }
            float piv = 1.f;
#pragma unroll
            for (int c = 0; c < 8; c++) {
                const float dv = Lb[c][c];
                bad = bad || !(dv > 0.f);
                if (tid == c) piv = dv;
                const float di = fast_rsqrt(dv);
#pragma unroll
                for (int r2 = c + 1; r2 < 8; r2++) Lb[r2][c] *= di;
                yb[c] *= di;
                const float lc = v[c] * di;
                v[c] = lc;
#pragma unroll
                for (int c3 = c + 1; c3 < 8; c3++) {
#pragma unroll
                    for (int r2 = c3; r2 < 8; r2++) Lb[r2][c3] = fmaf(-Lb[r2][c], Lb[c3][c], Lb[r2][c3]);
                    v[c3] = fmaf(-lc, Lb[c3][c], v[c3]);
                    yb[c3] = fmaf(-Lb[c3][c], yb[c], yb[c3]);
                }
                yi = fmaf(-lc, yb[c], yi);
            }
            if (tid < 8) {
                // column tid of the inverse factor; the finished right-hand side
                float yo = 0.f;
#pragma unroll
                for (int c = 0; c < 8; c++) if (tid == c) yo = yb[c];
                GR_PTR(float) p = sm.Ld + j * 64 + tid * 8;
                st_f4(p, make_float4(v[0], v[1], v[2], v[3]));
                st_f4(p + 4, make_float4(v[4], v[5], v[6], v[7]));
                sm.dl[r] = yo;
                pmin = fminf(pmin, __fdividef(piv, sm.dg[r]));
            } else {
                sm.yv[r] = yi;
                GR_PTR(float) p = sm.Lp + panel_row<C>(j, r);
                st_f4(p, make_float4(v[0], v[4], v[1], v[5]));
                st_f4(p + 4, make_float4(v[2], v[6], v[3], v[7]));
            }
        }
        __syncthreads();
        // rank-8 update of the tiles to the right (loads first; rows of the diagonal block itself only reach entries above
        // the diagonal)
        const bool onA = 2 * ra + 1 > j && 16 * ra < m, onB = 2 * rb + 1 > j && 16 * rb < m;
        if (onA || onB) {
            float fa[4], fb[4];
            float2 cv[C::kNB];
            auto load_rows = [&](int rt, float* f) {
                GR_PTR(const float) p = sm.Lp + panel_row<C>(j, max(16 * rt, 8 * j) + gid) + 2 * tig;
                const float2 f0 = ld_f2(p), f1 = ld_f2(p + 64);
                f[0] = -f0.x; f[1] = -f1.x; f[2] = -f0.y; f[3] = -f1.y;
            };
#pragma unroll
            for (int s = 0; s < C::kNB; s++)
                cv[s] = ld_f2(sm.Lp + panel_row<C>(j, 8 * max(cs + s * C::kS, j) + gid) + 2 * tig);
            load_rows(ra, fa);
            load_rows(rb, fb);
            {
                float al[4], bl[4], ah[4], bh[4];
#pragma unroll
                for (int z = 0; z < 4; z++) { split_tf32(fa[z], ah[z], al[z]); split_tf32(fb[z], bh[z], bl[z]); }
#pragma unroll
                for (int s = 0; s < C::kNB; s++) {
                    const int ni = cs + s * C::kS;
                    if (ni > j && 8 * ni < m) {
                        float ch[2], cl[2];
                        split_tf32(cv[s].x, ch[0], cl[0]); split_tf32(cv[s].y, ch[1], cl[1]);
                        if (s < C::kNA && onA) {
                            float* x = fr.A[s < C::kNA ? s : 0];
                            mma_tf32(x, al, ch); mma_tf32(x, ah, cl); mma_tf32(x, ah, ch);
                        }
                        if (onB) { mma_tf32(fr.B[s], bl, ch); mma_tf32(fr.B[s], bh, cl); mma_tf32(fr.B[s], bh, ch); }
                    }
                }
            }
        }
        // (the next panel goes to an area of its own: no barrier here)
    }
    if (tid < 32) {
        pmin = fminf(pmin, __shfl_xor_sync(0xffffffffu, pmin, 4));
        pmin = fminf(pmin, __shfl_xor_sync(0xffffffffu, pmin, 2));
        pmin = fminf(pmin, __shfl_xor_sync(0xffffffffu, pmin, 1));
        if (tid == 0) { sm.scal[SC_FAIL] = bad ? 1.0 : 0.0; sm.scal[SC_PIVOT] = (double)pmin; }
    }
}

// Backward substitution L^T x = sm.dl, in place, warp 0: eight unknowns at a time from the last panel up.
template <class C>
__device__ __noinline__ void backward_subst(int m, int* flag)
{
    const FSm<C> sm(flag);
    constexpr int kU = C::MP / 32;
    const int lane = threadIdx.x, e = lane & 7;
    if (lane >= 32) return;
    __syncwarp();
    float y[kU];
#pragma unroll
    for (int u = 0; u < kU; u++) y[u] = lane + 32 * u < m ? sm.dl[lane + 32 * u] : 0.f;
    __syncwarp();
#pragma unroll 1
    for (int j = (m - 1) >> 3; j >= 0; j--) {
        // x = (inverse of the diagonal block)^T y: lane e of every octet forms x_e = sum_c Ld[e][c] y_c
        float li[8], l[kU][8];
        {
            GR_PTR(const float) p = sm.Ld + 64 * j + 8 * e;
            const float4 lo = ld_f4(p), hi = ld_f4(p + 4);
            li[0] = lo.x; li[1] = lo.y; li[2] = lo.z; li[3] = lo.w; li[4] = hi.x; li[5] = hi.y; li[6] = hi.z; li[7] = hi.w;
        }
#pragma unroll
        for (int u = 0; u < kU; u++) {
            // rows 8 j .. 8 j + 7 of this lane's column (rows of its own diagonal block are not used)
            const int c = lane + 32 * u, pj = min(c >> 3, j);
            GR_PTR(const float) p = sm.Lp + panel_row<C>(pj, 8 * j) + panel_pos(c & 7);
#pragma unroll
            for (int z = 0; z < 8; z++) l[u][z] = p[8 * z];
        }
        float src = y[0];
#pragma unroll
        for (int u = 1; u < kU; u++) if ((8 * j) >> 5 == u) src = y[u];
        float x0 = 0.f, x1 = 0.f;
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
            x0 = fmaf(li[c], __shfl_sync(0xffffffffu, src, (8 * j + c) & 31), x0);
            x1 = fmaf(li[c + 1], __shfl_sync(0xffffffffu, src, (8 * j + c + 1) & 31), x1);
        }
        const float x = x0 + x1;
        if (lane < 8) sm.dl[8 * j + lane] = x;
        float a[kU], b[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) { a[u] = 0.f; b[u] = 0.f; }
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
            const float xa = __shfl_sync(0xffffffffu, x, c), xb = __shfl_sync(0xffffffffu, x, c + 1);
#pragma unroll
            for (int u = 0; u < kU; u++) { a[u] = fmaf(l[u][c], xa, a[u]); b[u] = fmaf(l[u][c + 1], xb, b[u]); }
        }
#pragma unroll
        for (int u = 0; u < kU; u++) if (lane + 32 * u < 8 * j) y[u] -= a[u] + b[u];
    }
}

// Right-hand side of the Newton system.  Along its own coordinate a token's flow behaves like a logistic curve
// g_i = c sigma(alpha_i - kappa): linear in w_i while the token is light, saturating at the flow c of the tuples it can win
// at all once it is heavy.  The curve through the current value and slope (H_ii = g_i (1 - g_i / c) gives c = g_i^2 / g2_i)
// is inverted exactly: H_ii (logit(rhs_i / c) - logit(g_i / c)) replaces rhs_i - g_i.  Near the solution the two agree to
// first order; far from it a token close to saturation is placed at once, and a light one gets the multiplicative
// update log(rhs_i / g_i).  A target at or beyond the saturation level says that the curve is off: plain residual.
__device__ __forceinline__ float newton_rhs(double g, double g2, double r)
{
    const float gf = (float)g, diff = (float)(r - g), hii = (float)(g - g2);
    const float room = 1.f - __fdividef((float)r * __fdividef((float)g2, gf), gf);
    const float arg = fmaxf(__fdividef(diff, gf * fmaxf(room, 1e-3f)), -0.999999f);
    return room > 1e-3f ? hii * (fabsf(arg) < 0.01f ? arg * fmaf(arg, fmaf(arg, 1.f / 3.f, -0.5f), 1.f) : __logf(1.f + arg)) : diff;
}

// Matrix-vector products with the half-precision matrices in sm.pi: thread t has row t / kNG and the (t % kNG)-th share of its
// columns, so that the shares of a row meet in neighbouring lanes and not through shared memory.  The vector's shares are four
// floats apart (their loads fall into different banks); three buffers behind what sum_copies uses.
template <class C, int kNG = C::kNG> __device__ __forceinline__ int vec_pos(int i) { return i + 4 * (i / (C::MP / kNG)); }
template <class C>
__device__ __forceinline__ GR_PTR(float) vec_buffer(const FSm<C>& sm, int which)
{
    constexpr int kLen = C::MP + 4 * C::kNG;
    static_assert(C::T * 16 + 3 * kLen * 4 <= C::kSPBytes, "vector buffers");
    return GR_MKPTR(float, reinterpret_cast<float*>(sm.base + C::oSP + C::T * 16) + which * kLen, kLen, sm.flag);
}
template <int kNG>
__device__ __forceinline__ float share_sum(float v)
{
    __syncwarp();
#pragma unroll
    for (int o = 1; o < kNG; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <class C, int kNG>
__device__ __forceinline__ void load_row(GR_PTR(const __half) mat, float* row)
{
    constexpr int kCol = C::MP / kNG;
    GR_PTR(const __half) np = mat + (threadIdx.x / kNG) * C::kNS + (threadIdx.x % kNG) * kCol;
#pragma unroll
    for (int c = 0; c < kCol; c += 8) {
        const uint4 v = ld_h8(np + c);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int z = 0; z < 4; z++) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[z]));
            row[c + 2 * z] = f.x; row[c + 2 * z + 1] = f.y;
        }
    }
}
template <class C, int kNG>
__device__ __forceinline__ float dot_row(const float* row, GR_PTR(const float) vec)
{
    constexpr int kCol = C::MP / kNG;
    GR_PTR(const float) vp = vec + (threadIdx.x % kNG) * (kCol + 4);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int c = 0; c < kCol; c += 4) {
        const float4 v = ld_f4(vp + c);
        a0 = fmaf(row[c], v.x, a0); a1 = fmaf(row[c + 1], v.y, a1); a2 = fmaf(row[c + 2], v.z, a2); a3 = fmaf(row[c + 3], v.w, a3);
    }
    return share_sum<kNG>((a0 + a1) + (a2 + a3));
}
template <class C>
__device__ __forceinline__ float row_times(GR_PTR(const __half) mat, GR_PTR(const float) vec)
{
    float row[C::MP / C::kNG];
    load_row<C, C::kNG>(mat, row);
    return dot_row<C, C::kNG>(row, vec);
}

template <class C> __device__ __forceinline__ float rs_ds(const FSm<C>& sm, int i) { return RSm<C, float>(sm).ds[i]; }

// fp32 evaluation at one point and what the Newton step needs from it, out of line (its registers, fragments included, stay
// its own).  Default: the Hessian scaled to unit diagonal, I - N with N_il = H_il / sqrt(H_ii H_ll), N in half precision
// (its error, 2^-11, is that of the contraction's operands) for cg_solve below; sm.dg receives 1 / sqrt(H_ii).
// With `chol` a Cholesky factorisation instead, for systems conjugate gradients do not get through.  `given`: the gradient
// and the diagonal part come from the caller, in fp64.
template <class C>
__device__ __noinline__ double2 eval_hessian(int m, int n, int slack, bool coarse, bool given, bool chol,
                                             double2 gg, int* flag)
{
    const FSm<C> sm(flag);
    const int tid = threadIdx.x, i = tid % C::MP, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
    Frags<C> fr;
    double g, g2;
    const double qstep = sm.scal[SC_QSTEP] * (coarse ? 2.0 : 1.0);
    // (a table's nodes all serve the Hessian, of the full trapezoid grid every other one)
    const int jstride = coarse || get_extent(sm).nodes > 0 ? 1 : 2;
    const double rhs = i < m ? sm.rhs[sm.ord[i]] : 0.0;
    const float zr = i < m ? (float)rhs : 1.f, zi = rsqrtf(zr);
    if constexpr (C::kContour) eval_contour<C, float, true>(sm, m, slack, qstep, jstride, sm.wd[i], i < m ? zi : 0.f, g, g2, fr);
    else eval_low<C>(sm, m, n, (float)sm.scal[SC_HS], slack, (float)qstep, jstride, sm.wf[i], i < m ? rs_ds<C>(sm, i) : 0.f, i < m ? zi : 0.f, g, g2, fr);
    if (given) { g = gg.x; g2 = gg.y; }
    if (chol) {
        // an outer block's function is constant along (1,...,1): that direction is pinned with 1/m everywhere
        const float add = slack ? 0.f : 1.f / (float)m;
        if (tid < C::MP) {
            sm.yv[i] = i < m ? newton_rhs(g, g2, rhs) : 0.f;
            sm.dg[i] = i < m ? (float)(g - g2) + add : 1.f;
            sm.wf[i] = zr * zi;                                // undoes the operands' scale
        }
        __syncthreads();
        factor<C>(sm, fr, m, add);
    } else {
        // (a diagonal that is not positive gives NaN, which the solve reports)
        GR_PTR(float) vec = vec_buffer(sm, 0);
        if (tid < C::MP) {
            const float rd = i < m ? rsqrtf((float)(g - g2)) : 1.f;
            sm.dg[i] = rd;
            sm.wf[i] = zr * zi * rd;
            vec[vec_pos<C>(i)] = i < m ? __fdividef(1.f, rd) : 0.f;
        }
        __syncthreads();
        const int ra = warp % C::kPr, rb = C::MP / 16 - 1 - ra, cs = warp / C::kPr;
        GR_PTR(__half) N = sm.pi;
        // Both triangles out of the fragments' lower one: an entry and its mirror image.  (Storing one triangle and reading the
        // other out of its columns afterwards took a barrier and twice the time.)
        auto put = [&](const float* v, int rt, int ni) {
            const int c0 = 8 * ni + 2 * tig, r0 = 16 * rt + gid;
            const float2 sc = ld_f2(sm.wf + c0);
            const float s0 = sm.wf[r0], s1 = sm.wf[r0 + 8];
            const float e[4] = {v[0] * s0 * sc.x, v[1] * s0 * sc.y, v[2] * s1 * sc.x, v[3] * s1 * sc.y};
#pragma unroll
            for (int z = 0; z < 2; z++) {
                const int r = r0 + 8 * z;                       // (eight rows further)
                const uint32_t h = pack_half(e[2 * z], e[2 * z + 1]);
                if (ni < 2 * rt) st_h2(N + r * C::kNS + c0, h);
                else {
                    // a tile on the diagonal: what lies above belongs to the mirror images, the diagonal itself is zero
                    if (c0 < r) N[r * C::kNS + c0] = __ushort_as_half((unsigned short)h);
                    if (c0 + 1 < r) N[r * C::kNS + c0 + 1] = __ushort_as_half((unsigned short)(h >> 16));
                    if (c0 == r || c0 + 1 == r) N[r * C::kNS + r] = __ushort_as_half((unsigned short)0);
                }
                if (c0 < r) N[c0 * C::kNS + r] = __ushort_as_half((unsigned short)h);
                if (c0 + 1 < r) N[(c0 + 1) * C::kNS + r] = __ushort_as_half((unsigned short)(h >> 16));
            }
        };
#pragma unroll
        for (int s = 0; s < C::kNB; s++) {
            const int ni = cs + s * C::kS;
            if (s < C::kNA && ni <= 2 * ra + 1) put(fr.A[s < C::kNA ? s : 0], ra, ni);
            if (ni <= 2 * rb + 1) put(fr.B[s], rb, ni);
        }
        __syncthreads();
        // row sums of |H| less the diagonal, for the diagonal that cg_solve sets
        const float nrow = row_times<C>(N, vec);
        if (tid % C::kNG == 0) sm.Ld[tid / C::kNG] = nrow;
    }
    double2 r; r.x = g; r.y = g2;
    return r;
}

// Newton step by conjugate gradients on the scaled Hessian; the step of token i is left in sm.yv[i], NaN when the residual did
// not fall by `rtol` in kFCgMax iterations.  Off the heavy-weight regime the scaled Hessian has all its eigenvalues
// within 0.8 - 1.5 but one, so four or five iterations give four digits.
// One thread per row (or share of a row), the row in registers; the pipelined form of the method (Ghysels and Vanroose), in which
// the scalar products of an iteration do not wait for its matrix product: one barrier each, where Chronopoulos and Gear's form
// with the shares summed through shared memory had three.  (50 tokens to 2e-4, one CTA alone: 3.7 k cycles.)
// The step's product with s, which goes into the common scale, is summed once at the end: carried along by the recurrences it drifts
// with them, and saves nothing (64 whole rows of 16 ids 94 us a call with the recurrence, 89 with the sum; 256 rows of n = 4, k = 8 58.0, 56.9).
// The one eigenvalue is the common scale of the weights, the direction (1,...,1): H 1 = s, s_i = g2_i / w_i the rate at
// which token i takes mass from the slack, tiny when the acceptance is close to one.  s is known exactly, so the diagonal
// is set from the row sums (sm.Ld), s_i + sum_l |H_il| (whatever the rounding of the off-diagonal part, the matrix then has the
// right action on that direction), and the direction itself is deflated: the iteration works on
// (I - s 1^T / sum s) H, and the step gets `shift`, the caller's answer for the common scale, less s . y / sum s.
// (kap = -1 / sum s, lin = sum rhs / sum s.)
// An outer block (slack == 0) has s = 0: the matrix is singular along the direction, e e^T / (e . e) is added, e = sqrt(H_ii)
// (kap = 1 / (e . e), lin = 0).
// Up to 32 tokens one warp does it all, a row per lane: its sums need no barrier and no shared memory, and an iteration takes half the
// time (64 whole rows of 16 ids, a call: 70.7 -> 67.7 us; 256 rows of n = 4, k = 8: 55.4 -> 54.0).
// In: sm.yv right-hand side, sm.dl s, visible to all.
template <class C>
__device__ __noinline__ void cg_solve(int m, int slack, float kap, float lin, float shift, float rtol, int* flag)
{
    constexpr bool kOne = C::MP == 32;                          // one warp
    constexpr int kNG = kOne ? 1 : C::kNG, kW = kOne ? 1 : C::kW, kCol = C::MP / kNG;       // copies, warps, columns of a share
    const FSm<C> sm(flag);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, i = tid / kNG;
    if (kOne && warp > 0) { __syncthreads(); return; }
    const bool on = i < m, lead = tid % kNG == 0;
    const float sd = sm.dg[i], rhs = sm.yv[i];
    float row[kCol];
    load_row<C, kNG>(sm.pi, row);
    // diagonal from the row sums; v: the deflated (slack) or added (outer block) direction, kap its factor
    const float si = on && slack ? sm.dl[i] : 0.f;
    const float diag = on ? sd * fmaf(si, sd, sm.Ld[i]) : 1.f;
    const float v = slack ? si * sd : (on ? __fdividef(1.f, sd) : 0.f);
    float r = on ? fmaf(-lin, v, rhs * sd) : 0.f, x = 0.f, p = 0.f, s = 0.f, z = 0.f, w = 0.f;
    // (1 / r.r of the last iteration and that times 1 / al: formed behind it, off the chain)
    float inv = 0.f, inva = 0.f, goal = 0.f;
    int it;
    bool done = false;
    // (the quadrature nodes' arrays, which only evaluations use, take the warps' sums: tok_reduce's may still be read)
    static_assert(2 * C::kW * 16 <= 2 * C::kQC * 8, "warp sums");
    GR_PTR(float) sums = GR_MKPTR(float, reinterpret_cast<float*>(sm.base + C::oTq), 4 * C::kQC, flag);
    // Sums over the rows.  The lanes that share a row hold the same numbers: each takes one of the three.
    auto row_sums = [&](float* d, GR_PTR(float) part) {
        __syncwarp();
        if constexpr (kNG >= 4) {
            float a = (lane & 3) == 0 ? d[0] : (lane & 3) == 1 ? d[1] : d[2];
#pragma unroll
            for (int o = kNG; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane < 3) part[4 * warp + lane] = a;
        } else if constexpr (kNG == 2) {
            float a = lane & 1 ? d[1] : d[0], b = d[2];
#pragma unroll
            for (int o = kNG; o < 32; o <<= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); b += __shfl_xor_sync(0xffffffffu, b, o); }
            if (lane < 2) part[4 * warp + lane] = a;
            if (lane == 0) part[4 * warp + 2] = b;
        } else {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int k = 0; k < 3; k++) d[k] += __shfl_xor_sync(0xffffffffu, d[k], o);
            }
            if (!kOne && lane == 0) st_f4(part + 4 * warp, make_float4(d[0], d[1], d[2], 0.f));
        }
    };
#pragma unroll 1
    for (it = -1; it <= kFCgMax; it++) {
        // products r.r, w.r, v.w (the first time only v.r) over the rows, and w (r) for the matrix product
        GR_PTR(float) vec = vec_buffer(sm, it & 1);
        const float in = it < 0 ? r : w;
        if (lead) vec[vec_pos<C, kNG>(i)] = in;
        float d[3] = {r * r, w * r, v * in};
        GR_PTR(float) part = sums + 4 * C::kW * (it & 1);
        row_sums(d, part);
        if constexpr (!kOne) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kW; u++) {
                const float4 t = ld_f4(part + 4 * u);
                const float tv[3] = {t.x, t.y, t.z};
#pragma unroll
                for (int k = 0; k < 3; k++) d[k] = u == 0 ? tv[k] : d[k] + tv[k];
            }
        }
        const float q = fmaf(v, kap * d[2], fmaf(diag, in, -dot_row<C, kNG>(row, vec)));
        if (it < 0) { w = q; continue; }
        const float gam = d[0];
        if (it == 0) goal = gam * rtol * rtol;
        if (gam <= goal) { done = true; break; }
        const float beta = gam * inv, den = fmaf(-beta * gam, inva, d[1]), al = __fdividef(gam, den);
        z = fmaf(beta, z, q); s = fmaf(beta, s, w); p = fmaf(beta, p, r);
        x = fmaf(al, p, x); r = fmaf(-al, s, r); w = fmaf(-al, z, w);
        inv = __fdividef(1.f, gam); inva = den * inv;
    }
    float y = x * sd;
    if (slack) {
        // the step's product with the direction, from the step itself: it decides where the common scale ends
        float t = v * x;
#pragma unroll
        for (int o = kNG; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if constexpr (!kOne) {
            GR_PTR(float) part = sums + 4 * C::kW * ((it + 1) & 1);
            if (lane == 0) part[warp] = t;
            __syncthreads();
            t = 0.f;
#pragma unroll
            for (int u = 0; u < kW; u++) t += part[u];
        }
        y += shift + kap * t;
    }
    // (not positive definite, NaN or slow: NaN)
    if (lead) sm.yv[i] = done ? y : __int_as_float(0x7fc00000);
    if (kOne || C::kNG > 1) __syncthreads();
}

// Starting point (log-weights, left in sm.yv): token i wins the share w_i / (slack + w_i + S_i) of the tuples that contain it, S_i = the
// weight it is up against.  A competitor j, present with probability pi_ij = Pr[i and j drafted] / Pr[i drafted],
// adds to S_i the weight e_j for which 1 / (A + e_j) = (1 - pi_ij) / A + pi_ij / (A + w_j), A = slack + w_i + S_i:
// e_j = A pi_ij / (A / w_j + 1 - pi_ij).  For w_j << A this is the mean-field value pi_ij w_j; a huge w_j counts for
// A pi_ij / (1 - pi_ij) only (token i simply loses the tuples that contain j).  fp32: it is a starting point.
// Rows and shares of columns as in the matrix products above (one barrier a sweep; three before).
template <class C>
__device__ __noinline__ void start_point(int m, int slack, int n, double Tm, int* flag)
{
    constexpr int kCol = C::MP / C::kNG;
    const FSm<C> sm(flag);
    const int tid = threadIdx.x, i = tid / C::kNG, share = tid % C::kNG;
    const bool on = i < m, lead = share == 0;
    const int pos = on ? sm.ord[i] : 0;
    const double rhs_i = on ? sm.rhs[pos] : 0.0, d_i = on ? sm.d[pos] : 0.0;
    // masses relative to the system's total: token avoided / a pair avoided, (1 - d_i / T)^n and (1 - (d_i + d_j) / T)^n
    const double iT = m_div(1.0, Tm);
    const float rel = (float)(d_i * iT);
    const double col_d = on ? ipow(fmax(1.0 - d_i * iT, 0.0), n) : 0.0;
    const float col = (float)col_d, ci = on ? (float)(1.0 - col_d) : 1.f, ic = __fdividef(1.f, ci);   // ci: Pr[token i drafted]
    const float rho = on ? fminf((float)(rhs_i * ipow(iT, n)) * ic, 0.999f) : 0.5f;
    const float odds = __fdividef(rho, 1.f - rho);
    float wi = slack ? odds : (on ? __fdividef((float)rhs_i, (float)d_i) : 1.f);
    // a rarely drafted token: Pr[j drafted | i drafted] tends to 1 - (1 - d_j / T)^(n - 1)
    const bool rare = ci < 0.02f;
    const float pres = 1.f - (rel < 1.f ? __fdividef(col, 1.f - rel) : 0.f);
    // (the table behind the vectors: masses, probabilities of being avoided, presences of a rare token's competitors.  Behind the last token:
    // avoided for certain, and an inverse weight that leaves nothing)
    GR_PTR(float) tab = GR_MKPTR(float, reinterpret_cast<float*>(sm.base + C::oPP), 3 * C::MP, sm.flag);
    static_assert(3 * C::MP * 4 <= C::kPPBytes + C::T * 16, "start table");
    // (bounds within which the product of two denominators below neither overflows nor vanishes)
    auto inverse = [&](float w) { return on ? fminf(fmaxf(__fdividef(1.f, w), 1e-18f), 1e15f) : 1e15f; };
    if (lead) { tab[i] = rel; tab[C::MP + i] = on ? col : 1.f; tab[2 * C::MP + i] = on ? pres : 0.f; vec_buffer(sm, 0)[vec_pos<C>(i)] = inverse(wi); }
    __syncthreads();
    // (eight columns at a time: their chains overlap, pairs of them in packed arithmetic.  A share of up to 32 columns stays in registers)
    constexpr bool kRegs = kCol <= 32;
    const int nc = (min(kCol, max(0, m - share * kCol)) + 7) >> 3;
    GR_PTR(__half) prow = sm.pi + i * C::kNS + share * kCol;
    F2 preg[kRegs ? kCol / 2 : 1];
    const F2 avoid(1.f - rel), nrel(-1.f);
    const float own = (1.f - col) * ic;
    auto presence = [&](int c, F2* o) {
        GR_PTR(const float) tp = tab + share * kCol + 8 * c;
        F2 x[4], b[4];
#pragma unroll
        for (int z = 0; z < 8; z += 4) {
            const float4 v = ld_f4(tp + z);
            x[z / 2] = fma(F2(v.x, v.y), nrel, avoid); x[z / 2 + 1] = fma(F2(v.z, v.w), nrel, avoid);
        }
        // both avoided: x^n
#pragma unroll
        for (int z = 0; z < 4; z++) b[z] = F2(1.f);
#pragma unroll 1
        for (int e = n; e > 0; e >>= 1) {
#pragma unroll
            for (int z = 0; z < 4; z++) { if (e & 1) b[z] = b[z] * x[z]; x[z] = x[z] * x[z]; }
        }
#pragma unroll
        for (int z = 0; z < 8; z += 4) {
            const float4 v = ld_f4(tp + C::MP + z), r = ld_f4(tp + 2 * C::MP + z);
            const F2 d0 = b[z / 2] - F2(v.x, v.y), d1 = b[z / 2 + 1] - F2(v.z, v.w);
            const float p[4] = {__saturatef(fmaf(d0.lo(), ic, own)), __saturatef(fmaf(d0.hi(), ic, own)),
                                __saturatef(fmaf(d1.lo(), ic, own)), __saturatef(fmaf(d1.hi(), ic, own))};
            const float q[4] = {r.x, r.y, r.z, r.w};
            float u[4];
#pragma unroll
            for (int y = 0; y < 4; y++) u[y] = share * kCol + 8 * c + z + y == i ? 0.f : rare ? q[y] : p[y];
            o[z / 2] = F2(u[0], u[1]); o[z / 2 + 1] = F2(u[2], u[3]);
        }
    };
    if constexpr (kRegs) {
#pragma unroll
        for (int c = 0; c < kCol / 2; c++) preg[c] = F2(0.f);
#pragma unroll
        for (int c = 0; c < kCol / 8; c++) if (c < nc) presence(c, preg + 4 * c);
    } else if (on) {
#pragma unroll 1
        for (int c = 0; c < nc; c++) {
            F2 o[4];
            presence(c, o);
            st_h8(prow + 8 * c, make_uint4(pack_half(o[0].lo(), o[0].hi()), pack_half(o[1].lo(), o[1].hi()), pack_half(o[2].lo(), o[2].hi()), pack_half(o[3].lo(), o[3].hi())));
        }
    }
    // (a thread reads back what it wrote)
    float A = (slack ? 1.f : 0.f) + wi;
    constexpr int sweeps = C::kSweeps;
#pragma unroll 1
    for (int sweep = 0; sweep < sweeps; sweep++) {
        // e_j / A = p / (1 / w_j + (1 - p) / A), two competitors to a reciprocal
        GR_PTR(const float) inv = vec_buffer(sm, sweep & 1) + share * (kCol + 4);
        const F2 invA(fminf(__fdividef(1.f, A), 1e15f));
        float acc[2] = {0.f, 0.f};
        auto group = [&](int c, const F2* pv) {
            const float4 w0 = ld_f4(inv + 8 * c), w1 = ld_f4(inv + 8 * c + 4);
            const F2 wv[4] = {F2(w0.x, w0.y), F2(w0.z, w0.w), F2(w1.x, w1.y), F2(w1.z, w1.w)};
#pragma unroll
            for (int z = 0; z < 4; z++) {
                const F2 b = fma(F2(1.f) - pv[z], invA, wv[z]);
                acc[z & 1] = fmaf(fmaf(pv[z].lo(), b.hi(), pv[z].hi() * b.lo()), __fdividef(1.f, b.lo() * b.hi()), acc[z & 1]);
            }
        };
        if constexpr (kRegs) {
#pragma unroll
            for (int c = 0; c < kCol / 8; c++) if (c < nc) group(c, preg + 4 * c);
        } else if (on) {
#pragma unroll 2
            for (int c = 0; c < nc; c++) {
                const uint4 pk = ld_h8(prow + 8 * c);
                const uint32_t u[4] = {pk.x, pk.y, pk.z, pk.w};
                F2 pv[4];
#pragma unroll
                for (int z = 0; z < 4; z++) {
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&u[z]));
                    pv[z] = F2(f.x, f.y);
                }
                group(c, pv);
            }
        }
        const float Si = share_sum<C::kNG>(acc[0] + acc[1]);
        if (on) {
            wi = odds * (slack ? 1.f + Si : fmaxf(Si, 1e-30f));
            A = (slack ? 1.f : 0.f) + wi + Si;
        }
        if (sweep + 1 < sweeps) {
            if (lead) vec_buffer(sm, (sweep + 1) & 1)[vec_pos<C>(i)] = inverse(wi);
            __syncthreads();
        }
    }
    if (lead) sm.yv[i] = on ? __logf(wi) : 0.f;
    __syncthreads();
}

// Newton iteration for one system.  Returns the status; sm.wd receives exp(alpha) at the last accepted point, the scalars the
// gradient norm and the number of evaluations.  Out of line, with what it does not change in shared memory: inlined into the
// kernel it had 600 to 1000 bytes of spills, which did not fit the first-level cache beside the shared memory and cost
// more than the evaluations' arithmetic (the same scalar code took three times as long as in the variant without them).
template <class C>
__device__ __noinline__ int fast_system(int m, int slack, int n, double hmass, int max_iters,
                                        const typename CircleOf<C::kContour>::type& circle, int* flag)
{
    const FSm<C> sm(flag);
    const int tid = threadIdx.x, i = tid % C::MP;
    const bool on = i < m, lead = tid < C::MP;
    int par = 0;
    float t0;                // the slack's share of the mass at the solution
    bool dominant;           // one token has most of the mass
    {
    const int pos = on ? sm.ord[i] : 0;
    const double d_i = on ? sm.d[pos] : 0.0, ds_i = d_i * sm.scal[SC_SIGMA];
    double tot[2] = {d_i, on ? sm.rhs[pos] : 0.0};
    tok_reduce<C, 2, 0, 0>(sm, tot, nullptr, nullptr, par);
    const double Tm = tot[0] + hmass;
    // mass of the tuples the system serves
    const double Tn = ipow(Tm, n);
    t0 = slack ? (float)(Tn - tot[1]) : 0.f;
    dominant = !(sm.d[sm.ord[m - 1]] < 0.6 * Tm);       // (ascending draft mass: the last is the largest)
    if (tid == 0) { sm.scal[SC_HS] = hmass * sm.scal[SC_SIGMA]; sm.scal[SC_TN] = Tn; }

    start_point<C>(m, slack, n, Tm, sm.flag);
    // scaled draft masses (and at short series their powers) for the evaluations
    if constexpr (C::kContour) {
        const double iT = m_div(1.0, Tm);
        contour_tables<C>(circle, m, d_i * iT, hmass * iT, Tn, sm.flag);
    } else if (lead) {
        sm.dsd[i] = ds_i;
        RSm<C, float> rs(sm);
        rs.ds[i] = (float)ds_i;
        if (C::NT <= 8) {
            float pw = (float)ds_i;
            const float f = pw;
#pragma unroll
            for (int c = 0; c < 8; c++) { sm.E[16 * (i >> 1) + 2 * c + (i & 1)] = pw; pw *= f; }     // (two tokens side by side)
        }
    }

    }
    // (the tokens' own numbers: the warps of their copies leave them out, where a reduction hands them the results)
    const bool act = on && (C::kTW == 1 || lead);
    double alpha = act ? (double)sm.yv[i] : 0.0;
    if (!slack) {
        const double mean = tok_sum<C>(sm, alpha, par) / (double)m;
        if (act) alpha -= mean;
    }
    alpha = fmin(fmax(alpha, -kFAlphaClamp), kFAlphaClamp);
    double alpha_prev = alpha;
    int status = GR_NOT_CONVERGED, it = 0, stalls = 0, was_kind = -1;
    double rn = 0.0;
    // (what steers the iteration only is fp32: it is compared with margins of three and more, and in fp64 cost 1 % at series of 16)
    float rprev = kFNone, lam = 1.f, dist = 0.f;
    bool ranged = false;                     // the extent of the weights is known for this point
    // Three modes.  Low: gradient and Hessian in fp32, conjugate gradients.  Chord: fp64 gradient, the last Hessian.  High:
    // fp64 gradient, fp32 Hessian of the same point, with `chol` a Cholesky factorisation.  A single token that dominates a
    // long series (its terms would cancel in fp32) starts in the last mode.
    enum { kLow, kChord, kHigh };
    int mode = (C::NT <= 8 || C::kContour || !dominant) ? kLow : kHigh;
    bool full_grid = false, predicted = false, chol = false;
#pragma unroll 1
    for (; it < max_iters; it++) {
        const double w_i = !act ? 0.0 : (mode == kLow ? (double)__expf((float)alpha) : m_exp(alpha));
        if (lead) { sm.wd[i] = w_i; sm.wf[i] = (float)w_i; }
        if (!ranged) {
            unsigned top[2] = {act ? fkey((float)alpha) : 0u, act ? fkey(-(float)alpha) : 0u};
            float wsum = act ? Rx<float>::ex((float)alpha) : 0.f;
            tok_reduce<C, 0, 1, 2>(sm, nullptr, &wsum, top, par);
            if (tid == 0) put_extent(sm, fkey_inv(top[0]), -fkey_inv(top[1]), wsum, n, slack);
        }
        ranged = false;
        __syncthreads();
        // On the trapezoid rule the step is doubled far from the solution (quadrature error ~1e-4, far below the gradient norm
        // there): half the nodes, every one of them a Hessian node.  Convergence is only declared on the full grid.
        const bool coarse = rprev > kFCoarse && !full_grid && mode != kChord && get_extent(sm).nodes == 0;
        const int kind = 2 * mode + (coarse ? 1 : 0);
        double2 gg = make_double2(0.0, 0.0);
        if (mode != kLow) gg = eval_fp64<C>(m, n, slack, coarse, sm.flag);
        if (mode == kHigh) __syncthreads();          // (sum_copies' array)
        if (mode != kChord)
            gg = eval_hessian<C>(m, n, slack, coarse, mode == kHigh, chol, gg, sm.flag);
        const double g = gg.x, g2 = gg.y, rhs_i = act ? sm.rhs[sm.ord[i]] : 0.0, tol = sm.scal[SC_TOL];
        // The residual, and what the step below needs of the tokens: right-hand side b of the Newton system, s_i = g2_i / w_i,
        // and the sums of b, s and the Hessian's diagonal.
        const float b = act ? newton_rhs(g, g2, rhs_i) : 0.f, s_i = act ? __fdividef((float)g2, (float)sm.wd[i]) : 0.f;
        if (!chol && lead) { sm.yv[i] = b; sm.dl[i] = s_i; }
        double rg[2] = {act ? g : 0.0, act ? fabs(g - rhs_i) : 0.0};
        float sums[3] = {b, slack ? s_i : 0.f, act ? (float)(g - g2) : 0.f};
        tok_reduce<C, 2, 3, 0>(sm, rg, sums, nullptr, par);
        if (C::kTW == 1) __syncthreads();
        rn = rg[1];
        // (residuals are only compared within one grid and one precision)
        const bool comparable = kind == was_kind && it > 0;
        was_kind = kind;
        // Stop on an evaluated residual.  (An fp32 evaluation by the fine sums or on the full grid is good to ~1e-6, where a dominant token's terms
        // cancel to 4e-5: enough to see a tolerance of 1e-4 and more met.  Between half the tolerance and the tolerance one more step, which costs a tenth of an
        // evaluation, leaves a residual far below it, unless steps have stopped helping.)
        if (rn <= tol && !coarse && (mode != kLow || tol >= kFLowEnds) && (rn <= 0.5 * tol || (comparable && rn > 0.5 * rprev))) {
            status = GR_OK; it++;
            break;
        }
        bool high = false;               // the same point again with an fp64 gradient on the full grid
        if (mode == kChord) {
            // the reused Hessian no longer serves: one of its own from here on
            high = !(rn <= 1.0e-3) || (comparable && !(rn < 0.3 * rprev));
        } else if (comparable && !(rn < rprev)) {
            if (mode == kLow && rn < kFLowFloor) high = true;          // at the noise of fp32
            else if (lam > 1.f / 64.f) {
                // the last step did not reduce the gradient norm: retry it at half length
                lam *= 0.5f;
                alpha = alpha_prev + 0.5 * (alpha - alpha_prev);
                continue;
            } else if (mode == kLow) {
                high = true; alpha = alpha_prev;
            } else {
                // A step that did not reduce the residual even at 1/64 of its length: the fp32 Newton system has reached
                // its accuracy for this instance.  Conjugate gradients give way to the factorisation; the second time there
                // the instance is handed to the general kernel, which starts from the last accepted point.
                if (chol && ++stalls >= 2) { alpha = alpha_prev; break; }
                if (!chol) {
                    // (the last accepted point once more: this one has no factorisation)
                    chol = true; alpha = alpha_prev; rprev = kFNone; lam = 1.f; was_kind = -1;
                    continue;
                }
            }
        }
        if (high) { mode = kHigh; full_grid = true; rprev = kFNone; lam = 1.f; was_kind = -1; continue; }
        // contraction of the last full step (same grid and precision on both sides)
        const float rho = (comparable && !coarse && lam == 1.f) ? __fdividef((float)rn, rprev) : kFNone;
        rprev = (float)rn; lam = 1.f;
        alpha_prev = alpha;
        // Newton step
        double dl;
        bool fail = false;
        float pivot = 1.f;
        float jump = 0.f;                // part of the step that is a common shift, not subject to the clamp
        if (!chol) {
            // The common scale of the weights.  The slack's share g0 = T^n - sum g is, along that scale, a falling logistic
            // curve whose slope is sum s; where its target t0 is far below (acceptance close to one), the curve is inverted
            // exactly, as the tokens' own curves are in newton_rhs: a Newton step would move the scale by one at most.
            float shift = 0.f;
            const float lin = slack ? __fdividef(sums[0], sums[1]) : 0.f;
            if (slack) {
                const double Tn = sm.scal[SC_TN];
                const float g0 = (float)(Tn - rg[0]), slope = sums[1];
                shift = lin;
                pivot = __fdividef(slope, sums[2]);                 // of the order of the smallest relative pivot
                float far = 0.f;
                if (g0 < kFSmallSlack * (float)Tn) {
                    // too small a difference for fp32; the slope, a sum of positive terms, is the share itself there, roughly: in fp64 it is for long jumps
                    // only (from 0.02 on the steps kept away from the solution: 1024 headline rows at a target temperature of 0.2 2620 us for 380)
                    far = __logf(__fdividef(fmaxf(slope, 1.0e-30f), fmaxf(t0, kFLeastSlack * (float)Tn)));
                    if (mode == kLow || fabsf(far) > kFScaleJumpFar) { shift = fminf(fmaxf(far, -16.f), 16.f); jump = shift; }
                } else if (t0 > 0.f && g0 > slope) {
                    // saturation level c0 from value and slope:  slope = g0 (1 - g0 / c0)
                    const float inv = __fdividef(g0 - slope, g0 * g0);                // 1 / c0
                    const float q = __fdividef(g0 * (1.f - t0 * inv), t0 * (1.f - g0 * inv));
                    far = q > 0.f ? __logf(q) : 0.f;
                    // (under a cap of one or two evaluations only a long one, which no Newton step replaces: what such a call leaves unconverged is what it
                    // was before there were shorter ones.  700 rows of n = 8, k = 50, target temperature 0.7, a cap of two: 505 within the tolerance, 698 with them)
                    const float least = max_iters < 3 ? kFScaleJumpFar : mode == kLow ? kFScaleJumpLow : kFScaleJump;
                    if (fabsf(far) > least) { shift = fminf(fmaxf(far, -16.f), 16.f); jump = shift; }
                }
            }
            // (far from the solution the step need not be solved to more than the model is worth)
            const float rtol = mode == kLow ? fminf(fmaxf(kFCgLow * (float)rn, kFCgTol), kFCgLoose) : kFCgTol;
            cg_solve<C>(m, slack, slack ? -__fdividef(1.f, sums[1]) : __fdividef(1.f, sums[2]), lin, shift, rtol, sm.flag);
            dl = act ? (double)sm.yv[i] : 0.0;
        } else {
            backward_subst<C>(m, sm.flag);
            __syncthreads();
            fail = sm.scal[SC_FAIL] != 0.0;
            pivot = (float)sm.scal[SC_PIVOT];
            dl = act ? (double)sm.dl[i] : 0.0;
            // proportional-fitting step  alpha += log(rhs / g)  (and the full grid from here on)
            if (fail) { full_grid = true; dl = act ? m_log(rhs_i / g) : 0.0; }
        }
        if (!slack) {
            const double mean = tok_sum<C>(sm, dl, par) / (double)m;
            if (act) dl -= mean;
        }
        // largest component, s2 = sum g dl^2 (see below), the extremes of the weights after the step, and whether it is a number
        double s2 = act ? g * dl * dl : 0.0;
        const float an = (float)fmin(fmax(alpha + dl, -kFAlphaClamp), kFAlphaClamp);
        unsigned top[3] = {act ? __float_as_uint(fabsf((float)(dl - (double)jump))) : 0u, act ? fkey(an) : 0u, act ? fkey(-an) : 0u};
        float wsum = act ? Rx<float>::ex(an) : 0.f;
        tok_reduce<C, 1, 1, 3>(sm, &s2, &wsum, top, par);
        const float dm = __uint_as_float(top[0]), far = dm + fabsf(jump);
        // (NaN for every thread or none)
        if (!(s2 < 1.0e300) || !(dm < kFNone)) {
            if (chol) break;                 // no usable step: the general kernel's
            // badly conditioned: the same point again with an fp64 gradient and a factorisation
            mode = kHigh; chol = true; full_grid = true; rprev = kFNone; was_kind = -1;
            continue;
        }
        if (tid == 0) put_extent(sm, fkey_inv(top[1]), -fkey_inv(top[2]), wsum, n, slack);
        ranged = !(dm > (float)kFStepClamp);
        // a full Newton step below 1e-11 in alpha: the weights cannot be improved at this quadrature accuracy
        if (!fail && mode != kLow && far < 1.0e-11f) { status = GR_OK; it++; break; }
        if (dm > (float)kFStepClamp && act) dl = jump + (dl - (double)jump) * (double)__fdividef((float)kFStepClamp, dm);
        alpha = fmin(fmax(alpha + dl, -kFAlphaClamp), kFAlphaClamp);
        // Stop on a predicted residual, without another evaluation, after a step from a point evaluated in fp64 on the
        // full grid.  Measured with this iteration against the oracle's residual at the weights returned, 14191 such stops at tolerances
        // of 1e-8 (quadrature steps 0.25 and 0.4), 3e-7 and 1e-5 on 28 kinds of rows: every benchmark shape, random rows of 16 to 128 tokens with 2 to 32 drafts,
        // whole and truncated, rows picked for prefixes that are almost tight (weights on several scales), and long series with a dominant token; 916 in outer blocks.  12960
        // were an instance's only system and are held one by one against what they left, less the floor of 3e-9:
        // (i) By the step (12261).  Second order: s2 = sum_i g_i delta_i^2 (each flow is a sum of terms exponential in alpha over
        // positive normalisers).  First order, after conjugate gradients: what the half-precision Hessian leaves of the residual (1202 stops
        // after a fresh one: 0.007 of it at most, 0.0125 on other draws of the same kinds), plus the distance to the point where a reused one was formed (11051 stops, distances of 0.004 in
        // the median, 0.03 in one of ten, 0.11 at most: 0.45 lin at most).  Left were never more than 13 % of 10 s2 + 3 lin, 38 % of the norm reported
        // and 10 % of the tolerance; lin is the larger term in all but 25.
        // (ii) By the ratio (699): the last full step on this grid contracted the residual by rho < 0.1, and the next one is taken
        // to contract by no less than that, its own length (along a direction in which the flows hardly change s2 says
        // nothing, and the length of the step times the residual is what it leaves) and the Hessian's share of (i), which already is twice what was seen and is held
        // with half the margin.  0.44 of the norm reported was left at most, 0.19 of the tolerance.
        // (Without the last, by contractions that the next step, with the same Hessian, did not repeat, up to 5 times the norm reported was left, and 0.77 of a
        // tolerance of 1e-8.  Held with a margin of three it costs up to 6 % of the instances of a dominant token an evaluation, with 1.5 half of those.)
        // Neither is trusted when the factorisation cancelled all but a few percent of some diagonal entry, or, after
        // conjugate gradients, when the common scale of the weights has a slope of that order: with weights of
        // 1e5 and more the fp32 system stops producing Newton steps, the residual stays where it is while the steps, and
        // with them s2, shrink.  (Relative pivots then lie below 4e-3, others above 3e-2.  An outer block has no common
        // scale: it is the direction that the system leaves out.)
        const bool trusted = !fail && pivot > (float)kFTrustPivot;
        if (mode == kLow) {
            // the next point is close enough: fp64 from here on, with this factorisation
            if (kFPredictBound * s2 < kFLowLeave && far <= 0.1f) { mode = trusted ? kChord : kHigh; full_grid = true; dist = far; }
        } else if (trusted && !coarse) {
            // (what a step by conjugate gradients leaves of the residual, at least)
            const float base = chol ? 0.f : (float)kFChordBase + (mode == kChord ? 2.f * dist : 0.f);
            const float lin = base * (float)rn, next = fmaxf(fmaxf(rho, far), base);
            const bool by_step = far <= (float)kFPredictStep && kFPredictSafety * s2 + 3.0 * (double)lin < tol;
            const bool by_ratio = rho < 0.1f && dm <= (float)kFStepClamp && kFRatioSafety * (double)fmaxf(rho, far) * rn < tol && kFBaseSafety * (double)lin < tol;
            if (by_step || by_ratio) {
                rn = by_step ? kFPredictBound * s2 + (double)lin : (double)next * rn;
                status = GR_OK; it++;
                predicted = true;
                break;
            }
            if (mode == kChord) dist += dm;
        }
    }
    // (not converged here: the last accepted point, the general kernel's starting point)
    if (lead) sm.wd[i] = act ? m_exp(status == GR_OK ? alpha : alpha_prev) : 0.0;
    if (tid == 0) { sm.scal[SC_GNORM] = rn; sm.scal[SC_ITERS] = (double)(it | (predicted ? kItersPredicted : 0)); }
    return status;
}

template <class C>
__global__ void __launch_bounds__(C::T, C::kCtas)
fast_solve_kernel(char* __restrict__ ws, char* __restrict__ params, int pstride, int kcap, int V, int n, int topk,
                  double temp_t, double temp_d, double tol, int max_iters, double qstep, double tau, double sigma,
                  float* __restrict__ alpha_out, int* __restrict__ status_out, FusedArgs fa,
                  const __grid_constant__ typename CircleOf<C::kContour>::type circle)
{
    __shared__ int s_sel;
    warm_tables();
    pdl_wait();
    GR_CHECK_FLAG_DECL;
    GR_CHECK_FLAG_INIT;
    const bool fused = fa.draft != nullptr;
    const int tid = threadIdx.x, lane = tid & 31;
    const long long b = blockIdx.x;
    char* pb = params + (size_t)b * pstride;
    ParamView pv = view_params(pb, kcap, V, GR_CHECK_FLAG);
    const WsView wv = view_ws(ws, b, GR_CHECK_FLAG);
    // (the record's lines on their way while its header is looked at)
    touch_lines(wv.h, ws_stride());
    if (kcap == 0 || wv.h->bad != 0 || wv.h->count <= 0) {
        if (tid == 0) write_no_rule(pv.h, n, wv.h->bad != 0, alpha_out, status_out, b);
        if (fused) {
            __syncthreads();
            fused_draw(fa, pv.h, b, n, smem_raw + C::oU, GR_CHECK_FLAG);
        }
        return;
    }
    constexpr int MP = C::MP;
    int* const ck = GR_CHECK_FLAG;
    const FSm<C> sm(ck);
    char* const sb = sm.base;

    // ---- distributions, ratio order, H*, residuals, blocks (arrays the solve does not need live in the union area)
    PrepSm ps;
    double* const ub = reinterpret_cast<double*>(sb + C::oU);
    ps.d = sm.d; ps.p = sm.rhs; ps.Dr = sm.Dr;
    ps.tg = GR_MKPTR(double, ub, MP, ck); ps.r = GR_MKPTR(double, ub + MP, MP, ck);
    ps.key = GR_MKPTR(double, ub + 2 * MP, MP, ck); ps.psi = GR_MKPTR(double, ub + 3 * MP, MP + 4, ck);
    int* const ui = reinterpret_cast<int*>(ub + 4 * MP + 4);
    ps.id = GR_MKPTR(int, ui, MP, ck); ps.itmp = GR_MKPTR(int, ui + MP, MP, ck);
    ps.blk = sm.blk; ps.red = sm.red; ps.out3 = sm.scal + SC_OUT;
    const PrepResult pr = prep_instance(ps, wv, pv.h, V, n, topk, temp_t, temp_d);
    const int k = pr.k, jstar = pr.jstar;
    // Truncated variant (Algorithm 1 with an error threshold): every system is solved on its truncation set alone,
    // to gradient norm 5 tau; the other tokens keep weight 0.
    const bool trunc = tau > 0.0;
    if (trunc) {
        truncation_sets(ps, sm.trunc, ps.itmp, k, jstar, n, tau);
        tol = 5.0 * tau;
    }
    if (tid == 0) { sm.scal[SC_TOL] = tol; sm.scal[SC_QSTEP] = qstep; sm.scal[SC_SIGMA] = sigma; }
    // with the drafted tuple at hand only the system it selects is solved
    const int sel = fused ? selected_system(fa.draft + (size_t)b * n, n, k, jstar, ps.id, sm.blk, &s_sel) : -2;
    // the rule's arrays, except the weights of the systems solved below
    for (int j = tid; j < kcap; j += C::T) {
        const bool in = j < k;
        pv.id[j] = in ? ps.id[j] : -1;
        pv.blk[j] = in ? sm.blk[j] : -2;
        pv.r[j] = in ? ps.r[j] : 0.0;
        pv.p[j] = in ? sm.rhs[j] : 0.0;
        pv.w[j] = in && !trunc ? 1.0 : 0.0;
    }
    __syncthreads();

    // ---- the systems: the inner one on H*, then every outer block with two or more tokens
    int status = GR_OK, iters_total = 0;
    double gnorm_total = 0.0;
    bool skipped = false;
    int lo = 0;
#pragma unroll 1
    while (lo < k && status == GR_OK) {
        const bool inner = lo < jstar;
        const int bk = sm.blk[lo];
        int hi = jstar;
        if (!inner) {
            // the first position of another block
            hi = k;
            for (int j0 = lo + 1; j0 < k; j0 += 32) {
                const unsigned other = __ballot_sync(0xffffffffu, j0 + lane < k && sm.blk[j0 + lane] != bk);
                if (other) { hi = j0 + __ffs(other) - 1; break; }
            }
        }
        // (a block of one token: its weight says nothing)
        if (!inner && hi - lo == 1 && !trunc) { lo = hi; continue; }
        const bool wanted = sel == -2 || (inner ? sel < 0 : sel == bk);
        // tokens of the system in ascending draft mass (fp32 is enough to order them), equal masses by position: a key of an earlier position
        // counts as larger where it is equal.  What is not in the truncation set, or behind the last token, has the key of none, far below all others.
        GR_PTR(unsigned) okey = GR_PCAST(unsigned, sm.wd);
        unsigned mine = 0u;
        const bool in = tid < hi - lo && (!trunc || sm.trunc[lo + tid] != 0);
        if (in) mine = 0x7fffffffu - __float_as_uint((float)sm.d[lo + tid]);
        if (tid < ((hi - lo + 3) & ~3)) okey[tid] = mine;
        const int m = __syncthreads_count(in);
        if (in) {
            int above = 0;
#pragma unroll 4
            for (int j = 0; j < hi - lo; j += 4) {
                const uint4 o = ld_u4(okey + j);
                above += (o.x + (j < tid ? 1u : 0u) > mine ? 1 : 0) + (o.y + (j + 1 < tid ? 1u : 0u) > mine ? 1 : 0) +
                         (o.z + (j + 2 < tid ? 1u : 0u) > mine ? 1 : 0) + (o.w + (j + 3 < tid ? 1u : 0u) > mine ? 1 : 0);
            }
            sm.ord[above] = lo + tid;
        }
        double hm = inner ? 0.0 : sm.Dr[lo];
        if (trunc && !inner) {
            // tuples counted: those inside (H* u T)^n, so the mass above the block is drf(H*) plus the T-part of the
            // higher-ratio outer blocks
            hm = sm.Dr[jstar];
            for (int j = jstar; j < lo; j++) hm += sm.trunc[j] ? sm.d[j] : 0.0;
        }
        __syncthreads();
        const int only = trunc && !inner && m == 1 ? sm.ord[0] : -1;
        if (only >= 0 && tid == 0) pv.w[only] = 1.0;
        const bool solve = inner ? m > 0 : m >= 2;
        // (a skipped inner system always leaves the rule partial)
        if (!wanted && (solve || inner)) skipped = true;
        if (solve && wanted) {
            const int st = fast_system<C>(m, inner ? 1 : 0, n, hm, max_iters, circle, ck);
            if (st != GR_OK) status = kNeedFallback;
            // (a thread reads back the weight it wrote)
            if (tid < m) pv.w[sm.ord[tid]] = sm.wd[tid];
            __syncthreads();
            gnorm_total += sm.scal[SC_GNORM]; iters_total = add_iters(iters_total, (int)sm.scal[SC_ITERS]);
        }
        __syncthreads();
        lo = hi;
    }
    if (status == GR_OK && skipped) status = GR_PARTIAL_RULE;
    write_rule_header(pv, pr, n, status, gnorm_total, iters_total, alpha_out, status_out, b, GR_CHECK_FLAG, wv.h->check);
    if (status == kNeedFallback && tid == 0) {
        const int i = atomicAdd(&reinterpret_cast<WsHeader*>(ws)->flagged, 1);
        reinterpret_cast<WsHeader*>(ws + (size_t)i * ws_stride())->flagged_id = (int)b;
    }
    if (fused && status != kNeedFallback) {
        __syncthreads();                       // the rule this CTA wrote is visible to its first warp
        fused_draw(fa, pv.h, b, n, smem_raw + C::oU, GR_CHECK_FLAG);
    }
}

template <class C>
int launch_fast_t(char* ws, char* params, int pstride, int kcap, int V, int n, int topk, double temp_t,
                  double temp_d, double tol, int max_iters, double qstep, double tau, int batch, float* alpha_out,
                  int* status_out, FusedArgs fa, cudaStream_t st)
{
    // function attributes belong to the device: set once per device
    static bool configured[kMaxDevices] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return GR_E_LAUNCH; }
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(fast_solve_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kBytes) != cudaSuccess)
            return GR_E_LAUNCH;
        // as much shared memory as the CTAs that fit an SM use, and no more: the rest is the first-level cache, which the
        // spills of the out-of-line calls live in
        constexpr int kTotal = 228 * 1024, kUsed = C::kCtas * (C::kBytes + 1024 + 64);
        constexpr int kPercent = kUsed >= kTotal ? 100 : (100 * kUsed + kTotal - 1) / kTotal;
        if (cudaFuncSetAttribute(fast_solve_kernel<C>, cudaFuncAttributePreferredSharedMemoryCarveout, kPercent) != cudaSuccess)
            return GR_E_LAUNCH;
        configured[dev] = true;
    }
    const double sigma = exp(lgamma((double)n + 1.0) / (double)n);       // sigma^n = n!
    typename CircleOf<C::kContour>::type circle;
    if constexpr (C::kContour) {
        // N points, a multiple of eight and at least n + 12: what is folded onto [lambda^n] from [lambda^(n + N)] is below
        // 1e-11 of it at this radius, and the mean loses one digit only (the saddle lies at |lambda| = n)
        const int N = 8 * ((n + 12 + 7) / 8);
        circle.np = N / 2;
        circle.r = 0.8 * (double)n;
        circle.factor = 2.0 / (double)N * exp(lgamma((double)n + 1.0) - (double)n * log(circle.r));
        for (int p = 0; p < circle.np; p++) {
            const double th = ((double)p + 0.5) * 2.0 * 3.14159265358979323846 / (double)N;
            circle.ct[p] = cos(th); circle.st[p] = sin(th); circle.nth[p] = fmod((double)n * th, 2.0 * 3.14159265358979323846);
        }
    }
    launch_pdl(fast_solve_kernel<C>, batch, C::T, C::kBytes, st, ws, params, pstride, kcap, V, n, topk, temp_t, temp_d, tol,
               max_iters, qstep, tau, sigma, alpha_out, status_out, fa, circle);
    return GR_OK;
}

// One translation unit per series length instantiates its kernels (they compile in parallel).
#define GR_FAST_ARGS                                                                                              \
    char *ws, char *params, int pstride, int kcap, int V, int n, int topk, double temp_t, double temp_d,   \
        double tol, int max_iters, double qstep, double tau, int batch, float *alpha_out, int *status_out,       \
        FusedArgs fa, cudaStream_t st
#define GR_FAST_PASS ws, params, pstride, kcap, V, n, topk, temp_t, temp_d, tol, max_iters, qstep, tau, batch, alpha_out, status_out, fa, st
#define GR_FAST_INSTANTIATE(NAME, ...)                                                                            \
    int launch_fast_##NAME(GR_FAST_ARGS) { return launch_fast_t<Cfg<__VA_ARGS__>>(GR_FAST_PASS); }

}  // namespace fast
}  // namespace gr
