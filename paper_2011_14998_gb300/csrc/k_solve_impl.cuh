// k_solve_impl.cuh -- formal solution along ray pairs and the mean intensity J
// (Eqs. 1-3, Sections 2.1.1-2.1.2).
//
// One warp per (origin, frequency tile); each lane carries BPL frequency bins
// (bin tile*32*BPL + lane + 32 i, i < BPL).  The warp walks every ray pair of
// its origin in ascending pair order.  Each half of the pair runs from the far
// end of its traced point list to the origin, in chunks of 32 points:
//   1. staging: lane j takes one point of the chunk -- its exact projected
//      distance Z (double), projected velocity difference delta = (v - v_o).d
//      and line data -- and, for the interval to the farther point, the number
//      of velocity samples (Section 2.1.1) and the constants of Eq. 2;
//   2. sample generation: the chunk's velocity samples (data linear in
//      distance between consecutive points, Section 2.1.1) are written to
//      shared memory as one record per sample, the lanes generating them in
//      parallel, so the frequency-independent work of a sample is done once
//      per warp instead of once per lane;
//   3. elimination: every lane reads each record (a broadcast) and, for each
//      of its bins,
//        * line optics: chi = chi_c + sum_l chi0_l exp(-a_l^2), eta likewise,
//          a_l the Doppler-shifted profile argument of line l at the bin;
//        * Eq. 2: the sample interval is split into
//          n_inter = ceil(max(chi) ds / dtau_max) equal parts, chi and eta
//          linear, trapezoidal dtau;
//        * Gaussian elimination of the Feautrier system (Eq. 1, second-order
//          boundary condition) in the scaled form of Rybicki & Hummer (1991):
//            boundary row:  Fh = 1 + dt/2,       D = 1/(1 + dt Fh), zh = D (S dt/2 + I)
//            interior row:  Fh = dtbar + D Fh,   D = 1/(1 + dt Fh), zh = D (dtbar S + zh)
//          with Fh = F_i / dtau_i and zh = z_i / dtau_i of the textbook 1+B
//          form, so no quantity overflows for small dtau and no difference of
//          nearly equal numbers is formed.  The boundary row is the interior row
//          applied to the state (Fh, D, zh, dtbar) = (1, 1, I, dt/2), and one
//          reciprocal 1 / (chi (1 + dt Fh)) per row yields both D and D S.
// The two half-sweeps meet at the origin row, which gives u without back
// substitution:  u_o = (dtbar S_o + zh- + zh+) / (dtbar + D- Fh- + D+ Fh+),
// an empty half contributing (zh, D Fh) = (I, 1).  J accumulates 2 w u in
// double precision with Neumaier's compensated sum.
//
// Template R selects the arithmetic: double (plain form: the samples are laid
// out exactly as the definition interpolates them, and Eq. 2 is evaluated as
// written) or float (single-precision bulk; Z and its differences and the J
// sum in double).
//
// Integer decisions of the single-precision form.  The velocity-sample count
// and Eq. 2's n_inter are the integers the double-precision definition gives.
// Each is first taken on the single-precision values together with a rigorous
// bound on their distance from the double-precision ones (the rounding of every
// operand and operation, the approximate reciprocal and exp2 at the error
// bounds below); where the bound does not separate the decision from the next
// integer it is redone in double precision from the double-precision point
// data, in the definition's order of operations.  The bound of Eq. 2 is folded
// into the per-interval threshold on chi, so the common case (no sub-interval
// anywhere in the warp) costs nothing extra.
#pragma once

#include <type_traits>

#include "f64_int.cuh"
#include "mgx_internal.cuh"

namespace mgx {

namespace {

constexpr unsigned kFull = 0xffffffffu;

template <typename R>
struct Ar;

// Double precision (plain form): the Gaussian exp(-a^2) and IEEE divisions.
template <>
struct Ar<double> {
    static constexpr double kArgScale = 1.0;
    static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
    static __device__ __forceinline__ double gauss(double a) { return exp(-(a * a)); }
    static __device__ __forceinline__ double src(double eta, double chi) { return eta / chi; }
};

// Single precision: the profile constants are prescaled by sqrt(log2 e), so
// exp(-a^2) = 2^(-a'^2) is one ex2.approx; reciprocals are rcp.approx.
template <>
struct Ar<float> {
    static constexpr double kArgScale = 1.2011224087864498;  // sqrt(log2(e))
    static __device__ __forceinline__ float rcp(float x) {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ float gauss(float a) {
        float r;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(-(a * a)));
        return r;
    }
    static __device__ __forceinline__ float src(float eta, float chi) { return eta * rcp(chi); }
};

// Error constants of the single-precision decisions: the unit roundoff and the
// relative errors taken for rcp.approx.ftz.f32 (documented at 1 ulp; 2 ulp
// taken) and ex2.approx.ftz.f32 (2^-20, well above what GB300 gives; a GPU
// test checks both bounds against double-precision references).
constexpr float kU = 5.9604644775390625e-8f;    // 2^-24
constexpr float kERcp = 2.384185791015625e-7f;  // 2^-22
constexpr float kEEx2 = 9.5367431640625e-7f;    // 2^-20
// |delta32 - delta64| <= kDeltaErr sum_i (|v_i| + |v_o,i|) |d_i| for the
// single-precision projection (operands rounded to single, then three
// products and two sums)
constexpr float kDeltaErr = 6.5f * kU;

// The point arrays of the form's precision, read from the mesh and line
// descriptors at each use (the descriptors live in constant or global memory,
// so no registers hold the pointers across the elimination loop).
template <typename R>
struct Pts;

template <>
struct Pts<double> {
    static __device__ __forceinline__ const double *vx(const DevMesh &m) { return m.vx; }
    static __device__ __forceinline__ const double *vy(const DevMesh &m) { return m.vy; }
    static __device__ __forceinline__ const double *vz(const DevMesh &m) { return m.vz; }
    static __device__ __forceinline__ const double *chi0(const DevLines &L) { return L.chi0; }
    static __device__ __forceinline__ const double *eta0(const DevLines &L) { return L.eta0; }
    static __device__ __forceinline__ const double *dvw(const DevLines &L) { return L.dvw; }
    static __device__ __forceinline__ const double *chic(const DevLines &L) { return L.chic; }
    static __device__ __forceinline__ const double *etac(const DevLines &L) { return L.etac; }
};

template <>
struct Pts<float> {
    static __device__ __forceinline__ const float *vx(const DevMesh &m) { return m.vxf; }
    static __device__ __forceinline__ const float *vy(const DevMesh &m) { return m.vyf; }
    static __device__ __forceinline__ const float *vz(const DevMesh &m) { return m.vzf; }
    static __device__ __forceinline__ const float *chi0(const DevLines &L) { return L.chi0f; }
    static __device__ __forceinline__ const float *eta0(const DevLines &L) { return L.eta0f; }
    static __device__ __forceinline__ const float *dvw(const DevLines &L) { return L.dvwf; }
    static __device__ __forceinline__ const float *chic(const DevLines &L) { return L.chicf; }
    static __device__ __forceinline__ const float *etac(const DevLines &L) { return L.etacf; }
};

// Values of one lane: a scalar, or two bins' single-precision values side by
// side (float2), on which GB300's packed instructions work (fma.rn.f32x2 and
// its kin): the same two IEEE operations in one issue slot.
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }

template <typename V>
__device__ __forceinline__ V vset(float x) {
    if constexpr (sizeof(V) == sizeof(float2) && !std::is_same_v<V, double>) return make_float2(x, x);
    else return V(x);
}

// Component c of a value.
__device__ __forceinline__ float vget(float x, int) { return x; }
__device__ __forceinline__ double vget(double x, int) { return x; }
__device__ __forceinline__ float vget(float2 x, int c) { return c ? x.y : x.x; }
template <typename T>
__device__ __forceinline__ void vput(T &x, int, T v) { x = v; }
__device__ __forceinline__ void vput(float2 &x, int c, float v) { (c ? x.y : x.x) = v; }

// One compiled form of the solve: the arithmetic R, the lines NL and bins per
// lane BPL it is compiled for, the scheme's order, the pivots' precision P.
// The single-precision second-order form holds its bins in pairs (kPacked): the
// optics and rows of two bins then take 20 issue slots instead of 36, and issue
// slots were what bounded the loop (77 % busy; FP32 lanes 39 %).  Together with
// the branch-free runs of consume_chunk and the lines left out (line_is_far) the
// solve of the 50 000-point wind fell from 86.1 to 70.8 ms, of a batch of five
// four-line models from 136.4 to 95.2 ms, J the same bit for bit.  What bounds it
// now is latency (issue 61 % busy): the reciprocal and exp2 on the recurrence's
// path and the staging's gathers, at 8 resident CTAs.
template <typename R_, int NL_, int BPL_, int ORD_, typename P_ = R_>
struct Form {
    using R = R_;
    using P = P_;
    static constexpr int NL = NL_, BPL = BPL_, ORD = ORD_;
    static constexpr bool kPacked = sizeof(R) == 4 && sizeof(P) == 4 && ORD == 2 && BPL % 2 == 0;
    // the double-precision second-order form: exponentials and divisions on the integer pipes
    static constexpr bool kInt = sizeof(R) == 8 && ORD == 2;
    using V = std::conditional_t<kPacked, float2, R>;
    using W = std::conditional_t<kPacked, float2, P>;
    static constexpr int kIn = kPacked ? 2 : 1;  // bins in a value
    static constexpr int NV = BPL / kIn;         // values per lane
};

// Per-bin constants: the Doppler-shifted profile argument of line l at this
// bin is (A[l] + B[l] delta) / dv (prescaled for the single-precision ex2).
template <typename V, int NL>
struct Bin {
    V A[NL], B[NL];
};

// Total opacity and emissivity of a sample for one bin: delta, rdv = 1/dv,
// continuum (cc, ec) and line-centre values ce[2l] = chi0_l, ce[2l+1] = eta0_l.
// Lines past the model's count have chi0 = eta0 = 0 and contribute nothing.
template <typename R, int NL>
__device__ __forceinline__ void optics(R delta, R rdv, R cc, R ec, const R *ce, const Bin<R, NL> &f, R &chi,
                                       R &eta) {
    chi = cc;
    eta = ec;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const R g = Ar<R>::gauss(fma(f.B[l], delta, f.A[l]) * rdv);
        chi = fma(ce[2 * l], g, chi);
        eta = fma(ce[2 * l + 1], g, eta);
    }
}

// One line's part of it for two bins.
__device__ __forceinline__ void add_line(float2 delta, float2 rdv, float2 c0, float2 e0, float2 A, float2 B,
                                         float2 &chi, float2 &eta) {
    const float2 a = vmul(vfma(B, delta, A), rdv);
    const float2 q = vmul(a, a);
    float2 g;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(g.x) : "f"(-q.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(g.y) : "f"(-q.y));
    chi = vfma(c0, g, chi);
    eta = vfma(e0, g, eta);
}

// State of the elimination of one bin along one half of a pair line.
// Starting from (Fh, D, zh, dtp) = (1, 1, I, 0) the interior row reproduces
// the second-order boundary row, and a half without points leaves exactly the
// empty-half coupling (D Fh, zh) = (1, I).
//
// The Hermitian scheme (ORD 4) also carries the source function of the last
// eliminated row (Sp) and of the current sample (Sc), the last increment (hp,
// negative before the first row) and its reciprocal (rh).
//
// P is the precision of the pivot recurrence (Fh, D and the increments dt):
// R, or double with R = float (the form with double-precision optical-depth
// increments and pivots, second-order scheme only).
template <typename R, typename P = R>
struct Sweep {
    P Fh, Dm, dtp;  // scaled 1+B quantities of the last eliminated row, half its dtau
    R zh;
    R chi, eta;     // optics of the current (not yet eliminated) sample
    R Sp, Sc, hp, rh;  // Hermitian scheme only
    uint64_t Y;        // double-precision pivots with R = float: D Fh as hold_y has it (Fh, Dm not kept)
};

// The second-order row below for two bins at once, operation for operation.
__device__ __forceinline__ void row2(Sweep<float2> &w, float2 chi, float2 eta, float2 dt) {
    const float2 half = make_float2(0.5f, 0.5f), one = make_float2(1.f, 1.f);
    const float2 dtb = vfma(dt, half, w.dtp);
    w.Fh = vfma(w.Dm, w.Fh, dtb);
    const float2 den = vmul(chi, vfma(dt, w.Fh, one));
    const float2 rr = make_float2(Ar<float>::rcp(den.x), Ar<float>::rcp(den.y));
    w.Dm = vmul(chi, rr);
    w.zh = vfma(dtb, vmul(eta, rr), vmul(w.Dm, w.zh));
    w.dtp = vmul(dt, half);
}

// Eliminate the row of the current sub-point (optics chi, eta) once the
// increment dt beyond it is known.  One reciprocal R = 1 / (chi (1 + dt Fh))
// gives D = chi R and D S = eta R.  The state carries half the previous
// increment, so dtbar = (dt_prev + dt) / 2 is one fused operation (the
// halvings are exact, so the rounding is that of the plain expression).
//
// ORD 4: the Hermitian row of Auer (1976) (Section 2.1) in the same scaled
// form.  With h- the previous and h+ the current increment, hbar their mean,
//   1 - lambda = (h-^2 + h- h+ - h+^2) / 12,  mu = (h+^2 + h- h+ - h-^2) / 12,
//   Fh = (hbar + lambda D Fh_prev) / (1 - mu),   D = 1 / (1 + h+ Fh),
//   zh = D (hbar r + lambda zh_prev) / (1 - mu),
//   hbar r = hbar S_i + ((1 - lambda) / h-) (S_{i-1} - S_i) + (mu / h+) (S_{i+1} - S_i),
// which is the textbook elimination with the compact weights
// a = (1 - lambda) / (h- hbar), g = mu / (h+ hbar), b = 1 - a - g, scaled by
// the increment beyond each row (F = h+ Fh, z = h+ zh).  A row whose two
// increments differ by more than a factor kHermRatio takes the second-order
// weights (lambda = 1, mu = 0): the compact weights grow like the ratio and
// would amplify the rounding of S next to a vanishing increment.  The first
// row of a half is the third-order boundary row (Auer 1967):
//   Fh = (1 + h/2) / (1 - h^2/6),  zh = D (h S_i / 3 + h S_{i+1} / 6 + I) / (1 - h^2/6).
constexpr double kHermRatio = 64.0;

// A non-negative value of the form in the pivots' precision.
template <typename P, typename R>
__device__ __forceinline__ P wide(R x) {
    if constexpr (sizeof(P) != sizeof(R)) return widen(x);
    else return x;
}

template <int ORD, typename R, typename P>
__device__ __forceinline__ void row(Sweep<R, P> &w, R chi, R eta, P dt, R Si, R Sn) {
    if constexpr (ORD == 2 && sizeof(P) != sizeof(R)) {
        // pivots of double's precision: D = 1 / (1 + dt Fh) in fixed point (pivot; of the
        // 22 FP64 instructions a row took, the reciprocal most, three are left); z in single
        // precision from D and S = eta / chi
        const P half = halve(dt), dtb = half + w.dtp;
        R Dr, bD;  // D and dtb D in single precision
        pivot(dt, dtb, w.Y, Dr, bD);
        w.zh = Dr * w.zh + bD * (eta * Ar<R>::rcp(chi));
        w.dtp = half;
    } else if constexpr (ORD == 2) {
        const P dtb = fma(dt, P(0.5), w.dtp);
        w.Fh = dtb + w.Dm * w.Fh;
        {
            const R rr = Ar<R>::rcp(chi * (R(1) + dt * w.Fh));
            w.Dm = chi * rr;
            w.zh = w.Dm * w.zh + dtb * (eta * rr);
        }
        w.dtp = dt * P(0.5);
    } else {
        static_assert(sizeof(P) == sizeof(R), "the Hermitian scheme keeps its pivots in the form's precision");
        const R rh = Ar<R>::rcp(dt);
        if (w.hp < R(0)) {  // boundary row
            const R k = Ar<R>::rcp(R(1) - dt * dt * R(1.0 / 6.0));
            w.Fh = fma(dt, R(0.5), R(1)) * k;
            const R D = Ar<R>::rcp(fma(dt, w.Fh, R(1)));
            w.zh = D * k * (dt * (Si * R(1.0 / 3.0) + Sn * R(1.0 / 6.0)) + w.zh);
            w.Dm = D;
        } else {
            const R hm = w.hp, p = hm * dt;
            const bool compact = !(dt > R(kHermRatio) * hm || hm > R(kHermRatio) * dt);
            const R oml = compact ? (hm * hm + p - dt * dt) * R(1.0 / 12.0) : R(0);  // 1 - lambda
            const R mu = compact ? (dt * dt + p - hm * hm) * R(1.0 / 12.0) : R(0);
            const R k = Ar<R>::rcp(R(1) - mu);
            const R hb = (hm + dt) * R(0.5);
            const R hr = hb * Si + oml * w.rh * (w.Sp - Si) + mu * rh * (Sn - Si);
            const R lam = R(1) - oml;
            w.Fh = k * (hb + lam * w.Dm * w.Fh);
            const R D = Ar<R>::rcp(fma(dt, w.Fh, R(1)));
            w.zh = D * k * (hr + lam * w.zh);
            w.Dm = D;
        }
        w.rh = rh;
        w.hp = dt;
        w.Sp = Si;
    }
}

// u at the origin row from the two half-sweeps (the origin row couples the
// last eliminated rows of both halves; no back substitution is needed).
// Second order: u_o = (dtbar S_o + zh- + zh+) / (dtbar + D- Fh- + D+ Fh+), an
// empty half contributing (D Fh, zh) = (1, I) through its initial state.
template <typename R, typename P>
__device__ __forceinline__ R origin_u2(const Sweep<R, P> &b, const Sweep<R, P> &f, R So) {
    const P dtb = b.dtp + f.dtp;  // the halves of the two last increments
    return R((dtb * P(So) + P(b.zh) + P(f.zh)) / (dtb + b.Dm * b.Fh + f.Dm * f.Fh));
}

// Hermitian scheme: with h- (h+) the last increment of the backward (forward)
// half and lambda- = 1 - (h-^2 + h- h+ - h+^2)/12, lambda+ = 1 - (h+^2 + h- h+ - h-^2)/12,
//   u_o = (hbar r_o + lambda- zh- + lambda+ zh+) / (hbar + lambda- D- Fh- + lambda+ D+ Fh+);
// with one half empty the origin row is the third-order boundary row,
//   u_o = (h S_o/3 + h S_1/6 + I + (1 - h^2/6) zh) / (1 + h/2 + (1 - h^2/6) D Fh);
// with both empty u_o = I.
template <typename R, typename P>
__device__ __forceinline__ R origin_u4(const Sweep<R, P> &b, const Sweep<R, P> &f, R So, R I) {
    if (b.hp < R(0) && f.hp < R(0)) return I;
    if (b.hp < R(0) || f.hp < R(0)) {
        const Sweep<R, P> &w = b.hp < R(0) ? f : b;
        const R h = w.hp, k1 = R(1) - h * h * R(1.0 / 6.0);
        return (h * (So * R(1.0 / 3.0) + w.Sp * R(1.0 / 6.0)) + I + k1 * w.zh) / (fma(h, R(0.5), R(1)) + k1 * w.Dm * w.Fh);
    }
    const R hm = b.hp, hp = f.hp, p = hm * hp;
    const bool compact = !(hp > R(kHermRatio) * hm || hm > R(kHermRatio) * hp);
    const R oml = compact ? (hm * hm + p - hp * hp) * R(1.0 / 12.0) : R(0);  // 1 - lambda-
    const R mu = compact ? (hp * hp + p - hm * hm) * R(1.0 / 12.0) : R(0);   // 1 - lambda+
    const R hb = (hm + hp) * R(0.5);
    const R hr = hb * So + oml * b.rh * (b.Sp - So) + mu * f.rh * (f.Sp - So);
    return (hr + (R(1) - oml) * b.zh + (R(1) - mu) * f.zh) /
           (hb + (R(1) - oml) * b.Dm * b.Fh + (R(1) - mu) * f.Dm * f.Fh);
}

// Where the ids of one half-ray are: entries k < n_main at main[k], the rest
// at tail[tail_off + k] (padded layout); cnt entries in all.
struct HalfList {
    const int32_t *main;
    const int32_t *tail;
    int64_t tail_off;
    int32_t n_main, cnt;
};

__device__ __forceinline__ HalfList half_list(const SolveArgs &a, int64_t h) {
    HalfList l;
    if (a.pad == 0) {
        l.main = a.idx + (a.offs[h] - a.base);
        l.cnt = l.n_main = int32_t(a.offs[h + 1] - a.offs[h]);
        l.tail = a.idx;
        l.tail_off = 0;
    } else {
        l.cnt = int32_t(a.lens[h]);
        l.main = a.idx + h * a.pad;
        l.n_main = l.cnt < a.pad ? l.cnt : a.pad;
        l.tail = a.tail;
        l.tail_off = a.offs[h] - a.base - a.pad;
    }
    return l;
}

// Layout of one velocity-sample record, as the bins read it: delta, 1/dv,
// continuum opacity and emissivity, half the distance to the previous sample,
// the Eq. 2 threshold on chi, then chi0 and eta0 of each line; padded to whole
// 16-byte words so that each word is one shared-memory load.  An infinite
// threshold (single precision) marks an interval on which no bin can need a
// split.  The packed form stores the values twice, so that a load yields the
// operand pair of the packed instructions (a register pair built from one
// loaded value would cost a move each; with more than two lines only the line
// values are stored once, for the sake of shared memory), with the lines that
// take part in the sample as a bit mask next to the threshold; the other
// single-precision forms with one line mark a sample in which it takes no part
// by a negative 1/dv.
template <class C>
struct Rec {
    using V = typename C::V;
    static constexpr bool kTwice = C::NL <= 2;  // packed: line values stored twice
    static constexpr int kVals = 6 + (C::kPacked && !kTwice ? 1 : 2) * C::NL;
    static constexpr int kPer16 = int(16 / sizeof(V));
    static constexpr int kStride = (kVals + kPer16 - 1) / kPer16 * kPer16;
};

// Per-warp shared staging: the sample records of the chunk being eliminated
// (kCap at a time), the chunk's points (slot 0 holds the point just farther
// than the chunk, slots 1..32 the chunk, far to near) with the constants of
// the interval from the farther point, and the warp's item.
template <class C>
struct Stage {
    using R = typename C::R;
    using V = typename C::V;
    static constexpr int NL = C::NL, BPL = C::BPL;
    static constexpr int kCap = sizeof(R) == 4 ? 32 : (NL <= 4 ? 32 : 16);
    static constexpr int kS = Rec<C>::kStride;
    static constexpr int kF = sizeof(R) == 4 ? 33 : 1;  // arrays of the single-precision decisions
    alignas(16) V rec[kCap * kS];
    alignas(16) V fA[NL][C::NV][32], fB[NL][C::NV][32];  // profile constants of each lane's bins (Bin)
    R d[33], w[33], cc[33], ec[33];         // delta, Doppler width, continuum
    R ce[2 * NL][33];                       // chi0 and eta0 per line
    R hq[33], thr[33];                      // half the sample spacing, Eq. 2 threshold
    R E[kF], qlo[kF], qhi[kF];              // bound of |chi - chi64|, Eq. 2 ratio factors
    unsigned char sk[kCap];                 // slot of each record
    R de0;                                  // single precision: bound of |delta - delta64| of the carried point
    double z[sizeof(R) == 8 ? 33 : 1];      // exact Z (single precision: the carried point's only)
    int id[33], nv[33], so[33];             // point (-1: the origin), velocity samples, their offset
    unsigned on[C::kInt ? kCap : 1];        // integer form: the lines that take part in each record
    unsigned m_block;                       // records at which a block of kBlock continuum rows starts
    double blk[C::kInt ? kCap / 8 : 1][C::kInt ? 6 : 1];  // and the blocks' maps (block of record s in blk[s / 8])
    double span;                            // integer form, one line: x_span dvw_o, the bins' half-range in km/s
    uint64_t uk[C::kInt && NL == 1 ? BPL : 1][C::kInt && NL == 1 ? 32 : 1];  // and each lane's bins' place in it, (ub / span + 1) / 2, in Q0.63
    R Am[NL], Bm[NL];                       // largest |A|, |B| of each line over the warp's bins
    double r[3], xo[3], vo[3];              // pair direction, origin position and velocity (double)
    R vor[3];                               // origin velocity in the form's precision
    int o, NB, tile;                        // origin, bins of the model, the warp's frequency tile
    HalfList hl;                            // traced list of the half being eliminated
    unsigned n_smp, n_extra, n_redo;        // work counters of the item (samples, extra sub-intervals, redone decisions)
    int fix[BPL][32];                       // Eq. 2 counts of a sample whose single-precision decision was left
                                            // open (0: not open; negative: to resolve, the bits of -chi)
    float wA[NL][2], wB[NL][2];             // single precision: smallest and largest A, B over the warp's bins
    unsigned m_split, m_new, m_wild;        // single-precision and integer forms: the round's records that may split; whose lines differ
                                            // from the record's before
};

// Bin i of the lane in the warp's tile (>= NB: beyond the last, inactive).
template <class C>
__device__ __forceinline__ int32_t lane_bin(const Stage<C> &sg, int i, int lane) {
    return sg.tile * 32 * C::BPL + lane + 32 * i;
}

// Per-lane state that lives across chunks of samples, kept in shared memory
// so that no register holds it across the out-of-line staging calls: the
// elimination state of each of the lane's bins (D and Fh enter every step only
// as their product, which is what is kept).  The pivot quantities (D Fh,
// dtb/2) are kept in the pivot precision.  What is needed only once per pair
// (the J sums, the origin's source function, the backward half's coupling to
// the origin row) stays in the item loop's registers.
template <class C>
struct Lane {
    static constexpr int kWR = C::ORD == 4 ? 6 : 3;  // zh, chi, eta (Hermitian: + Sp, Sc, hp; rh = 1/hp re-formed)
    typename C::W wp[2][C::NV][32];                  // D Fh, dtb/2
    typename C::V wr[kWR][C::NV][32];
};

// Projected distance Z = (x_n - x_o).d exactly as the tracer and its
// definition form it (explicitly rounded double operations in fixed order).
__device__ __forceinline__ double exact_Z(const DevMesh &m, int32_t id, double xo, double yo, double zo, double d0,
                                          double d1, double d2) {
    const double dx = __dsub_rn(__ldg(m.x + id), xo);
    const double dy = __dsub_rn(__ldg(m.y + id), yo);
    const double dz = __dsub_rn(__ldg(m.z + id), zo);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, d0), __dmul_rn(dy, d1)), __dmul_rn(dz, d2));
}

// Projected velocity difference (v_n - v_o).d in double precision, (x + y) + z
// with every product and sum rounded (the definition's order).
__device__ __forceinline__ double proj64(const DevMesh &m, int32_t id, const double *vo, double d0, double d1,
                                         double d2) {
    const double ux = __dsub_rn(__ldg(m.vx + id), vo[0]);
    const double uy = __dsub_rn(__ldg(m.vy + id), vo[1]);
    const double uz = __dsub_rn(__ldg(m.vz + id), vo[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(ux, d0), __dmul_rn(uy, d1)), __dmul_rn(uz, d2));
}

// Bound of |delta32 - delta64| of point id (-1: the origin) along d: the operands
// rounded to single, then three products and two sums.
template <class C>
__device__ __forceinline__ float delta_bound(const Stage<C> &sg, float vx, float vy, float vz, float f0, float f1,
                                             float f2) {
    return kDeltaErr * ((fabsf(vx) + fabsf(sg.vor[0])) * fabsf(f0) + (fabsf(vy) + fabsf(sg.vor[1])) * fabsf(f1) +
                        (fabsf(vz) + fabsf(sg.vor[2])) * fabsf(f2));
}

// Bound E of |chi32 - chi64| at every sample of the interval to the point in
// `slot` (both ends included), from the errors of delta (dea, deb at its ends,
// interpolation), dv, the profile constants, the profile argument, ex2 and the
// sums:
//   |g32 - g64| <= 0.7142 |da'| + 0.7358 rho + u/e + eps_ex2
// (0.7142 = max |d/da 2^(-a^2)|, 0.7358 = max |a d/da 2^(-a^2)|).  The error
// of a grows with |A|; far: the |a| beyond which bins need not be covered
// (infinite: every bin of the warp is).
template <class C>
__device__ __forceinline__ float opacity_bound(const Stage<C> &sg, int slot, float dea, float deb, float far) {
    const int pa = slot - 1;
    const float k6 = 6.f * kU + kERcp;  // interpolation in single precision
    const float wa = sg.w[pa], wb = sg.w[slot], ada = fabsf(sg.d[pa]), adb = fabsf(sg.d[slot]);
    const float dmax = fmaxf(ada, adb);
    const float edi = dea + deb + k6 * (ada + adb);
    const float rdvmin = 1.f / fminf(wa, wb);
    const float rho = kERcp + k6 * (wa + wb) * rdvmin + 4.f * kU;
    const float wfar = far * fmaxf(wa, wb);
    float E = 0.f, csum = fmaxf(sg.cc[pa], sg.cc[slot]);
#pragma unroll
    for (int l = 0; l < C::NL; ++l) {
        const float Am = fminf(sg.Am[l], sg.Bm[l] * dmax + wfar);
        const float dA = (3.f * kU * (Am + sg.Bm[l] * dmax) + sg.Bm[l] * edi) * rdvmin * (1.f + rho);
        const float Eg = 0.7142f * dA + 0.7358f * rho * 1.001f + 0.3679f * kU + kEEx2 + 2.f * dA * dA;
        const float c0a = sg.ce[2 * l][pa], c0b = sg.ce[2 * l][slot], c0m = fmaxf(c0a, c0b);
        E += c0m * Eg + k6 * (c0a + c0b) + kU * c0m;
        csum += c0m;
    }
    E += k6 * (sg.cc[pa] + sg.cc[slot]) + kU * fmaxf(sg.cc[pa], sg.cc[slot]) + float(C::NL + 1) * kU * csum;
    return E * 1.0625f;
}

// ---- double-precision redo of the single-precision form's decisions ------
// (rare: only where the single-precision bound leaves the integer open)

// Velocity samples of the interval between points ia and ib (-1: the origin)
// on the half along sgn r (Section 2.1.1): ceil(|delta_b - delta_a| /
// (dv_max min(dv_a, dv_b))) when the jump exceeds the limit, else 1.
__device__ __noinline__ int redo_velocity_samples(const DevMesh &m, const DevLines &Ln, const double *r,
                                                  const double *vo, int32_t o, double sgn, int32_t ia, int32_t ib,
                                                  double dv_max) {
    const double e0 = sgn * r[0], e1 = sgn * r[1], e2 = sgn * r[2];
    const double da = ia < 0 ? 0.0 : proj64(m, ia, vo, e0, e1, e2);
    const double db = ib < 0 ? 0.0 : proj64(m, ib, vo, e0, e1, e2);
    const double wa = Ln.dvw[ia < 0 ? o : ia], wb = Ln.dvw[ib < 0 ? o : ib];
    const double jump = fabs(__dsub_rn(db, da));
    const double lim = __dmul_rn(dv_max, fmin(wa, wb));
    if (!(jump > lim)) return 1;
    const double n = ceil(__ddiv_rn(jump, lim));
    return n > double(kMaxSubdiv) ? kMaxSubdiv + 1 : int(n);
}

// Eq. 2's n_inter for bin `bin` on the sub-interval between the velocity
// samples j-1 and j (counted from the farther point a, 0 = a, nv = b) of the
// interval from point ia to point ib, -1 being the origin.  The two samples are formed as the definition lays out the pair
// line: ordered along +r (the backward half from its far end, the forward half
// from the origin), each quantity interpolated linearly from the earlier point
// with t = i / nv; the opacity is the line optics of Magritte I evaluated in
// that order; n_inter = ceil(max(chi) ds / dtau_max), at least 1.
__device__ __noinline__ int redo_n_inter(const DevMesh &m, const DevLines &Ln, const double *r, const double *vo,
                                         int32_t o, double sgn, int32_t ia, int32_t ib, int nv, int j, int32_t bin,
                                         double dtau_max) {
    const bool bwd = sgn < 0.0;
    const double e0 = sgn * r[0], e1 = sgn * r[1], e2 = sgn * r[2];
    // the exact Z of the two points (0 at the origin, id -1)
    const double xo = m.x[o], yo = m.y[o], zo = m.z[o];
    const double za = ia < 0 ? 0.0 : exact_Z(m, ia, xo, yo, zo, e0, e1, e2);
    const double zb = ib < 0 ? 0.0 : exact_Z(m, ib, xo, yo, zo, e0, e1, e2);
    const int32_t p0 = bwd ? ia : ib, p1 = bwd ? ib : ia;  // base points in the definition's order
    const double z0 = bwd ? za : zb, z1 = bwd ? zb : za;
    const int ilo = bwd ? j - 1 : nv - j;  // indices of the two samples from p0
    const int32_t L = Ln.L, F = Ln.F, l = bin / F, k = bin - l * F;
    const double x = F == 1 ? 0.0
                            : __dadd_rn(-Ln.x_span, __ddiv_rn(__dmul_rn(2.0 * Ln.x_span, double(k)), double(F - 1)));
    const double ub = __dmul_rn(x, Ln.dvw[o]);
    const int32_t q0 = p0 < 0 ? o : p0, q1 = p1 < 0 ? o : p1;
    const double d0 = p0 < 0 ? 0.0 : proj64(m, p0, vo, e0, e1, e2);
    const double d1 = p1 < 0 ? 0.0 : proj64(m, p1, vo, e0, e1, e2);
    const double s0 = p0 < 0 ? 0.0 : sgn * z0, s1 = p1 < 0 ? 0.0 : sgn * z1;
    double chi[2], s[2];
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const int i = ilo + h;
        const bool at0 = i == 0, at1 = i == nv;
        const double t = __ddiv_rn(double(i), double(nv));
        auto lerp = [&](double a0, double a1) -> double {
            return at0 ? a0 : at1 ? a1 : __dadd_rn(a0, __dmul_rn(__dsub_rn(a1, a0), t));
        };
        s[h] = lerp(s0, s1);
        const double dl = lerp(d0, d1);
        const double dv = lerp(Ln.dvw[q0], Ln.dvw[q1]);
        double c = lerp(Ln.chic[q0], Ln.chic[q1]);
        for (int lp = 0; lp < L; ++lp) {
            const double c0 = lerp(Ln.chi0[int64_t(q0) * L + lp], Ln.chi0[int64_t(q1) * L + lp]);
            const double rr = Ln.ratio[l * MGX_MAX_LINES + lp];
            const double num = __dadd_rn(__dadd_rn(__dmul_rn(kC, __dsub_rn(rr, 1.0)), __dmul_rn(rr, ub)),
                                         __dmul_rn(__dmul_rn(rr, __dadd_rn(1.0, __ddiv_rn(ub, kC))), dl));
            const double arg = __ddiv_rn(num, dv);
            const double g = exp(-__dmul_rn(arg, arg));
            c = __dadd_rn(c, __dmul_rn(c0, g));
        }
        chi[h] = c;
    }
    const double n = ceil(__ddiv_rn(__dmul_rn(fmax(chi[0], chi[1]), __dsub_rn(s[1], s[0])), dtau_max));
    if (n > double(kMaxSubdiv)) return kMaxSubdiv + 1;
    return n < 1.0 ? 1 : int(n);
}

// ---- staging ----------------------------------------------------------------

// Point q of the half (q < cnt: traced entry cnt-1-q, far end first; q == cnt:
// the origin) into `slot`; its exact Z and (single precision) the bound of
// its delta's error are also returned, for the interval to it.
template <class C>
__device__ __forceinline__ void stage_point(const DevMesh &m, const DevLines &Ln, Stage<C> &sg, int32_t q, int32_t cnt,
                                            int slot, int sign, double &zq, typename C::R &deq) {
    using R = typename C::R;
    constexpr int NL = C::NL;
    const HalfList &hl = sg.hl;
    const double sgn = double(sign);
    const int32_t L = Ln.L;
    const double e0 = sgn * sg.r[0], e1 = sgn * sg.r[1], e2 = sgn * sg.r[2];
    int32_t id = sg.o;
    double z = 0.0;
    R d = R(0), de = R(0);
    // the traced ids stream through once: evict-first, so that they do not push the
    // mesh and the spilled item state out of L2
    if (q < cnt) {
        const int32_t k = cnt - 1 - q;
        id = k < hl.n_main ? __ldcs(hl.main + k) : __ldcs(hl.tail + (hl.tail_off + k));
    }
    float4 p0, p1, p2, p3;  // single precision: the point's record
    if constexpr (sizeof(R) == 4) {
        const float4 *rec = Ln.pt + 4 * int64_t(id);
        p0 = __ldg(rec);
        p1 = __ldg(rec + 1);
        p2 = __ldg(rec + 2);
        p3 = __ldg(rec + 3);
    }
    if (q < cnt) {
        if constexpr (sizeof(R) == 8) {
            z = exact_Z(m, id, sg.xo[0], sg.xo[1], sg.xo[2], e0, e1, e2);
            d = proj64(m, id, sg.vo, e0, e1, e2);
        } else {
            const double dx = __dsub_rn(__hiloint2double(__float_as_int(p0.y), __float_as_int(p0.x)), sg.xo[0]);
            const double dy = __dsub_rn(__hiloint2double(__float_as_int(p0.w), __float_as_int(p0.z)), sg.xo[1]);
            const double dz = __dsub_rn(__hiloint2double(__float_as_int(p1.y), __float_as_int(p1.x)), sg.xo[2]);
            z = __dadd_rn(__dadd_rn(__dmul_rn(dx, e0), __dmul_rn(dy, e1)), __dmul_rn(dz, e2));  // as exact_Z
            const float f0 = float(e0), f1 = float(e1), f2 = float(e2);
            const float vx = p1.z, vy = p1.w, vz = p2.x;
            const float ux = vx - sg.vor[0], uy = vy - sg.vor[1], uz = vz - sg.vor[2];
            d = fmaf(uz, f2, fmaf(uy, f1, ux * f0));
            de = delta_bound<C>(sg, vx, vy, vz, f0, f1, f2);
        }
    }
    sg.id[slot] = q < cnt ? id : -1;
    if constexpr (sizeof(R) == 8) sg.z[slot] = z;
    zq = z;
    deq = de;
    sg.d[slot] = d;
    constexpr int kIn = sizeof(R) == 4 ? (NL < 2 ? NL : 2) : 0;  // lines in the record
    if constexpr (sizeof(R) == 4) {
        sg.w[slot] = p2.y;
        sg.cc[slot] = p2.z;
        sg.ec[slot] = p2.w;
        sg.ce[0][slot] = p3.x;
        sg.ce[1][slot] = p3.y;
        if constexpr (NL > 1) {
            sg.ce[2][slot] = p3.z;
            sg.ce[3][slot] = p3.w;
        }
    } else {
        sg.w[slot] = __ldg(Pts<R>::dvw(Ln) + id);
        sg.cc[slot] = __ldg(Pts<R>::chic(Ln) + id);
        sg.ec[slot] = __ldg(Pts<R>::etac(Ln) + id);
    }
#pragma unroll
    for (int l = kIn; l < NL; ++l) {
        sg.ce[2 * l][slot] = l < L ? __ldg(Pts<R>::chi0(Ln) + int64_t(id) * L + l) : R(0);
        sg.ce[2 * l + 1][slot] = l < L ? __ldg(Pts<R>::eta0(Ln) + int64_t(id) * L + l) : R(0);
    }
}

// The interval from the point in slot-1 (farther) to the point in `slot`:
// its number of velocity samples (Section 2.1.1) and, in single precision,
// the constants of Eq. 2 with the bound on the opacity's error.  za, zb are
// the exact Z of the farther and the nearer point, dea, deb the bounds of
// their deltas' errors (single precision).
template <class C>
__device__ __forceinline__ int stage_interval(const DevMesh &m, const DevLines &Ln, const SolveArgs &a, Stage<C> &sg,
                                              int slot, int sign, double za, double zb, typename C::R dea,
                                              typename C::R deb) {
    using R = typename C::R;
    constexpr int NL = C::NL;
    const int pa = slot - 1;
    if constexpr (sizeof(R) == 8) {
        // as defined: ceil(|delta_b - delta_a| / (dv_max min(dv_a, dv_b))) when that exceeds one
        int nv = 1;
        if (a.dv_max > 0.0) {
            const double jump = fabs(sg.d[slot] - sg.d[pa]);
            const double lim = a.dv_max * fmin(sg.w[pa], sg.w[slot]);
            if (jump > lim) {
                const double n = ceil(jump / lim);
                nv = n > double(kMaxSubdiv) ? kMaxSubdiv + 1 : int(n);
            }
        }
        if (nv > kMaxSubdiv) {
            dev_fail(a.status, kDevSubdivLimit);
            nv = kMaxSubdiv;
        }
        if constexpr (C::kInt) {
            // the largest opacity any sample of the interval can reach; infinite, for plain_step,
            // where a source function may pass 2^291: with Q to 2^301, increments to 1e60 and eight
            // composed rows below 1e3 each (2^187), S Q times them stays below 2^1000
            R cb = fmax(sg.cc[pa], sg.cc[slot]);
            int top = max(__double2hiint(sg.ec[pa]), __double2hiint(sg.ec[slot]));
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                cb += fmax(sg.ce[2 * l][pa], sg.ce[2 * l][slot]);
                top = max(top, max(__double2hiint(sg.ce[2 * l + 1][pa]), __double2hiint(sg.ce[2 * l + 1][slot])));
            }
            if (top - min(__double2hiint(sg.cc[pa]), __double2hiint(sg.cc[slot])) > (290 << 20)) cb = INFINITY;
            sg.hq[slot] = cb * (1.0 + 0x1p-40);
        }
        return nv;
    } else {
        const float da = sg.d[pa], db = sg.d[slot], wa = sg.w[pa], wb = sg.w[slot];
        int nv = 1;
        if (a.dv_max > 0.0) {
            // q64 = jump64 / lim64 lies in [(jump - ej) / lim (1 - k), (jump + ej) / lim (1 + k)]
            const float jump = fabsf(db - da);
            const float ej = dea + deb + 2.f * kU * jump;
            const float rl = 1.f / (float(a.dv_max) * fminf(wa, wb));
            const float nhi = ceilf((jump + ej) * rl * (1.f + 16.f * kU));
            if (nhi > 1.f) {
                const float nlo = ceilf((jump - ej) * rl * (1.f - 16.f * kU));
                if (nlo == nhi) {
                    nv = nhi > float(kMaxSubdiv) ? kMaxSubdiv + 1 : int(nhi);
                } else {
                    nv = redo_velocity_samples(m, Ln, sg.r, sg.vo, sg.o, double(sign), sg.id[pa], sg.id[slot],
                                               a.dv_max);
                    atomicAdd(&sg.n_redo, 1u);
                }
                if (nv > kMaxSubdiv) {
                    dev_fail(a.status, kDevSubdivLimit);
                    nv = kMaxSubdiv;
                }
            }
        }
        const float ds = float(za - zb);  // distance increment, differenced in double
        const float rn = 1.f / float(nv);
        const float hs = ds * rn;
        const float E = opacity_bound<C>(sg, slot, dea, deb, INFINITY);
        // Eq. 2: n_inter = max(1, ceil(fl(fl(chi64 ds64) / dtau_max))); ds64, the
        // definition's sample spacing, is within (3u + rho_s) of hs, rho_s the
        // rounding of its interpolated distances (8 u64 max|Z| / hs)
        const float zmax = float(fmax(za, zb));
        const float kap = 15.f * kU + 9.0e-16f * zmax / hs + 1e-15f;
        const float dtm = float(a.dtau_max);
        sg.hq[slot] = 0.5f * hs;
        sg.thr[slot] = (dtm / hs) * (1.f - kap) - E * (1.f + 4.f * kU);
        const float qs = hs * float(1.0 / a.dtau_max);
        sg.qlo[slot] = qs * (1.f - kap);
        sg.qhi[slot] = qs * (1.f + kap);
        sg.E[slot] = E;
        return nv;
    }
}

// Whether line l takes no part in a sample of single precision, bit for bit:
// every bin of the warp gets chi = fma(c0, g, chi) = chi and eta likewise.
// A and B of the warp's bins lie in [wA[0], wA[1]] and [wB[0], wB[1]], and
// rounding is monotone, so fl(fl(B delta + A) rdv) of every bin lies between
// the same expression at the ends.  With |a| >= t on one side of zero,
// g <= 2^-t^2 (1 + kEEx2), and a product c0 g below half an ulp of chi, at
// least 2^-25 cc, rounds away: t^2 = 25.05 + log2(c0 / cc), likewise for eta,
// the margin covering lg2.approx, rcp.approx and this evaluation.  From
// |a| = 12.1 on ex2.approx.ftz(-a^2) is exactly 0, whatever the ratios.  On
// the 50 000-point wind the far wing then starts at |a'| of about 6.2
// instead of 12.1.
__device__ __forceinline__ bool line_is_far(float dl, float rdv, float cc, float ec, float c0, float e0,
                                            const float *wA, const float *wB) {
    if (c0 == 0.f && e0 == 0.f) return true;
    const float lo = fmaf(dl >= 0.f ? wB[0] : wB[1], dl, wA[0]) * rdv;
    const float hi = fmaf(dl >= 0.f ? wB[1] : wB[0], dl, wA[1]) * rdv;
    const float re = e0 > 0.f ? e0 * Ar<float>::rcp(ec) : 0.f;
    const float x = fmaxf(fmaxf(c0 * Ar<float>::rcp(cc), re), 1e-30f);
    const float t = fminf(sqrtf(fmaxf(25.05f + __log2f(x), 0.f)) * 1.0001f, 12.1f);
    return lo >= t || hi <= -t;
}

// The slot whose interval holds sample s_abs of the chunk: the last one whose
// samples start at or before it.
template <class C>
__device__ __forceinline__ int slot_of(const Stage<C> &sg, int s_abs, int nch) {
    int lo = 1, hi = nch;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sg.so[mid] <= s_abs) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The same for the double-precision integer form (far_profile).  The argument's
// range is formed in single precision; the margin on |a| covers its rounding.
__device__ __forceinline__ bool line_is_far(double dl, double rdv, double cc, double ec, double c0, double e0,
                                            const float *wA, const float *wB) {
    if (c0 == 0.0 && e0 == 0.0) return true;
    const float d = float(dl), rd = float(rdv);
    const float lo = fmaf(d >= 0.f ? wB[0] : wB[1], d, wA[0]) * rd;
    const float hi = fmaf(d >= 0.f ? wB[1] : wB[0], d, wA[1]) * rd;
    const float mar = 1e-6f * (fmaxf(fabsf(wA[0]), fabsf(wA[1])) + fmaxf(fabsf(wB[0]), fabsf(wB[1])) * fabsf(d)) * rd;
    const float t = far_profile(cc, ec, c0, e0);
    return lo - mar >= t || hi + mar <= -t;
}

// Record of the integer form: a quarter of the distance to the previous sample,
// eta_c / chi_c, chi_c, eta_c, the profile argument's two terms (a sample on
// which no line takes part: half the increment if it was so at the sample
// before too, and its sum with the one before), then chi0 and eta0 of each line.  One line: the argument of bin k is alpha + u_k gamma with
// u_k = (ub_k / span + 1) / 2 (the bin's velocity ub within its range +-span),
// alpha in Q6.57 and gamma scaled by the largest power
// of two that keeps it below 2^63 (the shift back in its lowest three bits),
// both from double products with their residuals, so that the cancellation
// between them costs nothing.  More lines, and one line where the origin's bins
// span 31 widths of the sample or the argument starts beyond what Q6.57 holds
// (kWide in `on`): delta and sqrt(log2 e) / dv.
// Returns the mask of the lines that take part, bit 31 set when some bin may
// need a split, bit 30 when the sample is outside what consume_int's arithmetic
// covers (consume_wide takes it, or plain_step).
constexpr unsigned kSplitBit = 0x80000000u, kWildBit = 0x40000000u, kLineBits = 0x3fffffffu;
constexpr unsigned kWide = 0x100u, kWideSplit = 0x200u;  // in `on`; kWideSplit: some bin may need a split

template <class C>
__device__ __forceinline__ unsigned gen_sample_int(Stage<C> &sg, int k, int nv, int j, int s_rec, int sign,
                                                   double dtau_max) {
    constexpr int NL = C::NL;
    double *o = sg.rec + s_rec * Stage<C>::kS;
    // as the definition lays the samples out: interpolated from the earlier point along +r
    const bool bwd = sign < 0;
    const double sgn = double(sign);
    const int b0 = bwd ? k - 1 : k, b1 = bwd ? k : k - 1;
    const int i = bwd ? j : nv - j, ip = bwd ? j - 1 : nv - j + 1;
    const double dn = double(nv);
    const float rn = Ar<float>::rcp(float(nv));
    auto frac = [&](int ii) -> double {  // ii / nv correctly rounded: the quotient with its residual added
        if (nv == 1) return 0.0;
        const double q = div_pos(double(ii), dn);
        return fma(fma(-q, dn, double(ii)), double(rn), q);
    };
    const double ti = frac(i), tp = frac(ip);
    auto at = [&](double x0, double x1, int ii, double t) -> double {
        return ii == 0 ? x0 : ii == nv ? x1 : __dadd_rn(x0, __dmul_rn(__dsub_rn(x1, x0), t));
    };
    const double s0 = sgn * sg.z[b0], s1 = sgn * sg.z[b1];
    const double ds = fabs(at(s0, s1, i, ti) - at(s0, s1, ip, tp));
    const double dl = at(sg.d[b0], sg.d[b1], i, ti), wv = at(sg.w[b0], sg.w[b1], i, ti);
    const double cc = at(sg.cc[b0], sg.cc[b1], i, ti), ec = at(sg.ec[b0], sg.ec[b1], i, ti);
    const double rs = div_pos(Ar<float>::kArgScale, wv);
    o[0] = 0.25 * ds;
    o[1] = div_pos(ec, cc);
    o[2] = cc;
    o[3] = ec;
    unsigned on = 0;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const double c0 = at(sg.ce[2 * l][b0], sg.ce[2 * l][b1], i, ti);
        const double e0 = at(sg.ce[2 * l + 1][b0], sg.ce[2 * l + 1][b1], i, ti);
        o[6 + 2 * l] = c0;
        o[7 + 2 * l] = e0;
        if (!line_is_far(dl, rs, cc, ec, c0, e0, sg.wA[l], sg.wB[l])) on |= 1u << l;
    }
    const double top = sg.hq[k];  // bound of chi on the interval
    unsigned cls = on;
    if (!(top * ds <= dtau_max * (1.0 - 0x1p-38))) cls |= kSplitBit;
    const bool wild = !(top * ds < 1e60) || !(cc > 1e-150);
    if constexpr (NL == 1) {
        if (on) {
            // gamma = 2 span (1 + delta/c) rs, alpha = delta rs - gamma / 2
            const double G = sg.span, q = G * (1.0 / kC);
            const double G1 = fma(q, dl, G), G1l = fma(q, dl, G - G1);
            const double gh = G1 * rs, gl = fma(G1, rs, -gh) + G1l * rs;
            const double ah = dl * rs, al = fma(dl, rs, -ah);
            const double am = ah - gh, z = am - ah;
            const double aml = ((ah - (am - z)) - (gh + z)) + (al - gl);
            const int ex = int(double_bits(gh) >> 52) - 1022;  // gh < 2^ex
            const int sh = ex < 1 ? 4 : ex > 5 ? 0 : 5 - ex;   // gamma 2^(57 + sh) = gh 2^(58 + sh) < 2^63
            const double up = bits_double(uint64_t(1023 + 58 + sh) << 52);
            const uint64_t g = uint64_t(__double2ll_rn(gh * up)) + uint64_t(__double2ll_rn(gl * up));
            o[4] = bits_double(uint64_t(__double2ll_rn(am * 0x1p57)) + uint64_t(__double2ll_rn(aml * 0x1p57)));
            o[5] = bits_double((g & ~uint64_t(7)) | uint64_t(sh));
            if (!(gh < 31.0 && gh >= 0.0 && am > -63.0 && am < 33.0) && !wild) {
                on |= cls & kSplitBit ? kWide | kWideSplit : kWide;
                cls |= kWildBit | kSplitBit;
                o[4] = dl;
                o[5] = rs;
            }
        }
    } else {
        o[4] = dl;
        o[5] = rs;
    }
    if (wild) {  // plain_step's layout: delta, dv
        cls |= kWildBit | kSplitBit;
        o[4] = dl;
        o[5] = wv;
    }
    sg.on[s_rec] = on;
    return cls;
}

// Record of sample s_abs of the chunk (relative to its first) into record s_rec.
// Returns (single precision) the mask of the lines that take part, bit 31 set when some bin may need a split.
template <class C>
__device__ __forceinline__ unsigned gen_sample(Stage<C> &sg, int s_abs, int s_rec, int nch, int sign,
                                               double dtau_max) {
    using R = typename C::R;
    constexpr int NL = C::NL;
    constexpr int kS = Stage<C>::kS;
    const int k = slot_of<C>(sg, s_abs, nch), nv = sg.nv[k], j = s_abs - sg.so[k] + 1;
    sg.sk[s_rec] = (unsigned char)k;
    if constexpr (sizeof(R) == 4) {
        const int pa = k - 1;
        float wv, dl, cc, ec, ce[2 * NL];
        if (j == nv) {
            dl = sg.d[k];
            wv = sg.w[k];
            cc = sg.cc[k];
            ec = sg.ec[k];
#pragma unroll
            for (int c = 0; c < 2 * NL; ++c) ce[c] = sg.ce[c][k];
        } else {
            const float t = float(j) * (1.f / float(nv));  // rn of the interval, formed again
            dl = fmaf(sg.d[k] - sg.d[pa], t, sg.d[pa]);
            wv = fmaf(sg.w[k] - sg.w[pa], t, sg.w[pa]);
            cc = fmaf(sg.cc[k] - sg.cc[pa], t, sg.cc[pa]);
            ec = fmaf(sg.ec[k] - sg.ec[pa], t, sg.ec[pa]);
#pragma unroll
            for (int c = 0; c < 2 * NL; ++c) ce[c] = fmaf(sg.ce[c][k] - sg.ce[c][pa], t, sg.ce[c][pa]);
        }
        const float rdv = Ar<float>::rcp(wv);
        // no bin can split anywhere on the interval when the largest opacity any
        // sample of it (or the point before it) can reach, continuum plus line
        // centres (the profile is at most 1; interpolation and the fused sums
        // round within (4 + NL) u), stays below the threshold: the record says so
        // with an infinite threshold and the step skips the vote
        float thr = sg.thr[k];
        float cb = fmaxf(sg.cc[pa], sg.cc[k]);
#pragma unroll
        for (int l = 0; l < NL; ++l) cb += fmaxf(sg.ce[2 * l][pa], sg.ce[2 * l][k]);
        if (cb * (1.f + (8 + 2 * NL) * kU) <= thr) thr = INFINITY;
        unsigned on = 0;  // the lines that take part
#pragma unroll
        for (int l = 0; l < NL; ++l)
            if (!line_is_far(dl, rdv, cc, ec, ce[2 * l], ce[2 * l + 1], sg.wA[l], sg.wB[l])) on |= 1u << l;
        if constexpr (C::kPacked) {
            float4 *o = reinterpret_cast<float4 *>(sg.rec + s_rec * kS);
            o[0] = make_float4(dl, dl, rdv, rdv);
            o[1] = make_float4(cc, cc, ec, ec);
            o[2] = make_float4(sg.hq[k], sg.hq[k], thr, __uint_as_float(on));
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                if constexpr (Rec<C>::kTwice)
                    o[3 + l] = make_float4(ce[2 * l], ce[2 * l], ce[2 * l + 1], ce[2 * l + 1]);
                else
                    reinterpret_cast<float2 *>(o + 3)[l] = make_float2(ce[2 * l], ce[2 * l + 1]);
            }
            return on | (thr != INFINITY ? 0x80000000u : 0u);
        } else {
            R *o = sg.rec + s_rec * kS;
            o[0] = dl;
            o[1] = NL == 1 && on == 0 ? -rdv : rdv;
            o[2] = cc;
            o[3] = ec;
            o[4] = sg.hq[k];
            o[5] = thr;
#pragma unroll
            for (int c = 0; c < 2 * NL; ++c) o[6 + c] = ce[c];
            return on | (thr != INFINITY ? 0x80000000u : 0u);
        }
    } else if constexpr (C::kInt) {
        return gen_sample_int<C>(sg, k, nv, j, s_rec, sign, dtau_max);
    } else {
        // the definition's layout: samples interpolated from the earlier point
        // along +r with t = i / nv, exact end points; ds between consecutive samples
        R *o = sg.rec + s_rec * kS;
        const bool bwd = sign < 0;
        const double sgn = double(sign);
        const int b0 = bwd ? k - 1 : k, b1 = bwd ? k : k - 1;
        const int i = bwd ? j : nv - j, ip = bwd ? j - 1 : nv - j + 1;
        auto at = [&](double x0, double x1, int ii) -> double {
            if (ii == 0) return x0;
            if (ii == nv) return x1;
            const double t = __ddiv_rn(double(ii), double(nv));
            return __dadd_rn(x0, __dmul_rn(__dsub_rn(x1, x0), t));
        };
        const double s0 = sgn * sg.z[b0], s1 = sgn * sg.z[b1];
        const double si = at(s0, s1, i), sp = at(s0, s1, ip);
        const double ds = bwd ? __dsub_rn(si, sp) : __dsub_rn(sp, si);
        o[0] = at(sg.d[b0], sg.d[b1], i);
        o[1] = 1.0 / at(sg.w[b0], sg.w[b1], i);
        o[2] = at(sg.cc[b0], sg.cc[b1], i);
        o[3] = at(sg.ec[b0], sg.ec[b1], i);
#pragma unroll
        for (int c = 0; c < 2 * NL; ++c) o[6 + c] = at(sg.ce[c][b0], sg.ce[c][b1], i);
        o[4] = 0.5 * ds;
        o[5] = (dtau_max / ds) * (1.0 - 0x1p-40);  // chi below this gives n_inter = 1
    }
    return 0u;
}

template <class C>
__device__ __forceinline__ void load_rec(const typename C::V *src, typename C::V (&v)[Stage<C>::kS]) {
    constexpr int kS = Stage<C>::kS;
    if constexpr (sizeof(typename C::V) == 4) {
#pragma unroll
        for (int c = 0; c < kS / 4; ++c) {
            const float4 t = reinterpret_cast<const float4 *>(src)[c];
            v[4 * c] = t.x;
            v[4 * c + 1] = t.y;
            v[4 * c + 2] = t.z;
            v[4 * c + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int c = 0; c < kS / 2; ++c) {
            const double2 t = reinterpret_cast<const double2 *>(src)[c];
            v[2 * c] = t.x;
            v[2 * c + 1] = t.y;
        }
    }
}

// Eq. 2's n_inter of one bin whose larger opacity cm may exceed the sample's
// threshold.  Double precision: as defined.  Single precision: certified from
// the bound E; 0 when the bound leaves the integer open (the caller has it
// redone in double precision).
template <class C>
__device__ __forceinline__ int n_inter(typename C::R cm, typename C::R hq, int k, const Stage<C> &sg,
                                       const SolveArgs &a) {
    using R = typename C::R;
    int n;
    if constexpr (sizeof(R) == 8) {
        const double nr = ceil((cm * (hq + hq)) / a.dtau_max);
        n = nr > double(kMaxSubdiv) ? kMaxSubdiv + 1 : nr <= 1.0 ? 1 : int(nr);
    } else {
        const float E = sg.E[k];
        const float nhi = ceilf((cm + E) * sg.qhi[k]);
        if (nhi <= 1.f) return 1;
        const float nlo = ceilf((cm - E) * sg.qlo[k]);
        if (nlo != nhi) return 0;
        n = nhi > float(kMaxSubdiv) ? kMaxSubdiv + 1 : int(nhi);
    }
    if (n > kMaxSubdiv) {
        dev_fail(a.status, kDevSubdivLimit);
        n = kMaxSubdiv;
    }
    return n;
}

// The Eq. 2 counts of sample s that its single-precision bound left open
// (sg.fix[i][lane] < 0), resolved into sg.fix: by a tighter bound, which leaves
// out the bins on which the line has no part (|a| >= 12.1, g = 0 in single
// precision and below 2^-146 in double), else in double precision.  With
// several lines the loop's bound carries their distance, hundreds of widths:
// on a two-line octree of 20 000 leaves the tighter one decides two thirds of
// the 5.6e5 open counts of a pass.  Out of line and outside the elimination
// loop, which it interrupts only for such a sample: a call inside the loop
// would cost the loop its registers.
template <class C>
__device__ __noinline__ void resolve_n_inter(Stage<C> &sg, const DevMesh &m, const DevLines &Ln, const SolveArgs &a,
                                             int sign, int s_abs) {
    const int lane = threadIdx.x & 31;
    const int k = sg.sk[s_abs % Stage<C>::kCap], j = s_abs - sg.so[k] + 1;
#pragma unroll 1
    for (int i = 0; i < C::BPL; ++i) {
        if (sg.fix[i][lane] >= 0) continue;
        if constexpr (sizeof(typename C::R) == 4) {
            const float cm = __int_as_float(sg.fix[i][lane] & 0x7fffffff);
            const float f0 = float(sg.r[0]), f1 = float(sg.r[1]), f2 = float(sg.r[2]);
            float de[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int id = sg.id[k - 1 + e];
                de[e] = id < 0 ? 0.f : delta_bound<C>(sg, __ldg(m.vxf + id), __ldg(m.vyf + id), __ldg(m.vzf + id), f0, f1, f2);
            }
            const float E = opacity_bound<C>(sg, k, de[0], de[1], 12.25f);
            const float nhi = ceilf((cm + E) * sg.qhi[k]), nlo = ceilf((cm - E) * sg.qlo[k]);
            if (nhi <= 1.f || nlo == nhi) {
                int n = nhi <= 1.f ? 1 : nhi > float(kMaxSubdiv) ? kMaxSubdiv + 1 : int(nhi);
                if (n > kMaxSubdiv) {
                    dev_fail(a.status, kDevSubdivLimit);
                    n = kMaxSubdiv;
                }
                sg.fix[i][lane] = n;
                continue;
            }
        }
        const int32_t b = lane_bin<C>(sg, i, lane);
        int n = redo_n_inter(m, Ln, sg.r, sg.vo, sg.o, double(sign), sg.id[k - 1], sg.id[k], sg.nv[k], j,
                             b < sg.NB ? b : sg.NB - 1, a.dtau_max);
        if (n > kMaxSubdiv) {
            dev_fail(a.status, kDevSubdivLimit);
            n = kMaxSubdiv;
        }
        sg.fix[i][lane] = n;
        atomicAdd(&sg.n_redo, 1u);
    }
    __syncwarp();
}

// The split counts (Eq. 2) of the lane's bins at a sample where some bin of
// the warp may need more than one.  Returns false, with the open bins marked
// in sg.fix, when a single-precision count is left open somewhere in the warp.
template <class C>
__device__ __forceinline__ bool split_counts(typename C::R hq, typename C::R thr, int s_abs, bool fixed,
                                             Stage<C> &sg, const SolveArgs &a, const typename C::V (&chi_q)[C::NV],
                                             const Sweep<typename C::V, typename C::W> (&w)[C::NV],
                                             int (&nis)[C::BPL]) {
    using R = typename C::R;
    const int lane = threadIdx.x & 31;
    const int k = sg.sk[s_abs % Stage<C>::kCap];
    bool open = false;
#pragma unroll
    for (int i = 0; i < C::BPL; ++i) {
        const R cm = fmax(vget(w[i / C::kIn].chi, i % C::kIn), vget(chi_q[i / C::kIn], i % C::kIn));
        int n = 1;
        if (cm > thr) {
            n = (fixed && sg.fix[i][lane] > 0) ? sg.fix[i][lane] : n_inter<C>(cm, hq, k, sg, a);
            open |= n == 0;
        }
        nis[i] = n;
        if constexpr (sizeof(R) == 4) {
            if (n == 0) nis[i] = __float_as_int(-cm);
        }
    }
    if constexpr (sizeof(R) == 4) {
        if (__any_sync(kFull, open)) {
#pragma unroll
            for (int i = 0; i < C::BPL; ++i) sg.fix[i][lane] = nis[i] < 0 ? nis[i] : 0;
            __syncwarp();
            return false;
        }
    }
    if (a.counters) {  // (uniform) only while profiling
        unsigned extra = 0;
#pragma unroll
        for (int i = 0; i < C::BPL; ++i)
            if (lane_bin<C>(sg, i, lane) < sg.NB) extra += unsigned(nis[i] - 1);
        extra = __reduce_add_sync(kFull, extra);
        if (lane == 0) sg.n_extra += extra;
    }
    return true;
}

// Packed form: words of a record, as pairs.
__device__ __forceinline__ void load_pair(const float2 *src, float2 &a, float2 &b) {
    const float4 t = *reinterpret_cast<const float4 *>(src);
    a = make_float2(t.x, t.y);
    b = make_float2(t.z, t.w);
}

// Packed form: the part of line l in a sample (record src) for every bin of
// the lane, A and B its profile constants.
template <class C>
__device__ __forceinline__ void one_line(const float2 *src, int l, float2 delta, float2 rdv, const float2 (&A)[C::NV],
                                         const float2 (&B)[C::NV], float2 (&chi_q)[C::NV], float2 (&eta_q)[C::NV]) {
    float2 c0, e0;
    if constexpr (Rec<C>::kTwice) {
        load_pair(src + 6 + 2 * l, c0, e0);
    } else {
        const float2 t = src[6 + l];
        c0 = make_float2(t.x, t.x);
        e0 = make_float2(t.y, t.y);
    }
#pragma unroll
    for (int i = 0; i < C::NV; ++i) add_line(delta, rdv, c0, e0, A[i], B[i], chi_q[i], eta_q[i]);
}

// Packed form: total opacity and emissivity of a sample for every bin of the
// lane, over the lines that take part (mask `on`, uniform over the warp).
template <class C>
__device__ __forceinline__ void all_lines(const float2 *src, unsigned on, const Stage<C> &sg, float2 (&chi_q)[C::NV],
                                          float2 (&eta_q)[C::NV]) {
    const int lane = threadIdx.x & 31;
    float2 delta, rdv, cc, ec;
    load_pair(src, delta, rdv);
    load_pair(src + 2, cc, ec);
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
        chi_q[i] = cc;
        eta_q[i] = ec;
    }
#pragma unroll 1
    for (; on; on &= on - 1) {
        const int l = C::NL == 1 ? 0 : __ffs(on) - 1;
        float2 A[C::NV], B[C::NV];
#pragma unroll
        for (int i = 0; i < C::NV; ++i) {
            A[i] = sg.fA[l][i][lane];
            B[i] = sg.fB[l][i][lane];
        }
        one_line<C>(src, l, delta, rdv, A, B, chi_q, eta_q);
    }
}

// Packed form: the rows of a sample without sub-intervals (hq: half its spacing).
template <class C>
__device__ __forceinline__ void rows_to(float2 hq, const float2 (&chi_q)[C::NV], const float2 (&eta_q)[C::NV],
                                        Sweep<float2> (&w)[C::NV]) {
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
        row2(w[i], w[i].chi, w[i].eta, vmul(hq, vadd(w[i].chi, chi_q[i])));
        w[i].chi = chi_q[i];
        w[i].eta = eta_q[i];
    }
}

// Packed form: one velocity sample (record src, sample s_abs of the chunk) of an
// interval on which some bin may need sub-intervals (Eq. 2, chi and eta
// linear).  Returns false, with nothing changed but the bins marked in sg.fix,
// when a count is left open somewhere in the warp; once it has been redone the
// sample is stepped again with `fixed` set, taking the counts from sg.fix.
template <class C>
__device__ __forceinline__ bool split_step(const float2 *src, int s_abs, bool fixed, Stage<C> &sg,
                                           const SolveArgs &a, Sweep<float2> (&w)[C::NV]) {
    float2 hq, tm;
    load_pair(src + 4, hq, tm);
    const float thr = tm.x;
    float2 chi_q[C::NV], eta_q[C::NV];
    all_lines<C>(src, __float_as_uint(tm.y), sg, chi_q, eta_q);
    float cm = 0.f;
#pragma unroll
    for (int i = 0; i < C::NV; ++i)
        cm = fmaxf(cm, fmaxf(fmaxf(w[i].chi.x, w[i].chi.y), fmaxf(chi_q[i].x, chi_q[i].y)));
    if (!__any_sync(kFull, cm > thr)) {
        rows_to<C>(hq, chi_q, eta_q, w);
        return true;
    }
    int nis[C::BPL];
    if (!split_counts<C>(hq.x, thr, s_abs, fixed, sg, a, chi_q, w, nis)) return false;
    // the sub-intervals of both bins of a value side by side, each bin taking its first n
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
        const int nx = nis[2 * i], ny = nis[2 * i + 1], n = nx > ny ? nx : ny;
        const float2 rni = make_float2(1.f / float(nx), 1.f / float(ny));
        const float2 hh = vmul(hq, rni);
        const float2 c0 = w[i].chi, e0 = w[i].eta;
        const float2 dchi = make_float2((chi_q[i].x - c0.x) * rni.x, (chi_q[i].y - c0.y) * rni.y);
        const float2 deta = make_float2((eta_q[i].x - e0.x) * rni.x, (eta_q[i].y - e0.y) * rni.y);
        float2 cprev = c0, eprev = e0;
#pragma unroll 1
        for (int k = 1; k <= n; ++k) {
            const float2 fk = make_float2(float(k), float(k));
            float2 ck = vfma(dchi, fk, c0), ek = vfma(deta, fk, e0);
            if (k >= nx) ck.x = chi_q[i].x, ek.x = eta_q[i].x;
            if (k >= ny) ck.y = chi_q[i].y, ek.y = eta_q[i].y;
            Sweep<float2> t = w[i];
            row2(t, cprev, eprev, vmul(hh, vadd(cprev, ck)));
            if (k <= nx) w[i].Fh.x = t.Fh.x, w[i].Dm.x = t.Dm.x, w[i].dtp.x = t.dtp.x, w[i].zh.x = t.zh.x;
            if (k <= ny) w[i].Fh.y = t.Fh.y, w[i].Dm.y = t.Dm.y, w[i].dtp.y = t.dtp.y, w[i].zh.y = t.zh.y;
            cprev = ck;
            eprev = ek;
        }
        w[i].chi = chi_q[i];
        w[i].eta = eta_q[i];
    }
    return true;
}

// The other forms: one velocity sample (record v, sample s_abs of the chunk) for every bin of the
// lane: line optics, Eq. 2 sub-intervals with linear chi and eta, elimination
// rows.  When no bin of the warp can need sub-intervals (the common case) the
// rows run as straight-line code, so the bins' chains interleave.  Single
// precision tests "possibly more than one sub-interval" on the lane's maximum
// of chi over its bins (this sample's and the previous one's) against the
// certified threshold; double precision per bin.  Returns false, with nothing
// changed, when a single-precision count is left open somewhere in the warp
// (sg.fix marks it); once it has been redone the sample is stepped again with
// `fixed` set, taking the counts from sg.fix.
template <class C>
__device__ __forceinline__ bool sample_step(const typename C::V (&v)[Stage<C>::kS], int s_abs, bool fixed, Stage<C> &sg,
                                            const SolveArgs &a, const Bin<typename C::V, C::NL> (&f)[C::NV],
                                            Sweep<typename C::V, typename C::W> (&w)[C::NV]) {
    using R = typename C::R;
    using P = typename C::P;
    constexpr int NL = C::NL;
    constexpr int BPL = C::BPL, ORD = C::ORD;
    const R dl = v[0], rdv = v[1], hq = v[4], thr = v[5];
    R chi_q[BPL], eta_q[BPL];
    if (sizeof(R) == 4 && NL == 1 && rdv < R(0)) {  // the line takes no part: the continuum
#pragma unroll
        for (int i = 0; i < BPL; ++i) {
            chi_q[i] = v[2];
            eta_q[i] = v[3];
        }
    } else {
#pragma unroll
        for (int i = 0; i < BPL; ++i) optics<R, NL>(dl, rdv, v[2], v[3], v + 6, f[i], chi_q[i], eta_q[i]);
    }
    bool go;  // no bin needs a split (n_inter = 1 for all)
    if constexpr (sizeof(R) == 4) {
        go = thr == R(INFINITY);  // uniform (the warp's record): no bin of the interval can split
        if (!go) {
            R cm = fmax(w[0].chi, chi_q[0]);
#pragma unroll
            for (int i = 1; i < BPL; ++i) cm = fmax(cm, fmax(w[i].chi, chi_q[i]));
            go = !__any_sync(kFull, cm > thr);
        }
    } else {
        bool split = false;
#pragma unroll
        for (int i = 0; i < BPL; ++i) split |= fmax(w[i].chi, chi_q[i]) > thr;
        go = !__any_sync(kFull, split);
    }
    if (go) {
#pragma unroll
        for (int i = 0; i < BPL; ++i) {
            R Sq = R(0);
            if constexpr (ORD == 4) Sq = Ar<R>::src(eta_q[i], chi_q[i]);
            row<ORD>(w[i], w[i].chi, w[i].eta, wide<P>(hq) * (wide<P>(w[i].chi) + wide<P>(chi_q[i])), w[i].Sc, Sq);
            w[i].chi = chi_q[i];
            w[i].eta = eta_q[i];
            w[i].Sc = Sq;
        }
        return true;
    }
    int nis[BPL];
    if (!split_counts<C>(hq, thr, s_abs, fixed, sg, a, chi_q, w, nis)) return false;
#pragma unroll
    for (int i = 0; i < BPL; ++i) {
        const int ni = nis[i];
        const R rni = R(1) / R(ni);
        const R hh = hq * rni;
        const R c0 = w[i].chi, e0 = w[i].eta;
        const R dchi = (chi_q[i] - c0) * rni, deta = (eta_q[i] - e0) * rni;
        R cprev = c0, eprev = e0, Sprev = w[i].Sc;
#pragma unroll 1
        for (int k = 1; k < ni; ++k) {
            const R ck = c0 + dchi * R(k), ek = e0 + deta * R(k);
            R Sk = R(0);
            if constexpr (ORD == 4) Sk = Ar<R>::src(ek, ck);
            row<ORD>(w[i], cprev, eprev, wide<P>(hh) * (wide<P>(cprev) + wide<P>(ck)), Sprev, Sk);
            cprev = ck;
            eprev = ek;
            Sprev = Sk;
        }
        R Sq = R(0);
        if constexpr (ORD == 4) Sq = Ar<R>::src(eta_q[i], chi_q[i]);
        row<ORD>(w[i], cprev, eprev, wide<P>(hh) * (wide<P>(cprev) + wide<P>(chi_q[i])), Sprev, Sq);
        w[i].chi = chi_q[i];
        w[i].eta = eta_q[i];
        w[i].Sc = Sq;
    }
    return true;
}

// The lane's sweep state to and from shared memory (D Fh kept as one value,
// read back as Fh = D Fh, D = 1).
template <class C>
__device__ __forceinline__ void put_sweep(Lane<C> &ln, const Sweep<typename C::V, typename C::W> (&w)[C::NV],
                                          int lane) {
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
        if constexpr (C::kPacked) ln.wp[0][i][lane] = vmul(w[i].Dm, w[i].Fh);
        else if constexpr (sizeof(typename C::P) != sizeof(typename C::R)) ln.wp[0][i][lane] = held_y(w[i].Y);
        else ln.wp[0][i][lane] = w[i].Dm * w[i].Fh;
        ln.wp[1][i][lane] = w[i].dtp;
        ln.wr[0][i][lane] = w[i].zh;
        ln.wr[1][i][lane] = w[i].chi;
        ln.wr[2][i][lane] = w[i].eta;
        if constexpr (C::ORD == 4) {
            ln.wr[3][i][lane] = w[i].Sp;
            ln.wr[4][i][lane] = w[i].Sc;
            ln.wr[5][i][lane] = w[i].hp;
        }
    }
}

template <class C>
__device__ __forceinline__ void get_sweep(const Lane<C> &ln, Sweep<typename C::V, typename C::W> (&w)[C::NV],
                                          int lane) {
    using V = typename C::V;
    using R = typename C::R;
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
        if constexpr (sizeof(typename C::P) != sizeof(typename C::R)) w[i].Y = hold_y(ln.wp[0][i][lane]);
        w[i].Fh = ln.wp[0][i][lane];
        w[i].Dm = vset<typename C::W>(1.f);
        w[i].dtp = ln.wp[1][i][lane];
        w[i].zh = ln.wr[0][i][lane];
        w[i].chi = ln.wr[1][i][lane];
        w[i].eta = ln.wr[2][i][lane];
        if constexpr (C::ORD == 4) {
            w[i].Sp = ln.wr[3][i][lane];
            w[i].Sc = ln.wr[4][i][lane];
            w[i].hp = ln.wr[5][i][lane];
            // the reciprocal of the last increment, formed again as the row formed it
            w[i].rh = w[i].hp < R(0) ? R(0) : Ar<R>::rcp(w[i].hp);
        } else {
            w[i].Sp = w[i].Sc = w[i].hp = w[i].rh = vset<V>(0.f);
        }
    }
}

template <class C>
__device__ __forceinline__ void get_bins(const Stage<C> &sg, Bin<typename C::V, C::NL> (&f)[C::NV], int lane) {
#pragma unroll
    for (int i = 0; i < C::NV; ++i) {
#pragma unroll
        for (int l = 0; l < C::NL; ++l) {
            f[i].A[l] = sg.fA[l][i][lane];
            f[i].B[l] = sg.fB[l][i][lane];
        }
    }
}

// Eliminate the samples of a staged chunk from sample `pos` on, generating the
// records kCap at a time (the round holding `pos` is already generated unless
// `fresh`).  The lane's state comes from and goes back to shared memory, so
// the registers hold it only here.  Returns the first sample not stepped
// (total when the chunk is done; else a sample whose single-precision Eq. 2
// count was left open, whose record round stays in place).  Kept out of line
// (one call per chunk): its loop then gets a register allocation of its own,
// unaffected by the calls of the code around it.  pend: a sample whose open
// counts have been redone into sg.fix (-1: none).
template <class C>
__device__ __noinline__ int consume_chunk(Stage<C> &sg, Lane<C> &ln, const SolveArgs &a, int total, int nch, int sign,
                                          int pos, int pend, bool fresh) {
    constexpr int kS = Stage<C>::kS, kCap = Stage<C>::kCap;
    const int lane = threadIdx.x & 31;
    Sweep<typename C::V, typename C::W> w[C::NV];
    Bin<typename C::V, C::NL> f[C::NV];
    get_sweep<C>(ln, w, lane);
    if constexpr (!C::kPacked) get_bins<C>(sg, f, lane);
    int r0 = pos / kCap * kCap, s = pos - r0;
#pragma unroll 1
    for (; r0 < total; r0 += kCap, s = 0, fresh = true) {
        const int nr = total - r0 < kCap ? total - r0 : kCap;
        if constexpr (C::kPacked) {
            // the round in runs of records on which no bin can split and the same lines take
            // part, so that the loops over the common classes (no line, one line) hold no
            // branch and the compiler interleaves one sample's optics with another's rows
            static_assert(kCap == 32, "one record per lane");
            unsigned m_split, m_new;
            if (fresh) {
                const unsigned cls = lane < nr ? gen_sample<C>(sg, r0 + lane, lane, nch, sign, a.dtau_max) : 0u;
                const unsigned up = __shfl_up_sync(kFull, cls, 1);
                m_split = __ballot_sync(kFull, cls >> 31);
                m_new = __ballot_sync(kFull, ((cls ^ up) & 0x7fffffffu) != 0u);
                if (lane == 0) {
                    sg.m_split = m_split;
                    sg.m_new = m_new;
                }
                __syncwarp();
            } else {
                m_split = sg.m_split;
                m_new = sg.m_new;
            }
            while (s < nr) {
                const float2 *src = sg.rec + s * kS;
                if ((m_split >> s) & 1u) {
                    if (!split_step<C>(src, r0 + s, r0 + s == pend, sg, a, w)) break;
                    ++s;
                    continue;
                }
                // the run ends at the next record that may split or has other lines
                const unsigned next = (m_split | m_new) & (0xfffffffeu << s);
                const int e = next ? min(__ffs(int(next)) - 1, nr) : nr;
                const float2 *end = sg.rec + e * kS;
                s = e;
                const unsigned on = __float_as_uint(src[5].y);
                float2 chi_q[C::NV], eta_q[C::NV];
                if (on == 0u) {
#pragma unroll 2
                    for (; src < end; src += kS) {
                        float2 cc, ec;
                        load_pair(src + 2, cc, ec);
#pragma unroll
                        for (int i = 0; i < C::NV; ++i) {
                            chi_q[i] = cc;
                            eta_q[i] = ec;
                        }
                        rows_to<C>(src[4], chi_q, eta_q, w);
                    }
                } else if (C::NL == 1 || (on & (on - 1)) == 0u) {
                    const int l = C::NL == 1 ? 0 : __ffs(int(on)) - 1;
                    float2 A[C::NV], B[C::NV];
#pragma unroll
                    for (int i = 0; i < C::NV; ++i) {
                        A[i] = sg.fA[l][i][lane];
                        B[i] = sg.fB[l][i][lane];
                    }
#pragma unroll 2
                    for (; src < end; src += kS) {
                        float2 delta, rdv, cc, ec;
                        load_pair(src, delta, rdv);
                        load_pair(src + 2, cc, ec);
#pragma unroll
                        for (int i = 0; i < C::NV; ++i) {
                            chi_q[i] = cc;
                            eta_q[i] = ec;
                        }
                        one_line<C>(src, l, delta, rdv, A, B, chi_q, eta_q);
                        rows_to<C>(src[4], chi_q, eta_q, w);
                    }
                } else {
#pragma unroll 1
                    for (; src < end; src += kS) {
                        all_lines<C>(src, on, sg, chi_q, eta_q);
                        rows_to<C>(src[4], chi_q, eta_q, w);
                    }
                }
            }
        } else if constexpr (sizeof(typename C::R) == 4 && sizeof(typename C::P) == 4) {
            // the scalar single-precision forms in runs too: records on which no bin can split,
            // with the continuum alone or with lines (12 000 points, Hermitian: 48.6 -> 42.9 ms;
            // with FP64 pivots, whose row is long, the one loop below is faster: 142 against 151)
            using R = typename C::R;
            static_assert(kCap == 32, "one record per lane");
            unsigned m_split, m_new;
            if (fresh) {
                const unsigned cls = lane < nr ? gen_sample<C>(sg, r0 + lane, lane, nch, sign, a.dtau_max) : 0u;
                const unsigned any = __ballot_sync(kFull, (cls & 0x7fffffffu) != 0u);
                m_split = __ballot_sync(kFull, cls >> 31);
                m_new = any ^ (any << 1);
                if (lane == 0) {
                    sg.m_split = m_split;
                    sg.m_new = m_new;
                    sg.m_wild = any;
                }
                __syncwarp();
            } else {
                m_split = sg.m_split;
                m_new = sg.m_new;
            }
            while (s < nr) {
                R v[kS];
                if ((m_split >> s) & 1u) {
                    load_rec<C>(sg.rec + s * kS, v);
                    if (!sample_step<C>(v, r0 + s, r0 + s == pend, sg, a, f, w)) break;
                    ++s;
                    continue;
                }
                const unsigned next = (m_split | m_new) & (0xfffffffeu << s);
                const int e = next ? min(__ffs(int(next)) - 1, nr) : nr;
                const bool lines = ((sg.m_wild >> s) & 1u) != 0u;
                auto rows = [&](const R (&chi_q)[C::BPL], const R (&eta_q)[C::BPL]) {
#pragma unroll
                    for (int i = 0; i < C::BPL; ++i) {
                        R Sq = R(0);
                        if constexpr (C::ORD == 4) Sq = Ar<R>::src(eta_q[i], chi_q[i]);
                        row<C::ORD>(w[i], w[i].chi, w[i].eta, v[4] * (w[i].chi + chi_q[i]), w[i].Sc, Sq);
                        w[i].chi = chi_q[i];
                        w[i].eta = eta_q[i];
                        w[i].Sc = Sq;
                    }
                };
                R chi_q[C::BPL], eta_q[C::BPL];
                if (lines) {
#pragma unroll 2
                    for (; s < e; ++s) {
                        load_rec<C>(sg.rec + s * kS, v);
#pragma unroll
                        for (int i = 0; i < C::BPL; ++i)
                            optics<R, C::NL>(v[0], v[1], v[2], v[3], v + 6, f[i], chi_q[i], eta_q[i]);
                        rows(chi_q, eta_q);
                    }
                } else {
#pragma unroll 2
                    for (; s < e; ++s) {
                        load_rec<C>(sg.rec + s * kS, v);
#pragma unroll
                        for (int i = 0; i < C::BPL; ++i) {
                            chi_q[i] = v[2];
                            eta_q[i] = v[3];
                        }
                        rows(chi_q, eta_q);
                    }
                }
            }
        } else {
            if (fresh) {
#pragma unroll 1
                for (int q = lane; q < nr; q += 32) gen_sample<C>(sg, r0 + q, q, nch, sign, a.dtau_max);
                __syncwarp();
            }
#pragma unroll 2
            for (; s < nr; ++s) {
                typename C::V v[kS];
                load_rec<C>(sg.rec + s * kS, v);
                if (!sample_step<C>(v, r0 + s, r0 + s == pend, sg, a, f, w)) break;
            }
        }
        if (s < nr) break;
        __syncwarp();
    }
    put_sweep<C>(ln, w, lane);
    __syncwarp();
    return r0 < total ? r0 + s : total;
}

// ---- the double-precision second-order form on the integer pipes -------------

// State of one bin: Y = D Fh and z of the scaled form above in homogeneous
// coordinates, Y = N / Q and z = W / Q, in which a row is linear and needs no
// reciprocal (dt the increment beyond the current sample, dtb its mean with the
// one before, S the current sample's source function):
//   N += dtb Q,  W += S dtb Q,  Q += dt N
// (D = Q / Q', so N' / Q' = D (dtb + Y) and W' / Q' = D (z + dtb S)).  Every
// term is positive (W's sign apart, which I_bdy may make negative), so nothing
// cancels; Q grows like e^tau and is scaled back when it passes 2^300.
struct IntSweep {
    double N, Q, W, T, S, h;  // T, S: opacity and source function of the current sample; h: half the last increment
};

__device__ __forceinline__ void int_rescale(IntSweep &w) {
    if (__double2hiint(w.Q) > 0x52b00000) {  // 2^300
        const double f = bits_double(uint64_t(2046 - (__double2hiint(w.Q) >> 20)) << 52);
        w.N *= f;
        w.Q *= f;
        w.W *= f;
    }
}

__device__ __forceinline__ void int_row(IntSweep &w, double S, double h, double b) {
    const double p = b * w.Q;  // b: dtb = the sum of the last half increment and this one
    w.N += p;
    w.W = fma(S, p, w.W);
    w.Q = fma(h, __hiloint2double(__double2hiint(w.N) + 0x100000, __double2loint(w.N)), w.Q);  // h 2N
    w.h = h;
    int_rescale(w);
}

// Opacity and emissivity of record src for bin i of the lane, over the lines in
// `on`; kDouble: the argument in double precision (more lines, or kWide).
template <class C, bool kDouble>
__device__ __forceinline__ void int_optics(const double *src, unsigned on, const Stage<C> &sg, const uint64_t *tab,
                                           int i, uint64_t u, double &chi, double &eta) {
    chi = src[2];
    eta = src[3];
    if constexpr (!kDouble) {
        if (!on) return;
        const double e = exp2_neg_sq(arg_magnitude(double_bits(src[4]), double_bits(src[5]), u), tab);
        chi = fma(src[6], e, chi);
        eta = fma(src[7], e, eta);
    } else {
        const int lane = threadIdx.x & 31;
#pragma unroll 1
        for (; on; on &= on - 1) {
            const int l = C::NL == 1 ? 0 : __ffs(int(on)) - 1;
            const double a = fabs(fma(sg.fB[l][i][lane], src[4], sg.fA[l][i][lane]) * src[5]);
            const double e = a < 31.0 ? exp2_neg_sq(uint64_t(__double2ll_rn(a * 0x1p57)), tab) : 0.0;
            chi = fma(src[6 + 2 * l], e, chi);
            eta = fma(src[7 + 2 * l], e, eta);
        }
    }
}

// A sample of an interval on which some bin may need sub-intervals (Eq. 2).
// The counts are the definition's: taken here where chi ds / dtau_max is
// farther than its rounding from an integer, else left open (false is
// returned, sg.fix marks the bins) and redone in the definition's own order.
template <class C, bool kDouble>
__device__ __forceinline__ bool int_split_step(const double *src, unsigned on, bool fixed, Stage<C> &sg,
                                               const SolveArgs &a, const uint64_t *tab,
                                               const uint64_t (&u)[C::BPL], IntSweep (&w)[C::BPL]) {
    const int lane = threadIdx.x & 31;
    double chi[C::BPL], eta[C::BPL];
    const double q = src[0];
    bool split = false;
#pragma unroll
    for (int i = 0; i < C::BPL; ++i) {
        int_optics<C, kDouble>(src, on, sg, tab, i, u[i], chi[i], eta[i]);
        split |= !(fmax(w[i].T, chi[i]) * (4.0 * q) <= a.dtau_max * (1.0 - 0x1p-45));
    }
    int n[C::BPL];
    if (__any_sync(kFull, split)) {
        bool open = false;
#pragma unroll
        for (int i = 0; i < C::BPL; ++i) {
            const double r = fmax(w[i].T, chi[i]) * (4.0 * q) / a.dtau_max;
            const double c = ceil(r);
            n[i] = c > double(kMaxSubdiv) ? kMaxSubdiv + 1 : c <= 1.0 ? 1 : int(c);
            const bool near = fabs(r - rint(r)) <= r * 0x1p-45 && r > 0.5;
            if (fixed && sg.fix[i][lane] > 0) {
                n[i] = sg.fix[i][lane];
            } else if (near) {
                n[i] = -1;
                open = true;
            } else if (n[i] > kMaxSubdiv) {
                dev_fail(a.status, kDevSubdivLimit);
                n[i] = kMaxSubdiv;
            }
        }
        if (__any_sync(kFull, open)) {
#pragma unroll
            for (int i = 0; i < C::BPL; ++i) sg.fix[i][lane] = n[i] < 0 ? -1 : 0;
            __syncwarp();
            return false;
        }
        if (a.counters) {
            unsigned extra = 0;
#pragma unroll
            for (int i = 0; i < C::BPL; ++i)
                if (lane_bin<C>(sg, i, lane) < sg.NB) extra += unsigned(n[i] - 1);
            extra = __reduce_add_sync(kFull, extra);
            if (lane == 0) sg.n_extra += extra;
        }
    } else {
#pragma unroll
        for (int i = 0; i < C::BPL; ++i) n[i] = 1;
    }
#pragma unroll
    for (int i = 0; i < C::BPL; ++i) {
        const double S = div_pos(eta[i], chi[i]);
        if (n[i] > 1) {  // chi and eta linear on the sub-intervals
            const double rn = 1.0 / double(n[i]), qs = q * rn;
            const double c0 = w[i].T, e0 = w[i].S * c0;
            const double dc = (chi[i] - c0) * rn, de = (eta[i] - e0) * rn;
            double cp = c0, Sp = w[i].S, h;
#pragma unroll 1
            for (int k = 1; k < n[i]; ++k) {
                const double ck = fma(dc, double(k), c0), ek = fma(de, double(k), e0);
                h = qs * (cp + ck);
                int_row(w[i], Sp, h, w[i].h + h);
                cp = ck;
                Sp = ek > 0.0 ? div_pos(ek, ck) : 0.0;
            }
            h = qs * (cp + chi[i]);
            int_row(w[i], Sp, h, w[i].h + h);
        } else {
            const double h = q * (w[i].T + chi[i]);
            int_row(w[i], w[i].S, h, w[i].h + h);
        }
        w[i].T = chi[i];
        w[i].S = S;
    }
    return true;
}

// Rows on which no line takes part are the same linear map for every bin:
//   (N, Q) -> ((1, b), (t, 1 + t b)) (N, Q),   W -> W + S b Q.
// Eight consecutive ones are composed into one map, six operations a bin in
// place of 32; the lanes hold one row each and compose them in three doubling
// steps (47 operations a round of records).  The map is held less the identity:
// an interval of many samples repeats one map, and its rounding, 2^-53 of 1, would
// add up block by block (-2e-14 of J over thousands of samples), where the sums
// with N and Q round differently each time.  A block starts at the third
// record of a run (the first two rows still depend on the bin), or where the
// last block ended.  Not where an increment is so large that the map's entries
// could leave the range of the state.  bound: the records at which a run
// begins.  Returns the records at which a block starts.
constexpr int kBlock = 8;

template <class C>
__device__ __forceinline__ unsigned compose_blocks(Stage<C> &sg, int lane, int nr, unsigned bound, bool far) {
    const double *o = sg.rec + lane * Stage<C>::kS;
    const unsigned ok = __ballot_sync(kFull, far && o[4] < 1e3);
    const int first = 31 - __clz(int(bound & (0xffffffffu >> (31 - lane))));  // of the lane's run (bit 0 is set)
    const int idx = lane - first;
    const unsigned need = 0xffu << lane;
    const bool start = idx >= 2 && (idx - 2) % kBlock == 0 && lane + kBlock <= nr && (ok & need) == need &&
                       (bound & (need & ~(1u << lane))) == 0u;
    const unsigned starts = __ballot_sync(kFull, start);
    if (starts == 0u) return 0u;
    double m11, m12 = 0.0, m21 = 0.0, m22 = 0.0, al, be = 0.0;
    if (lane > 1 && ((ok >> lane) & 1u)) {
        m12 = o[5];
        m21 = 2.0 * o[4];
        m22 = m21 * m12;
        be = o[1 - Stage<C>::kS] * m12;
    }
    {  // of single rows m11 and al are 0
        const double s12 = __shfl_down_sync(kFull, m12, 1), s21 = __shfl_down_sync(kFull, m21, 1);
        const double s22 = __shfl_down_sync(kFull, m22, 1), sb = __shfl_down_sync(kFull, be, 1);
        al = sb * m21;
        be = fma(sb, m22, sb + be);
        m11 = s12 * m21;
        const double n12 = fma(s12, m22, s12 + m12);
        m21 = fma(s22, m21, s21 + m21);
        m22 = fma(s21, m12, fma(s22, m22, s22 + m22));
        m12 = n12;
    }
#pragma unroll
    for (int d = 2; d < kBlock; d <<= 1) {
        const double s11 = __shfl_down_sync(kFull, m11, d), s12 = __shfl_down_sync(kFull, m12, d);
        const double s21 = __shfl_down_sync(kFull, m21, d), s22 = __shfl_down_sync(kFull, m22, d);
        const double sa = __shfl_down_sync(kFull, al, d), sb = __shfl_down_sync(kFull, be, d);
        al = fma(sa, m11, fma(sb, m21, sa + al));
        be = fma(sa, m12, fma(sb, m22, sb + be));
        const double n11 = fma(s11, m11, fma(s12, m21, s11 + m11)), n12 = fma(s11, m12, fma(s12, m22, s12 + m12));
        m21 = fma(s21, m11, fma(s22, m21, s21 + m21));
        m22 = fma(s21, m12, fma(s22, m22, s22 + m22));
        m11 = n11;
        m12 = n12;
    }
    if (start) {
        double *b = sg.blk[lane / kBlock];
        b[0] = m11;
        b[1] = m12;
        b[2] = m21;
        b[3] = m22;
        b[4] = al;
        b[5] = be;
    }
    return starts;
}

// The lane's state of the integer form to and from shared memory.
template <class C>
__device__ __forceinline__ void get_int(const Lane<C> &ln, IntSweep (&w)[C::BPL], int lane) {
#pragma unroll
    for (int i = 0; i < C::BPL; ++i) {
        w[i].N = ln.wp[0][i][lane];
        w[i].Q = 1.0;
        w[i].h = ln.wp[1][i][lane];
        w[i].W = ln.wr[0][i][lane];
        w[i].T = ln.wr[1][i][lane];
        w[i].S = ln.wr[2][i][lane];
    }
}

template <class C>
__device__ __forceinline__ void put_int(Lane<C> &ln, const IntSweep (&w)[C::BPL], int lane) {
#pragma unroll
    for (int i = 0; i < C::BPL; ++i) {
        ln.wp[0][i][lane] = div_pos(w[i].N, w[i].Q);
        ln.wp[1][i][lane] = w[i].h;
        ln.wr[0][i][lane] = copysign(div_pos(fabs(w[i].W), w[i].Q), w[i].W);
        ln.wr[1][i][lane] = w[i].T;
        ln.wr[2][i][lane] = w[i].S;
    }
}

// consume_chunk of the integer form.  Also returns at a sample that its
// arithmetic does not cover (sg.m_wild), for consume_wide or plain_step.
template <class C>
__device__ __noinline__ int consume_int(Stage<C> &sg, Lane<C> &ln, const SolveArgs &a, const uint64_t *tab, int total,
                                        int nch, int sign, int pos, int pend, bool fresh) {
    constexpr int kS = Stage<C>::kS, kCap = Stage<C>::kCap;
    const int lane = threadIdx.x & 31;
    IntSweep w[C::BPL];
    uint64_t u[C::BPL];
    get_int<C>(ln, w, lane);
#pragma unroll
    for (int i = 0; i < C::BPL; ++i) u[i] = C::NL == 1 ? sg.uk[i][lane] : 0;
    int r0 = pos / kCap * kCap, s = pos - r0;
#pragma unroll 1
    for (; r0 < total; r0 += kCap, s = 0, fresh = true) {
        const int nr = total - r0 < kCap ? total - r0 : kCap;
        unsigned m_split, m_new, m_wild, m_block;
        if (fresh) {
            const unsigned cls = lane < nr ? gen_sample<C>(sg, r0 + lane, lane, nch, sign, a.dtau_max) : 0u;
            const unsigned up = __shfl_up_sync(kFull, cls, 1);
            m_split = __ballot_sync(kFull, cls & kSplitBit);
            m_wild = __ballot_sync(kFull, cls & kWildBit);
            m_new = __ballot_sync(kFull, ((cls ^ up) & kLineBits) != 0u);
            if (lane == 0) {
                sg.m_split = m_split;
                sg.m_new = m_new;
                sg.m_wild = m_wild;
            }
            __syncwarp();
            if (lane > 0 && lane < nr && cls == 0u) {
                double *o = sg.rec + lane * kS;
                const double h = o[0] * (o[2 - kS] + o[2]);
                o[4] = h;
                o[5] = lane > 1 ? o[-kS] * (o[2 - 2 * kS] + o[2 - kS]) + h : h;
            }
            __syncwarp();
            m_block = compose_blocks<C>(sg, lane, nr, m_split | m_split << 1 | m_new | 1u,
                                        lane > 0 && lane < nr && cls == 0u);
            if (lane == 0) sg.m_block = m_block;
            __syncwarp();
        } else {
            m_split = sg.m_split;
            m_new = sg.m_new;
            m_wild = sg.m_wild;
            m_block = sg.m_block;
        }
        while (s < nr) {
            const double *src = sg.rec + s * kS;
            const unsigned on = sg.on[s];
            if ((m_split >> s) & 1u) {
                if ((m_wild >> s) & 1u) break;
                if (!int_split_step<C, (C::NL > 1)>(src, on, r0 + s == pend, sg, a, tab, u, w)) break;
                ++s;
                continue;
            }
            const unsigned next = (m_split | m_new) & (0xfffffffeu << s);
            const int e = next ? min(__ffs(int(next)) - 1, nr) : nr;
            const double *end = sg.rec + e * kS;
            const unsigned blocks = m_block >> s;
            const int s0 = s;
            s = e;
            if (on == 0u) {
                // the continuum: from the run's second sample on the increments are the same
                // for every bin, from the third their means too, and come with the record
                int k = 0;
#pragma unroll 1
                for (; src < end; src += kS, ++k) {
                    if ((blocks >> k) & 1u) {
                        const double *b = sg.blk[(s0 + k) / kBlock];
                        src += (kBlock - 1) * kS;  // to the block's last record
                        k += kBlock - 1;
#pragma unroll
                        for (int i = 0; i < C::BPL; ++i) {
                            const double N = w[i].N, Q = w[i].Q;
                            w[i].W = fma(b[4], N, fma(b[5], Q, w[i].W));
                            w[i].N = fma(b[0], N, fma(b[1], Q, N));
                            w[i].Q = fma(b[2], N, fma(b[3], Q, Q));
                            w[i].h = src[4];
                            w[i].T = src[2];
                            w[i].S = src[1];
                            int_rescale(w[i]);
                        }
                        continue;
                    }
#pragma unroll
                    for (int i = 0; i < C::BPL; ++i) {
                        const double h = k > 0 ? src[4] : src[0] * (w[i].T + src[2]);
                        int_row(w[i], w[i].S, h, k > 1 ? src[5] : w[i].h + h);
                        w[i].T = src[2];
                        w[i].S = src[1];
                    }
                }
            } else {
#pragma unroll 1
                for (; src < end; src += kS) {
#pragma unroll
                    for (int i = 0; i < C::BPL; ++i) {
                        double chi, eta;
                        int_optics<C, (C::NL > 1)>(src, on, sg, tab, i, u[i], chi, eta);
                        const double h = src[0] * (w[i].T + chi);
                        int_row(w[i], w[i].S, h, w[i].h + h);
                        w[i].T = chi;
                        w[i].S = div_pos(eta, chi);
                    }
                }
            }
        }
        if (s < nr) break;
        __syncwarp();
    }
    put_int<C>(ln, w, lane);
    __syncwarp();
    return r0 < total ? r0 + s : total;
}

// Of one line: the kWide samples from `pos` on that follow one another in the
// round, the profile argument in double precision.  Returns the sample after
// them, or the complement of one whose count was left open (int_split_step).  A
// function of its own: in consume_int's loop the choice cost every other sample
// (4001-point wind 101.3 -> 102.2 ms).  A slow wind of 4001 points, widths spread
// by 10 either way, bins to 4 and 16 widths: 67 -> 47 and 107 -> 52 ms against the
// plain step for every such sample.
template <class C>
__device__ __noinline__ int consume_wide(Stage<C> &sg, Lane<C> &ln, const SolveArgs &a, const uint64_t *tab, int total,
                                         int pos, int pend) {
    constexpr int kS = Stage<C>::kS, kCap = Stage<C>::kCap;
    const int lane = threadIdx.x & 31;
    IntSweep w[C::BPL];
    get_int<C>(ln, w, lane);
    const uint64_t none[C::BPL] = {};
    const int r0 = pos / kCap * kCap, nr = total - r0 < kCap ? total - r0 : kCap;
    int s = pos - r0;
    bool open = false;
#pragma unroll 1
    for (; s < nr && (sg.on[s] & kWide) != 0u; ++s) {
        const double *src = sg.rec + s * kS;
        if (sg.on[s] & kWideSplit) {
            open = !int_split_step<C, true>(src, 1u, r0 + s == pend, sg, a, tab, none, w);
            if (open) break;
            continue;
        }
#pragma unroll
        for (int i = 0; i < C::BPL; ++i) {
            double chi, eta;
            int_optics<C, true>(src, 1u, sg, tab, i, 0, chi, eta);
            const double h = src[0] * (w[i].T + chi);
            int_row(w[i], w[i].S, h, w[i].h + h);
            w[i].T = chi;
            w[i].S = div_pos(eta, chi);
        }
    }
    put_int<C>(ln, w, lane);
    __syncwarp();
    return open ? ~(r0 + s) : r0 + s;
}

// One sample of the integer form outside what its fixed-point arithmetic
// covers (optical depths beyond 1e60, continua below 1e-150, source functions
// beyond 2^290): the plain double-precision step.
template <class C>
__device__ __noinline__ void plain_step(Stage<C> &sg, Lane<C> &ln, const SolveArgs &a, int s_abs) {
    constexpr int NL = C::NL;
    const int lane = threadIdx.x & 31;
    const double *src = sg.rec + s_abs % Stage<C>::kCap * Stage<C>::kS;
    const double hq = 2.0 * src[0], rdv = 1.0 / src[5];
#pragma unroll 1
    for (int i = 0; i < C::BPL; ++i) {
        Bin<double, NL> f;
        double ce[2 * NL], chi, eta;
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            f.A[l] = sg.fA[l][i][lane];
            f.B[l] = sg.fB[l][i][lane];
            ce[2 * l] = src[6 + 2 * l];
            ce[2 * l + 1] = src[7 + 2 * l];
        }
        optics<double, NL>(src[4], rdv, src[2], src[3], ce, f, chi, eta);
        Sweep<double> w;
        w.Fh = ln.wp[0][i][lane];
        w.Dm = 1.0;
        w.dtp = ln.wp[1][i][lane];
        w.zh = ln.wr[0][i][lane];
        const double c0 = ln.wr[1][i][lane], e0 = ln.wr[2][i][lane] * c0;
        const double r = ceil(fmax(c0, chi) * (hq + hq) / a.dtau_max);
        int n = r > double(kMaxSubdiv) ? kMaxSubdiv + 1 : r <= 1.0 ? 1 : int(r);
        if (n > kMaxSubdiv) {
            dev_fail(a.status, kDevSubdivLimit);
            n = kMaxSubdiv;
        }
        if (n > 1 && lane_bin<C>(sg, i, lane) < sg.NB) atomicAdd(&sg.n_extra, unsigned(n - 1));
        const double rn = 1.0 / double(n), hh = hq * rn, dc = (chi - c0) * rn, de = (eta - e0) * rn;
        double cp = c0, ep = e0;
#pragma unroll 1
        for (int k = 1; k <= n; ++k) {
            const double ck = k == n ? chi : c0 + dc * double(k), ek = k == n ? eta : e0 + de * double(k);
            row<2>(w, cp, ep, hh * (cp + ck), 0.0, 0.0);
            cp = ck;
            ep = ek;
        }
        ln.wp[0][i][lane] = w.Dm * w.Fh;
        ln.wp[1][i][lane] = w.dtp;
        ln.wr[0][i][lane] = w.zh;
        ln.wr[1][i][lane] = chi;
        ln.wr[2][i][lane] = eta / chi;
    }
    __syncwarp();
}

// Copy the point data of slot `from` into slot 0 (the next chunk's farther point).
template <class C>
__device__ __forceinline__ void carry_slot(Stage<C> &sg, int from) {
    using R = typename C::R;
    constexpr int NL = C::NL;
    sg.d[0] = sg.d[from];
    sg.w[0] = sg.w[from];
    sg.cc[0] = sg.cc[from];
    sg.ec[0] = sg.ec[from];
#pragma unroll
    for (int c = 0; c < 2 * NL; ++c) sg.ce[c][0] = sg.ce[c][from];
    if constexpr (sizeof(R) == 8) sg.z[0] = sg.z[from];  // single precision: carried by stage_chunk
    sg.id[0] = sg.id[from];
}

// Stage the chunk of points qb .. qb+nch-1 of the half (slot 0 already holds
// the point farther than the chunk): points, intervals, and the offsets of
// their velocity samples.  Returns the chunk's number of samples.  Called once
// per 32 points and kept out of line, so that its double-precision and bound
// arithmetic does not add to the registers of the elimination loop.
template <class C>
__device__ __noinline__ int stage_chunk(const DevMesh &m, const DevLines &Ln, const SolveArgs &a, Stage<C> &sg,
                                        int32_t qb, int32_t cnt, int sign) {
    using R = typename C::R;
    const int lane = threadIdx.x & 31;
    const int32_t npt = cnt + 1;
    const int nch = npt - qb < 32 ? int(npt - qb) : 32;
    const int slot = lane + 1;
    const int32_t q = qb + lane;
    double zq = 0.0;
    R deq = R(0);
    if (lane < nch) stage_point<C>(m, Ln, sg, q, cnt, slot, sign, zq, deq);
    // the farther point's Z and delta bound: the previous lane's, or the carried point's for lane 0
    double zf = __shfl_up_sync(kFull, zq, 1);
    R def = __shfl_up_sync(kFull, deq, 1);
    if (lane == 0) {
        zf = sg.z[0];
        if constexpr (sizeof(R) == 4) def = sg.de0;
    }
    __syncwarp();
    if constexpr (sizeof(R) == 4) {
        if (lane == nch - 1) {  // the next chunk's farther point
            sg.z[0] = zq;
            sg.de0 = deq;
        }
    }
    int nvk = 0;  // the far end (q = 0) starts the line: no interval
    if (lane < nch && q > 0) nvk = stage_interval<C>(m, Ln, a, sg, slot, sign, zf, zq, def, deq);
    int incl = nvk;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, sh);
        if (lane >= sh) incl += t;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    if (lane < nch) {
        sg.nv[slot] = nvk;
        sg.so[slot] = incl - nvk;
    }
    if (lane == 0) sg.n_smp += unsigned(total);
    __syncwarp();
    return total;
}

// Eliminate one half of a pair line (direction sign r) from its far end up to
// (excluding) the origin row.  Leaves the origin row's coupling (D Fh, zh)
// and the last optical-depth increment in the lane's sweep state.
template <class C>
__device__ void half_sweep(const DevMesh &m, const DevLines &Ln, const SolveArgs &a, Stage<C> &sg, Lane<C> &ln,
                           int sign, const uint64_t *tab) {
    using R = typename C::R;
    using V = typename C::V;
    constexpr int NL = C::NL;
    const int lane = threadIdx.x & 31;
    {
        Sweep<V, typename C::W> w[C::NV];
#pragma unroll
        for (int i = 0; i < C::NV; ++i) {
            w[i].Fh = w[i].Dm = vset<typename C::W>(1.f);
            w[i].dtp = vset<typename C::W>(0.f);
            if constexpr (C::kPacked) w[i].zh = vset<V>(float(a.I_bdy));
            else w[i].zh = R(a.I_bdy);
            w[i].hp = vset<V>(-1.f);  // no row yet (Hermitian scheme)
            w[i].Sp = w[i].Sc = w[i].rh = w[i].chi = w[i].eta = vset<V>(0.f);
            w[i].Y = hold_y(1.0);
        }
        put_sweep<C>(ln, w, lane);
    }
    const int32_t cnt = sg.hl.cnt;
    __syncwarp();
    if (cnt == 0) return;
#pragma unroll 1
    for (int32_t qb = 0; qb <= cnt; qb += 32) {
        const int total = stage_chunk<C>(m, Ln, a, sg, qb, cnt, sign);
        const int nch = cnt + 1 - qb < 32 ? int(cnt + 1 - qb) : 32;
        if (qb == 0) {  // the far end: its optics; its row follows with the first increment
            R ce[2 * NL];
#pragma unroll
            for (int c = 0; c < 2 * NL; ++c) ce[c] = sg.ce[c][1];
            const R rdv = Ar<R>::rcp(sg.w[1]);
#pragma unroll
            for (int i = 0; i < C::BPL; ++i) {
                Bin<R, NL> f;
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    f.A[l] = vget(sg.fA[l][i / C::kIn][lane], i % C::kIn);
                    f.B[l] = vget(sg.fB[l][i / C::kIn][lane], i % C::kIn);
                }
                R chi, eta;
                optics<R, NL>(sg.d[1], rdv, sg.cc[1], sg.ec[1], ce, f, chi, eta);
                vput(ln.wr[1][i / C::kIn][lane], i % C::kIn, chi);
                vput(ln.wr[2][i / C::kIn][lane], i % C::kIn, C::kInt ? eta / chi : eta);
                if constexpr (C::ORD == 4) ln.wr[4][i][lane] = Ar<R>::src(eta, chi);
            }
            __syncwarp();
        }
        int pos = 0, pend = -1;
        bool fresh = true;
#pragma unroll 1
        for (;;) {
            if constexpr (C::kInt) {
                pos = consume_int<C>(sg, ln, a, tab, total, nch, sign, pos, pend, fresh);
                if (pos >= total) break;
                if ((sg.m_wild >> pos % Stage<C>::kCap) & 1u) {
                    int next = pos + 1;  // the complement of a sample left open
                    if (NL == 1 && (sg.on[pos % Stage<C>::kCap] & kWide) != 0u) {
                        if constexpr (NL == 1) next = consume_wide<C>(sg, ln, a, tab, total, pos, pend);
                    } else {
                        plain_step<C>(sg, ln, a, pos);
                    }
                    pos = next < 0 ? ~next : next;
                    if (pos >= total) break;
                    if (next >= 0) {
                        fresh = pos % Stage<C>::kCap == 0;
                        continue;
                    }
                }
            } else {
                pos = consume_chunk<C>(sg, ln, a, total, nch, sign, pos, pend, fresh);
                if (pos >= total) break;
            }
            resolve_n_inter<C>(sg, m, Ln, a, sign, pos);
            pend = pos;
            fresh = false;
        }
        if (lane == 0) carry_slot<C>(sg, nch);
        __syncwarp();
    }
}

// CTAs of 4 warps (2 in the double-precision Hermitian form, whose per-warp
// stage is twice as large); the minimum resident CTAs per SM caps the registers
// (65536 / (threads x CTAs)).  The packed form: 8 for one line (64 registers,
// 25 KB of shared memory each; the 50 000-point step takes 92.6 ms with 7, 89.9
// with 8, 91.4 with 9, where the loop spills), 7 and 6 for two and four lines,
// bounded by the staging.
template <class C>
struct Occ {
    static constexpr int NL = C::NL;
    static constexpr int kWarps = sizeof(typename C::R) == 8 && !C::kInt ? 2 : 4;
    static constexpr int kThreads = 32 * kWarps;
    static constexpr int kMinBlocks =
        C::kInt ? (NL == 1 ? 4 : NL <= 2 ? 3 : 2)
        : sizeof(typename C::R) == 8 ? 1
        : sizeof(typename C::P) == 8 ? (NL == 1 ? 4 : 2)
        : C::BPL == 4 ? 5
        : C::kPacked ? (NL == 1 ? 8 : NL == 2 ? 7 : NL <= 4 ? 6 : 4)
        : (NL == 1 ? 9 : NL == 2 ? 8 : NL <= 4 ? 6 : 3);
};

// J of origin a.o_begin + oc for the bins of frequency tile vt / a.parts, by one
// warp (a.parts > 1: u of its share vt % a.parts of the pairs).
template <class C>
__device__ __forceinline__ void solve_item(const DevMesh &m, const DevLines &Ln, const DevRays &Rs,
                                           const SolveArgs &a, int32_t oc, int32_t vt, Stage<C> &sg, Lane<C> &ln,
                                           int lane, const uint64_t *tab) {
    const int32_t tile = a.parts > 1 ? vt / a.parts : vt, part = vt - tile * a.parts;
    using R = typename C::R;
    using P = typename C::P;
    constexpr int NL = C::NL, BPL = C::BPL, ORD = C::ORD;
    const int32_t o = a.o_begin + oc;
    const int32_t L = Ln.L, F = Ln.F, NB = L * F;
    const double dvo = Ln.dvw[o];
    if (lane == 0) {
        sg.o = o;
        sg.NB = NB;
        sg.tile = tile;
        sg.xo[0] = m.x[o];
        sg.xo[1] = m.y[o];
        sg.xo[2] = m.z[o];
        sg.vo[0] = m.vx[o];
        sg.vo[1] = m.vy[o];
        sg.vo[2] = m.vz[o];
        sg.vor[0] = Pts<R>::vx(m)[o];
        sg.vor[1] = Pts<R>::vy(m)[o];
        sg.vor[2] = Pts<R>::vz(m)[o];
        sg.n_smp = sg.n_extra = sg.n_redo = 0u;
        sg.span = Ln.x_span * dvo;
    }
    // the origin's own optics give S_o
    R oce[2 * NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        oce[2 * l] = l < L ? __ldg(Pts<R>::chi0(Ln) + int64_t(o) * L + l) : R(0);
        oce[2 * l + 1] = l < L ? __ldg(Pts<R>::eta0(Ln) + int64_t(o) * L + l) : R(0);
    }
    const R rdvo = Ar<R>::rcp(__ldg(Pts<R>::dvw(Ln) + o));

    // frequency of each bin of this lane and its profile constants
    R So_[BPL];  // the source function at the origin of each bin
    float lA[NL][2], lB[NL][2];  // the smallest and largest A and B of each line over the lane's bins
#pragma unroll
    for (int i = 0; i < BPL; ++i) {
        const int32_t b = tile * 32 * BPL + lane + 32 * i;
        const int32_t bb = b < NB ? b : NB - 1;
        const int32_t l = bb / F, k = bb % F;
        const double x = (F == 1) ? 0.0 : -Ln.x_span + 2.0 * Ln.x_span * double(k) / double(F - 1);
        const double ub = x * dvo;
        if constexpr (C::kInt && NL == 1) {  // (ub / span + 1) / 2 in Q0.63, with the quotient's residual
            const double G = Ln.x_span * dvo, G2 = 2.0 * G, t = ub + G, tl = ub - (t - G);
            const double q = t / G2, r = (fma(-q, G2, t) + tl) / G2;
            long long u = 1ll << 62;
            if (G > 0.0) {
                u = q >= 1.0 ? INT64_MAX : __double2ll_rn(q * 0x1p63) + __double2ll_rn(r * 0x1p63);
                if (u < 0) u = 0;
            }
            sg.uk[i][lane] = uint64_t(u);
        }
        Bin<R, NL> f;
#pragma unroll
        for (int lp = 0; lp < NL; ++lp) {
            const double r = (lp < L) ? Ln.ratio[l * MGX_MAX_LINES + lp] : 1.0;
            f.A[lp] = R((kC * (r - 1.0) + r * ub) * Ar<R>::kArgScale);
            f.B[lp] = R(r * (1.0 + ub / kC) * Ar<R>::kArgScale);
            vput(sg.fA[lp][i / C::kIn][lane], i % C::kIn, f.A[lp]);
            vput(sg.fB[lp][i / C::kIn][lane], i % C::kIn, f.B[lp]);
            const float fa = float(f.A[lp]), fb = float(f.B[lp]);
            lA[lp][0] = i == 0 ? fa : fminf(lA[lp][0], fa);
            lA[lp][1] = i == 0 ? fa : fmaxf(lA[lp][1], fa);
            lB[lp][0] = i == 0 ? fb : fminf(lB[lp][0], fb);
            lB[lp][1] = i == 0 ? fb : fmaxf(lB[lp][1], fb);
        }
        R chi_o, eta_o;
        optics<R, NL>(R(0), rdvo, __ldg(Pts<R>::chic(Ln) + o), __ldg(Pts<R>::etac(Ln) + o), oce, f, chi_o, eta_o);
        So_[i] = eta_o / chi_o;
    }
    if constexpr (sizeof(R) == 4 || C::kInt) {
        // the ranges of A and B over the warp's bins (line_is_far) and the largest
        // |A|, |B| (the opacity bound of Eq. 2)
#pragma unroll
        for (int lp = 0; lp < NL; ++lp) {
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) {
                lA[lp][0] = fminf(lA[lp][0], __shfl_xor_sync(kFull, lA[lp][0], sh));
                lA[lp][1] = fmaxf(lA[lp][1], __shfl_xor_sync(kFull, lA[lp][1], sh));
                lB[lp][0] = fminf(lB[lp][0], __shfl_xor_sync(kFull, lB[lp][0], sh));
                lB[lp][1] = fmaxf(lB[lp][1], __shfl_xor_sync(kFull, lB[lp][1], sh));
            }
            if (lane == 0) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    sg.wA[lp][e] = lA[lp][e];
                    sg.wB[lp][e] = lB[lp][e];
                }
                sg.Am[lp] = fmaxf(fabsf(lA[lp][0]), fabsf(lA[lp][1]));
                sg.Bm[lp] = fmaxf(fabsf(lB[lp][0]), fabsf(lB[lp][1]));
            }
        }
    }

    const int64_t h0 = int64_t(oc) * Rs.npairs * 2;
    double js[BPL], jc[BPL];  // each bin's J: Neumaier sum and compensation
    P cpD[BPL], cpT[BPL];     // the backward half's coupling to the origin row: D Fh, dtb / 2,
    R cpZ[BPL], cpH[BPL], cpS[BPL];  // zh (Hermitian: + the last increment and S)
#pragma unroll
    for (int i = 0; i < BPL; ++i) js[i] = jc[i] = 0.0;
#pragma unroll 1
    for (int32_t p = int32_t(int64_t(Rs.npairs) * part / a.parts),
                 p1 = int32_t(int64_t(Rs.npairs) * (part + 1) / a.parts);
         p < p1; ++p) {
        const uint32_t ray = __ldg(Rs.rays + int64_t(o) * Rs.npairs + p);
        const int lev = int(ray >> 28);
        const int64_t hb = h0 + 2 * int64_t(p);
        if (lane < 3) sg.r[lane] = Rs.dir[3 * (level_offset(lev) + (ray & 0x0FFFFFFFu)) + lane];
        if (lane == 0) sg.hl = half_list(a, hb);
        __syncwarp();
        half_sweep<C>(m, Ln, a, sg, ln, -1, tab);
#pragma unroll
        for (int i = 0; i < BPL; ++i) {  // the backward half's coupling to the origin row
            const int v = i / C::kIn, c = i % C::kIn;
            cpD[i] = vget(ln.wp[0][v][lane], c);  // D Fh
            cpT[i] = vget(ln.wp[1][v][lane], c);  // dtb / 2
            cpZ[i] = vget(ln.wr[0][v][lane], c);  // zh
            if constexpr (ORD == 4) {
                cpH[i] = ln.wr[5][i][lane];  // hp
                cpS[i] = ln.wr[3][i][lane];  // Sp
            }
        }
        if (lane == 0) sg.hl = half_list(a, hb + 1);
        __syncwarp();
        half_sweep<C>(m, Ln, a, sg, ln, 1, tab);
        const double w2 = a.w2[lev];
#pragma unroll
        for (int i = 0; i < BPL; ++i) {
            const int v = i / C::kIn, c = i % C::kIn;
            Sweep<R, P> wf, wb;
            wf.Fh = vget(ln.wp[0][v][lane], c);
            wf.Dm = P(1);
            wf.dtp = vget(ln.wp[1][v][lane], c);
            wf.zh = vget(ln.wr[0][v][lane], c);
            if constexpr (ORD == 4) {
                wf.Sp = ln.wr[3][i][lane];
                wf.hp = ln.wr[5][i][lane];
                wf.rh = wf.hp < R(0) ? R(0) : Ar<R>::rcp(wf.hp);
            }
            wb.Fh = cpD[i];
            wb.Dm = P(1);
            wb.dtp = cpT[i];
            wb.zh = cpZ[i];
            if constexpr (ORD == 4) {
                wb.hp = cpH[i];
                wb.Sp = cpS[i];
                wb.rh = wb.hp < R(0) ? R(0) : Ar<R>::rcp(wb.hp);
            }
            const R So = So_[i];
            const R u = ORD == 4 ? origin_u4(wb, wf, So, R(a.I_bdy)) : origin_u2(wb, wf, So);
            const int32_t b = lane_bin<C>(sg, i, lane);
            if (a.u_out && b < NB) a.u_out[(int64_t(oc) * Rs.npairs + p) * NB + b] = double(u);
            const double xv = w2 * double(u);
            const double sum = js[i];
            const double t = sum + xv;  // Neumaier compensated sum
            if (fabs(sum) >= fabs(xv)) jc[i] += (sum - t) + xv;
            else jc[i] += (xv - t) + sum;
            js[i] = t;
        }
        __syncwarp();
    }
    unsigned n_act = 0;
#pragma unroll
    for (int i = 0; i < BPL; ++i) {
        const int32_t b = lane_bin<C>(sg, i, lane);
        if (b < NB) {
            if (a.parts == 1) a.J[int64_t(o) * NB + b] = js[i] + jc[i];
            ++n_act;
        }
    }
    if (a.counters) {
        // [0]: sub-intervals beyond one per sample (active bins); [1]: samples x active bins;
        // [4]: integer decisions redone in double precision
        unsigned long long na = n_act;
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1) na += __shfl_down_sync(kFull, na, sh);
        __syncwarp();
        if (lane == 0) {
            atomicAdd(a.counters, (unsigned long long)sg.n_extra);
            atomicAdd(a.counters + 1, (unsigned long long)sg.n_smp * na);
            atomicAdd(a.counters + 4, (unsigned long long)sg.n_redo);
        }
    }
}

// 2^(j/1024) in shared memory, after the warps' staging (the integer form).
__device__ const Exp2Table d_exp2_table{};

template <class C>
__device__ __forceinline__ const uint64_t *load_table(unsigned char *smem) {
    if constexpr (C::kInt) {
        uint64_t *tab = reinterpret_cast<uint64_t *>(smem + (sizeof(Stage<C>) + sizeof(Lane<C>)) * Occ<C>::kWarps);
        for (int j = threadIdx.x; j < 1024; j += Occ<C>::kThreads) tab[j] = d_exp2_table.v[j];
        __syncthreads();
        return tab;
    } else {
        return nullptr;
    }
}

// Grid-mapped launch: warp w of the grid solves item w = (oc * n_tiles + tile) * parts + part.
template <class C>
__global__ void __launch_bounds__(Occ<C>::kThreads, (Occ<C>::kMinBlocks))
k_solve(const __grid_constant__ DevMesh m, const __grid_constant__ DevLines Ln, const __grid_constant__ DevRays Rs,
        const __grid_constant__ SolveArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    Stage<C> *stage = reinterpret_cast<Stage<C> *>(smem);  // one per warp
    Lane<C> *lanes = reinterpret_cast<Lane<C> *>(smem + sizeof(Stage<C>) * Occ<C>::kWarps);
    const uint64_t *tab = load_table<C>(smem);
    const int lane = threadIdx.x & 31;
    const int64_t item = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
    const int64_t per = int64_t(a.n_tiles) * a.parts;
    if (item >= (a.o_end - a.o_begin) * per) return;
    solve_item<C>(m, Ln, Rs, a, int32_t(item / per), int32_t(item % per), stage[threadIdx.x >> 5],
                  lanes[threadIdx.x >> 5], lane, tab);
}

// Persistent launch over a work list of (model, origin, tile) items of many
// models: each warp takes the next item from a global counter until the list
// is exhausted.
template <class C>
__global__ void __launch_bounds__(Occ<C>::kThreads, (Occ<C>::kMinBlocks))
k_solve_queue(const BatchSlot *__restrict__ slots, const uint2 *__restrict__ work, int64_t n_work,
              unsigned long long *__restrict__ next) {
    extern __shared__ __align__(16) unsigned char smem[];
    Stage<C> *stage = reinterpret_cast<Stage<C> *>(smem);
    Lane<C> *lanes = reinterpret_cast<Lane<C> *>(smem + sizeof(Stage<C>) * Occ<C>::kWarps);
    const uint64_t *tab = load_table<C>(smem);
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned long long it = 0;
        if (lane == 0) it = atomicAdd(next, 1ull);
        it = __shfl_sync(kFull, it, 0);
        if (it >= (unsigned long long)n_work) return;
        const uint2 w = work[it];  // x = model << 16 | tile, y = origin
        const BatchSlot &s = slots[w.x >> 16];
        solve_item<C>(s.m, s.Ln, s.R, s.a, int32_t(w.y), int32_t(w.x & 0xffffu), stage[threadIdx.x >> 5],
                      lanes[threadIdx.x >> 5], lane, tab);
        __syncwarp();
    }
}

// Shared memory of a CTA of a solve kernel.
template <class C>
constexpr size_t solve_smem() {
    static_assert(sizeof(Stage<C>) % 16 == 0 && sizeof(Lane<C>) % 16 == 0, "16-byte aligned records");
    return (sizeof(Stage<C>) + sizeof(Lane<C>)) * Occ<C>::kWarps + (C::kInt ? sizeof(Exp2Table) : 0);
}

// Prefer the largest shared-memory carveout for a solve kernel (its resident
// CTAs are bounded by their per-warp staging) and allow its shared memory, on
// the current device.
template <class C, typename K>
void prefer_shared(K kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(solve_smem<C>()));
}

template <class C>
void launch_one(const DevMesh &m, const DevLines &Ln, const DevRays &R_, const SolveArgs &a, cudaStream_t st) {
    const int64_t n_items = int64_t(a.o_end - a.o_begin) * a.n_tiles * a.parts;
    if (n_items == 0) return;
    constexpr int tb = Occ<C>::kThreads;
    const unsigned grid = unsigned((n_items * 32 + tb - 1) / tb);
    prefer_shared<C>(k_solve<C>);
    k_solve<C><<<grid, tb, solve_smem<C>(), st>>>(m, Ln, R_, a);
}

template <typename R, int BPL, int ORD, typename P = R>
void launch_RB(const DevMesh &m, const DevLines &Ln, const DevRays &R_, const SolveArgs &a, cudaStream_t st) {
    if (Ln.L <= 1) launch_one<Form<R, 1, BPL, ORD, P>>(m, Ln, R_, a, st);
    else if (Ln.L <= 2) launch_one<Form<R, 2, BPL, ORD, P>>(m, Ln, R_, a, st);
    else if (Ln.L <= 4) launch_one<Form<R, 4, BPL, ORD, P>>(m, Ln, R_, a, st);
    else launch_one<Form<R, 8, BPL, ORD, P>>(m, Ln, R_, a, st);
}

template <class C>
void launch_queue_one(const BatchSlot *slots, const uint2 *work, int64_t n_work, unsigned long long *next,
                      cudaStream_t st) {
    int dev = 0, sms = 152, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr int tb = Occ<C>::kThreads, nw = Occ<C>::kWarps;
    prefer_shared<C>(k_solve_queue<C>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve_queue<C>, tb, solve_smem<C>());
    if (per_sm < 1) per_sm = 1;
    int64_t grid = int64_t(sms) * per_sm;
    const int64_t need = (n_work + nw - 1) / nw;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    k_solve_queue<C><<<unsigned(grid), tb, solve_smem<C>(), st>>>(slots, work, n_work, next);
}

template <typename R, int BPL, int ORD, typename P = R>
void launch_queue_RB(int max_lines, const BatchSlot *slots, const uint2 *work, int64_t n_work,
                     unsigned long long *next, cudaStream_t st) {
    if (max_lines <= 1) launch_queue_one<Form<R, 1, BPL, ORD, P>>(slots, work, n_work, next, st);
    else if (max_lines <= 2) launch_queue_one<Form<R, 2, BPL, ORD, P>>(slots, work, n_work, next, st);
    else if (max_lines <= 4) launch_queue_one<Form<R, 4, BPL, ORD, P>>(slots, work, n_work, next, st);
    else launch_queue_one<Form<R, 8, BPL, ORD, P>>(slots, work, n_work, next, st);
}

}  // namespace

template <int ORD>
void launch_solve_ord(const DevMesh &m, const DevLines &Ln, const DevRays &R, const SolveArgs &a, int precision,
                      cudaStream_t st) {
    const int bpl = solve_bins_per_lane(precision, ORD, Ln.L, Ln.L * Ln.F);
    if (precision == MGX_FP64 && ORD == 2 && bpl == 2) launch_RB<double, ORD == 2 ? 2 : 1, ORD>(m, Ln, R, a, st);
    else if (precision == MGX_FP64) launch_RB<double, 1, ORD>(m, Ln, R, a, st);
    else if (precision == MGX_FP32_DT64) launch_solve_dt64(m, Ln, R, a, bpl, st);
    else if (ORD == 2 && bpl == 4) launch_one<Form<float, 1, ORD == 2 ? 4 : 2, ORD>>(m, Ln, R, a, st);
    else if (bpl == 2) launch_RB<float, 2, ORD>(m, Ln, R, a, st);
    else launch_RB<float, 1, ORD>(m, Ln, R, a, st);
}

template <int ORD>
void launch_solve_queue_ord(int precision, int bins_per_lane, int max_lines, const BatchSlot *slots,
                            const uint2 *work, int64_t n_work, unsigned long long *next, cudaStream_t st) {
    if (n_work == 0) return;
    if (precision == MGX_FP64 && ORD == 2 && bins_per_lane == 2)
        launch_queue_RB<double, ORD == 2 ? 2 : 1, ORD>(max_lines, slots, work, n_work, next, st);
    else if (precision == MGX_FP64) launch_queue_RB<double, 1, ORD>(max_lines, slots, work, n_work, next, st);
    else if (precision == MGX_FP32_DT64)
        launch_solve_queue_dt64(bins_per_lane, max_lines, slots, work, n_work, next, st);
    else if (ORD == 2 && bins_per_lane == 4)
        launch_queue_one<Form<float, 1, ORD == 2 ? 4 : 2, ORD>>(slots, work, n_work, next, st);
    else if (bins_per_lane == 2) launch_queue_RB<float, 2, ORD>(max_lines, slots, work, n_work, next, st);
    else launch_queue_RB<float, 1, ORD>(max_lines, slots, work, n_work, next, st);
}

}  // namespace mgx
