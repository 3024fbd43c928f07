// Kernel function and pair separation shared by the pair kernels.
#pragma once

#include "neighbors.cuh"
#include "sph_internal.cuh"

namespace sph {

// Quintic spline in q (section 2, Eq. kernel) without sigma2, and its
// q-derivative, branch free: with a = max(3 - q, 0), b = max(2 - q, 0),
// c = max(1 - q, 0), w = a^5 - 6 b^5 + 15 c^5 and dw/dq = -5 a^4 + 30 b^4
// - 75 c^4 (every term vanishes where its base is clipped to zero).  The
// clip is one max instruction (a NaN q clips to zero).
// sigma2 = 7 / (478 pi h^2); dW/dr = sigma2 / h * dw(q).
__device__ __forceinline__ float clip0(float t) { return fmaxf(t, 0.0f); }
__device__ __forceinline__ double clip0(double t) { return fmax(t, 0.0); }

template <typename R>
__device__ __forceinline__ R qs_w(R q) {
    const R a = clip0(R(3) - q);
    const R b = clip0(R(2) - q);
    const R c = clip0(R(1) - q);
    const R a2 = a * a, b2 = b * b, c2 = c * c;
    return a2 * a2 * a - R(6) * (b2 * b2 * b) + R(15) * (c2 * c2 * c);
}

template <typename R>
__device__ __forceinline__ R qs_dw(R q) {
    const R a = clip0(R(3) - q);
    const R b = clip0(R(2) - q);
    const R c = clip0(R(1) - q);
    const R a2 = a * a, b2 = b * b, c2 = c * c;
    return R(-5) * (a2 * a2) + R(30) * (b2 * b2) - R(75) * (c2 * c2);
}

// a b + c d with the one product rounded first: the compiler may contract
// either one, and differently in each kernel a body is compiled into.
__device__ __forceinline__ double mad2(double a, double b, double c, double d) {
    return __fma_rn(a, b, __dmul_rn(c, d));
}

// a / b and 1/sqrt(x): IEEE in double; the fast FP32 forms (at most 2 ulp)
// in float, well inside the mixed path's tolerance.
__device__ __forceinline__ double fdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double frsqrt(double x) { return 1.0 / sqrt(x); }
__device__ __forceinline__ float frsqrt(float x) { return rsqrtf(x); }

// The FP64 pair sums of sets without walls (LEAN below) take their
// reciprocals from the hardware's 20-bit estimate and one third-order
// Householder step, with e = 1 - b y (reciprocal) or 1 - x y^2 (reciprocal
// square root) of at most 2^-19: the remainder e^3 lies below half an ulp,
// so the result is within 1.5 ulp for normal operands and results.  GB300
// issues one FP64 instruction per SM sub-partition every 64 cycles, and the
// pair sums are bound by that pipe: the correctly rounded divide and square
// root cost it tens of instructions a pair, these three and five.
//
// Sets with walls keep the correctly rounded sequence, operation for
// operation.  The rule looks at the walls alone; its reason is adaptation,
// which amplifies a last bit: a split parent's children sit on a hexagon,
// whose equal distances the merge search orders by their rounding, so after
// one bit the flow splits and merges other particles.  The flows past bodies
// adapt and have walls, their pair sums are a small part of an adaptive step
// (pass A and B 7 % of one of the 1:250 cylinder, 91k particles), and they
// keep their particle history.  The rule is not the reason on either side of
// it: a flow that adapts without walls (a vortex with a refined region, the
// background construction) takes these sums, and splits and merges by their
// rounding, not by the divisions'; a walled flow that never adapts (a
// channel) takes the slower sums.
template <typename R, bool LEAN>
constexpr bool lean64 = LEAN && sizeof(R) == 8;

__device__ __forceinline__ double frcp(double b) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = __fma_rn(-b, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}
__device__ __forceinline__ double frsqrt_lean(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = __fma_rn(-__dmul_rn(x, y), y, 1.0);
    return __fma_rn(__dmul_rn(y, e), __fma_rn(0.375, e, 0.5), y);
}

// LEAN FP64 pair sums: the quintic as one polynomial per unit piece, in t = 3 -
// q, 2 - q or 1 - q (0 <= t <= 1, so Horner's rule is well conditioned):
//   q in [2, 3): t^5
//   q in [1, 2): 1 + 5t + 10t^2 + 10t^3 + 5t^4 - 5t^5
//   q in [0, 1): 26 + 50t + 20t^2 - 20t^3 - 20t^4 + 10t^5
// and zero from q = 3 on (t = 0 on the first piece; a NaN q too).  The
// piece is chosen by q's high word and its coefficients, whose low words
// are zero, by integer selects; the FP64 pipe sees 5 operations for the
// derivative and 10 for both, against 14 and 17 for the clipped powers.
struct QsPiece {
    bool lt1, lt2;
    double t;
    __device__ __forceinline__ explicit QsPiece(double q) {
        const unsigned hi = (unsigned)__double2hiint(q);
        lt1 = hi < 0x3ff00000u;
        lt2 = hi < 0x40000000u;
        t = hi < 0x40080000u ? __dsub_rn(coef(1.0, 2.0, 3.0), q) : 0.0;
    }
    __device__ __forceinline__ double coef(double c1, double c2, double c3) const {
        return __hiloint2double(lt1 ? __double2hiint(c1)
                                    : lt2 ? __double2hiint(c2) : __double2hiint(c3), 0);
    }
};
// s = -(dw/dq) / 5
__device__ __forceinline__ double qs_s(double q) {
    const QsPiece p(q);
    double s = __fma_rn(p.coef(10.0, -5.0, 1.0), p.t, p.coef(-16.0, 4.0, 0.0));
    s = __fma_rn(s, p.t, p.coef(-12.0, 6.0, 0.0));
    s = __fma_rn(s, p.t, p.coef(8.0, 4.0, 0.0));
    return __fma_rn(s, p.t, p.coef(10.0, 1.0, 0.0));
}
__device__ __forceinline__ void qs_ws(double q, double &w, double &s) {
    const QsPiece p(q);
    w = __fma_rn(p.coef(10.0, -5.0, 1.0), p.t, p.coef(-20.0, 5.0, 0.0));
    w = __fma_rn(w, p.t, p.coef(-20.0, 10.0, 0.0));
    w = __fma_rn(w, p.t, p.coef(20.0, 10.0, 0.0));
    w = __fma_rn(w, p.t, p.coef(50.0, 5.0, 0.0));
    w = __fma_rn(w, p.t, p.coef(26.0, 1.0, 0.0));
    s = __fma_rn(p.coef(10.0, -5.0, 1.0), p.t, p.coef(-16.0, 4.0, 0.0));
    s = __fma_rn(s, p.t, p.coef(-12.0, 6.0, 0.0));
    s = __fma_rn(s, p.t, p.coef(8.0, 4.0, 0.0));
    s = __fma_rn(s, p.t, p.coef(10.0, 1.0, 0.0));
}
// Whether x >= 0 is a normal number (or infinite, or NaN), on the integer
// pipe.  A squared separation below that (r < 1.5e-154) counts as zero: the
// estimate above flushes it and returns infinity.  The kernels are at
// their r = 0 values to the last bit long before.
__device__ __forceinline__ bool is_normal(double x) {
    return (uint32_t)__double2hiint(x) >= 0x00100000u;
}

// Mixed pair sums of sets without walls (LEAN): two values share an
// instruction where the formulas come in pairs: the axes of a separation, u
// and v, the kernels of h_i and h_j.  Each half rounds like the scalar
// operation.  At 1M particles of the 1:250 strip pass B issues 178M warp
// instructions and is bound by the L1 data pipe of its record gathers (83 %
// of the peak; issue 59 %), pass A 206M and by issue (69 %; data pipe 46 %).
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ float lo(F2 a) {
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return x;
}
__device__ __forceinline__ float hi(F2 a) {
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
    return y;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, f2(-1.0f), a); }
__device__ __forceinline__ F2 clip2(F2 a) {
    return f2(fmaxf(lo(a), 0.0f), fmaxf(hi(a), 0.0f));
}
__device__ __forceinline__ float frcp_ftz(float b) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(b));
    return y;
}
constexpr float F32_LEAST = 1.17549435e-38f;   // least normal

// The bases of the clipped quintic (qs_w above) at two q = r / h each, nh =
// {-1 / h, -1 / h'}.  3 - q is rounded once and 2 - q and 1 - q follow from it
// exactly, so the rounding acts like one error of q, which mostly cancels in
// the derivative.  (Each base by its own FMA made the momentum rates of the
// 1:250 strip 6 % less accurate, all three from a rounded q pass B 5 %
// slower.)
struct Qs2 {
    F2 a, b, c;
    __device__ __forceinline__ Qs2(float r, F2 nh) {
        const F2 t = fma2(f2(r), nh, f2(3.0f));
        a = clip2(t);
        b = clip2(add2(t, f2(-1.0f)));
        c = clip2(add2(t, f2(-2.0f)));
    }
    // s = -(dw/dq) / 5
    __device__ __forceinline__ F2 s() const {
        const F2 a2 = mul2(a, a), b2 = mul2(b, b), c2 = mul2(c, c);
        return fma2(a2, a2, fma2(mul2(b2, f2(-6.0f)), b2, mul2(mul2(c2, f2(15.0f)), c2)));
    }
    __device__ __forceinline__ void ws(F2 &w, F2 &s) const {
        const F2 a2 = mul2(a, a), b2 = mul2(b, b), c2 = mul2(c, c);
        const F2 b6 = mul2(b2, f2(-6.0f)), c4 = mul2(mul2(c2, f2(15.0f)), c2);
        s = fma2(a2, a2, fma2(b6, b2, c4));
        w = fma2(mul2(a2, a2), a, fma2(mul2(b6, b2), b, mul2(c4, c)));
    }
};

// Separation r_i - r_j of anchor records (anchor_sep, both axes at once:
// the same values).
struct Sep2 {
    F2 xi, gi, nf, invn, A;
    __device__ __forceinline__ Sep2(const Anchor &an, const float4 &pi) {
        const unsigned g = __float_as_uint(pi.w);
        xi = f2(pi.x, pi.y);
        gi = f2(anchor_gx(g), anchor_gy(g));
        nf = f2(-an.nf[0], -an.nf[1]);
        invn = f2(an.invn[0], an.invn[1]);
        A = f2(an.A[0], an.A[1]);
    }
    __device__ __forceinline__ F2 get(const float4 &pj) const {
        const unsigned g = __float_as_uint(pj.w);
        F2 k = sub2(gi, f2(anchor_gx(g), anchor_gy(g)));
        const F2 t = add2(fma2(k, invn, f2(RINT_MAGIC)), f2(-RINT_MAGIC));
        k = fma2(t, nf, k);
        return fma2(k, A, sub2(xi, f2(pj.x, pj.y)));
    }
};

// Four values of one neighbour, loaded together.
template <typename R> struct V4;
template <> struct V4<float> { using T = float4; };
template <> struct V4<double> { using T = double4_32a; };

// The FP32 pass-B record of a neighbour, its two halves side by side: one
// 32-byte access (pass B is bound by the L1 data pipe of its gathers; two
// 16-byte ones took 5 % longer at 4.2M on the graded strip).
__device__ __forceinline__ void load8(const float4 *p, float4 &a, float4 &b) {
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}
__device__ __forceinline__ void store8(float4 *p, const float4 &a, const float4 &b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x),
                 "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

template <typename R>
__device__ __forceinline__ R sigma_norm() {
    return R(7.0 / (478.0 * PI));
}

// Separation r_i - r_j of list entry j: FP64 minimum image on the FP64
// path; on the mixed path rebuilt in FP32 from the anchor coordinates.
template <typename R> struct Sep;
template <> struct Sep<double> {
    double xi, yi;
    __device__ __forceinline__ void init(const Domain &, const double *x,
                                         const double *y, const float4 *, int i) {
        xi = x[i];
        yi = y[i];
    }
    __device__ __forceinline__ void get(const Domain &d, const Anchor &,
                                        const double *x, const double *y,
                                        const float4 *, int j, double &dx,
                                        double &dy, double &r2) const {
        dx = min_image(d, 0, __dsub_rn(xi, __ldg(&x[j])));
        dy = min_image(d, 1, __dsub_rn(yi, __ldg(&y[j])));
        r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    }
    // with h_j (FP64 array)
    __device__ __forceinline__ void get(const Domain &d, const Anchor &an,
                                        const double *x, const double *y,
                                        const double *h, const float4 *pk,
                                        int j, double &dx, double &dy,
                                        double &r2, double &hj) const {
        get(d, an, x, y, pk, j, dx, dy, r2);
        hj = __ldg(&h[j]);
    }
};
template <> struct Sep<float> {
    float4 pi;
    __device__ __forceinline__ void init(const Domain &, const double *,
                                         const double *, const float4 *pk, int i) {
        pi = pk[i];
    }
    __device__ __forceinline__ void get(const Domain &, const Anchor &an,
                                        const double *, const double *,
                                        const float4 *pk, int j, float &dx,
                                        float &dy, float &r2) const {
        anchor_sep(an, pi, __ldg(&pk[j]), dx, dy);
        r2 = fmaf(dx, dx, dy * dy);
    }
    // with h_j (from the anchor record)
    __device__ __forceinline__ void get(const Domain &, const Anchor &an,
                                        const double *, const double *,
                                        const double *, const float4 *pk,
                                        int j, float &dx, float &dy,
                                        float &r2, float &hj) const {
        const float4 pj = __ldg(&pk[j]);
        anchor_sep(an, pi, pj, dx, dy);
        r2 = fmaf(dx, dx, dy * dy);
        hj = pj.z;
    }
};


}  // namespace sph
