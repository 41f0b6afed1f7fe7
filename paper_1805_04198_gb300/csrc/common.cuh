// common.cuh -- numerics and small helpers shared by the libeik kernels.
//
// The local solver below is the Godunov upwind solve of Sec. 1.1 (eq.
// "godonuv") in the closed form of Sec. 3.2 (definition of C_H) with the
// per-axis neighbour choice of Alg. 3.  Every multiply and add is written with
// an explicitly rounded intrinsic so the compiler can never contract a pair
// into a fused multiply-add: the FP64 build then performs exactly the IEEE
// operations the method is defined by, in the order written here.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace eik {

constexpr unsigned FULL = 0xffffffffu;

template <class T> struct Num;

// Comparisons of FP64 values on the integer pipe.  The FP64 pipe of this GPU
// issues a warp instruction every 19 cycles per SM with 64 cycles of latency,
// and a double comparison or minimum costs 100 to 157 cycles there; the
// integer forms take about 25.  key() orders all non-NaN doubles as signed
// integers (-0 just below +0); mag() is the order of magnitudes, in which a
// NaN exceeds everything.
// The bits go through asm: the compiler turns an integer comparison of bit-cast
// doubles back into a floating-point one, which is slow and wrong for NaNs.
__device__ __forceinline__ long long bits64(double a) {
    long long x;
    asm("mov.b64 %0, %1;" : "=l"(x) : "d"(a));
    return x;
}
__device__ __forceinline__ long long key(double a) {
    const long long x = bits64(a);
    return x ^ ((x >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ long long mag(double a) { return bits64(a) & 0x7fffffffffffffffll; }

// Correctly rounded square root of a normal x with exponent in [-900, 900]
// (other values take the library root).  With x = 4^q m, m in [1, 4): an FP32
// reciprocal root and one FP32 correction give g, the root of m to 2^-43, as a
// multiple of 2^-43; the residual m - g^2 (at most 46 bits) is exact in one FP64
// FMA; its leading 24 bits times y / 2 give the rest of the root to 2^-12 of an
// ulp in fixed point.  Where that is within 2^-10.7 ulp of a rounding boundary
// (one root in 800) the exact residual of the result decides (Markstein, "IA-64
// and Elementary Functions", ch. 9): R = m - G^2 is a multiple of ulp^2, and G
// is the rounded root unless R > G ulp or R <= -G ulp (R < 0 where G is a power
// of two).  One operation on the FP64 pipe instead of about twenty dependent
// ones.  In two parts, so that several roots can be under way before the rare
// second part splits the warp.
struct Root64 {
    double x, m;
    long long out;  // bits of G
    int qe;         // 2^q for the exponent field
    bool unsure;
    __device__ __forceinline__ double value() const { return __longlong_as_double(out + ((long long)qe << 32)); }
};
__device__ __forceinline__ Root64 root_start(double x) {
    Root64 R;
    R.x = x;
    const int hi = __double2hiint(x);
    const int lo = __double2loint(x);
    const int e = (hi >> 20) - 1023;  // x > 0
    const int par = e & 1;
    R.qe = (e - par) << 19;
    const int mexp = par << 20;
    R.m = __hiloint2double((hi & 0xfffff) | (mexp + (1023 << 20)), lo);
    // m = mh + ml in FP32: 24 bits, the next 23
    const float mh = __int_as_float((__funnelshift_l(lo, hi, 3) & 0x7fffff) | ((mexp << 3) + (127 << 23)));
    const int mlx = (mexp << 3) + (104 << 23);
    const float ml = __fsub_rn(__int_as_float(mlx | (int)((unsigned)(lo << 3) >> 9)), __int_as_float(mlx));
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(mh));
    // in [1, 2), so that its FP64 ulp is 2^-52
    const float s = fminf(fmaxf(__fmul_rn(mh, y), 1.f), 1.99999988f);
    const float yh = __fmul_rn(0.5f, y);
    const float c = __fmul_rn(__fadd_rn(__fmaf_rn(-s, s, mh), ml), yh);
    // g = s + c, c in units of 2^-43 added to the bits of (double)s
    const int ci = __float_as_int(__fmaf_rn(c, 8796093022208.f, 12582912.f)) - 0x4b400000;
    const int sb = __float_as_int(s);
    const long long gb = (((long long)((sb >> 3) + (896 << 20)) << 32) | (unsigned)(sb << 29)) + ((long long)ci << 9);
    const double g = __longlong_as_double(gb);
    const double r = __fma_rn(-g, g, R.m);
    // r as FP32 (its leading bits, 2^-86 <= |r| <= 2^-40 or 0), the correction in 2^-12 ulp
    const int rh = __double2hiint(r), rl = __double2loint(r);
    const int rb = ((__funnelshift_l(rl, rh, 3) & 0x7fffffff) | (rh & 0x80000000)) - 0x40000000;
    const float rf = (rh & 0x7fffffff) == 0 ? 0.f : __int_as_float(rb);
    // + 2047: rounds to the nearest ulp by a shift
    const int f = __float_as_int(__fmaf_rn(__fmul_rn(rf, yh), 18446744073709551616.f, 12582912.f)) - (0x4b400000 - 2047);
    R.out = gb + (f >> 12);
    R.unsure = ((f + 3) & 4095) <= 4 || (unsigned)(e + 900) > 1800u;
    return R;
}
// `clamp`: the root of max(x, 0), 0 where x is NaN.
__device__ __forceinline__ void root_decide(Root64 &R, bool clamp = false) {
    if ((unsigned)((__double2hiint(R.x) >> 20) - 1023 + 900) > 1800u) {
        R.out = __double_as_longlong(__dsqrt_rn(clamp ? fmax(R.x, 0.0) : R.x));
        R.qe = 0;
        return;
    }
    const double G = __longlong_as_double(R.out);
    const long long Rb = bits64(__fma_rn(-G, G, R.m));
    const long long ub = R.out - (52ll << 52);  // G * ulp(G), G in [1, 2)
    const bool neg = Rb < 0;
    const long long Rm = Rb & 0x7fffffffffffffffll;
    // (G = 2, just above the largest root, stands at its lower neighbour's ulp)
    const bool off = (neg ? Rm >= ub : Rm > ub) || (neg && (R.out & 0xfffffffffffffll) == 0 && Rm > 0);
    if (off) R.out += neg ? -1 : 1;
}
__device__ __forceinline__ double sqrt_rn64(double x) {
    Root64 R = root_start(x);
    if (R.unsure) root_decide(R);
    return R.value();
}

template <> struct Num<float> {
    static __device__ __forceinline__ bool lt(float a, float b) { return a < b; }
    static __device__ __forceinline__ bool below(float a, float b) { return a < b; }
    static __device__ __forceinline__ bool lowers(float ut, float self) { return ut < self; }
    static __device__ __forceinline__ float mn(float a, float b) { return fminf(a, b); }
    static __device__ __forceinline__ bool within(float d, float rh) { return fabsf(d) < rh; }
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float sqrt_(float a) { return __fsqrt_rn(a); }
    static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
    static __device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }
    static __device__ __forceinline__ float nan() { return __int_as_float(0x7fffffff); }
    // Square root used inside the local solve.  FP32 storage carries a 1e-5
    // accuracy budget, so the single-instruction hardware approximation
    // (relative error ~1e-7, applied only to the increment of the two-term
    // branch) is used; FP64 keeps the correctly rounded root.
    static __device__ __forceinline__ float sqrt_solve(float a) {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
        return r;
    }
};

template <> struct Num<double> {
    // a < b as IEEE has it: the two zeros are equal, false where either is NaN.
    // Where a tie decides something (winds, Alg. 5)
    static __device__ __forceinline__ bool lt(double a, double b) {
        constexpr long long top = 0x7ff0000000000000ll;
        const long long x = key(a) - (bits64(a) >> 63), y = key(b) - (bits64(b) >> 63);
        return x < y && x >= -top && y <= top;
    }
    // a < b by the keys, for the values of a sweep: there a tie of zeros decides
    // at most the sign of a zero, and one comparison is enough
    static __device__ __forceinline__ bool below(double a, double b) { return key(a) < key(b); }
    // ut < self, false where ut is NaN (the keys of NaNs with the sign set, which
    // arithmetic gives, are below that of -inf).  For the three-term branch; the
    // two-term one gives no NaN, and the test would cost a small box 4%.
    static __device__ __forceinline__ bool lowers(double ut, double self) {
        const long long k = key(ut);
        return k < key(self) && (int)(k >> 32) >= (int)0x800fffff;
    }
    static __device__ __forceinline__ double mn(double a, double b) { return below(a, b) ? a : b; }
    // |d| < rh for rh >= 0, false where d is NaN
    static __device__ __forceinline__ bool within(double d, double rh) { return mag(d) < bits64(rh); }
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double sqrt_(double a) { return __dsqrt_rn(a); }
    static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
    static __device__ __forceinline__ double inf() { return __longlong_as_double(0x7ff0000000000000ll); }
    static __device__ __forceinline__ double nan() { return __longlong_as_double(0x7ff8000000000000ll); }
    static __device__ __forceinline__ double sqrt_solve(double a) { return sqrt_rn64(a); }
};

// The one NaN that the sweeps work with, nan(), has a key above that of +inf, and
// a sum with it is the same NaN.  As a value (Gamma where g is NaN) it is never
// the smaller neighbour; as r h (nodes that keep their value: Gamma, positions
// outside the grid) it gives a u~ that is below no value, whatever the neighbours.
// (r h = +inf does not: with a neighbour at -inf it gives the NaN with the sign
// set, whose key is below every value's.)
template <class T>
__device__ __forceinline__ T gamma_value(T g) {
    return g == g ? g : Num<T>::nan();
}

// Wind packing: component a in {-1,0,+1} stored as (w+1) in 2 bits at 2a.
// Sign = direction of travel: +1 when the upwind (smaller) neighbour is on the
// minus side of the axis.
__host__ __device__ __forceinline__ uint8_t wind_pack(int wx, int wy, int wz = 0) {
    return (uint8_t)((wx + 1) | ((wy + 1) << 2) | ((wz + 1) << 4));
}
__host__ __device__ __forceinline__ int wind_comp(uint8_t w, int a) { return (int)((w >> (2 * a)) & 3) - 1; }
constexpr uint8_t WIND_ZERO = 0x15;  // (0,0,0)
// Flag on a subdomain's copy of a coarse-set node (never on W or w^k): the node
// was inflow and the subdomain solve kept its Step 2 value U, so the copy
// echoes boundary data rather than a fine solution.
constexpr uint8_t WIND_ECHO = 0x80;

// Value of the local solve from the axis minima a, b: the two-term branch
// (a + b + sqrt(2 r^2 h^2 - (a-b)^2)) / 2 where |a - b| < r h, else the smaller
// one plus r h.  The discriminant needs no clamp while (r h)^2 is finite: where
// the two-term branch is taken it is at least (r h)^2; elsewhere its root is not
// selected.  Where both squares overflow it is NaN, which counts as 0 in FP64.
__device__ __forceinline__ float solve2(float a, float b, float rh, bool &two) {
    using N = Num<float>;
    const float d = N::sub(a, b);
    // rn(2 r h r h) = 2 rn(r h r h): one product, and the doubling in the FMA (for
    // r h below 2^-63, 1e-19, the product is subnormal and its root flushed to 0)
    const float disc = __fmaf_rn(2.f, N::mul(rh, rh), -N::mul(d, d));
    // (a + b + root) / 2 as one rounding of root / 2 + (a + b) / 2: halving is
    // exact, so this is the same value with a shorter chain behind the root
    const float u2 = __fmaf_rn(N::sqrt_solve(disc), 0.5f, N::mul(N::add(a, b), 0.5f));
    const float u1 = N::add(fminf(a, b), rh);
    two = fabsf(d) < rh;
    return two ? u2 : u1;
}
// FP64: eight operations on the FP64 pipe, the comparisons, the doubling and the
// halving on the integer pipe; in two parts like the root.  r h = +inf or NaN
// (fixed nodes) takes the one-term branch.
struct Solve64 {
    double ab, u1;
    Root64 root;
    bool two;
};
__device__ __forceinline__ Solve64 solve2_start(double a, double b, double rh) {
    using N = Num<double>;
    Solve64 S;
    const double d = N::sub(a, b);
    S.two = N::within(d, rh) && __double2hiint(rh) < 0x7ff00000;
    // 2 r h by its exponent (exact; where r h is subnormal its square is 0 in any
    // case; above the range another number whose product with r h is +inf too).
    // Not 2 (r h)^2: that loses the bits of a square just below the normal range.
    const unsigned rhi = (unsigned)__double2hiint(rh) + (1u << 20);
    const double rh2 = __hiloint2double((int)min(rhi, 0x7fefffffu), __double2loint(rh));
    const double disc = N::sub(N::mul(rh2, rh), N::mul(d, d));
    S.root = root_start(S.two ? disc : 1.0);
    S.ab = N::add(a, b);
    S.u1 = N::add(N::mn(a, b), rh);
    return S;
}
__device__ __forceinline__ double solve2_end(const Solve64 &S) {
    using N = Num<double>;
    const double w = N::add(S.ab, S.root.value());
    // w / 2 by its exponent, where that is exact (it always is but next to the
    // ends of the FP64 range)
    const int wh = __double2hiint(w);
    double u2 = __hiloint2double(wh - (1 << 20), __double2loint(w));
    if (S.two && ((unsigned)(wh & 0x7fffffff) - (2u << 20)) >= ((0x7ffu - 2u) << 20)) u2 = N::mul(w, 0.5);
    return S.two ? u2 : S.u1;
}
__device__ __forceinline__ double solve2(double a, double b, double rh, bool &two) {
    Solve64 S = solve2_start(a, b, rh);
    if (S.root.unsure) root_decide(S.root, true);
    two = S.two;
    return solve2_end(S);
}

// 2-D Godunov local solve.  vm*/vp* are the neighbours on the minus/plus side
// of each axis (+inf where missing: the one-sided rule of Sec. 1.1).  Returns
// u~ and the packed wind of the branch taken (zero wind when u~ is +inf).
// Both branches are evaluated and one is selected, so no warp diverges; the
// selected branch performs exactly the operations written in the paper's
// closed form.
template <class T>
__device__ __forceinline__ T local_solve2(T vmx, T vpx, T vmy, T vpy, T rh, uint8_t &wind) {
    using N = Num<T>;
    // Alg. 3: the smaller neighbour per axis; a tie goes to the plus side.
    const bool lx = N::lt(vmx, vpx), ly = N::lt(vmy, vpy);
    const T a = lx ? vmx : vpx, b = ly ? vmy : vpy;
    const int sa = lx ? 1 : -1, sb = ly ? 1 : -1;
    const bool ax = N::lt(a, b);
    bool two;
    T u = solve2(a, b, rh, two);
    if (!two) u = N::add(ax ? a : b, rh);  // (its own minimum differs only where a is NaN)
    wind = two ? wind_pack(sa, sb)
               : (N::lt(u, N::inf()) ? (ax ? wind_pack(sa, 0) : wind_pack(0, sb)) : WIND_ZERO);
    return u;
}

// Value-only variant used inside the sweeps (the wind is recomputed from the
// converged state, so the sweeps need only the value).
template <class T>
__device__ __forceinline__ T local_solve2_min(T a, T b, T rh) {
    bool two;
    return solve2(a, b, rh, two);
}
template <class T>
__device__ __forceinline__ T local_solve2_value(T vmx, T vpx, T vmy, T vpy, T rh) {
    return local_solve2_min(Num<T>::mn(vmx, vpx), Num<T>::mn(vmy, vpy), rh);
}

// 3-D Godunov local solve: axis minima sorted a_p0 <= a_p1 <= a_p2 (ties keep
// axis order); one term, else the paper's two-term formula on the two
// smallest, else the three-term quadratic written in t = u - a_p0:
//   t^2 + (t - d1)^2 + (t - d2)^2 = (r h)^2.
// The wind has the per-axis sign of Alg. 3 on the axes used.  With a_p2 = inf
// it reduces exactly to local_solve2.  The sort is done by ranks and selects
// (no indexed local arrays); the arithmetic is the same sequence of rounded
// operations on the sorted values.
template <class T>
__device__ __forceinline__ T local_solve3(const T *vm, const T *vp, T rh, uint8_t &wind) {
    using N = Num<T>;
    const bool l0 = N::lt(vm[0], vp[0]), l1 = N::lt(vm[1], vp[1]), l2 = N::lt(vm[2], vp[2]);
    const T a0 = l0 ? vm[0] : vp[0], a1 = l1 ? vm[1] : vp[1], a2 = l2 ? vm[2] : vp[2];
    // stable ranks: axis b precedes axis c when a_b < a_c, or a_b == a_c and b < c
    const bool b10 = N::lt(a1, a0), b20 = N::lt(a2, a0), b21 = N::lt(a2, a1);
    const int r0 = (b10 ? 1 : 0) + (b20 ? 1 : 0);
    const int r1 = (b10 ? 0 : 1) + (b21 ? 1 : 0);
    const int r2 = (b20 ? 0 : 1) + (b21 ? 0 : 1);
    const T v0 = r0 == 0 ? a0 : (r1 == 0 ? a1 : a2);
    const T v1 = r0 == 1 ? a0 : (r1 == 1 ? a1 : a2);
    const T v2 = r0 == 2 ? a0 : (r1 == 2 ? a1 : a2);
    const T d01 = N::sub(v0, v1);
    const bool two = fabs(d01) < rh;
    const T disc = N::sub(N::mul(N::mul(T(2), rh), rh), N::mul(d01, d01));
    const T u2 = N::mul(N::add(N::add(v0, v1), N::sqrt_solve(fmax(disc, T(0)))), T(0.5));
    const T u1 = N::add(v0, rh);
    const bool three = two && (u2 > v2);
    T u = two ? u2 : u1;
    if (three) {
        const T d1 = N::sub(v1, v0);
        const T d2 = N::sub(v2, v0);
        const T sd = N::add(d1, d2);
        T disc3 = N::sub(N::mul(sd, sd), N::mul(T(3), N::sub(N::add(N::mul(d1, d1), N::mul(d2, d2)), N::mul(rh, rh))));
        if (disc3 < T(0)) disc3 = T(0);
        u = N::add(v0, N::div(N::add(sd, N::sqrt_solve(disc3)), T(3)));
    }
    const int nt = three ? 3 : (two ? 2 : (u < N::inf() ? 1 : 0));  // axes used, by rank
    wind = wind_pack(r0 < nt ? (l0 ? 1 : -1) : 0, r1 < nt ? (l1 ? 1 : -1) : 0, r2 < nt ? (l2 ? 1 : -1) : 0);
    return u;
}

// x / 3, correctly rounded: the quotient by the rounded reciprocal corrected by
// its exact residual (Markstein, as above; equal to the division for every
// finite number but -0).  NaN at +-inf.
__device__ __forceinline__ float div3(float x) {
    const float c = 1.f / 3.f;
    const float q = __fmul_rn(x, c);
    return __fmaf_rn(__fmaf_rn(-3.f, q, x), c, q);
}
__device__ __forceinline__ double div3(double x) {
    const double c = 1.0 / 3.0;
    const double q = __dmul_rn(x, c);
    return __fma_rn(__fma_rn(-3.0, q, x), c, q);
}

// Value of the 3-D local solve from the three axis minima (the same rounded
// operations as local_solve3 on the sorted values): a sort of minima and maxima,
// no winds.  r h = NaN (fixed nodes) gives NaN, and so may squares that overflow:
// that lowers no value.
__device__ __forceinline__ float solve3(float m0, float m1, float m2, float rh) {
    using N = Num<float>;
    const float lo = fminf(m0, m1), hi = fmaxf(m0, m1);
    const float v0 = fminf(lo, m2), t = fmaxf(lo, m2);
    const float v1 = fminf(t, hi), v2 = fmaxf(t, hi);
    const float d1 = N::sub(v1, v0), d2 = N::sub(v2, v0);
    const float dd = N::mul(d1, d1), rr = N::mul(rh, rh);
    const float disc = __fmaf_rn(2.f, rr, -dd);
    const float u2 = __fmaf_rn(N::sqrt_solve(disc), 0.5f, N::mul(N::add(v0, v1), 0.5f));
    const bool two = d1 < rh;
    const float sd = N::add(d1, d2);
    const float disc3 = N::sub(N::mul(sd, sd), N::mul(3.f, N::sub(N::add(dd, N::mul(d2, d2)), rr)));
    const float u3 = N::add(v0, div3(N::add(sd, N::sqrt_solve(fmaxf(disc3, 0.f)))));
    const float u = two ? u2 : N::add(v0, rh);
    return two && u2 > v2 ? u3 : u;
}
__device__ __forceinline__ double solve3(double m0, double m1, double m2, double rh) {
    using N = Num<double>;
    const bool s01 = N::below(m1, m0);
    const double lo = s01 ? m1 : m0, hi = s01 ? m0 : m1;
    const bool s2 = N::below(m2, lo);
    const double v0 = s2 ? m2 : lo, t = s2 ? lo : m2;
    const bool s3 = N::below(t, hi);
    const double v1 = s3 ? t : hi, v2 = s3 ? hi : t;
    bool two;
    double u = solve2(v0, v1, rh, two);
    if (two && N::lt(v2, u)) {
        const double d1 = N::sub(v1, v0), d2 = N::sub(v2, v0);
        const double sd = N::add(d1, d2);
        double disc3 = N::sub(N::mul(sd, sd), N::mul(3.0, N::sub(N::add(N::mul(d1, d1), N::mul(d2, d2)), N::mul(rh, rh))));
        if (disc3 < 0.0) disc3 = 0.0;
        u = N::add(v0, div3(N::add(sd, sqrt_rn64(disc3))));
    }
    return u;
}

// Register cap of a sweep-engine kernel by element type (FP32, FP64): keeps
// the single-CTA launch shapes (up to 32 warps) and the co-residency of the
// cooperative multi-CTA forms.
template <class T, int F32, int F64> struct RegCap {
    static constexpr int v = sizeof(T) == 4 ? F32 : F64;
};

// Status codes mirrored from eik.h for device code.
constexpr int DEV_OK = 0;
constexpr int DEV_TIMEOUT = -4;

// Default iteration limit of every bounded device-side wait (iterations of at
// most ~1 us sleep each, so an expired wait reports within seconds).
constexpr long long SPIN_LIMIT_DEFAULT = 1ll << 22;

// The limit in force.  Each translation unit that waits has its own copy per
// device; eik_set_wait_limit writes every copy through the setter that the
// unit defines with EIK_SPIN_LIMIT_SETTER.  A kernel that waits reads it once
// when it starts (a global load on the path of a wait would delay the wait
// itself).
static __device__ long long g_spin_limit = SPIN_LIMIT_DEFAULT;
__device__ __forceinline__ long long spin_limit() { return *(volatile const long long *)&g_spin_limit; }
#define EIK_SPIN_LIMIT_SETTER(fname) \
    int fname(long long v) { return (int)cudaMemcpyToSymbol(g_spin_limit, &v, sizeof(v)); }

// Grid-wide barrier for cooperative launches (all CTAs co-resident).  bar[0]
// counts arrivals, bar[1] is the generation.  The wait is bounded by `lim`
// polls (the kernel reads spin_limit() once when it starts): on timeout the
// error word is set and false is returned to every thread of the CTA (the
// caller then returns with the whole CTA).
__device__ inline bool grid_barrier(unsigned *bar, int *err, long long lim) {
    __shared__ int s_barrier_ok;
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        volatile unsigned *vgen = bar + 1;
        const unsigned gen = *vgen;
        __threadfence();
        const unsigned arrived = atomicAdd(bar, 1u) + 1u;
        if (arrived == gridDim.x) {
            bar[0] = 0u;
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            long long it = 0;
            while (*vgen == gen) {
                if (++it > lim) {
                    atomicExch(err, DEV_TIMEOUT);
                    ok = false;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        s_barrier_ok = ok ? 1 : 0;
    }
    __syncthreads();
    ok = s_barrier_ok != 0;
    __syncthreads();  // s_barrier_ok is read by all before the next barrier writes it
    return ok;
}

// Per-node weight of Sec. 4.2 from du = u^k - u^{k-1} and the last n changes
// dC[s] of C_H(nbrs U): eq. secthetaest (weighted mean of the changes), the
// damping of eq. thetaest, the optional cap; `fallback` where undefined.  A is
// any argument block carrying the weights om[3] and the damping parameters sg
// (gamma), sd (delta), sx0 (x0) and cap.
template <class Args>
__device__ inline double theta_estimate(const Args &A, double du, const double *dC, int n, double fallback) {
    double den = 0.0, wsum = 0.0;
    for (int s = 0; s < n; ++s) {
        den = __dadd_rn(den, __dmul_rn(A.om[s], dC[s]));
        wsum = __dadd_rn(wsum, A.om[s]);
    }
    if (!(wsum > 0.0)) return fallback;
    den = __ddiv_rn(den, wsum);
    const double t = __ddiv_rn(du, den);
    if (!isfinite(t) || den == 0.0) return fallback;
    const double sig = __ddiv_rn(1.0, __dadd_rn(1.0, exp(__ddiv_rn(__dsub_rn(t, A.sx0), A.sg))));
    double v = __dadd_rn(__dmul_rn(sig, t), __dmul_rn(__dmul_rn(__dsub_rn(1.0, sig), A.sd), t));
    if (A.cap > 0.0 && v > A.cap) v = A.cap;
    return v > 0.0 ? v : 0.0;
}

}  // namespace eik
