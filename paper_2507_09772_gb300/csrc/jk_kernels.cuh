// Integral kernels of the JK build, compiled at run time by NVRTC for
// sm_103a, one instantiation per (l_a, l_b, l_c, l_d), fragmentation,
// density count, J/K flags and precision (the static parameters of Table 1 of
// the paper, except the primitive counts, which are loop limits read from the
// class pair: one launch then runs every class pair of the same angular
// momenta, see the class kernel). The library prepends
// jk_types.h and the generated rys_params.cuh.
//
// Method (Sec. 2 of the paper):
//   eq:rys0  (ab|cd) = sum over primitive quartets of c_a c_b c_c c_d (pq|rs)
//   eq:rys1  (pq|rs) = sum_r w_r (pq|rs)(t_r), N_r = floor(L/2) + 1 roots
//   eq:rys2  (pq|rs)(t_r) = I_x I_y I_z, each a 2D table over the Cartesian
//            exponents of the four centres, built per root by the vertical
//            recurrence on (A, C) and the horizontal transfers A->B, C->D
//   eq:jk    J_ab += T D_cd, J_cd += T D_ab, K_ac += T D_bd, K_ad += T D_bc,
//            K_bc += T D_ad, K_bd += T D_ac for each unique quartet (8-fold
//            symmetry, Sec. 2), scaled by the degeneracy factor f: 2f for J
//            and f for K into half matrices that are symmetrised afterwards.
//
// Thread mapping: a group of G = GA*GB*GC*GD threads evaluates one shell
// quartet. Each thread owns a fragment of FA x FB x FC x FD Cartesian
// components (the 1qnt fragmentation of Sec. 3.2; G = 1 is the 1q1t case of
// Sec. 3.1). With G == 1 the 2D tables live in registers; with G > 1 they
// live in shared memory, one set per group, built cooperatively per root and
// direction. A warp owns one bra pair at a time and scans its ket pairs in
// chunks of 32 candidates, screening each (Schwarz times density-block max),
// so the quartet list is never materialised; the J_ab partial stays in
// registers across the whole ket scan and is flushed once per bra pair.

#define JK_TWO_PI_2_5 34.986836655249725  // 2 pi^(5/2)

__device__ constexpr int jk_ncart(int l) { return (l + 1) * (l + 2) / 2; }

// Cartesian exponent along `axis` of component idx of a shell with angular
// momentum l: components ordered x descending, then y descending.
__device__ constexpr int jk_cart_exp(int l, int idx, int axis)
{
    int k = 0;
    for (int x = l; x >= 0; --x)
        for (int y = l - x; y >= 0; --y) {
            if (k == idx) return axis == 0 ? x : (axis == 1 ? y : l - x - y);
            ++k;
        }
    return 0;
}

// ------------------------------------------------- two-float arithmetic
// The split tier evaluates its quartets in pairs of floats (value h + l, 48
// bits). GB300 has 64 FP32 lanes per FP64 lane: one FP64 instruction holds the
// SM's FP64 pipe for as long as 64 FP32 instructions take to issue, a
// two-float product takes 4 to 7 of them and a sum 8 to 11 (measured: 2,400
// G/s two-float multiply-adds against 502 G/s DFMA). The algorithms are the
// error-free transformations of Dekker (Numer. Math. 18, 1971) and Knuth (The
// Art of Computer Programming 2, 4.2.2); the explicitly rounded intrinsics keep
// the compiler from contracting them. "Loose" results may carry an l of a few
// ulp of h; jk_norm brings it back below half an ulp.
struct jkdf {
    float h, l;
};
__device__ __forceinline__ jkdf jk_norm(jkdf a)
{
    const float s = __fadd_rn(a.h, a.l);
    return {s, __fadd_rn(a.l, -__fadd_rn(s, -a.h))};
}
// product (loose): h l' and l h' included, l l' (2^-48 of the result) dropped
__device__ __forceinline__ jkdf jk_mul(jkdf a, jkdf b)
{
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    return {p, __fmaf_rn(a.l, b.h, e)};
}
// sum (loose)
__device__ __forceinline__ jkdf jk_add(jkdf a, jkdf b)
{
    const float s = __fadd_rn(a.h, b.h), t = __fadd_rn(s, -a.h);
    const float e = __fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -t)), __fadd_rn(b.h, -t));
    return {s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ jkdf jk_neg(jkdf a) { return {-a.h, -a.l}; }
__device__ __forceinline__ jkdf jk_sub(jkdf a, jkdf b) { return jk_add(a, jk_neg(b)); }
// v += a b (loose)
__device__ __forceinline__ void jk_acc(jkdf &v, jkdf a, jkdf b) { v = jk_add(v, jk_mul(a, b)); }
__device__ __forceinline__ void jk_addto(jkdf &v, jkdf a) { v = jk_add(v, a); }
// times an exactly representable power of two
__device__ __forceinline__ jkdf jk_scale(jkdf a, float s) { return {__fmul_rn(a.h, s), __fmul_rn(a.l, s)}; }
// times a small integer (loose)
__device__ __forceinline__ jkdf jk_int(int n, jkdf a)
{
    if (n == 1) return a;
    const float p = __fmul_rn(a.h, (float)n);
    return {p, __fmaf_rn((float)n, a.l, __fmaf_rn((float)n, a.h, -p))};
}
template <typename R> struct JkConst {
    __device__ static __forceinline__ R get(double c) { return (R)c; }
};
template <> struct JkConst<jkdf> {   // compile-time constants only
    __device__ static __forceinline__ jkdf get(double c) { return {(float)c, (float)(c - (double)(float)c)}; }
};
// 1 / sqrt(x): the FP32 estimate y and its residual r = 1 - x y^2 = d - t (d =
// 1 - fl(x y^2) has a few bits, t the rest), y (1 + r/2 + 3 r^2 / 8) with the
// product y d / 2 kept exact (normalised; relative error 1.7e-14 at most and
// 1.3e-15 rms over 4e6 arguments with estimates within 2 ulp, emulated)
__device__ __forceinline__ jkdf jk_rsqrt(jkdf x)
{
    const float y = rsqrtf(x.h);
    const float p = __fmul_rn(y, y), e = __fmaf_rn(y, y, -p);
    const float h = __fmul_rn(x.h, p);
    const float t = __fmaf_rn(x.h, e, __fmaf_rn(x.l, p, __fmaf_rn(x.h, p, -h)));
    const float d = __fadd_rn(1.0f, -h), hd = __fmul_rn(0.5f, d), r = __fadd_rn(d, -t);
    const float q = __fmul_rn(y, hd);
    const float w = __fmaf_rn(y, __fmaf_rn(-0.5f, t, __fmul_rn(__fmul_rn(0.375f, r), r)), __fmaf_rn(y, hd, -q));
    const float s = __fadd_rn(y, q);
    return {s, __fadd_rn(__fadd_rn(q, -__fadd_rn(s, -y)), w)};
}
// the same names for the machine types
template <typename T> __device__ __forceinline__ T jk_norm(T a) { return a; }
template <typename T> __device__ __forceinline__ T jk_mul(T a, T b) { return a * b; }
template <typename T> __device__ __forceinline__ T jk_add(T a, T b) { return a + b; }
template <typename T> __device__ __forceinline__ T jk_sub(T a, T b) { return a - b; }
template <typename T> __device__ __forceinline__ T jk_neg(T a) { return -a; }
template <typename T> __device__ __forceinline__ void jk_acc(T &v, T a, T b) { v += a * b; }
template <typename T> __device__ __forceinline__ void jk_addto(T &v, T a) { v += a; }
template <typename T> __device__ __forceinline__ T jk_scale(T a, float s) { return a * (T)s; }
template <typename T> __device__ __forceinline__ T jk_int(int n, T a) { return T(n) * a; }

// Primitive-pair records by arithmetic, and their fields.
template <typename R> struct JkPP;
template <> struct JkPP<double> { typedef JkPrimPair64 T; };
template <> struct JkPP<float> { typedef JkPrimPair32 T; };
template <> struct JkPP<jkdf> { typedef JkPrimPairDf T; };
__device__ __forceinline__ float jk_pp_q(const JkPrimPair64 &r) { return r.qf; }
__device__ __forceinline__ float jk_pp_q(const JkPrimPair32 &r) { return r.q; }
__device__ __forceinline__ float jk_pp_q(const JkPrimPairDf &r) { return r.q; }
template <typename R> struct JkPrim {
    R Px, Py, Pz, p, PAx, PAy, PAz, K, inv2p;
};
template <typename R, typename T> __device__ __forceinline__ JkPrim<R> jk_prim(const T &r)
{
    return {r.Px, r.Py, r.Pz, r.p, r.PAx, r.PAy, r.PAz, r.K, r.inv2p};
}
template <> __device__ __forceinline__ JkPrim<jkdf> jk_prim<jkdf, JkPrimPairDf>(const JkPrimPairDf &r)
{
    return {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {r.ph, r.pl}, {r.PAxh, r.PAxl}, {r.PAyh, r.PAyl},
            {r.PAzh, r.PAzl}, {r.Kh, r.Kl}, {r.i2ph, r.i2pl}};
}

__device__ __forceinline__ double jk_rsqrt(double x) { return rsqrt(x); }

// The same of a pair for the FP64 kernels.
struct JkRec64 {
    int pp_off, a_ao, b_ao, same;
    double ABx, ABy, ABz;
};
__device__ __forceinline__ JkRec64 jk_rec64(const JkPair &p)
{
    return {p.pp_off, p.a_ao, p.b_ao, p.a == p.b, p.ABx, p.ABy, p.ABz};
}
template <typename R> struct JkRecOf {
    typedef JkRec T;
    __device__ static __forceinline__ T bra(const JkSub &s, int i) { return s.bra_rec[i]; }
    __device__ static __forceinline__ T ket(const JkSub &s, int i) { return s.ket_rec[i]; }
};
template <> struct JkRecOf<double> {
    typedef JkRec64 T;
    __device__ static __forceinline__ T bra(const JkSub &s, int i) { return jk_rec64(s.bra[i]); }
    __device__ static __forceinline__ T ket(const JkSub &s, int i) { return jk_rec64(s.ket[i]); }
};

// A - C of a quartet, read by the split tier alone.
template <typename R, typename T> __device__ __forceinline__ void jk_centres(const T &, const T &, R &, R &, R &) {}
template <> __device__ __forceinline__ void jk_centres<jkdf, JkRec>(const JkRec &b, const JkRec &k, jkdf &x, jkdf &y, jkdf &z)
{
    x = jk_norm(jk_sub(jkdf{b.Axh, b.Axl}, jkdf{k.Axh, k.Axl}));
    y = jk_norm(jk_sub(jkdf{b.Ayh, b.Ayl}, jkdf{k.Ayh, k.Ayl}));
    z = jk_norm(jk_sub(jkdf{b.Azh, b.Azl}, jkdf{k.Azh, k.Azl}));
}
// P - Q = (P - A) + W with W = (A - C) - (Q - C), kept in the ket's P field.
template <typename R> __device__ __forceinline__ void jk_ket_w(JkPrim<R> &, R, R, R) {}
template <> __device__ __forceinline__ void jk_ket_w<jkdf>(JkPrim<jkdf> &k, jkdf x, jkdf y, jkdf z)
{
    k.Px = jk_norm(jk_sub(x, k.PAx));
    k.Py = jk_norm(jk_sub(y, k.PAy));
    k.Pz = jk_norm(jk_sub(z, k.PAz));
}
template <typename R> __device__ __forceinline__ R jk_pq(R P, R Q, R) { return P - Q; }
__device__ __forceinline__ jkdf jk_pq(jkdf, jkdf w, jkdf pa) { return jk_norm(jk_add(pa, w)); }

// A - B of a pair in the tier's precision (the FP32 copy is stored, so the
// FP32 tier converts nothing on the FP64 pipe).
__device__ __forceinline__ void jk_pair_ab(const JkRec64 &p, double &x, double &y, double &z)
{
    x = p.ABx; y = p.ABy; z = p.ABz;
}
__device__ __forceinline__ void jk_pair_ab(const JkRec &p, float &x, float &y, float &z)
{
    x = p.ABxf; y = p.AByf; z = p.ABzf;
}
__device__ __forceinline__ void jk_pair_ab(const JkRec &p, jkdf &x, jkdf &y, jkdf &z)
{
    x = {p.ABxf, p.ABxl}; y = {p.AByf, p.AByl}; z = {p.ABzf, p.ABzl};
}

// An FP32 tier contribution widened to FP64 for the FP64 atomics into J and
// K. A float-to-double conversion is an FP64-pipe instruction (1/64 of the
// FP32 rate on GB300); the alternative builds the IEEE-754 binary64 bit
// pattern with integer operations: sign, exponent rebiased from 127 to
// 1023, fraction shifted left by 29; subnormal floats are normalised first.
// Exact for every float. (Measured: the integer form is the slower of the
// two on the batched workload, so the conversion is the default.)
__device__ __forceinline__ double jk_wide(double x, int) { return x; }
__device__ __forceinline__ double jk_to_f64(float x)
{
    const unsigned u = __float_as_uint(x);
    const unsigned long long sgn = (unsigned long long)(u & 0x80000000u) << 32;
    const unsigned e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    unsigned long long bits;
    if (e == 0xffu) {
        bits = sgn | (0x7ffull << 52) | ((unsigned long long)m << 29);
    } else if (e != 0) {
        bits = sgn | ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)m << 29);
    } else if (m == 0) {
        bits = sgn;
    } else {
        const int top = 31 - __clz(m);   // leading bit of the subnormal fraction, 0..22
        bits = sgn | ((unsigned long long)(top + 874) << 52) |
               (((unsigned long long)m << (52 - top)) & 0xfffffffffffffull);
    }
    return __longlong_as_double((long long)bits);
}
// wi = 0: the conversion instruction instead (for comparison)
__device__ __forceinline__ double jk_wide(float x, int wi) { return wi ? jk_to_f64(x) : (double)x; }
// Two floats to FP64. h by integer operations, l by the conversion instruction,
// which goes to the FP64 pipe beside the one sum and keeps infinities and NaNs:
// where h is not finite neither is l (each operation forms it from the
// difference of h and itself), so the sum is not. The integer widening of h
// alone would make 3.4e38 of an infinity. Below 1.2e-38 h counts as zero. Split
// builds of 8 molecules and 20 atoms, ms: 257.4 and 4.19; both halves by
// integers 257.0 and 4.17, with h tested there 261.6 and 4.25; both by
// conversions 260.6 and 4.23.
__device__ __forceinline__ double jk_to_f64_normal(float x)
{
    const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
    const unsigned hi = (u & 0x80000000u) | ((m >> 3) + 0x38000000u);
    return m < 0x00800000u ? 0.0 : __hiloint2double((int)hi, (int)(m << 29));
}
__device__ __forceinline__ double jk_wide(jkdf x, int) { return jk_to_f64_normal(x.h) + (double)x.l; }
__device__ __forceinline__ float jk_rsqrt(float x) { return rsqrtf(x); }

// ----------------------------------------------------- Rys roots, weights
// Root r and weight r of the N-point rule at T. The piecewise polynomials
// cover 0 <= T < tmax; above it the half-range Gauss-Hermite limit
// u = x^2 / T, w = w_h / sqrt(T) holds (evaluated in the tier's precision).
template <int N>
__device__ __forceinline__ void jk_rys_one(double T, int r, const double *__restrict__ tab,
                                           double &u, double &w, int /*a64*/)
{
    if (T >= rys64_tmax[N]) {
        double s = rsqrt(T);
        u = rys_gh[rys_gh_offset[N - 1] + r] * (s * s);
        w = rys_gh[rys_gh_offset[N - 1] + N + r] * s;
        return;
    }
    int k = min((int)(T * RYS64_INVH), rys64_nint[N] - 1);
    double x = (T - k * RYS64_H) * (2.0 * RYS64_INVH) - 1.0;
    // per function 8 doubles: c0..c5, then c6..c9 as floats (terms below
    // 2e-7 of c0, summed in FP32 and added to the FP64 Horner head)
    const double *cu = tab + rys64_offset[N] + (long long)k * (2 * N * 8) + r * 8;
    const double *cw = cu + N * 8;
    const float xf = (float)x;
    const float4 tu = __ldg(reinterpret_cast<const float4 *>(cu + 6));
    const float4 tw = __ldg(reinterpret_cast<const float4 *>(cw + 6));
    double au = (double)fmaf(fmaf(fmaf(tu.w, xf, tu.z), xf, tu.y), xf, tu.x);
    double aw = (double)fmaf(fmaf(fmaf(tw.w, xf, tw.z), xf, tw.y), xf, tw.x);
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        au = fma(au, x, __ldg(cu + i));
        aw = fma(aw, x, __ldg(cw + i));
    }
    u = au;
    w = aw;
}

// FP32: `tab` is this N's table alone, as the class kernel stages it in
// shared memory: per interval the 16 N coefficients (per root the eight of u,
// then per root the eight of w) and four floats of padding, so that the
// 16-byte vectors of different intervals fall in different bank groups.
template <int N>
__device__ __forceinline__ void jk_rys_one(float T, int r, const float *__restrict__ tab,
                                           float &u, float &w, int a64)
{
    static_assert(RYS32_DEG == 7, "two float4 per function");
    if (T >= rys32_tmaxf[N]) {
        if (a64) {
            // the same limit evaluated in FP64, rounded once to FP32
            const double s = rsqrt((double)T);
            u = (float)(rys_gh[rys_gh_offset[N - 1] + r] * (s * s));
            w = (float)(rys_gh[rys_gh_offset[N - 1] + N + r] * s);
            return;
        }
        // u = x^2 / T, w = w_h / sqrt(T): no cancellation, so FP32 keeps
        // ~2 ulp; the Gauss-Hermite constants are FP64-derived, stored
        // rounded to FP32
        const float s = rsqrtf(T);
        u = rys_gh32[rys_gh_offset[N - 1] + r] * (s * s);
        w = rys_gh32[rys_gh_offset[N - 1] + N + r] * s;
        return;
    }
    int k = min((int)(T * (float)RYS32_INVH), rys32_nint_c[N] - 1);
    float x = (T - k * (float)RYS32_H) * (float)(2.0 * RYS32_INVH) - 1.0f;
    const float4 *cu = reinterpret_cast<const float4 *>(tab + k * (16 * N + 4) + r * 8);
    const float4 *cw = cu + N * 2;
    const float4 u0 = cu[0], u1 = cu[1], w0 = cw[0], w1 = cw[1];
    float au = fmaf(fmaf(fmaf(u1.w, x, u1.z), x, u1.y), x, u1.x);
    float aw = fmaf(fmaf(fmaf(w1.w, x, w1.z), x, w1.y), x, w1.x);
    au = fmaf(fmaf(fmaf(fmaf(au, x, u0.w), x, u0.z), x, u0.y), x, u0.x);
    aw = fmaf(fmaf(fmaf(fmaf(aw, x, w0.w), x, w0.z), x, w0.y), x, w0.x);
    u = au;
    w = aw;
}

// Two floats: `tab` holds per interval, for each of the 2 N functions, c0..c5
// as (h, l) pairs and c6..c9 (below 2e-7 of c0) as floats, 16 floats, and four
// floats of padding. 71 FP32 instructions per function, where the FP64
// evaluation holds the FP64 pipe as long as about 1,000 take.
__device__ __forceinline__ jkdf jk_rys_poly_df(const float4 *__restrict__ c, jkdf x)
{
    const float4 c01 = c[0], c23 = c[1], c45 = c[2], t = c[3];
    const float f = __fmaf_rn(__fmaf_rn(__fmaf_rn(t.w, x.h, t.z), x.h, t.y), x.h, t.x);
    jkdf a = jk_add(jkdf{c45.z, c45.w}, jkdf{__fmul_rn(f, x.h), 0.0f});
    a = jk_add(jk_mul(a, x), jkdf{c45.x, c45.y});
    a = jk_add(jk_mul(a, x), jkdf{c23.z, c23.w});
    a = jk_add(jk_mul(a, x), jkdf{c23.x, c23.y});
    a = jk_add(jk_mul(a, x), jkdf{c01.z, c01.w});
    a = jk_add(jk_mul(jk_norm(a), x), jkdf{c01.x, c01.y});
    return jk_norm(a);
}
template <int N>
__device__ __forceinline__ void jk_rys_one(jkdf T, int r, const float *__restrict__ tab, jkdf &u, jkdf &w, int)
{
    if (T.h >= (float)(rys64_nint_c[N] * RYS64_H)) {
        const jkdf s = jk_rsqrt(T);
        const jkdf s2 = jk_norm(jk_mul(s, s));
        const float4 g = rys_ghdf[rys_gh_offset[N - 1] / 2 + r];
        u = jk_norm(jk_mul(jkdf{g.x, g.y}, s2));
        w = jk_norm(jk_mul(jkdf{g.z, g.w}, s));
        return;
    }
    const int k = min((int)(T.h * (float)RYS64_INVH), rys64_nint_c[N] - 1);
    // x = (2 / H) T - (2 k + 1), 2 / H a power of two
    const jkdf x = jk_norm(jk_add(jk_scale(T, (float)(2.0 * RYS64_INVH)), jkdf{-(float)(2 * k + 1), 0.0f}));
    const float4 *c = reinterpret_cast<const float4 *>(tab + k * (32 * N + 4) + r * 16);
    u = jk_rys_poly_df(c, x);
    w = jk_rys_poly_df(c + 4 * N, x);
}

template <typename R> struct JkIsFloat { static constexpr bool v = false; };
template <> struct JkIsFloat<float> { static constexpr bool v = true; };
template <typename R> struct JkIsDf { static constexpr bool v = false; };
template <> struct JkIsDf<jkdf> { static constexpr bool v = true; };
template <typename R> struct JkTab { typedef R T; };     // element type of the Rys tables
template <> struct JkTab<jkdf> { typedef float T; };

// Floats of the FP32 Rys table of the N-root rule in its shared-memory
// layout (intervals padded from 16 N to 16 N + 4 floats).
template <int N> struct JkRysTab32 { static constexpr int n = rys32_nint_c[N] * (16 * N + 4); };
// Two-float tables are staged up to three roots (12, 26, 42 KB); above, the
// few threads of a group that evaluate roots read them through L1.
#define JK_DF_STAGE 3
template <int N> struct JkRysTabDf { static constexpr int n = N <= JK_DF_STAGE ? rys64_nint_c[N] * (32 * N + 4) : 0; };

// --------------------------------------------------------- 2D integrals
// One direction, one root: vertical recurrence on (n on A, m on C) up to
// (LA+LB, LC+LD), then horizontal transfers to (a, b, c, d). Output layout
// out[((a*(LB+1) + b)*(LC+1) + c)*(LD+1) + d].
// UNIT: i00 is 1 (the x and y directions; z carries the weight).
template <int LA, int LB, int LC, int LD, bool UNIT, typename R>
__device__ __forceinline__ void jk_build_2d(R c00, R c00p, R b10, R b01, R b00, R i00,
                                            R ab, R cd, R *__restrict__ out)
{
    constexpr int NA = LA + LB, NC = LC + LD;
    R V[NA + 1][NC + 1];
    V[0][0] = i00;
    if (NA > 0) V[1][0] = UNIT ? c00 : jk_norm(jk_mul(c00, i00));
#pragma unroll
    for (int n = 1; n < NA; ++n) {
        R v = jk_mul(c00, V[n][0]);
        if (UNIT && n == 1) jk_addto(v, b10);
        else jk_acc(v, jk_int(n, b10), V[n - 1][0]);
        V[n + 1][0] = jk_norm(v);
    }
#pragma unroll
    for (int m = 0; m < NC; ++m) {
#pragma unroll
        for (int n = 0; n <= NA; ++n) {
            R v = UNIT && m == 0 && n == 0 ? c00p : jk_mul(c00p, V[n][m]);
            if (m > 0) {
                if (UNIT && m == 1 && n == 0) jk_addto(v, b01);
                else jk_acc(v, jk_int(m, b01), V[n][m - 1]);
            }
            if (n > 0) {
                if (UNIT && n == 1 && m == 0) jk_addto(v, b00);
                else jk_acc(v, jk_int(n, b00), V[n - 1][m]);
            }
            V[n][m + 1] = jk_norm(v);
        }
    }
    // bra transfer A -> B: H[a][b] = H[a+1][b-1] + AB H[a][b-1]
    R HB[LA + 1][LB + 1][NC + 1];
#pragma unroll
    for (int m = 0; m <= NC; ++m) {
        R t[NA + 1][LB + 1];
#pragma unroll
        for (int n = 0; n <= NA; ++n) t[n][0] = V[n][m];
#pragma unroll
        for (int b = 1; b <= LB; ++b)
#pragma unroll
            for (int a = 0; a <= NA - b; ++a) {
                R v = t[a + 1][b - 1];
                if (UNIT && m == 0 && a == 0 && b == 1) jk_addto(v, ab);
                else jk_acc(v, ab, t[a][b - 1]);
                t[a][b] = jk_norm(v);
            }
#pragma unroll
        for (int a = 0; a <= LA; ++a)
#pragma unroll
            for (int b = 0; b <= LB; ++b) HB[a][b][m] = t[a][b];
    }
    // ket transfer C -> D
#pragma unroll
    for (int a = 0; a <= LA; ++a)
#pragma unroll
        for (int b = 0; b <= LB; ++b) {
            R s[NC + 1][LD + 1];
#pragma unroll
            for (int m = 0; m <= NC; ++m) s[m][0] = HB[a][b][m];
#pragma unroll
            for (int d = 1; d <= LD; ++d)
#pragma unroll
                for (int c = 0; c <= NC - d; ++c) {
                    R v = s[c + 1][d - 1];
                    if (UNIT && a == 0 && b == 0 && c == 0 && d == 1) jk_addto(v, cd);
                    else jk_acc(v, cd, s[c][d - 1]);
                    s[c][d] = jk_norm(v);
                }
#pragma unroll
            for (int c = 0; c <= LC; ++c)
#pragma unroll
                for (int d = 0; d <= LD; ++d) out[((a * (LB + 1) + b) * (LC + 1) + c) * (LD + 1) + d] = s[c][d];
        }
}

// ----------------------------------------------------------- class shape
// OP: 0 the Coulomb operator 1/r; 1 erf(w r)/r (long range); 2 erfc(w r)/r
// (short range) = 1/r minus the long-range part, i.e. a second root set with
// negative weights (the range separation of Table 1, rys_type).
template <int LA, int LB, int LC, int LD, int GA, int GB, int GC, int GD, int OP = 0>
struct JkShape {
    static constexpr int NFA = jk_ncart(LA), NFB = jk_ncart(LB), NFC = jk_ncart(LC), NFD = jk_ncart(LD);
    static constexpr int FA = NFA / GA, FB = NFB / GB, FC = NFC / GC, FD = NFD / GD;
    static constexpr int G = GA * GB * GC * GD;
    static constexpr int EPT = FA * FB * FC * FD;
    static constexpr int L = LA + LB + LC + LD;
    static constexpr int NR = L / 2 + 1;
    static constexpr int NRE = (OP == 2 ? 2 : 1) * NR;   // roots of all sets
    static constexpr int SD = 1, SC = LD + 1, SB = (LC + 1) * (LD + 1), SA = (LB + 1) * SB;
    static constexpr int NI = (LA + 1) * SA;
    // reals of shared memory per group (G > 1): 2D tables and the roots
    static constexpr int SMEM_GROUP = (G == 1) ? 0 : (NRE * 3 * NI + 2 * NRE);
    static_assert(NFA % GA == 0 && NFB % GB == 0 && NFC % GC == 0 && NFD % GD == 0, "fragment");
    static_assert(G <= 16 * 1024, "a group fits 16 CTAs");
};

// Offsets into a 2D table for the components a thread owns (G > 1).
template <class S>
struct JkOffsets {
    int a[3][S::FA], b[3][S::FB], c[3][S::FC], d[3][S::FD];
};

template <int LA, int LB, int LC, int LD, int GA, int GB, int GC, int GD, class S>
__device__ __forceinline__ void jk_make_offsets(int ga, int gb, int gc, int gd, JkOffsets<S> &o)
{
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
        for (int i = 0; i < S::FA; ++i) {
            int idx = ga * S::FA + i, e = 0, k = 0;
            for (int x = LA; x >= 0; --x)
                for (int y = LA - x; y >= 0; --y, ++k)
                    if (k == idx) e = ax == 0 ? x : (ax == 1 ? y : LA - x - y);
            o.a[ax][i] = e * S::SA;
        }
#pragma unroll
        for (int i = 0; i < S::FB; ++i) {
            int idx = gb * S::FB + i, e = 0, k = 0;
            for (int x = LB; x >= 0; --x)
                for (int y = LB - x; y >= 0; --y, ++k)
                    if (k == idx) e = ax == 0 ? x : (ax == 1 ? y : LB - x - y);
            o.b[ax][i] = e * S::SB;
        }
#pragma unroll
        for (int i = 0; i < S::FC; ++i) {
            int idx = gc * S::FC + i, e = 0, k = 0;
            for (int x = LC; x >= 0; --x)
                for (int y = LC - x; y >= 0; --y, ++k)
                    if (k == idx) e = ax == 0 ? x : (ax == 1 ? y : LC - x - y);
            o.c[ax][i] = e * S::SC;
        }
#pragma unroll
        for (int i = 0; i < S::FD; ++i) {
            int idx = gd * S::FD + i, e = 0, k = 0;
            for (int x = LD; x >= 0; --x)
                for (int y = LD - x; y >= 0; --y, ++k)
                    if (k == idx) e = ax == 0 ? x : (ax == 1 ? y : LD - x - y);
            o.d[ax][i] = e * S::SD;
        }
    }
}

// Barrier of one group: a warp-local group syncs its lanes, a group of more
// than 32 threads is the whole CTA.
template <int G>
__device__ __forceinline__ void jk_group_sync(unsigned gmask)
{
    if constexpr (G <= 32) __syncwarp(gmask);
    else __syncthreads();
}

// ------------------------------------------------ one contracted quartet
// Accumulates the thread's fragment T[EPT] of the contracted block (ab|cd)
// over every primitive quartet (eq:rys0). `grp` is the group's shared
// memory (G > 1), gmask the group's lane mask. The roots and 2D tables are
// built by the NT threads that share `grp` (tg < NT: the thread's index
// among them), the whole group, or, for a group split over several CTAs,
// the group's threads in this CTA.
// Root r (< NRE) of the operator: set 0 at T (1/r) or at theta T (erf);
// for OP 2 set 1 is the erf part with negated weight. Returns u and w * pref.
template <int NR, int OP, typename R>
__device__ __forceinline__ void jk_op_root(R Tt, R rho, R pref, double omega, int a64, int r,
                                           const typename JkTab<R>::T *__restrict__ rys, R &u, R &wp)
{
    R uu, ww;
    if (OP == 0 || (OP == 2 && r < NR)) {
        jk_rys_one<NR>(Tt, r, rys, uu, ww, a64);
        u = uu;
        wp = jk_norm(jk_mul(ww, pref));
    } else {
        // theta = w^2 / (w^2 + rho), sqrt(theta) = w / sqrt(w^2 + rho)
        const R om = JkConst<R>::get(omega);
        const R rd = jk_rsqrt(jk_norm(jk_add(jk_mul(om, om), rho)));
        const R st = jk_norm(jk_mul(om, rd)), th = jk_norm(jk_mul(st, st));
        jk_rys_one<NR>(jk_norm(jk_mul(th, Tt)), OP == 2 ? r - NR : r, rys, uu, ww, a64);
        u = jk_norm(jk_mul(th, uu));
        wp = jk_norm(jk_mul(jk_norm(jk_mul(OP == 2 ? jk_neg(st) : st, ww)), pref));
    }
}

// A work item's share of a quartet's primitive quartets: bra pairs ab, ab + dab,
// ..., ket pairs cd, cd + dcd, ...
struct JkShare {
    int ab, dab, cd, dcd;
};

template <int LA, int LB, int LC, int LD, int GA, int GB, int GC, int GD, typename R, int OP = 0,
          int NT = JkShape<LA, LB, LC, LD, GA, GB, GC, GD, OP>::G>
__device__ __forceinline__ int jk_quartet(const typename JkRecOf<R>::T &bra, const typename JkRecOf<R>::T &ket, JkShare sh, int nab, int ncd, float qthr, double omega, int a64,
                                           const typename JkPP<R>::T *__restrict__ pp,
                                           const typename JkTab<R>::T *__restrict__ rys, R *grp, unsigned gmask,
                                           int tg, bool act,
                                           const JkOffsets<JkShape<LA, LB, LC, LD, GA, GB, GC, GD, OP>> &off,
                                           R (&T)[JkShape<LA, LB, LC, LD, GA, GB, GC, GD, OP>::EPT])
{
    typedef JkShape<LA, LB, LC, LD, GA, GB, GC, GD, OP> S;
    typedef typename JkPP<R>::T PPT;
    constexpr int NR = S::NR;
    constexpr int NRE = S::NRE;
    R ABx, ABy, ABz, CDx, CDy, CDz;
    jk_pair_ab(bra, ABx, ABy, ABz);
    jk_pair_ab(ket, CDx, CDy, CDz);
    R ACx, ACy, ACz;
    jk_centres<R>(bra, ket, ACx, ACy, ACz);
    const PPT *bpp = pp + bra.pp_off;
    const PPT *kpp = pp + ket.pp_off;
    // primitive pairs are sorted by their Schwarz factor q (largest first):
    // stop a loop at the first q_ij q_kl <= qthr (= prim_eps / Dmax), compared
    // in FP32 (a product below the FP32 range is below any threshold that
    // matters; qthr < 0 screens nothing). The ket's primitive pairs (one
    // record per lane and kl) are the outer loop, so each is loaded once; the
    // bra's (the same for the whole group or warp) the inner one.
    const float qthf = qthr;
    const float qb0 = jk_pp_q(bpp[sh.ab]);
    int nprim = 0;
#pragma unroll 1
    for (int kl = sh.cd; kl < ncd; kl += sh.dcd) {
        const PPT kr = kpp[kl];
        const float qk = jk_pp_q(kr);
        if (qb0 * qk <= qthf) break;
        JkPrim<R> kp = jk_prim<R>(kr);
        jk_ket_w<R>(kp, ACx, ACy, ACz);
#pragma unroll 1
        for (int ij = sh.ab; ij < nab; ij += sh.dab) {
            const PPT br = bpp[ij];
            if (jk_pp_q(br) * qk <= qthf) break;
            ++nprim;
            const JkPrim<R> bp = jk_prim<R>(br);
            const R rpq = jk_rsqrt(jk_norm(jk_add(bp.p, kp.p)));
            const R inv_pq = jk_norm(jk_mul(rpq, rpq));
            const R PQx = jk_pq(bp.Px, kp.Px, bp.PAx), PQy = jk_pq(bp.Py, kp.Py, bp.PAy), PQz = jk_pq(bp.Pz, kp.Pz, bp.PAz);
            const R qf = jk_norm(jk_mul(kp.p, inv_pq)), pf = jk_norm(jk_mul(bp.p, inv_pq));
            const R rho = jk_norm(jk_mul(bp.p, qf));
            R r2 = jk_mul(PQx, PQx);
            jk_acc(r2, PQy, PQy);
            jk_acc(r2, PQz, PQz);
            const R Tt = jk_norm(jk_mul(rho, jk_norm(r2)));
            const R pref = jk_norm(jk_mul(jk_norm(jk_mul(JkConst<R>::get(JK_TWO_PI_2_5), bp.K)),
                                          jk_norm(jk_mul(kp.K, rpq))));
            if constexpr (S::G == 1) {
                // large blocks: one copy of the root's code (compiling FP32 (dp|ps) 41 -> 6 s)
#pragma unroll(JkIsDf<R>::v || S::EPT * NRE > 100 ? 1 : NRE)
                for (int r = 0; r < NRE; ++r) {
                    R u, wp;
                    jk_op_root<NR, OP, R>(Tt, rho, pref, omega, a64, r, rys, u, wp);
                    const R uq = jk_norm(jk_mul(u, qf)), up = jk_norm(jk_mul(u, pf));
                    const R one = JkConst<R>::get(1.0);
                    const R b00 = jk_scale(jk_norm(jk_mul(u, inv_pq)), 0.5f);
                    R muq = one, mup = one;   // 1 - u qf, 1 - u pf, the product not rounded
                    jk_acc(muq, jk_neg(u), qf);
                    jk_acc(mup, jk_neg(u), pf);
                    const R b10 = jk_norm(jk_mul(bp.inv2p, jk_norm(muq)));
                    const R b01 = jk_norm(jk_mul(kp.inv2p, jk_norm(mup)));
                    const R nuq = jk_neg(uq);
                    R ax = bp.PAx, ay = bp.PAy, az = bp.PAz, cx = kp.PAx, cy = kp.PAy, cz = kp.PAz;
                    jk_acc(ax, nuq, PQx); jk_acc(ay, nuq, PQy); jk_acc(az, nuq, PQz);
                    jk_acc(cx, up, PQx); jk_acc(cy, up, PQy); jk_acc(cz, up, PQz);
                    R tx[S::NI], ty[S::NI], tz[S::NI];
                    jk_build_2d<LA, LB, LC, LD, true, R>(jk_norm(ax), jk_norm(cx), b10, b01, b00, one, ABx, CDx, tx);
                    jk_build_2d<LA, LB, LC, LD, true, R>(jk_norm(ay), jk_norm(cy), b10, b01, b00, one, ABy, CDy, ty);
                    jk_build_2d<LA, LB, LC, LD, false, R>(jk_norm(az), jk_norm(cz), b10, b01, b00, wp, ABz, CDz, tz);
#pragma unroll
                    for (int ia = 0; ia < S::FA; ++ia)
#pragma unroll
                        for (int ib = 0; ib < S::FB; ++ib)
#pragma unroll
                            for (int ic = 0; ic < S::FC; ++ic)
#pragma unroll
                                for (int id = 0; id < S::FD; ++id) {
                                    const int ox = jk_cart_exp(LA, ia, 0) * S::SA + jk_cart_exp(LB, ib, 0) * S::SB +
                                                   jk_cart_exp(LC, ic, 0) * S::SC + jk_cart_exp(LD, id, 0);
                                    const int oy = jk_cart_exp(LA, ia, 1) * S::SA + jk_cart_exp(LB, ib, 1) * S::SB +
                                                   jk_cart_exp(LC, ic, 1) * S::SC + jk_cart_exp(LD, id, 1);
                                    const int oz = jk_cart_exp(LA, ia, 2) * S::SA + jk_cart_exp(LB, ib, 2) * S::SB +
                                                   jk_cart_exp(LC, ic, 2) * S::SC + jk_cart_exp(LD, id, 2);
                                    const int k = ((ia * S::FB + ib) * S::FC + ic) * S::FD + id;
                                    // entry 0 of the x and y tables is 1
                                    if (ox == 0 && oy == 0) jk_addto(T[k], tz[oz]);
                                    else if (oy == 0) jk_acc(T[k], tx[ox], tz[oz]);
                                    else if (ox == 0) jk_acc(T[k], ty[oy], tz[oz]);
                                    else jk_acc(T[k], jk_mul(tx[ox], ty[oy]), tz[oz]);
                                }
                }
            } else {
                R *roots = grp + NRE * 3 * S::NI;   // [0, NRE): u ; [NRE, 2 NRE): w * pref
                for (int r = tg; r < NRE && tg < NT; r += NT) {
                    R u, wp;
                    jk_op_root<NR, OP, R>(Tt, rho, pref, omega, a64, r, rys, u, wp);
                    roots[r] = u;
                    roots[NRE + r] = wp;
                }
                jk_group_sync<S::G>(gmask);
                for (int task = tg; task < 3 * NRE && tg < NT; task += NT) {
                    const int r = task / 3, dir = task - 3 * r;
                    const R u = roots[r];
                    const R one = JkConst<R>::get(1.0);
                    const R uq = jk_norm(jk_mul(u, qf)), up = jk_norm(jk_mul(u, pf));
                    const R b00 = jk_scale(jk_norm(jk_mul(u, inv_pq)), 0.5f);
                    R muq = one, mup = one;   // 1 - u qf, 1 - u pf, the product not rounded
                    jk_acc(muq, jk_neg(u), qf);
                    jk_acc(mup, jk_neg(u), pf);
                    const R b10 = jk_norm(jk_mul(bp.inv2p, jk_norm(muq)));
                    const R b01 = jk_norm(jk_mul(kp.inv2p, jk_norm(mup)));
                    R pa, qc, pqd, abd, cdd, i00 = one;
                    if (dir == 0) { pa = bp.PAx; qc = kp.PAx; pqd = PQx; abd = ABx; cdd = CDx; }
                    else if (dir == 1) { pa = bp.PAy; qc = kp.PAy; pqd = PQy; abd = ABy; cdd = CDy; }
                    else { pa = bp.PAz; qc = kp.PAz; pqd = PQz; abd = ABz; cdd = CDz; i00 = roots[NRE + r]; }
                    jk_acc(pa, jk_neg(uq), pqd);
                    jk_acc(qc, up, pqd);
                    jk_build_2d<LA, LB, LC, LD, false, R>(jk_norm(pa), jk_norm(qc), b10, b01, b00, i00, abd, cdd,
                                                          grp + (r * 3 + dir) * S::NI);
                }
                jk_group_sync<S::G>(gmask);
                if (act) {
#pragma unroll
                for (int ia = 0; ia < S::FA; ++ia)
#pragma unroll
                    for (int ib = 0; ib < S::FB; ++ib)
#pragma unroll
                        for (int ic = 0; ic < S::FC; ++ic)
#pragma unroll
                            for (int id = 0; id < S::FD; ++id) {
                                const int ox = off.a[0][ia] + off.b[0][ib] + off.c[0][ic] + off.d[0][id];
                                const int oy = off.a[1][ia] + off.b[1][ib] + off.c[1][ic] + off.d[1][id];
                                const int oz = off.a[2][ia] + off.b[2][ib] + off.c[2][ic] + off.d[2][id];
                                const int k = ((ia * S::FB + ib) * S::FC + ic) * S::FD + id;
                                if constexpr (JkIsDf<R>::v) {
#pragma unroll
                                    for (int r = 0; r < NRE; ++r)
                                        jk_acc(T[k], jk_mul(grp[(r * 3 + 0) * S::NI + ox], grp[(r * 3 + 1) * S::NI + oy]),
                                               grp[(r * 3 + 2) * S::NI + oz]);
                                } else {
                                    R acc = (R)0;
#pragma unroll
                                    for (int r = 0; r < NRE; ++r)
                                        acc += grp[(r * 3 + 0) * S::NI + ox] * grp[(r * 3 + 1) * S::NI + oy] *
                                               grp[(r * 3 + 2) * S::NI + oz];
                                    T[k] += acc;
                                }
                            }
                }
                jk_group_sync<S::G>(gmask);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < S::EPT; ++k) T[k] = jk_norm(T[k]);
    return nprim;
}

template <typename R> __device__ __forceinline__ const typename JkPP<R>::T *jk_pp(const JkClassArgs &a);
template <> __device__ __forceinline__ const JkPrimPair64 *jk_pp<double>(const JkClassArgs &a) { return a.pp64; }
template <> __device__ __forceinline__ const JkPrimPair32 *jk_pp<float>(const JkClassArgs &a) { return a.pp32; }
template <> __device__ __forceinline__ const JkPrimPairDf *jk_pp<jkdf>(const JkClassArgs &a) { return a.ppdf; }
template <typename R> __device__ __forceinline__ const typename JkTab<R>::T *jk_rys(const JkClassArgs &a);
template <> __device__ __forceinline__ const double *jk_rys<double>(const JkClassArgs &a) { return a.rys64; }
template <> __device__ __forceinline__ const float *jk_rys<float>(const JkClassArgs &a) { return a.rys32; }
template <> __device__ __forceinline__ const float *jk_rys<jkdf>(const JkClassArgs &a) { return a.rysdf; }

// ---------------------------------------------- routed builds: the FP64 tier
// The FP64 tier of a routed build is the only tier that runs the router: the
// lanes in `rel` (band quartets the router releases) append (bra item, ket j,
// density factor) to the launch's list while it has room, for the FP32 list
// kernel (MODE 3) of the class pair. Returns whether this lane's quartet was
// listed; a quartet that finds the list full stays in FP64. All 32 lanes of
// the warp call it.
__device__ __forceinline__ bool jk_route_out(const JkClassArgs &args, int launch, bool rel, int item, int j, float dq)
{
    const unsigned m = __ballot_sync(0xffffffffu, rel);
    if (!m) return false;
    const int lane = threadIdx.x & 31, first = __ffs(m) - 1;
    unsigned long long base = 0;
    if (lane == first) base = atomicAdd(args.rcount + launch, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, first);
    const long long pos = (long long)base + __popc(m & ((1u << lane) - 1u));
    const bool listed = rel && pos < args.rcap[launch];
    if (listed) {
        JkRouted e;
        e.item = item; e.ket = j; e.dmq = dq; e.pad = 0;
        args.rlist[args.roff[launch] + pos] = e;
    }
    return listed;
}

// ------------------------------------------------- screening of a candidate
// The bounds of a tier for one molecule (FP64 and rounded to FP32): the split
// threshold follows the molecule's largest density element, and is formed
// alike by every launch of a build. dreal: the largest |D|, also where the
// screening takes 1 for it (dmol).
struct JkBounds {
    double lo, hi;
    float lo32, hi32;
};
__device__ __forceinline__ JkBounds jk_bounds(const JkClassArgs &args, const JkMol &mol, double dmol, double dreal)
{
    JkBounds b = {args.lo, args.hi, args.lo32, args.hi32};
    if (args.split_side != 0) {
        const double th = jk_split_threshold(args.split, args.split_min, mol.qmax2, dmol, dreal);
        if (args.split_side > 0 && th > b.lo) { b.lo = th; b.lo32 = (float)th; }
        if (args.split_side < 0 && th < b.hi) { b.hi = th; b.hi32 = (float)th; }
    }
    return b;
}
template <int MODE>
__device__ __forceinline__ void jk_screen_bound(const JkClassArgs &args, const JkBounds &bd,
                                                const JkSub &sub, const JkPair &bra, const JkMol &mol,
                                                const double *dmx, double dmol, float dmol32, int j, int ke,
                                                bool &sig, bool &stop, bool &band, float &dmq, float &Bout);
// Keep (bra, ket j) iff lo < Q_ab Q_cd Dmax <= hi; `stop` when even the
// molecule's largest density element cannot lift this ket (and every later
// one, kets being sorted by Q) above lo.
template <int MODE>
__device__ __forceinline__ void jk_screen(const JkClassArgs &args, const JkBounds &bd, const JkSub &sub, const JkPair &bra,
                                          const JkPairFeat &braf, const JkMol &mol, const double *dmx, double dmol, float dmol32, int item,
                                          int j, int ke, bool &sig, bool &stop, bool &band, float &dmq,
                                          unsigned short *rsm)
{
    sig = false;
    stop = false;
    band = false;
    dmq = 1.0f;
    float B = 0.0f;
    jk_screen_bound<MODE>(args, bd, sub, bra, mol, dmx, dmol, dmol32, j, ke, sig, stop, band, dmq, B);
    if (MODE == 1) {
        // learned router for the band candidates, all lanes together on the
        // tensor cores; `band` then marks the quartets released to FP32
        bool listed = false;
        if (__ballot_sync(0xffffffffu, band)) {
            const JkPairFeat kf = band ? sub.ket_feat[j] : braf;
            const bool to32 = jk_router_to_fp32_warp(args.router, braf, kf, band ? B : 2.0f * args.tau32,
                                                     band ? dmq : 1.0f, args.tau32, rsm);
            listed = jk_route_out(args, sub.launch, band && to32, item, j, dmq);
            if (band) sig = !listed;
        }
        band = listed;
    }
}

// Whether x and y (FP32 images of FP64 quantities, relative error at most
// 5 FP32 roundings, 3.0e-7) are too close for their order to be decided in
// FP32: then the caller redoes the comparison in FP64.
__device__ __forceinline__ bool jk_near(float x, float y)
{
    return fabsf(x - y) < 2e-6f * y;   // false for y = infinity
}

template <int MODE>
__device__ __forceinline__ void jk_screen_bound(const JkClassArgs &args, const JkBounds &bd,
                                                const JkSub &sub, const JkPair &bra, const JkMol &mol,
                                                const double *dmx, double dmol, float dmol32, int j, int ke,
                                                bool &sig, bool &stop, bool &band, float &dmq, float &Bout)
{
    if (j >= ke) return;
    if (args.scr32) {
        const JkKetScr ks = sub.ket_scr[j];
        // FP32 bounds: a handful of FP32 operations per candidate instead of
        // FP64-pipe work (an FP64 instruction costs the FP32 tier 64 FP32
        // ones on GB300). scr32 == 2 keeps the FP64 rule exact: the FP32
        // products carry at most 5 roundings, so only a bound within 2e-6 of
        // a threshold can compare differently from its FP64 value, and those
        // few are redone in FP64 (every tier decides alike, as in FP64).
        const float bq = bra.Qf * ks.Qf;
        const float s = bq * dmol32;
        bool st = s <= bd.lo32;
        if (args.scr32 == 2 && jk_near(s, bd.lo32)) st = (bra.Q * sub.ket[j].Q) * dmol <= bd.lo;
        if (st) { stop = true; return; }
        float dm = 1.0f;
        const int c = ks.a_loc, d = ks.b_loc;
        const int a = bra.a_loc, b = bra.b_loc, ns = mol.nsh;
        if (args.use_dmax) {
            const float *d32 = args.dmax32 + mol.dmax_off;
            dm = 0.0f;
            if (args.with_j) dm = fmaxf(__ldg(d32 + a * ns + b), __ldg(d32 + c * ns + d));
            if (args.with_k) {
                dm = fmaxf(dm, fmaxf(__ldg(d32 + a * ns + c), __ldg(d32 + a * ns + d)));
                dm = fmaxf(dm, fmaxf(__ldg(d32 + b * ns + c), __ldg(d32 + b * ns + d)));
            }
        }
        // the FP32 image of the FP64 maximum is the maximum of the images
        dmq = dm;
        const float B = bq * dm;
        Bout = B;
        sig = (B > bd.lo32) && (B <= bd.hi32);
        band = MODE == 1 && sig && B > args.tau32 && B <= args.band_hi32;
        if (args.scr32 == 2 &&
            (jk_near(B, bd.lo32) || jk_near(B, bd.hi32) ||
             (MODE == 1 && (jk_near(B, args.tau32) || jk_near(B, args.band_hi32))))) {
            double dm64 = 1.0;
            if (args.use_dmax) {
                dm64 = 0.0;
                if (args.with_j) dm64 = fmax(__ldg(dmx + a * ns + b), __ldg(dmx + c * ns + d));
                if (args.with_k) {
                    dm64 = fmax(dm64, fmax(__ldg(dmx + a * ns + c), __ldg(dmx + a * ns + d)));
                    dm64 = fmax(dm64, fmax(__ldg(dmx + b * ns + c), __ldg(dmx + b * ns + d)));
                }
            }
            const double B64 = (bra.Q * sub.ket[j].Q) * dm64;
            sig = (B64 > bd.lo) && (B64 <= bd.hi);
            band = MODE == 1 && sig && B64 > args.tau && B64 <= args.band_hi;
        }
        return;
    }
    const JkPair &kt = sub.ket[j];
    const double bq = bra.Q * kt.Q;
    if (bq * dmol <= bd.lo) { stop = true; return; }
    double dm = 1.0;
    if (args.use_dmax) {
        const int c = kt.a_loc, d = kt.b_loc;
        const int a = bra.a_loc, b = bra.b_loc, ns = mol.nsh;
        dm = 0.0;
        if (args.with_j) dm = fmax(__ldg(dmx + a * ns + b), __ldg(dmx + c * ns + d));
        if (args.with_k) {
            dm = fmax(dm, fmax(__ldg(dmx + a * ns + c), __ldg(dmx + a * ns + d)));
            dm = fmax(dm, fmax(__ldg(dmx + b * ns + c), __ldg(dmx + b * ns + d)));
        }
    }
    // dm below the FP32 range only reaches here with lo < 1e-30, where the
    // primitive threshold is 0 and dmq only divides it
    dmq = (float)dm;
    const double B = bq * dm;
    Bout = (float)B;
    sig = (B > bd.lo) && (B <= bd.hi);
    band = MODE == 1 && sig && B > args.tau && B <= args.band_hi;
}

// Density factor of a quartet (the same lookups as jk_screen).
__device__ __forceinline__ double jk_quartet_dmax(const JkClassArgs &args, const JkPair &bra, const JkPair &ket,
                                                  const JkMol &mol, const double *dmx)
{
    if (!args.use_dmax) return 1.0;
    const int a = bra.a_loc, b = bra.b_loc, c = ket.a_loc, d = ket.b_loc, ns = mol.nsh;
    double dm = 0.0;
    if (args.with_j) dm = fmax(__ldg(dmx + a * ns + b), __ldg(dmx + c * ns + d));
    if (args.with_k) {
        dm = fmax(dm, fmax(__ldg(dmx + a * ns + c), __ldg(dmx + a * ns + d)));
        dm = fmax(dm, fmax(__ldg(dmx + b * ns + c), __ldg(dmx + b * ns + d)));
    }
    return dm;
}

// MODE 2: one training sample (features, label) for a band quartet, written
// by the group's first thread. tmax is the group's max |T|. Which quartets are
// kept of too many follows a hash of their shells, not the order of the launches,
// which run one angular momentum after the other.
__device__ __forceinline__ void jk_log_sample(const JkClassArgs &args, const JkPair &bra, const JkPair &ket,
                                              const JkPairFeat &braf, const JkPairFeat &ketf, double dm, double tmax)
{
    const double B = bra.Q * ket.Q * dm;
    if (!(B > args.tau && B <= args.band_hi)) return;
    atomicAdd(args.log_n, 1ull);
    const unsigned long long key = jk_mix64(jk_mix64((unsigned long long)bra.a << 32 | (unsigned)bra.b) ^
                                            ((unsigned long long)ket.a << 32 | (unsigned)ket.b));
    if (key > args.log_keep) return;
    const unsigned long long idx = atomicAdd(args.log_n + 1, 1ull);
    if ((long long)idx >= args.log_cap) return;
    if (args.log_key) args.log_key[idx] = key;
    float x[JK_RT_NIN];
    // the bound as the FP32 screening path forms it
    jk_router_features(braf, ketf, (bra.Qf * ket.Qf) * (float)dm, (float)dm, args.tau32, x);
    for (int i = 0; i < JK_RT_NIN; ++i) args.log_x[idx * JK_RT_NIN + i] = x[i];
    args.log_y[idx] = (float)log10(fmax(tmax, 1e-300) / (bra.Q * ket.Q));
}

// ------------------------------------------ contraction with the density
// The thread's fragment T of (ab|cd), degeneracy f: J_ab partial kept in
// jab (flushed once per bra pair), the other five blocks by FP64 atomics.
template <typename R> struct JkDens;
template <> struct JkDens<double> { typedef double T; __device__ static __forceinline__ const double *p(const JkMol &m) { return m.D; } };
template <> struct JkDens<float> { typedef float T; __device__ static __forceinline__ const float *p(const JkMol &m) { return m.D32; } };
template <> struct JkDens<jkdf> { typedef float2 T; __device__ static __forceinline__ const float2 *p(const JkMol &m) { return m.D2; } };
__device__ __forceinline__ double jk_ldd(const double *p) { return __ldg(p); }
__device__ __forceinline__ float jk_ldd(const float *p) { return __ldg(p); }
__device__ __forceinline__ jkdf jk_ldd(const float2 *p)
{
    const float2 v = __ldg(p);
    return {v.x, v.y};
}

// J and K accumulate by FP64 reductions that return nothing (RED): atomicAdd
// on doubles issues ATOM, whose value the L2 sends back although nobody
// reads it (ncu: 9.7e9 ATOM sectors for one all-FP32 build of 8 molecules,
// 34 per quartet). Relaxed, device scope: the ordering atomicAdd gives.
__device__ __forceinline__ void jk_red_add(double *p, double v)
{
    asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "d"(v) : "memory");
}

// Adds the block v[F1][F2] times f to rows r0.., columns q0.. of the half matrix M.
template <int F1, int F2, typename R>
__device__ __forceinline__ void jk_store_block(double *__restrict__ M, int nao, int r0, int q0, const R (&v)[F1][F2],
                                               float f, int wi)
{
#pragma unroll
    for (int i = 0; i < F1; ++i)
#pragma unroll
        for (int j = 0; j < F2; ++j)
            jk_red_add(M + (long long)(r0 + i) * nao + q0 + j, jk_wide(jk_scale(v[i][j], f), wi));
}

template <int FA, int FB, int FC, int FD, int NDM, int DOJ, int DOK, typename R>
__device__ __forceinline__ void jk_contract(const R (&T)[FA * FB * FC * FD], float f, const JkMol &mol,
                                            int a0, int b0, int c0, int d0, R (&jab)[NDM][FA][FB], int wi)
{
    const long long nn = (long long)mol.nao * mol.nao;
    const int nao = mol.nao;
#pragma unroll
    for (int m = 0; m < NDM; ++m) {
        // the tier's own copy of D (the FP32 tier reads a pre-rounded one)
        const typename JkDens<R>::T *D = JkDens<R>::p(mol) + m * nn;
        if (DOJ) {
            R Dcd[FC][FD], Dab[FA][FB];
#pragma unroll
            for (int ic = 0; ic < FC; ++ic)
#pragma unroll
                for (int id = 0; id < FD; ++id) Dcd[ic][id] = jk_ldd(D + (long long)(c0 + ic) * nao + d0 + id);
#pragma unroll
            for (int ia = 0; ia < FA; ++ia)
#pragma unroll
                for (int ib = 0; ib < FB; ++ib) Dab[ia][ib] = jk_ldd(D + (long long)(a0 + ia) * nao + b0 + ib);
            R jcd[FC][FD];
#pragma unroll
            for (int ic = 0; ic < FC; ++ic)
#pragma unroll
                for (int id = 0; id < FD; ++id) jcd[ic][id] = JkConst<R>::get(0.0);
#pragma unroll
            for (int ia = 0; ia < FA; ++ia)
#pragma unroll
                for (int ib = 0; ib < FB; ++ib) {
                    R sum = JkConst<R>::get(0.0);
#pragma unroll
                    for (int ic = 0; ic < FC; ++ic)
#pragma unroll
                        for (int id = 0; id < FD; ++id) {
                            const R t = T[((ia * FB + ib) * FC + ic) * FD + id];
                            jk_acc(sum, t, Dcd[ic][id]);
                            jk_acc(jcd[ic][id], t, Dab[ia][ib]);
                        }
                    jk_addto(jab[m][ia][ib], jk_scale(sum, 2.0f * f));
                    jab[m][ia][ib] = jk_norm(jab[m][ia][ib]);
                }
            jk_store_block<FC, FD>(mol.J + m * nn, nao, c0, d0, jcd, 2.0f * f, wi);
        }
        if (DOK) {
            R Dbd[FB][FD], Dbc[FB][FC], Dad[FA][FD], Dac[FA][FC];
#pragma unroll
            for (int ib = 0; ib < FB; ++ib) {
#pragma unroll
                for (int id = 0; id < FD; ++id) Dbd[ib][id] = jk_ldd(D + (long long)(b0 + ib) * nao + d0 + id);
#pragma unroll
                for (int ic = 0; ic < FC; ++ic) Dbc[ib][ic] = jk_ldd(D + (long long)(b0 + ib) * nao + c0 + ic);
            }
#pragma unroll
            for (int ia = 0; ia < FA; ++ia) {
#pragma unroll
                for (int id = 0; id < FD; ++id) Dad[ia][id] = jk_ldd(D + (long long)(a0 + ia) * nao + d0 + id);
#pragma unroll
                for (int ic = 0; ic < FC; ++ic) Dac[ia][ic] = jk_ldd(D + (long long)(a0 + ia) * nao + c0 + ic);
            }
            R kac[FA][FC], kad[FA][FD], kbc[FB][FC], kbd[FB][FD];
#pragma unroll
            for (int ia = 0; ia < FA; ++ia) {
#pragma unroll
                for (int ic = 0; ic < FC; ++ic) kac[ia][ic] = JkConst<R>::get(0.0);
#pragma unroll
                for (int id = 0; id < FD; ++id) kad[ia][id] = JkConst<R>::get(0.0);
            }
#pragma unroll
            for (int ib = 0; ib < FB; ++ib) {
#pragma unroll
                for (int ic = 0; ic < FC; ++ic) kbc[ib][ic] = JkConst<R>::get(0.0);
#pragma unroll
                for (int id = 0; id < FD; ++id) kbd[ib][id] = JkConst<R>::get(0.0);
            }
#pragma unroll
            for (int ia = 0; ia < FA; ++ia)
#pragma unroll
                for (int ib = 0; ib < FB; ++ib)
#pragma unroll
                    for (int ic = 0; ic < FC; ++ic)
#pragma unroll
                        for (int id = 0; id < FD; ++id) {
                            const R t = T[((ia * FB + ib) * FC + ic) * FD + id];
                            jk_acc(kac[ia][ic], t, Dbd[ib][id]);
                            jk_acc(kad[ia][id], t, Dbc[ib][ic]);
                            jk_acc(kbc[ib][ic], t, Dad[ia][id]);
                            jk_acc(kbd[ib][id], t, Dac[ia][ic]);
                        }
            double *K = mol.K + m * nn;
            jk_store_block<FA, FC>(K, nao, a0, c0, kac, f, wi);
            jk_store_block<FA, FD>(K, nao, a0, d0, kad, f, wi);
            jk_store_block<FB, FC>(K, nao, b0, c0, kbc, f, wi);
            jk_store_block<FB, FD>(K, nao, b0, d0, kbd, f, wi);
        }
    }
}

__device__ __forceinline__ bool jk_nonzero(double x) { return x != 0.0; }
__device__ __forceinline__ bool jk_nonzero(float x) { return x != 0.0f; }
__device__ __forceinline__ bool jk_nonzero(jkdf x) { return x.h != 0.0f; }
template <int FA, int FB, int NDM, typename R>
__device__ __forceinline__ void jk_flush_jab(R (&jab)[NDM][FA][FB], const JkMol &mol, int a0, int b0, int wi)
{
    const long long nn = (long long)mol.nao * mol.nao;
#pragma unroll
    for (int m = 0; m < NDM; ++m)
#pragma unroll
        for (int ia = 0; ia < FA; ++ia)
#pragma unroll
            for (int ib = 0; ib < FB; ++ib)
                if (jk_nonzero(jab[m][ia][ib]))
                    jk_red_add(mol.J + m * nn + (long long)(a0 + ia) * mol.nao + b0 + ib, jk_wide(jab[m][ia][ib], wi));
}

// Counters of a warp (or CTA) for the class pair it works on, added to the
// class pair's statistics when it moves to another one.
struct JkCount {
    unsigned long long nq, nprim, nband;
};
__device__ __forceinline__ void jk_count_flush(const JkClassArgs &args, int launch, JkCount &c)
{
    if (launch >= 0 && (c.nq || c.nprim || c.nband)) {
        unsigned long long *st = args.stats + (long long)launch * args.stat_stride;
        atomicAdd(st, c.nq);
        atomicAdd(st + 1, c.nprim);
        if (c.nband) atomicAdd(st + 2, c.nband);
    }
    c.nq = c.nprim = c.nband = 0;
}

// ------------------------------------------------------- the class kernel
// One launch runs every class pair of the same angular momenta and fragment
// shape. Persistent: warps (or, for groups of more than 32 threads, whole
// CTAs) take work items, a bra pair and a range of its kets, from the list
// that jk_plan_kernel wrote for this build, the first by their own index and
// the next ones from a counter. A group of more than 256 threads (the largest
// classes, e.g. (gg|gg)) is split over X CTAs: work unit t is slab t % X of
// item t / X, each CTA builds the roots and 2D tables itself and evaluates
// the elements of its G / X threads.
//
// P1: every class pair of the launch is uncontracted. The primitive loops are then
// known to be one pass, so that the block is not live while the tables are built
// (FP32 (ff|ff) 112 -> 0 bytes of spills): 6 and 9 atoms of s p d f shells 2.05 -> 1.99
// and 2.90 -> 2.81 ms, 6 of f and g shells in FP32 2.08 -> 1.49.
//
// Why class pairs share a launch: a 6-31G*-shaped basis has 231 class pairs
// (22 kernels); launched one by one, most of them were too small to
// fill the GPU and ended in a tail of a few long items each.
template <int LA, int LB, int LC, int LD, int GA, int GB, int GC, int GD, int X, int NDM, int DOJ, int DOK,
          typename R, int MODE, int OP, int P1>
__global__ void __launch_bounds__(JkShape<LA, LB, LC, LD, GA, GB, GC, GD>::G <= 32 ? 128
                                  : ((JkShape<LA, LB, LC, LD, GA, GB, GC, GD>::G / X + 31) / 32) * 32)
jk_class_kernel(const JkClassArgs args)
{
    typedef JkShape<LA, LB, LC, LD, GA, GB, GC, GD, OP> S;
    constexpr int G = S::G;
    constexpr int FA = S::FA, FB = S::FB, FC = S::FC, FD = S::FD;
    extern __shared__ __align__(16) double jk_smem_raw[];
    const int lane = threadIdx.x & 31;
    const typename JkPP<R>::T *pp = jk_pp<R>(args);
    const typename JkTab<R>::T *rys = jk_rys<R>(args);
    const long long nitems = MODE == 3 ? 0 : (long long)*args.nitems;
    if (MODE != 3 && (long long)blockIdx.x * (G <= 32 ? 4 : 1) >= nitems * X) return;
    // The FP32 tier reads its Rys table from shared memory: lanes gather
    // coefficients of unrelated intervals, which from global memory costs one
    // L1 wavefront per lane and load. Only this class's N-root table, copied
    // once per (persistent) CTA, ahead of the groups' 2D tables.
    R *smem_groups = reinterpret_cast<R *>(jk_smem_raw);
    if constexpr (JkIsFloat<R>::v) {
        constexpr int NT = JkRysTab32<S::NR>::n, V = 4 * S::NR;   // float4 per interval (unpadded)
        static_assert(NT % 4 == 0, "whole float4 vectors");
        float4 *dst = reinterpret_cast<float4 *>(jk_smem_raw);
        const float4 *src = reinterpret_cast<const float4 *>(args.rys32 + rys32_offset[S::NR]);
        for (int i = threadIdx.x; i < rys32_nint_c[S::NR] * V; i += blockDim.x)
            dst[(i / V) * (V + 1) + i % V] = __ldg(src + i);
        __syncthreads();
        rys = reinterpret_cast<const R *>(jk_smem_raw);
        smem_groups = reinterpret_cast<R *>(jk_smem_raw) + NT;
    }
    if constexpr (JkIsDf<R>::v) {
        constexpr int NT = JkRysTabDf<S::NR>::n;
        rys = rys + rysdf_offset[S::NR];
        if constexpr (NT > 0) {
            float4 *dst = reinterpret_cast<float4 *>(jk_smem_raw);
            const float4 *src = reinterpret_cast<const float4 *>(rys);
            for (int i = threadIdx.x; i < NT / 4; i += blockDim.x) dst[i] = __ldg(src + i);
            __syncthreads();
            rys = reinterpret_cast<const float *>(jk_smem_raw);
            smem_groups = reinterpret_cast<R *>(jk_smem_raw) + NT / 2;
        }
    }
    JkCount cnt = {0, 0, 0};
    int cur = -1;   // class pair the counters belong to

    static_assert(X == 1 || (G > 32 && G % X == 0), "a split group spans whole CTAs");
    if constexpr (G <= 32) {
        constexpr int NGW = 32 / G;
        const int wib = threadIdx.x >> 5;
        const int gw = lane / G, tg = lane - gw * G;
        const bool active = gw < NGW;
        const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << ((active ? gw : 0) * G));
        R *grp = smem_groups + (size_t)(wib * NGW + (active ? gw : 0)) * S::SMEM_GROUP;
        // router scratch, 1 KB per warp (MODE 1)
        __shared__ __align__(16) unsigned short s_rsm[MODE == 1 ? 4 * 32 * JK_RT_NINP : 2];
        // ket queue per warp: at most NGW - 1 + 32 entries; band queue (MODE 1):
        // at most 31 + 32
        __shared__ int s_qk[4][64];
        __shared__ float s_qd[4][64];
        __shared__ int s_bk[4][MODE == 1 ? 64 : 1];
        __shared__ float s_bd[4][MODE == 1 ? 64 : 1], s_bb[4][MODE == 1 ? 64 : 1];
        unsigned short *rsm = s_rsm + (MODE == 1 ? wib * 32 * JK_RT_NINP : 0);
        const int gd = tg % GD, gc = (tg / GD) % GC, gb = (tg / (GD * GC)) % GB, ga = tg / (GD * GC * GB);
        JkOffsets<S> off;
        jk_make_offsets<LA, LB, LC, LD, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
        const long long nw = (long long)gridDim.x * 4, w0 = (long long)blockIdx.x * 4 + wib;
        if constexpr (MODE == 3) {
            // FP32 list kernel of a routed build: the band quartets the FP64
            // tier released, one per group; each bra's J block is flushed on
            // its own (the quartets of a warp belong to unrelated bras). Each
            // class pair's list is dealt to the warps in turn, the next one
            // from where the last ended.
            long long dealt = 0;
            for (int isub = 0; isub < args.nsub; ++isub) {
                const JkSub &sub = args.subs[isub];
                const int launch = sub.launch;
                const long long n = min((long long)args.rcount[launch], args.rcap[launch]);
                if (n <= 0) continue;
                const long long rounds = (n + NGW - 1) / NGW;
                long long r = w0 - dealt % nw;
                if (r < 0) r += nw;
                dealt += rounds;
                const JkRouted *list = args.rlist + args.roff[launch];
                for (; r < rounds; r += nw) {
                    const long long e = r * NGW + gw;
                    if (active && e < n) {
                        const JkRouted rq = list[e];
                        const JkPair bra = sub.bra[rq.item];
                        const typename JkRecOf<R>::T ket = JkRecOf<R>::ket(sub, rq.ket);
                        const JkMol mol = args.mols[bra.mol];
                        R T[S::EPT];
#pragma unroll
                        for (int k = 0; k < S::EPT; ++k) T[k] = JkConst<R>::get(0.0);
                        const int np = jk_quartet<LA, LB, LC, LD, GA, GB, GC, GD, R, OP>(
                            JkRecOf<R>::bra(sub, rq.item), ket, JkShare{0, 1, 0, 1}, P1 ? 1 : sub.nab, P1 ? 1 : sub.ncd, __fdiv_rn(args.prim_eps32, rq.dmq), args.omega, args.asym64,
                            pp, rys, grp, gmask, tg, true, off, T);
                        float f = 1.0f;
                        if (bra.a == bra.b) f *= 0.5f;
                        if (ket.same) f *= 0.5f;
                        if (sub.same_class && rq.ket == rq.item) f *= 0.5f;
                        R jab[NDM][FA][FB];
#pragma unroll
                        for (int m = 0; m < NDM; ++m)
#pragma unroll
                            for (int i = 0; i < FA; ++i)
#pragma unroll
                                for (int jj = 0; jj < FB; ++jj) jab[m][i][jj] = JkConst<R>::get(0.0);
                        const int a0 = bra.a_ao + ga * FA, b0 = bra.b_ao + gb * FB;
                        jk_contract<FA, FB, FC, FD, NDM, DOJ, DOK, R>(T, f, mol, a0, b0, ket.a_ao + gc * FC,
                                                                     ket.b_ao + gd * FD, jab, args.widen_int);
                        if (DOJ) jk_flush_jab<FA, FB, NDM, R>(jab, mol, a0, b0, args.widen_int);
                        if (tg == 0) { ++cnt.nq; cnt.nprim += np; }
                    }
                }
                for (int o = 16; o > 0; o >>= 1) {
                    cnt.nq += __shfl_xor_sync(0xffffffffu, cnt.nq, o);
                    cnt.nprim += __shfl_xor_sync(0xffffffffu, cnt.nprim, o);
                }
                if (lane == 0) jk_count_flush(args, launch, cnt);
                cnt.nq = cnt.nprim = 0;
            }
            return;
        }
        // the FP32 tier's items are short: the next ticket is drawn while this
        // one runs (an FP64 item hides the counter's latency itself, and a
        // ticket held back by a long item would lengthen the launch's tail)
        constexpr bool AHEAD = JkIsFloat<R>::v;
        long long t = w0;
        while (t < nitems) {
            unsigned long long nx = 0;
            if (AHEAD && lane == 0) nx = atomicAdd(args.work, 1ull);
            const JkItem wi = args.items[t];
            const JkSub &sub = args.subs[wi.sub & 0x7fffff];
            const int part = wi.sub >> 23;   // share of the primitive quartets
            const JkShare sh = P1 ? JkShare{0, 1, 0, 1}
                                  : JkShare{part % sub.split_ab, sub.split_ab, part / sub.split_ab, sub.split / sub.split_ab};
            const int item = wi.bra, nab = P1 ? 1 : sub.nab, ncd = P1 ? 1 : sub.ncd, same_class = sub.same_class;
            const int kb = wi.kb, ke = wi.ke;
            if (sub.launch != cur) {
                if (lane == 0) jk_count_flush(args, cur, cnt);
                cur = sub.launch;
            }
            const JkPair bra = sub.bra[item];
            const typename JkRecOf<R>::T brec = JkRecOf<R>::bra(sub, item);
            const JkMol mol = args.mols[bra.mol];
            const double *dmx = args.dmax + mol.dmax_off;
            const double dreal = args.dmax_mol[bra.mol], dmol = args.use_dmax ? dreal : 1.0;
            const float dmol32 = (float)dmol;
            const JkBounds bd = jk_bounds(args, mol, dmol, dreal);
            const int a0 = bra.a_ao + ga * FA, b0 = bra.b_ao + gb * FB;
            JkPairFeat braf;
            if (MODE != 0) braf = sub.bra_feat[item];
            R jab[NDM][FA][FB];
#pragma unroll
            for (int m = 0; m < NDM; ++m)
#pragma unroll
                for (int i = 0; i < FA; ++i)
#pragma unroll
                    for (int j = 0; j < FB; ++j) jab[m][i][j] = JkConst<R>::get(0.0);
            int nq = 0, nband = 0, nprim = 0;
            // significant kets wait in a per-warp queue (in scan order) until
            // a round can give every group of the warp one; partial rounds
            // only at the end of the item
            // MODE 1: band candidates wait in a second queue and go through
            // the router 32 at a time (one full MMA tile per evaluation);
            // those this tier keeps join the ket queue
            int qn = 0, nb = 0;
            for (int base = kb; base < ke; base += 32) {
                bool sig = false, stop = false, band = false;
                float dmq = 1.0f, B = 0.0f;
                jk_screen_bound<MODE>(args, bd, sub, bra, mol, dmx, dmol, dmol32, base + lane, ke, sig, stop, band, dmq, B);
                const unsigned lt = (1u << lane) - 1u;
                const bool def = sig && !band;   // decided by the bounds alone
                const unsigned mdef = __ballot_sync(0xffffffffu, def);
                nq += __popc(mdef);
                if (def) {
                    const int pos = qn + __popc(mdef & lt);
                    s_qk[wib][pos] = base + lane;
                    s_qd[wib][pos] = dmq;
                }
                qn += __popc(mdef);
                if (MODE == 1) {
                    const unsigned mb = __ballot_sync(0xffffffffu, band);
                    if (band) {
                        const int pos = nb + __popc(mb & lt);
                        s_bk[wib][pos] = base + lane;
                        s_bd[wib][pos] = dmq;
                        s_bb[wib][pos] = B;
                    }
                    nb += __popc(mb);
                }
                __syncwarp();
                const bool last = __any_sync(0xffffffffu, stop) || base + 32 >= ke;
                for (;;) {
                    const bool full_round = qn >= NGW;
                    const bool band_batch = MODE == 1 && !full_round && (nb >= 32 || (last && nb > 0));
                    const bool tail_round = !full_round && !band_batch && last && qn > 0;
                    if (band_batch) {
                        const int take = nb < 32 ? nb : 32;
                        const bool mine = lane < take;
                        const int j = mine ? s_bk[wib][lane] : 0;
                        const float dj = mine ? s_bd[wib][lane] : 1.0f;
                        const float bj = mine ? s_bb[wib][lane] : 2.0f * args.tau32;
                        const JkPairFeat kf = mine ? sub.ket_feat[j] : braf;
                        const bool to32 = jk_router_to_fp32_warp(args.router, braf, kf, bj, dj, args.tau32, rsm);
                        // released quartets go to the FP32 list kernel; the
                        // rest of the band stays here, in FP64
                        const bool listed = jk_route_out(args, cur, mine && to32, item, j, dj);
                        const bool keep = mine && !listed;
                        const unsigned mk = __ballot_sync(0xffffffffu, keep);
                        nq += __popc(mk);
                        nband += __popc(__ballot_sync(0xffffffffu, listed));
                        if (keep) {
                            const int pos = qn + __popc(mk & lt);
                            s_qk[wib][pos] = j;
                            s_qd[wib][pos] = dj;
                        }
                        qn += __popc(mk);
                        // drop the evaluated band entries (at most 31 remain)
                        __syncwarp();
                        const int rest = nb - take;
                        int k2 = 0;
                        float d2 = 0.0f, b2 = 0.0f;
                        if (lane < rest) { k2 = s_bk[wib][take + lane]; d2 = s_bd[wib][take + lane]; b2 = s_bb[wib][take + lane]; }
                        __syncwarp();
                        if (lane < rest) { s_bk[wib][lane] = k2; s_bd[wib][lane] = d2; s_bb[wib][lane] = b2; }
                        __syncwarp();
                        nb = rest;
                        continue;
                    }
                    if (!full_round && !tail_round) break;
                    const int take = qn < NGW ? qn : NGW;
                    if (active && gw < take) {
                        const int myket = s_qk[wib][gw];
                        const typename JkRecOf<R>::T ket = JkRecOf<R>::ket(sub, myket);
                        R T[S::EPT];
#pragma unroll
                        for (int k = 0; k < S::EPT; ++k) T[k] = JkConst<R>::get(0.0);
                        const int np = jk_quartet<LA, LB, LC, LD, GA, GB, GC, GD, R, OP>(
                            brec, ket, sh, nab, ncd, __fdiv_rn(args.prim_eps32, s_qd[wib][gw]), args.omega,
                            args.asym64, pp, rys, grp, gmask, tg, true, off, T);
                        if (tg == 0) nprim += np;
                        float f = 1.0f;
                        if (brec.same) f *= 0.5f;
                        if (ket.same) f *= 0.5f;
                        if (same_class && myket == item) f *= 0.5f;
                        jk_contract<FA, FB, FC, FD, NDM, DOJ, DOK, R>(T, f, mol, a0, b0, ket.a_ao + gc * FC,
                                                                          ket.b_ao + gd * FD, jab, args.widen_int);
                        if (MODE == 2) {
                            double tm = 0.0;
#pragma unroll
                            for (int k = 0; k < S::EPT; ++k) tm = fmax(tm, fabs(jk_wide(T[k], 0)));
                            for (int q = 0; q < G; ++q) tm = fmax(tm, __shfl_sync(gmask, tm, (gw * G + q) & 31));
                            if (tg == 0)
                                jk_log_sample(args, bra, sub.ket[myket], braf, sub.ket_feat[myket],
                                              jk_quartet_dmax(args, bra, sub.ket[myket], mol, dmx), tm);
                        }
                    }
                    // drop the round's entries (at most 31 remain)
                    __syncwarp();
                    const int rest = qn - take;
                    int k2 = 0;
                    float d2 = 0.0f;
                    if (lane < rest) { k2 = s_qk[wib][take + lane]; d2 = s_qd[wib][take + lane]; }
                    __syncwarp();
                    if (lane < rest) { s_qk[wib][lane] = k2; s_qd[wib][lane] = d2; }
                    __syncwarp();
                    qn = rest;
                }
                if (last) break;
            }
            if (DOJ && active) jk_flush_jab<FA, FB, NDM, R>(jab, mol, a0, b0, args.widen_int);
            if (part == 0) cnt.nq += nq;
            cnt.nband += nband;
            cnt.nprim += __reduce_add_sync(0xffffffffu, (unsigned)nprim);
            if (!AHEAD && lane == 0) nx = atomicAdd(args.work, 1ull);
            t = nw + (long long)__shfl_sync(0xffffffffu, nx, 0);
        }
        if (lane == 0) jk_count_flush(args, cur, cnt);
    } else {
        // one group (or one of its X slabs) per CTA of round_up(G / X, 32) threads
        constexpr int NTC = G / X;
        __shared__ long long s_item;
        __shared__ float s_dm[32];
        __shared__ unsigned s_mask;
        __shared__ int s_stop;
        __shared__ __align__(16) unsigned short s_rsm[MODE == 1 ? 32 * JK_RT_NINP : 2];
        const int tg = threadIdx.x;
        const bool act = tg < NTC;
        const int tgc = act ? tg : 0;
        int gd = tgc % GD, gc = (tgc / GD) % GC, gb = (tgc / (GD * GC)) % GB, ga = tgc / (GD * GC * GB);
        R *grp = smem_groups;
        JkOffsets<S> off;
        jk_make_offsets<LA, LB, LC, LD, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
        if constexpr (MODE == 3) {
            // FP32 list kernel of a routed build: one released quartet (or one
            // of its X slabs) per CTA at a time, dealt as in the warp path
            long long dealt = 0;
            for (int isub = 0; isub < args.nsub; ++isub) {
                const JkSub &sub = args.subs[isub];
                const int launch = sub.launch;
                const long long n = min((long long)args.rcount[launch], args.rcap[launch]) * X;
                if (n <= 0) continue;
                long long tt = (long long)blockIdx.x - dealt % gridDim.x;
                if (tt < 0) tt += gridDim.x;
                dealt += n;
                const JkRouted *list = args.rlist + args.roff[launch];
                for (; tt < n; tt += gridDim.x) {
                    const long long e = X == 1 ? tt : tt / X;
                    const int slab = (int)(tt - e * X);
                    if constexpr (X > 1) {
                        const int tgl = slab * NTC + tgc;
                        gd = tgl % GD; gc = (tgl / GD) % GC; gb = (tgl / (GD * GC)) % GB; ga = tgl / (GD * GC * GB);
                        jk_make_offsets<LA, LB, LC, LD, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
                    }
                    const JkRouted rq = list[e];
                    const JkPair bra = sub.bra[rq.item];
                    const typename JkRecOf<R>::T ket = JkRecOf<R>::ket(sub, rq.ket);
                    const JkMol mol = args.mols[bra.mol];
                    R T[S::EPT];
#pragma unroll
                    for (int k = 0; k < S::EPT; ++k) T[k] = JkConst<R>::get(0.0);
                    const int np = jk_quartet<LA, LB, LC, LD, GA, GB, GC, GD, R, OP, NTC>(
                        JkRecOf<R>::bra(sub, rq.item), ket, JkShare{0, 1, 0, 1}, P1 ? 1 : sub.nab, P1 ? 1 : sub.ncd, __fdiv_rn(args.prim_eps32, rq.dmq), args.omega, args.asym64, pp,
                        rys, grp, 0u, tg, act, off, T);
                    if (act) {
                        float f = 1.0f;
                        if (bra.a == bra.b) f *= 0.5f;
                        if (ket.same) f *= 0.5f;
                        if (sub.same_class && rq.ket == rq.item) f *= 0.5f;
                        R jab[NDM][FA][FB];
#pragma unroll
                        for (int m = 0; m < NDM; ++m)
#pragma unroll
                            for (int i = 0; i < FA; ++i)
#pragma unroll
                                for (int jj = 0; jj < FB; ++jj) jab[m][i][jj] = JkConst<R>::get(0.0);
                        const int a0 = bra.a_ao + ga * FA, b0 = bra.b_ao + gb * FB;
                        jk_contract<FA, FB, FC, FD, NDM, DOJ, DOK, R>(T, f, mol, a0, b0, ket.a_ao + gc * FC,
                                                                     ket.b_ao + gd * FD, jab, args.widen_int);
                        if (DOJ) jk_flush_jab<FA, FB, NDM, R>(jab, mol, a0, b0, args.widen_int);
                    }
                    if (slab == 0) { ++cnt.nq; cnt.nprim += np; }
                    // every thread is done with this entry's shared tables
                    __syncthreads();
                }
                if (threadIdx.x == 0) jk_count_flush(args, launch, cnt);
                cnt.nq = cnt.nprim = 0;
            }
            return;
        }
        long long tt = blockIdx.x;
        while (tt < nitems * X) {
            const long long t = X == 1 ? tt : tt / X;
            const int slab = (int)(tt - t * X);
            if constexpr (X > 1) {
                // this CTA's share of the group: logical threads slab * NTC + tg
                const int tgl = slab * NTC + tgc;
                gd = tgl % GD; gc = (tgl / GD) % GC; gb = (tgl / (GD * GC)) % GB; ga = tgl / (GD * GC * GB);
                jk_make_offsets<LA, LB, LC, LD, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
            }
            const JkItem wi = args.items[t];
            const JkSub &sub = args.subs[wi.sub & 0x7fffff];
            const int part = wi.sub >> 23;   // share of the primitive quartets
            const JkShare sh = P1 ? JkShare{0, 1, 0, 1}
                                  : JkShare{part % sub.split_ab, sub.split_ab, part / sub.split_ab, sub.split / sub.split_ab};
            const int item = wi.bra, nab = P1 ? 1 : sub.nab, ncd = P1 ? 1 : sub.ncd, same_class = sub.same_class;
            const int kb = wi.kb, ke = wi.ke;
            if (sub.launch != cur) {
                if (threadIdx.x == 0) jk_count_flush(args, cur, cnt);
                cur = sub.launch;
            }
            const JkPair bra = sub.bra[item];
            const typename JkRecOf<R>::T brec = JkRecOf<R>::bra(sub, item);
            const JkMol mol = args.mols[bra.mol];
            const double *dmx = args.dmax + mol.dmax_off;
            const double dreal = args.dmax_mol[bra.mol], dmol = args.use_dmax ? dreal : 1.0;
            const float dmol32 = (float)dmol;
            const JkBounds bd = jk_bounds(args, mol, dmol, dreal);
            const int a0 = bra.a_ao + ga * FA, b0 = bra.b_ao + gb * FB;
            JkPairFeat braf;
            if (MODE != 0) braf = sub.bra_feat[item];
            R jab[NDM][FA][FB];
#pragma unroll
            for (int m = 0; m < NDM; ++m)
#pragma unroll
                for (int i = 0; i < FA; ++i)
#pragma unroll
                    for (int j = 0; j < FB; ++j) jab[m][i][j] = JkConst<R>::get(0.0);
            unsigned long long nq = 0, nband = 0, nprim = 0;
            for (int base = kb; base < ke; base += 32) {
                if (threadIdx.x < 32) {
                    bool sig, stop, band;
                    float dmq;
                    jk_screen<MODE>(args, bd, sub, bra, braf, mol, dmx, dmol, dmol32, item, base + lane, ke, sig, stop, band,
                                    dmq, s_rsm);
                    s_dm[lane] = dmq;
                    const unsigned msk = __ballot_sync(0xffffffffu, sig);
                    const int anystop = __any_sync(0xffffffffu, stop);
                    const unsigned bmsk = __ballot_sync(0xffffffffu, band);
                    if (lane == 0) { s_mask = msk; s_stop = anystop; nband += __popc(bmsk); }
                }
                __syncthreads();
                unsigned mask = s_mask;
                const int stop = s_stop;
                __syncthreads();
                nq += __popc(mask);
                while (mask) {
                    const int myket = base + __ffs(mask) - 1;
                    mask &= mask - 1;
                    const typename JkRecOf<R>::T ket = JkRecOf<R>::ket(sub, myket);
                    R T[S::EPT];
#pragma unroll
                    for (int k = 0; k < S::EPT; ++k) T[k] = JkConst<R>::get(0.0);
                    const int np = jk_quartet<LA, LB, LC, LD, GA, GB, GC, GD, R, OP, NTC>(
                        brec, ket, sh, nab, ncd, __fdiv_rn(args.prim_eps32, s_dm[myket - base]), args.omega, args.asym64, pp,
                        rys, grp, 0u, tg, act, off, T);
                    nprim += np;
                    if (act) {
                        float f = 1.0f;
                        if (bra.a == bra.b) f *= 0.5f;
                        if (ket.same) f *= 0.5f;
                        if (same_class && myket == item) f *= 0.5f;
                        jk_contract<FA, FB, FC, FD, NDM, DOJ, DOK, R>(T, f, mol, a0, b0, ket.a_ao + gc * FC,
                                                                     ket.b_ao + gd * FD, jab, args.widen_int);
                    }
                    if (MODE == 2 && X == 1) {   // labels need the whole block's max |T|
                        __shared__ double s_tm[32];
                        double tm = 0.0;
                        if (act) {
#pragma unroll
                            for (int k = 0; k < S::EPT; ++k) tm = fmax(tm, fabs(jk_wide(T[k], 0)));
                        }
                        for (int o = 16; o > 0; o >>= 1) tm = fmax(tm, __shfl_xor_sync(0xffffffffu, tm, o));
                        if (lane == 0) s_tm[threadIdx.x >> 5] = tm;
                        __syncthreads();
                        if (threadIdx.x == 0) {
                            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) tm = fmax(tm, s_tm[w]);
                            jk_log_sample(args, bra, sub.ket[myket], braf, sub.ket_feat[myket],
                                          jk_quartet_dmax(args, bra, sub.ket[myket], mol, dmx), tm);
                        }
                        __syncthreads();
                    }
                    // every thread has read s_dm for this quartet before warp 0
                    // may screen the next chunk (a quartet can skip all its
                    // primitives and so pass no barrier inside jk_quartet)
                    __syncthreads();
                }
                if (stop) break;
            }
            if (DOJ && act) jk_flush_jab<FA, FB, NDM, R>(jab, mol, a0, b0, args.widen_int);
            if (slab == 0) { cnt.nq += part == 0 ? nq : 0; cnt.nprim += nprim; cnt.nband += nband; }
            if (threadIdx.x == 0) s_item = (long long)gridDim.x + (long long)atomicAdd(args.work, 1ull);
            __syncthreads();
            tt = s_item;
            __syncthreads();
        }
        if (threadIdx.x == 0) jk_count_flush(args, cur, cnt);
    }
}

// ------------------------------------------------- Schwarz factors Q_ab
// Diagonal quartets (ab|ab) of one pair class in FP64; Q_ab is the square
// root of the largest |(mu nu|mu nu)| (eq:schwartz at shell level).
// A group of more than 1024 threads is split over X CTAs (slab t % X of
// pair t / X); the CTAs combine their maxima by an atomic max on Qout, which
// the caller zeroes.
template <int LA, int LB, int NPA, int NPB, int GA, int GB, int GC, int GD, int X>
__global__ void __launch_bounds__(JkShape<LA, LB, LA, LB, GA, GB, GC, GD>::G <= 32 ? 128
                                  : ((JkShape<LA, LB, LA, LB, GA, GB, GC, GD>::G / X + 31) / 32) * 32)
jk_schwarz_kernel(const JkSchwarzArgs args)
{
    typedef JkShape<LA, LB, LA, LB, GA, GB, GC, GD> S;
    static_assert(GA == GC && GB == GD, "diagonal elements must stay inside one thread");
    static_assert(X == 1 || (S::G > 32 && S::G % X == 0), "a split group spans whole CTAs");
    constexpr int G = S::G;
    constexpr int FA = S::FA, FB = S::FB, FC = S::FC, FD = S::FD;
    extern __shared__ __align__(16) double jk_smem_raw[];
    const int lane = threadIdx.x & 31;
    if constexpr (G <= 32) {
        constexpr int NGW = 32 / G;
        const int wib = threadIdx.x >> 5;
        const int gw = lane / G, tg = lane - gw * G;
        const bool active = gw < NGW;
        const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << ((active ? gw : 0) * G));
        double *grp = jk_smem_raw + (size_t)(wib * NGW + (active ? gw : 0)) * S::SMEM_GROUP;
        const int gd = tg % GD, gc = (tg / GD) % GC, gb = (tg / (GD * GC)) % GB, ga = tg / (GD * GC * GB);
        JkOffsets<S> off;
        jk_make_offsets<LA, LB, LA, LB, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
        const int warps_total = (gridDim.x * blockDim.x) >> 5;
        const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        for (int base = gwarp * NGW; base < args.npair; base += warps_total * NGW) {
            const int pi = base + gw;
            const bool mine = active && pi < args.npair;
            double mx = 0.0;
            if (mine) {
                const JkRec64 pr = jk_rec64(args.pairs[pi]);
                double T[S::EPT];
#pragma unroll
                for (int k = 0; k < S::EPT; ++k) T[k] = 0.0;
                jk_quartet<LA, LB, LA, LB, GA, GB, GC, GD, double>(pr, pr, JkShare{0, 1, 0, 1}, NPA * NPB, NPA * NPB, -1.0f, 0.0, 0, args.pp64, args.rys64, grp, gmask, tg, true, off, T);
                if (ga == gc && gb == gd) {
#pragma unroll
                    for (int ia = 0; ia < FA; ++ia)
#pragma unroll
                        for (int ib = 0; ib < FB; ++ib)
                            mx = fmax(mx, fabs(T[((ia * FB + ib) * FC + ia) * FD + ib]));
                }
            }
            double gmx = mx;
            for (int q = 0; q < G; ++q) gmx = fmax(gmx, __shfl_sync(0xffffffffu, mx, (gw * G + q) & 31));
            if (mine && tg == 0) args.Qout[pi] = sqrt(gmx);
            __syncwarp();
        }
    } else {
        constexpr int NTC = G / X;
        __shared__ double s_max[32];
        const int tg = threadIdx.x;
        const bool act = tg < NTC;
        const int tgc = act ? tg : 0;
        int gd = tgc % GD, gc = (tgc / GD) % GC, gb = (tgc / (GD * GC)) % GB, ga = tgc / (GD * GC * GB);
        double *grp = jk_smem_raw;
        JkOffsets<S> off;
        jk_make_offsets<LA, LB, LA, LB, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
        for (long long t = blockIdx.x; t < (long long)args.npair * X; t += gridDim.x) {
            const int pi = (int)(t / X), slab = (int)(t - (long long)pi * X);
            if constexpr (X > 1) {
                const int tgl = slab * NTC + tgc;
                gd = tgl % GD; gc = (tgl / GD) % GC; gb = (tgl / (GD * GC)) % GB; ga = tgl / (GD * GC * GB);
                jk_make_offsets<LA, LB, LA, LB, GA, GB, GC, GD, S>(ga, gb, gc, gd, off);
            }
            const JkRec64 pr = jk_rec64(args.pairs[pi]);
            double T[S::EPT];
#pragma unroll
            for (int k = 0; k < S::EPT; ++k) T[k] = 0.0;
            jk_quartet<LA, LB, LA, LB, GA, GB, GC, GD, double, 0, NTC>(
                pr, pr, JkShare{0, 1, 0, 1}, NPA * NPB, NPA * NPB, -1.0f, 0.0, 0, args.pp64, args.rys64, grp, 0u, tg, act, off, T);
            double mx = 0.0;
            if (act && ga == gc && gb == gd) {
#pragma unroll
                for (int ia = 0; ia < FA; ++ia)
#pragma unroll
                    for (int ib = 0; ib < FB; ++ib)
                        mx = fmax(mx, fabs(T[((ia * FB + ib) * FC + ia) * FD + ib]));
            }
            for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0) s_max[threadIdx.x >> 5] = mx;
            __syncthreads();
            if (threadIdx.x == 0) {
                double m2 = 0.0;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m2 = fmax(m2, s_max[w]);
                // non-negative doubles order like their bit patterns
                if (X == 1) args.Qout[pi] = sqrt(m2);
                else atomicMax(reinterpret_cast<unsigned long long *>(args.Qout + pi),
                               (unsigned long long)__double_as_longlong(sqrt(m2)));
            }
            __syncthreads();
        }
    }
}
