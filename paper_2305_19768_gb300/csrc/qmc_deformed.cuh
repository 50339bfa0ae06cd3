// The deformed evaluator for sums ending at eps^0 or eps^1: contour-deformed sectors
// with d <= 3, at most two singular variables and exponents u0, u1, f0, f1,
// b_j that are integers of magnitude <= 4; in FP64 also F of total degree <= 2
// (every one-loop sector of the built-in integrals). Included by
// qmc_kernels.cu (parts 6, FP64, and 7, mixed precision) after qmc_real.cuh, whose front it shares.
//
// What bounds it: the FP64 pipe (76 % busy in the general kernel, at 175
// useful FP64 instructions per evaluation of the massive box and as many
// again switched off by predicates, which hold the pipe all the same). So:
//  * dimension, number of singular variables and corner are compile-time, and
//    what a sector lacks (couplings, U, regular factors) is skipped by
//    branches, uniform over the tile, not by predicates;
//  * with F quadratic, F(t) = c + b.t + t.A.t / 2, one real gradient
//    g = b + A t gives everything of the deformation, and the value on the
//    contour z = t - i y, y_j = lambda_j t_j (1 - t_j) g_j, is exactly
//      F(z) = [F(t) - y.A.y / 2] - i y.g,  F(t) = c + t.(b + g) / 2:
//    no complex monomials and no second-derivative tables;
//  * at a corner t_V = 0 the rows of the Jacobian of the zeroed variables are
//    diagonal with entries rho_j, which cancel the 1 / rho_j of the integrand:
//    determinant and products are formed over the other variables only;
//  * the Jacobian is 1 - i diag(p) M with p = lambda t (1 - t) and M symmetric,
//    M_jj = A_jj + (1 - 2t) / (t (1 - t)) g_j: its minors take one FMA each;
//  * x^-e enters as conj(x)^e / |x|^2e: the complex products collect in FP64,
//    the norms as mantissas, whose logarithm is also the corner's Re L; its
//    Im L is the sum of the factors' principal arguments, in 128-bit fixed point
//    (an integer arctangent), so that no branch has to be restored;
//  * transform, weight, the real factors of the deformation, 1/t, ln t,
//    reciprocals, logarithms and arguments run on the integer pipe (an FP64
//    negation or doubling by itself takes the FP64 pipe too: both go through
//    the bits), and the corners are folded variable by variable as in
//    qmc_real.cuh (complex corner series, real factors).
// Measured (evaluations/s, general kernel -> this one; FP64 instructions per
// evaluation): massive box, 64 points at n = 10007, 1.74e9 (175, and as many
// switched off) -> 5.9e9 (90) with the Jacobian entry by entry -> 7.4e9 (68,
// pipe 87 % busy); massless box, 16 physical points at n = 4001, 5.9e8 (555)
// -> 1.06e9 (453) with complex logarithms of the factors' product -> 1.86e9
// (204, 78 %); the massive box in mixed precision, 256 points at n = 1009,
// 2.85e9 -> 6.6e9. Arguments and their sums to FP64's relative precision at every
// size (qmc_iarg.h; 2^-57 fixed point before): the massless box at 60 points
// 1.94e9 -> 1.87e9.
// MIXED: derivatives of F and U(z), F(z) from FP32 monomial products in the
// order of the general mixed kernel, everything after them in FP64.

struct alignas(16) FdShared {
    uint64_t logtab[3 * QMC_LOG_TABLE_ROWS + 1];
    int64_t atan63[QMC_ATAN_TABLE_ROWS];   // atan(j / 64) 2^63
    uint32_t exps[QMC_MAXMONO];      // FP64: variables in slot order (singular first)
    uint4 mdesc[QMC_MAXMONO];        // MIXED: factors as in FxShared, original variable order
    double cval[QMC_MAXMONO];
    float cvalf[QMC_MAXMONO];
    // F(t) = qc[0] + sum_j t_j (qc[1+j] + qc[4+j] t_j) + qc[7] t_0 t_1 + qc[8] t_0 t_2 + qc[9] t_1 t_2 (slots)
    double qc[10];
    double qa[3];                    // 2 qc[4..6]
    int32_t qmask;                   // bits 0..2: qc[7..9] present; 3..5: qc[4..6]
    int32_t d, ns, nU, nF, dbase, prow;
    int32_t dFoff[3], dFn[3], Hoff[QMC_NHESS], Hn[QMC_NHESS];
    // MIXED: derivatives of F that are constants (F of degree <= 2 has only such
    // second ones): dF by variable, d2F by slot pair (diagonal, then 01, 02, 12)
    float gconst[3];
    double hconst[6];
    int32_t gvar, hvar;              // bits: those that are not
    int32_t perm[QMC_DMAX], slotof[QMC_DMAX], avar[QMC_DMAX], bvar[QMC_DMAX];
    double bd[QMC_DMAX], lam[QMC_DMAX];
    uint64_t lamm[QMC_DMAX];         // lambda as mantissa (0: none, or outside 2^-800 .. 2^1024), exponent and sign
    int32_t lame[QMC_DMAX], lamneg[QMC_DMAX];
    int32_t regular, u0, f0, u1, f1;
    double delta[QMC_DMAX];
    uint64_t dfix[QMC_DMAX], qz[QMC_DMAX];
    uint32_t rz[QMC_DMAX], zmod[QMC_DMAX];
    uint64_t minv;
    double w, mone, nzero;
    QmcJobDev job;
    unsigned long long tile;
    int cached_sector, cached_point, job_index;
    double red[16][8];
};
__device__ __forceinline__ FdShared &fd_shared() { return *reinterpret_cast<FdShared *>(qmc_fx_raw); }

// A squared norm as mantissa and exponent. Zero, subnormal, infinite and NaN
// ones get the exponent kFdBad, beyond anything that products of the others
// reach (|e| < 2^15), so that one look at a product's exponent finds them: a
// negative power or a logarithm of such a factor has no value, and the corner is
// NaN (mantissas alone would give a finite number, since conj(0) / 2^-1022 = 0).
constexpr int kFdBad = 1 << 20;
__device__ __forceinline__ FxM fd_of(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint32_t ex = (uint32_t)(b >> 52) & 0x7FFu;
    return FxM{(b << 11) | (1ULL << 63), ex - 1u < 0x7FEu ? (int)ex - 1023 : kFdBad};
}
__device__ __forceinline__ FxM fd_rcp(FxM a) {
    const qmc_xf r = qmc_xf_rcp3(qmc_xf{a.m, a.e, 0});
    return FxM{r.m, r.e};
}
__device__ __noinline__ double fd_half_log(FxM x) {
    return fx_half(qmc_ilog_xf(qmc_xf{x.m, x.e, 0}, fd_shared().logtab));
}

// sum + k arg(x + i y), |k| <= 4 (qmc_iarg.h). Out of line. In 64-bit fixed point
// (2^-57) a nearly real integrand's imaginary part, a sum of small arguments, had
// fewer bits than FP64 has.
__device__ __noinline__ qmc_u128 fd_addarg(qmc_u128 sum, double y, double x, int k, bool m0) {
    return qmc_iarg_add(sum, qmc_iarg(y, x, m0, fd_shared().atan63), k);
}
// -x or x on the sign bit (a negation by itself takes the FP64 pipe)
__device__ __forceinline__ double fd_signed(double x, bool neg) {
    return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}

// FP32 <-> FP64 conversions on the integer pipe (RN; subnormals, infinities and
// NaN too, behind one test)
__device__ __forceinline__ float fd_to_float(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7FFu) - 896;                    // FP32's biased exponent
    uint32_t m = (hi << 3 | lo >> 29) & 0x7FFFFFu, rest = lo << 3, out = (uint32_t)e << 23;
    if (__builtin_expect((uint32_t)e - 1u >= 254u, 0)) {
        out = 0;
        if (e >= 255) {                                                // infinite, too large, NaN
            m = 0x7F800000u | (e == 1151 && (m | rest) ? 0x400000u : 0u);
            rest = 0;
        } else if (e >= -24) {                                         // below FP32's normal range
            const uint64_t f = ((uint64_t)(m | 0x800000u) << 32 | rest) >> (1 - e);
            rest = (uint32_t)f | (rest ? 1u : 0u);
            m = (uint32_t)(f >> 32);
        } else {                                                       // below half the smallest
            m = rest = 0;
        }
    }
    out += m + ((rest > 0x80000000u || (rest == 0x80000000u && (m & 1u))) ? 1u : 0u);
    return __uint_as_float((hi & 0x80000000u) | out);
}
__device__ __forceinline__ double fd_to_double(float x) {
    const uint32_t b = __float_as_uint(x);
    uint32_t e = ((b >> 23) & 255u) + 896u, m = b & 0x7FFFFFu;
    if (__builtin_expect(e - 897u >= 254u, 0)) {
        if (e != 896u) {
            e = 2047u;                                                 // infinite, NaN
        } else {
            const int p = __clz((int)m) - 8;                           // 0 or subnormal
            e = m ? 897u - (uint32_t)p : 0u;
            m = (m << p) & 0x7FFFFFu;
        }
    }
    return __hiloint2double((int)((b & 0x80000000u) | (e << 20) | (m >> 3)), (int)(m << 29));
}

// complex arithmetic in FMAs (an FP64 multiply holds the pipe longer than an FMA)
struct FdOps {
    double mone, nzero, one;
    __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nzero); }
    __device__ __forceinline__ double add(double a, double b) const { return fma(b, one, a); }
    // 2 a on the exponent; behind one test, zero and subnormals on the mantissa,
    // and infinities and NaN stay
    __device__ __forceinline__ double dbl(double a) const {
        const uint64_t b = (uint64_t)__double_as_longlong(a), sign = b & 0x8000000000000000ULL;
        const uint32_t e = (uint32_t)(b >> 52) & 0x7FFu;
        if (__builtin_expect(e - 1u >= 0x7FDu, 0)) {
            const uint64_t v = e == 0 ? sign | (b << 1) : (e == 0x7FEu ? sign | 0x7FF0000000000000ULL : b);
            return __longlong_as_double((long long)v);
        }
        return __longlong_as_double((long long)(b + (1ULL << 52)));
    }
    __device__ __forceinline__ double sub(double a, double b) const { return fma(b, mone, a); }
    __device__ __forceinline__ dc mul(dc a, dc b) const {
        return dc{fma(a.re, b.re, mul(-a.im, b.im)), fma(a.re, b.im, mul(a.im, b.re))};
    }
    __device__ __forceinline__ dc sub(dc a, dc b) const { return dc{sub(a.re, b.re), sub(a.im, b.im)}; }
    // x^a, 1 <= a <= 4
    __device__ __forceinline__ dc pow(dc x, int a) const {
        if (a == 1) return x;
        const dc x2 = dc{fma(x.re, x.re, mul(-x.im, x.im)), mul(dbl(x.re), x.im)};
        if (a == 2) return x2;
        if (a == 3) return mul(x2, x);
        return dc{fma(x2.re, x2.re, mul(-x2.im, x2.im)), mul(dbl(x2.re), x2.im)};
    }
};

// The factors of a corner, out of line: inlined, their copies in every corner
// of every path overflowed the instruction cache when sectors of several shapes
// run side by side (the amplitude: 5 of 14 stall cycles per instruction).
// B x^e or, for e < 0, B conj(x)^-e
__device__ __noinline__ dc fd_mulpow(dc B, dc x, int e) {
    const FdShared &S = fd_shared();
    const FdOps o{S.mone, S.nzero, fd_signed(S.mone, true)};
    return o.mul(B, o.pow(e < 0 ? conj_(x) : x, e < 0 ? -e : e));
}
// a n^e, 1 <= e <= 4
__device__ __noinline__ FxM fd_mulnorm(FxM a, FxM n, int e) { return fx_norm(fx_mul(a, fx_pow(n, n, e))); }
// re^2 + im^2
__device__ __noinline__ FxM fd_norm2(double re, double im) {
    return fd_of(fma(re, re, fma(im, im, fd_shared().nzero)));
}

// MIXED: the thread's FP32 power tables (real rows, then complex rows, prow
// per variable) and the sums over them, products and sums in the order of the
// general mixed kernel; out of line, one copy for every polynomial and corner
template <int BLOCK> __device__ __forceinline__ unsigned char *fd_pt() {
    return qmc_fx_raw + sizeof(FdShared) + 16 * 3 * BLOCK;
}
template <int BLOCK> __device__ __forceinline__ void fd_put(int j, int prow, float x) {
    float *p = reinterpret_cast<float *>(fd_pt<BLOCK>()) + threadIdx.x + prow * j * BLOCK;
    p[0] = x;
    if (prow >= 2) {
        const float x2 = x * x;
        p[BLOCK] = x2;
        if (prow >= 3) p[2 * BLOCK] = x2 * x;
        if (prow >= 4) p[3 * BLOCK] = x2 * x2;
    }
}
template <int BLOCK> __device__ __forceinline__ void fd_putc(int j, int prow, fc x) {
    fc *p = reinterpret_cast<fc *>(fd_pt<BLOCK>() + 4 * 3 * prow * BLOCK) + threadIdx.x + prow * j * BLOCK;
    p[0] = x;
    if (prow >= 2) {
        const fc x2 = x * x;
        p[BLOCK] = x2;
        if (prow >= 3) p[2 * BLOCK] = x2 * x;
        if (prow >= 4) p[3 * BLOCK] = x2 * x2;
    }
}
template <class T>
__device__ __forceinline__ T fd_sum(const FdShared &S, const unsigned char *pt, int m0, int count) {
    constexpr int sc = (int)sizeof(T) / 4;
    auto ld = [&](uint32_t off) { return *reinterpret_cast<const T *>(pt + sc * off); };
    T s = zero<T>();
    for (int m = m0; m < m0 + count; ++m) {
        const uint4 D = S.mdesc[m];
        const float c = S.cvalf[m];
        if (D.w == 0) {
            s = m == m0 ? from_real<T>(c) : s + from_real<T>(c);
            continue;
        }
        T v = ld(D.x & 0xFFFFu);
        if (D.w > 1) {
            v = v * ld(D.x >> 16);
            if (D.w > 2) v = v * ld(D.y & 0xFFFFu);
        }
        s = m == m0 ? mulsc(v, c) : s + mulsc(v, c);
    }
    return s;
}
template <int BLOCK> __device__ __noinline__ float fd_poly(int m0, int count) {
    return fd_sum<float>(fd_shared(), fd_pt<BLOCK>() + 4 * threadIdx.x, m0, count);
}
template <int BLOCK> __device__ __noinline__ fc fd_polyc(int m0, int count) {
    const FdShared &S = fd_shared();
    return fd_sum<fc>(S, fd_pt<BLOCK>() + 4 * 3 * S.prow * BLOCK + 8 * threadIdx.x, m0, count);
}

struct FdPoint {
    // per slot: t, lambda t (1 - t), (1 - 2t) / (t (1 - t)), and lambda (1 - t) of the singular ones
    double t[3], p[3], k[3], s[3];
    float tf[3];                     // FP32 t, original variable order (MIXED)
};
struct FdCorner {
    dc B, L;                         // the corner value is B q
    FxM q;
};

// The corner with the slots of V at t = 0 (D variables, NS of them singular)
template <int D, int BLOCK, int NS, int HI, int V, bool MIXED>
__device__ __forceinline__ FdCorner fd_corner(const FdPoint &P, const FdOps &o, int prow, int &signfail) {
    const FdShared &S = fd_shared();
    constexpr bool lam = HI > 0 || V != 0;              // needs its eps exponent
    constexpr int NA = D - __builtin_popcount(V);       // variables left
    double g[D];                                        // dF/dt_j
    double e[D];                                        // F(t) = c + sum t_j e_j
    double Ad[D], Ao[3];                                // d2F: diagonal (MIXED), off-diagonal (01, 02, 12)
    dc F, U{1.0, 0.0};
    const bool needU = S.u0 != 0 || (lam && S.u1 != 0);
    const int qm = S.qmask;
    if constexpr (!MIXED) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            e[j] = S.qc[1 + j];
            if (!(V >> j & 1)) {
                if (qm >> (3 + j) & 1) e[j] = fma(S.qc[4 + j], P.t[j], e[j]);
#pragma unroll
                for (int k = j + 1; k < D; ++k)
                    if (!(V >> k & 1) && (qm >> (j + k - 1) & 1)) e[j] = fma(S.qc[6 + j + k], P.t[k], e[j]);
            }
            g[j] = e[j];
            if (!(V >> j & 1) && (qm >> (3 + j) & 1)) g[j] = fma(S.qc[4 + j], P.t[j], g[j]);
#pragma unroll
            for (int k = 0; k < D; ++k)
                if (k != j && (k < j || (V >> j & 1)) && !(V >> k & 1) && (qm >> (j + k - 1) & 1))
                    g[j] = fma(S.qc[6 + j + k], P.t[k], g[j]);
        }
    } else {
        // FP32 derivatives, original variable order
#pragma unroll
        for (int j = 0; j < D; ++j) fd_put<BLOCK>(j, prow, (V >> S.slotof[j] & 1) ? 0.0f : P.tf[j]);
        float gf[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int j = 0; j < D; ++j) {
            gf[j] = S.gconst[j];
            if (S.gvar >> j & 1) gf[j] = fd_poly<BLOCK>(S.dbase + S.dFoff[j], S.dFn[j]);
        }
        // to slot order
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const int pi = S.perm[i];
            g[i] = fd_to_double(pi == 0 ? gf[0] : (pi == 1 ? gf[1] : gf[2]));
#pragma unroll
            for (int k = i; k < D; ++k) {
                if ((V >> i & 1) || (V >> k & 1)) continue;
                const int at = i == k ? i : 2 + i + k;
                double h = S.hconst[at];
                if (S.hvar >> at & 1) {
                    const int a = min(pi, S.perm[k]), b = max(pi, S.perm[k]);
                    const int q = a * QMC_DMAX - a * (a - 1) / 2 + (b - a);
                    h = fd_to_double(fd_poly<BLOCK>(S.dbase + S.Hoff[q], S.Hn[q]));
                }
                if (i == k) Ad[i] = h;
                else Ao[i + k - 1] = h;
            }
        }
    }
    // y_j = lambda t (1 - t) g_j (z = t - i y); the Jacobian J = 1 - i V with
    // V = diag(p) M, M_jj = A_jj + k_j g_j, M_jk = A_jk: symmetric, so its
    // minors take one FMA each with the squares of the couplings
    double y[D], M[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        y[j] = M[j] = 0.0;
        if (V >> j & 1) continue;
        y[j] = o.mul(P.p[j], g[j]);
        M[j] = fma(P.k[j], g[j], MIXED ? Ad[j] : S.qa[j]);
    }
    dc J{1.0, 0.0};
    {
        int a[3] = {0, 0, 0}, na = 0;
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (!(V >> j & 1)) a[na++] = j;
        // M_x M_z - A_xz^2
        auto minor2 = [&](int x, int z) {
            if (!(qm >> (x + z - 1) & 1)) return o.mul(M[x], M[z]);
            const double A = MIXED ? Ao[x + z - 1] : S.qc[6 + x + z];
            return fma(M[x], M[z], o.mul(-A, A));
        };
        if constexpr (NA == 1) {
            J = dc{1.0, o.mul(-P.p[a[0]], M[a[0]])};
        } else if constexpr (NA == 2) {
            const int x = a[0], z = a[1];
            J.re = fma(o.mul(-P.p[x], P.p[z]), minor2(x, z), o.one);
            J.im = fma(-P.p[x], M[x], o.mul(-P.p[z], M[z]));
        } else if constexpr (NA == 3) {
            const double c01 = minor2(0, 1), c02 = minor2(0, 2), c12 = minor2(1, 2);
            double det = o.mul(M[0], c12);
            if (qm & 3) {
                // - A01^2 M2 - A02^2 M1 + 2 A01 A02 A12
                const double a01 = MIXED ? Ao[0] : S.qc[7], a02 = MIXED ? Ao[1] : S.qc[8], a12 = MIXED ? Ao[2] : S.qc[9];
                if (qm & 1) det = fma(o.mul(-a01, M[2]), a01, det);
                if (qm & 2) det = fma(o.mul(-a02, M[1]), a02, det);
                if ((qm & 7) == 7) det = fma(o.mul(o.dbl(a01), a02), a12, det);
            }
            const double p01 = o.mul(P.p[0], P.p[1]);
            J.re = fma(-p01, c01, fma(o.mul(-P.p[0], P.p[2]), c02, fma(o.mul(-P.p[1], P.p[2]), c12, o.one)));
            J.im = fma(-P.p[0], M[0], fma(-P.p[1], M[1], fma(-P.p[2], M[2], o.mul(o.mul(p01, P.p[2]), det))));
        }
    }
    // U and F on the contour
    if constexpr (!MIXED) {
        double re = S.qc[0], im = 0.0;
        bool first = true;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            if (V >> j & 1) continue;
            // t_j e_j - y_j (A_jj y_j / 2 + sum_{k > j} A_jk y_k);  -y_j g_j
            re = fma(P.t[j], e[j], re);
            double q = 0.0;
            bool any = false;
            if (qm >> (3 + j) & 1) {
                q = o.mul(S.qc[4 + j], y[j]);
                any = true;
            }
#pragma unroll
            for (int k = j + 1; k < D; ++k)
                if (!(V >> k & 1) && (qm >> (j + k - 1) & 1)) {
                    q = fma(S.qc[6 + j + k], y[k], any ? q : o.nzero);
                    any = true;
                }
            if (any) re = fma(-y[j], q, re);
            im = fma(-y[j], g[j], first ? o.nzero : im);
            first = false;
        }
        F = dc{re, im};
        if (needU) {
            // monomials by factors, uniform branches; t_V = 0 drops monomials
            U = dc{0.0, 0.0};
            uint32_t vm = 0;
#pragma unroll
            for (int j = 0; j < D; ++j)
                if (V >> j & 1) vm |= 15u << (4 * j);
            for (int m = 0; m < S.nU; ++m) {
                const uint32_t ex = S.exps[m];
                if (ex & vm) continue;
                const double c = S.cval[m];
                if (ex == 0) {
                    U.re = o.add(U.re, c);
                    continue;
                }
                dc v{1.0, 0.0};
                bool one = true;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    if (V >> j & 1) continue;
                    const dc z{P.t[j], -y[j]};
                    for (int q = (int)(ex >> (4 * j) & 15u); q > 0; --q) {
                        v = one ? z : o.mul(v, z);
                        one = false;
                    }
                }
                U = dc{fma(c, v.re, U.re), fma(c, v.im, U.im)};
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const int sl = S.slotof[j];
            double zi = 0.0;
            bool zeroed = false;
#pragma unroll
            for (int i = 0; i < D; ++i)
                if (sl == i) {
                    if (V >> i & 1) zeroed = true;
                    else zi = -y[i];
                }
            fd_putc<BLOCK>(j, prow, zeroed ? fc{0.0f, 0.0f} : fc{P.tf[j], fd_to_float(zi)});
        }
        if (needU) {
            const fc u = fd_polyc<BLOCK>(0, S.nU);
            U = dc{fd_to_double(u.re), fd_to_double(u.im)};
        }
        const fc f = fd_polyc<BLOCK>(S.nU, S.nF);
        F = dc{fd_to_double(f.re), fd_to_double(f.im)};
    }
    // F.im > 0 on the bits (not for NaN)
    if ((uint64_t)__double_as_longlong(F.im) - 1ULL < 0x7FF0000000000000ULL) ++signfail;
    // The corner value J / prod rho (kept singular) prod z^a (regular) U^u0
    // F^f0, a factor x^-e as conj(x)^e / |x|^2e: B collects the complex
    // products and q the real ones, in mantissas. Its exponent
    // L = sum of e ln x over rho^b, z^b, U^u1, F^f1: ln |x|^2 of the product
    // of norms in mantissas, and the sum of the principal arguments.
    FdCorner out;
    dc B = J;
    FxM den{1ULL << 63, 0}, np{1ULL << 63, 0}, nn{1ULL << 63, 0};
    qmc_u128 arg = 0;
    auto factor = [&](dc x, FxM n, int e0, int e1, bool m0) {
        if (e0) {
            B = fd_mulpow(B, x, e0);
            if (e0 < 0) den = fd_mulnorm(den, n, -e0);
        }
        if (lam && e1) {
            if (e1 > 0) np = fd_mulnorm(np, n, e1);
            else nn = fd_mulnorm(nn, n, -e1);
            arg = fd_addarg(arg, x.im, x.re, e1, m0);
        }
    };
#pragma unroll
    for (int j = 0; j < D; ++j) {
        if (j < NS) {
            // rho = 1 - i gl
            if ((V >> j & 1) && !lam) continue;
            const double gl = o.mul((V >> j & 1) ? S.lam[j] : P.s[j], g[j]);
            const FxM n = fd_of(fma(gl, gl, o.one));
            if (!(V >> j & 1)) {
                B = dc{fma(-gl, B.im, B.re), fma(gl, B.re, B.im)};
                den = fd_mulnorm(den, n, 1);
            }
            factor(dc{1.0, -gl}, n, 0, S.bvar[j], false);
        } else if (S.regular >> j & 1) {
            const dc z{P.t[j], -y[j]};
            factor(z, fd_norm2(z.re, z.im), S.avar[j], S.bvar[j], false);
        }
    }
    if (needU) factor(U, fd_norm2(U.re, U.im), S.u0, S.u1, false);
    factor(F, fd_norm2(F.re, F.im), S.f0, S.f1, true);
    // (den also beyond FP64's range: its reciprocal would vanish beside a finite B)
    if (den.e > 1020 || max(np.e, nn.e) > kFdBad / 2) B.re = B.im = __longlong_as_double(0x7FF8000000000000LL);
    out.B = B;
    out.q = fd_rcp(den);
    out.L = dc{0.0, 0.0};
    if constexpr (lam) out.L = dc{fd_half_log(fx_norm(fx_mul(np, fd_rcp(nn)))), qmc_iarg_sum(arg)};
    return out;
}

// Depth-first fold of the corners (see qmc_real.cuh), complex series
template <int D, int BLOCK, int NS, int HI, bool MIXED> struct FdFold {
    const FdPoint &P;
    const FdOps &o;
    const double (&h)[SlotArr<NS>::N][NS + HI + 1];
    int prow;
    int &signfail;
    FxM &q0;                          // NS = 0: the corner's real factor, left to the weight

    template <int Q, int V>
    __device__ __forceinline__ void run(dc (&out)[Q + __builtin_popcount(V) + HI + 1]) const {
        constexpr int pv = __builtin_popcount(V);
        if constexpr (Q == 0) {
            const FdCorner c = fd_corner<D, BLOCK, NS, HI, V, MIXED>(P, o, prow, signfail);
            if constexpr (NS == 0) {
                q0 = c.q;
                out[0] = c.B;
            } else {
                const double q = qmc_xf_to_double(qmc_xf{c.q.m, c.q.e, 0});
                out[0] = dc{o.mul(c.B.re, q), o.mul(c.B.im, q)};
            }
            if constexpr (pv + HI >= 1) out[1] = o.mul(out[0], c.L);
            if constexpr (pv + HI >= 2) out[2] = o.mul(out[1], dc{fx_half(c.L.re), fx_half(c.L.im)});
            if constexpr (pv + HI >= 3) out[3] = o.mul(out[2], dc{c.L.re * (1.0 / 3), c.L.im * (1.0 / 3)});
        } else {
            constexpr int n = Q + pv + HI;
            dc a[n], b[n + 1];
            run<Q - 1, V>(a);
            run<Q - 1, V | (1 << (Q - 1))>(b);
            out[0] = b[0];
#pragma unroll
            for (int k = 0; k < n; ++k) {
                a[k] = o.sub(a[k], b[k]);
                dc s = b[k + 1];
#pragma unroll
                for (int i = 0; i <= k; ++i) {
                    s.re = fma(h[Q - 1][k - i], a[i].re, s.re);
                    s.im = fma(h[Q - 1][k - i], a[i].im, s.im);
                }
                out[k + 1] = s;
            }
        }
    }
};

template <int D, int BLOCK, int NS, int HI, bool MIXED, int LMAX>
__device__ __forceinline__ void fd_points(const QmcLaunch &Lc, uint64_t k0, uint64_t kend, int lo, int nord,
                                          dc (&acc)[LMAX], int &signfail) {
    constexpr int NSA = SlotArr<NS>::N;
    const FdShared &S = fd_shared();
    const uint64_t n = S.job.n;
    const uint32_t n32 = (uint32_t)n;
    uint4 *const walk = reinterpret_cast<uint4 *>(qmc_fx_raw + sizeof(FdShared)) + threadIdx.x;
    {
        const uint64_t minv = S.minv;
#pragma unroll 1
        for (int i = 0; i < D; ++i) {
            uint64_t r0, Q, R;
            fx_divmod(k0 * (uint64_t)S.zmod[i], n, minv, r0);
            fx_fixdiv(r0, n, minv, Q, R);
            walk[i * BLOCK] = make_uint4((uint32_t)Q, (uint32_t)(Q >> 32), (uint32_t)r0, (uint32_t)R);
        }
    }
    const FdOps o{S.mone, S.nzero, fd_signed(S.mone, true)};
    constexpr int NO = NS + HI + 1;
    dc accN[NO];
#pragma unroll
    for (int i = 0; i < NO; ++i) accN[i] = dc{0.0, 0.0};
#pragma unroll 1
    for (uint64_t k = k0; k < kend; ++k) {
        FxM w{1ULL << 63, 0};
        FdPoint P;
        double hb[NSA], bl[NSA];
        bool zero = false;
        P.tf[0] = P.tf[1] = P.tf[2] = 1.0f;
#pragma unroll 1
        for (int i = 0; i < D; ++i) {
            const FxCoord u = fx_next(walk[i * BLOCK], S.zmod[i], S.qz[i], S.rz[i], n32, S.job.inv_n, S.delta[i],
                                      S.dfix[i], walk + i * BLOCK);
            zero |= u.y.m == 0;
            // t, 1 - t and 1 - 2t (c, negative for t > 1/2)
            FxM t, v, c;
            bool cneg;
            if (Lc.transform == 0) {
                const FxM s = fx_korobov(u);
                const FxM b = fx_one_minus(s);
                t = u.lower ? s : b;
                v = u.lower ? b : s;
                const uint64_t S2 = s.e >= -64 ? (s.m >> (-1 - s.e)) << 1 : 0;   // 2s (0 for s = 1/2)
                c = (S2 != 0 || s.e == -1) ? FxM{0 - S2, -1} : FxM{1ULL << 63, 0};
                cneg = !u.lower;
                w = fx_norm(fx_mul(w, FxM{__umul64hi(u.y.m, u.big), u.y.e}));
            } else {
                if (Lc.transform == 1) {                // baker: t = 2y
                    t = FxM{u.y.m, u.y.e + 1};
                    v = fx_norm(FxM{0 - 2 * u.Y, -1});  // 1 - 2y
                    if (u.Y == 0) v = FxM{1ULL << 63, 0};
                    if (u.Y == 1ULL << 63) v = FxM{1ULL << 63, -61};   // t = 1: p -> 0 with p k = -lambda
                } else {
                    t = u.lower ? u.y : FxM{u.big, -1};
                    v = u.lower ? FxM{u.big, -1} : u.y;
                }
                const double x = fx_pack(v) - fx_pack(t);
                cneg = x < 0.0;
                const qmc_xf xc = qmc_xf_of(fabs(x));
                c = FxM{xc.m, xc.m ? xc.e : 0};
            }
            const double td = fx_pack(t);
            P.t[i] = td;
            // the real factors of the deformation, by mantissas
            const FxM lm{S.lamm[i], S.lame[i]};
            const FxM tv = fx_norm(fx_mul(t, v));
            c = fx_norm(c);
            if (c.m == 0 || c.e < -64) c.m = 0;
            P.p[i] = P.k[i] = P.s[i] = 0.0;
            if (lm.m) {
                P.p[i] = fd_signed(fx_pack(fx_norm(fx_mul(lm, tv))), S.lamneg[i] != 0);
                if (i < NS) P.s[i] = fd_signed(fx_pack(fx_norm(fx_mul(lm, v))), S.lamneg[i] != 0);
            } else if (S.lam[i] != 0.0) {               // not finite, or its products may not be normal
                P.s[i] = S.lam[i] * fx_pack(v);
                P.p[i] = P.s[i] * td;
            }
            if (c.m) P.k[i] = fd_signed(fx_pack(fx_norm(fx_mul(c, fd_rcp(tv)))), cneg);
            if constexpr (MIXED) {
                const float f = fd_to_float(td);
                P.tf[S.perm[i]] = f;
            }
            if (i < NS && u.y.m) {
                const qmc_xf r = qmc_xf_rcp3(qmc_xf{t.m, t.e, 0});
                hb[i] = S.bd[i] * fx_pack(FxM{r.m, r.e});
                if (NS + HI > 1) bl[i] = S.bd[i] * qmc_ilog_core(t.e, t.m & 0x7FFFFFFFFFFFFFFFULL, S.logtab);
            }
        }
        if (zero) continue;
        double h[NSA][NO];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            h[q][0] = hb[q];
            if constexpr (NS + HI > 1) h[q][1] = o.mul(hb[q], bl[q]);
            if constexpr (NS + HI > 2) h[q][2] = o.mul(h[q][1], fx_half(bl[q]));
        }
        dc res[NO];
        FxM q0{1ULL << 63, 0};
        FdFold<D, BLOCK, NS, HI, MIXED>{P, o, h, Lc.prow, signfail, q0}.template run<NS, 0>(res);
        // the weight (1 without korobov3) and, for NS = 0, the corner's factor
        FxM wt{1ULL << 63, 0};
        if (Lc.transform == 0) wt = fx_norm(fx_mul(fx_mul(w, w), w));
        if constexpr (NS == 0) wt = fx_norm(fx_mul(wt, q0));
        const double W = qmc_xf_to_double(qmc_xf{wt.m, wt.e, 0});
#pragma unroll
        for (int i = 0; i < NO; ++i) {
            accN[i].re = fma(res[i].re, W, accN[i].re);
            accN[i].im = fma(res[i].im, W, accN[i].im);
        }
    }
#pragma unroll
    for (int q = 0; q < LMAX; ++q) {
        dc v{0.0, 0.0};
#pragma unroll
        for (int i = 0; i < NO; ++i)
            if (i == lo + q + NS) v = accN[i];
        if (q < nord) acc[q] = v;
    }
}

// Stage the sector of S.job at its kinematic point (all threads)
template <int BLOCK, bool MIXED>
__device__ __forceinline__ void fd_stage(FdShared &S, const QmcLaunch &Lc) {
    const int sidx = S.job.sector, pidx = S.job.point;
    if (sidx == S.cached_sector && pidx == S.cached_point) return;
    const QmcSectorDev *src = Lc.sectors + sidx;
    const int d = src->d, ns = src->ns, nU = src->nU, nF = src->nF;
    // FP64: only U and F are read; mixed precision also the derivatives of F
    const int nm = MIXED ? src->nmono : nU + nF;
    if (threadIdx.x < 10) S.qc[threadIdx.x] = 0.0;
    if (threadIdx.x >= 10 && threadIdx.x < 13) S.qa[threadIdx.x - 10] = 0.0;
    if (threadIdx.x == 13) S.qmask = S.gvar = S.hvar = 0;
    int slot[3], next = ns;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        bool sing = false;
        for (int q = 0; q < ns; ++q)
            if (src->sing[q] == j) {
                slot[j] = q;
                sing = true;
            }
        if (!sing) slot[j] = next++;
    }
    __syncthreads();
    const double *kin = Lc.kin + (size_t)pidx * Lc.ninv;
    for (int m = threadIdx.x; m < nm; m += BLOCK) {
        const QmcMono &Mo = Lc.monos[src->monoU + m];
        double v = Mo.coef[0];
        for (int i = 0; i < Lc.ninv && i + 1 < QMC_NCOEF; ++i) v = fma(Mo.coef[i + 1], kin[i], v);
        S.cval[m] = v;
        S.cvalf[m] = (float)v;
        if constexpr (MIXED) {
            uint32_t off[3] = {0, 0, 0}, k = 0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const uint32_t ej = (Mo.exps >> (4 * j)) & 15u;
                if (ej) {
                    const uint32_t at = (uint32_t)(Lc.prow * j + (int)ej - 1) * (BLOCK * 4);
                    if (k == 0) off[0] = at;
                    else if (k == 1) off[1] = at;
                    else off[2] = at;
                    ++k;
                }
            }
            S.mdesc[m] = make_uint4(off[0] | (off[1] << 16), off[2], 0, k);
        } else {
            uint32_t e = 0;
            int first = -1, second = -1;             // F: the one or two factors of a monomial
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const uint32_t ej = (Mo.exps >> (4 * j)) & 15u;
                e |= ej << (4 * slot[j]);
                for (uint32_t q = 0; q < ej; ++q) {
                    if (first < 0) first = slot[j];
                    else second = slot[j];
                }
            }
            S.exps[m] = e;
            if (m >= nU) {
                int idx = 0;
                if (first >= 0) idx = second < 0 ? 1 + first : (first == second ? 4 + first : 6 + first + second);
                atomicAdd(&S.qc[idx], v);
                if (idx >= 4 && idx < 7) atomicAdd(&S.qa[idx - 4], v + v);
                if (idx >= 4 && v != 0.0) atomicOr(&S.qmask, idx >= 7 ? 1 << (idx - 7) : 8 << (idx - 4));
            }
        }
    }
    if (threadIdx.x >= 32 && threadIdx.x < 35) {
        const int j = (int)threadIdx.x - 32;
        const int sl = j == 0 ? slot[0] : (j == 1 ? slot[1] : slot[2]);
        S.slotof[j] = sl;
        S.perm[sl] = j;
        S.avar[sl] = src->a[j];
        S.bvar[sl] = src->bi[j];
        S.bd[sl] = src->b[j];
        S.dFoff[j] = src->dFoff[j];
        S.dFn[j] = src->dFn[j];
    }
    if (threadIdx.x >= 64 && threadIdx.x < 64 + QMC_NHESS) {
        S.Hoff[threadIdx.x - 64] = src->Hoff[threadIdx.x - 64];
        S.Hn[threadIdx.x - 64] = src->Hn[threadIdx.x - 64];
    }
    if (threadIdx.x == 96) {
        S.d = d;
        S.ns = ns;
        S.nU = nU;
        S.nF = nF;
        S.dbase = nU + nF;
        S.prow = Lc.prow;
        S.u0 = (int)src->u0;
        S.f0 = (int)src->f0;
        S.u1 = src->u1i;
        S.f1 = src->f1i;
        int reg = 0;
        for (int j = 0; j < d; ++j)
            if ((src->regular_mask >> j) & 1) reg |= 1 << (j == 0 ? slot[0] : (j == 1 ? slot[1] : slot[2]));
        S.regular = reg;
        double w = src->weight_b;
        if (Lc.transform == 0)
            for (int j = 0; j < d; ++j) w *= 140.0;
        S.w = w;
        S.cached_sector = sidx;
        S.cached_point = pidx;
    }
    __syncthreads();
    if constexpr (MIXED) {
        // the constant derivatives (no monomial, or the constant one alone)
        if (threadIdx.x < 9) {
            const int i = threadIdx.x;
            int m0 = 0, n = 0;
            if (i < 3) {
                if (i < d) {
                    m0 = S.dFoff[i];
                    n = S.dFn[i];
                }
            } else {
                const int x = i < 6 ? i - 3 : (i == 8 ? 1 : 0), z = i < 6 ? x : (i == 6 ? 1 : 2);   // slots
                if (z < d) {
                    const int a = min(S.perm[x], S.perm[z]), b = max(S.perm[x], S.perm[z]);
                    const int q = a * QMC_DMAX - a * (a - 1) / 2 + (b - a);
                    m0 = S.Hoff[q];
                    n = S.Hn[q];
                }
            }
            const bool constant = n == 0 || (n == 1 && S.mdesc[S.dbase + m0].w == 0);
            const float v = n == 0 || !constant ? 0.0f : S.cvalf[S.dbase + m0];
            if (i < 3) {
                S.gconst[i] = v;
                if (!constant) atomicOr(&S.gvar, 1 << i);
            } else {
                S.hconst[i - 3] = (double)v;
                if (!constant) atomicOr(&S.hvar, 1 << (i - 3));
                // the coupling (slots 01, 02, 12) enters the minors
                if (i >= 6 && !(constant && v == 0.0f)) atomicOr(&S.qmask, 1 << (i - 6));
            }
        }
    }
}

// Resident 128-thread units the registers must allow. Measured at 4 and 6: FP64
// massive box 7.3e9 and 7.7e9 evaluations/s, massless box 1.86e9 and 1.72e9;
// mixed massive box 5.9e9 and 6.6e9; the mixed amplitude (sums to eps^1)
// 36.6 and 38.9 ms.
template <bool MIXED, int HI> constexpr int fd_min_units() { return MIXED && HI == 0 ? 6 : 4; }
template <bool MIXED, int BLOCK, int HI>
__global__ void __launch_bounds__(BLOCK, fd_min_units<MIXED, HI>() * 128 / BLOCK) qmc_deformed_kernel(QmcLaunch Lc, int ppt) {
    constexpr int LMAX = 4;
    FdShared &S = fd_shared();
    const int lo = Lc.lo, nord = Lc.norders;
    if (threadIdx.x == 0) {
        S.cached_sector = -1;
        S.cached_point = -1;
        S.mone = Lc.mone;
        S.nzero = Lc.nzero;
    }
    for (int i = threadIdx.x; i < 3 * QMC_LOG_TABLE_ROWS; i += BLOCK) S.logtab[i] = kLogTable[i];
    for (int i = threadIdx.x; i < QMC_ATAN_TABLE_ROWS; i += BLOCK)
        S.atan63[i] = __double2ll_rn(kAtanTable[2 * i] * 0x1p63) + __double2ll_rn(kAtanTable[2 * i + 1] * 0x1p63);
    for (;;) {
        __syncthreads();  // previous tile fully consumed
        if (threadIdx.x == 0) {
            const unsigned long long tile = atomicAdd(Lc.queue, 1ULL);
            S.tile = tile;
            if (tile < Lc.ntiles) {
                int lo_j = 0, hi_j = Lc.njobs - 1;
                while (lo_j < hi_j) {
                    const int mid = (lo_j + hi_j + 1) >> 1;
                    if (Lc.jobs[mid].tile_begin <= tile) lo_j = mid;
                    else hi_j = mid - 1;
                }
                S.job_index = lo_j;
            }
        }
        __syncthreads();
        const unsigned long long tile = S.tile;
        if (tile >= Lc.ntiles) break;
        {
            const int nw = sizeof(QmcJobDev) / 4;
            for (int i = threadIdx.x; i < nw; i += BLOCK)
                reinterpret_cast<int32_t *>(&S.job)[i] = reinterpret_cast<const int32_t *>(Lc.jobs + S.job_index)[i];
        }
        __syncthreads();
        fd_stage<BLOCK, MIXED>(S, Lc);
        const uint64_t local = tile - S.job.tile_begin;
        const uint64_t s = local / (uint64_t)S.job.tiles_per_shift;
        const uint64_t chunk = local - s * (uint64_t)S.job.tiles_per_shift;
        if ((int)threadIdx.x < S.d) {
            const int i = threadIdx.x, j = S.perm[i];
            const uint64_t nn = S.job.n;
            const uint64_t minv = ~0ULL / nn;
            const double dl = (S.job.flags & 1) ? 0.0 : splitmix_uniform(S.job.seed_state, s * S.d + j);
            S.delta[i] = dl;
            S.dfix[i] = (uint64_t)(dl * 18446744073709551616.0);   // exact: a multiple of 2^-53
            uint64_t zm, qz, rz;
            fx_divmod(S.job.z[j], nn, minv, zm);
            fx_fixdiv(zm, nn, minv, qz, rz);
            S.qz[i] = qz;
            S.rz[i] = (uint32_t)rz;
            S.zmod[i] = (uint32_t)zm;
            S.lam[i] = S.job.lambda[j];
            // (t (1 - t) >= 2^-212: from 2^-800 on its products with lambda are normal)
            const qmc_xf lx = qmc_xf_of(S.job.lambda[j]);
            const bool usual = lx.m && lx.e > -800 && lx.e < 1024;
            S.lamm[i] = usual ? lx.m : 0;
            S.lame[i] = usual ? lx.e : 0;
            S.lamneg[i] = lx.neg;
            if (i == 0) S.minv = minv;
        }
        __syncthreads();

        dc acc[LMAX];
#pragma unroll
        for (int q = 0; q < LMAX; ++q) acc[q] = dc{0.0, 0.0};
        int signfail = 0;
        const uint64_t kt0 = chunk * (uint64_t)Lc.tile_k;
        const uint64_t kt1 = min(S.job.n, kt0 + (uint64_t)Lc.tile_k);
        const uint64_t k0 = kt0 + (uint64_t)threadIdx.x * (uint64_t)ppt;
        if (k0 < kt1) {
            const uint64_t kend = min(kt1, k0 + (uint64_t)ppt);
            const int ns = S.ns;
            if (S.d == 3) {
                if (ns == 0) fd_points<3, BLOCK, 0, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
                else if (ns == 1) fd_points<3, BLOCK, 1, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
                else fd_points<3, BLOCK, 2, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
            } else if (S.d == 2) {
                if (ns == 0) fd_points<2, BLOCK, 0, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
                else if (ns == 1) fd_points<2, BLOCK, 1, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
                else fd_points<2, BLOCK, 2, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
            } else {
                if (ns == 0) fd_points<1, BLOCK, 0, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
                else fd_points<1, BLOCK, 1, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc, signfail);
            }
        }
        // sign-check failures of this tile: per job (if counted) and in total
        if (__ballot_sync(0xffffffffu, signfail != 0)) {
            const unsigned v = __reduce_add_sync(0xffffffffu, (unsigned)signfail);
            if ((threadIdx.x & 31) == 0) {
                atomicAdd(Lc.status, (unsigned long long)v);
                if (Lc.job_fail) atomicAdd(Lc.job_fail + S.job_index, v);
            }
        }
        // block reduction: warp sums, then warps in index order
        double flat[2 * LMAX];
#pragma unroll
        for (int q = 0; q < LMAX; ++q) {
            flat[2 * q] = acc[q].re;
            flat[2 * q + 1] = acc[q].im;
        }
        fx_block_sums(flat, 2 * nord, S.red);
        __syncthreads();
        if (threadIdx.x < 2 * nord) {
            double sum = 0.0;
            for (int wp = 0; wp < BLOCK / 32; ++wp) sum += S.red[wp][threadIdx.x];
            sum *= S.w;
            __stcs(&Lc.partials[tile * (uint64_t)(2 * nord) + threadIdx.x], sum);
            if (!isfinite(sum)) atomicAdd(Lc.status + 1, 1ULL);
        }
    }
}

template <bool MIXED, int BLOCK> constexpr int fd_dyn_smem(int prow) {
    return (int)sizeof(FdShared) + 16 * 3 * BLOCK + (MIXED ? 12 * 3 * prow * BLOCK : 0);
}

template <bool MIXED, int BLOCK, int HI> bool fd_allow() {
    static std::atomic<uint64_t> done{0};
    return qmc_allow_smem(done, qmc_deformed_kernel<MIXED, BLOCK, HI>, fd_dyn_smem<MIXED, BLOCK>(QMC_EMAX));
}

template <bool MIXED, int BLOCK, int HI>
int fd_launch(const QmcLaunch *L, int grid, cudaStream_t st) {
    if (L->prow < 1 || L->prow > QMC_EMAX || !fd_allow<MIXED, BLOCK, HI>()) return -1;
    qmc_deformed_kernel<MIXED, BLOCK, HI><<<grid, BLOCK, fd_dyn_smem<MIXED, BLOCK>(L->prow), st>>>(
        *L, (int)((L->tile_k + BLOCK - 1) / BLOCK));
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <bool MIXED, int BLOCK, int HI> int fd_occupancy(int prow) {
    if (!fd_allow<MIXED, BLOCK, HI>()) return 0;
    int v = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &v, qmc_deformed_kernel<MIXED, BLOCK, HI>, BLOCK, fd_dyn_smem<MIXED, BLOCK>(prow));
    return e == cudaSuccess ? v : 0;
}
