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
//  * transform, weight, 1/t, ln t, reciprocals and logarithms run on the
//    integer pipe, and the corners are folded variable by variable as in
//    qmc_real.cuh (complex corner series, real factors).
// Measured (evaluations/s, general kernel -> this one): massive box, 64 points
// at n = 10007, 1.74e9 -> 5.9e9 (90 FP64 instructions per evaluation, pipe
// 93 % busy); the same in mixed precision, 256 points at n = 1009,
// 2.85e9 -> 5.4e9; massless box, 16 physical points at n = 4001, 5.9e8 ->
// 1.06e9 (453, pipe 90 %). 16 warps (128 registers) beat 12 and 8 even with
// the FP64 kernel's spills.
// MIXED: derivatives of F and U(z), F(z) from FP32 monomial products in the
// order of the general mixed kernel, everything after them in FP64.

struct alignas(16) FdShared {
    uint64_t logtab[3 * QMC_LOG_TABLE_ROWS + 1];
    double atantab[2 * QMC_ATAN_TABLE_ROWS];
    uint32_t exps[QMC_MAXMONO];      // FP64: variables in slot order (singular first)
    uint4 mdesc[QMC_MAXMONO];        // MIXED: factors as in FxShared, original variable order
    double cval[QMC_MAXMONO];
    float cvalf[QMC_MAXMONO];
    // F(t) = qc[0] + sum_j t_j (qc[1+j] + qc[4+j] t_j) + qc[7] t_0 t_1 + qc[8] t_0 t_2 + qc[9] t_1 t_2 (slots)
    double qc[10];
    int32_t qmask;                   // bits 0..2: qc[7..9] present
    int32_t d, ns, nU, nF, dbase, prow;
    int32_t dFoff[3], dFn[3], Hoff[QMC_NHESS], Hn[QMC_NHESS];
    int32_t perm[QMC_DMAX], slotof[QMC_DMAX], avar[QMC_DMAX], bvar[QMC_DMAX];
    double bd[QMC_DMAX], lam[QMC_DMAX];
    int32_t regular, u0, f0, u1, f1;
    double delta[QMC_DMAX];
    uint64_t dfix[QMC_DMAX], qz[QMC_DMAX];
    uint32_t rz[QMC_DMAX], zmod[QMC_DMAX];
    uint64_t minv;
    double w, mone, nzero;
    QmcJobDev job;
    unsigned long long tile;
    int cached_sector, cached_point, job_index;
    double red[8][8];
};
__device__ __forceinline__ FdShared &fd_shared() { return *reinterpret_cast<FdShared *>(qmc_fx_raw); }

// 0.5 ln(a / b) of positive finite a, b, and 1 / x: integer pipe, out of line
__device__ __noinline__ double fd_half_log_ratio(double a, double b) {
    const qmc_xf x = qmc_xf_of(a), y = qmc_xf_of(b);
    if (x.m == 0 || y.m == 0) return a * (1.0 / b);      // (the integrand is singular there)
    const FxM q = fx_norm(fx_mul(FxM{x.m, x.e}, FxM{qmc_xf_rcp3(y).m, qmc_xf_rcp3(y).e}));
    return fx_half(qmc_ilog_xf(qmc_xf{q.m, q.e, 0}, fd_shared().logtab));
}
__device__ __noinline__ double fd_rcp(double x) {
    const qmc_xf a = qmc_xf_of(x);
    if (a.m == 0) return 1.0 / x;
    return qmc_xf_to_double(qmc_xf_rcp3(a));
}
__device__ __noinline__ double fd_atan2(double y, double x) { return qatan2(y, x, fd_shared().atantab); }

// FP32 <-> FP64 conversions on the integer pipe (normal range; below it 0)
__device__ __forceinline__ float fd_to_float(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(b >> 32);
    const int e = (int)((hi >> 20) & 0x7FFu) - 896;                    // FP32's biased exponent
    uint32_t m = (uint32_t)(b >> 29) & 0x7FFFFFu;
    const uint32_t rest = (uint32_t)b & 0x1FFFFFFFu;
    const uint32_t up = (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) ? 1u : 0u;
    const uint32_t v = ((uint32_t)e << 23) + m + up;
    return e >= 255 ? __double2float_rn(x) : (e > 0 ? __uint_as_float((hi & 0x80000000u) | v) : 0.0f);
}
__device__ __forceinline__ double fd_to_double(float x) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t e = (b >> 23) & 255u;
    if (e == 0) return 0.0;
    if (e == 255) return (double)x;
    const uint32_t hi = (b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7FFFFFu) >> 3);
    return __hiloint2double((int)hi, (int)(b << 29));
}

// complex arithmetic in FMAs (an FP64 multiply holds the pipe longer than an FMA)
struct FdOps {
    double mone, nzero;
    __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nzero); }
    __device__ __forceinline__ double add(double a, double b) const { return fma(b, -mone, a); }
    __device__ __forceinline__ double sub(double a, double b) const { return fma(b, mone, a); }
    __device__ __forceinline__ dc mul(dc a, dc b) const {
        return dc{fma(a.re, b.re, mul(-a.im, b.im)), fma(a.re, b.im, mul(a.im, b.re))};
    }
    __device__ __forceinline__ dc sub(dc a, dc b) const { return dc{sub(a.re, b.re), sub(a.im, b.im)}; }
    // num *= x^e or den *= x^-e
    __device__ __forceinline__ void ipow(dc x, int e, dc &num, bool &hn, dc &den, bool &hd) const {
        if (e == 0) return;
        const int a = e > 0 ? e : -e;
        dc p = x;
        if (a > 1) {
            const dc x2 = dc{fma(x.re, x.re, mul(-x.im, x.im)), mul(x.re + x.re, x.im)};
            p = a == 3 ? mul(x2, x) : x2;
            if (a == 4) p = dc{fma(x2.re, x2.re, mul(-x2.im, x2.im)), mul(x2.re + x2.re, x2.im)};
        }
        if (e > 0) {
            num = hn ? mul(num, p) : p;
            hn = true;
        } else {
            den = hd ? mul(den, p) : p;
            hd = true;
        }
    }
};

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
    double t[3], s[3], p[3], r[3];   // t; lambda (1 - t); lambda t (1 - t); lambda (1 - 2t)  (slots)
    float tf[3];                     // FP32 t, original variable order (MIXED)
};
struct FdCorner {
    dc B, L;
};

// The corner with the slots of V at t = 0 (D variables, NS of them singular)
template <int D, int BLOCK, int NS, int HI, int V, bool MIXED>
__device__ __forceinline__ FdCorner fd_corner(const FdPoint &P, const FdOps &o, int prow, int &signfail) {
    const FdShared &S = fd_shared();
    constexpr bool lam = HI > 0 || V != 0;              // needs its eps exponent
    constexpr int NA = D - __builtin_popcount(V);       // variables left
    double g[D];                                        // dF/dt_j
    double Vd[D], Vo[D][D];                             // J = 1 - i V: diagonal, off-diagonal
    double y[D];
    dc F, U{1.0, 0.0};
    const bool needU = S.u0 != 0 || (lam && S.u1 != 0);
#pragma unroll
    for (int j = 0; j < D; ++j)
#pragma unroll
        for (int k = 0; k < D; ++k) Vo[j][k] = 0.0;
    const int qm = MIXED ? 7 : S.qmask;
    if constexpr (!MIXED) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            g[j] = S.qc[1 + j];
            if (!(V >> j & 1)) g[j] = fma(S.qc[4 + j], P.t[j] + P.t[j], g[j]);
        }
#pragma unroll
        for (int j = 0; j < D; ++j)
#pragma unroll
            for (int k = j + 1; k < D; ++k)
                if (qm >> (j + k - 1) & 1) {
                    const double A = S.qc[6 + j + k];
                    if (!(V >> k & 1)) g[j] = fma(A, P.t[k], g[j]);
                    if (!(V >> j & 1)) g[k] = fma(A, P.t[j], g[k]);
                    if (!(V >> j & 1) && !(V >> k & 1)) {
                        Vo[j][k] = o.mul(A, P.p[j]);
                        Vo[k][j] = o.mul(A, P.p[k]);
                    }
                }
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (!(V >> j & 1)) Vd[j] = fma(S.qc[4 + j], P.p[j] + P.p[j], o.mul(P.r[j], g[j]));
    } else {
        // FP32 derivatives, original variable order
#pragma unroll
        for (int j = 0; j < D; ++j) fd_put<BLOCK>(j, prow, (V >> S.slotof[j] & 1) ? 0.0f : P.tf[j]);
        float gf[3], Hf[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            gf[j] = 0.0f;
            if (j < D) gf[j] = fd_poly<BLOCK>(S.dbase + S.dFoff[j], S.dFn[j]);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = j; k < 3; ++k) {
                Hf[j][k] = 0.0f;
                if (k < D) {
                    const int h = j * QMC_DMAX - j * (j - 1) / 2 + (k - j);
                    Hf[j][k] = fd_poly<BLOCK>(S.dbase + S.Hoff[h], S.Hn[h]);
                }
                Hf[k][j] = Hf[j][k];
            }
        // to slot order
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const int pi = S.perm[i];
            g[i] = fd_to_double(pi == 0 ? gf[0] : (pi == 1 ? gf[1] : gf[2]));
#pragma unroll
            for (int k = i; k < D; ++k) {
                if ((V >> i & 1) || (V >> k & 1)) continue;
                const int pk = S.perm[k];
                float h = 0.0f;
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int b = 0; b < 3; ++b)
                        if (pi == a && pk == b) h = Hf[a][b];
                const double H = fd_to_double(h);
                if (i == k) Vd[i] = fma(H, P.p[i], o.mul(P.r[i], g[i]));
                else {
                    Vo[i][k] = o.mul(H, P.p[i]);
                    Vo[k][i] = o.mul(H, P.p[k]);
                }
            }
        }
    }
    // rho_j = 1 - i g_j lambda_j (1 - t_j), z_j = t_j rho_j
    double gl[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        gl[j] = 0.0;
        y[j] = 0.0;
        if (V >> j & 1) gl[j] = o.mul(S.lam[j], g[j]);
        else {
            if (j < NS || needU || MIXED || (S.regular >> j & 1)) gl[j] = o.mul(P.s[j], g[j]);
            y[j] = o.mul(P.p[j], g[j]);
        }
    }
    // det J over the remaining variables
    dc J{1.0, 0.0};
    {
        int a[3] = {0, 0, 0}, na = 0;
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (!(V >> j & 1)) a[na++] = j;
        if constexpr (NA == 1) {
            J = dc{1.0, -Vd[a[0]]};
        } else if constexpr (NA == 2) {
            const int x = a[0], z = a[1];
            const double det = fma(Vd[x], Vd[z], o.mul(-Vo[x][z], Vo[z][x]));
            J = dc{1.0 - det, -(Vd[x] + Vd[z])};
        } else if constexpr (NA == 3) {
            double m01 = o.mul(Vd[0], Vd[1]), m02 = o.mul(Vd[0], Vd[2]), m12 = o.mul(Vd[1], Vd[2]);
            if (qm & 1) m01 = fma(-Vo[0][1], Vo[1][0], m01);
            if (qm & 2) m02 = fma(-Vo[0][2], Vo[2][0], m02);
            if (qm & 4) m12 = fma(-Vo[1][2], Vo[2][1], m12);
            double det = o.mul(Vd[0], m12);
            if (qm & 1) {
                double c = o.mul(Vo[1][0], Vd[2]);
                if ((qm & 6) == 6) c = fma(-Vo[1][2], Vo[2][0], c);
                det = fma(-Vo[0][1], c, det);
            }
            if (qm & 2) {
                double c = o.mul(-Vd[1], Vo[2][0]);
                if ((qm & 5) == 5) c = fma(Vo[1][0], Vo[2][1], c);
                det = fma(Vo[0][2], c, det);
            }
            J = dc{1.0 - o.add(o.add(m01, m02), m12), o.sub(det, o.add(o.add(Vd[0], Vd[1]), Vd[2]))};
        }
    }
    // U and F on the contour
    if constexpr (!MIXED) {
        double re = S.qc[0], im = 0.0;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            if (V >> j & 1) continue;
            // t_j (b_j + g_j) / 2 - y_j (A_jj y_j / 2 + sum_{k > j} A_jk y_k);  -y_j g_j
            re = fma(fx_half(P.t[j]), S.qc[1 + j] + g[j], re);
            double q = o.mul(S.qc[4 + j], y[j]);
#pragma unroll
            for (int k = j + 1; k < D; ++k)
                if (!(V >> k & 1) && (qm >> (j + k - 1) & 1)) q = fma(S.qc[6 + j + k], y[k], q);
            re = fma(-y[j], q, re);
            im = fma(-y[j], g[j], im);
        }
        F = dc{re, im};
        if (needU) {
            // monomials by factors, uniform branches; t_V = 0 drops monomials
            U = dc{0.0, 0.0};
            uint32_t vm = 0;
#pragma unroll
            for (int j = 0; j < D; ++j)
                if (V >> j & 1) vm |= 15u << (4 * j);
            dc z[D];
#pragma unroll
            for (int j = 0; j < D; ++j) z[j] = dc{P.t[j], -o.mul(P.t[j], gl[j])};
            for (int m = 0; m < S.nU; ++m) {
                const uint32_t e = S.exps[m];
                if (e & vm) continue;
                const double c = S.cval[m];
                if (e == 0) {
                    U.re = o.add(U.re, c);
                    continue;
                }
                dc v{1.0, 0.0};
                bool first = true;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    if (V >> j & 1) continue;
                    for (int q = (int)(e >> (4 * j) & 15u); q > 0; --q) {
                        v = first ? z[j] : o.mul(v, z[j]);
                        first = false;
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
                    else zi = o.mul(-P.t[i], gl[i]);
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
    if (__double_as_longlong(F.im) > 0) ++signfail;
    // B = det J / prod rho (kept singular) prod z^a (regular) U^u0 F^f0 and
    // the corner's exponent L = ln(prod rho^b prod z^b U^u1 F^f1), one complex
    // logarithm whose argument is restored to the sum of the factors'
    // principal arguments by an FP32 estimate
    FdCorner out{dc{1.0, 0.0}, dc{0.0, 0.0}};
    dc num = J, den{1.0, 0.0}, Xn{1.0, 0.0}, Xd{1.0, 0.0};
    bool hn = NA > 0, hd = false, xn = false, xd = false;
    float sarg = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
        if (j < NS) {
            const dc rho{1.0, -gl[j]};
            if (!(V >> j & 1)) {
                den = hd ? o.mul(den, rho) : rho;
                hd = true;
            }
            if constexpr (lam) {
                o.ipow(rho, S.bvar[j], Xn, xn, Xd, xd);
                sarg = fmaf((float)S.bvar[j], arg32(rho, false), sarg);
            }
        } else if (S.regular >> j & 1) {
            const dc z{P.t[j], -o.mul(P.t[j], gl[j])};
            o.ipow(z, S.avar[j], num, hn, den, hd);
            if constexpr (lam)
                if (S.bvar[j] != 0) {
                    o.ipow(z, S.bvar[j], Xn, xn, Xd, xd);
                    sarg = fmaf((float)S.bvar[j], arg32(z, false), sarg);
                }
        }
    }
    o.ipow(U, S.u0, num, hn, den, hd);
    o.ipow(F, S.f0, num, hn, den, hd);
    if (hd) {
        const double q = fd_rcp(fma(den.re, den.re, o.mul(den.im, den.im)));
        const dc di{o.mul(den.re, q), o.mul(-den.im, q)};
        out.B = hn ? o.mul(num, di) : di;
    } else {
        out.B = num;
    }
    if constexpr (lam) {
        if (S.u1 != 0) {
            o.ipow(U, S.u1, Xn, xn, Xd, xd);
            sarg = fmaf((float)S.u1, arg32(U, false), sarg);
        }
        if (S.f1 != 0) {
            o.ipow(F, S.f1, Xn, xn, Xd, xd);
            sarg = fmaf((float)S.f1, arg32(F, true), sarg);
        }
        const dc X = xd ? (xn ? o.mul(Xn, conj_(Xd)) : conj_(Xd)) : Xn;   // |Xd|^2 Xn / Xd
        const double phi = fd_atan2(X.im, X.re);
        const float kf = rintf((sarg - __double2float_rn(phi)) * 0.15915494f);
        const double nn = xn ? fma(Xn.re, Xn.re, o.mul(Xn.im, Xn.im)) : 1.0;
        const double nd = xd ? fma(Xd.re, Xd.re, o.mul(Xd.im, Xd.im)) : 1.0;
        out.L = dc{fd_half_log_ratio(nn, nd), kf == 0.0f ? phi : fma((double)kf, 2.0 * CUDART_PI, phi)};
    }
    return out;
}

// Depth-first fold of the corners (see qmc_real.cuh), complex series
template <int D, int BLOCK, int NS, int HI, bool MIXED> struct FdFold {
    const FdPoint &P;
    const FdOps &o;
    const double (&h)[SlotArr<NS>::N][NS + HI + 1];
    int prow;
    int &signfail;

    template <int Q, int V>
    __device__ __forceinline__ void run(dc (&out)[Q + __builtin_popcount(V) + HI + 1]) const {
        constexpr int pv = __builtin_popcount(V);
        if constexpr (Q == 0) {
            const FdCorner c = fd_corner<D, BLOCK, NS, HI, V, MIXED>(P, o, prow, signfail);
            out[0] = c.B;
            if constexpr (pv + HI >= 1) out[1] = o.mul(c.B, c.L);
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
    const FdOps o{S.mone, S.nzero};
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
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const FxCoord u = fx_next(walk[i * BLOCK], S.zmod[i], S.qz[i], S.rz[i], n32, S.job.inv_n, S.delta[i],
                                      S.dfix[i], walk + i * BLOCK);
            zero |= u.y.m == 0;
            // t and 1 - t
            FxM t, v;
            if (Lc.transform == 0) {
                const FxM s = fx_korobov(u);
                const FxM b = fx_one_minus(s);
                t = u.lower ? s : b;
                v = u.lower ? b : s;
                w = fx_norm(fx_mul(w, FxM{__umul64hi(u.y.m, u.big), u.y.e}));
            } else if (Lc.transform == 1) {             // baker
                t = FxM{u.y.m, u.y.e + 1};
                const uint64_t c = 0 - 2 * u.Y;         // 1 - 2y; 0 (u = 1/2): exactly zero
                v = fx_norm(FxM{c, -1});
                if (u.Y == 0) v = FxM{1ULL << 63, 0};
                if (u.Y == 1ULL << 63) v.m = 0;
            } else {
                t = u.lower ? u.y : FxM{u.big, -1};
                v = u.lower ? FxM{u.big, -1} : u.y;
            }
            const double td = fx_pack(t), vd = v.m ? fx_pack(v) : 0.0;
            P.t[i] = td;
            const double lm = S.lam[i];
            P.s[i] = o.mul(lm, vd);
            P.p[i] = o.mul(td, P.s[i]);
            P.r[i] = fma(-lm, td, P.s[i]);
            if constexpr (MIXED) {
                const float f = fd_to_float(td);
                const int pj = S.perm[i];
                if (pj == 0) P.tf[0] = f;
                else if (pj == 1) P.tf[1] = f;
                else P.tf[2] = f;
            }
            if (i < NS && u.y.m) {
                const qmc_xf r = qmc_xf_rcp3(qmc_xf{t.m, t.e, 0});
                hb[i] = S.bd[i] * fx_pack(FxM{r.m, r.e});
                if (NS + HI > 1) bl[i] = S.bd[i] * qmc_ilog_core(t.e, t.m & 0x7FFFFFFFFFFFFFFFULL, S.logtab);
            }
        }
        if (zero) continue;
        double W = 1.0;
        if (Lc.transform == 0) W = fx_pack(fx_norm(fx_mul(fx_mul(w, w), w)));
        double h[NSA][NO];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            h[q][0] = hb[q];
            if constexpr (NS + HI > 1) h[q][1] = o.mul(hb[q], bl[q]);
            if constexpr (NS + HI > 2) h[q][2] = o.mul(h[q][1], fx_half(bl[q]));
        }
        dc res[NO];
        FdFold<D, BLOCK, NS, HI, MIXED>{P, o, h, Lc.prow, signfail}.template run<NS, 0>(res);
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
    if (threadIdx.x == 10) S.qmask = 0;
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
                if (idx >= 7 && v != 0.0) atomicOr(&S.qmask, 1 << (idx - 7));
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
}

#ifndef QMC_FD_MINB
#define QMC_FD_MINB 4
#endif
template <bool MIXED, int BLOCK, int HI>
__global__ void __launch_bounds__(BLOCK, QMC_FD_MINB * 128 / BLOCK) qmc_deformed_kernel(QmcLaunch Lc, int ppt) {
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
    for (int i = threadIdx.x; i < 2 * QMC_ATAN_TABLE_ROWS; i += BLOCK) S.atantab[i] = kAtanTable[i];
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
        // block reduction: warp shuffles, then warps in index order
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int q = 0; q < LMAX; ++q) {
            if (q >= nord) continue;
            double vr = acc[q].re, vi = acc[q].im;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                vr += __shfl_down_sync(0xffffffffu, vr, off);
                vi += __shfl_down_sync(0xffffffffu, vi, off);
            }
            if (lane == 0) {
                S.red[warp][2 * q] = vr;
                S.red[warp][2 * q + 1] = vi;
            }
        }
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
    static const bool ok = cudaFuncSetAttribute(qmc_deformed_kernel<MIXED, BLOCK, HI>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                fd_dyn_smem<MIXED, BLOCK>(QMC_EMAX)) == cudaSuccess;
    return ok;
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
