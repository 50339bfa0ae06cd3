// The real evaluator on integers: undeformed sectors whose sums end at eps^0
// (d <= 3: or eps^1), whose exponents u0, u1, f0, f1 are integers of magnitude <= 4 and whose U
// and F have non-negative coefficients at the job's kinematic point with a
// constant term c0 >= (sum of coefficients) / 128 (the host checks this per
// job; see fx_job_ok in qmc_host.cpp). Every Euclidean sector of the built-in
// integrals is one. Included by qmc_kernels.cu (parts 4 and 5).
//
// What bounds it, and why integers. An FP64 warp instruction holds an SMSP's
// FP64 pipe for 64 cycles (FMA from registers) or 76 (add, multiply, FMA with
// a constant); a 64 x 64 -> high 64 integer product takes 16 issue cycles and
// a 64-bit add 4. Only the eps series need FP64's range and sign, so:
//  * the shifted lattice coordinate, the transform, its weight, 1/t and ln t
//    come from 64-bit mantissas (never packed into a double in between);
//  * U and F are sums of positive terms, so they are evaluated in fixed
//    point: t as t 2^64, coefficients scaled so that their sum stays below
//    2^64, each factor one high product, subset sums over the singular
//    variables plain 64-bit adds. A monomial may lose a unit, 2^-63 of the sum
//    of coefficients or less, so at most 2^-55 of any corner value (all are
//    >= c0, which the rule keeps above 1/128 of that sum); an FP64 monomial may
//    lose 2^-53 of itself and again of the sum it enters;
//  * a corner's powers and logarithm follow from those integers directly.
// FP64 is left with each corner's series (B L^i / i!), their combination and
// the accumulation. Sectors with three or four singular variables (EX below)
// take the general kernel's roundings up to the corner values instead: t to
// FP64, monomials and group sums in FP64, subset sums and corner products in
// 64-bit mantissas in the same order, and the Moebius transform before the
// fold. Their eps^0 sums cancel by up to 1e8, so that the last bit of one
// corner of one point near the border shows in a shift's sum at 1e-7: with
// other roundings, each as good, results would not be comparable between the
// kernels (with these they agree to 1e-15).
//
// The combination folds one singular variable at a time instead of forming
// the Moebius transform of all corners and then every pole set:
//   S(no variable, V) = corner series g_V,
//   S(Q, V) = (b/t) e^{eps b ln t} [S(Q-1, V) - S(Q-1, V + q)] + S(Q-1, V + q) / eps,
// q = Q - 1, t = t_q, b = b_q, which is b_q times the plus-distribution
// subtraction of t_q (1 / prod b_q joins the sector's constant factor). It
// takes 132 FP64 operations for four variables (217 before), and evaluated
// depth first it keeps one pending series per level instead of all sixteen.
//
// Layout: a thread keeps its lattice walk and its power table in shared memory
// and runs one rolled loop over the variables and one over the corners, so
// that 80 registers (d <= 6, 24 warps per SM) or 64 (d <= 3, 32 warps) hold
// the rest and the code stays small. 384-thread blocks for d <= 6 because a
// block carries the 24.6 KB logarithm table: two of them fit, six of 128 do
// not. Measured on the double box (n = 10007, evaluations/s): the general
// kernel 9.7e8; this one with fixed-point corners for every sector 1.91e9 at 16
// warps, 2.07e9 at 20, 2.14e9 at 24, and with the general kernel's roundings in
// the EX sectors 1.66e9 at 24, 1.62e9 at 20 and 1.53e9 at 16. The box
// (n = 100003) 4.2e9 -> 7.4e9 at 16 warps, 8.3e9 at 32.

// 64-bit mantissa and exponent: value m 2^(e - 63), m not necessarily normalised
struct FxM {
    uint64_t m;
    int e;
};
__device__ __forceinline__ FxM fx_mul(FxM a, FxM b) { return FxM{__umul64hi(a.m, b.m), a.e + b.e + 1}; }
__device__ __forceinline__ FxM fx_norm(FxM a) {
    const int c = __clzll((long long)a.m);
    return FxM{a.m << c, a.e - c};
}

struct alignas(16) FxShared {
    uint64_t logtab[3 * QMC_LOG_TABLE_ROWS + 1];
    // a monomial's factors as offsets of the power-table rows (4-byte units, 16
    // bits each, in x, y, z) and their count (w); its coefficient times 2^sh
    // (mixed precision: its FP32 value in the low word; three or four
    // singular variables: the FP64 value)
    uint4 mdesc[QMC_MAXMONO];
    uint64_t cfix[QMC_MAXMONO];
    int32_t gs[2][QMC_NGROUP + 1];   // first monomial of each singular-mask group of U, F
    int32_t emax[2], sh[2];          // largest coefficient exponent and the scale of each polynomial
    int32_t csum[2];
    // variables in slot order: the singular ones first
    int32_t perm[QMC_DMAX], avar[QMC_DMAX];
    double bvar[QMC_DMAX];
    int32_t d, ns, regular;          // regular: slots >= ns with a != 0 or b != 0
    int32_t hasC, hasL;              // some regular a > 0; some regular b != 0
    uint32_t ex;                     // u0, f0, u1, f1 as signed bytes
    double delta[QMC_DMAX];
    uint64_t dfix[QMC_DMAX], qz[QMC_DMAX];
    uint32_t rz[QMC_DMAX], zmod[QMC_DMAX];
    uint64_t minv;                   // floor((2^64 - 1) / n)
    double w;
    double mone, nzero;              // -1 and -0 (operands of FMAs that add and multiply)
    QmcJobDev job;
    unsigned long long tile;
    int cached_sector, cached_point, job_index;
    double red[16][6];
};
extern __shared__ __align__(16) unsigned char qmc_fx_raw[];
__device__ __forceinline__ FxShared &fx_shared() { return *reinterpret_cast<FxShared *>(qmc_fx_raw); }
// the thread's columns: the power table (8 bytes, or 4 in mixed precision, per
// entry, rows BLOCK entries apart) and, in front of it, the lattice walk
template <int DMAX, int BLOCK> __device__ __forceinline__ uint4 *fx_walk() {
    return reinterpret_cast<uint4 *>(qmc_fx_raw + sizeof(FxShared)) + threadIdx.x;
}
template <int DMAX, int BLOCK> __device__ __forceinline__ unsigned char *fx_pt(int esize) {
    return qmc_fx_raw + sizeof(FxShared) + 16 * DMAX * BLOCK + esize * threadIdx.x;
}

// Warp sums of N values per lane (N a power of two, <= 8): while more than one
// is left, the lanes of each pair keep half of them and hand over the others,
// so that eight values take 9 additions instead of 40 (an FP64 addition holds
// its pipe for 76 cycles; at four points a thread the 40 were a twelfth of the
// deformed kernel's FP64 work). The same pairs as a shuffle-down tree per
// value, so the same bits. Lane l returns the sum of value l / (32 / N).
template <int N> __device__ __forceinline__ double fx_warp_sum(double (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int h = N / 2; h >= 1; h /= 2, off /= 2) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double give = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
#pragma unroll
    for (int o = 16 / N; o >= 1; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}
// The block's warps write the sums of values [0, count) to red[warp][]
template <int LMAX, int W>
__device__ __forceinline__ void fx_block_sums(const double (&acc)[LMAX], int count, double (&red)[16][W]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto sum = [&](auto tag) {
        constexpr int N = decltype(tag)::value;
        double v[N];
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = i < LMAX ? acc[i < LMAX ? i : 0] : 0.0;
        const double s = fx_warp_sum<N>(v);
        const int q = lane / (32 / N);
        if (lane % (32 / N) == 0 && q < count) red[warp][q] = s;
    };
    if (count <= 1) sum(std::integral_constant<int, 1>{});
    else if (count <= 2) sum(std::integral_constant<int, 2>{});
    else if (count <= 4) sum(std::integral_constant<int, 4>{});
    else sum(std::integral_constant<int, 8>{});
}

// x / n and x mod n for n < 2^32 with minv = floor((2^64 - 1) / n): the
// quotient estimate is at most 2 short
__device__ __forceinline__ uint64_t fx_divmod(uint64_t x, uint64_t n, uint64_t minv, uint64_t &r) {
    uint64_t q = __umul64hi(x, minv);
    r = x - q * n;
    if (r >= n) { r -= n; ++q; }
    if (r >= n) { r -= n; ++q; }
    return q;
}
__device__ __forceinline__ void fx_fixdiv(uint64_t a, uint64_t n, uint64_t minv, uint64_t &q, uint64_t &rem) {
    uint64_t r1;
    const uint64_t q1 = fx_divmod(a << 32, n, minv, r1);
    const uint64_t q0 = fx_divmod(r1 << 32, n, minv, rem);
    q = (q1 << 32) | q0;
}

// The shifted coordinate u as the 64-bit fixed point U = u 2^64, for
// r/n >= 2^-12: the roundings of walk_coord (RN(r/n) to 53 bits, then
// RN of the sum with the shift, folded) done in place. 0 for u = 0.
__device__ __forceinline__ uint64_t fx_coord(uint64_t Q, uint32_t R, uint32_t n, uint64_t D) {
    const int sh = 11 - __clz((int)(uint32_t)(Q >> 32));                 // dropped bits of r/n, 0..11
    const uint32_t lo = (uint32_t)Q;
    const uint32_t half = (1u << sh) >> 1;
    // sh > 0: above half, or half with more below it (R) or an odd last bit;
    // sh = 0: the remainder alone decides
    const uint64_t r2 = 2 * (uint64_t)R;
    const uint32_t up0 = (r2 > n || (r2 == n && (lo & 1u))) ? 1u : 0u;
    const uint32_t bias = sh ? half - 1u + ((R != 0 || ((lo >> sh) & 1u)) ? 1u : 0u) : up0;
    uint64_t q = Q + bias;
    q &= ~(uint64_t)((1u << sh) - 1u);
    const uint64_t s = q + D;
    const bool wrap = s < q;                                             // u + shift >= 1
    const int sh2 = wrap ? 12 : 11 - __clz((int)(uint32_t)(s >> 32));    // s >= 2^52 without a wrap
    const uint32_t half2 = (1u << sh2) >> 1;
    const uint32_t bias2 = sh2 ? half2 - 1u + (((uint32_t)s >> sh2) & 1u) : 0u;
    return (s + bias2) & ~(uint64_t)((1u << sh2) - 1u);                  // a carry out leaves 0
}

// The lattice coordinate u as the smaller of u and 1 - u (y: normalised
// mantissa and exponent, m = 0 for u = 0; Y = y 2^64) and the larger one
// (big 2^-64 >= 1/2)
struct FxCoord {
    FxM y;
    uint64_t Y, big;
    bool lower;   // u < 1/2: u is y
};
// of the walk's state `st` (low, high word of Q; r; R), which then takes one
// step k -> k + 1 and goes to `next`
__device__ __forceinline__ FxCoord fx_next(uint4 st, uint32_t z, uint64_t qz, uint32_t rz, uint32_t n, double inv_n,
                                           double delta, uint64_t D, uint4 *next) {
    LatticeWalk lw;
    lw.Q = ((uint64_t)st.y << 32) | st.x;
    lw.r = st.z;
    lw.R = st.w;
    FxCoord c;
    uint64_t U;
    int e = 0;
    uint64_t M = 0;
    if (st.y >= (1u << 20)) {
        U = fx_coord(lw.Q, lw.R, n, D);
    } else {                                            // r/n < 2^-12: one in 4096
        const double u = lattice_coord(lw.r, (double)n, inv_n, delta);
        const uint64_t b = (uint64_t)__double_as_longlong(u);
        e = (int)(b >> 52) - 1023;
        M = b ? ((b & 0x000FFFFFFFFFFFFFULL) | (1ULL << 52)) << 11 : 0;
        U = e >= -64 ? M >> (-1 - e) : 0;               // exact for u >= 2^-11
        if (e >= -11) M = 0;
    }
    walk_step(lw, z, qz, rz, n);
    *next = make_uint4((uint32_t)lw.Q, (uint32_t)(lw.Q >> 32), lw.r, lw.R);
    c.lower = U < (1ULL << 63);
    c.Y = c.lower ? U : 0 - U;
    c.big = c.lower ? (U ? 0 - U : ~0ULL) : U;
    c.y = fx_norm(FxM{c.Y, -1});
    if (c.Y == 0) c.y.m = 0;                            // (the shift by 64 is undefined)
    if (M) c.y = FxM{M, e};
    return c;
}

// korobov3 of the smaller of u and 1 - u, y <= 1/2: s = y^4 (35 - 84y + 70y^2
// - 20y^3), the smaller of t and 1 - t (phi(1 - u) = 1 - phi(u)); P by Horner
// in Q57 (P >= 8). Relative error below 2^-58.
__device__ __forceinline__ FxM fx_korobov(const FxCoord &u) {
    // 20 y in Q57, rounded down
    const uint32_t ylo = (uint32_t)u.Y;
    const uint64_t y20 = (u.Y >> 3) + (u.Y >> 5) + ((((ylo & 7u) << 2) + (ylo & 31u)) >> 5);
    const uint64_t a1 = (70ULL << 57) - y20;
    const uint64_t a2 = (84ULL << 57) - __umul64hi(u.Y, a1);
    const uint64_t P = (35ULL << 57) - __umul64hi(u.Y, a2);
    const uint64_t p2 = __umul64hi(u.y.m, u.y.m);       // y^2 = p2 2^(2e - 62)
    const uint64_t p4 = __umul64hi(p2, p2);             // y^4 = p4 2^(4e - 60)
    const uint64_t hi = __umul64hi(p4, P), lo = p4 * P;
    const int c = __clzll((long long)hi);               // hi >= 2^56
    return FxM{(hi << c) | ((lo >> 1) >> (63 - c)), 10 - c + 4 * u.y.e};
}
// korobov3 of u in the general kernel's roundings (korobov_phi_fix: P by
// Horner on the smaller of u and 1 - u), the bits below the mantissa or-ed
// into its last one, so that it rounds to the same FP64 value
__device__ __forceinline__ FxM fx_korobov_ex(const FxCoord &u) {
    const uint64_t sm = u.lower ? ~0ULL : 0ULL;
    const uint64_t y = u.lower ? u.Y >> 2 : u.Y;
    const uint32_t ylo = (uint32_t)y;
    const uint64_t y20 = (y >> 1) + (y >> 3) + ((((ylo & 1u) << 2) + (ylo & 7u)) >> 3);   // 20 Y in Q57 / Q59
    const uint64_t a1 = (u.lower ? 70ULL << 57 : 10ULL << 59) + ((y20 ^ sm) - sm);
    const uint64_t a2 = (u.lower ? 84ULL << 57 : 4ULL << 59) + ((__umul64hi(u.Y, a1) ^ sm) - sm);
    const uint64_t P = (u.lower ? 35ULL << 57 : 1ULL << 59) + ((__umul64hi(u.Y, a2) ^ sm) - sm);
    const uint64_t M = u.lower ? u.y.m : u.big;
    const int e = u.lower ? u.y.e : -1;
    const uint64_t p2 = __umul64hi(M, M);
    const uint64_t p4 = __umul64hi(p2, p2);
    const uint64_t hi = __umul64hi(p4, P), lo = p4 * P;
    const int c = __clzll((long long)hi);
    return FxM{(hi << c) | ((lo >> 1) >> (63 - c)) | ((lo << c) ? 1ULL : 0ULL), 67 - c + 4 * e - (u.lower ? 57 : 59)};
}
// 1 - s for 0 < s <= 1/2 (2^-64 below 1 where s < 2^-64)
__device__ __forceinline__ FxM fx_one_minus(FxM s) {
    const uint64_t S = s.e >= -64 ? s.m >> (-1 - s.e) : 0;
    return FxM{S ? 0 - S : ~0ULL, -1};
}

// RN of a normalised mantissa in the normal range
__device__ __forceinline__ double fx_pack(FxM a) {
    uint64_t mant = a.m >> 11;
    const uint32_t low = (uint32_t)a.m & 0x7FFu;
    mant += (low > 0x400u || (low == 0x400u && (mant & 1))) ? 1 : 0;
    return __longlong_as_double((long long)(((uint64_t)(1023 + a.e - 1) << 52) + mant));
}
// x / 2 (0 below the normal range)
__device__ __forceinline__ double fx_half(double x) {
    const int h = __double2hiint(x);
    return (h & 0x7FF00000) > 0x00200000 ? __hiloint2double(h - 0x00100000, __double2loint(x)) : 0.0;
}

// One group's sum of monomials [m0, m1): out of line, one copy for every
// group of both polynomials. FP32 products in the order of the table for the
// mixed precision.
// EX: the sum in FP64, in the general kernel's order (its bits).
template <int DMAX, int BLOCK, bool MIXED, bool EX>
__device__ __noinline__ uint64_t fx_group(int m0, int m1, int sh) {
    const FxShared &S = fx_shared();
    if constexpr (MIXED) {
        const unsigned char *pt = fx_pt<DMAX, BLOCK>(4);
        auto ld = [&](uint32_t off) { return *reinterpret_cast<const float *>(pt + 4 * off); };
        float s = 0.0f;
        for (int m = m0; m < m1; ++m) {
            const uint4 D = S.mdesc[m];
            const float c = __uint_as_float((uint32_t)S.cfix[m]);
            if (D.w == 0) {
                s = m == m0 ? c : __fadd_rn(s, c);
                continue;
            }
            float v = ld(D.x & 0xFFFFu);
            if (D.w > 1) {
                v = __fmul_rn(v, ld(D.x >> 16));
                if (D.w > 2) {
                    v = __fmul_rn(v, ld(D.y & 0xFFFFu));
                    if (D.w > 3) {
                        v = __fmul_rn(v, ld(D.y >> 16));
                        if (D.w > 4) v = __fmul_rn(v, ld(D.z & 0xFFFFu));
                        if (D.w > 5) v = __fmul_rn(v, ld(D.z >> 16));
                    }
                }
            }
            s = m == m0 ? __fmul_rn(v, c) : __fmaf_rn(v, c, s);
        }
        if constexpr (EX) return (uint64_t)__double_as_longlong((double)s);
        // s 2^sh (s >= 0), rounded
        const uint32_t b = __float_as_uint(s);
        const uint64_t mant = (b & 0x7FFFFFu) | (b >= 0x800000u ? 0x800000u : 0u);
        const int x = (int)(b >> 23) - 150 + sh;
        return x >= 0 ? mant << x : (x > -26 ? (mant + (1ULL << (-x - 1))) >> -x : 0);
    } else if constexpr (EX) {
        const unsigned char *pt = fx_pt<DMAX, BLOCK>(8);
        auto ld = [&](uint32_t off) { return *reinterpret_cast<const double *>(pt + 4 * off); };
        double s = 0.0;
        for (int m = m0; m < m1; ++m) {
            const uint4 D = S.mdesc[m];
            const double c = __longlong_as_double((long long)S.cfix[m]);
            if (D.w == 0) {
                s = m == m0 ? c : __dadd_rn(s, c);
                continue;
            }
            double v = ld(D.x & 0xFFFFu);
            if (D.w > 1) {
                v = fma(v, ld(D.x >> 16), S.nzero);
                if (D.w > 2) {
                    v = fma(v, ld(D.y & 0xFFFFu), S.nzero);
                    if (D.w > 3) {
                        v = fma(v, ld(D.y >> 16), S.nzero);
                        if (D.w > 4) v = fma(v, ld(D.z & 0xFFFFu), S.nzero);
                        if (D.w > 5) v = fma(v, ld(D.z >> 16), S.nzero);
                    }
                }
            }
            s = fma(v, c, m == m0 ? S.nzero : s);
        }
        return (uint64_t)__double_as_longlong(s);
    } else {
        const unsigned char *pt = fx_pt<DMAX, BLOCK>(8);
        auto ld = [&](uint32_t off) { return *reinterpret_cast<const uint64_t *>(pt + 4 * off); };
        uint64_t s = (uint64_t)(m1 - m0) >> 1;      // the mean of the truncations below
        for (int m = m0; m < m1; ++m) {
            const uint4 D = S.mdesc[m];
            const uint64_t c = S.cfix[m];
            if (D.w == 0) {
                s += c;
                continue;
            }
            uint64_t v = ld(D.x & 0xFFFFu);
            if (D.w > 1) {
                v = __umul64hi(v, ld(D.x >> 16));
                if (D.w > 2) {
                    v = __umul64hi(v, ld(D.y & 0xFFFFu));
                    if (D.w > 3) {
                        v = __umul64hi(v, ld(D.y >> 16));
                        if (D.w > 4) v = __umul64hi(v, ld(D.z & 0xFFFFu));
                        if (D.w > 5) v = __umul64hi(v, ld(D.z >> 16));
                    }
                }
            }
            s += __umul64hi(v, c);
        }
        return s;
    }
}

// One corner: B = Cc U^u0 F^f0 rounded once and, with `lam`, the logarithm of
// U^u1 F^f1 (plus Lc). U, F are the fixed-point corner values (> 0). Out of
// line: up to sixteen call sites per tile path.
struct FxCorner {
    double B, L;
};
// x^k from x and 1/x, 1 <= |k| <= 4; each product drops at most one bit of the mantissa
__device__ __forceinline__ FxM fx_pow(FxM x, FxM r, int k) {
    const FxM b = k < 0 ? r : x;
    const int a = k < 0 ? -k : k;
    FxM p = b;
    if (a > 1) {
        p = fx_mul(b, b);
        if (a == 3) p = fx_mul(p, b);
        if (a == 4) p = fx_mul(p, p);
    }
    return p;
}
__device__ __noinline__ FxCorner fx_corner(uint64_t U, uint64_t F, FxM Cc, double Lc, bool lam) {
    const FxShared &S = fx_shared();
    const uint32_t ex = S.ex;
    const int u0 = (int8_t)ex, f0 = (int8_t)(ex >> 8), u1 = (int8_t)(ex >> 16), f1 = (int8_t)(ex >> 24);
    const FxM u = fx_norm(FxM{U, 63 - S.sh[0]}), f = fx_norm(FxM{F, 63 - S.sh[1]});
    FxM ru = u, rf = f;
    if (u0 < 0 || (lam && u1 < 0)) {
        const qmc_xf r = qmc_xf_rcp3(qmc_xf{u.m, u.e, 0});
        ru = FxM{r.m, r.e};
    }
    if (f0 < 0 || (lam && f1 < 0)) {
        const qmc_xf r = qmc_xf_rcp3(qmc_xf{f.m, f.e, 0});
        rf = FxM{r.m, r.e};
    }
    FxCorner out{1.0, 0.0};
    FxM b{1ULL << 63, 0};
    if (f0) b = fx_pow(f, rf, f0);
    if (u0) b = f0 ? fx_mul(b, fx_pow(u, ru, u0)) : fx_pow(u, ru, u0);
    if (S.hasC) b = fx_mul(b, Cc);
    b = fx_norm(b);
    out.B = qmc_xf_to_double(qmc_xf{b.m, b.e, 0});
    if (lam) {
        FxM x{1ULL << 63, 0};
        if (f1) x = fx_pow(f, rf, f1);
        if (u1) x = f1 ? fx_mul(x, fx_pow(u, ru, u1)) : fx_pow(u, ru, u1);
        x = fx_norm(x);
        out.L = qmc_ilog_xf(qmc_xf{x.m, x.e, 0}, S.logtab);
        if (S.hasL) out.L += Lc;
    }
    return out;
}

// The same for the EX sectors: FP64 values of U and F (positive), and the
// products of qmc_xf_mul in the order of corner_xf
__device__ __forceinline__ FxM fx_mulx(FxM a, FxM b) {
    const uint64_t h = __umul64hi(a.m, b.m);
    const int top = (int)(h >> 63);
    return FxM{top ? h : h << 1, a.e + b.e + top};
}
// x^k0 and x^k1 by repeated products of x or 1/x
__device__ __forceinline__ void fx_powx(FxM x, FxM r, int k0, int k1, FxM &p0, FxM &p1) {
    p0 = p1 = FxM{1ULL << 63, 0};
    const int n = max(max(k0, k1), 0), m = max(max(-k0, -k1), 0);
    FxM p = x;
    for (int i = 1; i <= n; ++i) {
        if (i > 1) p = fx_mulx(p, x);
        if (i == k0) p0 = p;
        if (i == k1) p1 = p;
    }
    p = r;
    for (int i = 1; i <= m; ++i) {
        if (i > 1) p = fx_mulx(p, r);
        if (i == -k0) p0 = p;
        if (i == -k1) p1 = p;
    }
}
__device__ __forceinline__ FxM fx_of(double x) {
    const qmc_xf a = qmc_xf_of(x);
    return FxM{a.m, a.e};
}
__device__ __noinline__ FxCorner fx_corner_ex(double U, double F, double Cc, double Lc, bool lam) {
    const FxShared &S = fx_shared();
    const uint32_t ex = S.ex;
    const int u0 = (int8_t)ex, f0 = (int8_t)(ex >> 8), u1 = (int8_t)(ex >> 16), f1 = (int8_t)(ex >> 24);
    const FxM u = fx_of(U), f = fx_of(F);
    FxM ru = u, rf = f;
    if (u0 < 0 || (lam && u1 < 0)) {
        const qmc_xf r = qmc_xf_rcp(qmc_xf{u.m, u.e, 0});
        ru = FxM{r.m, r.e};
    }
    if (f0 < 0 || (lam && f1 < 0)) {
        const qmc_xf r = qmc_xf_rcp(qmc_xf{f.m, f.e, 0});
        rf = FxM{r.m, r.e};
    }
    FxM pu0, pu1, pf0, pf1;
    fx_powx(u, ru, u0, lam ? u1 : 0, pu0, pu1);
    fx_powx(f, rf, f0, lam ? f1 : 0, pf0, pf1);
    const FxM b = fx_mulx(S.hasC ? fx_of(Cc) : FxM{1ULL << 63, 0}, fx_mulx(pu0, pf0));
    FxCorner out{qmc_xf_to_double(qmc_xf{b.m, b.e, 0}), 0.0};
    if (lam) {
        const FxM x = fx_mulx(pu1, pf1);
        out.L = qmc_ilog_xf(qmc_xf{x.m, x.e, 0}, S.logtab);
        if (S.hasL) out.L += Lc;
    }
    return out;
}
// Their subset sums over the singular variables, of non-negative FP64 values
// (subset_sums_xf without signs), rounded to FP64 in place
template <int NS> __device__ __noinline__ void fx_subset_ex(double *h) {
    constexpr int NG = 1 << NS;
    FxM x[NG];
#pragma unroll
    for (int g = 0; g < NG; ++g) x[g] = fx_of(h[g]);
#pragma unroll
    for (int q = 0; q < NS; ++q)
#pragma unroll
        for (int g = 0; g < NG; ++g)
            if (g & (1 << q)) {
                const FxM a = x[g], b = x[g ^ (1 << q)];
                const bool sw = b.e > a.e;
                const uint64_t big = sw ? b.m : a.m, small = sw ? a.m : b.m;
                const int e = sw ? b.e : a.e, d = sw ? b.e - a.e : a.e - b.e;
                const uint64_t s = big + (d < 64 ? small >> d : 0ULL);
                const bool c = s < big;
                x[g] = FxM{c ? (s >> 1) | (1ULL << 63) : s, e + (c ? 1 : 0)};
            }
#pragma unroll
    for (int g = 0; g < NG; ++g) h[g] = qmc_xf_to_double(qmc_xf{x[g].m, x[g].e, 0});
}

// Depth-first fold over the singular variables (see the top): out receives
// the orders eps^-Q .. eps^(|V| + HI), V the corner bits at and above Q and
// eps^HI the last order of the sums.
template <int NS, int HI> struct FxFold {
    const double (&B)[1 << NS];   // corner values and exponents
    const double (&L)[1 << NS];
    const double (&h)[SlotArr<NS>::N][NS + HI + 1];   // (b/t) (b ln t)^j / j! per slot
    double mone, nzero;

    template <int Q, int V>
    __device__ __forceinline__ void run(double (&out)[Q + __builtin_popcount(V) + HI + 1]) const {
        constexpr int pv = __builtin_popcount(V);
        if constexpr (Q == 0) {
            // B L^i / i!
            constexpr int N = pv + HI;
            const double l = N > 0 ? L[V] : 0.0;
            out[0] = B[V];
            if constexpr (N >= 1) out[1] = fma(out[0], l, nzero);
            if constexpr (N >= 2) out[2] = fma(out[1], fx_half(l), nzero);
            if constexpr (N >= 3) out[3] = fma(out[2], l * (1.0 / 3), nzero);
            if constexpr (N >= 4) out[4] = fma(out[3], fx_half(fx_half(l)), nzero);
        } else {
            constexpr int n = Q + pv + HI;
            double a[n], b[n + 1];
            run<Q - 1, V>(a);
            run<Q - 1, V | (1 << (Q - 1))>(b);
            out[0] = b[0];
#pragma unroll
            for (int k = 0; k < n; ++k) {
                a[k] = fma(b[k], mone, a[k]);
                double s = b[k + 1];
#pragma unroll
                for (int i = 0; i <= k; ++i) s = fma(h[Q - 1][k - i], a[i], s);
                out[k + 1] = s;
            }
        }
    }
};

// EX: the fold over the Moebius-transformed corner series D (series_fp64 and
// moebius_fp64 of the general kernel):
//   S(Q, P) = (b/t) e^{eps b ln t} S(Q-1, P) + S(Q-1, P + q) / eps
template <int NS, int HI> struct FxFoldD {
    const double (&D)[1 << NS][NS + HI + 1];
    const double (&h)[SlotArr<NS>::N][NS + HI + 1];

    template <int Q, int P>
    __device__ __forceinline__ void run(double (&out)[Q + __builtin_popcount(P) + HI + 1]) const {
        constexpr int n = Q + __builtin_popcount(P) + HI;
        if constexpr (Q == 0) {
#pragma unroll
            for (int i = 0; i <= n; ++i) out[i] = D[P][i];
        } else {
            double a[n], b[n + 1];
            run<Q - 1, P>(a);
            run<Q - 1, P | (1 << (Q - 1))>(b);
            out[0] = b[0];
#pragma unroll
            for (int k = 0; k < n; ++k) {
                double s = b[k + 1];
#pragma unroll
                for (int i = 0; i <= k; ++i) s = fma(h[Q - 1][k - i], a[i], s);
                out[k + 1] = s;
            }
        }
    }
};

// The thread's points [k0, kend) of the tile: acc[o] is the sum of W f_o,
// order eps^(lo + o).
template <int DMAX, int BLOCK, int NS, int HI, bool MIXED, int LMAX>
__device__ __forceinline__ void fx_points(const QmcLaunch &Lc, uint64_t k0, uint64_t kend, int lo, int nord,
                                          double (&acc)[LMAX]) {
    constexpr int NSA = SlotArr<NS>::N;
    constexpr int NG = 1 << NS;
    constexpr bool EX = NS >= 3;              // the general kernel's roundings (see the top)
    constexpr bool P64 = !MIXED && EX;        // FP64 monomials
    const FxShared &S = fx_shared();
    const int d = S.d;
    const uint64_t n = S.job.n;
    const uint32_t n32 = (uint32_t)n;
    uint4 *const walk = fx_walk<DMAX, BLOCK>();
    unsigned char *const pt = fx_pt<DMAX, BLOCK>(MIXED ? 4 : 8);
    {
        const uint64_t minv = S.minv;
#pragma unroll 1
        for (int i = 0; i < d; ++i) {
            uint64_t r0, Q, R;
            fx_divmod(k0 * (uint64_t)S.zmod[i], n, minv, r0);
            fx_fixdiv(r0, n, minv, Q, R);
            walk[i * BLOCK] = make_uint4((uint32_t)Q, (uint32_t)(Q >> 32), (uint32_t)r0, (uint32_t)R);
        }
    }
    constexpr int NO = NS + HI + 1;
    double accN[NO];
#pragma unroll
    for (int i = 0; i < NO; ++i) accN[i] = 0.0;
#pragma unroll 1
    for (uint64_t k = k0; k < kend; ++k) {
        FxM w{1ULL << 63, 0}, Cc{1ULL << 63, 0};
        double Lr = 0.0;
        double hb[NSA], bl[NSA];
        bool zero = false;
#pragma unroll 1
        for (int i = 0; i < d; ++i) {
            const uint4 st = walk[i * BLOCK];
            const FxCoord u = fx_next(st, S.zmod[i], S.qz[i], S.rz[i], n32, S.job.inv_n, S.delta[i], S.dfix[i],
                                      walk + i * BLOCK);
            if (u.y.m == 0) {                           // u = 0: the point contributes 0
                zero = true;
                continue;
            }
            FxM t;
            if (Lc.transform == 0) {
                if constexpr (EX) {
                    t = fx_korobov_ex(u);
                } else {
                    const FxM s = fx_korobov(u);
                    t = u.lower ? s : fx_one_minus(s);
                }
                // the weight: prod u (1 - u), cubed below
                w = fx_norm(fx_mul(w, FxM{__umul64hi(u.y.m, u.big), u.y.e}));
            } else if (Lc.transform == 1) {             // baker: 1 - |2u - 1|
                t = FxM{u.y.m, u.y.e + 1};
            } else {
                t = u.lower ? u.y : FxM{u.big, -1};
            }
            // powers of t for the polynomials
            if constexpr (MIXED) {
                float *p = reinterpret_cast<float *>(pt) + Lc.prow * i * BLOCK;
                // RN to 24 bits (t >= 2^-126 or 0)
                const uint32_t hw = (uint32_t)(t.m >> 32);
                uint32_t q = hw >> 8;
                const uint32_t rest = hw & 0xFFu;
                q += (rest > 0x80u || (rest == 0x80u && ((uint32_t)t.m != 0 || (q & 1u)))) ? 1u : 0u;
                const float x1 = t.e > -126 ? __uint_as_float(((uint32_t)(t.e + 126) << 23) + q) : 0.0f;
                p[0] = x1;
                if (Lc.prow >= 2) {
                    const float x2 = __fmul_rn(x1, x1);
                    p[BLOCK] = x2;
                    if (Lc.prow >= 3) p[2 * BLOCK] = __fmul_rn(x2, x1);
                    if (Lc.prow >= 4) p[3 * BLOCK] = __fmul_rn(x2, x2);
                }
            } else if constexpr (P64) {
                double *p = reinterpret_cast<double *>(pt) + Lc.prow * i * BLOCK;
                const double x1 = fx_pack(t);
                p[0] = x1;
                if (Lc.prow >= 2) {
                    const double x2 = x1 * x1;
                    p[BLOCK] = x2;
                    if (Lc.prow >= 3) p[2 * BLOCK] = x2 * x1;
                    if (Lc.prow >= 4) p[3 * BLOCK] = x2 * x2;
                }
            } else {
                uint64_t *p = reinterpret_cast<uint64_t *>(pt) + Lc.prow * i * BLOCK;
                const uint64_t x1 = t.e >= 0 ? ~0ULL : (t.e >= -64 ? t.m >> (-1 - t.e) : 0);
                p[0] = x1;
                if (Lc.prow >= 2) {
                    const uint64_t x2 = __umul64hi(x1, x1);
                    p[BLOCK] = x2;
                    if (Lc.prow >= 3) p[2 * BLOCK] = __umul64hi(x2, x1);
                    if (Lc.prow >= 4) p[3 * BLOCK] = __umul64hi(x2, x2);
                }
            }
            // 1/t and ln t of the singular variables; factors of the regular ones
            const bool reg = (S.regular >> i) & 1;
            if (i < NS || reg) {
                double l = 0.0;
                if (NS + HI > 1 || (NS + HI > 0 && reg)) l = qmc_ilog_core(t.e, t.m & 0x7FFFFFFFFFFFFFFFULL, S.logtab);
                if (i < NS) {
                    const qmc_xf r = qmc_xf_rcp3(qmc_xf{t.m, t.e, 0});
                    hb[i] = S.bvar[i] * fx_pack(FxM{r.m, r.e});
                    bl[i] = S.bvar[i] * l;
                } else {
                    const int a = S.avar[i];
                    if (a > 0) Cc = fx_norm(fx_mul(Cc, fx_pow(t, t, a)));
                    Lr = fma(S.bvar[i], l, Lr);
                }
            }
        }
        if (zero) continue;
        double W = 1.0;
        if (Lc.transform == 0) W = fx_pack(fx_norm(fx_mul(fx_mul(w, w), w)));
        // the polynomials: group sums, then subset sums over the singular
        // variables; the value at corner V (t_V = 0) is h[(NG-1) ^ V]
        double B[NG], L[NG];
        if constexpr (EX) {
            double hU[NG], hF[NG];
#pragma unroll 1
            for (int g = 0; g < NG; ++g) {
                const int u0 = S.gs[0][g], u1 = S.gs[0][g + 1], f0 = S.gs[1][g], f1 = S.gs[1][g + 1];
                hU[g] = 0.0;
                hF[g] = 0.0;
                if (u1 > u0) hU[g] = __longlong_as_double((long long)fx_group<DMAX, BLOCK, MIXED, EX>(u0, u1, 0));
                if (f1 > f0) hF[g] = __longlong_as_double((long long)fx_group<DMAX, BLOCK, MIXED, EX>(f0, f1, 0));
            }
            fx_subset_ex<NS>(hU);
            fx_subset_ex<NS>(hF);
            // (a product of t^a may lie below the normal range)
            const double Cd = S.hasC ? qmc_xf_to_double(qmc_xf{Cc.m, Cc.e, 0}) : 1.0;
#pragma unroll 1
            for (int V = 0; V < NG; ++V) {
                const FxCorner c = fx_corner_ex(hU[(NG - 1) ^ V], hF[(NG - 1) ^ V], Cd, Lr, HI > 0 || V != 0);
                B[V] = c.B;
                L[V] = c.L;
            }
        } else {
            uint64_t hU[NG], hF[NG];
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int u0 = S.gs[0][g], u1 = S.gs[0][g + 1], f0 = S.gs[1][g], f1 = S.gs[1][g + 1];
                hU[g] = 0;
                hF[g] = 0;
                if (u1 > u0) hU[g] = fx_group<DMAX, BLOCK, MIXED, EX>(u0, u1, S.sh[0]);
                if (f1 > f0) hF[g] = fx_group<DMAX, BLOCK, MIXED, EX>(f0, f1, S.sh[1]);
            }
#pragma unroll
            for (int q = 0; q < NS; ++q)
#pragma unroll
                for (int g = 0; g < NG; ++g)
                    if (g & (1 << q)) {
                        hU[g] += hU[g ^ (1 << q)];
                        hF[g] += hF[g ^ (1 << q)];
                    }
#pragma unroll 1
            for (int V = 0; V < NG; ++V) {
                const FxCorner c = fx_corner(hU[(NG - 1) ^ V], hF[(NG - 1) ^ V], Cc, Lr, HI > 0 || V != 0);
                B[V] = c.B;
                L[V] = c.L;
            }
        }
        double h[NSA][NO];
        const double mone = S.mone, nzero = S.nzero;
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            h[q][0] = hb[q];
            if constexpr (NS + HI > 1) h[q][1] = fma(hb[q], bl[q], nzero);
            if constexpr (NS + HI > 2) h[q][2] = fma(h[q][1], fx_half(bl[q]), nzero);
            if constexpr (NS + HI > 3) h[q][3] = fma(h[q][2], bl[q] * (1.0 / 3), nzero);
        }
        double res[NO];
        if constexpr (EX) {
            double D[NG][NO];
            series_fp64<NS, HI>(B, L, D);
            moebius_fp64<NS, HI>(D);
            FxFoldD<NS, HI>{D, h}.template run<NS, 0>(res);
        } else {
            FxFold<NS, HI>{B, L, h, mone, nzero}.template run<NS, 0>(res);
        }
#pragma unroll
        for (int i = 0; i < NO; ++i) accN[i] = fma(res[i], W, accN[i]);
    }
    // output order o is eps^(lo+o), i.e. index lo + o + NS of accN
#pragma unroll
    for (int o = 0; o < LMAX; ++o) {
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < NO; ++i)
            if (i == lo + o + NS) v = accN[i];
        if (o < nord) acc[o] = v;
    }
}

// Stage the sector of S.job at its kinematic point (all threads)
template <int BLOCK, bool MIXED>
__device__ __forceinline__ void fx_stage(FxShared &S, const QmcLaunch &Lc) {
    const int sidx = S.job.sector, pidx = S.job.point;
    if (sidx == S.cached_sector && pidx == S.cached_point) return;
    const QmcSectorDev *src = Lc.sectors + sidx;
    const int d = src->d, ns = src->ns, nU = src->nU, nm = nU + src->nF;
    if (threadIdx.x < 2) {
        S.emax[threadIdx.x] = -4096;
        S.csum[threadIdx.x] = 0;
    }
    __syncthreads();
    int slot[QMC_DMAX];
    int singmask = 0;
    {
        for (int q = 0; q < ns; ++q) singmask |= 1 << src->sing[q];
        int next = ns;
#pragma unroll
        for (int j = 0; j < QMC_DMAX; ++j) {
            slot[j] = next;
            if ((singmask >> j) & 1) {
                for (int q = 0; q < ns; ++q)
                    if (src->sing[q] == j) slot[j] = q;
            } else {
                ++next;
            }
        }
    }
    const double *kin = Lc.kin + (size_t)pidx * Lc.ninv;
    for (int m = threadIdx.x; m < nm; m += BLOCK) {
        const QmcMono &Mo = Lc.monos[src->monoU + m];
        double v = Mo.coef[0];
        for (int i = 0; i < Lc.ninv && i + 1 < QMC_NCOEF; ++i) v = fma(Mo.coef[i + 1], kin[i], v);
        // v >= 0 here, but -0.0 too: without its sign, which would read as an exponent bit
        const uint64_t vb = (uint64_t)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFULL;
        S.cfix[m] = vb;
        atomicMax(&S.emax[m < nU ? 0 : 1], (int)(vb >> 52) - 1023);
        uint32_t off[6] = {0, 0, 0, 0, 0, 0};
        uint32_t k = 0;
#pragma unroll
        for (int j = 0; j < QMC_DMAX; ++j) {
            const uint32_t ej = (Mo.exps >> (4 * j)) & 15u;
            if (ej) {
                const uint32_t o = (uint32_t)(Lc.prow * slot[j] + (int)ej - 1) * (BLOCK * (MIXED ? 1 : 2));
#pragma unroll
                for (int i = 0; i < 6; ++i)
                    if (i == (int)k) off[i] = o;
                ++k;
            }
        }
        S.mdesc[m] = make_uint4(off[0] | (off[1] << 16), off[2] | (off[3] << 16), off[4] | (off[5] << 16), k);
    }
    if (threadIdx.x <= QMC_NGROUP) {
        S.gs[0][threadIdx.x] = src->gU[threadIdx.x];
        S.gs[1][threadIdx.x] = nU + src->gF[threadIdx.x];
    }
    if (threadIdx.x >= 32 && threadIdx.x < 32 + QMC_DMAX) {
        const int j = (int)threadIdx.x - 32;
        int sl = 0;
#pragma unroll
        for (int i = 0; i < QMC_DMAX; ++i)
            if (i == j) sl = slot[i];
        if (sl < QMC_DMAX) {
            S.perm[sl] = j;
            S.avar[sl] = src->a[j];
            S.bvar[sl] = src->b[j];
        }
    }
    if (threadIdx.x == 64) {
        S.d = d;
        S.ns = ns;
        S.ex = ((uint32_t)(int)src->u0 & 255u) | (((uint32_t)(int)src->f0 & 255u) << 8) |
               (((uint32_t)src->u1i & 255u) << 16) | (((uint32_t)src->f1i & 255u) << 24);
        int reg = 0, hasC = 0, hasL = 0;
        for (int j = 0; j < d; ++j)
            if ((src->regular_mask >> j) & 1) {
                int sl = 0;
#pragma unroll
                for (int i = 0; i < QMC_DMAX; ++i)
                    if (i == j) sl = slot[i];
                reg |= 1 << sl;
                hasC |= src->a[j] > 0;
                hasL |= src->b[j] != 0.0;
            }
        S.regular = reg;
        S.hasC = hasC;
        S.hasL = hasL;
        double w = src->weight_b;
        if (Lc.transform == 0)
            for (int j = 0; j < d; ++j) w *= 140.0;
        S.w = w;
        S.cached_sector = sidx;
        S.cached_point = pidx;
    }
    __syncthreads();
    // the scale: the coefficients' sum, taken in units of 2^(emax - 16) and
    // rounded up with 2^-10 to spare, times 2^sh stays below 2^64
    for (int m = threadIdx.x; m < nm; m += BLOCK) {
        const int p = m < nU ? 0 : 1;
        const uint64_t b = S.cfix[m];
        const int be = (int)(b >> 52), x = S.emax[p] + 1023 + 36 - be;       // c = mant 2^(be - 1075)
        const uint64_t mant = (b & 0x000FFFFFFFFFFFFFULL) | (be ? 1ULL << 52 : 0);
        if (mant) atomicAdd(&S.csum[p], (x < 64 ? (int)(mant >> x) : 0) + 1);
    }
    __syncthreads();
    int sh[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int c = S.csum[p];
        sh[p] = 80 - (32 - __clz(c + (c >> 10) + 1)) - S.emax[p];
        if (threadIdx.x == 0) S.sh[p] = sh[p];
    }
    for (int m = threadIdx.x; m < nm; m += BLOCK) {
        const uint64_t b = S.cfix[m];
        if constexpr (MIXED) {
            S.cfix[m] = __float_as_uint((float)__longlong_as_double((long long)b));
        } else if (ns < 3) {                     // (three and more: the double itself)
            const int be = (int)(b >> 52);
            const uint64_t mant = (b & 0x000FFFFFFFFFFFFFULL) | (be ? 1ULL << 52 : 0);
            const int x = be - 1075 + sh[m < nU ? 0 : 1];            // c 2^sh = mant 2^x
            S.cfix[m] = x >= 0 ? mant << x : (x > -55 ? (mant + (1ULL << (-x - 1))) >> -x : 0);
        }
    }
}

// Resident 128-thread units the registers must allow: d <= 3, d <= 6
#ifndef QMC_FX_MINB
#define QMC_FX_MINB 8
#endif
#ifndef QMC_FX6_MINB
#define QMC_FX6_MINB 6
#endif
template <int DMAX, int SMAX, int LMAX, bool MIXED, int BLOCK, int HI>
__global__ void __launch_bounds__(BLOCK, (DMAX > 3 ? QMC_FX6_MINB : QMC_FX_MINB) * 128 / BLOCK) qmc_real_kernel(QmcLaunch Lc, int ppt) {
    FxShared &S = fx_shared();
    const int lo = Lc.lo, nord = Lc.norders;
    if (threadIdx.x == 0) {
        S.cached_sector = -1;
        S.cached_point = -1;
        S.mone = Lc.mone;
        S.nzero = Lc.nzero;
    }
    for (int i = threadIdx.x; i < 3 * QMC_LOG_TABLE_ROWS; i += BLOCK) S.logtab[i] = kLogTable[i];
    for (;;) {
        __syncthreads();  // previous tile fully consumed
        if (threadIdx.x == 0) {
            const unsigned long long tile = atomicAdd(Lc.queue, 1ULL);
            S.tile = tile;
            if (tile < Lc.ntiles) {
                // last job with tile_begin <= tile
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
        fx_stage<BLOCK, MIXED>(S, Lc);
        const uint64_t local = tile - S.job.tile_begin;
        const uint64_t s = local / (uint64_t)S.job.tiles_per_shift;
        const uint64_t chunk = local - s * (uint64_t)S.job.tiles_per_shift;
        if (threadIdx.x < QMC_DMAX && (int)threadIdx.x < S.d) {
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
            if (i == 0) S.minv = minv;
        }
        __syncthreads();

        double acc[LMAX];
#pragma unroll
        for (int o = 0; o < LMAX; ++o) acc[o] = 0.0;
        const uint64_t kt0 = chunk * (uint64_t)Lc.tile_k;
        const uint64_t kt1 = min(S.job.n, kt0 + (uint64_t)Lc.tile_k);
        const uint64_t k0 = kt0 + (uint64_t)threadIdx.x * (uint64_t)ppt;
        if (k0 < kt1) {
            const uint64_t kend = min(kt1, k0 + (uint64_t)ppt);
            const int ns = S.ns;
            if (ns == 0) fx_points<DMAX, BLOCK, 0, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc);
            else if (ns == 1) fx_points<DMAX, BLOCK, 1, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc);
            else if (ns == 2 || SMAX < 3) fx_points<DMAX, BLOCK, 2, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc);
            else if constexpr (SMAX >= 3) {
                if (ns == 3) fx_points<DMAX, BLOCK, 3, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc);
                else fx_points<DMAX, BLOCK, 4, HI, MIXED, LMAX>(Lc, k0, kend, lo, nord, acc);
            }
        }
        // block reduction: warp sums, then warps in index order
        fx_block_sums(acc, nord, S.red);
        __syncthreads();
        if (threadIdx.x < 2 * nord) {
            double sum = 0.0;
            if (!(threadIdx.x & 1)) {
                for (int wp = 0; wp < BLOCK / 32; ++wp) sum += S.red[wp][threadIdx.x >> 1];
                sum *= S.w;
            }
            __stcs(&Lc.partials[tile * (uint64_t)(2 * nord) + threadIdx.x], sum);
            if (!isfinite(sum)) atomicAdd(Lc.status + 1, 1ULL);
        }
    }
}

template <int DMAX, int BLOCK>
constexpr int fx_dyn_smem(int prow, bool mixed) {
    return (int)sizeof(FxShared) + 16 * DMAX * BLOCK + (mixed ? 4 : 8) * prow * DMAX * BLOCK;
}

template <int DMAX, int SMAX, int LMAX, bool MIXED, int BLOCK, int HI>
bool fx_allow() {
    static std::atomic<uint64_t> done{0};
    return qmc_allow_smem(done, qmc_real_kernel<DMAX, SMAX, LMAX, MIXED, BLOCK, HI>,
                          fx_dyn_smem<DMAX, BLOCK>(QMC_EMAX, MIXED));
}

// One block size per kernel: the tile's points over its threads, whatever
// block and points per thread made the tile
template <int DMAX, int SMAX, int LMAX, bool MIXED, int BLOCK, int HI>
int fx_launch(const QmcLaunch *L, int grid, cudaStream_t st) {
    if (L->prow < 1 || L->prow > QMC_EMAX || !fx_allow<DMAX, SMAX, LMAX, MIXED, BLOCK, HI>()) return -1;
    qmc_real_kernel<DMAX, SMAX, LMAX, MIXED, BLOCK, HI>
        <<<grid, BLOCK, fx_dyn_smem<DMAX, BLOCK>(L->prow, MIXED), st>>>(*L, (int)((L->tile_k + BLOCK - 1) / BLOCK));
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int DMAX, int SMAX, int LMAX, bool MIXED, int BLOCK, int HI>
int fx_occupancy(int prow) {
    if (!fx_allow<DMAX, SMAX, LMAX, MIXED, BLOCK, HI>()) return 0;
    int v = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &v, qmc_real_kernel<DMAX, SMAX, LMAX, MIXED, BLOCK, HI>, BLOCK, fx_dyn_smem<DMAX, BLOCK>(prow, MIXED));
    return e == cudaSuccess ? v : 0;
}
