// Prisms in block fixed point (fe_fixed.cuh), one zeta level of the six-point rule
// per thread: the sums of the FP64 form's level_sums and pair_blocks on integers.
//
// At a point with cofactor rows a_1..a_3 of J and det = det J, with f = w / |det|,
//   Gamma = B^T-contracted coefficients vol B C B^T,  B = diag(1, J^{-T}),
// has Gamma_ij = f a_i^T C3 a_j, Gamma_0j = f det c0 . a_j, Gamma_i0 = f det a_i . ci0 and
// Gamma_00 = f det^2 c00. The weights of the shape functions at a point are small
// rationals, 2 h_k = m_k / 6 and h_k = m_k / 12 with m_k = 4 for the point's own
// vertex and 1 otherwise: 1/6 goes into the value row (t6 = det / 6 for det), 1/12
// into a_3, and the sums over a level's points are then of integers:
//   SF_kk' = sum m_k m_k' G00 + m_k D_k' . G0 + m_k' D_k . G.0 + D_k G D_k',
//   SP_kk' = sum m_k' (m_k G03 + D_k . G.3),  SQ_kk' = sum m_k (m_k' G30 + D_k' . G3.),
//   SG_kk' = sum m_k m_k' G33,
//   BU_k = sum m_k d0 + D_k . dl,  BR_k = sum m_k dl_3
// (D = d lambda / d(xi, eta), D_0 = (-1, -1)). One exponent each for the cofactors
// (per coordinate axis, as in TetFx), det, f and the coefficients of all six points
// is agreed by the two threads from the first point of their levels with a spare
// bit; an element whose other points leave that range goes to the double form. a_3
// / 12 has an exponent of its own (flat and tall prisms have a_3 far from a_1, a_2):
// sums with a_3 once or twice are in units finer by 2^dz and 2^(2 dz) until the
// level's end.
#pragma once
#include "fe_fixed.cuh"

namespace fe {

// Largest magnitude of integers, by their high words: the largest and the smallest.
struct FxRange {
    int32_t mx, mn;
    FE_HD void add(int64_t a, int64_t b) {
        const int32_t u = fx_hi32(a), v = fx_hi32(b);
        mx = fx_maxi(fx_maxi(mx, u), v);
        mn = fx_mini(fx_mini(mn, u), v);
    }
    FE_HD uint32_t bits() const { return static_cast<uint32_t>(fx_maxi(mx, ~mn)); }
};

struct PrismFx {
    static constexpr int kMaxA = 12, kMaxDet = 24;
    // Evenness (as for TetFx; generic kind, whose coefficients are cut to one unit): the
    // kernels leave pairs to the double form whose diagonal diffusion coefficients spread
    // over more than kDiagSpread + 1 bits on a level (the largest of its points each, zeros
    // apart). 3,000 prisms of a slab with diffusion diag(1, e, e), median of the largest
    // relative error of an entry of A^e, fixed / double: e = 2^-4 0.95, 2^-6 1.9, 2^-8 3.7,
    // 2^-20 7.0 (in the norm of A^e 0.43 throughout); of 80,000 with the benchmark's
    // coefficients none is left. Unweighted, unlike TetFx's: every entry of a flat or tall
    // prism has a part along each axis (slab scaled by 2^-6 or 2^6 along z: 0.56 and 1.3).
    static constexpr int kDiagSpread = 6;
    static constexpr int kEdgeWin = TetFx::kEdgeWin;
    // |Gamma| < 2^59.4, Gamma_33 2^58.8 and in the value row 2^57.6: the level sums, of
    // 12, 18 and 42 of them, stay below 2^63
    static constexpr uint32_t kGammaHi = 0x0A800000, kGamma3Hi = 0x06E00000, kValueHi = 0x03000000;

    Fx2 cx[3], cy[3], cz[3][3];   // columns of J (d x / d xi, d eta; d zeta at point t), exponent of the edges
    Fx2 ncz0[3];
    int64_t r1[3], r2[3];         // cofactors a_1, a_2 of point 0, not yet normalised
    int64_t r3[3];                // a_3 / 12, likewise (in units finer by 4)
    Fx2 a3[3], a1[3], a2[3];
    int64_t half;
    int xe[3], xs, na, nd, dz, X[4], xf, Ec, Eb, xg, xl, lza, lzb, dP, dQ, dG, dV, dW;
    bool ok, neg;
    struct Sums {
        int64_t SF[9], SP[9], SQ[9], SG[6], BU[3], BR[3];
    } S;
    // a point: rows i of C^ (i = 3 the value row) against f a_j, columns a_m against ci0
    // and the value entry; then Gamma at the level's points
    int64_t Y[4][3], Z[3], y00, dl0, dl1, dl2, dl3;
    Fx2 t6, ft;
    bool ng;
    int s12, s3, sV, En[6];
    FxRange b12, b3, bV;   // of the products: axes with j = 1, 2, with j = 3, value row
    // Laplace: the points' G13, G23, G33 and load, the sums of G11, G12, G22
    int64_t G13[3], G23[3], G33[3], d0[3], S4[3];
    // Generic: 20 values per point kept in memory, v[20 t + i] (the thread's share of
    // the points' coefficients where those are per point: a point's are read before
    // its values are written): i = 0 G00, 1..3 G0j, 4..6 Gi0, 7.. Gij row by row, 16 the
    // load, 17.. dl
    int64_t *v;
    FxRange gb, g3, gv;
    int64_t SV[9], SW[2][6];   // the value row's part of SF, and of SP and SQ
    int64_t s4[4], p2[2][3], q2[2][3];

    FE_HD static void negate(const Fx2 a[3], Fx2 n[3]) {   // a's low limbs are above -2^31
#pragma unroll
        for (int i = 0; i < 3; ++i) n[i] = {-a[i].h, -a[i].l};
    }
    FE_HD static Fx2 limbs_neg(int64_t m) {   // limbs whose negatives exist
        Fx2 v = fx_limbs(m);
        v.l = v.l > -0x7FFFFFFF ? v.l : -0x7FFFFFFF;
        return v;
    }
    FE_HD static double flip(double v, bool ng) { return fx_double(fx_hi(v) ^ (ng ? 0x80000000u : 0u), fx_lo(v)); }
    FE_HD static Fx2 limbs_at(int64_t m, int n) {
        return fx_limbs(static_cast<int64_t>(static_cast<uint64_t>(m) << (n & 63)));
    }

    // Edges, the level's columns and point 0's cofactors. bits of a_1, a_2 and of a_3:
    // to agree on their shifts.
    template <class XS> FE_HD void begin(const XS &x, int l, uint32_t &bits, uint32_t &bits3) {
        double ed[15];
#pragma unroll
        for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int i = 0; i < 3; ++i)
#ifdef __CUDA_ARCH__
                ed[3 * k + i] = __dadd_rn(x(3 * (k + 1) + i), -x(i));
#else
                ed[3 * k + i] = x(3 * (k + 1) + i) - x(i);
#endif
        ok = true;
        neg = false;
        S4[0] = S4[1] = S4[2] = 0;
        gb = g3 = gv = {0, 0};
        int Ee[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            uint32_t e = fx_max3(fx_hi(ed[i]) & 0x7FFFFFFFu, fx_hi(ed[3 + i]), fx_hi(ed[6 + i]));
            e = fx_max3(e, fx_hi(ed[9 + i]), fx_hi(ed[12 + i]));
            Ee[i] = static_cast<int>(e >> 20);
            ok = ok && static_cast<unsigned>(Ee[i] - 1023 + kEdgeWin) <= 2u * kEdgeWin;
            xe[i] = Ee[i] - 1023 - 59;
        }
        half = static_cast<int64_t>(0x80000000u | static_cast<uint32_t>(Ee[0] & 0x7FF));
        // 61-bit integers of zb (the bottom nodes' weight on this level), 2/3, 1/3
        const Fx2 zb = fx_limbs(l ? 0x06C32C5D37E671D9ll : 0x193CD3A2C8198E27ll);
        const Fx2 c23 = fx_limbs(0x1555555555555555ll), c13 = fx_limbs(0x0AAAAAAAAAAAAAABll);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            int64_t m[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) m[k] = fx_from<7>(ed[3 * k + i], Ee[i] - fx_exp(ed[3 * k + i]));
            const int64_t ut = m[3] - m[2], vt = m[4] - m[2];
            cx[i] = limbs_neg(ut + fx_mul8(fx_limbs(m[0] - ut), zb));
            cy[i] = limbs_neg(vt + fx_mul8(fx_limbs(m[1] - vt), zb));
            const int64_t w0 = m[2], w1 = m[3] - m[0], w2 = m[4] - m[1];
            FxAcc s{0, 0};
            s.mul(fx_limbs((w0 + w1 + w2) >> 1), c23);   // (w0 + w1 + w2) / 12 = half of it, 2/3, 2^-2
            const int64_t wm = s.get<1>();
            cz[0][i] = limbs_neg(wm + (w0 >> 2));
            cz[1][i] = limbs_neg(wm + (w1 >> 2));
            cz[2][i] = limbs_neg(wm + (w2 >> 2));
        }
        Fx2 n[3];
        negate(cy, n);
        bits = bits3 = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            // 16 a_3 / 12 = (4 a_3) / 3
            FxAcc s{half >> 2, 0};
            s.mul(cx[(i + 1) % 3], cy[(i + 2) % 3]);
            s.mul(cx[(i + 2) % 3], n[(i + 1) % 3]);
            r3[i] = fx_mul8(fx_limbs(s.get<2>()), c13, half >> 3);
            bits3 |= fx_hi_bits(r3[i]);
        }
        cof(0);
#pragma unroll
        for (int i = 0; i < 3; ++i) bits |= fx_hi_bits(r1[i]) | fx_hi_bits(r2[i]);
    }
    // v[t] = x (the points run in a rolled loop: no indexed registers)
    FE_HD static void put(int64_t v[3], int t, int64_t x) {
        v[0] = t == 0 ? x : v[0];
        v[1] = t == 1 ? x : v[1];
        v[2] = t == 2 ? x : v[2];
    }
    // a_1 = c_y x c_z, a_2 = c_z x c_x of point t
    FE_HD void cof(int t) {
        Fx2 n[3], z[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            z[i].h = t == 0 ? cz[0][i].h : (t == 1 ? cz[1][i].h : cz[2][i].h);
            z[i].l = t == 0 ? cz[0][i].l : (t == 1 ? cz[1][i].l : cz[2][i].l);
        }
        negate(z, n);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            FxAcc s{half >> 2, 0};
            s.mul(cy[(i + 1) % 3], z[(i + 2) % 3]);
            s.mul(cy[(i + 2) % 3], n[(i + 1) % 3]);
            r1[i] = s.get<2>();
            FxAcc u{half >> 2, 0};
            u.mul(z[(i + 1) % 3], cx[(i + 2) % 3]);
            u.mul(n[(i + 2) % 3], cx[(i + 1) % 3]);
            r2[i] = u.get<2>();
        }
    }
    // The cofactors' common shifts from both levels' bits; point 0's det.
    FE_HD uint32_t set_a(uint32_t bits, uint32_t bits3) {
        na = fx_shift(bits) - 1;
        na = na > 0 ? na : 0;
        int na3 = fx_shift(bits3) - 1;
        na3 = na3 > 0 ? na3 : 0;
        ok = ok && na <= kMaxA && na3 <= kMaxA;
        dz = 2 + na3 - na;
        xs = xe[0] + xe[1] + xe[2] + 62 - na;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            X[i] = xs - xe[i];
            a3[i] = limbs_at(r3[i], na3);
        }
        return fx_hi_bits(det_raw());
    }
    // Normalises a_1, a_2; c_x . a_1
    FE_HD int64_t det_raw() {
        uint32_t b = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            b |= fx_hi_bits(r1[i]) | fx_hi_bits(r2[i]);
            a1[i] = limbs_at(r1[i], na);
            a2[i] = limbs_at(r2[i], na);
        }
        ok = ok && fx_shift(b) >= na;
        FxAcc s{0, 0};
#pragma unroll
        for (int i = 0; i < 3; ++i) s.mul(cx[i], a1[i]);
        return s.get<2>();
    }
    FE_HD void set_det(uint32_t bits) {
        nd = fx_shift(bits) - 1;
        nd = nd > 0 ? nd : 0;
        ok = ok && nd <= kMaxDet;
        const int xt = xs + 62 - nd;
        X[3] = xt - 2;
        xf = -121 - xt;
    }
    // Exponents of this level's weighted coefficients, the largest over the level's
    // points, column by column of C^ (the larger of the two levels' are common):
    // En[0..2] the axes, En[3] ci0 and c0j, En[4] c00, En[5] the load. c(20 q + j), q < np.
    // EVEN: with the test of kDiagSpread.
    template <int KIND, bool EVEN = false, class CS> FE_HD void exponents(const CS &c, int np) {
#pragma unroll
        for (int j = 0; j < 6; ++j) En[j] = -100000;
        if (KIND == 1) {
            int dmin = 1 << 20, dmax = -(1 << 20);
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const int o = i < 3 ? 4 * (i + 1) : (i == 3 ? 0 : 16);
                double v[4], u[4], w[4];
                fx_quad(c, o, v);
                fx_quad(c, np == 3 ? 20 + o : o, u);
                fx_quad(c, np == 3 ? 40 + o : o, w);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int e = static_cast<int>(fx_max3(fx_hi(v[j]) & 0x7FFFFFFFu, fx_hi(u[j]), fx_hi(w[j])) >> 20);
                    if (EVEN && i < 3 && j == i + 1 && e > 0) {
                        dmin = fx_mini(dmin, e);
                        dmax = fx_maxi(dmax, e);
                    }
                    if (i < 3)
                        En[j ? j - 1 : 3] = fx_maxi(En[j ? j - 1 : 3], e + (X[i] + X[j ? j - 1 : 3]));
                    else if (i == 3)
                        En[j ? 3 : 4] = fx_maxi(En[j ? 3 : 4], e + (X[3] + X[j ? j - 1 : 3]));
                    else
                        En[5] = fx_maxi(En[5], e + X[j ? j - 1 : 3]);
                }
            }
            if (EVEN) ok = ok && dmax - dmin <= kDiagSpread;
        } else {
            for (int q = 0; q < np; ++q) En[5] = fx_maxi(En[5], fx_exp(c(q)) + X[3]);
        }
    }
    template <int KIND> FE_HD void common_exponents() {
        Eb = En[5];
        if (KIND == 0)
            Ec = 1023 + 2 * fx_maxi(fx_maxi(X[0], X[1]), X[2]);   // see xgamma
        else
            Ec = fx_maxi(fx_maxi(fx_maxi(En[0], En[1]), En[2]), fx_maxi(En[3], En[4]));
    }
    // exponent of Gamma before the shifts: coefficients 2^(Ec - 1023 - 59), f a 2^(xf + 60),
    // their products / 2^60 and times a / 2^62; Laplace: f a 2^(xf + 61), times a / 2^62
    template <int KIND> FE_HD int xgamma() const { return KIND == 1 ? Ec - 1023 - 59 + xf + 182 : Ec - 1023 + xf + 61 + 62; }
    FE_HD int xload() const { return Eb - 1023 - 59 + 64; }
    // Windows of the common exponents; n values of this thread all zero otherwise
    template <int KIND, class CS> FE_HD void set_exponents(const CS &c, int np) {
        if (TetFx::outside(xgamma<KIND>())) {
            if (KIND == 0) ok = false;
            for (int q = 0; KIND == 1 && q < np; ++q)
                for (int j = 0; j < 16; ++j) ok = ok && c(20 * q + j) == 0.0;   // NaN compares unequal
            Ec -= xgamma<KIND>();
        }
        if (TetFx::outside(xload())) {
            for (int q = 0; q < np; ++q)
                for (int j = 16; j < 20; ++j) ok = ok && (KIND == 1 ? c(20 * q + j) : c(q)) == 0.0;
            Eb -= xload();
        }
    }

    // value i of the three points
    struct Points {
        int64_t q[3];
        FE_HD int64_t operator[](int t) const { return q[t]; }
        FE_HD int64_t sum() const { return q[0] + q[1] + q[2]; }
    };
    FE_HD Points at(int i) const { return {{v[i], v[20 + i], v[40 + i]}}; }
    // S_kk' = D_k . (w1, w2)_k', transposed on request
    FE_HD static void pi(const int64_t w1[3], const int64_t w2[3], int64_t s[9], bool tr) {
#pragma unroll
        for (int h = 0; h < 3; ++h) {
            s[tr ? 3 * h : h] = -(w1[h] + w2[h]);
            s[tr ? 3 * h + 1 : 3 + h] = w1[h];
            s[tr ? 3 * h + 2 : 6 + h] = w2[h];
        }
    }
    // m with weight m_k = 4 at t == k, 1 otherwise: sum_t m_k q_t
    template <class P> FE_HD static void weighted(const P &q, int64_t w[3]) {
        const int64_t T = q[0] + q[1] + q[2];
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = T + 3 * q[k];
    }
    // sum_t m_k m_k' q_t for (0,0), (1,1), (2,2), (0,1), (0,2), (1,2)
    template <class P> FE_HD static void weighted2(const P &q, int64_t w[6]) {
        const int64_t T = q[0] + q[1] + q[2];
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = T + 15 * q[k];
        w[3] = T + 3 * (q[0] + q[1]);
        w[4] = T + 3 * (q[0] + q[2]);
        w[5] = T + 3 * (q[1] + q[2]);
    }

    // Point t (a constant), first part: cofactors, det, f a_j and their products with
    // the coefficients; o: values per point (0: the element's). T12, T3 (point 0):
    // bounds of the axes' products with j = 1, 2 and j = 3, as powers of two from the
    // coefficients' exponents, to agree on their shifts.
    template <int KIND, class CS>
    FE_HD void products(const CS &c, int o, int t, int &T12, int &T3) {
        if (t > 0) cof(t);
        const int64_t dr = static_cast<int64_t>(static_cast<uint64_t>(det_raw()) << (nd & 63));
        const uint32_t hb = fx_hi_bits(dr);
        ok = ok && hb >= (1u << 26) && hb < (1u << 29);   // |det| in [2^58, 2^61)
        ng = dr < 0;
        neg = neg || ng;
        const double vn = fx_to(ng ? -dr : dr, -60);
        t6 = fx_limbs(fx_mul8(fx_limbs(dr), fx_limbs(0x1555555555555555ll)));   // (2/3) 2^61
        const double fd = fx_recip(vn, 4.0 / 3.0);
        const Fx2 f = fx_limbs(fx_from<8>(fd, 1025 - fx_exp(fd)));
        ft = fx_limbs(ng ? -0x038E38E38E38E38Ell : 0x038E38E38E38E38Ell);       // f t6 = +- 2^63 / 36
        Fx2 g[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                FxAcc s{half >> 4, 0};
                s.mul(f, j == 0 ? a1[i] : (j == 1 ? a2[i] : a3[i]));
                int top;
                if (KIND == 0) {
                    Y[i][j] = fx_shr(s.get<3>(), Ec - 1023 - 2 * X[i]);   // C = I: the axes' weights
                    top = 64 - fx_clz(fx_hi_bits(Y[i][j]));
                } else {
                    const int64_t v = s.get<4>();   // below 2^61.5: three products of it still sum to 63 bits
                    g[j][i] = fx_limbs(v);
                    top = 64 - fx_clz(fx_hi_bits(v)) - (Ec - En[i]);
                }
                if (t == 0) {
                    if (j < 2)
                        T12 = i + j == 0 ? top : fx_maxi(T12, top);
                    else
                        T3 = i == 0 ? top : fx_maxi(T3, top);
                }
            }
        b12 = b3 = bV = {0, 0};
        if constexpr (KIND == 1) {
            const int q = t * o;
            FxAcc z[3] = {{half >> 4, 0}, {half >> 4, 0}, {half >> 4, 0}};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                double v[4];
                fx_quad(c, i < 3 ? q + 4 * (i + 1) : q, v);
                Fx2 ck[3];
                const int w = Ec - X[i];
#pragma unroll
                for (int k = 0; k < 3; ++k) ck[k] = fx_limbs(fx_from<7>(v[k + 1], w - X[k] - fx_exp(v[k + 1])));
                const Fx2 c0 = fx_limbs(fx_from<7>(v[0], w - X[3] - fx_exp(v[0])));
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    FxAcc s{half >> 4, 0};
#pragma unroll
                    for (int k = 0; k < 3; ++k) s.mul(ck[k], g[j][k]);
                    Y[i][j] = s.get<4>();
                }
                if (i < 3) {
                    z[0].mul(a1[i], c0);
                    z[1].mul(a2[i], c0);
                    z[2].mul(a3[i], c0);
                } else {
                    FxAcc s{half >> 4, 0};
                    s.mul(c0, ft);
                    y00 = s.get<4>();
                }
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                Z[m] = z[m].get<4>();
                bV.add(Z[m], Y[3][m]);
            }
            bV.add(y00, y00);
            // load vector, with the sign of det
            double v[4];
            fx_quad(c, q + 16, v);
            Fx2 dk[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double dv = flip(v[k + 1], ng);
                dk[k] = fx_limbs(fx_from<7>(dv, Eb - X[k] - fx_exp(dv)));
            }
            dl1 = fx_dot3(dk, a1, half);
            dl2 = fx_dot3(dk, a2, half);
            dl3 = fx_dot3(dk, a3, half);
            dl0 = load(v[0]);
        } else {
            put(d0, t, load(c(t * o)));
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            b12.add(Y[i][0], Y[i][1]);
            b3.add(Y[i][2], Y[i][2]);
        }
    }
    FE_HD int64_t load(double v) const {
        const double dv = flip(v, ng);
        FxAcc s{half, 0};
        s.mul(t6, fx_limbs(fx_from<7>(dv, Eb - X[3] - fx_exp(dv))));
        return s.get();
    }
    // The products' shifts from both levels' bounds: below 3 2^58 (Laplace 2^58) at
    // point 0. The value row's from the common exponents.
    FE_HD static int room(int T) { return T >= 58 ? 0 : (T < -2 ? 60 : 58 - T); }
    FE_HD void set_products(int T12, int T3) {
        s12 = room(T12);
        s3 = room(T3);
        sV = room(fx_maxi(60 - (Ec - En[3]), 58 - (Ec - En[4])));
    }
    // Generic kind, after set_products, the same for both levels: whether the first point's
    // det and the products of coefficients and cofactors are not far below their bounds.
    // Stretched and sheared elements off the axes lose bits of both to the common units.
    // 1,500 prisms each, rms error in the norm of A^e against the double form of the
    // kernels, per element / per point: slab 0.51 / 0.55; stretched along any direction 2^3
    // times 1.1 / 1.1, 2^4 1.3 / 1.7, 2^5 2.2 / 2.0; sheared 2 to 1 0.73 / 0.75; what is kept
    // 0.8 at most. Slabs flattened or elongated 16 times along the axes are kept whole, of
    // 80,000 with all nodes jittered none was left. (Laplace kind: 0.5 to 0.83 without.)
    FE_HD bool even_shape() const { return nd <= 3 || (nd == 4 && s12 + s3 <= 1); }
    FE_HD static bool fits(uint32_t bits, int s) { return bits == 0 || fx_shift(bits) >= s; }
    // Second part: Gamma at the point.
    template <int KIND> FE_HD void gamma(int t) {
        ok = ok && fits(b12.bits(), s12) && fits(b3.bits(), s3) && (KIND == 0 || fits(bV.bits(), sV));
        const int64_t h1 = half >> 2;   // rounds get<2>
        Fx2 y[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) y[i][j] = limbs_at(Y[i][j], j < 2 ? s12 : s3);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
#pragma unroll
            for (int j = KIND == 1 ? 0 : m; j < 3; ++j) {
                FxAcc s{h1, 0};
#pragma unroll
                for (int i = 0; i < 3; ++i) s.mul(m == 0 ? a1[i] : (m == 1 ? a2[i] : a3[i]), y[i][j]);
                const int64_t G = s.get<2>();
                (m == 2 && j == 2 ? g3 : gb).add(G, G);
                if (KIND == 1)
                    v[20 * t + 7 + 3 * m + j] = G;
                else if (j < 2)
                    S4[m + j] += G;
                else
                    put(m == 0 ? G13 : (m == 1 ? G23 : G33), t, G);
            }
        }
        if constexpr (KIND == 1) {
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                FxAcc s{h1, 0};
                s.mul(limbs_at(Z[m], sV), ft);
                const int64_t g = s.get<2>();
                FxAcc u{h1, 0};
                u.mul(t6, limbs_at(Y[3][m], sV));
                const int64_t w = u.get<2>();
                v[20 * t + 4 + m] = g;
                v[20 * t + 1 + m] = w;
                gv.add(g, w);
            }
            FxAcc u{h1, 0};
            u.mul(t6, limbs_at(y00, sV));
            const int64_t g = u.get<2>();
            v[20 * t] = g;
            gv.add(g, g);
            v[20 * t + 16] = dl0;
            v[20 * t + 17] = dl1;
            v[20 * t + 18] = dl2;
            v[20 * t + 19] = dl3;
        }
    }
    // The level's sums over its points
    template <int KIND> FE_HD void sums() {
        ok = ok && gb.bits() < kGammaHi && g3.bits() < kGamma3Hi && gv.bits() < kValueHi;
        // sums with the points' weights; SF, SP and SQ are expanded from s4, p2 and q2 in
        // align (4 and 6 + 6 values across the exchange between the two threads instead of
        // 27: the per-point generic kernel fits 168 registers, 300,000 prisms 242 -> 224 us)
        if (KIND == 0) {
            s4[0] = S4[0];
            s4[1] = s4[2] = S4[1];
            s4[3] = S4[2];
            weighted(G13, p2[0]);
            weighted(G23, p2[1]);
            weighted2(G33, S.SG);
            weighted(d0, S.BU);
            S.BR[0] = S.BR[1] = S.BR[2] = 0;
        } else {
            int64_t w2[6], e1[3], e2[3], f1[3], f2[3];
            weighted2(at(0), w2);
            weighted(at(1), e1);
            weighted(at(2), e2);
            weighted(at(4), f1);
            weighted(at(5), f2);
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int kk = 0; kk < 3; ++kk) {
                    const int64_t de = kk == 0 ? -(e1[k] + e2[k]) : (kk == 1 ? e1[k] : e2[k]);
                    const int64_t df = k == 0 ? -(f1[kk] + f2[kk]) : (k == 1 ? f1[kk] : f2[kk]);
                    SV[3 * k + kk] = w2[k == kk ? k : k + kk + 2] + de + df;
                }
            weighted2(at(3), SW[0]);
            weighted2(at(6), SW[1]);
            s4[0] = at(7).sum();
            s4[1] = at(8).sum();
            s4[2] = at(10).sum();
            s4[3] = at(11).sum();
            weighted(at(9), p2[0]);
            weighted(at(12), p2[1]);
            weighted(at(13), q2[0]);
            weighted(at(14), q2[1]);
            weighted2(at(15), S.SG);
            weighted(at(16), S.BU);
            const int64_t l1 = at(17).sum(), l2 = at(18).sum();
            S.BU[0] -= l1 + l2;
            S.BU[1] += l1;
            S.BU[2] += l2;
            weighted(at(19), S.BR);
        }
        // leading zeros in units of SF and of BU: to agree on the units of the sums over
        // both levels
        dV = sV - s12;
        dW = dz + sV - s12;
        dP = dz + s3 - s12;
        dQ = dz;
        dG = 2 * dz + s3 - s12;
        uint32_t bf = 0, bp = 0, bq = 0, bg = 0, bu = 0, br = 0, bv = 0, bw = 0;
        {
            // (as they come out of align)
            int64_t w[9];
            expand4(s4, w);
#pragma unroll
            for (int k = 0; k < 9; ++k) bf |= fx_hi_bits(w[k]);
            pi(p2[0], p2[1], w, false);
#pragma unroll
            for (int k = 0; k < 9; ++k) bp |= fx_hi_bits(w[k]);
            if (KIND == 1) {
                pi(q2[0], q2[1], w, true);
#pragma unroll
                for (int k = 0; k < 9; ++k) bq |= fx_hi_bits(w[k]);
            }
        }
        if (KIND == 1) {
#pragma unroll
            for (int k = 0; k < 9; ++k) bv |= fx_hi_bits(SV[k]);
#pragma unroll
            for (int k = 0; k < 6; ++k) bw |= fx_hi_bits(SW[0][k]) | fx_hi_bits(SW[1][k]);
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) bg |= fx_hi_bits(S.SG[k]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            bu |= fx_hi_bits(S.BU[k]);
            if (KIND == 1) br |= fx_hi_bits(S.BR[k]);
        }
        // (minima of the leading zeros: nvcc 13.0 compiled the maxima of their negatives to
        // the maximum of the magnitudes)
        lza = fx_mini(fx_mini(fx_clz(bf), fx_clz(bp) + dP), fx_clz(bg) + dG);
        if (KIND == 1) lza = fx_mini(fx_mini(lza, fx_clz(bq) + dQ), fx_mini(fx_clz(bv) + dV, fx_clz(bw) + dW));
        lzb = fx_mini(fx_clz(bu), fx_clz(br) + dz);
    }
    // Brings the level's sums to common units from the smaller leading zeros of the two
    // levels: below 2^59, so that every entry is below 2^63.
    FE_HD static int64_t shift(int64_t m, int s) {   // m 2^s; an empty group's may be far
        const int l = s > 0 ? (s < 63 ? s : 63) : 0, r = s > 0 ? 0 : -s;
        return fx_shr(static_cast<int64_t>(static_cast<uint64_t>(m) << (l & 63)), r);
    }
    template <int KIND> FE_HD void align(int za, int zb) {
        // the largest part gets 6 leading zeros (two parts below 2^58 a sum below 2^59)
        const int sa = za - 6, sb = zb - 5;
        xg = xgamma<KIND>() - s12 - sa;
        xl = xload() - sb;
        int64_t f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] = KIND == 0 && k == 2 ? f[1] : shift(s4[k], sa);
        expand4(f, S.SF);
        shift3(p2, sa - dP);
        pi(p2[0], p2[1], S.SP, false);
        if (KIND == 0) {
            pi(p2[0], p2[1], S.SQ, true);
        } else {
            shift3(q2, sa - dQ);
            pi(q2[0], q2[1], S.SQ, true);
#pragma unroll
            for (int k = 0; k < 9; ++k) S.SF[k] += shift(SV[k], sa - dV);
        }
        if (KIND == 1) {
            int64_t p[2][6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                p[0][k] = shift(SW[0][k], sa - dW);
                p[1][k] = shift(SW[1][k], sa - dW);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int kk = 0; kk < 3; ++kk) {
                    S.SP[3 * k + kk] += p[0][k == kk ? k : k + kk + 2];
                    S.SQ[3 * k + kk] += p[1][k == kk ? k : k + kk + 2];
                }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) S.SG[k] = shift(S.SG[k], sa - dG);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            S.BU[k] = shift(S.BU[k], sb);
            if (KIND == 1) S.BR[k] = shift(S.BR[k], sb - dz);
        }
    }
    // D s D^T for the 2 x 2 matrix s (row-major), D = [-1 -1; 1 0; 0 1]
    FE_HD static void expand4(const int64_t s[4], int64_t w[9]) {
        w[4] = s[0];
        w[5] = s[1];
        w[7] = s[2];
        w[8] = s[3];
        w[3] = -(s[0] + s[1]);
        w[6] = -(s[2] + s[3]);
        w[1] = -(s[0] + s[2]);
        w[2] = -(s[1] + s[3]);
        w[0] = (s[0] + s[1]) + (s[2] + s[3]);
    }
    FE_HD static void shift3(int64_t w[2][3], int n) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            w[0][k] = shift(w[0][k], n);
            w[1][k] = shift(w[1][k], n);
        }
    }
    // This level's share of the four blocks (see the FP64 form's pair_blocks), doubled:
    // X + Y, X - Y the diagonal blocks, U + V, U - V the off-diagonal ones.
    template <class I> FE_HD void blocks(int l, int i, I &Xb, I &Yb, I &Ub, I &Vb) const {
        const int k = i / 3, kk = i % 3;
        const Fx2 cs = fx_limbs(l ? -kC2 : kC2);   // +- 1 / sqrt 3
        const Fx2 sf = fx_limbs(S.SF[i]);
        const int64_t spq = S.SP[i] + S.SQ[i];
        Xb = fx_mul8(sf, fx_limbs(0x1555555555555555ll)) + 2 * S.SG[k == kk ? k : k + kk + 2] -
             fx_mul8(fx_limbs(spq), cs);
        Ub = S.SF[i] - Xb;
        Yb = fx_mul8(sf, cs) - spq;
        Vb = S.SP[i] - S.SQ[i];
    }
    template <class I> FE_HD void loads(int l, int k, I &Xb, I &Yb) const {
        const Fx2 cs = fx_limbs(l ? -kC2 : kC2);
        Xb = S.BU[k];
        Yb = fx_mul8(fx_limbs(S.BU[k]), cs) - 2 * S.BR[k];
    }
    // results: entries of A^e from doubled sums, of b^e from doubled sums (times w = 1/6)
    FE_HD double out_a(int64_t v) const { return fx_to(v, xg - 1); }
    FE_HD double out_b(int64_t v) const {
        return fx_to(fx_mul8(fx_limbs(v >> 1), fx_limbs(0x1555555555555555ll)), xl - 2);
    }
    static constexpr int64_t kC2 = 0x1279A74590331C4Dll;   // 2^61 / sqrt 3
};

}  // namespace fe
