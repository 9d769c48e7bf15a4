// Block fixed-point arithmetic for the contractions of the FP64 form.
//
// This GPU issues 2 double operations per clock and SM, against 32 32x32+64-bit
// integer multiply-adds and 64-128 other integer operations. A double product
// summed into an accumulator costs one double instruction (64 cycles of a
// scheduler's pipe share per warp); the same product of two 61-bit integers costs
// three integer multiply-adds (12 cycles). The per-element contractions are sums
// of products of a few vectors, so each vector is converted once to integers with
// one exponent (that of its largest component), the sums of products run in
// 64-bit integers, and only the results are converted back, rounded once.
//
// A value is m 2^x with an integer |m| <= 2^61 and an exponent x shared by its
// vector; m is split into limbs m = h 2^32 + l with l signed. A sum of up to four
// products keeps the h h and the h l + l h parts (the l l part is below a quarter of
// a unit per product) and is rounded to units of 2^64: an error below about one
// unit in 2^58 times the largest product, against one in 2^53 for every operation
// of the double form. The callers normalise vectors between contractions and leave
// elements to the double form whose exponents are outside a window (see TetFx).
//
// Host and device code: the same functions run on the CPU in the tests.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define FE_HD __host__ __device__ __forceinline__
#else
#define FE_HD inline
#endif

namespace fe {

struct Fx2 {
    int32_t h, l;
};

// a b as mul.wide: ptxas then fuses the following 64-bit addition into one integer
// multiply-add. From a C++ product (or mad.wide) nvcc 13.0 made 2 to 3.6
// instructions per accumulated product (ncu instruction counts).
FE_HD int64_t fx_mulw(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
#else
    return int64_t(a) * b;
#endif
}

// Limbs of m, |m| <= 2^61: |h| <= 2^29, l in [-2^31, 2^31).
FE_HD Fx2 fx_limbs(int64_t m) {
    const uint32_t l = static_cast<uint32_t>(m);
    return {static_cast<int32_t>(static_cast<uint32_t>(static_cast<uint64_t>(m) >> 32) + (l >> 31)),
            static_cast<int32_t>(l)};
}

// Sum of products: mid = sum (h l' + l h'), hh = sum h h'. Four products of
// limbs within the bounds above stay within 63 bits.
struct FxAcc {
    int64_t mid, hh;
    FE_HD void mul(Fx2 a, Fx2 b) {
        mid += fx_mulw(a.h, b.l);
        mid += fx_mulw(a.l, b.h);
        hh += fx_mulw(a.h, b.h);
    }
    // in units of 2^64: rounded if mid started at 2^31, else truncated
    FE_HD int64_t get() const { return hh + (mid >> 32); }
    // in units of 2^(64 - N), truncated unless mid started at 2^(31 - N)
    template <int N> FE_HD int64_t get() const {
        return static_cast<int64_t>(static_cast<uint64_t>(hh) << N) + (mid >> (32 - N));
    }
};

// a b in units of 2^61 (rounded with round = 2^28)
FE_HD int64_t fx_mul8(Fx2 a, Fx2 b, int64_t round = 0) {
    FxAcc s{round, 0};
    s.mul(a, b);
    return s.get<3>();
}
FE_HD int64_t fx_dot3(const Fx2 a[3], const Fx2 b[3], int64_t half) {
    FxAcc s{half, 0};
    s.mul(a[0], b[0]);
    s.mul(a[1], b[1]);
    s.mul(a[2], b[2]);
    return s.get();
}

FE_HD int fx_maxi(int a, int b) { return a > b ? a : b; }
FE_HD int fx_mini(int a, int b) { return a < b ? a : b; }
// Leading zeros of a 32-bit word (32 for 0).
FE_HD int fx_clz(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __clz(static_cast<int>(v));
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
// Bits of the high word of |m| (of m's one's complement for negative m).
FE_HD uint32_t fx_hi_bits(int64_t m) {
    const int32_t h = static_cast<int32_t>(m >> 32);
    return static_cast<uint32_t>(h ^ (h >> 31));
}
FE_HD int32_t fx_hi32(int64_t m) { return static_cast<int32_t>(m >> 32); }
// The left shift that brings the largest of values with high-word bits `bits`
// (the OR of fx_hi_bits) to [2^60, 2^61). Values below 2^32 count as 2^32.
FE_HD int fx_shift(uint32_t bits) { return fx_clz(bits) - 3; }

FE_HD uint32_t fx_hi(double v) {
#ifdef __CUDA_ARCH__
    return static_cast<uint32_t>(__double2hiint(v));
#else
    uint64_t u;
    memcpy(&u, &v, 8);
    return static_cast<uint32_t>(u >> 32);
#endif
}
FE_HD uint32_t fx_lo(double v) {
#ifdef __CUDA_ARCH__
    return static_cast<uint32_t>(__double2loint(v));
#else
    uint64_t u;
    memcpy(&u, &v, 8);
    return static_cast<uint32_t>(u);
#endif
}
FE_HD double fx_double(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(lo));
#else
    const uint64_t u = (uint64_t(hi) << 32) | lo;
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}
// Biased exponent field of |v|.
FE_HD int fx_exp(double v) { return static_cast<int>((fx_hi(v) >> 20) & 0x7FFu); }

// m 2^-d, d >= 0, rounded down (0 or -1 for d > 63).
FE_HD int64_t fx_shr(int64_t m, int d) {
#ifdef __CUDA_ARCH__
    asm("shr.s64 %0, %0, %1;" : "+l"(m) : "r"(d));   // amounts above 63 count as 63
    return m;
#else
    return m >> (d > 63 ? 63 : d);
#endif
}

// v's significand 2^(52 + SH) scaled to an exponent field d above v's own,
// truncated toward zero: an integer below 2^(53 + SH) in magnitude. Zero (and a
// subnormal) gives 0 when d >= 64.
template <int SH> FE_HD int64_t fx_from(double v, int d) {
    const uint32_t h = fx_hi(v);
    uint64_t m = ((uint64_t((h & 0xFFFFFu) | 0x100000u) << 32) | fx_lo(v)) << SH;
#ifdef __CUDA_ARCH__
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(d));   // amounts above 63 give 0
#else
    m = d > 63 ? 0 : m >> d;
#endif
    int64_t r = static_cast<int64_t>(m);
#ifdef __CUDA_ARCH__
    asm("{\n .reg .pred p;\n setp.lt.s32 p, %1, 0;\n @p neg.s64 %0, %0;\n}" : "+l"(r) : "r"(h));
#else
    r = (h >> 31) ? -r : r;
#endif
    return r;
}

// m 2^x, rounded once; x within the normal range for every m != 0.
FE_HD double fx_to(int64_t m, int x) {
#ifdef __CUDA_ARCH__
    const double v = __ll2double_rn(m);
#else
    const double v = static_cast<double>(m);
#endif
    uint32_t h = fx_hi(v);
    const uint32_t s = static_cast<uint32_t>(x) << 20;
#ifdef __CUDA_ARCH__
    asm("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n @p add.u32 %0, %0, %1;\n}" : "+r"(h) : "r"(s));
#else
    h = h ? h + s : 0;   // |m| >= 1: h != 0
#endif
    return fx_double(h, fx_lo(v));
}

// w / v for normal v > 0 away from the range's ends: a float reciprocal of the
// leading 24 bits and one third-order Newton step (as recip_scaled).
FE_HD double fx_recip(double v, double w) {
#ifdef __CUDA_ARCH__
    const uint32_t hv = fx_hi(v);
    const float m = __uint_as_float(0x3F800000u | ((hv & 0xFFFFFu) << 3) | (fx_lo(v) >> 29));
    const uint32_t rb = __float_as_uint(__frcp_rn(m));
    const uint32_t yh = (((rb >> 23) + 1919u - (hv >> 20)) << 20) | ((rb & 0x7FFFFFu) >> 3);
    const double y0 = fx_double(yh, rb << 29);
    const double wy0 = __dmul_rn(w, y0);
    const double e = __fma_rn(-v, y0, 1.0);
    return __fma_rn(wy0, __fma_rn(e, e, e), wy0);
#else
    return w / v;
#endif
}

// The largest of three doubles' magnitudes by their high words (the first already
// without its sign). On the device the words compare as floats' magnitudes (one
// instruction, the signs dropped); a word that is a float NaN (|v| >= 2^1017,
// infinities, NaN) gives NaN, whose exponent field is outside every window.
FE_HD uint32_t fx_max3(uint32_t m, uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;"
        : "=f"(r)
        : "f"(__uint_as_float(m)), "f"(__uint_as_float(a)), "f"(__uint_as_float(b)));
    return __float_as_uint(r);
#else
    a &= 0x7FFFFFFFu;
    b &= 0x7FFFFFFFu;
    m = m > a ? m : a;
    return m > b ? m : b;
#endif
}
// Values j .. j + 3 of an accessor.
template <class S> FE_HD void fx_quad(const S &s, int j, double v[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = s(j + i);
}

// Tetrahedra with per-element coefficients in block fixed point. With the
// cofactor rows a_m = det J grad phi_m (m = 1..3, a_0 = -(a_1 + a_2 + a_3)),
// t = det J / 4 and f = W / |det J|,
//   A_rs = f (a_r, t) C^ (a_s, t)^T  (+ the same mass term again on the diagonal
//                                     for the four-point rule),
//   b_r  = sign(det J) W (a_r, t) . (d^1..d^3, d^0),
// C^ = [ c^{ij}  c^{i0} ; c^{0j}  kappa c^{00} ], kappa = 16 M2_01 / W (the sums of
// tet_generic_aug with sm = f t and mu = f t^2 kappa c^{00}): the coefficients enter
// as they are in memory, and f (a_s, t) needs nine products, f t being
// sign(det J) W / 4. Edges are differences in double (as the double form's).
//
// The coordinate axes carry an exponent each (that of the largest edge component
// along the axis), so that axis-aligned flat or long elements lose nothing: with
// D = diag(2^X) over the axes' cofactors and t, (a_r, t) = a^_r D and the integers
// a^_r meet the coefficients D C^ D, which share one exponent per element.
//
// False (nothing written) for elements that the double form takes: exponents of the
// edges or of the results outside the windows below (infinities and NaN among them),
// det J below 2^-20 of |edge| |cofactor| after that scaling (nearly or
// exactly degenerate: its sign and the degeneracy test are then those of the
// double form) or all cofactors below 2^-8 of |edge|^2 (nearly parallel edges).
struct TetFx {
    static constexpr int kMaxA = 12, kMaxDet = 24;   // largest normalising shifts (3 to 4 of them usual)
    // Edges within 2^+-80 bound every exponent sum below by |X_i + X_k - xt| <= 330:
    // results within 2^-700 .. 2^600 (of their last bit) then exclude an infinite or
    // NaN coefficient (2^1024 and more) and admit any within 2^+-300.
    static constexpr int kEdgeWin = 80, kLow = -700, kHigh = 600;
    // Evenness: an element's results share a unit (that of the largest), where double
    // gives every product its own. The kernels leave elements to the double form in which
    // this could cost more than double's own cancellation: generic ones whose weighted
    // diagonal diffusion coefficients that are not zero spread over more than
    // kDiagSpread + 1 bits (anisotropic diffusion along the axes, flat elements). 10,368
    // jittered tetrahedra with diffusion diag(1, e, e), 99% point of the largest relative
    // error of an entry of A^e, fixed / double: e = 2^-4 0.30, 2^-8 0.70, 2^-10 1.4, 2^-12 2.2,
    // 2^-20 33; with full random coefficients and the z axis scaled by 2^-3 1.05, 2^-5 3.4.
    // With the benchmark's coefficients one in 50,000 is left.
    static constexpr int kDiagSpread = 7;
    // and elements of either kind with a cofactor row below 2^-4 of the edges' products
    // along the axes (high words of the raw rows below kMinRow: a short or a long edge off
    // the axes). 10,368 tetrahedra, rms error in the norm of A^e, fixed / double: jittered
    // 0.53; one edge 2^4, 2^6, 2^8 times the others along (1, 1, 1) 1.25, 4.3, 31 (Laplace
    // kind the same); two edges of 2^-6 160; the ones that are kept 0.9 at most. Of 384,000
    // jittered tetrahedra one in 75,000 is left.
    static constexpr uint32_t kMinRow = 1u << 22;
    // and Laplace ones whose products are all below 2^52 units (high words of the diagonal
    // ones below kMinSum), where the axis with the largest exponent has small components: 8,000
    // tetrahedra stretched 2^5 times along any direction, 99% point of the error in the
    // norm of A^e, fixed / double: 3.3, of those that are kept 0.4. None of 384,000
    // jittered ones is left, and none for being flat or long along the axes.
    static constexpr int kMinSum = 1 << 20;
    FE_HD static bool outside(int x) { return static_cast<unsigned>(x - kLow) > static_cast<unsigned>(kHigh - kLow); }

    Fx2 a[3][3];        // cofactor rows 1..3, exponents X[0..2] along the axes
    Fx2 t;              // det / 4, exponent X[3]
    Fx2 f;              // W / |det|, exponent xf
    int64_t half;       // 2^31 (rounding of sums), from run-time data: see geometry
    int X[4], xf;
    bool neg;           // det < 0
    uint32_t low;       // high-word bits of the smallest raw cofactor row
    double vn;          // |det| / 4 / 2^(X[3] + 60), in [1, 2]

    template <class XS> FE_HD bool geometry(const XS &x) {
        double ed[9];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int i = 0; i < 3; ++i)
#ifdef __CUDA_ARCH__
                ed[3 * k + i] = __dadd_rn(x(3 * (k + 1) + i), -x(i));
#else
                ed[3 * k + i] = x(3 * (k + 1) + i) - x(i);
#endif
        int Ee[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Ee[i] = static_cast<int>(fx_max3(fx_hi(ed[i]) & 0x7FFFFFFFu, fx_hi(ed[3 + i]), fx_hi(ed[6 + i])) >> 20);
            if (static_cast<unsigned>(Ee[i] - 1023 + kEdgeWin) > 2u * kEdgeWin) return false;
        }
        // 2^31 up to 2^11, not a constant to the compiler: a constant start of a sum
        // of products kept ptxas from fusing the first product's addition
        half = static_cast<int64_t>(0x80000000u | static_cast<uint32_t>(Ee[0]));
        Fx2 e[3][3], n[3][3];   // edges and their negatives
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                Fx2 v = fx_limbs(fx_from<8>(ed[3 * k + i], Ee[i] - fx_exp(ed[3 * k + i])));
                v.l = v.l > -0x7FFFFFFF ? v.l : -0x7FFFFFFF;   // so that -l exists
                e[k][i] = v;
                n[k][i] = {-v.h, -v.l};
            }
        int64_t r[3][3];
        uint32_t bits = 0;
        low = 0xFFFFFFFFu;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int j = (m + 1) % 3, k = (m + 2) % 3;   // a_m = e_j x e_k
            uint32_t row = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                FxAcc s{half, 0};
                s.mul(e[j][(i + 1) % 3], e[k][(i + 2) % 3]);
                s.mul(e[j][(i + 2) % 3], n[k][(i + 1) % 3]);
                r[m][i] = s.get();
                row |= fx_hi_bits(r[m][i]);
            }
            bits |= row;
            low = low < row ? low : row;
        }
        const int na = fx_shift(bits);
        if (na > kMaxA) return false;
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int i = 0; i < 3; ++i) a[m][i] = fx_limbs(static_cast<int64_t>(static_cast<uint64_t>(r[m][i]) << na));
        const int xs = Ee[0] + Ee[1] + Ee[2] - 3 * (1023 + 60) + 64 - na;   // exponent of edge x cofactor
#pragma unroll
        for (int i = 0; i < 3; ++i) X[i] = xs - (Ee[i] - 1023 - 60);
        const int64_t d = fx_dot3(e[0], a[0], half);
        const int nd = fx_shift(fx_hi_bits(d));
        if (nd > kMaxDet) return false;
        const int64_t dm = static_cast<int64_t>(static_cast<uint64_t>(d) << nd);
        t = fx_limbs(dm);
        X[3] = xs + 62 - nd;
        neg = dm < 0;
        vn = fx_to(neg ? -dm : dm, -60);
        // f = W / |det| = (4/3) / vn 2^(-125 - X[3])
        const double fd = fx_recip(vn, 4.0 / 3.0);
        f = fx_limbs(fx_from<8>(fd, 1023 - fx_exp(fd)));
        xf = -125 - X[3];
        return true;
    }
    // f a_m in units of 2^(xf + X[i] + 61): at most (4/3) 2^60 (f t is +-(2/3) 2^60 of
    // 2^(xf + X[3] + 61))
    FE_HD void scaled(Fx2 fa[3][3]) const {
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int i = 0; i < 3; ++i) fa[m][i] = fx_limbs(fx_mul8(f, a[m][i]));
    }

    // |det J|
    FE_HD double volume() const { return fx_double(fx_hi(vn) + (static_cast<uint32_t>(X[3] + 62) << 20), fx_lo(vn)); }

    // Laplace kind: A_rs = f a_r . a_s (r, s = 1..3), row and column 0 from the
    // vanishing sums. False for elements that are left to the double form (kMinSum).
    FE_HD bool laplace(double A[16]) const {
        // the axes' products brought to the largest axis' exponent
        int xm = X[0] > X[1] ? X[0] : X[1];
        xm = xm > X[2] ? xm : X[2];
        const int xo = xf + 61 + 2 * xm + 64;
        int64_t row0[3] = {0, 0, 0};
        int sum = 0;
        Fx2 fa[3][3];
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int i = 0; i < 3; ++i) fa[m][i] = fx_limbs(fx_shr(fx_mul8(f, a[m][i]), 2 * (xm - X[i])));
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int s = r; s < 3; ++s) {
                const int64_t g = fx_dot3(fa[r], a[s], half);   // |g| < 2^60: the sums of nine below fit
                row0[s] -= g;
                if (r != s)
                    row0[r] -= g;
                else
                    sum = fx_maxi(sum, fx_hi32(g));
                A[4 * (r + 1) + s + 1] = A[4 * (s + 1) + r + 1] = fx_to(g, xo);
            }
#pragma unroll
        for (int s = 0; s < 3; ++s) A[1 + s] = A[4 * (1 + s)] = fx_to(row0[s], xo);
        A[0] = fx_to(-(row0[0] + row0[1] + row0[2]), xo);
        return sum >= kMinSum;
    }

    FE_HD bool even_rows() const { return low >= kMinRow; }
    // Generic kind: see kDiagSpread. (A zero's exponent field is 0: never the largest.)
    template <class CS> FE_HD bool even(const CS &c) const {
        int mn = 1 << 20, mx = -(1 << 20);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int f = fx_exp(c(5 + 5 * i)), e = f + 2 * X[i];
            mn = fx_mini(mn, f ? e : 1 << 20);
            mx = fx_maxi(mx, e);
        }
        return mx - mn <= kDiagSpread;
    }

    // Generic kind, MASS2: the four-point rule (kappa = 0.8, mass term twice on the
    // diagonal); else the one-point rule (kappa = 1). First everything that reads the
    // coefficients: P_rk = (a_r, t) . C^[.][k] (row 0 from the vanishing sum of the
    // a_r) in units of 2^(xo - xf - 61 - 64), pm = t kappa c^{00} in the same units,
    // and the load vector; then row by row A_r.
    struct Rows {
        int64_t P[4][4], pm;
        int xo;
    };
    template <bool MASS2, class CS> FE_HD bool columns(const CS &c, Rows &R, double b[4]) const {
        // exponents of D C^ D (axis 3: t) and of the weighted load coefficients
        int Ec, Eb;
        {
            double v[4];
            fx_quad(c, 0, v);
            Ec = fx_exp(v[0]) + 2 * X[3];
            int E3 = 0;                         // row and column of t, before its own X[3]
#pragma unroll
            for (int j = 0; j < 3; ++j) E3 = fx_maxi(E3, fx_exp(v[j + 1]) + X[j]);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                fx_quad(c, 4 * (i + 1), v);
                E3 = fx_maxi(E3, fx_exp(v[0]) + X[i]);
#pragma unroll
                for (int j = 0; j < 3; ++j) Ec = fx_maxi(Ec, fx_exp(v[j + 1]) + (X[i] + X[j]));
            }
            Ec = fx_maxi(Ec, E3 + X[3]);
            fx_quad(c, 16, v);
            Eb = fx_exp(v[0]) + X[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) Eb = fx_maxi(Eb, fx_exp(v[i + 1]) + X[i]);
        }
        R.xo = Ec - 1023 - 59 + xf + 189;
        int xb = Eb - 1023 - 60 - 63 + 61 + 64;
        // outside the window: exact zeros (no operator, no load) are fine
        if (outside(R.xo)) {
            for (int j = 0; j < 16; ++j)
                if (c(j) != 0.0) return false;   // NaN compares unequal
            Ec += -R.xo;                         // any exponent in the window: all integers are 0
            R.xo = 0;
        }
        if (outside(xb)) {
            for (int j = 16; j < 20; ++j)
                if (c(j) != 0.0) return false;
            Eb += -xb;
            xb = 0;
        }
#ifdef __CUDA_ARCH__
        asm volatile("" ::: "memory");   // read again below: 40 registers less than holding them
#endif
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int w = Ec - X[k];
            const int col = k == 3 ? 0 : k + 1;
            Fx2 ck[4];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const double v = c(4 * (i + 1) + col);
                ck[i] = fx_limbs(fx_from<7>(v, w - X[i] - fx_exp(v)));
            }
            const double v = c(col);
            int64_t m = fx_from<7>(v, w - X[3] - fx_exp(v));
            if (MASS2 && k == 3) m = fx_mul8(fx_limbs(m), fx_limbs(0x1999999999999999ll));   // 0.8 2^61
            ck[3] = fx_limbs(m);
            FxAcc T{half, 0};
            T.mul(t, ck[3]);
            const int64_t tk = T.get();
            int64_t p0 = tk * 4;
#pragma unroll
            for (int r = 1; r < 4; ++r) {
                FxAcc s = T;
#pragma unroll
                for (int i = 0; i < 3; ++i) s.mul(a[r - 1][i], ck[i]);
                R.P[r][k] = s.get();
                p0 -= R.P[r][k];
            }
            R.P[0][k] = p0;
            if (k == 3) R.pm = MASS2 ? tk : 0;
        }
        // load vector
        const Fx2 w = fx_limbs(neg ? -0x1555555555555555ll : 0x1555555555555555ll);   // sign(det) W = +-(4/3) 2^60 2^-63
        Fx2 d[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double v = c(17 + i);
            d[i] = fx_limbs(fx_mul8(fx_limbs(fx_from<8>(v, Eb - X[i] - fx_exp(v))), w));
        }
        const double v0 = c(16);
        const Fx2 d0 = fx_limbs(fx_mul8(fx_limbs(fx_from<8>(v0, Eb - X[3] - fx_exp(v0))), w));
        FxAcc T{half, 0};
        T.mul(t, d0);
        int64_t b0 = T.get() * 4;
#pragma unroll
        for (int r = 1; r < 4; ++r) {
            FxAcc s = T;
#pragma unroll
            for (int i = 0; i < 3; ++i) s.mul(a[r - 1][i], d[i]);
            const int64_t K = s.get();
            b0 -= K;
            b[r] = fx_to(K, xb);
        }
        b[0] = fx_to(b0, xb);
        return true;
    }
    // Row r (a constant after unrolling) of A^e. |P| < 2^59 in rows 1..3 and 2^61 in
    // row 0 (coefficients below 2^60): the normalising shift is not negative.
    template <bool MASS2> FE_HD void row(const Rows &R, const Fx2 fa[3][3], int r, double A[4]) const {
        const int64_t *P = R.P[r];
        const Fx2 ft = fx_limbs(neg ? -0x0AAAAAAAAAAAAAABll : 0x0AAAAAAAAAAAAAABll);   // f t = +-(2/3) 2^60
        const int32_t h[5] = {fx_hi32(P[0]), fx_hi32(P[1]), fx_hi32(P[2]), fx_hi32(P[3]), MASS2 ? fx_hi32(R.pm) : 0};
        int32_t mx = h[0], mn = h[0];
#pragma unroll
        for (int k = 1; k < (MASS2 ? 5 : 4); ++k) {
            mx = h[k] > mx ? h[k] : mx;
            mn = h[k] < mn ? h[k] : mn;
        }
        const int n = fx_shift(static_cast<uint32_t>(mx > ~mn ? mx : ~mn));
        const int x = R.xo - n;
        Fx2 p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) p[k] = fx_limbs(static_cast<int64_t>(static_cast<uint64_t>(P[k]) << n));
        FxAcc U{half, 0};
        U.mul(p[3], ft);
        int64_t k0 = U.get() * 4;
        const Fx2 pd = fx_limbs(static_cast<int64_t>(static_cast<uint64_t>(R.pm) << n));
#pragma unroll
        for (int s = 1; s < 4; ++s) {
            FxAcc v = U;
#pragma unroll
            for (int k = 0; k < 3; ++k) v.mul(p[k], fa[s - 1][k]);
            k0 -= v.get();
            if (MASS2 && s == r) v.mul(pd, ft);
            A[s] = fx_to(v.get(), x);
        }
        if (MASS2 && r == 0) {
            FxAcc v{half, 0};
            v.mul(pd, ft);
            k0 += v.get();
        }
        A[0] = fx_to(k0, x);
    }
    template <bool MASS2, class CS> FE_HD bool generic(const CS &c, double A[16], double b[4]) const {
        Rows R;
        if (!columns<MASS2>(c, R, b)) return false;
        Fx2 fa[3][3];
        scaled(fa);
#pragma unroll
        for (int r = 0; r < 4; ++r) row<MASS2>(R, fa, r, A + 4 * r);
        return true;
    }
};

}  // namespace fe
