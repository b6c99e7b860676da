// FP64-accurate SIP apply in 64-bit fixed point (eq. stiffness_form).
//
// Why: GB300 executes 2 FP64 operations per SM and clock, but 64 integer
// additions and 12 wide integer multiply-adds (measured lanes per clock and SM: DFMA and
// FP64 <-> integer conversions 2.0, DADD and DMUL 1.7, a 64-bit addition about 45,
// mad.wide.s32 12).  In the unnormalised Legendre basis the 1D
// factors of the operator are small integers: P_i(+-1) = (+-1)^i,
// P_i'(+-1) = (+-1)^(i+1) i(i+1)/2, int P_a' P_b' = m(m+1), int P_p P_q' = 2,
// so traces, jumps, strains and the lifting of the face terms need additions
// only.  Three kinds of real factors remain, all applied as 64 x 64-bit
// high products (three wide multiply-adds): the viscosities, the
// geometric / mass factors (hy/hx) 2/(2b+1), and the penalty.
//
// Scaling.  The coefficients of one component on element K become integers
// U = s_i s_j u 2^FRAC / 2^e, with 2^e just above the largest |u| of that component's
// modes but the constant one, and s_i = sqrt((2i+1)/2); FRAC is the largest for
// which no sum that is multiplied can reach 2^63 (55 bits at k = 5, 57 at k = 3): a
// finer grid than FP64's on the component's largest entry, and a coarser one than
// FP64's on an entry more than 2^(FRAC - 53) below it.  The result's error is thus
// bounded by 2^-53 of the largest term that the component brings into the element, not
// of each entry's own terms.  The constant mode (0, 0) has an exponent of its own:
// it enters the jumps of the lines m = 0 and the cross sums over them and nothing
// else, and a translation of both sides of a face leaves nothing, whatever else moves
// on top of it.  (With one exponent for all entries of an element, u_x = 1 and u_y of
// size 1e-12 left 20 of the 53 bits of what u_y gives, and a nearly rigid motion of a
// stiff inclusion is such a field; the separate exponents cost 2 to 10 % of an apply.)
// Sums over one component are exact; a jump is formed on the coarser grid of the
// face's two elements, the same on both sides.  Viscosities are 62-bit
// mantissas with exponents relative to the largest of K and its neighbours.
// Products are rounded to a unit that each line picks from the magnitudes it
// has, so a large factor (penalty, stiff neighbour, the other component) costs no
// resolution where what it multiplies is small or zero.  Rounding of traces thus
// cancels between the elements of a face as it does in FP64, which matters: the
// coarse levels amplify a net force on a floating stiff inclusion by 1e4 to 1e7.
//
// With kx_b = (hy/hx) 2/(2b+1), J = own - neighbour trace, d = reference normal
// derivative trace, s = +-1 the side, the result modes along an x-line (row b)
// are, for the normal component (tangential: the kx terms but the penalty
// halved),
//   W[a] = eta_K kx_b (4 g_a - sum_s s [s^a d_K + s^(a+1) a(a+1)/2 J])
//        + sum_s s^a ( (c/2) kx_b eta_max J - s eta_N kx_b d_N - s cross ),
//   g_a = sum_i m(m+1)/2 U_i over i = a mod 2, m = min(a, i),
//   cross = eta_K sum_{m<b, odd} J_t[m]            (normal component)
//           eta_K S_K + eta_N S_N, S = sum_{m>b, odd} v_n[m]   (tangential),
// and y = s_a s_b W.  Boundary faces are ghosts: v_N = -v or +v, d_N likewise.
//
// Host and device: tests/test_fix_host.py and tests/test_fix_parts.py compile this file
// with the host compiler and run the same phases tile by tile against the oracle and the
// operator in extended precision.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace sip {
namespace fix {

using i64 = long long;

#ifdef __CUDACC__
#define FIX_HD __host__ __device__ __forceinline__
#else
#define FIX_HD inline
#endif

constexpr double csqrt_it(double x, double g, int n) {
    return n == 0 ? g : csqrt_it(x, 0.5 * (g + x / g), n - 1);
}
constexpr double leg(int i) { return csqrt_it((2.0 * i + 1.0) / 2.0, 1.5, 50); }   // s_i
constexpr double leg_sum(int n) { return n == 0 ? 0.0 : leg(n - 1) + leg_sum(n - 1); }
constexpr double der_sum(int n) {
    return n == 0 ? 0.0 : leg(n - 1) * (n - 1) * n / 2.0 + der_sum(n - 1);
}
constexpr int floor_log2(double x) {   // x > 0
    int e = 0;
    while (x >= 2.0) { x *= 0.5; ++e; }
    while (x < 1.0) { x *= 2.0; --e; }
    return e;
}

// Largest magnitudes of the sums that are multiplied, for |u| < 1, in units
// of 2^FRAC (2 % above, for roundings: see shift_by).
template <int N>
struct Bound {
    static constexpr double v = leg_sum(N) * leg(N - 1);     // value trace
    static constexpr double d = der_sum(N) * leg(N - 1);     // derivative trace
    static constexpr double J = 2.0 * v;
    static constexpr double par() {   // largest sum of s_i over one parity
        double a = 0.0, b = 0.0;
        for (int i = 0; i < N; ++i) (i % 2 ? a : b) += leg(i);
        return a > b ? a : b;
    }
    static constexpr double X = 2.0 * par() * leg_sum(N);    // cross sums of a face
    static constexpr double G() {
        double best = 0.0;
        for (int a = 0; a < N; ++a) {
            double g = 0.0;
            for (int i = 0; i < N; ++i) {
                const int m = a < i ? a : i;
                if ((a + i) % 2 == 0) g += 0.5 * m * (m + 1) * leg(i);
            }
            g *= leg(N - 1);
            best = g > best ? g : best;
        }
        return best;
    }
    static constexpr double big(double a, double b) { return a > b ? a : b; }
    static constexpr double top = 1.02 * big(big(G(), d), big(J, X));
    static constexpr int FRAC = 62 - floor_log2(top);            // top 2^FRAC < 2^63
    static constexpr int TRI = N <= 2 ? 0 : (N == 3 ? 2 : (N <= 5 ? (N == 4 ? 3 : 4) : 4));
    // 2^TRI >= (N-1) N / 2, the largest derivative factor
};

// Biased exponents (of max |u| on an element) and viscosity exponents the
// fixed-point path covers; a tile with anything else (infinities, NaN, values
// near the ends of the FP64 range) takes the FP64 formulas.
constexpr int E_MIN = 300, E_MAX = 1800, ETA_E = 150;

// Scalar factors of one operator: 62-bit mantissas and binary exponents of
// kx_b and (c/2) kx_b per [direction][tangential mode].
struct Scal {
    i64 km[2][6], pm[2][6];
    int ek[2][6], ep[2][6];
    bool ok;
};

inline void norm62(double v, i64& m, int& e) {
    const double f = std::frexp(v, &e);
    m = i64(std::ldexp(f, 62));
}

// r = hy / hx, ch = c/2 = pen_x hx / 2; ok = false: factors out of range.
template <int N>
Scal make_scal(double r, double ch) {
    Scal s;
    std::memset(&s, 0, sizeof(s));
    if (!(r > 1e-6 && r < 1e6 && ch > 1e-9 && ch < 1e9)) return s;
    const double k0[2] = {2.0 * r, 2.0 / r};
    for (int dir = 0; dir < 2; ++dir)
        for (int b = 0; b < N; ++b) {
            const double k = k0[dir] / (2.0 * b + 1.0);
            norm62(k, s.km[dir][b], s.ek[dir][b]);
            norm62(k * ch, s.pm[dir][b], s.ep[dir][b]);
        }
    s.ok = true;
    return s;
}

// A 62-bit factor split into signed 32-bit halves.
struct Wt {
    int h, l;
};
FIX_HD Wt split(i64 w) {
    Wt s;
    s.l = int(w);
    s.h = int((w >> 32) - (s.l >> 31));
    return s;
}

// (t w) / 2^64 to nearest (within 3/4 of a unit), |t| < 2^63 - 2^32, |w| < 2^62.
FIX_HD i64 mulhi(i64 t, Wt w) {
    const int tl = int(t);
    const int th = int(t >> 32) - (tl >> 31);
    const i64 mid = i64(th) * w.l + 0x80000000LL + i64(tl) * w.h;
    return i64(th) * w.h + (mid >> 32);
}
// x 2^-n to nearest; n may be negative.  (Rounding down would add a constant
// force to every element, which the coarse levels amplify by the condition of
// their problem.)
struct Shift {
    int l, n;
    i64 half;
};
FIX_HD Shift shift_by(int n) {
    Shift s;
    s.l = n < 0 ? (n > -62 ? -n : 62) : 0;   // that far up: only zeros
    s.n = n < 0 ? 0 : (n < 62 ? n : 62);
    s.half = n < 59 ? (i64(1) << s.n) >> 1 : 0;   // at most 2^57: no overflow
    return s;
}
FIX_HD i64 shr(i64 x, Shift s) { return ((x << s.l) + s.half) >> s.n; }
// the same for n >= 0 and |x| < 2^62
struct Down {
    int n;
    i64 half;
};
FIX_HD Down down_by(int n) {
    Down s;
    s.n = n < 62 ? n : 62;
    s.half = (i64(1) << s.n) >> 1;
    return s;
}
FIX_HD i64 align(i64 x, Down s) { return (x + s.half) >> s.n; }
FIX_HD i64 prod(i64 t, Wt w, Shift s) { return shr(mulhi(t, w), s); }

// high word of |t| (bitwise complement for negative t), for magnitude bounds
FIX_HD unsigned mag(i64 t) {
    const int h = int(t >> 32);
    return unsigned(h ^ (h >> 31));
}
FIX_HD int bit_length(unsigned v) {
#ifdef __CUDA_ARCH__
    return 32 - __clz(int(v));
#else
    return v ? 32 - __builtin_clz(v) : 0;
#endif
}
FIX_HD int imax(int a, int b) { return a > b ? a : b; }
FIX_HD int imin(int a, int b) { return a < b ? a : b; }
// bit_length(mag(t)), or for zero a number that no unit depends on
constexpr int NONE = -16000;
FIX_HD int length(i64 t) { return t == 0 ? NONE : bit_length(mag(t)); }
FIX_HD int bit_length64(i64 t) {   // of |t|
#ifdef __CUDA_ARCH__
    return 64 - __clzll(t < 0 ? -t : t);
#else
    return t ? 64 - __builtin_clzll((unsigned long long)(t < 0 ? -t : t)) : 0;
#endif
}
FIX_HD Wt weight(i64 eta, i64 k) { return split(mulhi(eta, split(k)) << 2); }

FIX_HD i64 bits_of(double v) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    i64 b;
    std::memcpy(&b, &v, 8);
    return b;
#endif
}
FIX_HD double of_bits(i64 b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double v;
    std::memcpy(&v, &b, 8);
    return v;
#endif
}
FIX_HD i64 to_int(double v) {
#ifdef __CUDA_ARCH__
    return __double2ll_rn(v);
#else
    return std::llrint(v);
#endif
}
FIX_HD double to_fp(i64 v) {
#ifdef __CUDA_ARCH__
    return __ll2double_rn(v);
#else
    return double(v);
#endif
}
// v 2^e for a normal v whose result is normal
FIX_HD double scale2(double v, int e) { return of_bits(bits_of(v) + (i64(e) << 52)); }

// Mantissa in [2^61, 2^62) and exponent of a normal positive number.
FIX_HD i64 eta_mant(double v) {
    return ((bits_of(v) & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL) << 9;
}
FIX_HD int eta_exp(double v) { return int(bits_of(v) >> 52) - 1022; }

template <int C>
FIX_HD i64 mulc(i64 x) {   // C x by shifts and additions
    if constexpr (C == 0) return 0;
    else if constexpr (C == 1) return x;
    else if constexpr (C % 2 == 0) return mulc<C / 2>(x) << 1;
    else if constexpr (C == 3) return (x << 1) + x;
    else {
        static_assert(C == 15, "an odd factor without a form here (5, of A = 4: see tri)");
        return (x << 4) - x;
    }
}
template <int A>
FIX_HD i64 tri(i64 x) {   // A (A + 1) / 2 x
    if constexpr (A == 4) return ((x << 2) + x) << 1;
    else return mulc<A * (A + 1) / 2>(x);
}
FIX_HD i64 tri_rt(int a, i64 x) {
    return a == 0 ? 0
                  : (a == 1 ? x
                            : (a == 2 ? tri<2>(x)
                                      : (a == 3 ? tri<3>(x) : (a == 4 ? tri<4>(x) : tri<5>(x)))));
}

// Shared-memory layout of a tile of TW x TH elements.
template <int N, int TW, int TH>
struct Tile {
    static constexpr int NN = N * N, NB = 2 * NN;
    static constexpr int NEL = TW * TH, NH = 2 * TW + 2 * TH, NS = NEL + NH;
    static constexpr int NT = NEL * N;              // one thread per (element, line)
    // faces of the tile's elements: x-normals y (TW + 1) + x, then y-normals y TW + x
    static constexpr int NFX = (TW + 1) * TH, NF = NFX + TW * (TH + 1);
    // odd strides: lanes that walk entries of one element hit distinct banks
    static constexpr int XS = NB + 1, EP = NEL + 1;
    // entries of the elements; the constant modes on grids of their own, and in the
    // word behind the entries how far their exponents lie above the component's
    // (mean_pack)
    static constexpr int O_U = 0;                   // in 8-byte words
    static constexpr int O_T = O_U + NS * XS;       // traces [(F 2 + c) N + m][val, der][element]
    static constexpr int O_H = O_T + 16 * N * NEL;  // halo traces [c N + m][val, der][halo element]
    static constexpr int O_W = O_H + 4 * N * NH;    // results [mode][element]
    static constexpr int O_C = O_W + NB * EP;       // cross terms [mode][element]
    static constexpr int O_M = O_C + NB * NEL;      // constant modes' jumps [c][face]
    static constexpr int O_ETA = O_M + 2 * NF;
    // ints: e[NS] (expo_pack), surroundings[NEL] (expo_pack of E and E + ref), row units
    // [2 N][NEL]; then exponents of the jumps [c][face] (short)
    static constexpr int O_E = O_ETA + NS;
    static constexpr int I_R = NS, I_U = NS + NEL, I_M = I_U + 2 * N * NEL;
    static constexpr size_t BYTES = size_t(O_E) * 8 + size_t(I_M) * 4 + 2 * NF * 2;
    static_assert(NEL % 32 == 0, "a warp serves one line index");
};

struct Mesh {
    int nx, ny, ex0, ey0;
    int bc[4];
};

// Biased exponents of an element's components in one int, and those of its constant
// modes relative to them in one word.
FIX_HD int expo_pack(int e0, int e1) { return e0 + (e1 - e0) * 65536; }
FIX_HD int expo(int packed, int c) { return (packed & 0xffff) + (c ? packed >> 16 : 0); }
FIX_HD i64 mean_pack(int d0, int d1) { return i64(unsigned(d0)) | (i64(d1) << 32); }
FIX_HD int mean_above(i64 packed, int c) { return c ? int(packed >> 32) : int(packed); }

// Staged element s of the tile: its mesh position; false outside the mesh.
template <int N, int TW, int TH>
FIX_HD bool staged_at(const Mesh& g, int s, int& ex, int& ey) {
    using L = Tile<N, TW, TH>;
    int x, y;
    if (s < L::NEL) {
        x = s % TW;
        y = s / TW;
    } else {
        const int h = s - L::NEL;
        if (h < TW) { x = h; y = -1; }
        else if (h < 2 * TW) { x = h - TW; y = TH; }
        else if (h < 2 * TW + TH) { x = -1; y = h - 2 * TW; }
        else { x = TW; y = h - 2 * TW - TH; }
    }
    ex = g.ex0 + x;
    ey = g.ey0 + y;
    return ex >= 0 && ex < g.nx && ey >= 0 && ey < g.ny;
}

// Staged index of the element at (x, y) of the tile or its halo.
template <int N, int TW, int TH>
FIX_HD int staged_index(int x, int y) {
    using L = Tile<N, TW, TH>;
    if (x < 0) return L::NEL + 2 * TW + y;
    if (x >= TW) return L::NEL + 2 * TW + TH + y;
    if (y < 0) return L::NEL + x;
    if (y >= TH) return L::NEL + TW + x;
    return y * TW + x;
}

// Staged index of the neighbour of tile element el across face F.
template <int N, int TW, int TH>
FIX_HD int staged_nbr(int el, int F) {
    return staged_index<N, TW, TH>(el % TW + (F == 1 ? 1 : 0) - (F == 0 ? 1 : 0),
                                   el / TW + (F == 3 ? 1 : 0) - (F == 2 ? 1 : 0));
}

FIX_HD bool has_nbr(const Mesh& g, int ex, int ey, int F) {
    return F == 0 ? ex > 0 : (F == 1 ? ex < g.nx - 1 : (F == 2 ? ey > 0 : ey < g.ny - 1));
}

// Value and reference derivative at both ends of a line.
template <int N>
FIX_HD void ends(const i64 (&U)[N], i64 (&v)[2], i64 (&d)[2]) {
    i64 e = 0, o = 0, de = 0, dn = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (i % 2 == 0) {
            e += U[i];
            de += tri_rt(i, U[i]);
        } else {
            o += U[i];
            dn += tri_rt(i, U[i]);
        }
    }
    v[0] = e - o;
    v[1] = e + o;
    d[0] = dn - de;
    d[1] = dn + de;
}

// Entries of line m but the constant mode.
template <int N>
FIX_HD void load_line(const i64* u, int dir, int m, i64 (&U)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) U[i] = dir == 0 ? u[m * N + i] : u[i * N + m];
    if (m == 0) U[0] = 0;
}

// Jumps of the constant modes (whose value trace on the line m = 0 is the same at every
// end) across face f of the tile, the element on the low side less the one on the high
// side, per component on the finest grid that holds it, with that grid's exponent (NONE:
// no jump).  A ghost has the opposite value, or the same where the boundary condition
// leaves no jump.
template <int N, int TW, int TH>
FIX_HD void mean_jumps(const Mesh& g, const i64* su, const int* se, int f, i64* jump, short* expo_of) {
    using L = Tile<N, TW, TH>;
    constexpr int FRAC = Bound<N>::FRAC;
    const bool xn = f < L::NFX;
    const int r = xn ? f : f - L::NFX, w = xn ? TW + 1 : TW, x = r % w, y = r / w;
    const int at = xn ? g.ex0 + x : g.ey0 + y, end = xn ? g.nx : g.ny;   // of the high element
    const bool inside = at <= end && (xn ? g.ey0 + y < g.ny : g.ex0 + x < g.nx);
    const int l = staged_index<N, TW, TH>(x - (xn ? 1 : 0), y - (xn ? 0 : 1)), h = staged_index<N, TW, TH>(x, y);
    const i64 *u = su + l * L::XS, *v = su + h * L::XS;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        i64 d = 0;
        int lo = NONE;
        if (inside) {
            const int a = expo(se[l], c) + mean_above(u[L::NB], c), b = expo(se[h], c) + mean_above(v[L::NB], c);
            int e = imax(a, b);
            if (at > 0 && at < end) {
                d = align(u[c * L::NN], down_by(e - a)) - align(v[c * L::NN], down_by(e - b));
            } else {
                const int kind = g.bc[(xn ? 0 : 2) + (at > 0 ? 1 : 0)];
                e = at > 0 ? a : b;
                if (kind == 2 || (kind == 0 && c == (xn ? 0 : 1)))
                    d = at > 0 ? u[c * L::NN] << 1 : -(v[c * L::NN] << 1);
            }
            const int up = imax(FRAC - bit_length64(d), 0);
            if (d != 0) lo = e - up;
            d <<= up;
        }
        jump[c * L::NF + f] = d;
        expo_of[c * L::NF + f] = short(lo);
    }
}

// Phase 1: traces of the tile's elements (all faces) and of the halo
// elements (the face towards the tile); exponents of each element's surroundings.
template <int N, int TW, int TH>
FIX_HD void phase_traces(int tid, const Mesh& g, i64* sm) {
    using L = Tile<N, TW, TH>;
    i64 *su = sm + L::O_U, *st = sm + L::O_T, *sh = sm + L::O_H;
    const double* eta = reinterpret_cast<const double*>(sm + L::O_ETA);
    int* se = reinterpret_cast<int*>(sm + L::O_E);
    const int el = tid % L::NEL, m = tid / L::NEL;
    if (tid < L::NEL) {
        int ex, ey, E = 0, R = -2000;
        if (staged_at<N, TW, TH>(g, el, ex, ey)) {
            E = imax(expo(se[el], 0), expo(se[el], 1));
            R = eta_exp(eta[el]);
            for (int F = 0; F < 4; ++F)
                if (has_nbr(g, ex, ey, F)) {
                    const int n = staged_nbr<N, TW, TH>(el, F);
                    E = imax(E, imax(expo(se[n], 0), expo(se[n], 1)));
                    const int r = eta_exp(eta[n]);
                    R = r > R ? r : R;
                }
        }
        se[L::I_R + el] = expo_pack(E, E + R);
    }
    // from the last thread down: the first ones have the halo's traces below
#pragma unroll
    for (int r = 0; r < (L::NF + L::NT - 1) / L::NT; ++r) {
        const int f = r * L::NT + L::NT - 1 - tid;
        if (f < L::NF) mean_jumps<N, TW, TH>(g, su, se, f, sm + L::O_M, reinterpret_cast<short*>(se + L::I_M));
    }
#pragma unroll
    for (int dir = 0; dir < 2; ++dir)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            i64 U[N], v[2], d[2];
            load_line<N>(su + el * L::XS + c * L::NN, dir, m, U);
            ends<N>(U, v, d);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                i64* t = st + (((2 * dir + s) * 2 + c) * N + m) * 2 * L::NEL + el;
                t[0] = v[s];
                t[L::NEL] = d[s];
            }
        }
    for (int q = tid; q < L::NH * N; q += L::NT) {
        const int h = q % L::NH, mm = q / L::NH;
        const int F = h < TW ? 3 : (h < 2 * TW ? 2 : (h < 2 * TW + TH ? 1 : 0));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            i64 U[N], v[2], d[2];
            load_line<N>(su + (L::NEL + h) * L::XS + c * L::NN, F / 2, mm, U);
            ends<N>(U, v, d);
            i64* t = sh + (c * N + mm) * 2 * L::NH + h;
            t[0] = F & 1 ? v[1] : v[0];
            t[L::NH] = F & 1 ? d[1] : d[0];
        }
    }
}

// Phases 2 (DIR = 0, rows) and 3 (DIR = 1, columns): the line m of element el,
// both components.  Rows leave their part of W with its unit and the first
// half of the cross volume terms; columns add theirs and turn W into the FP64
// result.  os: alpha s_a s_b per mode.
template <int N, int TW, int TH, int DIR>
FIX_HD void phase_lines(int tid, const Mesh& g, const Scal& k, const double* os, i64* sm) {
    using L = Tile<N, TW, TH>;
    using B = Bound<N>;
    const i64 *su = sm + L::O_U, *st = sm + L::O_T, *sh = sm + L::O_H;
    i64 *sw = sm + L::O_W, *sc = sm + L::O_C;
    const double* seta = reinterpret_cast<const double*>(sm + L::O_ETA);
    int* se = reinterpret_cast<int*>(sm + L::O_E);
    int* unit = se + L::I_U;
    const int el = tid % L::NEL, m = tid / L::NEL;
    int ex, ey;
    if (!staged_at<N, TW, TH>(g, el, ex, ey)) return;
    // E: the reference exponent (offsets below it may be negative); of each component
    const int E = expo(se[L::I_R + el], 0), ref = se[L::I_R + el] >> 16, pK = se[el];
    const int oK[2] = {E - expo(pK, 0), E - expo(pK, 1)};   // exponent offsets: own
    const double etaK = seta[el];
    const i64 mK = eta_mant(etaK);
    const int rK = ref - eta_exp(etaK);
    const int ek = k.ek[DIR][m], ep = k.ep[DIR][m];
    const Wt wC = split(mK), wK = weight(mK, k.km[DIR][m]);
    // per side: neighbour traces (or a ghost's multiples), weights, exponents
    const i64 *op[2], *np[2];
    int ns[2], oN[2][2], rN[2], rP[2], kind[2];   // oN: offsets of the neighbour's components
    // per side and component: the grid of the jumps (its offset), own and neighbour traces
    // to it, the constant mode's jump.  Both sides of a face form a jump on one grid, so
    // that what one element gains the other loses, to the last bit of the jump.
    int oG[2][2];
    Down aK[2][2], aN[2][2];
    i64 mj[2][2];
    Wt wN[2], wP[2], wCN[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int F = 2 * DIR + s;
        op[s] = st + F * 4 * N * L::NEL + el;
        np[s] = op[s];
        ns[s] = L::NEL;
        kind[s] = 1 + g.bc[F];
        double eN = etaK;
        int pN = pK;
        if (has_nbr(g, ex, ey, F)) {
            const int n = staged_nbr<N, TW, TH>(el, F);
            kind[s] = 0;
            if (n < L::NEL) {
                np[s] = st + (F ^ 1) * 4 * N * L::NEL + n;
            } else {
                np[s] = sh + (n - L::NEL);
                ns[s] = L::NH;
            }
            pN = se[n];
            eN = seta[n];
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            oN[s][c] = E - expo(pN, c);
            oG[s][c] = imin(oK[c], oN[s][c]);
            mj[s][c] = 0;
            // the constant modes are part of the jumps on line 0, and of the tangential
            // component's in the normal one's cross sums on the odd lines
            if (m == 0 || (c != DIR && m % 2 == 1)) {
                const int f = c * L::NF + (DIR == 0 ? (el / TW) * (TW + 1) + el % TW + s : L::NFX + el + s * TW);
                const int lo = reinterpret_cast<const short*>(se + L::I_M)[f];
                oG[s][c] = imin(oG[s][c], E - lo);
                const i64 j = align(sm[L::O_M + f], down_by(E - oG[s][c] - lo));
                mj[s][c] = s ? j : -j;
            }
            aK[s][c] = down_by(oK[c] - oG[s][c]);
            aN[s][c] = down_by(oN[s][c] - oG[s][c]);
        }
        const i64 mN = eta_mant(eN);
        rN[s] = ref - eta_exp(eN);
        wN[s] = weight(mN, k.km[DIR][m]);
        wCN[s] = split(mN);
        const bool mine = etaK > eN;
        wP[s] = weight(mine ? mK : mN, k.pm[DIR][m]);
        rP[s] = mine ? rK : rN[s];
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const bool normal = c == DIR;
        const int half = normal ? 0 : 1;
        i64 U[N], v[2], d[2];
        load_line<N>(su + el * L::XS + c * L::NN, DIR, m, U);
        ends<N>(U, v, d);
        // per side: jump, own and neighbour derivative, own and neighbour cross sums;
        // offset of the own cross sums' grid
        i64 J[2], O[2], Dn[2], X[2], Xn[2];
        int oX[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            constexpr int tc = 1 - DIR;
            i64 x = normal && m % 2 == 1 ? mj[s][tc] : 0, xn = 0;
            const i64 jm = m == 0 ? mj[s][c] : 0;
            oX[s] = normal ? oG[s][tc] : oK[DIR];
            if (kind[s] == 0) {
                const i64* t = np[s] + (c * N + m) * 2 * ns[s];
                J[s] = align(v[s], aK[s][c]) - align(t[0], aN[s][c]) + jm;
                O[s] = d[s];
                Dn[s] = t[ns[s]];
                if (normal) {
                    for (int mm = m - 1; mm >= 0; mm -= 2)
                        x += align(op[s][(tc * N + mm) * 2 * L::NEL], aK[s][tc]) -
                             align(np[s][(tc * N + mm) * 2 * ns[s]], aN[s][tc]);
                } else {
                    for (int mm = m + 1; mm < N; mm += 2) {
                        x += op[s][(DIR * N + mm) * 2 * L::NEL];
                        xn += np[s][(DIR * N + mm) * 2 * ns[s]];
                    }
                }
            } else {
                // ghosts: Navier (1) v_n odd, d_n even, v_t even, d_t odd;
                // Neumann (2) all so that nothing remains;
                // Dirichlet (3) both values odd, both derivatives even
                const bool on = kind[s] == 3 || (kind[s] == 1 && normal);
                J[s] = on ? (align(v[s], aK[s][c]) << 1) + jm : 0;
                O[s] = on ? d[s] : 0;
                Dn[s] = O[s];
                if (kind[s] == 3) {
                    if (normal) {
                        for (int mm = m - 1; mm >= 0; mm -= 2)
                            x += align(op[s][(tc * N + mm) * 2 * L::NEL], aK[s][tc]) << 1;
                    } else {
                        for (int mm = m + 1; mm < N; mm += 2)
                            x += op[s][(DIR * N + mm) * 2 * L::NEL];
                        xn = x;
                    }
                }
            }
            X[s] = x;
            Xn[s] = xn;
        }
        // g_a by sums over one parity: i <= a with i(i+1)/2, i > a with a(a+1)/2
        i64 G[N], T[N];
        {
            i64 suf[N], pre[N];
#pragma unroll
            for (int a = N - 1; a >= 0; --a) suf[a] = a + 2 < N ? suf[a + 2] + U[a + 2] : 0;
#pragma unroll
            for (int a = 0; a < N; ++a) {
                pre[a] = (a >= 2 ? pre[a - 2] : 0) + tri_rt(a, U[a]);
                G[a] = pre[a] + tri_rt(a, suf[a]);
            }
        }
        if constexpr (DIR == 1) {   // second half of the cross volume terms
            i64 w[N];
#pragma unroll
            for (int j = 0; j < N; ++j) w[j] = sc[((1 - c) * L::NN + j * N + m) * L::NEL + el];
            if (c == 0) {
#pragma unroll
                for (int b = 0; b < N; ++b) T[b] = b >= 1 ? (b >= 2 ? T[b - 2] : 0) + w[b - 1] : 0;
            } else {
#pragma unroll
                for (int b = N - 1; b >= 0; --b)
                    T[b] = b + 1 < N ? (b + 2 < N ? T[b + 2] : 0) + w[b + 1] : 0;
            }
        }
        // unit 2^om (on the grid of exponent E) of this line's W: the largest of its
        // terms (magnitude times factor and viscosity, number of terms of the kind)
        // stays below 2^59, their sum below 2^62.  Zeros of the other component do not
        // count: on the grid of a large one they would coarsen what a small one gives.
        unsigned bG = mag(O[0]) | mag(O[1]);
        i64 nT = 0;
        unsigned bT = 0;
#pragma unroll
        for (int a = 1; a < N; ++a) bG |= mag(G[a]);
        if constexpr (DIR == 1) {
#pragma unroll
            for (int a = 0; a < N; ++a) {
                bT |= mag(T[a]);
                nT |= T[a];
            }
        }
        int wb = imax(bit_length(bG) + ek - oK[c], (nT == 0 ? NONE : bit_length(bT)) - oK[1 - c]) + 2 - rK;
        int lJ[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            lJ[s] = bit_length(mag(J[s]));
            wb = imax(wb, lJ[s] + imax(ep, ek + B::TRI) + 2 - oG[s][c] - rP[s]);
            wb = imax(wb, bit_length(mag(Dn[s])) + ek + 2 - oN[s][c] - rN[s]);
            wb = imax(wb, length(X[s]) + 2 - oX[s] - rK);
            wb = imax(wb, length(Xn[s]) + 2 - oN[s][DIR] - rN[s]);
        }
        const int om = wb + 32 + 3 - 62;
        // a high product of a term and a 62-bit mantissa is term * mantissa / 4
        i64 P[2], Q[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            // jumps are small next to the traces where the field is smooth: shifted up
            // by what their magnitude leaves before they meet the large factors
            const int js = imax(30 - lJ[s], 0);
            const i64 j = J[s] << js;
            i64 p = prod(O[s], wK, shift_by(om - 2 - ek + rK + half + oK[c])) +
                    prod(Dn[s], wN[s], shift_by(om - 2 - ek + rN[s] + half + oN[s][c]));
            p += prod(X[s], wC, shift_by(om - 2 + rK + oX[s]));
            if (!normal) p += prod(Xn[s], wCN[s], shift_by(om - 2 + rN[s] + oN[s][DIR]));
            P[s] = prod(j, wP[s], shift_by(om - 2 + js - ep + rP[s] + oG[s][c])) + (s ? -p : p);
            Q[s] = prod(j, wK, shift_by(om - 2 + js - ek + rK + half + oG[s][c]));
        }
        const Shift sG = shift_by(om - 4 - ek + rK + half + oK[c]), sT = shift_by(om - 4 + rK + oK[1 - c]);
        const i64 Pp = P[1] + P[0], Pm = P[1] - P[0];
        const i64 Qp = Q[1] + Q[0], Qm = Q[1] - Q[0];
#pragma unroll
        for (int a = 0; a < N; ++a) {
            i64 W = (a % 2 ? Pm : Pp) - tri_rt(a, a % 2 ? Qm : Qp);
            if (a > 0) W += prod(G[a], wK, sG);
            const int mode = c * L::NN + (DIR == 0 ? m * N + a : a * N + m);
            if constexpr (DIR == 0) {
                sw[mode * L::EP + el] = W;
            } else {
                W += prod(T[a], wC, sT);
                // both parts to the coarser of their units
                const int ur = unit[(c * N + a) * L::NEL + el], u = imax(ur, om);
                W = align(W, down_by(u - om)) + align(sw[mode * L::EP + el], down_by(u - ur));
                // y = alpha s_a s_b W 2^(E - 1022 + ref + u - FRAC)
                const double f = scale2(os[a * N + m], E - 1022 + ref + u - B::FRAC);
                sw[mode * L::EP + el] = bits_of(W == 0 ? 0.0 : to_fp(W) * f);
            }
        }
        if constexpr (DIR == 0) {   // first half of the cross volume terms, for component 1 - c
            unit[(c * N + m) * L::NEL + el] = om;
            i64 q[N];
            if (c == 1) {
#pragma unroll
                for (int a = N - 1; a >= 0; --a)
                    q[a] = a + 1 < N ? (a + 2 < N ? q[a + 2] : 0) + U[a + 1] : 0;
            } else {
#pragma unroll
                for (int a = 0; a < N; ++a) q[a] = a >= 1 ? (a >= 2 ? q[a - 2] : 0) + U[a - 1] : 0;
            }
#pragma unroll
            for (int a = 0; a < N; ++a) sc[(c * L::NN + m * N + a) * L::NEL + el] = q[a];
        }
    }
}

// Factor of an entry's conversion: s_i s_j 2^FRAC / 2^e.
template <int N>
FIX_HD double in_factor(double ss, int e) {
    return scale2(ss, Bound<N>::FRAC - (e - 1022));
}

}  // namespace fix
}  // namespace sip
