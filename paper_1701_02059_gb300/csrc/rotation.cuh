// The rotational half of the B-A-O-A update in fixed point on the integer
// pipes.  GB300 issues one FP64 instruction per 16 cycles and SM, so the
// director's and angular velocity's arithmetic in FP64 (projections, two
// Cayley maps, noise, renormalisation, conversions: about 100 FP64-pipe
// instructions a lipid) bounded the whole update; the same quantities as
// 64-bit fixed point cost 32 x 32 -> 64 multiply-adds, which run at 64 lanes
// per cycle and SM.  Measured on the 4M cell: see k_baoa_d.
//
// The results are the FP64 code's, bit for bit: every increment is rounded
// onto the 2^-40 grid, and the fixed-point value and the FP64 value of an
// increment differ by less than the thresholds below (the sum of both
// errors, in fractions of the grid), so they round alike unless the value
// lies within the threshold of a rounding boundary.  Such a value (about
// 1e-3 of the lipids a step), and any value outside the ranges stated below
// (torques of 2^8 eps, rotations of more than 2^-7 per half step, directors
// off unit length), makes rot_* return false (with the outputs undefined) and
// the caller takes the FP64 code.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>

namespace orbc {

#ifndef ORBC_HD
#define ORBC_HD __host__ __device__
#endif

// host-computed constants of one instance (real value c = m 2^-k, m in
// [2^61, 2^62), as the halves of m)
struct RotK {
    int ok;             // the ranges below hold for these constants
    int a_h, a_l, a_sh; // dt/4: a = (W << a_sh) m / 2^64 at 2^-64
    int hi_h, hi_l, hi_f;       // dt/2/I: dw at 2^-(40 + hi_f)
    int hi_t0, hi_t1;           // threshold hi_t0 + hi_t1 2^-8 |T|_1 (eps/16) of the kick, at 2^-(40 + hi_f)
    int cr_h, cr_l, cr_sl, cr_sr, cr_neg;   // exp(-gamma_r dt) - 1 (its magnitude)
    int sr_h, sr_l, sr_sl, sr_sr;           // noise amplitude per integer noise unit, grid units
    int sr_t0, sr_t1;                       // threshold sr_t0 + sr_t1 |z| 2^-32 of the noise, at 2^-(40 + kRotF)
    long long wlim;     // |W| below this
};
constexpr int kRotF = 18;   // fraction bits of the Ornstein-Uhlenbeck increment below the grid

// x = h 2^32 + l with l signed
struct Half { int h, l; };
ORBC_HD inline Half halves(long long x) {
    Half r;
    r.l = (int)(unsigned)(unsigned long long)x;
    r.h = (int)((x + 0x80000000ll) >> 32);
    return r;
}

// x = m 2^-k, m in [2^61, 2^62) in halves (k = 62 and m = 0 unless x > 0)
inline int norm61(double x, int& h, int& l) {
    h = l = 0;
    if (!(x > 0)) return 62;
    int e = 0;
    const double f = std::frexp(x, &e);
    const Half m = halves((long long)std::ldexp(f, 62));
    h = m.h;
    l = m.l;
    return 62 - e;
}

// The constants of one instance: dt/4, dt/2/I, exp(-gamma_r dt) - 1 and the
// noise amplitude per integer noise unit (grid units).
inline RotK rot_constants(double quarter_dt, double h_i, double cr_m1, double srn) {
    RotK R;
    auto shifts = [](int s, int& left, int& right) {
        left = std::max(s, 0);
        right = std::min(std::max(-s, 0), 63);
    };
    R.a_sh = 88 - norm61(quarter_dt, R.a_h, R.a_l);
    R.hi_f = norm61(h_i, R.hi_h, R.hi_l) - 51;
    const int cs = 82 - norm61(std::fabs(cr_m1), R.cr_h, R.cr_l);
    shifts(cs, R.cr_sl, R.cr_sr);
    R.cr_neg = cr_m1 < 0;
    const int ss = 57 - norm61(srn, R.sr_h, R.sr_l);
    shifts(srn > 0 ? ss : 0, R.sr_sl, R.sr_sr);
    // rounding thresholds: the kick with f = hi_f (3 units of 2^-50, 2 of the
    // result, 6 2^-53 dt/2/I per 1/16 eps), the noise with f = kRotF (3 units
    // of 2^-25, 3 of the result, 8 2^-53 s 2^32)
    const double kt0 = 3.0 * h_i * std::ldexp(1.0, R.hi_f - 10) + 2.0, kt1 = h_i * std::ldexp(6.0, R.hi_f - 17 + 8);
    const double nt0 = 3.0 * srn * std::ldexp(1.0, kRotF - 25) + 3.0, nt1 = srn * std::ldexp(8.0, 32 - 53 + kRotF);
    R.ok = R.a_sh >= 0 && R.a_sh <= 40 && R.hi_f >= 8 && R.hi_f <= 30 && R.cr_sl <= 40 && R.sr_sl <= 4 && kt0 < 32768.0 &&
           kt1 < 65535.0 && nt0 < 32768.0 && nt1 < 8192.0;
    R.hi_t0 = R.ok ? (int)std::ceil(kt0) : 0;
    R.hi_t1 = R.ok ? (int)std::ceil(kt1) : 0;
    R.sr_t0 = R.ok ? (int)std::ceil(nt0) + 1 : 0;
    R.sr_t1 = R.ok ? (int)std::ceil(nt1) : 0;
    R.wlim = R.ok ? 1ll << (62 - std::max(R.a_sh, R.cr_sl)) : 0;
    return R;
}

// (x y) 2^-64 without the product of the low halves (an error below one unit
// with the floor): hi and mid sums of one or several products
struct MulAcc {
    long long hi = 0, mid = 0;
    ORBC_HD inline void add(Half x, Half y) {
        hi += (long long)x.h * y.h;
        mid += (long long)x.h * y.l;
        mid += (long long)x.l * y.h;
    }
    ORBC_HD inline void sub(Half x, Half y) {   // (only high halves are negated: a low one may be -2^31)
        hi += (long long)(-x.h) * y.h;
        mid += (long long)(-x.h) * y.l;
        mid += (long long)x.l * (-y.h);
    }
    ORBC_HD inline long long get() const { return hi + (mid >> 32); }
};
ORBC_HD inline long long mulh(Half x, Half y) {
    MulAcc m;
    m.add(x, y);
    return m.get();
}
// round(x 2^-f); near: x 2^-f lies within thr 2^-f of a rounding boundary
ORBC_HD inline long long round_f(long long x, int f, int thr, bool& near) {
    const long long r = x + (1ll << (f - 1));
    near |= ((unsigned long long)(r + thr) & ((1ull << f) - 1ull)) <= 2ull * (unsigned)thr;
    return r >> f;
}
ORBC_HD inline bool below(long long x, long long lim) { return (unsigned long long)(x + lim) <= 2ull * (unsigned long long)lim; }

// the director at 2^-61, in halves
struct Dir { Half n[3]; };
ORBC_HD inline Dir dir_of(const long long nq[3]) {
    Dir d;
    for (int a = 0; a < 3; a++) d.n[a] = halves(nq[a] << 21);
    return d;
}
ORBC_HD inline bool dir_ok(const long long nq[3]) {
    const long long lim = (1ll << 40) + (1ll << 30);
    return below(nq[0], lim) && below(nq[1], lim) && below(nq[2], lim);
}

// w += reps round(dt/2/I (T - (T.n) n)); |T| < 2^40 (2^8 eps).
// Errors: T_perp 3 units of 2^-50 (one floor and the dropped low products
// per product sum), its product with dt/2/I 1.25 units of 2^-(40 + hi_f);
// FP64: 6 roundings of |T|_1 dt/2/I (three of the sum T.n, one each of
// its product with n, of the difference and of the product with dt/2/I).
ORBC_HD inline bool rot_kick(long long wq[3], const Dir& d, const long long Tq[3], const RotK& K, int reps) {
    const long long lim = 1ll << 40;
    if (!(below(Tq[0], lim) && below(Tq[1], lim) && below(Tq[2], lim))) return false;
    MulAcc s;                                                       // T.n at 2^-50
    int t1 = 3;
    for (int a = 0; a < 3; a++) {
        s.add(halves(Tq[a] << 21), d.n[a]);
        const int e = (int)(Tq[a] >> 28);
        t1 += e < 0 ? -e : e;
    }
    const int thr = K.hi_t0 + ((K.hi_t1 * t1) >> 8);                // |T|_1 < 2^14: no overflow (hi_t1 < 2^16)
    const Half S = halves(s.get() << 3);                            // at 2^-53
    const Half m{K.hi_h, K.hi_l};
    bool near = false;
    for (int a = 0; a < 3; a++) {
        const long long D = (Tq[a] << 18) - mulh(S, d.n[a]);        // at 2^-50
        wq[a] += reps * round_f(mulh(halves(D << 3), m), K.hi_f, thr, near);
    }
    return !near;
}

// n += round(2/(1 + |a|^2) (a x n - |a|^2 n)), a = dt/4 w, |a|^2 < 2^-14
// (the angular velocity is perpendicular to the director: a x (a x n) =
// -|a|^2 n).  2/(1 + aa) = 2 (1 - c), c = aa - aa^2 + aa^3 to 2^-55.
// Errors, in units of 2^-61 (2^-60 after the factor 2): a x n - aa n 2.5,
// the product with c 1.5, c itself 1; FP64: 20 roundings of |a| (below 3072
// |a| units of 2^-60, |a| < 2^-10 + 2^8 aa).
constexpr int kTurnThr = 6;     // 2^-60
ORBC_HD inline bool rot_turn(long long nq[3], const Dir& d, const long long wq[3], const RotK& K) {
    if (!(below(wq[0], K.wlim) && below(wq[1], K.wlim) && below(wq[2], K.wlim))) return false;
    const Half m{K.a_h, K.a_l};
    Half a[3];
    for (int q = 0; q < 3; q++) a[q] = halves(mulh(halves(wq[q] << K.a_sh), m));    // at 2^-64
    long long hi = 0, mid = 0;
    for (int q = 0; q < 3; q++) {
        hi += (long long)a[q].h * a[q].h;
        mid += (long long)a[q].h * a[q].l;
    }
    const long long aa = hi + (mid >> 31);                          // |a|^2 at 2^-64
    if ((unsigned long long)aa >= (1ull << 50)) return false;
    const int a44 = (int)(aa >> 20);                                // at 2^-44
    const long long aa2 = ((long long)a44 * a44) >> 24;             // at 2^-64
    const long long aa3 = ((long long)a44 * (int)(aa2 >> 10)) >> 34;
    const Half c = halves(aa - aa2 + aa3), A = halves(aa);
    const int thr = kTurnThr + 4 + (int)((3u * (unsigned)a44) >> 26);   // 3072 |a| < 3 + 3072 2^8 aa
    bool near = false;
    for (int q = 0; q < 3; q++) {
        const int u = q == 2 ? 0 : q + 1, w = q == 0 ? 2 : q - 1;
        MulAcc t;                                                   // a x n - |a|^2 n at 2^-61
        t.add(a[u], d.n[w]);
        t.sub(a[w], d.n[u]);
        t.sub(A, d.n[q]);
        const long long tv = t.get();
        const long long y = tv - mulh(c, halves(tv));               // (1 - c) t at 2^-61
        nq[q] += round_f(y, 20, thr, near);                    // 2 y at 2^-61 = y at 2^-60
    }
    return !near;
}

// w += round((exp(-gamma dt) - 1) w + s (z - (z.n) n)), z the integer noise
// 2 (word - 2^31) + 1.
// Errors: z_perp 3 units of 2^-25 (times s), 1.25 units of 2^-(40 + kRotF)
// per product; FP64: 8 roundings of s |z|.
ORBC_HD inline bool rot_noise(long long wq[3], const Dir& d, const unsigned zw[3], const RotK& K) {
    if (!(below(wq[0], K.wlim) && below(wq[1], K.wlim) && below(wq[2], K.wlim))) return false;
    long long z[3];
    unsigned zz = 0;                                                // |z|^2 2^-36
    MulAcc s;                                                       // z.n at 2^-25
    for (int a = 0; a < 3; a++) {
        z[a] = 2 * (long long)(int)(zw[a] ^ 0x80000000u) + 1;
        const int zs = (int)(z[a] >> 18);
        zz += (unsigned)(zs * zs);
        s.add(halves(z[a] << 28), d.n[a]);
    }
    // |z| 2^-32 < 1/2 + |z|^2 2^-65
    const int thr = K.sr_t0 + (int)(((unsigned)K.sr_t1 * (((1u << 28) + zz + (1u << 17)) >> 17)) >> 12);
    const Half S = halves(s.get() << 3);                            // at 2^-28
    const Half ms{K.sr_h, K.sr_l}, mc{K.cr_h, K.cr_l};
    bool near = false;
    for (int a = 0; a < 3; a++) {
        const long long P = (z[a] << 25) - mulh(S, d.n[a]);         // at 2^-25
        const long long zi = mulh(halves((P << K.sr_sl) >> K.sr_sr), ms);
        const long long wi = mulh(halves((wq[a] << K.cr_sl) >> K.cr_sr), mc);
        wq[a] += round_f(K.cr_neg ? zi - wi : zi + wi, kRotF, thr, near);
    }
    return !near;
}

// n <- n (1 - delta/2), delta = |n|^2 - 1 exact: with n = h 2^20 + l the
// excess |n|^2 - 2^80 is ((sum h^2 - 2^40) 2^19 + sum h l) 2^21 + sum l^2.
// Errors: 1.25 units of 2^-78, FP64 two roundings of at most 2^20 grid units.
ORBC_HD inline bool rot_renorm(long long nq[3]) {
    long long hh = 0, hl = 0, ll = 0;
    for (int a = 0; a < 3; a++) {
        const int l = (int)(((unsigned)(unsigned long long)nq[a] + 0x80000u) & 0xfffffu) - 0x80000;
        const int h = (int)((nq[a] - l) >> 20);
        hh += (long long)h * h;
        hl += (long long)h * l;
        ll += (long long)l * l;
    }
    const long long e = ((hh - (1ll << 40)) << 19) + hl;
    if (!below(e, 1ll << 40)) return false;
    const Half D = halves((e << 21) + ll);
    bool near = false;
    for (int a = 0; a < 3; a++) nq[a] -= round_f(mulh(halves(nq[a] << 21), D), 38, 1 << 18, near);
    return !near;
}

}  // namespace orbc
