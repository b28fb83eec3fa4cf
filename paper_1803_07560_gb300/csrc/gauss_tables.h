// gauss_tables.h -- the tables of the Gaussian sampler's Box-Muller pairs
// (mapped_kernels.cuh), computed by the compiler in double-double arithmetic
// (pairs of doubles; TwoSum of Knuth and TwoProduct of Dekker with Veltkamp's
// splitting, as in Ogita, Rump & Oishi, SIAM J. Sci. Comput. 26, 2005), so
// that every entry is known to twice a double's precision.
#pragma once

namespace bfi {
namespace tables {

struct DD {
    double h, l;
};

constexpr DD two_sum(double a, double b) {
    const double s = a + b, t = s - a;
    return DD{s, (a - (s - t)) + (b - t)};
}
constexpr DD two_prod(double a, double b) {
    const double ca = 134217729.0 * a, cb = 134217729.0 * b;  // 2^27 + 1
    const double ah = ca - (ca - a), al = a - ah, bh = cb - (cb - b), bl = b - bh, p = a * b;
    return DD{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD add(DD a, DD b) {
    const DD s = two_sum(a.h, b.h);
    return two_sum(s.h, s.l + (a.l + b.l));
}
constexpr DD mul(DD a, DD b) {
    const DD p = two_prod(a.h, b.h);
    return two_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD div(DD a, double d) {
    const double q = a.h / d;
    const DD p = two_prod(q, d);
    return two_sum(q, (((a.h - p.h) - p.l) + a.l) / d);
}

// cos and sin of pi i / 512, i = 0 .. 128, by their Taylor series.
struct Octant {
    double c[129], s[129], c_lo[129], s_lo[129];
};
constexpr Octant make_octant() {
    Octant o{};
    for (int i = 0; i <= 128; ++i) {
        const DD x = mul(DD{3.141592653589793, 1.2246467991473532e-16}, DD{i / 512.0, 0.0}), x2 = mul(x, x);
        DD c{1.0, 0.0}, s = x, tc{1.0, 0.0}, ts = x;
        for (int n = 1; n <= 12; ++n) {
            tc = div(mul(tc, x2), -(2.0 * n - 1.0) * (2.0 * n));
            ts = div(mul(ts, x2), -(2.0 * n) * (2.0 * n + 1.0));
            c = add(c, tc);
            s = add(s, ts);
        }
        o.c[i] = c.h;
        o.c_lo[i] = c.l;
        o.s[i] = s.h;
        o.s_lo[i] = s.l;
    }
    return o;
}

// For the 128 intervals of m in [3/4, 3/2) by its seven leading bits (2^-8 wide
// below 1, 2^-7 above): c near 1/m in 20 bits (1 next to m = 1) and 2 ln c =
// 4 artanh((c - 1) / (c + 1)); and 2 k ln 2.  The upper parts are multiples of
// 2^-44, so that their sum is exact.
struct Logs {
    double c[128], hi[128], lo[128], k_hi[34], k_lo[34];
};
constexpr double upper(double x) { return (x + 384.0) - 384.0; }  // to a multiple of 2^-44 (|x| < 128)
constexpr Logs make_logs() {
    Logs t{};
    for (int i = 0; i < 128; ++i) {
        const double m = i < 64 ? 0.75 + (i + 0.5) / 256.0 : 1.0 + (i - 64 + 0.5) / 128.0;
        const double c = i == 63 ? 1.0 : static_cast<int>(1048576.0 / m) / 1048576.0;
        const DD y = div(DD{c - 1.0, 0.0}, c + 1.0), y2 = mul(y, y);
        DD p = y, sum = y;
        for (int n = 1; n <= 20; ++n) {
            p = mul(p, y2);
            sum = add(sum, div(p, 2.0 * n + 1.0));
        }
        t.c[i] = c;
        t.hi[i] = upper(4.0 * sum.h);
        t.lo[i] = (4.0 * sum.h - t.hi[i]) + 4.0 * sum.l;
    }
    for (int k = 0; k < 34; ++k) {
        const DD e = mul(DD{1.3862943611198906, 4.638093627692599e-17}, DD{static_cast<double>(k), 0.0});
        t.k_hi[k] = upper(e.h);
        t.k_lo[k] = (e.h - t.k_hi[k]) + e.l;
    }
    return t;
}

}  // namespace tables
}  // namespace bfi
