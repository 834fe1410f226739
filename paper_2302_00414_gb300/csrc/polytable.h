// Window polynomials made on the host (no CUDA header is needed).
//
// For float64 Kaiser-Bessel plans, in double-double arithmetic (Dekker / Knuth
// error-free sums and products): tap s = 1..m is interpolated at n Chebyshev points of v, phi from the power series
// of I0, and rewritten in powers of v.  What is alike for every window (the change of basis, the series' reciprocals) is
// made once per process, 0.1 ms; a new window then takes 0.01 ms (m = 4) to 0.1 ms (m = 15) of a Grace core, a tap's nodes
// evaluated together.  With one node after the other, a division per term and Newton's form per tap it was 0.2 to
// 1.2 ms, beside the 0.3 to 0.4 ms of a small plan.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <vector>

namespace infft {

struct dd { double h, l; };
inline dd two_sum(double a, double b) { const double s = a + b, t = s - a; return {s, (a - (s - t)) + (b - t)}; }
inline dd operator+(dd a, dd b) { dd s = two_sum(a.h, b.h); s.l += a.l + b.l; return two_sum(s.h, s.l); }
inline dd operator-(dd a) { return {-a.h, -a.l}; }
inline dd operator*(dd a, dd b) {
    const double p = a.h * b.h, e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
    return two_sum(p, e);
}
inline dd operator/(dd a, dd b) {
    const double q1 = a.h / b.h;
    dd r = a + -(b * dd{q1, 0.0});
    const double q2 = r.h / b.h;
    r = r + -(b * dd{q2, 0.0});
    return two_sum(q1, q2) + dd{r.h / b.h, 0.0};
}

// what every window's table takes: the nodes, the map from values at them to powers of v, and 1 / i^2
template <int n>
struct PolyBasis {
    static constexpr int TERMS = 400;
    double x[n];
    dd map[n][n];   // [j][k]: coefficient k of the polynomial that is 1 at node j and 0 at the others
    dd inv2[TERMS];
    PolyBasis() {
        for (int k = 0; k < n; ++k) x[k] = std::cos(M_PI * (k + 0.5) / n);
        for (int j = 0; j < n; ++j) {   // prod (v - x_i) / (x_j - x_i) over i != j
            dd c[n];
            for (int k = 0; k < n; ++k) c[k] = dd{k == 0 ? 1.0 : 0.0, 0.0};
            dd scale{1.0, 0.0};
            for (int i = 0; i < n; ++i) {
                if (i == j) continue;
                for (int k = n - 1; k >= 1; --k) c[k] = c[k - 1] + -(c[k] * dd{x[i], 0.0});
                c[0] = -(c[0] * dd{x[i], 0.0});
                scale = scale * two_sum(x[j], -x[i]);
            }
            for (int k = 0; k < n; ++k) map[j][k] = c[k] / scale;
        }
        for (int i = 1; i < TERMS; ++i) inv2[i] = dd{1.0, 0.0} / dd{(double)i * i, 0.0};
    }
};

// coef[k stride + s - 1], k < n, s = 1..m
template <int n>
inline void kb_poly_table(int m, double beta, int stride, std::vector<double>& coef) {
    static const PolyBasis<n> B;
    coef.assign((size_t)n * stride, 0.0);
    const dd hb2 = dd{0.5 * beta, 0.0} * dd{0.5 * beta, 0.0}, m2 = dd{(double)m * m, 0.0};
    const dd im2 = dd{1.0, 0.0} / m2, one{1.0, 0.0};
    for (int s = 1; s <= m; ++s) {
        // delta = (v + 1) / 2 + m - s; z = (beta / 2)^2 (1 - (delta / m)^2); I0 = sum z^i / (i!)^2 as
        // 1 + z / 1 (1 + z / 4 (1 + z / 9 (..))).  The terms below 1e-13 of the sum are added up in doubles (to
        // 1e-29 of it), those before in double-doubles.
        dd z[n], f[n];
        double top = 0.0, tail[n];
        for (int k = 0; k < n; ++k) {
            const dd delta = two_sum(0.5 * B.x[k], 0.5) + dd{(double)(m - s), 0.0};
            z[k] = hb2 * (one + -((delta * delta) * im2));
            tail[k] = 1.0;
            top = std::max(top, z[k].h);
        }
        int last = 1, head = 0;
        for (double term = 1.0, sum = 1.0; last < PolyBasis<n>::TERMS - 1; ++last) {
            term *= top / ((double)last * last);
            sum += term;
            if (head == 0 && term < 1e-13 * sum) head = last;
            if (term < 1e-29 * sum) break;
        }
        for (int i = last; i > head; --i)
            for (int k = 0; k < n; ++k) tail[k] = 1.0 + z[k].h * B.inv2[i].h * tail[k];
        for (int k = 0; k < n; ++k) f[k] = dd{tail[k], 0.0};
        for (int i = head; i >= 1; --i)
            for (int k = 0; k < n; ++k) f[k] = one + (z[k] * B.inv2[i]) * f[k];
        dd c[n];
        for (int k = 0; k < n; ++k) c[k] = dd{0.0, 0.0};
        for (int j = 0; j < n; ++j)
            for (int k = 0; k < n; ++k) c[k] = c[k] + B.map[j][k] * f[j];
        for (int k = 0; k < n; ++k) coef[(size_t)k * stride + s - 1] = c[k].h;
    }
}

// The float32 table of the centred cardinal B-spline of order 2m: tap s at u in [0, 1] in powers of v = 2u - 1 up to
// v^(n - 1), coef[k stride + s - 1] for k < n, then what rounding took from k = 0.  The spline is a polynomial of degree
// 2m - 1 there: itself for n >= 2m, else its Chebyshev interpolant (m = 8, n = 11: off by less than 1e-11 of the
// largest value).
template <int n>
inline void bspline_poly_table(int m, int stride, std::vector<float>& coef) {
    coef.assign((size_t)(n + 1) * stride, 0.f);
    double node[n], f[n][17];   // values of every tap at the nodes, by the recursion of bspline_taps
    for (int k = 0; k < n; ++k) {
        node[k] = std::cos(M_PI * (k + 0.5) / n);
        const double u = 0.5 * (node[k] + 1.0);
        double w[16] = {1.0}, fact = 1.0;
        for (int o = 1; o < 2 * m; ++o) {
            fact *= o;
            w[o] = (1.0 - u) * w[o - 1];
            for (int j = o - 1; j >= 1; --j) w[j] = (u + j) * w[j] + (o + 1 - j - u) * w[j - 1];
            w[0] *= u;
        }
        for (int s = 1; s <= 2 * m; ++s) f[k][s] = w[2 * m - s] / fact;
    }
    for (int s = 1; s <= m; ++s) {
        double a[n] = {0.0}, t0[n] = {1.0}, t1[n] = {0.0, 1.0};   // powers of the sum, of T_(j-1) and of T_j
        for (int j = 0; j < n; ++j) {
            double c = 0.0;
            for (int k = 0; k < n; ++k) c += f[k][s] * std::cos(j * M_PI * (k + 0.5) / n);
            c *= (j == 0 ? 1.0 : 2.0) / n;
            const double* t = j == 0 ? t0 : t1;
            for (int k = 0; k < n; ++k) a[k] += c * t[k];
            if (j >= 1) {
                double t2[n];
                for (int k = 0; k < n; ++k) t2[k] = -t0[k] + (k > 0 ? 2.0 * t1[k - 1] : 0.0);
                for (int k = 0; k < n; ++k) { t0[k] = t1[k]; t1[k] = t2[k]; }
            }
        }
        for (int k = 0; k < n; ++k) coef[(size_t)k * stride + s - 1] = (float)a[k];
        coef[(size_t)n * stride + s - 1] = (float)(a[0] - (double)(float)a[0]);
    }
}

}  // namespace infft
