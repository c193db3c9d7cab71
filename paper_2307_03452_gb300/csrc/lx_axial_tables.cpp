// Host-side tables of the axial form (lx_axial.cu), in long double from closed forms and
// recurrences:
//  * real solid harmonics Y_lm = A_m(x, y) sum_j a_j rho^2j z^(l-m-2j) with A_m = Re, Im (x+iy)^m and
//    a_{j+1}/a_j = -(l-m-2j)(l-m-2j-1) / (4 (j+1)(j+1+m)), scaled so that Y_l0(0,0,1) = 1 and
//    rotations act orthogonally (Helgaker, Jorgensen & Olsen, Molecular Electronic-Structure
//    Theory, section 6.4); on x^l-normalised Gaussians they are unit-normalised;
//  * the axial part of a product, Y_lM Y_l'M -> sum_L G r^(l+l'-L) Y_L0, by Gauss-Legendre
//    quadrature of the azimuthal average;
//  * Laguerre inversion rho^2s A_M e^{-zeta rho^2} = sum_q tau (d_x^2 + d_y^2)^q A_M(d) e^{-zeta rho^2};
//  * three-term recurrence in l of the small Wigner functions d^l_{m'm} (Varshalovich, Moskalev &
//    Khersonskii, Quantum Theory of Angular Momentum, section 4.8).
#include <algorithm>
#include <cmath>
#include <mutex>

#include "lx_axial.cuh"

namespace lx {

namespace {

using ld = long double;

ld fact(int n) {
    ld r = 1;
    for (int i = 2; i <= n; ++i) r *= i;
    return r;
}
ld binom(int n, int k) { return k < 0 || k > n ? 0.0L : fact(n) / (fact(k) * fact(n - k)); }

// z series of Y_lm (m >= 0): coefficients of rho^2j z^(l-m-2j)
std::vector<ld> harmonic(int l, int m) {
    std::vector<ld> a{std::sqrt((m ? 2.0L : 1.0L) * fact(l - m) / fact(l + m)) * fact(l + m) /
                      (std::pow(2.0L, m) * fact(m) * fact(l - m))};
    for (int j = 0; j < (l - m) / 2; ++j)
        a.push_back(a.back() * -(ld)((l - m - 2 * j) * (l - m - 2 * j - 1)) / (4.0L * (j + 1) * (j + 1 + m)));
    return a;
}

// r^2k Y_{lm} as coefficients of rho^2q z^(l+2k-m-2q)
std::vector<ld> raised(int k, int l, int m) {
    const std::vector<ld> a = harmonic(l, m);
    std::vector<ld> v(a.size() + k, 0.0L);
    for (size_t j = 0; j < a.size(); ++j)
        for (int s = 0; s <= k; ++s) v[j + s] += a[j] * binom(k, s);
    return v;
}

std::vector<ld> inverse(std::vector<ld> a, int n) {
    std::vector<ld> b(n * n, 0.0L);
    for (int i = 0; i < n; ++i) b[i * n + i] = 1;
    for (int i = 0; i < n; ++i) {
        int p = i;
        for (int r = i + 1; r < n; ++r)
            if (std::fabs(a[r * n + i]) > std::fabs(a[p * n + i])) p = r;
        for (int c = 0; c < n; ++c) {
            std::swap(a[i * n + c], a[p * n + c]);
            std::swap(b[i * n + c], b[p * n + c]);
        }
        const ld d = a[i * n + i];
        for (int c = 0; c < n; ++c) {
            a[i * n + c] /= d;
            b[i * n + c] /= d;
        }
        for (int r = 0; r < n; ++r) {
            const ld f = a[r * n + i];
            if (r == i || f == 0) continue;
            for (int c = 0; c < n; ++c) {
                a[r * n + c] -= f * a[i * n + c];
                b[r * n + c] -= f * b[i * n + c];
            }
        }
    }
    return b;
}

}  // namespace

void make_axial_tables(AxHost& H) {
    // axial products
    constexpr int NQ = 32;  // degree 4 LMAX + 2 AX_LP = 56 < 2 NQ
    ld x[NQ], w[NQ], leg[2 * AX_LP + 1][NQ];
    for (int i = 0; i < NQ; ++i) {
        ld t = std::cos(3.14159265358979323846L * (i + 0.75L) / (NQ + 0.5L)), dp = 1;
        for (int it = 0; it < 20; ++it) {
            ld p0 = 1, p1 = t;
            for (int n = 1; n < NQ; ++n) {
                const ld p2 = ((2 * n + 1) * t * p1 - n * p0) / (n + 1);
                p0 = p1;
                p1 = p2;
            }
            dp = NQ * (p0 - t * p1) / (1 - t * t);
            t -= p1 / dp;
        }
        x[i] = t;
        w[i] = 2 / ((1 - t * t) * dp * dp);
        leg[0][i] = 1;
        leg[1][i] = t;
        for (int n = 1; n < 2 * AX_LP; ++n) leg[n + 1][i] = ((2 * n + 1) * t * leg[n][i] - n * leg[n - 1][i]) / (n + 1);
    }
    auto series = [&](int l, int m, int i) {
        const std::vector<ld> a = harmonic(l, m);
        ld s = 0;
        for (size_t j = 0; j < a.size(); ++j) s += a[j] * std::pow(1 - x[i] * x[i], (int)j) * std::pow(x[i], l - m - 2 * (int)j);
        return s;
    };
    std::vector<ld> y((size_t)AX_NL * AX_NL * NQ);
    for (int l = 0; l < AX_NL; ++l)
        for (int m = 0; m <= l; ++m)
            for (int i = 0; i < NQ; ++i) y[((size_t)l * AX_NL + m) * NQ + i] = series(l, m, i);
    int goff[AX_NL][AX_NL][AX_NL];
    for (int l = 0; l < AX_NL; ++l)
        for (int lp = l; lp < AX_NL; ++lp)
            for (int M = 0; M <= l; ++M) {
                goff[l][lp][M] = (int)H.g.size();
                for (int L = lp - l; L <= l + lp; L += 2) {
                    ld s = 0;
                    for (int i = 0; i < NQ; ++i)
                        s += w[i] * leg[L][i] * y[((size_t)l * AX_NL + M) * NQ + i] * y[((size_t)lp * AX_NL + M) * NQ + i] *
                             std::pow(1 - x[i] * x[i], M);
                    H.g.push_back((double)(s * (M ? 0.5L : 1.0L) * (2 * L + 1) / 2));
                }
            }
    // cylindrical operators (d_x^2 + d_y^2)^q d_z^(n-M-2q) A_M -> spherical (d^2)^k Y_{n-2k,M}
    for (int n = 0; n < AX_NL; ++n)
        for (int M = 0; M < AX_NL; ++M) {
            H.vinv_off.push_back((int)H.vinv.size());
            if (M > n) continue;
            const int nk = (n - M) / 2 + 1;
            std::vector<ld> v(nk * nk, 0.0L);
            for (int k = 0; k < nk; ++k) {
                const std::vector<ld> c = raised(k, n - 2 * k, M);
                for (int q = 0; q < nk; ++q) v[q * nk + k] = c[q];
            }
            for (ld t : inverse(v, nk)) H.vinv.push_back((double)t);
        }
    for (int M = 0; M < AX_NL; ++M)
        for (int s = 0; s < 8; ++s)
            for (int q = 0; q < 8; ++q)
                H.tau.push_back(q > s ? 0.0 : (double)(fact(s) / fact(q) * binom(s + M, s - q) *
                                                       std::pow(2.0L, -M - 2 * q)));
    // d chains (mp >= m >= 0): d^l_{mp,m} and d^l_{mp,-m} from l = mp up
    for (int mp = 0; mp < AX_NL; ++mp)
        for (int m = 0; m <= mp; ++m) {
            H.wig0.push_back((double)std::sqrt(binom(2 * mp, mp + m)));
            for (int l = 0; l < AX_NL; ++l) {
                const ld d = std::sqrt((ld)((l + 1) * (l + 1) - mp * mp) * ((l + 1) * (l + 1) - m * m));
                const bool in = l >= mp;
                H.wig.push_back(in ? (double)((l + 1) * (2 * l + 1) / d) : 0.0);
                H.wig.push_back(in && l ? (double)((ld)mp * m / ((ld)l * (l + 1))) : 0.0);
                H.wig.push_back(in && l ? (double)(std::sqrt((ld)(l * l - mp * mp) * (l * l - m * m)) * (l + 1) / (l * d)) : 0.0);
            }
        }
    // T(l, l', M, kappa) of every (Lb, Lk), stored for unordered (l, l')
    H.tinfo.assign((size_t)AX_NL * AX_NL * AX_NL * AX_NL, 0);
    for (int Lb = 0; Lb < AX_NL; ++Lb)
        for (int Lk = 0; Lk < AX_NL; ++Lk) {
            H.tent_off.push_back((int)H.tent.size());
            int at = 0;
            int* info = H.tinfo.data() + (size_t)(Lb * AX_NL + Lk) * AX_NL * AX_NL;
            for (int i = 0; i <= std::min(Lb, Lk); ++i)
                for (int j = i; j <= std::max(Lb, Lk); ++j) {
                    int n = 0;
                    if (i <= Lb && j <= Lk) n = std::max(n, (Lb - i) / 2 + (Lk - j) / 2 + 1);
                    if (j <= Lb && i <= Lk) n = std::max(n, (Lb - j) / 2 + (Lk - i) / 2 + 1);
                    if (!n) continue;
                    info[i * AX_NL + j] = info[j * AX_NL + i] = (at << 8) | n;
                    for (int M = 0; M <= i; ++M)
                        for (int ka = 0; ka < n; ++ka) {
                            const int N = 2 * ka + i + j, L0 = j - i;
                            H.tent.push_back(goff[i][j][M] | ((ax_bz(N) + (L0 >> 1)) << 14) | ((i + 1) << 23) | (ka ? 0 : 1 << 27));
                            ++at;
                        }
                }
            H.task_t_off.push_back((int)H.task_t.size());
            for (int nk = Lk / 2 + 1; nk >= 1; --nk) {
                for (int lp = 0; lp <= Lk; ++lp)
                    if ((Lk - lp) / 2 + 1 == nk)
                        for (int M = 0; M <= std::min(lp, Lb); ++M) H.task_t.push_back(lp | (M << 8));
                while (H.task_t.size() % 4) H.task_t.push_back(-1);
            }
        }
    H.tent_off.push_back((int)H.tent.size());
    H.task_t_off.push_back((int)H.task_t.size());
    for (int Lk = 0; Lk < AX_NL; ++Lk) {
        H.task_r_off.push_back((int)H.task_r.size());
        for (int nk = Lk / 2 + 1; nk >= 1; --nk) {
            for (int l = Lk; l >= 0; --l)
                if ((Lk - l) / 2 + 1 == nk)
                    for (int M = 0; M <= 2 * l; ++M) H.task_r.push_back(l | (M << 8));
            while (H.task_r.size() % 4) H.task_r.push_back(-1);
        }
    }
    H.task_r_off.push_back((int)H.task_r.size());
    // shell functions
    for (int l = 0; l <= LMAX; ++l)
        for (int solid = 0; solid < 2; ++solid) {
            AxShell& s = H.shell[l][solid];
            s.fn0 = (int)H.fns.size();
            s.ntot = nfun(l, solid);
            int at = 0;
            for (int lam = l; lam >= (solid ? l : 0); lam -= 2) {
                for (int m = 0; m <= lam; ++m) {
                    AxFn f{};
                    f.m = (int16_t)m;
                    f.lam = (int16_t)lam;
                    f.plus = (int16_t)(at + lam + m);
                    f.minus = (int16_t)(at + lam - m);
                    const std::vector<ld> c = raised((l - lam) / 2, lam, m);
                    for (size_t j = 0; j < c.size(); ++j) f.alpha[j] = (double)c[j];
                    H.fns.push_back(f);
                }
                at += 2 * lam + 1;
            }
            s.nfn = (int)H.fns.size() - s.fn0;
            s.wc0 = -1;
            if (solid) continue;
            // monomials in terms of the harmonics: the inverse of the harmonics' expansions
            const int nc = ncart(l);
            std::vector<ld> p((size_t)nc * nc, 0.0L);
            auto comp = [&](int ax, int ay, int az) { return (l - ax) * (l - ax + 1) / 2 + az + 0 * ay; };
            for (int i = 0; i < s.nfn; ++i) {
                const AxFn& f = H.fns[s.fn0 + i];
                const std::vector<ld> c = raised((l - f.lam) / 2, f.lam, f.m);
                for (size_t j = 0; j < c.size(); ++j)
                    for (int u = 0; u <= (int)j; ++u)
                        for (int t = 0; t <= f.m; ++t) {
                            const ld v = c[j] * binom((int)j, u) * binom(f.m, t) * ((t / 2) % 2 ? -1 : 1);
                            const int col = comp(f.m - t + 2 * ((int)j - u), t + 2 * u, l - f.m - 2 * (int)j);
                            if (t % 2 == 0) p[(size_t)f.plus * nc + col] += v;
                            else p[(size_t)f.minus * nc + col] += v;
                        }
            }
            const std::vector<ld> inv = inverse(p, nc);  // [monomial][harmonic]
            s.wc0 = (int)H.wc_row.size();
            for (int c = 0; c < nc; ++c) {
                H.wc_row.push_back((int)H.wc_idx.size());
                for (int h = 0; h < nc; ++h)
                    if (std::fabs(inv[(size_t)c * nc + h]) > 1e-13L) {
                        H.wc_idx.push_back(h);
                        H.wc_val.push_back((double)inv[(size_t)c * nc + h]);
                    }
            }
            H.wc_row.push_back((int)H.wc_idx.size());
        }
    // half rows of every pair class
    for (int la = 0; la <= LMAX; ++la)
        for (int lb = 0; lb <= LMAX; ++lb)
            for (int solid = 0; solid < 2; ++solid) {
                AxClass& c = H.cls[ax_class_id(la, lb, solid)];
                const AxShell &sa = H.shell[la][solid], &sb = H.shell[lb][solid];
                c.half0 = (int)H.halves.size();
                for (int fa = 0; fa < sa.nfn; ++fa)
                    for (int fb = 0; fb < sb.nfn; ++fb) {
                        const AxFn &A = H.fns[sa.fn0 + fa], &B = H.fns[sb.fn0 + fb];
                        const int pp = A.plus * sb.ntot + B.plus, mm = A.minus * sb.ntot + B.minus,
                                  mp = A.minus * sb.ntot + B.plus, pm = A.plus * sb.ntot + B.minus;
                        const int M0 = A.m + B.m, M1 = std::abs(A.m - B.m);
                        const bool both = A.m && B.m;
                        const int sine0 = both || A.m ? mp : (B.m ? pm : -1);
                        H.halves.push_back({(int16_t)fa, (int16_t)fb, (int16_t)M0, 0, (int16_t)pp, (int16_t)sine0, 0});
                        if (both)
                            H.halves.push_back(
                                {(int16_t)fa, (int16_t)fb, (int16_t)M1, 1, (int16_t)mm, (int16_t)(M1 ? pm : -1), 0});
                    }
                c.nhalf = (int)H.halves.size() - c.half0;
                std::stable_sort(H.halves.begin() + c.half0, H.halves.end(),
                                 [](const AxHalf& a, const AxHalf& b) { return a.M < b.M; });
                int off = 0;
                for (int i = c.half0; i < c.half0 + c.nhalf; ++i) {
                    H.halves[i].hoff = off;
                    for (int l = H.halves[i].M; l <= la + lb; ++l) off += (la + lb - l) / 2 + 1;
                }
                c.nh = off;
            }
}

const AxHost& axial_tables() {
    static std::once_flag once;
    static AxHost H;
    std::call_once(once, [] { make_axial_tables(H); });
    return H;
}

}  // namespace lx
