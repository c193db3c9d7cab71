// Axial form of the FP64 path: the two transforms of Eq. make-abq and Eq. make-abcd through
// frames in which they are sparse.
//
// A Hermite Gaussian is a polynomial in the derivatives d = d/dP of a Gaussian, and the
// integral of two of them that polynomial (the ket's with (-1)^degree, Eq. pq) applied to
// f(PQ) = [0]^(0).  Written over the operators S_klM = (d^2)^k Y_lM(d) (real solid harmonics of
// d, degree n = 2k + l) in a frame whose z axis is
//  * AB: shell functions of order m_a, m_b about AB only need M = +-m_a +- m_b, of the two kinds
//    (cosine, sine) one each: a pair's H has about one entry in twenty;
//  * PQ: S_klM S_k'l'M' f vanishes unless M = M', and is
//      T(l, l', M, k + k') = sum_L G(l, l', M, L) Z^L B_kappa(L),  kappa = k + k' + (l + l' - L) / 2,
//    with Z = |PQ| and B_kappa(L) = the radial part of (d^2)^kappa Y_L0(d) f:
//      B_0(L) = [0]^(L) (Eq. boys line), B_1(L) = pref (-2 rho)^(L+1) e^-T,
//      B_kappa+1(L) = (2L + 3) B_kappa(L + 1) + Z^2 B_kappa(L + 2)
//    (d^2 f is a Gaussian, so kappa >= 1 needs no difference of Boys functions);
//  * CD: as AB, for the ket.
// Rotations between the frames act on each l block alone (Wigner functions).  An uncontracted
// (ii|ii) quartet in solid functions executes 2.3e6 FMAs for the bra rotation, T, the ket rotation
// and the ket transform (1.4e6 on average in a 20-bohr cube, where half of the primitive quartets are far) and
// 0.8e6 to rotate its functions to the lab frame; H_ab [p+q] takes 3.5e7 and the second transform
// 1.3e7.  No step leaves FP64.  2,048 (ii|ii) quartets, solid, K = 1: 194.4 -> 13.6 ms; 200 Cartesian ones
// 169.1 -> 24.7 ms.  Against extended precision the two forms' errors are of one size (the largest 2e-15 to
// 1e-14 of the largest integral, up to 2.4 times the matrix form's where they are greater).
//
// Rows and columns are kept by half rows (AxHalf): the product of functions of orders m_a, m_b >= 0
// has orders m_a + m_b and |m_a - m_b|, each with a cosine and a sine member whose coefficients
// are the same; T sees both members through the same two sums
//   SC[k'l'M'] = sum_l dC^l[M'][M] sum_k h[kl] T(l, l', M', k + k'),   SS likewise with dS
// (dC, dS: the rotation by beta about y between cosine and between sine functions), and the
// azimuth gamma of PQ only mixes the members at the end: cosine row = cos(M gamma) SC - sin(M gamma) SS,
// sine row = sin(M gamma) SC + cos(M gamma) SS, where SC spans the cosine and SS the sine functions of
// the ket index.
//
// Kernels:
//   axial_pair_kernel    per primitive pair: zeta, P, h; per pair: frame, rotation to the lab
//   axial_boys_kernel    per primitive quartet: angles, B Z^L                (lx_boys_r.cu)
//   axial_wigner_kernel  per primitive quartet: rotation blocks
//   axial_main_kernel    per quartet and 8 half rows: T, ket rotation, ket transform
//   axial_rotate_kernel  function indices to the lab frame (and to Cartesian functions)
#include <algorithm>
#include <cmath>

#include "lx_axial.cuh"

namespace lx {

namespace {

struct AxDev {
    const double *g, *vinv, *tau, *wig0, *wig, *wc_val;
    const int *vinv_off, *tent, *tent_off, *tinfo, *task_t, *task_t_off, *task_r, *task_r_off, *wc_row, *wc_idx;
    const AxFn* fns;
    const AxHalf* halves;
    const AxClass* cls;
    AxShell shell[LMAX + 1][2];
};
__constant__ AxDev c_ax;

// Real rotation blocks of a rotation about y by beta, (c, s) = (cos, sin) of the angle of
// R = [[c, 0, s], [0, 1, 0], [-s, 0, c]] (Y_l(R v) = D Y_l(v)), for l <= lmax: C[ax_co(l) + m'(l+1) + m]
// between cosine and S[ax_so(l) + (m'-1) l + m-1] between sine functions.  One chain in l per
// (m' >= m >= 0), from the powers pw of cos and sin of the half angle.
constexpr int WIG_NP = 2 * AX_LP + 1;
__host__ __device__ inline int wigner_chains(int lmax) { return (lmax + 1) * (lmax + 2) / 2; }
// Powers 0 .. 2 lmax of b, the half angle's cos or sin, one thread.
__device__ inline void wigner_powers(int lmax, double b, double* pw) {
    double p = 1.0;
    for (int i = 0; i <= 2 * lmax; ++i) {
        pw[i] = p;
        p *= b;
    }
}
__device__ inline void wigner_chain(int i, int lmax, double c, const double* pw, double* C, double* S) {
    int mp = (int)((sqrtf(8.0f * i + 1.0f) - 1.0f) * 0.5f);
    while ((mp + 1) * (mp + 2) / 2 <= i) ++mp;
    while (mp * (mp + 1) / 2 > i) --mp;
    const int m = i - mp * (mp + 1) / 2;
    const double w0 = __ldg(c_ax.wig0 + i);
    // (-1)^(m' + m) d_{m',m} and (-1)^(m' + m) d_{m',-m}
    double x = w0 * pw[mp + m] * pw[WIG_NP + mp - m], y = w0 * pw[mp - m] * pw[WIG_NP + mp + m], xp = 0.0, yp = 0.0;
    const double flip = (mp + m) & 1 ? -1.0 : 1.0, par = m & 1 ? -1.0 : 1.0;
    const double* w = c_ax.wig + (size_t)i * AX_NL * 3;
    for (int l = mp; l <= lmax; ++l) {
        double vc, vs = 0.0;
        if (m) {
            vc = fma(par, y, x);
            vs = fma(-par, y, x);
        } else {
            vc = mp ? 1.4142135623730951 * x : x;
        }
        double* Cl = C + ax_co(l);
        Cl[mp * (l + 1) + m] = vc;
        Cl[m * (l + 1) + mp] = mp == m ? vc : flip * vc;
        if (m) {
            double* Sl = S + ax_so(l);
            Sl[(mp - 1) * l + m - 1] = vs;
            Sl[(m - 1) * l + mp - 1] = mp == m ? vs : flip * vs;
        }
        const double a = __ldg(w + 3 * l), b = __ldg(w + 3 * l + 1), cc = __ldg(w + 3 * l + 2);
        const double xn = fma(a * (c - b), x, -cc * xp), yn = fma(a * (c + b), y, -cc * yp);
        xp = x;
        yp = y;
        x = xn;
        y = yn;
    }
}

// Full blocks (2l+1)^2, l <= L, of the rotation Rz(a) Ry Rz(b): pa, pb = cos, sin of m a, m b; C, S the
// Y blocks; D[ax_do(l) + (l + m')(2l+1) + l + m], sine functions at m < 0.  The entries of all blocks
// are spread over `step` threads.
__device__ __forceinline__ void full_blocks(int L, const double* pa, const double* pb, const double* C,
                                            const double* S, double* D, int t0, int step) {
    int l = 0;
    for (int i = t0; i < ax_co(L + 1); i += step) {
        while (i >= ax_co(l + 1)) ++l;
        const int w = 2 * l + 1, e = i - ax_co(l), mp = e / (l + 1), m = e - mp * (l + 1);
        double* Dl = D + ax_do(l);
        const double c = C[i], s = mp && m ? S[ax_so(l) + (mp - 1) * l + m - 1] : 0.0;
        const double ca = pa[2 * mp], sa = pa[2 * mp + 1], cb = pb[2 * m], sb = pb[2 * m + 1];
        const double cc = c * cb, cs = c * sb, sc = -s * sb, ss = s * cb;
        Dl[(l + mp) * w + l + m] = ca * cc + sa * sc;
        if (m) Dl[(l + mp) * w + l - m] = ca * cs + sa * ss;
        if (mp) Dl[(l - mp) * w + l + m] = ca * sc - sa * cc;
        if (mp && m) Dl[(l - mp) * w + l - m] = ca * ss - sa * cs;
    }
}

// Rotation F with F n = e_z (z by -phi, then y by -theta) for a unit vector n; cp, sp = cos, sin phi.
__device__ inline void frame_of(const double n[3], double F[9], double& cp, double& sp, double& st) {
    st = ax_unit(n[0], n[1], cp, sp);
    const double ct = n[2];
    F[0] = ct * cp, F[1] = ct * sp, F[2] = -st;
    F[3] = -sp, F[4] = cp, F[5] = 0.0;
    F[6] = st * cp, F[7] = st * sp, F[8] = ct;
}

// ------------------------------------------------------------------ pairs

constexpr int AXP_THREADS = 128;
constexpr int AXP_NV = AX_NL;  // z-derivative orders of a pair
constexpr int AXP_SPREAD = 4 * AX_SMS;  // CTAs of a short list

// One CTA per primitive pair (item.q = pair, item.a = primitive pair kp).  With A and B on the z
// axis the expansion along z is the E recursion with P - A = zeta_b R / zeta, P - B = -zeta_a R / zeta,
// and across it Laguerre's: g[q][v] = sum_{ja, jb} a_ja a_jb tau(M, s, q) zeta^-(s+q+M) E[l_a - m_a - 2 ja]
// [l_b - m_b - 2 jb][v], s = ja + jb (+ min(m_a, m_b) for the order |m_a - m_b|); the (q, v) of one
// degree n then go over to (k, l = n - 2k).  One warp per half row.  3.8e4 FP64 instructions per
// (ii) pair against 3.5e5 for the matrix form's H: 7.0 -> 1.36 ms for 8,192 pairs.
__global__ void __launch_bounds__(AXP_THREADS) axial_pair_kernel(const AxPair* __restrict__ pairs,
                                                                 const WorkItem* __restrict__ items,
                                                                 const DShell* __restrict__ sh,
                                                                 const double* __restrict__ exps,
                                                                 const double* __restrict__ ncoef,
                                                                 double* __restrict__ ws, int solid) {
    __shared__ double E[(LMAX + 1) * (LMAX + 1)][AXP_NV + 1];
    __shared__ double zpow[32];
    __shared__ double g[AXP_THREADS / 32][8][AXP_NV];
    __shared__ double wt[AXP_THREADS / 32][16][8];  // weights of one half row: (ja, jb), q
    __shared__ double pw[2 * WIG_NP];
    __shared__ double s_pref;
    const WorkItem it = items[blockIdx.x];
    const AxPair pr = pairs[it.q];
    const DShell sa = sh[pr.sa], sb = sh[pr.sb];
    const int la = pr.la, lb = pr.lb, L = la + lb, kp = it.a, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ia = kp / sb.K, ib = kp - ia * sb.K;
    const double za = exps[sa.prim_off + ia], zb = exps[sb.prim_off + ib], zp = za + zb;
    const double AB[3] = {sb.A[0] - sa.A[0], sb.A[1] - sa.A[1], sb.A[2] - sa.A[2]};
    // Each of the serial preparations in a warp of its own: in all four they took half of the FP64
    // issues of a (dd) pair (36,697 primitive pairs 1.54 -> 0.71 ms)
    if (warp == 0) {  // z expansion, lanes over v
        double n[3];
        const double oz = 1.0 / zp;
        double R = ax_unit3(AB, n);
        if (za * zb * oz * R * R > 800.0) R = 0.0;  // the prefactor is 0: no power of R may make that NaN
        const double PA = zb * R * oz, PB = -za * R * oz, oo2p = 0.5 * oz;
        const int v = lane;
        if (v <= L + 1) E[0][min(v, AXP_NV)] = v == 0 ? 1.0 : 0.0;
        __syncwarp();
        for (int i = 0; i <= la; ++i)
            for (int j = i ? 0 : 1; j <= lb; ++j) {
                const double* p = j ? E[i * (lb + 1) + j - 1] : E[(i - 1) * (lb + 1)];
                const double x = j ? PB : PA;
                if (v <= L) {
                    double t = x * p[v];
                    if (v > 0) t += oo2p * p[v - 1];
                    if (v < L) t += (v + 1) * p[v + 1];
                    E[i * (lb + 1) + j][v] = t;
                }
                __syncwarp();
            }
    } else if (warp == 1) {
        double* info = ws + pr.info_off + 4 * (int64_t)kp;
        if (lane < 3 && blockIdx.y == 0) {
            info[1 + lane] = (za * sh[pr.sa].A[lane] + zb * sh[pr.sb].A[lane]) / zp;
        } else if (lane == 3 && blockIdx.y == 0) {
            info[0] = zp;
        } else if (lane == 4) {  // zeta^-(s+q+M), s + q + M <= L
            const double oz = 1.0 / zp;
            double p = 1.0;
            for (int i = 0; i <= L; ++i) {
                zpow[i] = p;
                p *= oz;
            }
        }
    } else if (warp == 2) {
        const double R2 = AB[0] * AB[0] + AB[1] * AB[1] + AB[2] * AB[2];
        if (lane == 0) s_pref = exp(-za * zb / zp * R2) * ncoef[sa.prim_off + ia] * ncoef[sb.prim_off + ib];
    } else if (kp == 0 && blockIdx.y == 0) {  // the pair's rotations
        double n[3], F[9], cp, sp, st, h[2];
        ax_unit3(AB, n);
        frame_of(n, F, cp, sp, st);
        double* rot = ws + pr.rot_off;
        const int lm = max(la, lb);
        ax_half(n[2], -st, h[0], h[1]);
        if (lane < 2) {
            wigner_powers(lm, lane ? h[1] : h[0], pw + lane * WIG_NP);
        } else if (lane == 2) {
            for (int i = 0; i < 9; ++i) rot[i] = F[i];
            double c = 1.0, s = 0.0;
            for (int m = 0; m <= LMAX; ++m) {
                rot[AX_ROT_CS + 2 * m] = c;
                rot[AX_ROT_CS + 2 * m + 1] = s;
                const double cn = c * cp - s * sp;
                s = c * sp + s * cp;
                c = cn;
            }
        }
        __syncwarp();
        for (int i = lane; i < wigner_chains(lm); i += 32)
            wigner_chain(i, lm, n[2], pw, rot + AX_ROT_C, rot + AX_ROT_C + ax_co(lm + 1));
    }
    __syncthreads();
    const double pref = s_pref;
    const AxClass cl = c_ax.cls[pr.cls];
    const AxFn* fa0 = c_ax.fns + c_ax.shell[la][solid].fn0;
    const AxFn* fb0 = c_ax.fns + c_ax.shell[lb][solid].fn0;
    double* h = ws + pr.h_off + (int64_t)kp * cl.nh;
    for (int r = blockIdx.y * (AXP_THREADS / 32) + warp; r < cl.nhalf; r += gridDim.y * (AXP_THREADS / 32)) {
        const AxHalf hr = c_ax.halves[cl.half0 + r];
        const AxFn &fa = fa0[hr.fa], &fb = fb0[hr.fb];
        const int ma = fa.m, mb = fb.m, M = hr.M;
        const int na = (la - ma) / 2, nb = (lb - mb) / 2, s0 = hr.slot ? min(ma, mb) : 0;
        const int nq = (L - M) / 2 + 1;  // q = 0 .. nq - 1, v = 0 .. L - M - 2q
        const double cf = pref * (ma && mb ? 0.5 : 1.0);
        // weights of the terms, then the sums over them for the pairs (q, v) that occur
        for (int e = lane; e < (na + 1) * 32; e += 32) {
            const int ja = e >> 5, jb = e >> 3 & 3, q = e & 7, s = ja + jb + s0;
            if (jb <= nb && q <= s)
                wt[warp][4 * ja + jb][q] =
                    cf * fa.alpha[ja] * fb.alpha[jb] * (__ldg(c_ax.tau + (M * 8 + s) * 8 + q) * zpow[s + q + M]);
        }
        __syncwarp();
        const int npair = nq * (L - M + 2 - nq);  // sum over q of L - M - 2q + 1
        for (int e = lane; e < npair; e += 32) {
            int q = 0, v = e;
            for (int nv = L - M + 1; v >= nv; nv -= 2, ++q) v -= nv;
            double t = 0.0;
            for (int ja = 0; ja <= na; ++ja)
                for (int jb = max(0, q - s0 - ja); jb <= nb; ++jb)
                    t = fma(wt[warp][4 * ja + jb][q], E[(la - ma - 2 * ja) * (lb + 1) + lb - mb - 2 * jb][v], t);
            g[warp][q][v] = t;
        }
        __syncwarp();
        // entries (l, k), l = M .. L, k = 0 .. (L - l) / 2, of degree n = 2k + l
        double* hp = h + hr.hoff;
        const int cnt = (r + 1 < cl.nhalf ? c_ax.halves[cl.half0 + r + 1].hoff : cl.nh) - hr.hoff;
        for (int e = lane; e < cnt; e += 32) {
            int l = M, k = e;
            for (int nk; k >= (nk = (L - l) / 2 + 1); ++l) k -= nk;
            const int n = 2 * k + l, nn = (n - M) / 2 + 1;
            const double* V = c_ax.vinv + __ldg(c_ax.vinv_off + n * AX_NL + M) + k * nn;
            double t = 0.0;
            for (int q = 0; q < nn; ++q) t = fma(__ldg(V + q), g[warp][q][n - M - 2 * q], t);
            hp[e] = pr.sign && (l & 1) ? -t : t;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ rotation blocks

// One CTA per primitive quartet (item.q, item.a = kp kket + kq): from the half angles about y and the
// phases of the table, the Y blocks of the bra rotation and of the rotation PQ -> CD, whose chains
// share the lanes, then the latter's full blocks (or its factors).  One warp where it holds all
// chains at once (L <= 4 on both sides), else two.  FP64 issue and the latency of a few dependent steps
// bound it: Boys values and tables of 1,024 contracted (ff|ff), K = 1..5 (85,000 primitive quartets), 2.61 ms
// with two warps whose sides took turns, 2.13 with the chains in one range, 1.56 with the half angles and
// 1.44 with the phases from axial_boys_kernel.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) axial_wigner_kernel(const AxQuartet* __restrict__ qd,
                                                               const WorkItem* __restrict__ items, int lmax,
                                                               double* __restrict__ ws) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double pw[2][2 * WIG_NP], ph[4 * AX_NL];  // ph: cos, sin of m a, then of m b: 4 (Lk + 1)
    double* C = sm;
    double* S = C + ax_co(lmax + 1);
    const WorkItem it = items[blockIdx.x];
    const AxQuartet q = qd[it.q];
    double* tab = ws + q.tab_off + (int64_t)it.a * q.tab_stride;
    const int tid = threadIdx.x, Lb = q.Lb, Lk = q.Lk;
    if (tid < 4) {  // powers for the bra (0, 1) and ket rotation (2, 3)
        const int side = tid >> 1;
        wigner_powers(side ? Lk : Lb, tab[4 * side + (tid & 1)], pw[side] + (tid & 1) * WIG_NP);
    }
    double* D = tab + ax_t_d(Lb, Lk);
    if (q.full)
        for (int i = tid; i < 4 * (Lk + 1); i += THREADS) ph[i] = D[i];
    __syncthreads();
    const int nb = wigner_chains(Lb), nk = wigner_chains(Lk);
    double* tc = tab + ax_t_c(Lb, Lk);
    for (int i = tid; i < nb + nk; i += THREADS) {
        const bool ket = i >= nb;
        const double ch = tab[ket ? 4 : 0], sh = tab[ket ? 5 : 1];
        wigner_chain(ket ? i - nb : i, ket ? Lk : Lb, (ch - sh) * (ch + sh), pw[ket], ket ? C : tc,
                     ket ? S : tc + ax_co(Lb + 1));
    }
    __syncthreads();
    if (q.full) {
        full_blocks(Lk, ph, ph + 2 * (Lk + 1), C, S, D, tid, THREADS);
    } else {
        const int nc = ax_co(Lk + 1), ns = ax_so(Lk + 1), np = 4 * (Lk + 1);
        for (int i = tid; i < nc; i += THREADS) D[np + i] = C[i];
        for (int i = tid; i < ns; i += THREADS) D[np + nc + i] = S[i];
    }
}

// ------------------------------------------------------------------ main kernel

__device__ __host__ inline int ax_nk(int L, int l) { return (L - l) / 2 + 1; }

// Shared memory (doubles) of the main kernel: h of 8 half rows, S (pyr(Lk) x 8), X (pyr(Lk) x 16),
// and the tables, where T and the bra blocks are replaced by the ket blocks.
__host__ __device__ inline int ax_count(int L) {  // (k, l) pairs, 2k + l <= L
    int n = 0;
    for (int l = 0; l <= L; ++l) n += ax_nk(L, l);
    return n;
}

// T tasks of one (l', M') for the lane's half row: all k' < NK.
template <int NK>
__device__ __forceinline__ void t_task(int lp, int Mp, int Lb, int lo, int M, const double* __restrict__ hs,
                                       const int* __restrict__ hpre, const int* __restrict__ tinfo,
                                       const double* __restrict__ T, const double* __restrict__ tc, double* __restrict__ sc_out,
                                       double* __restrict__ ss_out) {
    const double* ts = tc + ax_co(Lb + 1);
    double sc[NK], ss[NK];
#pragma unroll
    for (int j = 0; j < NK; ++j) sc[j] = ss[j] = 0.0;
    for (int l = Lb; l >= max(lo, Mp); --l) {
        const int nk = ax_nk(Lb, l), info = tinfo[l * AX_NL + lp];
        const double* t = T + (info >> 8) + Mp * (info & 255);
        const double* h = hs + hpre[l] * AX_NR;
        const double c = l >= M ? __ldg(tc + ax_co(l) + Mp * (l + 1) + M) : 0.0;
        const double s = l >= M && M && Mp ? __ldg(ts + ax_so(l) + (Mp - 1) * l + M - 1) : 0.0;
        double I[NK];
#pragma unroll
        for (int j = 0; j < NK; ++j) I[j] = 0.0;
        for (int k = 0; k < nk; ++k) {
            const double hk = h[k * AX_NR];
#pragma unroll
            for (int j = 0; j < NK; ++j) I[j] = fma(hk, t[k + j], I[j]);
        }
#pragma unroll
        for (int j = 0; j < NK; ++j) {
            sc[j] = fma(c, I[j], sc[j]);
            ss[j] = fma(s, I[j], ss[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        sc_out[j * AX_NR] = sc[j];
        if (Mp) ss_out[j * AX_NR] = ss[j];
    }
}

// Rotation tasks of one (l, M'') for the lane's half row: all k < NK, both members.
template <int NK>
__device__ __forceinline__ void r_task(int l, int mm, int mtop, bool first, double cM, double sM,
                                       const double* __restrict__ D, const double* __restrict__ SC,
                                       const double* __restrict__ SS, double* __restrict__ X) {
    double ra[NK], rb[NK];
#pragma unroll
    for (int j = 0; j < NK; ++j) ra[j] = rb[j] = 0.0;
    const double* d = D + mm * (2 * l + 1) + l;
    {
        const double a = d[0];
#pragma unroll
        for (int j = 0; j < NK; ++j) ra[j] = a * SC[j * AX_NR];
    }
    for (int m = 1; m <= mtop; ++m) {
        const double a = d[m], b = d[-m];
        const double* sc = SC + m * NK * AX_NR;
        const double* ss = SS + (m - 1) * NK * AX_NR;
#pragma unroll
        for (int j = 0; j < NK; ++j) {
            ra[j] = fma(a, sc[j * AX_NR], ra[j]);
            rb[j] = fma(b, ss[j * AX_NR], rb[j]);
        }
    }
    double* x = X + mm * NK * 2 * AX_NR;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        double2 v = make_double2(cM * ra[j] - sM * rb[j], sM * ra[j] + cM * rb[j]);
        double2* p = reinterpret_cast<double2*>(x + j * 2 * AX_NR);
        if (!first) {
            const double2 o = *p;
            v.x += o.x;
            v.y += o.y;
        }
        *p = v;
    }
}

// The same for a far primitive quartet (AX_FAR): k = k' = 0, 3 FMAs per (l, l', M') instead of
// (nk + 2) nk'.  With centers in a 20-bohr cube and exponents of 0.05 to 20 half of the primitive
// quartets are far: main kernel 12.5 -> 9.65 ms for 2,048 (ii|ii), 72.0 -> 45.4 ms for 200 mixed
// quartets with K = 1..5; within 6 bohr, where few are far, it costs nothing.
__device__ __forceinline__ void t_far(int lp, int Mp, int Lb, int lo, int M, const double* __restrict__ hs,
                                      const int* __restrict__ hpre, const int* __restrict__ tinfo,
                                      const double* __restrict__ T, const double* __restrict__ tc, double* __restrict__ sc_out,
                                      double* __restrict__ ss_out) {
    const double* ts = tc + ax_co(Lb + 1);
    double sc = 0.0, ss = 0.0;
    for (int l = Lb; l >= max(lo, Mp); --l) {
        const int info = tinfo[l * AX_NL + lp];
        const double I = hs[hpre[l] * AX_NR] * T[(info >> 8) + Mp * (info & 255)];
        const double c = l >= M ? __ldg(tc + ax_co(l) + Mp * (l + 1) + M) : 0.0;
        const double s = l >= M && M && Mp ? __ldg(ts + ax_so(l) + (Mp - 1) * l + M - 1) : 0.0;
        sc = fma(c, I, sc);
        ss = fma(s, I, ss);
    }
    *sc_out = sc;
    if (Mp) *ss_out = ss;
}

__device__ __forceinline__ void r_far(int l, int mm, int mtop, int nk, bool first, double cM, double sM,
                                      const double* __restrict__ D, const double* __restrict__ SC,
                                      const double* __restrict__ SS, double* __restrict__ X) {
    const double* d = D + mm * (2 * l + 1) + l;
    double ra = d[0] * SC[0], rb = 0.0;
    for (int m = 1; m <= mtop; ++m) {
        ra = fma(d[m], SC[m * nk * AX_NR], ra);
        rb = fma(d[-m], SS[(m - 1) * nk * AX_NR], rb);
    }
    double2 v = make_double2(cM * ra - sM * rb, sM * ra + cM * rb);
    double2* p = reinterpret_cast<double2*>(X + mm * nk * 2 * AX_NR);
    if (!first) {
        const double2 o = *p;
        v.x += o.x;
        v.y += o.y;
    }
    *p = v;
}

// One CTA per (quartet item.q, half rows item.a .. item.a + item.b - 1 of the bra class, part item.c
// of the ket primitives; 200 mixed quartets with K = 1..5: 42.9 -> 19.6 ms with the parts).  Lanes are
// the 8 half rows (then the 16 rows: cosine, sine), so every table value is a broadcast and
// every operand row one conflict-free shared access; groups of tasks are taken from shared
// counters, the longest first.  Every stage is bound by the FP64 pipe, which takes a warp instruction
// in 16 cycles: 100,000 of them per (ii|ii) quartet within 2 bohr, where none is far, 773 us of one SM or
// 10.4 ms for 2,048 quartets (measured 11.3, with 24 of 32 lanes filled), and 70,600 in a 20-bohr cube,
// 7.4 ms (8.4, with 22).
// KM: the largest k range, Lk / 2 + 1, that the group's shared memory admits.
template <int THREADS, int MINB, int KM>
__global__ void __launch_bounds__(THREADS, MINB) axial_main_kernel(const AxQuartet* __restrict__ qd,
                                                                   const AxPair* __restrict__ pairs,
                                                                   const WorkItem* __restrict__ items,
                                                                   const double* __restrict__ ws, double* wso,
                                                                   double* out) {
    extern __shared__ __align__(16) double sm[];
    static_assert(__alignof__(sm) >= alignof(double2), "r_task and r_far take X's entries in pairs");
    __shared__ int tinfo[AX_NL * AX_NL];
    __shared__ int hpre[AX_NL + 1], scp[AX_NL + 1], ssp[AX_NL + 1], xp[AX_NL + 1];
    __shared__ int ctr[3];
    __shared__ unsigned farw[LX_KMAX * LX_KMAX / 32];  // far flags of the primitives of one kq
    __shared__ double cg[AX_NR][2];
    __shared__ AxHalf hr[AX_NR];
    // the next group's launch (launch_axial_main) may fill the SMs once every CTA of this one runs
    asm volatile("griddepcontrol.launch_dependents;");
    const WorkItem it = items[blockIdx.x];
    const AxQuartet q = qd[it.q];
    const AxPair pb = pairs[q.pb], pk = pairs[q.pk];
    const int Lb = q.Lb, Lk = q.Lk, tid = threadIdx.x, lane = tid & 31;
    const AxClass cb = c_ax.cls[q.cb], ck = c_ax.cls[q.ck];
    const int pair_id = Lb * AX_NL + Lk;
    if (tid == 0) {
        int a = 0, b = 0, c = 0, d = 0;
        for (int l = 0; l <= AX_NL; ++l) {
            hpre[l] = a;
            scp[l] = b;
            ssp[l] = c;
            xp[l] = d;
            if (l <= Lb) a += ax_nk(Lb, l);
            if (l <= Lk) {
                const int n = ax_nk(Lk, l);
                b += n * (l + 1);
                c += n * l;
                d += n * (2 * l + 1);
            }
        }
        ctr[0] = ctr[1] = ctr[2] = 0;
    }
    if (tid >= 32 && tid < 32 + AX_NR) {
        const int r = tid - 32;
        AxHalf v{0, 0, 0, 0, -1, -1, 0};
        if (r < it.b) v = c_ax.halves[cb.half0 + it.a + r];
        hr[r] = v;
    }
    for (int i = tid; i < AX_NL * AX_NL; i += THREADS) tinfo[i] = c_ax.tinfo[pair_id * AX_NL * AX_NL + i];
    __syncthreads();
    const int nh = hpre[Lb + 1], nsc = scp[Lk + 1], nx = xp[Lk + 1];
    double* hs = sm;                      // nh x 8
    double* SC = hs + nh * AX_NR;         // pyr(Lk) x 8: cosine part, then sine part
    double* SS = SC + nsc * AX_NR;
    double* X = SC + nx * AX_NR;          // pyr(Lk) x 16
    double* T = X + nx * 2 * AX_NR;       // T and B Z^L, replaced by the ket blocks
    double* D = T;
    const int t0 = c_ax.tent_off[pair_id], nT = c_ax.tent_off[pair_id + 1] - t0;
    double* BZ = T + nT;
    const int lo = hr[0].M;  // half rows are ordered by M
    const int r8 = lane & 7, sub = lane >> 3;
    const int Mr = hr[r8].M;
    const int tt0 = c_ax.task_t_off[pair_id], ntt = (c_ax.task_t_off[pair_id + 1] - tt0) / 4;
    const int tr0 = c_ax.task_r_off[Lk], ntr = (c_ax.task_r_off[Lk + 1] - tr0) / 4;
    const int ncd = q.ncd;
    double* O = it.c ? wso + q.part_off + (int64_t)(it.c - 1) * q.nab * ncd : out + q.out_off;
    const int kq0 = (int)((int64_t)it.c * q.kket / q.nsplit), kq1 = (int)((int64_t)(it.c + 1) * q.kket / q.nsplit);

    for (int kq = kq0; kq < kq1; ++kq) {
        for (int i = tid; i < (q.kbra + 31) / 32 * 32; i += THREADS) {
            const bool f = i < q.kbra && ws[q.tab_off + (int64_t)(i * q.kket + kq) * q.tab_stride + AX_T_FAR] != 0.0;
            const unsigned m = __ballot_sync(0xffffffffu, f);
            if (lane == 0) farw[i >> 5] = m;
        }
        __syncthreads();
        // near primitives first: a far one only adds to the k' = 0 entries of X, which are all that the
        // ket transform reads if none is near
        int done = 0, near = 0;
        for (int kpp = 0; kpp < 2 * q.kbra; ++kpp) {
            const int kp = kpp < q.kbra ? kpp : kpp - q.kbra;
            const bool far = kpp >= q.kbra;
            if ((farw[kp >> 5] >> (kp & 31) & 1u) != (far ? 1u : 0u)) continue;
            near += !far;
            const double* tab = ws + q.tab_off + (int64_t)(kp * q.kket + kq) * q.tab_stride;
            const double* h = ws + pb.h_off + (int64_t)kp * pb.nh;
            for (int i = tid; i < ax_bz(Lb + Lk + 1); i += THREADS) BZ[i] = tab[AX_T_BZ + i];
            const double* tc = tab + ax_t_c(Lb, Lk);
            for (int i = tid; i < nh * AX_NR; i += THREADS) {
                const int r = i & (AX_NR - 1), e = i / AX_NR, e0 = hpre[hr[r].M];
                hs[i] = r < it.b && e >= e0 ? h[hr[r].hoff + e - e0] : 0.0;
            }
            if (tid < 2 * AX_NR) cg[tid >> 1][tid & 1] = tab[ax_t_cg(Lb, Lk) + 2 * hr[tid >> 1].M + (tid & 1)];
            if (tid == 0) ctr[1] = 0;
            __syncthreads();
            for (int i = tid; i < nT; i += THREADS) {
                const int e = __ldg(c_ax.tent + t0 + i), n = e >> 23 & 15;
                const double* gp = c_ax.g + (e & 0x3FFF);
                const double* bz = BZ + ((e >> 14) & 0x1FF);
                if (far) {
                    if (e >> 27) T[i] = __ldg(gp + n - 1) * bz[n - 1];
                    continue;
                }
                double t = 0.0;
                for (int s = 0; s < n; ++s) t = fma(__ldg(gp + s), bz[s], t);
                T[i] = t;
            }
            __syncthreads();
            for (;;) {
                int gi = 0;
                if (lane == 0) gi = atomicAdd(&ctr[0], 1);
                gi = __shfl_sync(0xffffffffu, gi, 0);
                if (gi >= ntt) break;
                const int task = __ldg(c_ax.task_t + tt0 + 4 * gi + sub);
                if (task < 0) continue;
                const int lp = task & 255, Mp = task >> 8, nk = ax_nk(Lk, lp);
                double* so = SC + (scp[lp] + Mp * nk) * AX_NR + r8;
                double* zo = SS + (ssp[lp] + (Mp - 1) * nk) * AX_NR + r8;
                if (far) {
                    t_far(lp, Mp, Lb, lo, Mr, hs + r8, hpre, tinfo, T, tc, so, zo);
                    continue;
                }
#define AX_T(N)                                                                                    \
    case N:                                                                                        \
        if constexpr (N <= KM) t_task<N>(lp, Mp, Lb, lo, Mr, hs + r8, hpre, tinfo, T, tc, so, zo);                    \
        break;
                switch (nk) { AX_T(1) AX_T(2) AX_T(3) AX_T(4) AX_T(5) AX_T(6) AX_T(7) AX_T(8) }
#undef AX_T
            }
            __syncthreads();
            if (tid == 0) ctr[0] = 0;
            const double* td = tab + ax_t_d(Lb, Lk);
            if (q.full) {
                for (int i = tid; i < ax_do(Lk + 1); i += THREADS) D[i] = td[i];
            } else {
                const double* C = td + 4 * (Lk + 1);
                full_blocks(Lk, td, td + 2 * (Lk + 1), C, C + ax_co(Lk + 1), D, tid, THREADS);
            }
            __syncthreads();
            const bool first = done++ == 0;
            const double cM = cg[r8][0], sM = cg[r8][1];
            for (;;) {
                int gi = 0;
                if (lane == 0) gi = atomicAdd(&ctr[1], 1);
                gi = __shfl_sync(0xffffffffu, gi, 0);
                if (gi >= ntr) break;
                const int task = __ldg(c_ax.task_r + tr0 + 4 * gi + sub);
                if (task < 0) continue;
                const int l = task & 255, mm = task >> 8, nk = ax_nk(Lk, l), mtop = min(l, Lb);
                if (far) {
                    r_far(l, mm, mtop, nk, first, cM, sM, D + ax_do(l), SC + scp[l] * AX_NR + r8,
                          SS + ssp[l] * AX_NR + r8, X + xp[l] * 2 * AX_NR + 2 * r8);
                    continue;
                }
#define AX_R(N)                                                                                    \
    case N:                                                                                        \
        if constexpr (N <= KM) r_task<N>(l, mm, mtop, first, cM, sM, D + ax_do(l), SC + scp[l] * AX_NR + r8,              \
                  SS + ssp[l] * AX_NR + r8, X + xp[l] * 2 * AX_NR + 2 * r8);                       \
        break;
                switch (nk) { AX_R(1) AX_R(2) AX_R(3) AX_R(4) AX_R(5) AX_R(6) AX_R(7) AX_R(8) }
#undef AX_R
            }
            __syncthreads();
        }
        // ket transform: half columns, lanes over 16 rows
        const double* hk = ws + pk.h_off + (int64_t)kq * pk.nh;
        const int row = lane & 15, half = lane >> 4;
        const int vrow = row & 1 ? hr[row >> 1].vs : hr[row >> 1].vc;
        for (;;) {
            int gi = 0;
            if (lane == 0) gi = atomicAdd(&ctr[2], 1);
            gi = __shfl_sync(0xffffffffu, gi, 0);
            const int c = 2 * gi + half;
            if (2 * gi >= ck.nhalf) break;
            if (c >= ck.nhalf) continue;
            const AxHalf hc = c_ax.halves[ck.half0 + c];
            const double* hv = hk + hc.hoff;
            const int M = hc.M;
            double vc = 0.0, vs = 0.0;
            for (int l = M; l <= Lk; ++l) {
                const int nk = ax_nk(Lk, l);
                const double* xc = X + (xp[l] + (l + M) * nk) * 2 * AX_NR + row;
                const double* xs = X + (xp[l] + (l - M) * nk) * 2 * AX_NR + row;
                for (int k = 0; k < (near ? nk : 1); ++k) {
                    const double w = __ldg(hv + k);
                    vc = fma(w, xc[k * 2 * AX_NR], vc);
                    vs = fma(w, xs[k * 2 * AX_NR], vs);
                }
                hv += nk;
            }
            if (vrow >= 0) {
                double* o = O + (int64_t)vrow * ncd;
                o[hc.vc] = kq > kq0 ? o[hc.vc] + vc : vc;
                if (hc.vs >= 0) o[hc.vs] = kq > kq0 ? o[hc.vs] + vs : vs;
            }
        }
        __syncthreads();
        if (tid == 0) ctr[2] = 0;
    }
    // ends after the groups before it, so that what follows in the stream sees them all
    if (tid == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------------------------ to the lab frame

// Both function indices (n1 x n2, item.q = quartet) of one side: the cosine/sine members of the
// half rows are combined into products of functions, each index is rotated from the pair's
// frame to the lab (transposed Y, then z) and, for Cartesian output, expanded over monomials.
// SIDE = 1: ket indices, `lanes` rows from item.a; SIDE = 0: bra indices, `lanes` columns from item.a.
// Bound by the FP64 pipe: 37,000 warp instructions per (ii|ii) quartet for both sides, 286 us of one SM
// or 3.85 ms for 2,048 quartets (measured 4.23, with 27 of 32 lanes filled; 200 Cartesian ones 14.0).  Neighbouring tasks of
// a warp take the same function of neighbouring lines, so that loop lengths do not differ within a
// warp (4.47 and 20.2 ms with neighbouring functions of one line); a tile of 16 lanes keeps the
// accesses of a half warp in 128 bytes and four CTAs on an SM (32 lanes: 5.64 ms).
template <int SIDE, int THREADS>
__global__ void __launch_bounds__(THREADS) axial_rotate_kernel(const AxQuartet* __restrict__ qd,
                                                                   const AxPair* __restrict__ pairs,
                                                                   const WorkItem* __restrict__ items, int lanes,
                                                                   const double* __restrict__ ws,
                                                                   double* __restrict__ out, int solid) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double rot[AX_ROT_C + 204 + 140];
    const WorkItem it = items[blockIdx.x];
    const AxQuartet q = qd[it.q];
    const AxPair pr = pairs[SIDE ? q.pk : q.pb];
    const int tid = threadIdx.x, ld = lanes + 1, lane = tid % lanes, t0 = tid / lanes, nt = THREADS / lanes;
    const AxShell s1 = c_ax.shell[pr.la][solid], s2 = c_ax.shell[pr.lb][solid];
    const AxFn *f1 = c_ax.fns + s1.fn0, *f2 = c_ax.fns + s2.fn0;
    const int n1 = s1.ntot, n2 = s2.ntot, n = n1 * n2, lm = max(pr.la, pr.lb);
    const int live = min(lanes, (SIDE ? q.nab : q.ncd) - it.a);
    double* a = sm;
    double* b = sm + n * ld;
    double* O = out + q.out_off;
    for (int i = tid; i < ax_rot_size(lm); i += THREADS) rot[i] = ws[pr.rot_off + i];
    const double *cs = rot + AX_ROT_CS, *C = rot + AX_ROT_C, *S = C + ax_co(lm + 1);
    if (SIDE) {
        for (int i = tid; i < live * n; i += THREADS) {
            const int r = i / n, c = i - r * n;
            double v = O[(int64_t)(it.a + r) * n + c];
            for (int p = 0; p + 1 < q.nsplit; ++p) v += ws[q.part_off + ((int64_t)p * q.nab + it.a + r) * n + c];
            a[c * ld + r] = v;
        }
    } else {
        if (lane < live)
            for (int r = t0; r < n; r += nt) a[r * ld + lane] = O[(int64_t)r * q.ncd + it.a + lane];
    }
    __syncthreads();
    if (lane < live) {
        for (int i = t0; i < s1.nfn * s2.nfn; i += nt) {
            const AxFn &x = f1[i / s2.nfn], &y = f2[i % s2.nfn];
            if (!x.m || !y.m) continue;
            double* pp = a + (x.plus * n2 + y.plus) * ld + lane;
            double* mm = a + (x.minus * n2 + y.minus) * ld + lane;
            double* mp = a + (x.minus * n2 + y.plus) * ld + lane;
            double* pm = a + (x.plus * n2 + y.minus) * ld + lane;
            const double c1 = *pp, c2 = *mm, z1 = *mp, z2 = x.m == y.m ? 0.0 : (x.m > y.m ? *pm : -*pm);
            *pp = c1 + c2;
            *mm = c2 - c1;
            *mp = z1 + z2;
            *pm = z1 - z2;
        }
    }
    __syncthreads();
    // one index: element (o, f) at o * so + f * sf; src -> dst
    auto turn = [&](const double* src, double* dst, const AxFn* fn, int nfn, int no, int so, int sf) {
        if (lane < live)
            for (int i = t0; i < no * nfn; i += nt) {
                const int f = i / no, o = i - f * no;
                const AxFn& F = fn[f];
                const int lam = F.lam, m = F.m, mid = F.plus - m;
                const double* v = src + (o * so + mid * sf) * ld + lane;
                const double* Cl = C + ax_co(lam) + m;
                const double* Sl = S + ax_so(lam) + m - 1;
                double c = Cl[0] * v[0], s = 0.0;
                for (int k = 1; k <= lam; ++k) c = fma(Cl[k * (lam + 1)], v[k * sf * ld], c);
                double* w = dst + o * so * ld + lane;
                if (m) {
                    for (int k = 1; k <= lam; ++k) s = fma(Sl[(k - 1) * lam], v[-k * sf * ld], s);
                    const double cm = cs[2 * m], sn = cs[2 * m + 1];
                    w[F.plus * sf * ld] = cm * c - sn * s;
                    w[F.minus * sf * ld] = sn * c + cm * s;
                } else {
                    w[F.plus * sf * ld] = c;
                }
            }
        __syncthreads();
    };
    auto expand = [&](const double* src, double* dst, const AxShell& s, int no, int so, int sf) {
        if (lane < live)
            for (int i = t0; i < no * s.ntot; i += nt) {
                const int c = i / no, o = i - c * no;
                const int b0 = __ldg(c_ax.wc_row + s.wc0 + c), b1 = __ldg(c_ax.wc_row + s.wc0 + c + 1);
                double t = 0.0;
                for (int e = b0; e < b1; ++e)
                    t = fma(__ldg(c_ax.wc_val + e), src[(o * so + __ldg(c_ax.wc_idx + e) * sf) * ld + lane], t);
                dst[(o * so + c * sf) * ld + lane] = t;
            }
        __syncthreads();
    };
    turn(a, b, f2, s2.nfn, n1, n2, 1);
    turn(b, a, f1, s1.nfn, n2, 1, n2);
    if (!solid) {
        expand(a, b, s2, n1, n2, 1);
        expand(b, a, s1, n2, 1, n2);
    }
    if (SIDE) {
        for (int i = tid; i < live * n; i += THREADS) {
            const int r = i / n, c = i - r * n;
            O[(int64_t)(it.a + r) * n + c] = a[c * ld + r];
        }
    } else if (lane < live) {
        for (int r = t0; r < n; r += nt) O[(int64_t)r * q.ncd + it.a + lane] = a[r * ld + lane];
    }
}

template <typename V>
cudaError_t upload(const std::vector<V>& v, const V** dst) {
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, sizeof(V) * (v.size() + 1));
    if (e != cudaSuccess) return e;
    if ((e = cudaMemcpy(p, v.data(), sizeof(V) * v.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
    *dst = static_cast<const V*>(p);
    return cudaSuccess;
}

constexpr int AX_SMEM_MAX = 227 * 1024;

}  // namespace

size_t axial_main_smem(int Lb, int Lk) {
    const AxHost& H = axial_tables();
    const int id = Lb * AX_NL + Lk, nT = H.tent_off[id + 1] - H.tent_off[id];
    const int tabs = std::max(nT + ax_bz(Lb + Lk + 1), ax_do(Lk + 1));
    return sizeof(double) * (size_t)(ax_count(Lb) * AX_NR + 3 * pyr(Lk) * AX_NR + tabs);
}

// The groups by shared memory: 1, 2, 3, 4 and 8 CTAs per SM of 512, 256, 256, 256 and 128 threads
// (CTAs that share an SM fill one another's gaps at barriers and table loads; small classes, with
// short stages, want the most warps).  n CTAs fit an SM's 228 KB if each takes 1,024 reserved bytes, 1,456 of
// static arrays and no more than the rest; the other limits are whole KB below that.  (ii|ii) needs
// 113,896 bytes, two per SM with the bra blocks left in global memory: its main kernel 9.65 -> 8.46 ms
// for 2,048 quartets against one CTA of 512 threads; (gg|gg) with 256 threads 4.41 ms for 8,192, with
// 128 5.34.
int axial_bin(int Lb, int Lk) {
    const size_t s = axial_main_smem(Lb, Lk);
    constexpr size_t two = 228 * 1024 / 2 - 1024 - 1456;
    const int bin = s <= 25 * 1024 ? 4 : s <= 54 * 1024 ? 3 : s <= 73 * 1024 ? 2 : s <= two ? 1 : 0;
    return std::min(bin, 8 - (Lk / 2 + 1));  // group b's kernel takes k ranges up to 8 - b
}

cudaError_t init_axial(const AxHost& H) {
    AxDev d{};
    cudaError_t e = cudaSuccess;
    const AxClass* cls = nullptr;
    std::vector<AxClass> c(H.cls, H.cls + (LMAX + 1) * (LMAX + 1) * 2);
    if ((e = upload(H.g, &d.g)) != cudaSuccess || (e = upload(H.vinv, &d.vinv)) != cudaSuccess ||
        (e = upload(H.tau, &d.tau)) != cudaSuccess || (e = upload(H.wig0, &d.wig0)) != cudaSuccess ||
        (e = upload(H.wig, &d.wig)) != cudaSuccess || (e = upload(H.wc_val, &d.wc_val)) != cudaSuccess ||
        (e = upload(H.vinv_off, &d.vinv_off)) != cudaSuccess || (e = upload(H.tent, &d.tent)) != cudaSuccess ||
        (e = upload(H.tent_off, &d.tent_off)) != cudaSuccess || (e = upload(H.tinfo, &d.tinfo)) != cudaSuccess ||
        (e = upload(H.task_t, &d.task_t)) != cudaSuccess || (e = upload(H.task_t_off, &d.task_t_off)) != cudaSuccess ||
        (e = upload(H.task_r, &d.task_r)) != cudaSuccess || (e = upload(H.task_r_off, &d.task_r_off)) != cudaSuccess ||
        (e = upload(H.wc_row, &d.wc_row)) != cudaSuccess || (e = upload(H.wc_idx, &d.wc_idx)) != cudaSuccess ||
        (e = upload(H.fns, &d.fns)) != cudaSuccess || (e = upload(H.halves, &d.halves)) != cudaSuccess ||
        (e = upload(c, &cls)) != cudaSuccess)
        return e;
    d.cls = cls;
    for (int l = 0; l <= LMAX; ++l)
        for (int s = 0; s < 2; ++s) d.shell[l][s] = H.shell[l][s];
    if ((e = cudaMemcpyToSymbol(c_ax, &d, sizeof(d))) != cudaSuccess) return e;
    const void* kernels[] = {(const void*)axial_main_kernel<512, 1, 8>, (const void*)axial_main_kernel<256, 2, 7>,
                             (const void*)axial_main_kernel<256, 3, 6>, (const void*)axial_main_kernel<256, 4, 5>,
                             (const void*)axial_main_kernel<128, 8, 4>,
                             (const void*)axial_rotate_kernel<0, 256>, (const void*)axial_rotate_kernel<1, 256>,
                             (const void*)axial_rotate_kernel<0, 1024>, (const void*)axial_rotate_kernel<1, 1024>};
    for (const void* k : kernels)
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, AX_SMEM_MAX - 8192)) != cudaSuccess)
            return e;
    return cudaSuccess;
}

cudaError_t launch_axial_pair(const AxPair* pairs, const WorkItem* items, int nitems, const DShell* sh,
                              const double* exps, const double* ncoef, double* ws, bool solid, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    // a short list spreads each pair's half rows over several CTAs, each with its own expansion along z:
    // 68 primitive pairs of up to (kk) 296 -> 66 us, 128 of (gg) 38 -> 29 us
    const int ny = std::max(1, std::min(8, AXP_SPREAD / nitems));
    axial_pair_kernel<<<dim3(nitems, ny), AXP_THREADS, 0, st>>>(pairs, items, sh, exps, ncoef, ws, solid ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_axial_wigner(const AxQuartet* qd, const WorkItem* items, int nitems, int lmax, double* ws,
                                cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const size_t smem = sizeof(double) * (size_t)(ax_co(lmax + 1) + ax_so(lmax + 1));
    if (2 * wigner_chains(lmax) <= 32)
        axial_wigner_kernel<32><<<nitems, 32, smem, st>>>(qd, items, lmax, ws);
    else
        axial_wigner_kernel<64><<<nitems, 64, smem, st>>>(qd, items, lmax, ws);
    return cudaGetLastError();
}

// One launch per group of shared-memory sizes.  The groups read what earlier kernels wrote and
// write apart, so a group need not wait for the one before it: it is launched to start once all of
// that one's CTAs run, and fills the SMs that its last, longest CTAs leave idle (7 mixed Cartesian
// quartets, K = 1..2, 0.46 -> 0.35 ms; 200 mixed ones 16.6 -> 16.3).
template <int THREADS, int MINB, int KM>
cudaError_t launch_group(int n, size_t smem, bool overlap, const AxQuartet* qd, const AxPair* pairs, const WorkItem* items,
                         double* ws, double* out, cudaStream_t st) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, axial_main_kernel<THREADS, MINB, KM>, qd, pairs, items, (const double*)ws, ws, out);
}

cudaError_t launch_axial_main(const AxQuartet* qd, const AxPair* pairs, const WorkItem* items, const int* counts,
                              const size_t* smem, double* ws, double* out, cudaStream_t st) {
    bool overlap = false;
    for (int b = 0; b < AX_NBIN; ++b) {
        const int n = counts[b];
        if (n <= 0) continue;
        cudaError_t e;
        switch (b) {
            case 0: e = launch_group<512, 1, 8>(n, smem[b], overlap, qd, pairs, items, ws, out, st); break;
            case 1: e = launch_group<256, 2, 7>(n, smem[b], overlap, qd, pairs, items, ws, out, st); break;
            case 2: e = launch_group<256, 3, 6>(n, smem[b], overlap, qd, pairs, items, ws, out, st); break;
            case 3: e = launch_group<256, 4, 5>(n, smem[b], overlap, qd, pairs, items, ws, out, st); break;
            default: e = launch_group<128, 8, 4>(n, smem[b], overlap, qd, pairs, items, ws, out, st); break;
        }
        if (e != cudaSuccess) return e;
        items += n;
        overlap = true;
    }
    return cudaSuccess;
}

cudaError_t launch_axial_rotate(int side, const AxQuartet* qd, const AxPair* pairs, const WorkItem* items, int nitems,
                                int lanes, size_t smem, const double* ws, double* out, bool solid, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    // at least 32 warps per SM: 256 threads where four CTAs fit, 1,024 otherwise
    const int s = solid ? 1 : 0;
    if (smem <= 54 * 1024) {
        if (side) axial_rotate_kernel<1, 256><<<nitems, 256, smem, st>>>(qd, pairs, items, lanes, ws, out, s);
        else axial_rotate_kernel<0, 256><<<nitems, 256, smem, st>>>(qd, pairs, items, lanes, ws, out, s);
    } else {
        if (side) axial_rotate_kernel<1, 1024><<<nitems, 1024, smem, st>>>(qd, pairs, items, lanes, ws, out, s);
        else axial_rotate_kernel<0, 1024><<<nitems, 1024, smem, st>>>(qd, pairs, items, lanes, ws, out, s);
    }
    return cudaGetLastError();
}

}  // namespace lx
