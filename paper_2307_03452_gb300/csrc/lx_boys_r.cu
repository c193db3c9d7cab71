// Boys function (Eq. boys) and the auxiliary Hermite integrals [r]^(m) (Eq. md1).
//
// Boys: for T < 36, F_mmax(T) from an 8-term Taylor expansion around the nearest point
// of a 0.1-spaced table of F_n(T_k), then the downward recursion
// F_m = (2T F_{m+1} + exp(-T)) / (2m+1); for T >= 36, F_0 = (1/2) sqrt(pi/T) (erf(sqrt T)
// differs from 1 by < 3e-17) and the upward recursion F_{m+1} = ((2m+1) F_m - exp(-T))/(2T).
//
// R: one warp per primitive quartet evaluates [r]^(m) for m = L-1 down to 0 in one shared
// array of pyr(L) doubles, overwriting [r]^(m+1) with [r]^(m) (the paper's in-place
// scheme, Section 3).  A position's inputs, at totals n-1 and n-2 of its n = |r|, lie below it, and
// within level m the positions are processed from the last down to the first: those below a block of
// positions still hold level m+1, and within a block every lane has read before any lane writes.
// In the batch kernel each CTA is that one warp, with shared memory for the chunk's
// largest L, so that as many quartets as shared memory allows run side by side.
#include <cmath>
#include <cstring>
#include <vector>

#include "lx_axial.cuh"
#include "lx_internal.cuh"

namespace lx {

namespace {

__device__ double g_boys[BOYS_NROW * BOYS_NPT];
// One step of Eq. md1 for every Hermite position h = hidx(t, u, v) with t + u + v >= 1,
// lowering the first nonzero direction d of (t, u, v):
//   [r]^(m) = X_d [r - 1_d]^(m+1) + (r_d - 1) [r - 2_d]^(m+1)
// x = hidx(r - 1_d) | hidx(r - 2_d) << 13 | d << 26 (the second position 0 when r_d = 1),
// (z, w) = the FP64 bits of r_d - 1 (low, high word), so that the step is one multiply and one
// FMA with no branch and no integer conversion.
__device__ int4 g_rec[NHERM_TOT];

constexpr double PI = 3.141592653589793238462643383279502884;

__device__ inline void set_status(unsigned* st, unsigned bit) { atomicOr(st, bit); }

// F_m(T) for m = 0..mmax (mmax <= LTOT) into F (any memory), one thread.
__device__ void boys_eval(int mmax, double T, double* F) {
    if (T < BOYS_TMAX) {
        const int k = __double2int_rn(T * (1.0 / BOYS_DT));
        const double d = k * BOYS_DT - T;  // -(T - T_k)
        // F_mmax(T) = sum_j F_{mmax+j}(T_k) (-(T - T_k))^j / j!
        const double* col = g_boys + k;
        double f = 0.0, pw = 1.0;
#pragma unroll
        for (int j = 0; j < BOYS_ORDER; ++j) {
            f += __ldg(col + (mmax + j) * BOYS_NPT) * pw;
            pw *= d / (j + 1);
        }
        F[mmax] = f;
        const double e = exp(-T), twoT = 2.0 * T;
        for (int m = mmax - 1; m >= 0; --m) {
            f = (twoT * f + e) / (2 * m + 1);
            F[m] = f;
        }
    } else {
        double f = 0.5 * sqrt(PI / T);
        F[0] = f;
        const double e = exp(-T), oo2T = 0.5 / T;
        for (int m = 0; m < mmax; ++m) {
            f = ((2 * m + 1) * f - e) * oo2T;
            F[m + 1] = f;
        }
    }
}

// B[m] *= pref (-2 rho)^m for m = 0..L (L <= LTOT < 32), one m per lane: the power is
// taken directly rather than as a running product, which keeps its rounding at one step.
__device__ inline void scale_base(int L, double rho, double pref, double* B, int lane) {
    if (lane <= L) {
        const double pw = pow(2.0 * rho, (double)lane);
        B[lane] *= (lane & 1) ? -pref * pw : pref * pw;
    }
}

// Positions h, h - 32, ..., h - 32 (N - 1) (those >= 1) of one order of Eq. md1: all lanes read their
// sources, then write.
template <int N>
__device__ __forceinline__ void hermite_r_block(int h, double X, double Y, double Z, double* R) {
    int4 e[N];
    double a[N], b[N];
#pragma unroll
    for (int u = 0; u < N; ++u) e[u] = __ldg(&g_rec[max(h - 32 * u, 1)]);
#pragma unroll
    for (int u = 0; u < N; ++u) {
        a[u] = R[e[u].x & 0x1FFF];
        b[u] = R[(e[u].x >> 13) & 0x1FFF];
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < N; ++u) {
        const int d = e[u].x >> 26;
        const double xd = d == 0 ? X : (d == 1 ? Y : Z);
        const double v = fma(__hiloint2double(e[u].w, e[u].z), b[u], xd * a[u]);
        if (h - 32 * u >= 1) R[h - 32 * u] = v;
    }
}

// In-place Eq. md1 on R[pyr(L)] (shared memory), by one warp.  B[m] = [0]^(m), m = 0..L.
// On return R holds [r]^(0).  A position's sources lie in the two shells below its own, so one
// order m is done from the last position down, several positions a lane at once (as many as are
// left fill), and the warp waits once between reading and writing a block.  Bound by the latency of
// a block's loads at 9 warps per SM (L = 24): with a shell at a time, one position a lane and a fifth of
// the lanes idle, 0.69 ms for 4,096 (ii|ii), so 0.39.
__device__ void hermite_r_warp(int L, double X, double Y, double Z, const double* B, double* R, int lane) {
    if (lane == 0) R[0] = B[L];
    __syncwarp();
    for (int m = L - 1; m >= 0; --m) {
        int top = pyr(L - m) - 1;
        for (; top > 96; top -= 128) hermite_r_block<4>(top - lane, X, Y, Z, R);
        for (; top > 32; top -= 64) hermite_r_block<2>(top - lane, X, Y, Z, R);
        if (top >= 1) hermite_r_block<1>(top - lane, X, Y, Z, R);
        if (lane == 0) R[0] = B[m];
        __syncwarp();
    }
}

constexpr int BR_WARPS = 4;  // warps per CTA of the stage entry point

// One more power: (h, l) = x^n as an unevaluated sum -> x^(n+1), so that the chain rounds once, at
// h + l.
__device__ inline void power_step(double x, double& h, double& l) {
    const double p = h * x;
    l = (__double2hiint(p) & 0x7FF00000) == 0x7FF00000 ? 0.0 : fma(l, x, fma(h, x, -p));
    h = p;
}

// [0]^(m) = (-2 rho)^m 2 pi^{5/2} / (zeta_p zeta_q sqrt(zeta_p + zeta_q)) F_m(T), m = 0..L, of each
// primitive quartet (item.q = quartet, item.a = kpq = kp kket + kq), into the first L + 1 entries of
// its [r]^(0).  One thread per primitive quartet: the Boys recursion is serial, with a division
// per order, so in the recursion kernel's warp it took as many FP64 issues for one quartet as here
// for 32.
constexpr int BASE_THREADS = 64;
__global__ void __launch_bounds__(BASE_THREADS) boys_base_kernel(const DQuartet* __restrict__ qd,
                                                                 const DPair* __restrict__ pairs,
                                                                 const WorkItem* __restrict__ items, int nitems,
                                                                 double* __restrict__ ws) {
    const int i = blockIdx.x * BASE_THREADS + threadIdx.x;
    if (i >= nitems) return;
    const WorkItem it = items[i];
    const DQuartet q = qd[it.q];
    const int kp = it.a / q.kket, kq = it.a - kp * q.kket;
    const double* ib = ws + pairs[q.pb].info_off + 4 * (int64_t)kp;
    const double* ik = ws + pairs[q.pk].info_off + 4 * (int64_t)kq;
    const double zp = ib[0], zq = ik[0];
    const double X = ib[1] - ik[1], Y = ib[2] - ik[2], Z = ib[3] - ik[3];
    const double rho = zp * zq / (zp + zq);
    double F[LTOT + 1];
    boys_eval(q.L, rho * (X * X + Y * Y + Z * Z), F);
    const double pref = 2.0 * PI * PI * sqrt(PI) / (zp * zq * sqrt(zp + zq));
    double* out = ws + q.rr_off + (int64_t)it.a * q.nr;
    double h = 1.0, l = 0.0;
    for (int m = 0; m <= q.L; ++m) {
        const double pw = h + l;
        out[m] = F[m] * ((m & 1) ? -pref * pw : pref * pw);
        power_step(2.0 * rho, h, l);
    }
}

// One single-warp CTA per primitive quartet: item.q = quartet, item.a = kpq = kp * kket + kq.  Its
// [0]^(m) are the first L + 1 entries of its [r]^(0) on entry.
__global__ void __launch_bounds__(32) boys_r_kernel(const DQuartet* __restrict__ qd, const DPair* __restrict__ pairs,
                                                    const WorkItem* __restrict__ items, double* __restrict__ ws) {
    extern __shared__ double smem[];
    const int lane = threadIdx.x & 31;
    const WorkItem it = items[blockIdx.x];
    const DQuartet q = qd[it.q];
    const int kpq = it.a;
    const int nr = q.nr;
    double* R = smem;
    double* B = R + nr;
    double* out = ws + q.rr_off + (int64_t)kpq * nr;
    if (lane <= q.L) B[lane] = out[lane];
    const int kp = kpq / q.kket, kq = kpq - kp * q.kket;
    const DPair pb = pairs[q.pb], pk = pairs[q.pk];
    const double* ib = ws + pb.info_off + 4 * (int64_t)kp;
    const double* ik = ws + pk.info_off + 4 * (int64_t)kq;
    const double X = ib[1] - ik[1], Y = ib[2] - ik[2], Z = ib[3] - ik[3];
    __syncwarp();
    hermite_r_warp(q.L, X, Y, Z, B, R, lane);
    for (int r = lane; r < nr; r += 32) out[r] = R[r];
}

// Axial form (lx_axial.cu): the angles of each primitive quartet's frames (item.q, item.a = kp kket +
// kq), as half angles and phases, and its table B_kappa(L) Z^L.  One CTA per `per` of them: first a
// thread each, in one warp for the geometry and in the other for the Boys values, some 300 FP64
// instructions with their divisions either way, then 8 lanes each for the table rows.  FP64 issue
// bounds it (one warp instruction in 16 cycles and SM), so full warps in the first part count: these and
// the rotation blocks of 165,856 primitive quartets of (dd|dd) 2.77 ms with 8 lanes doing alike, 1.32 so;
// `per` = 4 spreads a short list over the SMs (64 of (gg|gg) 52 us).  The
// powers of 2 rho and Z are one chain of products with their errors carried (7 FP64 instructions per
// degree for both; pow takes some 150 per power).
constexpr int AXB_THREADS = 64, AXB_PER = 32, AXB_PER_FEW = 4, AXB_FEW = 4096;
__global__ void __launch_bounds__(AXB_THREADS) axial_boys_kernel(const AxQuartet* __restrict__ qd,
                                                                 const AxPair* __restrict__ pairs,
                                                                 const WorkItem* __restrict__ items, int nitems,
                                                                 int per, double* __restrict__ ws) {
    // B_0(L), the kappa = 1 row from entry 1, Z^L; the second row of the recursion
    __shared__ double f_[AXB_PER][LTOT + 1], row_[AXB_PER][LTOT + 1], z_[AXB_PER][LTOT + 1],
        nxt_[AXB_THREADS / 8][LTOT + 1];
    __shared__ double r2_[AXB_PER];
    __shared__ double* tab_[AXB_PER];
    __shared__ int lt_[AXB_PER];
    const int lane = threadIdx.x & 31, item = blockIdx.x * per + lane;
    const bool boys = threadIdx.x >= 32;
    if (boys) lt_[lane] = -1;
    if (lane < per && item < nitems) {
        const WorkItem it = items[item];
        const AxQuartet& q = qd[it.q];
        const AxPair &pb = pairs[q.pb], &pk = pairs[q.pk];
        const int kp = it.a / q.kket, kq = it.a - kp * q.kket, Lt = q.Lb + q.Lk;
        const double* ib = ws + pb.info_off + 4 * (int64_t)kp;
        const double* ik = ws + pk.info_off + 4 * (int64_t)kq;
        const double *Fb = ws + pb.rot_off, *Fk = ws + pk.rot_off;
        const double zp = ib[0], zq = ik[0];
        const double v[3] = {ib[1] - ik[1], ib[2] - ik[2], ib[3] - ik[3]};
        const double R2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        double* tab = ws + q.tab_off + (int64_t)it.a * q.tab_stride;
        double n[3];
        const double Z = ax_unit3(v, n);
        if (boys) {
            const double rho = zp * zq / (zp + zq), T = rho * R2;
            const double pref = 2.0 * PI * PI * sqrt(PI) / (zp * zq * sqrt(zp + zq));
            double *f = f_[lane], *row = row_[lane], *z = z_[lane];
            boys_eval(Lt, T, f);
            const double ex = exp(-T);
            double ph = 1.0, pl = 0.0, zh = 1.0, zl = 0.0;
            for (int L = 0; L <= Lt; ++L) {
                const double pw = (L & 1 ? -pref : pref) * (ph + pl);
                f[L] *= pw;
                row[L] = pw * ex;
                z[L] = zh + zl;
                power_step(2.0 * rho, ph, pl);
                power_step(Z, zh, zl);
            }
            lt_[lane] = Lt;
            tab_[lane] = tab;
            r2_[lane] = fmin(R2, 1e300);
        } else {
            // bra rotation: PQ in the AB frame (no rotation for P = Q)
            double c = 1.0, s = 0.0, cg = 1.0, sg = 0.0;
            if (Z > 0.0) {
                c = Fb[6] * n[0] + Fb[7] * n[1] + Fb[8] * n[2];
                s = ax_unit(Fb[0] * n[0] + Fb[1] * n[1] + Fb[2] * n[2], Fb[3] * n[0] + Fb[4] * n[1] + Fb[5] * n[2], cg, sg);
            }
            const double nrm = 1.0 / sqrt(c * c + s * s);
            c *= nrm;
            s *= nrm;
            // PQ frame in the lab, and the ket rotation Rm = F_cd F_pq^T = Rz(a) Ry Rz(b)
            double Fp[9], Rm[9];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const double r0 = cg * Fb[i] + sg * Fb[3 + i];
                Fp[i] = c * r0 - s * Fb[6 + i];
                Fp[3 + i] = cg * Fb[3 + i] - sg * Fb[i];
                Fp[6 + i] = s * r0 + c * Fb[6 + i];
            }
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    Rm[3 * i + j] = Fk[3 * i] * Fp[3 * j] + Fk[3 * i + 1] * Fp[3 * j + 1] + Fk[3 * i + 2] * Fp[3 * j + 2];
            double cb, sb, c2 = Rm[8], s2 = ax_unit(Rm[6], Rm[7], cb, sb);
            const double nrm2 = 1.0 / sqrt(c2 * c2 + s2 * s2);
            c2 *= nrm2;
            s2 *= nrm2;
            // a from what Rz(b) and Ry leave of Rm, so that a and b stay consistent when s2 is tiny:
            // row 0 of Rm Rz(b)^T Ry^T with Rz(b)^T = [[cb, -sb], [sb, cb]], Ry^T = [[c2, 0, s2], [0, 1, 0], [-s2, 0, c2]]
            double ca = c2 * (Rm[0] * cb + Rm[1] * sb) - s2 * Rm[2], sa = Rm[1] * cb - Rm[0] * sb;
            const double nrm3 = 1.0 / sqrt(ca * ca + sa * sa);
            ca *= nrm3;
            sa *= nrm3;
            ax_half(c, -s, tab[0], tab[1]);
            ax_half(c2, -s2, tab[4], tab[5]);
            // cos and sin of m gamma for the bra; of m a, then m b, where the ket blocks will be
            ax_phases(q.Lb, cg, sg, tab + ax_t_cg(q.Lb, q.Lk));
            double* ab = tab + ax_t_d(q.Lb, q.Lk);
            ax_phases(q.Lk, ca, sa, ab);
            ax_phases(q.Lk, cb, sb, ab + 2 * (q.Lk + 1));
        }
    }
    __syncthreads();
    // 0 Z^L is taken as 0 and the square of Z kept finite: at separations where F_L underflows
    // the powers of Z may overflow
    const int sub = lane & 7, g = threadIdx.x >> 3;
    for (int i0 = 0; i0 < per; i0 += AXB_THREADS / 8) {
        const int i = i0 + g, Lt = lt_[i];
        const double* z = z_[i];
        double *f = f_[i], *cur = row_[i] + 1, *nxt = nxt_[g], *tab = tab_[i], *bz = tab + AX_T_BZ;
        const double R2f = r2_[i];
        for (int L = sub; L <= Lt; L += 8) {
            const double b0 = f[L], b = b0 != 0.0 ? b0 * z[L] : 0.0;
            bz[ax_bz(L) + (L >> 1)] = b;
            f[L] = AX_FAR * fabs(b);
        }
        __syncwarp();
        bool far = true;
        // every lane takes the warp's longest loop, for the barriers: the groups' degrees may differ
        const int Lw = __reduce_max_sync(0xffffffffu, Lt);
        for (int ka = 1; 2 * ka <= Lw; ++ka) {
            for (int L = sub; L <= Lt - 2 * ka; L += 8) {
                const double x = cur[L];
                const double b = x != 0.0 ? x * z[L] : 0.0;
                bz[ax_bz(2 * ka + L) + (L >> 1)] = b;
                far = far && fabs(b) <= f[2 * ka + L];
                if (L <= Lt - 2 * ka - 2) nxt[L] = fma(R2f, cur[L + 2], (2 * L + 3) * cur[L + 1]);
            }
            __syncwarp();
            double* t = cur;
            cur = nxt;
            nxt = t;
        }
        const unsigned all = __ballot_sync(0xffffffffu, far) >> (lane & 24) & 0xffu;
        if (Lt >= 0 && sub == 0) tab[AX_T_FAR] = all == 0xffu ? 1.0 : 0.0;
    }
}

__global__ void boys_stage_kernel(int mmax, const double* __restrict__ T, int64_t n, double* __restrict__ F,
                                  unsigned* status) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double t = T[i];
    double buf[LTOT + 1];
    if (!(t >= 0.0) || !isfinite(t)) {
        set_status(status, ST_BAD_INPUT);
        for (int m = 0; m <= mmax; ++m) F[i * (mmax + 1) + m] = nan("");
        return;
    }
    boys_eval(mmax, t, buf);
    for (int m = 0; m <= mmax; ++m) F[i * (mmax + 1) + m] = buf[m];
}

// Stage entry: params[5i..] = (rho, X, Y, Z, pref) -> R[i * pyr(L) ..].
__global__ void __launch_bounds__(BR_WARPS * 32) hermite_r_stage_kernel(int L, const double* __restrict__ params,
                                                                        int64_t n, double* __restrict__ Rout) {
    extern __shared__ double smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t item = (int64_t)blockIdx.x * BR_WARPS + warp;
    if (item >= n) return;
    const int nr = pyr(L);
    double* R = smem + warp * (nr + LTOT + 1);
    double* B = R + nr;
    const double rho = params[5 * item], X = params[5 * item + 1], Y = params[5 * item + 2],
                 Z = params[5 * item + 3], pref = params[5 * item + 4];
    if (lane == 0) boys_eval(L, rho * (X * X + Y * Y + Z * Z), B);
    __syncwarp();
    scale_base(L, rho, pref, B, lane);
    __syncwarp();
    hermite_r_warp(L, X, Y, Z, B, R, lane);
    for (int r = lane; r < nr; r += 32) Rout[item * nr + r] = R[r];
}

size_t br_smem(int L) { return sizeof(double) * BR_WARPS * (size_t)(pyr(L) + LTOT + 1); }

}  // namespace

cudaError_t init_boys_table(const double* host_table) {
    cudaError_t e = cudaMemcpyToSymbol(g_boys, host_table, sizeof(double) * BOYS_NROW * BOYS_NPT);
    if (e != cudaSuccess) return e;
    static_assert(NHERM_TOT <= 8192, "Hermite positions fit 13 bits");
    std::vector<int4> rec(NHERM_TOT, make_int4(0, 0, 0, 0));
    for (int n = 1; n <= LTOT; ++n)
        for (int i = 0; i <= n; ++i)
            for (int v = 0; v <= i; ++v) {
                const int u = i - v, t = n - i;
                const int d = t > 0 ? 0 : (u > 0 ? 1 : 2), rd = d == 0 ? t : (d == 1 ? u : v);
                const int dt = d == 0, du = d == 1, dv = d == 2;
                const int h1 = hidx(t - dt, u - du, v - dv);
                const int h2 = rd > 1 ? hidx(t - 2 * dt, u - 2 * du, v - 2 * dv) : 0;
                const double c = rd - 1;
                long long bits;
                std::memcpy(&bits, &c, sizeof(bits));
                rec[hidx(t, u, v)] = make_int4(h1 | (h2 << 13) | (d << 26), 0, (int)(bits & 0xFFFFFFFFll), (int)(bits >> 32));
            }
    if ((e = cudaMemcpyToSymbol(g_rec, rec.data(), sizeof(int4) * NHERM_TOT)) != cudaSuccess) return e;
    e = cudaFuncSetAttribute(boys_r_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(double) * (pyr(LTOT) + LTOT + 1)));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(hermite_r_stage_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)br_smem(LTOT));
}

cudaError_t launch_boys_r(const DQuartet* qd, const DPair* pairs, const WorkItem* items, int nitems, int lmax,
                          double* ws, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    if (lmax < 0 || lmax > LTOT) return cudaErrorInvalidValue;
    boys_base_kernel<<<(nitems + BASE_THREADS - 1) / BASE_THREADS, BASE_THREADS, 0, st>>>(qd, pairs, items, nitems, ws);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = sizeof(double) * (pyr(lmax) + LTOT + 1);
    boys_r_kernel<<<nitems, 32, smem, st>>>(qd, pairs, items, ws);
    return cudaGetLastError();
}

cudaError_t launch_axial_boys(const AxQuartet* qd, const AxPair* pairs, const WorkItem* items, int nitems, double* ws,
                              cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const int per = nitems > AXB_FEW ? AXB_PER : AXB_PER_FEW;
    axial_boys_kernel<<<(nitems + per - 1) / per, AXB_THREADS, 0, st>>>(qd, pairs, items, nitems, per, ws);
    return cudaGetLastError();
}

cudaError_t launch_boys(int mmax, const double* T, int64_t n, double* F, unsigned* status, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    boys_stage_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(mmax, T, n, F, status);
    return cudaGetLastError();
}

cudaError_t launch_hermite_r(int L, const double* params, int64_t n, double* R, unsigned* status, cudaStream_t st) {
    (void)status;
    if (n <= 0) return cudaSuccess;
    hermite_r_stage_kernel<<<(unsigned)((n + BR_WARPS - 1) / BR_WARPS), BR_WARPS * 32, br_smem(L), st>>>(L, params,
                                                                                                          n, R);
    return cudaGetLastError();
}

}  // namespace lx
