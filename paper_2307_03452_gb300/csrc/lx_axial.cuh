// Axial form of the FP64 path: tables, descriptors and launchers (the method is described at
// the top of lx_axial.cu).
#pragma once
#include <cstdint>
#include <vector>

#include "lx_internal.cuh"

namespace lx {

constexpr int AX_LP = 2 * LMAX;  // largest degree of one pair's operators (14)
constexpr int AX_NL = AX_LP + 1;
// Smallest matrix-form transforms, N_ab N_p N_q + N_ab N_q N_cd FMAs per primitive quartet, for
// which the axial form is taken: uncontracted, by output, and of at least AX_CONTRACTED primitive
// quartets.  Device times of all classes of s to k pairs near the lines, matrix form against axial
// form: 1,024 uncontracted quartets, solid, (fp|fs) (the lowest) 0.209 against 0.201 ms, (dd|dd) 0.32
// against 0.25, Cartesian just above its line (ff|ps) and (fd|pp) 1.2 to 1.5 times faster, just below it
// (gs|dd) 0.25 against 0.28; 256 quartets with K = 1..5, above the line (dd|dd) 3.7 against 1.9, (fp|fp) 3.5
// against 1.4, below it (dd|dp) 2.8 against 3.2.
constexpr int AX_CONTRACTED = 4;
constexpr int64_t AX_MIN_FMA_SOLID = 16000, AX_MIN_FMA_CART = 38000, AX_MIN_FMA_CONTRACTED = 26000;
constexpr int AX_SMS = 152;      // SMs of a GB300
constexpr int AX_ONE_WAVE = 4 * AX_SMS;  // main items that run at once, four to an SM
constexpr int AX_NR = 8;         // half rows of one CTA of the main kernel

// One harmonic component group of a shell: Y_lam,m r^(l - lam) for m >= 0 (and its sine partner
// if m > 0), as a polynomial A_m(x, y) sum_j alpha[j] rho^2j z^(l - m - 2j).
struct AxFn {
    int16_t m, lam;
    int16_t plus, minus;  // positions of the cosine and sine functions in the shell's list
    double alpha[LMAX / 2 + 1];
};
struct AxShell {   // one (l, output kind)
    int fn0, nfn;  // its AxFn entries
    int ntot;      // functions: 2l+1, or (l+1)(l+2)/2 (harmonics l, l-2, ... of a Cartesian shell)
    int wc0;       // Cartesian: start of its rows in wc_row (ntot + 1 bounds into wc); -1 for solid
};
// Half row of a pair class: the product of the m_a and m_b >= 0 functions fa, fb holds the
// azimuthal orders m_a + m_b (slot 0) and |m_a - m_b| (slot 1); its cosine and sine members are
// stored at functions vc, vs of the (a, b) block (vs = -1: no sine member).  The half rows of
// a class are ordered by M (the most work first).
struct AxHalf {
    int16_t fa, fb, M, slot, vc, vs;
    int32_t hoff;  // its entries (l = M.., k = 0..(L-l)/2) in the pair's h
};
struct AxClass {  // (l_a, l_b, output kind)
    int half0, nhalf, nh;
};
struct AxPair {
    int sa, sb, Kab, sign;
    int la, lb, cls, nh;
    int64_t h_off;     // doubles: [Kab][nh]
    int64_t info_off;  // doubles: [Kab][4] = zeta_p, P
    int64_t rot_off;   // doubles: AX_ROT (frame, phases, Y blocks)
};
struct AxQuartet {
    int pb, pk, kbra, kket;
    int Lb, Lk, nab, ncd;
    int cb, ck, tab_stride;
    int full;  // the tables hold the full ket blocks (else their factors)
    int64_t tab_off;  // doubles: [kbra][kket][tab_stride]
    int64_t out_off;
    // the ket primitives are summed in nsplit parts: part 0 in the output block, the others in
    // [nsplit - 1][nab ncd] doubles here, added when the ket indices are rotated
    int64_t part_off;
    int nsplit, pad;
};
// Primitive quartets per part: a CTA of the main kernel takes one part of one quartet, and with
// K = 5 on every shell (625 primitive quartets) one CTA would outlast the rest of a batch of some
// hundred quartets; of the largest classes 16 would.  So a part has as many as AX_PART_OPS, in units of
// pyr(Lk) (Lb + 1), about a primitive quartet's work in one CTA, and at most AX_PART.  Seven mixed
// Cartesian quartets, K = 1..2: main kernel 0.77 ms with 16 in every part, 0.46 so (0.53 at 12,000, 0.52 at
// 8,000); 200 mixed solid ones 17.4 -> 16.6.
constexpr int AX_PART = 16, AX_PART_OPS = 16000;
inline int ax_part(int Lb, int Lk) {
    const int ops = pyr(Lk) * (Lb + 1), n = AX_PART_OPS / ops;
    return n < 1 ? 1 : n < AX_PART ? n : AX_PART;
}

// Offsets of the l blocks: cosine blocks (l+1)^2, sine blocks l^2, full blocks (2l+1)^2.
__host__ __device__ inline int ax_co(int l) { return l * (l + 1) * (2 * l + 1) / 6; }
__host__ __device__ inline int ax_so(int l) { return (l - 1) * l * (2 * l - 1) / 6; }
__host__ __device__ inline int ax_do(int l) { return l * (2 * l - 1) * (2 * l + 1) / 3; }
// Row N of the table B_kappa(L) Z^L, 2 kappa + L = N: entries L = N mod 2, ..., N.
__host__ __device__ inline int ax_bz(int N) { return (N - 1) * (N - 1) / 4 + N; }
// Rotation data of a pair: frame (9), cos and sin of m phi (m = 0..LMAX), Y blocks l = 0..LMAX.
constexpr int AX_ROT_CS = 10, AX_ROT_C = AX_ROT_CS + 2 * (LMAX + 1);
__host__ __device__ inline int ax_rot_size(int l) { return AX_ROT_C + ax_co(l + 1) + ax_so(l + 1); }
// Table of a primitive quartet: cos and sin of the half angles about y (bra at 0, ket at 4), a flag (see
// AX_FAR), B Z^L, cos and sin of M gamma, Y blocks of the bra
// rotation, and of the ket rotation either the full blocks or, at about half the size, their
// factors: cos and sin of m a, of m b, Y blocks.
constexpr int AX_T_FAR = 10, AX_T_BZ = 12;
// A primitive quartet is far if every B_kappa(L) Z^L with kappa >= 1 (a polynomial times e^-T) is below
// AX_FAR of the B_0(N) Z^N of its degree N = 2 kappa + L: only T(l, l', M, 0) is then used, and of
// it the L = l + l' term, the interaction of multipoles.  AX_FAR = 2^-100: [r]^(0) of degree N reaches
// at least 2^-21 B_0(N) Z^N (the ratio of (2N-1)!! to N! at N = 24; 2^-25 at 28), so what is left out
// lies 2^-20 and more below one rounding of the matrix form's entries of the same degree.
constexpr double AX_FAR = 0x1p-100;
__host__ __device__ inline int ax_t_cg(int Lb, int Lk) { return AX_T_BZ + ax_bz(Lb + Lk + 1); }
__host__ __device__ inline int ax_t_c(int Lb, int Lk) { return ax_t_cg(Lb, Lk) + 2 * (Lb + 1); }
__host__ __device__ inline int ax_t_d(int Lb, int Lk) { return ax_t_c(Lb, Lk) + ax_co(Lb + 1) + ax_so(Lb + 1); }
__host__ __device__ inline int ax_t_size(int Lb, int Lk, bool full) {
    // full: the phases of the factors stand there first (more than the one block of Lk = 0)
    const int blocks = full ? ax_do(Lk + 1) : ax_co(Lk + 1) + ax_so(Lk + 1), ph = 4 * (Lk + 1);
    return (ax_t_d(Lb, Lk) + (full ? (blocks > ph ? blocks : ph) : ph + blocks) + 3) / 4 * 4;
}

// (c, s) = (x, y) / |(x, y)| and the length; (1, 0) for a null vector.  Scaled by the larger
// component first, so that the squares of tiny components cannot underflow.
__device__ inline double ax_unit(double x, double y, double& c, double& s) {
    const double m = fmax(fabs(x), fabs(y));
    c = 1.0;
    s = 0.0;
    if (!(m > 0.0)) return 0.0;
    const double a = x / m, b = y / m, n = sqrt(a * a + b * b);
    c = a / n;
    s = b / n;
    return m * n;
}
// n = v / |v| and the length, likewise; (0, 0, 1) for a null vector.
__device__ inline double ax_unit3(const double v[3], double n[3]) {
    const double m = fmax(fabs(v[0]), fmax(fabs(v[1]), fabs(v[2])));
    n[0] = n[1] = 0.0;
    n[2] = 1.0;
    if (!(m > 0.0)) return 0.0;
    const double a = v[0] / m, b = v[1] / m, c = v[2] / m, len = sqrt(a * a + b * b + c * c);
    n[0] = a / len;
    n[1] = b / len;
    n[2] = c / len;
    return m * len;
}

// cos and sin of half the angle of (c, s).
__device__ inline void ax_half(double c, double s, double& ch, double& sh) {
    ch = sqrt(fmax(0.0, 0.5 * (1.0 + c)));
    if (ch > 0.5) {
        sh = s / (2.0 * ch);
    } else {
        sh = sqrt(fmax(0.0, 0.5 * (1.0 - c)));
        ch = s / (2.0 * sh);
    }
}

// cos and sin of m times the angle of (c, s), m = 0..n.
__device__ inline void ax_phases(int n, double c, double s, double* o) {
    double x = 1.0, y = 0.0;
    for (int m = 0; m <= n; ++m) {
        o[2 * m] = x;
        o[2 * m + 1] = y;
        const double t = x * c - y * s;
        y = x * s + y * c;
        x = t;
    }
}

struct AxHost {
    std::vector<double> g;         // axial products G(l, l', M, L), l <= l'
    std::vector<double> vinv;      // cylindrical -> spherical operators of degree n, order M
    std::vector<int> vinv_off;     // [n][M]
    std::vector<double> tau;       // [M][s][q]
    std::vector<double> wig0;      // start of each d chain (mp, m)
    std::vector<double> wig;       // [chain][l][3]
    std::vector<int> tent;         // T entries of every (Lb, Lk)
    std::vector<int> tent_off;     // [Lb][Lk] + 1
    std::vector<int> tinfo;        // [Lb][Lk][l][l']: offset << 8 | entries per M
    std::vector<int> task_t;       // T tasks of every (Lb, Lk), groups of 4: l' | M' << 8, or -1
    std::vector<int> task_t_off;
    std::vector<int> task_r;       // rotation tasks of every Lk, groups of 4: l | (M + l) << 8
    std::vector<int> task_r_off;
    std::vector<AxFn> fns;
    AxShell shell[LMAX + 1][2];
    std::vector<AxHalf> halves;
    AxClass cls[(LMAX + 1) * (LMAX + 1) * 2];
    std::vector<int> wc_row, wc_idx;  // Cartesian conversion, sparse rows
    std::vector<double> wc_val;
};
inline int ax_class_id(int la, int lb, bool solid) { return (la * (LMAX + 1) + lb) * 2 + (solid ? 1 : 0); }
void make_axial_tables(AxHost& H);  // lx_axial_tables.cpp
const AxHost& axial_tables();       // built once per process

cudaError_t init_axial(const AxHost& H);
// Shared memory of one CTA of the main kernel.
size_t axial_main_smem(int Lb, int Lk);
cudaError_t launch_axial_pair(const AxPair* pairs, const WorkItem* items, int nitems, const DShell* sh,
                              const double* exps, const double* ncoef, double* ws, bool solid, cudaStream_t st);
cudaError_t launch_axial_boys(const AxQuartet* qd, const AxPair* pairs, const WorkItem* items, int nitems, double* ws,
                              cudaStream_t st);  // lx_boys_r.cu
cudaError_t launch_axial_wigner(const AxQuartet* qd, const WorkItem* items, int nitems, int lmax, double* ws,
                                cudaStream_t st);
// Size groups of the main kernel's launches.
constexpr int AX_NBIN = 5;
int axial_bin(int Lb, int Lk);
cudaError_t launch_axial_main(const AxQuartet* qd, const AxPair* pairs, const WorkItem* items, const int* counts,
                              const size_t* smem, double* ws, double* out, cudaStream_t st);
// Functions of both indices of one side rotated to the lab frame (and converted to Cartesian):
// ket indices over row tiles (side = 1), bra indices over column tiles (side = 0).
cudaError_t launch_axial_rotate(int side, const AxQuartet* qd, const AxPair* pairs, const WorkItem* items, int nitems,
                                int lanes, size_t smem, const double* ws, double* out, bool solid, cudaStream_t st);
// J/K digestion of the axial quartets' blocks (lx_jk.cu).
cudaError_t launch_jk_digest(const AxQuartet* qd, const AxPair* pairs, const DShell* sh, int nquartet,
                             const double* ws, bool solid, const double* D, int64_t nbf, double* J, double* K,
                             cudaStream_t st);
inline int axial_lanes(int n) { return n <= 784 ? 16 : 8; }
inline size_t axial_rotate_smem(int n, int lanes) { return sizeof(double) * 2 * (size_t)n * (lanes + 1); }

}  // namespace lx
