// Expansion kernels of the FMM / treecode: translation-operator tables (FP64 arithmetic,
// stored FP32), P2M, M2M, L2L, L2P and M2P (FP32).
//
// Notation (Section "Fast N-body simulation", Eq. 2-9): Y_n^m as Eq. 6 with the
// Condon-Shortley phase of Eq. 8; regular solid harmonics R_n^m(v) = |v|^n Y_n^m(v),
// irregular I_n^m(v) = |v|^(-n-1) Y_n^m(v).  Both are evaluated from Cartesian coordinates
// with the normalised three-term recurrence in n (Eq. 7 multiplied through by |v|^n) and the
// diagonal step R_m^m = -sqrt((2m-1)/(2m)) (x + iy) R_{m-1}^{m-1} (Eq. 8), so no
// trigonometric function is needed on the device.
//
//   P2M (Eq. 2):  M_n^m = sum_j q_j R_n^{-m}(x_j - c) = sum_j q_j conj(R_n^m(x_j - c))
//   L2P (Eq. 3):  phi = sum_{n,m} L_n^m R_n^m(x - c)
//   M2P (Eq. 2):  phi = sum_{n,m} M_n^m I_n^m(x - c)
// Gradients use the ladder relations of solid harmonics (d/dz and d/dx + i d/dy lower or
// raise the degree by one), which stay finite on the expansion's z axis.
// M2L (Eq. 4-5) and the M2M / L2L translations (Cheng, Greengard & Rokhlin 1999, cited by
// the paper for its translation operators) are linear maps on the real-packed coefficients;
// with coefficients scaled by the cell side they do not depend on the level, so each is a
// dense p^2 x p^2 FP32 matrix computed once per order in FP64.
#include "common.cuh"

#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

namespace gbfmm {

#define GBFMM_DISPATCH_P(P, CALL)      \
    switch (P) {                       \
    case 4: { constexpr int PQ = 4; CALL; } break;   \
    case 6: { constexpr int PQ = 6; CALL; } break;   \
    case 8: { constexpr int PQ = 8; CALL; } break;   \
    case 10: { constexpr int PQ = 10; CALL; } break; \
    }

constexpr int kMaxP = 10;
constexpr int kMaxDeg = 2 * kMaxP;  // harmonics up to degree 2P-2 (M2L) and P (M2P gradient)

// Recurrence and ladder constants, set once per device (init_expansion_constants).
__constant__ float c_rmm[kMaxDeg + 1];                 // sqrt((2m-1)/(2m))
__constant__ float c_ra[kMaxDeg + 1][kMaxDeg + 1];     // (2n+1) / sqrt((n+1-m)(n+1+m))
__constant__ float c_rb[kMaxDeg + 1][kMaxDeg + 1];     // sqrt((n-m)(n+m)) / sqrt((n+1-m)(n+1+m))
__constant__ float c_nbeta1[kMaxP + 1][kMaxP + 1];  // -beta_n^m of the real recurrences (P2M, P2L, M2P)
__device__ float d_kscale[kMaxP * kMaxP];           // k_n^m of the real-packed coefficient n^2 + ...
__constant__ float c_sq[2 * kMaxDeg + 4][2 * kMaxDeg + 4];  // sqrt(a*b)

void m2p_tables();

void init_expansion_constants()
{
    m2p_tables();
    float rmm[kMaxDeg + 1], ra[kMaxDeg + 1][kMaxDeg + 1], rb[kMaxDeg + 1][kMaxDeg + 1];
    float sq[2 * kMaxDeg + 4][2 * kMaxDeg + 4];
    for (int m = 0; m <= kMaxDeg; ++m) rmm[m] = m ? (float)sqrt((2.0 * m - 1.0) / (2.0 * m)) : 0.f;
    for (int n = 0; n <= kMaxDeg; ++n)
        for (int m = 0; m <= kMaxDeg; ++m) {
            double den = (double)(n + 1 - m) * (double)(n + 1 + m);
            ra[n][m] = (m <= n) ? (float)((2.0 * n + 1.0) / sqrt(den)) : 0.f;
            rb[n][m] = (m <= n) ? (float)(sqrt((double)(n - m) * (double)(n + m)) / sqrt(den)) : 0.f;
        }
    for (int a = 0; a < 2 * kMaxDeg + 4; ++a)
        for (int b = 0; b < 2 * kMaxDeg + 4; ++b) sq[a][b] = (float)sqrt((double)a * (double)b);
    cudaMemcpyToSymbol(c_rmm, rmm, sizeof(rmm));
    cudaMemcpyToSymbol(c_ra, ra, sizeof(ra));
    cudaMemcpyToSymbol(c_rb, rb, sizeof(rb));
    cudaMemcpyToSymbol(c_sq, sq, sizeof(sq));
}

// real-packed index of Re C_n^m / Im C_n^m
GB_HD constexpr int re_idx(int n, int m) { return m == 0 ? n * n : n * n + 2 * m - 1; }
GB_HD constexpr int im_idx(int n, int m) { return n * n + 2 * m; }

// ------------------------------------------------------------------------------------------
// Operator tables (FP64 arithmetic, one CTA per operator).
// All three column-major, [op][col][row], rows padded to PR = round_up(p^2, 8) with zeros:
//   M2L  code < 343 (offset source - target, in cells)
//   M2M  child position c (bit0 x, bit1 y, bit2 z), child -> parent
//   L2L  parent -> child c
// ------------------------------------------------------------------------------------------
struct C64 {
    double re, im;
};
GB_HD C64 cmul(C64 a, C64 b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
GB_HD C64 conj64(C64 a) { return {a.re, -a.im}; }

GB_HD void dof_decode(int i, int &n, int &m, int &im)
{
    n = 0;
    while ((n + 1) * (n + 1) <= i) ++n;
    int r = i - n * n;
    if (r == 0) {
        m = 0;
        im = 0;
    } else {
        m = (r + 1) / 2;
        im = (r % 2 == 0);
    }
}

GB_HD double fact64(int k)
{
    double f = 1.0;
    for (int i = 2; i <= k; ++i) f *= i;
    return f;
}
GB_HD double Anm64(int n, int m) { return 1.0 / sqrt(fact64(n - m) * fact64(n + m)); }
GB_HD double ipow_even(int e) { return ((e / 2) % 2 == 0) ? 1.0 : -1.0; }

// regular (irreg = 0) or irregular (irreg = 1) solid harmonics H[n(n+1)/2 + m], m >= 0, n < nmax
GB_HD void harmonics64(int nmax, double x, double y, double z, int irreg, C64 *H)
{
    double r2 = x * x + y * y + z * z;
    double ir2 = 1.0 / r2;
    C64 hmm = {irreg ? 1.0 / sqrt(r2) : 1.0, 0.0};
    for (int m = 0; m < nmax; ++m) {
        if (m > 0) {
            double f = -sqrt((2.0 * m - 1.0) / (2.0 * m)) * (irreg ? ir2 : 1.0);
            C64 t = cmul(C64{x, y}, hmm);
            hmm = {f * t.re, f * t.im};
        }
        H[m * (m + 1) / 2 + m] = hmm;
        for (int n = m; n + 1 < nmax; ++n) {
            C64 a = H[n * (n + 1) / 2 + m];
            C64 b = (n - 1 >= m) ? H[(n - 1) * n / 2 + m] : C64{0.0, 0.0};
            double s = sqrt((double)(n - m) * (double)(n + m));
            double d = 1.0 / sqrt((double)(n + 1 - m) * (double)(n + 1 + m));
            double ca = (2.0 * n + 1.0) * z, cb = s * (irreg ? 1.0 : r2);
            C64 v = {(ca * a.re - cb * b.re) * d, (ca * a.im - cb * b.im) * d};
            if (irreg) {
                v.re *= ir2;
                v.im *= ir2;
            }
            H[(n + 1) * (n + 2) / 2 + m] = v;
        }
    }
}

GB_HD C64 hfull(const C64 *H, int n, int m)
{
    return m >= 0 ? H[n * (n + 1) / 2 + m] : conj64(H[n * (n + 1) / 2 - m]);
}

// complex coefficient of input C_n^m in output D_j^k for the three operators
GB_HD C64 k_m2l(const C64 *I, int j, int k, int n, int m)
{
    double f = ipow_even(abs(k - m) - abs(k) - abs(m)) * Anm64(n, m) * Anm64(j, k) / Anm64(j + n, m - k) *
               ((j & 1) ? -1.0 : 1.0);
    C64 h = hfull(I, j + n, m - k);
    return {f * h.re, f * h.im};
}

GB_DEV C64 k_m2m(const C64 *R, int j, int k, int n, int m)
{
    if (j < n || abs(k - m) > j - n) return {0.0, 0.0};
    int nn = j - n, mm = k - m;
    double f = ipow_even(abs(k) - abs(mm) - abs(k - mm)) * Anm64(nn, mm) * Anm64(n, m) / Anm64(j, k) / ldexp(1.0, j);
    C64 h = hfull(R, nn, -mm);
    return {f * h.re, f * h.im};
}

GB_DEV C64 k_l2l(const C64 *R, int j, int k, int n, int m)
{
    if (n < j || abs(m - k) > n - j) return {0.0, 0.0};
    double f = ipow_even(abs(m) - abs(m - k) - abs(k)) * Anm64(n - j, m - k) * Anm64(j, k) / Anm64(n, m) /
               ldexp(1.0, n + 1);
    C64 h = hfull(R, n - j, m - k);
    return {f * h.re, f * h.im};
}

__global__ void k_build_ops(int P, float *m2l, float *m2m, float *l2l)
{
    __shared__ C64 H[(2 * kMaxP) * (2 * kMaxP + 1) / 2];
    const int op = blockIdx.x;
    const int PP = P * P;
    int kind;  // 0 m2l, 1 m2m, 2 l2l
    double v[3];
    bool used = true;
    if (op < kM2LCodes) {
        kind = 0;
        int dx = op % 7 - 3, dy = (op / 7) % 7 - 3, dz = op / 49 - 3;
        used = !(abs(dx) <= 1 && abs(dy) <= 1 && abs(dz) <= 1);
        v[0] = dx;  // target centre - source centre = -(source - target); the list stores
        v[1] = dy;  // source - target, so the operator is built for the negated offset below
        v[2] = dz;
        v[0] = -v[0];
        v[1] = -v[1];
        v[2] = -v[2];
    } else {
        int c = (op - kM2LCodes) % 8;
        kind = (op - kM2LCodes) < 8 ? 1 : 2;
        v[0] = (c & 1) - 0.5;  // child centre - parent centre, in child cells
        v[1] = ((c >> 1) & 1) - 0.5;
        v[2] = ((c >> 2) & 1) - 0.5;
    }
    if (threadIdx.x == 0 && used) harmonics64(kind == 0 ? 2 * P - 1 : P, v[0], v[1], v[2], kind == 0, H);
    __syncthreads();
    const int PR = (PP + 7) / 8 * 8;
    float *table = kind == 0 ? m2l + (size_t)op * PP * PR
                 : kind == 1 ? m2m + (size_t)(op - kM2LCodes) * PP * PR
                             : l2l + (size_t)(op - kM2LCodes - 8) * PP * PR;
    for (int e = threadIdx.x; e < PP * (PR - PP); e += blockDim.x)  // zero padding rows
        table[(size_t)(e / (PR - PP)) * PR + PP + e % (PR - PP)] = 0.f;
    for (int e = threadIdx.x; e < PP * PP; e += blockDim.x) {
        int row = e / PP, col = e % PP;
        float out = 0.f;
        if (used) {
            int j, k, rim, n, m, cim;
            dof_decode(row, j, k, rim);
            dof_decode(col, n, m, cim);
            C64 u = cim ? C64{0.0, 1.0} : C64{1.0, 0.0};
            C64 a, b = {0.0, 0.0};
            if (kind == 0) {
                a = k_m2l(H, j, k, n, m);
                if (m > 0) b = k_m2l(H, j, k, n, -m);
            } else if (kind == 1) {
                a = k_m2m(H, j, k, n, m);
                if (m > 0) b = k_m2m(H, j, k, n, -m);
            } else {
                a = k_l2l(H, j, k, n, m);
                if (m > 0) b = k_l2l(H, j, k, n, -m);
            }
            C64 val = cmul(a, u);
            C64 w = cmul(b, conj64(u));
            val.re += w.re;
            val.im += w.im;
            out = (float)(rim ? val.im : val.re);
        }
        table[(size_t)col * PR + row] = out;
    }
}

void launch_build_operators(int P, float *m2l_ops, float *m2m_ops, float *l2l_ops, cudaStream_t s)
{
    k_build_ops<<<kM2LCodes + 16, 256, 0, s>>>(P, m2l_ops, m2m_ops, l2l_ops);
    note_launches(1);
}

// ------------------------------------------------------------------------------------------
// Rotation factors of the M2L operators (host, FP64).  For an offset code with translation
// v = target centre - source centre and a rotation Q taking v / |v| to +z,
//   T_v = F^-1 C_|v| F,
// F: block-diagonal in the degree, the map of a degree-n coefficient block under the change
//    of frame x -> Q x (multipole and local blocks alike: both are sums of q f(rho) R_n^-m);
//    found by least squares from the blocks of point charges at sample directions and at their
//    rotated images (the map is exactly linear, so the fit is exact up to rounding);
// F^-1: the same for Q^T;
// C: the M2L operator of the coaxial translation (0, 0, |v|), which couples equal orders only,
//    with one real coefficient for the real and the imaginary parts.
// The factorisation is checked against the dense operator before it is used.
// Layout per code (kM2LCodes slots of m2l_rot_code_floats): F blocks (n = 0..P-1, (2n+1)^2 each,
// [row][col]), F^-1 blocks, then C blocks (m = 0..P-1, (P-m)^2 each, [j-m][n-m]), zero padding.
// ------------------------------------------------------------------------------------------
namespace {

void packed_block_regular(int n, const double x[3], double *out)
{
    C64 H[(kMaxDeg + 1) * (kMaxDeg + 2) / 2];
    harmonics64(n + 1, x[0], x[1], x[2], 0, H);
    for (int m = 0; m <= n; ++m) {
        const C64 r = H[n * (n + 1) / 2 + m];  // the block holds conj(R_n^m)
        if (m == 0) {
            out[0] = r.re;
        } else {
            out[2 * m - 1] = r.re;
            out[2 * m] = -r.im;
        }
    }
}

// solve G X = B for X (s x s, G symmetric positive definite), partial pivoting
bool solve_dense(int s, std::vector<double> G, std::vector<double> &B)
{
    for (int c = 0; c < s; ++c) {
        int piv = c;
        for (int r = c + 1; r < s; ++r)
            if (fabs(G[r * s + c]) > fabs(G[piv * s + c])) piv = r;
        if (fabs(G[piv * s + c]) < 1e-300) return false;
        if (piv != c)
            for (int k = 0; k < s; ++k) {
                std::swap(G[c * s + k], G[piv * s + k]);
                std::swap(B[c * s + k], B[piv * s + k]);
            }
        for (int r = 0; r < s; ++r) {
            if (r == c) continue;
            const double f = G[r * s + c] / G[c * s + c];
            if (f == 0.0) continue;
            for (int k = 0; k < s; ++k) {
                G[r * s + k] -= f * G[c * s + k];
                B[r * s + k] -= f * B[c * s + k];
            }
        }
    }
    for (int r = 0; r < s; ++r)
        for (int k = 0; k < s; ++k) B[r * s + k] /= G[r * s + r];
    return true;
}

// F_n for the frame change x -> Q x, row-major (2n+1)^2
bool rotation_block(int n, const double Q[9], double *F)
{
    const int s = 2 * n + 1, K = 2 * s + 3;
    std::vector<double> G(s * s, 0.0), Hm(s * s, 0.0), p(s), q(s);
    for (int i = 0; i < K; ++i) {
        double x[3] = {sin(1.31 * i + 0.7), cos(2.17 * i + 0.23), sin(0.93 * i + 1.1) + 0.3 * cos(3.7 * i)};
        const double nx = sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
        for (double &c : x) c /= nx;
        const double y[3] = {Q[0] * x[0] + Q[1] * x[1] + Q[2] * x[2], Q[3] * x[0] + Q[4] * x[1] + Q[5] * x[2],
                             Q[6] * x[0] + Q[7] * x[1] + Q[8] * x[2]};
        packed_block_regular(n, x, p.data());
        packed_block_regular(n, y, q.data());
        for (int a = 0; a < s; ++a)
            for (int b = 0; b < s; ++b) {
                G[a * s + b] += p[a] * p[b];
                Hm[a * s + b] += p[a] * q[b];  // (sum p q^T): F^T = G^-1 (sum p q^T)
            }
    }
    if (!solve_dense(s, G, Hm)) return false;
    for (int a = 0; a < s; ++a)
        for (int b = 0; b < s; ++b) F[a * s + b] = Hm[b * s + a];
    return true;
}

// the dense M2L operator (real-packed, [row][col]) of translation v, as k_build_ops builds it
void dense_m2l(int P, const double v[3], std::vector<double> &T)
{
    const int PP = P * P;
    std::vector<C64> H((2 * kMaxP) * (2 * kMaxP + 1) / 2);
    harmonics64(2 * P - 1, v[0], v[1], v[2], 1, H.data());
    T.assign((size_t)PP * PP, 0.0);
    for (int row = 0; row < PP; ++row)
        for (int col = 0; col < PP; ++col) {
            int j, k, rim, n, m, cim;
            dof_decode(row, j, k, rim);
            dof_decode(col, n, m, cim);
            const C64 u = cim ? C64{0.0, 1.0} : C64{1.0, 0.0};
            const C64 a = k_m2l(H.data(), j, k, n, m);
            const C64 b = m > 0 ? k_m2l(H.data(), j, k, n, -m) : C64{0.0, 0.0};
            C64 val = cmul(a, u);
            const C64 w = cmul(b, conj64(u));
            val.re += w.re;
            val.im += w.im;
            T[(size_t)row * PP + col] = rim ? val.im : val.re;
        }
}

}  // namespace

// floats per code: F, F^-1 and C, padded to a multiple of 4 (16-byte aligned codes)
size_t m2l_rot_code_floats(int P)
{
    size_t f = 0, c = 0;
    for (int n = 0; n < P; ++n) f += (size_t)(2 * n + 1) * (2 * n + 1);
    for (int m = 0; m < P; ++m) c += (size_t)(P - m) * (P - m);
    return (2 * f + c + 3) / 4 * 4;
}

int build_m2l_rot_table(int P, std::vector<float> &out)
{
    const int PP = P * P;
    const size_t RS = m2l_rot_code_floats(P);
    out.assign(RS * kM2LCodes, 0.f);
    std::vector<double> T, Cz, Fd((size_t)PP * PP), Fi((size_t)PP * PP);
    for (int code = 0; code < kM2LCodes; ++code) {
        const int dx = code % 7 - 3, dy = (code / 7) % 7 - 3, dz = code / 49 - 3;
        if (abs(dx) <= 1 && abs(dy) <= 1 && abs(dz) <= 1) continue;
        const double v[3] = {-(double)dx, -(double)dy, -(double)dz};  // target centre - source centre
        const double d = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        const double u[3] = {v[0] / d, v[1] / d, v[2] / d};
        double Q[9];  // rotation taking u to +z (Rodrigues about u x z)
        const double ax = u[1], ay = -u[0], s2 = ax * ax + ay * ay, c = u[2];
        if (s2 < 1e-30) {
            const double sg = c > 0 ? 1.0 : -1.0;  // u = +-z: identity or a half turn about x
            const double Qi[9] = {1, 0, 0, 0, sg, 0, 0, 0, sg};
            memcpy(Q, Qi, sizeof(Q));
        } else {
            const double sn = sqrt(s2), kx = ax / sn, ky = ay / sn, t = 1.0 - c;
            const double Qi[9] = {c + kx * kx * t, kx * ky * t, ky * sn, kx * ky * t, c + ky * ky * t, -kx * sn,
                                  -ky * sn, kx * sn, c};
            memcpy(Q, Qi, sizeof(Q));
        }
        const double Qt[9] = {Q[0], Q[3], Q[6], Q[1], Q[4], Q[7], Q[2], Q[5], Q[8]};
        const double z[3] = {0.0, 0.0, d};
        dense_m2l(P, v, T);
        dense_m2l(P, z, Cz);
        std::fill(Fd.begin(), Fd.end(), 0.0);
        std::fill(Fi.begin(), Fi.end(), 0.0);
        float *o = out.data() + RS * code;
        size_t at = 0;
        for (int pass = 0; pass < 2; ++pass)
            for (int n = 0; n < P; ++n) {
                const int s = 2 * n + 1;
                std::vector<double> B(s * s);
                if (!rotation_block(n, pass == 0 ? Q : Qt, B.data())) return -1;
                for (int a = 0; a < s; ++a)
                    for (int b = 0; b < s; ++b) {
                        (pass == 0 ? Fd : Fi)[(size_t)(n * n + a) * PP + n * n + b] = B[a * s + b];
                        o[at++] = (float)B[a * s + b];
                    }
            }
        // C: equal orders only, one coefficient for real and imaginary parts
        double cmax = 0.0, off = 0.0, imdiff = 0.0;
        for (int r = 0; r < PP; ++r)
            for (int cc = 0; cc < PP; ++cc) cmax = fmax(cmax, fabs(Cz[(size_t)r * PP + cc]));
        for (int r = 0; r < PP; ++r)
            for (int cc = 0; cc < PP; ++cc) {
                int j, k, rim, n, m, cim;
                dof_decode(r, j, k, rim);
                dof_decode(cc, n, m, cim);
                if (k != m || rim != cim) off = fmax(off, fabs(Cz[(size_t)r * PP + cc]));
            }
        for (int m = 0; m < P; ++m)
            for (int j = m; j < P; ++j)
                for (int n = m; n < P; ++n) {
                    const double cre = Cz[(size_t)(m == 0 ? j * j : j * j + 2 * m - 1) * PP + (m == 0 ? n * n : n * n + 2 * m - 1)];
                    if (m > 0) imdiff = fmax(imdiff, fabs(cre - Cz[(size_t)(j * j + 2 * m) * PP + n * n + 2 * m]));
                    o[at++] = (float)cre;
                }
        if (off > 1e-12 * cmax || imdiff > 1e-12 * cmax) return -2;
        // F^-1 C F against the dense operator
        std::vector<double> CF((size_t)PP * PP, 0.0);
        for (int r = 0; r < PP; ++r)
            for (int k2 = 0; k2 < PP; ++k2) {
                const double cv = Cz[(size_t)r * PP + k2];
                if (cv == 0.0) continue;
                for (int cc = 0; cc < PP; ++cc) CF[(size_t)r * PP + cc] += cv * Fd[(size_t)k2 * PP + cc];
            }
        double err = 0.0, tmax = 0.0;
        for (int r = 0; r < PP; ++r)
            for (int cc = 0; cc < PP; ++cc) {
                double acc = 0.0;
                for (int k2 = 0; k2 < PP; ++k2) acc += Fi[(size_t)r * PP + k2] * CF[(size_t)k2 * PP + cc];
                err = fmax(err, fabs(acc - T[(size_t)r * PP + cc]));
                tmax = fmax(tmax, fabs(T[(size_t)r * PP + cc]));
            }
        if (err > 1e-9 * tmax) return -3;
    }
    return 0;
}

// ------------------------------------------------------------------------------------------
// FP32 helpers
// ------------------------------------------------------------------------------------------

// ------------------------------------------------------------------------------------------
// Cell geometry tables.  The centre of a level-l cell with integer coordinates (ix, iy, iz) is
// origin + (i + 1/2) h_l per axis, h_l = side / 2^l, and its inverse side 1 / h_l: FP64
// expressions rounded to FP32.  FP64 runs at a small fraction of the FP32 rate, so they are
// evaluated once per level and axis (uniform tree) or once per cell (adaptive tree) into a
// table that the expansion kernels read, instead of once per particle or per (particle, cell)
// pair.
//   uniform: geo[l] = 1/h_l for l < kGeoLevels, then for l = 0..L the 2^l centre coordinates
//            along x, then y, then z, at offset kGeoLevels + 3 (2^l - 1)
//   adaptive: geom[c] = (cx, cy, cz, 1/h) of cell c
// ------------------------------------------------------------------------------------------
GB_DEV CellGeom geo_level_cell(const float *__restrict__ geo, int l, uint32_t key)
{
    int ix, iy, iz;
    demorton3(key, ix, iy, iz);
    const float *a = geo + kGeoLevels + 3 * ((1 << l) - 1);
    CellGeom g;
    g.cx = __ldg(a + ix);
    g.cy = __ldg(a + (1 << l) + iy);
    g.cz = __ldg(a + (2 << l) + iz);
    g.inv_h = __ldg(geo + l);
    return g;
}

GB_DEV CellGeom geo_cell(const float4 *__restrict__ geom, int64_t c)
{
    const float4 v = __ldg(&geom[c]);
    CellGeom g;
    g.cx = v.x;
    g.cy = v.y;
    g.cz = v.z;
    g.inv_h = v.w;
    return g;
}

// ------------------------------------------------------------------------------------------
// P2M: NL lanes per leaf; each strides over the leaf's particles and accumulates the full
// real-packed expansion in registers, then the lanes' sums are added through shared memory.
// ------------------------------------------------------------------------------------------
// acc += sum over particles j = b0 + lane, b0 + lane + NL, ... < e0 of q_j conj(H_n^m(x^_j)) / k_n^m,
// x^ = (x - c) / h, with H the regular harmonics R (P2M, Eq. 2) or the irregular harmonics I
// (P2L, Eq. 3), real-packed.  The harmonics of one m are a power of x + iy (irregular: over r^2)
// times real functions of one recurrence in n, H_n^m = k_n^m E_m g_n with
//   g_m = 1, g_n = u g_{n-1} - beta_n^m v g_{n-2},   (u, v) = (z, r^2), irregular (z, 1) / r^2,
// so a term costs 3 operations for the real recurrence and 2 sums instead of 8 or 10 with complex
// ones; the constants k enter once per expansion (lanes_store).
template <int P, bool IRREG, int NL>
GB_DEV void p2x_particles(float (&acc)[P * P], const float4 *__restrict__ sx, int b0, int e0, int lane,
                          const CellGeom &cg)
{
    for (int j = b0 + lane; j < e0; j += NL) {
        const float4 p = __ldg(&sx[j]);
        const float x = (p.x - cg.cx) * cg.inv_h, y = (p.y - cg.cy) * cg.inv_h, z = (p.z - cg.cz) * cg.inv_h;
        const float r2 = x * x + y * y + z * z;
        const float ir = IRREG ? rsqrt_ftz(r2) : 1.f, v = IRREG ? ir * ir : r2;
        const float u = IRREG ? z * v : z, xr = IRREG ? x * v : x, xi = IRREG ? y * v : y;
        float er = IRREG ? p.w * ir : p.w, ei = 0.f;  // E_m = q (1/r) (x + iy)^m
#pragma unroll
        for (int m = 0; m < P; ++m) {
            if (m == 1) {
                ei = xi * er;
                er = xr * er;
            } else if (m > 1) {
                const float tr = xr * er - xi * ei;
                ei = xr * ei + xi * er;
                er = tr;
            }
            float g1 = 1.f, g2 = 0.f;
#pragma unroll
            for (int n = m; n < P; ++n) {
                if (n == m) {
                    acc[re_idx(n, m)] += er;
                    if (m > 0) acc[im_idx(n, m)] -= ei;
                    continue;
                }
                const float g = n == m + 1 ? u : fmaf(c_nbeta1[n][m], n == m + 2 ? v : v * g2, u * g1);
                g2 = g1;
                g1 = g;
                acc[re_idx(n, m)] = fmaf(er, g, acc[re_idx(n, m)]);
                if (m > 0) acc[im_idx(n, m)] = fmaf(-ei, g, acc[im_idx(n, m)]);
            }
        }
    }
}

// The sums of acc over each NL lanes of the warp, times k_n^m, stored to (or added into) the
// lanes' dst (the same for the NL lanes; nullptr: nothing): a transpose through the warp's
// shared-memory scratch in two halves of the coefficients (each lane writes its row, then a lane
// per coefficient sums its column over the NL rows).  scr holds 32 x LD floats.
template <int P>
struct WarpSum {
    static constexpr int PP = P * P, H = (PP + 1) / 2, LD = H + 1;
};

template <int P, int NL>
GB_DEV void lanes_store(float (&acc)[P * P], float *dst, int lane, bool add, float *scr)
{
    using W = WarpSum<P>;
    constexpr int NG = 32 / NL;
#pragma unroll
    for (int part = 0; part < 2; ++part) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < W::H; ++i)
            if (part * W::H + i < W::PP) scr[lane * W::LD + i] = acc[part * W::H + i];
        __syncwarp();
        for (int i0 = 0; i0 < NG * W::H; i0 += 32) {
            const int e = i0 + lane, gr = min(e / W::H, NG - 1), i = e - gr * W::H, k = part * W::H + i;
            float *d = reinterpret_cast<float *>(
                __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst), gr * NL));
            if (i >= W::H || k >= W::PP || !d) continue;
            float v = 0.f;
#pragma unroll 8
            for (int r = 0; r < NL; ++r) v += scr[(gr * NL + r) * W::LD + i];
            v *= __ldg(&d_kscale[k]);
            d[k] = add ? d[k] + v : v;
        }
    }
}

template <int P, int NL>
__global__ void __launch_bounds__(128) k_p2m(int L, const float *__restrict__ geo, const float4 *__restrict__ sx,
                                             const int32_t *__restrict__ begin, const int32_t *__restrict__ end,
                                             float *__restrict__ M)
{
    __shared__ float scr[4][32 * WarpSum<P>::LD];
    const int lane = threadIdx.x & 31;
    const int64_t leaf = (blockIdx.x * (int64_t)4 + (threadIdx.x >> 5)) * (32 / NL) + lane / NL;
    const int64_t g = level_offset(L) + leaf;
    int b0 = 0, e0 = 0;
    if (leaf < (int64_t(1) << (3 * L))) b0 = begin[g], e0 = end[g];
    if (__all_sync(0xffffffffu, e0 <= b0)) return;
    float acc[P * P];
#pragma unroll
    for (int i = 0; i < P * P; ++i) acc[i] = 0.f;
    if (e0 > b0) {
        const CellGeom cg = geo_level_cell(geo, L, (uint32_t)leaf);
        p2x_particles<P, false, NL>(acc, sx, b0, e0, lane % NL, cg);
    }
    lanes_store<P, NL>(acc, e0 > b0 ? M + g * (P * P) : nullptr, lane, false, scr[threadIdx.x >> 5]);
}

// Lanes per leaf of P2M, by the expected number of leaves and not the counted one (a captured
// batch lays its trees out for more): 8 where the leaves fill the GPU at four to a warp (rounds of
// 8 waste fewer lanes than rounds of 32 on 15 to 40 particles, and 8 rows are added instead of
// 32), else 32, a leaf's particles in as few rounds as possible.  P2M, 32 lanes and complex
// recurrences -> 8 lanes and real ones: 1M uniform p = 10 64 -> 32 us, 5M p = 6 149 -> 62, 16M
// Plummer p = 8 1122 -> 407; P2L there 2036 -> 1108 (16 lanes a cell).
constexpr int64_t kP2MManyLeaves = 8 * 1024;

// P2M starts beside P2P, with priority.  An SM that runs it under another split of shared memory and L1
// than P2P's takes no P2P CTA until it is idle, and P2P's CTAs crowded onto the rest, eight on 60 SMs
// and none on 90 (100,000 Plummer particles, 465 leaves of up to 1024): so it asks for P2P's split.
// Forked evaluations with it: that one 3.59 .. 4.59 -> 3.21 ms, 400,009 with leaves of up to 512 3.45 -> 2.5.
template <class K>
static void p2m_carveout(K k)
{
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}

void launch_p2m(int P, int L, const float *geo, const float4 *sx, const int32_t *begin, const int32_t *end, float *M,
                cudaStream_t s)
{
    const int64_t nl = int64_t(1) << (3 * L);
    if (nl >= kP2MManyLeaves) {
        const unsigned grid = (unsigned)((nl + 15) / 16);
        GBFMM_DISPATCH_P(P, (p2m_carveout(k_p2m<PQ, 8>), k_p2m<PQ, 8><<<grid, 128, 0, s>>>(L, geo, sx, begin, end, M)));
    } else {
        const unsigned grid = (unsigned)((nl + 3) / 4);
        GBFMM_DISPATCH_P(P, (p2m_carveout(k_p2m<PQ, 32>), k_p2m<PQ, 32><<<grid, 128, 0, s>>>(L, geo, sx, begin, end, M)));
    }
    note_launches(1);
}

// ------------------------------------------------------------------------------------------
// M2M and L2L as batched FP32 contractions over 32 cells per CTA, the same register-blocked
// micro-kernel as M2L (4 operator rows x 8 cells per thread) on shared-memory-staged operands.
//   M2M (UP):  M~(parent q) = sum over child positions c of T^M2M_c M~(child 8q + c)
//   L2L (!UP): L~(child 8q + c) += T^L2L_c L~(parent q), one child position per CTA column
// M2M is block lower-triangular in degree (output degree j reads input degrees <= j) and L2L
// block upper-triangular (reads degrees >= j): each thread's k range is cut to its rows'
// degrees (rounded to whole k-groups of 4).
// ------------------------------------------------------------------------------------------
constexpr int kTrTN = 32, kTrCN = 8;
// k_m2m_small up to this many CTAs (700 parents at p = 10); beyond, k_translate's operator is staged
// for more cells (1,040 parents: 20 us either way)
constexpr int kTransSmallCtas = 4 * kSms;

template <int P, bool UP, int TN = kTrTN, int CN = kTrCN>
struct TransCfg {
    static constexpr int PP = P * P, PR = ops_rows_padded(P), SB = staged_col_stride(P);
    static constexpr int NCG = TN / CN, NRG = PR / 4, NT = ((NRG * NCG + 31) / 32) * 32;
    static constexpr int AF = PP * PR, BF = TN * SB;  // floats of one operator / one column block
    static constexpr int NBUF = UP ? 2 : 1;           // M2M walks 8 child positions: double-buffered
    static constexpr size_t kSmem = (size_t)NBUF * (AF + BF) * sizeof(float);
};

GB_DEV int degree_of(int r)
{
    int d = 0;
    while ((d + 1) * (d + 1) <= r) ++d;
    return d;
}

GB_DEV void cp_async16_t(void *dst, const void *src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(src_bytes)
                 : "memory");
}

// TN cells per CTA; the operator of each child position and the TN source columns are copied
// into shared memory with cp.async (zero-filled for missing cells), the next child position's
// copies in flight while the current one is applied
template <int P, bool UP, int TN, int CN>
__global__ void __launch_bounds__(TransCfg<P, UP, TN, CN>::NT) k_translate(int l, const int32_t *__restrict__ begin,
                                                                       const int32_t *__restrict__ end,
                                                                       const float *__restrict__ ops,
                                                                       float *__restrict__ X)
{
    using Cfg = TransCfg<P, UP, TN, CN>;
    constexpr int PP = Cfg::PP, PR = Cfg::PR, SB = Cfg::SB, NCG = Cfg::NCG, NRG = Cfg::NRG;
    extern __shared__ __align__(16) float tsm[];
    // parents: level l (M2M) or l - 1 (L2L)
    const int lp = UP ? l : l - 1;
    const int64_t np = int64_t(1) << (3 * lp);
    const int64_t q0 = blockIdx.x * (int64_t)TN;
    const int64_t offp = level_offset(lp), offc = level_offset(lp + 1);
    const int tid = threadIdx.x;
    const bool work = tid < NRG * NCG;
    const int cg = tid % NCG, rg = tid / NCG;
    int kbeg = 0, kend = PP;
    if (work) {
        const int r0 = min(rg * 4, PP - 1), r1 = min(rg * 4 + 3, PP - 1);
        if (UP) {
            const int d = degree_of(r1);
            kend = min(PP, ((d + 1) * (d + 1) + 3) / 4 * 4);
        } else {
            const int d = degree_of(r0);
            kbeg = (d * d) / 4 * 4;
        }
    }
    auto stage = [&](int c, int buf) {
        float *A = tsm + buf * (Cfg::AF + Cfg::BF);
        float *B = A + Cfg::AF;
        const float *src = ops + (size_t)c * PP * PR;
        for (int e = tid; e < PP * PR / 4; e += blockDim.x) cp_async16_t(A + 4 * e, src + 4 * e, 16u);
        for (int e = tid; e < TN * (PP / 4); e += blockDim.x) {
            const int i = e / (PP / 4), k4 = e % (PP / 4);
            const int64_t q = q0 + i;
            const float *gsrc = X;
            uint32_t bytes = 0;
            if (q < np) {
                const int64_t g = UP ? offc + 8 * q + c : offp + q;
                if (end[g] > begin[g]) {
                    gsrc = X + g * PP + 4 * k4;
                    bytes = 16u;
                }
            }
            cp_async16_t(B + i * SB + 4 * k4, gsrc, bytes);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float tot[4][CN];  // M2M: the child positions' sums, added in order (as k_m2m_small adds them)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < CN; ++j) tot[i][j] = 0.f;
    const int c_first = UP ? 0 : blockIdx.y, c_last = UP ? 7 : blockIdx.y;
    stage(c_first, 0);
    for (int c = c_first; c <= c_last; ++c) {
        const int buf = UP ? (c - c_first) & 1 : 0;
        if (c < c_last) {
            stage(c + 1, buf ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        if (work) {
            const float *Ar = tsm + buf * (Cfg::AF + Cfg::BF) + rg * 4;
            const float *Bc = tsm + buf * (Cfg::AF + Cfg::BF) + Cfg::AF + cg * SB;
            float acc[4][CN];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < CN; ++j) acc[i][j] = 0.f;
#pragma unroll 2
            for (int k = kbeg; k < kend; k += 4) {
                Frag<CN, 4> f;
                f.load(Ar, Bc, k, PR, NCG * SB);
                f.fma(acc);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < CN; ++j) tot[i][j] += acc[i][j];
        }
        __syncthreads();  // the buffer is refilled two positions later
    }
    if (!work) return;
#pragma unroll
    for (int j = 0; j < CN; ++j) {
        const int64_t q = q0 + cg + j * NCG;
        if (q >= np) continue;
        const int r = rg * 4;
        if (r >= PP) continue;
        const int64_t g = UP ? offp + q : offc + 8 * q + blockIdx.y;
        if (end[g] <= begin[g]) continue;
        float4 *dst = reinterpret_cast<float4 *>(X + g * PP + r);
        if (UP) {
            *dst = make_float4(tot[0][j], tot[1][j], tot[2][j], tot[3][j]);
        } else {
            float4 v = *dst;
            v.x += tot[0][j];
            v.y += tot[1][j];
            v.z += tot[2][j];
            v.w += tot[3][j];
            *dst = v;
        }
    }
}

// M2M of small levels.  k_translate takes the 8 child positions one after another, on few CTAs,
// each position waiting for its p^2 x p^2 operator: 9 / 16 / 22 us a level at p = 4 / 8 / 10 however
// few its cells.  Here a CTA takes 8 parents and one of SL slices of the output rows, and eight
// thread groups take the eight child positions at once: all copies (the slices of the eight
// operators and the columns, cut to the degrees the slice reads) are issued together and waited
// for once.  The groups' sums are added in child order through shared memory, so every sum is
// formed as in k_translate and k_translate_cells.  At p = 10 a level of
// 64 / 512 parents takes 7.5 / 13 us (k_translate 20); beside P2P small CTAs also find room sooner
// (16 parents and 143 KB a CTA: 10 us, and no gain in the 1M step).  L2L has one position per
// CTA already: the same form took 10 us there against 7.  `Cells` maps parent ordinals q < np to cells: parent(q),
// child(q, c), -1: none.
template <int P>
struct TransSmall {
    static constexpr int PP = P * P, PR = ops_rows_padded(P), SB = staged_col_stride(P);
    static constexpr int TN = 8, CN = 1, NCG = TN / CN, NRG = PR / 4;
    static constexpr int SL = P == 4 ? 1 : P == 6 ? 3 : P == 8 ? 4 : 7;  // row slices
    static constexpr int RGS = (NRG + SL - 1) / SL;         // row groups of a slice
    static constexpr int GT = RGS * NCG, NT = 8 * GT;       // threads of a child position, of the CTA
    static constexpr int LDA = 4 * RGS;
    static constexpr size_t kSmem = sizeof(float) * (8 * ((size_t)PP * LDA + (size_t)TN * SB) + (size_t)NT * CN * 4);
};

struct LevelCells {  // uniform tree: parents of level l, children of level l + 1
    int64_t offp, offc, n;
    const int32_t *begin, *end;
    GB_DEV int64_t np() const { return n; }
    GB_DEV int64_t some(int64_t g) const { return end[g] > begin[g] ? g : -1; }
    GB_DEV int64_t parent(int64_t q) const { return some(offp + q); }
    GB_DEV int64_t child(int64_t q, int c) const { return some(offc + 8 * q + c); }
};

struct SpanCells {  // adaptive tree: a span of cells; leaves among them are no parents
    Span par;
    const int32_t *child_of, *nchild;
    GB_DEV int64_t np() const { return span_count(par); }
    GB_DEV int64_t parent(int64_t q) const
    {
        const int64_t g = span_first(par) + q;
        return nchild[g] != 0 ? g : -1;
    }
    GB_DEV int64_t child(int64_t q, int c) const { return child_of[(span_first(par) + q) * 8 + c]; }
};

template <int P, class Cells>
__global__ void __launch_bounds__(TransSmall<P>::NT) k_m2m_small(Cells cells, const float *__restrict__ ops,
                                                                 float *__restrict__ M)
{
    using Cfg = TransSmall<P>;
    constexpr int PP = Cfg::PP, PR = Cfg::PR, SB = Cfg::SB, NCG = Cfg::NCG, TN = Cfg::TN, CN = Cfg::CN;
    constexpr int GT = Cfg::GT, LDA = Cfg::LDA, RGS = Cfg::RGS, NRG = Cfg::NRG;
    extern __shared__ __align__(16) float tsm[];
    __shared__ int64_t s_par[TN], s_child[8][TN];
    const int64_t np = cells.np();
    if (blockIdx.x * (int64_t)TN >= np) return;
    const int tid = threadIdx.x, rg0 = blockIdx.y * RGS, rg1 = min(rg0 + RGS, NRG);
    // the columns k that rows of degree d read: those of degrees <= d
    auto k_end = [](int r) { const int d = degree_of(min(r, PP - 1)); return min(PP, ((d + 1) * (d + 1) + 3) / 4 * 4); };
    const int ke = k_end(4 * rg1 - 1);
    float *B = tsm + 8 * PP * LDA, *red = B + 8 * TN * SB;
    for (int e = tid; e < 8 * PP * RGS; e += Cfg::NT) {
        const int r = e % RGS, k = (e / RGS) % PP, c = e / (RGS * PP);
        if (k < ke && rg0 + r < rg1)
            cp_async16_t(tsm + (c * PP + k) * LDA + 4 * r, ops + ((size_t)c * PP + k) * PR + 4 * (rg0 + r), 16u);
    }
    for (int64_t q0 = blockIdx.x * (int64_t)TN; q0 < np; q0 += (int64_t)gridDim.x * TN) {
        for (int e = tid; e < 9 * TN; e += Cfg::NT) {
            const int i = e % TN, c = e / TN - 1;
            const int64_t g = q0 + i >= np ? -1 : c < 0 ? cells.parent(q0 + i) : cells.child(q0 + i, c);
            (c < 0 ? s_par[i] : s_child[c][i]) = g;
        }
        __syncthreads();
        for (int e = tid; e < 8 * TN * (PP / 4); e += Cfg::NT) {
            const int k = 4 * (e % (PP / 4)), i = (e / (PP / 4)) % TN, c = e / (PP / 4 * TN);
            const int64_t g = s_child[c][i];
            if (k < ke) cp_async16_t(B + (c * TN + i) * SB + k, g >= 0 ? M + g * PP + k : M, g >= 0 ? 16u : 0u);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const int c = tid / GT, t = tid % GT, cg = t % NCG, rl = t / NCG, rg = rg0 + rl;
        float acc[4][CN];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CN; ++j) acc[i][j] = 0.f;
        if (rg < rg1) {
            const int kn = k_end(4 * rg + 3);
            const float *Ar = tsm + c * PP * LDA + 4 * rl, *Bc = B + (c * TN + cg) * SB;
#pragma unroll 2
            for (int k = 0; k < kn; k += 4) {
                Frag<CN, 4> f;
                f.load(Ar, Bc, k, LDA, NCG * SB);
                f.fma(acc);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CN; ++j) red[(i * CN + j) * Cfg::NT + tid] = acc[i][j];
        __syncthreads();
        for (int e = tid; e < 4 * CN * GT; e += Cfg::NT) {
            const int i = e % 4, tt = (e / 4) % GT, j = e / (4 * GT);
            const int r = 4 * (rg0 + tt / NCG) + i;
            const int64_t g = s_par[tt % NCG + j * NCG];
            if (g < 0 || rg0 + tt / NCG >= rg1 || r >= PP) continue;
            float v = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) v += red[(i * CN + j) * Cfg::NT + k * GT + tt];
            M[g * PP + r] = v;
        }
        __syncthreads();  // the columns and the sums are read: the next parents may be staged
    }
}

// false (nothing launched) on levels of more CTAs than kTransSmallCtas
template <int P, class Cells>
static bool launch_m2m_small(int64_t np, const Cells &cells, const float *ops, float *M, cudaStream_t s)
{
    using Cfg = TransSmall<P>;
    const int64_t ctas = (np + Cfg::TN - 1) / Cfg::TN;
    if (ctas * Cfg::SL > kTransSmallCtas) return false;
    cudaFuncSetAttribute(k_m2m_small<P, Cells>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem);
    k_m2m_small<P, Cells><<<dim3((unsigned)ctas, Cfg::SL), Cfg::NT, Cfg::kSmem, s>>>(cells, ops, M);
    note_launches(1);
    return true;
}

template <int P, bool UP, int TN, int CN>
static void launch_translate_tn(int l, const int32_t *begin, const int32_t *end, const float *ops, float *X,
                                cudaStream_t s)
{
    using Cfg = TransCfg<P, UP, TN, CN>;
    cudaFuncSetAttribute(k_translate<P, UP, TN, CN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem);
    const int64_t np = int64_t(1) << (3 * (UP ? l : l - 1));
    dim3 grid((unsigned)((np + TN - 1) / TN), UP ? 1 : 8);
    k_translate<P, UP, TN, CN><<<grid, Cfg::NT, Cfg::kSmem, s>>>(l, begin, end, ops, X);
    note_launches(1);
}

// cells per CTA: 32 (8 per thread) when the level has enough cells to fill the GPU twice over,
// else 16 (2 per thread): small levels are bound by the latency of staging the operators, and
// seven times the threads per cell cut it (M2M levels 2-4 of a 2^20-particle p = 10 tree:
// 150 us -> 68 us)
template <int P, bool UP>
static void launch_translate_t(int l, const int32_t *begin, const int32_t *end, const float *ops, float *X,
                               cudaStream_t s)
{
    const int lp = UP ? l : l - 1;
    const int64_t np = int64_t(1) << (3 * lp);
    if constexpr (UP)
        if (launch_m2m_small<P>(np, LevelCells{level_offset(lp), level_offset(lp + 1), np, begin, end}, ops, X, s)) return;
    const int64_t ctas32 = (np + 31) / 32 * (UP ? 1 : 8);
    if (ctas32 >= 2 * kSms)
        launch_translate_tn<P, UP, 32, 8>(l, begin, end, ops, X, s);
    else
        launch_translate_tn<P, UP, 16, 2>(l, begin, end, ops, X, s);
}

void launch_m2m(int P, int l, const int32_t *begin, const int32_t *end, const float *ops, float *M, cudaStream_t s)
{
    switch (P) {
    case 4: launch_translate_t<4, true>(l, begin, end, ops, M, s); break;
    case 6: launch_translate_t<6, true>(l, begin, end, ops, M, s); break;
    case 8: launch_translate_t<8, true>(l, begin, end, ops, M, s); break;
    case 10: launch_translate_t<10, true>(l, begin, end, ops, M, s); break;
    }
}

void launch_l2l(int P, int l, const int32_t *begin, const int32_t *end, const float *ops, float *Lc, cudaStream_t s)
{
    switch (P) {
    case 4: launch_translate_t<4, false>(l, begin, end, ops, Lc, s); break;
    case 6: launch_translate_t<6, false>(l, begin, end, ops, Lc, s); break;
    case 8: launch_translate_t<8, false>(l, begin, end, ops, Lc, s); break;
    case 10: launch_translate_t<10, false>(l, begin, end, ops, Lc, s); break;
    }
}

// ------------------------------------------------------------------------------------------
// L2P: one thread per particle (sorted order).  phi = (1/h) sum L~ R(x^), grad = (1/h^2) x
// ladder sums, x^ = (x - c) / h:
//   dphi/dz            = sum_{n<P-1} sum_m sqrt((n+1-m)(n+1+m)) L_{n+1}^m R_n^m
//   dphi/dx + i dphi/dy = sum_{n<P-1} sum_m s(m) sqrt((n+2-m)(n+1-m)) L_{n+1}^{m-1} R_n^m,
//   s(m) = +1 for m >= 1, -1 for m <= 0.
// ------------------------------------------------------------------------------------------
// With R_n^m = E_m g_n, E_m a constant times (x^ + i y^)^m and g_n real, every m needs three complex
// sums, F_m = sum L_n^m g_n, Z_m = sum sqrt((n+1-m)(n+1+m)) L_{n+1}^m g_n and
// A_m = sum sqrt((n+2-m)(n+1-m)) L_{n+1}^{m-1} g_n; the lowered term of dphi/dx + i dphi/dy follows
// from F_m and A_{m+1} as in M2P (there in powers of xi), with the constants' ratios
// E_m / (x^ + i y^) E_{m-1} = -c_rmm[m].  Half the operations of complex recurrences and four sums,
// and each coefficient is read once, a column of L at a time, instead of five times.
template <int P>
struct L2PState {
    float x, y, z, r2, rho2;
    float phi = 0.f, gz = 0.f, gr = 0.f, gi = 0.f;
    float er = 1.f, ei = 0.f, er1 = 0.f, ei1 = 0.f;  // E_m, E_{m-1}
    float fr1 = 0.f, fi1 = 0.f;                      // F_{m-1}
    float pr[P], pi[P];                              // L_n^{m-1}
};

// orders M, M + 1, ..., P (P: the last lowered term only)
template <int P, int M>
GB_DEV void l2p_orders(L2PState<P> &s, const float *__restrict__ Lg)
{
    float fr = 0.f, fi = 0.f, zr = 0.f, zi = 0.f, ar = 0.f, ai = 0.f;
    const float er2 = s.er1, ei2 = s.ei1;  // E_{m-2}
    if constexpr (M > 0 && M < P) {
        s.er1 = s.er, s.ei1 = s.ei;
        const float f = -c_rmm[M];
        s.er = f * (s.x * s.er1 - s.y * s.ei1);
        s.ei = f * (s.x * s.ei1 + s.y * s.er1);
    }
    if constexpr (M < P) {
        float cr[P], ci[P];
#pragma unroll
        for (int n = M; n < P; ++n) {
            cr[n] = __ldg(&Lg[re_idx(n, M)]);
            ci[n] = M > 0 ? __ldg(&Lg[im_idx(n, M)]) : 0.f;
        }
        float g1 = 1.f, g2 = 0.f;
#pragma unroll
        for (int n = M; n < P; ++n) {
            float g = 1.f;
            if (n > M) {
                g = c_ra[n - 1][M] * (s.z * g1);
                if (n > M + 1) g = fmaf(-c_rb[n - 1][M], s.r2 * g2, g);
                g2 = g1;
                g1 = g;
            }
            fr = fmaf(cr[n], g, fr);
            if (M > 0) fi = fmaf(ci[n], g, fi);
            if (n + 1 < P) {
                const float gs = c_sq[n + 1 - M][n + 1 + M] * g;
                zr = fmaf(cr[n + 1], gs, zr);
                if (M > 0) {
                    zi = fmaf(ci[n + 1], gs, zi);
                    const float ga = c_sq[n + 2 - M][n + 1 - M] * g;
                    ar = fmaf(s.pr[n + 1], ga, ar);
                    if (M > 1) ai = fmaf(s.pi[n + 1], ga, ai);
                }
            }
        }
        if (M == 0) {
            s.phi = fr;
            s.gz = zr;
        } else {
            s.phi = fmaf(2.f, s.er * fr - s.ei * fi, s.phi);
            s.gz = fmaf(2.f, s.er * zr - s.ei * zi, s.gz);
            s.gr += s.er * ar - s.ei * ai;
            s.gi += s.er * ai + s.ei * ar;
        }
#pragma unroll
        for (int n = M; n < P; ++n) {
            s.pr[n] = cr[n];
            s.pi[n] = ci[n];
        }
    }
    if constexpr (M >= 2) {  // the lowered term of order M - 1, with E_{M-2}
        const float e0 = M < P ? er2 : s.er1, e1 = M < P ? ei2 : s.ei1;
        const float cf = -2.f * (M - 1) * c_rmm[M - 1], ca = M < P ? c_rmm[M] * c_rmm[M - 1] * s.rho2 : 0.f;
        const float tr = fmaf(cf, s.fr1, ca * ar), ti = fmaf(cf, s.fi1, ca * ai);
        s.gr += e0 * tr - e1 * ti;
        s.gi -= e0 * ti + e1 * tr;
    }
    s.fr1 = fr;
    s.fi1 = fi;
    if constexpr (M < P) l2p_orders<P, M + 1>(s, Lg);
}

// value and gradient of the scaled local expansion Lg at x^ (multiplied by 1/h and 1/h^2)
template <int P>
GB_DEV float4 l2p_eval(const float *__restrict__ Lg, float x, float y, float z, float ih)
{
    L2PState<P> s;
    s.x = x, s.y = y, s.z = z;
    s.rho2 = x * x + y * y;
    s.r2 = s.rho2 + z * z;
    l2p_orders<P, 0>(s, Lg);
    const float ih2 = ih * ih;
    return make_float4(s.phi * ih, s.gr * ih2, s.gi * ih2, s.gz * ih2);
}

// the near-field compensated sums of particle i (sorted order: the sums, then their
// compensations) completed with the far field, in the order the P2P kernel adds it
GB_DEV float4 near_plus_far(const float4 *__restrict__ near, int64_t i, float4 f)
{
    const float4 s = near[2 * i], c = near[2 * i + 1];
    Kahan a{s.x, c.x}, bx{s.y, c.y}, by{s.z, c.z}, bz{s.w, c.w};
    a.add(f.x);
    bx.add(f.y);
    by.add(f.z);
    bz.add(f.w);
    return make_float4(a.s, bx.s, by.s, bz.s);
}

template <int P>
__global__ void __launch_bounds__(128) k_l2p(int L, const float *__restrict__ geo, int64_t n,
                                             const float4 *__restrict__ sx, const uint32_t *__restrict__ leafkey,
                                             const float *__restrict__ Lc, float4 *__restrict__ far,
                                             const float4 *__restrict__ near, const uint32_t *__restrict__ perm,
                                             float4 *__restrict__ out)
{
    constexpr int PP = P * P;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t key = leafkey[i];
    const int64_t g = level_offset(L) + key;
    const CellGeom cg = geo_level_cell(geo, L, key);
    float4 p = __ldg(&sx[i]);
    const float4 f = l2p_eval<P>(Lc + g * PP, (p.x - cg.cx) * cg.inv_h, (p.y - cg.cy) * cg.inv_h,
                                 (p.z - cg.cz) * cg.inv_h, cg.inv_h);
    if (near)
        out[perm[i]] = near_plus_far(near, i, f);
    else
        far[i] = f;
}

void launch_l2p(int P, int L, const float *geo, int64_t n, const float4 *sx, const uint32_t *leafkey, const float *Lc,
                float4 *far, cudaStream_t s, const float4 *near, const uint32_t *perm, float4 *out)
{
    if (n <= 0) return;
    unsigned grid = (unsigned)((n + 127) / 128);
    GBFMM_DISPATCH_P(P, (k_l2p<PQ><<<grid, 128, 0, s>>>(L, geo, n, sx, leafkey, Lc, far, near, perm, out)));
    note_launches(1);
}

// ------------------------------------------------------------------------------------------
// M2P (treecode far field; the adaptive FMM's W lists): the multipole of a source cell evaluated
// at a target particle.  With x^ = (x - c)/h:
//   phi = (1/h) sum M~_n^m I_n^m(x^)
//   dphi/dz             = -(1/h^2) sum sqrt((n+1-m)(n+1+m)) M~_n^m I_{n+1}^m
//   dphi/dx + i dphi/dy =  (1/h^2) sum s(m) sqrt((n+m+2)(n+m+1)) M~_n^m I_{n+1}^{m+1},
//   s(m) = +1 for m >= 0, -1 for m < 0.
// ------------------------------------------------------------------------------------------
// With xi = (x^ + i y^) / r^2 and u = z^ / r^2 the harmonics of one m are a power of xi times real
// functions of one recurrence in N,
//   I_N^m = (1/r) k_N^m xi^m g_N,   g_m = 1,  g_N = u g_{N-1} - beta_N^m (1/r^2) g_{N-2},
// the constants k absorbing the recurrence's factors (m2p_tables).  With three complex sums per m,
//   F_m = sum w k_N M_N^m g_N,   Z_m = -sum w k_N sqrt((N-m)(N+m)) M_{N-1}^m g_N,
//   A_m = sum k_N sqrt((N+m)(N+m-1)) M_{N-1}^{m-1} g_N          (w = 2 for m > 0, else 1)
// every m contributes Re(xi^m F_m) to phi, Re(xi^m Z_m) to dphi/dz and to dphi/dx + i dphi/dy
//   xi^m A_m + conj(xi^{m-1} (m F_m / r^2 + |xi|^2 A_{m+1}))     (the second for m >= 1),
// the lowered term following from (d/dx - i d/dy)(X^m h) = X^{m-1} (2 m h + |X|^2 2 dh/d(r^2)): 9
// FP32-pipe operations per (N, m) instead of the 14 of complex recurrences and four sums, and half
// their rounding error against FP64.
//
// Two source cells share every instruction (packed FP32, a lane each): per pair of cells the warp
// stages both expansions (cp.async, one step ahead) and folds the constants in, so that a record
// of three 16-byte loads per (N, m) holds {F re, F im}, {Z re, Z im}, {A re, A im}, each a (cell 0,
// cell 1) pair.  Issue-bound before (complex recurrences, one cell at a time: 73% issue, FP32 pipe
// 40% of active cycles).
//
// The four warps of a CTA take a target leaf, the sources of its rows dealt to them 2 G at a time
// (one warp a leaf: the longest rows were the tail, and half the GPU's warps idle); targets go in
// chunks of up to 32, and a chunk of T < 32 takes G = min(GMAX, 32 / T) pairs of cells a step (lane
// l: target l % T, pair l / T).  The lanes' partial sums are added in warp and group order.
// M2P alone, the earlier kernels (a warp or a CTA of 64 per leaf) -> this one: treecode, 131,072
// uniform p = 6 1325 -> 653 us, 50,021 Plummer p = 8 2348 -> 1023; W rows, 20,011 Plummer p = 4
// 59 -> 27, 400,009 p = 10 428 -> 234, 16M p = 8 3587 -> 2793.
template <int P>
struct M2PW {
    static constexpr int PP = P * P, NM = (P + 1) * (P + 2) / 2, NO = 6 * NM;
    static constexpr int GMAX = P <= 6 ? 4 : 2;
    static constexpr int kF = GMAX * NO * 8, kM = 2 * 2 * GMAX * PP * 4, kG = 2 * 2 * GMAX * 16;  // bytes per warp
    static constexpr int kWarp = kF + kM + kG;
    static_assert(kF % 16 == 0 && kM % 16 == 0 && GMAX * NO * 8 >= 32 * 16, "alignment; F also holds the lanes' sums");
};

GB_HD constexpr int nm_idx(int N, int m) { return N * (N + 1) / 2 + m; }

// from here on four leaves a CTA (most W rows of a large tree are empty); fewer leaves are spread
// over more CTAs (4,096 leaves, four a CTA: 887 us instead of 653)
constexpr int64_t kM2PManyLeaves = 1 << 16;
constexpr int kM2PMaxNO = 3 * (kMaxP + 1) * (kMaxP + 2);
// per compiled order (4, 6, 8, 10) and folded coefficient 6 nm_idx(N, m) + {F re, im, Z re, im, A re,
// im}: its source coefficient and factor (as bits); 0, 0 where there is none
__device__ int2 d_m2p_tab[4][kM2PMaxNO];
__constant__ uint64_t c_nbeta[kMaxP + 1][kMaxP + 1];  // (-beta, -beta) of (N, m)

// the host copies of those tables and of c_nbeta1 and d_kscale
struct M2PTables {
    int2 tab[4][kM2PMaxNO] = {};
    uint64_t nbeta[kMaxP + 1][kMaxP + 1] = {};
    float nbeta1[kMaxP + 1][kMaxP + 1] = {}, kscale[kMaxP * kMaxP] = {};
    M2PTables();
};

M2PTables::M2PTables()
{
    auto ra = [](int n, int m) { return (2.0 * n + 1.0) / sqrt((double)(n + 1 - m) * (n + 1 + m)); };
    auto rb = [](int n, int m) { return sqrt((double)(n - m) * (n + m)) / sqrt((double)(n + 1 - m) * (n + 1 + m)); };
    const int orders[4] = {4, 6, 8, 10};
    double gamma = 1.0;
    for (int m = 0; m <= kMaxP; ++m) {
        if (m > 0) gamma *= -sqrt((2.0 * m - 1.0) / (2.0 * m));
        const double w = m > 0 ? 2.0 : 1.0;
        double k = gamma;  // k_N^m
        for (int N = m; N <= kMaxP; ++N) {
            if (N > m) k *= ra(N - 1, m);
            if (N > m + 1) {
                const float f = (float)(-rb(N - 1, m) / (ra(N - 1, m) * ra(N - 2, m)));
                uint32_t bits;
                memcpy(&bits, &f, 4);
                nbeta[N][m] = (uint64_t)bits << 32 | bits;
                nbeta1[N][m] = f;
            }
            if (N < kMaxP) {
                kscale[re_idx(N, m)] = (float)k;
                if (m > 0) kscale[im_idx(N, m)] = (float)k;
            }
            for (int o = 0; o < 4; ++o) {
                const int P = orders[o];
                if (N > P) continue;
                auto put = [&](int j, int n, int mm, double c) {  // complex coefficient M_n^mm, factor c
                    const float f = (float)c;
                    int bits;
                    memcpy(&bits, &f, 4);
                    tab[o][6 * nm_idx(N, m) + 2 * j] = make_int2(re_idx(n, mm), bits);
                    if (mm > 0) tab[o][6 * nm_idx(N, m) + 2 * j + 1] = make_int2(im_idx(n, mm), bits);
                };
                if (N < P) put(0, N, m, k * w);
                if (N > m) put(1, N - 1, m, -k * w * sqrt((double)(N - m) * (N + m)));
                if (m > 0) put(2, N - 1, m - 1, k * sqrt((double)(N + m) * (N + m - 1)));
            }
        }
    }
}

void m2p_tables()
{
    static const M2PTables t;  // built once: contexts are created from several threads
    cudaMemcpyToSymbol(d_m2p_tab, t.tab, sizeof(t.tab));
    cudaMemcpyToSymbol(c_nbeta, t.nbeta, sizeof(t.nbeta));
    cudaMemcpyToSymbol(c_nbeta1, t.nbeta1, sizeof(t.nbeta1));
    cudaMemcpyToSymbol(d_kscale, t.kscale, sizeof(t.kscale));
}

GB_DEV uint64_t neg2(uint64_t v) { return v ^ 0x8000000080000000ull; }

// o += potential and gradient at p of the two cells of geometry g0, g1 and folded coefficients R
template <int P>
GB_DEV void m2p_pair(const ulonglong2 *__restrict__ R, float4 p, float4 g0, float4 g1, uint64_t (&o)[4])
{
    const uint64_t x = pack2((p.x - g0.x) * g0.w, (p.x - g1.x) * g1.w);
    const uint64_t y = pack2((p.y - g0.y) * g0.w, (p.y - g1.y) * g1.w);
    const uint64_t z = pack2((p.z - g0.z) * g0.w, (p.z - g1.z) * g1.w);
    float a, b;
    unpack2(fma2(x, x, fma2(y, y, mul2(z, z))), a, b);
    const uint64_t ir = pack2(rsqrt_ftz(a), rsqrt_ftz(b)), ir2 = mul2(ir, ir);
    const uint64_t u = mul2(z, ir2), xr = mul2(x, ir2), xi = mul2(y, ir2), nxi = neg2(xi);
    const uint64_t q2 = fma2(xr, xr, mul2(xi, xi));
    uint64_t er = 0, ei = 0, er1 = 0, ei1 = 0, er2, ei2;  // xi^m, xi^(m-1), xi^(m-2) (m = 0: 1, not held)
    uint64_t fr1 = 0, fi1 = 0;                             // F_{m-1}
    uint64_t phi = 0, gr = 0, gi = 0, gz = 0;
#pragma unroll
    for (int m = 0; m <= P; ++m) {
        er2 = er1, ei2 = ei1, er1 = er, ei1 = ei;
        if (m == 1) {
            er = xr, ei = xi;
        } else if (m > 1) {
            er = fma2(xr, er1, mul2(nxi, ei1));
            ei = fma2(xr, ei1, mul2(xi, er1));
        }
        uint64_t fr = 0, fi = 0, zr = 0, zi = 0, ar = 0, ai = 0, g1 = 0, g2 = 0;
#pragma unroll
        for (int N = m; N <= P; ++N) {
            const int q = 3 * nm_idx(N, m);
            if (N == m) {  // g = 1
                if (N < P) {
                    const ulonglong2 f = R[q];
                    fr = f.x, fi = f.y;
                }
                if (m > 0) {
                    const ulonglong2 c = R[q + 2];
                    ar = c.x, ai = c.y;
                }
                continue;
            }
            uint64_t g;
            if (N == m + 1)
                g = u;
            else
                g = fma2(c_nbeta[N][m], N == m + 2 ? ir2 : mul2(ir2, g2), mul2(u, g1));
            g2 = g1, g1 = g;
            if (N < P) {
                const ulonglong2 f = R[q];
                fr = fma2(f.x, g, fr);
                if (m > 0) fi = fma2(f.y, g, fi);
            }
            const ulonglong2 c = R[q + 1];
            if (N == m + 1) {
                zr = mul2(c.x, g);
                if (m > 0) zi = mul2(c.y, g);
            } else {
                zr = fma2(c.x, g, zr);
                if (m > 0) zi = fma2(c.y, g, zi);
            }
            if (m > 0) {
                const ulonglong2 d = R[q + 2];
                ar = fma2(d.x, g, ar);
                if (m > 1) ai = fma2(d.y, g, ai);
            }
        }
        if (m == 0) {
            phi = fr;
            gz = zr;
        } else {
            const uint64_t nei = neg2(ei);
            if (m < P) {
                phi = fma2(er, fr, fma2(nei, fi, phi));
                gz = fma2(er, zr, fma2(nei, zi, gz));
            }
            if (m == 1) {  // A_1 comes from the real M^0
                gr = mul2(er, ar);
                gi = mul2(ei, ar);
            } else {
                gr = fma2(er, ar, fma2(nei, ai, gr));
                gi = fma2(er, ai, fma2(ei, ar, gi));
                const uint64_t h = m == 2 ? ir2 : mul2(pack2((float)(m - 1), (float)(m - 1)), ir2);
                const uint64_t tr = fma2(h, fr1, mul2(q2, ar)), ti = fma2(h, fi1, mul2(q2, ai));
                if (m == 2) {
                    gr = add2(gr, tr);
                    gi = add2(gi, neg2(ti));
                } else {
                    gr = fma2(er2, tr, fma2(neg2(ei2), ti, gr));
                    gi = fma2(neg2(er2), ti, fma2(neg2(ei2), tr, gi));
                }
            }
        }
        fr1 = fr, fi1 = fi;
    }
    const uint64_t ih = pack2(g0.w, g1.w), s1 = mul2(ir, ih), s2 = mul2(s1, ih);
    o[0] = fma2(phi, s1, o[0]);
    o[1] = fma2(gr, s2, o[1]);
    o[2] = fma2(gi, s2, o[2]);
    o[3] = fma2(gz, s2, o[3]);
}

// Sources: the M2L rows of the leaf's ancestors at levels 2..L (uniform tree, UNI) or one row
// of a cell list (adaptive tree).  Writes far of every particle of the leaves.
// A CTA takes lpc leaves one after another; an empty row only stores zeros.
template <int P, bool UNI>
__global__ void __launch_bounds__(128, 5) k_m2p(int L, const float *__restrict__ geo, const int32_t *__restrict__ leaves,
                                             Span lv, int lpc, const float4 *__restrict__ geom,
                                             const int32_t *__restrict__ begin, const int32_t *__restrict__ end,
                                             const uint32_t *__restrict__ offs, const int32_t *__restrict__ ids,
                                             const float4 *__restrict__ sx, const float *__restrict__ M,
                                             float4 *__restrict__ far)
{
    using W = M2PW<P>;
    constexpr int PP = W::PP, NO = W::NO, C4 = PP / 4;
    extern __shared__ __align__(16) unsigned char m2p_sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float2 *F = reinterpret_cast<float2 *>(m2p_sm + warp * W::kWarp);
    float *sM = reinterpret_cast<float *>(m2p_sm + warp * W::kWarp + W::kF);
    float4 *sG = reinterpret_cast<float4 *>(m2p_sm + warp * W::kWarp + W::kF + W::kM);
    const int2 *tab = d_m2p_tab[P / 2 - 2];
    const int64_t w1 = min(span_count(lv), (int64_t)(blockIdx.x + 1) * lpc);
    for (int64_t w = blockIdx.x * (int64_t)lpc; w < w1; ++w) {
        const int64_t b = UNI ? level_offset(L) + w : (int64_t)leaves[w];
        const int b0 = begin[b], nt = end[b] - b0;
        if (!UNI && offs[b] == offs[b + 1]) {
            for (int t = threadIdx.x; t < nt; t += 128) far[b0 + t] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        for (int c0 = 0; c0 < nt; c0 += 32) {
            const int T = min(32, nt - c0);
            const int G = min(W::GMAX, 32 / T), S = 2 * G;
            const int t = lane % T, g = lane / T;
            const float4 p = __ldg(&sx[b0 + c0 + t]);
            uint64_t o[4] = {0, 0, 0, 0};
            auto row = [&](uint32_t e0, uint32_t e1, int l) {
                // one step's cells: lane j < S holds the id of cell j (-1: none, zero coefficients and
                // cell 0's geometry)
                auto id_at = [&](uint32_t e) { return lane < S && e + lane < e1 ? ids[e + lane] : -1; };
                auto fetch = [&](int id, int buf) {
                    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (id >= 0) {
                        const CellGeom cg = UNI ? geo_level_cell(geo, l, (uint32_t)(id - level_offset(l))) : geo_cell(geom, id);
                        q = make_float4(cg.cx, cg.cy, cg.cz, cg.inv_h);
                    }
                    const float4 q0 = make_float4(__shfl_sync(~0u, q.x, 0), __shfl_sync(~0u, q.y, 0),
                                                  __shfl_sync(~0u, q.z, 0), __shfl_sync(~0u, q.w, 0));
                    if (lane < S) sG[buf * 2 * W::GMAX + lane] = id >= 0 ? q : q0;
                    float *m = sM + buf * 2 * W::GMAX * PP;
                    for (int k0 = 0; k0 < S * C4; k0 += 32) {
                        const int k = k0 + lane, j = min(k / C4, S - 1);
                        const int idj = __shfl_sync(~0u, id, j);
                        if (k < S * C4)
                            cp_async16_t(m + 4 * k, M + (int64_t)max(idj, 0) * PP + 4 * (k - j * C4), idj >= 0 ? 16u : 0u);
                    }
                    asm volatile("cp.async.commit_group;" ::: "memory");
                };
                const uint32_t step = 4 * S;
                uint32_t e = e0 + warp * S;
                if (e >= e1) return;
                int buf = 0;
                fetch(id_at(e), 0);
                int next = id_at(e + step);
                for (; e < e1; e += step, buf ^= 1) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                    if (e + step < e1) {
                        fetch(next, buf ^ 1);
                        next = id_at(e + 2 * step);
                    }
                    const float *m = sM + buf * 2 * W::GMAX * PP;
                    for (int k = lane; k < NO; k += 32) {
                        const int2 c = __ldg(&tab[k]);
                        const float f = __int_as_float(c.y);
                        for (int pr = 0; pr < G; ++pr)
                            F[pr * NO + k] = make_float2(f * m[2 * pr * PP + c.x], f * m[(2 * pr + 1) * PP + c.x]);
                    }
                    __syncwarp();
                    if (g < G) {
                        const float4 *gg = sG + buf * 2 * W::GMAX + 2 * g;
                        m2p_pair<P>(reinterpret_cast<const ulonglong2 *>(F + g * NO), p, gg[0], gg[1], o);
                    }
                    __syncwarp();
                }
            };
            if (UNI) {
                for (int l = 2; l <= L; ++l) {
                    const int64_t a = level_offset(l) + (w >> (3 * (L - l)));
                    row(offs[a], offs[a + 1], l);
                }
            } else {
                row(offs[b], offs[b + 1], 0);
            }
            // the partial sums of the leaf's warps and groups, added in that order
            float4 v;
            float h;
            unpack2(o[0], v.x, h), v.x += h;
            unpack2(o[1], v.y, h), v.y += h;
            unpack2(o[2], v.z, h), v.z += h;
            unpack2(o[3], v.w, h), v.w += h;
            reinterpret_cast<float4 *>(F)[lane] = v;
            __syncthreads();
            if (warp == 0 && g == 0) {
                float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int ww = 0; ww < 4; ++ww) {
                    const float4 *part = reinterpret_cast<const float4 *>(m2p_sm + ww * W::kWarp);
                    for (int gg = 0; gg < G; ++gg) {
                        const float4 q = part[t + gg * T];
                        r.x += q.x;
                        r.y += q.y;
                        r.z += q.z;
                        r.w += q.w;
                    }
                }
                far[b0 + c0 + t] = r;
            }
            __syncthreads();
        }
    }
}

template <int P, bool UNI>
static void launch_m2p_t(int L, const float *geo, const int32_t *leaves, Span lv, const float4 *geom,
                         const int32_t *begin, const int32_t *end, const uint32_t *offs, const int32_t *ids,
                         const float4 *sx, const float *M, float4 *far, cudaStream_t s)
{
    constexpr int smem = 4 * M2PW<P>::kWarp;
    cudaFuncSetAttribute(k_m2p<P, UNI>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    const int lpc = lv.cap > kM2PManyLeaves ? 4 : 1;
    const unsigned grid = (unsigned)((lv.cap + lpc - 1) / lpc);
    k_m2p<P, UNI><<<grid, 128, smem, s>>>(L, geo, leaves, lv, lpc, geom, begin, end, offs, ids, sx, M, far);
    note_launches(1);
}

void launch_m2p(int P, int L, const float *geo, const float4 *sx, const int32_t *begin, const int32_t *end,
                const uint32_t *m2l_offs, const int32_t *m2l_ids, const float *M, float4 *far, cudaStream_t s)
{
    const Span lv = host_span(0, int64_t(1) << (3 * L));
    GBFMM_DISPATCH_P(P, (launch_m2p_t<PQ, true>(L, geo, nullptr, lv, nullptr, begin, end, m2l_offs, m2l_ids, sx, M,
                                                   far, s)));
}

// ==========================================================================================
// Adaptive tree: cells are given by index; each carries its level and 63-bit key prefix.
// ==========================================================================================
__global__ void k_cell_geom(Span cells, const int32_t *__restrict__ level, const uint64_t *__restrict__ key,
                            const Box *__restrict__ box, float4 *__restrict__ geom)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= span_count(cells)) return;
    const int64_t c = span_first(cells) + i;
    const CellGeom g = cell_geom63(*box, level[c], key[c]);
    geom[c] = make_float4(g.cx, g.cy, g.cz, g.inv_h);
}

void launch_cell_geom(Span cells, const int32_t *level, const uint64_t *key, const Box *box, float4 *geom,
                      cudaStream_t s)
{
    if (cells.cap <= 0) return;
    k_cell_geom<<<(unsigned)((cells.cap + 255) / 256), 256, 0, s>>>(cells, level, key, box, geom);
    note_launches(1);
}

// P2M at the listed leaves (levels >= 2), NL lanes per leaf
template <int P, int NL>
__global__ void __launch_bounds__(128) k_p2m_cells(const int32_t *__restrict__ leaves, Span lv,
                                                   const int32_t *__restrict__ level, const float4 *__restrict__ geom,
                                                   const int32_t *__restrict__ begin, const int32_t *__restrict__ count,
                                                   const float4 *__restrict__ sx, float *__restrict__ M)
{
    __shared__ float scr[4][32 * WarpSum<P>::LD];
    const int lane = threadIdx.x & 31;
    const int64_t w = (blockIdx.x * (int64_t)4 + (threadIdx.x >> 5)) * (32 / NL) + lane / NL;
    int32_t c = w < span_count(lv) ? leaves[w] : -1;
    if (c >= 0 && level[c] < 2) c = -1;
    if (__all_sync(0xffffffffu, c < 0)) return;
    float acc[P * P];
#pragma unroll
    for (int i = 0; i < P * P; ++i) acc[i] = 0.f;
    if (c >= 0) p2x_particles<P, false, NL>(acc, sx, begin[c], begin[c] + count[c], lane % NL, geo_cell(geom, c));
    lanes_store<P, NL>(acc, c >= 0 ? M + (int64_t)c * (P * P) : nullptr, lane, false, scr[threadIdx.x >> 5]);
}

// P2L over the X list (Eq. 3's L from the particles of each X leaf), NL lanes per cell; adds
// into the cell's local expansion
template <int P, int NL>
__global__ void __launch_bounds__(128) k_p2l_cells(Span cells, const int32_t *__restrict__ level,
                                                   const float4 *__restrict__ geom, const int32_t *__restrict__ begin,
                                                   const int32_t *__restrict__ count,
                                                   const uint32_t *__restrict__ x_offs,
                                                   const int32_t *__restrict__ x_ids, const float4 *__restrict__ sx,
                                                   float *__restrict__ Lc)
{
    __shared__ float scr[4][32 * WarpSum<P>::LD];
    const int lane = threadIdx.x & 31;
    const int64_t w = (blockIdx.x * (int64_t)4 + (threadIdx.x >> 5)) * (32 / NL) + lane / NL;
    const int64_t b = span_first(cells) + w;
    uint32_t e0 = 0, e1 = 0;
    if (w < span_count(cells) && level[b] >= 2) e0 = x_offs[b], e1 = x_offs[b + 1];
    if (__all_sync(0xffffffffu, e0 == e1)) return;
    float acc[P * P];
#pragma unroll
    for (int i = 0; i < P * P; ++i) acc[i] = 0.f;
    if (e0 < e1) {
        const CellGeom cg = geo_cell(geom, b);
        for (uint32_t e = e0; e < e1; ++e) {
            const int32_t c = x_ids[e];
            p2x_particles<P, true, NL>(acc, sx, begin[c], begin[c] + count[c], lane % NL, cg);
        }
    }
    lanes_store<P, NL>(acc, e0 < e1 ? Lc + b * (P * P) : nullptr, lane, true, scr[threadIdx.x >> 5]);
}

// L2P at every particle's leaf (leaves above level 2 carry no local expansion)
template <int P>
__global__ void __launch_bounds__(128) k_l2p_cells(int64_t n, const int32_t *__restrict__ leaf_of,
                                                   const int32_t *__restrict__ leaves,
                                                   const int32_t *__restrict__ level, const float4 *__restrict__ geom,
                                                   const float4 *__restrict__ sx, const float *__restrict__ Lc,
                                                   float4 *__restrict__ far, const float4 *__restrict__ near,
                                                   const uint32_t *__restrict__ perm, float4 *__restrict__ out,
                                                   const int32_t *__restrict__ abort)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n || (abort && *abort)) return;
    const int32_t lo = leaf_of[i], c = leaves ? leaves[lo] : lo;
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (level[c] >= 2) {
        const CellGeom cg = geo_cell(geom, c);
        float4 p = __ldg(&sx[i]);
        f = l2p_eval<P>(Lc + (int64_t)c * (P * P), (p.x - cg.cx) * cg.inv_h, (p.y - cg.cy) * cg.inv_h,
                        (p.z - cg.cz) * cg.inv_h, cg.inv_h);
    }
    if (near) {  // far holds the M2P (W list) sums
        const float4 w = far[i];
        f.x += w.x;
        f.y += w.y;
        f.z += w.z;
        f.w += w.w;
        out[perm[i]] = near_plus_far(near, i, f);
    } else {
        far[i] = f;
    }
}

// M2M (up) / L2L (down) over cells given by their parents' index range; children by position.
// As k_translate: the operator of each child position and the TN source columns are copied into
// shared memory with cp.async (zero-filled for missing children), the next child position's
// copies in flight while the current one is applied.
// LOOP: the CTAs take TN parents after TN (a captured level, whose count only the device knows: a
// launch over its whole capacity, most of it idle, cost a batch of 96 instances 3%).
template <int P, bool UP, int TN, int CN, bool LOOP>
__global__ void __launch_bounds__(TransCfg<P, UP, TN, CN>::NT) k_translate_cells(Span par,
                                                                         const int32_t *__restrict__ child_of,
                                                                         const int32_t *__restrict__ nchild,
                                                                         const float *__restrict__ ops,
                                                                         float *__restrict__ X)
{
    using Cfg = TransCfg<P, UP, TN, CN>;
    constexpr int PP = Cfg::PP, PR = Cfg::PR, SB = Cfg::SB, NCG = Cfg::NCG, NRG = Cfg::NRG;
    extern __shared__ __align__(16) float tsm[];
    int64_t q0 = blockIdx.x * (int64_t)TN;
    const int64_t lo = span_first(par), np = span_count(par);
    if (q0 >= np) return;  // the whole CTA: beyond the parents
    const int tid = threadIdx.x;
    const bool work = tid < NRG * NCG;
    const int cg = tid % NCG, rg = tid / NCG;
    int kbeg = 0, kend = PP;
    if (work) {
        const int r0 = min(rg * 4, PP - 1), r1 = min(rg * 4 + 3, PP - 1);
        if (UP) {
            const int d = degree_of(r1);
            kend = min(PP, ((d + 1) * (d + 1) + 3) / 4 * 4);
        } else {
            const int d = degree_of(r0);
            kbeg = (d * d) / 4 * 4;
        }
    }
    auto stage = [&](int c, int buf) {
        float *A = tsm + buf * (Cfg::AF + Cfg::BF);
        float *B = A + Cfg::AF;
        const float *src = ops + (size_t)c * PP * PR;
        for (int e = tid; e < PP * PR / 4; e += blockDim.x) cp_async16_t(A + 4 * e, src + 4 * e, 16u);
        for (int e = tid; e < TN * (PP / 4); e += blockDim.x) {
            const int i = e / (PP / 4), k4 = e % (PP / 4);
            const int64_t q = q0 + i;
            const float *gsrc = X;
            uint32_t bytes = 0;
            if (q < np) {
                const int64_t pcell = lo + q;
                const int64_t g = UP ? child_of[pcell * 8 + c] : (child_of[pcell * 8 + c] >= 0 ? pcell : -1);
                if (g >= 0) {
                    gsrc = X + g * PP + 4 * k4;
                    bytes = 16u;
                }
            }
            cp_async16_t(B + i * SB + 4 * k4, gsrc, bytes);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    do {
        float tot[4][CN];  // M2M: the child positions' sums, added in order (as k_m2m_small adds them)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CN; ++j) tot[i][j] = 0.f;
        const int c_first = UP ? 0 : blockIdx.y, c_last = UP ? 7 : blockIdx.y;
        stage(c_first, 0);
        for (int c = c_first; c <= c_last; ++c) {
            const int buf = UP ? (c - c_first) & 1 : 0;
            if (c < c_last) {
                stage(c + 1, buf ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            if (work) {
                const float *Ar = tsm + buf * (Cfg::AF + Cfg::BF) + rg * 4;
                const float *Bc = tsm + buf * (Cfg::AF + Cfg::BF) + Cfg::AF + cg * SB;
                float acc[4][CN];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < CN; ++j) acc[i][j] = 0.f;
#pragma unroll 2
                for (int k = kbeg; k < kend; k += 4) {
                    Frag<CN, 4> f;
                    f.load(Ar, Bc, k, PR, NCG * SB);
                    f.fma(acc);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < CN; ++j) tot[i][j] += acc[i][j];
            }
            __syncthreads();  // the buffer is refilled two positions later
        }
        if (work) {
#pragma unroll
            for (int j = 0; j < CN; ++j) {
                const int64_t q = q0 + cg + j * NCG;
                if (q >= np) continue;
                const int r = rg * 4;
                if (r >= PP) continue;
                const int64_t pcell = lo + q;
                int64_t g;
                if (UP) {
                    if (nchild[pcell] == 0) continue;  // a leaf keeps its P2M expansion
                    g = pcell;
                } else {
                    g = child_of[pcell * 8 + blockIdx.y];
                    if (g < 0) continue;
                }
                float4 *dst = reinterpret_cast<float4 *>(X + g * PP + r);
                if (UP) {
                    *dst = make_float4(tot[0][j], tot[1][j], tot[2][j], tot[3][j]);
                } else {
                    float4 v = *dst;
                    v.x += tot[0][j];
                    v.y += tot[1][j];
                    v.z += tot[2][j];
                    v.w += tot[3][j];
                    *dst = v;
                }
            }
        }
        q0 += (int64_t)gridDim.x * TN;
    } while (LOOP && q0 < np);
}

void launch_p2m_cells(int P, int64_t est_leaves, const int32_t *leaves, Span lv, const int32_t *level,
                      const float4 *geom, const int32_t *begin, const int32_t *count, const float4 *sx, float *M,
                      cudaStream_t s)
{
    if (lv.cap <= 0) return;
    if (est_leaves >= kP2MManyLeaves) {
        const unsigned grid = (unsigned)((lv.cap + 15) / 16);
        GBFMM_DISPATCH_P(P, (p2m_carveout(k_p2m_cells<PQ, 8>),
                             k_p2m_cells<PQ, 8><<<grid, 128, 0, s>>>(leaves, lv, level, geom, begin, count, sx, M)));
    } else {
        const unsigned grid = (unsigned)((lv.cap + 3) / 4);
        GBFMM_DISPATCH_P(P, (p2m_carveout(k_p2m_cells<PQ, 32>),
                             k_p2m_cells<PQ, 32><<<grid, 128, 0, s>>>(leaves, lv, level, geom, begin, count, sx, M)));
    }
    note_launches(1);
}

void launch_p2l_cells(int P, int64_t est_leaves, Span cells, const int32_t *level, const float4 *geom, const int32_t *begin,
                      const int32_t *count, const uint32_t *x_offs, const int32_t *x_ids, const float4 *sx, float *Lc,
                      cudaStream_t s)
{
    if (cells.cap <= 0) return;
    // an X leaf of 30 to 60 particles wastes fewer lanes in rounds of 16 (16M Plummer step 23.35 ->
    // 23.15 ms, 400,009 1696 -> 1686 us); few cells want them in few rounds (20,011: 386 against 389)
    if (est_leaves >= kP2MManyLeaves) {
        const unsigned grid = (unsigned)((cells.cap + 7) / 8);
        GBFMM_DISPATCH_P(P, (k_p2l_cells<PQ, 16><<<grid, 128, 0, s>>>(cells, level, geom, begin, count, x_offs, x_ids,
                                                                      sx, Lc)));
    } else {
        const unsigned grid = (unsigned)((cells.cap + 3) / 4);
        GBFMM_DISPATCH_P(P, (k_p2l_cells<PQ, 32><<<grid, 128, 0, s>>>(cells, level, geom, begin, count, x_offs, x_ids,
                                                                      sx, Lc)));
    }
    note_launches(1);
}

void launch_l2p_cells(int P, int64_t n, const int32_t *leaf_of, const int32_t *leaves, const int32_t *level, const float4 *geom,
                      const float4 *sx, const float *Lc, float4 *far, cudaStream_t s, const float4 *near,
                      const uint32_t *perm, float4 *out, const int32_t *abort)
{
    if (n <= 0) return;
    const unsigned grid = (unsigned)((n + 127) / 128);
    GBFMM_DISPATCH_P(P, (k_l2p_cells<PQ><<<grid, 128, 0, s>>>(n, leaf_of, leaves, level, geom, sx, Lc, far, near, perm, out,
                                                              abort)));
    note_launches(1);
}

void launch_m2p_cells(int P, const int32_t *leaves, Span lv, const float4 *geom, const int32_t *begin,
                      const int32_t *end, const uint32_t *w_offs, const int32_t *w_ids, const float4 *sx,
                      const float *M, float4 *far, cudaStream_t s)
{
    if (lv.cap <= 0) return;
    GBFMM_DISPATCH_P(P, (launch_m2p_t<PQ, false>(0, nullptr, leaves, lv, geom, begin, end, w_offs, w_ids, sx, M, far,
                                                 s)));
}

template <int P, bool UP, int TN, int CN, bool LOOP = false>
static void translate_cells_tn(Span par, const int32_t *child_of, const int32_t *nchild, const float *ops, float *X,
                               cudaStream_t s)
{
    using Cfg = TransCfg<P, UP, TN, CN>;
    const int smem = (int)Cfg::kSmem;  // operator + column block, double-buffered for M2M
    cudaFuncSetAttribute(k_translate_cells<P, UP, TN, CN, LOOP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    const int64_t items = LOOP ? std::max<int64_t>(1, par.likely()) : par.cap;
    dim3 grid((unsigned)((items + TN - 1) / TN), UP ? 1 : 8);
    k_translate_cells<P, UP, TN, CN, LOOP><<<grid, Cfg::NT, smem, s>>>(par, child_of, nchild, ops, X);
    note_launches(1);
}

// the cells-per-CTA choice of the uniform tree's translations (launch_translate_t), on the
// expected count
template <int P, bool UP>
static void translate_cells_t(Span par, const int32_t *child_of, const int32_t *nchild, const float *ops, float *X,
                              cudaStream_t s)
{
    if constexpr (UP)
        if (launch_m2m_small<P>(std::max<int64_t>(par.likely(), 1), SpanCells{par, child_of, nchild}, ops, X, s)) return;
    if (par.expect >= 0) return translate_cells_tn<P, UP, 16, 2, true>(par, child_of, nchild, ops, X, s);
    const int64_t np = par.cap, ctas32 = (np + 31) / 32 * (UP ? 1 : 8), ctas64 = (np + 63) / 64 * (UP ? 1 : 8);
    if constexpr (UP) {  // large levels: 128 (upward) or 64 cells per CTA share each staged operator
        if ((np + 127) / 128 >= 4 * kSms) return translate_cells_tn<P, UP, 128, 8>(par, child_of, nchild, ops, X, s);
    }
    if (ctas64 >= 4 * kSms)
        translate_cells_tn<P, UP, 64, 8>(par, child_of, nchild, ops, X, s);
    else if (ctas32 >= 2 * kSms)
        translate_cells_tn<P, UP, 32, 8>(par, child_of, nchild, ops, X, s);
    else
        translate_cells_tn<P, UP, 16, 2>(par, child_of, nchild, ops, X, s);
}

// ---- several small levels in one launch ---------------------------------------------------------
// A tree of 20,000 particles has six levels of 50 to 500 parents, each a launch of 5 us up and 5 us
// down for a microsecond of work.  One cluster of 8 CTAs takes a run of such levels: a CTA keeps its
// row slice of the eight operators in shared memory throughout, takes every (8 / SL)-th eight
// parents of a level, and a cluster barrier parts the levels.  Each sum is formed as in
// k_m2m_small and k_translate_cells.  20,011 Plummer particles, p = 4: the four top levels 19 -> 15.5 us
// up and 21 -> 16.5 down, the step 346 -> 332; a captured batch of 96 instances, whose launches cover
// three levels more than there are, 6.62 -> 6.28 ms.
constexpr int kChainCtas = 8;
struct ChainLevels {
    Span s[kGeoLevels];
    int n;
};

template <int P, bool UP>
__global__ void __cluster_dims__(kChainCtas, 1, 1) __launch_bounds__(TransSmall<P>::NT)
    k_translate_chain(const __grid_constant__ ChainLevels lv, const int32_t *__restrict__ child_of,
                      const int32_t *__restrict__ nchild, const float *__restrict__ ops, float *X)
{
    using Cfg = TransSmall<P>;
    constexpr int PP = Cfg::PP, PR = Cfg::PR, SB = Cfg::SB, TN = Cfg::TN, GT = Cfg::GT, LDA = Cfg::LDA;
    constexpr int RGS = Cfg::RGS, NRG = Cfg::NRG, SL = Cfg::SL, PER = kChainCtas / SL;
    static_assert(Cfg::CN == 1 && Cfg::NCG == TN, "a thread holds one parent's four rows");
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) float tsm[];
    __shared__ int64_t s_par[TN], s_child[8][TN];
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int rg0 = (rank % SL) * RGS, rg1 = min(rg0 + RGS, NRG);
    auto k_end = [](int r) { const int d = degree_of(min(r, PP - 1)); return min(PP, ((d + 1) * (d + 1) + 3) / 4 * 4); };
    auto k_beg = [](int r) { const int d = degree_of(min(r, PP - 1)); return (d * d) / 4 * 4; };
    const int ks = UP ? 0 : k_beg(4 * rg0), ke = UP ? k_end(4 * rg1 - 1) : PP;  // the columns the slice reads
    float *B = tsm + 8 * PP * LDA, *red = B + 8 * TN * SB;
    const bool active = rank < SL * PER;
    if (active) {
        for (int e = tid; e < 8 * PP * RGS; e += Cfg::NT) {
            const int r = e % RGS, k = (e / RGS) % PP, c = e / (RGS * PP);
            if (k >= ks && k < ke && rg0 + r < rg1)
                cp_async16_t(tsm + (c * PP + k) * LDA + 4 * r, ops + ((size_t)c * PP + k) * PR + 4 * (rg0 + r), 16u);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const int c = tid / GT, t = tid % GT, col = t % TN, rl = t / TN, rg = rg0 + rl;
    const int kb = UP ? 0 : k_beg(4 * rg), kn = UP ? k_end(4 * rg + 3) : PP;
    for (int li = 0; li < lv.n; ++li) {
        const int64_t np = span_count(lv.s[li]), lo = span_first(lv.s[li]);
        for (int64_t q0 = (int64_t)(rank / SL) * TN; active && q0 < np; q0 += (int64_t)PER * TN) {
            for (int e = tid; e < 9 * TN; e += Cfg::NT) {
                const int i = e % TN, ch = e / TN - 1;
                int64_t g = -1;
                if (q0 + i < np) g = ch >= 0 ? child_of[(lo + q0 + i) * 8 + ch] : nchild[lo + q0 + i] != 0 ? lo + q0 + i : -1;
                (ch < 0 ? s_par[i] : s_child[ch][i]) = g;
            }
            __syncthreads();
            for (int e = tid; e < (UP ? 8 : 1) * TN * (PP / 4); e += Cfg::NT) {
                const int k = 4 * (e % (PP / 4)), i = (e / (PP / 4)) % TN, ch = e / (PP / 4 * TN);
                const int64_t g = UP ? s_child[ch][i] : s_par[i];
                if (k >= ks && k < ke) cp_async16_t(B + (ch * TN + i) * SB + k, g >= 0 ? X + g * PP + k : X, g >= 0 ? 16u : 0u);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            float acc[4][1] = {{0.f}, {0.f}, {0.f}, {0.f}};
            if (rg < rg1) {
                const float *Ar = tsm + c * PP * LDA + 4 * rl, *Bc = B + ((UP ? c * TN : 0) + col) * SB;
#pragma unroll 2
                for (int k = kb; k < kn; k += 4) {
                    Frag<1, 4> f;
                    f.load(Ar, Bc, k, LDA, 0);
                    f.fma(acc);
                }
            }
            if (UP) {
#pragma unroll
                for (int i = 0; i < 4; ++i) red[i * Cfg::NT + tid] = acc[i][0];
                __syncthreads();
                for (int e = tid; e < 4 * GT; e += Cfg::NT) {
                    const int i = e % 4, tt = e / 4, r = 4 * (rg0 + tt / TN) + i;
                    const int64_t g = s_par[tt % TN];
                    if (g < 0 || rg0 + tt / TN >= rg1 || r >= PP) continue;
                    float v = 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) v += red[i * Cfg::NT + k * GT + tt];
                    X[g * PP + r] = v;
                }
            } else if (rg < rg1 && 4 * rg < PP && s_child[c][col] >= 0) {
                float4 *dst = reinterpret_cast<float4 *>(X + s_child[c][col] * PP + 4 * rg);
                float4 v = *dst;
                v.x += acc[0][0];
                v.y += acc[1][0];
                v.z += acc[2][0];
                v.w += acc[3][0];
                *dst = v;
            }
            __syncthreads();  // the columns and the sums are read: the next parents may be staged
        }
        __threadfence();
        cl.sync();  // the level is written before the next one's columns are read (cp.async.cg: from L2)
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // a CTA that had no parents: its operators
}

// levels of up to this many parents may share a launch: four rounds of eight parents a CTA
template <int P>
static constexpr int64_t chain_parents()
{
    return 4 * TransSmall<P>::TN * (kChainCtas / TransSmall<P>::SL);
}

template <int P, bool UP>
static void translate_levels_t(const Span *par, int n, const int32_t *child_of, const int32_t *nchild,
                               const float *ops, float *X, cudaStream_t s)
{
    for (int i = 0; i < n;) {
        ChainLevels lv;
        lv.n = 0;
        while (i + lv.n < n && par[i + lv.n].likely() <= chain_parents<P>()) {
            lv.s[lv.n] = par[i + lv.n];
            ++lv.n;
        }
        if (lv.n >= 2) {
            constexpr int smem = (int)TransSmall<P>::kSmem;
            cudaFuncSetAttribute(k_translate_chain<P, UP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            k_translate_chain<P, UP><<<kChainCtas, TransSmall<P>::NT, smem, s>>>(lv, child_of, nchild, ops, X);
            note_launches(1);
            i += lv.n;
        } else {
            if (par[i].cap > 0) translate_cells_t<P, UP>(par[i], child_of, nchild, ops, X, s);
            ++i;
        }
    }
}

void launch_translate_levels(int P, bool up, const Span *parents, int n, const int32_t *child_of,
                             const int32_t *nchild, const float *ops, float *X, cudaStream_t s)
{
    if (up) {
        GBFMM_DISPATCH_P(P, (translate_levels_t<PQ, true>(parents, n, child_of, nchild, ops, X, s)));
    } else {
        GBFMM_DISPATCH_P(P, (translate_levels_t<PQ, false>(parents, n, child_of, nchild, ops, X, s)));
    }
}
#undef GBFMM_DISPATCH_P

}  // namespace gbfmm
