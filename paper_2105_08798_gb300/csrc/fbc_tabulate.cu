// Kernel-table generation (setup, FP64).
//
// Stage 1 (periodic kernel): for every in-plane difference d that occurs and
// every repeat offset s in [0, L/2], the regularised image sum of Sec. 3.1
// (Eqs. 32, 35) extrapolated with Richardson's formula (Eq. 36):
//     G~(d, s) = G_n + sum_{m=n+1}^{n+N} W_m t_m,
//     G_n = G(d, s c) + sum_{m=1}^{n} t_m,
//     t_m = G(d, s c + m l3) + G(d, s c - m l3) - G(0, 0, m l3) - G(0, 0, -m l3),
// with W_m the cumulative weights computed on the host (algebraically the same
// as Eq. 36, arranged so that the large alternating weights only multiply the
// small increments t_m).  At s = L/2 the two centred representatives
// +-L/2 are averaged, which for a mirror-symmetric medium keeps the even
// entries and zeroes the odd ones.
//
// Stage 2 (line DFT): g^k(d) = sum_s G~(d, s) exp(-2 pi i k s / L) for
// k = 0..L/2.  With the mirror symmetry G~(d, L - s) = M G~(d, s) M,
// M = diag(1, 1, -1), the even entries give a cosine sum (real part) and the
// odd entries a sine sum (imaginary part):
//     A(k) = G(0) + (-1)^k G(L/2) + 2 sum_{s=1}^{L/2-1} G(s) cos(2 pi k s / L),
//     B(k) = -2 sum_{s=1}^{L/2-1} G(s) sin(2 pi k s / L).
//
// The continuum Green function (Eq. 33) is Kelvin's closed form for an
// isotropic medium and Barnett's integral over the unit circle normal to r,
//     G(r) = 1/(8 pi^2 |r|) int_0^{2 pi} (zz)^{-1} dpsi,
// for a cubic one, evaluated by the trapezoid rule on [0, pi) (the integrand
// has period pi) with the nodes' cosines and sines among the kernel's parameters.
//
// The reference terms G(0, 0, +-m l3) depend on m alone and are computed once; of each pair d, -d only one is
// evaluated.  Together four times fewer Green functions than one thread per (d, s) evaluating all of
// them: an isotropic slab of 4000 x 6000 columns, L = 256, 23.5 ms before, 8.9 ms now.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fbc_internal.cuh"

namespace fbc {
namespace {

// Which Green function a launch evaluates.  The polynomial form serves the plans of the FP64-accurate precisions whose
// medium and node count cubic_poly_form lets through.
// The others round the table to 32 bits or fewer, where a last-bit change of a few FP64 entries moves the
// rounding of some (1e-9 to 4e-9 of an update, more than those forms differ by from run to run): they and the
// H-matrix's FP32 table keep the node-by-node form's bits.
enum { kGreenIso = 0, kGreenNodes = 1, kGreenPoly = 2 };

// A launch's medium and quadrature nodes: kernel parameters, so that plans tabulated on different streams at the same
// time keep their own.
struct Medium {
    MaterialDev m;
    double pre;  // polynomial form: (scale of the constants) / (pi nquad)
};
// cos and sin of psi at the nodes (node by node), or of 2 psi, 4 psi and 6 psi
template <int KIND>
struct QuadNodes {
    double v[KIND == kGreenIso ? 1 : kMaxQuad][KIND == kGreenPoly ? 6 : 2];
};
static_assert(sizeof(Medium) + sizeof(QuadNodes<kGreenPoly>) + sizeof(TabulateParams) + 64 <= 32764, "kernel parameters");

// G as six entries (11, 12, 22, 33, 13, 23) of the symmetric tensor: Kelvin's closed form.
__device__ __forceinline__ void green_isotropic(const MaterialDev& mat, double rx, double ry, double rz, double g[6]) {
    const double R2 = rx * rx + ry * ry + rz * rz;
    const double R = sqrt(R2);
    const double pre = mat.kelvin_pre / R;
    const double iR2 = 1.0 / R2;
    const double a = mat.kelvin_a;
    g[0] = pre * (a + rx * rx * iR2);
    g[1] = pre * (rx * ry * iR2);
    g[2] = pre * (a + ry * ry * iR2);
    g[3] = pre * (a + rz * rz * iR2);
    g[4] = pre * (rx * rz * iR2);
    g[5] = pre * (ry * rz * iR2);
}

// Barnett's integral for a cubic medium node by node: the Christoffel matrix M of z = cos(psi) e1 + sin(psi) e2,
// its cofactors and a division at every node, about 88 FP64 operations each.
__device__ __forceinline__ void green_nodes(const MaterialDev& mat, const QuadNodes<kGreenNodes>& N, double rx, double ry,
                                            double rz, double g[6]) {
    const double R2 = rx * rx + ry * ry + rz * rz;
    const double R = sqrt(R2);
    // unit direction and an orthonormal pair spanning the plane normal to it
    const double iR = 1.0 / R;
    const double hx = rx * iR, hy = ry * iR, hz = rz * iR;
    double e1x, e1y, e1z;
    const double rho2 = hx * hx + hy * hy;
    if (rho2 > 1e-24) {
        const double ir = rsqrt(rho2);
        e1x = -hy * ir, e1y = hx * ir, e1z = 0.0;
    } else {
        e1x = 1.0, e1y = 0.0, e1z = 0.0;
    }
    const double e2x = hy * e1z - hz * e1y;
    const double e2y = hz * e1x - hx * e1z;
    const double e2z = hx * e1y - hy * e1x;
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0, s5 = 0;  // 11 22 33 23 13 12
    const int nq = mat.nquad;
    for (int q = 0; q < nq; q++) {
        const double cq = N.v[q][0], sq = N.v[q][1];
        const double zx = cq * e1x + sq * e2x;
        const double zy = cq * e1y + sq * e2y;
        const double zz = cq * e1z + sq * e2z;
        const double p[6] = {zx * zx, zy * zy, zz * zz, zy * zz, zx * zz, zx * zy};
        double m[6];
#pragma unroll
        for (int I = 0; I < 6; I++) {
            double v = 0.0;
#pragma unroll
            for (int J = 0; J < 6; J++) v = fma(mat.K[6 * I + J], p[J], v);
            m[I] = v;
        }
        // symmetric 3x3 inverse by the adjugate; m = (a, b, c, d, e, f) = (00, 11, 22, 12, 02, 01)
        const double a = m[0], b = m[1], c = m[2], d = m[3], e = m[4], f = m[5];
        const double A00 = b * c - d * d, A11 = a * c - e * e, A22 = a * b - f * f;
        const double A12 = e * f - a * d, A02 = d * f - b * e, A01 = d * e - c * f;
        const double idet = 1.0 / (a * A00 + f * A01 + e * A02);
        s0 = fma(A00, idet, s0);
        s1 = fma(A11, idet, s1);
        s2 = fma(A22, idet, s2);
        s3 = fma(A12, idet, s3);
        s4 = fma(A02, idet, s4);
        s5 = fma(A01, idet, s5);
    }
    // 2 * (pi / nq) / (8 pi^2 R) = 1 / (4 pi nq R)
    const double pre = 1.0 / (4.0 * M_PI * (double)nq * R);
    g[0] = pre * s0;
    g[1] = pre * s5;
    g[2] = pre * s1;
    g[3] = pre * s2;
    g[4] = pre * s4;
    g[5] = pre * s3;
}

// What the polynomial form below keeps for all points r = (d, z) of one in-plane difference d: rho = |d|, the in-plane unit vector e1 normal to r, and e1's part of the Christoffel matrix.
struct CubicDir {
    double rho2, rho, e1x, e1y, p[6], k11[6];
};

__device__ __forceinline__ void christoffel(const MaterialDev& mat, const double (&p)[6], double (&m)[6]) {
#pragma unroll
    for (int I = 0; I < 6; I++) {
        double v = 0.0;
#pragma unroll
        for (int J = 0; J < 6; J++) v = fma(mat.K[6 * I + J], p[J], v);
        m[I] = v;
    }
}

__device__ __forceinline__ CubicDir cubic_dir(const MaterialDev& mat, double rx, double ry) {
    CubicDir D;
    const bool line = rx == 0.0 && ry == 0.0;  // r along the line: any in-plane direction
    D.rho2 = fma(rx, rx, ry * ry);
    D.rho = sqrt(D.rho2);
    const double i = line ? 0.0 : 1.0 / D.rho2;
    D.e1x = line ? 1.0 : -ry / D.rho;
    D.e1y = line ? 0.0 : rx / D.rho;
    D.p[0] = line ? 1.0 : ry * ry * i;
    D.p[1] = rx * rx * i;
    D.p[2] = D.p[3] = D.p[4] = 0.0;
    D.p[5] = -(rx * ry) * i;
    christoffel(mat, D.p, D.k11);
    return D;
}

// The same sum with the work per node reduced; FP64 issue bounds the tabulation (this part's FP64 pipe runs at
// 1/64 of the FP32 rate).  2 M = u + v cos 2psi + w sin 2psi exactly, so its cofactors are trigonometric polynomials
// of degree 2 in 2 psi (five coefficients each, once per point) and its determinant one of degree 3 (seven), and
//     sum_q cof_ij(psi_q) / det(psi_q) = sum_t coef_ij,t  sum_q basis_t(psi_q) / det(psi_q):
// five sums serve all six entries.  With an even number of nodes psi and psi + pi/2 are both nodes; the even
// part E and odd part O of the determinant serve both, 1/(E+O) +- 1/(E-O) = (2 E, -2 O) / ((E+O)(E-O)), and
// one division serves two such pairs.  About 11 FP64 operations a node and 400 a point.  The coefficients' rounding is
// the same at every node and does not average out, so the directions enter as quotients of exact squares, the
// products are fused and the sums are taken in groups of eight pairs.  That rounding is relative to the largest
// products of the entries of M, not to the determinant at a node: the form serves the media cubic_poly_form lets through.
// The 1000 x 1500, L = 64 cubic slab's table: 112.3 ms with its first update before, 6.9 ms now;
// 4000 x 6000, L = 256: 1676 ms before, 97 ms now (433 ms with the node-by-node form).
__device__ __forceinline__ void green_cubic(const Medium& M, const QuadNodes<kGreenPoly>& N, const CubicDir& D, double rx,
                                            double ry, double rz, double g[6]) {
    const MaterialDev& mat = M.m;
    const double R2 = fma(rz, rz, D.rho2), R = sqrt(R2), iR = 1.0 / R, i2 = 1.0 / R2;
    const double hz = rz * iR, hr = D.rho * iR, zz = rz * rz * i2;
    double u[6], v[6], w[6];  // 2 M = u + v cos 2psi + w sin 2psi, entries (00, 11, 22, 12, 02, 01)
    {
        // e2 = (-hz e1y, hz e1x, hr)
        const double p22[6] = {zz * D.p[1], zz * D.p[0], D.rho2 * i2, -(rz * ry) * i2, -(rz * rx) * i2, -zz * D.p[5]};
        double k22[6];
        christoffel(mat, p22, k22);
        const double x = 2.0 * hz * D.p[5];
        const double p12[6] = {-x, x, 0.0, D.e1y * hr, D.e1x * hr, hz * (D.p[0] - D.p[1])};
        christoffel(mat, p12, w);
#pragma unroll
        for (int t = 0; t < 6; t++) u[t] = D.k11[t] + k22[t], v[t] = D.k11[t] - k22[t];
    }
    // cofactors times 2 in the basis (1, cos 2psi, sin 2psi, cos 4psi, sin 4psi)
    double A[6][5];  // 00, 11, 22, 12, 02, 01
    auto cof = [&](double (&q)[5], int i, int j, int k, int l) {  // m_i m_j - m_k m_l
        const double vv = fma(v[i], v[j], -(v[k] * v[l])), ww = fma(w[i], w[j], -(w[k] * w[l]));
        q[0] = fma(2.0, fma(u[i], u[j], -(u[k] * u[l])), vv + ww);
        q[1] = 2.0 * (fma(u[i], v[j], v[i] * u[j]) - fma(u[k], v[l], v[k] * u[l]));
        q[2] = 2.0 * (fma(u[i], w[j], w[i] * u[j]) - fma(u[k], w[l], w[k] * u[l]));
        q[3] = vv - ww;
        q[4] = fma(v[i], w[j], w[i] * v[j]) - fma(v[k], w[l], w[k] * v[l]);
    };
    cof(A[0], 1, 2, 3, 3);
    cof(A[1], 0, 2, 4, 4);
    cof(A[2], 0, 1, 5, 5);
    cof(A[3], 4, 5, 0, 3);
    cof(A[4], 3, 5, 1, 4);
    cof(A[5], 3, 4, 2, 5);
    // four times the determinant in the basis (1, cos, sin of 2psi, of 4psi, of 6psi)
    double d0 = 0, d1 = 0, d2 = 0, d3 = 0, d4 = 0, d5 = 0, d6 = 0;
    auto det = [&](int i, const double (&q)[5]) {
        const double ui = 2.0 * u[i], vi = v[i], wi = w[i];
        d0 = fma(ui, q[0], fma(vi, q[1], fma(wi, q[2], d0)));
        d1 = fma(ui, q[1], fma(2.0 * vi, q[0], fma(vi, q[3], fma(wi, q[4], d1))));
        d2 = fma(ui, q[2], fma(2.0 * wi, q[0], fma(vi, q[4], fma(-wi, q[3], d2))));
        d3 = fma(ui, q[3], fma(vi, q[1], fma(-wi, q[2], d3)));
        d4 = fma(ui, q[4], fma(vi, q[2], fma(wi, q[1], d4)));
        d5 = fma(vi, q[3], fma(-wi, q[4], d5));
        d6 = fma(vi, q[4], fma(wi, q[3], d6));
    };
    det(4, A[4]);
    det(5, A[5]);
    det(0, A[0]);
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0, t0 = 0, t1 = 0, t2 = 0, t3 = 0, t4 = 0;
    auto parts = [&](int q, double& E, double& O) {
        const double* n = N.v[q];
        E = fma(n[3], d4, fma(n[2], d3, d0));
        O = fma(n[5], d6, fma(n[4], d5, fma(n[1], d2, n[0] * d1)));
    };
    auto add = [&](int q, double e, double o) {  // e, o: the even and odd parts of the node's 1 / det
        const double* n = N.v[q];
        t0 += e;
        t1 = fma(n[0], o, t1);
        t2 = fma(n[1], o, t2);
        t3 = fma(n[2], e, t3);
        t4 = fma(n[3], e, t4);
    };
    auto join = [&]() {
        s0 += t0, s1 += t1, s2 += t2, s3 += t3, s4 += t4;
        t0 = t1 = t2 = t3 = t4 = 0.0;
    };
    const int nq = mat.nquad;
    double scale;
    if (nq % 4 == 0) {
        for (int q = 0; q < nq / 2; q += 2) {
            double E, O, F, Q;
            parts(q, E, O);
            parts(q + 1, F, Q);
            const double p = (E + O) * (E - O), r = (F + Q) * (F - Q);
            const double i = 1.0 / (p * r);
            const double ip = i * r, ir = i * p;
            add(q, E * ip, -O * ip);
            add(q + 1, F * ir, -Q * ir);
            if (q % 8 == 6) join();
        }
        scale = 2.0;
    } else {
        for (int q = 0; q < nq; q++) {
            double E, O;
            parts(q, E, O);
            const double i = 1.0 / (E + O);
            add(q, i, i);
            if (q % 8 == 7) join();
        }
        scale = 1.0;
    }
    join();
    const double pre = scale * M.pre * iR;
    auto entry = [&](const double (&q)[5]) {
        return pre * fma(q[0], s0, fma(q[1], s1, fma(q[2], s2, fma(q[3], s3, q[4] * s4))));
    };
    g[0] = entry(A[0]);
    g[1] = entry(A[5]);
    g[2] = entry(A[1]);
    g[3] = entry(A[2]);
    g[4] = entry(A[4]);
    g[5] = entry(A[3]);
}

// G(0, 0, m l3) + G(0, 0, -m l3) for the images m = 1 .. n + N (one block each, a thread per sign): the same for every
// difference and offset.
template <int KIND>
__global__ void k_reference(const __grid_constant__ Medium M, const __grid_constant__ QuadNodes<KIND> Q,
                            const __grid_constant__ TabulateParams T, double* __restrict__ ref) {
    const int m = blockIdx.x + 1;
    __shared__ double h[6];
    const double zm = (threadIdx.x ? -1.0 : 1.0) * ((double)m * ((double)T.L * T.c));
    double g[6];
    if constexpr (KIND == kGreenIso) {
        green_isotropic(M.m, 0.0, 0.0, zm, g);
    } else if constexpr (KIND == kGreenNodes) {
        green_nodes(M.m, Q, 0.0, 0.0, zm, g);
    } else {
        const CubicDir D = cubic_dir(M.m, 0.0, 0.0);
        green_cubic(M, Q, D, 0.0, 0.0, zm, g);
    }
    if (threadIdx.x == 1)
        for (int t = 0; t < 6; t++) h[t] = g[t];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int t = 0; t < 6; t++) ref[(m - 1) * 6 + t] = g[t] + h[t];
}

// Stage 1: one thread per (listed difference, s in [0, L/2]).  Of a pair of used differences d and -d only one
// is listed: G(-d, s) is G(d, s) with the odd entries (13, 23) negated, bit for bit, so stage 2 writes both.
template <int KIND>
__global__ void __launch_bounds__(128) k_periodic(const __grid_constant__ Medium M, const __grid_constant__ QuadNodes<KIND> Q,
                                                  const __grid_constant__ TabulateParams T, const int4* __restrict__ rep,
                                                  int n_rep, const double* __restrict__ ref, double* __restrict__ gs) {
    const int Lh = T.Lh;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long total = (long long)n_rep * (Lh + 1);
    if (tid >= total) return;
    const int di = (int)(tid / (Lh + 1));
    const int s = (int)(tid % (Lh + 1));
    const int4 d = rep[di];
    if (d.x == 0 && d.y == 0) {  // self-terms (FBC_PLAN_SELF_TERMS): filled by the lattice near field
        double* o0 = gs + ((size_t)di * (Lh + 1) + s) * 6;
        for (int t = 0; t < 6; t++) o0[t] = 0.0;
        return;
    }
    const double rx = (double)d.x, ry = (double)d.y;
    const double l3 = (double)T.L * T.c;
    const double z0 = (double)s * T.c;  // centred representative: s <= L/2
    CubicDir D;
    if (KIND == kGreenPoly) D = cubic_dir(M.m, rx, ry);
    auto green = [&](double z, double (&g)[6]) {
        if constexpr (KIND == kGreenIso) green_isotropic(M.m, rx, ry, z, g);
        else if constexpr (KIND == kGreenNodes) green_nodes(M.m, Q, rx, ry, z, g);
        else green_cubic(M, Q, D, rx, ry, z, g);
    };
    double acc[6], g[6], h[6];
    green(z0, acc);
    const int n = T.rich_n, N = T.rich_N;
    double tail[6] = {0, 0, 0, 0, 0, 0};
    for (int m = 1; m <= n + N; m++) {
        const double zm = (double)m * l3;
        green(z0 + zm, g);
        green(z0 - zm, h);
        const double* rf = ref + (m - 1) * 6;
        if (m <= n) {
#pragma unroll
            for (int t = 0; t < 6; t++) acc[t] += ((g[t] + h[t]) - rf[t]);
        } else {
            const double w = T.W[m - n - 1];
#pragma unroll
            for (int t = 0; t < 6; t++) tail[t] = fma(w, (g[t] + h[t]) - rf[t], tail[t]);
        }
    }
    double* o = gs + ((size_t)di * (Lh + 1) + s) * 6;
#pragma unroll
    for (int t = 0; t < 6; t++) o[t] = acc[t] + tail[t];
    if (s == Lh) {  // average of +L/2 and -L/2: odd entries cancel
        o[4] = 0.0;
        o[5] = 0.0;
    }
    if (s == 0) {  // exactly odd in s: zero at s = 0
        o[4] = 0.0;
        o[5] = 0.0;
    }
}

// Stage 2: one CTA per listed difference; threads over k.  The table entry of -d is that of d with the odd
// entries negated.
__global__ void k_line_dft(const __grid_constant__ TabulateParams T, const int4* __restrict__ rep,
                           const double* __restrict__ gs, const double2* __restrict__ twL, double* __restrict__ table) {
    extern __shared__ double sg[];  // [Lh+1][6]
    const int Lh = T.Lh, L = T.L, K = T.K;
    const int di = blockIdx.x;
    const double* src = gs + (size_t)di * (Lh + 1) * 6;
    for (int t = threadIdx.x; t < (Lh + 1) * 6; t += blockDim.x) sg[t] = src[t];
    __syncthreads();
    const int4 d = rep[di];
    const int ix = d.x - T.box_x0, iy = d.y - T.box_y0;
    const int mx = -d.x - T.box_x0, my = -d.y - T.box_y0;  // -d, in the box where it is used
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const double sgn = (k & 1) ? -1.0 : 1.0;
        double A0 = 0, A1 = 0, A2 = 0, A3 = 0, B4 = 0, B5 = 0;
        int ks = 0;
        for (int s = 1; s < Lh; s++) {
            ks += k;
            if (ks >= L) ks -= L;
            const double2 cs = twL[ks];
            const double* gp = sg + s * 6;
            A0 = fma(gp[0], cs.x, A0);
            A1 = fma(gp[1], cs.x, A1);
            A2 = fma(gp[2], cs.x, A2);
            A3 = fma(gp[3], cs.x, A3);
            B4 = fma(gp[4], cs.y, B4);
            B5 = fma(gp[5], cs.y, B5);
        }
        const double* g0 = sg;
        const double* gh = sg + Lh * 6;
        double v[6];
        v[0] = g0[0] + sgn * gh[0] + 2.0 * A0;
        v[1] = g0[1] + sgn * gh[1] + 2.0 * A1;
        v[2] = g0[2] + sgn * gh[2] + 2.0 * A2;
        v[3] = g0[3] + sgn * gh[3] + 2.0 * A3;
        v[4] = -2.0 * B4;
        v[5] = -2.0 * B5;
        double* o = table + (((size_t)k * T.Dy + iy) * T.Dx + ix) * 6;
#pragma unroll
        for (int t = 0; t < 6; t++) o[t] = v[t];
        if (d.z) {
            double* q = table + (((size_t)k * T.Dy + my) * T.Dx + mx) * 6;
#pragma unroll
            for (int t = 0; t < 6; t++) q[t] = t < 4 ? v[t] : -v[t];
        }
    }
}

// Derived tables for the reduced-precision contractions.
__global__ void k_derive_fp32(const double* __restrict__ t64, float* __restrict__ t32, size_t n) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t stride = (size_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) t32[i] = (float)t64[i];
}

// Double-float split: v = hi + lo with hi = fl32(v), lo = fl32(v - hi).  Stored
// per entry as the pairs (hi0, lo0, hi1, lo1, ..., hi5, lo5): three 16-byte
// records, the layout the contraction keeps in shared memory, so that a tile's
// sub-box is one tensor copy.
__global__ void k_derive_x2(const double* __restrict__ t64, float* __restrict__ tx2, size_t n_entries) {
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t stride = (size_t)gridDim.x * blockDim.x;
    for (; e < n_entries; e += stride) {
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const double v = t64[e * 6 + c];
            const float hi = (float)v;
            const float lo = (float)(v - (double)hi);
            tx2[e * 12 + 2 * c] = hi;
            tx2[e * 12 + 2 * c + 1] = lo;
        }
    }
}

}  // namespace

// Whether the polynomial form is as exact as the node-by-node one for a cubic medium: the cube of the mean eigenvalue of
// M(z) (its trace is C11 + 2 C44 for every unit z) over the smallest determinant at most 3, from 48 nodes on.  The
// determinant is linear in the elementary symmetric functions p, q of the squared components of z, so its minimum lies
// on the border of the range of (p, q), which the directions with squares (t, t, 1 - 2 t) reach.
// Errors against 64-bit mantissas (both forms emulated, 64 nodes, points of a slab), polynomial over node by node: 1500
// random media below 3, of |G| 0.71 to 0.89 on average and 1.03 at most, of the image sum 0.80 to 0.95 on average
// (single media scatter, 0.6 to 1.5).  Beyond, media of every bulk modulus: 1.2 at 4, 2 at 10, and without bound:
//     C11, C12, C44           quantity    rms error of |G|, nodes / poly     of the image sum
//     1.5, 1.0, 0.9              2.8        3.0e-16 / 3.0e-16              1.3e-13 / 1.4e-13
//     1.0, 0.9, 0.45             8.1        3.3e-16 / 6.3e-16              1.2e-13 / 2.7e-13
//     1.0, 0.2, 0.01           390          3.0e-16 / 5.8e-15              2.7e-14 / 1.3e-13
//     1.0, 0.99, 0.005        1500          6.6e-15 / 1.1e-13              6.9e-13 / 9.4e-12
// With fewer nodes the coefficients' rounding weighs more: below 3, 0.92 to 1.06 and 1.02 to 1.28 on average at 16 nodes,
// 0.75 to 0.86 and 0.88 to 1.04 at 48.
bool cubic_poly_form(const fbc_material& m, int nquad) {
    const double tr = m.C11 + 2.0 * m.C44, c11 = m.C11 / tr, c12 = m.C12 / tr, c44 = m.C44 / tr;  // any unit of stress
    const double h = c11 - c12 - 2.0 * c44;  // zero: isotropic
    double det = HUGE_VAL;
    for (int j = 0; j <= 96; j++) {  // (t = 0, 1/3, 1/2: the axes <100>, <111>, <110>)
        const double t = j / 192.0, r = 1.0 - 2.0 * t, p = t * (t + 2.0 * r), q = t * t * r;
        det = std::min(det, c11 * c44 * c44 + h * ((c11 + c12) * c44 * p + h * (c11 + 2.0 * c12 + c44) * q));
    }
    return nquad >= 48 && 1.0 <= 3.0 * 27.0 * det;
}

// A cubic plan's quadrature nodes and scaled constants, once.
static void make_tabulate_constants(Plan& P) {
    const int nq = P.mat.nquad;
    P.tab_nodes.assign((size_t)nq * 8, 0.0);  // [nq] cos, [nq] sin of psi, then [nq][6]
    for (int q = 0; q < nq; q++) {
        const double psi = M_PI * (double)q / (double)nq;
        P.tab_nodes[q] = cos(psi), P.tab_nodes[nq + q] = sin(psi);
        for (int j = 0; j < 3; j++) {
            const double a = M_PI * (double)((2LL * (j + 1) * q) % (2LL * nq)) / (double)nq;
            P.tab_nodes[(size_t)2 * nq + q * 6 + 2 * j] = cos(a);
            P.tab_nodes[(size_t)2 * nq + q * 6 + 2 * j + 1] = sin(a);
        }
    }
    // the constants scaled by a power of two to a largest magnitude in [1, 2): products of four
    // determinants stay in range whatever the unit of stress
    double top = 0.0;
    for (int t = 0; t < 36; t++) top = std::max(top, std::fabs(P.mat.K[t]));
    const double sc = std::ldexp(1.0, -std::ilogb(top));
    P.tab_mat = P.mat;
    for (int t = 0; t < 36; t++) P.tab_mat.K[t] = P.mat.K[t] * sc;
    P.tab_pre = sc / (M_PI * (double)nq);
}

// Stage 1 of nd listed differences from d0 on (ref: the images' reference sums).
template <int KIND>
static cudaError_t launch_periodic(Plan& P, int d0, int nd, double* ref, double* gs, cudaStream_t st) {
    if (KIND != kGreenIso && P.tab_nodes.empty()) make_tabulate_constants(P);
    Medium M;
    M.m = KIND == kGreenPoly ? P.tab_mat : P.mat, M.pre = P.tab_pre;
    QuadNodes<KIND> N{};
    if constexpr (KIND != kGreenIso) {
        const int nq = P.mat.nquad;
        const double* v = P.tab_nodes.data();
        for (int q = 0; q < nq; q++) {
            if constexpr (KIND == kGreenPoly) std::copy(v + 2 * nq + 6 * q, v + 2 * nq + 6 * q + 6, N.v[q]);
            else N.v[q][0] = v[q], N.v[q][1] = v[nq + q];
        }
    }
    if (d0 == 0) k_reference<KIND><<<P.tp.rich_n + P.tp.rich_N, 2, 0, st>>>(M, N, P.tp, ref);
    const long long threads = (long long)nd * (P.L / 2 + 1);
    k_periodic<KIND><<<(unsigned)((threads + 127) / 128), 128, 0, st>>>(M, N, P.tp, P.d_rep + d0, nd, ref, gs);
    return cudaGetLastError();
}

// The stage-1 buffer (differences in chunks of at most 256 MB) after the reference sums, and
// `stage2(d0, nd, gs)` for every chunk.
template <class F>
static cudaError_t tabulate_chunks(Plan& P, int kind, cudaStream_t st, F stage2) {
    if (P.n_rep == 0) return cudaSuccess;
    cudaError_t e;
    const size_t per_d = (size_t)(P.L / 2 + 1) * 6 * sizeof(double);
    const size_t n_ref = kMaxRichImages * 6;
    const int chunk = (int)std::min<size_t>((size_t)P.n_rep, std::max<size_t>(1, ((size_t)256 << 20) / per_d));
    double* buf = nullptr;
    if ((e = cudaMallocAsync((void**)&buf, n_ref * sizeof(double) + per_d * chunk, st))) return e;
    double* gs = buf + n_ref;
    for (int d0 = 0; d0 < P.n_rep && !e; d0 += chunk) {
        const int nd = std::min(chunk, P.n_rep - d0);
        e = kind == kGreenIso     ? launch_periodic<kGreenIso>(P, d0, nd, buf, gs, st)
            : kind == kGreenNodes ? launch_periodic<kGreenNodes>(P, d0, nd, buf, gs, st)
                                  : launch_periodic<kGreenPoly>(P, d0, nd, buf, gs, st);
        if (!e) e = stage2(d0, nd, gs);
    }
    cudaError_t e2 = cudaFreeAsync(buf, st);
    return e ? e : e2;
}

cudaError_t launch_tabulate(Plan& P, cudaStream_t st) {
    const size_t smem = (size_t)(P.L / 2 + 1) * 6 * sizeof(double);
    if (smem > 32 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_line_dft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e) return e;
    }
    const int kind = P.mat.kind == FBC_MATERIAL_ISOTROPIC          ? kGreenIso
                     : line_fp32(P.precision) || !P.tab_poly ? kGreenNodes
                                                             : kGreenPoly;
    return tabulate_chunks(P, kind, st, [&](int d0, int nd, const double* gs) {
        const int bt = std::min(256, std::max(32, ((P.K + 31) / 32) * 32));
        k_line_dft<<<nd, bt, smem, st>>>(P.tp, P.d_rep + d0, gs, P.d_twL, P.d_table);
        return cudaGetLastError();
    });
}

// Stage-1 output of a chunk of listed differences, rounded to FP32 and placed at each difference's
// cell of the box (and its mirror's, the odd entries negated): out[cell][s][6] for s = 0..L/2.
__global__ void k_real_space_scatter(const __grid_constant__ TabulateParams T, const int4* __restrict__ rep, int n_rep,
                                     const double* __restrict__ gs, float* __restrict__ out) {
    const int Lh = T.Lh;
    const long long per = (long long)(Lh + 1) * 6;
    const long long total = (long long)n_rep * per;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int di = (int)(t / per);
        const long long r = t - (long long)di * per;
        const int4 d = rep[di];
        const float v = (float)gs[t];
        out[((long long)(d.y - T.box_y0) * T.Dx + (d.x - T.box_x0)) * per + r] = v;
        if (d.z) out[((long long)(-d.y - T.box_y0) * T.Dx + (-d.x - T.box_x0)) * per + r] = r % 6 < 4 ? v : -v;
    }
}

cudaError_t launch_real_space_table(Plan& P, float* out, cudaStream_t st) {
    const size_t cells = (size_t)P.Dx * P.Dy;
    cudaError_t e = cudaMemsetAsync(out, 0, cells * (P.L / 2 + 1) * 6 * sizeof(float), st);
    if (e) return e;
    const int kind = P.mat.kind == FBC_MATERIAL_ISOTROPIC ? kGreenIso : kGreenNodes;
    return tabulate_chunks(P, kind, st, [&](int d0, int nd, const double* gs) {
        k_real_space_scatter<<<1216, 256, 0, st>>>(P.tp, P.d_rep + d0, nd, gs, out);
        return cudaGetLastError();
    });
}

cudaError_t launch_derive_tables(Plan& P, int precision, cudaStream_t st) {
    const size_t cells = (size_t)P.K * P.Dy * P.Dx;
    if (precision == FBC_PREC_FP32 || is_tensor_precision(precision)) {
        if (!P.d_table32 || !P.d_table_x2_k0) return cudaErrorInvalidValue;
        k_derive_fp32<<<1216, 256, 0, st>>>(P.d_table, P.d_table32, cells * 6);
        cudaError_t e = cudaGetLastError();
        if (e) return e;
        k_derive_x2<<<1216, 256, 0, st>>>(P.d_table, P.d_table_x2_k0, (size_t)P.Dy * P.Dx);  // k = 0 slice
        return cudaGetLastError();
    }
    if (is_fft_precision(precision)) return launch_fft_tables(P, precision, st);
    if (precision == FBC_PREC_F32X2 || precision == FBC_PREC_BF16X6) {
        if (!P.d_table_x2) return cudaErrorInvalidValue;
        k_derive_x2<<<1216, 256, 0, st>>>(P.d_table, P.d_table_x2, cells);
        return cudaGetLastError();
    }
    return cudaSuccess;
}

}  // namespace fbc
