// setup3d.cu -- 3-D setup kernels: trilinear Q1 assembly from the map
// (Sec. 2.1 in 3-D: 2x2x2 Gauss points, effective coefficient
// kappa det J J^-1 J^-T), operator-induced interpolation by hierarchical
// collapse (lines, then planes, then the cell centre) and Galerkin coarse
// operators P^T A P (Sec. 2.2), exports and the per-cell adjoint contraction.
#include "common.cuh"
#include "grid3.cuh"

namespace bmg {
namespace {

constexpr double kG0 = 0.21132486540518711775;
constexpr double kG1 = 0.78867513459481288225;

// Coefficient of a cell, as the metric it induces from adj(J) = det J J^-1
// (the 1/8 is the Gauss weight).  Scalar kappa: G = (kappa / det J) adj
// adj^T.  SPD tensor D (Sec. 2, Eq. pde): G = (1 / det J) adj D adj^T.
struct Scalar3 {
    double kap;
    __device__ __forceinline__ void metric(const double adj[3][3], double det, double G[3][3]) const {
        const double s = 0.125 * kap / det;
#pragma unroll
        for (int m = 0; m < 3; m++)
#pragma unroll
            for (int p = 0; p < 3; p++)
                G[m][p] = s * (adj[m][0] * adj[p][0] + adj[m][1] * adj[p][1] + adj[m][2] * adj[p][2]);
    }
};
struct Tensor3 {
    double d[3][3];
    __device__ __forceinline__ void metric(const double adj[3][3], double det, double G[3][3]) const {
        const double s = 0.125 / det;
        double t[3][3];   // adj D
#pragma unroll
        for (int m = 0; m < 3; m++)
#pragma unroll
            for (int c = 0; c < 3; c++) t[m][c] = adj[m][0] * d[0][c] + adj[m][1] * d[1][c] + adj[m][2] * d[2][c];
#pragma unroll
        for (int m = 0; m < 3; m++)
#pragma unroll
            for (int p = 0; p < 3; p++)
                G[m][p] = s * (t[m][0] * adj[p][0] + t[m][1] * adj[p][1] + t[m][2] * adj[p][2]);
    }
};

// Row `a` of the trilinear element matrix of cell (ci,cj,ck):
// Krow[b] = sum_q 1/8 grad(phi_a)^T G grad(phi_b), G from the cell's
// coefficient (above).  Corner b = bx + 2 by + 4 bz sits at node
// (ci+bx, cj+by, ck+bz).
template <class C>
__device__ bool element_row3d(const double* __restrict__ coords, int n, int ci, int cj, int ck, const C& coef, int a,
                              double Krow[8]) {
    const long long nn = (long long)n * n * n;
    double xa[3][8];
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const long long id = (long long)(ci + (b & 1)) + (long long)n * ((cj + ((b >> 1) & 1)) + (long long)n * (ck + (b >> 2)));
#pragma unroll
        for (int r = 0; r < 3; r++) xa[r][b] = coords[r * nn + id];
    }
#pragma unroll
    for (int b = 0; b < 8; b++) Krow[b] = 0.0;
    bool ok = true;
    for (int q = 0; q < 8; q++) {
        const double xi[3] = {(q & 1) ? kG1 : kG0, (q & 2) ? kG1 : kG0, (q & 4) ? kG1 : kG0};
        double g[8][3];
#pragma unroll
        for (int b = 0; b < 8; b++) {
            const double f0 = (b & 1) ? xi[0] : 1.0 - xi[0];
            const double f1 = (b & 2) ? xi[1] : 1.0 - xi[1];
            const double f2 = (b & 4) ? xi[2] : 1.0 - xi[2];
            const double d0 = (b & 1) ? 1.0 : -1.0, d1 = (b & 2) ? 1.0 : -1.0, d2 = (b & 4) ? 1.0 : -1.0;
            g[b][0] = d0 * f1 * f2;
            g[b][1] = f0 * d1 * f2;
            g[b][2] = f0 * f1 * d2;
        }
        double J[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
        for (int b = 0; b < 8; b++)
#pragma unroll
            for (int r = 0; r < 3; r++)
#pragma unroll
                for (int m = 0; m < 3; m++) J[r][m] += xa[r][b] * g[b][m];
        // adjugate (transpose of the cofactor matrix): J^-1 = adj / det
        double adj[3][3];
        adj[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
        adj[0][1] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
        adj[0][2] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
        adj[1][0] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
        adj[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
        adj[1][2] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
        adj[2][0] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
        adj[2][1] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
        adj[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
        const double det = J[0][0] * adj[0][0] + J[0][1] * adj[1][0] + J[0][2] * adj[2][0];
        if (!(det > 0.0)) ok = false;
        double G[3][3];
        coef.metric(adj, det, G);
        const double ga0 = G[0][0] * g[a][0] + G[0][1] * g[a][1] + G[0][2] * g[a][2];
        const double ga1 = G[1][0] * g[a][0] + G[1][1] * g[a][1] + G[1][2] * g[a][2];
        const double ga2 = G[2][0] * g[a][0] + G[2][1] * g[a][1] + G[2][2] * g[a][2];
#pragma unroll
        for (int b = 0; b < 8; b++) Krow[b] += ga0 * g[b][0] + ga1 * g[b][1] + ga2 * g[b][2];
    }
    return ok;
}

// Reference-cell derivatives of a trilinear field given at a cell's corners,
// kept in the form the Gauss loop needs.  d/dxi is bilinear in (eta, zeta),
// so it is interpolated from the four xi-edges' differences (first in eta, the
// value and its zeta slope kept); d/deta likewise; d/dzeta does not depend on
// zeta.  Formed once per cell: 48 FP64 operations, where a sum over the eight
// corners at every Gauss point takes 192.
struct EdgeMap3 {
    double u0[2], du[2];   // d/dxi at (eta_q, zeta = 0) and its zeta slope
    double v0[2], dv[2];   // d/deta at (xi_q, zeta = 0) and its zeta slope
    double w[2][2];        // d/dzeta at (xi_q, eta_p)
    __device__ __forceinline__ void set(const double x[8]) {
        const double ex[4] = {x[1] - x[0], x[3] - x[2], x[5] - x[4], x[7] - x[6]};   // [by + 2 bz]
        const double ey[4] = {x[2] - x[0], x[3] - x[1], x[6] - x[4], x[7] - x[5]};   // [bx + 2 bz]
        const double ez[4] = {x[4] - x[0], x[5] - x[1], x[6] - x[2], x[7] - x[3]};   // [bx + 2 by]
        const double ax = ex[1] - ex[0], bx = ex[3] - ex[2];
        const double ay = ey[1] - ey[0], by = ey[3] - ey[2];
        const double az = ez[1] - ez[0], bz = ez[3] - ez[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const double g = q ? kG1 : kG0;
            u0[q] = ex[0] + g * ax;
            du[q] = (ex[2] + g * bx) - u0[q];
            v0[q] = ey[0] + g * ay;
            dv[q] = (ey[2] + g * by) - v0[q];
            const double lo = ez[0] + g * az, hi = ez[2] + g * bz;   // at eta = 0, 1
            w[q][0] = lo + kG0 * (hi - lo);
            w[q][1] = lo + kG1 * (hi - lo);
        }
    }
    // derivatives at Gauss point (xi_q, eta_p) of the plane zeta = g
    __device__ __forceinline__ void at(int q, int p, double g, double& dxi, double& deta, double& dzeta) const {
        dxi = u0[p] + g * du[p];
        deta = v0[q] + g * dv[q];
        dzeta = w[q][p];
    }
};

// The three coordinates of a cell's trilinear map.
struct CellMap3 {
    EdgeMap3 c[3];
    __device__ __forceinline__ void load(const double* __restrict__ coords, int n, int ci, int cj, int ck) {
        const long long nn = (long long)n * n * n;
        const long long id = (long long)ci + (long long)n * (cj + (long long)n * ck);
        const long long sy = n, sz = (long long)n * n;
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const double* X = coords + r * nn + id;
            double x[8];
#pragma unroll
            for (int b = 0; b < 8; b++) x[b] = X[(b & 1) + sy * ((b >> 1) & 1) + sz * (b >> 2)];
            c[r].set(x);
        }
    }
    // adjugate rows (J^-1 = adj / det) and determinant at a Gauss point
    __device__ __forceinline__ double adjugate(int q, int p, double g, double adj[3][3]) const {
        double u[3], v[3], w[3];
#pragma unroll
        for (int r = 0; r < 3; r++) c[r].at(q, p, g, u[r], v[r], w[r]);
        cross(v, w, adj[0]);
        cross(w, u, adj[1]);
        cross(u, v, adj[2]);
        return u[0] * adj[0][0] + u[1] * adj[0][1] + u[2] * adj[0][2];
    }
    static __device__ __forceinline__ void cross(const double* a, const double* b, double* r) {
        r[0] = a[1] * b[2] - a[2] * b[1];
        r[1] = a[2] * b[0] - a[0] * b[2];
        r[2] = a[0] * b[1] - a[1] * b[0];
    }
};

// Contractions of two Gauss-point values with the products (1-t)^2, t(1-t),
// t^2 of the linear shape functions, as sum and difference (the squares are
// 1/3 +- 1/(2 sqrt 3) at the two points): where the metric is constant the
// entries keep the exact ratios 2 : 1 : 2, and the element's row sums stay
// exact zeros.
constexpr double kThird = 1.0 / 3.0, kSixth = 1.0 / 6.0, kHalfGap = 0.5 * (kG1 - kG0);

__device__ __forceinline__ void pair3(double s0, double s1, double out[3]) {
    const double S = s0 + s1, D = s0 - s1, t = kThird * S;
    out[0] = t + kHalfGap * D;
    out[1] = kSixth * S;
    out[2] = t - kHalfGap * D;
}
__device__ __forceinline__ void lin2(double s0, double s1, double out[2]) {
    out[0] = kG1 * s0 + kG0 * s1;
    out[1] = kG0 * s0 + kG1 * s1;
}

// Element matrix of one cell, K_ab = sum_q 1/8 grad(phi_a)^T G grad(phi_b), as
// its three blocks over the corners' z bits: K00 and K11 (symmetric, entries
// a' <= b' of the in-plane corners, in the order of sym4) and K01[a'][b']
// (a at z bit 0, b at z bit 1).  Sum factorisation: the shape functions are
// products of 1 - t, t per direction, so the 2x2x2 Gauss sum contracts one
// direction at a time, with per-plane (zeta) partial sums:
//   in-plane corners a' = ax + 2 ay, signs s = -1, +1 for bit 0, 1
//   Q[a'b'] = sx sx' M11[ay+by] + sy sy' M22[ax+bx] + sx sy' N12[ay][bx] + sx' sy N12[by][ax]
//   R[a'b'] = sx N13[ay+by][bx] + sy N23[ax+bx][by]
//   T[a'b'] = M33[ax+bx][ay+by]
//   K_ab = sum_zeta f_az f_bz Q + sz' f_az R[a'b'] + sz f_bz R[b'a'], + sz sz' T
// About 1100 FP64 operations a cell in all, against 8 rows x 8 points x
// about 140 for the direct sum.  Edge differences are formed before anything
// is summed, so the coordinates' magnitude does not cancel out of J.
__host__ __device__ constexpr int sym4(int a, int b) {   // a <= b
    return a * 4 - a * (a - 1) / 2 + (b - a);
}
template <class C>
__device__ __forceinline__ bool element3d(const CellMap3& M, const C& coef, double K00[10], double K11[10],
                                          double K01[16]) {
#pragma unroll
    for (int t = 0; t < 10; t++) K00[t] = K11[t] = 0.0;
#pragma unroll
    for (int t = 0; t < 16; t++) K01[t] = 0.0;
    double S33[2][2] = {{0, 0}, {0, 0}};
    bool ok = true;
#pragma unroll 1
    for (int qz = 0; qz < 2; qz++) {
        const double g = qz ? kG1 : kG0, h = qz ? kG0 : kG1;   // zeta, 1 - zeta
        double S11[2], S22[2] = {0, 0}, n12[2][2], n13[2][2], g12[2][2];
#pragma unroll
        for (int p = 0; p < 2; p++) {
            double g01[2], g02[2], s11[2];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                double adj[3][3], G[3][3];
                const double det = M.adjugate(q, p, g, adj);
                if (!(det > 0.0)) ok = false;
                coef.metric(adj, det, G);
                s11[q] = G[0][0];
                S22[q] += G[1][1];
                S33[q][p] += G[2][2];
                g01[q] = G[0][1];
                g02[q] = G[0][2];
                g12[q][p] = G[1][2];
            }
            S11[p] = s11[0] + s11[1];
            lin2(g01[0], g01[1], n12[p]);
            lin2(g02[0], g02[1], n13[p]);
        }
        double M11[3], M22[3], N12[2][2], N13[3][2], N23[3][2];
        pair3(S11[0], S11[1], M11);
        pair3(S22[0], S22[1], M22);
        {
            double n23[2][2];
            lin2(g12[0][0], g12[0][1], n23[0]);
            lin2(g12[1][0], g12[1][1], n23[1]);
#pragma unroll
            for (int b = 0; b < 2; b++) {
                double t2[2], t3[3];
                lin2(n12[0][b], n12[1][b], t2);
                N12[0][b] = t2[0];
                N12[1][b] = t2[1];
                pair3(n13[0][b], n13[1][b], t3);
                N13[0][b] = t3[0];
                N13[1][b] = t3[1];
                N13[2][b] = t3[2];
                pair3(n23[0][b], n23[1][b], t3);
                N23[0][b] = t3[0];
                N23[1][b] = t3[1];
                N23[2][b] = t3[2];
            }
        }
        double R[16];
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int b = 0; b < 4; b++) {
                const int ax = a & 1, ay = a >> 1, bx = b & 1, by = b >> 1;
                const double x = N13[ay + by][bx], y = N23[ax + bx][by];
                R[4 * a + b] = ax ? (ay ? x + y : x - y) : (ay ? y - x : -x - y);
            }
        const double w00 = h * h, w01 = kSixth, w11 = g * g;
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int b = a; b < 4; b++) {
                const int ax = a & 1, ay = a >> 1, bx = b & 1, by = b >> 1;
                const double m1 = M11[ay + by], m2 = M22[ax + bx], c1 = N12[ay][bx], c2 = N12[by][ax];
                double Q = ax == bx ? m1 : -m1;
                Q = ay == by ? Q + m2 : Q - m2;
                Q = ax == by ? Q + c1 : Q - c1;
                Q = bx == ay ? Q + c2 : Q - c2;
                const double rs = R[4 * a + b] + R[4 * b + a];
                const int t = sym4(a, b);
                K00[t] += w00 * Q;
                K00[t] -= h * rs;
                K11[t] += w11 * Q;
                K11[t] += g * rs;
                K01[4 * a + b] += w01 * Q;
                K01[4 * a + b] += h * R[4 * a + b];
                K01[4 * a + b] -= g * R[4 * b + a];
                if (a != b) {
                    K01[4 * b + a] += w01 * Q;
                    K01[4 * b + a] += h * R[4 * b + a];
                    K01[4 * b + a] -= g * R[4 * a + b];
                }
            }
    }
    // d/dzeta d/dzeta: xi pairs for both eta, then eta pairs
    double T[3][3];
    {
        double t0[3], t1[3];
        pair3(S33[0][0], S33[1][0], t0);
        pair3(S33[0][1], S33[1][1], t1);
#pragma unroll
        for (int x = 0; x < 3; x++) pair3(t0[x], t1[x], T[x]);
    }
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const double t = T[(a & 1) + (b & 1)][(a >> 1) + (b >> 1)];
            if (a <= b) {
                K00[sym4(a, b)] += t;
                K11[sym4(a, b)] += t;
            }
            K01[4 * a + b] -= t;
        }
    return ok;
}

__device__ __forceinline__ bool inner3(int n, int i, int j, int k) {
    return i >= 1 && j >= 1 && k >= 1 && i <= n - 2 && j <= n - 2 && k <= n - 2;
}

// coefficient of cell e: kappa[e], or the tensor planes D11, D12, D13, D22,
// D23, D33 (ne cells each)
template <bool TENSOR>
__device__ __forceinline__ auto cell_coef3(const double* __restrict__ c, long long ne, long long e) {
    if constexpr (TENSOR) {
        const double d11 = c[e], d12 = c[ne + e], d13 = c[2 * ne + e], d22 = c[3 * ne + e], d23 = c[4 * ne + e],
                     d33 = c[5 * ne + e];
        return Tensor3{{{d11, d12, d13}, {d12, d22, d23}, {d13, d23, d33}}};
    } else {
        return Scalar3{c[e]};
    }
}

// Gather assembly (no atomics).  A CTA owns a column of kAsm3N x kAsm3N nodes
// and a band of H node planes and marches up k one layer of cells at a time:
// its kAsm3C x kAsm3C threads form the element matrices of the layer's cells
// around the column (one cell each) into shared memory, then the node threads
// add the layer's entries to the plane below it, which that completes, and
// start the plane above.  A node's nine couplings to the plane below are
// complete after one layer and are stored at once, so only the five in-plane
// sums are carried to the next layer.  Each cell is formed once per column
// (a 16/15 halo in i and j, one layer per band) instead of once per node.
// FP64 arithmetic bounds this kernel (two FMA per SM and clock: one FP64
// instruction of a warp occupies a scheduler's unit for 64 cycles, so two
// warps per scheduler at up to 255 registers keep it busy); its 144 bytes per
// node take about a hundredth of its time.  129^3: 5.74 ms, where a thread per
// node forming eight matrix rows by the direct sum took 44.9 ms.
constexpr int kAsm3C = 16, kAsm3N = kAsm3C - 1, kAsm3Threads = kAsm3C * kAsm3C;
constexpr size_t kAsm3Smem = sizeof(double) * 36 * kAsm3Threads;

template <bool TENSOR>
__global__ void __launch_bounds__(kAsm3Threads, 1) k_assemble3d(int n, int ld, long long pl, int H,
                                                                const double* __restrict__ coords,
                                                                const double* __restrict__ kappa,
                                                                double* __restrict__ A, KState* st) {
    extern __shared__ __align__(16) unsigned char asm3_raw[];
    double* sK = reinterpret_cast<double*>(asm3_raw);   // [36][kAsm3Threads]: K00, K11, K01
    const long long ne = (long long)(n - 1) * (n - 1) * (n - 1);
    const int t = threadIdx.x;
    const int i0 = blockIdx.x * kAsm3N, j0 = blockIdx.y * kAsm3N;   // first node of the column
    const int k0 = blockIdx.z * H, k1 = min(k0 + H, n);             // node planes [k0, k1)
    const int ci = i0 - 1 + t % kAsm3C, cj = j0 - 1 + t / kAsm3C;   // this thread's cell column
    const bool cell_in = ci >= 0 && cj >= 0 && ci <= n - 2 && cj <= n - 2;
    const int ni = t % kAsm3N, nj = t / kAsm3N;                     // this thread's node of the column
    const int i = i0 + ni, j = j0 + nj;
    const bool node = t < kAsm3N * kAsm3N && i < n && j < n;
    const bool in2 = node && i >= 1 && j >= 1 && i <= n - 2 && j <= n - 2;
    const long long sz = (long long)ld * n, oij = (long long)i + (long long)ld * j;
    // slot of the cell that has this node as in-plane corner a' = (ax, ay)
    auto slot = [&](int a) { return (ni + 1 - (a & 1)) + kAsm3C * (nj + 1 - (a >> 1)); };
    double part[5] = {0, 0, 0, 0, 0};   // in-plane offsets 9..13 of the plane in progress
    // adds the block (K00 or K11) of corner a' = in-plane corner of the node
    auto add_plane = [&](int base) {
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const int a = 3 - c;        // cells in ascending order: the node is their corner 3, 2, 1, 0
            const double* K = sK + (size_t)base * kAsm3Threads + slot(a);
#pragma unroll
            for (int b = 0; b < 4; b++) {
                const int dx = (b & 1) - (a & 1), dy = (b >> 1) - (a >> 1);
                const int o = (dx + 1) + 3 * (dy + 1);
                if (o > 4) continue;
                const int lo = a < b ? a : b, hi = a < b ? b : a;
                part[o] += K[(size_t)sym4(lo, hi) * kAsm3Threads];
            }
        }
    };
    for (int ck = k0 - 1; ck < k1; ck++) {   // layers k0-1 .. k1-1
        if (ck >= 0 && ck <= n - 2 && cell_in) {
            CellMap3 M;
            M.load(coords, n, ci, cj, ck);
            const long long e = (long long)ci + (long long)(n - 1) * (cj + (long long)(n - 1) * ck);
            double K00[10], K11[10], K01[16];
            if (!element3d(M, cell_coef3<TENSOR>(kappa, ne, e), K00, K11, K01)) set_err(st, BMG_ERR_MAP_FOLDED);
#pragma unroll
            for (int q = 0; q < 10; q++) {
                sK[(size_t)q * kAsm3Threads + t] = K00[q];
                sK[(size_t)(10 + q) * kAsm3Threads + t] = K11[q];
            }
#pragma unroll
            for (int q = 0; q < 16; q++) sK[(size_t)(20 + q) * kAsm3Threads + t] = K01[q];
        }
        __syncthreads();
        if (ck >= k0 && node) {   // plane ck is complete with this layer above it
            const long long o = oij + sz * ck;
            const bool in = in2 && ck >= 1 && ck <= n - 2;
            if (in) add_plane(0);
#pragma unroll
            for (int q = 0; q < 5; q++) {
                const bool keep = in && inner3(n, i + q % 3 - 1, j + q / 3 - 1, ck);
                A[(long long)(9 + q) * pl + o] = keep ? part[q] : 0.0;
            }
        }
        if (ck + 1 < k1 && node) {   // this layer lies below plane ck + 1
            const int k = ck + 1;
            const long long o = oij + sz * k;
            const bool in = in2 && k >= 1 && k <= n - 2;
            double low[9];
#pragma unroll
            for (int q = 0; q < 9; q++) low[q] = 0.0;
#pragma unroll
            for (int q = 0; q < 5; q++) part[q] = 0.0;
            if (in) {
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    const int a = 3 - c;
                    const double* K = sK + (size_t)20 * kAsm3Threads + slot(a);
#pragma unroll
                    for (int b = 0; b < 4; b++) {
                        const int dx = (b & 1) - (a & 1), dy = (b >> 1) - (a >> 1);
                        low[(dx + 1) + 3 * (dy + 1)] += K[(size_t)(4 * b + a) * kAsm3Threads];
                    }
                }
                add_plane(10);
            }
#pragma unroll
            for (int q = 0; q < 9; q++) {
                const bool keep = in && inner3(n, i + q % 3 - 1, j + q / 3 - 1, k - 1);
                A[(long long)q * pl + o] = keep ? low[q] : 0.0;
            }
        }
        __syncthreads();
    }
}

// Launches k_assemble3d; planes per band: the one that minimises waves x
// (planes + 1 layer of pre-roll) at one CTA per SM.
template <bool TENSOR>
bmg_status launch_assemble3d(int n, int ld, long long pl, const double* coords, const double* coef, double* A,
                             KState* st, cudaStream_t s) {
    int dev = 0, sms = 0;
    BMG_CUDA(cudaGetDevice(&dev));
    BMG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    BMG_CUDA(cudaFuncSetAttribute(k_assemble3d<TENSOR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAsm3Smem));
    const int cols = cdiv(n, kAsm3N);
    int H = n;
    long long best = -1;
    for (int bands = 1; bands <= n; bands++) {
        const int h = cdiv(n, bands);
        const long long cost = (long long)cdiv((long long)cols * cols * cdiv(n, h), sms) * (h + 1);
        if (best < 0 || cost < best) {
            best = cost;
            H = h;
        }
    }
    k_assemble3d<TENSOR><<<dim3(cols, cols, cdiv(n, H)), kAsm3Threads, kAsm3Smem, s>>>(n, ld, pl, H, coords, coef, A, st);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

__global__ void k_set_stencil3d(int n, int ld, long long pl, const double* __restrict__ full, double* __restrict__ A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y, k = blockIdx.z;
    if (i >= n) return;
    const long long o = (long long)i + (long long)ld * (j + (long long)n * k);
    const bool in = inner3(n, i, j, k);
    const double* row = full + ((long long)i + (long long)n * (j + (long long)n * k)) * 27;
    for (int t = 0; t < 14; t++) {
        double v = 0.0;
        if (in && (t == 13 || inner3(n, i + off_x(t), j + off_y(t), k + off_z(t)))) v = row[t];
        A[(long long)t * pl + o] = v;
    }
}

struct CoarseDims {
    int nf, nc, ldc;
    long long plc;
    __device__ __forceinline__ long long at(int I, int J, int K) const {
        return (long long)I + (long long)ldc * (J + (long long)nc * K);
    }
    __device__ __forceinline__ bool inner(int I, int J, int K) const {
        return I >= 1 && J >= 1 && K >= 1 && I <= nc - 2 && J <= nc - 2 && K <= nc - 2;
    }
};

// Line points (one odd coordinate): collapse the 27-point row over the plane
// perpendicular to the odd axis.  Where the collapsed denominator is not
// positive the point uses its own couplings along the axis (a_000 > 0).
__global__ void k_interp_lines3d(Sten3<double> F, CoarseDims D, double* __restrict__ P, KState* st) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y, K = blockIdx.z;
    if (I >= D.nc) return;
    const long long oc = D.at(I, J, K);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int fi = 2 * I + (a == 0), fj = 2 * J + (a == 1), fk = 2 * K + (a == 2);
        double lo = 0.0, hi = 0.0;
        if (inner3(D.nf, fi, fj, fk)) {
            double S[3] = {0, 0, 0};
#pragma unroll
            for (int o = 0; o < 27; o++) {
                const int d = a == 0 ? off_x(o) : a == 1 ? off_y(o) : off_z(o);
                S[d + 1] += F.full(fi, fj, fk, o);
            }
            if (!(S[1] > 0.0)) {
                const int step = a == 0 ? 1 : a == 1 ? 3 : 9;   // offset of +e_a in the 27-numbering
                S[0] = F.full(fi, fj, fk, 13 - step);
                S[1] = F.full(fi, fj, fk, 13);
                S[2] = F.full(fi, fj, fk, 13 + step);
            }
            if (!(S[1] > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
            const int ax = a == 0 ? I : a == 1 ? J : K;
            lo = ax >= 1 ? -S[0] / S[1] : 0.0;
            hi = ax + 1 <= D.nc - 2 ? -S[2] / S[1] : 0.0;
        }
        const int base = kPBase(1 << a);
        P[(long long)base * D.plc + oc] = lo;
        P[(long long)(base + 1) * D.plc + oc] = hi;
    }
}

// Everything below is fixed by the offsets, so the loops unroll to plain
// loads and products (129^3 hierarchy: lines 175 us, planes 227 us, centres
// 139 us; with run-time weight look-ups 332, 846 and 718 us): which plane holds the weight of the fine point at
// offset g (in [-2, 2]^3 from the fine point 2(I,J,K)) to the coarse node
// (I,J,K) + e, and at which coarse node it is stored.
//   parity mask m of g, owner q = floor(g / 2), subset s = e - q of m
__host__ __device__ constexpr int half_floor(int g) { return g >= 0 ? g / 2 : -((1 - g) / 2); }
__host__ __device__ constexpr bool parent1(int g, int e) {   // one direction
    return e - half_floor(g) >= 0 && e - half_floor(g) <= (g & 1);
}
__host__ __device__ constexpr bool parent3(int gx, int gy, int gz, int ex, int ey, int ez) {
    return parent1(gx, ex) && parent1(gy, ey) && parent1(gz, ez);
}
__device__ __forceinline__ double weight3(const double* P, const CoarseDims& D, long long oc, int gx, int gy, int gz,
                                          int ex, int ey, int ez) {
    const int m = (gx & 1) | ((gy & 1) << 1) | ((gz & 1) << 2);
    if (m == 0) return 1.0;
    const int qx = half_floor(gx), qy = half_floor(gy), qz = half_floor(gz);
    const int s = (ex - qx) | ((ey - qy) << 1) | ((ez - qz) << 2);
    return P[(long long)(kPBase(m) + compress3(s, m)) * D.plc + oc + qx + (long long)D.ldc * (qy + (long long)D.nc * qz)];
}

// Plane points (two odd coordinates): collapse over the even axis, then solve
// the collapsed plane equation with the in-plane neighbours interpolated.
// Where the collapsed diagonal is not positive the point uses its own
// in-plane couplings (no collapse; the diagonal a_000 > 0).
__global__ void k_interp_planes3d(Sten3<double> F, CoarseDims D, double* __restrict__ P, KState* st) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y, K = blockIdx.z;
    if (I >= D.nc) return;
    const long long oc = D.at(I, J, K);
#pragma unroll
    for (int t = 0; t < 3; t++) {
        const int m = t == 0 ? 3 : t == 1 ? 5 : 6;
        const int e = 2 - t;                            // the even axis
        const int a0 = t == 2 ? 1 : 0, a1 = t == 0 ? 1 : 2;   // the odd axes
        const int fi = 2 * I + (m & 1), fj = 2 * J + ((m >> 1) & 1), fk = 2 * K + ((m >> 2) & 1);
        double w[4] = {0, 0, 0, 0};
        if (inner3(D.nf, fi, fj, fk)) {
            double cf[9];                               // in-plane offsets (d0 + 1) + 3 (d1 + 1)
#pragma unroll
            for (int q = 0; q < 9; q++) cf[q] = 0.0;
            auto dir = [](int o, int a) { return a == 0 ? off_x(o) : a == 1 ? off_y(o) : off_z(o); };
#pragma unroll
            for (int o = 0; o < 27; o++) cf[(dir(o, a0) + 1) + 3 * (dir(o, a1) + 1)] += F.full(fi, fj, fk, o);
            if (!(cf[4] > 0.0)) {
#pragma unroll
                for (int o = 0; o < 27; o++)
                    if (dir(o, e) == 0) cf[(dir(o, a0) + 1) + 3 * (dir(o, a1) + 1)] = F.full(fi, fj, fk, o);
            }
            const double d0 = cf[4];
            if (!(d0 > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const int s0 = c & 1, s1 = c >> 1;      // corner c of the odd-axis cell
                const int sx = a0 == 0 ? s0 : 0, sy = a0 == 1 ? s0 : a1 == 1 ? s1 : 0, sz = a1 == 2 ? s1 : 0;
                double acc = 0.0;
#pragma unroll
                for (int q = 0; q < 9; q++) {
                    if (q == 4) continue;
                    const int d0_ = q % 3 - 1, d1_ = q / 3 - 1;
                    const int gx = (m & 1) + (a0 == 0 ? d0_ : 0);
                    const int gy = ((m >> 1) & 1) + (a0 == 1 ? d0_ : a1 == 1 ? d1_ : 0);
                    const int gz = ((m >> 2) & 1) + (a1 == 2 ? d1_ : 0);
                    if (parent3(gx, gy, gz, sx, sy, sz)) acc += cf[q] * weight3(P, D, oc, gx, gy, gz, sx, sy, sz);
                }
                w[c] = D.inner(I + sx, J + sy, K + sz) ? -acc / d0 : 0.0;
            }
        }
#pragma unroll
        for (int c = 0; c < 4; c++) P[(long long)(kPBase(m) + c) * D.plc + oc] = w[c];
    }
}

// Cell centre (three odd coordinates): solve the full fine equation with the
// 26 neighbours interpolated by their own rows.
__global__ void k_interp_centre3d(Sten3<double> F, CoarseDims D, double* __restrict__ P, KState* st) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y, K = blockIdx.z;
    if (I >= D.nc) return;
    const long long oc = D.at(I, J, K);
    const int fi = 2 * I + 1, fj = 2 * J + 1, fk = 2 * K + 1;
    double w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (inner3(D.nf, fi, fj, fk)) {
        const double d0 = F.full(fi, fj, fk, 13);
        if (!(d0 > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
#pragma unroll
        for (int o = 0; o < 27; o++) {
            if (o == 13) continue;
            const double a = F.full(fi, fj, fk, o);
            const int gx = 1 + off_x(o), gy = 1 + off_y(o), gz = 1 + off_z(o);
#pragma unroll
            for (int s = 0; s < 8; s++)
                if (parent3(gx, gy, gz, s & 1, (s >> 1) & 1, s >> 2))
                    w[s] += a * weight3(P, D, oc, gx, gy, gz, s & 1, (s >> 1) & 1, s >> 2);
        }
#pragma unroll
        for (int s = 0; s < 8; s++) w[s] = D.inner(I + (s & 1), J + ((s >> 1) & 1), K + (s >> 2)) ? -w[s] / d0 : 0.0;
    }
#pragma unroll
    for (int s = 0; s < 8; s++) P[(long long)(kPBase(7) + s) * D.plc + oc] = w[s];
}

// Galerkin coarse operator: A_c(K, K+e) for the 14 stored offsets e, one
// thread per coarse node, as sum_f P(f, K) (A P)(f, K+e) over the fine points
// f = 2K + d, d in {-1,0,1}^3.  The eight f with three odd coordinates are left
// out: their interpolation solves their own fine equation, so (A P)(f, .) is
// zero there (to rounding).
//
// The in-plane offsets are unrolled; z is walked at run time over the (dz, oz)
// pairs whose neighbour plane 2K + dz + oz interpolates from coarse plane
// K + ez: three pairs for ez = -1 (nine in-plane e), seven for ez = 0 (the five
// stored ones).  About 1300 FP64 operations a coarse node from a loop body of
// a few hundred; unrolling all three directions took 950 operations but was
// ten times slower, its code outran the instruction caches (58% hits).
struct Rap3 {
    const double* A;      // fine operator at the fine point 2(I,J,K)
    long long pl;
    int ld;
    long long sz;         // fine plane of k
    const double* P;      // weights at the coarse node (I,J,K)
    long long plc;
    int ldc;
    long long szc;
};

// first weight plane of in-plane parity mask m and z parity pz, z parent bit b
__device__ __forceinline__ int wplane(int m, int pz, int b) {
    return pz ? kPBase(m | 4) + (b << ((m & 1) + (m >> 1))) : kPBase(m);
}

// One (dz, oz) pair: acc[t] += sum over (dx, dy) of P(f, K) times
// (A P)(f, K + e) restricted to the neighbours in plane dz + oz, for the
// in-plane offsets e = t (numbered as the nine-point stencil), t < NE.
template <int NE>
__device__ __forceinline__ void rap3_pair(const Rap3& R, int dz, int oz, int ez, double acc[NE]) {
    const int gz = dz + oz;                                 // in [-2, 1]
    const int qg = gz < 0 ? -1 : 0, qd = dz < 0 ? -1 : 0;   // owner planes of f + o and of f
    // weights of the neighbours: by in-plane parity mask
    const double* Pg[4];
#pragma unroll
    for (int m = 0; m < 4; m++) Pg[m] = R.P + wplane(m, gz & 1, ez - qg) * R.plc + qg * R.szc;
    const bool odd = gz & 1;
    const double* a_dir = R.A + (long long)(9 * (oz + 1)) * R.pl + dz * R.sz;                    // plane 9(oz+1) + o
    const double* a_mir = R.A + (long long)(26 - 9 * (oz + 1)) * R.pl + (dz + oz) * R.sz;        // plane 17 - 9 oz - o
#pragma unroll
    for (int f = 0; f < 9; f++) {
        const int dx = f % 3 - 1, dy = f / 3 - 1;
        if (dx != 0 && dy != 0 && dz != 0) continue;        // cell centres
        double T[NE];
#pragma unroll
        for (int t = 0; t < NE; t++) T[t] = 0.0;
#pragma unroll
        for (int o = 0; o < 9; o++) {
            const int ox = o % 3 - 1, oy = o / 3 - 1, gx = dx + ox, gy = dy + oy;
            const bool mir = oz > 0 || (oz == 0 && o > 4);
            const double a = mir ? a_mir[-(long long)o * R.pl + gx + (long long)gy * R.ld]
                                 : a_dir[(long long)o * R.pl + dx + (long long)dy * R.ld];
            const int m = (gx & 1) | ((gy & 1) << 1);
            const int qx = half_floor(gx), qy = half_floor(gy);
#pragma unroll
            for (int t = 0; t < NE; t++) {
                const int ex = t % 3 - 1, ey = t / 3 - 1;
                if (!parent1(gx, ex) || !parent1(gy, ey)) continue;
                const int c = compress3((ex - qx) | ((ey - qy) << 1), m);
                const double w = m || odd ? Pg[m][c * R.plc + qx + (long long)qy * R.ldc] : 1.0;
                T[t] += a * w;
            }
        }
        const int m = (dx & 1) | ((dy & 1) << 1), pz = dz & 1;
        double wK = 1.0;
        if (m || pz)
            wK = R.P[(wplane(m, pz, dz < 0) + compress3((dx < 0) | ((dy < 0) << 1), m)) * R.plc - (dx < 0) -
                     (dy < 0) * (long long)R.ldc + qd * R.szc];
#pragma unroll
        for (int t = 0; t < NE; t++) acc[t] += wK * T[t];
    }
}

// Four warps share 32 coarse nodes: the ten pairs go to four roles of about
// 380, 320, 350 and 290 operations, summed through shared memory.  On the
// small levels the chain of one thread's FP64 instructions is the kernel's
// time (64 cycles each: 73 us for the whole node), and a quarter of it is left;
// the roles rotate over the warps with the block so that the schedulers of an
// SM get equal shares.  129^3 hierarchy (six levels): 0.98 ms, 0.75 of it the
// finest; the kernel that looked every weight up at run time took 6.8 ms.
__global__ void __launch_bounds__(128, 3) k_rap3d(Sten3<double> F, CoarseDims D, const double* __restrict__ P,
                                                  double* __restrict__ Ac, KState* st) {
    __shared__ double part[2][9][32];
    const int lane = threadIdx.x, role = (threadIdx.y + blockIdx.y) & 3;
    const int I = blockIdx.x * 32 + lane;
    const int J = blockIdx.y, K = blockIdx.z;
    const bool in = D.inner(I, J, K);
    const long long oc = D.at(I, J, K);
    double lo[9], mid[5];
#pragma unroll
    for (int t = 0; t < 9; t++) lo[t] = 0.0;
#pragma unroll
    for (int t = 0; t < 5; t++) mid[t] = 0.0;
    if (in) {
        const Rap3 R{F.a + F.idx(2 * I, 2 * J, 2 * K), F.pl, F.ld, (long long)F.ld * F.n, P + oc, D.plc, D.ldc,
                     (long long)D.ldc * D.nc};
        // (dz, oz): ez = -1: (0,-1) | (-1,-1), (-1,0); ez = 0: (0,-1), (0,0), (0,1) | (-1,0), (-1,1), (1,-1), (1,0)
        if (role < 2) {
#pragma unroll 1
            for (int p = 0; p < 1 + role; p++) rap3_pair<9>(R, -role, role ? p - 1 : -1, -1, lo);
        } else {
#pragma unroll 1
            for (int p = 0; p < role + 1; p++)
                rap3_pair<5>(R, role == 2 ? 0 : p < 2 ? -1 : 1, role == 2 ? p - 1 : p < 2 ? p : p - 3, 0, mid);
        }
    }
    if (role == 1)
#pragma unroll
        for (int t = 0; t < 9; t++) part[0][t][lane] = lo[t];
    if (role == 3)
#pragma unroll
        for (int t = 0; t < 5; t++) part[1][t][lane] = mid[t];
    __syncthreads();
    if (I >= D.nc) return;
    // couplings to boundary coarse nodes are dropped
    if (role == 0) {
#pragma unroll
        for (int t = 0; t < 9; t++) {
            const bool keep = in && D.inner(I + t % 3 - 1, J + t / 3 - 1, K - 1);
            Ac[(long long)t * D.plc + oc] = keep ? lo[t] + part[0][t][lane] : 0.0;
        }
    } else if (role == 2) {
#pragma unroll
        for (int t = 0; t < 5; t++) {
            mid[t] += part[1][t][lane];
            const bool keep = in && D.inner(I + t % 3 - 1, J + t / 3 - 1, K);
            Ac[(long long)(9 + t) * D.plc + oc] = keep ? mid[t] : 0.0;
        }
        if (in && !(mid[4] > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
    }
}

__global__ void k_export_stencil3d(Sten3<double> F, double* __restrict__ out) {
    const int n = F.n;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y, k = blockIdx.z;
    if (i >= n) return;
    double* row = out + ((long long)i + (long long)n * (j + (long long)n * k)) * 27;
    const bool in = inner3(n, i, j, k);
    for (int o = 0; o < 27; o++) row[o] = in ? F.full(i, j, k, o) : 0.0;
}

__global__ void k_export_interp3d(const double* __restrict__ P, CoarseDims D, double* __restrict__ out) {
    const int nf = D.nf;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y, k = blockIdx.z;
    if (i >= nf) return;
    double* row = out + ((long long)i + (long long)nf * (j + (long long)nf * k)) * 8;
    for (int s = 0; s < 8; s++)
        row[s] = pweight3(P, D.ldc, D.nc, D.plc, nf, i, j, k, (i >> 1) + (s & 1), (j >> 1) + ((s >> 1) & 1),
                          (k >> 1) + (s >> 2));
}

// out_i = -sum over boundary nodes j of A_ij g_j at interior nodes i, as in 2-D.
__global__ void k_boundary_rhs3d(int n, const double* __restrict__ coords, const double* __restrict__ kappa,
                                 const double* __restrict__ g, double* __restrict__ out, KState* st) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y, k = blockIdx.z;
    if (i >= n) return;
    double acc = 0.0;
    if (inner3(n, i, j, k)) {
        bool ok = true;
        for (int cz = 0; cz < 2; cz++)
            for (int cy = 0; cy < 2; cy++)
                for (int cx = 0; cx < 2; cx++) {
                    const int ci = i - 1 + cx, cj = j - 1 + cy, ck = k - 1 + cz;
                    const int a = (1 - cx) + 2 * (1 - cy) + 4 * (1 - cz);
                    const double kap = kappa[(long long)ci + (long long)(n - 1) * (cj + (long long)(n - 1) * ck)];
                    double Kr[8];
                    ok &= element_row3d(coords, n, ci, cj, ck, Scalar3{kap}, a, Kr);
                    for (int b = 0; b < 8; b++) {
                        const int bi = ci + (b & 1), bj = cj + ((b >> 1) & 1), bk = ck + (b >> 2);
                        if (inner3(n, bi, bj, bk)) continue;
                        acc -= Kr[b] * g[(long long)bi + (long long)n * (bj + (long long)n * bk)];
                    }
                }
        if (!ok) set_err(st, BMG_ERR_MAP_FOLDED);
    }
    out[(long long)i + (long long)n * (j + (long long)n * k)] = acc;
}

// dL/dkappa_e = -lambda_e^T K_e^0 u_e = -sum_q 1/8 (adj^T grad lambda) .
// (adj^T grad u) / det: the two fields' gradients at the Gauss points instead
// of the element matrix, about 700 FP64 operations a cell (the eight matrix
// rows took 9000).  A cell whose lambda is zero is not checked for folding.
__global__ void k_adjoint_cells3d(int n, const double* __restrict__ coords, const double* __restrict__ u,
                                  const double* __restrict__ lam, double* __restrict__ g, KState* st) {
    const int ci = blockIdx.x * blockDim.x + threadIdx.x;
    const int cj = blockIdx.y, ck = blockIdx.z;
    if (ci >= n - 1) return;
    double ue[8], le[8];
    bool any = false;
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const int i = ci + (b & 1), j = cj + ((b >> 1) & 1), k = ck + (b >> 2);
        const long long id = (long long)i + (long long)n * (j + (long long)n * k);
        const bool in = inner3(n, i, j, k);
        ue[b] = in ? u[id] : 0.0;
        le[b] = in ? lam[id] : 0.0;
        any = any || !(le[b] == 0.0);
    }
    double s = 0.0;
    if (any) {
        CellMap3 M;
        EdgeMap3 U, L;
        M.load(coords, n, ci, cj, ck);
        U.set(ue);
        L.set(le);
        bool ok = true;
#pragma unroll 1
        for (int qz = 0; qz < 2; qz++) {
            const double z = qz ? kG1 : kG0;
#pragma unroll
            for (int qp = 0; qp < 4; qp++) {
                double adj[3][3], a[3], b[3];
                const double det = M.adjugate(qp & 1, qp >> 1, z, adj);
                if (!(det > 0.0)) ok = false;
                U.at(qp & 1, qp >> 1, z, a[0], a[1], a[2]);
                L.at(qp & 1, qp >> 1, z, b[0], b[1], b[2]);
                double t = 0.0;
#pragma unroll
                for (int r = 0; r < 3; r++)
                    t += (adj[0][r] * a[0] + adj[1][r] * a[1] + adj[2][r] * a[2]) *
                         (adj[0][r] * b[0] + adj[1][r] * b[1] + adj[2][r] * b[2]);
                s += t * (0.125 / det);
            }
        }
        if (!ok) set_err(st, BMG_ERR_MAP_FOLDED);
    }
    g[(long long)ci + (long long)(n - 1) * (cj + (long long)(n - 1) * ck)] = -s;
}

inline dim3 grid3(int ni, int nj, int nk) { return dim3(cdiv(ni, 64), nj, nk); }

}  // namespace

bmg_status assemble3d(Ctx& c, const double* coords, const double* kappa) {
    Level& L = c.lev[0];
    BMG_TRY(launch_assemble3d<false>(L.n, L.ld, L.plane, coords, kappa, L.A64, c.st, c.stream));
    c.launches++;
    return BMG_OK;
}

// As assemble_export2d: assembly into caller-given half planes, then export.
bmg_status assemble_export3d(int n, int ld, long long pl, const double* coords, const double* kappa, double* A,
                             KState* st, double* out, cudaStream_t s) {
    BMG_TRY(launch_assemble3d<false>(n, ld, pl, coords, kappa, A, st, s));
    k_export_stencil3d<<<grid3(n, n, n), 64, 0, s>>>(Sten3<double>{A, n, ld, pl}, out);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status assemble_tensor3d(Ctx& c, const double* coords, const double* D) {
    Level& L = c.lev[0];
    BMG_TRY(launch_assemble3d<true>(L.n, L.ld, L.plane, coords, D, L.A64, c.st, c.stream));
    c.launches++;
    return BMG_OK;
}

bmg_status boundary_rhs3d(Ctx& c, const double* coords, const double* kappa, const double* g, double* out) {
    const int n = c.lev[0].n;
    k_boundary_rhs3d<<<grid3(n, n, n), 64, 0, c.stream>>>(n, coords, kappa, g, out, c.st);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status set_stencil3d(Ctx& c, const double* full) {
    Level& L = c.lev[0];
    k_set_stencil3d<<<grid3(L.n, L.n, L.n), 64, 0, c.stream>>>(L.n, L.ld, L.plane, full, L.A64);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status setup_level3d(Ctx& c, int l) {
    Level& F = c.lev[l];
    Level& K = c.lev[l + 1];
    Sten3<double> fs{F.A64, F.n, F.ld, F.plane};
    CoarseDims D{F.n, K.n, K.ld, K.plane};
    const dim3 g = grid3(K.n, K.n, K.n);
    k_interp_lines3d<<<g, 64, 0, c.stream>>>(fs, D, F.P64, c.st);
    k_interp_planes3d<<<g, 64, 0, c.stream>>>(fs, D, F.P64, c.st);
    k_interp_centre3d<<<g, 64, 0, c.stream>>>(fs, D, F.P64, c.st);
    k_rap3d<<<dim3(cdiv(K.n, 32), K.n, K.n), dim3(32, 4), 0, c.stream>>>(fs, D, F.P64, K.A64, c.st);
    c.launches += 4;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status export_stencil3d(Ctx& c, int l, double* out) {
    Level& L = c.lev[l];
    k_export_stencil3d<<<grid3(L.n, L.n, L.n), 64, 0, c.stream>>>(Sten3<double>{L.A64, L.n, L.ld, L.plane}, out);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status export_interp3d(Ctx& c, int l, double* out) {
    Level& F = c.lev[l];
    Level& K = c.lev[l + 1];
    k_export_interp3d<<<grid3(F.n, F.n, F.n), 64, 0, c.stream>>>(F.P64, CoarseDims{F.n, K.n, K.ld, K.plane}, out);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status adjoint_cells3d(Ctx& c, const double* coords, const double* u, const double* lam, double* g) {
    const int n = c.lev[0].n;
    k_adjoint_cells3d<<<grid3(n - 1, n - 1, n - 1), 64, 0, c.stream>>>(n, coords, u, lam, g, c.st);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

}  // namespace bmg
