// setup2d.cu -- 2-D setup kernels: Q1 assembly from the map (Sec. 2.1),
// operator-induced interpolation and Galerkin coarse operators (Sec. 2.2),
// exports for diagnostics, and the per-cell adjoint contraction.
#include "common.cuh"

namespace bmg {
namespace {

// 2-point Gauss nodes on [0,1]: 1/2 -+ 1/(2 sqrt 3)
constexpr double kG0 = 0.21132486540518711775;
constexpr double kG1 = 0.78867513459481288225;

// Coefficient of a cell, as the metric it induces from adj(J) = det J J^-1.
// Scalar kappa: G = (kappa / det J) adj adj^T.  SPD tensor D (Sec. 2, Eq.
// pde): G = (1 / det J) adj D adj^T, i.e. det J J^-1 D J^-T (Sec. 2.1).
struct Scalar2 {
    double kap;
    __device__ __forceinline__ void metric(double J11, double J12, double J21, double J22, double det, double& G11,
                                           double& G12, double& G22) const {
        const double s = 0.25 * kap / det;
        G11 = s * (J22 * J22 + J12 * J12);
        G12 = -s * (J22 * J21 + J12 * J11);
        G22 = s * (J21 * J21 + J11 * J11);
    }
};
struct Tensor2 {
    double d11, d12, d22;
    __device__ __forceinline__ void metric(double J11, double J12, double J21, double J22, double det, double& G11,
                                           double& G12, double& G22) const {
        const double a11 = J22, a12 = -J12, a21 = -J21, a22 = J11;   // adj(J)
        const double t11 = a11 * d11 + a12 * d12, t12 = a11 * d12 + a12 * d22;
        const double t21 = a21 * d11 + a22 * d12, t22 = a21 * d12 + a22 * d22;
        const double s = 0.25 / det;
        G11 = s * (t11 * a11 + t12 * a12);
        G12 = s * (t11 * a21 + t12 * a22);
        G22 = s * (t21 * a21 + t22 * a22);
    }
};

// Reference-cell derivatives of a bilinear field given at a cell's corners:
// d/dxi is linear in eta and d/deta linear in xi, so each takes two values at
// the Gauss points (10 FP64 operations, against 32 for a sum over the four
// corners at every point).
struct EdgeMap2 {
    double u[2];   // d/dxi at eta_q
    double v[2];   // d/deta at xi_q
    __device__ __forceinline__ void set(const double x[4]) {
        const double e0 = x[1] - x[0], e1 = x[3] - x[2], f0 = x[2] - x[0], f1 = x[3] - x[1];
        const double de = e1 - e0, df = f1 - f0;
        u[0] = e0 + kG0 * de;
        u[1] = e0 + kG1 * de;
        v[0] = f0 + kG0 * df;
        v[1] = f0 + kG1 * df;
    }
};

struct CellMap2 {
    EdgeMap2 x, y;
    __device__ __forceinline__ void load(const double* __restrict__ X, const double* __restrict__ Y, int n, int ci,
                                         int cj) {
        const long long id = (long long)cj * n + ci;
        const double xa[4] = {X[id], X[id + 1], X[id + n], X[id + n + 1]};
        const double ya[4] = {Y[id], Y[id + 1], Y[id + n], Y[id + n + 1]};
        x.set(xa);
        y.set(ya);
    }
};

// Q1 element matrix of a cell: K_ab = sum_q 1/4 grad(phi_a)^T G grad(phi_b), G
// from the cell's coefficient (above), J = dx/dxi (isoparametric map).  Corner
// a = ax + 2 ay; the symmetric half a <= b in the order of sym4.  Sum
// factorisation over the 2x2 Gauss points: the shape functions are products of
// 1 - t, t per direction, so with s = -1, +1 for corner bit 0, 1
//   K_ab = sx sx' M11[ay+by] + sy sy' M22[ax+bx] + sx sy' N[ay][bx] + sx' sy N[by][ax],
// about 160 FP64 operations in all (the direct sum takes about 600).
// Returns false if det J <= 0.
__host__ __device__ constexpr int sym4(int a, int b) {   // a <= b
    return a * 4 - a * (a - 1) / 2 + (b - a);
}

// Contractions of two Gauss-point values with (1-t)^2, t(1-t), t^2 as sum and
// difference: (1-t)^2 and t^2 at the two points are 1/3 +- 1/(2 sqrt 3).  Where
// the metric is constant the difference vanishes and the entries keep the
// exact ratios 2 : 1 : 2, so an element's row sums, which every coarser level
// amplifies, come out as exact zeros.
constexpr double kThird = 1.0 / 3.0, kSixth = 1.0 / 6.0, kHalfGap = 0.5 * (kG1 - kG0);
__device__ __forceinline__ void pair3(double s0, double s1, double out[3]) {
    const double S = s0 + s1, D = s0 - s1, t = kThird * S;
    out[0] = t + kHalfGap * D;
    out[1] = kSixth * S;
    out[2] = t - kHalfGap * D;
}

template <class C>
__device__ __forceinline__ bool element2d(const CellMap2& M, const C& coef, double K[10]) {
    bool ok = true;
    double s11[2], g11[2][2], s22[2], g22[2][2], g12[2][2];   // [q: xi][p: eta]
#pragma unroll
    for (int p = 0; p < 2; p++)
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const double J11 = M.x.u[p], J12 = M.x.v[q], J21 = M.y.u[p], J22 = M.y.v[q];
            const double det = J11 * J22 - J12 * J21;
            if (!(det > 0.0)) ok = false;
            coef.metric(J11, J12, J21, J22, det, g11[q][p], g12[q][p], g22[q][p]);
        }
#pragma unroll
    for (int t = 0; t < 2; t++) {
        s11[t] = g11[0][t] + g11[1][t];
        s22[t] = g22[t][0] + g22[t][1];
    }
    double M11[3], M22[3];
    pair3(s11[0], s11[1], M11);
    pair3(s22[0], s22[1], M22);
    double N[2][2];
#pragma unroll
    for (int b = 0; b < 2; b++) {
        const double wa = b ? kG0 : kG1, wb = b ? kG1 : kG0;   // the xi factor of corner bit b at xi_0, xi_1
        const double n0 = wa * g12[0][0] + wb * g12[1][0], n1 = wa * g12[0][1] + wb * g12[1][1];
        N[0][b] = kG1 * n0 + kG0 * n1;
        N[1][b] = kG0 * n0 + kG1 * n1;
    }
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = a; b < 4; b++) {
            const int ax = a & 1, ay = a >> 1, bx = b & 1, by = b >> 1;
            const double m1 = M11[ay + by], m2 = M22[ax + bx], c1 = N[ay][bx], c2 = N[by][ax];
            double v = ax == bx ? m1 : -m1;
            v = ay == by ? v + m2 : v - m2;
            v = ax == by ? v + c1 : v - c1;
            v = bx == ay ? v + c2 : v - c2;
            K[sym4(a, b)] = v;
        }
    return ok;
}

// coefficient of cell e: kappa[e], or the tensor planes D11, D12, D22 (ne cells each)
template <bool TENSOR>
__device__ __forceinline__ auto cell_coef2(const double* __restrict__ c, long long ne, long long e) {
    if constexpr (TENSOR)
        return Tensor2{c[e], c[ne + e], c[2 * ne + e]};
    else
        return Scalar2{c[e]};
}

// Gather assembly (no atomics).  A CTA owns a strip of kAsmN node columns and
// a band of H node rows and marches up one row of cells at a time: each of
// its kAsmC threads forms one cell's matrix into shared memory, then the node
// threads add the row's entries to the node row below it, which that
// completes, and start the row above.  Couplings to boundary nodes are
// dropped; boundary rows are zero.  FP64 arithmetic bounds the kernel (two
// FMA per SM and clock), so the redundant cells count (one column in kAsmC,
// one row per band) and the 64 bytes per node do not.  Narrow strips keep
// the bands tall enough on small grids to give every SM work.
constexpr int kAsmC = 64, kAsmN = kAsmC - 1;

template <bool TENSOR>
__global__ void __launch_bounds__(kAsmC) k_assemble2d(int n, int ld, long long pl, int H,
                                                      const double* __restrict__ coords,
                                                      const double* __restrict__ kappa, double* __restrict__ A,
                                                      KState* st) {
    __shared__ double sK[10][kAsmC];
    const long long ne = (long long)(n - 1) * (n - 1);
    const int t = threadIdx.x;
    const int i0 = blockIdx.x * kAsmN;
    const int j0 = blockIdx.y * H, j1 = min(j0 + H, n);             // node rows [j0, j1)
    const int ci = i0 - 1 + t;                                      // cell column between nodes ci, ci + 1
    const int i = i0 + t;                                           // node column; its cells are slots t, t + 1
    const bool node = t < kAsmN && i < n;
    const bool in1 = node && i >= 1 && i <= n - 2;
    double C = 0, W = 0;                                            // of the row in progress
    for (int cj = j0 - 1; cj < j1; cj++) {
        if (cj >= 0 && cj <= n - 2 && ci >= 0 && ci <= n - 2) {
            CellMap2 M;
            M.load(coords, coords + (long long)n * n, n, ci, cj);
            double K[10];
            if (!element2d(M, cell_coef2<TENSOR>(kappa, ne, (long long)cj * (n - 1) + ci), K))
                set_err(st, BMG_ERR_MAP_FOLDED);
#pragma unroll
            for (int q = 0; q < 10; q++) sK[q][t] = K[q];
        }
        __syncthreads();
        if (cj >= j0 && node) {   // row cj: the cells above it, (i-1, cj) and (i, cj)
            const bool in = in1 && cj >= 1 && cj <= n - 2;
            const long long o = (long long)cj * ld + i;
            double NW = 0;
            if (in) {
                C += sK[sym4(1, 1)][t];
                if (i >= 2) {
                    W += sK[sym4(0, 1)][t];
                    if (cj + 1 <= n - 2) NW = sK[sym4(1, 2)][t];
                }
                C += sK[sym4(0, 0)][t + 1];
            }
            A[C2 * pl + o] = in ? C : 0.0;
            A[W2 * pl + o] = in ? W : 0.0;
            A[NW2 * pl + o] = NW;
        }
        if (cj + 1 < j1 && node) {   // row cj + 1: the cells below it, (i-1, cj) and (i, cj)
            const int j = cj + 1;
            const bool in = in1 && j >= 1 && j <= n - 2;
            const long long o = (long long)j * ld + i;
            double S = 0, SW = 0;
            C = W = 0;
            if (in) {
                C = sK[sym4(3, 3)][t];
                if (i >= 2) W = sK[sym4(2, 3)][t];
                if (j >= 2) {
                    S = sK[sym4(1, 3)][t];
                    if (i >= 2) SW = sK[sym4(0, 3)][t];
                }
                C += sK[sym4(2, 2)][t + 1];
                if (j >= 2) S += sK[sym4(0, 2)][t + 1];
            }
            A[S2 * pl + o] = S;
            A[SW2 * pl + o] = SW;
        }
        __syncthreads();
    }
}

// Launches k_assemble2d; rows per band: the ones that minimise (warps per
// scheduler) x (rows + 1 pre-roll row).  One warp's FP64 instruction holds its
// scheduler's unit for 64 cycles, so a row of cells costs each warp the same
// few microseconds whether or not the other schedulers have work.
template <bool TENSOR>
bmg_status launch_assemble2d(int n, int ld, long long pl, const double* coords, const double* coef, double* A,
                             KState* st, cudaStream_t s) {
    int dev = 0, sms = 0;
    BMG_CUDA(cudaGetDevice(&dev));
    BMG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int tx = cdiv(n, kAsmN);
    int H = 1;
    long long best = -1;
    for (int h = 1; h <= 64 && h <= n; h++) {
        const long long cost = (long long)cdiv(tx * cdiv(n, h) * (kAsmC / 32), 4 * sms) * (h + 1);
        if (best < 0 || cost < best) {
            best = cost;
            H = h;
        }
    }
    k_assemble2d<TENSOR><<<dim3(tx, cdiv(n, H)), kAsmC, 0, s>>>(n, ld, pl, H, coords, coef, A, st);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

// Full 9-entry rows -> symmetric half planes; couplings to boundary nodes
// and boundary rows are forced to zero.
__global__ void k_set_stencil2d(int n, int ld, long long pl, const double* __restrict__ full,
                                double* __restrict__ A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n) return;
    const long long o = (long long)j * ld + i;
    double C = 0, W = 0, S = 0, SW = 0, NW = 0;
    if (i >= 1 && j >= 1 && i <= n - 2 && j <= n - 2) {
        const double* row = full + ((long long)j * n + i) * 9;
        C = row[4];
        W = i > 1 ? row[3] : 0.0;
        S = j > 1 ? row[1] : 0.0;
        SW = (i > 1 && j > 1) ? row[0] : 0.0;
        NW = (i > 1 && j < n - 2) ? row[6] : 0.0;
    }
    A[C2 * pl + o] = C;
    A[W2 * pl + o] = W;
    A[S2 * pl + o] = S;
    A[SW2 * pl + o] = SW;
    A[NW2 * pl + o] = NW;
}

// Edge points of the fine grid, owned by coarse node (I,J):
//   (2I+1, 2J): collapse the stencil over dy -> weights -A_L/A_0, -A_R/A_0
//   (2I, 2J+1): collapse over dx               -> weights -A_S/A_0, -A_N/A_0
// Where the collapsed denominator A_0 is not positive the point uses its own
// couplings along the line instead (A_0 = a_00 > 0 for an SPD operator).
// Weights to boundary coarse nodes and rows of boundary fine points are 0.
__global__ void k_interp_edges2d(Sten2<double> F, int nf, int nc, int ldc, long long plc,
                                 double* __restrict__ P, KState* st) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y;
    if (I >= nc) return;
    const long long o = (long long)J * ldc + I;
    double xl = 0, xr = 0, ys = 0, yn = 0;
    {   // x-edge point
        const int i = 2 * I + 1, j = 2 * J;
        if (i <= nf - 2 && j >= 1 && j <= nf - 2) {
            double AL = F.full(i, j, -1, -1) + F.full(i, j, -1, 0) + F.full(i, j, -1, 1);
            double A0 = F.full(i, j, 0, -1) + F.full(i, j, 0, 0) + F.full(i, j, 0, 1);
            double AR = F.full(i, j, 1, -1) + F.full(i, j, 1, 0) + F.full(i, j, 1, 1);
            if (!(A0 > 0.0)) {
                AL = F.full(i, j, -1, 0);
                AR = F.full(i, j, 1, 0);
                A0 = F.c(i, j);
            }
            if (!(A0 > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
            xl = (I >= 1) ? -AL / A0 : 0.0;
            xr = (I + 1 <= nc - 2) ? -AR / A0 : 0.0;
        }
    }
    {   // y-edge point
        const int i = 2 * I, j = 2 * J + 1;
        if (i >= 1 && i <= nf - 2 && j <= nf - 2) {
            double AS = F.full(i, j, -1, -1) + F.full(i, j, 0, -1) + F.full(i, j, 1, -1);
            double A0 = F.full(i, j, -1, 0) + F.full(i, j, 0, 0) + F.full(i, j, 1, 0);
            double AN = F.full(i, j, -1, 1) + F.full(i, j, 0, 1) + F.full(i, j, 1, 1);
            if (!(A0 > 0.0)) {
                AS = F.full(i, j, 0, -1);
                AN = F.full(i, j, 0, 1);
                A0 = F.c(i, j);
            }
            if (!(A0 > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
            ys = (J >= 1) ? -AS / A0 : 0.0;
            yn = (J + 1 <= nc - 2) ? -AN / A0 : 0.0;
        }
    }
    P[PXL * plc + o] = xl;
    P[PXR * plc + o] = xr;
    P[PYS * plc + o] = ys;
    P[PYN * plc + o] = yn;
}

// Interior point (2I+1, 2J+1): solve the fine equation with its four C
// neighbours (coarse values) and four edge neighbours (their edge
// interpolation):  v = -(1/a00) sum_{d != 0} a_d v(i+d).
__global__ void k_interp_interior2d(Sten2<double> F, int nf, int nc, int ldc, long long plc,
                                    double* __restrict__ P, KState* st) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y;
    if (I >= nc) return;
    const long long o = (long long)J * ldc + I;
    double sw = 0, se = 0, nw = 0, ne = 0;
    const int i = 2 * I + 1, j = 2 * J + 1;
    if (i <= nf - 2 && j <= nf - 2) {
        const double a00 = F.c(i, j);
        if (!(a00 > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
        auto Pv = [&](int p, int II, int JJ) { return P[p * plc + (long long)JJ * ldc + II]; };
        // edge neighbours: south (i,j-1) = x-edge of (I,J); north (i,j+1) = x-edge of (I,J+1);
        //                  west (i-1,j) = y-edge of (I,J);  east (i+1,j) = y-edge of (I+1,J)
        const double aS = F.full(i, j, 0, -1), aN = F.full(i, j, 0, 1);
        const double aW = F.full(i, j, -1, 0), aE = F.full(i, j, 1, 0);
        const double sxl = Pv(PXL, I, J), sxr = Pv(PXR, I, J);
        const double nxl = Pv(PXL, I, J + 1), nxr = Pv(PXR, I, J + 1);
        const double wys = Pv(PYS, I, J), wyn = Pv(PYN, I, J);
        const double eys = Pv(PYS, I + 1, J), eyn = Pv(PYN, I + 1, J);
        const double inv = -1.0 / a00;
        sw = (F.full(i, j, -1, -1) + aS * sxl + aW * wys) * inv;
        se = (F.full(i, j, 1, -1) + aS * sxr + aE * eys) * inv;
        nw = (F.full(i, j, -1, 1) + aN * nxl + aW * wyn) * inv;
        ne = (F.full(i, j, 1, 1) + aN * nxr + aE * eyn) * inv;
        if (I < 1 || J < 1) sw = 0.0;
        if (I + 1 > nc - 2 || J < 1) se = 0.0;
        if (I < 1 || J + 1 > nc - 2) nw = 0.0;
        if (I + 1 > nc - 2 || J + 1 > nc - 2) ne = 0.0;
    }
    P[PSW * plc + o] = sw;
    P[PSE * plc + o] = se;
    P[PNW * plc + o] = nw;
    P[PNE * plc + o] = ne;
}

// Weight of fine node (fi,fj) to coarse node (KI,KJ).
__device__ __forceinline__ double pweight2(const double* __restrict__ P, int ldc, long long plc, int nf,
                                           int fi, int fj, int KI, int KJ) {
    if (fi < 1 || fj < 1 || fi > nf - 2 || fj > nf - 2) return 0.0;
    const int oi = fi & 1, oj = fj & 1, I = fi >> 1, J = fj >> 1;
    const int dI = KI - I, dJ = KJ - J;
    if (dI < 0 || dJ < 0 || dI > oi || dJ > oj) return 0.0;
    const long long o = (long long)J * ldc + I;
    if (!oi && !oj) return 1.0;
    if (oi && !oj) return P[(dI ? PXR : PXL) * plc + o];
    if (!oi && oj) return P[(dJ ? PYN : PYS) * plc + o];
    const int p = dJ ? (dI ? PNE : PNW) : (dI ? PSE : PSW);
    return P[p * plc + o];
}

// Weight of the fine point at offset (gx, gy) in [-2, 2]^2 from the fine point
// 2(I,J) to the coarse node (I+ex, J+ey); all offsets are compile-time constants
// at the call, so this is one load at a fixed offset from oc = (I,J).
__host__ __device__ constexpr int half_floor(int g) { return g >= 0 ? g / 2 : -((1 - g) / 2); }
__host__ __device__ constexpr bool parent1(int g, int e) {
    return e - half_floor(g) >= 0 && e - half_floor(g) <= (g & 1);
}
__device__ __forceinline__ double weight2(const double* __restrict__ P, int ldc, long long plc, long long oc, int gx,
                                          int gy, int ex, int ey) {
    const int qx = half_floor(gx), qy = half_floor(gy), dI = ex - qx, dJ = ey - qy;
    if (!(gx & 1) && !(gy & 1)) return 1.0;
    const int p = !(gy & 1) ? (dI ? PXR : PXL) : !(gx & 1) ? (dJ ? PYN : PYS) : dJ ? (dI ? PNE : PNW) : (dI ? PSE : PSW);
    return P[(long long)p * plc + oc + qx + (long long)ldc * qy];
}

// Galerkin coarse operator A_c = P^T A P, one thread per coarse node: the five
// stored entries A_c(K, K+e) = sum_f P(f,K) (A P)(f, K+e) over the fine points
// f = 2K + d, d in {-1,0,1}^2.  The four f with both coordinates odd are left
// out: their interpolation solves their own fine equation, so (A P)(f, .) is
// zero there (to rounding).  The offsets are constants, so the loops unroll to
// plain loads and about 120 FP64 operations a coarse node.
__global__ void k_rap2d(Sten2<double> F, int nf, const double* __restrict__ P, int nc, int ldc,
                        long long plc, double* __restrict__ Ac, KState* st) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y;
    if (I >= nc) return;
    const long long o = (long long)J * ldc + I;
    double out[NS2] = {0, 0, 0, 0, 0};
    if (I >= 1 && J >= 1 && I <= nc - 2 && J <= nc - 2) {
        constexpr int tdx[NS2] = {0, -1, 0, -1, -1};
        constexpr int tdy[NS2] = {0, 0, -1, -1, 1};
#pragma unroll
        for (int f = 0; f < 9; f++) {
            const int fx = f % 3 - 1, fy = f / 3 - 1;
            if (fx != 0 && fy != 0) continue;
            const double wK = weight2(P, ldc, plc, o, fx, fy, 0, 0);
#pragma unroll
            for (int e = 0; e < 9; e++) {
                const int dx = e % 3 - 1, dy = e / 3 - 1;
                const double a = wK * F.full(2 * I + fx, 2 * J + fy, dx, dy);
#pragma unroll
                for (int t = 0; t < NS2; t++) {
                    const int ex = t == 0 || t == 2 ? 0 : -1, ey = t == 2 || t == 3 ? -1 : t == 4 ? 1 : 0;
                    if (parent1(fx + dx, ex) && parent1(fy + dy, ey))
                        out[t] += a * weight2(P, ldc, plc, o, fx + dx, fy + dy, ex, ey);
                }
            }
        }
        // couplings to boundary coarse nodes are dropped
#pragma unroll
        for (int t = 1; t < NS2; t++) {
            const int LI = I + tdx[t], LJ = J + tdy[t];
            if (LI < 1 || LJ < 1 || LI > nc - 2 || LJ > nc - 2) out[t] = 0.0;
        }
        if (!(out[0] > 0.0)) set_err(st, BMG_ERR_SETUP_BREAKDOWN);
    }
#pragma unroll
    for (int t = 0; t < NS2; t++) Ac[t * plc + o] = out[t];
}

__global__ void k_export_stencil2d(Sten2<double> F, int n, double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n) return;
    double* row = out + ((long long)j * n + i) * 9;
    const bool in = i >= 1 && j >= 1 && i <= n - 2 && j <= n - 2;
    for (int o = 0; o < 9; o++) row[o] = in ? F.full(i, j, o % 3 - 1, o / 3 - 1) : 0.0;
}

__global__ void k_export_interp2d(const double* __restrict__ P, int nf, int ldc, long long plc,
                                  double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= nf) return;
    double* row = out + ((long long)j * nf + i) * 4;
    for (int s = 0; s < 4; s++)
        row[s] = pweight2(P, ldc, plc, nf, i, j, (i >> 1) + (s & 1), (j >> 1) + (s >> 1));
}

// out_i = -sum over boundary nodes j of A_ij g_j at interior nodes i (the
// couplings the assembly drops, applied to Dirichlet data g; Sec. 2, the
// lift term of Eq. weak_computational); g and out in the caller's n^2
// layout, out zero on the boundary.
__global__ void k_boundary_rhs2d(int n, const double* __restrict__ coords, const double* __restrict__ kappa,
                                 const double* __restrict__ g, double* __restrict__ out, KState* st) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n) return;
    double acc = 0.0;
    if (i >= 1 && j >= 1 && i <= n - 2 && j <= n - 2) {
        const double* X = coords;
        const double* Y = coords + (long long)n * n;
        bool ok = true;
#pragma unroll
        for (int cy = 0; cy < 2; cy++)
#pragma unroll
            for (int cx = 0; cx < 2; cx++) {
                const int ci = i - 1 + cx, cj = j - 1 + cy;
                const int a = (1 - cx) + 2 * (1 - cy);      // the node's corner in the cell
                CellMap2 M;
                M.load(X, Y, n, ci, cj);
                double K[10];
                ok &= element2d(M, Scalar2{kappa[(long long)cj * (n - 1) + ci]}, K);
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    const int bi = ci + (b & 1), bj = cj + (b >> 1);
                    if (bi >= 1 && bj >= 1 && bi <= n - 2 && bj <= n - 2) continue;
                    acc -= K[a < b ? sym4(a, b) : sym4(b, a)] * g[(long long)bj * n + bi];
                }
            }
        if (!ok) set_err(st, BMG_ERR_MAP_FOLDED);
    }
    out[(long long)j * n + i] = acc;
}

// dL/dkappa_e = -lambda_e^T K_e^0 u_e (u, lambda in the caller's n^2 layout) =
// -sum_q 1/4 (adj^T grad lambda) . (adj^T grad u) / det: the two fields'
// gradients at the Gauss points instead of the element matrix, about 130 FP64
// operations a cell.
__global__ void k_adjoint_cells2d(int n, const double* __restrict__ coords, const double* __restrict__ u,
                                  const double* __restrict__ lam, double* __restrict__ g, KState* st) {
    const int ci = blockIdx.x * blockDim.x + threadIdx.x;
    const int cj = blockIdx.y;
    if (ci >= n - 1) return;
    double ue[4], le[4];
#pragma unroll
    for (int a = 0; a < 4; a++) {
        const int i = ci + (a & 1), j = cj + (a >> 1);
        const bool in = i >= 1 && j >= 1 && i <= n - 2 && j <= n - 2;
        const long long id = (long long)j * n + i;
        ue[a] = in ? u[id] : 0.0;
        le[a] = in ? lam[id] : 0.0;
    }
    CellMap2 M;
    EdgeMap2 U, L;
    M.load(coords, coords + (long long)n * n, n, ci, cj);
    U.set(ue);
    L.set(le);
    bool ok = true;
    double s = 0.0;
#pragma unroll
    for (int p = 0; p < 2; p++)
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const double J11 = M.x.u[p], J12 = M.x.v[q], J21 = M.y.u[p], J22 = M.y.v[q];
            const double det = J11 * J22 - J12 * J21;
            if (!(det > 0.0)) ok = false;
            const double ux = J22 * U.u[p] - J21 * U.v[q], uy = J11 * U.v[q] - J12 * U.u[p];
            const double lx = J22 * L.u[p] - J21 * L.v[q], ly = J11 * L.v[q] - J12 * L.u[p];
            s += (ux * lx + uy * ly) * (0.25 / det);
        }
    if (!ok) set_err(st, BMG_ERR_MAP_FOLDED);
    g[(long long)cj * (n - 1) + ci] = -s;
}

inline dim3 grid_rows(int ni, int nj) { return dim3(cdiv(ni, 128), nj); }

}  // namespace

bmg_status assemble2d(Ctx& c, const double* coords, const double* kappa) {
    Level& L = c.lev[0];
    BMG_TRY(launch_assemble2d<false>(L.n, L.ld, L.plane, coords, kappa, L.A64, c.st, c.stream));
    c.launches++;
    return BMG_OK;
}

// The two kernels of bmg_assemble and bmg_get_stencil(0) on caller-given
// storage: half planes A (row length ld, plane stride pl) and error word st.
bmg_status assemble_export2d(int n, int ld, long long pl, const double* coords, const double* kappa, double* A,
                             KState* st, double* out, cudaStream_t s) {
    BMG_TRY(launch_assemble2d<false>(n, ld, pl, coords, kappa, A, st, s));
    k_export_stencil2d<<<grid_rows(n, n), 128, 0, s>>>(Sten2<double>{A, ld, pl}, n, out);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status assemble_tensor2d(Ctx& c, const double* coords, const double* D) {
    Level& L = c.lev[0];
    BMG_TRY(launch_assemble2d<true>(L.n, L.ld, L.plane, coords, D, L.A64, c.st, c.stream));
    c.launches++;
    return BMG_OK;
}

bmg_status boundary_rhs2d(Ctx& c, const double* coords, const double* kappa, const double* g, double* out) {
    const int n = c.lev[0].n;
    k_boundary_rhs2d<<<grid_rows(n, n), 128, 0, c.stream>>>(n, coords, kappa, g, out, c.st);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status set_stencil2d(Ctx& c, const double* full) {
    Level& L = c.lev[0];
    k_set_stencil2d<<<grid_rows(L.n, L.n), 128, 0, c.stream>>>(L.n, L.ld, L.plane, full, L.A64);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status setup_level2d(Ctx& c, int l) {
    Level& F = c.lev[l];
    Level& K = c.lev[l + 1];
    Sten2<double> fs{F.A64, F.ld, F.plane};
    k_interp_edges2d<<<grid_rows(K.n, K.n), 128, 0, c.stream>>>(fs, F.n, K.n, K.ld, K.plane, F.P64, c.st);
    k_interp_interior2d<<<grid_rows(K.n, K.n), 128, 0, c.stream>>>(fs, F.n, K.n, K.ld, K.plane, F.P64, c.st);
    k_rap2d<<<grid_rows(K.n, K.n), 128, 0, c.stream>>>(fs, F.n, F.P64, K.n, K.ld, K.plane, K.A64, c.st);
    c.launches += 3;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status export_stencil2d(Ctx& c, int l, double* out) {
    Level& L = c.lev[l];
    k_export_stencil2d<<<grid_rows(L.n, L.n), 128, 0, c.stream>>>(Sten2<double>{L.A64, L.ld, L.plane}, L.n, out);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status export_interp2d(Ctx& c, int l, double* out) {
    Level& F = c.lev[l];
    Level& K = c.lev[l + 1];
    k_export_interp2d<<<grid_rows(F.n, F.n), 128, 0, c.stream>>>(F.P64, F.n, K.ld, K.plane, out);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status adjoint_cells2d(Ctx& c, const double* coords, const double* u, const double* lam, double* g) {
    const int n = c.lev[0].n;
    k_adjoint_cells2d<<<grid_rows(n - 1, n - 1), 128, 0, c.stream>>>(n, coords, u, lam, g, c.st);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

}  // namespace bmg
