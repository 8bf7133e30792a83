// krylov.cu -- vector kernels of the preconditioned conjugate-gradient outer
// loop (FP64) and of the FP32 inner CG of the refinement mode: operator
// application fused with its dot product, fused x/r updates with ||r||^2,
// r.z / r.z_old with the CG coefficient, p update, layout packing.  2-D
// (9-point) and 3-D (27-point) rows.  All reductions are deterministic:
// per-block partials summed in a fixed order by the last block (grid_sum);
// scalars stay on the device in KState.
#include "common.cuh"

namespace bmg {
namespace {

// Rows of the padded layout: r in [0, n^(DIM-1)), columns i in [0, ld).
template <int DIM>
struct RowGrid {
    int n, ld;
    __device__ __forceinline__ int rows() const { return DIM == 2 ? n : n * n; }
    __device__ __forceinline__ bool row_inner(int r) const {
        if (DIM == 2) return r >= 1 && r <= n - 2;
        const int j = r % n, k = r / n;
        return j >= 1 && j <= n - 2 && k >= 1 && k <= n - 2;
    }
};

// neighbour offset of stored plane t (t < 13) in 3-D
__device__ __forceinline__ long long d3(int t, int ld, int n) {
    return (long long)(t % 3 - 1) + (long long)ld * (((t / 3) % 3 - 1) + (long long)n * (t / 9 - 1));
}

// sum_j a_ij x_j of row o (2-D, symmetric-half storage)
__device__ __forceinline__ double apply_row(const double* __restrict__ A, long long pl, int ld, const double* x,
                                            long long o) {
    double s = A[C2 * pl + o] * x[o];
    s += A[W2 * pl + o] * x[o - 1];
    s += A[W2 * pl + o + 1] * x[o + 1];
    s += A[S2 * pl + o] * x[o - ld];
    s += A[S2 * pl + o + ld] * x[o + ld];
    s += A[SW2 * pl + o] * x[o - ld - 1];
    s += A[SW2 * pl + o + ld + 1] * x[o + ld + 1];
    s += A[NW2 * pl + o] * x[o + ld - 1];
    s += A[NW2 * pl + o - ld + 1] * x[o - ld + 1];
    return s;
}

// True when every x_j row o (2-D) couples to is +-0 (bit test, no FP64 op):
// then (A x)_o is zero and the FP64 products can be skipped, e.g. for a zero
// initial guess, where the residual is b itself.
__device__ __forceinline__ bool row_x_zero(const double* x, int ld, long long o) {
    auto bits = [](double v) { return (unsigned long long)__double_as_longlong(v) << 1; };
    unsigned long long m = 0;
    // row by row and not unrolled: holding the neighbourhood in registers for
    // the products that follow costs more occupancy than reading it again
#pragma unroll 1
    for (int q = -1; q <= 1 && m == 0; q++) {
        const double* r = x + o + (long long)ld * q;
        m = bits(r[-1]) | bits(r[0]) | bits(r[1]);
    }
    return m == 0;
}

// Row sums s_i = sum_j a_ij of the FP64 operator (all stored couplings).
template <int DIM>
__device__ __forceinline__ double row_sum(const double* __restrict__ A, long long pl, int ld, int n, long long o) {
    if (DIM == 2)
        return A[C2 * pl + o] + A[W2 * pl + o] + A[W2 * pl + o + 1] + A[S2 * pl + o] + A[S2 * pl + o + ld] +
               A[SW2 * pl + o] + A[SW2 * pl + o + ld + 1] + A[NW2 * pl + o] + A[NW2 * pl + o - ld + 1];
    double s = A[13 * pl + o];
    for (int t = 0; t < 13; t++) s += A[(long long)t * pl + o] + A[(long long)t * pl + o - d3(t, ld, n)];
    return s;
}

// Compensated (Neumaier) FP32 accumulator for the inner CG's dot products.
struct Acc32 {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        c += fabsf(s) >= fabsf(x) ? (s - t) + x : (x - t) + s;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// alpha = r.z / p.Ap once p.Ap is known (one thread), and the pending step
__device__ __forceinline__ void set_alpha32(KState* st, double pq, int parity) {
    st->pq = pq;
    if (!(pq > 0.0)) {
        set_err(st, BMG_ERR_NOT_SPD);
        st->alpha = 0.0;
    } else {
        st->alpha = st->rz / pq;
    }
    if (parity == 0) st->alpha0 = st->alpha;
}

#define FOR_ROWS(g)                                                       \
    for (int r_ = blockIdx.x; r_ < (g).rows(); r_ += gridDim.x)           \
        for (int i_ = threadIdx.x; i_ < (g).ld; i_ += blockDim.x)

// FP64 products with the operator over the interior nodes: f(k, (A x)_k) for
// every node k.  With SKIP, rows whose x neighbourhood is +-0 (bit test, no
// FP64 operation) give zero without the products, e.g. for a zero initial
// guess.  FP64 lanes bound these kernels (a row-strided loop left up to 40% of
// them idle on 127 interior columns of 160 padded ones), then the loads:
//   2-D: tiles of 32 columns x 8 rows, H groups of 8 rows per CTA, a thread
//     per node;
//   3-D: tiles of 64 columns x 8 rows, H planes per CTA, a thread per column
//     pair (i, i + 1), i even, so that the loads are two wide and the zero
//     test reads nothing of its own.
// Boundary and padding entries are zero in every array and stay as they are.
template <int DIM>
struct NodeTiles {
    static constexpr int cols = DIM == 2 ? 32 : 64;
    int n, ld, H, ti, tj;
    template <bool SKIP, class F>
    __device__ __forceinline__ void products(const double* __restrict__ A, long long pl, const double* x,
                                             F&& f) const {
        const int t = (int)blockIdx.x, lane = (int)(threadIdx.x & 31), row = (int)(threadIdx.x >> 5);
        if constexpr (DIM == 2) {
            const int i = 1 + 32 * (t % ti) + lane;
            if (i > n - 2) return;
            const int j0 = 1 + 8 * H * (t / ti) + row;
            for (int s = 0; s < H; s++) {
                const int j = j0 + 8 * s;
                if (j > n - 2) break;
                const long long k = (long long)j * ld + i;
                f(k, SKIP && row_x_zero(x, ld, k) ? 0.0 : apply_row(A, pl, ld, x, k));
            }
        } else {
            const int i = 64 * (t % ti) + 2 * lane, j = 1 + 8 * (t / ti % tj) + row;
            if (i + 1 > n - 2 || j > n - 2) return;
            const int k0 = 1 + H * (t / (ti * tj));
            for (int k = k0; k < k0 + H && k <= n - 2; k++) {
                const long long o = (long long)i + (long long)ld * (j + (long long)n * k);
                double s0, s1;
                apply_pair<SKIP>(A, pl, x, i, o, s0, s1);
                if (i > 0) f(o, s0);
                f(o + 1, s1);
            }
        }
    }
    // rows o and o + 1 of A x (3-D): the diagonal, then each offset and its mirror
    template <bool SKIP>
    __device__ __forceinline__ void apply_pair(const double* __restrict__ A, long long pl, const double* x,
                                               int i, long long o, double& s0, double& s1) const {
        const long long sy = ld, sz = (long long)ld * n;
        double X[3][3][4];      // [dz + 1][dy + 1]: columns i - 1 .. i + 2
        unsigned long long m = 0;
#pragma unroll
        for (int z = 0; z < 3; z++)
#pragma unroll
            for (int y = 0; y < 3; y++) {
                const double* q = x + o + (y - 1) * sy + (z - 1) * sz;
                const double2 v = *reinterpret_cast<const double2*>(q);
                X[z][y][0] = i > 0 ? q[-1] : 0.0;
                X[z][y][1] = v.x;
                X[z][y][2] = v.y;
                X[z][y][3] = q[2];
                if (SKIP)
#pragma unroll
                    for (int c = 0; c < 4; c++) m |= (unsigned long long)__double_as_longlong(X[z][y][c]) << 1;
            }
        s0 = s1 = 0.0;
        if (SKIP && m == 0) return;
        {
            const double2 d = *reinterpret_cast<const double2*>(A + 13 * pl + o);
            s0 = d.x * X[1][1][1];
            s1 = d.y * X[1][1][2];
        }
#pragma unroll
        for (int t = 0; t < 13; t++) {
            const int dx = t % 3 - 1, dy = (t / 3) % 3 - 1, dz = t / 9 - 1;
            const double2 own = *reinterpret_cast<const double2*>(A + t * pl + o);
            const double* b = A + t * pl + o - dy * sy - dz * sz;   // the mirrors, stored at the node - d
            const double2 mr = *reinterpret_cast<const double2*>(b);
            const double m0 = dx == 0 ? mr.x : dx < 0 ? mr.y : i > 0 ? b[-1] : 0.0;
            const double m1 = dx == 0 ? mr.y : dx < 0 ? b[2] : mr.x;
            s0 += own.x * X[dz + 1][dy + 1][1 + dx];
            s0 += m0 * X[1 - dz][1 - dy][1 - dx];
            s1 += own.y * X[dz + 1][dy + 1][2 + dx];
            s1 += m1 * X[1 - dz][1 - dy][2 - dx];
        }
    }
};

// ---------------------------------------------------------------- layout
template <int DIM>
__global__ void k_pack_t(int n, int ld, const double* __restrict__ src, double* __restrict__ dst) {
    RowGrid<DIM> g{n, ld};
    FOR_ROWS(g) {
        const bool in = g.row_inner(r_) && i_ >= 1 && i_ <= n - 2;
        dst[(long long)r_ * ld + i_] = in ? src[(long long)r_ * n + i_] : 0.0;
    }
}

template <int DIM>
__global__ void k_unpack_t(int n, int ld, const double* __restrict__ src, double* __restrict__ dst) {
    RowGrid<DIM> g{n, ld};
    FOR_ROWS(g) {
        if (i_ < n) dst[(long long)r_ * n + i_] = src[(long long)r_ * ld + i_];
    }
}

// ---------------------------------------------------------------- FP64 outer CG
// r = b - A x ; st.rr = ||r||^2 (rows with a zero x neighbourhood: r = b)
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_residual64(NodeTiles<DIM> g, const double* __restrict__ A, long long pl,
                                                         const double* b, const double* x,
                                                         double* __restrict__ r, double* partials, KState* st) {
    pdl_wait();
    pdl_trigger();
    double acc = 0.0;
    g.template products<true>(A, pl, x, [&](long long k, double ax) {
        const double v = b[k] - ax;
        r[k] = v;
        acc += v * v;
    });
    double t;
    if (grid_sum(acc, partials, &st->counter[0], &t)) st->rr = t;
}

// The vector kernels below read pairs (planes hold a multiple of 32 values)
// on four CTAs per SM: every CTA's sum costs FP64 slots of its own, and with
// eight per SM, a shuffle tree in every warp, those took as long as the
// vectors (1025^2: r.z 17.5 us, update 16.4 us; now 11.4
// and 14.7 us).
__global__ void __launch_bounds__(kThreads) k_dot64(long long pairs, const double2* __restrict__ a,
                                                    const double2* __restrict__ b, double* partials, KState* st,
                                                    double* slot) {
    double acc = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pairs;
         k += (long long)gridDim.x * blockDim.x) {
        const double2 u = a[k], v = b[k];
        acc += u.x * v.x;
        acc += u.y * v.y;
    }
    double t;
    if (grid_sum(acc, partials, &st->counter[1], &t)) *slot = t;
}

// q = A p; st.pq = p.q; alpha = rz / pq
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_spmv_pq64(NodeTiles<DIM> g, const double* __restrict__ A, long long pl,
                                                        const double* p, double* __restrict__ q,
                                                        double* partials, KState* st) {
    pdl_wait();
    pdl_trigger();
    double acc = 0.0;
    g.template products<false>(A, pl, p, [&](long long k, double v) {
        q[k] = v;
        acc += p[k] * v;
    });
    double t;
    if (grid_sum(acc, partials, &st->counter[2], &t)) {
        st->pq = t;
        if (!(t > 0.0)) {
            set_err(st, BMG_ERR_NOT_SPD);
            st->alpha = 0.0;
        } else {
            st->alpha = st->rz / t;
        }
    }
}

// x += alpha p; r -= alpha q; st.rr = ||r||^2
__global__ void __launch_bounds__(kThreads) k_update_xr64(long long pairs, double2* x,
                                                          double2* r, const double2* p,
                                                          const double2* q, double* partials,
                                                          KState* st) {
    pdl_wait();
    pdl_trigger();
    const double alpha = st->alpha;
    double acc = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pairs;
         k += (long long)gridDim.x * blockDim.x) {
        double2 xv = x[k], rv = r[k];
        const double2 pv = p[k], qv = q[k];
        xv.x += alpha * pv.x;
        xv.y += alpha * pv.y;
        rv.x -= alpha * qv.x;
        rv.y -= alpha * qv.y;
        x[k] = xv;
        r[k] = rv;
        acc += rv.x * rv.x;
        acc += rv.y * rv.y;
    }
    double t;
    if (grid_sum(acc, partials, &st->counter[3], &t)) st->rr = t;
}

// r.z and (flexible) r.z_old in one pass, then beta in the last block; the
// first iteration has no beta.
template <bool FLEX>
__global__ void __launch_bounds__(kThreads) k_rz_beta64(long long pairs, const double2* r,
                                                        const double2* z,
                                                        const double2* zo, double* partials,
                                                        KState* st) {
    pdl_wait();
    pdl_trigger();
    double a1 = 0.0, a2 = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pairs;
         k += (long long)gridDim.x * blockDim.x) {
        const double2 rv = r[k], zv = z[k];
        a1 += rv.x * zv.x;
        a1 += rv.y * zv.y;
        if (FLEX) {
            const double2 ov = zo[k];
            a2 += rv.x * ov.x;
            a2 += rv.y * ov.y;
        }
    }
    double t1 = 0.0, t2 = 0.0;
    const bool lead = FLEX ? grid_sum2(a1, a2, partials, &st->counter[5], &t1, &t2)
                           : grid_sum(a1, partials, &st->counter[5], &t1);
    if (lead) {
        if (st->first) {
            st->beta = 0.0;
            st->first = 0;
        } else {
            st->beta = (FLEX ? t1 - t2 : t1) / st->rz;
        }
        st->rz = t1;
    }
}

// p = z + beta p
__global__ void __launch_bounds__(kThreads) k_p_update64(long long pairs, const double2* z,
                                                         double2* p, KState* st) {
    pdl_wait();
    pdl_trigger();
    const double beta = st->beta;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < pairs;
         k += (long long)gridDim.x * blockDim.x) {
        const double2 zv = z[k];
        double2 pv = p[k];
        pv.x = zv.x + beta * pv.x;
        pv.y = zv.y + beta * pv.y;
        p[k] = pv;
    }
}

// ---------------------------------------------------------------- refinement (FP32 inner CG)
// r32 = (float)(b - A x), ||r||^2 in FP64; resets the inner CG to its first step.
// Rows whose x neighbourhood is zero take r = b without the FP64 products
// (the FP64 rate, not HBM, bounds this kernel otherwise).
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_residual_to32_t(NodeTiles<DIM> g, const double* __restrict__ A,
                                                              long long pl, const double* b,
                                                              const double* x, float* __restrict__ r32,
                                                              double* partials, KState* st) {
    pdl_wait();
    pdl_trigger();
    double acc = 0.0;
    g.template products<true>(A, pl, x, [&](long long k, double ax) {
        const double v = b[k] - ax;
        r32[k] = (float)v;
        acc += v * v;
    });
    double t;
    if (grid_sum(acc, partials, &st->counter[0], &t)) {
        st->rr = t;
        st->first = 1;
        st->alpha0 = 0.0;
    }
}

template <int DIM>
__global__ void k_row_sums32_t(RowGrid<DIM> g, const double* __restrict__ A, long long pl, float* __restrict__ rs) {
    FOR_ROWS(g) {
        const long long k = (long long)r_ * g.ld + i_;
        double v = 0.0;
        if (g.row_inner(r_) && i_ >= 1 && i_ <= g.n - 2) v = row_sum<DIM>(A, pl, g.ld, g.n, k);
        rs[k] = (float)v;
    }
}

// x += alpha p straight into the FP64 iterate (an FP32 correction would cap
// the true residual near eps_32 ||A|| ||d|| / ||A d||, far above 1e-10 for a
// smooth correction d); r -= alpha q in FP32.  The FP64 iterate is touched
// every other iteration: an even one (PARITY 0) updates r alone and leaves its
// alpha in alpha0 (the product kernel puts it there), the odd one adds both
// steps, and k_flush_x32 adds what an odd count leaves.  24 instead of 32 bytes
// a node and iteration.  4097^2: 114 us a pair of iterations, 2 x 88 with x in
// every iteration; 157 with the conversion instruction in place of widen4,
// whose slots in the FP64 units then bound the odd iterations.
__device__ __forceinline__ void add_step(double2& x0, double2& x1, double alpha, float4 p) {
    double d[4];
    widen4(p, d);
    x0.x += alpha * d[0];
    x0.y += alpha * d[1];
    x1.x += alpha * d[2];
    x1.y += alpha * d[3];
}

template <int PARITY>
__global__ void __launch_bounds__(kThreads) k_update_xr32(long long quads, double2* x,
                                                          float4* r, const float4* p0,
                                                          const float4* p1,
                                                          const float4* q, const KState* st) {
    pdl_wait();
    pdl_trigger();
    const double alpha = st->alpha, alpha0 = st->alpha0;
    const float a32 = (float)alpha;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < quads;
         k += (long long)gridDim.x * blockDim.x) {
        const float4 qv = q[k];
        float4 rv = r[k];
        if (PARITY) {
            const float4 pv = p1[k];
            double2 x0 = x[2 * k], x1 = x[2 * k + 1];
            if (alpha0 != 0.0) add_step(x0, x1, alpha0, p0[k]);
            add_step(x0, x1, alpha, pv);
            x[2 * k] = x0;
            x[2 * k + 1] = x1;
        }
        rv.x -= a32 * qv.x;
        rv.y -= a32 * qv.y;
        rv.z -= a32 * qv.z;
        rv.w -= a32 * qv.w;
        r[k] = rv;
    }
}

// x += alpha0 p0: the step an even iteration left at the end of a run
__global__ void __launch_bounds__(kThreads) k_flush_x32(long long quads, double2* x,
                                                        const float4* p0, const KState* st) {
    pdl_wait();
    pdl_trigger();
    const double alpha0 = st->alpha0;
    if (alpha0 == 0.0) return;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < quads;
         k += (long long)gridDim.x * blockDim.x) {
        double2 x0 = x[2 * k], x1 = x[2 * k + 1];
        add_step(x0, x1, alpha0, p0[k]);
        x[2 * k] = x0;
        x[2 * k + 1] = x1;
    }
}

// r.z and r.z_old in one pass; the last block forms the flexible-CG beta.
// Four values a load, four CTAs per SM (as the FP64 vector kernels).
__global__ void __launch_bounds__(kThreads) k_rz_beta32_t(long long quads, const float4* r,
                                                          const float4* z,
                                                          const float4* zo, double* partials,
                                                          KState* st) {
    pdl_wait();
    pdl_trigger();
    Acc32 a1, a2;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < quads;
         k += (long long)gridDim.x * blockDim.x) {
        const float4 rv = r[k], zv = z[k], ov = zo[k];
        a1.add(rv.x * zv.x);
        a2.add(rv.x * ov.x);
        a1.add(rv.y * zv.y);
        a2.add(rv.y * ov.y);
        a1.add(rv.z * zv.z);
        a2.add(rv.z * ov.z);
        a1.add(rv.w * zv.w);
        a2.add(rv.w * ov.w);
    }
    double t1, t2;
    if (grid_sum2(a1.value(), a2.value(), partials, &st->counter[4], &t1, &t2)) {
        if (st->first) {
            st->beta = 0.0;
            st->first = 0;
            st->rzn = t1;   // the run's first r.z, for the host's prediction
        } else {
            st->beta = (t1 - t2) / st->rz;
        }
        st->rz = t1;
    }
}

inline double dofs0(const Ctx& c) {
    const double m = c.lev[0].n - 2;
    return c.dim == 2 ? m * m : m * m * m;
}

#define DISPATCH_DIM(c, KERNEL, ...)                                                                      \
    do {                                                                                                  \
        const Level& L_ = (c).lev[0];                                                                     \
        if ((c).dim == 2)                                                                                 \
            KERNEL<2><<<(c).red_blocks, kThreads, 0, (c).stream>>>(RowGrid<2>{L_.n, L_.ld}, __VA_ARGS__);  \
        else                                                                                              \
            KERNEL<3><<<(c).red_blocks, kThreads, 0, (c).stream>>>(RowGrid<3>{L_.n, L_.ld}, __VA_ARGS__);  \
        (c).launches++;                                                                                   \
    } while (0)

// The same for the node-tile kernels.
#define DISPATCH_TILES(c, KERNEL, ...)                                                                     \
    do {                                                                                                   \
        const Level& L_ = (c).lev[0];                                                                      \
        if ((c).dim == 2)                                                                                  \
            BMG_CUDA(launch_pdl(KERNEL<2>, dim3((c).nt_tiles), dim3(kThreads), 0, (c).stream,              \
                                NodeTiles<2>{L_.n, L_.ld, (c).nt_h, (c).nt_i, (c).nt_j}, __VA_ARGS__));    \
        else                                                                                               \
            BMG_CUDA(launch_pdl(KERNEL<3>, dim3((c).nt_tiles), dim3(kThreads), 0, (c).stream,              \
                                NodeTiles<3>{L_.n, L_.ld, (c).nt_h, (c).nt_i, (c).nt_j}, __VA_ARGS__));    \
        (c).launches++;                                                                                    \
    } while (0)

// CTAs of the reducing vector kernels: four per SM, fewer where a CTA would
// get less than two pairs a thread.
inline int vec_blocks(const Ctx& c) {
    const int want = cdiv(c.lev[0].plane / 2, 2 * kThreads);
    return want < 4 * c.sms ? want : 4 * c.sms;
}

}  // namespace

// Steps per tile of the node-tile kernels: the CTAs of an SM share its FP64
// units, so minimise CTAs per SM x steps (each CTA's reduction counted as
// one more), within the partials' buffer.
bmg_status node_tiles_prepare(Ctx& c) {
    BMG_CUDA(cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, c.device));
    const int m = c.lev[0].n - 2;
    const int ti = c.dim == 2 ? cdiv(m, NodeTiles<2>::cols) : cdiv(m + 1, NodeTiles<3>::cols);   // 3-D from column 0
    const int tj = cdiv(m, 8), steps = c.dim == 2 ? tj : m;
    const long long cols = c.dim == 2 ? ti : (long long)ti * tj;
    long long best = -1;
    for (int h = 1; h <= steps; h++) {
        const long long tiles = cols * cdiv(steps, h);
        if (tiles > kMaxBlocks) continue;
        const long long cost = (long long)cdiv(tiles, c.sms) * (h + 1);
        if (best < 0 || cost < best) {
            best = cost;
            c.nt_h = h;
            c.nt_tiles = (int)tiles;
        }
    }
    c.nt_i = ti;
    c.nt_j = tj;
    return best < 0 ? BMG_ERR_SHAPE : BMG_OK;
}

bmg_status k_pack(Ctx& c, const double* src, double* dst) {
    const Level& L = c.lev[0];
    if (c.dim == 2)
        k_pack_t<2><<<c.red_blocks, kThreads, 0, c.stream>>>(L.n, L.ld, src, dst);
    else
        k_pack_t<3><<<c.red_blocks, kThreads, 0, c.stream>>>(L.n, L.ld, src, dst);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_unpack(Ctx& c, const double* src, double* dst) {
    const Level& L = c.lev[0];
    if (c.dim == 2)
        k_unpack_t<2><<<c.red_blocks, kThreads, 0, c.stream>>>(L.n, L.ld, src, dst);
    else
        k_unpack_t<3><<<c.red_blocks, kThreads, 0, c.stream>>>(L.n, L.ld, src, dst);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_residual(Ctx& c, const double* b, const double* x, double* r) {
    const Level& L = c.lev[0];
    DISPATCH_TILES(c, k_residual64, L.A64, L.plane, b, x, r, c.partials, c.st);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_dot(Ctx& c, const double* a, const double* b, double* slot) {
    const Level& L = c.lev[0];
    k_dot64<<<vec_blocks(c), kThreads, 0, c.stream>>>(L.plane / 2, (const double2*)a, (const double2*)b, c.partials, c.st,
                                                      slot);
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_spmv_pq(Ctx& c, const double* p, double* q) {
    const Level& L = c.lev[0];
    prof_begin(c, BMG_PROF_SPMV, 0);
    DISPATCH_TILES(c, k_spmv_pq64, L.A64, L.plane, p, q, c.partials, c.st);
    prof_end(c, BMG_PROF_SPMV, 0, (c.ns + 2) * 8.0 * dofs0(c));
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_update_xr(Ctx& c) {
    const Level& L = c.lev[0];
    prof_begin(c, BMG_PROF_UPDATE, 0);
    BMG_CUDA(launch_pdl(k_update_xr64, dim3(vec_blocks(c)), dim3(kThreads), 0, c.stream, L.plane / 2, (double2*)c.x,
                        (double2*)c.r, (const double2*)c.p, (const double2*)c.q, c.partials, c.st));
    prof_end(c, BMG_PROF_UPDATE, 0, 6 * 8.0 * dofs0(c));
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_rz_beta(Ctx& c, const double* z, const double* zold, bool flexible) {
    const Level& L = c.lev[0];
    const double2 *r2 = (const double2*)c.r, *z2 = (const double2*)z, *o2 = (const double2*)zold;
    if (flexible)
        BMG_CUDA(launch_pdl(k_rz_beta64<true>, dim3(vec_blocks(c)), dim3(kThreads), 0, c.stream, L.plane / 2, r2, z2, o2,
                            c.partials, c.st));
    else
        BMG_CUDA(launch_pdl(k_rz_beta64<false>, dim3(vec_blocks(c)), dim3(kThreads), 0, c.stream, L.plane / 2, r2, z2,
                            o2, c.partials, c.st));
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_p_update(Ctx& c, const double* z) {
    const Level& L = c.lev[0];
    const int blocks = cdiv(L.plane / 2, 2 * kThreads);
    BMG_CUDA(launch_pdl(k_p_update64, dim3(blocks < c.red_blocks ? blocks : c.red_blocks), dim3(kThreads), 0, c.stream,
                        L.plane / 2, (const double2*)z, (double2*)c.p, c.st));
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_residual_to32(Ctx& c) {
    const Level& L = c.lev[0];
    DISPATCH_TILES(c, k_residual_to32_t, L.A64, L.plane, c.bvec, c.x, c.r32, c.partials, c.st);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

// p = z + beta p_old, q = A p and alpha = r.z / p.q in one pass; p goes to a
// second buffer, since p_old is still being read.  The product is in difference
// form, s_i p_i + sum_{j != i} a_ij (p_j - p_i), with the row sums s_i formed in
// FP64: the operator's rows nearly sum to zero, so the plain FP32 product loses
// the smooth part of A p to cancellation, and the differences keep FP32
// relative accuracy on every mode.
//
// 2-D: a warp owns a strip of 64 columns and a band of H
// rows and marches up the rows on its own, without barriers.  A lane holds the
// column pair (i, i + 1), i even, of the three rows in play in registers (p and
// the planes' values, loaded two wide); its neighbours' columns come by
// shuffle, and lanes 0 and 31 load the strip's edge columns.  The next row's
// raw values (z, p_old, planes) are in flight while a row is formed.  HBM
// bounds the kernel on large grids (36 bytes a node), the chain of row loads
// on small ones.  4097^2: 103 us, 65^2: 7 us, against 129 and 8.1 us for a
// thread per column, a block barrier per row and the planes in shared memory;
// with two CTAs an SM instead of three (92 registers a thread for 80) 120 us.
// A node's terms are summed in the order W, E, S, N, SW, NE, NW, SE.
__global__ void __launch_bounds__(kThreads, 3) k_pspmv2d_strips(int n, int ld, long long pl, int H, int strips, int bands,
                                                             const float* __restrict__ A,
                                                             const float* __restrict__ rs, const float* z,
                                                             const float* pold, float* __restrict__ p,
                                                             float* __restrict__ q, double* partials, KState* st,
                                                             int parity) {
    pdl_wait();
    pdl_trigger();
    const float beta = (float)st->beta;
    const int lane = threadIdx.x & 31;
    const int g = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    const int strip = g % strips, band = g / strips;
    Acc32 acc;
    if (band < bands) {
        const int j0 = 1 + band * H, j1 = min(j0 + H, n - 1);
        const int i = 64 * strip + 2 * lane;
        const bool act0 = i >= 1 && i <= n - 2, act1 = i + 1 <= n - 2;   // act0 implies act1 (n is odd)
        // raw values of a row: the pair's, and the edge column of lane 0 (left)
        // or lane 31 (right)
        struct Raw {
            float2 z, po, w, s, sw, nw, r;
            float ez, ep, ew, esw, enw;
        };
        const int ie = lane == 0 ? i - 1 : i + 2;
        const bool edge = lane == 0 ? i >= 2 : lane == 31 && ie <= n - 2;
        auto load = [&](int j, Raw& v) {
            v = Raw{};
            if (j < 1 || j > n - 2) return;
            const long long kr = (long long)j * ld;
            if (act1) {
                const long long k = kr + i;
                v.z = *reinterpret_cast<const float2*>(z + k);
                v.po = *reinterpret_cast<const float2*>(pold + k);
                v.w = *reinterpret_cast<const float2*>(A + W2 * pl + k);
                v.s = *reinterpret_cast<const float2*>(A + S2 * pl + k);
                v.sw = *reinterpret_cast<const float2*>(A + SW2 * pl + k);
                v.nw = *reinterpret_cast<const float2*>(A + NW2 * pl + k);
                v.r = *reinterpret_cast<const float2*>(rs + k);
            }
            if (edge) {
                const long long k = kr + ie;
                v.ez = z[k];
                v.ep = pold[k];
                if (lane == 31) {
                    v.ew = A[W2 * pl + k];
                    v.esw = A[SW2 * pl + k];
                    v.enw = A[NW2 * pl + k];
                }
            }
        };
        // p at columns i-1 .. i+2, W, SW, NW at i .. i+2, S and row sums at i, i+1
        struct Row {
            float pl, p0, p1, pr, w0, w1, w2, sw0, sw1, sw2, nw0, nw1, nw2, s0, s1, r0, r1;
        };
        auto form = [&](const Raw& v) {
            Row r;
            r.p0 = v.z.x + beta * v.po.x;
            r.p1 = v.z.y + beta * v.po.y;
            const float e = v.ez + beta * v.ep;
            r.pl = __shfl_up_sync(0xffffffffu, r.p1, 1);
            r.pr = __shfl_down_sync(0xffffffffu, r.p0, 1);
            r.w2 = __shfl_down_sync(0xffffffffu, v.w.x, 1);
            r.sw2 = __shfl_down_sync(0xffffffffu, v.sw.x, 1);
            r.nw2 = __shfl_down_sync(0xffffffffu, v.nw.x, 1);
            if (lane == 0) r.pl = e;
            if (lane == 31) {
                r.pr = e;
                r.w2 = v.ew;
                r.sw2 = v.esw;
                r.nw2 = v.enw;
            }
            r.w0 = v.w.x;
            r.w1 = v.w.y;
            r.sw0 = v.sw.x;
            r.sw1 = v.sw.y;
            r.nw0 = v.nw.x;
            r.nw1 = v.nw.y;
            r.s0 = v.s.x;
            r.s1 = v.s.y;
            r.r0 = v.r.x;
            r.r1 = v.r.y;
            return r;
        };
        Raw va, vb, vc;
        load(j0 - 1, va);
        load(j0, vb);
        load(j0 + 1, vc);
        Row rm = form(va), r0 = form(vb);
        for (int j = j0; j < j1; j++) {
            const Row rp = form(vc);
            load(j + 2, vc);
            float u = r0.r0 * r0.p0, v = r0.r1 * r0.p1;
            u += r0.w0 * (r0.pl - r0.p0);
            v += r0.w1 * (r0.p0 - r0.p1);
            u += r0.w1 * (r0.p1 - r0.p0);
            v += r0.w2 * (r0.pr - r0.p1);
            u += r0.s0 * (rm.p0 - r0.p0);
            v += r0.s1 * (rm.p1 - r0.p1);
            u += rp.s0 * (rp.p0 - r0.p0);
            v += rp.s1 * (rp.p1 - r0.p1);
            u += r0.sw0 * (rm.pl - r0.p0);
            v += r0.sw1 * (rm.p0 - r0.p1);
            u += rp.sw1 * (rp.p1 - r0.p0);
            v += rp.sw2 * (rp.pr - r0.p1);
            u += r0.nw0 * (rp.pl - r0.p0);
            v += r0.nw1 * (rp.p0 - r0.p1);
            u += rm.nw1 * (rm.p1 - r0.p0);
            v += rm.nw2 * (rm.pr - r0.p1);
            const long long k = (long long)j * ld + i;
            if (act0) {
                *reinterpret_cast<float2*>(p + k) = make_float2(r0.p0, r0.p1);
                *reinterpret_cast<float2*>(q + k) = make_float2(u, v);
                acc.add(r0.p0 * u);
                acc.add(r0.p1 * v);
            } else if (act1) {      // the boundary column and the first interior one
                p[k + 1] = r0.p1;
                q[k + 1] = v;
                acc.add(r0.p1 * v);
            }
            rm = r0;
            r0 = rp;
        }
    }
    double tot;
    if (grid_sum(acc.value(), partials, &st->counter[2], &tot)) {
        set_alpha32(st, tot, parity);
    }
}

bmg_status k_row_sums32(Ctx& c) {
    const Level& L = c.lev[0];
    DISPATCH_DIM(c, k_row_sums32_t, L.A64, L.plane, c.rs32);
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_rz_beta32(Ctx& c, const float* z, const float* zo) {
    const Level& L = c.lev[0];
    BMG_CUDA(launch_pdl(k_rz_beta32_t, dim3(vec_blocks(c)), dim3(kThreads), 0, c.stream, L.plane / 4,
                        (const float4*)c.r32, (const float4*)z, (const float4*)zo, c.partials, c.st));
    c.launches++;
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

// The same in 3-D: one CTA per tile of 64 columns x 8 rows and a band
// of k-planes, marching up k; p of the next plane, with a halo of one row and
// one column pair, goes from registers (loaded a step ahead) into a shared
// ring of 4 slots, so one barrier per plane suffices.
//
// A thread forms the column pair (i, i + 1), i even: its two nodes' 13 stored
// planes and 13 mirrors a(-d) (stored at the node - d) are two-wide loads
// straight from global memory, issued before the step's barrier so that they
// overlap the wait; the mirrors are other threads' own values, served by L1
// and L2.  HBM bounds the kernel (72 bytes a node).  257^3: 214 us, against
// 252 us with a thread per node and one-wide loads.  A node's terms are
// summed by offset, each followed by its mirror.
constexpr int kP3I = 64, kP3J = 8;
constexpr int kP3Pairs = kP3I / 2 + 2, kP3W = 2 * kP3Pairs, kP3H = kP3J + 2;   // halo tile: pairs a row, columns, rows
constexpr int kP3A = kP3W * kP3H;
constexpr int kP3Per = (kP3Pairs * kP3H + kThreads - 1) / kThreads;           // halo pairs per thread

__global__ void __launch_bounds__(kThreads) k_pspmv3d_direct(int n, int ld, long long pl, int H, int tiles_i,
                                                             int tiles_j, const float* __restrict__ A,
                                                             const float* __restrict__ rs,
                                                             const float* z,
                                                             const float* pold, float* __restrict__ p,
                                                             float* __restrict__ q, double* partials, KState* st,
                                                             int parity) {
    __shared__ __align__(8) float sP[4][kP3A];
    pdl_wait();
    pdl_trigger();
    const float beta = (float)st->beta;
    const int tid = threadIdx.x;
    const int tile = blockIdx.x;
    const int ti = tile % tiles_i, tj = (tile / tiles_i) % tiles_j, tk = tile / (tiles_i * tiles_j);
    const int i0 = ti * kP3I, j0 = 1 + tj * kP3J, k0 = 1 + tk * H;
    const int k1 = min(k0 + H, n - 1);
    const long long sy = ld, sz = (long long)ld * n;
    // halo pair u of the thread: columns i0 - 2 + 2 hp, row j0 - 1 + hj
    float2 rz[kP3Per], rpo[kP3Per];
    auto load = [&](int k) {
#pragma unroll
        for (int u = 0; u < kP3Per; u++) {
            const int h = tid + u * kThreads;
            const int hp = h % kP3Pairs, hj = h / kP3Pairs;
            const int i = i0 - 2 + 2 * hp, j = j0 - 1 + hj;
            const bool in = hj < kP3H && i >= 0 && i + 1 < ld && j <= n - 1 && k <= n - 1;
            const long long o = in ? (long long)i + sy * j + sz * k : 0;
            rz[u] = in ? *reinterpret_cast<const float2*>(z + o) : make_float2(0.f, 0.f);
            rpo[u] = in ? *reinterpret_cast<const float2*>(pold + o) : make_float2(0.f, 0.f);
        }
    };
    auto put = [&](int k) {
        float2* pp = reinterpret_cast<float2*>(sP[k & 3]);
#pragma unroll
        for (int u = 0; u < kP3Per; u++) {
            const int h = tid + u * kThreads;
            if (h < kP3Pairs * kP3H) pp[h] = make_float2(rz[u].x + beta * rpo[u].x, rz[u].y + beta * rpo[u].y);
        }
    };
    const int lane = tid & 31, row = tid >> 5;
    const int i = i0 + 2 * lane, j = j0 + row;
    const bool act0 = i >= 1 && i <= n - 2 && j <= n - 2, act1 = i + 1 <= n - 2 && j <= n - 2;
    const int hc = (row + 1) * kP3W + 2 * (lane + 1);
    load(k0 - 1);
    put(k0 - 1);
    load(k0);
    put(k0);
    load(k0 + 1);
    Acc32 acc;
    for (int k = k0; k < k1; k++) {
        put(k + 1);
        load(k + 2);
        const long long o = (long long)i + sy * j + sz * k;
        float2 a0[13], am[13];
        float as[13];
        float2 rsv = make_float2(0.f, 0.f);
        if (act1) {
#pragma unroll
            for (int t = 0; t < 13; t++) {
                const int dx = t % 3 - 1;
                a0[t] = __ldg(reinterpret_cast<const float2*>(A + t * pl + o));
                const float* b = A + t * pl + o - sy * ((t / 3) % 3 - 1) - sz * (t / 9 - 1);
                am[t] = __ldg(reinterpret_cast<const float2*>(b));
                as[t] = dx < 0 ? __ldg(b + 2) : dx > 0 && i > 0 ? __ldg(b - 1) : 0.f;
            }
            rsv = __ldg(reinterpret_cast<const float2*>(rs + o));
        }
        __syncthreads();
        if (act1) {
            const float* pm = sP[(k + 3) & 3];   // p at k-1
            const float* p0 = sP[k & 3];         // p at k
            const float* pp = sP[(k + 1) & 3];   // p at k+1
            const float2 pv = *reinterpret_cast<const float2*>(p0 + hc);
            float s0 = rsv.x * pv.x, s1 = rsv.y * pv.y;
#pragma unroll
            for (int t = 0; t < 13; t++) {
                const int dx = t % 3 - 1, dy = (t / 3) % 3 - 1, dz = t / 9 - 1;
                const int dh = dx + dy * kP3W;
                const float* pn = dz < 0 ? pm : p0;
                const float* pr = dz < 0 ? pp : p0;
                // the pair's mirrors sit at columns i - dx and i + 1 - dx
                const float m0 = dx == 0 ? am[t].x : dx < 0 ? am[t].y : as[t];
                const float m1 = dx == 0 ? am[t].y : dx < 0 ? as[t] : am[t].x;
                s0 += a0[t].x * (pn[hc + dh] - pv.x);
                s0 += m0 * (pr[hc - dh] - pv.x);
                s1 += a0[t].y * (pn[hc + 1 + dh] - pv.y);
                s1 += m1 * (pr[hc + 1 - dh] - pv.y);
            }
            if (act0) {
                p[o] = pv.x;
                q[o] = s0;
                acc.add(pv.x * s0);
            }
            p[o + 1] = pv.y;
            q[o + 1] = s1;
            acc.add(pv.y * s1);
        }
    }
    double tot;
    if (grid_sum(acc.value(), partials, &st->counter[2], &tot)) {
        set_alpha32(st, tot, parity);
    }
}

// Rows per band of k_pspmv2d_strips (planes per band in 3-D): minimise waves x
// (rows + 2 halo rows) at the kernel's occupancy, with at most kMaxBlocks tiles.
bmg_status pspmv_prepare(Ctx& c) {
    if (!c.rs32) return BMG_OK;
    if (c.dim == 3) {
        // bands of k-planes: minimise waves x (planes + 2) with at most kMaxBlocks tiles
        int sms = 0, occ = 0;
        BMG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c.device));
        BMG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_pspmv3d_direct, kThreads, 0));
        if (occ < 1) return BMG_ERR_DEVICE;
        const int m = c.lev[0].n - 2;
        const int ti = cdiv(m + 1, kP3I), tj = cdiv(m, kP3J);   // columns 0 .. n-2
        const long long slots = (long long)sms * occ;
        long long best = -1;
        for (int h = 1; h <= m; h++) {
            const long long tiles = (long long)ti * tj * cdiv(m, h);
            if (tiles > kMaxBlocks) continue;
            const long long cost = cdiv(tiles, slots) * (h + 2LL);
            if (best < 0 || cost < best) {
                best = cost;
                c.spmv_h = h;
                c.spmv_tiles_x = ti;
                c.spmv_tiles = (int)tiles;
            }
        }
        return best < 0 ? BMG_ERR_SHAPE : BMG_OK;
    }
    int sms = 0, occ = 0;
    BMG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c.device));
    BMG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_pspmv2d_strips, kThreads, 0));
    if (occ < 1) return BMG_ERR_DEVICE;
    const int m = c.lev[0].n - 2;
    const int strips = cdiv(m + 1, 64);    // columns 0 .. n-2
    const long long slots = (long long)sms * occ;
    long long best = -1;
    for (int h = 1; h <= m; h++) {
        const long long ctas = cdiv((long long)strips * cdiv(m, h), kThreads / 32);
        if (ctas > kMaxBlocks) continue;
        const long long cost = cdiv(ctas, slots) * (h + 2LL);
        if (best < 0 || cost < best) {
            best = cost;
            c.spmv_h = h;
            c.spmv_tiles_x = strips;
            c.spmv_tiles = (int)ctas;
        }
    }
    return best < 0 ? BMG_ERR_SHAPE : BMG_OK;
}

bmg_status k_pspmv32(Ctx& c, const float* z, int parity) {
    const Level& L = c.lev[0];
    if (c.spmv_h < 1) return BMG_ERR_STATE;   // pspmv_prepare has not run
    prof_begin(c, BMG_PROF_SPMV, 0);
    if (c.dim == 2) {
        BMG_CUDA(launch_pdl(k_pspmv2d_strips, dim3(c.spmv_tiles), dim3(kThreads), 0, c.stream, L.n, L.ld, L.plane,
                            c.spmv_h, c.spmv_tiles_x, cdiv(L.n - 2, c.spmv_h), L.A32, c.rs32, z, c.p32s[parity ^ 1],
                            c.p32s[parity], c.q32, c.partials, c.st, parity));
    } else {
        const int tj = cdiv(L.n - 2, kP3J);
        BMG_CUDA(launch_pdl(k_pspmv3d_direct, dim3(c.spmv_tiles), dim3(kThreads), 0, c.stream, L.n, L.ld, L.plane,
                            c.spmv_h, c.spmv_tiles_x, tj, L.A32, c.rs32, z, c.p32s[parity ^ 1], c.p32s[parity], c.q32,
                            c.partials, c.st, parity));
    }
    c.launches++;
    prof_end(c, BMG_PROF_SPMV, 0, (c.ns + 4) * 4.0 * dofs0(c));
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

bmg_status k_update_dr32(Ctx& c, int parity) {
    const Level& L = c.lev[0];
    const int want = cdiv(L.plane / 4, kThreads), blocks = want < 8 * c.sms ? want : 8 * c.sms;
    prof_begin(c, BMG_PROF_UPDATE, 0);
    auto kern = parity ? k_update_xr32<1> : k_update_xr32<0>;
    BMG_CUDA(launch_pdl(kern, dim3(blocks), dim3(kThreads), 0, c.stream, L.plane / 4, (double2*)c.x, (float4*)c.r32,
                        (const float4*)c.p32s[0], (const float4*)c.p32s[1], (const float4*)c.q32, c.st));
    // r, q in and r out; the odd iteration also both steps and x
    prof_end(c, BMG_PROF_UPDATE, 0, (parity ? 3 * 4.0 + 2 * 4.0 + 2 * 8.0 : 3 * 4.0) * dofs0(c));
    c.launches++;
    return BMG_OK;
}

bmg_status k_flush_dr32(Ctx& c) {
    const Level& L = c.lev[0];
    const int want = cdiv(L.plane / 4, kThreads), blocks = want < 8 * c.sms ? want : 8 * c.sms;
    BMG_CUDA(launch_pdl(k_flush_x32, dim3(blocks), dim3(kThreads), 0, c.stream, L.plane / 4, (double2*)c.x,
                        (const float4*)c.p32s[0], c.st));
    c.launches++;
    return BMG_OK;
}

}  // namespace bmg
