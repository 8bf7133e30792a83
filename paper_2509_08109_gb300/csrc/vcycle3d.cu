// vcycle3d.cu -- the V(1,1)-cycle on 3-D levels (27-point operators,
// 8-colour Gauss-Seidel with colour (i&1) + 2(j&1) + 4(k&1), forward colour
// order before the coarse correction and reverse after; residual;
// restriction P^T; prolongation with correction; exact solve on 3^3).
#include <type_traits>

#include "common.cuh"
#include "grid3.cuh"
#include "mbar.cuh"

namespace bmg {
namespace {

template <typename T>
struct L3 {
    const T* A;
    int n, ld;
    long long pl;
    __device__ __forceinline__ long long idx(int i, int j, int k) const {
        return (long long)i + (long long)ld * (j + (long long)n * k);
    }
};

// sum over the 26 off-diagonal couplings of row (i,j,k) applied to x
template <typename T>
__device__ __forceinline__ T offdiag3(const L3<T>& L, const T* __restrict__ x, int i, int j, int k) {
    const long long o = L.idx(i, j, k);
    const long long sy = L.ld, sz = (long long)L.ld * L.n;
    T s = 0;
#pragma unroll
    for (int t = 0; t < 13; t++) {
        const long long d = off_x(t) + sy * off_y(t) + sz * off_z(t);
        s += L.A[(long long)t * L.pl + o] * x[o + d];          // a(d) at the node
        s += L.A[(long long)t * L.pl + o - d] * x[o - d];      // a(-d) stored at the node - d
    }
    return s;
}

template <typename T>
__global__ void k_gs_colour3d(L3<T> L, const T* __restrict__ f, T* __restrict__ x, int ci, int cj, int ck) {
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ci;
    const int j = 2 * blockIdx.y + cj, k = 2 * blockIdx.z + ck;
    if (i < 1 || j < 1 || k < 1 || i > L.n - 2 || j > L.n - 2 || k > L.n - 2) return;
    const long long o = L.idx(i, j, k);
    x[o] = (f[o] - offdiag3(L, x, i, j, k)) / L.A[13 * L.pl + o];
}

// Colour-blocked rows: node t of colour col (t runs i fastest over that
// colour's interior nodes) keeps its 27 full-row entries at
// cb[cb_offset(col) + e * count(col) + t], so a colour sweep reads them
// coalesced instead of at stride 2 from the symmetric-half planes.
__global__ void k_cblocks3d(Sten3<float> S, float* __restrict__ cb) {
    const int n = S.n;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y, k = blockIdx.z;
    if (i < 1 || j < 1 || k < 1 || i > n - 2 || j > n - 2 || k > n - 2) return;
    const int col = (i & 1) | ((j & 1) << 1) | ((k & 1) << 2);
    const int ni = cb_side(n, i & 1), nj = cb_side(n, j & 1);
    // first interior index of parity p is 2 - p
    const long long t = (long long)((i - (2 - (i & 1))) >> 1) +
                        (long long)ni * (((j - (2 - (j & 1))) >> 1) + (long long)nj * ((k - (2 - (k & 1))) >> 1));
    const long long nc = cb_count(n, col);
    float* b = cb + cb_offset(n, col) + t;
    for (int e = 0; e < 27; e++) b[e * nc] = S.full(i, j, k, e);
}

// One colour of the FP32 smoother from the colour blocks: the same products
// summed in the same order as k_gs_colour3d (offset t, then its mirror).
__global__ void k_gs_colour3d_cb(const float* __restrict__ blk, long long nc, int ni, int nj, int i0, int j0,
                                 int k0, int n, int ld, const float* __restrict__ f, float* __restrict__ x) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= nc) return;
    const int a = (int)(t % ni);
    const long long r = t / ni;
    const int b = (int)(r % nj), cz = (int)(r / nj);
    const int i = i0 + 2 * a, j = j0 + 2 * b, k = k0 + 2 * cz;
    const long long o = (long long)i + (long long)ld * (j + (long long)n * k);
    const long long sy = ld, sz = (long long)ld * n;
    float s = 0.f;
#pragma unroll
    for (int e = 0; e < 13; e++) {
        const long long d = off_x(e) + sy * off_y(e) + sz * off_z(e);
        s += __ldcs(&blk[e * nc + t]) * x[o + d];
        s += __ldcs(&blk[(26 - e) * nc + t]) * x[o - d];
    }
    x[o] = (__ldcs(&f[o]) - s) / __ldcs(&blk[13 * nc + t]);
}

template <typename T>
struct V2 {
    T x, y;
};
template <typename T>
__device__ __forceinline__ V2<T> ld2(const T* p) {
    if constexpr (sizeof(T) == 4) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        return {v.x, v.y};
    } else {
        const double2 v = __ldg(reinterpret_cast<const double2*>(p));
        return {v.x, v.y};
    }
}

// the same without the read-only path (arrays another kernel has just written
// while this one was coming up), and the store
template <typename T>
__device__ __forceinline__ V2<T> ld2c(const T* p) {
    if constexpr (sizeof(T) == 4) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        return {v.x, v.y};
    } else {
        const double2 v = *reinterpret_cast<const double2*>(p);
        return {v.x, v.y};
    }
}
template <typename T>
__device__ __forceinline__ void st2(T* p, T a, T b) {
    if constexpr (sizeof(T) == 4)
        *reinterpret_cast<float2*>(p) = make_float2(a, b);
    else
        *reinterpret_cast<double2*>(p) = make_double2(a, b);
}

// mask of the non-zero components of offset t: the neighbour at offset t (or
// -t) of a point of colour col has colour col ^ mask
__host__ __device__ constexpr int off_mask(int t) { return (t % 3 != 1) | ((t / 3 % 3 != 1) << 1) | ((t / 9 != 1) << 2); }

// Residual after the forward 8-colour sweep from a zero guess: a point's own
// update zeroed its residual while the neighbours of later colours were
// still zero, so r = - sum over the neighbours of a later colour of a x, in
// the order of offdiag3.  A thread forms the column pair (2p, 2p + 1) of a
// row, so each point's terms are fixed at compile time (rows and planes of
// one parity are uniform over a CTA) and the loads are two wide; a thread per
// point left half the lanes of every term idle.  257^3 FP32: 148 us,
// the time of its 60 bytes a node at the copy rate (225 before); 129^3 FP64:
// 56 us.
template <typename T, int JODD, int KODD>
__device__ __forceinline__ void residual3d_pair(const L3<T>& L, const T* x, int i, long long o, T& r0, T& r1) {
    constexpr int c0 = 2 * JODD + 4 * KODD, c1 = c0 + 1;
    const long long sy = L.ld, sz = (long long)L.ld * L.n;
    T X[3][3][4];      // [dz + 1][dy + 1]: columns i - 1 .. i + 2
#pragma unroll
    for (int z = 0; z < 3; z++)
#pragma unroll
        for (int y = 0; y < 3; y++) {
            if (KODD && z != 1) continue;
            const T* q = x + o + (y - 1) * sy + (z - 1) * sz;
            const V2<T> v = ld2c(q);
            X[z][y][0] = i > 0 ? q[-1] : (T)0;
            X[z][y][1] = v.x;
            X[z][y][2] = v.y;
            X[z][y][3] = q[2];
        }
    T s0 = 0, s1 = 0;
#pragma unroll
    for (int t = 0; t < 13; t++) {
        const bool n0 = (c0 ^ off_mask(t)) > c0, n1 = (c1 ^ off_mask(t)) > c1;
        if (!n0 && !n1) continue;
        const int dx = off_x(t), dy = off_y(t), dz = off_z(t);
        const V2<T> own = ld2(L.A + t * L.pl + o);
        const T* b = L.A + t * L.pl + o - dy * sy - dz * sz;   // the mirrors, stored at the node - d
        const V2<T> m = ld2(b);
        if (n0) {
            s0 += own.x * X[dz + 1][dy + 1][1 + dx];
            s0 += (dx == 0 ? m.x : dx < 0 ? m.y : i > 0 ? __ldg(b - 1) : (T)0) * X[1 - dz][1 - dy][1 - dx];
        }
        if (n1) {
            s1 += own.y * X[dz + 1][dy + 1][2 + dx];
            s1 += (dx == 0 ? m.y : dx < 0 ? __ldg(b + 2) : m.x) * X[1 - dz][1 - dy][2 - dx];
        }
    }
    r0 = -s0;
    r1 = -s1;
}

template <typename T>
__global__ void __launch_bounds__(64) k_residual3d_sweep(L3<T> L, const T* x, T* __restrict__ r) {
    pdl_wait();
    pdl_trigger();
    const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int j = 1 + blockIdx.y, k = 1 + blockIdx.z;      // interior rows and planes
    if (i + 1 > L.n - 2) return;
    const long long o = L.idx(i, j, k);
    T r0, r1;
    if (k & 1) {
        if (j & 1)
            residual3d_pair<T, 1, 1>(L, x, i, o, r0, r1);
        else
            residual3d_pair<T, 0, 1>(L, x, i, o, r0, r1);
    } else {
        if (j & 1)
            residual3d_pair<T, 1, 0>(L, x, i, o, r0, r1);
        else
            residual3d_pair<T, 0, 0>(L, x, i, o, r0, r1);
    }
    if (i > 0) r[o] = r0;
    r[o + 1] = r1;
}

// b_c(K) = sum over the 27 fine neighbours f = 2K + d of P(f, K) r_f, in the
// order of d.  For an interior coarse node every such f is an interior fine
// node; its weight to K sits at the coarse node owning f (K - 1 in each
// direction where d = -1), in the plane of f's parity mask m and of the
// corner K - owner.  All of that is fixed by d, so the loop unrolls to plain
// loads.
template <typename T>
__device__ __forceinline__ void restrict_node3d(int nf, int ldf, const T* r, const T* __restrict__ P,
                                                int nc, int ldc, long long plc, T* __restrict__ bc, int I, int J,
                                                int K) {
    const long long oc = (long long)I + (long long)ldc * (J + (long long)nc * K);
    const long long of = 2LL * I + (long long)ldf * (2 * J + (long long)nf * 2 * K);
    T s = 0;
#pragma unroll
    for (int o = 0; o < 27; o++) {
        const int dx = off_x(o), dy = off_y(o), dz = off_z(o);
        const int m = (dx != 0) | ((dy != 0) << 1) | ((dz != 0) << 2);
        T w = (T)1;
        if (m) {
            const int sb = (dx < 0) | ((dy < 0) << 1) | ((dz < 0) << 2);
            const long long own = oc - (dx < 0) - (long long)ldc * ((dy < 0) + (long long)nc * (dz < 0));
            w = P[(long long)(kPBase(m) + compress3(sb, m)) * plc + own];
        }
        s += w * r[of + dx + (long long)ldf * (dy + (long long)nf * dz)];
    }
    bc[oc] = s;
}

template <typename T>
__global__ void k_restrict3d(int nf, int ldf, const T* r, const T* __restrict__ P, int nc, int ldc,
                             long long plc, T* __restrict__ bc) {
    pdl_wait();
    pdl_trigger();
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y, K = blockIdx.z;
    if (I < 1 || J < 1 || K < 1 || I > nc - 2 || J > nc - 2 || K > nc - 2) return;
    restrict_node3d<T>(nf, ldf, r, P, nc, ldc, plc, bc, I, J, K);
}

// x_f += sum over s subset of m of P(f, (I,J,K) + s) x_c((I,J,K) + s) for the
// eight fine points f = 2(I,J,K) + b (parity mask m = b) that coarse node
// (I,J,K) owns: one thread per coarse node, the 26 weights of its cell read
// once and contiguously across the warp.  Summation over s ascending, as the
// weights' own numbering.
template <typename T>
__device__ __forceinline__ void prolong_node3d(int nf, int ldf, T* __restrict__ x, const T* __restrict__ P, int nc,
                                               int ldc, long long plc, const T* xc, int I, int J,
                                               int K) {
    const long long oc = (long long)I + (long long)ldc * (J + (long long)nc * K);
    const long long sy = ldc, sz = (long long)ldc * nc;
    T c8[8];
#pragma unroll
    for (int q = 0; q < 8; q++) c8[q] = xc[oc + (q & 1) + sy * ((q >> 1) & 1) + sz * (q >> 2)];
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const int fi = 2 * I + (b & 1), fj = 2 * J + ((b >> 1) & 1), fk = 2 * K + (b >> 2);
        if (fi < 1 || fj < 1 || fk < 1 || fi > nf - 2 || fj > nf - 2 || fk > nf - 2) continue;
        T v = 0;
        if (b == 0) {
            v = c8[0];
        } else {
#pragma unroll
            for (int q = 0; q < 8; q++)
                if ((q & ~b) == 0) v += P[(long long)(kPBase(b) + compress3(q, b)) * plc + oc] * c8[q];
        }
        x[(long long)fi + (long long)ldf * (fj + (long long)nf * fk)] += v;
    }
}

template <typename T>
__global__ void k_prolong3d(int nf, int ldf, T* __restrict__ x, const T* __restrict__ P, int nc, int ldc,
                            long long plc, const T* __restrict__ xc) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y, K = blockIdx.z;
    if (I > nc - 2 || J > nc - 2 || K > nc - 2) return;
    prolong_node3d<T>(nf, ldf, x, P, nc, ldc, plc, xc, I, J, K);
}

inline dim3 g3(int ni, int nj, int nk) { return dim3(cdiv(ni, 64), nj, nk); }

// ---------------------------------------------------------------- tail
// The coarse end of the 3-D V-cycle (9^3, 5^3 and 3^3) in one launch of one
// CTA, every level in shared memory for the launch in a compact layout (n in
// place of the padded row length; 76 KB in FP32, 151 KB in FP64).  The
// operators and weights do not change between V-cycles: bmg_setup packs them
// once into the shared-memory image, which a launch stages with bulk copies.
// A barrier separates the colours, and a phase's time is the chain of one
// thread's instructions, of which a level of a few hundred points leaves
// nothing else to run meanwhile.  So:
//   - the diagonals are packed as reciprocals, and the coarsest unknown's
//     reciprocal is formed while the level above still runs;
//   - the forward sweep from the zero guess takes only the couplings to
//     earlier colours, and the residual after it only those to later colours;
//   - eight lanes share a point, each with at most two offsets and their
//     mirrors (FP64 at 9^3, where a colour's 64 points keep the FP64 units
//     busy: two lanes, the stored couplings and the mirrors);
//   - eight lanes share a coarse node of the restriction, and prolongation
//     runs one thread per fine point, all of one parity class in a warp.
//   - what a thread does in a level's colour phases is formed once per level,
//     and arrays are offsets from the shared image (pointers kept in a structure
//     became generic addresses).
// Measured per V-cycle: FP64 41 us (54 before the last two points; 206 when it
// started at 17^3, in global memory), FP32 19.7 us (25.5; 42 in its first form).
constexpr int kTail3Threads = 512;
constexpr int kTail3MaxN = 9;    // first tail level: n <= this
constexpr int kTail3Lev = 3;     // levels of a tail: 9, 5, 3 at most
constexpr unsigned kTail3Chunk = 16384;   // bytes per bulk copy

template <typename T>
struct Tail3Args {
    int nlev;
    int n;                 // nodes per side of the first
    const void* pack;      // packed operators and weights (shared-memory image)
    unsigned pack_bytes;   // its size, a multiple of 16
    const T* b;            // right-hand side of the first tail level
    T* x;                  // its finished iterate
    int ld;                // their row length
    const double* a64c;    // FP64 centre entry of the coarsest operator at (1,1,1)
    KState* st;
};

// first level of the tail, and the sizes of its packed image and vectors
int tail3_first(const Ctx& c) {
    int t = c.nlev - 1;
    while (t > 0 && c.lev[t - 1].n <= kTail3MaxN) t--;
    return t;
}
size_t tail3_pack_elems(const Ctx& c) {
    size_t e = 0;
    for (int l = tail3_first(c); l < c.nlev; l++) {
        const size_t n = c.lev[l].n, nc = l + 1 < c.nlev ? c.lev[l + 1].n : 0;
        e += NS3 * n * n * n + NP3 * nc * nc * nc;
    }
    return e;
}
size_t tail3_vec_elems(const Ctx& c) {
    size_t e = 0;
    for (int l = tail3_first(c); l < c.nlev; l++) e += 3 * (size_t)c.lev[l].n * c.lev[l].n * c.lev[l].n;
    return e;
}

// A level in shared memory: n^3 arrays, as element offsets from the image's
// start (stored pointers would lose their address space).
struct T3 {
    int n, nc;           // nodes per side, of the next level
    int A, P, b, x, r;
};

// lanes per point of a colour phase
template <typename T>
__device__ __forceinline__ int tail3_lanes(int n) { return sizeof(T) == 8 && n > 5 ? 2 : 8; }

// What a thread does in every colour phase of a level, formed once per level:
// its point, lane and share of the point's couplings (eight lanes: offsets lane
// and lane + 8).  n = 2^k + 1, and a colour's points are walked 2^(k-1) a side,
// leaving out the even coordinates' last one; all fit in one round (64 points
// of eight lanes at 9^3).
struct T3Lane {
    bool any;             // the warp has points
    int lane, lanes;
    int o, last;          // the all-even colour's point; bit d: it lies inside in direction d
    int da, db, pa, pb;   // index distance and plane offset
    int ma, mb;           // parity masks; 0: no offset
};
template <typename T>
__device__ __forceinline__ T3Lane tail3_lane(int n, int tid) {
    T3Lane q;
    q.lanes = tail3_lanes<T>(n);
    const int lgl = q.lanes == 8 ? 3 : 1, lg = 31 - __clz(n - 1) - 1, m = 1 << lg, n3 = n * n * n;
    q.lane = tid & (q.lanes - 1);
    const int t = tid >> lgl, I = t & (m - 1), J = (t >> lg) & (m - 1), K = t >> (2 * lg);
    q.any = (tid & ~31) >> lgl < m * m * m;
    q.o = 2 * (1 + I + n * (1 + J + n * (1 + K)));
    q.last = K < m ? (I < m - 1) | ((J < m - 1) << 1) | ((K < m - 1) << 2) : -8;
    const int a = tid & 7, b = a + 8;
    q.da = off_x(a) + n * (off_y(a) + n * off_z(a));
    q.db = off_x(b) + n * (off_y(b) + n * off_z(b));
    q.pa = a * n3;
    q.pb = b * n3;
    q.ma = off_mask(a);
    q.mb = b < 13 ? off_mask(b) : 0;
    return q;
}

// One colour: sel < 0: forward Gauss-Seidel update from the zero guess (the
// couplings to earlier colours); sel == 0: reverse update (all); sel > 0: the
// residual after the forward sweep into r (those to later colours).  The
// colour is a run-time value, uniform over the CTA: unrolled per colour the
// code outran the instruction cache (FP32 tail 72 us instead of 42).
template <typename T>
__device__ __forceinline__ void tail3_colour(T* sm, const T3& v, const T3Lane& ln, int col, int sel) {
    if (!ln.any) return;
    const int n = v.n, n3 = n * n * n;
    const T* A = sm + v.A;
    const T* x = sm + v.x;
    const int o = ln.o - ((col & 1) + n * (((col >> 1) & 1) + n * (col >> 2)));
    const bool on = ln.last >= 0 && ((ln.last | col) & 7) == 7;
    T s = 0, f = 0, dg = 0;
    if (on && sel <= 0) {
        f = sm[v.b + o];
        dg = A[13 * n3 + o];
    }
    if (ln.lanes == 8) {
        const bool ua = sel == 0 || ((col ^ ln.ma) > col) == (sel > 0);
        const bool ub = ln.mb && (sel == 0 || ((col ^ ln.mb) > col) == (sel > 0));
        T s1 = 0;
        if (on && ua) {
            s = A[ln.pa + o] * x[o + ln.da];
            s += A[ln.pa + o - ln.da] * x[o - ln.da];
        }
        if (on && ub) {
            s1 = A[ln.pb + o] * x[o + ln.db];
            s1 += A[ln.pb + o - ln.db] * x[o - ln.db];
        }
        s += s1;
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
    } else if (on) {
        const int h = ln.lane;
        T s1 = 0;   // two chains
#pragma unroll
        for (int q = 0; q < 13; q++) {
            const int c = col ^ off_mask(q);
            if (sel == 0 || (c > col) == (sel > 0)) {
                const int d = off_x(q) + n * (off_y(q) + n * off_z(q));
                const T a = A[q * n3 + (h ? o - d : o)], y = x[h ? o - d : o + d];
                if (q & 1)
                    s1 += a * y;
                else
                    s += a * y;
            }
        }
        s += s1;
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (on && ln.lane == 0) {
        if (sel > 0)
            sm[v.r + o] = -s;
        else   // FP64: f d - s d, one step less in the chain
            sm[v.x + o] = sizeof(T) == 8 ? f * dg - s * dg : (f - s) * dg;
    }
}

template <typename T>
__global__ void __launch_bounds__(kTail3Threads) k_vtail3d(Tail3Args<T> a) {
    extern __shared__ __align__(16) unsigned char t3_raw[];
    __shared__ T3 lv[kTail3Lev];
    __shared__ uint64_t bar;
    __shared__ int s_rw[27];   // restriction: weight plane (31: none) and, from bit 8, the owner's offset bits
    const int tid = threadIdx.x, nth = kTail3Threads;
    const int L = a.nlev;
    T* base = reinterpret_cast<T*>(t3_raw);
    if (tid == 0) {
        // the packed operators and weights, level after level
        mbar::init(&bar, 1);
        mbar::fence_init();
        mbar::expect_tx(&bar, a.pack_bytes);
        for (unsigned off = 0; off < a.pack_bytes; off += kTail3Chunk) {
            const unsigned len = a.pack_bytes - off < kTail3Chunk ? a.pack_bytes - off : kTail3Chunk;
            mbar::bulk_g2s(t3_raw + off, (const unsigned char*)a.pack + off, len, &bar);
        }
        int sp = 0, vp = (int)(a.pack_bytes / sizeof(T));
        for (int q = 0, n = a.n; q < L; q++, n = (n + 1) / 2) {
            T3& v = lv[q];
            const int n3 = n * n * n;
            v.n = n;
            v.nc = q + 1 < L ? (n + 1) / 2 : 0;
            v.A = sp;
            v.P = v.A + NS3 * n3;
            sp = v.P + NP3 * v.nc * v.nc * v.nc;
            v.b = vp;
            v.x = v.b + n3;
            v.r = v.x + n3;
            vp = v.r + n3;
        }
    }
    if (tid >= 32 && tid < 59) {
        const int o = tid - 32, dx = off_x(o), dy = off_y(o), dz = off_z(o);
        const int m = (dx != 0) | ((dy != 0) << 1) | ((dz != 0) << 2);
        const int sb = (dx < 0) | ((dy < 0) << 1) | ((dz < 0) << 2);
        s_rw[o] = (m ? kPBase(m) + compress3(sb, m) : 31) | (sb << 8);
    }
    // the coarsest operator's one entry
    const double ainv = tid == 0 ? 1.0 / *a.a64c : 0.0;
    __syncthreads();
    // meanwhile: zero vectors, then the first level's right-hand side
    {
        const int nv = lv[L - 1].r + lv[L - 1].n * lv[L - 1].n * lv[L - 1].n;
        for (int u = lv[0].b + tid; u < nv; u += nth) base[u] = (T)0;
    }
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    {
        // half a warp a row, every load before the first store
        constexpr int kPass = (kTail3MaxN * kTail3MaxN + kTail3Threads / 16 - 1) / (kTail3Threads / 16);
        const int n = lv[0].n, i = tid & 15, rows = i < n ? n * n : 0;
        T v[kPass];
#pragma unroll
        for (int q = 0; q < kPass; q++) {
            const int row = (tid >> 4) + q * (kTail3Threads / 16);
            v[q] = row < rows ? a.b[(long long)a.ld * row + i] : (T)0;
        }
#pragma unroll
        for (int q = 0; q < kPass; q++) {
            const int row = (tid >> 4) + q * (kTail3Threads / 16);
            if (row < rows) base[lv[0].b + row * n + i] = v[q];
        }
    }
    if (!__syncthreads_and(mbar::wait(&bar, 0))) {
        // record the expiry, give the copies in flight one more bounded wait
        // (the shared memory must outlive them) and leave
        if (tid == 0) set_err(a.st, BMG_ERR_TIMEOUT);
        mbar::wait(&bar, 0);
        return;
    }
    for (int l = 0; l + 1 < L; l++) {
        const T3 v = lv[l], w = lv[l + 1];
        const T3Lane ln = tail3_lane<T>(v.n, tid);
#pragma unroll 1
        for (int ph = 0; ph < 15; ph++) {      // colours 0..7 forward, residuals of colours 0..6
            tail3_colour<T>(base, v, ln, ph & 7, ph < 8 ? -1 : 1);
            if (ph < 8 || ph == 14) __syncthreads();
        }
        // restriction: the 27 fine neighbours of a coarse node over eight lanes
        const int n = v.n, nc = w.n, lg = 31 - __clz(nc - 1), mc = 1 << lg, nc3 = nc * nc * nc;
        for (int t0 = 0; t0 < mc * mc * mc; t0 += nth >> 3) {
            const int t = t0 + (tid >> 3);
            const int I = t & (mc - 1), J = (t >> lg) & (mc - 1), K = t >> (2 * lg);
            const bool on = I > 0 && J > 0 && K > 0 && K < mc;
            const int oc = I + nc * (J + nc * K), of = 2 * (I + n * (J + n * K));
            T s = 0;
            if (on)
                for (int o = tid & 7; o < 27; o += 8) {
                    const int pw = s_rw[o], sb = pw >> 8;
                    const T rv = base[v.r + of + off_x(o) + n * (off_y(o) + n * off_z(o))];
                    const int own = oc - (sb & 1) - nc * (((sb >> 1) & 1) + nc * (sb >> 2));
                    s += (pw & 31) == 31 ? rv : base[v.P + (pw & 31) * nc3 + own] * rv;
                }
            s += __shfl_xor_sync(0xffffffffu, s, 4);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            if (on && (tid & 7) == 0) base[w.b + oc] = s;
        }
        __syncthreads();
    }
    if (tid == 0) {   // coarsest: one unknown, in FP64
        const T3 v = lv[L - 1];
        const int o = 1 + v.n * (1 + v.n);
        base[v.x + o] = (T)((double)base[v.b + o] * ainv);
    }
    __syncthreads();
    for (int l = L - 2; l >= 0; l--) {
        const T3 v = lv[l], w = lv[l + 1];
        const int n = v.n, nc = w.n, lg = 31 - __clz(nc - 1), mc = 1 << lg, nc3 = nc * nc * nc;
        // cell (I, J, K) of the coarse level owns the fine points 2 (I, J, K) + b
        for (int t = tid; t < 8 * mc * mc * mc; t += nth) {
            const int I = t & (mc - 1), J = (t >> lg) & (mc - 1), K = (t >> (2 * lg)) & (mc - 1), b = t >> (3 * lg);
            const int i = 2 * I + (b & 1), j = 2 * J + ((b >> 1) & 1), k = 2 * K + (b >> 2);
            if (i == 0 || j == 0 || k == 0) continue;
            const int oc = I + nc * (J + nc * K);
            T s = 0;
            if (b == 0) {
                s = base[w.x + oc];
            } else {
                const T* P = base + v.P + kPBase(b) * nc3 + oc;
#pragma unroll
                for (int c = 0; c < 8; c++)
                    if ((c & ~b) == 0) {
                        s += *P * base[w.x + oc + (c & 1) + nc * (((c >> 1) & 1) + nc * (c >> 2))];
                        P += nc3;
                    }
            }
            base[v.x + i + n * (j + n * k)] += s;
        }
        __syncthreads();
        const T3Lane ln = tail3_lane<T>(n, tid);
#pragma unroll 1
        for (int col = 7; col >= 0; col--) {
            tail3_colour<T>(base, v, ln, col, 0);
            __syncthreads();
        }
    }
    {   // the first level's iterate to its array
        const int n = lv[0].n;
        for (int row = tid >> 4; row < n * n; row += nth >> 4)
            if ((tid & 15) < n) a.x[(long long)a.ld * row + (tid & 15)] = base[lv[0].x + row * n + (tid & 15)];
    }
}

// Packs one level: the operator's planes in compact rows (the diagonal as its
// reciprocal), then the weights on the next level's grid.
template <typename T>
__global__ void k_tail3_pack(const T* __restrict__ A, int n, int ld, long long pl, const T* __restrict__ P, int nc,
                             int ldc, long long plc, T* __restrict__ dst) {
    const int n3 = n * n * n, nc3 = nc * nc * nc, tot = NS3 * n3 + NP3 * nc3;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += gridDim.x * blockDim.x) {
        const bool op = e < NS3 * n3;
        const int m = op ? n : nc, m3 = op ? n3 : nc3, u = op ? e : e - NS3 * n3;
        const int t = u / m3, r = u - t * m3;
        const int i = r % m, j = (r / m) % m, k = r / (m * m);
        T w = op ? A[t * pl + (long long)i + (long long)ld * (j + (long long)n * k)]
                 : P[t * plc + (long long)i + (long long)ldc * (j + (long long)nc * k)];
        if (op && t == 13 && w != (T)0) w = (T)1 / w;
        dst[e] = w;
    }
}

// ---------------------------------------------------------------- half sweeps
// The 8-colour order visits all colours of the even k-planes (0..3) before
// those of the odd planes (4..7), and the only couplings between planes are
// the 18 z-couplings of a point, which all join planes of opposite parity.
// So each half of a sweep is, plane by plane, an independent 4-colour sweep
// of the plane with the couplings to its two neighbouring planes (whose
// values do not change during that half) taken as they stand:
//   forward (pre-smoothing, zero guess): the even planes first, whose odd
//     neighbours are still zero (in-plane couplings only), then the odd
//     planes against the finished even planes;
//   reverse (post-smoothing): the odd planes against the corrected even
//     planes, then the even planes against the finished odd planes.
// k_hsweep3d runs one such half for every plane of one parity at once: a
// CTA per (tile, plane) holds the plane's iterate over its tile and a halo
// in shared memory, with the two neighbouring planes' iterates beside it.
// Within a plane, colour (i&1) + 2(j&1) of the last phase depends on the
// first through a chain of at most three column steps and one row step, so
// a tile of TI x TJ owned points computes (TI + 6) x (TJ + 2) points
// and neighbouring tiles recompute each other's halo.  Each point's update
// is the per-colour kernels' update: the same 26 products summed in the
// same order (offset t, then its mirror); FP64 multiplies by the stored
// reciprocal of the diagonal, since FP64 arithmetic bounds it.
//
// Threads.  Lane p of a warp owns the column pair (ib + 2p, ib + 2p + 1) of
// a row; the two points of a pair have consecutive colours, so a thread
// loads both points' stencils with 2-wide vector loads when it updates the
// first and keeps the second one's in registers for the next phase.  The
// iterate rows in shared memory keep even and odd columns apart, so the
// neighbour reads of a phase (stride 2 in the natural layout) hit distinct
// banks.
//
// Inputs and outputs are separate arrays (xout is never read), so a CTA
// never sees a neighbour's finished values in place of the initial ones.
//
// Tile shapes.  W warps share a row (64 W computed columns) and S row slots
// give 2 S computed rows, 2 S - 2 of them owned.  FULL: the tile spans the
// whole row and needs no column halo; otherwise it owns 64 W - 6 columns.
// hsweep3d takes the full row up to 129: 58-column tiles compute 192 columns
// for the 127 points of a 129-node row (reverse sweep of one parity at 129^3:
// FP64 120 us, full row 95; FP32 32.6, full row 27.8) and 128 for 63.  At 257^3
// a row takes four warps, so either the rows' halo grows (four slots) or the
// CTA does: 257 us against 196 for the 58-column tiles (169 since their
// accesses are pairs and the first rows' stencils are fetched while the
// iterates are staged).  The levels up to 65 take the slots that leave the
// fewest row slots on the fullest of the chip's 152 SMs (CTAs an SM, rounded up, times
// S): at 65 five (eight tiles in 32 planes, two CTAs an SM), at 33 and below
// three.  FP64, a reverse half sweep: 65^3 22.0 -> 16.3 us with five slots for
// eight, 33^3 13.2 -> 11.1 and 17^3 12.9 -> 10.6 with three; 129^3 CG solve 6.48
// -> 6.24 ms.  The halo row that no owned row needs is left out: a
// seventh of the FP64 arithmetic of the four-slot tiles (129^3 FP64, reverse
// 100 -> 92 us, forward 79 -> 69 us).
template <int W_, int S_, bool FULL_>
struct HsShape {
    static constexpr int W = W_, S = S_;
    static constexpr bool FULL = FULL_;
    static constexpr int threads = 32 * W * S;
    static constexpr int TI = FULL ? 64 * W : 64 * W - 6;   // owned columns
    static constexpr int TJ = 2 * S - 2;                    // owned rows
    static constexpr int half = 32 * W + 2;                 // one parity's columns in a shared row
    static constexpr int cols = 2 * half;                   // shared row: columns ib-2 .. ib+64W+1
    static constexpr int rows = TJ + 4;                     // shared rows
    static constexpr int plane = rows * cols;
};

// In-plane couplings (offsets t >= 9 and their mirrors) that the update of a
// point of the plane's colour col needs: all of them in a reverse sweep, in a
// forward sweep from the zero guess those to the colours already updated.
__host__ __device__ constexpr bool hs_in(int t, int col, bool fwd) { return !fwd || (col ^ (off_mask(t) & 3)) < col; }
// plane of the diagonal: FP64 levels keep its reciprocal behind the operator
template <typename T>
constexpr int hs_diag() { return sizeof(T) == 8 ? NS3 : 13; }

template <typename T>
struct HS3Args {
    const T* A;          // symmetric-half planes (NS3)
    int n, ld;
    long long pl;
    const T* f;          // right-hand side
    const T* xcur;       // initial iterate of the swept planes (mode 2)
    const T* xz;         // iterate of the neighbouring planes (modes 1, 2)
    T* xout;             // swept planes' result (owned points)
    int parity;          // planes k with k & 1 == parity
};

// One pair's stencil: the 14 stored planes at both points (own) and, for
// each stored offset d, the mirror a(q, q - d) stored at q - d.
template <typename T, int MODE, bool FWD>
struct HsPair {
    T own0[NS3], own1[NS3];   // first (even column) / second point
    T mir0[13], mir1[13];
    T f0, f1;
    // JODD: the row's parity (its two points have colours 2 JODD, 2 JODD + 1)
    template <int JODD>
    static constexpr bool needs(int t) {
        return t < 9 ? MODE != 0   // z-couplings (mode 0: the odd planes are still zero)
                     : hs_in(t, 2 * JODD, FWD) || hs_in(t, 2 * JODD + 1, FWD);
    }
    template <int JODD>
    __device__ __forceinline__ void load(const HS3Args<T>& a, long long o0, bool first_ok) {
        const long long sz = (long long)a.ld * a.n;
#pragma unroll
        for (int t = 0; t < NS3; t++) {
            if (t < 13 && !needs<JODD>(t)) continue;
            const V2<T> v = ld2(a.A + (t == 13 ? hs_diag<T>() : t) * a.pl + o0);
            own0[t] = v.x;
            own1[t] = v.y;
        }
#pragma unroll
        for (int t = 0; t < 13; t++) {
            if (!needs<JODD>(t)) continue;
            const int dx = off_x(t), dy = off_y(t), dz = off_z(t);
            const long long m = o0 - (long long)dy * a.ld - dz * sz;   // node (i, j - dy, k - dz)
            const T* b = a.A + t * a.pl + m;
            const V2<T> v = ld2(b);
            if (dx == 0) {
                mir0[t] = v.x;
                mir1[t] = v.y;
            } else if (dx < 0) {             // mirrors at columns i + 1 and i + 2
                mir0[t] = v.y;
                mir1[t] = __ldg(b + 2);
            } else {                         // mirrors at columns i - 1 and i
                mir0[t] = first_ok ? __ldg(b - 1) : (T)0;
                mir1[t] = v.x;
            }
        }
    }
    __device__ __forceinline__ void load_f(const HS3Args<T>& a, long long o0) {
        const V2<T> v = ld2c(a.f + o0);
        f0 = v.x;
        f1 = v.y;
    }
};

// Gauss-Seidel update of one point from its stencil and the shared
// iterates.  ODD: the point is the pair's second (odd) column.  s: index of
// the point's row in the shared arrays (row start), p: the pair.
template <typename T, typename SH, int MODE, bool FWD, int JODD, bool ODD>
__device__ __forceinline__ T hs_update(const T* own, const T* mir, T f, const T* xc, const T* xb, const T* xa,
                                       int rs, int p) {
    // shared index of the neighbour at column offset dx, row offset dy
    auto at = [&](int dx, int dy) {
        const int c = ODD ? (dx == 0 ? SH::half + p + 1 : (dx < 0 ? p + 1 : p + 2))
                          : (dx == 0 ? p + 1 : (dx < 0 ? SH::half + p : SH::half + p + 1));
        return rs + dy * SH::cols + c;
    };
    T s = 0;
#pragma unroll
    for (int t = 0; t < 13; t++) {
        if (MODE == 0 && t < 9) continue;
        if (t >= 9 && !hs_in(t, 2 * JODD + ODD, FWD)) continue;
        const int dx = off_x(t), dy = off_y(t), dz = off_z(t);
        const T* xp = dz < 0 ? xb : xc;   // plane of q + d
        const T* xm = dz < 0 ? xa : xc;   // plane of q - d
        s += own[t] * xp[at(dx, dy)];
        s += mir[t] * xm[at(-dx, -dy)];
    }
    return sizeof(T) == 8 ? (f - s) * own[13] : (f - s) / own[13];
}

// MODE 0: zero initial iterate, no z-couplings (forward sweep of the even
// planes); MODE 1: zero initial iterate, z-couplings to xz (forward sweep of
// the odd planes); MODE 2: initial iterate xcur, z-couplings to xz (reverse
// sweeps).  FWD: colours of the plane ascending, else descending.
template <typename T, typename SH, int MODE, bool FWD>
__global__ void __launch_bounds__(SH::threads, (sizeof(T) == 8 ? 512 : 768) / SH::threads) k_hsweep3d(HS3Args<T> a) {
    extern __shared__ __align__(16) unsigned char hs_raw[];
    T* xc = reinterpret_cast<T*>(hs_raw);   // swept plane k
    T* xb = xc + SH::plane;                  // plane k - 1
    T* xa = xb + SH::plane;                  // plane k + 1
    const int n = a.n, ld = a.ld;
    const long long sz = (long long)ld * n;
    const int k = 2 - a.parity + 2 * (int)blockIdx.z;
    const int i0 = 1 + (int)blockIdx.x * SH::TI, j0 = 1 + (int)blockIdx.y * SH::TJ;
    const int ib = SH::FULL ? 0 : i0 - 3;    // first computed column (even)
    const int tid = threadIdx.x;
    const int slot = tid / (32 * SH::W);
    const int p = tid - 32 * SH::W * slot;   // the pair's index in the row
    const int i = ib + 2 * p;                // its first column
    HsPair<T, MODE, FWD> hold;
    bool ok0 = false, ok1 = false;
    using First = std::integral_constant<int, FWD ? 0 : 1>;
    using Second = std::integral_constant<int, FWD ? 1 : 0>;
    // the pair's rows: region row 2 slot + jpar, j = j0 - 1 + row (j0 - 1 is
    // even).  Owned rows of the second parity need the halo rows of the first
    // alone; the halo row of the second is left out.
    auto load = [&](auto jp) {
        constexpr int jpar = decltype(jp)::value;
        const int row = 2 * slot + jpar, j = j0 - 1 + row;
        const bool pv = j >= 1 && j <= n - 2 && i >= 0 && i <= n - 2 &&
                        (jpar == First::value || (row >= 1 && row <= SH::TJ));
        ok0 = pv && i >= 1;
        ok1 = pv && i + 1 <= n - 2;
        if (pv) hold.template load<jpar>(a, (long long)i + (long long)ld * j + sz * k, ok0);
    };
    auto load_f = [&](int jpar) {
        if (ok0 || ok1) hold.load_f(a, (long long)i + (long long)ld * (j0 - 1 + 2 * slot + jpar) + sz * k);
    };
    // the first rows' stencils, which no kernel of the iteration writes, are in
    // flight while the iterates are staged
    load(First{});
    pdl_wait();
    pdl_trigger();
    load_f(First::value);
    // Shared position (lr, lc) holds node (ib - 2 + lc, j0 - 2 + lr), even
    // columns before odd ones; boundary and padding entries of the arrays are
    // zero, so a pair is in or out as a whole.
    for (int q = tid; q < SH::rows * SH::half; q += SH::threads) {
        const int lr = q / SH::half, lp = q - lr * SH::half;
        const int ic = ib - 2 + 2 * lp, j = j0 - 2 + lr;
        const bool in = ic >= 0 && ic + 1 < ld && j >= 0 && j <= n - 1;
        const int s = lr * SH::cols + lp;
        const long long o = (long long)ic + (long long)ld * j + sz * k;
        V2<T> c{0, 0}, b{0, 0}, t{0, 0};
        if (in) {
            if (MODE == 2) c = ld2c(a.xcur + o);
            if (MODE >= 1) {
                b = ld2c(a.xz + o - sz);
                t = ld2c(a.xz + o + sz);
            }
        }
        xc[s] = c.x;
        xc[s + SH::half] = c.y;
        if (MODE >= 1) {
            xb[s] = b.x;
            xb[s + SH::half] = b.y;
            xa[s] = t.x;
            xa[s + SH::half] = t.y;
        }
    }
    __syncthreads();
    // one row parity: the pair's earlier colour, then the later one from the
    // registers (FWD: even column first; reverse: odd column first)
    auto phase = [&](auto jp, bool second) {
        constexpr int jpar = decltype(jp)::value;
        const int rs = (2 * slot + jpar + 1) * SH::cols;
        const bool do_odd = FWD ? second : !second;
        if (do_odd) {
            if (ok1)
                xc[rs + SH::half + p + 1] =
                    hs_update<T, SH, MODE, FWD, jpar, true>(hold.own1, hold.mir1, hold.f1, xc, xb, xa, rs, p);
        } else {
            if (ok0)
                xc[rs + p + 1] =
                    hs_update<T, SH, MODE, FWD, jpar, false>(hold.own0, hold.mir0, hold.f0, xc, xb, xa, rs, p);
        }
        __syncthreads();
    };
    phase(First{}, false);
    phase(First{}, true);
    load(Second{});
    load_f(Second::value);
    phase(Second{}, false);
    phase(Second{}, true);
    // every thread stores its pair of both rows
#pragma unroll
    for (int r = 0; r < 2; r++) {
        const int lrow = 2 * slot + r, j = j0 - 1 + lrow;
        if (lrow < 1 || lrow > SH::TJ || j > n - 2) continue;
        const bool w0 = i >= i0 && i < i0 + SH::TI && i <= n - 2;
        const bool w1 = i + 1 >= i0 && i + 1 < i0 + SH::TI && i + 1 <= n - 2;
        const T v0 = xc[(lrow + 1) * SH::cols + p + 1], v1 = xc[(lrow + 1) * SH::cols + SH::half + p + 1];
        T* o = a.xout + (long long)i + (long long)ld * j + sz * k;
        if (w0 && w1) {
            st2(o, v0, v1);
        } else if (w0) {
            o[0] = v0;
        } else if (w1) {
            o[1] = v1;
        }
    }
}

// x_out = x_in + P x_c at every interior fine point (out of place; the
// same sum as prolong_node3d).
template <typename T>
__global__ void k_prolong3d_to(int nf, int ldf, const T* xin, T* __restrict__ xout,
                               const T* __restrict__ P, int nc, int ldc, long long plc, const T* xc) {
    pdl_wait();
    pdl_trigger();
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = blockIdx.y, K = blockIdx.z;
    if (I > nc - 2 || J > nc - 2 || K > nc - 2) return;
    const long long oc = (long long)I + (long long)ldc * (J + (long long)nc * K);
    const long long sy = ldc, szc = (long long)ldc * nc;
    T c8[8];
#pragma unroll
    for (int q = 0; q < 8; q++) c8[q] = xc[oc + (q & 1) + sy * ((q >> 1) & 1) + szc * (q >> 2)];
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const int fi = 2 * I + (b & 1), fj = 2 * J + ((b >> 1) & 1), fk = 2 * K + (b >> 2);
        if (fi < 1 || fj < 1 || fk < 1 || fi > nf - 2 || fj > nf - 2 || fk > nf - 2) continue;
        T v = 0;
        if (b == 0) {
            v = c8[0];
        } else {
#pragma unroll
            for (int q = 0; q < 8; q++)
                if ((q & ~b) == 0) v += P[(long long)(kPBase(b) + compress3(q, b)) * plc + oc] * c8[q];
        }
        const long long o = (long long)fi + (long long)ldf * (fj + (long long)nf * fk);
        xout[o] = xin[o] + v;
    }
}

inline double dofs3(const Ctx& c, int l) {
    const double m = c.lev[l].n - 2;
    return m * m * m;
}

template <typename T>
const T* A_of(const Level& L) { return (const T*)(sizeof(T) == 4 ? (const void*)L.A32 : (const void*)L.A64); }
template <typename T>
const T* P_of(const Level& L) { return (const T*)(sizeof(T) == 4 ? (const void*)L.P32 : (const void*)L.P64); }

// one colour of the smoother on level l: colour blocks when the level has
// them (FP32), otherwise the symmetric-half planes
template <typename T>
bmg_status colour_sweep(Ctx& c, int l, const L3<T>& v, const T* f, T* x, int col, int h) {
    const Level& F = c.lev[l];
    const double N = dofs3(c, l);
    prof_begin(c, BMG_PROF_SMOOTH, l);
    if constexpr (sizeof(T) == 4) {
        if (F.cb) {
            const int pi = col & 1, pj = (col >> 1) & 1, pk = col >> 2;
            const long long nc = cb_count(F.n, col);
            const unsigned blocks = (unsigned)((nc + 255) / 256);
            k_gs_colour3d_cb<<<blocks, 256, 0, c.stream>>>(F.cb + cb_offset(F.n, col), nc, cb_side(F.n, pi),
                                                           cb_side(F.n, pj), 2 - pi, 2 - pj, 2 - pk, F.n, F.ld, f, x);
            c.launches++;
            prof_end(c, BMG_PROF_SMOOTH, l, (27.0 + 3.0) * sizeof(T) * N / 8);
            return BMG_OK;
        }
    }
    k_gs_colour3d<T><<<g3(h, h, h), 64, 0, c.stream>>>(v, f, x, col & 1, (col >> 1) & 1, col >> 2);
    c.launches++;
    prof_end(c, BMG_PROF_SMOOTH, l, (c.ns + 3) * sizeof(T) * N / 8);
    return BMG_OK;
}

}  // namespace

bmg_status colour_blocks3d(Ctx& c) {
    if (c.opts.precision != BMG_PREC_FP32 || c.dim != 3) return BMG_OK;
    for (int l = 0; l + 1 < c.nlev; l++) {
        const Level& L = c.lev[l];
        if (!L.cb) continue;
        k_cblocks3d<<<g3(L.n, L.n, L.n), 64, 0, c.stream>>>(Sten3<float>{L.A32, L.n, L.ld, L.plane}, L.cb);
        c.launches++;
    }
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

// One half sweep on level l (all planes of one parity); bytes for the
// profiler: per point of the parity its stored planes (in-plane ones only in
// mode 0), the mirrored z-planes of the plane above, the neighbouring
// planes' iterate, the right-hand side, the output and (mode 2) the input.
template <typename T, typename SH, int MODE, bool FWD>
bmg_status launch_hsweep3d(Ctx& c, const HS3Args<T>& a, int planes) {
    auto kern = k_hsweep3d<T, SH, MODE, FWD>;
    const int smem = (int)(3 * SH::plane * sizeof(T));
    if (smem > 48 * 1024) BMG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    BMG_CUDA(launch_pdl(kern, dim3(cdiv(a.n - 2, SH::TI), cdiv(a.n - 2, SH::TJ), planes), dim3(SH::threads), smem,
                        c.stream, a));
    c.launches++;
    return BMG_OK;
}

template <typename T, int MODE, bool FWD>
bmg_status hsweep3d(Ctx& c, int l, const T* f, const T* xcur, const T* xz, T* xout, int parity) {
    const Level& F = c.lev[l];
    const int planes = parity ? (F.n - 1) / 2 : (F.n - 3) / 2;
    if (planes < 1) return BMG_OK;
    const HS3Args<T> a{A_of<T>(F), F.n, F.ld, F.plane, f, xcur, xz, xout, parity};
    prof_begin(c, BMG_PROF_SMOOTH, l);
    bmg_status st;
    if (F.n <= 33)
        st = launch_hsweep3d<T, HsShape<1, 3, true>, MODE, FWD>(c, a, planes);
    else if (F.n <= 65)
        st = launch_hsweep3d<T, HsShape<1, 5, true>, MODE, FWD>(c, a, planes);
    else if (F.n <= 129)
        st = launch_hsweep3d<T, HsShape<2, 4, true>, MODE, FWD>(c, a, planes);
    else
        st = launch_hsweep3d<T, HsShape<1, 8, false>, MODE, FWD>(c, a, planes);
    const double per = MODE == 0 ? 5.0 + 2.0 : (MODE == 1 ? 14.0 + 9.0 + 2.0 + 2.0 : 14.0 + 9.0 + 2.0 + 3.0);
    prof_end(c, BMG_PROF_SMOOTH, l, per * sizeof(T) * dofs3(c, l) / 2);
    return st;
}

// The half-sweep legs of a level.
template <typename T>
bmg_status hs3_down(Ctx& c, int l, const T* f, T* x) {
    // even planes (their odd neighbours still zero), then odd planes
    BMG_TRY((hsweep3d<T, 0, true>(c, l, f, nullptr, nullptr, x, 0)));
    return hsweep3d<T, 1, true>(c, l, f, nullptr, x, x, 1);
}

template <typename T>
bmg_status hs3_up(Ctx& c, int l, const T* f, T* x, const T* xc) {
    // x + P x_c into the residual buffer (free until the next down leg), then
    // the odd planes against the corrected even planes, then the even planes
    // against the finished odd planes
    const Level& F = c.lev[l];
    const Level& K = c.lev[l + 1];
    T* xcor = (T*)F.r;
    prof_begin(c, BMG_PROF_PROLONG, l);
    BMG_CUDA(launch_pdl(k_prolong3d_to<T>, g3(K.n - 1, K.n - 1, K.n - 1), dim3(64), 0, c.stream, F.n, F.ld, x, xcor,
                        P_of<T>(F), K.n, K.ld, K.plane, xc));
    prof_end(c, BMG_PROF_PROLONG, l, (2.0 + c.np / 8.0 + 0.125) * sizeof(T) * dofs3(c, l));
    c.launches += 1;
    BMG_TRY((hsweep3d<T, 2, false>(c, l, f, xcor, xcor, x, 1)));
    return hsweep3d<T, 2, false>(c, l, f, xcor, x, x, 0);
}

template <typename T>
bmg_status vcycle3d_impl(Ctx& c, const T* b0, T* x0) {
    cudaStream_t s = c.stream;
    const int L = c.nlev;
    const double sz = sizeof(T);
    auto bl = [&](int l) { return l == 0 ? b0 : (const T*)c.lev[l].b; };
    auto xl = [&](int l) { return l == 0 ? x0 : (T*)c.lev[l].x; };
    // levels t .. L-1 run in the single-CTA tail
    const int t = tail3_first(c);
    for (int l = 0; l < t; l++) {
        const Level& F = c.lev[l];
        const Level& K = c.lev[l + 1];
        L3<T> v{A_of<T>(F), F.n, F.ld, F.plane};
        const int h = (F.n + 1) / 2;
        const double N = dofs3(c, l);
        if (c.use_hs3) {   // writes every interior node, reads none before
            BMG_TRY(hs3_down(c, l, bl(l), xl(l)));
        } else {
            BMG_CUDA(cudaMemsetAsync(xl(l), 0, sizeof(T) * F.plane, s));
            for (int col = 0; col < 8; col++) BMG_TRY(colour_sweep<T>(c, l, v, bl(l), xl(l), col, h));
        }
        prof_begin(c, BMG_PROF_RESIDUAL, l);
        BMG_CUDA(launch_pdl(k_residual3d_sweep<T>, g3((F.n - 1) / 2, F.n - 2, F.n - 2), dim3(64), 0, s, v, xl(l),
                            (T*)F.r));
        prof_end(c, BMG_PROF_RESIDUAL, l, (c.ns + 3) * sz * N);
        prof_begin(c, BMG_PROF_RESTRICT, l);
        BMG_CUDA(launch_pdl(k_restrict3d<T>, g3(K.n, K.n, K.n), dim3(64), 0, s, F.n, F.ld, (const T*)F.r, P_of<T>(F),
                            K.n, K.ld, K.plane, (T*)K.b));
        prof_end(c, BMG_PROF_RESTRICT, l, (1.0 + c.np / 8.0 + 0.125) * sz * N);
        c.launches += 2;   // residual, restriction (the colours count themselves)
    }
    {
        Tail3Args<T> a{};
        a.nlev = L - t;
        if (a.nlev > kTail3Lev) return BMG_ERR_STATE;   // n <= 9 has at most kTail3Lev levels
        a.n = c.lev[t].n;
        a.pack = c.tail_pack;
        a.pack_bytes = (unsigned)tail3_pack_bytes(c);
        a.b = bl(t);
        a.x = xl(t);
        a.ld = c.lev[t].ld;
        const Level& C = c.lev[L - 1];
        a.a64c = C.A64 + 13 * C.plane + (long long)C.ld * (1 + (long long)C.n) + 1;
        a.st = c.st;
        const size_t smem = a.pack_bytes + sizeof(T) * tail3_vec_elems(c);
        BMG_CUDA(cudaFuncSetAttribute(k_vtail3d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        BMG_CUDA(launch_pdl(k_vtail3d<T>, dim3(1), dim3(kTail3Threads), smem, s, a));
        c.launches++;
    }
    for (int l = t - 1; l >= 0; l--) {
        const Level& F = c.lev[l];
        const Level& K = c.lev[l + 1];
        L3<T> v{A_of<T>(F), F.n, F.ld, F.plane};
        const double N = dofs3(c, l);
        if (c.use_hs3) {
            BMG_TRY(hs3_up(c, l, bl(l), xl(l), xl(l + 1)));
            continue;
        }
        prof_begin(c, BMG_PROF_PROLONG, l);
        k_prolong3d<T><<<g3(K.n - 1, K.n - 1, K.n - 1), 64, 0, s>>>(F.n, F.ld, xl(l), P_of<T>(F), K.n, K.ld,
                                                                     K.plane, xl(l + 1));
        prof_end(c, BMG_PROF_PROLONG, l, (2.0 + c.np / 8.0 + 0.125) * sz * N);
        const int h = (F.n + 1) / 2;
        for (int col = 7; col >= 0; col--) BMG_TRY(colour_sweep<T>(c, l, v, bl(l), xl(l), col, h));
        c.launches += 1;   // prolongation
    }
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}

size_t tail3_pack_bytes(const Ctx& c) {
    return (tail3_pack_elems(c) * (c.opts.precision == BMG_PREC_FP32 ? 4 : 8) + 15) & ~(size_t)15;
}

namespace {
template <typename T>
bmg_status tail3_pack_impl(Ctx& c) {
    T* q = (T*)c.tail_pack;
    for (int l = tail3_first(c); l < c.nlev; l++) {
        const Level& F = c.lev[l];
        const bool last = l + 1 == c.nlev;
        const int nc = last ? 0 : c.lev[l + 1].n;
        const int tot = NS3 * F.n * F.n * F.n + NP3 * nc * nc * nc;
        k_tail3_pack<T><<<cdiv(tot, 256), 256, 0, c.stream>>>(A_of<T>(F), F.n, F.ld, F.plane, last ? nullptr : P_of<T>(F),
                                                             nc, last ? 0 : c.lev[l + 1].ld,
                                                             last ? 0 : c.lev[l + 1].plane, q);
        c.launches++;
        q += tot;
    }
    BMG_CUDA(cudaGetLastError());
    return BMG_OK;
}
}  // namespace

bmg_status tail3_pack(Ctx& c) {
    return c.opts.precision == BMG_PREC_FP32 ? tail3_pack_impl<float>(c) : tail3_pack_impl<double>(c);
}

template bmg_status vcycle3d_impl<double>(Ctx&, const double*, double*);
template bmg_status vcycle3d_impl<float>(Ctx&, const float*, float*);

}  // namespace bmg
