// common.cuh -- internal types and device helpers of libbmg.
//
// Internal layout.  Every level l of the hierarchy stores its grid
// (n_l nodes per side) with a padded row length ld_l (a multiple of 32
// elements, so every row starts on a 128-byte boundary in FP32 and a
// 256-byte boundary in FP64); one "plane" holds ld_l * n_l^(d-1) values,
// i fastest.  Padding and boundary entries are kept at zero in every array.
//
// Operators are stored as the symmetric half of the 9-point (2-D) or
// 27-point (3-D) stencil, one plane per stored offset (the symmetric
// storage of Sec. 4.1: five values per node in 2-D):
//   2-D: C (0,0), W (-1,0), S (0,-1), SW (-1,-1), NW (-1,+1);
//        a(+d) at node i is a(-d) stored at node i+d.
//   3-D: C and the 13 offsets that are lexicographically negative
//        (dz<0, or dz==0 and dy<0, or dz==dy==0 and dx<0).
// Interpolation P_l (level l+1 -> level l) is stored on the coarse grid,
// one plane per weight of the fine points owned by coarse node (I,J[,K])
// (the fine points 2I+{0,1}, 2J+{0,1}[, 2K+{0,1}] other than the C point):
//   2-D: PXL PXR  (2I+1,2J)   -> (I,J), (I+1,J)
//        PYS PYN  (2I,2J+1)   -> (I,J), (I,J+1)
//        PSW PSE PNW PNE (2I+1,2J+1) -> (I,J), (I+1,J), (I,J+1), (I+1,J+1)
//   3-D: 26 planes, see setup3d.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/bmg.h"
#include "fused2d.cuh"

namespace bmg {

constexpr int kMaxLevels = 20;
constexpr int kThreads = 256;
constexpr int kChipSms = 152;          // SMs of a GB300: grids whose size workspaces and results depend on
constexpr int kMaxBlocks = 4096;       // partials buffer size for reductions (two sums per block)
// refinement mode: most FP32 inner iterations between two FP64 residuals
// (slowly converging problems, e.g. the 3-D shell, need hundreds per solve)
constexpr int kMaxInner = 400;

enum Plane2 { C2 = 0, W2 = 1, S2 = 2, SW2 = 3, NW2 = 4, NS2 = 5 };
enum PPlane2 { PXL = 0, PXR = 1, PYS = 2, PYN = 3, PSW = 4, PSE = 5, PNW = 6, PNE = 7, NP2 = 8 };
constexpr int NS3 = 14;
constexpr int NP3 = 26;

// Device error word values mirror bmg_status.
struct KState {
    double bb;        // ||b||^2
    double rr;        // ||r||^2 (last reduction)
    double rz;        // r.z of the previous iteration
    double rzn;       // r.z of the first iteration of the current inner run (refinement mode)
    double pq;        // p.Aq
    double alpha, beta;
    double alpha0;    // refinement mode: step of the last even iteration, not yet in x
    double dot;       // scratch result of a plain dot product
    int err;          // first device error (bmg_status), 0 = none
    int first;        // 1 on the first iteration (p = z, no beta)
    unsigned int counter[8];
};

// CG scalars of one system (one right-hand side of one problem) in a
// batched solve; mirrors the fields of KState that the batched kernels use.
struct SysState {
    double bb;        // ||b||^2
    double rr;        // ||r||^2 of the last FP64 residual
    double rz;        // r.z of the previous inner iteration
    double pq;        // p.Ap
    double alpha, beta;
    double alpha0;    // step of the last even iteration, not yet in x
    double rz0;       // r.z of the first inner iteration of the current run
    double stop;      // the run ends for this system once r.z <= stop * rz0 (0: it takes its full count)
    int first;        // 1: the next inner iteration takes p = z
    int active;       // 0: converged, zero right-hand side or out of iterations: no updates
    int left;         // inner iterations this system still takes in the current run (its own
                      // count, refine_start's); at 0 it freezes
    int taken;        // inner iterations it took in the current run
};

// Right-hand sides per problem and row pairs per step of the batched
// streaming kernels (FP32 V-cycle).
constexpr int kBatchR = 4;
constexpr int kBatchK = 2;

// True when no system of problem p takes the current inner iteration: the
// batched kernels then skip the problem's work (its results would not be
// used: every one of its systems has alpha = 0 for the iteration).
__device__ __forceinline__ bool batch_frozen(const SysState* sys, int p) {
    const SysState* s = sys + (long long)p * kBatchR;
    for (int r = 0; r < kBatchR; r++)
        if (s[r].active && s[r].left > 0) return false;
    return true;
}

struct Level {
    int n = 0;            // nodes per side
    int ld = 0;           // padded row length
    long long plane = 0;  // elements per plane
    double* A64 = nullptr;
    float* A32 = nullptr;
    double* P64 = nullptr;    // interpolation from level+1 (planes on level+1's grid)
    float* P32 = nullptr;
    void* b = nullptr;        // V-cycle right-hand side (V-cycle precision)
    void* x = nullptr;        // V-cycle iterate
    void* r = nullptr;        // residual scratch
    float* cb = nullptr;      // 3-D FP32: full 27-entry rows in colour blocks (smoother)
};

struct ProfSlot {
    std::vector<cudaEvent_t> ev;   // start/end pairs
    int used = 0;
    double bytes = 0.0;
};

struct Batch;

struct Ctx {
    bmg_opts opts{};
    int dim = 2;
    int nlev = 0;
    int ns = 5, np = 8;       // stored stencil / interpolation planes
    Level lev[kMaxLevels];
    size_t ws_need = 0;
    char* ws = nullptr;
    cudaStream_t stream = nullptr;
    int device = -1;
    bool attached = false, have_op = false, have_setup = false;
    bool op_tensor = false;       // operator assembled from a diffusion tensor (no dL/dkappa)
    // finest-level FP64 Krylov vectors (internal padded layout)
    double *bvec = nullptr, *x = nullptr, *r = nullptr, *z[2] = {nullptr, nullptr};
    double *p = nullptr, *q = nullptr;
    double *stage_in = nullptr, *stage_out = nullptr;   // n^d doubles each, host staging
    // iterative refinement: FP32 inner CG vectors
    float *r32 = nullptr, *z32[2] = {nullptr, nullptr}, *p32 = nullptr, *q32 = nullptr;
    float* p32s[2] = {nullptr, nullptr};   // search directions, alternating (p is formed while p_old is read)
    float* rs32 = nullptr;        // FP32 row sums of the finest operator (difference-form products)
    FusedLevel fused_ir0;         // level-0 streaming kernels reading r32 (FP32)
    double* partials = nullptr;
    KState* st = nullptr;         // device
    KState* st_host = nullptr;    // pinned mirror
    long long launches = 0;
    int red_blocks = 0;           // fixed grid of the reducing kernels (deterministic)
    int sms = 0;                  // SMs of the device
    int nt_h = 0, nt_i = 0, nt_j = 0, nt_tiles = 0;   // node tiles of the FP64 products and residuals
    int spmv_h = 0, spmv_tiles_x = 0, spmv_tiles = 0;   // tiles of the 2-D refinement-mode operator product
    bool prof_on = false;
    ProfSlot prof[BMG_PROF_KINDS];
    bool use_fused = false;       // streaming V-cycle kernels (2-D)
    bool use_hs3 = false;         // 3-D: half-sweep kernels (one launch per colour parity of k)
    void* tail_pack = nullptr;    // operators and weights of the tail levels, packed (tail2d.cu, vcycle3d.cu)
    // CUDA graphs of one inner/outer iteration (two, for the alternating z buffers)
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t it_exec[2] = {nullptr, nullptr};
    long long it_kernels[2] = {0, 0};
    bool use_graphs = true;
    // bumped whenever launch shapes change (tile choices): graphs that other
    // objects capture around this context's kernels compare it
    unsigned long long shape_epoch = 0;
    FusedLevel fused[kMaxLevels];
    // several right-hand sides (opts.max_rhs > 1 on an eligible context): a
    // one-problem batch in a reserved part of the workspace, built on first use
    Batch* mrhs = nullptr;
    char* mrhs_ws = nullptr;
    size_t mrhs_bytes = 0;
};

// Event brackets around profiled launches (finest level only).
inline void prof_begin(Ctx& c, int kind, int level) {
    if (!c.prof_on || level != 0) return;
    ProfSlot& s = c.prof[kind];
    if ((size_t)(2 * s.used + 2) > s.ev.size()) {
        cudaEvent_t a, b;
        cudaEventCreate(&a);
        cudaEventCreate(&b);
        s.ev.push_back(a);
        s.ev.push_back(b);
    }
    cudaEventRecord(s.ev[2 * s.used], c.stream);
}

inline void prof_end(Ctx& c, int kind, int level, double bytes) {
    if (!c.prof_on || level != 0) return;
    ProfSlot& s = c.prof[kind];
    cudaEventRecord(s.ev[2 * s.used + 1], c.stream);
    s.used++;
    s.bytes += bytes;
}

// ------------------------------------------------------------------ helpers
#define BMG_CUDA(call)                                                      \
    do {                                                                    \
        cudaError_t e_ = (call);                                            \
        if (e_ != cudaSuccess) return BMG_ERR_DEVICE;                       \
    } while (0)

#define BMG_TRY(call)                                                       \
    do {                                                                    \
        bmg_status s_ = (call);                                             \
        if (s_ != BMG_OK) return s_;                                        \
    } while (0)

// Programmatic dependent launch: the kernels of an iteration are launched so
// that the next one's CTAs come up, set up their barriers and fetch what no
// kernel of the iteration writes (operators, weights) while the last CTAs of
// the one before still run.  pdl_wait() returns once every earlier kernel has
// finished and its writes are visible, so it stands before the first access to
// a vector or scalar.  __restrict__ would let the compiler take the wait for
// one that does not concern an array and move a load of it above; so in a
// waiting kernel, and in what it calls, only arrays that no kernel of the
// iteration writes (operators, weights, index lists) and arrays that this one
// writes and does not read carry it.  Without a trigger the next kernel comes up as this one's
// CTAs leave; pdl_trigger(), after the wait, calls it earlier, which pays only
// where this grid leaves SMs idle: a large one's CTAs lose their places to
// CTAs that wait (4097^2 solve 14.62 ms without triggers, 14.76 with; 65^2 1.00
// and 0.96 ms; without the attribute 14.61 and 1.03 ms).
constexpr unsigned kPdlGrid = kChipSms;
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
    if (gridDim.x * gridDim.y * gridDim.z <= kPdlGrid) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KA, typename... A>
cudaError_t launch_pdl(void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, KA(args)...);
}

// The four floats as doubles, exactly, by moving the fields of their binary32
// encoding (a normal number: exponent rebiased by 1023 - 127 = 0x380, fraction
// left-aligned; a zero keeps its sign).  Subnormal numbers, infinities and NaN,
// which are rare here, take the conversion instruction: it runs in the FP64
// units, of which an SM has two lanes' worth, and a vector update of FP32
// directions into an FP64 iterate spends half of its FP64 slots on it.
__host__ __device__ inline bool plain_f32(unsigned u) {   // zero or normal
    const unsigned t = u & 0x7fffffffu;
    return t == 0u || t - 0x00800000u < 0x7f000000u;
}
__host__ __device__ inline unsigned widen_hi(unsigned u) {
    const unsigned t = u & 0x7fffffffu;
    return (u & 0x80000000u) | (t ? (t >> 3) + 0x38000000u : 0u);
}
__host__ __device__ inline unsigned widen_lo(unsigned u) { return u << 29; }
__device__ __forceinline__ void widen4(float4 v, double* d) {
    const unsigned u[4] = {__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)};
    if (plain_f32(u[0]) && plain_f32(u[1]) && plain_f32(u[2]) && plain_f32(u[3])) {
#pragma unroll
        for (int q = 0; q < 4; q++) d[q] = __hiloint2double((int)widen_hi(u[q]), (int)widen_lo(u[q]));
    } else {
        d[0] = (double)v.x;
        d[1] = (double)v.y;
        d[2] = (double)v.z;
        d[3] = (double)v.w;
    }
}

inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

__device__ __forceinline__ void set_err(KState* st, int code) {
    atomicCAS(&st->err, 0, code);
}

// Symmetric-half 2-D stencil view.  a(i,j; dx,dy) for |dx|,|dy| <= 1.
template <typename T>
struct Sten2 {
    const T* a;
    int ld;
    long long pl;
    __device__ __forceinline__ T at(int p, int i, int j) const {
        return a[(long long)p * pl + (long long)j * ld + i];
    }
    __device__ __forceinline__ T c(int i, int j) const { return at(C2, i, j); }
    __device__ __forceinline__ T full(int i, int j, int dx, int dy) const {
        if (dx == 0 && dy == 0) return at(C2, i, j);
        if (dy == 0) return dx < 0 ? at(W2, i, j) : at(W2, i + 1, j);
        if (dx == 0) return dy < 0 ? at(S2, i, j) : at(S2, i, j + 1);
        if (dx < 0 && dy < 0) return at(SW2, i, j);
        if (dx > 0 && dy > 0) return at(SW2, i + 1, j + 1);
        if (dx < 0 && dy > 0) return at(NW2, i, j);
        return at(NW2, i + 1, j - 1);   // dx > 0, dy < 0
    }
};

// Block-wide sum (blockDim.x == kThreads) in a fixed order, valid in lane 0 of
// warp sum_warp(): one warp adds the other warps' values lane by lane and
// folds the lanes, 12 FP64 adds, where a shuffle tree in every warp takes 45 of
// the units' slots.  The warp rotates with the block, so that the blocks of an
// SM use different schedulers.
__device__ __forceinline__ int sum_warp() { return blockIdx.x % (kThreads / 32); }
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double sh[kThreads];
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    double s = 0.0;
    if ((int)(threadIdx.x >> 5) == sum_warp()) {
        const int l = threadIdx.x & 31;
        s = sh[l];
#pragma unroll
        for (int w = 1; w < kThreads / 32; w++) s += sh[l + 32 * w];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    return s;
}

// Deterministic grid reduction of N sums at once: each block stores its
// partials (N per block); the last block to arrive sums them in a fixed order.
// Returns true (in one thread of the last block only) with the totals in t.
template <int N>
__device__ __forceinline__ bool grid_sum_n(const double (&v)[N], double* partials, unsigned int* counter,
                                           double (&t)[N]) {
    __shared__ bool last;
    const bool lead = (int)threadIdx.x == 32 * sum_warp();
    double b[N];
#pragma unroll
    for (int q = 0; q < N; q++) b[q] = block_sum(v[q]);
    if (lead) {
#pragma unroll
        for (int q = 0; q < N; q++) partials[N * blockIdx.x + q] = b[q];
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int q = 0; q < N; q++) {
        double s = 0.0;
        for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) s += ((volatile double*)partials)[N * k + q];
        t[q] = block_sum(s);
    }
    if (lead) *counter = 0u;
    return lead;
}

__device__ __forceinline__ bool grid_sum2(double v1, double v2, double* partials, unsigned int* counter,
                                          double* t1, double* t2) {
    double t[2];
    if (!grid_sum_n<2>({v1, v2}, partials, counter, t)) return false;
    *t1 = t[0];
    *t2 = t[1];
    return true;
}

__device__ __forceinline__ bool grid_sum(double v, double* partials, unsigned int* counter, double* total) {
    double t[1];
    if (!grid_sum_n<1>({v}, partials, counter, t)) return false;
    *total = t[0];
    return true;
}

// ------------------------------------------------------------------ host launchers
// setup2d.cu
bmg_status assemble2d(Ctx& c, const double* coords, const double* kappa);
bmg_status assemble_tensor2d(Ctx& c, const double* coords, const double* D);
bmg_status boundary_rhs2d(Ctx& c, const double* coords, const double* kappa, const double* g, double* out);
bmg_status set_stencil2d(Ctx& c, const double* full);
bmg_status setup_level2d(Ctx& c, int l);
bmg_status export_stencil2d(Ctx& c, int l, double* out);
bmg_status export_interp2d(Ctx& c, int l, double* out);
bmg_status adjoint_cells2d(Ctx& c, const double* coords, const double* u, const double* lam, double* g);
// setup3d.cu
bmg_status assemble3d(Ctx& c, const double* coords, const double* kappa);
bmg_status assemble_tensor3d(Ctx& c, const double* coords, const double* D);
bmg_status boundary_rhs3d(Ctx& c, const double* coords, const double* kappa, const double* g, double* out);
bmg_status set_stencil3d(Ctx& c, const double* full);
bmg_status setup_level3d(Ctx& c, int l);
bmg_status export_stencil3d(Ctx& c, int l, double* out);
bmg_status export_interp3d(Ctx& c, int l, double* out);
bmg_status adjoint_cells3d(Ctx& c, const double* coords, const double* u, const double* lam, double* g);
// setup2d.cu / setup3d.cu, context-free: assembly into given half planes, then export
bmg_status assemble_export2d(int n, int ld, long long pl, const double* coords, const double* kappa, double* A,
                             KState* st, double* out, cudaStream_t s);
bmg_status assemble_export3d(int n, int ld, long long pl, const double* coords, const double* kappa, double* A,
                             KState* st, double* out, cudaStream_t s);
// batch2d.cu
bmg_status batch_attach(Batch& B, void* ws, size_t bytes, void* stream);
bmg_status batch_solve(Batch& B, int nrhs, const double* const* b, double* const* x, double tol, int maxit,
                       bmg_info* infos);
void batch_destroy(Batch* B);
size_t batch_single_bytes(Ctx& c);
bmg_status batch_single_create(Ctx& c, Batch** out);
// vcycle.cu: z = M r on the finest level (FP64 in/out, internal layout); dots
// (only where vcycle_forms_beta): the finest up kernel also forms beta from
// r.z (1) or r.z - r.zold (2)
bmg_status vcycle(Ctx& c, const double* r, double* z, const double* zold = nullptr, int dots = 0);
// fused2d.cu / tmaps.cu
int fused_rows_per_step(bool f32);
int fused_down_smem(bool f32, bool f64in, int wc);
int fused_up_smem(bool f32, bool f64in, int wc);
bmg_status fused_occupancy(bool f32, bool f64in, int wc, int* down_blocks, int* up_blocks);
bmg_status fused_down(Ctx& c, int l, bool ir = false);
bmg_status fused_up(Ctx& c, int l, void* out, bool ir = false, const void* zold = nullptr, int dots = 0);
bmg_status vcycle_f32(Ctx& c, float* z32, const float* zold = nullptr);
// batched streaming kernels (fused2d.cu): FP32, kBatchR right-hand sides, strip width 16 or 32
int batch_down_smem(int wc);
int batch_up_smem(int wc);
bmg_status batch_occupancy(int wc, int* down_blocks, int* up_blocks);
bmg_status batch_down(const CUtensorMap& mA, const CUtensorMap& mF, const FusedArgs& a, int grid, cudaStream_t s);
bmg_status batch_up(const CUtensorMap& mA, const CUtensorMap& mF, const CUtensorMap& mXp, const CUtensorMap& mXc,
                    const FusedArgs& a, int grid, cudaStream_t s);
// vcycle3d.cu: colour-blocked full rows of the FP32 levels (after demotion)
bmg_status colour_blocks3d(Ctx& c);
// interior nodes of colour col (parities col&1, col>>1&1, col>>2) on an n-grid,
// and the offset of that colour's block (27 entries per node) in Level::cb
__host__ __device__ inline int cb_side(int n, int parity) { return parity ? (n - 1) / 2 : (n - 2) / 2; }
__host__ __device__ inline long long cb_count(int n, int col) {
    return (long long)cb_side(n, col & 1) * cb_side(n, (col >> 1) & 1) * cb_side(n, col >> 2);
}
__host__ __device__ inline long long cb_offset(int n, int col) {
    long long o = 0;
    for (int q = 0; q < col; q++) o += 27 * cb_count(n, q);
    return o;
}
// tail2d.cu: the levels from the first one with n <= kTailMaxN (at least
// level 1) down to the coarsest, in one single-CTA launch
constexpr int kTailMaxN = 33;
struct TailArgs {
    int nlev;                     // levels in the tail (the last one has 3 nodes)
    int ns[kMaxLevels];           // nodes per side of each tail level
    const void* pack;             // packed operators and weights (shared-memory image)
    unsigned pack_bytes;          // its size, a multiple of 16
    const void* b0;               // right-hand side of the first tail level
    void* x0;                     // finished iterate of the first tail level
    int ld0;                      // row length of b0 and x0 (in nodes)
    const double* a64c;           // FP64 centre entry of the coarsest operator
    KState* st;
    const SysState* sys = nullptr;   // batched: the problem's systems (skips a frozen problem)
};
int tail_first_level(const Ctx& c);
bmg_status tail_args(const Ctx& c, const void* b0, void* x0, int ld0, KState* st, TailArgs* a);
size_t batch_tail_smem(const int* ns, int L);
bmg_status batch_tail(const TailArgs* args, int count, size_t smem, cudaStream_t s);
size_t tail_smem_bytes(const Ctx& c, int t);
size_t tail_pack_bytes(const Ctx& c);             // packed tail operators (0 outside 2-D)
bmg_status tail_pack(Ctx& c);                     // fills c.tail_pack (bmg_setup)
bmg_status tail_vcycle(Ctx& c, int t);
size_t tail3_pack_bytes(const Ctx& c);            // the same for the 3-D tail (vcycle3d.cu)
bmg_status tail3_pack(Ctx& c);
// whether the streaming kernels' finest up kernel can form beta (its tiles'
// sums fit the partials)
bool vcycle_forms_beta(const Ctx& c);
template <typename T>
bmg_status vcycle3d_impl(Ctx& c, const T* b0, T* x0);
bmg_status fused_prepare(Ctx& c);
bmg_status fused_configure(Ctx& c, int l, int wc, int hc, int hc_up);
bmg_status fused_autotune(Ctx& c, int reps, double* best_ms_total);
bmg_status demote_levels(Ctx& c);
bmg_status invert_diagonals(Ctx& c);   // FP64 contexts: 1 / diagonal into the plane behind every level's operator
// krylov.cu
bmg_status k_pack(Ctx& c, const double* src, double* dst);      // n^d -> padded, boundary zeroed
bmg_status k_unpack(Ctx& c, const double* src, double* dst);    // padded -> n^d
bmg_status k_residual(Ctx& c, const double* b, const double* x, double* r);  // r = b - A x; st.rr
bmg_status k_dot(Ctx& c, const double* a, const double* b, double* slot);    // *slot (device) = a.b
bmg_status k_spmv_pq(Ctx& c, const double* p, double* q);        // q = A p; alpha = rz / p.q
bmg_status k_update_xr(Ctx& c);                                   // x += alpha p; r -= alpha q; rr
bmg_status k_rz_beta(Ctx& c, const double* z, const double* zold, bool flexible);
bmg_status k_p_update(Ctx& c, const double* z);                   // p = z + beta p (or z)
// FP32 inner CG of the refinement mode
bmg_status k_row_sums32(Ctx& c);                // rs32 = row sums of A (computed in FP64)
bmg_status k_residual_to32(Ctx& c);             // r32 = (float)(b - A x); rr; resets the inner CG state
bmg_status k_rz_beta32(Ctx& c, const float* z, const float* zo);
bmg_status k_update_dr32(Ctx& c, int parity);    // r32 -= alpha q; odd parity: x (FP64) += both iterations' alpha p
// run lengths of the refinement mode, single, concurrent and batched (api.cu)
constexpr double kRefineFloor = 1e-6;   // reduction one FP32 inner solve can deliver
int refine_start(double want, double rho, int left);
int refine_next(const KState& h, double want, double rho, int done, int left);
double refine_rho(double rho, double red, int m);
bmg_status k_flush_dr32(Ctx& c);                 // x += the step an even last iteration left
bmg_status node_tiles_prepare(Ctx& c);           // tile shape of the FP64 products and residuals
bmg_status pspmv_prepare(Ctx& c);                // tile shape of the 2-D operator product
bmg_status k_pspmv32(Ctx& c, const float* z, int parity);   // p = z + beta p_old; q = A p; alpha

}  // namespace bmg

// The opaque context of the C ABI.
struct bmg_ctx {
    bmg::Ctx c;
};
