// batched.cu -- PCG on K right-hand sides at once (independent columns in lockstep).
//
// Block vectors are row-major [n][Kp].  Kp = K rounded up to 8 or 16, or to a multiple of 32: a warp owns
// one row of 32 J columns (lane l the J columns from l J on, one vector load), or for K <= 16 the R = 4
// or 2 rows that fill its lanes, since a warp instruction costs the same with idle lanes and FP64 issue
// is scarce on this part (the FP32 preconditioner's kernels take more rows to a warp, see Gather).  Every matrix entry is one broadcast load shared by all columns, and every
// gathered vector row is one coalesced load.  The matrix is read once per K solves instead of once per
// solve (SpMM).  Each column has its own alpha, beta and convergence flag; a converged column is frozen
// (alpha = 0) while the others continue, so each column reproduces the single-right-hand-side
// iteration.  Reductions are per column and finish in a fixed order.  The preconditioner is the
// handle's, applied column-wise by the same algorithms (Algorithm 2.1 with Algorithm 3.2 and the IC(0)
// solves); in FP32 it reads an FP32 copy of the residual, made once where the residual is updated
// (FP64 to FP32 conversions issue at FP64 rate, and each application read the residual five times).
#include <algorithm>
#include <type_traits>
#include <utility>

#include "device.cuh"
#include "handle.cuh"

namespace cpc {

namespace {

constexpr int BWARPS = 4;                 // warps per block of the SELL kernels, a row each
constexpr int BTPB = BWARPS * 32;
// Warps per block of the diagonal-form kernels and the vector passes.  Blocks start at about one a
// nanosecond on this part, which bounded these short rows at four warps a block (131,072 blocks: a fine
// colour step of 64 columns 135 us, 112 with 16 warps); the SELL kernels are slower in larger blocks
// (a level-1 colour step 41 and 51 us).
constexpr int DWARPS = 16;
constexpr int DTPB = DWARPS * 32;
constexpr int VWARPS = 8;                 // warps per block of the PCG vector kernels
constexpr int VTPB = VWARPS * 32;
constexpr int WSPLIT = 4;                 // warps that share a row in kb_gs_wide
constexpr int NB_STATE = 12;              // per-column scalar slots

// column-state layout: S[slot * Kp + col]
enum { S_BNORM = 0, S_RZ, S_RZOLD, S_PQ, S_ALPHA, S_BETA, S_RES, S_ACTIVE, S_K, S_STATUS, S_TOL, S_MAXIT };

template <class MT, class DT>
struct BV {                               // SELL view for the batched kernels
    int C;
    const int* __restrict__ perm;
    const int* __restrict__ cptr;
    const int* __restrict__ col;
    const MT* __restrict__ val;
    const DT* __restrict__ diag;
};

template <class MT, class DT>
BV<MT, DT> bview(const Sell& S, const MT* val, const DT* diag) {
    return BV<MT, DT>{S.C, S.perm.p, S.cptr.p, S.col.p, val, diag};
}

template <class... KArgs, class... Args>
void blaunch(void (*k)(KArgs...), int grid, int block, cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)std::max(1, grid), 1, 1);
    cfg.blockDim = dim3((unsigned)block, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CPC_CK(cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...));
}

// The columns of a lane: a warp holds R rows of 32 J / R columns, J neighbouring ones to a lane.
template <int J, int R>
struct Cols {
    static constexpr int W = 32 / R, KP = W * J;
    static __device__ __forceinline__ int sub() { return R == 1 ? 0 : (threadIdx.x & 31) / W; }
    static __device__ __forceinline__ int col() { return (R == 1 ? threadIdx.x & 31 : (threadIdx.x & 31) % W) * J; }
    // element of (row, the lane's first column)
    static __device__ __forceinline__ size_t at(int row) { return (size_t)row * KP + col(); }
};

// The columns of a lane in the preconditioner's kernels.  In FP32 they gather 16 bytes to a lane from two or
// four rows at a time (8 bytes for up to 16 columns), so that half or a quarter of the load instructions
// move the same bytes; a column's sums are the same.  64 solves and adjoints at 1M 255 -> 221 ms, 28 at 433k
// cells 87 -> 64 ms, 16 at 1M 148 -> 123 ms, 8 at 1M 98 -> 91 ms, 12 at 131k cells 28.0 -> 26.3 ms (with four
// columns to a lane 29.9).  Not in FP64, whose issue bounds them: fewer warps only lose (12 columns of a block
// solve 22.9 -> 27.9 ms, 32 at 590k cells 157 -> 159 ms).
template <int J, int R, class VT>
struct Gather {
    static constexpr int M = !std::is_same<VT, float>::value ? 1 : R == 1 && J <= 2 ? 4 / J : R >= 2 ? 2 : 1;
    static constexpr int j = J * M, r = R * M;
};

template <int J, class VT, class T>
__device__ __forceinline__ void ldv(const T* p, VT (&v)[J]) {
    if constexpr (std::is_same<T, float>::value && J == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        v[0] = Cv<VT>::f(t.x);
        v[1] = Cv<VT>::f(t.y);
    } else if constexpr (std::is_same<T, float>::value && J == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = Cv<VT>::f(t.x);
        v[1] = Cv<VT>::f(t.y);
        v[2] = Cv<VT>::f(t.z);
        v[3] = Cv<VT>::f(t.w);
    } else if constexpr (std::is_same<T, double>::value && J % 2 == 0) {
#pragma unroll
        for (int j = 0; j < J; j += 2) {
            const double2 t = *reinterpret_cast<const double2*>(p + j);
            v[j] = Cv<VT>::f(t.x);
            v[j + 1] = Cv<VT>::f(t.y);
        }
    } else {
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] = Cv<VT>::f(p[j]);
    }
}

template <int J, class T>
__device__ __forceinline__ void stv(T* p, const T (&v)[J]) {
    if constexpr (std::is_same<T, float>::value && J == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    } else if constexpr (std::is_same<T, float>::value && J == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (std::is_same<T, double>::value && J % 2 == 0) {
#pragma unroll
        for (int j = 0; j < J; j += 2) *reinterpret_cast<double2*>(p + j) = make_double2(v[j], v[j + 1]);
    } else {
#pragma unroll
        for (int j = 0; j < J; ++j) p[j] = v[j];
    }
}

// Blocks for nrows rows, one row per warp lane group.
template <int R>
inline int rows_grid(int nrows, int warps = BWARPS) { return (nrows + warps * R - 1) / (warps * R); }

// Calls f(std::integral_constant<int, ND>{}) with the padded diagonal count (4, 6 or 8).
template <class F>
void bwith_nd(int nd, F&& f) {
    if (nd <= 4) f(std::integral_constant<int, 4>{});
    else if (nd <= 6) f(std::integral_constant<int, 6>{});
    else f(std::integral_constant<int, 8>{});
}

// The row in slot s of a SELL layout: entries base + w C + r, w < width.
struct BRow {
    int base, width, r, C;
};
template <class MT, class DT>
__device__ __forceinline__ BRow brow_at(const BV<MT, DT>& A, int s, const int* end) {
    const int k = s / A.C;
    const int base = A.cptr[k];
    return BRow{base, (end[k] - base) / A.C, s - k * A.C, A.C};
}

// Columns and values of U entries w, w + step, ... of a row (past its end: column -1, value 0).
template <int U, class VT>
struct Entries {
    int c[U];
    VT a[U];
    template <class MT>
    __device__ __forceinline__ void load(const int* __restrict__ col, const MT* __restrict__ val, const BRow& t, int w, int step) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool on = w + u * step < t.width;
            const int e = t.base + (w + u * step) * t.C + t.r;
            c[u] = on ? col[e] : -1;
            a[u] = on ? Cv<VT>::f(val[e]) : VT(0);
        }
    }
};

// acc[j] += sum_w a_w x[col_w][j] over entries w0, w0 + step, ... of a row, U entries' gathers in flight
// together and the next entries' columns beside them; m holds the first ones, loaded by the caller before it
// waits for x.  Padding (-1) and marked columns (below -1) load nothing and add 0.  (With each batch's columns
// loaded before its own gathers a row cost two trips through L2 per batch and one more after the wait:
// 64 solves and adjoints at 1M 220 -> 203 ms, 28 at 433k cells 63.6 -> 53.2, a block solve of 12 22.9 -> 20.7.)
template <int J, int R, int U, class VT, class MT, class XT>
__device__ __forceinline__ void brow(const int* __restrict__ col, const MT* __restrict__ val, const BRow& t, int w0,
                                     int step, Entries<U, VT>& m, const XT* x, VT (&acc)[J]) {
    using L = Cols<J, R>;
    for (int w = w0; w < t.width; w += U * step) {
        VT xv[U][J];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (takes(m.c[u])) {
                ldv<J>(x + L::at(m.c[u]), xv[u]);
            } else {
#pragma unroll
                for (int j = 0; j < J; ++j) xv[u][j] = VT(0);
            }
        }
        Entries<U, VT> next;
        next.load(col, val, t, w + U * step, step);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < J; ++j) acc[j] += m.a[u] * xv[u][j];
        m = next;
    }
}

template <int J, class VT>
__device__ __forceinline__ void zero(VT (&v)[J]) {
#pragma unroll
    for (int j = 0; j < J; ++j) v[j] = VT(0);
}

// Gauss-Seidel over the slots [s0, s1) of one colour, all columns; the entries of a row end at end[k]
// (its chunk's last; in a sweep from a zero guess the entries of later colours, whose rows are zero, are
// left out: by end in FP64, by their mark in FP32).
template <int J, int R, class MT, class DT, class VT>
__global__ void __launch_bounds__(BTPB) kb_gs(BV<MT, DT> A, const int* __restrict__ end, int s0, int s1, const VT* f, VT* x) {
    using L = Cols<J, R>;
    const int s = s0 + (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= s1) return;
    pdl_launch_dependents();
    const int row = A.perm[s];                   // matrix data: before the wait
    const BRow t = brow_at(A, s, end);
    const VT dinv = Cv<VT>::f(A.diag[s]);        // the view's diagonal field holds 1 / a_ii
    Entries<4, VT> m;
    m.load(A.col, A.val, t, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J], fr[J];
    zero(acc);
    ldv<J>(f + L::at(row), fr);
    brow<J, R, 4>(A.col, A.val, t, 0, 1, m, x, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = (fr[j] - acc[j]) * dinv;
    stv<J>(x + L::at(row), acc);
}

// Gauss-Seidel for long rows in small colour groups (coarse levels): WSPLIT warps per R rows, warp w
// taking the entries w, w + WSPLIT, ...; the warps' partial sums are added in warp order through
// shared memory.  A step of a few thousand rows then costs a quarter of a row's chain of dependent
// loads instead of a whole one.  A block holds two such sets.
template <int J, int R, class MT, class DT, class VT>
__global__ void __launch_bounds__(64 * WSPLIT) kb_gs_wide(BV<MT, DT> A, const int* __restrict__ end, int s0, int s1,
                                                          const VT* f, VT* x) {
    using L = Cols<J, R>;
    __shared__ VT part[2][WSPLIT][J][32];
    const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) % WSPLIT, set = (threadIdx.x >> 5) / WSPLIT;
    const int sr = s0 + ((int)blockIdx.x * 2 + set) * R + L::sub();
    const int s = min(sr, s1 - 1);                           // (a repeated row is not written)
    pdl_launch_dependents();
    const int row = A.perm[s];
    const BRow t = brow_at(A, s, end);
    const VT dinv = Cv<VT>::f(A.diag[s]);
    Entries<4, VT> m;
    m.load(A.col, A.val, t, w, WSPLIT);
    pdl_wait();
    VT acc[J], fr[J];
    zero(acc);
    zero(fr);
    if (w == 0 && row >= 0) ldv<J>(f + L::at(row), fr);
    brow<J, R, 4>(A.col, A.val, t, w, WSPLIT, m, x, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) part[set][w][j][lane] = acc[j];
    __syncthreads();
    if (w != 0 || row < 0 || sr >= s1) return;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        VT v = part[set][0][j][lane];
        for (int q = 1; q < WSPLIT; ++q) v += part[set][q][j][lane];
        acc[j] = (fr[j] - v) * dinv;
    }
    stv<J>(x + L::at(row), acc);
}

// out = f - A x over all slots.
template <int J, int R, class MT, class DT, class VT>
__global__ void __launch_bounds__(BTPB) kb_resid(BV<MT, DT> A, int nslots, const VT* f, const VT* x, VT* __restrict__ out) {
    using L = Cols<J, R>;
    const int s = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= nslots) return;
    pdl_launch_dependents();
    const int row = A.perm[s];
    const BRow t = brow_at(A, s, A.cptr + 1);
    const VT d = Cv<VT>::f(A.diag[s]);
    Entries<4, VT> m;
    m.load(A.col, A.val, t, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J], fr[J];
    ldv<J>(x + L::at(row), acc);
    ldv<J>(f + L::at(row), fr);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] *= d;
    brow<J, R, 4>(A.col, A.val, t, 0, 1, m, x, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = fr[j] - acc[j];
    stv<J>(out + L::at(row), acc);
}

// out = f - A x after a forward sweep from a zero guess: (D + L) x = f holds row by row, so only the
// entries of later colours (from cmid on) are read, out_i = -sum_up a_ij x_j.
template <int J, int R, class MT, class DT, class VT>
__global__ void __launch_bounds__(BTPB) kb_resid_up(BV<MT, DT> A, const int* __restrict__ cmid, int nslots, const VT* x,
                                                    VT* __restrict__ out) {
    using L = Cols<J, R>;
    const int s = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= nslots) return;
    pdl_launch_dependents();
    const int row = A.perm[s];
    const int k = s / A.C, base = cmid[k];
    const BRow t{base, (A.cptr[k + 1] - base) / A.C, s - k * A.C, A.C};
    Entries<4, VT> m;
    m.load(A.col, A.val, t, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J];
    zero(acc);
    brow<J, R, 4>(A.col, A.val, t, 0, 1, m, x, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = -acc[j];
    stv<J>(out + L::at(row), acc);
}

// f_c = R r (entries up to end[k]: all, or the red columns of the finest level) and, with yx, the coarse
// level's first colour step from zero, x_c = f_c / a_ii on colour 0 (the sweep does not read the others).
template <int J, int R, class MT, class VT>
__global__ void __launch_bounds__(BTPB) kb_restrict(BV<MT, MT> M, const int* __restrict__ end, int nslots, const VT* x,
                                                    VT* __restrict__ y, VT* __restrict__ yx,
                                                    const int* __restrict__ colour, const VT* __restrict__ dnat) {
    using L = Cols<J, R>;
    const int s = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= nslots) return;
    pdl_launch_dependents();
    const int row = M.perm[s];
    const BRow t = brow_at(M, s, end);
    const bool c0 = yx && row >= 0 && colour[row] == 0;
    const VT dr = c0 ? dnat[row] : VT(0);
    Entries<4, VT> m;
    m.load(M.col, M.val, t, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J];
    zero(acc);
    brow<J, R, 4>(M.col, M.val, t, 0, 1, m, x, acc);
    stv<J>(y + L::at(row), acc);
    if (!c0) return;
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] *= dr;
    stv<J>(yx + L::at(row), acc);
}

// x += P e on the rows of slots [0, nslots)
template <int J, int R, class MT, class VT>
__global__ void __launch_bounds__(BTPB) kb_prolong(BV<MT, MT> P, int nslots, const VT* e, VT* __restrict__ x) {
    using L = Cols<J, R>;
    const int s = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= nslots) return;
    pdl_launch_dependents();
    const int row = P.perm[s];
    const BRow t = brow_at(P, s, P.cptr + 1);
    Entries<4, VT> m;
    m.load(P.col, P.val, t, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J], xr[J];
    zero(acc);
    ldv<J>(x + L::at(row), xr);
    brow<J, R, 4>(P.col, P.val, t, 0, 1, m, e, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] += xr[j];
    stv<J>(x + L::at(row), acc);
}

// x = A_c^{-1} f (dense) in FP64: a block per R * CROWS rows, its warps sharing the columns of A_c^{-1} in
// contiguous parts (one warp per row is a chain of 1,800 FP64 operations, 113 us; 17 this way), the partial
// sums added in warp order.  A warp takes CROWS rows at a time, since f is read from L2 once per block.
constexpr int CROWS = 4, CWARPS = 8;
template <int J, int R, class AT, class FT, class VT>
__global__ void __launch_bounds__(CWARPS * 32) kb_coarse(int n, const AT* __restrict__ Ainv, const FT* f, VT* __restrict__ x) {
    using L = Cols<J, R>;
    __shared__ VT part[CWARPS][CROWS][J][32];
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i0 = (blockIdx.x * R + L::sub()) * CROWS;
    const int per = (n + CWARPS - 1) / CWARPS, m0 = w * per, m1 = min(n, m0 + per);
    pdl_wait();
    VT acc[CROWS][J];
#pragma unroll
    for (int q = 0; q < CROWS; ++q) zero(acc[q]);
#pragma unroll 4
    for (int m = m0; m < m1; ++m) {
        VT fv[J];
        ldv<J>(f + L::at(m), fv);
#pragma unroll
        for (int q = 0; q < CROWS; ++q) {
            const VT a = i0 + q < n ? Cv<VT>::f(Ainv[(size_t)(i0 + q) * n + m]) : VT(0);
#pragma unroll
            for (int j = 0; j < J; ++j) acc[q][j] += a * fv[j];
        }
    }
#pragma unroll
    for (int q = 0; q < CROWS; ++q)
#pragma unroll
        for (int j = 0; j < J; ++j) part[w][q][j][lane] = acc[q][j];
    __syncthreads();
    if (w >= CROWS || i0 + w >= n) return;                  // warp q adds up row q
    VT v[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        v[j] = part[0][w][j][lane];
        for (int q = 1; q < CWARPS; ++q) v[j] += part[q][w][j][lane];
    }
    stv<J>(x + L::at(i0 + w), v);
}

// The same in FP32, a warp per SROWS R rows, each sum taken in column order by one lane.  f (466 KB for 64 FP32 columns at 1M) and the block's rows of A_c^{-1} pass
// through shared memory in tiles of CTILE columns, the next tile's loads in flight with the products: from
// L2 the sum is a chain of 1,823 loads, read once per row (107 us; 50 this way, 45 in FP64's order).
constexpr int SROWS = 2, CTILE = 32;
template <int J, int R, class AT, class FT, class VT>
__global__ void __launch_bounds__(CWARPS * 32) kb_coarse_seq(int n, const AT* __restrict__ Ainv, const FT* f, VT* __restrict__ x) {
    using L = Cols<J, R>;
    constexpr int KP = L::KP, ROWS = CWARPS * R * SROWS, TPB = CWARPS * 32;
    constexpr int FPT = (CTILE * KP + TPB - 1) / TPB, APT = (ROWS * CTILE + TPB - 1) / TPB;
    __shared__ __align__(16) VT fs[CTILE * KP];          // read by ldv, up to 16 bytes at a time
    __shared__ VT as[ROWS][CTILE + 1];
    pdl_launch_dependents();
    const int t = threadIdx.x, b0 = blockIdx.x * ROWS;
    const int r0 = ((t >> 5) * R + L::sub()) * SROWS;       // the lane's rows within the block
    VT fv[FPT], av[APT], acc[SROWS][J];
#pragma unroll
    for (int q = 0; q < SROWS; ++q) zero(acc[q]);
    auto load_a = [&](int m0) {
#pragma unroll
        for (int u = 0; u < APT; ++u) {
            const int e = t + u * TPB, r = e / CTILE, c = e % CTILE;
            av[u] = r < ROWS && b0 + r < n && m0 + c < n ? Cv<VT>::f(Ainv[(size_t)(b0 + r) * n + m0 + c]) : VT(0);
        }
    };
    auto load_f = [&](int m0) {
#pragma unroll
        for (int u = 0; u < FPT; ++u) {
            const int e = t + u * TPB;
            fv[u] = e < CTILE * KP && m0 + e / KP < n ? Cv<VT>::f(f[(size_t)m0 * KP + e]) : VT(0);
        }
    };
    load_a(0);
    pdl_wait();
    load_f(0);
    for (int m0 = 0; m0 < n; m0 += CTILE) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < FPT; ++u)
            if (t + u * TPB < CTILE * KP) fs[t + u * TPB] = fv[u];
#pragma unroll
        for (int u = 0; u < APT; ++u) {
            const int e = t + u * TPB;
            if (e / CTILE < ROWS) as[e / CTILE][e % CTILE] = av[u];
        }
        __syncthreads();
        if (m0 + CTILE < n) {
            load_a(m0 + CTILE);
            load_f(m0 + CTILE);
        }
        const int mc = min(CTILE, n - m0);
#pragma unroll 8
        for (int m = 0; m < mc; ++m) {
            VT v[J];
            ldv<J>(fs + m * KP + L::col(), v);
#pragma unroll
            for (int q = 0; q < SROWS; ++q)
#pragma unroll
                for (int j = 0; j < J; ++j) acc[q][j] += as[r0 + q][m] * v[j];
        }
    }
#pragma unroll
    for (int q = 0; q < SROWS; ++q)
        if (b0 + r0 + q < n) stv<J>(x + L::at(b0 + r0 + q), acc[q]);
}

// Triangular solves of one IC(0) level, all columns: y = t - L y; w = (y - U w) / d, z += w.
template <int J, int R, class MT, class VT>
__global__ void __launch_bounds__(BTPB) kb_lsolve(BV<MT, MT> A, int s0, int s1, const VT* t, VT* y) {
    using L = Cols<J, R>;
    const int s = s0 + (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= s1) return;
    pdl_launch_dependents();
    const int row = A.perm[s];
    const BRow b = brow_at(A, s, A.cptr + 1);
    Entries<4, VT> m;
    m.load(A.col, A.val, b, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J], tr[J];
    zero(acc);
    ldv<J>(t + L::at(row), tr);
    brow<J, R, 4>(A.col, A.val, b, 0, 1, m, y, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = tr[j] - acc[j];
    stv<J>(y + L::at(row), acc);
}

template <int J, int R, class MT, class VT>
__global__ void __launch_bounds__(BTPB) kb_usolve(BV<MT, MT> U, int s0, int s1, const VT* y, VT* w, VT* zadd) {
    using L = Cols<J, R>;
    const int s = s0 + (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= s1) return;
    pdl_launch_dependents();
    const int row = U.perm[s];
    const BRow b = brow_at(U, s, U.cptr + 1);
    const VT dinv = Cv<VT>::f(U.diag[s]);        // 1 / u_ii
    Entries<4, VT> m;
    m.load(U.col, U.val, b, 0, 1);
    pdl_wait();
    if (row < 0) return;
    VT acc[J], yr[J];
    zero(acc);
    ldv<J>(y + L::at(row), yr);
    brow<J, R, 4>(U.col, U.val, b, 0, 1, m, w, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = (yr[j] - acc[j]) * dinv;
    stv<J>(w + L::at(row), acc);
    if (!zadd) return;
    VT z[J];
    ldv<J>(zadd + L::at(row), z);
#pragma unroll
    for (int j = 0; j < J; ++j) z[j] += acc[j];
    stv<J>(zadd + L::at(row), z);
}

// ---------------------------------------------------------------------------------------------
// Diagonal form (Sell::ndiag > 0, structured fine level): the gathered rows are x[i + off_d], so a
// warp needs only its row index before it issues every gather, and the matrix values (one
// broadcast load per diagonal) and 1 / a_ii are loaded before griddepcontrol.wait.  Products are
// added in ascending column order, as in brow.
// ---------------------------------------------------------------------------------------------
template <class MT, class DT>
struct BD {
    int n, nslots;
    const int* __restrict__ perm;      // nullptr: natural order
    const MT* __restrict__ val;        // [ND][nslots]
    const DT* __restrict__ diag;
    DiaOff off;
};

template <class MT, class DT>
BD<MT, DT> bdview(const Sell& S, int n, const MT* val, const DT* diag, bool natural) {
    return BD<MT, DT>{n, S.nslots, natural ? nullptr : S.perm.p, val, diag, S.doff};
}

template <class MT, class DT>
__device__ __forceinline__ int bd_row(const BD<MT, DT>& A, int s) {
    return A.perm ? A.perm[s] : (s < A.n ? s : -1);
}

// acc[j] += sum_d v_d x[i + off_d][j] (all gathers issued before the products)
template <int J, int R, int ND, class VT, class XT>
__device__ __forceinline__ void bd_dot(const VT (&v)[ND], const DiaOff& off, int row, int n, const XT* x, VT (&acc)[J]) {
    VT xv[ND][J];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        int jr = row + off.o[d];
        jr = jr < 0 ? 0 : (jr >= n ? n - 1 : jr);
        ldv<J>(x + Cols<J, R>::at(jr), xv[d]);
    }
#pragma unroll
    for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int j = 0; j < J; ++j) acc[j] += v[d] * xv[d][j];
}

template <int J, int R, class MT, class DT, class VT, int ND>
__global__ void __launch_bounds__(DTPB) kb_gs_dia(BD<MT, DT> A, int s0, int s1, const VT* f, VT* x) {
    using L = Cols<J, R>;
    const int s = s0 + (blockIdx.x * DWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= s1) return;
    pdl_launch_dependents();
    const int row = bd_row(A, s);
    VT v[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) v[d] = Cv<VT>::f(A.val[(size_t)d * A.nslots + s]);
    const VT dinv = Cv<VT>::f(A.diag[s]);        // 1 / a_ii
    pdl_wait();
    if (row < 0) return;
    VT fr[J], acc[J];
    zero(acc);
    ldv<J>(f + L::at(row), fr);
    bd_dot<J, R, ND>(v, A.off, row, A.n, x, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = (fr[j] - acc[j]) * dinv;
    stv<J>(x + L::at(row), acc);
}

// out = f - A x on slots [0, s1), diagonal form.  ZERO: after a forward sweep from a zero guess on the
// first of two colours, whose f_i - a_ii x_i is 0.
template <int J, int R, class MT, class DT, class FT, class VT, int ND, bool ZERO>
__global__ void __launch_bounds__(DTPB) kb_resid_dia(BD<MT, DT> A, int s1, const FT* f, const VT* x, VT* __restrict__ out) {
    using L = Cols<J, R>;
    const int s = (blockIdx.x * DWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= s1) return;
    pdl_launch_dependents();
    const int row = bd_row(A, s);
    VT v[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) v[d] = Cv<VT>::f(A.val[(size_t)d * A.nslots + s]);
    const VT dg = Cv<VT>::f(A.diag[s]);
    pdl_wait();
    if (row < 0) return;
    VT acc[J], fr[J];
    zero(acc);
    zero(fr);
    if (!ZERO) {
        ldv<J>(x + L::at(row), acc);
        ldv<J>(f + L::at(row), fr);
#pragma unroll
        for (int j = 0; j < J; ++j) acc[j] *= dg;
    }
    bd_dot<J, R, ND>(v, A.off, row, A.n, x, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = fr[j] - acc[j];
    stv<J>(out + L::at(row), acc);
}

// B_co step (2) with red-black IC(0), black rows only (see the single right-hand-side path):
// z_b += (r_b - (A z)_b) / u_bb on the fine colour 1, diagonal form.
template <int J, int R, class MT, class DT, class VT, int ND>
__global__ void __launch_bounds__(DTPB) kb_bco_black_dia(BD<MT, DT> A, int s0, int s1, const VT* r,
                                                          const VT* __restrict__ uinv, VT* __restrict__ z) {
    using L = Cols<J, R>;
    const int s = s0 + (blockIdx.x * DWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (s >= s1) return;
    pdl_launch_dependents();
    const int row = bd_row(A, s);
    VT v[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) v[d] = Cv<VT>::f(A.val[(size_t)d * A.nslots + s]);
    const VT dg = Cv<VT>::f(A.diag[s]);
    const VT ui = row >= 0 ? uinv[row] : VT(0);
    pdl_wait();
    if (row < 0) return;
    VT zr[J], rr[J], acc[J];
    ldv<J>(z + L::at(row), zr);
    ldv<J>(r + L::at(row), rr);
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j] = dg * zr[j];
    bd_dot<J, R, ND>(v, A.off, row, A.n, z, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) zr[j] += (rr[j] - acc[j]) * ui;
    stv<J>(z + L::at(row), zr);
}

// First colour step of a sweep from a zero guess: x = f / a_ii on colour 0; the other rows are set to 0
// (the diagonal form gathers them with the value 0, and what a buffer held before may not be finite).
template <int J, int R, class VT>
__global__ void __launch_bounds__(DTPB) kb_first(int n, const VT* f, const int* __restrict__ colour,
                                                 const VT* __restrict__ dnat, VT* __restrict__ x) {
    using L = Cols<J, R>;
    const int i = (blockIdx.x * DWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (i >= n) return;
    pdl_launch_dependents();
    const bool c0 = colour[i] == 0;
    const VT d = dnat[i];
    pdl_wait();
    VT v[J];
    zero(v);
    if (c0) {
        ldv<J>(f + L::at(i), v);
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] *= d;
    }
    stv<J>(x + L::at(i), v);
}

// ---------------------------------------------------------------------------------------------
// Per-column reductions, in an order that depends on the number of rows alone: the rows are dealt to
// 4 vblocks(n) lane groups (row i to group i mod 4 vblocks), the groups are added by fours in order, and
// the last block adds these partial rows and runs `fin` per column.  How many groups a block holds (its
// warps times the rows of a warp) does not show in the sums.  ordered (FP32 preconditioner, see
// Level::skip_zeros): the partial rows are added one after another, a chain of 1,216 FP64 sums with the
// loads of the next rows beside it; else in parts by all threads, the parts in order.  One thread per
// column with one load in flight took 0.1 ms, three times an iteration.
// ---------------------------------------------------------------------------------------------
constexpr int VBLOCKS = 152 * 8;
__host__ __device__ inline int vblocks(int n) { return min(VBLOCKS, (n + 3) / 4); }
// Blocks for a pass over n rows.
template <int R>
inline int vgrid(int n) { return (vblocks(n) * 4 + VWARPS * R - 1) / (VWARPS * R); }
// The lane group's first row (none at or beyond n for a group past the last).
template <int J, int R>
__device__ __forceinline__ int vfirst(int n) {
    const int g = (blockIdx.x * VWARPS + (threadIdx.x >> 5)) * R + Cols<J, R>::sub();
    return g < vblocks(n) * 4 ? g : n;
}

// Rows whose loads a warp keeps in flight together: u of them, fewer where a lane has more columns.  The
// order of the sums is that of one row after another.  (64 columns at 1M, 608 blocks, one row against u:
// r.z 0.53 -> 0.31 ms, p 0.57 -> 0.24 ms, an iteration 9.84 -> 9.16 ms.)
__host__ __device__ constexpr int vrows(int J, int u) { return J <= 2 ? u : u / 2; }

template <int J, int R, class Fin>
__device__ void col_finish(int n, bool ordered, double (&v)[J], double* part, unsigned* ctr, Fin fin) {
    constexpr int KP = Cols<J, R>::KP, SETS = VWARPS * R / 4;
    __shared__ double sh[VWARPS * 128];
    __shared__ bool last;
    const int w = threadIdx.x >> 5, G = vblocks(n);
    const int sub = Cols<J, R>::sub(), col = Cols<J, R>::col();
#pragma unroll
    for (int j = 0; j < J; ++j) sh[(w * R + sub) * KP + col + j] = v[j];
    __syncthreads();
    for (int e = threadIdx.x; e < SETS * KP; e += VTPB) {
        const int b = e / KP, c = e % KP;
        if ((int)blockIdx.x * SETS + b >= G) break;
        double t = 0.0;
        for (int q = 0; q < 4; ++q) t += sh[(4 * b + q) * KP + c];
        part[((size_t)blockIdx.x * SETS + b) * KP + c] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ctr, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    constexpr int PER = 8;
    if (!ordered) {
        constexpr int PARTS = VTPB / KP;                     // (96 columns: some threads idle)
        const int per = (G + PARTS - 1) / PARTS, c = threadIdx.x % KP, p = threadIdx.x / KP, b1 = min(G, (p + 1) * per);
        double t = 0.0;
        if (p < PARTS)
            for (int b = p * per; b < b1; b += 2 * PER) {
                double u[2 * PER];
#pragma unroll
                for (int q = 0; q < 2 * PER; ++q) u[q] = b + q < b1 ? __ldcg(&part[(size_t)(b + q) * KP + c]) : 0.0;
#pragma unroll
                for (int q = 0; q < 2 * PER; ++q) t += u[q];
            }
        sh[threadIdx.x] = t;
        __syncthreads();
        if ((int)threadIdx.x < KP) {
            for (int q = 1; q < PARTS; ++q) t += sh[q * KP + threadIdx.x];
            fin(threadIdx.x, t);
        }
    } else {
        // tiles of rows through shared memory, the next one's loads in flight with a column's chain of sums
        constexpr int TILE = VTPB * PER / KP > VWARPS * 128 / KP ? VWARPS * 128 / KP : VTPB * PER / KP;
        double u[PER], t = 0.0;
        auto load = [&](int b) {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int e = (int)threadIdx.x + q * VTPB;
                u[q] = e < TILE * KP && b + e / KP < G ? __ldcg(&part[(size_t)b * KP + e]) : 0.0;
            }
        };
        load(0);
        for (int b = 0; b < G; b += TILE) {
            __syncthreads();
#pragma unroll
            for (int q = 0; q < PER; ++q)
                if ((int)threadIdx.x + q * VTPB < TILE * KP) sh[threadIdx.x + q * VTPB] = u[q];
            __syncthreads();
            if (b + TILE < G) load(b + TILE);
            if ((int)threadIdx.x < KP) {                     // (rows past the last are 0: t + 0 = t)
#pragma unroll
                for (int q = 0; q < TILE; ++q) t += sh[q * KP + threadIdx.x];
            }
        }
        if ((int)threadIdx.x < KP) fin(threadIdx.x, t);
    }
    __syncthreads();
    if (threadIdx.x == 0) *ctr = 0u;
}

// The residual in the preconditioner's precision (r32 null in FP64: the preconditioner reads r).
template <int J>
__device__ __forceinline__ void st_r32(float* r32, size_t o, const double (&r)[J]) {
    if (!r32) return;
    float t[J];
#pragma unroll
    for (int j = 0; j < J; ++j) t[j] = (float)r[j];
    stv<J>(r32 + o, t);
}

template <int J, int R>
__global__ void __launch_bounds__(VTPB) kb_init(int n, const double* b, double* __restrict__ x, double* __restrict__ r,
                                                 float* r32, double* part, unsigned* ctr, double* S, bool ordered) {
    using L = Cols<J, R>;
    constexpr int Kp = L::KP;
    pdl_launch_dependents();
    pdl_wait();
    double v[J], z[J];
    zero(v);
    zero(z);
    for (int i = vfirst<J, R>(n); i < n; i += 4 * vblocks(n)) {
        double bi[J];
        ldv<J>(b + L::at(i), bi);
        stv<J>(x + L::at(i), z);
        stv<J>(r + L::at(i), bi);
        st_r32<J>(r32, L::at(i), bi);
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] += bi[j] * bi[j];
    }
    col_finish<J, R>(n, ordered, v, part, ctr, [&](int c, double t) {
        const double bn = sqrt(t);
        S[S_BNORM * Kp + c] = bn;
        S[S_K * Kp + c] = 0.0;
        S[S_RZOLD * Kp + c] = 0.0;
        S[S_BETA * Kp + c] = 0.0;
        S[S_ALPHA * Kp + c] = 0.0;
        S[S_RES * Kp + c] = bn > 0.0 ? 1.0 : 0.0;
        const bool ok = isfinite(bn);
        S[S_STATUS * Kp + c] = ok ? (bn > 0.0 && S[S_MAXIT * Kp + c] <= 0.0 ? CPC_ENOCONV : CPC_OK) : CPC_EBREAKDOWN;
        S[S_ACTIVE * Kp + c] = (ok && bn > 0.0 && S[S_MAXIT * Kp + c] > 0.0) ? 1.0 : 0.0;
    });
}

// Any column still active?  Sets the loop condition (one warp).
__global__ void kb_any_active(int Kp, const double* S, cudaGraphConditionalHandle cond) {
    pdl_launch_dependents();
    pdl_wait();
    bool on = false;
    for (int c = threadIdx.x; c < Kp; c += 32) on |= S[S_ACTIVE * Kp + c] > 0.0;
    on = __any_sync(0xffffffffu, on);
    if (threadIdx.x == 0) cudaGraphSetConditional(cond, on ? 1u : 0u);
}

__global__ void kb_guard(cudaGraphConditionalHandle cond) {
    pdl_launch_dependents();
    pdl_wait();
    cudaGraphSetConditional(cond, 0u);
}

template <int J, int R, class ZT>
__global__ void __launch_bounds__(VTPB, 4) kb_rz(int n, const double* r, const ZT* z, double* part, unsigned* ctr, double* S, bool ordered) {
    using L = Cols<J, R>;
    constexpr int Kp = L::KP;
    pdl_launch_dependents();
    pdl_wait();
    constexpr int U = vrows(J, 4);
    const int step = 4 * vblocks(n);
    double v[J];
    zero(v);
    for (int i0 = vfirst<J, R>(n); i0 < n; i0 += U * step) {
        double ri[U][J], zi[U][J];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * step;
            if (i >= n) break;
            ldv<J>(r + L::at(i), ri[u]);
            ldv<J>(z + L::at(i), zi[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * step >= n) break;
#pragma unroll
            for (int j = 0; j < J; ++j) v[j] += ri[u][j] * zi[u][j];
        }
    }
    col_finish<J, R>(n, ordered, v, part, ctr, [&](int c, double t) {
        const bool act = S[S_ACTIVE * Kp + c] > 0.0;
        if (act && (!(t > 0.0) || !isfinite(t))) {
            S[S_STATUS * Kp + c] = CPC_EBREAKDOWN;
            S[S_ACTIVE * Kp + c] = 0.0;
        }
        S[S_BETA * Kp + c] = (S[S_K * Kp + c] == 0.0 || !act) ? 0.0 : t / S[S_RZOLD * Kp + c];
        S[S_RZ * Kp + c] = t;
        S[S_RZOLD * Kp + c] = t;
    });
}

template <int J, int R, class ZT>
__global__ void __launch_bounds__(VTPB, 4) kb_p(int n, const ZT* z, double* __restrict__ p, const double* S) {
    using L = Cols<J, R>;
    constexpr int Kp = L::KP;
    pdl_launch_dependents();
    pdl_wait();
    double beta[J], k[J];
    ldv<J>(S + S_BETA * Kp + L::col(), beta);
    ldv<J>(S + S_K * Kp + L::col(), k);
    constexpr int U = vrows(J, 4);
    const int step = 4 * vblocks(n);
    for (int i0 = vfirst<J, R>(n); i0 < n; i0 += U * step) {
        double zi[U][J], pi[U][J];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * step;
            if (i >= n) break;
            ldv<J>(z + L::at(i), zi[u]);
            ldv<J>(p + L::at(i), pi[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * step;
            if (i >= n) break;
#pragma unroll
            for (int j = 0; j < J; ++j) pi[u][j] = k[j] == 0.0 ? zi[u][j] : zi[u][j] + beta[j] * pi[u][j];
            stv<J>(p + L::at(i), pi[u]);
        }
    }
}

// p.q has been summed: alpha = (r.z) / (p.q), a column that is not positive stops.
__device__ __forceinline__ void fin_pq(double* S, int Kp, int c, double t) {
    const bool act = S[S_ACTIVE * Kp + c] > 0.0;
    S[S_PQ * Kp + c] = t;
    if (act && (!(t > 0.0) || !isfinite(t))) {
        S[S_STATUS * Kp + c] = CPC_EBREAKDOWN;
        S[S_ACTIVE * Kp + c] = 0.0;
    }
    S[S_ALPHA * Kp + c] = S[S_ACTIVE * Kp + c] > 0.0 ? S[S_RZ * Kp + c] / t : 0.0;
}

template <int J, int R>
__global__ void __launch_bounds__(VTPB) kb_spmv_pq(BV<double, double> A, int nslots, const double* p,
                                                    double* __restrict__ q, double* part, unsigned* ctr, double* S, bool ordered) {
    using L = Cols<J, R>;
    pdl_launch_dependents();
    pdl_wait();
    double v[J];
    zero(v);
    for (int s = vfirst<J, R>(nslots); s < nslots; s += 4 * vblocks(nslots)) {
        const int row = A.perm[s];
        if (row < 0) continue;
        double acc[J], pr[J];
        const double d = A.diag[s];
        ldv<J>(p + L::at(row), pr);
#pragma unroll
        for (int j = 0; j < J; ++j) acc[j] = d * pr[j];
        const BRow t = brow_at(A, s, A.cptr + 1);
        Entries<4, double> m;
        m.load(A.col, A.val, t, 0, 1);
        brow<J, R, 4>(A.col, A.val, t, 0, 1, m, p, acc);
        stv<J>(q + L::at(row), acc);
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] += pr[j] * acc[j];
    }
    col_finish<J, R>(nslots, ordered, v, part, ctr, [&](int c, double t) { fin_pq(S, L::KP, c, t); });
}

template <int J, int R, int ND>
__global__ void __launch_bounds__(VTPB) kb_spmv_pq_dia(BD<double, double> A, const double* p, double* __restrict__ q,
                                                        double* part, unsigned* ctr, double* S, bool ordered) {
    using L = Cols<J, R>;
    pdl_launch_dependents();
    pdl_wait();
    double v[J];
    zero(v);
    for (int s = vfirst<J, R>(A.nslots); s < A.nslots; s += 4 * vblocks(A.nslots)) {
        const int row = bd_row(A, s);
        if (row < 0) continue;
        double w[ND];
#pragma unroll
        for (int d = 0; d < ND; ++d) w[d] = A.val[(size_t)d * A.nslots + s];
        const double dg = A.diag[s];
        double acc[J], pr[J];
        ldv<J>(p + L::at(row), pr);
#pragma unroll
        for (int j = 0; j < J; ++j) acc[j] = dg * pr[j];
        bd_dot<J, R, ND>(w, A.off, row, A.n, p, acc);
        stv<J>(q + L::at(row), acc);
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] += pr[j] * acc[j];
    }
    col_finish<J, R>(A.nslots, ordered, v, part, ctr, [&](int c, double t) { fin_pq(S, L::KP, c, t); });
}

template <int J, int R>
__global__ void __launch_bounds__(VTPB, 4) kb_update(int n, double* __restrict__ x, double* __restrict__ r, float* r32,
                                                   const double* p, const double* q, double* part, unsigned* ctr, double* S, bool ordered) {
    using L = Cols<J, R>;
    constexpr int Kp = L::KP;
    pdl_launch_dependents();
    pdl_wait();
    double alpha[J], v[J];
    ldv<J>(S + S_ALPHA * Kp + L::col(), alpha);
    zero(v);
    constexpr int U = vrows(J, 2);
    const int step = 4 * vblocks(n);
    for (int i0 = vfirst<J, R>(n); i0 < n; i0 += U * step) {
        double xi[U][J], ri[U][J], pi[U][J], qi[U][J];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * step;
            if (i >= n) break;
            ldv<J>(x + L::at(i), xi[u]);
            ldv<J>(p + L::at(i), pi[u]);
            ldv<J>(r + L::at(i), ri[u]);
            ldv<J>(q + L::at(i), qi[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * step;
            if (i >= n) break;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                xi[u][j] += alpha[j] * pi[u][j];
                ri[u][j] -= alpha[j] * qi[u][j];
                v[j] += ri[u][j] * ri[u][j];
            }
            stv<J>(x + L::at(i), xi[u]);
            stv<J>(r + L::at(i), ri[u]);
            st_r32<J>(r32, L::at(i), ri[u]);
        }
    }
    col_finish<J, R>(n, ordered, v, part, ctr, [&](int c, double t) {
        if (S[S_ACTIVE * Kp + c] <= 0.0) return;
        const double k = S[S_K * Kp + c] + 1.0;
        S[S_K * Kp + c] = k;
        const double res = sqrt(t) / S[S_BNORM * Kp + c];
        S[S_RES * Kp + c] = res;
        if (!isfinite(res)) { S[S_STATUS * Kp + c] = CPC_EBREAKDOWN; S[S_ACTIVE * Kp + c] = 0.0; }
        else if (res < S[S_TOL * Kp + c]) { S[S_STATUS * Kp + c] = CPC_OK; S[S_ACTIVE * Kp + c] = 0.0; }
        else if (k >= S[S_MAXIT * Kp + c]) { S[S_STATUS * Kp + c] = CPC_ENOCONV; S[S_ACTIVE * Kp + c] = 0.0; }
    });
}

// [n][K] user layout <-> [n][Kp] internal layout, 32 rows per block of 8 warps.
__global__ void __launch_bounds__(256) kb_pack(int n, int K, int Kp, const double* in, double* __restrict__ out) {
    for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += gridDim.x * 8)
        for (int c = threadIdx.x & 31; c < Kp; c += 32) out[(size_t)i * Kp + c] = c < K ? in[(size_t)i * K + c] : 0.0;
}

__global__ void __launch_bounds__(256) kb_unpack(int n, int K, int Kp, const double* in, double* __restrict__ out) {
    for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += gridDim.x * 8)
        for (int c = threadIdx.x & 31; c < K; c += 32) out[(size_t)i * K + c] = in[(size_t)i * Kp + c];
}

// Adjoint sources from the forward solutions: b[i][c] = x[i][c] where b[i][c] != 0, else 0
// (the gradient of J_c = 1/2 sum over the source cells of column c of x^2); also saves x.
__global__ void kb_adjoint_rhs(int64_t nk, double* __restrict__ b, const double* x, double* __restrict__ xsave) {
    pdl_launch_dependents();
    pdl_wait();
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nk; t += (int64_t)gridDim.x * blockDim.x) {
        const double xi = x[t];
        xsave[t] = xi;
        b[t] = b[t] != 0.0 ? xi : 0.0;
    }
}

// ---------------------------------------------------------------------------------------------
// Recording (column-wise V-cycle, IC(0), B_co)
// ---------------------------------------------------------------------------------------------
// ------------------------------------------------------------------------------------------------
// Block PCG (O'Leary 1980): the K columns share one block Krylov space through K x K matrices.
// Not a method of the paper; the coupled counterpart of the batched solve above.  All K x K
// arithmetic is FP64 and every sum finishes in a fixed order.
// ------------------------------------------------------------------------------------------------
constexpr int KK_TPB = 256;
constexpr int KK_ELEMS = 2048;            // elements of U (and of V) staged per step of kk_gram
constexpr int KK_GRID = 152 * 2;          // blocks of kk_init / kk_gram / kk_update / kk_pupdate (fixed)
enum { KM_PQ = 0, KM_GAMMA, KM_GAMMA_NEW, KM_ALPHA, KM_BETA, KM_COUNT };
enum { KV_BNORM = 0, KV_RES, KV_COUNT };
enum { KF_BAD = 0, KF_DONE, KF_COUNT };

// part[block] = U^T V over the block's rows, on the 4 x 4 tiles (ti, tj) with ti <= tj of the
// KP x KP result; U is Z (preconditioner precision) or P, V is R or Q (FP64).  The NT upper tiles in
// row-major order belong to consecutive threads, and as many groups of NT threads as fit in the block
// share the staged rows (25 groups of 10 tiles for 16 columns, one of 136 for 64), so that whole warps
// work: an FP64 warp instruction costs the same with idle lanes, and FP64 issue is the bound of this
// kernel on this part.  The groups' tiles are added in group order.
template <int KP, class UT>
__global__ void __launch_bounds__(KK_TPB) kk_gram(int n, const UT* U, const double* V, double* __restrict__ part) {
    constexpr int T = KP / 4, NT = T * (T + 1) / 2, GROUPS = KK_TPB / NT, ROWS = KK_ELEMS / KP;
    extern __shared__ __align__(16) double ksm[];
    double* us = ksm;                      // [ROWS][KP]
    double* vs = ksm + KK_ELEMS;           // [ROWS][KP]
    const int t = threadIdx.x, grp = t / NT;
    int ti = 0, rem = t - grp * NT;
    while (rem >= T - ti) {
        rem -= T - ti;
        ++ti;
    }
    const int tj = ti + rem;
    const bool act = grp < GROUPS;
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = 0.0;
    const int per = (n + gridDim.x - 1) / gridDim.x;
    const int r0 = min(n, (int)blockIdx.x * per), r1 = min(n, r0 + per);
    for (int base = r0; base < r1; base += ROWS) {
        const int rows = min(ROWS, r1 - base);
        __syncthreads();
        for (int e = t; e < KK_ELEMS; e += KK_TPB) {
            const size_t g = (size_t)base * KP + e;
            us[e] = e < rows * KP ? (double)U[g] : 0.0;
            vs[e] = e < rows * KP ? V[g] : 0.0;
        }
        __syncthreads();
        if (act) {
            for (int rr = grp; rr < rows; rr += GROUPS) {
                double a[4], c[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    a[q] = us[rr * KP + ti * 4 + q];
                    c[q] = vs[rr * KP + tj * 4 + q];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int w = 0; w < 4; ++w) acc[q][w] = __fma_rn(a[q], c[w], acc[q][w]);
            }
        }
    }
    // the groups in turn add their tiles in shared memory (KP x KP <= 2 KK_ELEMS)
    for (int g = 0; g < GROUPS; ++g) {
        __syncthreads();
        if (grp == g)
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    double& o = ksm[(ti * 4 + q) * KP + tj * 4 + w];
                    o = g == 0 ? acc[q][w] : o + acc[q][w];
                }
    }
    __syncthreads();
    if (grp == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const int e = (ti * 4 + q) * KP + tj * 4 + w;
                part[(size_t)blockIdx.x * KP * KP + e] = ksm[e];
            }
}

// out = sum over blocks of part, a warp per entry (each lane its blocks in order, then a fixed tree);
// entry (i, j) and (j, i) both take the computed upper entry (min, max), so the result is exactly
// symmetric.
__global__ void __launch_bounds__(256) kk_gram_sum(int G, int Kp, const double* part, double* __restrict__ out) {
    const int e = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (e >= Kp * Kp) return;
    const int i = e / Kp, j = e - i * Kp;
    const double* p = part + (size_t)min(i, j) * Kp + max(i, j);
    double s = 0.0;
#pragma unroll 8
    for (int g = lane; g < G; g += 32) s += p[(size_t)g * Kp * Kp];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[e] = s;
}

// Y = S^{-1} W on the leading K x K blocks by Cholesky S = L L^T (one block; S symmetric).  out is
// Kp x Kp with zeros outside K x K.  A pivot that is not finite or at most 1e-12 times its diagonal
// entry s_kk (a block column within rounding of the span of the others) sets flag[KF_BAD].
// With copy_to, W is copied there afterwards (gamma_old <- gamma_new).
__global__ void __launch_bounds__(KK_TPB) kk_solve(int K, int Kp, const double* S, const double* W,
                                                   double* __restrict__ out, double* copy_to, int* flag) {
    extern __shared__ __align__(16) double ksm[];
    double* L = ksm;                       // [K][K]
    double* Y = ksm + K * K;               // [K][K]
    __shared__ int bad;
    const int t = threadIdx.x, nt = blockDim.x;
    if (t == 0) bad = 0;
    for (int e = t; e < K * K; e += nt) {
        const int i = e / K, j = e - (e / K) * K;
        L[e] = S[(size_t)i * Kp + j];
        Y[e] = W[(size_t)i * Kp + j];
    }
    __syncthreads();
    for (int k = 0; k < K; ++k) {
        if (t == 0) {
            const double d = L[k * K + k];
            if (!(d > 1e-12 * S[(size_t)k * Kp + k]) || !isfinite(d)) bad = 1;
            L[k * K + k] = sqrt(d > 0.0 && isfinite(d) ? d : 1.0);
        }
        __syncthreads();
        const double dk = L[k * K + k];
        for (int i = k + 1 + t; i < K; i += nt) L[i * K + k] /= dk;
        __syncthreads();
        const int m = K - k - 1;
        for (int e = t; e < m * m; e += nt) {
            const int i = k + 1 + e / m, j = k + 1 + (e - (e / m) * m);
            if (j <= i) L[i * K + j] -= L[i * K + k] * L[j * K + k];
        }
        __syncthreads();
    }
    for (int c = t; c < K; c += nt) {      // one right-hand-side column per thread
        for (int i = 0; i < K; ++i) {      // L z = w
            double s = Y[i * K + c];
            for (int q = 0; q < i; ++q) s -= L[i * K + q] * Y[q * K + c];
            Y[i * K + c] = s / L[i * K + i];
        }
        for (int i = K - 1; i >= 0; --i) { // L^T y = z
            double s = Y[i * K + c];
            for (int q = i + 1; q < K; ++q) s -= L[q * K + i] * Y[q * K + c];
            Y[i * K + c] = s / L[i * K + i];
        }
    }
    __syncthreads();
    for (int e = t; e < Kp * Kp; e += nt) {
        const int i = e / Kp, j = e - (e / Kp) * Kp;
        out[e] = (i < K && j < K) ? Y[i * K + j] : 0.0;
        if (copy_to) copy_to[e] = W[e];
    }
    if (t == 0 && bad) flag[KF_BAD] = 1;
}

// Entry k of a row held across its lanes.
template <int J, int R>
__device__ __forceinline__ double kk_lane(const double (&v)[J], int k) {
    if constexpr (R > 1) return __shfl_sync(0xffffffffu, v[0], Cols<J, R>::sub() * Cols<J, R>::W + k);
    else if constexpr (J == 1) return __shfl_sync(0xffffffffu, v[0], k);
    else return __shfl_sync(0xffffffffu, k % J ? v[1] : v[0], k / J);
}

// Per block, the column sums of v over the lanes in warp order, into part[block][KP].
template <int J, int R>
__device__ __forceinline__ void kk_block_cols(const double (&v)[J], double* ws, double* __restrict__ part) {
    using L = Cols<J, R>;
    const int w = threadIdx.x >> 5;
#pragma unroll
    for (int m = 0; m < J; ++m) ws[(w * R + L::sub()) * L::KP + L::col() + m] = v[m];
    __syncthreads();
    for (int c = threadIdx.x; c < L::KP; c += BTPB) {
        double s = 0.0;
        for (int q = 0; q < BWARPS * R; ++q) s += ws[q * L::KP + c];
        part[(size_t)blockIdx.x * L::KP + c] = s;
    }
}

// X += P alpha and R -= Q alpha (alpha in shared memory), and per block the column sums of r_ij^2.
template <int J, int R>
__global__ void __launch_bounds__(BTPB) kk_update(int n, int K, double* __restrict__ X, double* __restrict__ Rv, float* r32,
                                                  const double* P, const double* Q, const double* alpha,
                                                  double* __restrict__ part, const int* flag) {
    using L = Cols<J, R>;
    constexpr int Kp = L::KP;
    if (flag[KF_BAD]) return;              // a K x K solve failed: keep the last good iterate
    extern __shared__ __align__(16) double ksm[];
    double* al = ksm;                      // [Kp][Kp]
    double* ws = ksm + Kp * Kp;            // [BWARPS R][Kp]
    for (int e = threadIdx.x; e < Kp * Kp; e += BTPB) al[e] = alpha[e];
    __syncthreads();
    double rr[J];
    zero(rr);
    for (int i0 = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R; i0 < n; i0 += gridDim.x * BWARPS * R) {
        const bool on = i0 + L::sub() < n;
        const size_t o = L::at(i0 + L::sub());
        double p[J], q[J], dx[J], dr[J];
        zero(p);
        zero(q);
        zero(dx);
        zero(dr);
        if (on) {
            ldv<J>(P + o, p);
            ldv<J>(Q + o, q);
        }
        for (int k = 0; k < K; ++k) {
            const double pk = kk_lane<J, R>(p, k), qk = kk_lane<J, R>(q, k);
            double a[J];
            ldv<J>(al + k * Kp + L::col(), a);
#pragma unroll
            for (int m = 0; m < J; ++m) {
                dx[m] = __fma_rn(pk, a[m], dx[m]);
                dr[m] = __fma_rn(qk, a[m], dr[m]);
            }
        }
        if (!on) continue;
        double x[J], r[J];
        ldv<J>(X + o, x);
        ldv<J>(Rv + o, r);
#pragma unroll
        for (int m = 0; m < J; ++m) {
            x[m] += dx[m];
            r[m] -= dr[m];
            rr[m] = __fma_rn(r[m], r[m], rr[m]);
        }
        stv<J>(X + o, x);
        stv<J>(Rv + o, r);
        st_r32<J>(r32, o, r);
    }
    kk_block_cols<J, R>(rr, ws, part);
}

// P = Z + P beta, in place (a row is read by its own lanes before they write it).
template <int J, int R, class ZT>
__global__ void __launch_bounds__(BTPB) kk_pupdate(int n, int K, const ZT* Z, double* __restrict__ P, const double* beta,
                                                   const int* flag) {
    using L = Cols<J, R>;
    constexpr int Kp = L::KP;
    if (flag[KF_BAD]) return;
    extern __shared__ __align__(16) double ksm[];
    for (int e = threadIdx.x; e < Kp * Kp; e += BTPB) ksm[e] = beta[e];
    __syncthreads();
    for (int i0 = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R; i0 < n; i0 += gridDim.x * BWARPS * R) {
        const bool on = i0 + L::sub() < n;
        const size_t o = L::at(i0 + L::sub());
        double p[J], z[J], acc[J];
        zero(p);
        zero(z);
        zero(acc);
        if (on) {
            ldv<J>(P + o, p);
            ldv<J>(Z + o, z);
        }
        for (int k = 0; k < K; ++k) {
            const double pk = kk_lane<J, R>(p, k);
            double b[J];
            ldv<J>(ksm + k * Kp + L::col(), b);
#pragma unroll
            for (int m = 0; m < J; ++m) acc[m] = __fma_rn(pk, b[m], acc[m]);
        }
        if (!on) continue;
#pragma unroll
        for (int m = 0; m < J; ++m) z[m] += acc[m];
        stv<J>(P + o, z);
    }
}

template <class ZT>
__global__ void kk_copy(int64_t nk, const ZT* z, double* __restrict__ p) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nk; e += (int64_t)gridDim.x * blockDim.x)
        p[e] = (double)z[e];
}

// Q = A P with A in CSR.
template <int J, int R>
__global__ void __launch_bounds__(BTPB) kk_spmm(int n, const int* __restrict__ ptr, const int* __restrict__ col,
                                                const double* __restrict__ val, const double* P, double* __restrict__ Q) {
    using L = Cols<J, R>;
    const int i = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub();
    if (i >= n) return;
    double acc[J];
    zero(acc);
    const int e0 = ptr[i];
    const BRow t{e0, ptr[i + 1] - e0, 0, 1};
    Entries<4, double> m;
    m.load(col, val, t, 0, 1);
    brow<J, R, 4>(col, val, t, 0, 1, m, P, acc);
    stv<J>(Q + L::at(i), acc);
}

// R = B (and its copy in the preconditioner's precision), X = 0, and per block the column sums of b_ij^2.
template <int J, int R>
__global__ void __launch_bounds__(BTPB) kk_init(int n, const double* B, double* __restrict__ X, double* __restrict__ Rv,
                                                float* r32, double* __restrict__ part) {
    using L = Cols<J, R>;
    __shared__ double ws[BWARPS * R * L::KP];
    double s[J], z[J];
    zero(s);
    zero(z);
    for (int i = (blockIdx.x * BWARPS + (threadIdx.x >> 5)) * R + L::sub(); i < n; i += gridDim.x * BWARPS * R) {
        double v[J];
        ldv<J>(B + L::at(i), v);
        stv<J>(Rv + L::at(i), v);
        stv<J>(X + L::at(i), z);
        st_r32<J>(r32, L::at(i), v);
#pragma unroll
        for (int m = 0; m < J; ++m) s[m] = __fma_rn(v[m], v[m], s[m]);
    }
    kk_block_cols<J, R>(s, ws, part);
}

// One block of 8 warps, a warp per column.  Column norms from the partials (each lane its blocks in
// order, then a fixed tree).  init: bnorm_k = ||b_k||, a zero column sets KF_BAD.  Otherwise res_k =
// ||r_k|| / ||b_k||; KF_DONE = 1 when every column is below tol, and a residual that is not finite
// sets KF_BAD.
__global__ void __launch_bounds__(256) kk_check(int G, int Kp, int K, const double* part, double* __restrict__ vec, double tol,
                                                int init, int* flag) {
    __shared__ int all;
    if (threadIdx.x == 0) all = 1;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int c = threadIdx.x >> 5; c < K; c += 8) {
        double s = 0.0;
#pragma unroll 8
        for (int g = lane; g < G; g += 32) s += part[(size_t)g * Kp + c];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane != 0) continue;
        const double nrm = sqrt(s);
        if (init) {
            vec[KV_BNORM * Kp + c] = nrm;
            if (!(nrm > 0.0) || !isfinite(nrm)) atomicOr(&flag[KF_BAD], 1);
        } else {
            const double r = nrm / vec[KV_BNORM * Kp + c];
            vec[KV_RES * Kp + c] = r;
            if (!isfinite(r)) atomicOr(&flag[KF_BAD], 1);
            if (!(r < tol)) atomicAnd(&all, 0);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && !init) flag[KF_DONE] = all;
}

template <class VT> VT* bx(Batched& B, int l) { return (VT*)B.lx[l].p; }
template <class VT> VT* bf(Batched& B, int l) { return (VT*)B.lf[l].p; }
template <class VT> VT* br(Batched& B, int l) { return (VT*)B.lr[l].p; }

// One colour of a level; from_zero: in a forward sweep from a zero guess.
template <int J, int R, class VT>
void brec_gs(Level& L, int c, const VT* f, VT* x, cudaStream_t s, bool from_zero) {
    const int s0 = L.S.seg[c] * L.S.C, s1 = L.S.seg[c + 1] * L.S.C;
    if (s1 <= s0) return;
    const int g = rows_grid<R>(s1 - s0);
    if (L.S.ndiag) {
        bwith_nd(L.S.ndiag, [&](auto nd) {
            constexpr int ND = decltype(nd)::value;
            if constexpr (std::is_same<VT, double>::value)
                blaunch(kb_gs_dia<J, R, double, double, VT, ND>, rows_grid<R>(s1 - s0, DWARPS), DTPB, s,
                        bdview(L.S, L.n, (const double*)L.S.dval.p, (const double*)L.S.dinv.p, false), s0, s1, f, x);
            else
                blaunch(kb_gs_dia<J, R, float, float, VT, ND>, rows_grid<R>(s1 - s0, DWARPS), DTPB, s,
                        bdview(L.S, L.n, (const float*)L.S.dval32.p, (const float*)L.S.dinv32.p, false), s0, s1, f, x);
        });
        return;
    }
    const int* end = from_zero && L.skip_zeros() ? (const int*)L.S.cmid.p : (const int*)(L.S.cptr.p + 1);
    auto go = [&](auto view) {
        if (from_zero && !L.skip_zeros()) view.col = L.S.fcol.p;
        using V = decltype(view);
        using MT = std::remove_cv_t<std::remove_reference_t<decltype(*view.val)>>;
        using DT = std::remove_cv_t<std::remove_reference_t<decltype(*view.diag)>>;
        static_assert(std::is_same<V, BV<MT, DT>>::value, "");
        // long rows in a small colour group: a block per 2 R rows
        const bool lng = L.A.nnz >= (int64_t)16 * L.n;
        if (lng && (s1 - s0) <= 16384) blaunch(kb_gs_wide<J, R, MT, DT, VT>, (s1 - s0 + 2 * R - 1) / (2 * R), 64 * WSPLIT, s, view, end, s0, s1, f, x);
        else blaunch(kb_gs<J, R, MT, DT, VT>, g, BTPB, s, view, end, s0, s1, f, x);
    };
    if constexpr (std::is_same<VT, double>::value) go(bview(L.S, (const double*)L.S.val.p, (const double*)L.S.dinv.p));
    else if (L.vt == VT_BF16) go(bview(L.S, (const __nv_bfloat16*)L.S.val16.p, (const float*)L.S.dinv32.p));
    else go(bview(L.S, (const float*)L.S.val32.p, (const float*)L.S.dinv32.p));
}

// r = f - A x after a forward sweep (from a zero guess with from_zero).  In FP64, on a red-black level
// only the red rows are written: the black residual is zero up to rounding, and no transfer reads it.
template <int J, int R, class VT>
void brec_resid(Level& L, const VT* f, const VT* x, VT* r, cudaStream_t s, bool from_zero) {
    from_zero = from_zero && L.skip_zeros();
    if (L.S.ndiag) {
        const int s1 = L.red_black && L.skip_zeros() ? L.S.seg[1] * L.S.C : L.S.nslots;
        bwith_nd(L.S.ndiag, [&](auto nd) {
            constexpr int ND = decltype(nd)::value;
            auto go = [&](auto view, auto zero) {
                using MT = std::remove_cv_t<std::remove_reference_t<decltype(*view.val)>>;
                blaunch(kb_resid_dia<J, R, MT, MT, VT, VT, ND, decltype(zero)::value>, rows_grid<R>(s1, DWARPS), DTPB, s, view, s1, f, x, r);
            };
            auto both = [&](auto view) {
                if (from_zero && L.red_black) go(view, std::true_type{});
                else go(view, std::false_type{});
            };
            if constexpr (std::is_same<VT, double>::value)
                both(bdview(L.S, L.n, (const double*)L.S.dval.p, (const double*)L.S.diag.p, false));
            else
                both(bdview(L.S, L.n, (const float*)L.S.dval32.p, (const float*)L.S.diag32.p, false));
        });
        return;
    }
    const int g = rows_grid<R>(L.S.nslots);
    auto go = [&](auto view) {
        using MT = std::remove_cv_t<std::remove_reference_t<decltype(*view.val)>>;
        using DT = std::remove_cv_t<std::remove_reference_t<decltype(*view.diag)>>;
        if (from_zero) blaunch(kb_resid_up<J, R, MT, DT, VT>, g, BTPB, s, view, (const int*)L.S.cmid.p, L.S.nslots, x, r);
        else blaunch(kb_resid<J, R, MT, DT, VT>, g, BTPB, s, view, L.S.nslots, f, x, r);
    };
    if constexpr (std::is_same<VT, double>::value) go(bview(L.S, (const double*)L.S.val.p, (const double*)L.S.diag.p));
    else if (L.vt == VT_BF16) go(bview(L.S, (const __nv_bfloat16*)L.S.val16.p, (const float*)L.S.diag32.p));
    else go(bview(L.S, (const float*)L.S.val32.p, (const float*)L.S.diag32.p));
}

template <class VT>
BV<VT, VT> bfull(const Sell& S) {
    if constexpr (std::is_same<VT, double>::value) return bview(S, (const double*)S.val.p, (const double*)nullptr);
    else return bview(S, (const float*)S.val32.p, (const float*)nullptr);
}

template <class VT> const VT* bdnat(const Level& L);
template <> const double* bdnat<double>(const Level& L) { return L.dnat64.p; }
template <> const float* bdnat<float>(const Level& L) { return L.dnat32.p; }

// As rec_vcycle: with first_done the caller has applied the first colour step from the zero guess.
template <int J, int R, class VT>
void brec_vcycle(Handle& h, int l, const VT* f, VT* x, bool zero_guess, cudaStream_t s, bool first_done = false) {
    Batched& B = h.bat;
    const int nl = (int)h.lev.size();
    Level& L = h.lev[l];
    if (l == nl - 1) {
        constexpr int KP = Cols<J, R>::KP, JC = KP > 32 ? KP / 32 : 1, RC = KP > 32 ? 1 : 32 / KP;
        const VT* ai = std::is_same<VT, double>::value ? (const VT*)h.Ainv.p : (const VT*)h.Ainv32.p;
        if constexpr (std::is_same<VT, double>::value)
            blaunch(kb_coarse<JC, RC, VT, VT, VT>, (L.n + RC * CROWS - 1) / (RC * CROWS), CWARPS * 32, s, L.n, ai, f, x);
        else
            blaunch(kb_coarse_seq<JC, RC, VT, VT, VT>, (L.n + CWARPS * RC * SROWS - 1) / (CWARPS * RC * SROWS), CWARPS * 32, s, L.n,
                    ai, f, x);
        return;
    }
    if (zero_guess && !first_done)
        blaunch(kb_first<J, R, VT>, rows_grid<R>(L.n, DWARPS), DTPB, s, L.n, f, (const int*)L.colour.p, bdnat<VT>(L), x);
    for (int c = zero_guess ? 1 : 0; c < L.ncolours; ++c) brec_gs<J, R>(L, c, f, x, s, zero_guess);
    brec_resid<J, R>(L, f, (const VT*)x, br<VT>(B, l), s, zero_guess);
    Level& C = h.lev[l + 1];
    const bool last = l + 1 == nl - 1;
    blaunch(kb_restrict<J, R, VT, VT>, rows_grid<R>(L.SR.nslots), BTPB, s, bfull<VT>(L.SR),
            L.red_black && L.skip_zeros() ? (const int*)L.SR.cmid.p : (const int*)(L.SR.cptr.p + 1), L.SR.nslots, (const VT*)br<VT>(B, l),
            bf<VT>(B, l + 1), last ? (VT*)nullptr : bx<VT>(B, l + 1), (const int*)C.colour.p, bdnat<VT>(C));
    brec_vcycle<J, R, VT>(h, l + 1, bf<VT>(B, l + 1), bx<VT>(B, l + 1), !last, s, !last);
    const int ps = L.red_black ? L.SP.seg[1] * L.SP.C : L.SP.nslots;
    blaunch(kb_prolong<J, R, VT, VT>, rows_grid<R>(ps), BTPB, s, bfull<VT>(L.SP), ps, (const VT*)bx<VT>(B, l + 1), x);
    for (int c = L.ncolours - 1; c >= 0; --c) brec_gs<J, R>(L, c, f, x, s, false);
}

template <int J, int R, class VT>
void brec_ic(Handle& h, const VT* t, VT* y, VT* w, VT* zadd, cudaStream_t s) {
    BV<VT, VT> lv, uv;
    if constexpr (std::is_same<VT, double>::value) {
        lv = bview(h.L, (const double*)h.L.val.p, (const double*)nullptr);
        uv = bview(h.U, (const double*)h.U.val.p, (const double*)h.U.dinv.p);
    } else {
        lv = bview(h.L, (const float*)h.L.val32.p, (const float*)nullptr);
        uv = bview(h.U, (const float*)h.U.val32.p, (const float*)h.U.dinv32.p);
    }
    for (int g = 0; g + 1 < (int)h.L.seg.size(); ++g) {
        const int s0 = h.L.seg[g] * h.L.C, s1 = h.L.seg[g + 1] * h.L.C;
        blaunch(kb_lsolve<J, R, VT, VT>, rows_grid<R>(s1 - s0), BTPB, s, lv, s0, s1, t, y);
    }
    for (int g = 0; g + 1 < (int)h.U.seg.size(); ++g) {
        const int s0 = h.U.seg[g] * h.U.C, s1 = h.U.seg[g + 1] * h.U.C;
        blaunch(kb_usolve<J, R, VT, VT>, rows_grid<R>(s1 - s0), BTPB, s, uv, s0, s1, (const VT*)y, w, zadd);
    }
}

template <int J, int R, class VT>
void brec_precond(Handle& h, int which, const VT* r, VT* z, cudaStream_t s) {
    Batched& B = h.bat;
    VT* t = (VT*)B.t.p;
    VT* y = (VT*)B.y.p;
    const Sell& A = h.Anat;
    auto fine_resid = [&]() {
        const int g = rows_grid<R>(A.nslots);
        if (A.ndiag) {
            bwith_nd(A.ndiag, [&](auto nd) {
                constexpr int ND = decltype(nd)::value;
                if constexpr (std::is_same<VT, double>::value)
                    blaunch(kb_resid_dia<J, R, double, double, VT, VT, ND, false>, rows_grid<R>(A.nslots, DWARPS), DTPB, s,
                            bdview(A, h.n, (const double*)A.dval.p, (const double*)A.diag.p, true), A.nslots, r, (const VT*)z, t);
                else
                    blaunch(kb_resid_dia<J, R, float, float, VT, VT, ND, false>, rows_grid<R>(A.nslots, DWARPS), DTPB, s,
                            bdview(A, h.n, (const float*)A.dval32.p, (const float*)A.diag32.p, true), A.nslots, r, (const VT*)z, t);
            });
            return;
        }
        if constexpr (std::is_same<VT, double>::value)
            blaunch(kb_resid<J, R, double, double, VT>, g, BTPB, s, bview(A, (const double*)A.val.p, (const double*)A.diag.p), A.nslots, r, (const VT*)z, t);
        else
            blaunch(kb_resid<J, R, float, float, VT>, g, BTPB, s, bview(A, (const float*)A.val32.p, (const float*)A.diag32.p), A.nslots, r, (const VT*)z, t);
    };
    switch (which) {
        case CPC_PRECOND_BCO:
            brec_vcycle<J, R, VT>(h, 0, r, z, true, s);
            if (h.ic_rb && h.lev[0].S.ndiag) {                   // step (2): black rows, one pass
                const Sell& S0 = h.lev[0].S;
                const int s0 = S0.seg[1] * S0.C, s1 = S0.seg[2] * S0.C;
                if (s1 > s0)
                    bwith_nd(S0.ndiag, [&](auto nd) {
                        constexpr int ND = decltype(nd)::value;
                        if constexpr (std::is_same<VT, double>::value)
                            blaunch(kb_bco_black_dia<J, R, double, double, VT, ND>, rows_grid<R>(s1 - s0, DWARPS), DTPB, s,
                                    bdview(S0, h.n, (const double*)S0.dval.p, (const double*)S0.diag.p, false), s0, s1,
                                    r, (const VT*)h.ic_uinv64.p, z);
                        else
                            blaunch(kb_bco_black_dia<J, R, float, float, VT, ND>, rows_grid<R>(s1 - s0, DWARPS), DTPB, s,
                                    bdview(S0, h.n, (const float*)S0.dval32.p, (const float*)S0.diag32.p, false), s0,
                                    s1, r, (const VT*)h.ic_uinv32.p, z);
                    });
            } else {
                fine_resid();
                brec_ic<J, R, VT>(h, t, y, t, z, s);
            }
            brec_vcycle<J, R, VT>(h, 0, r, z, false, s);
            break;
        case CPC_PRECOND_AMG:
            brec_vcycle<J, R, VT>(h, 0, r, z, true, s);
            brec_vcycle<J, R, VT>(h, 0, r, z, false, s);
            break;
        case CPC_PRECOND_IC0:
            brec_ic<J, R, VT>(h, r, y, z, (VT*)nullptr, s);
            break;
        case CPC_PRECOND_BHAT:
            brec_vcycle<J, R, VT>(h, 0, r, z, true, s);
            brec_vcycle<J, R, VT>(h, 0, r, z, false, s);
            brec_ic<J, R, VT>(h, r, y, t, z, s);
            break;
        default:
            fail(CPC_EINVAL, "batched solve supports B_co, AMG, IC(0) and B^");
    }
}

// The residual as the preconditioner reads it.
template <class VT> const VT* bres(const Batched& B);
template <> const double* bres<double>(const Batched& B) { return B.r.p; }
template <> const float* bres<float>(const Batched& B) { return B.r32.p; }

template <int J, int R, class VT>
void brec_loop(Handle& h, cudaGraph_t g, cudaStream_t cs, cudaGraphNode_t* dep, size_t ndep, cudaGraphNode_t* out_node) {
    Batched& B = h.bat;
    const int Kp = B.Kp;
    const int n = h.n;
    cudaGraphConditionalHandle cond;
    CPC_CK(cudaGraphConditionalHandleCreate(&cond, g, 1u, cudaGraphCondAssignDefault));
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = cond;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    CPC_CK(cudaGraphAddNode(out_node, g, dep, nullptr, ndep, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    CPC_CK(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    blaunch(kb_guard, 1, 32, cs, cond);
    VT* z = (VT*)B.z.p;
    brec_precond<Gather<J, R, VT>::j, Gather<J, R, VT>::r, VT>(h, h.opt.precond, bres<VT>(B), z, cs);
    const int vg = vgrid<R>(n);
    const bool ord = !std::is_same<VT, double>::value;
    blaunch(kb_rz<J, R, VT>, vg, VTPB, cs, n, (const double*)B.r.p, (const VT*)z, B.partial.p, h.counter.p + 1, B.S.p, ord);
    blaunch(kb_p<J, R, VT>, vg, VTPB, cs, n, (const VT*)z, B.p.p, (const double*)B.S.p);
    const Sell& A = h.Anat;
    if (A.ndiag)
        bwith_nd(A.ndiag, [&](auto nd) {
            blaunch(kb_spmv_pq_dia<J, R, decltype(nd)::value>, vgrid<R>(A.nslots), VTPB, cs,
                    bdview(A, n, (const double*)A.dval.p, (const double*)A.diag.p, true), (const double*)B.p.p,
                    B.q.p, B.partial.p, h.counter.p + 1, B.S.p, ord);
        });
    else
        blaunch(kb_spmv_pq<J, R>, vgrid<R>(A.nslots), VTPB, cs, bview(A, (const double*)A.val.p, (const double*)A.diag.p),
                A.nslots, (const double*)B.p.p, B.q.p, B.partial.p, h.counter.p + 1, B.S.p, ord);
    blaunch(kb_update<J, R>, vg, VTPB, cs, n, B.x.p, B.r.p, B.r32.p, (const double*)B.p.p, (const double*)B.q.p, B.partial.p,
            h.counter.p + 1, B.S.p, ord);
    blaunch(kb_any_active, 1, 32, cs, Kp, (const double*)B.S.p, cond);
    CPC_CK(cudaStreamEndCapture(cs, &body));
}

// One graph: init, while(any active) { iteration }, [adjoint: sources, init, while {...}].  It works on the
// internal block vectors alone, so calls with other buffers replay it.
template <int J, int R, class VT>
void build_batched_graph(Handle& h, bool with_adjoint) {
    Batched& B = h.bat;
    const int Kp = B.Kp;
    const int n = h.n;
    cudaStream_t cs;
    CPC_CK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    struct SG { cudaStream_t s; ~SG() { cudaStreamDestroy(s); } } sg{cs};
    cudaGraph_t g;
    CPC_CK(cudaGraphCreate(&g, 0));
    const int vg = vgrid<R>(n);
    const bool ord = !std::is_same<VT, double>::value;
    auto capture_into = [&](cudaGraphNode_t* deps, size_t ndeps, auto&& body) -> std::vector<cudaGraphNode_t> {
        std::vector<cudaGraphNode_t> before;
        size_t nn = 0;
        CPC_CK(cudaGraphGetNodes(g, nullptr, &nn));
        before.resize(nn);
        CPC_CK(cudaGraphGetNodes(g, before.data(), &nn));
        CPC_CK(cudaStreamBeginCaptureToGraph(cs, g, deps, nullptr, ndeps, cudaStreamCaptureModeThreadLocal));
        body();
        CPC_CK(cudaStreamEndCapture(cs, &g));
        size_t nn2 = 0;
        CPC_CK(cudaGraphGetNodes(g, nullptr, &nn2));
        std::vector<cudaGraphNode_t> all(nn2);
        CPC_CK(cudaGraphGetNodes(g, all.data(), &nn2));
        std::vector<cudaGraphNode_t> added;
        for (auto nd : all) if (std::find(before.begin(), before.end(), nd) == before.end()) added.push_back(nd);
        // leaves among the added nodes
        std::vector<cudaGraphNode_t> leaves;
        for (auto nd : added) {
            size_t nout = 0;
            CPC_CK(cudaGraphNodeGetDependentNodes(nd, nullptr, nullptr, &nout));
            if (nout == 0) leaves.push_back(nd);
        }
        return leaves;
    };
    auto l1 = capture_into(nullptr, 0, [&] {
        blaunch(kb_init<J, R>, vg, VTPB, cs, n, (const double*)B.b.p, B.x.p, B.r.p, B.r32.p, B.partial.p, h.counter.p + 1, B.S.p, ord);
    });
    cudaGraphNode_t w1;
    brec_loop<J, R, VT>(h, g, cs, l1.data(), l1.size(), &w1);
    if (with_adjoint) {
        auto l2 = capture_into(&w1, 1, [&] {
            blaunch(kb_adjoint_rhs, 2048, 256, cs, (int64_t)n * Kp, B.b.p, (const double*)B.x.p, B.xfwd.p);
            CPC_CK(cudaMemcpyAsync(B.kfwd.p, B.S.p + (size_t)S_K * Kp, sizeof(double) * Kp, cudaMemcpyDeviceToDevice, cs));
            CPC_CK(cudaMemcpyAsync(B.kfwd.p + Kp, B.S.p + (size_t)S_STATUS * Kp, sizeof(double) * Kp, cudaMemcpyDeviceToDevice, cs));
            blaunch(kb_init<J, R>, vg, VTPB, cs, n, (const double*)B.b.p, B.x.p, B.r.p, B.r32.p, B.partial.p, h.counter.p + 1, B.S.p, ord);
        });
        cudaGraphNode_t w2;
        brec_loop<J, R, VT>(h, g, cs, l2.data(), l2.size(), &w2);
    }
    cudaGraphExec_t ge;
    CPC_CK(cudaGraphInstantiate(&ge, g, 0));
    B.graph = g;
    B.gexec = ge;
}


// Block PCG loop on the packed block vectors of h.bat (K <= Kp <= 64).  Each iteration:
//   Q = A P;  alpha = (P^T Q)^{-1} gamma;  X += P alpha, R -= Q alpha;  stop when every column
//   has ||r_k|| / ||b_k|| < tol;  Z = M R;  beta = gamma^{-1} (Z^T R);  gamma = Z^T R;  P = Z + P beta.
// The host reads two flags per iteration (one stream synchronisation).
template <int J, int R, class VT>
int solve_block_t(Handle& h, int K, const double* b, double* x, double tol, int maxit, int* iters, double* res) {
    Batched& B = h.bat;
    const int Kp = B.Kp, n = h.n;
    cudaStream_t s = h.s;
    const int64_t nk = (int64_t)n * Kp;
    auto km = [&](int i) { return B.kmat.p + (size_t)i * Kp * Kp; };
    constexpr int KP = Cols<J, R>::KP;
    const size_t gram_smem = 2 * (size_t)KK_ELEMS * sizeof(double);
    const size_t solve_smem = 2 * (size_t)K * K * sizeof(double);
    const size_t upd_smem = ((size_t)Kp * Kp + BWARPS * R * Kp) * sizeof(double);
    const size_t pup_smem = (size_t)Kp * Kp * sizeof(double);
    CPC_CK(cudaFuncSetAttribute(kk_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 64 * 64 * (int)sizeof(double)));
    const Csr& A = h.lev[0].A;
    VT* z = (VT*)B.z.p;
    auto gram = [&](const auto* U, const double* V, double* out) {
        kk_gram<KP><<<KK_GRID, KK_TPB, gram_smem, s>>>(n, U, V, B.kpart.p);
        kk_gram_sum<<<(Kp * Kp + 7) / 8, 256, 0, s>>>(KK_GRID, Kp, B.kpart.p, out);
    };
    int flags[KF_COUNT] = {0, 0};
    auto read_flags = [&]() {
        CPC_LAUNCH_CK();
        CPC_CK(cudaMemcpyAsync(flags, B.kflag.p, sizeof(flags), cudaMemcpyDeviceToHost, s));
        CPC_CK(cudaStreamSynchronize(s));
    };
    CPC_CK(cudaMemsetAsync(B.kflag.p, 0, sizeof(int) * KF_COUNT, s));
    CPC_CK(cudaMemsetAsync(B.kmat.p, 0, sizeof(double) * KM_COUNT * Kp * Kp, s));
    kb_pack<<<152 * 8, 256, 0, s>>>(n, K, Kp, b, B.b.p);
    kk_init<J, R><<<KK_GRID, BTPB, 0, s>>>(n, B.b.p, B.x.p, B.r.p, B.r32.p, B.kpart.p);
    kk_check<<<1, 256, 0, s>>>(KK_GRID, Kp, K, B.kpart.p, B.kvec.p, tol, 1, B.kflag.p);
    read_flags();
    if (flags[KF_BAD]) fail(CPC_EINVAL, "a right-hand-side column is zero or not finite");
    brec_precond<Gather<J, R, VT>::j, Gather<J, R, VT>::r, VT>(h, h.opt.precond, bres<VT>(B), z, s);       // Z = M R
    kk_copy<VT><<<2048, 256, 0, s>>>(nk, (const VT*)z, B.p.p);         // P = Z
    gram((const VT*)z, B.r.p, km(KM_GAMMA));                           // gamma = Z^T R
    int status = CPC_ENOCONV, it = 0;
    for (int k = 1; k <= maxit; ++k) {
        kk_spmm<J, R><<<rows_grid<R>(n), BTPB, 0, s>>>(n, A.ptr.p, A.col.p, A.val.p, (const double*)B.p.p, B.q.p);
        gram((const double*)B.p.p, B.q.p, km(KM_PQ));
        kk_solve<<<1, KK_TPB, solve_smem, s>>>(K, Kp, km(KM_PQ), km(KM_GAMMA), km(KM_ALPHA), nullptr, B.kflag.p);
        kk_update<J, R><<<KK_GRID, BTPB, upd_smem, s>>>(n, K, B.x.p, B.r.p, B.r32.p, B.p.p, B.q.p, km(KM_ALPHA), B.kpart.p,
                                                       B.kflag.p);
        kk_check<<<1, 256, 0, s>>>(KK_GRID, Kp, K, B.kpart.p, B.kvec.p, tol, 0, B.kflag.p);
        read_flags();
        if (flags[KF_BAD]) {                                           // X holds iteration k - 1
            status = CPC_EBREAKDOWN;
            it = k - 1;
            break;
        }
        it = k;
        if (flags[KF_DONE]) {
            status = CPC_OK;
            break;
        }
        if (k == maxit) break;
        brec_precond<Gather<J, R, VT>::j, Gather<J, R, VT>::r, VT>(h, h.opt.precond, bres<VT>(B), z, s);   // Z = M R
        gram((const VT*)z, B.r.p, km(KM_GAMMA_NEW));                   // Z^T R
        kk_solve<<<1, KK_TPB, solve_smem, s>>>(K, Kp, km(KM_GAMMA), km(KM_GAMMA_NEW), km(KM_BETA), km(KM_GAMMA),
                                               B.kflag.p);
        kk_pupdate<J, R, VT><<<KK_GRID, BTPB, pup_smem, s>>>(n, K, (const VT*)z, B.p.p, km(KM_BETA), B.kflag.p);
    }
    kb_unpack<<<152 * 8, 256, 0, s>>>(n, K, Kp, (const double*)B.x.p, x);
    CPC_LAUNCH_CK();
    std::vector<double> hv((size_t)KV_COUNT * Kp);
    CPC_CK(cudaMemcpyAsync(hv.data(), B.kvec.p, sizeof(double) * hv.size(), cudaMemcpyDeviceToHost, s));
    CPC_CK(cudaStreamSynchronize(s));
    *iters = it;
    if (res)
        for (int c = 0; c < K; ++c) res[c] = hv[(size_t)KV_RES * Kp + c];
    return status;
}

}  // namespace

void destroy_batched(Handle& h) {
    Batched& B = h.bat;
    if (B.gexec) cudaGraphExecDestroy(B.gexec);
    if (B.graph) cudaGraphDestroy(B.graph);
    B.gexec = nullptr;
    B.graph = nullptr;
}

// Columns the block vectors are padded to.
static int padded(int K) { return K <= 8 ? 8 : K <= 16 ? 16 : (K + 31) / 32 * 32; }

// Calls f(J, R) with the layout of Kp columns.
template <class F>
static auto with_cols(int Kp, F&& f) {
    using std::integral_constant;
    switch (Kp) {
        case 8: return f(integral_constant<int, 1>{}, integral_constant<int, 4>{});
        case 16: return f(integral_constant<int, 1>{}, integral_constant<int, 2>{});
        case 32: return f(integral_constant<int, 1>{}, integral_constant<int, 1>{});
        case 64: return f(integral_constant<int, 2>{}, integral_constant<int, 1>{});
        case 96: return f(integral_constant<int, 3>{}, integral_constant<int, 1>{});
        default: return f(integral_constant<int, 4>{}, integral_constant<int, 1>{});
    }
}

// Allocate the block vectors for K columns (kept across calls with the same padded width).
static void ensure_batched(Handle& h, int K, bool adjoint) {
    Batched& B = h.bat;
    const int Kp = padded(K);
    if (Kp > 128) fail(CPC_EINVAL, "at most 128 right-hand sides per batched call");
    const bool fp64 = h.opt.precision == CPC_PREC_FP64;
    const size_t vsz = fp64 ? sizeof(double) : sizeof(float);
    if (B.Kp != Kp) {
        destroy_batched(h);
        B = Batched{};
        const size_t nk = (size_t)h.n * Kp;
        B.b.alloc(nk); B.x.alloc(nk); B.r.alloc(nk); B.p.alloc(nk); B.q.alloc(nk); B.xfwd.alloc(nk);
        B.z.alloc(nk * vsz); B.t.alloc(nk * vsz); B.y.alloc(nk * vsz);
        if (!fp64) B.r32.alloc(nk);
        const int nl = (int)h.lev.size();
        B.lx.resize(nl); B.lf.resize(nl); B.lr.resize(nl);
        for (int l = 0; l < nl; ++l) {
            const size_t m = (size_t)h.lev[l].n * Kp * vsz;
            B.lx[l].alloc(m); B.lf[l].alloc(m); B.lr[l].alloc(m);
        }
        B.S.alloc((size_t)NB_STATE * Kp);
        B.partial.alloc((size_t)152 * 32 * Kp);
        B.kfwd.alloc(2 * (size_t)Kp);
        if (Kp <= 64) {
            B.kmat.alloc((size_t)KM_COUNT * Kp * Kp);
            B.kpart.alloc((size_t)KK_GRID * Kp * Kp);
            B.kvec.alloc((size_t)KV_COUNT * Kp);
            B.kflag.alloc(KF_COUNT);
        }
        B.Kp = Kp;                          // only now: a failed allocation leaves no layout behind
    }
    if (B.gexec && B.adjoint != adjoint) destroy_batched(h);
    B.adjoint = adjoint;
}

void solve_batched(Handle& h, int K, const double* b, double* x, double* lambda, double tol, int maxit,
                   int* iters, int* status, int* iters_adj, int* status_adj) {
    ensure_batched(h, K, lambda != nullptr);
    Batched& B = h.bat;
    const int Kp = B.Kp, n = h.n;
    if (!B.gexec)
        with_cols(Kp, [&](auto j, auto r) {
            constexpr int J = decltype(j)::value, R = decltype(r)::value;
            if (h.opt.precision == CPC_PREC_FP64) build_batched_graph<J, R, double>(h, lambda != nullptr);
            else build_batched_graph<J, R, float>(h, lambda != nullptr);
        });
    cudaStream_t s = h.s;
    std::vector<double> st((size_t)NB_STATE * Kp, 0.0);
    for (int c = 0; c < Kp; ++c) {
        st[(size_t)S_TOL * Kp + c] = tol;
        st[(size_t)S_MAXIT * Kp + c] = c < K ? (double)maxit : 0.0;
    }
    CPC_CK(cudaMemcpyAsync(B.S.p, st.data(), sizeof(double) * st.size(), cudaMemcpyHostToDevice, s));
    kb_pack<<<152 * 8, 256, 0, s>>>(n, K, Kp, b, B.b.p);
    CPC_CK(cudaGraphLaunch(B.gexec, s));
    kb_unpack<<<152 * 8, 256, 0, s>>>(n, K, Kp, (const double*)(lambda ? B.xfwd.p : B.x.p), x);
    if (lambda) kb_unpack<<<152 * 8, 256, 0, s>>>(n, K, Kp, (const double*)B.x.p, lambda);
    CPC_LAUNCH_CK();
    CPC_CK(cudaMemcpyAsync(st.data(), B.S.p, sizeof(double) * st.size(), cudaMemcpyDeviceToHost, s));
    std::vector<double> kf(2 * (size_t)Kp, 0.0);
    if (lambda) CPC_CK(cudaMemcpyAsync(kf.data(), B.kfwd.p, sizeof(double) * 2 * Kp, cudaMemcpyDeviceToHost, s));
    CPC_CK(cudaStreamSynchronize(s));
    for (int c = 0; c < K; ++c) {
        const int ki = (int)st[(size_t)S_K * Kp + c];
        const int si = (int)st[(size_t)S_STATUS * Kp + c];
        if (lambda) {
            iters[c] = (int)kf[c];
            if (status) status[c] = (int)kf[Kp + c];
            if (iters_adj) iters_adj[c] = ki;
            if (status_adj) status_adj[c] = si;
        } else {
            iters[c] = ki;
            if (status) status[c] = si;
        }
    }
}

int solve_block(Handle& h, int K, const double* b, double* x, double tol, int maxit, int* iters, double* res) {
    if (K < 1 || K > 64) fail(CPC_EINVAL, "block CG takes 1 to 64 right-hand sides");
    if (h.opt.precond == CPC_PRECOND_AMG_ILU) fail(CPC_EINVAL, "block CG supports B_co, AMG, IC(0) and B^");
    ensure_batched(h, K, false);
    return with_cols(h.bat.Kp, [&](auto j, auto r) {
        constexpr int J = decltype(j)::value, R = decltype(r)::value;
        if constexpr (J <= 2) {
            if (h.opt.precision == CPC_PREC_FP64) return solve_block_t<J, R, double>(h, K, b, x, tol, maxit, iters, res);
            return solve_block_t<J, R, float>(h, K, b, x, tol, maxit, iters, res);
        } else {
            return (int)CPC_EINVAL;
        }
    });
}

}  // namespace cpc
