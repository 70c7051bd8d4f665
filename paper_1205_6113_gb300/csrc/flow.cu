// flow.cu -- sweeps whose dependent steps are ordered by the data (see flow.cuh).
//
// A Gauss-Seidel sweep over g colours, or a triangular solve over g wavefronts, is a chain of g
// dependent steps.  One launch per step costs 1.2-3.9 us each, most of it launch and drain latency.
// Here the whole sweep is one launch: a warp takes one chunk of rows, loads the chunk's matrix data,
// then the new values it depends on, and loads again those that are still unset.  A value is its
// own flag (one aligned 4- or 8-byte store), so a step costs one trip through L2 and no fence, and
// chunks that are not on the chain overlap with it.
//
// Order and progress: chunks are handed out by a counter in group order, and a chunk depends only on
// rows of earlier groups, hence on chunks that running warps already hold; so whatever the
// scheduling, the earliest unfinished chunk never waits for one that has not started.  Sums are
// taken in entry order whatever the order of arrival, so results are reproducible to the bit.
// A wait gives up after a number of polls: it takes NaN for what is missing and sets *err.
#include "flow.cuh"
#include "handle.cuh"

namespace cpc {

namespace {

// Polls (a quarter of a microsecond each) after which a wait gives up: a chunk waits at most for the chunks
// in flight, one after another, each of `batches` batches of some ten polls; three times that, and at
// least half a second.
inline int flow_polls(int64_t chunks, int64_t batches) {
    return (int)std::min<int64_t>(std::max<int64_t>(32 * chunks * batches, 1 << 21), 1 << 30);
}

// v = *p if on, else v unchanged: a predicated load and no branch, so that the loads of a batch are
// all in flight before the first value is looked at (with a branch per load a poll took a round
// trip per entry: 77 against 29 us per sweep of the second coarse level at 1M).
__device__ __forceinline__ void flow_ld(unsigned long long& v, const double* p, bool on) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.relaxed.gpu.global.b64 %0, [%1];\n\t}"
                 : "+l"(v) : "l"(p), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void flow_ld(unsigned& v, const float* p, bool on) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.relaxed.gpu.global.b32 %0, [%1];\n\t}"
                 : "+r"(v) : "l"(p), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void flow_st(double* p, double v) {
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b == Unset<double>::bits) b = Unset<double>::nan;
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}
__device__ __forceinline__ void flow_st(float* p, float v) {
    unsigned b = __float_as_uint(v);
    if (b == Unset<float>::bits) b = Unset<float>::nan;
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(b) : "memory");
}
__device__ __forceinline__ double flow_val(unsigned long long b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ float flow_val(unsigned b) { return __uint_as_float(b); }

// Batch of up to M entries per lane of one part of a chunk: entries o, o + 32, ... < e.
template <int M, class VT, class MT>
struct FlowBatch {
    int c[M];
    VT v[M];
    int m;                                // entries per lane (warp-uniform), at most M
    __device__ __forceinline__ void load(const int* __restrict__ col, const MT* __restrict__ val, int o, int e, int left) {
        m = left < M ? left : M;
#pragma unroll
        for (int u = 0; u < M; ++u) {
            const int oo = o + u * 32;
            c[u] = oo < e ? col[oo] : -1;
            v[u] = oo < e ? Cv<VT>::f(val[oo]) : VT(0);
        }
    }
    __device__ __forceinline__ void add_old(const VT* x, VT& acc) {
        VT xv[M];
#pragma unroll
        for (int u = 0; u < M; ++u) xv[u] = c[u] >= 0 ? x[c[u]] : VT(0);
#pragma unroll
        for (int u = 0; u < M; ++u) {
            if (u >= m) break;
            acc += v[u] * xv[u];
        }
    }
    __device__ __forceinline__ void add_new(const VT* x, VT& acc, int* err, int polls) {
        using U = Unset<VT>;
        typename U::B b[M];
#pragma unroll
        for (int u = 0; u < M; ++u) {
            b[u] = 0;
            flow_ld(b[u], x + max(c[u], 0), c[u] >= 0);
        }
        for (int spin = 0;; ++spin) {
            bool miss = false;
#pragma unroll
            for (int u = 0; u < M; ++u) miss |= b[u] == U::bits;
            if (!__any_sync(0xffffffffu, miss)) break;
            if (spin == polls) {
                if (miss) *err = 1;
#pragma unroll
                for (int u = 0; u < M; ++u) b[u] = b[u] == U::bits ? U::nan : b[u];
                break;
            }
#pragma unroll
            for (int u = 0; u < M; ++u) flow_ld(b[u], x + max(c[u], 0), b[u] == U::bits);
        }
#pragma unroll
        for (int u = 0; u < M; ++u) {
            if (u >= m) break;
            acc += v[u] * flow_val(b[u]);
        }
    }
    // The same over a row whose entries keep their order: the new values of one part, the old ones of
    // the other, told apart by the mark.  MODE FLOW_FWD0 takes no old ones (they are zero).
    template <int MODE>
    __device__ __forceinline__ void add_mixed(const VT* xo, const VT* xn, VT& acc, int* err, int polls) {
        using U = Unset<VT>;
        typename U::B b[M];
        auto on = [&](int u) { return MODE == FLOW_FWD0 ? takes(c[u]) : c[u] != -1; };
        auto from = [&](int u) { return on(u) ? (is_later(c[u]) == (MODE == FLOW_BWD) ? xn : xo) + marked_col(c[u]) : xn; };
#pragma unroll
        for (int u = 0; u < M; ++u) {
            b[u] = 0;
            flow_ld(b[u], from(u), on(u));
        }
        for (int spin = 0;; ++spin) {
            bool miss = false;
#pragma unroll
            for (int u = 0; u < M; ++u) miss |= b[u] == U::bits;
            if (!__any_sync(0xffffffffu, miss)) break;
            if (spin == polls) {
                if (miss) *err = 1;
#pragma unroll
                for (int u = 0; u < M; ++u) b[u] = b[u] == U::bits ? U::nan : b[u];
                break;
            }
#pragma unroll
            for (int u = 0; u < M; ++u) flow_ld(b[u], from(u), b[u] == U::bits);
        }
#pragma unroll
        for (int u = 0; u < M; ++u) acc += v[u] * flow_val(b[u]);
    }
};

// WIDE: blocks of four warps, one chunk each.  Else blocks of one warp, which takes one chunk after
// another until none is left, and no shared memory: next to kernels without any, a block that wants some
// waits for an SM to empty before it can start (the IC(0) solves above: 190 us more an application).
template <class MT, class DT, class FT, class VT, int MODE, int M, bool WIDE>
__global__ void __launch_bounds__(WIDE ? 128 : 32) k_flow(SV<MT, DT> A, const int* __restrict__ cmid, int nchunks, const FT* f,
                                             const VT* xo, VT* xn, VT* unset, VT* zadd, unsigned* ctr, int* err, int polls) {
    constexpr bool UP = MODE == FLOW_BWD;
    constexpr bool TRI = MODE == FLOW_LOWER || MODE == FLOW_UPPER;
    // FP32 rows keep their entries in column order, the two parts mixed
    constexpr bool MIX = std::is_same<VT, float>::value && !TRI;
    constexpr bool OLD = !MIX && (MODE == FLOW_FWD || MODE == FLOW_BWD);
    const int lane = threadIdx.x & 31, C = A.C, r = lane & (C - 1), g = lane / C, o = g * C + r;
    bool waited = false;
    do {
        unsigned q = 0;
        if constexpr (WIDE) {
            __shared__ unsigned ticket;
            if (threadIdx.x == 0) ticket = atomicInc(ctr, gridDim.x - 1);
            __syncthreads();
            q = ticket * (blockDim.x >> 5) + (threadIdx.x >> 5);
        } else {
            // every warp draws once more than it has chunks, and the counter wraps to 0 at the last draw
            if (lane == 0) q = atomicInc(ctr, (unsigned)nchunks + gridDim.x - 1);
            q = __shfl_sync(0xffffffffu, q, 0);
        }
        if (q >= (unsigned)nchunks) return;
        const int k = UP ? nchunks - 1 - (int)q : (int)q;
        const int s = k * C + r;
        const int row = A.perm[s];
        const bool own = g == 0 && row >= 0;
        // [nb, ne): the entries with new values, [ob, oe): those with old values
        const int b0 = A.cptr[k], b2 = A.cptr[k + 1], b1 = TRI || MIX ? b2 : cmid[k];
        const int nb = UP && !MIX ? b1 : b0, ne = UP ? b2 : b1, ob = UP ? b0 : b1, oe = UP ? b1 : b2;
        FlowBatch<M, VT, MT> bn, bo;
        bn.load(A.col, A.val, nb + o, ne, (ne - nb + 31) >> 5);
        if (OLD) bo.load(A.col, A.val, ob + o, oe, (oe - ob + 31) >> 5);
        const VT dinv = MODE != FLOW_LOWER && own ? Cv<VT>::f(A.diag[s]) : VT(1);
        if (!waited) {
            pdl_wait();
            pdl_launch_dependents();
            waited = true;
        }
        VT fr = VT(0), zr = VT(0);
        if (own) {
            fr = Cv<VT>::f(f[row]);
            if (MODE == FLOW_UPPER && zadd) zr = zadd[row];
        }
        VT acc = VT(0);
        if (OLD) {
            bo.add_old(xo, acc);
            for (int p = 32 * M; p < oe - ob; p += 32 * M) {
                bo.load(A.col, A.val, ob + p + o, oe, (oe - ob - p + 31) >> 5);
                bo.add_old(xo, acc);
            }
        }
        auto add = [&] {
            if constexpr (MIX) bn.template add_mixed<MODE>(xo, xn, acc, err, polls);
            else bn.add_new(xn, acc, err, polls);
        };
        add();
        for (int p = 32 * M; p < ne - nb; p += 32 * M) {
            bn.load(A.col, A.val, nb + p + o, ne, (ne - nb - p + 31) >> 5);
            add();
        }
        for (int w = C; w < 32; w <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, w);
        if (own) {
            const VT x = MODE == FLOW_LOWER ? fr - acc : (fr - acc) * dinv;
            if (TRI && unset) flow_unset(unset + row);
            flow_st(xn + row, x);
            if (MODE == FLOW_UPPER && zadd) zadd[row] = zr + x;
        }
    } while (!WIDE);
}

int flow_sms() {
    static const int sms = [] {
        int dev = 0, n = 0;
        CPC_CK(cudaGetDevice(&dev));
        CPC_CK(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
        return n;
    }();
    return sms;
}

// Calls f(std::integral_constant<int, M>{}) with the batch of a kernel whose lanes hold at most `lanes` entries.
template <class F>
void with_m(int lanes, F&& f) {
    if (lanes <= 4) f(std::integral_constant<int, 4>{});
    else if (lanes <= 8) f(std::integral_constant<int, 8>{});
    else f(std::integral_constant<int, 16>{});
}

// Most entries that a lane takes of a row's new or old values: of one part in FP64, of the mixed row in FP32.
inline int sweep_lanes(const Sell& S, bool fp64) { return fp64 ? std::max(S.lanes_lo, S.lanes_up) : S.lanes; }

template <int MODE, class MT, class DT, class FT, class VT>
void flow_mode(const Sell& S, SV<MT, DT> v, const FT* f, const VT* xo, VT* xn, VT* unset, VT* zadd, unsigned* ctr,
               int* err, int polls, cudaStream_t s) {
    // Chunks in flight: four groups' worth, enough to have the matrix data of a chunk on hand when its
    // turn comes, and no more, since waiting warps slow the working ones down (IC(0) of 120,000 cells,
    // 25 chunks a level: 250 us with every chunk in flight, 150 with 304).  Where that is most of what
    // fits, blocks of four warps: one-warp blocks stop at 32 warps an SM and draw on the counter, 1.3 ns
    // a draw, once per chunk (18,000 chunks: 24 us against 15).
    const int ahead = std::max(2 * flow_sms(), (int)(4 * (int64_t)S.nchunks / std::max<int>(1, (int)S.seg.size() - 1)));
    const bool wide = ahead > 16 * flow_sms();
    const int lanes = MODE == FLOW_LOWER || MODE == FLOW_UPPER ? S.lanes : sweep_lanes(S, std::is_same<VT, double>::value);
    auto go = [&](auto m) {
        constexpr int M = decltype(m)::value;
        if (polls <= 0) polls = flow_polls(std::min(S.nchunks, wide ? 64 * flow_sms() : ahead), (lanes + M - 1) / M);
        if (wide)
            launch(k_flow<MT, DT, FT, VT, MODE, M, true>, (S.nchunks + 3) / 4, 128, s, v, (const int*)S.cmid.p, S.nchunks, f,
                   xo, xn, unset, zadd, ctr, err, polls);
        else
            launch(k_flow<MT, DT, FT, VT, MODE, M, false>, std::min(S.nchunks, ahead), 32, s, v, (const int*)S.cmid.p,
                   S.nchunks, f, xo, xn, unset, zadd, ctr, err, polls);
    };
    with_m(lanes, go);
}

// Warps of a level's sweep that the GPU holds at once.
template <class MT, class VT>
int flow_resident(int lanes) {
    int blocks = 0;
    with_m(lanes, [&](auto m) {
        CPC_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_flow<MT, VT, VT, VT, FLOW_FWD, decltype(m)::value, true>, 128, 0));
    });
    return 4 * blocks * flow_sms();
}

}  // namespace

// Wide colours fill the GPU for longer than a launch takes to start, and their launches keep more warps
// resident than a flow's waiting ones: 32,000 rows a colour (level 1 at 1M) take 49 us by launches and 50 by
// flow in FP64, 26 and 32 in FP32; 12,000 rows a colour 16.2 and 14.7 (FP32, 395,000 cells), 4,500 rows a colour
// 61 and 28.  Below that the chunks of a colour count, against the warps that the GPU holds (fewer where a
// lane takes 16 entries at a time): once they are not all resident a flow waits for its own chunks.  Launches and
// flow, us a full sweep, at chunks a colour per resident warp: FP64 0.83 68 and 57, 0.94 76 and 70, 1.02 59 and
// 53, 1.12 75 and 77, 1.49 67 and 85, 2.6 103 and 161 (with the sweep from zero, half a row, two cycles at 1.12
// 1,884 and 1,858, at 1.25 2,048 and 2,042, at 1.40 2,217 and 2,225; with at most 8 entries to a lane, at 1.32
// 1,838 and 1,773, at 1.58 2,192 and 2,151); FP32, which polls every entry of a row, 0.42
// 19 and 16, 0.66 47 and 42, 0.71 46 and 45, 0.84 46 and 54, 1.25 36 and 59, 2.0 52 and 115, and 83 and 109 at
// 0.55 with 30 entries to a lane, two batches.
bool gs_by_flow(const Sell& S, int n, VType vt) {
    constexpr int FLOW_ROWS = 24000;
    const int g = std::max(1, (int)S.seg.size() - 1), lanes = sweep_lanes(S, vt == VT_F64);
    if (n / g > FLOW_ROWS) return false;
    const double per = (double)S.nchunks / g;
    if (vt == VT_F64) return per <= (lanes <= 8 ? 1.6 : 1.25) * flow_resident<double, double>(lanes);
    const int res = vt == VT_BF16 ? flow_resident<__nv_bfloat16, float>(lanes) : flow_resident<float, float>(lanes);
    return per * std::max(1.0, lanes / 16.0) <= 0.75 * res;
}

template <class FT, class VT>
void rec_flow(FlowMode mode, const Sell& S, VType vt, const FT* f, const VT* xo, VT* xn, VT* unset, VT* zadd,
              unsigned* ctr, int* err, int polls, cudaStream_t s) {
    if (S.nchunks == 0) return;
    auto go = [&](auto v, auto md) {
        flow_mode<decltype(md)::value>(S, v, f, xo, xn, unset, zadd, ctr, err, polls, s);
    };
    auto sweep = [&](auto v) {
        if (mode == FLOW_FWD0) go(v, std::integral_constant<int, FLOW_FWD0>{});
        else if (mode == FLOW_FWD) go(v, std::integral_constant<int, FLOW_FWD>{});
        else go(v, std::integral_constant<int, FLOW_BWD>{});
    };
    auto solve = [&](auto v) {
        if (mode == FLOW_LOWER) go(v, std::integral_constant<int, FLOW_LOWER>{});
        else go(v, std::integral_constant<int, FLOW_UPPER>{});
    };
    auto flagged = [&](auto v) {
        v.col = S.fcol.p;
        return v;
    };
    const bool tri = mode == FLOW_LOWER || mode == FLOW_UPPER;
    if constexpr (std::is_same<VT, double>::value) {
        const auto v = view(S, (const double*)S.val.p, (const double*)S.dinv.p);
        if (tri) solve(v);
        else sweep(v);
    } else {
        if (tri) solve(view(S, (const float*)S.val32.p, (const float*)S.dinv32.p));
        else if (vt == VT_BF16) {
            if constexpr (std::is_same<FT, float>::value) sweep(flagged(view(S, (const __nv_bfloat16*)S.val16.p, (const float*)S.dinv32.p)));
        } else {
            sweep(flagged(view(S, (const float*)S.val32.p, (const float*)S.dinv32.p)));
        }
    }
    CPC_LAUNCH_CK();
}

template void rec_flow<double, double>(FlowMode, const Sell&, VType, const double*, const double*, double*, double*,
                                       double*, unsigned*, int*, int, cudaStream_t);
template void rec_flow<double, float>(FlowMode, const Sell&, VType, const double*, const float*, float*, float*, float*,
                                      unsigned*, int*, int, cudaStream_t);
template void rec_flow<float, float>(FlowMode, const Sell&, VType, const float*, const float*, float*, float*, float*,
                                     unsigned*, int*, int, cudaStream_t);

}  // namespace cpc
