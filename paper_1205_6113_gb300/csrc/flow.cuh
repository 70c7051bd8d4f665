// flow.cuh -- Gauss-Seidel sweeps and triangular solves as one launch each, rows ordered by their
// data instead of by launches.
#pragma once

#include "device.cuh"

namespace cpc {

// What a flow launch computes per row i (new: written by this launch, old: before it).
enum FlowMode {
    FLOW_FWD0 = 0,   // x_i = (f_i - sum_low a_ij x_j(new)) / a_ii: forward sweep from a zero guess
    FLOW_FWD = 1,    // x_i = (f_i - sum_low a_ij x_j(new) - sum_up a_ij x_j(old)) / a_ii
    FLOW_BWD = 2,    // x_i = (f_i - sum_up a_ij x_j(new) - sum_low a_ij x_j(old)) / a_ii, groups descending
    FLOW_LOWER = 3,  // y_i = t_i - sum_j l_ij y_j(new): unit lower factor, all of the row new
    FLOW_UPPER = 4   // w_i = (y_i - sum_j u_ij w_j(new)) / u_ii: upper factor, all of the row new
};

// A value not yet written by the running launch: a signalling NaN with a payload no kernel
// computes.  It is only ever moved and compared as an integer.
template <class VT> struct Unset;
template <> struct Unset<double> {
    using B = unsigned long long;
    static constexpr B bits = 0x7FF4C0DE5EED0001ull, nan = 0x7FF8000000000000ull;
};
template <> struct Unset<float> {
    using B = unsigned;
    static constexpr B bits = 0x7FA5EED1u, nan = 0x7FC00000u;
};

// Marks p unset, for the kernels that prepare a flow's output vector.
template <class VT>
__device__ __forceinline__ void flow_unset(VT* p) {
    *reinterpret_cast<typename Unset<VT>::B*>(p) = Unset<VT>::bits;
}

// Records a flow launch over all chunks of S.  f: right-hand side; xo: old values; xn: new values,
// unset on entry except where a row is already known; unset: own-row elements marked unset once f
// has been read (may be null, may be f's own storage); zadd: += the new value (may be null).
// ctr: a counter of this launch's own, 0 on entry and on exit; err: set to 1 when a wait gave up, after
// polls polls (0: a number that follows from S, flow.cu).  Every element of xn is written all the same.
template <class FT, class VT>
void rec_flow(FlowMode mode, const Sell& S, VType vt, const FT* f, const VT* xo, VT* xn, VT* unset, VT* zadd,
              unsigned* ctr, int* err, int polls, cudaStream_t s);

}  // namespace cpc
