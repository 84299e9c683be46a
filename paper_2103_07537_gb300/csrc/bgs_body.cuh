// Device-side building blocks of the block Gauss-Seidel smoother of
// Algorithm 1 (Sec. 4.3.2) shared by the per-colour kernels (k_solve.cu), the
// staged kernel (k_staged.cu) and the persistent sweep kernel (k_sweep.cu): the
// row sums of one field step and the update of a finished node.  Vectors are
// read through L2 (load_cg), see pdl_wait.
#pragma once

#include "common.cuh"

namespace bamg {

// One block of a field step of the smoother.  From a given iterate the step
// works in place on x_in: a finished node carries x_in + x~ in its field-f
// entries, so row f0 + r of A_{f,*} x_in + A_ff x~ (x~ of the lower colours)
// is one product per block with the neighbour's current entries -- one gather
// and B products, where x_in and x~ kept apart need two gathers, the colour
// flag and B + FB products.  The higher colours' nodes still hold x_in, and
// the nodes of one colour do not couple (the pattern is structurally symmetric:
// the setup refuses others), so no entry is read while its node is updated.  From the zero iterate (no x_in) the lower colours' x~ alone
// contribute.  arow = row f0 + r of the block; forced inline so that it stays
// in registers.
template <typename T, int B, int FB>
__device__ __forceinline__ void bgs_block(const BgsArgs& a, const T* xt, const T* x_in, int j, const T (&arow)[B],
                                          bool lower, T& acc) {
    if (x_in) {
        T xv[B];
        load_cg<T, B>(x_in + (size_t)j * B, xv);
#pragma unroll
        for (int c = 0; c < B; ++c) acc = fma(arow[c], xv[c], acc);
    } else if (lower) {
        T tv[FB];
        load_cg<T, FB>(xt + (size_t)j * FB, tv);
        // the field-f columns of the row, picked by selects over compile-time
        // register indices (an index computed from the field would put arow
        // in local memory)
#pragma unroll
        for (int c = 0; c < FB; ++c) {
            T av = arow[c];
#pragma unroll
            for (int ff = 1; ff < B / FB; ++ff) av = (ff == a.field) ? arow[ff * FB + c] : av;
            acc = fma(av, tv[c], acc);
        }
    }
}

// Node i's entries after its solve (m = field of the entry, e = its index in
// the vectors): x_out takes x_in with field f corrected by omega x~, and x_in
// itself becomes x_in + x~ in field f for the colours that follow.
template <typename T>
__device__ __forceinline__ void bgs_store(const BgsArgs& a, const T* x_in, size_t e, bool own, T xn, T om) {
    T v = x_in ? ld_cg(x_in + e) : T(0);
    if (own) {
        if (x_in) const_cast<T*>(x_in)[e] = v + xn;
        v = fma(om, xn, v);
    }
    static_cast<T*>(a.x_out)[e] = v;
}

template <typename T>
__device__ __forceinline__ T bgs_omega(const BgsArgs& a, int i) {
    return a.omega_node ? static_cast<const T*>(a.omega_node)[(size_t)i * a.F + a.field] : T(a.omega);
}

// the blocks kf, kf + S, kf + 2S, ... (< k1) of one matrix row, accumulated
// in that order into acc (bgs_block per block).  Software-pipelined: the
// next block's colour flag, column and matrix row are loaded before the
// current block's gathers, so each step waits for one gather latency rather
// than the column load followed by its gather.  The first block (column jf,
// flag lowf, row arf) is loaded by the caller, before its wait on the
// previous kernel; vb is the row's first block, VS the stride between
// blocks.  XIN: x_in is set (every block contributes; without it only blocks
// of lower colour do, and the others' rows are not loaded) -- a template
// flag, so that the loads of the next block do not wait on its colour flag.
template <typename T, int B, int FB, int S, bool XIN>
__device__ __forceinline__ void bgs_walk_x(const BgsArgs& a, const T* xt, const T* x_in, const T* __restrict__ vb,
                                           int VS, int k0, int kf, int k1, int jf, bool lowf, const T (&arf)[B],
                                           T& acc) {
    int j = jf;
    bool lw = lowf;
    T ar[B];
#pragma unroll
    for (int c = 0; c < B; ++c) ar[c] = arf[c];
#pragma unroll 2
    for (int k = kf;; k += S) {
        const int kn = k + S;
        const bool more = kn < k1;
        bool lwn = false;
        int jn = 0;
        T an[B];
        if (more) {
            if (!XIN) lwn = __ldg(a.lowk + kn) != 0;
            jn = __ldg(a.ci + kn);
            if (XIN || lwn) load_row<T, B>(vb + (size_t)(kn - k0) * VS, an);
        }
        if (XIN || lw) bgs_block<T, B, FB>(a, xt, XIN ? x_in : nullptr, j, ar, lw, acc);
        if (!more) break;
        j = jn;
        lw = lwn;
#pragma unroll
        for (int c = 0; c < B; ++c) ar[c] = an[c];
    }
}

template <typename T, int B, int FB, int S>
__device__ __forceinline__ void bgs_walk(const BgsArgs& a, const T* xt, const T* x_in, const T* __restrict__ vb,
                                         int VS, int k0, int kf, int k1, int jf, bool lowf, const T (&arf)[B],
                                         T& acc) {
    if (x_in) bgs_walk_x<T, B, FB, S, true>(a, xt, x_in, vb, VS, k0, kf, k1, jf, lowf, arf, acc);
    else bgs_walk_x<T, B, FB, S, false>(a, xt, x_in, vb, VS, k0, kf, k1, jf, lowf, arf, acc);
}

// Blocks of one row whose loads a thread issues together in the thread-per-row
// kernels (rows of 27 or 9 blocks split over 1 or 4 lanes): as many as keep the
// matrix rows and gathered vectors of a batch within 40 registers.
template <typename T, int B>
struct RowBatch {
    static constexpr int kRegs = 2 * B * (int)sizeof(T) / 4;
    static constexpr int kU = 40 / kRegs < 1 ? 1 : 40 / kRegs > 4 ? 4 : 40 / kRegs;
};

// The row sum of one thread: blocks kf, kf + G, ... (< k1), in that order, in
// batches whose columns and matrix rows are loaded together and then their
// gathers together.  (A rolled or unrolled loop waits for one block's column
// and gather after another: rows of 7 blocks per lane never reach the body of
// an eightfold unrolled loop.)  The first batch's columns and rows are loaded
// before the wait on the previous kernel.
template <typename T, int B, int FB, int G, int VS, bool XIN>
__device__ __forceinline__ T bgs_row_sum(const BgsArgs& a, const T* xt, const T* x_in, const T* __restrict__ vb,
                                         int k0, int kf, int k1) {
    constexpr int U = RowBatch<T, B>::kU;
    T acc = T(0);
    bool first = true;
    for (int k = kf; first || k < k1; k += U * G) {
        int j[U];
        bool on[U];
        T ar[U][B];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = k + u * G;
            on[u] = q < k1;
            j[u] = on[u] ? __ldg(a.ci + q) : 0;
            if (!XIN) on[u] = on[u] && __ldg(a.lowk + q) != 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (on[u]) load_row<T, B>(vb + (size_t)(k + u * G - k0) * VS, ar[u]);
        if (first) {
            first = false;
            pdl_wait();
            pdl_trigger();
        }
        constexpr int XB = XIN ? B : FB;
        T xv[U][XB];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (on[u]) {
                if constexpr (XIN) load_cg<T, B>(x_in + (size_t)j[u] * B, xv[u]);
                else load_cg<T, FB>(xt + (size_t)j[u] * FB, xv[u]);
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (on[u]) {
#pragma unroll
                for (int c = 0; c < XB; ++c) {
                    T av = ar[u][c];
                    if constexpr (!XIN) {
#pragma unroll
                        for (int ff = 1; ff < B / FB; ++ff) av = (ff == a.field) ? ar[u][ff * FB + c] : av;
                    }
                    acc = fma(av, xv[u][c], acc);
                }
            }
    }
    return acc;
}

}  // namespace bamg
