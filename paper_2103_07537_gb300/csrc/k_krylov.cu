// FP64 kernels of the outer flexible GMRES: Arnoldi orthogonalisation by
// classical Gram-Schmidt applied twice (CGS2), Givens rotations of the
// Hessenberg column, the triangular solve for y and the update x += Z y.
// (The paper applies its V-cycle inside GMRES: Sec. 3 and Sec. 5.1.)
//
// Reductions are deterministic: every vector is cut into the same fixed
// chunks (one CTA each), every chunk reduces in a fixed tree, and the sums
// of the chunk partials are formed in chunk order by the last CTA to finish
// (it takes a ticket with an atomic after a memory fence; no CTA waits for
// another).  The Givens update of the Hessenberg column runs in that same
// last CTA of the final reduction of an Arnoldi step.
#include <math.h>

#include "common.cuh"

namespace bamg {

constexpr int kKThreads = 256;
constexpr int kDotGroup = 16;  // dot products accumulated together per pass
// ||w1||^2 / ||w||^2 below which an Arnoldi step projects a second time
// (eta = 0.01: the first projection removed more than 99.99% of ||w||^2)
constexpr double kReorthRatio = 1e-4;

// fixed chunking of a vector of length N: at least 256 elements per chunk, at
// most two CTAs per SM of the GB300 (152 SMs).  The basis vectors are mostly
// L2-resident and the rate is set by the loads in flight across the GPU:
// measured on the solves here, 2048-element chunks (fewer CTAs) and four CTAs
// per SM (more block sums and partials) were both slower.
int krylov_chunks(long N) {
    long c = (N + 255) / 256;
    if (c > 2 * 152) c = 2 * 152;
    return (int)(c < 1 ? 1 : c);
}

__device__ __forceinline__ void chunk_range(long N, long* e0, long* e1) {
    const long per = (N + gridDim.x - 1) / gridDim.x;
    *e0 = (long)blockIdx.x * per;
    *e1 = min(N, *e0 + per);
}

// Dots of x with G vectors over the chunk (G fixed at compile time, so every
// issued FMA is a useful one: the FP64 pipe, 2 FMA per clock per SM on
// GB300, bounds these passes): vector g is Y_{v0+g}, or x itself for the last
// one when xx is set.  The block sums go to partial[(v0 + g) * nchunk + chunk].
template <int G>
__device__ __forceinline__ void chunk_dots_fixed(long e0, long e1, const double* __restrict__ x,
                                                 const double* __restrict__ Y, long ld, int v0, bool xx,
                                                 double* __restrict__ partial, double* sh) {
    const double* yp[G];
#pragma unroll
    for (int g = 0; g < G; ++g) yp[g] = (xx && g == G - 1) ? x : Y + (size_t)(v0 + g) * ld;
    double acc[G];
#pragma unroll
    for (int g = 0; g < G; ++g) acc[g] = 0.0;
    for (long e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        const double xe = x[e];
        double yv[G];
#pragma unroll
        for (int g = 0; g < G; ++g) yv[g] = yp[g][e];
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = fma(xe, yv[g], acc[g]);
    }
    // the block reduction works on a power-of-two width (its slices must tile
    // the CTA): the G sums padded with zeros, of which only G are formed
    constexpr int GP = G <= 1 ? 1 : G <= 2 ? 2 : G <= 4 ? 4 : G <= 8 ? 8 : 16;
    double accp[GP];
#pragma unroll
    for (int g = 0; g < GP; ++g) accp[g] = g < G ? acc[g] : 0.0;
    const double tot = block_sums<GP, kKThreads>(accp, G, sh);
    if ((int)threadIdx.x < G) partial[(size_t)(v0 + threadIdx.x) * gridDim.x + blockIdx.x] = tot;
}

// partial[v * nchunk + chunk] = sum_{e in chunk} x[e] * Y_v[e], v < nv, and
// if want_xx, partial[nv * nchunk + chunk] = sum x[e]^2: groups of kDotGroup
// vectors, then one group of the remaining count
__device__ void chunk_dots(long e0, long e1, const double* __restrict__ x, const double* __restrict__ Y,
                           long ld, int nv, int want_xx, double* __restrict__ partial) {
    // sized for the widest reduction (kDotGroup): narrower ones need less
    __shared__ double sh[(kKThreads + kKThreads / kDotGroup) * (kDotGroup + 1)];
    const int tot = nv + want_xx;
    int v0 = 0;
    for (; v0 + kDotGroup <= tot; v0 += kDotGroup)
        chunk_dots_fixed<kDotGroup>(e0, e1, x, Y, ld, v0, want_xx && v0 + kDotGroup == tot, partial, sh);
    const bool xx = want_xx != 0;
    switch (tot - v0) {
#define REM(R) \
    case R: chunk_dots_fixed<R>(e0, e1, x, Y, ld, v0, xx, partial, sh); break;
        REM(1) REM(2) REM(3) REM(4) REM(5) REM(6) REM(7) REM(8) REM(9) REM(10) REM(11) REM(12) REM(13) REM(14)
        REM(15)
#undef REM
        default: break;
    }
}

// True in every thread of the CTA that finishes last; that CTA has seen the
// partials of every other CTA.  Resets the ticket for the next launch.
__device__ __forceinline__ bool last_cta(unsigned* ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
        if (last) *ticket = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// out[v] = sum of the chunk partials partial[v * nchunk + c], a warp for four v
// at a time (their loads together); lane l sums chunks l, l+32, ... in four
// interleaved accumulators, a fixed order for a fixed chunk count
__device__ __forceinline__ void finish_sums(int nv, const double* partial, double* out) {
    constexpr int VU = 4;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int nchunk = gridDim.x;
    for (int v0 = threadIdx.x >> 5; v0 < nv; v0 += nw * VU) {
        double s[VU][4];
#pragma unroll
        for (int u = 0; u < VU; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[u][q] = 0.0;
        for (int c = lane; c < nchunk; c += 128)
#pragma unroll
            for (int u = 0; u < VU; ++u) {
                const int v = v0 + u * nw;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (v < nv && c + 32 * q < nchunk) s[u][q] += __ldcg(partial + (size_t)v * nchunk + c + 32 * q);
            }
#pragma unroll
        for (int u = 0; u < VU; ++u) {
            const int v = v0 + u * nw;
            if (v >= nv) break;  // (uniform)
            const double t = warp_sum((s[u][0] + s[u][1]) + (s[u][2] + s[u][3]));
            if (lane == 0) out[v] = t;
        }
    }
}

// Arnoldi bookkeeping by the whole CTA: column j of the Hessenberg matrix from
// h1 (+ h2) and ||w||, breakdown test, previous rotations, the new rotation, the
// residual estimate |g_{j+1}|.  scal = {h_{j+1,j}, |g_{j+1}|, breakdown, ||w||
// before orthogonalising}.  The column and the rotations are loaded and stored
// by all threads; one thread applies them in shared memory (a chain of two FP64
// operations per rotation instead of round trips through L2).
__device__ void givens_update(const GivensArgs& a, double wsq, bool with_h2) {
    __shared__ double col[kMaxRestart + 2], cs[kMaxRestart], sn[kMaxRestart];
    const int j = a.j, m = a.m, t = threadIdx.x;
    double* H = a.H;
    const double wn0 = sqrt(__ldcg(a.h1 + j + 1));  // ||w|| before orthogonalising
    if (t <= j) col[t] = __ldcg(a.h1 + t) + (with_h2 ? __ldcg(a.h2 + t) : 0.0);
    if (t < j) {
        cs[t] = __ldcg(a.cs + t);
        sn[t] = __ldcg(a.sn + t);
    }
    __syncthreads();
    if (t == 0) {
        const double hn = sqrt(wsq);
        const int breakdown = !(hn > 1e-14 * wn0);
        double x0 = col[0];
        for (int i = 0; i < j; ++i) {
            const double x1 = col[i + 1];
            col[i] = cs[i] * x0 + sn[i] * x1;
            x0 = -sn[i] * x0 + cs[i] * x1;
        }
        const double d = sqrt(x0 * x0 + hn * hn);
        const double c = d == 0.0 ? 1.0 : x0 / d, sj = d == 0.0 ? 0.0 : hn / d;
        a.cs[j] = c;
        a.sn[j] = sj;
        col[j] = d;
        const double gj = a.g[j];
        a.g[j + 1] = -sj * gj;
        a.g[j] = c * gj;
        a.scal[0] = hn;
        a.scal[1] = fabs(sj * gj);
        a.scal[2] = breakdown ? 1.0 : 0.0;
        a.scal[3] = wn0;
        // the step's outcome for the host, which waits for this kernel only
        a.host[0] = fabs(sj * gj);
        a.host[1] = breakdown ? 1.0 : 0.0;
        a.host[2] = 0.0;
        a.host[3] = (double)__ldcg(a.err);
        __threadfence_system();
    }
    __syncthreads();
    if (t <= j) H[(size_t)t * m + j] = col[t];
    if (t == j + 1) H[(size_t)t * m + j] = 0.0;
}

__global__ void __launch_bounds__(kKThreads) multi_dot_kernel(long N, const double* __restrict__ x,
                                                              const double* __restrict__ Y, long ld, int nv,
                                                              int want_xx, double* __restrict__ partial,
                                                              double* __restrict__ out, unsigned* ticket,
                                                              const unsigned* cond) {
    if (cond && __ldcg(cond) == 0u) return;  // a conditional pass that is not needed (every CTA)
    long e0, e1;
    chunk_range(N, &e0, &e1);
    chunk_dots(e0, e1, x, Y, ld, nv, want_xx, partial);
    if (last_cta(ticket)) finish_sums(nv + want_xx, partial, out);
}

// t[u] -= sum over G vectors v0 .. of h[v] Y_v[e + u * blockDim.x], u < E: the
// G * E loads are issued before the FMA chains
template <int G, int E>
__device__ __forceinline__ void axpy_group(double (&t)[E], const double* __restrict__ Y, long ld, long e, int v0,
                                           const double* sh_h) {
    double yv[G][E];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int u = 0; u < E; ++u) yv[g][u] = Y[(size_t)(v0 + g) * ld + e + u * (long)blockDim.x];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int u = 0; u < E; ++u) t[u] = fma(-sh_h[v0 + g], yv[g][u], t[u]);
}
// x[e + u * blockDim.x] -= sum_v h[v] Y_v there, u < E: groups of 8 vectors, the
// remainder as one group of its exact size (a vector at a time waits for each
// load).  Averages over 50 steps on 1.1 M unknowns, 25 vectors a pass: 99 us,
// this way 87 us; the FP64 pipe's floor is 49 us, HBM's 34 us
template <int E>
__device__ __forceinline__ void axpy_items(double* __restrict__ x, const double* __restrict__ Y, long ld, long e, int nv,
                                           const double* sh_h) {
    double t[E];
#pragma unroll
    for (int u = 0; u < E; ++u) t[u] = x[e + u * (long)blockDim.x];
    int v = 0;
    for (; v + 8 <= nv; v += 8) axpy_group<8, E>(t, Y, ld, e, v, sh_h);
    switch (nv - v) {
#define REM(R) \
    case R: axpy_group<R, E>(t, Y, ld, e, v, sh_h); break;
        REM(1) REM(2) REM(3) REM(4) REM(5) REM(6) REM(7)
#undef REM
        default: break;
    }
#pragma unroll
    for (int u = 0; u < E; ++u) x[e + u * (long)blockDim.x] = t[u];
}

// x -= sign * sum_v h[v] Y_v over the chunk, then (mode 1) the dots of the new
// x with Y_0..Y_{nv-1} into out, (mode 2) its squared norm into out (and the
// Givens update when do_givens), (mode 3) as 2, with the reorthogonalisation
// test of the Arnoldi step in the last CTA, (mode 0) nothing.  cond: the pass
// runs only where *cond is nonzero.
__global__ void __launch_bounds__(kKThreads) axpy_dot_kernel(long N, double* __restrict__ x,
                                                             const double* __restrict__ Y, long ld, int nv,
                                                             const double* __restrict__ h, double sign, int mode,
                                                             double* __restrict__ partial, double* __restrict__ out,
                                                             unsigned* ticket, GivensArgs ga, int do_givens,
                                                             const unsigned* cond) {
    if (cond && __ldcg(cond) == 0u) return;
    __shared__ double sh_h[kMaxRestart + 1];
    for (int v = threadIdx.x; v < nv; v += blockDim.x) sh_h[v] = sign * h[v];
    __syncthreads();
    long e0, e1;
    chunk_range(N, &e0, &e1);
    // two elements per thread at a time, one where the chunk ends
    for (long e = e0 + threadIdx.x; e < e1; e += 2 * (long)blockDim.x) {
        if (e + (long)blockDim.x < e1) axpy_items<2>(x, Y, ld, e, nv, sh_h);
        else axpy_items<1>(x, Y, ld, e, nv, sh_h);
    }
    if (mode == 0) return;
    __syncthreads();
    if (mode == 1) chunk_dots(e0, e1, x, Y, ld, nv, 0, partial);
    else chunk_dots(e0, e1, x, Y, ld, 0, 1, partial);
    if (last_cta(ticket)) {
        finish_sums(mode == 1 ? nv : 1, partial, out);
        __syncthreads();
        if (mode == 3) {
            // one projection is enough unless it removed nearly all of w
            // (||w1|| < eta ||w||, eta = 0.01); otherwise the step projects
            // again and its Givens update waits for that
            const double w1 = __ldcg(out), w0 = __ldcg(ga.h1 + ga.j + 1);
            const unsigned need = !(w1 >= kReorthRatio * w0);
            if (threadIdx.x == 0) {
                *ga.reorth = need;
                ga.host[4] = need ? 1.0 : 0.0;
            }
            if (!need) givens_update(ga, w1, false);
            else if (threadIdx.x == 0) {
                ga.host[2] = 1.0;
                ga.host[3] = (double)__ldcg(ga.err);
                __threadfence_system();
            }
        } else if (do_givens) {
            givens_update(ga, __ldcg(out), true);
        }
    }
}

int launch_multi_dot(long N, const double* x, const double* Y, long ld, int nv, int want_xx, double* partial,
                     double* out, unsigned* ticket, cudaStream_t s, const unsigned* cond) {
    multi_dot_kernel<<<krylov_chunks(N), kKThreads, 0, s>>>(N, x, Y, ld, nv, want_xx, partial, out, ticket, cond);
    return launched(1);
}
int launch_axpy_dot(long N, double* x, const double* Y, long ld, int nv, const double* h, double sign, int mode,
                    double* partial, double* out, unsigned* ticket, const GivensArgs* ga, cudaStream_t s,
                    const unsigned* cond) {
    GivensArgs g{};
    if (ga) g = *ga;
    axpy_dot_kernel<<<krylov_chunks(N), kKThreads, 0, s>>>(N, x, Y, ld, nv, h, sign, mode, partial, out, ticket, g,
                                                           ga ? 1 : 0, cond);
    return launched(1);
}

// y = H(0:k, 0:k)^{-1} g(0:k), upper triangular (k <= 64): one warp, a row's
// products spread over the lanes
__global__ void solve_upper_kernel(int k, int m, const double* __restrict__ H, const double* __restrict__ g,
                                   double* __restrict__ y) {
    __shared__ double ys[kMaxRestart];
    const int lane = threadIdx.x;
    if (lane >= 32 || blockIdx.x != 0) return;
    for (int i = k - 1; i >= 0; --i) {
        double s = 0.0;
        for (int c = i + 1 + lane; c < k; c += 32) s += H[(size_t)i * m + c] * ys[c];
        s = warp_sum(s);
        if (lane == 0) {
            ys[i] = (g[i] - s) / H[(size_t)i * m + i];
            y[i] = ys[i];
        }
        __syncwarp();
    }
}

// y = x / scal[0] unless the breakdown flag scal[2] is set; y32 (optional): the
// same rounded to FP32, the input of an FP32 cycle (its cast pass saved)
__global__ void scale_kernel(long N, const double* __restrict__ x, const double* __restrict__ scal,
                             double* __restrict__ y, float* __restrict__ y32, int check_breakdown) {
    if (check_breakdown && scal[2] != 0.0) return;
    // one division per thread and a product per element: an FP64 division
    // per element costs about ten FP64 operations, and GB300 issues two per
    // clock per SM (within an ulp of the quotient)
    const double rden = 1.0 / scal[0];
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < N; e += (long)gridDim.x * blockDim.x) {
        const double v = x[e] * rden;
        y[e] = v;
        if (y32) y32[e] = (float)v;
    }
}

// g = (beta, 0, ..., 0) with beta = sqrt(*bsq); scal[0] = beta
__global__ void init_g_kernel(int m, const double* __restrict__ bsq, double* __restrict__ g,
                              double* __restrict__ scal) {
    const int t = threadIdx.x;
    const double beta = sqrt(bsq[0]);
    for (int i = t; i <= m; i += blockDim.x) g[i] = (i == 0) ? beta : 0.0;
    if (t == 0) scal[0] = beta;
}

int launch_solve_upper(int k, int m, const double* H, const double* g, double* y, cudaStream_t s) {
    solve_upper_kernel<<<1, 32, 0, s>>>(k, m, H, g, y);
    return launched(1);
}
int launch_scale(long N, const double* x, const double* scal, double* y, float* y32, int check_breakdown,
                 cudaStream_t s) {
    long g = (N + 255) / 256;
    scale_kernel<<<(int)(g < 1216 ? (g > 0 ? g : 1) : 1216), 256, 0, s>>>(N, x, scal, y, y32, check_breakdown);
    return launched(1);
}
int launch_init_g(int m, const double* bsq, double* g, double* scal, cudaStream_t s) {
    init_g_kernel<<<1, 64, 0, s>>>(m, bsq, g, scal);
    return launched(1);
}

}  // namespace bamg
