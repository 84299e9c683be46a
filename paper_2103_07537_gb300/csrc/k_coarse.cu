// The V-cycle of the coarse levels (Fig. 1 of the paper from a given level
// down) in one launch of one thread-block cluster, the matrices and vectors of
// every level in the distributed shared memory of its CTAs.
//
// A small level's colour step is bound by latency: as a kernel of its own it
// costs 2.1 to 2.5 us (launch, dependent loads through L2, drain), nearly all
// of it independent of the level's size, and a cycle has 2 (n_pre + n_post)
// steps per field and level.  Here a step is one cluster barrier, a gather
// from distributed shared memory and the products: CTA c owns the nodes
// c per .. (c + 1) per - 1 of every level with their rows and vectors (copied in
// by cp.async ahead of the wait on the previous kernel) and reads its
// neighbours' values from the CTAs that own them.  Column indices, aggregates
// and member lists are kept as (owner << 16 | local index).
//
// Lanes: a node takes FB x G lanes of one warp (B x G in the residual), G
// lanes per scalar row, each taking every G-th block; the row sums meet by
// shuffles.  G = 2 in FP64, where a warp's FP64 instruction occupies its
// scheduler's pipe for 64 cycles and fuller lanes mean fewer of them, 4 in
// FP32.  The arithmetic of a step is that of the per-colour kernels (see
// bgs_block) up to the order of the row sums.
#include <cooperative_groups.h>

#include "bgs_body.cuh"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace bamg {

namespace {

constexpr int kCcThreads = 256;

template <typename T>
struct CcLanes {
    static constexpr int kG = sizeof(T) == 8 ? 2 : 4;
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Everything below addresses shared memory by byte offsets into the dynamic
// array (loads of the shared window, no generic addressing), and a peer's by the
// 32-bit cluster address of the same offset.
extern __shared__ __align__(16) unsigned char cc_sh[];

template <typename V>
__device__ __forceinline__ V* at(int off) {
    return reinterpret_cast<V*>(cc_sh + off);
}
__device__ __forceinline__ uint32_t cluster_addr(int off, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(a)
                 : "r"((uint32_t)__cvta_generic_to_shared(cc_sh) + (uint32_t)off), "r"(rank));
    return a;
}
__device__ __forceinline__ void ld_cluster(uint32_t a, float& v) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
__device__ __forceinline__ void ld_cluster(uint32_t a, double& v) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
// W values of the entry enc (owner << 16 | local) of a buffer of W per node
template <int W, typename T>
__device__ __forceinline__ void peer_row(int off, int enc, T (&v)[W]) {
    const uint32_t a = cluster_addr(off, enc >> 16) + (uint32_t)((enc & 0xffff) * W * (int)sizeof(T));
    constexpr int bytes = W * (int)sizeof(T);
    if constexpr (sizeof(T) == 4 && bytes % 16 == 0) {
#pragma unroll
        for (int c = 0; c < W; c += 4)
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v[c]), "=f"(v[c + 1]), "=f"(v[c + 2]), "=f"(v[c + 3])
                         : "r"(a + 4 * c));
    } else if constexpr (sizeof(T) == 4 && bytes % 8 == 0) {
#pragma unroll
        for (int c = 0; c < W; c += 2)
            asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v[c]), "=f"(v[c + 1]) : "r"(a + 4 * c));
    } else if constexpr (sizeof(T) == 8 && bytes % 16 == 0) {
#pragma unroll
        for (int c = 0; c < W; c += 2)
            asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[c]), "=d"(v[c + 1]) : "r"(a + 8 * c));
    } else {
#pragma unroll
        for (int c = 0; c < W; ++c) ld_cluster(a + (uint32_t)(c * (int)sizeof(T)), v[c]);
    }
}
// entry d of such a row
template <int W, typename T>
__device__ __forceinline__ T peer_entry(int off, int enc, int d) {
    T v;
    ld_cluster(cluster_addr(off, enc >> 16) + (uint32_t)(((enc & 0xffff) * W + d) * (int)sizeof(T)), v);
    return v;
}

// a level as one CTA sees it: its own nodes and the offsets of its slices
struct CcView {
    int nl, k0;  // own nodes, first stored block of the own rows
    int rp, vals, enc, lowk, dinv, omega, list, list_off, agg;  // omega: -1 for the scalar
    int x0, x1, rhs, xt;
};

// one colour of one field step on the CTA's own nodes (see bgs_tpr_kernel), from
// the iterate at xin (XIN; updated in place) or from zero, to xout; gout: the own
// slice of the result in global memory, or null
template <typename T, int B, int FB, bool XIN>
__device__ __forceinline__ void cc_colour(const CcView& L, int colour, int field, int xin, int xout, T* gout, T omega) {
    constexpr int G = CcLanes<T>::kG, LN = FB * G, NPW = 32 / LN, F = B / FB;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int q0 = at<int>(L.list_off)[colour], q1 = at<int>(L.list_off)[colour + 1];
    const int node = lane / LN, r = (lane - node * LN) / G, sl = lane % G;
    const int f0 = field * FB;
    for (int q = q0 + w * NPW; q < q1; q += (kCcThreads / 32) * NPW) {
        const bool act = node < NPW && q + node < q1;
        int i = 0;
        T acc = T(0);
        if (act) {
            i = at<int>(L.list)[q + node];
            const int ka = at<int>(L.rp)[i] - L.k0 + sl, k1 = at<int>(L.rp)[i + 1] - L.k0;
            constexpr int U = 3;  // blocks of a lane whose loads are issued together
            for (int k = ka; k < k1; k += U * G) {
                int enc[U];
                bool on[U];
                constexpr int XB = XIN ? B : FB;
                T ar[U][B], xv[U][XB];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    on[u] = k + u * G < k1;
                    const int kk = on[u] ? k + u * G : ka;
                    enc[u] = at<int>(L.enc)[kk];
                    if (!XIN) on[u] = on[u] && at<unsigned char>(L.lowk)[kk] != 0;
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (on[u]) {
                        peer_row<XB>(XIN ? xin : L.xt, enc[u], xv[u]);
                        load_row<T, B>(at<T>(L.vals) + (k + u * G) * B * B + (f0 + r) * B, ar[u]);
                    }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (on[u]) {
#pragma unroll
                        for (int c = 0; c < XB; ++c) {
                            T av = ar[u][c];
                            if constexpr (!XIN) {
#pragma unroll
                                for (int ff = 1; ff < F; ++ff) av = (ff == field) ? ar[u][ff * FB + c] : av;
                            }
                            acc = fma(av, xv[u][c], acc);
                        }
                    }
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const T t = act ? at<T>(L.rhs)[i * B + f0 + r] - acc : T(0);
        const T* D = at<T>(L.dinv) + (i * F + field) * FB * FB + (act ? r : 0) * FB;
        T xn = T(0);
#pragma unroll
        for (int c = 0; c < FB; ++c) xn = fma(D[c], __shfl_sync(0xffffffffu, t, node * LN + c * G), xn);
        if (act) {
            if (!XIN && sl == 0) at<T>(L.xt)[i * FB + r] = xn;
            // lane sl of row r takes the fields sl, sl + G, ... of the node's entries
            for (int m = sl; m < F; m += G) {
                const int e = i * B + m * FB + r;
                T v = XIN ? at<T>(xin)[e] : T(0);
                if (m == field) {
                    if (XIN) at<T>(xin)[e] = v + xn;
                    v = fma(L.omega >= 0 ? at<T>(L.omega)[i * F + field] : omega, xn, v);
                }
                at<T>(xout)[e] = v;
                if (gout) gout[e] = v;
            }
        }
    }
}

// res = rhs - A x on the CTA's own nodes
template <typename T, int B>
__device__ __forceinline__ void cc_residual(const CcView& L, int x, int res) {
    constexpr int G = CcLanes<T>::kG, LN = B * G, NPW = 32 / LN;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int node = lane / LN, r = (lane - node * LN) / G, sl = lane % G;
    for (int ib = w * NPW; ib < L.nl; ib += (kCcThreads / 32) * NPW) {
        const int i = ib + node;
        const bool act = node < NPW && i < L.nl;
        T acc = T(0);
        if (act) {
            const int k1 = at<int>(L.rp)[i + 1] - L.k0;
#pragma unroll 2
            for (int k = at<int>(L.rp)[i] - L.k0 + sl; k < k1; k += G) {
                T ar[B], xv[B];
                peer_row<B>(x, at<int>(L.enc)[k], xv);
                load_row<T, B>(at<T>(L.vals) + k * B * B + r * B, ar);
#pragma unroll
                for (int c = 0; c < B; ++c) acc = fma(ar[c], xv[c], acc);
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (act && sl == 0) at<T>(res)[i * B + r] = at<T>(L.rhs)[i * B + r] - acc;
    }
}

// own rows of y = Ainv x, x (spread over the CTAs at rhs) gathered at all; a warp per row
template <typename T, typename S, int B>
__device__ __forceinline__ void cc_coarsest(int rank, int n, int per, const S* __restrict__ ainv, int rhs, int all,
                                            int y) {
    const int nd = n * B, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < nd; e += kCcThreads) {
        const int i = e / B, own = i / per;
        at<T>(all)[e] = peer_entry<B, T>(rhs, (own << 16) | (i - own * per), e - i * B);
    }
    __syncthreads();
    const int r0 = rank * per * B, r1 = min(nd, r0 + per * B);
    for (int row = r0 + w; row < r1; row += kCcThreads / 32) {
        const S* a = ainv + (size_t)row * nd;
        constexpr int U = 8;  // columns of a lane loaded together
        S acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = S(0);
        for (int c = lane; c < nd; c += U * 32) {
            S av[U];
#pragma unroll
            for (int u = 0; u < U; ++u) av[u] = c + u * 32 < nd ? __ldg(a + c + u * 32) : S(0);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (c + u * 32 < nd) acc[u] = fma(av[u], (S)at<T>(all)[c + u * 32], acc[u]);
        }
        const S sum = warp_sum(((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7])));
        if (lane == 0) at<T>(y)[row - r0] = (T)sum;
    }
}

// count values at src of global memory into shared memory at off (a multiple of
// 16; 32 bytes of room beyond), in whole 16-byte units of the source (every
// buffer of the hierarchy has 64 bytes of room at its end); returns src's offset
template <typename V>
__device__ __forceinline__ int cc_copy(int off, const V* src, int count) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src), a16 = a & ~(uintptr_t)15;
    const int units = (int)((a + (size_t)count * sizeof(V) - a16 + 15) >> 4);
    const unsigned dst = (unsigned)__cvta_generic_to_shared(cc_sh) + (unsigned)off;
    for (int e = threadIdx.x; e < units; e += kCcThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * (unsigned)e), "l"(a16 + 16u * (size_t)e)
                     : "memory");
    return off + (int)(a - a16);
}

template <typename T, int B, int FB>
__global__ void __launch_bounds__(kCcThreads, 1) coarse_cycle_kernel(const __grid_constant__ CcArgs a, const T* rhs,
                                                                     T* out) {
    __shared__ CcView view[kCcLevels];
    constexpr int F = B / FB;
    const int rank = (int)cg::this_cluster().block_rank();
    const int last = a.nlev - 1;
#pragma unroll 1
    for (int l = 0; l <= last; ++l) {
        const CcLevel& L = a.lev[l];
        const int i0 = min(L.n, rank * L.per), nl = min(L.n, i0 + L.per) - i0;
        CcView v{};
        v.nl = nl;
        v.x0 = L.off[kCcX0];
        v.x1 = L.off[kCcX1];
        v.rhs = L.off[kCcRhs];
        v.xt = L.off[kCcXt];
        if (l < last) {
            const int k0 = L.bound[rank], nk = L.bound[rank + 1] - k0;
            v.k0 = k0;
            v.rp = cc_copy(L.off[kCcRp], L.rp + i0, nl + 1);
            v.vals = cc_copy(L.off[kCcVals], static_cast<const T*>(L.vals) + (size_t)k0 * B * B, nk * B * B);
            v.enc = cc_copy(L.off[kCcEnc], L.enc + k0, nk);
            v.lowk = cc_copy(L.off[kCcLow], L.lowk + k0, nk);
            v.dinv = cc_copy(L.off[kCcDinv], static_cast<const T*>(L.dinv) + (size_t)i0 * F * FB * FB, nl * F * FB * FB);
            v.omega = L.omega ? cc_copy(L.off[kCcOmega], static_cast<const T*>(L.omega) + (size_t)i0 * F, nl * F) : -1;
            v.list = cc_copy(L.off[kCcList], L.list + i0, nl);
            v.list_off = cc_copy(L.off[kCcListOff], L.list_off + rank * (L.colours + 1), L.colours + 1);
            v.agg = cc_copy(L.off[kCcAgg], L.agg + i0, nl);
        }
        if (threadIdx.x == 0) view[l] = v;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    pdl_wait();
    pdl_trigger();
    const int g0 = min(a.lev[0].n, rank * a.lev[0].per);
    {
        const int nl = min(a.lev[0].n, g0 + a.lev[0].per) - g0;
        T* r = at<T>(a.lev[0].off[kCcRhs]);
        for (int e = threadIdx.x; e < nl * B; e += kCcThreads) r[e] = ld_cg(rhs + (size_t)g0 * B + e);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    cluster_sync();  // every CTA has started and holds its slices, views and right-hand side
    const T omega = (T)a.omega;
    unsigned cur = 0u;  // bit l: which iterate of level l is current
#pragma unroll 1
    for (int l = 0; l < last; ++l) {
        const CcView V = view[l];
        const int colours = a.lev[l].colours;
        int c = -1;  // the zero iterate
        for (int t = 0; t < a.n_pre * F; ++t) {
            const int d = c == 0 ? 1 : 0;
            for (int q = 0; q < colours; ++q) {
                if (c < 0) cc_colour<T, B, FB, false>(V, q, t % F, 0, V.x0, nullptr, omega);
                else cc_colour<T, B, FB, true>(V, q, t % F, c ? V.x1 : V.x0, d ? V.x1 : V.x0, nullptr, omega);
                cluster_sync();
            }
            c = d;
        }
        if (c < 0) {
            for (int e = threadIdx.x; e < V.nl * B; e += kCcThreads) at<T>(V.x0)[e] = T(0);
            c = 0;
            cluster_sync();
        }
        cur |= (unsigned)c << l;
        const int res = c ? V.x0 : V.x1;
        cc_residual<T, B>(V, c ? V.x1 : V.x0, res);
        cluster_sync();
        // restriction: own coarse nodes, members ascending
        const int nl = view[l + 1].nl, rc = view[l + 1].rhs;
        const int* ap = a.lev[l].agg_ptr + min(a.lev[l + 1].n, rank * a.lev[l + 1].per);
        for (int e = threadIdx.x; e < nl * B; e += kCcThreads) {
            const int I = e / B, dd = e - I * B;
            const int p1 = __ldg(ap + I + 1);
            T s = T(0);
#pragma unroll 4
            for (int p = __ldg(ap + I); p < p1; ++p) s += peer_entry<B, T>(res, __ldg(a.lev[l].members + p), dd);
            at<T>(rc)[e] = s;
        }
        cluster_sync();
    }
    {
        const CcView V = view[last];
        if (a.inv32) cc_coarsest<T, float, B>(rank, a.lev[last].n, a.lev[last].per, a.inv32, V.rhs, V.xt, V.x0);
        else cc_coarsest<T, double, B>(rank, a.lev[last].n, a.lev[last].per, a.inv64, V.rhs, V.xt, V.x0);
        cluster_sync();
    }
#pragma unroll 1
    for (int l = last - 1; l >= 0; --l) {
        const CcView V = view[l];
        const int colours = a.lev[l].colours;
        int c = (int)(cur >> l & 1u);
        // prolongation and correction on the own nodes
        const int uc = cur >> (l + 1) & 1u ? view[l + 1].x1 : view[l + 1].x0;
        T* gout = l == 0 ? out + (size_t)g0 * B : nullptr;
        for (int e = threadIdx.x; e < V.nl * B; e += kCcThreads) {
            const int i = e / B;
            T* x = at<T>(c ? V.x1 : V.x0) + e;
            const T v = *x + peer_entry<B, T>(uc, at<int>(V.agg)[i], e - i * B);
            *x = v;
            if (gout && a.n_post == 0) gout[e] = v;
        }
        cluster_sync();
        for (int t = 0; t < a.n_post * F; ++t) {
            for (int q = 0; q < colours; ++q) {
                cc_colour<T, B, FB, true>(V, q, t % F, c ? V.x1 : V.x0, c ? V.x0 : V.x1,
                                          t == a.n_post * F - 1 ? gout : nullptr, omega);
                cluster_sync();
            }
            c = 1 - c;
        }
        cur = (cur & ~(1u << l)) | ((unsigned)c << l);
    }
}

__device__ __forceinline__ int cc_encode(int i, int per) {
    const int own = i / per;
    return (own << 16) | (i - own * per);
}
__global__ void cc_encode_kernel(long m, int per, const int* __restrict__ idx, int* __restrict__ enc) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < m) enc[e] = cc_encode(idx[e], per);
}
// CTA c's nodes by (colour, index), as local indices at list[c per ..], and their
// offsets per colour list_off[c][colours + 1]: one CTA of threads per cluster CTA
__global__ void __launch_bounds__(256) cc_list_kernel(int n, int per, int colours, const int* __restrict__ colour,
                                                      int* __restrict__ list, int* __restrict__ list_off) {
    const int i0 = min(n, (int)blockIdx.x * per), nl = min(n, i0 + per) - i0;
    __shared__ int sum[256];
    int base = 0;
    for (int c = 0; c < colours; ++c) {
        if (threadIdx.x == 0) list_off[blockIdx.x * (colours + 1) + c] = base;
        for (int b0 = 0; b0 < nl; b0 += 256) {
            const int i = b0 + threadIdx.x;
            const int is = i < nl && colour[i0 + i] == c;
            sum[threadIdx.x] = is;
            __syncthreads();
            for (int o = 1; o < 256; o <<= 1) {
                const int v = threadIdx.x >= o ? sum[threadIdx.x - o] : 0;
                __syncthreads();
                sum[threadIdx.x] += v;
                __syncthreads();
            }
            if (is) list[i0 + base + sum[threadIdx.x] - 1] = i;
            base += sum[255];
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) list_off[blockIdx.x * (colours + 1) + colours] = base;
}
// bound[c] = ptr of the first node of CTA c (c = 0..ctas)
__global__ void cc_bound_kernel(int n, int per, int ctas, const int* __restrict__ ptr, int* __restrict__ bound) {
    const int c = threadIdx.x;
    if (c <= ctas) bound[c] = ptr[min(n, c * per)];
}

template <typename T, int B, int FB>
cudaError_t cc_launch(const CcArgs& a, const T* rhs, T* out, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3((unsigned)a.ctas);
    cfg.blockDim = dim3(kCcThreads);
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = t_pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, coarse_cycle_kernel<T, B, FB>, a, rhs, out);
}

// shared memory and cluster size accepted by the device for this instance
template <typename T, int B, int FB>
bool cc_fits(int ctas, size_t smem) {
    if (cudaFuncSetAttribute(coarse_cycle_kernel<T, B, FB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCcMaxSmem) !=
            cudaSuccess ||
        (ctas > 8 && cudaFuncSetAttribute(coarse_cycle_kernel<T, B, FB>, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                          1) != cudaSuccess)) {
        (void)cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kCcThreads);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, coarse_cycle_kernel<T, B, FB>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return clusters >= 1;
}

}  // namespace

template <typename T>
int launch_coarse_cycle(int b, int fb, const CcArgs& a, const T* rhs, T* out, cudaStream_t s) {
    cudaError_t e = cudaErrorInvalidValue;
    switch (b * 16 + fb) {
#define CASE(BB, FF) \
    case BB * 16 + FF: e = cc_launch<T, BB, FF>(a, rhs, out, s); break;
        BAMG_BLOCK_SHAPES(CASE)
#undef CASE
        default: return BAMG_EUNSUPPORTED;
    }
    return e == cudaSuccess ? launched(1) : BAMG_ECUDA;
}
template int launch_coarse_cycle<double>(int, int, const CcArgs&, const double*, double*, cudaStream_t);
template int launch_coarse_cycle<float>(int, int, const CcArgs&, const float*, float*, cudaStream_t);

bool coarse_cycle_fits(int b, int fb, bool fp64, int ctas, size_t smem) {
    if (smem > (size_t)kCcMaxSmem) return false;
    switch (b * 16 + fb) {
#define CASE(BB, FF) \
    case BB * 16 + FF: return fp64 ? cc_fits<double, BB, FF>(ctas, smem) : cc_fits<float, BB, FF>(ctas, smem);
        BAMG_BLOCK_SHAPES(CASE)
#undef CASE
        default: return false;
    }
}

int launch_cc_encode(long m, int per, const int* idx, int* enc, cudaStream_t s) {
    if (m <= 0) return BAMG_OK;
    cc_encode_kernel<<<ceil_div(m, 256), 256, 0, s>>>(m, per, idx, enc);
    return launched(1);
}
int launch_cc_list(int n, int per, int ctas, int colours, const int* colour, int* list, int* list_off,
                   cudaStream_t s) {
    cc_list_kernel<<<ctas, 256, 0, s>>>(n, per, colours, colour, list, list_off);
    return launched(1);
}
int launch_cc_bound(int n, int per, int ctas, const int* ptr, int* bound, cudaStream_t s) {
    cc_bound_kernel<<<1, 32, 0, s>>>(n, per, ctas, ptr, bound);
    return launched(1);
}

}  // namespace bamg
