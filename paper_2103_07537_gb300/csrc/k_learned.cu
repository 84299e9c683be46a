// Learned damping weights (beyond the paper: the paper fixes one damping of
// its block Gauss-Seidel smoother near 0.5 and shows that the value decides
// convergence for small viscosity, Sec. 5).  A network 8 -> 64 -> 64 -> 2
// (tanh) maps features of a level's matrix to the smoother damping of every
// node and field (head 0) and to the prolongator smoothing weight of every
// aggregate and field (head 1).
//   features       features_kernel, agg_features_kernel (FP64 math, FP32 out)
//   inference      mlp_forward_kernel: FP16 parameters, FP32 arithmetic
//   training       mlp_grad_kernel (+ deterministic reduction), adam_kernel
// The network is small (4882 parameters): the kernels stage the parameters
// in shared memory as FP32 and use plain FMA; rows are independent.
#include <cuda_fp16.h>

#include "common.cuh"

namespace bamg {

constexpr int kNF = BAMG_NFEAT, kNH = BAMG_MLP_H, kNO = BAMG_MLP_OUT;
constexpr int kOW1 = 0, kOB1 = kOW1 + kNH * kNF, kOW2 = kOB1 + kNH, kOB2 = kOW2 + kNH * kNH, kOW3 = kOB2 + kNH,
              kOB3 = kOW3 + kNO * kNH, kOXM = kOB3 + kNO, kOXS = kOXM + kNF;
static_assert(kOXS + kNF == BAMG_MLP_NPARAMS, "parameter layout");
static_assert(kOXM == BAMG_MLP_NTRAIN, "parameter layout");

// ---------------------------------------------------------------------------
// features of node i, field f (see amg_features in bamg.h); thread per node
// ---------------------------------------------------------------------------
template <int B, int FB>
__global__ void features_kernel(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                const double* __restrict__ vals, const int* __restrict__ agg,
                                const int* __restrict__ agg_cnt, int level, float* __restrict__ out, int* err) {
    constexpr int F = B / FB;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double d[F], o[F], c[F], tr[F];
#pragma unroll
    for (int f = 0; f < F; ++f) d[f] = o[f] = c[f] = tr[f] = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        const double* blk = vals + (size_t)k * B * B;
        const int j = ci[k];
#pragma unroll
        for (int f = 0; f < F; ++f) {
#pragma unroll
            for (int g = 0; g < F; ++g) {
                double s = 0.0;
                for (int r = 0; r < FB; ++r)
                    for (int cc = 0; cc < FB; ++cc) {
                        const double v = blk[(f * FB + r) * B + g * FB + cc];
                        s += v * v;
                    }
                const double nrm = sqrt(s);
                if (g != f) c[f] += nrm;
                else if (j == i) d[f] = nrm;
                else o[f] += nrm;
            }
            if (j == i)
                for (int r = 0; r < FB; ++r) tr[f] += blk[(f * FB + r) * B + f * FB + r];
        }
    }
    double mean_log = 0.0;
#pragma unroll
    for (int f = 0; f < F; ++f) {
        if (!(d[f] > 0.0)) {
            set_error(err, kDevSingularBlock);
            return;
        }
        mean_log += log(d[f]);
    }
    mean_log /= F;
    const int a = agg[i];
    const double lsz = log((double)agg_cnt[a]);
#pragma unroll
    for (int f = 0; f < F; ++f) {
        float* x = out + ((size_t)i * F + f) * kNF;
        const double ld = log(d[f]);
        x[0] = (float)ld;
        x[1] = (float)(o[f] / d[f]);
        x[2] = (float)(c[f] / (d[f] + o[f]));
        x[3] = (float)(ld - mean_log);
        x[4] = (float)(tr[f] / (sqrt((double)FB) * d[f]));
        x[5] = (float)lsz;
        x[6] = (float)level;
        x[7] = (float)f;
    }
}

__global__ void agg_count_kernel(int n, int nc, const int* __restrict__ agg, int* __restrict__ cnt, int* err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int a = agg[i];
    if (a < 0 || a >= nc) {
        set_error(err, kDevBadPattern);
        return;
    }
    atomicAdd(cnt + a, 1);
}

// aggregate features: the mean of the member rows; thread per (I, f, m),
// members visited in ascending node order through the sorted member lists
__global__ void agg_features_kernel(int nc, int F, const int* __restrict__ agg_ptr, const int* __restrict__ members,
                                    const float* __restrict__ node_feat, float* __restrict__ out) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long)nc * F * kNF) return;
    const int I = (int)(e / (F * kNF));
    const int w = (int)(e % (F * kNF));
    double s = 0.0;
    const int q0 = agg_ptr[I], q1 = agg_ptr[I + 1];
    for (int q = q0; q < q1; ++q) s += (double)node_feat[(size_t)members[q] * F * kNF + w];
    out[e] = (float)(s / (double)(q1 - q0));
}

int launch_features(int b, int fb, int n, const int* rp, const int* ci, const double* vals, const int* agg,
                    const int* agg_cnt, int level, float* out, int* err, cudaStream_t s) {
    if (n <= 0) return BAMG_OK;
    const int grid = ceil_div(n, 128);
    switch (b * 16 + fb) {
#define CASE(BB, FF)                                                                                     \
    case BB * 16 + FF:                                                                                   \
        features_kernel<BB, FF><<<grid, 128, 0, s>>>(n, rp, ci, vals, agg, agg_cnt, level, out, err);    \
        break;
        BAMG_BLOCK_SHAPES(CASE)
#undef CASE
        default: return BAMG_EUNSUPPORTED;
    }
    return launched(1);
}

int launch_agg_count(int n, int nc, const int* agg, int* cnt, int* err, cudaStream_t s) {
    BAMG_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)(nc > 0 ? nc : 1), s));
    if (n <= 0) return BAMG_OK;
    agg_count_kernel<<<ceil_div(n, 256), 256, 0, s>>>(n, nc, agg, cnt, err);
    return launched(1);
}

int launch_agg_features(int nc, int F, const int* agg_ptr, const int* members, const float* node_feat, float* out,
                        cudaStream_t s) {
    if (nc <= 0) return BAMG_OK;
    agg_features_kernel<<<ceil_div((long)nc * F * kNF, 256), 256, 0, s>>>(nc, F, agg_ptr, members, node_feat, out);
    return launched(1);
}

// ---------------------------------------------------------------------------
// network
// ---------------------------------------------------------------------------
__global__ void pack_half_kernel(const float* __restrict__ p, uint16_t* __restrict__ p16) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < BAMG_MLP_NPARAMS) p16[e] = __half_as_ushort(__float2half_rn(p[e]));
}

__device__ __forceinline__ void stage_params(const uint16_t* __restrict__ p16, float* sp) {
    for (int e = threadIdx.x; e < BAMG_MLP_NPARAMS; e += blockDim.x) sp[e] = __half2float(__ushort_as_half(p16[e]));
    __syncthreads();
}

// One row (every sum from 0 in ascending index order, bias added last): h1[k]
// is produced one at a time and folded into the 64 accumulators of the second
// layer at once, so no activation array is indexed at run time and nothing
// spills.
__device__ __forceinline__ void row_infer(const float* __restrict__ sp, const float* __restrict__ x, float* y) {
    float xh[kNF], a2[kNH];
#pragma unroll
    for (int m = 0; m < kNF; ++m) xh[m] = (x[m] - sp[kOXM + m]) * sp[kOXS + m];
#pragma unroll
    for (int j = 0; j < kNH; ++j) a2[j] = 0.f;
    for (int k = 0; k < kNH; ++k) {
        float a = 0.f;
#pragma unroll
        for (int m = 0; m < kNF; ++m) a = fmaf(sp[kOW1 + k * kNF + m], xh[m], a);
        const float h = tanhf(a + sp[kOB1 + k]);
#pragma unroll
        for (int j = 0; j < kNH; ++j) a2[j] = fmaf(sp[kOW2 + j * kNH + k], h, a2[j]);
    }
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int j = 0; j < kNH; ++j) {
        const float h = tanhf(a2[j] + sp[kOB2 + j]);
        y0 = fmaf(sp[kOW3 + j], h, y0);
        y1 = fmaf(sp[kOW3 + kNH + j], h, y1);
    }
    y[0] = y0 + sp[kOB3];
    y[1] = y1 + sp[kOB3 + 1];
}

// grid-stride over rows: each CTA stages the parameters once
__global__ void __launch_bounds__(128) mlp_forward_kernel(const uint16_t* __restrict__ p16, const float* __restrict__ x,
                                                          int n, float* __restrict__ y) {
    __shared__ float sp[BAMG_MLP_NPARAMS];
    stage_params(p16, sp);
    for (long r = (long)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (long)gridDim.x * blockDim.x) {
        float xr[kNF], out[kNO];
#pragma unroll
        for (int m = 0; m < kNF; ++m) xr[m] = x[r * kNF + m];
        row_infer(sp, xr, out);
        y[r * kNO] = out[0];
        y[r * kNO + 1] = out[1];
    }
}

int launch_mlp_forward(const uint16_t* p16, const float* x, int n, float* y, cudaStream_t s) {
    if (n <= 0) return BAMG_OK;
    const int grid = ceil_div(n, 128) < 152 * 4 ? ceil_div(n, 128) : 152 * 4;
    mlp_forward_kernel<<<grid, 128, 0, s>>>(p16, x, n, y);
    return launched(1);
}

int launch_pack_half(const float* p, uint16_t* p16, cudaStream_t s) {
    pack_half_kernel<<<ceil_div(BAMG_MLP_NPARAMS, 256), 256, 0, s>>>(p, p16);
    return launched(1);
}

// Gradient of the mean squared error.  A CTA takes tiles of kTileRows rows
// (tile = its index, then every grid-th one).  Phase 1, eight threads per row
// (thread g the hidden units g, g + 8, ...): forward, dL/dy, back through both
// tanh layers; the activations and pre-activation gradients of the tile go to
// shared memory, row strides padded so that the eight units a row reads at
// once lie in distinct banks.  Phase 2: every thread adds the tile's rows, in
// ascending order, to its own parameter gradients in registers (a 4 x 4 patch
// of W2), written to partial[CTA][NTRAIN] after the last tile.  The partials
// are added in CTA order by grad_reduce_kernel: the sum depends on n alone.
// Latency-bound at the training batch of 4096 rows (128 tiles).  One thread per
// row and one output per thread took 62 us at that batch, this takes 21 us; the
// reduction, one thread per output over all tiles, 6.2 us, now 4.4 us; the whole
// step with Adam 71.7 -> 26.4 us.
constexpr int kTileRows = 32;
constexpr int kGradThreads = 256;
constexpr int kGradCtas = 304;  // at most two per SM
constexpr int kLd = kNH + 1;    // padded row stride
constexpr int kUnits = 8;       // hidden units of a thread

struct GradSmem {
    float w1[kNH][kNF + 1];
    float w2[kNH][kLd];
    float b1[kNH], b2[kNH], w3[kNO][kNH], b3[kNO], xm[kNF], xs[kNF];
    float h1[kTileRows][kLd];
    float h2[kTileRows][kLd];
    float da1[kTileRows][kLd];
    float da2[kTileRows][kLd];
    float xh[kTileRows][kNF + 1];
    float dy[kTileRows][kNO];
    float err2[kTileRows];
};

__global__ void __launch_bounds__(kGradThreads)
    mlp_grad_kernel(const uint16_t* __restrict__ p16, const float* __restrict__ x, const float* __restrict__ t,
                    const int* __restrict__ head, int n, int ntile, float* __restrict__ partial,
                    float* __restrict__ partial_loss) {
    extern __shared__ float4 smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    const int tid = threadIdx.x;
    for (int e = tid; e < BAMG_MLP_NPARAMS; e += kGradThreads) {
        const float v = __half2float(__ushort_as_half(p16[e]));
        if (e < kOB1) S.w1[e / kNF][e % kNF] = v;
        else if (e < kOW2) S.b1[e - kOB1] = v;
        else if (e < kOB2) S.w2[(e - kOW2) / kNH][(e - kOW2) % kNH] = v;
        else if (e < kOW3) S.b2[e - kOB2] = v;
        else if (e < kOB3) S.w3[(e - kOW3) / kNH][(e - kOW3) % kNH] = v;
        else if (e < kOXM) S.b3[e - kOB3] = v;
        else if (e < kOXS) S.xm[e - kOXM] = v;
        else S.xs[e - kOXS] = v;
    }
    const int row = tid / 8, g = tid & 7;        // phase 1: row of the tile, first unit
    const int tj = tid >> 4, tk = tid & 15;      // phase 2: W2 entries (tj + 16 a, tk + 16 b)
    float gw2[4][4] = {}, gw1[2] = {0.f, 0.f}, gsm = 0.f, loss = 0.f;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        __syncthreads();  // the parameters; the previous tile's phase 2
        const long r = (long)tile * kTileRows + row;
        const bool act = r < n;
        S.xh[row][g] = ((act ? x[r * kNF + g] : 0.f) - S.xm[g]) * S.xs[g];
        __syncwarp();  // a row's eight threads are lanes of one warp
        float h1[kUnits], h2[kUnits];
#pragma unroll
        for (int u = 0; u < kUnits; ++u) {
            const int k = g + 8 * u;
            float a = 0.f;
#pragma unroll
            for (int m = 0; m < kNF; ++m) a = fmaf(S.w1[k][m], S.xh[row][m], a);
            h1[u] = tanhf(a + S.b1[k]);
            S.h1[row][k] = h1[u];
        }
        __syncwarp();
        float a2[kUnits] = {};
#pragma unroll 4
        for (int k = 0; k < kNH; ++k) {
            const float h = S.h1[row][k];
#pragma unroll
            for (int u = 0; u < kUnits; ++u) a2[u] = fmaf(S.w2[g + 8 * u][k], h, a2[u]);
        }
        float y0 = 0.f, y1 = 0.f;
#pragma unroll
        for (int u = 0; u < kUnits; ++u) {
            const int j = g + 8 * u;
            h2[u] = tanhf(a2[u] + S.b2[j]);
            S.h2[row][j] = h2[u];
            y0 = fmaf(S.w3[0][j], h2[u], y0);
            y1 = fmaf(S.w3[1][j], h2[u], y1);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            y0 += __shfl_xor_sync(0xffffffffu, y0, o);
            y1 += __shfl_xor_sync(0xffffffffu, y1, o);
        }
        float dy0 = 0.f, dy1 = 0.f, e2 = 0.f;
        if (act) {
            const int hd = head[r];
            const float e = (hd == 0 ? y0 + S.b3[0] : y1 + S.b3[1]) - t[r];
            e2 = e * e;
            const float gr = 2.f * e / (float)n;
            dy0 = hd == 0 ? gr : 0.f;
            dy1 = hd == 0 ? 0.f : gr;
        }
        if (g == 0) {
            S.dy[row][0] = dy0;
            S.dy[row][1] = dy1;
            S.err2[row] = e2;
        }
#pragma unroll
        for (int u = 0; u < kUnits; ++u) {
            const int j = g + 8 * u;
            S.da2[row][j] = (dy0 * S.w3[0][j] + dy1 * S.w3[1][j]) * (1.f - h2[u] * h2[u]);
        }
        __syncwarp();
        float a1[kUnits] = {};
#pragma unroll 4
        for (int j = 0; j < kNH; ++j) {
            const float d = S.da2[row][j];
#pragma unroll
            for (int u = 0; u < kUnits; ++u) a1[u] = fmaf(S.w2[j][g + 8 * u], d, a1[u]);
        }
#pragma unroll
        for (int u = 0; u < kUnits; ++u) S.da1[row][g + 8 * u] = a1[u] * (1.f - h1[u] * h1[u]);
        __syncthreads();
#pragma unroll 2
        for (int q = 0; q < kTileRows; ++q) {
            float dj[4], hk[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                dj[u] = S.da2[q][tj + 16 * u];
                hk[u] = S.h1[q][tk + 16 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) gw2[u][v] = fmaf(dj[u], hk[v], gw2[u][v]);
        }
        // W1: entries tid and tid + 256 of 512; then b1, b2, W3 (one each) and b3, loss
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = (tid + u * kGradThreads) / kNF, m = (tid + u * kGradThreads) % kNF;
#pragma unroll 8
            for (int q = 0; q < kTileRows; ++q) gw1[u] = fmaf(S.da1[q][k], S.xh[q][m], gw1[u]);
        }
        if (tid < kNH) {
#pragma unroll 8
            for (int q = 0; q < kTileRows; ++q) gsm += S.da1[q][tid];
        } else if (tid < 2 * kNH) {
#pragma unroll 8
            for (int q = 0; q < kTileRows; ++q) gsm += S.da2[q][tid - kNH];
        } else {
            const int o = (tid - 2 * kNH) / kNH, j = (tid - 2 * kNH) % kNH;
#pragma unroll 8
            for (int q = 0; q < kTileRows; ++q) gsm = fmaf(S.dy[q][o], S.h2[q][j], gsm);
        }
        if (tid < kNO) {  // (b3: a second small sum of these threads, kept with the loss)
            for (int q = 0; q < kTileRows; ++q) loss += S.dy[q][tid];
        } else if (tid == kNO) {
            for (int q = 0; q < kTileRows; ++q) loss += S.err2[q];
        }
    }
    float* out = partial + (size_t)blockIdx.x * BAMG_MLP_NTRAIN;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) out[kOW2 + (tj + 16 * u) * kNH + tk + 16 * v] = gw2[u][v];
    out[kOW1 + tid] = gw1[0];
    out[kOW1 + tid + kGradThreads] = gw1[1];
    if (tid < kNH) out[kOB1 + tid] = gsm;
    else if (tid < 2 * kNH) out[kOB2 + tid - kNH] = gsm;
    else out[kOW3 + tid - 2 * kNH] = gsm;
    if (tid < kNO) out[kOB3 + tid] = loss;
    else if (tid == kNO) partial_loss[blockIdx.x] = loss;
}
static_assert(kNH * kNF == 2 * kGradThreads && kGradThreads == 4 * kNH && kNO == 2 && kTileRows * 8 == kGradThreads,
              "work split of mlp_grad_kernel");

// grad[o] = sum over the CTAs of partial[CTA][o]: a CTA takes 32 outputs, warp w
// the w-th eighth of the CTAs in ascending order, then the eighths in order;
// output NTRAIN is the loss, divided by n
__global__ void __launch_bounds__(256) grad_reduce_kernel(int nctas, int n, const float* __restrict__ partial,
                                                          const float* __restrict__ partial_loss,
                                                          float* __restrict__ grad, float* __restrict__ loss) {
    __shared__ float sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    const int per = (nctas + 7) / 8, c0 = w * per, c1 = min(nctas, c0 + per);
    float s = 0.f;
    if (o < BAMG_MLP_NTRAIN) {
#pragma unroll 8
        for (int c = c0; c < c1; ++c) s += partial[(size_t)c * BAMG_MLP_NTRAIN + o];
    } else if (o == BAMG_MLP_NTRAIN) {
        for (int c = c0; c < c1; ++c) s += partial_loss[c];
    }
    sh[w][lane] = s;
    __syncthreads();
    if (w != 0 || o > BAMG_MLP_NTRAIN) return;
    s = 0.f;
#pragma unroll
    for (int v = 0; v < 8; ++v) s += sh[v][lane];
    if (o < BAMG_MLP_NTRAIN) grad[o] = s;
    else *loss = s / (float)n;
}

static int grad_ctas(int n) {
    const int ntile = ceil_div(n, kTileRows);
    return ntile < kGradCtas ? ntile : kGradCtas;
}
size_t mlp_grad_workspace(int n) {
    return sizeof(float) * (size_t)grad_ctas(n) * (BAMG_MLP_NTRAIN + 1);
}

int launch_mlp_grad(const uint16_t* p16, const float* x, const float* t, const int* head, int n, float* grad,
                    float* loss, float* work, cudaStream_t s) {
    if (n < 1) return BAMG_EINVAL;
    const int nctas = grad_ctas(n);
    const size_t smem = sizeof(GradSmem);
    // more than 48 KB of dynamic shared memory needs the opt-in (idempotent)
    BAMG_CUDA_TRY(cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(GradSmem)));
    float* partial = work;
    float* partial_loss = work + (size_t)nctas * BAMG_MLP_NTRAIN;
    mlp_grad_kernel<<<nctas, kGradThreads, smem, s>>>(p16, x, t, head, n, ceil_div(n, kTileRows), partial,
                                                      partial_loss);
    grad_reduce_kernel<<<ceil_div(BAMG_MLP_NTRAIN + 1, 32), 256, 0, s>>>(nctas, n, partial, partial_loss, grad, loss);
    return launched(2);
}

// Adam with bias-corrected moments on the trained parameters; c1 = 1 -
// beta1^t, c2 = 1 - beta2^t; then the FP16 copy of every parameter
__global__ void adam_kernel(float* __restrict__ p, uint16_t* __restrict__ p16, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, float lr, float beta1, float beta2,
                            float eps, float c1, float c2) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= BAMG_MLP_NPARAMS) return;
    if (e < BAMG_MLP_NTRAIN) {
        const float gg = g[e];
        const float mm = beta1 * m[e] + (1.f - beta1) * gg;
        const float vv = beta2 * v[e] + (1.f - beta2) * gg * gg;
        m[e] = mm;
        v[e] = vv;
        p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
    p16[e] = __half_as_ushort(__float2half_rn(p[e]));
}

int launch_adam(float* p, uint16_t* p16, const float* g, float* m, float* v, float lr, float beta1, float beta2,
                float eps, float c1, float c2, cudaStream_t s) {
    adam_kernel<<<ceil_div(BAMG_MLP_NPARAMS, 256), 256, 0, s>>>(p, p16, g, m, v, lr, beta1, beta2, eps, c1, c2);
    return launched(1);
}

// ---------------------------------------------------------------------------
// weights of a level from the network outputs (same ranges as mlp_clip):
// out64[r] = clip_head(y[r][head]); *any = 1 if some value is nonzero
// ---------------------------------------------------------------------------
__device__ __forceinline__ double clip_weight(int head, double w) {
    if (head == 0) return !(w >= 0.05) ? 0.05 : (w > 1.5 ? 1.5 : w);
    return !(w >= 0.05) ? 0.0 : (w > 1.5 ? 1.5 : w);
}

__global__ void omega_from_mlp_kernel(int rows, int head, const float* __restrict__ y, double* __restrict__ out,
                                      int* __restrict__ any) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const double w = clip_weight(head, (double)y[(size_t)r * kNO + head]);
    out[r] = w;
    if (any && w > 0.0) atomicOr(any, 1);
}

int launch_omega_from_mlp(int rows, int head, const float* y, double* out, int* any, cudaStream_t s) {
    if (rows <= 0) return BAMG_OK;
    omega_from_mlp_kernel<<<ceil_div(rows, 256), 256, 0, s>>>(rows, head, y, out, any);
    return launched(1);
}

__global__ void fill_kernel(long m, double v, double* __restrict__ out) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < m) out[e] = v;
}

int launch_fill(long m, double v, double* out, cudaStream_t s) {
    if (m <= 0) return BAMG_OK;
    fill_kernel<<<ceil_div(m, 256), 256, 0, s>>>(m, v, out);
    return launched(1);
}

}  // namespace bamg

extern "C" double mlp_clip(int head, double w) {
    if (head == 0) return !(w >= 0.05) ? 0.05 : (w > 1.5 ? 1.5 : w);
    return !(w >= 0.05) ? 0.0 : (w > 1.5 ? 1.5 : w);
}
