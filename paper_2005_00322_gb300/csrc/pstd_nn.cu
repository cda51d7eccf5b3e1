// pstd_nn.cu -- kernels of the learned spectral operator (forward, backward, Adam).
//
// The network works in the wall-respecting sine/cosine basis of each axis
// (the truncated T1 of Table 2), so every operation is one of:
//   * a strided batched GEMM  C[b] = alpha A[b] B[b] + beta C[b]  with
//     arbitrary element strides (the per-axis transforms, the per-mode channel
//     mixing, the pointwise channel mixing and all their adjoints);
//   * per-channel elementwise work (lift, bias + ReLU, projection) and their
//     gradients, and per-channel reductions;
//   * an Adam update.
// The GEMM tiles 64 x 64 outputs per CTA (4 x 4 per thread) over 16-wide k
// slices staged in shared memory, FP32 throughout.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <type_traits>
#include <vector>

#include "pstd.h"

namespace {

// One CTA of 256 threads computes a BM x BN tile of C[b] (TM x TN per
// thread) over 16-wide k slices staged in shared memory.  Tile shapes:
// 64 x 64 for square-ish products, 256 x 16 / 16 x 256 for the tall or wide
// products with a mode count (16) on one side, 16 x 16 for the small per-line
// transforms, 32 x 32 for many channel-by-channel products (the weight gradients
// of 32 channels over 2048 chunks of 256 points: 152 us on 16 x 16 tiles).
template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(256) k_sgemm(pstd_gemm_desc d) {
    static_assert((BM / TM) * (BN / TN) == 256, "256 threads");
    constexpr int LA = 16 * BM / 256, LB = 16 * BN / 256;
    static_assert(LA >= 1 && LB >= 1, "tile too small");
    __shared__ float As[16][BM + 4];
    __shared__ float Bs[16][BN + 4];
    const int tid = threadIdx.x;
    const int tx = tid % (BN / TN), ty = tid / (BN / TN);
    const int64_t nb2 = d.batch2 > 1 ? d.batch2 : 1;
    const int64_t b1 = blockIdx.z / nb2, b2 = blockIdx.z - b1 * nb2;
    const int K = (nb2 > 1 && b2 == nb2 - 1) ? d.K_last : d.K;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const float* A = d.A + b1 * d.sAb + b2 * d.sAb2;
    const float* B = d.B + b1 * d.sBb + b2 * d.sBb2;
    float* C = d.C + b1 * d.sCb + b2 * d.sCb2;
    const bool a_kfast = d.sAk == 1 && d.sAm != 1;
    const bool b_kfast = d.sBk == 1 && d.sBn != 1;
    // This thread's slots in the staged k slice (consecutive threads walk the
    // operand's unit-stride index, so the global loads coalesce).
    int akk[LA], amm[LA], bkk[LB], bnn[LB];
#pragma unroll
    for (int i = 0; i < LA; ++i) {
        const int idx = tid + i * 256;
        akk[i] = a_kfast ? (idx & 15) : (idx / BM);
        amm[i] = a_kfast ? (idx >> 4) : (idx % BM);
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
        const int idx = tid + i * 256;
        bkk[i] = b_kfast ? (idx & 15) : (idx / BN);
        bnn[i] = b_kfast ? (idx >> 4) : (idx % BN);
    }
    float ra[LA], rb[LB];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int m = m0 + amm[i], k = k0 + akk[i];
            ra[i] = (m < d.M && k < K) ? A[m * d.sAm + k * d.sAk] : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int n = n0 + bnn[i], k = k0 + bkk[i];
            rb[i] = (n < d.N && k < K) ? B[k * d.sBk + n * d.sBn] : 0.0f;
        }
    };
    float acc[TM][TN] = {};
    if (K > 0) fetch(0);
    for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
        for (int i = 0; i < LA; ++i) As[akk[i]][amm[i]] = ra[i];
#pragma unroll
        for (int i = 0; i < LB; ++i) Bs[bkk[i]][bnn[i]] = rb[i];
        __syncthreads();
        if (k0 + 16 < K) fetch(k0 + 16);      // next slice in flight during this one's FMAs
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            float a[TM], bb[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
            for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx * TN + j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + ty * TM + i;
        if (m >= d.M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int n = n0 + tx * TN + j;
            if (n >= d.N) continue;
            float* c = &C[m * d.sCm + n * d.sCn];
            *c = d.beta != 0.0f ? d.alpha * acc[i][j] + d.beta * *c : d.alpha * acc[i][j];
        }
    }
}

// Row kernels: blockIdx.y is the row r = b C + c of a [B][C][P] tensor and
// the x blocks stride over its P points (no per-element index division).

// y[b, c, i] = act(x[b, c, i] + bias[c]) (act: 0 identity, 1 relu)
__global__ void k_bias_act(const float* x, const float* bias, float* y, int C, int64_t P, int act) {
    const int64_t r = blockIdx.y;
    const float bv = bias ? bias[r % C] : 0.0f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const float v = x[r * P + i] + bv;
        y[r * P + i] = act == 1 ? fmaxf(v, 0.0f) : v;
    }
}

// dx = dy * (pre > 0)  (relu) or dy (identity), in place allowed
__global__ void k_act_bwd(const float* dy, const float* pre, float* dx, int64_t n, int act) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x)
        dx[t] = (act == 1 && pre[t] <= 0.0f) ? 0.0f : dy[t];
}

// v[b, c, i] = w[c] p[b, i] + bias[c].  A thread writes G channels of its
// points (blockIdx.y = b and its group of channels): with a row of CTAs per
// (b, c) and one point per thread, 256 x 32 rows of 16383 points took 536 us for
// 537 MB; with all channels in a thread, one sample of 32 x 2^20 92 us against 39.
__global__ void k_lift(const float* p, const float* w, const float* bias, float* v, int C, int G, int64_t P) {
    const int ng = (C + G - 1) / G;
    const int64_t b = blockIdx.y / ng;
    const int c0 = (int)(blockIdx.y - b * ng) * G, c1 = c0 + G < C ? c0 + G : C;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const float x = p[b * P + i];
        float* q = v + (b * C + c0) * P + i;
#pragma unroll 8
        for (int c = c0; c < c1; ++c, q += P) *q = fmaf(w[c], x, bias[c]);
    }
}

// out[b, i] = sum_c w[c] v[b, c, i] + bias  (blockIdx.y = b)
__global__ void k_proj(const float* v, const float* w, const float* bias, float* out, int C, int64_t P) {
    const int64_t b = blockIdx.y;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        float acc = bias[0];
        for (int c = 0; c < C; ++c) acc = fmaf(w[c], v[(b * C + c) * P + i], acc);
        out[b * P + i] = acc;
    }
}

// dv[b, c, i] = w[c] dout[b, i]  (as k_lift)
__global__ void k_proj_bwd(const float* dout, const float* w, float* dv, int C, int G, int64_t P) {
    const int ng = (C + G - 1) / G;
    const int64_t b = blockIdx.y / ng;
    const int c0 = (int)(blockIdx.y - b * ng) * G, c1 = c0 + G < C ? c0 + G : C;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const float x = dout[b * P + i];
        float* q = dv + (b * C + c0) * P + i;
#pragma unroll 8
        for (int c = c0; c < c1; ++c, q += P) *q = w[c] * x;
    }
}

// Sums in FP64 run at a few operations per clock and SM, so a reduction is
// spread over the GPU: the R <= kRed CTAs of one cluster each add up a share, and
// the first adds the shares through distributed shared memory in a fixed order
// (no workspace, no atomics, the same bits each time).
constexpr int kRed = 8;
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}
// Sum over the cluster's R CTAs of `acc` over their threads (256), valid in
// thread 0 of rank 0.
__device__ double cluster_sum(double acc, unsigned R) {
    __shared__ double red[256];
    __shared__ double part;
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (R == 1) return red[0];
    if (threadIdx.x == 0) part = red[0];
    cluster_sync();
    double tot = 0.0;
    if (cluster_rank() == 0 && threadIdx.x == 0) {
        const unsigned mine = (unsigned)__cvta_generic_to_shared(&part);
        for (unsigned r = 0; r < R; ++r) {
            unsigned at;
            double v;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(mine), "r"(r));
            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(at));
            tot += v;
        }
    }
    cluster_sync();          // no CTA leaves while its share may be read
    return tot;
}

// g[c] = sum_{b, i} x[b, c, i] * (y ? y[b, c or -, i] : 1); y indexed [b, i] when ybc == 0
// One cluster of R CTAs per channel, which share out its samples (by_sample) or
// the points of each.  With one CTA per channel (32 of the SMs) 32 channels of
// 32 x 16383 points took 138 us of FP64 adds alone; with eight 4096 channels of
// 64 points 209 us against 21, and the points of 16 samples of 1024 shared out
// 29 us against 16.
__global__ void __launch_bounds__(256) k_chan_dot(const float* x, const float* y, int ybc, float* g, int64_t B, int C,
                                                  int64_t P, int R, int by_sample) {
    const int c = blockIdx.x / R;
    const int64_t rank = R > 1 ? cluster_rank() : 0;
    // four independent chains of adds and loads per thread
    double acc[4] = {};
    const int64_t step = (by_sample ? 1 : R) * 256, i0 = (by_sample ? 0 : rank * 256) + threadIdx.x;
    for (int64_t b = by_sample ? rank : 0; b < B; b += by_sample ? R : 1) {
        const float* xr = x + (b * C + c) * P;
        const float* yr = y ? (ybc ? y + (b * C + c) * P : y + b * P) : nullptr;
        int64_t i = i0;
        for (; i + 3 * step < P; i += 4 * step) {
            float xv[4], yv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                xv[q] = xr[i + q * step];
                yv[q] = yr ? yr[i + q * step] : 1.0f;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += (double)xv[q] * (double)yv[q];
        }
        for (; i < P; i += step) acc[0] += (double)xr[i] * (yr ? (double)yr[i] : 1.0);
    }
    // (rows too short for the unrolled loop skip the additions of its chains)
    const double own = 3 * step < P ? (acc[0] + acc[1]) + (acc[2] + acc[3]) : acc[0];
    const double tot = cluster_sum(own, R);
    if (rank == 0 && threadIdx.x == 0) g[c] = (float)tot;
}

// out[j] = sum_b x[b, j] (sum over the leading dimension), a thread per column:
// enough threads where there are many more columns than rows.
__global__ void k_sum_columns(const float* x, float* out, int64_t B, int64_t n) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int64_t b = 0; b < B; ++b) acc += x[b * n + j];
        out[j] = (float)acc;
    }
}
// As k_sum_columns with a CTA for 8 columns, its 32 groups of 8 threads every
// 32nd row each: 2048 x 1024 14 us against 294; but 1 x 2^20 285 against 10, 64 x
// 65536 45 against 23.
__global__ void __launch_bounds__(256) k_sum_lead(const float* x, float* out, int64_t B, int64_t n) {
    const int col = threadIdx.x & 7, grp = threadIdx.x >> 3;
    __shared__ double red[32][8];
    for (int64_t j0 = (int64_t)blockIdx.x * 8; j0 < n; j0 += (int64_t)gridDim.x * 8) {
        const int64_t j = j0 + col;
        double acc = 0.0;
        if (j < n)
            for (int64_t b = grp; b < B; b += 32) acc += x[b * n + j];
        red[grp][col] = acc;
        __syncthreads();
        if (grp == 0 && j < n) {
            double t = 0.0;
            for (int q = 0; q < 32; ++q) t += red[q][col];
            out[j] = (float)t;
        }
        __syncthreads();
    }
}

// Adam (Kingma & Ba) with bias correction; step t >= 1
__global__ void k_adam(float* w, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const float gg = g[t];
        const float mm = b1 * m[t] + (1.0f - b1) * gg;
        const float vv = b2 * v[t] + (1.0f - b2) * gg * gg;
        m[t] = mm;
        v[t] = vv;
        w[t] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
}

// Block-wide FP64 sum of one value per thread (blockDim.x a power of two <= 1024).
__device__ double block_sum(double v) {
    __shared__ double red[1024];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

// Mean squared error of out against target (one cluster): loss[0] =
// mean (out - t)^2, dout = (2 / n) (out - target).
__global__ void __launch_bounds__(256) k_mse(const float* out, const float* target, float* dout, float* loss,
                                             int64_t n) {
    double acc = 0.0;
    const float s = 2.0f / (float)n;
    for (int64_t t = cluster_rank() * blockDim.x + threadIdx.x; t < n; t += kRed * blockDim.x) {
        const float df = out[t] - target[t];
        acc += (double)df * (double)df;
        if (dout) dout[t] = s * df;
    }
    const double tot = cluster_sum(acc, kRed);
    if (cluster_rank() == 0 && threadIdx.x == 0) loss[0] = (float)(tot / (double)n);
}

// Per sample b (one CTA each): err[b] = ||a_b - r_b||_2 / ||r_b||_2.
__global__ void k_rel_err(const float* a, const float* r, float* err, int64_t P) {
    const int64_t b = blockIdx.x;
    double num = 0.0, den = 0.0;
    for (int64_t t = threadIdx.x; t < P; t += blockDim.x) {
        const double x = a[b * P + t], y = r[b * P + t];
        num += (x - y) * (x - y);
        den += y * y;
    }
    num = block_sum(num);
    den = block_sum(den);
    if (threadIdx.x == 0) err[b] = den > 0.0 ? (float)sqrt(num / den) : (float)sqrt(num);
}

// dst = src rounded to the nearest bfloat16 (ties to even), kept in FP32 storage.
__global__ void k_round_bf16(const float* src, float* dst, int64_t n) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        dst[t] = __bfloat162float(__float2bfloat16_rn(src[t]));
}

// rms[b] = sqrt(mean_i x[b, i]^2) (one CTA per sample, FP64 sum)
__global__ void k_row_rms(const float* x, float* rms, int64_t P) {
    const int64_t b = blockIdx.x;
    double acc = 0.0;
    for (int64_t i = threadIdx.x; i < P; i += blockDim.x) acc += (double)x[b * P + i] * x[b * P + i];
    acc = block_sum(acc);
    if (threadIdx.x == 0) rms[b] = (float)sqrt(acc / (double)P);
}

// y[b, i] = x[b, i] / s[b] (mode 0, s[b] == 0 gives 0) or x[b, i] * s[b] (mode 1)
__global__ void k_row_scale(const float* x, const float* sc, float* y, int64_t P, int mode) {
    const int64_t b = blockIdx.y;
    const float f = mode == 1 ? sc[b] : (sc[b] > 0.0f ? 1.0f / sc[b] : 0.0f);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x)
        y[b * P + i] = x[b * P + i] * f;
}

// ---- pointwise and spectral half of a layer in one pass ----------------------
// out[b, o, x, y] = act( sum_i W[o, i] v[b, i, x, y] + sum_k A[b, o, x, k] T[k, y] + bias[o] ),
// or, with `mask`, that value where mask > 0 and 0 elsewhere.  As separate
// products, bias and activation the field went through memory seven times;
// here v is read and out written once.  Each sum runs in index order and they
// are added last, so every value has the bits of the separate products (a relu
// argument near zero keeps its sign).
// A CTA of 4 warps takes nx <= kMixX consecutive x of a sample and 128 y, the next
// x's rows arriving (cp.async, second buffer) behind the current one's
// products: lanes walk y (4 each, 32 apart, so shared reads and global accesses
// are full lines), each warp has 8 output channels.  A CTA whose y end within 32
// or 64 takes 1 or 2 per lane, and warps beyond the channels only copy (4 channels
// of 129 x 9 points, 256 samples, four layers: 708 us without either).  256 samples of 32 channels
// of 129 x 127 points: 0.44 ms a layer against 1.9 ms for the separate launches;
// bound by shared-memory reads and issue (the multiply-adds alone are 0.17 ms,
// the field's bytes 0.16 ms).
constexpr int kMixC = 32, kMixK = 32, kMixX = 8, kMixY = 128;
struct MixArgs {
    const float* W;
    int64_t sWo, sWi;
    const float* v;
    const float* A;
    const float* T;
    int64_t sTk, sTy;
    const float* bias;
    const float* mask;
    float* out;
    int C, X, Y, K, act, nx;
};
__device__ __forceinline__ void copy4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// acc[m][q] += sum_j cf[j][m] rows[j][q], j ascending
template <int Q>
__device__ __forceinline__ void mix_rows(float (&acc)[8][Q], const float* cf, const float* rows, int n) {
    const float4* cp = (const float4*)cf;
#pragma unroll 4
    for (int j = 0; j < n; ++j, rows += kMixY, cp += kMixC / 4) {
        const float4 c0 = cp[0], c1 = cp[1];
        const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        float r[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) r[q] = rows[32 * q];
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
            for (int q = 0; q < Q; ++q) acc[m][q] = fmaf(c[m], r[q], acc[m][q]);
    }
}
inline size_t mix_smem(int C, int K) {
    return (size_t)(2 * C * kMixY + K * kMixY + C * kMixC + 2 * K * kMixC) * sizeof(float);
}
__global__ void __launch_bounds__(128) k_mix(MixArgs a) {
    extern __shared__ float sm[];
    float* const vr = sm;                               // [2][C][128]
    float* const tr = vr + 2 * a.C * kMixY;             // [K][128]
    float* const wc = tr + a.K * kMixY;                 // [C][32]: W of (input, output channel)
    float* const ac = wc + a.C * kMixC;                 // [2][K][32]: A of (mode, output channel)
    const int tid = threadIdx.x, lane = tid & 31, wrp = tid >> 5;
    const int y0 = blockIdx.x * kMixY, x0 = blockIdx.y * a.nx;
    const int ny = a.Y - y0 < kMixY ? a.Y - y0 : kMixY;
    const int64_t b = blockIdx.z, P = (int64_t)a.X * a.Y;
    const int x1 = x0 + a.nx < a.X ? x0 + a.nx : a.X;
    auto issue = [&](int x, int buf) {
        float* d = vr + buf * a.C * kMixY;
        for (int i = wrp; i < a.C; i += 4) {
            const float* src = a.v + (b * a.C + i) * P + (int64_t)x * a.Y + y0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int y = lane + 32 * q;
                if (y < ny) copy4(&d[i * kMixY + y], &src[y]);
            }
        }
        float* e = ac + buf * a.K * kMixC;
        for (int t = tid; t < a.K * a.C; t += 128) {
            const int o = t / a.K, k = t - o * a.K;
            copy4(&e[k * kMixC + o], &a.A[((b * a.C + o) * a.X + x) * a.K + k]);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    issue(x0, 0);
    // columns and channels past the end stay zero in both buffers
    for (int t = tid; t < 2 * a.C * kMixY; t += 128)
        if (t % kMixY >= ny) vr[t] = 0.0f;
    for (int t = tid; t < 2 * a.K * kMixC; t += 128)
        if (t % kMixC >= a.C) ac[t] = 0.0f;
    for (int t = tid; t < a.C * kMixC; t += 128) {
        const int i = t / kMixC, o = t % kMixC;
        wc[t] = o < a.C ? a.W[o * a.sWo + i * a.sWi] : 0.0f;
    }
    for (int t = tid; t < a.K * kMixY; t += 128) {
        const int k = t / kMixY, y = t % kMixY;
        tr[t] = y < ny ? a.T[k * a.sTk + (y0 + y) * a.sTy] : 0.0f;
    }
    auto rows = [&](auto nq) {
        constexpr int Q = decltype(nq)::value;
        for (int x = x0; x < x1; ++x) {
            const int buf = (x - x0) & 1;
            if (x + 1 < x1) {
                issue(x + 1, buf ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            float aw[8][Q] = {}, as[8][Q] = {};
            if (wrp * 8 < a.C) {
                mix_rows<Q>(as, ac + buf * a.K * kMixC + wrp * 8, tr + lane, a.K);
                mix_rows<Q>(aw, wc + wrp * 8, vr + buf * a.C * kMixY + lane, a.C);
            }
            __syncthreads();                       // this buffer may be refilled
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int o = wrp * 8 + m;
                if (o >= a.C) break;
                const int64_t off = (b * a.C + o) * P + (int64_t)x * a.Y + y0;
                const float bv = a.bias ? a.bias[o] : 0.0f;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int y = lane + 32 * q;
                    if (y >= ny) continue;
                    float z = aw[m][q] + as[m][q];
                    if (a.bias) z += bv;
                    if (a.act == 1) z = fmaxf(z, 0.0f);
                    if (a.mask && a.mask[off + y] <= 0.0f) z = 0.0f;
                    a.out[off + y] = z;
                }
            }
        }
    };
    if (ny <= 32) rows(std::integral_constant<int, 1>{});
    else if (ny <= 64) rows(std::integral_constant<int, 2>{});
    else rows(std::integral_constant<int, 4>{});
}

// Launch on clusters of R CTAs.
template <class... KA, class... CA>
cudaError_t launch_cluster(void (*k)(KA...), unsigned R, unsigned grid, cudaStream_t st, CA... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = R;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = R > 1;
    return cudaLaunchKernelEx(&cfg, k, static_cast<KA>(args)...);
}

dim3 row_grid(int64_t rows, int64_t P) {
    int64_t bx = (P + 255) / 256;
    return dim3((unsigned)(bx < 64 ? (bx > 0 ? bx : 1) : 64), (unsigned)rows);
}

// k_lift and k_proj_bwd: a thread per point (more than 64 CTAs a row: with 64, a
// row of 2^20 points took 55 us against 40), and as many channels in it as leave
// eight CTAs per SM.
int channel_group(int64_t B, int C, int64_t P) {
    const int64_t bx = (P + 255) / 256;
    int n = 1;                                   // groups
    while (n < C && B * n * bx < 152 * 8) n *= 2;
    return (C + n - 1) / n;
}
dim3 channel_grid(int64_t B, int C, int G, int64_t P) {
    const int64_t bx = (P + 255) / 256;
    return dim3((unsigned)(bx < 1 << 20 ? bx : 1 << 20), (unsigned)(B * ((C + G - 1) / G)));
}
unsigned blocks_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (unsigned)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}

int cuda_rc(cudaError_t e) { return e == cudaSuccess ? PSTD_OK : PSTD_ECUDA; }

}  // namespace

extern "C" {

int pstd_nn_gemm(const pstd_gemm_desc* d, void* stream) {
    if (!d || d->batch < 1 || d->M < 0 || d->N < 0 || d->K < 0 || !d->C) return PSTD_EINVAL;
    if (d->K > 0 && (!d->A || !d->B)) return PSTD_EINVAL;
    if (d->M == 0 || d->N == 0) return PSTD_OK;
    const int64_t nb2 = d->batch2 > 1 ? d->batch2 : 1;
    if (nb2 > 1 && (d->K_last < 0 || d->K_last > d->K || (d->K_last > 0 && (!d->A || !d->B)))) return PSTD_EINVAL;
    if (d->batch * nb2 > 65535 || (d->M + 255) / 256 > 65535) return PSTD_EINVAL;
    // The tile shape that computes the fewest padded outputs (ties: 64 x 64), the
    // small tiles charged for their operand traffic: 1056 x 1056 x 256 takes 29 us on
    // 64 x 64 tiles, 38 on 32 x 32.  32 x 32 tiles only where they fill the GPU (one
    // product 32 x 32 x 1024: 27 us, 19 on four 16 x 16 tiles).
    static const int shapes[5][2] = {{64, 64}, {256, 16}, {16, 256}, {16, 16}, {32, 32}};
    int best = 0;
    int64_t best_cost = -1;
    for (int t = 0; t < 5; ++t) {
        const int64_t bm = shapes[t][0], bn = shapes[t][1];
        const int64_t gm = (d->M + bm - 1) / bm;
        if (gm > 65535) continue;
        const int64_t gn = (d->N + bn - 1) / bn;
        if (t == 4 && gm * gn * d->batch * nb2 < 152) continue;
        const int64_t cost = gm * bm * gn * bn * (t == 3 ? 4 : t == 4 ? 3 : 2);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = t; }
    }
    const cudaStream_t st = (cudaStream_t)stream;
    const unsigned gz = (unsigned)(d->batch * nb2);
    const int bm = shapes[best][0], bn = shapes[best][1];
    const dim3 grid((unsigned)((d->N + bn - 1) / bn), (unsigned)((d->M + bm - 1) / bm), gz);
    switch (best) {
        case 0: k_sgemm<64, 64, 4, 4><<<grid, 256, 0, st>>>(*d); break;
        case 1: k_sgemm<256, 16, 4, 4><<<grid, 256, 0, st>>>(*d); break;
        case 2: k_sgemm<16, 256, 4, 4><<<grid, 256, 0, st>>>(*d); break;
        case 4: k_sgemm<32, 32, 2, 2><<<grid, 256, 0, st>>>(*d); break;
        default: k_sgemm<16, 16, 1, 1><<<grid, 256, 0, st>>>(*d); break;
    }
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_mix(const float* W, int w_transposed, const float* v, const float* A, const float* T, int t_by_mode,
                const float* bias, const float* mask, float* out, int64_t B, int C, int X, int Y, int K, int act,
                void* stream) {
    if (!W || !v || !A || !T || !out || B < 0 || C < 1 || X < 0 || Y < 0 || K < 1 || (act != 0 && act != 1))
        return PSTD_EINVAL;
    if (C > kMixC || K > kMixK || B > 65535 || (X + kMixX - 1) / kMixX > 65535) return PSTD_EUNSUPPORTED;
    if (B == 0 || X == 0 || Y == 0) return PSTD_OK;
    MixArgs a;
    a.W = W;
    a.sWo = w_transposed ? 1 : C;
    a.sWi = w_transposed ? C : 1;
    a.v = v;
    a.A = A;
    a.T = T;
    a.sTk = t_by_mode ? Y : 1;
    a.sTy = t_by_mode ? 1 : K;
    a.bias = bias;
    a.mask = mask;
    a.out = out;
    a.C = C;
    a.X = X;
    a.Y = Y;
    a.K = K;
    a.act = act;
    // eight x per CTA share its copy of W and T; fewer where that leaves SMs idle
    // (one sample of 32 channels of 129 x 127 points: 17 CTAs)
    const int64_t ny = (Y + kMixY - 1) / kMixY;
    a.nx = kMixX;
    while (a.nx > 1 && ny * ((X + a.nx - 1) / a.nx) * B < 2 * 152) a.nx /= 2;
    const dim3 grid((unsigned)ny, (unsigned)((X + a.nx - 1) / a.nx), (unsigned)B);
    const size_t smem = mix_smem(C, K);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_mix, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)mix_smem(kMixC, kMixK));
        if (e != cudaSuccess) return PSTD_ECUDA;
    }
    k_mix<<<grid, 128, smem, (cudaStream_t)stream>>>(a);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_bias_act(const float* x, const float* bias, float* y, int64_t B, int C, int64_t P, int act,
                     void* stream) {
    if (!x || !y || B < 0 || C < 1 || P < 0 || B * C > 65535 || (act != 0 && act != 1)) return PSTD_EINVAL;
    if (B == 0 || P == 0) return PSTD_OK;
    k_bias_act<<<row_grid(B * C, P), 256, 0, (cudaStream_t)stream>>>(x, bias, y, C, P, act);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_act_bwd(const float* dy, const float* pre, float* dx, int64_t n, int act, void* stream) {
    if (!dy || !dx || (act == 1 && !pre) || n < 0) return PSTD_EINVAL;
    k_act_bwd<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(dy, pre, dx, n, act);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_lift(const float* p, const float* w, const float* bias, float* v, int64_t B, int C, int64_t P,
                 void* stream) {
    if (!p || !w || !bias || !v || C < 1 || B < 0 || P < 0 || B * C > 65535) return PSTD_EINVAL;
    if (B == 0 || P == 0) return PSTD_OK;
    const int G = channel_group(B, C, P);
    k_lift<<<channel_grid(B, C, G, P), 256, 0, (cudaStream_t)stream>>>(p, w, bias, v, C, G, P);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_proj(const float* v, const float* w, const float* bias, float* out, int64_t B, int C, int64_t P,
                 void* stream) {
    if (!v || !w || !bias || !out || C < 1 || B < 0 || P < 0 || B > 65535) return PSTD_EINVAL;
    if (B == 0 || P == 0) return PSTD_OK;
    k_proj<<<row_grid(B, P), 256, 0, (cudaStream_t)stream>>>(v, w, bias, out, C, P);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_proj_bwd(const float* dout, const float* w, float* dv, int64_t B, int C, int64_t P, void* stream) {
    if (!dout || !w || !dv || C < 1 || B < 0 || P < 0 || B * C > 65535) return PSTD_EINVAL;
    if (B == 0 || P == 0) return PSTD_OK;
    const int G = channel_group(B, C, P);
    k_proj_bwd<<<channel_grid(B, C, G, P), 256, 0, (cudaStream_t)stream>>>(dout, w, dv, C, G, P);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_chan_dot(const float* x, const float* y, int y_has_channels, float* g, int64_t B, int C, int64_t P,
                     void* stream) {
    if (!x || !g || C < 1 || B < 0 || P < 0 || C > 0x7fffffff) return PSTD_EINVAL;
    // eight CTAs per channel while the channels alone leave SMs idle and each
    // share is worth a CTA; whole samples to a CTA where a sample's points would
    // not give each thread four
    const int R = C <= 2 * 152 && B * P >= 8192 ? kRed : 1;
    const int by_sample = R > 1 && B >= R && P < 4 * 256 * R;
    return cuda_rc(launch_cluster(k_chan_dot, R, (unsigned)C * R, (cudaStream_t)stream, x, y, y_has_channels, g, B, C,
                                  P, R, by_sample));
}

int pstd_nn_sum_lead(const float* x, float* out, int64_t B, int64_t n, void* stream) {
    if (!x || !out || B < 1 || n < 0) return PSTD_EINVAL;
    if (n == 0) return PSTD_OK;
    // (the two cost the same at 100 to 400 columns per row)
    if (n / 256 >= B) k_sum_columns<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(x, out, B, n);
    else k_sum_lead<<<blocks_for(n * 32), 256, 0, (cudaStream_t)stream>>>(x, out, B, n);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_adam(float* w, const float* g, float* m, float* v, int64_t n, float lr, float beta1, float beta2,
                 float eps, int64_t step, void* stream) {
    if (!w || !g || !m || !v || step < 1) return PSTD_EINVAL;
    const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
    k_adam<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(w, g, m, v, n, lr, beta1, beta2, eps, c1, c2);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_mse(const float* out, const float* target, float* dout, float* loss, int64_t n, void* stream) {
    if (!out || !target || !loss || n < 1) return PSTD_EINVAL;
    return cuda_rc(launch_cluster(k_mse, kRed, kRed, (cudaStream_t)stream, out, target, dout, loss, n));
}

int pstd_nn_rel_err(const float* a, const float* ref, float* err, int64_t B, int64_t P, void* stream) {
    if (!a || !ref || !err || B < 1 || B > 0x7fffffff || P < 1) return PSTD_EINVAL;
    k_rel_err<<<(unsigned)B, 256, 0, (cudaStream_t)stream>>>(a, ref, err, P);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_round_bf16(const float* src, float* dst, int64_t n, void* stream) {
    if (!src || !dst || n < 0) return PSTD_EINVAL;
    k_round_bf16<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(src, dst, n);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_row_rms(const float* x, float* rms, int64_t B, int64_t P, void* stream) {
    if (!x || !rms || B < 1 || B > 0x7fffffff || P < 1) return PSTD_EINVAL;
    k_row_rms<<<(unsigned)B, 256, 0, (cudaStream_t)stream>>>(x, rms, P);
    return cuda_rc(cudaGetLastError());
}

int pstd_nn_row_scale(const float* x, const float* s, float* y, int64_t B, int64_t P, int mode, void* stream) {
    if (!x || !s || !y || B < 0 || B > 65535 || P < 0 || (mode != 0 && mode != 1)) return PSTD_EINVAL;
    if (B == 0 || P == 0) return PSTD_OK;
    k_row_scale<<<row_grid(B, P), 256, 0, (cudaStream_t)stream>>>(x, s, y, P, mode);
    return cuda_rc(cudaGetLastError());
}

// The first K wall-respecting modes of one axis (Table 2, transform T1 of the
// wall pair), from their mode functions on the stored pressure nodes x_j:
//   NN  cos(pi k j / N)        j = 0..N     (T1 = C1)
//   ND  cos(pi (k+1/2) j / N)  j = 0..N-1   (T1 = C3)
//   DN  sin(pi (k+1/2) j / N)  j = 1..N     (T1 = S3)
//   DD  sin(pi (k+1) j / N)    j = 1..N-1   (T1 = S1)
// The unnormalised forward transform is T[k][j] = 2 w_j phi_k(x_j), with
// w_j = 1/2 on a stored wall node and 1 elsewhere (trapezoid weights); its
// inverse (Eq. inverse_transforms, implied period M = 2N for every pair) is
// I[j][k] = (1/M) 2 v_k phi_k(x_j) with v_k = 1/2 for the wall-constant
// modes (k = 0 and k = N of NN) and 1 elsewhere.  Built in FP64, rounded once.
int pstd_sno_basis(int ncells, int bc_left, int bc_right, int K, float* T, float* I) {
    if (ncells < 2 || K < 1 || !T || !I) return PSTD_EINVAL;
    if ((bc_left != PSTD_NEUMANN && bc_left != PSTD_DIRICHLET) ||
        (bc_right != PSTD_NEUMANN && bc_right != PSTD_DIRICHLET))
        return PSTD_EINVAL;
    const int N = ncells;
    const int lo = bc_left == PSTD_DIRICHLET ? 1 : 0;
    const int hi = bc_right == PSTD_DIRICHLET ? N - 1 : N;
    const int lp = hi - lo + 1;
    if (K > lp) return PSTD_EINVAL;
    const bool cosine = bc_left == PSTD_NEUMANN;
    const double shift = bc_left == bc_right ? (cosine ? 0.0 : 1.0) : 0.5;
    const double M = 2.0 * N;
    for (int k = 0; k < K; ++k) {
        const double kap = M_PI * (k + shift) / N;
        const double vk = (cosine && bc_right == PSTD_NEUMANN && (k == 0 || k == N)) ? 0.5 : 1.0;
        for (int jj = 0; jj < lp; ++jj) {
            const int j = jj + lo;
            const double phi = cosine ? std::cos(kap * j) : std::sin(kap * j);
            const double wj = ((j == 0 && bc_left == PSTD_NEUMANN) || (j == N && bc_right == PSTD_NEUMANN)) ? 0.5 : 1.0;
            T[(size_t)k * lp + jj] = (float)(2.0 * wj * phi);
            I[(size_t)jj * K + k] = (float)(2.0 * vk * phi / M);
        }
    }
    return PSTD_OK;
}

}  // extern "C"
