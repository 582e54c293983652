// The enhancement strategy's network on sm_103a (RA-Haar-tSVD, Eq. 24-25):
// a plain fully connected network that refines the mean patch of every
// group, trained by the library's own kernels with residual learning.
//
// The mean patch enters in the image's transform coordinates (k_mean_coefs:
// Eq. 19 without the Haar factor, [S^(1), sqrt 2 Re S^(2), sqrt 2 Im S^(2)],
// orthonormal, canonical eigenvector phases), where it is sparse, in units of
// its noise level s = sigma / sqrt(K).  Input: g(c / s), g(x) = x / (1 + |x|
// / 16), then sigma / 255, zero-padded to a multiple of 16; two hidden layers
// of 128 ReLU units; a linear output of C x 64 values, the residual in noise
// units: refined = c + s x output.  FP32 weights and arithmetic.  The layers are GEMMs
// over a batch of groups (k_gemm: 64 x 64 output tiles, 16-deep slabs in
// shared memory, 8 x 4 outputs per thread); the weight gradients (k_wgrad)
// reduce over the batch with a split of the reduction and a fixed-order sum
// of the parts, so training is deterministic.
//
// Denoising (hts_denoise_ra): the mean patch of every group, its coordinates
// and features with the call's estimated sigma (k_group_features), the network,
// the refined patch back in pixels (k_refined_patch), and the refined patches go to the
// tensor-core filter, which drops each group's first Haar row and
// adds the refined mean to every member's estimate instead (the same as
// replacing that row by sqrt(K) times the refined mean's transform and not
// thresholding it).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "hts_internal.h"

namespace hts {
namespace {

constexpr int HID = 128;
constexpr int NL = 3;
constexpr float ADAM_B1 = 0.9f, ADAM_B2 = 0.999f, ADAM_EPS = 1e-8f;
constexpr int TM = 64, TN = 64, TK = 16;  // GEMM tile
constexpr float SAT = 16.f;                // saturation of the input compression
constexpr float K3F = 0.57735026918962576f;  // 1/sqrt(3)
constexpr float SQ2 = 1.41421356237309505f;

}  // namespace
}  // namespace hts

struct hts_fcn {
    int C = 1, K = 16, device = 0, nparams = 0, t = 0, din = 0, dout = 0;
    int off[3] = {}, nin[3] = {}, nout[3] = {};
    float *w = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    size_t cap = 0;                       // samples the activation buffers hold
    float *X = nullptr;                   // features [n][din]
    float *act[3] = {};                   // layer outputs [n][nout[l]]
    size_t cap_train = 0;                 // samples the training buffers hold
    float *dy[3] = {};                    // gradients of the layer outputs [n][nout[l]]
    double *lpart = nullptr;              // per-block loss parts
    size_t cap_part = 0;
    float *part = nullptr;                // split-reduction parts, each a parameter vector
    double *loss = nullptr;               // accumulated loss
};

namespace hts {
namespace {

#define HTS_TRY(expr)                \
    do {                             \
        hts_status _s = (expr);      \
        if (_s != HTS_OK) return _s; \
    } while (0)

hts_status cu(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return HTS_OK;
    char buf[160];
    snprintf(buf, sizeof(buf), "%s: %s", what, cudaGetErrorString(e));
    cudaGetLastError();
    return report(e == cudaErrorMemoryAllocation ? HTS_ENOMEM : HTS_ECUDA, buf);
}

// C(m, n) = sum_k A(m, k) B(n, k) over a 64 x 64 tile, FP32, k in ascending order.  Bound by FP32 issue at large
// M and by load latency at small M: a block of 128 threads holds 8 x 4 outputs per thread (3 shared-memory float4
// reads per 32 FMAs), and the next 16-deep slab travels global memory -> registers while the current one is
// multiplied (two shared buffers, one barrier per slab).  AK / BK: the operand is contiguous along k (A[m * lda +
// k]), else along m / n (A[k * lda + m]); either way a thread loads float4s along the contiguous axis, which is why
// the leading dimensions and N (for BK false) are multiples of 4.  Before (4 x 4 outputs, scalar loads that strode
// over rows in the forward pass, no overlap): 38 us per GEMM of a 4096-sample training step, now 16 (between events).
constexpr int GT = 128;      // threads
constexpr int SLD = TM + 4;  // row stride of a shared slab (float4-aligned, 2-way conflicts at worst)
enum { EPI_BIAS = 0, EPI_BIAS_RELU = 1, EPI_MASK = 2, EPI_LOSS = 3, EPI_PART = 4 };

struct GemmArgs {
    const float *A, *B;
    int lda, ldb, M, N, K;
    const float *bias;  // EPI_BIAS, EPI_BIAS_RELU, EPI_LOSS
    const float *mask;  // EPI_MASK: times (mask > 0)
    float *out;         // [M][N]; EPI_LOSS: the gradient of the loss; EPI_PART: this block's part
    // EPI_LOSS: target (clean - noisy) / (sigma * rsqrt_k), loss parts per block
    const float *noisy, *clean, *sigma;
    float rsqrt_k, total;
    double *lpart;
    float *bsum;  // EPI_PART: the part's bias gradients (sums of A over k), written by the blocks with n0 = 0
};

template <bool KC>
__device__ __forceinline__ void load_slab(const float *__restrict__ P, int ld, int r0, int R, int k0, int k1, int tid,
                                          float4 (&v)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int e = tid + i * GT;
        const int r = r0 + (KC ? e >> 2 : (e & 15) * 4), k = k0 + (KC ? (e & 3) * 4 : e >> 4);
        const bool in = r < R && k < k1;
        v[i] = in ? *reinterpret_cast<const float4 *>(P + (KC ? (size_t)r * ld + k : (size_t)k * ld + r))
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

template <bool KC>
__device__ __forceinline__ void store_slab(float (&S)[TK][SLD], int tid, const float4 (&v)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int e = tid + i * GT;
        if (KC) {
            const int r = e >> 2, k = (e & 3) * 4;
            S[k][r] = v[i].x;
            S[k + 1][r] = v[i].y;
            S[k + 2][r] = v[i].z;
            S[k + 3][r] = v[i].w;
        } else {
            *reinterpret_cast<float4 *>(&S[e >> 4][(e & 15) * 4]) = v[i];
        }
    }
}

template <bool AK, bool BK, int EPI>
__device__ __forceinline__ void gemm_tile(const GemmArgs &g, int m0, int n0, int k0, int k1, int lblock) {
    __shared__ __align__(16) float sA[2][TK][SLD], sB[2][TK][SLD];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[8][4] = {}, bs[8] = {};
    float4 va[2], vb[2];
    load_slab<AK>(g.A, g.lda, m0, g.M, k0, k1, tid, va);
    load_slab<BK>(g.B, g.ldb, n0, g.N, k0, k1, tid, vb);
    store_slab<AK>(sA[0], tid, va);
    store_slab<BK>(sB[0], tid, vb);
    __syncthreads();
    int cur = 0;
    for (int kb = k0; kb < k1; kb += TK) {
        const bool more = kb + TK < k1;
        if (more) {
            load_slab<AK>(g.A, g.lda, m0, g.M, kb + TK, k1, tid, va);
            load_slab<BK>(g.B, g.ldb, n0, g.N, kb + TK, k1, tid, vb);
        }
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            float a[8], b[4];
            *reinterpret_cast<float4 *>(a) = *reinterpret_cast<const float4 *>(&sA[cur][kk][ty * 8]);
            *reinterpret_cast<float4 *>(a + 4) = *reinterpret_cast<const float4 *>(&sA[cur][kk][ty * 8 + 4]);
            *reinterpret_cast<float4 *>(b) = *reinterpret_cast<const float4 *>(&sB[cur][kk][tx * 4]);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            if (EPI == EPI_PART && n0 == 0) {
#pragma unroll
                for (int i = 0; i < 8; ++i) bs[i] += a[i];
            }
        }
        if (more) {  // the other buffer: its last readers passed the barrier of the previous slab
            cur ^= 1;
            store_slab<AK>(sA[cur], tid, va);
            store_slab<BK>(sB[cur], tid, vb);
            __syncthreads();
        }
    }
    const int gn = n0 + tx * 4;
    float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((EPI == EPI_BIAS || EPI == EPI_BIAS_RELU || EPI == EPI_LOSS) && gn < g.N)
        bias = *reinterpret_cast<const float4 *>(g.bias + gn);
    double ls = 0.0;  // EPI_LOSS: sum of squared errors
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int gm = m0 + ty * 8 + i;
        if (gm >= g.M || gn >= g.N) continue;
        const size_t o = (size_t)gm * g.N + gn;
        float r[4] = {acc[i][0], acc[i][1], acc[i][2], acc[i][3]};
        if (EPI == EPI_BIAS || EPI == EPI_BIAS_RELU || EPI == EPI_LOSS) {
            r[0] += bias.x;
            r[1] += bias.y;
            r[2] += bias.z;
            r[3] += bias.w;
        }
        if (EPI == EPI_BIAS_RELU) {
#pragma unroll
            for (int j = 0; j < 4; ++j) r[j] = fmaxf(r[j], 0.f);
        }
        if (EPI == EPI_MASK) {
            const float4 mk = *reinterpret_cast<const float4 *>(g.mask + o);
            r[0] = mk.x > 0.f ? r[0] : 0.f;
            r[1] = mk.y > 0.f ? r[1] : 0.f;
            r[2] = mk.z > 0.f ? r[2] : 0.f;
            r[3] = mk.w > 0.f ? r[3] : 0.f;
        }
        if (EPI == EPI_LOSS) {  // the caller's tensors: 4-byte alignment only
            const float unit = g.sigma[gm] * g.rsqrt_k;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float e = r[j] - (g.clean[o + j] - g.noisy[o + j]) / unit;
                r[j] = 2.f * e / g.total;
                ls = fma((double)e, (double)e, ls);  // (the product is exact)
            }
        }
        *reinterpret_cast<float4 *>(g.out + o) = make_float4(r[0], r[1], r[2], r[3]);
    }
    if (EPI == EPI_PART && n0 == 0 && tx == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (m0 + ty * 8 + i < g.M) g.bsum[m0 + ty * 8 + i] = bs[i];
    }
    if (EPI == EPI_LOSS) {
        __shared__ double red[GT / 32];
        double s = ls;
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0) red[tid >> 5] = s;
        __syncthreads();
        if (tid == 0) g.lpart[lblock] = (red[0] + red[1]) + (red[2] + red[3]);
    }
}

// blockIdx = (n tile, m tile)
template <bool BK, int EPI>
__global__ void __launch_bounds__(GT) k_gemm(const GemmArgs g) {
    gemm_tile<true, BK, EPI>(g, blockIdx.y * TM, blockIdx.x * TN, 0, g.K, blockIdx.y * gridDim.x + blockIdx.x);
}

// The weight and bias gradients of every layer in one launch: dW[m][n] = sum over the samples of dY[k][m] X[k][n],
// db[m] = sum dY[k][m].  Block (t, z): tile t of the layers' tiles over samples [z kchunk, (z + 1) kchunk); its sums
// go to part z, which has the layout of the parameter vector, so that one pass adds the parts in z order.  Three
// launches of their own (and a bias kernel of one thread per column: 107 us each) left most SMs idle.
struct WgradArgs {
    GemmArgs l[NL];  // A = dY, B = the layer's input, out / bsum: the layer's place in part 0
    int tile0[NL + 1], nt[NL];
    int kchunk, nparams;
};
__global__ void __launch_bounds__(GT) k_wgrad(const __grid_constant__ WgradArgs w) {
    int l = 0;
    while ((int)blockIdx.x >= w.tile0[l + 1]) ++l;
    const int t = blockIdx.x - w.tile0[l];
    GemmArgs g = w.l[l];
    g.out += (size_t)blockIdx.y * w.nparams;
    g.bsum += (size_t)blockIdx.y * w.nparams;
    const int k0 = blockIdx.y * w.kchunk;
    gemm_tile<false, false, EPI_PART>(g, (t / w.nt[l]) * TM, (t % w.nt[l]) * TN, k0, min(g.K, k0 + w.kchunk), 0);
}

// grad[e] += sum over z of parts[z][e], in z order; the last block adds the loss parts (a fixed order: 32 strided
// chains, then a tree).
__global__ void __launch_bounds__(256) k_sum_parts(const float *__restrict__ parts, int nz, int ne,
                                                   float *__restrict__ grad, const double *__restrict__ lpart, int nl,
                                                   double total, double *loss) {
    if (blockIdx.x == gridDim.x - 1) {
        if (threadIdx.x < 32) {
            double t = 0.0;
            for (int b = threadIdx.x; b < nl; b += 32) t += lpart[b];
#pragma unroll
            for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (threadIdx.x == 0) *loss += t / total;
        }
        return;
    }
    const int e = blockIdx.x * 256 + threadIdx.x;
    if (e >= ne) return;
    float s = 0.f;
#pragma unroll 8
    for (int z = 0; z < nz; ++z) s += parts[(size_t)z * ne + e];
    grad[e] += s;
}

// Mean patch of group r (channel t, pixel (u, v)) over its K members, members in order.
__global__ void k_group_means(const float *__restrict__ img, int H, int W, int C, const int32_t *__restrict__ idx, int K,
                              int nref, float *__restrict__ means) {
    const long total = (long)nref * C * 64;
    const size_t HW = (size_t)H * W;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int r = (int)(i / (C * 64)), e = (int)(i - (long)r * C * 64);
        const int t = e >> 6, u = (e >> 3) & 7, v = e & 7;
        float s = 0.f;
        for (int k = 0; k < K; ++k) {
            const int pos = idx[(long)r * K + k];
            s += img[t * HW + (size_t)pos + (size_t)u * W + v];
        }
        means[i] = s / (float)K;
    }
}

// Features: g(coordinate / s) with s = sigma / sqrt(K), g(x) = x / (1 + |x| / SAT); sigma / 255
// (sigma[i * sstride]); zeros.
__global__ void k_features(const float *__restrict__ coords, const float *__restrict__ sigma, int sstride, int n,
                           int d, int din, float rsqrt_k, float *__restrict__ X) {
    const long total = (long)n * din;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int s = (int)(i / din), c = (int)(i - (long)s * din);
        const float sg = sigma[(long)s * sstride];
        float v = 0.f;
        if (c < d) {
            const float x = coords[(long)s * d + c] / (sg * rsqrt_k);
            v = x / (1.f + fabsf(x) * (1.f / SAT));
        } else if (c == d) {
            v = sg * (1.f / 255.f);
        }
        X[i] = v;
    }
}

__global__ void k_fcn_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                           float *__restrict__ v, int n, float lr, float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = ADAM_B1 * m[i] + (1.f - ADAM_B1) * gi;
        const float vi = ADAM_B2 * v[i] + (1.f - ADAM_B2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + ADAM_EPS);
    }
}

// refined[i] = coords[i] + s out[i], s = sigma[sample * sstride] / sqrt(K)
__global__ void k_refine(const float *__restrict__ coords, const float *__restrict__ out, const float *__restrict__ sigma,
                         int sstride, int d, float rsqrt_k, long total, float *__restrict__ refined) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x)
        refined[i] = coords[i] + sigma[(i / d) * sstride] * rsqrt_k * out[i];
}

// Column c of an 8x8 basis (element (r, c) at r * 8 + c) multiplied by the conjugate phase of its
// largest-magnitude entry (ties to the lower row): the entry becomes real positive.  Eigenvectors are
// defined up to that phase; the network's coordinates need one fixed choice.
__device__ void canon_column(float *re, float *im, int c) {
    int best = 0;
    float bm = -1.f;
    for (int r = 0; r < 8; ++r) {
        const float x = re[r * 8 + c], y = im ? im[r * 8 + c] : 0.f;
        const float m2 = x * x + y * y;
        if (m2 > bm) {
            bm = m2;
            best = r;
        }
    }
    const float x = re[best * 8 + c], y = im ? im[best * 8 + c] : 0.f;
    const float inv = bm > 0.f ? rsqrtf(bm) : 1.f;
    const float pr = x * inv, pi = y * inv;  // phase; multiply the column by its conjugate
    for (int r = 0; r < 8; ++r) {
        const float a = re[r * 8 + c], b = im ? im[r * 8 + c] : 0.f;
        re[r * 8 + c] = a * pr + b * pi;
        if (im) im[r * 8 + c] = b * pr - a * pi;
    }
}

// Basis slices of the FP32 device copy ([j][U/V][8][8][re/im]) in shared memory, columns in the
// canonical phase (canon_column).
struct MeanBasis {
    float u0[64], v0[64], u1r[64], u1i[64], v1r[64], v1i[64];
};
template <int C>
__device__ void load_bases(const float *__restrict__ b32, MeanBasis &b) {
    const int t = threadIdx.x;
    if (t < 64) {
        b.u0[t] = b32[(0 * 64 + t) * 2];
        b.v0[t] = b32[(1 * 64 + t) * 2];
        if (C == 3) {
            b.u1r[t] = b32[(2 * 64 + t) * 2];
            b.u1i[t] = b32[(2 * 64 + t) * 2 + 1];
            b.v1r[t] = b32[(3 * 64 + t) * 2];
            b.v1i[t] = b32[(3 * 64 + t) * 2 + 1];
        }
    }
    __syncthreads();
    if (t < 8) canon_column(b.u0, nullptr, t);
    else if (t < 16) canon_column(b.v0, nullptr, t - 8);
    else if (C == 3 && t < 24) canon_column(b.u1r, b.u1i, t - 16);
    else if (C == 3 && t < 32) canon_column(b.v1r, b.v1i, t - 24);
    __syncthreads();
}

// The transforms below take PB patches at a time per block of 64 PB threads, thread t of a patch = pixel / coefficient
// (t >> 3, t & 7), and a block goes on to further patches, so that the bases are read and their phases fixed once.
// Every thread of the block calls them (barriers).
constexpr int PB = 4;
struct PatchBuf {
    float a0[64], ar[64], ai[64], b0[64], br[64], bi[64];
};

// Coordinates of the patch whose pixel values thread t holds in p (R, G, B or gray): the DFT along the channels,
// T = Phat V, S = U^H T (Eq. 19 without the Haar factor); o = [S^(1) | sqrt 2 Re S^(2) | sqrt 2 Im S^(2)] (orthonormal).
template <int C>
__device__ __forceinline__ void patch_forward(const MeanBasis &b, PatchBuf &w, int t, const float (&p)[C],
                                              float (&o)[C]) {
    __syncthreads();  // the buffer's last readers are done
    if (C == 1) {
        w.a0[t] = p[0];
    } else {
        const float R = p[0], G = p[C - 2], B = p[C - 1];
        w.a0[t] = ((R + G) + B) * K3F;
        w.ar[t] = (R - 0.5f * (G + B)) * K3F;
        w.ai[t] = (B - G) * 0.5f;
    }
    __syncthreads();
    const int hi = t >> 3, lo = t & 7;
    {  // T[i][b] = sum_j Phat[i][j] V[j][b], thread (i, b) = (hi, lo)
        float a0 = 0.f, ar = 0.f, ai = 0.f;
        for (int j = 0; j < 8; ++j) {
            a0 = fmaf(w.a0[hi * 8 + j], b.v0[j * 8 + lo], a0);
            if (C == 3) {
                const float xr = w.ar[hi * 8 + j], xi = w.ai[hi * 8 + j], yr = b.v1r[j * 8 + lo], yi = b.v1i[j * 8 + lo];
                ar = fmaf(xr, yr, fmaf(-xi, yi, ar));
                ai = fmaf(xr, yi, fmaf(xi, yr, ai));
            }
        }
        w.b0[t] = a0;
        w.br[t] = ar;
        w.bi[t] = ai;
    }
    __syncthreads();
    {  // S[a][b] = sum_i conj(U[i][a]) T[i][b], thread (a, b) = (hi, lo)
        float s0 = 0.f, sr = 0.f, si = 0.f;
        for (int i = 0; i < 8; ++i) {
            s0 = fmaf(b.u0[i * 8 + hi], w.b0[i * 8 + lo], s0);
            if (C == 3) {
                const float ur = b.u1r[i * 8 + hi], ui = b.u1i[i * 8 + hi], xr = w.br[i * 8 + lo], xi = w.bi[i * 8 + lo];
                sr = fmaf(ur, xr, fmaf(ui, xi, sr));
                si = fmaf(ur, xi, fmaf(-ui, xr, si));
            }
        }
        o[0] = s0;
        if (C == 3) {
            o[C - 2] = SQ2 * sr;
            o[C - 1] = SQ2 * si;
        }
    }
}

// The inverse: Phat = U S V^H per slice, then the inverse DFT along the channels.
template <int C>
__device__ __forceinline__ void patch_inverse(const MeanBasis &b, PatchBuf &w, int t, const float (&c)[C],
                                              float (&o)[C]) {
    __syncthreads();
    w.a0[t] = c[0];
    if (C == 3) {
        w.ar[t] = c[C - 2] * (1.f / SQ2);
        w.ai[t] = c[C - 1] * (1.f / SQ2);
    }
    __syncthreads();
    const int hi = t >> 3, lo = t & 7;
    {  // Q[a][j] = sum_b S[a][b] conj(V[j][b]), thread (a, j) = (hi, lo)
        float a0 = 0.f, ar = 0.f, ai = 0.f;
        for (int k = 0; k < 8; ++k) {
            a0 = fmaf(w.a0[hi * 8 + k], b.v0[lo * 8 + k], a0);
            if (C == 3) {
                const float xr = w.ar[hi * 8 + k], xi = w.ai[hi * 8 + k], yr = b.v1r[lo * 8 + k], yi = b.v1i[lo * 8 + k];
                ar = fmaf(xr, yr, fmaf(xi, yi, ar));
                ai = fmaf(xi, yr, fmaf(-xr, yi, ai));
            }
        }
        w.b0[t] = a0;
        w.br[t] = ar;
        w.bi[t] = ai;
    }
    __syncthreads();
    {  // Phat[i][j] = sum_a U[i][a] Q[a][j], thread (i, j) = (hi, lo); then the inverse channel DFT
        float f0 = 0.f, fr = 0.f, fi = 0.f;
        for (int a = 0; a < 8; ++a) {
            f0 = fmaf(b.u0[hi * 8 + a], w.b0[a * 8 + lo], f0);
            if (C == 3) {
                const float ur = b.u1r[hi * 8 + a], ui = b.u1i[hi * 8 + a], xr = w.br[a * 8 + lo], xi = w.bi[a * 8 + lo];
                fr = fmaf(ur, xr, fmaf(-ui, xi, fr));
                fi = fmaf(ur, xi, fmaf(ui, xr, fi));
            }
        }
        if (C == 1) {
            o[0] = f0;
        } else {
            o[0] = (f0 + 2.f * fr) * K3F;
            o[C - 2] = (f0 - fr - 1.7320508075688772f * fi) * K3F;
            o[C - 1] = (f0 - fr + 1.7320508075688772f * fi) * K3F;
        }
    }
}

// Patches (n x C x 64) to coordinates, or back (INV).
template <int C, bool INV>
__global__ void __launch_bounds__(64 * PB) k_mean_coefs(const float *__restrict__ in, int n,
                                                        const float *__restrict__ b32, float *__restrict__ out) {
    __shared__ MeanBasis b;
    __shared__ PatchBuf w[PB];
    const int t = threadIdx.x & 63, sub = threadIdx.x >> 6;
    load_bases<C>(b32, b);
    for (int r0 = blockIdx.x * PB; r0 < n; r0 += gridDim.x * PB) {
        const int r = r0 + sub;
        const float *src = in + (size_t)min(r, n - 1) * C * 64 + t;
        float x[C], y[C];
#pragma unroll
        for (int c = 0; c < C; ++c) x[c] = src[64 * c];
        if (INV) patch_inverse<C>(b, w[sub], t, x, y);
        else patch_forward<C>(b, w[sub], t, x, y);
        if (r < n) {
#pragma unroll
            for (int c = 0; c < C; ++c) out[(size_t)r * C * 64 + 64 * c + t] = y[c];
        }
    }
}

// The network's input from the groups in one pass: the mean patch of every group (as k_group_means), its coordinates
// (kept for the residual) and the features (as k_features) with the call's sigma.  Bound by L2 (K pixels read per value
// kept); as kernels of their own the three read and wrote the values between them and fixed the bases' phases per
// patch: 512 x 512 x 3, 81 us (between events), now 44.
template <int C>
__global__ void __launch_bounds__(64 * PB) k_group_features(const float *__restrict__ img, int H, int W,
                                                            const int32_t *__restrict__ idx, int K, int nref,
                                                            const float *__restrict__ b32, const DevState *st, int din,
                                                            float rsqrt_k, float *__restrict__ coords,
                                                            float *__restrict__ X) {
    __shared__ MeanBasis b;
    __shared__ PatchBuf w[PB];
    const int t = threadIdx.x & 63, sub = threadIdx.x >> 6;
    const size_t HW = (size_t)H * W, at = (size_t)(t >> 3) * W + (t & 7);
    const float sg = (float)st->sigma_hat;
    load_bases<C>(b32, b);
    for (int r0 = blockIdx.x * PB; r0 < nref; r0 += gridDim.x * PB) {
        const int r = r0 + sub;
        const int32_t *grp = idx + (size_t)min(r, nref - 1) * K;
        float m[C], o[C];
#pragma unroll
        for (int c = 0; c < C; ++c) m[c] = 0.f;
#pragma unroll 8
        for (int k = 0; k < K; ++k) {
            const float *src = img + (size_t)grp[k] + at;
#pragma unroll
            for (int c = 0; c < C; ++c) m[c] += src[c * HW];
        }
#pragma unroll
        for (int c = 0; c < C; ++c) m[c] = m[c] / (float)K;
        patch_forward<C>(b, w[sub], t, m, o);
        if (r < nref) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                coords[(size_t)r * C * 64 + 64 * c + t] = o[c];
                const float x = o[c] / (sg * rsqrt_k);
                X[(size_t)r * din + 64 * c + t] = x / (1.f + fabsf(x) * (1.f / SAT));
            }
            if (t < din - C * 64) X[(size_t)r * din + C * 64 + t] = t == 0 ? sg * (1.f / 255.f) : 0.f;
        }
    }
}

// The refined patch of every group in pixels: coordinates plus s times the network's output, then patch_inverse.
template <int C>
__global__ void __launch_bounds__(64 * PB) k_refined_patch(const float *__restrict__ coords,
                                                           const float *__restrict__ res, int n,
                                                           const float *__restrict__ b32, const DevState *st,
                                                           float rsqrt_k, float *__restrict__ patches) {
    __shared__ MeanBasis b;
    __shared__ PatchBuf w[PB];
    const int t = threadIdx.x & 63, sub = threadIdx.x >> 6;
    const float sg = (float)st->sigma_hat;
    load_bases<C>(b32, b);
    for (int r0 = blockIdx.x * PB; r0 < n; r0 += gridDim.x * PB) {
        const int r = r0 + sub;
        const size_t o = (size_t)min(r, n - 1) * C * 64 + t;
        float x[C], y[C];
#pragma unroll
        for (int c = 0; c < C; ++c) x[c] = coords[o + 64 * c] + sg * rsqrt_k * res[o + 64 * c];
        patch_inverse<C>(b, w[sub], t, x, y);
        if (r < n) {
#pragma unroll
            for (int c = 0; c < C; ++c) patches[o + 64 * c] = y[c];
        }
    }
}

void layout(hts_fcn *f) {
    f->din = (f->C * 64 + 1 + 15) / 16 * 16;
    f->dout = f->C * 64;
    const int ins[NL] = {f->din, HID, HID}, outs[NL] = {HID, HID, f->dout};
    int o = 0;
    for (int l = 0; l < NL; ++l) {
        f->nin[l] = ins[l];
        f->nout[l] = outs[l];
        f->off[l] = o;
        o += ins[l] * outs[l] + outs[l];
    }
    f->nparams = o;
}

hts_status ensure(hts_fcn *f, size_t n) {
    if (n > f->cap) {
        cudaFree(f->X);
        for (float *&p : f->act) {
            cudaFree(p);
            p = nullptr;
        }
        f->X = nullptr;
        f->cap = 0;
        HTS_TRY(cu(dev_malloc(&f->X, n * f->din * sizeof(float)), "cudaMalloc(fcn)"));
        for (int l = 0; l < NL; ++l) HTS_TRY(cu(dev_malloc(&f->act[l], n * f->nout[l] * sizeof(float)), "cudaMalloc(fcn)"));
        f->cap = n;
    }
    return HTS_OK;
}

// The buffers only training needs, for n samples in `nz` parts.
hts_status ensure_train(hts_fcn *f, size_t n, int nz) {
    if (n > f->cap_train) {
        for (float *&p : f->dy) {
            cudaFree(p);
            p = nullptr;
        }
        cudaFree(f->lpart);
        f->lpart = nullptr;
        f->cap_train = 0;
        for (int l = 0; l < NL; ++l) HTS_TRY(cu(dev_malloc(&f->dy[l], n * f->nout[l] * sizeof(float)), "cudaMalloc(fcn)"));
        const size_t blocks = ((n + TM - 1) / TM) * ((f->dout + TN - 1) / TN);
        HTS_TRY(cu(dev_malloc(&f->lpart, blocks * sizeof(double)), "cudaMalloc(fcn)"));
        f->cap_train = n;
    }
    const size_t need = (size_t)nz * f->nparams;
    if (need > f->cap_part) {
        cudaFree(f->part);
        f->part = nullptr;
        f->cap_part = 0;
        HTS_TRY(cu(dev_malloc(&f->part, need * sizeof(float)), "cudaMalloc(fcn)"));
        f->cap_part = need;
    }
    return HTS_OK;
}

int nsm() {
    int dev = 0, n = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

// Blocks of the patch kernels: eight per SM, as many as are resident.
int patch_blocks(int n) { return std::max(1, std::min((n + PB - 1) / PB, 8 * nsm())); }

template <bool BK, int EPI>
hts_status gemm(const GemmArgs &g, cudaStream_t s) {
    const dim3 grid((g.N + TN - 1) / TN, (g.M + TM - 1) / TM);
    {
        KTimer kt("k_fcn_gemm", s);
        k_gemm<BK, EPI><<<grid, GT, 0, s>>>(g);
    }
    return check_launch("k_fcn_gemm");
}

// Forward of n samples whose features are in f->X; output in f->act[2], or, with a target (noisy, clean, sigma of
// each), the loss gradient in f->dy[2] and the loss parts in f->lpart.
hts_status forward(hts_fcn *f, int n, cudaStream_t s, const float *noisy = nullptr, const float *clean = nullptr,
                   const float *sigma = nullptr) {
    const float *in = f->X;
    for (int l = 0; l < NL; ++l) {
        GemmArgs g{};
        g.A = in;
        g.B = f->w + f->off[l];
        g.lda = g.ldb = g.K = f->nin[l];
        g.M = n;
        g.N = f->nout[l];
        g.bias = f->w + f->off[l] + f->nout[l] * f->nin[l];
        g.out = f->act[l];
        if (l < NL - 1) {
            HTS_TRY((gemm<true, EPI_BIAS_RELU>(g, s)));
        } else if (!noisy) {
            HTS_TRY((gemm<true, EPI_BIAS>(g, s)));
        } else {
            g.out = f->dy[l];
            g.noisy = noisy;
            g.clean = clean;
            g.sigma = sigma;
            g.rsqrt_k = 1.f / std::sqrt((float)f->K);
            g.total = (float)((long)n * f->dout);
            g.lpart = f->lpart;
            HTS_TRY((gemm<true, EPI_LOSS>(g, s)));
        }
        in = f->act[l];
    }
    return HTS_OK;
}

// Tiles of layer l's weight gradient.
int wgrad_tiles(const hts_fcn *f, int l) { return (f->nout[l] + TM - 1) / TM * ((f->nin[l] + TN - 1) / TN); }

// Samples per part of the weight gradients: about four blocks per SM over all the layers' tiles, and at least 64.
int wgrad_chunk(const hts_fcn *f, int n) {
    long tiles = 0;
    for (int l = 0; l < NL; ++l) tiles += wgrad_tiles(f, l);
    const long c = ((long)n * tiles + 4 * nsm() - 1) / (4 * nsm());
    return (int)((std::max(c, 64l) + TK - 1) / TK * TK);
}

hts_status features(hts_fcn *f, const float *means, const float *sigma, int sstride, int n, cudaStream_t s) {
    const long total = (long)n * f->din;
    {
        KTimer kt("k_fcn_features", s);
        k_features<<<(unsigned)std::min<long>((total + 255) / 256, 4096), 256, 0, s>>>(
            means, sigma, sstride, n, f->dout, f->din, 1.f / std::sqrt((float)f->K), f->X);
    }
    return check_launch("k_fcn_features");
}

hts_status upload(hts_fcn *f, const float *host) {
    HTS_TRY(cu(cudaMemcpy(f->w, host, f->nparams * sizeof(float), cudaMemcpyHostToDevice), "cudaMemcpy"));
    for (float *p : {f->grad, f->m, f->v}) HTS_TRY(cu(cudaMemset(p, 0, f->nparams * sizeof(float)), "cudaMemset"));
    f->t = 0;
    return HTS_OK;
}

void free_fcn(hts_fcn *f) {
    if (!f) return;
    for (float *p : {f->w, f->grad, f->m, f->v, f->X, f->part}) cudaFree(p);
    for (float *p : f->act) cudaFree(p);
    for (float *p : f->dy) cudaFree(p);
    cudaFree(f->loss);
    cudaFree(f->lpart);
    delete f;
}

uint64_t splitmix64(uint64_t &x) {
    uint64_t z = (x += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

}  // namespace

hts_status launch_group_means(const float *img, const Geom &g, const int32_t *idx, float *means, cudaStream_t s) {
    const long total = (long)g.nref * g.C * 64;
    {
        KTimer kt("k_group_means", s);
        k_group_means<<<(unsigned)std::min<long>((total + 255) / 256, 8192), 256, 0, s>>>(img, g.H, g.W, g.C, idx,
                                                                                          g.K, g.nref, means);
    }
    return check_launch("k_group_means");
}

hts_status launch_mean_transform(const float *in, int n, int C, const float *b32, bool inverse, float *out,
                                 cudaStream_t s) {
    if (n == 0) return HTS_OK;
    const int nb = patch_blocks(n);
    KTimer kt(inverse ? "k_coefs_to_patch" : "k_mean_coefs", s);
    if (C == 1) {
        if (inverse) k_mean_coefs<1, true><<<nb, 64 * PB, 0, s>>>(in, n, b32, out);
        else k_mean_coefs<1, false><<<nb, 64 * PB, 0, s>>>(in, n, b32, out);
    } else {
        if (inverse) k_mean_coefs<3, true><<<nb, 64 * PB, 0, s>>>(in, n, b32, out);
        else k_mean_coefs<3, false><<<nb, 64 * PB, 0, s>>>(in, n, b32, out);
    }
    return check_launch(inverse ? "k_coefs_to_patch" : "k_mean_coefs");
}

// Refined mean patches (pixels) of the groups idx, with the call's sigma from the state, in out (N_ref x C x 64);
// coords: scratch of the same size.
hts_status fcn_refine_groups(hts_fcn *f, const float *img, const Geom &g, const int32_t *idx, const DevState *st,
                             const float *b32, float *coords, float *out, cudaStream_t s) {
    const int n = g.nref, nb = patch_blocks(n);
    const float rk = 1.f / std::sqrt((float)f->K);
    HTS_TRY(ensure(f, n));
    {
        KTimer kt("k_group_features", s);
        if (f->C == 1)
            k_group_features<1><<<nb, 64 * PB, 0, s>>>(img, g.H, g.W, idx, g.K, n, b32, st, f->din, rk, coords, f->X);
        else
            k_group_features<3><<<nb, 64 * PB, 0, s>>>(img, g.H, g.W, idx, g.K, n, b32, st, f->din, rk, coords, f->X);
    }
    HTS_TRY(check_launch("k_group_features"));
    HTS_TRY(forward(f, n, s));
    {
        KTimer kt("k_refined_patch", s);
        if (f->C == 1) k_refined_patch<1><<<nb, 64 * PB, 0, s>>>(coords, f->act[NL - 1], n, b32, st, rk, out);
        else k_refined_patch<3><<<nb, 64 * PB, 0, s>>>(coords, f->act[NL - 1], n, b32, st, rk, out);
    }
    return check_launch("k_refined_patch");
}

}  // namespace hts

using namespace hts;

extern "C" int hts_fcn_num_params(int C) {
    if (C != 1 && C != 3) return 0;
    hts_fcn f;
    f.C = C;
    layout(&f);
    return f.nparams;
}

extern "C" int hts_fcn_channels(const hts_fcn *f) { return f ? f->C : 0; }

extern "C" int hts_fcn_group_size(const hts_fcn *f) { return f ? f->K : 0; }

extern "C" hts_status hts_fcn_create(int C, int K, uint64_t seed, hts_fcn **out) {
    if (!out) return report(HTS_EINVAL, "NULL pointer");
    if (C != 1 && C != 3) return report(HTS_EINVAL, "C must be 1 or 3");
    if (K < 2 || K > 32 || (K & (K - 1))) return report(HTS_EINVAL, "K must be a power of 2 in 2..32");
    hts_fcn *f = new hts_fcn();
    f->C = C;
    f->K = K;
    layout(f);
    hts_status st = cu(cudaGetDevice(&f->device), "cudaGetDevice");
    for (float **p : {&f->w, &f->grad, &f->m, &f->v})
        if (st == HTS_OK) st = cu(dev_malloc(p, f->nparams * sizeof(float)), "cudaMalloc(fcn)");
    if (st == HTS_OK) st = cu(dev_malloc(&f->loss, sizeof(double)), "cudaMalloc(fcn)");
    if (st == HTS_OK) st = cu(cudaMemset(f->loss, 0, sizeof(double)), "cudaMemset");
    if (st != HTS_OK) {
        free_fcn(f);
        return st;
    }
    // He initialisation of the hidden layers, the output layer 0.1x smaller (starts near the identity
    // refinement), biases zero; Box-Muller on a splitmix64 stream
    std::vector<float> h(f->nparams, 0.f);
    uint64_t x = seed;
    for (int l = 0; l < NL; ++l) {
        const double sd = std::sqrt(2.0 / f->nin[l]) * (l == NL - 1 ? 0.1 : 1.0);
        for (int i = 0; i < f->nout[l] * f->nin[l]; ++i) {
            const double u1 = ((splitmix64(x) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
            const double u2 = ((splitmix64(x) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
            h[f->off[l] + i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
    }
    st = upload(f, h.data());
    if (st != HTS_OK) {
        free_fcn(f);
        return st;
    }
    *out = f;
    return HTS_OK;
}

extern "C" hts_status hts_fcn_free(hts_fcn *f) {
    free_fcn(f);
    return HTS_OK;
}

extern "C" hts_status hts_fcn_get_params(const hts_fcn *f, float *host) {
    if (!f || !host) return report(HTS_EINVAL, "NULL pointer");
    return cu(cudaMemcpy(host, f->w, f->nparams * sizeof(float), cudaMemcpyDeviceToHost), "cudaMemcpy");
}

extern "C" hts_status hts_fcn_set_params(hts_fcn *f, const float *host) {
    if (!f || !host) return report(HTS_EINVAL, "NULL pointer");
    return upload(f, host);
}

extern "C" hts_status hts_group_means(const float *img, int H, int W, int C, const hts_params *p, const int32_t *idx,
                                      float *means, void *stream) {
    Geom g;
    HTS_TRY(validate(H, W, C, p, &g));
    if (!img || !idx || !means) return report(HTS_EINVAL, "NULL pointer");
    return launch_group_means(img, g, idx, means, static_cast<cudaStream_t>(stream));
}

extern "C" hts_status hts_mean_coefs(const float *in, int n, int C, const hts_basis *basis, int inverse, float *out,
                                     void *stream) {
    if (!in || !basis || !out) return report(HTS_EINVAL, "NULL pointer");
    if (n < 0) return report(HTS_EINVAL, "n < 0");
    if (C != basis->C) return report(HTS_EINVAL, "basis built for another channel count");
    return launch_mean_transform(in, n, C, basis->b32, inverse != 0, out, static_cast<cudaStream_t>(stream));
}

extern "C" hts_status hts_fcn_refine(hts_fcn *f, const float *means, const float *sigma, int n, float *refined,
                                     void *stream) {
    if (!f || !means || !sigma || !refined) return report(HTS_EINVAL, "NULL pointer");
    if (n < 0) return report(HTS_EINVAL, "n < 0");
    if (n == 0) return HTS_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    HTS_TRY(ensure(f, n));
    HTS_TRY(features(f, means, sigma, 1, n, s));
    HTS_TRY(forward(f, n, s));
    const long total = (long)n * f->dout;
    {
        KTimer kt("k_fcn_refine", s);
        k_refine<<<(unsigned)std::min<long>((total + 255) / 256, 8192), 256, 0, s>>>(
            means, f->act[NL - 1], sigma, 1, f->dout, 1.f / std::sqrt((float)f->K), total, refined);
    }
    return check_launch("k_fcn_refine");
}

extern "C" hts_status hts_fcn_zero_grad(hts_fcn *f, void *stream) {
    if (!f) return report(HTS_EINVAL, "NULL pointer");
    return cu(cudaMemsetAsync(f->grad, 0, f->nparams * sizeof(float), static_cast<cudaStream_t>(stream)),
              "cudaMemsetAsync");
}

extern "C" hts_status hts_fcn_accumulate_grad(hts_fcn *f, const float *noisy_means, const float *clean_means,
                                              const float *sigma, int n, void *stream) {
    if (!f || !noisy_means || !clean_means || !sigma) return report(HTS_EINVAL, "NULL pointer");
    if (n <= 0) return report(HTS_EINVAL, "n must be > 0");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    HTS_TRY(ensure(f, n));
    HTS_TRY(features(f, noisy_means, sigma, 1, n, s));
    const int kchunk = wgrad_chunk(f, n), nz = (n + kchunk - 1) / kchunk;
    HTS_TRY(ensure_train(f, n, nz));
    HTS_TRY(forward(f, n, s, noisy_means, clean_means, sigma));
    // dX = (dY W) * (X > 0), the ReLU of the layer below
    for (int l = NL - 1; l > 0; --l) {
        GemmArgs g{};
        g.A = f->dy[l];
        g.B = f->w + f->off[l];
        g.lda = g.K = f->nout[l];
        g.ldb = g.N = f->nin[l];
        g.M = n;
        g.mask = f->act[l - 1];
        g.out = f->dy[l - 1];
        HTS_TRY((gemm<false, EPI_MASK>(g, s)));
    }
    WgradArgs w{};
    w.kchunk = kchunk;
    w.nparams = f->nparams;
    for (int l = 0; l < NL; ++l) {
        GemmArgs &g = w.l[l];
        g.A = f->dy[l];
        g.B = l == 0 ? f->X : f->act[l - 1];
        g.lda = g.M = f->nout[l];
        g.ldb = g.N = f->nin[l];
        g.K = n;
        g.out = f->part + f->off[l];
        g.bsum = g.out + f->nout[l] * f->nin[l];
        w.nt[l] = (f->nin[l] + TN - 1) / TN;
        w.tile0[l + 1] = w.tile0[l] + wgrad_tiles(f, l);
    }
    {
        KTimer kt("k_fcn_wgrad", s);
        k_wgrad<<<dim3(w.tile0[NL], nz), GT, 0, s>>>(w);
    }
    HTS_TRY(check_launch("k_fcn_wgrad"));
    {
        KTimer kt("k_sum_parts", s);
        k_sum_parts<<<(f->nparams + 255) / 256 + 1, 256, 0, s>>>(
            f->part, nz, f->nparams, f->grad, f->lpart, ((n + TM - 1) / TM) * ((f->dout + TN - 1) / TN),
            (double)n * f->dout, f->loss);
    }
    return check_launch("k_sum_parts");
}

extern "C" hts_status hts_fcn_take_loss(hts_fcn *f, double *loss_sum, void *stream) {
    if (!f || !loss_sum) return report(HTS_EINVAL, "NULL pointer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    HTS_TRY(cu(cudaMemcpyAsync(loss_sum, f->loss, sizeof(double), cudaMemcpyDeviceToHost, s), "cudaMemcpyAsync"));
    HTS_TRY(cu(cudaMemsetAsync(f->loss, 0, sizeof(double), s), "cudaMemsetAsync"));
    return cu(cudaStreamSynchronize(s), "cudaStreamSynchronize");
}

extern "C" hts_status hts_fcn_get_grad(const hts_fcn *f, float *host, void *stream) {
    if (!f || !host) return report(HTS_EINVAL, "NULL pointer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    HTS_TRY(cu(cudaMemcpyAsync(host, f->grad, f->nparams * sizeof(float), cudaMemcpyDeviceToHost, s),
               "cudaMemcpyAsync"));
    return cu(cudaStreamSynchronize(s), "cudaStreamSynchronize");
}

extern "C" hts_status hts_fcn_adam_step(hts_fcn *f, float lr, void *stream) {
    if (!f) return report(HTS_EINVAL, "NULL pointer");
    if (!(lr > 0.f) || !std::isfinite(lr)) return report(HTS_EINVAL, "lr must be > 0");
    f->t += 1;
    const float c1 = (float)(1.0 / (1.0 - std::pow((double)ADAM_B1, f->t)));
    const float c2 = (float)(1.0 / (1.0 - std::pow((double)ADAM_B2, f->t)));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    {
        KTimer kt("k_fcn_adam", s);
        k_fcn_adam<<<(f->nparams + 255) / 256, 256, 0, s>>>(f->w, f->grad, f->m, f->v, f->nparams, lr, c1, c2);
    }
    return check_launch("k_fcn_adam");
}
