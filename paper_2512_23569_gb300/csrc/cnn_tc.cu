// Tensor-core forward pass of the learned noise-level network (the
// convolutional estimate of the adaptive variant, Sec. III-C), used when
// denoising.
//
// A 3x3 convolution with zero padding is an implicit GEMM: for every tap
// (ky, kx), out[p][n] += sum_c in[p + (ky - 1, kx - 1)][c] w[n][c][ky][kx].
// A block takes a strip of 16 x 64 (16) output pixels and stages its input with a
// one-pixel halo in shared memory as planes of 8 channels: entry (g, py, px)
// is the 16-byte vector of channels 8g .. 8g + 7 of one pixel.  Eight 16 x 8
// pixel tiles of the strip are the MMA's M = 128 rows (tile row i = 8
// consecutive pixels of output row i, one core matrix), so the A operand of
// tap (ky, kx) is the staged region itself, its descriptor starting ky rows
// and kx pixels further on: core matrices one staged row apart along M and
// one channel plane apart along K.  No im2col copy is made.  B holds the
// layer's FP16 weights per tap (N = 32 output channels, or 16 of which one
// is used for the last layer); each tile accumulates 9 taps x (input
// channels / 16) MMAs of kind::f16 in its own 32 (16) tensor-memory columns.
// The epilogue reads a tile row per thread (tcgen05.ld), adds the bias,
// applies ReLU and writes FP16 planes for the next layer, or the FP32 log
// sigma map after the last layer.
//
// Layers: 0: image / 255 (rounded to FP16, channels padded to 16) -> 32;
// 1..3: 32 -> 32; 4: 32 -> 1.  Every mbarrier wait is bounded; a wait that
// gives up sets the network's error flag, the block waits (bounded) for its
// MMAs and releases its tensor memory, and the map is then filled with NaN
// so that the learned-map check falls back to the estimate.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "cnn_internal.h"
#include "hts_internal.h"
#include "tc_ptx.h"

namespace hts {
namespace {

constexpr int SY = 16;                   // output rows of a strip
constexpr int PY = SY + 2;               // staged rows (halo of one pixel)
constexpr int SX = 64, PX = SX + 2;      // output and staged columns of the weight gradient's strips
constexpr int NTH = 256;                 // 8 warps; warp w reads tensor-memory lanes 32 (w % 4) .. + 31
constexpr long long SPIN = 1ll << 22;
// At least this much shared memory per block: at most two blocks per SM, so
// their tensor memory (at most 2 x 256 columns) is always free to allocate.
constexpr size_t MIN_SMEM = 80 * 1024;

// Epilogues: bias and ReLU to FP16 planes (forward, hidden layers), column 0 plus bias to the FP32 map
// (forward, last layer), or the accumulated value times the ReLU mask of a stored activation to FP16 planes
// (backward: the gradient of a layer's input, zero where the activation is zero).
constexpr int EPI_RELU = 0, EPI_MAP = 1, EPI_MASK = 2;

// The layer's weights B[tap][g][n][k] = w[n][8 g + k][tap], laid out so in global memory, and its biases, into shared
// memory (gathering them from [n][ci][tap] took 2-byte loads with four divisions each: half of a small layer's time).
template <int CING, int NOUT, int EPI>
__device__ __forceinline__ void stage_weights(const __half *wp, const __half *wbias, int cout, __half *sB,
                                              float *sBias, int tid) {
    constexpr int NV = 9 * CING * NOUT, NE = (NV + NTH - 1) / NTH;
    uint4 v[NE];  // every load in flight before the first store
#pragma unroll
    for (int i = 0; i < NE; ++i)
        if (tid + i * NTH < NV) v[i] = reinterpret_cast<const uint4 *>(wp)[tid + i * NTH];
#pragma unroll
    for (int i = 0; i < NE; ++i)
        if (tid + i * NTH < NV) reinterpret_cast<uint4 *>(sB)[tid + i * NTH] = v[i];
    if (EPI != EPI_MASK)
        for (int n = tid; n < NOUT; n += NTH) sBias[n] = n < cout ? __half2float(wbias[n]) : 0.f;
}

// One tile row of the epilogue: thread m of lane quarter q holds output pixel (oy, ox); r: its NOUT
// accumulator columns (read by the caller).
template <int NOUT, int EPI>
__device__ __forceinline__ void epilogue_store(const uint32_t *r, const float *sBias, int H, int W, int oy, int ox,
                                               __half *hout, float *map, const __half *hmask) {
    if (oy >= H || ox >= W) return;
    const size_t HW = (size_t)H * W;
    if constexpr (EPI == EPI_MAP) {
        map[(size_t)oy * W + ox] = __uint_as_float(r[0]) + sBias[0];
    } else {
#pragma unroll
        for (int g = 0; g < NOUT / 8; ++g) {
            const size_t pix = (size_t)g * HW + (size_t)oy * W + ox;
            __align__(16) __half h[8];
            if (EPI == EPI_RELU) {
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    h[c] = __float2half_rn(fmaxf(__uint_as_float(r[8 * g + c]) + sBias[8 * g + c], 0.f));
            } else {
                const uint4 mv = reinterpret_cast<const uint4 *>(hmask)[pix];
                const __half *mk = reinterpret_cast<const __half *>(&mv);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    h[c] = __float2half_rn(__hgt(mk[c], __float2half_rn(0.f)) ? __uint_as_float(r[8 * g + c]) : 0.f);
            }
            reinterpret_cast<uint4 *>(hout)[pix] = *reinterpret_cast<const uint4 *>(h);
        }
    }
}

// MT: 16 x 8 pixel tiles (MMA M = 128) per strip, side by side.
template <int CING, int NOUT, int MT>
struct ConvTcLayout {
    static constexpr int SX = 8 * MT, PX = SX + 2;                  // output and staged columns of a strip
    static constexpr size_t a_bytes = (size_t)CING * PY * PX * 16;  // staged input planes
    static constexpr size_t b_off = a_bytes;
    static constexpr size_t b_bytes = (size_t)9 * CING * NOUT * 16;  // weights [tap][plane][n][8]
    static constexpr size_t bias_off = b_off + b_bytes;
    static constexpr size_t bar_off = bias_off + (size_t)NOUT * 4;
    static constexpr size_t slot_off = bar_off + 16;
    static constexpr size_t used = slot_off + 16;
    static constexpr size_t total = used > MIN_SMEM ? used : MIN_SMEM;
    static constexpr uint32_t tcols = MT * NOUT;  // 64 or 256
};

// CING: input planes of 8 channels (2 for layer 0, whose C <= 3 channels
// occupy plane 0 and plane 1 is zero; 4 otherwise).  NOUT: MMA N.
// IN_F32: the input is an FP32 planar C x H x W array (the image) times
// in_scale (1/255); otherwise FP16 planes hin[g][y][x][8].  EPI: the
// epilogue (EPI_RELU, EPI_MAP, EPI_MASK with the activation planes hmask).
template <int CING, int NOUT, int MT, bool IN_F32, int EPI>
__global__ void __launch_bounds__(NTH, 2)
    k_conv_tc(const float *img, int C, float in_scale, const __half *hin, int H, int W, const __half *wp,
              const __half *wbias, int cout, __half *__restrict__ hout, float *__restrict__ map, const __half *hmask,
              int *err) {
    using L = ConvTcLayout<CING, NOUT, MT>;
    constexpr int SX = L::SX, PX = L::PX;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint4 *sA = reinterpret_cast<uint4 *>(smem);
    __half *sB = reinterpret_cast<__half *>(smem + L::b_off);
    float *sBias = reinterpret_cast<float *>(smem + L::bias_off);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + L::bar_off);
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L::slot_off);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // layer 0 may follow the kernel that wrote its weights; a backward pass follows the loss, which waited for it
    if (EPI == EPI_MASK) stage_weights<CING, NOUT, EPI>(wp, wbias, cout, sB, sBias, tid);
    if (tid == 0) {
        tc::bar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) tc::tmem_alloc(slot, L::tcols);
    grid_wait();
    grid_launch();
    if (EPI != EPI_MASK) stage_weights<CING, NOUT, EPI>(wp, wbias, cout, sB, sBias, tid);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *slot;
    const uint32_t idesc = tc::idesc_f16(128, NOUT, false);
    const int nsx = (W + SX - 1) / SX, nstrip = ((H + SY - 1) / SY) * nsx;
    const size_t HW = (size_t)H * W;
    uint32_t phase = 0;

    for (int strip = blockIdx.x; strip < nstrip; strip += gridDim.x) {
        const int y0 = (strip / nsx) * SY, x0 = (strip % nsx) * SX;
        // ---- stage the input planes with the halo (zero outside the image)
        if constexpr (IN_F32) {
            // plane 0 only (the others stay zero from the first strip): every load of the thread's pixels
            // issued before the first conversion
            constexpr int NE = (PY * PX + NTH - 1) / NTH;
            float v[NE][3];
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                const int e = tid + i * NTH, py = e / PX, px = e - py * PX;
                const int y = y0 - 1 + py, x = x0 - 1 + px;
                const bool in = e < PY * PX && y >= 0 && y < H && x >= 0 && x < W;
#pragma unroll
                for (int c = 0; c < 3; ++c) v[i][c] = (in && c < C) ? img[c * HW + (size_t)y * W + x] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                const int e = tid + i * NTH;
                if (e < PY * PX) {
                    __align__(16) __half h[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) h[c] = __float2half_rn(c < 3 ? v[i][c] * in_scale : 0.f);
                    sA[e] = *reinterpret_cast<const uint4 *>(h);
                }
            }
            if (strip == (int)blockIdx.x)
                for (int e = PY * PX + tid; e < CING * PY * PX; e += NTH) sA[e] = make_uint4(0u, 0u, 0u, 0u);
        } else {
            for (int e = tid; e < CING * PY * PX; e += NTH) {
                const int g = e / (PY * PX), r = e - g * (PY * PX), py = r / PX, px = r - py * PX;
                const int y = y0 - 1 + py, x = x0 - 1 + px;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (y >= 0 && y < H && x >= 0 && x < W) v = reinterpret_cast<const uint4 *>(hin)[((size_t)g * H + y) * W + x];
                sA[e] = v;
            }
        }
        tc::fence_async_smem();
        __syncthreads();
        // ---- MMAs (one thread): tile j, tap (ky, kx), K step s = planes 2s, 2s + 1
        if (tid == 0) {
            tc::fence_after();
            const uint32_t a0 = tc::su32(sA), b0 = tc::su32(sB);
            for (int j = 0; j < MT; ++j)
                for (int tap = 0; tap < 9; ++tap) {
                    const int ky = tap / 3, kx = tap - 3 * ky;
#pragma unroll
                    for (int s = 0; s < CING / 2; ++s) {
                        const uint32_t aoff = (uint32_t)((((2 * s) * PY + ky) * PX + 8 * j + kx) * 16);
                        const uint32_t boff = (uint32_t)((tap * CING + 2 * s) * NOUT * 16);
                        const uint64_t ad = tc::sdesc(a0 + aoff, PY * PX * 16, PX * 16);
                        const uint64_t bd = tc::sdesc(b0 + boff, NOUT * 16, 128);
                        tc::mma_f16(tbase + j * NOUT, ad, bd, idesc, (tap | s) ? 1u : 0u);
                    }
                }
            tc::mma_commit(bar);
        }
        const bool done = tc::bar_wait(bar, phase, SPIN);
        if (__syncthreads_or(!done)) {
            if (tid == 0) {
                tc::bar_wait(bar, phase, SPIN);  // the MMAs must end before the memory is released
                atomicExch(err, 1);
            }
            break;
        }
        phase ^= 1u;
        tc::fence_after();
        // ---- epilogue: thread = pixel (row m of the tile), warps 0-3 even tiles, 4-7 odd tiles
        const int q = warp & 3, m = 32 * q + lane;
        const int oy = y0 + (m >> 3);
        for (int j = warp >> 2; j < MT; j += 2) {
            tc::converge();
            const int ox = x0 + 8 * j + (m & 7);
            const uint32_t taddr = tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(j * NOUT);
            uint32_t r[32];
            if (EPI == EPI_MAP) {
                r[0] = tc::tmem_ld1(taddr);
                tc::tmem_wait_ld(r[0]);
            } else {
                tc::tmem_ld32(taddr, r);
                tc::tmem_wait_ld(r);
            }
            epilogue_store<NOUT, EPI>(r, sBias, H, W, oy, ox, hout, map, hmask);
        }
        tc::fence_before();
        __syncthreads();  // tensor memory and the staged planes are free for the next strip
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, L::tcols);
}

// Hidden layers (1..4: four planes of 8 FP16 channels in), with the input staged by TMA: a block runs
// its strips (16 x 16 output pixels: two 16 x 8 tiles) in turn through a ring of NBH staging buffers.  The
// copies of the block's next NBH - 1 strips (4 x 18 x 18 boxes of 16-byte pixel vectors, zero outside the
// image) are in flight while a strip's MMAs and epilogue run; once a strip's MMAs have completed its buffer
// takes the copy of the strip NBH ahead.  Two blocks per SM (four 21 KB buffers each, 64 tensor-memory
// columns, at most 128 registers a thread): six input boxes in flight per SM keep enough reads outstanding
// for the memory's latency.  Waits bounded as in k_conv_tc; a block that gives up waits (bounded) for its
// copies in flight and its MMAs before it releases its shared and tensor memory.
constexpr int CING_H = 4;
constexpr int MTH = 2;                 // tiles per strip of the hidden layers
constexpr int NBH = 4;                 // staging buffers (ring)
constexpr int SXH = 8 * MTH, PXH = SXH + 2;
constexpr size_t TMA_BOX_BYTES = (size_t)CING_H * PY * PXH * 16;
constexpr size_t TMA_BUF = (TMA_BOX_BYTES + 1023) / 1024 * 1024;

template <int NOUT>
struct ConvTmaLayout {
    static constexpr size_t b_off = NBH * TMA_BUF;  // buffer k at k * TMA_BUF
    static constexpr size_t b_bytes = (size_t)9 * CING_H * NOUT * 16;
    static constexpr size_t bias_off = b_off + b_bytes;
    static constexpr size_t bar_off = (bias_off + (size_t)NOUT * 4 + 15) / 16 * 16;
    static constexpr size_t total = bar_off + (NBH + 1) * 8 + 16;  // NBH copy barriers, the MMA barrier, slot
    static constexpr uint32_t tcols = MTH * NOUT < 32 ? 32 : MTH * NOUT;
};

template <int NOUT, int EPI>
__global__ void __launch_bounds__(NTH, 2)
    k_conv_tma(const __grid_constant__ CUtensorMap tmap, int H, int W, const __half *wp, const __half *wbias, int cout,
               __half *__restrict__ hout, float *__restrict__ map, const __half *hmask, int *err) {
    using L = ConvTmaLayout<NOUT>;
    extern __shared__ __align__(1024) unsigned char smem[];
    __half *sB = reinterpret_cast<__half *>(smem + L::b_off);
    float *sBias = reinterpret_cast<float *>(smem + L::bias_off);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + L::bar_off);  // [NBH]: a staging buffer's copy landed
    uint64_t *mbar = full + NBH;                                       // the strip's MMAs completed
    uint32_t *slot = reinterpret_cast<uint32_t *>(full + NBH + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    stage_weights<CING_H, NOUT, EPI>(wp, wbias, cout, sB, sBias, tid);
    const int nsx = (W + SXH - 1) / SXH, nstrip = ((H + SY - 1) / SY) * nsx;
    if (tid == 0) {
        for (int k = 0; k <= NBH; ++k) tc::bar_init(&full[k], 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) tc::tmem_alloc(slot, L::tcols);
    tc::fence_async_smem();
    grid_wait();  // (the weights above were written before the layer before this one started its own work)
    grid_launch();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *slot;
    const uint32_t idesc = tc::idesc_f16(128, NOUT, false);
    auto issue_copy = [&](int strip, int b) {  // thread 0: the strip's input box into buffer b
        const int y0 = (strip / nsx) * SY, x0 = (strip % nsx) * SXH;
        tc::bar_arrive_expect_tx(&full[b], (uint32_t)TMA_BOX_BYTES);
        tc::tma_load_3d(smem + (size_t)b * TMA_BUF, &tmap, &full[b], 2 * (x0 - 1), y0 - 1, 0);
    };
    // The block's k-th strip goes through buffer k % NBH; copies issued (and waited for) in order, so copy k
    // lands on the (k / NBH)-th phase of its buffer's barrier.  The counts are the same on every thread.
    int issued = 0, waited = 0;
    for (int k = 0; k < NBH && (int)blockIdx.x + k * (int)gridDim.x < nstrip; ++k) {
        if (tid == 0) issue_copy(blockIdx.x + k * gridDim.x, k);
        ++issued;
    }
    bool failed = false;
    int i = 0;
    for (int strip = blockIdx.x; strip < nstrip; strip += gridDim.x, ++i) {
        const int b = i % NBH;
        const int y0 = (strip / nsx) * SY, x0 = (strip % nsx) * SXH;
        const bool landed = tc::bar_wait(&full[b], (uint32_t)((i / NBH) & 1), SPIN);
        if (__syncthreads_or(!landed)) {
            failed = true;
            break;
        }
        ++waited;
        if (tid == 0) {
            tc::fence_after();
            const uint32_t a0 = tc::su32(smem + (size_t)b * TMA_BUF), b0 = tc::su32(sB);
            for (int j = 0; j < MTH; ++j)
                for (int tap = 0; tap < 9; ++tap) {
                    const int ky = tap / 3, kx = tap - 3 * ky;
#pragma unroll
                    for (int ss = 0; ss < CING_H / 2; ++ss) {
                        const uint32_t aoff = (uint32_t)((((2 * ss) * PY + ky) * PXH + 8 * j + kx) * 16);
                        const uint32_t boff = (uint32_t)((tap * CING_H + 2 * ss) * NOUT * 16);
                        const uint64_t ad = tc::sdesc(a0 + aoff, PY * PXH * 16, PXH * 16);
                        const uint64_t bd = tc::sdesc(b0 + boff, NOUT * 16, 128);
                        tc::mma_f16(tbase + j * NOUT, ad, bd, idesc, (tap | ss) ? 1u : 0u);
                    }
                }
            tc::mma_commit(mbar);
        }
        const bool done = tc::bar_wait(mbar, (uint32_t)(i & 1), SPIN);
        if (__syncthreads_or(!done)) {
            if (tid == 0) tc::bar_wait(mbar, (uint32_t)(i & 1), SPIN);  // the MMAs end before the memory is released
            failed = true;
            break;
        }
        tc::fence_after();
        // buffer b is free (this strip's MMAs have read it): the copy of the strip NBH ahead
        const int ahead = strip + NBH * (int)gridDim.x;
        if (ahead < nstrip) {
            if (tid == 0) issue_copy(ahead, b);
            ++issued;
        }
        const int q = warp & 3, m = 32 * q + lane;
        const int oy = y0 + (m >> 3);
        for (int j = warp >> 2; j < MTH; j += 2) {
            tc::converge();
            const int ox = x0 + 8 * j + (m & 7);
            const uint32_t taddr = tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(j * NOUT);
            uint32_t r[32];
            if (EPI == EPI_MAP) {
                r[0] = tc::tmem_ld1(taddr);
                tc::tmem_wait_ld(r[0]);
            } else {
                tc::tmem_ld32(taddr, r);
                tc::tmem_wait_ld(r);
            }
            epilogue_store<NOUT, EPI>(r, sBias, H, W, oy, ox, hout, map, hmask);
        }
        tc::fence_before();
        __syncthreads();  // tensor memory is free for the next strip
    }
    if (failed && tid == 0) {
        atomicExch(err, 1);
        // copies still in flight must land before the block's shared memory is released
        for (int w = waited; w < issued; ++w) tc::bar_wait(&full[w % NBH], (uint32_t)((w / NBH) & 1), SPIN);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, L::tcols);
}

// The network's weights of layer l, its biases and their number, as conv_tc / conv_tma take them.
#define LW(n, l) (n)->wpk + (n)->pf[l], (n)->w16 + (n)->off[l] + (n)->cout[l] * (n)->cin[l] * 9, (n)->cout[l]
// The flipped weights of a backward pass through layer l (no biases).
#define LWB(n, l) (n)->wpk + (n)->pb[l], nullptr, 0

// After a forward whose wait gave up: the whole map becomes NaN.
__global__ void k_map_poison(float *map, size_t n, const int *err) {
    if (*err == 0) return;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        map[i] = __int_as_float(0x7fc00000);
}

// wp: the layer's packed weights (the network's, or the flipped ones of a backward pass).
template <int CING, int NOUT, int MT, bool IN_F32, int EPI>
hts_status conv_tc_mt(const hts_cnn *n, const __half *wp, const __half *wbias, int cout, const float *img, int C,
                      float in_scale, const __half *hin, int H, int W, __half *hout, float *map, const __half *hmask,
                      int nsm, cudaStream_t s) {
    using L = ConvTcLayout<CING, NOUT, MT>;
    const void *k = reinterpret_cast<const void *>(k_conv_tc<CING, NOUT, MT, IN_F32, EPI>);
    const hts_status st = allow_smem(k, L::total);
    if (st != HTS_OK) return st;
    const int nstrip = ((H + SY - 1) / SY) * ((W + L::SX - 1) / L::SX);
    const int grid = std::max(1, std::min(nstrip, 2 * nsm));
    return launch_chained("k_conv_tc", k_conv_tc<CING, NOUT, MT, IN_F32, EPI>, dim3(grid), NTH, L::total, s, img, C,
                          in_scale, hin, H, W, wp, wbias, cout, hout, map, hmask, n->err);
}

// Strips of 64 columns (the least halo) where they fill the two blocks of every SM, else of 16: on a 256 x 256 crop 64
// blocks of four times the work left most SMs idle (11.5 us a layer between events, now 9).
template <int CING, int NOUT, bool IN_F32, int EPI>
hts_status conv_tc(const hts_cnn *n, const __half *wp, const __half *wbias, int cout, const float *img, int C,
                   float in_scale, const __half *hin, int H, int W, __half *hout, float *map, const __half *hmask,
                   int nsm, cudaStream_t s) {
    if (((H + SY - 1) / SY) * ((W + 63) / 64) >= 2 * nsm)
        return conv_tc_mt<CING, NOUT, 8, IN_F32, EPI>(n, wp, wbias, cout, img, C, in_scale, hin, H, W, hout, map, hmask,
                                                      nsm, s);
    return conv_tc_mt<CING, NOUT, 2, IN_F32, EPI>(n, wp, wbias, cout, img, C, in_scale, hin, H, W, hout, map, hmask, nsm,
                                                  s);
}

// A hidden layer with the TMA-staged input: the tensor map describes hin as [plane][y][x][8 halves], read
// as 8-byte elements (3-D, innermost first: 2 W, H, 4 planes) with the box of one strip's staged input.
template <int NOUT, int EPI>
hts_status conv_tma(const hts_cnn *n, const __half *wp, const __half *wbias, int cout, const __half *hin, int H, int W,
                    __half *hout, float *map, const __half *hmask, int nsm, cudaStream_t s) {
    using L = ConvTmaLayout<NOUT>;
    const auto enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tensor_map_encoder());
    if (!enc) return report(HTS_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
    // 8-byte elements, two per pixel vector: each box row is one contiguous run of 2 PXH elements
    CUtensorMap tmap;
    const cuuint64_t dims[3] = {(cuuint64_t)W * 2, (cuuint64_t)H, (cuuint64_t)CING_H};
    const cuuint64_t strides[2] = {(cuuint64_t)W * 16, (cuuint64_t)H * W * 16};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * PXH), (cuuint32_t)PY, (cuuint32_t)CING_H};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<__half *>(hin), dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return report(HTS_ECUDA, "cuTensorMapEncodeTiled failed for a network layer");
    const void *k = reinterpret_cast<const void *>(k_conv_tma<NOUT, EPI>);
    const hts_status st = allow_smem(k, L::total);
    if (st != HTS_OK) return st;
    const int nstrip = ((H + SY - 1) / SY) * ((W + SXH - 1) / SXH);
    const int grid = std::max(1, std::min(nstrip, 2 * nsm));
    return launch_chained("k_conv_tma", k_conv_tma<NOUT, EPI>, dim3(grid), NTH, L::total, s, tmap, H, W, wp, wbias, cout,
                          hout, map, hmask, n->err);
}

// ------------------------------------------------------------------ training (backward) on the tensor cores

// Weight and bias gradients of every layer in one launch: per layer dW[co][ci][ky][kx] = sum_p dY[co](p) X[ci](p +
// (ky - 1, kx - 1)), db[co] = sum_p dY[co](p), a contraction over the pixels (the MMA's K): D_kx[(ky, ci)][co] +=
// A_kx[(ky, ci)][p] B[co][p].  A block takes strips of 8 x 64 pixels of one layer and stages X with a one-pixel halo
// as [row][plane][column] vectors of 8 channels and dY as planes.  In that order the 8-row groups (ky, plane) of A at
// a given kx lie one staged row piece (PX vectors) apart, so the descriptor of tap column kx, strip row r and 16
// pixels is the staged region itself (MN-major, M = 128: three ky, the rest of the rows multiply whatever follows
// and are not read back): no copy per tap, and every MMA of a strip issued at once.  An all-ones operand (its groups
// overlapping in 512 bytes) gives the bias gradient.  B is the staged dY row, MN-major as well (core matrices of 8
// pixels, planes 8 KB apart).  Every block accumulates its strips in tensor memory, rows then 16-pixel steps, and
// writes its sums once; k_wgrad_reduce adds the blocks' sums in block order.
// Bound by latency at the training crops' size (128 strips a layer): staging, about 4 us of MMAs whose 4 KB A
// operands come from shared memory, the read-back.  Three blocks per SM and the five layers side by side hide them:
// 256 x 256 x 3, between events, 33 us for the layers together (before, a launch per layer with a copy of every tap
// and a wait per strip row: 96 us); the reduction in one coalesced launch: 17 us (before 116).
constexpr int WSY = 8;            // strip rows
constexpr int WPY = WSY + 2;      // staged X rows
constexpr int WCH = SX;           // strip columns
constexpr int NWG = 5;            // layers

struct WgLayer {
    const void *x, *y;  // X: FP16 planes [cinx][H][W][8], or the FP32 image (planar, C channels; times 1/255);
                        // dY: FP16 planes [nply][H][W][8], or the FP32 gradient map (one channel; times y_scale)
    int x_f32, y_f32, C, cinx, nply;
    int rows;           // 72 cinx + 1: (tap, ci), then the bias row
    int cin, cout;
    size_t part;        // the layer's parts [block][rows][8 nply]
    float *grad;
};
struct WgradArgs {
    WgLayer l[NWG];     // in launch order
    int H, W, nblk;     // blocks per layer
    float y_scale;      // the loss scale dY carries (applied here when dY is the FP32 map)
    float *part;
    int *err;
};
struct WgradLayout {
    static constexpr size_t x_bytes = (size_t)4 * WPY * PX * 16;
    static constexpr size_t y_off = x_bytes, y_plane = (size_t)WSY * WCH * 16;
    static constexpr size_t one_off = y_off + 4 * y_plane;
    static constexpr size_t bar_off = one_off + 512;
    static constexpr size_t total = bar_off + 16;
    static constexpr uint32_t tcols = 128;  // three tap columns and the ones, 32 each
};
static_assert(WgradLayout::y_off % 128 == 0 && 3 * (WgradLayout::total + 1024) <= 228 * 1024, "three blocks per SM");
// the last MMA's A operand (16 groups from strip row 7, tap column 2, the last 16 pixels) stays in the staged bytes
static_assert(((WSY - 1 + 15) * PX + 2 + WCH) * 16 <= WgradLayout::one_off &&
                  (((WSY - 1) * 4 + 15) * PX + 2 + WCH) * 16 <= WgradLayout::one_off, "A stays in bounds");

__global__ void __launch_bounds__(NTH, 3) k_conv_wgrad(const __grid_constant__ WgradArgs a) {
    using L = WgradLayout;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint4 *sX = reinterpret_cast<uint4 *>(smem);
    uint4 *sY = reinterpret_cast<uint4 *>(smem + L::y_off);
    uint4 *s1 = reinterpret_cast<uint4 *>(smem + L::one_off);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + L::bar_off);
    uint32_t *slot = reinterpret_cast<uint32_t *>(bar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const WgLayer &l = a.l[blockIdx.y];
    const int H = a.H, W = a.W, cinx = l.cinx, nply = l.nply;
    const size_t HW = (size_t)H * W;
    if (tid < 32) s1[tid] = make_uint4(0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u);  // FP16 ones
    if (tid == 0) {
        tc::bar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) tc::tmem_alloc(slot, L::tcols);
    grid_wait();
    grid_launch();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *slot;
    const uint32_t idesc = tc::idesc_f16(128, 8 * nply, false) | (1u << 15) | (1u << 16);  // A and B MN-major
    const int nsx = (W + WCH - 1) / WCH, nstrip = ((H + WSY - 1) / WSY) * nsx;
    uint32_t phase = 0;
    bool first = true, failed = false;
    for (int strip = blockIdx.x; strip < nstrip; strip += gridDim.x) {
        const int y0 = (strip / nsx) * WSY, x0 = (strip % nsx) * WCH;
        // ---- stage X (halo, zero outside the image) and dY (zero outside)
        for (int e = tid; e < cinx * WPY * PX; e += NTH) {
            const int rg = e / PX, px = e - rg * PX, py = rg / cinx, gp = rg - py * cinx;
            const int y = y0 - 1 + py, x = x0 - 1 + px;
            const bool in = y >= 0 && y < H && x >= 0 && x < W;
            if (!l.x_f32) {
                const uint4 *src = static_cast<const uint4 *>(l.x);
                tc::cp_async16(sX + e, in ? src + ((size_t)gp * H + y) * W + x : src, in);
            } else {
                const float *img = static_cast<const float *>(l.x);
                __align__(16) __half h[8];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    h[c] = __float2half_rn(in && c < l.C ? img[c * HW + (size_t)y * W + x] * (1.f / 255.f) : 0.f);
                sX[e] = *reinterpret_cast<const uint4 *>(h);
            }
        }
        for (int e = tid; e < nply * WSY * WCH; e += NTH) {
            const int gp = e / (WSY * WCH), r = e - gp * (WSY * WCH), py = r / WCH, px = r - py * WCH;
            const int y = y0 + py, x = x0 + px;
            const bool in = y < H && x < W;
            if (!l.y_f32) {
                const uint4 *src = static_cast<const uint4 *>(l.y);
                tc::cp_async16(sY + e, in ? src + ((size_t)gp * H + y) * W + x : src, in);
            } else {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (in && gp == 0)
                    v.x = __half_as_ushort(
                        __float2half_rn(static_cast<const float *>(l.y)[(size_t)y * W + x] * a.y_scale));
                sY[e] = v;
            }
        }
        tc::cp_async_wait();
        tc::fence_async_smem();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
            const uint32_t xa = tc::su32(sX), ya = tc::su32(sY);
            const uint64_t od = tc::sdesc(tc::su32(s1), 128, 16);
            for (int r = 0; r < WSY; ++r)
#pragma unroll
                for (int kk = 0; kk < WCH / 16; ++kk) {
                    const uint64_t bd = tc::sdesc(ya + (uint32_t)(r * WCH + kk * 16) * 16, 128, (uint32_t)L::y_plane);
                    const uint32_t acc = (first && r == 0 && kk == 0) ? 0u : 1u;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx)
                        tc::mma_f16(tbase + kx * 32,
                                    tc::sdesc(xa + (uint32_t)(r * cinx * PX + kx + kk * 16) * 16, 128, PX * 16), bd,
                                    idesc, acc);
                    tc::mma_f16(tbase + 96, od, bd, idesc, acc);
                }
            tc::mma_commit(bar);
        }
        const bool done = tc::bar_wait(bar, phase, SPIN);
        if (__syncthreads_or(!done)) {
            if (tid == 0) {
                tc::bar_wait(bar, phase, SPIN);  // the MMAs must end before the memory is released
                atomicExch(a.err, 1);
            }
            failed = true;
            break;
        }
        phase ^= 1u;
        tc::fence_after();
        first = false;
    }
    // ---- the block's sums: row (tap, ci) or the bias row, 8 nply output channels
    if (!failed) {
        const int q = warp & 3, row = 32 * q + lane, gr = row >> 3, ch = row & 7;
        const int ky = gr / cinx, gp = gr - ky * cinx;
        for (int t = warp >> 2; t < 4; t += NTH / 128) {
            tc::converge();
            uint32_t v[32];
            tc::tmem_ld32(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(t * 32), v);
            tc::tmem_wait_ld(v);
            int orow = -1;
            if (t < 3) {
                if (ky < 3) orow = ((ky * 3 + t) * cinx + gp) * 8 + ch;  // (tap, ci)
            } else if (row == 0) {
                orow = l.rows - 1;  // the bias
            }
            if (orow >= 0) {
                uint4 *dst = reinterpret_cast<uint4 *>(a.part + l.part + ((size_t)blockIdx.x * l.rows + orow) * 8 * nply);
#pragma unroll
                for (int n = 0; n < 8; ++n)
                    if (n < 2 * nply) dst[n] = make_uint4(v[4 * n], v[4 * n + 1], v[4 * n + 2], v[4 * n + 3]);
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, L::tcols);
}

// grad[e] += (sum over the blocks, in block order, of their sums) / y_scale for every parameter of every layer
// (cout x cin x 9 weights, then cout biases); NaN everywhere after a wait that gave up.  A thread per element of a
// part, so that the reads are coalesced (the writes, one in nblk, scatter).
__global__ void __launch_bounds__(256) k_wgrad_reduce(const __grid_constant__ WgradArgs a) {
    const WgLayer &l = a.l[blockIdx.y];
    const int N = 8 * l.nply, j = blockIdx.x * 256 + threadIdx.x;
    grid_wait();
    grid_launch();
    if (j >= l.rows * N) return;
    const int row = j / N, co = j - row * N, cp = 8 * l.cinx, tap = row / cp, ci = row - tap * cp;
    const bool bias = row == l.rows - 1;
    if (co >= l.cout || (!bias && ci >= l.cin)) return;
    const float *p = a.part + l.part + j;
    const size_t stride = (size_t)l.rows * N;
    float s = 0.f;
    for (int b0 = 0; b0 < a.nblk; b0 += 32) {  // 32 loads in flight, added in block order
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = b0 + i < a.nblk ? p[(size_t)(b0 + i) * stride] : 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (b0 + i < a.nblk) s += v[i];
    }
    float *g = l.grad + (bias ? l.cout * l.cin * 9 + co : (co * l.cin + ci) * 9 + tap);
    *g = *a.err ? __int_as_float(0x7fc00000) : *g + s * (1.f / a.y_scale);
}

// Rows of a block's sums over all the layers, times their output channels.
constexpr size_t WG_PART = (size_t)(72 + 1) * 32 + 3 * (size_t)(72 * 4 + 1) * 32 + (size_t)(72 * 4 + 1) * 16;

// Every layer's gradients: x[l] the layer's input (the image for layer 0), dy[l] the gradient of its output.
hts_status conv_wgrad(hts_cnn *n, const float *img, __half *const *act, const float *d4, __half *const *dy,
                      float y_scale, int H, int W, int nsm, cudaStream_t s) {
    WgradArgs a{};
    a.H = H;
    a.W = W;
    a.nblk = std::max(1, std::min(((H + WSY - 1) / WSY) * ((W + WCH - 1) / WCH), nsm));
    a.y_scale = y_scale;
    a.part = n->tr_part;
    a.err = n->err;
    size_t part = 0;
    int most = 0;
    for (int i = 0; i < NWG; ++i) {
        const int l = (i + 1) % NWG;  // layer 0, the cheapest, last
        WgLayer &w = a.l[i];
        w.x = l == 0 ? static_cast<const void *>(img) : act[l - 1];
        w.y = l == NWG - 1 ? static_cast<const void *>(d4) : dy[l];
        w.x_f32 = l == 0;
        w.y_f32 = l == NWG - 1;
        w.C = n->C;
        w.cinx = l == 0 ? 1 : 4;
        w.nply = l == NWG - 1 ? 2 : 4;
        w.rows = 72 * w.cinx + 1;
        w.cin = n->cin[l];
        w.cout = n->cout[l];
        w.part = part;
        w.grad = n->grad + n->off[l];
        part += (size_t)a.nblk * w.rows * 8 * w.nply;
        most = std::max(most, w.rows * 8 * w.nply);
    }
    hts_status st = allow_smem(reinterpret_cast<const void *>(k_conv_wgrad), WgradLayout::total);
    if (st != HTS_OK) return st;
    st = launch_chained("k_conv_wgrad", k_conv_wgrad, dim3(a.nblk, NWG), NTH, WgradLayout::total, s, a);
    if (st != HTS_OK) return st;
    return launch_chained("k_wgrad_reduce", k_wgrad_reduce, dim3((most + 255) / 256, NWG), 256, 0, s, a);
}

}  // namespace

template <typename T>
hts_status grow_buf(T *&p, size_t &cap, size_t need) {
    if (need <= cap && p) return HTS_OK;
    cudaFree(p);
    p = nullptr;
    cap = 0;
    if (dev_malloc(&p, need * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return report(HTS_ENOMEM, "cudaMalloc(cnn inference buffers)");
    }
    cap = need;
    return HTS_OK;
}

hts_status cnn_ensure_h16(hts_cnn *n, int H, int W) {
    const size_t px = (size_t)H * W;
    if (px * 32 <= n->cap_h16 && n->h16[1]) return HTS_OK;
    size_t c0 = 0;
    hts_status st = grow_buf(n->h16[0], c0, px * 32);
    size_t c1 = 0;
    if (st == HTS_OK) st = grow_buf(n->h16[1], c1, px * 32);
    n->cap_h16 = st == HTS_OK ? px * 32 : 0;
    return st;
}

hts_status cnn_ensure_infer(hts_cnn *n, int H, int W, int nx) {
    hts_status st = cnn_ensure_h16(n, H, W);
    if (st == HTS_OK) st = grow_buf(n->map, n->cap_map, (size_t)H * W);
    return st == HTS_OK ? grow_buf(n->rows, n->cap_rows, (size_t)H * nx) : st;
}

hts_status cnn_forward_tc_into(hts_cnn *n, const float *img, int H, int W, __half *h0, __half *h1, float *map,
                               cudaStream_t s) {
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaMemsetAsync(n->err, 0, sizeof(int), s) != cudaSuccess) {
        cudaGetLastError();
        return report(HTS_ECUDA, "cudaMemsetAsync(cnn error flag)");
    }
    hts_status st = conv_tc<2, 32, true, EPI_RELU>(n, LW(n, 0), img, n->C, 1.f / 255.f, nullptr, H, W, h0, nullptr,
                                                   nullptr, nsm, s);
    if (st == HTS_OK) st = conv_tma<32, EPI_RELU>(n, LW(n, 1), h0, H, W, h1, nullptr, nullptr, nsm, s);
    if (st == HTS_OK) st = conv_tma<32, EPI_RELU>(n, LW(n, 2), h1, H, W, h0, nullptr, nullptr, nsm, s);
    if (st == HTS_OK) st = conv_tma<32, EPI_RELU>(n, LW(n, 3), h0, H, W, h1, nullptr, nullptr, nsm, s);
    if (st == HTS_OK) st = conv_tma<16, EPI_MAP>(n, LW(n, 4), h1, H, W, nullptr, map, nullptr, nsm, s);
    if (st != HTS_OK) return st;
    {
        KTimer kt("k_map_poison", s);
        k_map_poison<<<nsm, 256, 0, s>>>(map, (size_t)H * W, n->err);
    }
    return check_launch("k_map_poison");
}


// ------------------------------------------------------------------ tensor-core training step

hts_status cnn_train_ensure(hts_cnn *n, int H, int W, int nsm) {
    const size_t px = (size_t)H * W;
    if (px > n->tr_cap_px) {
        for (int i = 0; i < 4; ++i) {
            cudaFree(n->tr_act[i]);
            n->tr_act[i] = nullptr;
        }
        for (int i = 0; i < 4; ++i) {
            cudaFree(n->tr_dy[i]);
            n->tr_dy[i] = nullptr;
        }
        cudaFree(n->tr_map);
        cudaFree(n->tr_d0);
        n->tr_map = n->tr_d0 = nullptr;
        n->tr_cap_px = 0;
        size_t cap = 0;
        for (int i = 0; i < 4; ++i) {
            cap = 0;
            if (grow_buf(n->tr_act[i], cap, px * 32) != HTS_OK) return HTS_ENOMEM;
        }
        for (int i = 0; i < 4; ++i) {
            cap = 0;
            if (grow_buf(n->tr_dy[i], cap, px * 32) != HTS_OK) return HTS_ENOMEM;
        }
        cap = 0;
        if (grow_buf(n->tr_map, cap, px) != HTS_OK) return HTS_ENOMEM;
        cap = 0;
        if (grow_buf(n->tr_d0, cap, px) != HTS_OK) return HTS_ENOMEM;
        n->tr_cap_px = px;
    }
    return grow_buf(n->tr_part, n->tr_cap_part, (size_t)nsm * WG_PART);
}

// One image's loss and gradient on the tensor cores: the forward of cnn_forward_tc_into keeping every layer's
// FP16 activations, the loss gradient map 2 (out - target) / N_ref times the loss scale 2^(floor(log2 N_ref)
// + 2) (so (4, 8] times the error, well inside FP16's range) rounded to FP16, then from the last layer down the
// gradient of the layer input (the forward kernels with the flipped, transposed weights, times the ReLU mask of
// the stored activation, FP16), and every layer's weight and bias gradients at once (k_conv_wgrad, FP32
// accumulation, the scale divided out).
hts_status cnn_grad_tc(hts_cnn *n, const float *img, int H, int W, const Geom &g, const float *target,
                       cudaStream_t s) {
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    hts_status st = cnn_train_ensure(n, H, W, nsm);
    if (st != HTS_OK) return st;
    if (cudaMemsetAsync(n->err, 0, sizeof(int), s) != cudaSuccess) {
        cudaGetLastError();
        return report(HTS_ECUDA, "cudaMemsetAsync(cnn error flag)");
    }
    __half **a = n->tr_act;
    const float S = ldexpf(1.f, ilogb((double)g.nref) + 2);
    st = conv_tc<2, 32, true, EPI_RELU>(n, LW(n, 0), img, n->C, 1.f / 255.f, nullptr, H, W, a[0], nullptr, nullptr,
                                        nsm, s);
    for (int l = 1; l < 4 && st == HTS_OK; ++l)
        st = conv_tma<32, EPI_RELU>(n, LW(n, l), a[l - 1], H, W, a[l], nullptr, nullptr, nsm, s);
    if (st == HTS_OK) st = conv_tma<16, EPI_MAP>(n, LW(n, 4), a[3], H, W, nullptr, n->tr_map, nullptr, nsm, s);
    if (st == HTS_OK) st = cnn_loss(n, n->tr_map, H, W, g, target, n->tr_d0, s);
    __half **dy = n->tr_dy;
    if (st == HTS_OK)
        st = conv_tc<2, 32, true, EPI_MASK>(n, LWB(n, 4), n->tr_d0, 1, S, nullptr, H, W, dy[3], nullptr, a[3], nsm, s);
    for (int l = 3; l >= 1 && st == HTS_OK; --l)
        st = conv_tma<32, EPI_MASK>(n, LWB(n, l), dy[l], H, W, dy[l - 1], nullptr, a[l - 1], nsm, s);
    return st == HTS_OK ? conv_wgrad(n, img, a, n->tr_d0, dy, S, H, W, nsm, s) : st;
}

}  // namespace hts
