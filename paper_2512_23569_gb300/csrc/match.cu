// Grouping step of Haar-tSVD (Eq. 9, Alg. 1 step 1) on sm_103a.
//
// At the default grid step k_match_cells (below) shares the squared differences
// of neighbouring references; for other steps, windows above 31 and grids too
// small for it (cells_faster), k_match:
//
// A block of four warps takes a 2x2 block of reference patches and stages the
// union of their search regions of the matching planes in shared memory
// (gray image; for colour both the green channel and the channel sum R+G+B,
// since Eq. 9 picks one per reference).  Each warp takes one reference:
// lanes compute FP32 squared distances of 4 horizontally adjacent
// candidates per item (register-blocked), store every distance in shared
// memory and keep a sorted per-lane list of their 4 smallest keys (distance
// bits, raster index).  The (K-1)-th smallest key of the 32 lists bounds the
// true (K-1)-th from above; the warp then collects every candidate under the
// certified threshold (usually K-1 plus a few) and sorts only those.
//
// Exactness.  The group must equal the FP64 definition bit for bit: the K-1
// nearest candidates in ascending (distance, raster index), distances being
// the FP64 row-major sum of squared differences.  The FP32 distance d of a
// candidate whose FP64 distance is D obeys |d - D| <= eps D + beta sqrt(D) + g0
// (eps covers 66 roundings of the subtract / FMA chain; beta and g0 cover the
// rounding of the FP32 channel sum on the R+G+B plane, scaled by the largest
// |R|+|G|+|B| of the region; g0 also absorbs subnormal flushing).  If every
// adjacent pair among the first K sorted entries is separated by that bound,
// the FP32 order is the FP64 order.  Otherwise every entry that can still
// belong to the K-1 nearest is re-evaluated with the FP64 expression in the
// same operation order as the definition and ranked by (D, index).  When the
// candidate set exceeds what a warp handles (flat, noiseless inputs with
// massive ties), the reference goes to an exhaustive FP64 pass.
#include <algorithm>

#include "hts_internal.h"

namespace hts {
namespace {

constexpr float U32 = 5.9604644775390625e-08f;  // 2^-24
constexpr unsigned FULL = 0xffffffffu;
constexpr uint64_t EMPTY = ~0ull;

struct MatchArgs {
    const float *img;
    int H, W, C, step, R, nx, ny, nref;
    double gamma;
    int32_t *idx;
    uint8_t *green;
    int32_t *fb;
    DevState *st;
};

__device__ __forceinline__ uint64_t make_key(float d, int idx) {
    return ((uint64_t)__float_as_uint(d) << 32) | (uint32_t)idx;
}
__device__ __forceinline__ float key_dist(uint64_t k) { return __uint_as_float((uint32_t)(k >> 32)); }
__device__ __forceinline__ int key_idx(uint64_t k) { return (int)(uint32_t)(k & 0xffffffffu); }

template <int M>
__device__ __forceinline__ void topm_insert(uint64_t (&lst)[M], uint64_t key) {
    if (key >= lst[M - 1]) return;
#pragma unroll
    for (int i = M - 1; i > 0; --i) {
        const uint64_t prev = lst[i - 1], cur = lst[i];
        lst[i] = prev > key ? prev : (cur < key ? cur : key);
    }
    lst[0] = lst[0] < key ? lst[0] : key;
}

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const uint64_t w = __shfl_xor_sync(FULL, v, o);
        v = w < v ? w : v;
    }
    return v;
}

__device__ __forceinline__ float warp_max_f(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}

// Value of the matching plane in FP64, in the definition's operation order.
__device__ __forceinline__ double plane64(const float *__restrict__ img, size_t HW, int C, int green, size_t o) {
    if (C == 1) return (double)__ldg(img + o);
    if (green) return (double)__ldg(img + HW + o);
    return __dadd_rn(__dadd_rn((double)__ldg(img + o), (double)__ldg(img + HW + o)), (double)__ldg(img + 2 * HW + o));
}

// FP64 squared distance, row-major, no contraction (same order as the definition).
__device__ double exact_dist(const float *__restrict__ img, int W, size_t HW, int C, int green, int yr, int xr,
                             int yc, int xc) {
    double acc = 0.0;
    for (int u = 0; u < PS; ++u)
        for (int v = 0; v < PS; ++v) {
            const double a = plane64(img, HW, C, green, (size_t)(yr + u) * W + xr + v);
            const double b = plane64(img, HW, C, green, (size_t)(yc + u) * W + xc + v);
            const double d = __dsub_rn(a, b);
            acc = __dadd_rn(acc, __dmul_rn(d, d));
        }
    return acc;
}

// Eq. 9 on the reference patch in FP64 (sequential row-major sums, as the
// definition).  Lanes 0..2 each sum one channel; all lanes get the flag.
__device__ int gcp_green(const float *__restrict__ img, int W, size_t HW, int y, int x, double gamma, int lane) {
    double n2 = 0.0;
    if (lane < 3) {
        const float *ch = img + (size_t)lane * HW;
        for (int u = 0; u < PS; ++u)
            for (int v = 0; v < PS; ++v) {
                const double a = (double)__ldg(ch + (size_t)(y + u) * W + x + v);
                n2 = __dadd_rn(n2, __dmul_rn(a, a));
            }
    }
    const double r2 = __shfl_sync(FULL, n2, 0), g2 = __shfl_sync(FULL, n2, 1), b2 = __shfl_sync(FULL, n2, 2);
    const double nR = __dsqrt_rn(r2), nG = __dsqrt_rn(g2), nB = __dsqrt_rn(b2);
    const double lim = fmax(__ddiv_rn(nR, gamma), __ddiv_rn(nB, gamma));
    return nG >= lim ? 1 : 0;
}

// Certified interval of the FP64 distance given the FP32 one.
struct Bound {
    float eps, beta, g0;
    __device__ __forceinline__ float upper(float d) const {
        if (beta == 0.f) return __fdiv_rn(d + g0, 1.f - eps) * (1.f + 4.f * U32);
        const float a = 1.f - eps;
        const float s = (beta + sqrtf(beta * beta + 4.f * a * (g0 + d))) / (2.f * a);
        return s * s * (1.f + 8.f * U32);
    }
    __device__ __forceinline__ float lower(float d) const {
        if (d <= g0) return 0.f;
        if (beta == 0.f) return __fdiv_rn(d - g0, 1.f + eps) * (1.f - 4.f * U32);
        const float a = 1.f + eps;
        const float s = (-beta + sqrtf(beta * beta + 4.f * a * (d - g0))) / (2.f * a);
        return s * s * (1.f - 8.f * U32);
    }
};

constexpr int MW = 4;      // warps per block = a 2x2 block of reference patches sharing one staged region
constexpr int LTOP = 4;    // per-lane short list that bounds the (K-1)-th distance from above
constexpr int PMAX = 64;   // largest candidate set a warp certifies or re-ranks itself

// Eq. 9 with FP32 channel norms (64-term sums, relative error < 40 u): the
// decision is certain when nG^2 gamma^2 and max(nR^2, nB^2) differ by more
// than 1e-5 relative; otherwise the FP64 sequential definition decides.
__device__ int gcp_green_fast(const float *__restrict__ img, int W, size_t HW, int y, int x, double gamma, int lane) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = lane + 32 * q;
        const size_t o = (size_t)(y + (e >> 3)) * W + x + (e & 7);
        const float r = __ldg(img + o), g = __ldg(img + HW + o), b = __ldg(img + 2 * HW + o);
        s0 = fmaf(r, r, s0);
        s1 = fmaf(g, g, s1);
        s2 = fmaf(b, b, s2);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        s0 += __shfl_xor_sync(FULL, s0, o);
        s1 += __shfl_xor_sync(FULL, s1, o);
        s2 += __shfl_xor_sync(FULL, s2, o);
    }
    const float lhs = s1 * (float)(gamma * gamma), rhs = fmaxf(s0, s2);
    if (lhs > rhs * (1.f + 1e-5f) && lhs > 0.f) return 1;
    if (lhs < rhs * (1.f - 1e-5f)) return 0;
    return gcp_green(img, W, HW, y, x, gamma, lane);
}

// A warp's collected candidates: FP32 distances and raster indices, and the same sorted; PMAX entries each.
struct CandList {
    float *d, *sd;  // 16-byte aligned
    int *i, *si;
    double *d64;
    __device__ __forceinline__ CandList(void *list, void *scratch)
        : d(static_cast<float *>(list)), sd(static_cast<float *>(scratch)), i(reinterpret_cast<int *>(d + PMAX)),
          si(reinterpret_cast<int *>(sd + PMAX)), d64(reinterpret_cast<double *>(si + PMAX)) {}
    static constexpr int LIST = PMAX * 8, SCRATCH = PMAX * 16;  // bytes
};

// The group of one reference from its m collected candidates (K - 1 <= m <= PMAX, any order): sorted and, where the
// order is certain, written to out[1 ..] (returns 0); else the number of entries of c.si that may belong to the K-1
// nearest, for rerank_group.  One warp.
template <int K>
__device__ __forceinline__ int settle_group(const Bound &bd, const CandList &c, int m, int lane, int32_t *out) {
    if (lane < 4 && m + lane < PMAX) c.d[m + lane] = __int_as_float(0x7f800000);  // up to a multiple of 4
    __syncwarp();
    // ranks by distance, four comparisons per shared-memory load; equal distances collide and are ranked again with
    // the raster index
    const bool two = m > 32;
    const float inf = __int_as_float(0x7f800000);
    const float d0 = lane < m ? c.d[lane] : inf, d1 = lane + 32 < m ? c.d[lane + 32] : inf;
    const int i0 = lane < m ? c.i[lane] : 0, i1 = lane + 32 < m ? c.i[lane + 32] : 0;
    int r0 = 0, r1 = 0;
    for (int j = 0; j < m; j += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(c.d + j);
        r0 += (v.x < d0 ? 1 : 0) + (v.y < d0 ? 1 : 0) + (v.z < d0 ? 1 : 0) + (v.w < d0 ? 1 : 0);
        if (two) r1 += (v.x < d1 ? 1 : 0) + (v.y < d1 ? 1 : 0) + (v.z < d1 ? 1 : 0) + (v.w < d1 ? 1 : 0);
    }
    if (lane < m) c.si[r0] = i0;
    if (lane + 32 < m) c.si[r1] = i1;
    __syncwarp();
    const bool clash = (lane < m && c.si[r0] != i0) || (lane + 32 < m && c.si[r1] != i1);
    if (__any_sync(FULL, clash)) {
        r0 = r1 = 0;
        for (int j = 0; j < m; ++j) {
            const float v = c.d[j];
            const int w = c.i[j];
            r0 += (v < d0 || (v == d0 && w < i0)) ? 1 : 0;
            r1 += (v < d1 || (v == d1 && w < i1)) ? 1 : 0;
        }
        __syncwarp();
        if (lane < m) c.si[r0] = i0;
        if (lane + 32 < m) c.si[r1] = i1;
    }
    if (lane < m) c.sd[r0] = d0;
    if (lane + 32 < m) c.sd[r1] = d1;
    __syncwarp();
    bool ok = true;
    if (lane < K - 1 && lane + 1 < m) ok = bd.upper(c.sd[lane]) < bd.lower(c.sd[lane + 1]);
    if (__all_sync(FULL, ok)) {
        if (lane < K - 1) out[1 + lane] = c.si[lane];
        return 0;
    }
    const float thr = bd.upper(c.sd[K - 2]);
    int mp = 0;
    for (int i = 0; i < m; ++i) {
        if (bd.lower(c.sd[i]) > thr) break;
        mp = i + 1;
    }
    return mp;
}

// The K-1 nearest of the mp candidates `ids` by (FP64 distance, raster index) to out[1 ..]; d64: PMAX doubles of
// scratch.  One warp.
template <int K>
__device__ __forceinline__ void rerank_group(const MatchArgs &a, const int *ids, double *d64, int mp, int yr, int xr,
                                             int green, int lane, int32_t *out) {
    const size_t HW = (size_t)a.H * a.W;
    for (int i = lane; i < mp; i += 32) {
        const int id = ids[i];
        d64[i] = exact_dist(a.img, a.W, HW, a.C, green, yr, xr, id / a.W, id % a.W);
    }
    __syncwarp();
    for (int i = lane; i < mp; i += 32) {
        const double di = d64[i];
        const int ii = ids[i];
        int rank = 0;
        for (int j = 0; j < mp; ++j) {
            const double dj = d64[j];
            rank += (dj < di || (dj == di && ids[j] < ii)) ? 1 : 0;
        }
        if (rank < K - 1) out[1 + rank] = ii;
    }
    if (lane == 0) atomicAdd(&a.st->match_reranked, 1);
}

template <int K>
__global__ void __launch_bounds__(MW * 32) k_match(MatchArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int RHM = a.step + 2 * a.R + PS;          // region side bound
    const int NCM = (2 * a.R + 1) * (2 * a.R + 1);  // candidates per window bound
    const CandList cl(smem_raw + warp * (CandList::LIST + CandList::SCRATCH),
                      smem_raw + warp * (CandList::LIST + CandList::SCRATCH) + CandList::LIST);
    float *planeA = reinterpret_cast<float *>(smem_raw + (size_t)MW * (CandList::LIST + CandList::SCRATCH));
    float *planeS = planeA + RHM * RHM;
    float *dbuf = planeS + (a.C == 3 ? RHM * RHM : 0) + warp * NCM;
    __shared__ unsigned s_tmax;

    const int nbx = (a.nx + 1) >> 1;
    const int by = blockIdx.x / nbx, bx = blockIdx.x - by * nbx;
    const int gy = 2 * by + (warp >> 1), gx = 2 * bx + (warp & 1);
    const size_t HW = (size_t)a.H * a.W;
    // region = union of the block's windows (plus the patch extent)
    const int ya = grid_pos(2 * by, a.H, a.step), yb = grid_pos(min(2 * by + 1, a.ny - 1), a.H, a.step);
    const int xa = grid_pos(2 * bx, a.W, a.step), xb = grid_pos(min(2 * bx + 1, a.nx - 1), a.W, a.step);
    const int ry0 = max(0, ya - a.R), ry1 = min(a.H - PS, yb + a.R) + PS - 1;
    const int rx0 = max(0, xa - a.R), rx1 = min(a.W - PS, xb + a.R) + PS - 1;
    const int rh = ry1 - ry0 + 1, rw = rx1 - rx0 + 1;
    if (threadIdx.x == 0) s_tmax = 0u;
    __syncthreads();
    float tmax = 0.f;
    for (int e = threadIdx.x; e < rh * rw; e += blockDim.x) {
        const int yy = e / rw, xx = e - yy * rw;
        const size_t o = (size_t)(ry0 + yy) * a.W + (rx0 + xx);
        if (a.C == 1) {
            planeA[e] = __ldg(a.img + o);
        } else {
            const float R = __ldg(a.img + o), G = __ldg(a.img + HW + o), B = __ldg(a.img + 2 * HW + o);
            planeA[e] = G;
            planeS[e] = __fadd_rn(__fadd_rn(R, G), B);
            tmax = fmaxf(tmax, fabsf(R) + fabsf(G) + fabsf(B));
        }
    }
    tmax = warp_max_f(tmax);
    if (lane == 0) atomicMax(&s_tmax, __float_as_uint(tmax));  // non-negative floats order as their bits
    __syncthreads();
    if (gy >= a.ny || gx >= a.nx) return;  // no block-wide barrier below

    const int r = gy * a.nx + gx;
    const int yr = grid_pos(gy, a.H, a.step), xr = grid_pos(gx, a.W, a.step);
    const int green = (a.C == 3) ? gcp_green_fast(a.img, a.W, HW, yr, xr, a.gamma, lane) : 1;
    if (lane == 0 && a.green) a.green[r] = (uint8_t)green;
    const bool exact_plane = (a.C == 1) || green;
    const float *plane = exact_plane ? planeA : planeS;
    const float T3 = exact_plane ? 0.f : __uint_as_float(s_tmax);

    const int cy0 = max(0, yr - a.R), cy1 = min(a.H - PS, yr + a.R);
    const int cx0 = max(0, xr - a.R), cx1 = min(a.W - PS, xr + a.R);
    const int nrow = cy1 - cy0 + 1, ncol = cx1 - cx0 + 1, nc = nrow * ncol;
    const int oy = cy0 - ry0, ox = cx0 - rx0;

    float ar[NPIX];
    {
        const float *rp = plane + (yr - ry0) * rw + (xr - rx0);
#pragma unroll
        for (int u = 0; u < PS; ++u)
#pragma unroll
            for (int v = 0; v < PS; ++v) ar[u * PS + v] = rp[u * rw + v];
    }
    uint64_t lst[LTOP];
#pragma unroll
    for (int i = 0; i < LTOP; ++i) lst[i] = EMPTY;

    const int nq = (ncol + 3) >> 2;
    const int nitems = nrow * nq;
    for (int it = lane; it < nitems; it += 32) {
        const int i = it / nq, cxb = (it - i * nq) * 4;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        const float *base = plane + (oy + i) * rw + ox + cxb;
        const int lim = rw - ox - cxb;  // columns of the region right of this quad's first candidate
#pragma unroll
        for (int u = 0; u < PS; ++u) {
            const float *row = base + u * rw;
            float b[PS + 3];
#pragma unroll
            for (int t = 0; t < PS + 3; ++t) b[t] = (t < lim) ? row[t] : 0.f;
#pragma unroll
            for (int v = 0; v < PS; ++v) {
                const float av = ar[u * PS + v];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float e = __fsub_rn(av, b[v + t]);
                    d[t] = __fmaf_rn(e, e, d[t]);
                }
            }
        }
        const int gyy = cy0 + i;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int cx = cxb + t;
            if (cx < ncol) {
                const int gxx = cx0 + cx;
                if (gyy == yr && gxx == xr) {
                    dbuf[i * ncol + cx] = __int_as_float(0x7f800000);  // the reference itself: never collected
                } else {
                    dbuf[i * ncol + cx] = d[t];
                    topm_insert<LTOP>(lst, make_key(d[t], gyy * a.W + gxx));
                }
            }
        }
    }
    __syncwarp();

    // (K-1)-th smallest key of the union of the lane lists: an upper bound of the true one
    uint64_t tau = EMPTY;
    for (int j = 0; j < K - 1; ++j) {
        const uint64_t h = lst[0];
        const uint64_t mn = warp_min_u64(h);
        if (h == mn && mn != EMPTY) {
#pragma unroll
            for (int q = 0; q < LTOP - 1; ++q) lst[q] = lst[q + 1];
            lst[LTOP - 1] = EMPTY;
        }
        tau = mn;
    }
    int32_t *out = a.idx + (size_t)r * K;
    if (lane == 0) out[0] = yr * a.W + xr;
    Bound bd;
    bd.eps = 100.f * U32;
    bd.beta = exact_plane ? 0.f : 72.f * U32 * T3;
    bd.g0 = (exact_plane ? 0.f : 1200.f * U32 * U32 * T3 * T3) + 1e-30f;
    bool overflow = (tau == EMPTY);
    // collect every candidate whose distance may still matter
    int m = 0;
    if (!overflow) {
        const float T = bd.upper(bd.upper(key_dist(tau)));
        const unsigned lt = (1u << lane) - 1u;
        for (int c0 = 0; c0 < nc; c0 += 32) {
            const int c = c0 + lane;
            const float dv = (c < nc) ? dbuf[c] : __int_as_float(0x7f800000);
            const bool ok = dv <= T;
            const unsigned msk = __ballot_sync(FULL, ok);
            if (ok) {
                const int pos = m + __popc(msk & lt);
                if (pos < PMAX) {
                    const int ci = c / ncol;
                    cl.d[pos] = dv;
                    cl.i[pos] = (cy0 + ci) * a.W + cx0 + (c - ci * ncol);
                }
            }
            m += __popc(msk);
        }
        overflow = (m > PMAX) || (m < K - 1);
    }
    if (overflow) {
        if (lane == 0) {
            const int pos = atomicAdd(&a.st->match_fallback, 1);
            a.fb[pos] = r;
        }
        return;
    }
    __syncwarp();
    const int mp = settle_group<K>(bd, cl, m, lane, out);
    if (mp) rerank_group<K>(a, cl.si, cl.d64, mp, yr, xr, green, lane, out);
}

// ---- the default grid step (4): 4 x 4 cells shared by neighbouring references
//
// Two references 4 pixels apart share half their patches, and at one offset (dy, dx) the squared differences of the
// shared pixels are the same numbers: with the plane cut into 4 x 4 cells on the reference grid, a reference's
// distance at an offset is the sum of four cells' sums, and a cell's sum serves four references.  A block takes a
// tile of up to 8 x nry references; a thread takes an offset row dy and four consecutive dx, walks the tile's cell
// rows with the candidate row pieces sliding through registers (per cell and pixel row one 16-byte load of the
// reference, broadcast, and one of the candidates, conflict-free, for 32 operations), adds horizontally adjacent
// cells, keeps the row of these pairs in registers and adds the next one: about 43 operations a candidate where the
// distance alone took 128.  A row of references' distances goes to shared memory, and each warp settles a reference:
// a bound on the (K-1)-th distance from the two smallest of every lane (a sort of 32 values per list, no rounds of
// warp minima), the candidates under it, then as k_match; the few references whose order FP64 decides wait for the
// end of the tile, where they do not hold up a row.  Bound by issue (58-64 % active, 16 warps per SM) and, below
// 1000 tiles, by the uneven filling of the SMs.  Measured against a reference per warp (k_match): 768 x 1024 gray,
// K = 32, win 21: 184 us (562); 512 x 512 x 3, K = 16, win 31, beside the basis chain: 151 us (260); 1021 x 771 x 3:
// 352 us (683).
// Tiles are cut where the grid is: the last row / column of references, where H - 8 / W - 8 is no multiple of 4, are
// tiles of their own.
// Error: a term passes 2 roundings (difference, squared), at most 16 of the cell's chain and 2 of the cells' sums,
// 20 u together; Bound takes 32 u.
constexpr int CX = 8;          // references per tile row
constexpr int CT = 256;        // most threads: (2R + 1) * ceil((R4 + R + 1) / 4) <= 256, R4 = R rounded up to 4 (R <= 15)
constexpr float CEPS = 32.f * U32;
constexpr int NDEFER = 24;     // references a tile can leave to its end

struct CellArgs {
    MatchArgs m;
    int R4, G;                 // dx = 4 g + t - R4, g < G
    int nry;                   // reference rows per tile
    int rx, ry;                // references on the regular grid per row / column
    int ntx, nty;              // regular tiles
    int ncp;                   // floats per reference of the distance rows
    int rows, cols;            // staged region
};

// Ascending sort of one value per lane.
__device__ __forceinline__ float warp_sort(float v, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j; j >>= 1) {
            const float o = __shfl_xor_sync(FULL, v, j);
            const bool up = (lane & k) == 0 || k == 32, low = (lane & j) == 0;
            v = (up == low) ? fminf(v, o) : fmaxf(v, o);
        }
    return v;
}

template <int K>
__global__ void __launch_bounds__(CT, 2) k_match_cells(const __grid_constant__ CellArgs c) {
    constexpr int LT = K <= 16 ? 1 : 2;  // smallest distances of a lane that enter the bound
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const MatchArgs &a = c.m;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    const int npl = a.C == 3 ? 2 : 1, rw = c.cols;
    float *plane0 = reinterpret_cast<float *>(smem_raw);              // [npl][rows][cols]: gray or green, R + G + B
    float *dbuf = plane0 + (size_t)npl * c.rows * rw;                 // [CX][ncp] distances of a row of references
    unsigned char *list = reinterpret_cast<unsigned char *>(dbuf + (size_t)CX * c.ncp) + warp * CandList::LIST;
    __shared__ int defer[NDEFER * PMAX];  // candidates of the references left to the tile's FP64 re-rank
    __shared__ int4 s_defer[NDEFER];      // (reference, its position, candidates, plane)
    __shared__ int s_ndefer;
    __shared__ unsigned s_tmax;
    __shared__ unsigned s_use[2][8];  // per plane and reference row of the tile: the references that use it
    // ---- the tile: references (gy0 + i, gx0 + j) at (ya + 4 i, xa + 4 j), i < ni, j < nj
    const size_t HW = (size_t)a.H * a.W;
    int b = blockIdx.x, gy0, gx0, ni, nj;
    const int nreg = c.nty * c.ntx, nlc = a.nx > c.rx ? c.nty : 0, nlr = a.ny > c.ry ? c.ntx : 0;
    if (b < nreg) {
        gy0 = b / c.ntx * c.nry;
        gx0 = b % c.ntx * CX;
        ni = min(c.nry, c.ry - gy0);
        nj = min(CX, c.rx - gx0);
    } else if (b < nreg + nlc) {  // the last column, off the grid
        gy0 = (b - nreg) * c.nry;
        gx0 = c.rx;
        ni = min(c.nry, c.ry - gy0);
        nj = 1;
    } else {  // the last row, off the grid, and its corner
        gy0 = c.ry;
        gx0 = b < nreg + nlc + nlr ? (b - nreg - nlc) * CX : c.rx;
        ni = 1;
        nj = b < nreg + nlc + nlr ? min(CX, c.rx - gx0) : 1;
    }
    const int ya = grid_pos(gy0, a.H, 4), xa = grid_pos(gx0, a.W, 4);
    const int y0 = ya - a.R, x0 = xa - c.R4;  // region origin (may lie outside the image: zeros)
    if (tid == 0) {
        s_tmax = 0u;
        s_ndefer = 0;
    }
    if (tid < 16) s_use[tid >> 3][tid & 7] = 0u;
    for (int e = tid; e < CX * c.ncp; e += blockDim.x) dbuf[e] = __int_as_float(0x7f800000);  // the padding stays
    __syncthreads();
    float tmax = 0.f;
    const int nrow = 4 * (ni + 1) + 2 * a.R;
#pragma unroll 4
    for (int e = tid; e < nrow * rw; e += blockDim.x) {
        const int yy = e / rw, xx = e - yy * rw, y = y0 + yy, x = x0 + xx;
        const bool in = y >= 0 && y < a.H && x >= 0 && x < a.W;
        const size_t o = in ? (size_t)y * a.W + x : 0;
        if (a.C == 1) {
            plane0[e] = in ? __ldg(a.img + o) : 0.f;
        } else {
            const float r = __ldg(a.img + o), g = __ldg(a.img + HW + o), bl = __ldg(a.img + 2 * HW + o);
            plane0[e] = in ? g : 0.f;
            plane0[c.rows * rw + e] = in ? __fadd_rn(__fadd_rn(r, g), bl) : 0.f;
            if (in) tmax = fmaxf(tmax, fabsf(r) + fabsf(g) + fabsf(bl));
        }
    }
    tmax = warp_max_f(tmax);
    if (lane == 0) atomicMax(&s_tmax, __float_as_uint(tmax));  // non-negative floats order as their bits
    for (int q = warp; q < ni * nj; q += nw) {  // Eq. 9 flags
        const int i = q / nj, j = q - i * nj;
        const int green = a.C == 3 ? gcp_green_fast(a.img, a.W, HW, ya + 4 * i, xa + 4 * j, a.gamma, lane) : 1;
        if (lane == 0) {
            if (a.green) a.green[(size_t)(gy0 + i) * a.nx + gx0 + j] = (uint8_t)green;
            atomicOr(&s_use[green ? 0 : 1][i], 1u << j);
        }
    }
    __syncthreads();
    const float T3 = __uint_as_float(s_tmax);
    // ---- this thread's offsets: row ky (dy = ky - R), columns 4 g .. 4 g + 3
    const int ky = tid / c.G, g = tid - ky * c.G;
    const bool item = ky <= 2 * a.R;
    unsigned vt = 0u;  // its offsets inside the window, without the reference itself
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int dx = 4 * g + t - c.R4;
        if (item && dx >= -a.R && dx <= a.R && !(ky == a.R && dx == 0)) vt |= 1u << t;
    }
    const int wrow = 4 * c.G;
    for (int pass = 0; pass < npl; ++pass) {
        unsigned used = 0u;  // rows with a reference of this plane
        for (int i = 0; i < ni; ++i) used |= s_use[pass][i] ? 1u << i : 0u;
        if (!used) continue;
        const float *pa = plane0 + (size_t)pass * c.rows * rw + a.R * rw + c.R4;
        const float *pb = plane0 + (size_t)pass * c.rows * rw + (item ? ky * rw + 4 * g : 0);
        Bound bd;
        bd.eps = CEPS;
        bd.beta = pass == 0 ? 0.f : 72.f * U32 * T3;
        bd.g0 = (pass == 0 ? 0.f : 1200.f * U32 * U32 * T3 * T3) + 1e-30f;
        float4 hp[CX];  // the previous cell row's horizontal pairs
#pragma unroll
        for (int j = 0; j < CX; ++j) hp[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int cr = 0; cr <= ni; ++cr) {
            if (!(((used << 1) | used) >> cr & 1u)) continue;  // no reference of rows cr - 1, cr needs this cell row
            const bool emit = cr > 0 && (used >> (cr - 1) & 1u);
            const int cy = ya + 4 * (cr - 1) + ky - a.R;
            const unsigned vr = (cy >= 0 && cy <= a.H - PS) ? vt : 0u;
            if (item) {
                // the cells' sums, pixel row by pixel row (the rows rolled: unrolled, the loop outgrew the instruction
                // cache), the candidate pieces sliding through registers
                float s[CX + 1][4] = {};
#pragma unroll 1
                for (int u = 0; u < 4; ++u) {
                    const float4 *ra = reinterpret_cast<const float4 *>(pa + (4 * cr + u) * rw);
                    const float4 *rb = reinterpret_cast<const float4 *>(pb + (4 * cr + u) * rw);
                    float4 bl = rb[0];
#pragma unroll
                    for (int k = 0; k <= CX; ++k) {  // (all of them: a branch per cell would serialise the chains)
                        const float4 av = ra[k], bh = rb[k + 1];
                        const float aa[4] = {av.x, av.y, av.z, av.w};
                        const float bb[8] = {bl.x, bl.y, bl.z, bl.w, bh.x, bh.y, bh.z, bh.w};
#pragma unroll
                        for (int v = 0; v < 4; ++v)
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const float e = __fsub_rn(aa[v], bb[v + t]);
                                s[k][t] = __fmaf_rn(e, e, s[k][t]);
                            }
                        bl = bh;
                    }
                }
#pragma unroll
                for (int j = 0; j < CX; ++j) {
                    if (j >= nj) break;
                    const float4 h = make_float4(s[j][0] + s[j + 1][0], s[j][1] + s[j + 1][1], s[j][2] + s[j + 1][2],
                                                 s[j][3] + s[j + 1][3]);
                    if (emit) {
                        const float inf = __int_as_float(0x7f800000);
                        const int cx = xa + 4 * j + 4 * g - c.R4;  // the candidates' columns
                        float4 d;
                        d.x = (vr & 1u) && cx >= 0 && cx <= a.W - PS ? hp[j].x + h.x : inf;
                        d.y = (vr & 2u) && cx + 1 >= 0 && cx + 1 <= a.W - PS ? hp[j].y + h.y : inf;
                        d.z = (vr & 4u) && cx + 2 >= 0 && cx + 2 <= a.W - PS ? hp[j].z + h.z : inf;
                        d.w = (vr & 8u) && cx + 3 >= 0 && cx + 3 <= a.W - PS ? hp[j].w + h.w : inf;
                        *reinterpret_cast<float4 *>(dbuf + j * c.ncp + ky * wrow + 4 * g) = d;
                    }
                    hp[j] = h;
                }
            }
            if (!emit) continue;
            __syncthreads();
            // ---- the row's references of this plane, a warp each
            const unsigned use = s_use[pass][cr - 1];
            for (int j = warp; j < nj; j += nw) {
                if (!(use >> j & 1u)) continue;
                float *db = dbuf + j * c.ncp;
                const int r = (gy0 + cr - 1) * a.nx + gx0 + j, yr = ya + 4 * (cr - 1), xr = xa + 4 * j;
                int32_t *out = a.idx + (size_t)r * K;
                if (lane == 0) out[0] = yr * a.W + xr;
                // the reference's distances, once spent, make room for the sorted candidates
                const CandList cl(list, db);
                const int nch = (wrow * (2 * a.R + 1) + 31) >> 5;
                // entry i of this lane: 32 i + ((lane + 7 i) mod 32), so that neighbouring rows' equal dx differ in lane
                float m1 = __int_as_float(0x7f800000), m2 = m1;
#pragma unroll 8
                for (int i = 0; i < nch; ++i) {
                    const float v = db[32 * i + ((lane + 7 * i) & 31)];
                    if (LT == 2) m2 = fminf(m2, fmaxf(m1, v));
                    m1 = fminf(m1, v);
                }
                // a bound on the (K-1)-th distance: the (K-1)-th smallest of the lanes' minima (K = 16: 19 candidates
                // lie under it on average), or of their two smallest (K = 32: 33; one alone would give 71) -- the K-1
                // smallest of two ascending lists are min(A[i], B[K-2-i])
                const float A = warp_sort(m1, lane);
                float tau;
                if (LT == 1) {
                    tau = __shfl_sync(FULL, A, K - 2);
                } else {
                    const float bo = __shfl_sync(FULL, warp_sort(m2, lane), lane < K - 1 ? K - 2 - lane : 0);
                    tau = __uint_as_float(__reduce_max_sync(FULL, lane < K - 1 ? __float_as_uint(fminf(A, bo)) : 0u));
                }
                float T = bd.upper(bd.upper(tau));
                unsigned hit = 0u;
                int m = 0;
                float lo = 0.f;
                for (int it = 0;; ++it) {
                    hit = 0u;
#pragma unroll 8
                    for (int i = 0; i < nch; ++i) hit |= (db[32 * i + ((lane + 7 * i) & 31)] <= T ? 1u : 0u) << i;
                    m = __reduce_add_sync(FULL, __popc(hit));
                    if (m <= PMAX || it >= 24 || !(T < 3e38f)) break;
                    // too many: halve the bound as long as it keeps K - 1 candidates
                    int n = 0;
                    float mid;
                    for (;; ++it) {
                        mid = 0.5f * (lo + tau);
                        n = 0;
                        for (int i = 0; i < nch; ++i) n += db[32 * i + lane] <= mid ? 1 : 0;
                        n = __reduce_add_sync(FULL, n);
                        if (n >= K - 1 || it >= 24) break;
                        lo = mid;
                    }
                    if (n < K - 1) break;
                    tau = mid;
                    T = bd.upper(bd.upper(tau));
                }
                if (m > PMAX || m < K - 1 || !(T < 3e38f)) {  // the exhaustive FP64 pass
                    if (lane == 0) a.fb[atomicAdd(&a.st->match_fallback, 1)] = r;
                    continue;
                }
                int pos = __popc(hit);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(FULL, pos, o);
                    if (lane >= o) pos += v;
                }
                pos -= __popc(hit);
                for (; hit; hit &= hit - 1) {
                    const int i = __ffs(hit) - 1, e = 32 * i + ((lane + 7 * i) & 31), ey = e / wrow;
                    cl.d[pos] = db[e];
                    cl.i[pos++] = (yr + ey - a.R) * a.W + xr + (e - ey * wrow) - c.R4;
                }
                __syncwarp();
                const int mp = settle_group<K>(bd, cl, m, lane, out);
                if (mp) {  // FP64 is slow and its warp would hold up the row: kept for the end of the tile
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_ndefer, 1);
                    at = __shfl_sync(FULL, at, 0);
                    if (at < NDEFER) {
                        for (int i = lane; i < mp; i += 32) defer[at * PMAX + i] = cl.si[i];
                        if (lane == 0) s_defer[at] = make_int4(r, yr * a.W + xr, mp, pass == 0 ? 1 : 0);
                    } else {
                        rerank_group<K>(a, cl.si, cl.d64, mp, yr, xr, pass == 0 ? 1 : 0, lane, out);
                    }
                }
                __syncwarp();
                for (int e = wrow * (2 * a.R + 1) + lane; e < c.ncp; e += 32) db[e] = __int_as_float(0x7f800000);
            }
            __syncthreads();
        }
    }
    for (int e = warp; e < min(s_ndefer, NDEFER); e += nw) {  // the last barrier was the last row's
        const int4 f = s_defer[e];
        rerank_group<K>(a, defer + e * PMAX, reinterpret_cast<double *>(list), f.z, f.y / a.W, f.y % a.W, f.w, lane,
                        a.idx + (size_t)f.x * K);
        __syncwarp();
    }
}

// Offsets (threads) of the cell matcher's window.
inline int cell_groups(int R, int *R4) {
    *R4 = (R + 3) / 4 * 4;
    return (*R4 + R + 4) / 4;
}

template <int K>
hts_status launch_cells(const MatchArgs &a, cudaStream_t s) {
    CellArgs c{};
    c.m = a;
    c.G = cell_groups(a.R, &c.R4);
    const int items = (2 * a.R + 1) * c.G;
    const int threads = std::max(64, (items + 31) / 32 * 32);
    c.ry = (a.H - PS) / 4 + 1;
    c.rx = (a.W - PS) / 4 + 1;
    c.ntx = (c.rx + CX - 1) / CX;
    c.ncp = std::max((items * 4 + 31) / 32 * 32, CandList::SCRATCH / 4);
    c.cols = 4 * (CX + 1) + 4 * c.G;
    auto smem_of = [&](int nry) {
        return ((size_t)(a.C == 3 ? 2 : 1) * (4 * (nry + 1) + 2 * a.R) * c.cols + (size_t)CX * c.ncp) * sizeof(float) +
               (size_t)(threads / 32) * CandList::LIST;
    };
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // rows per tile: more share cells (n rows of references need n + 1 cell rows) but leave fewer blocks, and an SM
    // needs its 16 resident warps (the registers' limit) to hide a block's latencies: the work of a block, in thousands
    // of warp instructions (a cell row 1.4 per warp, a row of references settled 4, the staging 2 per 3000 values), times
    // the blocks of an SM and half a round of resident ones for the uneven end, or one round where they are fewer (no
    // uneven end where only two are resident and all are: 512 x 512 x 3, win 31, seven rows a tile 150 us, four 169).
    // With the blocks counted as if an SM ran them one by one, small windows (two to four warps a block) got tiles
    // whose blocks left the SMs idle: 301 x 417 gray, K = 16, win 9: 104 us, now 46; 512 x 640 x 3, K = 32, win 15:
    // 311 us, now 167.  Over 96 x 128 to 768 x 1024, K = 4 to 32 and windows 5 to 31 the choice is 2 % off the best.
    const double resident = 512.0 / threads;
    double best = 0.0;
    for (int n = 8; n >= 1; --n) {
        const long blocks = (long)c.ntx * ((c.ry + n - 1) / n);
        const double per_sm = (double)blocks / nsm;
        const double round = resident <= 2.0 && per_sm <= resident ? resident : std::max(resident, per_sm + 0.5 * resident);
        const double w = round *
                         ((n + 1) * 1.4 * (threads / 32) + n * 4.0 +
                          (a.C == 3 ? 2 : 1) * (4 * (n + 1) + 2 * a.R) * c.cols * (2.0 / 3000.0));
        if (best == 0.0 || w < best) {
            best = w;
            c.nry = n;
        }
    }
    c.nty = (c.ry + c.nry - 1) / c.nry;
    c.rows = 4 * (c.nry + 1) + 2 * a.R;
    const int blocks = c.ntx * c.nty + (a.nx > c.rx ? c.nty : 0) + (a.ny > c.ry ? c.ntx : 0) +
                       (a.nx > c.rx && a.ny > c.ry ? 1 : 0);
    const hts_status st0 = allow_smem(reinterpret_cast<const void *>(k_match_cells<K>), smem_of(c.nry));
    if (st0 != HTS_OK) return st0;
    {
        KTimer kt("k_match", s);
        k_match_cells<K><<<blocks, threads, smem_of(c.nry), s>>>(c);
    }
    return check_launch("k_match");
}

// Exhaustive FP64 matching of the references listed by k_match.
template <int K>
__global__ void __launch_bounds__(128) k_match_fallback(MatchArgs a) {
    constexpr int L = K - 1;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int count = *(volatile int *)&a.st->match_fallback;
    const size_t HW = (size_t)a.H * a.W;
    for (int f = gw; f < count; f += nw) {
        const int r = a.fb[f];
        const int yr = grid_pos(r / a.nx, a.H, a.step), xr = grid_pos(r % a.nx, a.W, a.step);
        const int green = (a.C == 3) ? gcp_green(a.img, a.W, HW, yr, xr, a.gamma, lane) : 1;
        const int cy0 = max(0, yr - a.R), cy1 = min(a.H - PS, yr + a.R);
        const int cx0 = max(0, xr - a.R), cx1 = min(a.W - PS, xr + a.R);
        const int ncol = cx1 - cx0 + 1, ncand = (cy1 - cy0 + 1) * ncol;
        double dl[L];
        int il[L];
#pragma unroll
        for (int i = 0; i < L; ++i) {
            dl[i] = __longlong_as_double(0x7ff0000000000000ll);  // +inf
            il[i] = 0x7fffffff;
        }
        for (int c = lane; c < ncand; c += 32) {
            const int cy = cy0 + c / ncol, cx = cx0 + c % ncol;
            if (cy == yr && cx == xr) continue;
            const double D = exact_dist(a.img, a.W, HW, a.C, green, yr, xr, cy, cx);
            const int id = cy * a.W + cx;
            if (D > dl[L - 1] || (D == dl[L - 1] && id > il[L - 1])) continue;
            // insertion keeping (D, id) ascending
#pragma unroll
            for (int i = L - 1; i > 0; --i) {
                const bool shift = (dl[i - 1] > D) || (dl[i - 1] == D && il[i - 1] > id);
                const bool here = !shift && ((dl[i] > D) || (dl[i] == D && il[i] > id));
                if (shift) { dl[i] = dl[i - 1]; il[i] = il[i - 1]; }
                else if (here) { dl[i] = D; il[i] = id; }
            }
            if ((dl[0] > D) || (dl[0] == D && il[0] > id)) { dl[0] = D; il[0] = id; }
        }
        int32_t *out = a.idx + (size_t)r * K;
        if (lane == 0) out[0] = yr * a.W + xr;
        for (int j = 0; j < L; ++j) {
            double bd = dl[0];
            int bi = il[0];
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                const double od = __shfl_xor_sync(FULL, bd, o);
                const int oi = __shfl_xor_sync(FULL, bi, o);
                if (od < bd || (od == bd && oi < bi)) { bd = od; bi = oi; }
            }
            // no candidate left with a distance (NaN pixels): the reference itself, a valid patch
            if (lane == 0) out[1 + j] = bi == 0x7fffffff ? yr * a.W + xr : bi;
            if (il[0] == bi && dl[0] == bd) {
#pragma unroll
                for (int q = 0; q < L - 1; ++q) { dl[q] = dl[q + 1]; il[q] = il[q + 1]; }
                dl[L - 1] = __longlong_as_double(0x7ff0000000000000ll);
                il[L - 1] = 0x7fffffff;
            }
        }
    }
}

// Exhaustive matching, in FP32, of the references the tensor-core matcher listed in a.fb (count in
// a.st->match_fallback): distances as FP32 fused multiply-adds in the definition's (u, v) order on the FP32 plane
// ((R + G) + B for the channel sum) -- the arithmetic of the tensor-core matcher's re-rank -- and the K-1 nearest by
// (distance, raster index).  The matching plane comes from a.green (Eq. 9 flags already decided).  A few references
// in a thousand on most images, over half of them on images full of gratings, whose equally good candidates crowd the
// matcher's bins.  One warp per reference: the region staged in shared memory, four consecutive candidates per lane
// and item with the reference in registers (three 16-byte loads of candidates, conflict-free, for 64 operations),
// distances to shared memory, then the bound from the lanes' minima and a sort of the few candidates under it.
// Bound by FP32 issue.  Before (a block per reference, two loads per pixel and candidate, per-thread insertion lists
// merged by one thread): 27 references / us at 1536 x 2048 x 3, now 96.
constexpr unsigned NONE = 0xffffffffu;  // no candidate: above every distance's bits
constexpr int RW = 4;                   // warps per block

struct RescueShape {
    int R4, G, cols, rows, ncp;  // as CellArgs; ncp: candidates, padded to whole chunks of 32
    __host__ __device__ explicit RescueShape(int R)
        : R4((R + 3) / 4 * 4), G((R4 + R + 4) / 4), cols(4 * G + 8), rows(2 * R + PS),
          ncp(((2 * R + 1) * 4 * G + 31) / 32 * 32) {}
    __host__ __device__ size_t floats() const { return (size_t)cols * rows + ncp + 4 * PMAX; }  // per warp
};

__device__ __forceinline__ unsigned warp_sort_u(unsigned v, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j; j >>= 1) {
            const unsigned o = __shfl_xor_sync(FULL, v, j);
            const bool up = (lane & k) == 0, low = (lane & j) == 0;
            v = (up == low) ? min(v, o) : max(v, o);
        }
    return v;
}

template <int K>
__global__ void __launch_bounds__(RW * 32) k_match_rescue(MatchArgs a) {
    constexpr int L = K - 1;
    constexpr int LT = K <= 16 ? 1 : 2;  // smallest distances of a lane that enter the bound (as k_match_cells)
    extern __shared__ __align__(16) float rs_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int count = *(volatile int *)&a.st->match_fallback;
    const size_t HW = (size_t)a.H * a.W;
    const RescueShape S(a.R);
    float *plane = rs_smem + warp * S.floats();                                // [rows][cols]
    unsigned *db = reinterpret_cast<unsigned *>(plane + S.cols * S.rows);      // [ncp] distances' bits, raster order
    unsigned *cd = db + S.ncp;                                                 // [PMAX] collected distances
    int *ci = reinterpret_cast<int *>(cd + PMAX), *si = ci + PMAX;             // and indices; sorted indices
    const int wrow = 4 * S.G, items = (2 * a.R + 1) * S.G, nch = S.ncp / 32;
    const unsigned below = (1u << lane) - 1u;
    for (int f = blockIdx.x * RW + warp; f < count; f += gridDim.x * RW) {
        const int r = a.fb[f];
        const int yr = grid_pos(r / a.nx, a.H, a.step), xr = grid_pos(r % a.nx, a.W, a.step);
        const int green = (a.C == 3) ? (int)a.green[r] : 1;
        const int y0 = yr - a.R, x0 = xr - S.R4;
        __syncwarp();  // the previous reference's values are read
        {  // the region, 16 elements in flight per lane (columns and rows advanced by 32 elements, no divisions)
            const bool one = a.C == 1 || green;  // the plane is one channel
            const float *ch = a.img + (a.C == 3 && green ? HW : 0);
            const int dq = 32 / S.cols, dr = 32 - dq * S.cols;
            int x = x0 + lane % S.cols, y = y0 + lane / S.cols;
            for (int e0 = lane; e0 < S.rows * S.cols; e0 += 16 * 32) {
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const bool in = e0 + 32 * i < S.rows * S.cols && y >= 0 && y < a.H && x >= 0 && x < a.W;
                    const size_t o = in ? (size_t)y * a.W + x : 0;
                    v[i] = in ? __ldg(ch + o) : 0.f;
                    if (!one && in) v[i] = (v[i] + __ldg(a.img + HW + o)) + __ldg(a.img + 2 * HW + o);
                    x += dr;
                    y += dq;
                    if (x >= x0 + S.cols) {
                        x -= S.cols;
                        ++y;
                    }
                }
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (e0 + 32 * i < S.rows * S.cols) plane[e0 + 32 * i] = v[i];
            }
        }
        __syncwarp();
        float ar[NPIX];
#pragma unroll
        for (int e = 0; e < NPIX; e += 4)
            *reinterpret_cast<float4 *>(ar + e) =
                *reinterpret_cast<const float4 *>(plane + (a.R + (e >> 3)) * S.cols + S.R4 + (e & 7));
        unsigned m1 = NONE, m2 = NONE;  // this lane's two smallest
        for (int it = lane; it < S.ncp / 4; it += 32) {
            uint4 d = make_uint4(NONE, NONE, NONE, NONE);
            if (it < items) {
                const int ky = it / S.G, g = it - ky * S.G;
                const float *row = plane + ky * S.cols + 4 * g;
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int u = 0; u < PS; ++u) {
                    float b[12];
#pragma unroll
                    for (int i = 0; i < 12; i += 4)
                        *reinterpret_cast<float4 *>(b + i) = *reinterpret_cast<const float4 *>(row + u * S.cols + i);
#pragma unroll
                    for (int v = 0; v < PS; ++v)
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const float e = ar[u * PS + v] - b[v + t];
                            acc[t] = fmaf(e, e, acc[t]);
                        }
                }
                const int cy = y0 + ky, cx = x0 + 4 * g, dx = 4 * g - S.R4;
                const bool rowok = cy >= 0 && cy <= a.H - PS;
                unsigned *dv = &d.x;
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (rowok && cx + t >= 0 && cx + t <= a.W - PS && dx + t >= -a.R && dx + t <= a.R &&
                        !(ky == a.R && dx + t == 0))
                        dv[t] = __float_as_uint(acc[t]);
            }
            *reinterpret_cast<uint4 *>(db + 4 * it) = d;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const unsigned v = (&d.x)[t];
                if (LT == 2) m2 = min(m2, max(m1, v));
                m1 = min(m1, v);
            }
        }
        __syncwarp();
        // a bound on the L-th distance: the L-th smallest of the lanes' smallest (K = 32: of their two smallest; of
        // two ascending lists the L smallest are min(A[i], B[L-1-i]))
        const unsigned A = warp_sort_u(m1, lane);
        unsigned T;
        if (LT == 1) {
            T = __shfl_sync(FULL, A, L - 1);
        } else {
            const unsigned bo = __shfl_sync(FULL, warp_sort_u(m2, lane), lane < L ? L - 1 - lane : 0);
            T = __reduce_max_sync(FULL, lane < L ? min(A, bo) : 0u);
        }
        // candidates below T and, in raster order, at T; more than the list holds (ties, a clustered bound): the exact
        // L-th distance by bisection, of which only the first ones in raster order can belong to the group
        int m = 0, nless = 0;
        for (int pass = 0; pass < 2; ++pass) {
            m = nless = 0;
            int cap = PMAX;  // of the candidates at T
            if (pass == 1) {
                // lo <= the L-th distance <= hi, both among the distances (so that ties, the common case, take few
                // rounds: bisecting the bits took 31), until the list holds all up to hi, or lo and hi meet
                unsigned lo = __shfl_sync(FULL, A, 0), hi = T;
                while (lo < hi) {
                    const unsigned mid = lo + (hi - lo) / 2;
                    int n = 0;
                    unsigned below = 0u, above = NONE;
#pragma unroll 8
                    for (int i = 0; i < nch; ++i) {
                        const unsigned v = db[32 * i + lane];
                        n += v <= mid ? 1 : 0;
                        below = max(below, v <= mid ? v : 0u);
                        above = min(above, v <= mid ? NONE : v);
                    }
                    n = __reduce_add_sync(FULL, n);
                    if (n >= L) hi = __reduce_max_sync(FULL, below);
                    else lo = __reduce_min_sync(FULL, above);
                    if (n >= L && n <= PMAX) break;
                }
                T = hi;
                int n = 0;
#pragma unroll 8
                for (int i = 0; i < nch; ++i) n += db[32 * i + lane] < T ? 1 : 0;
                n = __reduce_add_sync(FULL, n);
                if (n < L) cap = L - n;  // else the list holds them all
            }
            for (int i = 0; i < nch; ++i) {
                const int e = 32 * i + lane;
                const unsigned v = db[e];
                const bool at = v == T && v != NONE;
                const unsigned eq = __ballot_sync(FULL, at);
                const bool ok = v < T || (at && nless + __popc(eq & below) < cap);
                const unsigned msk = __ballot_sync(FULL, ok);
                const int pos = m + __popc(msk & below);
                if (ok && pos < PMAX) {
                    const int ky = e / wrow;
                    cd[pos] = v;
                    ci[pos] = (y0 + ky) * a.W + x0 + (e - ky * wrow);
                }
                m += __popc(msk);
                nless += __popc(eq);  // candidates at T so far
            }
            if (m <= PMAX) break;
        }
        __syncwarp();
        // ranks by (distance, raster index): the collected entries are in raster order, so an equal distance ranks
        // behind the ones collected before it
        const unsigned d0 = lane < m ? cd[lane] : NONE, d1 = lane + 32 < m ? cd[lane + 32] : NONE;
        int r0 = 0, r1 = 0;
        for (int j = 0; j < m; ++j) {
            const unsigned v = cd[j];
            r0 += (v < d0 || (v == d0 && j < lane)) ? 1 : 0;
            r1 += (v < d1 || (v == d1 && j < lane + 32)) ? 1 : 0;
        }
        if (lane < m) si[r0] = ci[lane];
        if (lane + 32 < m) si[r1] = ci[lane + 32];
        __syncwarp();
        int32_t *out = a.idx + (size_t)r * K;
        if (lane < K) out[lane] = lane == 0 || lane > m ? yr * a.W + xr : si[lane - 1];
    }
}

// k_match: one reference per warp.
template <int K>
hts_status launch_direct(const MatchArgs &a, cudaStream_t s) {
    const int RHM = a.step + 2 * a.R + PS;
    const int NCM = (2 * a.R + 1) * (2 * a.R + 1);
    const size_t smem = (size_t)MW * (CandList::LIST + CandList::SCRATCH) + (size_t)(a.C == 3 ? 2 : 1) * RHM * RHM * sizeof(float) +
                        (size_t)MW * NCM * sizeof(float);
    {
        const hts_status st0 = allow_smem(reinterpret_cast<const void *>(k_match<K>), smem);
        if (st0 != HTS_OK) return st0;
    }
    const int blocks = ((a.ny + 1) / 2) * ((a.nx + 1) / 2);
    {
        KTimer kt("k_match", s);
        k_match<K><<<blocks, MW * 32, smem, s>>>(a);
    }
    return check_launch("k_match");
}

// Whether the cell matcher takes a call at step 4 (windows whose offsets fit a block's threads: R <= 15).  Its blocks
// settle rows of eight references in turn, so small grids leave it few warps, and a small window's distances, which
// it halves, are the smaller part; the lines lie where a reference per warp (k_match) took as long (us, cells / k_match,
// both with k_match_fallback; K = 16 where not given): 96 x 128 x 3 (713 references), win 15: 67 / 53; 203 x 317 x 3
// (3950): 77 / 66, gray 44 / 46; 301 x 417 x 3 (7800): 76 / 86; 203 x 317 x 3, win 19: 68 / 73; 96 x 128 gray, win 21:
// 38 / 40, colour 63 / 58; 512 x 640 gray (20193), K = 8, win 5: 83 / 71; 1080 x 1920 (128851), win 5: 0.83 to 0.89 of
// k_match's time on gray, the same on colour.  At K = 32 k_match leaves most references of a wide window to the
// exhaustive pass (96 x 128 gray, win 31: 41 / 543).
inline bool cells_faster(int K, int C, int R, int nref) {
    int R4;
    if ((2 * R + 1) * cell_groups(R, &R4) > CT || (C == 3 && R <= 2)) return false;
    int need = R <= 3 ? 40000 : R <= 7 ? 7000 : R <= 9 || C == 3 ? 3000 : 500;
    if (K == 32 && R >= 13) need = 500;
    return nref >= (K == 2 ? 2 * need : need);
}

template <int K>
hts_status launch_k(const MatchArgs &a, cudaStream_t s) {
    const bool cells = a.step == 4 && cells_faster(K, a.C, a.R, a.nref);
    const hts_status st = cells ? launch_cells<K>(a, s) : launch_direct<K>(a, s);
    if (st != HTS_OK) return st;
    {
        KTimer kt("k_match_fallback", s);
        k_match_fallback<K><<<152, 128, 0, s>>>(a);
    }
    return check_launch("k_match_fallback");
}

// Eq. 9 flag of every reference patch, for the tensor-core matching path, which reads the flags instead of
// deciding them itself: two references per warp (a half-warp each, four pixels of the 8 x 8 patch per lane),
// the FP32 screen of gcp_green_fast (the same sums in another order, inside the same margin), and the FP64
// decision by the whole warp for a reference the screen leaves open.
__global__ void __launch_bounds__(128) k_gcp_flags(const float *__restrict__ img, int H, int W, int step, int nx,
                                                   int nref, double gamma, uint8_t *__restrict__ green) {
    const int lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15;
    const size_t HW = (size_t)H * W;
    const int nwarp = (gridDim.x * blockDim.x) >> 5;
    for (int r0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 2; r0 < nref; r0 += 2 * nwarp) {
        const int r = min(r0 + half, nref - 1);  // the last odd reference is decided twice, identically
        const int gy = r / nx, gx = r - gy * nx;
        const int yr = grid_pos(gy, H, step), xr = grid_pos(gx, W, step);
        float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = hl + 16 * q;
            const size_t o = (size_t)(yr + (e >> 3)) * W + xr + (e & 7);
            const float rv = __ldg(img + o), gv = __ldg(img + HW + o), bv = __ldg(img + 2 * HW + o);
            s0 = fmaf(rv, rv, s0);
            s1 = fmaf(gv, gv, s1);
            s2 = fmaf(bv, bv, s2);
        }
#pragma unroll
        for (int o = 8; o; o >>= 1) {
            s0 += __shfl_xor_sync(FULL, s0, o);
            s1 += __shfl_xor_sync(FULL, s1, o);
            s2 += __shfl_xor_sync(FULL, s2, o);
        }
        const float lhs = s1 * (float)(gamma * gamma), rhs = fmaxf(s0, s2);
        int flag = -1;  // -1: open
        if (lhs > rhs * (1.f + 1e-5f) && lhs > 0.f) flag = 1;
        else if (lhs < rhs * (1.f - 1e-5f)) flag = 0;
        const unsigned open = __ballot_sync(FULL, flag < 0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (open & (1u << (16 * h))) {  // the whole warp decides reference r0 + h in FP64
                const int rh = min(r0 + h, nref - 1);
                const int gyh = rh / nx, gxh = rh - gyh * nx;
                const int f = gcp_green(img, W, HW, grid_pos(gyh, H, step), grid_pos(gxh, W, step), gamma, lane);
                if (half == h) flag = f;
            }
        }
        if (hl == 0 && r0 + half < nref) green[r] = (uint8_t)flag;
    }
}

}  // namespace

hts_status launch_gcp_flags(const float *img, const Geom &g, double gamma_gcp, uint8_t *green, cudaStream_t s) {
    int blocks = (g.nref + 7) / 8;  // four warps of two references
    if (blocks > 152 * 16) blocks = 152 * 16;
    {
        KTimer kt("k_gcp_flags", s);
        k_gcp_flags<<<blocks, 128, 0, s>>>(img, g.H, g.W, g.step, g.nx, g.nref, gamma_gcp, green);
    }
    return check_launch("k_gcp_flags");
}

hts_status launch_match(const float *img, const Geom &g, double gamma_gcp, int32_t *idx, uint8_t *green,
                        int32_t *fallback_list, DevState *st, cudaStream_t s) {
    MatchArgs a;
    a.img = img;
    a.H = g.H;
    a.W = g.W;
    a.C = g.C;
    a.step = g.step;
    a.R = g.R;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nref = g.nref;
    a.gamma = gamma_gcp;
    a.idx = idx;
    a.green = green;
    a.fb = fallback_list;
    a.st = st;
    switch (g.K) {
        case 2: return launch_k<2>(a, s);
        case 4: return launch_k<4>(a, s);
        case 8: return launch_k<8>(a, s);
        case 16: return launch_k<16>(a, s);
        case 32: return launch_k<32>(a, s);
        default: return HTS_EUNSUPPORTED;
    }
}

hts_status launch_match_rescue(const float *img, const Geom &g, int32_t *idx, const uint8_t *green,
                               int32_t *fallback_list, DevState *st, cudaStream_t s) {
    MatchArgs a;
    a.img = img;
    a.H = g.H;
    a.W = g.W;
    a.C = g.C;
    a.step = g.step;
    a.R = g.R;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nref = g.nref;
    a.gamma = 0.0;
    a.idx = idx;
    a.green = const_cast<uint8_t *>(green);
    a.fb = fallback_list;
    a.st = st;
    const size_t smem = RW * RescueShape(g.R).floats() * sizeof(float);
    const void *fn = nullptr;
    switch (g.K) {
        case 2: fn = reinterpret_cast<const void *>(k_match_rescue<2>); break;
        case 4: fn = reinterpret_cast<const void *>(k_match_rescue<4>); break;
        case 8: fn = reinterpret_cast<const void *>(k_match_rescue<8>); break;
        case 16: fn = reinterpret_cast<const void *>(k_match_rescue<16>); break;
        case 32: fn = reinterpret_cast<const void *>(k_match_rescue<32>); break;
        default: return HTS_EUNSUPPORTED;
    }
    {
        const hts_status st0 = allow_smem(fn, smem);
        if (st0 != HTS_OK) return st0;
    }
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // four blocks an SM: resident together at windows up to 31 (44 KB of shared memory each); wider ones take fewer at
    // a time, down to one at 63 (149 KB), where the pass still takes no longer than with a block per reference
    // (400 x 400, step 1, win 63, 1187 references: 118 us, 147)
    const int blocks = 4 * nsm;
    {
        KTimer kt("k_match_rescue", s);
        switch (g.K) {
            case 2: k_match_rescue<2><<<blocks, RW * 32, smem, s>>>(a); break;
            case 4: k_match_rescue<4><<<blocks, RW * 32, smem, s>>>(a); break;
            case 8: k_match_rescue<8><<<blocks, RW * 32, smem, s>>>(a); break;
            case 16: k_match_rescue<16><<<blocks, RW * 32, smem, s>>>(a); break;
            default: k_match_rescue<32><<<blocks, RW * 32, smem, s>>>(a); break;
        }
    }
    return check_launch("k_match_rescue");
}

}  // namespace hts
