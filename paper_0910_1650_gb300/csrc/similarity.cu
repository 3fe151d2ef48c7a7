// ap_similarity: s(i,k) = -||x_i - x_k||^2 (Section 2) with the preferences
// p(k) on the diagonal (Algorithm 1 input) and the optional tie-break noise.
//
// Pipeline (all on the caller's stream, scratch in the caller's workspace):
//   1. column means of X in float64 (fixed-order two-stage reduction);
//   2. centred copy Xc = X - mean (float32, or bf16 for the tensor-core path),
//      zero padded to whole tiles, and squared norms of the centred rows
//      (of the bf16-rounded rows for the tensor-core path);
//   3. S = 2 Xc Xc^T - |x_i|^2 - |x_k|^2 clamped to <= 0 (SIMT float32 GEMM
//      here, tcgen05 GEMM in tc_gemm.cu);
//   4. preference: exact median of the n(n-1) off-diagonal values, both middle
//      order statistics at once, on order-preserving 32-bit keys: a sampled
//      bracket, one pass over S, and radix digits over what it encloses;
//   5. diagonal <- p, then s <- s + noise_rel*|s|*u(i,k) on every entry.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <map>
#include <array>
#include <climits>
#include <cmath>

#include <cuda_bf16.h>

#include <vector>

#include "common.cuh"

namespace apgb {

int32_t tc_similarity_bf16(const __nv_bfloat16* Xb, const float* nrm, int n, int dpad,
                           float* S, int64_t lds, int32_t* err, cudaStream_t s);
size_t tc_grouped_table_bytes(const int64_t* n, int32_t count);
int32_t tc_similarity_bf16_grouped(const __nv_bfloat16* Xb, const float* nrm, int64_t rows, int dpad,
                                   const int64_t* n, const int64_t* roff, float* const* S,
                                   const int64_t* lds, int32_t count, void* tables, int32_t* err,
                                   cudaStream_t s);
size_t tc_similarity_pad_rows();

// ---- 1. column means -----------------------------------------------------------
// Column sums of X over blocks of `rows` rows, bound by reading X.  Block: 32
// column lanes x 8 row lanes; row lane y sums rows y, y+8, ... of the row
// block, and the 8 lane sums are added in a fixed tree (deterministic).  VEC
// (X 16-byte aligned, ldx % 4 == 0): a column lane owns four columns and reads
// 16 bytes a row (10^6 x 128: 90 us where 4-byte loads took 119 us); else
// one.  A column's sum is the same bits either way.  Grid: (ceil(d / 32 or
// 128), ceil(n/rows)).  part[row block][j].
constexpr int kMeanRows = 256;

// One block of the column sums: column group bx, row block by.
template <bool VEC>
__device__ __forceinline__ void colsum_block(const float* __restrict__ X, int64_t n, int d, int64_t ldx,
                                             int64_t rows, double* part, int bx, int by) {
    constexpr int W = VEC ? 4 : 1;
    const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
    const int j = (bx * 32 + cx) * W;
    const int64_t r0 = (int64_t)by * rows;
    const int64_t r1 = min(n, r0 + rows);
    __shared__ double ps[8][32 * W];
    // Neumaier-compensated float32 sum of the lane's rows (float64 arithmetic is
    // scarce on this part); (s, c) carries the sum to well below float32 rounding
    float sm[W], cm[W];
#pragma unroll
    for (int e = 0; e < W; ++e) sm[e] = cm[e] = 0.f;
    auto add = [&](int e, float x) {
        const float t = sm[e] + x;
        cm[e] += (fabsf(sm[e]) >= fabsf(x)) ? (sm[e] - t) + x : (x - t) + sm[e];
        sm[e] = t;
    };
    if (VEC && j + 3 < d) {
#pragma unroll 8
        for (int64_t i = r0 + ry; i < r1; i += 8) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(X + i * ldx + j));
            add(0, x.x);
            add(W > 1 ? 1 : 0, x.y);
            add(W > 2 ? 2 : 0, x.z);
            add(W > 3 ? 3 : 0, x.w);
        }
    } else if (j < d) {
        for (int e = 0; e < W && j + e < d; ++e) {
            float s1 = 0.f, c1 = 0.f;
#pragma unroll 8
            for (int64_t i = r0 + ry; i < r1; i += 8) {
                const float x = X[i * ldx + j + e];
                const float t = s1 + x;
                c1 += (fabsf(s1) >= fabsf(x)) ? (s1 - t) + x : (x - t) + s1;
                s1 = t;
            }
#pragma unroll
            for (int q = 0; q < W; ++q)
                if (q == e) { sm[q] = s1; cm[q] = c1; }
        }
    }
#pragma unroll
    for (int e = 0; e < W; ++e) ps[ry][cx * W + e] = (double)sm[e] + (double)cm[e];
    __syncthreads();
    for (int c = threadIdx.x; c < 32 * W; c += blockDim.x) {
        const int k = bx * 32 * W + c;
        if (k < d)
            part[(int64_t)by * d + k] = ((ps[0][c] + ps[1][c]) + (ps[2][c] + ps[3][c])) +
                                        ((ps[4][c] + ps[5][c]) + (ps[6][c] + ps[7][c]));
    }
}

template <bool VEC>
__global__ void __launch_bounds__(256) colsum_partial_kernel(const float* __restrict__ X, int64_t n, int d,
                                                             int64_t ldx, int64_t rows, double* part) {
    colsum_block<VEC>(X, n, d, ldx, rows, part, blockIdx.x, blockIdx.y);
}

// The means from the row blocks' sums: 256 threads on LANES row lanes x 256 /
// LANES columns; lane y adds blocks y, y + LANES, ... in order, then the lane
// sums meet in a fixed tree.  Bound by float64 adds, of which an SM makes two
// a clock: 32 lanes x 8 columns spread many blocks over 4 times the SMs that 8
// x 32 reach (2048 blocks, d = 128: 15 us where 8 x 32 took 37 us; 50 blocks, d =
// 300: 4.7 and 6.0 us), but have the longer tree (16 blocks, d = 100: 4.0 us where
// 8 x 32 take 3.5).  The choice is the order of the sums, so the batched build
// makes the same one.
static __host__ __device__ __forceinline__ bool mean_by_32_lanes(int nb) { return nb > 16; }

template <int LANES>
__device__ __forceinline__ void colmean_block(const double* __restrict__ part, int nb, int d, int64_t n,
                                              float* mean, int bx) {
    constexpr int COLS = 256 / LANES;
    const int cx = threadIdx.x % COLS, ry = threadIdx.x / COLS;
    const int j = bx * COLS + cx;
    __shared__ double ps[LANES][COLS];
    double sm = 0.0;
    if (j < d) {
#pragma unroll 8
        for (int b = ry; b < nb; b += LANES) sm += part[(int64_t)b * d + j];
    }
    ps[ry][cx] = sm;
    __syncthreads();
    if (ry == 0 && j < d) {
        double v[LANES];
#pragma unroll
        for (int l = 0; l < LANES; ++l) v[l] = ps[l][cx];
#pragma unroll
        for (int w = LANES / 2; w > 0; w >>= 1)
#pragma unroll
            for (int e = 0; e < w; ++e) v[e] = v[2 * e] + v[2 * e + 1];
        mean[j] = (float)(v[0] / (double)n);
    }
}

// grid ceil(d / (256 / LANES)), 256 threads
template <int LANES>
__global__ void __launch_bounds__(256) colmean_kernel(const double* __restrict__ part, int nb, int d,
                                                      int64_t n, float* mean) {
    colmean_block<LANES>(part, nb, d, n, mean, blockIdx.x);
}

// ---- 2. centring, norms -----------------------------------------------------------
// One warp per (padded) row.  Rows >= n and columns >= d are written as zero.
// Block bx of a grid of gx blocks.
template <bool BF16>
__device__ __forceinline__ void centre_rows(const float* __restrict__ X, int n, int d, int64_t ldx,
                                            const float* __restrict__ mean, int npad, int dpad,
                                            void* out, float* nrm, int bx, int gx) {
    const int warps = blockDim.x >> 5, lid = threadIdx.x & 31;
    for (int i = bx * warps + (threadIdx.x >> 5); i < npad; i += gx * warps) {
        float acc = 0.f;
        for (int j = lid; j < dpad; j += 32) {
            float v = 0.f;
            if (i < n && j < d) v = X[(int64_t)i * ldx + j] - mean[j];
            if (BF16) {
                const __nv_bfloat16 b = __float2bfloat16_rn(v);
                reinterpret_cast<__nv_bfloat16*>(out)[(int64_t)i * dpad + j] = b;
                v = __bfloat162float(b);
            } else {
                reinterpret_cast<float*>(out)[(int64_t)i * dpad + j] = v;
            }
            acc = fmaf(v, v, acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lid == 0) nrm[i] = acc;
    }
}

// The same with four columns per lane and step (float4 loads, 8- or 16-byte
// stores); needs X 16-byte aligned with ldx % 4 == 0 (dpad % 64 == 0 holds).
// Each lane sums the squares of its own columns in order, then the warp adds
// the lane sums in a fixed butterfly, so the norms are deterministic.
template <bool BF16>
__device__ __forceinline__ void centre_rows4(const float* __restrict__ X, int n, int d, int64_t ldx,
                                             const float* __restrict__ mean, int npad, int dpad,
                                             void* out, float* nrm, int bx, int gx) {
    const int warps = blockDim.x >> 5, lid = threadIdx.x & 31;
    for (int i = bx * warps + (threadIdx.x >> 5); i < npad; i += gx * warps) {
        float acc = 0.f;
        for (int j = 4 * lid; j < dpad; j += 128) {
            float v[4];
            if (i < n && j + 3 < d) {
                const float4 x = *reinterpret_cast<const float4*>(X + (int64_t)i * ldx + j);
                const float4 m = *reinterpret_cast<const float4*>(mean + j);
                v[0] = x.x - m.x; v[1] = x.y - m.y; v[2] = x.z - m.z; v[3] = x.w - m.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    v[e] = (i < n && j + e < d) ? X[(int64_t)i * ldx + j + e] - mean[j + e] : 0.f;
            }
            if (BF16) {
                __nv_bfloat16 bv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    bv[e] = __float2bfloat16_rn(v[e]);
                    v[e] = __bfloat162float(bv[e]);
                }
                uint2 pk;
                pk.x = (uint32_t)__bfloat16_as_ushort(bv[0]) | ((uint32_t)__bfloat16_as_ushort(bv[1]) << 16);
                pk.y = (uint32_t)__bfloat16_as_ushort(bv[2]) | ((uint32_t)__bfloat16_as_ushort(bv[3]) << 16);
                *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + (int64_t)i * dpad + j) = pk;
            } else {
                *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + (int64_t)i * dpad + j) =
                    make_float4(v[0], v[1], v[2], v[3]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) acc = fmaf(v[e], v[e], acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lid == 0) nrm[i] = acc;
    }
}

template <bool BF16, bool VEC>
__global__ void centre_kernel(const float* __restrict__ X, int n, int d, int64_t ldx,
                              const float* __restrict__ mean, int npad, int dpad, void* out,
                              float* nrm) {
    if (VEC) centre_rows4<BF16>(X, n, d, ldx, mean, npad, dpad, out, nrm, blockIdx.x, gridDim.x);
    else centre_rows<BF16>(X, n, d, ldx, mean, npad, dpad, out, nrm, blockIdx.x, gridDim.x);
}

// ---- 3. SIMT float32 GEMM with the distance epilogue ---------------------------
// Bound by the float32 pipe (n^2 d multiply-adds on or above the diagonal at
// 10000 x 100 against 400 MB of writes).  S is symmetric but for the order in
// which the two norms are subtracted, so only the tiles on or above the
// diagonal are multiplied; a tile above it also writes its mirror image, with
// the norms subtracted in that element's own order.  The features' padding
// past the next multiple of 8 is not multiplied.  Every element's products are
// still added one by one in the order of the features: two columns per packed
// FMA, the next 16 features fetched while the current ones are used.
// 10000 points, d = 100: 270 us where multiplying the full square padded to 128
// features, one column per FMA and no fetch ahead, took 664 us.
constexpr int GT = 128, GK = 16;

// Tile t of the upper triangle of nt x nt tiles, row by row of the transpose:
// column block k0, row block i0 <= k0.
__device__ __forceinline__ void triangle_tile(int t, int& bi, int& bk) {
    bk = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while ((int64_t)(bk + 1) * (bk + 2) / 2 <= t) ++bk;
    while ((int64_t)bk * (bk + 1) / 2 > t) --bk;
    bi = t - (int)((int64_t)bk * (bk + 1) / 2);
}

static int triangle_tiles(int n) {
    const int64_t nt = (n + GT - 1) / GT;
    return (int)(nt * (nt + 1) / 2);
}

__global__ void __launch_bounds__(256, 2) sim_gemm_fp32_kernel(const float* __restrict__ Xc, int n, int d,
                                                               int dpad, const float* __restrict__ nrm,
                                                               float* __restrict__ S, int64_t lds, int vec_ok) {
    __shared__ __align__(16) float As[2][GK][GT];
    __shared__ __align__(16) float Bs[2][GK][GT];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    int bi, bk;
    triangle_tile(blockIdx.x, bi, bk);
    const int i0 = bi * GT, k0 = bk * GT;
    float2 acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);

    // features multiplied: d rounded up to 8 (dpad is a multiple of 64, the rest zeros)
    const int dk = (d + 7) / 8 * 8;
    const int lr = tid >> 1, lc = (tid & 1) * 8;
    const float* pa = Xc + (int64_t)(i0 + lr) * dpad + lc;
    const float* pb = Xc + (int64_t)(k0 + lr) * dpad + lc;
    float4 va[2], vb[2];
    auto fetch = [&](int kk) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            va[h] = __ldg(reinterpret_cast<const float4*>(pa + kk + 4 * h));
            vb[h] = __ldg(reinterpret_cast<const float4*>(pb + kk + 4 * h));
        }
    };
    auto put = [&](int buf) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            As[buf][lc + 4 * h + 0][lr] = va[h].x; As[buf][lc + 4 * h + 1][lr] = va[h].y;
            As[buf][lc + 4 * h + 2][lr] = va[h].z; As[buf][lc + 4 * h + 3][lr] = va[h].w;
            Bs[buf][lc + 4 * h + 0][lr] = vb[h].x; Bs[buf][lc + 4 * h + 1][lr] = vb[h].y;
            Bs[buf][lc + 4 * h + 2][lr] = vb[h].z; Bs[buf][lc + 4 * h + 3][lr] = vb[h].w;
        }
    };
    auto step = [&](int buf, int k) {
        const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]);
        const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][k][64 + ty * 4]);
        const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
        const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][k][64 + tx * 4]);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                              make_float2(b1.z, b1.w)};
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = __ffma2_rn(make_float2(av[a], av[a]), bv[b], acc[a][b]);
    };
    fetch(0);
    put(0);
    __syncthreads();
    int buf = 0;
    for (int kk = 0; kk < dk; kk += GK, buf ^= 1) {
        const bool more = kk + GK < dk;
        if (more) fetch(kk + GK);
        if (kk + GK <= dk) {
#pragma unroll
            for (int k = 0; k < GK; ++k) step(buf, k);
        } else {
#pragma unroll
            for (int k = 0; k < GK / 2; ++k) step(buf, k);
        }
        if (more) put(buf ^ 1);
        __syncthreads();
    }
    // this thread's rows i0 + ri(a) and columns k0 + ri(b)
    auto at = [](int t, int a) { return (a < 4 ? 4 * t + a : 64 + 4 * t + a - 4); };
    float ni[8], nk[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        ni[a] = nrm[i0 + at(ty, a)];
        nk[a] = nrm[k0 + at(tx, a)];
    }
    auto dot = [&](int a, int b) { return (b & 1) ? acc[a][b >> 1].y : acc[a][b >> 1].x; };
    auto put4 = [&](int row, int col, const float (&v)[4]) {
        if (row >= n) return;
        float* p = S + (int64_t)row * lds + col;
        if (vec_ok && col + 4 <= n) {
            *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (col + e < n) p[e] = v[e];
        }
    };
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + at(ty, a), k = k0 + at(tx, 4 * h);
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int b = 4 * h + e;
                v[e] = (k + e == i) ? 0.f : fminf(0.f, fmaf(2.f, dot(a, b), -ni[a]) - nk[b]);
            }
            put4(i, k, v);
        }
    if (bi == bk) return;
#pragma unroll
    for (int b = 0; b < 8; ++b)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int a = 4 * h + e;
                v[e] = fminf(0.f, fmaf(2.f, dot(a, b), -nk[b]) - ni[a]);
            }
            put4(k0 + at(tx, b), i0 + at(ty, 4 * h), v);
        }
}

// ---- 4. exact median by radix select -------------------------------------------
__device__ __forceinline__ uint32_t float_key(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
    const uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}

// The two middle order statistics of the n(n-1) off-diagonal entries of S, in
// one pass over S.  16384 entries drawn at random bracket the median
// (sample_kernel): the sample's order statistics 288 either side of its
// middle (4.5 standard deviations of a median's rank) enclose the wanted ranks
// but for about 1 matrix in 10^5.  bracket_pass reads S once, counts the
// entries below the bracket and copies those inside it (3.5 % on average) to
// a buffer; digit_kernel then selects by radix passes of 11 bits over the
// buffer, starting at the bracket's own highest bit.  Where the bracket missed
// or the buffer overflowed (a large share of equal entries), the digit passes
// read S itself from the top bit, so the result is exact either way.  The
// decision stays on the device.  20000 points (1.6 GB): 386 us, of which the
// pass is 321 (0.75 of the copy rate: with 3.5 % hits nearly every step of 512
// entries takes the tail of scan, second read and stores, behind four 16-byte
// loads a lane), the digits 53 and the sample 11, where three radix passes over
// S took 1025 us; 1000 points: 35 us (kSmallSelect) where they took 144 us (16
// blocks, most of the time waiting on shared-memory atomics).
constexpr int kSampleThreads = 1024;
constexpr int kSamplePer = 16;          // entries per thread (small selections: 4)
constexpr int kSample = kSampleThreads * kSamplePer;
constexpr int kSampleBins = 1024;       // two digits of 10 bits settle the bracket
// Buffer entries a warp takes at a time (more if a step's hits need it): enough
// that few of its steps wait for the atomic, few enough, where a warp has only
// a few rows, that the digit passes do not read mostly unused chunk ends.
__host__ __device__ constexpr int chunk_of(int n) { return n < 4096 ? 128 : 512; }
constexpr int kPassWarps = 8;           // warps per block of the pass

struct SelectState {
    uint32_t lo, range;       // the bracket: keys lo .. lo + range
    uint32_t prefix[2];       // known digits of (key - lo) of the two order statistics
    uint32_t known_mask;
    int32_t  direct;          // the digit passes read S (lo = 0), not the buffer
    uint64_t rank[2];         // ranks left inside the prefix
    unsigned long long less, inside, slots;   // entries below and inside the bracket; buffer taken
    unsigned ticket;          // blocks of a digit pass that have finished
    int32_t  bits;            // of range + 1: where the digits start
};

// One selection: a problem's S, its buffer and its blocks in the launch.
struct Select {
    const float* S;
    int64_t lds;
    int n;
    int b0, nb;               // blocks [b0, b0 + nb) of the pass
    int d0, dn;               // blocks [d0, d0 + dn) of a digit pass
    SelectState* st;
    unsigned long long* hist; // 2 x 2048 bins
    uint32_t* cand;           // the buffer, cap entries
    unsigned long long cap;
    float* pref;
};

// Up to this many points a selection's latency is what counts, and three launches
// do all of it: the sample's block draws it (a quarter of the entries), the pass
// over S has smaller blocks and counts the first digit of what it keeps, and
// one block takes the other digits and writes the diagonal (1000 points: the
// three 35 us and the whole call 111 us, where six launches took 58 and 126 us).
constexpr int kSmallSelect = 1500;

// Blocks of the pass over S: about 32K entries each, at most 8 per SM; of the
// digits of the buffer: about 8K of its entries each, at most 4 per SM (a block
// clears and adds up to 4096 bins).
static int pass_blocks(int n) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(1216, ((int64_t)n * n + 32767) / 32768));
}
static int digit_blocks(int n) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(608, (int64_t)n * n / (8192 * 28)));
}
// A 16th of the entries (the bracket holds 3.5 % on average), and every warp's last chunk.
static unsigned long long cand_cap(int n) {
    return (unsigned long long)n * (unsigned long long)n / 16 +
           (unsigned long long)std::max(pass_blocks(n), 8) * kPassWarps * 512;
}

// The sample: kSample entries of S at seeded random places off the diagonal, read
// by block bx of gx into the start of the candidate buffer (many blocks: one
// SM has too few reads in flight for 16384 scattered ones: 3.5 us and 7.7 for the
// bracket, together 17 when one block did both).
__device__ __forceinline__ float drawn(const Select& q, int e) {
    const uint64_t u = splitmix64_at(0x6d656469616eull, (uint64_t)e + 1);
    const int i = (int)(((u >> 32) * (uint64_t)q.n) >> 32);
    int k = (int)(((u & 0xffffffffull) * (uint64_t)(q.n - 1)) >> 32);
    k += k >= i;
    return __ldg(q.S + (int64_t)i * q.lds + k);
}
__device__ __forceinline__ void draw_block(const Select& q, int bx, int gx) {
    for (int e = bx * blockDim.x + threadIdx.x; e < kSample; e += gx * blockDim.x)
        q.cand[e] = __float_as_uint(drawn(q, e));
}

// The bracket of one problem (one block of kSampleThreads) from the drawn
// entries: the keys around the two ranks by
// two radix passes of 10 bits below the sample's own highest differing bit
// (the digits spread: a fixed top byte would put nearly every entry in one
// bin, whose shared-memory atomics wait for one another).  What the digits
// leave open widens the bracket.  The state and histograms start from here.
// PER entries per thread, drawn here (SELF) or before.
template <int PER, bool SELF>
__device__ __forceinline__ void sample_block(const Select& q) {
    // 4.5 standard deviations of a median's rank, sqrt(sample) / 2
    constexpr int SAMPLE = kSampleThreads * PER, HALF = PER == 16 ? 288 : 144;
    static_assert(PER == 16 || PER == 4, "half widths");
    __shared__ unsigned int h[2][kSampleBins];
    __shared__ unsigned int wsum[32];
    __shared__ uint32_t wmin[32], wmax[32];
    __shared__ int found[2];
    __shared__ unsigned int rem[2];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t key[PER];
    uint32_t kmin = 0xffffffffu, kmax = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        key[e] = float_key(SELF ? drawn(q, e * kSampleThreads + t)
                                : __uint_as_float(q.cand[e * kSampleThreads + t]));
    }
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        kmin = min(kmin, key[e]);
        kmax = max(kmax, key[e]);
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) { wmin[warp] = kmin; wmax[warp] = kmax; }
    for (int b = t; b < 4096; b += kSampleThreads) q.hist[b] = 0;
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, wmin[lane]);
    kmax = __reduce_max_sync(0xffffffffu, wmax[lane]);
    const int bits = 32 - __clz((int)(kmax - kmin));
    uint32_t pre[2] = {0, 0}, km = 0;
    unsigned int rank[2] = {SAMPLE / 2 - HALF, SAMPLE / 2 + HALF};
    int shift = bits;
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        const int width = min(10, shift);
        shift -= width;
        const uint32_t dm = (1u << width) - 1u;
        h[0][t] = 0;
        h[1][t] = 0;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const uint32_t rel = key[e] - kmin, dg = (rel >> shift) & dm;
            if ((rel & km) == pre[0]) atomicAdd(&h[0][dg], 1u);
            if ((rel & km) == pre[1]) atomicAdd(&h[1][dg], 1u);
        }
        __syncthreads();
        // thread t owns bin t of both histograms (each at most kSample: 15 bits),
        // scanned together in one word
        const unsigned int own = h[0][t] | (h[1][t] << 16);
        unsigned int x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned int w = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const unsigned int before = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
        x += (warp > 0 ? before : 0u) - own;                // exclusive
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const unsigned int lo = (x >> (16 * j)) & 0xffffu, c = (own >> (16 * j)) & 0xffffu;
            if (rank[j] >= lo && rank[j] < lo + c) {
                found[j] = t;
                rem[j] = rank[j] - lo;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            pre[j] |= (uint32_t)found[j] << shift;
            rank[j] = rem[j];
        }
        km |= dm << shift;
        __syncthreads();
    }
    if (t == 0) {
        SelectState s{};
        s.lo = kmin + pre[0];
        s.range = (pre[1] | ((1u << shift) - 1u)) - pre[0];
        const uint64_t m = (uint64_t)q.n * (uint64_t)(q.n - 1);
        s.rank[0] = (m - 1) / 2;
        s.rank[1] = m / 2;
        *q.st = s;
    }
}

// Four consecutive entries 4f .. 4f+3 of a row; entries past its end read as 0.
template <bool VEC>
__device__ __forceinline__ float4 entries4(const float* __restrict__ row, int f, int n) {
    if constexpr (VEC) {
        return __ldg(reinterpret_cast<const float4*>(row) + f);
    } else {
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = 4 * f + e < n ? __ldg(row + 4 * f + e) : 0.f;
        return make_float4(v[0], v[1], v[2], v[3]);
    }
}

// One entry of the pass: below the bracket, less grows by 1; not settled by the
// two comparisons (inside the bracket, a zero or infinity at its edge, NaN),
// mask grows by bit.  Counts are float32 (exact: at most 16 bits a mask, a row's
// entries a count), because the additions then go to the FMA pipe and leave the
// half-rate ALU pipe to the comparisons.
__device__ __forceinline__ void look(float v, float lo, float hi, float bit, float& less, float& mask) {
    asm("{\n\t.reg .pred p, r;\n\t"
        "setp.lt.f32 p, %2, %3;\n\t"
        "setp.gt.or.f32 r, %2, %4, p;\n\t"
        "@p add.f32 %0, %0, 0f3F800000;\n\t"
        "@!r add.f32 %1, %1, %5;\n\t}"
        : "+f"(less), "+f"(mask)
        : "f"(v), "f"(lo), "f"(hi), "f"(bit));
}

// The pass over S: warps take rows in turn; block bx of gx.  A step is 512
// entries of a row, 16 per lane: two float comparisons each settle all but
// the bracket's own; these (3.5 %) are read again as keys, so that NaN and
// signed zeros fall where their keys do, and written behind one another by a
// scan of the lanes' counts.
// HIST: counts the first digit of select_small_kernel along the way.
template <bool VEC, bool HIST = false>
__device__ __forceinline__ void bracket_pass(const Select& q, int bx, int gx) {
    const int lane = threadIdx.x & 31;
    const uint32_t lo = q.st->lo, range = q.st->range;
    const float flo = key_float(lo), fhi = key_float(lo + range);
    const int n = q.n, n4 = (n + 3) >> 2, nfull = n >> 2;
    unsigned less = 0, inside = 0;
    // the warp's current chunk of the buffer: entries [at, end)
    unsigned long long at = 0, end = 0;
    bool full = false;
    const int chunk = HIST ? 32 : chunk_of(n);              // (a warp has one or two rows there)
    const int bits = 32 - __clz((int)range), shift = bits > 11 ? bits - 11 : 0;
    for (int i = bx * kPassWarps + (threadIdx.x >> 5); i < n; i += gx * kPassWarps) {
        const float* row = q.S + (int64_t)i * q.lds;
        const int fi = i >> 2;
        float fless = 0.f;
        for (int f0 = 0; f0 < n4; f0 += 128) {
            float4 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int f = f0 + 32 * u + lane;
                x[u] = f < n4 ? entries4<VEC>(row, f, n) : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
            }
            float fmask = 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int f = f0 + 32 * u + lane;
                float v[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
                if (f == fi || f >= nfull) {
                    // the diagonal and what lies past the row's end: above every finite bracket
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (4 * f + e == i || 4 * f + e >= n) v[e] = INFINITY;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) look(v[e], flo, fhi, (float)(1 << (4 * u + e)), fless, fmask);
            }
            unsigned mask = (unsigned)fmask;
            if (!__any_sync(0xffffffffu, mask != 0)) continue;
            const int own = __popc(mask);
            int incl = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            unsigned long long pos = at + (incl - own), fresh = 0, take = 0;
            if (!full && at + total > end) {                // the entries past `end` open a new chunk
                // (a multiple of 4: the digit passes read 16 bytes at a time)
                take = max((unsigned long long)chunk, (at + total - end + 3) & ~3ull);
                if (lane == 0) fresh = atomicAdd(&q.st->slots, take);
                fresh = __shfl_sync(0xffffffffu, fresh, 0);
                full = fresh + take > q.cap;                // then the digit passes will read S
            }
            for (; mask; mask &= mask - 1, ++pos) {
                const int b = __ffs((int)mask) - 1, k = 4 * (f0 + 32 * (b >> 2) + lane) + (b & 3);
                uint32_t rel = 0xffffffffu;                 // beyond every range: does not count
                if (k != i && k < n) {
                    const uint32_t key = float_key(__ldg(row + k));
                    less += key < lo;
                    if (key - lo <= range) {
                        rel = key - lo;
                        ++inside;
                        if (HIST) atomicAdd(reinterpret_cast<unsigned int*>(q.hist) + ((rel >> shift) & 2047u), 1u);
                    }
                }
                if (!full) q.cand[pos < end ? pos : fresh + (pos - end)] = rel;
            }
            if (full) continue;
            if (at + total > end) {
                at = fresh + (at + total - end);
                end = fresh + take;
            } else {
                at += total;
            }
        }
        less += (unsigned)fless;
    }
    if (!full)
        for (unsigned long long x = at + lane; x < end; x += 32) q.cand[x] = 0xffffffffu;
    less = __reduce_add_sync(0xffffffffu, less);
    inside = __reduce_add_sync(0xffffffffu, inside);
    if (lane == 0) {
        if (less) atomicAdd(&q.st->less, (unsigned long long)less);
        if (inside) atomicAdd(&q.st->inside, (unsigned long long)inside);
    }
}

// The bin of a histogram of at most 2048 counts that holds rank r, and the
// rank left inside it (a block of 256 threads, eight bins each).
__device__ __forceinline__ void find_bin(const unsigned long long* h, int nb, unsigned long long r,
                                         unsigned long long* wsum, int* found, unsigned long long* rem) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned long long c[8], own = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) c[e] = 8 * t + e < nb ? __ldcg(h + 8 * t + e) : 0ull;
#pragma unroll
    for (int e = 0; e < 8; ++e) own += c[e];
    unsigned long long x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    unsigned long long at = x - own;
    for (int w = 0; w < warp; ++w) at += wsum[w];
    if (r >= at && r < at + own) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (r >= at && r < at + c[e]) {
                *found = 8 * t + e;
                *rem = r - at;
            }
            at += c[e];
        }
    }
    __syncthreads();
}

// Digit pass p (0, 1, 2): block bx of gx counts the digit of the entries that
// match each order statistic's known prefix (one histogram serves both while
// they share it); the last block to finish finds the two bins and advances
// the state.
template <bool VEC>
__device__ __forceinline__ void digit_pass(const Select& q, int p, int bx, int gx) {
    __shared__ unsigned int h[2][2048];
    __shared__ unsigned long long wsum[32], rem[2];
    __shared__ int found[2];
    __shared__ bool last;
    SelectState* st = q.st;
    // pass 0 settles what the bracket gave (every block reads the same values;
    // the last one writes them)
    uint32_t lo = st->lo, range = st->range;
    bool direct = st->direct != 0;
    uint64_t r0 = st->rank[0], r1 = st->rank[1];
    int bits = st->bits;
    if (p == 0) {
        const unsigned long long less = st->less, inside = st->inside;
        // a full buffer is one whose chunks passed its end; a bracket up to the
        // largest key would leave the unused entries' mark inside it
        direct = st->slots > q.cap || r0 < less || r1 >= less + inside || range == 0xffffffffu;
        if (direct) {
            lo = 0;
            range = 0xffffffffu;
        } else {
            r0 -= less;
            r1 -= less;
        }
        bits = 32 - __clz((int)range);
    }
    const int top = bits - 11 * p;                      // bits still unknown
    if (top <= 0 && p > 0) return;
    const int shift = max(0, top - 11), width = max(0, min(11, top)), nb = 1 << width;
    const uint32_t dm = (uint32_t)nb - 1u;
    const uint32_t km = p == 0 ? 0u : st->known_mask, p0 = p == 0 ? 0u : st->prefix[0], p1 = p == 0 ? 0u : st->prefix[1];
    const bool same = p0 == p1;
    for (int b = threadIdx.x; b < 2 * 2048; b += blockDim.x) (&h[0][0])[b] = 0;
    __syncthreads();
    auto count = [&](uint32_t rel) {
        const uint32_t dg = (rel >> shift) & dm;
        if ((rel & km) == p0) atomicAdd(&h[0][dg], 1u);
        if (!same && (rel & km) == p1) atomicAdd(&h[1][dg], 1u);
    };
    if (!direct) {
        const unsigned long long slots = st->slots;
        const uint4* c4 = reinterpret_cast<const uint4*>(q.cand);
        const unsigned long long n4 = slots / 4, step = (unsigned long long)gx * blockDim.x;
        for (unsigned long long x0 = (unsigned long long)bx * blockDim.x + threadIdx.x; x0 < n4; x0 += 4 * step) {
            uint4 v[4];                     // four loads in flight before the first count
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[u] = x0 + u * step < n4 ? __ldg(c4 + x0 + u * step)
                                          : make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (v[u].x <= range) count(v[u].x);
                if (v[u].y <= range) count(v[u].y);
                if (v[u].z <= range) count(v[u].z);
                if (v[u].w <= range) count(v[u].w);
            }
        }
    } else {
        const int n4 = (q.n + 3) >> 2;
        for (int i = bx; i < q.n; i += gx) {
            const float* row = q.S + (int64_t)i * q.lds;
            for (int f = threadIdx.x; f < n4; f += blockDim.x) {
                const float4 x = entries4<VEC>(row, f, q.n);
                const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (4 * f + e < q.n && 4 * f + e != i) count(float_key(v[e]));
            }
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const unsigned int c0 = h[0][b], c1 = same ? c0 : h[1][b];
        if (c0) atomicAdd(&q.hist[b], (unsigned long long)c0);
        if (c1) atomicAdd(&q.hist[2048 + b], (unsigned long long)c1);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == (unsigned)gx - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x < 2) {
        found[threadIdx.x] = nb - 1;                    // kept only if the counts were inconsistent
        rem[threadIdx.x] = 0;
    }
    __syncthreads();
    find_bin(q.hist, nb, r0, wsum, &found[0], &rem[0]);
    find_bin(q.hist + 2048, nb, r1, wsum, &found[1], &rem[1]);
    for (int b = threadIdx.x; b < 2 * 2048; b += blockDim.x) q.hist[b] = 0;
    if (threadIdx.x == 0) {
        st->lo = lo;
        st->range = range;
        st->direct = direct ? 1 : 0;
        st->bits = bits;
        st->prefix[0] = p0 | ((uint32_t)found[0] << shift);
        st->prefix[1] = p1 | ((uint32_t)found[1] << shift);
        st->known_mask = km | (dm << shift);
        st->rank[0] = rem[0];
        st->rank[1] = rem[1];
        st->ticket = 0;
    }
}

// All digits of a small selection in one block, histograms in shared memory, then
// the result and (diag not null) the diagonal.
template <bool VEC>
__global__ void __launch_bounds__(1024) select_small_kernel(Select q, float* diag, float* pref, float zero) {
    __shared__ unsigned int h[2][2048];
    __shared__ unsigned long long wsum[32];
    __shared__ int found[2];
    __shared__ uint64_t rem[2];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const SelectState s = *q.st;
    // as pass 0 of digit_pass
    const bool direct = s.slots > q.cap || s.rank[0] < s.less || s.rank[1] >= s.less + s.inside || s.range == 0xffffffffu;
    const uint32_t lo = direct ? 0u : s.lo, range = direct ? 0xffffffffu : s.range;
    uint64_t rank[2] = {direct ? s.rank[0] : s.rank[0] - s.less, direct ? s.rank[1] : s.rank[1] - s.less};
    uint32_t pre[2] = {0, 0}, km = 0;
    int shift = 32 - __clz((int)range);
    while (shift > 0) {
        const int width = min(11, shift);
        shift -= width;
        const uint32_t dm = (1u << width) - 1u;
        const bool same = pre[0] == pre[1];
        const bool counted = km == 0 && !direct;            // the first digit of the buffer's entries
        for (int b = t; b < 2 * 2048; b += 1024)
            (&h[0][0])[b] = counted && b < 2048 ? __ldcg(reinterpret_cast<const unsigned int*>(q.hist) + b) : 0u;
        __syncthreads();
        auto count = [&](uint32_t rel) {
            const uint32_t dg = (rel >> shift) & dm;
            if ((rel & km) == pre[0]) atomicAdd(&h[0][dg], 1u);
            if (!same && (rel & km) == pre[1]) atomicAdd(&h[1][dg], 1u);
        };
        if (counted) {
        } else if (!direct) {
            const uint4* c4 = reinterpret_cast<const uint4*>(q.cand);
            const unsigned n4 = (unsigned)(s.slots / 4);
            for (unsigned x0 = t; x0 < n4; x0 += 4 * 1024) {
                uint4 v[4];                         // four loads in flight before the first count
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = x0 + 1024 * u < n4 ? c4[x0 + 1024 * u]
                                              : make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (v[u].x <= range) count(v[u].x);
                    if (v[u].y <= range) count(v[u].y);
                    if (v[u].z <= range) count(v[u].z);
                    if (v[u].w <= range) count(v[u].w);
                }
            }
        } else {
            const int n4 = (q.n + 3) >> 2;
            for (int i = warp; i < q.n; i += 32) {
                const float* row = q.S + (int64_t)i * q.lds;
                for (int f = lane; f < n4; f += 32) {
                    const float4 x = entries4<VEC>(row, f, q.n);
                    const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (4 * f + e < q.n && 4 * f + e != i) count(float_key(v[e]));
                }
            }
        }
        __syncthreads();
        // thread t owns bins 2t and 2t + 1 of both histograms, scanned together
        const unsigned a0 = h[0][2 * t], a1 = h[0][2 * t + 1];
        const unsigned b0 = same ? a0 : h[1][2 * t], b1 = same ? a1 : h[1][2 * t + 1];
        const unsigned long long own = (unsigned long long)(a0 + a1) | ((unsigned long long)(b0 + b1) << 32);
        unsigned long long x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned long long w = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const unsigned long long before = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
        x += (warp > 0 ? before : 0ull) - own;              // exclusive
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint64_t base = j ? x >> 32 : x & 0xffffffffull;
            const unsigned c0 = j ? b0 : a0, c1 = j ? b1 : a1;
            if (rank[j] >= base && rank[j] < base + c0) {
                found[j] = 2 * t;
                rem[j] = rank[j] - base;
            } else if (rank[j] >= base + c0 && rank[j] < base + c0 + c1) {
                found[j] = 2 * t + 1;
                rem[j] = rank[j] - base - c0;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            pre[j] |= (uint32_t)found[j] << shift;
            rank[j] = rem[j];
        }
        km |= dm << shift;
        __syncthreads();
    }
    const float p = (float)(0.5 * ((double)key_float(lo + pre[0]) + (double)key_float(lo + pre[1])));
    if (t == 0) *pref = p;
    if (diag)
        for (int i = t; i < q.n; i += 1024) diag[(int64_t)i * q.lds + i] = p + zero;
}

__device__ __forceinline__ float select_result(const SelectState* st) {
    const double a = (double)key_float(st->lo + st->prefix[0]);
    const double b = (double)key_float(st->lo + st->prefix[1]);
    return (float)(0.5 * (a + b));
}

constexpr int kDrawBlocks = 64;

__global__ void __launch_bounds__(256) draw_kernel(Select q) { draw_block(q, blockIdx.x, gridDim.x); }

__global__ void __launch_bounds__(kSampleThreads) sample_kernel(Select q) { sample_block<kSamplePer, false>(q); }

__global__ void __launch_bounds__(kSampleThreads) sample_small_kernel(Select q) { sample_block<4, true>(q); }

template <bool VEC, bool HIST>
__global__ void __launch_bounds__(32 * kPassWarps, 4) bracket_kernel(Select q) {
    bracket_pass<VEC, HIST>(q, blockIdx.x, gridDim.x);
}

template <bool VEC>
__global__ void __launch_bounds__(256) digit_kernel(Select q, int p) {
    digit_pass<VEC>(q, p, blockIdx.x, gridDim.x);
}

__global__ void select_finish_kernel(const SelectState* st, float* pref) {
    *pref = select_result(st);
}

// ---- 5. diagonal and tie-break noise -----------------------------------------------
// p(i) from a device vector, a finished selection (whose result goes to pref)
// or a by-value scalar (in that order).
__global__ void diag_kernel(float* S, int n, int64_t lds, const float* __restrict__ pvec,
                            const SelectState* __restrict__ st, float* pref, float pval, float zero) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const float p = st ? select_result(st) : pval;
    if (st && i == 0) *pref = p;
    // zero: -0 (p as it is) or +0 (a preference of -0 becomes +0, as the noise makes it)
    if (i < n) S[(int64_t)i * lds + i] = (pvec ? pvec[i] : p) + zero;
}

__global__ void noise_kernel(float* S, int n, int64_t lds, double rel, uint64_t seed) {
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        float* row = S + (int64_t)i * lds;
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const double v = (double)row[k];
            const double u = unit_from_u64(splitmix64_at(seed, (uint64_t)i * n + k + 1));
            row[k] = (float)(v + rel * fabs(v) * u);
        }
    }
}

// ---- workspace ---------------------------------------------------------------------
struct SimWs {
    double* part;
    float* mean;
    void* xc;
    float* nrm;
    SelectState* sel;
    unsigned long long* hist;
    uint32_t* cand;
    float* pref;
    int32_t* err;
};

static int pad_rows(int n) {
    const int t = (int)std::max<size_t>(GT, tc_similarity_pad_rows());
    return (n + t - 1) / t * t;
}
static int pad_dim(int d) { return (d + 63) / 64 * 64; }
// Row blocks of the column means: 256 rows, or more so that there are at most
// 2048 blocks (the float64 combine of the partials is sequential per column).
static int64_t mean_rows(int64_t n, int64_t d) {
    // fewer rows where few columns leave most SMs without a block; not below 128 up
    // to 2048 points, where combining many partials costs more than it saves
    const int64_t spread = (n * ((d + 127) / 128) + 151) / 152;
    return std::max<int64_t>(std::max<int64_t>(n <= 2048 ? 128 : 32, std::min<int64_t>(kMeanRows, spread)), (n + 2047) / 2048);
}
static int mean_blocks(int64_t n, int64_t d) { return (int)((n + mean_rows(n, d) - 1) / mean_rows(n, d)); }

// The largest mean_blocks(m, d) of any m <= n: callers size for their largest
// set and then take the means of subsets in the same buffer, and mean_blocks
// falls at many n (d <= 128: 152 blocks at 4864 points, 148 at 4865).  Up to 2048
// points a block has at least 128 rows; beyond, rows >= m ceil(d / 128) / 152
// unless they are 256 or more.
static int64_t mean_blocks_cap(int64_t n, int64_t d) {
    if (n <= 2048) return (n + 127) / 128;
    const int64_t wide = (d + 127) / 128, spread = (151 + wide) / wide;
    return std::max({int64_t(16), spread, std::min<int64_t>((n + kMeanRows - 1) / kMeanRows, 2048)});
}

size_t column_mean_part_doubles(int64_t n, int d) { return (size_t)mean_blocks_cap(n, d) * (size_t)d; }

int32_t column_means(const float* X, int64_t n, int d, int64_t ldx, double* part, float* mean,
                     cudaStream_t s) {
    const int nb = mean_blocks(n, d);
    if (aligned16(X) && (ldx & 3) == 0)
        colsum_partial_kernel<true><<<dim3((d + 127) / 128, nb), 256, 0, s>>>(X, n, d, ldx, mean_rows(n, d), part);
    else
        colsum_partial_kernel<false><<<dim3((d + 31) / 32, nb), 256, 0, s>>>(X, n, d, ldx, mean_rows(n, d), part);
    if (mean_by_32_lanes(nb)) colmean_kernel<32><<<(d + 7) / 8, 256, 0, s>>>(part, nb, d, n, mean);
    else colmean_kernel<8><<<(d + 31) / 32, 256, 0, s>>>(part, nb, d, n, mean);
    note_launches(2);
    return last_error();
}

// The median's selection: state and result, histograms, buffer (n^2 / 16 words).
struct MedianWs {
    SelectState* sel;
    float* pref;
    unsigned long long* hist;
    uint32_t* cand;
};
static void take_median(Carver& c, int64_t n, MedianWs* w) {
    char* head = c.take<char>(sizeof(SelectState) + sizeof(float));
    w->sel = reinterpret_cast<SelectState*>(head);
    w->pref = reinterpret_cast<float*>(head + (head ? sizeof(SelectState) : 0));
    w->hist = c.take<unsigned long long>(4096);
    w->cand = c.take<uint32_t>(cand_cap((int)n));
}

// median: with what only the median preference needs.
static size_t carve_sim(void* ws, int64_t n, int64_t d, bool median, SimWs* w) {
    Carver c(ws);
    const int npad = pad_rows((int)n), dpad = pad_dim((int)d);
    w->part = c.take<double>(column_mean_part_doubles(n, (int)d));
    w->mean = c.take<float>(d);
    w->xc = c.take<float>((size_t)npad * dpad);   // large enough for either precision
    w->nrm = c.take<float>(npad);
    w->pref = c.take<float>(2);
    w->err = reinterpret_cast<int32_t*>(w->pref + 1);       // one copy brings both
    MedianWs m{};
    if (median) take_median(c, n, &m);
    w->sel = m.sel;
    w->hist = m.hist;
    w->cand = m.cand;
    return c.used;
}

// Enqueues the median of S's off-diagonal entries, to *pref, and (diag: S, for
// writing) onto the diagonal; zero as in diag_kernel.
static int32_t median_offdiag(const float* S, int n, int64_t lds, SelectState* sel, unsigned long long* hist,
                              uint32_t* cand, float* diag, float* pref, float zero, cudaStream_t s) {
    const int grid = n <= kSmallSelect ? (n * n + 8191) / 8192 : pass_blocks(n), dgrid = digit_blocks(n);
    const Select q{S, lds, n, 0, grid, 0, dgrid, sel, hist, cand, cand_cap(n), nullptr};
    const bool vec = aligned16(S) && (lds & 3) == 0, small = n <= kSmallSelect;
    if (small) {
        sample_small_kernel<<<1, kSampleThreads, 0, s>>>(q);
    } else {
        draw_kernel<<<kDrawBlocks, 256, 0, s>>>(q);
        sample_kernel<<<1, kSampleThreads, 0, s>>>(q);
    }
    if (small) {
        if (vec) bracket_kernel<true, true><<<grid, 32 * kPassWarps, 0, s>>>(q);
        else bracket_kernel<false, true><<<grid, 32 * kPassWarps, 0, s>>>(q);
    } else {
        if (vec) bracket_kernel<true, false><<<grid, 32 * kPassWarps, 0, s>>>(q);
        else bracket_kernel<false, false><<<grid, 32 * kPassWarps, 0, s>>>(q);
    }
    if (small) {
        if (vec) select_small_kernel<true><<<1, 1024, 0, s>>>(q, diag, pref, zero);
        else select_small_kernel<false><<<1, 1024, 0, s>>>(q, diag, pref, zero);
        note_launches(3);
        return last_error();
    }
    for (int p = 0; p < 3; ++p) {
        if (vec) digit_kernel<true><<<dgrid, 256, 0, s>>>(q, p);
        else digit_kernel<false><<<dgrid, 256, 0, s>>>(q, p);
    }
    if (diag) diag_kernel<<<(n + 255) / 256, 256, 0, s>>>(diag, n, lds, nullptr, sel, pref, 0.f, zero);
    else select_finish_kernel<<<1, 1, 0, s>>>(sel, pref);
    note_launches(7);
    return last_error();
}

// ---- the batched build ---------------------------------------------------------------
// ap_similarity_batched runs each stage above once for all problems of the
// batch: a launch's blocks are dealt out to problems by prefix counts, each
// block finds its problem by binary search and runs the single-problem code
// with its local block index, so every problem's S and preference are bit
// for bit those of ap_similarity.  Only the Gram products are launched per
// problem.
struct SimProblem {
    const float* X;
    float* S;
    int64_t lds;
    int n, npad;
    int64_t mrows;          // rows per column-sum block
    int nb;                 // column-sum blocks
    int part_b0;            // first column-sum block of the problem in the batched grid
    int centre_b0, centre_nb;
    Select sel;             // the median's selection (its blocks in the passes included)
    double* part;
    float* mean;
    void* xc;
    float* nrm;
    int64_t roff;           // first row of the problem in the centred-feature arena
};

// The problem whose blocks (first block b0(P[b])) include block `blk`.
template <class F>
__device__ __forceinline__ int sim_problem_of(const SimProblem* P, int count, int blk, F b0) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b0(P[mid]) <= blk) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// grid (sum of column-sum blocks, ceil(d / 32, or 128 for VEC))
template <bool VEC>
__global__ void __launch_bounds__(256) colsum_batched_kernel(const SimProblem* __restrict__ P, int count,
                                                             int d, int64_t ldx) {
    const int b = sim_problem_of(P, count, blockIdx.x, [](const SimProblem& q) { return q.part_b0; });
    const SimProblem& q = P[b];
    colsum_block<VEC>(q.X, q.n, d, ldx, q.mrows, q.part, blockIdx.y, blockIdx.x - q.part_b0);
}

// grid (problems, ceil(d/32)), 256 threads
__global__ void __launch_bounds__(256) colmean_batched_kernel(const SimProblem* __restrict__ P, int d) {
    const SimProblem& q = P[blockIdx.x];
    if (mean_by_32_lanes(q.nb)) {           // 8 columns at a time
        for (int t = 0; t < 4; ++t) {
            colmean_block<32>(q.part, q.nb, d, q.n, q.mean, 4 * blockIdx.y + t);
            __syncthreads();
        }
    } else {
        colmean_block<8>(q.part, q.nb, d, q.n, q.mean, blockIdx.y);
    }
}

// grid (sum of centring blocks)
template <bool BF16, bool VEC>
__global__ void centre_batched_kernel(const SimProblem* __restrict__ P, int count, int d, int64_t ldx,
                                      int dpad) {
    const int b = sim_problem_of(P, count, blockIdx.x, [](const SimProblem& q) { return q.centre_b0; });
    const SimProblem& q = P[b];
    if (VEC)
        centre_rows4<BF16>(q.X, q.n, d, ldx, q.mean, q.npad, dpad, q.xc, q.nrm, blockIdx.x - q.centre_b0,
                           q.centre_nb);
    else
        centre_rows<BF16>(q.X, q.n, d, ldx, q.mean, q.npad, dpad, q.xc, q.nrm, blockIdx.x - q.centre_b0,
                          q.centre_nb);
}

// grid (problems, blocks of each)
__global__ void __launch_bounds__(256) draw_batched_kernel(const SimProblem* __restrict__ P) {
    draw_block(P[blockIdx.x].sel, blockIdx.y, gridDim.y);
}

// grid (problems)
__global__ void __launch_bounds__(kSampleThreads) sample_batched_kernel(const SimProblem* __restrict__ P) {
    sample_block<kSamplePer, false>(P[blockIdx.x].sel);
}

// grid (sum of the problems' pass blocks)
template <bool VEC>
__global__ void __launch_bounds__(32 * kPassWarps, 4) bracket_batched_kernel(const SimProblem* __restrict__ P, int count) {
    const int b = sim_problem_of(P, count, blockIdx.x, [](const SimProblem& q) { return q.sel.b0; });
    const Select q = P[b].sel;
    bracket_pass<VEC>(q, blockIdx.x - q.b0, q.nb);
}

template <bool VEC>
__global__ void __launch_bounds__(256) digit_batched_kernel(const SimProblem* __restrict__ P, int count, int p) {
    const int b = sim_problem_of(P, count, blockIdx.x, [](const SimProblem& q) { return q.sel.d0; });
    const Select q = P[b].sel;
    digit_pass<VEC>(q, p, blockIdx.x - q.d0, q.dn);
}

// grid (problems, y); the median (median = 1) or the scalar p onto the diagonal
__global__ void diag_batched_kernel(const SimProblem* __restrict__ P, int median, float pval) {
    const SimProblem& q = P[blockIdx.x];
    const float p = median ? select_result(q.sel.st) : pval;
    if (median && blockIdx.y == 0 && threadIdx.x == 0) *q.sel.pref = p;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < q.n; i += gridDim.y * blockDim.x)
        q.S[(int64_t)i * q.lds + i] = p;
}

}  // namespace apgb

using namespace apgb;

APGB_API size_t ap_similarity_workspace_size(int64_t n, int64_t d) {
    if (n < 2 || d < 1 || n > INT_MAX / 2 || d > 65536) return 0;
    SimWs w;
    return carve_sim(nullptr, n, d, true, &w);
}

namespace apgb {

// Enqueues the whole similarity build of one problem on s (no synchronisation):
// means, centring (+ bf16 rounding), the Gram product with the distance
// epilogue, the preference and the optional noise.  pref_dev receives the
// median (AP_PREF_MEDIAN); err the tensor-core kernel's error flag.
static int32_t similarity_enqueue(const float* X, int ni, int di, int64_t ldx, float* S, int64_t lds,
                                  int32_t precision, int32_t pref_mode, const float* pref,
                                  double noise_rel, uint64_t seed, const SimWs& w, float* pref_dev,
                                  int32_t* err, cudaStream_t s) {
    const int npad = pad_rows(ni), dpad = pad_dim(di);
    AP_TRY(column_means(X, ni, di, ldx, w.part, w.mean, s));
    const int cgrid = std::min((npad + 7) / 8, 65535);
    const bool vx = aligned16(X) && (ldx & 3) == 0;
    if (precision == AP_PREC_FP32) {
        if (vx) centre_kernel<false, true><<<cgrid, 256, 0, s>>>(X, ni, di, ldx, w.mean, npad, dpad, w.xc, w.nrm);
        else centre_kernel<false, false><<<cgrid, 256, 0, s>>>(X, ni, di, ldx, w.mean, npad, dpad, w.xc, w.nrm);
        const int vec_ok = aligned16(S) && (lds & 3) == 0;
        sim_gemm_fp32_kernel<<<triangle_tiles(ni), 256, 0, s>>>(static_cast<const float*>(w.xc), ni, di, dpad,
                                                                w.nrm, S, lds, vec_ok);
        AP_TRY(last_error());
    } else {
        if (vx) centre_kernel<true, true><<<cgrid, 256, 0, s>>>(X, ni, di, ldx, w.mean, npad, dpad, w.xc, w.nrm);
        else centre_kernel<true, false><<<cgrid, 256, 0, s>>>(X, ni, di, ldx, w.mean, npad, dpad, w.xc, w.nrm);
        AP_TRY(last_error());
        AP_TRY(tc_similarity_bf16(static_cast<const __nv_bfloat16*>(w.xc), w.nrm, ni, dpad, S, lds,
                                  err, s));
    }
    const float zero = noise_rel > 0.0 ? 0.f : -0.f;
    if (pref_mode == AP_PREF_MEDIAN) {
        AP_TRY(median_offdiag(S, ni, lds, w.sel, w.hist, w.cand, S, pref_dev, zero, s));
    } else if (pref_mode == AP_PREF_SCALAR) {
        diag_kernel<<<(ni + 255) / 256, 256, 0, s>>>(S, ni, lds, nullptr, nullptr, nullptr, pref[0], zero);
    } else {
        diag_kernel<<<(ni + 255) / 256, 256, 0, s>>>(S, ni, lds, pref, nullptr, nullptr, 0.f, zero);
    }
    // s + noise_rel |s| u with u < 1 and noise_rel <= 2^-26 lies within half a
    // float32 ulp of s (at least 2^-25 |s|), so it rounds to s itself: the pass
    // (float64 arithmetic on every entry; 14.6 us at 1000 points) would change
    // nothing but a -0 on the diagonal, which diag_kernel has made +0
    if (noise_rel > 0x1p-26) {
        noise_kernel<<<std::min(ni, 8192), 256, 0, s>>>(S, ni, lds, noise_rel, seed);
        note_launches(1);
    }
    // centre, GEMM (the tensor-core one counts itself), a diagonal not written by the median
    note_launches((precision == AP_PREC_FP32 ? 2 : 1) + (pref_mode == AP_PREF_MEDIAN ? 0 : 1));
    return last_error();
}

static bool sim_args_ok(int32_t precision, int32_t pref_mode, const float* pref, double noise_rel) {
    if (precision != AP_PREC_FP32 && precision != AP_PREC_BF16) return false;
    if (pref_mode != AP_PREF_MEDIAN && pref_mode != AP_PREF_SCALAR && pref_mode != AP_PREF_VECTOR)
        return false;
    if (pref_mode != AP_PREF_MEDIAN && !pref) return false;
    return noise_rel >= 0.0 && std::isfinite(noise_rel);
}

}  // namespace apgb

APGB_API int32_t ap_similarity(const float* X, int64_t n, int64_t d, int64_t ldx, float* S,
                               int64_t lds, int32_t precision, int32_t pref_mode,
                               const float* pref, double noise_rel, uint64_t seed,
                               float* pref_out, void* ws, size_t ws_bytes, void* stream) {
    if (!X || !S || n < 2 || d < 1 || ldx < d || lds < n || n > INT_MAX / 2 || d > 65536)
        return AP_ERR_INVALID_ARG;
    if (!sim_args_ok(precision, pref_mode, pref, noise_rel)) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    SimWs w;
    const bool median = pref_mode == AP_PREF_MEDIAN;
    AP_TRY(check_ws(ws, ws_bytes, carve_sim(nullptr, n, d, median, &w)));
    carve_sim(ws, n, d, median, &w);
    AP_CUDA_TRY(cudaMemsetAsync(w.err, 0, sizeof(int32_t), s));
    AP_TRY(similarity_enqueue(X, (int)n, (int)d, ldx, S, lds, precision, pref_mode, pref, noise_rel,
                              seed, w, w.pref, w.err, s));
    struct { float pref; int32_t err; } h;
    AP_CUDA_TRY(cudaMemcpyAsync(&h, w.pref, sizeof(h), cudaMemcpyDeviceToHost, s));
    AP_CUDA_TRY(cudaStreamSynchronize(s));
    if (h.err) return AP_ERR_TIMEOUT;
    if (pref_out)
        *pref_out = pref_mode == AP_PREF_MEDIAN ? h.pref : pref_mode == AP_PREF_SCALAR ? pref[0] : NAN;
    return AP_OK;
}

namespace apgb {

// The Gram products of a batch are spread round-robin over kSimStreams
// library-owned streams (created once per device), so that the small
// problems' products overlap; they fork from and join back to the caller's
// stream through events.  Every other stage is one launch for the whole batch
// on the caller's stream.
constexpr int kSimStreams = 4;

static std::mutex g_sim_mu;
static std::map<int, std::array<cudaStream_t, kSimStreams>> g_sim_streams;

static int32_t sim_streams(std::array<cudaStream_t, kSimStreams>* out) {
    int dev = 0;
    AP_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(g_sim_mu);
    auto it = g_sim_streams.find(dev);
    if (it == g_sim_streams.end()) {
        std::array<cudaStream_t, kSimStreams> a{};
        for (auto& x : a) AP_CUDA_TRY(cudaStreamCreateWithFlags(&x, cudaStreamNonBlocking));
        it = g_sim_streams.emplace(dev, a).first;
    }
    *out = it->second;
    return AP_OK;
}

// Workspace of a batch: the problem table, every problem's column-sum
// partials, mean, centred copy, norms, select state and histograms, its
// preference and its Gram product's error flag.  host[b] receives problem b's
// pointers and block counts (problem fields filled by the caller).
static size_t carve_batched(void* ws, const int64_t* n, int32_t count, int64_t d, int32_t precision, bool median,
                            SimProblem** table, std::vector<SimProblem>* host, int32_t** err,
                            float** prefs, void** tables) {
    Carver c(ws);
    SimProblem* t = c.take<SimProblem>((size_t)count);
    float* pv = c.take<float>(2 * (size_t)count);           // the preferences, then the errors: one copy
    int32_t* e = pv ? reinterpret_cast<int32_t*>(pv + count) : nullptr;
    const int dpad = pad_dim((int)d);
    const size_t esz = precision == AP_PREC_FP32 ? sizeof(float) : sizeof(__nv_bfloat16);
    // every problem's centred rows (and norms) in one arena, problem b from row
    // roff_b (a multiple of the tensor-core tile), so that one grouped launch
    // covers the whole batch
    int64_t rows = 0;
    for (int32_t b = 0; b < count; ++b) rows += pad_rows((int)n[b]);
    unsigned char* xc_arena = c.take<unsigned char>((size_t)rows * dpad * esz);
    float* nrm_arena = c.take<float>((size_t)rows);
    void* tab = c.take<unsigned char>(tc_grouped_table_bytes(n, count));
    int part_b0 = 0, centre_b0 = 0, pass_b0 = 0, digit_b0 = 0;
    int64_t roff = 0;
    for (int32_t b = 0; b < count; ++b) {
        SimProblem q{};
        q.n = (int)n[b];
        q.npad = pad_rows(q.n);
        q.mrows = mean_rows(n[b], d);
        q.nb = mean_blocks(n[b], d);
        q.part_b0 = part_b0;
        part_b0 += q.nb;
        q.centre_nb = std::min((q.npad + 7) / 8, 65535);
        q.centre_b0 = centre_b0;
        centre_b0 += q.centre_nb;
        q.sel.n = q.n;
        q.sel.nb = pass_blocks(q.n);
        q.sel.b0 = pass_b0;
        pass_b0 += q.sel.nb;
        q.sel.dn = digit_blocks(q.n);
        q.sel.d0 = digit_b0;
        digit_b0 += q.sel.dn;
        q.part = c.take<double>((size_t)q.nb * d);
        q.mean = c.take<float>((size_t)d);
        q.roff = roff;
        q.xc = xc_arena ? xc_arena + (size_t)roff * dpad * esz : nullptr;
        q.nrm = nrm_arena ? nrm_arena + roff : nullptr;
        roff += q.npad;
        MedianWs m{};
        if (median) take_median(c, n[b], &m);
        q.sel.st = m.sel;
        q.sel.hist = m.hist;
        q.sel.cap = cand_cap(q.n);
        q.sel.cand = m.cand;
        q.sel.pref = pv ? pv + b : nullptr;
        if (host) (*host)[b] = q;
    }
    if (table) *table = t;
    if (err) *err = e;
    if (prefs) *prefs = pv;
    if (tables) *tables = tab;
    return c.used;
}

static bool batched_args_ok(const int64_t* n, int32_t count, int64_t d) {
    if (!n || count < 1 || d < 1 || d > 65536) return false;
    int64_t blocks = 0;
    for (int32_t b = 0; b < count; ++b) {
        if (n[b] < 2 || n[b] > INT_MAX / 2) return false;
        blocks += std::min<int64_t>(n[b], 4096);
    }
    return blocks <= INT_MAX;
}

}  // namespace apgb

APGB_API size_t ap_similarity_batched_workspace_size(const int64_t* n, int32_t count, int64_t d) {
    if (!batched_args_ok(n, count, d)) return 0;
    // the bf16 centred copy is the smaller; size for float32 so one query serves both
    return carve_batched(nullptr, n, count, d, AP_PREC_FP32, true, nullptr, nullptr, nullptr, nullptr, nullptr);
}

APGB_API int32_t ap_similarity_batched(const float* X, const int64_t* xoff, const int64_t* n,
                                       int32_t count, int64_t d, int64_t ldx, float* S,
                                       const int64_t* soff, const int64_t* lds, int32_t precision,
                                       int32_t pref_mode, const float* pref, float* pref_out,
                                       void* ws, size_t ws_bytes, void* stream) {
    if (!X || !xoff || !n || !S || !soff || !lds || ldx < d || !batched_args_ok(n, count, d))
        return AP_ERR_INVALID_ARG;
    if (pref_mode == AP_PREF_VECTOR || !sim_args_ok(precision, pref_mode, pref, 0.0))
        return AP_ERR_INVALID_ARG;
    int64_t nmax = 0;
    bool vec = true;
    for (int32_t b = 0; b < count; ++b) {
        if (lds[b] < n[b] || xoff[b] < 0 || soff[b] < 0) return AP_ERR_INVALID_ARG;
        nmax = std::max(nmax, n[b]);
        vec = vec && aligned16(S + soff[b]) && (lds[b] & 3) == 0;
    }
    // the bf16 path's tensor stores need 16-byte aligned rows of S
    if (precision != AP_PREC_FP32 && !vec) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool median = pref_mode == AP_PREF_MEDIAN;
    AP_TRY(check_ws(ws, ws_bytes, carve_batched(nullptr, n, count, d, AP_PREC_FP32, median, nullptr, nullptr, nullptr,
                                                nullptr, nullptr)));
    std::vector<SimProblem> host(count);
    SimProblem* table = nullptr;
    int32_t* err = nullptr;
    float* prefs = nullptr;
    void* tables = nullptr;
    carve_batched(ws, n, count, d, precision, median, &table, &host, &err, &prefs, &tables);
    int part_blocks = 0, centre_blocks = 0, pass_total = 0, digit_total = 0;
    for (int32_t b = 0; b < count; ++b) {
        host[b].X = X + xoff[b];
        host[b].S = S + soff[b];
        host[b].lds = lds[b];
        host[b].sel.S = host[b].S;
        host[b].sel.lds = lds[b];
        part_blocks += host[b].nb;
        centre_blocks += host[b].centre_nb;
        pass_total += host[b].sel.nb;
        digit_total += host[b].sel.dn;
    }
    const int di = (int)d, dpad = pad_dim(di);
    const bool bf16 = precision != AP_PREC_FP32;
    AP_CUDA_TRY(cudaMemcpyAsync(table, host.data(), sizeof(SimProblem) * count, cudaMemcpyHostToDevice, s));
    AP_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int32_t) * count, s));
    // 1-2. column means and the centred copies of every problem
    bool vx = (ldx & 3) == 0;
    for (int32_t b = 0; b < count; ++b) vx = vx && aligned16(X + xoff[b]);
    if (vx) colsum_batched_kernel<true><<<dim3(part_blocks, (di + 127) / 128), 256, 0, s>>>(table, count, di, ldx);
    else colsum_batched_kernel<false><<<dim3(part_blocks, (di + 31) / 32), 256, 0, s>>>(table, count, di, ldx);
    colmean_batched_kernel<<<dim3(count, (di + 31) / 32), 256, 0, s>>>(table, di);
    if (bf16) {
        if (vx) centre_batched_kernel<true, true><<<centre_blocks, 256, 0, s>>>(table, count, di, ldx, dpad);
        else centre_batched_kernel<true, false><<<centre_blocks, 256, 0, s>>>(table, count, di, ldx, dpad);
    } else {
        if (vx) centre_batched_kernel<false, true><<<centre_blocks, 256, 0, s>>>(table, count, di, ldx, dpad);
        else centre_batched_kernel<false, false><<<centre_blocks, 256, 0, s>>>(table, count, di, ldx, dpad);
    }
    note_launches(3);
    AP_TRY(last_error());
    // 3. the Gram products: bf16 as one persistent tensor-core launch over the
    //    tiles of every problem; float32 forked over the library's streams
    if (bf16) {
        std::vector<int64_t> roffs(count), nn(count), ld(count);
        std::vector<float*> Sp(count);
        int64_t rows = 0;
        for (int32_t b = 0; b < count; ++b) {
            roffs[b] = host[b].roff;
            nn[b] = host[b].n;
            ld[b] = host[b].lds;
            Sp[b] = host[b].S;
            rows = host[b].roff + host[b].npad;
        }
        AP_TRY(tc_similarity_bf16_grouped(static_cast<const __nv_bfloat16*>(host[0].xc), host[0].nrm, rows,
                                          dpad, nn.data(), roffs.data(), Sp.data(), ld.data(), count,
                                          tables, err, s));
    } else {
        std::array<cudaStream_t, kSimStreams> ss;
        AP_TRY(sim_streams(&ss));
        cudaEvent_t fork, join[kSimStreams];
        AP_CUDA_TRY(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
        for (auto& e : join) AP_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        struct Guard {
            cudaEvent_t f;
            cudaEvent_t* j;
            ~Guard() {
                cudaEventDestroy(f);
                for (int k = 0; k < kSimStreams; ++k) cudaEventDestroy(j[k]);
            }
        } guard{fork, join};
        AP_CUDA_TRY(cudaEventRecord(fork, s));
        for (int k = 0; k < kSimStreams; ++k) AP_CUDA_TRY(cudaStreamWaitEvent(ss[k], fork, 0));
        int32_t st = AP_OK;
        for (int32_t b = 0; b < count && st == AP_OK; ++b) {
            const SimProblem& q = host[b];
            cudaStream_t sk = ss[b % kSimStreams];
            const int vec_ok = aligned16(q.S) && (q.lds & 3) == 0;
            sim_gemm_fp32_kernel<<<triangle_tiles(q.n), 256, 0, sk>>>(static_cast<const float*>(q.xc), q.n, di,
                                                                      dpad, q.nrm, q.S, q.lds, vec_ok);
            note_launches(1);
            st = last_error();
        }
        // join: the caller's stream continues after every worker (also on error)
        for (int k = 0; k < kSimStreams; ++k) {
            AP_CUDA_TRY(cudaEventRecord(join[k], ss[k]));
            AP_CUDA_TRY(cudaStreamWaitEvent(s, join[k], 0));
        }
        AP_TRY(st);
    }
    // 4-5. the preferences and the diagonals
    const int dgy = (int)std::min<int64_t>((nmax + 255) / 256, 65535);
    if (pref_mode == AP_PREF_MEDIAN) {
        draw_batched_kernel<<<dim3(count, 16), 256, 0, s>>>(table);
        sample_batched_kernel<<<count, kSampleThreads, 0, s>>>(table);
        if (vec) bracket_batched_kernel<true><<<pass_total, 32 * kPassWarps, 0, s>>>(table, count);
        else bracket_batched_kernel<false><<<pass_total, 32 * kPassWarps, 0, s>>>(table, count);
        for (int p = 0; p < 3; ++p) {
            if (vec) digit_batched_kernel<true><<<digit_total, 256, 0, s>>>(table, count, p);
            else digit_batched_kernel<false><<<digit_total, 256, 0, s>>>(table, count, p);
        }
        diag_batched_kernel<<<dim3(count, dgy), 256, 0, s>>>(table, 1, 0.f);
        note_launches(7);
    } else {
        diag_batched_kernel<<<dim3(count, dgy), 256, 0, s>>>(table, 0, pref[0]);
        note_launches(1);
    }
    AP_TRY(last_error());
    std::vector<float> v(2 * (size_t)count);                // preferences, errors
    AP_CUDA_TRY(cudaMemcpyAsync(v.data(), prefs, sizeof(float) * v.size(), cudaMemcpyDeviceToHost, s));
    AP_CUDA_TRY(cudaStreamSynchronize(s));
    for (int32_t b = 0; b < count; ++b) {
        int32_t e;
        std::memcpy(&e, &v[(size_t)count + b], sizeof(e));
        if (e) return AP_ERR_TIMEOUT;
    }
    if (pref_out)
        for (int32_t b = 0; b < count; ++b)
            pref_out[b] = pref_mode == AP_PREF_MEDIAN ? v[b] : pref_mode == AP_PREF_SCALAR ? pref[0] : NAN;
    return AP_OK;
}

APGB_API size_t ap_preference_median_workspace_size(int64_t n) {
    if (n < 2 || n > INT_MAX / 2) return 0;
    Carver c(nullptr);
    MedianWs w;
    take_median(c, n, &w);
    return c.used;
}

APGB_API int32_t ap_preference_median(const float* S, int64_t n, int64_t ld, float* median,
                                      void* ws, size_t ws_bytes, void* stream) {
    if (!S || !median || n < 2 || n > INT_MAX / 2 || ld < n) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    AP_TRY(check_ws(ws, ws_bytes, ap_preference_median_workspace_size(n)));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Carver c(ws);
    MedianWs w;
    take_median(c, n, &w);
    AP_TRY(median_offdiag(S, (int)n, ld, w.sel, w.hist, w.cand, nullptr, w.pref, 0.f, s));
    float v = NAN;
    AP_CUDA_TRY(cudaMemcpyAsync(&v, w.pref, sizeof(float), cudaMemcpyDeviceToHost, s));
    AP_CUDA_TRY(cudaStreamSynchronize(s));
    *median = v;
    return AP_OK;
}
