// The learned warm start (not part of the paper; it plays the role Algorithm
// 2's merged availabilities play, and its exemplar score can choose
// Algorithm 3's landmarks).
//
// Per point k of S with preference scale p > 0, 25 features:
//   0-15  the 16 largest off-diagonal s(k,j), decreasing (ties: lower j first), / p
//   16-17 mean and standard deviation of the off-diagonal s(k,j), / p
//   18    s(k,k) / p
//   19-22 log(1 + #{j != k : s(k,j) >= -q p}) for q = 1/8, 1/4, 1/2, 1 (the
//         thresholds formed in float32): how many points lie within q times
//         the preference scale, i.e. how much support k could collect
//   23    D(k) - max_j D(j) over the 16 nearest j of k (those of features
//         0-15), with D = feature 20: positive where k is denser than all of
//         its neighbours, as exemplars tend to be
//   24    the fraction of those 16 neighbours with D(j) > D(k)
// A 25-256-256-3 network (ReLU) maps them to (c_hat, a_hat, logit): the
// predicted converged column value min(0, r(k,k) + a(k,k))/p that the warm
// start writes into column k, a(k,k)/p and the exemplar log-odds.  Training:
// mean over rows of (c_hat-t_c)^2 + (a_hat-t_a)^2 + softplus(logit) -
// t_e*logit, Adam.
//
// Parameters: one flat fp32 vector (W1 256x25, b1, W2 256x256, b2, W3 3x256,
// b3, mu 25, isd 25); the input is standardised first, x -> (x - mu) * isd,
// with mu and isd fixed (their gradient is zero, so Adam leaves them).  The
// products use a bf16 copy of the weights with fp32 accumulation.  All
// reductions (loss, weight gradients) run in a fixed order.
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace apgb {
namespace mlp {

constexpr int IN = 25, HID = 256, OUT = 3;
constexpr int F_DENS = 20;       // the density D(k) of features 23-24
constexpr int64_t OFF_W1 = 0, OFF_B1 = OFF_W1 + HID * IN, OFF_W2 = OFF_B1 + HID,
                  OFF_B2 = OFF_W2 + HID * HID, OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + OUT * HID,
                  OFF_MU = OFF_B3 + OUT, OFF_ISD = OFF_MU + IN, NP = OFF_ISD + IN;

// ---- features -------------------------------------------------------------------
constexpr int TOPK = 16;

// One warp per row of one problem.  The pass is bound by reading S (twice:
// the second time mostly from L2) and by about 25 instructions an entry, not
// by the selection:
//   scan 1  sums of e and e^2, where e = v - (a value inside the row): the mean
//           of 32 entries spread over it.  Entries close to one another lose
//           nothing to cancellation then, and e^2 exceeds the variance by a
//           factor of at most 1 + n / 32 on average, whatever the entries.  e is
//           a two-float difference (exact), the sums are two-float accumulators
//           (about 48 bits; packed f32x2: float64 arithmetic is scarce on this
//           part).  Also the four counts, and every lane's largest entry: the
//           16th largest of the 32 lane maxima is a value that at least 16
//           entries reach;
//   scan 2  the entries that reach it (about 22 on unordered data) go to a
//           list in shared memory; if the list fills up it is cut to its 16
//           best and the bar rises to the 16th of them;
//   then each listed entry's rank is the number of better ones (larger, or
//   equal with a lower index): ranks 0-15 are features 0-15.
// Writes features 0-15 and 18-22, the 16 neighbour indices (problem-local)
// and the sums (their pivot and unit in the places of features 16-17), from which
// features_finish_row makes 16-17 with whole warps of rows (a float64 division by
// one lane costs what 32 cost).
// The listing takes places by a shared atomic (the ranking does not depend on
// their order) and the counts are float32, whose additions are full rate.
// Six blocks per SM (40 registers) hide the scans' latencies: with the registers
// that the compiler takes by itself four fit and it takes 638 us.
// 48 problems of 200-4000 points (2.7e8 entries): 550 us (+ 24 us for the second
// pass; sums of v and v^2 themselves 543 + 27, but 2e-3 off in feature 17 at mean
// 1000 and spread 0.001; ballots, prefix counts and integer sums 637), where one
// block per row with 16 block-wide arg-max rounds and float64 sums took 8.1 ms.
constexpr int kListCap = 256;      // entries listed per warp
constexpr int kFeatWarps = 8;      // rows per block

struct FeatList {
    float v[kListCap];
    int j[kListCap];
    int have;
    float bv[TOPK];
    int bj[TOPK];
};

// The power of two nearest below 1 / scale, kept normal.
__device__ __forceinline__ float unit_of(float scale) {
    const int e = (int)(__float_as_uint(scale) >> 23);
    return __uint_as_float((uint32_t)max(1, 253 - e) << 23);
}

// s + c += x, exactly but for c's rounding (Knuth's two-sum), two columns at a time.
// A lane's c is a float32 sum of n / 64 errors: s + c carries about 48 bits.
__device__ __forceinline__ void two_add(float2& s, float2& c, float2 x) {
    const float2 mone = make_float2(-1.f, -1.f);
    const float2 t = __fadd2_rn(s, x);
    const float2 bp = __ffma2_rn(mone, s, t);
    const float2 ap = __ffma2_rn(mone, bp, t);
    c = __fadd2_rn(c, __fadd2_rn(__ffma2_rn(mone, ap, s), __ffma2_rn(mone, bp, x)));
    s = t;
}
// c += 1 where v >= t.
__device__ __forceinline__ void count_if_ge(float& c, float v, float t) {
    asm("{\n\t.reg .pred p;\n\tsetp.ge.f32 p, %1, %2;\n\t@p add.f32 %0, %0, 0f3F800000;\n\t}"
        : "+f"(c)
        : "f"(v), "f"(t));
}
// u v - p = d + e exactly (Knuth's two-sum with -p; u a power of two, nu = -u).
__device__ __forceinline__ float2 two_diff(float2 v, float2 u, float2 nu, float2 p, float2 np, float2& e) {
    const float2 mone = make_float2(-1.f, -1.f);
    const float2 d = __ffma2_rn(u, v, np);
    const float2 bp = __ffma2_rn(nu, v, d);
    const float2 nap = __ffma2_rn(mone, d, bp);
    e = __ffma2_rn(mone, __fadd2_rn(p, bp), __ffma2_rn(u, v, nap));
    return d;
}
__device__ __forceinline__ void two_add1(float& s, float& c, float x) {
    const float t = s + x, bp = t - s;
    c += (s - (t - bp)) + (x - bp);
    s = t;
}

// The 16 best of the list's cnt entries (cnt <= kListCap) to bv, bj, best first.
// The order in which the entries were listed does not matter.
__device__ __forceinline__ void rank_list(FeatList& L, int cnt, int lid) {
    for (int e0 = 0; e0 < cnt; e0 += 32) {
        const int at = e0 + lid;
        const float v = at < cnt ? L.v[at] : -INFINITY;
        const int j = at < cnt ? L.j[at] : INT_MAX;
        int rank = 0;
#pragma unroll 4
        for (int e = 0; e < cnt; ++e) {
            const float w = L.v[e];
            rank += w > v || (w == v && L.j[e] < j);
        }
        if (at < cnt && rank < TOPK) {
            L.bv[rank] = v;
            L.bj[rank] = j;
        }
    }
    __syncwarp();
}

// Four consecutive entries 4f .. 4f+3 of a row (vec: 16-byte aligned rows whose
// stride is a multiple of 4).  Past the row's end: whatever the padding holds, or
// 0, the largest similarity there is; the callers mask those out (j < n).
__device__ __forceinline__ float4 row4(const float* __restrict__ row, int f, int n, int vec) {
    if (vec) return __ldg(reinterpret_cast<const float4*>(row) + f);
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = 4 * f + e < n ? __ldg(row + 4 * f + e) : 0.f;
    return make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ void features_row(const float* __restrict__ S, int n, int64_t ld, int vec, float scale,
                                             int k, float* F, int32_t* nbr, float4* sums, FeatList& L) {
    const int lid = threadIdx.x & 31;
    const float* row = S + (int64_t)k * ld;
    const float inv_scale = 1.f / scale;
    float thr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) thr[q] = -(scale * (0.125f * (float)(1 << q)));   // exact: powers of 2
    const int n4 = (n + 3) >> 2, fk = k >> 2, nfull = n >> 2;
    // the pivot, and the sums' unit from the entries' size (not far below the scale's)
    const int at = (int)(((int64_t)lid * n) >> 5);
    const float sample = row[at == k ? (k > 0 ? k - 1 : 1) : at];
    float pivot = sample * 0.03125f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pivot += __shfl_xor_sync(0xffffffffu, pivot, o);
    const float unit = unit_of(fmaxf(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(sample)))),
                                     scale * 0x1p-40f));
    const float2 unit2 = make_float2(unit, unit), nunit2 = make_float2(-unit, -unit);
    const float2 pu = make_float2(pivot * unit, pivot * unit), npu = make_float2(-pu.x, -pu.y);
    float2 s1 = make_float2(0.f, 0.f), c1 = s1, s2 = s1, c2 = s1;
    // float32 counts (exact: a lane has at most n / 32 + 4 entries), since their
    // additions then go to the FMA pipe and not to the half-rate ALU pipe
    float fcnt[4] = {0.f, 0.f, 0.f, 0.f};
    float mx = -INFINITY;
#pragma unroll 2
    for (int f = lid; f < n4; f += 32) {
        const float4 x = row4(row, f, n, vec);
        float v[4] = {x.x, x.y, x.z, x.w};          // what is compared
        float u[4] = {x.x, x.y, x.z, x.w};          // what is summed
        if (f == fk || f >= nfull) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * f + e == k || 4 * f + e >= n) {
                    v[e] = -INFINITY;
                    u[e] = pivot;
                }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 l;
            const float2 w = two_diff(make_float2(u[2 * h], u[2 * h + 1]), unit2, nunit2, pu, npu, l);
            const float2 p = __fmul2_rn(w, w);
            const float2 e = __ffma2_rn(w, w, make_float2(-p.x, -p.y));     // w^2 = p + e exactly
            two_add(s1, c1, w);
            c1 = __fadd2_rn(c1, l);
            two_add(s2, c2, p);
            c2 = __fadd2_rn(c2, __ffma2_rn(__fadd2_rn(w, w), l, e));        // (w + l)^2 but for l^2
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int q = 0; q < 4; ++q) count_if_ge(fcnt[q], v[e], thr[q]);
        }
        mx = fmaxf(mx, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
    }
    // the sums over the warp, in a fixed order
    float t1 = s1.x, d1 = c1.x, t2 = s2.x, d2 = c2.x;
    two_add1(t1, d1, s1.y);
    two_add1(t2, d2, s2.y);
    d1 += c1.y;
    d2 += c2.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float y1 = __shfl_down_sync(0xffffffffu, t1, o), e1 = __shfl_down_sync(0xffffffffu, d1, o);
        const float y2 = __shfl_down_sync(0xffffffffu, t2, o), e2 = __shfl_down_sync(0xffffffffu, d2, o);
        two_add1(t1, d1, y1);
        two_add1(t2, d2, y2);
        d1 += e1;
        d2 += e2;
    }
    int cnt[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) cnt[q] = __reduce_add_sync(0xffffffffu, (int)fcnt[q]);
    // the 16th largest lane maximum: sort the 32 of them, largest first
#pragma unroll
    for (int w = 2; w <= 32; w <<= 1)
#pragma unroll
        for (int o = w >> 1; o > 0; o >>= 1) {
            const float y = __shfl_xor_sync(0xffffffffu, mx, o);
            const bool up = ((lid & w) == 0) == ((lid & o) == 0);           // this lane keeps the larger
            mx = up ? fmaxf(mx, y) : fminf(mx, y);
        }
    float bar = __shfl_sync(0xffffffffu, mx, TOPK - 1);
    int barj = INT_MAX;                             // an entry equal to bar must come before barj
    if (lid == 0) L.have = 0;
    __syncwarp();
#pragma unroll 1
    for (int f0 = 0; f0 < n4; f0 += 32) {
        const int f = f0 + lid;
        float v[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (f < n4) {
            const float4 x = row4(row, f, n, vec);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        }
        const bool maybe = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])) >= bar;
        if (!__any_sync(0xffffffffu, maybe)) continue;
        if (maybe) {
            // few lanes: each takes its places by an atomic (the ranking does not
            // depend on the order)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = 4 * f + e;
                if (v[e] > -INFINITY && (v[e] > bar || (v[e] == bar && j < barj)) && j != k && j < n) {
                    const int at = atomicAdd(&L.have, 1);
                    L.v[at] = v[e];
                    L.j[at] = j;
                }
            }
        }
        __syncwarp();
        if (L.have > kListCap - 128) {                  // room for the next 128: keep the best 16
            rank_list(L, L.have, lid);
            if (lid < TOPK) {
                L.v[lid] = L.bv[lid];
                L.j[lid] = L.bj[lid];
            }
            if (lid == 0) L.have = TOPK;
            __syncwarp();
            bar = L.v[TOPK - 1];
            barj = L.j[TOPK - 1];
            __syncwarp();
        }
    }
    __syncwarp();
    const int have = L.have;
    rank_list(L, have, lid);
    float* out = F + (int64_t)k * IN;
    if (lid < TOPK) {
        // fewer than 16 others: the last one is repeated (the point itself if there is none)
        const int r = min(lid, have - 1);
        out[lid] = (r >= 0 ? L.bv[r] : -INFINITY) * inv_scale;
        nbr[(int64_t)k * TOPK + lid] = r >= 0 ? L.bj[r] : k;
    }
    if (lid == 18) out[18] = row[k] * inv_scale;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (lid == 19 + q) out[19 + q] = log1pf((float)cnt[q]);
    if (lid == 0) {
        sums[k] = make_float4(t1, d1, t2, d2);
        out[16] = pivot;
        out[17] = unit;
    }
    __syncwarp();
}

static __device__ __forceinline__ int row_vec(const float* S, int64_t ld) {
    return (reinterpret_cast<uintptr_t>(S) & 15) == 0 && (ld & 3) == 0;
}

__global__ void __launch_bounds__(32 * kFeatWarps, 6) features_kernel(const float* __restrict__ S, int n, int64_t ld,
                                                                   float scale, float* F, int32_t* nbr,
                                                                   float4* sums) {
    __shared__ FeatList lists[kFeatWarps];
    const int wid = threadIdx.x >> 5, vec = row_vec(S, ld);
    for (int k = blockIdx.x * kFeatWarps + wid; k < n; k += gridDim.x * kFeatWarps)
        features_row(S, n, ld, vec, scale, k, F, nbr, sums, lists[wid]);
}

// Features 16-17 of row k from its sums, 23-24 from the densities of its 16
// neighbours.  Sums out of float32's range (entries that are infinite, NaN or
// more than about 1e18 times most others) are taken again in float64.
__device__ __forceinline__ void features_finish_row(const float* __restrict__ S, int64_t ld, int k, int n, float scale,
                                                    const float4* __restrict__ sums, const int32_t* __restrict__ nbr,
                                                    float* F) {
    const float4 t = sums[k];
    const double inv_scale = (double)(1.f / scale);
    double pivot = (double)F[(int64_t)k * IN + 16];
    const double unit = (double)F[(int64_t)k * IN + 17];
    double a = (double)t.x + (double)t.y, b = (double)t.z + (double)t.w;
    if (isfinite(a) && isfinite(b)) {
        a /= unit;
        b /= unit * unit;
    } else {
        a = b = pivot = 0.0;
        for (int j = 0; j < n; ++j)
            if (j != k) {
                const double v = (double)S[(int64_t)k * ld + j];
                a += v;
                b += v * v;
            }
    }
    const double dm = a / (double)(n - 1), m = pivot + dm;
    const double var = fmax(0.0, b / (double)(n - 1) - dm * dm);
    F[(int64_t)k * IN + 16] = (float)(m * inv_scale);
    F[(int64_t)k * IN + 17] = (float)(sqrt(var) * inv_scale);
    const float d = F[(int64_t)k * IN + F_DENS];
    float mx = -INFINITY;
    int denser = 0;
#pragma unroll
    for (int q = 0; q < TOPK; ++q) {
        const float dj = F[(int64_t)nbr[(int64_t)k * TOPK + q] * IN + F_DENS];
        mx = fmaxf(mx, dj);
        denser += dj > d;
    }
    F[(int64_t)k * IN + 23] = d - mx;
    F[(int64_t)k * IN + 24] = (float)denser * (1.f / TOPK);
}

__global__ void features_finish_kernel(const float* __restrict__ S, int64_t ld, int n, float scale, const float4* __restrict__ sums,
                                       const int32_t* __restrict__ nbr, float* F) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) features_finish_row(S, ld, k, n, scale, sums, nbr, F);
}

// ---- the same over a batch of problems (feature rows of problem b from frow) ----
struct BatchProblem {
    const float* S;         // the problem's S (row stride ld)
    float *R, *A;           // its messages (row stride ld)
    int64_t ld;
    int64_t frow;           // first row of the problem in the feature / output arenas
    int n;
    float scale;
    int b0, nb;             // feature blocks: [b0, b0 + nb)
    int w0;                 // first warm-start block (kWarmRows rows each)
    int pad;
};

// Largest b with key(P[b]) <= x (P sorted by key).
template <class F>
__device__ __forceinline__ int batch_problem_of(const BatchProblem* P, int count, int64_t x, F key) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (key(P[mid]) <= x) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(32 * kFeatWarps, 6) features_batched_kernel(const BatchProblem* __restrict__ P, int count,
                                                                           float* F, int32_t* nbr, float4* sums) {
    __shared__ FeatList lists[kFeatWarps];
    const int b = batch_problem_of(P, count, blockIdx.x, [](const BatchProblem& q) { return (int64_t)q.b0; });
    const BatchProblem& q = P[b];
    const int wid = threadIdx.x >> 5;
    const int k = (blockIdx.x - q.b0) * kFeatWarps + wid;
    if (k < q.n)
        features_row(q.S, q.n, q.ld, row_vec(q.S, q.ld), q.scale, k, F + q.frow * IN, nbr + q.frow * TOPK,
                     sums + q.frow, lists[wid]);
}

__global__ void features_finish_batched_kernel(const BatchProblem* __restrict__ P, int count, int64_t rows,
                                               const float4* __restrict__ sums, const int32_t* __restrict__ nbr,
                                               float* F) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= rows) return;
    const int b = batch_problem_of(P, count, t, [](const BatchProblem& q) { return q.frow; });
    const BatchProblem& q = P[b];
    features_finish_row(q.S, q.ld, (int)(t - q.frow), q.n, q.scale, sums + q.frow, nbr + q.frow * TOPK, F + q.frow * IN);
}

// Column j of the standardisation from F [rows x IN] (one block per column,
// float64 sums in a fixed order): mu = mean, isd = 1 / max(std, 1e-3) with the
// population standard deviation.
__global__ void standardisation_kernel(const float* __restrict__ F, int64_t rows, float* P) {
    __shared__ double s1[256], s2[256];
    const int j = blockIdx.x;
    double a = 0.0, b = 0.0;
    for (int64_t r = threadIdx.x; r < rows; r += blockDim.x) {
        const double v = (double)F[r * IN + j];
        a += v;
        b += v * v;
    }
    s1[threadIdx.x] = a;
    s2[threadIdx.x] = b;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            s1[threadIdx.x] += s1[threadIdx.x + w];
            s2[threadIdx.x] += s2[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double m = s1[0] / (double)rows;
        const double var = fmax(0.0, s2[0] / (double)rows - m * m);
        P[OFF_MU + j] = (float)m;
        P[OFF_ISD + j] = (float)(1.0 / fmax(sqrt(var), 1e-3));
    }
}

// ---- the network: forward, backward and Adam ------------------------------------
// A step of the network is bound by float32 arithmetic (activations and
// gradients stay float32, weights are bf16: about 74000 multiply-adds per row
// and direction), not by memory.  rows_kernel therefore takes a tile of 32
// rows through all three layers -- and, in training, back through them -- with
// the activations in shared memory: a thread owns 8 rows x 2 JC columns of the
// 256-wide layers, multiplies in packed f32x2, and prefetches the next 16 x 256
// weights into registers while the current ones are used.  The forward pass has
// several tiles per SM and JC = 4 (64 accumulators against 16 shared-memory
// words per step of k, so the FMA pipe and not shared memory is the limit); in
// training, where a batch has about one tile per SM, 256 threads with JC = 2 give
// every scheduler a second warp to fill the first one's waits (74 us a step
// where 128 threads took 80).  Every sum runs over k in turn from zero, so that
// a unit's sign, which decides where gradients flow, does not depend on the
// split.  A thread owns the same elements in every layer,
// so the ReLU masks stay in registers.  In training the block leaves its
// tiles' share of every gradient but W2's in one partial slot, and the rows'
// H1 and G2 for w2_grad_kernel, which splits the rows of G2^T H1 over blocks;
// adam_reduce_kernel adds the slots in a fixed order and takes the step.
// A training step on 4096 rows: three launches where separate layer kernels
// took 15 (weight gradients on at most 16 blocks, bias gradients one thread
// per column), 74 us where they took 1752 us.  The forward pass alone on
// 104000 rows: 408 us where four layer launches took about 870 us.
constexpr int TR = 32;                 // rows per tile
constexpr int RS = 36;                 // their stride in shared memory (16-byte groups, fewer bank conflicts)
constexpr int KC = 16;                 // weights staged per step: KC x 256
constexpr int kMaxSlots = 608;         // gradient partial slots: 4 tiles in flight per SM
constexpr int NSMALL = NP - 2 * IN - HID * HID;   // gradients but W2's, in parameter order
constexpr int SLOT = (NSMALL + 3) / 4 * 4;
constexpr int W2T = 128;               // w2_grad_kernel's tile

struct RowsSmem {
    float ws[2][KC][HID];              // staged weights (W1: ws as [IN][HID])
    float hs[HID * RS];                // activations / gradients of the tile, column by column
    float xs[IN * RS];                 // standardised inputs, column by column
    float w3[OUT][HID];
    float ys[OUT][TR], gs[OUT][TR];
};

// Eight bf16 starting at W (16-byte aligned when vec).
__device__ __forceinline__ uint4 load8(const __nv_bfloat16* __restrict__ W, int vec) {
    if (vec) return __ldg(reinterpret_cast<const uint4*>(W));
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        w[e] = (uint32_t)__bfloat16_as_ushort(W[2 * e]) | ((uint32_t)__bfloat16_as_ushort(W[2 * e + 1]) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// The next KC x 256 weights of W2 [256 x 256], k from k0: columns of the
// product are W2's rows going forward (k along a row), its columns going back
// (BACK: k is W2's row).
template <bool BACK, int RT>
__device__ __forceinline__ void fetch_w2(const __nv_bfloat16* __restrict__ W, int k0, int vec, uint4 (&pf)[512 / RT]) {
#pragma unroll
    for (int q = 0; q < 512 / RT; ++q) {
        const int e = threadIdx.x + q * RT;
        // 16 rows x 32 groups of eight; or 256 rows x 2 groups (a warp on 32 rows)
        if (BACK) pf[q] = load8(W + (int64_t)(k0 + (e >> 5)) * HID + 8 * (e & 31), vec);
        else pf[q] = load8(W + (int64_t)(e & 255) * HID + k0 + 8 * (e >> 8), vec);
    }
}
template <bool BACK, int RT>
__device__ __forceinline__ void put_w2(float (*ws)[HID], const uint4 (&pf)[512 / RT]) {
#pragma unroll
    for (int q = 0; q < 512 / RT; ++q) {
        const int e = threadIdx.x + q * RT;
        const float v[8] = {bf16_lo(pf[q].x), bf16_hi(pf[q].x), bf16_lo(pf[q].y), bf16_hi(pf[q].y),
                            bf16_lo(pf[q].z), bf16_hi(pf[q].z), bf16_lo(pf[q].w), bf16_hi(pf[q].w)};
        if (BACK) {
            float* at = &ws[e >> 5][8 * (e & 31)];
            *reinterpret_cast<float4*>(at) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(at + 4) = make_float4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) ws[8 * (e >> 8) + j][e & 255] = v[j];
        }
    }
}

// acc += (column k of act) x (row k of w): this thread's rows 8 wid .. and
// columns col + 64 j, + 1 (col: 2 lid, + 128 for the second four warps of eight).
template <int JC>
__device__ __forceinline__ void rank1(const float* act, const float* w, int wid, int col, float2 (&acc)[8][JC]) {
    const float4 a0 = *reinterpret_cast<const float4*>(act + 8 * wid);
    const float4 a1 = *reinterpret_cast<const float4*>(act + 8 * wid + 4);
    float2 b[JC];
#pragma unroll
    for (int j = 0; j < JC; ++j) b[j] = *reinterpret_cast<const float2*>(w + 64 * j + col);
    const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < JC; ++j) acc[r][j] = __ffma2_rn(make_float2(a[r], a[r]), b[j], acc[r][j]);
}

template <int JC>
__device__ __forceinline__ void clear(float2 (&acc)[8][JC]) {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < JC; ++j) acc[r][j] = make_float2(0.f, 0.f);
}

// acc = hs x W2 (or its transpose); leaves the block synchronised, hs free.
template <bool BACK, int JC>
__device__ __forceinline__ void layer2(RowsSmem& sm, const __nv_bfloat16* __restrict__ W, int vec, int wid, int col,
                                       float2 (&acc)[8][JC]) {
    constexpr int RT = 512 / JC;
    uint4 pf[JC];
    clear(acc);
    fetch_w2<BACK, RT>(W, 0, vec, pf);
    put_w2<BACK, RT>(sm.ws[0], pf);
    __syncthreads();
    for (int c = 0; c < HID / KC; ++c) {
        if (c + 1 < HID / KC) fetch_w2<BACK, RT>(W, (c + 1) * KC, vec, pf);
#pragma unroll
        for (int kk = 0; kk < KC; ++kk) rank1(sm.hs + (c * KC + kk) * RS, sm.ws[c & 1][kk], wid, col, acc);
        if (c + 1 < HID / KC) put_w2<BACK, RT>(sm.ws[(c + 1) & 1], pf);
        __syncthreads();
    }
}

// The thread's 8 x 2 JC elements into hs, and (out != null) into row-major
// out [rows x 256].
template <int JC>
__device__ __forceinline__ void put_tile(float* hs, float* out, const float2 (&v)[8][JC], int wid, int col, int64_t r0,
                                         int rows) {
#pragma unroll
    for (int j = 0; j < JC; ++j) {
        float* x = hs + (64 * j + col) * RS + 8 * wid;
        *reinterpret_cast<float4*>(x) = make_float4(v[0][j].x, v[1][j].x, v[2][j].x, v[3][j].x);
        *reinterpret_cast<float4*>(x + 4) = make_float4(v[4][j].x, v[5][j].x, v[6][j].x, v[7][j].x);
        *reinterpret_cast<float4*>(x + RS) = make_float4(v[0][j].y, v[1][j].y, v[2][j].y, v[3][j].y);
        *reinterpret_cast<float4*>(x + RS + 4) = make_float4(v[4][j].y, v[5][j].y, v[6][j].y, v[7][j].y);
    }
    if (out) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int64_t row = r0 + 8 * wid + r;
            if (row < rows)
#pragma unroll
                for (int j = 0; j < JC; ++j)
                    *reinterpret_cast<float2*>(out + row * HID + 64 * j + col) = v[r][j];
        }
    }
}

// Bias and ReLU; the mask has bit 8 r + 2 j + e for row r, column pair j, element e.
template <int JC>
__device__ __forceinline__ uint64_t bias_relu(float2 (&acc)[8][JC], const float* __restrict__ b, int col) {
    uint64_t m = 0;
#pragma unroll
    for (int j = 0; j < JC; ++j) {
        const float b0 = b[64 * j + col], b1 = b[64 * j + col + 1];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            acc[r][j].x = fmaxf(acc[r][j].x + b0, 0.f);
            acc[r][j].y = fmaxf(acc[r][j].y + b1, 0.f);
            m |= (uint64_t)(acc[r][j].x > 0.f) << (8 * r + 2 * j);
            m |= (uint64_t)(acc[r][j].y > 0.f) << (8 * r + 2 * j + 1);
        }
    }
    return m;
}

struct TrainOut {
    const float* T;           // targets [rows x 3]
    float *H1, *G2;           // [rows x 256]
    float* part;              // [gridDim.x][SLOT] gradients but W2's
    double* lpart;            // [gridDim.x] summed row losses
};

template <bool TRAIN>
__global__ void __launch_bounds__(TRAIN ? 256 : 128) rows_kernel(const float* __restrict__ P, const __nv_bfloat16* __restrict__ P16,
                                                  const float* __restrict__ F, int rows, int vec, float* Y,
                                                  TrainOut t) {
    extern __shared__ __align__(16) unsigned char rows_smem[];
    RowsSmem& sm = *reinterpret_cast<RowsSmem*>(rows_smem);
    constexpr int JC = TRAIN ? 2 : 4, RT = 512 / JC;
    const int tid = threadIdx.x, wid = (tid >> 5) & 3, lid = tid & 31;
    const int col = 2 * lid + (tid >> 7) * 128;            // (128 threads: 2 lid)
    const int tiles = (rows + TR - 1) / TR;
    for (int e = tid; e < OUT * HID; e += RT) (&sm.w3[0][0])[e] = __bfloat162float(P16[OFF_W3 + e]);
    float* part = TRAIN ? t.part + (int64_t)blockIdx.x * SLOT : nullptr;
    bool first = true;
    double lsum = 0.0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t r0 = (int64_t)tile * TR;
        __syncthreads();                                   // the previous tile is done with shared memory
        for (int e = tid; e < TR * IN; e += RT) {
            const int r = e / IN, k = e - r * IN;
            sm.xs[k * RS + r] = r0 + r < rows ? (F[r0 * IN + e] - P[OFF_MU + k]) * P[OFF_ISD + k] : 0.f;
        }
        float* w1 = &sm.ws[0][0][0];
        for (int e = tid; e < HID * IN; e += RT) {
            const int k = e / HID, o = e - k * HID;
            w1[e] = __bfloat162float(P16[OFF_W1 + o * IN + k]);
        }
        __syncthreads();
        float2 acc[8][JC];
        clear(acc);
#pragma unroll 5
        for (int k = 0; k < IN; ++k) rank1(sm.xs + k * RS, w1 + k * HID, wid, col, acc);
        const uint64_t m1 = bias_relu(acc, P + OFF_B1, col);
        put_tile(sm.hs, TRAIN ? t.H1 : nullptr, acc, wid, col, r0, rows);
        __syncthreads();
        layer2<false>(sm, P16 + OFF_W2, vec, wid, col, acc);
        const uint64_t m2 = bias_relu(acc, P + OFF_B2, col);
        put_tile(sm.hs, nullptr, acc, wid, col, r0, rows);
        __syncthreads();
        if (tid < OUT * TR) {                              // warp o: output o of the 32 rows
            float y0 = 0.f, y1 = 0.f, y2 = 0.f, y3 = 0.f;
#pragma unroll 4
            for (int k = 0; k < HID; k += 4) {
                const float4 w = *reinterpret_cast<const float4*>(&sm.w3[wid][k]);
                y0 = fmaf(sm.hs[k * RS + lid], w.x, y0);
                y1 = fmaf(sm.hs[(k + 1) * RS + lid], w.y, y1);
                y2 = fmaf(sm.hs[(k + 2) * RS + lid], w.z, y2);
                y3 = fmaf(sm.hs[(k + 3) * RS + lid], w.w, y3);
            }
            const float y = (y0 + y1) + (y2 + y3) + P[OFF_B3 + wid];
            if (TRAIN) sm.ys[wid][lid] = y;
            else if (r0 + lid < rows) Y[(r0 + lid) * OUT + wid] = y;
        }
        if (!TRAIN) continue;
        __syncthreads();
        if (tid < TR) {
            // the row's loss and dL/dY (divided by the row count)
            const bool in = r0 + lid < rows;
            const float inv = 1.f / (float)rows;
            const float* tr = t.T + (r0 + (in ? lid : 0)) * OUT;
            const float d = sm.ys[0][lid] - tr[0], e = sm.ys[1][lid] - tr[1], z = sm.ys[2][lid], tt = tr[2];
            const float sp = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));     // softplus(z)
            double l = in ? (double)(d * d + e * e + sp - tt * z) : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
            lsum += l;
            sm.gs[0][lid] = in ? 2.f * d * inv : 0.f;
            sm.gs[1][lid] = in ? 2.f * e * inv : 0.f;
            sm.gs[2][lid] = in ? (1.f / (1.f + expf(-z)) - tt) * inv : 0.f;
        }
        __syncthreads();
        auto add = [&](int at, float v) { part[at] = first ? v : part[at] + v; };
        constexpr int S_B2 = OFF_B2 - HID * HID, S_W3 = OFF_W3 - HID * HID, S_B3 = OFF_B3 - HID * HID;
        // layer 3: gW3 = G3^T H2, gb3
#pragma unroll
        for (int h = 0; h < HID / RT; ++h) {
            const int c = tid + h * RT;
            float g[OUT] = {};
#pragma unroll
            for (int r = 0; r < TR; r += 4) {
                const float4 x = *reinterpret_cast<const float4*>(sm.hs + c * RS + r);
#pragma unroll
                for (int o = 0; o < OUT; ++o) {
                    const float4 q = *reinterpret_cast<const float4*>(&sm.gs[o][r]);
                    g[o] = fmaf(q.x, x.x, g[o]);
                    g[o] = fmaf(q.y, x.y, g[o]);
                    g[o] = fmaf(q.z, x.z, g[o]);
                    g[o] = fmaf(q.w, x.w, g[o]);
                }
            }
#pragma unroll
            for (int o = 0; o < OUT; ++o) add(S_W3 + o * HID + c, g[o]);
        }
        if (tid < OUT) {
            float g = 0.f;
            for (int r = 0; r < TR; ++r) g += sm.gs[tid][r];
            add(S_B3 + tid, g);
        }
        // G2 = (G3 W3) where H2 > 0
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float g0 = sm.gs[0][8 * wid + r], g1 = sm.gs[1][8 * wid + r], g2 = sm.gs[2][8 * wid + r];
#pragma unroll
            for (int j = 0; j < JC; ++j) {
                const int c = 64 * j + col;
                const float2 w0 = *reinterpret_cast<const float2*>(&sm.w3[0][c]);
                const float2 w1v = *reinterpret_cast<const float2*>(&sm.w3[1][c]);
                const float2 w2v = *reinterpret_cast<const float2*>(&sm.w3[2][c]);
                const float vx = fmaf(g2, w2v.x, fmaf(g1, w1v.x, g0 * w0.x));
                const float vy = fmaf(g2, w2v.y, fmaf(g1, w1v.y, g0 * w0.y));
                acc[r][j] = make_float2((m2 >> (8 * r + 2 * j)) & 1 ? vx : 0.f,
                                        (m2 >> (8 * r + 2 * j + 1)) & 1 ? vy : 0.f);
            }
        }
        __syncthreads();                                   // H2 has been read
        put_tile(sm.hs, t.G2, acc, wid, col, r0, rows);
        __syncthreads();
#pragma unroll
        for (int h = 0; h < HID / RT; ++h) {               // gb2
            const int c = tid + h * RT;
            float g = 0.f;
#pragma unroll
            for (int r = 0; r < TR; r += 4) {
                const float4 x = *reinterpret_cast<const float4*>(sm.hs + c * RS + r);
                g += (x.x + x.y) + (x.z + x.w);
            }
            add(S_B2 + c, g);
        }
        // G1 = (G2 W2) where H1 > 0, then gW1 = G1^T X and gb1
        layer2<true>(sm, P16 + OFF_W2, vec, wid, col, acc);
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int j = 0; j < JC; ++j) {
                if (!((m1 >> (8 * r + 2 * j)) & 1)) acc[r][j].x = 0.f;
                if (!((m1 >> (8 * r + 2 * j + 1)) & 1)) acc[r][j].y = 0.f;
            }
        put_tile(sm.hs, nullptr, acc, wid, col, r0, rows);
        __syncthreads();
#pragma unroll
        for (int h = 0; h < HID / RT; ++h) {
            const int c = tid + h * RT;
            float g[IN] = {}, gb = 0.f;
#pragma unroll 2
            for (int r = 0; r < TR; r += 4) {
                const float4 y = *reinterpret_cast<const float4*>(sm.hs + c * RS + r);
                gb += (y.x + y.y) + (y.z + y.w);
#pragma unroll
                for (int k = 0; k < IN; ++k) {
                    const float4 x = *reinterpret_cast<const float4*>(sm.xs + k * RS + r);
                    g[k] = fmaf(y.x, x.x, g[k]);
                    g[k] = fmaf(y.y, x.y, g[k]);
                    g[k] = fmaf(y.z, x.z, g[k]);
                    g[k] = fmaf(y.w, x.w, g[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < IN; ++k) add(OFF_W1 + c * IN + k, g[k]);
            add(OFF_B1 + c, gb);
        }
        first = false;
    }
    if (TRAIN && tid == 0) t.lpart[blockIdx.x] = lsum;
}

// Partial slot z of gW2 = G2^T H1 over rows [z * per, (z + 1) * per): one
// 128 x 128 tile per block (grid (2, 2, splits)), 8 x 8 elements per thread.
__global__ void __launch_bounds__(256) w2_grad_kernel(const float* __restrict__ G, const float* __restrict__ H, int rows,
                                                      int per, float* part) {
    __shared__ __align__(16) float gs[2][KC][W2T], hs[2][KC][W2T];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int o0 = blockIdx.x * W2T, i0 = blockIdx.y * W2T;
    const int lo = blockIdx.z * per, hi = min(rows, lo + per);
    // a chunk: 16 rows x 32 groups of four columns of G and of H, two of each per thread
    float4 pg[2], ph[2];
    auto fetch = [&](int r0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + q * 256, r = r0 + (e >> 5), c = 4 * (e & 31);
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            pg[q] = r < hi ? *reinterpret_cast<const float4*>(G + (int64_t)r * HID + o0 + c) : z;
            ph[q] = r < hi ? *reinterpret_cast<const float4*>(H + (int64_t)r * HID + i0 + c) : z;
        }
    };
    auto put = [&](int b) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + q * 256;
            *reinterpret_cast<float4*>(&gs[b][e >> 5][4 * (e & 31)]) = pg[q];
            *reinterpret_cast<float4*>(&hs[b][e >> 5][4 * (e & 31)]) = ph[q];
        }
    };
    float2 acc[8][4];
    clear(acc);
    fetch(lo);
    put(0);
    __syncthreads();
    int b = 0;
    for (int r0 = lo; r0 < hi; r0 += KC, b ^= 1) {
        const bool more = r0 + KC < hi;
        if (more) fetch(r0 + KC);
#pragma unroll
        for (int k = 0; k < KC; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(&gs[b][k][4 * ty]);
            const float4 a1 = *reinterpret_cast<const float4*>(&gs[b][k][64 + 4 * ty]);
            const float4 b0 = *reinterpret_cast<const float4*>(&hs[b][k][4 * tx]);
            const float4 b1 = *reinterpret_cast<const float4*>(&hs[b][k][64 + 4 * tx]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 w[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                                 make_float2(b1.z, b1.w)};
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[r][j] = __ffma2_rn(make_float2(a[r], a[r]), w[j], acc[r][j]);
        }
        if (more) put(b ^ 1);
        __syncthreads();
    }
    float* out = part + (int64_t)blockIdx.z * HID * HID;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        float* row = out + (int64_t)(o0 + (r < 4 ? 4 * ty + r : 64 + 4 * ty + r - 4)) * HID + i0 + 4 * tx;
        *reinterpret_cast<float4*>(row) = make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
        *reinterpret_cast<float4*>(row + 64) = make_float4(acc[r][2].x, acc[r][2].y, acc[r][3].x, acc[r][3].y);
    }
}

// The gradient of every parameter from its partial slots (four lanes per
// parameter take every fourth slot, then meet in a fixed tree), Adam with
// bias correction, the bf16 copy, and (block 0) the mean loss.  mu and isd
// are fixed: their gradient is zero.
__global__ void __launch_bounds__(256) adam_reduce_kernel(float* P, float* m, float* v, const float* __restrict__ part,
                                                          int slots, const float* __restrict__ w2part, int splits,
                                                          const double* __restrict__ lpart, int rows, float lr, float b1,
                                                          float b2, float eps, float c1, float c2, __nv_bfloat16* P16,
                                                          float* grad, float* loss) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int i = (int)(t >> 2), q = (int)(t & 3);
    float g = 0.f;
    if (i < NP && i < OFF_MU) {
        const bool w2 = i >= OFF_W2 && i < OFF_B2;
        const float* at = w2 ? w2part + (i - OFF_W2) : part + (i < OFF_W2 ? i : i - HID * HID);
        const int64_t step = w2 ? HID * HID : SLOT;
        const int n = w2 ? splits : slots;
#pragma unroll 8
        for (int s = q; s < n; s += 4) g += at[s * step];
    }
    g += __shfl_xor_sync(0xffffffffu, g, 1);
    g += __shfl_xor_sync(0xffffffffu, g, 2);
    if (q == 0 && i < NP) {
        if (grad) grad[i] = g;
        const float mi = b1 * m[i] + (1.f - b1) * g;
        const float vi = b2 * v[i] + (1.f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        const float p = P[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        P[i] = p;
        P16[i] = __float2bfloat16_rn(p);
    }
    if (loss && blockIdx.x == 0 && threadIdx.x < 32) {
        double l = 0.0;
        for (int s = threadIdx.x; s < slots; s += 32) l += lpart[s];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (threadIdx.x == 0) *loss = (float)(l / (double)rows);
    }
}

__global__ void to_bf16_kernel(const float* __restrict__ P, int64_t np, __nv_bfloat16* P16) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np;
         i += (int64_t)gridDim.x * blockDim.x)
        P16[i] = __float2bfloat16_rn(P[i]);
}

__global__ void targets_kernel(const float* __restrict__ R, const float* __restrict__ A,
                               const int32_t* __restrict__ dec, int n, int64_t ld, float inv_scale,
                               float* T) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    T[k * 3 + 0] = fminf(0.f, R[(int64_t)k * ld + k] + A[(int64_t)k * ld + k]) * inv_scale;
    T[k * 3 + 1] = A[(int64_t)k * ld + k] * inv_scale;
    T[k * 3 + 2] = dec[k] == k ? 1.f : 0.f;
}

// Column-constant availabilities from the per-point predictions (the fixed
// point of Eq. 3-4 up to the i-th term): A(i,k) = min(0, c_hat_k p) for
// i != k, A(k,k) = max(0, a_hat_k p).  One block-row of A per block.
__global__ void warm_columns_kernel(const float* __restrict__ Y, int n, float scale, float* A,
                                    int64_t ld) {
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        float* row = A + (int64_t)i * ld;
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const float ch = Y[k * 3 + 0], ah = Y[k * 3 + 1];
            row[k] = (k == i) ? fmaxf(0.f, ah * scale) : fminf(0.f, ch * scale);
        }
    }
}

// The warm start of every problem of a batch: kWarmRows rows i of problem b per
// block; R(i,:) = 0 and A(i,:) the column-constant availabilities of b's
// predictions (as warm_columns_kernel).  Bound by writing R and A: a thread
// makes its columns' values once and writes them to every row of the block,
// 16 bytes at a time where the rows allow (2.7e8 entries: 355 us; one row per
// block and scalar stores took 486 us).
constexpr int kWarmRows = 16;

__global__ void __launch_bounds__(256) warm_batched_kernel(const BatchProblem* __restrict__ P, int count,
                                                           const float* __restrict__ Y) {
    const int b = batch_problem_of(P, count, blockIdx.x, [](const BatchProblem& q) { return (int64_t)q.w0; });
    const BatchProblem& q = P[b];
    const int i0 = (blockIdx.x - q.w0) * kWarmRows, i1 = min(q.n, i0 + kWarmRows);
    const float* y = Y + q.frow * OUT;
    const float scale = q.scale;
    auto value = [&](int i, int k) {
        return (k == i) ? fmaxf(0.f, y[k * 3 + 1] * scale) : fminf(0.f, y[k * 3] * scale);
    };
    int done = 0;                       // columns written by the vector path
    if (row_vec(q.R, q.ld) && row_vec(q.A, q.ld)) {
        for (int f = threadIdx.x; f < q.n >> 2; f += blockDim.x) {
            const int k = 4 * f;
            const float4 c = make_float4(value(-1, k), value(-1, k + 1), value(-1, k + 2), value(-1, k + 3));
            for (int i = i0; i < i1; ++i) {
                float4 v = c;
                if ((i >> 2) == f) v = make_float4(value(i, k), value(i, k + 1), value(i, k + 2), value(i, k + 3));
                reinterpret_cast<float4*>(q.R + (int64_t)i * q.ld)[f] = make_float4(0.f, 0.f, 0.f, 0.f);
                reinterpret_cast<float4*>(q.A + (int64_t)i * q.ld)[f] = v;
            }
        }
        done = q.n & ~3;
    }
    for (int k = done + threadIdx.x; k < q.n; k += blockDim.x)
        for (int i = i0; i < i1; ++i) {
            q.R[(int64_t)i * q.ld + k] = 0.f;
            q.A[(int64_t)i * q.ld + k] = value(i, k);
        }
}

struct MlpWs {
    float *H1, *G2, *part, *w2part;
    double* lpart;
};

static int row_tiles(int64_t rows) { return (int)((rows + TR - 1) / TR); }
static int grad_slots(int64_t rows) { return std::min(row_tiles(rows), kMaxSlots); }
// Rows per split of gW2: whole KC-row chunks, and splits enough for about one
// block per SM (four tiles of 128 x 128 each) but at least 32 rows, so that a
// small batch is not all partial sums.
static int w2_rows_per_split(int64_t rows) {
    const int64_t per = std::max<int64_t>(32, (rows + 37) / 38);
    return (int)((per + KC - 1) / KC * KC);
}
static int w2_splits(int64_t rows) {
    const int per = w2_rows_per_split(rows);
    return (int)((rows + per - 1) / per);
}

// The most splits of any smaller batch: the splits fall where a split grows by a
// chunk (38 at 1216 rows, 26 at 1217), and a workspace serves smaller batches.
static int64_t w2_splits_cap(int64_t rows) { return std::min<int64_t>((rows + 31) / 32, 38); }

static size_t carve(void* ws, int64_t rows, MlpWs* w) {
    Carver c(ws);
    w->H1 = c.take<float>((size_t)rows * HID);
    w->G2 = c.take<float>((size_t)rows * HID);
    w->part = c.take<float>((size_t)grad_slots(rows) * SLOT);
    w->w2part = c.take<float>((size_t)w2_splits_cap(rows) * HID * HID);
    w->lpart = c.take<double>(grad_slots(rows));
    return c.used;
}

template <bool TRAIN>
static int32_t launch_rows(const float* P, const __nv_bfloat16* P16, const float* F, int rows, float* Y,
                           const TrainOut& t, int grid, cudaStream_t s) {
    AP_CUDA_TRY(cudaFuncSetAttribute(rows_kernel<TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(RowsSmem)));
    rows_kernel<TRAIN><<<grid, TRAIN ? 256 : 128, sizeof(RowsSmem), s>>>(P, P16, F, rows, aligned16(P16) ? 1 : 0, Y, t);
    note_launches(1);
    return last_error();
}

static int32_t forward(const float* P, const __nv_bfloat16* P16, const float* F, int rows, float* Y, cudaStream_t s) {
    return launch_rows<false>(P, P16, F, rows, Y, TrainOut{}, std::min(row_tiles(rows), 8192), s);
}

}  // namespace mlp
}  // namespace apgb

using namespace apgb;
using namespace apgb::mlp;

APGB_API int64_t apl_param_count(void) { return NP; }

APGB_API size_t apl_features_workspace_size(int64_t n) {
    if (n < 2 || n > INT_MAX) return 0;
    Carver c(nullptr);
    c.take<int32_t>((size_t)n * TOPK);
    c.take<float4>((size_t)n);
    return c.used;
}

APGB_API int32_t apl_features(const float* S, int64_t n, int64_t ld, float scale, float* F,
                              void* ws, size_t ws_bytes, void* stream) {
    if (!S || !F || n < 2 || ld < n || n > INT_MAX || !(scale > 0.f)) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    AP_TRY(check_ws(ws, ws_bytes, apl_features_workspace_size(n)));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Carver c(ws);
    int32_t* nbr = c.take<int32_t>((size_t)n * TOPK);
    float4* sums = c.take<float4>((size_t)n);
    features_kernel<<<(int)std::min<int64_t>((n + kFeatWarps - 1) / kFeatWarps, 65535), 32 * kFeatWarps, 0, s>>>(
        S, (int)n, ld, scale, F, nbr, sums);
    features_finish_kernel<<<(int)((n + 255) / 256), 256, 0, s>>>(S, ld, (int)n, scale, sums, nbr, F);
    note_launches(2);
    return last_error();
}

APGB_API int32_t apl_targets(const float* R, const float* A, const int32_t* dec, int64_t n,
                             int64_t ld, float scale, float* T, void* stream) {
    if (!R || !A || !dec || !T || n < 1 || ld < n || n > INT_MAX || !(scale > 0.f))
        return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    targets_kernel<<<(int)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        R, A, dec, (int)n, ld, 1.f / scale, T);
    note_launches(1);
    return last_error();
}

APGB_API size_t apl_workspace_size(int64_t rows) {
    if (rows < 1 || rows > INT_MAX / HID) return 0;
    MlpWs w;
    return carve(nullptr, rows, &w);
}

APGB_API int32_t apl_sync_bf16(const float* P, void* P16, void* stream) {
    if (!P || !P16) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    to_bf16_kernel<<<(int)((NP + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        P, NP, static_cast<__nv_bfloat16*>(P16));
    note_launches(1);
    return last_error();
}

APGB_API int32_t apl_forward(const float* P, const void* P16, const float* F, int64_t rows,
                             float* Y, void* ws, size_t ws_bytes, void* stream) {
    if (!P || !P16 || !F || !Y || rows < 1 || rows > INT_MAX / HID) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    MlpWs w;
    AP_TRY(check_ws(ws, ws_bytes, carve(nullptr, rows, &w)));
    return forward(P, static_cast<const __nv_bfloat16*>(P16), F, (int)rows, Y, static_cast<cudaStream_t>(stream));
}

APGB_API int32_t apl_train_step(float* P, void* P16, float* M, float* V, int64_t step, float lr,
                                const float* F, const float* T, int64_t rows, float* loss,
                                float* grad_out, void* ws, size_t ws_bytes, void* stream) {
    if (!P || !P16 || !M || !V || !F || !T || rows < 1 || rows > INT_MAX / HID || step < 1 ||
        !(lr >= 0.f))
        return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    MlpWs w;
    AP_TRY(check_ws(ws, ws_bytes, carve(nullptr, rows, &w)));
    carve(ws, rows, &w);
    const int r = (int)rows, slots = grad_slots(rows), per = w2_rows_per_split(rows), splits = w2_splits(rows);
    AP_TRY(launch_rows<true>(P, static_cast<const __nv_bfloat16*>(P16), F, r, nullptr,
                             TrainOut{T, w.H1, w.G2, w.part, w.lpart}, slots, s));
    w2_grad_kernel<<<dim3(HID / W2T, HID / W2T, splits), 256, 0, s>>>(w.G2, w.H1, r, per, w.w2part);
    const float c1 = (float)(1.0 - std::pow(0.9, (double)step));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)step));
    adam_reduce_kernel<<<(int)((4 * NP + 255) / 256), 256, 0, s>>>(P, M, V, w.part, slots, w.w2part, splits, w.lpart, r,
                                                                   lr, 0.9f, 0.999f, 1e-8f, c1, c2,
                                                                   static_cast<__nv_bfloat16*>(P16), grad_out, loss);
    note_launches(2);
    return last_error();
}

APGB_API int32_t apl_warm_start(const float* Y, int64_t n, float scale, float* R, float* A,
                                int64_t ld, void* stream) {
    if (!Y || !R || !A || n < 1 || ld < n || n > INT_MAX || !(scale > 0.f)) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    AP_CUDA_TRY(cudaMemset2DAsync(R, ld * sizeof(float), 0, n * sizeof(float), n, s));
    warm_columns_kernel<<<(int)std::min<int64_t>(n, 4096), 256, 0, s>>>(Y, (int)n, scale, A, ld);
    note_launches(1);
    return last_error();
}

// ---- warm-started Algorithm 1, judged by the cold start ---------------------------
namespace apgb {
int32_t exemplars_impl(const float* S, const float* R, const float* A, int64_t n, int64_t ld,
                       int32_t* idx, ap_result* out, void* ws, size_t ws_bytes, cudaStream_t s);
size_t exemplars_ws_bytes(int64_t n);

struct RunWs {
    float *F, *Y, *R2, *A2;
    int32_t* idx2;
    void* mlp_ws;
    size_t mlp_bytes;
    void* sub_ws;
    size_t sub_bytes;
};

static size_t carve_run(void* ws, int64_t n, int64_t ld, RunWs* w) {
    const size_t mb = apl_workspace_size(n);
    const size_t sb = std::max({ap_iterate_workspace_size(n, ld), exemplars_ws_bytes(n),
                                apl_features_workspace_size(n)});
    Carver c(ws);
    w->F = c.take<float>((size_t)n * mlp::IN);
    w->Y = c.take<float>((size_t)n * mlp::OUT);
    w->R2 = c.take<float>((size_t)n * ld);
    w->A2 = c.take<float>((size_t)n * ld);
    w->idx2 = c.take<int32_t>(n);
    w->mlp_ws = c.take<char>(mb);
    w->mlp_bytes = mb;
    w->sub_ws = c.take<char>(sb);
    w->sub_bytes = sb;
    return (mb && sb) ? c.used : 0;
}
}  // namespace apgb

APGB_API size_t apl_ap_run_workspace_size(int64_t n, int64_t ld) {
    if (n < 2 || ld < n || n > INT_MAX / 256) return 0;
    RunWs w;
    return carve_run(nullptr, n, ld, &w);
}

APGB_API int32_t apl_ap_run(const float* S, int64_t n, int64_t ld, const float* P, const void* P16,
                            float scale, const ap_params* params, int32_t judge, float* R, float* A,
                            int32_t* idx, apl_result* out, void* ws, size_t ws_bytes, void* stream) {
    if (!S || !P || !P16 || !params || !R || !A || !idx || !out || n < 2 || ld < n ||
        n > INT_MAX / 256 || !(scale > 0.f))
        return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    RunWs w;
    const size_t need = carve_run(nullptr, n, ld, &w);
    if (need == 0) return AP_ERR_INVALID_ARG;
    AP_TRY(check_ws(ws, ws_bytes, need));
    carve_run(ws, n, ld, &w);
    cudaEvent_t ev[5];
    for (auto& e : ev) AP_CUDA_TRY(cudaEventCreate(&e));
    struct Guard {
        cudaEvent_t* e;
        ~Guard() { for (int i = 0; i < 5; ++i) cudaEventDestroy(e[i]); }
    } guard{ev};

    *out = apl_result{};
    AP_CUDA_TRY(cudaEventRecord(ev[0], s));
    AP_TRY(apl_features(S, n, ld, scale, w.F, w.sub_ws, w.sub_bytes, stream));
    AP_CUDA_TRY(cudaEventRecord(ev[1], s));
    AP_TRY(apl_forward(P, P16, w.F, n, w.Y, w.mlp_ws, w.mlp_bytes, stream));
    AP_TRY(apl_warm_start(w.Y, n, scale, R, A, ld, stream));
    AP_CUDA_TRY(cudaEventRecord(ev[2], s));
    ap_result rw;
    const int32_t sw = ap_iterate(S, R, A, n, ld, params, nullptr, &rw, w.sub_ws, w.sub_bytes, stream);
    if (sw < 0) return sw;
    const int32_t wi = rw.iters, wc = rw.converged;
    const int32_t swe = exemplars_impl(S, R, A, n, ld, idx, &rw, w.sub_ws, w.sub_bytes, s);
    if (swe < 0) return swe;
    rw.iters = wi;
    rw.converged = wc;
    rw.status = std::max(sw, swe);
    AP_CUDA_TRY(cudaEventRecord(ev[3], s));
    out->warm_iters = wi;
    out->warm_netsim = rw.netsim;
    out->result = rw;
    out->used_warm = 1;
    if (judge) {
        AP_CUDA_TRY(cudaMemset2DAsync(w.R2, ld * sizeof(float), 0, n * sizeof(float), n, s));
        AP_CUDA_TRY(cudaMemset2DAsync(w.A2, ld * sizeof(float), 0, n * sizeof(float), n, s));
        ap_result rc;
        const int32_t sc = ap_iterate(S, w.R2, w.A2, n, ld, params, nullptr, &rc, w.sub_ws,
                                      w.sub_bytes, stream);
        if (sc < 0) return sc;
        const int32_t ci = rc.iters, cc = rc.converged;
        const int32_t sce = exemplars_impl(S, w.R2, w.A2, n, ld, w.idx2, &rc, w.sub_ws,
                                           w.sub_bytes, s);
        if (sce < 0) return sce;
        rc.iters = ci;
        rc.converged = cc;
        rc.status = std::max(sc, sce);
        out->cold_iters = ci;
        out->cold_netsim = rc.netsim;
        // the judge: keep the warm result only within 0.5 % of the cold net similarity
        const bool ok = rw.n_exemplars > 0 && rc.n_exemplars > 0 &&
                        std::fabs(rw.netsim - rc.netsim) <= 0.005 * std::fabs(rc.netsim);
        if (!ok || rw.n_exemplars == 0) {
            out->used_warm = 0;
            out->result = rc;
            AP_CUDA_TRY(cudaMemcpy2DAsync(R, ld * sizeof(float), w.R2, ld * sizeof(float),
                                          n * sizeof(float), n, cudaMemcpyDeviceToDevice, s));
            AP_CUDA_TRY(cudaMemcpy2DAsync(A, ld * sizeof(float), w.A2, ld * sizeof(float),
                                          n * sizeof(float), n, cudaMemcpyDeviceToDevice, s));
            AP_CUDA_TRY(cudaMemcpyAsync(idx, w.idx2, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s));
        }
    }
    AP_CUDA_TRY(cudaEventRecord(ev[4], s));
    AP_CUDA_TRY(cudaEventSynchronize(ev[4]));
    float ms[4];
    for (int i = 0; i < 4; ++i) AP_CUDA_TRY(cudaEventElapsedTime(&ms[i], ev[i], ev[i + 1]));
    out->features_ms = ms[0];
    out->forward_ms = ms[1];
    out->warm_ms = ms[2];
    out->cold_ms = ms[3];
    return out->result.status;
}

// ---- the learned warm start over a batch of problems ------------------------------------
namespace apgb {
namespace mlp {

static size_t carve_batch(void* ws, const int64_t* n, int32_t count, BatchProblem** table, float** F,
                          int32_t** nbr, float4** sums, float** Y) {
    int64_t rows = 0;
    for (int32_t b = 0; b < count; ++b) rows += n[b];
    Carver c(ws);
    BatchProblem* t = c.take<BatchProblem>((size_t)count);
    float* f = c.take<float>((size_t)rows * IN);
    int32_t* nb = c.take<int32_t>((size_t)rows * TOPK);
    float4* sm = c.take<float4>((size_t)rows);
    float* y = c.take<float>((size_t)rows * OUT);
    if (sums) *sums = sm;
    if (table) *table = t;
    if (F) *F = f;
    if (nbr) *nbr = nb;
    if (Y) *Y = y;
    return c.used;
}

}  // namespace mlp
}  // namespace apgb

APGB_API size_t apl_warm_start_batched_workspace_size(const int64_t* n, int32_t count) {
    if (!n || count < 1) return 0;
    for (int32_t b = 0; b < count; ++b)
        if (n[b] < 2 || n[b] > INT_MAX) return 0;
    return carve_batch(nullptr, n, count, nullptr, nullptr, nullptr, nullptr, nullptr);
}

APGB_API int32_t apl_warm_start_batched(const float* S, float* R, float* A, const int64_t* offsets,
                                        const int64_t* n, const int64_t* ld, int32_t count,
                                        const float* scale, const float* P, const void* P16, float* Y,
                                        void* ws, size_t ws_bytes, void* stream) {
    if (!S || !R || !A || !offsets || !n || !ld || !scale || !P || !P16 || count < 1)
        return AP_ERR_INVALID_ARG;
    const size_t need = apl_warm_start_batched_workspace_size(n, count);
    if (!need) return AP_ERR_INVALID_ARG;
    int64_t rows = 0, blocks = 0;
    std::vector<BatchProblem> host(count);
    for (int32_t b = 0; b < count; ++b) {
        if (ld[b] < n[b] || offsets[b] < 0 || !(scale[b] > 0.f)) return AP_ERR_INVALID_ARG;
        BatchProblem& q = host[b];
        q.S = S + offsets[b];
        q.R = R + offsets[b];
        q.A = A + offsets[b];
        q.ld = ld[b];
        q.frow = rows;
        q.n = (int)n[b];
        q.scale = scale[b];
        q.nb = (int)((n[b] + kFeatWarps - 1) / kFeatWarps);
        q.b0 = (int)blocks;
        blocks += q.nb;
        rows += n[b];
    }
    if (blocks > INT_MAX || rows > INT_MAX) return AP_ERR_INVALID_ARG;
    int w0 = 0;
    for (int32_t b = 0; b < count; ++b) {
        host[b].w0 = w0;
        w0 += (host[b].n + kWarmRows - 1) / kWarmRows;
    }
    AP_TRY(require_sm103());
    AP_TRY(check_ws(ws, ws_bytes, need));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    BatchProblem* table = nullptr;
    float *F = nullptr, *Yw = nullptr;
    int32_t* nbr = nullptr;
    float4* sums = nullptr;
    carve_batch(ws, n, count, &table, &F, &nbr, &sums, &Yw);
    if (!Y) Y = Yw;
    AP_CUDA_TRY(cudaMemcpyAsync(table, host.data(), sizeof(BatchProblem) * count, cudaMemcpyHostToDevice, s));
    features_batched_kernel<<<(int)blocks, 32 * kFeatWarps, 0, s>>>(table, count, F, nbr, sums);
    features_finish_batched_kernel<<<(int)((rows + 255) / 256), 256, 0, s>>>(table, count, rows, sums, nbr, F);
    note_launches(2);
    AP_TRY(last_error());
    AP_TRY(forward(P, static_cast<const __nv_bfloat16*>(P16), F, (int)rows, Y, s));
    warm_batched_kernel<<<w0, 256, 0, s>>>(table, count, Y);
    note_launches(1);
    return last_error();
}

APGB_API int32_t apl_set_standardisation(float* P, const float* F, int64_t rows, void* stream) {
    if (!P || !F || rows < 1) return AP_ERR_INVALID_ARG;
    AP_TRY(require_sm103());
    standardisation_kernel<<<IN, 256, 0, static_cast<cudaStream_t>(stream)>>>(F, rows, P);
    note_launches(1);
    return last_error();
}

APGB_API int32_t apl_judge(const double* cold_netsim, const double* warm_netsim, int32_t count,
                           double tol, int32_t* use_warm) {
    if (!cold_netsim || !warm_netsim || !use_warm || count < 0 || !(tol >= 0.0)) return AP_ERR_INVALID_ARG;
    int32_t kept = 0;
    for (int32_t b = 0; b < count; ++b) {
        const double c = cold_netsim[b], w = warm_netsim[b];
        use_warm[b] = (std::isfinite(c) && std::isfinite(w) && std::fabs(w - c) <= tol * std::fabs(c)) ? 1 : 0;
        kept += use_warm[b];
    }
    return kept;
}
