// pair_tc.cu — SIS scores of the top level's binary candidates (§2.2 Eqs. 5-6) from fused
// tcgen05 products: the pair kernel of the FP32 and the mixed forms.
//
// With every operand x and its reciprocal z = 1/x centred (x' = x - A, A the FP64 mean), a
// candidate v = x_i g_j (g = x_j, z_j; and z_i x_j) has, over the samples,
//   var(v)   = A^2 Vg + B^2 Vx + (P2 - P1^2) + 2 A B P1 + 2 A P3 + 2 B P4
//   cov(v,r) = A Rg + B Rx + T
// with P1 = E x'g', P2 = E x'^2 g'^2, P3 = E x'g'^2, P4 = E x'^2 g', T = E (x'r) g' and the
// per-operand V = E x'^2, R = E x'r; and v = x_i +/- x_j has var = Vi + Vj +/- 2 P1 and
// cov = Ri +/- Rj.  So each pair needs five bilinear sums per product form, which is a
// contraction over the samples with the operand rows [x', x'^2] on one side and
// [x', x'^2, x'r] on the other: the tensor cores' job (15 sums per pair against 13 FP32
// instructions per pair and sample on the CUDA cores, whose FP32 pipe bounded that form).
// The variance does not depend on the target, so the first step of a fit stores 1/sd of
// every candidate and the later steps run the T sum alone.
//
// Precision: every row is scaled by a power of two and split into two FP16 parts hi + lo
// (|x - hi - lo| <= 2^-23 |x| beside the 2^-24 of its FP32 copy, down to 2^-39 of the row's
// largest value), and the products hi lo, lo hi, hi hi are accumulated in FP32.  The tensor
// cores drop up to about one unit in the last place of the accumulator per MMA, so a run is
// only 64 samples (the four hi hi MMAs of a run come last, on an accumulator that until then
// is 2^-11 of its final size) and the runs are added on the CUDA cores.  Sums over at most
// kMaxRuns runs are added in FP32, longer ones in chunks whose totals are added with compensation.
// Each key carries a bound of its error (pt_key); a key whose bound could matter next to the
// screening margin, where the candidate's terms nearly cancel, is left open and scored by
// k_pt_direct from the sums the definition writes, sample by sample, in FP32, or, where those are not
// sure either, by k_pt_exact in FP64.
//
// Measured against the CUDA-core kernel it replaced: 2.9e8 rung-3 candidates (1000 samples, 10 primaries), 40.6 ms
// a step -> 5.7 ms (first step), 2.4 ms (later ones), and 2.6 ms of open keys in the first step with 0.6 of
// those left to FP64; 402 operands over 65 536 samples, 7.9 ms a step -> 0.80 and 0.18 ms.  The mixed forms had their own split
// products (FP64 rows, chunk sums and scores): 4.9 ms a step there, and keys raised to their
// bound where they nearly cancel.  The rows, target rows and partials bound the long samples
// (HBM), the epilogue's FP32 adds the short ones.
#include "sis_device.cuh"
#include "tc_device.cuh"

#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace sg {

struct PairTc {
    int64_t P = 0, Q = 0;          // operands; pairs are (i, j), i < j, j >= Q (NEW_X_PREV: i < Q)
    int64_t Pi = 0;                // operands on the i side: [0, Pi)
    int Kpad = 0, runs = 0;        // samples padded to whole runs of 64
    __half* rows = nullptr;        // [set x, z][x', x'^2][hi, lo][P][Kpad]
    __half* rrows = nullptr;       // [set x, z][hi, lo][Pi][Kpad]: x'r, z'r of the step's target
    float* val32 = nullptr;        // [P][Kpad]: the operand values rounded to FP32 (open keys)
    float4* par = nullptr;         // [set][P]: mean, V, sample-0 value (scaled), log2 |sample 0|
    int* ex = nullptr;             // [set][P]: scale exponents (scaled = value 2^-ex)
    float* R = nullptr;            // [set][P]: E x'r, scaled
    float* w = nullptr;            // [+, -, i j, i / j, j / i][Pi][P - Q]: 1 / sd (scaled), negative where invalid
    unsigned long long* list = nullptr;   // open keys of the first step, those of every step, those left to FP64
    unsigned* count = nullptr;     // [0] open keys, [1] keys open at every step, [2] error flag, [3] left to FP64
    int64_t cap = 0;
    size_t n_w = 0;
    float* part = nullptr;         // chunk partials (long samples) of `batch` tiles
    int2* tiles[2] = {nullptr, nullptr};   // (i0, j0) per tile: five-sum and one-sum shapes
    int64_t n_tiles[2] = {0, 0}, batch[2] = {0, 0};
    int ni[2] = {0, 0}, chunks[2] = {1, 1}, run_len[2] = {0, 0};
    size_t part_bytes = 0;
    CUtensorMap mapM, mapN[2], mapR[2];
    std::vector<int2> tile_list[2];   // host copies of the tiles (the source of an asynchronous copy)
    bool ready = false;            // w and the lists hold this fit's operands
};

namespace {

constexpr int kPtM = 128;                  // j operands per tile: TMEM lanes
constexpr uint32_t kPtD2 = 160;            // column of the second accumulator block (five sums)
constexpr int kPtK = 64;                   // samples per run and stage
constexpr int kPtStages = 2;
constexpr int kPtEpiWarps = 12;            // epilogue warps: four lane quarters x thirds of the i operands
constexpr int kPtThreads = kPtEpiWarps * 32 + 64;   // then a TMA and an MMA warp
constexpr int kPtI5 = 48, kPtI1 = 240;     // largest i tile of the two shapes (240 accumulator columns)
constexpr int kMaxRuns = 32;               // runs added in FP32 (2048 samples)
constexpr float kU = 5.9604645e-8f;        // 2^-24
// largest errors, in units of 2^-24 and relative to the value: a row's x' as hi + lo (its FP32 copy
// and the parts), x'^2 (two copies, the square, the parts), x'r (hi + lo, the target's copy, the
// product, the parts), the part product lo lo that is left out, and a row's mean square V (the
// squares, four accumulators of up to four pairs, their sum, the warp's)
constexpr int kErrRow = 3, kErrSquare = 5, kErrTarget = 7, kErrLoLo = 4, kErrV = 17;
// ... of a sum of products over runs of 64: its two rows and lo lo at most (x'^2 g'^2 and x'r g'), one
// last-place unit of the accumulator at each of a run's four hi hi MMAs, the chunks and the scale;
// the additions of the runs come on top
constexpr int kErrSum = 2 * kErrSquare + kErrLoLo + 8 + 3;
static_assert(kErrTarget + kErrRow <= 2 * kErrSquare, "the largest pair of rows");
constexpr float kTolMany = 1.5e-4f;        // largest relative variance bound of a final key (score: half)
constexpr float kTolFew = 4e-5f;           // ... up to kFewRuns runs: FP32 sums that short are better than that
constexpr float kTolDirect = 1e-4f;        // ... of a key from the direct FP32 sums (k_pt_direct)
constexpr int kFewRuns = 4;
constexpr float kFloor = 1.82e-12f;        // 2^-39: parts below FP16's range, relative to a row's largest value

constexpr float kLogCap = 39.86324f;       // log2 of the value cap 1e12, and of its square with 1% to spare
constexpr float kLogRms = 79.74f;

__host__ __device__ constexpr int pt_m_kinds(int F) { return F == 5 ? 2 : 1; }   // row kinds staged per side
__host__ __device__ constexpr int pt_n_kinds(int F) { return F == 5 ? 3 : 1; }
constexpr uint32_t kRowBytes = kPtK * 2;

__host__ __device__ constexpr uint32_t pt_stage_bytes(int F, int ni) {
    return 2u * kRowBytes * (uint32_t)(pt_m_kinds(F) * kPtM + pt_n_kinds(F) * ni);
}

struct PtArgs {
    const Space* sp;
    int sec[4];
    int64_t P, Q, Pi;
    int N, Kpad, nxp, ntypes;
    const __half* rows;
    const float* val32;
    const double* val64;       // operand values and reciprocals (or null), feature-major, N samples
    const double* inv64;
    const double* tc64;
    double inv_n;
    int type[3];               // 0: x_i x_j and x_i +/- x_j, 1: x_i / x_j, 2: x_j / x_i
    const int2* tiles;
    int n_tiles, ni, chunks, run_len, runs;
    float scale;               // 2^-30 / N
    float tol;                 // relative variance bound of a final key; its covariance bound is half of it
    float eps;                 // bound on a sum's accumulation error, relative to E |product|
    const float4* par;
    const int* ex;
    const float* R;
    float* w;
    float* scores;
    const TargetStats* st;
    unsigned long long* list;
    unsigned* count;
    int64_t cap;
    float* part;
};

__device__ __forceinline__ float pow2f(int e) {      // 2^e, 0 below and infinity above FP32's range
    return e > 127 ? INFINITY : e < -126 ? 0.f : __int_as_float((e + 127) << 23);
}

// ---------------------------------------------------------------------------------
// operand rows
// ---------------------------------------------------------------------------------
// sum and maximum over the threads that share an operand: a warp (IT > 0) or a CTA (IT = 0)
template <bool CTA, typename T> __device__ __forceinline__ T group_sum(T v, T* sh) {
    v = warp_sum(v);
    if constexpr (CTA) {
        __syncthreads();
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
        __syncthreads();
        v = sh[0];
        for (int q = 1; q < (int)(blockDim.x >> 5); ++q) v += sh[q];
    }
    return v;
}
template <bool CTA> __device__ __forceinline__ int group_max(int v, int* sh) {
    v = __reduce_max_sync(0xffffffffu, v);
    if constexpr (CTA) {
        __syncthreads();
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
        __syncthreads();
        v = sh[0];
        for (int q = 1; q < (int)(blockDim.x >> 5); ++q) v = max(v, sh[q]);
    }
    return v;
}

// x and y in [-2^15, 2^15] as hi + lo
__device__ __forceinline__ void put_parts2(float x, float y, __half* hi, __half* lo) {
    const __half2 h = __floats2half2_rn(x, y);
    const float2 b = __half22float2(h);
    *reinterpret_cast<__half2*>(hi) = h;
    *reinterpret_cast<__half2*>(lo) = __floats2half2_rn(x - b.x, y - b.y);
}

// log2 |x| to about 2e-6, -inf for zero and subnormal values (x finite)
__device__ __forceinline__ float log2_abs(double x) {
    const int hi = __double2hiint(x) & 0x7fffffff;
    if ((hi >> 20) == 0) return -INFINITY;
    return (float)((hi >> 20) - 1023) + log2f(__int_as_float(0x3f800000 | ((hi & 0xfffff) << 3)));
}

// Rows of both sets of one operand: the mean (FP64), the exponent of the largest centred value
// (from the exponent bits: no FP64 comparison), the scaled rows and their squares.  The FP64
// pipe is the narrow one on this part (an FP64 warp instruction takes about 18 cycles of an
// SM), so FP64 work is kept to the sum and the centring of a value; it is rounded once to FP32
// and squared there.  IT > 0: one warp per operand with
// 2 IT values per lane in registers (a CTA's FP64 reductions would cost as much as its
// values); IT = 0: one CTA per operand, values read again.
template <int IT>
__global__ void __launch_bounds__(IT > 0 ? 128 : 512)
k_pt_rows(const double* __restrict__ val, const double* __restrict__ inv, const unsigned char* __restrict__ valid,
          int64_t P, int N, int Kpad, __half* __restrict__ rows, float* __restrict__ val32, float4* __restrict__ par,
          int* __restrict__ ex) {
    constexpr bool CTA = IT == 0;
    __shared__ double shd[16];
    __shared__ int shi[16];
    const int64_t f = CTA ? (int64_t)blockIdx.x : ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (f >= P) return;
    const int t = CTA ? (int)threadIdx.x : (int)(threadIdx.x & 31), nt = CTA ? (int)blockDim.x : 32;
    const bool ok = valid[f] != 0;
    const double inv_n = 1.0 / N;
    const double* v = val + (size_t)f * N;
#pragma unroll 1
    for (int set = 0; set < 2; ++set) {
        const double* u = set == 0 ? v : inv ? inv + (size_t)f * N : nullptr;
        auto load = [&](int i) { return !ok || i >= N ? 0.0 : u ? u[i] : 1.0 / v[i]; };
        double c[IT > 0 ? 2 * IT : 1];
        double s = 0.0;
        if constexpr (IT > 0) {
#pragma unroll
            for (int q = 0; q < IT; ++q) {
                const int i = 2 * (t + q * nt);
                c[2 * q] = load(i);
                c[2 * q + 1] = load(i + 1);
                s += c[2 * q] + c[2 * q + 1];
                if (set == 0 && i < Kpad)
                    *reinterpret_cast<float2*>(val32 + (size_t)f * Kpad + i) = make_float2(scaled_f32(c[2 * q], 0), scaled_f32(c[2 * q + 1], 0));
            }
        } else {
            for (int i = t; i < Kpad; i += nt) {
                const double x = load(i);
                s += x;
                if (set == 0) val32[(size_t)f * Kpad + i] = scaled_f32(x, 0);
            }
        }
        const double mean = group_sum<CTA>(s, shd) * inv_n;
        int hx = 0;                      // largest high word of |centred value|
        if constexpr (IT > 0) {
#pragma unroll
            for (int q = 0; q < 2 * IT; ++q) {
                const int i = 2 * (t + (q >> 1) * nt) + (q & 1);
                c[q] = i < N ? c[q] - mean : 0.0;
                hx = max(hx, __double2hiint(c[q]) & 0x7fffffff);
            }
        } else {
            for (int i = t; i < N; i += nt) hx = max(hx, __double2hiint(load(i) - mean) & 0x7fffffff);
        }
        hx = group_max<CTA>(hx, shi);
        const int be = hx >> 20;         // biased exponent of the largest value
        // unusable: a non-finite value (a zero's reciprocal), or no variation in FP32's range
        const bool bad = !ok || be == 0x7ff || be < 40;
        const int e = be - 1022;         // |centred| < 2^e
        __half* r0 = rows + (size_t)(set * 4) * P * Kpad + (size_t)f * Kpad;
        const size_t lo = (size_t)P * Kpad;
        __half* r1 = r0 + 2 * lo;
        float run[4] = {0.f, 0.f, 0.f, 0.f};
        double V = 0.0;
        auto put = [&](int i, double x, double y, float& sum) {
            const float a = bad ? 0.f : scaled_f32(x, 15 - e), b = bad ? 0.f : scaled_f32(y, 15 - e);
            const float a2 = a * a * 3.0517578125e-5f, b2 = b * b * 3.0517578125e-5f;      // times 2^15
            put_parts2(a, b, r0 + i, r0 + lo + i);
            put_parts2(a2, b2, r1 + i, r1 + lo + i);
            sum += a2 + b2;
        };
        if constexpr (IT > 0) {
#pragma unroll
            for (int q = 0; q < IT; ++q) {
                const int i = 2 * (t + q * nt);
                if (i < Kpad) put(i, c[2 * q], c[2 * q + 1], run[q & 3]);
            }
        } else {
            int q = 0;
            for (int i = 2 * t; i < Kpad; i += 2 * nt) {
                put(i, i < N ? load(i) - mean : 0.0, i + 1 < N ? load(i + 1) - mean : 0.0, run[0]);
                if ((++q & 7) == 0) { V += (double)run[0]; run[0] = 0.f; }
            }
        }
        float Vs;
        if constexpr (IT > 0) Vs = warp_sum((run[0] + run[1]) + (run[2] + run[3]));
        else Vs = (float)group_sum<CTA>(V + (double)run[0], shd);
        if (t == 0) {
            const double x0 = load(0);
            const float g = 3.0517578125e-5f;
            par[(size_t)set * P + f] = bad ? make_float4(0.f, 0.f, 0.f, INFINITY)
                                           : make_float4(scaled_f32(mean, -e), Vs * g * (float)inv_n, scaled_f32(x0, -e),
                                                         log2_abs(x0));
            ex[(size_t)set * P + f] = bad ? 0 : e;
        }
    }
}

// per step: R = E x'r of every operand and set, and the rows x'r of the i-side operands; a
// warp (or CTA, many samples) per operand, two samples per thread and round, products in FP32,
// runs of 16 added in FP64.  r is scaled by 2^-er, er the exponent of sd sqrt(N) >= max |r|.
template <bool CTA>
__global__ void __launch_bounds__(512) k_pt_target(const __half* __restrict__ rows, const float* __restrict__ r,
                                                   const TargetStats* __restrict__ st, int64_t P, int64_t Pi, int N,
                                                   int Kpad, __half* __restrict__ rrows, float* __restrict__ R) {
    __shared__ double shd[16];
    const int64_t f = CTA ? (int64_t)blockIdx.x : ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (f >= P) return;
    const int t = CTA ? (int)threadIdx.x : (int)(threadIdx.x & 31), nt = CTA ? (int)blockDim.x : 32;
    const size_t lo = (size_t)P * Kpad, rlo = (size_t)Pi * Kpad;
    const float rs = st->rscale;
    const bool write = f < Pi;
    const __half* x0 = rows + (size_t)f * Kpad;
    __half* o0 = rrows + (size_t)f * Kpad;
    float run[2] = {0.f, 0.f};
    double s[2] = {0.0, 0.0};
    int q = 0;
    for (int i = 2 * t; i < Kpad; i += 2 * nt) {
        const float ra = i < N ? r[i] * rs : 0.f, rb = i + 1 < N ? r[i + 1] * rs : 0.f;
#pragma unroll
        for (int set = 0; set < 2; ++set) {
            const __half* x = x0 + (size_t)(set * 4) * lo;
            const float2 h = __half22float2(*reinterpret_cast<const __half2*>(x + i));
            const float2 l = __half22float2(*reinterpret_cast<const __half2*>(x + lo + i));
            const float pa = (h.x + l.x) * ra, pb = (h.y + l.y) * rb;       // times 2^15
            run[set] += pa + pb;
            if (write) put_parts2(pa, pb, o0 + (size_t)(set * 2) * rlo + i, o0 + (size_t)(set * 2 + 1) * rlo + i);
        }
        if ((++q & 7) == 0) {
            s[0] += (double)run[0]; s[1] += (double)run[1];
            run[0] = run[1] = 0.f;
        }
    }
#pragma unroll
    for (int set = 0; set < 2; ++set) {
        const double v = group_sum<CTA>(s[set] + (double)run[set], shd);
        if (t == 0) R[(size_t)set * P + f] = (float)v * (3.0517578125e-5f / (float)N);
    }
}

// ---------------------------------------------------------------------------------
// keys
// ---------------------------------------------------------------------------------
struct PtSide { float m, V, s, x0, lg, R; int ex; };     // mean, E x'^2, its root, sample 0, log2, E x'r, exponent

__device__ __forceinline__ PtSide pt_side(const PtArgs& A, int set, int64_t f) {
    const float4 p = __ldg(A.par + (size_t)set * A.P + f);
    return PtSide{p.x, p.y, sqrtf(p.y), p.z, p.w, __ldg(A.R + (size_t)set * A.P + f), __ldg(A.ex + (size_t)set * A.P + f)};
}

struct PtKey { float key, w; };
__device__ __forceinline__ size_t w_index(const PtArgs& A, int op, int64_t i, int64_t j) {
    return ((size_t)op * (size_t)A.Pi + (size_t)i) * (size_t)(A.P - A.Q) + (size_t)(j - A.Q);
}

// key and 1/sd from the variance, its error bound dv, the covariance and its bound dc (both
// relative to the target's deviation) and the mean and its bound dm.  Rejected (w = -inf) only where
// the FP64 rules must reject: |v(sample 0)| > 1e12, a root mean square that even at the lower end of
// its bounds is above 1e12, or a deviation that even at the upper end of its bound is <= 1e-6
// max(|v0|, |mean|) with the mean at its lower end.  (Operands that span many decades and cancel,
// as a quotient of two of them does, leave a variance and a mean that are mostly rounding.)  Open
// (w = -dc) where the bounds could move the key by more than 7.5e-5 each (the selection's margin is
// 2e-4).  A key that only its bounds could reject is final: the FP64 re-score applies the rules.
__device__ __forceinline__ PtKey pt_key(float var, float dv, float cov, float dc, float v0, float mean, float dm, bool v0_ok,
                                        float rms2_max, float tol, float inv_sdr) {
    const float lo = fmaxf(fabsf(mean) - dm, 0.f), lim = (float)kConstRel * fmaxf(fabsf(v0), lo);
    if (!v0_ok || !(fmaf(lo, lo, var - dv) <= rms2_max) || !(var + dv > lim * lim)) return PtKey{-1.f, -INFINITY};
    const float w = __frsqrt_rn(var);
    if (!(dv <= tol * var) || !(dc * w <= 0.5f * tol)) return PtKey{-1.f, -fmaxf(dc, 1e-30f)};
    return PtKey{fabsf(cov) * w * inv_sdr, w};
}

// v = x g: x the i side (A), g the j side (B)
__device__ __forceinline__ PtKey pt_product(const PtArgs& A, const PtSide& a, const PtSide& b, float P1, float P4,
                                            float T, float P3, float P2, float inv_sdr) {
    const float AB = a.m * b.m;
    const float t1 = a.m * a.m * b.V, t2 = b.m * b.m * a.V, t3 = 2.f * AB * P1, t4 = 2.f * a.m * P3, t5 = 2.f * b.m * P4;
    const float p11 = P1 * P1;
    const float var = ((t1 + t2) + (P2 - p11)) + (t3 + (t4 + t5));
    const float fa = fabsf(a.m), fb = fabsf(b.m);
    const float S = t1 + t2 + P2 + p11 + fabsf(t3) + fabsf(t4) + fabsf(t5);
    const float fl = 2.f * kFloor * (a.s + b.s);
    const float q = sqrtf(fmaxf(P2, 0.f) + fl);              // >= root of E x'^2 g'^2 >= E |x'g'|
    // the sums' errors (E |x'g'^2| <= q s_g), V's and this expression's, the parts' floor
    const float dv = A.eps * (2.f * q * (fabsf(AB) + fabsf(P1) + fa * b.s + fb * a.s) + P2) + (kErrV + 8.f) * kU * S +
                     fl * (2.f + (1.f + 2.f * fa) * (1.f + 2.f * fb));
    const float cov = a.m * b.R + b.m * a.R + T;
    // T's error, R's (19 2^-24 E |x'r|) and the additions', the floors of x', g' and x'r: the last
    // is one of the target scaled into [-1, 1], whose deviation there is 1 / inv_sdr
    const float dc = A.eps * q + 20.f * kU * (fa * b.s + fb * a.s + q) +
                     2.f * kFloor * (a.s + b.s * (1.f + inv_sdr) + fa + fb);
    const float lg = a.lg + b.lg;
    const float dm = A.eps * q + 4.f * kU * (fabsf(AB) + fabsf(P1)) + 0.5f * fl;
    return pt_key(var, dv, cov, dc, a.x0 * b.x0, AB + P1, dm, lg <= kLogCap, exp2f(kLogRms - 2.f * (float)(a.ex + b.ex)),
                  A.tol, inv_sdr);
}

// v = x_i + sg x_j, in units of 2^max(exponents)
__device__ __forceinline__ PtKey pt_sum(const PtArgs& A, const PtSide& a, const PtSide& b, float sg, float P1,
                                        float inv_sdr) {
    const int em = max(a.ex, b.ex);
    const float fa = pow2f(a.ex - em), fb = sg * pow2f(b.ex - em);
    const float va = fa * fa * a.V, vb = fb * fb * b.V, c2 = 2.f * fa * fb * P1;
    const float var = va + vb + c2;
    const float sa = fa * a.s, sb = fabsf(fb) * b.s;
    // E |x_i' x_j'| <= s_i s_j
    const float dv = 2.f * A.eps * sa * sb + (kErrV + 4.f) * kU * (va + vb + fabsf(c2)) + 2.f * kFloor * fa * fabsf(fb) * (a.s + b.s);
    const float v0 = fa * a.x0 + fb * b.x0, mean = fa * a.m + fb * b.m;
    const bool ok = a.lg < INFINITY && b.lg < INFINITY && fabsf(v0) * pow2f(em) <= (float)kValueCap;
    return pt_key(var, dv, fa * a.R + fb * b.R, 20.f * kU * (sa + sb) + 2.f * kFloor * (fa + fabsf(fb)), v0, mean,
                  3.f * kU * (fa * fabsf(a.m) + fabsf(fb * b.m)), ok, exp2f(kLogRms - 2.f * (float)em),
                  A.tol, inv_sdr);
}

// first id of row i minus the column's offset: rank = base_i + j for candidates (i, j), j > i
__device__ __forceinline__ int64_t sym_base(int nxp, int64_t P, int64_t Q, int64_t i) {
    if (nxp) return i * (P - Q) - Q;
    const int64_t Ah = Q > 0 ? Q - 1 : 0;
    if (i < Ah) return i * (P - Q) - Q;
    return Ah * (P - Q) + tri_start(i - Ah, P - 1 - Ah) - i - 1;
}
__device__ __forceinline__ int64_t div_base(int nxp, int64_t P, int64_t Q, int64_t i) {
    if (nxp || i < Q) return i * (P - Q) - Q;
    return Q * (P - Q) + (i - Q) * (P - 1) - 1;
}
// ... and rank = base_j + i for the quotients x_j / x_i, i < j
__device__ __forceinline__ int64_t rdiv_base(int nxp, int64_t P, int64_t Q, int64_t j) {
    return Q * (P - Q) + (j - Q) * (nxp ? Q : P - 1);
}

// first ids of the sections + - * / of the top level (-1: operator not enabled)
struct PtBase { int64_t o[4]; };
__device__ __forceinline__ PtBase pt_bases(const PtArgs& A) {
    PtBase b;
#pragma unroll
    for (int o = 0; o < 4; ++o) b.o[o] = A.sec[o] >= 0 ? A.sp->sec[A.sec[o]].base : -1;
    return b;
}

// first id of row i of a product form, less the column's offset (types 0 and 1: id = base + j)
__device__ __forceinline__ int64_t row_base(const PtArgs& A, int type, int64_t i) {
    return type == 0 ? sym_base(A.nxp, A.P, A.Q, i) : type == 1 ? div_base(A.nxp, A.P, A.Q, i) : i;
}

// first step: keys and 1/sd of one pair from its five sums.  at: rank of (i, j) in its sections
__device__ __forceinline__ void pt_emit5(const PtArgs& A, const PtBase& B, int type, int64_t at, size_t wi, size_t wop,
                                         const PtSide& a, const PtSide& b, float P1, float P4, float T, float P3,
                                         float P2, bool in, float inv_sdr) {
    const PtKey k = pt_product(A, a, b, P1, P4, T, P3, P2, inv_sdr);
    if (type == 0) {
        const PtKey p = pt_sum(A, a, b, 1.f, P1, inv_sdr), m = pt_sum(A, a, b, -1.f, P1, inv_sdr);
        if (in && B.o[0] >= 0) { A.scores[B.o[0] + at] = p.key; A.w[wi] = p.w; }
        if (in && B.o[1] >= 0) { A.scores[B.o[1] + at] = m.key; A.w[wi + wop] = m.w; }
        if (in && B.o[2] >= 0) { A.scores[B.o[2] + at] = k.key; A.w[wi + 2 * wop] = k.w; }
    } else if (in) {
        A.scores[B.o[3] + at] = k.key;
        A.w[wi + (size_t)(type + 2) * wop] = k.w;
    }
}

__device__ __forceinline__ float later_key(float w, float cov, float inv_sdr) {
    return w < 0.f ? -1.f : fabsf(cov) * w * inv_sdr;
}

// bounded wait that also ends when another warp of the CTA has given up
__device__ __forceinline__ bool pt_wait(uint64_t* bar, uint32_t parity, const volatile int* failed) {
    for (long long it = 0; it < kWaitLimit; ++it) {
        uint32_t ok;
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 63) == 63 && *failed) return false;
    }
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(taddr));
}
// the loads above complete at tcgen05.wait::ld: values pass through here after it, so that no
// use of them can be scheduled before it
__device__ __forceinline__ void tmem_loaded8(float (&r)[8]) {
    asm volatile("" : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]));
}

struct PtSmem {
    uint64_t full[kPtStages], empty[kPtStages], tfull[2], tempty[2], done;
    uint32_t tmem;
    int failed;
};

// the i side of a tile as its warp's scoring reads it (shared memory, one broadcast per i)
template <int F> struct PtRow;
template <> struct PtRow<5> { PtSide s; int pad; int64_t base; };
template <> struct PtRow<1> { float m, R; int ex, pad; int64_t base; };
template <int F> __host__ __device__ constexpr uint32_t pt_row_bytes(int ni) {
    return (uint32_t)sizeof(PtRow<F>) * kPtEpiWarps * (uint32_t)(ni / 3);
}

// dynamic shared memory of k_pair_tc<F> with i tiles of ni
template <int F> constexpr size_t pt_smem_bytes(int ni) {
    return (size_t)kPtStages * pt_stage_bytes(F, ni) + 1024 + pt_row_bytes<F>(ni);
}

// Persistent: one CTA per SM walks the work units (tile of 128 j x ni i operands, product form,
// sample chunk).  A TMA warp stages a run's rows (two stages), an MMA warp issues its products
// into one of two TMEM buffers of 240 columns, twelve warps add the run's sums to their
// registers (80 per thread: lane = j, a third of the i columns) and score the tile at its end.
// F = 5: D1 = x_j' against [x_i' | x_i'^2 | x_i'r] and D2 = x_j'^2 against [x_i' | x_i'^2]
// (ni = 48: 144 + 96 columns); F = 1: x_j' against x_i'r (ni <= 240).  The second buffer lets
// the next run's MMAs overlap the additions; 240 columns are what the registers of a CTA's
// epilogue threads can accumulate.
template <int F>
__global__ void __launch_bounds__(kPtThreads, 1)
k_pair_tc(const __grid_constant__ CUtensorMap mapM, const __grid_constant__ CUtensorMap mapN,
          const __grid_constant__ CUtensorMap mapR, PtArgs A) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* stage0 = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ PtSmem S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t stage_bytes = pt_stage_bytes(F, A.ni);
    const uint32_t m_bytes = kPtM * kRowBytes, n_bytes = (uint32_t)A.ni * kRowBytes;   // one block of rows
    constexpr int MK = pt_m_kinds(F), NK = pt_n_kinds(F);
    const int per = A.n_tiles * A.ntypes, units = per * A.chunks;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPtStages; ++s) { mbar_init(&S.full[s], 1); mbar_init(&S.empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&S.tfull[b], 1); mbar_init(&S.tempty[b], kPtEpiWarps); }
        mbar_init(&S.done, 1);
        S.failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kPtEpiWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = S.tmem;
    volatile int* failed = &S.failed;

    if (warp == kPtEpiWarps) {
        if (lane == 0) {
            int g = 0;
            for (int u = blockIdx.x; u < units && !*failed; u += gridDim.x) {
                const int chunk = u / per, rem = u % per, type = A.type[rem % A.ntypes];
                const int2 t = A.tiles[rem / A.ntypes];
                const int sm = type == 1, sn = type == 2;                 // 1: reciprocals
                const int r0 = chunk * A.run_len, r1 = min(A.runs, r0 + A.run_len);
                for (int r = r0; r < r1; ++r, ++g) {
                    const int s = g % kPtStages;
                    if (g >= kPtStages && !pt_wait(&S.empty[s], ((uint32_t)(g / kPtStages) & 1u) ^ 1u, failed)) { *failed = 1; break; }
                    mbar_expect_tx(&S.full[s], stage_bytes);
                    unsigned char* d = stage0 + (size_t)s * stage_bytes;
                    for (int p = 0; p < 2; ++p)
                        for (int k = 0; k < MK; ++k, d += m_bytes)
                            tma_load_2d(d, &mapM, r * kPtK, (int)(((sm * 2 + k) * 2 + p) * A.P + t.y), &S.full[s]);
                    for (int p = 0; p < 2; ++p)
                        for (int k = 0; k < NK; ++k, d += n_bytes) {
                            if (k == NK - 1) tma_load_2d(d, &mapR, r * kPtK, (int)((sn * 2 + p) * A.Pi + t.x), &S.full[s]);
                            else tma_load_2d(d, &mapN, r * kPtK, (int)(((sn * 2 + k) * 2 + p) * A.P + t.x), &S.full[s]);
                        }
                }
            }
            // no copy may be in flight when the CTA ends
            for (int q = max(0, g - kPtStages); q < g; ++q) mbar_wait(&S.full[q % kPtStages], (uint32_t)(q / kPtStages) & 1u);
        }
    } else if (warp == kPtEpiWarps + 1) {
        if (lane == 0) {
            const uint32_t id1 = idesc_f16(0u, kPtM, NK * A.ni), id2 = idesc_f16(0u, kPtM, 2 * A.ni);
            int g = 0;
            for (int u = blockIdx.x; u < units && !*failed; u += gridDim.x) {
                const int chunk = u / per;
                const int r0 = chunk * A.run_len, r1 = min(A.runs, r0 + A.run_len);
                for (int r = r0; r < r1; ++r, ++g) {
                    const int s = g % kPtStages, b = g & 1;
                    if (g >= 2 && !pt_wait(&S.tempty[b], ((uint32_t)(g >> 1) & 1u) ^ 1u, failed)) { *failed = 1; break; }
                    if (!pt_wait(&S.full[s], (uint32_t)(g / kPtStages) & 1u, failed)) { *failed = 1; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t m0 = smem_u32(stage0 + (size_t)s * stage_bytes);
                    const uint32_t n0 = m0 + 2u * MK * m_bytes;
                    const uint32_t d1 = tmem + (uint32_t)b * 256u, d2 = d1 + kPtD2;
#pragma unroll
                    for (int p = 0; p < 3; ++p) {                       // lo hi, hi lo, hi hi
                        const int pm = p == 0, pn = p == 1;
                        const uint64_t dm = desc_sw128(m0 + (uint32_t)(pm * MK) * m_bytes);
                        const uint64_t dn = desc_sw128(n0 + (uint32_t)(pn * NK) * n_bytes);
                        const uint64_t dm2 = desc_sw128(m0 + (uint32_t)(pm * MK + MK - 1) * m_bytes);
#pragma unroll
                        for (int k = 0; k < kPtK / 16; ++k) {
                            mma_f16(d1, dm + (uint64_t)(2 * k), dn + (uint64_t)(2 * k), id1, p > 0 || k > 0);
                            if (F == 5) mma_f16(d2, dm2 + (uint64_t)(2 * k), dn + (uint64_t)(2 * k), id2, p > 0 || k > 0);
                        }
                    }
                    mma_commit(&S.empty[s]);
                    mma_commit(&S.tfull[b]);
                }
            }
            mma_commit(&S.done);
            if (!mbar_wait(&S.done, 0)) *failed = 1;       // every MMA done before TMEM is given back
        }
    } else {
        const int quad = warp & 3, hw = A.ni / 3, c0 = (warp >> 2) * hw;   // lanes 32 quad.., i columns c0 .. c0 + hw
        const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
        const float inv_sdr = A.st->inv_sdr;
        const PtBase bases = pt_bases(A);
        const int64_t PQ = A.P - A.Q;
        const size_t wop = (size_t)A.Pi * (size_t)PQ;
        PtRow<F>* rows = reinterpret_cast<PtRow<F>*>(stage0 + (size_t)kPtStages * stage_bytes) + warp * hw;
        constexpr int G = F == 5 ? 2 : 10;               // groups of eight i operands per thread
        int g = 0;
        for (int u = blockIdx.x; u < units && !*failed; u += gridDim.x) {
            const int chunk = u / per, rem = u % per, type = A.type[rem % A.ntypes];
            const int2 t = A.tiles[rem / A.ntypes];
            const int r0 = chunk * A.run_len, r1 = min(A.runs, r0 + A.run_len);
            const int nv = (int)min((int64_t)hw, A.Pi - t.x - c0);        // i operands of this warp
            if (A.chunks == 1) {
                __syncwarp();
                for (int q = lane; q < nv; q += 32) {
                    const int64_t i = t.x + c0 + q;
                    const PtSide a = pt_side(A, type == 2, i);
                    PtRow<F>& o = rows[q];
                    if constexpr (F == 5) o.s = a;
                    else { o.m = a.m; o.R = a.R; o.ex = a.ex; }
                    o.base = row_base(A, type, i);
                }
                __syncwarp();
            }
            float acc[F][G * 8];
#pragma unroll
            for (int f = 0; f < F; ++f)
#pragma unroll
                for (int q = 0; q < G * 8; ++q) acc[f][q] = 0.f;
            bool ok = true;
            for (int r = r0; r < r1; ++r, ++g) {
                const int b = g & 1;
                ok = pt_wait(&S.tfull[b], (uint32_t)(g >> 1) & 1u, failed);
                if (!__all_sync(0xffffffffu, ok)) { ok = false; *failed = 1; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = trow + (uint32_t)b * 256u;
                if constexpr (F == 5) {
#pragma unroll
                    for (int e = 0; e < G; ++e) {
                        float v[5][8];
#pragma unroll
                        for (int f = 0; f < 5; ++f)
                            tmem_ld8(base + (uint32_t)((f < 3 ? f * kPtI5 : (int)kPtD2 + (f - 3) * kPtI5) + 8 * e), v[f]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int f = 0; f < 5; ++f) {
                            tmem_loaded8(v[f]);
#pragma unroll
                            for (int q = 0; q < 8; ++q) acc[f][8 * e + q] += v[f][q];
                        }
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < G; e += 2) {                      // hw is a multiple of 16
                        if (8 * e >= hw) break;
                        float v[2][8];
                        tmem_ld8(base + (uint32_t)(8 * e), v[0]);
                        tmem_ld8(base + (uint32_t)(8 * e + 8), v[1]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int f = 0; f < 2; ++f) {
                            tmem_loaded8(v[f]);
#pragma unroll
                            for (int q = 0; q < 8; ++q) acc[0][8 * (e + f) + q] += v[f][q];
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.tempty[b]);
            }
            if (!ok) break;
            const int jl = quad * 32 + lane;
            if (A.chunks > 1) {
                float* o = A.part + ((size_t)u * (F * A.ni) + c0) * kPtM + jl;
#pragma unroll
                for (int e = 0; e < G; ++e)
                    if (8 * e < hw) {
#pragma unroll
                        for (int q = 8 * e; q < 8 * e + 8; ++q)
#pragma unroll
                            for (int f = 0; f < F; ++f) o[(size_t)(f * A.ni + q) * kPtM] = acc[f][q];
                    }
                continue;
            }
            const int64_t j = t.y + jl;
            const bool inj = j < A.P;
            const PtSide bj = pt_side(A, type == 1, inj ? j : A.P - 1);
            const int64_t add = type == 2 ? rdiv_base(A.nxp, A.P, A.Q, j) : j;
            const int64_t i_first = t.x + c0;
            // eight i at a time, the sums of the next eight moved down: one copy of the code
#pragma unroll 1
            for (int e = 0; 8 * e < nv; ++e) {
                const size_t w0 = (size_t)(i_first + 8 * e) * (size_t)PQ + (size_t)(j - A.Q);
                if constexpr (F == 5) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int ql = min(8 * e + q, nv - 1);
                        const PtRow<F>& row = rows[ql];
                        pt_emit5(A, bases, type, row.base + add, w0 + (size_t)q * (size_t)PQ, wop, row.s, bj,
                                 acc[0][q] * A.scale, acc[1][q] * A.scale, acc[2][q] * A.scale, acc[3][q] * A.scale,
                                 acc[4][q] * A.scale, inj && 8 * e + q < nv && i_first + 8 * e + q < j, inv_sdr);
                    }
                } else {
                    const int o0 = type == 0 ? 0 : type + 2, o1 = type == 0 ? 3 : type + 3;
#pragma unroll 1
                    for (int o = o0; o < o1; ++o) {
                        const int64_t sec = bases.o[o < 3 ? o : 3];
                        if (sec < 0) continue;
                        bool in[8];
                        float w[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            in[q] = inj && 8 * e + q < nv && i_first + 8 * e + q < j;
                            w[q] = in[q] ? __ldg(A.w + (size_t)o * wop + w0 + (size_t)q * (size_t)PQ) : 0.f;
                        }
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const PtRow<F>& row = rows[min(8 * e + q, nv - 1)];
                            float cov;
                            if (o < 2) {
                                const int em = max(row.ex, bj.ex);
                                const float b = pow2f(bj.ex - em) * bj.R;
                                cov = pow2f(row.ex - em) * row.R + (o == 0 ? b : -b);
                            } else {
                                cov = row.m * bj.R + bj.m * row.R + acc[0][q] * A.scale;
                            }
                            if (in[q]) A.scores[sec + row.base + add] = later_key(w[q], cov, inv_sdr);
                        }
                    }
                }
#pragma unroll
                for (int f = 0; f < F; ++f)
#pragma unroll
                    for (int q = 0; q + 8 < G * 8; ++q) acc[f][q] = acc[f][q + 8];
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && S.failed) atomicExch(A.count + 2, 1u);
    if (warp == kPtEpiWarps + 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// long samples: the chunks' sums added with their rounding errors carried along (two FP32
// values: about seven FP32 instructions a term where one FP64 addition takes as long as 70),
// then the same keys; one CTA per (tile, form, i), thread = j
template <int F>
__global__ void __launch_bounds__(kPtM) k_pt_reduce(PtArgs A) {
    const int per = A.n_tiles * A.ntypes;
    const int rem = blockIdx.x / A.ni, il = blockIdx.x % A.ni;
    const int type = A.type[rem % A.ntypes];
    const int2 t = A.tiles[rem / A.ntypes];
    const int64_t i = t.x + il, j = t.y + (int)threadIdx.x;
    if (i >= A.Pi) return;
    float s[F], lost[F];           // sum and what its roundings lost
#pragma unroll
    for (int f = 0; f < F; ++f) s[f] = lost[f] = 0.f;
#pragma unroll 4
    for (int c = 0; c < A.chunks; ++c) {
        const float* p = A.part + (size_t)(c * per + rem) * (F * A.ni) * kPtM + threadIdx.x;
#pragma unroll
        for (int f = 0; f < F; ++f) {
            const float x = p[(size_t)(f * A.ni + il) * kPtM], y = s[f] + x, z = y - s[f];
            lost[f] += (s[f] - (y - z)) + (x - z);
            s[f] = y;
        }
    }
    if (!(i < j && j < A.P)) return;
    float v[F];
#pragma unroll
    for (int f = 0; f < F; ++f) v[f] = (s[f] + lost[f]) * A.scale;
    const float inv_sdr = A.st->inv_sdr;
    const PtBase B = pt_bases(A);
    const PtSide b = pt_side(A, type == 1, j), a = pt_side(A, type == 2, i);
    const int64_t at = row_base(A, type, i) + (type == 2 ? rdiv_base(A.nxp, A.P, A.Q, j) : j);
    const size_t wop = (size_t)A.Pi * (size_t)(A.P - A.Q), wi = w_index(A, 0, i, j);
    if constexpr (F == 5) {
        pt_emit5(A, B, type, at, wi, wop, a, b, v[0], v[1], v[2], v[3], v[4], true, inv_sdr);
    } else {
        const int em = max(a.ex, b.ex);
        const float ra = pow2f(a.ex - em) * a.R, rb = pow2f(b.ex - em) * b.R;
        const float cov = a.m * b.R + b.m * a.R + v[0];
        if (type == 0) {
            if (B.o[0] >= 0) A.scores[B.o[0] + at] = later_key(A.w[wi], ra + rb, inv_sdr);
            if (B.o[1] >= 0) A.scores[B.o[1] + at] = later_key(A.w[wi + wop], ra - rb, inv_sdr);
            if (B.o[2] >= 0) A.scores[B.o[2] + at] = later_key(A.w[wi + 2 * wop], cov, inv_sdr);
        } else {
            A.scores[B.o[3] + at] = later_key(A.w[wi + (size_t)(type + 2) * wop], cov, inv_sdr);
        }
    }
}

// the open keys of the first step, listed from w (negative and finite); entries of disabled
// operators and of pairs outside i < j are zero
__global__ void __launch_bounds__(256) k_pt_open(PtArgs A, int64_t n) {
    const int lane = threadIdx.x & 31;
    const int64_t PQ = A.P - A.Q, step = (int64_t)gridDim.x * blockDim.x * 4;
    for (int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) * 4; e0 < n; e0 += step) {
        const int64_t e = e0 + 4 * lane;
        float v[4];
        if (e + 3 < n) {
            const float4 x = *reinterpret_cast<const float4*>(A.w + e);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = e + q < n ? A.w[e + q] : 0.f;
        }
        int c = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) c += v[q] < 0.f && v[q] > -INFINITY;
        if (!__any_sync(0xffffffffu, c)) continue;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        unsigned at = 0;
        if (lane == 31) at = atomicAdd(A.count, (unsigned)incl);
        int64_t slot = (int64_t)__shfl_sync(0xffffffffu, at, 31) + incl - c;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (v[q] < 0.f && v[q] > -INFINITY) {
                const int64_t row = (e + q) / PQ, j = A.Q + (e + q) - row * PQ, op = row / A.Pi, i = row - op * A.Pi;
                if (slot < A.cap)
                    A.list[slot] = ((unsigned long long)op << 61) | ((unsigned long long)i << 31) | (unsigned long long)j;
                ++slot;
            }
    }
}

// an open candidate, and where its key and 1/sd go
struct PtOpen { int op, type; int64_t i, j; };           // +, -, x_i x_j, x_i / x_j, x_j / x_i; product form
__device__ __forceinline__ PtOpen pt_open(unsigned long long word) {
    const int op = (int)(word >> 61);
    return PtOpen{op, op < 2 ? 0 : op - 2, (int64_t)((word >> 31) & 0x3FFFFFFFull), (int64_t)(word & 0x7FFFFFFFull)};
}
// exponent of the units of its 1/sd
__device__ __forceinline__ int pt_scale(const PtArgs& A, const PtOpen& o) {
    return o.op < 2 ? max(__ldg(A.ex + o.i), __ldg(A.ex + o.j))
                    : __ldg(A.ex + (o.type == 2 ? A.P : 0) + o.i) + __ldg(A.ex + (o.type == 1 ? A.P : 0) + o.j);
}
template <bool FIRST> __device__ __forceinline__ void pt_close(const PtArgs& A, unsigned long long word, const PtOpen& o, const PtKey& k) {
    const int64_t rank = o.type == 0 ? sym_base(A.nxp, A.P, A.Q, o.i) + o.j
                         : o.type == 1 ? div_base(A.nxp, A.P, A.Q, o.i) + o.j : rdiv_base(A.nxp, A.P, A.Q, o.j) + o.i;
    A.scores[A.sp->sec[A.sec[o.op < 3 ? o.op : 3]].base + rank] = k.key;
    if (FIRST) {
        const size_t wi = w_index(A, o.op, o.i, o.j);
        const float dc = -A.w[wi];
        if (k.w > 0.f && !(dc * k.w <= 0.5f * A.tol))
            A.list[A.cap + atomicAdd(A.count + 1, 1u)] = word;      // at most one entry per listed key
        A.w[wi] = k.w > 0.f ? k.w : -INFINITY;
    }
}

// open keys: one warp per candidate (one CTA, many samples), the sums of its definition sample by sample, in FP32 with
// runs of 32 samples per lane.  Products from the FP32 values, shifted by sample 0's product (a
// value near zero keeps its relative precision beside a reciprocal that is huge there); + and -
// from the centred values (hi + lo), which cancel without the values' own rounding.  A candidate
// that cancels so far that the operands' FP32 rounding or that of the shifted sums could move its
// key by more than three quarters of the screening margin, or that these sums reject, is left to
// k_pt_exact.  FIRST: stores 1/sd and lists the candidates whose covariance stays open at every
// step; later steps run those alone.
template <bool FIRST, bool CTA>
__global__ void __launch_bounds__(256) k_pt_direct(PtArgs A, const float* __restrict__ r) {
    __shared__ float sh[16];
    const int64_t n = min((int64_t)A.count[FIRST ? 0 : 1], A.cap);
    const int lane = CTA ? (int)threadIdx.x : (int)(threadIdx.x & 31);       // of the threads that share a candidate
    const int stride = CTA ? 2 * (int)blockDim.x : 64;
    const float inv_sdr = A.st->inv_sdr, rs = A.st->rscale, inv_n = 1.f / (float)A.N;
    const float sum_t = TgtView<float>::sum(A.st), sd_t = TgtView<float>::sd(A.st);
    const unsigned long long* list = FIRST ? A.list : A.list + A.cap;
    const size_t lo = (size_t)A.P * A.Kpad;
    for (int64_t e = CTA ? (int64_t)blockIdx.x : ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n;
         e += CTA ? (int64_t)gridDim.x : ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const unsigned long long word = list[e];
        const PtOpen o = pt_open(word);
        const int op = o.op, scale = pt_scale(A, o);
        const int64_t i = o.i, j = o.j;
        float t1 = 0.f, t2 = 0.f, tr = 0.f, s1 = 0.f, s2 = 0.f, sr = 0.f;
        int q = 0;
        auto add = [&](float u0, float u1, float y0, float y1) {
            s1 += u0 + u1;
            s2 = fmaf(u0, u0, fmaf(u1, u1, s2));
            sr = fmaf(u0, y0, fmaf(u1, y1, sr));
            if ((++q & 15) == 0) { t1 += s1; t2 += s2; tr += sr; s1 = s2 = sr = 0.f; }
        };
        auto total = [&]() {
            t1 = group_sum<CTA>(t1 + s1, sh); t2 = group_sum<CTA>(t2 + s2, sh); tr = group_sum<CTA>(tr + sr, sh);
        };
        PtKey k{-1.f, -INFINITY};
        bool sure = false;
        if (op < 2) {
            const PtSide a = pt_side(A, 0, i), b = pt_side(A, 0, j);
            const __half* xa = A.rows + (size_t)i * A.Kpad;
            const __half* xb = A.rows + (size_t)j * A.Kpad;
            const int em = scale;
            const float ca = pow2f(a.ex - em), cb = op == 1 ? -pow2f(b.ex - em) : pow2f(b.ex - em), g = 3.0517578125e-5f;
            for (int s = 2 * lane; s < A.Kpad; s += stride) {                      // padding: all zero
                const float2 ah = __half22float2(*reinterpret_cast<const __half2*>(xa + s));
                const float2 al = __half22float2(*reinterpret_cast<const __half2*>(xa + lo + s));
                const float2 bh = __half22float2(*reinterpret_cast<const __half2*>(xb + s));
                const float2 bl = __half22float2(*reinterpret_cast<const __half2*>(xb + lo + s));
                add(ca * ((ah.x + al.x) * g) + cb * ((bh.x + bl.x) * g), ca * ((ah.y + al.y) * g) + cb * ((bh.y + bl.y) * g),
                    s < A.N ? r[s] * rs : 0.f, s + 1 < A.N ? r[s + 1] * rs : 0.f);
            }
            total();
            const float v0 = ca * a.x0 + cb * b.x0;
            t1 *= inv_n;
            const float var = t2 * inv_n - t1 * t1;
            k = pt_key(var, 0.f, tr * inv_n, 0.f, v0, ca * a.m + cb * b.m, 0.f,
                       a.lg < INFINITY && b.lg < INFINITY && fabsf(v0) * pow2f(em) <= (float)kValueCap,
                       exp2f(kLogRms - 2.f * (float)em), A.tol, inv_sdr);
            // values kErrRow 2^-24 and 2^-39 off, in the sums of v r and of v^2
            const float off = 2.f * kErrRow * kU * (ca * a.s + fabsf(cb) * b.s) + 4.f * kFloor * (ca + fabsf(cb));
            sure = k.key >= 0.f && off * off <= kTolDirect * kTolDirect * var;
        } else {
            const bool quot = op > 2;
            const float* xa = A.val32 + (size_t)(op == 4 ? j : i) * A.Kpad;      // numerator
            const float* xb = A.val32 + (size_t)(op == 4 ? i : j) * A.Kpad;
            const float v0 = quot ? xa[0] * rcp<float>(xb[0]) : xa[0] * xb[0];
            for (int s = 2 * lane; s < A.N; s += stride) {
                const float2 x = *reinterpret_cast<const float2*>(xa + s);
                float2 z = *reinterpret_cast<const float2*>(xb + s);
                if (quot) { z.x = rcp<float>(z.x); z.y = rcp<float>(z.y); }
                const bool two = s + 1 < A.N;
                add(fmaf(x.x, z.x, -v0), two ? fmaf(x.y, z.y, -v0) : 0.f, r[s], two ? r[s + 1] : 0.f);
            }
            total();
            k.key = finalize<float>(t1, t2, tr, v0, A.N, sum_t, sd_t);
            if (k.key >= 0.f) {
                t1 *= inv_n;
                t2 *= inv_n;
                const float var = t2 - t1 * t1, mean = v0 + t1, half = 0.5f * kTolDirect;
                k.w = __frsqrt_rn(var) * pow2f(scale / 2) * pow2f(scale - scale / 2);
                // values 3 2^-24 off (two operands, the reciprocal), in the sums of v r and of v^2; sums of
                // u = v - v0 about 40 2^-24 of E u^2 off
                sure = k.w > 0.f && 36.f * kU * kU * (var + mean * mean) <= kTolDirect * kTolDirect * var && 60.f * kU * t2 <= half * var;
            }
        }
        if (lane == 0) {
            if (sure) pt_close<FIRST>(A, word, o, k);
            else A.list[2 * A.cap + atomicAdd(A.count + 3, 1u)] = word;
        }
    }
}

// key and 1/sd from the sums of u = v - v0: moments in FP64, root and quotients in FP32 (in FP64
// they took twice as long as 333 samples' sums).  Rejected where finalize<double> rejects.
__device__ __forceinline__ PtKey pt_key64(const PtArgs& A, double s1, double s2, double sr, double v0, int scale) {
    const double ms = s1 * A.inv_n, var = fma(s2, A.inv_n, -ms * ms), cov = fma(sr, A.inv_n, -ms * (A.st->tsum * A.inv_n));
    const double mean = v0 + ms, mx = fmax(fabs(v0), fabs(mean));
    const int hv = __double2hiint(var), hc = __double2hiint(cov) & 0x7fffffff;
    if (!(fabs(v0) <= kValueCap) || !(var > kConstRel * kConstRel * (1.0 - 1e-9) * mx * mx) || hv >= 0x7ff00000 || hc >= 0x7ff00000)
        return PtKey{-1.f, -INFINITY};
    const int h = ((hv >> 20) - 1023) >> 1;                            // var = m 4^h, m in [1, 4)
    const float rm = __frsqrt_rn(scaled_f32(var, -2 * h));
    const int er = 127 - (__float_as_int(A.st->rscale) >> 23);         // rscale = 2^-er
    return PtKey{fabsf(scaled_f32(cov, -h - er)) * rm * A.st->inv_sdr, rm * pow2f(scale - h)};
}

// ... and those from the FP64 operand values, summed in FP64: the margin that the selection relies
// on holds for every key.  Bound by the FP64 pipe, five operations a sample; there are few (0.1 to
// 6% of the open keys), so long samples take a cluster of four CTAs each.
constexpr int kExactCtas = 4;
template <bool FIRST, bool CTA>
__global__ void __launch_bounds__(256) k_pt_exact(PtArgs A) {
    __shared__ double sh[16], part[3];
    const int64_t n = min((int64_t)A.count[3], A.cap);
    namespace cg = cooperative_groups;
    const int rank = CTA ? (int)cg::this_cluster().block_rank() : 0;
    const int t = CTA ? rank * (int)blockDim.x + (int)threadIdx.x : (int)(threadIdx.x & 31);
    const int nt = CTA ? kExactCtas * (int)blockDim.x : 32;
    for (int64_t e = CTA ? (int64_t)blockIdx.x / kExactCtas : ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n;
         e += CTA ? (int64_t)gridDim.x / kExactCtas : ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const unsigned long long word = A.list[2 * A.cap + e];
        const PtOpen o = pt_open(word);
        const int64_t a = o.op == 4 ? o.j : o.i, b = o.op == 4 ? o.i : o.j;
        const bool inv = o.op > 2 && A.inv64;
        const double *xa = A.val64 + (size_t)a * A.N, *vb = A.val64 + (size_t)b * A.N, *xb = inv ? A.inv64 + (size_t)b * A.N : vb;
        auto value = [&](double x, double y, int s) {          // as the FP64 re-score's (opref_val)
            if (o.op == 0) return x + y;
            if (o.op == 1) return x - y;
            if (o.op == 2) return x * y;
            if (!inv) return x / y;
            return (__double2hiint(y) & 0x7ff00000) != 0x7ff00000 ? x * y : x / vb[s];
        };
        const double v0 = value(xa[0], xb[0], 0);
        double s1 = 0.0, s2 = 0.0, sr = 0.0;
        for (int s0 = t; s0 < A.N; s0 += 4 * nt) {            // four samples' loads in flight
            double x[4], y[4], r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int s = min(s0 + q * nt, A.N - 1);
                x[q] = xa[s]; y[q] = xb[s]; r[q] = A.tc64[s];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int s = s0 + q * nt;
                if (s >= A.N) break;
                const double u = value(x[q], y[q], s) - v0;
                s1 += u;
                s2 = fma(u, u, s2);
                sr = fma(u, r[q], sr);
            }
        }
        s1 = group_sum<CTA>(s1, sh); s2 = group_sum<CTA>(s2, sh); sr = group_sum<CTA>(sr, sh);
        if constexpr (CTA) {
            if (threadIdx.x == 0) { part[0] = s1; part[1] = s2; part[2] = sr; }
            cg::this_cluster().sync();
            if (t == 0)
                for (int q = 1; q < kExactCtas; ++q) {
                    const double* p = cg::this_cluster().map_shared_rank(part, q);
                    s1 += p[0]; s2 += p[1]; sr += p[2];
                }
            cg::this_cluster().sync();             // read before the next candidate's, and before a CTA ends
        }
        if (t == 0) pt_close<FIRST>(A, word, o, pt_key64(A, s1, s2, sr, v0, pt_scale(A, o)));
    }
}

// ids below the top level: |E x'r| / sqrt(E x'^2) of the operand itself
__global__ void __launch_bounds__(256) k_pt_low(PtArgs A, const unsigned char* __restrict__ valid) {
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f == 0) A.count[3] = 0u;               // (this step's keys left to FP64 are listed later)
    if (f >= A.P) return;
    const float4 p = A.par[f];
    A.scores[f] = valid[f] && p.w < INFINITY ? fabsf(A.R[f]) * __frsqrt_rn(p.y) * A.st->inv_sdr : -1.f;
}

bool pt_map(CUtensorMap* m, void* base, int64_t rows, int Kpad, int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)Kpad, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)Kpad * 2};
    const cuuint32_t box[2] = {kPtK, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, gdim, gstride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

namespace {

// Partial sums of long samples are kept for at most this much at a time, whole tiles of all chunks
// (one tile at least): 402 operands over 65 536 samples have 0.35 GB, 2355 over 16 384 would have 1.5.
constexpr size_t kPtPart = (size_t)1 << 30;
// The buffers may take this much, or half of what is left of the device beside the context's
// others: they make a fit faster, and the scores alone are as large as the deviations kept for
// later steps (half as large in the EQ2 grammar).
constexpr size_t kPtSmall = (size_t)1 << 30;

// i0 of the tiles of one row of j tiles: [0, end), every ni
int64_t pt_i_end(const PairTc& t, int64_t j0) { return std::min(t.Pi, std::min(j0 + kPtM, t.P) - 1); }

// sizes, tiles and chunks of a context's pair stage
void pt_layout(const sisso_ctx* c, PairTc& t) {
    const Space& sp = c->space;
    const int L = c->rung;
    t.P = sp.phi[L - 1];
    t.Q = L >= 2 ? sp.phi[L - 2] : 0;
    t.Pi = sp.grammar == SISSO_GRAMMAR_NEW_X_PREV && L >= 3 ? t.Q : t.P;
    t.runs = (c->N + kPtK - 1) / kPtK;
    t.Kpad = t.runs * kPtK;
    t.cap = (int64_t)1 << 22;
    t.n_w = 5 * (size_t)t.Pi * (size_t)(t.P - t.Q);
    t.part_bytes = 0;
    for (int v = 0; v < 2; ++v) {
        // i tiles: 48 for the five sums; for the one sum the multiple of 48 up to 240 that pads
        // the i operands least, the largest of those that leave every SM two units (long samples
        // are cut into chunks, so there a unit is a tile's chunk)
        t.ni[v] = kPtI5;
        if (v == 1) {
            auto padded = [&](int ni) { return (t.Pi + ni - 1) / ni * ni; };
            const int64_t nj = (t.P - t.Q + kPtM - 1) / kPtM, cuts = t.runs > kMaxRuns ? (t.runs + 15) / 16 : 1;
            for (int ni = 2 * kPtI5; ni <= kPtI1; ni += kPtI5)
                if (padded(ni) <= padded(t.ni[v]) && 3 * nj * ((t.Pi + ni - 1) / ni) * cuts >= 2 * c->sms) t.ni[v] = ni;
        }
        t.n_tiles[v] = 0;
        for (int64_t j0 = t.Q; j0 < t.P; j0 += kPtM) t.n_tiles[v] += (std::max<int64_t>(0, pt_i_end(t, j0)) + t.ni[v] - 1) / t.ni[v];
        // sample chunks: at most kMaxRuns runs each (the runs are added in FP32); a chunk of 16
        // runs or more costs the partials' round trip little, so long samples are cut until
        // every SM has about four units
        const int64_t units = std::max<int64_t>(1, 3 * t.n_tiles[v]);
        int64_t ch = (t.runs + kMaxRuns - 1) / kMaxRuns;
        if (ch > 1) ch = std::max(ch, std::min<int64_t>((t.runs + 15) / 16, (4 * c->sms + units - 1) / units));
        t.run_len[v] = (int)((t.runs + ch - 1) / ch);
        t.chunks[v] = (t.runs + t.run_len[v] - 1) / t.run_len[v];
        t.batch[v] = std::max<int64_t>(1, t.n_tiles[v]);
        if (t.chunks[v] > 1) {
            const size_t tile = sizeof(float) * 3 * (size_t)t.chunks[v] * (v == 0 ? 5 : 1) * t.ni[v] * kPtM;
            t.batch[v] = std::max<int64_t>(1, std::min<int64_t>(t.batch[v], (int64_t)(kPtPart / tile)));
            t.part_bytes = std::max(t.part_bytes, tile * (size_t)t.batch[v]);
        }
    }
}

size_t pt_bytes(const PairTc& t) {
    const size_t K = (size_t)t.Kpad, P = (size_t)t.P;
    return 20 * P * K + 8 * (size_t)t.Pi * K + 48 * P + sizeof(float) * t.n_w + sizeof(unsigned long long) * 3 * t.cap +
           t.part_bytes + sizeof(int2) * (size_t)(t.n_tiles[0] + t.n_tiles[1]);
}

}  // namespace

// Used for the FP32 and the mixed forms when the operands' FP32 and FP64 values are kept (8 GB of
// the former at most) and the buffers, 20 to 28 bytes per padded operand value and 20 per pair,
// fit; other contexts keep the CUDA-core kernel.
bool pair_tc_possible(const sisso_ctx* c) {
    const Space& sp = c->space;
    const int64_t P = sp.phi[c->rung - 1];
    const int64_t Kpad = ((int64_t)c->N + kPtK - 1) / kPtK * kPtK;
    bool any = false;
    for (int s = 0; s < sp.nsec; ++s) any |= sp.sec[s].level == c->rung && sp.sec[s].op <= DIV;
    if (!any || !c->opcache32 || !c->opval64 || P < 2 || P > ((int64_t)1 << 27) || P * Kpad * 16 > ((int64_t)40 << 30) ||
        encode_fn() == nullptr)
        return false;
    PairTc t;
    pt_layout(c, t);
    const size_t need = pt_bytes(t);
    return need <= kPtSmall || need <= memory_left(c) / 2;
}

// per-operand rows, tiles and buffers of a context (they depend on X only); without them
// (c->pt null) where the device has no room
sisso_status pair_tc_alloc(sisso_ctx* c) {
    PairTc* t = new (std::nothrow) PairTc();
    if (!t) return SISSO_ERR_OOM;
    c->pt = t;
    pt_layout(c, *t);
    std::vector<int2>* tiles = t->tile_list;
    for (int v = 0; v < 2; ++v) {
        tiles[v].reserve((size_t)t->n_tiles[v]);
        for (int64_t j0 = t->Q; j0 < t->P; j0 += kPtM)
            for (int64_t i0 = 0; i0 < pt_i_end(*t, j0); i0 += t->ni[v]) tiles[v].push_back(make_int2((int)i0, (int)j0));
    }
    const size_t K = (size_t)t->Kpad, P = (size_t)t->P;
    const std::string err = c->err;
    sisso_status st;
    if ((st = ctx_alloc(c, (void**)&t->rows, 16 * P * K, "pair rows")) ||
        (st = ctx_alloc(c, (void**)&t->rrows, 8 * (size_t)t->Pi * K, "pair target rows")) ||
        (st = ctx_alloc(c, (void**)&t->val32, 4 * P * K, "pair FP32 values")) ||
        (st = ctx_alloc(c, (void**)&t->par, sizeof(float4) * 2 * P, "pair operands")) ||
        (st = ctx_alloc(c, (void**)&t->ex, sizeof(int) * 2 * P, "pair exponents")) ||
        (st = ctx_alloc(c, (void**)&t->R, sizeof(float) * 2 * P, "pair R")) ||
        (st = ctx_alloc(c, (void**)&t->w, sizeof(float) * t->n_w, "pair 1/sd")) ||
        (st = ctx_alloc(c, (void**)&t->list, sizeof(unsigned long long) * 3 * t->cap, "pair open keys")) ||
        (st = ctx_alloc(c, (void**)&t->count, sizeof(unsigned) * 4, "pair counts")) ||
        (st = ctx_alloc(c, (void**)&t->part, t->part_bytes, "pair partials")) ||
        (st = ctx_alloc(c, (void**)&t->tiles[0], sizeof(int2) * tiles[0].size(), "pair tiles")) ||
        (st = ctx_alloc(c, (void**)&t->tiles[1], sizeof(int2) * tiles[1].size(), "pair tiles"))) {
        for (void* p : {(void*)t->rows, (void*)t->rrows, (void*)t->val32, (void*)t->par, (void*)t->ex, (void*)t->R, (void*)t->w,
                        (void*)t->list, (void*)t->count, (void*)t->part, (void*)t->tiles[0], (void*)t->tiles[1]})
            ctx_free(c, p);
        pair_tc_free(c);
        if (st == SISSO_ERR_OOM) { c->err = err; return SISSO_OK; }
        return st;
    }
    for (int v = 0; v < 2; ++v) {
        cudaMemcpyAsync(t->tiles[v], tiles[v].data(), sizeof(int2) * tiles[v].size(), cudaMemcpyHostToDevice, c->stream);
        if (!pt_map(&t->mapN[v], t->rows, 8 * t->P, t->Kpad, t->ni[v]) ||
            !pt_map(&t->mapR[v], t->rrows, 4 * t->Pi, t->Kpad, t->ni[v]))
            return fail(c, SISSO_ERR_CUDA, "pair tensor maps");
    }
    if (!pt_map(&t->mapM, t->rows, 8 * t->P, t->Kpad, kPtM)) return fail(c, SISSO_ERR_CUDA, "pair tensor maps");
    const unsigned gw = (unsigned)((t->P + 3) / 4);
#define SG_PT_ROWS(ITV, GRID, BLOCK) \
    k_pt_rows<ITV><<<GRID, BLOCK, 0, c->stream>>>(c->opval64, c->opinv64, c->subvalid, t->P, c->N, t->Kpad, t->rows, t->val32, t->par, t->ex)
    if (t->Kpad <= 256) SG_PT_ROWS(4, gw, 128);
    else if (t->Kpad <= 1024) SG_PT_ROWS(16, gw, 128);
    else SG_PT_ROWS(0, (unsigned)t->P, t->Kpad <= 4096 ? 256 : 512);
#undef SG_PT_ROWS
    c->stats.launches++;
    return check_cuda(c, cudaGetLastError(), "pair_tc_alloc");
}

void pair_tc_reset(sisso_ctx* c) { if (c->pt) c->pt->ready = false; }

void pair_tc_free(sisso_ctx* c) {
    delete c->pt;          // its device buffers are the context's (ctx_alloc)
    c->pt = nullptr;
}

// keys of the top level's binary sections for the current target (tc64 / tstats).  *overflow:
// more open keys than the list holds; the caller then scores the step with the CUDA-core kernel.
sisso_status pair_tc_scores(sisso_ctx* c, const int sec[4], bool* overflow) {
    PairTc* t = c->pt;
    *overflow = false;
    const int v = t->ready ? 1 : 0;
    PtArgs A{};
    A.sp = c->space_dev;
    for (int o = 0; o < 4; ++o) A.sec[o] = sec[o];
    A.P = t->P; A.Q = t->Q; A.Pi = t->Pi;
    A.nxp = c->space.grammar == SISSO_GRAMMAR_NEW_X_PREV && c->rung >= 3;
    if (sec[0] >= 0 || sec[1] >= 0 || sec[2] >= 0) A.type[A.ntypes++] = 0;
    if (sec[3] >= 0) { A.type[A.ntypes++] = 1; A.type[A.ntypes++] = 2; }
    A.ni = t->ni[v];
    A.chunks = t->chunks[v]; A.run_len = t->run_len[v]; A.runs = t->runs;
    A.N = c->N; A.Kpad = t->Kpad; A.rows = t->rows; A.val32 = t->val32;
    A.val64 = c->opval64; A.inv64 = c->opinv64; A.tc64 = c->tc64; A.inv_n = 1.0 / c->N;
    A.scale = (float)(1.0 / (1073741824.0 * c->N));
    A.eps = (float)((kErrSum + t->run_len[v]) * std::ldexp(1.0, -24));
    A.tol = t->runs <= kFewRuns ? kTolFew : kTolMany;
    A.par = t->par; A.ex = t->ex; A.R = t->R; A.w = t->w; A.scores = c->scores; A.st = c->tstats;
    A.list = t->list; A.count = t->count; A.cap = t->cap; A.part = t->part;
    if (v == 0) {
        cudaMemsetAsync(t->count, 0, sizeof(unsigned) * 4, c->stream);
        // entries no unit writes (pairs i >= j of one set, disabled operators) read as not open
        if (!A.nxp || sec[0] < 0 || sec[1] < 0 || sec[2] < 0 || sec[3] < 0) cudaMemsetAsync(t->w, 0, sizeof(float) * t->n_w, c->stream);
    }
    if (t->Kpad <= 2048)
        k_pt_target<false><<<(unsigned)((t->P + 7) / 8), 256, 0, c->stream>>>(t->rows, c->tc32, c->tstats, t->P, t->Pi, c->N, t->Kpad, t->rrows, t->R);
    else
        k_pt_target<true><<<(unsigned)t->P, 512, 0, c->stream>>>(t->rows, c->tc32, c->tstats, t->P, t->Pi, c->N, t->Kpad, t->rrows, t->R);
    k_pt_low<<<(unsigned)((t->P + 255) / 256), 256, 0, c->stream>>>(A, c->subvalid);
    const size_t smem = v == 0 ? pt_smem_bytes<5>(A.ni) : pt_smem_bytes<1>(A.ni);
    const bool many = t->Kpad > 4096;
    if (v == 0) allow_smem(k_pair_tc<5>, pt_smem_bytes<5>(kPtI5));
    else allow_smem(k_pair_tc<1>, pt_smem_bytes<1>(kPtI1));
    for (int64_t t0 = 0; t0 < t->n_tiles[v]; t0 += t->batch[v]) {          // (one batch unless the samples are cut)
        A.tiles = t->tiles[v] + t0;
        A.n_tiles = (int)std::min(t->batch[v], t->n_tiles[v] - t0);
        const int64_t units = (int64_t)A.n_tiles * A.ntypes * A.chunks;
        const int grid = (int)std::min<int64_t>(units, c->sms);
        const unsigned gr = (unsigned)(A.n_tiles * A.ntypes * A.ni);
        if (v == 0) {
            k_pair_tc<5><<<grid, kPtThreads, smem, c->stream>>>(t->mapM, t->mapN[0], t->mapR[0], A);
            if (A.chunks > 1) k_pt_reduce<5><<<gr, kPtM, 0, c->stream>>>(A);
        } else {
            k_pair_tc<1><<<grid, kPtThreads, smem, c->stream>>>(t->mapM, t->mapN[1], t->mapR[1], A);
            if (A.chunks > 1) k_pt_reduce<1><<<gr, kPtM, 0, c->stream>>>(A);
        }
        c->stats.launches += 1 + (A.chunks > 1);
    }
    cudaLaunchAttribute cluster{};
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim.x = kExactCtas;
    cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(256);
    cfg.stream = c->stream;
    cfg.attrs = &cluster;
    cfg.numAttrs = 1;
#define SG_PT_DIRECT(FIRST)                                                                              \
    do {                                                                                                  \
        if (many) {                                                                                       \
            k_pt_direct<FIRST, true><<<c->sms * 8, 256, 0, c->stream>>>(A, c->tc32);                      \
            cfg.gridDim = dim3((unsigned)(c->sms * 8 / kExactCtas * kExactCtas));                         \
            cudaLaunchKernelEx(&cfg, k_pt_exact<FIRST, true>, A);                                         \
        } else {                                                                                          \
            k_pt_direct<FIRST, false><<<c->sms * 8, 256, 0, c->stream>>>(A, c->tc32);                     \
            k_pt_exact<FIRST, false><<<c->sms * 8, 256, 0, c->stream>>>(A);                               \
        }                                                                                                 \
    } while (0)
    if (v == 0) {
        k_pt_open<<<(unsigned)std::max<size_t>(1, std::min<size_t>((size_t)c->sms * 8, (t->n_w + 1023) / 1024)), 256, 0, c->stream>>>(A, (int64_t)t->n_w);
        SG_PT_DIRECT(true);
    } else {
        SG_PT_DIRECT(false);
    }
#undef SG_PT_DIRECT
    c->stats.launches += 4 + (v == 0);
    // a launch that was refused leaves the last step's keys: waiting alone would not tell
    sisso_status st = check_cuda(c, cudaGetLastError(), "pair scores");
    if (st) return st;
    unsigned h[4] = {0, 0, 0, 0};
    cudaMemcpyAsync(h, t->count, sizeof(h), cudaMemcpyDeviceToHost, c->stream);
    if ((st = check_cuda(c, cudaStreamSynchronize(c->stream), "pair scores"))) return st;
    if (h[2]) return fail(c, SISSO_ERR_TIMEOUT, "pair scores: a bounded wait ran out");
    c->stats.pm_keys_direct += (int64_t)h[v == 0 ? 0 : 1];
    if ((int64_t)h[0] > t->cap) *overflow = true;
    else t->ready = true;
    return SISSO_OK;
}

}  // namespace sg
