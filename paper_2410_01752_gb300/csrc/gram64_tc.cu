// gram64_tc.cu — the FP64 Gram of the standardised subspace from exact tensor-core products.
//
// GB300's FP64 pipe bounds the plain kernel (k_gram_rows): 600 features over 65 536 samples are
// 1.2e10 fused multiply-adds, 20 ms.  Here every row is rounded once to a 55-bit integer
//     q = rint(z 2^(54 - e)),  |z| < 2^e for the whole row,
// written in base 256 with digits d0 .. d6 in [-128, 127] (d0 the leading one; the error-free slicing of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication", 2012), and the
// digit products are summed on the tensor cores as FP16 integers: a product is at most 2^14 and an
// accumulator takes at most 7 x 64 of them between two reads, so every partial sum is an integer
// below 2^23, which FP32 holds exactly whatever the order of the additions.  The sums S_w of equal
// weight w = i + j <= 7 (34 of the 49 products) are added as 64-bit integers, exactly again, also
// across CTAs.  What is left out, the products of weight 8 and more, is below 2^-61 of
// 2^(ei + ej) a sample at random signs, but of one sign between a row and itself, where it is
// 2^-63.6 4^e of the Gram's 1; the rounding of q is half a unit of 2^(e - 54).  Both are averaged over
// the samples, so the result is the Gram rounded once or twice to FP64: its error against longer
// sums is below that of the FP64 accumulation it replaces.  A pair of rows with ei + ej above
// kGWide, largest values of 45 deviations and more, would lose more than an FP64 rounding (5e-15 at
// 250 deviations: reciprocals of near-equal columns) and is summed in FP64 (k_gram64_wide).
//
// One CTA takes a 128 x 64 tile of the lower triangle and a run of 64-sample blocks: one warp
// streams the seven slices of both sides with TMA (two stages of 32 samples), one issues the 68
// tcgen05.mma of a stage ordered by weight into eight TMEM accumulators of 64 columns, and eight
// warps read an accumulator as soon as its weight is complete, while the next block's products of
// the weights already read proceed.
// Measured: 200, 400 and 600 features over 65 536 samples, 200 new each, 19.8 -> 3.0 ms (2.55 the
// products, 0.29 the digits, 0.15 the moments); the tensor pipe is 27% active, the epilogue
// warps wait for TMEM: eight accumulators of 64 columns leave none to double-buffer.
#include "tc_device.cuh"

#include <cuda_fp16.h>

#include <algorithm>

namespace sg {

namespace {

constexpr int kSl = 7;                    // digits
constexpr int kW = 8;                     // weights kept
constexpr int kGM = 128, kGN = 64;        // tile
constexpr int kGK = 32;                   // samples of a stage (64-byte rows)
constexpr int kGBlock = 64;               // samples between two reads of the accumulators
constexpr int kGStages = 2;
constexpr int kGThreads = 10 * 32;
constexpr int kGWide = 11;
constexpr uint32_t kGTileA = kGM * kGK * 2, kGTileB = kGN * kGK * 2;

struct Gram64Smem {
    uint8_t a[kGStages][kSl][kGTileA];
    uint8_t b[kGStages][kSl][kGTileB];
    uint64_t full[kGStages], empty[kGStages], acc_full[kW], acc_empty[kW];
    uint32_t tmem_base;
    int failed;
};

// digits of rows [row0, row0 + gridDim.x): one CTA per row, all on the integer pipe
__global__ void __launch_bounds__(512) k_gram_slices(const double* __restrict__ Z, int N, int Kpad, int row0, int R,
                                                     __half* __restrict__ sl, int* __restrict__ ex) {
    __shared__ unsigned long long red[16];
    const int row = row0 + blockIdx.x, t = threadIdx.x;
    const double* z = Z + (size_t)row * N;
    unsigned long long mx = 0;
    for (int i = t; i < N; i += 512) mx = max(mx, (unsigned long long)__double_as_longlong(z[i]) & 0x7FFFFFFFFFFFFFFFull);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((t & 31) == 0) red[t >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 16; ++q) mx = max(mx, red[q]);
    const int top = (int)(mx >> 52) + 1;                       // biased exponent of 2^e
    if (t == 0) ex[row] = top - 1023;
    for (int i0 = t * 8; i0 < Kpad; i0 += 512 * 8) {
        __half h[kSl][8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u;
            long long q = 0;
            if (i < N) {
                const unsigned long long bits = (unsigned long long)__double_as_longlong(z[i]);
                const int be = (int)((bits >> 52) & 2047u);
                const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (be ? 1ull << 52 : 0ull);
                const int sh = (be ? be : 1) - top + 2;        // <= 1
                if (sh >= 0) q = (long long)(m << sh);
                else if (sh > -55) q = (long long)((m + (1ull << (-sh - 1))) >> -sh);
                if (bits >> 63) q = -q;
            }
#pragma unroll
            for (int s = kSl - 1; s >= 0; --s) {
                const int d = s > 0 ? (int)(signed char)(q & 255) : (int)q;
                h[s][u] = __int2half_rn(d);
                q = (q - d) >> 8;
            }
        }
#pragma unroll
        for (int s = 0; s < kSl; ++s)
            *reinterpret_cast<uint4*>(sl + ((size_t)s * R + row) * Kpad + i0) = *reinterpret_cast<const uint4*>(h[s]);
    }
}

struct Gram64Args {
    int R, row0, n, tiles_n, splits, blocks, per;   // row stride of a slice, first new row, rows, col tiles, runs, 64-sample blocks, blocks of a run
    unsigned long long* acc;                          // [2][m_pad][n_pad]
    int n_pad;
    size_t plane;
    int* err;
};

__global__ void __launch_bounds__(kGThreads, 1)
k_gram64_tc(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, Gram64Args A) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Gram64Smem& S = *reinterpret_cast<Gram64Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x / A.splits, run = blockIdx.x % A.splits;
    const int tm = tile / A.tiles_n, tn = tile % A.tiles_n;
    const int i0 = A.row0 + tm * kGM, j0 = tn * kGN;                    // first rows of the tile
    const int b0 = run * A.per, nb = min(A.per, A.blocks - b0);         // its 64-sample blocks
    if (j0 > min(i0 + kGM, A.n) - 1 || nb <= 0) return;                 // above the diagonal (uniform)
    if (threadIdx.x == 0) {
        for (int s = 0; s < kGStages; ++s) { mbar_init(&S.full[s], 1); mbar_init(&S.empty[s], 1); }
        for (int w = 0; w < kW; ++w) { mbar_init(&S.acc_full[w], 1); mbar_init(&S.acc_empty[w], 8); }
        S.failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = S.tmem_base;
    const int stages = nb * (kGBlock / kGK);
    if (warp == 8 && lane == 0) {
        int issued = 0;
        bool ok = true;
        for (int k = 0; k < stages; ++k) {
            const int s = k % kGStages;
            if (k >= kGStages && !mbar_wait(&S.empty[s], ((uint32_t)(k / kGStages) & 1u) ^ 1u)) { ok = false; break; }
            mbar_expect_tx(&S.full[s], kSl * (kGTileA + kGTileB));
            const int x = b0 * kGBlock + k * kGK;
#pragma unroll
            for (int q = 0; q < kSl; ++q) {
                tma_load_2d(S.a[s][q], &map_a, x, q * A.R + i0, &S.full[s]);
                tma_load_2d(S.b[s][q], &map_b, x, q * A.R + j0, &S.full[s]);
            }
            ++issued;
        }
        if (!ok) {
            S.failed = 1;
            for (int k = (issued > kGStages ? issued - kGStages : 0); k < issued; ++k)
                mbar_wait(&S.full[k % kGStages], (uint32_t)(k / kGStages) & 1u);
        }
    } else if (warp == 9 && lane == 0) {
        bool ok = true;
        constexpr uint32_t idesc = idesc_f16(0, kGM, kGN);
        for (int k = 0; k < stages && ok; ++k) {
            const int s = k % kGStages;
            const bool first = k % (kGBlock / kGK) == 0, last = (k + 1) % (kGBlock / kGK) == 0;
            const int block = k / (kGBlock / kGK);
            if (!mbar_wait(&S.full[s], (uint32_t)(k / kGStages) & 1u)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t da = desc_sw64(smem_u32(S.a[s][0])), db = desc_sw64(smem_u32(S.b[s][0]));
#pragma unroll 1
            for (int w = 0; w < kW; ++w) {
                if (first && block > 0) {
                    if (!mbar_wait(&S.acc_empty[w], (uint32_t)(block - 1) & 1u)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                const int lo = max(0, w - (kSl - 1)), hi = min(w, kSl - 1);
#pragma unroll 1
                for (int i = lo; i <= hi; ++i) {
                    const uint64_t a = da + (uint64_t)(i * (kGTileA >> 4)), b = db + (uint64_t)((w - i) * (kGTileB >> 4));
#pragma unroll
                    for (int h = 0; h < kGK / 16; ++h)
                        mma_f16(tmem + (uint32_t)(w * kGN), a + (uint64_t)(2 * h), b + (uint64_t)(2 * h), idesc,
                                first && i == lo && h == 0 ? 0u : 1u);
                }
                if (last) mma_commit(&S.acc_full[w]);
            }
            if (ok) mma_commit(&S.empty[s]);
        }
        if (!ok) {
            S.failed = 1;
            // the loads in flight land before the CTA goes (bounded; the TMA thread waits for its own)
            mma_commit(&S.empty[0]);
        }
    } else if (warp < 8) {
        // warp: rows 32 (warp % 4) .., columns 32 (warp / 4) ..
        long long hi[32], lo[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
        bool ok = true;
        for (int block = 0; block < nb && ok; ++block) {
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                ok = ok && mbar_wait(&S.acc_full[w], (uint32_t)block & 1u);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t r[32];
                tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(w * kGN + (warp >> 2) * 32), r);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&S.acc_empty[w])) : "memory");
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const long long v = (long long)__float2int_rn(__uint_as_float(r[c])) * (1 << (8 * (3 - (w & 3))));
                    if (w < 4) hi[c] += v;
                    else lo[c] += v;
                }
            }
        }
        if (!ok) S.failed = 1;
        const int row = tm * kGM + (warp & 3) * 32 + lane;               // among the new rows
        const int gi = A.row0 + row;
        if (ok && gi < A.n) {
            unsigned long long* out = A.acc + (size_t)row * A.n_pad + j0 + (warp >> 2) * 32;
#pragma unroll
            for (int c = 0; c < 32; ++c)
                if (j0 + (warp >> 2) * 32 + c <= gi) {
                    atomicAdd(out + c, (unsigned long long)hi[c]);
                    atomicAdd(out + A.plane + c, (unsigned long long)lo[c]);
                }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && S.failed) atomicExch(A.err, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// G from the integer sums: sum q_i q_j = 2^72 (256^3 S_0 + .. + S_3) + 2^40 (256^3 S_4 + .. + S_7).
// Pairs with too wide a range, and all of them where a wait ran out (err: the sums are unusable), go
// to the list instead.
__global__ void k_gram64_finish(const unsigned long long* __restrict__ acc, size_t plane, int n_pad, const int* __restrict__ ex,
                                const int* __restrict__ err, int N, int row0, int n, int ld, double* __restrict__ G,
                                float* __restrict__ G32, int2* __restrict__ list, unsigned* __restrict__ count) {
    const bool bad = *err != 0;
    const int64_t total = (int64_t)(n - row0) * n;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / n), j = (int)(e % n), i = row0 + r;
        if (j > i) continue;
        if (bad || ex[i] + ex[j] > kGWide) { list[atomicAdd(count, 1u)] = make_int2(i, j); continue; }
        const long long hi = (long long)acc[(size_t)r * n_pad + j], lo = (long long)acc[plane + (size_t)r * n_pad + j];
        const double s = scalbn((double)hi * 4294967296.0 + (double)lo, ex[i] + ex[j] - 68) / N;
        G[(size_t)i * ld + j] = s;
        G[(size_t)j * ld + i] = s;
        G32[(size_t)i * ld + j] = (float)s;
        G32[(size_t)j * ld + i] = (float)s;
    }
}

// the listed entries, one CTA each
__global__ void __launch_bounds__(256) k_gram64_wide(const double* __restrict__ Z, int N, int ld, const int2* __restrict__ list,
                                                     const unsigned* __restrict__ count, double* __restrict__ G,
                                                     float* __restrict__ G32) {
    __shared__ double red[8];
    const unsigned m = *count;
    for (unsigned e = blockIdx.x; e < m; e += gridDim.x) {
        const int2 p = list[e];
        const double *a = Z + (size_t)p.x * N, *b = Z + (size_t)p.y * N;
        double s = 0.0;
        for (int t = threadIdx.x; t < N; t += 256) s += a[t] * b[t];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < 8; ++q) s += red[q];
            s /= N;
            G[(size_t)p.x * ld + p.y] = G[(size_t)p.y * ld + p.x] = s;
            G32[(size_t)p.x * ld + p.y] = G32[(size_t)p.y * ld + p.x] = (float)s;
        }
        __syncthreads();
    }
}

// b[i] = Z_i . y~ / N, one CTA per new row
__global__ void __launch_bounds__(256) k_gram64_b(const double* __restrict__ Z, const double* __restrict__ yc, int N, int row0,
                                                  double* __restrict__ b, float* __restrict__ b32) {
    __shared__ double red[8];
    const int i = row0 + blockIdx.x;
    const double* z = Z + (size_t)i * N;
    double s = 0.0;
    for (int t = threadIdx.x; t < N; t += 256) s += z[t] * yc[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) s += red[q];
        s /= N;
        b[i] = s;
        b32[i] = (float)s;
    }
}

bool gram64_map(CUtensorMap* m, const __half* base, int64_t rows, int64_t Kpad, int box) {
    const cuuint64_t dims[2] = {(cuuint64_t)Kpad, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)Kpad * 2};
    const cuuint32_t b[2] = {(cuuint32_t)kGK, (cuuint32_t)box}, es[2] = {1, 1};
    return encode_fn() &&
           encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, b, es,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t gram64_kpad(int N) { return ((int64_t)N + kGBlock - 1) / kGBlock * kGBlock; }

}  // namespace

// The rule: many samples, and enough multiply-adds that the FP64 pipe takes longer than the
// slices and the tiles' padding (n_new rows in tiles of 128): 5e8 multiply-adds, half of them left of
// the diagonal, are 0.5 ms of the FP64 pipe against 0.15 here.  The slices are kept for the
// context's later steps, 14 bytes a value.
bool gram64_tc_possible(int N, int n_new, int n, int n_cap) {
    return N >= 8192 && N <= (1 << 23) && (double)n_new * n * N >= 5e8 && gram64_kpad(N) * n_cap * 14 <= ((int64_t)16 << 30) &&
           encode_fn() != nullptr;
}

size_t gram64_tc_bytes(int N, int n_cap) { return (size_t)gram64_kpad(N) * n_cap * kSl * sizeof(__half); }

// rows [n_old, n) of G and b; slices of the rows below n_old from earlier calls (sl, ex: room for
// n_cap rows).  first: the first row without slices
sisso_status gram64_tc(sisso_ctx* c, const double* Z, const double* yc, int N, int first, int n_old, int n, int n_cap, int ld,
                       void* sl, int* ex, double* G, double* b, float* G32, float* b32) {
    const int Kpad = (int)gram64_kpad(N), n_new = n - n_old;
    __half* slices = static_cast<__half*>(sl);
    Gram64Args A{};
    A.R = n_cap; A.row0 = n_old; A.n = n;
    const int tiles_m = (n_new + kGM - 1) / kGM;
    A.tiles_n = (n + kGN - 1) / kGN;
    A.blocks = Kpad / kGBlock;
    const int tiles = tiles_m * A.tiles_n;
    // runs of samples: one wave of CTAs, at least eight blocks each
    A.splits = std::max(1, std::min(A.blocks / 8, c->sms / tiles));
    A.per = (A.blocks + A.splits - 1) / A.splits;
    A.n_pad = A.tiles_n * kGN;
    A.plane = (size_t)tiles_m * kGM * A.n_pad;
    // sums, the error flag and the list's length, the list
    sisso_status st = tmp_alloc(c, (void**)&A.acc, sizeof(unsigned long long) * (2 * A.plane + 1 + (size_t)n_new * n), "gram sums");
    if (st) return st;
    cudaMemsetAsync(A.acc, 0, sizeof(unsigned long long) * (2 * A.plane + 1), c->stream);
    A.err = reinterpret_cast<int*>(A.acc + 2 * A.plane);
    unsigned* wide = reinterpret_cast<unsigned*>(A.err + 1);
    int2* list = reinterpret_cast<int2*>(A.acc + 2 * A.plane + 1);
    CUtensorMap ma, mb;
    if (!gram64_map(&ma, slices, (int64_t)kSl * n_cap, Kpad, kGM) || !gram64_map(&mb, slices, (int64_t)kSl * n_cap, Kpad, kGN)) {
        cudaFreeAsync(A.acc, c->stream);
        return fail(c, SISSO_ERR_CUDA, "gram tensor maps");
    }
    k_gram_slices<<<n - first, 512, 0, c->stream>>>(Z, N, Kpad, first, n_cap, slices, ex);
    const size_t sm = sizeof(Gram64Smem) + 1024;
    cudaFuncSetAttribute(k_gram64_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_gram64_tc<<<tiles * A.splits, kGThreads, sm, c->stream>>>(ma, mb, A);
    k_gram64_finish<<<std::max(1, std::min(c->sms * 4, (int)(((int64_t)n_new * n + 255) / 256))), 256, 0, c->stream>>>(
        A.acc, A.plane, A.n_pad, ex, A.err, N, n_old, n, ld, G, G32, list, wide);
    k_gram64_wide<<<c->sms * 8, 256, 0, c->stream>>>(Z, N, ld, list, wide, G, G32);
    k_gram64_b<<<n_new, 256, 0, c->stream>>>(Z, yc, N, n_old, b, b32);
    c->stats.launches += 5;
    cudaFreeAsync(A.acc, c->stream);
    return check_cuda(c, cudaGetLastError(), "gram64_tc");
}

}  // namespace sg

// G = Z Z^T / N and b = Z yc / N in FP64 (host or device Z [n x N] and yc; outputs host), by the
// exact tensor-core products
extern "C" sisso_status sisso_gram_fp64(const double* Z, const double* yc, int n, int N, double* G, double* b) {
    using namespace sg;
    if (!Z || !yc || !G || !b || n < 1 || n > 65535 || N < 1 || N > (1 << 23)) return SISSO_ERR_ARG;
    sisso_ctx c;
    c.stream = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    c.opts.device = dev;
    cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev);
    double *dZ = nullptr, *dy = nullptr, *dG = nullptr, *db = nullptr;
    float *dG32 = nullptr, *db32 = nullptr;
    void* sl = nullptr;
    int* ex = nullptr;
    sisso_status st = SISSO_OK;
    auto al = [&](void** p, size_t bytes) { if (!st) st = tmp_alloc(&c, p, bytes, "gram"); };
    al((void**)&dZ, sizeof(double) * (size_t)n * N);
    al((void**)&dy, sizeof(double) * (size_t)N);
    al((void**)&dG, sizeof(double) * (size_t)n * n);
    al((void**)&db, sizeof(double) * (size_t)n);
    al((void**)&dG32, sizeof(float) * (size_t)n * n);
    al((void**)&db32, sizeof(float) * (size_t)n);
    al(&sl, gram64_tc_bytes(N, n));
    al((void**)&ex, sizeof(int) * (size_t)n);
    if (!st) {
        cudaMemcpyAsync(dZ, Z, sizeof(double) * (size_t)n * N, cudaMemcpyDefault, c.stream);
        cudaMemcpyAsync(dy, yc, sizeof(double) * (size_t)N, cudaMemcpyDefault, c.stream);
        st = gram64_tc(&c, dZ, dy, N, 0, 0, n, n, n, sl, ex, dG, db, dG32, db32);
    }
    if (!st) {
        cudaMemcpyAsync(G, dG, sizeof(double) * (size_t)n * n, cudaMemcpyDeviceToHost, c.stream);
        cudaMemcpyAsync(b, db, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost, c.stream);
        st = check_cuda(&c, cudaStreamSynchronize(c.stream), "gram");
    }
    for (void* p : {(void*)dZ, (void*)dy, (void*)dG, (void*)db, (void*)dG32, (void*)db32, sl, (void*)ex})
        if (p) cudaFreeAsync(p, c.stream);
    return st;
}
