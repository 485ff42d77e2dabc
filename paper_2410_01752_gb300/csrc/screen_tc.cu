// screen_tc.cu — split 16-bit tcgen05 products with FP64 chunk sums (sisso_bilinear_tc): C = L R^T
// over the samples, each row scaled by a power of two and split into 16-bit parts (FP16: hi + lo,
// BF16: hi + mid + lo); the part products kept (FP16: hh, hl, lh; BF16: hh, hm, mh, hl, lh, mm)
// give every sum to about 2^-21 of its Cauchy-Schwarz scale.  A CTA computes one 128 x 128 tile
// over a chunk of 1024 samples (FP32 accumulation in TMEM) and stores it; chunks are added in FP64.
#include "tc_device.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <vector>

namespace sg {
namespace {

constexpr int BM = 128, BN = 128, BK = 64;            // output tile; samples per stage
constexpr int kThreads = 128;
constexpr uint32_t kTileBytes = BM * BK * 2;
constexpr int kAcc = 4;                                // TMEM accumulators per tile, 128 columns each
constexpr uint32_t kTmemCols = 128 * kAcc;
constexpr int kAccBlocks = 4;                          // 64-sample blocks summed in one accumulator
constexpr int kChunkBlocks = kAcc * kAccBlocks;        // 64-sample blocks per chunk (1024 samples)
constexpr int kMaxParts = 6;

// one stage = one 64-sample block: every 16-bit part of the L tile and of the R tile
// (FP16: 2 + 2 tiles, 64 KB, three stages; BF16: 3 + 3 tiles, 96 KB, two stages), so each
// part is loaded once per block and the block's part products are issued back to back
template <int NP>
struct Smem {
    static constexpr int ST = NP == 2 ? 3 : 2;
    uint8_t a[ST][NP][kTileBytes];
    uint8_t b[ST][NP][kTileBytes];
    uint64_t full[ST], empty[ST], done;
    uint32_t tmem_base;
};

struct BilinArgs {
    int tiles_m, tiles_n;        // output tiles of this product
    int chunks, kb_per_chunk;    // sample chunks (in 64-sample blocks) and their length
    int nkb;                     // 64-sample blocks in all
    int l_row0, r_row0;          // first row of the product within a part block
    int l_part_rows, r_part_rows;// rows of one part block (the stride between parts)
    int npairs;                  // part products summed
    int lp[kMaxParts], rp[kMaxParts];
    float* C;                    // C[chunk * chunk_stride + row * ldc + col]
    int ldc;
    size_t chunk_stride;
    int* err;
    uint32_t idesc;
};

// One 128 x 128 tile of one sample chunk: TMA producer (warp 0), MMA issuer (warp 1), all
// four warps store the tile (warp w: rows 32w..32w+31).  The tensor cores' FP32 accumulation
// loses up to about one unit in the last place per MMA, so every run of kAccBlocks blocks
// goes to its own TMEM accumulator and the accumulators are added in FP64 before the store.
// Bounded waits; on timeout the error flag is raised and nothing is stored.
template <int NP>
__global__ void __launch_bounds__(kThreads, 1) k_bilin_tc(const __grid_constant__ CUtensorMap mapL,
                                                          const __grid_constant__ CUtensorMap mapR, BilinArgs A) {
    using SM = Smem<NP>;
    constexpr int ST = SM::ST;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SM& S = *reinterpret_cast<SM*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per_chunk = A.tiles_m * A.tiles_n;
    const int chunk = blockIdx.x / per_chunk, t = blockIdx.x % per_chunk;
    const int tm = t / A.tiles_n, tn = t % A.tiles_n;
    const int kb_lo = chunk * A.kb_per_chunk, kb_hi = min(A.nkb, kb_lo + A.kb_per_chunk);
    const int nk = max(0, kb_hi - kb_lo);

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) { mbar_init(&S.full[s], 1); mbar_init(&S.empty[s], 1); }
        mbar_init(&S.done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = S.tmem_base;
    __shared__ int failed;
    if (threadIdx.x == 0) failed = 0;
    __syncthreads();

    float* out = A.C + (size_t)chunk * A.chunk_stride + (size_t)(tm * BM + warp * 32 + lane) * A.ldc + tn * BN;
    if (nk > 0) {
        if (warp == 0 && lane == 0) {
            int issued = 0;
            for (int ks = 0; ks < nk; ++ks) {
                const int s = ks % ST;
                const uint32_t ph = (uint32_t)(ks / ST) & 1u;
                if (ks >= ST && !mbar_wait(&S.empty[s], ph ^ 1u)) { failed = 1; break; }
                mbar_expect_tx(&S.full[s], 2 * NP * kTileBytes);
                const int x = (kb_lo + ks) * BK;
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    tma_load_2d(S.a[s][q], &mapL, x, q * A.l_part_rows + A.l_row0 + tm * BM, &S.full[s]);
                    tma_load_2d(S.b[s][q], &mapR, x, q * A.r_part_rows + A.r_row0 + tn * BN, &S.full[s]);
                }
                ++issued;
            }
            if (failed)
                for (int ks = (issued > ST ? issued - ST : 0); ks < issued; ++ks)
                    mbar_wait(&S.full[ks % ST], (uint32_t)(ks / ST) & 1u);
        } else if (warp == 1 && lane == 0) {
            bool ok = true;
            for (int ks = 0; ks < nk; ++ks) {
                const int s = ks % ST;
                if (!mbar_wait(&S.full[s], (uint32_t)(ks / ST) & 1u)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem + (uint32_t)((ks / kAccBlocks) * 128);
                const bool first = ks % kAccBlocks == 0;
                for (int p = 0; p < A.npairs; ++p) {
                    const uint64_t da = desc_sw128(smem_u32(S.a[s][A.lp[p]])), db = desc_sw128(smem_u32(S.b[s][A.rp[p]]));
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        mma_f16(acc, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), A.idesc,
                                (!first || p > 0 || k > 0) ? 1u : 0u);
                }
                mma_commit(&S.empty[s]);
            }
            if (!ok) failed = 1;
            mma_commit(&S.done);
        }
        __syncwarp();
        const bool ready = mbar_wait(&S.done, 0);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncthreads();
        if (!ready || failed) {
            if (threadIdx.x == 0) atomicExch(A.err, 1);
        } else {
            const int used = (kb_hi - kb_lo + kAccBlocks - 1) / kAccBlocks;
#pragma unroll 1
            for (int cb = 0; cb < BN / 32; ++cb) {
                double v[32];
#pragma unroll
                for (int q = 0; q < 32; ++q) v[q] = 0.0;
#pragma unroll 1
                for (int a = 0; a < used; ++a) {
                    uint32_t r[32];
                    tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(a * 128 + cb * 32), r);
#pragma unroll
                    for (int q = 0; q < 32; ++q) v[q] += (double)__uint_as_float(r[q]);
                }
                float4* dst = reinterpret_cast<float4*>(out + cb * 32);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    dst[q] = make_float4((float)v[4 * q], (float)v[4 * q + 1], (float)v[4 * q + 2], (float)v[4 * q + 3]);
            }
        }
    } else {
        float4* dst = reinterpret_cast<float4*>(out);
        for (int q = 0; q < BN / 4; ++q) dst[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// ---- 16-bit parts --------------------------------------------------------------------
// x (already scaled, rounded once to FP32) as NP 16-bit parts whose sum is x to about 2^-22
// (FP16: two parts of 11 bits) or 2^-24 (BF16: three parts of 8 bits); the residuals are
// exact in FP32
template <typename H> __device__ __forceinline__ H to_h(float v);
template <> __device__ __forceinline__ __half to_h<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 to_h<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
__device__ __forceinline__ float from_h(__half v) { return __half2float(v); }
__device__ __forceinline__ float from_h(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename H, int NP>
__device__ __forceinline__ void split_parts(double xd, H (&h)[NP]) {
    float x = (float)xd;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        h[p] = to_h<H>(x);
        x -= from_h(h[p]);
    }
}

template <typename H, int NP>
__device__ __forceinline__ void put_parts(const H (&h)[NP], H* dst, size_t part_stride) {
#pragma unroll
    for (int p = 0; p < NP; ++p) dst[(size_t)p * part_stride] = h[p];
}

template <typename H, int NP>
__device__ __forceinline__ void store_parts(double x, H* dst, size_t part_stride) {
    H h[NP];
    split_parts<H, NP>(x, h);
    put_parts<H, NP>(h, dst, part_stride);
}

// power-of-two exponent e with max * 2^e in [2^14, 2^15) (0 for max = 0)
__device__ __forceinline__ int scale_exp(double mx) {
    if (!(mx > 0.0) || !isfinite(mx)) return 0;
    int q;
    frexp(mx, &q);
    return 15 - q;
}

__device__ __forceinline__ double wmax(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// out[r][c] = sum over chunks of C (FP64, in chunk order), unscaled by the rows' exponents
__global__ void k_bilin_reduce(const float* __restrict__ C, int chunks, size_t chunk_stride, int rows, int cols, int ldc,
                               const int* __restrict__ eL, const int* __restrict__ eR, double* __restrict__ out,
                               int ldo) {
    const int64_t total = (int64_t)rows * cols;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / cols), c = (int)(e % cols);
        const float* p = C + (size_t)r * ldc + c;
        double s = 0.0;
        for (int q = 0; q < chunks; ++q) s += (double)p[(size_t)q * chunk_stride];
        out[(size_t)r * ldo + c] = ldexp(s, -(eL[r] + eR[c]));
    }
}

// rows (FP64, row stride N) -> NP parts of 16 bits, scaled per row (one warp per row)
template <typename H, int NP>
__global__ void k_rows_parts(const double* __restrict__ src, int rows, int N, int rows_pad, int Kpad, H* __restrict__ dst,
                             int* __restrict__ ex) {
    const int f = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (f >= rows_pad) return;
    const size_t K = (size_t)Kpad, ps = (size_t)rows_pad * K;
    double mx = 0.0;
    if (f < rows)
        for (int i = lane; i < N; i += 32) mx = fmax(mx, fabs(src[(size_t)f * N + i]));
    const int e = scale_exp(wmax(mx));
    const double s = ldexp(1.0, e);
    for (int i = lane; i < Kpad; i += 32)
        store_parts<H, NP>(f < rows && i < N ? src[(size_t)f * N + i] * s : 0.0, dst + (size_t)f * K + i, ps);
    if (lane == 0) ex[f] = e;
}

// ---- host -----------------------------------------------------------------------------
struct Parts {
    int n;
    int lp[kMaxParts], rp[kMaxParts];
};
Parts parts_of(bool bf16) {
    if (bf16) return Parts{6, {0, 0, 1, 0, 2, 1}, {0, 1, 0, 2, 0, 1}};
    return Parts{3, {0, 0, 1}, {0, 1, 0}};
}
int nparts(bool bf16) { return bf16 ? 3 : 2; }

bool encode_map(EncodeTiledFn enc, CUtensorMap* map, bool bf16, void* base, int rows, int Kpad) {
    const cuuint64_t gdim[2] = {(cuuint64_t)Kpad, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)Kpad * 2};
    const cuuint32_t box[2] = {BK, BM};
    const cuuint32_t estride[2] = {1, 1};
    return enc(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, gdim, gstride, box,
               estride, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int chunks_of(int nkb, int& per) {
    const int ch = std::max(1, (nkb + kChunkBlocks - 1) / kChunkBlocks);
    per = (nkb + ch - 1) / ch;
    return (nkb + per - 1) / per;
}

// C (m_rows x n_rows of the product, FP64 into out) = L[l_row0 ..] R[r_row0 ..]^T over the
// samples, both sides given as parts; out is unscaled by eL / eR (offset to the product's rows)
cudaError_t bilin(cudaStream_t s, int sms, bool bf16, void* L, int l_part_rows, int l_row0, int m_rows, void* R,
                  int r_part_rows, int r_row0, int n_rows, int Kpad, float* part, int* err, const int* eL,
                  const int* eR, double* out, int ldo, int& launches) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const int np = nparts(bf16);
    CUtensorMap mL, mR;
    if (!encode_map(enc, &mL, bf16, L, np * l_part_rows, Kpad) || !encode_map(enc, &mR, bf16, R, np * r_part_rows, Kpad))
        return cudaErrorInvalidValue;
    const Parts pp = parts_of(bf16);
    BilinArgs A{};
    A.tiles_m = m_rows / BM;
    A.tiles_n = n_rows / BN;
    A.nkb = Kpad / BK;
    A.chunks = chunks_of(A.nkb, A.kb_per_chunk);
    A.l_row0 = l_row0; A.r_row0 = r_row0;
    A.l_part_rows = l_part_rows; A.r_part_rows = r_part_rows;
    A.npairs = pp.n;
    for (int q = 0; q < pp.n; ++q) { A.lp[q] = pp.lp[q]; A.rp[q] = pp.rp[q]; }
    A.C = part;
    A.ldc = n_rows;
    A.chunk_stride = (size_t)m_rows * n_rows;
    A.err = err;
    A.idesc = idesc_f16(bf16 ? 1u : 0u, BM, BN);
    const unsigned grid = (unsigned)A.tiles_m * A.tiles_n * A.chunks;
    if (bf16) {
        const size_t smem = sizeof(Smem<3>) + 1024;
        cudaFuncSetAttribute(k_bilin_tc<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_bilin_tc<3><<<grid, kThreads, smem, s>>>(mL, mR, A);
    } else {
        const size_t smem = sizeof(Smem<2>) + 1024;
        cudaFuncSetAttribute(k_bilin_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_bilin_tc<2><<<grid, kThreads, smem, s>>>(mL, mR, A);
    }
    const int64_t total = (int64_t)m_rows * n_rows;
    k_bilin_reduce<<<(int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * 8, (total + 255) / 256)), 256, 0, s>>>(
        part, A.chunks, A.chunk_stride, m_rows, n_rows, n_rows, eL + l_row0, eR + r_row0, out, ldo);
    launches += 2;
    return cudaGetLastError();
}

}  // namespace
}  // namespace sg

// sum_s L[i][s] R[j][s] (FP64 in and out, host memory) through the split 16-bit tensor-core
// product
extern "C" sisso_status sisso_bilinear_tc(const double* Lrows, const double* Rrows, int m, int n, int N, int kind,
                                          double* out) {
    using namespace sg;
    if (!Lrows || !Rrows || !out || m < 1 || n < 1 || N < 1 ||
        (kind != SISSO_PREC_MIXED_BF16 && kind != SISSO_PREC_MIXED_FP16) || m > 65536 || n > 65536)
        return SISSO_ERR_ARG;
    const bool bf16 = kind == SISSO_PREC_MIXED_BF16;
    const int np = nparts(bf16);
    const int mp = (m + BM - 1) / BM * BM, npad = (n + BN - 1) / BN * BN, Kpad = (N + BK - 1) / BK * BK;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int per;
    const int ch = chunks_of(Kpad / BK, per);
    double *dL = nullptr, *dR = nullptr, *dout = nullptr;
    void *hL = nullptr, *hR = nullptr;
    int *eL = nullptr, *eR = nullptr, *err = nullptr;
    float* part = nullptr;
    cudaError_t e = cudaSuccess;
    auto ck = [&](cudaError_t x) { if (e == cudaSuccess && x != cudaSuccess) e = x; };
    ck(cudaMalloc((void**)&dL, sizeof(double) * (size_t)m * N));
    ck(cudaMalloc((void**)&dR, sizeof(double) * (size_t)n * N));
    ck(cudaMalloc(&hL, (size_t)np * mp * Kpad * 2));
    ck(cudaMalloc(&hR, (size_t)np * npad * Kpad * 2));
    ck(cudaMalloc((void**)&eL, sizeof(int) * mp));
    ck(cudaMalloc((void**)&eR, sizeof(int) * npad));
    ck(cudaMalloc((void**)&err, sizeof(int)));
    ck(cudaMalloc((void**)&part, sizeof(float) * (size_t)ch * mp * npad));
    ck(cudaMalloc((void**)&dout, sizeof(double) * (size_t)mp * npad));
    int h_err = 0, launches = 0;
    if (e == cudaSuccess) {
        ck(cudaMemcpy(dL, Lrows, sizeof(double) * (size_t)m * N, cudaMemcpyHostToDevice));
        ck(cudaMemcpy(dR, Rrows, sizeof(double) * (size_t)n * N, cudaMemcpyHostToDevice));
        ck(cudaMemset(err, 0, sizeof(int)));
        if (bf16) {
            k_rows_parts<__nv_bfloat16, 3><<<(mp * 32 + 255) / 256, 256>>>(dL, m, N, mp, Kpad, (__nv_bfloat16*)hL, eL);
            k_rows_parts<__nv_bfloat16, 3><<<(npad * 32 + 255) / 256, 256>>>(dR, n, N, npad, Kpad, (__nv_bfloat16*)hR, eR);
        } else {
            k_rows_parts<__half, 2><<<(mp * 32 + 255) / 256, 256>>>(dL, m, N, mp, Kpad, (__half*)hL, eL);
            k_rows_parts<__half, 2><<<(npad * 32 + 255) / 256, 256>>>(dR, n, N, npad, Kpad, (__half*)hR, eR);
        }
        ck(cudaGetLastError());
        if (e == cudaSuccess)
            ck(bilin(0, sms, bf16, hL, mp, 0, mp, hR, npad, 0, npad, Kpad, part, err, eL, eR, dout, npad, launches));
        ck(cudaDeviceSynchronize());
        if (e == cudaSuccess) {
            ck(cudaMemcpy(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost));
            ck(cudaMemcpy2D(out, sizeof(double) * n, dout, sizeof(double) * npad, sizeof(double) * n, m,
                            cudaMemcpyDeviceToHost));
        }
    }
    cudaFree(dL); cudaFree(dR); cudaFree(hL); cudaFree(hR); cudaFree(eL); cudaFree(eR); cudaFree(err);
    cudaFree(part); cudaFree(dout);
    if (e != cudaSuccess) return SISSO_ERR_CUDA;
    return h_err ? SISSO_ERR_TIMEOUT : SISSO_OK;
}
