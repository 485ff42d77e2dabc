// l0_pair64.cuh — the exhaustive l0 search at D = 2 and 3 in FP64 throughout.
//
// Six FP64 operations a subset bound it: 3.6e7 subsets of 600 features are 0.5 ms of the FP64
// pipe.  The tiled FP32 sweep is not faster there (its units are too few to fill the SMs: 1.6 ms),
// and on strongly collinear subspaces, where FP32 leaves up to 70% of the subsets undecided, its
// FP64 confirmations took fifty times longer (2.5 ms for 2.2e5 subsets of 111 features).
//
// One CTA per first feature p (D = 3) and slice of rows i1; the reduced values of every feature
// x > p (r = G[p][x] / sqrt(G[p][p]), d = G[x][x] - r^2, n = b[x] - r w_p) and its row constants
// are tabulated in shared memory, then a warp takes a row and its lanes the columns x > i1:
//     g = G[i1][x] - r r',  t = g / d1,  d2 = d - g t,  num = n - t n1,
//     RSS / N = syy - w_p^2 - n1^2 / d1 - num^2 / d2
// A subset is dismissed when num^2 < K d2 with K = (RSS of {p, i1} - B - tie) / N less the bound of
// the solve's rounding, and d1, d2 >= 1e-6 (then num^2 < K d2 bounds the coefficient of x by
// 1e3 sqrt(K), and with it the coefficients' 1-norm by the row's s).  What is left goes to the
// same FP64 confirmation, band and tie rule as in the other forms.
#pragma once

#include "l0_tile.cuh"

namespace sg {
namespace {

constexpr double kPairPivot = 1e-6;
constexpr int kPairThreads = 256;

// per feature: reduced values, then its constants as a row
struct PairTab { double *r, *d, *n, *id, *nK; };       // 1/d1; -K before the threshold, in units of RSS / N

constexpr size_t kPair64Smem = (size_t)200 << 10;      // tables of up to 5120 features

__host__ __device__ constexpr size_t pair64_smem(int m) { return (size_t)m * 5 * sizeof(double); }

template <int D>
__global__ void __launch_bounds__(kPairThreads) k_l0_pair64(TileArgs A) {
    extern __shared__ __align__(16) unsigned char pair_smem[];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int p = D == 3 ? (int)blockIdx.x : -1, x0 = p + 1, m = A.n - x0;     // local feature x is x0 + x
    PairTab T;
    T.r = reinterpret_cast<double*>(pair_smem);
    T.d = T.r + m; T.n = T.d + m; T.id = T.n + m; T.nK = T.id + m;
    const double* G = A.G64;
    const double* b = A.b64;
    __shared__ double s_p[3];                                     // 1 / sqrt(G[p][p]) (0: singular), w_p
    if (tid == 0) {
        const double dp = D == 3 ? G[(size_t)p * A.ld64 + p] : 0.0;
        const double v = dp > kPivotMin + 1e-13 + 4e-15 * dp ? 1.0 / sqrt(dp) : 0.0;
        s_p[0] = v;
        s_p[1] = D == 3 ? b[p] * v : 0.0;
    }
    __syncthreads();
    const double inv = s_p[0], wp = s_p[1], base = A.syy64 - wp * wp;
    const bool okp = D == 2 || inv > 0.0;
    // the rounding bound needs no FP64: it is evaluated in FP32 and rounded up
    const float invf = (float)inv, vp = fabsf((float)wp * invf), ss = (float)A.sqrt_syy, c1 = 1.f + 3.1f * (float)(D + 1);
    for (int x = tid; x < m; x += kPairThreads) {
        const double r = D == 3 ? G[(size_t)p * A.ld64 + x0 + x] * inv : 0.0;
        const double d = G[(size_t)(x0 + x) * A.ld64 + x0 + x] - r * r, n = b[x0 + x] - r * wp;
        const bool ok = okp && d >= kPairPivot;
        const double id = ok ? 1.0 / d : 0.0, K0 = base - n * (n * id);
        // |gamma|_1 <= |p alone| + (1 + a1) |w1| + ((1 + a1) |g| / d1 + 1 + |x on p|) |num| / d2, with a1 and
        // |x on p| the coefficients on p, |g| <= sqrt(d1 d2'), d2' <= 1, |x on p| <= 1 / sqrt(G[p][p]) and
        // |num| / d2 <= sqrt(K / 1e-6)
        const float a1 = 1.f + fabsf((float)r * invf), idf = (float)id;
        const float s = vp + a1 * fabsf((float)n) * idf + (a1 * sqrtf(idf) + 1.f + invf) * 1e3f * sqrtf(fmaxf((float)K0, 0.f));
        const float err = 1.01f * 8.f * 1.1102230e-16f * (2.f * ss * s + c1 * s * s + (float)(D + 3) * 4.f * ss * ss);
        T.r[x] = r; T.d[x] = d; T.n[x] = n; T.id[x] = id;
        T.nK[x] = ok ? (double)err - K0 : INFINITY;
    }
    __syncthreads();
    const double inv_n = 1.0 / (double)A.N;
    double B = fmin((double)INFINITY, okey_inv(*(volatile unsigned long long*)A.ub_key));
    unsigned long long my_examined = 0, my_cand = 0;
    const int warps = kPairThreads / 32;
    for (int i1 = (int)blockIdx.y * warps + w; i1 < m - 1; i1 += (int)gridDim.y * warps) {
        const double ri = T.r[i1], id = T.id[i1], ni = T.n[i1];
        const double thr = B + A.tie64, nK = T.nK[i1] + thr * inv_n * (1.0 + 1e-15);
        const double* row = G + (size_t)(x0 + i1) * A.ld64 + x0;
        const unsigned long long next_key = *(volatile unsigned long long*)A.ub_key;
        for (int xb = i1 + 1; xb < m; xb += 32) {
            const int x = xb + lane;
            bool take = false;
            if (x < m) {
                const double g = D == 3 ? fma(-ri, T.r[x], row[x]) : row[x];
                const double t = g * id;
                const double d2 = fma(-g, t, T.d[x]), num = fma(-t, ni, T.n[x]);
                const double z = fma(nK, d2, num * num);
                // z < 0 and d2 >= 1e-6, on the high words (NaN is kept)
                const int zh = __double2hiint(z), dh = __double2hiint(d2);
                take = !(zh < 0 && (unsigned)zh < 0xfff00000u && dh >= __double2hiint(kPairPivot) + 1 && dh < 0x7ff00000);
            }
            if (!__any_sync(0xffffffffu, take)) continue;
            if (take) {
                int pos[D];
                if (D == 3) pos[0] = p;
                pos[D - 2] = x0 + i1;
                pos[D - 1] = x0 + x;
                ++my_cand;
                if (!clears64<D>(A.G64, A.b64, A.ld64, A.syy64, A.N, thr, pos)) {
                    const double r64 = rss64_fixed<D>(A.G64, A.b64, A.ld64, A.syy64, A.N, pos, nullptr);
                    if (r64 <= thr) {
                        add_band<D - 2>(A, pos, (float)r64);
                        if (r64 < B) { atomicMin(A.ub_key, okey(r64)); B = r64; }
                    }
                }
            }
            __syncwarp();
        }
        if (lane == 0) my_examined += (unsigned long long)(m - 1 - i1);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) B = fmin(B, __shfl_xor_sync(0xffffffffu, B, o));
        B = fmin(B, okey_inv(next_key));
    }
    my_examined = l0_warp_sum(my_examined);
    my_cand = l0_warp_sum(my_cand);
    if (lane == 0 && my_examined) {
        atomicAdd(A.examined, my_examined);
        atomicAdd(A.candidates, my_cand);
    }
}

}  // namespace
}  // namespace sg
