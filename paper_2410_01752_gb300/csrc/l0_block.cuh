// l0_block.cuh — the tiled l0 enumeration (l0_tile.cuh) for D = 4 and 5 with the prefix split in
// two: a CTA eliminates the first D - 3 features from the Gram once, in shared memory, and its
// warps sweep every (p, i1, i2) of the rest.
//
// k_l0_tile re-derives a prefix's reduced columns and rows in every warp's work unit; at D = 5 a
// prefix of three has on average only C(n, 5) / C(n, 3) = 4400 subsets at n = 300, and the unit's
// set-up and its short rows cost several times the sweep (1.4 warp instructions a subset, 0.25 in
// the sweep itself).  Here a work unit is a prefix of D - 3 features: the CTA forms
//     G'[x][y] = G[x][y] - sum R R   (y < x, packed strict lower triangle, shared memory)
// once for C(m, 3) subsets (m features to the right), and adding the next feature p needs one
// value per feature: r = G'[x][p] / sqrt(d'_p), dp = d' - r^2, np = n' - r w_p.  The warps take
// the p of a unit in turn and need no barrier.  Lanes are the rows i1 (their constants of the
// filter stay in registers); a column x > i1 costs two broadcast reads, three operations for its
// values and one row of G'.  The subset test is the filter of l0_tile.cuh with one fused
// multiply-add in the place of D - 2.
//
// The prefix is eliminated in FP64, its reduced features scaled to unit variance and then rounded
// to FP32, so that the FP32 error of a subset is relative to what the prefix leaves unexplained
// (syy' = syy - |w|^2 in the filter's e0 and e1, coefficients of the reduced features), not to the
// whole target.  The features are taken by their largest correlation with a feature of the greedy
// search: where a few features, or others that could stand in for them, reach the noise and every
// subset that holds them nearly ties, they are the prefix, and FP32 still tells those subsets
// apart (eliminated in FP32 and in the order of screening, up to 5.4e7 of the 1.96e10 subsets of
// such problems went to FP64 solves, which then took longer than the sweep).
// The sweep runs a shorter test that implies the filter (block_sweep_row) and only marks the
// columns it does not dismiss; they are decided after the sweep, so that no call stands between the
// row constants and their registers (with the calls inside, a third of the instructions were
// spills' and their operands').
// Measured at n = 300, D = 5 (1.96e10 subsets) over five problems: 20 to 25.5 ms (30 to 36 with the
// filter itself in the sweep, 43 and more by k_l0_tile); 0.6 warp instructions a subset at 56% of
// the issue slots.  Forms that took longer than k_l0_tile: lanes as columns with the row constants
// shuffled in (89 ms), and four warps sharing a p through a record table and a barrier (46 ms).
#pragma once

#include "l0_tile.cuh"

#include <type_traits>

namespace sg {
namespace {

// warps of a CTA (one p each at a time): sixteen and one CTA per SM while the triangle is large;
// up to kBSmallM features, four and four CTAs per SM, so that a unit's barriers hold up few warps
// (three quarters of the prefixes of n = 300 have that few features to the right)
constexpr int kBWarpsBig = 16, kBWarpsSmall = 4, kBSmallM = 150;
constexpr int kBRow = 6;                  // row groups of 32 swept together (their constants are 30 registers)
constexpr int kBQ = 64;                   // per-warp candidate queue
constexpr int kBMaxM = 320;               // features right of the CTA's prefix (204 KB triangle)

__host__ __device__ constexpr size_t block_smem_bytes(int m, int warps) {
    return sizeof(float) * ((size_t)m * (m - 1) / 2 + 36) + (sizeof(double2) + sizeof(float2)) * (size_t)m +
           sizeof(unsigned) * kBQ * warps;
}

// prefix of the CTA
struct BlockPre {
    int pre[2], last, ok;        // positions, the last of them; pivots usable
    double l10, inv[2], w[2];    // factor, 1 / diagonal, forward-solved moments
    float low;                   // the least pivot
    float base, e0, e1;          // syy' and the filter's errors at its scale
};

// the exact decision of one subset (feature positions ascending); returns the lane's new bound
template <int D>
__device__ __noinline__ double block_exact(const TileArgs& A, const int (&pos)[D], double B, double thr) {
    if (clears64<D>(A.G64, A.b64, A.ld64, A.syy64, A.N, thr, pos)) return B;
    const double r64 = rss64(A.G64, A.b64, A.ld64, A.syy64, A.N, D, pos, nullptr);
    if (!(r64 <= thr)) return B;
    add_band<D - 2>(A, pos, (float)r64);
    if (r64 < B) {
        atomicMin(A.ub_key, okey(r64));
        return r64;
    }
    return B;
}

// the warp's queued candidates (local positions p, i1, x in ten bits each), decided here or, with
// defer and while the list has room, left for k_l0_confirm: a p whose every extension nearly ties
// held one warp for milliseconds while the other SMs had nothing left to do (C(300, 4) with
// 22 000 candidates around one feature: 3.3 ms, 1.07 with the list, 0.5 where there are few)
template <int DC>
__device__ __noinline__ double block_flush(const TileArgs& A, const BlockPre* P, const unsigned* q, int qn, double B, bool defer) {
    const int lane = threadIdx.x & 31;
    const double thr = B + A.tie64;
    int64_t at = -1;
    if (defer) {
        if (lane == 0) at = (int64_t)atomicAdd(A.conf_count, (unsigned long long)qn);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (at + qn > A.conf_cap) {                               // full: the slots taken hold nothing
            for (int e = lane; e < qn; e += 32)
                if (at + e < A.conf_cap) A.conf[at + e] = ~0ull;
            at = -1;
        }
    }
    for (int e = lane; e < qn; e += 32) {
        const unsigned v = q[e];
        int pos[DC + 3];
#pragma unroll
        for (int m = 0; m < DC; ++m) pos[m] = A.perm[P->pre[m]];
        pos[DC] = A.perm[P->last + 1 + (int)(v & 1023u)];
        pos[DC + 1] = A.perm[P->last + 1 + (int)((v >> 10) & 1023u)];
        pos[DC + 2] = A.perm[P->last + 1 + (int)(v >> 20)];
#pragma unroll
        for (int i = 1; i < DC + 3; ++i)                      // ascending
#pragma unroll
            for (int j = i; j > 0; --j) {
                const int lo = min(pos[j - 1], pos[j]), hi = max(pos[j - 1], pos[j]);
                pos[j - 1] = lo;
                pos[j] = hi;
            }
        if (at >= 0) {
            uint64_t k = 0;
#pragma unroll
            for (int m = 0; m < DC + 3; ++m) k |= (uint64_t)pos[m] << (12 * m);
            A.conf[at + e] = k;
        } else {
            B = block_exact<DC + 3>(A, pos, B, thr);
        }
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) B = fmin(B, __shfl_xor_sync(0xffffffffu, B, o));
    return fmin(B, okey_inv(*(volatile unsigned long long*)A.ub_key));
}

// the deferred candidates, a thread each
template <int D>
__global__ void __launch_bounds__(128) k_l0_confirm(const __grid_constant__ TileArgs A) {
    const int64_t n = min((int64_t)*A.conf_count, A.conf_cap);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = A.conf[e];
        if (k == ~0ull) continue;
        int pos[D];
#pragma unroll
        for (int m = 0; m < D; ++m) pos[m] = (int)((k >> (12 * m)) & 4095u);
        const double B = fmin((double)INFINITY, okey_inv(*(volatile unsigned long long*)A.ub_key));    // (NaN: not set)
        block_exact<D>(A, pos, B, B + A.tie64);
    }
}

// the sweep's row constants of a lane, row groups j and j + 1 per register pair: -R[p][i1],
// -1/d1, -w1/sqrt(d1), -K2 and c (block_sweep_row)
struct RowsC { p2 nr[kBRow / 2], nid[kBRow / 2], nw[kBRow / 2], nK[kBRow / 2], c[kBRow / 2]; };

// the test of one subset: z < 0 and d2 > tau dismiss it
__device__ __forceinline__ void block_test(float gv, float r, float d, float n, float nr, float nid, float nw, float nK,
                                           float beta, float gamma, float& z, float& d2) {
    const float g = fmaf(nr, r, gv);
    d2 = fmaf(g * g, nid, d);
    const float num = fmaf(g, nw, n), n2 = num * num;
    z = fmaf(fmaf(beta, fabsf(num), fmaf(nK, d2, n2)), d2, gamma * n2);
}

// one column (r, d, n; gx its row of G' at this lane's rows) against C row groups with the sweep's
// test, num^2 - K2 d2 + c < 0: the largest value is folded into zmax.  dead: this lane's row of
// the last group is not left of x
template <int C>
__device__ __forceinline__ void block_col(const float* gx, float r, float d, float n, bool dead, const RowsC& R,
                                          float& zmax) {
    float gv[C];
#pragma unroll
    for (int j = 0; j < C; ++j) gv[j] = gx[32 * j];
    const p2 rx = pk2(r, r), dx = pk2(d, d), nx = pk2(n, n);
#pragma unroll
    for (int jp = 0; jp < C / 2; ++jp) {
        const p2 g = fma2(R.nr[jp], rx, pk2(gv[2 * jp], gv[2 * jp + 1]));
        const p2 d2 = fma2(mul2(g, g), R.nid[jp], dx);
        const p2 num = fma2(g, R.nw[jp], nx);
        float za, zb;
        up2(fma2(num, num, fma2(R.nK[jp], d2, R.c[jp])), za, zb);
        if (2 * jp + 1 == C - 1 && dead) zb = -INFINITY;
        zmax = fmaxf(fmaxf(zmax, za), zb);
    }
    if (C & 1) {
        constexpr int h = C / 2;
        float nr, nid, nw, nK, c, u;
        up2(R.nr[h], nr, u); up2(R.nid[h], nid, u); up2(R.nw[h], nw, u); up2(R.nK[h], nK, u); up2(R.c[h], c, u);
        const float g = fmaf(nr, r, gv[C - 1]), d2 = fmaf(g * g, nid, d), num = fmaf(g, nw, n);
        const float z = fmaf(num, num, fmaf(nK, d2, c));
        if (!dead) zmax = fmaxf(zmax, z);
    }
}

// one warp's p: the CTA's prefix plus p
struct BlockP {
    int p, m;
    bool ok;                     // pivots of the prefix and of p above tau
    float invd, w;               // 1 / sqrt(d'_p), w_p
    float A0, base, thrN;        // |w_p| / sqrt(d'_p), syy' - w_p^2, (B + tie) / N
    float e0, e1;                // the filter's errors at this prefix's scale
    float q2, rmax;              // largest |a2| and root of the largest dp
    int flushes;                 // full queues of this p (the first is decided at once, for its bound)
};
struct BlockRow { float r, d, n, l1; };      // R[p][x], dp, np, |coefficient on p|

__device__ __forceinline__ BlockRow block_feature(const BlockP& Q, const float* Gp, const float2* dn, int x) {
    const float r = Gp[x * (x - 1) / 2 + Q.p] * Q.invd;
    const float2 f = dn[x];
    return BlockRow{r, fmaf(-r, r, f.x), fmaf(-r, Q.w, f.y), fabsf(r * Q.invd)};
}

// the filter's constants of one row
struct RowC { float nr, nid, nw, nK, be, gm; };
__device__ __forceinline__ RowC block_row(const TileArgs& A, const BlockP& Q, const BlockRow& f) {
    const bool piv = Q.ok && f.d > A.tau;
    const float isd = __frsqrt_rn(f.d > 0.f ? f.d : 1.f), w1 = f.n * isd;
    const float S0 = 1.02f * (Q.A0 + (1.f + f.l1) * fabsf(w1) * isd);
    const float S1 = 1.02f * ((1.f + f.l1) * isd * Q.rmax * 1.0001f + 1.f + Q.q2);
    const float Kc = piv ? (Q.base - w1 * w1) - (Q.e0 + S0 * fmaf(A.e2, S0, Q.e1)) : -INFINITY;
    return RowC{-f.r, -(isd * isd), -(w1 * isd), Q.thrN - Kc, S1 * fmaf(2.f * A.e2, S0, Q.e1), A.e2 * S1 * S1};
}

// The sweep's test of the same row: six operations of two subsets each instead of ten and the
// smallest d2.  The filter dismisses a subset when
//     num^2 (d2 + gamma) + beta |num| d2 < K d2^2  and  d2 > tau,
// and with K > 0, t = max(gamma, tau) and d2 <= rmax^2 that follows from
//     num^2 + K t + beta sqrt(K) rmax < K d2:
// then num^2 < K d2, so gamma num^2 <= gamma K d2 and |num| < sqrt(K) rmax, and d2 > t.  Tested as
// num^2 - K2 d2 + c < 0 with room for the rounding of these expressions in K2 and c.  A column it
// does not dismiss is decided by the filter (block_take).
struct SweepC { float nK, c; };
__device__ __forceinline__ SweepC block_sweep_row(float tau, float rmax, const RowC& r) {
    const float K2 = -0.9999f * r.nK;
    const float c = 1.001f * (K2 * fmaxf(tau, r.gm) + r.be * sqrtf(fmaxf(K2, 0.f)) * rmax);
    return K2 > 0.f && c < INFINITY ? SweepC{-K2, c} : SweepC{0.f, 1.f};
}

struct BlockQueue { double B; int qn, taken; };

// a column some lane may keep: the decisions row group by row group, into the warp's queue
template <int DC>
__device__ __noinline__ BlockQueue block_take(const TileArgs& A, const BlockPre* P, BlockP& Q, const float* Gp,
                                              const float2* dn, int rb, int x, unsigned* q, int qn,
                                              double B) {
    const int lane = threadIdx.x & 31;
    int taken = 0;
    const BlockRow f = block_feature(Q, Gp, dn, x);
    const int end = min(x, rb + 32 * kBRow);            // the rows of this sweep
    for (int i = rb; i < end; i += 32) {
        const int i1 = i + lane;
        bool take = false;
        if (i1 < x) {
            const RowC c = block_row(A, Q, block_feature(Q, Gp, dn, i1));
            float z, d2;
            block_test(Gp[x * (x - 1) / 2 + i1], f.r, f.d, f.n, c.nr, c.nid, c.nw, c.nK, c.be, c.gm, z, d2);
            take = !((z < 0.f) & (d2 > A.tau));
        }
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        if (!mask) continue;
        if (take)
            q[qn + __popc(mask & ((1u << lane) - 1u))] = (unsigned)Q.p | ((unsigned)i1 << 10) | ((unsigned)x << 20);
        qn += __popc(mask);
        taken += __popc(mask);
        __syncwarp();
        if (qn >= 32) {
            B = block_flush<DC>(A, P, q, qn, B, Q.flushes > 0);
            qn = 0;
            if (lane == 0) ++Q.flushes;
            __syncwarp();
        }
    }
    return BlockQueue{B, qn, taken};
}

// the FP64 Gram and moments in the order of perm
__global__ void k_l0_reorder(const double* __restrict__ G, const double* __restrict__ b, int ld, int n,
                             const int* __restrict__ perm, double* __restrict__ Gq, double* __restrict__ bq) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
        const int i = e / n, j = e - i * n;
        Gq[e] = G[(size_t)perm[i] * ld + perm[j]];
        if (i == 0) bq[j] = b[perm[j]];
    }
}

// prefixes item0 .. of the colex order, M the most features right of one of them
template <int DC, int W>
__global__ void __launch_bounds__(W * 32, 16 / W) k_l0_block(const __grid_constant__ TileArgs A, int slices, int item0, int M) {
    extern __shared__ __align__(16) unsigned char block_smem[];
    __shared__ BlockPre P;
    __shared__ int s_item, s_p;
    __shared__ BlockP s_q[W];                                     // the warp's p, bound and subsets
    __shared__ double s_b[W];
    __shared__ unsigned long long s_seen[W];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    double2* rr = reinterpret_cast<double2*>(block_smem);         // R per feature (while the triangle is formed)
    float2* dn = reinterpret_cast<float2*>(rr + M);               // d', n' per feature; first its scale in .x
    float* Gp = reinterpret_cast<float*>(dn + M);                 // (x, y < x) at x (x - 1) / 2 + y
    unsigned* q = reinterpret_cast<unsigned*>(Gp + ((size_t)M * (M - 1) / 2 + 36)) + w * kBQ;
    const double inv_n = 1.0 / (double)A.N;
    if (lane == 0) {
        s_b[w] = fmin((double)INFINITY, okey_inv(*(volatile unsigned long long*)A.ub_key));
        s_seen[w] = 0;
    }
    __syncwarp();
    while (true) {
        __syncthreads();                                          // the last unit's buffers are free
        if (tid == 0) {
            s_item = item0 + atomicAdd(A.counter, 1);
            s_p = s_item % slices;
        }
        __syncthreads();
        const int item = s_item;
        if (item >= A.n_items) break;
        const int pre_rank = item / slices;
        if (tid == 0) {
            int pre[2] = {pre_rank, -1};
            if (DC == 2) {
                const int64_t m = colex_top2(pre_rank);
                pre[1] = (int)m;
                pre[0] = (int)(pre_rank - binom2(m));
            }
            P.last = pre[DC - 1];
            P.pre[0] = pre[0]; P.pre[1] = pre[1];
            const int f0 = pre[0], f1 = max(pre[1], 0);
            const double d0 = A.Gq[(size_t)f0 * A.n + f0];
            bool ok = d0 >= 1e-6;
            double low = d0;
            P.inv[0] = ok ? 1.0 / sqrt(d0) : 0.0;
            P.w[0] = A.bq[f0] * P.inv[0];
            P.l10 = 0.0; P.inv[1] = 0.0; P.w[1] = 0.0;
            if (DC == 2) {
                P.l10 = A.Gq[(size_t)f1 * A.n + f0] * P.inv[0];
                const double d1 = A.Gq[(size_t)f1 * A.n + f1] - P.l10 * P.l10;
                ok = ok && d1 >= 1e-6;
                low = fmin(low, d1);
                P.inv[1] = ok ? 1.0 / sqrt(d1) : 0.0;
                P.w[1] = (A.bq[f1] - P.l10 * P.w[0]) * P.inv[1];
            }
            const double s2 = A.syy64 - P.w[0] * P.w[0] - P.w[1] * P.w[1], share = s2 > 0.0 ? s2 / A.syy64 : 0.0;
            P.ok = ok && share > 1e-9;
            P.low = ok ? (float)low : 0.f;
            P.base = (float)s2;
            P.e0 = A.e0 * (float)share * 1.01f;
            P.e1 = A.e1 * (float)sqrt(share) * 1.01f;
        }
        __syncthreads();
        const int x0 = P.last + 1, m = A.n - x0;                  // local feature x is position x0 + x
        if (m < 3) continue;
        // ---- features right of the prefix, then the reduced triangle ---------------------
        const int q0 = P.pre[0], q1 = max(P.pre[1], 0);
        // FP64 leaves an error of about 2e-16 (r1^2 / d1 + 2 |r1| / sqrt(d1) + 2) in a reduced
        // variance h (d1 the second pivot, r1 the feature's value on it): h is resolved to FP32's
        // rounding where that is below 4e-8 h
        auto scale_of = [&](double h, double r1d) {
            const float r1 = fabsf((float)r1d), hf = (float)h;
            return P.ok && hf > 5e-9f * r1 * r1 / P.low + 1e-8f * r1 * rsqrtf(P.low) + 1e-8f ? rsqrtf(hf) : 0.f;
        };
        for (int x = tid; x < m; x += W * 32) {
            const int f = x0 + x;
            const double r0 = A.Gq[(size_t)q0 * A.n + f] * P.inv[0];
            const double r1 = DC == 2 ? (A.Gq[(size_t)q1 * A.n + f] - r0 * P.l10) * P.inv[1] : 0.0;
            rr[x] = make_double2(r0, r1);
            double h = A.Gq[(size_t)f * A.n + f] - r0 * r0;
            if (DC == 2) h -= r1 * r1;
            dn[x].x = scale_of(h, r1);
        }
        __syncthreads();
        for (int i = 1 + w; i < m; i += W) {
            const double2 ri = rr[i];
            const float si = dn[i].x;
            float* row = Gp + i * (i - 1) / 2;
            const double* src = A.Gq + (size_t)(x0 + i) * A.n + x0;
            for (int y = lane; y < i; y += 32) {
                const double2 ry = rr[y];
                double v = fma(-ri.x, ry.x, src[y]);
                if (DC == 2) v = fma(-ri.y, ry.y, v);
                row[y] = scaled_f32(v, 0) * (si * dn[y].x);
            }
        }
        __syncthreads();
        // variance (one to FP32 rounding; zero: unresolved, every subset kept) and moment
        for (int x = tid; x < m; x += W * 32) {
            const int f = x0 + x;
            const double2 r = rr[x];
            const float sc = dn[x].x;
            double h = A.Gq[(size_t)f * A.n + f] - r.x * r.x, n = A.bq[f] - r.x * P.w[0];
            if (DC == 2) { h -= r.y * r.y; n -= r.y * P.w[1]; }
            dn[x] = make_float2(sc > 0.f ? (float)h * sc * sc : 0.f, (float)n * sc);
        }
        __syncthreads();
        // ---- sweep: this warp's p ---------------------------------------------------------
        // (handed out largest triangle first: the warps finish together)
        int qn = 0;
        while (true) {
            int p = 0;
            if (lane == 0) p = atomicAdd(&s_p, slices);
            p = __shfl_sync(0xffffffffu, p, 0);
            if (p >= m - 2) break;
            const unsigned long long next_key = *(volatile unsigned long long*)A.ub_key;     // in flight
            BlockP Q;
            {
                const float2 f = dn[p];
                Q.p = p; Q.m = m; Q.flushes = 0;
                Q.ok = P.ok && f.x > A.tau;
                Q.invd = __frsqrt_rn(f.x > 0.f ? f.x : 1.f);
                Q.w = f.y * Q.invd;
                Q.A0 = fabsf(Q.w * Q.invd);
                Q.base = P.base - Q.w * Q.w;
                Q.e0 = P.e0; Q.e1 = P.e1;
                Q.thrN = __fmul_ru((float)((s_b[w] + A.tie64) * inv_n), 1.0000002f);
            }
            const float invd = Q.invd, wp = Q.w, tau = A.tau;
            float q2 = 0.f, dmax = 0.f;
            for (int x = p + 1 + lane; x < m; x += 32) {
                const BlockRow f = block_feature(Q, Gp, dn, x);
                q2 = fmaxf(q2, f.l1);
                dmax = fmaxf(dmax, f.d);
            }
            Q.q2 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(q2)));
            Q.rmax = sqrtf(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dmax))));
            __syncwarp();
            if (lane == 0) s_q[w] = Q;
            __syncwarp();
            // rows p + 1 .. m - 2, kBRow groups of 32 at a time: this lane's are i0 + 32 j
            for (int rb = p + 1; rb < m - 1; rb += 32 * kBRow) {
            const int i0 = rb + lane, groups = (m - 1 - rb + 31) >> 5;
            RowsC R;
#pragma unroll
            for (int jp = 0; jp < kBRow / 2; ++jp) {
                RowC c[2] = {{0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}};
                SweepC k[2] = {{0.f, 0.f}, {0.f, 0.f}};
                if (2 * jp < groups) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int i1 = i0 + 32 * (2 * jp + h);
                        if (i1 < m) {
                            c[h] = block_row(A, Q, block_feature(Q, Gp, dn, i1));
                            k[h] = block_sweep_row(tau, Q.rmax, c[h]);
                        }
                    }
                }
                R.nr[jp] = pk2(c[0].nr, c[1].nr); R.nid[jp] = pk2(c[0].nid, c[1].nid); R.nw[jp] = pk2(c[0].nw, c[1].nw);
                R.nK[jp] = pk2(k[0].nK, k[1].nK); R.c[jp] = pk2(k[0].c, k[1].c);
            }
            // columns to decide, one bit each: lane l holds those of rb + 1 + 32 l ..
            unsigned open = 0;
            // columns rb + 1 .. m - 1 in segments of equal row group count C, two at a time
            int x = rb + 1;
            const float* gx = Gp + x * (x - 1) / 2;               // row x of G'
            auto segment = [&](auto cc) {
                constexpr int C = decltype(cc)::value;
                const int end = C == kBRow ? m : min(m, rb + 1 + 32 * C);           // x - rb <= 32 C
                auto column = [&](const float* gr, int xc, float& zmax) {
                    const float r = gr[p] * invd;
                    const float2 f = dn[xc];
                    block_col<C>(gr + i0, r, fmaf(-r, r, f.x), fmaf(-r, wp, f.y), i0 + 32 * (C - 1) >= xc, R, zmax);
                };
                for (; x + 1 < end; x += 2) {                     // (an even number of columns from rb + 1: one word)
                    float zmax = -INFINITY;
                    column(gx, x, zmax);
                    column(gx + x, x + 1, zmax);
                    gx += 2 * x + 1;
                    if (__any_sync(0xffffffffu, !(zmax < 0.f)) && lane == ((x - rb - 1) >> 5)) open |= 3u << ((x - rb - 1) & 31);
                }
                if (x < end) {
                    float zmax = -INFINITY;
                    column(gx, x, zmax);
                    gx += x;
                    if (__any_sync(0xffffffffu, !(zmax < 0.f)) && lane == ((x - rb - 1) >> 5)) open |= 1u << ((x - rb - 1) & 31);
                    ++x;
                }
            };
            segment(std::integral_constant<int, 1>{});
            segment(std::integral_constant<int, 2>{});
            segment(std::integral_constant<int, 3>{});
            segment(std::integral_constant<int, 4>{});
            segment(std::integral_constant<int, 5>{});
            segment(std::integral_constant<int, 6>{});
            for (unsigned words = __ballot_sync(0xffffffffu, open != 0u); words; words &= words - 1u) {
                const int l = __ffs(words) - 1;
                for (unsigned o = __shfl_sync(0xffffffffu, open, l); o; o &= o - 1u) {
                    const BlockQueue t = block_take<DC>(A, &P, s_q[w], Gp, dn, rb, rb + 32 * l + __ffs(o), q, qn, s_b[w]);
                    qn = t.qn;
                    __syncwarp();
                    if (lane == 0) {
                        s_b[w] = t.B;
                        if (t.taken) atomicAdd(A.candidates, (unsigned long long)t.taken);
                    }
                    __syncwarp();
                }
            }
            }
            // rows p + 1 .. x - 1 of every column
            if (lane == 0) {
                s_seen[w] += (unsigned long long)(m - 1 - p) * (unsigned long long)(m - 2 - p) / 2;
                s_b[w] = fmin(s_b[w], okey_inv(next_key));
            }
            __syncwarp();
        }
        if (qn > 0) {                                      // the queue's entries are relative to this prefix
            const double B = block_flush<DC>(A, &P, q, qn, s_b[w], false);
            __syncwarp();
            if (lane == 0) s_b[w] = B;
        }
    }
    if (lane == 0) atomicAdd(A.examined, s_seen[w]);
}

}  // namespace
}  // namespace sg
