// fine_stencil.cuh -- parts shared by the kernels that apply the fine step's
// solve as a polynomial in the neighbour sum (fine_stencil.cu, fine_tiles.cu).
#pragma once

#include <cmath>

#include "fine.cuh"

namespace acpr {

// Coefficients of one call in the fields' precision.
template <typename T, int M>
struct Coef {
    T kappa, mdt;   // r = u + u (kappa + mdt u^2)
    T be0, b1;      // u' = r + be0 r + b1 T w_1
    T g[M];         // g[k], k = 0 .. M - 2: stage k, w = r + g[k] T (input)
    T a, dt;        // adjoint: lambda' = a mu + dt f'(u) (mu - mean)
};

template <typename T, int M>
Coef<T, M> make_coef(double a, double dt, const SolvePoly& p) {
    Coef<T, M> c{};
    c.kappa = T((a - 1.0) + dt);
    c.mdt = T(-dt);
    c.be0 = T(p.b[0] - 1.0);
    c.b1 = T(p.b[1]);
    // stage k applies the ratio of the coefficients M - k and M - k - 1
    for (int k = 0; k + 1 < M; ++k) {
        const double hi = p.b[M - k], lo = p.b[M - k - 1];
        c.g[k] = std::fabs(lo) > 1e-200 ? T(hi / lo) : T(0);
    }
    c.a = T(a);
    c.dt = T(dt);
    return c;
}

// A row in shared memory, a warp's lanes holding W adjacent columns each.
template <int W>
__device__ __forceinline__ void row_store(float* dst, const float (&x)[W], int lane) {
    // chunks of VW floats, chunk-major: lanes store consecutive vectors
    constexpr int VW = W % 4 == 0 ? 4 : W % 2 == 0 ? 2 : 1;
#pragma unroll
    for (int v = 0; v < W / VW; ++v) {
        float* p = dst + v * 32 * VW + lane * VW;
        if constexpr (VW == 4) *reinterpret_cast<float4*>(p) = make_float4(x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]);
        else if constexpr (VW == 2) *reinterpret_cast<float2*>(p) = make_float2(x[2 * v], x[2 * v + 1]);
        else *p = x[v];
    }
}
template <int W>
__device__ __forceinline__ void row_load(const float* src, float (&x)[W], int lane) {
    constexpr int VW = W % 4 == 0 ? 4 : W % 2 == 0 ? 2 : 1;
#pragma unroll
    for (int v = 0; v < W / VW; ++v) {
        const float* p = src + v * 32 * VW + lane * VW;
        if constexpr (VW == 4) {
            const float4 q = *reinterpret_cast<const float4*>(p);
            x[4 * v] = q.x; x[4 * v + 1] = q.y; x[4 * v + 2] = q.z; x[4 * v + 3] = q.w;
        } else if constexpr (VW == 2) {
            const float2 q = *reinterpret_cast<const float2*>(p);
            x[2 * v] = q.x; x[2 * v + 1] = q.y;
        } else {
            x[v] = *p;
        }
    }
}
// Left plus right neighbour of every column of a row.
template <int W>
__device__ __forceinline__ void hsum(const float (&x)[W], float (&h)[W], int lane) {
    const float l = __shfl_sync(0xffffffffu, x[W - 1], (lane + 31) & 31);
    const float r = __shfl_sync(0xffffffffu, x[0], (lane + 1) & 31);
#pragma unroll
    for (int c = 0; c < W; ++c) h[c] = (c ? x[c - 1] : l) + (c + 1 < W ? x[c + 1] : r);
}

// r <- p(Lap) r for the warp's H rows; halo(y, x) gives row y of r outside
// them (-M <= y < 0 or H <= y < H + M).  Rows stream through the M stages; a
// stage keeps its last row (p) and the three known neighbours of that row's
// cells (s), so T = ((left + right) + above) + below for every cell.
// SHIFT: plus `shift`, added to the small term: r + be0 r lies on the coarse
// grid of its binade, where a shift below half a unit would be rounded away in
// all of its cells alike.
template <int W, int H, int M, bool SHIFT, class Halo>
__device__ __forceinline__ void apply_poly(float (&r)[H][W], const Coef<float, M>& cf, int lane, float shift,
                                           Halo halo) {
    float s[M][W], p[M][W];
#pragma unroll
    for (int y = -M; y < H + M; ++y) {
        float x[W];
        if (y >= 0 && y < H) {
#pragma unroll
            for (int c = 0; c < W; ++c) x[c] = r[y][c];
        } else {
            halo(y, x);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const int yk = y - k, first = k - M;  // x is row yk of the stage's input, whose first row is `first`
            if (yk < first) break;
            float nx[W];
            const bool emit = yk >= first + 2;
            if (emit) {
                if (k < M - 1) {
                    float rr[W];
                    const int yr = yk - 1;
                    if (k == 0) {
#pragma unroll
                        for (int c = 0; c < W; ++c) rr[c] = p[0][c];
                    } else if (yr >= 0 && yr < H) {
#pragma unroll
                        for (int c = 0; c < W; ++c) rr[c] = r[yr][c];
                    } else {
                        halo(yr, rr);
                    }
#pragma unroll
                    for (int c = 0; c < W; ++c) nx[c] = fmaf(cf.g[k], s[k][c] + x[c], rr[c]);
                } else {
#pragma unroll
                    for (int c = 0; c < W; ++c) {
                        const float t0 = fmaf(cf.be0, r[yk - 1][c], r[yk - 1][c]);
                        r[yk - 1][c] = SHIFT ? t0 + fmaf(cf.b1, s[k][c] + x[c], shift) : fmaf(cf.b1, s[k][c] + x[c], t0);
                    }
                }
            }
            if (yk > first && yk < H + M - k - 1) {
                float h[W];
                hsum<W>(x, h, lane);
#pragma unroll
                for (int c = 0; c < W; ++c) s[k][c] = h[c] + p[k][c];
            }
#pragma unroll
            for (int c = 0; c < W; ++c) p[k][c] = x[c];
            if (!emit || k == M - 1) break;
#pragma unroll
            for (int c = 0; c < W; ++c) x[c] = nx[c];
        }
    }
}

constexpr float kFix = 16777216.f;  // 2^24: fixed point of the sums of r
constexpr long long kBadSum = (long long)(1ULL << 63);

// Sum over the warp's lanes of a 62-bit integer, on every lane.
__device__ __forceinline__ long long warp_sum_s64(long long v) {
    const int a0 = int(v & 0xfffff), a1 = int((v >> 20) & 0xfffff), a2 = int(v >> 40);
    return (long long)__reduce_add_sync(0xffffffffu, a0) + ((long long)__reduce_add_sync(0xffffffffu, a1) << 20) +
           ((long long)__reduce_add_sync(0xffffffffu, a2) << 40);
}

// Sum of the two rows' cells of a lane (the same order under every split).
template <int W>
__device__ __forceinline__ float pair_sum(const float (&x)[W], const float (&y)[W]) {
    float t[W];
#pragma unroll
    for (int c = 0; c < W; ++c) t[c] = x[c] + y[c];
#pragma unroll
    for (int o = W / 2; o > 0; o /= 2)
#pragma unroll
        for (int c = 0; c < o; ++c) t[c] += t[c + o];
    return t[0];
}

}  // namespace acpr
