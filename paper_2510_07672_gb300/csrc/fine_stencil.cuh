// fine_stencil.cuh -- parts shared by the kernels that apply the fine step's
// solve as a polynomial in the neighbour sum (fine_stencil.cu, fine_tiles.cu).
#pragma once

#include <cmath>
#include <type_traits>

#include "f32x2.cuh"
#include "fine.cuh"

namespace acpr {

// Coefficients of one call in the fields' precision.
template <typename T, int M>
struct Coef {
    T kappa, mdt;   // r = u + u (kappa + mdt u^2)
    T be0, b1;      // u' = r + be0 r + b1 T w_1
    T g[M];         // g[k], k = 0 .. M - 2: stage k, w = r + g[k] T (input)
    T a, dt;        // adjoint: lambda' = a mu + dt f'(u) (mu - mean)
    int run;        // steps between two measurements of the largest cell (mass model)
    double inv_sum;  // 1 / (a cells): sum of r -> mean of p(Lap) r (no division on the device: float64 is scarce)
};

template <typename T, int M>
Coef<T, M> make_coef(double a, double dt, double cells, const SolvePoly& p) {
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
    // A cell of size below one grows at most by (a + dt) / a a step, and a unit
    // serves two runs: 2^18 of the 2^19 that it leaves.
    c.run = int(std::fmin(64.0, std::fmax(4.0, 9.0 / std::log2((a + dt) / a))));
    c.inv_sum = 1.0 / (a * cells);
    return c;
}

// A lane's W adjacent columns of a row: pairs (column j, column j + W / 2) for
// even W, so that a column's neighbours are the adjacent pairs but at the ends
// and one paired instruction serves two cells; single columns for odd W.
template <int W>
struct Lane {
    static constexpr bool PAIR = W % 2 == 0;
    static constexpr int E = PAIR ? W / 2 : W;
    using V = std::conditional_t<PAIR, f32x2, float>;
};
template <int W>
using LaneV = typename Lane<W>::V;

__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ f32x2 vadd(f32x2 a, f32x2 b) { return f2_add(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ f32x2 vmul(f32x2 a, f32x2 b) { return f2_mul(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ f32x2 vfma(f32x2 a, f32x2 b, f32x2 c) { return f2_fma(a, b, c); }
template <typename V>
__device__ __forceinline__ V vset(float a) {
    if constexpr (sizeof(V) == 8) return f2(a, a);
    else return a;
}
__device__ __forceinline__ float lo_of(f32x2 v) {
    float a, b;
    f2split(v, a, b);
    return a;
}
__device__ __forceinline__ float hi_of(f32x2 v) {
    float a, b;
    f2split(v, a, b);
    return b;
}

// Columns in order <-> the lane's elements.
template <int W>
__device__ __forceinline__ void to_lane(const float (&c)[W], LaneV<W> (&x)[Lane<W>::E]) {
#pragma unroll
    for (int e = 0; e < Lane<W>::E; ++e) {
        if constexpr (Lane<W>::PAIR) x[e] = f2(c[e], c[e + W / 2]);
        else x[e] = c[e];
    }
}
template <int W>
__device__ __forceinline__ void from_lane(const LaneV<W> (&x)[Lane<W>::E], float (&c)[W]) {
#pragma unroll
    for (int e = 0; e < Lane<W>::E; ++e) {
        if constexpr (Lane<W>::PAIR) f2split(x[e], c[e], c[e + W / 2]);
        else c[e] = x[e];
    }
}

// A warp's row in shared memory, each lane's elements where only that lane
// looks for them: vectors of up to 16 bytes, consecutive over the lanes.
template <int W>
__device__ __forceinline__ void row_store(float* dst, const LaneV<W> (&x)[Lane<W>::E], int lane) {
    constexpr int E = Lane<W>::E;
    if constexpr (Lane<W>::PAIR && E % 2 == 0) {
#pragma unroll
        for (int v = 0; v < E / 2; ++v)
            reinterpret_cast<ulonglong2*>(dst)[v * 32 + lane] = make_ulonglong2(x[2 * v], x[2 * v + 1]);
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) reinterpret_cast<LaneV<W>*>(dst)[e * 32 + lane] = x[e];
    }
}
template <int W>
__device__ __forceinline__ void row_load(const float* src, LaneV<W> (&x)[Lane<W>::E], int lane) {
    constexpr int E = Lane<W>::E;
    if constexpr (Lane<W>::PAIR && E % 2 == 0) {
#pragma unroll
        for (int v = 0; v < E / 2; ++v) {
            const ulonglong2 q = reinterpret_cast<const ulonglong2*>(src)[v * 32 + lane];
            x[2 * v] = q.x;
            x[2 * v + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = reinterpret_cast<const LaneV<W>*>(src)[e * 32 + lane];
    }
}

// Left plus right neighbour of every column of a row; the neighbours of the
// run's ends are the next lanes' (the ring of lanes is the periodic row).
template <int W>
__device__ __forceinline__ void hsum(const LaneV<W> (&x)[Lane<W>::E], LaneV<W> (&h)[Lane<W>::E], int lane) {
    constexpr int E = Lane<W>::E;
    if constexpr (Lane<W>::PAIR) {
        const float l = __shfl_sync(0xffffffffu, hi_of(x[E - 1]), (lane + 31) & 31);
        const float r = __shfl_sync(0xffffffffu, lo_of(x[0]), (lane + 1) & 31);
        const f32x2 lv = f2(l, lo_of(x[E - 1])), rv = f2(hi_of(x[0]), r);
#pragma unroll
        for (int e = 0; e < E; ++e) h[e] = f2_add(e ? x[e - 1] : lv, e + 1 < E ? x[e + 1] : rv);
    } else {
        const float l = __shfl_sync(0xffffffffu, x[E - 1], (lane + 31) & 31);
        const float r = __shfl_sync(0xffffffffu, x[0], (lane + 1) & 31);
#pragma unroll
        for (int e = 0; e < E; ++e) h[e] = (e ? x[e - 1] : l) + (e + 1 < E ? x[e + 1] : r);
    }
}

// r = u + u (kappa + mdt u^2)
template <typename V>
__device__ __forceinline__ V rhs(V v, V mdt, V kappa) {
    return vfma(v, vfma(mdt, vmul(v, v), kappa), v);
}

// Bound of |r| over |u| <= m.
__device__ __forceinline__ float rhs_bound(float m, float mdt, float kappa) {
    return m * fmaxf(1.f + kappa, fabsf(fmaf(mdt, m * m, 1.f + kappa)));
}

// r <- p(Lap) r for the warp's H rows; halo(y, x) gives row y of r outside
// them (-M <= y < 0 or H <= y < H + M).  Rows stream through the M stages; a
// stage keeps its last row (p) and the three known neighbours of that row's
// cells (s), so T = ((left + right) + above) + below for every cell.
// SHIFT: plus `shift`, added to the small term: r + be0 r lies on the coarse
// grid of its binade, where a shift below half a unit would be rounded away in
// all of its cells alike.
// It is asked for (shift()) when the first row is complete.
template <int W, int H, int M, bool SHIFT, class Halo, class Shift>
__device__ __forceinline__ void apply_poly(LaneV<W> (&r)[H][Lane<W>::E], const Coef<float, M>& cf, int lane,
                                           Halo halo, Shift shift) {
    using V = LaneV<W>;
    constexpr int E = Lane<W>::E;
    V s[M][E], p[M][E];
    const V be0 = vset<V>(cf.be0), b1 = vset<V>(cf.b1);
    V sh = vset<V>(0.f);
#pragma unroll
    for (int y = -M; y < H + M; ++y) {
        V x[E];
        if (y >= 0 && y < H) {
#pragma unroll
            for (int c = 0; c < E; ++c) x[c] = r[y][c];
        } else {
            halo(y, x);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const int yk = y - k, first = k - M;  // x is row yk of the stage's input, whose first row is `first`
            if (yk < first) break;
            V nx[E];
            const bool emit = yk >= first + 2;
            if (emit) {
                if (k < M - 1) {
                    V rr[E];
                    const int yr = yk - 1;
                    if (k == 0) {
#pragma unroll
                        for (int c = 0; c < E; ++c) rr[c] = p[0][c];
                    } else if (yr >= 0 && yr < H) {
#pragma unroll
                        for (int c = 0; c < E; ++c) rr[c] = r[yr][c];
                    } else {
                        halo(yr, rr);
                    }
                    const V g = vset<V>(cf.g[k]);
#pragma unroll
                    for (int c = 0; c < E; ++c) nx[c] = vfma(g, vadd(s[k][c], x[c]), rr[c]);
                } else {
                    if (SHIFT && yk == 1) sh = vset<V>(shift());
#pragma unroll
                    for (int c = 0; c < E; ++c) {
                        const V t0 = vfma(be0, r[yk - 1][c], r[yk - 1][c]), t = vadd(s[k][c], x[c]);
                        r[yk - 1][c] = SHIFT ? vadd(t0, vfma(b1, t, sh)) : vfma(b1, t, t0);
                    }
                }
            }
            if (yk > first && yk < H + M - k - 1) {
                V h[E];
                hsum<W>(x, h, lane);
#pragma unroll
                for (int c = 0; c < E; ++c) s[k][c] = vadd(h[c], p[k][c]);
            }
#pragma unroll
            for (int c = 0; c < E; ++c) p[k][c] = x[c];
            if (!emit || k == M - 1) break;
#pragma unroll
            for (int c = 0; c < E; ++c) x[c] = nx[c];
        }
    }
}

// Sums of r in integers, exact up to the unit: any order and any split give the
// same bits.  The unit follows the field: a power of two 2^-scale such that the
// largest magnitude met, taken over the field at entry and every few steps, is
// below 2^room units, so a group's rounding is 2^-30 of that magnitude.  What is
// left of 62 bits is room for growth until the next measurement.
constexpr int kCellRoom = 40, kGroupRoom = 30;  // one cell of the entry sum; a group of cells of r
constexpr long long kBadSum = (long long)(1ULL << 63);
constexpr unsigned kAbsMask = 0x7fffffffu;

constexpr int log2i(int v) { return v > 1 ? 1 + log2i(v / 2) : 0; }
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }  // -126 <= k <= 127
__device__ __forceinline__ float pow2_inv(float p) { return __uint_as_float((254u << 23) - __float_as_uint(p)); }
// Scale by which every float of at most the magnitude `bits` (its bits without
// the sign) is below 2^room.
__device__ __forceinline__ int fix_scale(unsigned bits, int room) { return min(126, room + 126 - int(bits >> 23)); }

// Sum over the warp's lanes of a 62-bit integer, on every lane.
__device__ __forceinline__ long long warp_sum_s64(long long v) {
    const int a0 = int(v & 0xfffff), a1 = int((v >> 20) & 0xfffff), a2 = int(v >> 40);
    return (long long)__reduce_add_sync(0xffffffffu, a0) + ((long long)__reduce_add_sync(0xffffffffu, a1) << 20) +
           ((long long)__reduce_add_sync(0xffffffffu, a2) << 40);
}

// Sum of the two rows' cells of a lane (the same order under every split).
template <int W>
__device__ __forceinline__ float pair_sum(const LaneV<W> (&x)[Lane<W>::E], const LaneV<W> (&y)[Lane<W>::E]) {
    constexpr int E = Lane<W>::E;
    LaneV<W> t[E];
#pragma unroll
    for (int c = 0; c < E; ++c) t[c] = vadd(x[c], y[c]);
#pragma unroll
    for (int o = E / 2; o > 0; o /= 2)
#pragma unroll
        for (int c = 0; c < o; ++c) t[c] = vadd(t[c], t[c + o]);
    if constexpr (Lane<W>::PAIR) return lo_of(t[0]) + hi_of(t[0]);
    else return t[0];
}

}  // namespace acpr
