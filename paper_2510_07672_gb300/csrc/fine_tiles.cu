// fine_tiles.cu -- the fine step by the polynomial solve of fine_stencil.cu
// (float32, degree 2) for fields that no cluster holds: 1024 x 1024 grids and
// the periodic cube.  The step is then local to a few cells, so a block takes a
// tile with the cells around it that its result depends on, and no data moves
// between blocks within a launch.
#include "fine_tiles.cuh"

#include <algorithm>

#include "fine_stencil.cuh"

namespace acpr {

namespace {

// Mass-conserving model: the shift of step n needs the sum of r^n over the
// whole field.  From n = 1 it is accumulated (fixed point, integer atomics: any
// order gives the same bits) by launch n - 1, which makes u^n, in a unit that
// follows the largest cell of the last r measured before it: r^0 at entry, then
// every kMeasure-th launch.  The sums of u^0 and r^0 are float64 partial sums
// of kSumParts blocks.  Words per field: sum of r that keeps the entry mean
// (float64), three rotating sums of r, a mark for cells out of range, two
// rotating largest cells of r (their bits without the sign), the partial sums.
constexpr int kSumParts = 24, kSumThreads = 512;
constexpr int kMeasure = 8;  // (a unit leaves 2^14 and serves 9 steps: 2.9-fold growth a step)
static_assert(7 + 2 * kSumParts <= kSumWords, "words of a field");
struct Sums {
    long long* w;  // [kSumWords][fields]
    int fields;
    __device__ __forceinline__ double* goal(int f) const { return reinterpret_cast<double*>(w + f); }
    __device__ __forceinline__ long long* slot(int n, int f) const { return w + (long long)(1 + n % 3) * fields + f; }
    __device__ __forceinline__ long long* bad(int f) const { return w + 4LL * fields + f; }
    // largest cell of r as launch l knows it
    __device__ __forceinline__ unsigned* top(int l, int f) const {
        return reinterpret_cast<unsigned*>(w + (long long)(5 + (l / kMeasure & 1)) * fields + f);
    }
    // partial sums of u (which = 0) and r^0 (1)
    __device__ __forceinline__ double* part(int which, int i, int f) const {
        return reinterpret_cast<double*>(w + (long long)(7 + which * kSumParts + i) * fields + f);
    }
};

__device__ __forceinline__ void add_s64(long long* p, long long v) {
    atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v);
}

// Adds a lane's sums (and its out-of-range mark) to the field's.
__device__ __forceinline__ void flush_sum(const Sums& s, long long* dst, int f, long long acc, bool bad, int lane) {
    acc = warp_sum_s64(acc);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
        if (bad) atomicExch(reinterpret_cast<unsigned long long*>(s.bad(f)), 1ULL);
        else add_s64(dst, acc);
    }
}
// The same of the largest magnitude (not that of a NaN, which the sums find).
__device__ __forceinline__ void flush_max(unsigned* dst, float m, int lane) {
    const unsigned bits = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if (lane == 0) atomicMax(dst, bits);
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// What launch l of the mass model works with, by one warp of a block (float64
// instructions are scarce).  One block of the field (`first`) also keeps the
// goal and clears the words that the next launches add to.
struct LaunchSums {
    float shift;  // puts the mean of u^(l+1) at the entry mean
    float unit;   // of the sum of r^(l+1)
};
__device__ __forceinline__ void launch_sums(LaunchSums* out, const Sums& s, int l, int f, const Coef<float, 2>& cf, double a,
                                            int room, int lane, bool first) {
    double gap;  // the sum that r should have, less the one it has
    if (l == 0) {
        const double u = warp_sum(lane < kSumParts ? *s.part(0, lane, f) : 0.0);
        const double r = warp_sum(lane < kSumParts ? *s.part(1, lane, f) : 0.0);
        gap = a * u - r;
        if (first && lane == 0) *s.goal(f) = a * u;
    } else {
        gap = *s.goal(f) - double(*s.slot(l, f)) * double(pow2_inv(pow2f(fix_scale(*s.top(l - 1, f), room))));
    }
    if (lane) return;
    out->shift = *s.bad(f) ? __int_as_float(0x7fffffff) : float(gap * cf.inv_sum);
    out->unit = pow2f(fix_scale(*s.top(l, f), room));
    if (first) {
        *s.slot(l + 2, f) = 0;
        if (l % kMeasure == kMeasure / 2) *s.top(l + kMeasure, f) = 0;
    }
}
__device__ __forceinline__ bool measures(int l) { return l % kMeasure == kMeasure - 1; }

// s + e <- s + e + v, the rounding of s + v kept in e (TwoSum, Knuth).
__device__ __forceinline__ void two_sum(f32x2& s, f32x2& e, f32x2 v) {
    const f32x2 neg = f2(-1.f, -1.f);
    const f32x2 t = f2_add(s, v), b = f2_fma(s, neg, t);
    e = f2_add(e, f2_add(f2_fma(f2_fma(b, neg, t), neg, s), f2_fma(b, neg, v)));
    s = t;
}

// Partial sums of u and of r^0, exact to 2^-48 of each thread's, and the
// largest cell of r^0; parts blocks a field (the words of the others stay zero);
// cells a multiple of 4.
__global__ void __launch_bounds__(kSumThreads) entry_sums_kernel(FieldMap src, long long cells, Sums s, int parts, float mdt,
                                                                  float kappa) {
    const int f = blockIdx.x / parts, part = blockIdx.x % parts;
    const float4* u = reinterpret_cast<const float4*>(src.at(f, cells));
    const f32x2 m2 = f2(mdt, mdt), k2 = f2(kappa, kappa);
    f32x2 su = f2(0.f, 0.f), eu = su, sr = su, er = su;
    float top = 0.f;
    for (long long i = part * (long long)kSumThreads + threadIdx.x; i < cells / 4; i += parts * kSumThreads) {
        const float4 q = u[i];
        const f32x2 v[2] = {f2(q.x, q.y), f2(q.z, q.w)};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const f32x2 r = rhs(v[c], m2, k2);
            two_sum(su, eu, v[c]);
            two_sum(sr, er, r);
            top = fmaxf(top, fmaxf(fabsf(lo_of(r)), fabsf(hi_of(r))));
        }
    }
    auto total = [](f32x2 a, f32x2 b) {
        return warp_sum((double(lo_of(a)) + double(lo_of(b))) + (double(hi_of(a)) + double(hi_of(b))));
    };
    const double tu = total(su, eu), tr = total(sr, er);
    __shared__ double red[2][kSumThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    flush_max(s.top(0, f), top, lane);
    if (lane == 0) {
        red[0][warp] = tu;
        red[1][warp] = tr;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kSumThreads / 32; ++w) t += red[threadIdx.x][w];
        *s.part(threadIdx.x, part, f) = t;
    }
}

int entry_sums(const FieldMap& src, long long cells, const Sums& sums, const Coef<float, 2>& cf, cudaStream_t st) {
    ACPR_CUDA(cudaMemsetAsync(sums.w, 0, sizeof(long long) * kSumWords * sums.fields, st));
    // four vectors a thread or more: 32^3 takes 4 blocks
    const int parts = int(std::min<long long>(kSumParts, std::max<long long>(1, cells / (16 * kSumThreads))));
    entry_sums_kernel<<<unsigned(sums.fields) * parts, kSumThreads, 0, st>>>(src, cells, sums, parts, cf.mdt, cf.kappa);
    ACPR_LAUNCH_CHECK();
    return AC_OK;
}

// ------------------------------------------------------------ 1024 x 1024 --
// A block of 16 warps holds a tile of 144 x 256 cells in registers (a lane 9
// rows of 8 columns) and runs up to 4 steps on it, two rows and columns of the
// rim going stale per step; the inner 128 x 208 cells are stored (8 x 5 tiles,
// the last column of tiles cut; 71% of the computed cells): 4 steps cost one read and one write of the field where the
// Fourier passes moved 16 bytes a cell and step.  The mass model needs the
// field's sum each step and runs one step per launch.
// Bound: FP32 issue.  us a step, 32 fields: two Fourier passes 213, tiles 34.5 (scalar
// arithmetic on 7 columns a lane 48); mass-conserving 79 (one step a launch).
constexpr int kTW = 8, kTH = 9, kTWarps = 16, kRim = 8, kTSteps = 4;
constexpr int kTCols = 32 * kTW, kTRows = kTWarps * kTH;
constexpr int kBig = 1024;
constexpr int kTRoom = kGroupRoom - log2i(kTW);  // of a cell of r, in groups of a lane's row
constexpr int kTValidC = 208, kTValidR = kTRows - 2 * kRim;
constexpr int kTilesX = (kBig + kTValidC - 1) / kTValidC, kTilesY = kBig / kTValidR;
constexpr size_t kTileSmem = size_t(2) * 2 * kTWarps * 2 * kTCols * sizeof(float);
static_assert(kBig % kTValidR == 0 && kRim >= 2 * kTSteps && kTValidC + 2 * kRim <= kTCols && kTValidC % kTW == 0 && kRim % kTW == 0,
              "tiling");

template <bool MASS>
__global__ void __launch_bounds__(kTWarps * 32, 1) big_tile_kernel(FieldMap src, FieldMap dst, int steps,
                                                                   const __grid_constant__ Coef<float, 2> cf, Sums sums,
                                                                   int n_step, int last, double a) {
    constexpr int M = 2, E = Lane<kTW>::E;
    using V = LaneV<kTW>;
    constexpr long long NN = (long long)kBig * kBig;
    extern __shared__ __align__(16) float halo[];  // [buffer][0: above, 1: below][warp][M][kTCols]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int f = blockIdx.x / (kTilesX * kTilesY), tile = blockIdx.x % (kTilesX * kTilesY);
    const int tx = tile % kTilesX, ty = tile / kTilesX;
    const int row0 = ty * kTValidR - kRim + warp * kTH, col0 = tx * kTValidC - kRim + lane * kTW;
    const float* in = src.at(f, NN) + (col0 & (kBig - 1));
    V u[kTH][E];
#pragma unroll
    for (int y = 0; y < kTH; ++y) {
        const float4* p = reinterpret_cast<const float4*>(in + ((row0 + y) & (kBig - 1)) * kBig);
        const float4 q0 = p[0], q1 = p[1];
        const float c[kTW] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
        to_lane<kTW>(c, u[y]);
    }
    constexpr int BUF = 2 * kTWarps * M * kTCols;
    // the tile's first and last rows have no neighbour: they hand their rows to
    // a slot nobody needs, and read stale ones (their cells are rim)
    float* up = halo + (kTWarps + (warp > 0 ? warp - 1 : kTWarps - 1)) * M * kTCols;
    float* down = halo + (warp < kTWarps - 1 ? warp + 1 : 0) * M * kTCols;
    const float* above = halo + warp * M * kTCols;
    const float* below = halo + (kTWarps + warp) * M * kTCols;
    const V mdt = vset<V>(cf.mdt), kappa = vset<V>(cf.kappa);
    __shared__ LaunchSums now;
    if (MASS && warp == 0) launch_sums(&now, sums, n_step, f, cf, a, kTRoom, lane, tile == 0);
    for (int s = 0; s < steps; ++s) {
        const int buf = s & 1;
        if (!MASS || n_step == 0) {  // the mass model's launches hand on r
#pragma unroll
            for (int y = 0; y < kTH; ++y)
#pragma unroll
                for (int c = 0; c < E; ++c) u[y][c] = rhs(u[y][c], mdt, kappa);
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            row_store<kTW>(up + buf * BUF + m * kTCols, u[m], lane);
            row_store<kTW>(down + buf * BUF + m * kTCols, u[kTH - M + m], lane);
        }
        __syncthreads();
        apply_poly<kTW, kTH, M, MASS>(
            u, cf, lane,
            [&](int y, V(&x)[E]) {
                row_load<kTW>((y < 0 ? above + (y + M) * kTCols : below + (y - kTH) * kTCols) + buf * BUF, x, lane);
            },
            [&] { return now.shift; });  // written before the step's barrier
    }
    float* out = dst.at(f, NN) + col0;
    // whole lanes are rim or stored
    const bool keep = lane * kTW >= kRim && lane * kTW < kRim + kTValidC && col0 < kBig;
    long long acc = 0;
    bool bad = false;
    float top = 0.f;
#pragma unroll
    for (int y = 0; y < kTH; ++y) {
        const int lr = warp * kTH + y;
        if (lr < kRim || lr >= kRim + kTValidR || !keep) continue;
        if (MASS && !last) {
#pragma unroll
            for (int e = 0; e < E; ++e) u[y][e] = rhs(u[y][e], mdt, kappa);
        }
        float c[kTW];
        from_lane<kTW>(u[y], c);
        float4* p = reinterpret_cast<float4*>(out + (row0 + y) * kBig);
        p[0] = make_float4(c[0], c[1], c[2], c[3]);
        p[1] = make_float4(c[4], c[5], c[6], c[7]);
        if constexpr (MASS) {
            // a balanced tree: equal cells, a flat phase, add up exactly
            const V t2 = vadd(vadd(u[y][0], u[y][1]), vadd(u[y][2], u[y][3]));
            const float t = (lo_of(t2) + hi_of(t2)) * now.unit;
            acc += __float2ll_rn(t);
            bad |= !(fabsf(t) < 0x1p45f);  // 2^17 such sums stay below 2^62
            if (measures(n_step)) {
#pragma unroll
                for (int e = 0; e < kTW; ++e) top = fmaxf(top, fabsf(c[e]));
            }
        }
    }
    if (MASS && !last) {
        flush_sum(sums, sums.slot(n_step + 1, f), f, acc, bad, lane);
        if (measures(n_step)) flush_max(sums.top(n_step + 1, f), top, lane);
    }
}

// ------------------------------------------------------------------- cube --
// A block streams the planes i of a chunk through a strip of 36 rows (12 warps
// of 3 rows at N = 128, 9 of 4 below; a lane N / 32 columns of each; 32 rows are stored) of all N columns, as
// apply_poly streams rows: r(i) completes w(i - 1), w(i - 1) completes
// u'(i - 2).  One barrier per plane hands the warps' edge rows of r and w to
// the warps above and below.  A step reads and writes the fields once (the
// five Fourier passes: 40 bytes a cell).  Bound: the latency of a plane
// (loads, barrier, exchange), 4 TB/s of HBM traffic beside it.  us a step, mass / classic:
// 16 fields of 128^3  Fourier passes 372, streamed 86 / 75 (2 rows a warp 107 / 65, 4 rows 121 / 102; handing on r
// instead of u 103 / 93); 48 fields of 64^3 42 / 33.
constexpr int kCRows = 36, kCValid = kCRows - 4;
constexpr int kCRoom = kGroupRoom - 5;  // of a cell of r, in groups of up to 32
template <int N>
struct CubeShape {  // rows a warp, warps, CTAs per SM
    static constexpr int H = N == 128 ? 3 : 4, WARPS = kCRows / H, MINB = N == 128 ? 1 : 2;
};

template <int N, bool MASS>
__global__ void __launch_bounds__(CubeShape<N>::WARPS * 32, CubeShape<N>::MINB) cube_kernel(const float* __restrict__ u, float* __restrict__ uo,
                                                               int planes, const __grid_constant__ Coef<float, 2> cf,
                                                               Sums sums, int n_step, int last_step, double a) {
    constexpr int W = N / 32, E = Lane<W>::E, kCH = CubeShape<N>::H, kCWarps = CubeShape<N>::WARPS;
    using V = LaneV<W>;
    constexpr long long NN = (long long)N * N, NNN = NN * N;
    __shared__ __align__(16) float edge[2][2][2][kCWarps][N];  // [buffer][r, w][first, last row][warp]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int strips = N / kCValid;
    const int strip = blockIdx.x % strips, chunk = blockIdx.x / strips % (N / planes), f = blockIdx.x / (strips * (N / planes));
    const int i0 = chunk * planes, j0 = strip * kCValid - 2 + warp * kCH;
    const float* in = u + f * NNN;
    float* out = uo + f * NNN;
    __shared__ LaunchSums now;
    if constexpr (MASS) {
        if (warp == 0) launch_sums(&now, sums, n_step, f, cf, a, kCRoom, lane, strip == 0 && chunk == 0);
        __syncthreads();
    }
    const int up = warp > 0 ? warp - 1 : kCWarps - 1, down = warp < kCWarps - 1 ? warp + 1 : 0;
    auto load_plane = [&](int i, V(&x)[kCH][E]) {
        const float* p = in + (long long)((i + N) & (N - 1)) * NN + lane * W;
#pragma unroll
        for (int y = 0; y < kCH; ++y) {
            const float* q = p + ((j0 + y) & (N - 1)) * N;
            float c[W];
            if constexpr (W == 4) {
                const float4 v = *reinterpret_cast<const float4*>(q);
                c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
            } else if constexpr (W == 2) {
                const float2 v = *reinterpret_cast<const float2*>(q);
                c[0] = v.x; c[1] = v.y;
            } else {
                c[0] = *q;
            }
            to_lane<W>(c, x[y]);
        }
    };
    const V be0 = vset<V>(cf.be0), b1 = vset<V>(cf.b1), g = vset<V>(cf.g[0]), sh = vset<V>(MASS ? now.shift : 0.f);
    const V mdt = vset<V>(cf.mdt), kappa = vset<V>(cf.kappa);
    // rp, rq: r(i - 1), r(i - 2); s0: the five known neighbours of r(i - 1);
    // wp: w(i - 2); s1: the five known neighbours of w(i - 2)
    V even[kCH][E], odd[kCH][E], rp[kCH][E], rq[kCH][E], s0[kCH][E], wp[kCH][E], s1[kCH][E];
#pragma unroll
    for (int y = 0; y < kCH; ++y)
#pragma unroll
        for (int c = 0; c < E; ++c) rp[y][c] = rq[y][c] = s0[y][c] = wp[y][c] = s1[y][c] = vset<V>(0.f);
    load_plane(i0 - 2, even);
    load_plane(i0 - 1, odd);
    long long acc = 0;
    bool bad = false;
    float top = 0.f;
    // the next step's r over four planes (two of four rows), rows in balanced trees (equal cells, a
    // flat phase, add up exactly; one after another they all round alike, which
    // moved the mean by up to 4e-7 a call)
    V part[2][2];
    auto add_group = [&](V p) {
        float t;
        if constexpr (Lane<W>::PAIR) t = lo_of(p) + hi_of(p);
        else t = p;
        t *= now.unit;
        acc += __float2ll_rn(t);
        bad |= !(fabsf(t) < 0x1p44f);  // 2^17 such sums stay below 2^61
    };
    const bool last = n_step == last_step;
    // plane k from `nxt`, which then receives plane k + 2 (two sets in turn:
    // 47 / 33 us against 50 / 37 with a copy, 48 x 64^3)
    auto plane = [&](int k, int buf, V(&nxt)[kCH][E]) {
        V r[kCH][E], w[kCH][E];
#pragma unroll
        for (int y = 0; y < kCH; ++y)
#pragma unroll
            for (int c = 0; c < E; ++c) {
                r[y][c] = rhs(nxt[y][c], mdt, kappa);
                w[y][c] = vfma(g, vadd(s0[y][c], r[y][c]), rp[y][c]);  // w(k - 1)
            }
        if (k < planes) load_plane(i0 + k + 2, nxt);
        if (k >= 2) {
            float* p = out + (long long)(i0 + k - 2) * NN + lane * W;
            V rows[kCH];
#pragma unroll
            for (int y = 0; y < kCH; ++y) rows[y] = vset<V>(0.f);
#pragma unroll
            for (int y = 0; y < kCH; ++y) {
                V o[E];
#pragma unroll
                for (int c = 0; c < E; ++c) {
                    const V t = vadd(s1[y][c], w[y][c]), t0 = vfma(be0, rq[y][c], rq[y][c]);
                    o[c] = MASS ? vadd(t0, vfma(b1, t, sh)) : vfma(b1, t, t0);
                }
                float v[W];
                from_lane<W>(o, v);
                const int lr = warp * kCH + y;
                if (lr < 2 || lr >= 2 + kCValid) continue;
                float* q = p + (j0 + y) * N;
                if constexpr (W == 4) *reinterpret_cast<float4*>(q) = make_float4(v[0], v[1], v[2], v[3]);
                else if constexpr (W == 2) *reinterpret_cast<float2*>(q) = make_float2(v[0], v[1]);
                else *q = v[0];
                if constexpr (MASS) {
                    V rn[E];
#pragma unroll
                    for (int c = 0; c < E; ++c) rn[c] = rhs(o[c], mdt, kappa);
                    rows[y] = E == 2 ? vadd(rn[0], rn[E - 1]) : rn[0];
                }
            }
            if constexpr (MASS) {
                if constexpr (kCH == 3) {
                    const V g[2] = {vadd(rows[0], rows[1]), rows[2]};
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if ((k & 2) != 0) part[0][i] = buf ? vadd(part[0][i], g[i]) : g[i];  // (the first planes are k = 2, 3)
                        else if (buf == 0) part[1][i] = g[i];
                        else add_group(vadd(part[0][i], vadd(part[1][i], g[i])));
                    }
                } else {
                    const V g = vadd(vadd(rows[0], rows[1]), vadd(rows[2], rows[kCH - 1]));
                    if (buf == 0) part[0][0] = g;
                    else add_group(vadd(part[0][0], g));
                }
            }
        }
        if (MASS && measures(n_step)) {  // (of this step's r: the planes' ends part the instructions anyway)
#pragma unroll
            for (int y = 0; y < kCH; ++y) {
                float m[W];
                from_lane<W>(r[y], m);
#pragma unroll
                for (int c = 0; c < W; ++c) top = fmaxf(top, fabsf(m[c]));
            }
        }
        row_store<W>(edge[buf][0][0][warp], r[0], lane);
        row_store<W>(edge[buf][0][1][warp], r[kCH - 1], lane);
        row_store<W>(edge[buf][1][0][warp], w[0], lane);
        row_store<W>(edge[buf][1][1][warp], w[kCH - 1], lane);
        __syncthreads();
        // s = (((left + right) + above) + below) + the plane before
        auto neighbours = [&](const V(&x)[kCH][E], int which, const V(&prev)[kCH][E], V(&s)[kCH][E]) {
            V ab[E], be[E];
            row_load<W>(edge[buf][which][1][up], ab, lane);
            row_load<W>(edge[buf][which][0][down], be, lane);
#pragma unroll
            for (int y = 0; y < kCH; ++y) {
                V h[E];
                hsum<W>(x[y], h, lane);
#pragma unroll
                for (int c = 0; c < E; ++c)
                    s[y][c] = vadd(vadd(vadd(h[c], y ? x[y - 1][c] : ab[c]), y + 1 < kCH ? x[y + 1][c] : be[c]), prev[y][c]);
            }
        };
        neighbours(r, 0, rp, s0);
        neighbours(w, 1, wp, s1);
#pragma unroll
        for (int y = 0; y < kCH; ++y)
#pragma unroll
            for (int c = 0; c < E; ++c) {
                rq[y][c] = rp[y][c];
                rp[y][c] = r[y][c];
                wp[y][c] = w[y][c];
            }
    };
    for (int k = -2; k < planes + 2; k += 2) {  // (planes is even)
        plane(k, 0, even);
        plane(k + 1, 1, odd);
    }
    if (MASS && !last) {
        flush_sum(sums, sums.slot(n_step + 1, f), f, acc, bad, lane);
        if (measures(n_step)) flush_max(sums.top(n_step + 1, f), top, lane);
    }
}

template <int N>
int cube_steps(const SolvePoly& poly, double a, double dt, int mass, int steps, int fields, const float* u_in,
               float* u_out, float* tmp, Sums sums, cudaStream_t st) {
    constexpr long long NNN = (long long)N * N * N;
    const Coef<float, 2> cf = make_coef<float, 2>(a, dt, double(NNN), poly);
    if (mass) {
        FieldMap src{};
        src.base = const_cast<float*>(u_in);
        src.per_group = fields;
        const int rc = entry_sums(src, NNN, sums, cf, st);
        if (rc) return rc;
    }
    // the last step writes u_out, the ones before alternate with tmp; a first
    // step that writes u_out may not read cells there
    const float* cur = u_in;
    const uintptr_t from = reinterpret_cast<uintptr_t>(u_in), to = reinterpret_cast<uintptr_t>(u_out);
    if ((from > to ? from - to : to - from) < sizeof(float) * NNN * fields && steps % 2) {
        ACPR_CUDA(cudaMemcpyAsync(tmp, u_in, sizeof(float) * NNN * fields, cudaMemcpyDeviceToDevice, st));
        cur = tmp;
    }
    // planes per block: long chunks repeat fewer planes (4 each), short ones
    // fill the SMs; the fewest planes over all waves
    constexpr int strips = N / kCValid;
    const long long slots = (long long)sm_count() * CubeShape<N>::MINB;
    int planes = N;
    long long best = 1LL << 62;
    for (int p = N; p >= 8; p /= 2) {
        const long long cost = ((long long)fields * strips * (N / p) + slots - 1) / slots * (p + 4);
        if (cost < best) {
            best = cost;
            planes = p;
        }
    }
    for (int s = 0; s < steps; ++s) {
        float* dst = (steps - s) % 2 ? u_out : tmp;
        const unsigned grid = unsigned(fields) * strips * (N / planes);
        if (mass) cube_kernel<N, true><<<grid, CubeShape<N>::WARPS * 32, 0, st>>>(cur, dst, planes, cf, sums, s, steps - 1, a);
        else cube_kernel<N, false><<<grid, CubeShape<N>::WARPS * 32, 0, st>>>(cur, dst, planes, cf, sums, s, steps - 1, a);
        ACPR_LAUNCH_CHECK();
        cur = dst;
    }
    return AC_OK;
}

}  // namespace

int big_tiles_run(const SolvePoly& poly, double a, double dt, int mass, int fields, int steps, FieldMap src, FieldMap dst,
                  float* tmp, long long* sum_words, cudaStream_t st) {
    constexpr long long NN = (long long)kBig * kBig;
    const Coef<float, 2> cf = make_coef<float, 2>(a, dt, double(NN), poly);
    static DeviceSet configured;
    int rc = once_per_device(configured, [] {
        const int r = allow_smem(big_tile_kernel<true>, kTileSmem);
        return r ? r : allow_smem(big_tile_kernel<false>, kTileSmem);
    });
    if (rc) return rc;
    Sums sums{sum_words, fields};
    if (mass) {
        if ((rc = entry_sums(src, NN, sums, cf, st))) return rc;
    }
    FieldMap buf{};
    buf.base = tmp;
    buf.per_group = fields;
    const int per = mass ? 1 : kTSteps;
    const int launches = (steps + per - 1) / per;
    FieldMap cur = src;
    for (int l = 0, done = 0; l < launches; ++l) {
        const FieldMap to = (launches - l) % 2 ? dst : buf;  // the last launch writes dst
        const int k = std::min(per, steps - done);
        const unsigned grid = unsigned(fields) * (kTilesX * kTilesY);
        const int last = l == launches - 1;
        if (mass) big_tile_kernel<true><<<grid, kTWarps * 32, kTileSmem, st>>>(cur, to, k, cf, sums, done, last, a);
        else big_tile_kernel<false><<<grid, kTWarps * 32, kTileSmem, st>>>(cur, to, k, cf, sums, done, last, a);
        ACPR_LAUNCH_CHECK();
        cur = to;
        done += k;
    }
    return AC_OK;
}

int cube_run(const ac_params* p, const SolvePoly& poly, int steps, int fields, const float* u_in, float* u_out, float* tmp,
             long long* sum_words, cudaStream_t st) {
    const double a = 1.0 + p->S * p->dt;
    const int mass = p->variant == AC_MASS_CONSERVING;
    Sums sums{sum_words, fields};
    switch (p->n) {
        case 32: return cube_steps<32>(poly, a, p->dt, mass, steps, fields, u_in, u_out, tmp, sums, st);
        case 64: return cube_steps<64>(poly, a, p->dt, mass, steps, fields, u_in, u_out, tmp, sums, st);
        case 128: return cube_steps<128>(poly, a, p->dt, mass, steps, fields, u_in, u_out, tmp, sums, st);
        default: return AC_ERR_UNSUPPORTED;
    }
}

}  // namespace acpr
