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
// whole field.  It is accumulated (fixed point, integer atomics: any order
// gives the same bits) by the launch that makes u^n.  Words per field:
// entry sum of u, three rotating sums of r, a mark for cells out of range.
struct Sums {
    long long* w;  // [5][fields]
    int fields;
    __device__ __forceinline__ long long* entry(int f) const { return w + f; }
    __device__ __forceinline__ long long* slot(int n, int f) const { return w + (long long)(1 + n % 3) * fields + f; }
    __device__ __forceinline__ long long* bad(int f) const { return w + 4LL * fields + f; }
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

// Shift that puts the mean of the new field at the entry mean (one thread of a
// block computes it: float64 instructions are scarce).
__device__ __forceinline__ float step_shift(const Sums& s, int n, int f, double a, double inv_sum) {
    if (*s.bad(f)) return __int_as_float(0x7fffffff);
    const long long target = __double2ll_rn(a * double(*s.entry(f)));
    return float(target - *s.slot(n, f)) * (float(inv_sum) * (1.f / kFix));
}

// Entry sums of u and of r^0, kSumParts blocks a field; cells a multiple of 4.
constexpr int kSumParts = 32;
__global__ void __launch_bounds__(256) entry_sums_kernel(FieldMap src, long long cells, Sums s, float mdt, float kappa) {
    const int f = blockIdx.x / kSumParts;
    const float4* u = reinterpret_cast<const float4*>(src.at(f, cells));
    long long su = 0, sr = 0;
    bool bad = false;
    for (long long i = (blockIdx.x % kSumParts) * 256LL + threadIdx.x; i < cells / 4; i += kSumParts * 256LL) {
        const float4 q = u[i];
        const float v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float r = rhs(v[c], mdt, kappa);
            su += __float2ll_rn(v[c] * kFix);
            sr += __float2ll_rn(r * kFix);
            bad |= !(fabsf(v[c]) < 0x1p16f) | !(fabsf(r) < 0x1p16f);
        }
    }
    const int lane = threadIdx.x & 31;
    flush_sum(s, s.entry(f), f, su, bad, lane);
    flush_sum(s, s.slot(0, f), f, sr, bad, lane);
}

// ------------------------------------------------------------ 1024 x 1024 --
// A block of 16 warps holds a tile of 144 x 256 cells in registers (a lane 9
// rows of 8 columns) and runs up to 4 steps on it, two rows and columns of the
// rim going stale per step; the inner 128 x 208 cells are stored (8 x 5 tiles,
// the last column of tiles cut; 71% of the computed cells): 4 steps cost one read and one write of the field where the
// Fourier passes moved 16 bytes a cell and step.  The mass model needs the
// field's sum each step and runs one step per launch.
// Bound: FP32 issue.  us a step, 32 fields: two Fourier passes 213, tiles 34.5 (scalar
// arithmetic on 7 columns a lane 48); mass-conserving 82 (one step a launch).
constexpr int kTW = 8, kTH = 9, kTWarps = 16, kRim = 8, kTSteps = 4;
constexpr int kTCols = 32 * kTW, kTRows = kTWarps * kTH;
constexpr int kBig = 1024;
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
    __shared__ float shift_sh;
    if (MASS && threadIdx.x == 0) {
        shift_sh = step_shift(sums, n_step, f, a, cf.inv_sum);
        if (tile == 0) *sums.slot(n_step + 2, f) = 0;
    }
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
            [&] { return shift_sh; });  // written before the step's barrier
    }
    float* out = dst.at(f, NN) + col0;
    // whole lanes are rim or stored
    const bool keep = lane * kTW >= kRim && lane * kTW < kRim + kTValidC && col0 < kBig;
    long long acc = 0;
    bool bad = false;
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
            float t = 0.f;
#pragma unroll
            for (int e = 0; e < kTW; ++e) t += c[e];
            acc += __float2ll_rn(t * kFix);
            bad |= !(fabsf(t) < 0x1p18f);
        }
    }
    if (MASS && !last) flush_sum(sums, sums.slot(n_step + 1, f), f, acc, bad, lane);
}

// ------------------------------------------------------------------- cube --
// A block streams the planes i of a chunk through a strip of 36 rows (12 warps
// of 3 rows at N = 128, 9 of 4 below; a lane N / 32 columns of each; 32 rows are stored) of all N columns, as
// apply_poly streams rows: r(i) completes w(i - 1), w(i - 1) completes
// u'(i - 2).  One barrier per plane hands the warps' edge rows of r and w to
// the warps above and below.  A step reads and writes the fields once (the
// five Fourier passes: 40 bytes a cell).  Bound: the latency of a plane
// (loads, barrier, exchange), 4 TB/s of HBM traffic beside it.  us a step, mass / classic:
// 16 fields of 128^3  Fourier passes 372, streamed 89 / 75 (2 rows a warp 107 / 65, 4 rows 121 / 102; handing on r
// instead of u 103 / 93); 48 fields of 64^3 47 / 33.
constexpr int kCRows = 36, kCValid = kCRows - 4;
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
    __shared__ float shift_sh;
    if constexpr (MASS) {
        if (threadIdx.x == 0) {
            shift_sh = step_shift(sums, n_step, f, a, cf.inv_sum);
            if (strip == 0 && chunk == 0) *sums.slot(n_step + 2, f) = 0;
        }
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
    const V be0 = vset<V>(cf.be0), b1 = vset<V>(cf.b1), g = vset<V>(cf.g[0]), sh = vset<V>(MASS ? shift_sh : 0.f);
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
    // sums of u' and u'^3 over four planes (float32), then sum r = (1 + kappa) sum u' - dt sum u'^3 in fixed point
    V part = vset<V>(0.f), cubes = vset<V>(0.f);
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
#pragma unroll
                    for (int c = 0; c < E; ++c) {
                        part = vadd(part, o[c]);
                        cubes = vfma(vmul(o[c], o[c]), o[c], cubes);
                    }
                }
            }
            if (MASS && (k & 3) == 1) {
                part = vfma(mdt, cubes, vfma(kappa, part, part));
                float t;
                if constexpr (Lane<W>::PAIR) t = lo_of(part) + hi_of(part);
                else t = part;
                acc += __float2ll_rn(t * kFix);
                bad |= !(fabsf(t) < 0x1p20f);
                part = cubes = vset<V>(0.f);
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
    if (MASS && !last) flush_sum(sums, sums.slot(n_step + 1, f), f, acc, bad, lane);
}

int sm_count() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
            sms = 1;
    }
    return sms;
}

template <int N>
int cube_steps(const SolvePoly& poly, double a, double dt, int mass, int steps, int fields, const float* u_in,
               float* u_out, float* tmp, Sums sums, cudaStream_t st) {
    constexpr long long NNN = (long long)N * N * N;
    const Coef<float, 2> cf = make_coef<float, 2>(a, dt, double(NNN), poly);
    if (mass) {
        ACPR_CUDA(cudaMemsetAsync(sums.w, 0, sizeof(long long) * 5 * fields, st));
        FieldMap src{};
        src.base = const_cast<float*>(u_in);
        src.per_group = fields;
        entry_sums_kernel<<<unsigned(fields) * kSumParts, 256, 0, st>>>(src, NNN, sums, cf.mdt, cf.kappa);
        ACPR_LAUNCH_CHECK();
    }
    // the last step writes u_out, the ones before alternate with tmp
    const float* cur = u_in;
    if (u_in == u_out && steps % 2) {
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
    static bool configured = false;
    if (!configured) {
        ACPR_CUDA(cudaFuncSetAttribute(big_tile_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kTileSmem)));
        ACPR_CUDA(cudaFuncSetAttribute(big_tile_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kTileSmem)));
        configured = true;
    }
    Sums sums{sum_words, fields};
    if (mass) {
        ACPR_CUDA(cudaMemsetAsync(sums.w, 0, sizeof(long long) * 5 * fields, st));
        entry_sums_kernel<<<unsigned(fields) * kSumParts, 256, 0, st>>>(src, NN, sums, cf.mdt, cf.kappa);
        ACPR_LAUNCH_CHECK();
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
