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

// Shift that puts the mean of the new field at the entry mean.
__device__ __forceinline__ float step_shift(const Sums& s, int n, int f, double a, double cells) {
    if (*s.bad(f)) return __int_as_float(0x7fffffff);
    const long long target = __double2ll_rn(a * double(*s.entry(f)));
    return float(target - *s.slot(n, f)) * float(1.0 / (a * cells * double(kFix)));
}

__device__ __forceinline__ float rhs(float v, float mdt, float kappa) { return fmaf(v, fmaf(mdt, v * v, kappa), v); }

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
// A block of 16 warps holds a tile of 144 x 224 cells in registers (a lane 9
// rows of 7 columns) and runs up to 4 steps on it, two rows and columns of the
// rim going stale per step; the inner 128 x 208 cells are stored.  8 x 5 tiles
// cover the field (the last column of tiles is cut), 81% of the computed cells
// are stored: 4 steps cost one read and one write of the field where the
// Fourier passes moved 16 bytes a cell and step.  The mass model needs the
// field's sum each step and runs one step per launch.
// Bound: FP32 issue.  32 fields, 50 steps: two Fourier passes 10.67 ms, tiles 2.41 ms.
constexpr int kTW = 7, kTH = 9, kTWarps = 16, kRim = 8, kTSteps = 4;
constexpr int kTCols = 32 * kTW, kTRows = kTWarps * kTH;
constexpr int kTValidC = kTCols - 2 * kRim, kTValidR = kTRows - 2 * kRim;
constexpr int kBig = 1024;
constexpr int kTilesX = (kBig + kTValidC - 1) / kTValidC, kTilesY = kBig / kTValidR;
constexpr size_t kTileSmem = size_t(2) * 2 * kTWarps * 2 * kTCols * sizeof(float);
static_assert(kBig % kTValidR == 0 && kRim >= 2 * kTSteps, "tiling");

template <bool MASS>
__global__ void __launch_bounds__(kTWarps * 32, 1) big_tile_kernel(FieldMap src, FieldMap dst, int steps,
                                                                   const __grid_constant__ Coef<float, 2> cf, Sums sums,
                                                                   int n_step, double a) {
    constexpr int M = 2;
    constexpr long long NN = (long long)kBig * kBig;
    extern __shared__ __align__(16) float halo[];  // [buffer][0: above, 1: below][warp][M][kTCols]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int f = blockIdx.x / (kTilesX * kTilesY), tile = blockIdx.x % (kTilesX * kTilesY);
    const int tx = tile % kTilesX, ty = tile / kTilesX;
    const int row0 = ty * kTValidR - kRim + warp * kTH, col0 = tx * kTValidC - kRim + lane * kTW;
    const float* in = src.at(f, NN);
    float u[kTH][kTW];
#pragma unroll
    for (int y = 0; y < kTH; ++y)
#pragma unroll
        for (int c = 0; c < kTW; ++c) u[y][c] = in[((row0 + y) & (kBig - 1)) * kBig + ((col0 + c) & (kBig - 1))];
    constexpr int BUF = 2 * kTWarps * M * kTCols;
    // the tile's first and last rows have no neighbour: they hand their rows to
    // a slot nobody needs, and read stale ones (their cells are rim)
    float* up = halo + (kTWarps + (warp > 0 ? warp - 1 : kTWarps - 1)) * M * kTCols;
    float* down = halo + (warp < kTWarps - 1 ? warp + 1 : 0) * M * kTCols;
    const float* above = halo + warp * M * kTCols;
    const float* below = halo + (kTWarps + warp) * M * kTCols;
    float shift = 0.f;
    if constexpr (MASS) {
        shift = step_shift(sums, n_step, f, a, double(NN));
        if (tile == 0 && threadIdx.x == 0) *sums.slot(n_step + 2, f) = 0;
    }
    for (int s = 0; s < steps; ++s) {
        const int buf = s & 1;
#pragma unroll
        for (int y = 0; y < kTH; ++y)
#pragma unroll
            for (int c = 0; c < kTW; ++c) u[y][c] = rhs(u[y][c], cf.mdt, cf.kappa);
#pragma unroll
        for (int m = 0; m < M; ++m) {
            row_store<kTW>(up + buf * BUF + m * kTCols, u[m], lane);
            row_store<kTW>(down + buf * BUF + m * kTCols, u[kTH - M + m], lane);
        }
        __syncthreads();
        apply_poly<kTW, kTH, M, MASS>(u, cf, lane, shift, [&](int y, float(&x)[kTW]) {
            row_load<kTW>((y < 0 ? above + (y + M) * kTCols : below + (y - kTH) * kTCols) + buf * BUF, x, lane);
        });
    }
    float* out = dst.at(f, NN);
    long long acc = 0;
    bool bad = false;
#pragma unroll
    for (int y = 0; y < kTH; ++y) {
        const int lr = warp * kTH + y;
        if (lr < kRim || lr >= kRim + kTValidR) continue;
        float t = 0.f;
#pragma unroll
        for (int c = 0; c < kTW; ++c) {
            const int lc = lane * kTW + c;
            if (lc < kRim || lc >= kRim + kTValidC || col0 + c >= kBig) continue;
            out[(row0 + y) * kBig + col0 + c] = u[y][c];
            if constexpr (MASS) t += rhs(u[y][c], cf.mdt, cf.kappa);
        }
        if constexpr (MASS) {
            acc += __float2ll_rn(t * kFix);
            bad |= !(fabsf(t) < 0x1p18f);
        }
    }
    if constexpr (MASS) flush_sum(sums, sums.slot(n_step + 1, f), f, acc, bad, lane);
}

// ------------------------------------------------------------------- cube --
// A block streams the planes i of a chunk through a strip of 36 rows (9 warps,
// a lane 4 rows of N / 32 columns; 32 rows are stored) of all N columns, as
// apply_poly streams rows: r(i) completes w(i - 1), w(i - 1) completes
// u'(i - 2).  One barrier per plane hands the warps' edge rows of r and w to
// the warps above and below.  A step reads and writes the fields once (the
// five Fourier passes: 40 bytes a cell).  Bound: L2 / HBM and FP32 issue alike.
// 16 mass-conserving fields of 128^3, 20 steps: Fourier passes 7.45 ms, streamed 2.53 ms.
constexpr int kCWarps = 9, kCH = 4, kCRows = kCWarps * kCH, kCValid = kCRows - 4;

template <int N, bool MASS>
__global__ void __launch_bounds__(kCWarps * 32, 2) cube_kernel(const float* __restrict__ u, float* __restrict__ uo,
                                                               int planes, const __grid_constant__ Coef<float, 2> cf,
                                                               Sums sums, int n_step, double a) {
    constexpr int W = N / 32;
    constexpr long long NN = (long long)N * N, NNN = NN * N;
    __shared__ __align__(16) float edge[2][2][2][kCWarps][N];  // [buffer][r, w][first, last row][warp]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int strips = N / kCValid;
    const int strip = blockIdx.x % strips, chunk = blockIdx.x / strips % (N / planes), f = blockIdx.x / (strips * (N / planes));
    const int i0 = chunk * planes, j0 = strip * kCValid - 2 + warp * kCH;
    const float* in = u + f * NNN;
    float* out = uo + f * NNN;
    float shift = 0.f;
    if constexpr (MASS) {
        shift = step_shift(sums, n_step, f, a, double(NNN));
        if (strip == 0 && chunk == 0 && threadIdx.x == 0) *sums.slot(n_step + 2, f) = 0;
    }
    const int up = warp > 0 ? warp - 1 : kCWarps - 1, down = warp < kCWarps - 1 ? warp + 1 : 0;
    auto load_plane = [&](int i, float(&x)[kCH][W]) {
        const float* p = in + (long long)((i + N) & (N - 1)) * NN + lane * W;
#pragma unroll
        for (int y = 0; y < kCH; ++y) {
            const float* q = p + ((j0 + y) & (N - 1)) * N;
            if constexpr (W == 4) {
                const float4 v = *reinterpret_cast<const float4*>(q);
                x[y][0] = v.x; x[y][1] = v.y; x[y][2] = v.z; x[y][3] = v.w;
            } else if constexpr (W == 2) {
                const float2 v = *reinterpret_cast<const float2*>(q);
                x[y][0] = v.x; x[y][1] = v.y;
            } else {
                x[y][0] = *q;
            }
        }
    };
    // rp, rq: r(i - 1), r(i - 2); s0: the five known neighbours of r(i - 1);
    // wp: w(i - 2); s1: the five known neighbours of w(i - 2)
    float nxt[kCH][W], rp[kCH][W], rq[kCH][W], s0[kCH][W], wp[kCH][W], s1[kCH][W];
#pragma unroll
    for (int y = 0; y < kCH; ++y)
#pragma unroll
        for (int c = 0; c < W; ++c) rp[y][c] = rq[y][c] = s0[y][c] = wp[y][c] = s1[y][c] = 0.f;
    load_plane(i0 - 2, nxt);
    long long acc = 0;
    bool bad = false;
    for (int k = -2; k < planes + 2; ++k) {
        const int buf = k & 1;
        float r[kCH][W], w[kCH][W];
#pragma unroll
        for (int y = 0; y < kCH; ++y)
#pragma unroll
            for (int c = 0; c < W; ++c) {
                r[y][c] = rhs(nxt[y][c], cf.mdt, cf.kappa);
                w[y][c] = fmaf(cf.g[0], s0[y][c] + r[y][c], rp[y][c]);  // w(k - 1)
            }
        if (k < planes + 1) load_plane(i0 + k + 1, nxt);
        if (k >= 2) {
            float* p = out + (long long)(i0 + k - 2) * NN + lane * W;
#pragma unroll
            for (int y = 0; y < kCH; ++y) {
                float v[W];
#pragma unroll
                for (int c = 0; c < W; ++c) {
                    const float t = s1[y][c] + w[y][c], t0 = fmaf(cf.be0, rq[y][c], rq[y][c]);
                    v[c] = MASS ? t0 + fmaf(cf.b1, t, shift) : fmaf(cf.b1, t, t0);
                }
                const int lr = warp * kCH + y;
                if (lr < 2 || lr >= 2 + kCValid) continue;
                float* q = p + (j0 + y) * N;
                if constexpr (W == 4) *reinterpret_cast<float4*>(q) = make_float4(v[0], v[1], v[2], v[3]);
                else if constexpr (W == 2) *reinterpret_cast<float2*>(q) = make_float2(v[0], v[1]);
                else *q = v[0];
                if constexpr (MASS) {
                    float t = 0.f;
#pragma unroll
                    for (int c = 0; c < W; ++c) t += rhs(v[c], cf.mdt, cf.kappa);
                    acc += __float2ll_rn(t * kFix);
                    bad |= !(fabsf(t) < 0x1p16f);
                }
            }
        }
        row_store<W>(edge[buf][0][0][warp], r[0], lane);
        row_store<W>(edge[buf][0][1][warp], r[kCH - 1], lane);
        row_store<W>(edge[buf][1][0][warp], w[0], lane);
        row_store<W>(edge[buf][1][1][warp], w[kCH - 1], lane);
        __syncthreads();
        // s = (((left + right) + above) + below) + the plane before
        auto neighbours = [&](const float(&x)[kCH][W], int which, float(&prev)[kCH][W], float(&s)[kCH][W]) {
            float ab[W], be[W];
            row_load<W>(edge[buf][which][1][up], ab, lane);
            row_load<W>(edge[buf][which][0][down], be, lane);
#pragma unroll
            for (int y = 0; y < kCH; ++y) {
                float h[W];
                hsum<W>(x[y], h, lane);
#pragma unroll
                for (int c = 0; c < W; ++c)
                    s[y][c] = ((h[c] + (y ? x[y - 1][c] : ab[c])) + (y + 1 < kCH ? x[y + 1][c] : be[c])) + prev[y][c];
            }
        };
        neighbours(r, 0, rp, s0);
        neighbours(w, 1, wp, s1);
#pragma unroll
        for (int y = 0; y < kCH; ++y)
#pragma unroll
            for (int c = 0; c < W; ++c) {
                rq[y][c] = rp[y][c];
                rp[y][c] = r[y][c];
                wp[y][c] = w[y][c];
            }
    }
    if constexpr (MASS) flush_sum(sums, sums.slot(n_step + 1, f), f, acc, bad, lane);
}

template <int N>
int cube_steps(const SolvePoly& poly, double a, double dt, int mass, int steps, int fields, const float* u_in,
               float* u_out, float* tmp, Sums sums, cudaStream_t st) {
    constexpr long long NNN = (long long)N * N * N;
    const Coef<float, 2> cf = make_coef<float, 2>(a, dt, poly);
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
    // planes per block: long chunks repeat fewer planes, short ones fill the SMs
    constexpr int strips = N / kCValid;
    int planes = N < 32 ? N : 32;
    while (planes > 8 && (long long)fields * strips * (N / planes) < 200) planes /= 2;
    for (int s = 0; s < steps; ++s) {
        float* dst = (steps - s) % 2 ? u_out : tmp;
        const unsigned grid = unsigned(fields) * strips * (N / planes);
        if (mass) cube_kernel<N, true><<<grid, kCWarps * 32, 0, st>>>(cur, dst, planes, cf, sums, s, a);
        else cube_kernel<N, false><<<grid, kCWarps * 32, 0, st>>>(cur, dst, planes, cf, sums, s, a);
        ACPR_LAUNCH_CHECK();
        cur = dst;
    }
    return AC_OK;
}

}  // namespace

int big_tiles_run(const SolvePoly& poly, double a, double dt, int mass, int fields, int steps, FieldMap src, FieldMap dst,
                  float* tmp, long long* sum_words, cudaStream_t st) {
    constexpr long long NN = (long long)kBig * kBig;
    const Coef<float, 2> cf = make_coef<float, 2>(a, dt, poly);
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
        if (mass) big_tile_kernel<true><<<grid, kTWarps * 32, kTileSmem, st>>>(cur, to, k, cf, sums, done, a);
        else big_tile_kernel<false><<<grid, kTWarps * 32, kTileSmem, st>>>(cur, to, k, cf, sums, done, a);
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
