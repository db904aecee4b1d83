// fine_stencil.cu -- the fine propagator by a polynomial solve: the same
// stabilised step as fine.cu (Sec. 3.1),
//   (a - dt eps^2 Lap_h) u' = r,  r = u + u (kappa - dt u^2),  a = 1 + S dt,
//   kappa = S dt + dt,
// with A^{-1} applied as a polynomial of the 5-point stencil instead of a pair
// of Fourier transforms.  With lambda = dt eps^2 4 / h^2 the spectrum of
// -dt eps^2 Lap_h is [0, 2 lambda]; an interface resolved by a few cells and a
// step that resolves the dynamics make lambda about 25 dt (1e-3 at the paper's
// steps), A is within 1e-3 of a multiple of the identity, and the Chebyshev
// series of 1 / (a + s) on the spectrum converges by a factor rho = lambda / 4
// per degree: degree 2 is exact to 1e-9 and degree 4 to 4e-16.  A cell then
// costs 4 M + 4 operations (12 at degree 2) and M rows of neighbours where the
// Fourier solve costs about 75 instructions and two transposes over the
// cluster.  Steps too stiff for a built degree take the Fourier kernel.
//
// p(Lap) = sum_j b_j T^j (T: sum of the four neighbours), evaluated as
//   w_M = r,  w_j = r + (b_{j+1} / b_j) T w_{j+1},  u' = r + (b_0 - 1) r + b_1 T w_1,
// so every rounded coefficient multiplies a term of size lambda: a rounding of
// b_0 itself would be a gain error repeated in every step.  A cell's value is
// the same sequence of operations whatever the split into warps, CTAs and
// clusters, so the split follows the batch size and F stays one function.
//
// Mass-conserving model: beta shifts every cell alike, so u' = p(Lap) r + shift
// with the shift that puts the mean at the field's entry mean: mean(p(Lap) r) =
// mean(r) / a.  The sum of r over the field is formed in integers (fixed point:
// one word for float32, two for float64), which makes it independent of the
// order and of the split.  The unit follows the largest cell, so the mean is as
// exact for small, large, growing and decaying fields as for those of size one;
// only a field that outgrows its unit (float32: 2^18-fold in two runs of steps,
// see Coef::run, float64: 2^19-fold in one step; a blow-up) becomes not a number.
//
// Bound: FP32 (float64: FP64) issue and the step's barrier (512 fields of 256^2:
// FP32 pipe 62% busy, half of the issue slots).  Measured, Fourier kernel -> this one:
//   512 fields of 256^2, mass, 100 steps        11.40 -> 1.95 ms (2.21 with scalar instructions and 8x8x4)
//   21 fields of 512^2, 50 to 90 steps           3.01 -> 0.25 ms (0.37)
//   float64 256^2, 300 steps, their recomputation and adjoint  138 -> 22.5 ms (32.3 one after the other)
//   one step of one 128^2 field (call included)  16.4 -> 9.6 us
// Error against 64 bits after 100 float32 steps at 256^2: 1.5e-5 -> 1.5e-6.
#include <algorithm>
#include <cmath>

#include "fine_stencil.cuh"

namespace cg = cooperative_groups;

namespace acpr {

SolvePoly solve_poly(double a, double lam_scale, int dims, int precision, int min_degree, int max_degree) {
    SolvePoly out;
    // 1 / (C - x) on [-h, h], x = (lambda / 4) T, in Chebyshev polynomials of
    // z = x / h = T / (2 dims): c_0 = 1 / R, c_k = 2 rho^k / R
    const double h = 0.5 * dims * lam_scale, C = a + h;
    const double R = std::sqrt((C - h) * (C + h)), rho = h / (C + R);
    // The error is largest for the checkerboard mode, 4 rho^(M+1): at most one
    // rounding in float32, two in float64.  Against a long double
    // solve, 300 steps at 128^2 (lambda = 1.25e-3): degree 4 6e-14, degree 5
    // 2.6e-14, a float64 Fourier solve 5e-14; at 64^2 (1e-3), 400 steps:
    // degree 4 2.8e-14, Fourier 6e-14.  Against a float64 Fourier solve, whose
    // own rounding another Fourier solve shares in part: a Parareal solve at
    // 64^2 (1e-3, degree 4) 1.0e-13, the Fourier kernel 8.2e-14.
    const double tol = precision == AC_F64 ? 0x1p-52 : 0x1p-24;
    int M = std::max(1, min_degree);
    while (M <= max_degree && 4.0 * std::pow(rho, M + 1) > tol) ++M;
    // b_0 = 1 / a is applied as r + (b_0 - 1) r, whose rounding grows to a times
    // b_0's own: beyond a = 2 the Fourier solve is the more exact one
    if (M > max_degree || M > kMaxDegree || !(a > 0.0 && a <= 2.0) || !std::isfinite(rho)) return out;
    double c[kMaxDegree + 1];
    double sum = 0.0;
    for (int k = 0; k <= M; ++k) {
        c[k] = (k ? 2.0 : 1.0) * std::pow(rho, k) / R;
        sum += c[k];
    }
    c[M] += 1.0 / a - sum;  // exact for the mean mode (z = 1)
    // Chebyshev to monomials
    double t0[kMaxDegree + 1] = {1.0}, t1[kMaxDegree + 1] = {0.0, 1.0}, z[kMaxDegree + 1] = {};
    for (int k = 0; k <= M; ++k) {
        for (int j = 0; j <= k; ++j) z[j] += c[k] * t0[j];
        double t2[kMaxDegree + 1] = {};
        for (int j = 0; j <= M; ++j) t2[j] = (j ? 2.0 * t1[j - 1] : 0.0) - t0[j];
        std::copy(t1, t1 + kMaxDegree + 1, t0);
        std::copy(t2, t2 + kMaxDegree + 1, t1);
    }
    out.degree = M;
    for (int j = 0; j <= M; ++j) out.b[j] = z[j] / std::pow(2.0 * dims, j);
    return out;
}

namespace {

template <int P>
__device__ __forceinline__ void cl_arrive() {
    if constexpr (P > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
template <int P>
__device__ __forceinline__ void cl_wait() {
    if constexpr (P > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
}

template <int P, typename V>
__device__ __forceinline__ V* peer(V* local, int rank) {
    if constexpr (P > 1) return cg::this_cluster().map_shared_rank(local, rank);
    else return local;
}

// Field and step count of this block's work item.
struct Item {
    long long fin, fout;
    int steps;
};
__device__ __forceinline__ Item item_of(const FineArgs& args, int field) {
    Item it;
    it.steps = args.steps;
    if (args.work) {
        const int4 w = args.work[field];
        it.fin = w.x;
        it.fout = w.y;
        it.steps = w.z;
    } else {
        const int g = field / args.per_group, i = field % args.per_group;
        const long long pg = args.map ? args.map[g] : g;
        it.fin = pg * args.in_gs + args.in_off + i;
        it.fout = pg * args.out_gs + args.out_off + i;
    }
    return it;
}

// ------------------------------------------------ float32, in registers --
// A warp owns H full rows; lane l holds the W = N / 32 adjacent columns l W ..
// of each, so the horizontal neighbours at the run's ends come by one shuffle
// each way (the ring of lanes is the periodic row).  The rows of the warps
// above and below come through shared memory (`halo`), those of the
// neighbouring CTAs of the cluster through their shared memory: M rows each
// way per step, double-buffered, one cluster barrier per step.

// The lane's W columns of a row in global memory (row base, 16-byte aligned).
template <int W>
__device__ __forceinline__ void grow_load(const float* row, LaneV<W> (&x)[Lane<W>::E], int lane) {
    const float* p = row + lane * W;
    float c[W];
    if constexpr (W >= 4) {
#pragma unroll
        for (int v = 0; v < W / 4; ++v) {
            const float4 q = reinterpret_cast<const float4*>(p)[v];
            c[4 * v] = q.x; c[4 * v + 1] = q.y; c[4 * v + 2] = q.z; c[4 * v + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < W; ++i) c[i] = p[i];
    }
    to_lane<W>(c, x);
}
template <int W>
__device__ __forceinline__ void grow_store(float* row, const LaneV<W> (&x)[Lane<W>::E], int lane) {
    float* p = row + lane * W;
    float c[W];
    from_lane<W>(x, c);
    if constexpr (W >= 4) {
#pragma unroll
        for (int v = 0; v < W / 4; ++v)
            reinterpret_cast<float4*>(p)[v] = make_float4(c[4 * v], c[4 * v + 1], c[4 * v + 2], c[4 * v + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < W; ++i) p[i] = c[i];
    }
}

template <int N, int H, int NW, int P, int M>
struct RegShape {
    static constexpr int W = N / 32, R = NW * H;
    static constexpr size_t HALO = size_t(2) * 2 * NW * M * N;  // floats
    static constexpr size_t SMEM = HALO * sizeof(float) + (size_t(4) * P * NW + NW) * sizeof(long long);
    static constexpr int ROOM = kGroupRoom - log2i(2 * W);  // of a cell of r, in groups of two rows of a lane
    static_assert(R * P == N && H % 2 == 0 && H >= M && N % 32 == 0, "split");
};

template <int N, int H, int NW, int P, int M, bool MASS, bool ADJ>
__device__ __forceinline__ void stencil_reg_body(const FineArgs& args, const Coef<float, M>& cf, int field) {
    using Sh = RegShape<N, H, NW, P, M>;
    constexpr int W = Sh::W, R = Sh::R, E = Lane<W>::E;
    using V = LaneV<W>;
    constexpr long long NN = (long long)N * N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* halo = reinterpret_cast<float*>(smem_raw);  // [buffer][0: above, 1: below][warp][M][N]
    long long* tot = reinterpret_cast<long long*>(halo + Sh::HALO);  // [buffer][P NW] sums of the warps
    constexpr int AUX = 2 * P * NW;                                  // from there [buffer][P NW] the warps' largest cells
    double* goal = reinterpret_cast<double*>(tot + 2 * AUX);         // [NW] (the register it would take spills elsewhere)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int rank = 0;
    if constexpr (P > 1) rank = int(cg::this_cluster().block_rank());
    const Item it = item_of(args, field);
    const int row0 = rank * R + warp * H;
    const float* in = static_cast<const float*>(args.in) + it.fin * NN + (long long)row0 * N;
    float* out = static_cast<float*>(args.out) + it.fout * NN + (long long)row0 * N;
    float* traj = args.traj ? static_cast<float*>(args.traj) + field * NN + (long long)row0 * N : nullptr;
    const long long traj_step = (long long)args.num_fields * NN;

    V u[H][E];
#pragma unroll
    for (int y = 0; y < H; ++y) grow_load<W>(in + y * N, u[y], lane);
    if (traj) {
#pragma unroll
        for (int y = 0; y < H; ++y) grow_store<W>(traj + y * N, u[y], lane);
    }

    // where this warp's first and last M rows go: `below` of the warp above,
    // `above` of the warp below (in the neighbouring CTAs at the slab's ends)
    constexpr int BUF = 2 * NW * M * N;
    float* up = halo + (NW + (warp > 0 ? warp - 1 : NW - 1)) * M * N;
    float* down = halo + (warp < NW - 1 ? warp + 1 : 0) * M * N;
    if (P > 1 && warp == 0) up = peer<P>(up, (rank + P - 1) % P);
    if (P > 1 && warp == NW - 1) down = peer<P>(down, (rank + 1) % P);
    const float* above = halo + warp * M * N;
    const float* below = halo + (NW + warp) * M * N;

    // mass model: the sum of r that keeps the entry mean (goal), in units of 1 / unit
    long long target = 0;
    float unit = 0.f, inv_unit = 0.f;
    double msum = 0.0;      // adjoint: this warp's part of the sum of lambda
    auto publish = [&](int at, long long v) {
        for (int q = lane; q < P; q += 32) peer<P>(tot, q)[at + rank * NW + warp] = v;
    };
    auto largest = [&](const long long* from) {
        unsigned m = 0;
        for (int i = lane; i < P * NW; i += 32) m = max(m, unsigned(from[i]));
        return __reduce_max_sync(0xffffffffu, m);
    };
    // largest magnitude of the warp's cells, as bits (not that of a NaN, which
    // the sums below find)
    auto measure = [&] {
        float m[W] = {};
#pragma unroll
        for (int y = 0; y < H; ++y) {
            float v[W];
            from_lane<W>(u[y], v);
#pragma unroll
            for (int c = 0; c < W; ++c) m[c] = fmaxf(m[c], fabsf(v[c]));
        }
#pragma unroll
        for (int o = W / 2; o > 0; o /= 2)
#pragma unroll
            for (int c = 0; c < o; ++c) m[c] = fmaxf(m[c], m[c + o]);
        return __reduce_max_sync(0xffffffffu, __float_as_uint(m[0]));
    };
    // the sums of r while no cell of u is much larger than m
    auto set_unit = [&](unsigned m) {
        const float now = pow2f(fix_scale(__float_as_uint(rhs_bound(__uint_as_float(m), cf.mdt, cf.kappa)), Sh::ROOM));
        if (now == unit) return;
        unit = now;
        inv_unit = float(cf.inv_sum) * pow2_inv(unit);
        target = __double2ll_rn(goal[warp] * double(unit));
    };
    cl_arrive<P>();
    cl_wait<P>();  // every CTA of the cluster runs
    if constexpr (MASS && !ADJ) {
        const unsigned mine = measure();
        publish(AUX, mine);
        cl_arrive<P>();
        cl_wait<P>();
        const unsigned m = largest(tot + AUX);
        const float entry_unit = pow2f(fix_scale(m, kCellRoom));
        long long entry = 0;
        // entry sum, cell by cell
#pragma unroll
        for (int y = 0; y < H; ++y) {
            float v[W];
            from_lane<W>(u[y], v);
#pragma unroll
            for (int c = 0; c < W; ++c) entry += __float2ll_rn(v[c] * entry_unit);
        }
        publish(P * NW, warp_sum_s64(entry));
        cl_arrive<P>();
        cl_wait<P>();
        entry = 0;
        for (int i = lane; i < P * NW; i += 32) entry += tot[P * NW + i];
        entry = warp_sum_s64(entry);
        if (lane == 0) goal[warp] = args.a * double(entry) * double(pow2_inv(entry_unit));
        __syncwarp();
        set_unit(m);
    }

    // Runs of steps with one unit for the sums of r, from the largest cell at the
    // start of the run before: handed round with that run's first sums, it needs
    // no barrier, and nothing of it parts the instructions of a step (asked for
    // within the steps, even by branches not taken, it made them 5 to 10% longer;
    // between runs of 16 steps 1 to 5%).
    const int run = MASS && !ADJ ? cf.run : it.steps;
    for (int step = 0, odd = 0; step < it.steps; odd ^= 1) {
        const int tops = AUX + odd * P * NW;
        if constexpr (MASS && !ADJ) publish(tops, measure());
        for (const int end = it.steps - step > run ? step + run : it.steps; step < end; ++step) {
            const int buf = step & 1;
            // the rows that others wait for first
            auto rhs_row = [&](int y) {
                if constexpr (!ADJ) {
#pragma unroll
                    for (int c = 0; c < E; ++c) u[y][c] = rhs(u[y][c], vset<V>(cf.mdt), vset<V>(cf.kappa));
                }
            };
#pragma unroll
            for (int y = 0; y < H; ++y)
                if (y < M || y >= H - M) rhs_row(y);
#pragma unroll
            for (int m = 0; m < M; ++m) {
                row_store<W>(up + buf * BUF + m * N, u[m], lane);
                row_store<W>(down + buf * BUF + m * N, u[H - M + m], lane);
            }
            if constexpr (!MASS) cl_arrive<P>();
#pragma unroll
            for (int y = M; y < H - M; ++y) rhs_row(y);
            if constexpr (MASS) {
                if constexpr (!ADJ) {
                    long long acc = 0;
                    bool bad = false;
#pragma unroll
                    for (int y = 0; y < H; y += 2) {
                        const float t = pair_sum<W>(u[y], u[y + 1]) * unit;
                        acc += __float2ll_rn(t);
                        bad |= !(fabsf(t) < 0x1p49f);  // 2^13 such sums stay below 2^62
                    }
                    acc = warp_sum_s64(acc);
                    if (__any_sync(0xffffffffu, bad)) acc = kBadSum;
                    publish(buf * P * NW, acc);
                } else {
                    msum = 0.0;
#pragma unroll
                    for (int y = 0; y < H; y += 2) msum += double(pair_sum<W>(u[y], u[y + 1]));
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) msum += __shfl_xor_sync(0xffffffffu, msum, o);
                    publish(buf * P * NW, __double_as_longlong(msum));
                }
            }
            if constexpr (MASS) cl_arrive<P>();
            cl_wait<P>();
            // the shift of the mass model, and the adjoint's mean of mu
            float shift = 0.f;
            auto collect = [&]() -> float {
                const long long* tb = tot + buf * P * NW;
                if constexpr (!ADJ) {
                    long long t = 0;
                    bool bad = false;
#pragma unroll
                    for (int i0 = 0; i0 < P * NW; i0 += 32) {
                        const long long v = P * NW % 32 == 0 || i0 + lane < P * NW ? tb[i0 + lane] : 0;
                        t += v;
                        bad |= v == kBadSum;
                    }
                    t = warp_sum_s64(t);
                    shift = float(target - t) * inv_unit;
                    if (__any_sync(0xffffffffu, bad)) shift = __int_as_float(0x7fffffff);
                } else {
                    double t = 0.0;
                    for (int i = lane; i < P * NW; i += 32) t += __longlong_as_double(tb[i]);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                    shift = float(t * cf.inv_sum);
                }
                return shift;
            };
            apply_poly<W, H, M, MASS && !ADJ>(
                u, cf, lane,
                [&](int y, V(&x)[E]) {
                    row_load<W>((y < 0 ? above + (y + M) * N : below + (y - H) * N) + buf * BUF, x, lane);
                },
                collect);
            if constexpr (MASS && ADJ) collect();
            if constexpr (ADJ) {
                const float* un = static_cast<const float*>(args.states) +
                                  ((long long)(it.steps - 1 - step) * args.num_fields + field) * NN + (long long)row0 * N;
#pragma unroll
                for (int y = 0; y < H; ++y) {
                    V v[E];
                    grow_load<W>(un + y * N, v, lane);
                    const V one = vset<V>(1.f), m3 = vset<V>(-3.f), a = vset<V>(cf.a), dt = vset<V>(cf.dt), ms = vset<V>(-shift);
#pragma unroll
                    for (int c = 0; c < E; ++c) {
                        const V f = vmul(dt, vfma(m3, vmul(v[c], v[c]), one));
                        u[y][c] = vfma(a, u[y][c], vmul(f, vadd(u[y][c], ms)));
                    }
                }
            }
            if (traj) {
                float* ts = traj + (step + 1) * traj_step;
#pragma unroll
                for (int y = 0; y < H; ++y) grow_store<W>(ts + y * N, u[y], lane);
            }
        }
        if constexpr (MASS && !ADJ) set_unit(largest(tot + tops));
    }
#pragma unroll
    for (int y = 0; y < H; ++y) grow_store<W>(out + y * N, u[y], lane);
}

template <int N, int H, int NW, int P, int M, int MINB, bool MASS, bool ADJ>
__global__ void __launch_bounds__(NW * 32, MINB) stencil_reg_kernel(const __grid_constant__ FineArgs args,
                                                                    const __grid_constant__ Coef<float, M> cf) {
    stencil_reg_body<N, H, NW, P, M, MASS, ADJ>(args, cf, blockIdx.x / P);
}

// Adjoint steps of some fields and forward steps of others in one launch.
template <int N, int H, int NW, int P, int M, bool MASS>
__global__ void __launch_bounds__(NW * 32, 1) stencil_reg_pair_kernel(const __grid_constant__ FineArgs adj,
                                                                      const __grid_constant__ FineArgs fwd,
                                                                      const __grid_constant__ Coef<float, M> cf) {
    const int f = blockIdx.x / P;
    if (f < adj.num_fields) stencil_reg_body<N, H, NW, P, M, MASS, true>(adj, cf, f);
    else stencil_reg_body<N, H, NW, P, M, MASS, false>(fwd, cf, f - adj.num_fields);
}

// Launches a kernel in clusters of P CTAs.
template <typename K, typename... A>
int launch_clusters(K kern, DeviceSet& configured, int P, unsigned fields, int threads, size_t smem, cudaStream_t stream,
                    const A&... a) {
    const int rc = once_per_device(configured, [&] { return allow_smem(kern, smem, P); });
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(fields * unsigned(P), 1, 1);
    cfg.blockDim = dim3(unsigned(threads), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(P);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = P > 1 ? 1 : 0;
    ACPR_CUDA(cudaLaunchKernelEx(&cfg, kern, a...));
    count_launch();
    return AC_OK;
}

template <int N, int H, int NW, int P, int M, int MINB, bool MASS, bool ADJ>
int launch_reg_t(const FineArgs& args, const SolvePoly& poly, cudaStream_t stream) {
    using Sh = RegShape<N, H, NW, P, M>;
    static DeviceSet configured;
    return launch_clusters(stencil_reg_kernel<N, H, NW, P, M, MINB, MASS, ADJ>, configured, P, unsigned(args.num_fields), NW * 32, Sh::SMEM, stream, args,
                           make_coef<float, M>(args.a, args.dt, double(N) * N, poly));
}

template <int N, int H, int NW, int P, int M, bool MASS>
int launch_reg_pair(const FineArgs& adj, const FineArgs& fwd, const SolvePoly& poly, cudaStream_t stream) {
    static DeviceSet configured;
    return launch_clusters(stencil_reg_pair_kernel<N, H, NW, P, M, MASS>, configured, P,
                           unsigned(adj.num_fields + fwd.num_fields), NW * 32, RegShape<N, H, NW, P, M>::SMEM, stream, adj,
                           fwd, make_coef<float, M>(adj.a, adj.dt, double(N) * N, poly));
}

template <int N, int H, int NW, int P, int M, int MINB>
int launch_reg(const FineArgs& args, const SolvePoly& poly, cudaStream_t st) {
    if (args.adjoint)
        return args.mass ? launch_reg_t<N, H, NW, P, M, MINB, true, true>(args, poly, st)
                         : launch_reg_t<N, H, NW, P, M, MINB, false, true>(args, poly, st);
    return args.mass ? launch_reg_t<N, H, NW, P, M, MINB, true, false>(args, poly, st)
                     : launch_reg_t<N, H, NW, P, M, MINB, false, false>(args, poly, st);
}

// The split (rows a warp, warps a CTA, CTAs a field, CTAs per SM) by size and
// batch.  40 steps, us, mass-conserving / classic, measured for each line (the
// mass-conserving ones within 10% of the present sums'):
//   256: 4x4x16  1 field 60/36, 8 70/45; 8x4x8 (1 CTA per SM's registers)  8 fields 62/42, 24 87/67;
//        8x4x8 (4 CTAs)  38 fields 106/83, 512 825/650; 8x8x4 512 fields 923/645, 8x16x2 999/703
//   512: 8x4x16  1 field 105/70, 21 216/164, 64 599/504; 4x8x16  112/72, 317/206, 1033/677
//   128: 4x4x8   1 field 38/25, 16 44/31; 8x4x4  16 fields 44/29, 64 56/38, 128 82/58;
//        16x8x1  64 fields 83/49, 128 83/50, 512 261/166 (8x4x4 252/177)
//   64:  4x4x4   1 field 29/21, 76 40/29; 16x4x1  39/18, 76 40/18, 512 79/50
//   32:  8x4x1   1 field 22/14, 512 40/24; 4x8x1 22/13, 49/29
// Degrees 3 and 4 keep more rows of the stages in registers and hold fewer
// rows of the field.
template <int M>
int dispatch_reg(int n, const FineArgs& args, const SolvePoly& poly, cudaStream_t st) {
    const int F = args.num_fields;
    if constexpr (M == 2) {
        switch (n) {
            case 32: return launch_reg<32, 8, 4, 1, M, 1>(args, poly, st);
            case 64:
                if (args.mass && F <= 76) return launch_reg<64, 4, 4, 4, M, 1>(args, poly, st);
                return launch_reg<64, 16, 4, 1, M, 4>(args, poly, st);
            case 128:
                if (F <= 12) return launch_reg<128, 4, 4, 8, M, 1>(args, poly, st);
                if (F <= 96) return launch_reg<128, 8, 4, 4, M, 4>(args, poly, st);
                return launch_reg<128, 16, 8, 1, M, 2>(args, poly, st);
            case 256:
                if (F <= 6) return launch_reg<256, 4, 4, 16, M, 1>(args, poly, st);
                if (F <= 24) return launch_reg<256, 8, 4, 8, M, 1>(args, poly, st);
                return launch_reg<256, 8, 4, 8, M, 4>(args, poly, st);
            case 512: return launch_reg<512, 8, 4, 16, M, 2>(args, poly, st);
            default: return AC_ERR_UNSUPPORTED;
        }
    } else {
        switch (n) {
            case 32: return launch_reg<32, 4, 8, 1, M, 1>(args, poly, st);
            case 64: return launch_reg<64, 8, 8, 1, M, 1>(args, poly, st);
            case 128: return launch_reg<128, 8, 8, 2, M, 2>(args, poly, st);
            case 256: return launch_reg<256, 4, 8, 8, M, 2>(args, poly, st);
            case 512:
                if constexpr (M == 3) return launch_reg<512, 4, 8, 16, M, 1>(args, poly, st);
                return AC_ERR_UNSUPPORTED;
            default: return AC_ERR_UNSUPPORTED;
        }
    }
}

// -------------------------------------------------- any type, shared memory --
// The same solve with r and the stages in shared memory: cluster of P CTAs,
// CTA q holds rows [q R, q R + R) plus M halo rows each way; a stage is
// computed on the rows the later stages need (the halo shrinks by a row per
// stage), a CTA barrier between stages, one cluster barrier per step.  Used in
// float64, whose arithmetic (two lanes per SM and cycle) is the bound.
constexpr int kShThreads = 256;

template <typename T, int N, int P, int M>
struct ShShape {
    static constexpr int R = N / P, RH = R + 2 * M, RW = R + 2 * (M - 1);
    static constexpr int K = R * N / kShThreads;  // cells per thread
    static constexpr size_t SMEM =
        sizeof(T) * N * (size_t(2) * RH + size_t(M > 2 ? 2 : 1) * RW) + size_t(2 * 3 + 2) * P * 8 * sizeof(long long);
    static_assert(R >= M && R * N % kShThreads == 0, "split");
};

// Exact sum pieces of a float64, in units that follow the field: with the
// largest magnitude below 2^(e + 1), x = hi 2^(e - 24) + lo 2^(e - 68) to
// 2^(e - 69), for |x| < 2^(e + 20) (2^16 cells keep both words below 2^61).
struct Fix64 {
    int e;
    double m1, m2;  // adding and subtracting one rounds to its word's unit
    static __device__ __forceinline__ double pow2(int k) { return __longlong_as_double((long long)(k + 1023) << 52); }
    static __device__ __forceinline__ double pow2_15(int k) {  // 1.5 2^k
        return __longlong_as_double((long long)(k + 1023) << 52 | 1LL << 51);
    }
    // `key`: high word of the largest magnitude (infinities and NaN: any e)
    __device__ __forceinline__ explicit Fix64(unsigned key)
        : e(min(max(int(key >> 20) - 1023, -900), 990)), m1(pow2_15(e + 28)), m2(pow2_15(e - 16)) {}
    __device__ __forceinline__ void add(double x, long long& hi, long long& lo) const {
        const double t = x + m1;
        const double rem = x - (t - m1);
        const double t2 = rem + m2;
        hi += __double_as_longlong(t) - __double_as_longlong(m1);
        lo += __double_as_longlong(t2) - __double_as_longlong(m2);
    }
    // not a number where a magnitude left the range
    __device__ __forceinline__ double value(long long hi, long long lo, unsigned key) const {
        if (int(key >> 20) - 1023 > min(e + 19, 1009)) return __longlong_as_double(0x7ff8000000000000LL);
        return double(hi) * pow2(e - 24) + double(lo) * pow2(e - 68);
    }
};
__device__ __forceinline__ unsigned abs_key(double x) { return unsigned(__double2hiint(x)) & kAbsMask; }

template <typename T, int N, int P, int M, bool MASS, bool ADJ>
__device__ __forceinline__ void stencil_smem_body(const FineArgs& args, const Coef<T, M>& cf, int field) {
    using Sh = ShShape<T, N, P, M>;
    constexpr int R = Sh::R, RH = Sh::RH, RW = Sh::RW, K = Sh::K;
    constexpr long long NN = (long long)N * N;
    constexpr int WARPS = kShThreads / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* rbuf = reinterpret_cast<T*>(smem_raw);       // [2][RH][N], row 0 is row -M
    T* wbuf = rbuf + 2 * RH * N;                     // [1 or 2][RW][N], row 0 is row -(M-1)
    long long* tot = reinterpret_cast<long long*>(wbuf + (M > 2 ? 2 : 1) * RW * N);  // [buffer][P WARPS][hi, lo, largest]
    long long* aux = tot + 2 * 3 * P * WARPS;                                         // [P WARPS][hi, lo] of the entry sum
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int rank = 0;
    if constexpr (P > 1) rank = int(cg::this_cluster().block_rank());
    const Item it = item_of(args, field);
    const T* in = static_cast<const T*>(args.in) + it.fin * NN + (long long)rank * R * N;
    T* out = static_cast<T*>(args.out) + it.fout * NN + (long long)rank * R * N;
    T* traj = args.traj ? static_cast<T*>(args.traj) + field * NN + (long long)rank * R * N : nullptr;
    const long long traj_step = (long long)args.num_fields * NN;
    T* rup = peer<P>(rbuf, (rank + P - 1) % P);
    T* rdown = peer<P>(rbuf, (rank + 1) % P);

    T u[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        u[i] = in[tid + i * kShThreads];
        if (traj) traj[tid + i * kShThreads] = u[i];
    }
    // (integer sums: any order gives the same bits)
    auto warp_sums = [](long long& hi, long long& lo) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            hi += __shfl_xor_sync(0xffffffffu, hi, o);
            lo += __shfl_xor_sync(0xffffffffu, lo, o);
        }
    };
    auto publish = [&](long long hi, long long lo, unsigned key, int buf) {
        key = __reduce_max_sync(0xffffffffu, key);
        for (int q = lane; q < P; q += 32) {
            long long* p = peer<P>(tot, q) + ((buf * P + rank) * WARPS + warp) * 3;
            p[0] = hi;
            p[1] = lo;
            p[2] = key;
        }
    };
    auto collect = [&](int buf, long long& hi, long long& lo) -> unsigned {
        unsigned key = 0;
        hi = lo = 0;
        for (int i = lane; i < P * WARPS; i += 32) {
            const long long* p = tot + (buf * P * WARPS + i) * 3;
            hi += p[0];
            lo += p[1];
            key = max(key, unsigned(p[2]));
        }
        warp_sums(hi, lo);
        return __reduce_max_sync(0xffffffffu, key);
    };
    cl_arrive<P>();
    cl_wait<P>();
    double mean = 0.0;               // mean of r that keeps the entry mean
    long long ehi = 0, elo = 0;      // entry sum, in units of ufix
    unsigned key = 0, ukey = 0;      // largest magnitude of r, of the entry field
    if constexpr (MASS) {
#pragma unroll
        for (int i = 0; i < K; ++i) ukey = max(ukey, abs_key(double(u[i])));
        publish(0, 0, ukey, 1);
        cl_arrive<P>();
        cl_wait<P>();
        ukey = key = collect(1, ehi, elo);
        if constexpr (!ADJ) {
            const double m = __hiloint2double(int(ukey), -1);  // |r| <= m max(1 + kappa, |1 + kappa - dt m^2|) over |u| <= m
            key = abs_key(m * fmax(1.0 + cf.kappa, fabs(fma(double(cf.mdt), m * m, 1.0 + cf.kappa))));
            const Fix64 ufix(ukey);
#pragma unroll
            for (int i = 0; i < K; ++i) ufix.add(double(u[i]), ehi, elo);
            warp_sums(ehi, elo);
        }
    }

    for (int step = 0; step < it.steps; ++step) {
        const int buf = step & 1;
        T* r = rbuf + buf * RH * N;
        long long hi = 0, lo = 0;
        const Fix64 fix(key);
        unsigned largest = 0;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int e = tid + i * kShThreads, y = e / N;
            T v = u[i];
            if constexpr (!ADJ) v = fma(v, fma(cf.mdt, v * v, cf.kappa), v);
            r[M * N + e] = v;
            if (y < M) rup[buf * RH * N + (M + R) * N + e] = v;
            if (y >= R - M) rdown[buf * RH * N + e - (R - M) * N] = v;
            if constexpr (MASS) {
                fix.add(double(v), hi, lo);
                largest = max(largest, abs_key(double(v)));
            }
        }
        if constexpr (MASS) {
            warp_sums(hi, lo);
            publish(hi, lo, largest, buf);
            if (!ADJ && step == 0 && lane < P) {
                long long* p = peer<P>(aux, lane) + (rank * WARPS + warp) * 2;
                p[0] = ehi;
                p[1] = elo;
            }
        }
        cl_arrive<P>();
        cl_wait<P>();
        T shift = T(0);
        if constexpr (MASS) {
            if (!ADJ && step == 0) {
                ehi = elo = 0;
                for (int i = lane; i < P * WARPS; i += 32) {
                    ehi += aux[i * 2];
                    elo += aux[i * 2 + 1];
                }
                warp_sums(ehi, elo);
                mean = Fix64(ukey).value(ehi, elo, ukey) * (args.a * cf.inv_sum);
            }
            key = collect(buf, hi, lo);
            const double m = fix.value(hi, lo, key) * cf.inv_sum;
            shift = T(ADJ ? m : mean - m);
        }
        // stages: w_k on rows -(M-1-k) .. R + (M-1-k)
        const T* src = r;
        int srow = -M;  // row index of src's first stored row
#pragma unroll
        for (int k = 0; k < M - 1; ++k) {
            T* dst = wbuf + (k & 1) * RW * N;
            const int ext = M - 1 - k;
            const T g = cf.g[k];
            for (int e = tid; e < (R + 2 * ext) * N; e += kShThreads) {
                const int y = e / N - ext, x = e % N;
                const T* p = src + (y - srow) * N + x;
                const T* row = p - x;
                const T t = ((row[(x + N - 1) % N] + row[(x + 1) % N]) + p[-N]) + p[N];
                dst[(y + M - 1) * N + x] = fma(g, t, r[(y + M) * N + x]);
            }
            __syncthreads();
            src = dst;
            srow = -(M - 1);
        }
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int e = tid + i * kShThreads, y = e / N, x = e % N;
            const T* p = src + (y - srow) * N + x;
            const T* row = p - x;
            const T t = ((row[(x + N - 1) % N] + row[(x + 1) % N]) + p[-N]) + p[N];
            const T rv = r[(y + M) * N + x];
            const T t0 = fma(cf.be0, rv, rv);
            T v = MASS && !ADJ ? t0 + fma(cf.b1, t, shift) : fma(cf.b1, t, t0);
            if constexpr (ADJ) {
                const T w = static_cast<const T*>(args.states)[((long long)(it.steps - 1 - step) * args.num_fields + field) * NN +
                                                               (long long)rank * R * N + e];
                v = fma(cf.a, v, cf.dt * (T(1) - T(3) * w * w) * (v - shift));
            }
            u[i] = v;
            if (traj) traj[(step + 1) * traj_step + e] = v;
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i) out[tid + i * kShThreads] = u[i];
}

template <typename T, int N, int P, int M, bool MASS, bool ADJ>
__global__ void __launch_bounds__(kShThreads) stencil_smem_kernel(const __grid_constant__ FineArgs args,
                                                                  const __grid_constant__ Coef<T, M> cf) {
    stencil_smem_body<T, N, P, M, MASS, ADJ>(args, cf, blockIdx.x / P);
}

template <typename T, int N, int P, int M, bool MASS>
__global__ void __launch_bounds__(kShThreads) stencil_smem_pair_kernel(const __grid_constant__ FineArgs adj,
                                                                       const __grid_constant__ FineArgs fwd,
                                                                       const __grid_constant__ Coef<T, M> cf) {
    const int f = blockIdx.x / P;
    if (f < adj.num_fields) stencil_smem_body<T, N, P, M, MASS, true>(adj, cf, f);
    else stencil_smem_body<T, N, P, M, MASS, false>(fwd, cf, f - adj.num_fields);
}

template <typename T, int N, int P, int M, bool MASS, bool ADJ>
int launch_smem_t(const FineArgs& args, const SolvePoly& poly, cudaStream_t stream) {
    using Sh = ShShape<T, N, P, M>;
    static DeviceSet configured;
    return launch_clusters(stencil_smem_kernel<T, N, P, M, MASS, ADJ>, configured, P, unsigned(args.num_fields), kShThreads, Sh::SMEM, stream, args,
                           make_coef<T, M>(args.a, args.dt, double(N) * N, poly));
}

template <typename T, int N, int P, int M, bool MASS>
int launch_smem_pair(const FineArgs& adj, const FineArgs& fwd, const SolvePoly& poly, cudaStream_t stream) {
    static DeviceSet configured;
    return launch_clusters(stencil_smem_pair_kernel<T, N, P, M, MASS>, configured, P,
                           unsigned(adj.num_fields + fwd.num_fields), kShThreads, ShShape<T, N, P, M>::SMEM, stream, adj, fwd,
                           make_coef<T, M>(adj.a, adj.dt, double(N) * N, poly));
}

template <typename T, int N, int P, int M>
int launch_smem(const FineArgs& args, const SolvePoly& poly, cudaStream_t st) {
    if (args.adjoint)
        return args.mass ? launch_smem_t<T, N, P, M, true, true>(args, poly, st)
                         : launch_smem_t<T, N, P, M, false, true>(args, poly, st);
    return args.mass ? launch_smem_t<T, N, P, M, true, false>(args, poly, st)
                     : launch_smem_t<T, N, P, M, false, false>(args, poly, st);
}

template <int M>
int dispatch_smem(int n, const FineArgs& args, const SolvePoly& poly, cudaStream_t st) {
    switch (n) {
        case 32: return launch_smem<double, 32, 4, M>(args, poly, st);
        case 64:
            if constexpr (M <= 4) {
                if (args.num_fields <= 9) return launch_smem<double, 64, 16, M>(args, poly, st);
            }
            return launch_smem<double, 64, 8, M>(args, poly, st);
        case 128: return launch_smem<double, 128, 16, M>(args, poly, st);
        case 256: return launch_smem<double, 256, 16, M>(args, poly, st);
        default: return AC_ERR_UNSUPPORTED;
    }
}

template <bool MASS>
int dispatch_reg_pair(int n, const FineArgs& adj, const FineArgs& fwd, const SolvePoly& poly, cudaStream_t st) {
    switch (n) {  // the splits for few fields
        case 32: return launch_reg_pair<32, 8, 4, 1, 2, MASS>(adj, fwd, poly, st);
        case 64: return launch_reg_pair<64, 4, 4, 4, 2, MASS>(adj, fwd, poly, st);
        case 128: return launch_reg_pair<128, 4, 4, 8, 2, MASS>(adj, fwd, poly, st);
        case 256: return launch_reg_pair<256, 4, 4, 16, 2, MASS>(adj, fwd, poly, st);
        case 512: return launch_reg_pair<512, 8, 4, 16, 2, MASS>(adj, fwd, poly, st);
        default: return AC_ERR_UNSUPPORTED;
    }
}
template <int M, bool MASS>
int dispatch_smem_pair(int n, const FineArgs& adj, const FineArgs& fwd, const SolvePoly& poly, cudaStream_t st) {
    switch (n) {
        case 32: return launch_smem_pair<double, 32, 4, M, MASS>(adj, fwd, poly, st);
        case 64: return launch_smem_pair<double, 64, M <= 4 ? 16 : 8, M, MASS>(adj, fwd, poly, st);
        case 128: return launch_smem_pair<double, 128, 16, M, MASS>(adj, fwd, poly, st);
        case 256: return launch_smem_pair<double, 256, 16, M, MASS>(adj, fwd, poly, st);
        default: return AC_ERR_UNSUPPORTED;
    }
}

bool unaligned(const FineArgs& a) {
    return (reinterpret_cast<uintptr_t>(a.in) | reinterpret_cast<uintptr_t>(a.out) | reinterpret_cast<uintptr_t>(a.states) |
            reinterpret_cast<uintptr_t>(a.traj)) % 16;
}

}  // namespace

template <>
int launch_stencil<float>(int n, const FineArgs& args, cudaStream_t stream, bool* taken) {
    *taken = false;
    if (n < 32 || n > 512) return AC_OK;
    // rows move as vectors; callers that pass unaligned fields keep the Fourier kernels
    if (unaligned(args)) return AC_OK;
    // degree 4 rows of 512 columns would need 262 KB of halo buffers
    const SolvePoly p = solve_poly(args.a, args.lam_scale, 2, AC_F32, 2, n == 512 ? 3 : 4);
    if (!p.degree) return AC_OK;
    *taken = true;
    if (!args.num_fields) return AC_OK;
    switch (p.degree) {
        case 2: return dispatch_reg<2>(n, args, p, stream);
        case 3: return dispatch_reg<3>(n, args, p, stream);
        default: return dispatch_reg<4>(n, args, p, stream);  // n <= 256
    }
}

template <>
int launch_stencil<double>(int n, const FineArgs& args, cudaStream_t stream, bool* taken) {
    *taken = false;
    if (n < 32 || n > 256) return AC_OK;
    const SolvePoly p = solve_poly(args.a, args.lam_scale, 2, AC_F64, 4, 6);
    if (!p.degree) return AC_OK;
    *taken = true;
    if (!args.num_fields) return AC_OK;
    switch (p.degree) {
        case 4: return dispatch_smem<4>(n, args, p, stream);
        case 5: return dispatch_smem<5>(n, args, p, stream);
        default: return dispatch_smem<6>(n, args, p, stream);
    }
}

int launch_stencil_pair(int n, int precision, const FineArgs& adj, const FineArgs& fwd, cudaStream_t stream, bool* taken) {
    *taken = false;
    const bool f32 = precision == AC_F32;
    if (n < 32 || n > (f32 ? 512 : 256) || (f32 && (unaligned(adj) || unaligned(fwd)))) return AC_OK;
    const SolvePoly p = solve_poly(adj.a, adj.lam_scale, 2, precision, f32 ? 2 : 4, f32 ? 2 : 5);
    if (!p.degree) return AC_OK;
    *taken = true;
    if (f32) return adj.mass ? dispatch_reg_pair<true>(n, adj, fwd, p, stream) : dispatch_reg_pair<false>(n, adj, fwd, p, stream);
    if (p.degree == 4)
        return adj.mass ? dispatch_smem_pair<4, true>(n, adj, fwd, p, stream) : dispatch_smem_pair<4, false>(n, adj, fwd, p, stream);
    return adj.mass ? dispatch_smem_pair<5, true>(n, adj, fwd, p, stream) : dispatch_smem_pair<5, false>(n, adj, fwd, p, stream);
}

}  // namespace acpr
