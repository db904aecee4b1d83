// cnn_wgrad_tc.cu -- weight gradient of a hidden C -> C conv layer (C = 64)
// on the tensor cores:
//   dW[tap][co][ci] = sum over pixels p of dz(p, co) * a(p + off(tap), ci),
// off(tap) = (tap / 3 - 1, tap % 3 - 1) with periodic wrap, dz the gradient of
// the layer's pre-activation and a its input activation, both bf16 in the
// chunked layout [f][C/8][n][n][8].  Per tap this is a GEMM with M = co, N = ci
// and K = pixels.  In the chunked layout the 8 channels of a pixel are 16
// contiguous bytes and consecutive pixels follow each other, which is the
// "MN-major" no-swizzle core-matrix layout of the tcgen05 operands (a core
// matrix = 8 pixels x 8 channels, 128 contiguous bytes); A and B are read
// transposed (instruction descriptor bits 15 and 16), LBO = 128 bytes between
// pixel groups, SBO = the chunk-plane stride.
//
// Work unit: one activation row y of a 128-column block.  Tap row dy pairs it
// with the gradient row y + 1 - dy, so the unit's operand A is
//   rows y and y + 1 of dz side by side, M = 128 (dy = 1 and 0), and
//   row y - 1, M = 64 (dy = 2);
// dx is a shift of B's start address by one pixel.  Per 16 pixels that is three
// MMAs of 128 x 64 x 16 and three of 64 x 64 x 16 for all nine taps (one MMA of
// 64 x 64 x 16 per tap issued nine, and the pipe takes about as long for each).
// Two gradient rows are one operand when they lie in neighbouring ring slots:
// the ring has one more slot that repeats slot 0.  The bias gradient rides in
// the dx = 1 MMA: B there has two more planes, of ones, and the accumulator 16
// more columns, each sum_p dz(p, co).  One CTA per SM takes a contiguous range
// of units and keeps all accumulators in TMEM (448 columns); it reads every
// activation row and every gradient row of its range once.  The partials of the
// CTAs are summed in a fixed order, so the result is deterministic.
// Measured, a layer on 16 fields of 256^2: two CTAs per range with 5 and 4 taps
// each, M = 64, 64 ranges: 289 us; this form 127 us = 608 TFLOP/s.
//   warp 0, producer: gradient rows y - 1, y, y + 1 at a run's start, then row
//     y + 1 per unit, and activation row y (128 columns plus one pixel each
//     side, wrapped at the field's edge: bulk copy per chunk plane, wrapped
//     pixel by cp.async);
//   warp 1 (lane 0), MMA issuer: per unit 8 pixel groups, then releases the
//     activation row and the gradient row no later unit reads;
//   warps 2..5, epilogue: after the last MMA, read the accumulators and store
//     the partials.
// Every wait is bounded and sets the caller's status word when it gives up.
#include "cnn.cuh"
#include "tc_pipe.cuh"
#include "tc_ptx.cuh"

namespace acpr {

namespace {
constexpr int kWC = 64;                          // channels
constexpr int kWKC = kWC / 8;                    // chunk planes
constexpr int kWThreads = 32 * 6;                // producer, MMA, 4 epilogue warps
constexpr uint32_t kWAPlane = 130u * 16u;        // activation row: 128 pixels + 2 guard pixels
constexpr uint32_t kWASlot = (kWKC + 2) * kWAPlane;  // and two planes of ones
constexpr uint32_t kWDPlane = 128u * 16u;        // dz row: 128 pixels
constexpr uint32_t kWDSlot = kWKC * kWDPlane;
constexpr int kWRA = 5;                          // activation-row ring
constexpr int kWRD = 6;                          // dz-row ring (and one slot that repeats the first)
constexpr size_t kWCtlOff = size_t(kWRA) * kWASlot + size_t(kWRD + 1) * kWDSlot;
constexpr size_t kWSmem = kWCtlOff + 256;
// accumulator columns: dy = 0, 1 for dx = 0, 2, 1 (the last with the bias), dy = 2 for dx = 0, 1, 2
__host__ __device__ constexpr uint32_t w_col01(int dx) { return dx == 0 ? 0u : (dx == 1 ? 128u : 64u); }
__host__ __device__ constexpr uint32_t w_col2(int dx) { return 256u + 64u * uint32_t(dx); }
constexpr uint32_t kWColBias = 128 + kWC;

struct WCtl {
    uint64_t afull[kWRA], aempty[kWRA], dfull[kWRD], dempty[kWRD];
    uint64_t fin;
    uint32_t tmem;
    int abort;
};
static_assert(sizeof(WCtl) <= 256, "control block");
static_assert(kWSmem <= 227 * 1024, "shared memory");

bool g_wgrad_tc = true;
}  // namespace

void set_wgrad_tc(bool on) { g_wgrad_tc = on; }

__global__ void __launch_bounds__(kWThreads, 1)
wgrad_tc_kernel(const __nv_bfloat16* __restrict__ a, const __nv_bfloat16* __restrict__ dz, float* __restrict__ part,
                int n, int batch, int chunks, int* __restrict__ status) {
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* aring = smem;
    unsigned char* dring = smem + size_t(kWRA) * kWASlot;
    WCtl* ctl = reinterpret_cast<WCtl*>(smem + kWCtlOff);
    volatile int* abort_flag = &ctl->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ch = blockIdx.x;
    const int NB = n / 128;
    const size_t nn = size_t(n) * n;
    const long long total = (long long)batch * NB * n;
    const long long u0 = total * ch / chunks;
    const long long u1 = total * (ch + 1) / chunks;

    if (tid == 0) {
        for (int i = 0; i < kWRA; ++i) {
            tc::mbar_init(&ctl->afull[i], 1 + 32);  // byte count + the producer lanes' cp.async
            tc::mbar_init(&ctl->aempty[i], 1);
        }
        for (int i = 0; i < kWRD; ++i) {
            tc::mbar_init(&ctl->dfull[i], 1);
            tc::mbar_init(&ctl->dempty[i], 1);
        }
        tc::mbar_init(&ctl->fin, 1);
        ctl->abort = 0;
        tc::fence_mbar_init();
    }
    // the planes of ones (bf16 pairs) behind every activation row
    for (int i = tid; i < kWRA * int(2 * kWAPlane / 4); i += blockDim.x) {
        const int s = i / int(2 * kWAPlane / 4), e = i % int(2 * kWAPlane / 4);
        reinterpret_cast<uint32_t*>(aring + size_t(s) * kWASlot + kWKC * kWAPlane)[e] = 0x3F803F80u;
    }
    tc::fence_proxy_async_smem();
    if (warp == 1) tc::tmem_alloc(&ctl->tmem, 512u);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = ctl->tmem;

    if (warp == 0) {
        // ---- producer warp
        long long ja = 0, jd = 0;
        RingPos ra(kWRA), rd(kWRD);
        RowCursor cur(u0, n, NB);
        bool ok = true;
        for (long long u = u0; u < u1 && ok; ++u, cur.next()) {
            const int y = cur.y;
            const long long f = cur.f;
            const bool start = (u == u0) || (y == 0);
            const int x0 = cur.cb * 128;
            const bool wl = x0 == 0, wr = x0 + 128 == n;
            const int bx = wl ? x0 : x0 - 1;
            const uint32_t bbytes = uint32_t(130 - int(wl) - int(wr)) * 16u;
            const uint32_t boff = wl ? 16u : 0u;
            // activation row y
            {
                const int slot = ra.idx;
                bool free_slot = true;
                if (lane == 0 && ja >= kWRA) free_slot = p_wait(&ctl->aempty[slot], ra.phase ^ 1u, abort_flag, status);
                if (!__shfl_sync(0xffffffffu, free_slot, 0)) break;
                unsigned char* dst = aring + size_t(slot) * kWASlot;
                const __nv_bfloat16* src = a + (size_t(f) * kWKC * nn + size_t(y) * n) * 8;
                if (lane == 0) {
                    tc::mbar_arrive_expect_tx(&ctl->afull[slot], uint32_t(kWKC) * bbytes);
                    for (int kc = 0; kc < kWKC; ++kc)
                        tc::bulk_g2s(dst + size_t(kc) * kWAPlane + boff, src + (size_t(kc) * nn + size_t(bx)) * 8,
                                     bbytes, &ctl->afull[slot]);
                }
                if (lane < kWKC) {
                    unsigned char* d = dst + size_t(lane) * kWAPlane;
                    const __nv_bfloat16* r = src + size_t(lane) * nn * 8;
                    if (wl) cp_async16(d, r + size_t(n - 1) * 8);
                    if (wr) cp_async16(d + 129 * 16, r);
                }
                cp_async_arrive(&ctl->afull[slot]);
                ++ja;
                ra.next();
            }
            // gradient rows y - 1, y, y + 1 or y + 1
            for (int k = start ? 0 : 2; k < 3; ++k) {
                int yin = y - 1 + k;
                yin = yin < 0 ? yin + n : (yin >= n ? yin - n : yin);
                const int slot = rd.idx;
                bool free_slot = true;
                if (lane == 0 && jd >= kWRD) free_slot = p_wait(&ctl->dempty[slot], rd.phase ^ 1u, abort_flag, status);
                if (!__shfl_sync(0xffffffffu, free_slot, 0)) {
                    ok = false;
                    break;
                }
                if (lane == 0) {
                    const __nv_bfloat16* src = dz + (size_t(f) * kWKC * nn + size_t(yin) * n + size_t(x0)) * 8;
                    const int copies = slot == 0 ? 2 : 1;  // slot 0 also behind the last one
                    tc::mbar_arrive_expect_tx(&ctl->dfull[slot], uint32_t(copies) * kWDSlot);
                    for (int c = 0; c < copies; ++c) {
                        unsigned char* dst = dring + size_t(c ? kWRD : slot) * kWDSlot;
                        for (int kc = 0; kc < kWKC; ++kc)
                            tc::bulk_g2s(dst + size_t(kc) * kWDPlane, src + size_t(kc) * nn * 8, kWDPlane,
                                         &ctl->dfull[slot]);
                    }
                }
                ++jd;
                rd.next();
            }
        }
        // drain: every issued copy lands before the CTA may exit
        if (lane == 0) {
            for (long long x = ja > kWRA ? ja - kWRA : 0; x < ja; ++x)
                tc::mbar_wait_bounded(&ctl->afull[x % kWRA], uint32_t((x / kWRA) & 1), kTcSpin);
            for (long long x = jd > kWRD ? jd - kWRD : 0; x < jd; ++x)
                tc::mbar_wait_bounded(&ctl->dfull[x % kWRD], uint32_t((x / kWRD) & 1), kTcSpin);
        }
        cp_async_wait_all();
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer
            // bf16 A and B, f32 D, both operands MN-major (transposed)
            constexpr uint32_t tr = (1u << 15) | (1u << 16);
            constexpr uint32_t id01 = tc::idesc_bf16_f32(128, kWC) | tr, id01b = tc::idesc_bf16_f32(128, kWC + 16) | tr;
            constexpr uint32_t id2 = tc::idesc_bf16_f32(64, kWC) | tr;
            const uint64_t a_hi = tc::smem_desc(0, 128, kWDPlane);  // A = dz rows
            const uint64_t b_hi = tc::smem_desc(0, 128, kWAPlane);  // B = activation rows
            const uint32_t aring_u = tc::smem_u32(aring) >> 4, dring_u = tc::smem_u32(dring) >> 4;
            RingPos ra(kWRA), rd(kWRD);
            int pos[3] = {0, 0, 0};  // ring slots of the gradient rows y - 1, y, y + 1
            bool ok = true;
            uint32_t acc = 0;
            int y = int(u0 % n);
            for (long long u = u0; u < u1 && ok; ++u, y = (y + 1 == n ? 0 : y + 1)) {
                const bool start = (u == u0) || (y == 0);
                pos[0] = pos[1];
                pos[1] = pos[2];
                for (int k = start ? 0 : 2; k < 3 && ok; ++k) {
                    pos[k] = rd.idx;
                    ok = p_wait(&ctl->dfull[rd.idx], rd.phase, abort_flag, status);
                    rd.next();
                }
                if (ok) ok = p_wait(&ctl->afull[ra.idx], ra.phase, abort_flag, status);
                if (!ok) break;
                // the wrapped pixels came by cp.async (generic proxy); the MMAs read through the async proxy
                tc::fence_proxy_async_smem();
                tc::fence_after_sync();
                const uint32_t d01 = dring_u + uint32_t(pos[1]) * (kWDSlot >> 4);  // rows y, y + 1: slot pos[1] and the next
                const uint32_t d2 = dring_u + uint32_t(pos[0]) * (kWDSlot >> 4);
                const uint32_t r_u = aring_u + uint32_t(ra.idx) * (kWASlot >> 4);
#pragma unroll 1
                for (int kg = 0; kg < 8; ++kg) {
                    const uint64_t a01 = a_hi | uint64_t(d01 + uint32_t(kg * 16));
                    const uint64_t a2 = a_hi | uint64_t(d2 + uint32_t(kg * 16));
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        const uint64_t bd = b_hi | uint64_t(r_u + uint32_t(kg * 16 + dx));
                        tc::mma_bf16(tmem + w_col01(dx), a01, bd, dx == 1 ? id01b : id01, acc);
                        tc::mma_bf16(tmem + w_col2(dx), a2, bd, id2, acc);
                    }
                    acc = 1;
                }
                tc::mma_commit(&ctl->aempty[ra.idx]);
                ra.next();
                // row y - 1 is read by no later unit; at the end of a run neither are y, y + 1
                const bool cont = (u + 1 < u1) && (y + 1 != n);
                tc::mma_commit(&ctl->dempty[pos[0]]);
                if (!cont) {
                    tc::mma_commit(&ctl->dempty[pos[1]]);
                    tc::mma_commit(&ctl->dempty[pos[2]]);
                }
            }
            // every MMA issued completes before the accumulators are read and TMEM is freed
            tc::mma_commit(&ctl->fin);
            if (!ok) *abort_flag = 1;
        }
    } else {
        // ---- epilogue: the accumulators -> partials
        const int q = warp & 3;
        const bool ok = tc::mbar_wait_bounded(&ctl->fin, 0, kTcSpin);
        if (!ok) atomicExch(status, 3);
        tc::fence_after_sync();
        if (ok && !*abort_flag) {
            constexpr size_t kTapFloats = kWC * kWC + kWC;
            float* base = part + size_t(ch) * 9 * kTapFloats;
            auto store = [&](uint32_t col, int tap, int co, bool valid) {
                float* dst = base + size_t(tap) * kTapFloats + size_t(co) * kWC;
#pragma unroll 1
                for (int c0 = 0; c0 < kWC; c0 += 8) {
                    uint32_t v[8];
                    tc::tmem_ld8(tmem + (uint32_t(q * 32) << 16) + col + uint32_t(c0), v);
                    tc::tmem_wait_ld();
                    if (valid) {
                        reinterpret_cast<float4*>(dst + c0)[0] =
                            make_float4(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]),
                                        __uint_as_float(v[3]));
                        reinterpret_cast<float4*>(dst + c0)[1] =
                            make_float4(__uint_as_float(v[4]), __uint_as_float(v[5]), __uint_as_float(v[6]),
                                        __uint_as_float(v[7]));
                    }
                }
            };
            // M = 128: lane m holds row m (m < 64: dy = 1, else dy = 0); M = 64: rows 16 q .. 16 q + 15 in lanes 32 q ..
            const int m = 32 * q + lane;
            for (int dx = 0; dx < 3; ++dx) {
                store(w_col01(dx), (m < kWC ? 3 : 0) + dx, m & (kWC - 1), true);
                store(w_col2(dx), 6 + dx, 16 * q + (lane & 15), lane < 16);
            }
            uint32_t v[8];
            tc::tmem_ld8(tmem + (uint32_t(q * 32) << 16) + kWColBias, v);
            tc::tmem_wait_ld();
            if (m < kWC) base[kWC * kWC + m] = __uint_as_float(v[0]);  // sum of dz over the rows y (dy = 1)
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        // the MMA issuer's own completion wait (also when the epilogue gave up)
        if (lane == 0) tc::mbar_wait_bounded(&ctl->fin, 0, kTcSpin);
        __syncwarp();
        tc::tmem_dealloc(tmem, 512u);
    }
}

bool wgrad_tc_supported(int C, int n) { return g_wgrad_tc && C == kWC && n >= 128 && n % 128 == 0 && n <= 1024; }

int wgrad_tc_partials(int n, int batch, const __nv_bfloat16* a, const __nv_bfloat16* dz, float* part, int chunks,
                      int* status, cudaStream_t st) {
    if (!status) {
        set_error("tensor-core weight gradient: no status word");
        return AC_ERR_ARG;
    }
    static DeviceSet configured;
    const int rc = once_per_device(configured, [] { return allow_smem(wgrad_tc_kernel, kWSmem); });
    if (rc) return rc;
    wgrad_tc_kernel<<<chunks, kWThreads, kWSmem, st>>>(a, dz, part, n, batch, chunks, status);
    ACPR_LAUNCH_CHECK();
    return AC_OK;
}

}  // namespace acpr

extern "C" int cnn_train_set_wgrad_tc(int on) {
    acpr::set_wgrad_tc(on != 0);
    return AC_OK;
}
