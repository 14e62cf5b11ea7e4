// Convolution whose operands are exact sums of bf16 planes, on the tcgen05
// tensor cores: fp32 (three planes) and qint8 (one plane) implicit GEMM, NHWC.
//
//   fp32   2^24 x = x0 + x1 + x2 with x0 = bf16(2^24 x), x1 and x2 likewise of what
//          is left: 8 + 8 + 8 significant bits, so the sum is exact for every
//          |x| < 2^104 (unscaled, the last planes of an x below 2^-110 would fall
//          under bf16's smallest value).  The sums, 2^48 times the result, are
//          scaled back exactly; operands and sums too large for the planes are
//          recomputed (plain_sum).  Of the nine
//          plane products the six with i + j <= 2 are formed, each i + j in an
//          accumulator of its own; the dropped ones are below 2^-26 of |x w|.
//          With 64-channel tiles the planes of B lie behind one another as rows
//          of one operand: x0 [w0 w1 w2], x1 [w0 w1] and x2 [w0] are three MMAs
//          of N = 192, 128 and 64 whose columns land on the accumulator of
//          their i + j (an MMA of N = 64 alone takes as long to issue as one of
//          N = 128).  128-channel tiles take six MMAs and two accumulators
//          (x0 w0, the small products).
//   qint8  a code in [-127, 127] is a bf16 value, and a sum of at most 1024
//          code products stays below 2^24, so the fp32 accumulator holds the
//          integer sum exactly.
// Either way the accumulators are drained every few K steps and added up in
// registers (fp32 round-to-nearest, or int32): the tensor core's own
// accumulation does not round to nearest, and its error grows with the number
// of steps, not with their square root.
//
// Two launches: a kernel splits the activations into planes [planes][N H W][Cp]
// (Cp = C rounded up to 8; any C), then the persistent GEMM walks tiles of 128
// output pixels x BN channels.  A stage holds one 64-channel block of one tap:
// all planes of A as one TMA box and all planes of B as another (a box costs
// about the same whatever its size), so the six products of a stage read three
// + three staged blocks.  Warp 0 issues the copies (the first stages' weights
// before the dependency wait), warp 1 the MMAs, warps 2-9 drain: TMEM ->
// registers, and after a tile's last chunk bias, residual, activation or
// requantisation and 16-byte stores of a thread's own row (32 or 64 consecutive
// channels).  No staging: its 32 KB are a third fp32 stage, without which a
// stage's copy was exposed once its MMAs were done.
// What bounds it: 24 MMAs of K = 16 per stage and fp32 tile (six products),
// i.e. a sixth of the bf16 rate, against the FFMA rate that the CUDA-core
// routines stay below; small layers are bound by latency.  Every wait is
// bounded as in tc_conv.cuh.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <string>
#include <type_traits>
#include <vector>

#include "q8_common.cuh"
#include "tc_common.cuh"

namespace sn {
namespace k {
namespace tcs {

using namespace tc;

constexpr int SPLIT_THREADS = 320;  // producer, MMA issuer, eight epilogue warps
// K steps (64 values) per accumulator drain.  The tensor core truncates each
// accumulation of 16 products, an error of one sign where the products are: 128
// values a drain keep operands of one sign below the fp32 routines' error (256 ->
// 64 channels, 1x1, all positive: 1.6e-7 of the result, igemm_simt 2.2e-7; 256
// values a drain: 3.5e-7; the bottleneck at batch 8: 52.0 -> 53.2 us).  1024 code
// products stay exact in qint8.
constexpr int chunk_of(int planes) { return planes == 3 ? 2 : 16; }

struct SParams {
    int32_t N, H, W, C, K, P, Q, R, S;       // the layer (fix-up and output addressing)
    int32_t stride, ph, pw, dh, dw;
    int32_t Cp, cblocks, kiters;             // padded channels; 64-channel blocks; K steps per tile
    int32_t BW, BH, BNI, tq, tp, mtiles, ntiles, lbw, lbwh;
    int32_t gP, gQ, gN, gph, gpw;            // the pixel grid the tiles cover (plain layers: one row of N H W pixels)
    FastDiv fd_tq, fd_tp, fd_nt;
    const float *bias;
    void *y;
    const void *res;
    int *err;
    long long wait_limit;
    int32_t act, vec;                        // vec: output (and residual) accesses of 16 bytes (2), four elements (1), one (0)
    const float *x32, *w32;                  // fp32: the operands themselves (x NHWC, w [K][R*S][C])
    const float *ws;                         // qint8: weight scales
    float s_x, s_r, inv_out;
};

// the planes are those of SCALE * x and SCALE * w
constexpr float SCALE = 16777216.0f, UNSCALE = 1.0f / SCALE / SCALE;

// the sum of one output element in plain fp32, for one that the planes cannot
// carry: an infinity or a NaN among the operands (the planes of an infinity
// are inf, NaN, NaN), an operand from 2^104 on, or sums from 2^80 on
__device__ __noinline__ float plain_sum(const SParams &p, int64_t pix, int k) {
    const int q = (int)(pix % p.Q), pp = (int)((pix / p.Q) % p.P);
    const int64_t n = pix / ((int64_t)p.Q * p.P);
    float acc = 0.f;
    for (int r = 0; r < p.R; ++r) {
        const int h = pp * p.stride - p.ph + r * p.dh;
        if (h < 0 || h >= p.H) continue;
        for (int s = 0; s < p.S; ++s) {
            const int w = q * p.stride - p.pw + s * p.dw;
            if (w < 0 || w >= p.W) continue;
            const float *xp = p.x32 + ((n * p.H + h) * p.W + w) * p.C;
            const float *wp = p.w32 + ((int64_t)k * p.R * p.S + r * p.S + s) * p.C;
            for (int c = 0; c < p.C; ++c) acc = fmaf(xp[c], wp[c], acc);
        }
    }
    return acc;
}

template <int PLANES, int BN>
struct Lay {
    static constexpr uint32_t A_PL = BM * BK * 2, B_PL = BN * BK * 2;
    static constexpr uint32_t A_BYTES = PLANES * A_PL, STAGE = A_BYTES + PLANES * B_PL;
    static constexpr int STAGES = (226 * 1024 - 2048) / (int)STAGE < 8 ? (226 * 1024 - 2048) / (int)STAGE : 8;
    static constexpr bool STACK = PLANES == 3 && BN == 64;          // planes of B as rows of one operand
    static constexpr int ACC = PLANES == 1 ? 1 : STACK ? 3 : 2;     // accumulators per buffer
    static constexpr int BUF = STACK ? 256 : ACC * BN;              // TMEM columns from one buffer to the other
    static constexpr uint32_t COLS = 2 * BUF;
    static constexpr size_t SMEM = (size_t)STAGES * STAGE + 1024;
    static_assert(STAGES >= 2 && COLS <= 512, "stage ring and TMEM");
};

// TO: float (PLANES = 3), or the output type of a qint8 routine (PLANES = 1)
template <int PLANES, int BN, typename TO>
__global__ void __launch_bounds__(SPLIT_THREADS, 1)
    conv_split_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                      const __grid_constant__ CUtensorMap mA2, const __grid_constant__ CUtensorMap mA3,
                      const __grid_constant__ CUtensorMap mB, const __grid_constant__ SParams p) {
    using L = Lay<PLANES, BN>;
    constexpr int STAGES = L::STAGES, CH = chunk_of(PLANES);
    constexpr bool F32 = PLANES == 3;
    using Acc = typename std::conditional<F32, float, int>::type;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES];
    __shared__ __align__(8) uint64_t empty_bar[STAGES];
    __shared__ __align__(8) uint64_t accf_bar[2];
    __shared__ __align__(8) uint64_t acce_bar[2];
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_sh;
    __shared__ int issued_sh, consumed_sh;

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int total = p.mtiles * p.ntiles;
    const int nchunks = (p.kiters + CH - 1) / CH;
    if (threadIdx.x == 32) {  // the maps are kernel parameters, not data of the previous kernel
        const CUtensorMap *maps[5] = {&mB, &mA0, &mA1, &mA2, &mA3};
        for (int i = 0; i < (p.stride == 1 ? 2 : 5); ++i)
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(maps[i])) : "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf_bar[b], 1);
            mbar_init(&acce_bar[b], EPI_WARPS);
        }
        abort_sh = 0;
        issued_sh = consumed_sh = 0;
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc<1>(&tmem_sh, L::COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    griddep_launch();  // (behind the allocation: see tmem_alloc)
    // tile t: output channels n0.., pixel box at (q0, p0, i0)
    auto tile = [&](int t, int &n0, int &q0, int &p0, int &i0) {
        const int mt = (int)fdiv((uint32_t)t, p.fd_nt);
        n0 = (t - mt * p.ntiles) * BN;
        const int a = (int)fdiv((uint32_t)mt, p.fd_tq), b = (int)fdiv((uint32_t)a, p.fd_tp);
        q0 = (mt - a * p.tq) * p.BW;
        p0 = (a - b * p.tp) * p.BH;
        i0 = b * p.BNI;
    };
    if (warp == 0) {
        if (lane == 0) {  // ---------------- TMA producer
            int g = 0, s = 0;
            uint32_t par = 0;
            bool stop = false;
            // the weights of the first stages: not written by the previous kernel
            const int early = (int)blockIdx.x < total ? min(STAGES, p.kiters) : 0;
            {
                int n0, q0, p0, i0, tap = 0, cb = 0;
                tile((int)blockIdx.x, n0, q0, p0, i0);
                for (int i = 0; i < early; ++i) {
                    mbar_expect_tx(&full_bar[i], L::STAGE);
                    tma_4d<1>(su32(smem + i * L::STAGE) + L::A_BYTES, &mB, su32(&full_bar[i]), cb * BK, tap, n0, 0);
                    if (++cb == p.cblocks) {
                        cb = 0;
                        ++tap;
                    }
                }
            }
            griddep_wait();
            for (int t = blockIdx.x; t < total && !stop; t += gridDim.x) {
                int n0, q0, p0, i0;
                tile(t, n0, q0, p0, i0);
                int tap = 0, cb = 0, r = 0, ss = 0;
                for (int it = 0; it < p.kiters; ++it, ++g) {
                    if (!mbar_wait(&empty_bar[s], par ^ 1u, p.wait_limit)) {
                        atomicOr(p.err, ERR_TMA_WAIT);
                        abort_sh = 1;
                    }
                    // (a stage whose weights are on their way gets its activations whatever happened)
                    if (abort_sh && g >= early) {
                        stop = true;
                        break;
                    }
                    const uint32_t sa = su32(smem + s * L::STAGE), bar = su32(&full_bar[s]);
                    if (g >= early) mbar_expect_tx(&full_bar[s], L::STAGE);
                    const int oh = r * p.dh - p.gph, ow = ss * p.dw - p.gpw;
                    const CUtensorMap *m = &mA0;
                    int qa = q0 + ow, pa = p0 + oh;
                    if (p.stride != 1) {  // the even/odd row and column sub-lattices
                        const int bh = oh & 1, bw = ow & 1;
                        m = bh ? (bw ? &mA3 : &mA2) : (bw ? &mA1 : &mA0);
                        qa = q0 + ((ow - bw) >> 1);
                        pa = p0 + ((oh - bh) >> 1);
                    }
                    tma_5d<1>(sa, m, bar, cb * BK, qa, pa, i0, 0);
                    if (g >= early) tma_4d<1>(sa + L::A_BYTES, &mB, bar, cb * BK, tap, n0, 0);
                    issued_sh = g + 1;
                    if (++s == STAGES) {
                        s = 0;
                        par ^= 1u;
                    }
                    if (++cb == p.cblocks) {
                        cb = 0;
                        ++tap;
                        if (++ss == p.S) {
                            ss = 0;
                            ++r;
                        }
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {  // ---------------- MMA issuer
            const uint32_t idesc = idesc_f16<__nv_bfloat16>(BM, BN);
            const uint64_t desc0 = sdesc_sw128(su32(smem));
            int g = 0, s = 0, u = 0;  // u: accumulator buffer uses
            uint32_t par = 0;
            bool stop = false;
            for (int t = blockIdx.x; t < total && !stop; t += gridDim.x) {
                int cb = 0;
                for (int it = 0; it < p.kiters; ++it, ++g) {
                    const int b = u & 1;
                    const bool first = it % CH == 0;
                    if (first && !mbar_wait(&acce_bar[b], ((uint32_t)(u >> 1) & 1u) ^ 1u, p.wait_limit)) {
                        atomicOr(p.err, ERR_EPI_WAIT);
                        abort_sh = 1;
                        stop = true;
                    }
                    // (no look at abort_sh: a shared-memory access of this thread
                    // queues behind the MMAs' operand reads, ~200 cycles)
                    if (!stop && !mbar_wait(&full_bar[s], par, p.wait_limit)) {
                        atomicOr(p.err, ERR_MMA_WAIT);
                        abort_sh = 1;
                        stop = true;
                    }
                    if (stop) break;
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(b * L::BUF);
                    const uint64_t da = desc0 + (uint64_t)((s * L::STAGE) >> 4), db = da + (L::A_BYTES >> 4);
                    // 16-value steps of this block that hold channels (the rest is zero fill)
                    const int ks = min(BK / 16, (p.Cp - cb * BK + 15) / 16);
                    if constexpr (L::STACK) {
                        const uint32_t id3 = idesc_f16<__nv_bfloat16>(BM, 3 * BN), id2 = idesc_f16<__nv_bfloat16>(BM, 2 * BN);
                        auto step = [&](int k) {
                            umma<1>(d, da + 2 * k, db + 2 * k, id3, (!first || k > 0) ? 1u : 0u);
                            umma<1>(d + BN, da + (L::A_PL >> 4) + 2 * k, db + 2 * k, id2, 1u);
                            umma<1>(d + 2 * BN, da + 2 * (L::A_PL >> 4) + 2 * k, db + 2 * k, idesc, 1u);
                        };
                        if (ks == BK / 16) {
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k) step(k);
                        } else {
                            for (int k = 0; k < ks; ++k) step(k);
                        }
                    } else if constexpr (F32) {
                        // small products first within the block; each accumulator sums in its own order
                        constexpr int I[6] = {0, 1, 2, 0, 1, 0}, J[6] = {2, 1, 0, 1, 0, 0};
#pragma unroll
                        for (int e = 0; e < 6; ++e)
                            for (int k = 0; k < ks; ++k)
                                umma<1>(e == 5 ? d : d + BN, da + I[e] * (L::A_PL >> 4) + 2 * k,
                                        db + J[e] * (L::B_PL >> 4) + 2 * k, idesc,
                                        (!first || k > 0 || (e > 0 && e < 5)) ? 1u : 0u);
                    } else if (ks == BK / 16) {
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) umma<1>(d, da + 2 * k, db + 2 * k, idesc, (!first || k > 0) ? 1u : 0u);
                    } else {
                        for (int k = 0; k < ks; ++k) umma<1>(d, da + 2 * k, db + 2 * k, idesc, (!first || k > 0) ? 1u : 0u);
                    }
                    umma_commit<1>(&empty_bar[s]);
                    if ((it + 1) % CH == 0 || it + 1 == p.kiters) {
                        umma_commit<1>(&accf_bar[b]);
                        ++u;
                    }
                    if (++s == STAGES) {
                        s = 0;
                        par ^= 1u;
                    }
                    if (++cb == p.cblocks) cb = 0;
                }
            }
            consumed_sh = g;
        }
    } else {  // ---------------- epilogue: warps 2..9
        constexpr int HC = BN / 2;  // columns of this warp: half of the tile's
        const int half = (warp - 2) >> 2, g4 = warp & 3;
        const int tr = g4 * 32 + lane;  // this thread's row of the tile
        int u = 0;
        bool stop = false;
        griddep_wait();
        for (int t = blockIdx.x; t < total && !stop; t += gridDim.x) {
            int n0, q0, p0, i0;
            tile(t, n0, q0, p0, i0);
            const int q = q0 + (tr & (p.BW - 1)), pp = p0 + ((tr >> p.lbw) & (p.BH - 1)), n = i0 + (tr >> p.lbwh);
            const bool live = q < p.gQ && pp < p.gP && n < p.gN;
            const int64_t pix = live ? ((int64_t)n * p.gP + pp) * p.gQ + q : 0;
            // rows are handled by pairs of lanes when they are stored
            const bool live2 = __shfl_xor_sync(0xffffffffu, (int)live, 1);
            const int64_t pix2 = __shfl_xor_sync(0xffffffffu, (long long)pix, 1);
            if (F32 && p.res && live)  // its residual, on its way into L1 while the tile is accumulated
                for (int e = 0; e < HC && n0 + half * HC + e < p.K; e += 32)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(static_cast<const float *>(p.res) + pix * p.K + n0 + half * HC + e));
            Acc acc[HC];
#pragma unroll
            for (int e = 0; e < HC; ++e) acc[e] = 0;
            for (int c = 0; c < nchunks; ++c, ++u) {
                const int b = u & 1;
                const bool ok = mbar_wait(&accf_bar[b], (uint32_t)(u >> 1) & 1u, p.wait_limit);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) atomicOr(p.err, ERR_ACC_WAIT);
                    abort_sh = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                __syncwarp();
                const uint32_t ta = tmem + ((uint32_t)(g4 * 32) << 16) + (uint32_t)(b * L::BUF + half * HC);
#pragma unroll
                for (int j = 0; j < HC; j += 32) {
                    uint32_t v[32];
                    tmem_ld32(ta + j, v);
                    if constexpr (F32) {
                        uint32_t lo[32];
                        tmem_ld32(ta + BN + j, lo);
                        if constexpr (L::STACK) {
                            uint32_t l2[32];
                            tmem_ld32(ta + 2 * BN + j, l2);
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                lo[e] = __float_as_uint(__uint_as_float(lo[e]) + __uint_as_float(l2[e]));
                        }
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[j + e] += __uint_as_float(v[e]) + __uint_as_float(lo[e]);
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[j + e] += __float2int_rn(__uint_as_float(v[e]));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce_bar[b]);
            }
            if (stop) break;
            using TR = typename std::conditional<F32, float, int8_t>::type;  // residual element
            constexpr int G = 16;                                             // channels at a time
            // one 16-byte piece, four elements or one element at a time, as K and the bases allow
            auto group = [&](auto jc, auto epv) {
                constexpr int j = decltype(jc)::value;
                constexpr int EV = decltype(epv)::value;
                const int k = n0 + half * HC + j;
                const int64_t o0 = pix * p.K + k;
                float rv[G];
#pragma unroll
                for (int e = 0; e < G; ++e) rv[e] = 0.f;
                if (p.res && live) {
                    constexpr int ER = EV == 1 ? 1 : EV == 4 ? 4 : 16 / (int)sizeof(TR);
                    const TR *res = static_cast<const TR *>(p.res) + o0;
#pragma unroll
                    for (int e = 0; e < G; e += ER) {
                        if (k + e >= p.K) break;
                        const Vec<TR, ER> r = *reinterpret_cast<const Vec<TR, ER> *>(res + e);
#pragma unroll
                        for (int i = 0; i < ER; ++i) rv[e + i] = F32 ? (float)r.v[i] : __fmul_rn((float)r.v[i], p.s_r);
                    }
                }
                float bv[G];
                [[maybe_unused]] float sv[G];
#pragma unroll
                for (int e = 0; e < G; e += 4) {  // (the bias is zero-padded to a multiple of 256 channels)
                    const float4 b4 = __ldg(reinterpret_cast<const float4 *>(p.bias + k + e));
                    bv[e] = b4.x, bv[e + 1] = b4.y, bv[e + 2] = b4.z, bv[e + 3] = b4.w;
                    if constexpr (!F32) {  // (qint8: K is a multiple of four)
                        const float4 s4 = k + e < p.K ? __ldg(reinterpret_cast<const float4 *>(p.ws + k + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        sv[e] = s4.x, sv[e + 1] = s4.y, sv[e + 2] = s4.z, sv[e + 3] = s4.w;
                    }
                }
                TO o[G];
                if constexpr (F32) {
#pragma unroll
                    for (int e = 0; e < G; ++e) acc[j + e] *= UNSCALE;
                    // one test for the group: an infinity or a NaN has all exponent bits
                    bool odd_value = false;
#pragma unroll
                    for (int e = 0; e < G; ++e) odd_value |= (__float_as_uint(acc[j + e]) & 0x7f800000u) == 0x7f800000u;
                    if (odd_value && live) {
#pragma unroll
                        for (int e = 0; e < G; ++e)
                            if (k + e < p.K && !isfinite(acc[j + e])) acc[j + e] = plain_sum(p, pix, k + e);
                    }
                }
                auto finish = [&](auto act) {
#pragma unroll
                    for (int e = 0; e < G; ++e) {
                        if constexpr (F32) o[e] = act(acc[j + e] + bv[e] + rv[e]);
                        else o[e] = q8_out<TO>(act(__fadd_rn(__fadd_rn(__fmul_rn(__int2float_rn(acc[j + e]), __fmul_rn(p.s_x, sv[e])), bv[e]), rv[e])), p.inv_out);
                    }
                };
                if (p.act == SN_ACT_RELU || p.act == SN_ACT_RELU6)
                    finish([hi = p.act == SN_ACT_RELU ? INFINITY : 6.0f](float x) { return fminf(fmaxf(x, 0.0f), hi); });
                else if (p.act == SN_ACT_NONE)
                    finish([](float x) { return x; });
                else
                    finish([act = p.act](float x) {
                        if constexpr (F32) return act_apply(x, act);
                        else return q8_act(x, act);
                    });
                if constexpr (F32 && EV == 16) {
                    // 32 contiguous bytes of a row per pair of lanes: the even lane
                    // stores the first half of its own row, then of its neighbour's,
                    // the odd lane the second halves (16-byte stores of 32 different
                    // rows fill half a sector each)
                    const bool odd = lane & 1;
                    float *ya = static_cast<float *>(p.y) + (odd ? pix2 : pix) * p.K + k;   // the pair's even row
                    float *yb = static_cast<float *>(p.y) + (odd ? pix : pix2) * p.K + k;   // its odd row
                    const bool la = odd ? live2 : live, lb = odd ? live : live2;
#pragma unroll
                    for (int e = 0; e < G; e += 8) {
                        float got[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) got[i] = __shfl_xor_sync(0xffffffffu, odd ? o[e + i] : o[e + 4 + i], 1);
                        const int at = e + (odd ? 4 : 0);
                        if (k + at >= p.K) continue;
                        const float4 a = odd ? make_float4(got[0], got[1], got[2], got[3])
                                             : make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
                        const float4 b = odd ? make_float4(o[e + 4], o[e + 5], o[e + 6], o[e + 7])
                                             : make_float4(got[0], got[1], got[2], got[3]);
                        if (la) *reinterpret_cast<float4 *>(ya + at) = a;
                        if (lb) *reinterpret_cast<float4 *>(yb + at) = b;
                    }
                    return;
                }
                if (!live) return;
                TO *yo = static_cast<TO *>(p.y) + o0;
                constexpr int EO = EV == 1 ? 1 : EV == 4 ? 4 : 16 / (int)sizeof(TO);
#pragma unroll
                for (int e = 0; e < G; e += EO) {
                    if (k + e >= p.K) break;
                    Vec<TO, EO> w;
#pragma unroll
                    for (int i = 0; i < EO; ++i) w.v[i] = o[e + i];
                    *reinterpret_cast<Vec<TO, EO> *>(yo + e) = w;
                }
            };
            auto groups = [&](auto jc) {
                if (n0 + half * HC + decltype(jc)::value >= p.K) return;
                if (p.vec == 2) group(jc, std::integral_constant<int, 16>{});
                else if (p.vec == 1) group(jc, std::integral_constant<int, 4>{});
                else group(jc, std::integral_constant<int, 1>{});
            };
            groups(std::integral_constant<int, 0>{});
            groups(std::integral_constant<int, 16>{});
            if constexpr (HC == 64) {
                groups(std::integral_constant<int, 32>{});
                groups(std::integral_constant<int, 48>{});
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        if (abort_sh && lane == 0) {
            // let this CTA's copies and MMAs land before its memory goes away
            // (one deadline for the whole drain)
            const long long t0 = clock64();
            for (int g = consumed_sh; g < issued_sh; ++g)
                while (!mbar_try(&full_bar[g % STAGES], (uint32_t)(g / STAGES) & 1u) && clock64() - t0 < WAIT_LIMIT) {
                }
            if (consumed_sh > 0) {
                const int g = consumed_sh - 1;
                while (!mbar_try(&empty_bar[g % STAGES], (uint32_t)(g / STAGES) & 1u) && clock64() - t0 < WAIT_LIMIT) {
                }
            }
        }
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, L::COLS);
    }
}

// ------------------------------------------------------- operand planes
// the three bf16 planes of SCALE times an fp32 value
__device__ __forceinline__ void planes_of(float x, __nv_bfloat16 (&o)[3]) {
    x *= SCALE;
    o[0] = __float2bfloat16_rn(x);
    const float r = x - __bfloat162float(o[0]);
    o[1] = __float2bfloat16_rn(r);
    o[2] = __float2bfloat16_rn(r - __bfloat162float(o[1]));
}

// x [pixels][C] -> planes [PLANES][pixels][Cp], eight channels per thread, zero
// past C.  Memory bound: 4 C bytes read and 6 Cp written per fp32 pixel.
template <int PLANES, typename TI>
__global__ void __launch_bounds__(256) split_kernel(const TI *__restrict__ x, __nv_bfloat16 *__restrict__ o, uint32_t total,
                                                    int C, FastDiv fd_c8, int64_t plane, bool vec) {
    griddep_launch();
    griddep_wait();
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const uint32_t pix = fdiv(t, fd_c8);
    const int c0 = (int)(t - pix * fd_c8.d) * 8;
    const TI *xp = x + (int64_t)pix * C + c0;
    Vec<TI, 8> v;
    if (vec) {  // C % 8 == 0 and an aligned base
        v = *reinterpret_cast<const Vec<TI, 8> *>(xp);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v.v[e] = c0 + e < C ? xp[e] : TI(0);
    }
    Vec<__nv_bfloat16, 8> w[PLANES];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if constexpr (PLANES == 3) {
            __nv_bfloat16 pl[3];
            planes_of((float)v.v[e], pl);
#pragma unroll
            for (int i = 0; i < 3; ++i) w[i].v[e] = pl[i];
        } else {
            w[0].v[e] = __float2bfloat16_rn((float)v.v[e]);  // a code: exact
        }
    }
#pragma unroll
    for (int i = 0; i < PLANES; ++i) *reinterpret_cast<Vec<__nv_bfloat16, 8> *>(o + i * plane + (int64_t)t * 8) = w[i];
}

// weights, from fp32 [K][C][RS]: planes [PLANES][K][RS][Cp] and, fp32, the
// weights themselves as [K][RS][C] behind them
template <int PLANES>
__global__ void weight_split_kernel(const float *__restrict__ w, const float *__restrict__ scale,
                                    __nv_bfloat16 *__restrict__ o, float *__restrict__ w32, int64_t K, int64_t C,
                                    int64_t RS, int64_t Cp) {
    griddep_launch();
    griddep_wait();
    const int64_t total = K * RS * Cp;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = i % Cp, rs = (i / Cp) % RS, kk = i / (Cp * RS);
        const float v = c < C ? w[(kk * C + c) * RS + rs] : 0.f;
        if constexpr (PLANES == 3) {
            __nv_bfloat16 pl[3];
            planes_of(v, pl);
            for (int j = 0; j < 3; ++j) o[j * total + i] = pl[j];
            if (c < C) w32[(kk * RS + rs) * C + c] = v;
        } else {
            o[i] = __float2bfloat16_rn((float)q8_weight_code(v, scale[kk]));
        }
    }
}

// ------------------------------------------------------------- host side
struct SConfig {
    int BN, BW, BH, BNI;
    bool plain;
};

static int64_t padded_c(int64_t c) { return (c + 7) / 8 * 8; }

// tile parameters for a layer: output-channel tile 64 or 128, and for layers
// that are not a plain GEMM the one or two pixel boxes of 128 that waste least
static std::vector<SConfig> split_configs(const Layer &l, const Shape &in, sn_schema s) {
    std::vector<SConfig> out;
    const sn_conv_params &c = l.conv;
    if (l.type != SN_L_CONV2 || c.groups != 1 || s.layout != SN_NHWC || (s.dtype != SN_F32 && s.dtype != SN_QI8)) return out;
    if (c.sh != c.sw || (c.sh != 1 && c.sh != 2) || (c.sh == 2 && (in.h < 2 || in.w < 2))) return out;
    if (s.dtype == SN_QI8 && (in.c % 4 || c.c_out % 4)) return out;  // the layers of the dp4a routine
    const int64_t pixels = in.n * in.h * in.w, M = l.out.n * l.out.h * l.out.w;
    // 32-bit work indices and tensor-map extents
    if (pixels * padded_c(in.c) / 8 >= ((int64_t)1 << 31) || M >= ((int64_t)1 << 31) || c.c_out > MAX_K ||
        c.kh * c.kw > 65536 || (M / 128 + 65536) * ((c.c_out + 63) / 64) >= ((int64_t)1 << 31))
        return out;
    std::vector<int> bns = {64};
    if (c.c_out > 64) bns.push_back(128);
    const bool plain = c.kh == 1 && c.kw == 1 && c.sh == 1 && c.ph == 0 && c.pw == 0;
    if (plain) {
        for (int bn : bns) out.push_back({bn, 128, 1, 1, true});
        return out;
    }
    struct Geo {
        double waste;
        int bw, bh, bni;
    };
    std::vector<Geo> gs;
    const int64_t N = l.out.n, P = l.out.h, Q = l.out.w;
    for (int bw = 1; bw <= BM; bw *= 2)
        for (int bh = 1; bw * bh <= BM; bh *= 2) {
            const int bni = BM / (bw * bh);
            const double cover = (double)((Q + bw - 1) / bw * bw) * ((P + bh - 1) / bh * bh) * ((N + bni - 1) / bni * bni);
            gs.push_back({cover / (double)(N * P * Q), bw, bh, bni});
        }
    std::sort(gs.begin(), gs.end(), [](const Geo &a, const Geo &b) {
        if (a.waste != b.waste) return a.waste < b.waste;
        return a.bw != b.bw ? a.bw > b.bw : a.bh > b.bh;
    });
    for (size_t i = 0; i < gs.size() && i < 2; ++i)
        for (int bn : bns) out.push_back({bn, gs[i].bw, gs[i].bh, gs[i].bni, false});
    return out;
}

static bool enc(CUtensorMap *m, int rank, const void *base, const uint64_t *dims, const uint64_t *str,
                const uint32_t *box) {
    return tma_encode(m, SN_BF16, rank, base, dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

template <int PLANES, int BN, typename TO>
static cudaError_t launch_split(const CUtensorMap *mA, const CUtensorMap &mB, const SParams &p, cudaStream_t st) {
    using L = Lay<PLANES, BN>;
    auto kern = conv_split_kernel<PLANES, BN, TO>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<int64_t>((int64_t)p.mtiles * p.ntiles, num_sms());
    return launch_pdl(kern, dim3((unsigned)grid), dim3(SPLIT_THREADS), L::SMEM, st, mA[0], mA[1], mA[2], mA[3], mB, p);
}

}  // namespace tcs

int32_t conv_split_variants(const Layer &l, const Shape &in, sn_schema s) {
    return (int32_t)tcs::split_configs(l, in, s).size();
}

std::string conv_split_desc(const Layer &l, const Shape &in, sn_schema s, int32_t v) {
    const std::vector<tcs::SConfig> c = tcs::split_configs(l, in, s);
    if (v < 0 || v >= (int32_t)c.size()) return "?";
    char b[64];
    if (c[v].plain) snprintf(b, sizeof(b), "tc bn=%d plain", c[v].BN);
    else snprintf(b, sizeof(b), "tc bn=%d tile=%dx%dx%d", c[v].BN, c[v].BW, c[v].BH, c[v].BNI);
    return b;
}

// the activation planes
size_t conv_split_ws(const Layer &l, const Shape &in, sn_schema s) {
    (void)l;
    const size_t plane = (size_t)in.n * in.h * in.w * tcs::padded_c(in.c) * 2;
    return ((s.dtype == SN_F32 ? 3 : 1) * plane + 255) & ~size_t(255);
}

// prepared weights: the planes, then (256-byte aligned) fp32 [K][RS][C] or the
// qint8 channel scales [K]
static size_t split_planes_bytes(int64_t K, int64_t C, int64_t RS, int dt) {
    return ((size_t)(dt == SN_F32 ? 3 : 1) * K * RS * tcs::padded_c(C) * 2 + 255) & ~size_t(255);
}
size_t split_weight_bytes(int64_t K, int64_t C, int64_t RS, int dt) {
    return split_planes_bytes(K, C, RS, dt) + (dt == SN_F32 ? (size_t)K * RS * C : (size_t)K) * sizeof(float);
}

cudaError_t weight_split(const float *w, void *out, int dt, int64_t K, int64_t C, int64_t RS, cudaStream_t st) {
    float *tail = reinterpret_cast<float *>(static_cast<uint8_t *>(out) + split_planes_bytes(K, C, RS, dt));
    const int64_t Cp = tcs::padded_c(C), total = K * RS * Cp;
    auto *o = static_cast<__nv_bfloat16 *>(out);
    if (dt == SN_F32) {
        launch_pdl(tcs::weight_split_kernel<3>, grid_for(total, 256), 256, 0, st, w, (const float *)nullptr, o, tail, K, C,
                   RS, Cp);
    } else {
        const cudaError_t e = q8_weight_scales(w, tail, K, C * RS, st);
        if (e != cudaSuccess) return e;
        launch_pdl(tcs::weight_split_kernel<1>, grid_for(total, 256), 256, 0, st, w, (const float *)tail, o,
                   (float *)nullptr, K, C, RS, Cp);
    }
    return cudaGetLastError();
}

cudaError_t conv_split(const LaunchArgs &a, int32_t v) {
    using namespace tcs;
    const Layer &l = *a.layer;
    const Shape &in = a.in_shapes[0];
    const std::vector<SConfig> cfgs = split_configs(l, in, a.schema);
    if (v < 0 || v >= (int32_t)cfgs.size()) return cudaErrorInvalidValue;
    const SConfig cf = cfgs[v];
    const bool f32 = a.schema.dtype == SN_F32;
    const int planes = f32 ? 3 : 1;
    const sn_conv_params &c = l.conv;
    const int out_dt = out_dtype(a);
    if (!f32 && !scales_ok(a, a.in[1] ? 2 : 1)) return cudaErrorInvalidValue;
    if (!a.ws || a.ws_bytes < conv_split_ws(l, in, a.schema) || (uintptr_t)a.ws % 16 || (uintptr_t)a.wt % 16)
        return cudaErrorInvalidValue;
    SParams p{};
    p.N = (int)in.n, p.H = (int)in.h, p.W = (int)in.w, p.C = (int)in.c;
    p.K = c.c_out, p.P = (int)l.out.h, p.Q = (int)l.out.w, p.R = c.kh, p.S = c.kw;
    p.stride = c.sh, p.ph = c.ph, p.pw = c.pw, p.dh = c.dh, p.dw = c.dw;
    p.Cp = (int)padded_c(in.c);
    p.cblocks = (p.Cp + BK - 1) / BK;
    p.kiters = p.R * p.S * p.cblocks;
    p.act = c.act;
    p.bias = a.bias;
    p.y = a.out;
    p.res = a.in[1];
    p.err = device_error_word();
    p.wait_limit = a.wait_limit > 0 ? a.wait_limit : WAIT_LIMIT;
    {
        const int eo = dtype_size(out_dt), er = f32 ? 4 : 1;
        auto fits = [&](int bo, int br) {  // K and the bases admit pieces of bo and br bytes
            return p.K % (bo / eo) == 0 && (uintptr_t)a.out % bo == 0 &&
                   (!p.res || (p.K % (br / er) == 0 && (uintptr_t)p.res % br == 0));
        };
        p.vec = fits(16, 16) ? 2 : fits(4 * eo, 4 * er) ? 1 : 0;
    }
    const int64_t pixels = in.n * in.h * in.w, plane = pixels * p.Cp;
    auto *xs = static_cast<__nv_bfloat16 *>(a.ws);
    // the planes of the activations
    const uint32_t total = (uint32_t)(plane / 8);
    const FastDiv fc = make_fastdiv((uint32_t)(p.Cp / 8));
    const dim3 sg((total + 255) / 256);
    if (f32)
        launch_pdl(split_kernel<3, float>, sg, 256, 0, a.stream, (const float *)a.in[0], xs, total, p.C, fc, plane,
                   p.C % 8 == 0 && (uintptr_t)a.in[0] % 32 == 0);
    else
        launch_pdl(split_kernel<1, int8_t>, sg, 256, 0, a.stream, (const int8_t *)a.in[0], xs, total, p.C, fc, plane,
                   p.C % 8 == 0 && (uintptr_t)a.in[0] % 8 == 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // a plain layer's pixels are one row of N H W
    const int64_t gN = cf.plain ? 1 : in.n, gH = cf.plain ? 1 : in.h, gW = cf.plain ? pixels : in.w;
    p.gN = (int)gN, p.gP = cf.plain ? 1 : p.P, p.gQ = cf.plain ? (int)pixels : p.Q;
    p.gph = cf.plain ? 0 : p.ph, p.gpw = cf.plain ? 0 : p.pw;
    p.BW = cf.BW, p.BH = cf.BH, p.BNI = cf.BNI;
    p.tq = (p.gQ + cf.BW - 1) / cf.BW;
    p.tp = (p.gP + cf.BH - 1) / cf.BH;
    p.mtiles = p.tq * p.tp * ((p.gN + cf.BNI - 1) / cf.BNI);
    p.ntiles = (p.K + cf.BN - 1) / cf.BN;
    while ((1 << p.lbw) < cf.BW) ++p.lbw;
    while ((1 << p.lbwh) < cf.BW * cf.BH) ++p.lbwh;
    p.fd_tq = make_fastdiv((uint32_t)p.tq);
    p.fd_tp = make_fastdiv((uint32_t)p.tp);
    p.fd_nt = make_fastdiv((uint32_t)p.ntiles);
    const float *tail = reinterpret_cast<const float *>(static_cast<const uint8_t *>(a.wt) +
                                                        split_planes_bytes(p.K, p.C, p.R * p.S, a.schema.dtype));
    if (f32) {
        p.x32 = static_cast<const float *>(a.in[0]);
        p.w32 = tail;
    } else {
        p.ws = tail;
        const Q8Scales q = scales_of(a);
        p.s_x = q.s_x, p.s_r = q.s_r, p.inv_out = q.inv_out;
    }
    CUtensorMap mA[4], mB;
    {
        const uint64_t dims[4] = {(uint64_t)p.Cp, (uint64_t)p.R * p.S, (uint64_t)p.K, (uint64_t)planes};
        const uint64_t str[3] = {2ull * p.Cp, 2ull * p.R * p.S * p.Cp, 2ull * p.K * p.R * p.S * p.Cp};
        const uint32_t box[4] = {BK, 1, (uint32_t)cf.BN, (uint32_t)planes};
        if (!enc(&mB, 4, a.wt, dims, str, box)) return cudaErrorInvalidValue;
    }
    const uint32_t box[5] = {BK, (uint32_t)cf.BW, (uint32_t)cf.BH, (uint32_t)cf.BNI, (uint32_t)planes};
    const int st = p.stride;
    for (int bh = 0; bh < st; ++bh)
        for (int bw = 0; bw < st; ++bw) {
            const uint64_t dims[5] = {(uint64_t)p.Cp, (uint64_t)((gW - bw + st - 1) / st), (uint64_t)((gH - bh + st - 1) / st),
                                      (uint64_t)gN, (uint64_t)planes};
            const uint64_t str[4] = {2ull * st * p.Cp, 2ull * st * gW * p.Cp, 2ull * gH * gW * p.Cp, 2ull * plane};
            if (!enc(&mA[bh * 2 + bw], 5, xs + (bh * gW + bw) * p.Cp, dims, str, box)) return cudaErrorInvalidValue;
        }
    if (st == 1) mA[1] = mA[2] = mA[3] = mA[0];
#define SN_SPLIT_LAUNCH(PL, TO) \
    return cf.BN == 64 ? launch_split<PL, 64, TO>(mA, mB, p, a.stream) : launch_split<PL, 128, TO>(mA, mB, p, a.stream)
    if (f32) SN_SPLIT_LAUNCH(3, float);
    switch (out_dt) {
    case SN_QI8: SN_SPLIT_LAUNCH(1, int8_t);
    case SN_F16: SN_SPLIT_LAUNCH(1, __half);
    case SN_BF16: SN_SPLIT_LAUNCH(1, __nv_bfloat16);
    case SN_F32: SN_SPLIT_LAUNCH(1, float);
    default: return cudaErrorInvalidValue;
    }
#undef SN_SPLIT_LAUNCH
}

}  // namespace k
}  // namespace sn
