// A pointwise convolution and the depthwise convolution that alone reads it, as
// one kernel (NHWC, fp16 / bf16): the first half of an inverted residual block.
//
// A CTA takes one image, a band of output rows and 64 expanded channels.  It
// stages the band's input rows (whole rows are consecutive pixels: boxes of 128
// pixels x 64 channels) and its 64 weight rows, forms the expanded values with
// tcgen05 into tensor memory, adds bias and activation, rounds them to the type
// that the pointwise layer would have stored, and keeps them in shared memory
// over the staged input; the depthwise taps read them from there and only the
// depthwise result goes to memory.  Every value is what the two layers compute
// one after the other: the same products, the same order, the same roundings.
// (A cluster variant of the convolution adds up its CTAs' sums: their ranges of K
// steps get an accumulator each here.  Variants that group the steps otherwise
// are not paired.)
// What it saves is a launch and its dependency (about 3 of 8 us at batch 1) and
// the expanded map's trip through memory; what it costs is the KS - 1 halo rows
// of every band, expanded twice.  MobileNetV2
// at batch 1 (fp16): 212.7 -> 175.4 us a pass, an inverted residual block at
// batch 32 (28 x 28, 32 -> 192): 21.9 -> 18.4.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "tc_common.cuh"

namespace sn {
namespace k {
namespace fused {

using namespace tc;

constexpr int MAX_MT = 4;
constexpr int MAX_COLS = 256;  // of tensor memory: half of an SM's

struct FParams {
    int32_t H, W, C, E, P, Q, ph, pw;
    int32_t PB, cblocks, act_e, act_d;
    FastDiv fd_qb;  // column blocks of an output row
    const float *be, *bd;
    const void *wd;  // depthwise weights [KS * KS][E]
    void *y;
    int *err;
    long long wait_limit;
};

// T: storage type; KS: 3 or 5; SW: stride; NT: threads (512 while a CTA has an SM
// to itself, where the depthwise part is a latency); PARTS: accumulators that an
// expanded value is the sum of
template <typename T, int KS, int SW, int NT, int PARTS>
__global__ void __launch_bounds__(NT, 512 / NT)
    expand_dw_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB,
                     const __grid_constant__ FParams p, int MT, uint32_t tmem_cols) {
    constexpr int QB = 4;  // output columns per thread
    constexpr bool H2 = std::is_same<T, __half>::value && KS == 3;  // the packed fp16 accumulation of the 3x3 kernels
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t b_bar;
    __shared__ __align__(8) uint64_t full_bar[MAX_MT];
    __shared__ __align__(8) uint64_t accf_bar[MAX_MT];
    __shared__ uint4 dww[KS * KS * 8];
    __shared__ __align__(16) float be_sh[64], bd_sh[64];
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_sh;
    __shared__ int issued_sh, done_sh;

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t tile_bytes = (uint32_t)p.cblocks * (BM * BK * 2);  // one 128-pixel tile of A
    uint8_t *sb = smem + MT * tile_bytes;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int e0 = (int)blockIdx.x * 64, n = (int)blockIdx.z;
    const int p0 = (int)blockIdx.y * p.PB, p1 = min(p0 + p.PB, p.P);
    // the input rows inside the image that the band reads
    const int hs = max(p0 * SW - p.ph, 0), he = min((p1 - 1) * SW - p.ph + KS, p.H);
    const int px = (he - hs) * p.W, mtn = (px + BM - 1) / BM;  // mtn <= MT by the host's choice of PB
    if (threadIdx.x == 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mB)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mA)) : "memory");
    }
    if (threadIdx.x == 0) {
        mbar_init(&b_bar, 1);
        for (int i = 0; i < MAX_MT; ++i) {
            mbar_init(&full_bar[i], 1);
            mbar_init(&accf_bar[i], 1);
        }
        abort_sh = 0;
        issued_sh = done_sh = 0;
        fence_mbar_init();
    }
    // the depthwise weights of the slice (like all weights, not written by the previous kernel)
    for (int i = threadIdx.x; i < KS * KS * 8; i += NT) {
        const int c = e0 + (i & 7) * 8;
        dww[i] = c < p.E ? __ldg(reinterpret_cast<const uint4 *>(static_cast<const T *>(p.wd) + (int64_t)(i >> 3) * p.E + c))
                         : make_uint4(0u, 0u, 0u, 0u);
    }
    if (threadIdx.x < 64) {  // (zero-padded to 256 channels)
        be_sh[threadIdx.x] = __ldg(p.be + e0 + threadIdx.x);
        bd_sh[threadIdx.x] = __ldg(p.bd + e0 + threadIdx.x);
    }
    if (warp == 0) tmem_alloc<1>(&tmem_sh, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    griddep_launch();  // (behind the allocation: see tmem_alloc)
    if (threadIdx.x == 0) {
        mbar_expect_tx(&b_bar, (uint32_t)p.cblocks * (64 * BK * 2));
        for (int cb = 0; cb < p.cblocks; ++cb) tma_2d<1>(su32(sb + cb * (64 * BK * 2)), &mB, su32(&b_bar), cb * BK, e0);
    }
    griddep_wait();
    if (threadIdx.x == 0) {
        const int start = (n * p.H + hs) * p.W;  // the band's first pixel; pixels past its end are never read back
        for (int mt = 0; mt < mtn; ++mt) {
            mbar_expect_tx(&full_bar[mt], tile_bytes);
            for (int cb = 0; cb < p.cblocks; ++cb)
                tma_2d<1>(su32(smem + mt * tile_bytes + cb * (BM * BK * 2)), &mA, su32(&full_bar[mt]), cb * BK,
                          start + mt * BM);
        }
        issued_sh = mtn;
    }
    if (threadIdx.x == 32) {  // MMA issuer
        const uint32_t idesc = idesc_f16<T>(BM, 64);
        const uint64_t da0 = sdesc_sw128(su32(smem)), db0 = sdesc_sw128(su32(sb));
        bool ok = mbar_wait(&b_bar, 0u, p.wait_limit);
        int mt = 0;
        for (; mt < mtn && ok; ++mt) {
            ok = mbar_wait(&full_bar[mt], 0u, p.wait_limit);
            if (!ok) break;
            tc_fence_after();
            int cb = 0;
#pragma unroll
            for (int r = 0; r < PARTS; ++r)
                for (const int cb0 = cb, cb1 = p.cblocks * (r + 1) / PARTS; cb < cb1; ++cb) {
                    const int ks = min(BK / 16, (p.C - cb * BK + 15) / 16);  // 16-value steps that hold channels
                    for (int k = 0; k < ks; ++k)
                        umma<1>(tmem + (uint32_t)((mt * PARTS + r) * 64),
                                da0 + (uint64_t)((mt * tile_bytes + cb * (BM * BK * 2)) >> 4) + 2 * k,
                                db0 + (uint64_t)((cb * (64 * BK * 2)) >> 4) + 2 * k, idesc, (cb > cb0 || k > 0) ? 1u : 0u);
                }
            umma_commit<1>(&accf_bar[mt]);
        }
        if (!ok) {
            atomicOr(p.err, ERR_MMA_WAIT);
            abort_sh = 1;
        }
        done_sh = mt;
    }
    __syncwarp();
    // expanded values: warp w drains lanes 32 (w % 4) .., columns 32 (w / 4 % 2)
    // .. of every tile (256 threads) or every other one
    const int g4 = warp & 3, half = (warp >> 2) & 1;
    auto mid = [&](int i) { return smem + (i >> 7) * tile_bytes + (i & 127) * 128; };  // pixel i's 128 bytes
    for (int mt = warp >> 3; mt < mtn; mt += NT / 256) {
        const bool ok = mbar_wait(&accf_bar[mt], 0u, p.wait_limit);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicOr(p.err, ERR_ACC_WAIT);
            abort_sh = 1;
            break;
        }
        tc_fence_after();
        __syncwarp();
        uint32_t v[32];
        const uint32_t ta = tmem + ((uint32_t)(g4 * 32) << 16) + (uint32_t)(mt * PARTS * 64 + half * 32);
        tmem_ld32(ta, v);
#pragma unroll
        for (int r = 1; r < PARTS; ++r) {  // (from zero, as the cluster's CTAs add)
            uint32_t x[32];
            tmem_ld32(ta + (uint32_t)(r * 64), x);
#pragma unroll
            for (int e = 0; e < 32; ++e)
                v[e] = __float_as_uint((r == 1 ? 0.f + __uint_as_float(v[e]) : __uint_as_float(v[e])) + __uint_as_float(x[e]));
        }
        const int i = g4 * 32 + lane;
        uint8_t *row = mid(mt * BM + i);
        with_act2<T>(p.act_e, [&](auto fin) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 *b4 = reinterpret_cast<const float4 *>(be_sh + half * 32 + 8 * j);
                *reinterpret_cast<uint4 *>(row + (((half * 4 + j) ^ (i & 7)) << 4)) =
                    finish8<T>(v + 8 * j, b4[0], b4[1], false, make_uint4(0u, 0u, 0u, 0u), fin);
            }
        });
    }
    tc_fence_before();
    __syncthreads();
    // depthwise: QB columns x 8 channels per item, as the window kernel does it
    const int qblk = (int)p.fd_qb.d;
    const int items = abort_sh ? 0 : (p1 - p0) * qblk * 8;
    for (int it = threadIdx.x; it < items; it += NT) {
        const int v = it & 7, pr = (int)fdiv((uint32_t)(it >> 3), p.fd_qb), q0 = ((it >> 3) - pr * qblk) * QB;
        const int c0 = e0 + v * 8;
        if (c0 >= p.E) continue;
        const float4 b0 = *reinterpret_cast<const float4 *>(bd_sh + v * 8), b1 = *reinterpret_cast<const float4 *>(bd_sh + v * 8 + 4);
        const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        constexpr int WN = (QB - 1) * SW + KS;
        const int pout = p0 + pr, wbase = q0 * SW - p.pw;
        T *yrow = static_cast<T *>(p.y) + (((int64_t)n * p.P + pout) * p.Q) * p.E + c0;
        __half2 hacc[H2 ? QB : 1][4];
        float acc[H2 ? 1 : QB][8];
#pragma unroll
        for (int j = 0; j < QB; ++j) {
            if constexpr (H2) {
#pragma unroll
                for (int k = 0; k < 4; ++k) hacc[j][k] = __floats2half2_rn(b[2 * k], b[2 * k + 1]);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[j][e] = b[e];
            }
        }
        // (rolled: a thread has one item or two, so unrolled rows run once each and
        // wait for their instructions: 8 x 28 x 28 x 120, 5 x 5: 11.0 -> 10.3 us)
#pragma unroll 1
        for (int r = 0; r < KS; ++r) {
            const int h = pout * SW - p.ph + r;
            if (h < 0 || h >= p.H) continue;
            const int base = (h - hs) * p.W;
            uint4 win[WN];
#pragma unroll
            for (int t = 0; t < WN; ++t) {
                const int ww = wbase + t, i = base + ww;
                win[t] = (ww >= 0 && ww < p.W) ? *reinterpret_cast<const uint4 *>(mid(i) + ((v ^ (i & 7)) << 4))
                                                : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int s = 0; s < KS; ++s) {
                const uint4 wq = dww[(r * KS + s) * 8 + v];
#pragma unroll
                for (int j = 0; j < QB; ++j) {
                    const uint4 &xv = win[j * SW + s];
                    if constexpr (H2) {
                        const __half2 *xh = reinterpret_cast<const __half2 *>(&xv), *wh = reinterpret_cast<const __half2 *>(&wq);
#pragma unroll
                        for (int k = 0; k < 4; ++k) hacc[j][k] = __hfma2(xh[k], wh[k], hacc[j][k]);
                    } else {
                        mac2<T>(acc[j][0], acc[j][1], xv.x, wq.x);
                        mac2<T>(acc[j][2], acc[j][3], xv.y, wq.y);
                        mac2<T>(acc[j][4], acc[j][5], xv.z, wq.z);
                        mac2<T>(acc[j][6], acc[j][7], xv.w, wq.w);
                    }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < QB; ++j) {
            if (q0 + j >= p.Q) break;
            uint4 o;
            if constexpr (H2) {
                const __half2 z2 = __float2half2_rn(0.0f), six2 = __float2half2_rn(6.0f);
                __half2 *oh = reinterpret_cast<__half2 *>(&o);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    __half2 x = hacc[j][k];
                    if (p.act_d == SN_ACT_RELU) {
                        x = __hmax2(x, z2);
                    } else if (p.act_d == SN_ACT_RELU6) {
                        x = __hmin2(__hmax2(x, z2), six2);
                    } else if (p.act_d != SN_ACT_NONE) {
                        const float2 f = __half22float2(x);
                        x = __floats2half2_rn(act_apply(f.x, p.act_d), act_apply(f.y, p.act_d));
                    }
                    oh[k] = x;
                }
            } else {
                T *op = reinterpret_cast<T *>(&o);
#pragma unroll
                for (int e = 0; e < 8; ++e) op[e] = cvt<T>(act_apply(acc[j][e], p.act_d));
            }
            *reinterpret_cast<uint4 *>(yrow + (int64_t)(q0 + j) * p.E) = o;
        }
    }
    if (warp == 0) {
        if (abort_sh && lane == 0) {
            // let this CTA's copies and MMAs land before its memory goes away
            // (one deadline for the whole drain)
            const long long t0 = clock64();
            while (!mbar_try(&b_bar, 0u) && clock64() - t0 < WAIT_LIMIT) {
            }
            for (int i = 0; i < issued_sh; ++i)
                while (!mbar_try(&full_bar[i], 0u) && clock64() - t0 < WAIT_LIMIT) {
                }
            for (int i = 0; i < done_sh; ++i)
                while (!mbar_try(&accf_bar[i], 0u) && clock64() - t0 < WAIT_LIMIT) {
                }
        }
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, tmem_cols);
    }
}

// at least a third of an SM, so that no more than two CTAs share one: each
// holds at most half of its tensor memory, so neither waits for the other's
static size_t smem_of(int MT, int cblocks) {
    return std::max<size_t>((size_t)MT * cblocks * (BM * BK * 2) + (size_t)cblocks * (64 * BK * 2) + 1024, 80 * 1024);
}

}  // namespace fused

// the band height and the pixel tiles of a CTA: as few tiles as let the whole
// layer run as one wave of two CTAs an SM (one where the staged input takes more
// than half of it), so that at batch 1 the work spreads over the GPU and a
// larger layer has fewer halo rows.  No pair where four tiles are too few: a
// CTA's phases do not overlap, and several waves of them measured slower than
// the two layers (a block with its projection: 32 x 28 x 28, 32 -> 192: 17.8 ->
// 15.7 us and 14 x 14, 96 -> 576 at batch 1: 10.7 -> 8.9 in one wave; 32 x 56 x
// 56, 24 -> 144: 43.3 -> 47.5 and 32 x 112 x 112, 16 -> 96: 61 -> 84 in more)
ExpandDwPlan expand_dw_plan(const Layer &conv, const Shape &in, int32_t conv_variant, const Layer &dw, int32_t dw_variant,
                            sn_schema s) {
    using namespace fused;
    const ExpandDwPlan none{0, 0, 0, 0};
    const sn_conv_params &c = conv.conv, &d = dw.conv;
    if (conv.type != SN_L_CONV2 || dw.type != SN_L_DWCONV2 || s.layout != SN_NHWC || (s.dtype != SN_F16 && s.dtype != SN_BF16))
        return none;
    if (c.kh != 1 || c.kw != 1 || c.sh != 1 || c.sw != 1 || c.ph || c.pw || c.groups != 1 || c.c_in % 8 || c.c_out % 8) return none;
    if (d.c_in != c.c_out || d.kh != d.kw || (d.kh != 3 && d.kh != 5) || d.sh != d.sw || (d.sh != 1 && d.sh != 2) || d.dh != 1 ||
        d.dw != 1)
        return none;
    const int32_t parts = conv_tc_sum_parts(conv, in, s, conv_variant);
    if (parts < 1 || !dw_sums_as_window(dw, conv.out, s, dw_variant)) return none;
    const int64_t N = in.n, H = in.h, W = in.w, P = dw.out.h, slices = (c.c_out + 63) / 64;
    const int cblocks = (c.c_in + BK - 1) / BK;
    if (N > 65535 || P > 65535 || N * H * W >= ((int64_t)1 << 31) - BM * MAX_MT) return none;
    for (int MT = 1; MT <= MAX_MT; ++MT) {
        const size_t sm = smem_of(MT, cblocks);
        if (sm > 220 * 1024 || MT * parts * 64 > MAX_COLS) break;
        const int64_t rows = std::min<int64_t>(MT * BM / W, H);  // input rows that fit
        int64_t PB = rows >= H ? P : rows < d.kh ? 0 : (rows - d.kh) / d.sh + 1;
        if (PB < 1) continue;
        PB = std::min(PB, P);
        const int64_t bands = (P + PB - 1) / PB;
        PB = (P + bands - 1) / bands;
        const int64_t grid = slices * bands * N, slots = (int64_t)num_sms() * (sm <= 110 * 1024 ? 2 : 1);
        if (grid <= slots) return ExpandDwPlan{MT, (int32_t)PB, (int32_t)bands, parts};
    }
    return none;
}

cudaError_t expand_dw(const LaunchArgs &a, const LaunchArgs &b, const ExpandDwPlan &pl) {
    using namespace fused;
    const Layer &conv = *a.layer, &dw = *b.layer;
    const Shape &in = a.in_shapes[0];
    if (pl.MT < 1 || pl.parts < 1 || pl.MT * pl.parts * 64 > MAX_COLS || (uintptr_t)b.out % 16 || (uintptr_t)b.wt % 16) return cudaErrorInvalidValue;
    FParams p{};
    p.H = (int)in.h, p.W = (int)in.w, p.C = (int)in.c, p.E = conv.conv.c_out;
    p.P = (int)dw.out.h, p.Q = (int)dw.out.w, p.ph = dw.conv.ph, p.pw = dw.conv.pw;
    p.PB = pl.PB;
    p.cblocks = (p.C + BK - 1) / BK;
    p.act_e = conv.conv.act, p.act_d = dw.conv.act;
    p.fd_qb = make_fastdiv((uint32_t)((p.Q + 3) / 4));
    p.be = a.bias, p.bd = b.bias;
    p.wd = b.wt;
    p.y = b.out;
    p.err = device_error_word();
    p.wait_limit = a.wait_limit > 0 ? a.wait_limit : WAIT_LIMIT;
    CUtensorMap mA, mB;
    const int dt = a.schema.dtype;
    {
        const uint64_t dims[2] = {(uint64_t)p.C, (uint64_t)(in.n * in.h * in.w)}, str[1] = {2ull * p.C};
        const uint32_t box[2] = {BK, BM};
        if (!tma_encode(&mA, dt, 2, a.in[0], dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B)) return cudaErrorInvalidValue;
    }
    {
        const uint64_t dims[2] = {(uint64_t)p.C, (uint64_t)p.E}, str[1] = {2ull * p.C};
        const uint32_t box[2] = {BK, 64};
        if (!tma_encode(&mB, dt, 2, a.wt, dims, str, box, CU_TENSOR_MAP_SWIZZLE_128B)) return cudaErrorInvalidValue;
    }
    const size_t smem = smem_of(pl.MT, p.cblocks);
    uint32_t cols = 64;  // a power of two
    while (cols < (uint32_t)(pl.MT * pl.parts * 64)) cols *= 2;
    const dim3 grid((unsigned)((p.E + 63) / 64), (unsigned)pl.bands, (unsigned)in.n);
    const bool big = (int64_t)grid.x * grid.y * grid.z > num_sms();  // two CTAs share an SM
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        return launch_pdl(kern, grid, dim3(big ? 256u : 512u), smem, a.stream, mA, mB, p, (int)pl.MT, cols);
    };
    const int ks = dw.conv.kh, sw = dw.conv.sw;
#define SN_EXPAND_DW_P(T, KS, SW, PARTS) \
    return big ? go(expand_dw_kernel<T, KS, SW, 256, PARTS>) : go(expand_dw_kernel<T, KS, SW, 512, PARTS>)
#define SN_EXPAND_DW(T, KS, SW)                          \
    do {                                                 \
        if (pl.parts == 1) SN_EXPAND_DW_P(T, KS, SW, 1); \
        if (pl.parts == 2) SN_EXPAND_DW_P(T, KS, SW, 2); \
        if (pl.parts == 4) SN_EXPAND_DW_P(T, KS, SW, 4); \
        return cudaErrorInvalidValue;                    \
    } while (0)
#define SN_EXPAND_DW_T(T)                      \
    do {                                       \
        if (ks == 3 && sw == 1) SN_EXPAND_DW(T, 3, 1); \
        if (ks == 3) SN_EXPAND_DW(T, 3, 2);    \
        if (sw == 1) SN_EXPAND_DW(T, 5, 1);    \
        SN_EXPAND_DW(T, 5, 2);                 \
    } while (0)
    if (dt == SN_F16) SN_EXPAND_DW_T(__half);
    SN_EXPAND_DW_T(__nv_bfloat16);
#undef SN_EXPAND_DW_T
#undef SN_EXPAND_DW_P
#undef SN_EXPAND_DW
}

}  // namespace k
}  // namespace sn
