// Tensor-core implicit GEMM for layers too small to fill the GPU (batch 1, small
// maps): one tile per cluster, the tile's K steps split among the cluster's CTAs.
//
// What bounds such a layer is not the tensor core but a chain of latencies: the
// dependency release, the copies of all its K steps through one SM (about 350
// cycles a box for the thread that issues it), the MMAs, the drain.  So
//   * a cluster of NCL CTAs takes the 128-pixel x BN-channel tile, each CTA
//     1/NCL of the K steps (1 to 5 boxes of A instead of 9 to 36), and the
//     partial sums meet on chip: every CTA sends each peer the columns that the
//     peer finishes (st.async into its shared memory, counted by an mbarrier
//     there), adds its own BN/NCL columns in rank order, and stores them;
//   * the weights of the first K steps are copied before the dependency wait
//     (they are not written by the previous kernel), each stage by a warp of
//     its own, so that only boxes of A are left on the critical path;
//   * a CTA keeps to half an SM (three stages, one accumulator), so the next
//     kernel's CTAs can set up and copy their weights beside it;
//   * the residual's and the bias' loads are in flight before the accumulator
//     is ready; a cluster's rows go from registers straight to global memory, a
//     single CTA's tile through the stage memory and a TMA store.
// The sum of a tile is deterministic: fixed ranges, fixed order.  Waits are
// bounded as in tc_conv.cuh.
// Measured (fp16, a pass of a replayed net): MobileNetV2 at batch 1 239.6 ->
// 212.7 us (35 convolutions of 1 to 36 K steps), the 14 x 14 bottleneck 1024 ->
// 256 -> 256 -> 1024 at batch 1 20.6 -> 16.4 us (two of its layers were a K
// split through global memory with a reduction kernel each).
#include <cuda.h>

#include <algorithm>

#include "tc_common.cuh"

namespace sn {
namespace k {
namespace tc {

constexpr int LAT_STAGES = 3;
constexpr int LAT_THREADS = 32 * (4 + 1 + LAT_STAGES);  // epilogue, MMA, one producer per stage

// 16 bytes into a peer's shared memory, counted by the mbarrier there
__device__ __forceinline__ void st_async_v4(uint32_t caddr, uint32_t cbar, uint32_t a, uint32_t b, uint32_t c,
                                            uint32_t d) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(
                     caddr),
                 "r"(cbar), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

template <typename T, int BN, int NCL>
__global__ void __launch_bounds__(LAT_THREADS, 2)
    conv_tc_lat_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                       const __grid_constant__ CUtensorMap mA2, const __grid_constant__ CUtensorMap mA3,
                       const __grid_constant__ CUtensorMap mB, const __grid_constant__ CUtensorMap mY,
                       const __grid_constant__ Params p) {
    constexpr uint32_t A_BYTES = BM * BK * 2, STAGE = A_BYTES + BN * BK * 2;
    constexpr int CW = BN / NCL;  // columns this CTA finishes
    static_assert(CW >= 8 && CW % 8 == 0, "whole 16-byte pieces of a row");
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[LAT_STAGES];
    __shared__ __align__(8) uint64_t empty_bar[LAT_STAGES];
    __shared__ __align__(8) uint64_t accf_bar;
    __shared__ __align__(8) uint64_t x_bar[4];  // a warp's rows of every peer's partial sums have arrived
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_sh;
    __shared__ int issued_sh[LAT_STAGES], consumed_sh;
    __shared__ __align__(16) float bias_sh[BN];  // like all weights not written by the previous kernel

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // partial sums from the peers: [rank][CW / 4][128 rows] float4
    float4 *xch = reinterpret_cast<float4 *>(smem + LAT_STAGES * STAGE);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = NCL > 1 ? cluster_rank() : 0u;
    const int tile = (int)(blockIdx.x / NCL);
    const Work w = work_of(p, tile, BN, p.BW > 0, 1, 1);
    // this CTA's K steps
    const int it0 = p.kiters * (int)rank / NCL, it1 = p.kiters * ((int)rank + 1) / NCL, nit = it1 - it0;
    if (threadIdx.x == 32) {  // the maps are kernel parameters, not data of the previous kernel
        const CUtensorMap *maps[6] = {&mB, &mA0, &mA1, &mA2, &mA3, &mY};
        for (int i = 0; i < 6; ++i)
            if (i < 2 || (i < 5 ? p.stride != 1 : NCL == 1))
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(maps[i])) : "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < LAT_STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
            issued_sh[s] = 0;
        }
        mbar_init(&accf_bar, 1);
        for (int i = 0; i < 4; ++i) mbar_init(&x_bar[i], 1);
        abort_sh = 0;
        consumed_sh = 0;
        fence_mbar_init();
        if (NCL > 1)
            for (int i = 0; i < 4; ++i) mbar_expect_tx(&x_bar[i], (NCL - 1) * 32 * CW * 4);
    }
    if (threadIdx.x < BN) bias_sh[threadIdx.x] = __ldg(p.bias + w.n0 + threadIdx.x);  // zero-padded to 256 channels
    if (warp == 4) tmem_alloc<1>(&tmem_sh, BN);
    tc_fence_before();
    if (NCL > 1) cluster_sync_all();  // every CTA's barriers exist before a peer signals them
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    griddep_launch();  // (behind the allocation: see tmem_alloc)
    if (warp > 4) {
        if (lane == 0) {  // ---------------- producer of stage s: the K steps it0 + s, it0 + s + LAT_STAGES, ...
            const int s = warp - 5;
            const uint32_t sa = su32(smem + s * STAGE), bar = su32(&full_bar[s]);
            auto coords = [&](int it, int &c0, int &tap, int &r, int &ss) {
                tap = (int)fdiv((uint32_t)it, p.fd_spt);
                c0 = (it - tap * (int)p.fd_spt.d) * BK;
                r = (int)fdiv((uint32_t)tap, p.fd_S);
                ss = tap - r * (int)p.fd_S.d;
            };
            auto load_a = [&](int c0, int r, int ss) {
                if (p.BW > 0) {
                    const int oh = r * p.dh - p.ph, ow = ss * p.dw - p.pw;
                    const CUtensorMap *m = &mA0;
                    int qa = w.q0 + ow, pa = w.p0 + oh;
                    if (p.stride != 1) {  // even/odd sub-lattice maps
                        const int bh = oh & 1, bw = ow & 1;
                        m = bh ? (bw ? &mA3 : &mA2) : (bw ? &mA1 : &mA0);
                        qa = w.q0 + ((ow - bw) >> 1);
                        pa = w.p0 + ((oh - bh) >> 1);
                    }
                    tma_4d<1>(sa, m, bar, c0, qa, pa, w.i0);
                } else {
                    tma_2d<1>(sa, &mA0, bar, c0, (int)w.m0);
                }
            };
            int c0, tap, r, ss;
            if (s < nit) {
                coords(it0 + s, c0, tap, r, ss);
                mbar_expect_tx(&full_bar[s], STAGE);
                tma_3d<1>(sa + A_BYTES, &mB, bar, c0, tap, w.n0);
                griddep_wait();
                load_a(c0, r, ss);
                issued_sh[s] = 1;
            }
            uint32_t par = 0;
            for (int i = s + LAT_STAGES; i < nit; i += LAT_STAGES) {
                if (!mbar_wait(&empty_bar[s], par, p.wait_limit)) {
                    atomicOr(p.err, ERR_TMA_WAIT);
                    abort_sh = 1;
                }
                if (abort_sh) break;
                par ^= 1u;
                coords(it0 + i, c0, tap, r, ss);
                mbar_expect_tx(&full_bar[s], STAGE);
                load_a(c0, r, ss);
                tma_3d<1>(sa + A_BYTES, &mB, bar, c0, tap, w.n0);
                ++issued_sh[s];
            }
        }
    } else if (warp == 4) {
        if (lane == 0) {  // ---------------- MMA issuer
            const uint32_t idesc = idesc_f16<T>(BM, BN);
            const uint64_t desc0 = sdesc_sw128(su32(smem));
            int s = 0, i = 0;
            uint32_t par = 0;
            for (; i < nit; ++i) {
                // (no look at abort_sh: a shared-memory access of this thread queues
                // behind the MMAs' operand reads, ~200 cycles; every wait is bounded)
                if (!mbar_wait(&full_bar[s], par, p.wait_limit)) {
                    atomicOr(p.err, ERR_MMA_WAIT);
                    abort_sh = 1;
                    break;
                }
                tc_fence_after();
                const uint64_t da = desc0 + (uint64_t)((s * STAGE) >> 4), db = da + (A_BYTES >> 4);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) umma<1>(tmem, da + 2 * k, db + 2 * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
                umma_commit<1>(&empty_bar[s]);
                if (++s == LAT_STAGES) {
                    s = 0;
                    par ^= 1u;
                }
            }
            if (i == nit) umma_commit<1>(&accf_bar);
            consumed_sh = i;
        }
    } else if constexpr (NCL == 1) {  // ---------------- epilogue: warp w drains rows 32 w .. 32 w + 31
        // 32 columns at a time; the tile goes out through the stage memory, which
        // the MMAs are done with once the accumulator is ready: a warp's 32 rows x
        // 64 channels, 128-byte swizzled, one TMA store (clipped at the edges)
        const int r0 = warp * 32, row = r0 + lane;
        const bool imp = p.BW > 0;
        const int sq = w.q0 + (imp ? r0 & (p.BW - 1) : 0), sp = w.p0 + (imp ? (r0 >> p.lbw) & (p.BH - 1) : 0),
                  sn_ = w.i0 + (imp ? r0 >> p.lbwh : 0);
        bool valid;
        int64_t pix;
        if (imp) {
            const int q = w.q0 + (row & (p.BW - 1)), pp = w.p0 + ((row >> p.lbw) & (p.BH - 1)), n = w.i0 + (row >> p.lbwh);
            valid = q < p.Q && pp < p.P && n < p.N;
            pix = ((int64_t)n * p.P + pp) * p.Q + q;
        } else {
            pix = w.m0 + row;
            valid = pix < p.Mout;
        }
        const T *res = p.res && valid ? static_cast<const T *>(p.res) + pix * p.K : nullptr;
        uint4 rq[4];
        auto load_res = [&](int k) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                rq[j] = res && k + 8 * j < p.K ? *reinterpret_cast<const uint4 *>(res + k + 8 * j) : make_uint4(0u, 0u, 0u, 0u);
        };
        griddep_wait();
        load_res(w.n0);
        const bool ok = mbar_wait(&accf_bar, 0u, p.wait_limit);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicOr(p.err, ERR_ACC_WAIT);
            abort_sh = 1;
        } else {
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16);
            // (rolled: a CTA runs it once, so that straight-line code waits for its
            // instructions; ResNet-50 at batch 32: 653 -> 639 us)
            with_act2<T>(p.act, [&](auto fin) {
#pragma unroll 1
                for (int c = 0; c < BN / 32; ++c) {
                    const int k0 = w.n0 + 32 * c;
                    if (k0 >= p.K) break;
                    uint8_t *buf = smem + (c >> 1) * (BM * 128) + warp * 4096;
                    uint32_t v[32];
                    tmem_ld32(ta + 32 * c, v);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 *b4 = reinterpret_cast<const float4 *>(bias_sh + 32 * c + 8 * j);
                        const int piece = (c & 1) * 4 + j;
                        *reinterpret_cast<uint4 *>(buf + lane * 128 + ((piece ^ (lane & 7)) << 4)) =
                            finish8<T>(v + 8 * j, b4[0], b4[1], p.res != nullptr, rq[j], fin);
                    }
                    if (c + 1 < BN / 32) load_res(k0 + 32);
                    if ((c & 1) || k0 + 32 >= p.K) {  // the 64-channel block is complete
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            const int kb = w.n0 + 64 * (c >> 1);
                            if (imp) tma_store_4d(&mY, buf, kb, sq, sp, sn_);
                            else tma_store_2d(&mY, buf, kb, (int)(w.m0 + r0));
                            bulk_commit();
                        }
                        __syncwarp();
                    }
                }
            });
            if (lane == 0) bulk_wait_read_0();  // the stores have read the stage memory
            __syncwarp();
        }
    } else {  // ---------------- epilogue of a cluster: warp w drains rows 32 w .. 32 w + 31
        const int row = warp * 32 + lane;
        const int k0 = w.n0 + (int)rank * CW;  // first output channel of this CTA's columns
        bool valid;
        int64_t pix;
        if (p.BW > 0) {
            const int q = w.q0 + (row & (p.BW - 1)), pp = w.p0 + ((row >> p.lbw) & (p.BH - 1)), n = w.i0 + (row >> p.lbwh);
            valid = q < p.Q && pp < p.P && n < p.N;
            pix = ((int64_t)n * p.P + pp) * p.Q + q;
        } else {
            pix = w.m0 + row;
            valid = pix < p.Mout;
        }
        const float *bias = bias_sh + rank * CW;
        griddep_wait();
        uint4 res[CW / 8];
#pragma unroll
        for (int j = 0; j < CW / 8; ++j)
            res[j] = p.res && valid && k0 + 8 * j < p.K
                         ? *reinterpret_cast<const uint4 *>(static_cast<const T *>(p.res) + pix * p.K + k0 + 8 * j)
                         : make_uint4(0u, 0u, 0u, 0u);
        bool ok = mbar_wait(&accf_bar, 0u, p.wait_limit);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicOr(p.err, ERR_ACC_WAIT);
            abort_sh = 1;
            // the peers count on these bytes, and may leave only when they are there
#pragma unroll 1
            for (int i = 0; i < (NCL - 1) * (CW / 4); ++i) {
                const uint32_t dst = (rank + 1 + (uint32_t)(i / (CW / 4))) % NCL;
                const uint32_t at = su32(xch + ((int)rank * (CW / 4) + i % (CW / 4)) * BM + row);
                st_async_v4(mapa(at, dst), mapa(su32(&x_bar[warp]), dst), 0u, 0u, 0u, 0u);
            }
        } else {
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16);
            float own[CW];
            // the columns of each CTA of the cluster: a peer's go to it, this CTA's stay
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t v[32];
                tmem_ld32(ta + 32 * c, v);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int col = 32 * c + 4 * j;
                    const uint32_t dst = (uint32_t)(col / CW);
                    if (dst != rank) {
                        const uint32_t at = su32(xch + ((int)rank * (CW / 4) + (col % CW) / 4) * BM + row);
                        st_async_v4(mapa(at, dst), mapa(su32(&x_bar[warp]), dst), v[4 * j], v[4 * j + 1], v[4 * j + 2],
                                    v[4 * j + 3]);
                    }
                }
            }
            // this CTA's own columns: a runtime offset, so read again
#pragma unroll
            for (int c = 0; c < CW / 8; ++c) {
                uint32_t v[8];
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                             : "r"(ta + rank * CW + 8 * c));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int e = 0; e < 8; ++e) own[8 * c + e] = __uint_as_float(v[e]);
            }
            ok = mbar_wait_cluster(&x_bar[warp], 0u, p.wait_limit);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) {
                if (lane == 0) atomicOr(p.err, ERR_EPI_WAIT);
                abort_sh = 1;
            }
            if (ok) {
                float sum[CW];
#pragma unroll
                for (int e = 0; e < CW; ++e) sum[e] = 0.f;
#pragma unroll
                for (int r = 0; r < NCL; ++r)
#pragma unroll
                    for (int j = 0; j < CW / 4; ++j) {
                        float4 x = make_float4(own[4 * j], own[4 * j + 1], own[4 * j + 2], own[4 * j + 3]);
                        if (r != (int)rank) x = xch[(r * (CW / 4) + j) * BM + row];
                        sum[4 * j] += x.x, sum[4 * j + 1] += x.y, sum[4 * j + 2] += x.z, sum[4 * j + 3] += x.w;
                    }
                T *y = static_cast<T *>(p.y) + pix * p.K + k0;
                with_act2<T>(p.act, [&](auto fin) {
#pragma unroll
                    for (int j = 0; j < CW / 8; ++j) {
                        if (!valid || k0 + 8 * j >= p.K) break;
                        const float4 *b4 = reinterpret_cast<const float4 *>(bias + 8 * j);
                        *reinterpret_cast<uint4 *>(y + 8 * j) =
                            finish8<T>(sum + 8 * j, b4[0], b4[1], p.res != nullptr, res[j], fin);
                    }
                });
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        if (abort_sh && lane == 0) {
            // let this CTA's copies and MMAs and the peers' sums land before its
            // memory goes away (one deadline for the whole drain)
            const long long t0 = clock64();
            for (int i = 0; i < 4 && NCL > 1; ++i)
                while (!mbar_try(&x_bar[i], 0u) && clock64() - t0 < WAIT_LIMIT) {
                }
            for (int s = 0; s < LAT_STAGES; ++s)
                if (issued_sh[s] > 0)
                    while (!mbar_try(&full_bar[s], (uint32_t)(issued_sh[s] - 1) & 1u) && clock64() - t0 < WAIT_LIMIT) {
                    }
            if (consumed_sh > 0) {
                const int i = consumed_sh - 1;
                while (!mbar_try(&empty_bar[i % LAT_STAGES], (uint32_t)(i / LAT_STAGES) & 1u) &&
                       clock64() - t0 < WAIT_LIMIT) {
                }
            }
        }
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, BN);
    }
    // What the peers send has landed by now: the epilogue warps, or the drain
    // above, have waited for x_bar, and a CTA whose own sums are missing sends
    // zeros.  The barrier is for a CTA whose drain ran out.  (Relaxed: nothing read
    // after it depends on it; a releasing arrive would wait for this CTA's global
    // stores to be performed, ~1800 cycles.)
    if (NCL > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

template <typename T, int BN, int NCL>
static cudaError_t launch_lat_t(const CUtensorMap *mA, const CUtensorMap &mB, const CUtensorMap &mY, const Params &p,
                                cudaStream_t st) {
    // (at least a third of an SM: no more than two CTAs share one, so that a third
    // does not wait for tensor memory behind them)
    constexpr size_t need = (size_t)LAT_STAGES * (BM + BN) * BK * 2 + (NCL > 1 ? (size_t)BM * BN * 4 : 0) + 1024;
    constexpr size_t smem = need > 80 * 1024 ? need : 80 * 1024;
    auto kern = conv_tc_lat_kernel<T, BN, NCL>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3((unsigned)(p.mtiles * p.ntiles * NCL));
    cfg.blockDim = dim3(LAT_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_pdl
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 1;
    if (NCL > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = NCL;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kern, mA[0], mA[1], mA[2], mA[3], mB, mY, p);
}

template <typename T>
static cudaError_t launch_lat_d(int bn, int ncl, const CUtensorMap *mA, const CUtensorMap &mB, const CUtensorMap &mY,
                                const Params &p, cudaStream_t st) {
    if (bn == 128 && ncl == 1) return launch_lat_t<T, 128, 1>(mA, mB, mY, p, st);
    if (bn != 64) return cudaErrorInvalidValue;
    if (ncl == 1) return launch_lat_t<T, 64, 1>(mA, mB, mY, p, st);
    if (ncl == 2) return launch_lat_t<T, 64, 2>(mA, mB, mY, p, st);
    if (ncl == 4) return launch_lat_t<T, 64, 4>(mA, mB, mY, p, st);
    if (ncl == 8) return launch_lat_t<T, 64, 8>(mA, mB, mY, p, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_lat(int dtype, int bn, int ncl, const CUtensorMap *mA, const CUtensorMap &mB, const CUtensorMap &mY,
                       const Params &p, cudaStream_t st) {
    if (p.ksplit != 1 || p.y_nchw || p.kiters < ncl || (uintptr_t)p.y % 16) return cudaErrorInvalidValue;
    if (dtype == SN_BF16) return launch_lat_d<__nv_bfloat16>(bn, ncl, mA, mB, mY, p, st);
    return launch_lat_d<__half>(bn, ncl, mA, mB, mY, p, st);
}

}  // namespace tc
}  // namespace k
}  // namespace sn
