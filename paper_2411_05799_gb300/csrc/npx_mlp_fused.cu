// npx_mlp_fused.cu -- the surrogate network's inference in one kernel (tcgen05 / TMEM / TMA,
// sm_103a): every layer of 128 rows on one SM, the activations never leaving it.
//
// Layer by layer the activations of 65,536 rows (64 MB a layer) went out to L2 and back between
// five GEMM launches, and two more kernels packed the FP32 input and unpadded the output.  Here a
// persistent CTA takes 128 rows through the whole network:
//   - 128 KB of shared memory hold the rows' activations as the K-major, 128-byte-swizzled A
//     operand (up to 512 wide); warp 0 streams the weights through a ring of 256 x 64 boxes (three
//     of 32 KB: what is left), from L2, where they stay;
//   - warp 1 issues the MMAs of one 256-column block of a layer (a step) after the other, into the
//     two halves of tensor memory in turn;
//   - sixteen epilogue warps drain the other half: bias, GELU, rounding to BF16.  A layer's first
//     block waits in registers while the second block's MMAs still read the old activations; then
//     both go to shared memory in place of those, block by block, so that the next layer's first
//     MMAs run while its later columns are still being written.
// The products, their order, the bias, the GELU and the roundings are those of the layer-by-layer
// path, so the results are the same bit for bit.
// The input rows are loaded two rows at a time and the next tile's drawn into L2 ahead, and output
// rows without padding are staged as they lie in memory and leave as one bulk copy: chunk-wise
// loads and strided stores were two fifths of a tile's 120,000 cycles.  65,536 rows, 271 -> 4 x 512 ->
// 247: 225 us layer by layer, 197 with those, 137 now; what is left is the MMAs and the last block's
// epilogue of each layer.  (Weights by cluster multicast, and pairs of CTAs sharing each MMA, which
// halve or quarter the weights' traffic, measured no faster, 198 to 224 us, before those two: the
// ring was not what it waited for.)
// Waits are bounded as in npx_gemm.cu: a role that gives up sets the error flag and the others leave;
// an epilogue warp goes on or gives up as one.
#include <algorithm>
#include <cstring>

#include "../../include/npx_mlp.h"
#include "npx_internal.h"
#include "npx_tcgen05.cuh"

namespace npx {
namespace gemm {

constexpr int F_ROWS = 128, F_BN = 256, F_BK = 64, F_STAGES = 3, F_EPI = 16, F_THREADS = 32 * (2 + F_EPI);
constexpr int F_ACT = F_ROWS * FUSED_WIDTH * 2, F_CHUNK = F_ROWS * F_BK * 2, F_STAGE = F_BN * F_BK * 2;

struct FusedMaps {
    CUtensorMap w[FUSED_LAYERS];
};

// 16-byte unit u (8 BF16 columns) of row r in a 64-column chunk of the swizzled activations
__device__ __forceinline__ uint32_t act_offset(int col, int row) {
    return (uint32_t)((col >> 6) * F_CHUNK + row * 128 + ((((col & 63) >> 3) ^ (row & 7)) << 4));
}

__device__ __forceinline__ void act_store16(uint8_t *act, int col, int row, const uint32_t (&w)[8]) {
    *reinterpret_cast<uint4 *>(act + act_offset(col, row)) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4 *>(act + act_offset(col + 8, row)) = make_uint4(w[4], w[5], w[6], w[7]);
}

__device__ __forceinline__ void load_acc16(uint32_t taddr, const float *bias, float (&v)[16]) {
    uint32_t r[16];
    tmem_ld16_issue(taddr, r);
    const float4 *bb = reinterpret_cast<const float4 *>(bias);
    const float4 b0 = __ldg(bb), b1 = __ldg(bb + 1), b2 = __ldg(bb + 2), b3 = __ldg(bb + 3);
    tmem_wait_ld();
    const float b[16] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w, b2.x, b2.y, b2.z, b2.w, b3.x, b3.y, b3.z, b3.w};
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]) + b[i];
}

__device__ __forceinline__ void hidden16(uint32_t taddr, const float *bias, uint32_t (&w)[8]) {
    float v[16];
    load_acc16(taddr, bias, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(gelu(v[2 * i]), gelu(v[2 * i + 1]));
        w[i] = *reinterpret_cast<const uint32_t *>(&h);
    }
}

__global__ void __launch_bounds__(F_THREADS, 1)
mlp_fused_kernel(const __grid_constant__ FusedMaps maps, const __grid_constant__ FusedNet net,
                 const float *__restrict__ x, int n_in, const __nv_bfloat16 *__restrict__ xb, float *__restrict__ y,
                 int ldy, int ncols, int tiles, int *err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *act = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *ring = act + F_ACT;
    uint64_t *full = reinterpret_cast<uint64_t *>(ring + F_STAGES * F_STAGE);
    uint64_t *empty = full + F_STAGES;
    uint64_t *tfull = empty + F_STAGES;    // a step's accumulators complete
    uint64_t *tempty = tfull + 2;          // and drained
    uint64_t *aready = tempty + 2;         // columns 0-255 / 256-511 of a layer's input written
    uint64_t *staged = aready + 2;         // every epilogue warp is done with a tile's staged outputs
    uint64_t *freed = staged + 1;          // and the activations' memory can take the next tile
    uint64_t *done = freed + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    int *issued = reinterpret_cast<int *>(tmem_slot + 2), *consumed = reinterpret_cast<int *>(tmem_slot + 3);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, L = net.layers;

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"((uint32_t)(2 * F_BN))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < F_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], F_EPI);
            mbar_init(&aready[b], F_EPI);
        }
        mbar_init(staged, F_EPI);
        mbar_init(freed, 1);
        mbar_init(done, 1);
        *abort = 0;
        *issued = 0;
        *consumed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---- the weights, box by box in the order the MMAs take them
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x)
                for (int l = 0; l < L && ok; ++l)
                    for (int n0 = 0; n0 < net.n[l] && ok; n0 += F_BN)
                        for (int k0 = 0; k0 < net.k[l]; k0 += F_BK, ++g) {
                            const int s = g % F_STAGES;
                            if (g >= F_STAGES && !mbar_wait(&empty[s], (uint32_t)(((g / F_STAGES) - 1) & 1), abort)) {
                                ok = false;
                                break;
                            }
                            // (rows past the layer's width arrive as zeros and count towards the box)
                            mbar_expect_tx(&full[s], (uint32_t)(min(F_BN, net.n[l]) * F_BK * 2));
                            tma_load_2d(ring + s * F_STAGE, &maps.w[l], k0, n0, &full[s]);
                            *issued = g + 1;
                        }
            if (!ok) {
                *abort = 1;
                atomicExch(err, 1);
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer
        if (lane == 0) {
            int g = 0, step = 0, gen = 0;   // ring boxes, steps, layer inputs so far
            bool ok = true;
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x)
                for (int l = 0; l < L && ok; ++l, ++gen)
                    for (int n0 = 0; n0 < net.n[l] && ok; n0 += F_BN, ++step) {
                        const int b = step & 1;
                        if (step >= 2 && !mbar_wait(&tempty[b], (uint32_t)(((step >> 1) - 1) & 1), abort)) {
                            ok = false;
                            break;
                        }
                        const uint32_t d = tmem + (uint32_t)(b * F_BN);
                        const uint32_t idesc = idesc_bf16(F_ROWS, min(F_BN, net.n[l] - n0));
                        for (int k0 = 0; k0 < net.k[l]; k0 += F_BK, ++g) {
                            const int s = g % F_STAGES;
                            if (((k0 & 255) == 0 && !mbar_wait(&aready[k0 >> 8], (uint32_t)(gen & 1), abort)) ||
                                !mbar_wait(&full[s], (uint32_t)((g / F_STAGES) & 1), abort)) {
                                ok = false;
                                break;
                            }
                            *consumed = g + 1;
                            tc_fence_after();
                            const uint64_t da = sdesc_k_sw128(smem_u32(act + (k0 >> 6) * F_CHUNK));
                            const uint64_t db = sdesc_k_sw128(smem_u32(ring + s * F_STAGE));
#pragma unroll
                            for (int k = 0; k < F_BK / 16; ++k)
                                umma_bf16(d, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, (k0 | k) != 0);
                            umma_commit(&empty[s]);
                        }
                        if (!ok) break;
                        umma_commit(&tfull[b]);
                    }
            umma_commit(done);
            if (!ok) {
                *abort = 1;
                atomicExch(err, 2);
            }
        }
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 and a quarter of a step's columns
        const int e = warp - 2, q = warp & 3, part = e >> 2, row = q * 32 + lane;
        const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
        // (a row pitch of whole 16-byte units would put the lanes' rows on a few banks)
        const bool bulk = ncols == ldy && ldy <= F_ACT / (4 * F_ROWS) && (ldy & 3) != 0 &&
                          (reinterpret_cast<uintptr_t>(y) & 15) == 0;
        int step = 0, it = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++it) {
            // (the last tile's outputs were staged where these go)
            if (it > 0 && !mbar_wait_warp(freed, (uint32_t)((it - 1) & 1), abort)) {
                ok = false;
                break;
            }
            // the tile's rows into the activations (this warp: eight of them), zero-padded
            if (xb) {
                const int units = net.k[0] >> 3;
                const uint4 *src = reinterpret_cast<const uint4 *>(xb + (size_t)(t * F_ROWS + e * 8) * net.k[0]);
#pragma unroll 4
                for (int i = lane; i < 8 * units; i += 32) {
                    const int r = i / units, u = i - r * units;
                    *reinterpret_cast<uint4 *>(act + act_offset(u * 8, e * 8 + r)) = __ldg(src + i);
                }
            } else {
                // (all of two rows' loads first: they are rows of no alignment, four bytes a lane)
                const float *src = x + (size_t)(t * F_ROWS + e * 8) * n_in;
#pragma unroll
                for (int r = 0; r < 8; r += 2, src += 2 * n_in) {
                    float v[2][FUSED_WIDTH / 64][2];
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int c = 0; c < FUSED_WIDTH / 64; ++c) {
                            const int col = c * 64 + 2 * lane;
                            v[i][c][0] = col < n_in ? __ldg(src + i * n_in + col) : 0.f;
                            v[i][c][1] = col + 1 < n_in ? __ldg(src + i * n_in + col + 1) : 0.f;
                        }
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int c = 0; c < FUSED_WIDTH / 64; ++c) {
                            const int col = c * 64 + 2 * lane;
                            if (c * 64 < net.k[0])
                                *reinterpret_cast<__nv_bfloat162 *>(act + act_offset(col, e * 8 + r + i) + ((col & 7) << 1)) =
                                    __floats2bfloat162_rn(v[i][c][0], v[i][c][1]);
                        }
                }
                // the next tile's rows into L2 meanwhile
                if (t + gridDim.x < tiles) {
                    const char *next = reinterpret_cast<const char *>(x + (size_t)((t + gridDim.x) * F_ROWS + e * 8) * n_in);
                    for (int o = lane * 128; o < 32 * n_in; o += 32 * 128)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(next + o));
                }
            }
            fence_async_shared();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&aready[0]);
                mbar_arrive(&aready[1]);
            }
            for (int l = 0; l < L - 1 && ok; ++l) {
                const int N = net.n[l];
                const float *bias = net.bias[l];
                uint32_t keep[4][8];   // a first block's columns, until the second block's MMAs are done
                for (int n0 = 0; n0 < N; n0 += F_BN, ++step) {
                    const int b = step & 1, bn = min(F_BN, N - n0), nch = bn >> 6, c0 = part * (bn >> 2);
                    const bool last = n0 + F_BN >= N;
                    if (!mbar_wait_warp(&tfull[b], (uint32_t)((step >> 1) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    if (last && n0 > 0) {   // the old activations are no longer read
#pragma unroll
                        for (int c = 0; c < 4; ++c) act_store16(act, part * 64 + 16 * c, row, keep[c]);
                        fence_async_shared();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&aready[0]);
                    }
                    const uint32_t taddr = trow + (uint32_t)(b * F_BN + c0);
                    if (last) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            if (c < nch) {
                                uint32_t w[8];
                                hidden16(taddr + 16 * c, bias + n0 + c0 + 16 * c, w);
                                act_store16(act, n0 + c0 + 16 * c, row, w);
                            }
                        }
                        fence_async_shared();
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c) hidden16(taddr + 16 * c, bias + n0 + c0 + 16 * c, keep[c]);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&tempty[b]);
                        if (last) {
                            if (n0 == 0) mbar_arrive(&aready[0]);
                            mbar_arrive(&aready[1]);
                        }
                    }
                }
            }
            // the output layer: its accumulators are read once all its MMAs are done, so that the
            // activations' memory can stage the rows for full-line stores
            const int N = net.n[L - 1], nb = (N + F_BN - 1) / F_BN;
            for (int j = 0; j < nb && ok; ++j)
                if (!mbar_wait_warp(&tfull[(step + j) & 1], (uint32_t)(((step + j) >> 1) & 1), abort)) ok = false;
            if (!ok) break;
            tc_fence_after();
            // rows without padding between them are one block of memory: staged as they lie there, it
            // leaves as one bulk copy; wider or strided rows go out by 16 columns of 32 rows
            float *stage = bulk ? reinterpret_cast<float *>(act) + (size_t)row * ldy
                                : reinterpret_cast<float *>(act) + e * 512;   // 32 rows x 16 columns
            float *out = y + (size_t)(t * F_ROWS + q * 32) * ldy;
            for (int n0 = 0; n0 < N; n0 += F_BN, ++step) {
                const int b = step & 1, bn = min(F_BN, N - n0), nch = bn >> 6, c0 = part * (bn >> 2);
                const uint32_t taddr = trow + (uint32_t)(b * F_BN + c0);
#pragma unroll 1
                for (int c = 0; c < nch; ++c) {
                    const int col = n0 + c0 + 16 * c;
                    if (col >= ncols) break;
                    float v[16];
                    load_acc16(taddr + 16 * c, net.bias[L - 1] + col, v);
                    if (bulk) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (col + i < ncols) stage[col + i] = v[i];
                        continue;
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i)   // 16-byte units swizzled against bank conflicts
                        *reinterpret_cast<float4 *>(stage + lane * 16 + ((i ^ ((lane >> 1) & 3)) << 2)) =
                            make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    __syncwarp();
                    const int k = lane & 15;
                    if (col + k < ncols) {
#pragma unroll
                        for (int r = lane >> 4; r < 32; r += 2)
                            out[(size_t)r * ldy + col + k] = stage[r * 16 + (((k >> 2) ^ ((r >> 1) & 3)) << 2) + (k & 3)];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[b]);
            }
            if (bulk) fence_async_shared();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(staged);
                if (e == 0) {
                    if (!mbar_wait(staged, (uint32_t)(it & 1), abort)) {
                        *abort = 1;   // every warp gives up where it waits for freed
                        atomicExch(err, 3);
                    } else {
                        if (bulk) {
                            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                                             y + (size_t)t * F_ROWS * ldy),
                                         "r"(smem_u32(act)), "r"((uint32_t)(F_ROWS * 4 * ldy))
                                         : "memory");
                            bulk_commit();
                            bulk_wait_read<0>();
                        }
                        mbar_arrive(freed);
                    }
                }
            }
        }
        if (bulk && e == 0 && lane == 0) bulk_wait_all();   // the copies have landed before the CTA ends
        __syncwarp();
        if (!ok && lane == 0) {
            *abort = 1;
            atomicExch(err, 3);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // after a failure: let the copies still in flight land before the shared memory goes away
        for (int g = *consumed; g < *issued; ++g) mbar_wait(&full[g % F_STAGES], (uint32_t)((g / F_STAGES) & 1));
        if (!mbar_wait(done, 0)) atomicExch(err, 4);   // the MMAs end before their tensor memory is freed
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * F_BN)) : "memory");
    }
}

}  // namespace gemm

bool fused_fits(const FusedNet &net) {
    if (net.layers < 1 || net.layers > FUSED_LAYERS) return false;
    for (int l = 0; l < net.layers; ++l)
        if (net.k[l] < 64 || net.k[l] % 64 || net.k[l] > FUSED_WIDTH || net.n[l] < 128 || net.n[l] % 128 ||
            net.n[l] > FUSED_WIDTH)
            return false;
    return true;
}

cudaError_t launch_mlp_fused(const FusedNet &net, const float *x, int n_in, const __nv_bfloat16 *xb, float *y, int ldy,
                             int ncols, int rows, int *err, cudaStream_t st) {
    using namespace gemm;
    FusedMaps maps;
    memset(&maps, 0, sizeof maps);
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    for (int l = 0; l < net.layers; ++l) {
        const cuuint64_t dims[2] = {(cuuint64_t)net.k[l], (cuuint64_t)net.n[l]};
        const cuuint64_t strides[1] = {(cuuint64_t)net.k[l] * 2};
        const cuuint32_t box[2] = {(cuuint32_t)F_BK, (cuuint32_t)std::min(F_BN, net.n[l])};
        const cuuint32_t es[2] = {1, 1};
        if (fn(&maps.w[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(net.w[l]), dims, strides, box,
               es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    const int smem = 1024 + F_ACT + F_STAGES * F_STAGE + 256;
    cudaError_t e = cudaFuncSetAttribute(mlp_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int tiles = rows / F_ROWS;
    mlp_fused_kernel<<<std::min(tiles, sms), F_THREADS, smem, st>>>(maps, net, x, n_in, xb, y, ldy, ncols, tiles, err);
    return cudaGetLastError();
}

}  // namespace npx
