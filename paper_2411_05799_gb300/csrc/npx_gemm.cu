// npx_gemm.cu -- BF16 GEMM on the 5th-generation tensor cores (tcgen05 / TMEM / TMA, sm_103a)
// for the learned surrogate: C[M x N] = A[M x K] . B[N x K]^T, both operands K-major (row-major
// with K contiguous), FP32 accumulation in tensor memory, fused epilogues.
//
// A persistent, warp-specialised kernel: each CTA (one per SM) walks tiles of 128 x BN (and, for
// split K, one K range) in a static round-robin.  Warp 0 streams 128 x 64 and BN x 64 operand
// tiles with TMA (128-byte swizzle, the layout the UMMA shared-memory descriptors describe)
// through a STAGES-deep ring of shared-memory buffers; warp 1 issues one tcgen05.mma (M = 128,
// N = BN, K = 16) per 32-byte step of each 64-wide K block into one of two accumulators in tensor
// memory (2 x BN columns) and hands each ring buffer back with tcgen05.commit; sixteen epilogue warps
// read the other accumulator out (warp w owns TMEM lanes 32 (w % 4) .. + 31 and a quarter of
// the columns), apply the epilogue and release it, so a tile's epilogue overlaps the next tile's
// MMAs.  Every wait is bounded and also gives up once another role has failed: the failing role
// sets an error flag, the kernel drains the copies it started, waits for its MMAs, frees its
// tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstring>

#include "../../include/npx_mlp.h"
#include "npx_internal.h"
#include "npx_tcgen05.cuh"

namespace npx {
namespace gemm {

constexpr int BM = 128, BK = 64, STAGES = 4, EPI_WARPS = 16, THREADS = 32 * (2 + EPI_WARPS);

// 16 BF16 of each lane's row (32 rows a warp, even rows on even lanes) to or from memory: the lanes of
// a pair take the two halves of one row and then of the other, so that an access covers whole 32-byte
// sectors of 16 rows and not half sectors of 32.  At 8,192 rows a layer is one tile per SM, its
// epilogue a good part of the launch: with the two-row stores of C^T, GELU's inputs loaded ahead and
// the bias prefetched, four training minibatches went from 1,000 to 970 us.
__device__ __forceinline__ uint4 swap_pair(const uint4 &u) {
    return make_uint4(__shfl_xor_sync(0xffffffffu, u.x, 1), __shfl_xor_sync(0xffffffffu, u.y, 1),
                      __shfl_xor_sync(0xffffffffu, u.z, 1), __shfl_xor_sync(0xffffffffu, u.w, 1));
}

__device__ __forceinline__ void store_bf16x16(__nv_bfloat16 *base, long long ld, int row, int col, const float (&v)[16]) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t *>(&h);
    }
    const uint4 lo = make_uint4(w[0], w[1], w[2], w[3]), hi = make_uint4(w[4], w[5], w[6], w[7]);
    const bool odd = row & 1;
    const uint4 r = swap_pair(odd ? lo : hi);
    __nv_bfloat16 *o = base + (size_t)(row & ~1) * ld + col + (odd ? 8 : 0);
    *reinterpret_cast<uint4 *>(o) = odd ? r : lo;
    *reinterpret_cast<uint4 *>(o + ld) = odd ? hi : r;
}

__device__ __forceinline__ void load_pair(const __nv_bfloat16 *base, long long ld, int row, int col, uint4 (&u)[2]) {
    const __nv_bfloat16 *p = base + (size_t)(row & ~1) * ld + col + ((row & 1) ? 8 : 0);
    u[0] = *reinterpret_cast<const uint4 *>(p);
    u[1] = *reinterpret_cast<const uint4 *>(p + ld);
}

// The epilogue of 16 accumulator values of one row: v = acc[row, col .. col + 15].  With a store
// mode the row-major output goes to this thread's row of the warp's staging box (st: 16 BF16 or
// 16 FP32 values) instead of global memory; the warp then stores the box with TMA.
__device__ __forceinline__ void stage16(void *st, const float (&v)[16], bool f32) {
    if (f32) {
        float4 *o = reinterpret_cast<float4 *>(st);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
        uint4 *o = reinterpret_cast<uint4 *>(st);
        o[0] = make_uint4(w[0], w[1], w[2], w[3]);
        o[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

__device__ __forceinline__ void epilogue16(const npx_gemm_epilogue &ep, float (&v)[16], int row, int col, int split,
                                           int store_mode, void *st, const uint4 (&zp)[2]) {
    if (ep.mode == NPX_EPI_F32) {
        if (store_mode == 2) { stage16(st, v, true); return; }
        float4 *o = reinterpret_cast<float4 *>(ep.outf + (size_t)split * ep.split_stride + (size_t)row * ep.ldf + col);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        return;
    }
    if (ep.bias) {
        const float4 *bb = reinterpret_cast<const float4 *>(ep.bias + col);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 b = bb[i];
            v[4 * i] += b.x; v[4 * i + 1] += b.y; v[4 * i + 2] += b.z; v[4 * i + 3] += b.w;
        }
    }
    if (ep.mode == NPX_EPI_BIAS_GELU) {
        if (ep.zsave) store_bf16x16(static_cast<__nv_bfloat16 *>(ep.zsave), ep.ldz, row, col, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = gelu(v[i]);
    } else if (ep.mode == NPX_EPI_DGELU) {
        const bool odd = row & 1;
        const uint4 r = swap_pair(odd ? zp[0] : zp[1]);
        const uint4 u[2] = {odd ? r : zp[0], odd ? zp[1] : r};
        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(u);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 z = __bfloat1622float2(h[i]);
            v[2 * i] *= gelu_grad(z.x);
            v[2 * i + 1] *= gelu_grad(z.y);
        }
    }
    if (ep.outf) {
        if (store_mode == 2) {
            stage16(st, v, true);
        } else {
            float4 *o = reinterpret_cast<float4 *>(ep.outf + (size_t)row * ep.ldf + col);
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
    }
    if (ep.out) {
        if (store_mode == 1) stage16(st, v, false);
        else store_bf16x16(static_cast<__nv_bfloat16 *>(ep.out), ep.ldo, row, col, v);
    }
    if (ep.outT) {
        // lanes hold consecutive rows: each store instruction writes 64 contiguous bytes of one column,
        // or, where the columns start on 4 bytes, of two: a pair of lanes takes two rows of a column each
        __nv_bfloat16 *o = static_cast<__nv_bfloat16 *>(ep.outT) + (size_t)col * ep.ldt + row;
        if (((reinterpret_cast<uintptr_t>(ep.outT) & 3) | (ep.ldt & 1)) == 0) {
            const bool odd = row & 1;
            __nv_bfloat16 *oc = odd ? o + ep.ldt - 1 : o;   // (column col or col + 1, the pair's even row)
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
                const float r = __shfl_xor_sync(0xffffffffu, odd ? v[i] : v[i + 1], 1);
                *reinterpret_cast<__nv_bfloat162 *>(oc + (size_t)i * ep.ldt) =
                    odd ? __floats2bfloat162_rn(r, v[i + 1]) : __floats2bfloat162_rn(v[i], r);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) o[(size_t)i * ep.ldt] = __float2bfloat16_rn(v[i]);
        }
    }
}

// G products in one launch: their tiles (and split-K ranges) form one list, walked by the persistent
// blocks, so that a product's epilogues run under the next one's copies and MMAs.
template <int G>
struct Products {
    CUtensorMap a[G], b[G], out[G];
    int tiles_n[G], k_per_split[G], splits[G], first[G];   // first: the product's place in the list
    int n, total;
};

struct Tile {
    int p, m0, n0, split, kbeg, nk;
};

template <int BN, int G>
__device__ __forceinline__ Tile tile_at(const Products<G> &P, int t) {
    Tile r;
    r.p = 0;
    if (G > 1)
        while (r.p + 1 < P.n && t >= P.first[r.p + 1]) ++r.p;
    t -= P.first[r.p];
    const int splits = P.splits[r.p], tiles_n = P.tiles_n[r.p], rest = t / splits;
    r.split = t % splits;
    r.n0 = (rest % tiles_n) * BN;
    r.m0 = (rest / tiles_n) * BM;
    r.kbeg = r.split * P.k_per_split[r.p];
    r.nk = P.k_per_split[r.p] / BK;
    return r;
}

// STORE = 2: the FP32 row-major output (outf) leaves through per-warp shared-memory boxes and TMA
// stores (P.out), STORE = 1: the BF16 one (out) does; STORE = 0: every output is stored directly.
template <int BN, int STORE, int G>
__global__ void __launch_bounds__(THREADS, 1)
gemm_tn_kernel(const __grid_constant__ Products<G> P, npx_gemm_epilogue ep, int *err) {
    constexpr int store_mode = STORE;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
    uint8_t *sA = smem;
    uint8_t *sB = smem + STAGES * A_BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(sB + STAGES * B_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *tfull = empty + STAGES;     // accumulator b ready for the epilogue
    uint64_t *tempty = tfull + 2;         // accumulator b drained by the epilogue
    uint64_t *done = tempty + 2;          // every MMA of this CTA complete
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    int *issued = reinterpret_cast<int *>(tmem_slot + 2);      // k-blocks whose copies were started
    int *consumed = reinterpret_cast<int *>(tmem_slot + 3);    // k-blocks whose copies were waited for
    // per epilogue warp, a 2 KB staging area for the TMA store of the row-major output: two
    // 32 x 16 BF16 boxes (double-buffered) or one 32 x 16 FP32 box
    uint8_t *stage_base = sB + STAGES * B_BYTES + 1024;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total = P.total;

    if (warp == 1) {   // whole warp: allocate two accumulators of BN columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"((uint32_t)(2 * BN))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], EPI_WARPS);
        }
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
    // all of the above before the kernel ahead has ended (this one's shared memory leaves no room
    // for a second block, and so for a second TMEM allocation, on an SM)
    early_next();
    early_wait();

    if (warp == 0) {
        // ---- TMA producer
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
                const Tile T = tile_at<BN>(P, t);
                for (int kb = 0; kb < T.nk; ++kb, ++g) {
                    const int s = g % STAGES;
                    if (g >= STAGES && !mbar_wait(&empty[s], (uint32_t)(((g / STAGES) - 1) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&full[s], A_BYTES + B_BYTES);
                    tma_load_2d(sA + s * A_BYTES, &P.a[T.p], T.kbeg + kb * BK, T.m0, &full[s]);
                    tma_load_2d(sB + s * B_BYTES, &P.b[T.p], T.kbeg + kb * BK, T.n0, &full[s]);
                    *issued = g + 1;
                }
            }
            if (!ok) {
                *abort = 1;
                atomicExch(err, 1);
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16(BM, BN);
            int g = 0, tl = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x, ++tl) {
                const int b = tl & 1;
                if (tl >= 2 && !mbar_wait(&tempty[b], (uint32_t)(((tl >> 1) - 1) & 1), abort)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(b * BN);
                const int nk = tile_at<BN>(P, t).nk;
                for (int kb = 0; kb < nk; ++kb, ++g) {
                    const int s = g % STAGES;
                    if (!mbar_wait(&full[s], (uint32_t)((g / STAGES) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    *consumed = g + 1;
                    tc_fence_after();
                    const uint64_t da = sdesc_k_sw128(smem_u32(sA + s * A_BYTES));
                    const uint64_t db = sdesc_k_sw128(smem_u32(sB + s * B_BYTES));
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)   // 32 bytes along K per instruction
                        umma_bf16(d, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, (kb | k) != 0);
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
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 and column quarter (w - 2) / 4
        const int q = warp & 3, part = (warp - 2) >> 2;
        constexpr int COLS = BN / (EPI_WARPS / 4);
        uint8_t *stage = stage_base + (warp - 2) * 2048;
        const bool f32 = store_mode == 2;
        int nstore = 0;   // TMA stores issued by this warp
        int tl = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x, ++tl) {
            const int b = tl & 1;
            const Tile T = tile_at<BN>(P, t);
            const int n0 = T.n0, m0 = T.m0, split = T.split;
            const int row = m0 + q * 32 + lane;
            // GELU' reads its pre-activations one step ahead, the first ones while the products are still
            // being formed; the bias comes into L1 meanwhile
            uint4 zn[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
            const __nv_bfloat16 *zin = static_cast<const __nv_bfloat16 *>(ep.zin);
            if (ep.mode == NPX_EPI_DGELU) load_pair(zin, ep.ldzi, row, n0 + part * COLS, zn);
            if (ep.bias && lane < COLS / 32)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(ep.bias + n0 + part * COLS + 32 * lane));
            if (!mbar_wait_warp(&tfull[b], (uint32_t)((tl >> 1) & 1), abort)) {
                if (lane == 0) {
                    *abort = 1;
                    atomicExch(err, 3);
                }
                break;
            }
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN);
#pragma unroll 1
            for (int c0 = part * COLS; c0 < (part + 1) * COLS; c0 += 16) {
                uint32_t r[16];
                tmem_ld16_issue(taddr + (uint32_t)c0, r);
                tmem_wait_ld();
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
                const uint4 z[2] = {zn[0], zn[1]};
                if (ep.mode == NPX_EPI_DGELU && c0 + 16 < (part + 1) * COLS) load_pair(zin, ep.ldzi, row, n0 + c0 + 16, zn);
                uint8_t *box = nullptr;
                if (store_mode) {
                    // the staging box is free once the store that last read it has read it
                    box = stage + (f32 ? 0 : (nstore & 1) * 1024);
                    if (f32 ? nstore >= 1 : nstore >= 2) {
                        if (lane == 0) {
                            if (f32) bulk_wait_read<0>();
                            else bulk_wait_read<1>();
                        }
                        __syncwarp();
                    }
                }
                epilogue16(ep, v, row, n0 + c0, split, store_mode, box + lane * (f32 ? 64 : 32), z);
                if (store_mode) {
                    fence_async_shared();
                    __syncwarp();
                    if (lane == 0) {
                        if (f32) tma_store_3d(&P.out[T.p], n0 + c0, m0 + q * 32, split, box);
                        else tma_store_2d(&P.out[T.p], n0 + c0, m0 + q * 32, box);
                        bulk_commit();
                    }
                    ++nstore;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
        }
        if (store_mode && lane == 0) bulk_wait_all();   // the stores have landed before the CTA ends
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // after a failure: let the copies still in flight land before the shared memory goes away
        for (int g = *consumed; g < *issued; ++g) mbar_wait(&full[g % STAGES], (uint32_t)((g / STAGES) & 1));
        // every MMA issued by this CTA has completed before its tensor memory is freed
        if (!mbar_wait(done, 0)) atomicExch(err, 4);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * BN)) : "memory");
    }
}

// ------------------------------------------------------------------------ host side

// 2D map of a row-major [rows x cols] BF16 matrix read in boxes of box_rows x 64 (128 B rows)
static bool make_map(CUtensorMap *m, const void *ptr, int rows, int cols, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    const cuuint32_t es[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// map of the row-major output written by the epilogue's TMA stores, in boxes of 32 rows x 16
// columns: BF16 [rows x cols] with row stride ld (2-D), or FP32 split partials
// [splits][rows x cols] with row stride ld and split stride split_stride (3-D)
static bool make_out_map(CUtensorMap *m, void *ptr, bool f32, int rows, int cols, long long ld, int splits,
                         long long split_stride) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t es = f32 ? 4 : 2;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)splits};
    const cuuint64_t strides[2] = {(cuuint64_t)ld * es, (cuuint64_t)(splits > 1 ? split_stride : ld * rows) * es};
    const cuuint32_t box[3] = {16, 32, 1};
    const cuuint32_t el[3] = {1, 1, 1};
    return fn(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, f32 ? 3 : 2, ptr, dims,
              strides, box, el, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int STORE>
static size_t smem_bytes() {
    return 1024 + (size_t)STAGES * (BM * BK * 2 + BN * BK * 2) + 1024 + (STORE ? (size_t)EPI_WARPS * 2048 : 0);
}

static int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
            n = 1;
    }
    return n;
}

template <int BN, int STORE, int G>
static cudaError_t launch(const Products<G> &P, const npx_gemm_epilogue &ep, int *err, cudaStream_t st) {
    const size_t smem = smem_bytes<BN, STORE>();
    cudaError_t e = cudaFuncSetAttribute(gemm_tn_kernel<BN, STORE, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int grid = P.total < sm_count() ? P.total : sm_count();
    return launch_early(gemm_tn_kernel<BN, STORE, G>, grid, THREADS, smem, st, P, ep, err);
}

// the product's place after those in P
template <int G>
static void append(Products<G> &P, int M, int N, int K, int splits, int BN) {
    const int i = P.n++;
    P.tiles_n[i] = N / BN;
    P.k_per_split[i] = K / splits;
    P.splits[i] = splits;
    P.first[i] = P.total;
    P.total += (M / BM) * (N / BN) * splits;
}

// products of one launch, and those of them with tiles BN wide
constexpr int MAX_G = GEMM_GROUP;

template <int BN>
static int run_group(const GemmF32 *p, int n, int *err, cudaStream_t st) {
    Products<MAX_G> P;
    P.n = P.total = 0;
    npx_gemm_epilogue ep{};
    ep.mode = NPX_EPI_F32;
    for (int i = 0; i < n; ++i) {
        if ((p[i].N % 256 == 0 ? 256 : 128) == BN) {
            if (!make_map(&P.a[P.n], p[i].A, p[i].M, p[i].K, BM) || !make_map(&P.b[P.n], p[i].B, p[i].N, p[i].K, BN) ||
                !make_out_map(&P.out[P.n], p[i].out, true, p[i].M, p[i].N, p[i].N, p[i].splits, (long long)p[i].M * p[i].N))
                return set_last_error(NPX_ECUDA, "grouped product: tensor-map encoding failed");
            append(P, p[i].M, p[i].N, p[i].K, p[i].splits, BN);
            ep.outf = p[i].out;   // (stored through the maps)
        }
        if (P.n == MAX_G || (i == n - 1 && P.n)) {
            cudaError_t e = launch<BN, 2>(P, ep, err, st);
            if (e != cudaSuccess) return set_last_error(NPX_ECUDA, cudaGetErrorString(e));
            P.n = P.total = 0;
        }
    }
    return NPX_OK;
}

// The bounded barrier wait on its own: thread 0 waits on a barrier that nothing completes; with
// use_abort, warp 1 raises the abort flag after ABORT_NS.  out[0] = 1 if the wait gave up (0 if
// the phase completed), out[1] = the wait in microseconds.
constexpr unsigned long long ABORT_NS = 1000000ull;   // 1 ms
__global__ void __launch_bounds__(64) wait_selftest_kernel(int use_abort, int *out) {
    __shared__ uint64_t bar;
    __shared__ volatile int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (use_abort && threadIdx.x == 32) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < ABORT_NS) {
        }
        abort_flag = 1;
    }
    if (threadIdx.x == 0) {
        const unsigned long long t0 = global_ns();
        const bool ok = mbar_wait(&bar, 0, use_abort ? &abort_flag : nullptr);
        out[0] = ok ? 0 : 1;
        out[1] = (int)((global_ns() - t0) / 1000ull);
    }
}

// A warp's wait whose lanes see different outcomes: the lower half waits on a barrier that has
// completed, the upper half on one that nothing completes until warp 1 raises the abort flag.
// out[0] = lanes told that they may go on, out[1] = the same when every lane's barrier has completed.
__global__ void __launch_bounds__(64) warp_wait_selftest_kernel(int *out) {
    __shared__ uint64_t bars[2];
    __shared__ volatile int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_arrive(&bars[0]);
    }
    __syncthreads();
    if (threadIdx.x == 32) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < ABORT_NS) {
        }
        abort_flag = 1;
    }
    if (threadIdx.x < 32) {
        const bool split = mbar_wait_warp(&bars[threadIdx.x >> 4], 0, &abort_flag);
        const bool all = mbar_wait_warp(&bars[0], 0, &abort_flag);
        const unsigned a = __ballot_sync(0xffffffffu, split), b = __ballot_sync(0xffffffffu, all);
        if (threadIdx.x == 0) {
            out[0] = __popc(a);
            out[1] = __popc(b);
        }
    }
}

}  // namespace gemm
}  // namespace npx

extern "C" int npx_gemm_warp_wait_selftest(int *split, int *complete, void *stream) {
    if (!split || !complete) return npx::set_last_error(NPX_EINVAL, "npx_gemm_warp_wait_selftest: null argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * sizeof(int));
    if (e != cudaSuccess) return npx::set_last_error(NPX_ENOMEM, cudaGetErrorString(e));
    int h[2] = {-1, -1};
    npx::gemm::warp_wait_selftest_kernel<<<1, 64, 0, st>>>(d);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    if (e != cudaSuccess) return npx::set_last_error(NPX_ECUDA, cudaGetErrorString(e));
    *split = h[0];
    *complete = h[1];
    return NPX_OK;
}

extern "C" int npx_gemm_wait_selftest(int use_abort, int *timed_out, int *elapsed_us, void *stream) {
    if (!timed_out || !elapsed_us) return npx::set_last_error(NPX_EINVAL, "npx_gemm_wait_selftest: null argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * sizeof(int));
    if (e != cudaSuccess) return npx::set_last_error(NPX_ENOMEM, cudaGetErrorString(e));
    int h[2] = {-1, -1};
    npx::gemm::wait_selftest_kernel<<<1, 64, 0, st>>>(use_abort ? 1 : 0, d);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    if (e != cudaSuccess) return npx::set_last_error(NPX_ECUDA, cudaGetErrorString(e));
    *timed_out = h[0];
    *elapsed_us = h[1];
    return NPX_OK;
}

int npx::gemm_group(const GemmF32 *p, int n, int *err, cudaStream_t st) {
    if (int rc = gemm::run_group<256>(p, n, err, st)) return rc;
    return gemm::run_group<128>(p, n, err, st);
}

extern "C" int npx_gemm_bf16(const void *A, const void *B, int M, int N, int K, int splits,
                             const npx_gemm_epilogue *ep, int *err, void *stream) {
    using namespace npx::gemm;
    if (!A || !B || !ep || !err) return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: null argument");
    if (splits < 1) return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: splits must be >= 1");
    const int BN = (N % 256 == 0) ? 256 : 128;
    if (M < BM || M % BM || N < 128 || N % 128 || K < BK || K % (BK * splits))
        return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: M must be a multiple of 128, N of 128, K of 64 x splits");
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15)
        return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: A and B must be 16-byte aligned");
    if (ep->mode != NPX_EPI_BIAS && ep->mode != NPX_EPI_BIAS_GELU && ep->mode != NPX_EPI_DGELU && ep->mode != NPX_EPI_F32)
        return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: unknown epilogue mode");
    if (ep->mode == NPX_EPI_F32 ? !ep->outf : (!ep->out && !ep->outT && !ep->outf))
        return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: no output");
    if (ep->mode == NPX_EPI_DGELU && !ep->zin) return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: DGELU needs zin");
    // the epilogue stores 16-byte vectors: 16-byte aligned rows of the row-major outputs
    auto rows16 = [](const void *p, long long ld, int elem) {
        return !p || ((reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld * elem) % 16 == 0);
    };
    if (!rows16(ep->bias, 0, 4) || !rows16(ep->out, ep->ldo, 2) || !rows16(ep->zsave, ep->ldz, 2) ||
        !rows16(ep->zin, ep->ldzi, 2) || !rows16(ep->outf, ep->ldf, 4) ||
        (ep->outf && splits > 1 && (ep->split_stride * 4) % 16 != 0) ||
        (ep->outT && (reinterpret_cast<uintptr_t>(ep->outT) & 1)))
        return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: outputs, bias and zin need 16-byte aligned rows");
    if (splits > 1 && ep->mode != NPX_EPI_F32) return npx::set_last_error(NPX_EINVAL, "npx_gemm_bf16: split K needs the F32 epilogue");
    Products<1> P;
    P.n = P.total = 0;
    append(P, M, N, K, splits, BN);
    CUtensorMap &tout = P.out[0];
    if (!make_map(&P.a[0], A, M, K, BM) || !make_map(&P.b[0], B, N, K, BN))
        return npx::set_last_error(NPX_ECUDA, "npx_gemm_bf16: tensor-map encoding failed");
    // the row-major output leaves through per-warp staging boxes and TMA stores: FP32 (store
    // mode 2), or BF16 when it is the only row-major output (mode 1)
    memset(&tout, 0, sizeof tout);
    int store_mode = 0;
    if (ep->outf && !(ep->out && ep->mode != NPX_EPI_F32)) {
        if (!make_out_map(&tout, ep->outf, true, M, N, ep->ldf, ep->mode == NPX_EPI_F32 ? splits : 1, ep->split_stride))
            return npx::set_last_error(NPX_ECUDA, "npx_gemm_bf16: output tensor-map encoding failed");
        store_mode = 2;
    } else if (ep->out && !ep->outf && ep->mode != NPX_EPI_F32) {
        if (!make_out_map(&tout, ep->out, false, M, N, ep->ldo, 1, 0))
            return npx::set_last_error(NPX_ECUDA, "npx_gemm_bf16: output tensor-map encoding failed");
        store_mode = 1;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    if (store_mode == 2)
        e = BN == 256 ? launch<256, 2>(P, *ep, err, st) : launch<128, 2>(P, *ep, err, st);
    else if (store_mode == 1)
        e = BN == 256 ? launch<256, 1>(P, *ep, err, st) : launch<128, 1>(P, *ep, err, st);
    else
        e = BN == 256 ? launch<256, 0>(P, *ep, err, st) : launch<128, 0>(P, *ep, err, st);
    if (e != cudaSuccess) return npx::set_last_error(NPX_ECUDA, cudaGetErrorString(e));
    return NPX_OK;
}
