// npx_mlp.cu -- the learned surrogate's network on the tensor cores: forward, backward and Adam.
//
// Layers are GEMMs of npx_gemm.cu with fused epilogues: hidden layers write the pre-activation z
// (kept for the backward pass), the activation gelu(z) and its transpose (the B operand of the
// weight-gradient GEMM); the output layer writes FP32.  Backward: dY = 2 (y - t) / M, then for
// each layer dW = dZ^T X (split-K GEMM over the batch, partial sums reduced in FP32),
// db = column sums of dZ, and dZ_prev = (dZ W) * gelu'(z_prev) (GEMM with the GELU' epilogue,
// also writing its transpose).  Adam updates FP32 master weights and refreshes the BF16 copies
// W and W^T that the GEMMs read.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <random>
#include <string>
#include <vector>

#include "../../include/npx_mlp.h"
#include "npx_internal.h"

typedef __nv_bfloat16 bf16;

namespace {

int pad_to(int n, int m) { return (n + m - 1) / m * m; }

// Tiles of 32 x 32 elements go through shared memory so that both the row-major output and its
// transpose are written in full lines: block (32, 8), grid (cols / 32, rows / 32).

// X = bf16(x) zero-padded to in_p columns, and optionally X^T [in_p x M]
__global__ void __launch_bounds__(256) pack_input_kernel(const float *x, int M, int n_in, int in_p,
                                                         bf16 *X, bf16 *XT) {
    __shared__ bf16 tile[32][33];
    npx::early_next();
    npx::early_wait();
    const int k0 = blockIdx.x * 32, m0 = blockIdx.y * 32, tx = threadIdx.x, ty = threadIdx.y;
    const int k = k0 + tx;
    float f[4];   // (all loads first)
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = k < n_in ? x[(size_t)(m0 + ty + 8 * i) * n_in + k] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bf16 v = __float2bfloat16_rn(f[i]);
        X[(size_t)(m0 + ty + 8 * i) * in_p + k] = v;
        tile[ty + 8 * i][tx] = v;
    }
    if (!XT) return;   // block-uniform
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) XT[(size_t)(k0 + ty + 8 * i) * M + m0 + tx] = tile[tx][ty + 8 * i];
}

// dY = 2 (y - t) / M on real outputs, 0 on the padding, and dY^T; loss += sum (y - t)^2 / M
__global__ void __launch_bounds__(256) loss_grad_kernel(const float *Y, const float *T, int M, int n_out, int out_p,
                                                        bf16 *dY, bf16 *dYT, float *loss) {
    __shared__ bf16 tile[32][33];
    __shared__ float red[8];
    npx::early_next();
    npx::early_wait();
    const int j0 = blockIdx.x * 32, m0 = blockIdx.y * 32, tx = threadIdx.x, ty = threadIdx.y;
    const float inv = 1.f / (float)M;
    float sq = 0.f;
    const int j = j0 + tx;
    float y[4], t4[4];   // (all loads first)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const size_t m = m0 + ty + 8 * i;
        y[i] = j < n_out ? Y[m * out_p + j] : 0.f;
        t4[i] = j < n_out ? T[m * n_out + j] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float d = y[i] - t4[i];
        sq += d * d * inv;
        const bf16 g = __float2bfloat16_rn(2.f * d * inv);
        dY[(size_t)(m0 + ty + 8 * i) * out_p + j] = g;
        tile[ty + 8 * i][tx] = g;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) dYT[(size_t)(j0 + ty + 8 * i) * M + m0 + tx] = tile[tx][ty + 8 * i];
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (tx == 0) red[ty] = sq;
    __syncthreads();
    if (ty == 0 && tx == 0) {
        float t = 0.f;
        for (int i = 0; i < 8; ++i) t += red[i];
        if (t != 0.f) atomicAdd(loss, t);
    }
}

// What is left of a backward pass for up to WGROUP layers in one launch: the split-K partials of each
// weight gradient summed in split order, and each bias gradient, the sum over the M entries of a row
// of the layer's transposed output gradient GT [rows x M] (read from the transpose so that every load
// is a full line).  Bound by launches: layer by layer these were ten launches of 4 to 6 us each,
// 49 us of a 357 us minibatch of 8,192 rows (271 -> 4 x 512 -> 247); with Adam's ten below as one, a
// minibatch took 294 us (235 now).
constexpr int WGROUP = npx::GEMM_GROUP;   // layers whose weight gradients are formed together
struct GradLayer {
    const float *part;      // [splits][n], or NULL: the gradient is written already
    float *dW;
    const bf16 *GT;
    float *db;
    int splits, rows, first;    // first: the layer's first block
    long long n;
};
struct GradGroup {
    GradLayer l[WGROUP];
    int layers;
};

__global__ void __launch_bounds__(256) grads_finish_kernel(const __grid_constant__ GradGroup G, int M) {
    int k = 0;
    while (k + 1 < G.layers && (int)blockIdx.x >= G.l[k + 1].first) ++k;
    const GradLayer &g = G.l[k];
    npx::early_next();
    npx::early_wait();
    int blk = (int)blockIdx.x - g.first;
    if (blk >= g.rows) {   // four weights a thread
        const long long i = ((long long)(blk - g.rows) * 256 + threadIdx.x) * 4;
        if (i >= g.n) return;
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int s = 0; s < g.splits; ++s) {
            const float4 p = *reinterpret_cast<const float4 *>(g.part + (size_t)s * g.n + i);
            t.x += p.x; t.y += p.y; t.z += p.z; t.w += p.w;
        }
        *reinterpret_cast<float4 *>(g.dW + i) = t;
        return;
    }
    __shared__ float red[8];
    const bf16 *row = g.GT + (size_t)blk * M;
    float s = 0.f;
    for (int m = threadIdx.x * 8; m < M; m += 256 * 8) {
        const uint4 u = *reinterpret_cast<const uint4 *>(row + m);
        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
            const float2 f = __bfloat1622float2(h[k2]);
            s += f.x + f.y;
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int i = 0; i < 8; ++i) t += red[i];
        g.db[blk] = t;
    }
}

constexpr int GROUP = 16;
// Adam on FP32 master parameters of up to GROUP layers in one launch.  A block takes a 32 x 32 tile
// of a weight matrix, so that the refreshed BF16 copy and, through shared memory, its transpose are
// both written in full lines (element by element the transpose wrote two bytes to a sector), or 256
// biases.  It was ten launches of 4.5 us.
struct AdamLayer {
    float *W, *mW, *vW, *b, *mb, *vb;
    const float *dW, *db;
    bf16 *Wb, *WbT;
    int rows, cols, first;
};
struct AdamGroup {
    AdamLayer l[GROUP];
    int layers;
    float lr, b1, b2, eps, bc1, bc2;
};

__device__ __forceinline__ float adam_update(const AdamGroup &A, float *p, float *m, float *v, float gi) {
    const float mi = A.b1 * *m + (1.f - A.b1) * gi;
    const float vi = A.b2 * *v + (1.f - A.b2) * gi * gi;
    *m = mi;
    *v = vi;
    const float pi = *p - A.lr * (mi / A.bc1) / (sqrtf(vi / A.bc2) + A.eps);
    *p = pi;
    return pi;
}

__global__ void __launch_bounds__(256) adam_kernel(const __grid_constant__ AdamGroup A) {
    __shared__ bf16 tile[32][33];
    int k = 0;
    while (k + 1 < A.layers && (int)blockIdx.x >= A.l[k + 1].first) ++k;
    const AdamLayer &g = A.l[k];
    npx::early_next();
    npx::early_wait();
    const int blk = (int)blockIdx.x - g.first, tc = g.cols / 32, tiles = (g.rows / 32) * tc;
    if (blk >= tiles) {
        const int i = (blk - tiles) * 256 + threadIdx.x;
        if (i < g.rows) adam_update(A, g.b + i, g.mb + i, g.vb + i, g.db[i]);
        return;
    }
    const int r0 = blk / tc * 32, c0 = blk % tc * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const size_t e = (size_t)(r0 + ty + 8 * i) * g.cols + c0 + tx;
        const bf16 w = __float2bfloat16_rn(adam_update(A, g.W + e, g.mW + e, g.vW + e, g.dW[e]));
        g.Wb[e] = w;
        tile[ty + 8 * i][tx] = w;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) g.WbT[(size_t)(c0 + ty + 8 * i) * g.rows + r0 + tx] = tile[tx][ty + 8 * i];
}

__global__ void to_bf16_kernel(const float *p, long long n, int cols, int rows, bf16 *pb, bf16 *pbT) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bf16 b = __float2bfloat16_rn(p[i]);
    pb[i] = b;
    pbT[(size_t)(i % cols) * rows + (i / cols)] = b;
}

__global__ void unpad_kernel(const float *__restrict__ Y, int M, int out_p, int n_out, float *y) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)M * n_out) return;
    const int m = (int)(i / n_out), j = (int)(i % n_out);
    y[i] = Y[(size_t)m * out_p + j];
}

inline unsigned blocks_for(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// Column sums and sums of squares in FP64.  A cluster of MOM_CTAS blocks covers CW columns, its
// blocks and their MOM_THREADS / CW row lanes taking every MOM_CTAS * MOM_THREADS / CW-th row; each
// lane sums its rows in order, then a warp's lanes, a block's warps and the cluster's blocks are
// added in a fixed order (the blocks' sums over distributed shared memory, so there is no
// workspace and no atomic): every column's sum repeats bit for bit.
// Bound by the FP64 pipe (an add and a fused multiply-add per element, two lanes a clock and SM on
// this part), so the work has to reach every SM: 65,536 x 271 took 590 us on nine blocks of 32 columns
// each, 102 us on 272 (the first pass on new rows 1.80 ms and 0.17 ms).
constexpr int MOM_CTAS = 8, MOM_THREADS = 256;

template <int CW>
__global__ void __cluster_dims__(MOM_CTAS, 1, 1) __launch_bounds__(MOM_THREADS)
column_moments_kernel(const float *__restrict__ X, long long rows, int cols, double *sum, double *sumsq) {
    namespace cg = cooperative_groups;
    constexpr int TY = MOM_THREADS / CW, WARPS = MOM_THREADS / 32;
    __shared__ double red[WARPS][2][CW];
    __shared__ double part[2][CW];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tx = threadIdx.x % CW, ty = threadIdx.x / CW;
    const int c = (blockIdx.x / MOM_CTAS) * CW + tx, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long step = (long long)MOM_CTAS * TY;
    double s = 0.0, q = 0.0;
    if (c < cols) {
        const float *p = X + c;
        long long r = (long long)rank * TY + ty;
        for (; r + 7 * step < rows; r += 8 * step) {   // eight loads in flight
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = p[(r + k * step) * cols];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const double d = (double)v[k];
                s += d;
                q = fma(d, d, q);
            }
        }
        for (; r < rows; r += step) {
            const double d = (double)p[r * cols];
            s += d;
            q = fma(d, d, q);
        }
    }
#pragma unroll
    for (int o = 16; o >= CW; o >>= 1) {   // lanes of one column are CW apart
        s += __shfl_down_sync(0xffffffffu, s, o);
        q += __shfl_down_sync(0xffffffffu, q, o);
    }
    if (lane < CW) {
        red[warp][0][lane] = s;
        red[warp][1][lane] = q;
    }
    __syncthreads();
    if (threadIdx.x < 2 * CW) {
        const int k = threadIdx.x / CW, x = threadIdx.x % CW;
        double t = 0.0;
        for (int w = 0; w < WARPS; ++w) t += red[w][k][x];
        part[k][x] = t;
    }
    cl.sync();
    if (rank == 0 && threadIdx.x < 2 * CW) {
        const int k = threadIdx.x / CW, x = threadIdx.x % CW, col = (blockIdx.x / MOM_CTAS) * CW + x;
        double t = 0.0;
        for (int b = 0; b < MOM_CTAS; ++b) t += *cl.map_shared_rank(&part[k][x], b);
        if (col < cols) (k == 0 ? sum : sumsq)[col] += t;
    }
    cl.sync();   // no block leaves while its sums are read
}

}  // namespace

struct npx_mlp {
    npx_mlp_desc d{};
    cudaStream_t stream = nullptr, own = nullptr;
    int L = 0;                                  // layers (hidden + output)
    std::vector<int> din, dout, rin, rout;      // padded and real widths per layer
    std::vector<float *> W, b, mW, vW, mb, vb, dW, db;
    std::vector<bf16 *> Wb, WbT;
    bf16 *X0 = nullptr, *X0T = nullptr, *dY = nullptr, *dYT = nullptr;
    std::vector<bf16 *> Z, X, XT, dZ, dZT;      // hidden layers
    // split-K partials of the layers' weight gradients: one buffer, which each WGROUP layers use anew
    // (64 bytes a weight of a 512 x 512 layer: a buffer of every layer's own would be three quarters
    // of a deep network's memory)
    float *part = nullptr;
    float *Y = nullptr, *loss_tmp = nullptr;
    int *err = nullptr;
    int t = 0;
    std::vector<void *> bufs;
};

namespace {

template <class T>
bool dalloc(npx_mlp *n, T **p, size_t count) {
    void *q = nullptr;
    if (cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) return false;
    cudaMemset(q, 0, std::max<size_t>(count, 1) * sizeof(T));
    n->bufs.push_back(q);
    *p = static_cast<T *>(q);
    return true;
}

int gemm(npx_mlp *n, const void *A, const void *B, int M, int N, int K, int splits, const npx_gemm_epilogue &ep) {
    return npx_gemm_bf16(A, B, M, N, K, splits, &ep, n->err, n->stream);
}

npx_gemm_epilogue epi(int mode) {
    npx_gemm_epilogue e{};
    e.mode = mode;
    return e;
}

// splits of a weight gradient's K (the batch): as many as fill the chip; K = 0: the most of any batch
int pick_splits(int Mg, int Ng, int K) {
    const int tiles = (Mg / 128) * (Ng / (Ng % 256 == 0 ? 256 : 128));
    int s = 1;
    while (s * 2 * tiles <= 152 && K % (64 * s * 2) == 0 && s < 64) s *= 2;
    return s;
}

int check(npx_mlp *n, int M) {
    if (!n) return npx::set_last_error(NPX_EINVAL, "null network");
    if (M < 128 || M % 128 || M > n->d.max_batch)
        return npx::set_last_error(NPX_EINVAL, "M must be a multiple of 128 and at most max_batch");
    return NPX_OK;
}

#define CU(call)                                                                                 \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess) return npx::set_last_error(NPX_ECUDA, cudaGetErrorString(e_));    \
    } while (0)
#define RC(call)                    \
    do {                            \
        int r_ = (call);            \
        if (r_) return r_;          \
    } while (0)

// the layers, from the packed BF16 input X0
int forward_layers(npx_mlp *n, int M, bool train) {
    const bf16 *A = n->X0;
    for (int l = 0; l < n->L - 1; ++l) {
        npx_gemm_epilogue e = epi(NPX_EPI_BIAS_GELU);
        e.bias = n->b[l];
        e.out = n->X[l];
        e.ldo = n->dout[l];
        if (train) {
            e.zsave = n->Z[l];
            e.ldz = n->dout[l];
            e.outT = n->XT[l];
            e.ldt = M;
        }
        RC(gemm(n, A, n->Wb[l], M, n->dout[l], n->din[l], 1, e));
        A = n->X[l];
    }
    const int l = n->L - 1;
    npx_gemm_epilogue e = epi(NPX_EPI_BIAS);
    e.bias = n->b[l];
    e.outf = n->Y;
    e.ldf = n->dout[l];
    RC(gemm(n, A, n->Wb[l], M, n->dout[l], n->din[l], 1, e));
    return NPX_OK;
}

// The network as the fused inference kernel takes it; false when it does not fit (it then runs
// layer by layer).
bool fused_net(const npx_mlp *n, npx::FusedNet *f) {
    *f = npx::FusedNet{};
    if (n->L > npx::FUSED_LAYERS) return false;
    f->layers = n->L;
    for (int l = 0; l < n->L; ++l) {
        f->k[l] = n->din[l];
        f->n[l] = n->dout[l];
        f->bias[l] = n->b[l];
        f->w[l] = n->Wb[l];
    }
    return npx::fused_fits(*f);
}

int forward_impl(npx_mlp *n, const float *x, int M, bool train) {
    const int in_p = n->din[0];
    CU(npx::launch_early(pack_input_kernel, dim3(in_p / 32, M / 32), dim3(32, 8), 0, n->stream, x, M, n->d.n_in, in_p, n->X0,
                         train ? n->X0T : nullptr));
    return forward_layers(n, M, train);
}

}  // namespace

cudaStream_t npx::mlp_stream(const npx_mlp *n) { return n->stream; }
int npx::mlp_max_batch(const npx_mlp *n) { return n->d.max_batch; }
void npx::mlp_dims(const npx_mlp *n, int *n_in, int *n_out) {
    *n_in = n->d.n_in;
    *n_out = n->d.n_out;
}
__nv_bfloat16 *npx::mlp_input(npx_mlp *n, int *ld) {
    *ld = n->din[0];
    return n->X0;
}
int npx::mlp_forward_packed(npx_mlp *n, int M, int cols) {
    RC(check(n, M));
    npx::FusedNet f;
    if (!fused_net(n, &f)) return forward_layers(n, M, false);
    const int l = n->L - 1;
    f.n[l] = std::min(n->dout[l], pad_to(cols, 128));   // only the blocks of outputs that are read
    CU(npx::launch_mlp_fused(f, nullptr, 0, n->X0, n->Y, n->dout[l], cols, M, n->err, n->stream));
    return NPX_OK;
}
const float *npx::mlp_output(const npx_mlp *n, int *ld) {
    *ld = n->dout[n->L - 1];
    return n->Y;
}

extern "C" {

int npx_mlp_create(const npx_mlp_desc *d, npx_mlp **out) {
    if (!d || !out) return npx::set_last_error(NPX_EINVAL, "null argument");
    *out = nullptr;
    if (d->n_in < 1 || d->n_out < 1 || d->n_hidden < 128 || d->n_hidden % 128 || d->n_hidden_layers < 1 ||
        d->max_batch < 128 || d->max_batch % 128)
        return npx::set_last_error(NPX_EINVAL, "bad network sizes (hidden width and max_batch multiples of 128)");
    npx_mlp *n = new (std::nothrow) npx_mlp();
    if (!n) return npx::set_last_error(NPX_ENOMEM, "out of host memory");
    n->d = *d;
    n->stream = static_cast<cudaStream_t>(d->stream);
    if (!n->stream) {
        if (cudaStreamCreateWithFlags(&n->own, cudaStreamNonBlocking) != cudaSuccess) {
            delete n;
            return npx::set_last_error(NPX_ECUDA, "stream creation failed");
        }
        n->stream = n->own;
    }
    n->L = d->n_hidden_layers + 1;
    const int H = d->n_hidden, Mx = d->max_batch;
    for (int l = 0; l < n->L; ++l) {
        n->rin.push_back(l == 0 ? d->n_in : H);
        n->rout.push_back(l == n->L - 1 ? d->n_out : H);
        n->din.push_back(l == 0 ? pad_to(d->n_in, 128) : H);
        n->dout.push_back(l == n->L - 1 ? pad_to(d->n_out, 128) : H);
    }
    bool ok = true;
    n->W.resize(n->L); n->b.resize(n->L); n->mW.resize(n->L); n->vW.resize(n->L); n->mb.resize(n->L);
    n->vb.resize(n->L); n->dW.resize(n->L); n->db.resize(n->L); n->Wb.resize(n->L); n->WbT.resize(n->L);
    for (int l = 0; l < n->L && ok; ++l) {
        const size_t nw = (size_t)n->dout[l] * n->din[l];
        ok = dalloc(n, &n->W[l], nw) && dalloc(n, &n->mW[l], nw) && dalloc(n, &n->vW[l], nw) &&
             dalloc(n, &n->dW[l], nw) && dalloc(n, &n->Wb[l], nw) && dalloc(n, &n->WbT[l], nw) &&
             dalloc(n, &n->b[l], n->dout[l]) && dalloc(n, &n->mb[l], n->dout[l]) &&
             dalloc(n, &n->vb[l], n->dout[l]) && dalloc(n, &n->db[l], n->dout[l]);
    }
    size_t parts = 0, group = 0;   // (in the order of the backward pass, at the most splits of any batch)
    for (int l = n->L - 1; l >= 0; --l) {
        const int ms = pick_splits(n->dout[l], n->din[l], 0);
        if ((n->L - 1 - l) % WGROUP == 0) group = 0;
        group += ms > 1 ? (size_t)ms * n->dout[l] * n->din[l] : 0;
        parts = std::max(parts, group);
    }
    ok = ok && dalloc(n, &n->part, parts);
    n->Z.resize(n->L - 1); n->X.resize(n->L - 1); n->XT.resize(n->L - 1); n->dZ.resize(n->L - 1); n->dZT.resize(n->L - 1);
    for (int l = 0; l < n->L - 1 && ok; ++l)
        ok = dalloc(n, &n->Z[l], (size_t)Mx * H) && dalloc(n, &n->X[l], (size_t)Mx * H) &&
             dalloc(n, &n->XT[l], (size_t)Mx * H) && dalloc(n, &n->dZ[l], (size_t)Mx * H) &&
             dalloc(n, &n->dZT[l], (size_t)Mx * H);
    ok = ok && dalloc(n, &n->X0, (size_t)Mx * n->din[0]) && dalloc(n, &n->X0T, (size_t)Mx * n->din[0]) &&
         dalloc(n, &n->Y, (size_t)Mx * n->dout[n->L - 1]) && dalloc(n, &n->dY, (size_t)Mx * n->dout[n->L - 1]) &&
         dalloc(n, &n->dYT, (size_t)Mx * n->dout[n->L - 1]) && dalloc(n, &n->err, 1) && dalloc(n, &n->loss_tmp, 1);
    if (!ok) {
        npx_mlp_destroy(n);
        return npx::set_last_error(NPX_ENOMEM, "device allocation failed");
    }
    // He-normal initial weights (std sqrt(2 / fan_in)), zero biases
    std::mt19937_64 rng(d->seed);
    std::vector<float> host;
    for (int l = 0; l < n->L; ++l) {
        host.assign((size_t)n->dout[l] * n->din[l], 0.f);
        std::normal_distribution<float> nd(0.f, std::sqrt(2.f / n->rin[l]));
        for (int o = 0; o < n->rout[l]; ++o)
            for (int i = 0; i < n->rin[l]; ++i) host[(size_t)o * n->din[l] + i] = nd(rng);
        CU(cudaMemcpy(n->W[l], host.data(), host.size() * sizeof(float), cudaMemcpyHostToDevice));
        to_bf16_kernel<<<blocks_for((long long)host.size()), 256, 0, n->stream>>>(
            n->W[l], (long long)host.size(), n->din[l], n->dout[l], n->Wb[l], n->WbT[l]);
    }
    CU(cudaStreamSynchronize(n->stream));
    *out = n;
    return NPX_OK;
}

int npx_mlp_destroy(npx_mlp *n) {
    if (!n) return NPX_OK;
    if (n->stream) cudaStreamSynchronize(n->stream);
    for (void *p : n->bufs) cudaFree(p);
    if (n->own) cudaStreamDestroy(n->own);
    delete n;
    return NPX_OK;
}

size_t npx_mlp_param_count(const npx_mlp *n) {
    if (!n) return 0;
    size_t c = 0;
    for (int l = 0; l < n->L; ++l) c += (size_t)n->rout[l] * n->rin[l] + n->rout[l];
    return c;
}

static int copy_params(npx_mlp *n, float *host, size_t count, bool to_device, bool grads) {
    if (!n || !host) return npx::set_last_error(NPX_EINVAL, "null argument");
    if (count != npx_mlp_param_count(n)) return npx::set_last_error(NPX_EINVAL, "parameter count mismatch");
    CU(cudaStreamSynchronize(n->stream));
    int err = 0;
    CU(cudaMemcpy(&err, n->err, sizeof err, cudaMemcpyDeviceToHost));
    if (err) return npx::set_last_error(NPX_ETIMEOUT, "a tensor-core GEMM barrier timed out");
    size_t off = 0;
    for (int l = 0; l < n->L; ++l) {
        float *Wd = grads ? n->dW[l] : n->W[l];
        float *bd = grads ? n->db[l] : n->b[l];
        // rows of W are padded to din[l] columns: copy row by row with a 2D copy
        const size_t sp = (size_t)n->din[l] * sizeof(float), hp = (size_t)n->rin[l] * sizeof(float);
        if (to_device)
            CU(cudaMemcpy2D(Wd, sp, host + off, hp, hp, n->rout[l], cudaMemcpyHostToDevice));
        else
            CU(cudaMemcpy2D(host + off, hp, Wd, sp, hp, n->rout[l], cudaMemcpyDeviceToHost));
        off += (size_t)n->rout[l] * n->rin[l];
        if (to_device)
            CU(cudaMemcpy(bd, host + off, n->rout[l] * sizeof(float), cudaMemcpyHostToDevice));
        else
            CU(cudaMemcpy(host + off, bd, n->rout[l] * sizeof(float), cudaMemcpyDeviceToHost));
        off += n->rout[l];
        if (to_device && !grads) {
            const long long nw = (long long)n->dout[l] * n->din[l];
            to_bf16_kernel<<<blocks_for(nw), 256, 0, n->stream>>>(n->W[l], nw, n->din[l], n->dout[l], n->Wb[l],
                                                                  n->WbT[l]);
            CU(cudaGetLastError());
        }
    }
    CU(cudaStreamSynchronize(n->stream));
    return NPX_OK;
}

int npx_mlp_params_set(npx_mlp *n, const float *p, size_t c) { return copy_params(n, const_cast<float *>(p), c, true, false); }
int npx_mlp_params_get(npx_mlp *n, float *p, size_t c) { return copy_params(n, p, c, false, false); }
int npx_mlp_grads_get(npx_mlp *n, float *g, size_t c) { return copy_params(n, g, c, false, true); }

int npx_mlp_forward(npx_mlp *n, const float *x, float *y, int M) {
    RC(check(n, M));
    if (!x || !y) return npx::set_last_error(NPX_EINVAL, "null array");
    npx::FusedNet f;
    // (outputs that overlap the inputs need every input read first: layer by layer)
    const bool apart = x + (size_t)M * n->d.n_in <= y || y + (size_t)M * n->d.n_out <= x;
    if (apart && fused_net(n, &f)) {
        CU(npx::launch_mlp_fused(f, x, n->d.n_in, nullptr, y, n->d.n_out, n->d.n_out, M, n->err, n->stream));
        return NPX_OK;
    }
    RC(forward_impl(n, x, M, false));
    const int out_p = n->dout[n->L - 1];
    unpad_kernel<<<blocks_for((long long)M * n->d.n_out), 256, 0, n->stream>>>(n->Y, M, out_p, n->d.n_out, y);
    CU(cudaGetLastError());
    return NPX_OK;
}

int npx_mlp_backward(npx_mlp *n, const float *x, const float *t, int M, float *loss) {
    RC(check(n, M));
    if (!x || !t || !loss) return npx::set_last_error(NPX_EINVAL, "null array");
    RC(forward_impl(n, x, M, true));
    const int L = n->L, H = n->d.n_hidden, out_p = n->dout[L - 1];
    CU(cudaMemsetAsync(loss, 0, sizeof(float), n->stream));
    CU(npx::launch_early(loss_grad_kernel, dim3(out_p / 32, M / 32), dim3(32, 8), 0, n->stream, n->Y, t, M, n->d.n_out, out_p,
                         n->dY, n->dYT, loss));
    const bf16 *G = n->dY, *GT = n->dYT;     // gradient of the current layer's output
    std::vector<npx::GemmF32> wgrads;
    std::vector<GradLayer> finish;
    float *part = n->part;
    for (int l = L - 1; l >= 0; --l) {
        const int No = n->dout[l], Ni = n->din[l];
        // dW = G^T X_prev: A = G^T [No x M], B = X_prev^T [Ni x M]
        const bf16 *XprevT = l > 0 ? n->XT[l - 1] : n->X0T;
        const int splits = pick_splits(No, Ni, M);
        if ((L - 1 - l) % WGROUP == 0) part = n->part;
        float *out = splits > 1 ? part : n->dW[l];
        if (splits > 1) part += (size_t)splits * No * Ni;
        wgrads.push_back(npx::GemmF32{GT, XprevT, out, No, Ni, M, splits});
        finish.push_back(GradLayer{splits > 1 ? out : nullptr, n->dW[l], GT, n->db[l], splits, No, 0, (long long)No * Ni});
        if (l > 0) {
            // dZ_prev = (G W) * gelu'(Z_prev): A = G [M x No], B = W^T [Ni x No]
            npx_gemm_epilogue e2 = epi(NPX_EPI_DGELU);
            e2.zin = n->Z[l - 1];
            e2.ldzi = H;
            e2.out = n->dZ[l - 1];
            e2.ldo = H;
            e2.outT = n->dZT[l - 1];
            e2.ldt = M;
            RC(gemm(n, G, n->WbT[l], M, Ni, No, 1, e2));
            G = n->dZ[l - 1];
            GT = n->dZT[l - 1];
        }
    }
    // The weight gradients together, after the chain that the others hang on.  One alone is a tile of
    // a few K blocks for each SM, whose epilogue nothing hides: four minibatches of 8,192 rows
    // (271 -> 4 x 512 -> 247) 1,025 -> 1,002 us.
    // (WGROUP layers' partials at a time: the next layers' products overwrite them)
    for (int l = 0; l < L; l += WGROUP) {
        GradGroup group;
        group.layers = std::min(WGROUP, L - l);
        RC(npx::gemm_group(wgrads.data() + l, group.layers, n->err, n->stream));
        int blocks = 0;
        for (int k = 0; k < group.layers; ++k) {
            GradLayer &g = group.l[k] = finish[l + k];
            g.first = blocks;
            blocks += g.rows + (g.part ? (int)blocks_for(g.n / 4) : 0);
        }
        CU(npx::launch_early(grads_finish_kernel, blocks, 256, 0, n->stream, group, M));
    }
    return NPX_OK;
}

int npx_column_moments(const float *X, long long rows, int cols, double *sum, double *sumsq, void *stream) {
    if (!X || !sum || !sumsq || rows < 0 || cols < 1) return npx::set_last_error(NPX_EINVAL, "npx_column_moments: bad arguments");
    if (rows == 0) return NPX_OK;
    // the widest column group (8: full 32-byte sectors) whose clusters still give every SM a block
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto launch = [&](auto kernel, int cw) {
        kernel<<<(unsigned)((cols + cw - 1) / cw) * MOM_CTAS, MOM_THREADS, 0, st>>>(X, rows, cols, sum, sumsq);
    };
    if (cols > 8 * 18) launch(column_moments_kernel<8>, 8);
    else if (cols > 4 * 18) launch(column_moments_kernel<4>, 4);
    else launch(column_moments_kernel<2>, 2);
    CU(cudaGetLastError());
    return NPX_OK;
}

int npx_mlp_adam_step(npx_mlp *n) {
    if (!n) return npx::set_last_error(NPX_EINVAL, "null network");
    n->t += 1;
    const float b1 = n->d.beta1, b2 = n->d.beta2;
    const float bc1 = 1.f - std::pow(b1, (float)n->t), bc2 = 1.f - std::pow(b2, (float)n->t);
    AdamGroup A;
    A.lr = n->d.lr; A.b1 = b1; A.b2 = b2; A.eps = n->d.eps; A.bc1 = bc1; A.bc2 = bc2;
    A.layers = 0;
    int blocks = 0;
    for (int l = 0; l < n->L; ++l) {
        const int rows = n->dout[l], cols = n->din[l];
        A.l[A.layers++] = AdamLayer{n->W[l], n->mW[l], n->vW[l], n->b[l], n->mb[l], n->vb[l], n->dW[l], n->db[l],
                                    n->Wb[l], n->WbT[l], rows, cols, blocks};
        blocks += (rows / 32) * (cols / 32) + (int)blocks_for(rows);
        if (A.layers == GROUP || l == n->L - 1) {
            CU(npx::launch_early(adam_kernel, blocks, 256, 0, n->stream, A));
            A.layers = 0;
            blocks = 0;
        }
    }
    return NPX_OK;
}

int npx_mlp_set_lr(npx_mlp *n, float lr) {
    if (!n) return npx::set_last_error(NPX_EINVAL, "null network");
    if (!(lr > 0.f) || !std::isfinite(lr)) return npx::set_last_error(NPX_EINVAL, "learning rate must be positive");
    n->d.lr = lr;
    return NPX_OK;
}

}  // extern "C"
