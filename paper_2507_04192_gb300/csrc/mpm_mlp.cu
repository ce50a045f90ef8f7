// Small fully connected network trained and evaluated on the tcgen05 tensor
// cores: the learned warm start of the basal-friction inversion (a map from
// tracked-particle observations to per-segment friction coefficients).
//
// Layers: z_l = x_l W_l^T + b_l, x_{l+1} = GELU(z_l) (exact erf form) or
// max(z_l, 0) for the hidden layers, output y = lo + (hi - lo) sigmoid(z_last)
// or y = z_last (the coordinate network of Eq. nn_apprx).  Weights are kept in
// fp32 (Adam state too) with bf16 copies (and their transposes) as GEMM
// operands; activations and back-propagated gradients enter the GEMMs as bf16
// and every GEMM accumulates in fp32 in TMEM.  Loss: mean squared error.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mpm.h"
#include "mpm_umma.cuh"

using namespace mpm;

namespace {

__global__ void k_f32_to_bf16(const float *__restrict__ in, __nv_bfloat16 *__restrict__ out, int64_t n)
{
    pdl_enter();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __float2bfloat16_rn(in[i]);
}

// out[c][r] = in[r][c] (rows x cols -> cols x rows), bf16.
__global__ void k_transpose_bf16(const __nv_bfloat16 *__restrict__ in, __nv_bfloat16 *__restrict__ out, int rows,
                                 int cols)
{
    __shared__ __nv_bfloat16 tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int j = threadIdx.y; j < 32; j += blockDim.y) {
        const int r = r0 + j, c = c0 + threadIdx.x;
        if (r < rows && c < cols) tile[j][threadIdx.x] = in[(int64_t)r * cols + c];
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += blockDim.y) {
        const int c = c0 + j, r = r0 + threadIdx.x;
        if (r < rows && c < cols) out[(int64_t)c * rows + r] = tile[threadIdx.x][j];
    }
}

// Network input: bf16 rows and their transpose (cols x rows) in one pass; the step's
// loss is cleared on the way.
__global__ void __launch_bounds__(256) k_prepare_input(const float *__restrict__ x, __nv_bfloat16 *__restrict__ out,
                                                       __nv_bfloat16 *__restrict__ outT, int rows, int cols,
                                                       double *__restrict__ loss)
{
    __shared__ __nv_bfloat16 tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    pdl_enter();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *loss = 0.0;
    for (int j = ty; j < 32; j += 8) {
        const int r = r0 + j, c = c0 + tx;
        if (r < rows && c < cols) {
            const __nv_bfloat16 h = __float2bfloat16_rn(x[(int64_t)r * cols + c]);
            tile[j][tx] = h;
            out[(int64_t)r * cols + c] = h;
        }
    }
    __syncthreads();
    for (int j = ty; j < 32; j += 8) {
        const int c = c0 + j, r = r0 + tx;
        if (r < rows && c < cols) outT[(int64_t)c * rows + r] = tile[tx][j];
    }
}

// Gradient of the output layer's pre-activation, dz = g (hi - lo) s (1 - s) with s =
// sigmoid(z) (dz = g for the linear output), in fp32, bf16 and transposed bf16.
// With a loss pointer, src holds the targets, g = 2 (y - t) / n and the loss mean
// (y - t)^2 is added up, one atomic per block (one per warp: 8192 x 1024 outputs 106 us,
// 68 so); else src holds g = dL/dy.
__global__ void __launch_bounds__(256) k_output_grad(const float *__restrict__ y, const float *__restrict__ src,
                                                     const float *__restrict__ z, float *__restrict__ dz,
                                                     __nv_bfloat16 *__restrict__ dzb, __nv_bfloat16 *__restrict__ dzbT,
                                                     int rows, int cols, float lo, float hi, int linear,
                                                     double *__restrict__ loss)
{
    __shared__ __nv_bfloat16 tile[32][33];
    __shared__ double part[8];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    const int64_t n = (int64_t)rows * cols;
    pdl_enter();
    double acc = 0.0;
    const int c1 = c0 + tx;
    float gs[4], ys[4], zs[4];
    auto live = [&](int j) { return r0 + ty + 8 * j < rows && c1 < cols; };
    auto at = [&](int j) { return (int64_t)(r0 + ty + 8 * j) * cols + c1; };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!live(j)) continue;
        gs[j] = src[at(j)];
        ys[j] = y[at(j)];
        zs[j] = z[at(j)];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!live(j)) continue;
        float g = gs[j];
        if (loss != nullptr) {
            const float e = ys[j] - g;
            acc += (double)e * e;
            g = 2.0f * e / (float)n;
        }
        if (!linear) {
            const float s = 1.0f / (1.0f + expf(-zs[j]));
            g = g * (hi - lo) * s * (1.0f - s);
        }
        dz[at(j)] = g;
        const __nv_bfloat16 h = __float2bfloat16_rn(g);
        dzb[at(j)] = h;
        tile[ty + 8 * j][tx] = h;
    }
    if (loss != nullptr) {
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (tx == 0) part[ty] = acc;
    }
    __syncthreads();
    if (loss != nullptr && threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) acc += part[w];
        atomicAdd(loss, acc / (double)n);
    }
    for (int j = ty; j < 32; j += 8) {
        const int c = c0 + j, r = r0 + tx;
        if (r < rows && c < cols) dzbT[(int64_t)c * rows + r] = tile[tx][j];
    }
}

// The end of a training step over all layers, one launch (a training step was 38 small
// launches: separate conversions, transposes, column sums on one block, activation
// gradients, Adam and copies per layer; with those in the GEMM epilogues, k_output_grad
// and here it is 9, and 310 -> 70 us at batch 256 on 640-256-256-32; the loads of a
// block go ahead of its stores, which the compiler may not reorder: 13 us of it before):
// the bias gradients db[c] = sum_r dz[r][c], added in the order of the rows (blocks
// [0, n_bias), 32 columns each, 256 rows at a time through shared memory), and with
// update Adam on the fp32 master parameters (bias-corrected moments) with the weights'
// bf16 copies and transposes (32 x 32 tiles of the weights).
constexpr int kMaxLayers = 8;
struct StepEnd {
    struct Layer {
        float *W, *gW, *mW, *vW, *b, *gb, *mb, *vb;
        const float *dZ;
        __nv_bfloat16 *Wb, *WbT;
        int rows, cols;                        // N x K of the weights
        int bias0, tile0;                      // first block of the layer's biases, of its weight tiles
    } layer[kMaxLayers];
    int L, batch, n_bias;
    float lr, c1, c2;
    int update;
    const double *loss;
    double *loss_out;                          // when set, receives the step's loss
};

// Adam on one parameter p with gradient g and moments m, v.
__device__ __forceinline__ void adam(float &p, float g, float &m, float &v, const StepEnd &s)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    m = b1 * m + (1.f - b1) * g;
    v = b2 * v + (1.f - b2) * g * g;
    p -= s.lr * (m / s.c1) / (sqrtf(v / s.c2) + eps);
}

__global__ void __launch_bounds__(256) k_step_end(const __grid_constant__ StepEnd s)
{
    __shared__ float rows[256][32];
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, blk = blockIdx.x;
    pdl_enter();
    if (blk == 0 && threadIdx.x == 0 && s.loss_out != nullptr) *s.loss_out = *s.loss;
    int l = 0;
    if (blk < s.n_bias) {
        while (l + 1 < s.L && blk >= s.layer[l + 1].bias0) ++l;
        const StepEnd::Layer &y = s.layer[l];
        const int c = (blk - y.bias0) * 32 + tx;
        float sum = 0.f;
        for (int r0 = 0; r0 < s.batch; r0 += 256) {
            float d[32];                               // all loads before the first store
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int r = r0 + 8 * j + ty;
                d[j] = r < s.batch && c < y.rows ? y.dZ[(int64_t)r * y.rows + c] : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 32; ++j) rows[8 * j + ty][tx] = d[j];
            __syncthreads();
            if (ty == 0) {                             // the loads ahead of the chain of sums
                const int m = min(256, s.batch - r0);
                int j = 0;
                for (; j + 32 <= m; j += 32) {
                    float v[32];
#pragma unroll
                    for (int q = 0; q < 32; ++q) v[q] = rows[j + q][tx];
#pragma unroll
                    for (int q = 0; q < 32; ++q) sum += v[q];
                }
                for (; j < m; ++j) sum += rows[j][tx];
            }
            __syncthreads();
        }
        if (ty == 0 && c < y.rows) {
            y.gb[c] = sum;
            if (s.update) adam(y.b[c], sum, y.mb[c], y.vb[c], s);
        }
        return;
    }
    while (l + 1 < s.L && blk >= s.layer[l + 1].tile0) ++l;
    const StepEnd::Layer &y = s.layer[l];
    const int t = blk - y.tile0, tc = (y.cols + 31) / 32;
    const int r0 = t / tc * 32, c0 = t % tc * 32;
    // a thread's four elements are loaded before any is stored (their latencies overlap)
    float p[4], g[4], m[4], v[4];
    const int c1 = c0 + tx;
    auto live = [&](int j) { return r0 + ty + 8 * j < y.rows && c1 < y.cols; };
    auto at = [&](int j) { return (int64_t)(r0 + ty + 8 * j) * y.cols + c1; };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!live(j)) continue;
        p[j] = y.W[at(j)];
        g[j] = y.gW[at(j)];
        m[j] = y.mW[at(j)];
        v[j] = y.vW[at(j)];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!live(j)) continue;
        adam(p[j], g[j], m[j], v[j], s);
        y.W[at(j)] = p[j];
        y.mW[at(j)] = m[j];
        y.vW[at(j)] = v[j];
        y.Wb[at(j)] = __float2bfloat16_rn(p[j]);
        tile[ty + 8 * j][tx] = p[j];
    }
    __syncthreads();
    for (int j = ty; j < 32; j += 8) {
        const int c = c0 + j, r = r0 + tx;
        if (r < y.rows && c < y.cols) y.WbT[(int64_t)c * y.rows + r] = __float2bfloat16_rn(tile[tx][j]);
    }
}

int blocks_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 4096); }

}  // namespace

// Values of the pinned buffer of a network (with the status word after them).
constexpr size_t kHostRows = 4096;

struct mpm_mlp {
    int L = 0, max_batch = 0;
    std::vector<int> w;                           // widths, L + 1
    float lo = 0.f, hi = 1.f;
    int hidden_act = MPM_ACT_GELU, out_act = MPM_OUT_SIGMOID;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    std::vector<float *> W, b, gW, gb, mW, vW, mb, vb;     // fp32
    std::vector<__nv_bfloat16 *> Wb, WbT;                   // bf16 weight copies
    std::vector<__nv_bfloat16 *> X, XT;                     // layer inputs (bf16) and transposes, l = 0..L-1
    std::vector<float *> Z, dZ;                             // pre-activations and their gradients (fp32)
    std::vector<__nv_bfloat16 *> dZb, dZbT;
    float *Y = nullptr, *T = nullptr, *X0f = nullptr;
    double *loss = nullptr;
    int32_t *status = nullptr;                    // after Y's last row
    float *host = nullptr;                        // pinned, kHostRows values: small results on their way to the caller
    int64_t step = 0;
    std::string err;
};

namespace {

template <class T> int malloc_n(mpm_mlp *m, T **p, size_t count)
{
    if (cudaMalloc((void **)p, sizeof(T) * (count ? count : 1)) != cudaSuccess) {
        cudaGetLastError();
        m->err = "cudaMalloc failed";
        return MPM_ENOMEM;
    }
    return MPM_OK;
}

void refresh_bf16(mpm_mlp *m, int l)
{
    const int64_t n = (int64_t)m->w[l + 1] * m->w[l];
    k_f32_to_bf16<<<blocks_for(n), 256, 0, m->stream>>>(m->W[l], m->Wb[l], n);
    dim3 tb(32, 8), tg((m->w[l] + 31) / 32, (m->w[l + 1] + 31) / 32);
    k_transpose_bf16<<<tg, tb, 0, m->stream>>>(m->Wb[l], m->WbT[l], m->w[l + 1], m->w[l]);
}

// With train, the hidden layers' activations are also stored transposed (the weight
// gradients contract over the batch).
int forward(mpm_mlp *m, int B, bool train)
{
    for (int l = 0; l < m->L; ++l) {
        const int K = m->w[l], N = m->w[l + 1];
        // z = x W^T + b with the activation fused into the GEMM epilogue
        UmmaEpi epi;
        epi.bias = m->b[l];
        if (l + 1 < m->L) {
            epi.mode = m->hidden_act == MPM_ACT_RELU ? kEpiBiasRelu : kEpiBiasGelu;
            epi.xnext = m->X[l + 1];
            if (train) epi.xnextT = m->XT[l + 1];
        } else {
            epi.mode = m->out_act == MPM_OUT_LINEAR ? kEpiBiasLinear : kEpiBiasSigmoid;
            epi.y = m->Y;
            epi.lo = m->lo;
            epi.hi = m->hi;
        }
        cudaError_t e = umma_gemm_tma(B, N, K, m->X[l], K, m->Wb[l], K, m->Z[l], N, epi, m->status, m->stream);
        if (e != cudaSuccess) {
            m->err = std::string("gemm launch: ") + cudaGetErrorString(e);
            return MPM_ECUDA;
        }
    }
    return MPM_OK;
}

int check(mpm_mlp *m)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        m->err = cudaGetErrorString(e);
        return MPM_ECUDA;
    }
    return MPM_OK;
}

int status_code(mpm_mlp *m, int32_t st)
{
    if (st & kStatusTimeout) {
        m->err = "a bounded tensor-core wait ran out";
        return MPM_ETIMEOUT;
    }
    return MPM_OK;
}

int sync_status(mpm_mlp *m)
{
    int32_t st = 0;
    cudaError_t e = cudaMemcpyAsync(&st, m->status, sizeof st, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) {
        m->err = cudaGetErrorString(e);
        return MPM_ECUDA;
    }
    return status_code(m, st);
}

// Whether kernels may use a caller's device pointer in place: aligned, and memory that this
// device knows (its own, managed or pinned).  Any other pointer is left to a copy, which
// answers for it with an error where a kernel would fault.
bool in_place(const void *p, size_t align)
{
    if (reinterpret_cast<uintptr_t>(p) % align != 0) return false;
    cudaPointerAttributes a{};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type != cudaMemoryTypeUnregistered && (a.type != cudaMemoryTypeDevice || a.device == dev);
}

// Copies rows of floats at src to dev (a device buffer).
const float *copied(mpm_mlp *m, const float *src, float *dev, int64_t n, bool device)
{
    const cudaError_t e = cudaMemcpyAsync(dev, src, sizeof(float) * n,
                                          device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) return dev;
    cudaGetLastError();                           // reported by this call, not by the next one
    m->err = cudaGetErrorString(e);
    return nullptr;
}

// Network inputs at src on the device: src itself, or its copy in dev (host rows, and
// device rows that kernels cannot read in place).
const float *on_device(mpm_mlp *m, const float *src, float *dev, int64_t n, bool device)
{
    if (device && (reinterpret_cast<uintptr_t>(src) & 3) == 0) return src;
    return copied(m, src, dev, n, device);
}

// Back-propagation from the output layer's pre-activation gradient (dZ[L - 1] with its
// bf16 forms) and, with update, one Adam step; loss_out: device copy of the loss.
// Per layer one launch (two where a product fills the chip by itself) computes dW = dZ^T X
// and, for l > 0, dA = dZ W, whose epilogue forms the layer below's dZ; then one launch
// ends the step.
int backward_update(mpm_mlp *m, int B, double lr, int update, double *loss_out)
{
    const int L = m->L;
    for (int l = L - 1; l >= 0; --l) {
        const int K = m->w[l], N = m->w[l + 1];
        UmmaGemm g[2];
        g[0] = UmmaGemm{N, K, B, m->dZbT[l], B, m->XT[l], B, m->gW[l], K, UmmaEpi{}};
        if (l > 0) {
            UmmaEpi epi;
            epi.mode = m->hidden_act == MPM_ACT_RELU ? kEpiReluBack : kEpiGeluBack;
            epi.zprev = m->Z[l - 1];
            epi.xnext = m->dZb[l - 1];
            epi.xnextT = m->dZbT[l - 1];
            g[1] = UmmaGemm{B, K, N, m->dZb[l], N, m->WbT[l], N, m->dZ[l - 1], K, epi};
        }
        if (umma_gemms(g, l > 0 ? 2 : 1, m->status, m->stream) != cudaSuccess) return MPM_ECUDA;
    }
    if (update) m->step++;
    StepEnd s{};
    s.L = L;
    s.batch = B;
    s.lr = (float)lr;
    s.c1 = 1.f - powf(0.9f, (float)m->step);
    s.c2 = 1.f - powf(0.999f, (float)m->step);
    s.update = update != 0;
    s.loss = m->loss;
    s.loss_out = loss_out;
    int blocks = 0;
    for (int l = 0; l < L; ++l) {
        s.layer[l] = StepEnd::Layer{m->W[l], m->gW[l], m->mW[l], m->vW[l], m->b[l], m->gb[l], m->mb[l], m->vb[l],
                                    m->dZ[l], m->Wb[l], m->WbT[l], m->w[l + 1], m->w[l], blocks, 0};
        blocks += (m->w[l + 1] + 31) / 32;
    }
    s.n_bias = blocks;
    for (int l = 0; l < L && update; ++l) {
        s.layer[l].tile0 = blocks;
        blocks += ((m->w[l + 1] + 31) / 32) * ((m->w[l] + 31) / 32);
    }
    launch_after(k_step_end, blocks, 256, 0, m->stream, s);
    return MPM_OK;
}

// Queue the forward pass and the back-propagation of batch rows x (no
// synchronisation): of the mean squared error to the targets (with_loss), or of a
// given dL/dy (src).
int train_queue(mpm_mlp *m, int B, const float *x, const float *src, double lr, int update, bool device, bool with_loss,
                double *loss_out)
{
    const int L = m->L, nin = m->w[0], nout = m->w[L];
    const float *xd = on_device(m, x, m->X0f, (int64_t)B * nin, device);
    const float *sd = device && in_place(src, sizeof(float)) ? src : copied(m, src, m->T, (int64_t)B * nout, device);
    if (!xd || !sd) return MPM_ECUDA;
    launch_after(k_prepare_input, dim3((nin + 31) / 32, (B + 31) / 32), 256, 0, m->stream, xd, m->X[0], m->XT[0], B, nin,
                 m->loss);
    int rc = forward(m, B, true);
    if (rc != MPM_OK) return rc;
    launch_after(k_output_grad, dim3((nout + 31) / 32, (B + 31) / 32), 256, 0, m->stream, m->Y, sd, m->Z[L - 1],
                 m->dZ[L - 1], m->dZb[L - 1], m->dZbT[L - 1], B, nout, m->lo, m->hi, m->out_act == MPM_OUT_LINEAR,
                 with_loss ? m->loss : nullptr);
    rc = backward_update(m, B, lr, update, loss_out);
    return rc != MPM_OK ? rc : check(m);
}

}  // namespace

extern "C" {

int mpm_gemm_bf16(int M, int N, int K, const void *A, int lda, const void *B, int ldb, float *C, int ldc,
                  int32_t *status_dev, void *cuda_stream)
{
    if (M <= 0 || N <= 0 || K <= 0 || !A || !B || !C || lda < K || ldb < K || ldc < N || (lda % 8) || (ldb % 8) ||
        !status_dev)
        return MPM_EINVAL;
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) return MPM_EINVAL;
    cudaError_t e = umma_gemm_tma(M, N, K, (const __nv_bfloat16 *)A, lda, (const __nv_bfloat16 *)B, ldb, C, ldc, UmmaEpi{},
                              status_dev, (cudaStream_t)cuda_stream);
    return e == cudaSuccess ? MPM_OK : MPM_ECUDA;
}

int mpm_mlp_create(int n_layers, const int *widths, int max_batch, double out_lo, double out_hi, void *cuda_stream,
                   mpm_mlp **out)
{
    if (n_layers < 1 || n_layers > 8 || !widths || max_batch < 1 || max_batch > 65536 || !out || !(out_hi > out_lo))
        return MPM_EINVAL;
    for (int l = 0; l <= n_layers; ++l)
        if (widths[l] < 1 || widths[l] > 8192 || widths[l] % 8) return MPM_EINVAL;
    mpm_mlp *m = new mpm_mlp();
    m->L = n_layers;
    m->max_batch = (max_batch + 7) / 8 * 8;
    m->w.assign(widths, widths + n_layers + 1);
    m->lo = (float)out_lo;
    m->hi = (float)out_hi;
    if (cuda_stream) {
        m->stream = (cudaStream_t)cuda_stream;
    } else {
        if (cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete m;
            return MPM_ECUDA;
        }
        m->own_stream = true;
    }
    const int L = n_layers, B = m->max_batch;
    int rc = MPM_OK;
    auto resize = [&](auto &v) { v.assign(L, nullptr); };
    resize(m->W); resize(m->b); resize(m->gW); resize(m->gb); resize(m->mW); resize(m->vW); resize(m->mb);
    resize(m->vb); resize(m->Wb); resize(m->WbT); resize(m->X); resize(m->XT); resize(m->Z); resize(m->dZ);
    resize(m->dZb); resize(m->dZbT);
    for (int l = 0; l < L && rc == MPM_OK; ++l) {
        const size_t nw = (size_t)widths[l + 1] * widths[l], nb = widths[l + 1];
        rc = malloc_n(m, &m->W[l], nw);
        if (rc == MPM_OK) rc = malloc_n(m, &m->b[l], nb);
        if (rc == MPM_OK) rc = malloc_n(m, &m->gW[l], nw);
        if (rc == MPM_OK) rc = malloc_n(m, &m->gb[l], nb);
        if (rc == MPM_OK) rc = malloc_n(m, &m->mW[l], nw);
        if (rc == MPM_OK) rc = malloc_n(m, &m->vW[l], nw);
        if (rc == MPM_OK) rc = malloc_n(m, &m->mb[l], nb);
        if (rc == MPM_OK) rc = malloc_n(m, &m->vb[l], nb);
        if (rc == MPM_OK) rc = malloc_n(m, &m->Wb[l], nw);
        if (rc == MPM_OK) rc = malloc_n(m, &m->WbT[l], nw);
        if (rc == MPM_OK) rc = malloc_n(m, &m->X[l], (size_t)B * widths[l]);
        if (rc == MPM_OK) rc = malloc_n(m, &m->XT[l], (size_t)B * widths[l]);
        if (rc == MPM_OK) rc = malloc_n(m, &m->Z[l], (size_t)B * widths[l + 1]);
        if (rc == MPM_OK) rc = malloc_n(m, &m->dZ[l], (size_t)B * widths[l + 1]);
        if (rc == MPM_OK) rc = malloc_n(m, &m->dZb[l], (size_t)B * widths[l + 1]);
        if (rc == MPM_OK) rc = malloc_n(m, &m->dZbT[l], (size_t)B * widths[l + 1]);
    }
    if (rc == MPM_OK) rc = malloc_n(m, &m->Y, (size_t)B * widths[L] + 1);   // the status word after the outputs
    if (rc == MPM_OK && cudaMallocHost((void **)&m->host, kHostRows * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        m->err = "cudaMallocHost failed";
        rc = MPM_ENOMEM;
    }
    if (rc == MPM_OK) rc = malloc_n(m, &m->T, (size_t)B * widths[L]);
    if (rc == MPM_OK) rc = malloc_n(m, &m->X0f, (size_t)B * widths[0]);
    if (rc == MPM_OK) rc = malloc_n(m, &m->loss, 1);
    if (rc == MPM_OK) m->status = reinterpret_cast<int32_t *>(m->Y + (size_t)B * widths[L]);
    if (rc == MPM_OK && cudaMemsetAsync(m->status, 0, sizeof(int32_t), m->stream) != cudaSuccess) rc = MPM_ECUDA;
    if (rc != MPM_OK) {
        mpm_mlp_destroy(m);
        return rc;
    }
    *out = m;
    return MPM_OK;
}

void mpm_mlp_destroy(mpm_mlp *m)
{
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    for (auto *vec : {&m->W, &m->b, &m->gW, &m->gb, &m->mW, &m->vW, &m->mb, &m->vb, &m->Z, &m->dZ})
        for (float *p : *vec)
            if (p) cudaFree(p);
    for (auto *vec : {&m->Wb, &m->WbT, &m->X, &m->XT, &m->dZb, &m->dZbT})
        for (__nv_bfloat16 *p : *vec)
            if (p) cudaFree(p);
    for (void *p : {(void *)m->Y, (void *)m->T, (void *)m->X0f, (void *)m->loss})
        if (p) cudaFree(p);
    if (m->host) cudaFreeHost(m->host);
    if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

int64_t mpm_mlp_num_params(const mpm_mlp *m)
{
    if (!m) return MPM_EINVAL;
    int64_t n = 0;
    for (int l = 0; l < m->L; ++l) n += (int64_t)m->w[l + 1] * m->w[l] + m->w[l + 1];
    return n;
}

int mpm_mlp_set_params(mpm_mlp *m, const float *params)
{
    if (!m || !params) return MPM_EINVAL;
    const float *p = params;
    for (int l = 0; l < m->L; ++l) {
        const size_t nw = (size_t)m->w[l + 1] * m->w[l], nb = m->w[l + 1];
        if (cudaMemcpyAsync(m->W[l], p, sizeof(float) * nw, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
            cudaMemcpyAsync(m->b[l], p + nw, sizeof(float) * nb, cudaMemcpyHostToDevice, m->stream) != cudaSuccess)
            return MPM_ECUDA;
        cudaMemsetAsync(m->mW[l], 0, sizeof(float) * nw, m->stream);
        cudaMemsetAsync(m->vW[l], 0, sizeof(float) * nw, m->stream);
        cudaMemsetAsync(m->mb[l], 0, sizeof(float) * nb, m->stream);
        cudaMemsetAsync(m->vb[l], 0, sizeof(float) * nb, m->stream);
        refresh_bf16(m, l);
        p += nw + nb;
    }
    m->step = 0;
    int rc = check(m);
    return rc != MPM_OK ? rc : sync_status(m);
}

int mpm_mlp_get_params(mpm_mlp *m, float *params, int which)
{
    if (!m || !params || which < 0 || which > 1) return MPM_EINVAL;
    float *p = params;
    for (int l = 0; l < m->L; ++l) {
        const size_t nw = (size_t)m->w[l + 1] * m->w[l], nb = m->w[l + 1];
        const float *sw = which == 0 ? m->W[l] : m->gW[l];
        const float *sb = which == 0 ? m->b[l] : m->gb[l];
        if (cudaMemcpyAsync(p, sw, sizeof(float) * nw, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
            cudaMemcpyAsync(p + nw, sb, sizeof(float) * nb, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
            return MPM_ECUDA;
        p += nw + nb;
    }
    return sync_status(m);
}

int mpm_mlp_infer(mpm_mlp *m, int batch, const float *x, float *y, int device_ptrs)
{
    if (!m || !x || !y || batch < 1 || batch > m->max_batch) return MPM_EINVAL;
    const int64_t nx = (int64_t)batch * m->w[0];
    const float *xd = on_device(m, x, m->X0f, nx, device_ptrs != 0);
    if (!xd) return MPM_ECUDA;
    launch_after(k_f32_to_bf16, blocks_for(nx), 256, 0, m->stream, xd, m->X[0], nx);
    int rc = forward(m, batch, false);
    if (rc == MPM_OK) rc = check(m);
    if (rc != MPM_OK) return rc;
    const size_t n = (size_t)batch * m->w[m->L];
    // A network of small capacity, to the host: all its rows and the status word after them
    // come back in one copy through pinned memory (two pageable copies, each waited for by the
    // driver: one row through 640-256-256-32 built for 8 rows 59 us, 49 so).
    const size_t all = (size_t)m->max_batch * m->w[m->L] + 1;
    if (!device_ptrs && all <= kHostRows) {
        cudaError_t e = cudaMemcpyAsync(m->host, m->Y, sizeof(float) * all, cudaMemcpyDeviceToHost, m->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
        if (e != cudaSuccess) {
            m->err = cudaGetErrorString(e);
            return MPM_ECUDA;
        }
        int32_t st;
        std::memcpy(&st, m->host + all - 1, sizeof st);
        std::memcpy(y, m->host, sizeof(float) * n);
        return status_code(m, st);
    }
    if (cudaMemcpyAsync(y, m->Y, sizeof(float) * n, device_ptrs ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                        m->stream) != cudaSuccess)
        return MPM_ECUDA;
    return sync_status(m);
}

int mpm_mlp_train_step(mpm_mlp *m, int batch, const float *x, const float *target, double lr, int update,
                       double *loss_out, int device_ptrs)
{
    if (!m || !x || !target || batch < 8 || batch > m->max_batch || (batch % 8) || !(lr >= 0)) return MPM_EINVAL;
    int rc = train_queue(m, batch, x, target, lr, update, device_ptrs != 0, true, nullptr);
    if (rc != MPM_OK) return rc;
    if (loss_out &&
        cudaMemcpyAsync(loss_out, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
        return MPM_ECUDA;
    return sync_status(m);
}

int mpm_mlp_train_step_async(mpm_mlp *m, int batch, const float *x_dev, const float *target_dev, double lr,
                             double *loss_dev)
{
    if (!m || !x_dev || !target_dev || batch < 8 || batch > m->max_batch || (batch % 8) || !(lr >= 0))
        return MPM_EINVAL;
    const bool direct = loss_dev == nullptr || in_place(loss_dev, sizeof(double));   // a store of the last kernel
    int rc = train_queue(m, batch, x_dev, target_dev, lr, 1, true, true, direct ? loss_dev : nullptr);
    if (rc != MPM_OK) return rc;
    if (!direct &&
        cudaMemcpyAsync(loss_dev, m->loss, sizeof(double), cudaMemcpyDeviceToDevice, m->stream) != cudaSuccess)
        return MPM_ECUDA;
    return MPM_OK;
}

int mpm_mlp_backward(mpm_mlp *m, int batch, const float *x, const float *dy, double lr, int update, int device_ptrs)
{
    if (!m || !x || !dy || batch < 8 || batch > m->max_batch || (batch % 8) || !(lr >= 0)) return MPM_EINVAL;
    int rc = train_queue(m, batch, x, dy, lr, update, device_ptrs != 0, false, nullptr);
    return rc != MPM_OK ? rc : sync_status(m);
}

int mpm_mlp_set_activations(mpm_mlp *m, int hidden, int output)
{
    if (!m || (hidden != MPM_ACT_GELU && hidden != MPM_ACT_RELU) ||
        (output != MPM_OUT_SIGMOID && output != MPM_OUT_LINEAR))
        return MPM_EINVAL;
    m->hidden_act = hidden;
    m->out_act = output;
    return MPM_OK;
}

int mpm_mlp_last_error(const mpm_mlp *m, char *buf, int len)
{
    if (!m || !buf || len <= 0) return MPM_EINVAL;
    std::snprintf(buf, (size_t)len, "%s", m->err.c_str());
    return MPM_OK;
}

}  // extern "C"
