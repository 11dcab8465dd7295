// The learned CDF model: an FP32 MLP 8 -> 32 -> 32 -> 1 with ReLU, its
// forward pass, MSE loss gradient, Adam step, trainer and the compilation of
// the trained CDF into a sorted table of 4095 bucket splitters.
//
// Input x = the 8 prefix bytes of a rotation / 255; target t = the
// rotation's sorted rank / n, so the network approximates the CDF of 8-byte
// prefixes. Parameter layout (1,377 floats, row-major):
//   W1[32][8] | b1[32] | W2[32][32] | b2[32] | W3[32] | b3
// The loss over a batch is mean((y - t)^2); gradients are reduced in a fixed
// order (per-CTA partial sums, then CTA partials in index order), so runs are
// bit-reproducible. The MLP is FFMA work on CUDA cores: it is off the timed
// sort path (the sort only searches the compiled splitter table).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "bwt.h"
#include "plan_internal.h"

namespace bwt {

namespace {

constexpr int NP = BWT_MLP_NPARAMS;
constexpr int IN = 8, H = 32;
constexpr int OFF_W1 = 0, OFF_B1 = 256, OFF_W2 = 288, OFF_B2 = 1312, OFF_W3 = 1344, OFF_B3 = 1376;
constexpr int GS = 64;  // samples per CTA in the gradient kernel

__device__ __forceinline__ float mlp_eval(const float* __restrict__ P, const float* x, float* h1, float* h2) {
#pragma unroll
    for (int j = 0; j < H; ++j) {
        float a = P[OFF_B1 + j];
#pragma unroll
        for (int i = 0; i < IN; ++i) a = fmaf(P[OFF_W1 + j * IN + i], x[i], a);
        h1[j] = a > 0.f ? a : 0.f;
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
        float a = P[OFF_B2 + j];
#pragma unroll
        for (int i = 0; i < H; ++i) a = fmaf(P[OFF_W2 + j * H + i], h1[i], a);
        h2[j] = a > 0.f ? a : 0.f;
    }
    float y = P[OFF_B3];
#pragma unroll
    for (int i = 0; i < H; ++i) y = fmaf(P[OFF_W3 + i], h2[i], y);
    return y;
}

__global__ void __launch_bounds__(128) k_mlp_forward(const float* __restrict__ params, const float* __restrict__ x,
                                                     uint32_t count, float* __restrict__ y) {
    __shared__ float P[NP];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) P[i] = params[i];
    __syncthreads();
    const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= count) return;
    float xs[IN], h1[H], h2[H];
#pragma unroll
    for (int i = 0; i < IN; ++i) xs[i] = x[(size_t)s * IN + i];
    y[s] = mlp_eval(P, xs, h1, h2);
}

// Forward + backward of GS samples per CTA; writes the CTA's gradient sum
// (already divided by the batch size B) and its summed squared error.
// Samples are x[idx[first + s]] (or x[first + s] without idx).
//
// Four threads a sample: a warp computes one quarter of the units (8) for 32
// samples, so weights are read as broadcasts and every unit's sum is one
// thread's chain in the order of mlp_eval -- the same bits as one thread a
// sample. The gradient's 1,377 sums over the samples then spread over all 256
// threads. A step is latency (64 CTAs for a batch of 4,096): 98 steps of 4,096
// samples and the compilation took 5.75 ms with 64 threads a CTA and one thread
// a sample, 2.13 ms with four (13 us a gradient, 7 us a reduction, 0.15 ms the
// compilation), 1.54 ms as dependent launches (step_wait), 1.27-1.32 ms with the
// values of a unit in a row (four samples' values a 16-byte read) and
// four sums of W2 a thread sharing its reads: 8 shared-memory wavefronts for 16
// products instead of 32.
constexpr int TPS = 4;         // threads a sample
constexpr int GT = TPS * GS;   // threads
constexpr int UQ = H / TPS;    // units a thread
constexpr int GP = GS + 4;     // row length: 16-byte reads of eight lanes' rows fall in different banks
constexpr int GR = H / (GT / 32);  // rows of W2 a warp sums
static_assert(GT >= IN * H && IN % TPS == 0 && GR >= 1 && GT >= 128, "the sums' split over the threads");

// The launches of a training step follow each other as dependent launches: a
// kernel starts while the one before it ends, reads what no kernel of the
// training writes (samples, targets, order), and waits for its end and its
// results here. (Without the attribute at the launch both are empty.) What the
// kernels before it write is read after the wait and through plain pointers:
// const and __restrict__ together say that a value stands for the whole kernel,
// and the loads might then be moved ahead of the wait.
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void step_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__global__ void __launch_bounds__(GT) k_mlp_grad(const float* params, const float* __restrict__ x,
                                                 const float* __restrict__ t, const uint32_t* __restrict__ idx,
                                                 uint32_t first, uint32_t B, float* partial, float* loss_partial) {
    __shared__ __align__(16) float P[NP];
    // a row a unit (or input), a column a sample
    __shared__ __align__(16) float sx[IN][GP], sh1[H][GP], sh2[H][GP], sd1[H][GP], sd2[H][GP];
    __shared__ float sdy[GS], serr[GS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = (warp & 1) * 32 + lane, u0 = (warp >> 1) * UQ;  // the thread's sample and first unit
    const uint32_t b = blockIdx.x * GS + s;
    const bool valid = b < B;
    const uint32_t src = valid ? (idx ? idx[first + b] : first + b) : 0u;
    for (int i = u0 / UQ * (IN / TPS), n = 0; n < IN / TPS; ++i, ++n) sx[i][s] = valid ? x[(size_t)src * IN + i] : 0.f;
    const float want = valid && u0 == 0 ? t[src] : 0.f;
    step_wait();
    step_next();
    for (int i = threadIdx.x; i < NP; i += GT) P[i] = params[i];
    __syncthreads();
    if (valid) {
#pragma unroll
        for (int k = 0; k < UQ; ++k) {
            const int j = u0 + k;
            float a = P[OFF_B1 + j];
#pragma unroll
            for (int i = 0; i < IN; ++i) a = fmaf(P[OFF_W1 + j * IN + i], sx[i][s], a);
            sh1[j][s] = a > 0.f ? a : 0.f;
        }
    }
    __syncthreads();
    float h2[UQ];
    if (valid) {
        float h1[H];
#pragma unroll
        for (int i = 0; i < H; ++i) h1[i] = sh1[i][s];
#pragma unroll
        for (int k = 0; k < UQ; ++k) {
            const int j = u0 + k;
            float a = P[OFF_B2 + j];
#pragma unroll
            for (int i = 0; i < H; ++i) a = fmaf(P[OFF_W2 + j * H + i], h1[i], a);
            h2[k] = a > 0.f ? a : 0.f;
            sh2[j][s] = h2[k];
        }
    }
    __syncthreads();
    if (u0 == 0) {
        if (valid) {
            float y = P[OFF_B3];
#pragma unroll
            for (int i = 0; i < H; ++i) y = fmaf(P[OFF_W3 + i], sh2[i][s], y);
            const float e = y - want;
            serr[s] = e * e;
            sdy[s] = 2.f * e / (float)B;
        } else {
            serr[s] = 0.f;
            sdy[s] = 0.f;
        }
    }
    __syncthreads();
    if (valid) {
        const float dy = sdy[s];
#pragma unroll
        for (int k = 0; k < UQ; ++k) sd2[u0 + k][s] = h2[k] > 0.f ? dy * P[OFF_W3 + u0 + k] : 0.f;
    }
    __syncthreads();
    if (valid) {
        float d2[H];
#pragma unroll
        for (int j = 0; j < H; ++j) d2[j] = sd2[j][s];
#pragma unroll
        for (int k = 0; k < UQ; ++k) {
            const int i = u0 + k;
            float a = 0.f;
#pragma unroll
            for (int j = 0; j < H; ++j) a = fmaf(P[OFF_W2 + j * H + i], d2[j], a);
            sd1[i][s] = sh1[i][s] > 0.f ? a : 0.f;
        }
    } else {
        for (int k = 0; k < UQ; ++k) sd1[u0 + k][s] = sd2[u0 + k][s] = sh1[u0 + k][s] = sh2[u0 + k][s] = 0.f;
    }
    __syncthreads();
    float* out = partial + (size_t)blockIdx.x * NP;
    {  // W2: GR rows a warp, a column a lane
        float g[GR] = {};
#pragma unroll 4
        for (int q = 0; q < GS; q += 4) {
            const float4 h = *reinterpret_cast<const float4*>(&sh1[lane][q]);
#pragma unroll
            for (int k = 0; k < GR; ++k) {
                const float4 d = *reinterpret_cast<const float4*>(&sd2[warp * GR + k][q]);
                g[k] = fmaf(d.x, h.x, g[k]);
                g[k] = fmaf(d.y, h.y, g[k]);
                g[k] = fmaf(d.z, h.z, g[k]);
                g[k] = fmaf(d.w, h.w, g[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < GR; ++k) out[OFF_W2 + (warp * GR + k) * H + lane] = g[k];
    }
    if (threadIdx.x < IN * H) {  // W1: an entry a thread
        const int j = threadIdx.x / IN, i = threadIdx.x % IN;
        float g = 0.f;
#pragma unroll 4
        for (int q = 0; q < GS; q += 4) {
            const float4 d = *reinterpret_cast<const float4*>(&sd1[j][q]);
            const float4 v = *reinterpret_cast<const float4*>(&sx[i][q]);
            g = fmaf(d.x, v.x, g);
            g = fmaf(d.y, v.y, g);
            g = fmaf(d.z, v.z, g);
            g = fmaf(d.w, v.w, g);
        }
        out[OFF_W1 + threadIdx.x] = g;
    }
    // the biases, W3 and the loss: a warp each
    if (warp < 2) {
        const float* d = warp == 0 ? sd1[lane] : sd2[lane];
        float g = 0.f;
#pragma unroll 4
        for (int q = 0; q < GS; q += 4) {
            const float4 v = *reinterpret_cast<const float4*>(&d[q]);
            g += v.x;
            g += v.y;
            g += v.z;
            g += v.w;
        }
        out[(warp == 0 ? OFF_B1 : OFF_B2) + lane] = g;
    } else if (warp == 2) {
        float g = 0.f;
#pragma unroll 16
        for (int q = 0; q < GS; ++q) g = fmaf(sdy[q], sh2[lane][q], g);
        out[OFF_W3 + lane] = g;
    } else if (warp == 3 && lane < 2) {
        const float* d = lane == 0 ? sdy : serr;
        float g = 0.f;
#pragma unroll 16
        for (int q = 0; q < GS; ++q) g += d[q];
        if (lane == 0) out[OFF_B3] = g;
        else loss_partial[blockIdx.x] = g;
    }
}

// Sums the CTA partials in index order; optionally writes the gradient and
// the mean loss, and optionally applies one Adam step (Kingma and Ba 2015). A
// thread a parameter, 32 to a CTA so that the sums spread over the SMs, and 16
// partials loaded at a time: a sum is a chain of additions, not of loads.
__global__ void k_mlp_reduce(const float* partial, const float* loss_partial, int nblk, uint32_t B, float* grad_out,
                             float* loss_out, float* params, float* m, float* v, int step, float lr, float beta1,
                             float beta2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool adam = params && step > 0 && i < NP;
    float c1 = 1.f, c2 = 1.f, m0 = 0.f, v0 = 0.f, p0 = 0.f;
    if (adam) {
        c1 = 1.f - powf(beta1, (float)step);
        c2 = 1.f - powf(beta2, (float)step);
    }
    step_wait();
    step_next();
    if (adam) {
        m0 = m[i];
        v0 = v[i];
        p0 = params[i];
    }
    if (i == (int)(gridDim.x * blockDim.x) - 1 && loss_out) {  // past the parameters
        float l = 0.f;
#pragma unroll 16
        for (int b = 0; b < nblk; ++b) l += loss_partial[b];
        *loss_out = l / (float)B;
    }
    if (i >= NP) return;
    float g = 0.f;
#pragma unroll 16
    for (int b = 0; b < nblk; ++b) g += partial[(size_t)b * NP + i];
    if (grad_out) grad_out[i] = g;
    if (adam) {
        // the roundings spelled out: they do not hang on where the loads stand
        const float mi = fmaf(1.f - beta1, g, __fmul_rn(beta1, m0));
        const float vi = fmaf(__fmul_rn(1.f - beta2, g), g, __fmul_rn(beta2, v0));
        m[i] = mi;
        v[i] = vi;
        params[i] = p0 - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void k_adam(float* __restrict__ params, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int step, float lr, float beta1, float beta2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NP) return;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    const float mi = beta1 * m[i] + (1.f - beta1) * g[i];
    const float vi = beta2 * v[i] + (1.f - beta2) * g[i] * g[i];
    m[i] = mi;
    v[i] = vi;
    params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Bisection over the 64-bit key space, four neighbouring lanes per splitter:
// splitter j is the smallest key x (to 64-bit precision) with F(x) >= (j + 1) /
// 4096, where F = the MLP evaluated on x's 8 bytes mapped through norm. F need
// not be monotone; the table is sorted afterwards, and any sorted table gives
// exact results. A lane holds a quarter of the units (every unit's sum is one
// lane's chain in the order of mlp_eval, so F has the same bits) and the lanes
// exchange them by shuffles: the 64 evaluations of a splitter are one chain.
__global__ void __launch_bounds__(128) k_compile_splitters(const float* __restrict__ params,
                                                           const float* __restrict__ norm,
                                                           uint64_t* __restrict__ spl, uint32_t count) {
    __shared__ float P[NP];
    __shared__ float nrm[256];
    __shared__ __align__(16) float W1t[IN][H], W2t[H][H];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) P[i] = params[i];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) nrm[i] = norm[i];
    // W1 and W2 by input, so that a lane's eight units are two 16-byte loads
    // and the four lanes of a splitter use different banks
    for (int i = threadIdx.x; i < IN * H; i += blockDim.x) W1t[i % IN][i / IN] = params[OFF_W1 + i];
    for (int i = threadIdx.x; i < H * H; i += blockDim.x) W2t[i % H][i / H] = params[OFF_W2 + i];
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, quad = lane & ~3u;
    const uint32_t j = min((blockIdx.x * blockDim.x + threadIdx.x) >> 2, count - 1);
    const int u0 = (lane & 3) * UQ;  // this lane's first unit
    const float q = (float)(j + 1) / (float)(count + 1);
    uint64_t lo = 0, hi = ~0ull;  // invariant: F(hi) >= q is assumed at the top end
    for (int it = 0; it < 64; ++it) {  // lo == hi: an evaluation more changes nothing
        const uint64_t mid = lo + ((hi - lo) >> 1);
        float xs[IN], h1[UQ], h2[UQ];
#pragma unroll
        for (int b = 0; b < IN; ++b) xs[b] = nrm[(mid >> (56 - 8 * b)) & 0xff];
#pragma unroll
        for (int k = 0; k < UQ; ++k) {
            float a = P[OFF_B1 + u0 + k];
#pragma unroll
            for (int i = 0; i < IN; ++i) a = fmaf(W1t[i][u0 + k], xs[i], a);
            h1[k] = a > 0.f ? a : 0.f;
            h2[k] = P[OFF_B2 + u0 + k];
        }
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const float v = __shfl_sync(0xffffffffu, h1[i % UQ], quad + i / UQ);
#pragma unroll
            for (int k = 0; k < UQ; ++k) h2[k] = fmaf(W2t[i][u0 + k], v, h2[k]);
        }
        float y = P[OFF_B3];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const float a = h2[i % UQ];
            y = fmaf(P[OFF_W3 + i], __shfl_sync(0xffffffffu, a > 0.f ? a : 0.f, quad + i / UQ), y);
        }
        if (lo < hi) {
            if (y >= q) hi = mid; else lo = mid + 1;
        }
    }
    spl[j] = hi;
}

// Sorts the table in place (count <= 4096, one CTA, bitonic in shared memory),
// then spreads every run of equal splitters evenly over the key interval up
// to the next distinct splitter. Equal splitters come from a model that is
// flat across an interval and jumps at its end (the model reads the key as
// eight separate bytes, so it jumps at byte boundaries of the key): the run's
// share of the distribution lies in that interval, and even spacing there is
// the linear reading of the model's CDF across it. The table stays sorted.
__global__ void __launch_bounds__(1024) k_sort_splitters(uint64_t* __restrict__ spl, uint32_t count) {
    __shared__ uint64_t a[4096];
    for (uint32_t i = threadIdx.x; i < 4096; i += blockDim.x) a[i] = i < count ? spl[i] : ~0ull;
    __syncthreads();
    for (uint32_t k = 2; k <= 4096; k <<= 1)
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = threadIdx.x; i < 4096; i += blockDim.x) {
                const uint32_t ixj = i ^ j;
                if (ixj > i) {
                    const uint64_t x = a[i], y = a[ixj];
                    const bool up = (i & k) == 0;
                    if ((x > y) == up) {
                        a[i] = y;
                        a[ixj] = x;
                    }
                }
            }
            __syncthreads();
        }
    // every entry finds its run of equal splitters and its place in it
    for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) {
        const uint64_t base = a[i];
        uint32_t lo = 0, hi = i;  // first entry of the run
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (a[mid] < base) lo = mid + 1; else hi = mid;
        }
        const uint32_t first = lo;
        lo = i + 1;  // first entry after it
        hi = count;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (a[mid] <= base) lo = mid + 1; else hi = mid;
        }
        const uint64_t next = lo < count ? a[lo] : ~0ull;
        const uint32_t c = lo - first, r = i - first;
        spl[i] = r ? base + (uint64_t)((unsigned __int128)(next - base) * r / c) : base;
    }
}

struct MlpScratch {
    float* partial = nullptr;
    float* loss_partial = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    uint32_t cap_blocks = 0;
};

bwt_status ensure_scratch(MlpScratch& s, uint32_t nblk) {
    if (s.cap_blocks >= nblk) return BWT_OK;
    if (s.partial) cudaFree(s.partial);
    if (s.loss_partial) cudaFree(s.loss_partial);
    s.partial = nullptr;
    s.loss_partial = nullptr;
    if (cudaMalloc(&s.partial, sizeof(float) * NP * nblk) != cudaSuccess ||
        cudaMalloc(&s.loss_partial, sizeof(float) * nblk) != cudaSuccess) {
        cudaGetLastError();
        s.cap_blocks = 0;
        return BWT_ENOMEM;
    }
    s.cap_blocks = nblk;
    return BWT_OK;
}

void free_scratch(MlpScratch& s) {
    if (s.partial) cudaFree(s.partial);
    if (s.loss_partial) cudaFree(s.loss_partial);
    if (s.m) cudaFree(s.m);
    if (s.v) cudaFree(s.v);
    s = MlpScratch();
}

}  // namespace

}  // namespace bwt

using namespace bwt;

#define CKM(call)                                               \
    do {                                                        \
        cudaError_t _e = (call);                                \
        if (_e != cudaSuccess) return record_cuda(_e, #call);   \
    } while (0)

extern "C" bwt_status bwt_mlp_forward(const float* d_params, const float* d_x, uint32_t count, float* d_y,
                                      void* stream) {
    if (!d_params || (!d_x && count) || (!d_y && count)) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("mlp_forward");
    if (!count) return BWT_OK;
    k_mlp_forward<<<(count + 127) / 128, 128, 0, (cudaStream_t)stream>>>(d_params, d_x, count, d_y);
    CKM(cudaGetLastError());
    return BWT_OK;
}

extern "C" bwt_status bwt_mlp_loss_grad(const float* d_params, const float* d_x, const float* d_t, uint32_t count,
                                        float* d_grad, float* d_loss, void* stream) {
    if (!d_params || !d_x || !d_t || !d_grad || count == 0) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("mlp_loss_grad");
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t nblk = (count + GS - 1) / GS;
    MlpScratch s;
    bwt_status r = ensure_scratch(s, nblk);
    if (r != BWT_OK) return r;
    k_mlp_grad<<<nblk, GT, 0, st>>>(d_params, d_x, d_t, nullptr, 0, count, s.partial, s.loss_partial);
    k_mlp_reduce<<<NP / 32 + 1, 32, 0, st>>>(s.partial, s.loss_partial, (int)nblk, count, d_grad, d_loss,
                                                   nullptr, nullptr, nullptr, 0, 0.f, 0.f, 0.f, 0.f);
    cudaError_t e = cudaGetLastError();
    cudaStreamSynchronize(st);
    free_scratch(s);
    CKM(e);
    return BWT_OK;
}

extern "C" bwt_status bwt_mlp_adam_step(float* d_params, const float* d_grad, float* d_m, float* d_v, uint32_t step,
                                        float lr, void* stream) {
    if (!d_params || !d_grad || !d_m || !d_v || step == 0) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("mlp_adam");
    k_adam<<<(NP + 255) / 256, 256, 0, (cudaStream_t)stream>>>(d_params, d_grad, d_m, d_v, (int)step, lr, 0.9f,
                                                               0.999f, 1e-8f);
    CKM(cudaGetLastError());
    return BWT_OK;
}

namespace {

// dependent: the kernel before it in the stream is one of a training step (step_wait).
template <typename... P>
cudaError_t launch_step(void (*kernel)(P...), unsigned grid, unsigned threads, bool dependent, cudaStream_t st, P... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

extern "C" bwt_status bwt_model_train(float* d_params, const float* d_x, const float* d_t, uint32_t count,
                                      const uint32_t* d_order, uint32_t epochs, uint32_t batch, float lr,
                                      float* d_epoch_loss, void* stream) {
    if (!d_params || !d_x || !d_t || !d_order || count == 0 || batch == 0 || epochs == 0) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("mlp_train");
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t nblk = (batch + GS - 1) / GS;
    MlpScratch s;
    bwt_status r = ensure_scratch(s, nblk);
    if (r != BWT_OK) return r;
    float* batch_loss = nullptr;
    const uint32_t steps_per_epoch = (count + batch - 1) / batch;
    if (cudaMalloc(&s.m, sizeof(float) * NP) != cudaSuccess || cudaMalloc(&s.v, sizeof(float) * NP) != cudaSuccess ||
        cudaMalloc(&batch_loss, sizeof(float) * steps_per_epoch) != cudaSuccess) {
        cudaGetLastError();
        free_scratch(s);
        if (batch_loss) cudaFree(batch_loss);
        return BWT_ENOMEM;
    }
    cudaMemsetAsync(s.m, 0, sizeof(float) * NP, st);
    cudaMemsetAsync(s.v, 0, sizeof(float) * NP, st);
    int step = 0;
    std::vector<float> h_loss(steps_per_epoch);
    cudaError_t e = cudaSuccess;
    for (uint32_t ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        const uint32_t* order = d_order + (size_t)ep * count;
        for (uint32_t b0 = 0; b0 < count; b0 += batch) {
            const uint32_t B = std::min(batch, count - b0);
            const uint32_t nb = (B + GS - 1) / GS;
            ++step;
            // an epoch's first gradient follows work that is not a reduction: an ordinary launch
            e = launch_step(k_mlp_grad, nb, GT, b0 != 0, st, (const float*)d_params, d_x, d_t, order, b0, B, s.partial,
                            s.loss_partial);
            if (e != cudaSuccess) break;
            e = launch_step(k_mlp_reduce, NP / 32 + 1, 32, true, st, (const float*)s.partial, (const float*)s.loss_partial,
                            (int)nb, B, (float*)nullptr, batch_loss + b0 / batch, d_params, s.m, s.v, step, lr, 0.9f,
                            0.999f, 1e-8f);
            if (e != cudaSuccess) break;
        }
        if (d_epoch_loss && e == cudaSuccess) {
            // mean of the epoch's batch losses, computed on the host from a copy
            e = cudaMemcpyAsync(h_loss.data(), batch_loss, sizeof(float) * steps_per_epoch, cudaMemcpyDeviceToHost,
                                st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            double acc = 0;
            for (float v : h_loss) acc += v;
            const float mean = (float)(acc / steps_per_epoch);
            if (e == cudaSuccess) e = cudaMemcpyAsync(d_epoch_loss + ep, &mean, sizeof(float), cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        }
    }
    cudaStreamSynchronize(st);
    cudaFree(batch_loss);
    free_scratch(s);
    CKM(e);
    return BWT_OK;
}

extern "C" bwt_status bwt_model_compile(const float* d_params, const float* d_norm, uint64_t* d_splitters,
                                        void* stream) {
    if (!d_params || !d_norm || !d_splitters) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("mlp_compile");
    cudaStream_t st = (cudaStream_t)stream;
    k_compile_splitters<<<(4 * BWT_SPLITTERS + 127) / 128, 128, 0, st>>>(d_params, d_norm, d_splitters, BWT_SPLITTERS);
    k_sort_splitters<<<1, 1024, 0, st>>>(d_splitters, BWT_SPLITTERS);
    CKM(cudaGetLastError());
    return BWT_OK;
}
