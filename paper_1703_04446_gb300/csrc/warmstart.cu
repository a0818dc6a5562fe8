// Learned warm start: a small convolutional encoder-decoder that maps an image
// pair (T, R) to a starting velocity for the Gauss-Newton solve (Eq. 11).  The
// paper has no such network; it is an addition whose predictions the solver
// still checks and corrects.
//
// Network for m x m images, c base channels (B images per call):
//   e0 = relu(conv3(x, 2 -> c))                       m
//   e1 = relu(conv3(e0, c -> 2c, stride 2))           m/2
//   e2 = relu(conv3(e1, 2c -> 4c, stride 2))          m/4
//   e3 = relu(conv3(e2, 4c -> 8c, stride 2))          m/8
//   d2 = relu(conv3(up2(e3), 8c -> 4c)) + e2          m/4
//   d1 = relu(conv3(up2(d2), 4c -> 2c)) + e1          m/2
//   v  = scale * conv3(d1, 2c -> 2)                   m/2
// conv3: 3 x 3, zero padding 1; up2: nearest-neighbour doubling, folded into
// the convolution's input indexing.  Weights are used as bfloat16 (rounded from
// FP32 master weights after every Adam step); activations, gradients and
// accumulation are FP32.  Loss 1/2 mean((v - target)^2) / scale^2.
//
// The convolutions, their data gradients and their weight gradients run as
// implicit GEMMs on the tensor cores (conv_umma.cuh), each reading the bf16
// planes that the kernel before it wrote.  The first layer (two input channels,
// 18 products a value) has kernels of its own here: its forward pass on the tensor
// cores, its weight gradient in FP32; the ReLU masks, the loss and Adam are
// elementwise kernels.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "conv_umma.cuh"
#include "lgnk_internal.h"

namespace {

constexpr int kT = 256;
constexpr int kMaxSlices = 64;   // K slices of the weight-gradient GEMM (partials summed in order)

struct Layer {
    int ci, co, stride, up;   // input channels, output channels, stride, input upsampled
    int hin, hout;            // input and output side lengths (square)
    size_t woff, boff;        // offsets of W and b in the parameter vector
    // bf16 weight matrices of the tensor-core GEMMs, zero padded, K ordered
    // as the operand planes are (channel fastest):
    // forward wf[co][tap * cpi + ci] (cpi = ci rounded up to 16; rows to a
    // multiple of bnf, rows of ldf), data gradient
    // wd[ci][(tap * R + up position) * cpo + co] (cpo = co rounded up to 16, R = 4 when up)
    int cpi, cpo, bnf, ldf, rowsf, bnd, ldd, rowsd;
    __nv_bfloat16 *wf, *wd;
};

// The launch of one GEMM of a layer at one batch size: everything but the
// tensors of the call.  Kept per layer and kind for the last batch size.
struct Plan {
    int batch = 0;
    umma::ConvGemm g;
    CUtensorMap a, b;
    int grid = 0;
    size_t smem = 0;
};

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Launch as a programmatic dependent of the kernel before it on the stream
// (umma::dependency_wait): a pass is 13 to 60 kernels of a few microseconds, and
// each one's start-up overlaps the end of the one before.
template <class... KArgs, class... Args>
cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

struct Layers {
    Layer l[7];
};

// The GEMMs' weight matrices from the FP32 master weights (bf16, nearest), layer
// 1 + blockIdx.y (left as they are when a wait ran out, as the master weights are).
__global__ void pack_wmats_kernel(const float* p, const Layers all, const int* err) {
    umma::dependency_trigger();
    umma::dependency_wait();
    if (umma::ld(err) != 0) return;
    const Layer L = all.l[1 + blockIdx.y];
    const size_t nf = (size_t)L.rowsf * L.ldf, nd = (size_t)L.rowsd * L.ldd;
    const int R = L.up ? 4 : 1;
    const float* W = p + L.woff;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nf + nd; i += (size_t)gridDim.x * blockDim.x) {
        float v = 0.0f;
        if (i < nf) {
            const int n = (int)(i / L.ldf), k = (int)(i % L.ldf);
            const int t = k / L.cpi, c = k - t * L.cpi;
            if (n < L.co && t < 9 && c < L.ci) v = umma::ld(W + ((size_t)n * L.ci + c) * 9 + t);
            L.wf[i] = __float2bfloat16_rn(v);
        } else {
            const size_t j = i - nf;
            const int n = (int)(j / L.ldd), k = (int)(j % L.ldd);
            const int pos = k / L.cpo, cc = k - pos * L.cpo, t = pos / R;
            if (n < L.ci && t < 9 && cc < L.co) v = umma::ld(W + ((size_t)cc * L.ci + n) * 9 + t);
            L.wd[j] = __float2bfloat16_rn(v);
        }
    }
}

// The end of a layer's weight and bias gradients, partials summed in increasing
// order: dW[co][ci][tap] = sum_s part[s][co][tap cp + ci], and behind it
// db[co] = sum_s bpart[s][co].
__global__ void sum_slices_kernel(const float* part, const float* bpart, float* dW, int co,
                                  int ci, int cp, int slices, int bslices) {
    const int nw = co * ci * 9, rows = 9 * cp;
    umma::dependency_trigger();
    umma::dependency_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw + co; i += gridDim.x * blockDim.x) {
        float s = 0.0f;
        if (i < nw) {
            const int n = i / (ci * 9), r = i - n * ci * 9, c = r / 9, t = r - c * 9;
            const float* p = part + (size_t)n * rows + t * cp + c;
#pragma unroll 8
            for (int k = 0; k < slices; ++k) s += umma::ld(p + (size_t)k * co * rows);
        } else {
#pragma unroll 8
            for (int k = 0; k < bslices; ++k) s += umma::ld(bpart + (size_t)k * co + i - nw);
        }
        dW[i] = s;
    }
}

// The output gradient of a layer, dz = g (m > 0) (m: the ReLU's output, as FP32
// mr or as planes mp of cp channels; none: dz = g), as planes and as partial
// bias gradients bpart[s][co] (the sums over the pixels of block column s).
// One pass over g instead of a masking pass, a splitting pass and a bias pass
// (0.11 + 0.19 + 0.20 ms of a 128^2 batch-32 training step).  A thread handles 8
// channels of one pixel at a time; a warp covers 4 (2) neighbouring channel
// groups of 8 (16) pixels, so that reads (channel rows) and writes (pixels)
// both touch whole sectors.
constexpr int kBiasSlices = 152;     // at most: about one block a SM; also sizes the partials
__global__ void __launch_bounds__(kT) mask_split_kernel(const float* g, const float* mr,
                                                        const __nv_bfloat16* mp, __nv_bfloat16* planes,
                                                        float* bpart, int C, int cp, int P, int B, int gs) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pw = 32 / gs;      // pixels per warp
    const int c0 = (blockIdx.y * gs + lane / pw) * 8;
    const size_t n = (size_t)P * B, pe = n * cp;
    umma::dependency_trigger();
    umma::dependency_wait();
    float sum[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j] = 0.0f;
    const size_t step = (size_t)gridDim.x * (kT / 32) * pw;
    for (size_t pix = ((size_t)blockIdx.x * (kT / 32) + warp) * pw + lane % pw; pix < n; pix += step) {
        const size_t b = pix / P, o = pix - b * P, e = pix * cp + c0;
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = c0 + j < C ? umma::ld(g + (b * C + c0 + j) * P + o) : 0.0f;
        if (mr != nullptr) {
            float r[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) r[j] = c0 + j < C ? umma::ld(mr + (b * C + c0 + j) * P + o) : 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (!(r[j] > 0.0f)) v[j] = 0.0f;
        } else if (mp != nullptr) {
            __align__(16) __nv_bfloat16 m[8];
            *reinterpret_cast<uint4*>(m) = umma::ld(reinterpret_cast<const uint4*>(mp + e));
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (!(__bfloat162float(m[j]) > 0.0f)) v[j] = 0.0f;
        }
        umma::store_planes8(planes, pe, e, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) sum[j] += v[j];
    }
    __shared__ float red[kT / 32][4][8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        for (int w = pw / 2; w > 0; w >>= 1) sum[j] += __shfl_down_sync(0xffffffffu, sum[j], w, pw);
    if (lane % pw == 0) {
#pragma unroll
        for (int j = 0; j < 8; ++j) red[warp][lane / pw][j] = sum[j];
    }
    __syncthreads();
    if ((int)threadIdx.x < gs * 8) {
        const int gi = threadIdx.x / 8, j = threadIdx.x % 8, c = (blockIdx.y * gs + gi) * 8 + j;
        float s = 0.0f;
        for (int w = 0; w < kT / 32; ++w) s += red[w][gi][j];
        if (c < C) bpart[(size_t)blockIdx.x * C + c] = s;
    }
}

// The first layer, e0 = relu(conv(x = [T, R]) + b), written as the next layer's
// planes: M = 128 pixels, N = bn = C rounded up to 16, K = 9 taps x 8 channels (two
// used) rounded up to 80.  A thread makes one row of A: it reads the 18 inputs of
// its pixel and writes their planes to shared memory as 16-byte core-matrix rows
// (no TMA form fits: through tensor maps the rows are 32 bytes of mostly padding,
// 0.19 ms at batch 32, 128^2, against 0.10 ms for a generic gather); three CTAs of
// 128 threads per SM overlap the gather, the 15 MMAs and the stores, and the
// 6 bytes a value that it writes bound it.  K is summed as two taps per MMA step
// with the plane products innermost; the rounding of e0 decides its ReLU, and
// with it whole gradient entries.
constexpr int kFirstK = 10;       // 16-byte groups of K
__global__ void __launch_bounds__(128) conv_first_kernel(const float* T, const float* R,
                                                         const float* W, const float* bias,
                                                         __nv_bfloat16* planes, int C, int bn, int cp, int m, int B,
                                                         int tiles, int ncols, int* err, int* herr) {
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_base;
    __shared__ int dead;
    uint8_t* sb = sm + 3 * kFirstK * 2048;      // B: [k group][row] x 16 bytes; A: [plane][k group][row] x 16 bytes
    float* bs = reinterpret_cast<float*>(sb + kFirstK * bn * 16);
    const int tid = threadIdx.x, warp = tid >> 5;
    if (warp == 0) {
        asm volatile(
            "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(umma::smem_u32(&tmem_base)),
            "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        dead = 0;
        umma::mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    __syncthreads();
    umma::dependency_trigger();           // the CTA has its tensor memory (see dependency_trigger)
    umma::dependency_wait();
    for (int i = tid; i < kFirstK * bn; i += 128) {
        const int tap = i / bn, n = i - tap * bn;
        __align__(16) __nv_bfloat16 w[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
            w[c] = __float2bfloat16_rn(c < 2 && tap < 9 && n < C ? umma::ld(W + ((size_t)n * 2 + c) * 9 + tap) : 0.0f);
        *reinterpret_cast<uint4*>(sb + (size_t)i * 16) = *reinterpret_cast<const uint4*>(w);
    }
    for (int i = tid; i < bn; i += 128) bs[i] = i < C ? umma::ld(bias + i) : 0.0f;
#pragma unroll
    for (int p = 0; p < 3; ++p)
        *reinterpret_cast<uint4*>(sm + ((p * kFirstK + 9) * 128 + tid) * 16) = make_uint4(0, 0, 0, 0);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base, a0 = umma::smem_u32(sm), b0 = umma::smem_u32(sb);
    const uint32_t idesc = umma::instr_desc(umma::BM, bn, false);
    const size_t P = (size_t)m * m, n = P * B;
    bool ok = true;
    uint32_t phase = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, phase ^= 1u) {
        const size_t i = (size_t)tile * umma::BM + tid;
        const bool valid = i < n;
        const size_t b = i / P;
        const int o = (int)(i - b * P), y = o / m, x = o - y * m;
        float in[18];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int yy = y + t / 3 - 1, xx = x + t % 3 - 1;
            const bool in_img = valid && yy >= 0 && yy < m && xx >= 0 && xx < m;
            const size_t e = in_img ? b * P + (size_t)(yy * m + xx) : 0;
            in[2 * t] = in_img ? umma::ld(T + e) : 0.0f;
            in[2 * t + 1] = in_img ? umma::ld(R + e) : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            __nv_bfloat16 h[2], q[2], l[2];
            umma::split3(in[2 * t], h[0], q[0], l[0]);
            umma::split3(in[2 * t + 1], h[1], q[1], l[1]);
            uint4* dst = reinterpret_cast<uint4*>(sm + (t * 128 + tid) * 16);      // planes kFirstK x 128 rows apart
            dst[0] = make_uint4(*reinterpret_cast<const uint32_t*>(h), 0, 0, 0);
            dst[kFirstK * 128] = make_uint4(*reinterpret_cast<const uint32_t*>(q), 0, 0, 0);
            dst[2 * kFirstK * 128] = make_uint4(*reinterpret_cast<const uint32_t*>(l), 0, 0, 0);
        }
        asm volatile("fence.proxy.async.shared::cta;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int kk = 0; kk < kFirstK / 2; ++kk) {
                const uint64_t bd = umma::smem_desc(b0 + kk * 2 * bn * 16, (uint32_t)bn * 16, 128, 0);
#pragma unroll
                for (int p = 0; p < 3; ++p)
                    umma::mma_bf16(tmem, umma::smem_desc(a0 + (p * kFirstK + kk * 2) * 2048, 2048, 128, 0), bd, idesc,
                                   kk + p > 0 ? 1u : 0u);
            }
            umma::mma_commit(&bar);
        }
        ok = umma::mbar_wait(&bar, phase, &dead);
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        for (int c0 = 0; c0 < bn; c0 += 16) {
            uint32_t v[16];
            umma::tmem_ld16(v, tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0);
            asm volatile("tcgen05.wait::ld.sync.aligned;");
            if (!valid) continue;
            float z[16];
#pragma unroll
            for (int j = 0; j < 16; ++j)
                z[j] = c0 + j < C ? fmaxf(__uint_as_float(v[j]) + bs[c0 + j], 0.0f) : 0.0f;
            umma::store_planes8(planes, n * cp, i * cp + c0, z);
            umma::store_planes8(planes, n * cp, i * cp + c0 + 8, z + 8);
        }
    }
    if (!ok) {            // once more, bounded, for the MMAs in flight
        if (tid == 0) {
            umma::give_up(err, herr);
            for (long k = 0; k < umma::kWaitLimit && !umma::mbar_try(&bar, phase); ++k) {
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// Partial weight and bias gradients of the first layer from the gradient g of
// e0 (masked here by e0 > 0, its planes): part[s][co][(tap, ci)] and bpart[s][co]
// over the pixels of block column s.  A thread accumulates 18 x kFirstW products
// over its pixels; a block sums them once.
constexpr int kFirstW = 4;
__global__ void __launch_bounds__(kT) conv_first_wgrad_kernel(const float* T, const float* R,
                                                              const float* g,
                                                              const __nv_bfloat16* e0, float* part,
                                                              float* bpart, int C, int cp, int m, int B) {
    const int c0 = blockIdx.y * kFirstW, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t P = (size_t)m * m, n = P * B;
    umma::dependency_trigger();
    umma::dependency_wait();
    float acc[kFirstW][19];
#pragma unroll
    for (int j = 0; j < kFirstW; ++j)
#pragma unroll
        for (int k = 0; k < 19; ++k) acc[j][k] = 0.0f;
    for (size_t i = blockIdx.x * (size_t)kT + threadIdx.x; i < n; i += (size_t)gridDim.x * kT) {
        const size_t b = i / P;
        const int o = (int)(i - b * P), y = o / m, x = o - y * m;
        __align__(8) __nv_bfloat16 h[kFirstW];
        *reinterpret_cast<uint2*>(h) = umma::ld(reinterpret_cast<const uint2*>(e0 + i * cp + c0));
        float z[kFirstW];
#pragma unroll
        for (int j = 0; j < kFirstW; ++j) {
            z[j] = c0 + j < C ? umma::ld(g + (b * C + c0 + j) * P + o) : 0.0f;
            if (!(__bfloat162float(h[j]) > 0.0f)) z[j] = 0.0f;
            acc[j][18] += z[j];
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int yy = y + t / 3 - 1, xx = x + t % 3 - 1;
            const bool ok = yy >= 0 && yy < m && xx >= 0 && xx < m;
            const size_t e = b * P + (size_t)(ok ? yy * m + xx : 0);
            const float a = ok ? umma::ld(T + e) : 0.0f, r = ok ? umma::ld(R + e) : 0.0f;
#pragma unroll
            for (int j = 0; j < kFirstW; ++j) {
                acc[j][2 * t] = fmaf(a, z[j], acc[j][2 * t]);
                acc[j][2 * t + 1] = fmaf(r, z[j], acc[j][2 * t + 1]);
            }
        }
    }
    __shared__ float red[kT / 32][kFirstW * 19];
#pragma unroll
    for (int j = 0; j < kFirstW; ++j)
#pragma unroll
        for (int k = 0; k < 19; ++k) {
            float s = acc[j][k];
#pragma unroll
            for (int w = 16; w > 0; w >>= 1) s += __shfl_down_sync(0xffffffffu, s, w);
            if (lane == 0) red[warp][j * 19 + k] = s;
        }
    __syncthreads();
    for (int q = threadIdx.x; q < kFirstW * 19; q += kT) {
        const int j = q / 19, k = q % 19;
        float s = 0.0f;
        for (int w = 0; w < kT / 32; ++w) s += red[w][q];
        if (c0 + j >= C) continue;
        if (k < 18) part[((size_t)blockIdx.x * C + c0 + j) * 18 + k] = s;
        else bpart[(size_t)blockIdx.x * C + c0 + j] = s;
    }
}

// loss partials (FP64) and the gradient of the loss with respect to the
// unscaled output z (v = scale z): dz = (v - t) / (scale N).
__global__ void mse_kernel(const float* v, const float* t, float* dz, size_t n, float scale,
                           double* partial) {
    umma::dependency_trigger();
    umma::dependency_wait();
    double s = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float e = umma::ld(v + i) - umma::ld(t + i);
        s += (double)e * (double)e;
        dz[i] = e / (scale * (float)n);
    }
    __shared__ double red[kT];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = kT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

// No update from a step in which a wait ran out.
__global__ void adam_kernel(float* p, const float* g, float* m, float* s, size_t n, float lr, float c1, float c2,
                            const int* err) {
    umma::dependency_trigger();
    umma::dependency_wait();
    if (umma::ld(err) != 0) return;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = umma::ld(g + i);
        const float mi = 0.9f * umma::ld(m + i) + 0.1f * gi;
        const float si = 0.999f * umma::ld(s + i) + 0.001f * gi * gi;
        m[i] = mi;
        s[i] = si;
        p[i] = umma::ld(p + i) - lr * (mi / c1) / (sqrtf(si / c2) + 1e-8f);
    }
}

__global__ void give_up_kernel(int* err, int* herr) {
    umma::dependency_trigger();
    umma::dependency_wait();
    umma::give_up(err, herr);
}

inline int blocks_for(size_t n) {
    const size_t b = (n + kT - 1) / kT;
    return (int)(b < 4096 ? (b ? b : 1) : 4096);
}

}  // namespace

struct lgnk_ws {
    int m, c, max_batch;
    float scale;
    cudaStream_t stream;
    std::vector<Layer> L;
    size_t nparams;
    float *p, *g, *am, *as;     // master weights, gradients, Adam moments
    float *e1, *e2, *r4, *r5, *z6;   // activations that are read as FP32
    float *ga, *gb, *gc;        // gradients of e1 (and d1), e2 (and d2), and the others in turn
    float* wpart;               // per-slice weight-gradient partials
    float* bpart;               // per-slice bias-gradient partials
    __nv_bfloat16* planes[7];   // bf16 planes of the input of layer 1..6
    __nv_bfloat16* zplanes;     // of the output gradient at hand
    Plan plans[7][3];           // [layer][umma::Kind]
    int sms, smem_max;          // of the device: SMs, dynamic shared memory of the GEMM kernel
    float* gpart;               // split-K partial tiles of the FWD and BWD_DATA GEMMs
    size_t gpart_cap;           // floats it holds
    int *derr, *herr;           // set by a tensor-core kernel whose wait ran out (umma::give_up)
    double* partial;
    double* hres;
    long long steps;
    std::vector<void*> allocs;
    char err[256];
};

namespace {

lgnk_status ws_alloc(lgnk_ws* w, size_t bytes, void** out) {
    if (cudaMalloc(out, bytes ? bytes : 16) != cudaSuccess) {
        cudaGetLastError();
        snprintf(w->err, sizeof(w->err), "cudaMalloc(%zu) failed", bytes);
        return LGNK_ERR_OOM;
    }
    w->allocs.push_back(*out);
    return LGNK_OK;
}

template <typename T>
lgnk_status ws_alloc_n(lgnk_ws* w, size_t n, T** out) {
    void* p = nullptr;
    const lgnk_status s = ws_alloc(w, n * sizeof(T), &p);
    *out = static_cast<T*>(p);
    return s;
}

size_t act_size(const lgnk_ws* w, int layer_out_c, int side, int B) { return (size_t)B * layer_out_c * side * side; }

// K slices of a FWD / BWD_DATA GEMM with `tiles` output tiles and `chunks` K
// chunks: enough slices to give about two tiles to each of the device's SMs, each at
// least two chunks (1 when the tiles alone fill the GPU)
inline int split_slices(int tiles, int chunks, int sms) {
    if (tiles >= 2 * sms) return 1;
    const int s = std::min((2 * sms + tiles - 1) / tiles, std::max(1, chunks / 2));
    const int cps = (chunks + s - 1) / s;
    return (chunks + cps - 1) / cps;
}

// channels per row of an operand tile whose planes have cp channels
inline int row_channels(int cp) { return cp % 64 == 0 ? 64 : (cp % 32 == 0 ? 32 : 16); }

// The box of `total` positions (powers of two per axis) that covers a batch of
// side x side grids with the fewest boxes; among equals the widest, so that
// where the side divides, the boxes follow the pixels' linear order.
void choose_box(int side, int batch, int total, umma::ConvGemm* g) {
    long long best = -1;
    for (int bx = total; bx >= 1; bx /= 2)
        for (int by = total / bx; by >= 1; by /= 2) {
            const int bb = total / (bx * by);
            const long long n = (long long)((side + bx - 1) / bx) * ((side + by - 1) / by) * ((batch + bb - 1) / bb);
            if (best >= 0 && n >= best) continue;
            best = n;
            g->bx = bx;
            g->by = by;
            g->bb = bb;
        }
    g->tx = (side + g->bx - 1) / g->bx;
    g->ty = (side + g->by - 1) / g->by;
    g->tb = (batch + g->bb - 1) / g->bb;
}

// Everything of a layer's GEMM but its tensors, maps and stages.
umma::ConvGemm gemm_shape(const Layer& L, int kind, int B, int sms) {
    umma::ConvGemm g{};
    g.kind = kind;
    g.ci = L.ci;
    g.co = L.co;
    g.stride = L.stride;
    g.up = L.up;
    g.hin = L.hin;
    g.hout = L.hout;
    g.batch = B;
    g.cp = kind == umma::BWD_DATA ? L.cpo : L.cpi;
    g.kb = row_channels(g.cp);
    g.phases = (kind != umma::BWD_DATA && L.up) || (kind == umma::BWD_DATA && L.stride == 2) ? 4 : 1;
    if (kind == umma::BWD_WEIGHT) {
        g.N = L.co;
        g.kz = row_channels(L.cpo);
        g.bn = std::min(128, L.cpo);
        g.bn = round_up(g.bn, g.kz);
        g.ntn = (L.cpo + g.bn - 1) / g.bn;
        g.grid = L.up ? L.hin : L.hout;
        choose_box(g.grid, B, umma::BK, &g);
        g.mtiles = (9 * g.cp + umma::BM - 1) / umma::BM;
        g.chunks = g.phases * g.tx * g.ty * g.tb;
        const int tiles = g.mtiles * g.ntn;
        const int s = std::min(kMaxSlices, std::min(g.chunks, std::max(1, (2 * sms + tiles - 1) / tiles)));
        g.chunks_per_split = (g.chunks + s - 1) / s;
        g.splits = (g.chunks + g.chunks_per_split - 1) / g.chunks_per_split;
        g.items = tiles * g.splits;
        g.a_bytes = 3 * umma::BK * umma::BM * 2;
        g.stage_bytes = round_up(g.a_bytes + 3 * umma::BK * g.bn * 2, 1024);
    } else {
        const bool f = kind == umma::FWD;
        const int ho = f ? L.hout : L.hin;
        g.N = f ? L.co : L.ci;
        g.bn = f ? L.bnf : L.bnd;
        g.ntn = (f ? L.rowsf : L.rowsd) / g.bn;
        g.grid = g.phases == 4 ? ho / 2 : ho;
        choose_box(g.grid, B, umma::BM, &g);
        const int tiles = g.phases * g.tx * g.ty * g.tb * g.ntn;
        g.chunks = (9 * (!f && L.up ? 4 : 1) * g.cp + umma::BK - 1) / umma::BK;
        // the slices of K by the rows of D in tiles of 128, not by the boxes that cover them: they
        // set the rounding of the sums, and a ReLU's sign with it (a gradient's entries jump there)
        const int rows = (int)(((long long)B * ho * ho + umma::BM - 1) / umma::BM);
        const int s = split_slices(rows * g.ntn, g.chunks, sms);
        g.chunks_per_split = (g.chunks + s - 1) / s;
        g.splits = (g.chunks + g.chunks_per_split - 1) / g.chunks_per_split;
        g.items = tiles * g.splits;
        g.M = (long long)B * ho * ho;
        g.a_bytes = 3 * umma::BM * 2 * g.kb;
        g.stage_bytes = round_up(g.a_bytes + g.bn * 2 * g.kb, 1024);
    }
    g.ncols = g.bn <= 32 ? 32 : (g.bn <= 64 ? 64 : (g.bn <= 128 ? 128 : 256));
    return g;
}

typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_tiled() {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return reinterpret_cast<EncodeTiled>(fn);
}

inline CUtensorMapSwizzle swizzle_of(int kb) {
    return kb == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (kb == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

// Planes [3][B][h][h][cp] in boxes of 3 planes x (bb, by, bx) positions, `step`
// apart, x kb channels.
bool planes_map(EncodeTiled enc, CUtensorMap* m, __nv_bfloat16* p, int cp, int h, int B, int kb,
                const umma::ConvGemm& g, int step) {
    const cuuint64_t row = 2ull * cp, dims[5] = {(cuuint64_t)cp, (cuuint64_t)h, (cuuint64_t)h, (cuuint64_t)B, 3};
    const cuuint64_t strides[4] = {row, row * h, row * h * h, row * h * h * B};
    const cuuint32_t box[5] = {(cuuint32_t)kb, (cuuint32_t)(g.bx * step), (cuuint32_t)(g.by * step), (cuuint32_t)g.bb,
                               3};
    const cuuint32_t steps[5] = {1, (cuuint32_t)step, (cuuint32_t)step, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, p, dims, strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
               swizzle_of(kb), CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool weights_map(EncodeTiled enc, CUtensorMap* m, __nv_bfloat16* p, int ld, int rows, int kb, int bn) {
    const cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)rows}, strides[1] = {2ull * ld};
    const cuuint32_t box[2] = {(cuuint32_t)kb, (cuuint32_t)bn}, steps[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p, dims, strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
               swizzle_of(kb), CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The plan of layer l's GEMM at batch B, made on first use and when the batch
// size changes.
cudaError_t gemm_plan(lgnk_ws* w, int l, int kind, int B, Plan** out) {
    Plan& p = w->plans[l][kind];
    *out = &p;
    if (p.batch == B) return cudaSuccess;
    p.batch = 0;
    const Layer& L = w->L[l];
    p.g = gemm_shape(L, kind, B, w->sms);
    umma::ConvGemm& g = p.g;
    const EncodeTiled enc = encode_tiled();
    if (enc == nullptr) return cudaErrorNotSupported;
    bool ok;
    if (kind == umma::FWD) {
        ok = planes_map(enc, &p.a, w->planes[l], g.cp, L.hin, B, g.kb, g, L.stride) &&
             weights_map(enc, &p.b, L.wf, L.ldf, L.rowsf, g.kb, g.bn);
    } else if (kind == umma::BWD_DATA) {
        ok = planes_map(enc, &p.a, w->zplanes, g.cp, L.hout, B, g.kb, g, L.up ? 2 : 1) &&
             weights_map(enc, &p.b, L.wd, L.ldd, L.rowsd, g.kb, g.bn);
    } else {
        ok = planes_map(enc, &p.a, w->planes[l], g.cp, L.hin, B, g.kb, g, L.stride) &&
             planes_map(enc, &p.b, w->zplanes, L.cpo, L.hout, B, g.kz, g, L.up ? 2 : 1);
    }
    if (!ok) return cudaErrorInvalidValue;
    g.stages = std::min(umma::kMaxStages, (w->smem_max - 1024) / g.stage_bytes);
    if (g.stages < 1) return cudaErrorInvalidValue;
    p.smem = (size_t)g.stages * g.stage_bytes + 1024;
    p.grid = std::min(g.items, w->sms);
    g.err = w->derr;
    g.herr = w->herr;
    if (kind == umma::BWD_WEIGHT) g.part = w->wpart;
    else {
        g.part = w->gpart;
        if (g.splits > 1 && (size_t)g.splits * g.M * g.N > w->gpart_cap) return cudaErrorInvalidValue;
    }
    p.batch = B;
    return cudaSuccess;
}

cudaError_t launch_gemm(lgnk_ws* w, const Plan& p, const umma::ConvGemm& g) {
    cudaError_t e = launch(umma::conv_gemm_kernel, dim3(p.grid), umma::kThreads, p.smem, w->stream, p.a, p.b, g);
    if (e != cudaSuccess || g.kind == umma::BWD_WEIGHT || g.splits == 1) return e;
    return launch(umma::finish_split_kernel, dim3(blocks_for((size_t)g.M * ((g.N + 7) / 8))), kT, 0, w->stream, g,
                  g.splits);
}

// Layer l >= 1 from the planes of its input: out = scale (act(conv + b) + add)
// (FP32, may be NULL), r = act(conv + b) (may be NULL), and the next layer's
// planes if there is one.
cudaError_t conv_fwd(lgnk_ws* w, int l, float* out, float* r, const float* add, int relu, float scale, int B) {
    const Layer& L = w->L[l];
    Plan* p = nullptr;
    cudaError_t e = gemm_plan(w, l, umma::FWD, B, &p);
    if (e != cudaSuccess) return e;
    umma::ConvGemm g = p->g;
    g.out = out;
    g.r = r;
    g.add = add;
    g.bias = w->p + L.boff;
    g.relu = relu;
    g.scale = scale;
    g.nplanes = l < 6 ? w->planes[l + 1] : nullptr;
    g.ncp = l < 6 ? w->L[l + 1].cpi : 0;
    return launch_gemm(w, *p, g);
}

cudaError_t sum_slices(lgnk_ws* w, const Layer& L, int cp, int slices, int bslices) {
    const size_t n = (size_t)L.co * L.ci * 9 + L.co;
    return launch(sum_slices_kernel, dim3(blocks_for(n)), kT, 0, w->stream, w->wpart, w->bpart, w->g + L.woff, L.co,
                  L.ci, cp, slices, bslices);
}

// Backward of layer l >= 1 from the gradient gz of its ReLU's output (masked by
// that output, mr or mp; neither: gz is the gradient of the convolution): weight
// and bias gradients, and the input gradient into din (added when accumulate).
cudaError_t conv_bwd(lgnk_ws* w, int l, const float* gz, const float* mr, const __nv_bfloat16* mp, float* din,
                     int accumulate, int B) {
    const Layer& L = w->L[l];
    const int P = L.hout * L.hout, gs = L.cpo % 32 == 0 ? 4 : 2, per = kT / gs;     // pixels per block
    const int bs = (int)std::min<long long>(kBiasSlices, ((long long)P * B + per - 1) / per);
    cudaError_t e = launch(mask_split_kernel, dim3(bs, L.cpo / 8 / gs), kT, 0, w->stream, gz, mr, mp, w->zplanes,
                           w->bpart, L.co, L.cpo, P, B, gs);
    Plan* p = nullptr;
    if (e == cudaSuccess) e = gemm_plan(w, l, umma::BWD_WEIGHT, B, &p);
    if (e == cudaSuccess) e = launch_gemm(w, *p, p->g);
    if (e == cudaSuccess) e = sum_slices(w, L, L.cpi, p->g.splits, bs);
    if (e == cudaSuccess) e = gemm_plan(w, l, umma::BWD_DATA, B, &p);
    if (e != cudaSuccess) return e;
    umma::ConvGemm d = p->g;
    d.out = din;
    d.accumulate = accumulate;
    return launch_gemm(w, *p, d);
}

// refresh the GEMMs' bf16 weight matrices from the master weights
cudaError_t pack_weights(lgnk_ws* w) {
    Layers all;
    size_t n = 0;
    for (int l = 0; l < 7; ++l) {
        all.l[l] = w->L[l];
        if (l > 0) n = std::max(n, (size_t)w->L[l].rowsf * w->L[l].ldf + (size_t)w->L[l].rowsd * w->L[l].ldd);
    }
    return launch(pack_wmats_kernel, dim3(std::min(blocks_for(n), 608), 6), kT, 0, w->stream, w->p, all, w->derr);
}

// Shared memory of the first layer's kernel, and its CTAs per SM (bounded by
// that and by the 512 columns of tensor memory).
size_t first_smem(int bn) { return (size_t)3 * kFirstK * 2048 + (size_t)kFirstK * bn * 16 + (size_t)bn * 4; }
int first_ctas(int bn) { return bn <= 64 ? 3 : 2; }

// The network; with train, also what only the backward pass reads (r4, r5).
lgnk_status forward_pass(lgnk_ws* w, int B, const float* T, const float* R, float* v, bool train) {
    const Layer& L0 = w->L[0];
    const size_t n = (size_t)w->m * w->m * B;
    const int bn = w->L[1].cpi, tiles = (int)((n + umma::BM - 1) / umma::BM);
    const int ncols = bn <= 32 ? 32 : (bn <= 64 ? 64 : (bn <= 128 ? 128 : 256));
    const dim3 grid(std::min(tiles, first_ctas(bn) * w->sms));
    cudaError_t e = launch(conv_first_kernel, grid, 128, first_smem(bn), w->stream, T, R, w->p + L0.woff,
                           w->p + L0.boff, w->planes[1], L0.co, bn, bn, w->m, B, tiles, ncols, w->derr, w->herr);
    if (e == cudaSuccess) e = conv_fwd(w, 1, w->e1, nullptr, nullptr, 1, 1.0f, B);
    if (e == cudaSuccess) e = conv_fwd(w, 2, w->e2, nullptr, nullptr, 1, 1.0f, B);
    if (e == cudaSuccess) e = conv_fwd(w, 3, nullptr, nullptr, nullptr, 1, 1.0f, B);
    if (e == cudaSuccess) e = conv_fwd(w, 4, nullptr, train ? w->r4 : nullptr, w->e2, 1, 1.0f, B);
    if (e == cudaSuccess) e = conv_fwd(w, 5, nullptr, train ? w->r5 : nullptr, w->e1, 1, 1.0f, B);
    if (e == cudaSuccess) e = conv_fwd(w, 6, v, nullptr, nullptr, 0, w->scale, B);
    if (e != cudaSuccess) {
        snprintf(w->err, sizeof(w->err), "%s", cudaGetErrorString(e));
        return LGNK_ERR_CUDA;
    }
    return LGNK_OK;
}

// What a call on the network begins with (and a synchronising one ends with): an error if an
// earlier one's wait ran out, cleared as it is reported.
lgnk_status report_give_up(lgnk_ws* w) {
    if (*static_cast<volatile int*>(w->herr) == 0) return LGNK_OK;
    *static_cast<volatile int*>(w->herr) = 0;
    snprintf(w->err, sizeof(w->err), "a tensor-core convolution of an earlier call gave up waiting: its results are "
             "unfinished (the weights were not updated from them)");
    if (cudaMemsetAsync(w->derr, 0, sizeof(int), w->stream) != cudaSuccess) return LGNK_ERR_CUDA;
    return LGNK_ERR_INTERNAL;
}

}  // namespace

#define WS_CHECK(call)                                                              \
    do {                                                                            \
        cudaError_t e_ = (call);                                                    \
        if (e_ != cudaSuccess) {                                                    \
            snprintf(w->err, sizeof(w->err), "%s: %s", #call, cudaGetErrorString(e_)); \
            return LGNK_ERR_CUDA;                                                   \
        }                                                                           \
    } while (0)

extern "C" {

void lgnk_ws_destroy(lgnk_ws* w) {
    if (w == nullptr) return;
    for (void* p : w->allocs) cudaFree(p);
    if (w->hres) cudaFreeHost(w->hres);
    delete w;
}

lgnk_status lgnk_ws_create(int image_m, int base_channels, int max_batch, float output_scale, void* stream,
                           lgnk_ws** out) {
    if (out == nullptr) return LGNK_ERR_INVALID_ARG;
    *out = nullptr;
    if (image_m < 8 || image_m % 8 != 0 || image_m > 4096 || base_channels < 1 || base_channels > 256 ||
        max_batch < 1 || !(output_scale > 0.0f))
        return LGNK_ERR_INVALID_ARG;
    lgnk_ws* w = new (std::nothrow) lgnk_ws();
    if (w == nullptr) return LGNK_ERR_OOM;
    w->m = image_m;
    w->c = base_channels;
    w->max_batch = max_batch;
    w->scale = output_scale;
    w->stream = static_cast<cudaStream_t>(stream);
    const int c = base_channels, m = image_m;
    const int spec[7][5] = {{2, c, 1, 0, m},          {c, 2 * c, 2, 0, m},         {2 * c, 4 * c, 2, 0, m / 2},
                            {4 * c, 8 * c, 2, 0, m / 4}, {8 * c, 4 * c, 1, 1, m / 8}, {4 * c, 2 * c, 1, 1, m / 4},
                            {2 * c, 2, 1, 0, m / 2}};
    size_t off = 0;
    for (int l = 0; l < 7; ++l) {
        Layer L;
        L.ci = spec[l][0];
        L.co = spec[l][1];
        L.stride = spec[l][2];
        L.up = spec[l][3];
        L.hin = spec[l][4];
        L.hout = L.up ? 2 * L.hin : L.hin / L.stride;
        L.woff = off;
        off += (size_t)L.co * L.ci * 9;
        L.boff = off;
        off += L.co;
        w->L.push_back(L);
    }
    w->nparams = off;
    const int B = max_batch;
    lgnk_status s = LGNK_OK;
    auto fail = [&](lgnk_status st) {
        lgnk_ws_destroy(w);
        return st;
    };
    if ((s = ws_alloc_n(w, off, &w->p)) || (s = ws_alloc_n(w, off, &w->g)) || (s = ws_alloc_n(w, off, &w->am)) ||
        (s = ws_alloc_n(w, off, &w->as)) || (s = ws_alloc_n(w, 1, &w->derr)))
        return fail(s);
    {
        int dev = 0, optin = 0;
        cudaFuncAttributes fa{};
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&w->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, umma::conv_gemm_kernel) != cudaSuccess) {
            cudaGetLastError();
            return fail(LGNK_ERR_CUDA);
        }
        w->smem_max = optin - (int)fa.sharedSizeBytes;
        if (cudaFuncSetAttribute(conv_first_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)first_smem(256)) != cudaSuccess) {
            cudaGetLastError();
            return fail(LGNK_ERR_CUDA);
        }
        if (cudaFuncSetAttribute(umma::conv_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, w->smem_max) !=
            cudaSuccess) {
            cudaGetLastError();
            return fail(LGNK_ERR_CUDA);
        }
    }
    // the GEMMs' bf16 weight matrices (N per CTA up to 256, rows and K padded)
    size_t zmax = 0;
    for (int l = 0; l < 7; ++l) {
        Layer& L = w->L[l];
        const int R = L.up ? 4 : 1;
        L.cpi = round_up(L.ci, 16);
        L.cpo = round_up(L.co, 16);
        if (l == 0) continue;             // the first layer has kernels of its own
        L.bnf = std::min(256, L.cpo);
        L.rowsf = round_up(L.co, L.bnf);
        L.ldf = round_up(9 * L.cpi, umma::BK);
        L.bnd = std::min(256, L.cpi);
        L.rowsd = round_up(L.ci, L.bnd);
        L.ldd = round_up(9 * R * L.cpo, umma::BK);
        zmax = std::max(zmax, (size_t)B * L.hout * L.hout * L.cpo);
        if ((s = ws_alloc_n(w, (size_t)L.rowsf * L.ldf, &L.wf)) ||
            (s = ws_alloc_n(w, (size_t)L.rowsd * L.ldd, &L.wd)) ||
            (s = ws_alloc_n(w, (size_t)3 * B * L.hin * L.hin * L.cpi, &w->planes[l])))
            return fail(s);
    }
    if ((s = ws_alloc_n(w, 3 * zmax, &w->zplanes))) return fail(s);
    // split-K partials: the largest splits x M x N any batch size up to max_batch needs
    size_t gmax = 1;
    for (int b = 1; b <= B; ++b) {
        for (int l = 1; l < 7; ++l) {
            const Layer& L = w->L[l];
            for (int kind : {umma::FWD, umma::BWD_DATA}) {
                const umma::ConvGemm g = gemm_shape(L, kind, b, w->sms);
                if (g.splits > 1) gmax = std::max(gmax, (size_t)g.splits * (size_t)g.M * g.N);
            }
        }
    }
    w->gpart_cap = gmax;
    if ((s = ws_alloc_n(w, gmax, &w->gpart))) return fail(s);
    // gradients: ga of e1 and d1, gb of e2 and d2, gc the output's, e3's and e0's in turn
    if ((s = ws_alloc_n(w, act_size(w, 2 * c, m / 2, B), &w->e1)) ||
        (s = ws_alloc_n(w, act_size(w, 4 * c, m / 4, B), &w->e2)) ||
        (s = ws_alloc_n(w, act_size(w, 4 * c, m / 4, B), &w->r4)) ||
        (s = ws_alloc_n(w, act_size(w, 2 * c, m / 2, B), &w->r5)) ||
        (s = ws_alloc_n(w, act_size(w, 2, m / 2, B), &w->z6)) ||
        (s = ws_alloc_n(w, act_size(w, 2 * c, m / 2, B), &w->ga)) ||
        (s = ws_alloc_n(w, act_size(w, 4 * c, m / 4, B), &w->gb)) ||
        (s = ws_alloc_n(w, act_size(w, c, m, B), &w->gc)) || (s = ws_alloc_n(w, (size_t)4096, &w->partial)))
        return fail(s);
    size_t wmax = 0, bmax = 0;
    for (const Layer& L : w->L) {
        wmax = std::max(wmax, (size_t)L.co * L.cpi * 9);
        bmax = std::max(bmax, (size_t)L.co);
    }
    if ((s = ws_alloc_n(w, wmax * kMaxSlices, &w->wpart)) || (s = ws_alloc_n(w, bmax * kBiasSlices, &w->bpart)))
        return fail(s);
    if (cudaMallocHost((void**)&w->hres, 8 * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        w->hres = nullptr;
        return fail(LGNK_ERR_OOM);
    }
    w->herr = reinterpret_cast<int*>(w->hres + 7);
    *w->herr = 0;
    if (cudaMemsetAsync(w->p, 0, off * sizeof(float), w->stream) != cudaSuccess ||
        cudaMemsetAsync(w->am, 0, off * sizeof(float), w->stream) != cudaSuccess ||
        cudaMemsetAsync(w->as, 0, off * sizeof(float), w->stream) != cudaSuccess ||
        cudaMemsetAsync(w->derr, 0, sizeof(int), w->stream) != cudaSuccess || pack_weights(w) != cudaSuccess)
        return fail(LGNK_ERR_CUDA);
    *out = w;
    return LGNK_OK;
}

size_t lgnk_ws_num_params(const lgnk_ws* w) { return w ? w->nparams : 0; }

const char* lgnk_ws_last_error(const lgnk_ws* w) { return w ? w->err : "null network"; }

lgnk_status lgnk_ws_set_params(lgnk_ws* w, const float* params) {
    if (w == nullptr || params == nullptr) return LGNK_ERR_INVALID_ARG;
    WS_CHECK(cudaMemsetAsync(w->derr, 0, sizeof(int), w->stream));      // new weights, new start
    WS_CHECK(cudaMemcpyAsync(w->p, params, w->nparams * sizeof(float), cudaMemcpyDeviceToDevice, w->stream));
    WS_CHECK(pack_weights(w));
    WS_CHECK(cudaMemsetAsync(w->am, 0, w->nparams * sizeof(float), w->stream));
    WS_CHECK(cudaMemsetAsync(w->as, 0, w->nparams * sizeof(float), w->stream));
    w->steps = 0;
    return LGNK_OK;
}

lgnk_status lgnk_ws_get_params(lgnk_ws* w, float* params) {
    if (w == nullptr || params == nullptr) return LGNK_ERR_INVALID_ARG;
    if (const lgnk_status st = report_give_up(w)) return st;
    WS_CHECK(cudaMemcpyAsync(params, w->p, w->nparams * sizeof(float), cudaMemcpyDeviceToDevice, w->stream));
    return LGNK_OK;
}

lgnk_status lgnk_ws_get_grads(lgnk_ws* w, float* grads) {
    if (w == nullptr || grads == nullptr) return LGNK_ERR_INVALID_ARG;
    if (const lgnk_status st = report_give_up(w)) return st;
    WS_CHECK(cudaMemcpyAsync(grads, w->g, w->nparams * sizeof(float), cudaMemcpyDeviceToDevice, w->stream));
    return LGNK_OK;
}

lgnk_status lgnk_ws_predict(lgnk_ws* w, int batch, const float* T, const float* R, float* v) {
    if (w == nullptr || T == nullptr || R == nullptr || v == nullptr || batch < 1 || batch > w->max_batch)
        return LGNK_ERR_INVALID_ARG;
    if (const lgnk_status st = report_give_up(w)) return st;
    return forward_pass(w, batch, T, R, v, false);
}

lgnk_status lgnk_ws_train_step(lgnk_ws* w, int batch, const float* T, const float* R, const float* target, float lr,
                               double* loss) {
    if (w == nullptr || T == nullptr || R == nullptr || target == nullptr || batch < 1 || batch > w->max_batch)
        return LGNK_ERR_INVALID_ARG;
    const int B = batch;
    lgnk_status st = report_give_up(w);
    if (st == LGNK_OK) st = forward_pass(w, B, T, R, w->z6, true);
    if (st != LGNK_OK) return st;
    const int m = w->m;
    // loss and dz6 (gradient w.r.t. the unscaled output)
    const size_t nv = act_size(w, 2, m / 2, B);
    const int nb = blocks_for(nv) < 1024 ? blocks_for(nv) : 1024;
    float* dz6 = w->gc;
    WS_CHECK(launch(mse_kernel, dim3(nb), kT, 0, w->stream, w->z6, target, dz6, nv, w->scale, w->partial));
    // layer 6: d(d1) -> ga; d1 = r5 + e1, so ga is also the start of d(e1)
    WS_CHECK(conv_bwd(w, 6, dz6, nullptr, nullptr, w->ga, 0, B));
    // layer 5 (input up2(d2)): d(d2) -> gb, also the start of d(e2) (d2 = r4 + e2)
    WS_CHECK(conv_bwd(w, 5, w->ga, w->r5, nullptr, w->gb, 0, B));
    // layer 4 (input up2(e3)): d(e3) -> gc
    WS_CHECK(conv_bwd(w, 4, w->gb, w->r4, nullptr, w->gc, 0, B));
    // layer 3: d(e2) += ...; the masks of e3, e2, e1 are read from the planes
    WS_CHECK(conv_bwd(w, 3, w->gc, nullptr, w->planes[4], w->gb, 1, B));
    // layer 2: d(e1) += ...
    WS_CHECK(conv_bwd(w, 2, w->gb, nullptr, w->planes[3], w->ga, 1, B));
    // layer 1: d(e0) -> gc
    WS_CHECK(conv_bwd(w, 1, w->ga, nullptr, w->planes[2], w->gc, 0, B));
    // layer 0: weights only
    {
        const Layer& L = w->L[0];
        const size_t n = (size_t)m * m * B;
        // one wave of two blocks per SM
        const int groups = (L.co + kFirstW - 1) / kFirstW, wave = std::max(1, 2 * w->sms / groups);
        const int bs = (int)std::min<size_t>(std::min(kMaxSlices, wave), (n + kT - 1) / kT);
        WS_CHECK(launch(conv_first_wgrad_kernel, dim3(bs, groups), kT, 0, w->stream, T, R, w->gc, w->planes[1],
                        w->wpart, w->bpart, L.co, w->L[1].cpi, m, B));
        WS_CHECK(sum_slices(w, L, 2, bs, bs));
    }
    // Adam
    w->steps++;
    const float c1 = 1.0f - powf(0.9f, (float)w->steps), c2 = 1.0f - powf(0.999f, (float)w->steps);
    WS_CHECK(launch(adam_kernel, dim3(blocks_for(w->nparams)), kT, 0, w->stream, w->p, w->g, w->am, w->as, w->nparams,
                    lr, c1, c2, w->derr));
    WS_CHECK(pack_weights(w));
    if (loss != nullptr) {
        launch_reduce(w->partial, nb, w->partial + 2048, w->stream);
        WS_CHECK(cudaGetLastError());
        WS_CHECK(cudaMemcpyAsync(w->hres, w->partial + 2048, sizeof(double), cudaMemcpyDeviceToHost, w->stream));
        WS_CHECK(cudaStreamSynchronize(w->stream));
        if ((st = report_give_up(w)) != LGNK_OK) return st;
        *loss = 0.5 * w->hres[0] / (double)nv / ((double)w->scale * w->scale);
    }
    return LGNK_OK;
}

// For the tests: enqueues what a kernel whose wait ran out does.
void lgnk_internal_ws_give_up(lgnk_ws* w) { give_up_kernel<<<1, 1, 0, w->stream>>>(w->derr, w->herr); }

}  // extern "C"
