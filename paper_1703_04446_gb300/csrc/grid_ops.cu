// Grid utilities of the lgnk library: layout conversion between the ABI layout
// and the padded packed layout of the tracing kernels, reductions (the
// accumulators of fsum.cuh per element, FP64 from the block partials on),
// regularizer stencils (Sec. 2.1, Sec. 3.2), the per-axis DCT of the spectral
// preconditioner (Sec. 3.2) and the vector updates of PCG.
#include <cmath>

#include <algorithm>

#include "fsum.cuh"
#include "lgnk_internal.h"

namespace {

constexpr int kBlock = LGNK_BLOCK;

inline int nblocks_for(size_t count) {
    return (int)((count + kBlock - 1) / kBlock);
}

__device__ __forceinline__ size_t padded_size(const DevGrid& g) {
    return (size_t)g.mp[0] * g.mp[1] * g.mp[2];
}

// ---------------------------------------------------------------- packing --

// Axis coordinates of element i of an nx x ny (x nz) block, in 32-bit
// arithmetic: every array the library accepts has fewer than 2^31 elements
// (checked when the context is created), and a 64-bit division costs many
// times a 32-bit one.
__device__ __forceinline__ void split_xyz(unsigned i, unsigned nx, unsigned ny, int& x, int& y, int& z) {
    const unsigned r = i / nx;
    x = (int)(i - r * nx);
    const unsigned q = r / ny;
    y = (int)(r - q * ny);
    z = (int)q;
}

// Pair-packed time slices: element (m, node) holds the velocity at stage time
// t_m (linear in time between the K nodes) at the padded node and at its +x
// neighbour, [v(node) | v(node + 1)], as 8 floats (3D: xyz + zero pad, twice;
// 32 bytes) or 4 floats (2D).  One 256-bit (3D) or 128-bit (2D) load then
// returns both x-corners of a cell row.  With Gz given, the first nz slices of
// the gradients, which share the [slice][padded node] index, are zeroed in the
// same pass.
template <int D>
__device__ __forceinline__ void pack_velocity(const float* __restrict__ v, float* __restrict__ Vp, const DevGrid& g,
                                              const SliceTable& tab, void* Gz, int nz, unsigned block,
                                              unsigned blocks) {
    const size_t nodes = padded_size(g);
    const size_t total = nodes * tab.n;
    const size_t zero = Gz != nullptr ? nodes * nz : 0;
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    constexpr int PS = (D == 3) ? 8 : 4;
    for (size_t i = block * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)blocks * blockDim.x) {
        if (i < zero) {
            if (D == 3) reinterpret_cast<float4*>(Gz)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            else reinterpret_cast<float2*>(Gz)[i] = make_float2(0.0f, 0.0f);
        }
        const unsigned nn = (unsigned)nodes;
        const int m = (int)((unsigned)i / nn);
        const unsigned node = (unsigned)i - (unsigned)m * nn;
        const int j = tab.j[m];
        const float th = tab.th[m];
        int px, py, pz;
        split_xyz(node, (unsigned)g.mp[0], (unsigned)g.mp[1], px, py, pz);
        float out[PS];
#pragma unroll
        for (int q = 0; q < PS; ++q) out[q] = 0.0f;
        const int y = py - LGNK_PAD, z = (D == 3) ? pz - LGNK_PAD : 0;
        const bool yz_in = y >= 0 && y < g.m[1] && z >= 0 && z < g.m[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int x = px + h - LGNK_PAD;
            if (yz_in && x >= 0 && x < g.m[0]) {
                const size_t s = ((size_t)z * g.m[1] + y) * g.m[0] + x;
#pragma unroll
                for (int c = 0; c < D; ++c) {
                    const float a = v[((size_t)j * D + c) * Mv + s];
                    float val = a;
                    if (th != 0.0f) val = fmaf(th, v[((size_t)(j + 1) * D + c) * Mv + s] - a, a);
                    out[h * (PS / 2) + c] = val;
                }
            }
        }
        float4* o = reinterpret_cast<float4*>(Vp + i * PS);
        o[0] = make_float4(out[0], out[1], out[2], out[3]);
        if (D == 3) o[1] = make_float4(out[4], out[5], out[6], out[7]);
    }
}

// Cell coordinates of node s of an (unpadded) velocity block.
template <int D>
__device__ __forceinline__ void coords(size_t s, const DevGrid& g, int* c) {
    int z;
    split_xyz((unsigned)s, (unsigned)g.m[0], (unsigned)g.m[1], c[0], c[1], z);
    c[2] = (D == 3) ? z : 0;
}

// Adjoint of the slice packing for the gradient: node j of component c gets
// scale * sum_m w_j(m) G_m[node], w_j(m) = 1 - th[m] if j = j[m], th[m] if j = j[m] + 1.
template <int D>
__global__ void distribute_gradient_kernel(const float* __restrict__ Gp, float* __restrict__ out, DevGrid g, int K,
                                           SliceTable tab, float scale) {
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t nodes = padded_size(g);
    const size_t total = Mv * K;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)((unsigned)i / (unsigned)Mv);
        const size_t s = (unsigned)i - (unsigned)j * (unsigned)Mv;
        int x, y, z;
        split_xyz((unsigned)s, (unsigned)g.m[0], (unsigned)g.m[1], x, y, z);
        const size_t node =
            ((size_t)(z + (D == 3 ? LGNK_PAD : 0)) * g.mp[1] + (y + LGNK_PAD)) * g.mp[0] + (x + LGNK_PAD);
        float acc[3] = {0.0f, 0.0f, 0.0f};
        for (int m = 0; m < tab.n; ++m) {
            float w = 0.0f;
            if (tab.j[m] == j) w = 1.0f - tab.th[m];
            else if (tab.j[m] + 1 == j) w = tab.th[m];
            if (w == 0.0f) continue;
            const size_t e = (size_t)m * nodes + node;
            if (D == 3) {
                const float4 a = reinterpret_cast<const float4*>(Gp)[e];
                acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]); acc[2] = fmaf(w, a.z, acc[2]);
            } else {
                const float2 a = reinterpret_cast<const float2*>(Gp)[e];
                acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]);
            }
        }
#pragma unroll
        for (int c = 0; c < D; ++c) out[((size_t)j * D + c) * Mv + s] = scale * acc[c];
    }
}

__device__ __forceinline__ void pack_image(const float* __restrict__ T, float* __restrict__ Tp, const DevGrid& g, int d,
                                           unsigned block, unsigned blocks) {
    const size_t total = padded_size(g);
    for (size_t i = block * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)blocks * blockDim.x) {
        int px, py, pz;
        split_xyz((unsigned)i, (unsigned)g.mp[0], (unsigned)g.mp[1], px, py, pz);
        const int x = px - LGNK_PAD, y = py - LGNK_PAD, z = (d == 3) ? pz - LGNK_PAD : 0;
        const bool in = x >= 0 && x < g.m[0] && y >= 0 && y < g.m[1] && z >= 0 && z < g.m[2];
        Tp[i] = in ? T[((size_t)z * g.m[1] + y) * g.m[0] + x] : 0.0f;
    }
}

// Whether a Gauss-Newton product with the stationary velocity v is cheaper by tangent sweeps than
// by rows (trace_impl.cuh): a row costs a block for every cell its characteristic enters, and
// a second sweep past the blocks that a thread keeps.  At the speed of a node a
// characteristic crosses sum_a |v_a| / h_a cell faces; a warp takes the mean of 64 nodes
// spread evenly.  Rows win up to about 0.12 N faces, 1.1 at most (the limit, from the caller).
// Products on 128^3 voxels by rows / by the kernel before the rows / by this choice, us: velocity
// of 64^3 cells, N = 4, displacements up to 25 voxels 503 / 417 / 394; velocity of
// 128^3 cells, N = 8, 25 voxels 952 / 794 / 748, 8 voxels 654 / 690 / 639.  Taken in the
// packing, the sample costs the trace one load; taken by each of its warps it cost 2% with N = 8.
template <int D>
__device__ __forceinline__ void pack_many_cells(const float* __restrict__ v, const DevGrid& g, float limit, int* many) {
    constexpr int kNodes = 64;
    constexpr float step[3] = {0.8191725f, 0.6710436f, 0.5497005f};      // evenly spread points of the unit cube
    if (threadIdx.x >= 32) return;
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    float faces = 0.0f;
#pragma unroll
    for (int k = 0; k < kNodes / 32; ++k) {
        size_t e = 0;
#pragma unroll
        for (int a = D - 1; a >= 0; --a) {
            const float x = ((float)(threadIdx.x + 32 * k) + 0.5f) * step[a];
            e = e * (size_t)g.m[a] + (size_t)min((int)((x - floorf(x)) * (float)g.m[a]), g.m[a] - 1);
        }
#pragma unroll
        for (int a = 0; a < D; ++a) faces = fmaf(fabsf(v[a * Mv + e]), g.inv_h[a], faces);
    }
    const int total = __reduce_add_sync(0xffffffffu, (int)(fminf(faces, 4096.0f) * 1024.0f));
    if (threadIdx.x == 0) *many = (float)total > limit * (1024.0f * kNodes) ? 1 : 0;
}

// Everything a call lays out before its trace: the parts take consecutive
// blocks.  The parts are bound by memory at large sizes (the brain-scale product's
// 492 us are what its two packings and its clearing took) and by their launches
// at small ones, each about 4 us of the host and 2 us of the GPU: the 64 x 64
// forward 21.1 -> 18.1 us with one launch for two, the 256 x 256 mass-preserving
// product 103 -> 95 us with one for three and a clearing.
template <int D>
__global__ void __launch_bounds__(kBlock) pack_kernel(const PackArgs A) {
    unsigned b = blockIdx.x;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const unsigned n = (unsigned)A.blocks[k];
        if (b < n) {
            const bool last = k == 1 || A.v[1] == nullptr;
            pack_velocity<D>(A.v[k], A.vp[k], A.vg, A.tab, last ? A.Gz : nullptr, A.nz, b, n);
            return;
        }
        b -= n;
    }
    if (b < (unsigned)A.blocks[2]) {
        pack_image(A.image, A.imagep, A.ig, D, b, (unsigned)A.blocks[2]);
        return;
    }
    b -= (unsigned)A.blocks[2];
    if (b >= (unsigned)A.blocks[3]) {
        pack_many_cells<D>(A.v[0], A.vg, A.many_faces, A.many);
        return;
    }
    const size_t total = padded_size(A.ig);
    for (size_t i = b * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)A.blocks[3] * blockDim.x)
        A.zero[i] = 0.0f;
}

__global__ void unpack_image_kernel(const float* __restrict__ acc, float* __restrict__ out, DevGrid g, int d) {
    const size_t M = (size_t)g.m[0] * g.m[1] * g.m[2];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < M; i += (size_t)gridDim.x * blockDim.x) {
        int x, y, z;
        split_xyz((unsigned)i, (unsigned)g.m[0], (unsigned)g.m[1], x, y, z);
        const size_t p = ((size_t)(z + (d == 3 ? LGNK_PAD : 0)) * g.mp[1] + (y + LGNK_PAD)) * g.mp[0] + (x + LGNK_PAD);
        out[i] = acc[p];
    }
}

__global__ void repad_image_kernel(float* acc, DevGrid g, int d, float scale) {
    const size_t total = padded_size(g);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        int px, py, pz;
        split_xyz((unsigned)i, (unsigned)g.mp[0], (unsigned)g.mp[1], px, py, pz);
        const int x = px - LGNK_PAD, y = py - LGNK_PAD, z = (d == 3) ? pz - LGNK_PAD : 0;
        const bool in = x >= 0 && x < g.m[0] && y >= 0 && y < g.m[1] && z >= 0 && z < g.m[2];
        acc[i] = in ? scale * acc[i] : 0.0f;
    }
}

// ------------------------------------------------------------- reductions --

// res = u1 - R (Eq. 10): partial sums of res^2 per block (FP64); rp (padded) = scale * res.
__global__ void residual_kernel(const float* __restrict__ u1, const float* __restrict__ R, float* __restrict__ rp,
                                DevGrid g, int d, float scale, double* partial) {
    const size_t M = (size_t)g.m[0] * g.m[1] * g.m[2];
    lsum s = lsum_zero();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < M; i += (size_t)gridDim.x * blockDim.x) {
        const float ui = u1[i], Ri = R[i];
        const float r = ui - Ri;
        lsum_add_sqdiff(s, ui, Ri);
        if (rp != nullptr) {
            int x, y, z;
            split_xyz((unsigned)i, (unsigned)g.m[0], (unsigned)g.m[1], x, y, z);
            const size_t p =
                ((size_t)(z + (d == 3 ? LGNK_PAD : 0)) * g.mp[1] + (y + LGNK_PAD)) * g.mp[0] + (x + LGNK_PAD);
            rp[p] = scale * r;
        }
    }
    s = lsum_block_sum(s);
    if (threadIdx.x == 0) partial[blockIdx.x] = lsum_value(s);
}

__global__ void dot_kernel(const float* __restrict__ a, const float* __restrict__ b, size_t count, double* partial) {
    lsum s = lsum_zero();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        lsum_add_prod(s, a[i], b[i]);
    s = lsum_block_sum(s);
    if (threadIdx.x == 0) partial[blockIdx.x] = lsum_value(s);
}

// One or two inner products sharing the first operand, finished in the same
// launch: every block writes its partial sums (FP64, in the partial buffer's
// slots), and the last block to finish (a counter, reset by that block) adds
// the partials in a fixed order (deterministic) into sc[slot_b] (a.b) and
// sc[slot_c] (a.c, when c is given), then the PCG step lengths of step `mode`,
// in FP64, from the inner products in sc ([2] p.Hp, [3] r.r, [4] r.z new,
// [5] r.z current):
//   mode 0 (slot_b = 2): alpha = rz / pHp, or 0 when pHp is not positive; f[0] = alpha, f[1] = -alpha
//   mode 1 (slot_c = 4): beta = rz_new / rz, then rz = rz_new;             f[2] = beta
//
// End of one PCG iteration inside a device-side loop (a CUDA-graph while
// node; ctl given, slot_b = 3): the same tests the host loop makes, on
// sc[2] = p.Hp, sc[3] = r.r and the tolerance sc[6] = pcg_rtol |g|.  ctl: [0]
// iterations run, [1] accepted iterations, [2] 1 = non-positive curvature,
// 2 = non-finite, [3] the cap.  The loop continues while the handle is
// non-zero; the cap ends it.  Part of the iteration's last inner product (a
// kernel of its own took 2.3 us of a 2D iteration of 45 us).
//
// What bounds it is the FP64 rate of the sums and the chain of latencies after
// the loads (block sum, fence, counter, partials, final sum, scalars, divide,
// test), so the scalars are read while the partials are, a warp of its own
// makes the loop test, and up to 32 partials are summed by one warp.  With the
// block sums of fsum.cuh and half the blocks: r.r and r.z of 64 x 64 x 2 values
// 7.4 -> 5.8 us, of 64^3 x 3 values 14.7 -> 11.3 us (192 blocks of 1024 threads,
// whose FP64 additions of empty slots count too: 35 us).
__device__ __forceinline__ void dot_blocks_finish(lsum s, lsum t, bool two, double* partial, unsigned* counter,
                                                  double* sc, int slot_b, int slot_c, int mode, float* f,
                                                  int* ctl = nullptr, cudaGraphConditionalHandle handle = 0) {
    __shared__ double dred[2][32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    s = lsum_block_sum<0>(s);
    if (two) t = lsum_block_sum<1>(t);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = lsum_value(s);
        if (two) partial[gridDim.x + blockIdx.x] = lsum_value(t);
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double u = 0.0, w = 0.0;              // the totals, in thread 0
    double rz = 0.0, php = 0.0, tol = 0.0;
    int it = 0, cap = 0;
    if (threadIdx.x == 0 && mode >= 0) rz = sc[5];
    if (threadIdx.x == 32 && ctl != nullptr) {
        php = sc[2];
        tol = sc[6];
        it = ctl[0] + 1;
        cap = ctl[3];
    }
    const volatile double* vp = partial;
    const int n = (int)gridDim.x;
    if (n <= 32) {
        if (lane < n && warp == 0) {
            u = vp[lane];
            if (two) w = vp[n + lane];
        }
    } else {
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            u += vp[i];
            if (two) w += vp[n + i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            u += __shfl_down_sync(0xffffffffu, u, o);
            if (two) w += __shfl_down_sync(0xffffffffu, w, o);
        }
        if (lane == 0) {
            dred[0][warp] = u;
            dred[1][warp] = w;
        }
        __syncthreads();
        u = lane < nw ? dred[0][lane] : 0.0;
        w = lane < nw ? dred[1][lane] : 0.0;
    }
    if (warp == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            u += __shfl_down_sync(0xffffffffu, u, o);
            if (two) w += __shfl_down_sync(0xffffffffu, w, o);
        }
    }
    if (ctl != nullptr) {                 // r.r to the thread of the loop test
        __syncthreads();
        if (threadIdx.x == 0) dred[0][0] = u;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        sc[slot_b] = u;
        if (two) sc[slot_c] = w;
        if (mode == 0) {
            const double a = u > 0.0 ? rz / u : 0.0;
            f[0] = (float)a;
            f[1] = (float)-a;
        } else if (mode == 1) {
            f[2] = (float)(w / rz);
            sc[5] = w;
        }
        *counter = 0u;
    }
    if (threadIdx.x == 32 && ctl != nullptr) {
        const double rr = dred[0][0];
        ctl[0] = it;
        unsigned go = 0;
        if (!isfinite(php) || !isfinite(rr)) {
            ctl[2] = 2;
        } else if (!(php > 0.0)) {
            ctl[2] = 1;
        } else {
            ctl[1] = it;
            go = (sqrt(rr) <= tol || it >= cap) ? 0u : 1u;
        }
        cudaGraphSetConditional(handle, go);
    }
}

// kDotElems elements of a thread are loaded before the first is added.
constexpr int kDotElems = 4;

__global__ void dot_fused_kernel(const float* __restrict__ a, const float* __restrict__ b,
                                 const float* __restrict__ c, size_t count, double* partial, unsigned* counter,
                                 double* sc, int slot_b, int slot_c, int mode, float* f, int* ctl,
                                 cudaGraphConditionalHandle handle) {
    lsum s = lsum_zero(), t = lsum_zero();
    const size_t step = (size_t)gridDim.x * blockDim.x;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += kDotElems * step) {
        float x[kDotElems], y[kDotElems], z[kDotElems];
#pragma unroll
        for (int k = 0; k < kDotElems; ++k) {
            const size_t e = i + k * step;
            const bool in = e < count;
            x[k] = in ? a[e] : 0.0f;
            y[k] = in ? b[e] : 0.0f;
            z[k] = in && c != nullptr ? c[e] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < kDotElems; ++k) {
            if (i + k * step < count) {
                lsum_add_prod(s, x[k], y[k]);
                if (c != nullptr) lsum_add_prod(t, x[k], z[k]);
            }
        }
    }
    dot_blocks_finish(s, t, c != nullptr, partial, counter, sc, slot_b, slot_c, mode, f, ctl, handle);
}

// The end of a Gauss-Newton product inside PCG with the diffusion
// regularizer, in one pass over the velocity nodes: Hp = gscale * (slice
// gradients distributed to the time nodes) + rscale * (B^T B p) + gamma * p
// (the arithmetic of distribute_gradient_kernel and laplacian_kernel, in the
// same order), then p.Hp into sc[2] and the step length alpha (mode 0), as
// dot_fused_kernel does.  Launched with the same block count as the fused
// inner products (partial holds one pair per block).
template <int D, bool DOT>
__global__ void hess_finish_kernel(const float* __restrict__ Gp, const float* __restrict__ p, float* __restrict__ Hp,
                                   DevGrid g, int K, SliceTable tab, float gscale, float rscale, float gamma,
                                   double* partial, unsigned* counter, double* sc, float* f) {
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t nodes = padded_size(g);
    const size_t total = Mv * K;
    const size_t stride[3] = {1, (size_t)g.m[0], (size_t)g.m[0] * g.m[1]};
    lsum dsum = lsum_zero();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)((unsigned)i / (unsigned)Mv);
        const size_t sn = (unsigned)i - (unsigned)j * (unsigned)Mv;
        int c[3];
        coords<D>(sn, g, c);
        const size_t node =
            ((size_t)(c[2] + (D == 3 ? LGNK_PAD : 0)) * g.mp[1] + (c[1] + LGNK_PAD)) * g.mp[0] + (c[0] + LGNK_PAD);
        float acc[3] = {0.0f, 0.0f, 0.0f};
        for (int m = 0; m < tab.n; ++m) {
            float w = 0.0f;
            if (tab.j[m] == j) w = 1.0f - tab.th[m];
            else if (tab.j[m] + 1 == j) w = tab.th[m];
            if (w == 0.0f) continue;
            const size_t e = (size_t)m * nodes + node;
            if (D == 3) {
                const float4 a = reinterpret_cast<const float4*>(Gp)[e];
                acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]); acc[2] = fmaf(w, a.z, acc[2]);
            } else {
                const float2 a = reinterpret_cast<const float2*>(Gp)[e];
                acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]);
            }
        }
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const size_t k = ((size_t)j * D + q) * Mv + sn;
            const float xi = p[k];
            float lap = 0.0f;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                float t = 0.0f;
                if (c[a] > 0) t += xi - p[k - stride[a]];
                if (c[a] < g.m[a] - 1) t += xi - p[k + stride[a]];
                lap = fmaf(t, g.inv_h[a] * g.inv_h[a], lap);
            }
            float r = rscale * lap;
            if (gamma != 0.0f) r = fmaf(gamma, xi, r);
            r += gscale * acc[q];
            Hp[k] = r;
            if (DOT) lsum_add_prod(dsum, xi, r);
        }
    }
    if (DOT) dot_blocks_finish(dsum, lsum_zero(), false, partial, counter, sc, 2, 2, 0, f);
}

// x += f[0] p and r += f[1] Hp (the PCG updates with alpha, -alpha)
__global__ void pcg_update_xr_kernel(float* x, const float* __restrict__ p, float* r, const float* __restrict__ Hp,
                                     const float* __restrict__ f, size_t count) {
    const float a = f[0], b = f[1];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
        x[i] = fmaf(a, p[i], x[i]);
        r[i] = fmaf(b, Hp[i], r[i]);
    }
}

// After the device-side PCG loop: when its first iteration met non-positive
// curvature (ctl[2] = 1 with no accepted iteration), the step is the
// preconditioned steepest-descent direction, x = z.
__global__ void pcg_curvature_fix_kernel(float* x, const float* __restrict__ z, const int* __restrict__ ctl,
                                         size_t count) {
    if (!(ctl[2] == 1 && ctl[1] == 0)) return;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        x[i] = z[i];
}

// y = a x + b y, a = *ap when ap is given, b = *bp when bp is given.
__global__ void axpby_dev_kernel(float a, const float* __restrict__ ap, const float* __restrict__ x, float b,
                                 const float* __restrict__ bp, float* y, size_t count) {
    const float ea = ap ? *ap : a, eb = bp ? *bp : b;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        y[i] = fmaf(ea, x[i], eb * y[i]);
}

// Deterministic final sum of the per-block partials, in one block: eight
// loads of a thread in flight at a time (8192 partials of a 128^3 trace took 7 to
// 16 us one by one in 256 threads).
constexpr int kReduceBlock = 1024;
__global__ void __launch_bounds__(kReduceBlock)
    reduce_kernel(const double* __restrict__ partial, int count, double* out) {
    double s = 0.0;
    for (int i = threadIdx.x; i < count; i += 8 * kReduceBlock) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = i + k * kReduceBlock < count ? __ldg(partial + i + k * kReduceBlock) : 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) s += v[k];
    }
    __shared__ double red[kReduceBlock / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = red[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) out[0] = s;
    }
}

// ----------------------------------------------------------- regularizers --

// out = addsrc + scale * (B^T B x) + gamma * gsrc: the Neumann Laplacian of each
// (time node, component) block, B the forward difference between neighbouring
// cell centres (interior faces only).
template <int D>
__global__ void laplacian_kernel(const float* __restrict__ x, float* out, DevGrid g, int nblk, float scale,
                                 float gamma, const float* gsrc, const float* addsrc) {
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t total = Mv * nblk;
    const size_t stride[3] = {1, (size_t)g.m[0], (size_t)g.m[0] * g.m[1]};
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t s = (unsigned)i % (unsigned)Mv;
        int c[3];
        coords<D>(s, g, c);
        const float xi = x[i];
        float acc = 0.0f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            float t = 0.0f;
            if (c[a] > 0) t += xi - x[i - stride[a]];
            if (c[a] < g.m[a] - 1) t += xi - x[i + stride[a]];
            acc = fmaf(t, g.inv_h[a] * g.inv_h[a], acc);
        }
        float r = scale * acc;
        if (gsrc != nullptr) r = fmaf(gamma, gsrc[i], r);
        if (addsrc != nullptr) r += addsrc[i];
        out[i] = r;
    }
}

// div[j] = sum_a (x_a[i+1] - x_a[i-1]) / (2 h_a), ends mirrored (one-sided).
template <int D>
__global__ void divergence_kernel(const float* __restrict__ x, float* __restrict__ div, DevGrid g, int K) {
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t total = Mv * K;
    const size_t stride[3] = {1, (size_t)g.m[0], (size_t)g.m[0] * g.m[1]};
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t s = (unsigned)i % (unsigned)Mv;
        const size_t j = (unsigned)i / (unsigned)Mv;
        int c[3];
        coords<D>(s, g, c);
        float acc = 0.0f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const float* xa = x + (j * D + a) * Mv;
            const size_t up = (c[a] < g.m[a] - 1) ? s + stride[a] : s;
            const size_t dn = (c[a] > 0) ? s - stride[a] : s;
            acc += (xa[up] - xa[dn]) * (0.5f * g.inv_h[a]);
        }
        div[i] = acc;
    }
}

// out_c = addsrc + smu * (A x_c) + slm * (D_c^T div) + gamma * x_c (elastic operator).
template <int D>
__global__ void elastic_kernel(const float* __restrict__ x, const float* __restrict__ div, float* out, DevGrid g,
                               int K, float smu, float slm, float gamma, const float* addsrc) {
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t total = Mv * K * D;
    const size_t stride[3] = {1, (size_t)g.m[0], (size_t)g.m[0] * g.m[1]};
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t s = (unsigned)i % (unsigned)Mv;
        const size_t blk = (unsigned)i / (unsigned)Mv;
        const int comp = (int)(blk % D);
        const size_t j = blk / D;
        int c[3];
        coords<D>(s, g, c);
        const float xi = x[i];
        float lap = 0.0f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            float t = 0.0f;
            if (c[a] > 0) t += xi - x[i - stride[a]];
            if (c[a] < g.m[a] - 1) t += xi - x[i + stride[a]];
            lap = fmaf(t, g.inv_h[a] * g.inv_h[a], lap);
        }
        // transpose of the centred difference along axis comp
        const float* dj = div + j * Mv;
        const int ci = c[comp], m = g.m[comp];
        const size_t st = stride[comp];
        float dt = 0.0f;
        if (ci >= 1) dt += dj[s - st];
        if (ci == m - 1) dt += dj[s];
        if (ci + 1 <= m - 1) dt -= dj[s + st];
        if (ci == 0) dt -= dj[s];
        dt *= 0.5f * g.inv_h[comp];
        float r = smu * lap + slm * dt + gamma * xi;
        if (addsrc != nullptr) r += addsrc[i];
        out[i] = r;
    }
}

// ------------------------------------------------------------------ DCT --

// out[.., k, ..] = sum_i C[k][i] in[.., i, ..] along one axis (inverse: C[i][k]);
// C is the orthonormal DCT-II matrix of that axis.
__global__ void dct_axis_kernel(const float* __restrict__ in, float* __restrict__ out, const float* __restrict__ C,
                                DevGrid g, int nblk, int axis, int inverse) {
    const size_t Mv = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t total = Mv * nblk;
    const int m = g.m[axis];
    const size_t st = (axis == 0) ? 1 : (axis == 1 ? (size_t)g.m[0] : (size_t)g.m[0] * g.m[1]);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t s = (unsigned)i % (unsigned)Mv;
        const int k = (int)((s / st) % m);
        const size_t base = i - (size_t)k * st;
        float acc = 0.0f;
        if (inverse) {
            for (int q = 0; q < m; ++q) acc = fmaf(__ldg(C + (size_t)q * m + k), in[base + q * st], acc);
        } else {
            const float* row = C + (size_t)k * m;
            for (int q = 0; q < m; ++q) acc = fmaf(__ldg(row + q), in[base + q * st], acc);
        }
        out[i] = acc;
    }
}

// 16-byte asynchronous copy from global to shared memory (both addresses
// 16-byte aligned), cached in L2 only; cp_async_wait_all() waits for every
// copy this thread issued.  A CTA issues all its staging copies before the
// first wait, so a tile arrives in about one memory round trip.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}

// the same for 4 bytes (rows that are not 16-byte aligned)
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// The same transform for axes of at most kDctTileMax cells, as a small
// register-blocked matrix product staged in shared memory.  Each array block
// is viewed as [outer][m][inner] (inner = product of the cell counts of the
// axes below `axis`).  A CTA transforms 64 lines: 64 consecutive inner
// positions of one outer index (axis > 0), or 64 consecutive x rows (axis 0,
// inner = 1; loaded and stored through shared memory so that global accesses
// stay coalesced).  The coefficient matrix sits in shared memory transposed,
// [q][k], and the tile as [q][line]; a thread computes a 4 x 4 block of
// (output index k, line), reading one float4 of each per q for 16 FMAs.  Every
// output is accumulated over q in increasing order, as in dct_axis_kernel.
constexpr int kDctTileMax = 128;
constexpr int kDctLines = 64;
constexpr int kDctLS = kDctLines + 4;        // tile row stride (float4-aligned)

// The two tables of an axis of m <= kDctTileMax cells (C its orthonormal DCT-II
// matrix), read by every tiled transform, each 2 h rows (h = ceil(m/2)) of two parts of
// P4 = h rounded up to 4 floats, zero padded (m = 1: of one part).
//   forward row q: C[2j][q] | C[2j+1][q]
//   inverse row r < h: C[2r][j] | C[2r+1][j], row h + r: C[2r][m-1-j] | C[2r+1][m-1-j]
// The first h rows are what the transforms by halves need.  The direct sums read the
// inverse table as rows k of P4 floats, C[k][j], and the same mirrored h rows further on.
struct DctTable {
    const float* p;
    int m, h, P4, stride;     // cells; ceil(m/2); floats of a part and of a row
    __host__ __device__ __forceinline__ int step(bool full, bool inverse) const {     // from row to row
        return full && inverse ? P4 : stride;
    }
    __host__ __device__ __forceinline__ int part(bool full, bool inverse) const {     // offset of the second part
        return full && inverse ? h * stride : (m > 1 ? P4 : 0);
    }
};

inline DctTable dct_table(const float* p, int m) {
    DctTable t;
    t.p = p;
    t.m = m;
    t.h = (m + 1) / 2;
    t.P4 = (t.h + 3) & ~3;
    t.stride = m > 1 ? 2 * t.P4 : t.P4;
    return t;
}

// Output index (forward: mode, inverse: position) of column c of a table, -1 for padding.
__device__ __forceinline__ int dct_column(int c, int P4, int m, bool inverse) {
    const int j = c < P4 ? c : c - P4, h = (m + 1) / 2;
    if (inverse) return c < P4 ? (j < h ? j : -1) : (j < m - h ? m - 1 - j : -1);
    const int k = 2 * j + (c < P4 ? 0 : 1);
    return k < m ? k : -1;
}

template <bool XAXIS>
__global__ void __launch_bounds__(kBlock) dct_tile_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                          const DctTable tab, int inverse, long long inner,
                                                          long long lines, int vec_in) {
    extern __shared__ __align__(16) float sm[];
    const int m = tab.m, MP = tab.stride;        // columns, whole float4s
    float* Ct = sm;                              // the table of the direction
    float* tile = sm + 2 * tab.h * MP;           // [q][kDctLS], later the output stage of axis 0
    const int t = threadIdx.x, step = tab.step(true, inverse), part = tab.part(true, inverse);
    for (int e = t; e < 2 * tab.h * MP / 4; e += kBlock) cp_async16(Ct + 4 * e, tab.p + 4 * e);
    long long o = 0, i0 = 0, r0 = 0;
    if (XAXIS) {                                 // lines are rows: loaded transposed, element by element
        r0 = (long long)blockIdx.x * kDctLines;
        for (int e = t; e < kDctLines * m; e += kBlock) {
            const int l = e / m, q = e % m;
            tile[q * kDctLS + l] = (r0 + l < lines) ? __ldg(in + (size_t)(r0 + l) * m + q) : 0.0f;
        }
    } else {
        const long long tiles = (inner + kDctLines - 1) / kDctLines;
        o = blockIdx.x / tiles;
        i0 = (blockIdx.x - o * tiles) * kDctLines;
        if (vec_in) {                            // inner a multiple of 4, in 16-byte aligned
            for (int e = t; e < m * (kDctLines / 4); e += kBlock) {
                const int q = e / (kDctLines / 4), l = 4 * (e % (kDctLines / 4));
                if (i0 + l < inner) cp_async16(tile + q * kDctLS + l, in + ((size_t)o * m + q) * inner + i0 + l);
                else *reinterpret_cast<float4*>(tile + q * kDctLS + l) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
        } else {
            for (int e = t; e < kDctLines * m; e += kBlock) {
                const int q = e / kDctLines, l = e % kDctLines;
                tile[q * kDctLS + l] = (i0 + l < inner) ? __ldg(in + ((size_t)o * m + q) * inner + i0 + l) : 0.0f;
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();
    const int ntask = (MP / 4) * (kDctLines / 4);
    constexpr int SS = kDctTileMax + 1;          // output stage row stride (axis 0)
    float acc[2][4][4];                          // at most two tasks per thread (MP <= 128)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int task = t + r * kBlock;
        if (task >= ntask) break;
        const int kb = task / (kDctLines / 4), lb = task % (kDctLines / 4);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[r][i][j] = 0.0f;
        const float4* cp =
            reinterpret_cast<const float4*>(Ct + (4 * kb < tab.P4 ? 4 * kb : part + 4 * kb - tab.P4));
        const float4* xp = reinterpret_cast<const float4*>(tile) + lb;
#pragma unroll 4
        for (int q = 0; q < m; ++q) {
            const float4 c = cp[q * (step / 4)];
            const float4 x = xp[q * (kDctLS / 4)];
            const float cv[4] = {c.x, c.y, c.z, c.w}, xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[r][i][j] = fmaf(cv[i], xv[j], acc[r][i][j]);
        }
        if (!XAXIS) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = dct_column(4 * kb + i, tab.P4, m, inverse != 0);
                if (k < 0) continue;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const long long l = i0 + 4 * lb + j;
                    if (l < inner) out[((size_t)o * m + k) * inner + l] = acc[r][i][j];
                }
            }
        }
    }
    if (XAXIS) {
        __syncthreads();                         // the tile becomes the output stage [line][k]
        float* stage = tile;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int task = t + r * kBlock;
            if (task >= ntask) break;
            const int kb = task / (kDctLines / 4), lb = task % (kDctLines / 4);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = dct_column(4 * kb + i, tab.P4, m, inverse != 0);
                if (k < 0) continue;
#pragma unroll
                for (int j = 0; j < 4; ++j) stage[(4 * lb + j) * SS + k] = acc[r][i][j];
            }
        }
        __syncthreads();
        for (int e = t; e < kDctLines * m; e += kBlock) {
            const int l = e / m, k = e % m;
            if (r0 + l < lines) out[(size_t)(r0 + l) * m + k] = stage[l * SS + k];
        }
    }
}

// ---- transforms by halves.  The DCT-II rows are even or odd about the middle of
// the axis, C[k][m-1-q] = (-1)^k C[k][q], so with s_q = x_q + x_(m-1-q) and
// d_q = x_q - x_(m-1-q) the even modes are sums over s and the odd modes over d of
// half the length, and the inverse is x_q = E_q + O_q, x_(m-1-q) = E_q - O_q with
// E (O) the sum over the even (odd) modes: half the FMAs and half the table.
//
// The operand of either direction is a tile of lines in shared
// memory, [index][LS], first folded into s and d (forward).  A task is 4 even and 4
// odd outputs (forward: 8 consecutive modes; inverse: 4 q and their mirrors) of LT
// lines, done by one thread (LT = 8: 64 FMAs per 6 shared loads) or, where a CTA
// would have few threads, by two neighbouring lanes (SPLIT, LT = 4), one for the
// even and one for the odd part, which then exchange what the other stores.
//
// With FULL the same tasks sum over the whole axis in increasing index order.  The
// PCG of a 3D solve uses these (precond_apply): its iterates then keep the rounding of
// the direct sums.  The second Gauss-Newton step takes
// grad T, which jumps at image nodes, at end points of the first step's velocity, so
// a change of that velocity by a rounding can move a voxel's row of J by O(1).

// acc_e[i][l] = sum_r tab[r][j0 + i] E_r[l], acc_o = sum_r tab[r][po + j0 + i] O_r[l]
// over the m/2 pairs and the unpaired even row of an odd m; row r of the even
// (odd) operand is at even + r se (odd + r so).  FULL: over m rows of one operand.
template <int LT, bool FULL>
__device__ __forceinline__ void dct_half_product(const float* tab, int po, int stride, int m, int j0, const float* even,
                                                 int se, const float* odd, int so, float (&ae)[4][LT],
                                                 float (&ao)[4][LT]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int l = 0; l < LT; ++l) ae[i][l] = ao[i][l] = 0.0f;
    const int n = FULL ? m : m / 2;
    const float* te = tab + j0;
#pragma unroll 2
    for (int r = 0; r < n; ++r) {
        const float4 a = *reinterpret_cast<const float4*>(te);
        const float4 b = *reinterpret_cast<const float4*>(te + po);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
        float x[LT], y[FULL ? 1 : LT];
#pragma unroll
        for (int l = 0; l < LT; l += 4) {
            *reinterpret_cast<float4*>(x + l) = *reinterpret_cast<const float4*>(even + l);
            if constexpr (!FULL) *reinterpret_cast<float4*>(y + l) = *reinterpret_cast<const float4*>(odd + l);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int l = 0; l < LT; ++l) {
                ae[i][l] = fmaf(av[i], x[l], ae[i][l]);
                ao[i][l] = fmaf(bv[i], FULL ? x[l] : y[FULL ? 0 : l], ao[i][l]);
            }
        te += stride;
        even += se;
        odd += so;
    }
    if (!FULL && (m & 1)) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int l = 0; l < LT; ++l) ae[i][l] = fmaf(te[i], even[l], ae[i][l]);
    }
}

// The even (p = 0) or odd (p = 1) part of a task (FULL, forward: its first or last four modes).
template <bool FULL>
__device__ __forceinline__ void dct_half_part(const float* tab, int po, int stride, int m, bool inverse, const float* S,
                                              int LS, int j0, int l0, int p, float (&a)[4][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int l = 0; l < 4; ++l) a[i][l] = 0.0f;
    const int n = FULL ? m : m / 2, st = FULL ? LS : (inverse ? 2 * LS : (p ? -LS : LS));
    const float* t = tab + j0 + p * po;
    const float* x = S + l0 + (FULL ? 0 : (inverse ? p * LS : p * (m - 1) * LS));
    if (FULL && !inverse) {
        t = tab + j0 + 2 * p;
#pragma unroll 4
        for (int r = 0; r < n; ++r) {
            const float2 e = *reinterpret_cast<const float2*>(t), o = *reinterpret_cast<const float2*>(t + po);
            const float4 v = *reinterpret_cast<const float4*>(x);
            const float cv[4] = {e.x, o.x, e.y, o.y}, xv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int l = 0; l < 4; ++l) a[i][l] = fmaf(cv[i], xv[l], a[i][l]);
            t += stride;
            x += LS;
        }
        return;
    }
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
        const float4 c = *reinterpret_cast<const float4*>(t);
        const float4 v = *reinterpret_cast<const float4*>(x);
        const float cv[4] = {c.x, c.y, c.z, c.w}, xv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int l = 0; l < 4; ++l) a[i][l] = fmaf(cv[i], xv[l], a[i][l]);
        t += stride;
        x += st;
    }
    if (!FULL && (m & 1) && p == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int l = 0; l < 4; ++l) a[i][l] = fmaf(t[i], x[l], a[i][l]);
    }
}

// Line l of a split task: the four outputs this lane stores, from position
// `at` (dct_part_start) on.  Every lane of the warp calls it.
template <bool FULL>
__device__ __forceinline__ float4 dct_part_outputs(bool inverse, const float (&a)[4][4], int l, int p) {
    float v[4];
    if (inverse) {           // even lane E + O at j0 + i; odd lane E - O, mirrored (FULL: the sums themselves)
        float w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (FULL) {
                w[i] = a[i][l];
            } else {
                const float o = __shfl_xor_sync(0xffffffffu, a[i][l], 1);
                w[i] = p ? o - a[i][l] : a[i][l] + o;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = p ? w[3 - i] : w[i];
    } else if (FULL) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = a[i][l];
    } else {                 // modes e0 o0 e1 o1 (even lane), e2 o2 e3 o3 (odd lane)
        const float r0 = __shfl_xor_sync(0xffffffffu, p ? a[0][l] : a[2][l], 1);
        const float r1 = __shfl_xor_sync(0xffffffffu, p ? a[1][l] : a[3][l], 1);
        v[0] = p ? r0 : a[0][l];
        v[1] = p ? a[2][l] : r0;
        v[2] = p ? r1 : a[1][l];
        v[3] = p ? a[3][l] : r1;
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ int dct_part_start(bool inverse, int m, int j0, int p) {
    return inverse ? (p ? m - 4 - j0 : j0) : 2 * j0 + 4 * p;
}

// ... into a row of m values: positions below 0 or past m (forward), past the middle
// (inverse) are no outputs of this lane.
__device__ __forceinline__ void dct_store_part(float* dst, int m, int j0, int p, bool inverse, bool vec, float4 v) {
    const int at = dct_part_start(inverse, m, j0, p), h = (m + 1) / 2;
    if (vec && (inverse ? j0 + 4 <= m / 2 : at + 4 <= m)) {
        *reinterpret_cast<float4*>(dst + at) = v;
        return;
    }
    const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (inverse ? j0 + (p ? 3 - i : i) < h : at + i < m) dst[at + i] = x[i];
}

// x_q, x_(m-1-q) -> s_q, d_q in place (rows of a tile); every thread of the CTA.
__device__ __forceinline__ void dct_fold(float* S, int LS, int m, int lines) {
    const int c4 = (lines + 3) / 4, n = m / 2;
    for (int e = threadIdx.x; e < n * c4; e += blockDim.x) {
        const int q = e / c4, l = 4 * (e % c4);
        float4* p = reinterpret_cast<float4*>(S + q * LS + l);
        float4* r = reinterpret_cast<float4*>(S + (m - 1 - q) * LS + l);
        const float4 a = *p, b = *r;
        *p = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        *r = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
    }
}

// One direction of an axis on the tile S: the product of this thread's task.
template <int LT, bool FULL>
__device__ __forceinline__ void dct_half_axis(const float* tab, int po, int stride, int m, bool inverse, const float* S,
                                              int LS, int j0, int l0, float (&ae)[4][LT], float (&ao)[4][LT]) {
    if (FULL) dct_half_product<LT, true>(tab, po, stride, m, j0, S + l0, LS, S + l0, LS, ae, ao);
    else if (inverse) dct_half_product<LT, false>(tab, po, stride, m, j0, S + l0, 2 * LS, S + LS + l0, 2 * LS, ae, ao);
    else dct_half_product<LT, false>(tab, po, stride, m, j0, S + l0, LS, S + (m - 1) * LS + l0, -LS, ae, ao);
}

// The 8 outputs of line l of a task: forward, modes 2 j0 .. 2 j0 + 7 in v; inverse,
// positions j0 .. j0 + 3 in v[0..3] and m - 1 - j0 - 3 .. m - 1 - j0 in v[4..7].
template <int LT, bool FULL>
__device__ __forceinline__ void dct_outputs(bool inverse, const float (&ae)[4][LT], const float (&ao)[4][LT], int l,
                                            float* v) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (inverse) {
            v[i] = FULL ? ae[i][l] : ae[i][l] + ao[i][l];
            v[7 - i] = FULL ? ao[i][l] : ae[i][l] - ao[i][l];
        } else {
            v[2 * i] = ae[i][l];
            v[2 * i + 1] = ao[i][l];
        }
    }
}

// Stores the 8 outputs of one line into a row of m values at dst.
__device__ __forceinline__ void dct_store_line(float* dst, int m, int j0, bool inverse, bool vec, const float* v) {
    const int h = (m + 1) / 2, a = inverse ? j0 : 2 * j0, b = inverse ? m - 4 - j0 : 2 * j0 + 4;
    // whole groups: forward both halves inside m; inverse 4 positions below the middle, mirrors distinct
    if (vec && (inverse ? j0 + 4 <= m / 2 : b + 4 <= m)) {
        *reinterpret_cast<float4*>(dst + a) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(dst + b) = make_float4(v[4], v[5], v[6], v[7]);
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (inverse) {
            if (j0 + i < h) {
                dst[j0 + i] = v[i];
                dst[m - 1 - j0 - i] = v[7 - i];      // the middle of an odd m is written twice with the same value
            }
        } else {
            if (a + i < m) dst[a + i] = v[i];
            if (b + i < m) dst[b + i] = v[4 + i];
        }
    }
}

// Rows of a table that a transform stages.
template <bool FULL>
__host__ __device__ inline int dct_rows(int m) {
    return (FULL ? 2 : 1) * ((m + 1) / 2);
}

template <bool FULL>
__device__ __forceinline__ void dct_stage_table(float* dst, const DctTable& t) {
    const int n = dct_rows<FULL>(t.m) * t.stride / 4;
    for (int e = threadIdx.x; e < n; e += blockDim.x) cp_async16(dst + 4 * e, t.p + 4 * e);
}

// The last axis of the preconditioner in one pass: forward transform, the
// spectral scale inv_eig (per mode, the same for every block) and the inverse,
// with the scaled modes kept in shared memory in between.  A CTA takes
// LINES lines (64, or 32 where that leaves SMs without a CTA), a thread 8 outputs
// of 4 lines.
constexpr int kDctFusedLines = 64;

template <int LINES, bool SPLIT, bool FULL>
__global__ void __launch_bounds__(kBlock) dct_last_half_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                               const DctTable tf, const DctTable ti,
                                                               const float* __restrict__ inv_eig, int m,
                                                               long long inner, int vec_in) {
    constexpr int LS = LINES + 4, LT = 4;
    extern __shared__ __align__(16) float sm[];
    float* F = sm;
    float* I = F + dct_rows<FULL>(m) * tf.stride;
    float* tile = I + dct_rows<FULL>(m) * ti.stride;     // [q][LS], then the scaled modes [k][LS]
    dct_stage_table<FULL>(F, tf);
    dct_stage_table<FULL>(I, ti);
    const long long o = blockIdx.y, i0 = (long long)blockIdx.x * LINES;
    const int t = threadIdx.x;
    if (vec_in) {                     // inner a multiple of 4, in 16-byte aligned: whole float4s in or out
        for (int e = t; e < m * (LINES / 4); e += blockDim.x) {
            const int q = e / (LINES / 4), l = 4 * (e % (LINES / 4));
            if (i0 + l < inner) cp_async16(tile + q * LS + l, in + ((size_t)o * m + q) * inner + i0 + l);
            else *reinterpret_cast<float4*>(tile + q * LS + l) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    } else {
        for (int e = t; e < LINES * m; e += blockDim.x) {
            const int q = e / LINES, l = e % LINES;
            if (i0 + l < inner) cp_async4(tile + q * LS + l, in + ((size_t)o * m + q) * inner + i0 + l);
            else tile[q * LS + l] = 0.0f;
        }
    }
    cp_async_wait_all();
    __syncthreads();
    if (!FULL) {
        dct_fold(tile, LS, m, LINES);
        __syncthreads();
    }
    const int p = SPLIT ? t & 1 : 0, task = SPLIT ? t >> 1 : t;
    const int l0 = LT * (task % (LINES / LT)), j0 = 4 * (task / (LINES / LT));
    const int h = (m + 1) / 2;
    const bool act = j0 < h;
    float ae[4][LT], ao[4][LT];
    if (act) {
        const int po = tf.part(FULL, false), st = tf.step(FULL, false);
        if (SPLIT) dct_half_part<FULL>(F, po, st, m, false, tile, LS, j0, l0, p, ae);
        else dct_half_axis<LT, FULL>(F, po, st, m, false, tile, LS, j0, l0, ae, ao);
    }
    __syncthreads();                  // every thread is done reading the tile
    const bool vec = vec_in && i0 + l0 + LT <= inner;
    if (act) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < (SPLIT ? 1 : 2); ++q) {
                const int k = SPLIT && FULL ? 2 * j0 + 4 * p + i : 2 * (j0 + i) + (SPLIT ? p : q);
                if (k >= m) continue;
                const float4 v = q ? make_float4(ao[i][0], ao[i][1], ao[i][2], ao[i][3])
                                   : make_float4(ae[i][0], ae[i][1], ae[i][2], ae[i][3]);
                const float* e = inv_eig + (size_t)k * inner + i0 + l0;
                float4 sc;
                if (vec) {
                    sc = __ldg(reinterpret_cast<const float4*>(e));
                } else {
                    sc.x = i0 + l0 < inner ? __ldg(e) : 0.0f;
                    sc.y = i0 + l0 + 1 < inner ? __ldg(e + 1) : 0.0f;
                    sc.z = i0 + l0 + 2 < inner ? __ldg(e + 2) : 0.0f;
                    sc.w = i0 + l0 + 3 < inner ? __ldg(e + 3) : 0.0f;
                }
                *reinterpret_cast<float4*>(tile + k * LS + l0) =
                    make_float4(v.x * sc.x, v.y * sc.y, v.z * sc.z, v.w * sc.w);
            }
    }
    __syncthreads();
    if (act) {
        const int po = ti.part(FULL, true), st = ti.step(FULL, true);
        if (SPLIT) dct_half_part<FULL>(I, po, st, m, true, tile, LS, j0, l0, p, ae);
        else dct_half_axis<LT, FULL>(I, po, st, m, true, tile, LS, j0, l0, ae, ao);
    }
    const bool vec_out = vec && reinterpret_cast<uintptr_t>(out) % 16 == 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < (SPLIT ? 1 : 2); ++c) {
            const int mir = SPLIT ? p : c, q = mir ? m - 1 - j0 - i : j0 + i;
            float v[LT];
#pragma unroll
            for (int l = 0; l < LT; ++l) {
                if constexpr (FULL) {
                    v[l] = !SPLIT && c ? ao[i][l] : ae[i][l];
                } else if (SPLIT) {
                    const float o = __shfl_xor_sync(0xffffffffu, ae[i][l], 1);
                    v[l] = p ? o - ae[i][l] : ae[i][l] + o;
                } else {
                    v[l] = c ? ae[i][l] - ao[i][l] : ae[i][l] + ao[i][l];
                }
            }
            if (!act || j0 + i >= h) continue;
            float* d = out + ((size_t)o * m + q) * inner + i0 + l0;
            if (vec_out) {
                *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int l = 0; l < LT; ++l)
                    if (i0 + l0 + l < inner) d[l] = v[l];
            }
        }
}

// The y and x axes of the transform on whole xy planes (both at most
// kDctPlaneMax cells): a CTA holds one plane of one (block, z) in shared
// memory and applies the y axis and then the x axis, two products chained
// through shared memory.  The y result goes back transposed, [x][k], so that both
// products read float4 rows and the plane is loaded and stored row-major.  The
// two axes commute, so one order serves both directions.
constexpr int kDctPlaneMax = 128;
constexpr int kDctFullPlaneMax = 64;         // of the direct sums (their tables are twice as long)

// A thread's task in the plane kernels: LT = 8 lines, both parts; LT = 4 (split), one part.
template <int LT, bool FULL>
struct PlaneTask {
    static constexpr bool SPLIT = LT == 4;
    int j0, l0, p;
    bool act;
    float ae[4][LT], ao[SPLIT ? 1 : 4][SPLIT ? 1 : LT];

    // consecutive threads take consecutive output groups of one line group: the
    // transposed store and the store of the plane then write whole rows
    __device__ __forceinline__ void place(int m, int lines) {
        const int t = SPLIT ? threadIdx.x >> 1 : threadIdx.x, g = ((m + 1) / 2 + 3) / 4;
        p = SPLIT ? threadIdx.x & 1 : 0;
        j0 = 4 * (t % g);
        l0 = LT * (t / g);
        act = l0 < lines;
    }
    __device__ __forceinline__ void product(const float* tab, const DctTable& t, int m, bool inverse, const float* S,
                                            int LS) {
        if (!act) return;
        const int po = t.part(FULL, inverse), st = t.step(FULL, inverse);
        if constexpr (SPLIT) dct_half_part<FULL>(tab, po, st, m, inverse, S, LS, j0, l0, p, ae);
        else dct_half_axis<LT, FULL>(tab, po, st, m, inverse, S, LS, j0, l0, ae, ao);
    }
    // Stores the outputs of lines l0 .. as rows of m values, `row` floats apart;
    // scale: NULL or factors of the same layout (rows of m).  Every thread calls it.
    __device__ __forceinline__ void store(float* dst, size_t row, int m, int lines, bool inverse, bool vec,
                                          const float* scale) {
#pragma unroll
        for (int l = 0; l < LT; ++l) {
            const bool in = act && l0 + l < lines;
            if constexpr (SPLIT) {
                float4 v = dct_part_outputs<FULL>(inverse, ae, l, p);
                if (!in) continue;
                if (scale != nullptr) {
                    const int at = dct_part_start(inverse, m, j0, p);
                    const float* sc = scale + (size_t)(l0 + l) * m + at;
                    v.x *= at < m ? __ldg(sc) : 0.0f;
                    v.y *= at + 1 < m ? __ldg(sc + 1) : 0.0f;
                    v.z *= at + 2 < m ? __ldg(sc + 2) : 0.0f;
                    v.w *= at + 3 < m ? __ldg(sc + 3) : 0.0f;
                }
                dct_store_part(dst + (l0 + l) * row, m, j0, p, inverse, vec, v);
            } else {
                if (!in) continue;
                float v[8];
                dct_outputs<LT, FULL>(inverse, ae, ao, l, v);
                if (scale != nullptr) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        v[i] *= 2 * j0 + i < m ? __ldg(scale + (size_t)(l0 + l) * m + 2 * j0 + i) : 0.0f;
                }
                dct_store_line(dst + (l0 + l) * row, m, j0, inverse, vec, v);
            }
        }
    }
};

// Both products of the plane in S (rows [y][LS]), every thread of the CTA; the x
// product's outputs (lines = ky) stay in the task.
template <int LT, bool FULL>
__device__ __forceinline__ void plane_half_yx(const float* Ty, const DctTable& ty, const float* Tx, const DctTable& tx,
                                              float* S, int mx, int my, int LS, int LTR, bool inverse,
                                              PlaneTask<LT, FULL>& k) {
    if (!FULL && !inverse) {
        dct_fold(S, LS, my, mx);
        __syncthreads();
    }
    k.place(my, mx);
    k.product(Ty, ty, my, inverse, S, LS);
    __syncthreads();                      // every read of the plane is done
    k.store(S, LTR, my, mx, inverse, my % 4 == 0, nullptr);
    __syncthreads();
    if (!FULL && !inverse) {
        dct_fold(S, LTR, mx, my);
        __syncthreads();
    }
    k.place(mx, my);
    k.product(Tx, tx, mx, inverse, S, LTR);
}

// Stage a plane of `in` into S rows [y][LS].
__device__ __forceinline__ void plane_load(const float* __restrict__ in, size_t base, float* S, int mx, int my, int LS,
                                           int vec_in) {
    if (vec_in) {                         // mx a multiple of 4, in 16-byte aligned
        const int c4 = mx / 4;
        for (int e = threadIdx.x; e < my * c4; e += blockDim.x) {
            const int y = e / c4, x = 4 * (e % c4);
            cp_async16(S + y * LS + x, in + base + (size_t)y * mx + x);
        }
    } else {
        for (int e = threadIdx.x; e < my * mx; e += blockDim.x) {
            const int y = e / mx, x = e % mx;
            cp_async4(S + y * LS + x, in + base + e);
        }
    }
}

template <int LT, bool FULL>
__global__ void __launch_bounds__(kBlock) dct_plane_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                           const DctTable tx, const DctTable ty, int inverse, int mx,
                                                           int my, int vec_in, int vec_out) {
    extern __shared__ __align__(16) float sm[];
    const int LS = ((mx + 3) & ~3) + 4, LTR = ((my + 3) & ~3) + 4;   // row strides of [y][x] and of [x][k]
    float* Ty = sm;
    float* Tx = Ty + dct_rows<FULL>(my) * ty.stride;
    float* S = Tx + dct_rows<FULL>(mx) * tx.stride;  // the plane, later the y result transposed
    dct_stage_table<FULL>(Ty, ty);
    dct_stage_table<FULL>(Tx, tx);
    const size_t base = (size_t)blockIdx.x * mx * my;
    plane_load(in, base, S, mx, my, LS, vec_in);
    cp_async_wait_all();
    __syncthreads();
    PlaneTask<LT, FULL> k;
    plane_half_yx<LT, FULL>(Ty, ty, Tx, tx, S, mx, my, LS, LTR, inverse != 0, k);
    k.store(out + base, mx, mx, my, inverse != 0, vec_out != 0, nullptr);
}

// The whole 2D preconditioner on one plane (a (time node, component) block) in
// one CTA: forward, scale by inv_eig, inverse, with the scaled modes written
// back into the plane buffer between the two halves.  Few planes leave most SMs idle, but
// up to 128 x 128 the three launches of the per-axis path cost more: two planes of
// 65 x 65 33 -> 21 us, of 128 x 16 41 -> 11, of 128 x 128 51 -> 43, of 127 x 125 56 -> 51.
template <int LT>
__global__ void __launch_bounds__(kBlock) dct_plane2d_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                             const DctTable fx, const DctTable fy, const DctTable ix,
                                                             const DctTable iy, const float* __restrict__ inv_eig,
                                                             int mx, int my, int vec_in, int vec_out) {
    extern __shared__ __align__(16) float sm[];
    const int LS = ((mx + 3) & ~3) + 4, LTR = ((my + 3) & ~3) + 4;
    float* Fy = sm;
    float* Fx = Fy + dct_rows<false>(my) * fy.stride;
    float* Iy = Fx + dct_rows<false>(mx) * fx.stride;
    float* Ix = Iy + dct_rows<false>(my) * iy.stride;
    float* S = Ix + dct_rows<false>(mx) * ix.stride;
    dct_stage_table<false>(Fy, fy);
    dct_stage_table<false>(Fx, fx);
    dct_stage_table<false>(Iy, iy);
    dct_stage_table<false>(Ix, ix);
    const size_t base = (size_t)blockIdx.x * mx * my;
    plane_load(in, base, S, mx, my, LS, vec_in);
    cp_async_wait_all();
    __syncthreads();
    PlaneTask<LT, false> k;
    plane_half_yx<LT, false>(Fy, fy, Fx, fx, S, mx, my, LS, LTR, false, k);
    // the scaled modes back as rows [ky][LS] once every thread is done with the transposed buffer
    __syncthreads();
    k.store(S, LS, mx, my, false, mx % 4 == 0, inv_eig);
    __syncthreads();
    plane_half_yx<LT, false>(Iy, iy, Ix, ix, S, mx, my, LS, LTR, true, k);
    k.store(out + base, mx, mx, my, true, vec_out != 0, nullptr);
}

// Floats of an axis's staged table
template <bool FULL>
inline size_t staged_floats(int m) {
    return (size_t)dct_rows<FULL>(m) * dct_table(nullptr, m).stride;
}

// Shared memory of the plane kernels with `dirs` directions' tables.
template <bool FULL>
inline size_t dct_plane_smem(int mx, int my, int dirs) {
    const size_t LS = (size_t)((mx + 3) & ~3) + 4, LTR = (size_t)((my + 3) & ~3) + 4;
    const size_t plane = std::max((size_t)my * LS, (size_t)mx * LTR) + 8;    // (rows are read in groups of 8 lines)
    return (dirs * (staged_floats<FULL>(mx) + staged_floats<FULL>(my)) + plane) * sizeof(float);
}

// Threads with a task in a plane kernel, for either form (the larger of the two
// products); the split form where it needs at most kBlock.  Every launch has kBlock
// threads, or with many CTAs only those with a task (dct_threads).
inline int dct_plane_threads(int mx, int my, int lt) {
    const int ty = ((my + 1) / 2 + 3) / 4 * ((mx + lt - 1) / lt), tx = ((mx + 1) / 2 + 3) / 4 * ((my + lt - 1) / lt);
    return ((lt == 4 ? 2 : 1) * std::max(ty, tx) + 31) / 32 * 32;
}
// Threads of a CTA with `tasks` threads' tasks: kBlock where the CTAs hardly fill the
// GPU, since threads without a task help to stage and fold (a 70 x 70 plane alone: 30
// us with 96, 23 us with 128 threads); else just those, so that more CTAs fit (2160
// planes of 96 x 112: 204 against 180 us).
inline int dct_threads(int tasks, long long blocks) {
    return blocks < reduce_block_cap() / 2 ? kBlock : (tasks + 31) / 32 * 32;
}
inline bool dct_plane_split(int mx, int my) { return dct_plane_threads(mx, my, 4) <= kBlock; }

// Shared memory of dct_tile_kernel for an axis of m cells (bytes).
inline size_t dct_tile_smem(int m) {
    const size_t tile = std::max((size_t)m * kDctLS, (size_t)kDctLines * (kDctTileMax + 1));
    return (dct_table_floats(m) + tile) * sizeof(float);
}

__global__ void scale_modes_kernel(float* x, const float* __restrict__ inv_eig, size_t block_elems, size_t count) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        x[i] *= inv_eig[i % block_elems];
}

__global__ void add_scaled_kernel(float* out, const float* x, float ax, const float* y, float ay, size_t count) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        out[i] = fmaf(ax, x[i], ay * y[i]);
}

// ------------------------------------------------------------- multilevel --

// Coarse cell = average of the 2^d fine cells that tile it (fine m = 2 coarse m).
template <int D>
__global__ void restrict_image_kernel(const float* __restrict__ F, float* __restrict__ C, DevGrid cg) {
    const size_t Mc = (size_t)cg.m[0] * cg.m[1] * cg.m[2];
    const int fm0 = 2 * cg.m[0], fm1 = 2 * cg.m[1];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < Mc; i += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % cg.m[0]);
        const int y = (int)((i / cg.m[0]) % cg.m[1]);
        const int z = (int)(i / ((size_t)cg.m[0] * cg.m[1]));
        float s = 0.0f;
#pragma unroll
        for (int c = 0; c < (1 << D); ++c) {
            const int fx = 2 * x + (c & 1), fy = 2 * y + ((c >> 1) & 1), fz = D == 3 ? 2 * z + ((c >> 2) & 1) : 0;
            s += F[((size_t)fz * fm1 + fy) * fm0 + fx];
        }
        C[i] = s * (1.0f / (1 << D));
    }
}

// Fine velocity = coarse velocity interpolated (multilinear, zero outside the
// coarse grid) at the fine cell centres, per time node and component.
template <int D>
__global__ void prolong_velocity_kernel(const float* __restrict__ vc, float* __restrict__ vf, DevGrid cg, DevGrid fg,
                                        int blocks) {
    const size_t Mf = (size_t)fg.m[0] * fg.m[1] * fg.m[2];
    const size_t Mc = (size_t)cg.m[0] * cg.m[1] * cg.m[2];
    const size_t total = Mf * blocks;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t s = i % Mf;
        const size_t b = i / Mf;
        const int fi[3] = {(int)(s % fg.m[0]), (int)((s / fg.m[0]) % fg.m[1]), (int)(s / ((size_t)fg.m[0] * fg.m[1]))};
        int c0[3];
        float fr[3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const float x = fg.lo[a] + ((float)fi[a] + 0.5f) * fg.h[a];
            const float xi = (x - cg.lo[a]) * cg.inv_h[a] - 0.5f;
            const float fl = floorf(xi);
            c0[a] = (int)fl;
            fr[a] = xi - fl;
        }
        const float* src = vc + b * Mc;
        float acc = 0.0f;
#pragma unroll
        for (int c = 0; c < (1 << D); ++c) {
            float w = 1.0f;
            int idx[3] = {0, 0, 0};
            bool in = true;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const int bit = (c >> a) & 1;
                idx[a] = c0[a] + bit;
                w *= bit ? fr[a] : 1.0f - fr[a];
                in = in && idx[a] >= 0 && idx[a] < cg.m[a];
            }
            if (in) acc = fmaf(w, src[((size_t)idx[2] * cg.m[1] + idx[1]) * cg.m[0] + idx[0]], acc);
        }
        vf[b * Mf + s] = acc;
    }
}

// ------------------------------------------------- Jacobian determinant --

__device__ __forceinline__ void block_minmax(double& lo, double& hi) {
    __shared__ double slo[kBlock / 32], shi[kBlock / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_down_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_down_sync(0xffffffffu, hi, o));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        slo[warp] = lo;
        shi[warp] = hi;
    }
    __syncthreads();
    if (warp == 0) {
        lo = lane < kBlock / 32 ? slo[lane] : INFINITY;
        hi = lane < kBlock / 32 ? shi[lane] : -INFINITY;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fmin(lo, __shfl_down_sync(0xffffffffu, lo, o));
            hi = fmax(hi, __shfl_down_sync(0xffffffffu, hi, o));
        }
    }
}

// det grad y at the cell centres from the end points y [d][M]: central
// differences inside, one-sided at the ends; block min/max into partials.
template <int D>
__global__ void jacobian_det_kernel(const float* __restrict__ y, float* det, DevGrid g, double* pmin, double* pmax) {
    const size_t M = (size_t)g.m[0] * g.m[1] * g.m[2];
    const size_t stride[3] = {1, (size_t)g.m[0], (size_t)g.m[0] * g.m[1]};
    double lo = INFINITY, hi = -INFINITY;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < M; i += (size_t)gridDim.x * blockDim.x) {
        const int c[3] = {(int)(i % g.m[0]), (int)((i / g.m[0]) % g.m[1]), (int)(i / ((size_t)g.m[0] * g.m[1]))};
        double J[3][3];
#pragma unroll
        for (int b = 0; b < D; ++b) {
            const size_t up = c[b] < g.m[b] - 1 ? i + stride[b] : i;
            const size_t dn = c[b] > 0 ? i - stride[b] : i;
            const double span = (double)g.h[b] * (double)((up != i) + (dn != i));
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const float* ya = y + (size_t)a * M;
                J[a][b] = span > 0.0 ? ((double)ya[up] - (double)ya[dn]) / span : (a == b ? 1.0 : 0.0);
            }
        }
        double dt;
        if (D == 2) dt = J[0][0] * J[1][1] - J[0][1] * J[1][0];
        else
            dt = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) - J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                 J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
        if (det != nullptr) det[i] = (float)dt;
        lo = fmin(lo, dt);
        hi = fmax(hi, dt);
    }
    block_minmax(lo, hi);
    if (threadIdx.x == 0) {
        pmin[blockIdx.x] = lo;
        pmax[blockIdx.x] = hi;
    }
}

__global__ void minmax_final_kernel(const double* pmin, const double* pmax, int count, double* out) {
    double lo = INFINITY, hi = -INFINITY;
    for (int i = threadIdx.x; i < count; i += blockDim.x) {
        lo = fmin(lo, pmin[i]);
        hi = fmax(hi, pmax[i]);
    }
    block_minmax(lo, hi);
    if (threadIdx.x == 0) {
        out[0] = lo;
        out[1] = hi;
    }
}

inline int grid_for(size_t count) {
    const size_t b = (count + kBlock - 1) / kBlock;
    return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

}  // namespace

cudaError_t launch_pack(int d, PackArgs a, cudaStream_t s) {
    if (a.nz > a.tab.n || (a.v[0] == nullptr && a.v[1] != nullptr)) return cudaErrorInvalidValue;
    const size_t vn = (size_t)a.vg.mp[0] * a.vg.mp[1] * a.vg.mp[2] * a.tab.n;
    const size_t in = (size_t)a.ig.mp[0] * a.ig.mp[1] * a.ig.mp[2];
    for (int k = 0; k < 2; ++k) a.blocks[k] = a.v[k] != nullptr ? grid_for(vn) : 0;
    a.blocks[2] = a.image != nullptr ? grid_for(in) : 0;
    a.blocks[3] = a.zero != nullptr ? grid_for(in) : 0;
    if (a.many != nullptr && a.v[0] == nullptr) return cudaErrorInvalidValue;
    const int blocks = a.blocks[0] + a.blocks[1] + a.blocks[2] + a.blocks[3] + (a.many != nullptr ? 1 : 0);
    if (blocks == 0) return cudaSuccess;
    if (d == 3) pack_kernel<3><<<blocks, kBlock, 0, s>>>(a);
    else pack_kernel<2><<<blocks, kBlock, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_distribute_gradient(int d, const void* Gp, float* out, const DevGrid& g, int K,
                                       const SliceTable& t, float scale, cudaStream_t s) {
    const size_t total = (size_t)g.m[0] * g.m[1] * g.m[2] * K;
    if (d == 3) distribute_gradient_kernel<3><<<grid_for(total), kBlock, 0, s>>>((const float*)Gp, out, g, K, t, scale);
    else distribute_gradient_kernel<2><<<grid_for(total), kBlock, 0, s>>>((const float*)Gp, out, g, K, t, scale);
    return cudaGetLastError();
}

void make_node_table(int K, SliceTable* t) {
    t->n = K;
    for (int m = 0; m < K; ++m) {
        t->j[m] = m;
        t->th[m] = 0.0f;
    }
}

void make_slice_table(int K, int N, double t0, double dt, SliceTable* t) {
    if (K <= 1) {
        t->n = 1;
        t->j[0] = 0;
        t->th[0] = 0.0f;
        return;
    }
    t->n = 2 * N + 1;
    for (int m = 0; m < t->n; ++m) {
        double tm = t0 + m * 0.5 * dt;
        tm = tm < 0.0 ? 0.0 : (tm > 1.0 ? 1.0 : tm);
        const double sv = tm * (K - 1);
        int j = (int)std::floor(sv);
        if (j > K - 2) j = K - 2;
        t->j[m] = j;
        t->th[m] = (float)(sv - j);
    }
}

cudaError_t launch_unpack_image(const float* acc, float* out, const DevGrid& g, int d, cudaStream_t s) {
    const size_t M = (size_t)g.m[0] * g.m[1] * g.m[2];
    unpack_image_kernel<<<grid_for(M), kBlock, 0, s>>>(acc, out, g, d);
    return cudaGetLastError();
}

cudaError_t launch_repad_image(float* acc, const DevGrid& g, int d, float scale, cudaStream_t s) {
    const size_t total = (size_t)g.mp[0] * g.mp[1] * g.mp[2];
    repad_image_kernel<<<grid_for(total), kBlock, 0, s>>>(acc, g, d, scale);
    return cudaGetLastError();
}

// Blocks of the grid-stride reductions: four per SM of the current device
// (the SM count is read once per device ordinal).
int reduce_block_cap() {
    static int cap[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 4 * 152;
    }
    if (cap[dev] == 0) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
            cudaGetLastError();
            sms = 152;
        }
        cap[dev] = 4 * sms;
    }
    return cap[dev];
}

int residual_blocks(const DevGrid& g, int d) {
    (void)d;
    const size_t M = (size_t)g.m[0] * g.m[1] * g.m[2];
    const int b = nblocks_for(M);
    const int cap = reduce_block_cap();
    return b < cap ? b : cap;
}

cudaError_t launch_residual(const float* u1, const float* R, float* rp, const DevGrid& g, int d, float scale,
                            double* partial, int nblocks, cudaStream_t s) {
    residual_kernel<<<nblocks, kBlock, 0, s>>>(u1, R, rp, g, d, scale, partial);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const double* partial, int count, double* out, cudaStream_t s) {
    reduce_kernel<<<1, kReduceBlock, 0, s>>>(partial, count, out);
    return cudaGetLastError();
}

int dot_blocks(size_t count) {
    const int b = nblocks_for(count);
    const int cap = reduce_block_cap();
    return b < cap ? (b > 0 ? b : 1) : cap;
}

cudaError_t launch_dot_fused(const float* a, const float* b, const float* c, size_t count, double* partial,
                             int nblocks, unsigned* counter, double* sc, int slot_b, int slot_c, int mode, float* f,
                             cudaStream_t s, int* ctl, cudaGraphConditionalHandle handle) {
    // two blocks an SM at most: 11.3 us for 64^3 x 3 values, 12.9 with one, 11.6 with four
    const int blocks = nblocks < reduce_block_cap() / 2 ? nblocks : reduce_block_cap() / 2;
    dot_fused_kernel<<<blocks, kBlock, 0, s>>>(a, b, c, count, partial, counter, sc, slot_b, slot_c, mode, f, ctl,
                                                  handle);
    return cudaGetLastError();
}

cudaError_t launch_hess_finish(int d, const void* Gp, const float* p, float* Hp, const DevGrid& g, int K,
                               const SliceTable& t, float gscale, float rscale, float gamma, double* partial,
                               int nblocks, unsigned* counter, double* sc, float* f, cudaStream_t s) {
    // without partial: the product only, on a grid sized for the vector
    if (partial == nullptr) nblocks = grid_for((size_t)g.m[0] * g.m[1] * g.m[2] * K);
    if (d == 3) {
        if (partial) hess_finish_kernel<3, true><<<nblocks, kBlock, 0, s>>>((const float*)Gp, p, Hp, g, K, t, gscale,
                                                                             rscale, gamma, partial, counter, sc, f);
        else hess_finish_kernel<3, false><<<nblocks, kBlock, 0, s>>>((const float*)Gp, p, Hp, g, K, t, gscale, rscale,
                                                                     gamma, partial, counter, sc, f);
    } else {
        if (partial) hess_finish_kernel<2, true><<<nblocks, kBlock, 0, s>>>((const float*)Gp, p, Hp, g, K, t, gscale,
                                                                             rscale, gamma, partial, counter, sc, f);
        else hess_finish_kernel<2, false><<<nblocks, kBlock, 0, s>>>((const float*)Gp, p, Hp, g, K, t, gscale, rscale,
                                                                     gamma, partial, counter, sc, f);
    }
    return cudaGetLastError();
}

cudaError_t launch_pcg_update_xr(float* x, const float* p, float* r, const float* Hp, const float* f, size_t count,
                                 cudaStream_t s) {
    pcg_update_xr_kernel<<<grid_for(count), kBlock, 0, s>>>(x, p, r, Hp, f, count);
    return cudaGetLastError();
}

cudaError_t launch_pcg_curvature_fix(float* x, const float* z, const int* ctl, size_t count, cudaStream_t s) {
    const size_t want = (count + kBlock - 1) / kBlock;
    const int cap = reduce_block_cap();
    const int blocks = (int)(want < (size_t)cap ? (want > 0 ? want : 1) : (size_t)cap);
    pcg_curvature_fix_kernel<<<blocks, kBlock, 0, s>>>(x, z, ctl, count);
    return cudaGetLastError();
}

cudaError_t launch_axpby_dev(float a, const float* ap, const float* x, float b, const float* bp, float* y,
                             size_t count, cudaStream_t s) {
    axpby_dev_kernel<<<grid_for(count), kBlock, 0, s>>>(a, ap, x, b, bp, y, count);
    return cudaGetLastError();
}

cudaError_t launch_dot(const float* a, const float* b, size_t count, double* partial, int nblocks, cudaStream_t s) {
    dot_kernel<<<nblocks, kBlock, 0, s>>>(a, b, count, partial);
    return cudaGetLastError();
}

cudaError_t launch_laplacian(int d, const float* x, float* out, const DevGrid& g, int blocks_kd, float scale,
                             float gamma, const float* addsrc, cudaStream_t s) {
    return launch_laplacian_ext(d, x, out, g, blocks_kd, scale, gamma, gamma != 0.0f ? x : nullptr, addsrc, s);
}

cudaError_t launch_laplacian_ext(int d, const float* x, float* out, const DevGrid& g, int blocks_kd, float scale,
                                 float gamma, const float* gsrc, const float* addsrc, cudaStream_t s) {
    const size_t total = (size_t)g.m[0] * g.m[1] * g.m[2] * blocks_kd;
    const int grid = grid_for(total);
    if (d == 3) laplacian_kernel<3><<<grid, kBlock, 0, s>>>(x, out, g, blocks_kd, scale, gamma, gsrc, addsrc);
    else laplacian_kernel<2><<<grid, kBlock, 0, s>>>(x, out, g, blocks_kd, scale, gamma, gsrc, addsrc);
    return cudaGetLastError();
}

cudaError_t launch_divergence(int d, const float* x, float* div, const DevGrid& g, int K, cudaStream_t s) {
    const size_t total = (size_t)g.m[0] * g.m[1] * g.m[2] * K;
    if (d == 3) divergence_kernel<3><<<grid_for(total), kBlock, 0, s>>>(x, div, g, K);
    else divergence_kernel<2><<<grid_for(total), kBlock, 0, s>>>(x, div, g, K);
    return cudaGetLastError();
}

cudaError_t launch_elastic(int d, const float* x, const float* div, float* out, const DevGrid& g, int K,
                           float smu, float slm, float gamma, const float* addsrc, cudaStream_t s) {
    const size_t total = (size_t)g.m[0] * g.m[1] * g.m[2] * K * d;
    if (d == 3) elastic_kernel<3><<<grid_for(total), kBlock, 0, s>>>(x, div, out, g, K, smu, slm, gamma, addsrc);
    else elastic_kernel<2><<<grid_for(total), kBlock, 0, s>>>(x, div, out, g, K, smu, slm, gamma, addsrc);
    return cudaGetLastError();
}

// Raises the dynamic shared-memory limit of a kernel, once per device.
template <class K>
static cudaError_t raise_smem(K kernel, size_t bytes, bool (&done)[64]) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (done[dev]) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

cudaError_t launch_dct_axis(const float* in, float* out, const float* C, const DevGrid& g, int nblocks_kd, int axis,
                            bool inverse, cudaStream_t s) {
    const size_t total = (size_t)g.m[0] * g.m[1] * g.m[2] * nblocks_kd;
    const int m = g.m[axis];
    if (m > kDctTileMax) {
        dct_axis_kernel<<<grid_for(total), kBlock, 0, s>>>(in, out, C, g, nblocks_kd, axis, inverse ? 1 : 0);
        return cudaGetLastError();
    }
    const long long inner = axis == 0 ? 1 : (axis == 1 ? (long long)g.m[0] : (long long)g.m[0] * g.m[1]);
    const long long outer = (long long)(total / ((size_t)m * inner));
    // inner = 1: every (y, z, block) is one line
    const long long blocks =
        axis == 0 ? (outer + kDctLines - 1) / kDctLines : (inner + kDctLines - 1) / kDctLines * outer;
    const int vec_in = (inner % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0) ? 1 : 0;
    static bool done[2][64] = {};
    auto run = [&](auto kernel, long long lines, bool (&d)[64]) -> cudaError_t {
        const cudaError_t e = raise_smem(kernel, dct_tile_smem(kDctTileMax), d);
        if (e != cudaSuccess) return e;
        kernel<<<(unsigned)blocks, kBlock, dct_tile_smem(m), s>>>(in, out, dct_table(C, m), inverse, inner, lines,
                                                                  vec_in);
        return cudaGetLastError();
    };
    if (axis == 0) return run(dct_tile_kernel<true>, outer, done[0]);
    return run(dct_tile_kernel<false>, inner * m * outer, done[1]);
}

bool dct_table_ok(int m) { return m <= kDctTileMax; }

size_t dct_table_floats(int m) { return (size_t)2 * dct_table(nullptr, m).h * dct_table(nullptr, m).stride; }

void dct_tables(const float* C, int m, float* f, float* i) {
    const DctTable t = dct_table(nullptr, m);
    for (size_t e = 0; e < dct_table_floats(m); ++e) f[e] = i[e] = 0.0f;
    for (int r = 0; r < m; ++r)
        for (int j = 0; j < t.h; ++j) {
            float* fr = f + (size_t)r * t.stride + j;
            fr[0] = C[(size_t)(2 * j) * m + r];
            if (2 * j + 1 < m) fr[t.P4] = C[(size_t)(2 * j + 1) * m + r];
            float* ir = i + (size_t)r * t.P4 + j;
            ir[0] = C[(size_t)r * m + j];
            ir[t.h * t.stride] = C[(size_t)r * m + m - 1 - j];
        }
}

bool dct_plane_ok(int mx, int my, bool full) {
    const int most = full ? kDctFullPlaneMax : kDctPlaneMax;
    return mx <= most && my <= most;
}

template <int LT, bool FULL>
static cudaError_t run_plane(const float* in, float* out, const float* Tx, const float* Ty, bool inverse, int mx,
                             int my, long long planes, cudaStream_t s) {
    constexpr int most = FULL ? kDctFullPlaneMax : kDctPlaneMax;
    static bool done[64] = {};
    const cudaError_t e = raise_smem(dct_plane_kernel<LT, FULL>, dct_plane_smem<FULL>(most, most, 1), done);
    if (e != cudaSuccess) return e;
    const int vec_in = (mx % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0) ? 1 : 0;
    const int vec_out = (mx % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0) ? 1 : 0;
    dct_plane_kernel<LT, FULL><<<(unsigned)planes, dct_threads(dct_plane_threads(mx, my, LT), planes),
                                 dct_plane_smem<FULL>(mx, my, 1), s>>>(in, out, dct_table(Tx, mx), dct_table(Ty, my),
                                                                       inverse, mx, my, vec_in, vec_out);
    return cudaGetLastError();
}

cudaError_t launch_dct_plane(const float* in, float* out, const float* Tx, const float* Ty, bool inverse, bool full,
                             const DevGrid& g, long long planes, cudaStream_t s) {
    const int mx = g.m[0], my = g.m[1];
    if (!dct_plane_ok(mx, my, full) || planes < 1 || planes > 0x7fffffffLL) return cudaErrorNotSupported;
    if (dct_plane_split(mx, my))
        return full ? run_plane<4, true>(in, out, Tx, Ty, inverse, mx, my, planes, s)
                    : run_plane<4, false>(in, out, Tx, Ty, inverse, mx, my, planes, s);
    return full ? run_plane<8, true>(in, out, Tx, Ty, inverse, mx, my, planes, s)
                : run_plane<8, false>(in, out, Tx, Ty, inverse, mx, my, planes, s);
}

template <int LT>
static cudaError_t run_plane2d(const float* in, float* out, const float* Fx, const float* Fy, const float* Ix,
                               const float* Iy, const float* inv_eig, int mx, int my, int blocks, cudaStream_t s) {
    static bool done[64] = {};
    const cudaError_t e =
        raise_smem(dct_plane2d_kernel<LT>, dct_plane_smem<false>(kDctPlaneMax, kDctPlaneMax, 2), done);
    if (e != cudaSuccess) return e;
    const int vec_in = (mx % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0) ? 1 : 0;
    const int vec_out = (mx % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0) ? 1 : 0;
    dct_plane2d_kernel<LT><<<blocks, kBlock, dct_plane_smem<false>(mx, my, 2), s>>>(
        in, out, dct_table(Fx, mx), dct_table(Fy, my), dct_table(Ix, mx), dct_table(Iy, my), inv_eig, mx, my, vec_in,
        vec_out);
    return cudaGetLastError();
}

cudaError_t launch_dct_plane2d(const float* in, float* out, const float* Fx, const float* Fy, const float* Ix,
                               const float* Iy, const float* inv_eig, const DevGrid& g, int blocks, cudaStream_t s) {
    const int mx = g.m[0], my = g.m[1];
    if (!dct_plane_ok(mx, my, false) || blocks < 1) return cudaErrorNotSupported;
    return dct_plane_split(mx, my) ? run_plane2d<4>(in, out, Fx, Fy, Ix, Iy, inv_eig, mx, my, blocks, s)
                                   : run_plane2d<8>(in, out, Fx, Fy, Ix, Iy, inv_eig, mx, my, blocks, s);
}

template <int LINES, bool SPLIT, bool FULL>
static cudaError_t run_last(const float* in, float* out, const float* Tf, const float* Ti, const float* inv_eig, int m,
                            long long inner, int nblocks_kd, long long blocks, cudaStream_t s) {
    const auto bytes = [](int n) { return (2 * staged_floats<FULL>(n) + (size_t)n * (LINES + 4)) * sizeof(float); };
    static bool done[64] = {};
    const cudaError_t e = raise_smem(dct_last_half_kernel<LINES, SPLIT, FULL>, bytes(kDctTileMax), done);
    if (e != cudaSuccess) return e;
    const int groups = ((m + 1) / 2 + 3) / 4;
    const int vec_in = (inner % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0) ? 1 : 0;
    const dim3 grid((unsigned)((inner + LINES - 1) / LINES), (unsigned)nblocks_kd);
    const int threads = dct_threads((SPLIT ? 2 : 1) * groups * (LINES / 4), blocks);
    dct_last_half_kernel<LINES, SPLIT, FULL><<<grid, threads, bytes(m), s>>>(
        in, out, dct_table(Tf, m), dct_table(Ti, m), inv_eig, m, inner, vec_in);
    return cudaGetLastError();
}

cudaError_t launch_dct_last(const float* in, float* out, const float* Tf, const float* Ti, const float* inv_eig,
                            bool full, const DevGrid& g, int d, int nblocks_kd, cudaStream_t s) {
    const int m = g.m[d - 1];
    const long long inner = d == 2 ? (long long)g.m[0] : (long long)g.m[0] * g.m[1];
    if (m > kDctTileMax || nblocks_kd > 65535) return cudaErrorNotSupported;
    const long long blocks = (inner + kDctFusedLines - 1) / kDctFusedLines * nblocks_kd;
    const int groups = ((m + 1) / 2 + 3) / 4;
    if (blocks < reduce_block_cap() / 4)
        return full ? run_last<32, true, true>(in, out, Tf, Ti, inv_eig, m, inner, nblocks_kd, blocks, s)
                    : run_last<32, true, false>(in, out, Tf, Ti, inv_eig, m, inner, nblocks_kd, blocks, s);
    if (2 * groups * (kDctFusedLines / 4) <= kBlock)
        return full ? run_last<64, true, true>(in, out, Tf, Ti, inv_eig, m, inner, nblocks_kd, blocks, s)
                    : run_last<64, true, false>(in, out, Tf, Ti, inv_eig, m, inner, nblocks_kd, blocks, s);
    return full ? run_last<64, false, true>(in, out, Tf, Ti, inv_eig, m, inner, nblocks_kd, blocks, s)
                : run_last<64, false, false>(in, out, Tf, Ti, inv_eig, m, inner, nblocks_kd, blocks, s);
}

cudaError_t launch_scale_modes(float* x, const float* inv_eig, size_t block_elems, size_t count, cudaStream_t s) {
    scale_modes_kernel<<<grid_for(count), kBlock, 0, s>>>(x, inv_eig, block_elems, count);
    return cudaGetLastError();
}

cudaError_t launch_add_scaled(float* out, const float* x, float ax, const float* y, float ay, size_t count,
                              cudaStream_t s) {
    add_scaled_kernel<<<grid_for(count), kBlock, 0, s>>>(out, x, ax, y, ay, count);
    return cudaGetLastError();
}

cudaError_t launch_restrict_image(int d, const float* F, float* C, const DevGrid& cg, cudaStream_t s) {
    const size_t Mc = (size_t)cg.m[0] * cg.m[1] * cg.m[2];
    if (d == 3) restrict_image_kernel<3><<<grid_for(Mc), kBlock, 0, s>>>(F, C, cg);
    else restrict_image_kernel<2><<<grid_for(Mc), kBlock, 0, s>>>(F, C, cg);
    return cudaGetLastError();
}

cudaError_t launch_prolong_velocity(int d, const float* vc, float* vf, const DevGrid& cg, const DevGrid& fg,
                                    int blocks, cudaStream_t s) {
    const size_t total = (size_t)fg.m[0] * fg.m[1] * fg.m[2] * blocks;
    if (d == 3) prolong_velocity_kernel<3><<<grid_for(total), kBlock, 0, s>>>(vc, vf, cg, fg, blocks);
    else prolong_velocity_kernel<2><<<grid_for(total), kBlock, 0, s>>>(vc, vf, cg, fg, blocks);
    return cudaGetLastError();
}

cudaError_t launch_jacobian_det(int d, const float* y, float* det, const DevGrid& g, double* partial, double* out,
                                cudaStream_t s) {
    const size_t M = (size_t)g.m[0] * g.m[1] * g.m[2];
    const int nb = residual_blocks(g, d);
    double* pmin = partial;
    double* pmax = partial + nb;
    if (d == 3) jacobian_det_kernel<3><<<nb, kBlock, 0, s>>>(y, det, g, pmin, pmax);
    else jacobian_det_kernel<2><<<nb, kBlock, 0, s>>>(y, det, g, pmin, pmax);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    (void)M;
    minmax_final_kernel<<<1, kBlock, 0, s>>>(pmin, pmax, nb, out);
    return cudaGetLastError();
}
