// Tensor-core convolutions of the warm-start network: every 3x3 convolution
// and both of its gradients as an implicit GEMM on the 5th-generation tensor
// cores (tcgen05.mma, kind::f16: bf16 operands, FP32 accumulation in tensor
// memory), with the operands brought to shared memory by TMA.
//
//   forward       D[pixel][co]       = sum_(tap,ci) x_eff[pixel + tap][ci] W[co][ci][tap]
//   data gradient D[in pixel][ci]    = sum_(tap,up,co) dz[pixel - tap][co] W[co][ci][tap]
//   weight grad.  D[(tap,ci)][co]    = sum_pixel x_eff[pixel + tap][ci] dz[pixel][co]
//
// The network's FP32 activations and gradients enter as sums of three bf16
// planes, x = hi + mid + lo with hi = bf16(x), mid = bf16(x - hi), lo =
// bf16(x - hi - mid) (exact: each difference is exact in FP32 and has at most
// 16, then 8 significant bits), so the products the tensor cores form are the
// exact products of the FP32 values with the bf16 weights, accumulated in
// FP32: the arithmetic of the network as specified (bf16 weights, FP32
// activations and accumulation), not a bf16 approximation of it.  The weight
// gradient multiplies two FP32 operands; the six plane products whose
// exponents reach 2^-16 of the leading one are formed (the three dropped
// ones are below FP32 resolution).
//
// Operands.  The planes of a tensor are one NHWC array [3][B][h][h][cp] (cp:
// channels padded to a multiple of 16), described to TMA as a 5D tensor.  A
// box of spatial positions x `kb` channels x 3 planes of it is a whole operand
// tile in the tensor cores' swizzled layout: a row of shared memory is one
// pixel's channels.  A convolution's tap is a shift of the box (zero fill
// outside the image is the padding), a stride of two is a traversal stride of
// the tensor map, and what has no such form is cut into the four parities of
// the finer grid (`phases`): an upsampled input, and the data gradient of a
// stride-2 layer, whose pixels of one parity meet the same subset of the taps.
// The forward and data-gradient GEMMs read the tile K-major (K = channels of
// one tap), the weight gradient MN-major (K = pixels).
//
// A CTA is persistent (one per SM) and has a TMA warp, an MMA warp and four
// epilogue warps.  Tiles of 128 rows x bn columns (x a slice of K) are handed
// out in turn; operand stages form a ring with full / empty mbarriers, and two
// accumulators in tensor memory let the epilogue of one tile run under the
// MMAs of the next.  K runs in the order (tap, channel), 16 at a time with the
// plane products innermost, in one accumulator.
//
// The per-thread gather this replaces (cp.async of 16-byte chunks, one operand
// stage per CTA) waited on its copies: 0.40 ms for the 128 -> 64 channel
// upsampled layer at batch 32 (tensor pipe 7% active), and the weight
// gradient, which split FP32 elements on the fly, 1.7 ms.
//
// Every mbarrier wait is bounded; a wait that runs out sets an error flag and
// a flag that ends the CTA's other roles.  The TMA and the MMA role always end with a
// bounded wait for their copies and MMAs in flight (mbar_drain), and only then the
// CTA frees the tensor memory.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace umma {

constexpr int BM = 128;
constexpr int BK = 64;                      // K per chunk (the unit of the K split)
constexpr int kThreads = 192;               // TMA warp, MMA warp, four epilogue warps
constexpr int kMaxStages = 6;
constexpr long kWaitLimit = 1L << 22;       // mbarrier polls before giving up

enum Kind { FWD = 0, BWD_DATA = 1, BWD_WEIGHT = 2 };

struct ConvGemm {
    int kind;
    int ci, co, stride, up, hin, hout, batch;   // the layer and the batch
    int cp;                   // channels of the A planes (padded): FWD and BWD_WEIGHT the input's, BWD_DATA dz's
    int kb;                   // channels per row of the A tile (64, 32 or 16: its swizzle)
    int kz;                   // BWD_WEIGHT: the same for the dz tile
    int N;                    // columns of D
    int bn;                   // columns per tile: a multiple of 16, <= 256 (<= 128 for BWD_WEIGHT)
    int ntn;                  // column tiles
    int grid;                 // side of the grid of positions that is tiled
    int phases;               // 1, or 4 parities of the finer grid
    int bx, by, bb;           // box of positions (powers of two): 128, or 64 for BWD_WEIGHT (its K chunk)
    int tx, ty, tb;           // boxes per axis
    int mtiles;               // BWD_WEIGHT: tiles of 128 rows (tap, ci); else unused
    int chunks, chunks_per_split, splits;   // K chunks, and how they are split over tiles
    int items;                // tiles in all
    int stages, stage_bytes, a_bytes;
    int ncols;                // tensor-memory columns of one accumulator
    long long M;              // FWD, BWD_DATA: rows of D (pixels of the batch)
    float* part;              // FWD, BWD_DATA with splits > 1: raw partial tiles [split][N][M], finished by
                              // finish_split_kernel; BWD_WEIGHT: [split][co][9 cp]
    float* out;               // FWD: layer output (may be NULL); BWD_DATA: input gradient
    __nv_bfloat16* nplanes;   // FWD: the output's planes, the next layer's input (may be NULL)
    int ncp;                  // their channels (co padded to 16)
    float* r;                 // FWD: activation before the skip add (may be NULL)
    const float* add;         // FWD: skip tensor (may be NULL)
    const float* bias;        // FWD
    int relu;
    float scale;
    int accumulate;           // BWD_DATA: out += instead of out =
    int *err, *herr;          // give_up when a wait runs out
};

// A wait ran out: err (device memory) keeps the weights from being updated with what is
// unfinished, herr (pinned host memory) is what the network's next call reports.
__device__ __forceinline__ void give_up(int* err, int* herr) {
    atomicExch(err, 1);
    *reinterpret_cast<volatile int*>(herr) = 1;
}

// Every kernel of a network pass is launched as a programmatic dependent of the
// one before it: it may start (barriers, tensor memory, constants) while that
// one still runs, and touches global memory only after dependency_wait(), which
// returns when that kernel (which waited the same way) has completed.
//
// A kernel that allocates tensor memory triggers after the allocation, past the
// barrier that publishes its address.  tcgen05.alloc waits without a bound until the
// columns are free; a dependent that took them first would hold them in its
// dependency_wait(), for the very kernel that waits for the columns.  Since a
// dependent starts only when every CTA before it has triggered, every holder of
// columns waits for kernels that have theirs, so each allocation ends.
__device__ __forceinline__ void dependency_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads of global memory in these kernels.  A kernel may be resident while an earlier
// one (or the caller's own kernel before the pass) still writes what it reads, so its data is
// not read-only for the kernel's lifetime, which is what the non-coherent path (__ldg,
// const __restrict__) asks for: plain loads, volatile so that none moves above
// dependency_wait().
__device__ __forceinline__ float ld(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int ld(const int* p) {
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor.  kb = 64, 32, 16: a swizzled tile whose rows
// are 2 kb bytes (leading byte offset: MN blocks of an MN-major tile; stride byte
// offset: 8-row groups).  kb = 0: core matrices of 8 rows x 16 bytes without
// swizzle (K-major; leading byte offset: next along K, stride: next 8 rows).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo, int kb) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;   // descriptor version of this architecture
    d |= (uint64_t)(kb == 64 ? 2 : (kb == 32 ? 4 : (kb == 16 ? 6 : 0))) << 61;
    return d;
}

// Instruction descriptor of kind::f16: D FP32, A and B bf16, M x N; mn: both
// operands MN-major instead of K-major.
__device__ __forceinline__ uint32_t instr_desc(int M, int N, bool mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for the phase; false when the polls run out or another role gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* dead) {
    for (long i = 0; i < kWaitLimit; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 255) == 255 && *dead) return false;
    }
    *dead = 1;
    return false;
}

// Bounded wait that no other role's giving up cuts short: a role ends with it on the
// copies (MMAs) that it has issued, whichever role gave up, so that they land before
// the CTA frees its memory.  Without a give-up they have landed, or the epilogue waits for
// them anyway.
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity, volatile int* dead) {
    for (long i = 0; i < kWaitLimit; ++i)
        if (mbar_try(bar, parity)) return;
    *dead = 1;
}

__device__ __forceinline__ void tma_5d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int c, int x, int y,
                                       int b) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(dst),
        "l"(map), "r"(smem_u32(bar)), "r"(c), "r"(x), "r"(y), "r"(b), "r"(0)
        : "memory");
}

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int k, int row) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(map), "r"(smem_u32(bar)), "r"(k), "r"(row)
        : "memory");
}

// 16 columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_ld16(uint32_t (&v)[16], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(addr));
}

// x = hi + mid + lo exactly (see the file comment)
__device__ __forceinline__ void split3(float x, __nv_bfloat16& h, __nv_bfloat16& m, __nv_bfloat16& l) {
    h = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(h);
    m = __float2bfloat16_rn(r1);
    l = __float2bfloat16_rn(r1 - __bfloat162float(m));
}

// The planes of 8 channels of one pixel, at element e of planes of pe elements.
__device__ __forceinline__ void store_planes8(__nv_bfloat16* planes, size_t pe, size_t e, const float* v) {
    __align__(16) __nv_bfloat16 h[8], m[8], l[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) split3(v[j], h[j], m[j], l[j]);
    *reinterpret_cast<uint4*>(planes + e) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(planes + pe + e) = *reinterpret_cast<const uint4*>(m);
    *reinterpret_cast<uint4*>(planes + 2 * pe + e) = *reinterpret_cast<const uint4*>(l);
}

// One tile of work.  FWD, BWD_DATA: a box of 128 positions of one parity, a
// column tile and a slice of K.  BWD_WEIGHT: 128 rows (tap, ci), a column tile
// and a slice of the pixel chunks.
struct Item {
    int nt, sp, ph, x0, y0, b0, mt;
};

__device__ __forceinline__ void box_origin(const ConvGemm& g, int tile, int& x0, int& y0, int& b0) {
    x0 = (tile % g.tx) * g.bx;
    tile /= g.tx;
    y0 = (tile % g.ty) * g.by;
    b0 = (tile / g.ty) * g.bb;
}

__device__ __forceinline__ Item item_at(const ConvGemm& g, int i) {
    Item t;
    t.nt = i % g.ntn;
    i /= g.ntn;
    t.ph = t.x0 = t.y0 = t.b0 = t.mt = 0;
    if (g.kind == BWD_WEIGHT) {
        t.mt = i % g.mtiles;
        t.sp = i / g.mtiles;
        return t;
    }
    t.sp = i % g.splits;
    i /= g.splits;
    t.ph = i % g.phases;
    box_origin(g, i / g.phases, t.x0, t.y0, t.b0);
    return t;
}

// FWD, BWD_DATA: the K units (kb channels of one position pos: a tap, or a
// tap and an up position) of a tile's slice of K.
__device__ __forceinline__ void unit_range(const ConvGemm& g, int sp, int& u0, int& u1) {
    const int upc = BK / g.kb, npos = g.kind == BWD_DATA && g.up ? 36 : 9;
    u0 = sp * g.chunks_per_split * upc;
    u1 = min((sp + 1) * g.chunks_per_split * upc, npos * (g.cp / g.kb));
}

// Start of the source box along one axis for tap coordinate k (0..2), up
// position d, parity p and tile origin o; false when this parity does not
// meet the tap (stride-2 data gradient).
__device__ __forceinline__ bool axis_start(const ConvGemm& g, int o, int k, int d, int p, int& s) {
    if (g.kind == BWD_DATA) {
        if (g.up) {
            s = 2 * o + d + 1 - k;
        } else if (g.stride == 2) {
            if ((p + 1 - k) & 1) return false;
            s = o + (p + 1 - k) / 2;
        } else {
            s = o + 1 - k;
        }
    } else {
        s = g.up ? o + ((p + k - 1) >> 1) : g.stride * o + k - 1;
    }
    return true;
}

__device__ __forceinline__ bool unit_source(const ConvGemm& g, const Item& t, int u, int& c0, int& x, int& y) {
    const int upp = g.cp / g.kb, pos = u / upp;
    c0 = (u - pos * upp) * g.kb;
    const int R = g.kind == BWD_DATA && g.up ? 4 : 1, tap = pos / R, dd = pos - tap * R;
    const int ky = tap / 3, kx = tap - ky * 3;
    return axis_start(g, t.y0, ky, dd >> 1, t.ph >> 1, y) && axis_start(g, t.x0, kx, dd & 1, t.ph & 1, x);
}

__global__ void __launch_bounds__(kThreads, 1)
    conv_gemm_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
                     const ConvGemm g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], accf[2], acce[2];
    __shared__ uint32_t tmem_base;
    __shared__ int dead;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool bw = g.kind == BWD_WEIGHT;
    const uint32_t alloc_cols = 2u * (uint32_t)g.ncols;

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(alloc_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&amap) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&bmap) : "memory");
        dead = 0;
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&accf[s], 1);
            mbar_init(&acce[s], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    dependency_trigger();                 // the CTA has its tensor memory (see dependency_trigger)
    dependency_wait();
    const uint32_t tmem = tmem_base;
    const uint32_t smem0 = smem_u32(smem);
    const int S = g.stages;
    const uint32_t arow = 2u * (uint32_t)g.kb;                  // bytes of a row of the A tile
    const uint32_t zrow = 2u * (uint32_t)g.kz;                  // of the dz tile (BWD_WEIGHT)

    if (warp == 0) {
        // ---- TMA: one elected thread
        if (lane == 0) {
            int n = 0;                                          // stages filled so far
            bool ok = true;
            for (int it = blockIdx.x; ok && it < g.items; it += gridDim.x) {
                const Item t = item_at(g, it);
                if (!bw) {
                    int u0, u1;
                    unit_range(g, t.sp, u0, u1);
                    for (int u = u0; u < u1; ++u) {
                        int c0, x, y;
                        if (!unit_source(g, t, u, c0, x, y)) continue;
                        const int s = n % S;
                        if (n >= S && !(ok = mbar_wait(&empty[s], (uint32_t)((n / S - 1) & 1), &dead))) break;
                        const uint32_t sa = smem0 + (uint32_t)s * (uint32_t)g.stage_bytes;
                        mbar_expect(&full[s], 3u * BM * arow + (uint32_t)g.bn * arow);
                        tma_5d(sa, &amap, &full[s], c0, x, y, t.b0);
                        tma_2d(sa + (uint32_t)g.a_bytes, &bmap, &full[s], u * g.kb, t.nt * g.bn);
                        ++n;
                    }
                } else {
                    const int nblk = 9 * g.cp / g.kb, per = BM / g.kb, bpt = g.cp / g.kb;
                    const int b_lo = t.mt * per, b_hi = min(nblk, b_lo + per);
                    const int tiles = g.tx * g.ty * g.tb;
                    const int c_hi = min(g.chunks, (t.sp + 1) * g.chunks_per_split);
                    for (int c = t.sp * g.chunks_per_split; c < c_hi; ++c) {
                        const int ph = c / tiles;
                        int x0, y0, b0;
                        box_origin(g, c - ph * tiles, x0, y0, b0);
                        const int s = n % S;
                        if (n >= S && !(ok = mbar_wait(&empty[s], (uint32_t)((n / S - 1) & 1), &dead))) break;
                        const uint32_t sa = smem0 + (uint32_t)s * (uint32_t)g.stage_bytes;
                        const uint32_t ablk = 3u * BK * arow, zblk = 3u * BK * zrow;
                        mbar_expect(&full[s], (uint32_t)(b_hi - b_lo) * ablk + (uint32_t)(g.bn / g.kz) * zblk);
                        for (int b = b_lo; b < b_hi; ++b) {
                            const int tap = b / bpt, ky = tap / 3, kx = tap - ky * 3;
                            int x, y;
                            axis_start(g, y0, ky, 0, ph >> 1, y);
                            axis_start(g, x0, kx, 0, ph & 1, x);
                            tma_5d(sa + (uint32_t)(b - b_lo) * ablk, &amap, &full[s], (b - tap * bpt) * g.kb, x, y, b0);
                        }
                        for (int j = 0; j < g.bn / g.kz; ++j)
                            tma_5d(sa + (uint32_t)g.a_bytes + (uint32_t)j * zblk, &bmap, &full[s],
                                   t.nt * g.bn + j * g.kz, g.up ? 2 * x0 + (ph & 1) : x0,
                                   g.up ? 2 * y0 + (ph >> 1) : y0, b0);
                        ++n;
                    }
                }
            }
            for (int k = max(0, n - S); k < n; ++k) mbar_drain(&full[k % S], (uint32_t)((k / S) & 1), &dead);
        }
    } else if (warp == 1) {
        // ---- MMA: one elected thread
        if (lane == 0) {
            const uint32_t idesc = instr_desc(BM, g.bn, bw);
            // descriptors of a stage at address zero; planes are aplane (zplane) x 16 bytes apart
            const uint64_t adesc = bw ? smem_desc(0, 3u * BK * arow, 8 * arow, g.kb) : smem_desc(0, 16, 8 * arow, g.kb);
            const uint64_t bdesc =
                (bw ? smem_desc(0, 3u * BK * zrow, 8 * zrow, g.kz) : smem_desc(0, 16, 8 * arow, g.kb)) +
                ((uint32_t)g.a_bytes >> 4);
            const uint32_t aplane = (bw ? BK : BM) * arow / 16, zplane = BK * zrow / 16;
            const int nkk = g.kb / 16;
            int n = 0, a = 0;                                   // stages consumed, tiles begun
            bool ok = true;
            for (int it = blockIdx.x; ok && it < g.items; it += gridDim.x, ++a) {
                const Item t = item_at(g, it);
                const int ab = a & 1;
                if (a >= 2 && !(ok = mbar_wait(&acce[ab], (uint32_t)((a / 2 - 1) & 1), &dead))) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t d = tmem + (uint32_t)(ab * g.ncols);
                uint32_t issued = 0;
                int u0, u1;
                if (bw) {
                    u0 = t.sp * g.chunks_per_split;
                    u1 = min(g.chunks, u0 + g.chunks_per_split);
                } else {
                    unit_range(g, t.sp, u0, u1);
                }
                for (int u = u0; u < u1; ++u) {
                    int c0, x, y;
                    if (!bw && !unit_source(g, t, u, c0, x, y)) continue;
                    const int s = n % S;
                    if (!(ok = mbar_wait(&full[s], (uint32_t)((n / S) & 1), &dead))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    // descriptors differ by their start addresses (in 16 bytes) only
                    const uint32_t s4 = (smem0 + (uint32_t)s * (uint32_t)g.stage_bytes) >> 4;
                    const uint64_t ad = adesc + s4, bd = bdesc + s4;
                    if (!bw) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            if (kk < nkk) {
#pragma unroll
                                for (int p = 0; p < 3; ++p) {
                                    mma_bf16(d, ad + (uint32_t)p * aplane + 2 * kk, bd + 2 * kk, idesc, issued);
                                    issued = 1;
                                }
                            }
                        }
                    } else {
                        // 16 pixels at a time; plane pairs (dz, x) with pz + px <= 2
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
#pragma unroll
                            for (int pz = 0; pz < 3; ++pz) {
#pragma unroll
                                for (int px = 0; px + pz <= 2; ++px) {
                                    mma_bf16(d, ad + (uint32_t)px * aplane + kk * arow,
                                             bd + (uint32_t)pz * zplane + kk * zrow, idesc, issued);
                                    issued = 1;
                                }
                            }
                        }
                    }
                    mma_commit(&empty[s]);
                    ++n;
                }
                if (!ok) break;
                if (issued) mma_commit(&accf[ab]);
                else mbar_arrive(&accf[ab]);                    // an empty slice of K
            }
            if (n > 0) mbar_drain(&empty[(n - 1) % S], (uint32_t)(((n - 1) / S) & 1), &dead);
        }
    } else {
        // ---- epilogue: warp w reads the tensor-memory lanes 32 (w mod 4) ..
        const int quad = warp & 3, row = quad * 32 + lane;
        const int fine = g.phases == 4 && !bw ? 2 : 1;          // output positions per tiled position
        const int ho = g.kind == FWD ? g.hout : g.hin;          // side of the output
        int a = 0;
        bool ok = true;
        for (int it = blockIdx.x; ok && it < g.items; it += gridDim.x, ++a) {
            const Item t = item_at(g, it);
            const int ab = a & 1;
            ok = mbar_wait(&accf[ab], (uint32_t)((a / 2) & 1), &dead);
            if (__any_sync(0xffffffffu, !ok)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            bool empty_k = false;
            if (!bw && g.kind == BWD_DATA && g.splits > 1) {    // a slice whose taps this parity never meets
                int u0, u1, c0, x, y;
                unit_range(g, t.sp, u0, u1);
                empty_k = true;
                for (int u = u0; empty_k && u < u1; ++u) empty_k = !unit_source(g, t, u, c0, x, y);
            }
            // where this row goes
            bool valid;
            size_t P = (size_t)ho * ho, o = 0;
            int b = 0;
            if (bw) {
                o = (size_t)t.mt * BM + row;
                valid = o < (size_t)9 * g.cp;
            } else {
                const int px = t.x0 + row % g.bx, py = t.y0 + (row / g.bx) % g.by;
                b = t.b0 + row / (g.bx * g.by);
                valid = px < g.grid && py < g.grid && b < g.batch;
                o = (size_t)(py * fine + (fine == 2 ? t.ph >> 1 : 0)) * ho + px * fine + (fine == 2 ? t.ph & 1 : 0);
            }
            for (int c0 = 0; c0 < g.bn; c0 += 16) {
                uint32_t v[16];
                const uint32_t ta = tmem + (uint32_t)(ab * g.ncols) + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
                tmem_ld16(v, ta);
                asm volatile("tcgen05.wait::ld.sync.aligned;");
                if (!valid) continue;
                const int n0 = t.nt * g.bn + c0;
                if (bw || g.splits > 1) {
                    const size_t rows = bw ? (size_t)9 * g.cp : (size_t)g.M;
                    float* p = g.part + ((size_t)t.sp * g.N + n0) * rows + (bw ? o : (size_t)b * P + o);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (n0 + j < g.N) p[j * rows] = empty_k ? 0.0f : __uint_as_float(v[j]);
                } else if (g.kind == FWD) {
                    // the loads of a group of columns are all in flight before its stores
                    float z[16];
                    const size_t oi = ((size_t)b * g.co + n0) * P + o;
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        z[j] = g.add != nullptr && n0 + j < g.N ? ld(g.add + oi + j * P) : 0.0f;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const bool in = n0 + j < g.N;
                        float t1 = __uint_as_float(v[j]) + (in ? ld(g.bias + n0 + j) : 0.0f);
                        if (g.relu) t1 = fmaxf(t1, 0.0f);
                        if (g.r != nullptr && in) g.r[oi + j * P] = t1;
                        if (g.add != nullptr) t1 += z[j];
                        z[j] = in ? g.scale * t1 : 0.0f;
                        if (g.out != nullptr && in) g.out[oi + j * P] = z[j];
                    }
                    if (g.nplanes != nullptr && n0 < g.ncp) {
                        const size_t pe = (size_t)g.batch * P * g.ncp, e = ((size_t)b * P + o) * g.ncp + n0;
                        store_planes8(g.nplanes, pe, e, z);
                        store_planes8(g.nplanes, pe, e + 8, z + 8);
                    }
                } else {
                    float* p = g.out + ((size_t)b * g.ci + n0) * P + o;
                    float z[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) z[j] = g.accumulate && n0 + j < g.N ? ld(p + j * P) : 0.0f;
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (n0 + j < g.N) p[j * P] = z[j] + __uint_as_float(v[j]);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce[ab]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (tid == 0 && dead) give_up(g.err, g.herr);
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(alloc_cols));
}

// The end of a split-K FWD or BWD_DATA GEMM: the partial tiles summed over the
// splits in increasing order (deterministic), then the epilogue of the unsplit
// kernel.  One thread per 8 columns of a row, rows fastest.
__global__ void finish_split_kernel(const ConvGemm g, int splits) {
    const size_t M = (size_t)g.M, total = M * ((g.N + 7) / 8);
    const int h = g.kind == FWD ? g.hout : g.hin, C = g.kind == FWD ? g.co : g.ci;
    const size_t P = (size_t)h * h;
    dependency_trigger();
    dependency_wait();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int n0 = (int)(i / M) * 8;
        const size_t row = i - (size_t)(n0 / 8) * M, b = row / P, o = row - b * P;
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = 0.0f;
#pragma unroll 4
        for (int z = 0; z < splits; ++z) {
            const float* p = g.part + ((size_t)z * g.N + n0) * M + row;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (n0 + j < g.N) acc[j] += ld(p + j * M);
        }
        const size_t oi = (b * C + n0) * P + o;
        if (g.kind == FWD) {
            float z[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) z[j] = g.add != nullptr && n0 + j < g.N ? ld(g.add + oi + j * P) : 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool in = n0 + j < g.N;
                float t = acc[j] + (in ? ld(g.bias + n0 + j) : 0.0f);
                if (g.relu) t = fmaxf(t, 0.0f);
                if (g.r != nullptr && in) g.r[oi + j * P] = t;
                if (g.add != nullptr) t += z[j];
                z[j] = in ? g.scale * t : 0.0f;
                if (g.out != nullptr && in) g.out[oi + j * P] = z[j];
            }
            if (g.nplanes != nullptr) store_planes8(g.nplanes, M * g.ncp, row * g.ncp + n0, z);
        } else {
            float z[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) z[j] = g.accumulate && n0 + j < g.N ? ld(g.out + oi + j * P) : 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (n0 + j < g.N) g.out[oi + j * P] = z[j] + acc[j];
        }
    }
    // channels of the planes past the last column group
    if (g.kind == FWD && g.nplanes != nullptr && (g.N + 7) / 8 * 8 < g.ncp) {
        const float zero[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        for (size_t row = blockIdx.x * (size_t)blockDim.x + threadIdx.x; row < M; row += (size_t)gridDim.x * blockDim.x)
            store_planes8(g.nplanes, M * g.ncp, row * g.ncp + g.ncp - 8, zero);
    }
}

}  // namespace umma
