// Characteristic tracing kernels: one thread per voxel (= particle), RK4 state
// in registers (Alg. 1).  Included by trace2d.cu and trace3d.cu, each of which
// instantiates the family for one dimension.
//
// Modes (TraceMode):
//   FWD      trace, then transport gather u1 = T(y) (Eq. 6; optional SSD
//            partials, Eq. 10) or continuity splat of T(x_c) at y (Eq. 7).
//   JVP      trace with the forward-mode derivative of Alg. 1 applied to dv,
//            then du = grad T(y) . dy (transport) or the splat of
//            T(x_c) grad_y w . dy (continuity) (Sec. 3.2).
//   JTVP     trace recording the stages, seed the adjoint at the end point,
//            sweep the RK4 stages backwards scattering into the gradient.
//   HESS     transport only: the Gauss-Newton product J^T h^d J dv fused per
//            voxel (u1 at voxel i depends only on characteristic i, so the
//            JVP value feeds that voxel's JTVP seed directly).
//   HROW     the same product by rows (3D, stationary velocity): the adjoint
//            sweep seeded with grad T(y_i) yields the row J_i as a few blocks of
//            corner vectors; they are dotted with dv and scattered scaled by
//            h^d J_i dv (RowScatter).  Where the velocity crosses many cells, by
//            tangent sweeps as HESS (gauss_newton_tangent).
//   OBJGRAD  transport only: u1, SSD partials and the JTVP of h^d res fused.
//   ASM      transport only: the adjoint sweep seeded with grad T(y) yields
//            row i of J = d_v u1 (Sec. 3.3 assembles J as a sparse matrix);
//            its stage contributions are summed per (slice, cell) block in a
//            per-thread table and written out entry-major (ELL layout), and
//            ell_kernel then applies J, J^T and J^T h^d J.
//
// Position representation.  A characteristic starts at a cell centre x_c and
// its state is the FP32 displacement u = y - x_c.  Looking a point up on a grid
// uses the start's continuous grid index split into an integer I0 and a
// fraction F0 (on the image exact; on the velocity grid one FP32 FMA, see
// start_on_velocity): the cell is I0 + floor(F0 + u / h).  A
// characteristic that barely moves off a grid node therefore keeps the sign of
// its displacement (an absolute FP32 coordinate would round it away), and the
// cell choice at the kinks of the piecewise-linear interpolant agrees with an
// exact evaluation.
//
// Jacobian-free derivative products.  d_y I(v, y) enters only as J q (tangent)
// and J^T mu (adjoint), the gradient of the scalar interpolant of v . mu
// (coefficients contracted with mu first).  No d x d matrix lives in registers.
//
// Cells in registers.  A stage evaluates the interpolant of its velocity cell
// from registers and reads memory only when the cell or the stage's time slice
// changes; the adjoint's contributions to a cell are summed in registers (in
// moment form) and leave them only when the cell changes.
//
// What bounds these kernels: first the issue slots, now latency.  Paired FP32
// instructions, the row form of the Gauss-Newton product and the floor without
// conversions took the 128^3 product from 495M to 349M warp instructions (issue
// slots 0.70 -> 0.61 busy) and from 554 to 458 us; what the warps wait for is
// the cell's corners after a change (long scoreboard, at 16 warps per SM).
//
// Time slices.  Every RK4 stage time is t0 + m dt/2 (m = 0..2N), so the host
// packs the velocity (and the direction) at those 2N + 1 times, linearly
// interpolated between its K time nodes, as slices [m][node].  A stage reads
// the one slice of its time: a non-stationary field costs the same gathers as
// a stationary one (K = 1: a single slice), and no time interpolation happens
// in the kernels.
//
// Gradient scatter.  (d_v I)^T mu goes to the padded gradient accumulator with
// one vector reduction (red.global.add.v4.f32 / .v2) per corner of a finished
// block, executed by the L2 atomic units.  With K - 1 <= N the accumulator has
// the K time nodes (TM_NODES): a stage adds to the blocks of both nodes of its
// time cell, which at least one whole step shares, and a node's block is
// reduced once per cell.  Per stage time (TM_SLICES) it would be reduced at
// every second stage; measured on the brain-scale J^T (K = 9, N = 16) 7.8 ms
// with slices against 6.2 ms with nodes, and on the 128 x 150 x 128 product
// with K = 2, N = 5 1058 against 870 us (both with the other changes here).  A node's
// FP32 accumulator then takes all the stages that a slice each took before: errors
// against 64 bits 2.3e-7 -> 2.6e-7 (mass-preserving product, 96 x 112 x 80, K = 9),
// 1.1e-7 -> 1.6e-7 (objective's gradient, 80 x 70 x 60, K = 3).
// With shorter time cells (K - 1 > N) every stage time has two nodes of its own
// and the slices take half the reductions; a streaming kernel then distributes
// them onto the time nodes with the transposed time weights.  A shared-memory
// tile of the velocity grid was measured slower: float atomics on shared memory
// retry under the heavy same-address contention of neighbouring characteristics.
#pragma once

#include <type_traits>

#include "fsum.cuh"
#include "lgnk_internal.h"

namespace lgnk {

// Paired FP32 arithmetic: two values in one 64-bit register, one instruction
// for both (each half rounds as the scalar instruction does).  The tracing
// kernels are bound by issue slots, not by the FP32 lanes, so a pair costs
// half the slots of two scalars.  The pairs used below are the two x-corners
// (or the two coefficients that differ by a factor f_x) of one component:
// they leave poly_coeffs, the moment sums and poly_value as pairs and are
// never repacked inside a stage; only f_y, f_z and mu are duplicated.
using pair2 = unsigned long long;
__device__ __forceinline__ pair2 pk(float lo, float hi) {
    pair2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpk(pair2 p, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ float lo2(pair2 p) {
    float a, b;
    unpk(p, a, b);
    return a;
}
__device__ __forceinline__ float hi2(pair2 p) {
    float a, b;
    unpk(p, a, b);
    return b;
}
__device__ __forceinline__ pair2 fma2(pair2 a, pair2 b, pair2 c) {
    pair2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ pair2 mul2(pair2 a, pair2 b) {
    pair2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair2 sub2(pair2 a, pair2 b) {
    pair2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <int D> struct VecT;
template <> struct VecT<2> { using type = float2; };
template <> struct VecT<3> { using type = float4; };

__device__ __forceinline__ void red_vec(float2* p, const float* x, float w) {
    atomicAdd(p, make_float2(w * x[0], w * x[1]));
}
__device__ __forceinline__ void red_vec(float4* p, const float* x, float w) {
    atomicAdd(p, make_float4(w * x[0], w * x[1], w * x[2], 0.0f));
}

template <int D> struct TileShape;
template <> struct TileShape<2> { static constexpr int X = 16, Y = 16, Z = 1; };
template <> struct TileShape<3> { static constexpr int X = 8, Y = 8, Z = 4; };

// Voxel handled by this thread, of the tile that LGNK_BLOCK / threads CTAs share.
template <int D>
__device__ __forceinline__ void voxel_index(const TraceArgs& A, int threads, int* idx) {
    using TS = TileShape<D>;
    const int per = LGNK_BLOCK / threads;
    int b = blockIdx.x / per;
    const int bx = b % A.tiles[0];
    b /= A.tiles[0];
    const int by = b % A.tiles[1];
    const int bz = b / A.tiles[1];
    const int t = threadIdx.x + (blockIdx.x % per) * threads;
    idx[0] = bx * TS::X + t % TS::X;
    idx[1] = by * TS::Y + (t / TS::X) % TS::Y;
    idx[2] = bz * TS::Z + t / (TS::X * TS::Y);
}

// Start of one characteristic on one grid: its continuous grid index I0 + F0.
// Offsets t = F0 + u / h are clamped to [-2 - I0, m - I0 + 1/2], which keeps
// the lower corner I0 + floor(t) in [-2, m].
template <int D>
struct Start {
    int I0[D];
    float F0[D];
};

template <int D>
__device__ __forceinline__ void start_on_image(const int* idx, Start<D>& s) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
        s.I0[a] = idx[a];
        s.F0[a] = 0.0f;
    }
}

// Floor of t as floor(t) + kFloorMagic: adding 1.5 2^23 rounded down leaves
// the integer in the low mantissa bits (|t| < 2^22; grids have at most 2^20
// cells per axis), on the FP32 pipe, where floorf and the conversion to an
// integer take two instructions of the quarter-rate conversion unit.
constexpr float kFloorMagic = 12582912.0f;
constexpr int kFloorMagicBits = 0x4B400000;

// This thread's characteristic on the velocity grid, held for the whole trace:
// the fraction F0 of its start's continuous index, the clamps of the offset
// t = F0 + u / h (to [-2 - I0, m - I0 + 1/2], which keeps the lower corner in
// [-2, m]) and the constant of the linear cell index.
template <int D>
struct VelocityStart {
    float F0[D], lo[D], hi[D];
    unsigned c;
};

// (x_c - lo_v) / h_v - 1/2 = vxi_a + (i + 1/2) vxi_b, evaluated in FP32: exact where the
// grids' extents and cell counts make both constants short binary fractions (a velocity of a
// half or a quarter of the image's cells), else off by the constants' roundings and the
// FMA's, up to 1.2e-7 of the index: 1e-5 cells at 2^7 cells, 0.1 at the 2^20 that an axis may have.
template <int D>
__device__ __forceinline__ void start_on_velocity(const TraceArgs& A, const int* idx, VelocityStart<D>& s) {
    unsigned st = 1;
    s.c = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const float xi = fmaf((float)idx[a] + 0.5f, A.vxi_b[a], A.vxi_a[a]);
        const int i0 = min(max((int)floorf(xi), -2), A.vg.m[a]);
        s.F0[a] = xi - (float)i0;
        s.lo[a] = (float)(-2 - i0);
        s.hi[a] = (float)(A.vg.m[a] - i0) + 0.5f;
        s.c += st * (unsigned)(i0 + LGNK_PAD - kFloorMagicBits);
        st *= (unsigned)A.vg.mp[a];
    }
}

// Cell of the point at displacement u from the start, on the velocity grid:
// its linear padded index, and the fractional offsets f in [0, 1].  NaN maps
// to the lowest clamp, so any point addresses padded storage.  (The index
// arithmetic wraps: the magic's bits cancel against s.c.)
template <int D>
__device__ __forceinline__ int locate_velocity(const DevGrid& g, const VelocityStart<D>& s, const float* u, float* f) {
    unsigned b = 0;
    unsigned k[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        float t = fmaf(u[a], g.inv_h[a], s.F0[a]);
        t = fminf(fmaxf(t, s.lo[a]), s.hi[a]);
        const float r = __fadd_rd(t, kFloorMagic);
        f[a] = t - (r - kFloorMagic);
        k[a] = __float_as_uint(r);
    }
    if (D == 3) b = k[0] + (unsigned)g.mp[0] * (k[1] + (unsigned)g.mp[1] * k[D - 1]);
    else b = k[0] + (unsigned)g.mp[0] * k[1];
    return (int)(b + s.c);
}

// Cell of a point on a grid from the start's split index (the image at the
// end of the trace): per-axis padded index p of the lower corner, offsets f.
template <int D>
__device__ __forceinline__ void locate(const DevGrid& g, const Start<D>& s, const float* u, int* p, float* f) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
        float t = fmaf(u[a], g.inv_h[a], s.F0[a]);
        t = fminf(fmaxf(t, (float)(-2 - s.I0[a])), (float)(g.m[a] - s.I0[a]) + 0.5f);
        const float fl = floorf(t);
        f[a] = t - fl;
        p[a] = s.I0[a] + (int)fl + LGNK_PAD;
    }
}

template <int D>
__device__ __forceinline__ int linear(const DevGrid& g, const int* p) {
    if (D == 3) return p[0] + g.mp[0] * (p[1] + g.mp[1] * p[2]);
    return p[0] + g.mp[0] * p[1];
}

template <int D>
__device__ __forceinline__ int corner_offset(const DevGrid& g, int c) {
    int o = (c & 1) + ((c >> 1) & 1) * g.mp[0];
    if (D == 3) o += ((c >> 2) & 1) * g.mp[0] * g.mp[1];
    return o;
}

// Multilinear weight of corner c and (optionally) its derivative along each axis.
template <int D, bool GRAD>
__device__ __forceinline__ float corner_weight(int c, const float* f, const DevGrid& g, float* dw) {
    float w1[D];
#pragma unroll
    for (int a = 0; a < D; ++a) w1[a] = ((c >> a) & 1) ? f[a] : 1.0f - f[a];
    float w = w1[0];
#pragma unroll
    for (int a = 1; a < D; ++a) w *= w1[a];
    if (GRAD) {
#pragma unroll
        for (int a = 0; a < D; ++a) {
            float p = ((c >> a) & 1) ? g.inv_h[a] : -g.inv_h[a];
#pragma unroll
            for (int b = 0; b < D; ++b)
                if (b != a) p *= w1[b];
            dw[a] = p;
        }
    }
    return w;
}

// Both x-corners of a cell row from the pair-packed velocity: element e holds
// [v(node) | v(node + 1)] (3D: 32 bytes, one 256-bit load; 2D: 16 bytes).
__device__ __forceinline__ void load_pair3(const float* p, float* a, float* b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, _, %3, %4, %5, _}, [%6];"
        : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(b[0]), "=f"(b[1]), "=f"(b[2])
        : "l"(p));
}

template <int D>
__device__ __forceinline__ void pair_value(const float* __restrict__ V, size_t e, float* a, float* b) {
    constexpr int PS = (D == 3) ? 8 : 4;
    if (D == 3) {
        load_pair3(V + e * PS, a, b);
    } else {
        const float4 t = __ldg(reinterpret_cast<const float4*>(V + e * PS));
        a[0] = t.x; a[1] = t.y; b[0] = t.z; b[1] = t.w;
    }
}

// Element of corner (0, cy, cz) of the cell with lower corner `base` in the
// slice starting at element `s0`.
template <int D>
__device__ __forceinline__ size_t corner_elem(const DevGrid& g, size_t s0, int base, int cx, int cy, int cz) {
    int o = base + cx + cy * g.mp[0];
    if (D == 3) o += cz * g.mp[0] * g.mp[1];
    return s0 + (size_t)o;
}

// A pending cell block in moment form.  The block's corner vectors are
// sum_stages w_c(f) mu with w_c = prod_a (c_a ? f_a : 1 - f_a); expanding the
// product, they follow from the moments m_k = sum_stages phi_k(f) mu, phi_k =
// prod of the f_a over the axes a set in k (bit 0 x, bit 1 y, bit 2 z), by
// one subtraction per pair and axis: w_c = sum over subsets T of the axes
// with c_a = 0 of (-1)^|T| phi_(c + T).  A stage then costs the 2^d - 1 - d
// products of offsets, D adds and (2^d - 1) D FMAs (3D: 4 FMUL, 3 FADD, 21
// FFMA) instead of the corner weights and (2^d) D FMAs (12 FMUL, 3 FADD, 24
// FFMA); the conversion (12 FADD per component in 3D) is paid once per block.
// Blocks are held as pairs over the x axis, m[q][j] = (m_2j, m_2j+1) of
// component q.
template <int D>
struct Block {
    static constexpr int NP = 1 << (D - 1);     // pairs per component
    pair2 m[D][NP];
};

template <int D>
__device__ __forceinline__ void moments_add(Block<D>& B, const float* f, const float* mu) {
    constexpr int NP = Block<D>::NP;
    pair2 phi[NP];
    phi[0] = pk(1.0f, f[0]);
    phi[1] = mul2(pk(f[1], f[1]), phi[0]);
    if (D == 3) {
        const pair2 fz = pk(f[D - 1], f[D - 1]);
        phi[NP / 2] = mul2(fz, phi[0]);
        phi[NP - 1] = mul2(fz, phi[1]);
    }
#pragma unroll
    for (int q = 0; q < D; ++q) {
        const pair2 w = pk(mu[q], mu[q]);
#pragma unroll
        for (int k = 0; k < NP; ++k) B.m[q][k] = fma2(phi[k], w, B.m[q][k]);
    }
}

// The same with the corner weights themselves (the mass-preserving model): no corner is
// a difference of sums, for one FADD an axis and three more paired products a stage (3D), and
// without the conversion.  Error of J^T r against 64 bits, moments -> corners, 80 x 70 x 60 voxels:
// 4.1e-7 -> 2.7e-7; 96 x 112 x 80 with 9 time nodes, product: 2.84e-7 -> 2.61e-7; brain-scale
// product 10.03 -> 10.20 ms.  For the transport model moments are as exact as they ever were.
template <int D>
__device__ __forceinline__ void corners_add(Block<D>& B, const float* f, const float* mu) {
    constexpr int NP = Block<D>::NP;
    pair2 w[NP];
    const pair2 x = pk(1.0f - f[0], f[0]);
    const float y0 = 1.0f - f[1];
    w[0] = mul2(x, pk(y0, y0));
    w[1] = mul2(x, pk(f[1], f[1]));
    if (D == 3) {
        const float z0 = 1.0f - f[D - 1];
        const pair2 hi = pk(f[D - 1], f[D - 1]), lo = pk(z0, z0);
        w[NP / 2] = mul2(w[0], hi);
        w[NP - 1] = mul2(w[1], hi);
        w[0] = mul2(w[0], lo);
        w[1] = mul2(w[1], lo);
    }
#pragma unroll
    for (int q = 0; q < D; ++q) {
        const pair2 m = pk(mu[q], mu[q]);
#pragma unroll
        for (int k = 0; k < NP; ++k) B.m[q][k] = fma2(w[k], m, B.m[q][k]);
    }
}

template <int D, bool MOMENTS>
__device__ __forceinline__ void block_add(Block<D>& B, const float* f, const float* mu) {
    if constexpr (MOMENTS) moments_add<D>(B, f, mu);
    else corners_add<D>(B, f, mu);
}

// Moments to corner vectors, in place: afterwards m[q][j] holds corners
// (0, cy, cz) and (1, cy, cz), j = cy + 2 cz.
template <int D>
__device__ __forceinline__ void moments_to_corners(Block<D>& B) {
    constexpr int NP = Block<D>::NP;
#pragma unroll
    for (int q = 0; q < D; ++q) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            float a, b;
            unpk(B.m[q][k], a, b);
            B.m[q][k] = pk(a - b, b);
        }
#pragma unroll
        for (int b = 1; b < NP; b <<= 1)
#pragma unroll
            for (int k = 0; k < NP; ++k)
                if (!(k & b)) B.m[q][k] = sub2(B.m[q][k], B.m[q][k | b]);
    }
}

template <int D>
__device__ __forceinline__ void block_zero(Block<D>& B) {
#pragma unroll
    for (int q = 0; q < D; ++q)
#pragma unroll
        for (int k = 0; k < Block<D>::NP; ++k) B.m[q][k] = 0;
}

// Corner c of a block of corner vectors.
template <int D>
__device__ __forceinline__ void block_corner(const Block<D>& B, int c, float* x) {
#pragma unroll
    for (int q = 0; q < D; ++q) x[q] = (c & 1) ? hi2(B.m[q][c >> 1]) : lo2(B.m[q][c >> 1]);
}

// Adds w times a block of corner vectors at cell `key` to the gradients.
template <int D>
__device__ __forceinline__ void block_red(const DevGrid& g, typename VecT<D>::type* G, int key, const Block<D>& B,
                                          float w) {
#pragma unroll
    for (int c = 0; c < (1 << D); ++c) {
        float x[D];
        block_corner<D>(B, c, x);
        red_vec(G + corner_elem<D>(g, (size_t)key, 0, c & 1, (c >> 1) & 1, (c >> 2) & 1), x, w);
    }
}

// Destinations of the adjoint contributions w_c(f) mu.  The pending cell stays
// in registers (in moment form) and leaves them only when a stage falls in
// another cell (`emit`).  In time-node mode (NB = 2) a stage contributes to
// both nodes of its time cell, (1 - th) w_c mu to the block of node j and th w_c
// mu to that of node j + 1; node j's block is blk[j mod 2], so that when the
// sweep moves on to the next time cell one node is finished and the other's
// block stays where it is.  All keys are 32-bit element offsets (the packed
// velocity has fewer than 2^31 elements: checked when the context is created).

// Gradients and J^T r: the block's corners go to the slice (node) gradients
// with one vector reduction each.
template <int D, int NB>
struct BlockScatter {
    static constexpr bool MOMENTS = true;
    typename VecT<D>::type* G;
    int key, odd, sn;         // cell of the pending block(s) at its (earlier) node, -1 if none; NB = 2: that
                              // node's parity; elements per node
    Block<D> blk[NB];
};

template <int D, int NB>
__device__ __forceinline__ void scatter_emit(const DevGrid& g, BlockScatter<D, NB>& S, int b, int key) {
    moments_to_corners<D>(S.blk[b]);
    block_red<D>(g, S.G, key, S.blk[b], 1.0f);
}

// The same with the blocks kept as corner vectors (the mass-preserving model).
template <int D, int NB>
struct CornerScatter {
    static constexpr bool MOMENTS = false;
    typename VecT<D>::type* G;
    int key, odd, sn;
    Block<D> blk[NB];
};

template <int D, int NB>
__device__ __forceinline__ void scatter_emit(const DevGrid& g, CornerScatter<D, NB>& S, int b, int key) {
    block_red<D>(g, S.G, key, S.blk[b], 1.0f);
}

// The fused Gauss-Newton product by rows (MODE_HROW).  Row i of J is the adjoint
// sweep seeded with grad T(y_i), so one sweep yields both J_i dv (the blocks
// dotted with the direction's corners) and, scaled by h^d J_i dv, the row's
// contribution to J^T h^d J dv.  The blocks are kept until the dot product is
// known: the last in registers, the earlier ones (a trajectory leaves its
// velocity cell 0.4 times on average on the 128^3 workload) in a per-thread
// local array.  A row with more than CAP earlier blocks is swept a second time
// (`direct`) with the scaled seed and then scatters as the gradient does.
// Against a tangent sweep for J dv (MODE_HESS) this drops the direction's
// interpolation and the products d_y I q at every stage, 390 instead of 615
// FP32 operations per voxel-step, and adds the blocks' way through local
// memory once per row and cell: at 128^3 0.447 against 0.513 ms with N = 8, 0.279 against
// 0.293 ms with N = 4, but 0.200 against 0.190 ms with N = 2 (64 x 60 x 62:
// 61 / 70, 39 / 43, 30.5 / 28.6 us).  It stays with the tangent sweep in 2D (cheap
// stages: 10 to 20% slower by rows) and for K > 1 (a block per time node and
// cell: 5 to 40% slower).
template <int D, int NB>
struct RowScatter {
    static constexpr bool MOMENTS = true;
    static constexpr int CAP = 6;
    static constexpr int NV = (1 << D) * D / 4;      // float4s of a block
    typename VecT<D>::type* G;
    int key, odd, sn, n;
    bool direct;
    float du;                 // of the blocks that were not kept
    const float* dV;
    float4* st;               // [CAP][NV], moments
    int* stkey;               // [CAP]
    Block<D> blk[NB];
};

// The block of corner vectors . the direction at cell `key`
template <int D>
__device__ __forceinline__ float block_dot(const DevGrid& g, const float* __restrict__ dV, int key,
                                           const Block<D>& B) {
    float s = 0.0f;
#pragma unroll
    for (int j = 0; j < Block<D>::NP; ++j) {
        float lo[3], hi[3];
        pair_value<D>(dV, corner_elem<D>(g, (size_t)key, 0, 0, j & 1, j >> 1), lo, hi);
#pragma unroll
        for (int q = 0; q < D; ++q) {
            float a, b;
            unpk(B.m[q][j], a, b);
            s = fmaf(a, lo[q], s);
            s = fmaf(b, hi[q], s);
        }
    }
    return s;
}

template <int D>
__device__ __forceinline__ void block_store(float4* dst, const Block<D>& B) {
    constexpr int NP = Block<D>::NP, NV = (1 << D) * D / 4;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        float a[4];
        unpk(B.m[(2 * v) / NP][(2 * v) % NP], a[0], a[1]);
        unpk(B.m[(2 * v + 1) / NP][(2 * v + 1) % NP], a[2], a[3]);
        dst[v] = make_float4(a[0], a[1], a[2], a[3]);
    }
}

template <int D>
__device__ __forceinline__ void block_load(const float4* src, Block<D>& B) {
    constexpr int NP = Block<D>::NP, NV = (1 << D) * D / 4;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const float4 t = src[v];
        B.m[(2 * v) / NP][(2 * v) % NP] = pk(t.x, t.y);
        B.m[(2 * v + 1) / NP][(2 * v + 1) % NP] = pk(t.z, t.w);
    }
}

template <int D, int NB>
__device__ __forceinline__ void scatter_emit(const DevGrid& g, RowScatter<D, NB>& S, int b, int key) {
    if (S.direct) {
        moments_to_corners<D>(S.blk[b]);
        block_red<D>(g, S.G, key, S.blk[b], 1.0f);
    } else {
        if (S.n < RowScatter<D, NB>::CAP) {
            // converted and dotted after the sweep, where the warp's lanes are together again
            block_store<D>(S.st + S.n * RowScatter<D, NB>::NV, S.blk[b]);
            S.stkey[S.n] = key;
        } else {
            moments_to_corners<D>(S.blk[b]);
            S.du += block_dot<D>(g, S.dV, key, S.blk[b]);
        }
        S.n++;
    }
}

template <int D, int NB, template <int, int> class SC>
__device__ __forceinline__ void scatter_init(SC<D, NB>& S, void* G, int sn) {
    S.G = static_cast<typename VecT<D>::type*>(G);
    S.sn = sn;
    S.key = -1;
    S.odd = 0;
#pragma unroll
    for (int b = 0; b < NB; ++b) block_zero<D>(S.blk[b]);
}

// Element of the cell whose pending contributions blk[b] holds.
template <int D, int NB, template <int, int> class SC>
__device__ __forceinline__ int block_key(const SC<D, NB>& S, int b) {
    return NB == 2 && b != S.odd ? S.key + S.sn : S.key;
}

template <int D, int NB, template <int, int> class SC>
__device__ __forceinline__ void block_out(const DevGrid& g, SC<D, NB>& S, int b) {
    scatter_emit(g, S, b, block_key(S, b));
    block_zero<D>(S.blk[b]);
}

// Every pending block out.
template <int D, int NB, template <int, int> class SC>
__device__ __forceinline__ void scatter_finish(const DevGrid& g, SC<D, NB>& S) {
    if (S.key < 0) return;
#pragma unroll
    for (int b = 0; b < NB; ++b) block_out(g, S, b);
}

template <int D, int NB, template <int, int> class SC>
__device__ __forceinline__ void scatter_cell(const DevGrid& g, SC<D, NB>& S, int key, int odd) {
    if (key == S.key) return;
    if (S.key >= 0) {
        // the finished nodes: one of the two if only the time cell moved on by one
        const bool later = key == S.key + S.sn, earlier = key == S.key - S.sn;
        if (NB == 1 || !later || S.odd != 0)
            if (NB == 1 || !earlier || S.odd == 0) block_out(g, S, NB - 1);
        if (NB == 2)
            if ((!later || S.odd == 0) && (!earlier || S.odd != 0)) block_out(g, S, 0);
    }
    S.key = key;
    S.odd = odd;
}

// Add the contribution w_c(f) mu at cell `key` (NB = 2: of the earlier node,
// whose parity is odd, with the time offset th).
template <int D, int NB, template <int, int> class SC>
__device__ __forceinline__ void scatter_add(const DevGrid& g, SC<D, NB>& S, int key, int odd, float th, const float* f,
                                            const float* mu) {
    scatter_cell(g, S, key, odd);
    if (NB == 1) {
        block_add<D, SC<D, NB>::MOMENTS>(S.blk[0], f, mu);
    } else {
        const float t1 = odd ? 1.0f - th : th;      // weight of the odd node
        float m1[D], m0[D];
#pragma unroll
        for (int q = 0; q < D; ++q) {
            m1[q] = t1 * mu[q];
            m0[q] = mu[q] - m1[q];
        }
        block_add<D, SC<D, NB>::MOMENTS>(S.blk[0], f, m0);
        block_add<D, SC<D, NB>::MOMENTS>(S.blk[NB - 1], f, m1);
    }
}

// Destination of the adjoint contributions when a row of J is assembled: the
// row's (slice, cell) blocks, each the 2^d corner vectors sum_stages
// w_c(f) mu.  A trajectory stays within a few velocity cells, so a row has
// few blocks; a row that needs more than CAP sets `overflow`.  The keys live
// in a per-thread table (local memory); the blocks go straight to the row's
// slots of the global ELL array, entry j of voxel i at [j][i][corner][q], and
// a block met again is read back, added to and stored by the same thread.
template <int D>
struct AsmTable {
    static constexpr int CAP = D == 3 ? 16 : 32;
    long long key[CAP];
    int n;
    bool overflow;
};

// The block of the current cell is kept in registers until the cell changes;
// it is then committed to the row (kept in the table's local array it was
// placed in local memory: 1.23 ms for the 128^3 assembly, 0.79 ms apart).
template <int D, int NB>
struct AsmRow {
    static constexpr bool MOMENTS = true;
    static constexpr int B = (1 << D) * D;
    typename VecT<D>::type* G;
    AsmTable<D>* tab;
    float* row;               // entry 0 of this voxel's blocks in the ELL array
    size_t stride;            // floats from entry j to entry j + 1 of one voxel
    int key, odd, sn;
    Block<D> blk[NB];
};

// Adds the pending block to the row's entry of its cell (a new entry if the
// row has none yet).
template <int D, int NB>
__device__ __forceinline__ void scatter_emit(const DevGrid&, AsmRow<D, NB>& S, int b, int key) {
    constexpr int B = AsmRow<D, NB>::B;
    AsmTable<D>& T = *S.tab;
    moments_to_corners<D>(S.blk[b]);
    int j = T.n - 1;
#pragma unroll 1
    for (; j >= 0; --j)       // newest first: a trajectory revisits the cell it just left
        if (T.key[j] == key) break;
    const bool fresh = j < 0;
    if (fresh) {
        if (T.n == AsmTable<D>::CAP) {
            T.overflow = true;
            return;
        }
        j = T.n++;
        T.key[j] = key;
    }
    float x[B];               // [corner][component]
#pragma unroll
    for (int c = 0; c < (1 << D); ++c) block_corner<D>(S.blk[b], c, x + c * D);
    float4* dst = reinterpret_cast<float4*>(S.row + (size_t)j * S.stride);
#pragma unroll
    for (int k = 0; k < B / 4; ++k) {
        float4 w = make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
        if (!fresh) {
            const float4 o = dst[k];
            w.x += o.x;
            w.y += o.y;
            w.z += o.z;
            w.w += o.w;
        }
        dst[k] = w;
    }
}

// Stage time of stage st (0..3) of step k: slice 2k, 2k + 1, 2k + 1, 2k + 2.
template <int TM>
__device__ __forceinline__ int stage_slice(int k, int st) {
    return TM == TM_STEADY ? 0 : 2 * k + ((st + 1) >> 1);
}

// The multilinear interpolant of a cell in polynomial form, per component
//   3D: v(f) = a0 + a1 fx + a2 fy + a3 fz + a4 fx fy + a5 fx fz + a6 fy fz + a7 fx fy fz
//   2D: v(f) = a0 + a1 fx + a2 fy + a3 fx fy
// with f the fractional offsets in the cell, held as pairs over the x axis:
//   3D: (a0, a1), (a2, a4), (a3, a5), (a6, a7)     2D: (a0, a1), (a2, a3)
// so that fixing f_y (and f_z) is one paired FMA for both halves and f_x is
// applied last.  Coefficients of one component from its corner values, c[j] =
// corners (0, cy, cz) and (1, cy, cz), j = cy + 2 cz.
template <int D>
__device__ __forceinline__ void poly_coeffs(const pair2* c, pair2* a) {
    constexpr int NP = 1 << (D - 1);
    pair2 e[NP];              // (value, x difference) of every row of the cell
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        float lo, hi;
        unpk(c[j], lo, hi);
        e[j] = pk(lo, hi - lo);
    }
    a[0] = e[0];
    a[1] = sub2(e[1], e[0]);
    if (D == 3) {
        a[NP / 2] = sub2(e[NP / 2], e[0]);
        a[NP - 1] = sub2(sub2(e[NP - 1], e[NP / 2]), a[1]);
    }
}

// The interpolant with f_y (and f_z) applied: (value at f_x = 0, x slope).
// The order of the sums is fixed (f_y, then f_z, then f_x): the positions of
// every kernel that traces the same velocity agree bit for bit.
template <int D>
__device__ __forceinline__ pair2 poly_row(const pair2* a, const pair2* fd) {
    constexpr int NP = 1 << (D - 1);
    if (D == 2) return fma2(fd[0], a[1], a[0]);
    const pair2 t = fma2(fd[D - 2], a[NP - 1], a[1]);
    return fma2(fd[D - 2], a[NP / 2], fma2(fd[0], t, a[0]));
}

// f_y (and f_z) duplicated into pairs
template <int D>
__device__ __forceinline__ void dup_offsets(const float* f, pair2* fd) {
    fd[0] = pk(f[1], f[1]);
    if (D == 3) fd[D - 2] = pk(f[D - 1], f[D - 1]);
}

template <int D>
__device__ __forceinline__ float row_value(pair2 row, const float* f) {
    float v, gx;
    unpk(row, v, gx);
    return fmaf(f[0], gx, v);
}

// Derivatives along the fractional offsets (per cell width); the constant
// coefficient is not read.  The order of the sums is fixed (3D: f_z first for
// the x and y derivatives, f_x first for the z derivative): the rows of J, and
// with them a solve's iterates, keep their rounding whatever the pairing.
template <int D>
__device__ __forceinline__ void poly_grad(const pair2* a, const float* f, const pair2* fd, float* gr) {
    constexpr int NP = 1 << (D - 1);
    float t0, t1;
    if (D == 2) {
        unpk(a[1], t0, t1);
        gr[0] = fmaf(f[1], t1, hi2(a[0]));
        gr[1] = fmaf(f[0], t1, t0);
        return;
    }
    unpk(fma2(fd[D - 2], a[NP - 1], a[1]), t0, t1);
    gr[0] = fmaf(f[D - 1], hi2(a[NP / 2]), fmaf(f[1], t1, hi2(a[0])));
    gr[1] = fmaf(f[0], t1, t0);
    unpk(a[NP / 2], t0, t1);
    float u0, u1;
    unpk(a[NP - 1], u0, u1);
    gr[D - 1] = fmaf(f[1], fmaf(f[0], u1, u0), fmaf(f[0], t1, t0));
}

// The same interpolant as nested linear interpolations (x, then y, then z) of
// the corner values; c[j] = the two values along the last axis, j = cx (+ 2 cy
// in 3D), so that all but the last axis are paired.
template <int D>
__device__ __forceinline__ float lerp_value(const pair2* c, const float* f, const pair2* fx) {
    pair2 r;
    if (D == 2) {
        r = fma2(fx[0], sub2(c[1], c[0]), c[0]);
    } else {
        const pair2 a0 = fma2(fx[0], sub2(c[1], c[0]), c[0]);
        const pair2 a1 = fma2(fx[0], sub2(c[D], c[2]), c[2]);
        r = fma2(fx[D - 2], sub2(a1, a0), a0);
    }
    float lo, hi;
    unpk(r, lo, hi);
    return fmaf(f[D - 1], hi - lo, lo);
}

// ... with its product with qs (a direction in cell widths).
template <int D>
__device__ __forceinline__ float lerp_value_dot(const pair2* c, const float* f, const pair2* fx, const float* qs,
                                                float& dot) {
    float lo, hi, l0, l1;
    if (D == 2) {
        const pair2 d = sub2(c[1], c[0]);
        unpk(fma2(fx[0], d, c[0]), lo, hi);
        unpk(d, l0, l1);
        const float dl = hi - lo;
        dot = fmaf(fmaf(f[1], l1 - l0, l0), qs[0], dl * qs[1]);
        return fmaf(f[1], dl, lo);
    }
    const pair2 d0 = sub2(c[1], c[0]), d1 = sub2(c[D], c[2]);
    const pair2 a0 = fma2(fx[0], d0, c[0]);
    const pair2 dy = sub2(fma2(fx[0], d1, c[2]), a0);
    unpk(fma2(fx[D - 2], dy, a0), lo, hi);
    const float dl = hi - lo;
    // x and y slopes share the remaining interpolation: dot them first
    const pair2 dx = fma2(fx[D - 2], sub2(d1, d0), d0);
    unpk(fma2(dx, pk(qs[0], qs[0]), mul2(dy, pk(qs[1], qs[1]))), l0, l1);
    dot = fmaf(dl, qs[D - 1], fmaf(f[D - 1], l1 - l0, l0));
    return fmaf(f[D - 1], dl, lo);
}

// f_x (and f_y in 3D) duplicated into pairs, for the lerp forms
template <int D>
__device__ __forceinline__ void dup_offsets_x(const float* f, pair2* fx) {
    fx[0] = pk(f[0], f[0]);
    if (D == 3) fx[D - 2] = pk(f[1], f[1]);
}

// The corner values of a cell as pairs: over the x axis, c[q][cy + 2 cz], or,
// with LAST, over the last axis, c[q][cx (+ 2 cy)].
template <int D, bool LAST>
__device__ __forceinline__ void load_corners(const DevGrid& g, const float* __restrict__ V, int key,
                                             pair2 (&c)[D][1 << (D - 1)]) {
    constexpr int NP = 1 << (D - 1);
    float lo[NP][3], hi[NP][3];
#pragma unroll
    for (int j = 0; j < NP; ++j)
        pair_value<D>(V, corner_elem<D>(g, (size_t)key, 0, 0, j & 1, j >> 1), lo[j], hi[j]);
#pragma unroll
    for (int q = 0; q < D; ++q) {
        if (!LAST) {
#pragma unroll
            for (int j = 0; j < NP; ++j) c[q][j] = pk(lo[j][q], hi[j][q]);
        } else if (D == 2) {
            c[q][0] = pk(lo[0][q], lo[1][q]);
            c[q][1] = pk(hi[0][q], hi[1][q]);
        } else {
            c[q][0] = pk(lo[0][q], lo[NP / 2][q]);
            c[q][1] = pk(hi[0][q], hi[NP / 2][q]);
            c[q][NP / 2] = pk(lo[1][q], lo[NP - 1][q]);
            c[q][NP - 1] = pk(hi[1][q], hi[NP - 1][q]);
        }
    }
}

// The velocity cell a sweep last met, kept in registers: consecutive stages
// mostly fall in the same cell and slice (stages 2 and 3 share their time and
// nearly their position, stage 4 of a step is stage 1 of the next), so a stage
// reads memory only when its cell or slice changes.  FORM: the polynomial
// coefficients, or the corner values for the nested interpolation.  The
// forward sweep of the transport model evaluates coefficients, that of the
// mass-preserving model corner values: the form fixes the rounding of the
// positions, and with it on which side of a cell face a characteristic ends.
enum CellForm { POLY = 0, CORNERS = 1 };
template <int D, int FORM>
struct Cell {
    static constexpr int NP = 1 << (D - 1);
    int key;                  // element of the cached cell, -1 when empty (32 bits: the packed velocity has
                              // fewer than 2^31 elements, checked when the context is created)
    pair2 e[D][NP];
};

template <int D, int FORM>
__device__ __forceinline__ void cell_at(const DevGrid& g, const float* __restrict__ V, int key, Cell<D, FORM>& C) {
    if (key == C.key) return;
    C.key = key;
    if constexpr (FORM == CORNERS) {
        load_corners<D, true>(g, V, key, C.e);
    } else {
        pair2 c[D][1 << (D - 1)];
        load_corners<D, false>(g, V, key, c);
#pragma unroll
        for (int q = 0; q < D; ++q) poly_coeffs<D>(c[q], C.e[q]);
    }
}

// T(y) and optionally grad T(y) from the padded image, y at displacement u.
template <int D, bool GRAD>
__device__ __forceinline__ float sample_image(const DevGrid& g, const Start<D>& s, const float* __restrict__ Tp,
                                              const float* u, float* grad) {
    int p[D];
    float f[D];
    locate<D>(g, s, u, p, f);
    const int base = linear<D>(g, p);
    float val = 0.0f;
    if (GRAD) {
#pragma unroll
        for (int a = 0; a < D; ++a) grad[a] = 0.0f;
    }
#pragma unroll
    for (int c = 0; c < (1 << D); ++c) {
        const float t = __ldg(Tp + base + corner_offset<D>(g, c));
        float dw[D];
        const float w = corner_weight<D, GRAD>(c, f, g, dw);
        val = fmaf(w, t, val);
        if (GRAD) {
#pragma unroll
            for (int a = 0; a < D; ++a) grad[a] = fmaf(dw[a], t, grad[a]);
        }
    }
    return val;
}

// The push-forward through a shared-memory tile (Eq. 7 with the default
// particle width; every thread of the CTA calls it, inactive ones with
// active = false).  The CTA's particles start on one 8 x 8 x 4 (3D) or
// 16 x 16 (2D) tile of voxels and a smooth flow keeps their end cells
// together, so the CTA reduces the box of their cells; when the box with its
// upper corners holds at most kSplatTile cells, the particles add their
// corner masses into a zeroed tile in shared memory and the CTA then adds
// each nonzero cell of the tile to the image with one global atomic, instead
// of one per particle and corner.  A larger box (large displacements) takes
// the per-particle global atomics.  Measured on the brain-scale forward and
// JVP: 2.06 / 4.01 ms against 1.99 / 3.97 ms with the box reduction but
// direct global atomics (1.93 / 3.85 ms with the splat inline in the trace):
// the L2 atomics are not what bounds these kernels.  Combining, before the
// shared atomic, the lanes of a warp whose corner lands in the same cell
// (__match_any_sync, one leader per cell) measured 2.14 / 4.12 ms: for a
// given corner the lanes' cells are distinct unless the flow compresses, so
// the match finds no peers and costs its instructions.
constexpr int kSplatTile = 2048;

template <int D, bool TANGENT>
__device__ __forceinline__ void splat_tiled(const DevGrid& g, float* acc, bool active, const int* p, const float* f,
                                            float mass, const float* dp) {
    __shared__ float tile[kSplatTile];
    __shared__ int wbox[LGNK_BLOCK / 32][6];
    float x[1 << D];
#pragma unroll
    for (int c = 0; c < (1 << D); ++c) {
        float dw[D];
        const float w = corner_weight<D, TANGENT>(c, f, g, dw);
        if (TANGENT) {
            float t = 0.0f;
#pragma unroll
            for (int a = 0; a < D; ++a) t = fmaf(dw[a], dp[a], t);
            x[c] = t * mass;
        } else {
            x[c] = w * mass;
        }
    }
    // the box of the CTA's cells (lower corners), per axis
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int lo[3] = {0, 0, 0}, hi[3] = {-1, -1, -1};
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int l = __reduce_min_sync(0xffffffffu, active ? p[a] : 0x7fffffff);
        const int h = __reduce_max_sync(0xffffffffu, active ? p[a] : -0x7fffffff);
        if (lane == 0) {
            wbox[warp][a] = l;
            wbox[warp][3 + a] = h;
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < D; ++a) {
        lo[a] = wbox[0][a];
        hi[a] = wbox[0][3 + a];
#pragma unroll
        for (int w = 1; w < LGNK_BLOCK / 32; ++w) {
            lo[a] = min(lo[a], wbox[w][a]);
            hi[a] = max(hi[a], wbox[w][3 + a]);
        }
    }
    if (hi[0] < lo[0]) return;            // no active particle in the CTA
    int ext[3] = {1, 1, 1};
    long long vol = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        ext[a] = hi[a] - lo[a] + 2;
        vol *= ext[a];
    }
    if (vol > kSplatTile) {
        if (active) {
            const int base = linear<D>(g, p);
#pragma unroll
            for (int c = 0; c < (1 << D); ++c) atomicAdd(acc + base + corner_offset<D>(g, c), x[c]);
        }
        return;
    }
    const int nv = (int)vol;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) tile[i] = 0.0f;
    __syncthreads();
    const int lb = active ? (p[0] - lo[0]) + ext[0] * ((p[1] - lo[1]) + (D == 3 ? ext[1] * (p[D - 1] - lo[D - 1]) : 0))
                          : 0;
#pragma unroll
    for (int c = 0; c < (1 << D); ++c) {
        const int l = lb + (c & 1) + ((c >> 1) & 1) * ext[0] + (D == 3 ? ((c >> 2) & 1) * ext[0] * ext[1] : 0);
        if (active) atomicAdd(&tile[l], x[c]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
        const float v = tile[i];
        if (v != 0.0f) {
            int r = i;
            const int ix = r % ext[0];
            r /= ext[0];
            int gi;
            if (D == 3) {
                const int iy = r % ext[1];
                const int iz = r / ext[1];
                gi = (lo[0] + ix) + g.mp[0] * ((lo[1] + iy) + g.mp[1] * (lo[D - 1] + iz));
            } else {
                gi = (lo[0] + ix) + g.mp[0] * (lo[1] + r);
            }
            atomicAdd(acc + gi, v);
        }
    }
}

// General-width PIC push-forward (Eqs. 7-8): the particle is the tensor
// product of unit-mass hats max(0, 1 - |s| / rho) / rho of half-width rho
// cells; cell c (node coordinates [c - 1/2, c + 1/2]) receives the exact
// integral of the particle over it, a difference of the hat's antiderivative,
// so the weights of a particle sum to one.  Cells outside the grid are
// dropped.  rho <= 3.5 keeps a particle within kHatMax cells per axis.
constexpr int kHatMax = 8;

__device__ __forceinline__ float hat_cdf(float s) {
    s = fminf(fmaxf(s, -1.0f), 1.0f);
    return s <= 0.0f ? 0.5f * (1.0f + s) * (1.0f + s) : 1.0f - 0.5f * (1.0f - s) * (1.0f - s);
}

__device__ __forceinline__ float hat_pdf(float s) { return fmaxf(0.0f, 1.0f - fabsf(s)); }

// Cells [I0 + c0, I0 + c0 + n) of one axis that a particle at node coordinate
// I0 + t overlaps inside the grid, their weights and d(weight)/dy.
__device__ __forceinline__ void hat_axis(float t, float rho, int I0, int m, float inv_h, int& c0, int& n, float* w,
                                         float* dw) {
    t = fminf(fmaxf(t, -(float)I0 - rho - 2.0f), (float)(m - I0) + rho + 2.0f);   // also maps NaN into range
    const int lo = max((int)floorf(t - rho + 0.5f), -I0);
    const int hi = min((int)floorf(t + rho + 0.5f), m - 1 - I0);
    c0 = lo;
    n = min(hi - lo + 1, kHatMax);
    const float ir = 1.0f / rho;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const float c = (float)(lo + j);
        const float s1 = (c + 0.5f - t) * ir, s0 = (c - 0.5f - t) * ir;
        w[j] = hat_cdf(s1) - hat_cdf(s0);
        dw[j] = (hat_pdf(s0) - hat_pdf(s1)) * ir * inv_h;
    }
}

// KIND 0: acc += mass w (push-forward); KIND 1: acc += mass (grad_y w . dp)
// (its tangent); KIND 2: grad = sum_c grad_y w_c F_c (the transpose's seed).
// acc and F are padded image grids.
template <int D, int KIND>
__device__ __noinline__ void pic_hat(const DevGrid& g, const int* I0, const float* u, const float* rho, float* acc,
                                     const float* __restrict__ F, float mass, const float* dp, float* grad) {
    int c0[3] = {0, 0, 0}, n[3] = {1, 1, 1};
    float w[3][kHatMax], dw[3][kHatMax];
    w[2][0] = 1.0f;
    dw[2][0] = 0.0f;
#pragma unroll
    for (int a = 0; a < D; ++a)
        hat_axis(u[a] * g.inv_h[a], rho[a], I0[a], g.m[a], g.inv_h[a], c0[a], n[a], w[a], dw[a]);
    float gsum[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 1
    for (int kz = 0; kz < n[2]; ++kz) {
#pragma unroll 1
        for (int ky = 0; ky < n[1]; ++ky) {
            const float wyz = w[1][ky] * w[2][kz];
            const float dyz = dw[1][ky] * w[2][kz], ydz = w[1][ky] * dw[2][kz];
            int p[3];
            p[1] = I0[1] + c0[1] + ky + LGNK_PAD;
            p[2] = D == 3 ? I0[2] + c0[2] + kz + LGNK_PAD : 0;
#pragma unroll 1
            for (int kx = 0; kx < n[0]; ++kx) {
                p[0] = I0[0] + c0[0] + kx + LGNK_PAD;
                const int o = linear<D>(g, p);
                const float gx = dw[0][kx] * wyz, gy = w[0][kx] * dyz, gz = w[0][kx] * ydz;
                if (KIND == 0) {
                    atomicAdd(acc + o, mass * w[0][kx] * wyz);
                } else if (KIND == 1) {
                    float x = fmaf(gx, dp[0], gy * dp[1]);
                    if (D == 3) x = fmaf(gz, dp[2], x);
                    atomicAdd(acc + o, mass * x);
                } else {
                    const float f = __ldg(F + o);
                    gsum[0] = fmaf(gx, f, gsum[0]);
                    gsum[1] = fmaf(gy, f, gsum[1]);
                    gsum[2] = fmaf(gz, f, gsum[2]);
                }
            }
        }
    }
    if (KIND == 2) {
#pragma unroll
        for (int a = 0; a < D; ++a) grad[a] = gsum[a];
    }
}

// What the forward sweep records of a stage for the adjoint sweep: the
// stage's cell on the velocity grid (linear padded index) and its fractional
// offsets in it, as one 16-byte word (f0, f1, f2 or 0, base).  The adjoint
// then needs no second lookup of the stage position.
template <int D>
__device__ __forceinline__ float4 stage_word(int base, const float* f) {
    return make_float4(f[0], f[1], D == 3 ? f[D - 1] : 0.0f, __int_as_float(base));
}

template <int D>
__device__ __forceinline__ int stage_from_word(const float4 w, float* f) {
    f[0] = w.x;
    f[1] = w.y;
    if (D == 3) f[D - 1] = w.z;
    return __float_as_int(w.w);
}

// The forward sweep: RK4 on the displacement u (Alg. 1 without the
// derivative).  With REC, each stage's cell and offsets are recorded for the
// adjoint sweep (the trajectory is not stored in global memory: the record is
// a per-thread local array).
template <int D, int TM, int FORM, bool REC>
__device__ __forceinline__ void value_sweep(const TraceArgs& A, const VelocityStart<D>& sv, const float* V, float* u,
                                            float4* rec) {
    Cell<D, FORM> C;
    C.key = -1;
    const float dt = A.dt, hdt = 0.5f * A.dt;
#pragma unroll 1
    for (int k = 0; k < A.N; ++k) {
        float us[D], acc[D];
#pragma unroll
        for (int a = 0; a < D; ++a) us[a] = u[a];
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            float f[D];
            const int base = locate_velocity<D>(A.vg, sv, us, f);
            if (REC) rec[4 * k + st] = stage_word<D>(base, f);
            const int m = stage_slice<TM>(k, st), key = m * (int)A.slice_nodes + base;
            cell_at<D, FORM>(A.vg, V, key, C);
            pair2 fd[D - 1];
            if (FORM == CORNERS) dup_offsets_x<D>(f, fd);
            else dup_offsets<D>(f, fd);
#pragma unroll
            for (int q = 0; q < D; ++q) {
                const float v =
                    FORM == CORNERS ? lerp_value<D>(C.e[q], f, fd) : row_value<D>(poly_row<D>(C.e[q], fd), f);
                acc[q] = st == 0 ? v : (st == 3 ? acc[q] + v : fmaf(2.0f, v, acc[q]));
                if (st < 3) us[q] = fmaf(st == 2 ? dt : hdt, v, u[q]);
            }
        }
#pragma unroll
        for (int a = 0; a < D; ++a) u[a] = fmaf(A.dt6, acc[a], u[a]);
    }
}

// The forward sweep with the derivative recursion of Alg. 1 applied to dv:
// D_s = I(dv, y_s, t_s) + d_y I(v, y_s, t_s) (dy + c_s dt D_{s-1}).
template <int D, int TM, int FORM, bool REC>
__device__ __forceinline__ void tangent_sweep(const TraceArgs& A, const VelocityStart<D>& sv, const float* V,
                                              const float* dV, float* u, float* dy, float4* rec) {
    Cell<D, FORM> C;
    Cell<D, POLY> B;
    C.key = -1;           // of both cells
    const float dt = A.dt, hdt = 0.5f * A.dt;
#pragma unroll 1
    for (int k = 0; k < A.N; ++k) {
        float us[D], q[D], acc[D], dacc[D];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            us[a] = u[a];
            q[a] = dy[a];
        }
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            float f[D], vs[D], ds[D], qs[D];
            const int base = locate_velocity<D>(A.vg, sv, us, f);
            if (REC) rec[4 * k + st] = stage_word<D>(base, f);
            const int m = stage_slice<TM>(k, st), key = m * (int)A.slice_nodes + base;
            if (key != C.key) {       // both fields' loads in flight together
                C.key = key;
                pair2 c[D][1 << (D - 1)], b[D][1 << (D - 1)];
                load_corners<D, FORM == CORNERS>(A.vg, V, key, c);
                load_corners<D, false>(A.vg, dV, key, b);
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    if (FORM == CORNERS) {
#pragma unroll
                        for (int j = 0; j < (1 << (D - 1)); ++j) C.e[a][j] = c[a][j];
                    } else {
                        poly_coeffs<D>(c[a], C.e[a]);
                    }
                    poly_coeffs<D>(b[a], B.e[a]);
                }
            }
#pragma unroll
            for (int a = 0; a < D; ++a) qs[a] = q[a] * A.vg.inv_h[a];
            pair2 fd[D - 1];
            dup_offsets<D>(f, fd);
            if constexpr (FORM == CORNERS) {
                pair2 fx[D - 1];
                dup_offsets_x<D>(f, fx);
#pragma unroll
                for (int a = 0; a < D; ++a) vs[a] = lerp_value_dot<D>(C.e[a], f, fx, qs, ds[a]);
            } else {
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    float gr[D];
                    vs[a] = row_value<D>(poly_row<D>(C.e[a], fd), f);
                    poly_grad<D>(C.e[a], f, fd, gr);
                    float jq = gr[D - 1] * qs[D - 1];
#pragma unroll
                    for (int b = D - 2; b >= 0; --b) jq = fmaf(gr[b], qs[b], jq);
                    ds[a] = jq;
                }
            }
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const float d = row_value<D>(poly_row<D>(B.e[a], fd), f) + ds[a];
                acc[a] = st == 0 ? vs[a] : (st == 3 ? acc[a] + vs[a] : fmaf(2.0f, vs[a], acc[a]));
                dacc[a] = st == 0 ? d : (st == 3 ? dacc[a] + d : fmaf(2.0f, d, dacc[a]));
                if (st < 3) {
                    us[a] = fmaf(st == 2 ? dt : hdt, vs[a], u[a]);
                    q[a] = fmaf(st == 2 ? dt : hdt, d, dy[a]);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < D; ++a) {
            u[a] = fmaf(A.dt6, acc[a], u[a]);
            dy[a] = fmaf(A.dt6, dacc[a], dy[a]);
        }
    }
}

// The adjoint sweep: from lam, the adjoint of the end point, scatter every
// stage's contribution and leave in lam the adjoint of the start.  Stages in
// reverse, D_s = I(dv, y_s) + J_s (dy + c_s dt D_{s-1}):
//   mu_4 = dt/6 lam, mu_3 = dt/3 lam + dt nu_4, mu_2 = dt/3 lam + dt/2 nu_3,
//   mu_1 = dt/6 lam + dt/2 nu_2, nu_s = J_s^T mu_s, lam += nu_1 + .. + nu_4
// with J_s^T mu the gradient of the scalar interpolant of v . mu.  The records
// are read one stage ahead of their use: they come from L2 more often than
// from L1 (the records of the resident threads exceed the L1), and the load is
// then in flight during a stage's arithmetic.
template <int D, int TM, int NB, template <int, int> class SC>
__device__ __forceinline__ void adjoint_sweep(const TraceArgs& A, const float* V, SC<D, NB>& S, const float4* rec,
                                              float* lam, Cell<D, POLY>& C) {
    constexpr int NP = 1 << (D - 1);
    const float dt = A.dt, hdt = 0.5f * A.dt, c16 = A.dt6, c13 = 2.0f * A.dt6;
    float4 word = rec[4 * A.N - 1];
#pragma unroll 1
    for (int k = A.N - 1; k >= 0; --k) {
        float nu[D], acc[D];
#pragma unroll
        for (int st = 3; st >= 0; --st) {
            float f[D], mu[D];
            const int base = stage_from_word<D>(word, f);
            word = rec[st > 0 ? 4 * k + st - 1 : max(4 * k - 1, 0)];
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const float c = (st == 1 || st == 2) ? c13 : c16;
                mu[a] = st == 3 ? c * lam[a] : fmaf(c, lam[a], (st == 2 ? dt : hdt) * nu[a]);
            }
            const int m = stage_slice<TM>(k, st);
            cell_at<D, POLY>(A.vg, V, m * (int)A.slice_nodes + base, C);
            pair2 sc[NP];         // coefficients of the scalar interpolant of v . mu
#pragma unroll
            for (int q = 0; q < D; ++q) {
                const pair2 w = pk(mu[q], mu[q]);
#pragma unroll
                for (int j = 0; j < NP; ++j) sc[j] = q == 0 ? mul2(C.e[0][j], w) : fma2(C.e[q][j], w, sc[j]);
            }
            pair2 fd[D - 1];
            dup_offsets<D>(f, fd);
            float gr[D];
            poly_grad<D>(sc, f, fd, gr);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                nu[a] = gr[a] * A.vg.inv_h[a];
                acc[a] = st == 3 ? nu[a] : acc[a] + nu[a];
            }
            if (NB == 2) scatter_add(A.vg, S, A.tj[m] * (int)A.slice_nodes + base, A.tj[m] & 1, A.tth[m], f, mu);
            else scatter_add(A.vg, S, m * (int)A.slice_nodes + base, 0, 0.0f, f, mu);
        }
#pragma unroll
        for (int a = 0; a < D; ++a) lam[a] += acc[a];
    }
}

// The fused Gauss-Newton product of one voxel (RowScatter): the row's sweep,
// then its blocks dotted with the direction and, scaled by h^d J_i dv, into
// the gradients; a row whose blocks did not fit is swept again with the scaled
// seed.
template <int D, int TM, int NB>
__device__ __forceinline__ void gauss_newton_row(const TraceArgs& A, const float* V, RowScatter<D, NB>& S,
                                                 const float4* rec, const float* gT, Cell<D, POLY>& C) {
    constexpr int NV = RowScatter<D, NB>::NV, CAP = RowScatter<D, NB>::CAP;
    S.direct = false;
    S.n = 0;
    S.du = 0.0f;
    float lam[D];
#pragma unroll
    for (int a = 0; a < D; ++a) lam[a] = gT[a];
#pragma unroll 1
    for (;;) {
        adjoint_sweep<D, TM>(A, V, S, rec, lam, C);
        if (S.direct) {
            scatter_finish(A.vg, S);
            return;
        }
        float du = S.du;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            moments_to_corners<D>(S.blk[b]);
            du += block_dot<D>(A.vg, S.dV, block_key(S, b), S.blk[b]);
        }
        const int kept = min(S.n, CAP);
        Block<D> B;
#pragma unroll 1
        for (int j = 0; j < kept; ++j) {
            block_load<D>(S.st + j * NV, B);
            moments_to_corners<D>(B);
            du += block_dot<D>(A.vg, S.dV, S.stkey[j], B);
            block_store<D>(S.st + j * NV, B);
        }
        const float s = A.cellvol * du;
        if (S.n <= CAP) {
#pragma unroll
            for (int b = 0; b < NB; ++b) block_red<D>(A.vg, S.G, block_key(S, b), S.blk[b], s);
#pragma unroll 1
            for (int j = 0; j < S.n; ++j) {
                block_load<D>(S.st + j * NV, B);
                block_red<D>(A.vg, S.G, S.stkey[j], B, s);
            }
            return;
        }
        S.direct = true;
        S.key = -1;
#pragma unroll
        for (int b = 0; b < NB; ++b) block_zero<D>(S.blk[b]);
#pragma unroll
        for (int a = 0; a < D; ++a) lam[a] = s * gT[a];
    }
}

// The same product of one voxel by a tangent sweep, where the rule of pack_many_cells says so (A.many):
// a launch-wide choice, since CTAs of both kinds together evict each other's instructions
// (chosen per warp 778 us where rows alone took 710).
template <int D, int TM, int FORM, int NB>
__device__ __forceinline__ void gauss_newton_tangent(const TraceArgs& A, const int* idx, const VelocityStart<D>& sv,
                                                     float4* rec) {
    const float* V = static_cast<const float*>(A.V);
    float u[D], dy[D], lam[D], du = 0.0f;
#pragma unroll
    for (int a = 0; a < D; ++a) u[a] = dy[a] = 0.0f;
    tangent_sweep<D, TM, FORM, true>(A, sv, V, static_cast<const float*>(A.dV), u, dy, rec);
    Start<D> si;
    start_on_image<D>(idx, si);
    sample_image<D, true>(A.ig, si, A.Tp, u, lam);
#pragma unroll
    for (int a = 0; a < D; ++a) du = fmaf(lam[a], dy[a], du);
#pragma unroll
    for (int a = 0; a < D; ++a) lam[a] *= A.cellvol * du;
    Cell<D, POLY> C;
    C.key = -1;
    BlockScatter<D, NB> S;
    scatter_init(S, A.G, (int)A.slice_nodes);
    adjoint_sweep<D, TM>(A, V, S, rec, lam, C);
    scatter_finish(A.vg, S);
}

// Finish one assembled row: its keys at [e][voxel] (the blocks are already
// in place, [e][voxel][corner][q], written by asm_commit) and its length.
template <int D>
__device__ __forceinline__ void write_row(const TraceArgs& A, const AsmTable<D>& S, int vox) {
    const long long M = (long long)A.ig.m[0] * A.ig.m[1] * (D == 3 ? A.ig.m[2] : 1);
    if (S.overflow || S.n > A.ewidth) {
        A.ecnt[vox] = 0;
        atomicExch(A.eflag, 1);
        return;
    }
    A.ecnt[vox] = S.n;
#pragma unroll 1
    for (int j = 0; j < S.n; ++j) A.ekey[j * M + vox] = S.key[j];
}

// Products with the assembled J, one thread per voxel i (row i):
//   ELL_JVP   out_i = J_i dv = sum_e sum_c blk_e[c] . dV[key_e + corner c]
//   ELL_JTVP  G[key_e + corner c] += r_i blk_e[c]
//   ELL_HESS  both, with the weight h^d (J_i dv) (the Gauss-Newton data term)
// Most rows have one block: the first is loaded without waiting for the row
// length (every row has at least one) and kept in registers for both the
// gather and the scatter; further blocks are read in a loop (twice for HESS).
constexpr int kEllRegBlocks = 1;
// 128-thread CTAs (measured 0.116 -> 0.109 ms against 256 on the 128^3 matvec)
constexpr int kEllBlock = 128;

// 32 bytes from the read-only path in one 256-bit load (p 32-byte aligned)
__device__ __forceinline__ void load8(const float* p, float* v) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
        : "l"(p));
}

// Entry j of row i: its key and its block, read as 256-bit loads (a block is
// 96 bytes in 3D, 32 in 2D, so every block starts on a 32-byte boundary); a
// warp's load then touches half as many L1 wavefronts as with 128-bit loads.
template <int D>
__device__ __forceinline__ void ell_load(const EllArgs& A, long long i, int j, long long& key, float* b) {
    constexpr int B = (1 << D) * D;
    key = __ldg(A.ekey + j * A.M + i);
    const float* p = A.eblk + ((size_t)j * A.M + i) * B;
#pragma unroll
    for (int k = 0; k < B / 8; ++k) load8(p + 8 * k, b + 8 * k);
}

template <int D>
__device__ __forceinline__ float ell_dot(const EllArgs& A, const float* __restrict__ dV, long long key,
                                         const float* b) {
    float s = 0.0f;
#pragma unroll
    for (int r = 0; r < (1 << (D - 1)); ++r) {     // rows of x-pairs (cy, cz); corner (0, cy, cz) is 2 r
        float lo[3], hi[3];
        pair_value<D>(dV, corner_elem<D>(A.vg, (size_t)key, 0, 0, r & 1, r >> 1), lo, hi);
#pragma unroll
        for (int q = 0; q < D; ++q) {
            s = fmaf(b[2 * r * D + q], lo[q], s);
            s = fmaf(b[(2 * r + 1) * D + q], hi[q], s);
        }
    }
    return s;
}

template <int D>
__device__ __forceinline__ void ell_scatter(const EllArgs& A, long long key, const float* b, float w) {
    using VT = typename VecT<D>::type;
    VT* G = static_cast<VT*>(A.G);
#pragma unroll
    for (int c = 0; c < (1 << D); ++c)
        red_vec(G + corner_elem<D>(A.vg, (size_t)key, 0, c & 1, (c >> 1) & 1, (c >> 2) & 1), b + c * D, w);
}

// Scatter of the first blocks of a warp's rows with neighbouring rows merged:
// voxels next to each other in x mostly trace through the same velocity cell
// or the next one along x.  A run of lanes with equal keys adds its weighted
// blocks two by two through shuffles and only the lane at an even position of
// the run reduces (about half the global reductions); then a reducing lane
// whose next reducing lane holds the cell one step along x (key + 1: corner
// (1, cy, cz) of cell k is node k + 1 + cy mx + cz mx my, corner (0, cy, cz)
// of cell k + 1) hands it the four corner vectors of that face and reduces
// only its other four corners.  Every lane of the warp calls it; lanes
// without a block pass a key no other lane has.
template <int D>
__device__ __forceinline__ void ell_scatter_merged(const EllArgs& A, long long key, const float* b, float w) {
    constexpr int C = 1 << D, B = C * D;
    using VT = typename VecT<D>::type;
    VT* G = static_cast<VT*>(A.G);
    const int lane = threadIdx.x & 31;
    const long long prev = __shfl_up_sync(0xffffffffu, key, 1);
    const long long next = __shfl_down_sync(0xffffffffu, key, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || prev != key);
    const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));   // the run's first lane
    const bool absorbed = ((lane - start) & 1) != 0;
    const bool absorber = !absorbed && lane < 31 && next == key;
    float wb[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
        wb[k] = w * b[k];
        const float o = __shfl_down_sync(0xffffffffu, wb[k], 1);
        if (absorber) wb[k] += o;
    }
    const bool reducer = !absorbed && key >= 0;
    const unsigned red = __ballot_sync(0xffffffffu, reducer);
    const unsigned above = lane == 31 ? 0u : red & (0xfffffffeu << lane);
    const unsigned below = red & ((1u << lane) - 1u);
    const int nxt = above != 0u ? __ffs((int)above) - 1 : lane;     // the next and previous reducing lanes
    const int prv = below != 0u ? 31 - __clz((int)below) : lane;
    const long long knext = __shfl_sync(0xffffffffu, key, nxt);
    const long long kprev = __shfl_sync(0xffffffffu, key, prv);
    const bool give = reducer && nxt != lane && knext == key + 1;
    const bool take = reducer && prv != lane && kprev + 1 == key;
#pragma unroll
    for (int c = 1; c < C; c += 2) {
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const float o = __shfl_sync(0xffffffffu, wb[c * D + q], prv);
            if (take) wb[(c - 1) * D + q] += o;
        }
    }
    if (reducer) {
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (!((c & 1) && give))
                red_vec(G + corner_elem<D>(A.vg, (size_t)key, 0, c & 1, (c >> 1) & 1, (c >> 2) & 1), wb + c * D, 1.0f);
    }
}


template <int D, int EMODE>
__global__ void __launch_bounds__(kEllBlock) ell_kernel(const EllArgs A) {
    constexpr int B = (1 << D) * D;
    constexpr int RB = kEllRegBlocks;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < A.M;           // lanes past the end stay for the warp's shuffles
    const float* dV = static_cast<const float*>(A.dV);
    const int n = valid ? __ldg(A.ecnt + i) : 0;
    long long kr[RB > 0 ? RB : 1];
    float br[RB > 0 ? RB : 1][B];
#pragma unroll
    for (int j = 0; j < RB; ++j)
        if (valid && (j == 0 || j < n)) ell_load<D>(A, i, j, kr[j], br[j]);
    float s = 0.0f;
    if (EMODE != ELL_JTVP) {
#pragma unroll
        for (int j = 0; j < RB; ++j)
            if (j < n) s += ell_dot<D>(A, dV, kr[j], br[j]);
#pragma unroll 1
        for (int j = RB; j < n; ++j) {
            long long k;
            float b[B];
            ell_load<D>(A, i, j, k, b);
            s += ell_dot<D>(A, dV, k, b);
        }
        if (EMODE == ELL_JVP) {
            if (valid) A.out[i] = s;
            return;
        }
        s *= A.cellvol;
    } else {
        s = valid ? A.r[i] : 0.0f;
    }
    // the first block: merged across the warp; keys are non-negative element offsets
    ell_scatter_merged<D>(A, n > 0 ? kr[0] : -1 - (long long)(threadIdx.x & 31), br[0], s);
#pragma unroll
    for (int j = 1; j < RB; ++j)
        if (j < n) ell_scatter<D>(A, kr[j], br[j], s);
#pragma unroll 1
    for (int j = RB; j < n; ++j) {
        long long k;
        float b[B];
        ell_load<D>(A, i, j, k, b);
        ell_scatter<D>(A, k, b, s);
    }
}

template <int D>
static cudaError_t launch_ell_dim(int mode, const EllArgs& a, cudaStream_t s) {
    const long long blocks = (a.M + kEllBlock - 1) / kEllBlock;
    if (blocks < 1 || blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    switch (mode) {
        case ELL_JVP: ell_kernel<D, ELL_JVP><<<(unsigned)blocks, kEllBlock, 0, s>>>(a); break;
        case ELL_JTVP: ell_kernel<D, ELL_JTVP><<<(unsigned)blocks, kEllBlock, 0, s>>>(a); break;
        case ELL_HESS: ell_kernel<D, ELL_HESS><<<(unsigned)blocks, kEllBlock, 0, s>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Threads of a CTA and CTAs per SM that the register budget is set for.  A CTA
// covers a tile of voxels where it writes the tile's partial sums and half a
// tile where nothing is summed: 465 -> 454 us for the 128^3 product by rows, 6.29
// -> 6.10 ms for the brain-scale J^T, from the shorter wait for a CTA's last
// warp.  The 3D kernels hold a cell's coefficients and a pending block (24
// registers each, 48 for the two nodes of a time cell) and run at 128
// registers: at 96 they spill (the brain-scale J^T 8.2 ms), at 168 too few warps
// run (7.0 ms).  The forward sweep holds the coefficients only and runs at 80.
template <int D, int TM, int MODEL, int MODE>
struct TraceOccupancy {
    static constexpr int threads =
        MODE == MODE_JTVP || MODE == MODE_HESS || MODE == MODE_HROW ? LGNK_BLOCK / 2 : LGNK_BLOCK;
    static constexpr int ctas = D == 3 ? (MODE == MODE_FWD ? 3 : 2) : (MODE == MODE_FWD ? 4 : 3);
    static constexpr int value = ctas * (LGNK_BLOCK / threads);
};

template <int D, int TM, int MODEL, int MODE>
__global__ void
__launch_bounds__((TraceOccupancy<D, TM, MODEL, MODE>::threads), (TraceOccupancy<D, TM, MODEL, MODE>::value))
    trace_kernel(const TraceArgs A) {
    constexpr int THREADS = TraceOccupancy<D, TM, MODEL, MODE>::threads;
    constexpr bool TRANSPORT = MODEL == LGNK_TRANSPORT;
    constexpr int FORM = TRANSPORT ? POLY : CORNERS;
    constexpr bool ROWS = MODE == MODE_HROW;
    constexpr bool TANGENT = MODE == MODE_JVP || MODE == MODE_HESS;
    constexpr bool ADJOINT = MODE != MODE_FWD && MODE != MODE_JVP;
    constexpr int NB = TM == TM_NODES ? 2 : 1;
    using BS = typename std::conditional<TRANSPORT, BlockScatter<D, NB>, CornerScatter<D, NB>>::type;
    using SC = typename std::conditional<MODE == MODE_ASM, AsmRow<D, NB>,
                                         typename std::conditional<ROWS, RowScatter<D, NB>, BS>::type>::type;
    const float* V = static_cast<const float*>(A.V);
    const float* dV = static_cast<const float*>(A.dV);
    lsum ssd = lsum_zero();  // res^2 of this thread's voxel (FWD with R, OBJGRAD, ASM with R)
    int entries = 0;         // MODE_ASM: blocks of this thread's row

    bool far = false;         // MODE_HROW: by tangent sweeps after all
    if constexpr (ROWS) far = *A.many != 0;
    int idx[3];
    voxel_index<D>(A, THREADS, idx);
    const bool active = idx[0] < A.ig.m[0] && idx[1] < A.ig.m[1] && (D == 2 || idx[2] < A.ig.m[2]);
    int sp[D];                // continuity FWD / JVP: the end cell, offsets, mass and dy of the splat
    float sf[D], sdy[D], smass = 0.0f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        sp[a] = 0;
        sf[a] = 0.0f;
        sdy[a] = 0.0f;
    }
    if (active) {
        const int vox = idx[0] + A.ig.m[0] * (idx[1] + A.ig.m[1] * (D == 3 ? idx[2] : 0));
        float u[D], dy[D];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            u[a] = 0.0f;
            dy[a] = 0.0f;
        }
        VelocityStart<D> sv;
        start_on_velocity<D>(A, idx, sv);
        // the stages, recorded for the adjoint sweep in a per-thread local
        // array.  Kept in shared memory instead, the record shrank the L1
        // that the gathers use and measured slower (0.828 against 0.814 ms
        // for an earlier 128^3 product).
        float4 rec[ADJOINT ? 4 * LGNK_MAX_STEPS : 1];
        if constexpr (ROWS) {
            if (far) {
                gauss_newton_tangent<D, TM, FORM, NB>(A, idx, sv, rec);
                return;
            }
        }
        if constexpr (TANGENT) tangent_sweep<D, TM, FORM, ADJOINT>(A, sv, V, dV, u, dy, rec);
        else value_sweep<D, TM, FORM, ADJOINT>(A, sv, V, u, rec);
        if (A.yout != nullptr) {
            const int M = A.ig.m[0] * A.ig.m[1] * (D == 3 ? A.ig.m[2] : 1);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const float xc = A.ig.lo[a] + ((float)idx[a] + 0.5f) * A.ig.h[a];
                A.yout[(size_t)a * M + vox] = xc + u[a];
            }
        }

        float lam[D];
        Start<D> si;
        start_on_image<D>(idx, si);
        if constexpr (TRANSPORT) {
            if constexpr (MODE == MODE_FWD) {
                const float val = sample_image<D, false>(A.ig, si, A.Tp, u, nullptr);
                A.u1[vox] = val;
                if (A.R != nullptr) lsum_add_sqdiff(ssd, val, A.R[vox]);
            } else {
                float gT[D];
                const float val = sample_image<D, true>(A.ig, si, A.Tp, u, gT);
                if constexpr (TANGENT) {
                    float du = 0.0f;
#pragma unroll
                    for (int a = 0; a < D; ++a) du = fmaf(gT[a], dy[a], du);
                    if (MODE == MODE_JVP) A.u1[vox] = du;
                    const float s = A.cellvol * du;      // MODE_HESS: the seed h^d J dv
#pragma unroll
                    for (int a = 0; a < D; ++a) lam[a] = s * gT[a];
                } else {
                    float s = 1.0f;                      // MODE_HROW and MODE_ASM: the row of J
                    if (MODE == MODE_JTVP) s = A.r[vox];
                    if (MODE == MODE_OBJGRAD || (MODE == MODE_ASM && A.R != nullptr)) {
                        const float Rv = A.R[vox];
                        lsum_add_sqdiff(ssd, val, Rv);
                        const float w = A.cellvol * (val - Rv);
                        if (MODE == MODE_ASM) A.u1[vox] = w;     // the gradient's weights h^d res
                        else s = w;
                    }
#pragma unroll
                    for (int a = 0; a < D; ++a) lam[a] = s * gT[a];
                }
            }
        } else {
            const float mass = __ldg(A.T + vox);
            if (A.pic_rho[0] > 0.0f) {
                if (MODE == MODE_FWD) {
                    pic_hat<D, 0>(A.ig, si.I0, u, A.pic_rho, A.acc, nullptr, mass, nullptr, nullptr);
                } else if (MODE == MODE_JVP) {
                    pic_hat<D, 1>(A.ig, si.I0, u, A.pic_rho, A.acc, nullptr, mass, dy, nullptr);
                } else if (MODE == MODE_JTVP) {
                    float gr[D];
                    pic_hat<D, 2>(A.ig, si.I0, u, A.pic_rho, nullptr, A.r, 0.0f, nullptr, gr);
#pragma unroll
                    for (int a = 0; a < D; ++a) lam[a] = mass * gr[a];
                }
            } else if (MODE == MODE_FWD || MODE == MODE_JVP) {
                locate<D>(A.ig, si, u, sp, sf);   // splat after the trace, with the whole CTA
                smass = mass;
#pragma unroll
                for (int a = 0; a < D; ++a) sdy[a] = dy[a];
            } else if (MODE == MODE_JTVP) {
                float gr[D];
                sample_image<D, true>(A.ig, si, A.r, u, gr);
#pragma unroll
                for (int a = 0; a < D; ++a) lam[a] = mass * gr[a];
            }
        }

        if constexpr (ADJOINT) {
            Cell<D, POLY> C;
            C.key = -1;
            SC S;
            scatter_init(S, A.G, (int)A.slice_nodes);
            if constexpr (ROWS) {
                float4 rowst[RowScatter<D, NB>::CAP * RowScatter<D, NB>::NV];
                int rowkey[RowScatter<D, NB>::CAP];
                S.dV = dV;
                S.st = rowst;
                S.stkey = rowkey;
                gauss_newton_row<D, TM>(A, V, S, rec, lam, C);
            } else if constexpr (MODE == MODE_ASM) {
                AsmTable<D> row_table;        // the keys of the row being assembled
                row_table.n = 0;
                row_table.overflow = false;
                S.tab = &row_table;
                const size_t Mi = (size_t)A.ig.m[0] * A.ig.m[1] * (D == 3 ? A.ig.m[2] : 1);
                S.stride = Mi * AsmRow<D, NB>::B;
                S.row = A.eblk + (size_t)vox * AsmRow<D, NB>::B;
                adjoint_sweep<D, TM>(A, V, S, rec, lam, C);
                scatter_finish(A.vg, S);
                write_row<D>(A, row_table, vox);
                entries = row_table.n;
            } else {
                adjoint_sweep<D, TM>(A, V, S, rec, lam, C);
                scatter_finish(A.vg, S);
            }
        }
    }
    if constexpr (!TRANSPORT && (MODE == MODE_FWD || MODE == MODE_JVP)) {
        if (A.pic_rho[0] <= 0.0f) splat_tiled<D, MODE == MODE_JVP>(A.ig, A.acc, active, sp, sf, smass, sdy);
    }

    if constexpr (TRANSPORT && (MODE == MODE_OBJGRAD || MODE == MODE_FWD || MODE == MODE_ASM)) {
        if (A.partial != nullptr) {
            const lsum s = lsum_block_sum(ssd);
            if (threadIdx.x == 0) A.partial[blockIdx.x] = lsum_value(s);
        }
    }
    if constexpr (MODE == MODE_ASM) {
        if (A.cpartial != nullptr) {
            __shared__ int rowsum[THREADS / 32];
            const int w = __reduce_add_sync(0xffffffffu, entries);
            if ((threadIdx.x & 31) == 0) rowsum[threadIdx.x >> 5] = w;
            __syncthreads();
            if (threadIdx.x == 0) {
                int c = 0;
#pragma unroll
                for (int i = 0; i < THREADS / 32; ++i) c += rowsum[i];
                A.cpartial[blockIdx.x] = (double)c;
            }
        }
    }
}

template <int D, int TM, int MODEL, int MODE>
static cudaError_t launch_one(const TraceArgs& a0, cudaStream_t s) {
    TraceArgs a = a0;
    int ts[3];
    trace_tile_shape(D, ts);
    for (int i = 0; i < 3; ++i) a.tiles[i] = (a.ig.m[i] + ts[i] - 1) / ts[i];
    const int blocks = a.tiles[0] * a.tiles[1] * a.tiles[2];
    constexpr int threads = TraceOccupancy<D, TM, MODEL, MODE>::threads;
    trace_kernel<D, TM, MODEL, MODE><<<blocks * (LGNK_BLOCK / threads), threads, 0, s>>>(a);
    return cudaGetLastError();
}

template <int D, int TM>
static cudaError_t launch_dim(int model, int mode, const TraceArgs& a, cudaStream_t s) {
    if (model == LGNK_TRANSPORT) {
        switch (mode) {
            case MODE_FWD: return launch_one<D, TM, LGNK_TRANSPORT, MODE_FWD>(a, s);
            case MODE_JVP: return launch_one<D, TM, LGNK_TRANSPORT, MODE_JVP>(a, s);
            case MODE_JTVP: return launch_one<D, TM, LGNK_TRANSPORT, MODE_JTVP>(a, s);
            case MODE_HESS: return launch_one<D, TM, LGNK_TRANSPORT, MODE_HESS>(a, s);
            case MODE_HROW:
                if constexpr (D == 3 && TM == TM_STEADY) return launch_one<D, TM, LGNK_TRANSPORT, MODE_HROW>(a, s);
                break;
            case MODE_OBJGRAD: return launch_one<D, TM, LGNK_TRANSPORT, MODE_OBJGRAD>(a, s);
            case MODE_ASM:      // rows are kept per (slice, cell)
                if constexpr (TM != TM_NODES) return launch_one<D, TM, LGNK_TRANSPORT, MODE_ASM>(a, s);
                break;
        }
    } else {
        switch (mode) {
            case MODE_FWD: return launch_one<D, TM, LGNK_CONTINUITY, MODE_FWD>(a, s);
            case MODE_JVP: return launch_one<D, TM, LGNK_CONTINUITY, MODE_JVP>(a, s);
            case MODE_JTVP: return launch_one<D, TM, LGNK_CONTINUITY, MODE_JTVP>(a, s);
        }
    }
    return cudaErrorInvalidValue;
}

template <int D>
static cudaError_t launch_trace_dim(TimeMode tm, int model, int mode, const TraceArgs& a, cudaStream_t s) {
    switch (tm) {
        case TM_STEADY: return launch_dim<D, TM_STEADY>(model, mode, a, s);
        case TM_SLICES: return launch_dim<D, TM_SLICES>(model, mode, a, s);
        case TM_NODES: return launch_dim<D, TM_NODES>(model, mode, a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lgnk
