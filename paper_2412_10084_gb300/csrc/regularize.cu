// Grid-level training terms of ProbeSDF (Sec. 3.3, Eqs. 11-15).
//
//   smooth_kernel         s = G(s_hat): 5^3 Gaussian (sigma = 1 node, separable,
//                         replicated edge nodes), or G^T with the transposed 1D
//                         operators (edge outputs gather the replicated taps)
//   sdf_reg_kernel        L_sdf, L_Eik and L_normal on the smoothed SDF, their
//                         gradients scaled by (1 + 5 |s|)^-1: the
//                         central-difference adjoint as a gather
//                         (both z-streaming, on dense grids and on sparse
//                         16^3-node bricks behind a brick table)
//   plane_reg_kernel      L_features: forward differences inside each tile plane
//   probe_reg_kernel      L_probes: ordered pairs of 6-neighbour probes
//
// Streaming stencils over HBM-resident grids; loss values are summed per CTA
// and added to device accumulators.
#include <cmath>
#include <type_traits>

#include "internal.h"

namespace psdf {

namespace {

// ---------------------------------------------------------------------------
// z-streaming stencils.  A CTA owns an OX x OY column tile and walks z; every
// thread owns one (x, y) column of the tile or of its halo.  Neighbours along
// z are the thread's own registers, neighbours in the plane come from shared
// memory.  Stage k of a plane runs one step after stage k - 1, on what the step
// before wrote (two buffers per stage), so a step has a single barrier.
// ---------------------------------------------------------------------------

constexpr int HALO = 2;      // smoothing: 5 taps
constexpr int REG_HALO = 3;  // regularisers: s -> normal -> gradient -> output
constexpr int SB = 16;       // brick edge

struct Taps {
    float w[5];
};

__device__ __forceinline__ int clampi(int v, int lo, int hi)
{
    return v < lo ? lo : (v > hi ? hi : v);
}

// Columns of a tile in order of their distance to it: the OX x OY outputs
// first, then ring 1, 2, .. of the halo (top row, bottom row, the two sides).
// A stage that needs fewer columns than the one before thus leaves whole warps
// out instead of the border lanes of every row.
template <int OX_, int OY_, int H_>
struct Tile {
    static constexpr int OX = OX_, OY = OY_, H = H_;
    static constexpr int kCols = (OX + 2 * H) * (OY + 2 * H);  // columns, halo included
    static constexpr int kThreads = (kCols + 31) & ~31;
    // columns within ring r
    static __host__ __device__ constexpr int cols(int r) { return (OX + 2 * r) * (OY + 2 * r); }
    static __device__ __forceinline__ void column(int e, int& x, int& y)
    {
        if (e < OX * OY) {
            x = e % OX;
            y = e / OX;
            return;
        }
        e -= OX * OY;
#pragma unroll
        for (int r = 1; r <= H; ++r) {
            const int w = OX + 2 * r, n = 2 * w + 2 * (OY + 2 * r) - 4;
            if (e < n) {
                if (e < 2 * w) {
                    x = e % w - r;
                    y = e < w ? -r : OY - 1 + r;
                } else {
                    e -= 2 * w;
                    x = (e & 1) ? OX - 1 + r : -r;
                    y = 1 - r + (e >> 1);
                }
                return;
            }
            e -= n;
        }
        x = y = 0;  // threads past the last column: never used
    }
};

// Dense tiles: 32 outputs in x keep the rows of every array whole 128-byte
// lines.  Brick tiles: a brick's 16 x 16 columns.
using DenseSmooth = Tile<32, 16, HALO>;
using BrickSmooth = Tile<SB, SB, HALO>;
using DenseReg = Tile<32, 16, REG_HALO>;
using BrickReg = Tile<SB, SB, REG_HALO>;

// Where a kernel's planes lie.  Dense: node (x, y, z) is element
// (z Ry + y) Rx + x, and CTA z covers planes [z zc, z zc + zc).  Sparse bricks:
// node `local` of slot b is element b * 4096 + local; a CTA owns `seg` <= kMaxSeg bricks
// of a brick column, whose stored bricks it walks run by run.
struct Domain {
    int R[3];
    int zc;
    const int* table;  // [B2][B1][B0]: slot, or -1 (outside [0, n_bricks) counts as absent)
    int B[3], n_bricks, seg;
};

constexpr int kMaxSeg = 8;

// Slots of the brick columns that a CTA's tile and halo lie in: its own and its
// 8 neighbours, from the brick below its segment to the one above (-1: absent or
// outside the grid).  Read once, all entries at a time: the walks then look
// slots up in shared memory instead of waiting for the table brick after brick.
struct SlotTable {
    int slot[9][kMaxSeg + 2];
};

template <bool SPARSE>
__device__ __forceinline__ void load_slots(const Domain& D, SlotTable& S)
{
    if constexpr (SPARSE) {
        const int n = D.seg + 2;
        for (int i = threadIdx.x; i < 9 * n; i += blockDim.x) {
            const int c = i / n, k = i % n;
            const int x = blockIdx.x + c % 3 - 1, y = blockIdx.y + c / 3 - 1;
            const int z = blockIdx.z * D.seg + k - 1;
            int s = -1;
            if (x >= 0 && x < D.B[0] && y >= 0 && y < D.B[1] && z >= 0 && z < D.B[2])
                s = __ldg(D.table + (int64_t(z) * D.B[1] + y) * D.B[0] + x);
            S.slot[c][k] = s < D.n_bricks ? max(s, -1) : -1;
        }
        __syncthreads();
    }
}

// The next run of planes [z0, z1) of this CTA, from `at` on (a brick, sparse;
// negative: from the start); false when there is none.  CTA-uniform.
template <bool SPARSE>
__device__ __forceinline__ bool next_run(const Domain& D, const SlotTable& S, int& at, int& z0,
                                         int& z1)
{
    if constexpr (!SPARSE) {
        if (at >= 0) return false;
        at = 0;
        z0 = blockIdx.z * D.zc;
        z1 = min(z0 + D.zc, D.R[2]);
        return true;
    } else {
        const int first = blockIdx.z * D.seg, last = min(first + D.seg, D.B[2]);
        const int* own = S.slot[4] + 1 - first;
        int b = at < 0 ? first : at;
        while (b < last && own[b] < 0) ++b;
        if (b >= last) return false;
        int e = b + 1;
        while (e < last && own[e] >= 0) ++e;
        at = e;
        z0 = b * SB;
        z1 = e * SB;
        return true;
    }
}

// A thread's column, walked plane by plane: `e` is the node of the current
// plane in the arrays, -1 where it is not stored (sparse: its brick is absent).
template <bool SPARSE>
struct Walk {
    int e;
    int step;          // nodes between planes
    int xy;            // offset inside a plane
    const int* slots;  // sparse: the slots of the column's bricks, by brick
    // column (x, y), inside the grid
    __device__ __forceinline__ Walk(const Domain& D, const SlotTable& S, int x, int y)
    {
        if constexpr (SPARSE) {
            const int c = ((y >> 4) - int(blockIdx.y) + 1) * 3 + (x >> 4) - int(blockIdx.x) + 1;
            slots = S.slot[c] + 1 - int(blockIdx.z) * D.seg;
            xy = ((y & 15) << 4) | (x & 15);
            step = 256;
        } else {
            xy = y * D.R[0] + x;
            step = D.R[0] * D.R[1];
        }
        e = -1;
    }
    // to plane z (inside the grid)
    __device__ __forceinline__ void seek(const Domain& D, int z)
    {
        if constexpr (SPARSE) {
            const int slot = slots[z >> 4];
            e = slot < 0 ? -1 : slot * 4096 + ((z & 15) << 8) + xy;
        } else {
            e = z * step + xy;
        }
    }
    // from plane z - 1 to plane z, both inside the grid
    __device__ __forceinline__ void next(const Domain& D, int z)
    {
        if (SPARSE && (z & 15) == 0)
            seek(D, z);
        else if (!SPARSE || e >= 0)
            e += step;
    }
};

using Yes = std::true_type;
using No = std::false_type;

// 1D pass of 5 taps.  Transposed, at output node k of an axis of n nodes: v0 .. v4 are input
// nodes k - 2 .. k + 2 (0 outside the grid).  Inside the axis, output k takes
// input i with the weight w[k - i + 2] that the forward gave input k in output
// i; the replicated edge taps add (w0 + w1) x in[0] + w0 x in[1] at k = 0 and
// (w3 + w4) x in[n-1] + w4 x in[n-2] at k = n - 1 (`first`, `last`).
template <bool TRANSPOSE>
__device__ __forceinline__ float conv5(float v0, float v1, float v2, float v3, float v4,
                                       bool first, bool last, const Taps& T)
{
    if constexpr (!TRANSPOSE) {
        return fmaf(T.w[4], v4,
                    fmaf(T.w[3], v3, fmaf(T.w[2], v2, fmaf(T.w[1], v1, T.w[0] * v0))));
    } else {
        float acc = fmaf(T.w[0], v4,
                         fmaf(T.w[1], v3, fmaf(T.w[2], v2, fmaf(T.w[3], v1, T.w[4] * v0))));
        if (first) acc = fmaf(T.w[0] + T.w[1], v2, fmaf(T.w[0], v3, acc));
        if (last) acc = fmaf(T.w[3] + T.w[4], v2, fmaf(T.w[4], v1, acc));
        return acc;
    }
}

struct Smooth {
    Domain D;
    const float* in;  // element e at in[e * in_stride]
    int in_stride;
    float* out;       // likewise
    int out_stride;
    float empty;      // sparse, forward: the value of a node of an absent brick
    int accumulate;
};

// s = G(s_hat) or G^T.  What a node costs beyond memory is one load, two
// 5-tap passes over shared memory (x, then y) and one over registers (z); the
// next four planes (and what the outputs add to) are in flight meanwhile.
//
// Bound: HBM, by the 4-byte SDF slots of the 16-byte records (whole sectors are
// moved: 0.57 GB for a 256^3 grid).  Measured on 256^3 node records: s 93 us,
// G^T 95 us (a 32 x 8 x 8 tile with its halo gathered at once: 109 and 155 us);
// on 47.6 M stored nodes of a 512^3 grid 285 and 302 us (20^3 tiles gathered per
// brick with an index division per element: 573 and 774 us).
//
// Outside the grid the forward reads the replicated edge node and the
// transpose 0; in an absent brick the forward reads `empty` and the transpose
// 0 (an absent node's s is fixed, so it carries no gradient).
template <class T, bool SPARSE, bool TRANSPOSE>
__global__ void __launch_bounds__(T::kThreads, SPARSE ? 3 : 2) smooth_kernel(Smooth P, Taps taps)
{
    // row pitch of the shared planes: 16-wide rows, two to a warp, fall on
    // different halves of the banks
    constexpr int W = T::OX == 16 ? 48 : T::OX + 2 * HALO;
    __shared__ float S[2][W * (T::OY + 2 * HALO)];  // loaded plane
    __shared__ float X[2][W * (T::OY + 2 * HALO)];  // after the x pass
    __shared__ SlotTable slots;
    const Domain& D = P.D;
    load_slots<SPARSE>(D, slots);
    const int x0 = blockIdx.x * T::OX, y0 = blockIdx.y * T::OY;
    int lx, ly;
    T::column(threadIdx.x, lx, ly);
    const bool mine = threadIdx.x < T::kCols;
    const int gx = x0 + lx, gy = y0 + ly;
    const int pos = (ly + HALO) * W + lx + HALO;
    const bool do_x = mine && lx >= 0 && lx < T::OX;
    const bool do_y = threadIdx.x < T::OX * T::OY;
    const bool do_out = do_y && gx < D.R[0] && gy < D.R[1];
    const bool in_xy = gx >= 0 && gx < D.R[0] && gy >= 0 && gy < D.R[1];
    const bool reads = mine && (!TRANSPOSE || in_xy);
    const int cx = clampi(gx, 0, D.R[0] - 1), cy = clampi(gy, 0, D.R[1] - 1);
    Walk<SPARSE> in(D, slots, cx, cy), ahead(D, slots, cx, cy), out(D, slots, cx, cy);
    const float none = TRANSPOSE ? 0.0f : P.empty;
    auto value = [&]() -> float {
        return reads && (!SPARSE || in.e >= 0) ? __ldg(P.in + int64_t(in.e) * P.in_stride) : none;
    };
    auto edge_value = [&](int z) -> float {
        return TRANSPOSE && (z < 0 || z >= D.R[2]) ? 0.0f : value();
    };
    int at = -1, z0, z1;
    while (next_run<SPARSE>(D, slots, at, z0, z1)) {
        // planes z0 - 2 .. z1 + 1 enter, kAhead of them in flight.  The x pass
        // of plane z runs in step z, the y pass in step z + 2, and output plane
        // z leaves in step z + 4.  The loop is unrolled over the period of the
        // register rings (5) and of the shared buffers (2); steps away from the
        // ends of the run and of the grid test no plane index.
        constexpr int kAhead = 4;
        float v[5], r[5];  // loaded planes; planes after the y pass
        float old[5];      // what the outputs add to
        const int zb = z0 - HALO;
        in.seek(D, max(zb, 0));
        v[0] = edge_value(zb);
#pragma unroll
        for (int i = 1; i < kAhead; ++i) {
            if (zb + i > 0 && zb + i < D.R[2]) in.next(D, zb + i);
            v[i] = edge_value(zb + i);
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) r[i] = old[i] = 0.0f;
        out.seek(D, z0);
        ahead.seek(D, z0);
        auto step = [&](auto inner, int u, int z) {
            constexpr bool kInner = decltype(inner)::value;
            if (mine) S[u & 1][pos] = v[u % 5];
            if (kInner || z + kAhead < z1 + HALO) {
                if (kInner || (z + kAhead > 0 && z + kAhead < D.R[2])) in.next(D, z + kAhead);
                v[(u + kAhead) % 5] = kInner ? value() : edge_value(z + kAhead);
            }
            if (P.accumulate && do_out && (kInner || (z >= z0 && z < z1))) {
                if (z > z0) ahead.next(D, z);
                old[u % 5] = P.out[int64_t(ahead.e) * P.out_stride];
            }
            const int zo = z - 4;
            if (do_y) {
                const float* c = &X[u & 1][pos];  // the x pass of plane z - 2
                r[u % 5] = conv5<TRANSPOSE>(c[-2 * W], c[-W], c[0], c[W], c[2 * W],
                                            gy == 0, gy == D.R[1] - 1, taps);
            }
            if (do_out && (kInner || zo >= z0)) {
                P.out[int64_t(out.e) * P.out_stride] =
                    old[(u + 1) % 5] + conv5<TRANSPOSE>(r[(u + 1) % 5], r[(u + 2) % 5], r[(u + 3) % 5],
                                           r[(u + 4) % 5], r[u % 5], !kInner && zo == 0,
                                           !kInner && zo == D.R[2] - 1, taps);
                if (kInner || zo + 1 < z1) out.next(D, zo + 1);
            }
            __syncthreads();  // plane z is in S; the x pass's buffer is read
            if (do_x) {
                const float* c = &S[u & 1][pos];
                X[u & 1][pos] = conv5<TRANSPOSE>(c[-2], c[-1], c[0], c[1], c[2], gx == 0,
                                                 gx == D.R[0] - 1, taps);
            }
        };
        const int lo = z0 + 5, hi = min(z1 + HALO, D.R[2]) - kAhead;  // inner steps [lo, hi)
        for (int zs = zb; zs < z1 + 4; zs += 10) {
#pragma unroll
            for (int u = 0; u < 10; ++u) {
                const int z = zs + u;
                if (z >= z1 + 4) break;
                if (z >= lo && z < hi)
                    step(Yes(), u, z);
                else
                    step(No(), u, z);
            }
        }
        __syncthreads();  // the last reads of S and X, before the next run's writes
    }
}

// Block sum of up to three loss partials, added to acc[0..n-1] (skipped when acc is null).
__device__ __forceinline__ void block_loss(float a, float b, float c, float* acc, int n)
{
    __shared__ float part[3][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
        c += __shfl_xor_sync(0xffffffffu, c, off);
    }
    if (lane == 0) {
        part[0][warp] = a;
        part[1][warp] = b;
        part[2][warp] = c;
    }
    __syncthreads();
    if (acc && threadIdx.x < n) {
        float s = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += part[threadIdx.x][w];
        atomicAdd(acc + threadIdx.x, s);
    }
    __syncthreads();
}

// 1 / x for 1 <= x, and 1 / sqrt(x) for x in [1e-16, 1e30): the hardware's
// approximations with one Newton-Raphson step.  Over all mantissas the first is
// 1.0f / x to the bit below 1e30 (from there on, |s| past 2e29, it is the
// approximation alone: squares of such values have no FP32), the second at most 1.00
// units in the last place off (1.0f / sqrtf(x): 1.49).  The root itself is sqrtf: x
// times the second was up to 0.75 units off and not the nearest in 12 % of the cases.
__device__ __forceinline__ float reciprocal(float x)
{
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return x < 1e30f ? fmaf(r, fmaf(-x, r, 1.0f), r) : r;
}

__device__ __forceinline__ float inverse_root(float x)
{
    float r;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    const float e = fmaf(-(x * r), r, 1.0f);  // 1 - x r^2
    return fmaf(0.5f * r, e, r);
}

// Asynchronous 4-byte copies into shared memory, in groups of one step.
__device__ __forceinline__ void copy_async4(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}

__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// All but the newest N groups of this thread have landed.
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

struct SdfReg {
    Domain D;
    const float* s_hat;  // element e at s_hat[e]
    const float* s;      // smoothed, element stride s_stride
    int s_stride;
    float* d_s;          // gradient w.r.t. s (accumulated), stride d_stride
    int d_stride;
    float* d_s_hat;      // gradient w.r.t. s_hat (accumulated), laid out as s_hat
    float* loss;         // [3]: L_sdf, L_Eik, L_normal (accumulated)
    float inv2h[3];      // 1 / (2 h_a)
    float lam_sdf, lam_eik, lam_normal;
    float empty;         // sparse: the value of a node of an absent brick
};

// L_sdf, L_Eik and L_normal with their gradients, z-streaming.  Step z loads s
// plane z, computes N = {normal, voxel weight} of plane z - 1, G = dObjective /
// d(grad s) of plane z - 2 and the outputs of plane z - 3:
//   ds_i = own L_sdf term + sum_a (G_a(i - e_a) - G_a(i + e_a)) / 2h_a
// (the central-difference adjoint as a gather, so every output has one writer
// and no atomics are needed).  A node that is not interior has no normal; its
// weight is stored as -1.
//
// Bound: issue (73 % of the slots) and, on bricks, the serial chain of a step;
// HBM would take 0.15 ms at 256^3.  s and the own values arrive by asynchronous
// copies three planes ahead, which cost no registers.  Steps and warps whose
// columns and planes all lie inside take straight-line code.  Measured: 256^3
// 0.268 ms (0.421 with three barriers a plane and every neighbour read from
// shared memory), 47.6 M stored nodes of a 512^3 grid 1.14 ms (1.29 ms).  Dense
// tile: 32 x 16 outputs in 864 threads, 1 CTA per SM; 32 x 12 and 32 x 8 with 2
// CTAs recompute more halo (0.29 and 0.38 ms).
//
// Sparse bricks: s is that of the full grid with every node of an absent brick
// at `empty` (as the render and the smoothing read it), and the terms are those
// of the stored nodes: an absent node gets voxel weight 0, so its own Eikonal
// term and the normal pairs it owns add nothing, while its normal still enters
// the pairs its stored neighbours own.  Gradients are written for the stored
// nodes only (an absent node's s is not a parameter).
template <class T>
struct RegSmem {
    static constexpr int H = REG_HALO;
    static constexpr int kOwn = T::OX * T::OY;
    // row pitches: of s, two 16-wide rows of a warp on different halves of the
    // banks; of N (whole 16-byte lanes) and G, the row itself
    static constexpr int kWS = T::OX == 16 ? 48 : T::OX + 2 * H, kWN = T::OX + 2 * H;
    float4 N[2][T::kCols];
    float2 G[2][T::kCols];
    float s[6][kWS * (T::OY + 2 * H)];  // planes z - 1 .. z + 3
    float own[3][6][kOwn];              // s_hat and d s_hat of plane z - 1, d s of plane z - 3
};

template <class T, bool SPARSE>
__global__ void __launch_bounds__(T::kThreads, SPARSE ? 2 : 1) sdf_reg_kernel(SdfReg P)
{
    using M = RegSmem<T>;
    constexpr int H = REG_HALO, kWS = M::kWS, kWN = M::kWN;
    constexpr int kAhead = 3;  // planes in flight
    extern __shared__ __align__(16) uint8_t reg_smem[];
    M& S = *reinterpret_cast<M*>(reg_smem);
    __shared__ SlotTable slots;
    const Domain& D = P.D;
    load_slots<SPARSE>(D, slots);
    const int x0 = blockIdx.x * T::OX, y0 = blockIdx.y * T::OY;
    const int Rx = D.R[0], Ry = D.R[1], Rz = D.R[2];
    int lx, ly;
    T::column(threadIdx.x, lx, ly);
    const int tid = threadIdx.x;
    const int gx = x0 + lx, gy = y0 + ly;
    const int pos = (ly + H) * kWN + lx + H, pos_s = (ly + H) * kWS + lx + H;
    const bool do_s = tid < T::cols(3), do_n = tid < T::cols(2), do_g = tid < T::cols(1);
    const bool in_xy = do_s && gx >= 0 && gx < Rx && gy >= 0 && gy < Ry;
    const bool own_xy = tid < T::OX * T::OY && in_xy;
    const bool n_xy = gx > 0 && gy > 0 && gx < Rx - 1 && gy < Ry - 1;  // interior in x and y
    // warp-uniform: every lane an output column off the grid's faces
    const bool full = __all_sync(0xffffffffu, own_xy && n_xy);
    const float cn = 2.0f * P.lam_normal;
    Walk<SPARSE> in(D, slots, clampi(gx, 0, Rx - 1), clampi(gy, 0, Ry - 1));
    float l_sdf = 0.0f, l_eik = 0.0f, l_nrm = 0.0f;
    int at = -1, z0, z1;
    while (next_run<SPARSE>(D, slots, at, z0, z1)) {
        // Rings in registers, unrolled over their period: the column's nodes of
        // planes z - 2 .. z + 3, s of three planes, N of three, its 1 / rho and
        // Eikonal factors of two, the L_sdf term and G_z of three.
        int e[6] = {};
        float s[3], ir[2], ee[2], ke[2], own[3], gz[3];
        float4 n[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            s[i] = own[i] = gz[i] = 0.0f;
            n[i] = make_float4(0.f, 0.f, 0.f, -1.f);
            if (i < 2) ir[i] = ee[i] = ke[i] = 0.0f;
        }
        const int zb = z0 - H;
        // plane z + 3 of s and the own values of the step that it enters in,
        // asynchronously: s is 0 outside the grid and `empty` in absent bricks
        auto fetch = [&](auto inner, int z, int slot) {
            constexpr bool kInner = decltype(inner)::value;
            const bool in_z = kInner || (z >= 0 && z < Rz);
            if (do_s) {
                float* dst = &S.s[slot][pos_s];
                if (!in_z || !in_xy)
                    *dst = 0.0f;
                else if (SPARSE && e[slot] < 0)
                    *dst = P.empty;
                else
                    copy_async4(dst, P.s + int64_t(e[slot]) * P.s_stride);
            }
            if (own_xy) {
                const int e1 = e[(slot + 5) % 6], e3 = e[(slot + 3) % 6];  // planes z - 1, z - 3
                if (kInner || (z - 1 >= z0 && z - 1 < z1)) {
                    copy_async4(&S.own[0][slot][tid], P.s_hat + e1);
                    copy_async4(&S.own[1][slot][tid], P.d_s_hat + e1);
                }
                if (kInner || (z - 3 >= z0 && z - 3 < z1))
                    copy_async4(&S.own[2][slot][tid], P.d_s + int64_t(e3) * P.d_stride);
            }
            copy_commit();
        };
        auto walk = [&](int z, int slot) {  // the node of plane z
            if (z > 0 && z < Rz) in.next(D, z);
            e[slot] = in.e;
        };
        in.seek(D, max(zb, 0));
        e[0] = in.e;
        fetch(No(), zb, 0);
        walk(zb + 1, 1);
        fetch(No(), zb + 1, 1);
        walk(zb + 2, 2);
        fetch(No(), zb + 2, 2);
        auto step = [&](auto inner, int u, int z) {
            // inner: a step away from the ends, in a warp of interior output
            // columns: straight-line code
            constexpr bool kInner = decltype(inner)::value;
            const int zo = z - 3;
            const int e_out = e[(u + 3) % 6];
            if (kInner || z + kAhead < z1 + H) {
                walk(z + kAhead, (u + kAhead) % 6);
                fetch(inner, z + kAhead, (u + kAhead) % 6);
            } else {
                copy_commit();  // an empty group keeps the count
            }
            const int p = u & 1, q = p ^ 1;  // planes z - 2 and z - 1, z - 3 of N and G
            const int iC = u % 3, iB = (u + 2) % 3, iA = (u + 1) % 3;
            const float sp = s[iC] = (kInner || do_s) ? S.s[u][pos_s] : 0.0f;
            const float sc = s[iB], sm = s[iA];
            const float w = reciprocal(fmaf(5.0f, fabsf(sc), 1.0f));
            // ---- Eq. 11 of plane z - 1 ----
            own[iC] = 0.0f;
            if (kInner || (own_xy && z - 1 >= z0 && z - 1 < z1)) {
                const float r = sc - S.own[0][u][tid];
                l_sdf = fmaf(r, r, l_sdf);
                own[iC] = P.lam_sdf * w * 2.0f * r;
                P.d_s_hat[e[(u + 5) % 6]] = S.own[1][u][tid] - own[iC];
            }
            // ---- N of plane z - 1: gradient, normal, weight at interior nodes ----
            if (kInner || do_n) {
                n[iC] = make_float4(0.f, 0.f, 0.f, -1.f);
                if (kInner || (n_xy && z - 1 > 0 && z - 1 < Rz - 1)) {
                    const float* c = &S.s[(u + 5) % 6][pos_s];
                    const float g0 = (c[1] - c[-1]) * P.inv2h[0];
                    const float g1 = (c[kWS] - c[-kWS]) * P.inv2h[1];
                    const float g2 = (sp - sm) * P.inv2h[2];
                    const float gg = fmaf(g2, g2, fmaf(g1, g1, g0 * g0));
                    const float wn = (SPARSE && !kInner && e[(u + 5) % 6] < 0) ? 0.0f : w;
                    // rho = sqrt(|g|^2 + 1e-24); from 1e-16 on it equals |g| in FP32
                    const float gn = sqrtf(gg);
                    float rho = gn, ratio = 1.0f, irho = inverse_root(gg);
                    if (!(gg >= 1e-16f && gg < 1e30f)) {
                        rho = sqrtf(gg + 1e-24f);
                        irho = 1.0f / rho;
                        ratio = gn > 0.0f ? rho / gn : 0.0f;
                    }
                    ir[q] = irho;
                    ee[q] = gn - 1.0f;
                    // Eq. 12: its gradient is ke n
                    ke[q] = P.lam_eik * wn * 2.0f * ee[q] * ratio;
                    if (rho > 0.0f) n[iC] = make_float4(g0 * irho, g1 * irho, g2 * irho, wn);
                }
                S.N[q][pos] = n[iC];
            }
            // ---- G of plane z - 2: Eikonal and normal adjoints w.r.t. grad s ----
            gz[iC] = 0.0f;
            if (kInner || do_g) {
                // Eq. 13: pairs (j, j + e_a) owned by j, (j - e_a, j) owned by the
                // neighbour; a node without a normal (w = -1) takes part in none
                const float n0 = n[iB].x, n1 = n[iB].y, n2 = n[iB].z;
                const bool has = !(n[iB].w < 0.0f);
                const float kw = has ? cn * n[iB].w : 0.0f;
                const float4* c = &S.N[p][pos];
                float d0 = 0.f, d1 = 0.f, d2 = 0.f, lq = 0.f;
                auto up = [&](const float4& v) {
                    const float q0 = n0 - v.x, q1 = n1 - v.y, q2 = n2 - v.z;
                    const bool pair = !(v.w < 0.0f);
                    const float k = pair ? kw : 0.0f;
                    const float qq = fmaf(q2, q2, fmaf(q1, q1, q0 * q0));
                    lq += pair ? qq : 0.0f;
                    d0 = fmaf(k, q0, d0);
                    d1 = fmaf(k, q1, d1);
                    d2 = fmaf(k, q2, d2);
                };
                auto down = [&](const float4& v) {
                    const float k = v.w < 0.0f ? 0.0f : cn * v.w;
                    d0 = fmaf(k, n0 - v.x, d0);
                    d1 = fmaf(k, n1 - v.y, d1);
                    d2 = fmaf(k, n2 - v.z, d2);
                };
                up(c[1]);
                down(c[-1]);
                up(c[kWN]);
                down(c[-kWN]);
                down(n[iA]);
                up(n[iC]);
                if ((kInner || (own_xy && z - 2 >= z0 && z - 2 < z1)) && has) {
                    l_eik = fmaf(ee[p], ee[p], l_eik);
                    l_nrm += lq;
                }
                // dg = ke n + (d - n (n . d)) / rho
                const float nd = -fmaf(n2, d2, fmaf(n1, d1, n0 * d0));
                d0 = has ? fmaf(ke[p], n0, fmaf(n0, nd, d0) * ir[p]) : 0.0f;
                d1 = has ? fmaf(ke[p], n1, fmaf(n1, nd, d1) * ir[p]) : 0.0f;
                gz[iC] = has ? fmaf(ke[p], n2, fmaf(n2, nd, d2) * ir[p]) : 0.0f;
                S.G[p][pos] = make_float2(d0, d1);
            }
            // ---- outputs of plane z - 3 ----
            if (kInner || (own_xy && zo >= z0)) {
                const float2* c = &S.G[q][pos];
                const float adj = fmaf(c[-1].x - c[1].x, P.inv2h[0],
                                       fmaf(c[-kWN].y - c[kWN].y, P.inv2h[1],
                                            (gz[iA] - gz[iC]) * P.inv2h[2]));
                P.d_s[int64_t(e_out) * P.d_stride] = S.own[2][u][tid] + (own[iA] + adj);
            }
        };
        // inner steps [lo, hi): the fetched plane z + 3 and its own values lie
        // in the run and in the grid, and so does every plane that is used
        const int lo = z0 + H, hi = min(z1, Rz) - kAhead;
        for (int zs = zb; zs < z1 + H; zs += 6) {
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                const int z = zs + u;
                if (z >= z1 + H) break;
                copy_wait<kAhead - 1>();
                // plane z has landed; N of plane z - 2 and G of z - 3 are written.  The
                // one barrier of a step, ahead of the branch, which differs by warp.
                __syncthreads();
                if (full && z >= lo && z < hi)
                    step(Yes(), u, z);
                else
                    step(No(), u, z);
            }
        }
        copy_wait<0>();
        __syncthreads();  // the last reads, before the next run's writes
    }
    block_loss(l_sdf, l_eik, l_nrm, P.loss, 3);
}

// L_features: planes as 16-byte texels {f0, f1, f2, 0}; gradient gathered per
// texel from its (up to 4) in-plane neighbours.
__global__ void __launch_bounds__(256) plane_reg_kernel(const float4* __restrict__ planes,
                                                        int64_t n_texels, float lam,
                                                        float4* __restrict__ grad, float* loss)
{
    float l = 0.0f;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n_texels;
         i += int64_t(gridDim.x) * blockDim.x) {
        const int c = static_cast<int>(i % 16), r = static_cast<int>((i / 16) % 16);
        const float4 v = __ldg(planes + i);
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        auto pair = [&](const float4& u, float sgn) {  // sgn * (v - u) enters the gradient
            g.x += sgn * 2.0f * lam * (v.x - u.x);
            g.y += sgn * 2.0f * lam * (v.y - u.y);
            g.z += sgn * 2.0f * lam * (v.z - u.z);
        };
        if (c > 0) pair(__ldg(planes + i - 1), 1.0f);
        if (r > 0) pair(__ldg(planes + i - 16), 1.0f);
        if (c < 15) {
            const float4 u = __ldg(planes + i + 1);
            pair(u, 1.0f);
            const float dx = u.x - v.x, dy = u.y - v.y, dz = u.z - v.z;
            l += dx * dx + dy * dy + dz * dz;
        }
        if (r < 15) {
            const float4 u = __ldg(planes + i + 16);
            pair(u, 1.0f);
            const float dx = u.x - v.x, dy = u.y - v.y, dz = u.z - v.z;
            l += dx * dx + dy * dy + dz * dz;
        }
        float4 o = grad[i];
        o.x += g.x;
        o.y += g.y;
        o.z += g.z;
        grad[i] = o;
    }
    block_loss(l, 0.0f, 0.0f, loss, 1);
}

// L_probes over [Pz][Py][Px][l*l * n_a] coefficient vectors, read as float4.
__global__ void __launch_bounds__(256) probe_reg_kernel(const float4* __restrict__ b, int Px,
                                                        int Py, int Pz, int n4, float lam,
                                                        float4* __restrict__ grad, float* loss)
{
    const int64_t n = int64_t(Px) * Py * Pz * n4;
    float l = 0.0f;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t node = i / n4;
        const int x = static_cast<int>(node % Px), y = static_cast<int>((node / Px) % Py);
        const int z = static_cast<int>(node / (int64_t(Px) * Py));
        const float4 v = __ldg(b + i);
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        const int64_t step[3] = {int64_t(n4), int64_t(Px) * n4, int64_t(Px) * Py * n4};
        const int pos[3] = {x, y, z}, lim[3] = {Px, Py, Pz};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#pragma unroll
            for (int sgn = -1; sgn <= 1; sgn += 2) {
                const int q = pos[a] + sgn;
                if (q < 0 || q >= lim[a]) continue;
                const float4 u = __ldg(b + i + sgn * step[a]);
                const float dx = v.x - u.x, dy = v.y - u.y, dz = v.z - u.z, dw = v.w - u.w;
                g.x += 4.0f * lam * dx;
                g.y += 4.0f * lam * dy;
                g.z += 4.0f * lam * dz;
                g.w += 4.0f * lam * dw;
                l += dx * dx + dy * dy + dz * dz + dw * dw;  // each ordered pair once
            }
        }
        float4 o = grad[i];
        o.x += g.x;
        o.y += g.y;
        o.z += g.z;
        o.w += g.w;
        grad[i] = o;
    }
    block_loss(l, 0.0f, 0.0f, loss, 1);
}

Taps gauss_taps()
{
    Taps T;
    double w[5], sum = 0.0;
    for (int j = 0; j < 5; ++j) {
        const double k = j - HALO;
        w[j] = std::exp(-0.5 * k * k);
        sum += w[j];
    }
    for (int j = 0; j < 5; ++j) T.w[j] = static_cast<float>(w[j] / sum);
    return T;
}

int sms()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

int blocks(int64_t n)
{
    const int64_t b = (n + 255) / 256;
    const int64_t cap = int64_t(sms()) * 16;
    return static_cast<int>(b < 1 ? 1 : (b < cap ? b : cap));
}

}  // namespace

namespace {

// Planes per CTA of a dense z-streaming kernel: the split of z into equal
// chunks whose waves of resident CTAs take the fewest steps (a chunk costs its
// planes plus `extra` steps of halo and pipeline).
int dense_chunk(int64_t tiles, int Rz, int resident, int extra)
{
    const int64_t slots = int64_t(sms()) * resident;
    int best = Rz;
    int64_t cost = INT64_MAX;
    for (int n = 1; n <= (Rz + 3) / 4 && n <= 65535; ++n) {
        const int zc = (Rz + n - 1) / n;
        const int64_t waves = (tiles * ((Rz + zc - 1) / zc) + slots - 1) / slots;
        if (waves * (zc + extra) < cost) {
            cost = waves * (zc + extra);
            best = zc;
        }
    }
    return best;
}

template <class T>
dim3 dense_domain(const int R[3], int resident, int extra, Domain& D)
{
    for (int a = 0; a < 3; ++a) {
        D.R[a] = R[a];
        D.B[a] = 0;
    }
    D.table = nullptr;
    D.n_bricks = D.seg = 0;
    const int tx = (R[0] + T::OX - 1) / T::OX, ty = (R[1] + T::OY - 1) / T::OY;
    D.zc = dense_chunk(int64_t(tx) * ty, R[2], resident, extra);
    return dim3(tx, ty, (R[2] + D.zc - 1) / D.zc);
}

// Sparse: a CTA walks up to kMaxSeg bricks along z, so that neighbouring stored
// bricks share their halo planes and pipeline and fewer CTAs find nothing stored.
// The number doubles as long as 12 CTAs per SM remain, four times the resident
// ones: it goes by the table, stored or not, because an empty CTA still costs its
// launch and its look at the table.  Measured, all three kernels, with 1 / 2 / 4 / 8
// bricks: 512^3 with 11 468 stored bricks 2.05 / 1.81 / 1.64 / 1.61 ms, 1024^3 with
// 2400 2.93 / 1.73 / 1.15 / 0.85 ms, 384^3 with 2400 0.55 / 0.47 / 0.46 / 0.46 ms,
// 256^3 with 2432 442 / 416 / 424 / 454 us, 128^3 with 300 86 / 110 / 138 / 238 us.
dim3 brick_domain(const int R[3], const int* table, int n_bricks, Domain& D)
{
    for (int a = 0; a < 3; ++a) {
        D.R[a] = R[a];
        D.B[a] = R[a] / SB;
    }
    D.zc = 0;
    D.table = table;
    D.n_bricks = n_bricks;
    const int64_t columns = int64_t(D.B[0]) * D.B[1], enough = 12 * sms();
    auto ctas = [&](int seg) { return columns * ((D.B[2] + seg - 1) / seg); };
    D.seg = 1;
    while (D.seg < kMaxSeg && D.seg < D.B[2] && ctas(2 * D.seg) >= enough) D.seg *= 2;
    return dim3(D.B[0], D.B[1], (D.B[2] + D.seg - 1) / D.seg);
}

template <class T, bool SPARSE>
cudaError_t launch_reg(const SdfReg& P, dim3 grid, cudaStream_t stream)
{
    constexpr int kBytes = static_cast<int>(sizeof(RegSmem<T>));
    auto kernel = sdf_reg_kernel<T, SPARSE>;
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
    if (e != cudaSuccess) return e;
    kernel<<<grid, T::kThreads, kBytes, stream>>>(P);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_smooth(const int R[3], const float* in, int in_stride, float* out,
                          int out_stride, bool transpose, bool accumulate, cudaStream_t stream)
{
    using T = DenseSmooth;
    Smooth P;
    const dim3 grid = dense_domain<T>(R, 2, 6, P.D);
    P.in = in;
    P.in_stride = in_stride;
    P.out = out;
    P.out_stride = out_stride;
    P.empty = 0.0f;
    P.accumulate = accumulate ? 1 : 0;
    if (transpose)
        smooth_kernel<T, false, true><<<grid, T::kThreads, 0, stream>>>(P, gauss_taps());
    else
        smooth_kernel<T, false, false><<<grid, T::kThreads, 0, stream>>>(P, gauss_taps());
    return cudaGetLastError();
}

cudaError_t launch_smooth_sparse(const int R[3], const int* table, int n_bricks, const float* in,
                                 int64_t in_base, int in_stride, float* out, int64_t out_base,
                                 int out_stride, float empty, bool transpose, bool accumulate,
                                 cudaStream_t stream)
{
    using T = BrickSmooth;
    Smooth P;
    const dim3 grid = brick_domain(R, table, n_bricks, P.D);
    P.in = in + in_base;
    P.in_stride = in_stride;
    P.out = out + out_base;
    P.out_stride = out_stride;
    P.empty = empty;
    P.accumulate = accumulate ? 1 : 0;
    if (transpose)
        smooth_kernel<T, true, true><<<grid, T::kThreads, 0, stream>>>(P, gauss_taps());
    else
        smooth_kernel<T, true, false><<<grid, T::kThreads, 0, stream>>>(P, gauss_taps());
    return cudaGetLastError();
}

cudaError_t launch_sdf_reg(const int R[3], const float h[3], const float* s_hat, const float* s,
                           int s_stride, float lam_sdf, float lam_eik, float lam_normal,
                           float* d_s, int d_stride, float* d_s_hat, float* loss,
                           cudaStream_t stream, const int* table, int n_bricks, float empty)
{
    SdfReg P;
    P.s_hat = s_hat;
    P.s = s;
    P.s_stride = s_stride;
    P.d_s = d_s;
    P.d_stride = d_stride;
    P.d_s_hat = d_s_hat;
    P.loss = loss;
    for (int a = 0; a < 3; ++a) P.inv2h[a] = 0.5f / h[a];
    P.lam_sdf = lam_sdf;
    P.lam_eik = lam_eik;
    P.lam_normal = lam_normal;
    P.empty = empty;
    if (table) {
        return launch_reg<BrickReg, true>(P, brick_domain(R, table, n_bricks, P.D), stream);
    }
    return launch_reg<DenseReg, false>(P, dense_domain<DenseReg>(R, 1, 6, P.D), stream);
}

cudaError_t launch_plane_reg(const float4* planes, int64_t n_texels, float lam, float4* grad,
                             float* loss, cudaStream_t stream)
{
    plane_reg_kernel<<<blocks(n_texels), 256, 0, stream>>>(planes, n_texels, lam, grad, loss);
    return cudaGetLastError();
}

cudaError_t launch_probe_reg(const float4* b, const int P[3], int n4, float lam, float4* grad,
                             float* loss, cudaStream_t stream)
{
    probe_reg_kernel<<<blocks(int64_t(P[0]) * P[1] * P[2] * n4), 256, 0, stream>>>(
        b, P[0], P[1], P[2], n4, lam, grad, loss);
    return cudaGetLastError();
}

}  // namespace psdf
