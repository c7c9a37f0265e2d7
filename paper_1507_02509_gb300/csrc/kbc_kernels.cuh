// Kernels of the fused pull-stream + collide step and its helpers.
//
// Data layout in device memory (one population field):
//   S f[9][plane], plane >= nx * ny, row-major [ny][nx] inside a plane, x
//   fastest; plane is padded so every plane starts on a 256-byte boundary.
// Two fields (A, B) alternate: a step reads A and writes B (pull pattern:
// f_i(x) = f'_i(x - v_i) with periodic wrap, Eq. Egeneral).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <type_traits>

#include "kbc_collide.cuh"
#include "kbc_ff.cuh"

namespace kbc {

struct StepArgs {
    int nx, ny;
    long long plane;     // elements between population planes
    CodecScale cs;
    CollideParams<float> pf;   // collision constants, computed on the host
    CollideParams<double> pd;
    double beta;               // relaxation parameter (Grad initialisation)
    int* fix_count;      // two counters, used alternately by successive steps
    int* fix_list;       // node indices recorded for the FP64 re-evaluation
    int fix_slot;        // counter used by this step
    int* flag;           // set to 1 when a node's density is not finite
    int rev;             // 1: blocks take the field from its end (see sweep_block)
    int ywrap;           // 1: periodic in y; 0: a y-slab whose rows -1 and ny are
                         // ghost rows holding the neighbouring slabs' populations
};

// The block's place in the field.  Successive steps of a field beyond L2 sweep
// it in opposite directions: what a step wrote last is still in L2 and is
// what the next one reads first, which saves part of the traffic of fields up
// to a few times that size (float LBGK 1536^2 25.1 -> 21.5 us a step, 2048^2
// 44.5 -> 40.1, 4096^2 172.5 -> 167.7, B 4095 x 4096 192 -> 184).  Within L2
// the order only costs (1024^2 LBGK 7.4 -> 7.9).
__device__ __forceinline__ unsigned sweep_block(const StepArgs& a)
{
    return a.rev ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
}

// Source row of a pull that lands on row sy (y - b, so -1 <= sy <= ny):
// periodic wrap, or on a y-slab the ghost row itself.
__device__ __forceinline__ int pull_row(int sy, const StepArgs& a)
{
    if (!a.ywrap) return sy;
    return sy < 0 ? sy + a.ny : (sy >= a.ny ? sy - a.ny : sy);
}

// ---------------------------------------------------------------- launches
//
// The kernels of a step are launched with programmatic stream serialisation:
// the launch of a kernel and the start of its blocks overlap the end of the
// kernel before it, 0.2 us a kernel in a replayed graph (64^2, float: LBGK
// 1.75 -> 1.55 us a step, B with its guard pass 3.02 -> 2.70 us).  Every
// kernel starts with chain_enter(), which waits until the one before has
// completed and its writes are visible; nothing is read or written before
// that, and every thread passes it, so a kernel's completion still implies
// that of all before it.  No kernel lets the next one start early
// (griddepcontrol.launch_dependents): blocks placed while others still run
// crowd onto the SMs that empty first (200^2 double LBGK 8.9 -> 15.6 us a
// step, 512^2 float B 5.1 -> 6.5 us).
__device__ __forceinline__ void chain_enter()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Loads of the field.  Coherent and ordered after chain_enter(): the kernel
// before may still be writing the field while this kernel's blocks start, so
// the read-only path, whose loads the compiler may move, is not for them.
__device__ __forceinline__ unsigned short ld_field(const unsigned short* p)
{
    unsigned v;
    asm volatile("ld.global.u16 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return (unsigned short)v;
}
__device__ __forceinline__ int ld_count(const int* p)
{
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float ld_field(const float* p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double ld_field(const double* p)
{
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_field(const uint2* p)
{
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_field(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

// ---------------------------------------------------------------- vectors

template <int BYTES> struct RawT;
template <> struct RawT<16> { using type = uint4; };
template <> struct RawT<8> { using type = uint2; };
template <> struct RawT<4> { using type = unsigned int; };

template <class S, int NV>
struct Vec {
    static constexpr int kBytes = int(sizeof(S)) * NV;
    using Raw = typename RawT<kBytes>::type;
    union U {
        Raw r;
        S s[NV];
    };
    __device__ __forceinline__ static void load(const S* p, S (&v)[NV])
    {
        U u;
        u.r = ld_field(reinterpret_cast<const Raw*>(p));
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = u.s[k];
    }
    __device__ __forceinline__ static void store(S* p, const S (&v)[NV])
    {
        U u;
#pragma unroll
        for (int k = 0; k < NV; ++k) u.s[k] = v[k];
        *reinterpret_cast<Raw*>(p) = u.r;
    }
};

template <class S> __device__ __forceinline__ S shfl_up1(S v)
{
    if constexpr (sizeof(S) == 2) {
        return (S)__shfl_up_sync(0xffffffffu, (unsigned)v, 1);
    } else {
        return __shfl_up_sync(0xffffffffu, v, 1);
    }
}
template <class S> __device__ __forceinline__ S shfl_down1(S v)
{
    if constexpr (sizeof(S) == 2) {
        return (S)__shfl_down_sync(0xffffffffu, (unsigned)v, 1);
    } else {
        return __shfl_down_sync(0xffffffffu, v, 1);
    }
}

template <typename T> __device__ __forceinline__ const CollideParams<T>& params_of(const StepArgs& a);
template <> __device__ __forceinline__ const CollideParams<float>& params_of<float>(const StepArgs& a)
{
    return a.pf;
}
template <> __device__ __forceinline__ const CollideParams<double>& params_of<double>(const StepArgs& a)
{
    return a.pd;
}

// Appends up to NV nodes per lane to the re-evaluation list: bit k of `hits`
// marks node n0 + k * stride.  All lanes of the warp call it.  One atomic
// addition per warp reserves the entries (one per lane with a hit, all on the
// same counter, took 60 us of a step with 250 k hits); they are written in
// the order k, lane, which keeps neighbouring nodes together.
template <int NV>
__device__ __forceinline__ void record_fix(unsigned hits, int n0, int stride, const StepArgs& a)
{
    if (!__any_sync(0xffffffffu, hits != 0u)) return;
    unsigned vote[NV];
    int all = 0;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        vote[k] = __ballot_sync(0xffffffffu, (hits >> k) & 1u);
        all += __popc(vote[k]);
    }
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == 0) base = atomicAdd(a.fix_count + a.fix_slot, all);
    base = __shfl_sync(0xffffffffu, base, 0);
    const int cap = a.nx * a.ny;  // the list holds one entry per node
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int idx = base + __popc(vote[k] & ((1u << lane) - 1u));
        if (((hits >> k) & 1u) && idx < cap) a.fix_list[idx] = n0 + k * stride;
        base += __popc(vote[k]);
    }
}

// ---------------------------------------------------------------- step, rows

// Collides the NV nodes one thread holds.  Sets `bad` when a density is not
// finite; bit k of the result marks a guard hit of node k.  PAIRS: collide
// nodes 2j, 2j + 1 in one packed lane pair (float, NV even; the same bits as
// one node at a time, about half the arithmetic instructions, twice the
// registers of the collision).
template <int VAR, bool U, bool PAIRS = false, typename T, int NV>
__device__ __forceinline__ unsigned collide_vec(T (&f)[NV][9], const CollideParams<T>& p, bool& bad)
{
    unsigned hits = 0u;
    if constexpr (PAIRS && std::is_same<T, float>::value && NV % 2 == 0) {
#pragma unroll
        for (int k = 0; k < NV; k += 2) {
            T r0, r1;
            unsigned h;
            collide_pair<VAR, U>(f[k], f[k + 1], p, r0, r1, h);
            bad |= !isfinite(r0) || !isfinite(r1);
            hits |= h << k;
        }
    } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            T rho;
            bool hit;
            collide_node<VAR, U>(f[k], p, rho, hit);
            bad |= !isfinite(rho);
            hits |= (hit ? 1u : 0u) << k;
        }
    }
    return hits;
}

//
// One thread updates NV consecutive nodes of one row with 16-byte loads and
// stores per population plane.  Populations moving along x (a = +-1) need
// the neighbour one element to the left/right: it comes from the adjacent
// lane by a warp shuffle, and lanes 0 / 31 fetch it from memory (periodic
// wrap at the row ends).  Requires nx % (32 NV) == 0; a 1-D grid of
// nbx * ny blocks, nbx = ceil(nx / (BLOCK NV)) blocks per row; warps past
// the row end exit as a whole.
// PAIRS: the four nodes are collided as two packed lane pairs, which takes 40%
// fewer instructions and up to 128 registers: 8 resident blocks per SM (10, of
// 96 registers, for the natural-basis variants and LBGK) instead of 12.  Half
// storage fits them; float spills 4 bytes (A), 12 (B), 32 (C) and 48 (D).
// That is the faster side where instructions bound the step: half storage
// (4096^2 C 143 -> 122 us, bulk copies 126; 1024^2 B 10.5 -> 9.5), and
// float fields that stay in L2 (1024^2 B 12.2 -> 11.6, C 11.4 -> 10.8);
// where HBM does, the lower occupancy costs more than it saves (4096^2
// float B 180 -> 182, half LBGK 103 -> 105).
template <int VAR, class C, bool PAIRS> constexpr int row_min_blocks()
{
    return !PAIRS ? C::kRowMinBlocks : (VAR == kA || VAR == kB) ? 8 : 10;
}

template <int VAR, class C, int NV, int BLOCK, bool PAIRS>
__global__ void __launch_bounds__(BLOCK, row_min_blocks<VAR, C, PAIRS>())
step_rows(const typename C::S* __restrict__ src, typename C::S* __restrict__ dst, StepArgs a,
          int nbx)
{
    using S = typename C::S;
    using T = typename C::T;
    // the pairs' kernels are bound by instructions: no alternating sweeps there
    const unsigned blk = PAIRS ? blockIdx.x : sweep_block(a);
    const int y = blk / nbx;
    const int bx = blk - y * nbx;
    const int x0 = (bx * BLOCK + threadIdx.x) * NV;
    chain_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.fix_count)
        a.fix_count[a.fix_slot ^ 1] = 0;  // free the other counter for the next step
    if (x0 >= a.nx) return;               // whole warps only (nx % (32 NV) == 0)
    const int lane = threadIdx.x & 31;
    const int ym = pull_row(y - 1, a);
    const int yp = pull_row(y + 1, a);
    const int xl = (x0 == 0) ? a.nx - 1 : x0 - 1;
    const int xr = (x0 + NV == a.nx) ? 0 : x0 + NV;

    S raw[9][NV];
    S edge[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ai = i % 3 - 1, bi = i / 3 - 1;
        const int sy = (bi == 1) ? ym : (bi == -1 ? yp : y);   // source row y - b
        const S* row = src + (long long)i * a.plane + (long long)sy * a.nx;
        Vec<S, NV>::load(row + x0, raw[i]);
        if (ai == 1) {
            edge[i] = S(0);
            if (lane == 0) edge[i] = ld_field(row + xl);
        } else if (ai == -1) {
            edge[i] = S(0);
            if (lane == 31) edge[i] = ld_field(row + xr);
        }
    }
    T f[NV][9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ai = i % 3 - 1;
        if (ai == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) f[k][i] = C::load(raw[i][k], i, a.cs);
        } else if (ai == 1) {  // source x - 1
            S left = shfl_up1(raw[i][NV - 1]);
            if (lane == 0) left = edge[i];
            f[0][i] = C::load(left, i, a.cs);
#pragma unroll
            for (int k = 1; k < NV; ++k) f[k][i] = C::load(raw[i][k - 1], i, a.cs);
        } else {               // source x + 1
            S right = shfl_down1(raw[i][0]);
            if (lane == 31) right = edge[i];
#pragma unroll
            for (int k = 0; k < NV - 1; ++k) f[k][i] = C::load(raw[i][k + 1], i, a.cs);
            f[NV - 1][i] = C::load(right, i, a.cs);
        }
    }
    bool bad = false;
    const unsigned hits = collide_vec<VAR, C::kUnits, PAIRS>(f, params_of<T>(a), bad);
    if constexpr (VAR != kLBGK) {
        if (a.fix_list) record_fix<NV>(hits, y * a.nx + x0, 1, a);
    }
    if (bad) *a.flag = 1;
    const long long o = (long long)y * a.nx + x0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if constexpr (std::is_same<C, CodecF16>::value && NV % 2 == 0) {
            unsigned pk[NV / 2];
#pragma unroll
            for (int k = 0; k < NV; k += 2) pk[k / 2] = C::store2(f[k][i], f[k + 1][i], i, a.cs);
            Vec<unsigned, NV / 2>::store(reinterpret_cast<unsigned*>(dst + (long long)i * a.plane + o), pk);
        } else {
            S out[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) out[k] = C::store(f[k][i], i, a.cs);
            Vec<S, NV>::store(dst + (long long)i * a.plane + o, out);
        }
    }
}

// ---------------------------------------------------------------- step, nodes
//
// Any nx, ny; same arithmetic as step_rows.  Nodes are taken in memory order
// across the rows: a warp holds 32 K consecutive nodes, each thread K of
// them 32 apart (collided in packed lane pairs for float and half with K > 1),
// so every load and store is coalesced whatever the width.  A warp whose
// nodes lie in one row, away from its ends, addresses every population as
// one offset shared by the warp plus the thread's index; the others wrap per
// thread.  Bound by the latency of the collision: K = 4 gives it two
// independent pairs (4095 x 4096, float B, all sweeps in one direction: K = 4
// 193 us, K = 2 248 us, one node at a time 237 us; one node per thread with a
// 64-bit division before, 281 us; 185 us with alternating sweeps); float C
// needs 94 registers and runs at the copy bandwidth with ten blocks per SM (176
// us against 189 us with eight), half C spills 64 bytes there.  A grid whose
// nodes find a thread each at once takes K = 1 (256^2, float B: 3.1 us a step
// against 3.3 for the vector rows).  Double is bound by the FP64 pipe and takes
// K = 1 everywhere (64^2: 7.8 us against 13.9 with the two nodes a thread of
// the vector rows, 2048^2 1486 against 1503 us).
constexpr int kFlatBlock = 64;
// Nodes per thread on a grid that fills the GPU, and resident blocks per SM
// the kernel is compiled for.
template <int VAR, class C> constexpr int flat_nodes()
{
    return std::is_same<C, CodecF64>::value ? 1 : (VAR == kLBGK ? 2 : 4);
}
template <int VAR, class C, int K> constexpr int flat_min_blocks()
{
    return std::is_same<C, CodecF64>::value ? 1 : (K < 4 ? 12 : (VAR == kC || VAR == kD) ? 10 : 8);
}

template <int VAR, class C, int K>
__global__ void __launch_bounds__(kFlatBlock, flat_min_blocks<VAR, C, K>())
step_nodes(const typename C::S* __restrict__ src, typename C::S* __restrict__ dst, StepArgs a)
{
    using S = typename C::S;
    using T = typename C::T;
    chain_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.fix_count) a.fix_count[a.fix_slot ^ 1] = 0;
    const int total = a.nx * a.ny;
    const int lane = threadIdx.x & 31;
    // first node of the warp (uniform), its row and column
    const unsigned w0 = (sweep_block(a) * kFlatBlock + (threadIdx.x & ~31u)) * K;
    if (w0 >= (unsigned)total) return;
    const int y0 = (int)(w0 / (unsigned)a.nx), x0 = (int)w0 - y0 * a.nx;
    const bool yin = !a.ywrap || (y0 > 0 && y0 + 1 < a.ny);
    S raw[K][9];
    if (yin && x0 > 0 && x0 + 32 * K < a.nx) {
        const S* base = src + w0 + lane;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const S* pl = base + ((long long)i * a.plane - vb(i) * (long long)a.nx - va(i));
#pragma unroll
            for (int k = 0; k < K; ++k) raw[k][i] = ld_field(pl + 32 * k);
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            int n = (int)w0 + 32 * k + lane;
            if ((unsigned)n >= (unsigned)total) n = total - 1;  // idle lanes repeat the last node
            const int y = (int)((unsigned)n / (unsigned)a.nx), x = n - y * a.nx;
            const int ym = pull_row(y - 1, a), yp = pull_row(y + 1, a);
            const int xl = x == 0 ? a.nx - 1 : x - 1, xr = x + 1 == a.nx ? 0 : x + 1;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int sy = vb(i) == 1 ? ym : (vb(i) == -1 ? yp : y);
                const int sx = va(i) == 1 ? xl : (va(i) == -1 ? xr : x);
                raw[k][i] = ld_field(src + (long long)i * a.plane + (long long)sy * a.nx + sx);
            }
        }
    }
    T f[K][9];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int i = 0; i < 9; ++i) f[k][i] = C::load(raw[k][i], i, a.cs);
    bool bad = false;
    const unsigned hits = collide_vec<VAR, C::kUnits, (K > 1)>(f, params_of<T>(a), bad);
    if (bad) *a.flag = 1;
    unsigned live = 0u;
#pragma unroll
    for (int k = 0; k < K; ++k) live |= (w0 + 32 * k + lane < (unsigned)total ? 1u : 0u) << k;
    if constexpr (VAR != kLBGK) {
        if (a.fix_list) record_fix<K>(hits & live, (int)w0 + lane, 32, a);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int n = (int)w0 + 32 * k + lane;
        if ((live >> k) & 1u) {
#pragma unroll
            for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = C::store(f[k][i], i, a.cs);
        }
    }
}

// ---------------------------------------------------------------- all-FP64 step
//
// One node per thread with the whole collision in double whatever the
// storage; used for the exact-gamma mode (root of Eq. result1), whose Newton
// iteration runs in double.
template <int VAR, class C>
__global__ void __launch_bounds__(256)
step_nodes_f64(const typename C::S* __restrict__ src, typename C::S* __restrict__ dst, StepArgs a)
{
    chain_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.fix_count) a.fix_count[a.fix_slot ^ 1] = 0;
    const long long total = (long long)a.nx * a.ny;
    CollideParams<double> p = a.pd;
    p.guard = 0.0;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total;
         n += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(n / a.nx), x = (int)(n - (long long)y * a.nx);
        double f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int ai = i % 3 - 1, bi = i / 3 - 1;
            int sx = x - ai, sy = y - bi;
            sx = sx < 0 ? sx + a.nx : (sx >= a.nx ? sx - a.nx : sx);
            sy = pull_row(sy, a);
            f[i] = C::to_f64(ld_field(src + (long long)i * a.plane + (long long)sy * a.nx + sx), i, a.cs);
        }
        double rho;
        bool hit;
        collide_node<VAR>(f, p, rho, hit);
        if (!isfinite(rho)) *a.flag = 1;
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = C::from_f64(f[i], i, a.cs);
    }
}

// ---------------------------------------------------------------- FP64 re-evaluation
//
// Recomputes, entirely in double, the nodes the step recorded (entropic
// denominator at or below the guard) from the same source field, and
// overwrites their stored result.
template <int VAR, class C>
__global__ void __launch_bounds__(256)
step_fixup(const typename C::S* __restrict__ src, typename C::S* __restrict__ dst, StepArgs a)
{
    using S = typename C::S;
    chain_enter();
    const int recorded = ld_count(a.fix_count + a.fix_slot);
    const int count = recorded < a.nx * a.ny ? recorded : a.nx * a.ny;
    if (count == 0) return;
    // node t goes to block t % gridDim.x: the few recorded nodes spread over
    // every SM's FP64 pipe instead of filling the first blocks
    for (int t = threadIdx.x * gridDim.x + blockIdx.x; t < count; t += gridDim.x * blockDim.x) {
        const int n = ld_count(a.fix_list + t);
        const int y = n / a.nx, x = n - y * a.nx;
        double f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int ai = i % 3 - 1, bi = i / 3 - 1;
            int sx = x - ai, sy = y - bi;
            sx = sx < 0 ? sx + a.nx : (sx >= a.nx ? sx - a.nx : sx);
            sy = pull_row(sy, a);
            f[i] = C::to_f64(ld_field(src + (long long)i * a.plane + (long long)sy * a.nx + sx), i, a.cs);
        }
        CollideParams<double> q = a.pd;
        q.guard = 0.0;
        double rho;
        bool hit;
        collide_node<VAR>(f, q, rho, hit);
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = C::from_f64(f[i], i, a.cs);
    }
}

// ---------------------------------------------------------------- init / io

// out of line: the rarely taken branch of the two below, which keeps the order
// of operations that the stored float and half values have always had.
// rho = 1 and u = 0 (of either sign) give f = W, for which no error bound
// settles anything and which fluid at rest has in every node: stored without the
// double computation (4096^2 float at rest 1959 -> 363 us).
template <class C>
__device__ __noinline__ void feq_node_general(double r, double x, double y,
                                              typename C::S* __restrict__ dst, long long n, const StepArgs& a)
{
    if (__double_as_longlong(r) == 0x3ff0000000000000ll &&
        ((__double_as_longlong(x) | __double_as_longlong(y)) << 1) == 0ll) {
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = typename C::S(0);
        return;
    }
    const double usq15 = 1.5 * (x * x + y * y);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const double xi = va(i) * x + vb(i) * y;
        const double P = xi * (3.0 + 4.5 * xi) - usq15;
        const double dev = wgt(i) * ((r - 1.0) + r * P);
        dst[(long long)i * a.plane + n] = C::from_f64(dev, i, a.cs);
    }
}

// f = f^eq(rho, u) (Eq. Eq) of one node, stored as deviations from W_i;
// computed in double, in the moment form
//   f^eq_i - W_i = W_i (q + 3 v_i.j + rho (4.5 (v_i.u)^2 - 1.5 u^2)),
// q = rho - 1, j = rho u: 28 FP64 instructions where nine polynomials took 61.
template <class C>
__device__ __forceinline__ void feq_node(double r, double x, double y, typename C::S* __restrict__ dst,
                                         long long n, const StepArgs& a)
{
    // infinities, NaN and magnitudes whose products may overflow: the general
    // form, whose terms turn into NaN together
    const int top = max(max(__double2hiint(r) & 0x7fffffff, __double2hiint(x) & 0x7fffffff),
                        __double2hiint(y) & 0x7fffffff);
    if (top >= 0x52b00000) {  // 2^300
        feq_node_general<C>(r, x, y, dst, n, a);
        return;
    }
    const double q = r - 1.0, jx = r * x, jy = r * y;
    const double A = jx * x, B = jy * y, xy = 0.25 * (jx * y);
    const double S = A + B, q9 = (1.0 / 9.0) * q;
    const double ex = fma(1.0 / 3.0, A, fma(-1.0 / 6.0, B, q9));
    const double ey = fma(1.0 / 3.0, B, fma(-1.0 / 6.0, A, q9));
    const double g = fma(1.0 / 12.0, S, 0.25 * q9);
    const double dp = g + xy, dm = g - xy, sp = jx + jy, sm = jx - jy;
    double d[9];
    d[4] = fma(-2.0 / 3.0, S, 4.0 * q9);
    d[5] = fma(1.0 / 3.0, jx, ex);
    d[3] = fma(-1.0 / 3.0, jx, ex);
    d[7] = fma(1.0 / 3.0, jy, ey);
    d[1] = fma(-1.0 / 3.0, jy, ey);
    d[8] = fma(1.0 / 12.0, sp, dp);
    d[0] = fma(-1.0 / 12.0, sp, dp);
    d[2] = fma(1.0 / 12.0, sm, dm);
    d[6] = fma(-1.0 / 12.0, sm, dm);
#pragma unroll
    for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = C::from_f64(d[i], i, a.cs);
}

// Two nodes n0, n1 (n1 < 0: none) of the equilibrium for float or half
// storage in pairs of floats, packed over the nodes: the moment form of
// feq_node with the factors 1/9, 1/3 and 1 (float) or S, 3 S and 9 S (half
// codes are (f - W) S / W) on q, the first- and second-order terms.  Error
// bound, relative: the inputs 2^-48, rho 2^-47, a product 2^-45 more (see
// FF), so j 2^-44.5, and A, B and C9, of three more factors, 2^-43.3; then at
// most four additions, 2^-46 of M each, M the sum of the terms' magnitudes (for
// the rest population its own two terms').  2^-42.7 in all, of which 2^-42 M
// leaves a third, and the double computation's own error is 2^-50 M.
template <class C>
__device__ __forceinline__ void feq_pair(const double (&r)[2], const double (&x)[2], const double (&y)[2],
                                         typename C::S* __restrict__ dst, long long n0, long long n1,
                                         const StepArgs& a)
{
    using L = Lf2;
    constexpr bool half = std::is_same<C, CodecF16>::value;
    float h[3][2], l[3][2];
    bool ok[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        ok[k] = split_double(r[k] - 1.0, h[0][k], l[0][k]);
        ok[k] = split_double(x[k], h[1][k], l[1][k]) && ok[k];
        ok[k] = split_double(y[k], h[2][k], l[2][k]) && ok[k];
    }
    const FF<L> q(L(h[0][0], h[0][1]), L(l[0][0], l[0][1]));
    const FF<L> u(L(h[1][0], h[1][1]), L(l[1][0], l[1][1]));
    const FF<L> v(L(h[2][0], h[2][1]), L(l[2][0], l[2][1]));
    FF<L> rho = two_sum(L(1.0f), q.h);
    rho = fast_two_sum(rho.h, rho.l + q.l);
    const FF<L> jx = rho * u, jy = rho * v;
    FF<L> c1, c3;
    FF<L> q1, C9;
    const FF<L> xy = jx * v;
    if constexpr (half) {
        const float S = a.cs.scale;
        const float s3 = 3.0f * S, s9 = 9.0f * S;
        c3 = FF<L>(L(s3), L(__fmaf_rn(3.0f, S, -s3)));
        q1 = FF<L>(q.h, q.l) * FF<L>(L(S), L(0.0f));
        C9 = xy * FF<L>(L(s9), L(__fmaf_rn(9.0f, S, -s9)));
    } else {
        c1 = FF<L>(L(ff_hi(1.0 / 9.0)), L(ff_lo(1.0 / 9.0)));
        c3 = FF<L>(L(ff_hi(1.0 / 3.0)), L(ff_lo(1.0 / 3.0)));
        q1 = q * c1;
        C9 = xy;
    }
    const FF<L> A = (jx * u) * c3, B = (jy * v) * c3, px = jx * c3, py = jy * c3;
    const FF<L> S3 = A + B;
    const FF<L> ex = (q1 + A) + scale(B, -0.5f), ey = (q1 + B) + scale(A, -0.5f);
    const FF<L> g = q1 + S3;
    const FF<L> dp = g + C9, dm = g - C9, sp = px + py, sm = px - py;
    FF<L> d[9];
    d[4] = add_raw(q1, scale(S3, -0.5f));
    d[5] = add_raw(ex, px);
    d[3] = add_raw(ex, -px);
    d[7] = add_raw(ey, py);
    d[1] = add_raw(ey, -py);
    d[8] = add_raw(dp, sp);
    d[0] = add_raw(dp, -sp);
    d[2] = add_raw(dm, sm);
    d[6] = add_raw(dm, -sm);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float m4 = fabsf(q1.h.get(k)) + fabsf(A.h.get(k)) + fabsf(B.h.get(k));
        const float m = 2.0f * m4 + fabsf(C9.h.get(k)) + fabsf(px.h.get(k)) + fabsf(py.h.get(k));
        // below 2^-28 the inputs' cut at 2^-74 would count; above, overflow
        bool fine = ok[k] && m > (half ? 0x1p-28f * a.cs.scale : 0x1p-28f) && m < 0x1p60f;
        const long long n = k ? n1 : n0;
        typename C::S out[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            // the stored value is the sum over 4 (float, diagonals) or times 4 (float, rest)
            const float w = half ? 1.0f : (wclass(i) == 0 ? 0.25f : wclass(i) == 2 ? 4.0f : 1.0f);
            const float err = (i == 4 ? m4 : m) * (0x1p-42f * w);
            round_sure(d[i].h.get(k) * w, d[i].l.get(k) * w, err, out[i], fine);
        }
        if (n >= 0) {
            if (fine) {
#pragma unroll
                for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = out[i];
            } else {
                feq_node_general<C>(r[k], x[k], y[k], dst, n, a);
            }
        }
    }
}

// Two nodes per thread for float and half storage (grid stride apart, so
// that every access stays coalesced): about 200 instructions a node, two of
// them FP64, against 67 FP64 instructions before; 4096^2 from device fields
// 1906 -> 360 us (float), 2187 -> 372 us (half), 1635 -> 994 us (double), 80 us
// of each the caller's copy of u into one array.
template <class C>
__global__ void __launch_bounds__(256)
init_feq(const double* __restrict__ rho, const double* __restrict__ ux,
         const double* __restrict__ uy, typename C::S* __restrict__ dst, StepArgs a)
{
    const long long total = (long long)a.nx * a.ny;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if constexpr (std::is_same<C, CodecF64>::value) {
        for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total; n += stride)
            feq_node<C>(rho[n], ux[n], uy[n], dst, n, a);
    } else {
        for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total; n += 2 * stride) {
            const long long n1 = n + stride < total ? n + stride : -1;
            const long long m = n1 >= 0 ? n1 : n;
            const double r[2] = {rho[n], rho[m]}, x[2] = {ux[n], ux[m]}, y[2] = {uy[n], uy[m]};
            feq_pair<C>(r, x, y, dst, n, n1, a);
        }
    }
}

// Grad's approximation (Eq. Grad) with Pi = Pi^eq + Pi^(1) (Eq. Peq,
// Eq. P1AC), velocity gradients by periodic central differences.
template <class C>
__global__ void init_grad(const double* __restrict__ rho, const double* __restrict__ ux,
                          const double* __restrict__ uy, typename C::S* __restrict__ dst,
                          StepArgs a)
{
    const long long total = (long long)a.nx * a.ny;
    // cs^2 = 1/3: the divisions by cs^2 and 2 cs^4 of Eq. Grad are the
    // multiplications by 3 and 4.5 (double division is many FP64-pipe
    // instructions, and this kernel is bound by that pipe)
    const double cs2 = 1.0 / 3.0;
    const double half_inv_beta = 0.5 / a.beta;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total;
         n += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(n / a.nx), x = (int)(n - (long long)y * a.nx);
        const long long row = (long long)y * a.nx;
        const long long xp = row + (x + 1 == a.nx ? 0 : x + 1);
        const long long xm = row + (x == 0 ? a.nx - 1 : x - 1);
        const long long yp = (long long)(y + 1 == a.ny ? 0 : y + 1) * a.nx + x;
        const long long ym = (long long)(y == 0 ? a.ny - 1 : y - 1) * a.nx + x;
        // du[a][b] = d u_b / d x_a
        const double dxux = 0.5 * (ux[xp] - ux[xm]), dxuy = 0.5 * (uy[xp] - uy[xm]);
        const double dyux = 0.5 * (ux[yp] - ux[ym]), dyuy = 0.5 * (uy[yp] - uy[ym]);
        const double r = rho[n], u0 = ux[n], u1 = uy[n];
        const double c = r * cs2 * half_inv_beta;
        // non-equilibrium-shifted stress minus the isotropic part rho cs2 delta
        const double sxx = r * u0 * u0 - c * 2.0 * dxux;
        const double syy = r * u1 * u1 - c * 2.0 * dyuy;
        const double sxy = r * u0 * u1 - c * (dxuy + dyux);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double vx = va(i), vy = vb(i);
            const double lin = 3.0 * r * (u0 * vx + u1 * vy);
            const double quad = sxx * (vx * vx - cs2) + syy * (vy * vy - cs2) + 2.0 * sxy * vx * vy;
            const double fi = wgt(i) * (r + lin + 4.5 * quad);
            dst[(long long)i * a.plane + n] = C::from_f64(fi - wgt(i), i, a.cs);
        }
    }
}

template <class C>
__global__ void set_populations(const double* __restrict__ f, typename C::S* __restrict__ dst,
                                StepArgs a)
{
    const long long total = (long long)a.nx * a.ny;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total;
         n += (long long)gridDim.x * blockDim.x) {
        double v[9];  // all loads first: the conversions branch
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = f[(long long)i * total + n];
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = C::from_f64(v[i] - wgt(i), i, a.cs);
    }
}

template <class C>
__global__ void get_populations(const typename C::S* __restrict__ src, double* __restrict__ f,
                                StepArgs a)
{
    const long long total = (long long)a.nx * a.ny;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total;
         n += (long long)gridDim.x * blockDim.x) {
        typename C::S v[9];  // all loads first: the conversions branch
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = src[(long long)i * a.plane + n];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[(long long)i * total + n] = C::to_f64(v[i], i, a.cs) + wgt(i);
    }
}

// f[k][9] = populations of node nodes[k]; bad indices set *bad and are skipped
template <class C>
__global__ void probe_nodes(const typename C::S* __restrict__ src, const long long* __restrict__ nodes,
                            int count, double* __restrict__ f, int* bad, StepArgs a)
{
    const long long total = (long long)a.nx * a.ny;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
        const long long n = nodes[k];
        if (n < 0 || n >= total) {
            *bad = 1;
            continue;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i)
            f[(long long)k * 9 + i] = C::to_f64(src[(long long)i * a.plane + n], i, a.cs) + wgt(i);
    }
}

// rho and u of a node in double (from the stored deviations).  Float and
// half storage: exact integer sums, rounded once (FixedSums), so that six
// FP64 instructions and three conversions remain of about forty; a node
// whose values do not share a unit takes the double sums.  Bound by the FP64
// pipe; 4096^2 moments 1106 -> 327 us (float), 1266 -> 364 us (half),
// 828 -> 700 us (double, shared differences and rcp_pos), against 150, 127
// and 241 us for the bytes.
template <class C>
__device__ __forceinline__ void node_macro(const typename C::S* __restrict__ src, long long n,
                                           const StepArgs& a, double& rho, double& ux, double& uy)
{
    typename C::S c[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) c[i] = src[(long long)i * a.plane + n];
    if constexpr (fixed_of<C>::kHas) {
        FixedSums s;
        if (fixed_of<C>::sums(c, a.cs, s)) {
            rho = __fma_rn(s.unit, (double)s.drho, 1.0);
            // where rho nearly vanishes (or is negative) the rounding of the
            // half storage's unit would be all that is left of it
            if (__double2hiint(rho) >= 0x3eb00000) {  // 2^-20
                const double ir = rcp_pos(rho) * s.unit;
                ux = (double)s.jx * ir;
                uy = (double)s.jy * ir;
                return;
            }
        }
    }
    double d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = C::to_f64(c[i], i, a.cs);
    // differences of opposite populations: j keeps its relative accuracy
    // where it is far smaller than the populations
    const double a08 = d[8] - d[0], a26 = d[2] - d[6];
    rho = 1.0 + (((d[0] + d[8]) + (d[2] + d[6])) + ((d[1] + d[7]) + (d[3] + d[5])) + d[4]);
    const double irho = rcp_pos(rho);  // one reciprocal for both components
    ux = ((a08 + a26) + (d[5] - d[3])) * irho;
    uy = ((a08 - a26) + (d[7] - d[1])) * irho;
}

template <class C>
__global__ void __launch_bounds__(256)
moments(const typename C::S* __restrict__ src, double* __restrict__ rho,
        double* __restrict__ ux, double* __restrict__ uy, StepArgs a)
{
    const long long total = (long long)a.nx * a.ny;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < total;
         n += (long long)gridDim.x * blockDim.x) {
        double r, x, y;
        node_macro<C>(src, n, a, r, x, y);
        rho[n] = r;
        ux[n] = x;
        uy[n] = y;
    }
}

// ---------------------------------------------------------------- diagnostics
//
// Per block: FP64 partial sums of mass and momentum, the count, mean and sum
// of squared deviations (M2) of |u|^2/2 and of w^2/2, and gamma (sum, min,
// max) over a grid-stride range of nodes, written to part[block][11].  gamma
// is that of the collision the next step performs, evaluated in double.
// Means and M2 are accumulated per thread by Welford's update and combined
// across threads and blocks by Chan et al.'s pairwise formula, so the
// standard deviations need no E[x^2] - E[x]^2 difference (which cancels).
// Deterministic: fixed grid, fixed reduction order.
constexpr int kDiagParts = 11;
constexpr int kDiagBlock = 256;

// Welford's running update of mean m and M2 q with one value x, rn = 1 / n
// with n the count including x.  The counts of both quantities of a thread
// are the same, so one reciprocal (rcp_pos) serves both; with a division
// each they took a tenth of the kernels' FP64 instructions.
__device__ __forceinline__ void welford_add(double rn, double& m, double& q, double x)
{
    const double d = x - m;
    m = __fma_rn(d, rn, m);
    q = __fma_rn(d, x - m, q);
}

// Chan, Golub and LeVeque's combination of two partial (n, m, q) sets: the
// second is folded into the first.  Both quantities of a set have the same
// counts, so their factors nb / n and na nb / n are formed once (with four
// divisions a fold, the reductions' chains took half of the time of a call on
// a small grid).
struct ChanFactors {
    double fm, fq;
    bool first, second;  // whether either set is empty
    __device__ __forceinline__ ChanFactors(double na, double nb) : first(na == 0.0), second(nb == 0.0)
    {
        const double r = first || second ? 0.0 : rcp_pos(na + nb);
        fm = nb * r;
        fq = na * fm;
    }
    __device__ __forceinline__ void merge(double& ma, double& qa, double mb, double qb) const
    {
        if (second) return;
        if (first) {
            ma = mb;
            qa = qb;
            return;
        }
        const double d = mb - ma;
        ma = __fma_rn(d, fm, ma);
        qa += __fma_rn(d * d, fq, qb);
    }
};

// Tiles of the diagnostics kernels: kTileW x kTileH nodes per block
// iteration (two per thread), with rho and u computed once per position of
// the tile and its halo into shared memory (periodic wrap), so that the
// central-difference stencils read them there instead of recomputing them.
constexpr int kTileW = 64, kTileH = 8;

__device__ __forceinline__ int wrap_mod(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// Folds partial set b into partial set a of the diagnostics; element k of a
// set is at a[k * sa] (b[k * sb]).
__device__ __forceinline__ void diag_fold(double* a, int sa, const double* b, int sb)
{
    a[0] += b[0];
    a[sa] += b[sb];
    a[2 * sa] += b[2 * sb];
    const double na = a[3 * sa], nb = b[3 * sb];
    const ChanFactors f(na, nb);
    f.merge(a[4 * sa], a[5 * sa], b[4 * sb], b[5 * sb]);
    f.merge(a[6 * sa], a[7 * sa], b[6 * sb], b[7 * sb]);
    a[3 * sa] = na + nb;
    a[8 * sa] += b[8 * sb];
    a[9 * sa] = fmin(a[9 * sa], b[9 * sb]);
    a[10 * sa] = fmax(a[10 * sa], b[10 * sb]);
}

template <int VAR, class C>
__global__ void __launch_bounds__(kDiagBlock)
diag_partial(const typename C::S* __restrict__ src, double* __restrict__ part, StepArgs a)
{
    constexpr int HW = kTileW + 2, HH = kTileH + 2;  // one-node halo
    __shared__ double sr[HH][HW], sux[HH][HW], suy[HH][HW];
    // mass, px, py, n, mean and M2 of |u|^2/2, of w^2/2, gamma sum, min, max
    double acc[kDiagParts] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 1e300, -1e300};
    CollideParams<double> p = a.pd;
    p.guard = 0.0;
    const int ntx = (a.nx + kTileW - 1) / kTileW, nty = (a.ny + kTileH - 1) / kTileH;
    const long long ntiles = (long long)ntx * nty;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int x0 = (int)(tile % ntx) * kTileW, y0 = (int)(tile / ntx) * kTileH;
        __syncthreads();  // the previous tile's readers are done with the arrays
        for (int q = threadIdx.x; q < HH * HW; q += blockDim.x) {
            const int qy = q / HW, qx = q - qy * HW;
            const int gx = wrap_mod(x0 + qx - 1, a.nx);
            int gy = y0 + qy - 1;
            if (a.ywrap) {
                gy = wrap_mod(gy, a.ny);
            } else if (gy > a.ny) {  // y-slab: rows -1 and ny are ghost rows; beyond, unused
                sr[qy][qx] = sux[qy][qx] = suy[qy][qx] = 0.0;
                continue;
            }
            node_macro<C>(src, (long long)gy * a.nx + gx, a, sr[qy][qx], sux[qy][qx], suy[qy][qx]);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < kTileW * kTileH; k += blockDim.x) {
            const int ly = k / kTileW, lx = k - ly * kTileW;
            const int x = x0 + lx, y = y0 + ly;
            if (x >= a.nx || y >= a.ny) continue;
            const int cx = lx + 1, cy = ly + 1;
            const double r = sr[cy][cx], ux = sux[cy][cx], uy = suy[cy][cx];
            acc[0] += r;
            acc[1] += r * ux;
            acc[2] += r * uy;
            const double ke = 0.5 * (ux * ux + uy * uy);
            const double w = 0.5 * (suy[cy][cx + 1] - suy[cy][cx - 1]) - 0.5 * (sux[cy + 1][cx] - sux[cy - 1][cx]);
            const double zz = 0.5 * w * w;
            acc[3] += 1.0;
            const double rn = rcp_pos(acc[3]);
            welford_add(rn, acc[4], acc[5], ke);
            welford_add(rn, acc[6], acc[7], zz);
            const int xl = x == 0 ? a.nx - 1 : x - 1, xr = x + 1 == a.nx ? 0 : x + 1;
            const int ym = pull_row(y - 1, a), yp = pull_row(y + 1, a);
            typename C::S raw[9];
            double f[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int sy = vb(i) == 1 ? ym : (vb(i) == -1 ? yp : y);
                const int sx = va(i) == 1 ? xl : (va(i) == -1 ? xr : x);
                raw[i] = src[(long long)i * a.plane + (long long)sy * a.nx + sx];
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = C::to_f64(raw[i], i, a.cs);
            double rr;
            bool hit;
            const double g = collide_node<VAR>(f, p, rr, hit);
            acc[8] += g;
            acc[9] = fmin(acc[9], g);
            acc[10] = fmax(acc[10], g);
        }
    }
    __shared__ double sm[kDiagParts][kDiagBlock];
#pragma unroll
    for (int k = 0; k < kDiagParts; ++k) sm[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int s = kDiagBlock / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) diag_fold(&sm[0][threadIdx.x], kDiagBlock, &sm[0][threadIdx.x + s], kDiagBlock);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < kDiagParts; ++k) part[(long long)blockIdx.x * kDiagParts + k] = sm[k][0];
    }
}

// Palinstrophy and entropy density per block: part[block][5] = count, and
// the mean and M2 (Welford / Chan, as in diag_partial) of P = |grad w|^2 / 2
// (w and its gradient by periodic central differences, the same w as
// diag_partial) and of the entropy density of Eq. S,
// s = -sum_i f_i ln(f_i / W_i) = -sum_i f_i log1p(d_i / W_i).
constexpr int kDiagExtParts = 5;

__device__ __forceinline__ void diag_ext_fold(double* a, int sa, const double* b, int sb)
{
    const double na = a[0], nb = b[0];
    const ChanFactors f(na, nb);
    f.merge(a[sa], a[2 * sa], b[sb], b[2 * sb]);
    f.merge(a[3 * sa], a[4 * sa], b[3 * sb], b[4 * sb]);
    a[0] = na + nb;
}

// The library's logarithm out of line: code that hardly any node takes should
// not cost the others registers.
static __device__ __noinline__ double log1p_one(double x) { return log1p(x); }

// Bound by the FP64 pipe (4096^2 float 10.3 ms with the library's logarithm and
// an IEEE division per moment, 4.1 ms now).  Four blocks per SM, all of the
// grid: 64 registers, of which doubles spill 116 bytes; with 78 and three
// blocks the fourth quarter of the grid runs alone (1024^2 float 324 -> 411 us).
template <class C>
__global__ void __launch_bounds__(kDiagBlock, 4)
diag_ext_partial(const typename C::S* __restrict__ src, double* __restrict__ part, StepArgs a)
{
    // u on the tile with a two-node halo, w on the tile with a one-node halo
    constexpr int UW = kTileW + 4, UH = kTileH + 4, WW = kTileW + 2, WH = kTileH + 2;
    __shared__ double sux[UH][UW], suy[UH][UW], sw[WH][WW];
    __shared__ EntropyLogs logs;
    logs.fill();
    double acc[kDiagExtParts] = {0, 0, 0, 0, 0};  // n, mean and M2 of P, of s
    const int ntx = (a.nx + kTileW - 1) / kTileW, nty = (a.ny + kTileH - 1) / kTileH;
    const long long ntiles = (long long)ntx * nty;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int x0 = (int)(tile % ntx) * kTileW, y0 = (int)(tile / ntx) * kTileH;
        __syncthreads();
        for (int q = threadIdx.x; q < UH * UW; q += blockDim.x) {
            const int qy = q / UW, qx = q - qy * UW;
            const int gx = wrap_mod(x0 + qx - 2, a.nx), gy = wrap_mod(y0 + qy - 2, a.ny);
            double r;
            node_macro<C>(src, (long long)gy * a.nx + gx, a, r, sux[qy][qx], suy[qy][qx]);
        }
        __syncthreads();
        // w = d uy/dx - d ux/dy by central differences
        for (int q = threadIdx.x; q < WH * WW; q += blockDim.x) {
            const int qy = q / WW, qx = q - qy * WW, cy = qy + 1, cx = qx + 1;
            sw[qy][qx] = 0.5 * (suy[cy][cx + 1] - suy[cy][cx - 1]) - 0.5 * (sux[cy + 1][cx] - sux[cy - 1][cx]);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < kTileW * kTileH; k += blockDim.x) {
            const int ly = k / kTileW, lx = k - ly * kTileW;
            const int xn = x0 + lx, y = y0 + ly;
            if (xn >= a.nx || y >= a.ny) continue;
            const int cx = lx + 1, cy = ly + 1;
            const double wx = 0.5 * (sw[cy][cx + 1] - sw[cy][cx - 1]);
            const double wy = 0.5 * (sw[cy + 1][cx] - sw[cy - 1][cx]);
            const double pp = 0.5 * (wx * wx + wy * wy);
            const long long n = (long long)y * a.nx + xn;
            // s = -sum W_i (1 + x_i) ln(1 + x_i), x_i = d_i / W_i
            typename C::S raw[9];
            double x[9], se = 0.0;
            bool near = true;
#pragma unroll
            for (int i = 0; i < 9; ++i) raw[i] = src[(long long)i * a.plane + n];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                x[i] = C::relative(raw[i], i, a.cs);
                near &= (__double2hiint(x[i]) & 0x7fffffff) < 0x3fe00000;  // |x| < 1/2
            }
            if (near) {
                // sums by weight class; the weights are 1, 4 and 16 times 1/36
                double sum[3] = {0.0, 0.0, 0.0};
                long long units = 0;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    long long unit;
                    sum[wclass(i)] += logs.near(x[i], leading(x[i]), unit);
                    units += unit << (2 * wclass(i));
                }
                se = -__fma_rn(EntropyLogs::as_double(units), 0x1p-46 * wgt(0),
                               __fma_rn(wgt(0), sum[0], __fma_rn(wgt(1), sum[1], wgt(4) * sum[2])));
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const double d = C::to_f64(src[(long long)i * a.plane + n], i, a.cs);
                    se -= (wgt(i) + d) * log1p_one(d * inv_wgt(i));
                }
            }
            acc[0] += 1.0;
            const double rn = rcp_pos(acc[0]);
            welford_add(rn, acc[1], acc[2], pp);
            welford_add(rn, acc[3], acc[4], se);
        }
    }
    __shared__ double sm[kDiagExtParts][kDiagBlock];
#pragma unroll
    for (int k = 0; k < kDiagExtParts; ++k) sm[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int s = kDiagBlock / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            diag_ext_fold(&sm[0][threadIdx.x], kDiagBlock, &sm[0][threadIdx.x + s], kDiagBlock);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < kDiagExtParts; ++k) part[(long long)blockIdx.x * kDiagExtParts + k] = sm[k][0];
    }
}

// Reduces part[nblocks][5] into out[4] = (mean P, std P, mean s, std s).
__global__ void diag_ext_final(const double* __restrict__ part, int nblocks,
                               double* __restrict__ out, long long total);

// Reduces part[nblocks][11] (fixed order) into out[KBC_DIAG_N], or with raw
// into the merged partial set out[11] (the layout of one block's part).
__global__ void diag_final(const double* __restrict__ part, int nblocks, double* __restrict__ out,
                           long long total, int raw);

}  // namespace kbc
