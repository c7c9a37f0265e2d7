// Host-side launchers, one explicit instantiation per storage codec
// (kbc_f64.cu, kbc_f32.cu, kbc_f16.cu).
#pragma once

#include <type_traits>

#include <cuda_runtime.h>

#include "kbc_adjoint.cuh"
#include "kbc_adjoint_async.cuh"
#include "kbc_guard.cuh"
#include "kbc_kernels.cuh"
#include "kbc_tma.cuh"

namespace kbc {

// Unique id of the current context, which tells one created after
// cudaDeviceReset from the one before; 0 when it cannot be had.
unsigned long long current_context_id();

// rows: vectorised row kernel (nx % (32 * kVec) == 0); nodes: any width;
// bulk: persistent bulk-copy kernel (nx % kTmaTile == 0, F32/F16)
enum class StepKind { rows, nodes, bulk };

// Whether every node finds a thread of its own in the first wave of
// step_nodes: 1024 threads (16 blocks of 64) are resident per SM.
inline bool flat_small(int nx, int ny, int num_sms) { return (long long)nx * ny <= (long long)num_sms * 1024; }

// Whether the two fields of a step stay in L2 (129 MB, of which 100 MB hold
// them without the rest of the step pushing them out: what half B gains by the
// kernels for either side changes sign between 94 and 113 MB; 1024^2 float, 75
// MB, is inside, 1536^2, 170 MB, outside).
inline bool rows_in_l2(long long total, size_t elem) { return 18.0 * (double)elem * (double)total <= 100e6; }

struct Launch {
    const void* src;
    void* dst;
    StepArgs a;
    int variant;
    StepKind kind;
    bool all_f64;   // whole collision in double (exact-gamma mode)
    bool fixup;     // FP64 re-evaluation pass after the step
    cudaStream_t stream;
    int num_sms;
};

// Records msg as the message of kbc_last_error(NULL) and returns code (for
// the entry points that take no handle).
int handle_free_error(int code, const char* msg);

constexpr int kRowBlock = 64;
constexpr int kNodeBlock = 256;

// Launch with programmatic stream serialisation (the kernels start with
// chain_enter(); see there).
template <class... P, class... Q>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t s, Q... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

inline int grid_for(long long total, int block, int num_sms, int per_sm)
{
    long long b = (total + block - 1) / block;
    long long cap = (long long)num_sms * per_sm;
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

template <int VAR, class C>
cudaError_t launch_step_v(const Launch& L)
{
    using S = typename C::S;
    const S* src = static_cast<const S*>(L.src);
    S* dst = static_cast<S*>(L.dst);
    const long long total = (long long)L.a.nx * L.a.ny;
    if (L.all_f64)
        return launch_chained(step_nodes_f64<VAR, C>, grid_for(total, kNodeBlock, L.num_sms, 16), kNodeBlock, 0,
                              L.stream, src, dst, L.a);
    cudaError_t e = cudaSuccess;
    if constexpr (!std::is_same<C, CodecF64>::value) {
        if (L.kind == StepKind::bulk) {
            constexpr size_t smem = tma_smem_bytes<S, kTmaTile>();
            constexpr int threads = kTmaTile / C::kVec + 32;
            static int per_sm = 0;  // resident CTAs per SM, from the occupancy calculator
            if (per_sm == 0) {
                e = cudaFuncSetAttribute(step_tma<VAR, C, kTmaTile>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
                if (e != cudaSuccess) return e;
                int n = 0;
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, step_tma<VAR, C, kTmaTile>,
                                                                  threads, smem);
                if (e != cudaSuccess) return e;
                per_sm = n > 0 ? n : 1;
            }
            const long long tiles = (long long)(L.a.nx / kTmaTile) * L.a.ny;
            long long grid = (long long)L.num_sms * per_sm;
            if (grid > tiles) grid = tiles;
            e = launch_chained(step_tma<VAR, C, kTmaTile>, grid, threads, smem, L.stream, src, dst, L.a);
        }
    }
    if (L.kind == StepKind::rows) {
        constexpr int NV = C::kVec;
        const int nbx = (L.a.nx + kRowBlock * NV - 1) / (kRowBlock * NV);
        const long long grid = (long long)nbx * L.a.ny;
        // see step_rows for what either form is the faster one at
        constexpr bool f32 = std::is_same<C, CodecF32>::value, f16 = std::is_same<C, CodecF16>::value;
        const bool pairs = f16 ? VAR != kLBGK || rows_in_l2(total, sizeof(S))
                               : f32 && VAR != kLBGK && rows_in_l2(total, sizeof(S));
        if constexpr ((f32 && VAR != kLBGK) || f16) {
            if (pairs)
                e = launch_chained(step_rows<VAR, C, NV, kRowBlock, true>, grid, kRowBlock, 0, L.stream, src, dst,
                                   L.a, nbx);
        }
        if constexpr (!f16 || VAR == kLBGK) {
            if (!pairs)
                e = launch_chained(step_rows<VAR, C, NV, kRowBlock, false>, grid, kRowBlock, 0, L.stream, src, dst,
                                   L.a, nbx);
        }
    } else if (L.kind == StepKind::nodes) {
        constexpr int K = flat_nodes<VAR, C>();
        if (K > 1 && !flat_small(L.a.nx, L.a.ny, L.num_sms)) {
            constexpr int per = kFlatBlock * K;
            e = launch_chained(step_nodes<VAR, C, K>, (total + per - 1) / per, kFlatBlock, 0, L.stream, src, dst, L.a);
        } else {
            e = launch_chained(step_nodes<VAR, C, 1>, (total + kFlatBlock - 1) / kFlatBlock, kFlatBlock, 0, L.stream,
                               src, dst, L.a);
        }
    }
    if constexpr (VAR != kLBGK) {
        if (L.fixup && e == cudaSuccess) {
            if constexpr (std::is_same<C, CodecF32>::value) {
                GuardParams gp;
                gp.n2b_h = (float)(-L.a.pd.two_beta);
                gp.n2b_l = (float)(-L.a.pd.two_beta - (double)gp.n2b_h);
                gp.nb = (float)(-L.a.pd.one_m_2beta);
                gp.settle = (double)L.a.pf.guard <= kGuardSettle;
                e = launch_chained(step_guard<VAR>, L.num_sms, kGuardBlock, 0, L.stream, src, dst, L.a, gp);
            } else if constexpr (std::is_same<C, CodecF16>::value) {
                e = launch_chained(step_fixup<VAR, C>, L.num_sms * 2, kNodeBlock, 0, L.stream, src, dst, L.a);
            }
        }
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <class C>
cudaError_t launch_step(const Launch& L)
{
    switch (L.variant) {
    case kLBGK: return launch_step_v<kLBGK, C>(L);
    case kA: return launch_step_v<kA, C>(L);
    case kB: return launch_step_v<kB, C>(L);
    case kC: return launch_step_v<kC, C>(L);
    case kD: return launch_step_v<kD, C>(L);
    default: return cudaErrorInvalidValue;
    }
}

template <class C>
cudaError_t launch_init(const double* rho, const double* ux, const double* uy, void* dst,
                        const StepArgs& a, bool grad, cudaStream_t s, int num_sms)
{
    const long long total = (long long)a.nx * a.ny;
    const int g = grid_for(total, kNodeBlock, num_sms, 16);
    if (grad)
        init_grad<C><<<g, kNodeBlock, 0, s>>>(rho, ux, uy, static_cast<typename C::S*>(dst), a);
    else
        init_feq<C><<<g, kNodeBlock, 0, s>>>(rho, ux, uy, static_cast<typename C::S*>(dst), a);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_set(const double* f, void* dst, const StepArgs& a, cudaStream_t s, int num_sms)
{
    const long long total = (long long)a.nx * a.ny;
    set_populations<C><<<grid_for(total, kNodeBlock, num_sms, 16), kNodeBlock, 0, s>>>(
        f, static_cast<typename C::S*>(dst), a);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_get(const void* src, double* f, const StepArgs& a, cudaStream_t s, int num_sms)
{
    const long long total = (long long)a.nx * a.ny;
    get_populations<C><<<grid_for(total, kNodeBlock, num_sms, 16), kNodeBlock, 0, s>>>(
        static_cast<const typename C::S*>(src), f, a);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_moments(const void* src, double* rho, double* ux, double* uy,
                           const StepArgs& a, cudaStream_t s, int num_sms)
{
    const long long total = (long long)a.nx * a.ny;
    moments<C><<<grid_for(total, kNodeBlock, num_sms, 16), kNodeBlock, 0, s>>>(
        static_cast<const typename C::S*>(src), rho, ux, uy, a);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_probe(const void* src, const long long* nodes, int count, double* f, int* bad,
                         const StepArgs& a, cudaStream_t s, int num_sms)
{
    probe_nodes<C><<<grid_for(count, kNodeBlock, num_sms, 4), kNodeBlock, 0, s>>>(
        static_cast<const typename C::S*>(src), nodes, count, f, bad, a);
    return cudaGetLastError();
}

// number of partial-sum blocks the diagnostics use for this grid
inline int diag_blocks(long long total, int num_sms)
{
    return grid_for(total, kDiagBlock, num_sms, 4);
}

template <class C>
cudaError_t launch_diag(const void* src, double* part, int nblocks, double* out, int variant,
                        const StepArgs& a, cudaStream_t s, int raw)
{
    const typename C::S* p = static_cast<const typename C::S*>(src);
    switch (variant) {
    case kLBGK: diag_partial<kLBGK, C><<<nblocks, kDiagBlock, 0, s>>>(p, part, a); break;
    case kA: diag_partial<kA, C><<<nblocks, kDiagBlock, 0, s>>>(p, part, a); break;
    case kB: diag_partial<kB, C><<<nblocks, kDiagBlock, 0, s>>>(p, part, a); break;
    case kC: diag_partial<kC, C><<<nblocks, kDiagBlock, 0, s>>>(p, part, a); break;
    case kD: diag_partial<kD, C><<<nblocks, kDiagBlock, 0, s>>>(p, part, a); break;
    default: return cudaErrorInvalidValue;
    }
    diag_final<<<1, kDiagBlock, 0, s>>>(part, nblocks, out, (long long)a.nx * a.ny, raw);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_diag_ext(const void* src, double* part, int nblocks, double* out,
                            const StepArgs& a, cudaStream_t s)
{
    diag_ext_partial<C><<<nblocks, kDiagBlock, 0, s>>>(static_cast<const typename C::S*>(src), part, a);
    diag_ext_final<<<1, kDiagBlock, 0, s>>>(part, nblocks, out, (long long)a.nx * a.ny);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- adjoint

// Blocks of the objective and of the reverse steps, one beta partial sum each.
inline int adj_blocks(long long total, int num_sms) { return grid_for(total, 256, num_sms, 8); }

// One reverse step: FP32 storage prefetches each thread's operands by
// asynchronous copies (adj_step_async); the other storages load them node
// by node (adj_step).
template <int VAR, class C>
cudaError_t launch_adj_step_v(const typename C::S* g, const typename C::T* li, typename C::T* lo,
                              double* part, unsigned* fixmask, int nblocks, const StepArgs& a, cudaStream_t s,
                              int num_sms)
{
    cudaError_t e;
    if constexpr (std::is_same<C, CodecF32>::value) {
        // one wave of resident blocks (adj_min_blocks per SM), each with its
        // share of the segments: a second, partly filled wave would start
        // its prefetch pipeline anew
        const int wave = num_sms * adj_min_blocks<VAR, float>();
        e = launch_chained(adj_step_async<VAR>, nblocks < wave ? nblocks : wave, kAdjBlock, 0, s, g, li, lo, part,
                           fixmask, a);
    } else
        e = launch_chained(adj_step<VAR, C>, nblocks, kAdjBlock, 0, s, g, li, lo, part, fixmask, a);
    if constexpr (VAR != kLBGK && !std::is_same<typename C::T, double>::value) {
        // the double redo scans one mask word per thread: a grid sized to the
        // mask (at most the step's), so small grids do not pay for idle blocks;
        // its beta partial sums land in part[0 .. fblocks) in a fixed order
        const long long words = ((long long)a.nx * a.ny + 31) / 32;
        const int fblocks = (int)((words + 255) / 256 < nblocks ? (words + 255) / 256 : nblocks);
        if (e == cudaSuccess)
            e = launch_chained(adj_fixup<VAR, C>, fblocks, 256, 0, s, g, li, lo, part, fixmask, a);
    }
    return e;
}

template <class C>
cudaError_t launch_adj_step(int variant, const void* g, const void* lam_in, void* lam_out,
                            double* part, unsigned* fixmask, int nblocks, const StepArgs& a,
                            cudaStream_t s, int num_sms)
{
    using S = typename C::S;
    using T = typename C::T;
    const S* gp = static_cast<const S*>(g);
    const T* li = static_cast<const T*>(lam_in);
    T* lo = static_cast<T*>(lam_out);
    cudaError_t e;
    switch (variant) {
    case kLBGK: e = launch_adj_step_v<kLBGK, C>(gp, li, lo, part, fixmask, nblocks, a, s, num_sms); break;
    case kA: e = launch_adj_step_v<kA, C>(gp, li, lo, part, fixmask, nblocks, a, s, num_sms); break;
    case kB: e = launch_adj_step_v<kB, C>(gp, li, lo, part, fixmask, nblocks, a, s, num_sms); break;
    case kC: e = launch_adj_step_v<kC, C>(gp, li, lo, part, fixmask, nblocks, a, s, num_sms); break;
    case kD: e = launch_adj_step_v<kD, C>(gp, li, lo, part, fixmask, nblocks, a, s, num_sms); break;
    default: return cudaErrorInvalidValue;
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <class C>
cudaError_t launch_adj_objective(const void* g, const double* tx, const double* ty, int objective,
                                 void* lam, double* part, int nblocks, const StepArgs& a,
                                 cudaStream_t s)
{
    adj_objective<C><<<nblocks, 256, 0, s>>>(static_cast<const typename C::S*>(g), tx, ty, objective,
                                             static_cast<typename C::T*>(lam), part, a);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_adj_grad_u0(const double* rho0, const double* ux0, const double* uy0,
                               const void* lam, double* gx, double* gy, const StepArgs& a,
                               cudaStream_t s, int num_sms)
{
    const long long total = (long long)a.nx * a.ny;
    adj_grad_u0<C><<<grid_for(total, 256, num_sms, 16), 256, 0, s>>>(
        rho0, ux0, uy0, static_cast<const typename C::T*>(lam), gx, gy, a);
    return cudaGetLastError();
}

// explicit instantiations live in the per-codec translation units
#define KBC_DECLARE_CODEC(C)                                                                   \
    extern template cudaError_t launch_step<C>(const Launch&);                                \
    extern template cudaError_t launch_init<C>(const double*, const double*, const double*,   \
                                               void*, const StepArgs&, bool, cudaStream_t,    \
                                               int);                                          \
    extern template cudaError_t launch_set<C>(const double*, void*, const StepArgs&,          \
                                              cudaStream_t, int);                             \
    extern template cudaError_t launch_get<C>(const void*, double*, const StepArgs&,          \
                                              cudaStream_t, int);                             \
    extern template cudaError_t launch_moments<C>(const void*, double*, double*, double*,     \
                                                  const StepArgs&, cudaStream_t, int);        \
    extern template cudaError_t launch_diag<C>(const void*, double*, int, double*, int,       \
                                               const StepArgs&, cudaStream_t, int);           \
    extern template cudaError_t launch_probe<C>(const void*, const long long*, int, double*,  \
                                                int*, const StepArgs&, cudaStream_t, int);    \
    extern template cudaError_t launch_diag_ext<C>(const void*, double*, int, double*,        \
                                                   const StepArgs&, cudaStream_t);            \
    extern template cudaError_t launch_adj_step<C>(int, const void*, const void*, void*,      \
                                                   double*, unsigned*, int, const StepArgs&,  \
                                                   cudaStream_t, int);                        \
    extern template cudaError_t launch_adj_objective<C>(const void*, const double*,           \
                                                        const double*, int, void*, double*,   \
                                                        int, const StepArgs&, cudaStream_t);  \
    extern template cudaError_t launch_adj_grad_u0<C>(const double*, const double*,           \
                                                      const double*, const void*, double*,    \
                                                      double*, const StepArgs&, cudaStream_t, \
                                                      int);

#define KBC_DEFINE_CODEC(C)                                                                    \
    template cudaError_t launch_step<C>(const Launch&);                                       \
    template cudaError_t launch_init<C>(const double*, const double*, const double*, void*,   \
                                        const StepArgs&, bool, cudaStream_t, int);            \
    template cudaError_t launch_set<C>(const double*, void*, const StepArgs&, cudaStream_t,   \
                                       int);                                                  \
    template cudaError_t launch_get<C>(const void*, double*, const StepArgs&, cudaStream_t,   \
                                       int);                                                  \
    template cudaError_t launch_moments<C>(const void*, double*, double*, double*,            \
                                           const StepArgs&, cudaStream_t, int);               \
    template cudaError_t launch_diag<C>(const void*, double*, int, double*, int,              \
                                        const StepArgs&, cudaStream_t, int);                  \
    template cudaError_t launch_probe<C>(const void*, const long long*, int, double*, int*,   \
                                         const StepArgs&, cudaStream_t, int);                 \
    template cudaError_t launch_diag_ext<C>(const void*, double*, int, double*,               \
                                            const StepArgs&, cudaStream_t);                   \
    template cudaError_t launch_adj_step<C>(int, const void*, const void*, void*, double*,    \
                                            unsigned*, int, const StepArgs&, cudaStream_t,    \
                                            int);                                             \
    template cudaError_t launch_adj_objective<C>(const void*, const double*, const double*,   \
                                                 int, void*, double*, int, const StepArgs&,   \
                                                 cudaStream_t);                               \
    template cudaError_t launch_adj_grad_u0<C>(const double*, const double*, const double*,   \
                                               const void*, double*, double*,                 \
                                               const StepArgs&, cudaStream_t, int);

#ifndef KBC_CODEC_TU
KBC_DECLARE_CODEC(CodecF64)
KBC_DECLARE_CODEC(CodecF32)
KBC_DECLARE_CODEC(CodecF16)
#endif

}  // namespace kbc
