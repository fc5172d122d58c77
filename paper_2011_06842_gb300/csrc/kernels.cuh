// Kernels of the FEWHA hot path and the per-precision implementation
// object that launches them (internal to libfewha).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <cstddef>
#include <cstring>
#include <type_traits>
#include <vector>

#include "mcao.cuh"
#include "plan.h"
#include "solver.cuh"

namespace fewha {

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T *dyn_smem()
{
    extern __shared__ __align__(16) unsigned char fewha_smem[];
    return reinterpret_cast<T *>(fewha_smem);
}

// Kernel arguments are copied into shared memory once: the phases are not
// inlined and take them by reference, which would otherwise place them in
// local memory (a load through the L1 for every field read).
template <typename T, typename S>
__device__ __forceinline__ void args_to_smem(const Args<T, S> &src, Args<T, S> &dst)
{
    const int4 *s = reinterpret_cast<const int4 *>(&src);
    int4 *d = reinterpret_cast<int4 *>(&dst);
    for (int e = threadIdx.x; e < (int)(sizeof(Args<T, S>) / sizeof(int4)); e += blockDim.x) d[e] = s[e];
    __syncthreads();
}

// --- the operator by itself: y = M x, b = W^{-T} A^T C^{-1} s, nodal = W^{-1} c --
// The solver's phases as a chain of kernels.  Split form (split_levels): the
// coarser synthesis levels on one CTA per layer, the finest split_depth levels
// tiled over all CTAs, and back the same way; whole form: every level on the
// layer's CTA.  One CTA per layer for every level left 143 of 152 SMs idle for
// most of an ELT application.
// The kernels are launched with programmatic stream serialisation: each
// lets the next one start (its launch, its arguments into shared memory) and
// waits for the previous one's results before it touches memory.  The first
// of a chain is launched without it.
// ELT, us per call before and after: apply FP64 274 and 77, FP32 50 and 36; rhs
// with 16-bit slopes 35.5 and 25.9; fit FP32 20.3 and 20.1, FP64 147 and 33.
__device__ __forceinline__ void pdl_begin()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Several vectors at once: vector v is applied by CTAs [v*per, (v+1)*per) with
// its own scratch buffers, so the transforms of all vectors run side by side.
constexpr int kMaxVec = FEWHA_MAX_MULTI;

template <typename T, typename S>
struct MultiArgs {
    Args<T, S> a[kMaxVec];
    int per;
};

template <typename T, typename S>
__device__ __forceinline__ void op_args(const Args<T, S> &P, Args<T, S> &A)
{
    args_to_smem(P, A);
    pdl_begin();
}
template <typename T, typename S>
__device__ __forceinline__ void op_args(const MultiArgs<T, S> &P, Args<T, S> &A)
{
    args_to_smem(P.a[blockIdx.x / P.per], A);
    pdl_begin();
}

// W^{-1} x: the coarser levels (whole form: every level, to nodal)
template <typename T, typename S, class P, bool WHOLE>
__global__ void __launch_bounds__(kThreads, 1) k_op_coarse(const __grid_constant__ P p)
{
    __shared__ __align__(16) Args<T, S> A;
    op_args(p, A);
    phase_coarse_synth<WHOLE>(A, A.x, dyn_smem<T>());
}

// W^{-1} x: tiled level LV (0 = finest, to nodal)
template <typename T, typename S, class P, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_op_synth(const __grid_constant__ P p)
{
    __shared__ __align__(16) Args<T, S> A;
    op_args(p, A);
    phase_fine_synth<LV>(A, A.x, dyn_smem<T>());
}

// psi = Gamma^T C Gamma P nodal (RHS = false) or Gamma^T C s (RHS = true)
template <typename T, typename S, class P, bool RHS>
__global__ void __launch_bounds__(kThreads, 1) k_op_wfs(const __grid_constant__ P p)
{
    __shared__ __align__(16) Args<T, S> A;
    op_args(p, A);
    wfs_phase<T, S, RHS>(A, dyn_smem<T>());
}

// u = P^T psi
template <typename T, typename S, class P>
__global__ void __launch_bounds__(kThreads, 1) k_op_gather(const __grid_constant__ P p)
{
    __shared__ __align__(16) Args<T, S> A;
    op_args(p, A);
    band_gather<T, S>(A, dyn_smem<T>());
}

// W^{-T} u: tiled level LV (split form)
template <typename T, typename S, class P, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_op_analysis(const __grid_constant__ P p)
{
    __shared__ __align__(16) Args<T, S> A;
    op_args(p, A);
    phase_D1<LV>(A, dyn_smem<T>());
}

// y = W^{-T} u + alpha D x (RHS = false) or y = W^{-T} u (RHS = true)
template <typename T, typename S, class P, bool RHS, bool WHOLE>
__global__ void __launch_bounds__(kThreads, 1) k_op_update(const __grid_constant__ P p)
{
    __shared__ __align__(16) Args<T, S> A;
    op_args(p, A);
    constexpr int W = VW<T>::W;
    analysis_update<WHOLE>(A, dyn_smem<T>(), [&](long e, const T (&v)[W]) {
        T y[W], x[W], ad[W];
        if (!RHS) {
            vld(A.x + e, x);
            vld_nc(A.geo.alpha_d + e, ad);
        }
#pragma unroll
        for (int i = 0; i < W; i++) y[i] = RHS ? v[i] : v[i] + ad[i] * x[i];
        vst(A.y + e, y);
    });
}

// --- mirror side of the reconstructor loop (Algorithm 3) --------------------
// One deformable mirror conjugated to the ground with its actuators on the
// (n_s+1)^2 pupil nodes (reading of the fitting operator F).
template <typename T>
struct FitTab {
    long off[FEWHA_MAX_LAYERS];
    int n[FEWHA_MAX_LAYERS];
    int L, m;
    const int *fk;  // [L][m] lower node of pupil index j (both axes)
    const T *fw;    // [L][m] fractional position
};

// a~ = F W^{-1} c with nodal = W^{-1} c already in place: on-axis bilinear
// sample of every layer at every actuator, summed over layers.
template <typename T, typename S>
__global__ void k_fit(const __grid_constant__ FitTab<T> F, const S *__restrict__ nodal, T *__restrict__ a)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= F.m * F.m) return;
    const int i = e / F.m, j = e - i * F.m;
    T v = 0;
    for (int l = 0; l < F.L; l++) {
        const int n = F.n[l];
        const int kx = F.fk[l * F.m + j], ky = F.fk[l * F.m + i];
        const T wx = F.fw[l * F.m + j], wy = F.fw[l * F.m + i];
        const S *Lp = nodal + F.off[l] + (long)ky * n + kx;
        const T v00 = Cv<S>::ld(Lp[0]), v01 = Cv<S>::ld(Lp[1]);
        const T v10 = Cv<S>::ld(Lp[n]), v11 = Cv<S>::ld(Lp[n + 1]);
        v += (T(1) - wy) * ((T(1) - wx) * v00 + wx * v01) + wy * ((T(1) - wx) * v10 + wx * v11);
    }
    a[e] = v;
}

// Pseudo-open-loop slopes: s_out = s + Gamma a for every guide star (the
// ground mirror adds the same phase to every sensor).
template <typename T, typename S>
__global__ void k_pol(const S *s_in, const T *__restrict__ a, S *s_out, int G, int ns)  // s_out may be s_in
{
    const int m = ns + 1, per = ns * ns;
    const long total = (long)G * per;
    for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int g = (int)(idx / per), e = (int)(idx - (long)g * per);
        const int i = e / ns, j = e - i * ns;
        const T p00 = a[i * m + j], p01 = a[i * m + j + 1];
        const T p10 = a[(i + 1) * m + j], p11 = a[(i + 1) * m + j + 1];
        const T gx = T(0.5) * ((p01 - p00) + (p11 - p10));
        const T gy = T(0.5) * ((p10 - p00) + (p11 - p01));
        const size_t b = (size_t)g * 2 * per;
        s_out[b + e] = Cv<S>::st(Cv<S>::ld(s_in[b + e]) + gx);
        s_out[b + per + e] = Cv<S>::st(Cv<S>::ld(s_in[b + per + e]) + gy);
    }
}

// Gain control: closed loop a_next = a_i + gain (a~ - a_{i-1}); open loop
// a_next = (1 - gain) a_i + gain a~.
template <typename T>
__global__ void k_control(int closed, T gain, const T *__restrict__ am1, const T *__restrict__ ai,
                          const T *__restrict__ af, T *__restrict__ an, int na)
{
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < na; e += gridDim.x * blockDim.x)
        an[e] = closed ? ai[e] + gain * (af[e] - am1[e]) : (T(1) - gain) * ai[e] + gain * af[e];
}

// --- solver phases, one kernel each (FEWHA_LAUNCH_PHASES) -------------------
#define FEWHA_PHASE_GUARD                                             \
    __shared__ Scal sc;                                               \
    __shared__ double sred[kSred];                                   \
    __shared__ __align__(16) Args<T, S> A;                            \
    args_to_smem(Ap, A);                                              \
    (void)sred;                                                       \
    if (ldcgi(&A.rec->done) || ldcgi(&A.rec->status)) return;         \
    const Basis b = basis_info(A);                                    \
    (void)b;

// R1: weighted slopes -> psi, and the Gram matrix of the old basis
template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_rhs_wfs(const __grid_constant__ Args<T, S> Ap)
{
    __shared__ __align__(16) Args<T, S> A;
    args_to_smem(Ap, A);
    if (!A.rhs_in_state) wfs_phase<T, S, true>(A, dyn_smem<T>());
    const Basis b = basis_info(A);
    if (b.kv > 0) phase_gram<T, S>(A, b, dyn_smem<T>(), (int)(A.smem_bytes / sizeof(T)));
}

// R2: u = P^T psi; the last CTA also factorises the Gram matrix
template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_rhs_gather(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    if (!A.rhs_in_state) band_gather<T, S>(A, dyn_smem<T>());
    if (b.kv > 0 && A.vrank() == A.ncta - 1) phase_factor<T, S>(A, b, sc);
}

// R3: the finest analysis level of u (split form), then b, r0 and P^T r0
template <typename T, typename S, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_rhs_D1(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    if (!A.rhs_in_state) phase_D1<LV>(A, dyn_smem<T>());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_rhs_update(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    if (A.rhs_in_state)
        phase_rhs_update<T, S, true>(A, b, dyn_smem<T>(), sred);
    else
        phase_rhs_update<T, S, false>(A, b, dyn_smem<T>(), sred);
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_init(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    if (b.kv > 0) phase_init<T, S>(A, b, sc, sred);
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_UA1(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    phase_UA1<T, S>(A, b, k, dyn_smem<T>(), sc, sred);
}

template <typename T, typename S, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_A2(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    phase_A2<LV>(A, b, k, dyn_smem<T>());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_B(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    typename AccT<T>::type acc[1] = {wfs_phase<T, S, false>(A, dyn_smem<T>())};
    const int slots[1] = {kSlotB + (k & 1)};
    block_partials<1>(acc, A.part, slots, sred, A.vrank());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_C(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    phase_C<T, S>(A, b, k, dyn_smem<T>(), sc);
}

template <typename T, typename S, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_D1(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    phase_D1<LV>(A, dyn_smem<T>());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_D2E(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    phase_D2E<T, S>(A, b, k, dyn_smem<T>(), sred);
}

// residual replacement after iteration k (phases TU, TA2, TB, TC, TD1, TE)
template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_TU(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    phase_TU<T>(*TrView<T, S>::get(A), dyn_smem<T>());
}

template <typename T, typename S, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_TA2(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    const Args<T, T> &V = *TrView<T, S>::get(A);
    phase_fine_synth<LV>(V, V.c, dyn_smem<T>());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_TB(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    wfs_phase<T, T, false>(*TrView<T, S>::get(A), dyn_smem<T>());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_TC(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    band_gather<T, T>(*TrView<T, S>::get(A), dyn_smem<T>());
}

template <typename T, typename S, int LV>
__global__ void __launch_bounds__(kThreads, 1) k_TD1(const __grid_constant__ Args<T, S> Ap)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    phase_D1<LV>(*TrView<T, S>::get(A), dyn_smem<T>());
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_TE(const __grid_constant__ Args<T, S> Ap, int k)
{
    FEWHA_PHASE_GUARD
    (void)sc;
    phase_TE<T>(*TrView<T, S>::get(A), b, k, dyn_smem<T>(), sred);
}

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 1) k_finish(const __grid_constant__ Args<T, S> Ap)
{
    __shared__ Scal sc;
    __shared__ __align__(16) Args<T, S> A;
    args_to_smem(Ap, A);
    if (A.c_out) phase_store_c<T, S>(A, blockIdx.x, gridDim.x);  // this launch's CTAs
    if (A.vrank() != 0) return;
    const Basis b = basis_info(A);
    int K = ldcgi(&A.rec->done) ? ldcgi(&A.rec->iters) : A.max_iter;
    phase_finish<T, S>(A, b, K, sc);
}

// Residual replacement after iteration k inside the persistent kernel (phases
// TU, TA2, TB, TC, TD1, TE, each followed by the group's barrier); false when a
// barrier reports an error.  ti: trace slot of the next barrier.
template <typename T>
__device__ __forceinline__ bool true_residual_phases(const Args<T, T> &V, const Basis &b, int k, double *sred,
                                                     int rank, int &ti)
{
    T *sm = dyn_smem<T>();
    const bool split = split_levels(V), deep = split && split_depth(V.geo) > 1;
    auto sync = [&](int tag) -> bool {
        unsigned long long *slot = (V.trace && ti < V.trace_cap) ? V.trace + 4 * ti : nullptr;
        if (slot && rank == 0 && threadIdx.x == 0) slot[3] = (unsigned long long)tag;
        ti++;
        return grid_sync(V.rec, V.timeout_ns, V.ncta, rank, slot);
    };
    phase_TU<T>(V, sm);
    if (!sync(20)) return false;
    if (deep) {
        phase_fine_synth<1>(V, V.c, sm);
        if (!sync(26)) return false;
    }
    if (split) {
        phase_fine_synth(V, V.c, sm);
        if (!sync(21)) return false;
    }
    wfs_phase<T, T, false>(V, sm);
    if (!sync(22)) return false;
    band_gather<T, T>(V, sm);
    if (!sync(23)) return false;
    if (split) {
        phase_D1(V, sm);
        if (!sync(24)) return false;
    }
    if (deep) {
        phase_D1<1>(V, sm);
        if (!sync(27)) return false;
    }
    phase_TE<T>(V, b, k, sm, sred);
    return sync(25);
}

// --- the whole time step of one instance, run by its group of CTAs ----------
// TR: the kernel variant with the residual replacement (fewha_solve_opts.
// true_res_every > 0); RIS: the variant for a right-hand side already in the
// state (fewha_solve_opts.rhs_in_state).  The default variant carries the
// code of neither, so its register allocation does not depend on them.
template <typename T, typename S, bool TR, bool RIS = false>
__device__ void solve_body(const Args<T, S> &A, Scal &sc, double *sred)
{
    T *sm = dyn_smem<T>();
    const unsigned long long to = A.timeout_ns;
    const Basis b = basis_info(A);
    const int rank = A.vrank();
    int ti = 0;  // trace slot of the next barrier
    // barrier of the group with the optional phase trace (tag = phase id)
    auto sync = [&](int tag) -> bool {
        unsigned long long *slot = (A.trace && ti < A.trace_cap) ? A.trace + 4 * ti : nullptr;
        if (slot && rank == 0 && threadIdx.x == 0) slot[3] = (unsigned long long)tag;
        bool ok = grid_sync(A.rec, to, A.ncta, rank, slot);
        ti++;
        return ok;
    };
    int K = A.max_iter;
    const bool split = split_levels(A);  // uniform over the instance's CTAs
    const bool deep = split && split_depth(A.geo) > 1;
    const Args<T, T> *V = nullptr;  // residual replacement's view of the arguments
    if constexpr (TR) V = TrView<T, S>::get(A);
    trace_begin(A.trace != nullptr);
    constexpr bool rhs = !RIS;  // form the right-hand side (else it is in the state)
    do {
        if (rhs) wfs_phase<T, S, true>(A, sm);
        if (b.kv > 0) phase_gram<T, S>(A, b, sm, (int)(A.smem_bytes / sizeof(T)));
        if ((rhs || b.kv > 0) && !sync(1)) break;
        if (rhs) band_gather<T, S>(A, sm);
        if (b.kv > 0 && rank == A.ncta - 1) phase_factor<T, S>(A, b, sc);
        if ((rhs || b.kv > 0) && !sync(2)) break;
        if (split && rhs) {
            phase_D1(A, sm);  // the finest analysis level of u
            if (!sync(6)) break;
            if (deep) {
                phase_D1<1>(A, sm);
                if (!sync(7)) break;
            }
        }
        phase_rhs_update<T, S, RIS>(A, b, sm, sred);  // b, r0 and P^T r0
        if (!sync(3)) break;
        if (b.kv > 0) {
            phase_init<T, S>(A, b, sc, sred);
            if (!sync(5)) break;
        }
        for (int k = 0; k < A.max_iter; k++) {
            // UA1's partial sums join the WFS phase's block reduction
            typename AccT<T>::type ua[2];
            if (!phase_UA1<T, S>(A, b, k, sm, sc, sred, true, ua)) {
                K = k;
                break;
            }
            if (!sync(10)) break;
            if (deep) {
                phase_A2<1>(A, b, k, sm);
                if (!sync(17)) break;
            }
            if (split) {
                phase_A2(A, b, k, sm);
                if (!sync(16)) break;
            }
            {
                typename AccT<T>::type acc[3] = {wfs_phase<T, S, false>(A, sm), ua[0], ua[1]};
                const int slots[3] = {kSlotB + (k & 1), kSlotA + (k & 1) * 2, kSlotA + (k & 1) * 2 + 1};
                block_partials<3>(acc, A.part, slots, sred, rank);
            }
            if (!sync(12)) break;
            if (!phase_C<T, S>(A, b, k, sm, sc, true)) {
                K = k;
                break;
            }
            if (!sync(13)) break;
            if (split) {
                phase_D1(A, sm);
                if (!sync(14)) break;
            }
            if (deep) {
                phase_D1<1>(A, sm);
                if (!sync(18)) break;
            }
            phase_D2E<T, S>(A, b, k, sm, sred, &sc.alpha);
            if (!sync(15)) break;
            // residual replacement: r = b - M c, then iteration k+1's scalars
            // come from it
            if constexpr (TR) {
                if ((k + 1) % A.true_res_every == 0 && !true_residual_phases<T>(*V, b, k, sred, rank, ti)) break;
            }
        }
    } while (0);
    // on a device-side error the stats carry the status; the other fields are
    // then not meaningful
    if (A.c_out) phase_store_c<T, S>(A, rank, A.ncta);
    if (rank == 0) phase_finish<T, S>(A, b, K, sc);
}

// One instance on the whole grid (cooperative launch).
template <typename T, typename S, bool TR, bool RIS = false>
__global__ void __launch_bounds__(kThreads, 1) k_solve_persistent(const __grid_constant__ Args<T, S> Ap)
{
    __shared__ Scal sc;
    __shared__ double sred[kSred];
    __shared__ __align__(16) Args<T, S> A;
    args_to_smem(Ap, A);
    solve_body<T, S, TR, RIS>(A, sc, sred);
}

// Many instances in one cooperative launch: CTA c runs instance cta_inst[c]
// with the group of CTAs [inst.cta0, inst.cta0 + inst.ncta).
template <typename T, typename S, bool TR>
__global__ void __launch_bounds__(kThreads, 1) k_solve_batched(const Args<T, S> *inst, const int *cta_inst,
                                                              int nrounds, int total, Record *brec,
                                                              unsigned long long timeout_ns)
{
    // Instances run in rounds: in round r, CTA c runs instance cta_inst[r * total + c]
    // (-1: idle in this round); a barrier over the whole launch separates rounds, so
    // one launch can give a few large instances many CTAs and then the small ones.
    __shared__ Scal sc;
    __shared__ double sred[kSred];
    __shared__ __align__(16) Args<T, S> A;
    for (int r = 0; r < nrounds; r++) {
        const int i = cta_inst[r * total + blockIdx.x];
        if (i >= 0) {
            args_to_smem(inst[i], A);
            solve_body<T, S, TR>(A, sc, sred);
        }
        if (r + 1 < nrounds && !grid_sync(brec, timeout_ns, total, blockIdx.x)) return;
    }
}

// Resets the record flags and the barrier of every instance of a batch.
template <typename T, typename S>
__global__ void k_batch_reset(const Args<T, S> *inst, int n, Record *brec)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        brec->status = 0;
        brec->bar.count = brec->bar.gen = 0;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        Record *r = inst[i].rec;
        r->status = r->done = r->iters = r->chol_ok = 0;
        r->bar.count = r->bar.gen = 0;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
#define CK(x)                                   \
    do {                                        \
        cudaError_t _e = (x);                   \
        if (_e != cudaSuccess) return FEWHA_ERR_CUDA; \
    } while (0)

template <typename T>
static int upload(const std::vector<T> &v, T **d)
{
    *d = nullptr;
    if (v.empty()) return FEWHA_OK;
    if (cudaMalloc(d, v.size() * sizeof(T)) != cudaSuccess) return FEWHA_ERR_NOMEM;
    CK(cudaMemcpy(*d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
    return FEWHA_OK;
}

struct ImplBase {
    virtual ~ImplBase() {}
    virtual int init(int grid) = 0;
    virtual int get_invJ(double *host) const = 0;
    virtual int apply(const void *x, void *y, cudaStream_t s) = 0;
    // mirror side of Algorithm 3 (ground DM on the pupil nodes)
    virtual int fit(const void *c, void *a, cudaStream_t s) = 0;
    virtual int pol_slopes(const void *s_in, const void *a, void *s_out, cudaStream_t s) = 0;
    virtual int control(int closed, double gain, const void *am1, const void *ai, const void *af, void *an,
                        cudaStream_t s) = 0;
    // MCAO fitting onto several mirrors: plan (tables, work vectors), fit, free
    virtual int mcao_create(const fewha_mcao_desc *d, void **plan, long *n_act) = 0;
    virtual int mcao_fit(void *plan, const void *c, void *a, int iters, cudaStream_t s) = 0;
    virtual void mcao_destroy(void *plan) = 0;
    // y_v = M x_v for v < nvec (x_v = x + v*ldx, y_v = y + v*ldy), nvec <= kMaxVec
    virtual int apply_multi(const void *x, long ldx, void *y, long ldy, int nvec, cudaStream_t s) = 0;
    virtual int rhs(const void *sl, void *b, cudaStream_t s) = 0;
    virtual int solve(const void *sl, void *c, const fewha_state *st, const fewha_solve_opts *o,
                      fewha_stats *stats, cudaStream_t s) = 0;
    virtual int set_invJ(const std::vector<double> &invJ) = 0;
    // C_eta^{-1}: weight of guide star g on its lit subapertures (plan.geom.gs[g].weight)
    virtual int set_weights() = 0;
    virtual void set_trace(unsigned long long *buf, int cap) = 0;
    virtual void set_timeout(unsigned long long ns) = 0;
    // --- batched launch support (many instances, one cooperative kernel) ---
    virtual size_t args_size() const = 0;
    virtual int precision_id() const = 0;
    // WFS tile shape for a group of `ctas` CTAs, and the dynamic shared memory it needs
    virtual int tiles_for(int ctas, int *ty, int *tx) const = 0;
    virtual size_t smem_for(int ty, int tx) const = 0;
    // the same, with what a faster plan needs if a group of nct CTAs runs it (a
    // batch's solver, or the operator chain)
    virtual size_t smem_want(int ty, int tx, int nct, bool chain) const = 0;
    // host copy of this instance's kernel arguments for one time step
    virtual int batch_args(void *out, const void *sl, void *c, const fewha_state *st, const fewha_solve_opts *o,
                           fewha_stats *stats, int cta0, int ncta, int ty, int tx, size_t smem) const = 0;
    // CTAs that can be co-resident for the batched kernel with `smem` bytes
    virtual int batch_capacity(size_t smem, int *max_ctas) const = 0;
    virtual int launch_batched(const void *d_args, const int *d_map, int n, int total, size_t smem, int nrounds,
                               Record *brec, int true_res, cudaStream_t s) const = 0;
    // y = M x with every scratch buffer carved from caller-provided device
    // memory (no allocation); FEWHA_ERR_SCRATCH if `bytes` is too small.
    virtual int apply_in_scratch(const void *x, void *y, void *scratch, size_t bytes, cudaStream_t s) = 0;
    virtual void launch_info(fewha_launch_info *out) const = 0;
    // P^T band heights (layer rows) on the largest and on the smaller layers, for every launch; and back to
    // the library's choice
    virtual int set_bands(int rows_large, int rows_small) = 0;
    virtual int auto_bands() = 0;
    // P^T bands that a group of nct CTAs with sm bytes of shared memory runs
    virtual int group_bands(int nct, size_t sm) const = 0;
};

template <typename T, typename S>
struct Impl : ImplBase {
    const Plan &P;
    Args<T, S> base{};
    int ncta = 1;
    size_t smem = 0;
    std::vector<void *> owned;
    const int *fit_k = nullptr;          // fitting tables (device)
    const T *fit_w = nullptr;
    unsigned char *multi_buf = nullptr;  // scratch of apply_multi (allocated on first use)
    size_t multi_stride = 0;

    static constexpr int kBandLarge = 8, kBandSmall = 4;  // default P^T band heights (plan_bands)
    size_t sm_fixed = 0;  // dynamic shared memory of every phase but the WFS tiles
    size_t sm_base = 0;   // of the layer and WFS phases alone (before the P^T bands)
    size_t sm_layer_ = 0; // of the layer phases alone
    size_t sm_fine_ = 0;  // of the tiled wavelet levels alone
    size_t ll_elems() const { return (size_t)P.n / 4 + P.n / 16 + 1; }  // Args::ll
    // Args::ll of W^{-1} c (fit, mcao_fit).  A loop may fit one frame while it forms the
    // next right-hand side on another stream of the same handle: the two calls write no buffer in common.
    T *ll_nodal = nullptr;
    std::vector<void *> band_owned;  // device tables of the P^T bands (replaced by plan_bands)
    int band_rows_large = 0, band_rows_small = 0;
    bool bands_set = false;  // by a caller (set_bands): they hold for every group
    // Second P^T band plan, for groups with several bands per CTA: the tallest
    // bands (kBandOutputs outputs each).  Staging and contracting one pass of a band
    // (the guide stars whose pupil rows fit at once) takes a CTA about 3.2 us in FP32
    // and 3.8 us in FP64, and every adjoint value it stages 1.3 and 2.6 ns more, so a
    // pass costs as much as kPassValues values (within 20 % on one CTA, band heights
    // 2 to 128, 7 geometries; a 16-row band of a 64^2 ELT layer takes 14 us, its four
    // 4-row bands 19).  A batch of 24 tiny, 24 medium and 16 ELT instances: 2425 us
    // with one plan, 2270 with two.
    static constexpr int kPassValues = sizeof(T) == 8 ? 1500 : 2500;
    Geo<T> few{};
    std::vector<void *> few_owned;
    size_t few_fixed = 0;  // its sm_fixed; 0: no such plan
    std::vector<long> band_cost;  // of the bands of the last plan, in staged values
    // by the CTAs of a group (from 0): whether it runs the second plan in the
    // solver and in the operator chain (choose_plans)
    std::vector<char> few_solver, few_chain;

    explicit Impl(const Plan &p) : P(p) {}

    // WFS tile bytes: per-layer halo values and the weighted slopes
    size_t wfs_bytes(int ty, int tx) const
    {
        return ((size_t)P.L * (ty + 2) * (tx + 2) + 2 * (size_t)(ty + 1) * (tx + 1)) * sizeof(T);
    }

    // WFS tiles of ty x tx pupil nodes on every sensor's grid: tiles per row
    // and the cumulative work-item count per sensor
    void set_tiles(Geo<T> &G, int ty, int tx) const
    {
        G.tile_y = ty;
        G.tile_x = tx;
        G.gs_tile0[0] = 0;
        for (int g = 0; g < P.G; g++) {
            G.gs_tiles_x[g] = (P.gm[g] + tx - 1) / tx;
            G.gs_tile0[g + 1] = G.gs_tile0[g] + G.gs_tiles_x[g] * ((P.gm[g] + ty - 1) / ty);
        }
    }

    // WFS tile shape: a square tile if the caller fixed one, else the shape
    // (8..32 nodes per side) whose work per round of `ctas` CTAs is least
    // among those whose shared memory fits
    int tiles_for(int ctas, int *ty_out, int *tx_out) const override
    {
        double best = 1e300;
        *ty_out = *tx_out = 0;
        const int cand[4] = {8, 16, 24, 32};
        for (int a = 0; a < 4; a++)
            for (int c = 0; c < 4; c++) {
                int ty = cand[a], tx = cand[c];
                if (P.geom.tile) ty = tx = P.geom.tile;
                if (wfs_bytes(ty, tx) > 200 * 1024) continue;
                int tiles = 0;
                for (int g = 0; g < P.G; g++) tiles += ((P.gm[g] + ty - 1) / ty) * ((P.gm[g] + tx - 1) / tx);
                const int rounds = (tiles + ctas - 1) / ctas;
                const double cost = rounds * ((double)(ty + 2) * (tx + 2) + 64.0);
                if (cost < best - 1e-9) {
                    best = cost;
                    *ty_out = ty;
                    *tx_out = tx;
                }
            }
        return *ty_out ? FEWHA_OK : FEWHA_ERR_GEOMETRY;
    }

    size_t smem_for(int ty, int tx) const override { return std::max(sm_fixed, wfs_bytes(ty, tx)); }
    // with room for the second band plan if the group runs it (shared memory that
    // is not needed costs L1 cache: 3 % of an ELT step on 72 CTAs)
    size_t smem_want(int ty, int tx, int nct, bool chain) const override
    {
        return std::max(smem_for(ty, tx), few_wanted(nct, chain) ? few_fixed : 0);
    }

    bool few_wanted(int nct, bool chain) const
    {
        const std::vector<char> &v = chain ? few_chain : few_solver;
        return !bands_set && nct < (int)v.size() && v[nct];
    }

    // Which groups run the second plan: those whose CTAs then have fewer bands and
    // whose busiest CTA does not take longer (to 2 %, the model's reach).  Fewer
    // bands alone are not enough: LTAO on 36 CTAs 855 us a step with 8- and 4-row
    // bands and 1012 with the tallest, ELT in FP64 on 48 CTAs 1175 and 1275, against
    // 2248 and 1841 for the 16 m telescope on one CTA.  In the operator chain, where the
    // gather is a kernel of its own, fewer bands win whenever the standard plan
    // stages weight tables per band (ELT in FP64, 8 vectors: 352 and 319 us); without
    // the tables the model holds there too (LTAO, 4 vectors: 112 and 129 us).
    void choose_plans(const std::vector<long> &few_cost)
    {
        const Geo<T> &G = base.geo;
        few_solver.assign(G.nbands + 1, 0);  // on more CTAs every band has its own
        few_chain = few_solver;
        for (int n = 1; n <= G.nbands; n++) {
            if ((few.nbands + n - 1) / n >= (G.nbands + n - 1) / n) continue;
            auto busiest = [n](const std::vector<long> &cost) {
                std::vector<long> cta(n, 0);
                for (size_t w = 0; w < cost.size(); w++) cta[w % n] += cost[w];
                return *std::max_element(cta.begin(), cta.end());
            };
            few_solver[n] = busiest(few_cost) < 1.02 * busiest(band_cost);
            few_chain[n] = G.stage_tab || few_solver[n];
        }
    }

    // the P^T band plan for a group of nct CTAs with sm bytes of shared memory
    void choose_bands(Geo<T> &G, int nct, size_t sm, bool chain) const
    {
        if (!few_wanted(nct, chain) || few_fixed > sm) return;
        G.nbands = few.nbands;
        G.band_layer = few.band_layer, G.band_row0 = few.band_row0, G.band_rows = few.band_rows;
        G.band_ilo = few.band_ilo, G.band_ihi = few.band_ihi;
        G.band_gend = few.band_gend, G.band_gc = few.band_gc, G.band_gr = few.band_gr;
        G.rows_chunk = few.rows_chunk, G.stage_tab = few.stage_tab;
        G.band_ycnt = few.band_ycnt, G.band_yrow = few.band_yrow, G.band_yw = few.band_yw;
        G.ybr = few.ybr, G.ymax = few.ymax;
    }
    size_t args_size() const override { return sizeof(Args<T, S>); }
    int precision_id() const override
    {
        return sizeof(T) == 8 ? FEWHA_F64 : (sizeof(S) == 2 ? FEWHA_BF16S : FEWHA_F32);
    }
    ~Impl() override
    {
        for (void *q : owned) cudaFree(q);
        for (void *q : band_owned) cudaFree(q);
        for (void *q : few_owned) cudaFree(q);
    }

    template <typename U>
    int up(const std::vector<U> &v, const U **d)
    {
        U *dd;
        int st = upload(v, &dd);
        if (dd) owned.push_back(dd);
        *d = dd;
        return st;
    }
    template <typename U>
    int upb(const std::vector<U> &v, const U **d)  // a P^T band table (replaced by plan_bands)
    {
        U *dd;
        int st = upload(v, &dd);
        if (dd) band_owned.push_back(dd);
        *d = dd;
        return st;
    }
    template <typename U>
    int alloc(size_t count, U **d)
    {
        if (cudaMalloc(d, count * sizeof(U)) != cudaSuccess) return FEWHA_ERR_NOMEM;
        owned.push_back(*d);
        CK(cudaMemset(*d, 0, count * sizeof(U)));
        return FEWHA_OK;
    }

    // P^T work items and their tables: bands of rows_large layer rows on the
    // largest layers and rows_small on the smaller ones (at most kBandOutputs
    // outputs each); with the staging groups, tap lists and the shared memory
    // they need.  Replaces the tables of an earlier call.
    int plan_bands(int rows_large, int rows_small)
    {
        if (rows_large < 1 || rows_small < 1) return FEWHA_ERR_ARG;
        Geo<T> &G = base.geo;
        int st;
        int nmax = 0;
        for (int l = 0; l < P.L; l++) nmax = std::max(nmax, P.geom.layers[l].n);
        for (void *q : band_owned) cudaFree(q);
        band_owned.clear();
        // bands of BR rows with BR * n_l <= kBandOutputs outputs; by default 8
        // rows on the largest layers and 4 on the smaller ones (their coarser
        // grid touches about twice as many pupil rows per layer row, so a
        // half-height band balances the staged work)
        std::vector<int> bl, br0, brs;
        int n_largest = 0;
        for (int l = 0; l < P.L; l++) n_largest = std::max(n_largest, P.geom.layers[l].n);
        for (int l = 0; l < P.L; l++) {
            const int n = P.geom.layers[l].n;
            int BR = std::max(1, std::min(n, std::min(kBandOutputs / n, n < n_largest ? rows_small : rows_large)));
            for (int a0 = 0; a0 < n; a0 += BR) {
                bl.push_back(l);
                br0.push_back(a0);
                brs.push_back(std::min(BR, n - a0));
            }
        }
        G.nbands = (int)bl.size();
        band_cost.assign(G.nbands, 0);
        std::vector<int> bilo((size_t)P.G * G.nbands), bihi((size_t)P.G * G.nbands);
        int max_rows = 1, max_rows_sum = 1;
        std::vector<int> rows_sum(G.nbands, 0);
        for (int g = 0; g < P.G; g++)
            for (int w = 0; w < G.nbands; w++) {
                int lo = P.gm[g], hi = 0;
                size_t by = ((size_t)g * P.L + bl[w]) * 2 + 1;
                for (int a = br0[w]; a < br0[w] + brs[w]; a++) {
                    int alo = P.alo[by * FEWHA_MAX_GRID + a], ahi = P.ahi[by * FEWHA_MAX_GRID + a];
                    if (alo < ahi) {
                        lo = std::min(lo, alo);
                        hi = std::max(hi, ahi);
                    }
                }
                if (lo >= hi) lo = hi = 0;
                bilo[(size_t)g * G.nbands + w] = lo;
                bihi[(size_t)g * G.nbands + w] = hi;
                max_rows = std::max(max_rows, hi - lo);
                band_cost[w] += (long)(hi - lo) * P.gm[g];
                rows_sum[w] += hi - lo;
                max_rows_sum = std::max(max_rows_sum, rows_sum[w]);
            }
        if ((st = upb(bl, &G.band_layer)) || (st = upb(br0, &G.band_row0)) || (st = upb(brs, &G.band_rows)) ||
            (st = upb(bilo, &G.band_ilo)) || (st = upb(bihi, &G.band_ihi)))
            return st;
        // band_gather stages rows_chunk psi rows and their x-contraction
        // (all guide stars of a band at once when they fit, else in groups)
        const size_t row_bytes = (size_t)(P.m_max + nmax) * sizeof(T);
        const size_t smem_cap = 200 * 1024;  // 227 KB per CTA minus the static shared memory
        size_t smem = sm_base;
        size_t want = (size_t)max_rows_sum * row_bytes;
        if (want > smem) smem = std::min(want, smem_cap);
        G.rows_chunk = (int)std::min<size_t>(max_rows_sum, smem / row_bytes);
        if (smem > smem_cap || G.rows_chunk < max_rows) return FEWHA_ERR_GEOMETRY;
        {
            // guide stars of each band in groups of consecutive guide stars whose
            // pupil rows fit rows_chunk staged rows
            std::vector<int> gend((size_t)P.G * G.nbands), gc((size_t)P.G * G.nbands), gr((size_t)P.G * G.nbands);
            for (int w = 0; w < G.nbands; w++)
                for (int g0 = 0, g1; g0 < P.G; g0 = g1) {
                    int rows_tot = 0;
                    for (g1 = g0; g1 < P.G; g1++) {
                        const size_t i = (size_t)g1 * G.nbands + w;
                        if (rows_tot + bihi[i] - bilo[i] > G.rows_chunk) break;
                        rows_tot += bihi[i] - bilo[i];
                    }
                    if (g1 == g0) return FEWHA_ERR_GEOMETRY;  // rows_chunk >= max_rows
                    band_cost[w] += kPassValues;
                    for (int g = g0, c = 0, r = 0; g < g1; g++) {
                        const size_t i = (size_t)g * G.nbands + w;
                        gend[i] = g1;
                        gc[i] = c;
                        gr[i] = r;
                        c += (bihi[i] - bilo[i]) * P.gm[g];
                        r += bihi[i] - bilo[i];
                    }
                }
            if ((st = upb(gend, &G.band_gend)) || (st = upb(gc, &G.band_gc)) || (st = upb(gr, &G.band_gr))) return st;
            // y-contraction lists: for band row r of band w and the group that
            // starts at g0, the staged row (gr + pupil row - ilo) and weight of
            // each tap, guide star after guide star
            int ybr = 1, ymax = 1;
            for (int w = 0; w < G.nbands; w++) ybr = std::max(ybr, brs[w]);
            auto ytaps = [&](int w, int g, int r, std::vector<std::pair<int, double>> *out) {
                const size_t t = ((size_t)g * P.L + bl[w]) * 2 + 1;
                const int a = br0[w] + r, lo = P.alo[t * FEWHA_MAX_GRID + a], hi = P.ahi[t * FEWHA_MAX_GRID + a];
                const size_t i = (size_t)g * G.nbands + w;
                int cnt = 0;
                const size_t tb = P.tab(g, bl[w], 1);
                for (int j = lo; j < hi; j++, cnt++) {
                    if (!out) continue;
                    const double w0 = P.fw[tb + j];
                    out->push_back({gr[i] + (j - bilo[i]), P.fk[tb + j] == a ? 1.0 - w0 : w0});
                }
                return cnt;
            };
            for (int w = 0; w < G.nbands; w++)
                for (int g0 = 0; g0 < P.G; g0 = gend[(size_t)g0 * G.nbands + w])
                    for (int r = 0; r < brs[w]; r++) {
                        int c = 0;
                        for (int g = g0; g < gend[(size_t)g0 * G.nbands + w]; g++) c += ytaps(w, g, r, nullptr);
                        ymax = std::max(ymax, c);
                    }
            std::vector<int> ycnt((size_t)G.nbands * P.G * ybr, 0), yrow(ycnt.size() * ymax, 0);
            std::vector<T> yw(ycnt.size() * ymax, T(0));
            for (int w = 0; w < G.nbands; w++)
                for (int g0 = 0; g0 < P.G; g0 = gend[(size_t)g0 * G.nbands + w])
                    for (int r = 0; r < brs[w]; r++) {
                        std::vector<std::pair<int, double>> taps;
                        for (int g = g0; g < gend[(size_t)g0 * G.nbands + w]; g++) ytaps(w, g, r, &taps);
                        const size_t e = ((size_t)w * P.G + g0) * ybr + r;
                        ycnt[e] = (int)taps.size();
                        for (size_t t = 0; t < taps.size(); t++) {
                            yrow[e * ymax + t] = taps[t].first;
                            yw[e * ymax + t] = (T)taps[t].second;
                        }
                    }
            G.ybr = ybr;
            G.ymax = ymax;
            if ((st = upb(ycnt, &G.band_ycnt)) || (st = upb(yrow, &G.band_yrow)) || (st = upb(yw, &G.band_yw)))
                return st;
        }
        size_t sm_fixed = std::max(sm_layer_, std::min(want, smem_cap));
        // P^T x weight tables of one band (all guide stars) staged beside the
        // psi rows when kTabPT entries per thread and the shared memory suffice
        const size_t tab_entries = (size_t)P.G * nmax;
        const size_t tab_bytes = tab_entries * (kAdjW * sizeof(T) + 2 * sizeof(int));
        const size_t gather_bytes = (size_t)G.rows_chunk * row_bytes + tab_bytes;
        G.stage_tab = 0;
        if (tab_entries <= (size_t)kTabPT * kThreads && gather_bytes <= smem_cap) {
            G.stage_tab = 1;
            smem = std::max(smem, gather_bytes);
            sm_fixed = std::max(sm_fixed, gather_bytes);
        }
        this->smem = smem;
        this->sm_fixed = sm_fixed;
        base.smem_bytes = smem;
        band_rows_large = rows_large;
        band_rows_small = rows_small;
        return FEWHA_OK;
    }

    int init(int grid) override
    {
        Geo<T> &G = base.geo;
        G.G = P.G;
        G.L = P.L;
        G.ns = P.ns;
        G.m = P.m;
        G.n = P.n;
        for (int g = 0; g < P.G; g++) {
            G.gs_ns[g] = P.gns[g];
            G.gs_m[g] = P.gm[g];
            G.gs_tab[g] = P.tab_off[g];
            G.gs_psi[g] = P.psi_off[g];
            G.gs_sl[g] = P.slope_off[g];
            G.gs_mask[g] = P.mask_off[g];
        }
        G.m_max = P.m_max;
        for (int l = 0; l < P.L; l++) {
            G.lay_n[l] = P.geom.layers[l].n;
            G.lay_J[l] = P.geom.layers[l].J;
            G.lay_off[l] = P.lay_off[l];
            G.inv_delta[l] = (T)(1.0 / P.geom.layers[l].delta);
        }
        G.lay_off[P.L] = P.lay_off[P.L];
        G.ll_off[0] = 0;
        for (int l = 0; l < P.L; l++) {
            const long h = P.geom.layers[l].n / 2;
            G.ll_off[l + 1] = G.ll_off[l] + h * h;
        }
        // The split form costs an iteration two phases and two barriers (on 152 CTAs
        // 4.4 us in FP32, 7 to 10 us in FP64) and takes the finest level and three
        // quarters of the update off the layer CTAs.  By the largest layer, us a
        // step of six iterations whole / split, recycling the last direction and
        // all eight:
        //   FP32   32^2  194 / 235, 268 / 313     64^2  237 / 269, 326 / 343
        //         128^2  395 / 341, 559 / 432
        //   FP64   32^2  321 / 344, 557 / 570     64^2  620 / 445, 930 / 681
        //         128^2 1816 / 639, 2446 / 908
        // With all of 16 directions the first three are 897 / 1041, 1141 / 1139 and
        // (FP64 32^2) 1829 / 1816 us for 18 iterations.
        {
            int nmax = 0;
            for (int l = 0; l < P.L; l++) nmax = std::max(nmax, P.geom.layers[l].n);
            G.split_min = nmax > (sizeof(T) == 8 ? 32 : 64) ? 2 * P.L : kMaxCtas + 1;
        }
        // two tiled levels where a layer CTA's block would be 64^2 in FP64 (split_depth)
        {
            int nmax = 0;
            bool ok = sizeof(T) == 8;
            for (int l = 0; l < P.L; l++) {
                const fewha_layer &ly = P.geom.layers[l];
                nmax = std::max(nmax, ly.n);
                ok = ok && ly.J >= 2 && ly.n >= 32;
            }
            G.depth = ok && nmax >= 128 ? 2 : 1;
        }
        G.n_taps = (int)P.taps.size();
        for (int t = 0; t < kMaxT; t++) {
            G.h[t] = t < G.n_taps ? (T)P.taps[t] : T(0);
            G.g[t] = t < G.n_taps ? (T)(((t & 1) ? -1.0 : 1.0) * P.taps[G.n_taps - 1 - t]) : T(0);
        }
        // WFS tiles for the whole grid
        {
            int dev0, nsm0;
            CK(cudaGetDevice(&dev0));
            CK(cudaDeviceGetAttribute(&nsm0, cudaDevAttrMultiProcessorCount, dev0));
            int ty, tx;
            if (tiles_for(grid > 0 ? grid : nsm0, &ty, &tx)) return FEWHA_ERR_GEOMETRY;
            set_tiles(G, ty, tx);
        }
        int st;
        if ((st = up(P.fk, &G.fk)) || (st = up(P.alo, &G.alo)) || (st = up(P.ahi, &G.ahi))) return st;
        std::vector<T> fw(P.fw.begin(), P.fw.end());
        std::vector<T> ad(P.alpha_d.begin(), P.alpha_d.end());
        std::vector<T> one(P.n, T(1));
        if ((st = up(fw, &G.fw)) || (st = up(weight_table(), &G.wmask)) || (st = up(ad, &G.alpha_d)) ||
            (st = up(one, &G.invJ)))
            return st;
        for (int l = 0; l < P.L; l++) {
            int lg = 0;
            while ((1 << lg) < P.geom.layers[l].n) lg++;
            G.lay_lg[l] = lg;
        }
        // compact P_g^T weights: per layer node, its pupil-node range and weights
        {
            size_t nt = (size_t)P.G * P.L * 2 * FEWHA_MAX_GRID;
            std::vector<int> alo(nt, 0), acnt(nt, 0);
            std::vector<T> aw(nt * kAdjW, T(0));
            for (size_t t = 0; t < (size_t)P.G * P.L * 2; t++)
                for (int k = 0; k < FEWHA_MAX_GRID; k++) {
                    int lo = P.alo[t * FEWHA_MAX_GRID + k], hi = P.ahi[t * FEWHA_MAX_GRID + k];
                    if (hi - lo > kAdjW) return FEWHA_ERR_GEOMETRY;
                    alo[t * FEWHA_MAX_GRID + k] = lo;
                    acnt[t * FEWHA_MAX_GRID + k] = hi - lo;
                    const size_t tb = P.tab((int)(t / (2 * P.L)), (int)((t / 2) % P.L), (int)(t % 2));
                    for (int j = lo; j < hi; j++) {
                        double w0 = P.fw[tb + j];
                        aw[(t * FEWHA_MAX_GRID + k) * kAdjW + (j - lo)] = (T)(P.fk[tb + j] == k ? 1.0 - w0 : w0);
                    }
                }
            if ((st = up(alo, &G.adj_lo)) || (st = up(acnt, &G.adj_cnt)) || (st = up(aw, &G.adj_w))) return st;
            {
                std::vector<T> fw2(P.fit_w.begin(), P.fit_w.end());
                if ((st = up(P.fit_k, &fit_k)) || (st = up(fw2, &fit_w))) return st;
            }
        }
        if ((st = alloc((size_t)P.n, &base.nodal)) || (st = alloc((size_t)P.n, &base.u)) ||
            (st = alloc((size_t)P.n, &base.wq)) ||
            (st = alloc((size_t)P.psi_off[P.G], &base.psi)) || (st = alloc(ll_elems(), &base.ll)) ||
            (st = alloc((size_t)kSlots * kMaxCtas, &base.part)) || (st = alloc((size_t)1, &base.rec)))
            return st;
        if constexpr (std::is_same<T, S>::value) {
            base.nodal_t = base.nodal;
            base.psi_t = base.psi;
        } else {  // BF16 storage: the residual replacement stores its intermediates in T
            if ((st = alloc((size_t)P.n, &base.nodal_t)) || (st = alloc((size_t)P.psi_off[P.G], &base.psi_t)))
                return st;
        }
        // launch geometry: dynamic shared memory = max over phases
        int nmax = 0;
        for (int l = 0; l < P.L; l++) nmax = std::max(nmax, P.geom.layers[l].n);
        size_t sm_layer = (size_t)nmax * (nmax + 1) * sizeof(T);  // pitch n + 1
        G.pingpong = sizeof(T) == 4 ? 1 : 0;  // FP32: second buffer for out-of-place DWT passes
        if (G.pingpong) sm_layer *= 2;
        const size_t sm_wfs = wfs_bytes(G.tile_y, G.tile_x);
        // tiles of the finest wavelet level (analysis: input window and row-pass
        // output; synthesis: four subband windows and the column-pass output)
        size_t sm_fine = 0;
        {
            const int Lt = (int)P.taps.size();
            for (int l = 0; l < P.L; l++) {
                const size_t t = std::min(kFineTile, P.geom.layers[l].n / 2);
                const size_t ia = (2 * t + Lt - 2), wa = t + Lt / 2 - 1;
                sm_fine = std::max(sm_fine, std::max(ia * ia + ia * 2 * t, 4 * wa * wa + 2 * t * 2 * wa) * sizeof(T));
            }
        }
        sm_layer = std::max(sm_layer, sm_fine);
        sm_fine_ = sm_fine;
        smem = std::max(sm_layer, sm_wfs);
        sm_base = smem;
        sm_layer_ = sm_layer;
        std::vector<long> few_cost;
        if ((st = plan_bands(FEWHA_MAX_GRID, FEWHA_MAX_GRID)) == FEWHA_OK) {
            few = G;
            few_owned.swap(band_owned);
            few_fixed = sm_fixed;
            few_cost = band_cost;
        } else if (st != FEWHA_ERR_GEOMETRY) {
            return st;  // (too many rows for the shared memory: no second plan)
        }
        if ((st = plan_bands(kBandLarge, kBandSmall))) return st;
        if (few_fixed > 0) choose_plans(few_cost);
        if ((st = alloc(ll_elems(), &ll_nodal))) return st;
        int dev, nsm;
        CK(cudaGetDevice(&dev));
        CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        // the attribute allows the cap, so that plan_bands may change smem later
        auto setattr = [&](const void *f) {
            return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        };
        CK((op_attributes<Args<T, S>>()));
        CK((op_attributes<MultiArgs<T, S>>()));
        CK(setattr((const void *)k_op_wfs<T, S, Args<T, S>, true>));
        CK(setattr((const void *)k_op_update<T, S, Args<T, S>, true, false>));
        CK(setattr((const void *)k_op_update<T, S, Args<T, S>, true, true>));
        CK(setattr((const void *)k_rhs_wfs<T, S>));
        CK(setattr((const void *)k_rhs_D1<T, S, 0>));
        CK(setattr((const void *)k_rhs_D1<T, S, 1>));
        CK(setattr((const void *)k_rhs_update<T, S>));
        CK(setattr((const void *)k_rhs_gather<T, S>));
        CK(setattr((const void *)k_init<T, S>));
        CK(setattr((const void *)k_UA1<T, S>));
        CK(setattr((const void *)k_A2<T, S, 0>));
        CK(setattr((const void *)k_A2<T, S, 1>));
        CK(setattr((const void *)k_B<T, S>));
        CK(setattr((const void *)k_C<T, S>));
        CK(setattr((const void *)k_D1<T, S, 0>));
        CK(setattr((const void *)k_D1<T, S, 1>));
        CK(setattr((const void *)k_D2E<T, S>));
        CK(setattr((const void *)k_finish<T, S>));
        CK(setattr((const void *)k_TU<T, S>));
        CK(setattr((const void *)k_TA2<T, S, 0>));
        CK(setattr((const void *)k_TA2<T, S, 1>));
        CK(setattr((const void *)k_TB<T, S>));
        CK(setattr((const void *)k_TC<T, S>));
        CK(setattr((const void *)k_TD1<T, S, 0>));
        CK(setattr((const void *)k_TD1<T, S, 1>));
        CK(setattr((const void *)k_TE<T, S>));
        CK(setattr((const void *)k_solve_persistent<T, S, false>));
        CK(setattr((const void *)k_solve_persistent<T, S, true>));
        CK(setattr((const void *)k_solve_persistent<T, S, false, true>));
        CK(setattr((const void *)k_solve_persistent<T, S, true, true>));
        CK(cudaFuncSetAttribute((const void *)k_solve_batched<T, S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                200 * 1024));
        CK(cudaFuncSetAttribute((const void *)k_solve_batched<T, S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                200 * 1024));
        int per_sm = 0;
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve_persistent<T, S, false>, kThreads, smem));
        if (per_sm < 1) return FEWHA_ERR_CUDA;
        {
            int per_sm_tr = 0;
            CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_tr, k_solve_persistent<T, S, true>, kThreads,
                                                             smem));
            per_sm = std::min(per_sm, per_sm_tr);
            if (per_sm < 1) return FEWHA_ERR_CUDA;
        }
        ncta = grid > 0 ? grid : nsm;
        if (ncta > nsm * per_sm) ncta = nsm * per_sm;
        if (ncta > kMaxCtas) ncta = kMaxCtas;
        base.timeout_ns = 1000000000ull;
        base.ncta = ncta;
        base.cta0 = 0;
        base.smem_bytes = smem;
        return FEWHA_OK;
    }

    int set_bands(int rows_large, int rows_small) override
    {
        if (rows_large < 1 || rows_small < 1) return FEWHA_ERR_ARG;
        CK(cudaDeviceSynchronize());  // the tables may be in use
        const int ol = band_rows_large, os = band_rows_small;
        int st = plan_bands(rows_large, rows_small);
        if (st != FEWHA_OK) {
            plan_bands(ol, os);  // keep the earlier plan
            return st;
        }
        bands_set = true;
        return FEWHA_OK;
    }

    int auto_bands() override
    {
        CK(cudaDeviceSynchronize());  // the tables may be in use
        const int st = plan_bands(kBandLarge, kBandSmall);
        if (st == FEWHA_OK) bands_set = false;
        return st;
    }

    int group_bands(int nct, size_t sm) const override
    {
        Geo<T> G = base.geo;
        choose_bands(G, nct, sm, false);
        return G.nbands;
    }

    void launch_info(fewha_launch_info *out) const override
    {
        out->ctas = ncta;
        out->threads = kThreads;
        out->smem_bytes = (long)smem;
        out->split_levels = ncta >= base.geo.split_min ? 1 : 0;
        out->staged_tables = base.geo.stage_tab;
        out->wfs_tile_y = base.geo.tile_y;
        out->wfs_tile_x = base.geo.tile_x;
        out->pt_bands = base.geo.nbands;
        out->pt_rows_chunk = base.geo.rows_chunk;
        out->pt_rows_large = band_rows_large;
        out->pt_rows_small = band_rows_small;
    }

    int get_invJ(double *host) const override
    {
        std::vector<T> v(P.n);
        CK(cudaMemcpy(v.data(), base.geo.invJ, P.n * sizeof(T), cudaMemcpyDeviceToHost));
        for (long i = 0; i < P.n; i++) host[i] = (double)v[i];
        return FEWHA_OK;
    }

    // C_eta^{-1} per slope: 1/sigma_g^2 on lit subapertures, 0 elsewhere
    std::vector<T> weight_table() const
    {
        std::vector<T> wm((size_t)P.mask_off[P.G]);
        for (int g = 0; g < P.G; g++)
            for (long i = P.mask_off[g]; i < P.mask_off[g + 1]; i++)
                wm[i] = P.mask[i] ? (T)P.geom.gs[g].weight : T(0);
        return wm;
    }

    int set_weights() override
    {
        const std::vector<T> wm = weight_table();
        CK(cudaMemcpy(const_cast<T *>(base.geo.wmask), wm.data(), wm.size() * sizeof(T), cudaMemcpyHostToDevice));
        return FEWHA_OK;
    }

    int set_invJ(const std::vector<double> &invJ) override
    {
        std::vector<T> v(invJ.begin(), invJ.end());
        CK(cudaMemcpy(const_cast<T *>(base.geo.invJ), v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
        return FEWHA_OK;
    }

    void set_timeout(unsigned long long ns) override { base.timeout_ns = ns; }

    void set_trace(unsigned long long *buf, int cap) override
    {
        base.trace = buf;
        base.trace_cap = buf ? cap : 0;
    }

    int launch_check() { return cudaGetLastError() == cudaSuccess ? FEWHA_OK : FEWHA_ERR_CUDA; }

    template <class A>
    static cudaError_t op_attributes()
    {
        for (const void *f : {(const void *)k_op_coarse<T, S, A, false>, (const void *)k_op_coarse<T, S, A, true>,
                              (const void *)k_op_synth<T, S, A, 0>, (const void *)k_op_synth<T, S, A, 1>,
                              (const void *)k_op_wfs<T, S, A, false>, (const void *)k_op_gather<T, S, A>,
                              (const void *)k_op_analysis<T, S, A, 0>, (const void *)k_op_analysis<T, S, A, 1>,
                              (const void *)k_op_update<T, S, A, false, false>,
                              (const void *)k_op_update<T, S, A, false, true>}) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }

    // One kernel of an operator chain; after the first, with programmatic
    // stream serialisation (see pdl_begin).
    struct OpChain {
        int grid;
        cudaStream_t s;
        bool first;
        cudaError_t err;
        template <class K, class A>
        void operator()(K kern, size_t sm, const A &args)
        {
            if (err != cudaSuccess) return;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(grid);
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = sm;
            cfg.stream = s;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = first ? 0 : 1;
            err = cudaLaunchKernelEx(&cfg, kern, args);
            first = false;
        }
    };

    // Form of the chain for `group` CTAs per vector.  Split costs two more
    // kernels (four with two tiled levels) and pays where the solver's split form
    // does (Geo::split_min); in FP32 from four CTAs per layer: with fewer, the
    // tiled kernels take several rounds (9 ELT layers, 5 vectors of 30 CTAs:
    // 94.7 us split, 79.9 us whole).
    bool op_split(int group) const
    {
        return group >= base.geo.split_min && (sizeof(T) == 8 || group >= 4 * P.L);
    }

    // nodal = W^{-1} x; group: CTAs per vector
    template <class A>
    void op_idwt(OpChain &run, const A &args, int group, size_t sm) const
    {
        if (!op_split(group)) {
            run(k_op_coarse<T, S, A, true>, sm, args);
            return;
        }
        run(k_op_coarse<T, S, A, false>, sm, args);
        if (base.geo.depth > 1) run(k_op_synth<T, S, A, 1>, sm_fine_, args);
        run(k_op_synth<T, S, A, 0>, sm_fine_, args);
    }

    // u = P^T psi and W^{-T} u up to its last part
    template <class A>
    void op_adjoint(OpChain &run, const A &args, int group, size_t sm) const
    {
        run(k_op_gather<T, S, A>, sm, args);
        if (!op_split(group)) return;
        run(k_op_analysis<T, S, A, 0>, sm_fine_, args);
        if (base.geo.depth > 1) run(k_op_analysis<T, S, A, 1>, sm_fine_, args);
    }

    template <class A>
    int op_apply(const A &args, int grid, int group, size_t sm, cudaStream_t s) const
    {
        OpChain run{grid, s, true, cudaSuccess};
        op_idwt(run, args, group, sm);
        run(k_op_wfs<T, S, A, false>, sm, args);
        op_adjoint(run, args, group, sm);
        if (op_split(group))
            run(k_op_update<T, S, A, false, false>, sm, args);
        else
            run(k_op_update<T, S, A, false, true>, sm, args);
        return run.err == cudaSuccess ? FEWHA_OK : FEWHA_ERR_CUDA;
    }

    int op_nodal(const void *c, cudaStream_t s) const
    {
        Args<T, S> A = base;
        A.x = static_cast<const T *>(c);
        A.ll = ll_nodal;
        OpChain run{ncta, s, true, cudaSuccess};
        op_idwt(run, A, ncta, smem);
        return run.err == cudaSuccess ? FEWHA_OK : FEWHA_ERR_CUDA;
    }

    int apply(const void *x, void *y, cudaStream_t s) override
    {
        Args<T, S> A = base;
        A.x = static_cast<const T *>(x);
        A.y = static_cast<T *>(y);
        return op_apply(A, ncta, ncta, smem, s);
    }

    int fit(const void *c, void *a, cudaStream_t s) override
    {
        if (!P.fit_ok) return FEWHA_ERR_GEOMETRY;
        const int st = op_nodal(c, s);  // nodal = W^{-1} c
        if (st != FEWHA_OK) return st;
        FitTab<T> F{};
        for (int l = 0; l < P.L; l++) {
            F.off[l] = P.lay_off[l];
            F.n[l] = P.geom.layers[l].n;
        }
        F.L = P.L;
        F.m = P.m;
        F.fk = fit_k;
        F.fw = fit_w;
        k_fit<T, S><<<(P.m * P.m + 255) / 256, 256, 0, s>>>(F, base.nodal, static_cast<T *>(a));
        return launch_check();
    }

    // MCAO fitting plan: device tables and work vectors of one mirror system
    struct McaoPlan {
        McaoArgs<T, S> M{};
        std::vector<void *> owned;
        ~McaoPlan()
        {
            for (void *q : owned) cudaFree(q);
        }
    };

    int mcao_create(const fewha_mcao_desc *d, void **out, long *n_act) override
    {
        if (d->n_dm < 1 || d->n_dm > FEWHA_MAX_DM || d->n_dir < 1 || d->n_dir > FEWHA_MAX_DIR)
            return FEWHA_ERR_ARG;
        const int m = P.m, L = P.L, D = d->n_dm, T_ = d->n_dir;
        int nmax = 0;
        for (int k = 0; k < D; k++) {
            if (d->dm_n[k] < 2 || !(d->dm_pitch[k] > 0) || !std::isfinite(d->dm_pitch[k]) ||
                !std::isfinite(d->dm_h[k]) || d->dm_h[k] < 0)
                return FEWHA_ERR_ARG;
            nmax = std::max(nmax, d->dm_n[k]);
        }
        for (int t = 0; t < T_; t++)
            if (!std::isfinite(d->dir_x[t]) || !std::isfinite(d->dir_y[t])) return FEWHA_ERR_ARG;
        // bilinear tables: pupil node j at x = -D/2 + j ds; layer node k at
        // (k - n/2) d_l; actuator i at (i - (n-1)/2) pitch
        std::vector<int> lk((size_t)T_ * L * 2 * m), dk((size_t)T_ * D * 2 * m);
        std::vector<T> lw(lk.size()), dw(dk.size());
        std::vector<int> alo((size_t)T_ * D * 2 * nmax, 0), ahi(alo.size(), 0);
        auto table = [&](double shift, double spacing, double centre, int n, int *k_out, T *w_out) {
            for (int j = 0; j < m; j++) {
                const double f = (-0.5 * P.geom.D + j * P.ds + shift) / spacing + centre;
                const int k = (int)std::floor(f);
                if (k < 0 || k + 1 > n - 1) return false;
                k_out[j] = k;
                w_out[j] = (T)(f - k);
            }
            return true;
        };
        for (int t = 0; t < T_; t++) {
            for (int l = 0; l < L; l++) {
                const fewha_layer &ly = P.geom.layers[l];
                for (int ax = 0; ax < 2; ax++) {
                    const size_t b = (((size_t)t * L + l) * 2 + ax) * m;
                    const double th = ax == 0 ? d->dir_x[t] : d->dir_y[t];
                    if (!table(th * ly.h, P.lay_d[l], 0.5 * ly.n, ly.n, &lk[b], &lw[b])) return FEWHA_ERR_GEOMETRY;
                }
            }
            for (int k = 0; k < D; k++)
                for (int ax = 0; ax < 2; ax++) {
                    const size_t b = (((size_t)t * D + k) * 2 + ax) * m;
                    const double th = ax == 0 ? d->dir_x[t] : d->dir_y[t];
                    if (!table(th * d->dm_h[k], d->dm_pitch[k], 0.5 * (d->dm_n[k] - 1), d->dm_n[k], &dk[b], &dw[b]))
                        return FEWHA_ERR_GEOMETRY;
                    const size_t rb = (((size_t)t * D + k) * 2 + ax) * nmax;
                    for (int i = 0; i < d->dm_n[k]; i++) {
                        int lo = m, hi = 0;
                        for (int j = 0; j < m; j++)
                            if (dk[b + j] == i || dk[b + j] + 1 == i) {
                                lo = std::min(lo, j);
                                hi = std::max(hi, j + 1);
                            }
                        if (lo >= hi) lo = hi = 0;
                        alo[rb + i] = lo;
                        ahi[rb + i] = hi;
                    }
                }
        }
        auto *pl = new McaoPlan();
        McaoArgs<T, S> &M = pl->M;
        M.L = L;
        M.D = D;
        M.ndir = T_;
        M.m = m;
        M.nmax = nmax;
        for (int l = 0; l < L; l++) {
            M.lay_off[l] = P.lay_off[l];
            M.lay_n[l] = P.geom.layers[l].n;
        }
        M.dm_off[0] = 0;
        for (int k = 0; k < D; k++) {
            M.dm_n[k] = d->dm_n[k];
            M.dm_off[k + 1] = M.dm_off[k] + (long)d->dm_n[k] * d->dm_n[k];
        }
        const long na = M.dm_off[D];
        int st = FEWHA_OK;
        auto put_i = [&](const std::vector<int> &v, const int **dst) {
            int *dd = nullptr;
            if (upload(v, &dd)) return false;
            pl->owned.push_back(dd);
            *dst = dd;
            return true;
        };
        auto put_t = [&](const std::vector<T> &v, const T **dst) {
            T *dd = nullptr;
            if (upload(v, &dd)) return false;
            pl->owned.push_back(dd);
            *dst = dd;
            return true;
        };
        auto make = [&](size_t bytes, void **dst) {
            if (cudaMalloc(dst, bytes) != cudaSuccess) return false;
            pl->owned.push_back(*dst);
            return true;
        };
        const int *c_lk, *c_dk, *c_alo, *c_ahi;
        const T *c_lw, *c_dw;
        void *r, *p, *p2, *q, *y, *part, *rec;
        if (!put_i(lk, &c_lk) || !put_t(lw, &c_lw) || !put_i(dk, &c_dk) || !put_t(dw, &c_dw) ||
            !put_i(alo, &c_alo) || !put_i(ahi, &c_ahi) || !make(na * sizeof(T), &r) || !make(na * sizeof(T), &p) ||
            !make(na * sizeof(T), &p2) ||
            !make(na * sizeof(T), &q) || !make((size_t)T_ * m * m * sizeof(T), &y) ||
            !make(2 * kMaxCtas * sizeof(double), &part) || !make(sizeof(Record), &rec))
            st = FEWHA_ERR_CUDA;
        if (st) {
            delete pl;
            return st;
        }
        M.lk = c_lk;
        M.lw = c_lw;
        M.dk = c_dk;
        M.dw = c_dw;
        M.alo = c_alo;
        M.ahi = c_ahi;
        M.r = static_cast<T *>(r);
        M.p = static_cast<T *>(p);
        M.p2 = static_cast<T *>(p2);
        M.q = static_cast<T *>(q);
        M.y = static_cast<T *>(y);
        M.part = static_cast<double *>(part);
        M.rec = static_cast<Record *>(rec);
        *out = pl;
        *n_act = na;
        return FEWHA_OK;
    }

    int mcao_fit(void *plan, const void *c, void *a, int iters, cudaStream_t s) override
    {
        if (iters < 0 || iters > FEWHA_MAX_ITER) return FEWHA_ERR_ARG;
        auto *pl = static_cast<McaoPlan *>(plan);
        const int st = op_nodal(c, s);  // nodal = W^{-1} c
        if (st != FEWHA_OK) return st;
        McaoArgs<T, S> M = pl->M;
        M.nodal = base.nodal;
        M.a = static_cast<T *>(a);
        M.iters = iters;
        M.timeout_ns = base.timeout_ns;
        CK(cudaMemsetAsync(M.rec, 0, sizeof(Record), s));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ncta);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        CK(cudaLaunchKernelEx(&cfg, k_mcao_fit<T, S>, M));
        return launch_check();
    }

    void mcao_destroy(void *plan) override { delete static_cast<McaoPlan *>(plan); }

    int pol_slopes(const void *s_in, const void *a, void *s_out, cudaStream_t s) override
    {
        for (int g = 0; g < P.G; g++)  // the mirror's actuators sit on the geometry's pupil grid
            if (P.gns[g] != P.ns) return FEWHA_ERR_GEOMETRY;
        k_pol<T, S><<<256, 256, 0, s>>>(static_cast<const S *>(s_in), static_cast<const T *>(a),
                                        static_cast<S *>(s_out), P.G, P.ns);
        return launch_check();
    }

    int control(int closed, double gain, const void *am1, const void *ai, const void *af, void *an,
                cudaStream_t s) override
    {
        const int na = P.m * P.m;
        k_control<T><<<(na + 255) / 256, 256, 0, s>>>(closed, (T)gain, static_cast<const T *>(am1),
                                                      static_cast<const T *>(ai), static_cast<const T *>(af),
                                                      static_cast<T *>(an), na);
        return launch_check();
    }

    int apply_multi(const void *x, long ldx, void *y, long ldy, int nvec, cudaStream_t s) override
    {
        static_assert(sizeof(MultiArgs<T, S>) <= 32000, "kernel parameter size");
        if (nvec < 1 || nvec > kMaxVec || ldx < P.n || ldy < P.n) return FEWHA_ERR_ARG;
        auto up256 = [](size_t v) { return (v + 255) & ~(size_t)255; };
        if (!multi_buf) {
            multi_stride = up256((size_t)P.n * sizeof(S)) + up256((size_t)P.psi_off[P.G] * sizeof(S)) +
                           2 * up256((size_t)P.n * sizeof(T)) + up256(ll_elems() * sizeof(T));
            if (alloc(multi_stride * kMaxVec, &multi_buf)) return FEWHA_ERR_NOMEM;
        }
        const int per = std::max(1, ncta / nvec);
        int ty, tx;
        if (tiles_for(per, &ty, &tx)) return FEWHA_ERR_GEOMETRY;
        const size_t sm = smem_want(ty, tx, per, true);
        MultiArgs<T, S> M{};
        M.per = per;
        for (int v = 0; v < nvec; v++) {
            Args<T, S> A = base;
            unsigned char *b = multi_buf + (size_t)v * multi_stride;
            A.nodal = reinterpret_cast<S *>(b);
            A.psi = reinterpret_cast<S *>(b + up256((size_t)P.n * sizeof(S)));
            A.u = reinterpret_cast<T *>(b + up256((size_t)P.n * sizeof(S)) + up256((size_t)P.psi_off[P.G] * sizeof(S)));
            A.wq = A.u + up256((size_t)P.n * sizeof(T)) / sizeof(T);
            A.ll = A.wq + up256((size_t)P.n * sizeof(T)) / sizeof(T);
            A.x = static_cast<const T *>(x) + (size_t)v * ldx;
            A.y = static_cast<T *>(y) + (size_t)v * ldy;
            A.cta0 = v * per;
            A.ncta = per;
            set_tiles(A.geo, ty, tx);
            choose_bands(A.geo, per, sm, true);
            A.smem_bytes = sm;
            A.trace = nullptr;
            A.trace_cap = 0;
            M.a[v] = A;
        }
        return op_apply(M, per * nvec, per, sm, s);
    }

    int apply_in_scratch(const void *x, void *y, void *scratch, size_t bytes, cudaStream_t s) override
    {
        // layout: nodal layers | adjoint wavefronts | P^T output | level-1 and -2
        // approximations | operator output before + alpha D x (in the nodal
        // layers' place when they have the same type: it is written after they
        // were last read).  Every buffer is written before it is read.
        auto up256 = [](size_t v) { return (v + 255) & ~(size_t)255; };
        const size_t o_psi = up256((size_t)P.n * sizeof(S));
        const size_t o_u = up256(o_psi + (size_t)P.psi_off[P.G] * sizeof(S));
        const size_t o_ll = up256(o_u + (size_t)P.n * sizeof(T));
        const size_t o_wq = std::is_same<T, S>::value ? 0 : up256(o_ll + ll_elems() * sizeof(T));
        const size_t need = std::max(up256(o_ll + ll_elems() * sizeof(T)), up256(o_wq + (size_t)P.n * sizeof(T)));
        // the size test of the entry point's contract (fewha.h): a record, partial
        // sums of every CTA, nodal layers, adjoint wavefronts and P^T output; the
        // first two are counted and no longer stored
        const size_t contract = up256(sizeof(Record)) + up256((size_t)kSlots * kMaxCtas * sizeof(double)) +
                                up256(o_u + (size_t)P.n * sizeof(T));
        if (contract > bytes || need > bytes) return FEWHA_ERR_SCRATCH;
        unsigned char *base_p = static_cast<unsigned char *>(scratch);
        Args<T, S> A = base;
        A.nodal = reinterpret_cast<S *>(base_p);
        A.psi = reinterpret_cast<S *>(base_p + o_psi);
        A.u = reinterpret_cast<T *>(base_p + o_u);
        A.ll = reinterpret_cast<T *>(base_p + o_ll);
        A.wq = reinterpret_cast<T *>(base_p + o_wq);
        A.trace = nullptr;
        A.trace_cap = 0;
        A.x = static_cast<const T *>(x);
        A.y = static_cast<T *>(y);
        return op_apply(A, ncta, ncta, smem, s);
    }

    int rhs(const void *sl, void *b, cudaStream_t s) override
    {
        Args<T, S> A = base;
        A.slopes = static_cast<const S *>(sl);
        A.y = static_cast<T *>(b);
        OpChain run{ncta, s, true, cudaSuccess};
        run(k_op_wfs<T, S, Args<T, S>, true>, smem, A);
        op_adjoint(run, A, ncta, smem);
        if (op_split(ncta))
            run(k_op_update<T, S, Args<T, S>, true, false>, smem, A);
        else
            run(k_op_update<T, S, Args<T, S>, true, true>, smem, A);
        return run.err == cudaSuccess ? FEWHA_OK : FEWHA_ERR_CUDA;
    }

    Args<T, S> solve_args(const void *sl, void *c, const fewha_state *st, const fewha_solve_opts *o,
                          fewha_stats *stats) const
    {
        Args<T, S> A = base;
        A.slopes = static_cast<const S *>(sl);
        A.c = static_cast<T *>(c);
        A.r = static_cast<T *>(st->r_prev);
        A.b_prev = static_cast<T *>(st->b_prev);
        A.P = static_cast<T *>(st->basis_P);
        A.Q = static_cast<T *>(st->basis_Q);
        A.pq = st->basis_pq;
        A.meta = st->meta;
        A.kcap = st->k_cap;
        A.max_iter = o->max_iter;
        A.rtol = o->rtol;
        A.augmented = o->augmented ? 1 : 0;
        A.recycle_all = o->recycle_mode == FEWHA_RECYCLE_ALL ? 1 : 0;
        A.true_res_every = o->true_res_every;
        A.rhs_in_state = o->rhs_in_state ? 1 : 0;
        A.c_out = static_cast<T *>(o->c_out);
        A.stats = stats;
        return A;
    }

    int batch_args(void *out, const void *sl, void *c, const fewha_state *st, const fewha_solve_opts *o,
                   fewha_stats *stats, int cta0, int nct, int ty, int tx, size_t sm) const override
    {
        Args<T, S> A = solve_args(sl, c, st, o, stats);
        A.c_out = nullptr;  // the batch calls have no second destination
        A.cta0 = cta0;
        A.ncta = nct;
        set_tiles(A.geo, ty, tx);
        choose_bands(A.geo, nct, sm, false);
        A.smem_bytes = sm;
        A.trace = nullptr;
        A.trace_cap = 0;
        std::memcpy(out, &A, sizeof(A));
        return FEWHA_OK;
    }

    int batch_capacity(size_t sm, int *max_ctas) const override
    {
        int dev, nsm, per_sm = 0;
        CK(cudaGetDevice(&dev));
        CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        int per_sm_tr = 0;
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve_batched<T, S, false>, kThreads, sm));
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_tr, k_solve_batched<T, S, true>, kThreads, sm));
        *max_ctas = std::min(nsm * std::min(per_sm, per_sm_tr), kMaxCtas);
        return FEWHA_OK;
    }

    int launch_batched(const void *d_args, const int *d_map, int n, int total, size_t sm, int nrounds,
                       Record *brec, int true_res, cudaStream_t s) const override
    {
        const Args<T, S> *args = static_cast<const Args<T, S> *>(d_args);
        k_batch_reset<T, S><<<(n + 255) / 256, 256, 0, s>>>(args, n, brec);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(total);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = sm;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        // a round may run as long as one time step of its slowest instance
        const unsigned long long to = base.timeout_ns * 4;
        if (true_res)
            CK(cudaLaunchKernelEx(&cfg, k_solve_batched<T, S, true>, args, d_map, nrounds, total, brec, to));
        else
            CK(cudaLaunchKernelEx(&cfg, k_solve_batched<T, S, false>, args, d_map, nrounds, total, brec, to));
        return cudaGetLastError() == cudaSuccess ? FEWHA_OK : FEWHA_ERR_CUDA;
    }

    int solve(const void *sl, void *c, const fewha_state *st, const fewha_solve_opts *o,
              fewha_stats *stats, cudaStream_t s) override
    {
        Args<T, S> A = solve_args(sl, c, st, o, stats);
        CK(cudaMemsetAsync(A.rec, 0, offsetof(Record, rz), s));
        CK(cudaMemsetAsync(&A.rec->bar, 0, sizeof(Bar), s));
        if (A.trace) CK(cudaMemsetAsync(A.trace, 0, (size_t)A.trace_cap * 4 * sizeof(unsigned long long), s));
        if (o->launch_mode == FEWHA_LAUNCH_PERSISTENT) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(ncta);
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = smem;
            cfg.stream = s;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeCooperative;
            attr[0].val.cooperative = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            const bool tr = A.true_res_every > 0, ris = A.rhs_in_state != 0;
            if (tr && ris)
                CK(cudaLaunchKernelEx(&cfg, k_solve_persistent<T, S, true, true>, A));
            else if (tr)
                CK(cudaLaunchKernelEx(&cfg, k_solve_persistent<T, S, true>, A));
            else if (ris)
                CK(cudaLaunchKernelEx(&cfg, k_solve_persistent<T, S, false, true>, A));
            else
                CK(cudaLaunchKernelEx(&cfg, k_solve_persistent<T, S, false>, A));
            return launch_check();
        }
        const bool deep = A.geo.depth > 1 && ncta >= A.geo.split_min;  // split_levels, split_depth
        k_rhs_wfs<T, S><<<ncta, kThreads, smem, s>>>(A);
        k_rhs_gather<T, S><<<ncta, kThreads, smem, s>>>(A);
        k_rhs_D1<T, S, 0><<<ncta, kThreads, smem, s>>>(A);
        if (deep) k_rhs_D1<T, S, 1><<<ncta, kThreads, smem, s>>>(A);
        k_rhs_update<T, S><<<ncta, kThreads, smem, s>>>(A);
        k_init<T, S><<<ncta, kThreads, smem, s>>>(A);
        for (int k = 0; k < A.max_iter; k++) {
            k_UA1<T, S><<<ncta, kThreads, smem, s>>>(A, k);
            if (deep) k_A2<T, S, 1><<<ncta, kThreads, smem, s>>>(A, k);
            k_A2<T, S, 0><<<ncta, kThreads, smem, s>>>(A, k);
            k_B<T, S><<<ncta, kThreads, smem, s>>>(A, k);
            k_C<T, S><<<ncta, kThreads, smem, s>>>(A, k);
            k_D1<T, S, 0><<<ncta, kThreads, smem, s>>>(A, k);
            if (deep) k_D1<T, S, 1><<<ncta, kThreads, smem, s>>>(A, k);
            k_D2E<T, S><<<ncta, kThreads, smem, s>>>(A, k);
            if (A.true_res_every > 0 && (k + 1) % A.true_res_every == 0) {
                k_TU<T, S><<<ncta, kThreads, smem, s>>>(A);
                if (deep) k_TA2<T, S, 1><<<ncta, kThreads, smem, s>>>(A);
                k_TA2<T, S, 0><<<ncta, kThreads, smem, s>>>(A);
                k_TB<T, S><<<ncta, kThreads, smem, s>>>(A);
                k_TC<T, S><<<ncta, kThreads, smem, s>>>(A);
                k_TD1<T, S, 0><<<ncta, kThreads, smem, s>>>(A);
                if (deep) k_TD1<T, S, 1><<<ncta, kThreads, smem, s>>>(A);
                k_TE<T, S><<<ncta, kThreads, smem, s>>>(A, k);
            }
        }
        k_finish<T, S><<<1, kThreads, smem, s>>>(A);
        return launch_check();
    }
};


ImplBase *make_impl_f64(const Plan &p);
// Working-precision implementation of a handle and the device it was created
// on (defined with the C ABI).
ImplBase *handle_impl(void *handle);
int handle_device(const void *handle);
// Device address of the allocation-free entry point's static scratch on the
// current device; the first call on a device loads the module that holds it.
int noalloc_prepare();
ImplBase *make_impl_f32(const Plan &p);
ImplBase *make_impl_bf16(const Plan &p);

}  // namespace fewha
