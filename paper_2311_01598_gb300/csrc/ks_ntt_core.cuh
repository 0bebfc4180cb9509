// ks_ntt_core.cuh -- limb addressing and the row/column NTT pass bodies shared
// by the stage kernels (ks_kernels.cu) and the Output-Centric fused kernels
// (ks_oc.cu).  See ks_device.cuh for the decomposition.
#pragma once
#include "ks_device.cuh"
#include "ks_launch.h"

namespace ks {

struct LimbRef {
    const u64 *src;
    u64 *dst;
    const ulonglong2 *scale;
    int t, tf, b;
    bool skip;
};

__device__ __forceinline__ LimbRef limb_ref(const LimbMaps &ms, int lg, int nq, int alpha, int logN)
{
    const int jb = find_slot(ms.pre, ms.n, lg);
    const LimbMap &m = ms.m[jb];
    const int l = lg - ms.pre[jb];
    const int a = l / m.per, b = l % m.per;
    const int t = m.toff + b;
    const size_t o = ((size_t)a * m.row_stride + m.aoff + b) << logN;
    LimbRef r;
    r.src = m.src ? m.src + o : nullptr;
    r.dst = m.dst ? m.dst + o : nullptr;
    r.scale = m.scale;
    r.t = t;
    r.b = b;
    r.tf = full_tower(t, m.nact, nq);
    r.skip = m.skip_base >= 0 && t < m.nact && (t / alpha) == a + m.skip_base;
    return r;
}

// Padded index inside a shared-memory row: one spare word after every group
// of MB words keeps the second-round reads of a row free of bank conflicts.
template <class S>
__device__ __forceinline__ int rpad(int c)
{
    return c + c / S::MB;
}

// First-round twiddles of one row (local stages s < RB, group g < 2^s),
// copied by the row's own TB threads into sh[2^s - 1 + g]: one load each,
// issued together with the row's data loads, so the first round's
// butterflies read shared memory instead of waiting on dependent L2 loads
// (the first round's twiddles are common to the whole row; the second
// round's differ per thread and stay in the table).
template <class S>
__device__ __forceinline__ void stage_row_round1(ulonglong2 *sh, const ulonglong2 *t, int G, int tau)
{
    for (int f = tau; f < S::REGB - 1; f += S::TB) {
        const int st = 31 - __clz(f + 1);
        sh[f] = __ldg(t + (G << st) + f + 1 - (1 << st));
    }
}
// Twiddle fetcher of the forward row pass: first round from the staged row
// block, second round from the tower table.
template <class S>
struct TwStaged {
    const ulonglong2 *sh;
    const ulonglong2 *t;
    int G;
    __device__ __forceinline__ ulonglong2 operator()(int s, int i) const { return sh[(1 << s) - 1 + i]; }
    template <int NG> __device__ __forceinline__ ulonglong2 r2(int s, int, int tau, int gg, int g2) const
    {
        return __ldg(t + (G << s) + (g2 * NG + gg) * S::TB + tau);
    }
    template <int NG> __device__ __forceinline__ ulonglong2 r2v(int s, int tau, int gg, int g2) const
    {
        return ldg_now(t + (G << s) + (g2 * NG + gg) * S::TB + tau);
    }
};

// Row pass of the forward NTT on one row held by TB threads: x enters and
// leaves in the first-round layout (x[k] is element k*TB + tau of the row),
// srow is the row's padded shared-memory buffer.  Contains block barriers:
// every thread of the block must call it.
// pf: the folds this set's transforms need (Tables::pm_fold, uniform).
template <class S, int AR, class TW>
__device__ __forceinline__ void row_fwd_core(u64 (&x)[S::REGB], const TW &tw, u64 *srow, int tau, const ModR<AR> &m,
                                             int pf)
{
    constexpr int M = S::MB, NG = S::REGB / S::MB;
    if (AR == AR_PM && (pf & PM_FOLD_ROW)) fold_all<S::REGB, AR>(x, m);
    fwd_round1<S::RB, AR>(x, tw, m);
#pragma unroll
    for (int k = 0; k < S::REGB; ++k) srow[rpad<S>(k * S::TB + tau)] = x[k];
    // the second round's first twiddles while the values are in shared memory:
    // their L2 latency passes behind the barrier (494 -> 478 us for 1920 limbs of
    // 2^16; seven of the fifteen spill, 494)
    constexpr int NP = S::REGB >= 16 ? 5 : 3;
    ulonglong2 pre[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
        const int q = e / NG, s2 = q == 0 ? 0 : q < 3 ? 1 : 2;
        pre[e] = tw.template r2v<NG>(S::RB + s2, tau, e % NG, q + 1 - (1 << s2));
    }
    __syncthreads();
#pragma unroll
    for (int gg = 0; gg < NG; ++gg)
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) x[gg * M + k2] = srow[rpad<S>((tau * NG + gg) * M + k2)];
    if (AR == AR_PM && (pf & PM_FOLD_MID)) fold_all<S::REGB, AR>(x, m);
    fwd_round2<S::LB, S::RB, AR, NP>(x, tau, tw, m, pre);
    __syncthreads();
#pragma unroll
    for (int gg = 0; gg < NG; ++gg)
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) srow[rpad<S>((tau * NG + gg) * M + k2)] = x[gg * M + k2];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < S::REGB; ++k) x[k] = srow[rpad<S>(k * S::TB + tau)];
    __syncthreads();
}

// Row pass of the inverse NTT (stages logN-1 .. LA), same layout contract.
template <class S, int AR, class TW>
__device__ __forceinline__ void row_inv_core(u64 (&x)[S::REGB], const TW &tw, u64 *srow, int tau, const ModR<AR> &m)
{
    constexpr int M = S::MB, NG = S::REGB / S::MB;
#pragma unroll
    for (int k = 0; k < S::REGB; ++k) srow[rpad<S>(k * S::TB + tau)] = x[k];
    // the first stage's twiddles while the values are in shared memory, as in the
    // forward pass (192 -> 180 us for 640 limbs of 2^16)
    constexpr int NP = S::REGB / 2;
    ulonglong2 pre[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) pre[e] = tw.template r2v<NG>(S::LB - 1, tau, e % NG, e / NG);
    __syncthreads();
#pragma unroll
    for (int gg = 0; gg < NG; ++gg)
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) x[gg * M + k2] = srow[rpad<S>((tau * NG + gg) * M + k2)];
    inv_round2<S::LB, S::RB, AR, NP>(x, tau, tw, m, pre);
    __syncthreads();
#pragma unroll
    for (int gg = 0; gg < NG; ++gg)
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) srow[rpad<S>((tau * NG + gg) * M + k2)] = x[gg * M + k2];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < S::REGB; ++k) x[k] = srow[rpad<S>(k * S::TB + tau)];
    __syncthreads();
    fold_all<S::REGB, AR>(x, m);
    inv_round1<S::RB, AR>(x, tw, m);
}

// A forward output as the key product takes it: canonical or lazy in the
// other forms (below kFwdLazy*q), folded below 2^(b+1) plus a little here.
template <int AR>
__device__ __forceinline__ u64 key_input(u64 x, const ModR<AR> &m)
{
    return fold<AR>(x, m);
}
// Any 64-bit value -> [0, q).
template <int AR>
__device__ __forceinline__ u64 canon_any(u64 x, const ModC &mc)
{
    if constexpr (AR == AR_PM)
        return pm_canon(x, mc.q, mc.pm_c2, mc.pm_k);
    else
        return reduce_any(x, mc.q, mc.one_sh);
}
// End of an inverse transform: the scale (W a twiddle-form pair when SC) and
// the reduction to [0, q).  x below 4q (AR_GEN, AR_SP) or any (AR_PM).
template <int AR, bool SC>
__device__ __forceinline__ u64 inv_finish(u64 x, const ulonglong2 &W, const ModC &mc)
{
    if constexpr (AR == AR_PM) {
        if (SC) x = pm_mul(x, W, mc.pm_c2, mc.pm_k);
        return pm_canon(x, mc.q, mc.pm_c2, mc.pm_k);
    } else {
        if (SC) x = shoup_lazy(x, W.x, W.y, mc.q);
        return reduce4(x, mc.q, 2 * mc.q);
    }
}

// Runs FN<AR>(...) for the parameter set's butterfly form.
#define KS_DISPATCH_AR(T, CALL)                \
    switch ((T).arith) {                       \
    case AR_PM: { constexpr int AR = AR_PM; CALL; break; } \
    case AR_SP: { constexpr int AR = AR_SP; CALL; break; } \
    default: { constexpr int AR = AR_GEN; CALL; break; }   \
    }
// The same for kernels without a special-form instance (AR_SP sets use AR_GEN).
#define KS_DISPATCH_AR2(T, CALL)               \
    switch ((T).arith) {                       \
    case AR_PM: { constexpr int AR = AR_PM; CALL; break; } \
    default: { constexpr int AR = AR_GEN; CALL; break; }   \
    }

}  // namespace ks
