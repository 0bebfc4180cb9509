// ks_ntt_cluster.cu -- one-launch NTT over thread-block clusters.
//
// The two-pass NTT (ks_kernels.cu) runs its column and row passes as two
// launches, the limb going through L2/HBM in between.  Here one cluster of C
// CTAs transforms one limb in a single launch: CTA r runs the column pass on
// columns [r*COLS, (r+1)*COLS) and keeps its block in shared memory; after a
// cluster barrier it gathers rows [r*ROWS, (r+1)*ROWS) from the blocks of all
// C CTAs through distributed shared memory and runs the row pass.  The
// inverse runs the row pass first and gathers columns.  The butterflies,
// twiddles and value ranges are those of the two-pass kernels, so the outputs
// are bit-identical to theirs.
//
// Shared memory per CTA: one buffer (the CTA's block of the limb, the column
// pass's transpose, then the row buffers), the column twiddles and the staged
// first-round row twiddles: 42 KB at N = 2^16.  A second cluster barrier
// after the gather frees the buffer for reuse and keeps every CTA alive while
// others read its block.
#include "ks_cluster.cuh"

namespace ks {

namespace {

// Forward NTT (input below 4q; output canonical with CANON, else lazy, at most flz).
// grid (C, limbs), cluster (C, 1, 1): every CTA of a cluster has the same
// limb, so the early exits below are uniform over the cluster.  early: the next
// kernel may start with this one, else as its blocks end (early_start).
template <class S, int MUL, bool CANON, int AR>
__global__ void __launch_bounds__(Cl<S, MUL>::THREADS, Cl<S, MUL>::MINB) k_fwd_cl(Tables T, LimbMaps ms, int early)
{
    if (early) pdl_start();
    typedef Cl<S, MUL> G_;
    constexpr int COLS = G_::COLS, ROWS = G_::ROWS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    u64 *buf = reinterpret_cast<u64 *>(smem_raw);
    ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(buf + G_::BUFW);
    ulonglong2 *tsh_all = tws + (1 << S::LA);
    const int lg = blockIdx.y + blockIdx.z * gridDim.y;
    if (lg >= ms.pre[ms.n]) return pdl_wait();
    const LimbRef L = limb_ref(ms, lg, T.nq, T.alpha, S::LOGN);
    if (L.skip) return;
    const ModC &mc = T.modc[L.tf];
    const ModR<AR> md = mod_fwd<AR>(mc);
    const int r = cluster_rank();
    const ulonglong2 *twt = T.tw + ((size_t)L.tf << S::LOGN);
    {
        // column pass on this CTA's columns; the block stays in buf as
        // buf[h*COLS + cc] (row h, column r*COLS + cc)
        for (int i = threadIdx.x; i < (1 << S::LA); i += G_::THREADS) tws[i] = twt[i];
        const int cc = threadIdx.x % COLS, tau = threadIdx.x / COLS;
        const int c = r * COLS + cc;
        u64 x[S::REGA];
        pdl_wait();
#pragma unroll
        for (int k = 0; k < S::REGA; ++k) x[k] = L.src[((size_t)(k * S::TA + tau) << S::LB) + c];
        __syncthreads();
        fwd_round1<S::RA, AR>(x, TwSmem{tws}, md);
#pragma unroll
        for (int k = 0; k < S::REGA; ++k) buf[(k * S::TA + tau) * COLS + cc] = x[k];
        __syncthreads();
        constexpr int M = S::TA, NG = S::REGA / S::TA;
#pragma unroll
        for (int gg = 0; gg < NG; ++gg)
#pragma unroll
            for (int k2 = 0; k2 < M; ++k2) x[gg * M + k2] = buf[((tau * NG + gg) * M + k2) * COLS + cc];
        if (AR == AR_PM && (T.pm_fold & PM_FOLD_MID)) fold_all<S::REGA, AR>(x, md);
        fwd_round2<S::LA, S::RA, AR>(x, tau, TwSmem{tws}, md);
        __syncthreads();  // every read of the transpose precedes the block's writes
#pragma unroll
        for (int gg = 0; gg < NG; ++gg)
#pragma unroll
            for (int k2 = 0; k2 < M; ++k2) buf[((tau * NG + gg) * M + k2) * COLS + cc] = x[gg * M + k2];
    }
    cluster_barrier();  // every CTA's block is complete
    // row pass on rows [r*ROWS, (r+1)*ROWS): element c of row h lives in
    // CTA c / COLS at buf[h*COLS + c % COLS]
    const int rr = threadIdx.x / S::TB, tau = threadIdx.x % S::TB;
    const int h = r * ROWS + rr;
    const int G = (1 << S::LA) + h;
    u64 x[S::REGB];
#pragma unroll
    for (int k = 0; k < S::REGB; ++k) {
        const int c = k * S::TB + tau;
        x[k] = ld_dsmem(dsmem_addr(buf + h * COLS + c % COLS, c / COLS));
    }
    ulonglong2 *tsh = tsh_all + rr * S::REGB;
    stage_row_round1<S>(tsh, twt, G, tau);
    cluster_barrier();  // no CTA reads another's block after this point
    row_fwd_core<S, AR>(x, TwStaged<S>{tsh, twt, G}, buf + rr * S::ROWPAD, tau, md, T.pm_fold);
    u64 *gout = L.dst + ((size_t)h << S::LB);
#pragma unroll
    for (int k = 0; k < S::REGB; ++k) gout[k * S::TB + tau] = CANON ? canon_any<AR>(x[k], mc) : x[k];
}

// Inverse NTT (input below 4q), then the scale (SC: the job's per-entry scale
// where its map has one, else N^-1); output canonical.
template <class S, int MUL, bool SC, int AR>
__global__ void __launch_bounds__(Cl<S, MUL>::THREADS, Cl<S, MUL>::MINB) k_inv_cl(Tables T, LimbMaps ms, int early)
{
    if (early) pdl_start();
    typedef Cl<S, MUL> G_;
    constexpr int COLS = G_::COLS, ROWS = G_::ROWS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    u64 *buf = reinterpret_cast<u64 *>(smem_raw);
    ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(buf + G_::BUFW);
    const int lg = blockIdx.y + blockIdx.z * gridDim.y;
    if (lg >= ms.pre[ms.n]) return pdl_wait();
    const LimbRef L = limb_ref(ms, lg, T.nq, T.alpha, S::LOGN);
    if (L.skip) return;
    const ModC &mc = T.modc[L.tf];
    const ModR<AR> md = mod_inv<AR>(mc);
    const int r = cluster_rank();
    const ulonglong2 *itw = T.itw + ((size_t)L.tf << S::LOGN);
    for (int i = threadIdx.x; i < (1 << S::LA); i += G_::THREADS) tws[i] = itw[i];
    {
        // row pass on rows [r*ROWS, (r+1)*ROWS); the block stays in buf as
        // buf[(h - r*ROWS) * 2^LB + c]
        const int rr = threadIdx.x / S::TB, tau = threadIdx.x % S::TB;
        const int h = r * ROWS + rr;
        const TwRow<S> tw{itw, (1 << S::LA) + h};
        const u64 *gin = L.src + ((size_t)h << S::LB);
        u64 x[S::REGB];
        pdl_wait();
#pragma unroll
        for (int k = 0; k < S::REGB; ++k) x[k] = gin[k * S::TB + tau];
        row_inv_core<S, AR>(x, tw, buf + rr * S::ROWPAD, tau, md);  // ends with buf free
#pragma unroll
        for (int k = 0; k < S::REGB; ++k) buf[rr * (1 << S::LB) + k * S::TB + tau] = x[k];
    }
    cluster_barrier();  // every CTA's block (and tws) is complete
    // column pass on columns [r*COLS, (r+1)*COLS): row h lives in CTA h / ROWS
    const int cc = threadIdx.x % COLS, tau = threadIdx.x / COLS;
    const int c = r * COLS + cc;
    constexpr int M = S::TA, NG = S::REGA / S::TA;
    u64 x[S::REGA];
#pragma unroll
    for (int gg = 0; gg < NG; ++gg)
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) {
            const int h = (tau * NG + gg) * M + k2;
            x[gg * M + k2] = ld_dsmem(dsmem_addr(buf + (h % ROWS) * (1 << S::LB) + c, h / ROWS));
        }
    cluster_barrier();  // no CTA reads another's block after this point
    fold_all<S::REGA, AR>(x, md);
    inv_round2<S::LA, S::RA, AR>(x, tau, TwSmem{tws}, md);
#pragma unroll
    for (int gg = 0; gg < NG; ++gg)
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) buf[((tau * NG + gg) * M + k2) * COLS + cc] = x[gg * M + k2];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < S::REGA; ++k) x[k] = buf[(k * S::TA + tau) * COLS + cc];
    fold_all<S::REGA, AR>(x, md);
    inv_round1<S::RA, AR>(x, TwSmem{tws}, md);
    ulonglong2 f = make_ulonglong2(0, 0);
    if (SC) f = L.scale ? L.scale[L.b] : make_ulonglong2(mc.ninv, mc.ninv_sh);
#pragma unroll
    for (int k = 0; k < S::REGA; ++k)
        L.dst[((size_t)(k * S::TA + tau) << S::LB) + c] = inv_finish<AR, SC>(x[k], f, mc);
}

template <class S, int MUL>
struct ClKernels {
    typedef Cl<S, MUL> G;
    template <int AR> static bool prepare()
    {
        return cluster_prepare(k_fwd_cl<S, MUL, false, AR>, G::C, G::THREADS, G::SMEM) &&
               cluster_prepare(k_fwd_cl<S, MUL, true, AR>, G::C, G::THREADS, G::SMEM) &&
               cluster_prepare(k_inv_cl<S, MUL, false, AR>, G::C, G::THREADS, G::SMEM) &&
               cluster_prepare(k_inv_cl<S, MUL, true, AR>, G::C, G::THREADS, G::SMEM);
    }
    // per device: attributes set and the cluster shape accepted
    static bool ready()
    {
        static std::atomic<uint64_t> done{0}, ok{0};
        once_per_device(done, [] {
            const bool r = prepare<AR_GEN>() && prepare<AR_PM>();
            int dev = 0;
            if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
            if (r) ok.fetch_or(1ull << (dev & 63));
        });
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
        return (ok.load() >> (dev & 63)) & 1;
    }
};

template <class KERN>
static cudaError_t launch_cluster(KERN kern, int C, int threads, int smem, int limbs, const Tables &T,
                                  const LimbMaps &m, int early, cudaStream_t st)
{
    const unsigned gy = (unsigned)std::min(limbs, 32768);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C, gy, (unsigned)((limbs + (int)gy - 1) / (int)gy));
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_dep
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, T, m, early);
}

// Returns KS_EUNSUPPORTED (nothing launched) when the shape or the device
// cannot run the cluster form.
template <class S, int MUL>
static int fwd_cl_SM(const Tables &T, const LimbMaps &m, bool canonical, bool alone, cudaStream_t st)
{
    typedef Cl<S, MUL> G;
    if constexpr (!G::OK) {
        return KS_EUNSUPPORTED;
    } else {
        if (!ClKernels<S, MUL>::ready()) return KS_EUNSUPPORTED;
        cudaError_t e;
        const int limbs = m.pre[m.n];
        constexpr int C = G::C, TH = G::THREADS, SM = G::SMEM;
        const int early = early_start(T, limbs, (size_t)limbs * C, G::MINB, alone);
        if (canonical)
            KS_DISPATCH_AR2(T, KS_LAUNCH(st, "ntt_fwd_cl", (e = launch_cluster(k_fwd_cl<S, MUL, true, AR>, C, TH, SM, limbs,
                                                                               T, m, early, st))))
        else
            KS_DISPATCH_AR2(T, KS_LAUNCH(st, "ntt_fwd_cl", (e = launch_cluster(k_fwd_cl<S, MUL, false, AR>, C, TH, SM, limbs,
                                                                               T, m, early, st))))
        if (e != cudaSuccess) return fail(KS_ECUDA, std::string("cluster NTT launch: ") + cudaGetErrorString(e));
        return KS_OK;
    }
}

template <class S, int MUL>
static int inv_cl_SM(const Tables &T, const LimbMaps &m, bool scaled, bool alone, cudaStream_t st)
{
    typedef Cl<S, MUL> G;
    if constexpr (!G::OK) {
        return KS_EUNSUPPORTED;
    } else {
        if (!ClKernels<S, MUL>::ready()) return KS_EUNSUPPORTED;
        cudaError_t e;
        const int limbs = m.pre[m.n];
        constexpr int C = G::C, TH = G::THREADS, SM = G::SMEM;
        const int early = early_start(T, limbs, (size_t)limbs * C, G::MINB, alone);
        if (scaled)
            KS_DISPATCH_AR2(T, KS_LAUNCH(st, "ntt_inv_cl", (e = launch_cluster(k_inv_cl<S, MUL, true, AR>, C, TH, SM, limbs,
                                                                               T, m, early, st))))
        else
            KS_DISPATCH_AR2(T, KS_LAUNCH(st, "ntt_inv_cl", (e = launch_cluster(k_inv_cl<S, MUL, false, AR>, C, TH, SM, limbs,
                                                                               T, m, early, st))))
        if (e != cudaSuccess) return fail(KS_ECUDA, std::string("cluster NTT launch: ") + cudaGetErrorString(e));
        return KS_OK;
    }
}

// T.ntt_cluster: 1 = CTAs of the two-pass size, 2 = CTAs twice as wide
template <class S>
static int fwd_cl_S(const Tables &T, const LimbMaps &m, bool canonical, bool alone, cudaStream_t st)
{
    return T.ntt_cluster == 2 ? fwd_cl_SM<S, 2>(T, m, canonical, alone, st) : fwd_cl_SM<S, 1>(T, m, canonical, alone, st);
}
template <class S>
static int inv_cl_S(const Tables &T, const LimbMaps &m, bool scaled, bool alone, cudaStream_t st)
{
    return T.ntt_cluster == 2 ? inv_cl_SM<S, 2>(T, m, scaled, alone, st) : inv_cl_SM<S, 1>(T, m, scaled, alone, st);
}

#define KS_CL_DISPATCH(logN, FN, ...)                         \
    switch (logN) {                                           \
    case 10: return FN<ShapeOf<10>::T>(__VA_ARGS__);          \
    case 11: return FN<ShapeOf<11>::T>(__VA_ARGS__);          \
    case 12: return FN<ShapeOf<12>::T>(__VA_ARGS__);          \
    case 13: return FN<ShapeOf<13>::T>(__VA_ARGS__);          \
    case 14: return FN<ShapeOf<14>::T>(__VA_ARGS__);          \
    case 15: return FN<ShapeOf<15>::T>(__VA_ARGS__);          \
    case 16: return FN<ShapeOf<16>::T>(__VA_ARGS__);          \
    case 17: return FN<ShapeOf<17>::T>(__VA_ARGS__);          \
    default: return KS_EUNSUPPORTED;                          \
    }

}  // namespace

bool ntt_cluster_shape(int logN)
{
    switch (logN) {
    case 10: return Cl<ShapeOf<10>::T, 1>::OK;
    case 11: return Cl<ShapeOf<11>::T, 1>::OK;
    case 12: return Cl<ShapeOf<12>::T, 1>::OK;
    case 13: return Cl<ShapeOf<13>::T, 1>::OK;
    case 14: return Cl<ShapeOf<14>::T, 1>::OK;
    case 15: return Cl<ShapeOf<15>::T, 1>::OK;
    case 16: return Cl<ShapeOf<16>::T, 1>::OK;
    case 17: return Cl<ShapeOf<17>::T, 1>::OK;
    default: return false;
    }
}

int launch_ntt_fwd_cluster(const Tables &T, const LimbMaps &m, bool canonical, cudaStream_t st, bool alone)
{
    KS_CL_DISPATCH(T.logN, fwd_cl_S, T, m, canonical, alone, st);
}

int launch_ntt_inv_cluster(const Tables &T, const LimbMaps &m, bool scaled, cudaStream_t st, bool alone)
{
    KS_CL_DISPATCH(T.logN, inv_cl_S, T, m, scaled, alone, st);
}

}  // namespace ks
