// ks_internal.h -- internal types of the key-switching library (host + device).
//
// Layout of everything the library keeps on the device (one parameter set):
//   modc[t]          per-tower constants, t over the full basis q_0..q_L, p_0..p_{K-1}
//   tw[t][N]         forward twiddles (w, floor(w*2^64/q), or an AR_PM pair) in bit-reversed order:
//                    tw[t][i] = psi^brv(i) for the Cooley-Tukey NTT
//   itw[t][N]        inverse twiddles psi^-brv(i) for the Gentleman-Sande iNTT
//   up_pre[...]      ModUp P1 scale N^-1 * (Q_j/q_i)^-1 mod q_i per (digit, active
//                    towers, source tower)
//   up_mat[...]      ModUp P2 matrix (Q_j/q_i) mod r per (digit, active towers,
//                    source tower, target tower), split in two 28-bit halves
//   dn_mat[k][i]     ModDown P2 matrix (P/p_k) * P^-1 mod q_i (P^-1 of P4 folded in)
//   key_sc[t]        per-tower factor folded into the stored key: P^-1 on Q towers
//                    (ModDown P4), N^-1 * (P/p_k)^-1 on P towers (ModDown P1 + P2
//                    prescale), times 2^64 for the Montgomery product of P4
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/ks.h"

namespace ks {

typedef uint64_t u64;
typedef uint32_t u32;

constexpr int kMaxQ = 64;
constexpr int kMaxP = 32;
constexpr int kMaxT = kMaxQ + kMaxP;
constexpr int kMinLogN = 10;
constexpr int kMaxLogN = 17;
constexpr int kMaxPrimeBits = 56;  // 28-bit split products in BConv; 4q < 2^58 in the NTT
constexpr int kSplit = 28;

// Butterfly form of a parameter set's primes (ks_device.cuh), and the folds
// its AR_PM forward transforms need: at the start of the row pass, and between
// the two rounds of each pass.
enum { AR_GEN = 0, AR_SP = 1, AR_PM = 2 };
enum { PM_FOLD_ROW = 1, PM_FOLD_MID = 2 };
constexpr u64 kFwdLazy = 72;  // AR_GEN, AR_SP: forward outputs are below kFwdLazy * q

// Per-tower constants.
struct ModC {
    u64 q;       // modulus
    u64 q2;      // 2q
    u64 mont;    // -q^-1 mod 2^64 (Montgomery reduction)
    u64 one_sh;  // floor(2^64 / q): Shoup companion of 1
    u64 r28, r28_sh;  // 2^28 mod q and its Shoup companion
    u64 r56, r56_sh;  // 2^56 mod q and its Shoup companion
    u64 ninv, ninv_sh;  // N^-1 mod q as a pair of the set's form (Shoup, or AR_PM)
    u64 r2;             // 2^128 mod q (into Montgomery form)
    u64 flz;            // multiple of q no forward NTT output (lazy) exceeds; flz + q < 2^64
    // q = 2^b - c just below a power of two (arith AR_PM, ks_device.cuh)
    u64 pm_T;     // multiple of q no lazy product exceeds
    u64 pm_D;     // multiple of q no value of an inverse round exceeds
    u32 pm_c2;    // 2^(b+1) - 2q
    u32 pm_k;     // b - 31
    u64 pad;
};

// Device tables of one parameter set, passed to kernels by value.
// A key as the kernels read it: a full key, or a compressed one (b stored,
// a regenerated from a_seed; see key_a_word in ks_device.cuh).
struct KeyView {
    const u64 *evk;
    u64 a_seed;
    int comp;
};

struct Tables {
    const ModC *modc;
    const ulonglong2 *tw;
    const ulonglong2 *itw;
    const ulonglong2 *up_pre;
    const u64 *up_mat;
    const u64 *dn_mat;
    const ulonglong2 *key_sc;   // Montgomery-form fold factors (see header)
    const ulonglong2 *plain_sc; // the same factors without 2^64
    const int *up_mat_lvl;    // ModUp matrix offset of digit j at level nact: [(nact-1)*ndig + j]
    // tensor-core base conversion: per-target B slabs (null when unsupported
    // or switched off) and the ModUp slab base of digit j at level nact
    const uint4 *up_tc;
    const int *up_tc_lvl;
    const uint4 *dn_tc;
    int ntt_cluster;  // host side: NTTs as one cluster launch where supported
    int row_stage;    // host side: forward row passes staged by bulk copies (k_fwd_row_st)
    int arith;        // butterfly form the primes allow (AR_GEN, AR_SP, AR_PM: ks_device.cuh); AR_PM sets hold
                      // tw, itw, the ModUp P1 factors and N^-1 as AR_PM pairs instead of Shoup pairs
    int pm_fold;      // AR_PM: folds the forward transforms need (PM_FOLD_*)
    int tc_pm_b;      // tensor-core base conversion: the moduli's common bit length where its folding epilogue
    int tc_pm_up, tc_pm_dn;  // serves the set (ModUp, ModDown; tc_reduce_pm), else 0
    int tc_below54;   // every modulus is below 2^54: 9-bit constant slices (tensor-core BConv)
    int logN;
    int nq, kp, alpha, ndig;
};

// Offsets of the ModUp tables for digit j with `a` active towers.
struct UpOffsets {
    std::vector<int> pre;  // [j * (alpha + 1) + a]
    std::vector<int> mat;
};

struct Workspace;
struct HostStage;

}  // namespace ks

struct ks_params {
    int logN = 0;
    uint32_t N = 0;
    int nq = 0, kp = 0, dnum = 0, alpha = 0, ndig = 0;
    int device = 0;
    std::vector<uint64_t> q, p, psi;  // psi over the full basis
    ks::UpOffsets up_off;
    // device allocations
    ks::ModC *d_modc = nullptr;
    ulonglong2 *d_tw = nullptr, *d_itw = nullptr;
    ulonglong2 *d_up_pre = nullptr;
    ulonglong2 *d_up_pre_lvl = nullptr;  // [nq levels][nq]: ModUp P1 factor per level
    int *d_up_mat_lvl = nullptr;         // [nq levels][ndig]: ModUp matrix offsets per level
    uint4 *d_up_tc = nullptr, *d_dn_tc = nullptr;  // tensor-core BConv slabs
    int *d_up_tc_lvl = nullptr;
    int bconv_tensor = -1;               // tensor-core BConv: -1 by size, 0 never, 1 wherever supported
    int ntt_cluster = 0;                 // NTTs as one cluster launch where supported
    int row_stage = 0;                   // forward row passes staged by bulk copies
    int batch_lanes = 2;                 // internal streams a large Output-Centric batch is split over
    cudaStream_t lane_st[4] = {};        // created on first use
    cudaEvent_t lane_ev[5] = {};
    std::mutex lane_mu;                  // one batch at a time enqueues on the lanes
    uint64_t *d_up_mat = nullptr;
    uint64_t *d_dn_mat = nullptr;
    ulonglong2 *d_key_sc = nullptr, *d_plain_sc = nullptr;
    ks::Tables tables{};
    // per-stream scratch
    std::mutex mu;
    std::map<void *, ks::Workspace *> ws;
    // default schedule (KS_OC / KS_AUTO without a tuned entry)
    ks_schedule sched{KS_OC, 1, 64, 0, -1, -1};
    // tuning cache: (job-count bucket, mean-level bucket) -> schedule;
    // every access holds tune_mu (KS_AUTO calls on several threads share it)
    std::map<std::pair<uint32_t, uint32_t>, ks_schedule> tune;
    mutable std::mutex tune_mu;
    // learned cost model consulted by KS_AUTO on a tuning-cache miss (not
    // owned), its target normalisation and its one-row input/output buffers
    ks_mlp *cost_model = nullptr;
    float cm_mean = 0.f, cm_scale = 1.f;
    float *d_cm_x = nullptr, *d_cm_y = nullptr;
    // double-buffered device staging of ks_switch_batch_host
    std::mutex host_mu;
    ks::HostStage *stage = nullptr;
};

struct ks_key {
    const ks_params *params = nullptr;
    // full key: [ndig][2][nq+kp][N]; compressed: [ndig][nq+kp][N] (b only);
    // Montgomery form with key_sc folded in
    uint64_t *d_evk = nullptr;
    size_t bytes = 0;
    int compressed = 0;
    uint64_t a_seed = 0;  // compressed: seed of the regenerated a half
    // tower shard (ks_key_shard): the limbs of full Q towers [q0, q1) and
    // special towers [p0, p1) only, [ndig][2][(q1-q0)+(p1-p0)][N]; used by
    // the ks_shard_* calls only
    int shard = 0;
    uint32_t q0 = 0, q1 = 0, p0 = 0, p1 = 0;
};

namespace ks {
// Whether the base conversions of nsrc sources to ntgt targets use the tensor
// cores.  By size: the tensor-core kernel has one CTA an SM, which allocates
// tensor memory, stages its targets and then runs producers, MMA and epilogue one
// after the other, 1.5 to 8 us a launch before its rate counts, and an output
// costs it the same at one source as at nine; the CUDA-core kernel starts at once
// and pays by the source.  One key switch (OC) and 24, us, tensor / CUDA cores:
//   L+1, K, dnum     N = 2^12                  2^13                      2^14                      2^15
//   3, 1, 3     35.3/31.1  84.7/72.5     50.3/42.6  122/94         60.9/57.4  178/140        69.3/72.1  306/251
//   6, 2, 3     36.6/33.6  92.1/72.0     57.9/49.7  149/126        64.6/69.8  253/230        76.8/89.8  481/457
//   9, 3, 3     41.5/38.1  109/102       59.3/62.7  186/190        68.6/86.2  341/371        92.3/101   667/755
//   12, 2, 6    44.8/44.5  170/163       66.4/66.9  306/317        85.1/93.6  595/642        108/114    1178/1299
//   24, 8, 3    52.5/57.3                74.7/80.4                 93.0/110                  124/140
// so the line is drawn at 2^17 multiply-adds a digit (9 targets at three sources
// and 2^12, 6 at two and 2^13, 8 at one and 2^14).  The smallest sets of the larger
// rings fall below it too.  For a lone switch of theirs the sign changes from set
// to set, as the places of the small launches' blocks do; from four jobs on the
// CUDA cores win in all of them (1, 4 and 24 jobs):
//   3, 1, 3     2^15: 71.8/73.9  111/97    309/253
//   2, 1, 2     2^15: 66.2/76.3  97.3/79.8 225/174     2^16: 73.5/65.6  123/112   396/308
//   1, 1, 1     2^16: 66.6/75.1  97.0/87.2 265/190     2^17: 93.8/79.2  142/124   487/364
inline bool bconv_tc_chosen(const ks_params *P, int nsrc, int ntgt)
{
    if (P->bconv_tensor >= 0) return P->bconv_tensor != 0;
    return ((size_t)nsrc * ntgt << P->logN) > (size_t)1 << 17;
}
inline bool up_tc_chosen(const ks_params *P) { return bconv_tc_chosen(P, P->alpha, P->nq + P->kp - P->alpha); }
inline bool dn_tc_chosen(const ks_params *P) { return bconv_tc_chosen(P, P->kp, P->nq); }

inline KeyView key_view(const ks_key *K) { return KeyView{K->d_evk, K->a_seed, K->compressed}; }
}  // namespace ks

namespace ks {

// Every kernel launch of the library runs inside a LaunchScope: the scope
// counts the launch and, while profiling is on, brackets it with CUDA events
// recorded on the launch stream (ks_profile_collect sums them per name).
class LaunchScope {
  public:
    LaunchScope(cudaStream_t st, const char *name);
    ~LaunchScope();
    LaunchScope(const LaunchScope &) = delete;
    LaunchScope &operator=(const LaunchScope &) = delete;

  private:
    cudaStream_t st_;
    long rec_ = -1;
};
#define KS_LAUNCH(st, name, ...)              \
    do {                                      \
        ::ks::LaunchScope ks_scope_(st, name); \
        __VA_ARGS__;                          \
    } while (0)

// Launch of a kernel that begins with pdl_start and whose every block calls
// pdl_wait, before it touches anything earlier work may write and before it
// leaves (ks_device.cuh): the launch may start
// while the stream's previous kernel drains (programmatic dependent launch), so
// its dispatch, its descriptors and the constants it stages overlap that
// kernel's last wave.  Ordering is the stream's: pdl_wait returns when the
// previous kernel is complete and its writes visible, and that kernel waited for
// the one before it.  12 launches at N = 2^16, one key switch: 218 -> 195 us; at
// N = 2^12: 59 -> 36 us; batches of 16 and more: no difference.
template <class T> struct Same {
    typedef T type;
};
template <class... KA>
inline void launch_dep(cudaStream_t st, void (*kern)(KA...), dim3 grid, dim3 block, size_t smem,
                       const typename Same<KA>::type &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *ptrs[] = {const_cast<void *>(static_cast<const void *>(&args))...};
    cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kern), ptrs);
}

// Per-device one-time setup (kernel attributes are per device context):
// runs setup() once for the current device; callers on other threads wait
// for it to finish.  done is the caller's static bit set of devices.
inline std::mutex &setup_mutex()
{
    static std::mutex m;
    return m;
}
template <class F>
inline void once_per_device(std::atomic<uint64_t> &done, F &&setup)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        dev = 0;
    }
    const uint64_t bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return;
    std::lock_guard<std::mutex> g(setup_mutex());
    if (done.load(std::memory_order_relaxed) & bit) return;
    setup();
    done.fetch_or(bit, std::memory_order_release);
}

// Thread-local error message (ks_last_error).
void set_error(const std::string &msg);
int fail(int code, const std::string &msg);

// Host number theory (ks_host.cpp).
bool is_prime_u64(u64 n);
int gen_primes(int logN, int bits, int count, std::vector<u64> &out);
int gen_special_primes(int bits, int count, std::vector<u64> &out);
u64 find_psi(u64 q, int logN);
u64 mulmod_h(u64 a, u64 b, u64 m);
u64 powmod_h(u64 b, u64 e, u64 m);
u64 invmod_h(u64 a, u64 m);
u64 shoup_h(u64 w, u64 q);  // floor(w * 2^64 / q)

// Batch execution under a schedule (ks_api.cu), used by the autotuner.
int run_batch(ks_params *P, uint32_t n, const ks_job *jobs, const ks_schedule &sc, cudaStream_t st);
int check_batch(const ks_params *P, uint32_t n, const ks_job *jobs);
int check_schedule(const ks_schedule *sc);
// Tuning-cache signature of a batch.
std::pair<uint32_t, uint32_t> tune_signature(uint32_t n, uint32_t mean_level);
// The schedule the parameter set's cost model predicts fastest for a batch
// (ks_tune.cu): runs the model's forward kernel on st and reads the
// predictions back (synchronises st).  h_pred (nullable) receives the raw
// outputs (predicted log ms per key switch).
int predict_schedule(ks_params *P, uint32_t n, const ks_job *jobs, cudaStream_t st, ks_schedule *out, float *h_pred);
// MLP internals used by the schedule predictor (ks_mlp.cu).
int mlp_io_dims(const ks_mlp *M, int *in, int *out);
int mlp_reserve(ks_mlp *M, int batch);
// Fill a key buffer with pseudo-random canonical residues (ks_kernels.cu).
int launch_key_random(const Tables &T, u64 *evk, uint64_t seed, cudaStream_t st);

// Build every host table and upload it (ks_host.cpp).
int build_tables(ks_params *P);
void free_tables(ks_params *P);

}  // namespace ks
