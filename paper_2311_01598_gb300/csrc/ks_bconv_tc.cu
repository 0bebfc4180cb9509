// ks_bconv_tc.cu -- fast base conversion (ModUp P2, ModDown P2) on the
// 5th-generation tensor cores (tcgen05, accumulators in tensor memory).
//
// The conversion z_t = sum_i y_i c_{i,t} mod r_t is a product of a
// [coefficients x sources] matrix by a [sources x targets] matrix of
// constants below 2^56.  Exactness with f16 operands: y_i (canonical, < 2^56)
// is cut into 7 bytes y_{i,a}, so y_i c_{i,t} = sum_a y_{i,a} 2^(8a) c_{i,t}.
// The shift of byte a is folded into the constant, c'_{i,a,t} = 2^(8a)
// c_{i,t} mod r_t, and each c' is cut into W-bit slices c'_{i,a,t,b}
// (W = 8: 7 slices; W = 9: 6 slices, when every modulus is below 2^54 and the
// sources fit one K block); then
//   z_t == sum_b 2^(Wb) P_{t,b}  (mod r_t),
//   P_{t,b} = sum_i sum_a y_{i,a} c'_{i,a,t,b},
// and every P_{t,b} (at most 18 sources x 7 bytes x 255^2, or 9 x 7 x 255 x
// 511 with W = 9, below 2^23) is an exact integer in the fp32 accumulator.
// One MMA of M=128 coefficients, K = 7*(sources) padded to 64 (up to 9 sources) or 128 (up to 18: two K
// blocks), N = 8 per target (7 byte rows used) computes
// all P_{t,b} of up to 32 targets.  19 to 36 sources take two such A tiles with
// an accumulator each, added in the epilogue (16 targets at a time).  The A
// tile holds the byte slices of y
// (built by the CTA from the source limbs), the B tile the per-target slabs
// B[b][7i+a] = c'_{i,a,t,b} (precomputed on the host, 1 KB a K block).  The
// epilogue reads the 6 or 7 sums from tensor memory and recombines them into
// S = sum_{i,a} y_{i,a} c'_{i,a,t} exactly; S <= 126*255*r < 2^15 r.  For moduli
// just below a power of two (AR_PM, ks_device.cuh) the top bits of S are folded
// by r = 2^b - c (tc_reduce_pm), an output below 4r; otherwise one Montgomery
// step by 2^32 (constants carry 2^32) leaves (S + m r)/2^32 below 2r.  Either
// is the same residue as the CUDA-core kernels' lazy output.
//
// Operand layout: the canonical K-major layout without swizzle: 8x16-byte
// core matrices, K-adjacent core matrices 128 bytes apart (LBO), 8-row
// groups 1024 bytes a K block apart (SBO); B slabs of 8 rows concatenate.
#include <algorithm>

#include "ks_device.cuh"
#include "ks_launch.h"

namespace ks {

namespace {

constexpr int TC_M = 128;            // coefficients per MMA tile
constexpr int TC_TB = 32;            // targets per MMA (8 accumulator columns each)
constexpr uint32_t TC_LBO = 128;
// KB K blocks of 64: K = 64*KB columns (7 x up to 9*KB sources, the last
// column the bias), 8-row groups K/8*128 bytes apart, slabs of 8 rows.
template <int KB> struct TcK {
    static constexpr int K = 64 * KB;
    static constexpr uint32_t SBO = (K / 8) * 128;
    static constexpr int SLAB = 8 * K * 2;  // bytes of one target slab
    static constexpr int SRC = 9 * KB;            // sources of one A tile
    static constexpr int ATILE = TC_M * K * 2;    // bytes of an A tile
};
// Targets of one item: both accumulator buffers hold NS accumulators of 8
// columns a target in 512 columns of tensor memory.
template <int NS> struct TcTargets {
    static constexpr int N = TC_TB / NS;
};
static_assert(TcK<1>::SLAB == 2 * kTcSlabHalves && TcK<2>::SLAB == 4 * kTcSlabHalves, "slab size");
constexpr int TC_WAIT_LIMIT = 1 << 24;  // mbarrier polls before giving up

__device__ int g_tc_error;  // set when an MMA completion wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

template <int KB>
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)((TC_LBO >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((TcK<KB>::SBO >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of this architecture; no swizzle
    return d;
}
// kind::f16 instruction descriptor: D f32, A and B f16, both K-major.
__device__ __forceinline__ uint32_t tc_idesc(int n)
{
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}
template <int KB>
__host__ __device__ __forceinline__ uint32_t tc_off(int r, int k)
{
    return (uint32_t)((r / 8) * TcK<KB>::SBO + (k / 8) * TC_LBO + (r % 8) * 16 + (k % 8) * 2);
}
// Two bytes as an exact f16 pair: byte a0 of word x (low half) and byte a1 of
// word y (high half).  0x6400 | b is the f16 of 1024 + b (b < 1024), so one
// byte permute, one logic op and one packed subtraction of 1024 give (b0, b1).
// The selector is a constant once the callers' loops are unrolled.
__device__ __forceinline__ uint32_t f16x2_bytes(uint32_t x, uint32_t y, uint32_t a0, uint32_t a1)
{
    const uint32_t sel = a0 | ((4u + a1) << 8);  // x.byte[a0] -> byte 0, y.byte[a1] -> byte 2
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(y), "r"(sel));
    d = (d & 0x00FF00FFu) | 0x64006400u;
    uint32_t r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(d), "r"(0x64006400u));
    return r;
}

// The shifted partial sums of one target (W-bit slices: 7 for W = 8, 6 for
// W = 9), recombined and reduced by one Montgomery step by 2^32.  v[b] are the
// raw accumulator bits 0x4B000000 + P_b (bias column); the bias is removed
// once per group (modulo 2^64: the exact sums fit).  qinv = -q^-1 mod 2^32.
template <int W>
__device__ __forceinline__ u64 tc_reduce(const uint32_t *v, u64 q, uint32_t qinv)
{
    constexpr u64 B = 0x4B000000ull;
    constexpr u64 B5 = B * (1ull + (1ull << W) + (1ull << (2 * W)) + (1ull << (3 * W)) + (1ull << (4 * W)));
    u64 a0 = 0;
#pragma unroll
    for (int b = 0; b < 5; ++b) a0 += (u64)v[b] << (W * b);
    a0 -= B5;                           // P_0 + ... + P_4 2^(4W) < 2^(23 + 4W + 1)
    u64 a1;                             // the sums above, at 2^(5W)
    if constexpr (W == 8)
        a1 = (u64)v[5] + ((u64)v[6] << 8) - B * 0x0101ull;
    else
        a1 = (u64)v[5] - B;
    const u64 t1 = a1 << (5 * W);
    const u64 lo = a0 + t1;
    const uint32_t hi = (uint32_t)(a1 >> (64 - 5 * W)) + (lo < t1 ? 1u : 0u);  // S = lo + hi 2^64
    // (S + m q) / 2^32 with m = -S q^-1 mod 2^32: the low word of S + m q is 0
    const uint32_t l0 = (uint32_t)lo, l1 = (uint32_t)(lo >> 32);
    const uint32_t m = l0 * qinv;
    const u64 w = (u64)m * (uint32_t)q + l0;
    return (u64)m * (uint32_t)(q >> 32) + (w >> 32) + l1 + ((u64)hi << 32);
}

// The same recombination for moduli r = 2^b - c.  Neighbouring sums pair up in
// 32 bits, a_{2i} = P_{2i} + P_{2i+1} 2^W (W = 9: at most 9*7*255*511*513 <
// 2^32; W = 8 and up to 36 sources in NS accumulators: 36*7*255*255*257 < 2^32;
// the shifted accumulator's bias, NS * 75 * 2^24 << W, vanishes modulo 2^32, so
// one constant per pair takes the bias out), and the bits of S from b up are
// multiplied by c:
//   W = 9: S = a01 + a23 2^18 + a45 2^36,
//   W = 8: S = a01 + a23 2^16 + (a45 + P_6 2^16) 2^32.
// Outputs are below 4r (tc_pm_ok, checked for the set on the host).  15-17
// instructions an output against 35 for the Montgomery form (ModUp conversion of
// 16 key switches, N = 2^16, 24 + 8 primes, 3 digits: 235 -> 219 us).
template <int W, int NS>
__device__ __forceinline__ u64 tc_reduce_pm(const uint32_t *v, uint32_t c, int b)
{
    constexpr uint32_t B = NS * 0x4B000000u;
    const uint32_t a01 = v[0] - B + (v[1] << W);
    const uint32_t a23 = v[2] - B + (v[3] << W);
    const uint32_t a45 = v[4] - B + (v[5] << W);
    if constexpr (W == 9) {
        const u64 x = mul_wide(a23, 1u << 18);
        const uint32_t hi = (uint32_t)(x >> 32) + ((a45 & ((1u << (b - 36)) - 1)) << 4);
        return mad_wide(a45 >> (b - 36), c, ((u64)hi << 32) | (uint32_t)x) + a01;
    } else {
        const u64 u = mul_wide(v[6] - B, 1u << 16) + a45;
        const u64 x = mul_wide(a23, 1u << 16);
        const uint32_t hi = (uint32_t)(x >> 32) + ((uint32_t)u & ((1u << (b - 32)) - 1));
        return mad_wide((uint32_t)(u >> (b - 32)), c, ((u64)hi << 32) | (uint32_t)x) + a01;
    }
}

// 16 consecutive accumulator columns of this warp's 32 lanes (no wait).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}

__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t phase)
{
    uint32_t done = 0;
    for (int it = 0; it < TC_WAIT_LIMIT && !done; ++it)
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(mbar), "r"(phase)
            : "memory");
    return done != 0;
}

// One unit of work: a tile of 128 coefficients for one block of at most 32
// targets (16 with two A tiles) of one (job, digit) (ModUp) or (job, polynomial) (ModDown).
struct TcItem {
    const u64 *src;     // source tower 0 at the tile's first coefficient; tower i at + i*N
    int nsrc;           // source towers (<= 36)
    int G;              // targets (0: nothing to do)
    int sbase;          // slab index base (ModUp: of the digit at this level)
    int t_first, ov_at, ov, nact, t_base;  // target numbering (ModUp)
    u64 *dst0;          // output base: target t at dst0 + (t - t_base)*N
};

template <int MODE>
__device__ __forceinline__ TcItem tc_item(const Tables &T, const BUpJobs &bu, const BDnJobs &bd, int item, int XT,
                                          int TBN, int TB)
{
    const size_t N = (size_t)1 << T.logN;
    const int xt = item % XT, r = item / XT, tb = r % TBN, z = r / TBN;
    TcItem it;
    if (MODE == 0) {
        const int jb = find_slot(bu.zpre, bu.n, z);
        const BUpJob &J = bu.job[jb];
        const int j = J.jsel >= 0 ? J.jsel : z - bu.zpre[jb];
        const int lo = j * T.alpha, hi = min(lo + T.alpha, J.nact);
        const int olo = max(lo, J.t_begin), ohi = min(hi, J.t_end);
        it.ov = ohi > olo ? ohi - olo : 0;
        it.ov_at = olo;
        const int nb = (J.t_end - J.t_begin) - it.ov;
        const int u0 = tb * TB;
        it.G = max(0, min(TB, nb - u0));
        it.t_first = J.t_begin + u0;
        it.nact = J.nact;
        it.t_base = J.t_base;
        it.nsrc = hi - lo;
        it.src = J.y + (size_t)lo * N + (size_t)xt * TC_M;
        it.sbase = T.up_tc_lvl[(size_t)(J.nact - 1) * T.ndig + j];
        it.dst0 = J.D + (size_t)(J.jsel >= 0 ? 0 : j) * J.dstride + (size_t)xt * TC_M;
    } else {
        const int jb = find_slot(bd.zpre, bd.n, z);
        const BDnJob &J = bd.job[jb];
        const int x = z - bd.zpre[jb];
        const int i0 = tb * TB;
        it.G = max(0, min(TB, J.nact - i0));
        it.t_first = i0;
        it.ov = 0;
        it.ov_at = 0;
        it.nact = J.nact;
        it.t_base = 0;
        it.nsrc = T.kp;
        it.src = J.cp + (size_t)x * J.cp_stride + (size_t)J.nact * N + (size_t)xt * TC_M;
        it.sbase = 0;
        it.dst0 = J.v + (size_t)x * J.v_stride + (size_t)xt * TC_M;
    }
    return it;
}

// target g of an item: compact tower, full tower, slab
template <int MODE>
__device__ __forceinline__ void tc_target(const Tables &T, const TcItem &it, int g, int &t, int &tf, int &slab)
{
    if (MODE == 0) {
        t = it.t_first + g;
        if (it.ov > 0 && t >= it.ov_at) t += it.ov;
        tf = full_tower(t, it.nact, T.nq);
        slab = it.sbase + tf;
    } else {
        t = it.t_first + g;
        tf = t;
        slab = t;
    }
}

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t a)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
// OR of a flag over the threads of a named barrier.
template <int ID, int COUNT>
__device__ __forceinline__ bool bar_or(bool f)
{
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((uint32_t)f), "n"(ID), "n"(COUNT)
        : "memory");
    return r != 0;
}

constexpr int TC_PROD = 256;                  // producer threads (warps 0-7): two groups, one thread per tile row
constexpr int TC_CONS_WARPS = 16;             // consumer warps: 4 lane quarters x 4 target groups
constexpr int TC_PIPE_THREADS = TC_PROD + 32 * TC_CONS_WARPS;
constexpr int TC_TILE_COST = 18;              // work of an A tile in epilogues of one target (TcSplit)
constexpr uint32_t TC_PIPE_COLS = 512;        // two accumulators of 256 columns

// Row m of an A tile from its sources' words (zero past the item's sources):
// column 7i + a = byte a of source i, the last column the bias.
template <int KB>
__device__ __forceinline__ void tc_build_row(unsigned char *sa, int m, const u64 (&y)[TcK<KB>::SRC])
{
    constexpr int K = TcK<KB>::K;
    constexpr int SRC = TcK<KB>::SRC;  // with two K blocks column 126 is spare (0)
#pragma unroll
    for (int c = 0; c < K / 8; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const int k0 = 8 * c + e, k1 = k0 + 1;
            const int a0 = k0 % 7, a1 = k1 % 7;
            const uint32_t x0 = k0 / 7 < SRC ? (uint32_t)(y[k0 / 7 < SRC ? k0 / 7 : 0] >> (32 * (a0 / 4))) : 0u;
            if (k1 == K - 1) {  // the last slice byte, then the bias 2048 (f16 0x6800)
                w[e / 2] = (f16x2_bytes(x0, 0u, (uint32_t)(a0 % 4), 0u) & 0xFFFFu) | 0x68000000u;
            } else {
                const uint32_t x1 = (uint32_t)(y[k1 / 7] >> (32 * (a1 / 4)));  // k1 < K - 1: a source's byte
                w[e / 2] = f16x2_bytes(x0, x1, (uint32_t)(a0 % 4), (uint32_t)(a1 % 4));
            }
        }
        *reinterpret_cast<uint4 *>(sa + tc_off<KB>(m, 8 * c)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Runs of items per CTA with about equal work: items of job j cost w[j] (their
// targets plus the cost of building an A tile); cpre are the costs of the jobs
// before, ipre their items.  Equal counts instead left the CTAs that drew the
// top-level jobs of a mixed batch working alone at the end.
struct TcSplit {
    int n;
    uint32_t cpre[kMaxBatch + 1];
    int ipre[kMaxBatch + 1];
    uint16_t w[kMaxBatch];
};
__device__ __forceinline__ int tc_run_start(const TcSplit &sp, int cta, int ctas)
{
    if (cta >= ctas) return sp.ipre[sp.n];
    const uint32_t at = (uint32_t)((u64)sp.cpre[sp.n] * (uint32_t)cta / (uint32_t)ctas);
    int lo = 0, hi = sp.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sp.cpre[mid] <= at)
            lo = mid;
        else
            hi = mid - 1;
    }
    return sp.ipre[lo] + (int)((at - sp.cpre[lo]) / sp.w[lo]);
}

// Persistent pipelined base conversion: each CTA (one per SM) takes a
// contiguous run of items.  For every stretch of items that differ only in
// their coefficients, the producer warps stage the B slabs and the targets'
// outputs and constants once.  Two producer groups of 128 threads, a thread per
// tile row, take the stretch's items in turn, each with its own A tiles and
// accumulator buffer: build the A tile from the sources in registers, issue the
// loads of the group's next item, then one thread issues the MMAs and commits
// them to acc_full.  Consumer warps wait on acc_full, run the epilogue and
// release the buffer through acc_empty; an item of no targets ends them.  Every
// wait is bounded: on timeout the kernel sets g_tc_error and its threads leave
// their loops.
// What bounds it: the consumers' integer work at 24 targets an item (some 50
// cycles of a scheduler an output, six warps each), the producers' chain (source
// loads, tile, fence, barrier, issue) at few.  Measured for the ModUp conversion
// of 16 key switches at N = 2^16 (24576 items of 24 targets): one group of 256
// threads that fetched the targets' constants for every item 219 us (the load's
// 700 cycles in its serial chain), targets staged once a stretch 193, two groups
// 169.  More overlap only added instructions: consumers split between the
// buffers 180, four half-item buffers 176, a warp of its own for the issue 182,
// sources copied three items ahead 173.
// KB: K blocks of an A tile; NS: A tiles (and accumulators) an item; PM: the
// set's moduli are 2^b - c, b = T.tc_pm_b (tc_reduce_pm).
template <int MODE, int KB, int NS, int W, bool PM>
__global__ void __launch_bounds__(TC_PIPE_THREADS, 1) k_bconv_tc(Tables T, BUpJobs bu, BDnJobs bd, const uint4 *slabs,
                                                                int XT, int TBN, int TB, TcSplit split)
{
    constexpr int K = TcK<KB>::K, ATILE = TcK<KB>::ATILE, SLAB = TcK<KB>::SLAB;
    constexpr int TBM = TcTargets<NS>::N;
    extern __shared__ unsigned char tc_dyn[];
    unsigned char *sa0 = tc_dyn + ((128 - (smem_u32(tc_dyn) & 127)) & 127);  // [2 buffers][NS] A tiles
    unsigned char *sb = sa0 + 2 * NS * ATILE;                               // [NS][TBM] B slabs
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
    __shared__ uint32_t tbase_s;
    __shared__ u64 *s_dst[TBM];       // output of each target at the stretch's first coefficient
    __shared__ u64 s_q[TBM];
    __shared__ uint32_t s_red[TBM];   // -q^-1 mod 2^32, or c (PM)
    __shared__ int s_G[2], s_off[2];  // of the item in each buffer: targets, coefficients past the stretch's first
    pdl_start();
    const int i0 = tc_run_start(split, blockIdx.x, gridDim.x), i1 = tc_run_start(split, blockIdx.x + 1, gridDim.x);
    if (i0 >= i1) return pdl_wait();
    const size_t N = (size_t)1 << T.logN;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 2);              // MMA commit + producer release of the item
            mbar_init(smem_u32(&acc_empty[b]), TC_CONS_WARPS);  // one arrival per consumer warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tbase_s)),
                     "r"(TC_PIPE_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = tbase_s;
    pdl_wait();

    if (tid < TC_PROD) {
        // ------------------------------------------------------------ producers
        const int m = tid % TC_M, grp = tid / TC_M;  // tile row, group (items and buffer of this parity)
        const uint32_t full = smem_u32(&acc_full[grp]), empty = smem_u32(&acc_empty[grp]);
        unsigned char *sa = sa0 + grp * (NS * ATILE);
        int k0 = 0;  // items before the stretch
        bool ok = true;
        for (int item = i0; item < i1;) {
            const TcItem it = tc_item<MODE>(T, bu, bd, item, XT, TBN, TB);
            const int n = min(i1 - item, XT - item % XT);
            item += n;
            if (it.G == 0) continue;
            // new targets: every earlier item must be done with the slabs and tables
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int used = (k0 + 1 - b) >> 1;  // items that took buffer b
                ok = ok && (used == 0 || tc_wait(smem_u32(&acc_empty[b]), (uint32_t)((used - 1) & 1)));
            }
            if (bar_or<3, TC_PROD>(!ok)) {
                ok = false;
                break;
            }
            {
                // G slabs, and a zero slab after an odd G (the MMA's N is a
                // multiple of 16 columns: two targets)
                constexpr int WS = SLAB / 16;
                const int Gp = (it.G + 1) & ~1;
                for (int idx = tid; idx < Gp * NS * WS; idx += TC_PROD) {
                    const int g = idx / (NS * WS), w = idx % (NS * WS);
                    uint4 val = make_uint4(0u, 0u, 0u, 0u);
                    if (g < it.G) {
                        int t, tf, slab;
                        tc_target<MODE>(T, it, g, t, tf, slab);
                        val = slabs[(size_t)slab * (NS * WS) + w];
                    }
                    reinterpret_cast<uint4 *>(sb + ((w / WS) * TBM + g) * SLAB)[w % WS] = val;
                }
            }
            if (tid < it.G) {
                int t, tf, slab;
                tc_target<MODE>(T, it, tid, t, tf, slab);
                s_dst[tid] = it.dst0 + (size_t)(t - it.t_base) * N;
                if (!PM) s_q[tid] = T.modc[tf].q;
                s_red[tid] = PM ? T.modc[tf].pm_c2 >> 1 : (uint32_t)T.modc[tf].mont;
            }
            // the slabs' writes ordered before the other group's MMAs too
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bar_or<3, TC_PROD>(false);
            int k = k0 + ((k0 ^ grp) & 1);  // the group's first item of the stretch
            const u64 *src = it.src + (size_t)(k - k0) * TC_M + m;
            u64 y[TcK<KB>::SRC];
            auto load = [&](int s) {
#pragma unroll
                for (int u = 0; u < TcK<KB>::SRC; ++u) {
                    const int i = s * TcK<KB>::SRC + u;
                    y[u] = i < it.nsrc ? src[(size_t)i * N] : 0;
                }
            };
            if (k < k0 + n) load(0);
            for (; k < k0 + n; k += 2) {
                // the accumulators and A tiles of this buffer were last used by item k-2
                const int used = k >> 1;
                ok = used == 0 || tc_wait(empty, (uint32_t)((used - 1) & 1));
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    tc_build_row<KB>(sa + s * ATILE, m, y);
                    if (s + 1 < NS) load(s + 1);
                }
                if (k + 2 < k0 + n) {  // in flight while this item is issued and the buffer awaited
                    src += 2 * TC_M;
                    load(0);
                }
                if (m == 0) {
                    s_G[grp] = it.G;
                    s_off[grp] = (k - k0) * TC_M;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (grp == 0 ? bar_or<1, TC_M>(!ok) : bar_or<2, TC_M>(!ok)) {
                    ok = false;
                    break;
                }
                if (m == 0) {
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t idesc = tc_idesc(8 * ((it.G + 1) & ~1));
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const uint32_t dcol = tbase + (uint32_t)(grp * 256 + s * 8 * TBM);
#pragma unroll
                        for (int kk = 0; kk < K / 16; ++kk) {
                            const uint64_t ad = tc_desc<KB>(smem_u32(sa + s * ATILE) + kk * 2 * TC_LBO);
                            const uint64_t bdsc = tc_desc<KB>(smem_u32(sb + s * TBM * SLAB) + kk * 2 * TC_LBO);
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dcol),
                                "l"(ad), "l"(bdsc), "r"(idesc), "r"((uint32_t)kk));
                        }
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(full)
                                 : "memory");
                    mbar_arrive(full);  // releases the targets' tables and the item's G and offset
                }
            }
            k0 += n;
        }
        const bool mine = (k0 & 1) == grp;  // the group whose buffer comes next
        const int used = (k0 + 1 - grp) >> 1;
        if (m == 0) {
            // the consumers' end: an item of no targets, once its buffer is free
            if (ok && mine && used > 0) ok = tc_wait(empty, (uint32_t)((used - 1) & 1));
            if (ok && mine) {
                s_G[grp] = 0;
                mbar_arrive(full);
                mbar_arrive(full);
            }
            if (!ok) {
                atomicExch(&g_tc_error, 1);
                // bounded waits for MMAs still in flight before the memory is freed
                tc_wait(full, 0);
                tc_wait(full, 1);
            }
        }
    } else {
        // ------------------------------------------------------------ consumers
        const int cw = warp - TC_PROD / 32, quarter = cw % 4, part = cw / 4;
        const int row = quarter * 32 + lane;
        const uint32_t tq = tbase + ((uint32_t)(quarter * 32) << 16);
        bool ok = true;
        auto reduce = [&](const uint32_t *v, int g) {
            if constexpr (PM)
                return tc_reduce_pm<W, NS>(v, s_red[g], T.tc_pm_b);
            else
                return tc_reduce<W>(v, s_q[g], s_red[g]);
        };
        for (int k = 0;; ++k) {
            const int buf = k & 1;
            const bool got = tc_wait(smem_u32(&acc_full[buf]), (uint32_t)((k >> 1) & 1));
            if (__any_sync(0xffffffffu, !got)) {  // the warp's lanes agree (tcgen05.ld is warp-collective)
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int G = s_G[buf], NP = (G + 1) / 2;
            if (G == 0) break;
            const int at = s_off[buf] + row;
            // target pairs (2p, 2p+1: 16 columns) strided over the four warps
            // of a lane quarter, two tensor-memory loads in flight per wait
            for (int p = part; p < NP; p += NS == 1 ? 8 : 4) {
                uint32_t v[16], w[16];
                const uint32_t taddr = tq + (uint32_t)(buf * 256 + 16 * p);
                const bool two = NS == 1 && p + 4 < NP;
                tmem_ld16(taddr, v);
                if (NS == 2)
                    tmem_ld16(taddr + 8 * TBM, w);
                else if (two)
                    tmem_ld16(taddr + 64, w);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (NS == 2) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] += w[i];
                }
                const int g = 2 * p;
                s_dst[g][at] = reduce(v, g);
                if (g + 1 < G) s_dst[g + 1][at] = reduce(v + 8, g + 1);
                if (two) {
                    s_dst[g + 8][at] = reduce(w, g + 8);
                    if (g + 9 < G) s_dst[g + 9][at] = reduce(w + 8, g + 9);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[buf]));
        }
        if (!ok && lane == 0) atomicExch(&g_tc_error, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(TC_PIPE_COLS));
}

// Dynamic shared memory: two buffers of NS A tiles (16 KB, or 32 KB with two K
// blocks) and the B slabs (1 or 2 KB a target and tile), padded so that one CTA
// holds an SM (it takes all 512 columns of tensor memory).
template <int KB, int NS> constexpr int tc_pipe_smem()
{
    return std::max(120 * 1024, 2 * NS * TcK<KB>::ATILE + NS * TcTargets<NS>::N * TcK<KB>::SLAB + 128);
}
static_assert(tc_pipe_smem<2, 2>() <= 200 * 1024, "shared memory of an SM");

}  // namespace

bool bconv_tc_supported(const Tables &T, int nsrc)
{
    return nsrc <= tc_max_sources(T.tc_pm_b) && (((size_t)1 << T.logN) % (size_t)TC_M) == 0;
}

static int sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        n = 1;
    }
    return n;
}

template <int MODE, int KB, int NS, int W, bool PM>
static int launch_tc(const Tables &T, const BUpJobs &bu, const BDnJobs &bd, int span, const uint4 *slabs, cudaStream_t st,
                     const char *name)
{
    // target blocks of equal size (at most 32, or 16 with two tiles): 38 targets run as 19 + 19
    constexpr int TBM = TcTargets<NS>::N;
    const int TBN = (span + TBM - 1) / TBM;
    const int TB = (span + TBN - 1) / TBN;
    static std::atomic<uint64_t> attr{0};
    once_per_device(attr, [] {
        cudaFuncSetAttribute(k_bconv_tc<MODE, KB, NS, W, PM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             tc_pipe_smem<KB, NS>());
    });
    const int XT = (int)(((size_t)1 << T.logN) / TC_M);
    // Cost of an item: its targets' epilogues plus the A tile, averaged over the
    // job's target blocks (measured 0.46 us + 0.0245 us a target: 18 targets' worth).
    TcSplit sp;
    sp.n = MODE == 0 ? bu.n : bd.n;
    u64 cost = 0, items = 0;  // at most 64 jobs x 64 digits x 1024 tiles x 6 blocks of cost 50: below 2^31
    for (int j = 0; j < sp.n; ++j) {
        const int z = MODE == 0 ? bu.zpre[j + 1] - bu.zpre[j] : bd.zpre[j + 1] - bd.zpre[j];
        const int targets = MODE == 0 ? bu.job[j].t_end - bu.job[j].t_begin : bd.job[j].nact;
        sp.w[j] = (uint16_t)(std::min(targets / TBN, TB) + TC_TILE_COST);
        sp.cpre[j] = (uint32_t)cost;
        sp.ipre[j] = (int)items;
        items += (u64)XT * TBN * z;
        cost += (u64)XT * TBN * z * sp.w[j];
    }
    if (items == 0) return KS_OK;
    sp.cpre[sp.n] = (uint32_t)cost;
    sp.ipre[sp.n] = (int)items;
    const int grid = (int)std::min<u64>(items, (u64)sm_count());
    constexpr int SM = tc_pipe_smem<KB, NS>();
    KS_LAUNCH(st, name,
              (launch_dep(st, k_bconv_tc<MODE, KB, NS, W, PM>, grid, TC_PIPE_THREADS, SM, T, bu, bd, slabs, XT, TBN, TB, sp)));
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? KS_OK : fail(KS_ECUDA, std::string(name) + " (tensor cores) launch: " + cudaGetErrorString(e));
}

// The kernel of a conversion with nsrc sources.
template <int MODE>
static int launch_tc_for(const Tables &T, const BUpJobs &bu, const BDnJobs &bd, int nsrc, int span, const uint4 *slabs,
                         cudaStream_t st, const char *name)
{
    const int kb = tc_kblocks(nsrc), bits = tc_slice_bits(kb, T.tc_below54);
    if (MODE == 0 ? T.tc_pm_up : T.tc_pm_dn) {
        if (kb == 4) return launch_tc<MODE, 2, 2, 8, true>(T, bu, bd, span, slabs, st, name);
        if (kb == 2) return launch_tc<MODE, 2, 1, 8, true>(T, bu, bd, span, slabs, st, name);
        return bits == 9 ? launch_tc<MODE, 1, 1, 9, true>(T, bu, bd, span, slabs, st, name)
                         : launch_tc<MODE, 1, 1, 8, true>(T, bu, bd, span, slabs, st, name);
    }
    if (kb == 2) return launch_tc<MODE, 2, 1, 8, false>(T, bu, bd, span, slabs, st, name);
    return bits == 9 ? launch_tc<MODE, 1, 1, 9, false>(T, bu, bd, span, slabs, st, name)
                     : launch_tc<MODE, 1, 1, 8, false>(T, bu, bd, span, slabs, st, name);
}

int launch_bconv_up_tc(const Tables &T, const BUpJobs &b, cudaStream_t st)
{
    const int span = bup_span(T, b);
    if (span <= 0) return KS_OK;
    BDnJobs none;
    none.n = 0;
    return launch_tc_for<0>(T, b, none, T.alpha, span, T.up_tc, st, "bconv_up");
}

int launch_bconv_down_tc(const Tables &T, const BDnJobs &b, cudaStream_t st)
{
    int span = 0;
    for (int i = 0; i < b.n; ++i) span = std::max(span, b.job[i].nact);
    if (span <= 0) return KS_OK;
    BUpJobs none;
    none.n = 0;
    return launch_tc_for<1>(T, none, b, T.kp, span, T.dn_tc, st, "bconv_down");
}

int tc_error_flag(bool clear)
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    if (clear && v) {
        const int z = 0;
        cudaMemcpyToSymbol(g_tc_error, &z, sizeof(int));
    }
    return v;
}

// Host: the B slab of one target of modulus r: rows b (slice b of the
// folded constant, W bits; rows past the slices zero), columns k = 7i + a
// (source i, byte a of y): slice b of c_i * 2^(8a) mod r, times 2^32 for the
// Montgomery epilogue; the last column holds the bias.
template <int KB>
static void tc_slab_kb(const u64 *c, int n, u64 r, int W, bool pm, uint16_t *slab)
{
    constexpr int K = TcK<KB>::K;
    const int NSL = W == 8 ? 7 : 6;
    const u64 f = pm ? 1 : (u64)(((unsigned __int128)1 << 32) % r);
    u64 sh[7];  // 2^(8a), with the epilogue's factor
    for (int a = 0; a < 7; ++a) sh[a] = mulmod_h(f, powmod_h(2, 8 * (u64)a, r), r);
    for (int k = 0; k < K; ++k) {
        const int i = k / 7, a = k % 7;
        const u64 cf = (k < K - 1 && i < n) ? mulmod_h(c[i], sh[a], r) : 0;
        for (int b = 0; b < 8; ++b) {
            const uint32_t sl = b < NSL ? (uint32_t)((cf >> (W * b)) & ((1u << W) - 1)) : 0u;
            // f16 of an integer below 2048
            uint16_t bits = 0;
            if (sl) {
                int e = 31 - __builtin_clz(sl);                   // exponent
                uint32_t mant = (sl << (10 - e)) & 0x3FF;          // 10 fraction bits
                bits = (uint16_t)(((15 + e) << 10) | mant);
            }
            slab[tc_off<KB>(b, k) / 2] = bits;
        }
    }
    // the last column (never a slice: 9*KB sources use the columns before it)
    // holds 4096 in the used slice rows; times the A tile's 2048 there it
    // adds 2^23, so the fp32 accumulator of P (< 2^23) reads 2^23 + P: its
    // bits are 0x4B000000 + P
    for (int b = 0; b < NSL; ++b) slab[tc_off<KB>(b, K - 1) / 2] = (uint16_t)((15 + 12) << 10);
}

void tc_slab(const std::vector<u64> &c, u64 r, int kblocks, int bits, bool pm, uint16_t *slab)
{
    const int n = (int)c.size();
    if (kblocks == 1) {
        tc_slab_kb<1>(c.data(), n, r, bits, pm, slab);
    } else {
        const int s0 = std::min(n, TcK<2>::SRC);  // sources of the first tile
        tc_slab_kb<2>(c.data(), s0, r, 8, pm, slab);
        if (kblocks == 4) tc_slab_kb<2>(c.data() + s0, n - s0, r, 8, pm, slab + TcK<2>::SLAB / 2);
    }
}

// Whether tc_reduce_pm's output stays below 4q (the NTT's input bound) for
// moduli q = 2^b - c, c at most cmax.
bool tc_pm_ok(int bits, int b, u64 cmax)
{
    typedef unsigned __int128 u128;
    const u128 q4 = 4 * (((u128)1 << b) - cmax), word = (u128)1 << 32;
    if (bits == 9)
        return b >= 40 && b <= 54 && word + (word << 18) + ((u128)1 << b) + (((word - 1) >> (b - 36)) * cmax) < q4;
    return b >= 40 && b <= 56 && word + (word << 16) + ((u128)1 << b) + (((word << 8) + word) >> (b - 32)) * cmax < q4;
}

}  // namespace ks
