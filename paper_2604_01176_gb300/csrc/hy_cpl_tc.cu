// hy_cpl_tc.cu -- phase A of the float alpha-beta coupling on the fifth-
// generation tensor cores (tcgen05, accumulators in tensor memory).
//
// Per alpha string J (one persistent CTA per SM, grid-stride over J) and
// column tile of 128 beta strings b':
//   T[J][m][b'] = sum_t W_J[m][t] G_J[t][b']        m < nexa (tensor cores)
//   T[J][nexa][b'] = sum_t Wd_J[t] G_J[t][b']         (diagonal slot, FP32 SIMT)
// with the beta excitation types t = r*16 + s (r created in b', s its
// partner's orbital; s = r the diagonal pair), G_J[t][b'] = sign * psi[J][b'
// with r -> s] (zero where b' has no such excitation), W_J[m][t] the coupling
// coefficient of the m-th single-excitation partner of J and Wd_J[t] the
// diagonal coefficient sum_{p in J} V[p][p][t] (the same quantities as the
// SIMT kernel k_cpl_gemm, hy_sigma.cu).  Phase B (k_cpl_gather) is shared.
//
// FP32 accuracy from TF32 inputs: every operand is split x = hi + lo with hi
// the top 19 bits (exact in TF32) and lo = x - hi, and the tensor cores add
// hi*hi + hi*lo + lo*hi (the lo*lo term is below 2^-22 relative).
//
// Shared memory per CTA: psi's row J (every gather of G_J reads it), W_J in
// FP32, and two stages of MMA operands -- W hi/lo for 32 types (64 x 32) and
// G hi/lo for 32 types x 128 columns -- in the no-swizzle K-major layout
// (8-row x 16-byte core matrices; consecutive cores along K 128 bytes apart,
// along M/N `sbo` bytes apart).  All threads build one stage while the
// tensor cores multiply the other; the beta excitation entries of the next
// chunk are loaded while the current one is built.  A warp of its own issues
// the MMAs (M = 64, N = 128, K = 8), so its wait for the tensor cores to
// accept them never stalls a builder, and commits each stage to its mbarrier.
// Every wait is bounded (spin_limit polls of the mbarrier): on a timeout the
// kernel records it in *status, waits (bounded) for its own MMAs, frees its
// tensor memory and returns.
#include "hy_kernels.cuh"
#include "hy_tc.cuh"

#include <algorithm>

namespace hy {
namespace k {

namespace {

// warps 0-7 build G, warps 8-11 build W chunks, warp 12 issues the MMAs
constexpr int kTcThreads = 416;
constexpr int kGThreadsTc = 256;
constexpr int kAWarps = 4;
constexpr int kIssueWarp = 12;
constexpr int kTcN = 128;          // columns per tile (MMA N)
constexpr int kTcM = 64;           // MMA M (single-excitation slots, zero padded)
constexpr int kTcKc = 32;          // types per chunk (two values of r)
constexpr int kTcK = 256;          // padded types (16 r x 16 s)
constexpr uint32_t kTmemCols = 128;
constexpr uint32_t kSbo = (kTcKc / 4) * 128;    // 8 rows (A) / columns (B) of a chunk
constexpr int kWRow = kTcK + 4;                           // padded row: 8 rows hit 32 banks
constexpr size_t kWBytes = size_t(kTcM) * kWRow * 4;       // W_J in FP32, 65 KB
constexpr size_t kABytes = size_t(kTcM) * kTcKc * 4;       // one A chunk, 8 KB
constexpr size_t kBBytes = size_t(kTcN) * kTcKc * 4;       // one G chunk, 16 KB
constexpr size_t kStage = 2 * kABytes + 2 * kBBytes;       // hi, lo of both

// kind::tf32, FP32 accumulate, K-major A and B, M = 64, N = 128
constexpr uint32_t kIdesc = (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(kTcN >> 3) << 17) |
                            (uint32_t(kTcM >> 4) << 24);

__device__ __forceinline__ void mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
                 ::"r"(tmem), "l"(a), "l"(b), "r"(kIdesc), "r"(acc));
}

__device__ __forceinline__ void commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(saddr(bar)) : "memory");
}

// bounded wait for the phase with parity `par` of an mbarrier: at most
// `limit` polls
__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t par, long long limit)
{
    uint32_t done = 0;
    for (long long it = 0; it < limit; ++it) {
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     "selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(saddr(bar)), "r"(par) : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_ld32(uint32_t addr, float *v)
{
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
                   "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
                   "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace

size_t cpl_tc_smem(int64_t Nb)
{
    // W_J | 2 stages | Wd [256] | diag partials [2][128] | 2 mbarriers +
    // tensor-memory slot | psi row J
    return kWBytes + 2 * kStage + kTcK * 4 + 2 * kTcN * 4 + 64 + size_t((Nb + 3) / 4 * 16);
}

// issue = 0 is a test mode: nothing is multiplied or committed, so every
// stage barrier stays pending and the builders' bounded waits run out (the
// kernel then reports a timeout in *status and returns; no MMA is in flight)
__global__ void __launch_bounds__(kTcThreads, 1)
k_cpl_tc(CplDenseArgs a, int *status, long long spin_limit, int issue)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    float *Wf = reinterpret_cast<float *>(sm);                  // [64][kWRow]
    unsigned char *stg = sm + kWBytes;                          // stage s at s * kStage
    float *Wd = reinterpret_cast<float *>(stg + 2 * kStage);
    float *dpart = Wd + kTcK;                                   // [2][kTcN]
    uint64_t *bar = reinterpret_cast<uint64_t *>(dpart + 2 * kTcN);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 2);
    float *prow = reinterpret_cast<float *>(bar + 8);           // psi[J][0 .. Nb)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, nn = n * n, nexa = a.nexa;
    const int free_b = n - __popc(a.bstr[0]);                 // empty orbitals of a beta string
    const int nch = (n + 1) / 2;                              // chunks of two r values
    const int64_t Nb = a.Nb;
    const int slots = nexa + 1;

    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&bar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&bar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(saddr(tslot)), "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    uint32_t issued0 = 0, issued1 = 0;   // commits made to each stage's barrier
    uint32_t waited0 = 0, waited1 = 0;   // commits already waited for
    bool ok = true;
    // wait until every commit made to a stage so far has completed
    auto drain = [&](uint64_t *b, uint32_t &waited, uint32_t issued) {
        while (ok && waited < issued) {
            if (!wait_bar(b, waited & 1u, spin_limit)) {
                ok = false;             // this commit is still out: waited for at the end
                atomicExch(status, 1);
                break;
            }
            ++waited;
        }
    };
    const bool gb = tid < kGThreadsTc;                        // a G builder
    const int col = tid & (kTcN - 1), half = (tid >> 7) & 1;  // 2 G builders per column

    for (int64_t jj = blockIdx.x; jj < a.nJ && ok; jj += gridDim.x) {
        const int64_t J = a.jlist ? int64_t(a.jlist[jj]) : jj;
        // W_J in FP32 for the 64 MMA rows, Wd_J for the diagonal slot and
        // psi's row J.  The previous J's MMAs have all been waited for.
        const uint32_t jm = a.astr[J];
        for (int idx = tid; idx < kTcM * kTcK; idx += blockDim.x) {
            const int m = idx / kTcK, tp = idx % kTcK;
            const int r = tp >> 4, s = tp & 15;
            float v = 0.0f;
            if (m < nexa && r < n && s < n) {
                const uint32_t u = a.aex[J * nexa + m];
                const int pj = (u >> 16) & 15, qj = (u >> 20) & 15;
                v = a.V[size_t(qj * n + pj) * nn + r * n + s];
                if (u >> 31) v = -v;
            }
            Wf[m * kWRow + tp] = v;
        }
        for (int tp = tid; tp < kTcK; tp += blockDim.x) {
            const int r = tp >> 4, s = tp & 15;
            float v = 0.0f;
            if (r < n && s < n)
                for (uint32_t mm = jm; mm; mm &= mm - 1) {
                    const int p = __ffs(mm) - 1;
                    v += a.V[size_t(p * n + p) * nn + r * n + s];
                }
            Wd[tp] = v;
        }
        const float *src = a.psi + J * Nb;
        for (int64_t i = tid; i < Nb; i += blockDim.x) prow[i] = __ldg(src + i);
        __syncthreads();
        for (int64_t b0 = 0; b0 < Nb && ok; b0 += kTcN) {
            const int64_t b = b0 + col;
            const bool live = gb && b < Nb;
            const uint32_t bm = live ? a.bstr[b] : 0u;
            float dsum = 0.0f;
            bool first = true;
            // beta excitation entries of this thread's r for chunk c, loaded
            // one chunk ahead: u[s] is the entry of (r created in b', s empty
            // in b') -- entry f0 + (empty orbitals below s) of b', since a
            // string lists its excitations by created orbital, then by empty
            // orbital, ascending -- or 0 (a packed entry is never 0: p != q)
            uint32_t un[16];
            auto load_entries = [&](int c, uint32_t *u) {
                const int r = 2 * c + half;
                const bool has = live && r < n && ((bm >> r) & 1u);
                const int f0 = has ? __popc(bm & ((1u << r) - 1u)) * free_b : 0;
#pragma unroll
                for (int s = 0; s < 16; ++s) {
                    const bool emp = has && s < n && !((bm >> s) & 1u);
                    const int q = s - __popc(bm & ((1u << s) - 1u));
                    u[s] = emp ? __ldg(a.bexT + size_t(f0 + q) * Nb + b) : 0u;
                }
            };
            load_entries(0, un);
            for (int c = 0; c < nch && ok; ++c) {
                const int st = c & 1;
                if (st == 0) drain(&bar[0], waited0, issued0);   // the MMAs that last read
                else drain(&bar[1], waited1, issued1);           // this stage
                uint32_t u[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) u[q] = un[q];
                if (c + 1 < nch) load_entries(c + 1, un);
                // this thread's 16 types: r = 2c + half, s = 0..15
                const int r = 2 * c + half;
                float g[16];
#pragma unroll
                for (int s = 0; s < 16; ++s) g[s] = 0.0f;
                if (live && r < n && ((bm >> r) & 1u)) {
                    const float diag = prow[b];           // the diagonal pair (r, r)
#pragma unroll
                    for (int s = 0; s < 16; ++s) {
                        float v = 0.0f;
                        if (u[s]) {
                            const float pv = prow[u[s] & 0xFFFFu];
                            v = (u[s] >> 31) ? -pv : pv;
                        } else if (s == r) {
                            v = diag;
                        }
                        g[s] = v;
                        dsum = fmaf(Wd[r * 16 + s], v, dsum);
                    }
                }
                unsigned char *Ah = stg + st * kStage, *Al = Ah + kABytes;
                unsigned char *Bh = Al + kABytes, *Bl = Bh + kBBytes;
                if (gb) {
#pragma unroll
                    for (int s4 = 0; s4 < 4; ++s4) {
                        float4 h, l;
                        split(g[4 * s4 + 0], h.x, l.x);
                        split(g[4 * s4 + 1], h.y, l.y);
                        split(g[4 * s4 + 2], h.z, l.z);
                        split(g[4 * s4 + 3], h.w, l.w);
                        const uint32_t off = kmaj(col, half * 16 + 4 * s4, kSbo);
                        *reinterpret_cast<float4 *>(Bh + off) = h;
                        *reinterpret_cast<float4 *>(Bl + off) = l;
                    }
                } else if (warp < kIssueWarp) {
                    // this chunk's 64 x 32 block of W_J, split: a warp writes
                    // one whole 8 x 4 core matrix (128 contiguous bytes) per step
                    const int w4 = warp - kGThreadsTc / 32;
#pragma unroll
                    for (int e = 0; e < (kTcM * kTcKc) / (32 * kAWarps); ++e) {
                        const int core = w4 + e * kAWarps;                 // 0 .. 63
                        const int m = (core >> 3) * 8 + (lane >> 2);       // 8 cores along K per row group
                        const int k = (core & 7) * 4 + (lane & 3);
                        float hi, lo;
                        split(Wf[m * kWRow + c * kTcKc + k], hi, lo);
                        const uint32_t off = uint32_t(core) * 128u + uint32_t(lane) * 4u;
                        *reinterpret_cast<float *>(Ah + off) = hi;
                        *reinterpret_cast<float *>(Al + off) = lo;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                ok = __syncthreads_and(ok) != 0;      // block-uniform from here
                if (!ok) break;
                // the issuing warp builds nothing: its wait for the tensor
                // cores to accept the MMAs stays off the builders' path
                if (warp == kIssueWarp && lane == 0 && issue) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t ah = saddr(Ah), al = saddr(Al), bh = saddr(Bh), bl = saddr(Bl);
#pragma unroll
                    for (int ks = 0; ks < kTcKc / 8; ++ks) {
                        const uint32_t ko = uint32_t(ks) * 256u;
                        mma(tmem, sdesc(ah + ko, kSbo), sdesc(bh + ko, kSbo), first ? 0u : 1u);
                        mma(tmem, sdesc(ah + ko, kSbo), sdesc(bl + ko, kSbo), 1u);
                        mma(tmem, sdesc(al + ko, kSbo), sdesc(bh + ko, kSbo), 1u);
                        first = false;
                    }
                    commit(&bar[st]);
                }
                first = false;
                if (st == 0) ++issued0; else ++issued1;
            }
            if (gb) dpart[half * kTcN + col] = dsum;
            drain(&bar[0], waited0, issued0);
            drain(&bar[1], waited1, issued1);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            ok = __syncthreads_and(ok) != 0;
            if (!ok) break;
            // epilogue: rows 16w .. 16w + 15 sit in lanes 0..15 of sub-partition w
            if (warp < 4) {
                const int m = warp * 16 + lane;
                const uint32_t rowaddr = tmem + (uint32_t(warp * 32) << 16);
#pragma unroll
                for (int cb = 0; cb < kTcN / 32; ++cb) {
                    float v[32];
                    tmem_ld32(rowaddr + uint32_t(cb * 32), v);
                    if (lane < 16 && m < nexa) {
                        float *dst = a.T + (J * slots + m) * a.Nbp + b0 + cb * 32;
#pragma unroll
                        for (int i = 0; i < 32; i += 4)
                            if (b0 + cb * 32 + i + 3 < Nb)
                                *reinterpret_cast<float4 *>(dst + i) =
                                    make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                            else
                                for (int q = 0; q < 4; ++q)
                                    if (b0 + cb * 32 + i + q < Nb) dst[i + q] = v[i + q];
                    }
                }
            } else if (tid < 128 + kTcN) {
                const int cc = tid - 128;
                if (b0 + cc < Nb)
                    a.T[(J * slots + nexa) * a.Nbp + b0 + cc] = dpart[cc] + dpart[kTcN + cc];
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();
        }
    }
    // on a timeout, give the MMAs still in flight a bounded chance to finish, whatever
    // the limit of the other waits (test mode: nothing was issued, nothing will come)
    if (!ok && issue) {
        const long long drain_limit = spin_limit > (1ll << 24) ? spin_limit : 1ll << 24;
        while (waited0 < issued0) wait_bar(&bar[0], (waited0++) & 1u, drain_limit);
        while (waited1 < issued1) wait_bar(&bar[1], (waited1++) & 1u, drain_limit);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem), "r"(kTmemCols));
}

// ---------------------------------------------------------------------------
// The same contraction for wider beta spaces (k_cpl_tcw): W_J stays in shared
// memory for all column tiles of J, already split (n x 8 KB), an operand stage
// is the 16 types of one r, and the roles run apart, joined by mbarriers only:
//   * two groups of eight warps build alternate stages.  A thread owns a column
//     and eight s; its eight partners' places and signs are one 16-byte load
//     from a table made when the Hamiltonian is (cpl_entries: 16 bits each,
//     absent pairs point at a zero behind psi's row), so a stage is eight
//     gathers, splits and four 16-byte stores;
//   * one warp issues the MMAs of a stage (six) and commits it;
//   * four warps read finished accumulators (two in tensor memory, used in turn)
//     while the next tile is multiplied.
// The diagonal slot is one more row of W_J where 64 rows have room for it (all but 8
// electrons in 16 orbitals: DIAG, summed in FP32 by the builders).  W_J is rounded
// when it is split and the small products go first (hy_same.cu): the error of the
// float H|psi> against double, 11 orbitals, 6+5, 2.2e-7 -> 1.8e-7 (relative, l2).
// r that no column of a tile holds is skipped.  k_cpl_tc's block-wide barrier
// per chunk left it at 3,600 clocks per 32 types, 768 of them tensor time.
// Bound by the hand-over of stages (build, fence, arrive, issue, commit): with
// gathers, stores or MMAs left out one at a time it loses 0-13 %, with all of them
// half.  Stages of 8 types (twice the hand-overs) cost 30 %, four groups of four
// warps, a column's 16 types to a thread, 6-20 %; an issuing warp that meets and
// elects anew at each stage 8 %.  Measured, whole float H|psi> with the same-spin parts
// by rows: 16 orbitals, 8+8 (64 of 129 ms left of the coupling's) 205 -> 141 ms; 13
// orbitals, 7+6: 2,989 -> 1,583 us; 11 orbitals, 6+5: 285 -> 162 us; also with few
// strings: 12 orbitals, 2+2: 62.6 -> 56 us.  The diagonal's sums by their own loop,
// all loads at once, gave 11 orbitals 5 % and 13 orbitals 2 % of that.
// ---------------------------------------------------------------------------
namespace {

constexpr int kTwBuilders = 512, kTwThreads = kTwBuilders + 128 + 32;
constexpr int kTwIssueWarp = 20;
constexpr uint32_t kTwSbo = 512;                        // 16 types of 8 rows
constexpr size_t kTwA = size_t(kTcM) * 16 * 4;          // one r of W_J, hi or lo: 4 KB
constexpr size_t kTwB = size_t(kTcN) * 16 * 4;          // one r of a tile, hi or lo: 8 KB
constexpr int kTwMaxStages = 4;

// small block of barriers and flags at the front of shared memory
struct TwCtl {
    uint64_t full[kTwMaxStages], empty[kTwMaxStages], acc_full[2], acc_empty[2], fin;
    uint32_t tmem;
    int dead;                                           // a wait ran out somewhere
};

__device__ __forceinline__ void arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}

// whether the phase with parity `par` has completed: a plain test, as
// try_wait's suspended thread wakes late
__device__ __forceinline__ bool test_bar(uint64_t *bar, uint32_t par)
{
    uint32_t done;
    asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 "selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(saddr(bar)), "r"(par) : "memory");
    return done != 0;
}

// bounded wait that also ends when another role has given up
__device__ __forceinline__ bool tw_wait(TwCtl *c, uint64_t *bar, uint32_t par, long long limit,
                                        int *status)
{
    for (long long it = 0; it < limit; ++it) {
        if (test_bar(bar, par)) return true;
        if (*reinterpret_cast<volatile int *>(&c->dead)) return false;
    }
    *reinterpret_cast<volatile int *>(&c->dead) = 1;
    atomicExch(status, 1);
    return false;
}

// the same for a whole warp: one lane polls (32 lanes of 20 warps polling slow
// the barrier unit down for everyone)
__device__ __forceinline__ bool tw_wait_warp(TwCtl *c, uint64_t *bar, uint32_t par, long long limit,
                                             int *status)
{
    int ok = 1;
    if ((threadIdx.x & 31) == 0) ok = tw_wait(c, bar, par, limit, status);
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// barrier of the builders (all of them, always); whether v holds in every one
__device__ __forceinline__ bool builders_and(bool v)
{
    int r;
    __syncwarp();
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.s32 p, %1, 0;\n"
                 "bar.red.and.pred q, 1, %2, p;\nselp.s32 %0, 1, 0, q;\n}"
                 : "=r"(r) : "r"(int(v)), "n"(kTwBuilders) : "memory");
    return r != 0;
}

}  // namespace

size_t cpl_tcw_smem(int64_t Nb, int n, int stages)
{
    // control | W_J hi, lo | stages | Wd | diagonal partials [2][4][128] | psi row and a zero
    return 256 + size_t(n) * 2 * kTwA + stages * 2 * kTwB + 256 * 4 + 2 * 4 * kTcN * 4 +
           size_t((Nb + 1 + 3) / 4 * 16);
}

template <bool DIAG>
__global__ void __launch_bounds__(kTwThreads, 1)
k_cpl_tcw(CplDenseArgs a, int nst, int *status, long long spin_limit, int issue)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    TwCtl *ctl = reinterpret_cast<TwCtl *>(sm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, nn = n * n, nexa = a.nexa, slots = nexa + 1;
    const int Nb = int(a.Nb), tiles = (Nb + kTcN - 1) / kTcN;
    unsigned char *Wa = sm + 256;                           // [n][hi, lo][64 x 16]
    unsigned char *stg = Wa + size_t(n) * 2 * kTwA;         // [nst][hi, lo][128 x 16]
    float *Wd = reinterpret_cast<float *>(stg + size_t(nst) * 2 * kTwB);  // [16][16]
    float *dpart = Wd + 256;                                // [2][4][128]
    float *prow = dpart + 2 * 4 * kTcN;                     // [Nb + 1]

    if (tid == 0) {
        auto init = [](uint64_t *b, int cnt) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(cnt));
        };
        for (int i = 0; i < nst; ++i) {
            init(&ctl->full[i], 8);
            init(&ctl->empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            init(&ctl->acc_full[i], 1);
            init(&ctl->acc_empty[i], 4);
        }
        init(&ctl->fin, 1);
        ctl->dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(saddr(&ctl->tmem)), "r"(2 * kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = ctl->tmem;

    if (tid < kTwBuilders) {
        // ---- builders ----------------------------------------------------
        // two groups of eight warps take the r in turn; r number i goes to stage
        // i % nst, a thread fills half of a column's types
        const int par = warp >> 3, half = (warp >> 2) & 1, col = tid & (kTcN - 1);
        const uint32_t none = uint32_t(Nb * 4) | (uint32_t(Nb * 4) << 16);
        const uint32_t off = kmaj(col, half * 8, kTwSbo);
        const unsigned char *row = reinterpret_cast<const unsigned char *>(prow);
        uint32_t it = 0;            // r of all tiles so far
        int slot = par, use = 0;    // where this group's next r goes, how often used
        uint32_t tile_no = 0;
        bool ok = true;
        // this group's r of a tile whose first r has number i: every second set bit
        auto own = [&](uint32_t tm, uint32_t i) {
            return ((i ^ uint32_t(par)) & 1u) ? tm & (tm - 1) : tm;
        };
        auto load = [&](int tile, uint32_t m, int r) {
            return ((m >> r) & 1u)
                ? __ldg(reinterpret_cast<const uint4 *>(a.entries) +
                        ((size_t(tile) * a.nocc + __popc(m & ((1u << r) - 1u))) * kTcN + col) * 2 + half)
                : make_uint4(none, none, none, none);
        };
        auto mask = [&](int tile) {
            const int b = tile * kTcN + col;
            return b < Nb ? __ldg(a.bstr + b) : 0u;
        };
        // tables run ahead across tiles and J: e the entry of the next own stage,
        // bm the column's string in this tile, bn in the next
        uint32_t bm = mask(0), bn = mask(tiles > 1 ? 1 : 0), tm = __ldg(a.tmask);
        uint4 e = make_uint4(none, none, none, none);
        if (own(tm, 0)) e = load(0, bm, __ffs(own(tm, 0)) - 1);
        for (int64_t jj = blockIdx.x; jj < a.nJ; jj += gridDim.x) {
            const int64_t J = a.jlist ? int64_t(a.jlist[jj]) : jj;
            // the previous J: its row is read by all builders, its W_J by the MMAs
            // (the last of them done, all are).  A builder whose wait ran out comes
            // here too: the block's builders stop together
            if (it && ok) {
                const uint32_t last = it - 1;
                ok = tw_wait_warp(ctl, &ctl->empty[last % nst], (last / nst) & 1u, spin_limit, status);
            }
            ok = builders_and(ok);
            if (!ok) break;
            const float *src = a.psi + J * Nb;
            for (int i = tid; i < Nb; i += kTwBuilders) prow[i] = __ldg(src + i);
            if (tid == 0) prow[Nb] = 0.0f;
            const uint32_t jm = a.astr[J];
            auto diag_coef = [&](int r, int s) {         // sum_{p in J} V[pp][rs]
                float v = 0.0f;
                if (r < n && s < n) {
                    const float *V = a.V + r * n + s;        // the loads go out together
#pragma unroll
                    for (int p = 0; p < 16; ++p)
                        if ((jm >> p) & 1u) v += __ldg(V + size_t(p * n + p) * nn);
                }
                return v;
            };
            // a thread's m and k4 are the same for all its r
            const uint32_t u = (tid & 63) < nexa ? __ldg(a.aex + J * nexa + (tid & 63)) : 0u;
#pragma unroll 4
            for (int i = tid; i < n * kTcM * 4; i += kTwBuilders) {
                const int m = i & 63, k4 = (i >> 6) & 3, r = i >> 8;
                float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (m < nexa) {
                    const int pj = (u >> 16) & 15, qj = (u >> 20) & 15;
                    const float *V = a.V + size_t(qj * n + pj) * nn + r * n;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (4 * k4 + q < n) v[q] = (u >> 31) ? -__ldg(V + 4 * k4 + q) : __ldg(V + 4 * k4 + q);
                } else if (!DIAG && m == nexa) {
                    continue;
                }
                float4 h, l;
                split_rn(v[0], h.x, l.x);
                split_rn(v[1], h.y, l.y);
                split_rn(v[2], h.z, l.z);
                split_rn(v[3], h.w, l.w);
                unsigned char *dst = Wa + size_t(r) * 2 * kTwA + kmaj(m, 4 * k4, kTwSbo);
                *reinterpret_cast<float4 *>(dst) = h;
                *reinterpret_cast<float4 *>(dst + kTwA) = l;
            }
            for (int i = tid; i < n * 16; i += kTwBuilders) {
                const int r = i >> 4, sp = i & 15;
                const float v = diag_coef(r, sp);
                if (DIAG) {
                    Wd[i] = v;
                } else {                     // one more row of W_J
                    float h, l;
                    split_rn(v, h, l);
                    unsigned char *dst = Wa + size_t(r) * 2 * kTwA + kmaj(nexa, sp, kTwSbo);
                    *reinterpret_cast<float *>(dst) = h;
                    *reinterpret_cast<float *>(dst + kTwA) = l;
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            builders_and(true);
            for (int tile = 0; tile < tiles && ok; ++tile, ++tile_no) {
                const int next = tile + 1 < tiles ? tile + 1 : 0;
                const uint32_t tn = __ldg(a.tmask + next), stages = __popc(tm);
                const uint32_t bnn = mask(next + 1 < tiles ? next + 1 : 0);
                uint32_t left = own(tm, it);
                float dsum = 0.0f;
                while (left && ok) {
                    const int r = __ffs(left) - 1;
                    left &= left - 1;
                    if (left) left &= left - 1;
                    // the next own stage's entries, here or in the next tile
                    uint4 nx = e;
                    if (left) {
                        nx = load(tile, bm, __ffs(left) - 1);
                    } else {
                        const uint32_t on = own(tn, it + stages);
                        if (on) nx = load(next, bn, __ffs(on) - 1);
                    }
                    const uint32_t w[4] = {e.x, e.y, e.z, e.w};
                    float h[8], l[8];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        // four times the place in the row, and the sign
                        const float x = *reinterpret_cast<const float *>(row + (w[q] & 0xFFFCu));
                        const float y = *reinterpret_cast<const float *>(row + ((w[q] >> 16) & 0xFFFCu));
                        const float xs = __uint_as_float(__float_as_uint(x) ^ (w[q] << 31));
                        const float ys = __uint_as_float(__float_as_uint(y) ^ ((w[q] << 15) & 0x80000000u));
                        if (DIAG) {
                            const float2 c = *reinterpret_cast<const float2 *>(Wd + r * 16 + half * 8 + 2 * q);
                            dsum = fmaf(c.x, xs, dsum);
                            dsum = fmaf(c.y, ys, dsum);
                        }
                        split(xs, h[2 * q], l[2 * q]);
                        split(ys, h[2 * q + 1], l[2 * q + 1]);
                    }
                    // the MMAs that read this stage last
                    if (use)
                        ok = tw_wait_warp(ctl, &ctl->empty[slot], (use - 1) & 1u, spin_limit, status);
                    if (!ok) break;
                    unsigned char *Bh = stg + size_t(slot) * 2 * kTwB, *Bl = Bh + kTwB;
                    *reinterpret_cast<float4 *>(Bh + off) = make_float4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<float4 *>(Bh + off + 128) = make_float4(h[4], h[5], h[6], h[7]);
                    *reinterpret_cast<float4 *>(Bl + off) = make_float4(l[0], l[1], l[2], l[3]);
                    *reinterpret_cast<float4 *>(Bl + off + 128) = make_float4(l[4], l[5], l[6], l[7]);
                    if (DIAG && !left) {
                        // the tile's last stage of this group: its part of the
                        // diagonal slot, once that tile's place has been read
                        const uint32_t buf = tile_no & 1u, used = tile_no >> 1;
                        if (used)
                            ok = tw_wait_warp(ctl, &ctl->acc_empty[buf], (used - 1) & 1u, spin_limit,
                                      status);
                        if (!ok) break;
                        dpart[(buf * 4 + par * 2 + half) * kTcN + col] = dsum;
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) arrive(&ctl->full[slot]);
                    for (slot += 2; slot >= nst; slot -= nst) ++use;
                    e = nx;
                }
                // a tile without a stage of this group leaves e for the one after it
                if (!own(tm, it)) {
                    const uint32_t on = own(tn, it + stages);
                    if (on) e = load(next, bn, __ffs(on) - 1);
                }
                it += stages;
                bm = bn;
                bn = bnn;
                tm = tn;
            }
        }
    } else if (warp == kTwIssueWarp) {
        // ---- MMA issue -----------------------------------------------------
        // the whole warp walks the stages (uniform registers hold the operand
        // descriptors), one lane, elected once, issues.  Nothing in the loops needs the
        // lanes together: a limit that runs out between two lanes' polls parts them.
        // One lane polling for all costs 5 % (16 orbitals) to 12 % of the sweep, electing
        // and meeting again at each stage 3 to 10 %
        const bool lead = elect_one();
        uint32_t tile_no = 0;
        int slot = 0, use = 0;
        bool ok = true;
        const uint32_t wa = saddr(Wa), sa = saddr(stg);
        for (int64_t jj = blockIdx.x; jj < a.nJ && ok; jj += gridDim.x)
            for (int tile = 0; tile < tiles && ok; ++tile, ++tile_no) {
                const uint32_t buf = tile_no & 1u, used = tile_no >> 1;
                if (used)
                    ok = tw_wait(ctl, &ctl->acc_empty[buf], (used - 1) & 1u, spin_limit, status);
                const uint32_t d = tmem + buf * kTmemCols;
                uint32_t acc = 0;
                for (uint32_t left = __ldg(a.tmask + tile); left && ok; left &= left - 1) {
                    ok = tw_wait(ctl, &ctl->full[slot], use & 1u, spin_limit, status);
                    if (ok && issue) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t ah = wa + uint32_t(__ffs(left) - 1) * uint32_t(2 * kTwA);
                        const uint32_t bh = sa + uint32_t(slot) * uint32_t(2 * kTwB);
                        if (lead) {
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks) {      // the small products first
                                const uint64_t da = sdesc(ah + ks * 256u, kTwSbo);
                                const uint64_t db = sdesc(bh + ks * 256u, kTwSbo);
                                mma(d, da, db + (kTwB >> 4), ks ? 1u : acc);
                                mma(d, da + (kTwA >> 4), db, 1u);
                            }
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks)
                                mma(d, sdesc(ah + ks * 256u, kTwSbo), sdesc(bh + ks * 256u, kTwSbo), 1u);
                            commit(&ctl->empty[slot]);
                        }
                        acc = 1u;
                    }
                    if (++slot == nst) {
                        slot = 0;
                        ++use;
                    }
                }
                if (ok && issue && lead) commit(&ctl->acc_full[buf]);
            }
        // every MMA issued is done before the tensor memory goes back
        if (issue) {
            if (lead) commit(&ctl->fin);
            __syncwarp();
            wait_bar(&ctl->fin, 0, spin_limit > (1ll << 24) ? spin_limit : 1ll << 24);
        }
        __syncwarp();
    } else {
        // ---- epilogue --------------------------------------------------------
        const int ew = warp - kTwBuilders / 32;        // sub-partition: warp % 4
        const int rows = DIAG ? nexa : slots;
        uint32_t it = 0, tile_no = 0;
        bool ok = true;
        for (int64_t jj = blockIdx.x; jj < a.nJ && ok; jj += gridDim.x) {
            const int64_t J = a.jlist ? int64_t(a.jlist[jj]) : jj;
            for (int tile = 0; tile < tiles && ok; ++tile, ++tile_no) {
                const uint32_t buf = tile_no & 1u, stages = __popc(__ldg(a.tmask + tile));
                const uint32_t g1 = (it & 1u) * 2;      // parts of the first stage's group
                it += stages;
                ok = tw_wait_warp(ctl, &ctl->acc_full[buf], (tile_no >> 1) & 1u, spin_limit, status);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int b0 = tile * kTcN, m = ew * 16 + lane;
                const uint32_t rowaddr = tmem + buf * kTmemCols + (uint32_t(ew * 32) << 16);
                float *dst = a.T + (J * slots + m) * a.Nbp + b0;
#pragma unroll
                for (int cb = 0; cb < kTcN / 32; ++cb) {
                    float v[32];
                    tmem_ld32(rowaddr + uint32_t(cb * 32), v);
                    if (lane < 16 && m < rows) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4)
                            if (b0 + cb * 32 + i < int(a.Nbp))      // Nbp: Nb rounded up to 64
                                *reinterpret_cast<float4 *>(dst + cb * 32 + i) =
                                    make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                    }
                }
                // the diagonal slot: 32 columns a warp; a group without a stage in
                // this tile (one r only) has left nothing
                const int c = ew * 32 + lane;
                if (DIAG && b0 + c < Nb) {
                    const float *d = dpart + buf * 4 * kTcN + c;
                    const float s = stages >= 2 ? (d[0] + d[kTcN]) + (d[2 * kTcN] + d[3 * kTcN])
                                                : d[g1 * kTcN] + d[(g1 + 1) * kTcN];
                    a.T[(J * slots + nexa) * a.Nbp + b0 + c] = s;
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive(&ctl->acc_empty[buf]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem), "r"(2 * kTmemCols));
}

// entries and the r each tile holds (k_cpl_tcw), from the packed beta
// excitations: entry (tile, i, column, s) belongs to the i-th occupied orbital r
// of the column's string: its partner with r -> s (s empty), itself (s = r), or
// the zero behind psi's row; four times the place in the row, plus the sign
__global__ void __launch_bounds__(256)
k_cpl_entries(const uint32_t *__restrict__ bstr, const uint32_t *__restrict__ bexT, int Nb, int n,
              int nocc, int tiles, uint16_t *__restrict__ entries, uint32_t *__restrict__ tmask)
{
    const int64_t total = int64_t(tiles) * nocc * kTcN * 16;
    for (int64_t id = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; id < total;
         id += int64_t(gridDim.x) * blockDim.x) {
        const int s = int(id & 15), col = int(id >> 4) & (kTcN - 1);
        const int ti = int(id / (16 * kTcN)), i = ti % nocc, tile = ti / nocc, b = tile * kTcN + col;
        uint32_t e = uint32_t(Nb) * 4;
        if (b < Nb) {
            const uint32_t m = bstr[b];
            uint32_t mm = m;
            for (int k = 0; k < i; ++k) mm &= mm - 1;
            const int r = __ffs(mm) - 1;
            if (s == r) {
                e = uint32_t(b) * 4;
            } else if (s < n && !((m >> s) & 1u)) {
                const int f = i * (n - nocc) + s - __popc(m & ((1u << s) - 1u));
                const uint32_t u = bexT[size_t(f) * Nb + b];
                e = (u & 0x3FFFu) * 4 | (u >> 31);
            }
            if (s == 0 && i == 0) atomicOr(tmask + tile, m);
        }
        entries[id] = uint16_t(e);
    }
}

size_t cpl_entries_count(int64_t Nb, int nocc)
{
    return size_t((Nb + kTcN - 1) / kTcN) * nocc * kTcN * 16;
}

// tmask: (Nb + 127) / 128 words, zeroed
cudaError_t cpl_entries(const uint32_t *bstr, const uint32_t *bexT, int64_t Nb, int n, int nocc,
                        uint16_t *entries, uint32_t *tmask, int num_sms, cudaStream_t st)
{
    const int tiles = int((Nb + kTcN - 1) / kTcN);
    k_cpl_entries<<<unsigned(8 * num_sms), 256, 0, st>>>(bstr, bexT, int(Nb), n, nocc, tiles, entries,
                                                        tmask);
    hy::count_launch();
    return cudaGetLastError();
}

cudaError_t coupling_tc(const CplDenseArgs &a, int *status, long long spin_limit, int issue,
                        int num_sms, cudaStream_t st)
{
    if (a.Na == 0 || a.Nb == 0) return cudaSuccess;
    if (a.nexa > kTcM || a.n > 16) return cudaErrorInvalidValue;
    if (a.entries) {
        int nst = kTwMaxStages;
        while (nst > 2 && cpl_tcw_smem(a.Nb, a.n, nst) > 227 * 1024) --nst;
        const size_t smem = cpl_tcw_smem(a.Nb, a.n, nst);
        auto run = [&](auto *kernel) {
            const cudaError_t e = allow_smem(kernel, smem);
            if (e != cudaSuccess || a.nJ == 0) return e;
            kernel<<<unsigned(std::min<int64_t>(num_sms, a.nJ)), kTwThreads, smem, st>>>(
                a, nst, status, spin_limit, issue);
            hy::count_launch();
            return cudaGetLastError();
        };
        return a.nexa < kTcM ? run(k_cpl_tcw<false>) : run(k_cpl_tcw<true>);
    }
    const size_t smem = cpl_tc_smem(a.Nb);
    cudaError_t err = allow_smem(k_cpl_tc, smem);
    if (err != cudaSuccess) return err;
    if (a.nJ == 0) return cudaSuccess;
    int64_t grid = num_sms;
    if (grid > a.nJ) grid = a.nJ;
    k_cpl_tc<<<unsigned(grid), kTcThreads, smem, st>>>(a, status, spin_limit, issue);
    hy::count_launch();
    return cudaGetLastError();
}

}  // namespace k
}  // namespace hy
