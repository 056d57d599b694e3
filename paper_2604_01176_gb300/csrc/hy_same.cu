// hy_same.cu -- same-spin part of the float H|psi> for wider spaces, on the
// fifth-generation tensor cores.
//
//   Y[r][c] = sum_J M[r][J] X[J][c],   Y row-major [N][ncols]
//
// M couples strings up to two excitations apart: 7-40 % of it is there, but in no
// blocks to speak of (16 orbitals, 8 electrons: 76 % of its 256 x 32 blocks hold
// something).  Row by row (k_spmm) every multiply-add takes its own four bytes
// of X through L1 and L2: 33 ms for 12,870 strings squared, 14 % of the FP32 rate.
// As a dense product with its empty blocks left out it has twelve times the
// multiply-adds, three TF32 products each (hi*hi, hi*lo, lo*hi; hy_cpl_tc.cu), and
// still ends sooner.
//
// Both factors lie in memory as MMA operands, hi and lo: M's off-diagonal part once
// per Hamiltonian, with its first float sweep (same_used, same_fill: 256 rows by 32 columns that hold anything),
// X per call (k_same_x, from either layout of psi, so the beta side needs no
// transposed copy).  A pair of CTAs (cta_group::2) multiplies 256 columns of X (its
// M side, so that a lane of tensor memory is a column and rows of Y are written
// whole) by 256 rows (N).  A stage is 32 J: two bulk copies of 32 KB into each CTA,
// twelve MMAs (1,536 clocks).  Splitting X on the way in instead, by eight warps, took
// 2,900 clocks a stage: its loads wait for lines of the little L1 that is left.
//   * warps 0-7 take finished accumulators out (two, each half of tensor memory,
//     in turn): the tensor cores cut sums off toward zero, so 64 J are added there
//     and the rest in FP32 registers.  Error of the float H|psi> against double, 14
//     orbitals, 7+7, with the same coupling: 3.3e-7 by rows (k_spmm), 3.2e-7 with 128
//     J, 2.7e-7 with 64, 2.6e-7 with 32 (5 % slower); hi not rounded to nearest, 128 J:
//     4.4e-7 (2.1e-7 with 64 J since the coupling rounds too, hy_cpl_tc.cu);
//   * warp 8 starts the copies;
//   * warp 9 issues the MMAs in the leading CTA and passes the other one's stages
//     on to it.
// The diagonal is large and needs no sum: Y starts as diag * X in FP32, and the sum
// is added to it once.
// Waits are bounded as in hy_cpl_tc.cu.
// A dense product multiplies amplitudes by zeros too: one that is not finite, or so
// large that its rounded half is not, would spoil rows that M does not couple to it.
// Packing X looks for such a one, and k_same_rows then does both sides over, row by
// row; else it ends at once (6 of 969 us at 13 orbitals, 7+5, with the looking).
// Measured: 12,870 strings squared 33.0 -> 12.3 ms a side (71 % of the MMA rate,
// the rest between stages: 128 KB of L2 reads a pair and 1,536 clocks), 1,716 360 ->
// 73 us; whole float H|psi>, 16 orbitals, 8+8, 140.5 -> 99.0 ms; 13 orbitals, 7+5, 1,389
// -> 974 us; 12 orbitals, 6+6, 490 -> 444 us.
#include "hy_kernels.cuh"
#include "hy_tc.cuh"

#include <algorithm>

namespace hy {
namespace k {

namespace {

constexpr int kSmRows = 256, kSmCols = 256, kSmK = 32;      // a pair's tile and a stage
constexpr int kSmStages = 3;
constexpr int kSmGroup = 2;                                 // stages per accumulator
constexpr int kSmSum = 256, kSmThreads = kSmSum + 64;
constexpr uint32_t kSmSbo = kSmK / 4 * 128;                 // 1024
constexpr uint32_t kSmOp = 128 * kSmK * 4;                  // hi or lo of 128 rows or columns, 16 KB
constexpr uint32_t kSmStage = 4 * kSmOp;                    // X hi, lo, M hi, lo
constexpr uint32_t kSmBlock = 2 * 2 * kSmOp;                // a pack's block: both CTAs

struct SmCtl {
    uint64_t full[kSmStages], pfull[kSmStages], empty[kSmStages];
    uint64_t acc_full[2], acc_empty[2], fin;
    uint32_t tmem;
    int dead;
};
constexpr size_t kSmBase = 1024;
constexpr long long kSmDrain = 1ll << 24;   // polls, whatever the limit of the other waits
static_assert(sizeof(SmCtl) <= kSmBase, "control block");
constexpr size_t kSmSmem = kSmBase + size_t(kSmStages) * kSmStage;

// kind::tf32, FP32 accumulate, K-major A and B, M = 256 over both CTAs, N = 256
constexpr uint32_t kSmIdesc = (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(kSmRows >> 3) << 17) |
                              (uint32_t(kSmCols >> 4) << 24);

__device__ __forceinline__ void mma2(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n}"
                 ::"r"(tmem), "l"(a), "l"(b), "r"(kSmIdesc), "r"(acc));
}

// arrives at this barrier of both CTAs when the MMAs issued so far are done
__device__ __forceinline__ void commit2(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster"
                 ".multicast::cluster.b64 [%0], %1;"
                 ::"r"(saddr(bar)), "h"(uint16_t(3)) : "memory");
}

// arrives at the leading CTA's barrier
__device__ __forceinline__ void arrive_leader(uint64_t *bar)
{
    asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %0, 0;\n"
                 "mbarrier.arrive.shared::cluster.b64 _, [a];\n}"
                 ::"r"(saddr(bar)) : "memory");
}

__device__ __forceinline__ bool sm_test(uint64_t *bar, uint32_t par)
{
    uint32_t done;
    asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 "selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(saddr(bar)), "r"(par) : "memory");
    return done != 0;
}

// bounded wait for what is in flight for sure
__device__ __forceinline__ void drain(uint64_t *bar, uint32_t par)
{
    for (long long it = 0; it < kSmDrain && !sm_test(bar, par); ++it) {}
}

// bounded wait that also ends when another role has given up
__device__ __forceinline__ bool sm_wait(SmCtl *c, uint64_t *bar, uint32_t par, long long limit,
                                        int *status)
{
    for (long long it = 0; it < limit; ++it) {
        if (sm_test(bar, par)) return true;
        if (*reinterpret_cast<volatile int *>(&c->dead)) return false;
    }
    *reinterpret_cast<volatile int *>(&c->dead) = 1;
    atomicExch(status, 1);
    return false;
}

__device__ __forceinline__ bool sm_wait_warp(SmCtl *c, uint64_t *bar, uint32_t par, long long limit,
                                             int *status)
{
    int ok = 1;
    if ((threadIdx.x & 31) == 0) ok = sm_wait(c, bar, par, limit, status);
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// tile number -> row block and column block: eight row blocks at a time, so that
// the pairs at work share both operands in L2
struct SmTile {
    int rb, cb;
};
__device__ __forceinline__ SmTile sm_tile(int t, int nrb, int ncb)
{
    const int per = 8 * ncb, g = t / per, in = t - g * per;
    const int rows = min(8, nrb - 8 * g);
    return SmTile{8 * g + in % rows, in / rows};
}

}  // namespace

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSmThreads, 1)
k_same(SameArgs a, int *status, long long spin_limit)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    SmCtl *ctl = reinterpret_cast<SmCtl *>(sm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int rb0 = int(a.row0 / kSmRows), nrb = int((a.row1 - 1) / kSmRows) + 1 - rb0;
    const int ncb = int((a.ncols + kSmCols - 1) / kSmCols);
    const int64_t nch = (a.N + kSmK - 1) / kSmK;
    const int ntile = nrb * ncb, first = int(blockIdx.x >> 1), step = int(gridDim.x >> 1);

    if (tid == 0) {
        auto init = [](uint64_t *b, int cnt) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(cnt));
        };
        for (int i = 0; i < kSmStages; ++i) {
            init(&ctl->full[i], 1);
            init(&ctl->pfull[i], 1);
            init(&ctl->empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            init(&ctl->acc_full[i], 1);
            init(&ctl->acc_empty[i], 16);
        }
        init(&ctl->fin, 1);
        ctl->dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(saddr(&ctl->tmem)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = ctl->tmem;

    if (warp < 8) {
        // ---- sums ----------------------------------------------------------
        const int half = warp >> 2;                     // 128 rows of the tile
        const uint32_t taddr = tmem + (uint32_t((warp & 3) * 32) << 16) + uint32_t(half * 128);
        uint32_t grp = 0;
        bool ok = true;
        for (int t = first; t < ntile && ok; t += step) {
            const SmTile tl = sm_tile(t, nrb, ncb);
            const int cb = 2 * tl.cb + int(rank), xcol = (warp & 3) * 32 + lane;
            const int64_t c = int64_t(cb) * 128 + xcol;
            const int64_t r0 = int64_t(rb0 + tl.rb) * kSmRows + half * 128;
            const int cnt = int(a.base[rb0 + tl.rb + 1] - a.base[rb0 + tl.rb]);
            const int jlo = int(max(int64_t(0), a.row0 - r0)), jhi = int(min(int64_t(128), a.row1 - r0));
            float *y = a.Y + (r0 - a.row0) * a.ncols + c;
            if (c < a.ncols) {
                const unsigned char *x = a.xpack + (size_t(cb) * nch + size_t(r0 / kSmK)) * 2 * kSmOp;
#pragma unroll 4
                for (int j4 = jlo & ~3; j4 < jhi; j4 += 4) {
                    const unsigned char *p = x + size_t(j4 / kSmK) * 2 * kSmOp + kmaj(xcol, j4 & (kSmK - 1), kSmSbo);
                    const float4 h = __ldg(reinterpret_cast<const float4 *>(p));
                    const float4 l = __ldg(reinterpret_cast<const float4 *>(p + kSmOp));
                    const float v[4] = {h.x + l.x, h.y + l.y, h.z + l.z, h.w + l.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (j4 + q >= jlo && j4 + q < jhi)
                            y[(j4 + q) * a.ncols] = __ldg(a.diag + r0 + j4 + q) * v[q];
                }
            }
            float acc[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.0f;
            for (int s = 0; s < cnt && ok; s += kSmGroup, ++grp) {
                const uint32_t buf = grp & 1u;
                ok = sm_wait_warp(ctl, &ctl->acc_full[buf], (grp >> 1) & 1u, spin_limit, status);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    uint32_t v[16];
                    tmem_ld16(taddr + buf * 256u + uint32_t(q * 16), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[16 * q + i] += __uint_as_float(v[i]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive_leader(&ctl->acc_empty[buf]);
            }
            if (c < a.ncols && cnt) {
                // one addition to the place this thread wrote above
#pragma unroll
                for (int j = 0; j < 128; ++j)
                    if (j >= jlo && j < jhi)
                        asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;"
                                     ::"l"(y + j * a.ncols), "f"(acc[j]) : "memory");
            }
        }
    } else if (warp == 8) {
        // ---- copies --------------------------------------------------------
        if (lane == 0) {
            int slot = 0, use = 0;
            uint32_t issued = 0;
            bool ok = true;
            for (int t = first; t < ntile && ok; t += step) {
                const SmTile tl = sm_tile(t, nrb, ncb);
                const int64_t b0 = a.base[rb0 + tl.rb];
                const int cnt = int(a.base[rb0 + tl.rb + 1] - b0);
                const unsigned char *x = a.xpack + size_t(2 * tl.cb + int(rank)) * nch * 2 * kSmOp;
                const unsigned char *m = a.pack + size_t(b0) * kSmBlock + rank * 2 * kSmOp;
                int id = cnt ? int(__ldg(a.list + b0)) : 0;
                for (int s = 0; s < cnt; ++s) {
                    const int next = s + 1 < cnt ? int(__ldg(a.list + b0 + s + 1)) : 0;
                    if (use) ok = sm_wait(ctl, &ctl->empty[slot], (use - 1) & 1u, spin_limit, status);
                    if (!ok) break;
                    const uint32_t st = saddr(sm + kSmBase) + uint32_t(slot) * kSmStage;
                    const uint32_t bar = saddr(&ctl->full[slot]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                 ::"r"(bar), "r"(kSmStage) : "memory");
                    auto copy = [&](uint32_t dst, const unsigned char *src) {
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
                                     "[%0], [%1], %2, [%3];"
                                     ::"r"(dst), "l"(src), "r"(2 * kSmOp), "r"(bar) : "memory");
                    };
                    copy(st, x + size_t(id) * 2 * kSmOp);
                    copy(st + 2 * kSmOp, m + size_t(s) * kSmBlock);
                    ++issued;
                    id = next;
                    if (++slot == kSmStages) {
                        slot = 0;
                        ++use;
                    }
                }
            }
            // copies that nobody may have waited for end before the block does
            for (uint32_t i = issued > kSmStages ? issued - kSmStages : 0; i < issued; ++i)
                drain(&ctl->full[i % kSmStages], (i / kSmStages) & 1u);
        }
        __syncwarp();
    } else {
        // ---- MMA issue (leader), or passing this CTA's stages on -------------
        const uint32_t sa = saddr(sm + kSmBase);
        int slot = 0, use = 0;
        uint32_t grp = 0;
        bool ok = true;
        for (int t = first; t < ntile && ok; t += step) {
            const SmTile tl = sm_tile(t, nrb, ncb);
            const int cnt = int(a.base[rb0 + tl.rb + 1] - a.base[rb0 + tl.rb]);
            for (int s = 0; s < cnt; ++s) {
                const uint32_t buf = grp & 1u, in = uint32_t(s % kSmGroup);
                const bool last = in == kSmGroup - 1 || s == cnt - 1;
                if (rank == 0 && in == 0 && grp >= 2)
                    ok = sm_wait_warp(ctl, &ctl->acc_empty[buf], ((grp >> 1) - 1) & 1u, spin_limit, status);
                if (ok) ok = sm_wait_warp(ctl, &ctl->full[slot], use & 1u, spin_limit, status);
                if (ok && rank == 0) ok = sm_wait_warp(ctl, &ctl->pfull[slot], use & 1u, spin_limit, status);
                if (!ok) break;
                if (rank == 0) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t x = sa + uint32_t(slot) * kSmStage, m = x + 2 * kSmOp;
                    const uint32_t d = tmem + buf * 256u;
                    if (elect_one()) {
                        // the small products first: sums are cut at their size then
#pragma unroll
                        for (int ks = 0; ks < kSmK / 8; ++ks) {
                            const uint64_t dx = sdesc(x + ks * 256u, kSmSbo);
                            const uint64_t dm = sdesc(m + ks * 256u, kSmSbo);
                            mma2(d, dx, dm + (kSmOp >> 4), (in | uint32_t(ks)) ? 1u : 0u);
                            mma2(d, dx + (kSmOp >> 4), dm, 1u);
                        }
#pragma unroll
                        for (int ks = 0; ks < kSmK / 8; ++ks)
                            mma2(d, sdesc(x + ks * 256u, kSmSbo), sdesc(m + ks * 256u, kSmSbo), 1u);
                        commit2(&ctl->empty[slot]);
                        if (last) commit2(&ctl->acc_full[buf]);
                    }
                    __syncwarp();
                } else if (lane == 0) {
                    arrive_leader(&ctl->pfull[slot]);
                }
                __syncwarp();
                if (last) ++grp;
                if (++slot == kSmStages) {
                    slot = 0;
                    ++use;
                }
            }
        }
        // every MMA issued is done, and its signs are in, before either CTA leaves
        if (rank == 0 && elect_one()) commit2(&ctl->fin);
        __syncwarp();
        drain(&ctl->fin, 0);
        __syncwarp();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 9)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------------------------
// X as operands: block [128 columns][32 J], hi then lo, zero outside.  Bound by
// memory (4 bytes read, 8 written an element).
//   TRANS: element (J, c) is src[c * stride + J], else src[J * stride + c]
//   bad (or null): set to 1 if an element has no finite halves
// ---------------------------------------------------------------------------
template <bool TRANS>
__global__ void __launch_bounds__(256)
k_same_x(const float *__restrict__ src, int64_t stride, int N, int64_t ncols, int64_t nch,
         unsigned char *__restrict__ out, int *__restrict__ bad)
{
    bool odd = false;
    // lanes along the direction that is contiguous in src
    const int t = threadIdx.x;
    const int64_t ch = TRANS ? blockIdx.x : blockIdx.y, cb = TRANS ? blockIdx.y : blockIdx.x;
    unsigned char *blk = out + (size_t(cb) * nch + size_t(ch)) * 2 * kSmOp;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int xcol = TRANS ? (t >> 3) + 32 * i : t & 127;
        const int k4 = TRANS ? t & 7 : (t >> 7) + 2 * i;
        const int64_t c = cb * 128 + xcol;
        const int J = int(ch) * kSmK + 4 * k4;
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = c < ncols && J + q < N ? __ldg(TRANS ? src + c * stride + J + q : src + (J + q) * stride + c)
                                          : 0.0f;
        float4 h, l;
        split_rn(v[0], h.x, l.x);
        split_rn(v[1], h.y, l.y);
        split_rn(v[2], h.z, l.z);
        split_rn(v[3], h.w, l.w);
        const uint32_t off = kmaj(xcol, 4 * k4, kSmSbo);
        *reinterpret_cast<float4 *>(blk + off) = h;
        *reinterpret_cast<float4 *>(blk + kSmOp + off) = l;
        // x, or hi alone, infinite or NaN: lo is then too
        auto none = [](float x) { return (__float_as_uint(x) & 0x7F800000u) == 0x7F800000u; };
        odd = odd || none(l.x) || none(l.y) || none(l.z) || none(l.w);
    }
    if (bad && odd) *bad = 1;
}

// Both sides by rows, as k_spmm sums them, if bad[0]; the last block clears it
// (bad[1]: blocks done)
__global__ void __launch_bounds__(256)
k_same_rows(SameRows a, int *bad)
{
    if (*reinterpret_cast<volatile int *>(bad) == 0) return;
    const int64_t nr = a.row1 - a.row0, ca = (a.Nb + 255) / 256, cb = (nr + 255) / 256;
    const int64_t na = nr * ca, items = na + a.Nb * cb;
    for (int64_t i = blockIdx.x; i < items; i += gridDim.x) {
        const bool al = i < na;
        const int64_t j = al ? i : i - na, r = al ? a.row0 + j / ca : j / cb;
        const int64_t c = (al ? j % ca : j % cb) * 256 + threadIdx.x;
        if (c >= (al ? a.Nb : nr)) continue;
        const int32_t *ptr = al ? a.aptr : a.bptr, *col = al ? a.acol : a.bcol;
        const float *val = al ? a.aval : a.bval;
        const float *x = al ? a.psi + c : a.psi + (a.row0 + c) * a.Nb;
        const int64_t step = al ? a.Nb : 1;
        float s[2] = {0.0f, 0.0f};
        const int k0 = ptr[r], k1 = ptr[r + 1];
        for (int k = k0; k < k1; ++k) s[(k - k0) & 1] = fmaf(val[k], x[col[k] * step], s[(k - k0) & 1]);
        (al ? a.sigma + (r - a.row0) * a.Nb : a.tau + r * nr)[c] = s[0] + s[1];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(bad + 1, 1) == int(gridDim.x) - 1) bad[0] = bad[1] = 0;
    }
}

// ---------------------------------------------------------------------------
// M as operands.  used[row block][32 columns] -> places in the list (host side sums
// the counts), then every nonzero to its place in both halves
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_same_used(const int32_t *__restrict__ ptr, const int32_t *__restrict__ col, int N, int nch,
            uint32_t *__restrict__ place, int32_t *__restrict__ count)
{
    const int rb = blockIdx.x;
    uint32_t *p = place + size_t(rb) * nch;             // zero before
    const int r = rb * kSmRows + int(threadIdx.x);
    if (r < N)
        for (int k = ptr[r]; k < ptr[r + 1]; ++k)
            if (col[k] != r) p[col[k] / kSmK] = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        int n = 0;
        for (int i = 0; i < nch; ++i)
            if (p[i]) p[i] = uint32_t(++n);             // 1 + place
        count[rb] = n;
    }
}

__global__ void __launch_bounds__(256)
k_same_fill(const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
            const float *__restrict__ val, int N, int nch, const uint32_t *__restrict__ place,
            const int64_t *__restrict__ base, uint16_t *__restrict__ list,
            unsigned char *__restrict__ pack, float *__restrict__ diag)
{
    const int r = blockIdx.x, rb = r / kSmRows, m = r & (kSmRows - 1);
    const uint32_t *p = place + size_t(rb) * nch;
    if (m == 0)
        for (int i = threadIdx.x; i < nch; i += blockDim.x)
            if (p[i]) list[base[rb] + p[i] - 1] = uint16_t(i);
    for (int k = ptr[r] + int(threadIdx.x); k < ptr[r + 1]; k += blockDim.x) {
        const int c = col[k];
        if (c == r) {
            diag[r] = val[k];
            continue;
        }
        float h, l;
        split_rn(val[k], h, l);
        unsigned char *dst = pack + size_t(base[rb] + p[c / kSmK] - 1) * kSmBlock +
                             size_t(m >> 7) * 2 * kSmOp + kmaj(m & 127, c & (kSmK - 1), kSmSbo);
        *reinterpret_cast<float *>(dst) = h;
        *reinterpret_cast<float *>(dst + kSmOp) = l;
    }
}

int same_row_blocks(int64_t N) { return int((N + kSmRows - 1) / kSmRows); }
int same_chunks(int64_t N) { return int((N + kSmK - 1) / kSmK); }
size_t same_block_bytes() { return kSmBlock; }
// of X; the columns of both CTAs of a pair, and 256 rows, which the last block of
// rows reads (its diagonal) and multiplies whole
size_t same_x_bytes(int64_t N, int64_t ncols)
{
    return size_t((ncols + kSmCols - 1) / kSmCols) * 2 * size_t(same_chunks(N)) * 2 * kSmOp;
}

cudaError_t same_used(const int32_t *ptr, const int32_t *col, int64_t N, uint32_t *place,
                      int32_t *count, cudaStream_t st)
{
    k_same_used<<<unsigned(same_row_blocks(N)), 256, 0, st>>>(ptr, col, int(N), same_chunks(N), place, count);
    hy::count_launch();
    return cudaGetLastError();
}

cudaError_t same_fill(const int32_t *ptr, const int32_t *col, const float *val, int64_t N,
                      const uint32_t *place, const int64_t *base, uint16_t *list,
                      unsigned char *pack, float *diag, cudaStream_t st)
{
    k_same_fill<<<unsigned(N), 256, 0, st>>>(ptr, col, val, int(N), same_chunks(N), place, base, list,
                                             pack, diag);
    hy::count_launch();
    return cudaGetLastError();
}

// CTA pairs that run at once (0: none)
int same_pairs()
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = kSmSmem;
    int n = 0;
    if (allow_smem(k_same, kSmSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_same, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t same_rows(const SameRows &a, int *bad, int num_sms, cudaStream_t st)
{
    k_same_rows<<<unsigned(2 * num_sms), 256, 0, st>>>(a, bad);
    hy::count_launch();
    return cudaGetLastError();
}

cudaError_t same(const SameArgs &a, const float *src, int64_t stride, bool trans, int pairs, int *status,
                 int *bad, long long spin_limit, cudaStream_t st)
{
    if (a.row1 <= a.row0 || a.ncols == 0) return cudaSuccess;
    const int64_t nch = same_chunks(a.N), ncb = (a.ncols + kSmCols - 1) / kSmCols;
    if (trans) {
        const dim3 grid(unsigned(nch), unsigned(2 * ncb));
        k_same_x<true><<<grid, 256, 0, st>>>(src, stride, int(a.N), a.ncols, nch, a.xpack, bad);
    } else {
        const dim3 grid(unsigned(2 * ncb), unsigned(nch));
        k_same_x<false><<<grid, 256, 0, st>>>(src, stride, int(a.N), a.ncols, nch, a.xpack, bad);
    }
    hy::count_launch();
    const cudaError_t e = allow_smem(k_same, kSmSmem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = ((a.row1 - 1) / kSmRows + 1 - a.row0 / kSmRows) * ncb;
    k_same<<<unsigned(2 * std::min<int64_t>(pairs, tiles)), kSmThreads, kSmSmem, st>>>(a, status, spin_limit);
    hy::count_launch();
    return cudaGetLastError();
}

}  // namespace k
}  // namespace hy
