// hy_screen32.cu -- the gradient screen of a whole pool on a float state, with
// the float sums of k_grad_partial (hy_sweeps.cu) bit for bit.
//
// k_grad_partial sums, per (operator, row chunk, thread t of 256), the pairs of
// rows chunk, chunk + CH, ... and columns t, t + 256, ... of each constituent in
// float, one row after another, and leaves the thread in double.  That order is
// kept here, thread by thread; what changes is who shares a row.  An operator's
// block loads four amplitudes from L2 and a table entry per pair and waits for
// each row in turn (7.2 ms for the 28-qubit qubit pool, 5 ns x SM a pair, where
// the arithmetic needs 0.1).  Here
//   * alpha-beta constituents: a CTA takes one alpha pattern and several beta
//     patterns.  Its alpha pairs' rows (psi, sigma interleaved) are staged in
//     shared memory one pair ahead (cp.async), a thread keeps its table entries
//     of all its patterns in registers, so that a pair is two 8-byte shared
//     loads: bound by their bank conflicts (a pattern's strings are spread, so
//     sixteen lanes meet about three to a bank; separate 4-byte planes, staged
//     16 bytes at a time, meet more and measured 6.3 ms);
//   * the other constituents (one spin only) run as blocks of the same launch
//     behind them, their entries in registers and several rows in flight (L2).
// Per-operator kernel -> here: 213 k determinants (spin-adapted / qubit pool)
// 240 / 184 -> 150 us, 854 k 614 / 450 -> 359, 2.9 M 1,862 / 1,481 -> 1,210, 11.8 M
// 9,304 / 7,167 -> 5,660, 41 M 50 -> 32 ms.  At 16 orbitals a pair's rows fill the
// SM and a CTA has too few patterns for staging them (250 -> 277 ms): the
// per-operator kernel stays there (kScreen32MaxPairs).
#include "hy_kernels.cuh"

namespace hy {
namespace k {

namespace {

__device__ __forceinline__ float neg_if(float x, uint32_t sbit)
{
    return __uint_as_float(__float_as_uint(x) ^ sbit);
}

// sigma(Cd) psi(d) - sigma(d) psi(Cd), rounded as k_grad_partial rounds it
__device__ __forceinline__ float pair_term(float s2, float p1, float s1, float p2)
{
    return __fmaf_rn(s2, p1, -__fmul_rn(s1, p2));
}

__device__ __forceinline__ void copy4(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                 ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}

// rows A, A' of one alpha pair: plane 0 = (psi, sigma)[A], plane 1 = [A']
__device__ __forceinline__ void stage_pair(float2 *buf, const float *psi, const float *sig,
                                           uint32_t u, int Nb, int pitch)
{
    const int64_t o1 = int64_t(u & 0x7FFFu) * Nb, o2 = int64_t((u >> 15) & 0x7FFFu) * Nb;
    for (int b = threadIdx.x; b < Nb; b += blockDim.x) {
        copy4(&buf[b].x, psi + o1 + b);
        copy4(&buf[b].y, sig + o1 + b);
        copy4(&buf[pitch + b].x, psi + o2 + b);
        copy4(&buf[pitch + b].y, sig + o2 + b);
    }
}

// beta-only constituent: the thread's KK entries in registers, UR rows in
// flight; returns the thread's float sum over rows chunk, chunk + CH, ...
template <int KK, int UR>
__device__ float beta_rows(const float *psi, const float *sig, const uint32_t *be, int cnt, int t,
                           int Na, int Nb, int chunk, int CH)
{
    uint32_t e[KK];
#pragma unroll
    for (int k = 0; k < KK; ++k) e[k] = t + 256 * k < cnt ? __ldg(be + t + 256 * k) : 0u;
    float part = 0.f;
    for (int r0 = chunk; r0 < Na; r0 += UR * CH) {
        float row[UR];
#pragma unroll
        for (int i = 0; i < UR; ++i) {
            const int r = r0 + i * CH;
            const float *p = psi + int64_t(r) * Nb, *s = sig + int64_t(r) * Nb;
            row[i] = 0.f;
            if (r < Na)
#pragma unroll
                for (int k = 0; k < KK; ++k)
                    if (t + 256 * k < cnt) {
                        const int B = e[k] & 0x7FFFu, B2 = (e[k] >> 15) & 0x7FFFu;
                        row[i] = __fadd_rn(row[i], neg_if(pair_term(s[B2], p[B], s[B], p[B2]),
                                                          e[k] & 0x80000000u));
                    }
        }
#pragma unroll
        for (int i = 0; i < UR; ++i)
            if (r0 + i * CH < Na) part = __fadd_rn(part, row[i]);
    }
    return part;
}

// alpha-only constituent: contiguous columns t, t + 256, ... of its row pairs
__device__ float alpha_rows(const float *psi, const float *sig, const uint32_t *ae, int rows, int t,
                            int Nb, int chunk, int CH)
{
    float part = 0.f;
    for (int rr = chunk; rr < rows; rr += CH) {
        const uint32_t u = __ldg(ae + rr);
        const int64_t o1 = int64_t(u & 0x7FFFu) * Nb, o2 = int64_t((u >> 15) & 0x7FFFu) * Nb;
        const float *pA = psi + o1, *sA = sig + o1, *pA2 = psi + o2, *sA2 = sig + o2;
        float row = 0.f;
#pragma unroll 4
        for (int b = t; b < Nb; b += 256)
            row = __fadd_rn(row, pair_term(sA2[b], pA[b], sA[b], pA2[b]));
        part = __fadd_rn(part, neg_if(row, u & 0x80000000u));
    }
    return part;
}

}  // namespace

// G groups of 256 threads.  Blocks below a.n_ab: (chunk, alpha pattern, share
// of the beta patterns), at most G * PB of them; the others: one single-spin
// constituent and chunk per group.  NK: entries of a beta single pattern per
// thread; DB: two staging buffers.
template <int NK, int PB, int G, bool DB>
__global__ void __launch_bounds__(256 * G)
k_screen32(Screen32Args a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[8 * G][PB];
    const int tid = threadIdx.x, t = tid & 255, grp = tid >> 8, lane = tid & 31, warp = tid >> 5;
    const int Nb = a.Nb, Na = a.Na, CH = a.CH;
    float part[PB];
#pragma unroll
    for (int p = 0; p < PB; ++p) part[p] = 0.f;
    int np = 0;                       // values this group produces
    int64_t v0 = 0;                   // first of them
    int chunk;
    if (int(blockIdx.x) < a.n_ab) {
        const int pg = int(blockIdx.x) % a.n_pg, q = int(blockIdx.x) / a.n_pg;
        const int ia = q % a.nA;
        chunk = q / a.nA;
        const int c0 = a.nB * pg / a.n_pg, c1 = a.nB * (pg + 1) / a.n_pg;
        const int g0 = c0 + (c1 - c0) * grp / G, g1 = c0 + (c1 - c0) * (grp + 1) / G;
        np = g1 - g0;
        v0 = int64_t(ia) * a.nB + g0;
        // two planes of Nb amplitudes and a zero one that absent entries read
        const int pitch = Nb + 1;
        float2 *buf = reinterpret_cast<float2 *>(smem_raw);
        for (int i = tid; i < (DB ? 4 : 2); i += blockDim.x) buf[i * pitch + Nb] = make_float2(0.f, 0.f);
        uint32_t e[PB][NK];
#pragma unroll
        for (int p = 0; p < PB; ++p) {
            const int id = p < np ? a.lb[g0 + p] : 0;
            const int cnt = p < np ? int(a.bcnt[id]) : 0;
            const uint32_t *be = a.bent + (p < np ? a.boff[id] : 0);
#pragma unroll
            for (int k = 0; k < NK; ++k)
                e[p][k] = t + 256 * k < cnt ? __ldg(be + t + 256 * k) : uint32_t(Nb) | (uint32_t(Nb) << 15);
        }
        const int ida = a.la[ia], rows = int(a.acnt[ida]);
        const uint32_t *ae = a.aent + a.aoff[ida];
        if (DB && chunk < rows) stage_pair(buf, a.psi, a.sigma, __ldg(ae + chunk), Nb, pitch);
        if (DB) asm volatile("cp.async.commit_group;" ::: "memory");
        int cur = 0;
        for (int rr = chunk; rr < rows; rr += CH) {
            const uint32_t u = __ldg(ae + rr);
            if (DB) {
                // the next pair into the other buffer, read last an iteration ago
                if (rr + CH < rows)
                    stage_pair(buf + (cur ^ 1) * 2 * pitch, a.psi, a.sigma, __ldg(ae + rr + CH), Nb, pitch);
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                stage_pair(buf, a.psi, a.sigma, u, Nb, pitch);
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            const float2 *x = buf + cur * 2 * pitch, *y = x + pitch;
#pragma unroll
            for (int p = 0; p < PB; ++p) {
                float row = 0.f;
#pragma unroll
                for (int k = 0; k < NK; ++k) {
                    const float2 d = x[e[p][k] & 0x7FFFu], c = y[(e[p][k] >> 15) & 0x7FFFu];
                    row = __fadd_rn(row, neg_if(pair_term(c.y, d.x, d.y, c.x), e[p][k] & 0x80000000u));
                }
                part[p] = __fadd_rn(part[p], neg_if(row, u & 0x80000000u));
            }
            __syncthreads();
            if (DB) cur ^= 1;
        }
    } else {
        const int64_t o = int64_t(int(blockIdx.x) - a.n_ab) * G + grp;
        chunk = int(o % CH);
        const int id = int(o / CH);
        if (id < a.npA + a.npB) {
            np = 1;
            v0 = int64_t(a.nA) * a.nB + id;
            if (id < a.npA) {
                part[0] = alpha_rows(a.psi, a.sigma, a.aent + a.aoff[id], int(a.acnt[id]), t, Nb, chunk, CH);
            } else {
                const int ib = id - a.npA, cnt = int(a.bcnt[ib]);
                const uint32_t *be = a.bent + a.boff[ib];
                if (cnt <= 256)
                    part[0] = beta_rows<1, 8>(a.psi, a.sigma, be, cnt, t, Na, Nb, chunk, CH);
                else if (cnt <= 1024)
                    part[0] = beta_rows<4, 2>(a.psi, a.sigma, be, cnt, t, Na, Nb, chunk, CH);
                else
                    part[0] = beta_rows<14, 1>(a.psi, a.sigma, be, cnt, t, Na, Nb, chunk, CH);
            }
        }
    }
    // double from here: lanes, then the group's warps in order
#pragma unroll
    for (int p = 0; p < PB; ++p) {
        double s = double(part[p]);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) red[warp][p] = s;
    }
    __syncthreads();
    if (t < np) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += red[grp * 8 + w][t];
        a.partials[(v0 + t) * CH + chunk] = s;
    }
}

// g of every operator from its constituents' values (a warp per operator,
// lanes over the chunks)
__global__ void __launch_bounds__(256)
k_screen32_final(Screen32Args a, const OpDev *__restrict__ opd, const ConsDev *__restrict__ cons,
                 const int32_t *__restrict__ aslot, const int32_t *__restrict__ bslot, int64_t n_ops,
                 double *__restrict__ g)
{
    const int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n_ops) return;
    const OpDev od = opd[i];
    double tot = 0.0;
    for (int c = 0; c < od.nc; ++c) {
        const ConsDev cd = cons[c == 0 ? od.c0 : od.c1];
        const int64_t v = cd.ap >= 0 && cd.bp >= 0 ? int64_t(aslot[cd.ap]) * a.nB + bslot[cd.bp]
                        : int64_t(a.nA) * a.nB + (cd.ap >= 0 ? cd.ap : a.npA + cd.bp);
        double s = 0.0;
        for (int j = lane; j < a.CH; j += 32) s += a.partials[v * a.CH + j];
        tot += double(cd.eps) * s;
    }
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
    if (lane == 0) g[i] = 2.0 * tot;
}

namespace {

template <int NK, int PB, int G, bool DB>
cudaError_t run32(Screen32Args &a, cudaStream_t st)
{
    a.n_pg = a.nB > 0 ? (a.nB + G * PB - 1) / (G * PB) : 0;
    a.n_ab = a.CH * a.nA * a.n_pg;
    const int64_t others = (int64_t(a.npA + a.npB) * a.CH + G - 1) / G;
    const size_t smem = size_t(DB ? 4 : 2) * (size_t(a.Nb) + 1) * sizeof(float2);
    auto *kern = k_screen32<NK, PB, G, DB>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<unsigned(a.n_ab + others), 256 * G, smem, st>>>(a);
    hy::count_launch();
    return cudaGetLastError();
}

}  // namespace

// entries per thread (NK) x patterns (PB) within ~21 registers; 16 to 18
// patterns per CTA, so that staging a pair (an element per copy) costs less than
// reading it (8 patterns: 7.3 ms at 14 orbitals, 16: 5.7)
cudaError_t screen32(Screen32Args a, int bs_cnt, const OpDev *opd, const ConsDev *cons,
                     const int32_t *aslot, const int32_t *bslot, int64_t n_ops, double *g,
                     cudaStream_t st)
{
    if (n_ops == 0) return cudaSuccess;
    const cudaError_t e = bs_cnt <= 256 ? run32<1, 9, 2, true>(a, st)
                        : bs_cnt <= 512 ? run32<2, 5, 2, true>(a, st)
                        : bs_cnt <= 1024 ? run32<4, 4, 4, true>(a, st)
                                         : run32<7, 3, 4, false>(a, st);
    if (e != cudaSuccess) return e;
    k_screen32_final<<<unsigned((n_ops + 7) / 8), 256, 0, st>>>(a, opd, cons, aslot, bslot, n_ops, g);
    hy::count_launch();
    return cudaGetLastError();
}

}  // namespace k
}  // namespace hy
