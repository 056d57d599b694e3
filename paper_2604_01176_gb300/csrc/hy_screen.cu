// hy_screen.cu -- the gradient screen of whole pools in double precision,
// g_k = 2 <sigma|A_k psi> for every operator of one or many molecules in one
// launch.
//
// For a constituent C with sign s on the pair d -> C d,
//   <sigma|(C - C^dagger) psi> = sum_d s [sigma(Cd) psi(d) - sigma(d) psi(Cd)],
// and the pairs factor into string pairs of the two spins.  A pool holds few
// distinct string patterns (at 32 qubits 64 singles and 784 doubles per spin)
// in many combinations (3,376 operators), so instead of one pass over the
// state per operator the work is cut by pattern:
//
//   * alpha-beta tasks: for an alpha single pattern (or the alpha identity),
//     a task stages the psi and sigma rows A, A' of some of its pairs in
//     shared memory and sums every beta single pattern (and the beta
//     identity) over them.  A row is read once for all nb * vb beta patterns;
//   * same-spin tasks: rows (or columns) of psi and sigma are staged and every
//     beta (alpha) double pattern summed over them.
//
// What bounds it: the FP64 pipe.  A pair costs two FMAs (the sign is applied
// to an operand by an integer XOR; the per-operator kernel k_grad_partial
// spends three FP64 instructions and four gathers from L2 on it), two 16-byte
// shared loads of (psi, sigma) and a table entry.  Measured: 1,463 -> 520 us for
// the 24-qubit pool (1.28e8 pairs; 406 us at the FP64 rate), 8.4 -> 2.7 ms for
// the pools of 20 molecules of 8 to 12 orbitals.  Three configurations by
// string count (build_screen_plan): 0 and 1 differ in the vectors staged by a
// same-spin task (4 and 2 per string: two CTAs, or one, per SM), 2 serves
// string counts whose two alpha-beta planes exceed one SM's shared memory
// (n = 16): each of the two terms of a pair is then summed in its own pass
// over planes of 8 bytes per string.  All orders are fixed.
//
// Float screens keep the per-operator order of k_grad_partial (hy_sweeps.cu):
// their sums run in float, so another order gives other results.
#include "hy_kernels.cuh"

#include <type_traits>

namespace hy {
namespace k {

namespace {

constexpr int kScThreads = 512, kScWarps = kScThreads / 32;
constexpr int kScSeg = 5;      // patterns a warp's share of <= 64 patterns can touch

__device__ __forceinline__ double flip(double x, uint32_t sbit)
{
    return __hiloint2double(__double2hiint(x) ^ int(sbit), __double2loint(x));
}
// s * (psi(d) sigma(Cd) - sigma(d) psi(Cd)), or one of its two products
__device__ __forceinline__ void term(double &t, const double2 &u, const double2 &v, uint32_t sbit)
{
    t = fma(flip(u.x, sbit), v.y, t);
    t = fma(flip(u.y, sbit ^ 0x80000000u), v.x, t);
}
__device__ __forceinline__ void term(double &t, const double &u, const double &v, uint32_t sbit)
{
    t = fma(flip(u, sbit), v, t);
}

// entries of one pattern part over a staged group, LANES threads at a time: the
// entry loads of four strides go out together, ahead of their shared loads
template <typename U, int Q, int LANES>
__device__ __forceinline__ void sum_pairs(double &t, const uint32_t *__restrict__ ent, int n, int lane,
                                          const U *p1, const U *p2, int pitch)
{
    for (int e = lane; e < n; e += 4 * LANES) {
        uint32_t u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = e + LANES * i < n ? __ldg(ent + e + LANES * i) : 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (e + LANES * i < n) {
                const int B = u[i] & 0x7FFFu, B2 = (u[i] >> 15) & 0x7FFFu;
                const uint32_t sb = u[i] & 0x80000000u;
#pragma unroll
                for (int q = 0; q < Q; ++q) term(t, p1[B + q * pitch], p2[B2 + q * pitch], sb);
            }
    }
}

__device__ __forceinline__ double warp_total(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// stage the planes of an alpha pair (A, A', sign sa): u = row A, v = sa * row A'
__device__ __forceinline__ void stage_ab(double2 *p1, double2 *p2, const double *psi,
                                         const double *sig, int Nb, int64_t A, int64_t A2,
                                         uint32_t sa, int)
{
    const double *pA = psi + A * Nb, *sA = sig + A * Nb, *pA2 = psi + A2 * Nb, *sA2 = sig + A2 * Nb;
    for (int b = threadIdx.x; b < Nb; b += kScThreads) {
        p1[b] = make_double2(pA[b], sA[b]);
        p2[b] = make_double2(flip(pA2[b], sa), flip(sA2[b], sa));
    }
}
// pass 0: psi_A, sa sigma_A'; pass 1: sigma_A, -sa psi_A'
__device__ __forceinline__ void stage_ab(double *p1, double *p2, const double *psi,
                                         const double *sig, int Nb, int64_t A, int64_t A2,
                                         uint32_t sa, int pass)
{
    const double *x = (pass ? sig : psi) + A * Nb, *y = (pass ? psi : sig) + A2 * Nb;
    const uint32_t f = pass ? sa ^ 0x80000000u : sa;
    for (int b = threadIdx.x; b < Nb; b += kScThreads) {
        p1[b] = x[b];
        p2[b] = flip(y[b], f);
    }
}

}  // namespace

// kind 0: alpha-beta task (idx = alpha pattern, nA = the identity); kind 1:
// alpha doubles over columns; kind 2: beta doubles over rows.  chunk: the
// task's groups are chunk, chunk + CH, ...; slice: its share of the patterns (one
// slice unless the groups are too few, CUT: the plan has several somewhere, which
// costs the other plans 1 to 2 us).  OCC: CTAs that fit an SM's shared memory;
// one alone has twice the registers (16 orbitals, 8+8: 300 -> 289 ms, 15, 8+7: 58.3 -> 55.4)
template <int CFG, int OCC, bool CUT>
__global__ void __launch_bounds__(kScThreads, OCC)
k_screen(ScreenArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[kScWarps][kScSeg + 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int4 tk = a.tasks[blockIdx.x];
    const ScreenMol &m = a.mols[tk.x];
    const double *psi = a.psi + m.off, *sig = a.sigma + m.off;
    const int Na = m.Na, Nb = m.Nb;
    const int kind = tk.y, chunk = CUT ? tk.w & 0xFFFF : tk.w, slice = CUT ? tk.w >> 16 : 0;
    int CH = m.ch[kind];

    if (kind == 0) {
        using U = std::conditional_t<CFG == 2, double, double2>;
        U *p1 = reinterpret_cast<U *>(smem_raw), *p2 = p1 + Nb;
        const int ia = tk.z;
        const bool ident = ia == m.nA;
        if (CUT && ident) CH = m.chi;
        const int cnt = ident ? Na : int(m.acnt[m.la[ia]]);
        const uint32_t *ae = ident ? nullptr : m.aent + m.aoff[m.la[ia]];
        // this warp's share [lo, hi) of the pairs of the slice's beta singles [b0, b1),
        // cut by pattern
        const uint32_t *bent = m.bent;
        const int nB = m.nB, cb = nB > 0 ? int(m.bcnt[m.lb[0]]) : 0;
        int b0 = 0, b1 = nB;
        if (CUT) {
            const int Z = m.zs[ident ? 1 : 0];
            b0 = nB * slice / Z;
            b1 = nB * (slice + 1) / Z;
        }
        const int tot = (b1 - b0) * cb;
        const int lo = b0 * cb + int(int64_t(tot) * warp / kScWarps);
        const int hi = b0 * cb + int(int64_t(tot) * (warp + 1) / kScWarps);
        int so[kScSeg];
        int sn[kScSeg];
        const int first = cb > 0 ? lo / cb : 0;
#pragma unroll
        for (int s = 0; s < kScSeg; ++s) {
            const int p = first + s;
            const int e0 = max(lo, p * cb), e1 = min(hi, (p + 1) * cb);
            sn[s] = p < b1 && e1 > e0 ? e1 - e0 : 0;
            so[s] = sn[s] ? int(m.boff[m.lb[p]]) + (e0 - p * cb) : 0;
        }
        double acc[kScSeg], aid = 0.0;
#pragma unroll
        for (int s = 0; s < kScSeg; ++s) acc[s] = 0.0;
        for (int g = chunk; g < cnt; g += CH) {
            const uint32_t u = ae ? __ldg(ae + g) : uint32_t(g) | (uint32_t(g) << 15);
            const int64_t A = u & 0x7FFFu, A2 = (u >> 15) & 0x7FFFu;
            const uint32_t sa = u & 0x80000000u;
            for (int pass = 0; pass < (CFG == 2 ? 2 : 1); ++pass) {
                __syncthreads();
                stage_ab(p1, p2, psi, sig, Nb, A, A2, sa, pass);
                __syncthreads();
#pragma unroll
                for (int s = 0; s < kScSeg; ++s)
                    if (sn[s]) sum_pairs<U, 1, 32>(acc[s], bent + so[s], sn[s], lane, p1, p2, 0);
                if (!ident && (!CUT || slice == 0))
                    for (int b = tid; b < Nb; b += kScThreads) term(aid, p1[b], p2[b], 0u);
            }
        }
        // per warp and segment, then per pattern over the warps in order
        __syncthreads();
#pragma unroll
        for (int s = 0; s < kScSeg; ++s) {
            const double v = warp_total(acc[s]);
            if (lane == 0) red[warp][s] = sn[s] ? v : 0.0;
        }
        const double v = warp_total(aid);
        if (lane == 0) red[warp][kScSeg] = v;
        __syncthreads();
        double *out = a.partials + m.base[0] + (int64_t(ia) * (CUT ? m.ch[0] : CH) + chunk) * (nB + 1);
        for (int i = tid; i <= b1 - b0; i += kScThreads) {
            const int p = i < b1 - b0 ? b0 + i : nB;
            if (CUT && p == nB && slice) break;
            double s = 0.0;
            if (p == nB) {
                for (int w = 0; w < kScWarps; ++w) s += red[w][kScSeg];
            } else {
                for (int w = 0; w < kScWarps; ++w) {
                    const int l = b0 * cb + int(int64_t(tot) * w / kScWarps);
                    const int q = p - l / cb;       // segment of warp w for pattern p
                    if (q >= 0 && q < kScSeg) s += red[w][q];
                }
            }
            out[p] = s;
        }
        return;
    }

    // same-spin doubles: V vectors of Ns amplitudes, element s of vector v at
    // v * vst + s * sst
    constexpr int Q = CFG == 0 ? 4 : CFG == 1 ? 2 : 1;      // vectors per group
    const bool al = kind == 1;
    const int Ns = al ? Na : Nb, V = al ? Nb : Na;
    const int64_t sst = al ? Nb : 1, vst = al ? 1 : Nb;
    const int nAll = al ? m.nRa : m.nRb;
    int r0 = 0, nR = nAll;
    if (CUT) {
        const int Z = m.zs[kind + 1];
        r0 = nAll * slice / Z;
        nR = nAll * (slice + 1) / Z - r0;
    }
    const int32_t *ids = (al ? m.ra : m.rb) + r0;
    const uint32_t *ent = al ? m.aent : m.bent;
    const int64_t *off = al ? m.aoff : m.boff, *cnts = al ? m.acnt : m.bcnt;
    double2 *pl = reinterpret_cast<double2 *>(smem_raw);                // [Q][Ns]
    double *acc = reinterpret_cast<double *>(pl + size_t(Q) * Ns);      // [nR padded to 4]
    for (int i = tid; i < (nR + 3) / 4 * 4; i += kScThreads) acc[i] = 0.0;
    const int cnt = int(cnts[ids[0]]);
    for (int v0 = chunk * Q; v0 < V; v0 += CH * Q) {
        __syncthreads();
        auto put = [&](int s, int r) {
            const int64_t o = int64_t(v0 + r) * vst + s * sst;
            pl[r * Ns + s] = v0 + r < V ? make_double2(psi[o], sig[o]) : make_double2(0.0, 0.0);
        };
        if (al) {               // a string's Q neighbouring columns share its sectors
            for (int i = tid; i < Ns * Q; i += kScThreads) put(i / Q, i % Q);
        } else {
            for (int r = 0; r < Q; ++r)
                for (int s = tid; s < Ns; s += kScThreads) put(s, r);
        }
        __syncthreads();
        // eight lanes per pattern: a double has few pairs (70 at 12 orbitals),
        // so a whole warp on one leaves lanes idle (27 %) and pays a longer sum
        for (int p = tid >> 3; p < (nR + 3) / 4 * 4; p += kScThreads / 8) {
            double t = 0.0;
            if (p < nR) sum_pairs<double2, Q, 8>(t, ent + off[ids[p]], cnt, lane & 7, pl, pl, Ns);
            for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if ((lane & 7) == 0) acc[p] += t;
        }
    }
    __syncthreads();
    double *out = a.partials + m.base[kind] + int64_t(chunk) * nAll + r0;
    for (int i = tid; i < nR; i += kScThreads) out[i] = acc[i];
}

// g of every operator: its constituents' values, each the sum of its tasks'
// partials in task order (a warp per operator, lanes over the tasks)
__global__ void __launch_bounds__(256)
k_screen_final(const ScreenMol *__restrict__ mols, int count, const double *__restrict__ partials,
               int64_t n_ops, double *__restrict__ g)
{
    const int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n_ops) return;
    int lo = 0, hi = count;                       // molecule: gbase <= i < next gbase
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (mols[mid].gbase <= i) lo = mid; else hi = mid;
    }
    const ScreenMol &m = mols[lo];
    const OpDev od = m.opd[i - m.gbase];
    double tot = 0.0;
    for (int c = 0; c < od.nc; ++c) {
        const ConsDev cd = m.cons[c == 0 ? od.c0 : od.c1];
        const int sa = cd.ap < 0 ? m.nA : m.aslot[cd.ap];     // >= 0: alpha-beta row
        const int sb = cd.bp < 0 ? m.nB : m.bslot[cd.bp];
        const double *p;
        int64_t stride;
        int ch;
        if (sa >= 0 && sb >= 0) {
            ch = sa == m.nA ? m.chi : m.ch[0];
            stride = m.nB + 1;
            p = partials + m.base[0] + int64_t(sa) * m.ch[0] * stride + sb;
        } else if (sa < 0) {
            ch = m.ch[1];
            stride = m.nRa;
            p = partials + m.base[1] + (-1 - sa);
        } else {
            ch = m.ch[2];
            stride = m.nRb;
            p = partials + m.base[2] + (-1 - sb);
        }
        double s = 0.0;
        for (int j = lane; j < ch; j += 32) s += p[j * stride];
        tot += double(cd.eps) * s;
    }
    tot = warp_total(tot);
    if (lane == 0) g[i] = 2.0 * tot;
}

template <int CFG, int OCC>
cudaError_t screen_cfg(const ScreenArgs &a, bool cut, int n_tasks, size_t smem, cudaStream_t st)
{
    auto run = [&](auto *kernel) {
        const cudaError_t e = allow_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        kernel<<<unsigned(n_tasks), kScThreads, smem, st>>>(a);
        hy::count_launch();
        return cudaGetLastError();
    };
    return cut ? run(k_screen<CFG, OCC, true>) : run(k_screen<CFG, OCC, false>);
}

cudaError_t screen_all(const ScreenArgs &a, int cfg, bool cut, int n_tasks, size_t smem, int count,
                       int64_t n_ops, double *g, cudaStream_t st)
{
    if (n_ops == 0) return cudaSuccess;
    const bool two = smem <= 113 * 1024;
    const cudaError_t e = cfg == 0 ? screen_cfg<0, 2>(a, cut, n_tasks, smem, st)
                        : cfg == 1 ? (two ? screen_cfg<1, 2>(a, cut, n_tasks, smem, st)
                                          : screen_cfg<1, 1>(a, cut, n_tasks, smem, st))
                                   : screen_cfg<2, 1>(a, cut, n_tasks, smem, st);
    if (e != cudaSuccess) return e;
    k_screen_final<<<unsigned((n_ops + 7) / 8), 256, 0, st>>>(a.mols, count, a.partials, n_ops, g);
    hy::count_launch();
    return cudaGetLastError();
}

}  // namespace k
}  // namespace hy
