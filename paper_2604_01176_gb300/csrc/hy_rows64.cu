// hy_rows64.cu -- sigma = H psi in double precision for beta string spaces of
// up to kRowsMaxNb strings (13 orbitals at half filling), one molecule or
// many, in one launch.  A CTA computes one output alpha row a' on a chunk of
// at most kRowsCols columns, a column per thread, all three parts of
//   sigma[a'][b'] = sum_J Ma[a'][J] psi[J][b']                (alpha part)
//                 + sum_K Mb[b'][K] psi[a'][K]                (beta part)
//                 + sum_{e in X(a'), f in X(b')} C_e[f] psi[J_e][K_f]
//
// Bound: the FP64 pipe (one DFMA per coupling; 2 per clock and SM).  What the
// sweep in parts (hy_sigma.cu: CSR product, transpose, CSR product, transposed
// add, coupling) spends beside that at these sizes, and what is done here:
//   * the diagonal beta term's half-mask tables are built per alpha partner
//     with 2 x 256 x 8 additions, 12 % of the DFMAs at 12 orbitals and more
//     than all of them at 8: here a table covers half of the n orbitals, each
//     entry is one addition to the entry without its top bit;
//   * a partner row is staged, then multiplied, 37 times per row: here two
//     partners per slice are staged interleaved, so that one 16-byte load
//     brings both and a column's excitation entry is read once for them;
//   * 924 whole rows on 304 CTA slots run in four waves for 3.04 waves of
//     work: chunks of columns make three times as many tasks;
//   * small systems pay for five dependent launches, and their few warps for
//     long chains of FMAs (a warp's DFMA occupies its quarter of the SM for 64
//     clocks): there the partners of a row are split over ES = 4 slices of the
//     CTA, whose sums are added in order at the end.
// Measured, sweep in parts -> rows: 400 determinants 117 -> 14 us, 63,504 264 ->
// 141 us, 853,776 4,020 -> 3,030 us (2,580 us at the measured 0.60 TFMA/s), 20
// molecules of 8 to 12 orbitals 17.1 -> 14.3 ms.
// The beta part reads its table by column (entry k of all columns contiguous,
// built from the CSR table when the Hamiltonian is).  Every element's sum has
// a fixed order that depends on its row and column only.
#include "hy_kernels.cuh"

namespace hy {
namespace k {

namespace {

__device__ __forceinline__ double flip_sign(double x, uint32_t sbit)
{
    return __hiloint2double(__double2hiint(x) ^ int(sbit), __double2loint(x));
}

// staged values of a slice: two alpha partners per index
struct RowsSmem {
    double2 *R, *C, *TL, *TH;       // psi rows, coefficients, diagonal half tables
};

__host__ __device__ __forceinline__ int low_bits(int n) { return (n + 1) / 2; }

__host__ __device__ __forceinline__ int64_t slice_units(int64_t Nb, int n)
{
    return Nb + n * n + (int64_t(1) << low_bits(n)) + (int64_t(1) << (n - low_bits(n)));
}

__device__ __forceinline__ RowsSmem rows_smem(unsigned char *base, int slice, int Nb, int n)
{
    RowsSmem s;
    s.R = reinterpret_cast<double2 *>(base) + slice * slice_units(Nb, n);
    s.C = s.R + Nb;
    s.TL = s.C + n * n;
    s.TH = s.TL + (1 << low_bits(n));
    return s;
}

}  // namespace

size_t rows64_smem(int64_t Nb, int n, int slices)
{
    return size_t(slices) * size_t(slice_units(Nb, n)) * 16;
}

// CTA: slices x columns threads (columns: chunk width rounded up to a warp)
template <int ES>
__global__ void __launch_bounds__(ES == 1 ? kRowsCols : ES * kRowsColsSmall)
k_rows64(const __grid_constant__ Rows64Args a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double part[ES == 1 ? 1 : (ES - 1) * kRowsColsSmall];
    __shared__ double red[32];
    __shared__ uint32_t ent[2 * ES];
    constexpr int E = 2 * ES;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int cols = nt / ES, slice = ES == 1 ? 0 : tid / cols, ct = tid - slice * cols;
    int mol = 0;
    int64_t t = blockIdx.x;
    if (a.tasks) {
        const int2 tk = a.tasks[blockIdx.x];
        mol = tk.x;
        t = tk.y;
    }
    const Rows64Mol &m = a.mols ? a.mols[mol] : a.mol;
    const int Nb = int(m.m.Nb), n = m.m.n, nn = n * n, nexa = m.m.nexa, nexb = m.m.nexb;
    const int chunks = m.chunks;
    const int64_t ar = m.row0 + t / chunks;
    const int ck = int(t % chunks);
    const int c0 = int(int64_t(Nb) * ck / chunks), c1 = int(int64_t(Nb) * (ck + 1) / chunks);
    const int b = c0 + ct;
    const bool act = b < c1;
    const double *psi = a.psi + m.m.offset;
    const RowsSmem s = rows_smem(smem_raw, slice, Nb, n);
    const uint32_t bm = act ? m.m.bstr[b] : 0u;
    const uint32_t am = m.m.astr[ar];
    double acc = 0.0, acc1 = 0.0;

    // alpha part: rows J of psi, coalesced; the table row is the same for all
    // threads of a slice
    if (act) {
        const int32_t *col = m.m.Ma_col;
        const double *val = m.m.Ma_val;
        const int p0 = m.m.Ma_ptr[ar], len = m.m.Ma_ptr[ar + 1] - p0;
        int k = p0 + len * slice / ES;
        const int k1 = p0 + len * (slice + 1) / ES;
        for (; k + 7 < k1; k += 8) {
            double x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = psi[int64_t(__ldg(col + k + i)) * Nb + b];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc = fma(__ldg(val + k + i), x[i], acc);
        }
        for (; k < k1; ++k) acc = fma(__ldg(val + k), psi[int64_t(__ldg(col + k)) * Nb + b], acc);
    }

    // groups of E alpha partners, the row itself (diagonal alpha part) first
    for (int e0 = -1; e0 < nexa; e0 += E) {
        const int ne = min(E, nexa - e0);
        __syncthreads();
        if (tid < ne) ent[tid] = e0 + tid < 0 ? uint32_t(ar) : m.m.aex[ar * nexa + e0 + tid];
        __syncthreads();
        // partner j: slice j / 2, component j % 2; the row itself goes to
        // component 0 of every slice's first group only where it is read (the
        // beta part below reads slice 0's)
        for (int j = 0; j < ne; ++j) {
            const bool diag = e0 + j < 0;
            const uint32_t u = ent[j];
            const double *src = psi + int64_t(diag ? ar : u & 0xFFFFu) * Nb;
            const RowsSmem d = rows_smem(smem_raw, j >> 1, Nb, n);
            double *R = reinterpret_cast<double *>(d.R) + (j & 1);
            double *C = reinterpret_cast<double *>(d.C) + (j & 1);
            for (int i = tid; i < Nb; i += nt) R[2 * i] = src[i];
            const uint32_t sb = diag ? 0u : u & 0x80000000u;
            const double *V = m.m.V + size_t(((u >> 16) & 15) * n + ((u >> 20) & 15)) * nn;
            for (int i = tid; i < nn; i += nt) {
                double v = 0.0;
                if (diag) {
                    for (uint32_t mm = am; mm; mm &= mm - 1) {
                        const int p = __ffs(mm) - 1;
                        v += m.m.V[size_t(p * n + p) * nn + i];
                    }
                } else {
                    v = flip_sign(V[i], sb);
                }
                C[2 * i] = v;
            }
        }
        __syncthreads();
        // diagonal beta tables of the group: entry m is the entry without m's
        // top bit plus that orbital's coefficient (level by level, one warp
        // per partner and half)
        for (int w = tid >> 5; w < 2 * ne; w += nt >> 5) {
            const int j = w >> 1, lane = tid & 31, hl = low_bits(n);
            const int bits = (w & 1) ? n - hl : hl, o = (w & 1) ? hl : 0;
            const RowsSmem d = rows_smem(smem_raw, j >> 1, Nb, n);
            double *T = reinterpret_cast<double *>((w & 1) ? d.TH : d.TL) + (j & 1);
            const double *C = reinterpret_cast<const double *>(d.C) + (j & 1);
            if (lane == 0) T[0] = 0.0;
            __syncwarp();
            for (int l = 0; l < bits; ++l) {
                const double c = C[2 * ((o + l) * n + o + l)];
                for (int i = lane; i < (1 << l); i += 32) T[2 * ((1 << l) + i)] = T[2 * i] + c;
                __syncwarp();
            }
        }
        __syncthreads();
        if (!act) continue;
        if (e0 < 0) {       // beta part, from the row itself (partner 0 of this group)
            const double2 *row = rows_smem(smem_raw, 0, Nb, n).R;
            const int len = m.m.Mb_ptr[b + 1] - m.m.Mb_ptr[b];
            const double *val = m.Mb_colv + b;
            const uint16_t *col = m.Mb_colc + b;
            int k = len * slice / ES;
            const int k1 = len * (slice + 1) / ES;
            for (; k + 3 < k1; k += 4) {
                double v[4];
                int c[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v[i] = __ldg(val + size_t(k + i) * Nb);
                    c[i] = __ldg(col + size_t(k + i) * Nb);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) acc = fma(v[i], row[c[i]].x, acc);
            }
            for (; k < k1; ++k)
                acc = fma(__ldg(val + size_t(k) * Nb), row[int(__ldg(col + size_t(k) * Nb))].x, acc);
        }
        // this slice's partners: both, or (last group) one or none
        const int mine = ne - 2 * slice;
        if (mine <= 0) continue;
        const int h = low_bits(n);
        const double2 tl = s.TL[bm & ((1u << h) - 1u)], th = s.TH[bm >> h], rb = s.R[b];
        const uint32_t *bx = m.m.bexT + b;
        acc = fma(tl.x + th.x, rb.x, acc);
        if (mine >= 2) {
            acc1 = fma(tl.y + th.y, rb.y, acc1);
#pragma unroll 4
            for (int f = 0; f < nexb; ++f) {
                const uint32_t u = __ldg(bx + size_t(f) * Nb);
                const uint32_t sb = u & 0x80000000u;
                const double2 c = s.C[((u >> 16) & 15) * n + ((u >> 20) & 15)], r = s.R[u & 0xFFFFu];
                acc = fma(flip_sign(c.x, sb), r.x, acc);
                acc1 = fma(flip_sign(c.y, sb), r.y, acc1);
            }
        } else {
#pragma unroll 4
            for (int f = 0; f < nexb; ++f) {
                const uint32_t u = __ldg(bx + size_t(f) * Nb);
                const double c = s.C[((u >> 16) & 15) * n + ((u >> 20) & 15)].x;
                acc = fma(flip_sign(c, u & 0x80000000u), s.R[u & 0xFFFFu].x, acc);
            }
        }
    }
    acc += acc1;
    if (ES > 1) {
        if (slice > 0) part[(slice - 1) * kRowsColsSmall + ct] = acc;
        __syncthreads();
        if (slice == 0)
            for (int i = 0; i < ES - 1; ++i) acc += part[i * kRowsColsSmall + ct];
    }
    if (act && slice == 0) a.sigma[m.m.offset + (ar - m.row0) * Nb + b] = acc;
    if (a.row_energy) {
        double v = act && slice == 0 ? acc * psi[ar * Nb + b] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        if (tid == 0) {
            double e = 0.0;
            for (int w = 0; w < (nt >> 5); ++w) e += red[w];
            a.row_energy[m.task_base + t] = e;
        }
    }
}

cudaError_t rows64(const Rows64Args &a, int64_t n_tasks, int slices, int cols, size_t smem,
                   cudaStream_t st)
{
    if (n_tasks <= 0) return cudaSuccess;
    auto run = [&](auto *kernel) {
        cudaError_t e = allow_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        kernel<<<unsigned(n_tasks), unsigned(slices * cols), smem, st>>>(a);
        hy::count_launch();
        return cudaGetLastError();
    };
    return slices == 1 ? run(k_rows64<1>) : run(k_rows64<kRowsSlices>);
}

// the beta CSR table by column: entry k of string b at [k][b]
__global__ void __launch_bounds__(256)
k_rows64_table(const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
               const double *__restrict__ val, int Nb, double *__restrict__ cv,
               uint16_t *__restrict__ cc)
{
    const int b = int((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5);
    if (b >= Nb) return;
    const int k0 = ptr[b], len = ptr[b + 1] - k0;
    for (int k = threadIdx.x & 31; k < len; k += 32) {
        cv[size_t(k) * Nb + b] = val[k0 + k];
        cc[size_t(k) * Nb + b] = uint16_t(col[k0 + k]);
    }
}

cudaError_t rows64_table(const int32_t *ptr, const int32_t *col, const double *val, int Nb,
                         double *cv, uint16_t *cc, cudaStream_t st)
{
    if (Nb <= 0) return cudaSuccess;
    k_rows64_table<<<unsigned((Nb + 7) / 8), 256, 0, st>>>(ptr, col, val, Nb, cv, cc);
    hy::count_launch();
    return cudaGetLastError();
}

}  // namespace k
}  // namespace hy
