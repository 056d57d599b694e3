// hy_dense.cu -- state preparation and ansatz gradient of a small dense state
// in one launch each.
//
// A dense evaluation of an ansatz of L operators is a chain of 2 L to 4 L pair
// rotations and L gradients, every one a pass over a few thousand pairs: as
// separate launches each costs 4 to 5 us whatever its size (63,504
// determinants: 85 launches an evaluation).  Here one cluster of kDenseCtas
// CTAs walks the whole chain, the cluster barrier (hardware, well below a
// microsecond) in the place of the launch boundary.  The vectors are spread
// over the CTAs' shared memories (up to kDenseMaxN determinants: psi, or phi
// and lambda, 4,096 amplitudes of each per CTA), partners read and written
// through distributed shared memory.
//
// Bound: the latency of a pass (pair, amplitudes, store, barrier).  Four
// evaluations of 12 operators at 20 qubits: 4,284 us with a launch per pass and
// one thread summing each gradient's chunks, 2,475 with that sum by a warp and
// H psi by rows, 1,631 with the chain in one launch on vectors in L2 (3 us a
// rotation), 1,340 on vectors in shared memory with the pairs of a pass dealt to
// all SMs (of which H psi 564).
#include <cooperative_groups.h>

#include "hy_kernels.cuh"

namespace cg = cooperative_groups;

namespace hy {
namespace k {

namespace {

constexpr int kDenseCtas = 16, kDenseThreads = 1024, kDenseAll = kDenseCtas * kDenseThreads;

// One step of the chain: a pass over the pairs (rr, t) of a constituent's
// alpha x beta pattern.
enum { kTerm = 1, kRotate = 2, kBarrier = 4 };      // barrier: after the pass
template <typename T>
struct DenseStep {
    const uint32_t *ae, *be;
    int rows, cols;
    T c, s;                  // cos theta, eps sin theta (of the rotation applied)
    int16_t eps, flags, op;
};

template <typename T>
__device__ __forceinline__ DenseStep<T> step_of(const DensePool &p, const ConsDev &cd, double c,
                                                double s, int op, int flags)
{
    DenseStep<T> r;
    r.ae = cd.ap < 0 ? nullptr : p.aent + p.aoff[cd.ap];
    r.be = cd.bp < 0 ? nullptr : p.bent + p.boff[cd.bp];
    r.rows = cd.ap < 0 ? p.Na : int(p.acnt[cd.ap]);
    r.cols = cd.bp < 0 ? p.Nb : int(p.bcnt[cd.bp]);
    r.c = T(c);
    r.s = T(double(cd.eps) * s);
    r.eps = int16_t(cd.eps);
    r.op = int16_t(op);
    r.flags = int16_t(flags);
    return r;
}

struct DensePair {
    int x, y;                // determinant and its image
    bool sa, sb;             // negative alpha / beta sign
};

template <typename T>
__device__ __forceinline__ DensePair pair_at(const DenseStep<T> &d, int idx, int Nb)
{
    const int rr = idx / d.cols, t = idx - rr * d.cols;
    const uint32_t u = d.ae ? __ldg(d.ae + rr) : uint32_t(rr) | (uint32_t(rr) << 15);
    const uint32_t v = d.be ? __ldg(d.be + t) : uint32_t(t) | (uint32_t(t) << 15);
    DensePair q;
    q.x = int(u & 0x7FFFu) * Nb + int(v & 0x7FFFu);
    q.y = int((u >> 15) & 0x7FFFu) * Nb + int((v >> 15) & 0x7FFFu);
    q.sa = u >> 31;
    q.sb = v >> 31;
    return q;
}

// a thread's place in a pass: warps dealt to the CTAs in turn, so that a pass of
// a few thousand pairs uses every SM's FP64 pipe
__device__ __forceinline__ int chain_thread(int rank)
{
    return (int(threadIdx.x >> 5) * kDenseCtas + rank) * 32 + int(threadIdx.x & 31);
}

// A thread's first pair of a step, its table entries loaded before the barrier
// that precedes the step.
template <typename T>
__device__ __forceinline__ DensePair first_pair(const DenseStep<T> &d, int g0, int Nb)
{
    return g0 < d.rows * d.cols ? pair_at(d, g0, Nb) : DensePair{0, 0, false, false};
}

// first step of every operator (nsteps of operator l from count(nc)); first
// has L + 1 entries; ends with a block barrier
template <typename F>
__device__ __forceinline__ void index_steps(const DensePool &p, const int32_t *ops, int L,
                                            int16_t *first, F count)
{
    for (int l = threadIdx.x; l < L; l += kDenseThreads) first[l + 1] = int16_t(count(p.opd[ops[l]].nc));
    __syncthreads();
    if (threadIdx.x == 0) {
        first[0] = 0;
        for (int l = 0; l < L; ++l) first[l + 1] = int16_t(first[l + 1] + first[l]);
    }
    __syncthreads();
}

// a vector over the cluster's shared memories: amplitude i in CTA i >> shift
template <typename T>
struct DenseVec {
    T *loc;
    int shift;
    __device__ __forceinline__ T &at(int i) const
    {
        return cg::this_cluster().map_shared_rank(loc, i >> shift)[i & ((1 << shift) - 1)];
    }
};

// the roundings of the per-rotation kernels, in float too: a b + c d as one
// multiplication and one fused multiply-add
__device__ __forceinline__ float mul_add2(float a, float b, float c, float d)
{
    return __fmaf_rn(a, b, __fmul_rn(c, d));
}
__device__ __forceinline__ double mul_add2(double a, double b, double c, double d)
{
    return fma(a, b, c * d);
}

template <typename T>
__device__ __forceinline__ void rotate(T &x, T &y, const DensePair &q, T c, T s_eps)
{
    T sg = s_eps;
    if (q.sa) sg = -sg;
    if (q.sb) sg = -sg;
    const T xv = x, yv = y;
    x = mul_add2(c, xv, -sg, yv);
    y = mul_add2(sg, xv, c, yv);
}

// sum of one double per thread over the cluster, in rank order, in every
// thread; red: 33 doubles
__device__ __forceinline__ double cluster_sum(cg::cluster_group &cl, double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kDenseThreads / 32; ++w) s += red[w];
        red[32] = s;
    }
    cl.sync();
    double s = 0.0;
    for (int r = 0; r < kDenseCtas; ++r) s += cl.map_shared_rank(red, r)[32];
    return s;
}

}  // namespace

// psi = U_L .. U_1 |HF>; float states divided by their FP64 norm, tracked
// through the rotations as in k_excite_n
template <typename T>
__global__ void __launch_bounds__(kDenseThreads, 1)
k_dense_prepare(DensePool p, const int32_t *__restrict__ ops, const double *__restrict__ cs, int L,
                T *__restrict__ psi, double *__restrict__ norm2, int shift)
{
    constexpr bool track = sizeof(T) == sizeof(float);
    extern __shared__ __align__(16) unsigned char dsm[];
    DenseStep<T> *steps = reinterpret_cast<DenseStep<T> *>(dsm);       // [2 L]
    const DenseVec<T> v{reinterpret_cast<T *>(steps + 2 * L), shift};
    cg::cluster_group cl = cg::this_cluster();
    __shared__ double red[33];
    __shared__ int16_t first[kDenseMaxOps + 1];
    const int g0 = chain_thread(int(cl.block_rank()));
    // this CTA's amplitudes [i0, i1)
    const int N = p.Na * p.Nb, i0 = min(N, int(cl.block_rank()) << shift);
    const int i1 = min(N, i0 + (1 << shift));
    for (int i = i0 + int(threadIdx.x); i < i1; i += kDenseThreads) v.loc[i - i0] = i == 0 ? T(1) : T(0);
    index_steps(p, ops, L, first, [](int nc) { return nc; });
    for (int l = threadIdx.x; l < L; l += kDenseThreads) {
        const OpDev od = p.opd[ops[l]];
        for (int q = 0; q < od.nc; ++q)
            steps[first[l] + q] = step_of<T>(p, p.cons[q == 0 ? od.c0 : od.c1], cs[2 * l],
                                             cs[2 * l + 1], l, kRotate | kBarrier);
    }
    __syncthreads();
    const int S = first[L];
    ProdAcc<T> acc;
    DensePair nxt = S > 0 ? first_pair(steps[0], g0, p.Nb) : DensePair{};
    cl.sync();
    for (int k = 0; k < S; ++k) {
        const DenseStep<T> &d = steps[k];
        for (int i = g0; i < d.rows * d.cols; i += kDenseAll) {
            const DensePair pr = i == g0 ? nxt : pair_at(d, i, p.Nb);
            T &vx = v.at(pr.x), &vy = v.at(pr.y);
            const T x = vx, y = vy;
            T nx = x, ny = y;
            rotate(nx, ny, pr, d.c, d.s);
            vx = nx;
            vy = ny;
            if (track) {
                acc.add(nx, nx);
                acc.add(ny, ny);
                acc.add(-x, x);
                acc.add(-y, y);
            }
        }
        if (k + 1 < S) nxt = first_pair(steps[k + 1], g0, p.Nb);
        cl.sync();
    }
    T f = T(1);
    if (track && L > 0) {
        const double n2 = 1.0 + cluster_sum(cl, acc.total(), red);
        if (g0 == 0) *norm2 = n2;
        f = T(1.0 / sqrt(n2));
        cl.sync();           // no CTA leaves while others may read its sum
    }
    for (int i = i0 + int(threadIdx.x); i < i1; i += kDenseThreads)
        psi[i] = track && L > 0 ? v.loc[i - i0] * f : v.loc[i - i0];
}

// dE/dtheta_l = 2 <lam_l | A_l phi_l>, phi and lam walked back from psi and
// sigma = H psi.  The constituents of an operator commute with one another, so
// in double a constituent's term is summed and both vectors rotated by it in
// one pass; in float all terms are taken before any rotation, each pair's term
// formed in float as k_grad_partial forms it (bit for bit: with one pair per
// thread and chunk there, its float partial sums are single terms).
template <typename T>
__global__ void __launch_bounds__(kDenseThreads, 1)
k_dense_gradient(DensePool p, const int32_t *__restrict__ ops, const double *__restrict__ cs, int L,
                 const T *__restrict__ psi, const T *__restrict__ sigma, double *__restrict__ g,
                 int shift)
{
    constexpr bool f32 = sizeof(T) == sizeof(float);
    extern __shared__ __align__(16) unsigned char dsm[];
    double *warp_g = reinterpret_cast<double *>(dsm);                          // [L][32]
    DenseStep<T> *steps = reinterpret_cast<DenseStep<T> *>(warp_g + size_t(L) * 32);   // [4 L]
    const DenseVec<T> phi{reinterpret_cast<T *>(steps + 4 * L), shift};
    const DenseVec<T> lam{phi.loc + (1 << shift), shift};
    cg::cluster_group cl = cg::this_cluster();
    __shared__ int16_t first[kDenseMaxOps + 1];
    const int rank = int(cl.block_rank()), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g0 = chain_thread(rank);
    const int N = p.Na * p.Nb, i0 = min(N, rank << shift), i1 = min(N, i0 + (1 << shift));
    for (int i = i0 + int(threadIdx.x); i < i1; i += kDenseThreads) {
        phi.loc[i - i0] = psi[i];
        lam.loc[i - i0] = sigma[i];
    }
    index_steps(p, ops, L, first, [](int nc) { return f32 && nc > 1 ? 2 * nc : nc; });
    const int S = first[L];
    for (int l = threadIdx.x; l < L; l += kDenseThreads) {
        const OpDev od = p.opd[ops[l]];
        const bool split = f32 && od.nc > 1;
        int k = S - first[l + 1];                    // the last operator goes first
        for (int pass = split ? 0 : 1; pass < 2; ++pass)
            for (int q = 0; q < od.nc; ++q) {
                int fl = pass == 0 ? kTerm : split ? kRotate : kTerm | kRotate;
                if (l == 0) fl &= ~kRotate;
                if (l > 0 && ((fl & kRotate) || q == od.nc - 1)) fl |= kBarrier;
                steps[k++] = step_of<T>(p, p.cons[q == 0 ? od.c0 : od.c1], cs[2 * l],
                                        -cs[2 * l + 1], l, fl);
            }
    }
    __syncthreads();
    DensePair nxt = S > 0 ? first_pair(steps[0], g0, p.Nb) : DensePair{};
    cl.sync();
    double tot = 0.0;
    for (int k = 0; k < S; ++k) {
        const DenseStep<T> &d = steps[k];
        const int fl = d.flags;
        if (fl & (kTerm | kRotate))
            for (int i = g0; i < d.rows * d.cols; i += kDenseAll) {
                const DensePair pr = i == g0 ? nxt : pair_at(d, i, p.Nb);
                T &fx = phi.at(pr.x), &fy = phi.at(pr.y), &gx = lam.at(pr.x), &gy = lam.at(pr.y);
                T px = fx, py = fy, lx = gx, ly = gy;
                if (fl & kTerm) {
                    const bool neg = (pr.sa != pr.sb) != (d.eps < 0);
                    if constexpr (f32) {
                        const double t = double(mul_add2(ly, px, -lx, py));
                        tot += neg ? -t : t;
                    } else {         // the FP64 pipe bounds the pass: two FMAs
                        tot = fma(neg ? -ly : ly, px, tot);
                        tot = fma(neg ? lx : -lx, py, tot);
                    }
                }
                if (fl & kRotate) {
                    rotate(px, py, pr, d.c, d.s);
                    rotate(lx, ly, pr, d.c, d.s);
                    fx = px;
                    fy = py;
                    gx = lx;
                    gy = ly;
                }
            }
        const int op = d.op;
        if (k + 1 < S) nxt = first_pair(steps[k + 1], g0, p.Nb);
        if (k + 1 == S || steps[k + 1].op != op) {
            for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
            if (lane == 0) warp_g[op * 32 + warp] = tot;
            tot = 0.0;
        }
        if (fl & kBarrier) cl.sync();
    }
    // warps in order, then the CTAs' sums in rank order
    __syncthreads();
    for (int l = threadIdx.x; l < L; l += kDenseThreads) {
        double s = 0.0;
        for (int w = 0; w < 32; ++w) s += warp_g[l * 32 + w];
        warp_g[l * 32] = s;
    }
    cl.sync();
    if (rank == 0)
        for (int l = threadIdx.x; l < L; l += kDenseThreads) {
            double s = 0.0;
            for (int r = 0; r < kDenseCtas; ++r) s += cl.map_shared_rank(warp_g, r)[l * 32];
            g[l] = 2.0 * s;
        }
    cl.sync();               // no CTA leaves while others may read its sums
}

// amplitudes per CTA as a power of two
int dense_shift(const DensePool &p)
{
    int s = 0;
    while ((int64_t(kDenseCtas) << s) < int64_t(p.Na) * p.Nb) ++s;
    return s;
}

namespace {
// one cluster of kDenseCtas CTAs (beyond the portable eight: opted into)
template <typename... P>
cudaError_t cluster_config(void (*kernel)(P...), size_t smem, cudaLaunchAttribute &at,
                           cudaLaunchConfig_t &cfg)
{
    cudaError_t e = allow_smem(kernel, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kDenseCtas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(kDenseCtas);
    cfg.blockDim = dim3(kDenseThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return e;
}

template <typename... P, typename... A>
cudaError_t launch_cluster(void (*kernel)(P...), size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg{};
    cudaError_t e = cluster_config(kernel, smem, at, cfg);
    if (e != cudaSuccess) return e;
    cfg.stream = st;
    e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    hy::count_launch();
    return e;
}

template <typename... P>
bool cluster_fits(void (*kernel)(P...), size_t smem)
{
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg{};
    int n = 0;
    if (cluster_config(kernel, smem, at, cfg) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess)
        return n > 0;
    cudaGetLastError();
    return false;
}

template <typename T>
size_t prepare_smem(int L, int shift)
{
    return size_t(L) * 2 * sizeof(DenseStep<T>) + (size_t(1) << shift) * sizeof(T);
}
template <typename T>
size_t gradient_smem(int L, int shift)
{
    return size_t(L) * (32 * sizeof(double) + 4 * sizeof(DenseStep<T>)) + (size_t(2) << shift) * sizeof(T);
}
}  // namespace

template <typename T>
bool dense_fits(int Na, int Nb)
{
    DensePool p{};
    p.Na = Na;
    p.Nb = Nb;
    const int shift = dense_shift(p);
    return cluster_fits(k_dense_prepare<T>, prepare_smem<T>(kDenseMaxOps, shift)) &&
           cluster_fits(k_dense_gradient<T>, gradient_smem<T>(kDenseMaxOps, shift));
}

template <typename T>
cudaError_t dense_prepare(const DensePool &p, const int32_t *ops, const double *cs, int L, T *psi,
                          double *norm2, cudaStream_t st)
{
    const int shift = dense_shift(p);
    return launch_cluster(k_dense_prepare<T>, prepare_smem<T>(L, shift), st, p, ops, cs, L, psi, norm2, shift);
}

template <typename T>
cudaError_t dense_gradient(const DensePool &p, const int32_t *ops, const double *cs, int L,
                           const T *psi, const T *sigma, double *g, cudaStream_t st)
{
    const int shift = dense_shift(p);
    return launch_cluster(k_dense_gradient<T>, gradient_smem<T>(L, shift), st, p, ops, cs, L, psi, sigma, g, shift);
}

template bool dense_fits<double>(int, int);
template bool dense_fits<float>(int, int);
template cudaError_t dense_prepare<double>(const DensePool &, const int32_t *, const double *, int,
                                           double *, double *, cudaStream_t);
template cudaError_t dense_prepare<float>(const DensePool &, const int32_t *, const double *, int,
                                          float *, double *, cudaStream_t);
template cudaError_t dense_gradient<double>(const DensePool &, const int32_t *, const double *, int,
                                            const double *, const double *, double *, cudaStream_t);
template cudaError_t dense_gradient<float>(const DensePool &, const int32_t *, const double *, int,
                                           const float *, const float *, double *, cudaStream_t);

}  // namespace k
}  // namespace hy
