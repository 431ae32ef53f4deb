// ik_field.cu -- field solve (a5): lap(phi) = -rho/eps0, E = -grad(phi).
//
// Sec. 4.3: finite-volume discretisation (the 3D standard stencil is the
// 7-point one) solved by geometric multigrid V-cycles with red-black
// Gauss-Seidel smoothing, exit at a relative residual of 1e-10.  Boundary
// conditions of Sec. 5.1: plane electrodes (Dirichlet, phi = 0 at z = lo,
// E0 L at z = hi; ghost 2 phi_b - phi_1) and homogeneous Neumann side faces
// (ghost = phi_1).  Cell-centred hierarchy down to 4^3: averaging
// restriction, trilinear cell-centred prolongation, and at the bottom red-black
// sweeps in FP32 or the level's eigenvectors in the 64-bit forms (the paper
// uses BiCGSTAB there).
//
// Two forms: V-cycles on the system in 64-bit fixed point (the FP64 form; with
// FP64 V-cycles where the integers' range does not serve), or FP32 V-cycles
// on the correction equation inside residual iterative refinement
// (phi += V32(b - A phi) until the residual meets the tolerance).
// Realizations are stacked (slowest index) and solved together; each has
// its own convergence test.  Norms are reduced in a fixed order.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <type_traits>

#include <cooperative_groups.h>

#include "../../include/itokmc.h"
#include "ik_common.cuh"
#include "ik_state.h"

namespace ik {

namespace {

namespace cg = cooperative_groups;

struct Geo {      // one level, all realizations
    int n, log2n, R;
    uint64_t cells;   // R n^3
};

__device__ __forceinline__ void decode(uint64_t t, int log2n, int& r, int& k, int& j, int& i)
{
    const int n = 1 << log2n;
    i = (int)(t & (uint64_t)(n - 1));
    j = (int)((t >> log2n) & (uint64_t)(n - 1));
    k = (int)((t >> (2 * log2n)) & (uint64_t)(n - 1));
    r = (int)(t >> (3 * log2n));
}

// Sum of interior neighbours and the diagonal count n_int + 2 n_D of the
// homogeneous operator at (k, j, i).
template <class T>
__device__ __forceinline__ T nbr_sum(const T* __restrict__ phi, uint64_t idx, int n, int i, int j, int k,
                                     int& diag)
{
    const uint64_t sy = (uint64_t)n, sz = (uint64_t)n * n;
    T s = 0;
    diag = 0;
    if (i > 0) { s = phi[idx - 1]; ++diag; }     // the sum starts at the first neighbour
    if (i < n - 1) { s += phi[idx + 1]; ++diag; }
    if (j > 0) { s += phi[idx - sy]; ++diag; }
    if (j < n - 1) { s += phi[idx + sy]; ++diag; }
    if (k > 0) { s += phi[idx - sz]; ++diag; } else diag += 2;
    if (k < n - 1) { s += phi[idx + sz]; ++diag; } else diag += 2;
    return s;
}

// diag as a T without a conversion instruction.
template <class T>
__device__ __forceinline__ T diag_val(int d)
{
    switch (d) {
    case 4: return (T)4;
    case 5: return (T)5;
    case 6: return (T)6;
    case 7: return (T)7;
    case 8: return (T)8;
    case 9: return (T)9;
    default: return (T)d;
    }
}

// 1/diag for the diagonal counts 4..9 (a multiply instead of a divide).
template <class T>
__device__ __forceinline__ T inv_diag(int d)
{
    if (d == 6) return (T)(1.0 / 6.0);
    return d == 5 ? (T)(1.0 / 5.0) : d == 7 ? (T)(1.0 / 7.0) : d == 4 ? (T)(1.0 / 4.0) : d == 8 ? (T)(1.0 / 8.0) : (T)(1.0 / 9.0);
}

// The arithmetic of the multigrid on values of type T.  float and double round
// each operation in the order written.  long long is the fixed-point form of
// the FP64 solve (see field_solve): sums are exact, the relaxed value and the
// interpolated correction are rounded to the nearest unit.  GB300 has 2 FP64
// lanes per SM and clock and 64 or more integer ones, so a relaxed cell costs
// about 30 integer instructions in the place of 7 FP64 ones that occupy the
// pipe for as long as 220.
template <class T>
struct MG {
    static __device__ __forceinline__ T relax(T sum, T rhs, int diag) { return (sum - rhs) * inv_diag<T>(diag); }
    static __device__ __forceinline__ T resid(T sum, T rhs, T phi, int diag) { return fma(diag_val<T>(diag), phi, rhs - sum); }
    static __device__ __forceinline__ T half(T acc) { return acc * (T)0.5; }
    static __device__ __forceinline__ T axpy3(T a, T b) { return fma((T)3, a, b); }
    static __device__ __forceinline__ T div64(T a) { return a * (T)(1.0 / 64.0); }
};
template <>
struct MG<long long> {
    // t / d to within a unit for |t| < 2^62: the product with floor(2^63 / d) =
    // mh 2^32 + ml (ml signed), without the product of the low halves
    static __device__ __forceinline__ long long mul(long long t, int mh, int ml)
    {
        const int th = (int)(t >> 32);
        const unsigned tl = (unsigned)t;
        const long long mid = (long long)th * ml + (long long)((unsigned long long)tl * (unsigned)mh);
        return (((long long)th * mh) << 1) + (mid >> 31);
    }
    static __device__ __forceinline__ void magic(int diag, int& mh, int& ml)
    {
        mh = diag == 6 ? 0x15555555 : diag == 5 ? 0x1999999a : diag == 7 ? 0x12492492
           : diag == 4 ? 0x20000000 : diag == 8 ? 0x10000000 : 0x0e38e38e;
        ml = diag == 6 ? 0x55555555 : diag == 5 ? -0x66666667 : diag == 7 ? 0x49249249 : diag == 9 ? 0x38e38e38 : 0;
    }
    static __device__ __forceinline__ long long relax(long long sum, long long rhs, int diag)
    {
        int mh, ml;
        magic(diag, mh, ml);
        return mul(sum - rhs + 3, mh, ml);
    }
    static __device__ __forceinline__ long long resid(long long sum, long long rhs, long long phi, int diag)
    {
        return rhs - sum + (long long)diag * phi;
    }
    static __device__ __forceinline__ long long half(long long acc) { return (acc + 1) >> 1; }
    static __device__ __forceinline__ long long axpy3(long long a, long long b) { return a + (a << 1) + b; }
    static __device__ __forceinline__ long long div64(long long a) { return (a + 32) >> 6; }
};

// A cell's divisor prepared for several relaxations.
template <class T>
struct Inv {
    T v;
    __device__ __forceinline__ Inv() {}
    __device__ __forceinline__ explicit Inv(int d) : v(inv_diag<T>(d)) {}
    static __device__ __forceinline__ Inv zero() { Inv i; i.v = (T)0; return i; }
    __device__ __forceinline__ T relax(T sum, T rhs) const { return (sum - rhs) * v; }
};
template <>
struct Inv<long long> {
    int mh, ml;
    __device__ __forceinline__ Inv() {}
    __device__ __forceinline__ explicit Inv(int d) { MG<long long>::magic(d, mh, ml); }
    static __device__ __forceinline__ Inv zero() { Inv i; i.mh = i.ml = 0; return i; }
    __device__ __forceinline__ long long relax(long long sum, long long rhs) const
    {
        return MG<long long>::mul(sum - rhs + 3, mh, ml);
    }
};

// Diagonal count of cell (i, j, k): 6, one less per Neumann side face, one
// more per electrode face.
__device__ __forceinline__ int diag_count(int i, int j, int k, int n)
{
    return 6 - (i == 0) - (i == n - 1) - (j == 0) - (j == n - 1) + (k == 0) + (k == n - 1);
}

template <class T>
__global__ void k_smooth(T* __restrict__ phi, const T* __restrict__ rhs, Geo G, int color)
{
    const uint64_t half = G.cells >> 1;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < half; t += (uint64_t)gridDim.x * blockDim.x) {
        // t enumerates (r, k, j, ih); i = 2 ih + parity
        const int n = G.n;
        const int ih = (int)(t & (uint64_t)(n / 2 - 1));
        const int j = (int)((t >> (G.log2n - 1)) & (uint64_t)(n - 1));
        const int k = (int)((t >> (2 * G.log2n - 1)) & (uint64_t)(n - 1));
        const uint64_t r = t >> (3 * G.log2n - 1);
        const int i = 2 * ih + ((j + k + color) & 1);
        const uint64_t idx = ((r * n + k) * n + j) * n + i;
        int diag;
        const T s = nbr_sum(phi, idx, n, i, j, k, diag);
        phi[idx] = MG<T>::relax(s, rhs[idx], diag);
    }
}

// Residual at fine cells, averaged over the 8 children of each coarse cell
// into the coarse right-hand side.  Every level stores h^2 b (the multigrid
// systems are scaled by h^2), so the coarse value h_c^2 mean(r) is half the
// sum of the children's h_f^2 r = h_f^2 b - (neighbour sum - diag phi).
// A thread reads its 2 x 2 x 2 cells and their rim by rows of pairs: 12 pairs
// and 8 single values for eight residuals.
template <class T>
struct __align__(2 * sizeof(T)) Pair { T v[2]; };

template <class T>
__global__ void __launch_bounds__(256) k_resid_restrict(const T* __restrict__ phi, const T* __restrict__ rhs,
                                                        T* __restrict__ rhs_c, Geo Gc, int nf)
{
    const int nc = Gc.n;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < Gc.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, K, J, I;
        decode(t, Gc.log2n, r, K, J, I);
        const uint64_t sy = (uint64_t)nf, sz = (uint64_t)nf * nf;
        const T* p = phi + ((uint64_t)r * nf + 2 * K) * sz + (2 * J) * sy + 2 * I;
        const T* b = rhs + (p - phi);
        auto row = [&](int k, int j, bool in) {    // the x pair of plane k, row j from the thread's own
            Pair<T> v;
            v.v[0] = v.v[1] = (T)0;
            if (in) v = *reinterpret_cast<const Pair<T>*>(p + (int64_t)k * (int64_t)sz + (int64_t)j * (int64_t)sy);
            return v;
        };
        const bool xl = I > 0, xr = I < nc - 1, yl = J > 0, yr = J < nc - 1, zl = K > 0, zr = K < nc - 1;
        // own pairs with a row before and after, per plane; the planes before and after
        Pair<T> v[4][4];
#pragma unroll
        for (int k = -1; k <= 2; ++k)
#pragma unroll
            for (int j = -1; j <= 2; ++j) {
                const bool edge_k = k < 0 || k > 1, edge_j = j < 0 || j > 1;
                if (edge_k && edge_j) continue;
                v[k + 1][j + 1] = row(k, j, (k >= 0 || zl) && (k <= 1 || zr) && (j >= 0 || yl) && (j <= 1 || yr));
            }
        T acc = 0;
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint64_t o = (uint64_t)k * sz + (uint64_t)j * sy;
                const Pair<T> c = v[k + 1][j + 1], f = *reinterpret_cast<const Pair<T>*>(b + o);
                const T left = xl ? p[o - 1] : (T)0, right = xr ? p[o + 2] : (T)0;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    T s = (x ? c.v[0] : left) + (x ? right : c.v[1]);      // a side without a cell adds zero
                    s += v[k + 1][j].v[x];
                    s += v[k + 1][j + 2].v[x];
                    s += v[k][j + 1].v[x];
                    s += v[k + 2][j + 1].v[x];
                    acc += MG<T>::resid(s, f.v[x], c.v[x], diag_count(2 * I + x, 2 * J + j, 2 * K + k, nf));
                }
            }
        rhs_c[t] = MG<T>::half(acc);
    }
}

// phi_f += trilinear cell-centred interpolation of the coarse correction:
// weights 3/4, 1/4 per axis written as (3 a + b) / 4 with fused multiply-
// adds (ghosts: Neumann e, Dirichlet -e, i.e. (3 a - a) / 4 in z).
template <class T>
__device__ __forceinline__ T prolong_at(const T* __restrict__ ec, int nc, int i, int j, int k)
{
    const int I = i >> 1, J = j >> 1, K = k >> 1;
    int I2 = I + ((i & 1) ? 1 : -1), J2 = J + ((j & 1) ? 1 : -1), K2 = K + ((k & 1) ? 1 : -1);
    T sz = (T)1;
    if (I2 < 0 || I2 >= nc) I2 = I;
    if (J2 < 0 || J2 >= nc) J2 = J;
    if (K2 < 0 || K2 >= nc) { K2 = K; sz = (T)-1; }
    const int iz[2] = { K, K2 }, iy[2] = { J, J2 };
    T m[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        T q[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const T* row = ec + ((int64_t)iz[c] * nc + iy[b]) * nc;
            q[b] = MG<T>::axpy3(row[I], row[I2]);
        }
        m[c] = MG<T>::axpy3(q[0], q[1]);
    }
    return MG<T>::div64(MG<T>::axpy3(m[0], sz < (T)0 ? -m[1] : m[1]));
}

// A thread takes the x pair (2 I, 2 I + 1) of rows 2 J and 2 J + 1 of plane k:
// three coarse values in each of 2 x 3 rows serve four cells (eight loads and
// index computations per cell otherwise).  Each cell gets prolong_at's
// operations.
template <class T>
__global__ void __launch_bounds__(256) k_prolong(T* __restrict__ phi_f, const T* __restrict__ e_c, Geo Gf)
{
    const int n = Gf.n, nc = n / 2, lc = Gf.log2n - 1;
    const uint64_t groups = Gf.cells >> 2;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < groups; t += (uint64_t)gridDim.x * blockDim.x) {
        const int I = (int)(t & (uint64_t)(nc - 1)), J = (int)((t >> lc) & (uint64_t)(nc - 1));
        const int k = (int)((t >> (2 * lc)) & (uint64_t)(n - 1));
        const uint64_t r = t >> (2 * lc + Gf.log2n);
        const int K = k >> 1;
        int K2 = K + ((k & 1) ? 1 : -1);
        bool neg = false;
        if (K2 < 0 || K2 >= nc) { K2 = K; neg = true; }
        const int Il = I > 0 ? I - 1 : I, Ir = I < nc - 1 ? I + 1 : I;
        const int Jl = J > 0 ? J - 1 : J, Jr = J < nc - 1 ? J + 1 : J;
        T m[2][2][2];                              // [plane][fine row][cell]
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const T* pl = e_c + (r * nc + (c ? K2 : K)) * (uint64_t)nc * nc;
            const T *r0 = pl + J * nc, *rl = pl + Jl * nc, *rr = pl + Jr * nc;
            const T a = r0[I], al = r0[Il], ar = r0[Ir];
            const T b = rl[I], bl = rl[Il], br = rl[Ir];
            const T d = rr[I], dl = rr[Il], dr = rr[Ir];
            const T q0 = MG<T>::axpy3(a, al), q1 = MG<T>::axpy3(a, ar);
            m[c][0][0] = MG<T>::axpy3(q0, MG<T>::axpy3(b, bl));
            m[c][0][1] = MG<T>::axpy3(q1, MG<T>::axpy3(b, br));
            m[c][1][0] = MG<T>::axpy3(q0, MG<T>::axpy3(d, dl));
            m[c][1][1] = MG<T>::axpy3(q1, MG<T>::axpy3(d, dr));
        }
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            Pair<T>* p = reinterpret_cast<Pair<T>*>(phi_f + ((r * n + k) * n + 2 * J + y) * (uint64_t)n + 2 * I);
            Pair<T> v = *p;
#pragma unroll
            for (int x = 0; x < 2; ++x) v.v[x] += MG<T>::div64(MG<T>::axpy3(m[0][y][x], neg ? -m[1][y][x] : m[1][y][x]));
            *p = v;
        }
    }
}

// The same with kp fine planes per thread, from the bottom up: a coarse plane's
// interpolation is formed once for the two fine planes on either side.
template <class T>
__global__ void __launch_bounds__(256) k_prolong_march(T* __restrict__ phi_f, const T* __restrict__ e_c, Geo Gf, int kp)
{
    const int n = Gf.n, nc = n / 2, lc = Gf.log2n - 1;
    const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const int I = (int)(t & (uint64_t)(nc - 1)), J = (int)((t >> lc) & (uint64_t)(nc - 1));
    const uint64_t z = (t >> (2 * lc)) * (uint64_t)kp, r = z >> Gf.log2n;      // first plane over all realizations
    if (z >= Gf.cells >> (2 * Gf.log2n)) return;
    const int k0 = (int)(z & (uint64_t)(n - 1));
    const int il = I > 0 ? -1 : 0, ir = I < nc - 1 ? 1 : 0;
    const int64_t jl = J > 0 ? -nc : 0, jr = J < nc - 1 ? nc : 0;
    struct M { T v[2][2]; };                       // in-plane interpolation: [fine row][cell]
    auto plane = [&](int K, M& m) {                // ghosts beyond the electrodes: the outermost plane, negated
        const bool neg = K < 0 || K >= nc;
        const int Kc = K < 0 ? 0 : (K >= nc ? nc - 1 : K);
        const T *r0 = e_c + ((r * nc + Kc) * (uint64_t)nc + J) * (uint64_t)nc + I, *rl = r0 + jl, *rr = r0 + jr;
        const T a = r0[0], al = r0[il], ar = r0[ir];
        const T b = rl[0], bl = rl[il], br = rl[ir];
        const T d = rr[0], dl = rr[il], dr = rr[ir];
        const T q0 = MG<T>::axpy3(a, al), q1 = MG<T>::axpy3(a, ar);
        m.v[0][0] = MG<T>::axpy3(q0, MG<T>::axpy3(b, bl));
        m.v[0][1] = MG<T>::axpy3(q1, MG<T>::axpy3(b, br));
        m.v[1][0] = MG<T>::axpy3(q0, MG<T>::axpy3(d, dl));
        m.v[1][1] = MG<T>::axpy3(q1, MG<T>::axpy3(d, dr));
        if (neg)
#pragma unroll
            for (int q = 0; q < 4; ++q) m.v[q >> 1][q & 1] = -m.v[q >> 1][q & 1];
    };
    T* f = phi_f + (z * (uint64_t)n + 2 * J) * (uint64_t)n + 2 * I;
    M own, oth;                                    // plane k's coarse plane and the one beside it
    plane(k0 >> 1, own);
    plane((k0 >> 1) + ((k0 & 1) ? 1 : -1), oth);
    for (int k = k0;; ++k, f += (int64_t)n * n) {
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            Pair<T>* p = reinterpret_cast<Pair<T>*>(f + y * n);
            Pair<T> v = *p;
#pragma unroll
            for (int x = 0; x < 2; ++x) v.v[x] += MG<T>::div64(MG<T>::axpy3(own.v[y][x], oth.v[y][x]));
            *p = v;
        }
        if (k + 1 == k0 + kp) break;
        if (k & 1) {
            const M m = own;
            own = oth;
            oth = m;
        } else {
            plane((k >> 1) + 1, oth);
        }
    }
}

// FP64 residual, its squared norm per block (fixed order), and optionally
// the FP32 copy for the inner V-cycle.  A block covers items*256 cells of
// one realization.
constexpr int NORM_TPB = 256;

__global__ void __launch_bounds__(NORM_TPB) k_resid_norm(const double* __restrict__ phi, const double* __restrict__ rhs,
                                                         float* __restrict__ r32, Geo G,
                                                         double* __restrict__ part, int with_b, int items)
{
    __shared__ double red[NORM_TPB / 32][2];
    const uint64_t base = ((uint64_t)blockIdx.x * NORM_TPB) * items;
    double acc = 0.0, bacc = 0.0;
    for (int q = 0; q < items; ++q) {
        const uint64_t t = base + (uint64_t)q * NORM_TPB + threadIdx.x;
        if (t >= G.cells) break;
        int r, k, j, i;
        decode(t, G.log2n, r, k, j, i);
        int diag;
        const double s = nbr_sum(phi, t, G.n, i, j, k, diag);
        const double res = rhs[t] - (s - (double)diag * phi[t]);
        if (r32) r32[t] = (float)res;
        acc = __fma_rn(res, res, acc);
        if (with_b) bacc = __fma_rn(rhs[t], rhs[t], bacc);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, d);
        bacc += __shfl_xor_sync(0xffffffffu, bacc, d);
    }
    if ((threadIdx.x & 31) == 0) { red[threadIdx.x >> 5][0] = acc; red[threadIdx.x >> 5][1] = bacc; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < NORM_TPB / 32; ++w) { a += red[w][0]; b += red[w][1]; }
        part[2 * (uint64_t)blockIdx.x] = a;
        part[2 * (uint64_t)blockIdx.x + 1] = b;
    }
}

// Per realization (one block each): fixed-order strided sums, then a fixed
// tree in shared memory -- the same result on every run.  fs (FP64 form): the
// largest |Phi| of the check is closed.
__global__ void __launch_bounds__(256) k_norm_final(const double* __restrict__ part, int blocks_per_real, int R,
                                                    double* __restrict__ out, FixScale* __restrict__ fs = nullptr)
{
    __shared__ double sa[256], sb[256];
    const int r = blockIdx.x;
    double a = 0.0, b = 0.0;
    for (int q = threadIdx.x; q < blocks_per_real; q += 256) {
        a += part[2 * ((uint64_t)r * blocks_per_real + q)];
        b += part[2 * ((uint64_t)r * blocks_per_real + q) + 1];
    }
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            sa[threadIdx.x] += sa[threadIdx.x + w];
            sb[threadIdx.x] += sb[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[2 * r] = sa[0];
        out[2 * r + 1] = sb[0];
        if (fs) {
            fs[r].seen = fs[r].max_fix;
            fs[r].max_fix = 0;
        }
    }
}

__global__ void k_add_correction(double* __restrict__ phi, const float* __restrict__ e, uint64_t cells)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cells; t += (uint64_t)gridDim.x * blockDim.x)
        phi[t] += (double)e[t];
}

// ---- fixed-point potential (mixed field form)
// The potential is held as Phi = phi 2^F (int64) and the right-hand side as
// B = round(h^2 2^F b), so the residual h^2 2^F (b - A phi) = B - (sum of
// neighbours - diag Phi) is exact integer arithmetic (FP64 runs at a small
// fraction of the integer rate on GB300).  The FP32 residual r = R 2^-F / h^2
// feeds the FP32 correction V-cycles; squared norms are summed in FP32 per
// thread and FP64 across the block in a fixed order.
constexpr long long PHI_LIM = 1ll << 59;

// The cells of one block: a column of TX x TY cells over ZC planes of one
// realization, one (x, y) per thread, marching up in z with the planes below
// and at the cell in registers; the row's and the next rows' values were just
// loaded by the block (a block of consecutive cells reads three planes from L2
// for each one).
struct MarchGeo {
    int tx, log2tx, zc;          // x cells of a block (a power of two), planes of a block
    int bx, bxy, bpr;            // blocks per row of blocks, per plane of blocks, per realization
};

__host__ __device__ inline MarchGeo march_geo(int n)
{
    MarchGeo m;
    m.tx = n < 64 ? n : 64;
    m.log2tx = 0;
    while ((1 << m.log2tx) < m.tx) ++m.log2tx;
    const int ty = NORM_TPB / m.tx < n ? NORM_TPB / m.tx : n;
    m.zc = n <= 64 ? 4 : 16;     // small grids: more blocks rather than longer marches
    m.bx = n / m.tx;
    m.bxy = m.bx * (n / ty);
    m.bpr = m.bxy * (n / m.zc);
    return m;
}

// Calls f(cell index, value, neighbour sum, diagonal) for the thread's cells.
template <class F>
__device__ __forceinline__ void march_cells(const long long* __restrict__ Phi, int n, const MarchGeo& m, F f)
{
    const int ty = NORM_TPB / m.tx < n ? NORM_TPB / m.tx : n;
    const int r = blockIdx.x / m.bpr, b = blockIdx.x - r * m.bpr, bz = b / m.bxy, bb = b - bz * m.bxy, by = bb / m.bx,
              bx = bb - by * m.bx;
    const int row = threadIdx.x >> m.log2tx;
    if (row >= ty) return;
    const int i = bx * m.tx + (threadIdx.x & (m.tx - 1)), j = by * ty + row, k0 = bz * m.zc;
    const int64_t sy = n, sz = (int64_t)n * n;
    uint64_t t = (uint64_t)r * n * sz + (uint64_t)k0 * sz + (uint64_t)j * sy + i;
    const int dxy = 6 - (i == 0) - (i == n - 1) - (j == 0) - (j == n - 1);
    long long below = k0 > 0 ? Phi[t - sz] : 0, own = Phi[t];
#pragma unroll 2
    for (int q = 0; q < m.zc; ++q, t += sz) {
        const int k = k0 + q;
        const long long above = k < n - 1 ? Phi[t + sz] : 0;
        const long long xm = i > 0 ? Phi[t - 1] : 0, xp = i < n - 1 ? Phi[t + 1] : 0;
        const long long ym = j > 0 ? Phi[t - sy] : 0, yp = j < n - 1 ? Phi[t + sy] : 0;
        f(t, own, (xm + xp + ym) + (yp + below + above), dxy + (k == 0) + (k == n - 1));
        below = own;
        own = above;
    }
}

__global__ void __launch_bounds__(NORM_TPB) k_resid_fixed(const long long* __restrict__ Phi,
                                                          const long long* __restrict__ B, float* __restrict__ r32,
                                                          Geo G, float sc, double* __restrict__ part, int with_b,
                                                          MarchGeo m)
{
    __shared__ double red[NORM_TPB / 32][2];
    float acc = 0.f, bacc = 0.f;
    bool bad = false;
    march_cells(Phi, G.n, m, [&](uint64_t t, long long pc, long long s, int diag) {
        bad |= pc >= PHI_LIM || pc <= -PHI_LIM;
        const long long b = B[t];
        const float res = __ll2float_rn(MG<long long>::resid(s, b, pc, diag)) * sc;
        r32[t] = res;
        acc = __fmaf_rn(res, res, acc);
        if (with_b) {
            const float bf = __ll2float_rn(b) * sc;
            bacc = __fmaf_rn(bf, bf, bacc);
        }
    });
    double a = bad ? (double)INFINITY : (double)acc, bb = (double)bacc;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, d);
        bb += __shfl_xor_sync(0xffffffffu, bb, d);
    }
    if ((threadIdx.x & 31) == 0) { red[threadIdx.x >> 5][0] = a; red[threadIdx.x >> 5][1] = bb; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double x = 0.0, y = 0.0;
        for (int w = 0; w < NORM_TPB / 32; ++w) { x += red[w][0]; y += red[w][1]; }
        part[2 * (uint64_t)blockIdx.x] = x;
        part[2 * (uint64_t)blockIdx.x + 1] = y;
    }
}

// Phi += round(e 2^F) for the FP32 correction e (volts).
__global__ void k_add_fixed(long long* __restrict__ Phi, const float* __restrict__ e, float scale, uint64_t cells)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cells; t += (uint64_t)gridDim.x * blockDim.x)
        Phi[t] += __float2ll_rn(e[t] * scale);
}

// E = -grad(phi) from the fixed-point potential: the neighbour differences
// are exact integers, scaled by 2^-F / 2h (FP64 into E64 and/or FP32 into E32).
__global__ void k_efield_fixed(const long long* __restrict__ Phi, E64* __restrict__ E, float4* __restrict__ E32,
                               Geo G, double sc, long long Phi_top)
{
    const float scf = (float)sc;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, k, j, i;
        decode(t, G.log2n, r, k, j, i);
        const int n = G.n;
        const uint64_t sy = (uint64_t)n, sz = (uint64_t)n * n;
        const long long c = Phi[t];
        const long long xm = i > 0 ? Phi[t - 1] : c, xp = i < n - 1 ? Phi[t + 1] : c;
        const long long ym = j > 0 ? Phi[t - sy] : c, yp = j < n - 1 ? Phi[t + sy] : c;
        const long long zm = k > 0 ? Phi[t - sz] : -c, zp = k < n - 1 ? Phi[t + sz] : 2 * Phi_top - c;
        if (E) {
            const double ex = (double)(xm - xp) * sc, ey = (double)(ym - yp) * sc, ez = (double)(zm - zp) * sc;
            const double m = sqrt((ex * ex + ey * ey) + ez * ez);
            reinterpret_cast<double2*>(E + t)[0] = make_double2(ex, ey);
            reinterpret_cast<double2*>(E + t)[1] = make_double2(ez, m);
            if (E32) E32[t] = make_float4((float)ex, (float)ey, (float)ez, (float)m);
        } else {
            const float ex = __ll2float_rn(xm - xp) * scf, ey = __ll2float_rn(ym - yp) * scf,
                        ez = __ll2float_rn(zm - zp) * scf;
            E32[t] = make_float4(ex, ey, ez, sqrtf(ex * ex + ey * ey + ez * ez));
        }
    }
}

// ---- the FP64 form's fixed-point cycles
// The FP64 solve runs its V-cycles on 64-bit integers: Phi = phi 2^F and B =
// h^2 b 2^F, |Phi| below 2^57 (2^-57 of the bound on |phi|, FP64 keeps 2^-53
// of the value), with the relaxations, residuals and transfers of MG<long
// long>.  The potential is FP64 before and after (the start guess, the
// checkpoint, itokmc_read_densities).  Each realization has its own scale: a
// member of a batch keeps its bits beside one of a far higher potential.
// FIX_LIM marks an iterate that left its range: the solve then goes on with
// FP64 cycles.  Sums, residuals and relaxations hold for |Phi| below it; the
// interpolation forms 64 times a correction and holds for corrections below
// 2^57, which the scales leave room for: guess and solution are at most half of
// a bound below 2^57 each.  A correction beyond that (a cycle that overshoots, a
// step whose potential grows more than fivefold) wraps, and the next check finds
// a residual that has not fallen.
constexpr long long FIX_LIM = 1ll << 59;

// The bits by which a scale can go up that a loose bound (k_fix_scale) left too
// low: the largest |Phi| (seen) holds fewer bits than a double.  It goes to [2^55,
// 2^56); B (from max_b) and the electrode stay below 2^60 and 2^58.
constexpr int FIX_BITS = 53;
__host__ __device__ inline int lead_bit(unsigned long long v)
{
    int l = 0;
    while ((v >> l) > 1) ++l;
    return l;
}
__host__ __device__ inline int fix_shift(const FixScale& f)
{
    if (f.seen == 0 || f.seen >= (1ull << FIX_BITS)) return 0;
    if (f.max_b == 0 && f.top == 0) return 0;      // no charge and no applied field: the guess decays to zero
    int sh = 55 - lead_bit(f.seen);
    const int eb = (int)(f.max_b >> 52) - 1023 + f.F;          // |B| < 2^(eb + 1)
    if (f.max_b && sh > 58 - eb) sh = 58 - eb;
    const int et = lead_bit((unsigned long long)(f.top < 0 ? -f.top : f.top));
    if (f.top && sh > 56 - et) sh = 56 - et;
    return sh > 0 ? sh : 0;
}

// x 2^F rounded to the nearest integer, |x| 2^F < 2^62, by integer steps.
__device__ __forceinline__ long long to_fixed(double x, int F)
{
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;                                       // zero (or subnormal)
    const long long m = (b & 0xfffffffffffffll) | (1ll << 52);
    const int sh = e - 1075 + F;
    const long long v = sh >= 0 ? m << sh : (sh < -54 ? 0ll : (m + (1ll << (-sh - 1))) >> -sh);
    return b < 0 ? -v : v;
}

// The start guess (extrapolated in time when asked) and the largest |guess|
// and |h^2 b| (the electrode's share of the top layer's b taken out), as the
// bits of the non-negative doubles.  Block row r: realization r.
__global__ void __launch_bounds__(256) k_fix_start(double* __restrict__ phi, double* __restrict__ prev, int extrapolate,
                                                   int have, const double* __restrict__ rhs, Geo G, double bc,
                                                   FixScale* __restrict__ fs)
{
    unsigned long long mp = 0, mb = 0;
    const uint64_t n3 = 1ull << (3 * G.log2n), o = blockIdx.y * n3;
    fs += blockIdx.y;
    phi += o;
    rhs += o;
    if (prev) prev += o;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < n3; t += (uint64_t)gridDim.x * blockDim.x) {
        double v = phi[t];
        if (extrapolate) {
            const double old = v;
            if (have) {
                v = (v + v) - prev[t];
                phi[t] = v;
            }
            prev[t] = old;
        }
        double b = rhs[t];
        if ((t >> (2 * G.log2n)) == (uint64_t)(G.n - 1)) b += bc;
        const unsigned long long vb = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull,
                                 bb = (unsigned long long)__double_as_longlong(b) & 0x7fffffffffffffffull;
        mp = vb > mp ? vb : mp;
        mb = bb > mb ? bb : mb;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, mp, d), c = __shfl_xor_sync(0xffffffffu, mb, d);
        mp = a > mp ? a : mp;
        mb = c > mb ? c : mb;
    }
    __shared__ unsigned long long sp[8], sb[8];
    if ((threadIdx.x & 31) == 0) { sp[threadIdx.x >> 5] = mp; sb[threadIdx.x >> 5] = mb; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            mp = sp[w] > mp ? sp[w] : mp;
            mb = sb[w] > mb ? sb[w] : mb;
        }
        atomicMax(&fs->max_phi, mp);
        atomicMax(&fs->max_b, mb);
    }
}

// The scale of each realization.  Mc bounds |phi| of the solution: electrode
// potential plus the 1D Dirichlet bound max|h^2 b| n^2 / 8, doubled.  A guess
// extrapolated from the last steps is near the solution: four times its modulus
// bounds it (Mc is loose by orders of magnitude for a localised charge; a single
// cell's potential is about a quarter of its |h^2 b|, so that at least FIX_BITS
// bits hold it).  near: 1 unless the guess is so far below the bound that the
// charge may be another one (a looser scale is raised after the first cycle), 2 in
// any case (replayed steps, whose scale stays).  use64: the guess is not finite or
// far above the solution.
__global__ void k_fix_scale(FixScale* fs, int R, double phi_top, int n, int near, int rescale)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    fs += r;
    if (rescale == 2) fs->seen = fs->max_fix;                   // of k_fix_max
    fs->sh = rescale ? fix_shift(*fs) : 0;
    if (rescale) {                                              // of a running solve
        fs->F += fs->sh;
    } else {
        const double mp = __longlong_as_double((long long)fs->max_phi), mb = __longlong_as_double((long long)fs->max_b);
        const double Mc = 2.0 * (fabs(phi_top) + mb * (double)n * (double)n / 8.0);
        double M = near && mp > 0.0 && (near == 2 || mp * 16384.0 >= Mc) ? fmin(Mc, fmax(4.0 * mp, 2.0 * (mb + fabs(phi_top)))) : fmax(Mc, 2.0 * mp);
        M = fmax(M, 0x1p-400);
        fs->use64 = !(mp <= 16.0 * Mc) || !(Mc < 0x1p400);
        if (!(M < 0x1p400)) M = 1.0;
        fs->F = 57 - (ilogb(M) + 1);
    }
    fs->max_fix = 0;
    fs->down = scalbn(1.0, -fs->F);
    fs->top = to_fixed(phi_top, fs->F);
}

// The largest |Phi|.  Block row r: realization r.
__global__ void __launch_bounds__(256) k_fix_max(const long long* __restrict__ Phi, uint64_t n3, FixScale* __restrict__ fs)
{
    const uint64_t o = blockIdx.y * n3;
    unsigned long long mx = 0;
    for (uint64_t t = o + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < o + n3; t += (uint64_t)gridDim.x * blockDim.x) {
        const long long v = Phi[t];
        const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
        mx = a > mx ? a : mx;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, mx, d);
        mx = a > mx ? a : mx;
    }
    __shared__ unsigned long long sm[8];
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) mx = sm[w] > mx ? sm[w] : mx;
        atomicMax(&fs[blockIdx.y].max_fix, mx);
    }
}

// Phi and B from phi and the right-hand side; rescale: Phi shifted up by sh
// bits and B formed again at the new scale.  Block row r: realization r.
__global__ void k_fix_load(const double* __restrict__ phi, const double* __restrict__ rhs, long long* __restrict__ Phi,
                           long long* __restrict__ B, uint64_t n3, const FixScale* __restrict__ fs, int rescale)
{
    fs += blockIdx.y;
    const int F = fs->F, sh = fs->sh;
    if (fs->use64 || (rescale && sh == 0)) return;
    const uint64_t o = blockIdx.y * n3;
    for (uint64_t t = o + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < o + n3; t += (uint64_t)gridDim.x * blockDim.x) {
        Phi[t] = rescale ? Phi[t] << sh : to_fixed(phi[t], F);
        B[t] = to_fixed(rhs[t], F);
    }
}

// The potential back in FP64.  Block row r: realization r.
__global__ void k_fix_store(const long long* __restrict__ Phi, double* __restrict__ phi, uint64_t n3,
                            const FixScale* __restrict__ fs)
{
    const double sc = fs[blockIdx.y].down;
    const uint64_t o = blockIdx.y * n3;
    for (uint64_t t = o + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < o + n3; t += (uint64_t)gridDim.x * blockDim.x)
        phi[t] = (double)Phi[t] * sc;
}

// Squared norms of the exact integer residual and of B in FP64, summed in the
// order of k_resid_fixed, and the largest |Phi|.  The norms decide where the
// cycles end.
__global__ void __launch_bounds__(NORM_TPB) k_resid_norm_fix(const long long* __restrict__ Phi,
                                                             const long long* __restrict__ B, Geo G,
                                                             double* __restrict__ part, int with_b, MarchGeo m,
                                                             FixScale* __restrict__ fs)
{
    __shared__ double red[NORM_TPB / 32][2];
    __shared__ unsigned long long redm[NORM_TPB / 32];
    double acc = 0.0, bb = 0.0;
    unsigned long long mx = 0;
    fs += blockIdx.x / m.bpr;
    march_cells(Phi, G.n, m, [&](uint64_t t, long long pc, long long s, int diag) {
        const long long b = B[t];
        const unsigned long long ap = (unsigned long long)(pc < 0 ? -pc : pc);
        mx = ap > mx ? ap : mx;
        const double res = __ll2double_rn(MG<long long>::resid(s, b, pc, diag));
        acc = __fma_rn(res, res, acc);
        if (with_b) {
            const double bf = __ll2double_rn(b);
            bb = __fma_rn(bf, bf, bb);
        }
    });
    double a = fs->use64 || mx >= (unsigned long long)FIX_LIM ? (double)INFINITY : acc;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, d);
        bb += __shfl_xor_sync(0xffffffffu, bb, d);
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, d);
        mx = o > mx ? o : mx;
    }
    if ((threadIdx.x & 31) == 0) { red[threadIdx.x >> 5][0] = a; red[threadIdx.x >> 5][1] = bb; redm[threadIdx.x >> 5] = mx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double x = 0.0, y = 0.0;
        for (int w = 0; w < NORM_TPB / 32; ++w) {
            x += red[w][0];
            y += red[w][1];
            mx = redm[w] > mx ? redm[w] : mx;
        }
        part[2 * (uint64_t)blockIdx.x] = x;
        part[2 * (uint64_t)blockIdx.x + 1] = y;
        atomicMax(&fs->max_fix, mx);
    }
}

// E = -grad(phi) from the fixed-point potential (exact integer differences
// times 2^-F / 2h) into E, and the potential itself in FP64.
__global__ void k_efield_fix(const long long* __restrict__ Phi, E64* __restrict__ E, float4* __restrict__ E32,
                             double* __restrict__ phi, Geo G, double inv2h, const FixScale* __restrict__ fs)
{
    const float inv2hf = (float)inv2h;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, k, j, i;
        decode(t, G.log2n, r, k, j, i);
        if (fs[r].use64) continue;                // nothing was solved here (replayed steps: the host solves again)
        const double down = fs[r].down, sc = down * inv2h;
        const long long top2 = 2 * fs[r].top;
        const int n = G.n;
        const uint64_t sy = (uint64_t)n, sz = (uint64_t)n * n;
        const long long c = Phi[t];
        const long long xm = i > 0 ? Phi[t - 1] : c, xp = i < n - 1 ? Phi[t + 1] : c;
        const long long ym = j > 0 ? Phi[t - sy] : c, yp = j < n - 1 ? Phi[t + sy] : c;
        const long long zm = k > 0 ? Phi[t - sz] : -c, zp = k < n - 1 ? Phi[t + sz] : top2 - c;
        phi[t] = (double)c * down;
        if (E) {
            const double ex = (double)(xm - xp) * sc, ey = (double)(ym - yp) * sc, ez = (double)(zm - zp) * sc;
            const double m = sqrt((ex * ex + ey * ey) + ez * ez);
            reinterpret_cast<double2*>(E + t)[0] = make_double2(ex, ey);
            reinterpret_cast<double2*>(E + t)[1] = make_double2(ez, m);
            if (E32) E32[t] = make_float4((float)ex, (float)ey, (float)ez, (float)m);
        } else {
            // as k_efield: differences in FP64, scaling and |E| in FP32
            const float ex = (float)((double)(xm - xp) * down) * inv2hf, ey = (float)((double)(ym - yp) * down) * inv2hf,
                        ez = (float)((double)(zm - zp) * down) * inv2hf;
            E32[t] = make_float4(ex, ey, ez, sqrtf(ex * ex + ey * ey + ez * ez));
        }
    }
}

// B = round(b h^2 2^F) with b formed exactly as the FP64 right-hand side.
__global__ void k_rhs_fixed(const int64_t* __restrict__ rho, long long* __restrict__ B, Geo G, double qscale,
                            double bc_top, double bfix)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        const int k = (int)((t >> (2 * G.log2n)) & (uint64_t)(G.n - 1));
        const int64_t q = rho[t];
        long long v = 0;                          // a cell without charge below the electrode's
        if (q != 0 || k == G.n - 1) {
            double b = -((double)q * qscale);
            if (k == G.n - 1) b = b - bc_top;
            v = __double2ll_rn(b * bfix);
        }
        B[t] = v;
    }
}

// Phi <- round(Phi 2^-sh) when the fixed-point scale is lowered.
__global__ void k_shift_fixed(long long* __restrict__ Phi, int sh, uint64_t cells)
{
    const long long half = 1ll << (sh - 1);
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cells; t += (uint64_t)gridDim.x * blockDim.x)
        Phi[t] = (Phi[t] + half) >> sh;
}

// Phi <- 2 Phi - prev, prev <- the old Phi (with no previous potential yet:
// prev <- Phi only).
__global__ void k_extrapolate(long long* __restrict__ phi, long long* __restrict__ prev, uint64_t cells, bool have)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cells; t += (uint64_t)gridDim.x * blockDim.x) {
        const long long v = phi[t];
        if (have) phi[t] = (v + v) - prev[t];
        prev[t] = v;
    }
}

__global__ void k_phi_to_double(const long long* __restrict__ Phi, double* __restrict__ out, double sc, uint64_t cells)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cells; t += (uint64_t)gridDim.x * blockDim.x)
        out[t] = (double)Phi[t] * sc;
}

// E = -grad(phi) by centred differences with the boundary ghosts, and |E|.
// FP64 form: everything in FP64 into E64.  Mixed form (E == nullptr): the
// differences of neighbouring potentials in FP64 (they cancel most digits),
// the scaling and |E| in FP32, into E32 only.
__global__ void k_efield(const double* __restrict__ phi, E64* __restrict__ E, float4* __restrict__ E32, Geo G,
                         double h, double phi_top)
{
    const float inv2h = (float)(1.0 / (2.0 * h));
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, k, j, i;
        decode(t, G.log2n, r, k, j, i);
        const int n = G.n;
        const uint64_t sy = (uint64_t)n, sz = (uint64_t)n * n;
        const double c = phi[t];
        const double xm = i > 0 ? phi[t - 1] : c, xp = i < n - 1 ? phi[t + 1] : c;
        const double ym = j > 0 ? phi[t - sy] : c, yp = j < n - 1 ? phi[t + sy] : c;
        const double zm = k > 0 ? phi[t - sz] : -c, zp = k < n - 1 ? phi[t + sz] : 2.0 * phi_top - c;
        if (E) {
            const double ex = (xm - xp) / (2.0 * h), ey = (ym - yp) / (2.0 * h), ez = (zm - zp) / (2.0 * h);
            const double m = sqrt((ex * ex + ey * ey) + ez * ez);
            reinterpret_cast<double2*>(E + t)[0] = make_double2(ex, ey);
            reinterpret_cast<double2*>(E + t)[1] = make_double2(ez, m);
            if (E32) E32[t] = make_float4((float)ex, (float)ey, (float)ez, (float)m);
        } else {
            const float ex = (float)(xm - xp) * inv2h, ey = (float)(ym - yp) * inv2h, ez = (float)(zm - zp) * inv2h;
            E32[t] = make_float4(ex, ey, ez, sqrtf(ex * ex + ey * ey + ez * ez));
        }
    }
}

int gridsz(uint64_t n, int tpb) {
    uint64_t b = (n + tpb - 1) / tpb;
    if (b > 152 * 32) b = 152 * 32;
    return (int)(b < 1 ? 1 : b);
}

Geo geo(const Dev& d, int l, int R)
{
    Geo g;
    g.n = d.lev[l].n;
    g.log2n = 0;
    while ((1 << g.log2n) < g.n) ++g.log2n;
    g.R = R;
    g.cells = (uint64_t)R * g.n * g.n * g.n;
    return g;
}

// Blocks for a pass whose block row r takes realization r.
dim3 grid_per_real(const Geo& G)
{
    const int cap = 152 * 32 / G.R, b = gridsz(G.cells / G.R, 256);
    return dim3(b < cap ? b : (cap > 1 ? cap : 1), G.R);
}

// ---------------------------------------------------------------------------
// The coarse end of the V-cycle (levels of at most 32^3 cells) in one launch:
// a cluster of 8 blocks per realization.  The 32^3 and 16^3 levels are split
// into slabs of n/8 planes.  A thread owns an x pair of cells in every plane
// of its block's slab and keeps their values, right-hand sides and divisors
// in registers; the values also lie in shared memory, one array per colour
// with a rim of zeros, for the neighbours in x and y.  A half-sweep stores the
// slab's two outer planes into the neighbour blocks' halo planes (distributed
// shared memory) and ends with a cluster barrier.  The 8^3 level runs in the
// cluster's first block, the 4^3 bottom (48 red-black sweep pairs) in one warp
// with the cells in registers (64-bit forms: solved by its eigenvectors).
// What bounds it is a chain of latencies (22 cluster barriers from 32^3 down with
// two sweeps before and after; in FP32 96 warp half-sweeps at the bottom), not
// bandwidth: 29 us in fixed point, 25 us in FP32 from 32^3 down (33 and 28 with
// the interpolation cell by cell, every thread's fence at the barriers, a divisor
// formed per cell and the loads after the zeros; clusters of 16 blocks took 1 us
// off when they found 16 free SMs in one GPC, which other streams' kernels may
// hold); one block per realization from 16^3 down took 159 us in FP64 and 96 us in
// FP32, after 10 launches for the 32^3 level.
constexpr int COARSE_N = 32, COARSE_CL = 8, COARSE_TPB = 512, BOTTOM_SWEEPS = 48;

template <class T>
struct CoarseTop {       // the level the kernel starts at (n <= COARSE_N)
    T* phi;
    const T* rhs;
    int n;
};

// One half-sweep of the 4^3 level by one warp: a lane holds the colour-0 and
// the colour-1 cell of the x pair (2 ih, 2 ih + 1) of its row, five shuffles
// bring the neighbours of the relaxed one (other: the lane's cell of the other
// colour; xl the lane of the x neighbour outside the pair).
template <class T>
__device__ __forceinline__ T bottom_update(T other, T rhs, const Inv<T>& inv, int xl, unsigned ok, unsigned lane)
{
    const unsigned full = 0xffffffffu;
    const T xo = __shfl_sync(full, other, xl);
    const T ym = __shfl_sync(full, other, lane - 2), yp = __shfl_sync(full, other, lane + 2);
    const T zm = __shfl_sync(full, other, lane - 8), zp = __shfl_sync(full, other, lane + 8);
    T s = other + ((ok & 1u) ? xo : (T)0);
    s += (ok & 2u) ? ym : (T)0;
    s += (ok & 4u) ? yp : (T)0;
    s += (ok & 8u) ? zm : (T)0;
    s += (ok & 16u) ? zp : (T)0;
    return inv.relax(s, rhs);
}

template <class T>
__device__ void bottom_solve(T* phi, const T* rhs, unsigned lane)
{
    const int ih = lane & 1, j = (lane >> 1) & 3, k = lane >> 3;
    const int p0 = (j + k) & 1, p1 = p0 ^ 1;
    const int c0 = (k * 4 + j) * 4 + 2 * ih + p0, c1 = (k * 4 + j) * 4 + 2 * ih + p1;
    const int x0 = (int)lane + (p0 ? 1 : -1), x1 = (int)lane + (p1 ? 1 : -1);
    const unsigned yz = (j > 0 ? 2u : 0u) | (j < 3 ? 4u : 0u) | (k > 0 ? 8u : 0u) | (k < 3 ? 16u : 0u);
    const unsigned ok0 = yz | (p0 ? (ih < 1) : (ih > 0)), ok1 = yz | (p1 ? (ih < 1) : (ih > 0));
    const Inv<T> i0(diag_count(2 * ih + p0, j, k, 4)), i1(diag_count(2 * ih + p1, j, k, 4));
    T a = phi[c0], b = phi[c1];
    const T ra = rhs[c0], rb = rhs[c1];
#pragma unroll 1
    for (int it = 0; it < BOTTOM_SWEEPS; ++it) {
        a = bottom_update(b, ra, i0, x0, ok0, lane);
        b = bottom_update(a, rb, i1, x1, ok1, lane);
    }
    phi[c0] = a;
    phi[c1] = b;
}

// The 4^3 level solved by its eigenvectors, for the 64-bit forms: cosines along
// x and y (Neumann sides), sines along z (electrodes), six products with 4 x 4
// matrices by 64 threads; all threads of the block call this.  The sweeps
// above leave 4e-5 of the bottom's error; 1.6k clocks against 18k for them in
// fixed point.
__constant__ double BOTTOM_C[16] = {   // normalised cos(pi m (i + 1/2) / 4), row m
    0.5, 0.5, 0.5, 0.5,
    0.65328148243818826, 0.27059805007309850, -0.27059805007309850, -0.65328148243818826,
    0.5, -0.5, -0.5, 0.5,
    0.27059805007309850, -0.65328148243818826, 0.65328148243818826, -0.27059805007309850 };
__constant__ double BOTTOM_S[16] = {   // normalised sin(pi (m + 1) (k + 1/2) / 4), row m
    0.27059805007309850, 0.65328148243818826, 0.65328148243818826, 0.27059805007309850,
    0.5, 0.5, -0.5, -0.5,
    0.65328148243818826, -0.27059805007309850, -0.27059805007309850, 0.65328148243818826,
    0.5, -0.5, 0.5, -0.5 };
__constant__ double BOTTOM_L[5] = {    // 2 - 2 cos(pi m / 4)
    0.0, 0.58578643762690485, 2.0, 3.4142135623730949, 4.0 };

template <class T>
__device__ void bottom_solve_exact(T* phi, const T* rhs, double* w)
{
    const int t = threadIdx.x, i = t & 3, j = (t >> 2) & 3, k = t >> 4;
    double* a = w;
    double* b = w + 64;
    if (t < 64) a[t] = (double)rhs[t];
    __syncthreads();
    // forward along z, y, x, divide, back along x, y, z
#pragma unroll 1
    for (int st = 0; st < 6; ++st) {
        if (t < 64) {
            const int ax = st < 3 ? 2 - st : st - 3;
            const int row = ax == 0 ? i : (ax == 1 ? j : k), step = 1 << (2 * ax), first = t - row * step;
            const double* Q = ax == 2 ? BOTTOM_S : BOTTOM_C;
            double s = 0.0;
#pragma unroll
            for (int m = 0; m < 4; ++m) s = __fma_rn(st < 3 ? Q[row * 4 + m] : Q[m * 4 + row], a[first + m * step], s);
            if (st == 2) s = -s / ((BOTTOM_L[i] + BOTTOM_L[j]) + BOTTOM_L[k + 1]);
            b[t] = s;
        }
        __syncthreads();
        double* x = a; a = b; b = x;
    }
    if (t < 64) phi[t] = std::is_same<T, long long>::value ? (T)__double2ll_rn(a[t]) : (T)a[t];
    __syncthreads();
}

// The planes of one level in one block: PL own planes and a halo plane below
// and above, each as two colour arrays with a rim of zeros.
template <int N, int PLANES>
struct SlabShape {
    static constexpr int PL = PLANES, W = N / 2 + 2, PLANE = (N + 2) * W, COLOR = (PL + 2) * PLANE, SIZE = 2 * COLOR;
    static constexpr int PAIRS = N * N / 2;                     // threads that own a pair column
};

template <class T>
struct CoarseSmem {
    T p32[SlabShape<32, 4>::SIZE], p16[SlabShape<16, 2>::SIZE], p8[SlabShape<8, 8>::SIZE];
    T res[4 * 1024];               // residuals of a level's slab, then corrections of the level below, in cell order
    T r16[2 * 256], r8[512], e8[512];
    T p4[64], r4[64];
    double w4[128];                // the bottom's transforms
};

// A thread's pair column of a level: PER planes of the PLANES in the block.
template <class T, int N, int PLANES, int PER>
struct Slab {
    using S = SlabShape<N, PLANES>;
    static constexpr int PL = PER;
    T v[PL][2], r[PL][2];          // value and right-hand side per plane and colour
    Inv<T> inv[PL][2];
    T *own, *below, *above;        // the level's array here and in the neighbour blocks (nullptr: none)
    int at, ih, j, k0;             // the pair's place in a plane's rim array; the slab's first plane
    bool act;

    __device__ __forceinline__ void init(T* base, T* lower, T* upper, int first)
    {
        const int z = threadIdx.x / S::PAIRS * PER;     // the column's first plane in the slab
        own = base; below = lower; above = upper; k0 = first + z;
        act = z < PLANES;
        ih = threadIdx.x % (N / 2);
        j = threadIdx.x / (N / 2) % N;
        at = z * S::PLANE + (j + 1) * S::W + ih + 1;
        // between the electrodes a column has two divisors
        const int dy = 6 - (j == 0) - (j == N - 1);
        const Inv<T> even(dy - (ih == 0)), odd(dy - (ih == N / 2 - 1));
#pragma unroll
        for (int q = 0; q < PL; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                inv[q][c] = par(q, c) ? odd : even;
                if ((q == 0 && k0 == 0) || (q == PL - 1 && k0 + q == N - 1))
                    inv[q][c] = Inv<T>(diag_count(2 * ih + par(q, c), j, k0 + q, N));
                v[q][c] = r[q][c] = (T)0;
            }
    }
    // x parity of the colour-c cell of own plane q
    __device__ __forceinline__ int par(int q, int c) const { return (j + k0 + q + c) & 1; }
    // its place in cell order, from the column's first plane
    __device__ __forceinline__ int cell(int q, int p) const { return (q * N + j) * N + 2 * ih + p; }
    __device__ __forceinline__ T sum(int q, int c) const
    {
        const int o = c ^ 1;
        const T* b = own + o * S::COLOR + (q + 1) * S::PLANE + at;
        T s = v[q][o] + b[par(q, c) ? 1 : -1];
        s += b[-S::W];
        s += b[S::W];
        s += q > 0 ? v[q - 1][o] : b[-S::PLANE];
        s += q < PL - 1 ? v[q + 1][o] : b[S::PLANE];
        return s;
    }
    __device__ __forceinline__ void put(int q, int c, T w)
    {
        v[q][c] = w;
        own[c * S::COLOR + (q + 1) * S::PLANE + at] = w;
        if (q == 0 && below) below[c * S::COLOR + (PL + 1) * S::PLANE + at] = w;
        if (q == PL - 1 && above) above[c * S::COLOR + at] = w;
    }
    __device__ __forceinline__ void relax(int c)
    {
        if (!act) return;
        T w[PL];
#pragma unroll
        for (int q = 0; q < PL; ++q) w[q] = inv[q][c].relax(sum(q, c), r[q][c]);
#pragma unroll
        for (int q = 0; q < PL; ++q) put(q, c, w[q]);
    }
    // right-hand side from cell order
    __device__ __forceinline__ void set_rhs(const T* rhs)
    {
        if (!act) return;
#pragma unroll
        for (int q = 0; q < PL; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) r[q][c] = rhs[cell(q, par(q, c))];
    }
    __device__ __forceinline__ void residuals(T* res) const
    {
        if (!act) return;
#pragma unroll
        for (int q = 0; q < PL; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                res[cell(q, par(q, c))] =
                    MG<T>::resid(sum(q, c), r[q][c], v[q][c], diag_count(2 * ih + par(q, c), j, k0 + q, N));
    }
    // values in cell order, with the halo planes first and last
    __device__ __forceinline__ void values(T* out) const
    {
        if (!act) return;
#pragma unroll
        for (int q = -1; q <= PL; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                out[cell(q + 1, par(q, c))] = own[c * S::COLOR + (q + 1) * S::PLANE + at];
    }
    // plus the correction of the level below (cell order, planes from z0 on):
    // prolong_at's operations, with each coarse plane's share formed once
    __device__ __forceinline__ void correct(const T* ec, int z0)
    {
        static_assert(PL == 1 || PL % 2 == 0, "a column of several planes starts at an even one");
        if (!act) return;
        constexpr int NC = N / 2;
        const int J = j >> 1, il = ih > 0 ? -1 : 0, ir = ih < NC - 1 ? 1 : 0;
        const int dj = (j & 1) ? (J < NC - 1 ? NC : 0) : (J > 0 ? -NC : 0);
        auto plane = [&](int K, Pair<T>& m) {
            const bool neg = K < 0 || K >= NC;
            const T* a = ec + ((neg ? (K < 0 ? 0 : NC - 1) : K) - z0) * (NC * NC) + J * NC + ih;
            const T* b = a + dj;
            m.v[0] = MG<T>::axpy3(MG<T>::axpy3(a[0], a[il]), MG<T>::axpy3(b[0], b[il]));
            m.v[1] = MG<T>::axpy3(MG<T>::axpy3(a[0], a[ir]), MG<T>::axpy3(b[0], b[ir]));
            if (neg) { m.v[0] = -m.v[0]; m.v[1] = -m.v[1]; }
        };
        Pair<T> own, oth;
        plane(k0 >> 1, own);
        plane((k0 >> 1) + ((k0 & 1) ? 1 : -1), oth);
#pragma unroll
        for (int q = 0; q < PL; ++q) {
            if (q & 1) {
                plane(((k0 + q) >> 1) + 1, oth);
            } else if (q > 0) {
                const Pair<T> m = own;
                own = oth;
                oth = m;
            }
            const T c0 = MG<T>::div64(MG<T>::axpy3(own.v[0], oth.v[0]));
            const T c1 = MG<T>::div64(MG<T>::axpy3(own.v[1], oth.v[1]));
            const bool p = par(q, 0);
            put(q, 0, v[q][0] + (p ? c1 : c0));
            put(q, 1, v[q][1] + (p ? c0 : c1));
        }
    }
};

// Half the sums of eight residuals (cell order, planes 2 K and 2 K + 1 of an
// N x N slab) into planes of the level below.
template <class T, int N>
__device__ __forceinline__ void restrict_planes(const T* res, T* rc, int planes)
{
    constexpr int NC = N / 2;
    for (int t = threadIdx.x; t < planes * NC * NC; t += COARSE_TPB) {
        const int I = t % NC, J = (t / NC) % NC, K = t / (NC * NC);
        T acc = (T)0;
#pragma unroll
        for (int c = 0; c < 8; ++c) acc += res[((2 * K + (c >> 2)) * N + 2 * J + ((c >> 1) & 1)) * N + 2 * I + (c & 1)];
        rc[t] = MG<T>::half(acc);
    }
}

// cluster.sync() with one warp's fence for the block: the block's stores come
// before its barrier, and the fence after it is cumulative.
__device__ __forceinline__ void cluster_step()
{
    __syncthreads();
    if (threadIdx.x < 32) asm volatile("fence.acq_rel.cluster;" ::: "memory");
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// zero: the starting level's potential is taken as zero (not read).
template <class T>
__global__ void __cluster_dims__(COARSE_CL, 1, 1) __launch_bounds__(COARSE_TPB, 1)
    k_vcycle_coarse(CoarseTop<T> top, int zero, int nu1, int nu2)
{
    extern __shared__ __align__(16) unsigned char csm[];
    CoarseSmem<T>& S = *reinterpret_cast<CoarseSmem<T>*>(csm);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), n = top.n;
    const uint64_t base = (uint64_t)(blockIdx.x / COARSE_CL) * n * n * n;
    T* gp = top.phi + base;
    const T* gr = top.rhs + base;
    Slab<T, 32, 4, 4> a;
    Slab<T, 16, 2, 2> b;
    Slab<T, 8, 8, 1> c;
    auto lower = [&](T* p) { return rank > 0 ? cl.map_shared_rank(p, rank - 1) : nullptr; };
    auto upper = [&](T* p) { return rank < COARSE_CL - 1 ? cl.map_shared_rank(p, rank + 1) : nullptr; };
    a.init(S.p32, lower(S.p32), upper(S.p32), rank * 4);
    b.init(S.p16, lower(S.p16), upper(S.p16), rank * 2);
    c.init(S.p8, nullptr, nullptr, 0);
    // the starting level's right-hand side, on its way while the zeros are
    // written, and potential
    if (n == 32) a.set_rhs(gr + (int64_t)a.k0 * 1024);
    if (n == 16) b.set_rhs(gr + (int64_t)b.k0 * 256);
    if (n == 8 && rank == 0) c.set_rhs(gr + (int64_t)c.k0 * 64);
    // zeros everywhere (rims, domain halos, the corrections' start)
    {
        constexpr int WORDS = (SlabShape<32, 4>::SIZE + SlabShape<16, 2>::SIZE + SlabShape<8, 8>::SIZE) * (int)sizeof(T) / 16;
        static_assert(WORDS * 16 == (int)offsetof(CoarseSmem<T>, res), "the three levels first, in whole 16-byte words");
        for (int t = threadIdx.x; t < WORDS; t += COARSE_TPB) reinterpret_cast<uint4*>(&S)[t] = make_uint4(0, 0, 0, 0);
    }
    auto load = [&](auto& L, int N) {
        const int64_t o = (int64_t)L.k0 * N * N;
        if (!L.act) return;
#pragma unroll
        for (int q = 0; q < L.PL; ++q)
#pragma unroll
            for (int x = 0; x < 2; ++x) L.put(q, x, gp[o + L.cell(q, L.par(q, x))]);
    };
    cluster_step();                                    // zeros in place before a neighbour's store
    if (!zero) {
        if (n == 32) load(a, 32);
        if (n == 16) load(b, 16);
        if (n == 8 && rank == 0) load(c, 8);
        cluster_step();
    }
    if (n >= 32) {
        for (int it = 0; it < nu1; ++it) {
            a.relax(0); cluster_step();
            a.relax(1); cluster_step();
        }
        a.residuals(S.res);
        __syncthreads();
        restrict_planes<T, 32>(S.res, S.r16, 2);
        __syncthreads();
        b.set_rhs(S.r16);
    }
    if (n >= 16) {
        for (int it = 0; it < nu1; ++it) {
            b.relax(0); cluster_step();
            b.relax(1); cluster_step();
        }
        b.residuals(S.res);
        __syncthreads();
        restrict_planes<T, 16>(S.res, cl.map_shared_rank(S.r8, 0) + rank * 64, 1);
        cluster_step();
    }
    if (rank == 0) {
        if (n >= 16) c.set_rhs(S.r8 + c.k0 * 64);
        for (int it = 0; it < nu1; ++it) {
            c.relax(0); __syncthreads();
            c.relax(1); __syncthreads();
        }
        c.residuals(S.res + c.k0 * 64);
        __syncthreads();
        restrict_planes<T, 8>(S.res, S.r4, 4);
        if (threadIdx.x < 64) S.p4[threadIdx.x] = (T)0;
        __syncthreads();
        if constexpr (sizeof(T) == 8) {
            bottom_solve_exact(S.p4, S.r4, S.w4);
        } else {
            if (threadIdx.x < 32) bottom_solve(S.p4, S.r4, threadIdx.x);
            __syncthreads();
        }
        c.correct(S.p4, 0);
        __syncthreads();
        for (int it = 0; it < nu2; ++it) {
            c.relax(1); __syncthreads();
            c.relax(0); __syncthreads();
        }
        if (c.act)
#pragma unroll
            for (int x = 0; x < 2; ++x) (n == 8 ? gp : S.e8)[c.k0 * 64 + c.cell(0, c.par(0, x))] = c.v[0][x];
    }
    if (n >= 16) {
        cluster_step();
        const T* e0 = cl.map_shared_rank(S.e8, 0);
        for (int t = threadIdx.x; t < 512; t += COARSE_TPB) S.res[t] = e0[t];
        __syncthreads();
        b.correct(S.res, 0);
        cluster_step();
        for (int it = 0; it < nu2; ++it) {
            b.relax(1); cluster_step();
            b.relax(0); cluster_step();
        }
    }
    auto store = [&](auto& L, int N) {
        if (!L.act) return;
#pragma unroll
        for (int q = 0; q < L.PL; ++q)
#pragma unroll
            for (int x = 0; x < 2; ++x) gp[(int64_t)L.k0 * N * N + L.cell(q, L.par(q, x))] = L.v[q][x];
    };
    if (n >= 32) {
        b.values(S.res);
        __syncthreads();
        a.correct(S.res, rank * 2 - 1);
        cluster_step();
        for (int it = 0; it < nu2; ++it) {
            a.relax(1); cluster_step();
            a.relax(0); cluster_step();
        }
        store(a, 32);
    } else if (n == 16) {
        store(b, 16);
    }
    cluster_step();                     // no block's shared memory goes while another may still write to it
}

// ---------------------------------------------------------------------------
// Two red-black sweeps (four half-sweeps) of a level of at least 64^3 cells in
// one pass over memory.  A block owns a TX x TY column of a z chunk and
// marches up in z: while plane t (with a halo of four cells on each side)
// enters, half-sweep K runs on plane t - K, so that each plane is read once,
// relaxed four times and written once.  A thread keeps its x pairs of cells
// of the last planes in registers, one value of each colour (A: the colour of
// the first half-sweep, B: the other): a cell's z neighbours and one x
// neighbour are its own, of the other colour whatever the plane.  The other x
// neighbour and the two y neighbours come from a ring of planes in shared
// memory, one half plane per colour (no bank conflicts).  They were last
// written a step before (half-sweep K of step t reads what half-sweep K - 1
// left on the same plane in step t - 1), so one barrier per step orders
// everything.  In step t the cell that half-sweep K relaxes has x parity
// (y + t + c0 + 1) mod 2 for every K.  The next plane's values are loaded
// into registers a step ahead; the right-hand side never leaves them.  Pairs
// at the rim of the halo relax with what lies beside them; what is wrong
// there moves one cell inwards per half-sweep and ends before the tile.  Out
// of place (dst must not be src): neighbouring blocks read the halo's old
// values.  src == nullptr: a zero initial guess.  Every cell gets the
// operations of four plain half-sweeps in their order, so the result is the
// same to the last bit.  Cells outside the domain relax like the others, with
// a divisor of zero: no branch per cell (FP32 at 512^3 564 -> 521 us, fixed
// point at 256^3 202 -> 180 us).  Two sweeps of 256^3 cells: 180 us in fixed
// point (128 blocks on 152 SMs, which issue 65% of the time; the next plane's
// loads are the largest stall) against 508 us for four FP64 half-sweeps (FP64
// pipe 82% busy).
//
// The tile: 64 x 32 in FP32 (two pairs per thread), 32 x 32 in 64 bits.  A
// 64^3 level has too few of these for the chip's SMs: 32 x 16 there, with one
// pair per thread (17.9 -> 12.2 us in fixed point, 16.0 -> 10.4 us in FP32: a
// step takes as long as its warps need to issue).
template <class T, int TX_, int TY_, int PP_>
struct SweepTile {
    static constexpr int TX = TX_, TY = TY_, H = 4;
    static constexpr int EX = TX + 2 * H, EY = TY + 2 * H, PX = EX / 2;
    static constexpr int PP = PP_, NT = PX * EY / PP, RING = 5;
    static constexpr int GUARD = PX + 1;           // elements before and after the ring that rim pairs read
    static constexpr size_t SMEM = sizeof(T) * (RING * EX * EY + 2 * GUARD);
    static_assert(PX * EY == PP * NT && NT % PX == 0 && (PP == 1 || EY / PP % 2 == 0), "whole pairs per thread, rows of one parity");
};

template <class T, class Q>
__global__ void __launch_bounds__(Q::NT, 1)
    k_sweep4(const T* __restrict__ src, const T* __restrict__ rhs, T* __restrict__ dst, int n, int c0, int zc)
{
    constexpr int H = Q::H, PP = Q::PP, PX = Q::PX, EY = Q::EY, DY = EY / PP, PLH = PX * EY;   // PLH: the cells of one colour
    extern __shared__ __align__(16) unsigned char ssm[];
    T* ring = reinterpret_cast<T*>(ssm) + Q::GUARD;
    const int tiles_x = n / Q::TX;
    const int x0 = (int)(blockIdx.x % tiles_x) * Q::TX - H, y0 = (int)(blockIdx.x / tiles_x) * Q::TY - H;
    const int z0 = (int)blockIdx.y * zc, z1 = z0 + zc;
    const int64_t nn = (int64_t)n * n;
    // a thread's pairs lie DY rows apart (an even number): one x, one parity
    const int px = (int)threadIdx.x % PX, ey0 = (int)threadIdx.x / PX, gi = x0 + 2 * px, gj0 = y0 + ey0;
    const unsigned odd = (unsigned)(gj0 + c0);
    const int off0 = gj0 * n + gi;
    bool in[PP], tile[PP];                         // inside the domain; inside the block's own column
    Inv<T> i0[PP], i1[PP];                         // of the even and the odd cell; outside the domain zero: cells stay zero
    auto diag = [&](int m, int x) { return 6 - (gj0 + m * DY == 0) - (gj0 + m * DY == n - 1) - (x ? gi + 2 == n : gi == 0); };
#pragma unroll
    for (int m = 0; m < PP; ++m) {
        const int ey = ey0 + m * DY, gj = gj0 + m * DY;
        in[m] = gi >= 0 && gi < n && gj >= 0 && gj < n;       // pairs lie wholly inside or outside
        tile[m] = px >= H / 2 && px < PX - H / 2 && ey >= H && ey < EY - H;
        i0[m] = in[m] ? Inv<T>(diag(m, 0)) : Inv<T>::zero();
        i1[m] = in[m] ? Inv<T>(diag(m, 1)) : Inv<T>::zero();
    }
    // in step t: v[K] and r[K - 1] are plane t - K's values and right-hand
    // side, colour A in .v[0], colour B in .v[1]
    Pair<T> v[H + 2][PP], r[H][PP], nv[PP], nr[PP];
    auto plane_of = [&](int p) { return ((int64_t)blockIdx.z * n + p) * nn; };
    auto fetch = [&](const T* __restrict__ a, int p, Pair<T>* to) {
        const T* pl = a + plane_of(p);
#pragma unroll
        for (int m = 0; m < PP; ++m) {
            to[m].v[0] = to[m].v[1] = (T)0;
            if (in[m] && p >= 0 && p < n) to[m] = *reinterpret_cast<const Pair<T>*>(pl + (off0 + m * DY * n));
        }
    };
#pragma unroll
    for (int m = 0; m < PP; ++m) {
        nv[m].v[0] = nv[m].v[1] = (T)0;
#pragma unroll
        for (int K = 0; K < H + 2; ++K) v[K][m] = nv[m];
#pragma unroll
        for (int K = 0; K < H; ++K) r[K][m] = nv[m];
    }
    if (src) fetch(src, z0 - H, nv);
    int s = 0;                                     // ring slot of plane t
    // one step; EDGE: some plane of it is outside the march's range or at a
    // domain face (else no plane needs a look)
    auto step = [&](auto edge, int t) {
        constexpr bool EDGE = decltype(edge)::value;
        const bool par = (odd + (unsigned)t + 1u) & 1u;
        const int xo = par ? 1 : -1;
        Inv<T> ic[PP];
#pragma unroll
        for (int m = 0; m < PP; ++m) {
            ic[m] = par ? i1[m] : i0[m];
            T* c = ring + s * (2 * PLH) + threadIdx.x + m * Q::NT;
            if (src) {
                v[0][m].v[0] = par ? nv[m].v[0] : nv[m].v[1];
                v[0][m].v[1] = par ? nv[m].v[1] : nv[m].v[0];
            }
            c[0] = v[0][m].v[0];
            c[PLH] = v[0][m].v[1];
        }
        if (src) fetch(src, t + 1, nv);
        fetch(rhs, t, nr);
#pragma unroll
        for (int K = 1; K <= H; ++K) {
            const int p = t - K;
            if (EDGE && (p < 0 || p >= n || p < z0 - (H - K) || p >= z1 + (H - K))) continue;
            const int c = (K & 1) ? 0 : 1, o = c ^ 1;         // relaxed colour and the other
            const int dz = EDGE ? (p == 0) + (p == n - 1) : 0;
            T* plane = ring + (s >= K ? s - K : s + Q::RING - K) * (2 * PLH) + threadIdx.x;
#pragma unroll
            for (int m = 0; m < PP; ++m) {
                const T* oth = plane + o * PLH + m * Q::NT;
                T sum = v[K][m].v[o] + oth[xo];
                sum += oth[-PX];
                sum += oth[PX];
                sum += v[K + 1][m].v[o];
                sum += v[K - 1][m].v[o];
                T w = ic[m].relax(sum, r[K - 1][m].v[c]);
                if (EDGE && dz && in[m]) w = Inv<T>(diag(m, par) + dz).relax(sum, r[K - 1][m].v[c]);
                v[K][m].v[c] = w;
                if (K < H) plane[c * PLH + m * Q::NT] = w;
                if (K == H && tile[m]) {
                    Pair<T> q;
                    q.v[0] = par ? v[H][m].v[0] : w;
                    q.v[1] = par ? w : v[H][m].v[0];
                    *reinterpret_cast<Pair<T>*>(dst + plane_of(p) + (off0 + m * DY * n)) = q;
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < PP; ++m) {
#pragma unroll
            for (int K = H + 1; K > 0; --K) v[K][m] = v[K - 1][m];
#pragma unroll
            for (int K = H - 1; K > 0; --K) r[K][m] = r[K - 1][m];
            r[0][m].v[0] = par ? nr[m].v[0] : nr[m].v[1];
            r[0][m].v[1] = par ? nr[m].v[1] : nr[m].v[0];
        }
        s = s + 1 == Q::RING ? 0 : s + 1;
    };
#pragma unroll 1
    for (int t = z0 - H; t < z1 + H; ++t) {
        if (t - H >= z0 && t <= z1 && t - H > 0 && t < n) step(std::false_type{}, t);
        else step(std::true_type{}, t);
    }
}

template <class T>
T* lphi(MGLevel& L);
template <>
double* lphi<double>(MGLevel& L) { return L.phi; }
template <>
float* lphi<float>(MGLevel& L) { return L.phi32; }
template <>
long long* lphi<long long>(MGLevel& L) { return L.phi_fix; }
template <class T>
T* lrhs(MGLevel& L);
template <>
double* lrhs<double>(MGLevel& L) { return L.rhs; }
template <>
float* lrhs<float>(MGLevel& L) { return L.rhs32; }
template <>
long long* lrhs<long long>(MGLevel& L) { return L.rhs_fix; }

constexpr int SMALL_R = 4;

// Two sweeps of level l from src (nullptr: zeros) into dst.  The z chunk is
// the one with the least modelled time: waves of resident blocks (one per SM)
// times the planes each block marches over, the chunk and its halo of 2 x 4.
template <class T, class Q>
void launch_sweep4_tile(const T* src, const T* rhs, T* dst, const Geo& G, int c0, cudaStream_t s)
{
    allow_smem(k_sweep4<T, Q>, Q::SMEM);
    const uint64_t tiles = (uint64_t)(G.n / Q::TX) * (G.n / Q::TY);
    int zc = G.n;
    uint64_t best = ~0ull;
    for (int c = G.n; c >= 4; c >>= 1) {
        const uint64_t blocks = tiles * G.R * (G.n / c), cost = ((blocks + 151) / 152) * (c + 2 * Q::H);
        if (cost < best) { best = cost; zc = c; }
    }
    ++g_launches;
    k_sweep4<T, Q><<<dim3((unsigned)tiles, G.n / zc, G.R), Q::NT, Q::SMEM, s>>>(src, rhs, dst, G.n, c0, zc);
}

template <class T>
void launch_sweep4(const T* src, const T* rhs, T* dst, const Geo& G, int c0, cudaStream_t s)
{
    constexpr int TX = sizeof(T) == 4 ? 64 : 32;
    if (G.n == 64 && G.R < SMALL_R) launch_sweep4_tile<T, SweepTile<T, 32, 16, 1>>(src, rhs, dst, G, c0, s);
    else launch_sweep4_tile<T, SweepTile<T, TX, 32, TX / 32>>(src, rhs, dst, G, c0, s);
}

// FP32 grids of 2^25 cells and more march over eight planes (512^3: 235 us
// against 300 us, 16 x 128^3: 61 against 76); at 2^24 cells both take 33 us,
// smaller ones want the threads (64^3: 4.5 us against 5.6), and 64-bit values
// the registers (256^3 in fixed point: 50 us against 59).
template <class T>
void launch_prolong(T* phi, const T* ec, const Geo& G, cudaStream_t s)
{
    ++g_launches;
    if constexpr (sizeof(T) == 4) {
        if (G.cells >= (1u << 25)) {
            constexpr int kp = 8;
            k_prolong_march<T><<<(unsigned)((G.cells / (4 * kp) + 255) / 256), 256, 0, s>>>(phi, ec, G, kp);
            return;
        }
    }
    k_prolong<T><<<gridsz(G.cells / 4, 256), 256, 0, s>>>(phi, ec, G);
}

// One V-cycle from level l; zero: the level's potential counts as zero (it is
// not read).  Levels of 64^3 and more take two sweeps per pass, between the
// level's two arrays; an odd sweep runs as two plain half-sweeps in place.
template <class T>
void vcycle(Dev& d, int l, int R, int nu1, int nu2, cudaStream_t s, bool zero)
{
    MGLevel& L = d.lev[l];
    const Geo G = geo(d, l, R);
    T* const phi = lphi<T>(L);
    const T* rhs = lrhs<T>(L);
    if (L.n <= COARSE_N) {
        allow_smem(k_vcycle_coarse<T>, sizeof(CoarseSmem<T>));
        ++g_launches;
        k_vcycle_coarse<T><<<R * COARSE_CL, COARSE_TPB, sizeof(CoarseSmem<T>), s>>>(CoarseTop<T>{ phi, rhs, G.n }, zero,
                                                                                    nu1, nu2);
        return;
    }
    const int tpb = 256;
    T* cur = phi;
    auto sweeps = [&](int nu, int c0) {
        for (; nu >= 2; nu -= 2) {
            T* to = cur == phi ? reinterpret_cast<T*>(L.alt) : phi;
            launch_sweep4<T>(zero ? nullptr : cur, rhs, to, G, c0, s);
            cur = to;
            zero = false;
        }
        if (zero) cudaMemsetAsync(cur, 0, G.cells * sizeof(T), s);
        zero = false;
        if (nu == 1)
            for (int c = 0; c < 2; ++c) {
                ++g_launches;
                k_smooth<T><<<gridsz(G.cells / 2, tpb), tpb, 0, s>>>(cur, rhs, G, c0 ^ c);
            }
    };
    sweeps(nu1, 0);
    MGLevel& C = d.lev[l + 1];
    const Geo Gc = geo(d, l + 1, R);
    ++g_launches;
    k_resid_restrict<T><<<gridsz(Gc.cells, tpb), tpb, 0, s>>>(cur, rhs, lrhs<T>(C), Gc, G.n);
    vcycle<T>(d, l + 1, R, nu1, nu2, s, true);
    launch_prolong<T>(cur, lphi<T>(C), G, s);
    sweeps(nu2, 1);
    if (cur != phi) cudaMemcpyAsync(phi, cur, G.cells * sizeof(T), cudaMemcpyDeviceToDevice, s);
}


// ------------------------------------------------------------------ semi-implicit
// Variable-coefficient operator of the semi-implicit coupling (Sec. 4.3, Eq.
// poisson_simp): div(c grad phi) with c = 1 + sigma dt / eps0 per cell; the
// coefficient of an interior face is the mean of its two cells', a boundary
// face takes the cell's own (Neumann sides: no flux; Dirichlet electrodes:
// ghost 2 phi_b - phi_1, i.e. 2 c on the diagonal).  With c = 1 it is the
// operator above.  The systems are scaled by h^2 like the constant-
// coefficient ones.  Per level the face coefficients (fx, fy, fz: the +x,
// +y, +z face of each cell, 0 on the boundary), the diagonal and its
// inverse are formed once per solve (k_vc_faces), so a smoothing update is
// six fused multiply-adds and one multiply.
__global__ void k_vc_faces(const double* __restrict__ c, double* __restrict__ fx, double* __restrict__ fy,
                           double* __restrict__ fz, double* __restrict__ dg, double* __restrict__ idg, Geo G)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, k, j, i;
        decode(t, G.log2n, r, k, j, i);
        const int n = G.n;
        const uint64_t sy = (uint64_t)n, sz = (uint64_t)n * n;
        const double ci = c[t];
        const double xm = i > 0 ? 0.5 * (c[t - 1] + ci) : 0.0, xp = i < n - 1 ? 0.5 * (ci + c[t + 1]) : 0.0;
        const double ym = j > 0 ? 0.5 * (c[t - sy] + ci) : 0.0, yp = j < n - 1 ? 0.5 * (ci + c[t + sy]) : 0.0;
        const double zm = k > 0 ? 0.5 * (c[t - sz] + ci) : 2.0 * ci, zp = k < n - 1 ? 0.5 * (ci + c[t + sz]) : 2.0 * ci;
        fx[t] = xp;
        fy[t] = yp;
        fz[t] = k < n - 1 ? zp : 0.0;
        const double d = ((((xm + xp) + ym) + yp) + zm) + zp;
        dg[t] = d;
        idg[t] = 1.0 / d;
    }
}

// Off-diagonal sum of the variable-coefficient operator at (k, j, i).
__device__ __forceinline__ double vcf_sum(const double* __restrict__ phi, const double* __restrict__ fx,
                                          const double* __restrict__ fy, const double* __restrict__ fz, uint64_t idx,
                                          int n, int i, int j, int k)
{
    const uint64_t sy = (uint64_t)n, sz = (uint64_t)n * n;
    double s = 0.0;
    if (i > 0) s = __fma_rn(fx[idx - 1], phi[idx - 1], s);
    if (i < n - 1) s = __fma_rn(fx[idx], phi[idx + 1], s);
    if (j > 0) s = __fma_rn(fy[idx - sy], phi[idx - sy], s);
    if (j < n - 1) s = __fma_rn(fy[idx], phi[idx + sy], s);
    if (k > 0) s = __fma_rn(fz[idx - sz], phi[idx - sz], s);
    if (k < n - 1) s = __fma_rn(fz[idx], phi[idx + sz], s);
    return s;
}

struct VCArrays {        // one level's operator (kernel argument)
    const double* fx;
    const double* fy;
    const double* fz;
    const double* dg;
    const double* idg;
};

__global__ void k_smooth_vc(double* __restrict__ phi, const double* __restrict__ rhs, VCArrays A, Geo G, int color)
{
    const uint64_t half = G.cells >> 1;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < half; t += (uint64_t)gridDim.x * blockDim.x) {
        const int n = G.n;
        const int ih = (int)(t & (uint64_t)(n / 2 - 1));
        const int j = (int)((t >> (G.log2n - 1)) & (uint64_t)(n - 1));
        const int k = (int)((t >> (2 * G.log2n - 1)) & (uint64_t)(n - 1));
        const uint64_t r = t >> (3 * G.log2n - 1);
        const int i = 2 * ih + ((j + k + color) & 1);
        const uint64_t idx = ((r * n + k) * n + j) * n + i;
        const double sum = vcf_sum(phi, A.fx, A.fy, A.fz, idx, n, i, j, k);
        phi[idx] = (sum - rhs[idx]) * A.idg[idx];
    }
}

// Residual h^2 (b - A phi) at fine cells, half the sum of 8 children into the
// coarse right-hand side (the convention of k_resid_restrict).
__global__ void k_resid_restrict_vc(const double* __restrict__ phi, const double* __restrict__ rhs, VCArrays A,
                                    double* __restrict__ rhs_c, Geo Gc, int nf)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < Gc.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, K, J, I;
        decode(t, Gc.log2n, r, K, J, I);
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
            const uint64_t idx = (((uint64_t)r * nf + k) * nf + j) * nf + i;
            const double sum = vcf_sum(phi, A.fx, A.fy, A.fz, idx, nf, i, j, k);
            acc += rhs[idx] - __fma_rn(-A.dg[idx], phi[idx], sum);
        }
        rhs_c[t] = acc * 0.5;
    }
}

// Coarse coefficient: the mean of the 8 children.
__global__ void k_coef_restrict(const double* __restrict__ cf, double* __restrict__ cc, Geo Gc, int nf)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < Gc.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, K, J, I;
        decode(t, Gc.log2n, r, K, J, I);
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
            acc += cf[(((uint64_t)r * nf + k) * nf + j) * nf + i];
        }
        cc[t] = acc * 0.125;
    }
}

// The coarse end of the variable-coefficient V-cycle (levels of at most 16^3
// cells) in one launch, one block per realization.
constexpr int COARSE_VC_N = 16;

struct CoarseVC {
    int nlev;
    int n[MAX_LEVELS];
    double* phi[MAX_LEVELS];
    double* rhs[MAX_LEVELS];
    VCArrays A[MAX_LEVELS];
};

__device__ void blk_smooth_vc(double* phi, const double* rhs, const VCArrays& A, uint64_t off, int n, int color)
{
    const int half = n * n * n / 2;
    for (int t = threadIdx.x; t < half; t += blockDim.x) {
        const int ih = t % (n / 2), j = (t / (n / 2)) % n, k = t / (n * n / 2);
        const int i = 2 * ih + ((j + k + color) & 1);
        const uint64_t idx = ((uint64_t)k * n + j) * n + i;
        const double sum = vcf_sum(phi, A.fx + off, A.fy + off, A.fz + off, idx, n, i, j, k);
        phi[idx] = (sum - rhs[idx]) * A.idg[off + idx];
    }
    __syncthreads();
}

__global__ void __launch_bounds__(512) k_vcycle_coarse_vc(CoarseVC C, int nu1, int nu2, int bottom_sweeps)
{
    const uint64_t r = blockIdx.x;
    auto cells = [&](int l) { return (uint64_t)C.n[l] * C.n[l] * C.n[l]; };
    const int L = C.nlev - 1;
    for (int l = 0; l < L; ++l) {
        const uint64_t off = r * cells(l);
        double* phi = C.phi[l] + off;
        const double* rhs = C.rhs[l] + off;
        for (int it = 0; it < nu1; ++it) {
            blk_smooth_vc(phi, rhs, C.A[l], off, C.n[l], 0);
            blk_smooth_vc(phi, rhs, C.A[l], off, C.n[l], 1);
        }
        const int nf = C.n[l], nc = nf / 2;
        const uint64_t offc = r * cells(l + 1);
        for (int t = threadIdx.x; t < nc * nc * nc; t += blockDim.x) {
            const int I = t % nc, J = (t / nc) % nc, K = t / (nc * nc);
            double acc = 0.0;
            for (int q = 0; q < 8; ++q) {
                const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q >> 2);
                const uint64_t idx = ((uint64_t)k * nf + j) * nf + i;
                const double sum = vcf_sum(phi, C.A[l].fx + off, C.A[l].fy + off, C.A[l].fz + off, idx, nf, i, j, k);
                acc += rhs[idx] - __fma_rn(-C.A[l].dg[off + idx], phi[idx], sum);
            }
            C.rhs[l + 1][offc + t] = acc * 0.5;
            C.phi[l + 1][offc + t] = 0.0;
        }
        __syncthreads();
    }
    {
        const uint64_t off = r * cells(L);
        for (int it = 0; it < bottom_sweeps; ++it) {
            blk_smooth_vc(C.phi[L] + off, C.rhs[L] + off, C.A[L], off, C.n[L], 0);
            blk_smooth_vc(C.phi[L] + off, C.rhs[L] + off, C.A[L], off, C.n[L], 1);
        }
    }
    for (int l = L - 1; l >= 0; --l) {
        const uint64_t off = r * cells(l);
        double* phi = C.phi[l] + off;
        const double* ec = C.phi[l + 1] + r * cells(l + 1);
        const int nf = C.n[l];
        for (int t = threadIdx.x; t < nf * nf * nf; t += blockDim.x) {
            const int i = t % nf, j = (t / nf) % nf, k = t / (nf * nf);
            phi[t] += prolong_at(ec, nf / 2, i, j, k);
        }
        __syncthreads();
        for (int it = 0; it < nu2; ++it) {
            blk_smooth_vc(phi, C.rhs[l] + off, C.A[l], off, nf, 1);
            blk_smooth_vc(phi, C.rhs[l] + off, C.A[l], off, nf, 0);
        }
    }
}

// Squared norms of the residual and of the right-hand side per realization
// (blockIdx.y): one partial pair per block in part[2 (r gridDim.x + x)],
// summed in a fixed order by k_norm_final, so the convergence test (and with
// it the cycle count and the potential) is the same on every run.  256
// threads per block.
__global__ void __launch_bounds__(256) k_resid_norm_vc(const double* __restrict__ phi, const double* __restrict__ rhs,
                                                       VCArrays A, Geo G, double* __restrict__ part)
{
    const uint64_t r = blockIdx.y;
    const uint64_t per = (uint64_t)G.n * G.n * G.n;
    double s0 = 0.0, s1 = 0.0;
    for (uint64_t u = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; u < per; u += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t t = r * per + u;
        int rr, k, j, i;
        decode(t, G.log2n, rr, k, j, i);
        const double sum = vcf_sum(phi, A.fx, A.fy, A.fz, t, G.n, i, j, k);
        const double res = rhs[t] - __fma_rn(-A.dg[t], phi[t], sum);
        s0 += res * res;
        s1 += rhs[t] * rhs[t];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    __shared__ double w0[8], w1[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { w0[wid] = s0; w1[wid] = s1; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { a += w0[q]; b += w1[q]; }
        const uint64_t o = 2 * (r * gridDim.x + blockIdx.x);
        part[o] = a;
        part[o + 1] = b;
    }
}

// h^2 b = h^2 (-rho/eps0) with the top electrode term weighted by the
// boundary cell's coefficient.
__global__ void k_rhs_vc(const int64_t* __restrict__ rho, const double* __restrict__ c, double* __restrict__ rhs, Geo G,
                         double qscale, double bc_top, double h2)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G.cells; t += (uint64_t)gridDim.x * blockDim.x) {
        int r, k, j, i;
        decode(t, G.log2n, r, k, j, i);
        double b = -((double)rho[t] * qscale);
        if (k == G.n - 1) b = b - c[t] * bc_top;
        rhs[t] = b * h2;
    }
}

// c = 1 + sigma dt / eps0, sigma = q_e mu n_e (Eq. conductivity) from the
// fixed-point CIC electron count.
__global__ void k_coef_from_ne(const unsigned long long* __restrict__ ne_fix, double* __restrict__ c, uint64_t cells,
                               double per_cell, double qmu, double dt_eps)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cells; t += (uint64_t)gridDim.x * blockDim.x) {
        const double ne = ((double)ne_fix[t] * per_cell);
        const double sigma = qmu * ne;
        c[t] = 1.0 + sigma * dt_eps;
    }
}

}  // namespace

constexpr int MAX_REAL_NORM = 4096;

// Replays (capturing first if needed) the graph of kind k on stream s:
// k = 0: one FP64 V-cycle; k = 1: two FP32 V-cycles from a zero correction;
// k = 3: one fixed-point V-cycle.  The launches of a cycle depend only on the
// level pointers and the smoother counts, so one capture per (nu1, nu2) serves every solve.
// Launches directly when d.direct_cycles is set (a solve on per-call
// buffers, whose graphs could not be reused) or capture is not possible.
void run_cycles(Dev& d, int k, int R, int nu1, int nu2, cudaStream_t s)
{
    auto direct = [&]() {
        if (k == 0) {
            vcycle<double>(d, 0, R, nu1, nu2, s, false);
        } else if (k == 3) {
            vcycle<long long>(d, 0, R, nu1, nu2, s, false);
        } else {
            vcycle<float>(d, 0, R, nu1, nu2, s, true);
            vcycle<float>(d, 0, R, nu1, nu2, s, false);
        }
    };
    if (d.direct_cycles) {
        direct();
        return;
    }
    if (d.vgraph[k] && (d.vgraph_nu[k][0] != nu1 || d.vgraph_nu[k][1] != nu2)) {
        cudaGraphExecDestroy(d.vgraph[k]);
        d.vgraph[k] = nullptr;
    }
    if (!d.vgraph[k]) {
        cudaGraph_t g = nullptr;
        if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            cudaGetLastError();
            direct();
            return;
        }
        const unsigned long long l0 = g_launches.load();
        direct();
        const unsigned long long nk = g_launches.load() - l0;
        g_launches -= nk;                         // captured, not run
        if (cudaStreamEndCapture(s, &g) != cudaSuccess || !g ||
            cudaGraphInstantiate(&d.vgraph[k], g, 0) != cudaSuccess) {
            cudaGetLastError();
            if (g) cudaGraphDestroy(g);
            d.vgraph[k] = nullptr;
            direct();
            return;
        }
        cudaGraphDestroy(g);
        d.vgraph_nu[k][0] = nu1;
        d.vgraph_nu[k][1] = nu2;
        d.vgraph_kernels[k] = nk;
    }
    g_launches += d.vgraph_kernels[k];
    cudaGraphLaunch(d.vgraph[k], s);
}

// Lowers the fixed-point potential's scale to F bits (F < d.phi_F): the
// potential and the kept previous one shifted right by the difference.
void lower_phi_scale(const Params& P, Dev& d, int F, cudaStream_t s)
{
    if (F >= d.phi_F) return;
    const Geo G0 = geo(d, 0, P.R);
    ++g_launches;
    k_shift_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(reinterpret_cast<long long*>(d.lev[0].phi), d.phi_F - F,
                                                       G0.cells);
    if (d.phi_prev && d.have_prev) {
        ++g_launches;
        k_shift_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(reinterpret_cast<long long*>(d.phi_prev), d.phi_F - F,
                                                           G0.cells);
    }
    d.phi_F = F;
}

// FP64 form, before the cycles: start guess, scale, Phi and B.
// Returns whether the scale may have been taken from the guess (else it is from
// the bound).
bool fix_begin(const Params& P, Dev& d, bool extrapolate, bool replayed, cudaStream_t s)
{
    MGLevel& L0 = d.lev[0];
    const Geo G0 = geo(d, 0, P.R);
    double qscale, bc_top;
    rhs_consts(P, qscale, bc_top);
    const bool ex = extrapolate && d.phi_prev;
    cudaMemsetAsync(d.fix, 0, P.R * sizeof(FixScale), s);
    g_launches += 3;
    k_fix_start<<<grid_per_real(G0), 256, 0, s>>>(L0.phi, reinterpret_cast<double*>(d.phi_prev), ex, d.have_prev, L0.rhs,
                                                  G0, bc_top * (L0.h * L0.h), d.fix);
    k_fix_scale<<<(P.R + 255) / 256, 256, 0, s>>>(d.fix, P.R, P.E0 * (P.hi[2] - P.lo[2]), G0.n,
                                                 ex && d.have_prev ? (replayed ? 2 : 1) : 0, 0);
    k_fix_load<<<grid_per_real(G0), 256, 0, s>>>(L0.phi, L0.rhs, L0.phi_fix, L0.rhs_fix, G0.cells / P.R, d.fix, 0);
    const bool near = ex && d.have_prev;
    if (ex) d.have_prev = true;
    d.fix_result = true;
    return near;
}

// precision: 0 V-cycles in 64-bit fixed point, followed by FP64 ones where the
// integers do not serve (a start guess or an iterate beyond their range, a
// tolerance below what they reach); 1 FP32 V-cycles in FP64 residual refinement;
// 2 FP32 V-cycles in fixed-point residual refinement (potential in units of
// 2^-phi_F V, right-hand side prepared by the charge kernel).  Returns 0 on
// convergence, ITOKMC_ERR_NOCONV (-6) if max_cycles is reached or the potential
// of form 2 leaves its range.
int field_solve(const Params& P, Dev& d, int precision, double rtol, int nu1, int nu2, unsigned long long rho_absmax,
                int max_cycles, cudaStream_t s, int* cycles_out, double* rel_out, bool extrapolate)
{
    const int R = P.R;
    MGLevel& L0 = d.lev[0];
    const Geo G0 = geo(d, 0, R);
    const uint64_t per_real = G0.cells / R;
    const int items = (int)(per_real / NORM_TPB < 8 ? per_real / NORM_TPB : 8);
    const int nblk = (int)(G0.cells / ((uint64_t)NORM_TPB * items));
    const int bpr = nblk / R;
    const MarchGeo march = march_geo(G0.n);     // the integer residuals' blocks
    double* h_norm = d.norm_host;       // R (2 + FIX_DOUBLES) doubles of host memory owned by the caller
    double bnorm[MAX_REAL_NORM];
    if (R > MAX_REAL_NORM) return -1;
    double worst = 0.0;
    int cyc = 0;
    int status = -6;
    const bool fixed = precision == 2;
    bool fix = precision == 0;          // FP64 form in fixed point (until it cannot go on)
    d.fix_result = false;
    long long* Phi = reinterpret_cast<long long*>(L0.phi);
    long long* Bfix = reinterpret_cast<long long*>(L0.rhs);
    if (fixed) {
        // scale from a bound on |phi| (lowered only: the warm start is shifted)
        lower_phi_scale(P, d, phi_fixed_bits(phi_bound(P, rho_absmax)), s);
        double qscale, bc_top;
        rhs_consts(P, qscale, bc_top);
        ++g_launches;
        k_rhs_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(d.rho, Bfix, G0, qscale, bc_top,
                                                         L0.h * L0.h * std::ldexp(1.0, d.phi_F));
        // initial guess 2 phi_k - phi_{k-1} (the previous potential is kept)
        if (extrapolate && d.phi_prev) {
            ++g_launches;
            k_extrapolate<<<gridsz(G0.cells, 256), 256, 0, s>>>(Phi, reinterpret_cast<long long*>(d.phi_prev), G0.cells,
                                                               d.have_prev);
            d.have_prev = true;
        }
    }
    bool near = false;                  // fixed point: the scale is from a guess that ought to be near
    if (fix) near = fix_begin(P, d, extrapolate, false, s);
    const float rsc = (float)std::ldexp(1.0, -d.phi_F);
    const float esc = (float)std::ldexp(1.0, d.phi_F);
    // FP64 form: the residual norm only serves the convergence test, so
    // it is evaluated at cycle 0 and then at the cycle the observed
    // convergence factor predicts (refinement forms need the residual every
    // outer iteration as the right-hand side of the correction).
    int next_check = 0;
    bool first = true;                  // the check takes the right-hand sides' norms too
    double rho_est = 0.1, prev_rel = -1.0;
    int prev_cyc = 0;
    for (cyc = 0; cyc <= max_cycles; ++cyc) {
        if (precision == 0 && cyc < next_check && cyc < max_cycles) {
            run_cycles(d, fix ? 3 : 0, R, nu1, nu2, s);
            continue;
        }
        ++g_launches;
        if (fixed)
            k_resid_fixed<<<R * march.bpr, NORM_TPB, 0, s>>>(Phi, Bfix, L0.rhs32, G0, rsc, d.norm_part, first, march);
        else if (fix)
            k_resid_norm_fix<<<R * march.bpr, NORM_TPB, 0, s>>>(L0.phi_fix, L0.rhs_fix, G0, d.norm_part, first, march, d.fix);
        else
            k_resid_norm<<<nblk, NORM_TPB, 0, s>>>(L0.phi, L0.rhs, precision == 1 ? L0.rhs32 : nullptr, G0,
                                                   d.norm_part, first, items);
        ++g_launches;
        k_norm_final<<<R, 256, 0, s>>>(d.norm_part, fixed || fix ? march.bpr : bpr, R, d.norm_out, fix ? d.fix : nullptr);
        cudaMemcpyAsync(h_norm, d.norm_out, 2 * R * sizeof(double), cudaMemcpyDeviceToHost, s);
        if (fix) cudaMemcpyAsync(h_norm + 2 * R, d.fix, R * sizeof(FixScale), cudaMemcpyDeviceToHost, s);
        if (cudaStreamSynchronize(s) != cudaSuccess) return -3;
        worst = 0.0;
        bool done = true;
        for (int r = 0; r < R; ++r) {
            if (first) bnorm[r] = h_norm[2 * r + 1];
            const double rn = std::sqrt(h_norm[2 * r]), bn = std::sqrt(bnorm[r]);
            const double rel = bn > 0.0 ? rn / bn : rn;
            if (rel > worst || !(rel == rel)) worst = rel;
            if (!(rn <= rtol * bn)) done = false;
        }
        first = false;
        bool few = false;               // a scale that may be too low
        if (fix) {
            const FixScale* fs = reinterpret_cast<const FixScale*>(h_norm + 2 * R);
            bool range = std::isfinite(worst), finer = false;
            for (int r = 0; r < R; ++r) {
                range = range && !fs[r].use64 && fs[r].seen < (unsigned long long)FIX_LIM;
                finer = finer || fix_shift(fs[r]) > 0;
                const unsigned long long top = (unsigned long long)(fs[r].top < 0 ? -fs[r].top : fs[r].top);
                few = few || (bnorm[r] > 0.0 && std::max(fs[r].seen, top) < (1ull << (FIX_BITS + 1)));
            }
            if (range && finer && cyc > 0 && cyc < max_cycles) {
                // a loose bound left the leading bits unused: more of them, and
                // a cycle that fills them
                g_launches += 2;
                k_fix_scale<<<(R + 255) / 256, 256, 0, s>>>(d.fix, R, P.E0 * (P.hi[2] - P.lo[2]), G0.n, 0, 1);
                k_fix_load<<<grid_per_real(G0), 256, 0, s>>>(L0.phi, L0.rhs, L0.phi_fix, L0.rhs_fix, per_real, d.fix, 1);
                first = true;
                done = false;
            } else if (!range && near) {
                // the solution is far above the guess: once more, at the bound's scale
                near = false;
                g_launches += 2;
                k_fix_scale<<<(R + 255) / 256, 256, 0, s>>>(d.fix, R, P.E0 * (P.hi[2] - P.lo[2]), G0.n, 0, 0);
                k_fix_load<<<grid_per_real(G0), 256, 0, s>>>(L0.phi, L0.rhs, L0.phi_fix, L0.rhs_fix, per_real, d.fix, 0);
                first = true;
                prev_rel = -1.0;
                next_check = 0;
                cyc = -1;
                continue;
            } else if (!range || (!done && prev_rel >= 0.0 && worst > 0.9 * prev_rel)) {
                // out of the integer range (the cycles start again from the
                // guess), or no further progress in it (they go on): FP64 cycles
                if (range) {
                    ++g_launches;
                    k_fix_store<<<grid_per_real(G0), 256, 0, s>>>(L0.phi_fix, L0.phi, per_real, d.fix);
                }
                fix = false;
                d.fix_result = false;
                first = true;
                prev_rel = -1.0;
                cyc = range ? cyc - 1 : -1;                 // the check again, in FP64
                next_check = cyc + 1;
                continue;
            }
        }
        // a guess that needs no cycle stays as it is
        if (fix && done && cyc == 0 && !near) d.fix_result = false;
        if (done) { status = 0; break; }
        if (cyc == max_cycles || !std::isfinite(worst)) break;
        if (precision == 0) {
            if (prev_rel > 0.0 && worst > 0.0 && cyc > prev_cyc) {
                rho_est = std::pow(worst / prev_rel, 1.0 / (cyc - prev_cyc));
                rho_est = std::min(0.5, std::max(0.02, rho_est));
            }
            const double need = worst > 0.0 ? std::log(rtol / worst) / std::log(rho_est) : 1.0;
            next_check = cyc + std::max(1, (int)std::floor(need));
        }
        prev_rel = worst;
        prev_cyc = cyc;
        if (precision >= 1) {
            // inner solve of A e = r in FP32: two V-cycles per outer residual
            run_cycles(d, 1, R, nu1, nu2, s);
            ++g_launches;
            if (fixed)
                k_add_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(Phi, L0.phi32, esc, G0.cells);
            else
                k_add_correction<<<gridsz(G0.cells, 256), 256, 0, s>>>(L0.phi, L0.phi32, G0.cells);
        } else {
            run_cycles(d, fix ? 3 : 0, R, nu1, nu2, s);
            if (fix && few && cyc == 0) {
                // after one cycle the potential is known well enough for a
                // scale that the bound left too low (no wait for it)
                g_launches += 3;
                const dim3 few_blocks(std::min<unsigned>(grid_per_real(G0).x, std::max(1, 152 * 8 / R)), R);
                k_fix_max<<<few_blocks, 256, 0, s>>>(L0.phi_fix, per_real, d.fix);
                k_fix_scale<<<(R + 255) / 256, 256, 0, s>>>(d.fix, R, P.E0 * (P.hi[2] - P.lo[2]), G0.n, 0, 2);
                k_fix_load<<<grid_per_real(G0), 256, 0, s>>>(L0.phi, L0.rhs, L0.phi_fix, L0.rhs_fix, per_real, d.fix, 1);
                first = true;
            }
        }
    }
    if (cycles_out) *cycles_out = cyc;
    if (rel_out) *rel_out = worst;
    return status;
}

// The solve of field_solve with a fixed number of cycles and no host
// synchronisation, for steps replayed from a captured graph: the same
// launches (the fixed-point scale is kept: a step that needs a lower one is
// solved again by field_solve afterwards), then the residual and right-hand
// side norms of every realization in d.norm_out, which the host checks after
// the step.  cycles: V-cycles (FP64), or outer corrections of two FP32
// V-cycles each (refinement forms).
void field_solve_fixed(const Params& P, Dev& d, int precision, int nu1, int nu2, int cycles, cudaStream_t s)
{
    const int R = P.R;
    MGLevel& L0 = d.lev[0];
    const Geo G0 = geo(d, 0, R);
    const uint64_t per_real = G0.cells / R;
    const int items = (int)(per_real / NORM_TPB < 8 ? per_real / NORM_TPB : 8);
    const int nblk = (int)(G0.cells / ((uint64_t)NORM_TPB * items));
    const int bpr = nblk / R;
    const MarchGeo march = march_geo(G0.n);     // the integer residuals' blocks
    const bool fixed = precision == 2;
    long long* Phi = reinterpret_cast<long long*>(L0.phi);
    long long* Bfix = reinterpret_cast<long long*>(L0.rhs);
    d.fix_result = false;
    if (fixed) {
        double qscale, bc_top;
        rhs_consts(P, qscale, bc_top);
        ++g_launches;
        k_rhs_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(d.rho, Bfix, G0, qscale, bc_top,
                                                         L0.h * L0.h * std::ldexp(1.0, d.phi_F));
        if (d.phi_prev) {
            ++g_launches;
            k_extrapolate<<<gridsz(G0.cells, 256), 256, 0, s>>>(Phi, reinterpret_cast<long long*>(d.phi_prev), G0.cells,
                                                               d.have_prev);
            d.have_prev = true;
        }
    } else if (precision == 0) {
        fix_begin(P, d, true, true, s);
    }
    const float rsc = (float)std::ldexp(1.0, -d.phi_F);
    const float esc = (float)std::ldexp(1.0, d.phi_F);
    auto resid = [&](bool first) {
        ++g_launches;
        if (fixed)
            k_resid_fixed<<<R * march.bpr, NORM_TPB, 0, s>>>(Phi, Bfix, L0.rhs32, G0, rsc, d.norm_part, first, march);
        else if (precision == 0)
            k_resid_norm_fix<<<R * march.bpr, NORM_TPB, 0, s>>>(L0.phi_fix, L0.rhs_fix, G0, d.norm_part, first, march, d.fix);
        else
            k_resid_norm<<<nblk, NORM_TPB, 0, s>>>(L0.phi, L0.rhs, L0.rhs32, G0, d.norm_part, first, items);
    };
    for (int c = 0; c < cycles; ++c) {
        if (precision == 0) {
            run_cycles(d, 3, R, nu1, nu2, s);
            continue;
        }
        resid(false);
        run_cycles(d, 1, R, nu1, nu2, s);
        ++g_launches;
        if (fixed)
            k_add_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(Phi, L0.phi32, esc, G0.cells);
        else
            k_add_correction<<<gridsz(G0.cells, 256), 256, 0, s>>>(L0.phi, L0.phi32, G0.cells);
    }
    resid(true);
    ++g_launches;
    k_norm_final<<<R, 256, 0, s>>>(d.norm_part, precision == 1 ? bpr : march.bpr, R, d.norm_out);
}

// The FP32 value of a double that is one (false: it is not, or is not a normal
// number).
__device__ __forceinline__ bool as_float(double v, float& f)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (b << 1 == 0) { f = 0.f; return true; }
    if ((b & 0x1fffffffull) != 0 || e < 1023 - 126 || e > 1023 + 126) return false;
    f = __uint_as_float((uint32_t)((b >> 32) & 0x80000000u) | ((uint32_t)(e - 896) << 23) | (uint32_t)((b >> 29) & 0x7fffffu));
    return true;
}

// |E| of three FP32 components rounded to FP32 as (float)sqrt((ex ex + ey ey) +
// ez ez) in FP64 is, from sums of two floats (relative error below 2^-40):
// false where that is too near a rounding boundary to tell, or out of range.
__device__ __forceinline__ bool norm3(float x, float y, float z, float& m)
{
    const float a = x * x, b = y * y, c = z * z;
    const float ea = __fmaf_rn(x, x, -a), eb = __fmaf_rn(y, y, -b), ec = __fmaf_rn(z, z, -c);
    const float s1 = a + b, t1 = s1 - a, e1 = (a - (s1 - t1)) + (b - t1);       // two-sums
    const float s = s1 + c, t2 = s - s1, e2 = (s1 - (s - t2)) + (c - t2);
    const float lo = ((ea + eb) + ec) + (e1 + e2);
    if (!(s > 1e-20f && s < 1e30f)) return false;
    const float r = sqrtf(s);
    const float d = __fdiv_rn(__fmaf_rn(-r, r, s) + lo, r + r);                  // sqrt(s + lo) = r + d
    m = r + d;
    const float off = fabsf((r - m) + d);                                        // what the rounding left
    const float half = 0.5f * (__uint_as_float(__float_as_uint(m) + 1u) - m);
    // (a power of two has its lower boundary at half the distance)
    return fabsf(off - half) > half * 1e-3f && fabsf(off - 0.5f * half) > half * 1e-3f;
}

// The handle's field from three blocks of components: E64 (FP64 form) or
// float4 (mixed form).  An FP32 field (one read from the mixed form) takes
// |E| without the FP64 pipe, whose square root bounds the pass otherwise.
__global__ void k_pack_field(const double* __restrict__ E3, E64* __restrict__ E, float4* __restrict__ E32, uint64_t G)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G; t += (uint64_t)gridDim.x * blockDim.x) {
        const double ex = E3[t], ey = E3[G + t], ez = E3[2 * G + t];
        float fx, fy, fz, fm;
        if (!E && as_float(ex, fx) && as_float(ey, fy) && as_float(ez, fz) && norm3(fx, fy, fz, fm)) {
            E32[t] = make_float4(fx, fy, fz, fm);
            continue;
        }
        const double m = sqrt((ex * ex + ey * ey) + ez * ez);
        if (E) {
            reinterpret_cast<double2*>(E + t)[0] = make_double2(ex, ey);
            reinterpret_cast<double2*>(E + t)[1] = make_double2(ez, m);
        }
        if (E32) E32[t] = make_float4((float)ex, (float)ey, (float)ez, (float)m);
    }
}

// Field readback: from the FP64 field, or from the FP32 one (mixed form).
__global__ void k_unpack_field(const E64* __restrict__ E, const float4* __restrict__ E32, double* __restrict__ E3,
                               uint64_t G)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < G; t += (uint64_t)gridDim.x * blockDim.x) {
        if (E) {
            const E64 e = E[t];
            E3[t] = e.x; E3[G + t] = e.y; E3[2 * G + t] = e.z;
        } else {
            const float4 e = E32[t];
            E3[t] = e.x; E3[G + t] = e.y; E3[2 * G + t] = e.z;
        }
    }
}

void launch_pack_field(const Params& P, Dev& d, const double* E3, cudaStream_t s)
{
    const uint64_t G = (uint64_t)P.R * P.n3;
    ++g_launches;
    k_pack_field<<<gridsz(G, 256), 256, 0, s>>>(E3, d.E, d.E32, G);
}

void launch_unpack_field(const Params& P, Dev& d, double* E3, cudaStream_t s)
{
    const uint64_t G = (uint64_t)P.R * P.n3;
    ++g_launches;
    k_unpack_field<<<gridsz(G, 256), 256, 0, s>>>(d.E, d.E32, E3, G);
}

void launch_efield(const Params& P, Dev& d, cudaStream_t s) { launch_efield_to(P, d, s, d.E, d.E32); }

// E = -grad(phi) into the given FP64 and/or FP32 field arrays.
void launch_efield_to(const Params& P, Dev& d, cudaStream_t s, E64* E, float4* E32)
{
    const Geo G0 = geo(d, 0, P.R);
    const double phi_top = P.E0 * (P.hi[2] - P.lo[2]);
    ++g_launches;
    if (d.fix_result) {
        // of a solve in fixed point: E and the FP64 potential in one pass
        k_efield_fix<<<gridsz(G0.cells, 256), 256, 0, s>>>(d.lev[0].phi_fix, E, E32, d.lev[0].phi, G0,
                                                          1.0 / (2.0 * d.lev[0].h), d.fix);
        d.fix_result = false;
    } else if (d.phi_F > 0)
        k_efield_fixed<<<gridsz(G0.cells, 256), 256, 0, s>>>(
            reinterpret_cast<const long long*>(d.lev[0].phi), E, E32, G0,
            std::ldexp(1.0, -d.phi_F) / (2.0 * d.lev[0].h), std::llrint(std::ldexp(phi_top, d.phi_F)));
    else
        k_efield<<<gridsz(G0.cells, 256), 256, 0, s>>>(d.lev[0].phi, E, E32, G0, d.lev[0].h, phi_top);
}

// The potential as FP64 volts into out (R n^3).
void launch_phi_to_double(const Params& P, Dev& d, double* out, cudaStream_t s)
{
    const Geo G0 = geo(d, 0, P.R);
    ++g_launches;
    k_phi_to_double<<<gridsz(G0.cells, 256), 256, 0, s>>>(reinterpret_cast<const long long*>(d.lev[0].phi), out,
                                                          std::ldexp(1.0, -d.phi_F), G0.cells);
}


// ------------------------------------------------------------------ semi-implicit solve
VCArrays vc_arrays(const Dev& d, int l)
{
    const VCLevel& V = d.vc[l];
    return VCArrays{ V.fx, V.fy, V.fz, V.dg, V.idg };
}

// One V-cycle of the variable-coefficient system from level l (RB-GS, the
// colour order of the constant-coefficient cycle); levels of at most 16^3
// cells run in the fused coarse kernel, whose coarsest level is relaxed by
// 48 sweep pairs.
static void vcycle_vc(const Dev& d, int l, int R, int nu1, int nu2, cudaStream_t s)
{
    const Geo G = geo(d, l, R);
    double* phi = d.lev[l].phi;
    const double* rhs = d.lev[l].rhs;
    const int tpb = 256;
    if (G.n <= COARSE_VC_N && d.nlev - l >= 2) {
        CoarseVC C{};
        C.nlev = d.nlev - l;
        for (int q = 0; q < C.nlev; ++q) {
            C.n[q] = d.lev[l + q].n;
            C.phi[q] = d.lev[l + q].phi;
            C.rhs[q] = d.lev[l + q].rhs;
            C.A[q] = vc_arrays(d, l + q);
        }
        ++g_launches;
        k_vcycle_coarse_vc<<<R, 512, 0, s>>>(C, nu1, nu2, 48);
        return;
    }
    const VCArrays A = vc_arrays(d, l);
    auto sweep = [&](int color) {
        ++g_launches;
        k_smooth_vc<<<gridsz(G.cells / 2, tpb), tpb, 0, s>>>(phi, rhs, A, G, color);
    };
    for (int it = 0; it < nu1; ++it) { sweep(0); sweep(1); }
    const Geo Gc = geo(d, l + 1, R);
    ++g_launches;
    k_resid_restrict_vc<<<gridsz(Gc.cells, tpb), tpb, 0, s>>>(phi, rhs, A, d.lev[l + 1].rhs, Gc, G.n);
    cudaMemsetAsync(d.lev[l + 1].phi, 0, Gc.cells * sizeof(double), s);
    vcycle_vc(d, l + 1, R, nu1, nu2, s);
    launch_prolong<double>(phi, d.lev[l + 1].phi, G, s);
    for (int it = 0; it < nu2; ++it) { sweep(1); sweep(0); }
}

// One variable-coefficient V-cycle from the graph of kind 2 (captured once
// per smoother pair: the operator arrays keep their addresses).
static void run_cycle_vc(Dev& d, int R, int nu1, int nu2, cudaStream_t s)
{
    const int k = 2;
    if (d.direct_cycles) { vcycle_vc(d, 0, R, nu1, nu2, s); return; }
    if (d.vgraph[k] && (d.vgraph_nu[k][0] != nu1 || d.vgraph_nu[k][1] != nu2)) {
        cudaGraphExecDestroy(d.vgraph[k]);
        d.vgraph[k] = nullptr;
    }
    if (!d.vgraph[k]) {
        cudaGraph_t g = nullptr;
        if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            cudaGetLastError();
            vcycle_vc(d, 0, R, nu1, nu2, s);
            return;
        }
        const unsigned long long l0 = g_launches.load();
        vcycle_vc(d, 0, R, nu1, nu2, s);
        const unsigned long long nk = g_launches.load() - l0;
        g_launches -= nk;
        if (cudaStreamEndCapture(s, &g) != cudaSuccess || !g ||
            cudaGraphInstantiate(&d.vgraph[k], g, 0) != cudaSuccess) {
            cudaGetLastError();
            if (g) cudaGraphDestroy(g);
            d.vgraph[k] = nullptr;
            vcycle_vc(d, 0, R, nu1, nu2, s);
            return;
        }
        cudaGraphDestroy(g);
        d.vgraph_nu[k][0] = nu1;
        d.vgraph_nu[k][1] = nu2;
        d.vgraph_kernels[k] = nk;
    }
    g_launches += d.vgraph_kernels[k];
    cudaGraphLaunch(d.vgraph[k], s);
}

// Coefficients of the semi-implicit field (Sec. 4.7 step 1) into c0 from the
// electron deposit in d.ne_fix (the particles at the start of the step).
void launch_semi_coef(const Params& P, Dev& d, double* c0, cudaStream_t s)
{
    const Geo G0 = geo(d, 0, P.R);
    const double dV = P.h[0] * P.h[1] * P.h[2];
    const double per_cell = std::ldexp(1.0, -3 * P.frac_bits) / dV;
    ++g_launches;
    k_coef_from_ne<<<gridsz(G0.cells, 256), 256, 0, s>>>(d.ne_fix, c0, G0.cells, per_cell, 1.602176634e-19 * P.mu,
                                                          P.dt / 8.8541878128e-12);
}

// Semi-implicit field (Sec. 4.7 step 3, FP64 form): the level-0
// coefficients in d.vc[0].c (launch_semi_coef), restricted to the coarser
// levels, each level's face coefficients and diagonal, the right-hand side
// from d.rho (the charge of the diffused particles), FP64 V-cycles until
// ||r|| <= rtol ||b|| per realization, then E = -grad(phi) into d.E.  acc 2 R
// doubles of device scratch, acc_host its pinned mirror.  Returns 0, -6 (no
// convergence) or -3 (CUDA error).
int field_solve_vc(const Params& P, Dev& d, double* acc, double* acc_host, double rtol, int nu1, int nu2,
                   int max_cycles, cudaStream_t s, int* cycles_out, double* rel_out)
{
    const int R = P.R;
    const Geo G0 = geo(d, 0, R);
    const int tpb = 256;
    for (int l = 0; l + 1 < d.nlev; ++l) {
        const Geo Gc = geo(d, l + 1, R);
        ++g_launches;
        k_coef_restrict<<<gridsz(Gc.cells, tpb), tpb, 0, s>>>(d.vc[l].c, d.vc[l + 1].c, Gc, d.lev[l].n);
    }
    for (int l = 0; l < d.nlev; ++l) {
        const Geo G = geo(d, l, R);
        const VCLevel& V = d.vc[l];
        ++g_launches;
        k_vc_faces<<<gridsz(G.cells, tpb), tpb, 0, s>>>(V.c, V.fx, V.fy, V.fz, V.dg, V.idg, G);
    }
    double qscale, bc_top;
    rhs_consts(P, qscale, bc_top);
    ++g_launches;
    k_rhs_vc<<<gridsz(G0.cells, tpb), tpb, 0, s>>>(d.rho, d.vc[0].c, d.lev[0].rhs, G0, qscale, bc_top,
                                                    P.h[2] * P.h[2]);
    const VCArrays A0 = vc_arrays(d, 0);
    int cyc = 0, status = -6;
    double worst = 0.0;
    for (cyc = 0; cyc <= max_cycles; ++cyc) {
        g_launches += 2;
        const uint64_t per = G0.cells / (uint64_t)R;
        const dim3 ng((unsigned)gridsz(per, tpb), (unsigned)R);
        k_resid_norm_vc<<<ng, tpb, 0, s>>>(d.lev[0].phi, d.lev[0].rhs, A0, G0, d.norm_part);
        k_norm_final<<<R, 256, 0, s>>>(d.norm_part, (int)ng.x, R, acc);
        cudaMemcpyAsync(acc_host, acc, 2 * R * sizeof(double), cudaMemcpyDeviceToHost, s);
        if (cudaStreamSynchronize(s) != cudaSuccess) return -3;
        worst = 0.0;
        bool done = true;
        for (int r = 0; r < R; ++r) {
            const double rn = std::sqrt(acc_host[2 * r]), bn = std::sqrt(acc_host[2 * r + 1]);
            const double rel = bn > 0.0 ? rn / bn : rn;
            if (rel > worst || !(rel == rel)) worst = rel;
            if (!(rn <= rtol * bn)) done = false;
        }
        if (done) { status = 0; break; }
        if (cyc == max_cycles || !std::isfinite(worst)) break;
        run_cycle_vc(d, R, nu1, nu2, s);
    }
    if (cycles_out) *cycles_out = cyc;
    if (rel_out) *rel_out = worst;
    launch_efield_to(P, d, s, d.E, d.E32);
    return status;
}

}  // namespace ik

// ===========================================================================
// Field solve without device allocation (itokmc_field_solve_noalloc).
//
// Some callers cannot call cudaMalloc: a host program whose device memory
// belongs to another runtime's pool with a fixed budget, code that must not
// incur the implicit device synchronisation of cudaMalloc/cudaFree inside a
// latency-critical loop, or a plugin whose host forbids new device
// allocations.  For them the multigrid scratch (coarse levels, FP32 copies,
// right-hand side, norm partials and the packed field) lives in this
// file-scope device array, which every GPU that loads the library keeps
// until the process exits.  The caller passes the charge, the potential and
// the field buffers.
// ===========================================================================
namespace ik {
namespace {

constexpr size_t NOALLOC_BYTES = 16u << 20;     // 16 MiB: grids up to 64^3
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

std::mutex g_noalloc_mtx;
constexpr int NOALLOC_MAX_DEV = 64;
void* g_noalloc_ptr[NOALLOC_MAX_DEV] = {};

// h^2 b with b = -rho/eps0 and the electrode potentials folded in (as the
// step does).
__global__ void k_rhs_from_rho(const int64_t* __restrict__ rho, double* __restrict__ rhs, int n, int log2n,
                               double qscale, double phi_top, double h)
{
    const uint64_t cells = (uint64_t)n * n * n;
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < cells; g += (uint64_t)gridDim.x * blockDim.x) {
        const int k = (int)(g >> (2 * log2n));
        double b = -((double)rho[g] * qscale) / 8.8541878128e-12;
        if (k == n - 1) b = b - 2.0 * phi_top / (h * h);
        rhs[g] = b * (h * h);
    }
}

size_t carve(size_t& off, size_t bytes)
{
    const size_t at = off;
    off = (off + bytes + 255) & ~(size_t)255;
    return at;
}

}  // namespace
}  // namespace ik

extern "C" int itokmc_field_solve_noalloc(const itokmc_config* cfg, const int64_t* rho, double* phi, double* E,
                                          int32_t* cycles_out, double* rel_out)
{
    using namespace ik;
    if (!cfg || !rho || !phi || !E) { set_global_error("field_solve_noalloc: NULL argument"); return ITOKMC_ERR_ARG; }
    const int n = cfg->n[0];
    if (cfg->n_realizations != 1 || cfg->n[1] != n || cfg->n[2] != n || n < 8 || (n & (n - 1))) {
        set_global_error("field_solve_noalloc: one realization on an n^3 grid, n a power of two >= 8");
        return ITOKMC_ERR_ARG;
    }
    if (n > ITOKMC_NOALLOC_MAX_N) {
        set_global_error("field_solve_noalloc: grid larger than ITOKMC_NOALLOC_MAX_N (64) cells per axis");
        return ITOKMC_ERR_ARG;
    }
    if ((cfg->precision != ITOKMC_FP64 && cfg->precision != ITOKMC_MIXED) ||
        (cfg->field_precision != -1 && cfg->field_precision != ITOKMC_FP64 && cfg->field_precision != ITOKMC_MIXED)) {
        set_global_error("field_solve_noalloc: precision must be ITOKMC_FP64 or ITOKMC_MIXED (field_precision also -1)");
        return ITOKMC_ERR_ARG;
    }
    const int fp = cfg->field_precision < 0 ? cfg->precision : cfg->field_precision;
    // FP64 V-cycles, or FP32 V-cycles inside FP64 residual refinement
    const int prec = fp == ITOKMC_MIXED ? 1 : 0;
    cudaStream_t s = (cudaStream_t)cfg->stream;
    // set-up once per device, with that device current: the device address
    // of the scratch array (its name is only a stand-in in host code)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEV) {
        cudaGetLastError();
        set_global_error("field_solve_noalloc: no current CUDA device");
        return ITOKMC_ERR_CUDA;
    }
    unsigned char* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mtx);
        if (!g_noalloc_ptr[dev]) {
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                set_global_error("field_solve_noalloc: cudaGetSymbolAddress of the scratch array failed");
                return ITOKMC_ERR_CUDA;
            }
            g_noalloc_ptr[dev] = p;
        }
        base = static_cast<unsigned char*>(g_noalloc_ptr[dev]);
    }
    // lay the hierarchy out in the scratch array
    Params P{};
    P.n = n; P.n3 = n * n * n; P.R = 1;
    while ((1 << P.log2n) < n) ++P.log2n;
    for (int a = 0; a < 3; ++a) {
        P.lo[a] = cfg->lo[a]; P.hi[a] = cfg->hi[a]; P.h[a] = (cfg->hi[a] - cfg->lo[a]) / n;
        P.rh[a] = 1.0 / P.h[a];
    }
    P.E0 = cfg->E0;
    P.frac_bits = cfg->frac_bits;
    Dev d;
    d.direct_cycles = true;            // no graph objects: nothing is instantiated per call
    // the field is formed after the cycles, so its array shares its place with
    // the finest level's right-hand sides and second array
    // the cycles load and store the potential by pairs: a caller's array that
    // is not aligned to them (the ABI asks for a double's alignment) is solved
    // in a copy, which shares that place too
    const bool copy = reinterpret_cast<uintptr_t>(phi) % (2 * sizeof(double)) != 0;
    size_t off = 0;
    d.E = reinterpret_cast<E64*>(base + carve(off, (size_t)P.n3 * sizeof(E64)));
    d.E32 = nullptr;
    size_t top = 0;
    int l = 0;
    for (int m = n; m >= 4 && l < MAX_LEVELS; m >>= 1, ++l) {
        MGLevel& L = d.lev[l];
        const size_t cells = (size_t)m * m * m;
        size_t& at = l == 0 ? top : off;
        L.n = m;
        L.h = P.h[0] * (double)(n / m);
        L.phi = l == 0 && !copy ? phi : reinterpret_cast<double*>(base + carve(at, cells * sizeof(double)));
        L.rhs = reinterpret_cast<double*>(base + carve(at, cells * sizeof(double)));
        L.alt = base + carve(at, cells * sizeof(double));
        L.rhs_fix = reinterpret_cast<long long*>(l == 0 ? base + carve(at, cells * sizeof(long long))
                                                        : reinterpret_cast<unsigned char*>(L.rhs));
        L.phi_fix = reinterpret_cast<long long*>(l == 0 ? base + carve(off, cells * sizeof(long long))
                                                        : reinterpret_cast<unsigned char*>(L.phi));
        L.phi32 = reinterpret_cast<float*>(base + carve(off, cells * sizeof(float)));
        L.rhs32 = reinterpret_cast<float*>(base + carve(off, cells * sizeof(float)));
    }
    d.nlev = l;
    d.norm_part = reinterpret_cast<double*>(base + carve(off, 2 * ((size_t)P.n3 / 256 + 16) * sizeof(double)));
    d.norm_out = reinterpret_cast<double*>(base + carve(off, 2 * sizeof(double)));
    d.fix = reinterpret_cast<FixScale*>(base + carve(off, sizeof(FixScale)));
    if (top > (size_t)P.n3 * sizeof(E64)) {
        set_global_error("field_solve_noalloc: scratch layout exceeds the static array");
        return ITOKMC_ERR_ARG;
    }
    if (off > NOALLOC_BYTES) {
        set_global_error("field_solve_noalloc: scratch layout exceeds the static array");
        return ITOKMC_ERR_ARG;
    }
    alignas(FixScale) double norm_host[2 + FIX_DOUBLES];   // stack memory: no allocation
    d.norm_host = norm_host;
    const double dV = P.h[0] * P.h[1] * P.h[2];
    const double qscale = 1.602176634e-19 * ldexp(1.0, -3 * P.frac_bits) / dV;
    const double phi_top = P.E0 * (P.hi[2] - P.lo[2]);
    ++g_launches;
    k_rhs_from_rho<<<gridsz((uint64_t)P.n3, 256), 256, 0, s>>>(rho, d.lev[0].rhs, n, P.log2n, qscale, phi_top, P.h[0]);
    const size_t phi_bytes = (size_t)P.n3 * sizeof(double);
    if (copy) cudaMemcpyAsync(d.lev[0].phi, phi, phi_bytes, cudaMemcpyDeviceToDevice, s);
    int cycles = 0;
    double rel = 0.0;
    const int st = field_solve(P, d, prec, cfg->mg_rtol, cfg->mg_nu1, cfg->mg_nu2, 0ull, cfg->mg_max_cycles, s, &cycles,
                               &rel);
    if (cycles_out) *cycles_out = cycles;
    if (rel_out) *rel_out = rel;
    if (st == -3) {
        set_global_error("field_solve_noalloc: CUDA error in the multigrid");
        return ITOKMC_ERR_CUDA;
    }
    if (copy) {
        cudaMemcpyAsync(phi, d.lev[0].phi, phi_bytes, cudaMemcpyDeviceToDevice, s);
        d.lev[0].phi = phi;
    }
    launch_efield(P, d, s);
    const uint64_t G = (uint64_t)P.n3;
    ++g_launches;
    k_unpack_field<<<gridsz(G, 256), 256, 0, s>>>(d.E, nullptr, E, G);
    const cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_global_error("field_solve_noalloc: CUDA error");
        return ITOKMC_ERR_CUDA;
    }
    if (st != 0) {
        set_global_error("field_solve_noalloc: multigrid did not reach mg_rtol within mg_max_cycles");
        return ITOKMC_ERR_NOCONV;
    }
    return ITOKMC_OK;
}
