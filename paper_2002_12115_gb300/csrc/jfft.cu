// 3-D complex FFT block of libjac (include/jfft.h): the FFT workload of the
// paper's evaluation (NAS.FT, Section 5.1.1) and the function-block offload
// it names as next step (Section 6), device-resident on GB300.
//
// One kernel launch per axis.  A CTA owns W whole lines along the axis of
// the pass and transforms them in registers and shared memory:
//   * mixed-radix Stockham FFT of length N = R1 R2 R3 (radices 2..16):
//     stage s reads R values at stride N / R, multiplies by the twiddles
//     W_{Ns R}^{(j mod Ns) r} (from a table per stage computed on the host in
//     FP64), does an R-point DFT in registers (radix-2 decimation in
//     frequency with constant twiddles, its bit-reversed output order folded
//     into the register indices) and writes R values at stride Ns, Ns = R1
//     ... R(s-1);
//   * the first stage reads global memory and the last writes it; the
//     stages between exchange through a padded shared-memory tile;
//   * passes along y and z give a CTA W lines of consecutive x (W * element
//     size = 128 bytes), lanes running over those lines, so every global
//     access is a run of 128 bytes; the pass along x gives a CTA W rows with
//     lanes running along the row;
//   * the spectral step multiplies the data by exp(-4 pi^2 alpha t |kbar|^2)
//     as the first pass loads it (a per-CTA table of the factor along the
//     axis times one factor per line), and the last pass scales by 1/N as it
//     stores and sums |u|^2 per CTA in FP64; a one-CTA kernel then adds the
//     per-CTA sums in a fixed order, so the energy is bitwise reproducible.
// What bounds a pass: FP32 passes of 512 points run at 4-5 TB/s of their own
// reads and writes even when all of them hit L2, so instructions and latency
// bound them, not DRAM; FP64 passes are bound by the FP64 pipe.  Hence
// element offsets of a butterfly are constants (shared memory, twiddles) or a
// running pointer (global), indices are 32 bits, and factors of 1 are not
// multiplied by.  Before and after, on one GB300: x pass of 512x512x512 FP32
// in 64 -> 48 registers; forward and one spectral step on 512^3 FP32 2.75 ->
// 2.42 ms, on 256x256x128 FP64 2.67 -> 2.36 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/jfft.h"
#include "jac_common.cuh"
#include "jac_internal.h"

namespace jfft {

template <typename T>
struct alignas(2 * sizeof(T)) C2 {
    T x, y;
};

template <typename T>
__device__ __forceinline__ C2<T> operator+(C2<T> a, C2<T> b) { return {a.x + b.x, a.y + b.y}; }
template <typename T>
__device__ __forceinline__ C2<T> operator-(C2<T> a, C2<T> b) { return {a.x - b.x, a.y - b.y}; }

// z * w (INV = false) or z * conj(w) (INV = true)
template <typename T, bool INV>
__device__ __forceinline__ C2<T> cmul(C2<T> z, C2<T> w)
{
    if (INV) return {z.x * w.x + z.y * w.y, z.y * w.x - z.x * w.y};
    return {z.x * w.x - z.y * w.y, z.x * w.y + z.y * w.x};
}

// cos(2 pi m / 16)
__host__ __device__ constexpr double cos16(int m)
{
    m &= 15;
    if (m > 8) m = 16 - m;
    return m == 0   ? 1.0
           : m == 1 ? 0.92387953251128675613
           : m == 2 ? 0.70710678118654752440
           : m == 3 ? 0.38268343236508977173
           : m == 4 ? 0.0
           : m == 5 ? -0.38268343236508977173
           : m == 6 ? -0.70710678118654752440
           : m == 7 ? -0.92387953251128675613
                    : -1.0;
}

// z * exp(-+ 2 pi i m / 16) (forward: minus), m a compile-time constant
// after unrolling; the trivial factors 1 and -+i cost no multiply.
template <typename T, bool INV, int M>
__device__ __forceinline__ C2<T> rot16(C2<T> z)
{
    constexpr int m = M & 15;
    if constexpr (m == 0) {
        return z;
    } else if constexpr (m == 4) {
        return INV ? C2<T>{-z.y, z.x} : C2<T>{z.y, -z.x};
    } else {
        constexpr T c = (T)cos16(m), s = (T)cos16(m + 12);   // sin(2 pi m / 16)
        return INV ? C2<T>{z.x * c - z.y * s, z.x * s + z.y * c} : C2<T>{z.x * c + z.y * s, z.y * c - z.x * s};
    }
}

// One level of the in-register radix-2 decimation-in-frequency DFT of R
// points: butterflies of span HALF, then the next level.  After all levels
// X[k] sits at v[brev(k)].
template <typename T, int R, int HALF, bool INV>
struct Dif {
    template <int BLK, int K>
    static __device__ __forceinline__ void bfly(C2<T> *v)
    {
        if constexpr (BLK < R) {
            if constexpr (K < HALF) {
                const C2<T> a = v[BLK + K], b = v[BLK + K + HALF];
                v[BLK + K] = a + b;
                v[BLK + K + HALF] = rot16<T, INV, K * (8 / HALF)>(a - b);
                bfly<BLK, K + 1>(v);
            } else {
                bfly<BLK + 2 * HALF, 0>(v);
            }
        }
    }
    static __device__ __forceinline__ void run(C2<T> *v)
    {
        bfly<0, 0>(v);
        Dif<T, R, HALF / 2, INV>::run(v);
    }
};
template <typename T, int R, bool INV>
struct Dif<T, R, 0, INV> {
    static __device__ __forceinline__ void run(C2<T> *) {}
};

__host__ __device__ constexpr int brev(int k, int R)
{
    int r = 0;
    for (int b = 1; b < R; b <<= 1) {
        r = (r << 1) | (k & 1);
        k >>= 1;
    }
    return r;
}

// Radices of a length-N transform: up to three stages of at most 16.
template <int N>
struct Radix {
    static constexpr int R1 = N <= 16 ? N : (N == 32 ? 4 : (N == 64 ? 8 : (N == 128 ? 8 : (N == 256 ? 16 :
                                                            (N == 512 ? 8 : 4)))));
    static constexpr int R2 = N <= 16 ? 1 : (N == 32 ? 8 : (N == 64 ? 8 : (N == 128 ? 16 : (N == 256 ? 16 :
                                                            (N == 512 ? 8 : 16)))));
    static constexpr int R3 = N <= 256 ? 1 : (N == 512 ? 8 : 16);
    static constexpr int RMAX = R1 > R2 ? (R1 > R3 ? R1 : R3) : (R2 > R3 ? R2 : R3);
    static_assert(R1 * R2 * R3 == N, "radix plan");
    // The twiddles of the second and third stage: W^{jm r} of its length for
    // jm < NS and r = 1 .. R-1 at [(r - 1) NS + jm], so that a butterfly reads
    // them at constant offsets from jm.  N - R1 values in all.
    static constexpr int TW3 = R1 * (R2 - 1), TW = N - R1;
};

// Elements of a line each thread holds.  The pass along x keeps the
// largest radix (more lanes along each row); the passes along y and z take
// up to 16, so that fewer threads serve a line and a CTA of at most 512
// threads covers up to 256 bytes of consecutive x.
template <typename T, int N, bool YZ>
__host__ __device__ constexpr int elems_per_thread()
{
    constexpr int rmax = Radix<N>::RMAX;
    constexpr int want = N / 16 > rmax ? N / 16 : rmax;
    return YZ ? (want < 16 ? want : 16) : rmax;
}

// CTAs per SM the kernel is built for: for FP32, two 512-thread CTAs of the
// passes along y and z and four 256-thread CTAs of the pass along x (at
// most 64 registers a thread), so that one CTA's loads overlap another's
// butterflies; FP64 (bound by its ALU) keeps the registers it wants.
template <typename T, bool YZ>
__host__ __device__ constexpr int min_ctas_per_sm()
{
    return sizeof(T) == 4 ? (YZ ? 2 : 4) : 1;
}

// Shared-memory index of element e of a line: one pad element after every
// 16 (FP32) or 8 (FP64) elements, so that butterfly writes at stride R do
// not fall on one bank.
template <typename T>
__host__ __device__ constexpr int pad_idx(int e)
{
    return sizeof(T) == 4 ? e + (e >> 4) : e + (e >> 3);
}
// pad_idx(a + x) = pad_idx(a) + pad_idx(x) for the indices of a stage: a lies
// in a block of S elements that starts at a multiple of S (a power of two)
// and x is a multiple of S, or the roles are swapped, so no carry crosses the
// pad's digits.  The elements of a butterfly are then constants apart.

// Row stride of the tile (elements): the padded line plus one, with the
// stride odd in units of 32 bytes, so that lanes on different lines at the
// same element do not share a bank.
template <typename T, int N>
__host__ __device__ constexpr int row_stride()
{
    constexpr int a = sizeof(T) == 4 ? 16 : 8;
    return (pad_idx<T>(N - 1) + 1 + a - 1) / a * a + 1;
}

struct PassArgs {
    const void *in;
    void *out;
    const void *tw;          // this axis' twiddles by stage (Radix<N>; forward sign)
    int n1, n2, n3;
    int axis;                // 0: x, 1: y, 2: z
    int W;                   // lines per CTA
    double scale;            // applied by the last stage (1 or 1/N)
    int factor;              // multiply by the spectral factor on load (first pass of a step)
    const void *fa;          // factor tables exp(c kbar^2) (element type T): this pass's axis,
    const void *fb;          // and the line's other two axes (for the pass along x: y, then z)
    const void *fc;
    double *partials;        // per-CTA sums of |u|^2 (written when energy != NULL)
    double *energy;
};

__device__ __forceinline__ double kbar2(int k, int n)
{
    const int s = k < (n + 1) / 2 ? k : k - n;
    return (double)s * (double)s;
}

// Programmatic dependent launch: a pass lets the next launch of the stream
// start its prologue as soon as every CTA of this one runs, and waits for
// everything before it in the stream ahead of its own first data access.
using jac::launch_dependents;
using jac::wait_prior_grids;

// The spectral factor along each axis, exp(c kbar^2) for every index of
// n1, then n2, then n3 (FP64 exp, stored as T): one small launch per step,
// so that a pass multiplies by a table entry per element and one per line.
template <typename T>
__global__ void k_fft_factors(double c, int n1, int n2, int n3, T *f1, T *f2, T *f3)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    launch_dependents();
    wait_prior_grids();            // an earlier step may still read the tables
    if (i < n1) f1[i] = (T)exp(c * kbar2(i, n1));
    else if (i < n1 + n2) f2[i - n1] = (T)exp(c * kbar2(i - n1, n2));
    else if (i < n1 + n2 + n3) f3[i - n1 - n2] = (T)exp(c * kbar2(i - n1 - n2, n3));
}

// 8 or 16 bytes global -> shared without a register round trip.
template <typename E>
__device__ __forceinline__ void copy_async(E *smem_dst, const E *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(smem_dst)),
                 "l"(src), "n"((int)sizeof(E))
                 : "memory");
}

// A thread's elements of a line are t + k TT, k = 0 .. RMAX-1; butterfly q of
// a radix-R stage holds those with k = q + r RMAX / R.  The first stage's
// inputs from `line` (this line's first element; es: its element stride).
template <typename T, int N, int R, int RMAX>
__device__ __forceinline__ void load_line(C2<T> (&v)[RMAX], const C2<T> *line, unsigned es, int t)
{
    constexpr int TT = N / RMAX, BPT = RMAX / R;
    const C2<T> *p = line + (unsigned)t * es;
#pragma unroll
    for (int k = 0; k < RMAX; ++k, p += TT * es) v[(k % BPT) * R + k / BPT] = *p;
}

// The last stage's outputs to `line`.
template <typename T, int N, int R, int RMAX>
__device__ __forceinline__ void store_line(const C2<T> (&v)[RMAX], C2<T> *line, unsigned es, int t)
{
    constexpr int TT = N / RMAX, BPT = RMAX / R;
    C2<T> *p = line + (unsigned)t * es;
#pragma unroll
    for (int k = 0; k < RMAX; ++k, p += TT * es) *p = v[(k % BPT) * R + brev(k / BPT, R)];
}

// One Stockham stage for the BPT = RMAX / R butterflies of this thread: the
// first finds its inputs in v, the last leaves its outputs there (the output
// of index j + r N/R at v[q R + brev(r)]).
template <typename T, int N, int R, int RMAX, int NS, bool INV, bool FIRST, bool LAST>
__device__ __forceinline__ void stage(C2<T> (&v)[RMAX], C2<T> *row, const C2<T> *tw, int t)
{
    constexpr int TT = N / RMAX;       // threads per line
    constexpr int BPT = RMAX / R;      // butterflies per thread
    if constexpr (!FIRST) {
#pragma unroll
        for (int q = 0; q < BPT; ++q) {
            const C2<T> *p = row + pad_idx<T>(t + q * TT);
#pragma unroll
            for (int r = 0; r < R; ++r) v[q * R + r] = p[pad_idx<T>(r * (N / R))];
        }
    }
    if constexpr (!FIRST && !LAST) __syncthreads();   // every read of the tile before any write
#pragma unroll
    for (int q = 0; q < BPT; ++q) {
        if constexpr (NS > 1) {
            const C2<T> *w = tw + ((t + q * TT) & (NS - 1));
#pragma unroll
            for (int r = 1; r < R; ++r) v[q * R + r] = cmul<T, INV>(v[q * R + r], w[(r - 1) * NS]);
        }
        Dif<T, R, R / 2, INV>::run(&v[q * R]);
    }
    if constexpr (!LAST) {
#pragma unroll
        for (int q = 0; q < BPT; ++q) {
            const int j = t + q * TT;
            C2<T> *p = row + pad_idx<T>((j / NS) * NS * R + (j & (NS - 1)));
#pragma unroll
            for (int r = 0; r < R; ++r) p[pad_idx<T>(r * NS)] = v[q * R + brev(r, R)];
        }
        __syncthreads();
    }
}

template <typename T, int N, bool INV, bool YZ>
__global__ void __launch_bounds__(YZ ? 512 : 256, min_ctas_per_sm<T, YZ>()) k_fft_pass(const PassArgs a)
{
    using RX = Radix<N>;
    constexpr int RMAX = elems_per_thread<T, N, YZ>();   // elements per thread
    constexpr int TT = N / RMAX;
    constexpr int RS = row_stride<T, N>();
    extern __shared__ __align__(16) unsigned char jfft_smem[];
    constexpr int R1 = RX::R1, R2 = RX::R2, R3 = RX::R3;
    const int W = a.W;
    C2<T> *tile = reinterpret_cast<C2<T> *>(jfft_smem);
    C2<T> *tw = tile + (R2 > 1 ? W * RS : 0);
    T *fe = reinterpret_cast<T *>(tw + RX::TW);
    T *fl = fe + N;
    __shared__ double red[512];

    // This thread's line and position in it.  Element indices are at most
    // 2^30 (three extents of 1024), so 32 bits hold them.
    int w, t;
    if (!YZ) { t = threadIdx.x % TT; w = threadIdx.x / TT; }
    else { w = threadIdx.x % W; t = threadIdx.x / W; }
    const unsigned n1 = (unsigned)a.n1, n2 = (unsigned)a.n2;
    unsigned lb, es = 1;           // first element of the line, element stride
    int ia = 0, ib = 0;            // pass along x: the line's indices on the other two axes
    if (!YZ) {
        const unsigned row = blockIdx.x * W + w;                 // row = z * n2 + y
        lb = row * n1;
        ia = (int)(row % n2);
        ib = (int)(row / n2);
    } else {
        const unsigned xt = blockIdx.x % (n1 / W);
        const unsigned o = blockIdx.x / (n1 / W);                // z (y pass) or y (z pass)
        lb = (a.axis == 1 ? o * n1 * n2 : o * n1) + xt * W + w;
        es = a.axis == 1 ? n1 : n1 * n2;
    }

    launch_dependents();
    // the twiddles into shared memory (constant since the plan was made, so
    // their copies need not wait for earlier launches) ...
    const C2<T> *gtw = static_cast<const C2<T> *>(a.tw);
    if constexpr (R2 > 1)
        for (int m = threadIdx.x; m < RX::TW; m += blockDim.x) copy_async(&tw[m], &gtw[m]);
    asm volatile("cp.async.commit_group;" ::: "memory");
    wait_prior_grids();
    // ... and, with them in flight, this thread's part of its line
    const C2<T> *gin = static_cast<const C2<T> *>(a.in) + lb;
    C2<T> *gout = static_cast<C2<T> *>(a.out) + lb;
    C2<T> v[RMAX];
    load_line<T, N, R1, RMAX>(v, gin, es, t);
    if (!YZ && a.factor) {         // the spectral factor along this axis and of this line
        const T *gfa = static_cast<const T *>(a.fa);
        for (int m = threadIdx.x; m < N; m += blockDim.x) fe[m] = gfa[m];
        if (t == 0) fl[w] = static_cast<const T *>(a.fb)[ia] * static_cast<const T *>(a.fc)[ib];
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    const bool want_energy = YZ && a.energy != nullptr;
    if (!YZ && a.factor) {
        const T flw = fl[w];
#pragma unroll
        for (int q = 0; q < RMAX / R1; ++q)
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const T f = fe[t + q * TT + r * (N / R1)] * flw;
                v[q * R1 + r].x *= f;
                v[q * R1 + r].y *= f;
            }
    }
    C2<T> *row = tile + w * RS;
    constexpr int RL = R3 > 1 ? R3 : (R2 > 1 ? R2 : R1);         // radix of the last stage
    if constexpr (R2 == 1) {
        stage<T, N, R1, RMAX, 1, INV, true, true>(v, row, tw, t);
    } else {
        stage<T, N, R1, RMAX, 1, INV, true, false>(v, row, tw, t);
        if constexpr (R3 == 1) {
            stage<T, N, R2, RMAX, R1, INV, false, true>(v, row, tw, t);
        } else {
            stage<T, N, R2, RMAX, R1, INV, false, false>(v, row, tw, t);
            stage<T, N, R3, RMAX, R1 * R2, INV, false, true>(v, row, tw + RX::TW3, t);
        }
    }
    // Only the last pass of an inverse transform scales; elsewhere the factor
    // is 1 and its two multiplies per point (of about 25 in FP64, which its
    // pipe bounds) are left out.
    if (YZ && a.scale != 1.0) {
        const T scale = (T)a.scale;
#pragma unroll
        for (int q = 0; q < RMAX; ++q) { v[q].x *= scale; v[q].y *= scale; }
    }
    // the stride once more, opaque: without it the 16 offsets of the loads are
    // kept in registers for the stores (and spill)
    if (YZ) asm volatile("" : "+r"(es));
    store_line<T, N, RL, RMAX>(v, gout, es, t);
    T esum = (T)0;
    if (want_energy) {             // this thread's |u|^2, summed in T over its outputs
#pragma unroll
        for (int q = 0; q < RMAX / RL; ++q)
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                const C2<T> x = v[q * RL + brev(r, RL)];
                esum = fma(x.x, x.x, fma(x.y, x.y, esum));
            }
    }
    if (!want_energy) return;

    // energy: a pairwise tree over the block in T (warp shuffles, then the
    // warps' sums in shared memory; log2 of the block's size roundings, and
    // FP64 only for the CTA's one partial -- GB300's FP64 pipe is narrow);
    // k_fft_energy adds the partials after the pass
    __shared__ T tred[32];
    T v_e = esum;
    if ((blockDim.x & 31) == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v_e += __shfl_down_sync(0xffffffffu, v_e, o);
        if ((threadIdx.x & 31) == 0) tred[threadIdx.x >> 5] = v_e;
        __syncthreads();
        if (threadIdx.x < 32) {
            const int nw = blockDim.x >> 5;
            T x = threadIdx.x < nw ? tred[threadIdx.x] : (T)0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (threadIdx.x == 0) a.partials[blockIdx.x] = (double)x;
        }
    } else {                                   // blocks of fewer than 32 threads (short lines)
        red[threadIdx.x] = (double)v_e;
        __syncthreads();
        if (threadIdx.x == 0) {
            double sum = 0.0;
            for (unsigned i = 0; i < blockDim.x; ++i) sum += red[i];
            a.partials[blockIdx.x] = sum;
        }
    }
}

// Sum of the n per-CTA energy partials of the last pass, in a fixed order:
// thread t adds the partials t, t + 512, ... (four independent loads in
// flight), then a pairwise tree over the 512 threads.  One CTA of 512
// threads.  It may start while that pass still writes the partials, so the
// pointer is not __restrict__ and they are read through L2, after the wait.
__global__ void __launch_bounds__(512) k_fft_energy(const double *partials, int n, double *energy)
{
    __shared__ double red[512];
    const int t = threadIdx.x;
    launch_dependents();
    wait_prior_grids();
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int b = t; b < n; b += 4 * 512) {
        s0 += __ldcg(partials + b);
        if (b + 512 < n) s1 += __ldcg(partials + b + 512);
        if (b + 1024 < n) s2 += __ldcg(partials + b + 1024);
        if (b + 1536 < n) s3 += __ldcg(partials + b + 1536);
    }
    red[t] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    for (int h = 256; h > 0; h >>= 1) {
        if (t < h) red[t] += red[t + h];
        __syncthreads();
    }
    if (t == 0) *energy = red[0];
}

// ---------------------------------------------------------------- host
namespace {

bool pow2_in_range(int n) { return n >= JFFT_MIN_N && n <= JFFT_MAX_N && (n & (n - 1)) == 0; }

size_t elem_bytes(jfft_prec p) { return p == JFFT_C64 ? 16 : 8; }

size_t round256(size_t x) { return (x + 255) / 256 * 256; }

// Largest radix of a length-N transform (Radix<N>::RMAX), on the host.
int rmax_of(int N)
{
    if (N <= 16) return N;
    return (N == 32 || N == 64 || N == 512) ? 8 : 16;
}

// Radix<N>::R1, R2, R3 on the host.
void radices_of(int N, int r[3])
{
    static const int table[11][3] = {{1, 1, 1}, {2, 1, 1},  {4, 1, 1},   {8, 1, 1}, {16, 1, 1},   {4, 8, 1},
                                     {8, 8, 1}, {8, 16, 1}, {16, 16, 1}, {8, 8, 8}, {4, 16, 16}};
    int e = 0;
    while ((1 << e) < N) ++e;
    for (int q = 0; q < 3; ++q) r[q] = table[e][q];
}

// Elements per thread (elems_per_thread<T, N, YZ> on the host).
int elems_of(int N, jfft_prec prec, bool yz)
{
    (void)prec;
    const int rmax = rmax_of(N);
    if (!yz) return rmax;
    return std::min(std::max(N / 16, rmax), 16);
}

// Lines per CTA of a pass (see the kernel's mapping): rows of about 256
// threads for the pass along x; for y and z, 256 bytes of consecutive x
// (32 FP32 or 16 FP64 complex values), at most 512 threads.
int lines_per_cta(int axis, int N, const int n[3], jfft_prec prec)
{
    const int tt = N / elems_of(N, prec, axis != 0);
    if (axis == 0) return std::max(1, std::min(256 / tt, n[1] * n[2]));
    return std::max(1, std::min(std::min(prec == JFFT_C64 ? 16 : 32, n[0]), 512 / tt));
}

long long ctas_of_pass(int axis, const int n[3], int W)
{
    if (axis == 0) return (long long)n[1] * n[2] / W;
    return (long long)(n[0] / W) * (axis == 1 ? n[2] : n[1]);
}

int threads_of_pass(int N, int W, jfft_prec prec, bool yz) { return (N / elems_of(N, prec, yz)) * W; }

struct Layout {
    size_t tw[3];       // offsets of the twiddle tables
    size_t fac[3];      // offsets of the spectral factor tables
    size_t partials;
    size_t total;
    long long max_ctas;
};

Layout layout(const int n[3], jfft_prec prec)
{
    Layout L;
    size_t off = 256;                     // header (reserved)
    for (int a = 0; a < 3; ++a) {
        L.tw[a] = off;
        off += round256((size_t)n[a] * elem_bytes(prec));
    }
    for (int a = 0; a < 3; ++a) {
        L.fac[a] = off;
        off += round256((size_t)n[a] * elem_bytes(prec) / 2);
    }
    L.max_ctas = 0;
    for (int a = 0; a < 3; ++a)
        L.max_ctas = std::max(L.max_ctas, ctas_of_pass(a, n, lines_per_cta(a, n[a], n, prec)));
    L.partials = off;
    off += round256((size_t)L.max_ctas * sizeof(double));
    L.total = off;
    return L;
}

jac_status check_shape(int n1, int n2, int n3, jfft_prec prec)
{
    if (!pow2_in_range(n1) || !pow2_in_range(n2) || !pow2_in_range(n3)) {
        jac::set_thread_error("every extent must be a power of two in [" + std::to_string(JFFT_MIN_N) + ", " +
                              std::to_string(JFFT_MAX_N) + "]");
        return JAC_EINVAL;
    }
    if (prec != JFFT_C64 && prec != JFFT_C32) {
        jac::set_thread_error("unknown FFT precision");
        return JAC_EINVAL;
    }
    return JAC_OK;
}

}  // namespace

// A launch that may start before the stream's previous one has ended (its
// kernel waits for it, see wait_prior_grids).
template <typename... P, typename... A>
jac_status launch_chained(void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                          const char *what, A... args)
{
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
    if (e == cudaSuccess) return JAC_OK;
    jac::set_thread_error(std::string(what) + ": " + cudaGetErrorString(e));
    return JAC_ECUDA;
}

// Launch of one pass: the kernel instantiation for (T, N, INV).
template <typename T, bool INV, bool YZ>
jac_status launch_pass_t(int N, const PassArgs &a, unsigned grid, unsigned block, cudaStream_t st)
{
    size_t smem = 0;
    void (*kern)(PassArgs) = nullptr;
    switch (N) {
#define JFFT_CASE(NN)                                                                                       \
    case NN:                                                                                                \
        kern = k_fft_pass<T, NN, INV, YZ>;                                                                  \
        smem = (Radix<NN>::R2 > 1 ? (size_t)a.W * row_stride<T, NN>() * sizeof(C2<T>) : 0) +               \
               (size_t)Radix<NN>::TW * sizeof(C2<T>) + (size_t)NN * sizeof(T) + (size_t)a.W * sizeof(T);    \
        break;
        JFFT_CASE(2) JFFT_CASE(4) JFFT_CASE(8) JFFT_CASE(16) JFFT_CASE(32) JFFT_CASE(64) JFFT_CASE(128)
        JFFT_CASE(256) JFFT_CASE(512) JFFT_CASE(1024)
#undef JFFT_CASE
    default:
        jac::set_thread_error("unsupported FFT length");
        return JAC_EINVAL;
    }
    smem = (smem + 15) / 16 * 16;
    // opt in to more than the default dynamic shared memory (the kernel's
    // static reduction buffer counts against the same 48 KB); once per
    // kernel and size
    if (smem > 32 * 1024) {
        static std::mutex mu;
        static std::vector<std::pair<const void *, size_t>> done;
        std::lock_guard<std::mutex> lk(mu);
        auto it = std::find_if(done.begin(), done.end(), [&](const std::pair<const void *, size_t> &d) {
            return d.first == (const void *)kern;
        });
        if (it == done.end() || it->second < smem) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) {
                jac::set_thread_error(std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e));
                return JAC_ECUDA;
            }
            if (it == done.end()) done.emplace_back((const void *)kern, smem);
            else it->second = smem;
        }
    }
    return launch_chained(kern, grid, block, smem, st, "FFT pass launch", a);
}

}  // namespace jfft

struct jfft_plan {
    int n[3] = {0, 0, 0};
    jfft_prec prec = JFFT_C32;
    cudaStream_t stream = nullptr;
    char *ws = nullptr;
    jfft::Layout L{};
    std::string err;
};

namespace {

jac_status plan_fail(jfft_plan *p, jac_status s, const std::string &m)
{
    if (p) p->err = m;
    jac::set_thread_error(m);
    return s;
}

jac_status plan_from_thread(jfft_plan *p, jac_status s)
{
    if (s != JAC_OK && p) p->err = jac::thread_last_error();
    return s;
}

// The three passes of one transform.  first_in: the input of the first
// pass; every later pass works in place on `out`.
jac_status run3(jfft_plan *p, const void *in, void *out, bool inv, double scale, bool factor, double c,
                double *energy)
{
    if (!p) return plan_fail(p, JAC_EINVAL, "plan is NULL");
    if (!in || !out || (reinterpret_cast<uintptr_t>(in) & 15) || (reinterpret_cast<uintptr_t>(out) & 15))
        return plan_fail(p, JAC_EINVAL, "data arrays must be non-NULL and 16-byte aligned");
    if (in != out) {
        const size_t bytes = (size_t)p->n[0] * p->n[1] * p->n[2] * jfft::elem_bytes(p->prec);
        const char *a = static_cast<const char *>(in), *b = static_cast<const char *>(out);
        if (a < b + bytes && b < a + bytes) return plan_fail(p, JAC_EINVAL, "in and out overlap without being equal");
    }
    if (factor) {
        const unsigned blocks = (unsigned)(p->n[0] + p->n[1] + p->n[2] + 255) / 256;
        char *f[3] = {p->ws + p->L.fac[0], p->ws + p->L.fac[1], p->ws + p->L.fac[2]};
        const jac_status s =
            p->prec == JFFT_C32
                ? jfft::launch_chained(jfft::k_fft_factors<float>, blocks, 256, 0, p->stream, "factor launch", c, p->n[0],
                                       p->n[1], p->n[2], reinterpret_cast<float *>(f[0]),
                                       reinterpret_cast<float *>(f[1]), reinterpret_cast<float *>(f[2]))
                : jfft::launch_chained(jfft::k_fft_factors<double>, blocks, 256, 0, p->stream, "factor launch", c,
                                       p->n[0], p->n[1], p->n[2], reinterpret_cast<double *>(f[0]),
                                       reinterpret_cast<double *>(f[1]), reinterpret_cast<double *>(f[2]));
        if (s != JAC_OK) return plan_from_thread(p, s);
    }
    for (int axis = 0; axis < 3; ++axis) {
        const int N = p->n[axis];
        jfft::PassArgs a;
        std::memset(&a, 0, sizeof(a));
        a.in = axis == 0 ? in : out;
        a.out = out;
        a.tw = p->ws + p->L.tw[axis];
        a.n1 = p->n[0]; a.n2 = p->n[1]; a.n3 = p->n[2];
        a.axis = axis;
        a.W = jfft::lines_per_cta(axis, N, p->n, p->prec);
        a.scale = axis == 2 ? scale : 1.0;
        a.factor = (factor && axis == 0) ? 1 : 0;
        a.fa = p->ws + p->L.fac[0];
        a.fb = p->ws + p->L.fac[1];
        a.fc = p->ws + p->L.fac[2];
        if (axis == 2 && energy) {
            a.energy = energy;
            a.partials = reinterpret_cast<double *>(p->ws + p->L.partials);
        }
        const unsigned grid = (unsigned)jfft::ctas_of_pass(axis, p->n, a.W);
        const unsigned block = (unsigned)jfft::threads_of_pass(N, a.W, p->prec, axis != 0);
        jac_status s;
        const bool yz = axis != 0;
        if (p->prec == JFFT_C32)
            s = inv ? (yz ? jfft::launch_pass_t<float, true, true>(N, a, grid, block, p->stream)
                          : jfft::launch_pass_t<float, true, false>(N, a, grid, block, p->stream))
                    : (yz ? jfft::launch_pass_t<float, false, true>(N, a, grid, block, p->stream)
                          : jfft::launch_pass_t<float, false, false>(N, a, grid, block, p->stream));
        else
            s = inv ? (yz ? jfft::launch_pass_t<double, true, true>(N, a, grid, block, p->stream)
                          : jfft::launch_pass_t<double, true, false>(N, a, grid, block, p->stream))
                    : (yz ? jfft::launch_pass_t<double, false, true>(N, a, grid, block, p->stream)
                          : jfft::launch_pass_t<double, false, false>(N, a, grid, block, p->stream));
        if (s != JAC_OK) return plan_from_thread(p, s);
        if (axis == 2 && energy) {
            s = jfft::launch_chained(jfft::k_fft_energy, 1, 512, 0, p->stream, "energy launch",
                                     reinterpret_cast<const double *>(p->ws + p->L.partials), (int)grid, energy);
            if (s != JAC_OK) return plan_from_thread(p, s);
        }
    }
    return JAC_OK;
}

}  // namespace

extern "C" {

jac_status jfft_workspace_size(int n1, int n2, int n3, jfft_prec prec, size_t *bytes)
{
    if (!bytes) return plan_fail(nullptr, JAC_EINVAL, "bytes is NULL");
    jac_status s = jfft::check_shape(n1, n2, n3, prec);
    if (s != JAC_OK) return s;
    const int n[3] = {n1, n2, n3};
    *bytes = jfft::layout(n, prec).total;
    return JAC_OK;
}

jac_status jfft_plan_create(jfft_plan **out, int n1, int n2, int n3, jfft_prec prec, void *stream, void *workspace,
                            size_t ws_bytes)
{
    if (!out) return plan_fail(nullptr, JAC_EINVAL, "out is NULL");
    *out = nullptr;
    jac_status s = jfft::check_shape(n1, n2, n3, prec);
    if (s != JAC_OK) return s;
    const int n[3] = {n1, n2, n3};
    const jfft::Layout L = jfft::layout(n, prec);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return plan_fail(nullptr, JAC_EINVAL, "workspace must be non-NULL and 256-byte aligned");
    if (ws_bytes < L.total)
        return plan_fail(nullptr, JAC_EINVAL, "workspace too small: need " + std::to_string(L.total) + " bytes");
    jfft_plan *p = new (std::nothrow) jfft_plan;
    if (!p) return plan_fail(nullptr, JAC_ENOMEM, "host allocation failed");
    p->n[0] = n1; p->n[1] = n2; p->n[2] = n3;
    p->prec = prec;
    p->stream = static_cast<cudaStream_t>(stream);
    p->ws = static_cast<char *>(workspace);
    p->L = L;
    // twiddle tables of the stages (Radix<N>), exp(-2 pi i jm r / (NS R)), in FP64 on the host, stored in the
    // plan's precision
    std::vector<unsigned char> host(L.fac[0] - 256, 0);
    const double pi = 3.14159265358979323846264338327950288;
    for (int a = 0; a < 3; ++a) {
        unsigned char *dst = host.data() + (L.tw[a] - 256);
        int r3[3];
        jfft::radices_of(n[a], r3);
        int at = 0;
        for (int st = 1, ns = r3[0]; st < 3; ns *= r3[st], ++st)
            for (int r = 1; r < r3[st]; ++r)
                for (int jm = 0; jm < ns; ++jm, ++at) {
                    const int m = jm * r;                    // of ns * r3[st] points
                    const double ang = 2.0 * pi * m / (ns * r3[st]);
                    const double re = std::cos(ang), im = -std::sin(ang);
                    if (prec == JFFT_C64) {
                        const double v[2] = {re, im};
                        std::memcpy(dst + (size_t)at * 16, v, 16);
                    } else {
                        const float v[2] = {(float)re, (float)im};
                        std::memcpy(dst + (size_t)at * 8, v, 8);
                    }
                }
    }
    cudaError_t e = cudaMemsetAsync(p->ws, 0, 256, p->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p->ws + 256, host.data(), host.size(), cudaMemcpyHostToDevice, p->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    if (e != cudaSuccess) {
        delete p;
        return plan_fail(nullptr, JAC_ECUDA, std::string("plan set-up: ") + cudaGetErrorString(e));
    }
    *out = p;
    return JAC_OK;
}

jac_status jfft_destroy(jfft_plan *p)
{
    if (!p) return JAC_OK;
    cudaStreamSynchronize(p->stream);
    delete p;
    return JAC_OK;
}

const char *jfft_last_error(const jfft_plan *p) { return p ? p->err.c_str() : jac::thread_last_error(); }

jac_status jfft_forward(jfft_plan *p, const void *in, void *out)
{
    return run3(p, in, out, false, 1.0, false, 0.0, nullptr);
}

jac_status jfft_inverse(jfft_plan *p, const void *in, void *out)
{
    if (!p) return plan_fail(p, JAC_EINVAL, "plan is NULL");
    return run3(p, in, out, true, 1.0 / ((double)p->n[0] * p->n[1] * p->n[2]), false, 0.0, nullptr);
}

jac_status jfft_evolve(jfft_plan *p, const void *U, double alpha, double t, void *out, double *d_energy)
{
    if (!p) return plan_fail(p, JAC_EINVAL, "plan is NULL");
    if (!std::isfinite(alpha) || !std::isfinite(t) || alpha * t < 0.0)
        return plan_fail(p, JAC_EINVAL, "alpha and t must be finite with alpha * t >= 0");
    const double pi = 3.14159265358979323846264338327950288;
    const double c = -4.0 * pi * pi * alpha * t;
    return run3(p, U, out, true, 1.0 / ((double)p->n[0] * p->n[1] * p->n[2]), true, c, d_energy);
}

}  // extern "C"
