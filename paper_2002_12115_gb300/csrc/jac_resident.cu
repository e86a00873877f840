// Resident sweeps of libjac: small grids whose coefficients fit in the shared
// memory of all SMs together.
//
// The streaming kernel (jac_sweep_kernel.cuh) reads every coefficient again
// in every sweep and ends each sweep with a grid barrier and a refill of its
// rings; on small grids that fixed cost, not bandwidth, is what a sweep takes
// (33x33x65 FP64: 6.4 us a sweep, of which 2.1 us is FP64 arithmetic).  Here
// every CTA owns one box of the grid for all sweeps of a call: full rows in i,
// bj x bk rows in (j, k).
//   * The box's coefficients are copied into shared memory once per call, one
//     point's values in 16-byte vectors (array v of all points, so that the
//     lanes of a warp read consecutive vectors).
//   * The state of the box with a one-row halo lives in shared memory, double
//     buffered.  Only rows next to another box go through global memory (the
//     caller's state buffers, L2): the owner stores them, releases a flag,
//     and each of the up to eight neighbours polls that flag and copies its
//     part of the halo.  No CTA waits for more than its neighbours.
//   * Compute warps (one point per lane and turn, consecutive lanes along i)
//     update the rows next to other boxes first; while eight communication
//     warps, one per neighbour direction, publish and collect, the compute
//     warps update the inner rows.
//   * Safety of the two state buffers: a box stores sweep t+2's rows over
//     sweep t's only after every neighbour released sweep t+1's flag, which
//     it does after it copied sweep t's halo.
//   * With a history every state of the call is stored whole, each to its own
//     array (the reverse pass recomputes a checkpoint segment that way, in one
//     launch instead of one per sweep).
//   * The update is the streaming kernels' arithmetic in the same order, so
//     the state is bitwise theirs.  The last sweep stores the whole box; its ss
//     values, left in shared memory, give the residual (one partial per CTA).
//   * Every wait is bounded; on expiry the CTA sets the workspace error word
//     and returns, and the last CTA writes NaN as the residual.
// What is left is the exchange between neighbours (3.3 us: the stores reach
// L2, the flag follows, is seen, and the rows come back) plus the arithmetic
// (FP64) or the shared-memory reads of 19 state values and the coefficients
// per point (FP32).  Measured, us a sweep, streaming -> resident:
//   17x17x17 FP64 6.3 -> 3.7      33x33x65 FP64 6.4 -> 5.1   49x49x97 FP64 15.9 -> 10.9
//   33x33x65 FP32 4.5 -> 3.5      77x53x101 FP32 7.0 -> 4.8  65x65x129 FP32 6.5 -> 4.7
//   65x65x129 BF16 6.1 -> 4.2
// (80 registers at 768 threads: ptxas spills 20 bytes in FP32, 24 with BF16
// coefficients, 36 in FP64.)  Wide, flat grids are faster streaming: the rule is
// resident_pays in jac_sweep.cu.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>

#include "jac_internal.h"
#include "jac_sweep_kernel.cuh"

namespace jac {

namespace {

constexpr int kComputeWarps = 16, kCommWarps = 8;
constexpr int kWarps = kComputeWarps + kCommWarps;
constexpr int kCompute = 32 * kComputeWarps, kThreads = 32 * kWarps;
constexpr int kFlagStride = 8;                  // words between flags: one 32-byte sector each
constexpr size_t kSmemBudget = 225 * 1024;

struct ResArgs {
    const void *coef[12];      // JAC_A0 .. JAC_BND
    void *p_buf[2];            // state t of the call is in p_buf[t & 1]
    int I, J, K, pitch;
    int nj, nk;                // boxes along j and k
    int ucap, rcap;            // most points and rows of a box
    int bjm, bkm;              // most rows of a box along j and k
    int ws;                    // shared-memory row length (elements)
    int n_iter;
    double omega;
    double *partials;          // one per CTA
    double *res;
    unsigned *flags;           // one per CTA, kFlagStride words apart
    char *hist;                // not NULL: state t + 1 whole at hist + t * hist_stride
    size_t hist_stride;        // instead of in p_buf[(t + 1) & 1]
    WsHeader *hdr;
    unsigned long long wait_ns;   // limit of every wait on another CTA
    unsigned gbar_extra;       // added to the barrier's target: 0, except when a test of the failure path
                               // makes it unreachable
};

// Boxes split n rows into parts of nearly equal length.
__host__ __device__ inline int part_begin(int n, int parts, int b) { return (int)((long long)n * b / parts); }

// One point's coefficients as VEC 16-byte vectors.
template <typename T, typename C>
struct PointCoef;

template <>
struct PointCoef<double, double> {
    static constexpr int VEC = 6;
    double a0, a1, a2, a3, b0, b1, b2, c0, c1, c2, wk, bn;
    __device__ __forceinline__ void get(const uint4 *v, int cap)
    {
        double2 x;
        x = *reinterpret_cast<const double2 *>(v); a0 = x.x; a1 = x.y;
        x = *reinterpret_cast<const double2 *>(v + cap); a2 = x.x; a3 = x.y;
        x = *reinterpret_cast<const double2 *>(v + 2 * cap); b0 = x.x; b1 = x.y;
        x = *reinterpret_cast<const double2 *>(v + 3 * cap); b2 = x.x; c0 = x.y;
        x = *reinterpret_cast<const double2 *>(v + 4 * cap); c1 = x.x; c2 = x.y;
        x = *reinterpret_cast<const double2 *>(v + 5 * cap); wk = x.x; bn = x.y;
    }
    static __device__ __forceinline__ void put(uint4 *v, int cap, const void *const *coef, size_t off)
    {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            double2 x;
            x.x = __ldg(static_cast<const double *>(coef[2 * q]) + off);
            x.y = __ldg(static_cast<const double *>(coef[2 * q + 1]) + off);
            *reinterpret_cast<double2 *>(v + q * cap) = x;
        }
    }
};

template <>
struct PointCoef<float, float> {
    static constexpr int VEC = 3;
    float a0, a1, a2, a3, b0, b1, b2, c0, c1, c2, wk, bn;
    __device__ __forceinline__ void get(const uint4 *v, int cap)
    {
        float4 x;
        x = *reinterpret_cast<const float4 *>(v); a0 = x.x; a1 = x.y; a2 = x.z; a3 = x.w;
        x = *reinterpret_cast<const float4 *>(v + cap); b0 = x.x; b1 = x.y; b2 = x.z; c0 = x.w;
        x = *reinterpret_cast<const float4 *>(v + 2 * cap); c1 = x.x; c2 = x.y; wk = x.z; bn = x.w;
    }
    static __device__ __forceinline__ void put(uint4 *v, int cap, const void *const *coef, size_t off)
    {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            float4 x;
            x.x = __ldg(static_cast<const float *>(coef[4 * q]) + off);
            x.y = __ldg(static_cast<const float *>(coef[4 * q + 1]) + off);
            x.z = __ldg(static_cast<const float *>(coef[4 * q + 2]) + off);
            x.w = __ldg(static_cast<const float *>(coef[4 * q + 3]) + off);
            *reinterpret_cast<float4 *>(v + q * cap) = x;
        }
    }
};

template <>
struct PointCoef<float, __nv_bfloat16> {
    static constexpr int VEC = 2;
    float a0, a1, a2, a3, b0, b1, b2, c0, c1, c2, wk, bn;
    static __device__ __forceinline__ float lo(unsigned x) { return __uint_as_float(x << 16); }
    static __device__ __forceinline__ float hi(unsigned x) { return __uint_as_float(x & 0xffff0000u); }
    __device__ __forceinline__ void get(const uint4 *v, int cap)
    {
        uint4 x = *v;
        a0 = lo(x.x); a1 = hi(x.x); a2 = lo(x.y); a3 = hi(x.y);
        b0 = lo(x.z); b1 = hi(x.z); b2 = lo(x.w); c0 = hi(x.w);
        x = v[cap];
        c1 = lo(x.x); c2 = hi(x.x); bn = lo(x.y); wk = __uint_as_float(x.z);
    }
    static __device__ __forceinline__ unsigned bits(const void *p, size_t off)
    {
        return __ldg(static_cast<const unsigned short *>(p) + off);
    }
    static __device__ __forceinline__ void put(uint4 *v, int cap, const void *const *coef, size_t off)
    {
        uint4 x;
        x.x = bits(coef[0], off) | bits(coef[1], off) << 16;
        x.y = bits(coef[2], off) | bits(coef[3], off) << 16;
        x.z = bits(coef[4], off) | bits(coef[5], off) << 16;
        x.w = bits(coef[6], off) | bits(coef[7], off) << 16;
        v[0] = x;
        x.x = bits(coef[8], off) | bits(coef[9], off) << 16;
        x.y = bits(coef[11], off);                                   // bnd
        x.z = __float_as_uint(__ldg(static_cast<const float *>(coef[10]) + off));   // wrk1
        x.w = 0u;
        v[cap] = x;
    }
};

// ss of the point at P in a state with row stride W and plane stride Z; the
// operations of the streaming kernels, in their order.  FP64 leaves out the
// multiply by bnd where the whole box has bnd = 1 (not masked).
template <typename T, typename C>
__device__ __forceinline__ T res_ss(const T *P, int W, int Z, const PointCoef<T, C> &k, bool masked)
{
    const T c = P[0], xp = P[1], xm = P[-1], yp = P[W], ym = P[-W], zp = P[Z], zm = P[-Z];
    if constexpr (sizeof(T) == 4) {
        const T bij = ((P[W + 1] - P[-W + 1]) - P[W - 1]) + P[-W - 1];
        const T bjk = ((P[Z + W] - P[-Z + W]) - P[Z - W]) + P[-Z - W];
        const T bik = ((P[Z + 1] - P[-Z + 1]) - P[Z - 1]) + P[-Z - 1];
        return ss_f32<sizeof(C) == 2>(c, xp, xm, yp, ym, zp, zm, bij, bjk, bik, k.a0, k.a1, k.a2, k.a3, k.b0, k.b1,
                                      k.b2, k.c0, k.c1, k.c2, k.wk, k.bn);
    } else {
        const T bij = (P[W + 1] - P[-W + 1]) - (P[W - 1] - P[-W - 1]);
        const T bjk = (P[Z + W] - P[Z - W]) - (P[-Z + W] - P[-Z - W]);
        const T bik = (P[Z + 1] - P[Z - 1]) - (P[-Z + 1] - P[-Z - 1]);
        T s0 = k.wk;
        s0 = fma(k.a0, xp, s0);
        s0 = fma(k.a1, yp, s0);
        s0 = fma(k.a2, zp, s0);
        s0 = fma(k.b0, bij, s0);
        s0 = fma(k.b1, bjk, s0);
        s0 = fma(k.b2, bik, s0);
        s0 = fma(k.c0, xm, s0);
        s0 = fma(k.c1, ym, s0);
        s0 = fma(k.c2, zm, s0);
        T ss = fma(s0, k.a3, -c);
        if (masked) ss *= k.bn;
        return ss;
    }
}

template <typename T, typename C>
__global__ void __launch_bounds__(kThreads, 1) k_resident(const __grid_constant__ ResArgs a)
{
    using PC = PointCoef<T, C>;
    constexpr int TV = 16 / (int)sizeof(T);            // elements of a 16-byte vector
    extern __shared__ __align__(16) unsigned char res_smem[];
    __shared__ volatile int s_abort;
    __shared__ int s_masked;
    __shared__ double s_part[kWarps];
    __shared__ int s_last;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, b = blockIdx.x;
    const int nj = a.nj, nk = a.nk, tj = b % nj, tk = b / nj;
    const int j0 = 1 + part_begin(a.J - 2, nj, tj), bj = 1 + part_begin(a.J - 2, nj, tj + 1) - j0;
    const int k0 = 1 + part_begin(a.K - 2, nk, tk), bk = 1 + part_begin(a.K - 2, nk, tk + 1) - k0;
    const int I = a.I, bi = I - 2, W = a.ws, Z = W * (bj + 2);
    const int rows = bj * bk, units = rows * bi;
    const size_t plane = (size_t)a.J * a.pitch;

    uint4 *coefs = reinterpret_cast<uint4 *>(res_smem);
    int2 *rowtab = reinterpret_cast<int2 *>(res_smem + (size_t)PC::VEC * 16 * a.ucap);
    const int sbytes = a.ws * (a.bjm + 2) * (a.bkm + 2);             // elements of one state copy
    T *st0 = reinterpret_cast<T *>(res_smem + (size_t)PC::VEC * 16 * a.ucap + ((size_t)a.rcap * 8 + 15) / 16 * 16);
    T *st1 = st0 + sbytes;

    if (tid == 0) {
        s_abort = 0;
        s_masked = 0;
        __stcg(a.flags + (size_t)b * kFlagStride, 0u);
        __threadfence();
        atomicAdd(&a.hdr->gbar, 1u);                   // every flag is zero once all G arrived
    }
    // The box's rows, those next to another box (or face) first.
    const int edge_rows = (bk <= 2 || bj <= 2) ? rows : 2 * bj + 2 * (bk - 2);
    for (int r = tid; r < rows; r += kThreads) {
        int jj, kk;
        if (edge_rows == rows) { kk = r / bj; jj = r - kk * bj; }
        else if (r < 2 * bj) { kk = r < bj ? 0 : bk - 1; jj = r < bj ? r : r - bj; }
        else if (r < edge_rows) { kk = 1 + (r - 2 * bj) / 2; jj = (r & 1) ? bj - 1 : 0; }
        else { kk = 1 + (r - edge_rows) / (bj - 2); jj = 1 + (r - edge_rows) % (bj - 2); }
        // .x: the row in a shared-memory state, .y: in a state buffer
        rowtab[r] = make_int2(((kk + 1) * (bj + 2) + jj + 1) * W, ((k0 + kk) * a.J + j0 + jj) * a.pitch);
    }
    // State 0 with its halo, into both copies (faces never change).
    {
        const T *src = static_cast<const T *>(a.p_buf[0]);
        const int vpr = W / TV, n = (bj + 2) * (bk + 2) * vpr;
        for (int x = tid; x < n; x += kThreads) {
            const int row = x / vpr, col = x - row * vpr;
            const int kk = row / (bj + 2), jj = row - kk * (bj + 2);
            const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(src + (size_t)(k0 - 1 + kk) * plane +
                                                                   (size_t)(j0 - 1 + jj) * a.pitch) + col);
            reinterpret_cast<uint4 *>(st0)[x] = v;
            reinterpret_cast<uint4 *>(st1)[x] = v;
        }
    }
    __syncthreads();
    for (int u = tid; u < units; u += kThreads) {
        const int r = u / bi;
        const size_t off = (size_t)rowtab[r].y + 1 + (u - r * bi);
        PC::put(coefs + u, a.ucap, a.coef, off);
        if constexpr (sizeof(T) == 8)
            if (__ldg(static_cast<const double *>(a.coef[JAC_BND - 1]) + off) != 1.0) s_masked = 1;
    }
    __syncthreads();
    const bool masked = s_masked != 0;

    const T omega = (T)a.omega;
    const bool compute = warp < kComputeWarps;
    // Points u0 .. u1-1 of the box: ss from `old`, the new value into `nxt`
    // and, if `out` is not NULL, into the state buffer; with `res` nxt takes
    // ss instead.
    auto update = [&](int u0, int u1, const T *old, T *nxt, T *out, bool res) {
        int r = (u0 + tid) / bi, i = (u0 + tid) - r * bi;
        const int dr = kCompute / bi, di = kCompute - dr * bi;
#pragma unroll 2
        for (int u = u0 + tid; u < u1; u += kCompute) {
            const int2 row = rowtab[r];
            PC k;
            k.get(coefs + u, a.ucap);
            const T *P = old + row.x + 1 + i;
            const T ss = res_ss<T, C>(P, W, Z, k, masked);
            const T v = fma(omega, ss, P[0]);
            nxt[row.x + 1 + i] = res ? ss : v;
            if (out) out[(size_t)row.y + 1 + i] = v;
            r += dr;
            i += di;
            if (i >= bi) { i -= bi; ++r; }
        }
    };

    // This communication warp's neighbour: the box at (tj + dj, tk + dk) and
    // its part of the halo, rows (hj .., hk ..) of the shared state.
    const int d = compute ? 4 : (warp - kComputeWarps) + (warp - kComputeWarps >= 4 ? 1 : 0);
    const int dj = d % 3 - 1, dk = d / 3 - 1;
    const bool has_nb = !compute && tj + dj >= 0 && tj + dj < nj && tk + dk >= 0 && tk + dk < nk;
    const unsigned *nb_flag = a.flags + (size_t)(b + dj + dk * nj) * kFlagStride;
    const int hj = dj < 0 ? 0 : (dj == 0 ? 1 : bj + 1), hk = dk < 0 ? 0 : (dk == 0 ? 1 : bk + 1);
    const int hnj = dj == 0 ? bj : 1, hnk = dk == 0 ? bk : 1;
    const bool publisher = warp == kComputeWarps;

    bool ok = true;
    for (int t = 0; t < a.n_iter; ++t) {
        const T *old = (t & 1) ? st1 : st0;
        T *nxt = (t & 1) ? st0 : st1;
        T *out = a.hist ? reinterpret_cast<T *>(a.hist + (size_t)t * a.hist_stride)
                        : static_cast<T *>(a.p_buf[(t + 1) & 1]);
        const bool last = t == a.n_iter - 1;
        if (last) {
            if (compute) update(0, units, old, nxt, out, a.res != nullptr);
            break;
        }
        if (compute) update(0, edge_rows * bi, old, nxt, out, false);
        __syncthreads();                               // the box's outer rows are stored
        if (compute) {
            update(edge_rows * bi, units, old, nxt, a.hist ? out : nullptr, false);
        } else {
            if (publisher && lane == 0) {
                // orders the box's stores (before the barrier) ahead of the flag
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.flags + (size_t)b * kFlagStride),
                             "r"((unsigned)(t + 1)) : "memory");
            }
            if (has_nb) {
                bool got = true;
                if (lane == 0) {
                    if (t == 0) got = wait_counter_bounded(&a.hdr->gbar, (unsigned)G + a.gbar_extra, a.wait_ns);
                    if (got && ld_acquire_gpu(nb_flag) < (unsigned)(t + 1)) {
                        const unsigned long long t0 = globaltimer_ns();
                        while (ld_acquire_gpu(nb_flag) < (unsigned)(t + 1))
                            if (globaltimer_ns() - t0 > a.wait_ns) { got = false; break; }
                    }
                    if (!got) s_abort = 1;
                }
                got = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
                __syncwarp();                          // the other lanes' loads follow lane 0's acquire
                if (got) {
                    const int vpr = W / TV, n = hnj * hnk * vpr;
                    const int drow = 32 / vpr, dcol = 32 - drow * vpr;
                    int row = lane / vpr, col = lane - row * vpr;
                    constexpr int D = 8;               // vectors in flight per lane
                    for (int x0 = lane; x0 < n; x0 += 32 * D) {
                        uint4 v[D];
                        int at[D];
#pragma unroll
                        for (int q = 0; q < D; ++q) {
                            if (x0 + 32 * q < n) {
                                const int kk = hk + (dk == 0 ? (dj == 0 ? 0 : row) : 0);
                                const int jj = hj + (dj == 0 ? row : 0);
                                at[q] = (kk * (bj + 2) + jj) * vpr + col;
                                v[q] = __ldcg(reinterpret_cast<const uint4 *>(out + (size_t)(k0 - 1 + kk) * plane +
                                                                              (size_t)(j0 - 1 + jj) * a.pitch) + col);
                            }
                            row += drow;
                            col += dcol;
                            if (col >= vpr) { col -= vpr; ++row; }
                        }
#pragma unroll
                        for (int q = 0; q < D; ++q)
                            if (x0 + 32 * q < n) reinterpret_cast<uint4 *>(nxt)[at[q]] = v[q];
                    }
                }
            }
        }
        __syncthreads();                               // the new state of the box and its halo
        if (s_abort) { ok = false; break; }            // the same for every thread: set before the barrier
    }
    if (!ok && tid == 0) atomicExch(&a.hdr->errword, (int)JAC_ETIMEOUT);

    // This CTA's residual partial, from the ss values of the last sweep: FP32
    // squares of the (at most four) points of an aligned vector are summed in
    // FP32, the rest in FP64, as in the streaming kernel.  The last CTA sums
    // the partials in a fixed order and leaves the header zero.
    __syncthreads();
    double acc = 0.0;
    if (ok && a.res != nullptr) {
        const T *ss = (a.n_iter & 1) ? st1 : st0;
        const int vpr = W / TV;
        for (int x = tid; x < rows * vpr; x += kThreads) {
            const int r = x / vpr, i = (x - r * vpr) * TV;
            const T *v = ss + rowtab[r].x + i;
            float sq = 0.0f;
#pragma unroll
            for (int e = 0; e < TV; ++e) {
                if (i + e < 1 || i + e > I - 2) continue;
                if constexpr (sizeof(T) == 4) sq = fmaf(v[e], v[e], sq);
                else acc = fma(v[e], v[e], acc);
            }
            if constexpr (sizeof(T) == 4) acc += (double)sq;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) s_part[warp] = acc;
    }
    __syncthreads();
    if (warp == 0) {
        const double sum = warp_sum(a.res != nullptr && lane < kWarps ? s_part[lane] : 0.0, 0.0);
        if (lane == 0) {
            __stcg(a.partials + b, sum);
            __threadfence();
            s_last = atomicAdd(&a.hdr->counter, 1u) == (unsigned)G - 1;
        }
    }
    __syncthreads();
    if (!s_last || warp != 0) return;
    __threadfence();
    if (a.res != nullptr) {
        const double sum = sum_partials(a.partials, G, lane);
        if (lane == 0) *a.res = workspace_failed(a.hdr) ? __longlong_as_double(0x7ff8000000000000ll) : sum;
    }
    if (lane == 0) {
        a.hdr->gbar = 0u;
        a.hdr->counter = 0u;
        __threadfence();
    }
}

jac_status res_fail(jac_status s, const std::string &m)
{
    set_thread_error(m);
    return s;
}

int vectors_per_point(jac_prec prec) { return prec == JAC_F64 ? 6 : (prec == JAC_F32 ? 3 : 2); }

size_t resident_smem(jac_prec prec, int units, int rows, int ws, int bj, int bk)
{
    const size_t state = (size_t)ws * (bj + 2) * (bk + 2) * (prec == JAC_F64 ? 8 : 4);
    return (size_t)vectors_per_point(prec) * 16 * units + ((size_t)rows * 8 + 15) / 16 * 16 + 2 * state;
}

template <typename T, typename C>
jac_status launch_resident(const ResArgs &a, unsigned nblocks, size_t smem, cudaStream_t st)
{
    static std::once_flag once;
    static cudaError_t err = cudaSuccess;
    std::call_once(once, [] {
        err = cudaFuncSetAttribute(k_resident<T, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget);
    });
    if (err != cudaSuccess) return res_fail(JAC_ECUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(err));
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(nblocks);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;       // neighbours wait on one another: all CTAs resident
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_resident<T, C>, a);
    if (e != cudaSuccess) return res_fail(JAC_ECUDA, std::string("resident launch: ") + cudaGetErrorString(e));
    return JAC_OK;
}

}  // namespace

// The boxes of a grid over at most `sms` CTAs, and whether they fit in shared
// memory: of the splits of the J-2 x K-2 rows into nj x nk boxes the one whose
// largest box takes the least time by this model of a sweep, in ns: the rows
// next to other boxes at tu per point (128 points at a time: one per lane of
// a warp on each of the SM's four FP64 pipes), then the exchange, which the
// inner rows overlap, and the halo rows it collects.  tu and the exchange are
// measured on 33x33x65 FP64 and 77x53x101 FP32; BF16 takes FP32's.  The model
// orders the splits of one grid and leaves out how wide the halo rows are; what
// a sweep takes is estimated by resident_us in jac_sweep.cu.  Against the split with the fewest
// points in its largest box, which left 77x53x101 FP32 no inner rows (17 x 2
// instead of 9 x 4): 5.7 -> 4.8 us a sweep.
bool resident_shape(int I, int J, int K, jac_prec prec, int sms, ResidentShape *out)
{
    const int nji = J - 2, nki = K - 2, bi = I - 2;
    const int ws = (int)round_up((size_t)I, prec == JAC_F64 ? 2 : 4);
    const long long pts = (long long)nji * nki * bi;
    // more points than all shared memory holds, or more than 32-bit offsets
    if (pts * vectors_per_point(prec) * 16 > (long long)sms * (long long)kSmemBudget) return false;
    if ((long long)jac_pitch(I) * J * K > 0x7fffffffLL) return false;
    const double tu = prec == JAC_F64 ? 5.7 : 0.47, exchange = 3000.0;
    auto time_of = [&](long long rows) { return tu * (double)((rows * bi + 127) / 128 * 128); };
    double best = -1.0;
    for (int nj = 1; nj <= std::min(nji, sms); ++nj) {
        const int nk = std::min(nki, sms / nj);
        const int bj = (nji + nj - 1) / nj, bk = (nki + nk - 1) / nk;
        const long long rows = (long long)bj * bk;
        if (rows * bi > 65536) continue;               // far past any shared memory
        const long long edge = (bj <= 2 || bk <= 2) ? rows : 2LL * (bj + bk) - 4;
        const double cost = time_of(edge) + std::max(exchange, time_of(rows - edge)) + 2.0 * (2 * (bj + bk) + 4);
        if (best >= 0.0 && cost >= best) continue;
        const size_t smem = resident_smem(prec, (int)(rows * bi), (int)rows, ws, bj, bk);
        if (smem > kSmemBudget) continue;
        best = cost;
        *out = ResidentShape{nj, nk, bj, bk, ws, smem};
    }
    return best >= 0.0;
}

size_t resident_workspace_bytes(const ResidentShape &s)
{
    const size_t ctas = (size_t)s.nj * s.nk;
    return kWsHeaderBytes + round_up(ctas * sizeof(double), 256) + ctas * kFlagStride * sizeof(unsigned);
}

jac_status resident_run(const jac_grid *g, const ResidentShape &s, int n_iter, double *d_residual, void *workspace,
                        cudaStream_t st, void *hist, size_t hist_stride, const LaunchOpts *opts)
{
    const unsigned ctas = (unsigned)(s.nj * s.nk);
    ResArgs a;
    std::memset(&a, 0, sizeof(a));
    for (int q = JAC_A0; q <= JAC_BND; ++q) a.coef[q - 1] = g->coef[q];
    a.p_buf[0] = g->p[0];
    a.p_buf[1] = g->p[1];
    a.I = g->I; a.J = g->J; a.K = g->K;
    a.pitch = jac_pitch(g->I);
    a.nj = s.nj; a.nk = s.nk;
    a.bjm = s.bj; a.bkm = s.bk;
    a.rcap = s.bj * s.bk;
    a.ucap = a.rcap * (g->I - 2);
    a.ws = s.ws;
    a.n_iter = n_iter;
    a.omega = g->omega;
    char *w = static_cast<char *>(workspace);
    a.hdr = reinterpret_cast<WsHeader *>(w);
    a.partials = reinterpret_cast<double *>(w + kWsHeaderBytes);
    a.flags = reinterpret_cast<unsigned *>(w + kWsHeaderBytes + round_up(ctas * sizeof(double), 256));
    a.res = d_residual;
    a.hist = static_cast<char *>(hist);
    a.hist_stride = hist_stride;
    a.wait_ns = opts && opts->wait_ns ? opts->wait_ns : kWaitLimitNs;
    a.gbar_extra = opts ? opts->gbar_extra : 0;
    switch (g->prec) {
    case JAC_F64: return launch_resident<double, double>(a, ctas, s.smem, st);
    case JAC_F32: return launch_resident<float, float>(a, ctas, s.smem, st);
    default: return launch_resident<float, __nv_bfloat16>(a, ctas, s.smem, st);
    }
}

}  // namespace jac
