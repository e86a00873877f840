// Conversions between dense arrays (i fastest) and the storage layout
// (pitched rows, each array in its own element type): the device side of the
// hoisted copy-in and copy-out (Sections 3.2-3.3 of the paper).
//
// Bound by memory: 8 (FP64 source) plus 2, 4 or 8 bytes per point and array.
//   * One launch packs every array of a copy-in and writes p to both state
//     buffers (blockIdx.y is the array).  On a batch's grid of a few thousand
//     points, fourteen launches of 3 us each were what a copy-in cost.
//   * A block takes whole rows, about kBatch elements of storage at a time,
//     its threads running along them, so that every lane has an element
//     whatever the row length, and kPer loads of a thread are in flight.  The
//     row of an element is one multiply (no 64-bit division).
//   * FP64 <-> FP32 conversions are integer arithmetic: the conversion
//     instructions run on GB300's FP64 pipe (2 per SM and clock), which alone
//     takes longer than the memory traffic.
// Copy-in and copy-out of a grid, against thirteen launches with a 64-bit
// division and a hardware conversion per element, plus a copy of p:
// 513x513x1025 FP32 9.46 -> 7.27 ms (6.0 TB/s) and 0.70 -> 0.52 ms;
// 129x129x257 FP32 211 -> 105 us and 10.9 -> 8.5 us; 257x257x513 with BF16
// coefficients 1218 -> 866 us; the 512 grids of a batch 22.3 -> 5.4 ms.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "jac_common.cuh"
#include "jac_internal.h"

namespace jac {

namespace {

// FP64 -> FP32 -> BF16, each RNE; FP32 numbers keep their value in FP32 and
// FP64 storage, so both sources give the same storage values.
template <typename C, typename S>
__device__ __forceinline__ C to_storage(S x)
{
    if constexpr (sizeof(C) == sizeof(S)) return x;
    else if constexpr (sizeof(C) == 8) return widen(x);
    else {
        float f;
        if constexpr (sizeof(S) == 8) f = narrow(x);
        else f = x;
        if constexpr (sizeof(C) == 2) return __float2bfloat16_rn(f);
        else return f;
    }
}

// Storage value to dense value of type D.
template <typename D, typename C>
__device__ __forceinline__ D from_storage(C x)
{
    if constexpr (sizeof(C) == 2) return from_storage<D>(__bfloat162float(x));
    else if constexpr (sizeof(C) == sizeof(D)) return x;
    else if constexpr (sizeof(D) == 8) return widen(x);
    else return narrow(x);
}

constexpr int kThreads = 256, kPer = 8, kBatch = kThreads * kPer;

// Rows of `len` elements that a block takes at a time: about kBatch elements.
int rows_at_once(int len) { return std::max(1, kBatch / len); }

// l / len for 0 <= l < max(kBatch, len) and len >= 3: the high word of
// l * ceil(2^32 / len) is exact where l * len < 2^32, and for a longer row
// every l < len gives 0.
struct RowDiv {
    unsigned magic;
    int len;
    __device__ __forceinline__ int operator()(int l) const { return l < len ? 0 : (int)__umulhi((unsigned)l, magic); }
};
RowDiv row_div(int len) { return RowDiv{(unsigned)((0x100000000ull + len - 1) / len), len}; }

template <typename S>
struct PackArgs {
    const S *src[JAC_NFIELDS];
    void *dst[JAC_NFIELDS];
    void *dst2;                          // second destination of array 0 (NULL: none)
    unsigned char elem[JAC_NFIELDS];     // bytes of a storage element
    int I, pitch;
    int rpb;                             // rows_at_once(pitch)
    RowDiv div;                          // by pitch
    size_t rows;                         // J * K
};

template <typename S, typename C>
__device__ __forceinline__ void pack_rows(const PackArgs<S> &a, const S *src, C *dst, C *dst2)
{
    for (size_t row0 = (size_t)blockIdx.x * a.rpb; row0 < a.rows; row0 += (size_t)gridDim.x * a.rpb) {
        const int n = (int)(a.rows - row0 < (size_t)a.rpb ? a.rows - row0 : (size_t)a.rpb) * a.pitch;
        const S *s = src + row0 * a.I;
        const size_t off = row0 * a.pitch;
        for (int l0 = threadIdx.x; l0 < n; l0 += kBatch) {
            S v[kPer];
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int l = l0 + u * kThreads, r = a.div(l), i = l - r * a.pitch;
                v[u] = (l < n && i < a.I) ? __ldcs(s + (size_t)r * a.I + i) : S(0);
            }
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int l = l0 + u * kThreads;
                if (l < n) {
                    const C c = to_storage<C>(v[u]);
                    dst[off + l] = c;
                    if (dst2) dst2[off + l] = c;
                }
            }
        }
    }
}

template <typename S>
__global__ void __launch_bounds__(kThreads) k_pack(const __grid_constant__ PackArgs<S> a)
{
    const int f = blockIdx.y;
    void *d2 = f == 0 ? a.dst2 : nullptr;
    switch (a.elem[f]) {
    case 8: pack_rows(a, a.src[f], static_cast<double *>(a.dst[f]), static_cast<double *>(d2)); break;
    case 4: pack_rows(a, a.src[f], static_cast<float *>(a.dst[f]), static_cast<float *>(d2)); break;
    default: pack_rows(a, a.src[f], static_cast<__nv_bfloat16 *>(a.dst[f]), static_cast<__nv_bfloat16 *>(d2));
    }
}

// Storage layout to dense values of type D (FP32 from FP64 storage: RNE);
// rpb and div are of the dense row length I.
template <typename C, typename D>
__global__ void __launch_bounds__(kThreads)
k_unpack(const C *__restrict__ src, D *__restrict__ dst, int I, int pitch, int rpb, RowDiv div, size_t rows)
{
    for (size_t row0 = (size_t)blockIdx.x * rpb; row0 < rows; row0 += (size_t)gridDim.x * rpb) {
        const int n = (int)(rows - row0 < (size_t)rpb ? rows - row0 : (size_t)rpb) * I;
        const C *s = src + row0 * pitch;
        D *d = dst + row0 * I;
        for (int l0 = threadIdx.x; l0 < n; l0 += kBatch) {
            C v[kPer];
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int l = l0 + u * kThreads, r = div(l);
                if (l < n) v[u] = s[(size_t)r * pitch + (l - r * I)];
            }
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int l = l0 + u * kThreads;
                if (l < n) d[l] = from_storage<D>(v[u]);
            }
        }
    }
}

jac_status pack_fail(jac_status s, const std::string &m)
{
    set_thread_error(m);
    return s;
}

jac_status launched(const char *what)
{
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? JAC_OK : pack_fail(JAC_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Blocks for `rows` rows, rpb at a time: no more than several full waves.
unsigned row_blocks(size_t rows, int rpb)
{
    return (unsigned)std::min<size_t>((rows + rpb - 1) / rpb, (size_t)device_sm_count() * 64);
}

bool bad_dims(int I, int J, int K) { return I < 3 || J < 3 || K < 3; }

template <typename S>
jac_status pack_impl(int I, int J, int K, jac_prec prec, int first, int n, const S *const *src, void *const *dst,
                     void *dst2, cudaStream_t st)
{
    if (bad_dims(I, J, K) || first < 0 || first + n > JAC_NFIELDS) return pack_fail(JAC_EINVAL, "bad pack arguments");
    PackArgs<S> a;
    for (int q = 0; q < n; ++q) {
        if (!src[q] || !dst[q]) return pack_fail(JAC_EINVAL, "bad pack arguments");
        a.src[q] = src[q];
        a.dst[q] = dst[q];
        a.elem[q] = (unsigned char)elem_bytes(prec, first + q);
    }
    a.dst2 = dst2;
    a.I = I;
    a.pitch = jac_pitch(I);
    a.rpb = rows_at_once(a.pitch);
    a.div = row_div(a.pitch);
    a.rows = (size_t)J * K;
    k_pack<S><<<dim3(row_blocks(a.rows, a.rpb), (unsigned)n), kThreads, 0, st>>>(a);
    return launched("pack launch");
}

template <typename D>
jac_status unpack_impl(int I, int J, int K, jac_prec prec, int which, const void *src, D *dst, cudaStream_t st)
{
    if (bad_dims(I, J, K) || which < 0 || which >= JAC_NFIELDS || !src || !dst)
        return pack_fail(JAC_EINVAL, "bad unpack arguments");
    const int pitch = jac_pitch(I), rpb = rows_at_once(I);
    const size_t rows = (size_t)J * K;
    const unsigned blocks = row_blocks(rows, rpb);
    const RowDiv div = row_div(I);
    switch (elem_bytes(prec, which)) {
    case 8: k_unpack<<<blocks, kThreads, 0, st>>>(static_cast<const double *>(src), dst, I, pitch, rpb, div, rows); break;
    case 4: k_unpack<<<blocks, kThreads, 0, st>>>(static_cast<const float *>(src), dst, I, pitch, rpb, div, rows); break;
    default: k_unpack<<<blocks, kThreads, 0, st>>>(static_cast<const __nv_bfloat16 *>(src), dst, I, pitch, rpb, div, rows);
    }
    return launched("unpack launch");
}

}  // namespace

jac_status pack_dev(int I, int J, int K, jac_prec prec, int which, const double *src, void *dst, cudaStream_t st,
                    void *dst2)
{
    if (which < 0 || which >= JAC_NFIELDS) return pack_fail(JAC_EINVAL, "bad pack arguments");
    return pack_impl<double>(I, J, K, prec, which, 1, &src, &dst, dst2, st);
}

jac_status pack_fields(int I, int J, int K, jac_prec prec, const double *const *src, void *const *dst, void *p2,
                       cudaStream_t st)
{
    return pack_impl<double>(I, J, K, prec, 0, JAC_NFIELDS, src, dst, p2, st);
}

jac_status pack_fields_f32(int I, int J, int K, jac_prec prec, const float *const *src, void *const *dst, void *p2,
                           cudaStream_t st)
{
    return pack_impl<float>(I, J, K, prec, 0, JAC_NFIELDS, src, dst, p2, st);
}

jac_status unpack_dev(int I, int J, int K, jac_prec prec, int which, const void *src, double *dst, cudaStream_t st)
{
    return unpack_impl<double>(I, J, K, prec, which, src, dst, st);
}

jac_status unpack_dev_f32(int I, int J, int K, jac_prec prec, int which, const void *src, float *dst, cudaStream_t st)
{
    return unpack_impl<float>(I, J, K, prec, which, src, dst, st);
}

}  // namespace jac

extern "C" {

jac_status jac_pack_dev(int I, int J, int K, jac_prec prec, int which, const double *d_src, void *d_dst, void *stream)
{
    return jac::pack_dev(I, J, K, prec, which, d_src, d_dst, static_cast<cudaStream_t>(stream));
}

jac_status jac_unpack_dev(int I, int J, int K, jac_prec prec, int which, const void *d_src, double *d_dst,
                          void *stream)
{
    return jac::unpack_dev(I, J, K, prec, which, d_src, d_dst, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
