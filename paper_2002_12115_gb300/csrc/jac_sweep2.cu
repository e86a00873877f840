// Two fused sweeps per pass (temporal blocking by two) for FP32 storage.
//
// A pass reads the state p_t and writes p_{t+2}; the intermediate state
// p_{t+1} of a tile lives only in shared memory.  Every coefficient plane is
// then read from memory once for two point-updates.  Each update is the
// same arithmetic as the single-sweep kernel (ss_f32_ec; a3 S - 1, which
// depends only on the coefficients, is formed by sweep 1 and carried in
// registers to sweep 2 at the same point), so a pass gives bitwise the state
// of two single sweeps.
//
// Kernel design (persistent, warp-specialised, one CTA per SM, all passes of
// a call in one cooperative launch):
//   * an item is a tile of the 128 columns i0 .. i0+127 (i0 a multiple of
//     128) x R2 = 8 rows in (i, j) of output points over `kdepth` output
//     planes kb .. ke-1.  Sweep 1 runs over the tile's columns, the
//     R1 = R2 + 2 rows j0-1 .. j0+R2 and the planes kb-1 .. ke; sweep 2 over
//     the R2 inner rows and planes kb .. ke-1.  Tiles do not overlap: sweep 2
//     at columns i0 and i0+127 needs sweep 1 at columns i0-1 and i0+128 too;
//   * items are numbered along i, then j, then k, and CTA b takes items b,
//     b + G, ... of every pass (a fixed assignment also keeps the order of the
//     residual's sum).  A tile shares two columns (whole sectors, in twelve
//     arrays) and two rows with its neighbours along i and j: 1.32 times the
//     bytes where each reads them from DRAM.  They are in L2 when the tiles
//     are worked on at the same time, so the producers keep in step by a clock:
//     the sum of all CTAs' planes / 4.  None starts a plane more than 8 planes
//     ahead of the average (it waits 20 us at most, then goes on); the CTA
//     furthest behind never waits.  Batched, the grids' items differ in size:
//     they are taken by ticket, whichever CTA is free, without the clock;
//   * the queue entry of a CTA's next item carries its pass.
//     Before the state of pass t the producer waits until every item of the
//     passes before is stored (a counter; each sweep-2 warp adds one per item);
//   * warp 10 (one lane) copies, in the order they are used, the planes of
//     p_t with a halo of 4 columns and 2 rows into a ring of 4 slots, and the
//     twelve coefficient tiles (128 x R1) of every sweep-1 plane into a ring
//     of 3 stages;
//   * warps 0 .. R1-1 compute sweep 1, one row each, into a ring of 4
//     intermediate planes.  A row that is an output row too keeps its twelve
//     coefficients and a3 S - 1 in tensor memory (13 values per point, three
//     planes; tcgen05.st/ld with each lane's own points), so that sweep 2
//     reads neither global memory nor a stage that would have to be kept;
//   * warps 12 .. 19 compute sweep 2, one row each, a plane behind the newest
//     intermediate plane.  A row's sweep-2 warp has the index of its sweep-1
//     warp modulo 4, since a warp reaches only its quarter of tensor memory;
//   * warp 11 (the edge warp, 20 lanes) computes sweep 1 at columns i0-1 and
//     i0+128 of the R1 rows, from the state ring and coefficients it loads
//     from global memory one plane ahead;
//   * both sweeps take the update in two parts (ss_axes, ss_rest), and sweep 1
//     forms the b brackets before it loads a coefficient, so that 96 registers
//     hold one part's coefficients and the state values still needed but for 12
//     bytes that ptxas spills (4 with MID, 64 without that order).  Spilled
//     registers go through an L1 of a few KB, behind the copies' traffic;
//   * two points share an instruction (f32x2) where both operands lie in
//     aligned register pairs: a3 S - 1 and the axis terms;
//   * every wait is bounded; on expiry the kernel sets the workspace error
//     word, drains its own copies, frees its tensor memory and returns;
//   * batched (BATCH): the items of many grids in one list, each grid with its
//     own descriptor in device memory; no residual (a batch ends with single
//     sweeps);
//   * a one-pass call may also store sweep 1's state at the points the
//     items own (MID, Sweep2Args::mid): the reverse pass recomputes two
//     checkpoint-segment states per launch that way;
//   * STALL: a test of the failure path, with its own wait limit and a barrier
//     between passes that no CTA reaches.
//
// What bounds it: latency and issue of 18 compute warps where the state stays in
// L2 (a step of a CTA, one plane of a tile, both sweeps, takes 1.34 us), and
// DRAM elsewhere: 513x513x1025 reads and writes 1.05 times the bytes a pass
// needs at 6.2 TB/s.  Kept against, on one GB300 (Gpt/s, FP32):
//                                             129x129x257   257x257x513   513x513x1025
//   both sweeps in one warp, coefficients of
//     sweep 2 read again from L2 (41% of all
//     L2 reads)                                                   141            145
//   ... kept in tensor memory                                     150            153
//   separate warps for the two sweeps                             164            143
//   ... and items by ticket                        161            171            150
//   barriers tested together, 12 B spilled, f32x2  189            172            158
//   i-neighbours first, all CTAs in step
//     (this kernel)                                192            216            208
// The order alone (by ticket) ran at 184 and 157, the clock alone at 174 and
// 160; the clock's lead of 1 to 8 ticks made 1% of difference.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>

#include "jac_internal.h"
#include "jac_sweep_kernel.cuh"

namespace jac {

struct Sweep2Shape {
    static constexpr int VI = 4, TI = 128, H = 4;
    static constexpr int R2 = 8, R1 = R2 + 2;                // output rows, sweep-1 rows (= consumer warps)
    static constexpr int PW = TI + 2 * H, PH = R1 + 2;       // state plane box
    static constexpr int P_BYTES = PW * PH * 4;              // 6528
    static constexpr int TILE = TI * R1 * 4;                 // one coefficient tile, 5120
    static constexpr int C_BYTES = 12 * TILE;                // one stage
    static constexpr int Q_BYTES = TI * R1 * 4;              // one intermediate plane
    static constexpr int RP = 4, RC = 3, RQ = 4;
    static constexpr size_t SMEM = (size_t)RP * P_BYTES + (size_t)RQ * Q_BYTES + (size_t)RC * C_BYTES + 128;
    static constexpr int TM_SLOT = 13 * VI;                  // tensor-memory columns of one row: 12 coefficients, a3 S - 1
    static constexpr int TM_SLOTS = 3;                       // planes m-2 .. m
    static constexpr int TM_COLS = 512;                      // allocated (a power of two)
    static constexpr int EDGE_WARP = R1 + 1;                 // sweep 1 at the two columns past the tile
    static constexpr int WARP2 = R1 + 2;                     // first of the R2 sweep-2 warps
    static constexpr int THREADS = 32 * (R1 + 2 + R2);
    static constexpr int NQ = 4;                             // item queue of a CTA
    static constexpr uint32_t END = 0xffffffffu;             // no further item
    static constexpr uint32_t TICK = 4;                      // planes of a tick of the clock
    static constexpr uint32_t LEAD = 2;                      // ticks a CTA may be ahead of the average
    static constexpr unsigned long long CLOCK_WAIT_NS = 20000;   // then it goes on all the same
    static_assert(P_BYTES % 128 == 0 && Q_BYTES % 128 == 0 && C_BYTES % 128 == 0, "slot alignment");
    static_assert(R2 / 4 * TM_SLOTS * TM_SLOT <= TM_COLS && WARP2 % 4 == 0 && R2 % 4 == 0, "tensor memory columns");
};

struct Sweep2Desc {
    CUtensorMap p[2];          // state buffers, box (PW, PH, 1)
    CUtensorMap coef[12];      // JAC_A0 .. JAC_BND (index q-1), box (TI, R1, 1)
    const float *coef_ptr[12]; // the same arrays, for the edge warp's loads
    void *p_buf[2];
    int I, J, K, pitch;
    int kdepth, nti, ntj, nkb, nitems;
};

struct Sweep2Args {
    const Sweep2Desc *descs;   // batched: one per grid
    const int *item_base;      // batched: first item of each grid (ascending)
    int ngrids, nitems;        // grids and items of a pass

    int n_pass, par;           // pass t reads p[(t + par) & 1], writes the other
    double omega;
    double *partials;          // gridDim.x
    double *res;               // residual of the last pass's second sweep (NULL: none)
    float *mid;                // one-pass calls: also store sweep 1's state here (NULL: no)
    WsHeader *hdr;
    int l2_keep_state;
    unsigned l2_keep_coef;
    unsigned long long wait_ns;   // STALL: limit of the waits on other warps and CTAs
    unsigned gbar_extra;       // STALL: added to the targets between passes, which makes them unreachable
};

struct Item2 {
    int ti, i0, j0, kb, nout;
};

__device__ __forceinline__ Item2 decode_item2(const Sweep2Desc &d, int item)
{
    using S = Sweep2Shape;
    Item2 it;
    it.ti = item % d.nti;
    const int r = item / d.nti;
    const int tj = r % d.ntj;
    const int kk = r / d.ntj;
    it.i0 = it.ti * S::TI;
    it.j0 = 1 + tj * S::R2;
    it.kb = 1 + kk * d.kdepth;
    it.nout = min(d.K - 1, it.kb + d.kdepth) - it.kb;
    return it;
}

// Batched: the grid of an item, the last one whose first item is not past it;
// `item` becomes its number within the grid.
__device__ __forceinline__ const Sweep2Desc *find_grid(const Sweep2Args &a, int &item)
{
    int lo = 0, hi = a.ngrids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&a.item_base[mid]) <= item) lo = mid;
        else hi = mid - 1;
    }
    item -= __ldg(&a.item_base[lo]);
    return a.descs + lo;
}

// VI values of an intermediate-plane row (no halo) with the left and right
// neighbours by lane shuffles; the edge lanes get `left` / `right`.
__device__ __forceinline__ void q_ext(const float *row, int lane, float left, float right, float (&e)[6])
{
    const float4 v = *reinterpret_cast<const float4 *>(row + 4 * lane);
    e[1] = v.x; e[2] = v.y; e[3] = v.z; e[4] = v.w;
    const float l = __shfl_up_sync(0xffffffffu, e[4], 1);
    const float r = __shfl_down_sync(0xffffffffu, e[1], 1);
    e[0] = (lane == 0) ? left : l;
    e[5] = (lane == 31) ? right : r;
}

// Tensor memory as a per-lane scratchpad: a warp reaches the 32 lanes of its
// quarter (warp index mod 4); lane l of the warp owns column values of lane l.
__device__ __forceinline__ void tmem_alloc(uint32_t *smem_addr, int cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_addr)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, int cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
// Four arrays of four values (one lane's) to or from 16 columns.
__device__ __forceinline__ void tmem_st16(uint32_t addr, const float (&a)[4], const float (&b)[4], const float (&c)[4],
                                          const float (&d)[4])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(addr),
        "f"(a[0]), "f"(a[1]), "f"(a[2]), "f"(a[3]), "f"(b[0]), "f"(b[1]), "f"(b[2]), "f"(b[3]), "f"(c[0]), "f"(c[1]),
        "f"(c[2]), "f"(c[3]), "f"(d[0]), "f"(d[1]), "f"(d[2]), "f"(d[3])
        : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t addr, const float (&a)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a[0]), "f"(a[1]),
                 "f"(a[2]), "f"(a[3])
                 : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&a)[4], float (&b)[4], float (&c)[4], float (&d)[4])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3]), "=f"(b[0]), "=f"(b[1]), "=f"(b[2]), "=f"(b[3]), "=f"(c[0]),
          "=f"(c[1]), "=f"(c[2]), "=f"(c[3]), "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(addr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t addr, float (&a)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3])
                 : "r"(addr)
                 : "memory");
}
// Order this warp's tensor-memory accesses before a barrier that it arrives
// at, and after one that it waited for.
__device__ __forceinline__ void tmem_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Ties loaded values to the wait before it: no use of them moves above it.
__device__ __forceinline__ void tmem_loaded(float (&a)[4])
{
    asm volatile("" : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3])::"memory");
}

// Two FP32 numbers in one register pair: one instruction for two points where
// both operands lie in aligned pairs.  Each half rounds like the single
// instruction, so the values are bitwise the same.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ void fast_two_sum_acc2(f32x2 &hi, f32x2 &lo, f32x2 b)
{
    const f32x2 s = add2(hi, b);
    lo = add2(lo, sub2(b, sub2(s, hi)));
    hi = s;
}

// a3s_minus_one<false> of four points.
__device__ __forceinline__ void a3s_minus_one4(const float (&a3)[4], const float (&a0)[4], const float (&a1)[4],
                                               const float (&a2)[4], const float (&c0)[4], const float (&c1)[4],
                                               const float (&c2)[4], float (&ec)[4])
{
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
        f32x2 hi = pack2(fmaxf(a0[e], c0[e]), fmaxf(a0[e + 1], c0[e + 1])), lo = pack2(0.0f, 0.0f);
        fast_two_sum_acc2(hi, lo, pack2(fminf(a0[e], c0[e]), fminf(a0[e + 1], c0[e + 1])));
        fast_two_sum_acc2(hi, lo, pack2(a1[e], a1[e + 1]));
        fast_two_sum_acc2(hi, lo, pack2(c1[e], c1[e + 1]));
        fast_two_sum_acc2(hi, lo, pack2(a2[e], a2[e + 1]));
        fast_two_sum_acc2(hi, lo, pack2(c2[e], c2[e + 1]));
        const f32x2 s = pack2(a3[e], a3[e + 1]);
        unpack2(fma2(s, lo, fma2(s, hi, pack2(-1.0f, -1.0f))), ec[e], ec[e + 1]);
    }
}

// ss_axes of four points; x, yp, ym, zp, zm with one value past each end.  The
// differences along i, whose operands are shifted by one point, are formed
// singly, into aligned pairs.
__device__ __forceinline__ void ss_axes4(const float (&x)[6], const float (&yp)[6], const float (&ym)[6],
                                         const float (&zp)[6], const float (&zm)[6], const float (&a0)[4],
                                         const float (&a1)[4], const float (&a2)[4], const float (&c0)[4],
                                         const float (&c1)[4], const float (&c2)[4], const float (&wk)[4],
                                         float (&d)[4])
{
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
        const f32x2 c = pack2(x[e + 1], x[e + 2]);
        f32x2 s = pack2(wk[e], wk[e + 1]);
        s = fma2(pack2(a0[e], a0[e + 1]), pack2(x[e + 2] - x[e + 1], x[e + 3] - x[e + 2]), s);
        s = fma2(pack2(a1[e], a1[e + 1]), sub2(pack2(yp[e + 1], yp[e + 2]), c), s);
        s = fma2(pack2(a2[e], a2[e + 1]), sub2(pack2(zp[e + 1], zp[e + 2]), c), s);
        s = fma2(pack2(c0[e], c0[e + 1]), pack2(x[e] - x[e + 1], x[e + 1] - x[e + 2]), s);
        s = fma2(pack2(c1[e], c1[e + 1]), sub2(pack2(ym[e + 1], ym[e + 2]), c), s);
        s = fma2(pack2(c2[e], c2[e + 1]), sub2(pack2(zm[e + 1], zm[e + 2]), c), s);
        unpack2(s, d[e], d[e + 1]);
    }
}

template <bool BATCH, bool MID, bool STALL>
__global__ void __launch_bounds__(Sweep2Shape::THREADS, 1)
k_sweep2(const __grid_constant__ Sweep2Desc d, const Sweep2Args a)
{
    using S = Sweep2Shape;
    constexpr int VI = S::VI, TI = S::TI, H = S::H, R1 = S::R1, RP = S::RP, RC = S::RC, RQ = S::RQ;
    extern __shared__ unsigned char dsm2_raw[];
    unsigned char *base =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(dsm2_raw) + 127) & ~uintptr_t(127));
    unsigned char *ring_q = base + (size_t)RP * S::P_BYTES;
    unsigned char *ring_c = ring_q + (size_t)RQ * S::Q_BYTES;
    __shared__ __align__(8) uint64_t p_full[RP], p_empty[RP], c_full[RC], c_empty[RC], q_full[RQ], q_empty[RQ],
        i_full[S::NQ], i_empty[S::NQ], cons_bar;
    __shared__ uint32_t s_item[S::NQ];
    __shared__ volatile int s_abort;
    __shared__ uint32_t s_tmem;
    __shared__ double s_part[S::R2];
    __shared__ float q_edge[RQ][R1][2];   // sweep-1 values at columns i0-1 and i0+128, per row

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int G = gridDim.x;
    // A test of the failure path has a kernel of its own: arguments in place of
    // these constants cost 3% of 513x513x1025 (1277 -> 1317 us a sweep).
    const unsigned long long limit = STALL ? a.wait_ns : kWaitLimitNs;
    const unsigned extra = STALL ? a.gbar_extra : 0u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < RP; ++s) { mbar_init(&p_full[s], 1); mbar_init(&p_empty[s], R1 + 1); }
        for (int s = 0; s < RC; ++s) { mbar_init(&c_full[s], 1); mbar_init(&c_empty[s], R1); }
        for (int s = 0; s < RQ; ++s) { mbar_init(&q_full[s], R1 + 1); mbar_init(&q_empty[s], S::R2); }
        for (int s = 0; s < S::NQ; ++s) { mbar_init(&i_full[s], 1); mbar_init(&i_empty[s], R1 + 1 + S::R2); }
        mbar_init(&cons_bar, S::R2);
        s_abort = 0;
        fence_mbar_init();
    }
    if (warp == S::EDGE_WARP) tmem_alloc(&s_tmem, S::TM_COLS);
    __syncthreads();

    // The next entry of the CTA's item queue (every warp but the producer's
    // reads each entry): pass * nitems + item, or END; false: give up.
    uint32_t ic = 0;
    auto next_item = [&](uint32_t &entry) -> bool {
        bool r = mbar_wait_bounded(&i_full[ic % S::NQ], (ic / S::NQ) & 1, limit);
        r = __all_sync(0xffffffffu, r && !s_abort);
        entry = s_item[ic % S::NQ];
        __syncwarp();
        if (lane == 0) mbar_arrive(&i_empty[ic % S::NQ]);
        ++ic;
        return r;
    };
    const uint32_t nitems = (uint32_t)(BATCH ? a.nitems : d.nitems);

    if (warp == R1) {
        // ------------------------------------------------------------ producer
        // One lane copies, per item, the coefficient stage of each sweep-1
        // plane (twelve 128 x R1 tiles) and the state planes of p_t with a
        // halo of 4 columns and 2 rows, in the order the consumers use them:
        // state planes 0 and 1, then per step s state plane s+2 and stage
        // s+1.  Before the state of pass t >= 1 it waits until the passes
        // before are stored (the first stage of an item does not need it).
        if (lane == 0) {
            // Coefficients make way for a state that stays in L2, but not
            // before a neighbour along i has read the columns it shares
            // (129x129x257, one tile: 22.6 -> 21.6 us a sweep; 250x129x257,
            // two: 44.6 -> 54.0 if they did).
            const uint64_t pol_c = l2_policy(a.l2_keep_state && (BATCH || d.nti == 1) ? -1 : 0);
            const uint64_t pol_keep = l2_policy(1);
            const uint64_t pol_p = l2_policy(a.l2_keep_state ? 1 : 0);
            uint32_t pc = 0, cc = 0;
            bool ok = true;
            const CUtensorMap *pm = nullptr, *cm = d.coef;
            auto put_state = [&](const Item2 &it, int q) -> bool {
                const uint32_t slot = pc % RP, use = pc / RP;
                if (use > 0 && !mbar_wait_bounded(&p_empty[slot], (use - 1) & 1, limit)) return false;
                if (s_abort) return false;
                mbar_arrive_expect_tx(&p_full[slot], (uint32_t)S::P_BYTES);
                tma_load_3d_hint(base + (size_t)slot * S::P_BYTES, pm, &p_full[slot], it.i0 - H, it.j0 - 2,
                                 it.kb - 2 + q, pol_p);
                ++pc;
                return true;
            };
            auto put_coef = [&](const Item2 &it, int q) -> bool {
                const uint32_t slot = cc % RC, use = cc / RC;
                if (use > 0 && !mbar_wait_bounded(&c_empty[slot], (use - 1) & 1, limit)) return false;
                if (s_abort) return false;
                unsigned char *st = ring_c + (size_t)slot * S::C_BYTES;
                mbar_arrive_expect_tx(&c_full[slot], (uint32_t)S::C_BYTES);
                for (int k = JAC_A0; k <= JAC_BND; ++k)
                    tma_load_3d_hint(st + (size_t)(k - 1) * S::TILE, (BATCH ? cm : d.coef) + (k - 1), &c_full[slot], it.i0,
                                     it.j0 - 1, it.kb - 1 + q, ((a.l2_keep_coef >> k) & 1u) ? pol_keep : pol_c);
                ++cc;
                return true;
            };
            // Items by CTA number in every pass (batched: in the order of
            // their numbers, whichever CTA is free, by ticket).  The clock
            // counts the ticks of all CTAs; one that takes part in fewer
            // items or planes than others adds the rest when it is done.
            uint32_t ip = 0, entry = blockIdx.x, pass = 0;
            const uint32_t total = (uint32_t)a.n_pass * nitems;
            const uint32_t ticks = BATCH ? 0 : ((uint32_t)d.kdepth + 2 + S::TICK - 1) / S::TICK;   // of an item
            const uint32_t rounds = (nitems + (uint32_t)G - 1) / (uint32_t)G;   // items of a CTA in a pass
            uint32_t round = 0;
            [[maybe_unused]] uint32_t clock = 0;      // as last read
            while (ok) {
                const uint32_t qslot = ip % S::NQ;
                if (ip >= S::NQ && !(ok = mbar_wait_bounded(&i_empty[qslot], ((ip / S::NQ) - 1) & 1, limit))) break;
                s_item[qslot] = entry;
                mbar_arrive(&i_full[qslot]);
                ++ip;
                if (entry == S::END) break;
                [[maybe_unused]] uint32_t ticket = 0;
                if constexpr (BATCH) ticket = (uint32_t)G + atomicAdd(&a.hdr->ticket, 1u);   // used after this item
                const uint32_t t = entry / nitems;
                Item2 it;
                if constexpr (BATCH) {
                    int item = (int)(entry - t * nitems);
                    const Sweep2Desc *g = find_grid(a, item);
                    it = decode_item2(*g, item);
                    pm = &g->p[(t + a.par) & 1];
                    cm = g->coef;
                } else {
                    it = decode_item2(d, (int)(entry - t * nitems));
                    pm = ((t + a.par) & 1) ? &d.p[1] : &d.p[0];
                }
                if (!(ok = put_coef(it, 0))) break;
                if (t > pass) {            // every item of the passes before is stored
                    pass = t;
                    if (!(ok = wait_counter_bounded(&a.hdr->gbar, t * nitems * S::R2 + extra, limit))) break;
                    fence_proxy_async_global();
                }
                if (!(ok = put_state(it, 0) && put_state(it, 1))) break;
                for (int q = 0; q < it.nout + 2 && ok; ++q) {
                    if (!BATCH && q % S::TICK == 0) {
                        // not far ahead of the average: rows and columns that
                        // tiles share are then still in L2
                        atomicAdd(&a.hdr->clock, 1u);
                        const uint32_t mine = ((t * rounds + round) * ticks + q / S::TICK - S::LEAD) * (uint32_t)G;
                        if ((int)(mine - clock) > 0) {
                            const unsigned long long t0 = globaltimer_ns();
                            do {
                                clock = ld_relaxed_gpu(&a.hdr->clock);
                            } while ((int)(mine - clock) > 0 && globaltimer_ns() - t0 < S::CLOCK_WAIT_NS);
                        }
                    }
                    ok = put_state(it, q + 2);
                    if (ok && q + 1 < it.nout + 2) ok = put_coef(it, q + 1);
                }
                if constexpr (BATCH) {
                    entry = ticket < total ? ticket : S::END;
                } else {
                    uint32_t rest = ticks - ((uint32_t)it.nout + 2 + S::TICK - 1) / S::TICK;
                    ++round;
                    if (entry - t * nitems + (uint32_t)G < nitems) {
                        entry += (uint32_t)G;
                    } else {
                        rest += (rounds - round) * ticks;
                        round = 0;
                        entry = t + 1 < (uint32_t)a.n_pass ? (t + 1) * nitems + blockIdx.x : S::END;
                    }
                    if (rest > 0) atomicAdd(&a.hdr->clock, rest);
                }
            }
            if (!ok) {
                s_abort = 1;
                atomicExch(&a.hdr->errword, (int)JAC_ETIMEOUT);
            }
            for (uint32_t s = 0; s < (uint32_t)RC && s < cc; ++s) {   // land every issued copy
                const uint32_t last = cc - 1 - ((cc - 1 - s) % RC);
                (void)mbar_wait_bounded(&c_full[s], (last / RC) & 1);
            }
            for (uint32_t s = 0; s < (uint32_t)RP && s < pc; ++s) {
                const uint32_t last = pc - 1 - ((pc - 1 - s) % RP);
                (void)mbar_wait_bounded(&p_full[s], (last / RP) & 1);
            }
        }
    } else if (warp == S::EDGE_WARP) {
        // ----------------------------------------------------------- edge warp
        // Lane 2r + e (r < R1) computes sweep 1 at row j0-1+r and column
        // i0-1 (e = 0) or i0+128 (e = 1), the neighbours that sweep 2 needs
        // past the tile's 128 columns, with the consumers' arithmetic.  Its
        // twelve coefficients come from global memory one plane ahead.
        const int r = lane >> 1, side = lane & 1;
        const bool act = lane < 2 * R1;
        const float omega = (float)a.omega;
        int I = d.I, J = d.J, K = d.K, pitch = d.pitch;
        [[maybe_unused]] const Sweep2Desc *g = nullptr;
        const int x = side ? H + TI : H - 1;             // the column in the state box
        const int r0 = r * S::PW, r1 = (r + 1) * S::PW, r2 = (r + 2) * S::PW;
        uint32_t pc = 0, qc = 0;
        bool ok = true;
        uint32_t entry;
        while ((ok = next_item(entry)) && entry != S::END) {
            Item2 it;
            if constexpr (BATCH) {
                int item = (int)(entry % nitems);
                g = find_grid(a, item);
                it = decode_item2(*g, item);
                I = g->I; J = g->J; K = g->K; pitch = g->pitch;
            } else {
                it = decode_item2(d, (int)(entry % nitems));
            }
            const int j = it.j0 - 1 + r;
            const int ie = side ? it.i0 + TI : it.i0 - 1;
            const bool col_in = act && (j >= 1) && (j <= J - 2) && (ie >= 1) && (ie <= I - 2);
            float cf[12], cn[12];
            auto load_coef = [&](int m, float (&v)[12]) {
                if (col_in && m >= 1 && m <= K - 2) {
                    const size_t off = ((size_t)m * J + (size_t)j) * (size_t)pitch + (size_t)ie;
#pragma unroll
                    for (int q = 0; q < 12; ++q) v[q] = __ldg((BATCH ? g->coef_ptr[q] : d.coef_ptr[q]) + off);
                } else {
#pragma unroll
                    for (int q = 0; q < 12; ++q) v[q] = 0.0f;
                }
            };
            load_coef(it.kb - 1, cf);
            for (int s = 0; s < it.nout + 2; ++s) {
                const int m = it.kb - 1 + s;
                const bool gone = s_abort;
                if (s == 0) {
                    ok = mbar_wait_bounded(&p_full[pc % RP], (pc / RP) & 1, limit) &&
                         mbar_wait_bounded(&p_full[(pc + 1) % RP], ((pc + 1) / RP) & 1, limit);
                }
                const uint32_t q2 = pc + s + 2;
                ok = ok && mbar_wait_bounded(&p_full[q2 % RP], (q2 / RP) & 1, limit);
                const uint32_t qs = qc + s;
                if (qs >= RQ) ok = ok && mbar_wait_bounded(&q_empty[qs % RQ], ((qs / RQ) - 1) & 1, limit);
                ok = __all_sync(0xffffffffu, ok && !gone);
                if (!ok) break;
                if (s + 1 < it.nout + 2) load_coef(m + 1, cn);
                if (act) {
                    const float *Pm = reinterpret_cast<const float *>(base + (size_t)((pc + s) % RP) * S::P_BYTES);
                    const float *Pk =
                        reinterpret_cast<const float *>(base + (size_t)((pc + s + 1) % RP) * S::P_BYTES);
                    const float *Pp = reinterpret_cast<const float *>(base + (size_t)(q2 % RP) * S::P_BYTES);
                    const float c = Pk[r1 + x];
                    float out = c;
                    if (col_in && m >= 1 && m <= K - 2) {
                        const float bij = ((Pk[r2 + x + 1] - Pk[r0 + x + 1]) - Pk[r2 + x - 1]) + Pk[r0 + x - 1];
                        const float bjk = ((Pp[r2 + x] - Pm[r2 + x]) - Pp[r0 + x]) + Pm[r0 + x];
                        const float bik = ((Pp[r1 + x + 1] - Pm[r1 + x + 1]) - Pp[r1 + x - 1]) + Pm[r1 + x - 1];
                        const float ss = ss_f32<false>(c, Pk[r1 + x + 1], Pk[r1 + x - 1], Pk[r2 + x], Pk[r0 + x],
                                                       Pp[r1 + x], Pm[r1 + x], bij, bjk, bik, cf[0], cf[1], cf[2],
                                                       cf[3], cf[4], cf[5], cf[6], cf[7], cf[8], cf[9], cf[10],
                                                       cf[11]);
                        out = fmaf(omega, ss, c);
                    }
                    q_edge[qs % RQ][r][side] = out;
                }
#pragma unroll
                for (int q = 0; q < 12; ++q) cf[q] = cn[q];
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&q_full[qs % RQ]);            // the edge values of intermediate plane s
                    mbar_arrive(&p_empty[(pc + s) % RP]);     // state plane m-1 is done
                }
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&p_empty[(pc + it.nout + 2) % RP]);
                mbar_arrive(&p_empty[(pc + it.nout + 3) % RP]);
            }
            pc += it.nout + 4;
            qc += it.nout + 2;
        }
        if (!ok) {
            s_abort = 1;
            atomicExch(&a.hdr->errword, (int)JAC_ETIMEOUT);
        }
    } else if (warp < R1) {
        // ------------------------------------------------------- sweep-1 warps
        const int w = warp;                         // row j0-1+w of every item
        const float omega = (float)a.omega;
        const uint64_t st_pol = l2_policy(a.l2_keep_state ? 1 : 0);
        int I = d.I, J = d.J, K = d.K, pitch = d.pitch;
        [[maybe_unused]] const Sweep2Desc *g = nullptr;
        const bool do2 = (w >= 1) && (w <= R1 - 2);  // this warp's row is an output row too
        const uint32_t tm = s_tmem + ((uint32_t)(w & 3) << 21) + (uint32_t)(((w - 1) >> 2) * S::TM_SLOTS * S::TM_SLOT);
        uint32_t pc = 0, qc = 0;
        bool ok = true;
        uint32_t entry;
        while ((ok = next_item(entry)) && entry != S::END) {
            Item2 it;
            if constexpr (BATCH) {
                int item = (int)(entry % nitems);
                g = find_grid(a, item);
                it = decode_item2(*g, item);
                I = g->I; J = g->J; K = g->K; pitch = g->pitch;
            } else {
                it = decode_item2(d, (int)(entry % nitems));
            }
            const int j = it.j0 - 1 + w;
            const int ib = it.i0 + VI * lane;
            const bool row1_in = (j >= 1) && (j <= J - 2);
            bool in_i[VI], owned[VI];
            bool all_owned = true;
#pragma unroll
            for (int e = 0; e < VI; ++e) {
                in_i[e] = (ib + e >= 1) && (ib + e <= I - 2);
                owned[e] = do2 && row1_in && in_i[e];
                all_owned = all_owned && owned[e];
            }
            const int r0 = w * S::PW, r1 = (w + 1) * S::PW, r2 = (w + 2) * S::PW;   // rows j-1, j, j+1
            const int cidx = w * TI + VI * lane;

            for (int s = 0; s < it.nout + 2; ++s) {
                const int m = it.kb - 1 + s;                 // sweep-1 plane
                const uint32_t qs = qc + s;
                const bool gone = s_abort;
                if (s == 0) {
                    ok = mbar_wait_bounded(&p_full[pc % RP], (pc / RP) & 1, limit) &&
                         mbar_wait_bounded(&p_full[(pc + 1) % RP], ((pc + 1) / RP) & 1, limit);
                }
                const uint32_t q2 = pc + s + 2;
                // The newest state plane, the stage and a free intermediate
                // plane (whose phase before the first use counts as
                // complete), tested together: one latency when all are there.
                const bool got_p = mbar_try_wait(&p_full[q2 % RP], (q2 / RP) & 1);
                const bool got_c = mbar_try_wait(&c_full[qs % RC], (qs / RC) & 1);
                const bool got_q = mbar_try_wait(&q_empty[qs % RQ], ((qs / RQ) - 1) & 1);
                ok = ok && !gone;
                if (!__all_sync(0xffffffffu, ok && got_p && got_c && got_q)) {
                    ok = ok && mbar_wait_bounded(&p_full[q2 % RP], (q2 / RP) & 1, limit) &&
                         mbar_wait_bounded(&c_full[qs % RC], (qs / RC) & 1, limit) &&
                         mbar_wait_bounded(&q_empty[qs % RQ], ((qs / RQ) - 1) & 1, limit);
                    ok = __all_sync(0xffffffffu, ok);
                }
                if (!ok) break;
                if (do2) tmem_after_sync();                  // sweep 2 is done with the slot of plane s-3
                const float *Pm = reinterpret_cast<const float *>(base + (size_t)((pc + s) % RP) * S::P_BYTES);
                const float *Pk =
                    reinterpret_cast<const float *>(base + (size_t)((pc + s + 1) % RP) * S::P_BYTES);
                const float *Pp = reinterpret_cast<const float *>(base + (size_t)(q2 % RP) * S::P_BYTES);
                const unsigned char *cs = ring_c + (size_t)(qs % RC) * S::C_BYTES;
                float ek0[VI + 2], ek1[VI + 2], ek2[VI + 2], em1[VI + 2], ep1[VI + 2];
                float vm0[VI], vm2[VI], vp0[VI], vp2[VI];
                load_ext<float, VI, H>(Pk + r0, lane, 32, ek0);
                load_ext<float, VI, H>(Pk + r1, lane, 32, ek1);
                load_ext<float, VI, H>(Pk + r2, lane, 32, ek2);
                load_ext<float, VI, H>(Pm + r1, lane, 32, em1);
                load_ext<float, VI, H>(Pp + r1, lane, 32, ep1);
                lds_vec<float, VI>(Pm + r0 + H + VI * lane, vm0);
                lds_vec<float, VI>(Pm + r2 + H + VI * lane, vm2);
                lds_vec<float, VI>(Pp + r0 + H + VI * lane, vp0);
                lds_vec<float, VI>(Pp + r2 + H + VI * lane, vp2);
                const bool in1 = row1_in && (m >= 1) && (m <= K - 2);
                const uint32_t at = tm + (qs % S::TM_SLOTS) * S::TM_SLOT;
                auto coef = [&](int q, float (&v)[VI]) {
                    lds_vec<float, VI>(reinterpret_cast<const float *>(cs + (q - 1) * S::TILE) + cidx, v);
                };
                // The coefficients in the two parts of the update, so that
                // only one part's are held in registers at a time; an
                // output row keeps them for sweep 2 at this plane.
                float bij[VI], bjk[VI], bik[VI];
#pragma unroll
                for (int e = 0; e < VI; ++e) {
                    bij[e] = ((ek2[e + 2] - ek0[e + 2]) - ek2[e]) + ek0[e];
                    bjk[e] = ((vp2[e] - vm2[e]) - vp0[e]) + vm0[e];
                    bik[e] = ((ep1[e + 2] - em1[e + 2]) - ep1[e]) + em1[e];
                }
                // formed before the coefficients are loaded: 12 bytes are spilled instead of 64
                tmem_loaded(bij); tmem_loaded(bjk); tmem_loaded(bik);
                float dd[VI], ec[VI];
                {
                    float wk[VI], a0[VI], a1[VI], a2[VI], c0[VI], c1[VI], c2[VI];
                    coef(JAC_WRK1, wk); coef(JAC_A0, a0); coef(JAC_A1, a1); coef(JAC_A2, a2);
                    coef(JAC_C0, c0); coef(JAC_C1, c1); coef(JAC_C2, c2);
                    if (do2) {
                        tmem_st16(at, wk, a0, a1, a2);
                        tmem_st4(at + 16, c0);
                        tmem_st4(at + 20, c1);
                        tmem_st4(at + 24, c2);
                    }
                    float a3[VI];
                    coef(JAC_A3, a3);
                    ss_axes4(ek1, ek2, ek0, ep1, em1, a0, a1, a2, c0, c1, c2, wk, dd);
                    a3s_minus_one4(a3, a0, a1, a2, c0, c1, c2, ec);
                }
                float out[VI];
                {
                    float b0[VI], b1[VI], b2[VI], a3[VI], bn[VI];
                    coef(JAC_B0, b0); coef(JAC_B1, b1); coef(JAC_B2, b2); coef(JAC_A3, a3); coef(JAC_BND, bn);
                    if (do2) {
                        tmem_st4(at + 28, b0);
                        tmem_st4(at + 32, b1);
                        tmem_st16(at + 36, b2, a3, bn, ec);
                    }
#pragma unroll
                    for (int e = 0; e < VI; ++e) {
                        const float c = ek1[e + 1];
                        const float ss = ss_rest(dd[e], c, bij[e], bjk[e], bik[e], a3[e], b0[e], b1[e], b2[e],
                                                 bn[e], ec[e]);
                        out[e] = (in1 && in_i[e]) ? fmaf(omega, ss, c) : c;
                    }
                }
                float *qrow = reinterpret_cast<float *>(ring_q + (size_t)(qs % RQ) * S::Q_BYTES) + w * TI;
                *reinterpret_cast<float4 *>(qrow + VI * lane) = make_float4(out[0], out[1], out[2], out[3]);
                if (MID && m >= it.kb && m < it.kb + it.nout) {
                    // the intermediate state at this item's own points
                    const size_t offm = ((size_t)m * J + (size_t)j) * (size_t)pitch + (size_t)ib;
                    if (all_owned) {
                        store_vec<float, VI>(a.mid + offm, out, st_pol);
                    } else {
#pragma unroll
                        for (int e = 0; e < VI; ++e)
                            if (owned[e]) a.mid[offm + e] = out[e];
                    }
                }
                if (do2) {
                    tmem_wait_st();
                    tmem_before_sync();
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&q_full[qs % RQ]);            // intermediate plane s: this row written
                    mbar_arrive(&p_empty[(pc + s) % RP]);     // state plane m-1 is done
                    mbar_arrive(&c_empty[qs % RC]);     // stage s is done
                }
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) {                      // the item's last state planes
                mbar_arrive(&p_empty[(pc + it.nout + 2) % RP]);
                mbar_arrive(&p_empty[(pc + it.nout + 3) % RP]);
            }
            pc += it.nout + 4;
            qc += it.nout + 2;
        }
        if (!ok) {
            s_abort = 1;
            atomicExch(&a.hdr->errword, (int)JAC_ETIMEOUT);
        }
    } else {
        // ------------------------------------------------------- sweep-2 warps
        // A row's sweep-2 warp has the index of its sweep-1 warp modulo 4: the
        // two share a quarter of the tensor memory.
        const int w = (warp - S::WARP2) == 0 ? S::R2 : warp - S::WARP2;   // row j0-1+w of every item
        const float omega = (float)a.omega;
        const uint64_t st_pol = l2_policy(a.l2_keep_state ? 1 : 0);
        int I = d.I, J = d.J, pitch = d.pitch;
        const uint32_t tm = s_tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(((w - 1) >> 2) * S::TM_SLOTS * S::TM_SLOT);
        uint32_t qc = 0;
        bool ok = true;
        double acc = 0.0;
        uint32_t sync_phase = 0;
        auto cons_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(&cons_bar);
            const bool r = mbar_wait_bounded(&cons_bar, sync_phase & 1, limit);
            ++sync_phase;
            return __all_sync(0xffffffffu, r);
        };
        uint32_t entry;
        while ((ok = next_item(entry)) && entry != S::END) {
            const uint32_t t = entry / nitems;
            Item2 it;
            float *p_out;
            if constexpr (BATCH) {
                int item = (int)(entry - t * nitems);
                const Sweep2Desc *g = find_grid(a, item);
                it = decode_item2(*g, item);
                I = g->I; J = g->J; pitch = g->pitch;
                p_out = static_cast<float *>(g->p_buf[(t + 1 + a.par) & 1]);
            } else {
                it = decode_item2(d, (int)(entry - t * nitems));
                p_out = static_cast<float *>(((t + 1 + a.par) & 1) ? d.p_buf[1] : d.p_buf[0]);
            }
            const bool res = !BATCH && (t == (uint32_t)a.n_pass - 1) && (a.res != nullptr);
            const int j = it.j0 - 1 + w;
            const int ib = it.i0 + VI * lane;
            const bool row_in = j <= J - 2;
            bool owned[VI], all_owned = true;
#pragma unroll
            for (int e = 0; e < VI; ++e) {
                owned[e] = row_in && (ib + e >= 1) && (ib + e <= I - 2);
                all_owned = all_owned && owned[e];
            }
            const int q0 = (w - 1) * TI, q1 = w * TI, q2r = (w + 1) * TI;
            for (int s = 3; s < it.nout + 3; ++s) {
                // output plane kb-3+s from intermediate planes s-3 .. s-1
                const uint32_t qs = qc + s;
                const size_t off = ((size_t)(it.kb - 3 + s) * J + (size_t)j) * (size_t)pitch + (size_t)ib;
                const bool gone = s_abort;
                if (s == 3)
                    ok = mbar_wait_bounded(&q_full[qc % RQ], (qc / RQ) & 1, limit) &&
                         mbar_wait_bounded(&q_full[(qc + 1) % RQ], ((qc + 1) / RQ) & 1, limit);
                ok = ok && mbar_wait_bounded(&q_full[(qs - 1) % RQ], ((qs - 1) / RQ) & 1, limit);
                ok = __all_sync(0xffffffffu, ok && !gone);
                if (!ok) break;
                tmem_after_sync();
                const float *Qm =
                    reinterpret_cast<const float *>(ring_q + (size_t)((qs - 3) % RQ) * S::Q_BYTES);
                const float *Qk =
                    reinterpret_cast<const float *>(ring_q + (size_t)((qs - 2) % RQ) * S::Q_BYTES);
                const float *Qp =
                    reinterpret_cast<const float *>(ring_q + (size_t)((qs - 1) % RQ) * S::Q_BYTES);
                // columns i0-1 and i0+128 come from the edge warp
                const float(*Em)[2] = q_edge[(qs - 3) % RQ];
                const float(*Ek)[2] = q_edge[(qs - 2) % RQ];
                const float(*Ep)[2] = q_edge[(qs - 1) % RQ];
                float ek0[VI + 2], ek1[VI + 2], ek2[VI + 2], em1[VI + 2], ep1[VI + 2];
                float vm0[VI], vm2[VI], vp0[VI], vp2[VI];
                q_ext(Qk + q0, lane, Ek[w - 1][0], Ek[w - 1][1], ek0);
                q_ext(Qk + q1, lane, Ek[w][0], Ek[w][1], ek1);
                q_ext(Qk + q2r, lane, Ek[w + 1][0], Ek[w + 1][1], ek2);
                q_ext(Qm + q1, lane, Em[w][0], Em[w][1], em1);
                q_ext(Qp + q1, lane, Ep[w][0], Ep[w][1], ep1);
                lds_vec<float, VI>(Qm + q0 + VI * lane, vm0);
                lds_vec<float, VI>(Qm + q2r + VI * lane, vm2);
                lds_vec<float, VI>(Qp + q0 + VI * lane, vp0);
                lds_vec<float, VI>(Qp + q2r + VI * lane, vp2);
                const uint32_t at = tm + ((qs - 2) % S::TM_SLOTS) * S::TM_SLOT;
                float dd[VI], out[VI];
                {
                    float wk[VI], a0[VI], a1[VI], a2[VI], c0[VI], c1[VI], c2[VI];
                    tmem_ld16(at, wk, a0, a1, a2);
                    tmem_ld4(at + 16, c0);
                    tmem_ld4(at + 20, c1);
                    tmem_ld4(at + 24, c2);
                    tmem_wait_ld();
                    tmem_loaded(wk); tmem_loaded(a0); tmem_loaded(a1); tmem_loaded(a2);
                    tmem_loaded(c0); tmem_loaded(c1); tmem_loaded(c2);
                    ss_axes4(ek1, ek2, ek0, ep1, em1, a0, a1, a2, c0, c1, c2, wk, dd);
                }
                float ss2 = 0.0f;
                {
                    float b0[VI], b1[VI], b2[VI], a3[VI], bn[VI], ec[VI];
                    tmem_ld4(at + 28, b0);
                    tmem_ld4(at + 32, b1);
                    tmem_ld16(at + 36, b2, a3, bn, ec);
                    tmem_wait_ld();
                    tmem_loaded(b0); tmem_loaded(b1); tmem_loaded(b2);
                    tmem_loaded(a3); tmem_loaded(bn); tmem_loaded(ec);
#pragma unroll
                    for (int e = 0; e < VI; ++e) {
                        const float c = ek1[e + 1];
                        const float bij = ((ek2[e + 2] - ek0[e + 2]) - ek2[e]) + ek0[e];
                        const float bjk = ((vp2[e] - vm2[e]) - vp0[e]) + vm0[e];
                        const float bik = ((ep1[e + 2] - em1[e + 2]) - ep1[e]) + em1[e];
                        const float ss = ss_rest(dd[e], c, bij, bjk, bik, a3[e], b0[e], b1[e], b2[e], bn[e], ec[e]);
                        out[e] = owned[e] ? fmaf(omega, ss, c) : c;
                        if (res && owned[e]) ss2 = fmaf(ss, ss, ss2);
                    }
                }
                if (res) acc += (double)ss2;
                if (all_owned) {
                    store_vec<float, VI>(p_out + off, out, st_pol);
                } else {
#pragma unroll
                    for (int e = 0; e < VI; ++e)
                        if (owned[e]) p_out[off + e] = out[e];
                }
                tmem_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&q_empty[(qs - 3) % RQ]);   // intermediate plane s-3 done
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) {                      // the item's last intermediate planes
                mbar_arrive(&q_empty[(qc + it.nout) % RQ]);
                mbar_arrive(&q_empty[(qc + it.nout + 1) % RQ]);
            }
            qc += it.nout + 2;
            if (t + 1 < (uint32_t)a.n_pass) {
                // publish this row's part of the item to every CTA's TMA reads
                fence_proxy_async_global();
                __syncwarp();
                if (lane == 0) {
                    __threadfence();
                    atomicAdd(&a.hdr->gbar, 1u);
                }
            }
        }
        if (!BATCH && ok && a.res != nullptr) {
            double v = acc;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) s_part[w - 1] = v;
            ok = cons_sync();
            if (ok && warp == S::WARP2) {
                const double sum = warp_sum(lane < S::R2 ? s_part[lane] : 0.0, 0.0);
                if (lane == 0) a.partials[blockIdx.x] = sum;
            }
        }
        if (!ok) {
            s_abort = 1;
            atomicExch(&a.hdr->errword, (int)JAC_ETIMEOUT);
        }
    }

    // CTA epilogue: the last CTA to finish sums the partials in a fixed order
    // and resets the workspace counters for the next launch.
    // If any CTA gave up a wait, the residual is written as NaN.
    __syncthreads();
    if (warp == S::EDGE_WARP) {
        tmem_after_sync();
        tmem_dealloc(s_tmem, S::TM_COLS);
    }
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&a.hdr->counter, 1u);
        s_last = (prev == (unsigned)G - 1);
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (warp == 0) {
            if (a.res != nullptr) {
                const double sum = sum_partials(a.partials, G, lane);
                if (lane == 0)
                    *a.res = (s_abort || workspace_failed(a.hdr)) ? __longlong_as_double(0x7ff8000000000000ll) : sum;
            }
            if (lane == 0) {
                a.hdr->gbar = 0u;
                a.hdr->counter = 0u;
                a.hdr->ticket = 0u;
                a.hdr->clock = 0u;
                __threadfence();
            }
        }
    }
}

// ------------------------------------------------------------ host side
namespace {

jac_status fail2(jac_status st, const std::string &msg)
{
    set_thread_error(msg);
    return st;
}

}  // namespace

// Tiles in i: columns 128 n .. 128 n + 127, until one holds column I-2.
int sweep2_tiles_i(int I)
{
    using S = Sweep2Shape;
    return (I - 2) / S::TI + 1;
}

// Output planes per item: the depth that minimises the steps of a pass, the
// rounds of items over `ctas` CTAs times the steps of an item (its planes, the
// two extra planes of sweep 1 and about two steps of start-up); ties go to the
// shallower.  steps: that minimum.
int sweep2_kdepth(long cols, int nk, int ctas, long *steps = nullptr)
{
    if (nk <= 2) {
        if (steps) *steps = ((cols + ctas - 1) / ctas) * (nk + 4);
        return std::max(nk, 1);
    }
    long best_cost = -1;
    int best = 2;
    int prev = -1;
    for (int n = 1; n <= nk; ++n) {
        const int kd = std::max(2, (nk + n - 1) / n);
        if (kd == prev) continue;
        prev = kd;
        const long items = cols * (long)((nk + kd - 1) / kd);
        const long rounds = (items + ctas - 1) / ctas;
        const long cost = rounds * (long)(kd + 4);
        if (best_cost < 0 || cost < best_cost || (cost == best_cost && kd < best)) {
            best_cost = cost;
            best = kd;
        }
    }
    if (steps) *steps = best_cost;
    return best;
}

// Steps of a pass over the grid (one tile of 1024 points, both sweeps, each).
long sweep2_steps(const jac_grid *g, int sms)
{
    const long nti = sweep2_tiles_i(g->I), ntj = (g->J - 2 + Sweep2Shape::R2 - 1) / Sweep2Shape::R2;
    long steps = 0;
    sweep2_kdepth(nti * ntj, g->K - 2, sms, &steps);
    return steps;
}

// Passes of `nitems` items that one launch can count in 32 bits (even).
static int passes_per_launch(long long nitems)
{
    return (int)std::min<long long>(0x7ffffffe, (0xffff0000ll / (nitems * Sweep2Shape::R2)) & ~1ll);
}

int sweep2_batch_launches(int nitems, int n_pass)
{
    const int most = std::max(2, passes_per_launch(nitems));
    return n_pass / most + (n_pass % most != 0);
}

int sweep2_launches(const jac_grid *g, int n_pass, int sms)
{
    const long cols = (long)sweep2_tiles_i(g->I) * ((g->J - 2 + Sweep2Shape::R2 - 1) / Sweep2Shape::R2);
    const int kd = sweep2_kdepth(cols, g->K - 2, sms);
    return sweep2_batch_launches((int)(cols * ((g->K - 2 + kd - 1) / kd)), n_pass);
}

size_t sweep2_workspace_bytes(const jac_grid *g)
{
    using S = Sweep2Shape;
    const long long cols = (long long)sweep2_tiles_i(g->I) * ((g->J - 2 + S::R2 - 1) / S::R2);
    const int sms = device_sm_count();
    const int kd = sweep2_kdepth(cols, g->K - 2, sms);
    const long long items = cols * ((g->K - 2 + kd - 1) / kd);
    return kWsHeaderBytes + round_up((size_t)std::min<long long>(items, sms) * sizeof(double), 256);
}

namespace {

// Descriptor of one grid: tensor maps, tiling and item count.
jac_status build_desc2(Sweep2Desc *d, const jac_grid *g, int kdepth)
{
    using S = Sweep2Shape;
    std::memset(d, 0, sizeof(*d));
    d->I = g->I; d->J = g->J; d->K = g->K;
    d->pitch = jac_pitch(g->I);
    d->nti = sweep2_tiles_i(g->I);
    d->ntj = (g->J - 2 + S::R2 - 1) / S::R2;
    d->kdepth = kdepth;
    d->nkb = (g->K - 2 + kdepth - 1) / kdepth;
    const long long items = (long long)d->nti * d->ntj * d->nkb;
    if (items > 0x3fffffffLL) return fail2(JAC_EINVAL, "grid too large for the two-sweep launch shape");
    d->nitems = (int)items;
    d->p_buf[0] = g->p[0];
    d->p_buf[1] = g->p[1];
    jac_status s;
    for (int b = 0; b < 2; ++b)
        if ((s = encode_box_map(&d->p[b], g->p[b], 4, d->pitch, d->pitch, g->J, g->K, S::PW, S::PH)) != JAC_OK)
            return s;
    for (int q = JAC_A0; q <= JAC_BND; ++q) {
        if ((s = encode_box_map(&d->coef[q - 1], g->coef[q], 4, d->pitch, d->pitch, g->J, g->K, S::TI, S::R1)) !=
            JAC_OK)
            return s;
        d->coef_ptr[q - 1] = static_cast<const float *>(g->coef[q]);
    }
    return JAC_OK;
}

// All passes of a call.  Items of all passes and the arrivals of the pass
// barrier are counted in 32 bits: very long calls take several launches, each
// of an even number of passes.
template <bool BATCH, bool MID, bool STALL>
jac_status launch2(const Sweep2Desc &d, Sweep2Args a, unsigned nblocks, cudaStream_t st)
{
    using S = Sweep2Shape;
    static std::once_flag attr_once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(attr_once, [] {
        attr_err = cudaFuncSetAttribute(k_sweep2<BATCH, MID, STALL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)S::SMEM);
    });
    if (attr_err != cudaSuccess)
        return fail2(JAC_ECUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(attr_err));
    const int most = passes_per_launch(a.nitems);
    if (most < 2 && a.n_pass > most) return fail2(JAC_EINVAL, "grid too large for the two-sweep launch shape");
    double *const res = a.res;
    for (int left = a.n_pass; left > 0;) {
        a.n_pass = std::min(left, most);
        left -= a.n_pass;
        a.res = left == 0 ? res : nullptr;
        cudaLaunchConfig_t cfg;
        std::memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(nblocks);
        cfg.blockDim = dim3(S::THREADS);
        cfg.dynamicSmemBytes = S::SMEM;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_sweep2<BATCH, MID, STALL>, d, a);
        if (e != cudaSuccess) return fail2(JAC_ECUDA, std::string("two-sweep launch: ") + cudaGetErrorString(e));
    }
    return JAC_OK;
}

}  // namespace

jac_status sweep2_run(const jac_grid *g, int kdepth, int n_pass, double *d_residual, void *workspace,
                      size_t ws_bytes, cudaStream_t st, void *mid, const LaunchOpts *opts)
{
    if (mid != nullptr && n_pass != 1) return fail2(JAC_EINVAL, "the intermediate state needs a one-pass call");
    const long cols = (long)sweep2_tiles_i(g->I) * ((g->J - 2 + Sweep2Shape::R2 - 1) / Sweep2Shape::R2);
    const int sms = device_sm_count();
    Sweep2Desc d;
    jac_status s = build_desc2(&d, g, kdepth > 0 ? kdepth : sweep2_kdepth(cols, g->K - 2, sms));
    if (s != JAC_OK) return s;
    const unsigned nblocks = (unsigned)std::min(d.nitems, sms);
    if (ws_bytes < kWsHeaderBytes + (size_t)nblocks * sizeof(double))
        return fail2(JAC_EINVAL, "workspace too small for the two-sweep launch");
    Sweep2Args a;
    std::memset(&a, 0, sizeof(a));
    a.ngrids = 1;
    a.nitems = d.nitems;
    a.n_pass = n_pass;
    a.omega = g->omega;
    a.partials = reinterpret_cast<double *>(static_cast<char *>(workspace) + kWsHeaderBytes);
    a.res = d_residual;
    a.mid = static_cast<float *>(mid);
    a.hdr = static_cast<WsHeader *>(workspace);
    SweepArgs la;
    std::memset(&la, 0, sizeof(la));
    set_l2_policy(la, g->prec, (size_t)d.pitch * g->J * g->K);
    a.l2_keep_state = la.l2_keep_state;
    a.l2_keep_coef = la.l2_keep_coef;
    if (opts && (opts->wait_ns != 0 || opts->gbar_extra != 0)) {
        a.wait_ns = opts->wait_ns ? opts->wait_ns : kWaitLimitNs;
        a.gbar_extra = opts->gbar_extra;
        return launch2<false, false, true>(d, a, nblocks, st);
    }
    return mid != nullptr ? launch2<false, true, false>(d, a, nblocks, st)
                          : launch2<false, false, false>(d, a, nblocks, st);
}

// ---- batches: the descriptors of many grids in device memory
size_t sweep2_desc_bytes() { return sizeof(Sweep2Desc); }

jac_status sweep2_batch_desc(void *desc, const jac_grid *g, int kdepth, int *items)
{
    Sweep2Desc d;                  // tensor maps are encoded at multiples of 64; desc may lie anywhere
    const jac_status s = build_desc2(&d, g, kdepth);
    if (s != JAC_OK) return s;
    std::memcpy(desc, &d, sizeof(d));
    *items = d.nitems;
    return JAC_OK;
}

jac_status sweep2_batch_run(const void *descs, const int *item_base, int ngrids, int nitems, int n_pass, int par,
                            double omega, void *workspace, cudaStream_t st)
{
    Sweep2Args a;
    std::memset(&a, 0, sizeof(a));
    a.descs = static_cast<const Sweep2Desc *>(descs);
    a.item_base = item_base;
    a.ngrids = ngrids;
    a.nitems = nitems;
    a.n_pass = n_pass;
    a.par = par;
    a.omega = omega;
    a.hdr = static_cast<WsHeader *>(workspace);
    Sweep2Desc unused;
    std::memset(&unused, 0, sizeof(unused));
    return launch2<true, false, false>(unused, a, (unsigned)std::min(nitems, device_sm_count()), st);
}

}  // namespace jac
