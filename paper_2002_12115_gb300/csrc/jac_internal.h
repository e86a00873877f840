// Internal interfaces shared by the translation units of libjac.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <string>

#include "../../include/jacobi.h"

namespace jac {

struct GridDesc;
struct SweepArgs;
struct WsHeader;

const char *thread_last_error();
void set_thread_error(const std::string &m);

jac_status validate_grid(const jac_grid *g);
jac_plan resolve_plan(const jac_grid *g, const jac_plan *plan);
jac_plan resolve_plan_sms(const jac_grid *g, const jac_plan *plan, int sms);
// Bytes of workspace a sweep with this resolved plan needs, and those with
// which every path open to `plan` may run (more where it is all zero).
size_t sweep_workspace_bytes(const jac_grid *g, const jac_plan &p);
size_t sweep_workspace_reported(const jac_grid *g, const jac_plan *plan);
// Launch options of the single-grid sweep.  wait_ns and gbar_extra are set
// only by a test of the failure path: a shorter limit for the waits on other
// warps and CTAs, and an offset that makes the launch's grid barrier
// unreachable.  They do not change the kernel, except that a grid of one
// resident box, which waits for nobody, streams.
// no_residual: nobody reads this launch's residual, so none is summed.
struct LaunchOpts {
    unsigned long long wait_ns = 0;
    unsigned gbar_extra = 0;
    bool no_residual = false;
};
jac_status sweep_dev(const jac_grid *g, const jac_plan *plan, int n_iter, double *d_residual, void *workspace,
                     size_t ws_bytes, void *stream, const LaunchOpts *opts = nullptr);
// Dense FP64 (or FP32) arrays into storage layout and back (jac_pack.cu).
// pack_fields packs all thirteen arrays of a grid in one launch, p into dst[0]
// and p2; pack_dev packs one array, into dst and, if not NULL, dst2.
jac_status pack_dev(int I, int J, int K, jac_prec prec, int which, const double *src, void *dst, cudaStream_t st,
                    void *dst2 = nullptr);
jac_status pack_fields(int I, int J, int K, jac_prec prec, const double *const *src, void *const *dst, void *p2,
                       cudaStream_t st);
jac_status pack_fields_f32(int I, int J, int K, jac_prec prec, const float *const *src, void *const *dst, void *p2,
                           cudaStream_t st);
jac_status unpack_dev(int I, int J, int K, jac_prec prec, int which, const void *src, double *dst,
                      cudaStream_t st);
jac_status unpack_dev_f32(int I, int J, int K, jac_prec prec, int which, const void *src, float *dst,
                          cudaStream_t st);
jac_status workspace_check(void *workspace, cudaStream_t st);
jac_status workspace_read(void *workspace, cudaStream_t st, WsHeader *out);
int device_sm_count();
size_t device_l2_bytes();
void set_l2_policy(SweepArgs &a, jac_prec prec, size_t points);
int vector_points(jac_prec prec);
int max_row_fold(jac_prec prec, int tj);
bool warps_supported(jac_prec prec, int tj);
int best_tile_i(int I, int J, jac_prec prec, int tj);
jac_status check_plan(jac_prec prec, const jac_plan &p, int *rw_out, int *tj_out);
jac_status build_desc(GridDesc *d, const jac_grid *g, const jac_plan &p, int item_base);
template <bool BATCH>
jac_status launch_sweep(jac_prec prec, int tj, const GridDesc &d0, const SweepArgs &a, unsigned nblocks,
                        cudaStream_t st);
// Two-sweep passes (FP32 storage): n_pass passes of two sweeps each, in one
// cooperative launch (very long calls: several); pass t reads p[t & 1] and
// writes the other buffer.  The residual of the last sweep goes to d_residual
// (NULL: none).  kdepth 0: the default depth.  mid (one-pass calls only) also
// receives the state after the first sweep at every interior point; its faces
// are left as they are.  opts: only its wait_ns and gbar_extra are read; with
// either one set mid is not written.
jac_status sweep2_run(const jac_grid *g, int kdepth, int n_pass, double *d_residual, void *workspace,
                      size_t ws_bytes, cudaStream_t st, void *mid = nullptr, const LaunchOpts *opts = nullptr);
// Whether the library's plan for this grid takes two-sweep passes (fuse 0).
bool two_sweep_default(const jac_grid *g);
size_t sweep2_workspace_bytes(const jac_grid *g);
// Steps of a two-sweep pass over the grid on `sms` SMs, and the launches that
// n_pass of them take.
long sweep2_steps(const jac_grid *g, int sms);
int sweep2_launches(const jac_grid *g, int n_pass, int sms);
// Two-sweep passes of a batch: descriptors (sweep2_desc_bytes each, built on
// the host at any address, used from device memory at a multiple of 64) and
// first items of its grids.  No residual; n_pass even; pass t reads
// p[(t + par) & 1].
size_t sweep2_desc_bytes();
jac_status sweep2_batch_desc(void *desc, const jac_grid *g, int kdepth, int *items);
int sweep2_batch_launches(int nitems, int n_pass);
jac_status sweep2_batch_run(const void *descs, const int *item_base, int ngrids, int nitems, int n_pass, int par,
                            double omega, void *workspace, cudaStream_t st);
// Resident sweeps (jac_resident.cu): the boxes of a small grid, one per CTA,
// whose coefficients stay in shared memory for all sweeps of a call.
struct ResidentShape {
    int nj, nk;        // boxes along j and k
    int bj, bk;        // most rows of a box along j and k
    int ws;            // shared-memory row length (elements)
    size_t smem;       // dynamic shared memory of a CTA
};
// False where the grid does not fit in the shared memory of `sms` SMs.
bool resident_shape(int I, int J, int K, jac_prec prec, int sms, ResidentShape *out);
size_t resident_workspace_bytes(const ResidentShape &s);
// d_residual NULL: no residual is summed.  hist not NULL: state t + 1 goes
// whole to hist + t * hist_stride (bytes; faces and padding already there)
// and p[1] is not used.  opts: only its wait_ns and gbar_extra are read.
jac_status resident_run(const jac_grid *g, const ResidentShape &s, int n_iter, double *d_residual, void *workspace,
                        cudaStream_t st, void *hist = nullptr, size_t hist_stride = 0,
                        const LaunchOpts *opts = nullptr);
// Whether a call of n_iter sweeps with this plan and workspace can run resident.
bool use_resident(const jac_grid *g, const jac_plan *plan, int n_iter, size_t ws_bytes, ResidentShape *r);
jac_status adjoint_step_dev(const jac_grid *g, const void *p_t, const void *lam_in, void *lam_out, double *g_wrk1,
                            double *g_a3, double *const *g_coef, int kdepth, void *workspace, size_t ws_bytes,
                            cudaStream_t st);
// 3-D tensor map of one storage-layout array (row pitch `pitch` elements)
// with extent (extent_i, J, K), so that columns at i >= extent_i read as
// zero, and a (bx, by, 1) box.
jac_status encode_box_map(CUtensorMap *m, const void *base, size_t elem, int extent_i, int pitch, int J, int K,
                          int bx, int by);

}  // namespace jac
