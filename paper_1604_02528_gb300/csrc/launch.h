// Host-side launchers of the sm_103a kernels (internal).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace selinv {

// counts kernel launches issued by the library (reported by selinv_launch_count)
void note_launch(int n = 1);

cudaError_t configure_selinv_kernels();
// L_KK^{-1} and Dinv_K by one CTA per supernode of at most 32 columns; large = 1:
// of any width (real, 194 KB of shared memory): the adjoints' one launch for all
// supernodes when none of them is on the tensor cores
cudaError_t launch_linv(int dtype, const ProbDesc *d, const int2 *work, int nwork, int large, cudaStream_t st);
// L_KK^{-1} of supernodes wider than 32 columns, kLinvCols columns per work entry
constexpr int kLinvCols = 8;
cudaError_t launch_linv_cols(int dtype, const ProbDesc *d, const int2 *work, int nwork, cudaStream_t st);
constexpr int kDinvTile = 16;
cudaError_t launch_dinv(int dtype, const ProbDesc *d, const int2 *work, int nwork, cudaStream_t st);
cudaError_t launch_selinv(int dtype, int bucket, const ProbDesc *d, const Item *items, int n,
                          cudaStream_t st);
// FP64 products of the level schedule (kernels_fma.cu): Lhat (narrow: s <= 16,
// tiles of kFmaNarrowRows rows; else of kFmaLhatRows, columns by kFmaCols),
// A^{-1}_{C,K} by tiles of `rows` rows x `cols` columns (16 or 32), and the
// diagonal block by 16 x 16 tiles; cl CTAs each
constexpr int kFmaCols = 32, kFmaLhatRows = 32, kFmaNarrowRows = 128;
cudaError_t launch_fma_lhat(int dtype, int narrow, const ProbDesc *d, const Item *items, int n, cudaStream_t st);
cudaError_t launch_fma_rows(int dtype, int rows, int cols, int cl, const ProbDesc *d, const Item *items, int n,
                            cudaStream_t st);
cudaError_t launch_fma_diag(int dtype, int cl, const ProbDesc *d, const Item *items, int n, cudaStream_t st);
cudaError_t configure_ozaki_kernels();
cudaError_t configure_tc_kernels();
cudaError_t launch_selinv_tc(int tn, const ProbDesc *d, const Item *items, int n, long long *slab,
                             long long wait_limit, cudaStream_t st);
cudaError_t launch_tc_reduce(int tn, const ProbDesc *d, const Item *items, const int4 *red, int n,
                             const long long *slab, cudaStream_t st);
cudaError_t configure_tcw_kernels();
cudaError_t launch_selinv_tcw(int cplx, const ProbDesc *d, const Item *items, int n, long long *slab,
                              long long wait_limit, cudaStream_t st);
cudaError_t launch_lhat_tcw(int cplx, const ProbDesc *d, const Item *items, int n, long long wait_limit, cudaStream_t st);
// mode 1: the reverse pass' update matrix, 2: the factorization's
cudaError_t launch_syrk_tcw(int mode, const ProbDesc *d, const Item *items, int n, long long wait_limit,
                            cudaStream_t st);
cudaError_t launch_tcw_reduce(int cplx, const ProbDesc *d, const Item *items, const int4 *red, int n,
                              const long long *slab, cudaStream_t st);
cudaError_t launch_diag_fin(const ProbDesc *d, const Item *items, int n, cudaStream_t st);
cudaError_t launch_diag_tc(int tn, int cplx, const ProbDesc *d, const Item *items, int n, long long wait_limit,
                           cudaStream_t st);
// complex left operands: of Lhat, or (linv) of L_KK^{-1}
cudaError_t launch_digits_z(int linv, const ProbDesc *d, const int2 *work, int nwork, cudaStream_t st);
cudaError_t launch_diag_fin_z(const ProbDesc *d, const Item *items, int n, cudaStream_t st);
cudaError_t launch_check_finite(const void *x, int64_t n_doubles, int *status, cudaStream_t st);
cudaError_t launch_selinv_persist(int dtype, const ProbDesc *d, const Item *items, const int8_t *buckets,
                                  int n, int *ticket, long long spin_limit, int wait_on_unset,
                                  cudaStream_t st);
cudaError_t launch_linv_digits(const ProbDesc *d, const int2 *work, int nwork, cudaStream_t st);
cudaError_t launch_lhat_oz(int tn, const ProbDesc *d, const Item *items, int n, cudaStream_t st);
// Narrow supernodes (at most kNarrowS columns, narrow_elems of shared memory
// within kNarrowSmem: two CTAs per SM): cl CTAs and smem bytes each
constexpr int kNarrowS = 16;
constexpr int kNarrowSmem = 110 * 1024, kNarrowAlone = 116 * 1024;
int narrow_elems(int s, int c, int cl, int lu);
cudaError_t configure_narrow_kernels();
cudaError_t launch_selinv_narrow(int dtype, int cl, int lu, int smem, const ProbDesc *d, const Item *items, int n,
                                 cudaStream_t st);
cudaError_t launch_push(int dtype, int kind, int bucket, const ProbDesc *d, const Item *items, int n,
                        cudaStream_t st);
cudaError_t launch_lhat_digits(const ProbDesc *d, const int2 *work, int nwork, cudaStream_t st);
cudaError_t launch_diag_oz(const ProbDesc *d, const Item *items, int n, cudaStream_t st);
cudaError_t launch_selinv_oz(int tn, const ProbDesc *d, const Item *items, int n, cudaStream_t st);

}  // namespace selinv
