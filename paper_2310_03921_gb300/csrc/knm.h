// K_NM assembly kernels (internal).
#pragma once

#include "gap_internal.h"
#include "knm_gemm.h"

// Jacobian rows of the force-row GEMM: target-major rows in T (CUDA-core
// forms, see knm.cu), or the triples of the tensor-core form.
struct KnmRows {
    void *A;        // [rows][D16] T
    int *src_sign;  // [rows] +(atom+1) own row, -(atom+1) incoming row
    int *seg;       // [rows] segment (3 * target + xyz) of each row
    KnmTriples tri;
};

gap_status gap_knm_segments(int n, const int *offsets, const int *atom_cfg, int *seg_start, int *out_row,
                            cudaStream_t st);
template <typename T>
gap_status gap_jacobian_rows(const SoapGeom &g, const T *tab, int n, const PairList &pl, const int *species,
                             const T *coef, const T *phat, const T *pnorm, KnmRows &out, cudaStream_t st);
// The tensor-core form's triples (mu_all NULL: J . mu written as 0).
gap_status gap_jacobian_triples(const SoapGeom &g, const float *tab, int n, const PairList &pl, const int *species,
                                const float *coef, const float *phat, const float *pnorm, const int *gp_of_atom,
                                const float *mu_all, const KnmTriples &tr, cudaStream_t st);
// Compressed descriptors (p~ = Q p renormalised): V = J Q^T for rows J
// [nrow][ldj] in T and Q [Dg][D] (CUDA-core forms; V [nrow][ldv], columns
// Dg .. ldv - 1 untouched) ...
template <typename T>
gap_status gap_rows_times_qt(long nrow, int D, const T *J, int ldj, int Dg, const T *Q, T *V, int ldv,
                             cudaStream_t st);
// ... and the compressed rows J~ = (|p| / |p~|) (I - p_hat~ p_hat~^T) V of each
// row's source atom, [nrow][Dg16] into out.A (T; may alias V when ldv ==
// Dg16) or, SPLIT, into the planes of out.tri with J~ . mu~ of the source
// atom's GP (mu_all [n_gp][Dg16]) into its meta; src_sign is read for the
// CUDA-core forms, out.tri.src for SPLIT.
template <typename T, bool SPLIT>
gap_status gap_jacobian_compress(long nrow, int Dg, int Dg16, const T *V, int ldv, const int *src_sign,
                                 const int *gp_of_atom, const T *phatc, const T *pnorm, const T *pnormc,
                                 const float *mu_all, KnmRows &out, cudaStream_t st);
template <typename T>
gap_status gap_knm_qpow_simt(const T *phat, int D, const int *rows, int nrows, const T *X, int M, double delta,
                             int zeta, T *Wp, T *kq, int ld, cudaStream_t st);
template <typename T>
gap_status gap_knm_force_simt(const T *A, int D, int D16, long nrow, const int *seg, int n_seg, const int *seg_start,
                              const int *out_row, const int *src_sign, const T *X, int M, const T *Wp, int ldw,
                              double *K, int ldk, int col_out0, T *P, int ldp, cudaStream_t st);
template <typename T>
gap_status gap_knm_energy(int n_configs, const int *cfg_off, const T *kq, int ld, int M, double *K, int ldk,
                          int col_out0, cudaStream_t st);
