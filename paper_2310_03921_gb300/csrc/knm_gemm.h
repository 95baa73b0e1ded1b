// K_NM force rows on the tensor cores (internal).
#pragma once

#include "gap_internal.h"

// A batch's Jacobian rows come in triples (x, y, z of one source atom's
// derivative with respect to one target atom), ordered by (GP of the source,
// target atom, own triple then neighbours): triple q holds rows 3 q .. 3 q + 2.
// Incoming triples are stored negated, so that every row is scaled by
// +W'[source].
struct KnmTriples {
    __nv_bfloat16 *hi, *lo, *mid;  // [3 triples][ld] BF16 planes of J (mid: three-plane split)
    float4 *meta;                  // [triples] J . mu of the three rows, then the source's row among its GP's atoms
    int *dest;                     // [triples] first of the target's three K rows at a target's last triple, else -1
    int *src;                      // [triples] source atom (compressed descriptors; else NULL)
    const int *first;              // [n_gp n + 1] first triple of (GP, target)
    const int *slot;               // [P] pair (j -> i): place of i's triple among those of target j and i's GP
    const int *rank;               // [n] an atom's row among its GP's atoms
    const int *atom_cfg;           // [n]
};

constexpr int kKnmMaxGPs = 8;
struct KnmGP {
    int M, M_pad, R;                            // sparse points, their padding, atoms of the GP
    const __nv_bfloat16 *B_hi, *B_lo, *B_mid;   // [M_pad][K] centred sparse points
    const float *Wp, *kq;                       // [R][M_pad] W' and k of the GP's atoms
    const int *rows;                            // [R] its atoms, ascending
    int col0;                                   // its first column of K
};

// slot[P] and counts[n_gp][n] (triples per GP and target; scanned into
// KnmTriples::first by the caller) of a pair list.
gap_status gap_knm_slots(int n, int n_gp, const int *offsets, const int *nbr_j, const int *gp_of_atom, int *slot,
                         int *counts, cudaStream_t st);
// Work ranges of the force GEMM: ints of scratch it needs.
size_t gap_knm_bounds_ints(int n_gp);
// K[dest + a][col0 + m] = sum over the target's triples of W'[source][m]
// (J_a . (x_m - mu) + J_a . mu) for every GP with atoms and sparse points, one
// launch.  K (the product's inner size) is a multiple of 16; nsplit as in
// TcOperands; n_triples the host's count (all GPs).
gap_status gap_knm_force_tc(const KnmTriples &t, long n_triples, int n, int K, int nsplit, const KnmGP *gps, int n_gp,
                            int *bounds, double *Kout, long ldk, int *err, cudaStream_t st);
// Energy rows K[c + 3 first atom of c][col0 + m] = sum of kq over the configuration's atoms of each GP.
gap_status gap_knm_energy_tc(int n_configs, const int *cfg_off, const KnmGP *gps, int n_gp, double *Kout, long ldk,
                             cudaStream_t st);
