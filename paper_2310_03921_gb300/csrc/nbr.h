// Neighbour search workspace and entry points (internal).
#pragma once

#include <vector>

#include "gap_internal.h"

struct CellGeom {
    double cell[9], inv[9];
    double rc2;
    float rc2_loose;  // squared cutoff widened past the FP32 rounding of cart32: the prefilter bound
    float rc2_tight;  // squared cutoff narrowed by the same margin: below it a pair is surely inside
    int nb[3], R[3], pbc[3];
    int bin0;
};

struct NbrWork {
    CellGeom *geo = nullptr;
    int *cfg_offsets = nullptr;
    D4 *cart = nullptr;        // wrapped atoms, Cartesian (x, y, z, near)
    float4 *cart32 = nullptr;  // FP32 copy of cart (prefilter of the candidate scans)
    int *atom_cfg = nullptr, *atom_bin = nullptr, *bin_atoms = nullptr, *counts = nullptr;
    int *bin_count = nullptr, *bin_start = nullptr;
    int *scan_tmp = nullptr, *total = nullptr;
    int *err = nullptr;  // of the caller (gap_neighbours)
    long long *keys = nullptr;
    PairList pairs{};
    // Graph mode (a captured MD step): no host synchronisation; the pair
    // arrays have a fixed capacity, cell geometry and configuration offsets
    // stay as the last ordinary build uploaded them.  A build that would
    // exceed the capacity leaves every atom without pairs and sets err bit 1.
    bool graph = false;
    int pair_cap = 0;
    size_t cap_geo = 0, cap_cfg = 0, cap_cart = 0, cap_acfg = 0, cap_abin = 0, cap_batoms = 0, cap_counts = 0,
           cap_offsets = 0, cap_bcount = 0, cap_bstart = 0, cap_scan = 0, cap_total = 0,
           cap_keys = 0, cap_i = 0, cap_j = 0, cap_rev = 0, cap_v64 = 0, cap_v32 = 0, cap_c32 = 0;

    gap_status reserve_atoms(int n, int n_configs, int n_bins);
    gap_status reserve_pairs(int P);
    void release();
};

gap_status gap_cell_geometry(const gap_batch *b, double rc, std::vector<CellGeom> &geo, int &n_bins);
// The call's device error words (err, cleared by the caller): a species
// outside 0 .. S - 1 sets err[1] (species NULL: not checked), the build's own
// code goes to err[kNbrErr].
constexpr int kNbrErr = 8;
// Builds the sorted CSR pair list of the batch on `st` (positions and species
// on the device).  Synchronises once to read the pair count (not in graph mode).
gap_status gap_neighbours(NbrWork &w, const gap_batch *b, const double *d_pos, const int *d_species, int S, double rc,
                          int *err, cudaStream_t st);
// The status of a build's error word: GAP_ECAPACITY for a graph-mode build
// beyond its pair capacity.
gap_status gap_neighbours_status(const NbrWork &w, int code);
// A scan with a capacity: see k_scan_out.
struct ScanCap {
    int cap = 0;
    int *used = nullptr, *err = nullptr;
};
gap_status gap_scan(const int *in, int n, int *out, int *tmp, int *total, cudaStream_t st, ScanCap cap = {});
size_t gap_scan_tmp_ints(int n);
