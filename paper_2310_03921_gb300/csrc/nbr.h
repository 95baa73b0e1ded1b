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
    int *scan_tmp = nullptr;
    int *total = nullptr, *err = nullptr;  // in the caller's words (gap_neighbours)
    long long *keys = nullptr;
    PairList pairs{};
    // Graph mode (a captured MD step): no host synchronisation; the pair
    // arrays have a fixed capacity, cell geometry and configuration offsets
    // stay as the last ordinary build uploaded them.  A build that would
    // exceed the capacity leaves every atom without pairs and sets err bit 1.
    bool graph = false;
    int pair_cap = 0;
    // Pinned copy of the cell geometry and offsets on its way to the device
    // (in_flight until the caller has synchronised), and the most pairs per
    // atom any finished build of this workspace had: the pair capacity of a
    // build that does not wait for its pair count (gap_neighbours).
    void *stage = nullptr;
    bool in_flight = false;
    int n_atoms = 0;
    double pairs_per_atom = 0.0;
    size_t cap_stage = 0;
    size_t cap_geo = 0, cap_cart = 0, cap_acfg = 0, cap_abin = 0, cap_batoms = 0, cap_counts = 0,
           cap_offsets = 0, cap_bcount = 0, cap_bstart = 0, cap_scan = 0,
           cap_keys = 0, cap_i = 0, cap_j = 0, cap_rev = 0, cap_v64 = 0, cap_v32 = 0, cap_c32 = 0;

    gap_status reserve_atoms(int n, int n_configs, int n_bins);
    gap_status reserve_pairs(int P);
    void release();
};

gap_status gap_cell_geometry(const gap_batch *b, double rc, std::vector<CellGeom> &geo, int &n_bins);
// A call's device words (int [kWords], cleared by the caller) and their
// pinned host copy: a species outside 0 .. S - 1 sets [1] (species NULL: not
// checked), the build's own code goes to [kNbrErr], the pair count to
// [kNbrTotal] (the pairs in the lists to the next), the rows of each GP to
// [kGpCounts ..].
constexpr int kNbrErr = 8, kNbrTotal = 16, kGpCounts = 18, kWords = 32;
// Builds the sorted CSR pair list of the batch on `st` (positions and species
// on the device).  Synchronises once to read the words (`host`) and with them
// the pair count, except in graph mode and when `ahead` is allowed and the
// workspace has finished a build before: the arrays then get room for the
// most pairs per atom seen so far (2^20 pairs in all at most, else it waits),
// and a batch with more empties every list
// and ends in GAP_ECAPACITY (gap_neighbours_done), to be run again without
// `ahead`, as is a call whose room ahead could not be had (GAP_ENOMEM).
gap_status gap_neighbours(NbrWork &w, const gap_batch *b, const double *d_pos, const int *d_species, int S, double rc,
                          int *words, int *host, bool ahead, cudaStream_t st);
// The status of a build from its words on the host, the stream synchronised.
gap_status gap_neighbours_done(NbrWork &w, const int *host);
// A scan with a capacity: see k_scan_out.
struct ScanCap {
    int cap = 0;
    int *used = nullptr, *err = nullptr;
};
gap_status gap_scan(const int *in, int n, int *out, int *tmp, int *total, cudaStream_t st, ScanCap cap = {});
size_t gap_scan_tmp_ints(int n);
