// Cell-list neighbour search with periodic images.
//
// Every directed pair (i, j, T) with |r_j + T - r_i| < r_c is listed, where
// T runs over all lattice translations (j = i allowed for T != 0): the
// connectivity "based on the cutoff" of Sec. 3.1.1 and the sum over all
// neighbours of Eq. 19.  Per configuration, fractional coordinates are
// wrapped into [0, 1) along periodic axes and binned on a grid whose bins are
// at least r_c wide in perpendicular width, or, for cells thinner than r_c,
// one bin per axis searched over several images.  Each atom's list is sorted
// by (j, shift), so the output does not depend on the order in which atomics
// filled the bins.
#include "gap_internal.h"
#include "nbr.h"

#include <cmath>
#include <cstring>
#include <vector>

namespace {

constexpr int kShiftBias = 128;

// A lattice shift packed into 24 bits, ordered as (sx, sy, sz).
__device__ __forceinline__ int shift_code(int sx, int sy, int sz)
{
    return ((sx + kShiftBias) << 16) | ((sy + kShiftBias) << 8) | (sz + kShiftBias);
}
constexpr int kNoShift = (kShiftBias << 16) | (kShiftBias << 8) | kShiftBias;

__device__ __forceinline__ long long pair_key(int j, int code) { return ((long long)j << 24) | (long long)code; }

__device__ __forceinline__ int config_of(const int *offsets, int n_configs, int i)
{
    int lo = 0, hi = n_configs - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (offsets[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// What a build needs of the batch; err[1] is set for a species outside 0 .. S - 1.
struct BinInputs {
    int n, n_configs, S;
    const double *pos;
    const int *species, *offsets;
    const CellGeom *geo;
    int *err;
};

// Atom i: wrapped Cartesian coordinates, configuration and bin (returned).
__device__ __forceinline__ int bin_atom(const BinInputs &in, int i, D4 *cart, float4 *cart32, int *atom_cfg,
                                        int *atom_bin)
{
    const double *pos = in.pos;
    const int *offsets = in.offsets;
    const int n_configs = in.n_configs;
    const CellGeom *geo = in.geo;
    if (in.species && (in.species[i] < 0 || in.species[i] >= in.S)) atomicOr(in.err + 1, 1);
    int c = config_of(offsets, n_configs, i);
    const CellGeom &g = geo[c];
    double p[3] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]};
    int b[3];
    double fr[3];
    for (int k = 0; k < 3; ++k) {
        double s = p[0] * g.inv[k] + p[1] * g.inv[3 + k] + p[2] * g.inv[6 + k];
        if (g.pbc[k]) {
            s -= floor(s);
            if (s >= 1.0) s = 0.0;
        }
        int bk = (int)floor(s * g.nb[k]);
        bk = bk < 0 ? 0 : (bk >= g.nb[k] ? g.nb[k] - 1 : bk);
        fr[k] = s;
        b[k] = bk;
    }
    int gb = g.bin0 + (b[0] * g.nb[1] + b[1]) * g.nb[2] + b[2];
    // the wrapped atom in Cartesian coordinates; w = 1 marks fractional
    // coordinates within [-4, 4] (always so along periodic directions), where
    // the FP32 copy is close enough for the prefilter
    const bool near = fabs(fr[0]) <= 4.0 && fabs(fr[1]) <= 4.0 && fabs(fr[2]) <= 4.0;
    double x[3];
    for (int a = 0; a < 3; ++a) x[a] = fr[0] * g.cell[a] + fr[1] * g.cell[3 + a] + fr[2] * g.cell[6 + a];
    cart[i] = D4{x[0], x[1], x[2], near ? 1.0 : 0.0};
    cart32[i] = make_float4((float)x[0], (float)x[1], (float)x[2], near ? 1.f : 0.f);
    atom_cfg[i] = c;
    atom_bin[i] = gb;
    return gb;
}

__global__ void k_bin(BinInputs in, D4 *__restrict__ cart, float4 *__restrict__ cart32, int *__restrict__ atom_cfg,
                      int *__restrict__ atom_bin, int *__restrict__ bin_count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < in.n) atomicAdd(&bin_count[bin_atom(in, i, cart, cart32, atom_cfg, atom_bin)], 1);
}

// A bin's places are taken from the end of its count.
__global__ void k_scatter(int n, const int *__restrict__ atom_bin, const int *__restrict__ bin_start,
                          int *__restrict__ bin_count, int *__restrict__ bin_atoms)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int gb = atom_bin[i];
    int slot = atomicSub(&bin_count[gb], 1) - 1;
    bin_atoms[bin_start[gb] + slot] = i;
}

// Exclusive prefix of v over the 1024 threads of a block; *total their sum.
__device__ __forceinline__ int block_prefix(int v, int *warp_tot, int *total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();  // warp_tot of an earlier call is read
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    int t = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
    }
    *total = __shfl_sync(0xffffffffu, t, 31);
    const int before = __shfl_sync(0xffffffffu, t, w > 0 ? w - 1 : 0);
    return (w > 0 ? before : 0) + x - v;
}

// The whole binning of a small batch (up to kSmallAtoms atoms and kSmallBins
// bins) in one block: at these sizes a build is launch latency, and this is
// one launch for a clear, the bins, a scan and the scatter (2 us each).  One
// SM's FP64 pipe takes the ~40 FP64 instructions of 256 atoms in about 3 us;
// beyond that the spread kernels are faster.
constexpr int kSmallAtoms = 256, kSmallBins = 4096;
__global__ void __launch_bounds__(1024)
k_bin_small(BinInputs in, int n_bins, D4 *__restrict__ cart, float4 *__restrict__ cart32, int *__restrict__ atom_cfg,
            int *__restrict__ atom_bin, int *__restrict__ bin_start, int *__restrict__ bin_atoms)
{
    __shared__ int cnt[kSmallBins], warp_tot[32];
    const int i = threadIdx.x;
    for (int b = i; b < n_bins; b += 1024) cnt[b] = 0;
    __syncthreads();
    int gb = 0;
    if (i < in.n) {
        gb = bin_atom(in, i, cart, cart32, atom_cfg, atom_bin);
        atomicAdd(&cnt[gb], 1);
    }
    __syncthreads();
    const int items = (n_bins + 1023) / 1024;  // consecutive bins of this thread
    int sum = 0, total;
    for (int k = 0; k < items; ++k) {
        const int b = i * items + k;
        if (b < n_bins) sum += cnt[b];
    }
    int at = block_prefix(sum, warp_tot, &total);
    for (int k = 0; k < items; ++k) {
        const int b = i * items + k;
        if (b < n_bins) {
            const int c = cnt[b];
            bin_start[b] = at;
            cnt[b] = at;  // becomes the bin's next free place
            at += c;
        }
    }
    if (i == 0) bin_start[n_bins] = total;
    __syncthreads();
    if (i < in.n) bin_atoms[atomicAdd(&cnt[gb], 1)] = i;
}

// floor(a / n) for n > 0.
__device__ __forceinline__ int floor_div(int a, int n) { return a >= 0 ? a / n : -((n - 1 - a) / n); }

// Per warp: the non-empty bins of the current chunk of 32 bins around the
// atom (their lattice shifts in FP64 and FP32, the offset taking a candidate's
// number to its slot of bin_atoms, the packed shift) and the candidates that
// wait for the exact test.
constexpr int kNbrQueue = 64;
struct NbrScan {
    double T[32][3];
    float4 T32[32];
    int first[32], code[32];
    int2 queue[kNbrQueue];  // (atom, bin slot)
};

// Visits every candidate (j, shift) of atom i, one warp per atom, 32 at a
// time; f(hit, j, code, v, r2) is called by every lane with uniform control
// flow (it may use warp votes), hit marking a pair within the cutoff.  The
// bins around the atom ((2R+1)^3, 32 at a time: lane b resolves bin b's
// periodic shift and atom range) are flattened into one run of candidates,
// which the lanes take 32 at a time through an FP32 prefilter: the cutoff
// widened by 5 10^-4 rc + 3 10^-5 of the cell's edge lengths, beyond the error
// of the FP32 coordinates and shifts (~4 10^-6 of the edges at 60 images;
// atoms far outside the box of a non-periodic direction skip it).  The
// survivors (~15%) queue in shared memory and take the exact FP64 test 32 at
// a time.  GB300's FP64 pipe takes about 64 cycles per warp instruction
// whatever the active lanes, and bounded this scan: so every FP64 instruction
// works on a full warp, the exact test is r = (x_j - x_i) + T on wrapped
// Cartesian coordinates (six additions; the reverse pair gets exactly the
// negative), the shifts T are formed once per bin (not at all for an atom
// whose bins need none), and bin wrapping is integer arithmetic.  The pair
// set is the FP64 one.  (With FP64 fractional coordinates, divisions and
// square roots a step of 32768 atoms took 0.13 ms longer, 512 four-species
// boxes 0.4 ms.)
// SURE (counting only): a candidate whose FP32 distance is below the cutoff
// narrowed by the same margin is inside for FP64 too; it is counted in
// sure_hits without the exact test, which then sees only the thin shell
// between the two bounds.
template <bool SURE, typename F>
__device__ __forceinline__ void warp_candidates(int i, int lane, const D4 *__restrict__ cart,
                                                const float4 *__restrict__ cart32, const int *__restrict__ atom_cfg,
                                                const int *__restrict__ atom_bin, const CellGeom *__restrict__ geo,
                                                const int *__restrict__ bin_start,
                                                const int *__restrict__ bin_atoms, NbrScan &sc, F &&f, int &sure_hits)
{
    const CellGeom &g = geo[atom_cfg[i]];
    const D4 xi = cart[i];
    const float4 xi32 = cart32[i];
    const int nb0 = g.nb[0], nb1 = g.nb[1], nb2 = g.nb[2], ib = atom_bin[i] - g.bin0;
    const int b2 = ib % nb2, b1 = (ib / nb2) % nb1, b0 = ib / (nb2 * nb1);
    const double rc2 = g.rc2;
    const float loose = g.rc2_loose, tight = g.rc2_tight;
    const unsigned lt = (1u << lane) - 1u;
    int qn = 0;  // queued candidates
    // the exact test of queue[0 .. cnt) (cnt <= 32), one per lane
    auto drain = [&](int cnt) {
        bool hit = false;
        int j = -1, code = 0;
        double v[3] = {0.0, 0.0, 0.0}, r2 = 0.0;
        if (lane < cnt) {
            const int2 e = sc.queue[lane];
            j = e.x;
            code = sc.code[e.y];
            const D4 xj = cart[j];
            v[0] = (xj.x - xi.x) + sc.T[e.y][0];
            v[1] = (xj.y - xi.y) + sc.T[e.y][1];
            v[2] = (xj.z - xi.z) + sc.T[e.y][2];
            r2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
            hit = r2 < rc2;
        }
        f(hit, j, code, v, r2);
    };
    const int wx = 2 * g.R[0] + 1, wy = 2 * g.R[1] + 1, wz = 2 * g.R[2] + 1, nbins = wx * wy * wz;
    for (int c0b = 0; c0b < nbins; c0b += 32) {
        int st = 0, cnt = 0, sx = 0, sy = 0, sz = 0;
        const int bb = c0b + lane;
        if (bb < nbins) {
            int nz = b2 + bb % wz - g.R[2], ny = b1 + (bb / wz) % wy - g.R[1], nx = b0 + bb / (wz * wy) - g.R[0];
            bool ok = true;
            if (g.pbc[0]) { sx = floor_div(nx, nb0); nx -= sx * nb0; }
            else ok = ok && nx >= 0 && nx < nb0;
            if (g.pbc[1]) { sy = floor_div(ny, nb1); ny -= sy * nb1; }
            else ok = ok && ny >= 0 && ny < nb1;
            if (g.pbc[2]) { sz = floor_div(nz, nb2); nz -= sz * nb2; }
            else ok = ok && nz >= 0 && nz < nb2;
            if (ok) {
                const int gb = g.bin0 + (nx * nb1 + ny) * nb2 + nz;
                st = bin_start[gb];
                cnt = bin_start[gb + 1] - st;
            }
        }
        // exclusive prefix of the bin sizes
        int pre = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, pre, o);
            if (lane >= o) pre += t;
        }
        const int total = __shfl_sync(0xffffffffu, pre, 31);
        pre -= cnt;
        const unsigned full = __ballot_sync(0xffffffffu, cnt > 0);
        const int code = shift_code(sx, sy, sz);
        const bool shifted = __ballot_sync(0xffffffffu, cnt > 0 && code != kNoShift) != 0;
        __syncwarp();  // the previous chunk's drain has read the tables
        if (cnt > 0) {
            const int slot = __popc(full & lt);
            double T[3] = {0.0, 0.0, 0.0};
            if (shifted)
                for (int a = 0; a < 3; ++a)
                    T[a] = (double)sx * g.cell[a] + (double)sy * g.cell[3 + a] + (double)sz * g.cell[6 + a];
            for (int a = 0; a < 3; ++a) sc.T[slot][a] = T[a];
            sc.T32[slot] = make_float4((float)T[0], (float)T[1], (float)T[2], 0.f);
            sc.first[slot] = st - pre;
            sc.code[slot] = code;
        }
        __syncwarp();
        for (int c0 = 0; c0 < total; c0 += 32) {
            const int c = c0 + lane;
            // the bin of candidate c: bins that start at or before it, from
            // the starts in this window and the number before it
            const unsigned heads =
                __reduce_or_sync(0xffffffffu, cnt > 0 && pre >= c0 && pre < c0 + 32 ? 1u << (pre - c0) : 0u);
            const int slot = __popc(__ballot_sync(0xffffffffu, cnt > 0 && pre < c0)) +
                             __popc(heads & (lt | (1u << lane))) - 1;
            bool pass = false, sure = false;
            int j = -1;
            if (c < total) {
                j = bin_atoms[sc.first[slot] + c];
                if (!(j == i && sc.code[slot] == kNoShift)) {
                    pass = true;
                    const float4 xj = cart32[j], T = sc.T32[slot];
                    if (xi32.w != 0.f && xj.w != 0.f) {
                        const float d0 = (xj.x - xi32.x) + T.x, d1 = (xj.y - xi32.y) + T.y, d2 = (xj.z - xi32.z) + T.z;
                        const float r2f = d0 * d0 + d1 * d1 + d2 * d2;
                        pass = r2f < loose;
                        if (SURE && r2f < tight) {
                            sure = true;
                            pass = false;
                        }
                    }
                }
            }
            if (SURE) sure_hits += __popc(__ballot_sync(0xffffffffu, sure));
            const unsigned pm = __ballot_sync(0xffffffffu, pass);
            if (pass) sc.queue[qn + __popc(pm & lt)] = make_int2(j, slot);
            qn += __popc(pm);
            __syncwarp();
            if (qn >= 32) {
                drain(32);
                __syncwarp();
                qn -= 32;
                if (lane < qn) sc.queue[lane] = sc.queue[32 + lane];
                __syncwarp();
            }
        }
        if (qn > 0) {  // before the next chunk's tables
            drain(qn);
            qn = 0;
        }
    }
}

constexpr int kNbrWarps = 4;   // warps (atoms) per block
constexpr int kNbrSort = 128;   // pairs per atom sorted in shared memory

__global__ void __launch_bounds__(32 * kNbrWarps)
k_count_warp(int n, const D4 *__restrict__ cart, const float4 *__restrict__ cart32,
             const int *__restrict__ atom_cfg, const int *__restrict__ atom_bin, const CellGeom *__restrict__ geo,
             const int *__restrict__ bin_start, const int *__restrict__ bin_atoms, int *__restrict__ counts)
{
    __shared__ NbrScan scan[kNbrWarps];
    const int i = blockIdx.x * kNbrWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n) return;
    int c = 0, sure = 0;
    warp_candidates<true>(i, lane, cart, cart32, atom_cfg, atom_bin, geo, bin_start, bin_atoms, scan[threadIdx.x >> 5],
                          [&](bool hit, int, int, const double *, double) {
                              c += __popc(__ballot_sync(0xffffffffu, hit));
                          },
                          sure);
    if (lane == 0) counts[i] = c + sure;
}

// The pairs of atom i sorted by (j, shift): gathered in shared memory and
// placed by rank (keys are distinct), or, beyond kNbrSort pairs, written in
// scan order and insertion-sorted by one lane.
__global__ void __launch_bounds__(32 * kNbrWarps)
k_fill_warp(int n, const D4 *__restrict__ cart, const float4 *__restrict__ cart32,
            const int *__restrict__ atom_cfg, const int *__restrict__ atom_bin, const CellGeom *__restrict__ geo,
            const int *__restrict__ bin_start, const int *__restrict__ bin_atoms, const int *__restrict__ offsets,
            int cap, long long *__restrict__ keys, int *__restrict__ pair_i, int *__restrict__ nbr_j,
            D4 *__restrict__ vec64, float4 *__restrict__ vec32, int *__restrict__ err)
{
    __shared__ __align__(16) long long skey[kNbrWarps][kNbrSort];
    __shared__ D4 svec[kNbrWarps][kNbrSort];
    __shared__ NbrScan scan[kNbrWarps];
    const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kNbrWarps + wi;
    if (i >= n) return;
    const int p0 = offsets[i], p1 = offsets[i + 1], np = p1 - p0;
    if (p1 > cap) {
        if (lane == 0) atomicOr(err, 1);
        return;
    }
    const bool local = np <= kNbrSort;
    int w = 0;  // pairs found so far
    int no_sure = 0;
    warp_candidates<false>(i, lane, cart, cart32, atom_cfg, atom_bin, geo, bin_start, bin_atoms, scan[wi],
                    [&](bool hit, int j, int code, const double *v, double r2) {
                        const unsigned m = __ballot_sync(0xffffffffu, hit);
                        if (hit) {
                            const int pos = w + __popc(m & ((1u << lane) - 1u));
                            if (pos < np) {
                                const long long key = pair_key(j, code);
                                const D4 d{v[0], v[1], v[2], sqrt64(r2)};
                                if (local) {
                                    skey[wi][pos] = key;
                                    svec[wi][pos] = d;
                                } else {
                                    keys[p0 + pos] = key;
                                    vec64[p0 + pos] = d;
                                }
                            }
                        }
                        w += __popc(m);
                    },
                    no_sure);
    if (w != np) {
        if (lane == 0) atomicOr(err, 2);
        return;
    }
    if (local) {
        __syncwarp();
        for (int e = lane; e < np; e += 32) {
            const long long k = skey[wi][e];
            int rank = 0, e2 = 0;
            for (; e2 + 2 <= np; e2 += 2) {  // two keys per 16-byte load
                const longlong2 k2 = *reinterpret_cast<const longlong2 *>(&skey[wi][e2]);
                rank += (k2.x < k ? 1 : 0) + (k2.y < k ? 1 : 0);
            }
            if (e2 < np) rank += skey[wi][e2] < k ? 1 : 0;
            const D4 d = svec[wi][e];
            keys[p0 + rank] = k;
            vec64[p0 + rank] = d;
            pair_i[p0 + rank] = i;
            nbr_j[p0 + rank] = (int)(k >> 24);
            vec32[p0 + rank] = make_float4((float)d.x, (float)d.y, (float)d.z, (float)d.w);
        }
        return;
    }
    __syncwarp();
    if (lane == 0) {
        for (int a = p0 + 1; a < p1; ++a) {
            const long long k = keys[a];
            const D4 v = vec64[a];
            int bq = a - 1;
            while (bq >= p0 && keys[bq] > k) {
                keys[bq + 1] = keys[bq];
                vec64[bq + 1] = vec64[bq];
                --bq;
            }
            keys[bq + 1] = k;
            vec64[bq + 1] = v;
        }
    }
    __syncwarp();
    for (int a = p0 + lane; a < p1; a += 32) {
        pair_i[a] = i;
        nbr_j[a] = (int)(keys[a] >> 24);
        const D4 v = vec64[a];
        vec32[a] = make_float4((float)v.x, (float)v.y, (float)v.z, (float)v.w);
    }
}

__global__ void k_reverse(int n, const int *__restrict__ offsets, const long long *__restrict__ keys,
                          int *__restrict__ rev, int *__restrict__ err)
{
    int i = blockIdx.x;
    for (int p = offsets[i] + threadIdx.x; p < offsets[i + 1]; p += blockDim.x) {
        long long k = keys[p];
        int j = (int)(k >> 24);
        int sx = (int)((k >> 16) & 255) - kShiftBias, sy = (int)((k >> 8) & 255) - kShiftBias,
            sz = (int)(k & 255) - kShiftBias;
        long long want = pair_key(i, shift_code(-sx, -sy, -sz));
        int lo = offsets[j], hi = offsets[j + 1] - 1, found = -1;
        while (lo <= hi) {
            int mid = (lo + hi) >> 1;
            long long km = keys[mid];
            if (km == want) { found = mid; break; }
            if (km < want) lo = mid + 1;
            else hi = mid - 1;
        }
        rev[p] = found;
        if (found < 0) atomicOr(err, 4);
    }
}

// ------------------------------------------------- exclusive scan of ints
constexpr int kScanOne = 8192, kScanTile = 4096;  // ints of the one-block form; per block else

// Sums of kScanTile ints each.
__global__ void __launch_bounds__(1024) k_scan_sums(const int *__restrict__ in, int n, int *__restrict__ sums)
{
    __shared__ int warp_tot[32];
    int v = 0, total;
#pragma unroll
    for (int k = 0; k < kScanTile / 1024; ++k) {
        const int i = blockIdx.x * kScanTile + k * 1024 + threadIdx.x;
        if (i < n) v += in[i];
    }
    block_prefix(v, warp_tot, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// out[0 .. n] of a block's `per` ints (a thread takes consecutive ones), after
// the sums of the blocks before it (sums == NULL: one block).  With a cap
// (graph mode): a total beyond it empties every list (out = 0), so that no
// later kernel reads past the pair arrays, and sets err bit 0.
__global__ void __launch_bounds__(1024)
k_scan_out(const int *__restrict__ in, int n, int per, const int *__restrict__ sums, int *__restrict__ out,
           int *__restrict__ total_out, ScanCap cap)
{
    __shared__ int warp_tot[32];
    int base = 0, grand = 0;
    if (sums) {
        int before = 0, all = 0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += 1024) {
            const int s = sums[b];
            all += s;
            if (b < (int)blockIdx.x) before += s;
        }
        block_prefix(before, warp_tot, &base);
        block_prefix(all, warp_tot, &grand);
    }
    const int items = per / 1024, i0 = blockIdx.x * per + threadIdx.x * items;
    int v = 0, total;
    for (int k = 0; k < items; ++k)
        if (i0 + k < n) v += in[i0 + k];
    int at = base + block_prefix(v, warp_tot, &total);
    if (!sums) grand = total;
    const bool over = cap.used && grand > cap.cap;
    for (int k = 0; k < items; ++k)
        if (i0 + k < n) {
            const int x = in[i0 + k];
            out[i0 + k] = over ? 0 : at;
            at += x;
        }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        out[n] = over ? 0 : grand;
        if (total_out) *total_out = grand;
        if (cap.used) {
            *cap.used = over ? 0 : grand;
            if (over) atomicOr(cap.err, 1);
        }
    }
}

}  // namespace

// Exclusive scan of n ints into out[0..n] (out[n] = total): one launch up to
// 8192 ints (the scans of a small step were six launches), else two, the
// blocks of the second adding up the sums of those before them.
gap_status gap_scan(const int *in, int n, int *out, int *tmp, int *total, cudaStream_t st, ScanCap cap)
{
    if (n <= kScanOne) {
        const int per = n <= 1024 ? 1024 : (n + 1023) / 1024 * 1024;
        gap_count_launch();
        k_scan_out<<<1, 1024, 0, st>>>(in, n, per, nullptr, out, total, cap);
        return gap_cuda_status(cudaGetLastError(), "k_scan_out");
    }
    const int nb = (int)(((long)n + kScanTile - 1) / kScanTile);
    gap_count_launch();
    k_scan_sums<<<nb, 1024, 0, st>>>(in, n, tmp);
    GAP_TRY_CUDA(cudaGetLastError());
    gap_count_launch();
    k_scan_out<<<nb, 1024, 0, st>>>(in, n, kScanTile, tmp, out, total, cap);
    return gap_cuda_status(cudaGetLastError(), "k_scan_out");
}

size_t gap_scan_tmp_ints(int n) { return n > 0 ? ((size_t)n + kScanTile - 1) / kScanTile + 4 : 4; }

// The cell geometries' part of the device buffer they share with the offsets.
static size_t geo_bytes(int n_configs) { return (sizeof(CellGeom) * (size_t)(n_configs + 1) + 255) / 256 * 256; }

// Host-side geometry of each configuration's bin grid.
gap_status gap_cell_geometry(const gap_batch *b, double rc, std::vector<CellGeom> &geo, int &n_bins)
{
    geo.resize(b->n_configs);
    n_bins = 0;
    for (int c = 0; c < b->n_configs; ++c) {
        CellGeom &g = geo[c];
        const double *m = b->cell + 9 * c;
        double det = m[0] * (m[4] * m[8] - m[5] * m[7]) - m[1] * (m[3] * m[8] - m[5] * m[6]) +
                     m[2] * (m[3] * m[7] - m[4] * m[6]);
        if (!(std::fabs(det) > 1e-12)) {
            gap_set_error("cell of configuration " + std::to_string(c) + " is singular");
            return GAP_EINVAL;
        }
        double inv[9] = {(m[4] * m[8] - m[5] * m[7]) / det, (m[2] * m[7] - m[1] * m[8]) / det,
                         (m[1] * m[5] - m[2] * m[4]) / det, (m[5] * m[6] - m[3] * m[8]) / det,
                         (m[0] * m[8] - m[2] * m[6]) / det, (m[2] * m[3] - m[0] * m[5]) / det,
                         (m[3] * m[7] - m[4] * m[6]) / det, (m[1] * m[6] - m[0] * m[7]) / det,
                         (m[0] * m[4] - m[1] * m[3]) / det};
        long long nbins = 1;
        for (int k = 0; k < 3; ++k) {
            double width = 1.0 / std::sqrt(inv[k] * inv[k] + inv[3 + k] * inv[3 + k] + inv[6 + k] * inv[6 + k]);
            int nb = (int)std::floor(width / rc);
            if (nb < 1) nb = 1;
            if (nb > 1024) nb = 1024;
            int R = (int)std::ceil(rc * nb / width - 1e-12);
            if (R < 1) R = 1;
            g.pbc[k] = b->pbc[3 * c + k] ? 1 : 0;
            if (g.pbc[k] && R > 60) {
                gap_set_error("cell of configuration " + std::to_string(c) + " is too thin for the cutoff");
                return GAP_EINVAL;
            }
            g.nb[k] = nb;
            g.R[k] = R;
            nbins *= nb;
        }
        for (int k = 0; k < 9; ++k) {
            g.cell[k] = m[k];
            g.inv[k] = inv[k];
        }
        g.rc2 = rc * rc;
        // FP32 coordinates and shifts carry ~6e-8 of their size, up to 60 cell
        // edges, per component: a bound above that error
        double span = 0.0;
        for (int k = 0; k < 3; ++k) span += std::sqrt(m[3 * k] * m[3 * k] + m[3 * k + 1] * m[3 * k + 1] + m[3 * k + 2] * m[3 * k + 2]);
        const double rl = rc * (1.0 + 5e-4) + 3e-5 * span, rt = rc * (1.0 - 5e-4) - 3e-5 * span;
        g.rc2_loose = (float)(rl * rl);
        g.rc2_tight = rt > 0.0 ? (float)(rt * rt) : 0.f;
        g.bin0 = n_bins;
        if ((long long)n_bins + nbins > (1LL << 30)) {
            gap_set_error("too many neighbour bins");
            return GAP_EINVAL;
        }
        n_bins += (int)nbins;
    }
    return GAP_OK;
}

// Most pairs a build makes room for without waiting for their number: 2^20,
// about 100 MB of pair arrays.  The wait costs ~20 us, 1% of a call with that
// many pairs (1.5 ms and more); beyond, a workspace that once met a dense cell
// would hold its density times the atoms of a large sparse one.
constexpr int kAheadPairs = 1 << 20;
// Most geometry a handle keeps pinned: about 80 thousand configurations.
constexpr size_t kMaxStage = 16 << 20;

gap_status gap_neighbours(NbrWork &w, const gap_batch *b, const double *d_pos, const int *d_species, int S, double rc,
                          int *words, int *host, bool ahead, cudaStream_t st)
{
    int n = b->n_atoms;
    std::vector<CellGeom> geo;
    int n_bins = 0;
    GAP_TRY(gap_cell_geometry(b, rc, geo, n_bins));
    GAP_TRY(w.reserve_atoms(n, b->n_configs, n_bins));
    int *err = words;
    w.err = words + kNbrErr;
    w.total = words + kNbrTotal;
    w.n_atoms = n;
    if (!w.graph) {
        // geometry and offsets in one copy from pinned memory, or, beyond what a
        // handle should keep pinned (or where none is to be had), in two from
        // the host's own, which wait for the stream
        const size_t og = geo_bytes(b->n_configs), bytes = og + sizeof(int) * (b->n_configs + 1);
        if (w.in_flight) {  // an earlier call ended in an error before it synchronised
            GAP_TRY_CUDA(cudaDeviceSynchronize());
            w.in_flight = false;
        }
        if (bytes > w.cap_stage && bytes <= kMaxStage) {
            if (w.stage) cudaFreeHost(w.stage);
            w.stage = nullptr;
            w.cap_stage = 0;
            if (cudaMallocHost(&w.stage, bytes + bytes / 4) == cudaSuccess) {
                w.cap_stage = bytes + bytes / 4;
            } else {
                cudaGetLastError();
                w.stage = nullptr;
            }
        }
        if (bytes <= w.cap_stage) {
            if (!geo.empty()) std::memcpy(w.stage, geo.data(), sizeof(CellGeom) * geo.size());
            if (b->n_configs > 0)
                std::memcpy(static_cast<char *>(w.stage) + og, b->config_offsets, sizeof(int) * (b->n_configs + 1));
            GAP_TRY_CUDA(cudaMemcpyAsync(w.geo, w.stage, bytes, cudaMemcpyHostToDevice, st));
            w.in_flight = true;
        } else if (b->n_configs > 0) {
            GAP_TRY_CUDA(cudaMemcpyAsync(w.geo, geo.data(), sizeof(CellGeom) * geo.size(), cudaMemcpyHostToDevice, st));
            GAP_TRY_CUDA(cudaMemcpyAsync(w.cfg_offsets, b->config_offsets, sizeof(int) * (b->n_configs + 1),
                                         cudaMemcpyHostToDevice, st));
        }
    }
    const BinInputs in{n, b->n_configs, S, d_pos, d_species, w.cfg_offsets, w.geo, err};
    if (n > 0 && n <= kSmallAtoms && n_bins <= kSmallBins) {
        gap_count_launch();
        k_bin_small<<<1, 1024, 0, st>>>(in, n_bins, w.cart, w.cart32, w.atom_cfg, w.atom_bin, w.bin_start, w.bin_atoms);
        GAP_TRY_CUDA(cudaGetLastError());
    } else if (n > 0) {
        const int T = 128, gridN = (n + T - 1) / T;
        GAP_TRY_CUDA(cudaMemsetAsync(w.bin_count, 0, sizeof(int) * (n_bins + 1), st));
        gap_count_launch();
        k_bin<<<gridN, T, 0, st>>>(in, w.cart, w.cart32, w.atom_cfg, w.atom_bin, w.bin_count);
        GAP_TRY_CUDA(cudaGetLastError());
        GAP_TRY(gap_scan(w.bin_count, n_bins, w.bin_start, w.scan_tmp, nullptr, st));
        gap_count_launch();
        k_scatter<<<gridN, T, 0, st>>>(n, w.atom_bin, w.bin_start, w.bin_count, w.bin_atoms);
        GAP_TRY_CUDA(cudaGetLastError());
    }
    if (n > 0) {
        gap_count_launch();
        const int gridW = (n + kNbrWarps - 1) / kNbrWarps;
        k_count_warp<<<gridW, 32 * kNbrWarps, 0, st>>>(n, w.cart, w.cart32, w.atom_cfg, w.atom_bin, w.geo,
                                                       w.bin_start, w.bin_atoms, w.counts);
        GAP_TRY_CUDA(cudaGetLastError());
    }
    // room for the pairs: a capacity, or (after a wait) their number
    ahead = ahead && !w.graph && w.pairs_per_atom > 0.0;
    const double room = std::ceil(1.05 * w.pairs_per_atom * n) + 64.0;
    if (room > (double)kAheadPairs) ahead = false;
    int P = w.graph ? w.pair_cap : ahead ? (int)room : 0;
    const bool capped = w.graph || ahead;
    GAP_TRY(gap_scan(w.counts, n, w.pairs.offsets, w.scan_tmp, w.total, st,
                     capped ? ScanCap{P, w.total + 1, w.err} : ScanCap{}));
    w.pairs.count = capped ? w.total + 1 : w.total;
    if (!capped) {
        GAP_TRY_CUDA(cudaMemcpyAsync(host, words, sizeof(int) * kWords, cudaMemcpyDeviceToHost, st));
        GAP_TRY_CUDA(cudaStreamSynchronize(st));
        w.in_flight = false;
        P = host[kNbrTotal];
    }
    GAP_TRY(w.reserve_pairs(P));
    w.pairs.n_pairs = P;
    if (n > 0) {
        gap_count_launch();
        k_fill_warp<<<(n + kNbrWarps - 1) / kNbrWarps, 32 * kNbrWarps, 0, st>>>(
            n, w.cart, w.cart32, w.atom_cfg, w.atom_bin, w.geo, w.bin_start, w.bin_atoms, w.pairs.offsets, P, w.keys,
            w.pairs.i, w.pairs.j, w.pairs.vec64, w.pairs.vec32, w.err);
        GAP_TRY_CUDA(cudaGetLastError());
        gap_count_launch();
        k_reverse<<<n, 64, 0, st>>>(n, w.pairs.offsets, w.keys, w.pairs.rev, w.err);
        GAP_TRY_CUDA(cudaGetLastError());
    }
    return GAP_OK;
}

gap_status gap_neighbours_done(NbrWork &w, const int *host)
{
    const int e = host[kNbrErr];
    w.in_flight = false;
    if (w.n_atoms > 0) {
        const double ppa = (double)host[kNbrTotal] / w.n_atoms;
        if (ppa > w.pairs_per_atom) w.pairs_per_atom = ppa;
    }
    if (e & 1) {  // without a graph the caller runs the call again, and sets an error if that fails
        if (w.graph)
            gap_set_error("more neighbour pairs than the pair capacity (" + std::to_string(w.pair_cap) +
                          ") of the captured step");
        return GAP_ECAPACITY;
    }
    if (e) {
        gap_set_error("neighbour list inconsistency (code " + std::to_string(e) + ")");
        return GAP_ECUDA;
    }
    return GAP_OK;
}

// ------------------------------------------------------------ workspace
static gap_status grow(void **p, size_t &cap, size_t bytes)
{
    if (bytes <= cap && *p) return GAP_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    cap = 0;
    size_t b = bytes + bytes / 4 + 256;
    cudaError_t e = gap_dev_malloc(p, b);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();  // the caller may go on with a smaller request
        gap_set_error(std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
        return GAP_ENOMEM;
    }
    cap = b;
    return GAP_OK;
}

gap_status NbrWork::reserve_atoms(int n, int n_configs, int n_bins)
{
    GAP_TRY(grow((void **)&geo, cap_geo, geo_bytes(n_configs) + sizeof(int) * (n_configs + 2)));
    cfg_offsets = reinterpret_cast<int *>(reinterpret_cast<char *>(geo) + geo_bytes(n_configs));
    GAP_TRY(grow((void **)&cart, cap_cart, sizeof(D4) * (size_t)(n + 1)));
    GAP_TRY(grow((void **)&cart32, cap_c32, sizeof(float4) * (size_t)(n + 1)));
    GAP_TRY(grow((void **)&atom_cfg, cap_acfg, sizeof(int) * (size_t)(n + 1)));
    GAP_TRY(grow((void **)&atom_bin, cap_abin, sizeof(int) * (size_t)(n + 1)));
    GAP_TRY(grow((void **)&bin_atoms, cap_batoms, sizeof(int) * (size_t)(n + 1)));
    GAP_TRY(grow((void **)&counts, cap_counts, sizeof(int) * (size_t)(n + 1)));
    GAP_TRY(grow((void **)&pairs.offsets, cap_offsets, sizeof(int) * (size_t)(n + 2)));
    GAP_TRY(grow((void **)&bin_count, cap_bcount, sizeof(int) * (size_t)(n_bins + 2)));
    GAP_TRY(grow((void **)&bin_start, cap_bstart, sizeof(int) * (size_t)(n_bins + 2)));
    size_t t = gap_scan_tmp_ints(n > n_bins ? n : n_bins);
    GAP_TRY(grow((void **)&scan_tmp, cap_scan, sizeof(int) * t));
    return GAP_OK;
}

gap_status NbrWork::reserve_pairs(int P)
{
    size_t p = (size_t)(P > 0 ? P : 1);
    GAP_TRY(grow((void **)&keys, cap_keys, sizeof(long long) * p));
    GAP_TRY(grow((void **)&pairs.i, cap_i, sizeof(int) * p));
    GAP_TRY(grow((void **)&pairs.j, cap_j, sizeof(int) * p));
    GAP_TRY(grow((void **)&pairs.rev, cap_rev, sizeof(int) * p));
    GAP_TRY(grow((void **)&pairs.vec64, cap_v64, sizeof(D4) * p));
    GAP_TRY(grow((void **)&pairs.vec32, cap_v32, sizeof(float4) * p));
    return GAP_OK;
}

void NbrWork::release()
{
    if (stage) cudaFreeHost(stage);
    void *ps[] = {geo, cart, cart32, atom_cfg, atom_bin, bin_atoms, counts, pairs.offsets, bin_count,
                  bin_start, scan_tmp, keys, pairs.i, pairs.j, pairs.rev, pairs.vec64, pairs.vec32};
    for (void *p : ps)
        if (p) cudaFree(p);
    *this = NbrWork();
}
