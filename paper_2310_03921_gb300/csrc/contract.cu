// Kernel contraction of the sparse GP (Eqs. 2, 3 and 13): for the atoms of one
// central species and that species' M sparse points,
//   q_im = p_hat_i . x_m,   eps_i = delta^2 sum_m alpha_m q_im^zeta,
//   g_i  = d eps_i / d p_hat_i = sum_m W_im x_m,  W_im = zeta delta^2 alpha_m q_im^(zeta-1).
// Two SIMT (CUDA-core) GEMMs, templated on the arithmetic type: the plain
// FP64 path and an FP32 variant.  The tensor-core form lives in tc_gemm.cu;
// this file also holds its operand preparation (centring on the mean sparse
// point mu: a_i = p_hat_i - mu, b_m = x_m - mu, q = a.b + a.mu + x_m.mu, and the
// BF16 hi/lo split) and the per-atom finalisation of both forms.
#include <vector>

#include "contract.h"

namespace {

constexpr int TM = 64, TN = 64, TK = 16;

// W[r][m] and per-(row, column tile) partial energies.
template <typename T>
__global__ void __launch_bounds__(256)
k_simt_qW(const T *__restrict__ phat, int D, const int *__restrict__ rows, const int *__restrict__ nrows_p,
          const T *__restrict__ X, const T *__restrict__ alpha, int M, T d2, int zeta, T *__restrict__ W, int ldw,
          double *__restrict__ eps_part, int n_tiles)
{
    __shared__ T As[TK][TM + 1], Bs[TK][TN + 1];
    const int nrows = *nrows_p;
    const int r0 = blockIdx.y * TM, m0 = blockIdx.x * TN;
    if (r0 >= nrows) return;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T acc[4][4] = {};
    for (int k0 = 0; k0 < D; k0 += TK) {
        for (int e = threadIdx.x; e < TK * TM; e += 256) {
            int kk = e % TK, rr = e / TK;
            int r = r0 + rr, k = k0 + kk;
            As[kk][rr] = (r < nrows && k < D) ? phat[(size_t)rows[r] * D + k] : T(0);
            int m = m0 + rr;
            Bs[kk][rr] = (m < M && k < D) ? X[(size_t)m * D + k] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            T a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { a[u] = As[kk][ty * 4 + u]; b[u] = Bs[kk][tx * 4 + u]; }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] += a[u] * b[v];
        }
        __syncthreads();
    }
    __shared__ double red[TM][17];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        int r = r0 + ty * 4 + u;
        double e = 0.0;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            int m = m0 + tx * 4 + v;
            if (r < nrows && m < M) {
                T q = acc[u][v], qz = T(1);
                for (int z = 1; z < zeta; ++z) qz *= q;
                T a = d2 * alpha[m];
                e += (double)(a * qz * q);
                W[(size_t)r * ldw + m] = T(zeta) * a * qz;
            }
        }
        red[ty * 4 + u][tx] = e;
    }
    __syncthreads();
    if (threadIdx.x < TM) {
        int r = r0 + threadIdx.x;
        double e = 0.0;
        for (int t = 0; t < 16; ++t) e += red[threadIdx.x][t];
        if (r < nrows) eps_part[(size_t)r * n_tiles + blockIdx.x] = e;
    }
}

// g[rows[r]][d] = sum_m W[r][m] X[m][d]
template <typename T>
__global__ void __launch_bounds__(256)
k_simt_G(const T *__restrict__ W, int ldw, const int *__restrict__ rows, const int *__restrict__ nrows_p,
         const T *__restrict__ X, int M, int D, T *__restrict__ g, int ldg)
{
    __shared__ T As[TK][TM + 1], Bs[TK][TN + 1];
    const int nrows = *nrows_p;
    const int r0 = blockIdx.y * TM, d0 = blockIdx.x * TN;
    if (r0 >= nrows) return;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T acc[4][4] = {};
    for (int k0 = 0; k0 < M; k0 += TK) {
        for (int e = threadIdx.x; e < TK * TM; e += 256) {
            int kk = e % TK, rr = e / TK;
            int r = r0 + rr, k = k0 + kk;
            As[kk][rr] = (r < nrows && k < M) ? W[(size_t)r * ldw + k] : T(0);
            int kb = e / TN, dd = e % TN;
            int d = d0 + dd, m = k0 + kb;
            Bs[kb][dd] = (m < M && d < D) ? X[(size_t)m * D + d] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            T a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { a[u] = As[kk][ty * 4 + u]; b[u] = Bs[kk][tx * 4 + u]; }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] += a[u] * b[v];
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        int r = r0 + ty * 4 + u;
        if (r >= nrows) continue;
        int atom = rows[r];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            int d = d0 + tx * 4 + v;
            if (d < D) g[(size_t)atom * ldg + d] = acc[u][v];
        }
    }
}

// eps of each row from its column tiles' partial energies: a warp per row.
__global__ void __launch_bounds__(128)
k_eps_rows(const int *__restrict__ rows, const int *__restrict__ nrows_p, const double *__restrict__ eps_part,
           int n_tiles, double *__restrict__ eps)
{
    const int r = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= *nrows_p) return;
    double e = 0.0;
    for (int t = lane; t < n_tiles; t += 32) e += eps_part[(size_t)r * n_tiles + t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) eps[rows[r]] = e;
}

// ------------------------------------------------ the same on small tiles
// 8 x 8 outputs per block, the K sum split four ways over its 256 threads and
// the four partial sums added in a fixed order.  The 64 x 64 tiles above keep
// a small product on few SMs (64 atoms x 100 points: two blocks, a serial
// chain over K of 134 us); these spread it over R M / 64 blocks.  In FP64
// they are the better tile at every size: GB300's FP64 pipe holds a warp
// instruction for ~64 cycles, which covers two shared-memory reads and the
// tile loads per FMA.  In FP32 the reads bound them, so they serve only
// products whose 64 x 64 tiles would leave most SMs idle (small_tiles).
// Whole predictions with 64 x 64 and 8 x 8 tiles, n_max 8, l_max 6: FP64 215
// atoms x 4000 points 5371 and 1216 us, 4095 x 2000 9089 and 8392 us; FP32 215
// x 4000 (252 tiles and 16) 905 and 461 us.  One FP32 product by its number of
// 64 x 64 tiles, 64 x 64 and 8 x 8, inner size 252: 8 tiles 41 and 10 us, 32
// tiles 43 and 17, 64 tiles 43 and 31, 96 tiles 43 and 32, 128 tiles 43 and
// 52, 512 tiles 73 and 177; inner size 2000: 4 tiles 276 and 27, 32 tiles 278
// and 103, 64 tiles 277 and 183, 108 tiles 281 and 300.  They cross near 100
// tiles whatever the inner size; the line lies at 48, well on the side where
// the small tiles win.
constexpr int kST = 8, kSK = 64, kSplit = 4;

// acc = sum over this thread's quarter of K of A(r, k) B(k, c); load(e, kk, rr)
// fills the staged operands.
template <typename T, typename LoadA, typename LoadB>
__device__ __forceinline__ T small_tile_sum(int K, T (&As)[kSK][kST + 1], T (&Bs)[kSK][kST + 1],
                                            T (&red)[kSplit][kST * kST], LoadA &&la, LoadB &&lb)
{
    const int cell = threadIdx.x & 63, split = threadIdx.x >> 6, r = cell >> 3, c = cell & 7;
    T acc = T(0);
    for (int k0 = 0; k0 < K; k0 += kSK) {
#pragma unroll
        for (int u = 0; u < kSK * kST / 256; ++u) {
            la(k0, (int)threadIdx.x + 256 * u);
            lb(k0, (int)threadIdx.x + 256 * u);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kSK / kSplit; ++kk) acc += As[split * (kSK / kSplit) + kk][r] * Bs[split * (kSK / kSplit) + kk][c];
        __syncthreads();
    }
    red[split][cell] = acc;
    __syncthreads();
    return (red[0][cell] + red[1][cell]) + (red[2][cell] + red[3][cell]);
}

template <typename T>
__global__ void __launch_bounds__(256)
k_small_qW(const T *__restrict__ phat, int D, const int *__restrict__ rows, const int *__restrict__ nrows_p,
           const T *__restrict__ X, const T *__restrict__ alpha, int M, T d2, int zeta, T *__restrict__ W, int ldw,
           double *__restrict__ eps_part, int n_tiles)
{
    __shared__ T As[kSK][kST + 1], Bs[kSK][kST + 1];
    __shared__ T red[kSplit][kST * kST];
    __shared__ int atom[kST];
    const int nrows = *nrows_p;
    const int r0 = blockIdx.y * kST, m0 = blockIdx.x * kST;
    if (r0 >= nrows) return;
    if (threadIdx.x < kST) atom[threadIdx.x] = r0 + (int)threadIdx.x < nrows ? rows[r0 + threadIdx.x] : -1;
    __syncthreads();
    const T q = small_tile_sum<T>(
        D, As, Bs, red,
        [&](int k0, int e) {
            const int kk = e % kSK, rr = e / kSK, k = k0 + kk;
            As[kk][rr] = (atom[rr] >= 0 && k < D) ? phat[(size_t)atom[rr] * D + k] : T(0);
        },
        [&](int k0, int e) {
            const int kk = e % kSK, rr = e / kSK, k = k0 + kk, m = m0 + rr;
            Bs[kk][rr] = (m < M && k < D) ? X[(size_t)m * D + k] : T(0);
        });
    if (threadIdx.x >= kST * kST) return;
    const int r = r0 + (threadIdx.x >> 3), m = m0 + (threadIdx.x & 7);
    double e = 0.0;
    if (r < nrows && m < M) {
        T qz = T(1);
        for (int z = 1; z < zeta; ++z) qz *= q;
        const T a = d2 * alpha[m];
        e = (double)(a * qz * q);
        W[(size_t)r * ldw + m] = T(zeta) * a * qz;
    }
#pragma unroll
    for (int o = kST / 2; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 7) == 0 && r < nrows) eps_part[(size_t)r * n_tiles + blockIdx.x] = e;
}

template <typename T>
__global__ void __launch_bounds__(256)
k_small_G(const T *__restrict__ W, int ldw, const int *__restrict__ rows, const int *__restrict__ nrows_p,
          const T *__restrict__ X, int M, int D, T *__restrict__ g, int ldg)
{
    __shared__ T As[kSK][kST + 1], Bs[kSK][kST + 1];
    __shared__ T red[kSplit][kST * kST];
    const int nrows = *nrows_p;
    const int r0 = blockIdx.y * kST, d0 = blockIdx.x * kST;
    if (r0 >= nrows) return;
    const T v = small_tile_sum<T>(
        M, As, Bs, red,
        [&](int k0, int e) {
            const int kk = e % kSK, rr = e / kSK, k = k0 + kk;
            As[kk][rr] = (r0 + rr < nrows && k < M) ? W[(size_t)(r0 + rr) * ldw + k] : T(0);
        },
        [&](int k0, int e) {
            const int dd = e % kST, kk = e / kST, k = k0 + kk;
            Bs[kk][dd] = (k < M && d0 + dd < D) ? X[(size_t)k * D + d0 + dd] : T(0);
        });
    if (threadIdx.x >= kST * kST) return;
    const int r = r0 + (threadIdx.x >> 3), d = d0 + (threadIdx.x & 7);
    if (r < nrows && d < D) g[(size_t)rows[r] * ldg + d] = v;
}

// Whether the small tiles serve a product of rows x cols outputs.
template <typename T> bool small_tiles(int rows, int cols)
{
    if (sizeof(T) == 8) return (rows + kST - 1) / kST <= 65535;  // grid y
    return (long)((rows + TM - 1) / TM) * ((cols + TN - 1) / TN) <= 48;
}

// ---------------------------------------------------------------- rows
constexpr int kRowsOne = 8192, kRowsTile = 1024;  // atoms of the one-block form; per block else
constexpr int kMaxGPs = 8;

// Atoms of each GP (species below n_gp) in kRowsTile consecutive atoms.  one:
// a single species; the host takes its count as n without reading it back, so
// every atom has a row whatever its species says (a wrong one fails the call).
__global__ void __launch_bounds__(kRowsTile)
k_gp_counts(int n, int n_gp, bool one, const int *__restrict__ species, int *__restrict__ block_counts)
{
    __shared__ int cnt[kMaxGPs];
    if (threadIdx.x < kMaxGPs) cnt[threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * kRowsTile + threadIdx.x;
    const int z = i < n ? (one ? 0 : species[i]) : -1;
    for (int s = 0; s < n_gp; ++s) {
        const unsigned m = __ballot_sync(0xffffffffu, z == s);
        if ((threadIdx.x & 31) == 0 && m) atomicAdd(&cnt[s], __popc(m));
    }
    __syncthreads();
    if (threadIdx.x < n_gp) block_counts[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = cnt[threadIdx.x];
}

// rows[s][.] = the atoms of GP s in index order, rank = an atom's place among
// them, gp_of_atom (-1 without a GP), counts[s].  One block over all atoms
// (block_counts NULL, tiles in turn), or a block per tile after
// k_gp_counts, whose counts of the tiles before it each block adds up.  One
// or two launches for all GPs; a flag, scan and compaction per GP were six.
__global__ void __launch_bounds__(kRowsTile)
k_gp_rows(int n, int n_gp, bool one, const int *__restrict__ species, const int *__restrict__ block_counts,
          int *__restrict__ rows, int *__restrict__ counts, int *__restrict__ gp_of_atom, int *__restrict__ rank)
{
    __shared__ int wcnt[kMaxGPs][33], base[kMaxGPs];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // base[s]: GP s's rows before this block; one writer per entry before the barrier
    if (block_counts) {
        if (w < n_gp) {
            int sum = 0, all = 0;
            for (int b = lane; b < (int)gridDim.x; b += 32) {
                const int c = block_counts[(size_t)w * gridDim.x + b];
                all += c;
                if (b < (int)blockIdx.x) sum += c;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sum += __shfl_xor_sync(0xffffffffu, sum, o);
                all += __shfl_xor_sync(0xffffffffu, all, o);
            }
            if (lane == 0) {
                base[w] = sum;
                if (blockIdx.x == 0) counts[w] = all;
            }
        }
    } else if (threadIdx.x < kMaxGPs) {
        base[threadIdx.x] = 0;
    }
    __syncthreads();
    const int t0 = block_counts ? blockIdx.x : 0, t1 = block_counts ? blockIdx.x + 1 : (n + kRowsTile - 1) / kRowsTile;
    for (int t = t0; t < t1; ++t) {
        const int i = t * kRowsTile + threadIdx.x;
        const int z = i < n ? (one ? 0 : species[i]) : -1;
        int before = 0;
        for (int s = 0; s < n_gp; ++s) {
            const unsigned m = __ballot_sync(0xffffffffu, z == s);
            if (lane == 0) wcnt[s][w] = __popc(m);
            if (z == s) before = __popc(m & ((1u << lane) - 1u));
        }
        __syncthreads();
        if (w < n_gp) {  // exclusive prefix over the 32 warps
            const int c = wcnt[w][lane];
            int x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            wcnt[w][lane] = base[w] + x - c;
            if (lane == 31) wcnt[w][32] = base[w] + x;
        }
        __syncthreads();
        if (i < n) {
            const bool in = z >= 0 && z < n_gp;
            gp_of_atom[i] = in ? z : -1;
            if (in) {
                const int r = wcnt[z][w] + before;
                rows[(size_t)z * n + r] = i;
                rank[i] = r;
            }
        }
        __syncthreads();
        if (threadIdx.x < n_gp) base[threadIdx.x] = wcnt[threadIdx.x][32];
        __syncthreads();
    }
    if (!block_counts && threadIdx.x < n_gp) counts[threadIdx.x] = base[threadIdx.x];
}

// -------------------------------------------------- tensor-core operands
// a = p_hat - mu split into BF16 hi + lo (columns D..ld-1 zero); t = a . mu.
__global__ void k_split_rows(const float *__restrict__ phat, int D, int ld, const int *__restrict__ rows, int nrows,
                             const float *__restrict__ mu, __nv_bfloat16 *__restrict__ Ahi,
                             __nv_bfloat16 *__restrict__ Alo, __nv_bfloat16 *__restrict__ Amid,
                             float *__restrict__ t_row)
{
    int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    int lane = threadIdx.x & 31;
    if (r >= nrows) return;
    const float *p = phat + (size_t)rows[r] * D;
    float t = 0.f;
    for (int d = lane; d < ld; d += 32) {
        float a = d < D ? p[d] - mu[d] : 0.f;
        __nv_bfloat16 h = __float2bfloat16_rn(a);
        Ahi[(size_t)r * ld + d] = h;
        float rest = a - __bfloat162float(h);
        if (Amid) {
            __nv_bfloat16 m = __float2bfloat16_rn(rest);
            Amid[(size_t)r * ld + d] = m;
            rest -= __bfloat162float(m);
        }
        Alo[(size_t)r * ld + d] = __float2bfloat16_rn(rest);
        t += a * mu[d];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) t_row[r] = t;
}

// eps, wsum and g of the atoms of one GP from the tensor-core partials.
// LANES lanes per row: the column-tile partials of eps and sum_m W summed in
// FP64 (lanes over partials, then a fixed shuffle tree), and, where the
// gradient product ran in parts of K (g not NULL), their sum in order to the
// row's atom; else the product has written g itself (copying every row here
// made a call of 512 four-species boxes 3843 us, 3749 then).  The FP64 pipe
// bounds the sums (two instructions per partial and per shuffle, ~19 cycles
// each per SM): eight lanes per row halve them; a whole warp per row where a
// few rows have g to copy.  32768 rows x 32 partials: 35 us with a warp per
// row, 15 us with eight lanes.
template <int LANES>
__global__ void __launch_bounds__(128) k_tc_finalize(const int *__restrict__ rows, int nrows,
                                                     const float *__restrict__ eps_part,
                                                     const float *__restrict__ wsum_part, int n_part,
                                                     const float *__restrict__ Gs, int parts, int D16,
                                                     double *__restrict__ eps,
                                                     float *__restrict__ wsum, float *__restrict__ g)
{
    const int r = blockIdx.x * (128 / LANES) + threadIdx.x / LANES, lane = threadIdx.x % LANES;
    const bool in = r < nrows;
    double e = 0.0, w = 0.0;
    for (int t = in ? lane : n_part; t < n_part; t += LANES) {
        e += eps_part[(size_t)r * n_part + t];
        w += wsum_part[(size_t)r * n_part + t];
    }
#pragma unroll
    for (int o = LANES / 2; o; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        w += __shfl_xor_sync(0xffffffffu, w, o);
    }
    if (!in) return;
    const int atom = rows[r];
    if (lane == 0) {
        eps[atom] = e;
        wsum[atom] = (float)w;
    }
    if (g)
        for (int d = lane; d < D16; d += LANES) {
            float v = Gs[(size_t)r * D16 + d];
            for (int p = 1; p < parts; ++p) v += Gs[((size_t)p * nrows + r) * D16 + d];
            g[(size_t)atom * D16 + d] = v;
        }
}

gap_status tc_finalize(const int *rows, int nrows, const TcScratch &sc, int n_part, int parts, int D16, double *eps,
                       float *wsum, float *g, cudaStream_t st)
{
    gap_count_launch();
    if (g && parts > 1)
        k_tc_finalize<32><<<(nrows + 3) / 4, 128, 0, st>>>(rows, nrows, sc.eps_part, sc.wsum_part, n_part, sc.Gs, parts,
                                                           D16, eps, wsum, g);
    else
        k_tc_finalize<8><<<(nrows + 15) / 16, 128, 0, st>>>(rows, nrows, sc.eps_part, sc.wsum_part, n_part, nullptr, 1,
                                                            D16, eps, wsum, nullptr);
    return gap_cuda_status(cudaGetLastError(), "k_tc_finalize");
}

}  // namespace

template <typename T>
gap_status gap_contract_simt(const T *phat, int D, int D16, const int *rows, const int *nrows_dev, int max_rows,
                             const T *X, const T *alpha, int M, double delta, int zeta, T *W, double *eps_part,
                             T *g, double *eps, cudaStream_t st)
{
    if (max_rows <= 0 || M <= 0) return GAP_OK;
    const int n_tiles = gap_contract_simt_parts<T>(max_rows, M);
    gap_prof_begin(ST_GEMM_Q, st);
    gap_count_launch();
    if (small_tiles<T>(max_rows, M)) {
        k_small_qW<T><<<dim3(n_tiles, (max_rows + kST - 1) / kST), 256, 0, st>>>(
            phat, D, rows, nrows_dev, X, alpha, M, (T)(delta * delta), zeta, W, M, eps_part, n_tiles);
    } else {
        k_simt_qW<T><<<dim3(n_tiles, (max_rows + TM - 1) / TM), 256, 0, st>>>(
            phat, D, rows, nrows_dev, X, alpha, M, (T)(delta * delta), zeta, W, M, eps_part, n_tiles);
    }
    GAP_TRY_CUDA(cudaGetLastError());
    gap_prof_end(ST_GEMM_Q, st);
    gap_prof_begin(ST_GEMM_G, st);
    if (g) {
        gap_count_launch();
        if (small_tiles<T>(max_rows, D))
            k_small_G<T><<<dim3((D + kST - 1) / kST, (max_rows + kST - 1) / kST), 256, 0, st>>>(W, M, rows, nrows_dev,
                                                                                                X, M, D, g, D16);
        else
            k_simt_G<T><<<dim3((D + TN - 1) / TN, (max_rows + TM - 1) / TM), 256, 0, st>>>(W, M, rows, nrows_dev, X, M,
                                                                                           D, g, D16);
        GAP_TRY_CUDA(cudaGetLastError());
    }
    gap_count_launch();
    k_eps_rows<<<(max_rows + 3) / 4, 128, 0, st>>>(rows, nrows_dev, eps_part, n_tiles, eps);
    GAP_TRY_CUDA(cudaGetLastError());
    gap_prof_end(ST_GEMM_G, st);
    return GAP_OK;
}

template gap_status gap_contract_simt<double>(const double *, int, int, const int *, const int *, int, const double *,
                                              const double *, int, double, int, double *, double *, double *, double *,
                                              cudaStream_t);
template gap_status gap_contract_simt<float>(const float *, int, int, const int *, const int *, int, const float *,
                                             const float *, int, double, int, float *, double *, float *, double *,
                                             cudaStream_t);

int gap_contract_simt_tiles(int M) { return M > 0 ? (M + TN - 1) / TN : 0; }
template <typename T> int gap_contract_simt_parts(int rows, int M)
{
    const int tile = small_tiles<T>(rows, M) ? kST : TN;
    return M > 0 ? (M + tile - 1) / tile : 0;
}
template int gap_contract_simt_parts<double>(int, int);
template int gap_contract_simt_parts<float>(int, int);

// The same two GEMMs as gap_contract_simt<double> on the identity row list,
// launched without stage profiling (used by the allocation-free entry point).
gap_status gap_contract_simt_fixed(const double *phat, int D, int ldg, const int *rows, const int *nrows_dev,
                                   int n_rows, const double *X, const double *alpha, int M, double delta, int zeta,
                                   double *W, double *eps_part, double *g, double *eps, cudaStream_t st)
{
    if (n_rows <= 0 || M <= 0) return GAP_OK;
    const int n_tiles = gap_contract_simt_tiles(M);
    dim3 g1(n_tiles, (n_rows + TM - 1) / TM);
    gap_count_launch();
    k_simt_qW<double><<<g1, 256, 0, st>>>(phat, D, rows, nrows_dev, X, alpha, M, delta * delta, zeta, W, M,
                                           eps_part, n_tiles);
    GAP_TRY_CUDA(cudaGetLastError());
    dim3 g2((D + TN - 1) / TN, (n_rows + TM - 1) / TM);
    gap_count_launch();
    k_simt_G<double><<<g2, 256, 0, st>>>(W, M, rows, nrows_dev, X, M, D, g, ldg);
    GAP_TRY_CUDA(cudaGetLastError());
    gap_count_launch();
    k_eps_rows<<<(n_rows + 3) / 4, 128, 0, st>>>(rows, nrows_dev, eps_part, n_tiles, eps);
    return gap_cuda_status(cudaGetLastError(), "k_eps_rows");
}

gap_status gap_gp_rows(int n, int n_gp, bool one, const int *species, int *tmp, int *rows, int *counts,
                       int *gp_of_atom, int *rank, cudaStream_t st)
{
    if (n_gp > kMaxGPs) {
        gap_set_error("too many GPs");
        return GAP_EINVAL;
    }
    if (n == 0) {
        if (n_gp > 0) GAP_TRY_CUDA(cudaMemsetAsync(counts, 0, sizeof(int) * n_gp, st));
        return GAP_OK;
    }
    if (n <= kRowsOne) {
        gap_count_launch();
        k_gp_rows<<<1, kRowsTile, 0, st>>>(n, n_gp, one, species, nullptr, rows, counts, gp_of_atom, rank);
        return gap_cuda_status(cudaGetLastError(), "k_gp_rows");
    }
    const int nb = (n + kRowsTile - 1) / kRowsTile;
    gap_count_launch();
    k_gp_counts<<<nb, kRowsTile, 0, st>>>(n, n_gp, one, species, tmp);
    GAP_TRY_CUDA(cudaGetLastError());
    gap_count_launch();
    k_gp_rows<<<nb, kRowsTile, 0, st>>>(n, n_gp, one, species, tmp, rows, counts, gp_of_atom, rank);
    return gap_cuda_status(cudaGetLastError(), "k_gp_rows");
}

size_t gap_gp_rows_tmp_ints(int n, int n_gp)
{
    return ((size_t)n + kRowsTile - 1) / kRowsTile * (n_gp > 0 ? n_gp : 1) + 1;
}

gap_status gap_split_rows(const float *phat, int D, int D16, const int *rows, int nrows, const float *mu,
                          __nv_bfloat16 *Ahi, __nv_bfloat16 *Alo, __nv_bfloat16 *Amid, float *t_row, cudaStream_t st)
{
    if (nrows <= 0) return GAP_OK;
    gap_count_launch();
    k_split_rows<<<(nrows + 3) / 4, 128, 0, st>>>(phat, D, D16, rows, nrows, mu, Ahi, Alo, Amid, t_row);
    return gap_cuda_status(cudaGetLastError(), "k_split_rows");
}

int gap_contract_parts(const int *rows, const int *M_pad, int n, int D16, int nsplit, int q)
{
    if (n == 1 && gap_tc_variant_forced(nsplit)) return 1;  // the forced tile, not the split's own
    // column tile: a split product runs on 128 x 128 tiles, a group on its own
    const int bn = n == 1 ? 128 : gap_tc_grouped_col_tile(nsplit);
    long tiles = 0;
    for (int k = 0; k < n; ++k) tiles += (long)((rows[k] + 127) / 128) * ((D16 + bn - 1) / bn);
    return gap_tc_ksplit(tiles, M_pad[q]);
}

gap_status gap_contract_tc(const float *phat, int D, int D16, const int *rows, int nrows, const TcModelGP &gp,
                           double delta, int zeta, int nsplit, TcScratch &sc, double *eps, float *wsum, float *g,
                           int *err, cudaStream_t st)
{
    if (nrows <= 0 || gp.M <= 0) return GAP_OK;
    const bool three = nsplit == 3;
    gap_prof_begin(ST_SPLIT, st);
    gap_count_launch();
    k_split_rows<<<(nrows + 3) / 4, 128, 0, st>>>(phat, D, D16, rows, nrows, gp.mu, sc.A_hi, sc.A_lo,
                                                   three ? sc.A_mid : nullptr, sc.t_row);
    GAP_TRY_CUDA(cudaGetLastError());
    TcOperands op1{sc.A_hi, sc.A_lo, gp.B_hi, gp.B_lo, nrows, gp.M_pad, D16, D16, D16, nsplit,
                   three ? sc.A_mid : nullptr, three ? gp.B_mid : nullptr};
    TcEpilogue ep1{};
    ep1.s_col = gp.s_col;
    ep1.alpha_col = gp.alpha;
    ep1.t_row = sc.t_row;
    ep1.d2 = (float)(delta * delta);
    ep1.zeta = zeta;
    ep1.W_hi = g ? sc.W_hi : nullptr;
    ep1.W_lo = g ? sc.W_lo : nullptr;
    ep1.W_mid = g && three ? sc.W_mid : nullptr;
    ep1.ldw = gp.M_pad;
    ep1.eps_part = sc.eps_part;
    ep1.wsum_part = sc.wsum_part;
    // the energy partials per column tile of the variant the tuner picks
    int groups = 2;
    const int bn = gap_tc_plan(op1, ep1, EPI_KERNEL, err, st, &groups);
    const int n_part = groups * ((gp.M_pad + bn - 1) / bn);
    ep1.n_part = n_part;
    gap_prof_end(ST_SPLIT, st);
    gap_prof_begin(ST_GEMM_Q, st);
    GAP_TRY(gap_tc_gemm(op1, ep1, EPI_KERNEL, err, st));
    gap_prof_end(ST_GEMM_Q, st);
    TcOperands op2{sc.W_hi, sc.W_lo, gp.BT_hi, gp.BT_lo, nrows, D16, gp.M_pad, gp.M_pad, gp.M_pad, nsplit,
                   three ? sc.W_mid : nullptr, three ? gp.BT_mid : nullptr};
    op2.ksplit = gap_contract_parts(&nrows, &gp.M_pad, 1, D16, nsplit, 0);
    TcEpilogue ep2{};
    const bool split = op2.ksplit > 1;
    ep2.C = split ? sc.Gs : g;
    ep2.row_map = split ? nullptr : rows;
    ep2.ldc = D16;
    if (g) {
        gap_prof_begin(ST_GEMM_G, st);
        GAP_TRY(gap_tc_gemm(op2, ep2, EPI_STORE, err, st));
        gap_prof_end(ST_GEMM_G, st);
    }
    gap_prof_begin(ST_FINALIZE, st);
    GAP_TRY(tc_finalize(rows, nrows, sc, n_part, op2.ksplit, D16, eps, wsum, g, st));
    gap_prof_end(ST_FINALIZE, st);
    return GAP_OK;
}

gap_status gap_contract_tc_groups(const float *phat, int D, int D16, const int *const *rows, const int *nrows,
                                  const TcModelGP *gps, int n, double delta, int zeta, int nsplit,
                                  const TcScratch *sc, double *eps, float *wsum, float *g, int *err, cudaStream_t st)
{
    const bool three = nsplit == 3;
    const int bn = gap_tc_grouped_col_tile(nsplit);
    std::vector<TcOperands> op1(n), op2(n);
    std::vector<TcEpilogue> ep1(n), ep2(n);
    std::vector<int> mpad(n);
    for (int q = 0; q < n; ++q) mpad[q] = gps[q].M_pad;
    gap_prof_begin(ST_SPLIT, st);
    for (int q = 0; q < n; ++q) {
        const TcModelGP &gp = gps[q];
        op1[q] = TcOperands{};
        op2[q] = TcOperands{};
        ep1[q] = TcEpilogue{};
        ep2[q] = TcEpilogue{};
        if (nrows[q] <= 0 || gp.M <= 0) continue;
        gap_count_launch();
        k_split_rows<<<(nrows[q] + 3) / 4, 128, 0, st>>>(phat, D, D16, rows[q], nrows[q], gp.mu, sc[q].A_hi,
                                                          sc[q].A_lo, three ? sc[q].A_mid : nullptr, sc[q].t_row);
        GAP_TRY_CUDA(cudaGetLastError());
        op1[q] = TcOperands{sc[q].A_hi, sc[q].A_lo, gp.B_hi, gp.B_lo, nrows[q], gp.M_pad, D16, D16, D16, nsplit,
                            three ? sc[q].A_mid : nullptr, three ? gp.B_mid : nullptr};
        TcEpilogue &e = ep1[q];
        e.s_col = gp.s_col;
        e.alpha_col = gp.alpha;
        e.t_row = sc[q].t_row;
        e.d2 = (float)(delta * delta);
        e.zeta = zeta;
        e.W_hi = g ? sc[q].W_hi : nullptr;
        e.W_lo = g ? sc[q].W_lo : nullptr;
        e.W_mid = g && three ? sc[q].W_mid : nullptr;
        e.ldw = gp.M_pad;
        e.eps_part = sc[q].eps_part;
        e.wsum_part = sc[q].wsum_part;
        e.n_part = 2 * ((gp.M_pad + bn - 1) / bn);
        op2[q] = TcOperands{sc[q].W_hi, sc[q].W_lo, gp.BT_hi, gp.BT_lo, nrows[q], D16, gp.M_pad, gp.M_pad, gp.M_pad,
                            nsplit, three ? sc[q].W_mid : nullptr, three ? gp.BT_mid : nullptr};
        op2[q].ksplit = gap_contract_parts(nrows, mpad.data(), n, D16, nsplit, q);
        const bool split = op2[q].ksplit > 1;
        ep2[q].C = split ? sc[q].Gs : g;
        ep2[q].row_map = split ? nullptr : rows[q];
        ep2[q].ldc = D16;
    }
    gap_prof_end(ST_SPLIT, st);
    gap_prof_begin(ST_GEMM_Q, st);
    GAP_TRY(gap_tc_gemm_grouped(op1.data(), ep1.data(), n, EPI_KERNEL, err, st));
    gap_prof_end(ST_GEMM_Q, st);
    if (g) {
        gap_prof_begin(ST_GEMM_G, st);
        GAP_TRY(gap_tc_gemm_grouped(op2.data(), ep2.data(), n, EPI_STORE, err, st));
        gap_prof_end(ST_GEMM_G, st);
    }
    gap_prof_begin(ST_FINALIZE, st);
    for (int q = 0; q < n; ++q) {
        if (nrows[q] <= 0 || gps[q].M <= 0) continue;
        GAP_TRY(tc_finalize(rows[q], nrows[q], sc[q], ep1[q].n_part, op2[q].ksplit, D16, eps, wsum, g, st));
    }
    gap_prof_end(ST_FINALIZE, st);
    return GAP_OK;
}
