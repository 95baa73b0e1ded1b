// SOAP expansion, power spectrum and its backward pass, per-pair forces.
//
//   expansion      c^g_{n lm} = sum_j wacc[g][Z_j] f_cut(r_ij) I_nl(r_ij) Y_lm(u_ij)
//                  + central term                                   (Eqs. 19-20, 25)
//   power spectrum p_{a a' l} = s_aa' sum_m c_{a lm} c_{a' lm}, p_hat = p / |p|
//                                                                   (Eqs. 22-24)
//   backward       h = (g - (g . p_hat) p_hat) / |p|, g = d eps / d p_hat;
//                  gamma_{a lm} = sum_a' H_{a a' l} c_{a' lm} with H = sqrt2 h off
//                  the diagonal and 2 h on it; Gamma^z_{n lm} = sum_g wacc[g][z] gamma
//   pair force     d eps_i / d r_ij = sum_lm Gamma^{Z_j}_{n lm} d(R_nl Y_lm)/d r_ij
//                  (Eq. 3 through the chain rule)
//
// Kernels are templated on (n_max, l_max, groups) and on the arithmetic type
// (double for the plain FP64 path, float for the tensor-core path).
#include "gap_internal.h"
#include "soap.h"

namespace {

template <typename T> struct V4;
template <> struct V4<double> { typedef D4 type; };
template <> struct V4<float> { typedef float4 type; };

template <typename T> __device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename T> __device__ __forceinline__ T wacc(const SoapGeom &g, int grp, int z);
template <> __device__ __forceinline__ double wacc<double>(const SoapGeom &g, int grp, int z)
{
    return g.wacc64[grp * GAP_MAX_SPECIES + z];
}
template <> __device__ __forceinline__ float wacc<float>(const SoapGeom &g, int grp, int z)
{
    return g.wacc32[grp * GAP_MAX_SPECIES + z];
}

// channel a of coupling block b -> (group, radial n)
__device__ __forceinline__ void chan(const SoapGeom &g, int b, int a, int N, int &grp, int &n)
{
    if (g.mixed) { grp = b; n = a; }
    else { grp = a / N; n = a % N; }
}

__device__ __forceinline__ int pair_index(int Nc, int a, int ap)  // a <= ap
{
    return a * Nc - (a * (a - 1)) / 2 + (ap - a);
}

// N consecutive values (global or shared memory) as 16- or 8-byte vector
// loads where N sizeof(T) allows it (the rows start on multiples of
// N sizeof(T)).
template <int N, typename T> __device__ __forceinline__ void load_n(const T *p, T (&out)[N])
{
    if constexpr ((N * sizeof(T)) % 16 == 0) {
#pragma unroll
        for (int k = 0; k < N * (int)sizeof(T) / 16; ++k)
            reinterpret_cast<float4 *>(out)[k] = reinterpret_cast<const float4 *>(p)[k];
    } else {
#pragma unroll
        for (int k = 0; k < N * (int)sizeof(T) / 8; ++k)
            reinterpret_cast<float2 *>(out)[k] = reinterpret_cast<const float2 *>(p)[k];
    }
}

// ------------------------------------------------------------ expansion
// The accumulation c_{n lm} += w R_nl Y_lm gives each lane the m values of
// one l, in runs of at most S (the smallest S with sum_l ceil((2l+1)/S) <= 32
// runs): per pair a lane then loads its N values R_nl once for all its m.
template <int L> __host__ __device__ constexpr int expand_slots()
{
    for (int S = 1; S < 2 * L + 1; ++S) {
        int runs = 0;
        for (int l = 0; l <= L; ++l) runs += (2 * l + 1 + S - 1) / S;
        if (runs <= 32) return S;
    }
    return 2 * L + 1;
}

// Row stride of the staged Y_lm: (L+1)^2 made odd, so that the lanes' rows
// fall in distinct banks.
__host__ __device__ constexpr int expand_ylm_stride(int L) { return (L + 1) * (L + 1) | 1; }

// Neighbour pairs staged per batch of k_expand.
constexpr int kExpandBatch = 16;

// Shared memory per warp of k_expand, in elements: the pair staging area
// (Y_lm, R_nl, channel weights and the radial-table position of a batch of
// pairs) and, reusing it afterwards, the coefficients and the power spectrum
// (GA N (L+1)^2 + D).
__host__ __device__ constexpr int expand_stride(int N, int L, int GA, int D)
{
    return (kExpandBatch * (expand_ylm_stride(L) + N * (L + 1) + GA + 3) > GA * N * (L + 1) * (L + 1) + D
                ? kExpandBatch * (expand_ylm_stride(L) + N * (L + 1) + GA + 3)
                : GA * N * (L + 1) * (L + 1) + D) + 3 & ~3;
}

template <int N, int L, int GA, typename T, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
k_expand(SoapGeom geo, const T *__restrict__ tab, int n_atoms, const int *__restrict__ offsets,
         const int *__restrict__ nbr_j, const typename V4<T>::type *__restrict__ vec, const int *__restrict__ species,
         T *__restrict__ coef, T *__restrict__ phat, T *__restrict__ pnorm)
{
    constexpr int LM = (L + 1) * (L + 1);
    constexpr int LMS = expand_ylm_stride(L);
    constexpr int NL = N * (L + 1);
    constexpr int S = expand_slots<L>();
    const int STRIDE = expand_stride(N, L, GA, geo.D);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *base = reinterpret_cast<T *>(smem_raw) + (threadIdx.x >> 5) * STRIDE;
    constexpr int BP = kExpandBatch;
    static_assert(N % 2 == 0 && (BP * LMS) % 4 == 0, "vector reads of the radial values");
    T *Ysm = base, *Rsm = base + BP * LMS, *Wsm = Rsm + BP * NL, *Psm = Wsm + BP * GA;  // Psm [3][BP]: k, u, f
    int *Ksm = reinterpret_cast<int *>(Psm);
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (i >= n_atoms) return;
    const T rc = (T)geo.rc, dw = (T)geo.d, inv_h = T(1) / (T)geo.h;
    typedef typename Coef4<T>::type C4;
    const C4 *tab4 = reinterpret_cast<const C4 *>(tab);

    // this lane's run: degree my_l, entries my_lm .. my_lm + my_cnt - 1
    int my_l = 0, my_lm = 0, my_cnt = 0;
    {
        int run = 0;
#pragma unroll
        for (int l = 0; l <= L; ++l)
#pragma unroll
            for (int m0 = 0; m0 < 2 * l + 1; m0 += S) {
                if (run == lane) {
                    my_l = l;
                    my_lm = l * l + m0;
                    my_cnt = 2 * l + 1 - m0 < S ? 2 * l + 1 - m0 : S;
                }
                ++run;
            }
    }
    T acc[S][GA][N];
#pragma unroll
    for (int o = 0; o < S; ++o)
#pragma unroll
        for (int g = 0; g < GA; ++g)
#pragma unroll
            for (int n = 0; n < N; ++n) acc[o][g][n] = T(0);

    // central Gaussian: lm = 0 only, the first slot of lane 0
    if (lane == 0 && geo.cw != 0.0) {
        const T y00 = T(0.28209479177387814347);  // 1 / (2 sqrt(pi))
        int zi = species[i];
        if (zi < 0 || zi >= geo.S) zi = 0;  // out of range: the call fails (species check)
#pragma unroll
        for (int g = 0; g < GA; ++g)
#pragma unroll
            for (int n = 0; n < N; ++n) acc[0][g][n] += wacc<T>(geo, g, zi) * (T)geo.cw * tab[4 * n] * y00;
    }

    const int p0 = offsets[i], p1 = offsets[i + 1];
    for (int base_p = p0; base_p < p1; base_p += BP) {
        const int cnt = min(BP, p1 - base_p);
        const int p = base_p + lane;
        if (lane < cnt) {
            typename V4<T>::type v = vec[p];
            T r = v.w, ir = T(1) / r;
            ylm_all<L, T>(geo, v.x * ir, v.y * ir, v.z * ir, Ysm + lane * LMS);
            T df;
            const T f = fcut_dev<T>(r, rc, dw, &df);
            const RadialPos<T> rp = radial_pos<T>(r, inv_h, geo.G);
            Ksm[lane] = rp.k;
            Psm[BP + lane] = rp.u;
            Psm[2 * BP + lane] = f;
            int z = species[nbr_j[p]];
            if (z < 0 || z >= geo.S) z = 0;  // out of range: the call fails (species check)
#pragma unroll
            for (int g = 0; g < GA; ++g) Wsm[lane * GA + g] = wacc<T>(geo, g, z);
        }
        __syncwarp();
        // f R_nl of all pairs, the warp over (pair, entry): each pair's
        // table interval is one contiguous row of NL coefficient quads; four
        // loads in flight per lane
        const int total = cnt * NL;
        for (int e0 = lane; e0 < total; e0 += 128) {
            C4 c[4];
            T u[4], f[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int e = e0 + 32 * k;
                if (e < total) {
                    const int t = e / NL;
                    u[k] = Psm[BP + t];
                    f[k] = Psm[2 * BP + t];
                    c[k] = tab4[(size_t)Ksm[t] * NL + (e - t * NL)];
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int e = e0 + 32 * k;
                if (e < total) Rsm[e] = f[k] * (c[k].x + u[k] * (c[k].y + u[k] * (c[k].z + u[k] * c[k].w)));
            }
        }
        __syncwarp();
        for (int t = 0; t < cnt; ++t) {
            const T *Yt = Ysm + t * LMS + my_lm;
            T rv[N], yv[S];
            load_n<N, T>(Rsm + t * NL + my_l * N, rv);
#pragma unroll
            for (int o = 0; o < S; ++o) yv[o] = o < my_cnt ? Yt[o] : T(0);
#pragma unroll
            for (int g = 0; g < GA; ++g) {
                const T wg = Wsm[t * GA + g];
#pragma unroll
                for (int o = 0; o < S; ++o) {
                    const T wy = wg * yv[o];
#pragma unroll
                    for (int n = 0; n < N; ++n) acc[o][g][n] += rv[n] * wy;
                }
            }
        }
        __syncwarp();
    }

    // coefficients to shared memory (reusing the staging area) and to global
    T *csm = base;
    T *psm = base + GA * N * LM;
#pragma unroll
    for (int o = 0; o < S; ++o) {
        const int lm = my_lm + o;
        if (o < my_cnt) {
#pragma unroll
            for (int g = 0; g < GA; ++g)
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    csm[(g * N + n) * LM + lm] = acc[o][g][n];
                    coef[((size_t)i * GA * N + g * N + n) * LM + lm] = acc[o][g][n];
                }
        }
    }
    __syncwarp();
    // power spectrum
    T ss = T(0);
    const int D = geo.D;
    // entries in the l order of the descriptor table: the lanes of a warp
    // run m-loops of one length, with no index decoding
    for (int k = lane; k < D; k += 32) {
        const int4 e = __ldg(geo.dtab + k);
        const int d = e.x, l = e.w & 0xff;
        const T *c1 = csm + e.y, *c2 = csm + e.z;
        T s = T(0);
        for (int m = 0; m <= 2 * l; ++m) s += c1[m] * c2[m];
        if (e.w >> 8) s *= T(1.41421356237309504880);
        psm[d] = s;
        ss += s * s;
    }
    ss = warp_sum(ss);
    T nrm = sqrt(ss), inv = T(1) / nrm;
    __syncwarp();
    for (int d = lane; d < D; d += 32) phat[(size_t)i * D + d] = psm[d] * inv;
    if (lane == 0) pnorm[i] = nrm;
}

// N values to consecutive places, as 16- or 8-byte stores where N sizeof(T)
// allows it (the rows start on multiples of N sizeof(T)).
template <int N, typename T> __device__ __forceinline__ void store_n(T *__restrict__ p, const T (&v)[N])
{
    if constexpr ((N * sizeof(T)) % 16 == 0) {
#pragma unroll
        for (int k = 0; k < N * (int)sizeof(T) / 16; ++k)
            reinterpret_cast<float4 *>(p)[k] = reinterpret_cast<const float4 *>(v)[k];
    } else {
#pragma unroll
        for (int k = 0; k < N * (int)sizeof(T) / 8; ++k)
            reinterpret_cast<float2 *>(p)[k] = reinterpret_cast<const float2 *>(v)[k];
    }
}

// ------------------------------------------------------------ backward chain
// Gam[i][z][lm][n] for every neighbour species z; a warp per atom.  h =
// (g - (g . p_hat) p_hat) / |p| goes to shared memory, then a lane takes the
// (l, m) of its turn with all its channels in registers: the c_{a, lm} of the
// Nc coupled channels once, then every h_{aa'l} (a broadcast or neighbouring
// words: l is the fastest index) serves two FMAs, and Gamma^z is formed from
// the lane's own gammas and stored as runs of N.  With a lane per (channel,
// lm) entry (index arithmetic and two shared reads per FMA) a step of 512
// four-species boxes took 0.9 ms longer, of 32768 atoms 0.11 ms.  MIXED: GA separate blocks of N channels (Eq. 25), else
// one block of GA N channels.
template <int N, int L, int GA, bool MIXED, typename T>
__global__ void __launch_bounds__(128)
k_chain(SoapGeom geo, int n_atoms, const T *__restrict__ gvec, const T *__restrict__ wsum,
        const T *__restrict__ mu, const int *__restrict__ gp_of_atom, const T *__restrict__ phat,
        const T *__restrict__ pnorm, const T *__restrict__ coef, T *__restrict__ Gam)
{
    constexpr int LM = (L + 1) * (L + 1), NB = MIXED ? GA : 1, NC = MIXED ? N : GA * N, PER = NC * (NC + 1) / 2 * (L + 1);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int D = geo.D, warps = blockDim.x >> 5;
    T *hsm = reinterpret_cast<T *>(smem_raw) + (size_t)(threadIdx.x >> 5) * D;
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * warps + (threadIdx.x >> 5);
    if (i >= n_atoms) return;
    const int s = gp_of_atom ? gp_of_atom[i] : 0;
    // g = G + wsum * mu (tensor-core path stores the centred product separately)
    const bool centred = wsum && s >= 0;
    const T ws = centred ? wsum[i] : T(0);
    const T *mus = centred ? mu + (size_t)s * geo.D16 : nullptr;
    const T *gi = gvec + (size_t)i * geo.D16, *pi = phat + (size_t)i * D;
    T gp = T(0);
#pragma unroll 4
    for (int d = lane; d < D; d += 32) {
        T g = gi[d];
        if (centred) g += ws * mus[d];
        hsm[d] = g;
        gp += g * pi[d];
    }
    gp = warp_sum(gp);
    const T inv = T(1) / pnorm[i];
#pragma unroll 4
    for (int d = lane; d < D; d += 32) hsm[d] = (hsm[d] - gp * pi[d]) * inv;
    __syncwarp();
    const T *ci = coef + (size_t)i * GA * N * LM;
    for (int lm = lane; lm < LM; lm += 32) {
        const int l = (int)sqrtf((float)lm + 0.5f);  // floor(sqrt(lm)), lm < 121
        T gam[NB * NC];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            T c[NC], off[NC];
#pragma unroll
            for (int a = 0; a < NC; ++a) {
                c[a] = ci[(b * NC + a) * LM + lm];
                off[a] = T(0);
            }
            const T *h = hsm + b * PER + l;
#pragma unroll
            for (int a = 0, k = 0; a < NC; ++a) {
                const T haa = h[(k++) * (L + 1)];
#pragma unroll
                for (int a2 = a + 1; a2 < NC; ++a2) {
                    const T hv = h[(k++) * (L + 1)];
                    off[a] += hv * c[a2];
                    off[a2] += hv * c[a];
                }
                gam[b * NC + a] = T(2) * haa * c[a];
            }
#pragma unroll
            for (int a = 0; a < NC; ++a) gam[b * NC + a] += T(1.41421356237309504880) * off[a];
        }
        // Gam[i][z][lm][n]: the pair-force kernel reads the n values of one lm
        // as vectors
        for (int z = 0; z < geo.S; ++z) {
            T out[N];
#pragma unroll
            for (int n = 0; n < N; ++n) out[n] = T(0);
#pragma unroll
            for (int g = 0; g < GA; ++g) {
                const T w = wacc<T>(geo, g, z);
#pragma unroll
                for (int n = 0; n < N; ++n) out[n] += w * gam[g * N + n];
            }
            store_n<N, T>(Gam + ((size_t)(i * (size_t)geo.S + z) * LM + lm) * N, out);
        }
    }
}

// ------------------------------------------------------------ pair forces
// The radial coefficients of entries n, n + 1 of one (interval, l): 32 bytes
// in FP32 (one 256-bit load; N is even, so pairs start on 32 bytes).
template <typename T> struct Coef2;
template <> struct Coef2<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float *p)
    {
        asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
            : "l"(p));
    }
};
template <> struct Coef2<double> {
    D4 a, b;
    __device__ __forceinline__ void load(const double *p)
    {
        a = reinterpret_cast<const D4 *>(p)[0];
        b = reinterpret_cast<const D4 *>(p)[1];
    }
};

// fpair[p] = d eps_i / d r_ij for pair p = (i -> j), a thread per pair.  With
// A_lm = sum_n Gamma_{n lm} R_nl and B_lm = sum_n Gamma_{n lm} dR_nl the force is
// a sum over the polynomial forms Y_lm = K Q_l^|m|(z) {C_m, S_m}; its l sums are
// taken first, per m, for the three factors they leave (x and y derivatives,
// z derivative, value), so an (l, m) costs 2 N + 3 FMAs, and the C_m, S_m
// enter once at the end.  The projection of the gradient onto the sphere
// needs only the total.  The table rows bound it (1.2 KB per pair at n = l =
// 8, from L2 where L1 misses): read as whole lines, 32 bytes per load.
template <int N, int L, typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 2 : 4)
k_pairforce(SoapGeom geo, const T *__restrict__ tab, int n_pairs, const int *__restrict__ n_valid,
            const int *__restrict__ pair_i, const int *__restrict__ nbr_j,
            const typename V4<T>::type *__restrict__ vec, const int *__restrict__ species,
            const T *__restrict__ Gam, T *__restrict__ fpair)
{
    constexpr int LM = (L + 1) * (L + 1);
    constexpr int NL = N * (L + 1);
    static_assert(N % 2 == 0, "entries are read in pairs");
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pairs || p >= *n_valid) return;
    const int i = pair_i[p];
    const int zr = species[nbr_j[p]], z = zr >= 0 && zr < geo.S ? zr : 0;  // out of range: the call fails
    const T *Gm = Gam + ((size_t)i * geo.S + z) * N * LM;
    typename V4<T>::type v = vec[p];
    const T r = v.w, ir = T(1) / r;
    const T ux = v.x * ir, uy = v.y * ir, uz = v.z * ir;
    T df;
    const T f = fcut_dev<T>(r, (T)geo.rc, (T)geo.d, &df);
    const T inv_h = T(1) / (T)geo.h;
    const RadialPos<T> rp = radial_pos<T>(r, inv_h, geo.G);
    const T *row = tab + (size_t)rp.k * NL * 4;
    const T fh = f * inv_h, u2 = T(2) * rp.u, u3 = T(3) * rp.u * rp.u;

    // per m >= 0 and its negative: sum_l A K Q_l^m, sum_l A K Q_l^{m+1}, sum_l B K Q_l^m
    T P[L + 1], Pn[L + 1], Z[L + 1], Zn[L + 1], V[L + 1], Vn[L + 1];
#pragma unroll
    for (int m = 0; m <= L; ++m) P[m] = Pn[m] = Z[m] = Zn[m] = V[m] = Vn[m] = T(0);
    T q1[L + 2], q2[L + 2];
#pragma unroll
    for (int l = 0; l <= L; ++l) {
        T R[N], dR[N];
#pragma unroll
        for (int n = 0; n < N; n += 2) {
            Coef2<T> c;
            c.load(row + 4 * (l * N + n));
            const T I0 = c.a.x + rp.u * (c.a.y + rp.u * (c.a.z + rp.u * c.a.w));
            const T I1 = c.b.x + rp.u * (c.b.y + rp.u * (c.b.z + rp.u * c.b.w));
            R[n] = f * I0;
            R[n + 1] = f * I1;
            dR[n] = df * I0 + fh * (c.a.y + u2 * c.a.z + u3 * c.a.w);
            dR[n + 1] = df * I1 + fh * (c.b.y + u2 * c.b.z + u3 * c.b.w);
        }
        T q[L + 2];
#pragma unroll
        for (int m = 0; m <= L + 1; ++m) {
            if (m > l) { q[m] = T(0); continue; }
            if (m == l) q[m] = (l == 0) ? T(1) : T(2 * l - 1) * q1[l - 1];
            else if (m == l - 1) q[m] = T(2 * l - 1) * uz * q1[m];
            else q[m] = (T(2 * l - 1) * uz * q1[m] - T(l + m - 1) * q2[m]) * (T(1) / T(l - m));  // l, m unrolled: a constant
        }
#pragma unroll
        for (int m = 0; m <= L; ++m) {
            if (m > l) continue;
            const T k = ylm_k<T>(geo, l, m), kq = k * q[m], kz = k * q[m + 1];
            T G[N];
            load_n<N, T>(Gm + (l * l + l + m) * N, G);
            T A = T(0), B = T(0);
#pragma unroll
            for (int n = 0; n < N; ++n) { A += G[n] * R[n]; B += G[n] * dR[n]; }
            P[m] += A * kq;
            Z[m] += A * kz;
            V[m] += B * kq;
            if (m > 0) {
                load_n<N, T>(Gm + (l * l + l - m) * N, G);
                A = B = T(0);
#pragma unroll
                for (int n = 0; n < N; ++n) { A += G[n] * R[n]; B += G[n] * dR[n]; }
                Pn[m] += A * kq;
                Zn[m] += A * kz;
                Vn[m] += B * kq;
            }
        }
#pragma unroll
        for (int m = 0; m <= L; ++m) {
            if (m > l) continue;
            q2[m] = q1[m];
            q1[m] = q[m];
        }
    }
    // (C_m, S_m) = (x + i y)^m; d/dx of C_m, S_m is m (C_{m-1}, S_{m-1}), d/dy m (-S_{m-1}, C_{m-1})
    T sU = V[0], sx = T(0), sy = T(0), sz = Z[0], C = T(1), Sn = T(0);
#pragma unroll
    for (int m = 1; m <= L; ++m) {
        sx += T(m) * (C * P[m] + Sn * Pn[m]);
        sy += T(m) * (C * Pn[m] - Sn * P[m]);
        const T c2 = ux * C - uy * Sn;
        Sn = ux * Sn + uy * C;
        C = c2;
        sz += C * Z[m] + Sn * Zn[m];
        sU += C * V[m] + Sn * Vn[m];
    }
    sU -= ir * (ux * sx + uy * sy + uz * sz);
    fpair[3 * (size_t)p] = sU * ux + sx * ir;
    fpair[3 * (size_t)p + 1] = sU * uy + sy * ir;
    fpair[3 * (size_t)p + 2] = sU * uz + sz * ir;
}

// ------------------------------------------------------------ two-body term
// E(r) and dE/dr of the two-body pair energy, evaluated directly (FP64).
__device__ double twobody_exact(const TwoBodyDev &tb, double r, double *dE)
{
    double df;
    const double f = fcut_dev<double>(r, tb.rc, tb.d, &df);
    const double t2 = tb.theta * tb.theta, d2 = tb.delta * tb.delta;
    double es = 0.0, des = 0.0;
    for (int m = 0; m < tb.m; ++m) {
        const double dx = r - tb.x[m];
        const double k = exp(-dx * dx / (2.0 * t2));
        es += tb.a[m] * k;
        des += tb.a[m] * (df - f * dx / t2) * k;
    }
    *dE = d2 * des;
    return d2 * f * es;
}

// Interval k of the two-body table: cubic Hermite coefficients in u = (r - r_k)/h
// from the exact values and derivatives at both knots.
__global__ void k_twobody_table(TwoBodyDev tb, D4 *__restrict__ tab)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= tb.g_in + tb.g_out) return;
    const double r0 = k < tb.g_in ? k * tb.h_in : (tb.rc - tb.d) + (k - tb.g_in) * tb.h_out;
    const double h = k < tb.g_in ? tb.h_in : tb.h_out;
    double d0, d1;
    const double e0 = twobody_exact(tb, r0, &d0), e1 = twobody_exact(tb, r0 + h, &d1);
    tab[k] = D4{e0, h * d0, 3.0 * (e1 - e0) - h * (2.0 * d0 + d1), 2.0 * (e0 - e1) + h * (d0 + d1)};
}

// Lanes that share one atom's pairs in the per-atom sums below.  An atom has
// 25-40 pairs: eight lanes leave a chain of four or five dependent loads (one
// thread per atom walked all of them: 30 us of latency at 64 atoms), and a
// block still covers 16 atoms.
constexpr int kPairLanes = 8;

template <typename T> __device__ __forceinline__ T group_sum(T v)
{
#pragma unroll
    for (int o = kPairLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Two-body term of every atom from the tabulated E(r), FP64 in every
// precision mode (the term is large next to the 1e-4 eV/A force bound): half
// of each pair's energy to eps2, and, when fw2 is given, the atom's force and
// virial (F, then W_xx W_yy W_zz W_yz W_xz W_xy: it is symmetric).  The pair's
// two directions carry opposite derivatives, so the reverse pair is not read:
// F_i = sum_p 2 f[p], W_i = -sum_p f[p] (x) r_p with f = E'(r) / 2 u.
// Bound by the FP64 pipe (about 25 FP64 instructions per pair).
__global__ void __launch_bounds__(128)
k_twobody(int n_atoms, const int *__restrict__ offsets, const D4 *__restrict__ vec, TwoBodyDev tb,
          double *__restrict__ eps2, double *__restrict__ fw2)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) / kPairLanes, sub = threadIdx.x % kPairLanes;
    const double rt = tb.rc - tb.d, inv_in = 1.0 / tb.h_in, inv_out = 1.0 / tb.h_out;
    double e = 0.0, F[3] = {0, 0, 0}, W[6] = {0, 0, 0, 0, 0, 0};
    const int p1 = i < n_atoms ? offsets[i + 1] : 0;
    for (int p = i < n_atoms ? offsets[i] + sub : 0; p < p1; p += kPairLanes) {
        const D4 v = vec[p];
        const double r = v.w;
        if (r >= tb.rc) continue;
        const bool in = r < rt;
        const double inv = in ? inv_in : inv_out, s = (in ? r : r - rt) * inv;
        const int k = min((int)s, (in ? tb.g_in : tb.g_out) - 1);
        const double u = s - k;
        const D4 a = tb.tab[in ? k : tb.g_in + k];
        e += a.x + u * (a.y + u * (a.z + u * a.w));
        if (fw2) {
            const double c = divide64((a.y + u * (2.0 * a.z + 3.0 * u * a.w)) * inv, r);
            const double fx = c * v.x, fy = c * v.y, fz = c * v.z;
            F[0] += fx;
            F[1] += fy;
            F[2] += fz;
            W[0] -= fx * v.x;
            W[1] -= fy * v.y;
            W[2] -= fz * v.z;
            W[3] -= fy * v.z;
            W[4] -= fx * v.z;
            W[5] -= fx * v.y;
        }
    }
    e = group_sum(e);
#pragma unroll
    for (int a = 0; a < 3; ++a) F[a] = group_sum(F[a]);
#pragma unroll
    for (int a = 0; a < 6; ++a) W[a] = group_sum(W[a]);
    if (i < n_atoms && sub == 0) {
        eps2[i] = 0.5 * e;
        if (fw2) {
#pragma unroll
            for (int a = 0; a < 3; ++a) fw2[9 * (size_t)i + a] = F[a];
#pragma unroll
            for (int a = 0; a < 6; ++a) fw2[9 * (size_t)i + 3 + a] = 0.5 * W[a];
        }
    }
}

// ------------------------------------------------------ forces and virials
// Running sums of the pair terms.  FP64 terms are summed in FP64; FP32 terms
// (and the exact products of two of them) in three FP32 words: two-sum and
// two-product (Ogita, Rump and Oishi 2005) pass every rounding error on to the
// next word, so the sum is good to more than FP64's 53 bits.  One FP64
// instruction holds GB300's FP64 pipe for ~64 cycles per warp where the
// thirteen FP32 ones of a term take thirteen.  Every operation is rounded by
// itself: contracted into a multiply-add, s + p would hold p's rounding error
// already and sub_product count it twice.  (Products below 2^-102 keep an
// absolute error of 2^-149.)
template <typename T> struct PairSum;
template <> struct PairSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void sub_product(double a, double b) { s -= a * b; }
    // adds what the lane at distance o sends
    __device__ __forceinline__ void receive(const PairSum &sent, int o) { s += __shfl_xor_sync(0xffffffffu, sent.s, o); }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct PairSum<float> {
    float s = 0.f, c = 0.f, e = 0.f;
    // a + x rounded; the error to r
    static __device__ __forceinline__ float two_sum(float a, float x, float &r)
    {
        const float t = __fadd_rn(a, x), b = __fsub_rn(t, a);
        r = __fadd_rn(__fsub_rn(a, __fsub_rn(t, b)), __fsub_rn(x, b));
        return t;
    }
    __device__ __forceinline__ void carry(float x)
    {
        float r;
        c = two_sum(c, x, r);
        e = __fadd_rn(e, r);
    }
    __device__ __forceinline__ void add(float x)
    {
        float r;
        s = two_sum(s, x, r);
        carry(r);
    }
    __device__ __forceinline__ void sub_product(float a, float b)
    {
        const float p = -__fmul_rn(a, b);
        carry(-__fmaf_rn(a, b, p));
        add(p);
    }
    __device__ __forceinline__ void receive(const PairSum &sent, int o)
    {
        const float s2 = __shfl_xor_sync(0xffffffffu, sent.s, o), c2 = __shfl_xor_sync(0xffffffffu, sent.c, o),
                    e2 = __shfl_xor_sync(0xffffffffu, sent.e, o);
        add(s2);
        carry(c2);
        e = __fadd_rn(e, e2);
    }
    __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)e); }
};

// Halves the entries of two lanes at distance o: the upper half of them goes to
// the lane with bit o set, each lane adding the other's share of its half.
template <typename S, int N>
__device__ __forceinline__ void share(const S (&all)[N], S (&mine)[N / 2], int o)
{
    const bool up = (threadIdx.x & o) != 0;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const S sent = up ? all[k] : all[N / 2 + k];
        mine[k] = up ? all[N / 2 + k] : all[k];
        mine[k].receive(sent, o);
    }
}

// The sums of one atom's pairs p0 + sub, p0 + sub + kPairLanes, ... over its
// eight lanes.  Of the twelve (F, then W row-major, zero unless virial) lane
// sub gets entries first_entry(sub) and, in even lanes, the next: the lanes
// halve the entries three times (11 additions a lane where a butterfly over
// all of them takes 36).
__device__ __forceinline__ int first_entry(int sub) { return 6 * (sub >> 2) + 3 * ((sub >> 1) & 1) + 2 * (sub & 1); }

template <typename S, typename T, typename V>
__device__ __forceinline__ void sum_pairs(S (&mine)[2], int p0, int p1, int sub, const int *__restrict__ rev,
                                          const V *__restrict__ vec, const T *__restrict__ fpair, bool virial)
{
    S acc[12], half[6], quarter[4];
    for (int p = p0 + sub; p < p1; p += kPairLanes) {
        const size_t q = 3 * (size_t)rev[p];
        const V v = vec[p];
        T fp[3], fq[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            fp[a] = fpair[3 * (size_t)p + a];
            fq[a] = fpair[q + a];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc[a].add(fp[a]);
            acc[a].add(-fq[a]);
        }
        if (virial) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                acc[3 + 3 * a].sub_product(fp[a], v.x);
                acc[4 + 3 * a].sub_product(fp[a], v.y);
                acc[5 + 3 * a].sub_product(fp[a], v.z);
            }
        }
    }
    static_assert(kPairLanes == 8, "three halvings");
    share(acc, half, 4);
    S three[3];
    share(half, three, 2);
#pragma unroll
    for (int k = 0; k < 3; ++k) quarter[k] = three[k];
    quarter[3] = S{};
    share(quarter, mine, 1);
}

// F_j = sum_{p in pairs(j)} (f[p] - f[rev p]);  W_j = -sum_{p in pairs(j)} f[p] (x) r_p,
// plus the two-body force and virial of the atom (fw2, see k_twobody).
// kPairLanes lanes per atom: latency bounds it at few atoms (a captured step of
// 64 atoms took 151 us with a thread per atom, 120 us with eight lanes).  Three
// words per sum instead of two, with the halved entries in place of a butterfly:
// a step of 64 atoms 73.8 -> 74.2 us, of 32768 1284 -> 1277 us.
template <typename T>
__global__ void __launch_bounds__(128)
k_gather(int n_atoms, const int *__restrict__ offsets, const int *__restrict__ rev,
         const typename V4<T>::type *__restrict__ vec, const T *__restrict__ fpair, const double *__restrict__ fw2,
         double *__restrict__ forces, double *__restrict__ vir_atom)
{
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) / kPairLanes, sub = threadIdx.x % kPairLanes;
    const int p0 = j < n_atoms ? offsets[j] : 0, p1 = j < n_atoms ? offsets[j + 1] : 0;
    PairSum<T> mine[2];
    sum_pairs(mine, p0, p1, sub, rev, vec, fpair, vir_atom != nullptr);
    double v[2] = {mine[0].value(), mine[1].value()};
    if constexpr (sizeof(T) == 4) {
        // beyond FP32's range (or infinite, or no number): the FP64 sum
        const bool wide[2] = {!(fabsf(mine[0].s) <= 3.402823466e38f), !(fabsf(mine[1].s) <= 3.402823466e38f)};
        if (__any_sync(0xffffffffu, wide[0] || wide[1])) {
            PairSum<double> sums[2];
            sum_pairs(sums, p0, p1, sub, rev, vec, fpair, vir_atom != nullptr);
#pragma unroll
            for (int h = 0; h < 2; ++h) v[h] = wide[h] ? sums[h].s : v[h];
        }
    }
    if (j >= n_atoms) return;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int q = first_entry(sub) + h;
        if (h > (~sub & 1)) continue;  // odd lanes own one entry
        // the two-body term's symmetric virial is stored xx yy zz yz xz xy: the
        // place of entry q, four bits each
        if (fw2) v[h] += fw2[9 * (size_t)j + ((0x567648783210ull >> (4 * q)) & 15)];
        if (q < 3) {
            if (forces) forces[3 * (size_t)j + q] = v[h];
        } else if (vir_atom) {
            vir_atom[9 * (size_t)j + q - 3] = v[h];
        }
    }
}

// Energy (eps + eps2) and virial sums of each configuration, over chunks of
// atoms (block (c, k): atoms k chunk .. of configuration c), so that a large
// configuration spreads over many SMs; with one chunk per configuration the
// sums are final, else k_config_final adds the chunks (fixed order:
// deterministic).  Also writes the local energies eps + eps2.  The FP64 pipe
// bounds it: one atom per thread (256 atoms per chunk), then each warp sums
// whole columns over the block (13 FP64 adds per column).  Chunks of 2048
// where 256 would need too many blocks or partial sums (grid y is limited to
// 65535; 2^20 chunks hold 84 MB).
constexpr int kCfgThreads = 256;

int config_chunk(int n_configs, int max_atoms)
{
    const long nchunk = ((long)max_atoms + kCfgThreads - 1) / kCfgThreads;
    return nchunk <= 65535 && (nchunk <= 1 || nchunk * n_configs <= (1L << 20)) ? kCfgThreads : 2048;
}

__device__ __forceinline__ void config_store(int c, int a, double s, double *energy, double *virial)
{
    if (a == 0) {
        if (energy) energy[c] = s;
    } else if (virial) {
        virial[9 * (size_t)c + a - 1] = s;
    }
}

__global__ void __launch_bounds__(kCfgThreads)
k_config_part(int nchunk, int chunk, const int *__restrict__ cfg_off, const double *__restrict__ eps,
              const double *__restrict__ eps2, const double *__restrict__ vir_atom, double *__restrict__ part,
              double *__restrict__ energy, double *__restrict__ virial, double *__restrict__ local_e)
{
    __shared__ double red[10][kCfgThreads];
    const int c = blockIdx.x, k = blockIdx.y;
    const int i0 = cfg_off[c] + k * chunk, iend = cfg_off[c + 1], i1 = iend - i0 < chunk ? iend : i0 + chunk;
    const int nq = vir_atom ? 10 : 1;
    double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = i0 + (int)threadIdx.x; i < i1; i += kCfgThreads) {
        const double e = eps[i] + (eps2 ? eps2[i] : 0.0);
        if (local_e) local_e[i] = e;
        acc[0] += e;
        if (vir_atom)
#pragma unroll
            for (int a = 0; a < 9; ++a) acc[1 + a] += vir_atom[9 * (size_t)i + a];
    }
#pragma unroll
    for (int a = 0; a < 10; ++a)
        if (a < nq) red[a][threadIdx.x] = acc[a];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int a = warp; a < nq; a += kCfgThreads / 32) {
        double s = 0.0;
#pragma unroll
        for (int t = 0; t < kCfgThreads / 32; ++t) s += red[a][32 * t + lane];
        s = warp_sum(s);
        if (lane == 0) {
            if (nchunk == 1) config_store(c, a, s, energy, virial);
            else part[((size_t)c * nchunk + k) * 10 + a] = s;
        }
    }
}

// Block per configuration, warp per column: lanes over chunks.
__global__ void __launch_bounds__(320)
k_config_final(int nchunk, int nq, const double *__restrict__ part, double *__restrict__ energy,
               double *__restrict__ virial)
{
    const int c = blockIdx.x, a = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (a >= nq) return;
    double s = 0.0;
    for (int k = lane; k < nchunk; k += 32) s += part[((size_t)c * nchunk + k) * 10 + a];
    s = warp_sum(s);
    if (lane == 0) config_store(c, a, s, energy, virial);
}

// ----------------------------------------------------------- dispatching
constexpr size_t kMaxSmem = 227 * 1024;  // opt-in dynamic shared memory per block

template <typename T> struct Launch {
    template <int N, int L, int GA>
    static gap_status expand(const SoapGeom &g, const T *tab, int n, const PairList &pl, const int *species, T *coef,
                             T *phat, T *pnorm, cudaStream_t st)
    {
        constexpr int WARPS = 2;
        const size_t shm = sizeof(T) * WARPS * (size_t)expand_stride(N, L, GA, g.D);
        if (shm > kMaxSmem) {
            gap_set_error("descriptor too large for the expansion kernel's shared memory");
            return GAP_EUNSUPPORTED;
        }
        auto kern = k_expand<N, L, GA, T, WARPS>;
        if (shm > 48 * 1024)
            GAP_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
        const typename V4<T>::type *vec;
        if constexpr (sizeof(T) == 8) vec = pl.vec64; else vec = pl.vec32;
        gap_count_launch();
        kern<<<(n + WARPS - 1) / WARPS, 32 * WARPS, shm, st>>>(g, tab, n, pl.offsets, pl.j, vec, species, coef, phat,
                                                              pnorm);
        return gap_cuda_status(cudaGetLastError(), "k_expand");
    }
    template <int N, int L, int GA>
    static gap_status chain(const SoapGeom &g, int n, const T *gvec, const T *wsum, const T *mu, const int *gp_of_atom,
                            const T *phat, const T *pnorm, const T *coef, T *Gam, cudaStream_t st)
    {
        // Four atoms per block once that fills the chip, one for few atoms.  One
        // and four: 32768 atoms, (n, l) = (6, 4) 34 and 25 us, (8, 8) 63 and 56,
        // four species unmixed (8, 6) 2735 and 2283; 1728 atoms the same but for
        // the unmixed ones (199 and 133); 144 atoms unmixed 45 and 53.  FP64, four
        // mixed species: 1000 atoms 74 and 81, 1728 atoms 116 and 116, 3584 atoms
        // 225 and 225.  (Unmixed descriptors alone would change over at about one
        // atom per SM.)
        const int warps = n >= 2048 && 4 * sizeof(T) * (size_t)g.D <= kMaxSmem ? 4 : 1;
        const size_t shm = sizeof(T) * (size_t)g.D * warps;
        if (shm > kMaxSmem) {
            gap_set_error("descriptor too large for the chain kernel's shared memory");
            return GAP_EUNSUPPORTED;
        }
        auto kern = GA > 1 && g.mixed ? k_chain<N, L, GA, (GA > 1), T> : k_chain<N, L, GA, false, T>;
        if (shm > 48 * 1024)
            GAP_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
        gap_count_launch();
        kern<<<(n + warps - 1) / warps, 32 * warps, shm, st>>>(g, n, gvec, wsum, mu, gp_of_atom, phat, pnorm, coef, Gam);
        return gap_cuda_status(cudaGetLastError(), "k_chain");
    }
    template <int N, int L, int GA>
    static gap_status pairforce(const SoapGeom &g, const T *tab, const PairList &pl, const int *species,
                                const T *Gam, T *fpair, cudaStream_t st)
    {
        if (pl.n_pairs == 0) return GAP_OK;
        const typename V4<T>::type *vec;
        if constexpr (sizeof(T) == 8) vec = pl.vec64; else vec = pl.vec32;
        gap_count_launch();
        // One warp per block while that spreads the warps over more SMs (the
        // FP64 pipe and L1 are per SM); the FP64 form's registers allow no more
        // warps per SM in larger blocks either.  FP32 with 32 and 128 threads, (n,
        // l) = (8, 8): 1800 pairs 12.2 and 13.3 us, 28 thousand 16.3 and 17.1, 56
        // thousand 22.5 and 25.6, 918 thousand 242 and 250; (2, 1): 28 thousand
        // 6.8 and 6.5, 918 thousand 22.5 and 16.3.  Beyond 32 thousand the
        // difference is 1 to 3% either way but for the smallest shape, which
        // blocks of one warp would slow down.
        const int threads = sizeof(T) == 8 || pl.n_pairs <= 32 * 1024 ? 32 : 128;
        k_pairforce<N, L, T><<<(pl.n_pairs + threads - 1) / threads, threads, 0, st>>>(
            g, tab, pl.n_pairs, pl.count, pl.i, pl.j, vec, species, Gam, fpair);
        return gap_cuda_status(cudaGetLastError(), "k_pairforce");
    }
};

// Supported (n_max, l_max, groups) instantiations.
#define GAP_SHAPES(X)  \
    X(2, 1, 1)         \
    X(4, 3, 1)         \
    X(4, 3, 2)         \
    X(4, 3, 4)         \
    X(6, 4, 1)         \
    X(6, 6, 1)         \
    X(8, 4, 1)         \
    X(8, 6, 1)         \
    X(8, 4, 5)         \
    X(8, 6, 4)         \
    X(8, 8, 1)         \
    X(10, 8, 1)

}  // namespace

bool gap_shape_supported(int N, int L, int GA)
{
#define X(n, l, ga) if (N == n && L == l && GA == ga) return true;
    GAP_SHAPES(X)
#undef X
    return false;
}

template <typename T>
gap_status gap_expand(const SoapGeom &g, const T *tab, int n, const PairList &pl, const int *species, T *coef, T *phat,
                      T *pnorm, cudaStream_t st)
{
    if (n == 0) return GAP_OK;
#define X(nn, ll, ga) \
    if (g.N == nn && g.L == ll && g.GA == ga) return Launch<T>::template expand<nn, ll, ga>(g, tab, n, pl, species, coef, phat, pnorm, st);
    GAP_SHAPES(X)
#undef X
    gap_set_error("unsupported (n_max, l_max, groups)");
    return GAP_EUNSUPPORTED;
}

template <typename T>
gap_status gap_chain(const SoapGeom &g, int n, const T *gvec, const T *wsum, const T *mu, const int *gp_of_atom,
                     const T *phat, const T *pnorm, const T *coef, T *Gam, cudaStream_t st)
{
    if (n == 0) return GAP_OK;
#define X(nn, ll, ga) \
    if (g.N == nn && g.L == ll && g.GA == ga) return Launch<T>::template chain<nn, ll, ga>(g, n, gvec, wsum, mu, gp_of_atom, phat, pnorm, coef, Gam, st);
    GAP_SHAPES(X)
#undef X
    gap_set_error("unsupported (n_max, l_max, groups)");
    return GAP_EUNSUPPORTED;
}

template <typename T>
gap_status gap_pairforce(const SoapGeom &g, const T *tab, const PairList &pl, const int *species, const T *Gam,
                         T *fpair, cudaStream_t st)
{
#define X(nn, ll, ga) \
    if (g.N == nn && g.L == ll) return Launch<T>::template pairforce<nn, ll, 1>(g, tab, pl, species, Gam, fpair, st);
    GAP_SHAPES(X)
#undef X
    gap_set_error("unsupported (n_max, l_max)");
    return GAP_EUNSUPPORTED;
}

gap_status gap_twobody_table(const TwoBodyDev &tb, D4 *tab, cudaStream_t st)
{
    const int G = tb.g_in + tb.g_out;
    gap_count_launch();
    k_twobody_table<<<(G + 127) / 128, 128, 0, st>>>(tb, tab);
    return gap_cuda_status(cudaGetLastError(), "k_twobody_table");
}

gap_status gap_twobody(int n, const PairList &pl, const TwoBodyDev &tb, double *fw2, double *eps2, cudaStream_t st)
{
    if (n == 0) return GAP_OK;
    constexpr int kAtoms = 128 / kPairLanes;  // per block
    gap_count_launch();
    k_twobody<<<(n + kAtoms - 1) / kAtoms, 128, 0, st>>>(n, pl.offsets, pl.vec64, tb, eps2, fw2);
    return gap_cuda_status(cudaGetLastError(), "k_twobody");
}

template <typename T>
gap_status gap_gather(int n, const PairList &pl, const T *fpair, const double *fw2, double *forces, double *vir_atom,
                      cudaStream_t st)
{
    if (n == 0) return GAP_OK;
    const typename V4<T>::type *vec;
    if constexpr (sizeof(T) == 8) vec = pl.vec64; else vec = pl.vec32;
    constexpr int kAtoms = 128 / kPairLanes;  // per block
    gap_count_launch();
    k_gather<T><<<(n + kAtoms - 1) / kAtoms, 128, 0, st>>>(n, pl.offsets, pl.rev, vec, fpair, fw2, forces, vir_atom);
    return gap_cuda_status(cudaGetLastError(), "k_gather");
}

size_t gap_config_part_doubles(int n_configs, int max_atoms)
{
    const int chunk = config_chunk(n_configs, max_atoms);
    return 10 * (size_t)n_configs * (max_atoms > chunk ? (max_atoms + chunk - 1) / chunk : 1);
}

gap_status gap_config_sums(int n_configs, const int *cfg_off, int max_atoms, const double *eps, const double *eps2,
                           const double *vir_atom, double *energy, double *virial, double *local_e, double *part,
                           cudaStream_t st)
{
    if (n_configs == 0) return GAP_OK;
    const int chunk = config_chunk(n_configs, max_atoms), nchunk = max_atoms > chunk ? (max_atoms + chunk - 1) / chunk : 1;
    gap_count_launch();
    k_config_part<<<dim3(n_configs, nchunk), kCfgThreads, 0, st>>>(nchunk, chunk, cfg_off, eps, eps2, vir_atom, part,
                                                                   energy, virial, local_e);
    GAP_TRY_CUDA(cudaGetLastError());
    if (nchunk == 1) return GAP_OK;
    gap_count_launch();
    k_config_final<<<n_configs, 320, 0, st>>>(nchunk, vir_atom ? 10 : 1, part, energy, virial);
    return gap_cuda_status(cudaGetLastError(), "k_config_final");
}

#define INST(T)                                                                                                      \
    template gap_status gap_expand<T>(const SoapGeom &, const T *, int, const PairList &, const int *, T *, T *, T *, \
                                      cudaStream_t);                                                                 \
    template gap_status gap_chain<T>(const SoapGeom &, int, const T *, const T *, const T *, const int *, const T *,  \
                                     const T *, const T *, T *, cudaStream_t);                                       \
    template gap_status gap_pairforce<T>(const SoapGeom &, const T *, const PairList &, const int *, const T *, T *,    \
                                         cudaStream_t);                                                              \
    template gap_status gap_gather<T>(int, const PairList &, const T *, const double *, double *, double *,          \
                                      cudaStream_t);
INST(double)
INST(float)
