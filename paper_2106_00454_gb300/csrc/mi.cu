// mi.cu -- matrix-inversion (MI) solution of the LS equation (Sec. 2.1), the
// paper's comparison method, batched over (sample, channel, energy).
//
// The real K-matrix with the Haftel-Tabakin pole subtraction on the grid
// {k_j} (N_Q Gauss-Legendre points mapped by k = c tan(pi (1 + x) / 4)) plus
// the on-shell point p:
//   D_j = w_j k_j^2 2 mu / (p^2 - k_j^2)  (j < N_Q),
//   D_N = -2 mu p^2 sum_j w_j / (p^2 - k_j^2),
//   (1 - V D) K = V,
// with the on-shell K, T = (1 + i pi mu p K)^-1 K, S = 1 - 2 pi i mu p T and
// the phases.  As in the paper's timing study (Sec. 6) the equation is solved
// at n_I interpolation energies and the phase shifts are interpolated linearly
// in T_lab to the requested energies, from which the np total cross section
// follows.
//
// GB300 layout: the potential terms on the grid are computed once per channel
// set (k_mi_pot_grid) and the on-shell rows once per energy list
// (k_mi_pot_onshell).  Many systems go through one eigendecomposition per
// (sample, channel) (k_mi_energies below).  Few of them, and those it leaves,
// are solved by elimination: k_mi_solve runs persistent CTAs, each owning a slot of
// FP64 scratch for one (sample, channel) matrix V = V0 + sum_a c_a V_a, and for
// every energy of its chunk inverts 1 - V D in FP32 in shared memory (Gauss-Jordan, partial
// pivoting; FP32 issues at 58x the FP64 rate) and refines the solution to FP64
// accuracy with FP64 residuals r = b - (x - V (D x)) (classical iterative
// refinement: every step is two matrix-vector products).
#include <math.h>

#include "potential.cuh"
#include "wpcd_internal.cuh"

namespace wpcd {

constexpr int kMiThreads = 512;  // one CTA per SM for coupled systems: 16 warps to hide latency
constexpr int kMiMaxRefine = 30;

// ------------------------------------------------------------------------------------- grid
__global__ void k_mi_grid(int NQ, double cmap, const double *glx, const double *glw, double *k, double *w)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= NQ) return;
    const double th = kPi * (1.0 + glx[j]) / 4.0, cth = cos(th);
    k[j] = cmap * tan(th);
    w[j] = cmap * (kPi / 4.0) * glw[j] / (cth * cth);
}

cudaError_t launch_mi_grid(int NQ, double cmap, const double *glx, const double *glw, double *k, double *w,
                           cudaStream_t st)
{
    k_mi_grid<<<(NQ + 127) / 128, 128, 0, counted(st)>>>(NQ, cmap, glx, glw, k, w);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------- potential
__device__ __forceinline__ int mi_lblock(const MiChanDev &c, int a)
{
    return c.coupled ? (a == 0 ? c.J - 1 : c.J + 1) : c.l;
}

// Grid part of V_t for every channel: entries (a, i), (b, j) with i, j < N_Q;
// one thread per grid pair i <= j (the mirror follows from V^{l'l}(p', p) =
// V^{ll'}(p, p')).  Vg of channel c: [n_terms][n][n] at c.vg_off, n = K (N_Q+1).
template <int GEN>
__global__ void __launch_bounds__(128) k_mi_pot_grid(const MiChanDev *chans, int n_ch, int NQ, const double *kg,
                                                     int Lmax, const double *gp, const double *angx,
                                                     const double *angw, int n_terms, double *Vg)
{
    __shared__ double wpl[kAngleQ][kLmaxReg + 1];
    __shared__ double ax[kAngleQ];
    const int Lm = (Lmax < kLmaxReg) ? Lmax : kLmaxReg;
    if (GEN == WPCD_GEN_YUKAWA) {
        angle_tables(angx, angw, Lm, wpl, ax);
        __syncthreads();
    }
    const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= (long long)NQ * (NQ + 1) / 2) return;
    int j = (int)((sqrt(8.0 * (double)b + 1.0) - 1.0) * 0.5);
    while ((long long)(j + 1) * (j + 2) / 2 <= b) ++j;
    while ((long long)j * (j + 1) / 2 > b) --j;
    const int i = (int)(b - (long long)j * (j + 1) / 2);
    const double pp = kg[i], p = kg[j];
    double I1[kLmaxReg + 1], I2[kLmaxReg + 1], I3[kLmaxReg + 1], R = 0.0;
    if (GEN == WPCD_GEN_YUKAWA) yukawa_angle_integrals(gp, wpl, ax, Lm, pp, p, I1, I2, I3, R);
    const int M = NQ + 1;
    for (int c = 0; c < n_ch; ++c) {
        const MiChanDev ch = chans[c];
        const int n = ch.n;
        for (int al = 0; al < ch.K; ++al)
            for (int be = 0; be < ch.K; ++be) {
                double tv[kMaxTerms];
                potential_terms<GEN>(gp, ch.s, ch.J, ch.tz, mi_lblock(ch, al), mi_lblock(ch, be), pp, p, I1, I2, I3,
                                     R, tv);
                for (int t = 0; t < n_terms; ++t) {
                    double *V = Vg + ch.vg_off + (size_t)t * n * n;
                    V[(size_t)(al * M + i) * n + (be * M + j)] = tv[t];
                    V[(size_t)(be * M + j) * n + (al * M + i)] = tv[t];
                }
            }
    }
}

// On-shell column of V_t at each energy: V_t^{l_a l_b}(q_i, p_e) for q_i = k_i
// (i < N_Q) and q_N = p_e.  Von of channel c: [n_I][n_terms][K][K][N_Q+1] at
// c.von_off.  One thread per (energy, i).
template <int GEN>
__global__ void __launch_bounds__(128) k_mi_pot_onshell(const MiChanDev *chans, int n_ch, int NQ, const double *kg,
                                                        int n_I, const double *e_int, int Lmax, const double *gp,
                                                        const double *angx, const double *angw, int n_terms,
                                                        double *Von)
{
    __shared__ double wpl[kAngleQ][kLmaxReg + 1];
    __shared__ double ax[kAngleQ];
    const int Lm = (Lmax < kLmaxReg) ? Lmax : kLmaxReg;
    if (GEN == WPCD_GEN_YUKAWA) {
        angle_tables(angx, angw, Lm, wpl, ax);
        __syncthreads();
    }
    const int M = NQ + 1;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n_I * M) return;
    const int e = b / M, i = b - e * M;
    const double p = sqrt(kMn * e_int[e] / 2.0) / kHbarc;
    const double pp = i < NQ ? kg[i] : p;
    double I1[kLmaxReg + 1], I2[kLmaxReg + 1], I3[kLmaxReg + 1], R = 0.0;
    if (GEN == WPCD_GEN_YUKAWA) yukawa_angle_integrals(gp, wpl, ax, Lm, pp, p, I1, I2, I3, R);
    for (int c = 0; c < n_ch; ++c) {
        const MiChanDev ch = chans[c];
        for (int al = 0; al < ch.K; ++al)
            for (int be = 0; be < ch.K; ++be) {
                double tv[kMaxTerms];
                potential_terms<GEN>(gp, ch.s, ch.J, ch.tz, mi_lblock(ch, al), mi_lblock(ch, be), pp, p, I1, I2, I3,
                                     R, tv);
                for (int t = 0; t < n_terms; ++t)
                    Von[ch.von_off + ((((size_t)e * n_terms + t) * ch.K + al) * ch.K + be) * M + i] = tv[t];
            }
    }
}

cudaError_t launch_mi_pot(int gen, const MiChanDev *chans_dev, int n_ch, int NQ, const double *kg, int Lmax,
                          const double *gp_dev, const double *angx, const double *angw, int n_terms, double *Vg,
                          cudaStream_t st)
{
    const long long pairs = (long long)NQ * (NQ + 1) / 2;
    const unsigned grid = (unsigned)((pairs + 127) / 128);
    if (gen == WPCD_GEN_YUKAWA)
        k_mi_pot_grid<WPCD_GEN_YUKAWA><<<grid, 128, 0, counted(st)>>>(chans_dev, n_ch, NQ, kg, Lmax, gp_dev, angx, angw,
                                                             n_terms, Vg);
    else
        k_mi_pot_grid<WPCD_GEN_YAMAGUCHI><<<grid, 128, 0, counted(st)>>>(chans_dev, n_ch, NQ, kg, 0, gp_dev, nullptr, nullptr,
                                                                n_terms, Vg);
    return cudaGetLastError();
}

cudaError_t launch_mi_onshell(int gen, const MiChanDev *chans_dev, int n_ch, int NQ, const double *kg, int n_I,
                              const double *e_int, int Lmax, const double *gp_dev, const double *angx,
                              const double *angw, int n_terms, double *Von, cudaStream_t st)
{
    const unsigned grid = (unsigned)((n_I * (NQ + 1) + 127) / 128);
    if (gen == WPCD_GEN_YUKAWA)
        k_mi_pot_onshell<WPCD_GEN_YUKAWA><<<grid, 128, 0, counted(st)>>>(chans_dev, n_ch, NQ, kg, n_I, e_int, Lmax, gp_dev, angx,
                                                                angw, n_terms, Von);
    else
        k_mi_pot_onshell<WPCD_GEN_YAMAGUCHI><<<grid, 128, 0, counted(st)>>>(chans_dev, n_ch, NQ, kg, n_I, e_int, 0, gp_dev,
                                                                   nullptr, nullptr, n_terms, Von);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------- solve
// Shared memory of one CTA for matrices up to n: A float [n][ld] | D double [M] |
// b, x, r double [2][n] | y float [2][n] | perm int [n, even] | reduction double [64].
__host__ __device__ inline int mi_ld(int n) { return (n + 3) & ~3; }  // rows padded to 16 bytes (float4 access)

__host__ __device__ inline size_t mi_smem(int n, int M)
{
    size_t a = (size_t)n * mi_ld(n) * 4;
    a = (a + 15) & ~(size_t)15;
    return a + (size_t)M * 8 + 3 * (size_t)2 * n * 8 + (size_t)2 * n * 4 + (size_t)(n + (n & 1)) * 4 + 64 * 8;
}

size_t mi_smem_bytes(int n, int M) { return mi_smem(n, M); }

// Maximum over the CTA that propagates NaN (fmax would drop it).
__device__ __forceinline__ double nan_max(double a, double b) { return (b > a || b != b) ? b : a; }

__device__ __forceinline__ double mi_block_max(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v = nan_max(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = nan_max(t, red[w]);
    return t;
}

__device__ __forceinline__ double mi_block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

// T = (1 + i pi mu p K)^-1 K of the on-shell K (2 x 2 frame) and the phases of S.
__device__ __forceinline__ void mi_phases(int K, double p, const double *Km, double *po)
{
    const double g = kPi * kMu * p;
    double T[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (K == 1) {
        const double dre = 1.0, dim = g * Km[0], dd = dre * dre + dim * dim;
        T[0] = Km[0] * dre / dd;
        T[1] = -Km[0] * dim / dd;
    } else {
        // M = 1 + i g K (complex 2 x 2); T = M^-1 K
        const double m00r = 1.0, m00i = g * Km[0], m01i = g * Km[1], m10i = g * Km[2], m11r = 1.0,
                     m11i = g * Km[3];
        // det = m00 m11 - m01 m10
        const double detr = m00r * m11r - m00i * m11i + m01i * m10i;
        const double deti = m00r * m11i + m00i * m11r;
        const double dd = detr * detr + deti * deti;
        // inverse = [[m11, -m01], [-m10, m00]] / det
        const double ir = detr / dd, ii = -deti / dd;
        const double inv[8] = {m11r * ir - m11i * ii, m11r * ii + m11i * ir,  // (0,0)
                               m01i * ii, -m01i * ir,                          // (0,1) = -i m01i / det
                               m10i * ii, -m10i * ir,                          // (1,0)
                               m00r * ir - m00i * ii, m00r * ii + m00i * ir};  // (1,1)
        for (int a = 0; a < 2; ++a)
            for (int bb = 0; bb < 2; ++bb) {
                double re = 0.0, im = 0.0;
                for (int k = 0; k < 2; ++k) {
                    re += inv[(a * 2 + k) * 2] * Km[k * 2 + bb];
                    im += inv[(a * 2 + k) * 2 + 1] * Km[k * 2 + bb];
                }
                T[(a * 2 + bb) * 2] = re;
                T[(a * 2 + bb) * 2 + 1] = im;
            }
    }
    phases_of_T(K, p, T, po);
}

// The most refinement steps of a (sample, channel), -1 (a failed system) sticking.
__device__ __forceinline__ void mi_worst(int *status, int worst)
{
    if (worst < 0) {
        atomicExch(status, -1);
        return;
    }
    int old = atomicAdd(status, 0);
    while (old >= 0 && old < worst) {
        const int was = atomicCAS(status, old, worst);
        if (was == old) break;
        old = was;
    }
}

// Items (sample, work channel, chunk of ne energies) of one block size; CTA
// blockIdx.x owns scratch slot Vs + blockIdx.x n^2 and walks the items item =
// blockIdx.x, + gridDim.x, ...  redo (may be NULL; with ne = 1): only the systems
// with redo[(smp n_ch_total + channel) n_I + energy] != 0.  status is zero on entry.
// Outputs per (sample, channel, energy): phases ph [S][n_ch][n_I][3] (degrees)
// and, if k_out, the on-shell K [S][n_ch][n_I][2][2].
__global__ void __launch_bounds__(kMiThreads) k_mi_solve(const MiChanDev *chans, const int *work_ch, int n_work,
                                                         int n_ch_total, int n_samples, int NQ, const double *kg,
                                                         const double *wg, int n_terms, const double *coeffs,
                                                         const double *Vg, const double *Von, int n_I,
                                                         const double *e_int, double *Vs_all, double *ph,
                                                         double *k_out, int *status, int *err, int ne, int n_chunk,
                                                         const int *redo)
{
    const int M = NQ + 1;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    if ((size_t)dyn_smem_bytes() < mi_smem(chans[work_ch[0]].n, M)) {  // launch/layout mismatch
        if (tid == 0) record_error(err, kDevBadSize);
        return;
    }
    extern __shared__ __align__(16) double mi_sm[];
    unsigned char *sb = reinterpret_cast<unsigned char *>(mi_sm);
    const int n0 = chans[work_ch[0]].n;  // every work channel of a launch has the same n
    const int ld = mi_ld(n0);
    size_t off = ((size_t)n0 * ld * 4 + 15) & ~(size_t)15;
    float *A = reinterpret_cast<float *>(sb);
    double *D = reinterpret_cast<double *>(sb + off);
    double *bv = D + M, *xv = bv + 2 * n0, *rv = xv + 2 * n0;
    float *yv = reinterpret_cast<float *>(rv + 2 * n0);
    int *perm = reinterpret_cast<int *>(yv + 2 * n0);
    double *red = reinterpret_cast<double *>(perm + n0 + (n0 & 1));
    double *Vs = Vs_all + (size_t)blockIdx.x * 2 * n0 * n0;  // V, then the FP64 fallback matrix

    for (long long item = blockIdx.x; item < (long long)n_samples * n_work * n_chunk; item += gridDim.x) {
        const int sw = (int)(item / n_chunk), chunk = (int)(item - (long long)sw * n_chunk);
        const int smp = sw / n_work, cidx = work_ch[sw - smp * n_work];
        if (redo && redo[((size_t)smp * n_ch_total + cidx) * n_I + chunk] == 0) continue;
        const MiChanDev ch = chans[cidx];
        const int n = ch.n, K = ch.K;
        const double *cf = coeffs ? coeffs + (size_t)smp * (n_terms - 1) : nullptr;
        const double *Vgc = Vg + ch.vg_off;
        // V = V0 + sum_a c_a V_a on the grid part (the on-shell rows follow per energy)
        for (int e = tid; e < n * n; e += nt) {
            const int r = e / n, c = e - r * n;
            if (r % M == NQ || c % M == NQ) continue;
            double v = Vgc[e];
            for (int t = 1; t < n_terms; ++t) v = fma(cf[t - 1], Vgc[(size_t)t * n * n + e], v);
            Vs[e] = v;
        }
        int worst = 0;
        const int ie1 = min(n_I, (chunk + 1) * ne);
        for (int ie = chunk * ne; ie < ie1; ++ie) {
            const double p = sqrt(kMn * e_int[ie] / 2.0) / kHbarc, p2 = p * p;
            // D and the on-shell rows and columns of V at this energy
            double part = 0.0;
            for (int j = tid; j < NQ; j += nt) {
                const double den = p2 - kg[j] * kg[j];
                D[j] = wg[j] * kg[j] * kg[j] * 2.0 * kMu / den;
                part += wg[j] / den;
            }
            const double sum = mi_block_sum(part, red);
            if (tid == 0) D[NQ] = -2.0 * kMu * p2 * sum;
            const double *Vo = Von + ch.von_off + (size_t)ie * n_terms * K * K * M;
            for (int e = tid; e < K * K * M; e += nt) {
                const int al = e / (K * M), be = (e / M) % K, i = e % M;
                double v = Vo[e];
                for (int t = 1; t < n_terms; ++t) v = fma(cf[t - 1], Vo[(size_t)t * K * K * M + e], v);
                Vs[(size_t)(al * M + i) * n + (be * M + NQ)] = v;  // V^{l_a l_b}(q_i, p)
                Vs[(size_t)(be * M + NQ) * n + (al * M + i)] = v;  // V^{l_b l_a}(p, q_i), the same value
            }
            __syncthreads();
            // A = 1 - V D (FP32), right-hand sides b_bb = V[:, (bb, N)] (FP64)
            for (int e = tid; e < n * n; e += nt) {
                const int r = e / n, c = e - r * n;
                A[(size_t)r * ld + c] = (float)((r == c ? 1.0 : 0.0) - Vs[e] * D[c % M]);
            }
            for (int e = tid; e < K * n; e += nt) {
                const int bb = e / n, r = e - bb * n;
                bv[bb * n0 + r] = Vs[(size_t)r * n + (bb * M + NQ)];
                xv[bb * n0 + r] = 0.0;
                rv[bb * n0 + r] = bv[bb * n0 + r];
            }
            for (int r = tid; r < n; r += nt) {
                perm[r] = r;
                for (int c = n; c < ld; ++c) A[(size_t)r * ld + c] = 0.0f;
            }
            __syncthreads();
            // In-place Gauss-Jordan inversion with partial pivoting (rows swapped
            // in place, perm[] tracks them): afterwards A holds W with
            // W (P r) = (1 - V D)^-1 r, (P r)_k = r_perm[k].
            for (int k = 0; k < n; ++k) {
                if (warp == 0) {
                    float best = -1.0f;
                    int bi = k;
                    for (int r = k + lane; r < n; r += 32) {
                        const float v = fabsf(A[(size_t)r * ld + k]);
                        if (v > best) { best = v; bi = r; }
                    }
                    for (int o = 16; o > 0; o >>= 1) {
                        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
                    }
                    if (lane == 0) {
                        reinterpret_cast<int *>(red)[0] = bi;
                        reinterpret_cast<float *>(red)[1] = A[(size_t)bi * ld + k];  // the pivot
                    }
                }
                __syncthreads();
                const int pr = reinterpret_cast<int *>(red)[0];
                const float rinv = 1.0f / reinterpret_cast<float *>(red)[1];
                if (pr != k) {
                    for (int c = tid; c < n; c += nt) {
                        const float t = A[(size_t)k * ld + c];
                        A[(size_t)k * ld + c] = A[(size_t)pr * ld + c];
                        A[(size_t)pr * ld + c] = t;
                    }
                    if (tid == 0) {
                        const int t = perm[k];
                        perm[k] = perm[pr];
                        perm[pr] = t;
                    }
                    __syncthreads();
                }
                // the other rows' column-k entries, then row k divided by the pivot
                for (int r = tid; r < n; r += nt) yv[r] = r == k ? 0.0f : A[(size_t)r * ld + k];
                for (int c = tid; c < n; c += nt) A[(size_t)k * ld + c] = c == k ? rinv : A[(size_t)k * ld + c] * rinv;
                __syncthreads();
                // eliminate column k from every other row (one warp per row); the
                // column-k entry becomes -f / pivot (the in-place inverse column)
                // (four columns per lane: the padding columns n..ld-1 stay finite and unused)
                const float4 *Ak4 = reinterpret_cast<const float4 *>(A + (size_t)k * ld);
                for (int r = warp; r < n; r += nw) {
                    if (r == k) continue;
                    const float f = yv[r];
                    float4 *Ar4 = reinterpret_cast<float4 *>(A + (size_t)r * ld);
                    for (int c = lane; c < (ld >> 2); c += 32) {
                        const float4 a = Ar4[c], b = Ak4[c];
                        Ar4[c] = make_float4(fmaf(-f, b.x, a.x), fmaf(-f, b.y, a.y), fmaf(-f, b.z, a.z), fmaf(-f, b.w, a.w));
                    }
                    __syncwarp();  // the lane that updated column k has written it
                    if (lane == 0) A[(size_t)r * ld + k] = -f * A[(size_t)k * ld + k];
                }
                __syncthreads();
            }
            // iterative refinement: y = W (P r) in FP32, x += y, r = b - (x - V D x) in FP64
            bool conv = false;
            int it = 0;
            double ym_prev = 0.0;
            for (; it < kMiMaxRefine && !conv; ++it) {
                double ym = 0.0, xm = 0.0;  // NaN-propagating maxima: a NaN never passes as converged
                for (int r = warp; r < n; r += nw)
                    for (int bb = 0; bb < K; ++bb) {
                        float acc = 0.0f;
                        for (int c = lane; c < n; c += 32)
                            acc = fmaf(A[(size_t)r * ld + c], (float)rv[bb * n0 + perm[c]], acc);
                        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                        if (lane == 0) {
                            const double y = (double)acc, xn = xv[bb * n0 + r] + y;
                            xv[bb * n0 + r] = xn;
                            const double ay = fabs(y), ax = fabs(xn);
                            ym = (ay > ym || ay != ay) ? ay : ym;
                            xm = (ax > xm || ax != ax) ? ax : xm;
                        }
                    }
                ym = mi_block_max(ym, red);
                xm = mi_block_max(xm, red + 32);
                // done when the correction is negligible, or when it has stopped
                // shrinking at the accuracy floor of the FP64 residual (about
                // cond(A) u_64, the accuracy of an FP64 factorisation too)
                conv = ym <= 1e-14 * xm || (it > 0 && ym > 0.25 * ym_prev && ym <= 1e-9 * xm);
                ym_prev = ym;
                if (conv) break;  // (uniform: conv comes from CTA-wide maxima)
                // r = b - x + V (D x): one warp per row, lanes over the columns
                for (int r = warp; r < n; r += nw)
                    for (int bb = 0; bb < K; ++bb) {
                        double acc = 0.0;
                        const double *Vr = Vs + (size_t)r * n;
                        double acc2 = 0.0;  // two chains keep two loads in flight
                        int c = lane;
                        for (; c + 32 < n; c += 64) {
                            const int c1 = c + 32;
                            acc = fma(Vr[c] * D[c < M ? c : c - M], xv[bb * n0 + c], acc);
                            acc2 = fma(Vr[c1] * D[c1 < M ? c1 : c1 - M], xv[bb * n0 + c1], acc2);
                        }
                        if (c < n) acc = fma(Vr[c] * D[c < M ? c : c - M], xv[bb * n0 + c], acc);
                        acc += acc2;
                        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                        if (lane == 0) rv[bb * n0 + r] = bv[bb * n0 + r] - xv[bb * n0 + r] + acc;
                    }
                __syncthreads();
            }
            int steps = conv ? it + 1 : it;  // the loop left by break on convergence
            if (!conv) {
                // The FP32 inverse is too inexact for refinement to converge
                // (cond(A) u_32 ~ 1): solve this system by FP64 Gauss-Jordan
                // elimination with partial pivoting in the slot's second FP64
                // matrix (global memory; rare, so plain), right-hand sides
                // carried along.
                double *G = Vs + (size_t)n0 * n0;
                for (int e = tid; e < n * n; e += nt) {
                    const int r = e / n, c = e - r * n;
                    G[e] = (r == c ? 1.0 : 0.0) - Vs[e] * D[c < M ? c : c - M];
                }
                for (int e = tid; e < K * n; e += nt) xv[(e / n) * n0 + e % n] = bv[(e / n) * n0 + e % n];
                __syncthreads();
                bool ok = true;
                for (int k = 0; k < n; ++k) {
                    if (warp == 0) {
                        double best = -1.0;
                        int bi = k;
                        for (int r = k + lane; r < n; r += 32) {
                            const double v = fabs(G[(size_t)r * n + k]);
                            if (v > best) { best = v; bi = r; }
                        }
                        for (int o = 16; o > 0; o >>= 1) {
                            const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
                        }
                        if (lane == 0) reinterpret_cast<int *>(red)[0] = bi;
                    }
                    __syncthreads();
                    const int pr = reinterpret_cast<int *>(red)[0];
                    if (pr != k) {
                        for (int c = tid; c < n; c += nt) {
                            const double t = G[(size_t)k * n + c];
                            G[(size_t)k * n + c] = G[(size_t)pr * n + c];
                            G[(size_t)pr * n + c] = t;
                        }
                        if (tid < K) {
                            const double t = xv[tid * n0 + k];
                            xv[tid * n0 + k] = xv[tid * n0 + pr];
                            xv[tid * n0 + pr] = t;
                        }
                    }
                    __syncthreads();
                    const double piv = G[(size_t)k * n + k];
                    if (piv == 0.0) ok = false;
                    const double rinv = piv != 0.0 ? 1.0 / piv : 0.0;
                    __syncthreads();  // every thread holds the pivot before row k is rescaled
                    for (int c = tid; c < n; c += nt) G[(size_t)k * n + c] *= rinv;
                    if (tid < K) xv[tid * n0 + k] *= rinv;
                    __syncthreads();
                    for (int r = warp; r < n; r += nw) {
                        if (r == k) continue;
                        const double f = G[(size_t)r * n + k];
                        __syncwarp();
                        for (int c = lane; c < n; c += 32) G[(size_t)r * n + c] -= f * G[(size_t)k * n + c];
                        if (lane < K) xv[lane * n0 + r] -= f * xv[lane * n0 + k];
                    }
                    __syncthreads();
                }
                if (ok) {
                    conv = true;
                    steps = kMiMaxRefine + 1;  // marks the FP64 fallback in the status
                }
            }
            if (!conv) worst = -1;
            else if (worst >= 0 && steps > worst) worst = steps;
            if (tid == 0) {
                // on-shell K and its phases
                double Km[4] = {0, 0, 0, 0};
                for (int a = 0; a < K; ++a)
                    for (int bb = 0; bb < K; ++bb) Km[a * 2 + bb] = xv[bb * n0 + a * M + NQ];
                const size_t o = ((size_t)smp * n_ch_total + cidx) * n_I + ie;
                mi_phases(K, p, Km, ph + o * 3);
                if (k_out)
                    for (int k = 0; k < 4; ++k) k_out[o * 4 + k] = Km[k];
            }
            __syncthreads();
        }
        if (tid == 0) {
            mi_worst(&status[(size_t)smp * n_ch_total + cidx], worst);
            if (worst < 0) record_error(err, kDevNoConverge);
        }
    }
}

// status zeroed by the caller; n_chunk chunks of ne energies per (sample, channel).
cudaError_t launch_mi_solve(const MiChanDev *chans_dev, const int *work_dev, int n_work, int n, int n_ch_total,
                            int n_samples, int NQ, const double *kg, const double *wg, int n_terms,
                            const double *coeffs, const double *Vg, const double *Von, int n_I, const double *e_int,
                            double *Vs, int slots, double *ph, double *k_out, int *status, int *err, cudaStream_t st,
                            int ne, const int *redo)
{
    const size_t smem = mi_smem(n, NQ + 1);
    if (smem > 227 * 1024 || ne < 1 || (redo && ne != 1)) return cudaErrorInvalidValue;
    raise_smem_limit((const void *)k_mi_solve, smem);
    k_mi_solve<<<slots, kMiThreads, smem, counted(st)>>>(chans_dev, work_dev, n_work, n_ch_total, n_samples, NQ, kg, wg, n_terms,
                                                coeffs, Vg, Von, n_I, e_int, Vs, ph, k_out, status, err, ne,
                                                (n_I + ne - 1) / ne, redo);
    return cudaGetLastError();
}

int mi_slots_per_sm(int n, int NQ)
{
    const size_t smem = mi_smem(n, NQ + 1);
    raise_smem_limit((const void *)k_mi_solve, smem);
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_mi_solve, kMiThreads, smem);
    return blocks;
}

// ------------------------------------------------------------------------------------- solve, all energies at once
// With w = D y, (1 - V D) y = r reads (D^-1 - V) w = r, and on the grid
//     D_j^-1 = (p^2 - k_j^2) / (2 mu w_j k_j^2)
// is affine in p^2: V - D^-1 = S^-1 (Ht - p^2) S^-1 with S_j = sqrt(2 mu w_j) k_j and
// Ht = diag(k^2) + S V S, the same for every energy.  One eigendecomposition
// Ht = Q diag(lambda) Q^T per (sample, channel) thus inverts the grid part at every
// energy, M^-1 = S Q (lambda - p^2)^-1 Q^T S, and the on-shell point is a K x K border:
//     w_p = (1/D_N - R)^-1 (r_p - v^T M^-1 r_g),  w_g = -M^-1 (r_g + v w_p),
//     R = V_pp - v^T M^-1 v,  v = V(grid, p).
// Q is held in FP32 and lambda - p^2 formed in FP64, so every direction is
// inverted to FP32's relative accuracy, close poles included; FP64 residuals
// of the original system then refine the solution to FP64 as for the FP32
// inverse of k_mi_solve (which takes the systems that do not converge here).
// Per energy this costs K n^2 FP64 multiply-adds a residual (the bound: two or
// three of them) instead of an n^3 elimination whose n steps wait for each other:
// 64 samples x 15 channels x 32 energies, N_Q = 96: 134.4 -> 16.4 ms, errors against
// 64 bits unchanged (the eigendecompositions are 10 ms of it).  The rest of the pass is
// kept off the FP64 pipe where it can be: -w / D as a product with (k^2 - p^2) / (2 mu w
// k^2), one reciprocal for D and the sum in D_N, V summed over one triangle (20.9 -> 20.1).

// S V_t S over the grid and k^2, from the grid terms of every channel.
__global__ void __launch_bounds__(256) k_mi_scale(const MiChanDev *chans, int n_ch, int NQ, const double *kg,
                                                  const double *wg, int n_terms, const double *Vg, double *Vt,
                                                  const long long *vt_off, double *k2)
{
    const int c = blockIdx.y;
    const MiChanDev ch = chans[c];
    const int M = NQ + 1, ng = ch.K * NQ;
    if (c == 0)
        for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < NQ; j += (long long)gridDim.x * blockDim.x)
            k2[j] = kg[j] * kg[j];
    const long long total = (long long)n_terms * ng * ng;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int t = (int)(e / ((long long)ng * ng)), rc = (int)(e - (long long)t * ng * ng), r = rc / ng, q = rc - r * ng;
        const int i = r % NQ, j = q % NQ;
        const double v = Vg[ch.vg_off + ((size_t)t * ch.n + (r / NQ) * M + i) * ch.n + (q / NQ) * M + j];
        const double si = sqrt(2.0 * kMu * wg[i]) * kg[i], sj = sqrt(2.0 * kMu * wg[j]) * kg[j];
        Vt[vt_off[c] + e] = v * (si * sj);
    }
}

cudaError_t launch_mi_scale(const MiChanDev *chans_dev, int n_ch, int NQ, const double *kg, const double *wg, int n_terms,
                            const double *Vg, double *Vt, const long long *vt_off, double *k2, cudaStream_t st)
{
    k_mi_scale<<<dim3(64, n_ch), 256, 0, counted(st)>>>(chans_dev, n_ch, NQ, kg, wg, n_terms, Vg, Vt, vt_off, k2);
    return cudaGetLastError();
}

constexpr int kMeCols = 8;      // right-hand sides a pass carries: 8 / K energies
// 16 warps for coupled channels (14 row-block tasks of the residual), 8 for uncoupled ones (7 to 8),
// two or three of which share an SM
__host__ __device__ inline int me_threads(int K) { return K == 2 ? 512 : 256; }
constexpr int kMeMaxRefine = 10;

__host__ __device__ inline int me_ldq(int ng) { return ng | 1; }  // odd row pitch of Q: conflict-free along both indices

// Q float [ng][ldq] | z, x, b double [ng][8] | T = M^-1 v, u, h float [ng][8] | lambda, S double [ng] |
// 1 / (2 mu w k^2) double [NQ] | D double [NQ][8 / K] | per column: p^2, D_N, x_p, r_p, y_p ... double [8 x 16] | maxima double [16][16]
__host__ __device__ inline size_t me_smem(int ng, int NQ, int K)
{
    size_t b = ((size_t)ng * me_ldq(ng) * 4 + 15) & ~(size_t)15;
    b += (size_t)3 * ng * kMeCols * 8 + (size_t)3 * ng * kMeCols * 4 + (size_t)2 * ng * 8;
    b += (size_t)(NQ + (NQ & 1)) * 8 + (size_t)NQ * (kMeCols / K) * 8 + (size_t)8 * 16 * 8 + (size_t)32 * kMeCols * 8;
    return b;
}

// u = Q^T (S o rhs) in FP32, divided by lambda - p^2, then h = S o (Q u): h = M^-1 rhs
// for the pass's columns (rhs FP64 [ng][8], h float [ng][8]).
__device__ __forceinline__ void me_apply(int ng, int NQ, int ldq, const float *Q, const double *lam, const double *Sg,
                                         const double *p2c, const double *rhs, float *u, float *h)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    // h as the FP32 copy of S o rhs first
    for (int e = tid; e < ng * kMeCols; e += nt) h[e] = (float)(rhs[e] * Sg[e / kMeCols]);
    __syncthreads();
    for (int task = tid; task < ng * 2; task += nt) {  // (eigenvector i, four columns)
        const int q = task / ng, i = task - q * ng;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r = 0; r < ng; ++r) {
            const float v = Q[r * ldq + i];
            const float4 b = *reinterpret_cast<const float4 *>(h + r * kMeCols + 4 * q);
            a.x = fmaf(v, b.x, a.x);
            a.y = fmaf(v, b.y, a.y);
            a.z = fmaf(v, b.z, a.z);
            a.w = fmaf(v, b.w, a.w);
        }
        const double l = lam[i], *p = p2c + 4 * q;
        a.x *= 1.0f / (float)(l - p[0]);
        a.y *= 1.0f / (float)(l - p[1]);
        a.z *= 1.0f / (float)(l - p[2]);
        a.w *= 1.0f / (float)(l - p[3]);
        *reinterpret_cast<float4 *>(u + i * kMeCols + 4 * q) = a;
    }
    __syncthreads();
    for (int task = tid; task < ng * 2; task += nt) {  // (grid point r, four columns)
        const int q = task / ng, r = task - q * ng;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = 0; i < ng; ++i) {
            const float v = Q[r * ldq + i];
            const float4 b = *reinterpret_cast<const float4 *>(u + i * kMeCols + 4 * q);
            a.x = fmaf(v, b.x, a.x);
            a.y = fmaf(v, b.y, a.y);
            a.z = fmaf(v, b.z, a.z);
            a.w = fmaf(v, b.w, a.w);
        }
        const float s = (float)Sg[r];
        *reinterpret_cast<float4 *>(h + r * kMeCols + 4 * q) = make_float4(s * a.x, s * a.y, s * a.z, s * a.w);
    }
    __syncthreads();
}

// One CTA per (sample, work channel), slot Vs + blockIdx.x ng^2 for its V on the grid.
__global__ void __launch_bounds__(512, 1) k_mi_energies(const MiChanDev *chans, const ChanDev *eig_ch, const int *work_ch, int n_work,
                                                            int n_ch_total, int sample0, int n_samples, int NQ,
                                                            const double *kg, const double *wg, int n_terms,
                                                            const double *coeffs, const double *Vg, const double *Von,
                                                            int n_I, const double *e_int, const double *eps_all,
                                                            const double *Q_all, const int *eig_status,
                                                            const int *eig_err, double *Vs_all, double *ph,
                                                            double *k_out, int *status, int *redo, int *err)
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int K = chans[work_ch[0]].K, M = NQ + 1, ng = K * NQ, ldq = me_ldq(ng), EC = kMeCols / K;
    if ((size_t)dyn_smem_bytes() < me_smem(ng, NQ, K)) {
        if (tid == 0) record_error(err, kDevBadSize);
        return;
    }
    extern __shared__ __align__(16) unsigned char me_sm[];
    float *Q = reinterpret_cast<float *>(me_sm);
    double *z = reinterpret_cast<double *>(me_sm + (((size_t)ng * ldq * 4 + 15) & ~(size_t)15));  // D x, or a right-hand side
    double *x = z + (size_t)ng * kMeCols, *b = x + (size_t)ng * kMeCols;
    double *lam = b + (size_t)ng * kMeCols, *Sg = lam + ng;
    double *iw = Sg + ng;                                  // [NQ]: 1 / (2 mu w k^2)
    double *D = iw + NQ + (NQ & 1);                        // [NQ][EC] (T, u, h further on need 16 bytes)
    double *p2c = D + (size_t)NQ * EC;                     // per column: p^2
    double *DNc = p2c + 8, *xp = DNc + 8, *rp = xp + 16, *Rm = rp + 16, *Vpp = Rm + 16, *wp = Vpp + 16;  // [8][K] each
    double *ymx = wp + 16, *ypr = ymx + 8;                 // maxima of the correction, this step's and the last one's
    int *nst = reinterpret_cast<int *>(ypr + 8);           // per column: 0, or the step it converged at
    double *red = p2c + 8 * 16;                            // [32][8]
    float *T = reinterpret_cast<float *>(red + 32 * kMeCols), *u = T + (size_t)ng * kMeCols, *h = u + (size_t)ng * kMeCols;
    double *V = Vs_all + (size_t)blockIdx.x * ng * ng;

    for (int item = blockIdx.x; item < n_samples * n_work; item += gridDim.x) {
        const int smp = sample0 + item / n_work, cidx = work_ch[item % n_work];
        const MiChanDev ch = chans[cidx];
        const ChanDev ec = eig_ch[cidx];
        const double *cf = coeffs ? coeffs + (size_t)smp * (n_terms - 1) : nullptr;
        const double *Vgc = Vg + ch.vg_off;
        const double *Qg = Q_all + ec.c_off + (size_t)(smp - sample0) * ng * ng;
        const double *lg = eps_all + ec.eps_off + (size_t)(smp - sample0) * ng;
        // eigenpairs that a solve did not converge to, or a product that timed out did not write, could
        // pass for a solution (vectors of zeros give a correction of zero): all energies by elimination
        if (*eig_err != 0 || eig_status[(size_t)(smp - sample0) * n_ch_total + cidx] < 0) {
            for (int ie = tid; ie < n_I; ie += nt) redo[((size_t)smp * n_ch_total + cidx) * n_I + ie] = 1;
            if (tid == 0) status[(size_t)smp * n_ch_total + cidx] = 0;
            continue;
        }
        __syncthreads();  // the last item is done with shared memory
        for (int r = warp; r < ng; r += nw) {  // V is symmetric: the upper triangle, mirrored
            const size_t orow = (size_t)((r / NQ) * M + r % NQ) * ch.n;
            for (int c = lane; c < ng; c += 32) {
                Q[r * ldq + c] = (float)Qg[(size_t)r * ng + c];
                if (c < r) continue;
                const size_t o = orow + (c / NQ) * M + c % NQ;
                double v = Vgc[o];
                for (int t = 1; t < n_terms; ++t) v = fma(cf[t - 1], Vgc[(size_t)t * ch.n * ch.n + o], v);
                V[(size_t)r * ng + c] = v;
                V[(size_t)c * ng + r] = v;
            }
        }
        for (int i = tid; i < ng; i += nt) {
            lam[i] = lg[i];
            Sg[i] = sqrt(2.0 * kMu * wg[i % NQ]) * kg[i % NQ];
            if (i < NQ) iw[i] = 1.0 / (wg[i] * kg[i] * kg[i] * 2.0 * kMu);
        }
        int worst = 0;
        for (int e0 = 0; e0 < n_I; e0 += EC) {
            // columns c = (energy el = c / K, right-hand side bb = c % K); past the last energy the last one again
            __syncthreads();
            for (int el = warp; el < EC; el += nw) {
                const int ie = min(e0 + el, n_I - 1);
                const double p = sqrt(kMn * e_int[ie] / 2.0) / kHbarc, p2 = p * p;
                double part = 0.0;
                for (int j = lane; j < NQ; j += 32) {
                    const double rden = 1.0 / (p2 - kg[j] * kg[j]);
                    D[j * EC + el] = wg[j] * kg[j] * kg[j] * 2.0 * kMu * rden;
                    part = fma(wg[j], rden, part);
                }
                for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
                if (lane < K) {
                    p2c[el * K + lane] = p2;
                    DNc[el * K + lane] = -2.0 * kMu * p2 * part;
                }
            }
            // v_{(a, i), bb} at the column's energy, V_pp, and the first right-hand side b = v
            for (int e = tid; e < (ng + K) * kMeCols; e += nt) {
                const int r = e / kMeCols, c = e - r * kMeCols, el = c / K, bb = c - el * K;
                const int ie = min(e0 + el, n_I - 1);
                const int a = r < ng ? r / NQ : r - ng, i = r < ng ? r % NQ : NQ;
                const double *Vo = Von + ch.von_off + (size_t)ie * n_terms * K * K * M + (size_t)(a * K + bb) * M + i;
                double v = Vo[0];
                for (int t = 1; t < n_terms; ++t) v = fma(cf[t - 1], Vo[(size_t)t * K * K * M], v);
                if (r < ng) {
                    b[r * kMeCols + c] = v;
                    x[r * kMeCols + c] = 0.0;
                } else {
                    Vpp[c * 2 + a] = v;
                    rp[c * 2 + a] = v;
                    xp[c * 2 + a] = 0.0;
                }
            }
            if (tid < kMeCols) nst[tid] = 0;
            __syncthreads();
            me_apply(ng, NQ, ldq, Q, lam, Sg, p2c, b, u, h);
            for (int e = tid; e < ng * kMeCols; e += nt) T[e] = h[e];
            __syncthreads();
            // R = V_pp - v^T T, one warp per (column, row block)
            for (int w = warp; w < kMeCols * K; w += nw) {
                const int c = w / K, a = w - c * K, ca = (c / K) * K + a;  // v of block a at this energy: column ca
                double s = 0.0;
                for (int r = lane; r < ng; r += 32) s = fma(b[r * kMeCols + ca], (double)T[r * kMeCols + c], s);
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) Rm[c * 2 + a] = Vpp[c * 2 + a] - s;
            }
            __syncthreads();
            int it = 0;
            bool done = false;
            for (; it < kMeMaxRefine && !done; ++it) {
                if (it > 0) {
                    // h = M^-1 r for the residual in z
                    me_apply(ng, NQ, ldq, Q, lam, Sg, p2c, z, u, h);
                }
                // r_p - v^T h (the first step: h = T, so this is R), then w_p and the correction of x_p
                for (int w = warp; w < kMeCols * K; w += nw) {
                    const int c = w / K, a = w - c * K, ca = (c / K) * K + a;
                    double s = 0.0;
                    for (int r = lane; r < ng; r += 32) s = fma(b[r * kMeCols + ca], (double)h[r * kMeCols + c], s);
                    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if (lane == 0) wp[c * 2 + a] = rp[c * 2 + a] - s;
                }
                __syncthreads();
                if (tid < kMeCols) {
                    const int c = tid, k0 = (c / K) * K;
                    const double DN = DNc[c];
                    if (K == 1) {
                        wp[c * 2] = DN * wp[c * 2] / (1.0 - DN * Rm[c * 2]);
                    } else {  // (1 - D_N R) w = D_N s, R[a][b] = Rm of column b, block a
                        const double a00 = 1.0 - DN * Rm[k0 * 2], a01 = -DN * Rm[(k0 + 1) * 2], a10 = -DN * Rm[k0 * 2 + 1],
                                     a11 = 1.0 - DN * Rm[(k0 + 1) * 2 + 1];
                        const double det = a00 * a11 - a01 * a10, s0 = DN * wp[c * 2], s1 = DN * wp[c * 2 + 1];
                        wp[c * 2] = (a11 * s0 - a01 * s1) / det;
                        wp[c * 2 + 1] = (a00 * s1 - a10 * s0) / det;
                    }
                }
                __syncthreads();
                // y_g = -(h + T w_p) / D, y_p = w_p / D_N; x += y, z = D x, the maxima of |y| and |x|
                double ym[kMeCols / 4], xm[kMeCols / 4];  // this thread's columns are tid % 4, + 4
                for (int q = 0; q < kMeCols / 4; ++q) ym[q] = xm[q] = 0.0;
                for (int e = tid; e < ng * 4; e += nt) {
                    const int r = e >> 2, j = r % NQ;
                    const double k2 = kg[j] * kg[j], iwj = iw[j];
#pragma unroll
                    for (int q = 0; q < kMeCols / 4; ++q) {
                        const int c = (e & 3) + 4 * q, k0 = (c / K) * K;
                        float w = h[r * kMeCols + c];
                        double t = (double)w;
                        for (int a = 0; a < K; ++a) t = fma((double)T[r * kMeCols + k0 + a], wp[c * 2 + a], t);
                        const double y = t * ((k2 - p2c[c]) * iwj), xn = x[r * kMeCols + c] + y;  // -t / D
                        x[r * kMeCols + c] = xn;
                        z[r * kMeCols + c] = D[j * EC + c / K] * xn;
                        ym[q] = nan_max(ym[q], fabs(y));
                        xm[q] = nan_max(xm[q], fabs(xn));
                    }
                }
                // lanes with the same tid % 4 hold the same columns
#pragma unroll
                for (int q = 0; q < kMeCols / 4; ++q) {
                    for (int o = 16; o >= 4; o >>= 1) {
                        ym[q] = nan_max(ym[q], __shfl_xor_sync(0xffffffffu, ym[q], o));
                        xm[q] = nan_max(xm[q], __shfl_xor_sync(0xffffffffu, xm[q], o));
                    }
                    if (lane < 4) {
                        red[warp * kMeCols + lane + 4 * q] = ym[q];
                        red[(16 + warp) * kMeCols + lane + 4 * q] = xm[q];
                    }
                }
                __syncthreads();
                if (tid < kMeCols) {
                    const int c = tid;
                    double y = 0.0, xx = 0.0;
                    for (int w = 0; w < nw; ++w) {
                        y = nan_max(y, red[w * kMeCols + c]);
                        xx = nan_max(xx, red[(16 + w) * kMeCols + c]);
                    }
                    for (int a = 0; a < K; ++a) {
                        const double yp = wp[c * 2 + a] / DNc[c];
                        xp[c * 2 + a] += yp;
                        y = nan_max(y, fabs(yp));
                        xx = nan_max(xx, fabs(xp[c * 2 + a]));
                    }
                    const double pr = ypr[c];
                    ypr[c] = y;
                    ymx[c] = y;
                    // done when the correction is negligible, when the next one will be (it shrinks by the
                    // same factor y / pr again, to below the rounding of x), or when it has stopped shrinking at
                    // the accuracy floor of the FP64 residual
                    const bool conv = y <= 1e-14 * xx || (it > 0 && y <= 1e-3 * pr && y * y <= 2e-15 * xx * pr) ||
                                      (it > 0 && y > 0.25 * pr && y <= 1e-9 * xx);
                    if (conv && nst[c] == 0) nst[c] = it + 1;
                    if (!conv) nst[c] = 0;
                }
                __syncthreads();
                done = true;
                for (int c = 0; c < kMeCols; ++c) done &= nst[c] != 0;
                if (done) break;
                // z <- r = b - x + V (D x), grid part: lanes along the rows (V is symmetric: row c of V is
                // its column), four columns per thread; the results wait for everyone's reads of z
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
                const int rq = warp & 1, rr = (warp >> 1) * 32 + lane;  // one task a warp (the launch checks)
                if (rr < ng) {
                    const double *Vr = V + rr;
#pragma unroll 4
                    for (int c = 0; c < ng; ++c) {
                        const double v = Vr[(size_t)c * ng];
                        const double2 z0 = *reinterpret_cast<const double2 *>(z + c * kMeCols + 4 * rq);
                        const double2 z1 = *reinterpret_cast<const double2 *>(z + c * kMeCols + 4 * rq + 2);
                        acc[0] = fma(v, z0.x, acc[0]);
                        acc[1] = fma(v, z0.y, acc[1]);
                        acc[2] = fma(v, z1.x, acc[2]);
                        acc[3] = fma(v, z1.y, acc[3]);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int c = 4 * rq + j, k0 = (c / K) * K;
                        // the on-shell column: v_a D_N x_p[a]
                        for (int bb = 0; bb < K; ++bb) acc[j] = fma(b[rr * kMeCols + k0 + bb], DNc[c] * xp[c * 2 + bb], acc[j]);
                        acc[j] = b[rr * kMeCols + c] - x[rr * kMeCols + c] + acc[j];
                    }
                }
                // r_p = V_pp - x_p + v^T (D x_g) + V_pp D_N x_p
                for (int w = warp; w < kMeCols * K; w += nw) {
                    const int c = w / K, a = w - c * K, k0 = (c / K) * K;
                    double s = 0.0;
                    for (int r = lane; r < ng; r += 32) s = fma(b[r * kMeCols + k0 + a], z[r * kMeCols + c], s);
                    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if (lane == 0) {
                        for (int bb = 0; bb < K; ++bb) s = fma(Vpp[(k0 + bb) * 2 + a], DNc[c] * xp[c * 2 + bb], s);
                        rp[c * 2 + a] = Vpp[c * 2 + a] - xp[c * 2 + a] + s;
                    }
                }
                __syncthreads();
                if (rr < ng)
#pragma unroll
                    for (int j = 0; j < 4; ++j) z[rr * kMeCols + 4 * rq + j] = acc[j];
                __syncthreads();
            }
            for (int c = 0; c < kMeCols; ++c) worst = max(worst, nst[c]);
            if (tid < EC && e0 + tid < n_I) {
                const int ie = e0 + tid;
                bool ok = true;
                for (int bb = 0; bb < K; ++bb) ok &= nst[tid * K + bb] != 0;
                redo[((size_t)smp * n_ch_total + cidx) * n_I + ie] = ok ? 0 : 1;
                double Km[4] = {0, 0, 0, 0};
                for (int a = 0; a < K; ++a)
                    for (int bb = 0; bb < K; ++bb) Km[a * 2 + bb] = xp[(tid * K + bb) * 2 + a];
                const size_t o = ((size_t)smp * n_ch_total + cidx) * n_I + ie;
                mi_phases(K, sqrt(kMn * e_int[ie] / 2.0) / kHbarc, Km, ph + o * 3);
                if (k_out)
                    for (int k = 0; k < 4; ++k) k_out[o * 4 + k] = Km[k];
            }
        }
        if (tid == 0) status[(size_t)smp * n_ch_total + cidx] = worst;  // the elimination kernel adds what it redoes
    }
}

bool mi_energies_fit(int NQ, int K) { return me_smem(K * NQ, NQ, K) <= 227 * 1024 && (K * NQ + 31) / 32 * 2 <= me_threads(K) / 32; }

int mi_energies_per_sm(int NQ, int K)
{
    const size_t smem = me_smem(K * NQ, NQ, K);
    raise_smem_limit((const void *)k_mi_energies, smem);
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_mi_energies, me_threads(K), smem);
    return blocks;
}

// n_samples samples from sample0; eps / Q: the eigenpairs of this range (eig_ch offsets), eig_status their
// solves' status [sample][n_ch_total], eig_err their error word.
cudaError_t launch_mi_energies(const MiChanDev *chans_dev, const ChanDev *eig_ch, const int *work_dev, int n_work, int K,
                               int n_ch_total, int sample0, int n_samples, int NQ, const double *kg, const double *wg,
                               int n_terms, const double *coeffs, const double *Vg, const double *Von, int n_I,
                               const double *e_int, const double *eps, const double *Q, const int *eig_status,
                               const int *eig_err, double *Vs, int slots, double *ph, double *k_out, int *status, int *redo,
                               int *err, cudaStream_t st)
{
    const size_t smem = me_smem(K * NQ, NQ, K);
    if (!mi_energies_fit(NQ, K)) return cudaErrorInvalidValue;
    raise_smem_limit((const void *)k_mi_energies, smem);
    k_mi_energies<<<slots, me_threads(K), smem, counted(st)>>>(chans_dev, eig_ch, work_dev, n_work, n_ch_total, sample0,
                                                            n_samples, NQ, kg, wg, n_terms, coeffs, Vg, Von, n_I, e_int,
                                                            eps, Q, eig_status, eig_err, Vs, ph, k_out, status, redo, err);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------- observables
// Phases at the requested energies by linear interpolation in T_lab between
// consecutive interpolation energies (end segments extended, delta unwrapped
// by multiples of 180 deg), and the np total cross section.  One thread per
// (sample, energy).
__global__ void k_mi_observables(const MiChanDev *chans, int n_ch, int n_samples, int n_I, const double *e_int,
                                 const double *ph, int n_E, const double *e_lab, double *delta, double *sigma)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n_samples * n_E) return;
    const int e = (int)(idx % n_E), smp = (int)(idx / n_E);
    const double E = e_lab[e], p = sqrt(kMn * E / 2.0) / kHbarc, rad = kPi / 180.0;
    int lo = -1, hi = n_I - 1;  // largest j with e_int[j] <= E
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (e_int[mid] <= E) lo = mid;
        else hi = mid - 1;
    }
    const int j = lo < 0 ? 0 : (lo > n_I - 2 ? n_I - 2 : lo);
    const double w = (E - e_int[j]) / (e_int[j + 1] - e_int[j]);
    double acc = 0.0;
    for (int c = 0; c < n_ch; ++c) {
        const MiChanDev ch = chans[c];
        const double *pc = ph + ((size_t)smp * n_ch + c) * n_I * 3;
        double out[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < ch.K; ++k) {
            const double d0 = pc[3 * j + k];
            double d1 = pc[3 * (j + 1) + k];
            d1 += 180.0 * round((d0 - d1) / 180.0);
            double d = d0 + w * (d1 - d0);
            if (isfinite(d)) {
                while (d > 90.0) d -= 180.0;
                while (d <= -90.0) d += 180.0;
            }
            out[k] = d;
        }
        if (ch.K == 2) out[2] = pc[3 * j + 2] + w * (pc[3 * (j + 1) + 2] - pc[3 * j + 2]);
        if (delta) {
            double *d = delta + (((size_t)smp * n_ch + c) * n_E + e) * 3;
            d[0] = out[0];
            d[1] = out[1];
            d[2] = out[2];
        }
        if (ch.tz == 0) {
            if (ch.K == 1) {
                acc += (2.0 * ch.J + 1.0) * (1.0 - cos(2.0 * out[0] * rad));
            } else {
                const double c2e = cos(2.0 * out[2] * rad);
                acc += (2.0 * ch.J + 1.0) *
                       ((1.0 - c2e * cos(2.0 * out[0] * rad)) + (1.0 - c2e * cos(2.0 * out[1] * rad)));
            }
        }
    }
    if (sigma) sigma[idx] = kPi / (2.0 * p * p) * 10.0 * acc;
}

cudaError_t launch_mi_observables(const MiChanDev *chans_dev, int n_ch, int n_samples, int n_I, const double *e_int,
                                  const double *ph, int n_E, const double *e_lab, double *delta, double *sigma,
                                  cudaStream_t st)
{
    const size_t total = (size_t)n_samples * n_E;
    k_mi_observables<<<(unsigned)((total + 127) / 128), 128, 0, counted(st)>>>(chans_dev, n_ch, n_samples, n_I, e_int, ph, n_E,
                                                                       e_lab, delta, sigma);
    return cudaGetLastError();
}

}  // namespace wpcd
