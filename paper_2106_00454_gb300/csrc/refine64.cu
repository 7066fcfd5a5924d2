// refine64.cu -- FP64 eigenpairs from an FP32 eigensolve (the FP64 path of (a3)).
//
// The FP64 pipe issues two fused multiply-adds per clock and SM, 1/58 of the
// FP32 rate, so the FP64 path lets the FP32 Jacobi kernels find approximate
// eigenvectors X and brings them to FP64 with products on the tensor cores
// (exact digit products, ozaki.cu).  Each iteration forms, with the FP64 H,
//     Y = H X,  S = X^T Y,  G = X^T X,  lambda_i = S_ii / G_ii,
//     s_ij = S_ij - (lambda_i + lambda_j) G_ij / 2   (the off-diagonal of the
//            Rayleigh matrix after symmetric orthonormalisation, to first order)
// and updates X <- X (I + E), E_ij = s_ij / (lambda_j - lambda_i) - G_ij / 2,
// E being the first-order correction of Ogita & Aishima ("Iterative refinement
// for symmetric eigenvalue decomposition", 2018), split into its antisymmetric
// (rotation) and symmetric (orthonormalisation) parts.  First order is not
// enough for a pair whose eigenvalues lie closer together than the FP32 solve
// resolves (the two branches of a coupled channel at high l, or a chance
// crossing): such pairs are turned by plane rotations of s, G and the columns of
// X first, in FP64, pair by pair and rescanned until none is left.  A pair with
// |s_ij| below the rounding of the products is left alone: its quotient is noise,
// and the FP64 Jacobi kernel's stopping test would leave it too.
//
// An item is done once, after the first iteration, an update's ||E||_F^2 <= kDoneE2 =
// 2e-14: what is left of the off-diagonal, and the error of the eigenvalues, which come
// from before the update, are second order in E and so below 2e-14 ||H||_F.  That bound is
// seldom met: the second iteration's E is mostly the rounding of the products over small
// gaps, whose second order is below the rounding of X.  Measured at 2e-14 and at 1e-15
// alike: residual 3.9e-15 ||H||_F, eigenvalues 6e-16, orthogonality 2.6e-14 at n = 200 (FP64
// Jacobi alone, which stops at off(A) <= 1e-15 ||H||_F: 3e-15, 1e-15, 1e-12), at 18.0 and
// 20.1 ms for 128 samples x 15 channels at N_WP = 100, as the tighter one sends more items
// through a third iteration; 2e-16 leaves items to FP64 Jacobi (85 ms).  Two iterations
// usually do it, the third runs only for the items that need it, and an item
// that is not done after that (or whose eigenvalues do not fit FP32) is solved again
// by the FP64 Jacobi kernel (the caller's fallback over done[b] == 0).
//
// The FP32 solve may start from C0^T H C0, C0 the eigenvectors of diag(H0) + V0 (built
// once per set): nearly diagonal, about half the sweeps, and the longest chains (a
// channel with a bound state, 12 sweeps) shorten most.  It only supplies the start: H
// itself is never rotated here.  Start from H -> from the basis, ms a call: 20 channels at
// N_WP = 100, one sample, 5.47 -> 3.20; at N_WP = 150, 8 samples, 14.8 -> 11.2; 15 channels of
// N_WP 40/64/100, 32 samples 4.42 -> 3.96, 256 19.7 -> 18.4, 1024 74.1 -> 69.1.
//
// Measured against FP64 Jacobi alone (its rotations are bound by the FP64 pipe):
// 20 channels at N_WP = 100, one sample, 153 -> 3.2 to 4.0 ms a solve (by the sample); 15
// channels of N_WP 40/64/100, 256 samples, 333 -> 18.7 ms; 20 channels at N_WP = 150, 8
// samples, 843 to 918 -> 10.5 to 12.0 ms; 1S0 at N_WP = 32, 0.69 -> 0.29 ms; errors against
// 64-bit LAPACK unchanged (T 3e-14 to 1.2e-12 in both).  Up to n = 16 FP64 Jacobi is faster
// (runtime.cu).
//
// The update is X + X E with E small: the digit product's rounding, relative
// to E's columns, then vanishes beside X, and X keeps its 53 bits.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>

#include "wpcd_internal.cuh"

namespace wpcd {

// Pairs are turned above these angles: in the first iteration 2^-13, whose square
// the second one corrects; from then on 2^-26, so that nothing of their square is
// left.  The second list is short (at n = 300 up to ~40 pairs of a coupled channel,
// whose s only the second iteration's products resolve); where it is not, only what
// first order cannot take is turned, and the item goes on to the next iteration.
constexpr float kFirstAngle = 1.2207031e-4f, kLaterAngle = 1.4901161e-8f, kMaxAngle = 0.02f;
constexpr float kDoneE2 = 2e-14f;     // ||E||_F <= 1.4e-7; the bound on what its square leaves (above)
// Pairs turned per scan: 64 up to n = 512, 512 above.  Pairs that first order cannot take grow in
// number with n, and a first iteration that leaves them is not made good by the other two: with
// 64 everywhere, dense matrices above n = 512 and one in eight of the projected coupled ones at
// N_WP = 512 went to FP64 Jacobi (3 matrices of n = 514 1980 -> 26 ms, 8 of n = 1024 31 s -> 180 ms;
// those that finished before, n = 600, 62 -> 64 ms).
constexpr int kPairCap = 512, kPairFew = 64;
constexpr int kPairScans = 6;

// One CTA per item, or a cluster of them (CL) where the items are few: the CTAs take the
// rows in turn, the pairs found and the rows' sums of E^2 meet in the first one's shared
// memory, and what others may have written is read past the L1.  No result depends on how
// many share an item (||E||^2 is summed by rows).  Bound by the FP64 pipe where the chip is
// full, by the latency of S and G where it is not (64 matrices of n = 200, one CTA each, 0.40
// and 0.64 ms for the two iterations, the sort 0.12).  One CTA an item -> up to eight, a whole
// solve: 20 channels at N_WP = 100, one sample, 3.70 -> 3.11 ms; N_WP = 150, 8 samples, 11.9 ->
// 10.7; 15 channels N_WP 40/64/100, 256 samples, unchanged.  S, G and X change only where pairs are turned; E goes to
// E_all (the buffer of the next X, whose old content is dead).  FP64 where it
// must be: the Rayleigh quotients, the differences and s (both cancel for close
// eigenvalues) and the sums; the quotient s / d is formed in FP32, with one
// correction step for the angles above 2^-26, so its error stays below 2^-50.
template <bool CL>
__global__ void __launch_bounds__(256) k_r64_update(int n, double *S_all, double *G_all, double *X_all,
                                                    double *E_all, double *lam_all, int *done, int it)
{
    extern __shared__ double sm64[];
    double *lam = sm64;                                          // n
    double *hl = lam + n;                                        // n: lambda / 2
    unsigned *pr = reinterpret_cast<unsigned *>(hl + n);         // kPairCap: the scan's pairs, unordered
    unsigned *ps = pr + kPairCap;                                // kPairCap: the same in order
    float *al = reinterpret_cast<float *>(ps + kPairCap);        // n: |lambda| times the rounding of the products
    float *rs = al + n;                                          // n: the rows' sums of E^2
    __shared__ double red[32];
    __shared__ int s_cnt;
    const int cr = CL ? (int)cooperative_groups::this_cluster().block_rank() : 0;
    const int cn = CL ? (int)cooperative_groups::this_cluster().num_blocks() : 1;
    const int b = blockIdx.x / cn;
    if (done[b] != 0) return;
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, nwarp = nt >> 5;
    auto sync = [&]() {
        if (CL) cooperative_groups::this_cluster().sync();
        else __syncthreads();
    };
    unsigned *pr0 = CL ? cooperative_groups::this_cluster().map_shared_rank(pr, 0) : pr;
    float *rs0 = CL ? cooperative_groups::this_cluster().map_shared_rank(rs, 0) : rs;
    int *cnt0 = CL ? cooperative_groups::this_cluster().map_shared_rank(&s_cnt, 0) : &s_cnt;
    const int w0 = cr * nwarp + warp, ws = cn * nwarp, t0 = cr * nt + tid, ts = cn * nt;  // over the cluster
    auto ld = [](const double *q) { return CL ? __ldcg(q) : *q; };
    const size_t off = (size_t)b * n * n;
    double *S = S_all + off, *G = G_all + off, *X = X_all + off, *E = E_all + off;
    const float round = it == 0 ? 2.910383e-11f : 8.881784e-16f;  // 2^-35 (39-bit products), 2^-50 (55-bit)
    bool above = false, enough = false;
    for (int i = tid; i < n; i += nt) {
        const double l = ld(S + (size_t)i * n + i) / ld(G + (size_t)i * n + i);
        const float lf = fabsf(f32_trunc(l));
        lam[i] = l;
        hl[i] = 0.5 * l;
        al[i] = round * lf;
        above |= !(lf < 1.2676506e30f);  // 2^100
        enough |= lf > 8.6736174e-19f;   // 2^-60
    }
    // the tests below are in FP32: H's scale has to leave them room on both sides
    if (__syncthreads_or(above) || !__syncthreads_or(enough)) return;
    float ang = it == 0 ? kFirstAngle : kLaterAngle;
    const int cap = n > 512 ? kPairCap : kPairFew;
    bool plain = true;  // S holds S (not yet s)
    bool clear = false, later = false;
    for (int scan = 0;; ++scan) {
        if (cr == 0 && tid == 0) s_cnt = 0;
        sync();
        for (int i = w0; i < n; i += ws) {
            const double li = lam[i], hi = hl[i];
            const float ai = al[i];
            const double *Si = S + (size_t)i * n, *Gi = G + (size_t)i * n;
            double *Ei = E + (size_t)i * n;
            float e2 = 0.0f;
            double sj = lane < n ? ld(Si + lane) : 0.0, gj = lane < n ? ld(Gi + lane) : 0.0;
            for (int j = lane; j < n; j += 32) {
                const double g = gj, sv = sj;
                if (j + 32 < n) {  // the next step's values on their way
                    sj = ld(Si + j + 32);
                    gj = ld(Gi + j + 32);
                }
                double ev;
                if (j == i) {
                    ev = 0.5 * (1.0 - g);
                } else {
                    const double s = plain ? fma(-(hi + hl[j]), g, sv) : sv;
                    const double d = lam[j] - li;
                    const float sf = f32_trunc(s), df = f32_trunc(d);
                    double th = 0.0;
                    const float as = fabsf(sf), ad = fabsf(df);
                    if (as > fmaxf(ai, al[j])) {
                        if (as > ang * ad && i < j) {
                            const int k = atomicAdd(cnt0, 1);
                            if (k < kPairCap) pr0[k] = ((unsigned)i << 16) | (unsigned)j;
                        }
                        if (as <= kMaxAngle * ad) {
                            const float rd = __frcp_rn(df), t0 = sf * rd;
                            th = f64_of(t0);
                            if (fabsf(t0) > 1.5e-8f) th += f64_of(f32_trunc(fma(-th, d, s)) * rd);
                        }
                    }
                    ev = fma(-0.5, g, th);
                }
                Ei[j] = ev;
                const float ef = f32_trunc(ev);
                e2 = fmaf(ef, ef, e2);
            }
            for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
            if (lane == 0) rs0[i] = e2;
        }
        sync();
        const int m = *cnt0;
        if (m > cap && ang < kMaxAngle) {  // too many: turn only those beyond first order
            ang = kMaxAngle;
            later = true;
            sync();  // every thread has read the count
            continue;
        }
        if (m == 0 || m > cap || scan >= kPairScans) {
            clear = m == 0 && !later;
            break;
        }
        // ---- turn the scan's pairs, in index order (the order of the list does not matter)
        if (cr != 0) {
            for (int k = tid; k < m; k += nt) pr[k] = pr0[k];
            __syncthreads();
        }
        for (int k = tid; k < m; k += nt) {
            const unsigned v = pr[k];
            int r = 0;
            for (int q = 0; q < m; ++q) r += pr[q] < v;
            ps[r] = v;
        }
        if (plain) {
            for (int i = w0; i < n; i += ws)
                for (int j = lane; j < n; j += 32) {
                    const size_t e = (size_t)i * n + j;
                    S[e] = i == j ? lam[i] : fma(-(hl[i] + hl[j]), ld(G + e), ld(S + e));
                }
            plain = false;
        }
        sync();
        for (int k = 0; k < m; ++k) {
            const int i = (int)(ps[k] >> 16), j = (int)(ps[k] & 0xFFFFu);
            const double s = ld(S + (size_t)i * n + j), a = ld(S + (size_t)i * n + i), q = ld(S + (size_t)j * n + j);
            double c = 1.0, sn = 0.0;
            if (s != 0.0) {
                const double tau = (q - a) / (2.0 * s);
                const double t = fabs(tau) > 1e150 ? 0.5 / tau
                                                   : (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(fma(tau, tau, 1.0)));
                c = 1.0 / sqrt(fma(t, t, 1.0));
                sn = t * c;
            }
            sync();  // every thread has read the pair's block
            for (int r = t0; r < n; r += ts)  // columns i, j
                for (int w = 0; w < 3; ++w) {
                    double *M = w == 0 ? S : w == 1 ? G : X;
                    const double x = ld(M + (size_t)r * n + i), y = ld(M + (size_t)r * n + j);
                    M[(size_t)r * n + i] = fma(-sn, y, c * x);
                    M[(size_t)r * n + j] = fma(sn, x, c * y);
                }
            sync();
            for (int r = t0; r < n; r += ts)  // rows i, j
                for (int w = 0; w < 2; ++w) {
                    double *M = w == 0 ? S : G;
                    const double x = ld(M + (size_t)i * n + r), y = ld(M + (size_t)j * n + r);
                    M[(size_t)i * n + r] = fma(-sn, y, c * x);
                    M[(size_t)j * n + r] = fma(sn, x, c * y);
                }
            sync();
            if (tid == 0) {
                if (cr == 0) S[(size_t)i * n + j] = S[(size_t)j * n + i] = 0.0;
                lam[i] = ld(S + (size_t)i * n + i);
                lam[j] = ld(S + (size_t)j * n + j);
                hl[i] = 0.5 * lam[i];
                hl[j] = 0.5 * lam[j];
            }
            sync();
        }
    }
    sync();  // the first CTA's shared memory has been read
    if (cr != 0) return;
    double *lo = lam_all + (size_t)b * n;
    for (int i = tid; i < n; i += nt) lo[i] = lam[i];
    double e2 = 0.0;
    for (int i = tid; i < n; i += nt) e2 += (double)rs[i];
    const double t2 = cta_sum64(e2, red);
    // (the first iteration's eigenvalues come from 39-bit products)
    if (tid == 0 && it > 0 && clear && t2 <= (double)kDoneE2) done[b] = it + 1;
}

// Sorted eigenpairs of the items that are done, into the eigen-buffer layout;
// the vectors of an item done at iteration k lie in X0 (k even) or X1 (k odd).
// An item whose FP32 solve hit its sweep cap counts as not done; left (may be NULL)
// counts the items that are not.
__global__ void __launch_bounds__(256) k_r64_sort(const ChanDev *chans, const int *work, int nw, int sample0, int n,
                                                  const double *lam_s, const double *X0, const double *X1, int *done,
                                                  const int *status_all, int n_ch_total, double *eps_all,
                                                  double *X_all, unsigned long long *left)
{
    extern __shared__ long long sm64s[];
    long long *key = sm64s;                         // n: the eigenvalues as integers in the same order
    int *rank = reinterpret_cast<int *>(key + n);   // n
    const int b = blockIdx.x, part = blockIdx.y, parts = gridDim.y;
    const int wc = b % nw, smp = sample0 + b / nw;
    const int d = done[b];
    const bool failed = status_all[(size_t)smp * n_ch_total + work[wc]] <= 0;
    if (d == 0 || failed) {
        __syncthreads();
        if (threadIdx.x == 0 && part == 0) {
            done[b] = 0;
            if (left) atomicAdd(left, 1ull);
        }
        return;
    }
    const ChanDev ch = chans[work[wc]];
    const double *Xs = ((d & 1) ? X1 : X0) + (size_t)b * n * n;
    double *X = X_all + ch.c_off + (size_t)smp * n * n;
    double *eps = eps_all + ch.eps_off + (size_t)smp * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const long long v = __double_as_longlong(lam_s[(size_t)b * n + i] + 0.0);  // no negative zero
        key[i] = v < 0 ? v ^ 0x7fffffffffffffffll : v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const long long ki = key[i];
        int r = 0;
        for (int j = 0; j < n; ++j) r += (key[j] < ki) || (key[j] == ki && j < i);
        rank[i] = r;
        if (part == 0) eps[r] = lam_s[(size_t)b * n + i];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    for (int row = part * nwarp + warp; row < n; row += parts * nwarp)
        for (int c = lane; c < n; c += 32) X[(size_t)row * n + rank[c]] = Xs[(size_t)row * n + c];
}

static size_t r64_smem(int n) { return (size_t)n * (2 * 8 + 2 * 4) + kPairCap * 2 * sizeof(unsigned); }

// CTAs that share an item in k_r64_update and k_r64_sort: up to two of 256
// threads on each SM (clusters wait for room beside other kernels, so a full chip
// does better without: up to eight cost 19.2 -> 20.1 ms at 256 samples), two rows or more a warp.
static int r64_share(int items, int n)
{
    const long long room = 2ll * device_sms();
    int cl = 8;
    while (cl > 1 && ((long long)items * cl > room || n < 16 * cl)) cl /= 2;
    return cl;
}

static cudaError_t launch_r64_update(int items, int n, double *S, double *G, double *X, double *E, double *lam, int *done,
                                     int it, cudaStream_t st)
{
    const int cl = r64_share(items, n);
    if (cl == 1) {
        k_r64_update<false><<<items, 256, r64_smem(n), counted(st)>>>(n, S, G, X, E, lam, done, it);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(items * cl));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = r64_smem(n);
    cfg.stream = counted(st);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_r64_update<true>, n, S, G, X, E, lam, done, it);
}

// Digits per product: the first iteration only has to leave errors that the
// second squares away (39-bit products); from then on Y, S and G carry 55 bits.
// E is small, so X E needs its leading 31 bits (kDigE), and so does the change of
// basis X = C0 X' of a start in the mean-potential eigenbasis, which the
// iterations refine.
constexpr int kDigFirst = 5, kDigLast = 7;

// X, Y (then E and the next X), G, S, lambda; digit slices of H's rows (kDigFirst and
// kDigLast planes), X's columns and Y's columns (kDigLast each), X's rows and E's columns
// (kDigE) with their exponents.
size_t refine64_scratch_per_item(int n)
{
    return (size_t)4 * n * n * 8 + (size_t)n * 8 +
           (oz_slice_elems(n, kDigFirst) + 3 * oz_slice_elems(n, kDigLast) + 2 * oz_slice_elems(n, kDigE)) * 2 +
           (size_t)5 * n * 4 + 512;
}

// Where the FP32 solve leaves its vectors (rotated: in the mean-potential basis), and its eigenvalues.
double *refine64_start(void *scratch, int items, int n, bool rotated)
{
    return static_cast<double *>(scratch) + (rotated ? (size_t)items * n * n : 0);
}
double *refine64_lambda(void *scratch, int items, int n)
{
    return static_cast<double *>(scratch) + (size_t)4 * items * n * n;
}

// The items of one bucket chunk, in scratch blocks X, Y, G, S of items n^2 doubles
// each, lambda after them, and done[items] ints.  On entry the FP32 solve's vectors at
// refine64_start; on return the done items' eigenpairs are in eps_all / X_all and
// done[b] == 0 marks the ones that the caller solves by other means.  chans, coeffs: H is
// summed from its terms, never from the FP32 solve's basis.  rot_s, rot_e: kDigE digit
// slices of the rows of the nw channels' C0 when the vectors are given in that basis.
cudaError_t launch_refine64(const ChanDev *chans, const int *work, int nw, int n_samples, int sample0, int n, int n_terms,
                            const double *coeffs, void *scratch, int *done, const int *status_all, int n_ch_total,
                            double *eps_all, double *X_all, cudaStream_t st, int *err, const __nv_bfloat16 *rot_s,
                            const int *rot_e, unsigned long long *left)
{
    const int items = n_samples * nw;
    const size_t nn = (size_t)items * n * n;
    double *X0 = static_cast<double *>(scratch);
    double *X1 = X0 + nn, *G = X1 + nn, *S = G + nn, *lam = S + nn;
    const uintptr_t s0 = (reinterpret_cast<uintptr_t>(lam + (size_t)items * n) + 255) & ~(uintptr_t)255;
    const size_t s5 = (size_t)items * oz_slice_elems(n, kDigFirst), se = (size_t)items * oz_slice_elems(n, kDigLast),
                 sE = (size_t)items * oz_slice_elems(n, kDigE);
    __nv_bfloat16 *sH5 = reinterpret_cast<__nv_bfloat16 *>(s0);
    __nv_bfloat16 *sH7 = sH5 + s5, *sXc = sH7 + se, *sXr = sXc + 2 * se, *sEc = sXr + sE;
    int *eH = reinterpret_cast<int *>(sEc + sE);
    int *eXc = eH + (size_t)items * n, *eYc = eXc + (size_t)items * n, *eXr = eYc + (size_t)items * n;
    int *eEc = eXr + (size_t)items * n;
    cudaError_t e = cudaMemsetAsync(done, 0, sizeof(int) * items, st);
    if (e != cudaSuccess) return e;
#define CKR(x)                       \
    do {                             \
        if ((e = (x)) != cudaSuccess) \
            return e;                \
    } while (0)
    if (rot_s) {  // X = C0 X'
        CKR(launch_oz_split(n, items, true, X1, sEc, eEc, st, OzSkip(), kDigE));
        CKR(launch_oz_gemm_slices(n, items, rot_s, rot_e, sEc, eEc, X0, st, kDigE, false, err, nw, nullptr, OzSkip(), kDigE));
    }
    CKR(launch_oz_hsum(chans, work, nw, n_samples, sample0, n, n_terms, coeffs, sH5, sH7, eH, st));
    double *x = X0, *xn = X1;
    for (int it = 0; it < kRefine64Iters; ++it) {
        OzSkip sk;
        sk.done = it > 0 ? done : nullptr;
        sk.it = it;
        const int dg = it == 0 ? kDigFirst : kDigLast;
        CKR(launch_oz_split(n, items, true, x, sXc, eXc, st, sk, dg));
        CKR(launch_oz_gemm_slices(n, items, it == 0 ? sH5 : sH7, eH, sXc, eXc, xn, st, dg, false, err, 0, nullptr, sk, dg));  // Y = H X
        // G = X^T X and S = X^T Y in one launch: the column slices of Y follow those of X
        __nv_bfloat16 *sYc = sXc + (size_t)items * oz_slice_elems(n, dg);
        OzSkip two = sk;
        two.mod = items;
        CKR(launch_oz_split(n, items, true, xn, sYc, eYc, st, sk, dg));
        CKR(launch_oz_gemm_slices(n, 2 * items, sXc, eXc, sXc, eXc, G, st, dg, true, err, items, nullptr, two, dg));
        CKR(launch_r64_update(items, n, S, G, x, xn, lam, done, it, st));  // E over Y
        CKR(launch_oz_split(n, items, false, x, sXr, eXr, st, sk, kDigE));
        CKR(launch_oz_split(n, items, true, xn, sEc, eEc, st, sk, kDigE));
        CKR(launch_oz_gemm_slices(n, items, sXr, eXr, sEc, eEc, xn, st, kDigE, false, err, 0, x, sk, kDigE));  // X + X E
        double *t = x;
        x = xn;
        xn = t;
    }
#undef CKR
    k_r64_sort<<<dim3(items, r64_share(items, n)), 256, (size_t)n * 12, counted(st)>>>(chans, work, nw, sample0, n, lam, X0, X1, done, status_all,
                                                            n_ch_total, eps_all, X_all, left);
    return cudaGetLastError();
}

}  // namespace wpcd
