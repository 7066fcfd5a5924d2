// saclay.cu -- spin observables of np scattering (App. A) from the phase
// shifts: the M-matrix partial-wave expansion, the Saclay amplitudes a..e and
// dsigma/dOmega, batched over (sample, energy, angle).
//
// With the incoming momentum along z and phi = 0, momentum-space partial waves
// and every np channel once,
//   M^s_{m'm}(theta) = sqrt(4 pi)/(2 i p) sum_{J,l,l'} sqrt(2l+1)
//       C(l' (m-m') s m' | J m) C(l 0 s m | J m) (S_{l'l} - delta_{l'l}) Y_{l'}^{m-m'}(theta, 0),
// S rebuilt from the (Stapp) phases.  Parity, M_{-m'-m} = (-1)^{m-m'} M_{m'm}
// (l + l' is even), leaves six functions of the angle: the singlet M_ss and
// M_11, M_1-1, M_10, M_01, M_00.  The amplitudes are M's coefficients in
//   M = [(a+b) + (a-b)(s1.n)(s2.n) + (c+d)(s1.m)(s2.m) + (c-d)(s1.l)(s2.l) + e(s1+s2).n] / 2,
// l, m, n along p + p', p - p', p x p'.  With (s1.v)(s2.v) = 2 (S.v)^2 - 1 the
// traces that define them are, in the six functions,
//   a = (M_11 + M_00 - M_1-1)/2,  b = (M_11 + M_1-1 + M_ss)/2,  c = (M_11 + M_1-1 - M_ss)/2,
//   d = [cos(theta) (M_1-1 + M_00 - M_11) - sqrt 2 sin(theta) (M_01 + M_10)]/2,
//   e = i (M_10 - M_01)/sqrt 2,
// and dsigma/dOmega = Tr(M M^+)/4.
//
// The kernel is bound by the FP64 pipe (two multiply-adds a clock and SM), so
// nothing is done twice: the sum over channels depends on (sample, energy)
// alone and runs once per pair, into coefficients B_f[l'] of each function in
// Y_{l'}^{mu}; the harmonics depend on the angle alone and are tabulated once
// per CTA; a point is then six sums over l' of 2 multiply-adds.  256 samples x
// 128 energies x 32 angles, J <= 4: 18.4 -> 0.44 ms a call (the sum over channels and
// the harmonics at every point before), 92 MB of outputs in 14 us at the copy rate.
#include <math.h>

#include "wpcd_internal.cuh"

namespace wpcd {

constexpr int kSacThreads = 256;
constexpr int kSacChunk = 8;  // channels whose S - 1 one pass holds

struct Cplx {
    double re, im;
};
__device__ __forceinline__ Cplx cmul(Cplx a, Cplx b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }

// Shared memory of one CTA: B double2 [P][L1][6] | S - 1 double2 [P][kSacChunk][3] | Y double [3][L1][TC] |
// normalisations double [3][L1] | cos, sin [TC each].
__host__ __device__ inline size_t sac_smem(int P, int L1, int TC)
{
    return ((size_t)P * L1 * 6 + (size_t)P * kSacChunk * 3) * 16 + ((size_t)3 * L1 * TC + 3 * L1 + 2 * TC) * 8;
}

// CTA (x, y, z): pairs x P .. + P - 1 of (sample, energy), TC angles from y TC on and, where the angles
// need more rows than a grid has, z gridDim.y TC further on.
__global__ void __launch_bounds__(kSacThreads) k_saclay(const SacChanDev *chans, int n_ch, long long n_pairs, int n_E,
                                                        const double *e_lab, const double *delta, int n_th,
                                                        const double *theta, double *abcde, double *dsig, int P,
                                                        int L1, int TC)
{
    extern __shared__ double2 sac_sm[];
    double2 *B = sac_sm;
    double2 *A = B + (size_t)P * L1 * 6;
    double *Y = reinterpret_cast<double *>(A + (size_t)P * kSacChunk * 3);
    double *nrm = Y + (size_t)3 * L1 * TC;
    double *ct = nrm + 3 * L1, *st = ct + TC;
    const int tid = threadIdx.x, nt = blockDim.x;
    const long long pair0 = (long long)blockIdx.x * P;
    const unsigned first = (blockIdx.z * gridDim.y + blockIdx.y) * (unsigned)TC;  // below 2^31 + 65535 TC
    if (first >= (unsigned)n_th) return;
    const int np = (int)min((long long)P, n_pairs - pair0);
    const int th0 = (int)first, nth = min(TC, n_th - th0);

    // ---- Y_l^mu(theta, 0), Condon-Shortley phase, mu = 0, 1, 2
    for (int e = tid; e < 3 * L1; e += nt) {  // sqrt((2l+1)/(4 pi) (l-mu)!/(l+mu)!), with (-1)^mu
        const int mu = e / L1, l = e - mu * L1;
        double ratio = 1.0;
        for (int k = l - mu + 1; k <= l + mu; ++k) ratio /= k;  // l >= mu (the others are not used)
        const double y = l >= mu ? sqrt((2.0 * l + 1.0) / (4.0 * kPi) * ratio) : 0.0;
        nrm[e] = mu == 1 ? -y : y;
    }
    for (int t = tid; t < nth; t += nt) sincos(theta[th0 + t], &st[t], &ct[t]);
    __syncthreads();
    for (int e = tid; e < 3 * nth; e += nt) {
        const int mu = e / nth, t = e - mu * nth;
        const double x = ct[t], s = st[t];
        double *y = Y + (size_t)mu * L1 * TC + t;
        double p1 = mu == 0 ? 1.0 : mu == 1 ? s : 3.0 * s * s, p0 = 0.0;  // P_mu^mu without the phase
        for (int l = 0; l < L1; ++l) {
            if (l < mu) {
                y[(size_t)l * TC] = 0.0;
                continue;
            }
            if (l > mu) {
                const double pn = ((2.0 * l - 1.0) * x * p1 - (l + mu - 1.0) * p0) / (l - mu);
                p0 = p1;
                p1 = pn;
            }
            y[(size_t)l * TC] = nrm[mu * L1 + l] * p1;
        }
    }

    // ---- B_f[l'] of every pair, the channels in passes of kSacChunk
    for (int e = tid; e < np * L1 * 6; e += nt) B[e] = make_double2(0.0, 0.0);
    for (int c0 = 0; c0 < n_ch; c0 += kSacChunk) {
        const int nc = min(kSacChunk, n_ch - c0);
        __syncthreads();  // the last pass has read A
        for (int e = tid; e < np * nc; e += nt) {
            const int k = e / nc, c = e - k * nc;
            const SacChanDev &ch = chans[c0 + c];
            if (ch.tz != 0) continue;
            const long long pair = pair0 + k, smp = pair / n_E;
            const int en = (int)(pair - smp * n_E);
            const double *ph = delta + ((smp * n_ch + c0 + c) * n_E + en) * 3;
            double2 *a = A + ((size_t)k * kSacChunk + c) * 3;
            Cplx em, ep;  // e^{i delta}: angles in half turns, pi delta / 180
            sincospi(ph[0] * (1.0 / 180.0), &em.im, &em.re);
            const Cplx s11 = cmul(em, em);
            if (ch.K == 1) {
                a[0] = make_double2(s11.re - 1.0, s11.im);
            } else {
                double ce, se;
                sincospi(ph[1] * (1.0 / 180.0), &ep.im, &ep.re);
                sincospi(ph[2] * (1.0 / 90.0), &se, &ce);
                const Cplx s22 = cmul(ep, ep), m = cmul(em, ep);
                a[0] = make_double2(ce * s11.re - 1.0, ce * s11.im);
                a[1] = make_double2(ce * s22.re - 1.0, ce * s22.im);
                a[2] = make_double2(-se * m.im, se * m.re);  // i sin(2 eps) e^{i (dm + dp)}
            }
        }
        __syncthreads();
        for (int e = tid; e < np * L1; e += nt) {
            const int k = e / L1, l = e - k * L1;
            double2 *b = B + (size_t)e * 6;
            for (int c = 0; c < nc; ++c) {
                const SacChanDev &ch = chans[c0 + c];
                if (ch.tz != 0) continue;
                const double2 *a = A + ((size_t)k * kSacChunk + c) * 3;
                for (int ip = 0; ip < ch.K; ++ip) {
                    if (ch.l[ip] != l) continue;
                    for (int il = 0; il < ch.K; ++il) {
                        const double2 v = ip != il ? a[2] : a[ip];
                        const double *w = ch.w[ip * 2 + il];
                        if (ch.s == 0) {
                            b[0].x = fma(w[0], v.x, b[0].x);
                            b[0].y = fma(w[0], v.y, b[0].y);
                        } else {
                            for (int f = 1; f < 6; ++f) {
                                b[f].x = fma(w[f], v.x, b[f].x);
                                b[f].y = fma(w[f], v.y, b[f].y);
                            }
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int k = tid; k < np; k += nt)  // 1 / (2 p), where S - 1 was
        A[k].x = 1.0 / (2.0 * (sqrt(kMn * e_lab[(pair0 + k) % n_E] / 2.0) / kHbarc));
    __syncthreads();
    for (int e = tid; e < np * L1 * 6; e += nt) {  // / (2 i p)
        const double f = A[e / (L1 * 6)].x;
        const double2 v = B[e];
        B[e] = make_double2(v.y * f, -v.x * f);
    }
    __syncthreads();

    // ---- the points of the CTA, angles fastest (a warp's lanes share a pair when it has 32 angles)
    for (int e = tid; e < np * nth; e += nt) {
        const int k = e / nth, t = e - k * nth;
        const double2 *b = B + (size_t)k * L1 * 6;
        Cplx M[6];
#pragma unroll
        for (int f = 0; f < 6; ++f) M[f] = {0.0, 0.0};
        for (int l = 0; l < L1; ++l, b += 6) {
            const double y0 = Y[(size_t)l * TC + t], y1 = Y[((size_t)L1 + l) * TC + t],
                         y2 = Y[((size_t)2 * L1 + l) * TC + t];
#pragma unroll
            for (int f = 0; f < 6; ++f) {
                const double2 v = b[f];
                const double y = f == 2 ? y2 : (f == 3 || f == 4) ? y1 : y0;
                M[f].re = fma(v.x, y, M[f].re);
                M[f].im = fma(v.y, y, M[f].im);
            }
        }
        const Cplx ss = M[0], m11 = M[1], m1m = M[2], m10 = M[3], m01 = M[4], m00 = M[5];
        const size_t o = (size_t)(pair0 + k) * n_th + th0 + t;
        if (abcde) {
            const double h = 0.70710678118654752440, hc = 0.5 * ct[t], hs = h * st[t];
            const Cplx p = {m11.re + m1m.re, m11.im + m1m.im}, q = {m11.re - m1m.re, m11.im - m1m.im};
            const double2 out[5] = {make_double2(0.5 * (q.re + m00.re), 0.5 * (q.im + m00.im)),
                                    make_double2(0.5 * (p.re + ss.re), 0.5 * (p.im + ss.im)),
                                    make_double2(0.5 * (p.re - ss.re), 0.5 * (p.im - ss.im)),
                                    make_double2(hc * (m00.re - q.re) - hs * (m01.re + m10.re),
                                                 hc * (m00.im - q.im) - hs * (m01.im + m10.im)),
                                    make_double2(h * (m01.im - m10.im), h * (m10.re - m01.re))};
            if ((reinterpret_cast<uintptr_t>(abcde) & 15) == 0) {
#pragma unroll
                for (int f = 0; f < 5; ++f) reinterpret_cast<double2 *>(abcde)[o * 5 + f] = out[f];
            } else {  // a caller's buffer on an odd 8-byte boundary
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    abcde[o * 10 + 2 * f] = out[f].x;
                    abcde[o * 10 + 2 * f + 1] = out[f].y;
                }
            }
        }
        if (dsig) {
            double two = 0.0, one = 0.0;
#pragma unroll
            for (int f = 1; f < 5; ++f) two = fma(M[f].re, M[f].re, fma(M[f].im, M[f].im, two));
            one = fma(ss.re, ss.re, fma(ss.im, ss.im, fma(m00.re, m00.re, m00.im * m00.im)));
            dsig[o] = 2.5 * fma(2.0, two, one);  // Tr(M M^+)/4, fm^2 -> mb
        }
    }
}

// Angles up to 32 a CTA (a warp shares a pair's coefficients) and as many pairs as
// make ~1024 points, at most 32: the tables then cost a few percent of the points.
cudaError_t launch_saclay(const SacChanDev *chans_dev, int n_ch, int n_samples, int n_E, const double *e_lab,
                          const double *delta, int n_th, const double *theta, double *abcde, double *dsig, int Lmax,
                          cudaStream_t st)
{
    const long long n_pairs = (long long)n_samples * n_E;
    if (Lmax < 0 || Lmax > kMaxJ + 1) return cudaErrorInvalidValue;
    const int L1 = Lmax + 1, TC = n_th < 32 ? n_th : 32;
    int P = 1024 / TC < 32 ? 1024 / TC : 32;
    while (P > 1 && sac_smem(P, L1, TC) > 48 * 1024) P /= 2;
    const unsigned tbs = (unsigned)((n_th - 1) / TC + 1), rows = tbs < 65535u ? tbs : 65535u;
    const dim3 grid((unsigned)((n_pairs + P - 1) / P), rows, (tbs + rows - 1) / rows);
    k_saclay<<<grid, kSacThreads, sac_smem(P, L1, TC), counted(st)>>>(chans_dev, n_ch, n_pairs, n_E, e_lab, delta,
                                                                      n_th, theta, abcde, dsig, P, L1, TC);
    return cudaGetLastError();
}

}  // namespace wpcd
