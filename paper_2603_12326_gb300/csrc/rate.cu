// Momentum binning of the loss tables and the nonrelativistic halo rate.
//
// dR/dw = (rho_chi/m_chi)(1/rho_T) sigma_e/(8 pi^2 alpha mu^2)
//         int dq q^3 |F_DM(q)|^2 Im[-1/eps(w,q)] eta(v_min),   v_min = q/(2 m_chi) + w/q
// (end of Appendix A with Eqs. (general_rate), (v_min), (F_DM)); eta is the
// mean inverse speed above v_min of the truncated Maxwellian halo.  The
// recoil spectrum is Eq. (excitation_rate) with the step ionisation model.
// Everything here is FP64: the rate accumulates over q and w.
#include "qcx_internal.h"

namespace {

// CODATA 2018 and unit conversions (natural units, eV)
constexpr double kAlpha = 1.0 / 137.035999084;
constexpr double kMe = 510998.95000;            // eV
constexpr double kHbarC = 1.973269804e-5;       // eV cm
constexpr double kHbar = 6.582119569e-16;       // eV s
constexpr double kC = 299792.458;               // km/s
constexpr double kEvPerKg = 5.609588603804452e35;
constexpr double kYear = 365.25 * 24.0 * 3600.0;
constexpr double kHartree = 27.211386245988;    // eV
constexpr double kAme = kAlpha * kMe;           // eV per bohr^-1
constexpr double kPi = 3.141592653589793;

// mean inverse speed above vmin of f ~ exp(-|v + vE|^2/v0^2), |v + vE| < vesc (units of c); pref = 1 / (2 n_esc v0 y),
// ez = exp(-z^2), erfz = erf(z) do not depend on vmin
struct Halo {
    double v0, y, z, pref, ez, erfz;
};
__device__ Halo halo_of(double v0, double vesc, double vE) {
    Halo h;
    h.v0 = v0;
    h.y = vE / v0;
    h.z = vesc / v0;
    h.ez = exp(-h.z * h.z);
    h.erfz = erf(h.z);
    const double nesc = h.erfz - 2.0 / sqrt(kPi) * h.z * h.ez;
    h.pref = 1.0 / (2.0 * nesc * v0 * h.y);
    return h;
}
__device__ double eta_halo(double vmin, const Halo& h) {
    const double x = vmin / h.v0, y = h.y, z = h.z;
    if (x < z - y) return h.pref * (erf(x + y) - erf(x - y) - 4.0 / sqrt(kPi) * y * h.ez);
    if (x < z + y) return h.pref * (h.erfz - erf(x - y) - 2.0 / sqrt(kPi) * (z + y - x) * h.ez);
    return 0.0;
}

// One CTA per frequency, threads over the q bins: the integrand in parallel, the trapezoids in a fixed order (each
// thread its own, a tree over the threads).  A thread per frequency walked the bins serially, two or three error
// functions each (120 bins: 217 -> 15 us).
constexpr int RATE_THREADS = 128;
__global__ void __launch_bounds__(RATE_THREADS) k_rate(int nq, const double* q_bohr, int nw, const double* w_ha,
                                                       const double* L, qcx_halo_params p, double* dRdw) {
    __shared__ double g[RATE_THREADS + 1], sum[RATE_THREADS];
    const int iw = blockIdx.x;
    const Halo h = halo_of(p.v0_kms / kC, p.vesc_kms / kC, p.vE_kms / kC);
    const double n_chi = p.rho_chi_GeV_cm3 * 1e9 / p.m_chi_eV * kHbarC * kHbarC * kHbarC;
    const double rho_T = p.rho_T_g_cm3 * kEvPerKg * 1e-3 * kHbarC * kHbarC * kHbarC;
    const double sigma = p.sigma_e_cm2 / (kHbarC * kHbarC);
    const double mu = p.m_chi_eV * kMe / (p.m_chi_eV + kMe);
    const double pref = n_chi / rho_T * sigma / (8.0 * kPi * kPi * kAlpha * mu * mu);
    const double wv = w_ha[iw] * kHartree;
    double acc = 0.0;
    for (int i0 = 0; i0 < nq; i0 += RATE_THREADS) {
        const int i = i0 + threadIdx.x;
        double v = 0.0;
        if (i < nq) {
            const double qv = q_bohr[i] * kAme;
            double F2 = 1.0;
            if (p.m_med_eV >= 0.0) {
                const double f = (kAme * kAme + p.m_med_eV * p.m_med_eV) / (qv * qv + p.m_med_eV * p.m_med_eV);
                F2 = f * f;
            }
            const double vmin = qv / (2.0 * p.m_chi_eV) + wv / qv;
            v = qv * qv * qv * F2 * L[(size_t)i * nw + iw] * eta_halo(vmin, h);
        }
        g[threadIdx.x + 1] = v;
        __syncthreads();
        if (i < nq && i > 0) acc += 0.5 * (g[threadIdx.x + 1] + g[threadIdx.x]) * (q_bohr[i] * kAme - q_bohr[i - 1] * kAme);
        __syncthreads();
        if (threadIdx.x == RATE_THREADS - 1) g[0] = v;
        __syncthreads();
    }
    sum[threadIdx.x] = acc;
    __syncthreads();
    for (int d = RATE_THREADS / 2; d > 0; d >>= 1) {
        if (threadIdx.x < d) sum[threadIdx.x] += sum[threadIdx.x + d];
        __syncthreads();
    }
    if (threadIdx.x == 0) dRdw[iw] = pref * sum[0] * kEvPerKg * (kYear / kHbar);
}

// One warp per ionisation bin: lanes over the frequencies (the step of a frequency needs an FP64 division each, and one
// thread walked them all), then a tree.
__global__ void k_recoil(int nw, const double* w_ha, const double* dRdw, double wgap, double wpp, int nQ,
                         double* out) {
    const int Q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5) + 1, lane = threadIdx.x & 31;
    if (Q > nQ) return;
    const double dw = (w_ha[1] - w_ha[0]) * kHartree;
    double acc = 0.0;
    for (int i = lane; i < nw; i += 32) {
        const double wv = w_ha[i] * kHartree;
        if (wv < wgap) continue;
        const int Qi = 1 + (int)floor((wv - wgap) / wpp);
        if (Qi == Q) acc += dRdw[i] * dw;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) out[Q - 1] = acc;
}

// out[bin][w] = mean over (q, G) with |q+G| in [edges[bin], edges[bin+1]) of L[which][w][G].  One warp per (bin, 32 w):
// lanes first find a bin's members 32 G at a time, then every lane adds them for its frequency in (q, G) order.
__global__ void k_bin(int nsel, const double* const* Ls, const double* const* qm, const int* ngs, int nw,
                      int which, int nbin, const double* edges, double* out, double* cnt) {
    const int wblk = (nw + 31) / 32;
    const int id = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (id >= nbin * wblk) return;
    const int bin = id / wblk, iw = (id - bin * wblk) * 32 + lane;
    const double lo = edges[bin], hi = edges[bin + 1];
    double s = 0.0;
    int c = 0;
    for (int q = 0; q < nsel; ++q) {
        const int ng = ngs[q];
        const double* qmq = qm[q];
        const double* Lq = Ls[q] + ((size_t)which * nw + min(iw, nw - 1)) * ng;
        for (int g0 = 0; g0 < ng; g0 += 32) {
            const double m = g0 + lane < ng ? qmq[g0 + lane] : -1.0;
            unsigned in = __ballot_sync(0xffffffffu, g0 + lane < ng && m >= lo && m < hi);
            c += __popc(in);
            for (; in; in &= in - 1) s += Lq[g0 + __ffs(in) - 1];
        }
    }
    if (iw < nw) out[(size_t)bin * nw + iw] = c ? s / c : 0.0;
    if (iw == 0) cnt[bin] = (double)c;
}

}  // namespace

cudaError_t qcx_launch_bin(qcx_ctx* ctx, int nsel, const double* const* d_L, const double* const* d_qmag,
                           const int* d_ng, int nw, int which, int nbin, const double* d_edges, double* d_out,
                           double* d_cnt) {
    const long long n = (long long)nbin * ((nw + 31) / 32);      // warps
    k_bin<<<(unsigned)((n + 3) / 4), 128, 0, ctx->stream>>>(nsel, d_L, d_qmag, d_ng, nw, which, nbin, d_edges, d_out,
                                                   d_cnt);
    return cudaGetLastError();
}

cudaError_t qcx_launch_recoil(cudaStream_t st, int nw, const double* d_w, const double* d_dRdw, double wgap_eV,
                              double wpp_eV, int nQ, double* d_dRQ) {
    k_recoil<<<(nQ + 3) / 4, 128, 0, st>>>(nw, d_w, d_dRdw, wgap_eV, wpp_eV, nQ, d_dRQ);
    return cudaGetLastError();
}

cudaError_t qcx_launch_rate(qcx_ctx* ctx, int nqbin, const double* d_q, int nw, const double* d_w,
                            const double* d_L, const qcx_halo_params& p, double* d_dRdw, int nQ,
                            double* d_dRQ) {
    k_rate<<<nw, RATE_THREADS, 0, ctx->stream>>>(nqbin, d_q, nw, d_w, d_L, p, d_dRdw);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || nQ <= 0) return e;
    k_recoil<<<(nQ + 3) / 4, 128, 0, ctx->stream>>>(nw, d_w, d_dRdw, p.w_gap_eV, p.w_pp_eV, nQ, d_dRQ);
    return cudaGetLastError();
}
