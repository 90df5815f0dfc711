// FP64 chi0 (Eq. (RPA)) on the tcgen05 tensor cores, exact to the last bits of FP64 by integer slices.
//
//   chi0_GG'(w) = pref sum_t conj(rho_t(G)) x_t(w, G'),   x = W_t(w) rho_t(G')  (FP64),
//
// is one real product with k = 2t + part,
//   D[m][n] = sum_k A[m][k] B[n][k],   m = (G block of 64, re | im, G in block),   n = (w, G'),
//   A re rows (Re rho, Im rho), im rows (-Im rho, Re rho);   B (Re x, Im x).
// Every row is scaled by a power of two to |v| < 1 and written as an integer q = rint(2^62 v) in eight signed
// base-256 digits, each exact in BF16 (the scheme of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with
// fixed slices).  The 36 digit products of order i + j <= 7 are formed on the tensor cores; those left out are below
// 2^-63 of the row maxima's product.  A product of digits is at most 2^14, so the sum of the (at most eight) products
// of one order over 128 k stays below 2^24 and is exact in the FP32 accumulator: after each such window the sums are
// read out as integers and added into two 64-bit integers per element (orders 0-3 and 4-7).  No rounding happens
// before the final conversion; the K range is split over CTAs and the splits are added in FP64 in a fixed order.
// Bound of an element's error: ~2^-61 of (row maximum of |A|) x (sum of the row of |B|) and the reverse, which is not the
// plain sum's bound over sum |A||B|: terms far below their row's maximum are held in fewer bits.  Measured over that
// sum, element by element against sums in extended precision (N_t = 48, 960, 4536; eta = 2e-2 to 2e-12 Hartree,
// frequencies on and beside resonances): 0.8e-15 to 1.1e-14, the plain kernel 1.2e-15 to 5.8e-14, the slices closer in
// all 27 cases.
//
// What bounds it: the plain kernel is bound by the GB300's FP64 pipe (1.06 TFLOP/s): 42 ms per frequency at N_G =
// 181, N_t = 65536.  Here a frequency costs 36 BF16 products of the same shape on the tensor cores.  Operand
// digits go through global memory: A once per call, B once per frequency (both read back by TMA), so that a CTA's
// stage is 96 KB of copies against 72 MMAs of 128 x 64 x 16; the copies (~42 B/clk per SM, near what the SM takes
// in) and the MMAs are about balanced.  Eight orders x 64 columns fill the 512 TMEM columns, which is why the tile
// is 64 wide and the read-out does not overlap the MMAs (a window is 4 stages, ~9k cycles; a read-out ~1.5k).
// Measured: N_G = 181, N_t = 65536, 8 frequencies 339 -> 14 ms (products 11.2, digits 2.3, maxima 0.35).
#include "qcx_internal.h"
#include "tc_ptx.cuh"

#include <algorithm>

namespace {

constexpr int NS = 8;                       // digits per value
constexpr int OZ_BITS = 62;
constexpr int OZ_THREADS = 320;             // TMA, MMA, 8 read-out warps
constexpr int OZ_NSTAGE = 2;
constexpr int OZ_M = 128;
constexpr int OZ_NMAX = 64;
constexpr int OZ_WINDOW = 4;                // K stages (of 32) whose sums stay below 2^24
constexpr int OZ_KWIN = OZ_WINDOW * KSTEP;  // 128
constexpr uint32_t OZ_ATILE = OZ_M * ROWB;
constexpr int OZ_BAD = 1 << 20;             // exponent of a row that holds an infinity or NaN
constexpr int OZ_EMIN = -900;               // rows below 2^-900 count as zero
static_assert((1 << 14) * NS * OZ_KWIN <= (1 << 24), "window sums must be exact in FP32");

// e with |x| < 2^e from the high word of |x| (largest over a row)
__device__ __forceinline__ int exponent_of(unsigned hi) {
    const int e = (int)(hi >> 20) & 0x7ff;
    return e == 0x7ff ? OZ_BAD : max(e - 1022, OZ_EMIN);
}
__device__ __forceinline__ unsigned hi_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ double pow2(int e) { return scalbn(1.0, e); }    // 0 for a row with OZ_BAD

__device__ __forceinline__ unsigned block_max(unsigned v) {
    __shared__ unsigned red[8];
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[threadIdx.x & 7];
    v = __reduce_max_sync(0xffffffffu, v);
    __syncthreads();
    return v;
}

// W_t(w) and max(|Re W|, |Im W|) of a group of frequencies
__global__ void k_oz_weights(int nw, long long nt, int nv, int nc, const double* Ek, const double* Ekq, const double* w,
                             double eta, double2* W, double* winf) {
    const long long n = (long long)nw * nt;
    const int nvc = nv * nc;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int iw = (int)(i / nt);
        const long long t = i - (long long)iw * nt;
        const long long k = t / nvc;
        const int rem = (int)(t - k * nvc);
        const int v = rem / nc, c = rem - v * nc;
        const double dE = Ekq[k * nc + c] - Ek[k * nv + v];
        const double a = w[iw] - dE, b = w[iw] + dE;
        const double d1 = 1.0 / (a * a + eta * eta), d2 = 1.0 / (b * b + eta * eta);
        const double2 x = make_double2(a * d1 - b * d2, eta * (d2 - d1));
        W[i] = x;
        // a NaN must survive the maximum
        winf[i] = fabs(x.x) + fabs(x.y);
    }
}

// exponents of the rho rows: one CTA per G
__global__ void __launch_bounds__(256) k_oz_rowmax(long long nt, const double2* R, int* eA) {
    const double2* r = R + (long long)blockIdx.x * nt;
    unsigned m = 0;
    for (long long t = threadIdx.x; t < nt; t += 256) m = max(m, max(hi_abs(r[t].x), hi_abs(r[t].y)));
    m = block_max(m);
    if (threadIdx.x == 0) eA[blockIdx.x] = exponent_of(m);
}

// exponents of the rows x(w, G'): |x| < 2 max_t winf |rho|; CTA (G', 4 frequencies)
__global__ void __launch_bounds__(256) k_oz_xmax(int ng, int nw, long long nt, const double2* R, const double* winf, int* eB) {
    const int G = blockIdx.x, w0 = blockIdx.y * 4;
    const double2* r = R + (long long)G * nt;
    unsigned m[4] = {0, 0, 0, 0};
    for (long long t = threadIdx.x; t < nt; t += 256) {
        const double2 z = r[t];
        const double a = fabs(z.x) + fabs(z.y);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (w0 + u < nw) m[u] = max(m[u], hi_abs(a * winf[(long long)(w0 + u) * nt + t]));
    }
    for (int u = 0; u < 4; ++u) {
        const unsigned v = block_max(m[u]);
        if (threadIdx.x == 0 && w0 + u < nw) eB[(w0 + u) * ng + G] = exponent_of(v);
    }
}

// digits of the two parts of a value, most significant first, as packed BF16 pairs
__device__ __forceinline__ void digits(double re, double im, double scale, uint32_t (&d)[NS]) {
    long long a = __double2ll_rn(re * scale), b = __double2ll_rn(im * scale);
#pragma unroll
    for (int i = NS - 1; i >= 0; --i) {
        const int x = i ? (int)(signed char)(a & 0xff) : (int)a;
        const int y = i ? (int)(signed char)(b & 0xff) : (int)b;
        a = (a - x) >> 8;
        b = (b - y) >> 8;
        d[i] = pack_bf16((float)x, (float)y);
    }
}

// digits of rho over transitions t0 .. t0 + nt2 - 1 into [NS][arows][nt2] (pairs): re rows and im rows of every 64-G block
__global__ void __launch_bounds__(256) k_oz_slice_a(int ng, long long nt, long long t0, int nt2, int arows, const double2* R,
                                                    const int* eA, uint32_t* P) {
    const int tl = blockIdx.x * 256 + threadIdx.x;
    if (tl >= nt2) return;
    const long long t = t0 + tl;
    const size_t plane = (size_t)arows * nt2;
    for (int j = 0; j < 16; ++j) {
        const int G = blockIdx.y * 16 + j;                      // up to the padded block of 64
        uint32_t d[NS] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (G < ng && t < nt) {
            const double2 r = R[(long long)G * nt + t];
            digits(r.x, r.y, pow2(OZ_BITS - eA[G]), d);
        }
        uint32_t* p = P + (size_t)((G >> 6) * 128 + (G & 63)) * nt2 + tl;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            p[i * plane] = d[i];
            // (-Im, Re): halves swapped, the new low half negated
            p[i * plane + (size_t)64 * nt2] = __byte_perm(d[i], 0u, 0x1032) ^ 0x00008000u;
        }
    }
}

// digits of x = W rho into [NS][nw][ngp][nt2] (pairs)
__global__ void __launch_bounds__(256) k_oz_slice_x(int ng, int ngp, int nw, long long nt, long long t0, int nt2,
                                                    const double2* R, const double2* W, const int* eB, uint32_t* P) {
    const int tl = blockIdx.x * 256 + threadIdx.x;
    if (tl >= nt2) return;
    const long long t = t0 + tl;
    const int iw = blockIdx.z;
    const size_t plane = (size_t)nw * ngp * nt2;
    const double2 w = t < nt ? W[(long long)iw * nt + t] : make_double2(0.0, 0.0);
    for (int j = 0; j < 16; ++j) {
        const int G = blockIdx.y * 16 + j;
        uint32_t d[NS] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (G < ng && t < nt) {
            const double2 r = R[(long long)G * nt + t];
            digits(fma(w.x, r.x, -w.y * r.y), fma(w.x, r.y, w.y * r.x), pow2(OZ_BITS - 1 - eB[iw * ng + G]), d);
        }
        uint32_t* p = P + ((size_t)iw * ngp + G) * nt2 + tl;
#pragma unroll
        for (int i = 0; i < NS; ++i) p[i * plane] = d[i];
    }
}

struct OzArgs {
    int ng, ngp, nw, n_tile, n_chunks, arows, brows;
    int kstages, per_split;           // stages of 32 in this K chunk; stages per split (a multiple of the window)
    uint32_t tmem_cols;
    const int* eA;                    // [ng]
    const int* eB;                    // [nw][ng]
    double* part;                     // [split][nw][ngp][arows]
    int accumulate;                   // add to part (later K chunks)
    int* status;
    long long wait_limit;
    int withhold;                     // fault injection: no copies, so that the consumers' first waits run out
};

__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, OzArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gb = blockIdx.x;
    const int iw = blockIdx.y / a.n_chunks, n0 = (blockIdx.y % a.n_chunks) * a.n_tile;
    const int s0 = blockIdx.z * a.per_split;
    const int nst = min(a.per_split, a.kstages - s0);           // a multiple of the window, > 0
    const uint32_t btile = (uint32_t)a.n_tile * ROWB;
    const uint32_t stage_bytes = NS * (OZ_ATILE + btile);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + OZ_NSTAGE * stage_bytes);   // [NSTAGE]
    uint64_t* empty = full + OZ_NSTAGE;                                             // [NSTAGE]
    uint64_t* acc_full = empty + OZ_NSTAGE;
    uint64_t* drained = acc_full + 1;
    uint64_t* mma_done = drained + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_NSTAGE; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(drained, 8);
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, a.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int nwin = nst / OZ_WINDOW;

    if (warp == 0) {
        if (lane == 0) {
            int last = -1;
            for (int it = 0; it < (a.withhold ? 0 : nst); ++it) {
                const int s = it % OZ_NSTAGE;
                const uint32_t ph = (uint32_t)(it / OZ_NSTAGE) & 1u;
                if (!mbar_wait(&empty[s], ph ^ 1u, abort_flag, a.status, a.wait_limit)) break;
                unsigned char* st = base + s * stage_bytes;
                mbar_arrive_tx(&full[s], stage_bytes);
                const int x = (s0 + it) * KSTEP;
                for (int i = 0; i < NS; ++i) {
                    tma_load_2d(st + i * OZ_ATILE, &ma, &full[s], x, i * a.arows + gb * OZ_M);
                    tma_load_2d(st + NS * OZ_ATILE + i * btile, &mb, &full[s], x, i * a.brows + iw * a.ngp + n0);
                }
                last = it;
            }
            // copies still in flight land before the CTA can exit
            for (int it = max(0, last - OZ_NSTAGE + 1); it <= last; ++it)
                mbar_wait(&full[it % OZ_NSTAGE], (uint32_t)(it / OZ_NSTAGE) & 1u, abort_flag, a.status,
                          CLEANUP_WAIT_LIMIT, false);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = make_idesc(OZ_M, a.n_tile);
            bool ok = true;
            for (int win = 0; win < nwin && ok; ++win) {
                if (win && !(ok = mbar_wait(drained, (uint32_t)(win - 1) & 1u, abort_flag, a.status, a.wait_limit))) break;
                for (int u = 0; u < OZ_WINDOW; ++u) {
                    const int it = win * OZ_WINDOW + u;
                    const int s = it % OZ_NSTAGE;
                    if (!(ok = mbar_wait(&full[s], (uint32_t)(it / OZ_NSTAGE) & 1u, abort_flag, a.status, a.wait_limit)))
                        break;
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(base + s * stage_bytes), b0 = a0 + NS * OZ_ATILE;
                    for (int kk = 0; kk < KSTEP / 16; ++kk) {
                        const uint32_t off = kk * 32;
                        for (int g = 0; g < NS; ++g) {
                            const uint32_t d = tmem + (uint32_t)(g * a.n_tile);
                            for (int i = 0; i <= g; ++i)
                                umma_bf16(d, sw64_desc(a0 + i * OZ_ATILE + off), sw64_desc(b0 + (g - i) * btile + off), idesc,
                                          (u | kk | i) ? 1u : 0u);
                        }
                    }
                    umma_commit(&empty[s]);
                }
                if (ok) umma_commit(acc_full);
            }
            // no MMA may still be running when TMEM is freed (also on the abort path)
            umma_commit(mma_done);
            mbar_wait(mma_done, 0, abort_flag, a.status, CLEANUP_WAIT_LIMIT, false);
        }
    } else {
        const int q = warp & 3, hc = (warp - 2) >> 2;           // TMEM lane quadrant, column half
        const int half = a.n_tile >> 1;                          // a multiple of 8, at most 32
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        long long hi[OZ_NMAX / 2], lo[OZ_NMAX / 2];
#pragma unroll
        for (int c = 0; c < OZ_NMAX / 2; ++c) hi[c] = lo[c] = 0;
        bool ok = true;
        for (int win = 0; win < nwin && ok; ++win) {
            if (!(ok = warp_wait(acc_full, (uint32_t)win & 1u, abort_flag, a.status, a.wait_limit))) break;
            tc_fence_after();
            const uint32_t tb = tmem + lane_off + (uint32_t)(hc * half);
#pragma unroll
            for (int c8 = 0; c8 < OZ_NMAX / 16; ++c8)
                if (c8 * 8 < half) {
#pragma unroll
                    for (int g2 = 0; g2 < NS; g2 += 4) {
                        uint32_t r[4][8];
#pragma unroll
                        for (int u = 0; u < 4; ++u) tmem_ld8(tb + (uint32_t)((g2 + u) * a.n_tile + c8 * 8), r[u]);
                        tmem_wait_ld();
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const long long v = (long long)__float2int_rn(__uint_as_float(r[u][i])) * (1 << (8 * (3 - u)));
                                if (g2 == 0)
                                    hi[c8 * 8 + i] += v;
                                else
                                    lo[c8 * 8 + i] += v;
                            }
                    }
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(drained);
        }
        if (ok) {
            const int row = q * 32 + lane, G = gb * 64 + (row & 63);
            double* out = a.part + (((size_t)blockIdx.z * a.nw + iw) * a.ngp) * a.arows + (size_t)gb * OZ_M + row;
            if (G < a.ng) {
                const int ea = a.eA[G];
#pragma unroll
                for (int c = 0; c < OZ_NMAX / 2; ++c) {
                    const int H = n0 + hc * half + c;
                    if (c < half && H < a.ng) {
                        const int eb = a.eB[iw * a.ng + H];
                        double v;
                        if (ea >= OZ_BAD || eb >= OZ_BAD)
                            v = nan("");
                        else
                            // digit products of order g carry 2^(8 (14 - g)); x was scaled by one bit less
                            v = scalbn(fma((double)hi[c], 4294967296.0, (double)lo[c]), 56 - 2 * OZ_BITS + 1 + ea + eb);
                        double* o = out + (size_t)H * a.arows;
                        *o = a.accumulate ? *o + v : v;
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, a.tmem_cols);
    }
}

// chi0 = pref x the splits in order; eps = 1 - v^1/2 chi0 v^1/2.  part is [split][nw][ngp (G')][arows (G)].  NaN after a wait
// that gave up, since the host may look at the status later than at the results.
__global__ void k_oz_finish(int ng, int ngp, int nw, int arows, int nsplit, const double* part, double pref, const double* vs,
                            const int* status, double2* eps, double2* chi) {
    const int G = blockIdx.x * 32 + threadIdx.x, H = blockIdx.y * 8 + threadIdx.y, iw = blockIdx.z;
    __shared__ double2 tile[8][33];
    double2 c = make_double2(0.0, 0.0);
    if (G < ng && H < ng) {
        const size_t row = (size_t)(G >> 6) * 128 + (G & 63);
        for (int z = 0; z < nsplit; ++z) {
            const double* p = part + (((size_t)z * nw + iw) * ngp + H) * arows + row;
            c.x += p[0];
            c.y += p[64];
        }
    }
    if (*status) c = make_double2(nan(""), nan(""));
    tile[threadIdx.y][threadIdx.x] = make_double2(pref * c.x, pref * c.y);
    __syncthreads();
    const int id = threadIdx.y * 32 + threadIdx.x, h = id & 7, g = id >> 3;
    const int G2 = blockIdx.x * 32 + g, H2 = blockIdx.y * 8 + h;
    if (G2 < ng && H2 < ng) {
        const double2 ch = tile[h][g];
        const double vv = vs[G2] * vs[H2];
        const size_t o = ((size_t)iw * ng + G2) * ng + H2;
        eps[o] = make_double2((G2 == H2 ? 1.0 : 0.0) - vv * ch.x, -vv * ch.y);
        if (chi) chi[o] = ch;
    }
}

// digit planes of one pass (both operands): frequencies are taken in groups and transitions in chunks to stay below
constexpr size_t OZ_PLANE_BYTES = 4ull << 30;
constexpr int OZ_W_GROUP = 8;

}  // namespace

// Tensor-core route of the FP64 chi0; cudaErrorMemoryAllocation when its work space does not fit.
cudaError_t qcx_launch_chi0_fp64_tc(qcx_ctx* ctx, QSlot& s, int iq, double pref, double2* chi, int* d_status) {
    const int ng = s.ng, nw = s.nw;
    const long long nt = (long long)ctx->nk * ctx->nv * ctx->nc;
    const int ngp = (ng + 15) / 16 * 16, gbs = (ng + 63) / 64, arows = gbs * 128;
    const int n_tile = std::min(OZ_NMAX, ngp), n_chunks = (ngp + n_tile - 1) / n_tile;
    const int wg = std::min(nw, OZ_W_GROUP);
    // transitions per chunk: 64 per window of 128 k
    const long long all = (nt + 63) / 64 * 64;
    const size_t per_t = (size_t)NS * 4 * (arows + (size_t)wg * ngp);
    const int nt2 = (int)std::min<long long>(all, std::max<long long>(64, (long long)(OZ_PLANE_BYTES / per_t) / 64 * 64));
    const int kst = nt2 / 16;                                     // K stages of a chunk
    const int tiles = gbs * n_chunks * wg;
    const int windows = kst / OZ_WINDOW;
    const int want = std::min(windows, std::max(1, (2 * 152 + tiles - 1) / tiles));
    const int per_split = (windows + want - 1) / want * OZ_WINDOW;
    const int nsplit = (kst + per_split - 1) / per_split;

    OzBufs& b = ctx->oz;
    cudaError_t e;
    if ((e = b.a.ensure((size_t)NS * 4 * arows * nt2)) != cudaSuccess ||
        (e = b.b.ensure((size_t)NS * 4 * wg * ngp * nt2)) != cudaSuccess ||
        (e = b.w.ensure((size_t)wg * nt * (sizeof(double2) + sizeof(double)))) != cudaSuccess ||
        (e = b.e.ensure(sizeof(int) * (size_t)(ng + wg * ng))) != cudaSuccess ||
        (e = b.part.ensure(sizeof(double) * (size_t)nsplit * wg * ngp * arows)) != cudaSuccess) {
        b.release();
        return e;
    }
    cudaStream_t st = ctx->stream;
    const double2* R = s.rho.as<double2>();
    double2* W = b.w.as<double2>();
    double* winf = reinterpret_cast<double*>(W + (size_t)wg * nt);
    int* eA = b.e.as<int>();
    int* eB = eA + ng;
    OzArgs a{};
    a.ng = ng;
    a.ngp = ngp;
    a.n_tile = n_tile;
    a.n_chunks = n_chunks;
    a.arows = arows;
    a.eA = eA;
    a.eB = eB;
    a.part = b.part.as<double>();
    a.status = d_status;
    a.wait_limit = ctx->wait_limit;
    a.withhold = ctx->withhold_copies;
    a.kstages = kst;
    a.per_split = per_split;
    a.tmem_cols = 32;
    while (a.tmem_cols < (uint32_t)(NS * n_tile)) a.tmem_cols *= 2;
    const size_t smem = 1024 + OZ_NSTAGE * (size_t)NS * (OZ_ATILE + n_tile * ROWB) + (2 * OZ_NSTAGE + 3) * 8 + 16;
    if ((e = qcx_allow_smem((const void*)k_oz_gemm)) != cudaSuccess) return e;
    k_oz_rowmax<<<ng, 256, 0, st>>>(nt, R, eA);
    CUtensorMap ma, mb;
    if (!qcx_make_bf16_map(&ma, b.a.p, 2LL * nt2, NS * arows, OZ_M, KSTEP)) return cudaErrorInvalidValue;
    bool a_ready = false;
    for (int w0 = 0; w0 < nw; w0 += wg) {
        const int m = std::min(wg, nw - w0);
        a.nw = m;
        a.brows = m * ngp;
        if (!qcx_make_bf16_map(&mb, b.b.p, 2LL * nt2, NS * m * ngp, n_tile, KSTEP)) return cudaErrorInvalidValue;
        k_oz_weights<<<(int)std::min<long long>(((long long)m * nt + 255) / 256, 4096), 256, 0, st>>>(
            m, nt, ctx->nv, ctx->nc, ctx->d_Ek.as<double>(), ctx->d_Ekq.as<double>() + (size_t)iq * ctx->nk * ctx->nc,
            s.w.as<double>() + w0, s.eta, W, winf);
        k_oz_xmax<<<dim3(ng, (m + 3) / 4), 256, 0, st>>>(ng, m, nt, R, winf, eB);
        for (long long t0 = 0; t0 < all; t0 += nt2) {
            const unsigned tb = (nt2 + 255) / 256;
            if (!a_ready) k_oz_slice_a<<<dim3(tb, gbs * 4), 256, 0, st>>>(ng, nt, t0, nt2, arows, R, eA, b.a.as<uint32_t>());
            a_ready = nt2 == all;                                // one chunk: the rho digits serve every group
            k_oz_slice_x<<<dim3(tb, ngp / 16, m), 256, 0, st>>>(ng, ngp, m, nt, t0, nt2, R, W, eB, b.b.as<uint32_t>());
            a.accumulate = t0 > 0;
            k_oz_gemm<<<dim3(gbs, n_chunks * m, nsplit), OZ_THREADS, smem, st>>>(ma, mb, a);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        k_oz_finish<<<dim3((ng + 31) / 32, (ng + 7) / 8, m), dim3(32, 8), 0, st>>>(
            ng, ngp, m, arows, nsplit, a.part, pref, s.vs.as<double>(), d_status, s.eps.as<double2>() + (size_t)w0 * ng * ng,
            chi ? chi + (size_t)w0 * ng * ng : nullptr);
    }
    return cudaGetLastError();
}
