// Mixed-precision chi0 (Eq. (RPA)) for many frequencies: the direct sum with its frequency dependence taken out of
// the contraction.
//
// W_t(w) = 1/(w - dE_t + i eta) - 1/(w + dE_t + i eta) is, as a function of dE, analytic but for poles a distance eta
// from the real axis.  On an interval of half width a it is therefore reproduced by the polynomial through n Chebyshev
// points up to ~rho^-n of its largest value there, rho = eta/a + sqrt(1 + (eta/a)^2) (Trefethen, Approximation
// Theory and Approximation Practice, 2013, ch. 8), for every w at once: with a = 2 eta/3 and n = 16, 1e-8, below the
// FP32 rounding of W itself.  So the energies are cut into panels of width 2a and
//
//   S_pj[G][G'] = sum_{t in panel p} l_j(dE_t) conj(rho_t(G)) rho_t(G'),   l_j the Lagrange polynomial of node j,
//   chi0(w)     = pref sum_pj W(w; E_pj) S_pj.
//
// Each transition is contracted 16 times (in one triangle: S_pj is Hermitian) instead of once per frequency, and the
// frequencies see N_b = 16 x panels nodes instead of N_t transitions.  Precision: operands as in the direct kernel
// (rho~ in two BF16 planes against l rho~ in three terms, five products); the tensor core truncates its FP32 sums with
// every MMA, which shrinks them by ~7e-8 per MMA of a window in the mean, so the leading product has its own
// accumulator, in windows of 4 MMAs added in FP32 registers (at most 64 windows: longer panels are cut into segments
// with their own S), and the other four, 2^-8 of it, share one for the whole segment.   (All five in one accumulator
// with windows of 20: error of the loss 4.2e-6 where the direct kernel has 2.5e-6.)  W and S in three terms, six
// products (k_spec_kk_tc, the same two accumulators), node chunks added in FP64.  The diagonal from the three-term
// |rho|^2: FP32 sums of 128 transitions added in FP64 and rounded to FP32 per node, FP32 sums of 32 nodes added in FP64.
// Re W and Im W meet S separately, so the loss is not left over from products of size |Re W||rho|^2 as in the
// direct kernel: measured error of the loss with local fields 1.4e-6 against the direct kernel's 2.3e-6 (200 w, N_G = 181).
//
// Steps: energy range; stable radix sort of the transitions by panel; plan (segments, 16-transition stages); Lagrange
// weights; rho~ gathered into stage-contiguous, pre-swizzled tiles (a stage is one plain bulk copy per plane);
// k_pn_gram, which writes S as BF16 planes; contraction with W; diagonal; Dyson step.
//
// k_pn_gram is k_chi0_tc (same roles, same stage) made persistent over (segment, G' block, G chunk, node): segments are
// ~15 stages long, so the drain warps write one item's S while the next one's MMAs run.  Tiles cover each pair of G'
// blocks once (pair_cover).  A stage of 128 columns takes ~1680 cycles: 640 of MMA issue, ~1020 of shared-memory traffic
// (operands of the MMAs 80 KB, A tiles written 24 KB, copies and reads 24 KB at 128 B per cycle), the rest the ring's
// hand-overs, so fewer and wider tiles win.
// Measured (one q, 200 w, N_t = 65536, N_G = 181): chi0 14.8 -> 2.9 ms (S 1.19, contraction with W 1.03, gather 0.15);
// 100 w, N_t = 57344, N_G = 531: 56 -> 21 ms.
#include "qcx_internal.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cmath>

namespace {

constexpr int PN_NODES = 16;                // nodes per panel
constexpr double PN_HALF = 2.0 / 3.0;       // panel half width / eta
constexpr int PN_SEG = 2048;                // transitions per segment (64 accumulation windows)
constexpr int PN_TPS = KSTEP / 2;           // transitions per K stage
constexpr int PN_MAXPANELS = 65536;
constexpr int PN_CHUNK_NODES = 4096;        // nodes contracted with W in one FP32 chain
constexpr size_t GATHER_BYTES = 48ull << 20; // rows of rho~ that the gather reads together (the L2 has 129 MB)
constexpr size_t PN_BYTES = 4ull << 30;     // S of a chunk of segments

// ------------------------------------------------------------------ energies, sort, plan
__device__ __forceinline__ unsigned long long order_key(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return b >> 63 ? ~b : b | (1ull << 63);
}
__device__ __forceinline__ double transition(long long t, int nv, int nc, const double* Ek, const double* Ekq) {
    const int nvc = nv * nc;
    const long long k = t / nvc;
    const int rem = (int)(t - k * nvc);
    const int v = rem / nc, c = rem - v * nc;
    return Ekq[k * nc + c] - Ek[k * nv + v];
}

// out: {~key(min) as a maximum, key(max), 1 if any is not finite}
__global__ void __launch_bounds__(256) k_pn_range(long long nt, int nv, int nc, const double* Ek, const double* Ekq,
                                                  unsigned long long* out) {
    unsigned long long lo = 0, hi = 0;
    bool bad = false;
    for (long long t = blockIdx.x * 256LL + threadIdx.x; t < nt; t += 256LL * gridDim.x) {
        const double e = transition(t, nv, nc, Ek, Ekq);
        bad |= !isfinite(e);
        const unsigned long long k = order_key(e);
        lo = max(lo, ~k);
        hi = max(hi, k);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = max(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    bad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(out, lo);
        atomicMax(out + 1, hi);
        if (bad) atomicMax(out + 2, 1ull);
    }
}

__global__ void k_pn_keys(long long nt, int nv, int nc, const double* Ek, const double* Ekq, double e0, double width,
                          int npanel, uint32_t* keys) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nt; t += (long long)gridDim.x * blockDim.x)
        keys[t] = (uint32_t)min(npanel - 1, max(0, (int)((transition(t, nv, nc, Ek, Ekq) - e0) / width)));
}

// Stable LSD radix sort, digits of nd values.  One warp per 1024 items, in order, so equal keys keep their order and
// every sum below runs in a fixed order.
constexpr int RS_ITEMS = 1024, RS_DIGITS = 1024;
__global__ void __launch_bounds__(32) k_pn_hist(long long n, int nd, int shift, int mask, const uint32_t* keys, int* cnt) {
    __shared__ int h[RS_DIGITS];
    const int lane = threadIdx.x;
    for (int d = lane; d < nd; d += 32) h[d] = 0;
    __syncwarp();
    const long long i0 = (long long)blockIdx.x * RS_ITEMS;
    for (int r = 0; r < RS_ITEMS; r += 32)
        if (i0 + r + lane < n) atomicAdd(&h[(keys[i0 + r + lane] >> shift) & mask], 1);
    __syncwarp();
    for (int d = lane; d < nd; d += 32) cnt[(size_t)d * gridDim.x + blockIdx.x] = h[d];
}
__global__ void __launch_bounds__(1024) k_pn_scan(long long n, int* v) {      // exclusive, in place, one block
    __shared__ int part[32];
    __shared__ int carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    for (long long i0 = 0; i0 < n; i0 += 4096) {
        __syncthreads();
        int x[4], s = 0;
        const long long i = i0 + threadIdx.x * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u] = i + u < n ? v[i + u] : 0;
            s += x[u];
        }
        int inc = s;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) part[warp] = inc;
        __syncthreads();
        int base = carry;
        for (int w = 0; w < warp; ++w) base += part[w];
        int run = base + inc - s;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i + u < n) v[i + u] = run;
            run += x[u];
        }
        __syncthreads();
        if (threadIdx.x == 1023) carry = base + inc;
    }
}
// vin null: the values are the item numbers
__global__ void __launch_bounds__(32) k_pn_scatter(long long n, int nd, int shift, int mask, const uint32_t* kin,
                                                   const int* vin, const int* cnt, uint32_t* kout, int* vout) {
    __shared__ int base[RS_DIGITS];
    const int lane = threadIdx.x;
    for (int d = lane; d < nd; d += 32) base[d] = cnt[(size_t)d * gridDim.x + blockIdx.x];
    __syncwarp();
    const long long i0 = (long long)blockIdx.x * RS_ITEMS;
    for (int r = 0; r < RS_ITEMS; r += 32) {
        const long long i = i0 + r + lane;
        const bool on = i < n;
        const uint32_t k = on ? kin[i] : 0u;
        const int v = on ? (vin ? vin[i] : (int)i) : 0;
        const int d = on ? (int)((k >> shift) & mask) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(same & ((1u << lane) - 1));
        const int at = on ? base[d] + rank : 0;
        __syncwarp();
        if (on) {
            if (rank == 0) base[d] = at + __popc(same);
            kout[at] = k;
            vout[at] = v;
        }
        __syncwarp();
    }
}

// Segments of the non-empty panels in order: seg {panel, first sorted item, items, first stage}; total {segments, stages}.
__global__ void __launch_bounds__(1024) k_pn_plan(int n, int npanel, const uint32_t* keys, int4* seg, int* total) {
    __shared__ int ps[1024], pt[1024];
    const int per = (npanel + 1023) / 1024;
    const int lo = min(npanel, (int)threadIdx.x * per), hi = min(npanel, lo + per);
    auto first = [&](int p) {                              // items with a key below p
        int a = 0, b = n;
        while (a < b) {
            const int m = (a + b) >> 1;
            if (keys[m] < (uint32_t)p)
                a = m + 1;
            else
                b = m;
        }
        return a;
    };
    int ns = 0, nst = 0;
    const int begin = first(lo);
    for (int pass = 0, s = 0, st = 0; pass < 2; ++pass) {
        int at = begin;
        for (int p = lo; p < hi; ++p) {
            const int e = first(p + 1);
            for (; at < e; at += min(PN_SEG, e - at)) {
                const int c = min(PN_SEG, e - at);
                if (pass) seg[s] = make_int4(p, at, c, st);
                ++s;
                st += (c + PN_TPS - 1) / PN_TPS;
            }
            at = e;
        }
        if (pass == 0) {
            ns = s;
            nst = st;
            ps[threadIdx.x] = ns;
            pt[threadIdx.x] = nst;
            __syncthreads();
            for (int d = 1; d < 1024; d <<= 1) {
                const int a = threadIdx.x >= (unsigned)d ? ps[threadIdx.x - d] : 0;
                const int b = threadIdx.x >= (unsigned)d ? pt[threadIdx.x - d] : 0;
                __syncthreads();
                ps[threadIdx.x] += a;
                pt[threadIdx.x] += b;
                __syncthreads();
            }
            s = ps[threadIdx.x] - ns;
            st = pt[threadIdx.x] - nst;
            if (threadIdx.x == 1023) {
                total[0] = ps[1023];
                total[1] = pt[1023];
            }
        }
    }
}

// ------------------------------------------------------------------ weights, operands
// node j of [-1, 1]: Chebyshev points of the first kind
__device__ __forceinline__ double node_x(int j) { return cospi((2 * j + 1) / (2.0 * PN_NODES)); }

// Per segment: the transitions of its stages (-1 where padded) and their Lagrange weights in barycentric form (Berrut
// and Trefethen, SIAM Rev. 46, 2004): l_j(x) = [b_j/(x - x_j)] / sum_i b_i/(x - x_i), b_j = (-1)^j sin((2j+1) pi/2n).
__global__ void __launch_bounds__(128) k_pn_weights(const int4* seg, const int* perm, int nv, int nc, const double* Ek,
                                                    const double* Ekq, double e0, double width, long long ldl, int* tr,
                                                    float* Lw) {
    __shared__ double xs[PN_NODES], bs[PN_NODES];
    if (threadIdx.x < PN_NODES) {
        xs[threadIdx.x] = node_x(threadIdx.x);
        const double s = sinpi((2 * (int)threadIdx.x + 1) / (2.0 * PN_NODES));
        bs[threadIdx.x] = threadIdx.x & 1 ? -s : s;
    }
    __syncthreads();
    const int4 g = seg[blockIdx.x];
    const int padded = (g.z + PN_TPS - 1) / PN_TPS * PN_TPS;
    const double mid = e0 + (g.x + 0.5) * width, inv = 2.0 / width;
    for (int i = threadIdx.x; i < padded; i += 128) {
        const long long o = (long long)g.w * PN_TPS + i;
        const int t = i < g.z ? perm[g.y + i] : -1;
        tr[o] = t;
        double l[PN_NODES], sum = 0.0;
        int hit = -1;
        if (t >= 0) {
            const double x = (transition(t, nv, nc, Ek, Ekq) - mid) * inv;
#pragma unroll
            for (int j = 0; j < PN_NODES; ++j) {
                const double d = x - xs[j];
                if (d == 0.0) hit = j;
                l[j] = bs[j] / d;
                sum += l[j];
            }
        }
        const double r = 1.0 / sum;
#pragma unroll
        for (int j = 0; j < PN_NODES; ++j)
            Lw[j * ldl + o] = t < 0 ? 0.f : (hit >= 0 ? (hit == j ? 1.f : 0.f) : (float)(l[j] * r));
    }
}

// rho~ (first two planes) into stage tiles [stage][ngp rows][64 bytes], 64-byte swizzle, and |rho|^2 (three planes) as
// [transition][ngp].  Thread: 4 transitions of one G; a warp covers 8 G, so its writes are contiguous.  Sorted
// transitions lie anywhere in a row of rho~, so the 4-byte reads use a sector eight times over the whole pass: G is
// walked in groups of 2^lg rows whose three planes stay in the L2 while all stages read them.
// One q, N_t = 65536, N_G = 181: all rows at once 336 us, groups of 32 148 us.
__global__ void __launch_bounds__(256) k_pn_gather(int ngp, int lg, long long nst, const int* tr, const uint32_t* p0,
                                                   const uint32_t* p1, const uint32_t* p2, long long kp2,
                                                   unsigned char* t0, unsigned char* t1, float* r2) {
    const long long per = nst << lg, n = ((ngp + (1 << lg) - 1) >> lg) * per * 4;
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += 256LL * gridDim.x) {
        const int j = (int)(i & 3);
        const long long grp = (i >> 2) / per, row = (i >> 2) - grp * per;
        const int G = (int)(grp << lg) + (int)(row & ((1 << lg) - 1));
        const long long st = row >> lg;
        if (G >= ngp) continue;
        const int4 t = *reinterpret_cast<const int4*>(tr + st * PN_TPS + 4 * j);
        const int tt[4] = {t.x, t.y, t.z, t.w};
        uint32_t a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long o = (long long)G * kp2 + tt[u];
            a[u] = tt[u] >= 0 ? p0[o] : 0u;
            b[u] = tt[u] >= 0 ? p1[o] : 0u;
            const uint32_t c = tt[u] >= 0 ? p2[o] : 0u;
            const float2 fa = bf2(a[u]), fb = bf2(b[u]), fc = bf2(c);
            const float re = (fa.x + fb.x) + fc.x, im = (fa.y + fb.y) + fc.y;
            r2[(st * PN_TPS + 4 * j + u) * ngp + G] = re * re + im * im;
        }
        const size_t o = (size_t)st * ngp * ROWB + sw64_off(G, j);
        *reinterpret_cast<uint4*>(t0 + o) = make_uint4(a[0], a[1], a[2], a[3]);
        *reinterpret_cast<uint4*>(t1 + o) = make_uint4(b[0], b[1], b[2], b[3]);
    }
}

// W(w; E_b) of every node: FP32 table [nw][ld] and three BF16 planes [rows][ld], row 2 w + r; zero in the padding
__global__ void k_pn_ktab(int nw, int rows, long long ld, int nb, const double* w, double eta, const int4* seg, double e0,
                          double width, float2* K, __nv_bfloat16* p0, __nv_bfloat16* p1, __nv_bfloat16* p2) {
    const long long n = (long long)(rows / 2) * ld;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int iw = (int)(i / ld);
        const long long b = i - (long long)iw * ld;
        float2 v = make_float2(0.f, 0.f);
        if (iw < nw && b < nb) {
            const double E = e0 + width * (seg[b / PN_NODES].x + 0.5 + 0.5 * node_x((int)(b % PN_NODES)));
            const double x1 = w[iw] - E, x2 = w[iw] + E;
            const double n1 = x1 * x1 + eta * eta, n2 = x2 * x2 + eta * eta;
            const double r = 1.0 / (n1 * n2);
            const double d1 = n2 * r, d2 = n1 * r;
            v = make_float2((float)(x1 * d1 - x2 * d2), (float)(eta * (d2 - d1)));
        }
        if (iw < nw) K[i] = v;
        uint32_t q0, q1, q2;
        split3(v.x, v.y, q0, q1, q2);
        const long long o = 2LL * iw * ld + b;
        const uint32_t q[3] = {q0, q1, q2};
        __nv_bfloat16* p[3] = {p0, p1, p2};
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            p[u][o] = __ushort_as_bfloat16((unsigned short)(q[u] & 0xffffu));
            p[u][o + ld] = __ushort_as_bfloat16((unsigned short)(q[u] >> 16));
        }
    }
}

// ------------------------------------------------------------------ S on the tensor cores
// Warp roles, register budgets, ring and windows of k_chi0_tc.
constexpr int PG_THREADS = 640;
constexpr int PG_LAUNCH_REGS = 96;
constexpr int PG_REG_CTRL = 40, PG_REG_AGEN = 64, PG_REG_DRAIN = 152;
static_assert(128 * PG_REG_CTRL + 256 * PG_REG_AGEN + 256 * PG_REG_DRAIN <= PG_THREADS * PG_LAUNCH_REGS,
              "warpgroup register budgets exceed the launch allocation");
constexpr int PG_MMA2 = 2, PG_AGEN0 = 4, PG_DRAIN0 = 12;
constexpr int PG_NSTAGE = 4;                // ring at least; one more stage where the shared memory holds it
constexpr int PG_PROMOTE = 2;
constexpr int PG_AWARPS = 4;                // warps that form one stage's A tiles (two such groups)
constexpr int PG_NMAX = 128;                // columns of a tile at most
constexpr int PG_MAXHALF = PG_NMAX / 2;
constexpr int PG_GBLK = 64;
constexpr uint32_t PG_ATILE = 128 * ROWB;
constexpr int PG_SMEM_LIMIT = 232448;
static_assert(PN_SEG / PN_TPS / PG_PROMOTE <= 64, "FP32 register sums of at most 64 windows");

struct PgArgs {
    int ng, ngp, n_max, with_src;         // widest tile; whether tiles may lack their own G' rows
    int ntile;                            // tiles per segment
    const int4* tiles;                    // {G' block, first column, columns, A rows from B}
    const int4* seg;                      // segments of this chunk
    int nseg;
    const unsigned char* t0;              // stage tiles of the two planes
    const unsigned char* t1;
    const float* Lw;                      // [16][ldl]
    long long ldl;
    int npair_row;                        // 32-tiles per row of the pair triangle
    long long ncol, plane;                // columns of S (2 x 1024 x pairs), elements of a plane
    __nv_bfloat16* S;                     // three planes [node][ncol], column ((pair 32 + G in 32) 2 + part) 32 + (G' in 32)
    int* status;
    long long wait_limit;
    int withhold;                         // fault injection: no copies
};

struct PgItem {
    int gb, n0, n, from_b, node, stage0, nst, slot;
};
__device__ __forceinline__ PgItem pg_item(const PgArgs& a, int it) {
    PgItem r;
    r.node = it % PN_NODES;
    const int q = it / PN_NODES;
    const int4 t = a.tiles[q % a.ntile];
    r.slot = q / a.ntile;
    const int4 s = a.seg[r.slot];
    r.gb = t.x;
    r.n0 = t.y;
    r.n = t.z;
    r.from_b = t.w;
    r.stage0 = s.w;
    r.nst = (s.z + PN_TPS - 1) / PN_TPS;
    return r;
}

template <int NST> __global__ void __launch_bounds__(PG_THREADS, 1) k_pn_gram(const __grid_constant__ PgArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bplane = (uint32_t)a.n_max * ROWB;
    const uint32_t splane = a.with_src ? (uint32_t)PG_GBLK * ROWB : 0u;
    const uint32_t aoff = 2 * (bplane + splane);
    const uint32_t stage_bytes = aoff + 3 * PG_ATILE;
    unsigned char* tail = base + NST * stage_bytes;
    float* Lbuf = reinterpret_cast<float*>(tail);                 // [NST][16]
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail + NST * PN_TPS * sizeof(float));
    uint64_t* full_b = bars;                                       // [2 NST] by stage mod 2 NST (see k_chi0_tc)
    uint64_t* full_a = bars + 2 * NST;                       // [2 NST]
    uint64_t* empty = bars + 4 * NST;                        // [NST]
    uint64_t* acc_full = bars + 5 * NST;                     // [2]
    uint64_t* drained = acc_full + 2;                              // [2]
    uint64_t* mma_done = drained + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * NST; ++s) {
            mbar_init(&full_b[s], 1);
            mbar_init(&full_a[s], PG_AWARPS);
        }
        for (int s = 0; s < NST; ++s) mbar_init(&empty[s], 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&drained[b], 8);
        }
        mbar_init(mma_done, 2);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, 4 * PG_NMAX);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int nitem = a.nseg * a.ntile * PN_NODES;
    // gs and gw count this CTA's stages and windows over all its items

    if (warp < PG_AGEN0) {
        regs_dec<PG_REG_CTRL>();
        if (warp == 0) {
            if (lane == 0) {
                int gs = 0;
                bool ok = true;
                // with copies withheld nothing is issued and the consumers' first waits run out
                for (int im = a.withhold ? nitem : blockIdx.x; im < nitem && ok; im += gridDim.x) {
                    const PgItem m = pg_item(a, im);
                    const uint32_t bb = (uint32_t)m.n * ROWB;
                    const uint32_t b1 = (uint32_t)min(m.n, a.ngp - m.n0) * ROWB;   // the columns wrap around ngp
                    const uint32_t sb = m.from_b ? 0u : (uint32_t)min(PG_GBLK, a.ngp - m.gb * PG_GBLK) * ROWB;
                    for (int it = 0; it < m.nst; ++it, ++gs) {
                        const int s = gs % NST;
                        if (!(ok = mbar_wait(&empty[s], ((uint32_t)(gs / NST) & 1u) ^ 1u, abort_flag, a.status,
                                             a.wait_limit)))
                            break;
                        uint64_t* fb = &full_b[gs % (2 * NST)];
                        unsigned char* st = base + s * stage_bytes;
                        const size_t stage = (size_t)(m.stage0 + it);
                        const size_t top = stage * a.ngp * ROWB, row = top + (size_t)m.n0 * ROWB;
                        mbar_arrive_tx(fb, 2 * (bb + sb) + PN_TPS * (uint32_t)sizeof(float));
                        bulk_load(Lbuf + s * PN_TPS, a.Lw + m.node * a.ldl + stage * PN_TPS, PN_TPS * sizeof(float), fb);
                        bulk_load(st, a.t0 + row, b1, fb);
                        bulk_load(st + bplane, a.t1 + row, b1, fb);
                        if (b1 < bb) {
                            bulk_load(st + b1, a.t0 + top, bb - b1, fb);
                            bulk_load(st + bplane + b1, a.t1 + top, bb - b1, fb);
                        }
                        if (sb) {
                            const size_t src = (stage * a.ngp + (size_t)m.gb * PG_GBLK) * ROWB;
                            bulk_load(st + 2 * bplane, a.t0 + src, sb, fb);
                            bulk_load(st + 2 * bplane + splane, a.t1 + src, sb, fb);
                        }
                    }
                }
                // every copy in flight lands before the CTA can exit
                for (int it = max(0, gs - NST); it < gs; ++it)
                    mbar_wait(&full_b[it % (2 * NST)], (uint32_t)(it / (2 * NST)) & 1u, abort_flag, a.status,
                              CLEANUP_WAIT_LIMIT, false);
            }
        } else if (warp == 1 || warp == PG_MMA2) {
            if (lane == 0) {
                const int par = warp == 1 ? 0 : 1;
                int gs = 0, gw = 0;
                bool ok = true;
                for (int im = blockIdx.x; im < nitem && ok; im += gridDim.x) {
                    const PgItem m = pg_item(a, im);
                    const uint32_t idesc = make_idesc(128, m.n);
                    for (int it0 = 0; it0 < m.nst && ok; it0 += PG_PROMOTE, ++gw) {
                        const int len = min(PG_PROMOTE, m.nst - it0);
                        if ((gw & 1) != par) {
                            gs += len;
                            continue;
                        }
                        if (gw >= 2 && !(ok = mbar_wait(&drained[par], (uint32_t)((gw - 2) >> 1) & 1u, abort_flag, a.status,
                                                        a.wait_limit)))
                            break;
                        // leading products, and the four of order 2^-8 and below (drained once per item)
                        const uint32_t d = tmem + (uint32_t)par * PG_NMAX, dl = d + 2 * PG_NMAX;
                        const bool first = it0 < 2 * PG_PROMOTE;       // this issuer's first window of the item
                        for (int u = 0; u < len; ++u, ++gs) {
                            const int s = gs % NST;
                            if (!(ok = mbar_wait(&full_a[gs % (2 * NST)], (uint32_t)(gs / (2 * NST)) & 1u,
                                                 abort_flag, a.status, a.wait_limit)))
                                break;
                            tc_fence_after();
                            const uint32_t b0 = smem_u32(base + s * stage_bytes), b1 = b0 + bplane;
                            const uint32_t a0 = b0 + aoff, a1 = a0 + PG_ATILE, a2 = a1 + PG_ATILE;
#pragma unroll
                            for (int kk = 0; kk < KSTEP / 16; ++kk) {
                                const uint32_t off = kk * 32;
                                umma_bf16(d, sw64_desc(a0 + off), sw64_desc(b0 + off), idesc, (u == 0 && kk == 0) ? 0u : 1u);
                                umma_bf16(dl, sw64_desc(a0 + off), sw64_desc(b1 + off), idesc,
                                          (first && u == 0 && kk == 0) ? 0u : 1u);
                                umma_bf16(dl, sw64_desc(a1 + off), sw64_desc(b0 + off), idesc, 1u);
                                umma_bf16(dl, sw64_desc(a1 + off), sw64_desc(b1 + off), idesc, 1u);
                                umma_bf16(dl, sw64_desc(a2 + off), sw64_desc(b0 + off), idesc, 1u);
                            }
                            umma_commit(&empty[s]);
                        }
                        if (ok) umma_commit(&acc_full[par]);
                    }
                }
                // no MMA of either issuer may still be running when TMEM is freed (also on the abort path)
                umma_commit(mma_done);
                mbar_wait(mma_done, 0, abort_flag, a.status, CLEANUP_WAIT_LIMIT, false);
            }
        }
    } else if (warp < PG_DRAIN0) {
        regs_dec<PG_REG_AGEN>();
        // A stage takes a warp mostly latency (its wait, loads, fence), so two groups of four warps take alternate stages
        // (eight warps on every stage: 1224 us where this takes 1186, N_G = 181; 10.8 and 10.3 ms, N_G = 531)
        const int g = threadIdx.x - 32 * PG_AGEN0, group = g / (32 * PG_AWARPS);
        const int j = g & 3, go = (g >> 2) & 31;                   // 4 transitions of G' rows go and go + 32
        int gs = 0;
        bool ok = true;
        for (int im = blockIdx.x; im < nitem && ok; im += gridDim.x) {
            const PgItem m = pg_item(a, im);
            const uint32_t src = m.from_b ? 0u : 2 * bplane, src_plane = m.from_b ? bplane : splane;
            for (int it = 0; it < m.nst; ++it, ++gs) {
                if ((gs & 1) != group) continue;
                const int s = gs % NST, s2 = gs % (2 * NST);
                if (!(ok = warp_wait(&full_b[s2], (uint32_t)(gs / (2 * NST)) & 1u, abort_flag, a.status, a.wait_limit)))
                    break;
                unsigned char* st = base + s * stage_bytes;
                const float4 l = reinterpret_cast<const float4*>(Lbuf + s * PN_TPS)[j];
                const float lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int row = go + 32 * r;
                    uint32_t re0[4] = {0, 0, 0, 0}, re1[4] = {0, 0, 0, 0}, re2[4] = {0, 0, 0, 0};
                    if (m.gb * PG_GBLK + row < a.ng) {
                        const uint32_t coff = src + sw64_off(row, j);
                        const uint4 h0 = *reinterpret_cast<const uint4*>(st + coff);
                        const uint4 h1 = *reinterpret_cast<const uint4*>(st + src_plane + coff);
                        const uint32_t v0[4] = {h0.x, h0.y, h0.z, h0.w}, v1[4] = {h1.x, h1.y, h1.z, h1.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 f0 = bf2(v0[q]), f1 = bf2(v1[q]);   // rho~ = f0 + f1 is exact in FP32
                            split3(lv[q] * (f0.x + f1.x), lv[q] * (f0.y + f1.y), re0[q], re1[q], re2[q]);
                        }
                    }
                    unsigned char* o_re = st + aoff + sw64_off(row, j);
                    unsigned char* o_im = st + aoff + sw64_off(64 + row, j);
                    *reinterpret_cast<uint4*>(o_re) = make_uint4(re0[0], re0[1], re0[2], re0[3]);
                    *reinterpret_cast<uint4*>(o_re + PG_ATILE) = make_uint4(re1[0], re1[1], re1[2], re1[3]);
                    *reinterpret_cast<uint4*>(o_re + 2 * PG_ATILE) = make_uint4(re2[0], re2[1], re2[2], re2[3]);
                    *reinterpret_cast<uint4*>(o_im) = make_uint4(perm_im(re0[0]), perm_im(re0[1]), perm_im(re0[2]), perm_im(re0[3]));
                    *reinterpret_cast<uint4*>(o_im + PG_ATILE) =
                        make_uint4(perm_im(re1[0]), perm_im(re1[1]), perm_im(re1[2]), perm_im(re1[3]));
                    *reinterpret_cast<uint4*>(o_im + 2 * PG_ATILE) =
                        make_uint4(perm_im(re2[0]), perm_im(re2[1]), perm_im(re2[2]), perm_im(re2[3]));
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full_a[s2]);
            }
        }
    } else {
        regs_inc<PG_REG_DRAIN>();
        const int q = warp & 3, hc = (warp - PG_DRAIN0) >> 2;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        float part[PG_MAXHALF];
        int gw = 0;
        bool ok = true;
        for (int im = blockIdx.x; im < nitem && ok; im += gridDim.x) {
            const PgItem m = pg_item(a, im);
            const int half = m.n >> 1, nch16 = half >> 4;
            const bool tail8 = (half & 15) != 0;
#pragma unroll
            for (int i = 0; i < PG_MAXHALF; ++i) part[i] = 0.0f;
            for (int it0 = 0; it0 < m.nst && ok; it0 += PG_PROMOTE, ++gw) {
                const int b = gw & 1;
                if (!(ok = warp_wait(&acc_full[b], (uint32_t)(gw >> 1) & 1u, abort_flag, a.status, a.wait_limit))) break;
                tc_fence_after();
                // with an issuer's last window of the item, its low-order sums too
                const int nsum = it0 + 2 * PG_PROMOTE >= m.nst ? 2 : 1;
                for (int z = 0; z < nsum; ++z) {
                    const uint32_t tb = tmem + lane_off + (uint32_t)((b + 2 * z) * PG_NMAX + hc * half);
#pragma unroll
                    for (int grp = 0; grp < PG_MAXHALF / 32; ++grp) {
                        uint32_t r[2][16];
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            if (grp * 2 + u < nch16) tmem_ld16(tb + (uint32_t)((grp * 2 + u) * 16), r[u]);
                        tmem_wait_ld();
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            if (grp * 2 + u < nch16) {
#pragma unroll
                                for (int i = 0; i < 16; ++i) part[(grp * 2 + u) * 16 + i] += __uint_as_float(r[u][i]);
                            }
                    }
                    if (tail8) {
                        uint32_t r8[8];
                        tmem_ld8(tb + (uint32_t)(nch16 * 16), r8);
                        tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < PG_MAXHALF; c += 8)
                            if (c == nch16 * 16) {
#pragma unroll
                                for (int i = 0; i < 8; ++i) part[c + i] += __uint_as_float(r8[i]);
                            }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&drained[b]);
            }
            if (!ok) break;
            // S of this item in three BF16 terms: the warp's 32 rows are one 32-tile of G'.  Above the diagonal two
            // columns at a time, even lanes writing the first as pairs of rows, odd lanes the second; below it (another
            // block's columns, wrapped) the conjugate, eight columns of a row at a time
            const int gi = m.gb * 2 + (q & 1), part_im = q >> 1;   // G' tile; real or imaginary rows
            if (gi < a.npair_row) {
                __nv_bfloat16* S = a.S + ((size_t)m.slot * PN_NODES + m.node) * a.ncol + part_im * 32;
                const int c0 = m.n0 + hc * half;
#pragma unroll
                for (int c = 0; c < PG_MAXHALF; c += 8) {
                    if (c >= half) break;
                    const int G0 = c0 + c < a.ngp ? c0 + c : c0 + c - a.ngp, hi = G0 >> 5;
                    if (hi >= gi) {
                        const int p = gi * a.npair_row - gi * (gi - 1) / 2 + hi - gi;
                        const bool odd = lane & 1;
                        uint32_t* o = reinterpret_cast<uint32_t*>(S + (size_t)(p * 32 + (G0 & 31) + (odd ? 1 : 0)) * 64 + (lane & ~1));
#pragma unroll
                        for (int u = 0; u < 8; u += 2, o += 64) {
                            const float other = __shfl_xor_sync(0xffffffffu, odd ? part[c + u] : part[c + u + 1], 1);
                            uint32_t s0, s1, s2;
                            split3(odd ? other : part[c + u], odd ? part[c + u + 1] : other, s0, s1, s2);
                            o[0] = s0;
                            o[a.plane / 2] = s1;
                            o[a.plane] = s2;
                        }
                    } else if (hi >> 1 != m.gb) {
                        const int p = hi * a.npair_row - hi * (hi - 1) / 2 + gi - hi;
                        const float sg = part_im ? -1.0f : 1.0f;
                        uint32_t s0[4], s1[4], s2[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            split3(sg * part[c + 2 * u], sg * part[c + 2 * u + 1], s0[u], s1[u], s2[u]);
                        uint4* o = reinterpret_cast<uint4*>(S + (size_t)(p * 32 + lane) * 64 + (G0 & 31));
                        o[0] = make_uint4(s0[0], s0[1], s0[2], s0[3]);
                        o[a.plane / 8] = make_uint4(s1[0], s1[1], s1[2], s1[3]);
                        o[a.plane / 4] = make_uint4(s2[0], s2[1], s2[2], s2[3]);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 4 * PG_NMAX);
    }
}

// ------------------------------------------------------------------ diagonal, Dyson step
// Sd[b][G] = sum_t l_j |rho_t(G)|^2: CTA (segment, 128 G)
__global__ void __launch_bounds__(128) k_pn_diag(int ngp, const int4* seg, const float* r2, const float* Lw, long long ldl,
                                                 float* Sd) {
    __shared__ float l[PN_NODES][128];
    const int4 g = seg[blockIdx.x];
    const int G = blockIdx.y * 128 + threadIdx.x;
    const int n = (g.z + PN_TPS - 1) / PN_TPS * PN_TPS;
    const long long o = (long long)g.w * PN_TPS;
    double sum[PN_NODES];
    float acc[PN_NODES];
#pragma unroll
    for (int j = 0; j < PN_NODES; ++j) {
        sum[j] = 0.0;
        acc[j] = 0.f;
    }
    for (int i0 = 0; i0 < n; i0 += 128) {
        const int m = min(128, n - i0);
        __syncthreads();
        for (int j = 0; j < PN_NODES; ++j)
            if (threadIdx.x < m) l[j][threadIdx.x] = Lw[j * ldl + o + i0 + threadIdx.x];
        __syncthreads();
        if (G < ngp)
            for (int i = 0; i < m; ++i) {
                const float x = r2[(o + i0 + i) * ngp + G];
#pragma unroll
                for (int j = 0; j < PN_NODES; ++j) acc[j] = fmaf(l[j][i], x, acc[j]);
            }
#pragma unroll
        for (int j = 0; j < PN_NODES; ++j) {
            sum[j] += (double)acc[j];
            acc[j] = 0.f;
        }
    }
    if (G < ngp)
#pragma unroll
        for (int j = 0; j < PN_NODES; ++j) Sd[((size_t)blockIdx.x * PN_NODES + j) * ngp + G] = (float)sum[j];
}

// part[z][w][G] = sum over the nodes of range z of W(w; E_b) Sd[b][G]; CTA 32 w x 32 G, thread 2 x 2, sums of
// 32 in FP32 added in FP64 (factors as FP32 pairs changed nothing in the loss).
__global__ void __launch_bounds__(256) k_pn_diag_chi(int nw, int ng, int ngp, int nb, int per, const float2* K, long long ld,
                                                     const float* Sd, double2* part) {
    __shared__ float2 Ks[32][33];
    __shared__ float Rs[32][33];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int G0 = blockIdx.x * 32, w0 = blockIdx.y * 32;
    const int b_lo = blockIdx.z * per, b_hi = min(nb, b_lo + per);
    double2 sum[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) sum[i][j] = make_double2(0.0, 0.0);
    for (int b0 = b_lo; b0 < b_hi; b0 += 32) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = threadIdx.x + 256 * r, a = i & 31, c = i >> 5;
            Ks[a][c] = b0 + a < b_hi && w0 + c < nw ? K[(long long)(w0 + c) * ld + b0 + a] : make_float2(0.f, 0.f);
            Rs[c][a] = b0 + c < b_hi && G0 + a < ng ? Sd[(size_t)(b0 + c) * ngp + G0 + a] : 0.f;
        }
        __syncthreads();
        float2 acc[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int b = 0; b < 32; ++b) {
            const float2 k[2] = {Ks[b][ty], Ks[b][ty + 16]};
            const float r[2] = {Rs[b][tx], Rs[b][tx + 16]};
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    acc[i][j].x = fmaf(k[i].x, r[j], acc[i][j].x);
                    acc[i][j].y = fmaf(k[i].y, r[j], acc[i][j].y);
                }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                sum[i][j].x += (double)acc[i][j].x;
                sum[i][j].y += (double)acc[i][j].y;
            }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int w = w0 + ty + 16 * i, G = G0 + tx + 16 * j;
            if (w < nw && G < ng) part[((size_t)blockIdx.z * nw + w) * ng + G] = sum[i][j];
        }
}

// eps^T (row G', column G) = delta - v^1/2 chi0 v^1/2 from the unscaled chi [w][G][G'], its diagonal from the ranges of
// part; optionally chi0 itself.  Block (32, 8): a 32 x 32 tile through shared memory.
__global__ void __launch_bounds__(256) k_pn_dyson(int ng, int nw, int nz, const double2* chi, const double2* part, double pref,
                                                  const double* vs, double2* eps, double2* chi_out) {
    __shared__ double2 t[32][33];
    const int w = blockIdx.z, G0 = blockIdx.y * 32, H0 = blockIdx.x * 32;
    const size_t o = (size_t)w * ng * ng;
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int G = G0 + j, H = H0 + threadIdx.x;
        if (G >= ng || H >= ng) continue;
        double2 c = chi[o + (size_t)G * ng + H];
        if (G == H) {
            c = make_double2(0.0, 0.0);
            for (int z = 0; z < nz; ++z) {
                const double2 v = part[((size_t)z * nw + w) * ng + G];
                c.x += v.x;
                c.y += v.y;
            }
        }
        t[j][threadIdx.x] = c;
        if (chi_out) chi_out[o + (size_t)G * ng + H] = make_double2(pref * c.x, pref * c.y);
    }
    __syncthreads();
    // three FP64 operations per element: the pipe, not memory, is what this kernel could be bound by
    const double vG = G0 + threadIdx.x < ng ? pref * vs[G0 + threadIdx.x] : 0.0;
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int H = H0 + j, G = G0 + threadIdx.x;
        if (G >= ng || H >= ng) continue;
        const double2 c = t[threadIdx.x][j];
        const double vv = vG * vs[H];
        eps[o + (size_t)H * ng + G] = make_double2(fma(-vv, c.x, G == H ? 1.0 : 0.0), -vv * c.y);
    }
}

inline int blocks(long long n, int t, int cap = 16384) { return (int)std::min<long long>((n + t - 1) / t, cap); }

}  // namespace

// Estimated times (us, measured rates of this GPU).  Direct: 0.85 us x SMs per K stage of a (G' block, chunk, w); panels:
// 0.62 per stage of a tile and node and 1.2 per item, 0.65 per (128 x 128) stage of the contraction with W, the passes
// over S and the gathered operands at ~3 TB/s, and ~200 for the launches and two host round trips.
static double direct_us(const QSlot& s, long long nt) {
    const int chunks = (s.ngp + 191) / 192;
    return (double)((s.ng + 63) / 64) * chunks * s.nw * (double)((nt + 15) / 16) * 0.85 / 152.0;
}
static double panel_us(const QSlot& s, long long nt, double stages, double segs, int ntile) {
    const double T = (s.ng + 31) / 32, pairs = T * (T + 1) / 2, nodes = segs * PN_NODES;
    const double gram = ntile * PN_NODES * (stages * 0.62 + segs * 1.2) / 152.0;
    const double kk = (2.0 * s.nw + 127) / 128 * pairs * 16 * nodes / 32 * 0.65 / 152.0;
    const double bytes = pairs * 1024 * nodes * 12.0 + (double)nt * s.ngp * 40.0 + 48.0 * s.nw * s.ng * (double)s.ng;
    return gram + kk + bytes / 3e6 + 200.0;
}

// The pairs of G' blocks as tiles {G' block, first column, columns (wrapping around ngp), A rows from B}: either every
// block with the columns from its own on (the upper triangle), or with its own and the next floor(blocks / 2) around the
// circle (the pairs half way around an even circle once).  The time of a tile hardly depends on its width, so the one
// with fewer tiles: around the circle for 3 blocks (3 against 4: one q, N_G = 181, 1508 -> 1224 us with the deeper
// ring) and for 7 and 11 or more of an odd number.  Tiles that hold their own rows also need
// no copy of them, which leaves room for a fifth stage.
static std::vector<int4> pair_cover(int ng, int ngp) {
    const int nb = (ng + PG_GBLK - 1) / PG_GBLK;
    std::vector<int4> cover[2];
    for (int gb = 0; gb < nb; ++gb)
        for (int ring = 0; ring < 2; ++ring) {
            const int up = ring ? nb / 2 - (nb % 2 == 0 && gb >= nb / 2) : nb - 1 - gb;      // further blocks
            const int end = (gb + up) % nb;                                                  // the last of them
            const int len = std::min(ngp, (end + 1) * PG_GBLK) - gb * PG_GBLK + (gb + up >= nb ? ngp : 0);
            const int nch = (len + PG_NMAX - 1) / PG_NMAX, step = ((len + nch - 1) / nch + 15) / 16 * 16;
            for (int c = 0; c < len; c += step)
                cover[ring].push_back(make_int4(gb, (gb * PG_GBLK + c) % ngp, std::min(step, len - c), c == 0));
        }
    return cover[cover[1].size() < cover[0].size()];
}

// Tries the panel route.  *used = false (and cudaSuccess) when the direct kernel is to run instead: the estimate above is
// not better, the energies are not finite or span too many panels, or the work space does not fit.
cudaError_t qcx_launch_chi0_panels(qcx_ctx* ctx, QSlot& s, int iq, double2* d_chi, int* d_status, bool* used) {
    *used = false;
    const int ng = s.ng, ngp = s.ngp, nw = s.nw;
    const long long nt = (long long)ctx->nk * ctx->nv * ctx->nc;
    const double direct = direct_us(s, nt);
    // below this the host round trips alone would cost what there is to gain
    if (direct < 600.0) return cudaSuccess;
    const int T32 = (ng + 31) / 32, ntp = T32 * (T32 + 1) / 2;
    if (nw > 65535 || ntp * 16 > 65535) return cudaSuccess;      // grid limits
    const std::vector<int4> tiles = pair_cover(ng, ngp);
    int n_max = 16;
    bool with_src = false;
    for (const int4& t : tiles) {
        n_max = std::max(n_max, t.z);
        with_src |= !t.w;
    }
    const int ntile = (int)tiles.size();
    if (panel_us(s, nt, (double)nt / PN_TPS, 1.0, ntile) >= 0.8 * direct) return cudaSuccess;

    cudaStream_t st = ctx->stream;
    PanelBufs& b = ctx->panels;
    cudaError_t e;
    auto fits = [&](DevBuf& d, size_t n) {
        e = d.ensure(n);
        if (e == cudaErrorMemoryAllocation) cudaGetLastError();
        return e == cudaSuccess;
    };
    auto give_up = [&]() {                       // what did fit would be missing for the direct kernel and the inverse
        b.release();
        return e == cudaErrorMemoryAllocation ? cudaSuccess : e;
    };
    const double* Ek = ctx->d_Ek.as<double>();
    const double* Ekq = ctx->d_Ekq.as<double>() + (size_t)iq * ctx->nk * ctx->nc;
    if (!fits(b.small, 64)) return give_up();
    unsigned long long* d_range = b.small.as<unsigned long long>();
    int* d_total = reinterpret_cast<int*>(d_range + 4);
    if ((e = cudaMemsetAsync(d_range, 0, 64, st)) != cudaSuccess) return e;
    k_pn_range<<<blocks(nt, 256, 152), 256, 0, st>>>(nt, ctx->nv, ctx->nc, Ek, Ekq, d_range);
    unsigned long long range[3];
    if ((e = cudaMemcpyAsync(range, d_range, sizeof(range), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return e;
    auto value = [](unsigned long long k) {
        const unsigned long long u = k >> 63 ? k & ~(1ull << 63) : ~k;
        double x;
        std::memcpy(&x, &u, sizeof(x));
        return x;
    };
    if (range[2]) return cudaSuccess;
    const double e0 = value(~range[0]), e1 = value(range[1]), width = 2.0 * PN_HALF * s.eta;
    if (!((e1 - e0) / width < PN_MAXPANELS - 1)) return cudaSuccess;
    const int npanel = std::max(1, (int)std::floor((e1 - e0) / width) + 1);

    // transitions by panel
    const int nblk = (int)((nt + RS_ITEMS - 1) / RS_ITEMS);
    const bool two = npanel > RS_DIGITS;
    const int nd = two ? 256 : npanel;
    const size_t max_seg = (size_t)npanel + (size_t)(nt / PN_SEG) + 1;
    if (!fits(b.keys, 2 * sizeof(uint32_t) * (size_t)nt) || !fits(b.perm, 2 * sizeof(int) * (size_t)nt) ||
        !fits(b.cnt, sizeof(int) * (size_t)nd * nblk) || !fits(b.seg, sizeof(int4) * (max_seg + ntile)))
        return give_up();
    uint32_t* k0 = b.keys.as<uint32_t>();
    uint32_t* k1 = k0 + nt;
    int* v0 = b.perm.as<int>();
    int* v1 = v0 + nt;
    int4* seg = b.seg.as<int4>();
    int4* d_tiles = seg + max_seg;
    if ((e = cudaMemcpyAsync(d_tiles, tiles.data(), sizeof(int4) * ntile, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    k_pn_keys<<<blocks(nt, 256, 1024), 256, 0, st>>>(nt, ctx->nv, ctx->nc, Ek, Ekq, e0, width, npanel, k0);
    for (int pass = 0; pass < (two ? 2 : 1); ++pass) {
        const int shift = 8 * pass, mask = two ? 255 : 0xffff;
        k_pn_hist<<<nblk, 32, 0, st>>>(nt, nd, shift, mask, pass ? k1 : k0, b.cnt.as<int>());
        k_pn_scan<<<1, 1024, 0, st>>>((long long)nd * nblk, b.cnt.as<int>());
        k_pn_scatter<<<nblk, 32, 0, st>>>(nt, nd, shift, mask, pass ? k1 : k0, pass ? v1 : nullptr, b.cnt.as<int>(),
                                          pass ? k0 : k1, pass ? v0 : v1);
    }
    const uint32_t* ks = two ? k0 : k1;
    const int* perm = two ? v0 : v1;
    k_pn_plan<<<1, 1024, 0, st>>>((int)nt, npanel, ks, seg, d_total);
    int total[2];
    if ((e = cudaMemcpyAsync(total, d_total, sizeof(total), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return e;
    const int nseg = total[0];
    const long long nst = total[1];
    if (panel_us(s, nt, (double)nst, nseg, ntile) >= 0.8 * direct) return cudaSuccess;

    // chunks of segments: nodes per FP32 chain and bytes of S bounded
    const size_t per_seg = (size_t)PN_NODES * ntp * 1024 * 6 * sizeof(__nv_bfloat16);
    const int cap = (int)std::max<size_t>(2, std::min<size_t>(PN_CHUNK_NODES / PN_NODES, PN_BYTES / per_seg)) / 2 * 2;
    const int nchunk = (nseg + cap - 1) / cap;
    const int cseg = ((nseg + nchunk - 1) / nchunk + 1) / 2 * 2;                // even: node chunks are multiples of 32
    const int nbc = cseg * PN_NODES;
    const long long ldl = nst * PN_TPS;
    const int nb = nseg * PN_NODES;
    const long long ldk = (long long)nchunk * nbc;
    const int mtiles = (2 * nw + 127) / 128, ntiles = ntp * 16;
    const size_t kn = (size_t)mtiles * 128 * ldk, sn = (size_t)ntiles * 128 * nbc;
    const size_t tile_bytes = (size_t)nst * ngp * ROWB;
    const int nz = std::max(1, std::min(16, nb / 256)), per = ((nb + nz - 1) / nz + 31) / 32 * 32;
    if (!fits(b.tr, sizeof(int) * (size_t)ldl) || !fits(b.Lw, sizeof(float) * PN_NODES * (size_t)ldl) ||
        !fits(b.tiles, 2 * tile_bytes) || !fits(b.r2, sizeof(float) * (size_t)ldl * ngp) ||
        !fits(b.ktab, sizeof(float2) * (size_t)nw * ldk) || !fits(b.kplanes, 3 * kn * sizeof(__nv_bfloat16)) ||
        !fits(b.splanes, 3 * sn * sizeof(__nv_bfloat16)) ||
        !fits(b.Sd, sizeof(float) * (size_t)nb * ngp) || !fits(b.part, sizeof(double2) * (size_t)nz * nw * ng) ||
        !fits(b.chi, sizeof(double2) * (size_t)nw * ng * ng) || !fits(b.tp, sizeof(int2) * ntp))
        return give_up();
    std::vector<int2> tp;
    for (int gi = 0; gi < T32; ++gi)
        for (int hi = gi; hi < T32; ++hi) tp.push_back(make_int2(hi, gi));    // S element: G in tile hi, G' in tile gi
    if ((e = cudaMemcpyAsync(b.tp.p, tp.data(), sizeof(int2) * ntp, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    *used = true;

    k_pn_weights<<<nseg, 128, 0, st>>>(seg, perm, ctx->nv, ctx->nc, Ek, Ekq, e0, width, ldl, b.tr.as<int>(), b.Lw.as<float>());
    const uint32_t* p0 = reinterpret_cast<const uint32_t*>(s.rho.p);
    const size_t plane = (size_t)ngp * (s.kp / 2);
    unsigned char* t0 = b.tiles.as<unsigned char>();
    int lg = 5;                                              // 8 rows at least: a warp's writes stay contiguous
    while (lg > 3 && (size_t)(s.kp / 2) * 12 << lg > GATHER_BYTES) --lg;
    const long long grows = (ngp + (1 << lg) - 1) >> lg << lg;
    k_pn_gather<<<blocks(nst * grows * 4, 256), 256, 0, st>>>(ngp, lg, nst, b.tr.as<int>(), p0, p0 + plane, p0 + 2 * plane,
                                                            s.kp / 2, t0, t0 + tile_bytes, b.r2.as<float>());
    __nv_bfloat16* kp = b.kplanes.as<__nv_bfloat16>();
    k_pn_ktab<<<blocks((long long)mtiles * 64 * ldk, 256), 256, 0, st>>>(nw, mtiles * 128, ldk, nb, s.w.as<double>(), s.eta, seg,
                                                                         e0, width, b.ktab.as<float2>(), kp, kp + kn, kp + 2 * kn);
    k_pn_diag<<<dim3(nseg, (ngp + 127) / 128), 128, 0, st>>>(ngp, seg, b.r2.as<float>(), b.Lw.as<float>(), ldl, b.Sd.as<float>());
    k_pn_diag_chi<<<dim3((ng + 31) / 32, (nw + 31) / 32, nz), 256, 0, st>>>(nw, ng, ngp, nb, per, b.ktab.as<float2>(), ldk,
                                                                            b.Sd.as<float>(), b.part.as<double2>());
    PgArgs a{};
    a.ng = ng;
    a.ngp = ngp;
    a.n_max = n_max;
    a.with_src = with_src;
    a.ntile = ntile;
    a.tiles = d_tiles;
    a.t0 = t0;
    a.t1 = t0 + tile_bytes;
    a.Lw = b.Lw.as<float>();
    a.ldl = ldl;
    a.npair_row = T32;
    a.ncol = (long long)ntiles * 128;
    a.plane = a.ncol * nbc;
    a.S = b.splanes.as<__nv_bfloat16>();
    a.status = d_status;
    a.wait_limit = ctx->wait_limit;
    a.withhold = ctx->withhold_copies;
    auto ring_bytes = [&](size_t nst) {
        return 1024 + nst * (2 * (n_max + (with_src ? PG_GBLK : 0)) * ROWB + 3 * PG_ATILE + PN_TPS * sizeof(float)) +
               (5 * nst + 5) * sizeof(uint64_t) + 16;
    };
    const bool deep = ring_bytes(PG_NSTAGE + 1) <= PG_SMEM_LIMIT;
    const size_t smem = ring_bytes(PG_NSTAGE + deep);
    const auto gram = deep ? k_pn_gram<PG_NSTAGE + 1> : k_pn_gram<PG_NSTAGE>;
    if (smem > PG_SMEM_LIMIT) return cudaErrorInvalidValue;
    if ((e = qcx_allow_smem((const void*)gram)) != cudaSuccess) return e;
    // the register budgets assume this launch allocation (see k_chi0_tc)
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, (const void*)gram)) != cudaSuccess) return e;
    if (fa.numRegs != PG_LAUNCH_REGS) return cudaErrorNotSupported;
    CUtensorMap kmaps[3], smaps[3];
    __nv_bfloat16* sp = b.splanes.as<__nv_bfloat16>();
    for (int i = 0; i < 3; ++i)
        if (!qcx_make_bf16_map(&kmaps[i], kp + i * kn, ldk, mtiles * 128, 128, 32) ||
            !qcx_make_bf16_map(&smaps[i], sp + i * sn, ntiles * 128, nbc, 32, 64))
            return cudaErrorInvalidValue;
    for (int c = 0; c < nchunk; ++c) {
        const int s0 = c * cseg, m = std::min(cseg, nseg - s0);
        if (m <= 0) break;
        a.seg = seg + s0;
        a.nseg = m;
        gram<<<std::min(152, m * ntile * PN_NODES), PG_THREADS, smem, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // an odd number of segments leaves 16 points of the last stage
        for (int i = 0; i < 3 && m * PN_NODES % KSTEP; ++i)
            if ((e = cudaMemsetAsync(sp + i * sn + (size_t)m * PN_NODES * a.ncol, 0, PN_NODES * a.ncol * sizeof(__nv_bfloat16),
                                     st)) != cudaSuccess)
                return e;
        e = qcx_spec_tc_kk(st, kmaps, smaps, mtiles, ntiles, nw, ng, m * PN_NODES, c * nbc, b.tp.as<int2>(), c > 0,
                           b.chi.as<double2>(), d_status, ctx->wait_limit);
        if (e != cudaSuccess) return e;
    }
    const double* L = ctx->lattice;
    const double vol = fabs(L[0] * (L[4] * L[8] - L[5] * L[7]) - L[1] * (L[3] * L[8] - L[5] * L[6]) +
                            L[2] * (L[3] * L[7] - L[4] * L[6]));
    k_pn_dyson<<<dim3(T32, T32, nw), dim3(32, 8), 0, st>>>(ng, nw, nz, b.chi.as<double2>(), b.part.as<double2>(),
                                                           2.0 / (ctx->nk * vol), s.vs.as<double>(), s.eps.as<double2>(), d_chi);
    return cudaGetLastError();
}
