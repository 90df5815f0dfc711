// Inverse of the dielectric matrices and the loss functions.
//
// eps(w, q+G) = 1/[eps^-1]_GG (Eq. (eps_LFE)); eps^noLFE = eps_GG
// (Eq. (eps_noLFE)); L = Im[-1/eps] (Eq. (dynamic_structure_factor)).
//
// Every (q, w) block is inverted by blocked Gauss-Jordan elimination with partial
// (row) pivoting.  The FP64 path does this in double.  The mixed path
// does it in FP32 on the rounded copy of the FP64 matrix and records the
// condition estimate kappa_1 = |A|_1 |X|_1.  Blocks with kappa_1 above the
// context's threshold (default 1e4; the ill-conditioned ones, near the
// plasmon) then get one FP64 correction of the diagonal against the FP64
// matrix: with R = I - A X, [A^-1]_jj = X_jj + (X R)_jj + O(|R|^2).  The other
// blocks take L_LFE from the quadratic form below, which keeps the relative
// accuracy of X; on the 10 000 blocks of the 181-G workload the 981 with
// kappa_1 in (1e3, 1e4] agree with their FP64-corrected loss to 1.8e-5.
#include "qcx_internal.h"
#include "cplx.cuh"

#include <algorithm>

namespace {

// Blocked in-place Gauss-Jordan over all matrices at once.  Per panel of PB columns:
//
//   k_inv_panel   one CTA per matrix holds the n x PB panel in shared memory and eliminates its columns with
//                 partial pivoting over the rows not used yet (rows are not moved: the CTA records which row
//                 serves as pivot of which column);
//   k_inv_update  every other column at once, out of place (src -> dst), as a product with inner length PB:
//                     dst[i][j] = (i in panel ? 0 : src[p(i)][j]) + sum_c M[i][c] src[p(k0 + c)][j],
//                 where M is the eliminated panel (for a pivot row the inverse of the pivot block, for any other
//                 row minus its multipliers) and p the panel's row exchange.
//
// What bounds it: the rank-1 form rewrote the whole matrix for every one of the n columns (n^3 elements through
// L2, one CTA per matrix, or through shared memory with a cluster barrier per column); this form touches it
// n/PB times and spends 8 n^3 flops in a product that the FP32 (FP64) pipe bounds, with tiles of all matrices in
// one grid.  PB = 32 (FP32) keeps the panel's serial part (two CTA barriers per column, ~0.3 us) below the
// update's time.  Measured (GB300): 200 matrices of 181: 3.33 -> 0.65 ms; 100 of 531: 177 -> 4.9 ms; FP64, 8 of 181:
// 10.8 -> 2.0 ms.
// With P A = rows in pivot order, the eliminated matrix is (P A)^-1, so its column k is the inverse's column
// row(k): the last update writes its columns there.
constexpr int UPD = 64;                     // update tile edge
template <typename T> struct InvCfg;
template <> struct InvCfg<float> { static constexpr int PB = 32; };
template <> struct InvCfg<double> { static constexpr int PB = 16; };
constexpr size_t PANEL_SMEM = 200 * 1024;   // the panel narrows above this (from n = 774 on in FP32 and FP64)
constexpr int PANEL_ROWS = 4;               // rows per thread of the panel at most (n <= 4096)

template <typename T> __device__ __forceinline__ T cabs2(cplx<T> z) { return z.x * z.x + z.y * z.y; }
// |z| without overflow of the squares
__device__ __forceinline__ float cabs_safe(float2 z) {
    const float x = fabsf(z.x), y = fabsf(z.y), m = fmaxf(x, y), r = fminf(x, y);
    if (!(m > 0.f)) return m;
    const float t = r / m;
    return m * sqrtf(fmaf(t, t, 1.f));
}

// order of a squared magnitude as an integer: NaN below everything, zero 1, larger magnitudes larger
__device__ __forceinline__ unsigned long long mag_key(float v) {
    return v >= 0.f ? (unsigned long long)__float_as_uint(v) + 1ull : 0ull;
}
__device__ __forceinline__ unsigned long long mag_key(double v) {
    return v >= 0.0 ? (unsigned long long)__double_as_longlong(v) + 1ull : 0ull;
}
// largest key of the warp; with ties the first lane's `row` wins
template <typename T> __device__ __forceinline__ void warp_best(unsigned long long& key, int& row);
template <> __device__ __forceinline__ void warp_best<float>(unsigned long long& key, int& row) {
    const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)key);
    const int r = (unsigned)key == m ? row : 0x7fffffff;
    row = __reduce_min_sync(0xffffffffu, r);
    key = m;
}
template <> __device__ __forceinline__ void warp_best<double>(unsigned long long& key, int& row) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32) == hi ? (unsigned)key : 0u);
    const unsigned long long m = ((unsigned long long)hi << 32) | lo;
    const int r = key == m ? row : 0x7fffffff;
    row = __reduce_min_sync(0xffffffffu, r);
    key = m;
}

// The matrices of a call: all of order n, or (inst) a batch of uneven ones with their own offsets.  A panel is pb columns;
// matrix b has ceil(n_b / pb) of them, and the last update lands in the first of the two buffers.
struct InvShape {
    int n, pb;
    const BatchInst* inst;
    int b0;                                 // first matrix of the launch
    size_t mat0, vec0;                      // where the second copy's matrices and the panels' rows begin
    __device__ int order(int b) const { return inst ? inst[b].ng : n; }
    __device__ size_t mat(int b) const { return inst ? (size_t)inst[b].work_off : (size_t)b * n * n; }
    __device__ size_t mat2(int b) const { return mat(b) - mat0; }
    __device__ size_t vec(int b) const { return (inst ? (size_t)inst[b].vec_off : (size_t)b * n) - vec0; }
};

// FP64 matrices -> work precision; eps_GG, the loss without local fields, |A|_1 (largest column sum) and the
// starting row order.  Grid (matrix, 64 columns); 64 columns x 4 row groups per CTA.
template <typename T>
__global__ void __launch_bounds__(256) k_inv_load(int n, const double2* A, cplx<T>* X, double* anorm, double2* eps_diag,
                                                  double* L_nolfe, int* rows, int* flags) {
    __shared__ double sums[4][64];
    const int b = blockIdx.x, tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int j = blockIdx.y * 64 + tx;
    A += (size_t)b * n * n;
    X += (size_t)b * n * n;
    double cs = 0.0;
    if (j < n)
        for (int i = ty; i < n; i += 4) {
            const double2 z = A[(size_t)i * n + j];
            const cplx<T> x = mk<T>((T)z.x, (T)z.y);
            X[(size_t)i * n + j] = x;
            if constexpr (sizeof(T) == 4) cs += (double)cabs_safe(x);
            if (i == j) {
                eps_diag[(size_t)b * n + i] = z;
                L_nolfe[(size_t)b * n + i] = z.y / (z.x * z.x + z.y * z.y);
                rows[(size_t)b * n + i] = i;
            }
        }
    if (blockIdx.y == 0 && threadIdx.x == 0) flags[b] = 0;
    if constexpr (sizeof(T) == 4) {
        sums[ty][tx] = cs;
        __syncthreads();
        if (ty == 0 && j < n) {
            cs = (sums[0][tx] + sums[1][tx]) + (sums[2][tx] + sums[3][tx]);
            atomicMax(reinterpret_cast<unsigned long long*>(anorm + b), (unsigned long long)__double_as_longlong(cs));
        }
    }
}

// One panel: columns k0 .. k0 + nb - 1 of every row.  Warps: RW row warps x column groups of bc columns; a thread
// eliminates in its rows (row, row + 32 RW, ...) and its group's columns.  M[c][i] gets the eliminated panel in the
// new row order, perm the exchange (new position -> old position), rows the original row of each position.
template <typename T>
__global__ void __launch_bounds__(1024) k_inv_panel(InvShape sh, int p_, int RW, int bc, const cplx<T>* X, const cplx<T>* B2,
                                                    cplx<T>* M, int* perm, int* rows, int* flags) {
    using C = cplx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = sh.b0 + blockIdx.x, n = sh.order(b), npan = (n + sh.pb - 1) / sh.pb;
    if (p_ >= npan || flags[b]) return;
    const int k0 = p_ * sh.pb, nb = min(sh.pb, n - k0);
    const C* src = (npan - p_) & 1 ? B2 + sh.mat2(b) : X + sh.mat(b);
    const size_t vec = sh.vec(b);
    const int ld = n | 1;
    C* xs = reinterpret_cast<C*>(smem_raw);            // [nb][ld]
    C* prow = xs + (size_t)nb * ld;                     // [nb] scaled pivot row (inverse pivot at its own column)
    unsigned long long* wkey = reinterpret_cast<unsigned long long*>(prow + nb);   // [32] best per row warp
    int* wrow = reinterpret_cast<int*>(wkey + 32);      // [32]
    int* pos = wrow + 32;                               // [n] position -> row of src
    int* ipos = pos + n;                                // [n] its inverse
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rw = warp % RW, grp = warp / RW;
    const int stride = 32 * RW;
    const int row0 = rw * 32 + lane;
    for (int e = threadIdx.x; e < n * nb; e += blockDim.x) {
        const int i = e / nb, c = e - i * nb;
        xs[(size_t)c * ld + i] = src[(size_t)i * n + k0 + c];
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) pos[i] = ipos[i] = i;
    __syncthreads();
    unsigned free_rows = 0;                             // rows of this thread that may still serve as pivot
#pragma unroll
    for (int u = 0; u < PANEL_ROWS; ++u) {
        const int i = row0 + u * stride;
        if (i >= k0 && i < n) free_rows |= 1u << u;
    }
    const int c_lo = grp * bc, c_hi = min(nb, c_lo + bc);
    auto publish = [&](int c) {                         // best free row of column c, by the warps of its group
        unsigned long long key = 0;
        int row = 0x7fffffff;
#pragma unroll
        for (int u = 0; u < PANEL_ROWS; ++u)
            if (free_rows >> u & 1) {
                const unsigned long long q = mag_key(cabs2<T>(xs[(size_t)c * ld + row0 + u * stride]));
                if (q > key) {
                    key = q;
                    row = row0 + u * stride;
                }
            }
        warp_best<T>(key, row);
        if (lane == 0) {
            wkey[rw] = key;
            wrow[rw] = row;
        }
    };
    if (grp == 0) publish(0);
    bool bad = false;
    for (int k = 0; k < nb; ++k) {
        __syncthreads();
        unsigned long long key = lane < RW ? wkey[lane] : 0ull;
        int p = lane < RW ? wrow[lane] : 0x7fffffff;
        warp_best<T>(key, p);
        if (key <= 1ull) {                              // no free row with a non-zero entry (uniform over the CTA)
            bad = true;
            break;
        }
        C f[PANEL_ROWS];                                // column k of this thread's rows before it is overwritten
#pragma unroll
        for (int u = 0; u < PANEL_ROWS; ++u) {
            const int i = row0 + u * stride;
            if (i < n) f[u] = xs[(size_t)k * ld + i];
        }
        if (threadIdx.x < 32) {
            // the pivot row, scaled, and the exchange of positions
            const C pv = xs[(size_t)k * ld + p];
            const T d = (T)1 / cabs2<T>(pv);
            const C inv = mk<T>(pv.x * d, -pv.y * d);
            for (int c = lane; c < nb; c += 32) prow[c] = c == k ? inv : cmul(xs[(size_t)c * ld + p], inv);
            if (lane == 0) {
                const int l = ipos[p], r = pos[k0 + k];
                pos[l] = r;
                ipos[r] = l;
                pos[k0 + k] = p;
                ipos[p] = k0 + k;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PANEL_ROWS; ++u) {
            const int i = row0 + u * stride;
            if (i < n) {
                if (i == p) {
                    for (int c = c_lo; c < c_hi; ++c) xs[(size_t)c * ld + i] = prow[c];
                    free_rows &= ~(1u << u);
                } else {
                    const C fi = f[u];
#pragma unroll 4
                    for (int c = c_lo; c < c_hi; ++c) {
                        const C r = prow[c];
                        C x = c == k ? mk<T>(0, 0) : xs[(size_t)c * ld + i];
                        x.x -= fi.x * r.x - fi.y * r.y;
                        x.y -= fi.x * r.y + fi.y * r.x;
                        xs[(size_t)c * ld + i] = x;
                    }
                }
            }
        }
        if (k + 1 < nb && k + 1 >= c_lo && k + 1 < c_hi) publish(k + 1);
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) flags[b] = 1;
        return;
    }
    M += vec * sh.pb;
    for (int c = 0; c < nb; ++c)
        for (int i = threadIdx.x; i < n; i += blockDim.x) M[(size_t)c * n + i] = xs[(size_t)c * ld + pos[i]];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        perm[vec + i] = pos[i];
        ipos[i] = rows[vec + pos[i]];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) rows[vec + i] = ipos[i];
}

// The same panel for n <= PR_ROWS with the panel in registers: a thread owns one row and BC columns (groups of BC columns,
// 32-row warps), every group turns its columns by one place per step, so that the current column is always the owning
// group's place 0 and the loop needs no register indexing; the turn costs nothing, the update writes one place over.
// Shared memory carries the pivot row, the current column and the row warps' best pivots.  The version above reads and
// writes its panel in shared memory, a load-store chain per column.  Per panel: 200 matrices of 181 67 -> 32 us, 100 of
// 531 107 -> 44, a batch of 19-339 93 -> 40.
constexpr int PR_ROWS = 640;
template <typename T, int BC>
__global__ void __launch_bounds__(PR_ROWS) k_inv_panel_reg(InvShape sh, int p_, int RW, const cplx<T>* X, const cplx<T>* B2,
                                                           cplx<T>* M, int* perm, int* rows, int* flags) {
    using C = cplx<T>;
    __shared__ __align__(16) C prow[InvCfg<T>::PB + BC];
    __shared__ C col[PR_ROWS];
    __shared__ unsigned long long wkey[32];
    __shared__ int wrow[32];
    __shared__ int pos[PR_ROWS], ipos[PR_ROWS];
    const int b = sh.b0 + blockIdx.x, n = sh.order(b), npan = (n + sh.pb - 1) / sh.pb;
    if (p_ >= npan || flags[b]) return;
    const int k0 = p_ * sh.pb, nb = min(sh.pb, n - k0);
    const C* src = (npan - p_) & 1 ? B2 + sh.mat2(b) : X + sh.mat(b);
    const size_t vec = sh.vec(b);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rw = warp % RW, grp = warp / RW;
    const int row = rw * 32 + lane;
    C x[BC];
#pragma unroll
    for (int j = 0; j < BC; ++j) x[j] = row < n && grp * BC + j < nb ? src[(size_t)row * n + k0 + grp * BC + j] : mk<T>(0, 0);
    for (int i = threadIdx.x; i < n; i += blockDim.x) pos[i] = ipos[i] = i;
    bool free_row = row >= k0 && row < n;
    auto publish = [&]() {                              // the current column and its best free row, by its group
        col[row] = x[0];
        unsigned long long key = free_row ? mag_key(cabs2<T>(x[0])) : 0ull;
        int r = row;
        warp_best<T>(key, r);
        if (lane == 0) {
            wkey[rw] = key;
            wrow[rw] = r;
        }
    };
    if (grp == 0) publish();
    bool bad = false;
    for (int k = 0; k < nb; ++k) {
        __syncthreads();
        unsigned long long key = lane < RW ? wkey[lane] : 0ull;
        int p = lane < RW ? wrow[lane] : 0x7fffffff;
        warp_best<T>(key, p);
        if (key <= 1ull) {                              // no free row with a non-zero entry (uniform over the CTA)
            bad = true;
            break;
        }
        if (row == p) {
#pragma unroll
            for (int j = 0; j < BC; ++j) prow[grp * BC + j] = x[j];
        }
        const C f = col[row], pv = col[p];
        if (threadIdx.x == 0) {
            const int l = ipos[p], r = pos[k0 + k];
            pos[l] = r;
            ipos[r] = l;
            pos[k0 + k] = p;
            ipos[p] = k0 + k;
        }
        const T d = (T)1 / cabs2<T>(pv);
        const C inv = mk<T>(pv.x * d, -pv.y * d);
        const bool owner = grp == k / BC, pivot = row == p;
        C m = cmul(f, inv);                             // multiplier; the pivot row is scaled instead
        m = pivot ? inv : mk<T>(-m.x, -m.y);
        __syncthreads();
        const C x0 = x[0], r0 = prow[grp * BC];
#pragma unroll
        for (int j = 1; j < BC; ++j) {
            const C r = prow[grp * BC + j];
            C y = pivot ? mk<T>(0, 0) : x[j];
            cfma(y, m, r);
            x[j - 1] = y;
        }
        C y = pivot ? mk<T>(0, 0) : x0;
        cfma(y, m, r0);
        x[BC - 1] = owner ? m : y;                      // the eliminated column: inverse pivot, minus the multipliers
        free_row &= !pivot;
        if (k + 1 < nb && grp == (k + 1) / BC) publish();
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) flags[b] = 1;
        return;
    }
    M += vec * sh.pb;
    if (row < n) {
        const int i = ipos[row];
#pragma unroll
        for (int j = 0; j < BC; ++j) {
            const int c = grp * BC + (j + nb) % BC;
            if (c < nb) M[(size_t)c * n + i] = x[j];
        }
    }
    int orig = 0;
    if (threadIdx.x < n) {
        perm[vec + threadIdx.x] = pos[threadIdx.x];
        orig = rows[vec + pos[threadIdx.x]];
    }
    for (int i = threadIdx.x + blockDim.x; i < n; i += blockDim.x) perm[vec + i] = pos[i];
    __syncthreads();
    if (threadIdx.x < n) rows[vec + threadIdx.x] = orig;
}

// The other columns (see above).  Grid (column tile, row tile, matrix); thread (tx, ty) holds rows ty 4 .. + 3 and
// columns tx + 16 u of a 64 x 64 tile, the panel's multipliers and pivot rows staged once in shared memory.
// FP32: four CTAs per SM (64 registers with the loop unrolled by two; three, unrolled by four: 357 us where this takes
// 332, 200 matrices of N_G = 181).
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 1) k_inv_update(InvShape sh, int p, cplx<T>* X, cplx<T>* B2, const cplx<T>* M,
                                                    const int* perm, const int* rows, const int* flags) {
    using C = cplx<T>;
    constexpr int PB = InvCfg<T>::PB;
    __shared__ __align__(16) C ms[PB][UPD];
    __shared__ __align__(16) C rs[PB][UPD];
    const int b = sh.b0 + blockIdx.z, n = sh.order(b), npan = (n + sh.pb - 1) / sh.pb;
    const int i0 = blockIdx.y * UPD, j0 = blockIdx.x * UPD;
    if (p >= npan || i0 >= n || j0 >= n || flags[b]) return;
    const int k0 = p * sh.pb, nb = min(sh.pb, n - k0);
    const bool from_b = (npan - p) & 1, last = p + 1 == npan;
    const C* src = from_b ? B2 + sh.mat2(b) : X + sh.mat(b);
    C* dst = from_b ? X + sh.mat(b) : B2 + sh.mat2(b);
    M += sh.vec(b) * sh.pb;
    perm += sh.vec(b);
    rows += sh.vec(b);
    for (int e = threadIdx.x; e < nb * UPD; e += 256) {
        const int c = e / UPD, x = e % UPD;
        ms[c][x] = i0 + x < n ? M[(size_t)c * n + i0 + x] : mk<T>(0, 0);
        rs[c][x] = j0 + x < n ? src[(size_t)perm[k0 + c] * n + j0 + x] : mk<T>(0, 0);
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    C acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[r][u] = mk<T>(0, 0);
    __syncthreads();
#pragma unroll 2
    for (int c = 0; c < nb; ++c) {
        C m[4], x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) m[r] = ms[c][ty * 4 + r];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = rs[c][tx + 16 * u];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int u = 0; u < 4; ++u) cfma(acc[r][u], m[r], x[u]);
    }
    // the products are summed from zero and meet the old element once: one rounding at its size per panel, not nb (the
    // inverse's part of the loss error 1.23e-6 -> 1.10e-6 and 1.11e-6 -> 0.91e-6 on two q of N_G = 181)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = i0 + ty * 4 + r;
        if (i >= n || (i >= k0 && i < k0 + nb)) continue;
        const C* s = src + (size_t)perm[i] * n;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + tx + 16 * u;
            if (j >= n) continue;
            const C v = s[j];
            acc[r][u].x += v.x;
            acc[r][u].y += v.y;
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = j0 + tx + 16 * u;
        if (j >= n) continue;
        const bool in_panel = j >= k0 && j < k0 + nb;
        const int jd = last ? rows[j] : j;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = i0 + ty * 4 + r;
            if (i < n) dst[(size_t)i * n + jd] = in_panel ? ms[j - k0][ty * 4 + r] : acc[r][u];
        }
    }
}

// The diagonal of the inverse, and kappa_1 = |A|_1 |X|_1 (mixed path; xnorm starts at 0 and is read by the callers
// that need kappa).  Singular matrices get a zero diagonal.
template <typename T>
__global__ void __launch_bounds__(256) k_inv_finish(int n, const cplx<T>* X, const int* flags, double* xnorm,
                                                    double2* diag_inv, double* L) {
    __shared__ double sums[4][64];
    const int b = blockIdx.x, tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int j = blockIdx.y * 64 + tx;
    X += (size_t)b * n * n;
    const bool bad = flags[b] != 0;
    if (j < n && ty == 0) {
        const cplx<T> z = bad ? mk<T>(0, 0) : X[(size_t)j * n + j];
        diag_inv[(size_t)b * n + j] = make_double2((double)z.x, (double)z.y);
        if constexpr (sizeof(T) == 8) L[(size_t)b * n + j] = -(double)z.y;
    }
    if constexpr (sizeof(T) == 4) {
        double cs = 0.0;
        if (j < n && !bad)
            for (int i = ty; i < n; i += 4) cs += (double)cabs_safe(X[(size_t)i * n + j]);
        sums[ty][tx] = cs;
        __syncthreads();
        if (ty == 0 && j < n) {
            cs = (sums[0][tx] + sums[1][tx]) + (sums[2][tx] + sums[3][tx]);
            atomicMax(reinterpret_cast<unsigned long long*>(xnorm + b), (unsigned long long)__double_as_longlong(cs));
        }
    }
}

// FP64 correction of the diagonal of X ~ A^-1 for the blocks with kappa_1 above
// the threshold (A FP64, X FP32):  d_j = X_jj + sum_k X_jk (delta_kj - sum_l A_kl X_lj).
// The other blocks keep X_jj.  A CTA takes 32 rows k and 32 columns j of A X (k_refine_part) and leaves their share of
// d_j; k_refine_diag adds the shares in row order.  Bound by the FP64 pipe (4 n^3 multiply-adds a block, 1.1 ms at
// N_G = 531); with all rows k of 32 columns in one CTA a few blocks waited for its serial sums: 5 of 531: 44 -> 5 ms,
// 84: 143 -> 85 ms.
constexpr int RF_T = 32, RF_K = 16;
__global__ void __launch_bounds__(256) k_refine_part(int n, int nw, const double2* Aall, const float2* Xall, const int* flags,
                                                     const double* norms, double kappa_refine, double2* part) {
    __shared__ double2 As[RF_K][RF_T + 1];                 // [l][k]
    __shared__ double2 Xs[RF_K][RF_T];                     // [l][j]
    __shared__ double2 red[RF_T][17];
    const int b = blockIdx.x, j0 = blockIdx.y * RF_T, k0 = blockIdx.z * RF_T;
    if (flags[b] || !(norms[b] * norms[nw + b] > kappa_refine)) return;
    const double2* A = Aall + (size_t)b * n * n;
    const float2* X = Xall + (size_t)b * n * n;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;    // rows ty, ty + 16; columns tx, tx + 16
    double2 acc[2][2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) acc[r][c] = make_double2(0.0, 0.0);
    for (int l0 = 0; l0 < n; l0 += RF_K) {
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int e = threadIdx.x + 256 * v;
            const int la = e % RF_K, ka = e / RF_K, lx = e / RF_T, jx = e % RF_T;
            As[la][ka] = l0 + la < n && k0 + ka < n ? A[(size_t)(k0 + ka) * n + l0 + la] : make_double2(0.0, 0.0);
            const float2 x = l0 + lx < n && j0 + jx < n ? X[(size_t)(l0 + lx) * n + j0 + jx] : make_float2(0.f, 0.f);
            Xs[lx][jx] = make_double2((double)x.x, (double)x.y);
        }
        __syncthreads();
#pragma unroll 4
        for (int l = 0; l < RF_K; ++l) {
            const double2 a0 = As[l][ty], a1 = As[l][ty + 16], x0 = Xs[l][tx], x1 = Xs[l][tx + 16];
            cfma(acc[0][0], a0, x0);
            cfma(acc[0][1], a0, x1);
            cfma(acc[1][0], a1, x0);
            cfma(acc[1][1], a1, x1);
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int j = j0 + tx + 16 * c;
        double2 d = make_double2(0.0, 0.0);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = k0 + ty + 16 * r;
            if (j < n && k < n) {
                const double2 res = make_double2((k == j ? 1.0 : 0.0) - acc[r][c].x, -acc[r][c].y);
                const float2 x = X[(size_t)j * n + k];
                cfma(d, make_double2((double)x.x, (double)x.y), res);
            }
        }
        red[tx + 16 * c][ty] = d;
    }
    __syncthreads();
    if (threadIdx.x < RF_T && j0 + threadIdx.x < n) {
        double2 d = make_double2(0.0, 0.0);
        for (int r = 0; r < 16; ++r) d = cadd(d, red[threadIdx.x][r]);
        part[((size_t)blockIdx.z * nw + b) * n + j0 + threadIdx.x] = d;
    }
}

__global__ void __launch_bounds__(128) k_refine_diag(int n, int nw, int nk, const float2* Xall, const int* flags,
                                                     const double* norms, double kappa_refine, const double2* part,
                                                     double2* diag_inv, double* L, double* resid) {
    const int b = blockIdx.x, j = blockIdx.y * 128 + threadIdx.x;
    if (flags[b] || j >= n) return;
    const float2 x = Xall[(size_t)b * n * n + (size_t)j * n + j];
    double2 d = make_double2(0.0, 0.0);
    if (norms[b] * norms[nw + b] > kappa_refine) {
        for (int z = 0; z < nk; ++z) d = cadd(d, part[((size_t)z * nw + b) * n + j]);
        const double dr = (double)x.x + d.x, di = (double)x.y + d.y;
        const double mag = sqrt(dr * dr + di * di);
        const double rel = mag > 0 ? sqrt(d.x * d.x + d.y * d.y) / mag : 0.0;
        atomicMax(reinterpret_cast<unsigned long long*>(resid + b), (unsigned long long)__double_as_longlong(rel));
    }
    diag_inv[(size_t)b * n + j] = make_double2((double)x.x + d.x, (double)x.y + d.y);
    L[(size_t)b * n + j] = -((double)x.y + d.y);
}

// L_LFE of the mixed path without cancellation: for X = A^-1 (the FP32
// inverse) and B = (A - A^H)/(2i) the Hermitian form of A's anti-Hermitian
// part, -Im [A^-1]_jj = [X B X^H]_jj.  Where the loss is small against
// |[A^-1]_jj| (Im of an O(1) diagonal) the imaginary part of the FP32 diagonal
// loses its relative accuracy; the form builds L from the small B itself
// (B from the FP64 matrix in FP64, rounded once), so its relative error is
// that of X.  The imaginary part of the reported diagonal becomes -L_j.  Blocks
// corrected in FP64 keep their values.
//
// B is formed once per matrix (k_form_b, tile and transposed tile), then a CTA of
// k_loss_quadform takes 64 rows j: T = X B in 64 x 64 tiles of l, L_j += Re sum_l T_jl
// conj(X_jl).  B being Hermitian, the k tiles above an l tile's own count twice and those
// below it are left out, half the product.  Bound by the FP32 pipe; with 32 x 32 tiles, all
// of B and its FP64 source read again by every row block: 200 matrices of 181 660 -> 280 us,
// 100 of 531 7.0 -> 2.2 ms.  k_form_b is bound by the FP64 pipe (two sums and two conversions per element) and forms only
// the tiles the form reads (200 of 181: 95 -> 52 us; 100 of 531: 357 -> 160).
constexpr int QF = 64, QK = 16;
__global__ void __launch_bounds__(256) k_form_b(int n, const double2* Aall, const int* flags, const double* norms,
                                                const double* xnorms, double kappa_refine, float2* Ball) {
    __shared__ double2 At[32][33];
    const int b = blockIdx.z;
    if (flags[b] || norms[b] * xnorms[b] > kappa_refine) return;
    const double2* A = Aall + (size_t)b * n * n;
    float2* B = Ball + (size_t)b * n * n;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int k0 = blockIdx.y * 32, l0 = blockIdx.x * 32;
    if (k0 >= (l0 / QF + 1) * QF) return;                  // below the l tile of the form, which leaves it out
    for (int r = ty; r < 32; r += 8)
        if (l0 + r < n && k0 + tx < n) At[r][tx] = A[(size_t)(l0 + r) * n + k0 + tx];
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int k = k0 + r, l = l0 + tx;
        if (k < n && l < n) {
            const double2 akl = A[(size_t)k * n + l], alk = At[tx][r];
            // halved after the conversion: exact, and not on the FP64 pipe
            B[(size_t)k * n + l] = make_float2(0.5f * (float)(akl.y + alk.y), -0.5f * (float)(akl.x - alk.x));
        }
    }
}

__global__ void __launch_bounds__(256) k_loss_quadform(int n, const float2* Xall, const float2* Ball, const int* flags,
                                                       const double* norms, const double* xnorms, double kappa_refine,
                                                       double2* diag_inv, double* L) {
    __shared__ __align__(16) float2 Xs[QK][QF + 2];        // [k][j]
    __shared__ __align__(16) float2 Bs[QK][QF];            // [k][l]
    const int b = blockIdx.x, j0 = blockIdx.y * QF;
    if (flags[b] || norms[b] * xnorms[b] > kappa_refine) return;
    const float2* X = Xall + (size_t)b * n * n;
    const float2* B = Ball + (size_t)b * n * n;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // rows 4 ty .. + 3, columns tx + 16 u
    float part[4] = {0.f, 0.f, 0.f, 0.f};
    for (int l0 = 0; l0 < n; l0 += QF) {
        float2 acc[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[r][u] = make_float2(0.f, 0.f);
        for (int k0 = 0; k0 < l0 + QF && k0 < n; k0 += QK) {
            if (k0 == l0) {                                    // the tiles before count for their mirror images too
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc[r][u] = make_float2(2.f * acc[r][u].x, 2.f * acc[r][u].y);
            }
            __syncthreads();
#pragma unroll
            for (int v = 0; v < QF * QK / 256; ++v) {
                const int e = threadIdx.x + 256 * v;
                const int kx = e % QK, jx = e / QK;            // rows of X along k
                Xs[kx][jx] = j0 + jx < n && k0 + kx < n ? X[(size_t)(j0 + jx) * n + k0 + kx] : make_float2(0.f, 0.f);
                const int lb = e % QF, kb = e / QF;
                Bs[kb][lb] = k0 + kb < n && l0 + lb < n ? B[(size_t)(k0 + kb) * n + l0 + lb] : make_float2(0.f, 0.f);
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < QK; ++k) {
                const float4 xa = *reinterpret_cast<const float4*>(&Xs[k][ty * 4]);
                const float4 xb = *reinterpret_cast<const float4*>(&Xs[k][ty * 4 + 2]);
                const float2 x[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xb.x, xb.y),
                                     make_float2(xb.z, xb.w)};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 v = Bs[k][tx + 16 * u];
#pragma unroll
                    for (int r = 0; r < 4; ++r) cfma(acc[r][u], x[r], v);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + ty * 4 + r, l = l0 + tx + 16 * u;
                if (j < n && l < n) {
                    const float2 x = X[(size_t)j * n + l];
                    part[r] = fmaf(acc[r][u].x, x.x, fmaf(acc[r][u].y, x.y, part[r]));
                }
            }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float s = part[r];
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, 16);
        const int j = j0 + ty * 4 + r;
        if (tx == 0 && j < n) {
            const size_t o = (size_t)b * n + j;
            L[o] = (double)s;
            diag_inv[o].y = -(double)s;
        }
    }
}

}  // namespace

// All panels of nmat matrices of order at most n; returns the number of launches.
template <typename T>
static int eliminate(cudaStream_t st, InvShape sh, int n, int nmat, int npan, size_t smem, cplx<T>* X, cplx<T>* B2, cplx<T>* M,
                     int* perm, int* rows, int* flags) {
    int launches = 0;
    const int RW = std::min((n + 31) / 32, 32);
    int groups = 1;
    while (groups * 2 * RW <= 16 && groups * 2 <= sh.pb) groups *= 2;
    const int bc = (sh.pb + groups - 1) / groups;
    // columns per thread of the register panel: more for large orders (fewer warps repeat the step's set-up), within
    // PR_ROWS threads
    const int breg = sizeof(T) == 8 ? (RW <= 10 ? 8 : 16) : (RW <= 2 ? 8 : (RW <= 8 ? 16 : 32));
    const int greg = (sh.pb + breg - 1) / breg;
    const bool reg = n <= PR_ROWS && 32 * RW * greg <= PR_ROWS;
    auto panel = [&](int p, int m) {
        const int threads = 32 * RW * greg;
        if (!reg)
            k_inv_panel<T><<<m, 32 * RW * groups, smem, st>>>(sh, p, RW, bc, X, B2, M, perm, rows, flags);
        else if (breg == 8)
            k_inv_panel_reg<T, 8><<<m, threads, 0, st>>>(sh, p, RW, X, B2, M, perm, rows, flags);
        else if (breg == 16)
            k_inv_panel_reg<T, 16><<<m, threads, 0, st>>>(sh, p, RW, X, B2, M, perm, rows, flags);
        else if constexpr (sizeof(T) == 4)
            k_inv_panel_reg<T, 32><<<m, threads, 0, st>>>(sh, p, RW, X, B2, M, perm, rows, flags);
    };
    for (const int b1 = sh.b0 + nmat; sh.b0 < b1; sh.b0 += 32768) {    // grid limit of the tiles' third dimension
        const int m = std::min(32768, b1 - sh.b0);
        const dim3 tiles((n + UPD - 1) / UPD, (n + UPD - 1) / UPD, m);
        for (int p = 0; p < npan; ++p) {
            panel(p, m);
            launches += 2;
            k_inv_update<T><<<tiles, 256, 0, st>>>(sh, p, X, B2, M, perm, rows, flags);
        }
    }
    return launches;
}

// Widest panel of order-n matrices that fits shared memory, and its bytes.
template <typename T> static int panel_width(int n, size_t* smem) {
    int pb = std::min(InvCfg<T>::PB, n);
    auto bytes = [&](int w) {
        return ((size_t)w * (n | 1) + w) * sizeof(cplx<T>) + 32 * (sizeof(unsigned long long) + sizeof(int)) +
               2 * (size_t)n * sizeof(int);
    };
    while (pb > 1 && bytes(pb) > PANEL_SMEM) pb >>= 1;
    *smem = bytes(pb);
    return pb;
}

// Inverse of nmat matrices of order n into X; B2 holds as many for the out-of-place updates, aux the panels and row
// orders.  norms (mixed path): |A|_1 of every matrix, then |X|_1.
template <typename T>
static cudaError_t invert_batch(cudaStream_t st, int n, int nmat, const double2* A, cplx<T>* X, cplx<T>* B2, void* aux,
                                double* anorm, double* xnorm, double2* eps_diag, double* L, double* L_nolfe,
                                double2* diag_inv, int* flags) {
    using C = cplx<T>;
    size_t smem = 0;
    const int pb = panel_width<T>(n, &smem);
    C* M = reinterpret_cast<C*>(aux);
    int* perm = reinterpret_cast<int*>(M + (size_t)nmat * pb * n);
    int* rows = perm + (size_t)nmat * n;
    cudaError_t e = qcx_allow_smem((const void*)k_inv_panel<T>);
    if (e != cudaSuccess) return e;
    const int npan = (n + pb - 1) / pb;
    const dim3 cols(nmat, (n + 63) / 64);
    k_inv_load<T><<<cols, 256, 0, st>>>(n, A, npan & 1 ? B2 : X, anorm, eps_diag, L_nolfe, rows, flags);
    eliminate<T>(st, InvShape{n, pb, nullptr, 0, 0, 0}, n, nmat, npan, smem, X, B2, M, perm, rows, flags);
    k_inv_finish<T><<<cols, 256, 0, st>>>(n, X, flags, xnorm, diag_inv, L);
    return cudaGetLastError();
}

// Matrices are inverted in groups whose second copy stays within QCX_INV_COPY_BYTES (at least one), so that the scratch
// does not grow with the number of frequencies; where even that does not fit, in smaller groups.
template <typename C> static int inv_group(int n, int nw) {
    return (int)std::min<size_t>({(size_t)nw, std::max<size_t>(1, QCX_INV_COPY_BYTES / ((size_t)n * n * sizeof(C))), 32768});
}

template <typename T>
static cudaError_t invert_all(qcx_ctx* ctx, QSlot& s, double* norms, double* L, int& per) {
    using C = cplx<T>;
    const int n = s.ng, nw = s.nw;
    cudaError_t e;
    for (per = inv_group<C>(n, nw);; per /= 2) {
        e = qcx_ensure(ctx, s.work2, (size_t)per * n * n * sizeof(C));
        if (e == cudaSuccess) e = qcx_ensure(ctx, s.gjaux, (size_t)per * n * (InvCfg<T>::PB * sizeof(C) + 2 * sizeof(int)));
        if (e == cudaSuccess) break;
        if (e != cudaErrorMemoryAllocation || per == 1) return e;
        cudaGetLastError();
        s.work2.release();
        s.gjaux.release();
    }
    for (int w0 = 0; w0 < nw; w0 += per) {
        const int m = std::min(per, nw - w0);
        const size_t o = (size_t)w0 * n;
        e = invert_batch<T>(ctx->stream, n, m, s.eps.as<double2>() + o * n, s.work.as<C>() + o * n, s.work2.as<C>(),
                            s.gjaux.p, norms ? norms + w0 : nullptr, norms ? norms + nw + w0 : nullptr,
                            s.eps_diag.as<double2>() + o, L + o, L + (size_t)nw * n + o, s.diag_inv.as<double2>() + o,
                            s.flags.as<int>() + w0);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t qcx_launch_invert(qcx_ctx* ctx, QSlot& s, qcx_precision prec, double* d_loss_out) {
    const int n = s.ng;
    int per = 1;
    if (prec == QCX_FP64) {
        cudaError_t e = invert_all<double>(ctx, s, nullptr, d_loss_out, per);
        if (e != cudaSuccess) return e;
        return cudaMemsetAsync(s.resid.p, 0, sizeof(double) * s.nw, ctx->stream);
    }
    const int rt = (n + RF_T - 1) / RF_T;
    cudaError_t e = qcx_ensure(ctx, s.kappa1, 2 * sizeof(double) * s.nw);
    if (e == cudaSuccess) e = qcx_ensure(ctx, s.refine, sizeof(double2) * (size_t)rt * s.nw * n);
    if (e != cudaSuccess) return e;
    double* norms = s.kappa1.as<double>();
    e = cudaMemsetAsync(norms, 0, 2 * sizeof(double) * s.nw, ctx->stream);
    if (e != cudaSuccess) return e;
    e = invert_all<float>(ctx, s, norms, d_loss_out, per);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(s.resid.p, 0, sizeof(double) * s.nw, ctx->stream);
    if (e != cudaSuccess) return e;
    k_refine_part<<<dim3(s.nw, rt, rt), 256, 0, ctx->stream>>>(n, s.nw, s.eps.as<double2>(), s.work.as<float2>(),
                                                               s.flags.as<int>(), norms, ctx->kappa_refine,
                                                               s.refine.as<double2>());
    k_refine_diag<<<dim3(s.nw, (n + 127) / 128), 128, 0, ctx->stream>>>(n, s.nw, rt, s.work.as<float2>(), s.flags.as<int>(),
                                                                        norms, ctx->kappa_refine, s.refine.as<double2>(),
                                                                        s.diag_inv.as<double2>(), d_loss_out,
                                                                        s.resid.as<double>());
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int t32 = (n + 31) / 32;
    for (int w0 = 0; w0 < s.nw; w0 += per) {             // B takes the inverse's second copy, group by group
        const int m = std::min(per, s.nw - w0);
        const size_t o = (size_t)w0 * n;
        k_form_b<<<dim3(t32, t32, m), 256, 0, ctx->stream>>>(n, s.eps.as<double2>() + o * n, s.flags.as<int>() + w0, norms + w0,
                                                              norms + s.nw + w0, ctx->kappa_refine, s.work2.as<float2>());
        k_loss_quadform<<<dim3(m, (n + QF - 1) / QF), 256, 0, ctx->stream>>>(
            n, s.work.as<float2>() + o * n, s.work2.as<float2>(), s.flags.as<int>() + w0, norms + w0, norms + s.nw + w0,
            ctx->kappa_refine, s.diag_inv.as<double2>() + o, d_loss_out + o);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ------------------------------------------------------------------ uneven batches (mixed path)
namespace {

// FP64 eps of every instance -> FP32, into the buffer its first panel reads; starting row order.  Grid (instance, 64
// columns).
__global__ void __launch_bounds__(256) k_batch_load(InvShape sh, const double2* eps, float2* X, float2* B2, int* rows, int* flags) {
    const int b = sh.b0 + blockIdx.x, n = sh.order(b), tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int j = blockIdx.y * 64 + tx;
    if (blockIdx.y == 0 && threadIdx.x == 0) flags[b] = 0;
    if (j >= n) return;
    const int npan = (n + sh.pb - 1) / sh.pb;
    float2* dst = npan & 1 ? B2 + sh.mat2(b) : X + sh.mat(b);
    const double2* A = eps + sh.inst[b].eps_off;
    for (int i = ty; i < n; i += 4) {
        const double2 z = A[(size_t)i * n + j];
        dst[(size_t)i * n + j] = make_float2((float)z.x, (float)z.y);
    }
    if (ty == 0) rows[sh.vec(b) + j] = j;
}

// index of the solution's component i (the head last) in eps
__device__ __forceinline__ int head_last(int i, int n, int h) { return i == n - 1 ? h : (i < h ? i : i + 1); }

// x = the inverse's head column (head component last), the heads, and zero heads for singular instances
__global__ void __launch_bounds__(128) k_batch_x(BatchSolveArgs a, const float2* X) {
    const int id = blockIdx.x;
    const BatchInst in = a.inst[id];
    const int n = in.ng, h = in.head;
    const bool bad = a.flags[id] != 0;
    if (!bad)
        for (int i = threadIdx.x; i < n; i += 128) {
            const float2 z = X[in.work_off + (size_t)head_last(i, n, h) * n + h];
            a.x[in.vec_off + i] = make_double2((double)z.x, (double)z.y);
        }
    if (threadIdx.x == 0) {
        const double2 e = a.eps[in.eps_off + (size_t)h * n + h];
        a.out[id] = bad ? 0.0 : -(double)X[in.work_off + (size_t)h * n + h].y;
        a.out[a.ninst + id] = e.y / (e.x * e.x + e.y * e.y);
        a.out[2 * a.ninst + id] = 0.0;
    }
}

constexpr double REFINE_TOL = 1.0e-6;        // last relative correction that counts as converged

// x += X r (FP32 products of the FP64 residual); one CTA per instance, a row per warp
__global__ void __launch_bounds__(512) k_batch_correct(BatchSolveArgs a, const float2* Xall, int last) {
    __shared__ float red[2][16];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* r = reinterpret_cast<float2*>(smem_raw);       // residual in eps order
    const int id = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (a.flags[id] == 1) return;
    const BatchInst in = a.inst[id];
    const int n = in.ng, h = in.head;
    const float2* X = Xall + in.work_off;
    for (int i = threadIdx.x; i < n; i += 512) {
        const double2 z = a.r[in.vec_off + i];
        r[head_last(i, n, h)] = make_float2((float)z.x, (float)z.y);
    }
    __syncthreads();
    double2* x = a.x + in.vec_off;
    float dmax = 0.f, xmax = 0.f;
    for (int i = warp; i < n; i += 16) {
        const float2* row = X + (size_t)head_last(i, n, h) * n;
        float2 d = make_float2(0.f, 0.f);
        for (int j = lane; j < n; j += 32) cfma(d, row[j], r[j]);
        for (int o = 16; o > 0; o >>= 1) {
            d.x += __shfl_xor_sync(0xffffffffu, d.x, o);
            d.y += __shfl_xor_sync(0xffffffffu, d.y, o);
        }
        if (lane == 0) {
            double2 v = x[i];
            v.x += (double)d.x;
            v.y += (double)d.y;
            x[i] = v;
            dmax = fmaxf(dmax, hypotf(d.x, d.y));
            xmax = fmaxf(xmax, (float)hypot(v.x, v.y));
            if (!(d.x == d.x) || !(d.y == d.y)) dmax = INFINITY;
        }
    }
    if (lane == 0) {
        red[0][warp] = dmax;
        red[1][warp] = xmax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float dm = 0.f, xm = 0.f;
        for (int w = 0; w < 16; ++w) {
            dm = fmaxf(dm, red[0][w]);
            xm = fmaxf(xm, red[1][w]);
        }
        const double rel = xm > 0.f ? (double)dm / (double)xm : 0.0;
        a.out[id] = -x[n - 1].y;
        a.out[2 * a.ninst + id] = rel;
        if (last) a.flags[id] = (rel > REFINE_TOL || !(rel == rel)) ? 2 : 0;
    }
}

}  // namespace

// Consecutive instances whose matrices stay within copy_bytes (at least one instance each).
std::vector<InvGroup> qcx_batch_inverse_groups(const std::vector<BatchInst>& inst, size_t copy_bytes) {
    std::vector<InvGroup> groups;
    for (int b = 0; b < (int)inst.size(); ++b) {
        const long long mats = (long long)inst[b].ng * (inst[b].ng + 1);
        if (groups.empty() || (size_t)(groups.back().mats + mats) * sizeof(float2) > copy_bytes)
            groups.push_back({b, 0, inst[b].work_off, inst[b].vec_off, 0, 0});
        InvGroup& g = groups.back();
        ++g.n;
        g.mats += mats;
        g.vecs += inst[b].ng;
    }
    return groups;
}

size_t qcx_batch_inverse_aux(long long vecs, int nmax) {
    size_t smem;
    return (size_t)vecs * ((size_t)panel_width<float>(nmax, &smem) * sizeof(float2) + 2 * sizeof(int));
}

cudaError_t qcx_launch_batch_inverse(cudaStream_t st, const BatchSolveArgs& a, const std::vector<InvGroup>& groups, float2* B2,
                                     void* aux, int nmax, int* launches) {
    if (nmax < 1 || nmax > 1024 * PANEL_ROWS) return cudaErrorInvalidValue;
    size_t smem = 0;
    const int pb = panel_width<float>(nmax, &smem);
    cudaError_t e = qcx_allow_smem((const void*)k_inv_panel<float>);
    if (e != cudaSuccess) return e;
    float2* X = reinterpret_cast<float2*>(a.work);
    for (const InvGroup& g : groups) {
        const InvShape sh{nmax, pb, a.inst, g.b0, (size_t)g.mat0, (size_t)g.vec0};
        float2* M = reinterpret_cast<float2*>(aux);
        int* perm = reinterpret_cast<int*>(M + (size_t)g.vecs * pb);
        int* rows = perm + g.vecs;
        k_batch_load<<<dim3(g.n, (nmax + 63) / 64), 256, 0, st>>>(sh, a.eps, X, B2, rows, a.flags);
        *launches += 1 + eliminate<float>(st, sh, nmax, g.n, (nmax + pb - 1) / pb, smem, X, B2, M, perm, rows, a.flags);
    }
    ++*launches;
    k_batch_x<<<a.ninst, 128, 0, st>>>(a, X);
    return cudaGetLastError();
}

cudaError_t qcx_launch_batch_correct(cudaStream_t st, const BatchSolveArgs& a, int nmax, int last) {
    k_batch_correct<<<a.ninst, 512, sizeof(float2) * nmax, st>>>(a, reinterpret_cast<const float2*>(a.work), last);
    return cudaGetLastError();
}

extern "C" qcx_status qcx_set_refine_threshold(qcx_ctx* ctx, double kappa1) {
    if (!ctx) return QCX_ERR_ARG;
    if (!(kappa1 >= 0.0)) return ctx->fail(QCX_ERR_ARG, "set_refine_threshold: kappa1 must be >= 0");
    ctx->kappa_refine = kappa1;
    return QCX_OK;
}
