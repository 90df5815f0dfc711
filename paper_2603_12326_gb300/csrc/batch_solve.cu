// Heads of the inverse dielectric matrices of a batch of uneven (q, w)
// instances: L_LFE = -Im [eps^-1]_{00} (Eq. (eps_LFE)) and L_noLFE =
// -Im (1/eps_00) (Eq. (eps_noLFE)).
//
// FP64 path: only the head of eps^-1 is needed, so no inverse is formed.  With the head
// row and column moved last (A' = P^T eps P), [eps^-1]_{00} is the last
// component of the solution of A' x = e_last; LU elimination with partial
// pivoting of the augmented matrix [A' | e_last] leaves that component as
// y_last / u_last,last, with no back substitution (k_lu_head: one CTA per instance
// at a time, instance lists per CTA built on the host, largest first, so the batch is one
// persistent launch; right-looking blocked LU on a work copy in global memory: rows are
// never moved, a row map in shared memory records the pivot order; per panel of PB columns
// the panel is factored in shared memory and the trailing columns, right-hand side included,
// are processed CW at a time).
//
// Mixed path: the blocked FP32 inverse of the per-q path over all instances (invert.cu); its
// head column is x, refined with the FP64 residual r = e_last - A' x (k_resid: 32 rows per CTA,
// all instances at once, so the FP64 work is spread over the whole GPU) and d = X r.  A CTA per
// instance left the largest instance's elimination on one SM as the critical path.
#include "qcx_internal.h"
#include "cplx.cuh"

namespace {

constexpr int LU_THREADS = 256;
constexpr int NWARP = LU_THREADS / 32;
constexpr int CW = 64;                       // trailing columns per chunk
constexpr int RG = LU_THREADS / CW;          // row groups of the trailing update
constexpr int PB = 16;                       // panel columns

// logical index -> index in eps with the head moved last
__device__ __forceinline__ int head_last(int i, int n, int h) { return i == n - 1 ? h : (i < h ? i : i + 1); }

template <typename C> __device__ __forceinline__ C czero() {
    C z;
    z.x = 0;
    z.y = 0;
    return z;
}
template <typename C> __device__ __forceinline__ C cinv(C a) {
    const auto d = 1 / (a.x * a.x + a.y * a.y);
    C z;
    z.x = a.x * d;
    z.y = -a.y * d;
    return z;
}
// acc -= a * b
template <typename C> __device__ __forceinline__ void cfms(C& acc, C a, C b) {
    acc.x = fma(-a.x, b.x, acc.x);
    acc.x = fma(a.y, b.y, acc.x);
    acc.y = fma(-a.x, b.y, acc.y);
    acc.y = fma(-a.y, b.x, acc.y);
}
template <typename T> __device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(LU_THREADS) k_lu_head(BatchSolveArgs a, int nmax) {
    using T = double;
    using C = double2;
    extern __shared__ __align__(16) unsigned char sm[];
    C* P = reinterpret_cast<C*>(sm);                  // [nmax][PB] panel, logical row order
    C* Li = P + (size_t)nmax * PB;                    // [PB][PB] L11^-1 (then U blocks)
    C* As = Li + PB * PB;                             // [PB][CW] A12 chunk
    C* Ub = As + PB * CW;                             // [PB][CW] U12 chunk
    int* rmap = reinterpret_cast<int*>(Ub + PB * CW); // [nmax]
    __shared__ T red_v[NWARP];
    __shared__ int red_i[NWARP];
    __shared__ int s_p, s_bad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    for (int ii = a.cta_off[blockIdx.x]; ii < a.cta_off[blockIdx.x + 1]; ++ii) {
        const int id = a.cta_ids[ii];
        const BatchInst in = a.inst[id];
        const int n = in.ng, h = in.head, ld = n + 1;
        const double2* A = a.eps + in.eps_off;
        C* M = reinterpret_cast<C*>(a.work) + in.work_off;
        for (long long e = threadIdx.x; e < (long long)n * ld; e += LU_THREADS) {
            const int i = (int)(e / ld), j = (int)(e - (long long)i * ld);
            C v;
            if (j == n) {
                v.x = (i == n - 1) ? T(1) : T(0);
                v.y = 0;
            } else {
                const double2 z = A[(size_t)head_last(i, n, h) * n + head_last(j, n, h)];
                v.x = (T)z.x;
                v.y = (T)z.y;
            }
            M[e] = v;
        }
        for (int i = threadIdx.x; i < n; i += LU_THREADS) rmap[i] = i;
        if (threadIdx.x == 0) s_bad = 0;
        __syncthreads();

        for (int k0 = 0; k0 < n; k0 += PB) {
            const int kb = min(PB, n - k0), R = n - k0;
            for (int e = threadIdx.x; e < R * PB; e += LU_THREADS) {
                const int r = e / PB, c = e - r * PB;
                P[e] = c < kb ? M[(size_t)rmap[k0 + r] * ld + k0 + c] : czero<C>();
            }
            __syncthreads();
            for (int kk = 0; kk < kb; ++kk) {
                // pivot: largest |P_r,kk| over r >= kk (smallest r on ties)
                T best = -1;
                int bi = R;
                for (int r = kk + threadIdx.x; r < R; r += LU_THREADS) {
                    const C z = P[r * PB + kk];
                    const T v = z.x * z.x + z.y * z.y;
                    if (v > best) {
                        best = v;
                        bi = r;
                    }
                }
                for (int o = 16; o > 0; o >>= 1) {
                    const T ov = __shfl_down_sync(0xffffffffu, best, o);
                    const int oi = __shfl_down_sync(0xffffffffu, bi, o);
                    if (ov > best || (ov == best && oi < bi)) {
                        best = ov;
                        bi = oi;
                    }
                }
                if (lane == 0) {
                    red_v[warp] = best;
                    red_i[warp] = bi;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    T bv = red_v[0];
                    int bix = red_i[0];
                    for (int w = 1; w < NWARP; ++w)
                        if (red_v[w] > bv || (red_v[w] == bv && red_i[w] < bix)) {
                            bv = red_v[w];
                            bix = red_i[w];
                        }
                    if (!(bv > 0) || bix >= R) {
                        s_bad = 1;
                        bix = kk;
                    }
                    s_p = bix;
                    if (bix != kk) {
                        const int t = rmap[k0 + kk];
                        rmap[k0 + kk] = rmap[k0 + bix];
                        rmap[k0 + bix] = t;
                    }
                }
                __syncthreads();
                if (s_bad) break;
                const int p = s_p;
                if (p != kk && threadIdx.x < PB) {
                    const C t = P[kk * PB + threadIdx.x];
                    P[kk * PB + threadIdx.x] = P[p * PB + threadIdx.x];
                    P[p * PB + threadIdx.x] = t;
                }
                __syncthreads();
                const C inv = cinv(P[kk * PB + kk]);
                for (int r = kk + 1 + threadIdx.x; r < R; r += LU_THREADS) {
                    const C l = cmul(P[r * PB + kk], inv);
                    P[r * PB + kk] = l;
                    for (int c = kk + 1; c < kb; ++c) cfms(P[r * PB + c], l, P[kk * PB + c]);
                }
                __syncthreads();
            }
            if (s_bad) break;
            for (int e = threadIdx.x; e < R * kb; e += LU_THREADS) {
                const int r = e / kb, c = e - r * kb;
                M[(size_t)rmap[k0 + r] * ld + k0 + c] = P[r * PB + c];
            }
            if (threadIdx.x < kb) {
                // column c of L11^-1 by forward substitution (unit diagonal)
                const int c = threadIdx.x;
                for (int i = 0; i < kb; ++i) {
                    C y = czero<C>();
                    if (i == c) y.x = 1;
                    else if (i > c)
                        for (int l = c; l < i; ++l) cfms(y, P[i * PB + l], Li[l * PB + c]);
                    Li[i * PB + c] = y;
                }
            }
            __syncthreads();
            for (int c0 = k0 + kb; c0 <= n; c0 += CW) {
                const int cw = min(CW, n + 1 - c0);
                for (int e = threadIdx.x; e < kb * CW; e += LU_THREADS) {
                    const int i = e / CW, c = e - i * CW;
                    As[e] = c < cw ? M[(size_t)rmap[k0 + i] * ld + c0 + c] : czero<C>();
                }
                __syncthreads();
                for (int e = threadIdx.x; e < kb * CW; e += LU_THREADS) {
                    const int i = e / CW, c = e - i * CW;
                    C s = czero<C>();
                    for (int l = 0; l <= i; ++l) cfma(s, Li[i * PB + l], As[l * CW + c]);
                    Ub[e] = s;
                    if (c < cw) M[(size_t)rmap[k0 + i] * ld + c0 + c] = s;
                }
                __syncthreads();
                const int c = threadIdx.x % CW, rg = threadIdx.x / CW;
                if (c < cw) {
                    C u[PB];
#pragma unroll
                    for (int l = 0; l < PB; ++l) u[l] = l < kb ? Ub[l * CW + c] : czero<C>();
                    for (int r = kb + rg; r < R; r += 4 * RG) {
                        C* dst[4];
                        C acc[4];
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int rr = r + v * RG;
                            dst[v] = rr < R ? M + (size_t)rmap[k0 + rr] * ld + c0 + c : nullptr;
                            acc[v] = dst[v] ? *dst[v] : czero<C>();
                        }
#pragma unroll
                        for (int l = 0; l < PB; ++l)
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                const int rr = min(r + v * RG, R - 1);
                                cfms(acc[v], P[rr * PB + l], u[l]);
                            }
#pragma unroll
                        for (int v = 0; v < 4; ++v)
                            if (dst[v]) *dst[v] = acc[v];
                    }
                }
                __syncthreads();
            }
        }
        const double2 ehh = A[(size_t)h * n + h];
        const double Lno = ehh.y / (ehh.x * ehh.x + ehh.y * ehh.y);
        if (s_bad) {
            if (threadIdx.x == 0) {
                a.flags[id] = 1;
                a.out[id] = 0.0;
                a.out[a.ninst + id] = Lno;
                a.out[2 * a.ninst + id] = 0.0;
            }
            __syncthreads();
            continue;
        }
        if (threadIdx.x == 0) {
            const C* rowp = M + (size_t)rmap[n - 1] * ld;
            const C xl = cmul(rowp[n], cinv(rowp[n - 1]));
            a.flags[id] = 0;
            a.out[id] = -(double)xl.y;
            a.out[a.ninst + id] = Lno;
            a.out[2 * a.ninst + id] = 0.0;
        }
        __syncthreads();
    }
}

// r = e_last - A' x in FP64; task = {instance, first of 32 rows}, 4 rows per warp
__global__ void __launch_bounds__(256) k_resid(BatchSolveArgs a, const int2* tasks) {
    const int2 tk = tasks[blockIdx.x];
    const BatchInst in = a.inst[tk.x];
    const int n = in.ng, h = in.head;
    const double2* A = a.eps + in.eps_off;
    const double2* x = a.x + in.vec_off;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (a.flags[tk.x] == 1) return;
    for (int v = 0; v < 4; ++v) {
        const int i = tk.y + warp * 4 + v;
        if (i >= n) break;
        const double2* row = A + (size_t)head_last(i, n, h) * n;
        double sx = 0.0, sy = 0.0;
        for (int j = lane; j < n; j += 32) {
            const double2 av = row[head_last(j, n, h)], xv = x[j];
            sx = fma(av.x, xv.x, fma(-av.y, xv.y, sx));
            sy = fma(av.x, xv.y, fma(av.y, xv.x, sy));
        }
        sx = warp_sum(sx);
        sy = warp_sum(sy);
        if (lane == 0) a.r[in.vec_off + i] = make_double2((i == n - 1 ? 1.0 : 0.0) - sx, -sy);
    }
}

size_t lu_smem(int nmax) {
    return ((size_t)nmax * PB + PB * PB + 2 * PB * CW) * sizeof(double2) + nmax * sizeof(int);
}

}  // namespace

cudaError_t qcx_launch_lu_head(cudaStream_t st, const BatchSolveArgs& a, int grid, int nmax) {
    if (grid < 1 || nmax < 1) return cudaErrorInvalidValue;
    const size_t smem = lu_smem(nmax);
    const cudaError_t e = qcx_allow_smem((const void*)k_lu_head, 1024);
    if (e != cudaSuccess) return e;
    k_lu_head<<<grid, LU_THREADS, smem, st>>>(a, nmax);
    return cudaGetLastError();
}

cudaError_t qcx_launch_resid(cudaStream_t st, const BatchSolveArgs& a, const int2* tasks, int ntask) {
    if (ntask < 1) return cudaErrorInvalidValue;
    k_resid<<<ntask, 256, 0, st>>>(a, tasks);
    return cudaGetLastError();
}
