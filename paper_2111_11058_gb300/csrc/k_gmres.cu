// k_gmres.cu -- batched right-preconditioned restarted GMRES on the reduced
// CBFM system A (G^CBF)^{-1} y = b (paper Eq. (CBFM_outer)); x = (G^CBF)^{-1} y
// (Eq. (CBFM_inner)).
//
// Every right-hand side runs its own GMRES (x0 = 0, Givens rotations, stop
// when ||b - A P y|| / ||b|| <= tol); the kernels process all of them at once
// and skip the ones that have converged.  The operator B = A P is formed once
// (cbfm_cmp_setup) so an iteration needs one product B v, done in FP64
// (CBFM_FP64) or with B in complex64 and FP32 accumulation (CBFM_MIXED).
// Arnoldi orthogonalisation, Hessenberg matrix and residual are FP64 in both:
// classical Gram-Schmidt with a second pass only where the first one
// cancelled strongly (||w_after|| < ||w_before|| / sqrt 2, the Daniel-Gragg-
// Kaufman-Stewart criterion).
#include <algorithm>
#include <atomic>
#include <vector>

#include "internal.cuh"

namespace cbfm {

namespace {

constexpr int JB = 8;          // basis vectors per block in k_dots

// Two orders of the FP64 sums.  The slowly converging systems without the CMP
// (the conventional MoM, restarted every few hundred steps) carry a change of
// rounding through hundreds of steps: their iterates, stopped at the same
// tolerance, move by up to 1e-4 of the currents when only the order of a sum
// changes.  They keep one fixed order (ORD: k_dots<true>, k_orth_ord, k_update_y, k_finish_ord,
// k_matvec64_ord; four partial sums over the basis, one over the columns of the
// product), so that results stay reproducible; the systems with the CMP, which
// do not amplify it (1e-13), take the faster order.
constexpr double DGKS_ETA = 0.70710678118654752, DGKS_ETA2 = 0.5;   // 1 / sqrt 2 and its square

__device__ __forceinline__ double block_sum(double v, double *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[i];
    return s;   // valid in thread 0
}

// sum of the nc partial sums p (fixed order), in every lane of the warp
__device__ __forceinline__ double warp_total(const double *__restrict__ p, int nc) {
    double s = 0.0;
    for (int i = threadIdx.x & 31; i < nc; i += 32) s += p[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// h[r][j] = sum_i conj(V[j][r][i]) w[r][i], j = j0 + warp, for the right-hand
// sides still iterating: one warp per basis vector (JB warps per block), four
// partial sums per lane to keep the FP64 pipe busy, warp-shuffle reduction
// only.  First pass (part == NULL): the x == 0 blocks also store ||w||^2 in
// nrm2.  Second pass: only where the first cancelled strongly, ||w||^2 after
// it (the sum of part[r][0..nc)) below DGKS_ETA2 nrm2; the x == 0 blocks
// store that decision in flag and count the work (reo_work += k + 1).
template <bool ORD>
__global__ void __launch_bounds__(32 * JB) k_dots(int64_t n, int nrhs, int k, const z64 *__restrict__ V,
                                                  const z64 *__restrict__ w, z64 *__restrict__ h, int hld,
                                                  const int *__restrict__ done, double *__restrict__ nrm2,
                                                  const double *__restrict__ part, int nc, int *__restrict__ flag,
                                                  unsigned long long *__restrict__ reo_work) {
    const int r = blockIdx.y;
    if (done[r]) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (part) {
        __shared__ int s_again;
        if (ORD) {   // the sum over w itself, in the order of k_finish_ord
            double s = 0;
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += norm2(w[(int64_t)r * n + i]);
            __shared__ double sh[32];
            s = block_sum(s, sh);
            if (threadIdx.x == 0) s_again = sqrt(s) < DGKS_ETA * sqrt(nrm2[r]);
        } else if (warp == 0) {
            const double s = warp_total(part + (int64_t)r * nc, nc);
            if (lane == 0) s_again = s < DGKS_ETA2 * nrm2[r];
        }
        __syncthreads();
        const int again = s_again;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            flag[r] = again;
            if (again) atomicAdd(reo_work, (unsigned long long)(k + 1));
        }
        if (!again) return;
    }
    const int j = blockIdx.x * JB + warp;
    const z64 *x = w + (int64_t)r * n;
    if (j <= k) {
        const z64 *v = V + ((int64_t)j * nrhs + r) * n;
        double re[4] = {0, 0, 0, 0}, im[4] = {0, 0, 0, 0};
        int64_t i = lane;
        for (; i + 96 < n; i += 128) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const z64 a = v[i + 32 * u], b = x[i + 32 * u];
                if (ORD) {
                    re[u] += a.re * b.re + a.im * b.im;
                    im[u] += a.re * b.im - a.im * b.re;
                    continue;
                }
                re[u] = fma(a.im, b.im, fma(a.re, b.re, re[u]));   // written as a sum it is a product, an FMA and an add
                im[u] = fma(-a.im, b.re, fma(a.re, b.im, im[u]));
            }
        }
        for (; i < n; i += 32) {
            const z64 a = v[i], b = x[i];
            if (ORD) {
                re[0] += a.re * b.re + a.im * b.im;
                im[0] += a.re * b.im - a.im * b.re;
                continue;
            }
            re[0] = fma(a.im, b.im, fma(a.re, b.re, re[0]));
            im[0] = fma(-a.im, b.re, fma(a.re, b.im, im[0]));
        }
        double sr = (re[0] + re[1]) + (re[2] + re[3]), si = (im[0] + im[1]) + (im[2] + im[3]);
        for (int o = 16; o > 0; o >>= 1) {
            sr += __shfl_xor_sync(0xffffffffu, sr, o);
            si += __shfl_xor_sync(0xffffffffu, si, o);
        }
        if (lane == 0) h[(int64_t)r * hld + j] = z64(sr, si);
    }
    if (!part && blockIdx.x == 0 && warp == JB - 1) {
        double s0 = 0, s1 = 0;
        int64_t i = lane;
        for (; i + 32 < n; i += 64) {
            s0 += norm2(x[i]);
            s1 += norm2(x[i + 32]);
        }
        for (; i < n; i += 32) s0 += norm2(x[i]);
        double s = s0 + s1;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) nrm2[r] = s;
    }
}

// ORD: w[r][i] -= sum_{j<=k} V[j][r][i] h[r][j] for the rows with mask[r] == want, in four partial sums over j = u, u +
// 4, ... (the last k + 1 mod 4 terms in the first one, which starts at w), added as (0 + 1) + (2 + 3).  A warp takes one
// partial sum of 32 entries, a block all four: four times the blocks of a thread that walks all of an entry's
// terms, for small systems, and the same FP64 work, which bounds it on large ones (two lanes per entry, one for each
// component, loaded every basis element twice: 99 us against 78 at n = 2304, 32 right-hand sides).
__global__ void __launch_bounds__(128) k_orth_ord(int64_t n, int nrhs, int k, const z64 *__restrict__ V,
                                                  const z64 *__restrict__ h, int hld, const int *__restrict__ mask,
                                                  int want, z64 *__restrict__ w) {
    const int r = blockIdx.y;
    if (mask[r] != want) return;
    const int u = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * 32LL + lane;
    __shared__ z64 s_acc[3][32];
    const z64 *hr = h + (int64_t)r * hld;
    z64 acc(0, 0);
    if (i < n) {
        const z64 *v = V + (int64_t)r * n + i;
        const int64_t stride = (int64_t)nrhs * n;
        if (u == 0) acc = w[(int64_t)r * n + i];
        auto sub = [&](z64 a, z64 b) {
            acc.re = __dsub_rn(acc.re, fma(a.re, b.re, -__dmul_rn(a.im, b.im)));
            acc.im = __dsub_rn(acc.im, fma(a.im, b.re, __dmul_rn(a.re, b.im)));
        };
        const int kmain = (k + 1) & ~3;
        int j = u;
        for (; j + 12 < kmain; j += 16) {
            z64 a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                a[q] = v[(j + 4 * q) * stride];
                b[q] = hr[j + 4 * q];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) sub(a[q], b[q]);
        }
        for (; j < kmain; j += 4) sub(v[j * stride], hr[j]);
        if (u == 0)
            for (j = kmain; j <= k; ++j) sub(v[j * stride], hr[j]);
    }
    if (u > 0) s_acc[u - 1][lane] = acc;
    __syncthreads();
    if (u == 0 && i < n) w[(int64_t)r * n + i] = (acc + s_acc[0][lane]) + (s_acc[1][lane] + s_acc[2][lane]);
}

// ORD: y[rhs] += sum_{j < kc} z_j V[j][rhs], ascending j
__global__ void k_update_y(int64_t n, int nrhs, int m, const z64 *__restrict__ V, const z64 *__restrict__ z,
                           const int *__restrict__ kconv, const int *__restrict__ active, z64 *__restrict__ y) {
    const int r = blockIdx.y;
    if (!active[r]) return;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    z64 acc = y[(int64_t)r * n + i];
    for (int j = 0; j < kconv[r]; ++j) acc += V[((int64_t)j * nrhs + r) * n + i] * z[(int64_t)r * m + j];
    y[(int64_t)r * n + i] = acc;
}

// w[r][i] += sgn sum_{j < cnt[r] or m} V[j][r][i] h[r][j] for the rows with
// mask[r] == want.  A block takes 32 entries i and deals the basis vectors j
// to its eight warps (a block per 256 entries with the loop over j in every
// thread left one right-hand side of 222 unknowns on one SM: 41 us a call
// against 5), summed through shared memory in warp order; part[r][block]
// receives the squared norm of the block's new entries when given.
__global__ void __launch_bounds__(256) k_combine(int64_t n, int nrhs, int m, const int *__restrict__ cnt,
                                                 const z64 *__restrict__ V, const z64 *__restrict__ h, int hld,
                                                 const int *__restrict__ mask, int want, double sgn,
                                                 z64 *__restrict__ w, double *__restrict__ part) {
    const int r = blockIdx.y;
    if (mask[r] != want) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * 32LL + lane;
    const int nj = cnt ? cnt[r] : m;
    __shared__ double s_acc[8][64];
    double re[2] = {0, 0}, im[2] = {0, 0};
    if (i < n) {
        const z64 *v = V + (int64_t)r * n + i;
        const int64_t stride = (int64_t)nrhs * n;
        const z64 *hr = h + (int64_t)r * hld;
        int j = warp;
        for (; j + 24 < nj; j += 32) {
            z64 a[4], c[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = v[(j + 8 * u) * stride];
                c[u] = hr[j + 8 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                re[u & 1] = fma(a[u].re, c[u].re, re[u & 1]);
                im[u & 1] = fma(a[u].re, c[u].im, im[u & 1]);
                re[u & 1] = fma(-a[u].im, c[u].im, re[u & 1]);
                im[u & 1] = fma(a[u].im, c[u].re, im[u & 1]);
            }
        }
        for (; j < nj; j += 8) {
            const z64 a = v[j * stride], c = hr[j];
            re[0] = fma(a.re, c.re, re[0]);
            im[0] = fma(a.re, c.im, im[0]);
            re[0] = fma(-a.im, c.im, re[0]);
            im[0] = fma(a.im, c.re, im[0]);
        }
    }
    s_acc[warp][2 * lane] = re[0] + re[1];
    s_acc[warp][2 * lane + 1] = im[0] + im[1];
    __syncthreads();
    if (warp < 2) {   // thread t: component t of the block's 32 complex entries
        const int t = threadIdx.x;
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) s += s_acc[q][t];
        double x = 0.0;
        if (blockIdx.x * 32LL + (t >> 1) < n) {
            double *p = reinterpret_cast<double *>(w + (int64_t)r * n + blockIdx.x * 32LL) + t;
            x = fma(sgn, s, *p);
            *p = x;
        }
        if (part) {
            x *= x;
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            __shared__ double s_h[2];
            if (lane == 0) s_h[warp] = x;
            asm volatile("bar.sync 1, 64;" ::: "memory");
            if (t == 0) part[(int64_t)r * gridDim.x + blockIdx.x] = s_h[0] + s_h[1];
        }
    }
}

// Column k of H for every active rhs: h1 (+ h2 if reorthogonalised), ||w||;
// previous rotations, new rotation, residual, convergence; V[k+1] = w / ||w||
// (and its complex64 copy x32 when given).
//
// The k previous rotations take a_0 = col[0] through a_{j+1} = c_j col[j+1] -
// conj(s_j) a_j, an affine map per step, and leave col[j] = c_j a_j + s_j
// col[j+1].  One thread walking them paid an FP64 instruction's ~64 clocks for
// each of 12 operations a step (51 us at k = 184).  Warps 0-3 instead compose
// the maps of a chunk per lane, scan the chunks over the lanes and the four
// warps, and walk their chunk again from the right start; warps 4-7 scale
// V[k+1] meanwhile.
constexpr int FIN_LANES = 128;
__device__ __forceinline__ void affine_after(z64 &A, z64 &B, z64 A1, z64 B1) {   // (A, B) o (A1, B1)
    z64 b = B;
    cfma(b, A, B1);
    B = b;
    A = A * A1;
}
struct RotState {   // one right-hand side's least-squares state of a cycle (see gmres_solve)
    z64 *H, *sn, *g;
    double *cs, *resid;
    const double *bnorm;
    int *done, *flag, *kconv, *n_active;   // flag, n_active: NULL in the cluster kernel
    double tol;
};
// The new rotation that zeroes (a, nrm) in column k, the residual and the convergence test (one thread).
__device__ __forceinline__ void new_rotation(const RotState &S, int r, int k, int m, int last, double nrm, z64 a) {
    z64 *Hr = S.H + (int64_t)r * (m + 1) * m;
    z64 *gr = S.g + (int64_t)r * (m + 1);
    // new rotation zeroing (a, nrm)
    double na = sqrt(norm2(a)), nb = nrm;
    double cc;
    z64 ss;
    if (nb == 0.0) { cc = 1.0; ss = z64(0, 0); }
    else if (na == 0.0) { cc = 0.0; ss = z64(1, 0); }
    else {
        double t = sqrt(na * na + nb * nb);
        cc = na / t;
        ss = a * (nb / (na * t));            // (a/|a|) nb / t, nb real
    }
    S.cs[(int64_t)r * m + k] = cc;
    S.sn[(int64_t)r * m + k] = ss;
    Hr[(int64_t)k * m + k] = cc * a + ss * nb;
    z64 gk = gr[k];
    gr[k] = cc * gk;
    gr[k + 1] = -(conj(ss) * gk);
    double res = sqrt(norm2(gr[k + 1])) / S.bnorm[r];
    S.resid[r] = res;
    if (res <= S.tol || nb == 0.0 || last) {
        S.kconv[r] = k + 1;
        S.done[r] = res <= S.tol || nb == 0.0 ? 1 : 2;
        if (S.flag) S.flag[r] = 0;
    } else if (S.n_active) {
        atomicAdd(S.n_active + k, 1);
    }
}
// Column k (col[0..k], shared) and the norm of the new vector through the previous rotations and a new one; called by
// FIN_LANES threads (four whole warps, named barrier 1).
__device__ __forceinline__ void rotate_column(const RotState &S, int r, int k, int m, int last, double nrm, int tid,
                                              const z64 *col, z64 *s_A, z64 *s_B) {
    const int lane = tid & 31, warp = tid >> 5;
    const double *cr = S.cs + (int64_t)r * m;
    const z64 *sr = S.sn + (int64_t)r * m;
    const int chunk = (k + FIN_LANES - 1) / FIN_LANES, j0 = min(k, tid * chunk), j1 = min(k, j0 + chunk);
    const z64 a0 = col[0];
    z64 A(1, 0), B(0, 0);
    for (int j = j0; j < j1; ++j) {
        const z64 al = -conj(sr[j]);
        z64 b = cr[j] * col[j + 1];
        cfma(b, al, B);
        B = b;
        A = A * al;
    }
    // inclusive scan of the chunks' maps over the warp, then over the warps
    for (int o = 1; o < 32; o <<= 1) {
        const z64 A1(__shfl_up_sync(0xffffffffu, A.re, o), __shfl_up_sync(0xffffffffu, A.im, o));
        const z64 B1(__shfl_up_sync(0xffffffffu, B.re, o), __shfl_up_sync(0xffffffffu, B.im, o));
        if (lane >= o) affine_after(A, B, A1, B1);
    }
    if (lane == 31) {
        s_A[warp] = A;
        s_B[warp] = B;
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    z64 a = a0;   // the value entering this warp's, then this lane's chunk
    for (int q = 0; q < warp; ++q) {
        z64 t = s_B[q];
        cfma(t, s_A[q], a);
        a = t;
    }
    {
        const z64 A1(__shfl_up_sync(0xffffffffu, A.re, 1), __shfl_up_sync(0xffffffffu, A.im, 1));
        z64 t(__shfl_up_sync(0xffffffffu, B.re, 1), __shfl_up_sync(0xffffffffu, B.im, 1));
        if (lane > 0) {
            cfma(t, A1, a);
            a = t;
        }
    }
    z64 *Hr = S.H + (int64_t)r * (m + 1) * m;
    for (int j = j0; j < j1; ++j) {
        const z64 b = col[j + 1];
        const double c = cr[j];
        const z64 s = sr[j];
        Hr[(int64_t)j * m + k] = c * a + s * b;
        z64 t = c * b;
        cfma(t, -conj(s), a);
        a = t;
    }
    // the lane whose chunk ends at k holds a_k (lane 0 when there is no rotation yet)
    if (k == 0 ? tid == 0 : (j0 < k && j1 == k)) {
        new_rotation(S, r, k, m, last, nrm, a);
    }
}

__global__ void __launch_bounds__(256) k_finish(int64_t n, int nrhs, int k, int m, int last,
                                                const z64 *__restrict__ h1, const z64 *__restrict__ h2, int hld,
                                                const __grid_constant__ RotState S, const double *__restrict__ part1,
                                                const double *__restrict__ part2, int nc, const z64 *__restrict__ w,
                                                z64 *__restrict__ V, c32 *__restrict__ x32) {
    const int r = blockIdx.x;
    if (S.done[r]) return;
    __shared__ z64 col[1024];
    __shared__ z64 s_A[4], s_B[4];
    __shared__ double s_nrm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool re = S.flag[r] != 0;
    for (int j = tid; j <= k; j += blockDim.x) {
        z64 v = h1[(int64_t)r * hld + j];
        if (re) v += h2[(int64_t)r * hld + j];
        col[j] = v;
    }
    if (warp == 4) {
        const double s = sqrt(warp_total((re ? part2 : part1) + (int64_t)r * nc, nc));
        if (lane == 0) s_nrm = s;
    }
    __syncthreads();
    const double nrm = s_nrm;
    if (warp >= 4) {
        const double inv = (nrm > 0.0) ? 1.0 / nrm : 0.0;
        const z64 *x = w + (int64_t)r * n;
        z64 *vn = V + ((int64_t)(k + 1) * nrhs + r) * n;
        for (int64_t i = tid - 128; i < n; i += 128) {
            const z64 v = x[i] * inv;
            vn[i] = v;
            if (x32) x32[(int64_t)r * n + i] = c32((float)v.re, (float)v.im);
        }
        return;
    }
    rotate_column(S, r, k, m, last, nrm, tid, col, s_A, s_B);
}

// ORD: column k and V[k+1] = w / ||w|| as k_finish, the norm and the rotations in one fixed order: a_{j+1} walked step by
// step by two lanes (real and imaginary part: three dependent FP64 operations a step), col[j] = c_j a_j + s_j
// col[j+1] by all threads afterwards.  Dynamic shared memory: finish_ord_smem(k).
constexpr size_t finish_ord_smem(int k) { return (size_t)(k + 1) * (3 * sizeof(z64) + sizeof(double)); }
__global__ void __launch_bounds__(256) k_finish_ord(int64_t n, int nrhs, int k, int m, int last,
                                                    const z64 *__restrict__ h1, const z64 *__restrict__ h2, int hld,
                                                    const __grid_constant__ RotState S, const z64 *__restrict__ w,
                                                    z64 *__restrict__ V, c32 *__restrict__ x32) {
    const int r = blockIdx.x;
    if (S.done[r]) return;
    extern __shared__ __align__(16) unsigned char fo_raw[];
    z64 *col = reinterpret_cast<z64 *>(fo_raw), *av = col + k + 1, *ssn = av + k + 1;
    double *scs = reinterpret_cast<double *>(ssn + k + 1);
    __shared__ double sh[32], s_nrm;
    const int tid = threadIdx.x;
    const bool re = S.flag[r] != 0;
    for (int j = tid; j <= k; j += blockDim.x) {
        z64 v = h1[(int64_t)r * hld + j];
        if (re) v += h2[(int64_t)r * hld + j];
        col[j] = v;
        if (j < k) {
            scs[j] = S.cs[(int64_t)r * m + j];
            ssn[j] = S.sn[(int64_t)r * m + j];
        }
    }
    const z64 *x = w + (int64_t)r * n;
    double s = 0;
    for (int64_t i = tid; i < n; i += blockDim.x) s += norm2(x[i]);
    s = block_sum(s, sh);   // contains __syncthreads: col, scs and ssn are visible afterwards
    if (tid == 0) s_nrm = sqrt(s);
    __syncthreads();
    const double nrm = s_nrm;
    if (tid < 32) {
        const int c = tid & 1;
        double own = c == 0 ? col[0].re : col[0].im;
        for (int j = 0; j < k; ++j) {
            const double oth = __shfl_xor_sync(0xffffffffu, own, 1);
            if (tid < 2) reinterpret_cast<double *>(av + j)[c] = own;
            const double b = reinterpret_cast<const double *>(col + j + 1)[c];
            const double x1 = fma(ssn[j].re, own, (c == 0 ? ssn[j].im : -ssn[j].im) * oth);   // conj(s) a
            own = fma(scs[j], b, -x1);
        }
        const double oth = __shfl_xor_sync(0xffffffffu, own, 1);
        if (tid == 0) new_rotation(S, r, k, m, last, nrm, z64(own, oth));
    } else {
        const double inv = (nrm > 0.0) ? 1.0 / nrm : 0.0;
        z64 *vn = V + ((int64_t)(k + 1) * nrhs + r) * n;
        for (int64_t i = tid - 32; i < n; i += blockDim.x - 32) {
            const z64 v = x[i] * inv;
            vn[i] = v;
            if (x32) x32[(int64_t)r * n + i] = c32((float)v.re, (float)v.im);
        }
    }
    __syncthreads();
    z64 *Hr = S.H + (int64_t)r * (m + 1) * m;
    for (int j = tid; j < k; j += blockDim.x) {
        const z64 a = av[j], b = col[j + 1];
        Hr[(int64_t)j * m + k] = scs[j] * a + ssn[j] * b;
    }
}

// out[r] = M in[r], M complex64 n x n row-major, in complex64, FP32 sums over
// ascending k, for the right-hand sides still iterating (done == NULL: all).
// Tiles of 16 output rows x RT right-hand sides, 256 threads with two outputs
// each (RT = 32) or 128 with one (RT = 8, for few right-hand sides).  Both operands
// come through a three-stage cp.async pipeline of 32 values of k; the rows of a
// stage are 272 bytes apart, so that eight rows' 16-byte reads (two values of
// k) fall into different banks.  Bound: FP32 multiply-adds at one warp per
// scheduler (n = 2304, 32 right-hand sides: 680 M FMA, 18 us at full rate).
// Before: no pipeline, and every block converted the FP64 input again on
// the FP64 pipe (362 us).  n is even (two halves), so 16-byte chunks never straddle a row's end.
constexpr int MV_N = 16, MV_K = 32, MV_PITCH = MV_K + 2, MV_STAGES = 3;
__device__ __forceinline__ void cp16(void *dst, const void *src, bool live) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(live ? 16 : 0)
                 : "memory");
}
template <int RT>
__global__ void __launch_bounds__(RT == 32 ? 256 : 128) k_matvec32(int64_t n, int nrhs, const c32 *__restrict__ M,
                                                  const c32 *__restrict__ in, z64 *__restrict__ out,
                                                  const int *__restrict__ done) {
    constexpr int NT = RT == 32 ? 256 : 128, NR = RT * MV_N / NT;   // threads, right-hand sides per thread
    __shared__ __align__(16) c32 Ms[MV_STAGES][MV_N][MV_PITCH];
    __shared__ __align__(16) c32 Xs[MV_STAGES][RT][MV_PITCH];
    const int tid = threadIdx.x, tx = tid % MV_N, ty = tid / MV_N;
    const int64_t r0 = (int64_t)blockIdx.y * RT, c0 = (int64_t)blockIdx.x * MV_N;
    bool any = false;
    for (int a = 0; a < RT; ++a) any |= r0 + a < nrhs && (!done || done[r0 + a] == 0);
    if (!any) return;
    const int nst = (int)((n + MV_K - 1) / MV_K);
    auto fetch = [&](int s) {
        if (s < nst) {
            const int b = s % MV_STAGES;
            for (int q = tid; q < (MV_N + RT) * (MV_K / 2); q += NT) {
                const int row = q / (MV_K / 2), c = 2 * (q % (MV_K / 2));
                const int64_t kx = (int64_t)s * MV_K + c;
                if (row < MV_N) {
                    const bool live = c0 + row < n && kx < n;
                    cp16(&Ms[b][row][c], live ? M + (c0 + row) * n + kx : M, live);
                } else {
                    const int64_t r = r0 + row - MV_N;
                    const bool live = r < nrhs && kx < n;
                    cp16(&Xs[b][row - MV_N][c], live ? in + r * n + kx : in, live);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    c32 acc[NR];
    for (int a = 0; a < NR; ++a) acc[a] = c32(0, 0);
    for (int s = 0; s < MV_STAGES - 1; ++s) fetch(s);
    for (int s = 0; s < nst; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(MV_STAGES - 2) : "memory");
        __syncthreads();   // stage s has landed for every thread; stage s - 1 is no longer read
        fetch(s + MV_STAGES - 1);
        const int b = s % MV_STAGES;
#pragma unroll
        for (int kk = 0; kk < MV_K; kk += 2) {
            float4 xa[NR];
#pragma unroll
            for (int a = 0; a < NR; ++a) xa[a] = *reinterpret_cast<const float4 *>(&Xs[b][ty + 16 * a][kk]);
            const float4 mb = *reinterpret_cast<const float4 *>(&Ms[b][tx][kk]);
#pragma unroll
            for (int a = 0; a < NR; ++a) {
                cfma(acc[a], c32(xa[a].x, xa[a].y), c32(mb.x, mb.y));
                cfma(acc[a], c32(xa[a].z, xa[a].w), c32(mb.z, mb.w));
            }
        }
    }
    const int64_t c = c0 + tx;
    for (int a = 0; a < NR; ++a) {
        const int64_t r = r0 + ty + 16 * a;
        if (r >= nrhs || c >= n || (done && done[r] != 0)) continue;
        out[r * n + c] = z64((double)acc[a].re, (double)acc[a].im);
    }
}

// The FP64 product: one warp per output row and RW right-hand sides, the lanes
// over k, so that every FP64 warp instruction has 32 useful lanes whatever the
// number of right-hand sides (32 x 16 tiles spent 134 us on n = 222 and one).
template <int RW>
__global__ void __launch_bounds__(256) k_matvec64(int64_t n, int nrhs, const z64 *__restrict__ M,
                                                  const z64 *__restrict__ in, z64 *__restrict__ out,
                                                  const int *__restrict__ done) {
    const int lane = threadIdx.x & 31;
    const int64_t c = blockIdx.x * 8LL + (threadIdx.x >> 5);
    const int r0 = blockIdx.y * RW;
    bool any = false;
#pragma unroll
    for (int a = 0; a < RW; ++a) any |= r0 + a < nrhs && (!done || done[r0 + a] == 0);
    if (!any || c >= n) return;
    z64 acc[RW][2];
#pragma unroll
    for (int a = 0; a < RW; ++a) acc[a][0] = acc[a][1] = z64(0, 0);
    const z64 *m = M + c * n;
    int u = 0;
    for (int64_t k = lane; k < n; k += 32, u ^= 1) {
        const z64 b = m[k];
#pragma unroll
        for (int a = 0; a < RW; ++a)
            if (r0 + a < nrhs) {
                const z64 x = in[(int64_t)(r0 + a) * n + k];
                if (u) cfma(acc[a][1], x, b);
                else cfma(acc[a][0], x, b);
            }
    }
#pragma unroll
    for (int a = 0; a < RW; ++a) {
        if (r0 + a >= nrhs) break;
        z64 s = acc[a][0] + acc[a][1];
        for (int o = 16; o > 0; o >>= 1) {
            s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
            s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
        }
        if (lane == 0 && (!done || done[r0 + a] == 0)) out[(int64_t)(r0 + a) * n + c] = s;
    }
}

// ORD: the FP64 product with one sum over ascending k per component: a warp
// takes 16 output rows (two lanes each, real and imaginary part) of one
// right-hand side, four right-hand sides a block, both operands through a
// three-stage cp.async pipeline.  Bound: the chain of 2 n dependent FP64 FMAs
// (n = 960: 64 us; a thread with four outputs and both components took 520 us).
constexpr int MO_K = 16, MO_PITCH = MO_K + 1, MO_R = 4;
__global__ void __launch_bounds__(32 * MO_R) k_matvec64_ord(int64_t n, int nrhs, const z64 *__restrict__ M,
                                                            const z64 *__restrict__ in, z64 *__restrict__ out,
                                                            const int *__restrict__ done) {
    __shared__ __align__(16) z64 Ms[MV_STAGES][MV_N][MO_PITCH];
    __shared__ __align__(16) z64 Xs[MV_STAGES][MO_R][MO_PITCH];
    const int tid = threadIdx.x, lane = tid & 31, row = lane >> 1, c = lane & 1, q = tid >> 5;
    const int64_t r0 = (int64_t)blockIdx.y * MO_R, c0 = (int64_t)blockIdx.x * MV_N;
    bool any = false;
    for (int a = 0; a < MO_R; ++a) any |= r0 + a < nrhs && (!done || done[r0 + a] == 0);
    if (!any) return;
    const bool mine = r0 + q < nrhs && (!done || done[r0 + q] == 0);   // the same in a warp
    const int nst = (int)((n + MO_K - 1) / MO_K);
    auto fetch = [&](int s) {
        if (s < nst) {
            const int b = s % MV_STAGES;
            for (int e = tid; e < (MV_N + MO_R) * MO_K; e += 32 * MO_R) {
                const int rw = e / MO_K, kk = e % MO_K;
                const int64_t kx = (int64_t)s * MO_K + kk;
                if (rw < MV_N) {
                    const bool live = c0 + rw < n && kx < n;
                    cp16(&Ms[b][rw][kk], live ? M + (c0 + rw) * n + kx : M, live);
                } else {
                    const int64_t r = r0 + rw - MV_N;
                    const bool live = r < nrhs && kx < n;
                    cp16(&Xs[b][rw - MV_N][kk], live ? in + r * n + kx : in, live);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    double acc = 0.0;
    for (int s = 0; s < MV_STAGES - 1; ++s) fetch(s);
    for (int s = 0; s < nst; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(MV_STAGES - 2) : "memory");
        __syncthreads();
        fetch(s + MV_STAGES - 1);
        const int b = s % MV_STAGES;
        if (mine) {
#pragma unroll
            for (int kk = 0; kk < MO_K; ++kk) {
                const z64 x = Xs[b][q][kk], e = Ms[b][row][kk];
                acc = fma(x.re, c == 0 ? e.re : e.im, acc);
                acc = fma(x.im, c == 0 ? -e.im : e.re, acc);
            }
        }
    }
    if (mine && c0 + row < n) reinterpret_cast<double *>(out + (r0 + q) * n + c0 + row)[c] = acc;
}

// The same sums in tiles of 32 right-hand sides x 16 output rows, four outputs a thread: a CTA's four warps keep its SM's
// FP64 pipe full (1024 clocks a value of k), where the kernel above spends issue slots on the operands of two
// multiply-adds a lane and reaches 0.57 of the pipe.  For many right-hand sides: product of n = 2304 and 64 of them
// 2.4 ms against 3.9, 128 4.7 against 7.5; with few, whole tiles are padding (n = 960, 24: 0.60 against 0.32).
constexpr int MT_R = 32, MT_K = 32;
__global__ void __launch_bounds__(128) k_matvec64_tile(int64_t n, int nrhs, const z64 *__restrict__ M,
                                                       const z64 *__restrict__ in, z64 *__restrict__ out,
                                                       const int *__restrict__ done) {
    __shared__ z64 Xs[MT_K][MT_R + 1];
    __shared__ z64 Ms[MT_K][MV_N + 1];
    const int tid = threadIdx.x, tx = tid % 8, ty = tid / 8;
    const int64_t r0 = (int64_t)blockIdx.y * MT_R, c0 = (int64_t)blockIdx.x * MV_N;
    bool any = false;
    for (int a = 0; a < MT_R; ++a) any |= r0 + a < nrhs && (!done || done[r0 + a] == 0);
    if (!any) return;
    z64 acc[2][2];
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b) acc[a][b] = z64(0, 0);
    for (int64_t k0 = 0; k0 < n; k0 += MT_K) {
        for (int e = tid; e < (MT_R + MV_N) * MT_K; e += 128) {
            const int row = e / MT_K, kk = e % MT_K;
            const int64_t kx = k0 + kk, r = r0 + row, c = c0 + row - MT_R;
            if (row < MT_R) Xs[kk][row] = r < nrhs && kx < n ? in[r * n + kx] : z64(0, 0);
            else Ms[kk][row - MT_R] = c < n && kx < n ? M[c * n + kx] : z64(0, 0);
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < MT_K; ++kk) {
            const z64 x[2] = {Xs[kk][ty], Xs[kk][ty + 16]}, m[2] = {Ms[kk][tx], Ms[kk][tx + 8]};
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    z64 &o = acc[a][b];
                    o.re = fma(x[a].im, -m[b].im, fma(x[a].re, m[b].re, o.re));
                    o.im = fma(x[a].im, m[b].re, fma(x[a].re, m[b].im, o.im));
                }
        }
        __syncthreads();
    }
    for (int a = 0; a < 2; ++a) {
        const int64_t r = r0 + ty + 16 * a;
        if (r >= nrhs || (done && done[r] != 0)) continue;
        for (int b = 0; b < 2; ++b) {
            const int64_t c = c0 + tx + 8 * b;
            if (c < n) out[r * n + c] = acc[a][b];
        }
    }
}

// ------------------------------------------------- whole cycle on a cluster
// The Arnoldi cycle of few right-hand sides of moderate order in one launch: a
// cluster of CC CTAs per right-hand side.  As separate kernels an iteration is
// six dependent launches of ~7 us that mostly wait (45 us at n = 222, one
// right-hand side, whatever its work); here it is three hardware cluster
// barriers (two more where the second Gram-Schmidt pass runs).  CTA c owns the
// entries [c per, (c + 1) per) of w and of every basis vector.  Iteration k:
//   x = V[k] = w / ||w|| staged in shared memory by every CTA (own entries written to V);
//   own rows of w' = B x;                                                | barrier
//   h_j = V[j]^H w', one warp per j over all warps of the cluster;       | barrier
//   own entries w' -= sum_j V[j] h_j, partial norms;                     | barrier
// The rotations of column k (four extra warps of CTA 0) run beside the product and
// the dot products of iteration k + 1; a convergence is seen after its second
// barrier, so the cycle runs at most one iteration too many.  Every thread of
// the cluster reaches every barrier: all decisions are taken from values written
// before the barrier ahead of them.
// The complex64 product sums over ascending k in one thread per row, as the
// kernels above do.
constexpr int GC_WARPS = 8, GC_THREADS = 32 * GC_WARPS + FIN_LANES;
constexpr int GC_NMAX = 1024, GC_CL = 16;
constexpr int GC_K = 16, GC_PITCH = GC_K + 2;   // complex64 product: values of k per stage
struct GmresCl {
    int64_t n;
    int nrhs, m, mc, hld;
    const z64 *M64;
    const c32 *M32;
    z64 *V, *w, *h1, *h2;      // w: two buffers of nrhs x n; h1, h2: two buffers of nrhs x hld (by the parity of k)
    double *part;              // nrhs x 2 (parity of k) x 3 x 16 partial norms: before, after the first, the second pass
    unsigned long long *reo;
    RotState rot;
};
__device__ __forceinline__ void cl_arrive_all() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait_all() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ z64 ldcg(const z64 *p) {
    const double2 v = __ldcg(reinterpret_cast<const double2 *>(p));
    return z64(v.x, v.y);
}

template <bool F32>
__global__ void __launch_bounds__(GC_THREADS) k_gmres_cl(const __grid_constant__ GmresCl P) {
    constexpr int CC = GC_CL, ROWS = GC_NMAX / CC;   // most entries a CTA owns
    __shared__ __align__(16) z64 x_s[F32 ? 1 : GC_NMAX];
    __shared__ __align__(16) c32 x32_s[F32 ? GC_NMAX : 2];
    __shared__ __align__(16) c32 Ms[F32 ? 2 : 1][F32 ? ROWS : 1][GC_PITCH];
    __shared__ z64 s_acc[32 * GC_WARPS];
    __shared__ double s_red[GC_WARPS];
    __shared__ z64 col[1024], s_A[4], s_B[4];
    const int r = blockIdx.x / CC, c = blockIdx.x % CC;
    if (P.rot.done[r]) return;   // the whole cluster
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = (int)P.n;
    const int per = (n + CC - 1) / CC, i0 = min(n, c * per), own = min(n, i0 + per) - i0;
    const int64_t nn = (int64_t)P.nrhs * P.n;
    const bool rotw = warp >= GC_WARPS;
    int W = 8;                                     // entries per slot of the update
    while (W < per) W <<= 1;
    // sum of the CC partial norms p, in every thread
    auto total = [&](const double *p) {
        double s = lane < CC ? __ldcg(p + lane) : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    auto cta_sync = [&] { asm volatile("bar.sync 2, 256;" ::: "memory"); };   // the GC_WARPS computing warps
    double nrm = 0.0;
    bool again = false;
    for (int k = 0;; ++k) {
        const bool fin = k == P.mc;   // the cycle is over: only the last column's rotations remain
        double *part = P.part + ((int64_t)r * 2 + (k & 1)) * 3 * 16;
        z64 *w = P.w + (int64_t)(k & 1) * nn + (int64_t)r * P.n;
        const z64 *wp = P.w + (int64_t)((k & 1) ^ 1) * nn + (int64_t)r * P.n;
        z64 *h1 = P.h1 + ((int64_t)(k & 1) * P.nrhs + r) * P.hld, *h2 = P.h2 + ((int64_t)(k & 1) * P.nrhs + r) * P.hld;
        if (rotw) {
            cl_arrive_all();
            if (c == 0 && k > 0) {   // column k - 1
                const z64 *g1 = P.h1 + ((int64_t)((k & 1) ^ 1) * P.nrhs + r) * P.hld;
                const z64 *g2 = P.h2 + ((int64_t)((k & 1) ^ 1) * P.nrhs + r) * P.hld;
                const int q = tid - 32 * GC_WARPS;
                for (int j = q; j < k; j += FIN_LANES) {
                    z64 v = ldcg(g1 + j);
                    if (again) v += ldcg(g2 + j);
                    col[j] = v;
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                rotate_column(P.rot, r, k - 1, P.m, fin ? 1 : 0, nrm, q, col, s_A, s_B);
                __syncwarp();
            }
            cl_wait_all();
            if (fin) break;
            cl_arrive_all();
            cl_wait_all();
        } else {
            if (fin) {
                cl_arrive_all();
                cl_wait_all();
                break;
            }
            // x = V[k]
            const double inv = k == 0 ? 1.0 : (nrm > 0.0 ? 1.0 / nrm : 0.0);
            z64 *vk = P.V + ((int64_t)k * P.nrhs + r) * P.n;
            for (int i = tid; i < n; i += 32 * GC_WARPS) {
                z64 v = ldcg(k == 0 ? vk + i : wp + i);
                if (k > 0) {
                    v = v * inv;
                    if (i >= i0 && i < i0 + own) vk[i] = v;
                }
                if (F32) x32_s[i] = c32((float)v.re, (float)v.im);
                else x_s[i] = v;
            }
            cta_sync();
            // own rows of the product, and their squared norm
            double s2 = 0.0;
            if (F32) {
                const int nst = (n + GC_K - 1) / GC_K;
                auto fetch = [&](int s) {
                    if (s < nst)
                        for (int q = tid; q < own * (GC_K / 2); q += 32 * GC_WARPS) {
                            const int row = q / (GC_K / 2), cc = 2 * (q % (GC_K / 2)), kx = s * GC_K + cc;
                            const bool live = kx < n;
                            cp16(&Ms[s & 1][row][cc], P.M32 + (int64_t)(i0 + row) * n + (live ? kx : 0), live);
                        }
                    asm volatile("cp.async.commit_group;" ::: "memory");
                };
                c32 acc(0, 0);
                fetch(0);
                for (int s = 0; s < nst; ++s) {
                    fetch(s + 1);
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    cta_sync();
                    if (tid < own) {
                        const int ke = min(GC_K, n - s * GC_K);   // even
                        const float4 *xp = reinterpret_cast<const float4 *>(x32_s + s * GC_K);
#pragma unroll 8
                        for (int kk = 0; kk < ke; kk += 2) {
                            const float4 xv = xp[kk >> 1], mv = *reinterpret_cast<const float4 *>(&Ms[s & 1][tid][kk]);
                            cfma(acc, c32(xv.x, xv.y), c32(mv.x, mv.y));
                            cfma(acc, c32(xv.z, xv.w), c32(mv.z, mv.w));
                        }
                    }
                    cta_sync();   // before stage s + 2 overwrites this one
                }
                if (tid < own) {
                    const z64 v((double)acc.re, (double)acc.im);
                    w[i0 + tid] = v;
                    s2 = fma(v.re, v.re, v.im * v.im);
                }
            } else {
                for (int i = warp; i < own; i += GC_WARPS) {
                    const z64 *mr = P.M64 + (int64_t)(i0 + i) * n;
                    z64 a0(0, 0), a1(0, 0);
                    int kk = lane;
                    for (; kk + 32 < n; kk += 64) {
                        const z64 b0 = mr[kk], b1 = mr[kk + 32];
                        cfma(a0, x_s[kk], b0);
                        cfma(a1, x_s[kk + 32], b1);
                    }
                    if (kk < n) cfma(a0, x_s[kk], mr[kk]);
                    a0 += a1;
                    for (int o = 16; o > 0; o >>= 1) {
                        a0.re += __shfl_xor_sync(0xffffffffu, a0.re, o);
                        a0.im += __shfl_xor_sync(0xffffffffu, a0.im, o);
                    }
                    if (lane == 0) {
                        w[i0 + i] = a0;
                        s2 += fma(a0.re, a0.re, a0.im * a0.im);
                    }
                }
            }
            for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            if (lane == 0) s_red[warp] = s2;
            cta_sync();
            if (tid == 0) {
                double t = 0.0;
                for (int q = 0; q < GC_WARPS; ++q) t += s_red[q];
                part[c] = t;
            }
            cl_arrive_all();
            cl_wait_all();
            // h_j = V[j]^H w
            for (int pass = 0;; ++pass) {
                z64 *h = pass == 0 ? h1 : h2;
                for (int j = c * GC_WARPS + warp; j <= k; j += CC * GC_WARPS) {
                    const z64 *v = P.V + ((int64_t)j * P.nrhs + r) * P.n;
                    double re[2] = {0, 0}, im[2] = {0, 0};
                    int i = lane;
                    for (; i + 32 < n; i += 64) {
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const z64 a = ldcg(v + i + 32 * u), b = ldcg(w + i + 32 * u);
                            re[u] = fma(a.im, b.im, fma(a.re, b.re, re[u]));
                            im[u] = fma(-a.im, b.re, fma(a.re, b.im, im[u]));
                        }
                    }
                    if (i < n) {
                        const z64 a = ldcg(v + i), b = ldcg(w + i);
                        re[0] = fma(a.im, b.im, fma(a.re, b.re, re[0]));
                        im[0] = fma(-a.im, b.re, fma(a.re, b.im, im[0]));
                    }
                    double sr = re[0] + re[1], si = im[0] + im[1];
                    for (int o = 16; o > 0; o >>= 1) {
                        sr += __shfl_xor_sync(0xffffffffu, sr, o);
                        si += __shfl_xor_sync(0xffffffffu, si, o);
                    }
                    if (lane == 0) h[j] = z64(sr, si);
                }
                cl_arrive_all();
                cl_wait_all();
                if (pass == 0 && k > 0 && __ldcg(P.rot.done + r)) return;   // column k - 1 converged (all threads alike)
                // own entries of w -= sum_j V[j] h_j
                {
                    const int i = tid % W, slot = tid / W, ns = 32 * GC_WARPS / W;
                    double re[2] = {0, 0}, im[2] = {0, 0};
                    if (i < own) {
                        const z64 *v = P.V + (int64_t)r * P.n + i0 + i;
                        const int64_t stride = (int64_t)P.nrhs * P.n;
                        int j = slot;
                        for (; j + ns <= k; j += 2 * ns) {
                            const z64 a0 = ldcg(v + j * stride), a1 = ldcg(v + (j + ns) * stride);
                            const z64 c0 = ldcg(h + j), c1 = ldcg(h + j + ns);
                            re[0] = fma(-a0.im, c0.im, fma(a0.re, c0.re, re[0]));
                            im[0] = fma(a0.im, c0.re, fma(a0.re, c0.im, im[0]));
                            re[1] = fma(-a1.im, c1.im, fma(a1.re, c1.re, re[1]));
                            im[1] = fma(a1.im, c1.re, fma(a1.re, c1.im, im[1]));
                        }
                        if (j <= k) {
                            const z64 a0 = ldcg(v + j * stride), c0 = ldcg(h + j);
                            re[0] = fma(-a0.im, c0.im, fma(a0.re, c0.re, re[0]));
                            im[0] = fma(a0.im, c0.re, fma(a0.re, c0.im, im[0]));
                        }
                    }
                    s_acc[tid] = z64(re[0] + re[1], im[0] + im[1]);
                    cta_sync();
                    double t2 = 0.0;
                    if (tid < 2 * own) {
                        const double *a = reinterpret_cast<const double *>(s_acc) + tid;
                        double t = 0.0;
                        for (int q = 0; q < ns; ++q) t += a[2 * W * q];
                        double *p = reinterpret_cast<double *>(w + i0) + tid;
                        t = __ldcg(p) - t;
                        *p = t;
                        t2 = t * t;
                    }
                    for (int o = 16; o > 0; o >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, o);
                    if (lane == 0) s_red[warp] = t2;
                    cta_sync();
                    if (tid == 0) {
                        double t = 0.0;
                        for (int q = 0; q < GC_WARPS; ++q) t += s_red[q];
                        part[16 * (1 + pass) + c] = t;
                    }
                }
                cl_arrive_all();
                cl_wait_all();
                if (pass == 1) break;
                // again where the first pass cancelled strongly
                if (!(total(part + 16) < DGKS_ETA2 * total(part))) break;
            }
        }
        if (rotw) {   // the same barriers and decisions as the computing warps
            if (k > 0 && __ldcg(P.rot.done + r)) return;
            cl_arrive_all();
            cl_wait_all();
        }
        const double s1 = total(part + 16);
        again = s1 < DGKS_ETA2 * total(part);
        if (again && rotw)
            for (int b = 0; b < 2; ++b) {
                cl_arrive_all();
                cl_wait_all();
            }
        nrm = sqrt(again ? total(part + 32) : s1);
        if (again && c == 0 && tid == 0) atomicAdd(P.reo, (unsigned long long)(k + 1));
    }
}

// Back-substitution H(0:kc,0:kc) z = g(0:kc), one block per rhs (column oriented).
__global__ void k_backsolve(int nrhs, int m, const z64 *__restrict__ H, z64 *__restrict__ g,
                            const int *__restrict__ kconv, const int *__restrict__ active, z64 *__restrict__ z) {
    const int r = blockIdx.x;
    if (!active[r]) return;
    const int kc = kconv[r];
    const z64 *Hr = H + (int64_t)r * (m + 1) * m;
    z64 *gr = g + (int64_t)r * (m + 1);
    z64 *zr = z + (int64_t)r * m;
    __shared__ z64 zj;
    for (int j = kc - 1; j >= 0; --j) {
        if (threadIdx.x == 0) {
            z64 d = Hr[(int64_t)j * m + j];
            zj = (norm2(d) > 0.0) ? cdiv(gr[j], d) : z64(0, 0);
            zr[j] = zj;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < j; i += blockDim.x) gr[i] -= Hr[(int64_t)i * m + j] * zj;
        __syncthreads();
    }
}

// start of a cycle: r = b - w (w = B y, or 0), beta = ||r||, V[0] = r / beta, g = beta e1
__global__ void k_start(int64_t n, int nrhs, int m, const z64 *__restrict__ b, const z64 *__restrict__ w, int have_w,
                        z64 *__restrict__ V, z64 *__restrict__ g, const double *__restrict__ bnorm,
                        double *__restrict__ resid, int *__restrict__ done, double tol, c32 *__restrict__ x32) {
    const int r = blockIdx.x;
    double s = 0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        z64 v = b[(int64_t)r * n + i];
        if (have_w) v -= w[(int64_t)r * n + i];
        s += norm2(v);
    }
    __shared__ double sh[32];
    __shared__ double beta;
    s = block_sum(s, sh);
    if (threadIdx.x == 0) {
        beta = sqrt(s);
        z64 *gr = g + (int64_t)r * (m + 1);
        for (int j = 0; j <= m; ++j) gr[j] = z64(0, 0);
        gr[0] = z64(beta, 0);
        double res = (bnorm[r] > 0.0) ? beta / bnorm[r] : 0.0;
        resid[r] = res;
        if (done[r] != 1) done[r] = (res <= tol || beta == 0.0) ? 1 : 0;
    }
    __syncthreads();
    const double inv = (beta > 0.0) ? 1.0 / beta : 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        z64 v = b[(int64_t)r * n + i];
        if (have_w) v -= w[(int64_t)r * n + i];
        v = v * inv;
        V[(int64_t)r * n + i] = v;
        if (x32) x32[(int64_t)r * n + i] = c32((float)v.re, (float)v.im);
    }
}

__global__ void k_norms(int64_t n, int nrhs, const z64 *__restrict__ b, double *__restrict__ out) {
    const int r = blockIdx.x;
    double s = 0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += norm2(b[(int64_t)r * n + i]);
    __shared__ double sh[32];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) out[r] = sqrt(s);
}

}  // namespace

// out[r] = M in[r] for the rows with done[r] == 0 (NULL: all): M32 in complex64 with FP32 sums (in32: the rows rounded
// to complex64, or NULL to round in here), else M64 in FP64
static void apply_rows(int64_t n, const z64 *M64, const c32 *M32, const z64 *in, const c32 *in32, z64 *out, int nrhs,
                       const int *done, bool ord, cudaStream_t st) {
    DevBuf<c32> tmp;
    if (M32 && !in32) {
        tmp.alloc((size_t)nrhs * n);
        launch_z64_to_c32(in, tmp.p, (int64_t)nrhs * n, st);
        in32 = tmp.p;
    }
    ProfScope ps_("k_matvec", st);
    if (M32) {
        const unsigned gx = (unsigned)((n + MV_N - 1) / MV_N);
        // one output per thread while the blocks of 8 right-hand sides still fit the SMs once (n = 2304: 12 us
        // against 20 us of a half-empty 32 tile)
        if (nrhs <= 8) k_matvec32<8><<<dim3(gx, (unsigned)((nrhs + 7) / 8)), 128, 0, st>>>(n, nrhs, M32, in32, out, done);
        else k_matvec32<32><<<dim3(gx, (unsigned)((nrhs + 31) / 32)), 256, 0, st>>>(n, nrhs, M32, in32, out, done);
    } else if (ord) {
        // tiles where their waves (n x 1024 clocks each) beat the row kernel's n^2 nrhs x 3.5 / SMs clocks
        const int64_t gx = (n + MV_N - 1) / MV_N, gt = (nrhs + MT_R - 1) / MT_R;
        const int64_t waves = (gx * gt + sm_count() - 1) / sm_count();
        if (1024.0 * waves * sm_count() < 3.5 * (double)n * nrhs) {
            k_matvec64_tile<<<dim3((unsigned)gx, (unsigned)gt), 128, 0, st>>>(n, nrhs, M64, in, out, done);
            launched("k_matvec");
            return;
        }
        const dim3 g((unsigned)((n + MV_N - 1) / MV_N), (unsigned)((nrhs + MO_R - 1) / MO_R));
        k_matvec64_ord<<<g, 32 * MO_R, 0, st>>>(n, nrhs, M64, in, out, done);
    } else {
        const unsigned gx = (unsigned)((n + 7) / 8);
        if (nrhs == 1) k_matvec64<1><<<dim3(gx, 1), 256, 0, st>>>(n, nrhs, M64, in, out, done);
        else k_matvec64<4><<<dim3(gx, (unsigned)((nrhs + 3) / 4)), 256, 0, st>>>(n, nrhs, M64, in, out, done);
    }
    launched("k_matvec");
}

// out[r] = done[r] == 0 (or done NULL) ? in[r] : 0 (rows of length n)
__global__ void k_mask_rows(int64_t n, int nrhs, const int *__restrict__ done, const z64 *__restrict__ in,
                            z64 *__restrict__ out) {
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n * nrhs;
         idx += (int64_t)gridDim.x * blockDim.x)
        out[idx] = !done || done[idx / n] == 0 ? in[idx] : z64(0, 0);
}

static void apply_B(Red &rd, int pc, const z64 *in, const c32 *in32, z64 *out, int nrhs, const int *done,
                    cudaStream_t st) {
    DevBuf<z64> v, z;
    if (pc == CBFM_PC_CMP_INEXACT) {   // A (G^CBF)^{-1} in: the inner GMRES, then the product with A
        // rows the mask leaves out may hold stale basis vectors: they enter the inner solve as zero
        v.alloc((size_t)nrhs * rd.n);
        z.alloc((size_t)nrhs * rd.n);
        const int64_t work = rd.n * nrhs;
        k_mask_rows<<<(unsigned)std::min<int64_t>((work + 255) / 256, 65535), 256, 0, st>>>(rd.n, nrhs, done, in, v.p);
        launched("k_mask_rows");
        cmp_inner_apply(rd, v.p, z.p, nrhs, st);
        in = z.p;
        in32 = nullptr;
    }
    const bool mixed = rd.prec != CBFM_FP64;
    apply_rows(rd.n, mixed ? nullptr : pc_op64(rd, pc), mixed ? pc_op32(rd, pc) : nullptr, in, in32, out, nrhs, done,
               pc != CBFM_PC_CMP, st);
}

static void set_finish_smem() {   // once per device: columns of up to 1023 entries
    static std::atomic<bool> done[64];
    int dev = 0;
    CBFM_CUDA(cudaGetDevice(&dev));
    if (dev < 64 && done[dev].load(std::memory_order_acquire)) return;
    CBFM_CUDA(cudaFuncSetAttribute(k_finish_ord, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)finish_ord_smem(1023)));
    if (dev < 64) done[dev].store(true, std::memory_order_release);
}
static cudaLaunchConfig_t gmres_cl_cfg(int nrhs, cudaStream_t st, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nrhs * GC_CL), 1, 1);
    cfg.blockDim = dim3(GC_THREADS, 1, 1);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = GC_CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}
static void launch_gmres_cl(const GmresCl &P, bool f32, cudaStream_t st) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = gmres_cl_cfg(P.nrhs, st, at);
    if (f32) CBFM_CUDA(cudaLaunchKernelEx(&cfg, k_gmres_cl<true>, P));
    else CBFM_CUDA(cudaLaunchKernelEx(&cfg, k_gmres_cl<false>, P));
}
// Clusters of the cycle kernel that can be resident at once on this device (0: none, the size is not portable).
static int gmres_clusters(bool f32) {
    static std::atomic<int> known[64][2];   // zero-initialised: 0 = not asked yet, else the count + 1
    int dev = 0;
    CBFM_CUDA(cudaGetDevice(&dev));
    if (dev < 64) {
        const int k = known[dev][f32].load(std::memory_order_acquire);
        if (k) return k - 1;
    }
    int nc = 0;
    auto ask = [&](auto *f) {
        if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return;
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg = gmres_cl_cfg(1, 0, at);
        if (cudaOccupancyMaxActiveClusters(&nc, f, &cfg) != cudaSuccess) nc = 0;
    };
    if (f32) ask(k_gmres_cl<true>);
    else ask(k_gmres_cl<false>);
    (void)cudaGetLastError();   // a refused non-portable size is not an error here
    if (dev < 64) known[dev][f32].store(nc + 1, std::memory_order_release);
    return nc;
}

GmresOut gmres_solve(Red &rd, const z64 *d_b, int nrhs, double tol, int maxit, int restart, int pc, z64 *d_x,
                     cudaStream_t st) {
    const int64_t n = rd.n;
    CBFM_REQUIRE(nrhs <= 65535, "nrhs must be <= 65535");
    const int m = std::max(1, std::min<int>(std::min(restart, 1023),
                                            (int)std::min<int64_t>(maxit, std::max<int64_t>(n, 1))));
    DevBuf<z64> V, H, sn, g, y, w, hb1, hb2, zs;
    DevBuf<double> cs, bnorm, resid, nrm0, part1, part2;
    DevBuf<c32> x32;   // the newest basis vectors rounded to complex64 (mixed precision)
    DevBuf<int> done, kconv, active, nact, flag;
    const int nc = (int)((n + 31) / 32);   // blocks of k_combine per right-hand side
    DevBuf<unsigned long long> reo;
    reo.alloc(1);
    V.alloc((size_t)(m + 1) * nrhs * n);
    H.alloc((size_t)nrhs * (m + 1) * m);
    sn.alloc((size_t)nrhs * m);
    cs.alloc((size_t)nrhs * m);
    g.alloc((size_t)nrhs * (m + 1));
    y.alloc((size_t)nrhs * n);
    w.alloc((size_t)nrhs * n);
    hb1.alloc((size_t)nrhs * (m + 1));
    hb2.alloc((size_t)nrhs * (m + 1));
    zs.alloc((size_t)nrhs * m);
    bnorm.alloc(nrhs);
    resid.alloc(nrhs);
    nrm0.alloc(nrhs);
    done.alloc(nrhs);
    kconv.alloc(nrhs);
    active.alloc(nrhs);
    flag.alloc(nrhs);
    part1.alloc((size_t)nrhs * nc);
    part2.alloc((size_t)nrhs * nc);
    if (rd.prec != CBFM_FP64) x32.alloc((size_t)nrhs * n);
    nact.alloc(m + 1);
    // the polled active count lands in a pinned word kept per host thread (one API call at a
    // time per thread), so a solve -- and every inner solve of the inexact CMP -- does no
    // host allocation and no cudaFreeHost
    struct PinnedWord {
        int *p = nullptr;
        ~PinnedWord() {
            if (p) cudaFreeHost(p);
        }
    };
    static thread_local PinnedWord t_nact;
    if (t_nact.p == nullptr) CBFM_CUDA(cudaMallocHost((void **)&t_nact.p, sizeof(int)));
    int *h_nact = t_nact.p;
    CBFM_CUDA(cudaMemsetAsync(y.p, 0, sizeof(z64) * nrhs * n, st));
    CBFM_CUDA(cudaMemsetAsync(H.p, 0, sizeof(z64) * nrhs * (m + 1) * m, st));
    CBFM_CUDA(cudaMemsetAsync(done.p, 0, sizeof(int) * nrhs, st));
    CBFM_CUDA(cudaMemsetAsync(flag.p, 0, sizeof(int) * nrhs, st));
    CBFM_CUDA(cudaMemsetAsync(reo.p, 0, sizeof(unsigned long long), st));
    double pass1 = 0.0, nmatvec = 0.0;   // algorithmic work counters (profiling)
    {
        ProfScope ps_("k_norms", st);
        k_norms<<<nrhs, 256, 0, st>>>(n, nrhs, d_b, bnorm.p);
        launched("k_norms");
    }

    const int hld = m + 1;
    const RotState rot{H.p, sn.p, g.p, cs.p, resid.p, bnorm.p, done.p, flag.p, kconv.p, nact.p, tol};
    // few right-hand sides of moderate order: a cluster each, if all are resident at once (n = 222, one: 12 us an
    // iteration against 45 us of separate launches; at n = 1024 and 1000 steps both are bound by the FP64 pipes, of 16
    // SMs and of all)
    const bool ord = pc != CBFM_PC_CMP;
    const bool cl = n <= GC_NMAX && !ord && nrhs <= gmres_clusters(rd.prec != CBFM_FP64);
    DevBuf<z64> w2, hc;
    DevBuf<double> partc;
    if (cl) {
        w2.alloc((size_t)2 * nrhs * n);
        hc.alloc((size_t)4 * nrhs * hld);
        partc.alloc((size_t)nrhs * 2 * 3 * 16);
    }
    if (ord) set_finish_smem();
    const int CHECK = 4;   // iterations between convergence polls
    std::vector<int> h_iters(nrhs, 0), h_done(nrhs, 0), h_kc(nrhs, 0), h_act(nrhs, 0);
    int total = 0;
    bool first = true;
    while (total < maxit) {
        if (!first) apply_B(rd, pc, y.p, nullptr, w.p, nrhs, nullptr, st);
        {
            ProfScope ps_("k_start", st);
            k_start<<<nrhs, 256, 0, st>>>(n, nrhs, m, d_b, w.p, first ? 0 : 1, V.p, g.p, bnorm.p, resid.p, done.p,
                                          tol, x32.p);
            launched("k_start");
        }
        first = false;
        CBFM_CUDA(cudaMemcpyAsync(h_done.data(), done.p, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, st));
        CBFM_CUDA(cudaStreamSynchronize(st));
        int nrun = 0;
        for (int r = 0; r < nrhs; ++r) {
            h_act[r] = h_done[r] == 1 ? 0 : 1;
            nrun += h_act[r];
        }
        if (nrun == 0) break;
        CBFM_CUDA(cudaMemcpyAsync(active.p, h_act.data(), sizeof(int) * nrhs, cudaMemcpyHostToDevice, st));
        CBFM_CUDA(cudaMemsetAsync(kconv.p, 0, sizeof(int) * nrhs, st));
        CBFM_CUDA(cudaMemsetAsync(nact.p, 0, sizeof(int) * (m + 1), st));
        const int mc = std::min(m, maxit - total);
        int k = 0;
        if (cl) {
            GmresCl P{n, nrhs, m, mc, hld, nullptr, nullptr, V.p, w2.p, hc.p, hc.p + 2 * (int64_t)nrhs * hld, partc.p, reo.p, rot};
            P.rot.flag = P.rot.n_active = nullptr;
            if (rd.prec != CBFM_FP64) P.M32 = pc_op32(rd, pc);
            else P.M64 = pc_op64(rd, pc);
            ProfScope ps_("k_gmres_cl", st);
            launch_gmres_cl(P, rd.prec != CBFM_FP64, st);
            launched("k_gmres_cl");
        }
        for (; !cl && k < mc; ++k) {
            const z64 *vk = V.p + (int64_t)k * nrhs * n;
            apply_B(rd, pc, vk, x32.p, w.p, nrhs, done.p, st);
            const dim3 gd((unsigned)((k + 1 + JB - 1) / JB), nrhs), gu((unsigned)nc, nrhs);
            for (int pass = 0; pass < 2; ++pass) {
                z64 *hb = pass == 0 ? hb1.p : hb2.p;
                {
                    ProfScope ps_("k_dots", st);
                    auto *f = ord ? k_dots<true> : k_dots<false>;
                    f<<<gd, 32 * JB, 0, st>>>(n, nrhs, k, V.p, w.p, hb, hld, done.p, nrm0.p,
                                              pass == 0 ? nullptr : part1.p, nc, flag.p, reo.p);
                    launched("k_dots");
                }
                ProfScope ps_("k_orth_update", st);
                // the second pass on the rows k_dots flagged (a finished row's flag is zero)
                const int *mask = pass == 0 ? done.p : flag.p;
                if (ord) k_orth_ord<<<gu, 128, 0, st>>>(n, nrhs, k, V.p, hb, hld, mask, pass, w.p);
                else
                    k_combine<<<gu, 256, 0, st>>>(n, nrhs, k + 1, nullptr, V.p, hb, hld, mask, pass, -1.0, w.p,
                                                  pass == 0 ? part1.p : part2.p);
                launched("k_orth_update");
            }
            const int last = (k + 1 == mc) ? 1 : 0;
            {
                ProfScope ps_("k_finish", st);
                if (ord)
                    k_finish_ord<<<nrhs, 256, finish_ord_smem(k), st>>>(n, nrhs, k, m, last, hb1.p, hb2.p, hld, rot, w.p,
                                                                        V.p, x32.p);
                else
                    k_finish<<<nrhs, 256, 0, st>>>(n, nrhs, k, m, last, hb1.p, hb2.p, hld, rot, part1.p, part2.p, nc, w.p,
                                                   V.p, x32.p);
                launched("k_finish");
            }
            if ((k + 1) % CHECK == 0 || last) {
                CBFM_CUDA(cudaMemcpyAsync(h_nact, nact.p + k, sizeof(int), cudaMemcpyDeviceToHost, st));
                CBFM_CUDA(cudaStreamSynchronize(st));
                if (*h_nact == 0) {
                    ++k;
                    break;
                }
            }
        }
        CBFM_CUDA(cudaMemcpyAsync(h_kc.data(), kconv.p, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, st));
        CBFM_CUDA(cudaMemcpyAsync(h_done.data(), done.p, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, st));
        CBFM_CUDA(cudaStreamSynchronize(st));
        for (int r = 0; r < nrhs; ++r)
            if (h_act[r]) {
                if (cl) k = std::max(k, h_kc[r]);
                h_iters[r] += h_kc[r];
                pass1 += 0.5 * (double)h_kc[r] * (h_kc[r] + 1);
                nmatvec += h_kc[r] + 1;
            }
        total += k;
        {
            ProfScope ps_("k_backsolve", st);
            k_backsolve<<<nrhs, 128, 0, st>>>(nrhs, m, H.p, g.p, kconv.p, active.p, zs.p);
            launched("k_backsolve");
        }
        {
            ProfScope ps_("k_update_y", st);
            if (ord)
                k_update_y<<<dim3((unsigned)((n + 255) / 256), nrhs), 256, 0, st>>>(n, nrhs, m, V.p, zs.p, kconv.p,
                                                                                    active.p, y.p);
            else
                k_combine<<<dim3((unsigned)nc, nrhs), 256, 0, st>>>(n, nrhs, 0, kconv.p, V.p, zs.p, m, active.p, 1, 1.0, y.p,
                                                                nullptr);
            launched("k_update_y");
        }
        bool all = true;
        for (int r = 0; r < nrhs; ++r) all &= (h_done[r] == 1);
        if (all) break;
        for (int r = 0; r < nrhs; ++r)
            if (h_done[r] == 2) h_done[r] = 0;
        CBFM_CUDA(cudaMemcpyAsync(done.p, h_done.data(), sizeof(int) * nrhs, cudaMemcpyHostToDevice, st));
        CBFM_CUDA(cudaMemsetAsync(H.p, 0, sizeof(z64) * nrhs * (m + 1) * m, st));
    }
    // x = P y
    if (pc == CBFM_PC_CMP) apply_rows(n, rd.Ginv.p, nullptr, y.p, nullptr, d_x, nrhs, nullptr, false, st);
    else if (pc == CBFM_PC_TDIAG) tdiag_recover(rd, y.p, d_x, nrhs, st);
    else if (pc == CBFM_PC_CMP_INEXACT) cmp_inner_apply(rd, y.p, d_x, nrhs, st);
    else CBFM_CUDA(cudaMemcpyAsync(d_x, y.p, sizeof(z64) * nrhs * n, cudaMemcpyDeviceToDevice, st));
    GmresOut out;
    out.iters = h_iters;
    out.resid.resize(nrhs);
    CBFM_CUDA(cudaMemcpyAsync(out.resid.data(), resid.p, sizeof(double) * nrhs, cudaMemcpyDeviceToHost, st));
    CBFM_CUDA(cudaMemcpyAsync(h_done.data(), done.p, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, st));
    CBFM_CUDA(cudaStreamSynchronize(st));
    for (int r = 0; r < nrhs; ++r)
        if (h_done[r] != 1) out.iters[r] = -std::abs(out.iters[r]) - 1;   // marks non-convergence
    if (g_prof.load()) {
        unsigned long long p2 = 0;
        CBFM_CUDA(cudaMemcpy(&p2, reo.p, sizeof(p2), cudaMemcpyDeviceToHost));
        const double cb = sizeof(z64);
        // dot products and updates: 8 flops per complex multiply-add, one basis element read each
        prof_add_work("k_dots", 8.0 * n * (pass1 + p2), cb * n * (pass1 + p2));
        prof_add_work("k_orth_update", 8.0 * n * (pass1 + p2), cb * n * (pass1 + p2));
        const double eb = rd.prec != CBFM_FP64 ? sizeof(c32) : sizeof(z64);
        prof_add_work("k_matvec", 8.0 * n * n * (nmatvec + (pc == CBFM_PC_CMP ? nrhs : 0)), eb * n * n * (nmatvec + 1.0));
    }
    return out;
}

}  // namespace cbfm
