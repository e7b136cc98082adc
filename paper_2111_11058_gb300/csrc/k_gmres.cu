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
#include <vector>

#include "internal.cuh"

namespace cbfm {

namespace {

constexpr int JB = 8;          // basis vectors per block in k_dots
constexpr double DGKS_ETA2 = 0.5;   // (1 / sqrt 2)^2

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
        if (warp == 0) {
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
                re[u] = fma(a.im, b.im, fma(a.re, b.re, re[u]));   // written as a sum it is a product, an FMA and an add
                im[u] = fma(-a.im, b.re, fma(a.re, b.im, im[u]));
            }
        }
        for (; i < n; i += 32) {
            const z64 a = v[i], b = x[i];
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
__global__ void __launch_bounds__(256) k_finish(int64_t n, int nrhs, int k, int m, int last,
                                                const z64 *__restrict__ h1, const z64 *__restrict__ h2,
                                                int *__restrict__ flag, int hld, z64 *__restrict__ H,
                                                double *__restrict__ cs, z64 *__restrict__ sn, z64 *__restrict__ g,
                                                const double *__restrict__ bnorm, double tol, int *__restrict__ done,
                                                int *__restrict__ kconv, double *__restrict__ resid,
                                                int *__restrict__ n_active, const double *__restrict__ part1,
                                                const double *__restrict__ part2, int nc, const z64 *__restrict__ w,
                                                z64 *__restrict__ V, c32 *__restrict__ x32) {
    const int r = blockIdx.x;
    if (done[r]) return;
    __shared__ z64 col[1024];
    __shared__ z64 s_A[4], s_B[4];
    __shared__ double s_nrm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool re = flag[r] != 0;
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
    const double *cr = cs + (int64_t)r * m;
    const z64 *sr = sn + (int64_t)r * m;
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
    z64 *Hr = H + (int64_t)r * (m + 1) * m;
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
        z64 *gr = g + (int64_t)r * (m + 1);
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
        cs[(int64_t)r * m + k] = cc;
        sn[(int64_t)r * m + k] = ss;
        Hr[(int64_t)k * m + k] = cc * a + ss * nb;
        z64 gk = gr[k];
        gr[k] = cc * gk;
        gr[k + 1] = -(conj(ss) * gk);
        double res = sqrt(norm2(gr[k + 1])) / bnorm[r];
        resid[r] = res;
        if (res <= tol || nb == 0.0) {
            kconv[r] = k + 1;
            done[r] = 1;
            flag[r] = 0;
        } else if (last) {
            kconv[r] = k + 1;
            done[r] = 2;
            flag[r] = 0;
        } else {
            atomicAdd(n_active + k, 1);
        }
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
                       const int *done, cudaStream_t st) {
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
    apply_rows(rd.n, mixed ? nullptr : pc_op64(rd, pc), mixed ? pc_op32(rd, pc) : nullptr, in, in32, out, nrhs, done, st);
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
        for (; k < mc; ++k) {
            const z64 *vk = V.p + (int64_t)k * nrhs * n;
            apply_B(rd, pc, vk, x32.p, w.p, nrhs, done.p, st);
            const dim3 gd((unsigned)((k + 1 + JB - 1) / JB), nrhs), gu((unsigned)nc, nrhs);
            for (int pass = 0; pass < 2; ++pass) {
                z64 *hb = pass == 0 ? hb1.p : hb2.p;
                {
                    ProfScope ps_("k_dots", st);
                    k_dots<<<gd, 32 * JB, 0, st>>>(n, nrhs, k, V.p, w.p, hb, hld, done.p, nrm0.p,
                                                   pass == 0 ? nullptr : part1.p, nc, flag.p, reo.p);
                    launched("k_dots");
                }
                ProfScope ps_("k_orth_update", st);
                // the second pass on the rows k_dots flagged (a finished row's flag is zero)
                k_combine<<<gu, 256, 0, st>>>(n, nrhs, k + 1, nullptr, V.p, hb, hld, pass == 0 ? done.p : flag.p, pass,
                                              -1.0, w.p, pass == 0 ? part1.p : part2.p);
                launched("k_orth_update");
            }
            const int last = (k + 1 == mc) ? 1 : 0;
            {
                ProfScope ps_("k_finish", st);
                k_finish<<<nrhs, 256, 0, st>>>(n, nrhs, k, m, last, hb1.p, hb2.p, flag.p, hld, H.p, cs.p, sn.p, g.p,
                                               bnorm.p, tol, done.p, kconv.p, resid.p, nact.p, part1.p, part2.p, nc, w.p,
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
        total += k;
        CBFM_CUDA(cudaMemcpyAsync(h_kc.data(), kconv.p, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, st));
        CBFM_CUDA(cudaMemcpyAsync(h_done.data(), done.p, sizeof(int) * nrhs, cudaMemcpyDeviceToHost, st));
        CBFM_CUDA(cudaStreamSynchronize(st));
        for (int r = 0; r < nrhs; ++r)
            if (h_act[r]) {
                h_iters[r] += h_kc[r];
                pass1 += 0.5 * (double)h_kc[r] * (h_kc[r] + 1);
                nmatvec += h_kc[r] + 1;
            }
        {
            ProfScope ps_("k_backsolve", st);
            k_backsolve<<<nrhs, 128, 0, st>>>(nrhs, m, H.p, g.p, kconv.p, active.p, zs.p);
            launched("k_backsolve");
        }
        {
            ProfScope ps_("k_update_y", st);
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
    if (pc == CBFM_PC_CMP) apply_rows(n, rd.Ginv.p, nullptr, y.p, nullptr, d_x, nrhs, nullptr, st);
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
