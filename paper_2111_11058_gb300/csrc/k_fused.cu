// k_fused.cu -- Galerkin assembly fused with the projection onto the CBFs
// (paper Eq. (CBFM_outer) with Eqs. (CBF_matrix_JM), (CBF_matrix_MJ); Z from
// Eqs. (K), (T), (Z) of Sec. II-B), mixed-precision path.  No local-block or
// RWG matrix exists in device memory: each cell pair (m, n) is one work item of
// a persistent kernel that forms the four blocks of A,
//   A_mn = [[C^J_m^H Ks C^M_n, C^J_m^H Ta C^J_n], [C^M_m^H Tb C^M_n, C^M_m^H Ks C^J_n]],
// from the triangles that support the cells' RWG functions -- and, since Z_nm is
// the transpose of Z_mn operator by operator, A_nm from the same entries (m <= n).
//
// Work item (m, n).  T_m = triangles carrying an RWG of cell m (test side), T_n
// likewise (trial side).  One stage per trial triangle s:
//   1. the warps evaluate the pairs (t, s), t in T_m, a test triangle per lane, 32
//      consecutive pairs of the item's list (t fastest) per task: far pairs by the
//      FP32 barycentric quadrature (far_bary.cuh), near pairs from the FP64 blocks
//      of the near-pair stage;
//   2. each lane splits its entries into TF32 hi/lo and stores them as the B operand
//      of the stage, row = cell-m RWG i, columns along K = (side of i that t is,
//      edge b of s, re/im).  An RWG has one triangle on each side and s its own
//      columns, so every element has exactly one writer: no atomic adds, no zeroing,
//      no pass over the tile, and the sums over the sides and the edges are K sums;
//   3. the warp that completes the stage has one thread issue tcgen05.mma kind::tf32
//      (hi*hi + hi*lo + lo*hi),
//        Y^T[w][i] += sum_K C_n[K][w] Z_op[i][K],
//      with the CBF coefficients of s's edges as the A operand (M = 128 lanes: 2 per
//      CBF, real and imaginary rows of the expanded complex product, and 2 more of
//      conj(C_n) for A_nm); Y^T accumulates in tensor memory over the item.  Lanes
//      [0, 2L) and [2L, 4L) of the Ks accumulator hold Y for C^M and C^J; the Ta and Tb
//      products share a second accumulator (Ta on lanes [0, 2L) with C^J, Tb on
//      [2L, 4L) with C^M; each operand is zero on the other's lanes); lanes [4L, 8L)
//      repeat this for the conjugates.
// After the last stage all warps read Y^T from tensor memory and form C_m^H Y (A_mn)
// and Y^T C_m (A_nm) on the CUDA cores (FP32), writing the blocks of A directly --
// every entry of A has exactly one writer, and the sums have a fixed order.
//
// Tasks go round robin to the warps over the CTA's whole sequence of items, so a warp
// never waits for another between tasks: it computes into registers and meets the
// others only at the store, where the stage two before its own must have left the
// operand buffer.  Cells with more CBFs than 16 (8 L lanes) or tiles that do not fit
// beside the doubled operand run over all ordered cell pairs instead.
//
// Bound: the FP32 quadrature's latency and instruction fetch (one CTA of 12 warps
// per SM by registers, issue active 49 %).  The spheroid of 32 400 unknowns (96
// cells, L = 8): 31 ms, against 77 ms with ordered cell pairs, the general
// quadrature and shared-memory atomic adds into the tile.  Measured and not taken:
// a pair on two lanes, one medium each (16 warps of 128 registers), 34 ms, and 20
// warps of 96, 38 ms; both orbits unrolled, 33 ms.
//
// Entries: barycentric far pairs and the near pairs' short closed forms, whatever the CBFs' spread (SPREAD_ASM rules
// the unfused form only).  17 generated CBF sets (spread 40 to 1.9e3) against 64 bits: A 0.57 times, the RCS 0.87 times
// and the currents 1.00 times the errors of the earlier kernel with the general quadrature; A 0.4 to 0.8 times those
// of the unfused form.
//
// Triangle pairs whose triangles carry RWGs of several cells are evaluated once
// per cell pair they feed (about 1.15 x per side on the RCB cells used here).
//
// Every mbarrier wait is bounded; on expiry the kernel records an error code,
// stops at the next task, frees its tensor memory and returns.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <numeric>
#include <vector>

#include "far_bary.cuh"
#include "tc_ptx.cuh"

namespace cbfm {

namespace {

using namespace fm;
using namespace tc;

constexpr int FU_THREADS = 384;
constexpr int FU_WARPS = FU_THREADS / 32;
constexpr int FU_PARTS = FU_WARPS / 4;   // warps per lane quarter of tensor memory
constexpr int FU_LMAX = 32;      // largest L_m (4 L lanes of the accumulator <= 128)
constexpr int FU_LSYM = 16;      // largest L_m with the conjugate lanes (8 L <= 128)
constexpr int FU_NMAX = 256;     // largest N_m (MMA N)
constexpr int FU_RING = 8;       // cell-pair items held in shared memory at once
constexpr int FU_AHEAD = 4;      // items fetched ahead of the one whose first stage is issued
constexpr uint32_t FU_NONE16 = 0xffffu;

struct FusedJob {
    const double *rec64;
    const int32_t *vid;
    const float *trial;          // FuTrial of every list entry
    const float *farT;           // test-side far records, field-major over the list entries (stride ntl)
    const int32_t *vidT;
    int64_t ntl;
    const int4 *tl;
    const int32_t *tl_off, *cell_off;
    const int32_t *near_row;
    const int2 *near_ent;
    const c32 *near_val;
    const float *aimg;           // per list entry: its CBF operand, 2 planes x 3 operators x rows x 8 floats,
    const int64_t *aimg_off;     //   swizzled as in shared memory; cell c's entries from float offset aimg_off[c]
    const c32 *CM32, *CJ32;      // complex64 CBF blocks (test side of the epilogue)
    const int64_t *boff, *coff;
    const int32_t *L;
    c32 *A;
    int64_t nh, n;
    MediaT<float> md;
    double alpha;
};

// The tensor cores round their FP32 sums toward zero at every step, two K steps of
// three products per trial triangle.  Where tensor memory has room for a second set
// of accumulators the two small products (hi*lo, lo*hi) go there, and a pair's trial
// triangles are taken in two segments whose parts of A are added with rounding;
// otherwise in four.  Relative errors of A against FP64, one segment and one set:
// 1.15e-5 on a spheroid of 7200 unknowns in 24 cells, so 1.9e-6 (chunks of eight
// summed columns in one set, six steps per chunk: 3.4e-6); in 96 cells 6.0e-7 (9.1e-7).
__host__ __device__ inline int fu_segments(int nacc) { return nacc == 2 ? 2 : 4; }

// One segment of a cell-pair work item (shared memory); job < 0: no more work.
struct FuItem {
    int job, m, n, t0, nT, s0, nS, Lm, Ln, Nm, Np, rows;
    int e0;      // first trial entry within the cell's list
    int first;   // first segment of its cell pair
    int left, lseg;   // trial entries and segments of the cell pair after this one
    FusedJob J;
};

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// A warp's trial triangle: far record, vertex ids, triangle.
struct FuTrial {
    float f[FB_REC];
    int32_t vid[3], tri;
};

// The 27 entries of test list entry ti (triangle t) with trial triangle S.
// Returns false if a near pair is missing from the near list.
__device__ __forceinline__ bool fused_pair(const FusedJob &J, int64_t ti, int t, const FuTrial &S, c32 *v) {
    const float *rt = J.farT + ti;
    const int64_t L = J.ntl;
    const int32_t vt[3] = {J.vidT[ti], J.vidT[ti + L], J.vidT[ti + 2 * L]};
    float rec[FB_REC];
#pragma unroll
    for (int f = 0; f <= FB_H; ++f) rec[f] = rt[f * L];
    float dc[3];
    if (is_near_b<float>(rec, S.f, J.rec64 + (int64_t)t * TRI_REC, J.rec64 + (int64_t)S.tri * TRI_REC, vt, S.vid,
                         J.alpha, dc)) {
        int code = -1;
        for (int e = J.near_row[t], e1 = J.near_row[t + 1]; e < e1; ++e) {
            const int2 en = J.near_ent[e];
            if (en.x == S.tri) {
                code = en.y;
                break;
            }
        }
        const c32 *b = J.near_val + (int64_t)max(code >> 1, 0) * NCOMP;
        const int sa = code & 1 ? 1 : 3, sb = code & 1 ? 3 : 1;   // the block of (s, t) is the transpose
#pragma unroll
        for (int op = 0; op < 3; ++op)
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int bb = 0; bb < 3; ++bb) v[op * 9 + 3 * a + bb] = b[op * 9 + sa * a + sb * bb];
        return code >= 0;
    }
    far_bary<float, true>(rec + FB_P, rec + FB_C, S.f + FB_P, S.f + FB_C, dc, J.md, v);
    return true;
}

// Shared-memory plan (bytes from the 1024-aligned base):
//   A images (the CBF operand), two buffers: hi then lo plane, 3 operators x RA rows x 32 B (one K step);
//   the RWG tile (B operand), two buffers: hi then lo plane, 3 operators x NP rows x 64 B (two K steps, one per
//   side: real parts of edges 0, 1, 2 of s, zero, imaginary parts, zero);
//   the warps' trial triangles.
// laid out [A0 | A1 | Z0 | Z1 | trial].  An A operand is read 128 rows deep from its
// base; rows past its image land in the next region (lanes that are not used).
// ls (at most 64 rows): Ta and Tb take the lanes 64 .. 127 of the accumulator Ks
// uses, so that a set of accumulators needs NP columns and two sets always fit
// tensor memory; a plane's regions are Ks, zeros, Ta, zeros, Tb (RA = 64 rows each),
// Ks read from its own and Ta, Tb from the zeros before them (adding zeros is exact).
// acol: columns of an accumulator set, nacc: sets.
struct FuPlan {
    int RA, NP, sym, ls, nacc;
    uint32_t a_op, z_op, z_base, t_base, total, acol;
};

__device__ __forceinline__ uint32_t fu_a(const FuPlan &P, int b, int plane, int op) {   // image of an operator
    return P.ls ? (uint32_t)(b * 10 + plane * 5 + 2 * op) * P.a_op : (uint32_t)(b * 6 + plane * 3 + op) * P.a_op;
}
__device__ __forceinline__ uint32_t fu_z(const FuPlan &P, int b, int plane, int op) {
    return P.z_base + (uint32_t)(b * 6 + plane * 3 + op) * P.z_op;
}

// Stores a pair's entries into the tile at shared-memory address z (hi planes; the
// lo planes lie 3 z_op further): te.y, te.z hold the rows of the test triangle's
// edges and, from bit 16 of te.z, which side of each RWG it is.  Eight lanes with
// consecutive rows fill distinct 16-byte slots (swizzle), as the list order mostly gives.
__device__ __forceinline__ void fused_store(uint32_t z, uint32_t z_op, int4 te, const c32 *v) {
    const uint32_t rows[3] = {(uint32_t)te.y & 0xffffu, ((uint32_t)te.y >> 16) & 0xffffu, (uint32_t)te.z & 0xffffu};
    auto put = [&](uint32_t o, float x0, float x1, float x2) {
        float h[3], l[3];
        split(x0, h[0], l[0]);
        split(x1, h[1], l[1]);
        split(x2, h[2], l[2]);
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(o), "f"(h[0]), "f"(h[1]), "f"(h[2]), "f"(0.f)
                     : "memory");
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(o + 3 * z_op), "f"(l[0]), "f"(l[1]), "f"(l[2]),
                     "f"(0.f)
                     : "memory");
    };
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const uint32_t r = rows[a];
        if (r == FU_NONE16) continue;
        const uint32_t side = ((uint32_t)te.z >> (16 + a)) & 1u;
        const uint32_t o0 = z + swz64((int)r, (int)(8u * side)), o1 = z + swz64((int)r, (int)(8u * side + 4u));
#pragma unroll
        for (int op = 0; op < 3; ++op) {
            const c32 *x = v + 9 * op + 3 * a;
            put(o0 + op * z_op, x[0].re, x[1].re, x[2].re);
            put(o1 + op * z_op, x[0].im, x[1].im, x[2].im);
        }
    }
}

// One thread fetches the CTA's item `seq` into its ring slot (job < 0: the work is exhausted): the next segment of
// the cell pair of item seq - 1, or the first one of a new pair.
__device__ void fu_fetch(const FusedJob *jobs, const int4 *items, int nitems, unsigned *counter, FuItem *ring, int seq,
                         const FuPlan &P) {
    FuItem &o = ring[seq % FU_RING];
    const FuItem &p = ring[(seq + FU_RING - 1) % FU_RING];
    if (seq > 0 && p.job >= 0 && p.left > 0) {
        o = p;
        o.first = 0;
        o.e0 = p.e0 + p.nS;
        o.s0 = p.s0 + p.nS;
        o.nS = (p.left + p.lseg - 1) / p.lseg;
        o.left = p.left - o.nS;
        o.lseg = p.lseg - 1;
        return;
    }
    const int it = (int)atomicAdd(counter, 1u);
    if (it >= nitems) {
        o.job = -1;
        return;
    }
    const int4 im = __ldg(items + it);
    o.J = jobs[im.x];
    const FusedJob &J = o.J;
    o.job = im.x;
    o.m = im.y;
    o.n = im.z;
    o.t0 = J.tl_off[im.y];
    o.nT = J.tl_off[im.y + 1] - o.t0;
    o.s0 = J.tl_off[im.z];
    const int n = J.tl_off[im.z + 1] - o.s0, ns = fu_segments(P.nacc);
    o.nS = (n + ns - 1) / ns;
    o.left = n - o.nS;
    o.lseg = ns - 1;
    o.e0 = 0;
    o.first = 1;
    o.Lm = J.L[im.y];
    o.Ln = J.L[im.z];
    o.Nm = J.cell_off[im.y + 1] - J.cell_off[im.y];
    o.Np = (o.Nm + 15) & ~15;
    o.rows = (P.sym ? 8 : 4) * o.Ln;
}

// Starts the asynchronous copies of the CBF operand of trial entry si of an item
// into buffer b (one thread; completion on `bar`).
__device__ __forceinline__ void fu_load_a(const FuPlan &P, uint32_t sbase, int b, const FuItem &it,
                                          int si, uint64_t *bar, int *issued) {
    const FusedJob &J = it.J;
    const uint32_t seg = (uint32_t)it.rows * 32u;   // bytes of one operator's rows in one plane
    mbar_expect_tx(bar, 6 * seg);
    ++*issued;
    const float *src = J.aimg + J.aimg_off[it.n] + (int64_t)(it.e0 + si) * (6 * (seg / 4));
    for (int q = 0; q < 6; ++q)
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                sbase + fu_a(P, b, q / 3, q % 3)),
            "l"(src + (int64_t)q * (seg / 4)), "r"(seg), "r"(smem_u32(bar))
            : "memory");
}

// The blocks of A of item `pip`, whose last MMAs are done.  Warp w reads tensor-memory lanes 32 (w mod 4) ... + 31; the FU_PARTS
// warps of a lane quarter share the CBFs l of cell m.  Lane r holds, for every RWG
// i of cell m (column i of its accumulator), the real (r even) or imaginary (r odd)
// part of Y[i][w], w = (r mod 2 L_n) / 2: of C^M_n (lanes [0, 2 L)) and C^J_n
// ([2 L, 4 L)) in the Ks accumulator, C^J_n with Ta and C^M_n with Tb in the other;
// lanes [4 L, 8 L) the same of the conjugates (ls: lanes 64 on are the other's).  The first half gives
// sum_i conj(C_m[i][l]) Y[i][w] of A_mn, the second sum_i Y[i][w] C_m[i][l] of A_nm.
// Not inlined: it runs once per item between a
// task's quadrature and its stores, and its registers should be spilled only then.
constexpr int FU_LB = 3;   // CBFs of cell m per pass over the accumulator
__device__ __noinline__ void fu_epilogue(const FuItem *pip, uint32_t tmem, uint32_t set2, int ls, int warp, int lane) {
    const FuItem &pi = *pip;
    tc_fence_after();
    const FusedJob &J = pi.J;
    const int Ln = pi.Ln, Lm = pi.Lm, Nm = pi.Nm, Np = pi.Np;
    const int quarter = warp & 3;
    const int lpart = (Lm + FU_PARTS - 1) / FU_PARTS, l0 = (warp >> 2) * lpart, l1 = min(l0 + lpart, Lm);
    if (32 * (ls ? quarter & 1 : quarter) < pi.rows) {
        const int r = 32 * (ls ? quarter & 1 : quarter) + lane;
        const bool cj = r >= 4 * Ln;
        const bool valid = r < pi.rows && !(cj && pi.m == pi.n);
        const int rr = cj ? r - 4 * Ln : r;
        const bool upper = rr >= 2 * Ln;
        const int w = (rr - (upper ? 2 * Ln : 0)) >> 1, ri = r & 1;
        const int64_t cm = J.coff[pi.m], cn = J.coff[pi.n];
#pragma unroll 1
        for (int g = ls ? quarter >> 1 : 0; g < (ls ? (quarter >> 1) + 1 : 2); ++g) {
            const bool eq = (g == 0) == upper;
#pragma unroll 1
            for (int lb = l0; lb < l1; lb += FU_LB) {
                PF acc[FU_LB];   // sums of Re c y and Im c y
#pragma unroll
                for (int l = 0; l < FU_LB; ++l) acc[l] = pmk(0.f, 0.f);
                const int nl = l1 - lb;
                // lanes 0-15 hold 16 rows of C^J, lanes 16-31 of C^M (the next 16 in flight), read by shuffles
                const c32 *Cl = (lane < 16 ? J.CJ32 : J.CM32) + J.boff[pi.m] + lb;
                auto fetch = [&](int i0, c32 *c) {
                    const int i = i0 + (lane & 15);
#pragma unroll
                    for (int l = 0; l < FU_LB; ++l) c[l] = i < Nm && l < nl ? Cl[(int64_t)i * Lm + l] : c32(0.f, 0.f);
                };
                c32 cn_[FU_LB];
                fetch(0, cn_);
#pragma unroll 1
                for (int i0 = 0; i0 < Nm; i0 += 16) {
                    c32 cc[FU_LB];
#pragma unroll
                    for (int l = 0; l < FU_LB; ++l) cc[l] = cn_[l];
                    fetch(i0 + 16, cn_);
                    uint32_t y[16];
                    const uint32_t ta = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)((ls ? 0 : g * Np) + i0);
                    tmem_ld16(ta, y);
                    if (set2) {   // the small products
                        uint32_t z[16];
                        tmem_ld16(ta + set2, z);
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            y[q] = __float_as_uint(__uint_as_float(y[q]) + __uint_as_float(z[q]));
                    }
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        // rows past N_m: zero coefficients (their columns hold sums of finite tile entries)
                        const float yv = __uint_as_float(y[q]);
                        const PF yy = pmk(yv, yv);
#pragma unroll
                        for (int l = 0; l < FU_LB; ++l) {
                            const float cr = __shfl_sync(0xffffffffu, cc[l].re, q + (upper ? 16 : 0));
                            const float ci = __shfl_sync(0xffffffffu, cc[l].im, q + (upper ? 16 : 0));
                            acc[l] = pfma(pmk(cr, ci), yy, acc[l]);
                        }
                    }
                }
#pragma unroll
                for (int l = 0; l < FU_LB; ++l) {
                    // even lanes hold c y_re, odd ones c y_im; conj(c) for A_mn
                    const float p = plo(acc[l]), q = cj ? phi(acc[l]) : -phi(acc[l]);
                    const float p1 = __shfl_xor_sync(0xffffffffu, p, 1), q1 = __shfl_xor_sync(0xffffffffu, q, 1);
                    if (valid && ri == 0 && l < nl) {
                        const int64_t am = cm + lb + l, an = cn + w;
                        // A_mn: rows J-tested (lower) / M-tested (upper); A_nm: columns M (upper) / J (lower)
                        const int64_t row = cj ? (eq ? 0 : J.nh) + an : (upper ? J.nh : 0) + am;
                        const int64_t col = cj ? (upper ? 0 : J.nh) + am : (eq ? J.nh : 0) + an;
                        c32 *dst = J.A + row * J.n + col;
                        c32 a(p - q1, q + p1);
                        if (!pi.first) a += *dst;   // this thread wrote it for the item's segment before
                        *dst = a;
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncwarp();
}

__global__ void __launch_bounds__(FU_THREADS, 1)
    k_fused(const FusedJob *__restrict__ jobs, const int4 *__restrict__ items, int nitems,
            unsigned int *__restrict__ counter, int *__restrict__ err, const FuPlan plan, uint32_t tmem_cols) {
    extern __shared__ uint8_t fu_raw[];
    __shared__ uint64_t mma_bar[2], aimg_bar[2], epi_bar;
    __shared__ unsigned done_ctr[2];           // pairs stored into each operand buffer since the launch
    __shared__ int a_issued[2], a_waited[2];   // operand copies started / waited for, per buffer
    __shared__ FuItem s_it[FU_RING];
    __shared__ int s_nseq, s_issued, s_abort;  // items fetched; stages issued to the tensor cores; a wait expired
    __shared__ uint32_t s_tmem;
    uint8_t *sm = (uint8_t *)(((uintptr_t)fu_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(sm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&mma_bar[b], 1);
            mbar_init(&aimg_bar[b], 1);
            done_ctr[b] = 0;
            a_issued[b] = a_waited[b] = 0;
        }
        mbar_init(&epi_bar, FU_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        for (int q = 0; q < FU_AHEAD; ++q) fu_fetch(jobs, items, nitems, counter, s_it, q, plan);
        s_nseq = FU_AHEAD;
        s_issued = 0;
    }
    // the tiles' zero columns and the zero rows of ls (and everything else of both operands) once
    for (uint32_t o = (uint32_t)tid * 16u; o < plan.t_base; o += FU_THREADS * 16u)
        *reinterpret_cast<float4 *>(sm + o) = make_float4(0.f, 0.f, 0.f, 0.f);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 32 && s_it[0].job >= 0)
        fu_load_a(plan, sbase, 0, s_it[0], 0, &aimg_bar[0], &a_issued[0]);   // stage k + 1's: service of stage k
    const uint32_t tmem = s_tmem;
    FuTrial *trial = reinterpret_cast<FuTrial *>(sm + plan.t_base) + 2 * warp;

    int seq = 0, epi = 0;      // item of this warp's next task; items whose epilogue it has done
    int kbase = 0;             // stage number of the item's first stage
    unsigned base[2] = {0, 0}; // pairs of the items before, per operand buffer
    int pos = warp;            // next task within the item
    bool ok = true;
    // Waits (bounded) for a shared counter to pass x; whole warp.
    auto passed = [&](volatile int *ctr, int x) {
        int good = 1;
        if (lane == 0) {
            const uint64_t t0 = gtimer();
            while (*ctr <= x) {
                if (*(volatile int *)&s_abort || gtimer() - t0 > TC_WAIT_NS) {
                    good = 0;
                    break;
                }
            }
            __threadfence_block();
        }
        return __shfl_sync(0xffffffffu, good, 0) != 0;
    };
    // Stage k's MMAs are done: stage k + 1 has been issued (after waiting for them), or k is the last one issued and
    // its barrier phase is over.  The barrier alone would not tell: it distinguishes only neighbouring phases, and
    // a warp can be several stages ahead of or behind the issue.
    auto ready = [&](int k) {
        const int n = *(volatile int *)&s_issued;
        return n > k + 1 || (n == k + 1 && mbar_try(&mma_bar[k & 1], (k >> 1) & 1));
    };
    auto stage_done = [&](int k) {   // waits (bounded) for it; whole warp
        int good = 1;
        if (lane == 0) {
            const uint64_t t0 = gtimer();
            while (!ready(k)) {
                if (*(volatile int *)&s_abort || gtimer() - t0 > TC_WAIT_NS) {
                    good = 0;
                    break;
                }
            }
            __threadfence_block();
        }
        return __shfl_sync(0xffffffffu, good, 0) != 0;
    };
    // the epilogues of the items before `seq` that this warp still owes
    auto settle = [&]() {
        while (ok && epi < seq) {
            int klast = kbase - 1;   // last stage of item epi
            for (int q = seq - 1; q > epi; --q) klast -= s_it[q % FU_RING].nS;
            ok = stage_done(klast);
            if (ok) fu_epilogue(&s_it[epi % FU_RING], tmem, plan.nacc == 2 ? plan.acol : 0u, plan.ls, warp, lane);
            if (lane == 0) mbar_arrive(&epi_bar);
            ++epi;
        }
        if (!ok) {
            atomicExch(err, 6);
            *(volatile int *)&s_abort = 1;
        }
    };
    while (ok) {
        if (!passed(&s_nseq, seq)) {
            atomicExch(err, 5);
            *(volatile int *)&s_abort = 1;
        }
        if (__any_sync(0xffffffffu, *(volatile int *)&s_abort)) break;
        const FuItem &it = s_it[seq % FU_RING];
        const bool end = it.job < 0;
        const int nT = it.nT, nS = it.nS;
        const int ntask = end ? 0 : nT >= 32 ? (nT * nS + 31) >> 5 : nS;
        // Others wait for this warp's epilogues (an item's first MMAs need those of the item before), so it does not
        // run further ahead than the items that are fetched without it.
        if (end || (pos >= ntask && seq - epi >= FU_AHEAD - 1)) {
            settle();
            if (end) break;
            if (!ok) continue;
        }
        if (pos >= ntask) {
            const int n0 = (nS + ((kbase & 1) ^ 1)) >> 1;   // stages of the item in buffer 0
            base[0] += (unsigned)(nT * n0);
            base[1] += (unsigned)(nT * (nS - n0));
            pos -= ntask;
            kbase += nS;
            ++seq;
            continue;
        }
        const FusedJob &J = it.J;
        // ---- this task's pairs: (ti, s_first + sl), one per lane
        int s_first, ti, sl = 0;
        bool valid;
        if (nT >= 32) {
            s_first = (32 * pos) / nT;
            ti = 32 * pos - s_first * nT + lane;
            if (ti >= nT) {
                ti -= nT;
                sl = 1;
            }
            valid = s_first + sl < nS;
        } else {
            s_first = pos;
            ti = lane;
            valid = ti < nT;
        }
        const int nst = __any_sync(0xffffffffu, valid && sl == 1) ? 2 : 1;   // stages the task feeds
        constexpr int TW = sizeof(FuTrial) / 4;
        if (lane < TW)
            for (int h = 0; h < nst; ++h)
                reinterpret_cast<float *>(trial + h)[lane] = J.trial[(int64_t)(it.s0 + s_first + h) * TW + lane];
        __syncwarp();
        const int64_t te_i = it.t0 + ti;
        c32 v[NCOMP];
        int4 te = make_int4(0, -1, -1, 0);
        if (valid) {
            te = J.tl[te_i];
            if (!fused_pair(J, te_i, te.x, trial[sl], v)) atomicExch(err, 7);
        }
        __syncwarp();
        // ---- epilogues of the items before, now that this warp holds a task of a later one
        settle();
        if (!ok) break;
#pragma unroll 1
        for (int h = 0; h < nst && ok; ++h) {
            const int si = s_first + h, k = kbase + si, b = k & 1;
            // the operand buffer: stage k - 2's MMAs must have read it
            if (k >= 2 && !stage_done(k - 2)) {
                atomicExch(err, 9);
                *(volatile int *)&s_abort = 1;
                ok = false;
                break;
            }
            const bool mine = valid && sl == h;
            if (mine) fused_store(sbase + fu_z(plan, b, 0, 0), plan.z_op, te, v);
            fence_proxy_async_smem();   // generic-proxy writes -> tensor-core reads
            __syncwarp();
            const unsigned cnt = __popc(__ballot_sync(0xffffffffu, mine));
            // pairs in buffer b once stage k is complete
            const unsigned full = base[b] + (unsigned)(nT * (si / 2 + 1));
            int last = 0;
            if (lane == 0) {
                __threadfence_block();
                last = atomicAdd(&done_ctr[b], cnt) + cnt == full;
                __threadfence_block();
            }
            // ---- service of stage k by the warp that completed it
            if (last) {
                // one MMA issue at a time, in order: stage k - 1's must be done (it also frees A[b ^ 1])
                if (k >= 1 && !mbar_wait(&mma_bar[b ^ 1], ((k - 1) >> 1) & 1)) ok = false;
                if (si == 0) {
                    const int ns = seq + FU_AHEAD;
                    fu_fetch(jobs, items, nitems, counter, s_it, ns, plan);
                    __threadfence_block();
                    *(volatile int *)&s_nseq = ns + 1;
                }
                if (ok) {
                    if (si + 1 < nS) fu_load_a(plan, sbase, b ^ 1, it, si + 1, &aimg_bar[b ^ 1], &a_issued[b ^ 1]);
                    else if (s_it[(seq + 1) % FU_RING].job >= 0)
                        fu_load_a(plan, sbase, b ^ 1, s_it[(seq + 1) % FU_RING], 0, &aimg_bar[b ^ 1],
                                  &a_issued[b ^ 1]);
                }
                // an item's first MMAs overwrite the accumulators: the previous item's epilogue must be done
                if (ok && si == 0 && seq > 0) ok = mbar_wait(&epi_bar, (seq - 1) & 1);
                if (ok && mbar_wait(&aimg_bar[b], (k >> 1) & 1)) ++a_waited[b];   // the stage's CBF operand has landed
                else ok = false;
                if (!ok) {
                    atomicExch(err, 8);
                    *(volatile int *)&s_abort = 1;
                } else {
                    tc_fence_after();
                    const uint32_t idesc = idesc_tf32(it.Np);
#pragma unroll 1
                    for (int op = 0; op < 3; ++op) {
                        const uint32_t d = tmem + (op == 0 || plan.ls ? 0u : (uint32_t)it.Np);
                        const uint32_t ds = d + (plan.nacc == 2 ? plan.acol : 0u);   // the small products
                        const uint32_t up = op > 0 && plan.ls ? plan.a_op : 0u;   // from the zeros before the image
                        const uint64_t a_h = sdesc32(sbase + fu_a(plan, b, 0, op) - up);
                        const uint64_t a_l = sdesc32(sbase + fu_a(plan, b, 1, op) - up);
                        const uint32_t b_h = sbase + fu_z(plan, b, 0, op), b_l = sbase + fu_z(plan, b, 1, op);
                        const uint32_t fresh = si == 0 && op < (plan.ls ? 1 : 2);
#pragma unroll
                        for (int side = 0; side < 2; ++side) {
                            const uint32_t o = side * 32;   // 8 TF32 along K inside the 64-byte row
                            mma_tf32(d, a_h, sdesc64(b_h + o), idesc, fresh && side == 0 ? 0u : 1u);
                            mma_tf32(ds, a_h, sdesc64(b_l + o), idesc, fresh && side == 0 && ds != d ? 0u : 1u);
                            mma_tf32(ds, a_l, sdesc64(b_h + o), idesc, 1);
                        }
                    }
                    mma_commit(&mma_bar[b]);
                    __threadfence_block();
                    *(volatile int *)&s_issued = k + 1;
                }
            }
            ok = __all_sync(0xffffffffu, ok);
        }
        pos += FU_WARPS;
    }
    tc_fence_before();
    __syncthreads();
    // after an expired wait, operand copies may still be in flight: let them land (bounded) before exit
    if (tid == 32)
        for (int b = 0; b < 2; ++b)
            while (a_waited[b] < a_issued[b]) {
                if (!mbar_wait(&aimg_bar[b], a_waited[b] & 1)) atomicExch(err, 10);
                ++a_waited[b];
            }
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
}

// ------------------------------------------------------------ host tables
uint32_t morton10(uint32_t x) {
    x &= 0x3ff;
    x = (x | (x << 16)) & 0x030000ff;
    x = (x | (x << 8)) & 0x0300f00f;
    x = (x | (x << 4)) & 0x030c30c3;
    x = (x | (x << 2)) & 0x09249249;
    return x;
}

std::mutex g_fused_mu;

// Field-major copies of the far records and vertex ids of the list entries (test side), and the entries' FuTrial.
__global__ void k_tl_soa(int64_t ntl, const int4 *__restrict__ tl, const float *__restrict__ rec,
                         const int32_t *__restrict__ vid, float *__restrict__ farT, int32_t *__restrict__ vidT,
                         float *__restrict__ trial) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ntl * FB_REC;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i % ntl, f = i / ntl;
        const int t = tl[e].x;
        farT[i] = rec[(int64_t)t * FB_REC + f];
        if (f < 3) vidT[i] = vid[3 * (int64_t)t + f];
    }
    constexpr int TW = sizeof(FuTrial) / 4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ntl * TW; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / TW;
        const int f = (int)(i - e * TW), t = tl[e].x;
        trial[i] = f < FB_REC ? rec[(int64_t)t * FB_REC + f]
                              : __int_as_float(f < FB_REC + 3 ? vid[3 * (int64_t)t + f - FB_REC] : t);
    }
}

}  // namespace

FusedTables &fused_tables(Mesh &m, cudaStream_t st) {
    std::lock_guard<std::mutex> lk(g_fused_mu);
    if (m.fused) return *m.fused;
    const HostMesh &h = m.h;
    const int nc = h.ncell;
    const int64_t nt = h.nt;
    std::vector<int32_t> ecell(h.ne);
    for (int c = 0; c < nc; ++c)
        for (int32_t e = h.cell_off[c]; e < h.cell_off[c + 1]; ++e) ecell[e] = c;
    // spatial order of the triangles (Morton code of the centroid in the bounding box)
    std::vector<double> cen(3 * nt);
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    for (int64_t t = 0; t < nt; ++t)
        for (int d = 0; d < 3; ++d) {
            double x = 0;
            for (int a = 0; a < 3; ++a) x += h.verts[3 * h.tris[3 * t + a] + d];
            cen[3 * t + d] = x / 3.0;
            lo[d] = std::min(lo[d], x / 3.0);
            hi[d] = std::max(hi[d], x / 3.0);
        }
    std::vector<uint32_t> key(nt);
    for (int64_t t = 0; t < nt; ++t) {
        uint32_t q[3];
        for (int d = 0; d < 3; ++d) {
            const double span = hi[d] - lo[d];
            q[d] = span > 0 ? (uint32_t)std::min(1023.0, (cen[3 * t + d] - lo[d]) / span * 1023.0) : 0u;
        }
        key[t] = morton10(q[0]) | (morton10(q[1]) << 1) | (morton10(q[2]) << 2);
    }
    std::vector<std::vector<int32_t>> lists(nc);
    for (int64_t t = 0; t < nt; ++t) {
        int seen[3] = {-1, -1, -1};
        for (int a = 0; a < 3; ++a) {
            const int c = ecell[h.tri_edge[3 * t + a]];
            if (c != seen[0] && c != seen[1]) lists[c].push_back((int32_t)t);
            seen[a] = c;
        }
    }
    auto ft = std::make_shared<FusedTables>();
    ft->tl_off.assign(nc + 1, 0);
    std::vector<int4> ent;
    std::vector<int32_t> tcell;
    for (int c = 0; c < nc; ++c) {
        auto &L = lists[c];
        std::stable_sort(L.begin(), L.end(), [&](int32_t a, int32_t b) { return key[a] < key[b]; });
        ft->tl_off[c] = (int32_t)ent.size();
        ft->nmax = std::max(ft->nmax, h.cell_off[c + 1] - h.cell_off[c]);
        for (int32_t t : L) {
            uint32_t rows[3], side = 0;
            for (int a = 0; a < 3; ++a) {
                const int32_t e = h.tri_edge[3 * t + a];
                rows[a] = FU_NONE16;
                if (ecell[e] != c) continue;
                rows[a] = (uint32_t)(e - h.cell_off[c]);
                if (h.edge_tri[2 * e] != t) side |= 1u << a;
            }
            ent.push_back(make_int4(t, (int)(rows[0] | (rows[1] << 16)), (int)(rows[2] | (side << 16)), 0));
            tcell.push_back(c);
        }
    }
    ft->tl_off[nc] = (int32_t)ent.size();
    // list positions of the two triangles of every RWG function (both carry it, so both are in its cell's list)
    std::vector<int2> rpos(h.ne, make_int2(-1, -1));
    for (int c = 0; c < nc; ++c)
        for (int32_t q = ft->tl_off[c]; q < ft->tl_off[c + 1]; ++q) {
            const int32_t t = ent[q].x;
            for (int a = 0; a < 3; ++a) {
                const int32_t e = h.tri_edge[3 * t + a];
                if (ecell[e] != c) continue;
                if (h.edge_tri[2 * e] == t) rpos[e].x = q - ft->tl_off[c];
                if (h.edge_tri[2 * e + 1] == t) rpos[e].y = q - ft->tl_off[c];
            }
        }
    for (int64_t e = 0; e < h.ne; ++e)
        CBFM_REQUIRE(rpos[e].x >= 0 && rpos[e].y >= 0, "triangle tables: an RWG function's triangle is missing");
    CBFM_REQUIRE(ft->nmax <= 0xfffe, "cell too large for the fused tables");
    // near list as CSR over the test triangle, both orientations
    std::vector<int32_t> np(2 * m.n_near);
    if (m.n_near)
        CBFM_CUDA(cudaMemcpyAsync(np.data(), m.near_pairs.p, np.size() * 4, cudaMemcpyDeviceToHost, st));
    CBFM_CUDA(cudaStreamSynchronize(st));
    std::vector<int32_t> rowc(nt + 1, 0);
    for (int64_t l = 0; l < m.n_near; ++l) {
        rowc[np[2 * l] + 1]++;
        if (np[2 * l] != np[2 * l + 1]) rowc[np[2 * l + 1] + 1]++;
    }
    for (int64_t t = 0; t < nt; ++t) rowc[t + 1] += rowc[t];
    std::vector<int2> ne(rowc[nt]);
    std::vector<int32_t> fill(rowc.begin(), rowc.end() - 1);
    for (int64_t l = 0; l < m.n_near; ++l) {
        const int32_t t = np[2 * l], s = np[2 * l + 1];
        ne[fill[t]++] = make_int2(s, (int)(2 * l));
        if (t != s) ne[fill[s]++] = make_int2(t, (int)(2 * l + 1));
    }
    CBFM_REQUIRE(2 * m.n_near < (1ll << 31), "near list too long for the fused tables");
    ft->n_near = m.n_near;
    auto up = [&](auto &buf, const auto &v) {
        buf.alloc(std::max<size_t>(1, v.size()));
        if (!v.empty())
            CBFM_CUDA(cudaMemcpyAsync(buf.p, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice, st));
    };
    up(ft->tl, ent);
    up(ft->dtl_off, ft->tl_off);
    up(ft->tl_cell, tcell);
    up(ft->rwg_pos, rpos);
    up(ft->near_row, rowc);
    up(ft->near_ent, ne);
    {
        const int64_t ntl = (int64_t)ent.size();
        ft->farT.alloc((size_t)std::max<int64_t>(1, ntl) * FB_REC);
        ft->vidT.alloc((size_t)std::max<int64_t>(1, ntl) * 3);
        ft->trial.alloc((size_t)std::max<int64_t>(1, ntl) * (sizeof(FuTrial) / 4));
        const unsigned g = (unsigned)std::min<int64_t>((ntl * FB_REC + 255) / 256, 8 * (int64_t)sm_count());
        if (ntl) {
            k_tl_soa<<<g, 256, 0, st>>>(ntl, ft->tl.p, m.far32.p, m.tri_vid.p, ft->farT.p, ft->vidT.p,
                                         ft->trial.p);
            launched("k_tl_soa");
        }
    }
    CBFM_CUDA(cudaStreamSynchronize(st));
    m.fused = ft;
    return *ft;
}

namespace {

FuPlan fu_plan(int lmax, int nmax, int sym, int ls) {
    FuPlan p;
    const int lp = (lmax + 1) & ~1;   // rows per A image, a multiple of 8
    p.sym = sym;
    p.ls = ls;
    p.RA = ls ? 64 : std::max(8, sym ? 8 * lmax : 4 * lp);
    p.NP = std::max(16, (nmax + 15) & ~15);
    p.acol = (uint32_t)(ls ? p.NP : 2 * p.NP);
    p.nacc = 2 * p.acol <= 512 ? 2 : 1;
    p.a_op = (uint32_t)p.RA * 32u;
    p.z_op = (uint32_t)p.NP * 64u;
    p.z_base = (ls ? 20 : 12) * p.a_op;
    p.t_base = p.z_base + 12 * p.z_op;
    // the last A image (buffer 1, lo, Tb) is read 128 rows deep: keep that inside the allocation
    p.total = std::max<uint32_t>(p.t_base + 2 * FU_WARPS * (uint32_t)sizeof(FuTrial), p.z_base - p.a_op + 128u * 32u);
    return p;
}
constexpr uint32_t FU_SMEM = 227u * 1024u - 1024u;   // dynamic shared memory less the alignment of its base
constexpr uint32_t FU_STATIC = 4096u;                // at least the kernel's static shared memory

// Cells the fused form takes: CBFs up to FU_LMAX, RWG functions up to FU_NMAX, and both within
// 768 bytes of operand per CBF lane and RWG row (the ordered plan fits whenever this holds).
bool fu_takes(int lmax, int nmax) {
    const int ra = std::max(8, 4 * ((lmax + 1) & ~1)), np = std::max(16, (nmax + 15) & ~15);
    return lmax <= FU_LMAX && nmax <= FU_NMAX && 768u * (uint32_t)(ra + np) <= FU_SMEM;
}
// m <= n pairs with the conjugate lanes where the lanes and the doubled operand fit (half the quadrature), and Ta, Tb on
// lanes 64 .. 127 where the rows leave them free.
FuPlan fu_choose(int lmax, int nmax) {
    for (int sym = lmax <= FU_LSYM ? 1 : 0; sym >= 0; --sym)
        for (int ls = (sym ? 8 : 4) * lmax <= 64 ? 1 : 0; ls >= 0; --ls) {
            const FuPlan p = fu_plan(lmax, nmax, sym, ls);
            if (p.total + FU_STATIC <= FU_SMEM) return p;
        }
    return fu_plan(lmax, nmax, 0, 0);
}

// CBF operand of every list entry of a mesh, in the shared-memory layout of the
// fused kernel: for entry e (trial triangle of cell n, columns = its edges in n),
// plane (hi, lo) x operator (Ks, Ta, Tb) x rows x 8 floats, each 32-byte row
// swizzled.  Row r = 2 w + (re, im) expands CBF w of C^M_n (Ks rows [0, 2 L),
// Tb rows [2 L, 4 L)) or C^J_n (Ks rows [2 L, 4 L), Ta rows [0, 2 L)):
// (w, re) = (c_re, -c_im), (w, im) = (c_im, c_re) along the columns; the other
// half of Ta and Tb is zero.  Rows [4 L, 8 L) (sym) are the same of conj(c).  TF32
// split hi = tf32(x), lo = tf32(x - hi) of the FP64 coefficient.
__global__ void k_entry_aimg(int64_t ntl, const int4 *__restrict__ tl, const int32_t *__restrict__ tl_cell,
                             const int32_t *__restrict__ tl_off, const int64_t *__restrict__ off,
                             const int32_t *__restrict__ L, const int64_t *__restrict__ boff,
                             const z64 *__restrict__ CM, const z64 *__restrict__ CJ, int sym, float *__restrict__ img) {
    const int64_t e = blockIdx.x;
    if (e >= ntl) return;
    const int n = tl_cell[e], Ln = L[n], rows = (sym ? 8 : 4) * Ln;
    const int64_t bo = boff[n];
    const int4 te = tl[e];
    const uint32_t jl[4] = {(uint32_t)te.y & 0xffffu, ((uint32_t)te.y >> 16) & 0xffffu, (uint32_t)te.z & 0xffffu, FU_NONE16};
    float *dst = img + off[n] + (e - tl_off[n]) * (6 * rows * 8);
    for (int idx = threadIdx.x; idx < 3 * rows * 8; idx += blockDim.x) {
        const int op = idx / (rows * 8), rem = idx - op * rows * 8;
        const int r = rem >> 3, f = rem & 7;
        const int b = f & 3, comp = f >> 2;
        const bool cj = r >= 4 * Ln;
        const int rr = cj ? r - 4 * Ln : r;
        const bool upper = rr >= 2 * Ln;
        const int w = (rr - (upper ? 2 * Ln : 0)) >> 1, ri = r & 1;
        const uint32_t j = b == 0 ? jl[0] : b == 1 ? jl[1] : b == 2 ? jl[2] : FU_NONE16;
        const z64 *src = op == 0 ? (upper ? CJ : CM) : op == 1 ? (upper ? nullptr : CJ) : (upper ? CM : nullptr);
        double val = 0.0;
        if (src && j != FU_NONE16) {
            const z64 q = src[bo + (int64_t)j * Ln + w];
            const double im = cj ? -q.im : q.im;
            val = ri == 0 ? (comp == 0 ? q.re : -im) : (comp == 0 ? im : q.re);
        }
        float hi, lo;
        split64(val, hi, lo);
        const uint32_t o = swz32(r, f) >> 2;
        dst[(int64_t)(0 * 3 + op) * rows * 8 + o] = hi;
        dst[(int64_t)(1 * 3 + op) * rows * 8 + o] = lo;
    }
}

}  // namespace

bool fused_fits(const Mesh &m, const Cbf &c) {
    int lmax = 0, nmax = 0;
    for (int k = 0; k < m.h.ncell; ++k) {
        lmax = std::max(lmax, c.L[k]);
        nmax = std::max(nmax, m.h.cell_off[k + 1] - m.h.cell_off[k]);
    }
    return fu_takes(lmax, nmax);
}

namespace {

// One launch of the fused kernel over the cell pairs of jobs [j0, j1) (their
// combined shared-memory plan fits).
void fused_launch(std::vector<FusedJob> &jobs, const std::vector<std::pair<double, int4>> &items_all, int j0, int j1,
                  const FuPlan &plan, cudaStream_t st) {
    std::vector<std::pair<double, int4>> items;
    for (const auto &it : items_all)
        if (it.second.x >= j0 && it.second.x < j1) items.push_back({it.first, make_int4(it.second.x - j0, it.second.y, it.second.z, 0)});
    if (items.empty()) return;
    // largest items first (the persistent CTAs take them in this order)
    std::stable_sort(items.begin(), items.end(), [](const auto &x, const auto &y) { return x.first > y.first; });
    std::vector<int4> hit(items.size());
    for (size_t i = 0; i < items.size(); ++i) hit[i] = items[i].second;
    CBFM_REQUIRE(plan.total + FU_STATIC <= FU_SMEM, "fused assembly: shared-memory plan too large");
    const uint32_t tcols = plan.nacc * plan.acol <= 256 ? 256u : 512u;
    const int nj = j1 - j0;
    DevBuf<FusedJob> djobs;
    DevBuf<int4> ditems;
    DevBuf<unsigned int> counter;
    DevBuf<int> err;
    djobs.alloc(nj);
    ditems.alloc(hit.size());
    counter.alloc(1);
    err.alloc(1);
    CBFM_CUDA(cudaMemcpyAsync(djobs.p, jobs.data() + j0, sizeof(FusedJob) * nj, cudaMemcpyHostToDevice, st));
    CBFM_CUDA(cudaMemcpyAsync(ditems.p, hit.data(), sizeof(int4) * hit.size(), cudaMemcpyHostToDevice, st));
    CBFM_CUDA(cudaMemsetAsync(counter.p, 0, sizeof(unsigned int), st));
    CBFM_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
    const size_t smem = plan.total + 1024;
    // the same limit from every thread: a smaller one set in between would fail the other's launch
    CBFM_CUDA(cudaFuncSetAttribute(k_fused, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)(FU_SMEM + 1024 - FU_STATIC)));
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)hit.size(), sm_count());
    {
        ProfScope ps_("k_fused", st);
        k_fused<<<grid, FU_THREADS, smem, st>>>(djobs.p, ditems.p, (int)hit.size(), counter.p, err.p, plan, tcols);
        launched("k_fused");
    }
    int herr = 0;
    CBFM_CUDA(cudaMemcpyAsync(&herr, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    CBFM_CUDA(cudaStreamSynchronize(st));
    if (herr == 7) throw Fail{CBFM_ECUDA, "fused assembly: a near pair is missing from the near list"};
    if (herr) throw Fail{CBFM_ETIMEOUT, "fused assembly: a tensor-core wait expired (code " + std::to_string(herr) + ")"};
}

}  // namespace

// Size of the unfused form, as bytes of its local blocks, RWG operators (complex64 and as split planes) and Y^T.  The
// complex64 operators are no longer formed (the gather writes the planes), but the line that mixed_takes_fused draws with
// this sum lies where the fused form is the faster one already: cube of 6912 triangles, just above it, 15.2 ms fused
// and 26.9 unfused for L = 8 (17.3 and 27.1 for 14, 33.4 and 32.8 for 20), spheroid of 6960 16.5 and 35.4; cube of 3072,
// below it, 4.6 and 3.1.
double unfused_scratch_bytes(const Mesh &m, const Cbf &c) {
    const double nt = (double)m.h.nt, ne = (double)m.h.ne, nh = (double)c.nhalf;
    const double ldz = std::ceil(2.0 * ne / 32.0) * 32.0;
    return 27.0 * nt * nt * 8 + 3.0 * ne * ne * 8 + 6.0 * ne * ldz * 4 + 8.0 * 2 * nh * ldz * 4;
}

bool mixed_takes_fused(const Mesh &m, const Cbf &c) {
    if (!fused_fits(m, c)) return false;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return unfused_scratch_bytes(m, c) > std::min(0.25 * (double)free_b, 16.0 * (1ull << 30));
}

void assemble_project_fused(const std::vector<Mesh *> &ms, const std::vector<Cbf *> &cs, const std::vector<c32 *> &A,
                            cudaStream_t st) {
    const int nj = (int)ms.size();
    if (nj == 0) return;
    // near-pair blocks (FP64 closed forms), compact, one launch for all meshes
    std::vector<DevBuf<c32>> nearv(nj);
    std::vector<c32 *> nearp(nj);
    for (int k = 0; k < nj; ++k) {
        nearv[k].alloc((size_t)std::max<int64_t>(1, ms[k]->n_near) * NCOMP);
        nearp[k] = nearv[k].p;
    }
    near_blocks_compact(ms, nearp, st, true);
    std::vector<FusedJob> jobs(nj);
    std::vector<std::pair<double, int4>> items;
    std::vector<DevBuf<int32_t>> dL(nj), dcoff32(nj);
    std::vector<DevBuf<int64_t>> dboff(nj), dcoff(nj);
    std::vector<DevBuf<float>> aimg(nj);
    std::vector<DevBuf<int64_t>> daoff(nj);
    // launches over consecutive jobs of one form (each job's own, so that a mesh gets the same A alone and in a
    // batch) whose combined shared-memory plan fits
    struct Group {
        int j0, j1, lmax, nmax;
        FuPlan plan;
    };
    std::vector<Group> groups;
    std::vector<int> jsym(nj, 0);
    for (int k = 0; k < nj; ++k) {
        int l = 0, n = 0;
        for (int a = 0; a < ms[k]->h.ncell; ++a) {
            l = std::max(l, (int)cs[k]->L[a]);
            n = std::max(n, (int)(ms[k]->h.cell_off[a + 1] - ms[k]->h.cell_off[a]));
        }
        CBFM_REQUIRE(l <= FU_LMAX && n <= FU_NMAX, "fused assembly: cell beyond the tile limits");
        const FuPlan own = fu_choose(l, n);
        jsym[k] = own.sym;
        if (!groups.empty()) {
            Group &g = groups.back();
            const FuPlan both = fu_plan(std::max(g.lmax, l), std::max(g.nmax, n), own.sym, own.ls);
            if (g.plan.sym == own.sym && g.plan.ls == own.ls && g.plan.nacc == own.nacc && both.nacc == own.nacc &&
                both.total + FU_STATIC <= FU_SMEM) {
                g = Group{g.j0, k + 1, std::max(g.lmax, l), std::max(g.nmax, n), both};
                continue;
            }
        }
        groups.push_back(Group{k, k + 1, l, n, own});
    }
    double far_flop = 0.0, bytes = 0.0;
    for (int k = 0; k < nj; ++k) {
        Mesh &m = *ms[k];
        Cbf &c = *cs[k];
        FusedTables &ft = fused_tables(m, st);
        const int nc = m.h.ncell;
        dL[k].alloc(nc);
        dboff[k].alloc(nc + 1);
        dcoff[k].alloc(nc + 1);
        dcoff32[k].alloc(nc + 1);
        CBFM_CUDA(cudaMemcpyAsync(dL[k].p, c.L.data(), 4 * nc, cudaMemcpyHostToDevice, st));
        CBFM_CUDA(cudaMemcpyAsync(dboff[k].p, c.boff.data(), 8 * (nc + 1), cudaMemcpyHostToDevice, st));
        CBFM_CUDA(cudaMemcpyAsync(dcoff[k].p, c.coff.data(), 8 * (nc + 1), cudaMemcpyHostToDevice, st));
        CBFM_CUDA(cudaMemcpyAsync(dcoff32[k].p, m.h.cell_off.data(), 4 * (nc + 1), cudaMemcpyHostToDevice, st));
        FusedJob &J = jobs[k];
        J.rec64 = m.tri64.p;
        J.vid = m.tri_vid.p;
        J.trial = ft.trial.p;
        J.farT = ft.farT.p;
        J.vidT = ft.vidT.p;
        J.ntl = ft.tl_off[nc];
        J.tl = ft.tl.p;
        J.tl_off = ft.dtl_off.p;
        J.cell_off = dcoff32[k].p;
        J.near_row = ft.near_row.p;
        J.near_ent = ft.near_ent.p;
        J.near_val = nearp[k];
        {
            // CBF operand images of every list entry (whole 16-byte pieces)
            std::vector<int64_t> coffs(nc);
            int64_t tot = 0;
            for (int a = 0; a < nc; ++a) {
                coffs[a] = tot;
                tot += (int64_t)(ft.tl_off[a + 1] - ft.tl_off[a]) * 6 * (jsym[k] ? 8 : 4) * c.L[a] * 8;
            }
            daoff[k].alloc(coffs.size());
            aimg[k].alloc((size_t)std::max<int64_t>(16, tot));
            CBFM_CUDA(cudaMemcpyAsync(daoff[k].p, coffs.data(), 8 * coffs.size(), cudaMemcpyHostToDevice, st));
            CBFM_REQUIRE(((uintptr_t)aimg[k].p & 15) == 0, "fused assembly: operand images not 16-byte aligned");
            if (J.ntl > 0) {
                k_entry_aimg<<<(unsigned)J.ntl, 256, 0, st>>>(J.ntl, ft.tl.p, ft.tl_cell.p, ft.dtl_off.p, daoff[k].p,
                                                              dL[k].p, dboff[k].p, c.CM.p, c.CJ.p, jsym[k], aimg[k].p);
                launched("k_entry_aimg");
            }
        }
        J.aimg = aimg[k].p;
        J.aimg_off = daoff[k].p;
        J.CM32 = c.CM32.p;
        J.CJ32 = c.CJ32.p;
        J.boff = dboff[k].p;
        J.coff = dcoff[k].p;
        J.L = dL[k].p;
        J.A = A[k];
        J.nh = c.nhalf;
        J.n = 2 * c.nhalf;
        J.md = media_t<float>(media_full(m.k1, m.k2, m.eta1, m.eta2));
        J.alpha = m.alpha;
        for (int a = 0; a < nc; ++a) {
            const int32_t na = ft.tl_off[a + 1] - ft.tl_off[a];
            CBFM_REQUIRE(c.L[a] == 0 || na > 0, "fused assembly: a cell with CBFs has no triangles");
            if (c.L[a] == 0) continue;
            for (int b = jsym[k] ? a : 0; b < nc; ++b) {
                if (c.L[b] == 0) continue;
                const int32_t nb = ft.tl_off[b + 1] - ft.tl_off[b];
                const bool swap = jsym[k] && na < nb;   // the longer list fills the lanes
                items.push_back({(double)na * nb, swap ? make_int4(k, b, a, 0) : make_int4(k, a, b, 0)});
            }
        }
        const double ntd = (double)m.h.nt;   // far pairs, ordered or unordered
        far_flop += (ntd * ntd - (2.0 * m.n_near - ntd)) * (jsym[k] ? 0.5 : 1.0) * 49.0 * FAR_FLOP_PER_POINT_PAIR;
        bytes += ntd * FB_REC * 4 + (double)m.n_near * NCOMP * 8 + 2.0 * c.boff[nc] * 24 + (double)J.n * J.n * 8;
    }
    for (const Group &g : groups) fused_launch(jobs, items, g.j0, g.j1, g.plan, st);
    prof_add_work("k_fused", far_flop, bytes);
}

}  // namespace cbfm
