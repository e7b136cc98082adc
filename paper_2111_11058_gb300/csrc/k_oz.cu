// k_oz.cu -- FP64 complex products on the tensor cores: every FP64 operand is
// cut into seven signed 8-bit digits of a fixed-point number per row (digits of
// one row share the row's power-of-two scale), the digits travel as FP16, and
// the products of digits are summed exactly in the FP32 accumulators (error-
// free splitting after K. Ozaki, T. Ogita, S. Oishi, S. Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012).
//
// Why.  GB300 has two FP64 multiply-adds per clock and SM; the block solver's
// products run at that rate (~1 TFLOP/s) on the FP64 units whatever their
// schedule.  One real product of digits costs 28 FP16 tensor-core products (the
// digit pairs i + j <= 6), at ~4096 multiply-adds per clock and SM: 35 times
// the FP64 rate at full issue, and no serial chains.
//
// Accuracy.  A row is scaled by 2^E, |x| < 2^E, and rounded to 55 fractional
// bits, x = 2^(E - 55) sum_i d_i 256^(6-i) with d_i in [-128, 128].  The pairs
// i + j >= 7 are left out, so an entry of the product is off by about
// 2^-56 max|a_k| max|b_k| sqrt(K) (a random walk), against sqrt(K) times the
// rms of a_k b_k times 2^-53 sqrt(K) / 4 from the roundings of a sum in FP64.
// Rows and columns of the like size throughout lose nothing by this; where the entries of a row differ by orders of
// magnitude and meet small ones of the column, FP64 sums are the better (operators of FP64 systems, cell blocks of Z,
// everything in the long restarted solves without the CMP: OzHold, internal.cuh).
// All sums in between are integers and exact: a digit pair's product is at most
// 2^14, at most 7 pairs x 128 values of k meet in one accumulator (< 2^24),
// and every 128 values of k the accumulators are drained into two 64-bit
// integers per entry; the K ranges of a tile's CTAs are added as integers
// (any order, same bits) and the result is rounded once to FP64.  The error is
// measured against 128-bit sums in tests/test_matmul_f64_gpu.py.
//
// Complex products become real ones: the left operand's rows are the interleaved
// complex rows, each column b of the right operand becomes two rows
// (b_re, -b_im, ...) and (b_im, b_re, ...), and entry (r, j) leaves in columns
// 2j and 2j + 1.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

#include <cooperative_groups.h>

#include "internal.cuh"
#include "tc_ptx.cuh"

namespace cbfm {

namespace cg = cooperative_groups;
thread_local OzWork *g_oz = nullptr;
thread_local int g_oz_hold = OZ_FREE;

namespace {

using namespace tc;

constexpr int OZ_S = 7;          // digits per operand
constexpr int OZ_BK = 32;        // reals of K per stage (one 64-byte swizzled row per digit)
constexpr int OZ_M = 128;        // left rows per tile
constexpr int OZ_N = 64;         // right rows per tile (32 complex columns)
constexpr int OZ_NC = OZ_N / 2;
constexpr int OZ_A_SLICE = OZ_M * OZ_BK * 2, OZ_B_SLICE = OZ_N * OZ_BK * 2;
constexpr int OZ_A_STAGE = OZ_S * OZ_A_SLICE, OZ_B_STAGE = OZ_S * OZ_B_SLICE;
constexpr int OZ_STAGE = OZ_A_STAGE + OZ_B_STAGE;   // 86 016 bytes
constexpr int OZ_NSTAGE = 2;
constexpr int OZ_CHUNK = 4;      // stages between two drains of the accumulators (K = 128)
constexpr int OZ_EPI = 256;      // threads of the 8 draining warps
constexpr int OZ_THREADS = OZ_EPI + 64;
constexpr int OZ_SMEM = OZ_NSTAGE * OZ_STAGE + 1024;
constexpr int OZ_TMEM = 512;
constexpr int OZ_BAD = 0x7fff;   // row exponent of a row with an infinity or NaN

// ------------------------------------------------------------------ packing
// One CTA cuts 8 rows of one operand: row exponent first (a maximum over the
// row), then the digits.  Lane (rr, ch) of a warp owns 4 complex values of row
// rr in each K block, so that it writes one 16-byte chunk per digit and a warp
// 512 consecutive bytes.  The values of a warp's first four K blocks stay in
// registers between the two passes (K <= 1024 complex: each operand is read
// once).  Bound: the digits' stores, 14 bytes per real (28 for the right
// operand, whose rows are written twice) through L2.
constexpr int PK_WARPS = 16, PK_KEEP = 4;

struct OzPack {
    const void *X;         // complex128, or complex64 (widened exactly) where f32 is set
    int64_t off, rs, cs;   // element (row r, k): X[off + r rs + k cs]
    int conj, f32;
    int rows;              // rows in use (the rest of the last tile is zero)
    int groups;            // 8-row groups, padding included
    int expand;            // right operand: two real rows per row
    uint8_t *out;
    int *E;                // exponent field of each row's largest entry
};
struct OzPack2 {
    OzPack p[2];
    int K, nkb;
};

// fixed-point value (55 fractional bits below 2^E) of the double with bit pattern b in a row of exponent field er
__device__ __forceinline__ long long oz_fix(double x, int er) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    long long m = b & 0xfffffffffffffLL;
    if (ex) m |= 1LL << 52;
    const int sh = er + (er == 0) - ex - (ex == 0);   // >= 0; subnormals count as exponent field 1
    long long q;
    if (sh <= 2) q = m << (2 - sh);
    else if (sh >= 57) q = 0;
    else q = (m + (1LL << (sh - 3))) >> (sh - 2);
    return b < 0 ? -q : q;
}
constexpr long long OZ_BIAS = 0x0080808080808080LL;

// digit s of two biased fixed-point values as an FP16 pair
template <int S>
__device__ __forceinline__ uint32_t oz_digit(unsigned long long t0, unsigned long long t1) {
    uint32_t w;
    if (S == 0) {   // 0..256: nine bits
        w = ((uint32_t)(t0 >> 48) & 0x1ffu) | ((uint32_t)(t1 >> 48) << 16);
        w += 0x64006400u;
    } else {
        constexpr int byte = 6 - S;   // 5..0
        const uint32_t a = byte >= 4 ? (uint32_t)(t0 >> 32) : (uint32_t)t0;
        const uint32_t b = byte >= 4 ? (uint32_t)(t1 >> 32) : (uint32_t)t1;
        constexpr uint32_t k = byte & 3;
        w = __byte_perm(a, b, k | (k << 4) | ((4 + k) << 8) | ((4 + k) << 12));
        w = (w & 0x00ff00ffu) | 0x64006400u;
    }
    const __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&w), __half2half2(__ushort_as_half(0x6480)));   // - 1152
    return *reinterpret_cast<const uint32_t *>(&h);
}
template <int S>
__device__ __forceinline__ void oz_store(uint8_t *dst, int slice, const unsigned long long (&a)[4],
                                         const unsigned long long (&b)[4]) {
    *reinterpret_cast<uint4 *>(dst + (size_t)S * slice) =
        make_uint4(oz_digit<S>(a[0], b[0]), oz_digit<S>(a[1], b[1]), oz_digit<S>(a[2], b[2]), oz_digit<S>(a[3], b[3]));
    if constexpr (S + 1 < OZ_S) oz_store<S + 1>(dst, slice, a, b);
}

__global__ void __launch_bounds__(32 * PK_WARPS) k_oz_pack(const __grid_constant__ OzPack2 pp) {
    const int which = (int)blockIdx.x >= pp.p[0].groups;
    const OzPack &P = pp.p[which];
    const int g = (int)blockIdx.x - (which ? pp.p[0].groups : 0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rr = lane >> 2, ch = lane & 3;
    const int r = g * 8 + rr;
    const bool live = r < P.rows;
    const int64_t x0 = P.off + (int64_t)r * P.rs;
    __shared__ uint32_t s_mx[PK_WARPS][8];
    double2 keep[PK_KEEP][4];
    uint32_t mx = 0;
    auto load = [&](int kb, double2 (&v)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = kb * 16 + ch * 4 + q;
            v[q] = make_double2(0.0, 0.0);
            if (live && k < pp.K) {
                const int64_t i = x0 + (int64_t)k * P.cs;
                if (P.f32) {
                    const float2 f = reinterpret_cast<const float2 *>(P.X)[i];
                    v[q] = make_double2((double)f.x, (double)f.y);
                } else {
                    v[q] = reinterpret_cast<const double2 *>(P.X)[i];
                }
            }
        }
    };
    auto top = [&](const double2 (&v)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            mx = max(mx, max((uint32_t)__double2hiint(v[q].x) & 0x7fffffffu, (uint32_t)__double2hiint(v[q].y) & 0x7fffffffu));
    };
#pragma unroll
    for (int i = 0; i < PK_KEEP; ++i) {
        const int kb = warp + i * PK_WARPS;
        if (kb < pp.nkb) load(kb, keep[i]);
    }
#pragma unroll
    for (int i = 0; i < PK_KEEP; ++i)
        if (warp + i * PK_WARPS < pp.nkb) top(keep[i]);
    for (int kb = warp + PK_KEEP * PK_WARPS; kb < pp.nkb; kb += PK_WARPS) {
        double2 v[4];
        load(kb, v);
        top(v);
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    if (ch == 0) s_mx[warp][rr] = mx;
    __syncthreads();
    mx = 0;
    for (int w = 0; w < PK_WARPS; ++w) mx = max(mx, s_mx[w][rr]);
    int er = (int)(mx >> 20);
    const bool bad = er == 0x7ff;
    if (warp == 0 && ch == 0) P.E[r] = bad ? OZ_BAD : er;
    const int tile_rows = P.expand ? OZ_NC : OZ_M, slice = P.expand ? OZ_B_SLICE : OZ_A_SLICE;
    const int row = P.expand ? 2 * (r % tile_rows) : r % tile_rows;
    uint8_t *base = P.out + (size_t)(r / tile_rows) * pp.nkb * OZ_S * slice;
    auto put = [&](int kb, const double2 (&v)[4]) {
        unsigned long long re[4], im[4], ni[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const long long a = bad ? 0 : oz_fix(v[q].x, er);
            long long b = bad ? 0 : oz_fix(v[q].y, er);
            if (P.conj) b = -b;
            re[q] = (unsigned long long)(a + OZ_BIAS);
            im[q] = (unsigned long long)(b + OZ_BIAS);
            ni[q] = (unsigned long long)(OZ_BIAS - b);
        }
        uint8_t *d = base + (size_t)kb * OZ_S * slice;
        if (P.expand) {   // rows (b_re, -b_im) and (b_im, b_re)
            oz_store<0>(d + row * 64 + ((ch ^ ((row >> 1) & 3)) << 4), slice, re, ni);
            oz_store<0>(d + (row + 1) * 64 + ((ch ^ ((row >> 1) & 3)) << 4), slice, im, re);
        } else {
            oz_store<0>(d + row * 64 + ((ch ^ ((row >> 1) & 3)) << 4), slice, re, im);
        }
    };
#pragma unroll
    for (int i = 0; i < PK_KEEP; ++i)
        if (warp + i * PK_WARPS < pp.nkb) put(warp + i * PK_WARPS, keep[i]);
    for (int kb = warp + PK_KEEP * PK_WARPS; kb < pp.nkb; kb += PK_WARPS) {
        double2 v[4];
        load(kb, v);
        put(kb, v);
    }
}

// ------------------------------------------------------------------ product
struct OzArgs {
    const uint8_t *A, *B;
    const int *EA, *EB;
    z64 *C;
    int64_t ldc;
    int rows, cols;        // left rows and right (complex) columns in use
    int nkb, tn, cs;       // K stages, right tiles, CTAs (of one cluster) per tile
    int swap;              // 1: entry (r, j) goes to C[j][r]
    int accumulate, neg;
    int *err;
};

__device__ __forceinline__ uint32_t idesc_f16(int n) {   // D F32, A and B FP16, both K-major, M = 128
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
            dtmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// eight columns of the accumulators of G consecutive digit sums (64 columns apart), waited for
#define OZ_LD8(v, o, t) \
    "=r"(v[o]), "=r"(v[o + 1]), "=r"(v[o + 2]), "=r"(v[o + 3]), "=r"(v[o + 4]), "=r"(v[o + 5]), "=r"(v[o + 6]), "=r"(v[o + 7])
__device__ __forceinline__ void tmem_ld_3x8(uint32_t t, uint32_t (&v)[24]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%24];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%25];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%26];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : OZ_LD8(v, 0, t), OZ_LD8(v, 8, t), OZ_LD8(v, 16, t)
        : "r"(t), "r"(t + 64), "r"(t + 128)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_4x8(uint32_t t, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : OZ_LD8(v, 0, t), OZ_LD8(v, 8, t), OZ_LD8(v, 16, t), OZ_LD8(v, 24, t)
        : "r"(t), "r"(t + 64), "r"(t + 128), "r"(t + 192)
        : "memory");
}
#undef OZ_LD8

__device__ __forceinline__ long long oz_int(uint32_t bits) { return (long long)__float2int_rn(__uint_as_float(bits)); }

// (H 2^32 + L) 2^(EA + EB - 62 - 2 x 1022) rounded to nearest even, assembled by integer operations (an FP64 conversion
// would hold the FP64 pipe for 64 clocks per warp); NaN where a row held one
__device__ __forceinline__ double oz_round(long long H, long long L, int ea, int eb) {
    if (ea == OZ_BAD || eb == OZ_BAD) return __longlong_as_double(0x7ff8000000000000LL);
    unsigned long long lo = (unsigned long long)L + ((unsigned long long)H << 32);
    long long hi = (H >> 32) + (L >> 63) + (lo < (unsigned long long)L ? 1 : 0);
    const bool neg = hi < 0;
    if (neg) {
        lo = 0ULL - lo;
        hi = ~hi + (lo == 0 ? 1 : 0);
    }
    if ((hi | (long long)lo) == 0) return 0.0;
    // the 64 leading bits and whether anything lies below them
    const int lz = hi ? __clzll(hi) : 64 + __clzll((long long)lo);
    unsigned long long top;
    bool sticky;
    if (lz == 0) {
        top = (unsigned long long)hi;
        sticky = lo != 0;
    } else if (lz < 64) {
        top = ((unsigned long long)hi << lz) | (lo >> (64 - lz));
        sticky = (lo << lz) != 0;
    } else {
        top = lz == 64 ? lo : lo << (lz - 64);
        sticky = false;
    }
    // value = top 2^(64 - lz) ..., top in [2^63, 2^64)
    int e = 127 - lz + (ea + (ea == 0)) + (eb + (eb == 0)) - 62 - 2 * 1022 + 1023;
    unsigned long long m = top >> 11;
    const unsigned long long rest = (top & 0x7ff) | (sticky ? 1 : 0);
    if (rest > 0x400 || (rest == 0x400 && (m & 1))) ++m;
    if (m >> 53) {
        m >>= 1;
        ++e;
    }
    double v;
    if (e >= 1 && e <= 2046) v = __longlong_as_double((long long)((unsigned long long)e << 52 | (m & 0xfffffffffffffULL)));
    else v = ldexp((double)m, e - 1075);
    return neg ? -v : v;
}

__device__ __forceinline__ void oz_write(const OzArgs &P, int r, int j, double re, double im) {
    if (r >= P.rows || j >= P.cols) return;
    z64 *c = P.C + (P.swap ? (int64_t)j * P.ldc + r : (int64_t)r * P.ldc + j);
    if (P.neg) {
        re = -re;
        im = -im;
    }
    if (P.accumulate) {
        const double2 o = *reinterpret_cast<const double2 *>(c);
        re += o.x;
        im += o.y;
    }
    *reinterpret_cast<double2 *>(c) = make_double2(re, im);
}

// One CTA per tile of 128 left rows x 32 complex columns, or a cluster of cs
// CTAs that share the tile's K stages and add their integer sums through
// distributed shared memory (every CTA then rounds and writes 32 / cs
// columns).  Warp 8 fetches the stages (two bulk copies of packed digits
// each), warp 9 issues the MMAs: left digit i meets the right digits 0 .. 6 - i,
// which lie behind one another in shared memory, in one or two MMAs of up to 256
// columns that end in the accumulators of the digit sums i .. 6, so a left
// digit is read once per 256 columns (10 MMAs per 16 of K instead of 28).  The
// 448 accumulator columns leave no room for a second set: the MMAs wait while warps
// 0-7 drain them every 128 of K, and the stage loads go on.
__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz_gemm(const __grid_constant__ OzArgs P) {
    extern __shared__ __align__(16) unsigned char oz_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[OZ_NSTAGE], empty[OZ_NSTAGE], acc_full, acc_free;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)blockIdx.x % P.cs, tile = (int)blockIdx.x / P.cs;
    const int mt = tile / P.tn, nt = tile % P.tn;
    const int per = (P.nkb + P.cs - 1) / P.cs;
    const int s0 = min(P.nkb, rank * per), ns = min(P.nkb, s0 + per) - s0;
    if (tid == 0) {
        for (int i = 0; i < OZ_NSTAGE; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        mbar_init(&acc_full, 1);
        mbar_init(&acc_free, OZ_EPI / 32);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(OZ_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int nchunk = (ns + OZ_CHUNK - 1) / OZ_CHUNK;
    auto fail = [&] {
        atomicExch(&s_abort, 1);
        atomicExch(P.err, 1);
    };
    long long H[32], L[32];
    if (warp == 8) {
        if (lane == 0) {
            const uint8_t *ga = P.A + ((size_t)mt * P.nkb + s0) * OZ_A_STAGE;
            const uint8_t *gb = P.B + ((size_t)nt * P.nkb + s0) * OZ_B_STAGE;
            int issued = 0;
            for (int s = 0; s < ns; ++s) {
                const int b = s % OZ_NSTAGE;
                if (s >= OZ_NSTAGE && !mbar_wait(&empty[b], ((s / OZ_NSTAGE) - 1) & 1)) {
                    fail();
                    break;
                }
                unsigned char *st = sm + b * OZ_STAGE;
                mbar_expect_tx(&full[b], OZ_STAGE);
                bulk_load(st, ga + (size_t)s * OZ_A_STAGE, OZ_A_STAGE, &full[b]);
                bulk_load(st + OZ_A_STAGE, gb + (size_t)s * OZ_B_STAGE, OZ_B_STAGE, &full[b]);
                ++issued;
            }
            // its own copies have landed before the CTA may leave or reuse the buffers
            for (int s = max(0, issued - OZ_NSTAGE); s < issued; ++s)
                if (!mbar_wait(&full[s % OZ_NSTAGE], (s / OZ_NSTAGE) & 1)) fail();
        }
    } else if (warp == 9) {
        if (lane == 0) {
            bool ok = true;
            for (int c = 0; c < nchunk && ok; ++c) {
                if (c > 0 && !mbar_wait(&acc_free, (c - 1) & 1)) {
                    fail();
                    break;
                }
                tc_fence_after();
                const int e = min(ns, (c + 1) * OZ_CHUNK);
                for (int s = c * OZ_CHUNK; s < e; ++s) {
                    const int b = s % OZ_NSTAGE;
                    if (!mbar_wait(&full[b], (s / OZ_NSTAGE) & 1)) {
                        fail();
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(sm + b * OZ_STAGE), sb = sa + OZ_A_STAGE;
#pragma unroll
                    for (int kk = 0; kk < OZ_BK / 16; ++kk) {
                        const uint32_t first = (s == c * OZ_CHUNK && kk == 0) ? 0u : 1u;
#pragma unroll
                        for (int i = 0; i < OZ_S; ++i) {
                            const uint64_t ad = sdesc64(sa + i * OZ_A_SLICE + kk * 32);
                            const int nj = OZ_S - i, n0 = nj < 4 ? nj : 4;
                            const uint32_t acc = i == 0 ? first : 1u;   // digit 0 touches every accumulator first
                            mma_f16(tmem + i * OZ_N, ad, sdesc64(sb + kk * 32), idesc_f16(n0 * OZ_N), acc);
                            if (nj > 4)
                                mma_f16(tmem + (i + 4) * OZ_N, ad, sdesc64(sb + 4 * OZ_B_SLICE + kk * 32),
                                        idesc_f16((nj - 4) * OZ_N), acc);
                        }
                    }
                    mma_commit(&empty[b]);
                }
                if (ok) mma_commit(&acc_full);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 32; ++q) H[q] = L[q] = 0;
        const uint32_t tb = tmem + ((uint32_t)(warp & 3) << 21) + (warp >> 2) * 32;
        for (int c = 0; c < nchunk; ++c) {
            if (!__all_sync(0xffffffffu, mbar_wait(&acc_full, c & 1))) {
                fail();
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int q0 = 0; q0 < 32; q0 += 8) {
                uint32_t u[24];
                tmem_ld_3x8(tb + q0, u);
#pragma unroll
                for (int q = 0; q < 8; ++q) H[q0 + q] += (oz_int(u[q]) << 16) + (oz_int(u[8 + q]) << 8) + oz_int(u[16 + q]);
                uint32_t w[32];
                tmem_ld_4x8(tb + 3 * OZ_N + q0, w);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    L[q0 + q] += (oz_int(w[q]) << 24) + (oz_int(w[8 + q]) << 16) + (oz_int(w[16 + q]) << 8) + oz_int(w[24 + q]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_free);
        }
    }
    __syncthreads();   // every MMA has been drained and every copy has landed (or the waits gave up)
    const int row = tid & 127;
    const int r = mt * OZ_M + row;
    if (P.cs == 1) {
        if (tid < OZ_EPI && !s_abort) {
            const int ea = P.EA[r];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int j = nt * OZ_NC + (warp >> 2) * 16 + q;
                const int eb = P.EB[j];
                oz_write(P, r, j, oz_round(H[2 * q], L[2 * q], ea, eb), oz_round(H[2 * q + 1], L[2 * q + 1], ea, eb));
            }
        }
    } else {
        cg::cluster_group cl = cg::this_cluster();
        long long *Hs = reinterpret_cast<long long *>(sm), *Ls = Hs + OZ_N * OZ_M;
        if (tid < OZ_EPI) {
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                const int o = ((warp >> 2) * 32 + q) * OZ_M + row;
                Hs[o] = H[q];
                Ls[o] = L[q];
            }
        }
        cl.sync();
        if (tid < OZ_EPI && !s_abort) {
            const int nj = OZ_NC / P.cs;
            const int ea = P.EA[r];
            for (int q = tid >> 7; q < nj; q += 2) {
                const int j = rank * nj + q;
                long long h[2] = {0, 0}, l[2] = {0, 0};
                for (int p = 0; p < P.cs; ++p) {
                    const long long *ph = cl.map_shared_rank(Hs, p), *pl = ph + OZ_N * OZ_M;
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        h[x] += ph[(2 * j + x) * OZ_M + row];
                        l[x] += pl[(2 * j + x) * OZ_M + row];
                    }
                }
                const int eb = P.EB[nt * OZ_NC + j];
                oz_write(P, r, nt * OZ_NC + j, oz_round(h[0], l[0], ea, eb), oz_round(h[1], l[1], ea, eb));
            }
        }
        cl.sync();   // no CTA leaves while another reads its sums
    }
    if (warp == 9)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM) : "memory");
}

struct Shape {
    bool swap;
    int64_t rows, cols, mt, nt;   // left rows, right complex columns and their tiles
    size_t bytes;
};
// The operand that becomes the left one: the choice with fewer tiles (the left side is padded to 128, the right
// one to 32), and with equal tiles the one that packs less (a right row is packed twice).
Shape oz_shape(int64_t M, int64_t N, int64_t K) {
    Shape best{};
    int64_t cost = 0;
    const size_t nkb = (size_t)((K + 15) / 16);
    for (int sw = 0; sw < 2; ++sw) {
        Shape s;
        s.swap = sw != 0;
        s.rows = sw ? N : M;
        s.cols = sw ? M : N;
        s.mt = (s.rows + OZ_M - 1) / OZ_M;
        s.nt = (s.cols + OZ_NC - 1) / OZ_NC;
        s.bytes = nkb * (s.mt * (size_t)OZ_A_STAGE + s.nt * (size_t)OZ_B_STAGE) +
                  4 * (size_t)(s.mt * OZ_M + s.nt * OZ_NC) + 1024;
        const int64_t c = s.mt * s.nt;
        if (sw == 0 || c < cost || (c == cost && s.bytes < best.bytes)) {
            best = s;
            cost = c;
        }
    }
    return best;
}

template <typename F>
void set_smem_once(F *f, int bytes) {
    static std::atomic<bool> done[64];
    int dev = 0;
    CBFM_CUDA(cudaGetDevice(&dev));
    if (dev < 64 && done[dev].load(std::memory_order_acquire)) return;
    CBFM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    if (dev < 64) done[dev].store(true, std::memory_order_release);
}

}  // namespace

namespace {

// 8-row groups of an operand: the left one padded to OZ_M rows per tile, the right one to OZ_NC complex columns
OzPack pack_of(const void *X, bool f32, int64_t off, int64_t rs, int64_t cs, bool conj, int64_t rows, bool right,
               uint8_t *out, int *E) {
    OzPack p;
    p.X = X;
    p.off = off;
    p.rs = rs;
    p.cs = cs;
    p.conj = conj;
    p.f32 = f32;
    p.rows = (int)rows;
    const int64_t t = right ? OZ_NC : OZ_M;
    p.groups = (int)((rows + t - 1) / t * t / 8);
    p.expand = right;
    p.out = out;
    p.E = E;
    return p;
}
OzPack pack_a(const GemmDesc &d, int op, const z64 *A, bool right, uint8_t *out, int *E) {   // rows of op(A)
    const bool row = op == 0 || op == 3;
    return pack_of(A, false, d.a_off, row ? d.lda : 1, row ? 1 : d.lda, op >= 2, d.M, right, out, E);
}
OzPack pack_b(const GemmDesc &d, int op, const z64 *B, bool right, uint8_t *out, int *E) {   // columns of op(B)
    const bool row = op == 0 || op == 3;
    return pack_of(B, false, d.b_off, row ? 1 : d.ldb, row ? d.ldb : 1, op >= 2, d.N, right, out, E);
}
void launch_pack(const OzPack *p, int np, int64_t K, cudaStream_t st) {
    OzPack2 pp{};
    for (int i = 0; i < np; ++i) pp.p[i] = p[i];
    pp.K = (int)K;
    pp.nkb = (int)((K + 15) / 16);
    int g = p[0].groups + (np > 1 ? p[1].groups : 0);
    ProfScope ps_("k_oz_pack", st);
    k_oz_pack<<<g, 32 * PK_WARPS, 0, st>>>(pp);
    launched("k_oz_pack");
}
void launch_gemm(OzArgs g, int64_t mt, cudaStream_t st) {
    // CTAs per tile: the K stages are shared while the tiles leave SMs idle, down to half a drain's worth of stages
    // (block solve of the 9216-unknown cube: 120 products 3.45 -> 3.20 ms against a whole one, 3.13 ms with clusters of
    // 16, which cost the 2304-unknown cube's more than they give; the sums are integers, so the split has no say in them)
    const int64_t tiles = mt * g.tn;
    int cs = 1;
    while (cs < 8 && tiles * cs * 2 <= sm_count() && g.nkb >= OZ_CHUNK * cs) cs *= 2;
    g.cs = cs;
    set_smem_once(k_oz_gemm, OZ_SMEM);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * cs), 1, 1);
    cfg.blockDim = dim3(OZ_THREADS, 1, 1);
    cfg.dynamicSmemBytes = OZ_SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ProfScope ps_("k_oz_gemm", st);
    CBFM_CUDA(cudaLaunchKernelEx(&cfg, k_oz_gemm, g));
    launched("k_oz_gemm");
}
// this thread's scratch of at least `bytes`, or a buffer of the call's own
struct Scratch {
    DevBuf<unsigned char> own;
    DevBuf<int> own_err;
    unsigned char *p;
    int *err;
    cudaStream_t st;
    Scratch(size_t bytes, cudaStream_t s) : st(s) {
        if (g_oz) {
            if (g_oz->buf.n < bytes) g_oz->buf.alloc(bytes);
            p = g_oz->buf.p;
            err = g_oz->err;
        } else {
            own.alloc(bytes);
            own_err.alloc(1);
            CBFM_CUDA(cudaMemsetAsync(own_err.p, 0, sizeof(int), st));
            p = own.p;
            err = own_err.p;
        }
    }
    void check() {   // without an OzWork: wait and report
        if (g_oz) return;
        int h = 0;
        CBFM_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
        CBFM_CUDA(cudaStreamSynchronize(st));
        if (h) throw Fail{CBFM_ETIMEOUT, "tensor-core FP64 product: a device wait expired"};
    }
};

}  // namespace

bool oz_takes(int64_t M, int64_t N, int64_t K) {
    if (g_oz_hold >= OZ_FP64_SUMS || M < 1 || N < 1 || K < 1 || M > (1 << 24) || N > (1 << 24) || K > (1 << 18)) return false;
    const Shape s = oz_shape(M, N, K);
    if (s.bytes > ((size_t)2 << 30) || s.mt * s.nt > (1 << 24)) return false;
    return 1.0 * M * N * K > 2.0e6;
}

void gemm_oz(const GemmDesc &d, int opA, int opB, const z64 *A, const z64 *B, z64 *C, bool accumulate, cudaStream_t st,
             bool neg) {
    const Shape s = oz_shape(d.M, d.N, d.K);
    const int nkb = (int)((d.K + 15) / 16);
    const size_t na = (size_t)s.mt * nkb * OZ_A_STAGE, nbb = (size_t)s.nt * nkb * OZ_B_STAGE;
    Scratch ws(s.bytes, st);
    int *EA = reinterpret_cast<int *>(ws.p + na + nbb), *EB = EA + s.mt * OZ_M;
    OzPack p[2];
    if (s.swap) {
        p[0] = pack_b(d, opB, B, false, ws.p, EA);
        p[1] = pack_a(d, opA, A, true, ws.p + na, EB);
    } else {
        p[0] = pack_a(d, opA, A, false, ws.p, EA);
        p[1] = pack_b(d, opB, B, true, ws.p + na, EB);
    }
    prof_add_work("k_oz_gemm", 8.0 * d.M * d.N * d.K, 16.0 * (d.M * d.K + d.K * d.N + d.M * d.N));
    launch_pack(p, 2, d.K, st);
    launch_gemm(OzArgs{ws.p, ws.p + na, EA, EB, C + d.c_off, d.ldc, (int)s.rows, (int)s.cols, nkb, (int)s.nt, 1,
                       s.swap ? 1 : 0, accumulate ? 1 : 0, neg ? 1 : 0, ws.err},
                s.mt, st);
    ws.check();
}

void OzMat::pack(const c32 *X, int64_t n_rows, int64_t n_k, int64_t ld, cudaStream_t st) {
    rows = n_rows;
    K = n_k;
    const int64_t mt = (rows + OZ_M - 1) / OZ_M;
    const size_t na = (size_t)mt * ((K + 15) / 16) * OZ_A_STAGE;
    buf.alloc(na + 4 * (size_t)(mt * OZ_M));
    const OzPack p = pack_of(X, true, 0, ld, 1, false, rows, false, buf.p, reinterpret_cast<int *>(buf.p + na));
    launch_pack(&p, 1, K, st);
}

void gemm_oz_rows(const OzMat &M, const z64 *in, int64_t ldi, z64 *out, int64_t ldo, int64_t n, cudaStream_t st) {
    const int64_t mt = (M.rows + OZ_M - 1) / OZ_M, nt = (n + OZ_NC - 1) / OZ_NC;
    const int nkb = (int)((M.K + 15) / 16);
    const size_t na = (size_t)mt * nkb * OZ_A_STAGE, nbb = (size_t)nt * nkb * OZ_B_STAGE;
    Scratch ws(nbb + 4 * (size_t)(nt * OZ_NC), st);
    int *EB = reinterpret_cast<int *>(ws.p + nbb);
    const OzPack p = pack_of(in, false, 0, ldi, 1, false, n, true, ws.p, EB);
    prof_add_work("k_oz_gemm", 8.0 * M.rows * n * M.K, 16.0 * (M.rows * M.K + n * (M.rows + M.K)));
    launch_pack(&p, 1, M.K, st);
    launch_gemm(OzArgs{M.buf.p, ws.p, reinterpret_cast<const int *>(M.buf.p + na), EB, out, ldo, (int)M.rows, (int)n,
                       nkb, (int)nt, 1, 1, 0, 0, ws.err},
                mt, st);
    ws.check();
}

}  // namespace cbfm
