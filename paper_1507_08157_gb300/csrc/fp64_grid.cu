// Float64 grid contractions on the tensor cores: response density and potential integrals of FP64
// contexts (Secs. II C, III A) by error-free splitting (Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59 (2012) 95; on tensor cores: Mukunoki, Ozaki, Ogita and Imamura, ISC 2020).
//
// This part executes about two float64 multiply-adds per cycle and SM, and the CUDA-core kernels ran
// at that rate. Here a value x with |x| < 2^E becomes the integer q = round(x 2^(62 - E)), written
// in nine balanced digits of seven bits, q = sum_i d_i 128^(8 - i), -64 <= d_i <= 63 (the first to 64), each
// exact in float16. A product sum over K terms is
//
//   sum x y = 2^(Ex + Ey - 124) sum_l 128^(16 - l) D_l,     D_l = sum_{i + j = l} sum_K x_i y_j,
//
// and each D_l, l <= 8, is an integer below 2^24 (9 pairs x 455 terms x 64 x 64; past that only the
// lowest level can round, at 2^-80 of the result's range), so the float32 accumulators of
// kind::f16 hold it exactly. The levels l > 8 and the rounding of q leave an error of about 2^-63 of
// 2^(Ex + Ey) per term.
// The density's scales are those of a sum: one per point, of the tile's chi there, and one per phi, of
// its P over the tile's chi. Where both are reached by different chi, a sum can still be small against
// them, so every point compares the largest of its terms T phi with the largest that its scales
// allow: below 2^-9 of it (0.03 % of the points for P without structure), or where a tile's P is not
// finite or its columns' scales lie too far apart, the point is summed in float64. So the error is that of
// float64 sums or below at every point: relative to the sum of the terms' sizes at most 6.1e-16, root
// mean square 9.6e-17, where float64 sums have 8.2e-16 and 1.2e-16 (emulated, 8 atoms, 48^3); with P's
// rows in blocks of 1, 1e-6 and 1e-12, 7.2e-16 and 9.7e-17 against 9.3e-16 and 1.2e-16. (Entry point, 32
// atoms and 3 states: P without structure or decaying with distance 1.05 and 1.07 ms, such rows, where
// 40 % of the points are summed again, 7.5; CUDA cores 17.2 to 18.0.) One scale for
// the chi table and one for a state's P left no digit right where chi is below 1e-16 of its largest value.
// The integrals' scales are chi's and (V phi)'s largest values on the tile, each function its own. An
// entry's error is about 2^-63 of the sum over tiles of 512 times their product, below that of a float64
// sum wherever the entry's terms come within 2^-10 of it; entries of functions that only graze each
// other have the same absolute error and fewer digits than a float64 sum would give them. A tile whose
// V is not finite is summed in float64. Largest error of small-8's entries, of the largest entry (emulated): V
// without structure 3.3e-16, float64 sums 6.4e-16; V a Gaussian of 1 A, 3.6e-16 and 7.5e-16 (with one
// scale for all of V 6e-11).
//
// The digits of B are stacked along N (32 columns each), the accumulators of the levels along the
// columns of TMEM (32 each): for digit i of A one MMA of N = 32 (9 - i) columns, placed at level i,
// makes all its products with the digits j <= 8 - i of B. Nine MMAs (the first cut in two at 256
// columns) per 16 of K instead of 45.
//
// Both kernels: 320 threads; warp 8 brings the digit tiles of chi (128 x 64, 16 KB) through a ring by
// TMA from tables made at creation, eight warps make the digits of B for the next K block while
// warp 9 issues the MMAs of this one, then combine the levels in integers and float64. Every wait is
// bounded.
// Measured (GB300, stage, CUDA events, CUDA-core kernel and this): 8 atoms, 48^3, 1 state: density 0.57
// and 0.08 ms, integrals 1.05 and 0.07; 32 atoms with 4 + 9 functions, 90^3, 3 states: density 19.3 and
// 0.98 ms, integrals 21.2 and 0.85. A block has one set of
// accumulators, so that its MMAs (45 digit products in 10 MMAs) and its float64 epilogue take turns: at 32
// atoms the tensor pipe is busy 27 % (density) and 39 % (integrals), the float64 pipe 42 and 37 %. In small
// systems a block's start and end count as well.
#include "tc_common.cuh"
#include "tddft_internal.h"

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

namespace tddft {

using namespace tc;

bool encode_map_2d(CUtensorMap *map, CUtensorMapDataType dt, const void *ptr, unsigned long long inner,
                   unsigned long long rows, unsigned long long row_bytes, unsigned box_inner, unsigned box_rows);

namespace {

constexpr int ND = 9;                // digits, and levels kept
constexpr int SHIFT = 62;            // |q| <= 2^62
constexpr int NB = 32;               // B columns of one digit
constexpr int THREADS64 = 320;       // warps 0-7 make B and combine, 8 TMA, 9 MMA
constexpr int A_RING = 8, A_TILE = 16384;
constexpr int B_KMAJ = ND * NB * 128;           // integrals: rows (digit, phi) of 64 points
constexpr int B_NMAJ = (ND + 1) / 2 * 8192;     // density: blocks of 64 columns (two digits) x 64 chi
constexpr int MAX_K = 448;           // chi summed in one accumulator

struct __align__(8) Shared64 {
    unsigned long long a_full[A_RING], a_empty[A_RING];
    unsigned long long b_full[2], b_empty[2];
    unsigned long long acc_full, acc_empty, drain;
    unsigned int tmem_base;
    int abort;
    double part[128];                // density: the second half's sums and exponents
    int most[128], found[128];
    unsigned lost[4];                // points to sum in float64
    int vmax[8], down[NB];           // integrals: V's exponents by warp, the columns' scales
};

__device__ __forceinline__ void init64(Shared64 *c) {
    for (int i = 0; i < A_RING; ++i) {
        mbar_init(&c->a_full[i], 1);
        mbar_init(&c->a_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
        mbar_init(&c->b_full[i], 8);
        mbar_init(&c->b_empty[i], 1);
    }
    mbar_init(&c->acc_full, 1);
    mbar_init(&c->acc_empty, 8);
    mbar_init(&c->drain, 1);
    c->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// 2^(62 - E) of a column's values (0 of a column of zeros)
__device__ __forceinline__ double column_scale(int E) {
    return E < -900 || E > 1024 ? 0.0 : __hiloint2double((1023 + SHIFT - E) << 20, 0);
}

// q + sum_i 64 128^i: the digits plus 64, seven bits each and eight for the first, up to 128
__device__ __forceinline__ unsigned long long biased(double scaled) {
    constexpr unsigned long long C = 0x2040810204081020ull << 1;   // 64 (1 + 128 + ... + 128^8)
    return (unsigned long long)__double2ll_rn(scaled) + C;
}
// two digits (plus 64) as float16 pair: 1024 + d is exact, then 1088 is taken off
__device__ __forceinline__ unsigned digit_pair(unsigned a, unsigned b) {
    const unsigned v = 0x64006400u | a | (b << 16);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), __half2half2(__ushort_as_half(0x6440)));
    return *reinterpret_cast<const unsigned *>(&h);
}
__device__ __forceinline__ unsigned digit(unsigned long long u, int j) {
    const unsigned d = (unsigned)(u >> (7 * (ND - 1 - j)));
    return j == 0 ? d : d & 127u;
}

// an integer below 2^51 in size as float64 with one addition
__device__ __forceinline__ double to_double(long long v) {
    return __longlong_as_double(0x4330000000000000ll + (1ll << 51) + v) - 6755399441055744.0;
}
// sum_l 128^(8 - l) D_l of the nine level sums (float32 integers). |D_l| <= (l + 1) 512 64 64, so that
// both halves stay below 2^50.
__device__ __forceinline__ double combine_levels(const float (*D)[8], int e) {
    long long hi = 0, lo = 0;
#pragma unroll
    for (int l = 0; l < 5; ++l) hi = hi * 128 + (int)__float2int_rn(D[l][e]);
#pragma unroll
    for (int l = 5; l < ND; ++l) lo = lo * 128 + (int)__float2int_rn(D[l][e]);
    return fma(to_double(hi), 268435456.0, to_double(lo));
}
// E with |x| < 2^E of one value: VAL_ZERO of zero, VAL_BAD of infinity and NaN
constexpr int VAL_ZERO = -8192, VAL_BAD = 8191;
__device__ __forceinline__ int value_exponent(double x) {
    const int h = __double2hiint(x) & 0x7fffffff, f = h >> 20;
    return (h | __double2loint(x)) == 0 ? VAL_ZERO : f == 2047 ? VAL_BAD : max(f, 1) - 1022;
}
// exponent field of x (0: zero or below the normal range, 2047: infinity or NaN)
__device__ __forceinline__ int expo_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

__device__ __forceinline__ void tmem_ld8(unsigned taddr, float *v) {
    unsigned r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 " tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// The MMAs of one K block of 64: the nine digit tiles of A against B (descriptor low words b + kk bk).
// bx: distance to digit 8 of B. False after an expired wait.
__device__ __forceinline__ bool mma_block(Shared64 *ctl, volatile int *abort, unsigned a_lo, unsigned &qa, unsigned tmem,
                                          unsigned b, unsigned bk, unsigned bx, unsigned idesc_flags, bool first,
                                          long long wlim) {
    for (int i = 0; i < ND; ++i, ++qa) {
        const unsigned st = qa % A_RING;
        if (!mbar_wait(&ctl->a_full[st], (qa / A_RING) & 1, abort, wlim)) return false;
        tc_fence_after();
        const unsigned a = a_lo + st * (A_TILE >> 4);
        const unsigned idesc = idesc_f16(128, min(256, NB * (ND - i))) | idesc_flags;
#pragma unroll
        for (unsigned kk = 0; kk < 4; ++kk) {
            const unsigned acc = (first && i == 0 && kk == 0) ? 0u : 1u;
            mma_f16(tmem + i * NB, desc_of(a + 2 * kk), desc_of(b + kk * bk), idesc, acc);
            if (i == 0)   // digit 8 of B, level 8
                mma_f16(tmem + 8 * NB, desc_of(a + 2 * kk), desc_of(b + bx + kk * bk), idesc_f16(128, NB) | idesc_flags, acc);
        }
        mma_commit(&ctl->a_empty[st]);
    }
    return true;
}

// ---- potential integrals: D[a][b] = sum_r chi_a(r) (V_s phi_b)(r) --------------------------------------
// Block = (item, state): at most 128 chi and 32 phi of a tile, K = its 512 points.
__global__ void __launch_bounds__(THREADS64, 1) integrals64_kernel(
    const __grid_constant__ CUtensorMap mX,   // chi digits [digit * slots + slot][512], box 64 x 128
    int n, int nt, int k, const IItem *__restrict__ items, long long slots, const int *__restrict__ cids,
    const double *__restrict__ cval, const int *__restrict__ pids, const double *__restrict__ pval,
    const int *__restrict__ cexp, const short *__restrict__ pexp, int nchi, int nphi, const double *__restrict__ V, double dV,
    double *__restrict__ out, int *err, long long wlim) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<unsigned long long>(smem_raw) + 1023ull) & ~1023ull);
    unsigned char *A = base, *B = base + A_RING * A_TILE;
    double *Vt = reinterpret_cast<double *>(B + 2 * B_KMAJ);
    short *Ve = reinterpret_cast<short *>(Vt + TILE_PTS);
    Shared64 *ctl = reinterpret_cast<Shared64 *>(Ve + TILE_PTS);
    volatile int *abort = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x % k;
    const IItem d = items[blockIdx.x / k];
    const long long n3 = (long long)n * n * n;
    if (threadIdx.x == 0) init64(ctl);
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = ctl->tmem_base;
    constexpr int KB = TILE_PTS / 64;

    if (warp == 8) {
        if (lane == 0) {
            unsigned q = 0;
            for (; q < KB * ND; ++q) {
                const unsigned st = q % A_RING;
                if (q >= A_RING && !mbar_wait(&ctl->a_empty[st], (q / A_RING - 1) & 1, abort, wlim)) break;
                mbar_expect_tx(&ctl->a_full[st], A_TILE);
                tma_load_2d(A + st * A_TILE, &mX, &ctl->a_full[st], (int)(q / ND) * 64, (int)((q % ND) * slots + d.c0));
            }
            // after an abort, the loads already issued land before the block exits
            if (*abort)
                for (unsigned i = q > A_RING ? q - A_RING : 0; i < q; ++i)
                    mbar_drain(&ctl->a_full[i % A_RING], (i / A_RING) & 1, wlim);
        }
    } else if (warp == 9) {
        if (elect_one()) {
            const unsigned a_lo = desc_lo(smem_u32(A));
            unsigned qa = 0;
            bool ok = true;
            for (unsigned kb = 0; kb < KB && ok; ++kb) {
                ok = mbar_wait(&ctl->b_full[kb & 1], (kb >> 1) & 1, abort, wlim);
                if (!ok) break;
                tc_fence_after();
                ok = mma_block(ctl, abort, a_lo, qa, tmem, desc_lo(smem_u32(B + (kb & 1) * B_KMAJ)), 2u, (8 * NB * 128) >> 4,
                               0u, kb == 0, wlim);
                mma_commit(&ctl->b_empty[kb & 1]);
            }
            mma_commit(&ctl->acc_full);
            if (*abort) {
                mma_commit(&ctl->drain);
                mbar_drain(&ctl->drain, 0, wlim);
            }
        }
    } else {
        // V on the tile and its exponents, then V scaled by the largest (as it is where it is not finite)
        const int tx = d.t / (nt * nt), ty = (d.t / nt) % nt, tz = d.t % nt;
        double vr[2];
        int etv = VAL_ZERO;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int lp = threadIdx.x + h * 256;
            const int gx = tx * TILE + (lp >> 6), gy = ty * TILE + ((lp >> 3) & 7), gz = tz * TILE + (lp & 7);
            vr[h] = (gx < n && gy < n && gz < n) ? V[(long long)s * n3 + ((long long)gx * n + gy) * n + gz] : 0.0;
            const int E = value_exponent(vr[h]);
            Ve[lp] = (short)E;
            etv = max(etv, E);
        }
        etv = __reduce_max_sync(0xffffffffu, etv);
        if (lane == 0) ctl->vmax[warp] = etv;
        asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 8; ++i) etv = max(etv, ctl->vmax[i]);
        const bool bad = etv == VAL_BAD;
        etv = etv == VAL_ZERO || bad ? 0 : max(etv, -900);
        const double vs = __hiloint2double((1023 + SHIFT - etv) << 20, 0);
#pragma unroll
        for (int h = 0; h < 2; ++h) Vt[threadIdx.x + h * 256] = bad ? vr[h] : vr[h] * vs;
        // digits of V phi: thread = (phi b, octet o of the K block's points). phi takes the exponent of the
        // scale 2^E of its column of products without V's: phi 2^-down, |V phi| < 2^(etv + down)
        const int o = threadIdx.x & 7, b = threadIdx.x >> 3;
        bool ok = true;
        int down;
        {
            unsigned m = 0xc000c000u, pm = 0xe000e000u;       // pairs of exponents: V phi, phi
            const uint4 *pe = reinterpret_cast<const uint4 *>(pexp + (long long)(d.p0 + b) * TILE_PTS + o * 8);
            const uint4 *ve = reinterpret_cast<const uint4 *>(Ve + o * 8);
            if (b < d.np)
#pragma unroll
                for (int kb = 0; kb < KB; ++kb) {
                    const uint4 x = __ldg(pe + kb * 8), y = ve[kb * 8];
                    m = __vmaxs2(m, __vmaxs2(__vmaxs2(__vadd2(x.x, y.x), __vadd2(x.y, y.y)),
                                             __vmaxs2(__vadd2(x.z, y.z), __vadd2(x.w, y.w))));
                    pm = __vmaxs2(pm, __vmaxs2(__vmaxs2(x.x, x.y), __vmaxs2(x.z, x.w)));
                }
#pragma unroll
            for (int i = 1; i < 8; i *= 2) {
                m = __vmaxs2(m, __shfl_xor_sync(0xffffffffu, m, i));
                pm = __vmaxs2(pm, __shfl_xor_sync(0xffffffffu, pm, i));
            }
            const int mw = max((int)(short)(m & 0xffffu), (int)(short)(m >> 16));
            const int mp = max((int)(short)(pm & 0xffffu), (int)(short)(pm >> 16));
            // 2^900 at most above phi's largest value, so that no phi leaves the range
            down = mw < VAL_ZERO / 2 || bad ? 0 : max(max(mw - etv, mp - 900), -1000);
            if (o == 0) ctl->down[b] = down;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        auto scaled = [&](double x) {
            const int hi = __double2hiint(x), ef = (hi >> 20) & 0x7ff;
            return ef != 0 && ef > down ? __hiloint2double(hi - down * (1 << 20), __double2loint(x)) : 0.0;
        };
        for (int kb = 0; kb < KB; ++kb) {
            unsigned long long u[8];
            const double2 *pp = reinterpret_cast<const double2 *>(pval + (long long)(d.p0 + b) * TILE_PTS + kb * 64 + o * 8);
            const double2 *vv = reinterpret_cast<const double2 *>(Vt + kb * 64 + o * 8);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double2 p = b < d.np && !bad ? __ldg(pp + e) : make_double2(0.0, 0.0);
                const double2 v = bad ? make_double2(0.0, 0.0) : vv[e];
                u[2 * e] = biased(scaled(p.x) * v.x);
                u[2 * e + 1] = biased(scaled(p.y) * v.y);
            }
            if (kb >= 2 && !mbar_wait_warp(&ctl->b_empty[kb & 1], ((kb >> 1) - 1) & 1, abort, wlim)) {
                ok = false;
                break;
            }
            unsigned char *Bk = B + (kb & 1) * B_KMAJ;
#pragma unroll
            for (int j = 0; j < ND; ++j) {
                uint4 x;
                x.x = digit_pair(digit(u[0], j), digit(u[1], j));
                x.y = digit_pair(digit(u[2], j), digit(u[3], j));
                x.z = digit_pair(digit(u[4], j), digit(u[5], j));
                x.w = digit_pair(digit(u[6], j), digit(u[7], j));
                *reinterpret_cast<uint4 *>(Bk + sw128_offset(j * NB + b, o)) = x;
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->b_full[kb & 1]);
        }
        ok = ok && __all_sync(0xffffffffu, mbar_wait(&ctl->acc_full, 0, abort, wlim) && !*abort);
        tc_fence_after();
        // rows of chi over warps 0-3 and 4-7, the phi halves between the two groups
        const int a = (warp & 3) * 32 + lane;
        const int ea = 56 - 2 * SHIFT + etv + (a < d.nc ? cexp[d.c0 + a] : 0);
        double *o_row = out + (long long)s * nchi * nphi + (a < d.nc ? (long long)cids[d.c0 + a] * nphi : 0);
        for (int c = (warp >> 2) * 16; c < (warp >> 2) * 16 + 16 && c < d.np; c += 8) {
            float D[ND][8];
#pragma unroll
            for (int l = 0; l < ND; ++l) tmem_ld8(tmem + l * NB + c + ((unsigned)((warp & 3) * 32) << 16), D[l]);
            if (!ok || a >= d.nc || bad) continue;
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (c + e < d.np) {
                    double x = combine_levels(D, e);
                    const int f = expo_field(x), up = ea + ctl->down[c + e];
                    if (f != 0) x = f + up > 0 ? __hiloint2double(__double2hiint(x) + up * (1 << 20), __double2loint(x)) : ldexp(x, up);
                    atomicAdd(o_row + pids[d.p0 + c + e], dV * x);
                }
        }
        // V not finite on the tile: the sums in float64
        if (ok && bad && a < d.nc)
            for (int c = (warp >> 2) * 16; c < (warp >> 2) * 16 + 16 && c < d.np; ++c) {
                const double *x = cval + (long long)(d.c0 + a) * TILE_PTS, *y = pval + (long long)(d.p0 + c) * TILE_PTS;
                double v = 0.0;
                for (int i = 0; i < TILE_PTS; ++i) v = fma(__ldg(x + i), __ldg(y + i) * Vt[i], v);
                atomicAdd(o_row + pids[d.p0 + c], dV * v);
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
    if (threadIdx.x == 0 && ctl->abort) atomicExch(err, 1);
}

// ---- response density: rho(r) = sum_b phi_b(r) sum_a chi_a(r) P_ab ------------------------------------
// scales of the P columns (a phi over the chi of a tile's list) and the rows (a point over them)
constexpr int COL_ZERO = -20000;     // a column of zeros
constexpr int ROW_ZERO = -20000;     // no chi is nonzero at the point
constexpr int TILE_F64 = 20000;      // (of a tile's largest column) the whole tile in float64
constexpr int LOST_BITS = 9;         // terms this far below their scales: the point in float64

// cexp[s][slot]: |P_ab| < 2^E over the tile's chi; ctop[s][listed tile]: the largest E of the tile's columns,
// or TILE_F64 where P is not finite or a column's scale is more than 2^900 below the largest or below
// 2^-900. Block = (listed tile, state). 32 atoms, 3 states: 17 us.
__global__ void __launch_bounds__(256) column_exponents_kernel(const int *__restrict__ tiles, int ntiles,
                                                               const int *__restrict__ coff, const int *__restrict__ cids,
                                                               const int *__restrict__ poff, const int *__restrict__ pids,
                                                               int nphi, const double *__restrict__ P, long long sP,
                                                               long long pslots, int *__restrict__ cexp,
                                                               int *__restrict__ ctop) {
    __shared__ int mx[NB], top, low;
    const int t = tiles[blockIdx.x], s = blockIdx.y;
    const int c0 = coff[t], nc = coff[t + 1] - c0, p0 = poff[t], np = poff[t + 1] - p0;
    const double *Ps = P + (long long)s * sP;
    const int qd = threadIdx.x & 7, a0 = threadIdx.x >> 3;
    if (threadIdx.x == 0) top = COL_ZERO, low = TILE_F64;
    for (int b0 = 0; b0 < np; b0 += NB) {
        const int nb = min(NB, np - b0);
        if (threadIdx.x < NB) mx[threadIdx.x] = 0;
        __syncthreads();
        // of the high words without sign, and 1 where only the low word is not zero
        int m[4] = {0, 0, 0, 0};
        if (qd * 4 < nb) {
            const int col = pids[p0 + b0 + qd * 4];
#pragma unroll 4
            for (int a = a0; a < nc; a += 32) {
                const double2 *p = reinterpret_cast<const double2 *>(Ps + (long long)cids[c0 + a] * nphi + col);
                const double2 x = __ldg(p), y = __ldg(p + 1);
                const double v[4] = {x.x, x.y, y.x, y.y};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    m[e] = max(m[e], max(__double2hiint(v[e]) & 0x7fffffff, __double2loint(v[e]) != 0 ? 1 : 0));
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            m[e] = max(m[e], __shfl_xor_sync(0xffffffffu, m[e], 8));
            m[e] = max(m[e], __shfl_xor_sync(0xffffffffu, m[e], 16));
            if ((threadIdx.x & 31) < 8) atomicMax(&mx[qd * 4 + e], m[e]);
        }
        __syncthreads();
        if (threadIdx.x < nb) {
            const int h = mx[threadIdx.x], f = h >> 20;
            const int E = h == 0 ? COL_ZERO : f == 2047 ? TILE_F64 : max(f, 1) - 1022;
            cexp[(long long)s * pslots + p0 + b0 + threadIdx.x] = E;
            if (E != COL_ZERO) {
                atomicMax(&top, E);
                atomicMin(&low, E);
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) ctop[(long long)s * ntiles + blockIdx.x] = top != COL_ZERO && (low < -900 || low < top - 900) ? TILE_F64 : top;
}

// Block = (tile, 128 of its points, state); for every 32 phi (and every 448 chi) the product
// T[r][b] = sum_a chi_a(r) P_ab, whose levels each thread combines and multiplies by phi.
__global__ void __launch_bounds__(THREADS64, 1) density64_kernel(
    const __grid_constant__ CUtensorMap mX,   // chi digits [(digit * nchunks + chunk) * 512 + point][64], box 64 x 128
    int n, int nt, int k, int ntiles, const int *__restrict__ tiles, const int *__restrict__ coff,
    const int *__restrict__ cids, const double *__restrict__ cval, const int *__restrict__ cfirst, long long nchunks,
    const int *__restrict__ poff, const int *__restrict__ pids, const double *__restrict__ pval, int nphi,
    const double *__restrict__ P, long long sP, const int *__restrict__ rexp, const int *__restrict__ cexp,
    const int *__restrict__ ctop, long long pslots, double *__restrict__ rho, int *err, long long wlim) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<unsigned long long>(smem_raw) + 1023ull) & ~1023ull);
    unsigned char *A = base, *B = base + A_RING * A_TILE;
    Shared64 *ctl = reinterpret_cast<Shared64 *>(B + 2 * B_NMAJ);
    volatile int *abort = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // states fastest, then the point blocks: blocks that share a tile's tables run together
    const int s = blockIdx.x % k, pb = blockIdx.x / k % 4, ti = blockIdx.x / k / 4, t = tiles[ti];
    const int c0 = coff[t], nc = coff[t + 1] - c0, p0 = poff[t], np = poff[t + 1] - p0;
    const int top = ctop[(long long)s * ntiles + ti];
    const bool f64 = top == TILE_F64;
    const int KB = (nc + 63) / 64, NY = f64 ? 0 : (np + NB - 1) / NB, NZ = (nc + MAX_K - 1) / MAX_K;
    constexpr int ZB = MAX_K / 64;       // K blocks of one accumulation
    if (threadIdx.x == 0) init64(ctl);
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = ctl->tmem_base;

    if (warp == 8) {
        if (lane == 0) {
            unsigned q = 0;
            const unsigned total = (unsigned)(NY * KB * ND);
            for (; q < total; ++q) {
                const unsigned st = q % A_RING;
                if (q >= A_RING && !mbar_wait(&ctl->a_empty[st], (q / A_RING - 1) & 1, abort, wlim)) break;
                mbar_expect_tx(&ctl->a_full[st], A_TILE);
                const long long ch = (long long)(q % ND) * nchunks + cfirst[t] + q / ND % KB;
                tma_load_2d(A + st * A_TILE, &mX, &ctl->a_full[st], 0, (int)(ch * TILE_PTS + pb * 128));
            }
            // after an abort, the loads already issued land before the block exits
            if (*abort)
                for (unsigned i = q > A_RING ? q - A_RING : 0; i < q; ++i)
                    mbar_drain(&ctl->a_full[i % A_RING], (i / A_RING) & 1, wlim);
        }
    } else if (warp == 9) {
        if (elect_one()) {
            const unsigned a_lo = desc_lo(smem_u32(A));
            unsigned qa = 0, qb = 0, acc = 0;
            bool ok = true;
            for (int y = 0; y < NY && ok; ++y)
                for (int z = 0; z < NZ && ok; ++z, ++acc) {
                    if (acc > 0 && !mbar_wait(&ctl->acc_empty, (acc - 1) & 1, abort, wlim)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    for (int kb = z * ZB; kb < min(KB, (z + 1) * ZB) && ok; ++kb, ++qb) {
                        ok = mbar_wait(&ctl->b_full[qb & 1], (qb >> 1) & 1, abort, wlim);
                        if (!ok) break;
                        tc_fence_after();
                        // B is N-major (bit 16): 16 chi are 2048 bytes on, digit 8 starts block 4
                        ok = mma_block(ctl, abort, a_lo, qa, tmem, desc_lo_mn(smem_u32(B + (qb & 1) * B_NMAJ), 8192), 128u,
                                       (4 * 8192) >> 4, 1u << 16, kb == z * ZB, wlim);
                        mma_commit(&ctl->b_empty[qb & 1]);
                    }
                    if (ok) mma_commit(&ctl->acc_full);
                }
            if (*abort) {
                mma_commit(&ctl->drain);
                mbar_drain(&ctl->drain, 0, wlim);
            }
        }
    } else {
        const double *Ps = P + (long long)s * sP;
        const int *ce = cexp + (long long)s * pslots + p0;
        const int lp = pb * 128 + (warp & 3) * 32 + lane, hb = warp >> 2;
        unsigned qb = 0, acc = 0;
        bool ok = true;
        double r = 0.0;
        int most = COL_ZERO, found = 2 * COL_ZERO;   // exponents: of the terms that the scales allow, of the terms
        const int rx = rexp[t * TILE_PTS + lp];
        for (int y = 0; y < NY && ok; ++y) {
            const int b0 = y * NB, nb = min(NB, np - b0);
            // digits of P: thread = (chi row, phi quad), twice; zeros past the lists
            const int qd = threadIdx.x & 7;
            double sc[4] = {0.0, 0.0, 0.0, 0.0};
            int col = 0;
            if (qd * 4 < nb) {
                const int4 E = *reinterpret_cast<const int4 *>(ce + b0 + qd * 4);
                sc[0] = column_scale(E.x), sc[1] = column_scale(E.y), sc[2] = column_scale(E.z), sc[3] = column_scale(E.w);
                col = pids[p0 + b0 + qd * 4];
            }
            for (int z = 0; z < NZ && ok; ++z, ++acc) {
                for (int kb = z * ZB; kb < min(KB, (z + 1) * ZB); ++kb, ++qb) {
                    if (qb >= 2 && !mbar_wait_warp(&ctl->b_empty[qb & 1], ((qb >> 1) - 1) & 1, abort, wlim)) {
                        ok = false;
                        break;
                    }
                    unsigned char *Bk = B + (qb & 1) * B_NMAJ;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int a = (threadIdx.x + h * 256) >> 3;
                        double v[4] = {0.0, 0.0, 0.0, 0.0};
                        if (kb * 64 + a < nc && qd * 4 < nb) {
                            const double2 *p = reinterpret_cast<const double2 *>(
                                Ps + (long long)cids[c0 + kb * 64 + a] * nphi + col);
                            const double2 x = __ldg(p), y2 = __ldg(p + 1);
                            v[0] = x.x, v[1] = x.y, v[2] = y2.x, v[3] = y2.y;
                        }
                        unsigned long long u[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) u[e] = biased(v[e] * sc[e]);
#pragma unroll
                        for (int j = 0; j < ND; ++j) {
                            const uint2 x = make_uint2(digit_pair(digit(u[0], j), digit(u[1], j)),
                                                       digit_pair(digit(u[2], j), digit(u[3], j)));
                            *reinterpret_cast<uint2 *>(Bk + (j >> 1) * 8192 + sw128_offset(a, (j & 1) * 4 + (qd >> 1)) +
                                                       (qd & 1) * 8) = x;
                        }
                    }
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->b_full[qb & 1]);
                }
                ok = ok && __all_sync(0xffffffffu, mbar_wait(&ctl->acc_full, acc & 1, abort, wlim) && !*abort);
                tc_fence_after();
                if (!ok) break;
                for (int c = hb * 16; c < hb * 16 + 16 && c < nb; c += 8) {
                    float D[ND][8];
#pragma unroll
                    for (int l = 0; l < ND; ++l) tmem_ld8(tmem + l * NB + c + ((unsigned)((warp & 3) * 32) << 16), D[l]);
#pragma unroll
                    for (int h = 0; h < 8; h += 4)
                        if (c + h < nb) {
                            const int4 E4 = __ldg(reinterpret_cast<const int4 *>(ce + b0 + c + h));
                            const int E[4] = {E4.x, E4.y, E4.z, E4.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const double ph = __ldg(pval + (long long)(p0 + b0 + c + h + e) * TILE_PTS + lp);
                                double x = combine_levels(D, h + e);         // zero or at least 1 in size
                                const int fp = expo_field(ph), fx = expo_field(x), w = fp != 0 ? fp + E[e] : 2 * COL_ZERO;
                                most = max(most, w);
                                if (fx != 0) {
                                    found = max(found, w + fx);
                                    x = __hiloint2double(__double2hiint(x) + (E[e] - top) * (1 << 20), __double2loint(x));
                                }
                                r = fma(x, ph, r);
                            }
                        }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->acc_empty);
            }
        }
        // the two halves of the phi meet (warps 0-7 only: a barrier of their own)
        const int p = (warp & 3) * 32 + lane;
        const int gx = t / (nt * nt) * TILE + (lp >> 6), gy = (t / nt) % nt * TILE + ((lp >> 3) & 7),
                  gz = t % nt * TILE + (lp & 7);
        const bool inside = gx < n && gy < n && gz < n;
        if (hb == 1) {
            ctl->part[p] = r;
            ctl->most[p] = most;
            ctl->found[p] = found;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (hb == 0) {
            r += ctl->part[p];
            most = max(most, ctl->most[p]);
            found = max(found, ctl->found[p]);
            // the term of both scales, 2^(rx + E) phi, has x = 2^(2 SHIFT - 56)
            const bool lost = f64 || (rx != ROW_ZERO && most > COL_ZERO / 2 && found < most + 1023 + 2 * SHIFT - 56 - LOST_BITS);
            if (ok && inside && !lost)
                rho[(long long)s * n * n * n + ((long long)gx * n + gy) * n + gz] = top == COL_ZERO ? 0.0 : ldexp(r, 56 - 2 * SHIFT + rx + top);
            const unsigned b = __ballot_sync(0xffffffffu, inside && lost);
            if (lane == 0) ctl->lost[warp] = b;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        // those points in float64: short lists by a warp each, others one after the other by all eight
        // (threads along the phi quads, then the chi)
        const int G = nc * np <= 4096 ? 32 : 256, tid = threadIdx.x & (G - 1);
        const int nq = np / 4, lanes = nq > 16 ? 32 : nq > 8 ? 16 : 8, q0 = tid % lanes, a0 = tid / lanes;
        for (int w = 0, i = 0; w < 4; ++w)
            for (unsigned left = ctl->lost[w]; left != 0; left &= left - 1, ++i) {
                if (G == 32 && (i & 7) != warp) continue;
                const int lpl = pb * 128 + w * 32 + __ffs(left) - 1;
                double v = 0.0;
                for (int q = q0; q < nq; q += lanes) {
                    const double *Pq = Ps + pids[p0 + q * 4], *ph = pval + (long long)(p0 + q * 4) * TILE_PTS + lpl;
                    double x[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
                    for (int a = a0; a < nc; a += G / lanes) {
                        const double ch = __ldg(cval + (long long)(c0 + a) * TILE_PTS + lpl);
                        const double2 *pp = reinterpret_cast<const double2 *>(Pq + (long long)cids[c0 + a] * nphi);
                        const double2 y = __ldg(pp), z = __ldg(pp + 1);
                        x[0] = fma(ch, y.x, x[0]);
                        x[1] = fma(ch, y.y, x[1]);
                        x[2] = fma(ch, z.x, x[2]);
                        x[3] = fma(ch, z.y, x[3]);
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) v = fma(x[e], __ldg(ph + e * TILE_PTS), v);
                }
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (G == 256) {
                    if (lane == 0) ctl->part[warp] = v;
                    asm volatile("bar.sync 1, 256;" ::: "memory");
                    v = 0.0;
                    for (int u = 0; u < 8; ++u) v += ctl->part[u];
                    asm volatile("bar.sync 1, 256;" ::: "memory");
                }
                if (tid == 0) {
                    const int hx = t / (nt * nt) * TILE + (lpl >> 6), hy = (t / nt) % nt * TILE + ((lpl >> 3) & 7),
                              hz = t % nt * TILE + (lpl & 7);
                    rho[(long long)s * n * n * n + ((long long)hx * n + hy) * n + hz] = v;
                }
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
    if (threadIdx.x == 0 && ctl->abort) atomicExch(err, 1);
}

// ---- tables and scales --------------------------------------------------------------------------------
// largest |x| of every row of len values (bit pattern; bits zeroed before). blockIdx.y = row.
__global__ void __launch_bounds__(256) max64_kernel(const double *__restrict__ x, long long len,
                                                    unsigned long long *__restrict__ bits) {
    const double *p = x + (long long)blockIdx.y * len;
    unsigned long long m = 0;   // of non-negative doubles the bits order as the values, NaN last
#pragma unroll 4
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < len; i += gridDim.x * 256ll) {
        const unsigned long long v = (unsigned long long)__double_as_longlong(p[i]) & 0x7fffffffffffffffull;
        m = v > m ? v : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
        m = v > m ? v : m;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(&bits[blockIdx.y], m);
}

// exponent E of every slot, max |value| < 2^E, at least -900 (0 for a slot of zeros); one warp per slot
__global__ void __launch_bounds__(256) slot_exponent_kernel(const double *__restrict__ val, long long slots,
                                                            int *__restrict__ out) {
    const long long sl = blockIdx.x * 8ll + (threadIdx.x >> 5);
    if (sl >= slots) return;
    double m = 0.0;
    for (int i = threadIdx.x & 31; i < TILE_PTS; i += 32) m = fmax(m, fabs(val[sl * TILE_PTS + i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = 0;
    if (m > 0.0) frexp(m, &e);
    if ((threadIdx.x & 31) == 0) out[sl] = max(e, -900);
}

__global__ void value_exponents_kernel(const double *__restrict__ val, long long values, short *__restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < values; i += (long long)gridDim.x * blockDim.x)
        out[i] = (short)value_exponent(val[i]);
}

// digit tables of chi: function-major [digit][slot][512], each slot by its own scale
__global__ void chi_digits_fm_kernel(const double *__restrict__ val, long long values, const int *__restrict__ cexp,
                                     unsigned short *__restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < values; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long u = biased(ldexp(val[i], SHIFT - cexp[i / TILE_PTS]));
#pragma unroll
        for (int j = 0; j < ND; ++j) out[j * values + i] = (unsigned short)digit_pair(digit(u, j), 64u);
    }
}
// exponent E of every point of a tile, max over its chi of |value| < 2^E, at least -900 (ROW_ZERO where
// all are zero). One thread per point.
__global__ void __launch_bounds__(256) point_exponent_kernel(const double *__restrict__ val, const int *__restrict__ off,
                                                             int ntiles, int *__restrict__ out) {
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= (long long)ntiles * TILE_PTS) return;
    const int t = (int)(i / TILE_PTS), p = (int)(i % TILE_PTS);
    double m = 0.0;
    for (int sl = off[t]; sl < off[t + 1]; ++sl) m = fmax(m, fabs(val[(long long)sl * TILE_PTS + p]));
    int e = 0;
    if (m > 0.0) frexp(m, &e);
    out[i] = m > 0.0 ? max(e, -900) : ROW_ZERO;
}
// and point-major in chunks of 64 slots of a tile, zero padded, each point by its own scale:
// [digit][chunk][512][64]
__global__ void chi_digits_pm_kernel(const double *__restrict__ val, const int *__restrict__ off,
                                     const int *__restrict__ chunk_tile, const int *__restrict__ chunk_j, long long nchunks,
                                     const int *__restrict__ rexp, unsigned short *__restrict__ out) {
    const long long tot = nchunks * TILE_PTS * 64;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
        const long long ch = e / (TILE_PTS * 64);
        const int rem = (int)(e - ch * (TILE_PTS * 64)), p = rem / 64, t = chunk_tile[ch], sl = chunk_j[ch] * 64 + rem % 64;
        const int ex = rexp[t * TILE_PTS + p];
        const bool in = sl < off[t + 1] - off[t] && ex != ROW_ZERO;
        const unsigned long long u = biased(in ? ldexp(val[(long long)(off[t] + sl) * TILE_PTS + p], SHIFT - ex) : 0.0);
#pragma unroll
        for (int j = 0; j < ND; ++j) out[j * tot + e] = (unsigned short)digit_pair(digit(u, j), 64u);
    }
}

size_t smem64_int() { return 1024 + A_RING * A_TILE + 2 * B_KMAJ + TILE_PTS * (sizeof(double) + sizeof(short)) + sizeof(Shared64); }
size_t smem64_den() { return 1024 + A_RING * A_TILE + 2 * B_NMAJ + sizeof(Shared64); }

void max64(cudaStream_t st, const double *x, long long len, int rows, unsigned long long *bits) {
    check(cudaMemsetAsync(bits, 0, sizeof(unsigned long long) * rows, st), "memset max64");
    const long long per = std::max(8, 1216 / rows);
    max64_kernel<<<dim3((unsigned)std::max<long long>(1, std::min<long long>(per, (len + 1023) / 1024)), rows), 256, 0, st>>>(
        x, len, bits);
    check_launch("max64_kernel");
}

}  // namespace

// Digit tables and lists of a context: coff, poff on the host as on the device. False (and nothing made)
// when a tile's TMA rows would not fit 31 bits, a table holds values beyond any orbital's, or the tables
// would take more than half of the free memory: the contractions then run on the CUDA cores, as
// they did where only the float64 tables fit. G.pm is null where the density's do not fit beside
// the integrals'.
bool fp64_grid_build(cudaStream_t st, Mem &out, const TileSet<double> &chi, const TileSet<double> &phi,
                     const std::vector<int> &coff, const std::vector<int> &poff, bool quads, Fp64Grid &result) try {
    const int ntl = chi.ntiles;
    const long long slots = coff[ntl], values = slots * TILE_PTS;
    std::vector<int> tiles, first(ntl + 1, 0), ct, cj;
    std::vector<IItem> items;
    for (int t = 0; t < ntl; ++t) {
        const int nc = coff[t + 1] - coff[t], np = poff[t + 1] - poff[t], nch = (nc + 63) / 64;
        first[t + 1] = first[t] + nch;
        for (int j = 0; j < nch; ++j) ct.push_back(t), cj.push_back(j);
        if (nc == 0 || np == 0) continue;
        tiles.push_back(t);
        for (int c = 0; c < nc; c += 128)
            for (int b = 0; b < np; b += NB)
                items.push_back(IItem{t, coff[t] + c, std::min(128, nc - c), poff[t] + b, std::min(NB, np - b)});
    }
    const long long nchunks = first[ntl];
    if (tiles.empty() || ND * slots > 0x7fffffffll || ND * nchunks * TILE_PTS > 0x7fffffffll) return false;
    std::stable_sort(tiles.begin(), tiles.end(), [&](int a, int b) {
        return (long long)(coff[a + 1] - coff[a]) * (poff[a + 1] - poff[a]) >
               (long long)(coff[b + 1] - coff[b]) * (poff[b + 1] - poff[b]);
    });
    const long long pslots = poff[ntl];
    // 18 bytes per chi value function-major, as many and the padding point-major, 2 per phi value
    const size_t fm_bytes = (size_t)ND * values * 2 + (size_t)pslots * TILE_PTS * 2;
    const size_t pm_bytes = quads ? (size_t)ND * nchunks * TILE_PTS * 64 * 2 + (size_t)ntl * TILE_PTS * 4 : 0;
    size_t room = 0, total = 0;
    if (cudaMemGetInfo(&room, &total) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (fm_bytes > room / 2) return false;
    const bool make_pm = quads && fm_bytes + pm_bytes <= room / 2;
    Mem mem;
    Fp64Grid G;
    unsigned long long *bits = mem.alloc<unsigned long long>(2), h[2];
    max64(st, chi.val, values, 1, bits);
    max64(st, phi.val, pslots * TILE_PTS, 1, bits + 1);
    check(cudaMemcpyAsync(h, bits, sizeof h, cudaMemcpyDeviceToHost, st), "D2H table maxima");
    check(cudaStreamSynchronize(st), "sync table maxima");
    double m[2];
    static_assert(sizeof m == sizeof h, "bits of a double");
    std::memcpy(m, h, sizeof m);
    // tables with infinities, NaN or values beyond any orbital's stay on the CUDA cores
    if (!(m[0] < 1e100) || !(m[1] < 1e100)) return false;
    auto up = [&](const auto &v) {
        using E = typename std::decay<decltype(v[0])>::type;
        E *p = mem.alloc<E>(v.size());
        check(cudaMemcpy(p, v.data(), v.size() * sizeof(E), cudaMemcpyHostToDevice), "upload FP64 grid lists");
        return p;
    };
    G.slots = slots;
    G.fm = mem.alloc<unsigned short>((size_t)ND * values);
    G.cexp = mem.alloc<int>(slots);
    G.pexp = mem.alloc<short>((size_t)pslots * TILE_PTS);
    slot_exponent_kernel<<<(unsigned)((slots + 7) / 8), 256, 0, st>>>(chi.val, slots, G.cexp);
    check_launch("slot_exponent_kernel");
    value_exponents_kernel<<<8 * 152, 256, 0, st>>>(phi.val, pslots * TILE_PTS, G.pexp);
    check_launch("value_exponents_kernel");
    chi_digits_fm_kernel<<<8 * 1216, 256, 0, st>>>(chi.val, values, G.cexp, G.fm);
    check_launch("chi_digits_fm_kernel");
    G.items = up(items);
    G.nitems = (long long)items.size();
    if (make_pm) {
        G.nchunks = nchunks;
        G.pm = mem.alloc<unsigned short>((size_t)ND * nchunks * TILE_PTS * 64);
        Mem tmp;
        int *dct = tmp.alloc<int>(ct.size()), *dcj = tmp.alloc<int>(cj.size());
        check(cudaMemcpy(dct, ct.data(), ct.size() * sizeof(int), cudaMemcpyHostToDevice), "upload chunk tiles");
        check(cudaMemcpy(dcj, cj.data(), cj.size() * sizeof(int), cudaMemcpyHostToDevice), "upload chunk index");
        G.rexp = mem.alloc<int>((size_t)ntl * TILE_PTS);
        point_exponent_kernel<<<(unsigned)(((long long)ntl * TILE_PTS + 255) / 256), 256, 0, st>>>(chi.val, chi.off, ntl, G.rexp);
        check_launch("point_exponent_kernel");
        chi_digits_pm_kernel<<<8 * 1216, 256, 0, st>>>(chi.val, chi.off, dct, dcj, nchunks, G.rexp, G.pm);
        check_launch("chi_digits_pm_kernel");
        check(cudaStreamSynchronize(st), "sync digit tables");
        G.tiles = up(tiles);
        G.ntiles = (int)tiles.size();
        G.cfirst = up(first);
        G.covers = G.ntiles == ntl;
        G.pslots = pslots;
    }
    out.ptrs.insert(out.ptrs.end(), mem.ptrs.begin(), mem.ptrs.end());
    mem.ptrs.clear();
    result = G;
    return true;
} catch (const std::bad_alloc &) {
    return false;
}

// rho [k][n^3] of P [k][nchi][nphi] (16-byte aligned rows); exps: k (pslots + ntiles) words
void response_density_fp64(cudaStream_t st, const GridShape &g, const TileSet<double> &chi, const TileSet<double> &phi,
                           const Fp64Grid &G, int nphi, const double *P, long long sP, int k, double *rho,
                           int *exps, int *err) {
    if (k <= 0) return;
    ProfScope ps(st, ST_DENSITY, 2.0 * k * g.pair_points, 8.0 * (g.table_values + (double)k * g.n * g.n * g.n));
    if (!G.covers) check(cudaMemsetAsync(rho, 0, sizeof(double) * (size_t)k * g.n * g.n * g.n, st), "memset rho");
    int *top = exps + k * G.pslots;
    column_exponents_kernel<<<dim3(G.ntiles, k), 256, 0, st>>>(G.tiles, G.ntiles, chi.off, chi.ids, phi.off, phi.ids, nphi, P,
                                                              sP, G.pslots, exps, top);
    check_launch("column_exponents_kernel");
    CUtensorMap mx;
    if (!encode_map_2d(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, G.pm, 64ull, (unsigned long long)(ND * G.nchunks) * TILE_PTS,
                       128ull, 64, 128))
        throw CudaError{cudaErrorInvalidValue, "cuTensorMapEncodeTiled (density64)"};
    static const bool attr = [&]() {
        check(cudaFuncSetAttribute(density64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64_den()),
              "attr density64");
        return true;
    }();
    (void)attr;
    const long long blocks = 4LL * G.ntiles * k;
    if (blocks > 0x7fffffffll) throw CudaError{cudaErrorInvalidValue, "density64: too many blocks"};
    density64_kernel<<<(unsigned)blocks, THREADS64, smem64_den(), st>>>(
        mx, g.n, g.nt, k, G.ntiles, G.tiles, chi.off, chi.ids, chi.val, G.cfirst, G.nchunks, phi.off, phi.ids, phi.val, nphi, P,
        sP, G.rexp, exps, top, G.pslots, rho, err, active_wait_limit());
    check_launch("density64_kernel");
}

// out [k][nchi][nphi] of V [k][n^3]
void potential_integrals_fp64(cudaStream_t st, const GridShape &g, const TileSet<double> &chi, const TileSet<double> &phi,
                              const Fp64Grid &G, int nchi, int nphi, const double *V, int k, double *out,
                              int *err) {
    if (k <= 0) return;
    ProfScope ps(st, ST_INTEGRALS, 2.0 * k * g.pair_points,
                 8.0 * (g.table_values + (double)k * g.n * g.n * g.n + (double)k * nchi * nphi));
    check(cudaMemsetAsync(out, 0, sizeof(double) * (size_t)k * nchi * nphi, st), "memset(integrals)");
    CUtensorMap mx;
    if (!encode_map_2d(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, G.fm, (unsigned long long)TILE_PTS,
                       (unsigned long long)(ND * G.slots), (unsigned long long)TILE_PTS * 2, 64, 128))
        throw CudaError{cudaErrorInvalidValue, "cuTensorMapEncodeTiled (integrals64)"};
    static const bool attr = [&]() {
        check(cudaFuncSetAttribute(integrals64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64_int()),
              "attr integrals64");
        return true;
    }();
    (void)attr;
    const long long blocks = G.nitems * k;
    if (blocks > 0x7fffffffll) throw CudaError{cudaErrorInvalidValue, "integrals64: too many blocks"};
    integrals64_kernel<<<(unsigned)blocks, THREADS64, smem64_int(), st>>>(
        mx, g.n, g.nt, k, G.items, G.slots, chi.ids, chi.val, phi.ids, phi.val, G.cexp, G.pexp, nchi, nphi, V, g.dV, out, err,
        active_wait_limit());
    check_launch("integrals64_kernel");
}

}  // namespace tddft
