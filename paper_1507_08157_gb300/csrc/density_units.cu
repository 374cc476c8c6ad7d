// Response density of a system whose tiles' phi lists are whole aligned quads (four consecutive
// functions, the first a multiple of four: every set of four per atom), mixed precision:
//
//   rho_s(r) = sum_b phi_b(r) T_s[r][b],   T_s[r][b] = sum_a chi_a(r) P_s,ab     (Secs. II C, III A)
//
// as tcgen05 kind::f16 products. The persistent kernel walks items: a whole grid tile (512 points)
// whose chi come in chunks of at most 128, or half a tile (256 points) with up to 256 chi. Per chunk
// of chi, and for each chunk of at most 64 phi and each pair of states, it multiplies
//
//   A  [512 or 256 points][chi] float16, K-major, brought once by TMA from a chunked point-major
//      table and kept for all phi chunks and states (128 KB);
//   B  [chi][phi quad][2 states][4] float16, N-major, gathered by five warps into a ring of stages of
//      32 chi (8 KB); of a last state without a partner [chi][phi], half as wide;
//   D  one accumulator of up to 128 columns per 128 points, four in TMEM (512 columns); two groups
//      of four warps multiply each by phi, which they keep in registers across the states.
//
// The gather reads P from a float16 copy laid out [state pair][phi quad][chi][2][4], made first by
// one pass over P: a 16-byte piece serves two states, the pieces of one quad's consecutive chi lie
// next to each other (an atom's chi make one run), and no conversion remains in the loop. The
// chunks of a tile follow one another in one block and the thread that owns a point adds to it, so
// the sum over a tile's functions has one order and needs no atomics.
//
// Why this shape: the gather is the scarce part. Every piece of P goes through the load/store unit
// once per item, whatever the number of points, so an item takes as many points as TMEM holds
// accumulators for and two states share a piece. Versions with 8-byte pieces (one state), 256
// points an item and asynchronous copies took 60 cycles per 32 pieces and 1.26 ms where this takes
// 0.59; one that streamed chi from L2 for every state and converted float32 P in the gather
// took 1.55 ms (140 atoms, 10 states, 135^3, GB300).
// Measured (GB300, whole stage, CUDA events, before and after): 140 atoms, 4 + 9 functions each, 135^3,
// 10 states 1.59 and 0.59 ms; 200 atoms, 4 + 4, 0.1 per A^3, 120^3, 5 states 0.80 and 0.51; the same at
// 60 atoms, 90^3 3.08 and 0.12, at 20 atoms with 2 states 0.35 and 0.036 (those two took the per-tile
// kernel); 200 atoms, 4 + 9, 180^3, 4 states 1.87 and 1.26. Not bound by HBM (0.17 ms of tables at 140
// atoms): 5400 MMAs, 9900 warp loads of the gather and 710 accumulators per SM share 1.1 M cycles,
// and the epilogue's path per accumulator (TMEM loads and dependent multiply-adds) is the longest.
// A state without a partner takes half a pair's gather, MMAs and epilogue (three states of the 200
// atoms 0.43 and 0.36 ms). One state of a dense cluster takes the streaming kernel at the end.
#include "tc_common.cuh"
#include "tddft_internal.h"

#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

namespace tddft {

using namespace tc;

bool encode_map_2d(CUtensorMap *map, CUtensorMapDataType dt, const void *ptr, unsigned long long inner,
                   unsigned long long rows, unsigned long long row_bytes, unsigned box_inner, unsigned box_rows);

namespace {

constexpr int DU_THREADS = 768;      // warps 0-15 epilogue, 16 TMA, 17-21 gather, 22-23 MMA
constexpr int DU_GATHER = 5;         // gathering warps
constexpr int DU_ROWS = 32;          // chi of a B stage
constexpr int DU_STAGES = 12;        // B stages (8 KB); at least the eight of one pair on half a tile
constexpr int A_BYTES = 131072, B_STAGE = 8192;

struct __align__(8) DuShared {
    unsigned long long a_full[4];    // per 64 chi
    unsigned long long a_empty;
    unsigned long long b_full[DU_STAGES];
    unsigned long long b_empty[DU_STAGES];
    unsigned long long acc_full[4];
    unsigned long long acc_empty[4];
    unsigned long long drain[2];
    unsigned int tmem_base;
    int abort;
};

// float16 power-of-two scale of a state from the bits of its largest |P|: 2^-e with
// 2^(e-1) < max <= 2^e (1 for an all-zero or non-finite state)
__device__ __forceinline__ float state_scale(unsigned bits) {
    const float m = __uint_as_float(bits);
    int e = 0;
    if (!(m > 0.0f && isfinite(m))) return 1.0f;
    frexpf(m, &e);
    return ldexpf(1.0f, -e);
}

// PHI32: phi in float32 (at most 32 per unit, the same registers) instead of float16
template <bool PHI32>
__global__ void __launch_bounds__(DU_THREADS, 1) density_units_kernel(
    const __grid_constant__ CUtensorMap mX,   // chunked point-major chi [chunk * 512 + point][64] f16, box 64 x 256
    int n, int nt, int k, int groups, const DItem *__restrict__ list, int nitems, const DUnit *__restrict__ units,
    const int *__restrict__ cids, const int *__restrict__ pids, int nchi, const uint4 *__restrict__ P16, long long sP16,
    const unsigned short *__restrict__ phi_pmc, const float *__restrict__ pval, const float *__restrict__ scale,
    float *__restrict__ rho, int chunked, int adds, int *err, long long wlim) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<unsigned long long>(smem_raw) + 1023ull) & ~1023ull);
    unsigned char *A = base, *B = base + A_BYTES;
    DuShared *ctl = reinterpret_cast<DuShared *>(B + DU_STAGES * B_STAGE);
    volatile int *abort = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 4; ++i) {
            mbar_init(&ctl->a_full[i], 1);
            mbar_init(&ctl->acc_full[i], 1);
            mbar_init(&ctl->acc_empty[i], 4);
        }
        mbar_init(&ctl->a_empty, 2);
        for (int i = 0; i < DU_STAGES; ++i) {
            mbar_init(&ctl->b_full[i], 1);
            mbar_init(&ctl->b_empty[i], 2);
        }
        for (int i = 0; i < 2; ++i) mbar_init(&ctl->drain[i], 1);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 22) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = ctl->tmem_base;
    // work item it: list entry it / groups with the state pairs pairs g / groups .. of group it % groups
    const int pairs = (k + 1) / 2;
    auto pairs_of = [&](int it, int &q0, int &q1) {
        const int g = it % groups;
        q0 = (int)((long long)pairs * g / groups);
        q1 = (int)((long long)pairs * (g + 1) / groups);
    };

    // accumulator of block mh of pair q: one per block on a whole tile, two sets in turn on half a tile
    auto acc_of = [](int nmh, int q, int mh) { return nmh == 4 ? mh : (q & 1) * 2 + mh; };

    if (warp == 16) {
        if (lane == 0) {
            unsigned loads = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
                const DItem d = list[it / groups];
                for (int ui = d.u0; ui < d.u1 && ok; ++ui) {
                    const DUnit u = units[ui];
                    if (!(u.chi_use & DUnit::FIRST)) continue;
                    if (loads > 0 && !mbar_wait(&ctl->a_empty, (loads - 1) & 1, abort, wlim)) {
                        ok = false;
                        break;
                    }
                    ++loads;
                    const int KB = (u.nc + 63) / 64;
                    for (int kb = 0; kb < 4; ++kb) {
                        if (kb >= KB) {      // keeps the barriers' phases in step
                            mbar_arrive(&ctl->a_full[kb]);
                            continue;
                        }
                        mbar_expect_tx(&ctl->a_full[kb], d.nmh * 16384);
                        for (int h = 0; h < d.nmh / 2; ++h)
                            tma_load_2d(A + kb * d.nmh * 16384 + h * 32768, &mX, &ctl->a_full[kb], 0,
                                        (u.cch + kb) * TILE_PTS + d.point0 + h * 256);
                    }
                }
            }
            // after an abort, the loads already issued land before the block exits
            if (*abort && loads > 0)
                for (int kb = 0; kb < 4; ++kb) mbar_drain(&ctl->a_full[kb], (loads - 1) & 1, wlim);
        }
    } else if (warp >= 22) {
        // MMA issuers: warp 22 + i issues the products of the 128-point blocks of parity i. One issuing
        // thread takes about 120 cycles an MMA where the tensor pipe needs 64 (M 128, N 128, K 16).
        if (elect_one()) {
            const int par = warp & 1;
            const unsigned a_lo = desc_lo(smem_u32(A)), b_lo = desc_lo_mn(smem_u32(B), B_STAGE / 2);
            unsigned loads = 0, buse = 0;   // A loads, laps of the B ring so far
            unsigned uses[2] = {0, 0};      // of accumulators par and par + 2
            int bi = 0;                     // next B stage
            bool ok = true;
            for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
                const DItem d = list[it / groups];
                int q0, q1;
                pairs_of(it, q0, q1);
                for (int ui = d.u0; ui < d.u1 && ok; ++ui) {
                    const DUnit u = units[ui];
                    const int KS = (u.nc + DU_ROWS - 1) / DU_ROWS;
                    const int tail = u.nc - (KS - 1) * DU_ROWS;   // chi of the last stage
                    const unsigned idesc2 = idesc_f16(128, (u.np + 15) / 16 * 32) | (1u << 16);   // B is N-major
                    const unsigned idesc1 = idesc_f16(128, (u.np + 15) / 16 * 16) | (1u << 16);
                    if (u.chi_use & DUnit::FIRST) ++loads;
                    for (int q = q0; q < q1 && ok; ++q) {
                        const unsigned idesc = 2 * q + 1 < k ? idesc2 : idesc1;
                        for (int mh = par; mh < d.nmh; mh += 2) {
                            const int acc = acc_of(d.nmh, q, mh);
                            const unsigned d0 = tmem + acc * 128, au = acc >> 1 ? uses[1]++ : uses[0]++;
                            if (au > 0 && !mbar_wait(&ctl->acc_empty[acc], (au - 1) & 1, abort, wlim)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const bool last = mh + 2 >= d.nmh;
                            unsigned a = a_lo + mh * 1024, use = buse;
                            int st = bi;
                            for (int ks = 0; ks < KS; ++ks) {
                                if (mh == par) {   // the pair's stages (and, the first time, the chi blocks)
                                    if ((q == q0 && (u.chi_use & DUnit::FIRST) && (ks & 1) == 0 &&
                                         !mbar_wait(&ctl->a_full[ks >> 1], (loads - 1) & 1, abort, wlim)) ||
                                        !mbar_wait(&ctl->b_full[st], use & 1, abort, wlim)) {
                                        ok = false;
                                        break;
                                    }
                                    tc_fence_after();
                                }
                                const unsigned b = b_lo + st * (B_STAGE >> 4);
                                mma_f16(d0, desc_of(a), desc_of(b), idesc, ks > 0 ? 1u : 0u);
                                if (ks < KS - 1 || tail > 16) mma_f16(d0, desc_of(a + 2), desc_of(b + 128), idesc, 1u);
                                if (last) mma_commit(&ctl->b_empty[st]);
                                a += (ks & 1) ? d.nmh * 1024 - 4 : 4;
                                if (++st == DU_STAGES) st = 0, ++use;
                            }
                            if (!ok) break;
                            mma_commit(&ctl->acc_full[acc]);
                        }
                        bi += KS;
                        if (bi >= DU_STAGES) bi -= DU_STAGES, ++buse;
                    }
                    if (ok && (u.chi_use & DUnit::LAST)) mma_commit(&ctl->a_empty);
                }
            }
            // after an abort, the MMAs already issued finish before TMEM is freed
            if (*abort) {
                mma_commit(&ctl->drain[par]);
                mbar_drain(&ctl->drain[par], 0, wlim);
            }
        }
    } else if (warp >= 17) {
        // gather: B stage rows = 32 of the unit's chi (K), columns = its phi quads times two states. The
        // stages go to the warps in turn, a whole stage to one warp (lane = row, all quads), so that
        // waits, fence and arrival are paid once per stage.
        const int w = warp - 17;
        int bi = w, turn = 0;   // the warp's next stage; stage count modulo the warps
        unsigned buse = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
            const DItem d = list[it / groups];
            int q0, q1;
            pairs_of(it, q0, q1);
            for (int ui = d.u0; ui < d.u1 && ok; ++ui) {
                const DUnit u = units[ui];
                const int KS = (u.nc + DU_ROWS - 1) / DU_ROWS, nq = (u.np + 15) / 16 * 4;
                // lane j: the row of quad j in P16 (-1 past the list)
                const int qr = lane * 4 < u.np ? (pids[u.p0 + lane * 4] >> 2) * nchi : -1;
                for (int q = q0; q < q1 && ok; ++q) {
                    const uint4 *Ps = P16 + (long long)q * sP16;
                    for (int ks = 0; ks < KS; ++ks) {
                        const bool mine = turn == w;
                        turn = turn == DU_GATHER - 1 ? 0 : turn + 1;
                        if (!mine) continue;
                        const int a = ks * DU_ROWS + lane;
                        const int id = a < u.nc ? cids[u.c0 + a] : -1;
                        // rows past the list up to a multiple of 16 are read too: zeros
                        unsigned char *b = B + bi * B_STAGE + lane * 128;
                        const unsigned x = (lane & 7) << 4;
                        if (2 * q + 1 == k) {     // a state without a partner: pieces of two quads
                            const uint2 *Pl = reinterpret_cast<const uint2 *>(Ps);
                            uint4 v[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const int r0 = __shfl_sync(0xffffffffu, qr, 2 * j), r1 = __shfl_sync(0xffffffffu, qr, 2 * j + 1);
                                const uint2 y0 = (id >= 0 && r0 >= 0) ? __ldg(Pl + (r0 + id)) : make_uint2(0u, 0u);
                                const uint2 y1 = (id >= 0 && r1 >= 0) ? __ldg(Pl + (r1 + id)) : make_uint2(0u, 0u);
                                v[j] = make_uint4(y0.x, y0.y, y1.x, y1.y);
                            }
                            if (buse > 0) ok = mbar_wait_warp(&ctl->b_empty[bi], (buse - 1) & 1, abort, wlim);
                            if (ok)
#pragma unroll
                                for (int j = 0; j < 8; ++j)
                                    if (2 * j < nq) *reinterpret_cast<uint4 *>(b + ((j << 4) ^ x)) = v[j];
                        } else {
                            for (int h = 0; h * 8 < nq; ++h) {
                                uint4 v[8];
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    const int row = __shfl_sync(0xffffffffu, qr, h * 8 + j);
                                    v[j] = (id >= 0 && row >= 0) ? __ldg(Ps + (row + id)) : make_uint4(0u, 0u, 0u, 0u);
                                }
                                if (h == 0 && buse > 0 && !mbar_wait_warp(&ctl->b_empty[bi], (buse - 1) & 1, abort, wlim)) {
                                    ok = false;
                                    break;
                                }
#pragma unroll
                                for (int j = 0; j < 8; ++j)
                                    if (h * 8 + j < nq)
                                        *reinterpret_cast<uint4 *>(b + h * (B_STAGE / 2) + ((j << 4) ^ x)) = v[j];
                            }
                        }
                        if (!ok) break;
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&ctl->b_full[bi]);
                        bi += DU_GATHER;
                        if (bi >= DU_STAGES) {
                            bi -= DU_STAGES;
                            ++buse;
                        }
                    }
                }
            }
        }
    } else {
        // epilogue: group g takes accumulator g; a thread owns one point of an item and keeps its phi for
        // all states of a unit. Columns: per quad the four phi of the pair's first state, then of its
        // second. Sixteen warps, because a warp's path here is latency: loads out of TMEM and two
        // chains of fused multiply-adds.
        const int grp = warp >> 2;
        const long long n3 = (long long)n * n * n;
        unsigned uses = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
            const DItem d = list[it / groups];
            int q0, q1;
            pairs_of(it, q0, q1);
            const int lp = d.point0 + (d.nmh == 4 ? grp : grp & 1) * 128 + (warp & 3) * 32 + lane;
            const int gx = d.t / (nt * nt) * TILE + (lp >> 6), gy = (d.t / nt) % nt * TILE + ((lp >> 3) & 7),
                      gz = d.t % nt * TILE + (lp & 7);
            const bool inside = gx < n && gy < n && gz < n;
            float *out = rho + ((long long)gx * n + gy) * n + gz;
            for (int ui = d.u0; ui < d.u1 && ok; ++ui) {
                const int np = units[ui].np, ncol = (np + 15) / 16 * 32;
                unsigned ph[32];   // 64 float16 or 32 float32
                if (PHI32) {
                    const float *s = pval + (long long)units[ui].p0 * TILE_PTS + lp;
#pragma unroll
                    for (int b = 0; b < 32; ++b) ph[b] = b < np ? __float_as_uint(__ldg(s + b * TILE_PTS)) : 0u;
                } else {
                    const uint4 *s = reinterpret_cast<const uint4 *>(phi_pmc + ((long long)units[ui].pch * TILE_PTS + lp) * 32);
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        if (x < 4 || np > 32) {
                            const uint4 y = __ldg(s + (x >> 2) * (TILE_PTS * 4) + (x & 3));
                            ph[x * 4] = y.x;
                            ph[x * 4 + 1] = y.y;
                            ph[x * 4 + 2] = y.z;
                            ph[x * 4 + 3] = y.w;
                        }
                }
                for (int q = q0; q < q1; ++q) {
                    if (d.nmh == 2 && (q & 1) != grp >> 1) continue;
                    const int s0 = 2 * q, s1 = min(2 * q + 1, k - 1);
                    float *o0 = out + s0 * n3, *o1 = out + s1 * n3;
                    // a later unit of the tile goes on from the point's sums so far (scales are powers of two:
                    // exact), or, with `adds`, adds to them; chunked: dot products of 32 phi, added in
                    // order, else running sums
                    float t0 = 0.0f, t1 = 0.0f;
                    if (!adds && ui > d.u0 && inside) {
                        t0 = *o0 * scale[s0];
                        t1 = *o1 * scale[s1];
                    }
                    const float inv0 = scale[k + s0], inv1 = scale[k + s1];
                    ok = __all_sync(0xffffffffu, mbar_wait(&ctl->acc_full[grp], uses & 1, abort, wlim) && !*abort);
                    ++uses;
                    tc_fence_after();
                    if (!ok) break;
                    float r0 = chunked ? 0.0f : t0, r1 = chunked ? 0.0f : t1;
                    const unsigned ta = tmem + grp * 128 + ((unsigned)((warp & 3) * 32) << 16);
                    if (s1 == s0) {
                        // a state without a partner: column b is phi b
#pragma unroll
                        for (int c = 0; c < (PHI32 ? 2 : 4); ++c)
                            if (c * 32 < ncol) {
                                float v[16];
                                tmem_ld16(ta + c * 16, v);
#pragma unroll
                                for (int e = 0; e < 16; e += 2) {
                                    if (PHI32) {
                                        r0 = __fadd_rn(r0, __fmul_rn(v[e], __uint_as_float(ph[(c * 16 + e) & 31])));
                                        r0 = __fadd_rn(r0, __fmul_rn(v[e + 1], __uint_as_float(ph[(c * 16 + e + 1) & 31])));
                                    } else {
                                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&ph[c * 8 + e / 2]));
                                        r0 = fmaf(v[e], f.x, r0);
                                        r0 = fmaf(v[e + 1], f.y, r0);
                                    }
                                }
                                if (!PHI32 && chunked && ((c & 1) || (c + 1) * 32 >= ncol)) {
                                    t0 += r0;
                                    r0 = 0.0f;
                                }
                            }
                    } else
#pragma unroll
                    for (int c = 0; c < (PHI32 ? 4 : 8); ++c)
                        if (c * 16 < ncol) {
                            float v[16];
                            tmem_ld16(ta + c * 16, v);
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                float f[4];
                                if (PHI32) {
#pragma unroll
                                    for (int e = 0; e < 4; ++e) f[e] = __uint_as_float(ph[(c * 8 + j * 4 + e) & 31]);
                                } else {
                                    const float2 x = __half22float2(*reinterpret_cast<const __half2 *>(&ph[c * 4 + j * 2]));
                                    const float2 y = __half22float2(*reinterpret_cast<const __half2 *>(&ph[c * 4 + j * 2 + 1]));
                                    f[0] = x.x, f[1] = x.y, f[2] = y.x, f[3] = y.y;
                                }
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    if (PHI32) {   // rounded as in the per-tile kernel's float32 sums
                                        r0 = __fadd_rn(r0, __fmul_rn(v[8 * j + e], f[e]));
                                        r1 = __fadd_rn(r1, __fmul_rn(v[8 * j + 4 + e], f[e]));
                                    } else {
                                        r0 = fmaf(v[8 * j + e], f[e], r0);
                                        r1 = fmaf(v[8 * j + 4 + e], f[e], r1);
                                    }
                                }
                            }
                            if (!PHI32 && chunked && ((c & 3) == 3 || (c + 1) * 16 >= ncol)) {
                                t0 += r0, t1 += r1;
                                r0 = r1 = 0.0f;
                            }
                        }
                    if (!PHI32 && chunked) r0 = t0, r1 = t1;
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->acc_empty[grp]);
                    if (inside) {
                        if (adds) {
                            atomicAdd(o0, r0 * inv0);
                            if (s1 > s0) atomicAdd(o1, r1 * inv1);
                        } else {
                            *o0 = r0 * inv0;
                            if (s1 > s0) *o1 = r1 * inv1;
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 22) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
    if (threadIdx.x == 0 && ctl->abort) atomicExch(err, 1);
}

// largest |P_s| of every state (bit pattern; bits zeroed before). blockIdx.y = state.
__global__ void __launch_bounds__(256) max_bits_kernel(const float *__restrict__ P, long long len,
                                                       unsigned *__restrict__ bits) {
    const float *p = P + (long long)blockIdx.y * len;
    float m = 0.0f;
#pragma unroll 8
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < len; i += gridDim.x * 256ll) m = fmaxf(m, fabsf(p[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&bits[blockIdx.y], __float_as_uint(m));
}

// P16[s / 2][q][a][s % 2][4] = float16(P[s][a][4q .. 4q+3] * scale_s), the last state of an odd count
// [q][a][4]: 32 x 32 (chi, quad) tiles of a state pair through shared memory, both sides in rows
// of 16-byte pieces. scale [k] and its inverse [k] are left for the kernel.
__global__ void __launch_bounds__(256) pack_quads_kernel(const float *__restrict__ P, long long sP, int nchi, int nphi,
                                                         int k, const unsigned *__restrict__ bits,
                                                         uint4 *__restrict__ out, long long sout,
                                                         float *__restrict__ scale) {
    __shared__ uint4 t[32][33];
    const int sp = blockIdx.z, a0 = blockIdx.y * 32, q0 = blockIdx.x * 32, nq = nphi / 4;
    const int s0 = 2 * sp;
    const bool two = s0 + 1 < k;
    const float c0 = state_scale(bits[s0]), c1 = two ? state_scale(bits[s0 + 1]) : 1.0f;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
        scale[s0] = c0;
        scale[k + s0] = 1.0f / c0;
        if (two) {
            scale[s0 + 1] = c1;
            scale[k + s0 + 1] = 1.0f / c1;
        }
    }
    const float *Ps = P + (long long)s0 * sP;
    auto half4 = [](float4 v, float c) {
        const __half2 lo = __floats2half2_rn(v.x * c, v.y * c), hi = __floats2half2_rn(v.z * c, v.w * c);
        return make_uint2(*reinterpret_cast<const unsigned *>(&lo), *reinterpret_cast<const unsigned *>(&hi));
    };
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int a = a0 + i, q = q0 + threadIdx.x;
        if (a < nchi && q < nq) {
            const float4 *p = reinterpret_cast<const float4 *>(Ps + (long long)a * nphi) + q;
            const uint2 x = half4(*p, c0);
            const uint2 y = two ? half4(*reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(p) + sP), c1)
                                : make_uint2(0u, 0u);
            t[i][threadIdx.x] = make_uint4(x.x, x.y, y.x, y.y);
        }
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int q = q0 + i, a = a0 + threadIdx.x;
        if (a < nchi && q < nq) {
            const uint4 x = t[threadIdx.x][i];
            const long long o = (long long)q * nchi + a;
            if (two) out[(long long)sp * sout + o] = x;
            else reinterpret_cast<uint2 *>(out + (long long)sp * sout)[o] = make_uint2(x.x, x.y);
        }
    }
}

// ---- one state on dense tiles ---------------------------------------------------------------------------
// The kernel above keeps chi for all states, so that one state alone waits for each 128 KB of it. Where
// lists are long (no tile's chi fit one of its accumulations) one state is faster with chi streamed:
// units of at most 5 x 64 chi and 4 x 32 phi of a tile, each adding its part to rho with float32
// reductions. Persistent, one block per SM over (unit, state): warp 4 brings 128 points x 64 chi at a
// time by TMA through a ring, warp 5 issues the MMAs (M = 128 points, N = 128 phi, K = the unit's chi),
// warps 6-7 and 12-15 gather the next item's float32 P (scaled to float16) into the other B buffer, and
// two groups of four warps multiply their accumulator by phi. Every wait is bounded.
// Measured (entry point with its conversions, one state, the kernel above and this): clusters at 0.1
// atoms per A^3 with 4 + 4 functions, 200 atoms 295 and 264 us, 150 atoms 164 and 146; 110 atoms with 4 + 9
// 172 and 155. With five states of 200 atoms the kernel above is the faster (0.88 and 0.59 ms). Lists that
// fit the per-tile kernels keep the items (no line between the two was looked for among them).
constexpr int DS_THREADS = 512, DS_GATHER = 192, DS_STAGES = 4;
constexpr int DS_KB = 5, DS_NB = 128;      // chi blocks of 64 and phi of a unit
struct __align__(8) DsShared {
    unsigned long long a_full[DS_STAGES], a_empty[DS_STAGES];
    unsigned long long acc_full[2], acc_empty[2];
    unsigned long long b_full[2], b_free[2];
    unsigned long long drain;
    unsigned int tmem_base;
    int abort;
};

__global__ void __launch_bounds__(DS_THREADS, 1) density_stream_kernel(
    const __grid_constant__ CUtensorMap mX,   // [chi chunk * 512 + point][64] f16, box 64 x 128
    int n, int nt, int k, const DUnit *__restrict__ units, int nitems, const int *__restrict__ cids,
    const int *__restrict__ pids, int nphi, const unsigned short *__restrict__ phi_pmc,
    const float *__restrict__ P, long long sP, const unsigned *__restrict__ bits, float *__restrict__ rho,
    int *err, long long wlim) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<unsigned long long>(smem_raw) + 1023ull) & ~1023ull);
    constexpr int NB = DS_NB;
    unsigned char *A = base;                                      // ring [STAGES][128 x 128 B]
    unsigned char *Bb = base + DS_STAGES * 16384;              // [2][DS_KB][NB x 128 B]
    constexpr size_t bsize = (size_t)DS_KB * NB * 128;
    DsShared *ctl = reinterpret_cast<DsShared *>(Bb + 2 * bsize);
    volatile int *abort = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n3 = (long long)n * n * n;
    if (threadIdx.x == 0) {
        for (int i = 0; i < DS_STAGES; ++i) {
            mbar_init(&ctl->a_full[i], 1);
            mbar_init(&ctl->a_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&ctl->acc_full[i], 1);
            mbar_init(&ctl->acc_empty[i], 128);
            mbar_init(&ctl->b_full[i], DS_GATHER);
            mbar_init(&ctl->b_free[i], 1);
        }
        mbar_init(&ctl->drain, 1);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(256));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = ctl->tmem_base;

    if (warp == 4) {
        if (lane == 0) {
            long long q = 0;
            for (int it = blockIdx.x; it < nitems && !*abort; it += gridDim.x) {
                const DUnit u = units[it / k];
                const int KB = (u.nc + 63) / 64;
                for (int pb = 0; pb < TILE_PTS / 128; ++pb)
                    for (int kb = 0; kb < KB; ++kb, ++q) {
                        const int st = (int)(q % DS_STAGES);
                        const long long use = q / DS_STAGES;
                        if (use > 0 && !mbar_wait(&ctl->a_empty[st], (unsigned)((use - 1) & 1), abort, wlim)) break;
                        mbar_expect_tx(&ctl->a_full[st], 16384);
                        tma_load_2d(A + st * 16384, &mX, &ctl->a_full[st], 0, (u.cch + kb) * TILE_PTS + pb * 128);
                    }
            }
            if (*abort)
                for (long long j = q > DS_STAGES ? q - DS_STAGES : 0; j < q; ++j)
                    mbar_drain(&ctl->a_full[j % DS_STAGES], (unsigned)((j / DS_STAGES) & 1), wlim);
        }
    } else if (warp == 5) {
        if (lane == 0) {
            const unsigned idesc = idesc_f16(128, NB);
            long long q = 0, pbg = 0;
            int j = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x, ++j) {
                const DUnit u = units[it / k];
                const int KB = (u.nc + 63) / 64;
                const int buf = j & 1;
                if (!mbar_wait(&ctl->b_full[buf], (unsigned)((j >> 1) & 1), abort, wlim)) break;
                tc_fence_after();
                const unsigned char *B = Bb + buf * bsize;
                for (int pb = 0; pb < TILE_PTS / 128 && ok; ++pb, ++pbg) {
                    const int acc = (int)(pbg & 1);
                    const long long ause = pbg >> 1;
                    if (ause > 0 && !mbar_wait(&ctl->acc_empty[acc], (unsigned)((ause - 1) & 1), abort, wlim)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    for (int kb = 0; kb < KB; ++kb, ++q) {
                        const int st = (int)(q % DS_STAGES);
                        if (!mbar_wait(&ctl->a_full[st], (unsigned)((q / DS_STAGES) & 1), abort, wlim)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const unsigned a = smem_u32(A + st * 16384), bb = smem_u32(B + (size_t)kb * NB * 128);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_f16(tmem + acc * 128, smem_desc(a + kk * 32), smem_desc(bb + kk * 32), idesc,
                                    (kb > 0 || kk > 0) ? 1u : 0u);
                        mma_commit(&ctl->a_empty[st]);
                    }
                    if (!ok) break;
                    mma_commit(&ctl->acc_full[acc]);
                }
                if (!ok) break;
                mma_commit(&ctl->b_free[buf]);
            }
            if (*abort) {
                mma_commit(&ctl->drain);
                mbar_drain(&ctl->drain, 0, wlim);
            }
        }
    } else if ((warp >= 6 && warp < 8) || warp >= 12) {
        // the P block of each item (rows = the unit's phi, K = its chi) by phi quads, zeros past
        // the unit's counts (every row and K column of the buffer is written)
        const int rank = (warp < 8 ? warp - 6 : warp - 10) * 32 + lane;   // warps 6, 7, 12-15: 0 .. 191
        int j = 0;
        for (int it = blockIdx.x; it < nitems; it += gridDim.x, ++j) {
            const DUnit u = units[it / k];
            const int s = it % k;
            const int KB = (u.nc + 63) / 64;
            const int buf = j & 1;
            if (j >= 2 && !mbar_wait_warp(&ctl->b_free[buf], (unsigned)(((j >> 1) - 1) & 1), abort, wlim)) break;
            unsigned char *B = Bb + buf * bsize;
            const float sc = state_scale(bits[s]);
            const float *Ps = P + (long long)s * sP;
            constexpr int nq = NB / 4;
            const int total = nq * KB * 8;
            for (int i0 = rank; i0 < total; i0 += 2 * DS_GATHER) {
                float4 v[2][8];
#pragma unroll
                for (int uu = 0; uu < 2; ++uu) {
                    const int idx = i0 + uu * DS_GATHER;
                    const int qd = idx % nq, ch = idx / nq;
                    const bool live = idx < total && qd * 4 < u.np;
                    const float *Pq = Ps + (live ? pids[u.p0 + qd * 4] : 0);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int a = (ch >> 3) * 64 + (ch & 7) * 8 + e;
                        v[uu][e] = (live && a < u.nc)
                                       ? __ldg(reinterpret_cast<const float4 *>(Pq + (long long)cids[u.c0 + a] * nphi))
                                       : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    }
                }
#pragma unroll
                for (int uu = 0; uu < 2; ++uu) {
                    const int idx = i0 + uu * DS_GATHER;
                    if (idx >= total) continue;
                    const int qd = idx % nq, ch = idx / nq;
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        unsigned short h[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float x = r == 0 ? v[uu][e].x : r == 1 ? v[uu][e].y : r == 2 ? v[uu][e].z : v[uu][e].w;
                            h[e] = __half_as_ushort(__float2half_rn(x * sc));
                        }
                        uint4 qv;
                        qv.x = h[0] | ((unsigned)h[1] << 16);
                        qv.y = h[2] | ((unsigned)h[3] << 16);
                        qv.z = h[4] | ((unsigned)h[5] << 16);
                        qv.w = h[6] | ((unsigned)h[7] << 16);
                        *reinterpret_cast<uint4 *>(B + (size_t)(ch >> 3) * NB * 128 + sw128_offset(qd * 4 + r, ch & 7)) = qv;
                    }
                }
            }
            fence_async_smem();
            mbar_arrive(&ctl->b_full[buf]);
        }
    } else {
        // epilogue groups: warps 0-3 accumulator 0 (even point blocks), warps 8-11 accumulator 1
        const int eg = warp < 4 ? 0 : 1, quarter = warp & 3;
        long long ause = 0;
        for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
            const DUnit u = units[it / k];
            const int s = it % k;
            const int tx = u.t / (nt * nt), ty = (u.t / nt) % nt, tz = u.t % nt;
            const float inv = 1.0f / state_scale(bits[s]);
            bool stop = false;
            for (int pb = eg; pb < TILE_PTS / 128; pb += 2, ++ause) {
                const bool ok = __all_sync(0xffffffffu, mbar_wait(&ctl->acc_full[eg], (unsigned)(ause & 1), abort, wlim) && !*abort);
                tc_fence_after();
                const int lp = pb * 128 + quarter * 32 + lane;
                float r = 0.0f;
                if (ok) {
                    for (int c = 0; c < u.np; c += 32) {
                        const uint4 *q = reinterpret_cast<const uint4 *>(
                            phi_pmc + ((long long)(u.pch + c / 32) * TILE_PTS + lp) * 32);
                        uint4 ph[4];
#pragma unroll
                        for (int w = 0; w < 4; ++w) ph[w] = __ldg(q + w);
                        float v[32];
                        tmem_ld32(tmem + eg * 128 + ((unsigned)(quarter * 32) << 16) + (unsigned)c, v);
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            const __half2 *hh = reinterpret_cast<const __half2 *>(&ph[w]);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 f2 = __half22float2(hh[e]);
                                r = fmaf(v[8 * w + 2 * e], f2.x, r);
                                r = fmaf(v[8 * w + 2 * e + 1], f2.y, r);
                            }
                        }
                    }
                }
                tc_fence_before();
                mbar_arrive(&ctl->acc_empty[eg]);
                if (!ok) {
                    stop = true;
                    break;
                }
                const int gx = tx * TILE + (lp >> 6), gy = ty * TILE + ((lp >> 3) & 7), gz = tz * TILE + (lp & 7);
                if (gx < n && gy < n && gz < n)
                    atomicAdd(rho + (long long)s * n3 + ((long long)gx * n + gy) * n + gz, r * inv);
            }
            if (stop) break;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
    }
    if (threadIdx.x == 0 && ctl->abort) atomicExch(err, 1);
}
size_t density_stream_smem() { return 1024 + (size_t)DS_STAGES * 16384 + 2 * (size_t)DS_KB * DS_NB * 128 + sizeof(DsShared); }

size_t density_units_smem() { return 1024 + A_BYTES + (size_t)DU_STAGES * B_STAGE + sizeof(DuShared); }

}  // namespace

// rho [k][n^3] of P [k][nchi][nphi] (16-byte aligned, nphi and sP multiples of 4). P16: scratch of
// 2 ceil(k / 2) nchi nphi float16; bits: k words; scale: 2 k words.
void response_density_units(cudaStream_t st, const GridShape &g, const TileSet<float> &chi, const TileSet<float> &phi,
                            const unsigned short *chi_pmc, long long nchunks_chi, const unsigned short *phi_pmc,
                            const DUnitList &ul, int nchi, int nphi, const float *P, long long sP, int k, float *rho,
                            unsigned short *P16, unsigned *bits, float *scale, int *err) {
    if (k <= 0) return;
    if (!P16) throw CudaError{cudaErrorInvalidValue, "density units: no scratch for the packed kernels"};
    ProfScope ps(st, ST_DENSITY, 2.0 * k * g.pair_points, 2.0 * g.table_values + 4.0 * k * g.n * g.n * g.n);
    const long long n3 = (long long)g.n * g.n * g.n;
    if (!ul.covers || ul.adds) check(cudaMemsetAsync(rho, 0, sizeof(float) * (size_t)k * n3, st), "memset rho");
    if (ul.nitems == 0) return;
    check(cudaMemsetAsync(bits, 0, sizeof(unsigned) * k, st), "memset maxabs");
    const int per = std::max(8, 1216 / k);
    max_bits_kernel<<<dim3((unsigned)std::min<long long>(per, (sP + 2047) / 2048), k), 256, 0, st>>>(P, sP, bits);
    check_launch("max_bits_kernel");
    const long long s16 = (long long)nchi * (nphi / 4);
    const int pairs = (k + 1) / 2;
    pack_quads_kernel<<<dim3((nphi / 4 + 31) / 32, (nchi + 31) / 32, pairs), dim3(32, 8), 0, st>>>(
        P, sP, nchi, nphi, k, bits, reinterpret_cast<uint4 *>(P16), s16, scale);
    check_launch("pack_quads_kernel");
    CUtensorMap mx;
    if (!encode_map_2d(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, chi_pmc, 64ull, (unsigned long long)nchunks_chi * TILE_PTS,
                       128ull, 64, 256))
        throw CudaError{cudaErrorInvalidValue, "cuTensorMapEncodeTiled (density units)"};
    static const bool attr = [&]() {
        check(cudaFuncSetAttribute(density_units_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)density_units_smem()),
              "attr density_units");
        check(cudaFuncSetAttribute(density_units_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)density_units_smem()),
              "attr density_units");
        return true;
    }();
    (void)attr;
    int dev = 0, sms = 0;
    check(cudaGetDevice(&dev), "cudaGetDevice");
    check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
    // an item keeps its chi for all states; only where that leaves fewer than eight items per SM are
    // the pairs cut into groups, so that the last round of items stays a small part
    const int groups = (int)std::min<long long>(pairs, std::max<long long>(1, (8LL * sms + ul.nitems - 1) / ul.nitems));
    const long long nitems = (long long)ul.nitems * groups;
    if (nitems > (1LL << 31) - 1) throw CudaError{cudaErrorInvalidValue, "density units: too many items"};
    auto kern = ul.phi32 ? density_units_kernel<true> : density_units_kernel<false>;
    kern<<<(int)std::min<long long>(sms, nitems), DU_THREADS, density_units_smem(), st>>>(
        mx, g.n, g.nt, k, groups, ul.items, (int)nitems, ul.units, chi.ids, phi.ids, nchi,
        reinterpret_cast<const uint4 *>(P16), s16, phi_pmc, phi.val, scale, rho, ul.chunked ? 1 : 0, ul.adds ? 1 : 0, err,
        active_wait_limit());
    check_launch("density_units_kernel");
}

// rho [k][n^3] of P [k][nchi][nphi] by the streaming kernel (P rows 16-byte aligned); units: at most 320 chi
// and 128 phi of a tile each; bits: k words.
void response_density_stream(cudaStream_t st, const GridShape &g, const TileSet<float> &chi, const TileSet<float> &phi,
                             const unsigned short *chi_pmc, long long nchunks_chi, const unsigned short *phi_pmc,
                             const DUnit *units, int nunits, int nphi, const float *P, long long sP, int k, float *rho,
                             unsigned *bits, int *err) {
    if (k <= 0) return;
    ProfScope ps(st, ST_DENSITY, 2.0 * k * g.pair_points, 2.0 * g.table_values + 4.0 * k * g.n * g.n * g.n);
    check(cudaMemsetAsync(rho, 0, sizeof(float) * (size_t)k * g.n * g.n * g.n, st), "memset rho");
    const long long nitems = (long long)nunits * k;
    if (nitems == 0) return;
    if (nitems > (1LL << 31) - 1) throw CudaError{cudaErrorInvalidValue, "density stream: too many items"};
    check(cudaMemsetAsync(bits, 0, sizeof(unsigned) * k, st), "memset maxabs");
    const int per = std::max(8, 1216 / k);
    max_bits_kernel<<<dim3((unsigned)std::min<long long>(per, (sP + 2047) / 2048), k), 256, 0, st>>>(P, sP, bits);
    check_launch("max_bits_kernel");
    CUtensorMap mx;
    if (!encode_map_2d(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, chi_pmc, 64ull, (unsigned long long)nchunks_chi * TILE_PTS,
                       128ull, 64, 128))
        throw CudaError{cudaErrorInvalidValue, "cuTensorMapEncodeTiled (density stream)"};
    static const bool attr = [&]() {
        check(cudaFuncSetAttribute(density_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)density_stream_smem()),
              "attr density_stream");
        return true;
    }();
    (void)attr;
    int dev = 0, sms = 0;
    check(cudaGetDevice(&dev), "cudaGetDevice");
    check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
    density_stream_kernel<<<(int)std::min<long long>(sms, nitems), DS_THREADS, density_stream_smem(), st>>>(
        mx, g.n, g.nt, k, units, (int)nitems, chi.ids, phi.ids, nphi, phi_pmc, P, sP, bits, rho, err, active_wait_limit());
    check_launch("density_stream_kernel");
}

}  // namespace tddft
