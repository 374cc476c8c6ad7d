// Potential integrals of a system whose tiles' phi lists are whole aligned quads (four consecutive
// functions, the first a multiple of four), mixed precision:
//
//   V_s,ab = dV sum_r chi_a(r) V_s(r) phi_b(r)      (Eqs. operator_TDA / operator_RPA)
//
// as tcgen05 kind::f16 products per grid tile, D[a][(s, b)] = sum_r X[a][r] W[(s, b)][r] with
// W = V_s(r) phi_b(r) and K = the tile's 512 points. The persistent kernel walks items (tile, at most
// 128 of its chi, group of states) and, inside an item, chunks of at most 48 phi and pairs of states:
//
//   X  [128 chi][512 points] float16, K-major in eight slices of 64 points, brought by TMA from the
//      function-major table once per item (128 KB); a slice is refilled for the next item as soon
//      as the last pair is past it;
//   phi in registers: producer warp w holds the chunk's phi on the 64 points of slice w and writes
//      W's slice w for every pair of states into a stage of its own (12 KB, K-major);
//   D  one accumulator of 2 x 48 columns per pair, four in TMEM, added to the output by two groups
//      of four warps in turn.
//
// The output of the reduction is laid out [state][phi quad][chi][4], so that the 16-byte additions
// of consecutive chi fall into the same sectors (an atom's chi make one run), and is put in row
// order by one pass at the end.
//
// Why this shape: with one (tile, state) per block every state re-read X and phi from L2 (12 GB a
// call at 140 atoms and 10 states), scaled phi in place between the copy and the MMAs, and spread its
// additions over one sector each. Here X and phi are read once per item, and V (2 KB a state) is all
// that streams.
// Measured (GB300, whole stage, CUDA events, before and after): 140 atoms, 4 + 9 functions each, 135^3,
// 10 states 1.68 and 0.77 ms, 7 states 1.20 and 0.64; 200 atoms, 180^3, 4 states 3.58 and 1.70; 20
// atoms, 90^3, 2 states 0.044 and 0.037. At 140 atoms no unit is at its limit: tensor pipe 26 % (N = 96),
// L1 and shared memory 43 % (X is read once per pair of states), L2's reductions 15 % (1.28 GB in 16-byte
// pieces), issue slots 46 %; the warps wait for loads, out of TMEM above all.
#include "tc_common.cuh"
#include "tddft_internal.h"

#include <cuda_fp16.h>

#include <algorithm>

namespace tddft {

using namespace tc;

bool encode_map_2d(CUtensorMap *map, CUtensorMapDataType dt, const void *ptr, unsigned long long inner,
                   unsigned long long rows, unsigned long long row_bytes, unsigned box_inner, unsigned box_rows);

namespace {

constexpr int IU_THREADS = 576;      // warps 0-7 produce W, 8-15 epilogue, 16 TMA, 17 MMA
constexpr int SLICES = 8;            // 64-point K slices of a tile, and stages of W
constexpr int IU_PHI = 48;           // most phi of a chunk
constexpr int X_SLICE = 16384, W_STAGE = 2 * IU_PHI * 128;

struct __align__(8) IuShared {
    unsigned long long x_full[SLICES];
    unsigned long long x_empty[SLICES];
    unsigned long long w_full[SLICES];
    unsigned long long w_empty[SLICES];
    unsigned long long acc_full[4];
    unsigned long long acc_empty[4];
    unsigned long long drain;
    unsigned int tmem_base;
    int abort;
};

// float16 power-of-two scale of a state from the bits of its largest |V| (as the density's)
__device__ __forceinline__ float v_scale(unsigned bits) {
    const float m = __uint_as_float(bits);
    int e = 0;
    if (!(m > 0.0f && isfinite(m))) return 1.0f;
    frexpf(m, &e);
    return ldexpf(1.0f, -e);
}

__device__ __forceinline__ void red_add_v4(float *addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

// phi chunk y of mp of a list of np: whole groups of 16, evenly cut
__device__ __forceinline__ void phi_chunk(int np, int mp, int y, int &b0, int &nb) {
    const int g = (np + 15) / 16;
    b0 = g * y / mp * 16;
    nb = min(g * (y + 1) / mp * 16, np) - b0;
}

__global__ void __launch_bounds__(IU_THREADS, 1) integrals_units_kernel(
    const __grid_constant__ CUtensorMap mX,   // function-major chi [slot][512] f16, box 64 points x 128 slots
    int n, int nt, int k, int groups, int pch, const IItem *__restrict__ list, int nitems, const int *__restrict__ cids,
    const int *__restrict__ pids, int nchi, int nquads, const unsigned short *__restrict__ phi_fm,
    const float *__restrict__ V, const unsigned *__restrict__ bits, float dV, float *__restrict__ out, int *err,
    long long wlim) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<unsigned long long>(smem_raw) + 1023ull) & ~1023ull);
    unsigned char *X = base, *W = base + SLICES * X_SLICE;
    IuShared *ctl = reinterpret_cast<IuShared *>(W + SLICES * W_STAGE);
    volatile int *abort = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n3 = (long long)n * n * n;
    if (threadIdx.x == 0) {
        for (int i = 0; i < SLICES; ++i) {
            mbar_init(&ctl->x_full[i], 1);
            mbar_init(&ctl->x_empty[i], 1);
            mbar_init(&ctl->w_full[i], 1);
            mbar_init(&ctl->w_empty[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(&ctl->acc_full[i], 1);
            mbar_init(&ctl->acc_empty[i], 4);
        }
        mbar_init(&ctl->drain, 1);
        ctl->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 17) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = ctl->tmem_base;
    // work item it: list entry it / groups with the state pairs of group it % groups
    const int pairs = (k + 1) / 2;
    auto pairs_of = [&](int it, int &q0, int &q1) {
        const int g = it % groups;
        q0 = (int)((long long)pairs * g / groups);
        q1 = (int)((long long)pairs * (g + 1) / groups);
    };

    if (warp == 16) {
        if (lane == 0) {
            unsigned loads = 0;
            int sl = 0;
            for (int it = blockIdx.x; it < nitems && !*abort; it += gridDim.x, ++loads) {
                const IItem d = list[it / groups];
                for (sl = 0; sl < SLICES; ++sl) {
                    if (loads > 0 && !mbar_wait(&ctl->x_empty[sl], (loads - 1) & 1, abort, wlim)) break;
                    mbar_expect_tx(&ctl->x_full[sl], X_SLICE);
                    tma_load_2d(X + sl * X_SLICE, &mX, &ctl->x_full[sl], sl * 64, d.c0);
                }
            }
            // after an abort, the loads already issued land before the block exits: the last of every slice
            // (loads counts the item whose slices 0 .. sl - 1 were issued last)
            if (*abort && loads > 0)
                for (int i = 0; i < SLICES; ++i) {
                    if (i < sl) mbar_drain(&ctl->x_full[i], (loads - 1) & 1, wlim);
                    else if (loads > 1) mbar_drain(&ctl->x_full[i], (loads - 2) & 1, wlim);
                }
        }
    } else if (warp == 17) {
        // MMA issuer
        if (elect_one()) {
            const unsigned x_lo = desc_lo(smem_u32(X)), w_lo = desc_lo(smem_u32(W));
            unsigned loads = 0, j = 0;   // items and pairs so far
            bool ok = true;
            for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x, ++loads) {
                const int np = list[it / groups].np, mp = (np + pch - 1) / pch;
                int q0, q1;
                pairs_of(it, q0, q1);
                for (int y = 0; y < mp && ok; ++y) {
                    int b0, nb;
                    phi_chunk(np, mp, y, b0, nb);
                    const unsigned idesc = idesc_f16(128, (nb + 15) / 16 * 32);
                    for (int q = q0; q < q1 && ok; ++q, ++j) {
                        const bool first = y == 0 && q == q0, last = y == mp - 1 && q == q1 - 1;
                        const unsigned acc = j & 3, au = j >> 2;
                        if (au > 0 && !mbar_wait(&ctl->acc_empty[acc], (au - 1) & 1, abort, wlim)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const unsigned d0 = tmem + acc * 128;
#pragma unroll
                        for (unsigned sl = 0; sl < SLICES; ++sl) {
                            if ((first && !mbar_wait(&ctl->x_full[sl], loads & 1, abort, wlim)) ||
                                !mbar_wait(&ctl->w_full[sl], j & 1, abort, wlim)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const unsigned x = x_lo + sl * (X_SLICE >> 4), w = w_lo + sl * (W_STAGE >> 4);
                            mma_f16(d0, desc_of(x), desc_of(w), idesc, sl > 0 ? 1u : 0u);
                            mma_f16(d0, desc_of(x + 2), desc_of(w + 2), idesc, 1u);
                            mma_f16(d0, desc_of(x + 4), desc_of(w + 4), idesc, 1u);
                            mma_f16(d0, desc_of(x + 6), desc_of(w + 6), idesc, 1u);
                            mma_commit(&ctl->w_empty[sl]);
                            if (last) mma_commit(&ctl->x_empty[sl]);
                        }
                        if (ok) mma_commit(&ctl->acc_full[acc]);
                    }
                }
            }
            // after an abort, the MMAs already issued finish before TMEM is freed
            if (*abort) {
                mma_commit(&ctl->drain);
                mbar_drain(&ctl->drain, 0, wlim);
            }
        }
    } else if (warp < 8) {
        // producer of slice `warp`: lane = octet of points (lane & 7) and phi rows (lane >> 3) + 4 i
        const int o = lane & 7, r = lane >> 3;
        unsigned j = 0;
        for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
            const IItem d = list[it / groups];
            const int mp = (d.np + pch - 1) / pch;
            int q0, q1;
            pairs_of(it, q0, q1);
            const int gx = d.t / (nt * nt) * TILE + warp, gy = (d.t / nt) % nt * TILE + o, gz = d.t % nt * TILE;
            const bool row_in = gx < n && gy < n;
            const float *vp = V + ((long long)gx * n + gy) * n + gz;
            for (int y = 0; y < mp; ++y) {
                int b0, nb;
                phi_chunk(d.np, mp, y, b0, nb);
                const int NB = (nb + 15) / 16 * 16;
                uint4 ph[IU_PHI / 4];
                const uint4 *pp = reinterpret_cast<const uint4 *>(phi_fm + (long long)(d.p0 + b0 + r) * TILE_PTS + warp * 64) + o;
#pragma unroll
                for (int i = 0; i < IU_PHI / 4; ++i)
                    if (r + 4 * i < nb) ph[i] = __ldg(pp + i * (4 * TILE_PTS / 8));
                for (int q = q0; q < q1; ++q, ++j) {
                    const int s0 = 2 * q, s1 = min(2 * q + 1, k - 1);
                    float v0[8], v1[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const bool in = row_in && gz + e < n;
                        v0[e] = in ? __ldg(vp + s0 * n3 + e) : 0.0f;
                        v1[e] = in ? __ldg(vp + s1 * n3 + e) : 0.0f;
                    }
                    const float c0 = v_scale(bits[s0]), c1 = v_scale(bits[s1]);
#pragma unroll
                    for (int e = 0; e < 8; ++e) v0[e] *= c0, v1[e] *= c1;
                    // after an abort the warp walks on to the end without waiting: its stores stay inside the
                    // stage, and nothing reads them (leaving the loop by a vote of the lanes took 4 % of the kernel)
                    if (j > 0) mbar_wait(&ctl->w_empty[warp], (j - 1) & 1, abort, wlim);
                    unsigned char *w = W + warp * W_STAGE;
#pragma unroll
                    for (int i = 0; i < IU_PHI / 4; ++i) {
                        const int b = r + 4 * i;
                        if (b < nb) {
                            const __half2 *h = reinterpret_cast<const __half2 *>(&ph[i]);
                            uint4 x, y2;
                            __half2 *hx = reinterpret_cast<__half2 *>(&x), *hy = reinterpret_cast<__half2 *>(&y2);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 f = __half22float2(h[e]);
                                hx[e] = __floats2half2_rn(f.x * v0[2 * e], f.y * v0[2 * e + 1]);
                                hy[e] = __floats2half2_rn(f.x * v1[2 * e], f.y * v1[2 * e + 1]);
                            }
                            *reinterpret_cast<uint4 *>(w + sw128_offset(b, o)) = x;
                            *reinterpret_cast<uint4 *>(w + sw128_offset(NB + b, o)) = y2;
                        }
                    }
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->w_full[warp]);
                }
            }
        }
    } else {
        // epilogue: group e (warps 8-11, 12-15) takes the pairs of parity e; lane = chi row
        const unsigned grp = (warp >> 2) & 1;
        const int a = (warp & 3) * 32 + lane;
        unsigned j = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
            const IItem d = list[it / groups];
            const int mp = (d.np + pch - 1) / pch;
            int q0, q1;
            pairs_of(it, q0, q1);
            const int id = a < d.nc ? cids[d.c0 + a] : -1;
            for (int y = 0; y < mp && ok; ++y) {
                int b0, nb;
                phi_chunk(d.np, mp, y, b0, nb);
                const int NB = (nb + 15) / 16 * 16;
                // lane i: the output offset of the chunk's quad i
                const int qr = lane * 4 < nb ? (pids[d.p0 + b0 + lane * 4] >> 2) * nchi : 0;
                for (int q = q0; q < q1; ++q, ++j) {
                    if ((j & 1) != grp) continue;
                    const unsigned acc = j & 3;
                    ok = __all_sync(0xffffffffu, mbar_wait(&ctl->acc_full[acc], (j >> 2) & 1, abort, wlim) && !*abort);
                    tc_fence_after();
                    if (!ok) break;
                    const unsigned ta = tmem + acc * 128 + ((unsigned)((warp & 3) * 32) << 16);
                    const int ns = 2 * q + 1 < k ? 2 : 1;
                    for (int h = 0; h < ns; ++h) {
                        const int s = 2 * q + h;
                        const float f = dV / v_scale(bits[s]);
                        float *o = out + ((long long)s * nquads * nchi + id) * 4;
                        for (int c = 0; c < NB; c += 16) {
                            float v[16];
                            tmem_ld16(ta + h * NB + c, v);
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int row = __shfl_sync(0xffffffffu, qr, c / 4 + i);
                                if (id >= 0 && c + 4 * i < nb)
                                    red_add_v4(o + (long long)row * 4, f * v[4 * i], f * v[4 * i + 1], f * v[4 * i + 2],
                                               f * v[4 * i + 3]);
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->acc_empty[acc]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 17) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
    if (threadIdx.x == 0 && ctl->abort) atomicExch(err, 1);
}

// largest |V_s| of every state (bit pattern; bits zeroed before). blockIdx.y = state.
__global__ void __launch_bounds__(256) v_max_kernel(const float *__restrict__ V, long long n3,
                                                    unsigned *__restrict__ bits) {
    const float *v = V + (long long)blockIdx.y * n3;
    float m = 0.0f;
#pragma unroll 8
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n3; i += gridDim.x * 256ll) m = fmaxf(m, fabsf(v[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&bits[blockIdx.y], __float_as_uint(m));
}

// out[s][a][4q .. 4q+3] = in[s][q][a][4]: 32 x 32 (quad, chi) tiles through shared memory
__global__ void __launch_bounds__(256) unpack_quads_kernel(const float4 *__restrict__ in, int nchi, int nquads,
                                                           float4 *__restrict__ out) {
    __shared__ float4 t[32][33];
    const int a0 = blockIdx.x * 32, q0 = blockIdx.y * 32;
    const long long so = (long long)blockIdx.z * nchi * nquads;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int q = q0 + i, a = a0 + threadIdx.x;
        if (q < nquads && a < nchi) t[i][threadIdx.x] = in[so + (long long)q * nchi + a];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int a = a0 + i, q = q0 + threadIdx.x;
        if (q < nquads && a < nchi) out[so + (long long)a * nquads + q] = t[threadIdx.x][i];
    }
}

size_t integrals_units_smem() { return 1024 + (size_t)SLICES * X_SLICE + (size_t)SLICES * W_STAGE + sizeof(IuShared); }

}  // namespace

// quads [k][nphi / 4][nchi][4] of V [k][n^3]; out, where not null, also in row order [k][nchi][nphi].
// list: tiles with both chi and phi in chunks of at most 128 chi; pch: most phi of a chunk (a multiple
// of 16, <= 48); bits: k words.
void potential_integrals_units(cudaStream_t st, const GridShape &g, const TileSet<float> &chi, const TileSet<float> &phi,
                               const unsigned short *chi_fm16, int nslots, const unsigned short *phi_fm16,
                               const IItem *list, int nlist, int pch, int nchi, int nphi, const float *V, int k,
                               float *quads, float *out, unsigned *bits, int *err) {
    if (k <= 0) return;
    ProfScope ps(st, ST_INTEGRALS, 2.0 * k * g.pair_points,
                 2.0 * g.table_values + 4.0 * k * g.n * g.n * g.n + 4.0 * k * nchi * nphi);
    const long long n3 = (long long)g.n * g.n * g.n;
    check(cudaMemsetAsync(quads, 0, sizeof(float) * (size_t)k * nchi * nphi, st), "memset(integrals)");
    if (nlist > 0) {
        check(cudaMemsetAsync(bits, 0, sizeof(unsigned) * k, st), "memset vmaxabs");
        const int per = std::max(8, 1216 / k);
        v_max_kernel<<<dim3((unsigned)std::min<long long>(per, (n3 + 2047) / 2048), k), 256, 0, st>>>(V, n3, bits);
        check_launch("v_max_kernel");
        CUtensorMap mx;
        if (!encode_map_2d(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, chi_fm16, (unsigned long long)TILE_PTS,
                           (unsigned long long)nslots, (unsigned long long)TILE_PTS * 2, 64, 128))
            throw CudaError{cudaErrorInvalidValue, "cuTensorMapEncodeTiled (integrals units)"};
        static const bool attr = [&]() {   // once per process, thread-safe
            check(cudaFuncSetAttribute(integrals_units_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)integrals_units_smem()),
                  "attr integrals_units");
            return true;
        }();
        (void)attr;
        int dev = 0, sms = 0;
        check(cudaGetDevice(&dev), "cudaGetDevice");
        check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
        // an item keeps its chi for all states; only where that leaves fewer than eight items per SM
        // are the pairs cut into groups, so that the last round of items stays a small part
        const int pairs = (k + 1) / 2;
        const int groups = (int)std::min<long long>(pairs, std::max<long long>(1, (8LL * sms + nlist - 1) / nlist));
        const long long nitems = (long long)nlist * groups;
        if (nitems > (1LL << 31) - 1) throw CudaError{cudaErrorInvalidValue, "integrals units: too many items"};
        integrals_units_kernel<<<(int)std::min<long long>(sms, nitems), IU_THREADS, integrals_units_smem(), st>>>(
            mx, g.n, g.nt, k, groups, pch, list, (int)nitems, chi.ids, phi.ids, nchi, nphi / 4, phi_fm16, V, bits,
            (float)g.dV, quads, err, active_wait_limit());
        check_launch("integrals_units_kernel");
    }
    if (out) {
        unpack_quads_kernel<<<dim3((nchi + 31) / 32, (nphi / 4 + 31) / 32, k), dim3(32, 8), 0, st>>>(
            reinterpret_cast<const float4 *>(quads), nchi, nphi / 4, reinterpret_cast<float4 *>(out));
        check_launch("unpack_quads_kernel");
    }
}

}  // namespace tddft
