// Internal declarations shared by the translation units of libtddft.
#pragma once

#include "device_memory.h"

#include <cuda_runtime.h>

#include <cstdint>
#include <new>
#include <string>
#include <vector>

namespace tddft {

constexpr int TILE = 8;                  // grid tile edge (points); a tile holds 512 points
constexpr int TILE_PTS = TILE * TILE * TILE;

struct CudaError {
    cudaError_t code;
    std::string where;
};

void check(cudaError_t e, const char *where);   // throws CudaError on failure
void check_launch(const char *where);           // cudaGetLastError after a launch

// ---- per-stage launch timing (CUDA events on the launching stream) -------------------------------
enum Stage {
    ST_GEMM = 0, ST_DENSITY, ST_INTEGRALS, ST_FFT, ST_TRACE, ST_VECTOR, ST_SMALL, ST_COUNT
};
const char *stage_name(int s);

struct Profiler;                        // defined in profile.cu
Profiler *&active_profiler();           // thread-local; null when profiling is off

// Limit of every bounded wait inside the tensor-core kernels, in clock64 ticks: thread-local, set
// for the duration of a call from the context's options (tddft_options.spin_limit_cycles) and read
// by the launchers, which pass it to the kernels.
constexpr long long DEFAULT_WAIT_LIMIT = 4000000000LL;   // about 2 s at 2 GHz
long long &active_wait_limit();

// Records an event pair around one launch when a profiler is active; `flops` and `bytes` are the
// algorithmic counts of the launch.
struct ProfScope {
    Profiler *p;
    cudaStream_t st;
    int stage;
    double flops, bytes;
    void *ev0;
    ProfScope(cudaStream_t st, int stage, double flops, double bytes);
    ~ProfScope();
};

// Per-tile lists of the functions whose support touches the tile, and their values on the
// tile's 512 points (local index (lx*8 + ly)*8 + lz; zero outside the support and the grid).
template <typename T>
struct TileSet {
    int ntiles = 0;
    int max_per_tile = 0;
    const int *off = nullptr;     // [ntiles+1] slot offsets
    const int *ids = nullptr;     // [slots] function index
    const T *val = nullptr;       // [slots][512]
};

// One unit of the tensor-core integrals launches: a grid tile with a chunk of its chi slots (at
// most three 128-row blocks) and a chunk of its phi slots (at most 128). A tile whose lists fit is
// one unit; a denser tile is cut into several units, each adding its part into the output.
struct VTile {
    int t;        // grid tile (whose 512 points the unit sums over)
    int c0, nc;   // first chi slot, count
    int p0, np;   // first phi slot, count
    int pad;
};

// One unit of the tensor-core density: a chunk of a tile's chi slots (at most two blocks of 64 on a
// whole tile, four on half a tile) and of its phi slots (at most 64, in chunks of 32), with the
// indices of their first 64-wide chi chunk and 32-wide phi chunk in the chunked point-major tables.
struct DUnit {
    enum { FIRST = 1, LAST = 2 };
    int t;         // grid tile
    int c0, nc;    // first chi slot, count
    int p0, np;    // first phi slot, count
    int cch;       // first chi chunk
    int pch;       // first phi chunk
    int chi_use;   // FIRST / LAST unit of a run with the same chi chunk
};

// One item: 128 nmh points (nmh 4 or 2) of tile t from its point point0 on, and its units
struct DItem {
    int t, point0, nmh, u0, u1;
};

// the density's items and units (device arrays)
struct DUnitList {
    const DItem *items = nullptr;
    const DUnit *units = nullptr;
    int nitems = 0;
    int cut[2] = {256, 64};   // most chi of an item, phi of a unit
    bool covers = false;      // every tile of the grid has both chi and phi
    bool phi32 = false;       // phi in float32 instead of float16 (at most 32 per unit)
    bool adds = false;        // units add to rho (float32 reductions, in their order) instead of carrying a sum
    bool chunked = false;     // a point's sum over phi in dot products of 32, else one running sum
};

// One item of the tensor-core integrals on units: at most 128 chi slots of a tile, all its phi slots
struct IItem {
    int t, c0, nc, p0, np;
};

// Tables of the float64 grid contractions on the tensor cores (device arrays): seven-bit digits of chi
// as float16, function-major and, where phi lists are whole aligned quads, point-major
struct Fp64Grid {
    unsigned short *fm = nullptr, *pm = nullptr;
    long long slots = 0, nchunks = 0, nitems = 0;
    const IItem *items = nullptr;   // integrals: at most 128 chi and 32 phi of a tile
    const int *tiles = nullptr;     // density: tiles with both chi and phi, densest first
    const int *cfirst = nullptr;    // first 64-wide chi chunk of each tile
    int *cexp = nullptr;                    // of every chi slot: |value| < 2^exp
    short *pexp = nullptr;                  // of every phi value
    int *rexp = nullptr;                    // of every point of every tile: |chi| < 2^exp
    long long pslots = 0;                   // phi slots
    int ntiles = 0;
    bool covers = false;            // the listed tiles are all tiles of the grid
};

struct GridShape {
    int n;          // points per side
    int nt;         // tiles per side = ceil(n / 8)
    double cell;
    double dV;
    double pair_points = 0.0;   // sum over grid points of (#chi nonzero) * (#phi nonzero)
    double table_values = 0.0;  // nonzero tabulated values of chi and phi
};

// ---------------------------------------------------------------------------------------------
// float32 matrices that stay fixed while registered: the tensor-core GEMM keeps their split
// (hi/lo, K-major) copies; unregister before freeing them
void tc_register_constant(const float *p);
void tc_unregister_constant(const float *p);

// dense GEMM, row-major: C[b] = alpha * op(A[b]) op(B[b]) + beta * C[b]. approx: a float32
// product on the tensor cores may take one TF32 MMA instead of the three-term split (about 1e-3
// relative error; for operands whose errors the method tolerates, such as a preconditioner's)
template <typename T>
void gemm(cudaStream_t st, bool ta, bool tb, int M, int N, int K, T alpha, const T *A, int lda,
          long long sA, const T *B, int ldb, long long sB, T beta, T *C, int ldc, long long sC,
          int batch, bool approx = false);

// ---------------------------------------------------------------------------------------------
// grid work
template <typename T>
void response_density(cudaStream_t st, const GridShape &g, const TileSet<T> &chi,
                      const TileSet<T> &phi, int nphi, const T *P, long long sP, int k, T *rho);

template <typename T>
void potential_integrals(cudaStream_t st, const GridShape &g, const TileSet<T> &chi,
                         const TileSet<T> &phi, int nchi, int nphi, const T *V, int k, T *out);

// V_s = v_H[rho_s] + fxc * rho_s for k states; work: complex buffer of ceil(k/2) * n^3; tw: the grid
// size's twiddles from fft_twiddles (2 n values of T)
template <typename T>
void hartree_fxc(cudaStream_t st, const GridShape &g, const T *rho, const T *fxc, int k, T *V,
                 void *work, const T *tw);
template <typename T>
void fft_twiddles(cudaStream_t st, int n, T *tw);

void fxc_lda(cudaStream_t st, const double *n0, double *fxc, long long npts);

bool fft_size_ok(int n);

// ---------------------------------------------------------------------------------------------
// solver primitives
// Trace products of blocks of k rows (rows len apart): for every job and q < nset <= 4,
// g[q][i * ldg + j] = sum_e x_i[e] y[q]_j[e], i, j < k (float64 result; fixed reduction order). A job's x
// is read once for all its sets. scratch: >= gram_scratch_doubles(64, 32) doubles.
constexpr int GRAM_JOBS = 3;
template <typename T>
struct GramBlock {
    const T *x;
    int nset;
    const T *y[4];
    double *g[4];
};
long long gram_scratch_doubles(int nx, int ny);
template <typename T>
void gram_blocks(cudaStream_t st, int k, int njob, const GramBlock<T> *job, int ldg, long long len, double *scratch);

// out_i = base_i + sum_j C[i*ldc + j] * in_j (C float64 on the device), out != in, rows len apart.
template <typename T>
void combine(cudaStream_t st, const double *C, int ldc, int nout, int nin, const T *in, const T *base, T *out,
             long long len);

// X_i <- sum_j C_ij (X_j + lam D_j) for narr <= 4 arrays of k p rows (C = Cp) and k q rows (Cq), in place;
// lam a device scalar, or NULL: X_i <- sum_j C_ij X_j (D is not read)
template <typename T>
void step_combine(cudaStream_t st, int k, const double *Cp, const double *Cq, const double *lam, T *const *X,
                  const T *const *D, int narr, long long len);

// X_b[e] *= mask[e % len] for b < nb
template <typename T>
void mask_mul(cudaStream_t st, T *X, const T *mask, long long len, int nb);

template <typename Tin, typename Tout>
void convert(cudaStream_t st, const Tin *in, Tout *out, long long n);

// y_b += sgn * a[b * a_stride] * x_b over nb blocks of len; a on the device (float64)
template <typename T>
void axpy_dev(cudaStream_t st, const double *a, int a_stride, double sgn, T *y, const T *x,
              long long len, int nb);

// ---------------------------------------------------------------------------------------------
// small float64 linear algebra on the device (one thread; k <= KMAX)
constexpr int KMAX = 16;

// Status word bits written by the small kernels
enum { DEV_OK = 0, DEV_BREAKDOWN = 1, DEV_NAN = 2, DEV_NAN_EVAL = 3, DEV_NAN_LINE = 4, DEV_NAN_INIT = 5 };

}  // namespace tddft
