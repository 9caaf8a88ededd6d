// sm_103a kernels of the phMG hot path.
//
//   spmv_*            CSR SpMV / fused residual r = b - K x (Eq. 3.1, 3.2
//                     residuals), prolongation y += P x and restriction y = R x
//                     (Sec. 3.1 transfers).
//   patch_gather      K_i = I_i K I_i^T from the CSR operator (Eq. 3.4,
//                     Sec. 3.4 assembled-matrix patch extraction).
//   gj_inverse_*      batched partial-pivot Gauss-Jordan inversion of the
//                     patch matrices in FP64 (exact patch solves, Sec. 3.4).
//   patch_apply       y_i = W_i K_i^{-1} (I_i r) for every patch (one ASM
//                     sweep, Eq. 3.4), streamed from HBM.
//   pull_scatter      z = sum_i I_i^T y_i as a deterministic gather over the
//                     DoF -> (patch slot) transpose map, fused with the
//                     Chebyshev / damped update.
//   mdot / maxpy ...  FGMRES and Arnoldi vector kernels (FP64).
//   hess_*            small Hessenberg / Givens kernels run by one thread.
//
// All kernels take plain device pointers; grids are sized by the host.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace skern {

constexpr int GJ_SMEM_MAX_N = 160;   // FP64 patch held in shared memory up to this size

// Programmatic dependent launch: a kernel launched with the programmatic
// stream serialisation attribute may start while the kernel before it on the
// stream is still running.  pdl_wait() blocks until that kernel has finished
// and its writes are visible; every kernel of the V-cycle calls it before it
// reads an input another kernel writes, or writes anything, and may read
// constant data (operators, patch factors, maps) before it.  pdl_release()
// lets the next kernel's blocks be scheduled once every block of this one has
// called it or exited.  Both are no-ops in a kernel launched without the
// attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ----------------------------------------------------------------- SpMV ---
enum SpmvMode { SPMV_SET = 0, SPMV_ADD = 1, SPMV_RESID = 2 };

// One LANES-wide group of threads per row; values of type T accumulate in T.
// mode SET:   y = A x        ADD: y += A x        RESID: y = b - A x
// MV: blockIdx.y selects the vector; the V-cycle's kernels then work on
// gridDim.y vectors stored one after another (the velocity components of FBF),
// each with the arithmetic of a single one.  (Templates: the offsets cost a
// single vector's small kernels 1-4%.)
template <typename T, int LANES, int MODE, bool MV>
__global__ void __launch_bounds__(256) spmv_csr(int nrows, int ncols, const int* __restrict__ rp,
                                                const int* __restrict__ ci, const T* __restrict__ av,
                                                const T* __restrict__ x, T* __restrict__ y, const T* __restrict__ b) {
    if (MV) {
        x += (long long)blockIdx.y * ncols;
        y += (long long)blockIdx.y * nrows;
        if (MODE == SPMV_RESID) b += (long long)blockIdx.y * nrows;
    }
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = gtid / LANES;
    const int lane = threadIdx.x % LANES;
    // the operator is constant: its first round of column and value loads
    // is issued before waiting for the kernel that wrote x (and b)
    const bool live = row < nrows;
    const int s = live ? __ldg(rp + row) : 0, e = live ? __ldg(rp + row + 1) : 0;
    int c[4];
    T a[4];
    int base = s + lane;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int p = base + u * LANES;
        const bool ok = p < e;
        c[u] = ok ? __ldg(ci + p) : 0;
        a[u] = ok ? __ldg(av + p) : T(0);
    }
    pdl_wait();
    pdl_release();
    if (!live) return;   // whole LANES-group exits together (LANES divides 32)
    T acc = 0;
    // four entries per lane per round: their column and value loads, then
    // their x loads, are issued together (a row of ~40 entries takes one
    // round at 16 lanes instead of a chain of three dependent load pairs)
    for (;;) {
#pragma unroll
        for (int u = 0; u < 4; ++u) acc += a[u] * x[c[u]];
        base += 4 * LANES;
        if (base >= e) break;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int p = base + u * LANES;
            const bool ok = p < e;
            c[u] = ok ? __ldg(ci + p) : 0;
            a[u] = ok ? __ldg(av + p) : T(0);
        }
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o, LANES);
    if (lane == 0) {
        if (MODE == SPMV_SET) y[row] = acc;
        else if (MODE == SPMV_ADD) y[row] += acc;
        else y[row] = b[row] - acc;
    }
}

// y = A x (SET) or y = b - A x (RESID) in FP32 for a Stokes operator as the device
// assembly writes it: the rows of a velocity node's D components have their
// entries in the same places (the velocity block, with the same values and the
// columns of the component, then the pressures, with the same columns), and a
// pressure row holds the components' blocks one after another, node by node
// alike.  A group of LANES threads takes a node's D rows, or a pressure row, so
// that one column index serves D entries, a velocity value D rows and a gathered
// pressure D rows: 4 instead of 6 (2D) or 5 instead of 9 (3D) loads for D
// entries, and D times as many gathers in flight per thread.  The gathers' latency
// bounds it (cold caches, against spmv_csr): 64 x 64 P4 26.2 -> 23.6 us, 3D P3
// 16^3 70 -> 56, 256 x 256 P4 231 -> 199 us (0.7 GB less the shared entries).  In FP64,
// bound by the FP64 pipe, it measured no faster and is not used.
template <int LANES, int MODE, int D>
__global__ void __launch_bounds__(256) spmv_stokes(int nvf, int nq, const int* __restrict__ rp,
                                                   const int* __restrict__ ci, const float* __restrict__ av,
                                                   const float* __restrict__ x, float* __restrict__ y, const float* __restrict__ b) {
    constexpr int U = 4;
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) / LANES;
    const int lane = threadIdx.x % LANES;
    const bool live = g < nvf + nq, vel = g < nvf;
    const int row = vel ? g : g - nvf + D * nvf;
    int s[D];
    s[0] = live ? __ldg(rp + row) : 0;
    int len = live ? __ldg(rp + row + 1) - s[0] : 0;
#pragma unroll
    for (int c = 1; c < D; ++c) s[c] = live && vel ? __ldg(rp + row + c * nvf) : 0;
    if (!vel) {
        len /= D;
#pragma unroll
        for (int c = 1; c < D; ++c) s[c] = s[0] + c * len;
    }
    int col[U];
    float a[D][U];
    auto load = [&](int p0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = p0 + u * LANES;
            const bool ok = p < len;
            col[u] = ok ? __ldg(ci + s[0] + p) : 0;
            a[0][u] = ok ? __ldg(av + s[0] + p) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = p0 + u * LANES;
            const bool own = p < len && !(vel && col[u] < nvf);      // B's entries; the velocity block's are shared
#pragma unroll
            for (int c = 1; c < D; ++c) a[c][u] = own ? __ldg(av + s[c] + p) : a[0][u];
        }
    };
    int p = lane;
    load(p);
    pdl_wait();
    pdl_release();
    if (!live) return;   // whole LANES-group exits together (LANES divides 32)
    float acc[D];
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] = 0;
    for (;;) {
        float xv[D][U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool one = vel && col[u] >= nvf;                   // a pressure: the same for every component
            xv[0][u] = x[col[u]];
#pragma unroll
            for (int c = 1; c < D; ++c) xv[c][u] = one ? xv[0][u] : x[col[u] + c * nvf];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int c = 0; c < D; ++c) acc[c] += a[c][u] * xv[c][u];
        p += U * LANES;
        if (p >= len) break;
        load(p);
    }
    if (!vel) {
#pragma unroll
        for (int c = 1; c < D; ++c) acc[0] += acc[c];
    }
    // every live lane takes part in every shuffle: a warp may hold the last
    // velocity nodes and the first pressure rows
#pragma unroll
    for (int c = 0; c < D; ++c) {
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) acc[c] += __shfl_down_sync(0xffffffffu, acc[c], o, LANES);
        if (lane == 0 && (c == 0 || vel)) {
            const int i = row + c * nvf;
            y[i] = MODE == SPMV_SET ? acc[c] : b[i] - acc[c];
        }
    }
}

// ------------------------------------------------------- vector kernels ---
template <typename TO, typename TI>
__global__ void convert_vec(int n, const TI* __restrict__ x, TO* __restrict__ y) {
    pdl_wait();
    pdl_release();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = (TO)x[i];
}

template <typename T>
__global__ void fill_vec(long long n, T v, T* __restrict__ y) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) y[i] = v;
}

// y = a x + b y
template <typename T>
__global__ void axpby(int n, T a, const T* __restrict__ x, T b, T* __restrict__ y) {
    pdl_wait();
    pdl_release();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = a * x[i] + b * y[i];
}

// y = x * (1 / *s)   (device scalar divisor, FGMRES / Arnoldi normalisation)
__global__ void scale_by_inv(int n, const double* __restrict__ x, const double* __restrict__ s, double* __restrict__ y);

// y = x - K x is not needed; the FGMRES/Arnoldi reductions:
// partial[b*m + i] = sum over this block's rows of V[i][k] * w[k]
__global__ void mdot_partial(int n, int m, const double* __restrict__ V, long long ldv,
                             const double* __restrict__ w, double* __restrict__ partial);
// out[i] = sum_b partial[b*m + i] (fixed order), optionally accumulated
// into acc[i] as well; if sqrt_out, out[0] = sqrt(sum).
__global__ void mdot_final(int nblocks, int m, const double* __restrict__ partial, double* __restrict__ out,
                           double* __restrict__ acc, int sqrt_out);
// Same reduction in one launch (last block finishes in a fixed order);
// MDOT_BLOCKS blocks of MDOT_THREADS threads; ticket must start at 0 and is reset.
constexpr int MDOT_BLOCKS = 152, MDOT_THREADS = 256;
void mdot_fused(int n, int m, const double* V, long long ldv, const double* w, double* partial, unsigned int* ticket,
                double* out, double* acc, int sqrt_out, cudaStream_t s);
// w <- w - V h; out[0..m) = V^T w, out[m] = w^T w of the updated w,
// acc[i] += out[i] (i < m); MDOT_BLOCKS blocks of MDOT_THREADS threads, m <= 31.
void maxpy_mdot(int n, int m, const double* V, long long ldv, const double* h, double* w, double* partial,
                unsigned int* ticket, double* out, double* acc, cudaStream_t s);
// w <- (w - V h) / nu, nu = sqrt(max(*nrm2 - |h|^2, 0)), *hn = nu
__global__ void maxpy_normalise(int n, int m, const double* __restrict__ V, long long ldv, const double* __restrict__ h,
                                const double* __restrict__ nrm2, double* __restrict__ w, double* __restrict__ hn);
// w[k] += sign * sum_i h[i] V[i][k]
__global__ void maxpy(int n, int m, const double* __restrict__ V, long long ldv, const double* __restrict__ h,
                      double sign, double* __restrict__ w);

// ------------------------------------------------------ DoF -> slot map ---
// slot_count (cnt zeroed) -> exclusive scan of cnt into soff[0..n] ->
// slot_fill (cur zeroed) -> slot_sort: sidx lists every DoF's slots in
// increasing order, wt[j] = 1 / multiplicity.
__global__ void slot_count(long long nent, const int* __restrict__ pdofs, int* __restrict__ cnt);
__global__ void slot_fill(long long nent, const int* __restrict__ pdofs, const int* __restrict__ soff, int* __restrict__ cur,
                          int* __restrict__ sidx);
__global__ void slot_sort(int n, const int* __restrict__ soff, int* __restrict__ sidx, double* __restrict__ wt);

// ------------------------------------------------------------- patches ---
// Dense K_i (row-major n_i x n_i, FP64) gathered from the CSR of K: one CTA
// per patch; column positions found by binary search in the sorted patch DoF
// list.  out must be zeroed by the caller.
__global__ void patch_gather(int npatch, const int* __restrict__ poff, const int* __restrict__ pdofs,
                             const long long* __restrict__ moff, const int* __restrict__ rp,
                             const int* __restrict__ ci, const double* __restrict__ av, double* __restrict__ out);

// In-place Gauss-Jordan inversion with partial pivoting of every patch
// matrix (row-major, FP64), shared-memory variant (n_i <= GJ_SMEM_MAX_N).
// Writes K_i^{-1} column-major with leading dimension ld64 (FP64) and, if
// inv32 != nullptr, ld32 (FP32); the row-major inverse is also written back
// to `work` when keep_rowmajor.  status[patch] = 0, or 1 + pivot step of the
// first zero pivot.  retry: only the patches whose status is not 0.
__global__ void gj_inverse_smem(int npatch, const int* __restrict__ poff, const long long* __restrict__ moff,
                                double* __restrict__ work, const long long* __restrict__ off64, double* __restrict__ inv64,
                                const long long* __restrict__ off32, float* __restrict__ inv32,
                                int* __restrict__ status, int retry);
// Same algorithm operating on the matrix in global memory (large patches).
__global__ void gj_inverse_global(int npatch, const int* __restrict__ poff, const long long* __restrict__ moff,
                                  double* __restrict__ work, const long long* __restrict__ off64, double* __restrict__ inv64,
                                  const long long* __restrict__ off32, float* __restrict__ inv32,
                                  int* __restrict__ status, int* __restrict__ ipiv_ws, double* __restrict__ col_ws,
                                  int retry);

// Block (Schur-complement) inverse of saddle-structured Vanka patches:
// K_i = [L 0 B_0^T; 0 L B_1^T; B_0 B_1 0] with one SPD velocity block L per
// component (vector Laplacian), pnv[p] velocity nodes per component.  FP64;
// SPD blocks inverted by Gauss-Jordan without pivoting; status as above.
// Patches whose scratch (saddle_scratch doubles) is <= max_scratch run in
// shared memory (saddle_inverse_smem), the others in the global scratch at
// soff[p] (saddle_inverse_global).
__host__ __device__ inline long long saddle_scratch(int d, int n, int nv) {
    const int np = n - d * nv, npp = np | 1;
    const int mx = nv > np ? nv : np;
    return (long long)nv * nv + 2LL * d * nv * npp + (long long)np * np + 3LL * mx + 2;
}
constexpr long long SADDLE_SMEM_MAX_DOUBLES = 25600;   // 200 KB of shared memory
// scratch of the factored-only inversion (one component's B^T and W at a
// time, the two-pivot sweep's columns, and one bit mask per pressure column
// of B^T: its nonzero rows)
// Pair-packed upper triangle of a symmetric n x n matrix: rows pr and
// n - 1 - pr share the n + 1 slots from pr (n + 1), in the order of the
// sweeps' row-pair mapping; entry (a, b), a <= b, sits at pp_row(n, a) + b.
__host__ __device__ inline long long pp_size(int n) { return (long long)((n + 1) / 2) * (n + 1); }
__host__ __device__ inline int pp_row(int n, int a) { return 2 * a < n ? a * n : (n - 1 - a) * (n + 1) + 1; }
// pp: the velocity block pair-packed (the shared-memory kernel) or full
// (the global-scratch kernel, whose lane accesses then stay coalesced)
__host__ __device__ inline long long saddle_scratch_factored(int d, int n, int nv, bool pp = true) {
    const int np = n - d * nv, npp = np | 1;
    const int mx = nv > np ? nv : np;
    return (pp ? pp_size(nv) : (long long)nv * nv) + 2LL * nv * npp + (long long)np * np + 7LL * mx + 2 + (long long)np * ((nv + 63) / 64);
}
// (saddle_inverse_smem leaves patches with max(nv, np) >= skip_from alone.)
// Outputs (each may be NULL): explicit inverses inv64 / inv32 (column-major,
// leading dimension n rounded up to 2 / 4), the factored form fac64 / fac32
// at foff64[p] / foff32[p] (saddle_factor_len), and, if back, the explicit
// inverse row-major in place of K_i.  saddle_inverse_smem with work == NULL
// (factored form only) reads each patch's rows of the CSR operator (rp, ci,
// av) directly, its sorted DoF list pdofs[poff[p] ..) held in shared memory
// at double offset sd_off (after the scratch).
__global__ void saddle_inverse_smem(int npatch, int d, const int* __restrict__ poff, const int* __restrict__ pnv,
                                    const long long* __restrict__ moff, double* __restrict__ work,
                                    const long long* __restrict__ off64, double* __restrict__ inv64,
                                    const long long* __restrict__ off32, float* __restrict__ inv32,
                                    const long long* __restrict__ foff64, double* __restrict__ fac64,
                                    const long long* __restrict__ foff32, float* __restrict__ fac32, int back,
                                    int packed, long long max_scratch, int skip_from, const int* __restrict__ pdofs,
                                    const int* __restrict__ rp, const int* __restrict__ ci, const double* __restrict__ av,
                                    int sd_off, int* __restrict__ status);
__global__ void saddle_inverse_global(int npatch, int d, const int* __restrict__ poff, const int* __restrict__ pnv,
                                      const long long* __restrict__ moff, double* __restrict__ work,
                                      const long long* __restrict__ off64, double* __restrict__ inv64,
                                      const long long* __restrict__ off32, float* __restrict__ inv32,
                                      const long long* __restrict__ foff64, double* __restrict__ fac64,
                                      const long long* __restrict__ foff32, float* __restrict__ fac32, int back,
                                      int packed, long long max_scratch, const long long* __restrict__ soff,
                                      double* __restrict__ scratch, int* __restrict__ status);
// The factored form of the listed patches from the CSR operator, on 4 x 4 tiles
// in shared memory, one CTA of 512, 256 or 128 threads per patch.  max4: the largest
// of nv and np in tiles of four; max_np, max_n: the largest np and n; soff: each
// listed patch's place in the scratch (saddle_tiles_scratch doubles).
constexpr size_t SADDLE_TILES_SMEM_MAX = 226 * 1024;
// A launch's patches take at most this many doubles of scratch (4 GB): about three
// times what is kept of a patch, so that a level with all its patches at once could
// fill the memory that its operator and bases need.  Some 5500 patches of P8 and
// 30,000 of P5 make one launch; a larger level pays a last wave per 40 waves.
constexpr long long SADDLE_TILES_SCRATCH_MAX = 1LL << 29;
// Patches of max(nv, np) from here on are tiled even where the pivot-pair
// kernel's shared memory would hold them.  At 91 nodes (P5 64 x 64) tiles take
// 7.4 ms against 8.9; at 61 (P4 64 x 64, where the 4 x 4 inverses and the padding
// weigh more) 2.94 against 2.42, at 37 (P3 128 x 128) 3.65 against 3.20.  The line
// lies between; 3D P2 stars (65 nodes, one pressure) are on its slower side by
// 10% (2.40 against 2.16 ms on 16^3).
constexpr int SADDLE_TILES_MIN_N = 80;
// and from this many on, unless the level's larger ones need the tiles anyway: they
// are a launch of their own behind the others', whose time a small level pays on top
// (P5 16 x 16 0.74 ms on pivot pairs, 0.45 + 0.59 with tiles; 28 x 28 1.93, 0.46 + 1.77; 32 x 32
// with 961 stars 2.57, 0.46 + 2.18, its setup 5.50 and 5.90; 64 x 64 8.9, 0.49 + 7.4; P4 on the
// disk, a few stars of 81 nodes among 1943, 1.50, 1.37 + 0.27).  Below another level,
// beside whose inversion it runs, half as many: under P8 32 x 32 the 961 P5 stars are
// better on tiles (setup 31.4 ms against 33.1).
constexpr int SADDLE_TILES_MIN_COUNT = 152 * 8, SADDLE_TILES_MIN_BELOW = 152 * 4;
__host__ __device__ inline size_t saddle_tiles_smem(int d, int max4, int max_np, int max_n) {
    const size_t nt = (size_t)max4 * (max4 + 1) / 2;
    return nt * (128 + 4) + sizeof(double) * (32 * (size_t)max4 + 32) + sizeof(int) * ((size_t)max_np * (d + 1) + max_n);
}
__host__ __device__ inline long long saddle_tiles_scratch(int d, int n, int nv) {
    const long long dnv = (long long)d * nv, np = n - dnv;
    return dnv * ((np + 3) & ~3LL) + dnv * np + (dnv * np + 1) / 2;
}
#define SADDLE_TILES_ARGS                                                                                              \
    int d, const int *__restrict__ list, const int *__restrict__ poff, const int *__restrict__ pnv,                    \
        const long long *__restrict__ foff64, double *__restrict__ fac64, const long long *__restrict__ foff32,        \
        float *__restrict__ fac32, int packed, const int *__restrict__ pdofs, const int *__restrict__ rp,              \
        const int *__restrict__ ci, const double *__restrict__ av, int max4, int max_np,                               \
        const long long *__restrict__ soff, double *scratch, int *__restrict__ status
__global__ void saddle_inverse_tiles_512(SADDLE_TILES_ARGS);
__global__ void saddle_inverse_tiles_256(SADDLE_TILES_ARGS);
__global__ void saddle_inverse_tiles_128(SADDLE_TILES_ARGS);
#undef SADDLE_TILES_ARGS
// Explicit inverses of SPD blocks of lo < n <= hi (work row-major, kept),
// outputs and status as gj_inverse_*; spd_tiles_smem(min(hi, largest n)) bytes.
// Up to SPD_TILES_SMALL_N four CTAs of 128 threads share an SM.
constexpr int SPD_TILES_SMALL_N = 88, SPD_TILES_MAX_N = 220;
__host__ __device__ inline size_t spd_tiles_smem(int n) {
    const size_t n4 = (n + 3) / 4, nt = n4 * (n4 + 1) / 2;
    return nt * (128 + 4) + sizeof(double) * (32 * n4 + 32);
}
#define SPD_TILES_ARGS                                                                                                 \
    int lo, int hi, const int *__restrict__ poff, const long long *__restrict__ moff, const double *__restrict__ work, \
        const long long *__restrict__ off64, double *__restrict__ inv64, const long long *__restrict__ off32,          \
        float *__restrict__ inv32, int *__restrict__ status
__global__ void spd_inverse_tiles_128(SPD_TILES_ARGS);
__global__ void spd_inverse_tiles_512(SPD_TILES_ARGS);
#undef SPD_TILES_ARGS
// Elements of one patch's factored inverse (Li, W, Si with leading
// dimensions rounded up to vec = 2 (FP64) or 4 (FP32)).  Li's form, packed:
// 0 column-major; 1 its upper triangle row by row (nv (nv + 1) / 2 entries,
// rounded up to vec: the row-wise bulk-copy apply); 2 the 4 x 4 tiles of its upper
// triangle, zero padded, 16-byte group r ntile + t holding row r of tile t (the
// FP32 apply on tiles).
__host__ __device__ inline long long saddle_factor_lenL(int nv, int vec, int packed) {
    const long long n4 = (nv + 3) / 4;
    if (packed == 2) return 8 * n4 * (n4 + 1);
    return packed ? ((long long)nv * (nv + 1) / 2 + vec - 1) / vec * vec : (long long)((nv + vec - 1) / vec * vec) * nv;
}
__host__ __device__ inline long long saddle_factor_len(int d, int n, int nv, int vec, int packed = 0) {
    const int np = n - d * nv;
    const long long ldw = (d * nv + vec - 1) / vec * vec, lds = (np + vec - 1) / vec * vec;
    return saddle_factor_lenL(nv, vec, packed) + ldw * np + lds * np;
}
// One ASM sweep with the factored inverses streamed from global memory, one
// CTA of 128 or 256 threads per patch, D = 2 or 3 components; xs_len >= the largest patch.  Shared
// memory (bytes): the groups' partial sums and the patch's vectors (the
// residual in two orders, y, t and s).  A level whose largest patch needs more
// than SADDLE_APPLY_SMEM_MAX (the kernels' shared-memory attribute) by
// saddle_apply_limit is refused.
constexpr size_t SADDLE_APPLY_SMEM_MAX = 200 * 1024;
__host__ __device__ inline size_t saddle_apply_smem(int elem_bytes, int d, long long xs_len, int threads) {
    const long long xl = (xs_len + 3) & ~3LL;
    return (size_t)16 * threads * d + (size_t)elem_bytes * ((d == 3 ? 4 : d) * ((xl / d + 4) & ~3LL) + 3 * xl + 4);
}
__host__ __device__ inline size_t saddle_apply_limit(long long xs_len) { return (size_t)(6144 + 40 * xs_len); }
// Threads per patch: 256 while all patches fit in about one wave of the CTAs of 128
// (seven per SM), where a patch's own chain is what takes the time (FP32, 3D P3, 369
// patches 32.5 us against 71; SV P4, 370, 32.5 against 55.6; P8 16 x 16, 289, 45 against 71;
// P8 32 x 32, 1089, 130 against 143; FP64 P6 16 x 16, 289, 53 against 59).  Beyond it the
// smaller CTAs cover each other's barriers better (3D P3 16^3, 4913, 144 against 170; SV P3
// disk, 1438, 32.6 against 38.9; FP64 P5 stars, 1089, 90 against 117).  In FP32, with half as
// many row groups a patch, the line is eight per SM.
inline int saddle_apply_threads(int elem_bytes, int npatch) { return npatch <= 152 * (elem_bytes == 4 ? 8 : 7) ? 256 : 128; }
#define SADDLE_APPLY_DECL(T, NAME)                                                                                     \
    __global__ void NAME(const int* __restrict__ poff, const int* __restrict__ pdofs, const int* __restrict__ pnv,     \
                         const long long* __restrict__ foff, const T* __restrict__ fac, const T* __restrict__ r,       \
                         const T* __restrict__ wt, T* __restrict__ Y, int xs_len);
SADDLE_APPLY_DECL(float, saddle_apply_f32_2d_128)
SADDLE_APPLY_DECL(float, saddle_apply_f32_3d_128)
SADDLE_APPLY_DECL(double, saddle_apply_f64_2d_128)
SADDLE_APPLY_DECL(double, saddle_apply_f64_3d_128)
SADDLE_APPLY_DECL(float, saddle_apply_f32_2d_256)
SADDLE_APPLY_DECL(float, saddle_apply_f32_3d_256)
SADDLE_APPLY_DECL(double, saddle_apply_f64_2d_256)
SADDLE_APPLY_DECL(double, saddle_apply_f64_3d_256)
#undef SADDLE_APPLY_DECL
// The same sweep with one CTA per patch whose factored block is brought into
// shared memory by one bulk copy (buf_bytes >= the largest block, a
// multiple of 128; xs_len >= the largest patch).  *status = 1 if a CTA gave
// up waiting for its copy (bounded wait).
constexpr int SA_BULK_THREADS = 128;
constexpr long long SA_WAIT_LIMIT = 1ll << 22;
__host__ __device__ inline size_t saddle_apply_bulk_smem(int buf_bytes, int elem_bytes, int xs_len) {
    return (size_t)buf_bytes + (size_t)elem_bytes * 5 * xs_len;
}
__global__ void saddle_apply_bulk_f32(int d, const int* __restrict__ poff, const int* __restrict__ pdofs,
                                      const int* __restrict__ pnv, const long long* __restrict__ foff,
                                      const float* __restrict__ fac, const float* __restrict__ r,
                                      const float* __restrict__ wt, float* __restrict__ Y, int buf_bytes,
                                      int xs_len, int* __restrict__ status);
__global__ void saddle_apply_bulk_f64(int d, const int* __restrict__ poff, const int* __restrict__ pdofs,
                                      const int* __restrict__ pnv, const long long* __restrict__ foff,
                                      const double* __restrict__ fac, const double* __restrict__ r,
                                      const double* __restrict__ wt, double* __restrict__ Y, int buf_bytes,
                                      int xs_len, int* __restrict__ status);

// The FP32 sweep with Li on tiles (packed = 2): buf_bytes >= the largest block
// rounded up to 128 bytes, in 3D plus tile_part_bytes of the largest patch (its
// partial sums; in 2D they fit over Li).  saddle_tile_apply_<dim>_<threads>_<tiles per thread>.
__host__ __device__ inline int tile_part_bytes(int d, int n4) { return (4 * d * n4 + 4) * n4 * 4; }
__host__ __device__ inline size_t saddle_tile_apply_smem(int buf_bytes, int d, int xs_len) {
    return (size_t)buf_bytes + 4 * (5 * (size_t)((xs_len + 7) & ~3) + 4 * d);
}
#define SADDLE_TILE_APPLY_ARGS                                                                                      \
    const int *__restrict__ poff, const int *__restrict__ pdofs, const int *__restrict__ pnv,                       \
        const long long *__restrict__ foff, const float *__restrict__ fac, const float *__restrict__ r,             \
        const float *__restrict__ wt, float *__restrict__ Y, int buf_bytes, int xs_len, int *__restrict__ status
#define SADDLE_TILE_APPLY_DECL(D)                                         \
    __global__ void saddle_tile_apply_##D##d_32_1(SADDLE_TILE_APPLY_ARGS);  \
    __global__ void saddle_tile_apply_##D##d_64_1(SADDLE_TILE_APPLY_ARGS);  \
    __global__ void saddle_tile_apply_##D##d_128_1(SADDLE_TILE_APPLY_ARGS); \
    __global__ void saddle_tile_apply_##D##d_160_1(SADDLE_TILE_APPLY_ARGS); \
    __global__ void saddle_tile_apply_##D##d_256_1(SADDLE_TILE_APPLY_ARGS); \
    __global__ void saddle_tile_apply_##D##d_256_2(SADDLE_TILE_APPLY_ARGS);
SADDLE_TILE_APPLY_DECL(2)
SADDLE_TILE_APPLY_DECL(3)
#undef SADDLE_TILE_APPLY_DECL
using saddle_tile_apply_t = void (*)(SADDLE_TILE_APPLY_ARGS);
#undef SADDLE_TILE_APPLY_ARGS
// threads per CTA for npatch patches of at most n4 tile rows (0: too many
// tiles): one tile a thread where a CTA of up to 256 holds them, so that small
// patches take little of an SM and many of them are in flight; two above.  With
// 128 threads for all, 64 x 64 P4 took 29 us (24.5 with 160) and its 4225 P2
// stars 12.3 (8.6 with 32); a level too small to fill the SMs (one warp a patch
// takes the longest there: 6.4 us against 5.9 for 1089 stars) keeps two warps.
constexpr int SADDLE_TILE_APPLY_MAX = 512, SADDLE_TILE_APPLY_WARP_MIN = 152 * 16;
inline int saddle_tile_apply_threads(int n4, int npatch) {
    const int t = n4 * (n4 + 1) / 2;
    if (t <= 64) return t <= 32 && npatch >= SADDLE_TILE_APPLY_WARP_MIN ? 32 : 64;
    return t <= 128 ? 128 : t <= 160 ? 160 : t <= SADDLE_TILE_APPLY_MAX ? 256 : 0;
}
// Levels that keep the row-wise bulk-copy apply in FP32: one pressure per patch (P2),
// a largest patch, which sets threads and shared memory for all, with far more tiles
// than most, and enough patches for the SMs' places to count.  Mean over largest 0.23: the P2 level
// of SV on the refined disk (5671 patches, 91 tiles) 18.1 us against 22.3, 3D P2 with one
// star of 115 nodes (4505) 38.7 against 57.8; 0.33: 3D P2, 95 nodes (2465) 24.7 against
// 28.6; 0.39 (2057 patches) 22.5 on both sides; 0.47: P4 around a vertex of nine cells 52.5
// against 44.5 on tiles.  With 1438 patches or fewer there is no such loss (0.22: 11.4
// against 11.7 us; 669 patches, 0.23: 17.8 against 16.7), and with many pressures the
// tiles' products with W outweigh it (SV P3, up to 73 nodes, 3137 patches: 84 against 55).
constexpr int SADDLE_TILE_UNEVEN_FROM = 152 * 8;
inline bool saddle_tile_uneven(long long sum_tiles, int n4, int max_np, int npatch) {
    const int t = n4 * (n4 + 1) / 2;
    return max_np <= 1 && t > 64 && npatch > SADDLE_TILE_UNEVEN_FROM && 5 * sum_tiles < 2LL * t * npatch;
}

// One ASM sweep (Eq. 3.4): Y[poff[i] + a] = w[dof_a] * sum_b Kinv_i[a][b] r[dof_b].
// FP32: float4 loads of 4 consecutive rows per thread; FP64: double2 loads
// of 2 rows.  One CTA of PATCH_APPLY_THREADS per patch and vector (blockIdx.y;
// vectors of n DoFs and nslot slots).
constexpr int PATCH_APPLY_THREADS = 128;
__global__ void patch_apply_f32(int npatch, const int* __restrict__ poff, const int* __restrict__ pdofs,
                                const long long* __restrict__ ioff, const float* __restrict__ inv,
                                const float* __restrict__ r, const float* __restrict__ wt, float* __restrict__ Y, int n,
                                long long nslot);
__global__ void patch_apply_f64(int npatch, const int* __restrict__ poff, const int* __restrict__ pdofs,
                                const long long* __restrict__ ioff, const double* __restrict__ inv,
                                const double* __restrict__ r, const double* __restrict__ wt, double* __restrict__ Y, int n,
                                long long nslot);

// out[j] = alpha * sum_{s in slots(j)} Y[s] + beta * out[j]  (slots in a
// fixed order, so the sum is bitwise reproducible).  Fused Chebyshev
// bookkeeping: xmode PULL_X_SET also sets x[j] = out[j], PULL_X_ADD adds
// x[j] += out[j]; with rdst != NULL, rdst[j] = bsrc[j].
enum PullX { PULL_X_NONE = 0, PULL_X_SET = 1, PULL_X_ADD = 2 };
// PRE = 8 slots at a time cover every DoF of a structured mesh at once, but cost
// 48 registers in FP64 (32 in FP32): levels beyond one wave of such CTAs take 4
// there (256 x 256 P4 73 -> 57 us, 128 x 128 P4 23 -> 19), smaller ones, where the chain
// of loads counts, 8 (one V-cycle of P2 8 x 8 50.5 us against 51.2).
constexpr int PULL_WIDE_MAX_64 = 152 * 5 * 256;
template <typename T, bool MV, int PRE>
__global__ void __launch_bounds__(256) pull_scatter(int n, const int* __restrict__ soff, const int* __restrict__ sidx,
                                                    const T* __restrict__ Y, T alpha, T beta, T* __restrict__ out,
                                                    T* __restrict__ x, int xmode, const T* __restrict__ bsrc,
                                                    T* __restrict__ rdst, long long nslot) {
    if (MV) {                                     // vectors of n DoFs and nslot slots, one after another
        Y += blockIdx.y * nslot;
        out += (long long)blockIdx.y * n;
        if (x) x += (long long)blockIdx.y * n;
        if (rdst) {
            bsrc += (long long)blockIdx.y * n;
            rdst += (long long)blockIdx.y * n;
        }
    }
    // the map is constant: the first DoF's slots (PRE at most) are fetched before
    // the wait for the kernel that wrote Y; the others one by one in the wide FP64
    // form, whose small levels hardly have any (a loop around them costs it 3 us a
    // V-cycle of P2 8 x 8), else PRE at a time
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    int q = 0, e = 0, idx[PRE];
    if (j < n) {
        q = __ldg(soff + j);
        e = __ldg(soff + j + 1);
#pragma unroll
        for (int u = 0; u < PRE; ++u) idx[u] = q + u < e ? __ldg(sidx + q + u) : 0;
    }
    pdl_wait();
    pdl_release();
    for (; j < n;) {
        T s = 0;
        auto slots = [&] {
            T y[PRE];
#pragma unroll
            for (int u = 0; u < PRE; ++u)
                if (q + u < e) y[u] = Y[idx[u]];
#pragma unroll
            for (int u = 0; u < PRE; ++u)
                if (q + u < e) s += y[u];
        };
        if constexpr (sizeof(T) == 8 && PRE == 8) {
            slots();
            for (int k = q + PRE; k < e; ++k) s += Y[__ldg(sidx + k)];
        } else {
            for (;;) {
                slots();
                q += PRE;
                if (q >= e) break;
#pragma unroll
                for (int u = 0; u < PRE; ++u) idx[u] = q + u < e ? __ldg(sidx + q + u) : 0;
            }
        }
        const T o = beta == T(0) ? alpha * s : alpha * s + beta * out[j];
        out[j] = o;
        if (xmode == PULL_X_SET) x[j] = o;
        else if (xmode == PULL_X_ADD) x[j] += o;
        if (rdst) rdst[j] = bsrc[j];
        j += gridDim.x * blockDim.x;
        if (j < n) {
            q = __ldg(soff + j);
            e = __ldg(soff + j + 1);
#pragma unroll
            for (int u = 0; u < PRE; ++u) idx[u] = q + u < e ? __ldg(sidx + q + u) : 0;
        }
    }
}

// ------------------------------------------------------ coarse solve ---
// One Gauss-Jordan step k on a dense row-major n x n FP64 matrix in global
// memory: pivot search, row swap, pivot-row scaling and copy of column k
// (single CTA), then the rank-1 elimination over all rows (whole grid).
__global__ void gj_step_pivot(int n, int k, double* __restrict__ A, int* __restrict__ ipiv,
                              double* __restrict__ colk, int* __restrict__ status);
__global__ void gj_step_eliminate(int n, int k, double* __restrict__ A, const double* __restrict__ colk);
__global__ void gj_unpivot_rows(int n, double* __restrict__ A, const int* __restrict__ ipiv);
// Blocked Gauss-Jordan inverse of one n x n row-major matrix on every SM,
// B <= GJB_MAX_B pivots per panel: for each panel gj_block_panel (one CTA,
// gj_block_panel_smem bytes), gj_block_swap (one thread per column),
// gj_block_update (grid ceil(n/32) x ceil(n/32)); then gj_unpivot_rows.
constexpr int GJB_THREADS = 512, GJB_MAX_B = 32;
__host__ __device__ inline size_t gj_block_panel_smem(int n, int B) { return (size_t)n * B * sizeof(double); }
__global__ void gj_block_panel(int n, int k0, int B, double* __restrict__ A, int* __restrict__ ipiv,
                               double* __restrict__ Pk, int* __restrict__ status);
__global__ void gj_block_swap(int n, int k0, int B, double* __restrict__ A, const int* __restrict__ ipiv,
                              double* __restrict__ Yb);
__global__ void gj_block_update(int n, int k0, int B, double* __restrict__ A, const double* __restrict__ Pk,
                                const double* __restrict__ Yb);
constexpr int GJC_CTAS = 16, GJC_THREADS = 512;
// The panel on one cluster of GJC_CTAS CTAs (rows split among them):
// gj_cluster_panel_smem_doubles(n, B) doubles of dynamic shared memory.
__host__ __device__ inline long long gj_cluster_panel_smem_doubles(int n, int B) {
    const long long R = (n + GJC_CTAS - 1) / GJC_CTAS;
    return 2 * R * B + 2LL * B + R;
}
__global__ void gj_cluster_panel(int n, int k0, int B, double* __restrict__ A, int* __restrict__ ipiv,
                                 double* __restrict__ Pk, int* __restrict__ status);


// y[i] = sum_j A[i][j] x[j] for i < nout (row-major, leading dimension lda),
// one warp per row, accumulated in FP64 whatever the vectors' type (an FP32
// x is widened exactly, y rounded once)
template <typename TI, typename TO, bool MV>
__global__ void __launch_bounds__(256) dense_gemv(int nout, int ncol, int lda, const double* __restrict__ A,
                                                  const TI* __restrict__ x, TO* __restrict__ y) {
    if (MV) {
        x += (long long)blockIdx.y * ncol;
        y += (long long)blockIdx.y * nout;
    }
    const int lane = threadIdx.x & 31;
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    // A is constant: the row's first entries are fetched before the wait
    constexpr int PRE = 8;
    double a[PRE];
#pragma unroll
    for (int u = 0; u < PRE; ++u) {
        const int j = lane + 32 * u;
        a[u] = row < nout && j < ncol ? __ldg(A + (long long)row * lda + j) : 0.0;
    }
    pdl_wait();
    pdl_release();
    if (row >= nout) return;
    double s = 0;
#pragma unroll
    for (int u = 0; u < PRE; ++u) {
        const int j = lane + 32 * u;
        if (j < ncol) s += a[u] * (double)x[j];
    }
    for (int j = lane + 32 * PRE; j < ncol; j += 32) s += __ldg(A + (long long)row * lda + j) * (double)x[j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) y[row] = (TO)s;
}

// --------------------------------------------------- small Hessenberg ---
// FGMRES: apply the previous Givens rotations to column j of H (stored
// [restart+1][restart] row-major), build rotation j, update g; resid[0] = |g[j+1]|.
// hcol holds h[0..j]; hnorm[0] = h[j+1].
__global__ void fgmres_givens(int j, int ldh, double* __restrict__ H, const double* __restrict__ hcol,
                              const double* __restrict__ hnorm, double* __restrict__ cs, double* __restrict__ sn,
                              double* __restrict__ g, double* __restrict__ resid);
// y = H[0:m,0:m]^{-1} g (upper triangular back substitution)
__global__ void fgmres_backsolve(int m, int ldh, const double* __restrict__ H, const double* __restrict__ g,
                                 double* __restrict__ y);
// Arnoldi: store column j of H (h[0..j], hnorm) into Hs [(m+1) x m].
__global__ void arnoldi_store(int j, int m, double* __restrict__ Hs, const double* __restrict__ h,
                              const double* __restrict__ hnorm);
constexpr int HESS_MAX = 16;
struct cplx { double re, im; };
__host__ __device__ void hessenberg_eig_core(int m, int ld, const double* Hs, double* out, cplx (*A)[HESS_MAX],
                                             cplx* cr, cplx* sr);
// Eigenvalues of the leading m x m block of an upper Hessenberg matrix
// (row-major, leading dimension ld) by the shifted QR iteration in complex
// arithmetic; out[0] = largest real part, out[1] = 1 if not converged.
// Host and device callable; the library runs it on the host.
// ------------------------------------------------------ solve plumbing ---
// b_free[r] = (F restricted) computed by the host-built maps:
// x_free gathers: out[i] = in[idx[i]]; scatter: out[idx[i]] = in[i]
template <typename T>
__global__ void gather_idx(int n, const int* __restrict__ idx, const T* __restrict__ in, T* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = in[idx[i]];
}
template <typename T>
__global__ void scatter_idx(int n, const int* __restrict__ idx, const T* __restrict__ in, T* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[idx[i]] = in[i];
}
// x[i] -= mean; mean = (sum_i w[i] x[i]) / wsum from a device scalar
__global__ void sub_scalar(int n, double* __restrict__ x, const double* __restrict__ num, double den);
// z[qcell[e][a]] = scale[e] * sum_b minv[a][b] y[qcell[e][b]]: a block-diagonal
// operator whose blocks are one reference matrix times a per-cell scale (the
// cells own disjoint index sets)
__global__ void block_mass_inverse(int nc, int nb, const int* __restrict__ qcell, const double* __restrict__ minv,
                                   const double* __restrict__ scale, const double* __restrict__ y, double* __restrict__ z);
// rows [0, nr), columns [0, nc) of a CSR: per-row counts, then (after a scan
// into brp) the entries in their row order, FP64 and optionally FP32
__global__ void csr_block_count(int nr, int nc, const int* __restrict__ rp, const int* __restrict__ ci, int* __restrict__ len);
__global__ void csr_block_fill(int nr, int nc, const int* __restrict__ rp, const int* __restrict__ ci,
                               const double* __restrict__ v, const int* __restrict__ brp, int* __restrict__ bci,
                               double* __restrict__ bv, float* __restrict__ bv32);
// x[i] -= w[i] * num[0] / den
// FP64 pipe peak probe: every thread runs 8 independent FMA chains of
// `iters` steps (x = x * a + b); out is written only if the sum equals the
// impossible value `never`, which keeps the chains live.
__global__ void fp64_fma_probe(long long iters, double a, double b, double never, double* __restrict__ out);

__global__ void sub_weighted(int n, double* __restrict__ x, const double* __restrict__ w, const double* __restrict__ num,
                             double den);

}  // namespace skern
