// FP64 kernels of the batched FGMRES; see batched.cuh.  Vectors of a batch
// are interleaved DoF-major, X[r * M + c] (DoF r, right-hand side c), so that
// a sparse row or a basis row of all the right-hand sides is one contiguous
// run, and every column is an independent FGMRES (Sec. 4) in lockstep.
#include "batched.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace sbat {

namespace {

constexpr int NBMAX = 32;           // basis vectors in one multi-dot (restart + 1 <= 32)
constexpr int DOT_CTAS = 152 * 4;   // the most CTAs of a multi-dot

// Y = A X (MODE 0) or Y = B - A X (MODE 2), FP64; M / 2 lanes per row, one
// double2 of right-hand sides per lane.
template <int MODE>
__global__ void __launch_bounds__(256) k_spmm64(int nr, int m, const int* __restrict__ rp, const int* __restrict__ ci,
                                                const double* __restrict__ av, const double2* __restrict__ X,
                                                double2* __restrict__ Y, const double2* __restrict__ B) {
    const int L = m >> 1;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long gt = blockIdx.x * (long long)blockDim.x + threadIdx.x; gt < (long long)nr * L; gt += stride) {
        const int row = (int)(gt / L), c2 = (int)(gt - (long long)row * L);
        const int s = __ldg(rp + row), e = __ldg(rp + row + 1);
        double2 acc = make_double2(0.0, 0.0);
        int p = s;
        for (; p + 2 <= e; p += 2) {
            const int c0 = __ldg(ci + p), c1 = __ldg(ci + p + 1);
            const double a0 = __ldg(av + p), a1 = __ldg(av + p + 1);
            const double2 x0 = __ldg(X + (long long)c0 * L + c2), x1 = __ldg(X + (long long)c1 * L + c2);
            acc.x = fma(a0, x0.x, acc.x);
            acc.y = fma(a0, x0.y, acc.y);
            acc.x = fma(a1, x1.x, acc.x);
            acc.y = fma(a1, x1.y, acc.y);
        }
        for (; p < e; ++p) {
            const double a = __ldg(av + p);
            const double2 x = __ldg(X + (long long)__ldg(ci + p) * L + c2);
            acc.x = fma(a, x.x, acc.x);
            acc.y = fma(a, x.y, acc.y);
        }
        if (MODE == 0) Y[gt] = acc;
        else { const double2 b = B[gt]; Y[gt] = make_double2(b.x - acc.x, b.y - acc.y); }
    }
}

// ---- classical Gram-Schmidt twice, per column ---------------------------
// Three passes over the basis for the new vector w (the single-vector cgs2's
// fusion): h1 = V^T w;  w <- w - V h1, h2 = V^T w, |w|^2;  w <- (w - V h2) / nu.
// The FP64 pipe bounds them (2 FMA lanes per SM and clock: 4 FMAs per basis
// entry take 1.8 times what reading it three times takes), so the
// accumulators are unrolled to NB, the smallest class (with_nb) that holds nb:
// unrolled to 32 for every nb, the dots of 32 columns on 128 x 128 P3 took
// 838 us, now 311 us at nb = 9 to 12 (86% of the FP64 peak's 268 us at 12);
// the whole orthogonalisation of a step went from 2.5 to 1.0 ms on average.
// A thread keeps one column c for all its rows (m divides the CTA's 256 threads).
template <int NB>
constexpr int dot_ctas_per_sm() { return NB <= 8 ? 4 : 2; }

// The CTA's sums of acc[0 .. na) over its row lanes -> partial[blk][i][c] (and
// of extra as i = na with EXTRA), 16 accumulators at a time through shared memory.
template <bool EXTRA, int NB>
__device__ __forceinline__ void col_block_partials(int m, int na, const double (&acc)[NB], double extra,
                                                   double* __restrict__ partial) {
    constexpr int NA = NB + (EXTRA ? 1 : 0), CH = NA < 16 ? NA : 16;
    const int mc = na + (EXTRA ? 1 : 0);
    __shared__ double red[CH][256];
    const int rl = 256 / m;
#pragma unroll
    for (int i0 = 0; i0 < NA; i0 += CH) {
        if (i0 >= mc) break;
#pragma unroll
        for (int q = 0; q < CH; ++q)
            if (i0 + q < NA) {
                double v = acc[i0 + q < NB ? i0 + q : 0];
                if (EXTRA && i0 + q == na) v = extra;
                red[q][threadIdx.x] = v;
            }
        __syncthreads();
        for (int t = threadIdx.x; t < CH * m; t += 256) {
            const int q = t / m, c = t - q * m;
            if (i0 + q < mc) {
                double s = 0.0;
                for (int x = 0; x < rl; ++x) s += red[q][x * m + c];
                partial[((long long)blockIdx.x * (NBMAX + 1) + i0 + q) * m + c] = s;
            }
        }
        __syncthreads();
    }
}

// partial[blk][i][c] = sum over the CTA's rows of V_i[r][c] W[r][c], i < nb
template <int NB>
__global__ void __launch_bounds__(256, dot_ctas_per_sm<NB>()) k_col_dots(int n, int m, int nb,
                                                                         const double* __restrict__ V, long long ldv,
                                                                         const double* __restrict__ W,
                                                                         double* __restrict__ partial) {
    double acc[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) acc[i] = 0.0;
    const long long nm = (long long)n * m;
    for (long long t = blockIdx.x * 256LL + threadIdx.x; t < nm; t += gridDim.x * 256LL) {
        const double w = W[t];
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (i < nb) acc[i] = fma(V[i * ldv + t], w, acc[i]);
    }
    col_block_partials<false>(m, nb, acc, 0.0, partial);
}

// W <- W - V H, then the dots of the new W with the basis (i < nb) and itself (i = nb)
template <int NB>
__global__ void __launch_bounds__(256, dot_ctas_per_sm<NB>()) k_col_update_dots(int n, int m, int nb,
                                                                                const double* __restrict__ V, long long ldv,
                                                                                const double* __restrict__ H,
                                                                                double* __restrict__ W,
                                                                                double* __restrict__ partial) {
    extern __shared__ double hs[];                // [nb][m]
    for (int t = threadIdx.x; t < nb * m; t += 256) hs[t] = H[t];
    __syncthreads();
    double acc[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) acc[i] = 0.0;
    const int c = threadIdx.x % m;
    const long long nm = (long long)n * m;
    double nrm = 0.0;
    for (long long t = blockIdx.x * 256LL + threadIdx.x; t < nm; t += gridDim.x * 256LL) {
        double w = W[t];
        if constexpr (NB <= 16) {
            // V's entries stay in registers between the two uses
            double v[NB];
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nb) v[i] = V[i * ldv + t];
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nb) w = fma(-hs[i * m + c], v[i], w);
            W[t] = w;
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nb) acc[i] = fma(v[i], w, acc[i]);
        } else {
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nb) w = fma(-hs[i * m + c], V[i * ldv + t], w);
            W[t] = w;
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nb) acc[i] = fma(V[i * ldv + t], w, acc[i]);
        }
        nrm = fma(w, w, nrm);
    }
    col_block_partials<true>(m, nb, acc, nrm, partial);   // the norm behind the nb dots
}

// out[i][c] = sum_blk partial[blk][i][c] (fixed order: 1024 / m interleaved
// block sums, then those in turn), acc[i][c] += out[i][c] for i < nacc;
// sqrt_out: out = sqrt(out) (column norms).  One CTA per i.
__global__ void __launch_bounds__(1024) k_col_reduce(int nblk, int m, const double* __restrict__ partial,
                                                     double* __restrict__ out, double* __restrict__ acc, int nacc,
                                                     int sqrt_out) {
    __shared__ double red[1024];
    const int i = blockIdx.x, c = threadIdx.x % m, g = threadIdx.x / m, G = 1024 / m;
    double s = 0.0;
#pragma unroll 8
    for (int b = g; b < nblk; b += G) s += partial[((long long)b * (NBMAX + 1) + i) * m + c];
    red[threadIdx.x] = s;
    __syncthreads();
    if (g > 0) return;
    for (int q = 1; q < G; ++q) s += red[q * m + c];
    if (sqrt_out) s = sqrt(s);
    out[i * m + c] = s;
    if (i < nacc) acc[i * m + c] += s;
}

// Vout = (W - V H) / nu, hn[c] = nu = sqrt(H[nb][c] - sum_i H[i][c]^2), with H[nb] =
// |W|^2 before the update (Pythagoras); 0 where nu = 0 (padding, a zero column).
// The second pass's H is O(eps) relative to the vector before the first one, so
// the difference loses no accuracy unless that vector lay in the span to about
// eps (a column whose Krylov space has closed while others go on).  Where it
// cancels by more than a factor of four, Vout stays unscaled, hn[c] = -1, and
// col_givens measures and scales the vector.
__global__ void __launch_bounds__(256) k_col_normalise(int n, int m, int nb, const double* __restrict__ V, long long ldv,
                                                       const double* __restrict__ H, const double* __restrict__ W,
                                                       double* __restrict__ Vout, double* __restrict__ hn) {
    extern __shared__ double hs[];                // [nb][m], then [m] 1 / nu
    for (int t = threadIdx.x; t < nb * m; t += 256) hs[t] = H[t];
    __syncthreads();
    if (threadIdx.x < m) {
        double q = H[nb * m + threadIdx.x];
        for (int i = 0; i < nb; ++i) q = fma(-hs[i * m + threadIdx.x], hs[i * m + threadIdx.x], q);
        const bool exact = q >= 0.25 * H[nb * m + threadIdx.x];     // (false for NaN)
        const double nu = exact ? sqrt(q) : 1.0;
        hs[nb * m + threadIdx.x] = nu > 0.0 ? 1.0 / nu : 0.0;
        if (blockIdx.x == 0) hn[threadIdx.x] = exact ? nu : -1.0;
    }
    __syncthreads();
    const int c = threadIdx.x % m;
    const double inv = hs[nb * m + c];
    const long long nm = (long long)n * m;
    for (long long t = blockIdx.x * 256LL + threadIdx.x; t < nm; t += gridDim.x * 256LL) {
        double s = W[t];
        int i = 0;
        for (; i + 4 <= nb; i += 4) {
            double v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = V[(i + u) * ldv + t];
#pragma unroll
            for (int u = 0; u < 4; ++u) s = fma(-hs[(i + u) * m + c], v[u], s);
        }
        for (; i < nb; ++i) s = fma(-hs[i * m + c], V[i * ldv + t], s);
        Vout[t] = inv > 0.0 ? s * inv : 0.0;
    }
}

// Vout[r][c] = W[r][c] / h[c] (0 where h[c] == 0: a column already exact)
__global__ void k_col_scale(long long nm, int m, const double* __restrict__ W, const double* __restrict__ h,
                            double* __restrict__ Vout) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nm; t += (long long)gridDim.x * blockDim.x) {
        const double d = h[t % m];
        Vout[t] = d > 0.0 ? W[t] / d : 0.0;
    }
}

// one CTA per column c: scale its new basis vector where col_normalise left that
// open (hn[c] < 0; rare, so one CTA's strided reads will do), then append
// (hcol[.][c], hn[c]) as column j of the column's Hessenberg matrix, apply the
// previous rotations, form the next, update g and the residual estimate (the
// single-RHS fgmres_givens per column)
__global__ void __launch_bounds__(256) k_col_givens(int j, int m, int ldh, int n, double* __restrict__ Vn,
                                                    double* __restrict__ H, const double* __restrict__ hcol,
                                                    double* __restrict__ hn, double* __restrict__ cs,
                                                    double* __restrict__ sn, double* __restrict__ g,
                                                    double* __restrict__ resid) {
    __shared__ double red[256];
    const int c = blockIdx.x;
    double nu = hn[c];
    if (nu < 0.0) {
        double s = 0.0;
        for (long long r = threadIdx.x; r < n; r += 256) s = fma(Vn[r * m + c], Vn[r * m + c], s);
        red[threadIdx.x] = s;
        __syncthreads();
        s = 0.0;
        for (int t = 0; t < 256; ++t) s += red[t];
        nu = sqrt(s);
        for (long long r = threadIdx.x; r < n; r += 256) Vn[r * m + c] = nu > 0.0 ? Vn[r * m + c] / nu : 0.0;
    }
    if (threadIdx.x > 0) return;
    hn[c] = nu;
    double* Hc = H + (long long)c * ldh * ldh;
    double* csc = cs + (long long)c * ldh;
    double* snc = sn + (long long)c * ldh;
    double* gc = g + (long long)c * (ldh + 1);
    for (int i = 0; i <= j; ++i) Hc[i * ldh + j] = hcol[i * m + c];
    Hc[(j + 1) * ldh + j] = nu;
    for (int i = 0; i < j; ++i) {
        const double a = Hc[i * ldh + j], b = Hc[(i + 1) * ldh + j];
        Hc[i * ldh + j] = csc[i] * a + snc[i] * b;
        Hc[(i + 1) * ldh + j] = -snc[i] * a + csc[i] * b;
    }
    const double a = Hc[j * ldh + j], b = Hc[(j + 1) * ldh + j];
    const double den = hypot(a, b);
    double cc = 1.0, ss = 0.0;
    if (den > 0.0) { cc = a / den; ss = b / den; }
    csc[j] = cc;
    snc[j] = ss;
    Hc[j * ldh + j] = den > 0.0 ? den : a;
    Hc[(j + 1) * ldh + j] = 0.0;
    gc[j + 1] = -ss * gc[j];
    gc[j] = cc * gc[j];
    resid[c] = fabs(gc[j + 1]);
}

// y = H^-1 g per column (upper triangular, jend columns); a zero pivot (a
// column whose Krylov space was exhausted earlier) contributes y = 0
__global__ void k_col_backsolve(int jend, int m, int ldh, const double* __restrict__ H, const double* __restrict__ g,
                                double* __restrict__ y) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m) return;
    const double* Hc = H + (long long)c * ldh * ldh;
    const double* gc = g + (long long)c * (ldh + 1);
    double* yc = y + (long long)c * (ldh + 1);
    for (int i = jend - 1; i >= 0; --i) {
        double s = gc[i];
        for (int l = i + 1; l < jend; ++l) s -= Hc[i * ldh + l] * yc[l];
        yc[i] = Hc[i * ldh + i] != 0.0 ? s / Hc[i * ldh + i] : 0.0;
    }
}

// X[r][c] += sum_{j < jend} y[c][j] Z_j[r][c]
__global__ void k_col_xupdate(long long nm, int m, int jend, int ldy, const double* __restrict__ Z, long long ldz,
                              const double* __restrict__ y, double* __restrict__ X) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nm; t += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(t % m);
        double s = X[t];
        for (int j = 0; j < jend; ++j) s = fma(y[(long long)c * ldy + j], Z[j * ldz + t], s);
        X[t] = s;
    }
}

// g[c][0] = beta[c], the rest 0; V0[r][c] = R[r][c] / beta[c]
__global__ void k_col_start(int m, int ldg, const double* __restrict__ beta, double* __restrict__ g) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m * ldg) return;
    const int c = t / ldg, i = t - c * ldg;
    g[t] = i == 0 ? beta[c] : 0.0;
}

// FP64 [nrhs][n] <-> FP64 interleaved [n][m] (zero columns nrhs .. m - 1)
__global__ void k_pack64(int n, int nrhs, int m, const double* __restrict__ r, double* __restrict__ X) {
    const long long total = (long long)n * m;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(t / m), c = (int)(t - (long long)j * m);
        X[t] = c < nrhs ? r[(long long)c * n + j] : 0.0;
    }
}
__global__ void k_unpack64(int n, int nrhs, int m, const double* __restrict__ X, double* __restrict__ z) {
    const long long total = (long long)n * nrhs;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(t / n), j = (int)(t - (long long)c * n);
        z[t] = X[(long long)j * m + c];
    }
}
// FP64 interleaved <-> FP32 interleaved (same layout)
__global__ void k_to32(long long nm, const double* __restrict__ x, float* __restrict__ y) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nm; t += (long long)gridDim.x * blockDim.x)
        y[t] = (float)x[t];
}
__global__ void k_to64(long long nm, const float* __restrict__ x, double* __restrict__ y) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nm; t += (long long)gridDim.x * blockDim.x)
        y[t] = (double)x[t];
}

inline int grid_of(long long n, int block = 256) {
    long long g = (n + block - 1) / block;
    if (g > 152LL * 16) g = 152LL * 16;
    return (int)(g < 1 ? 1 : g);
}

// calls f(integral constant NB) with the smallest unrolling that holds nb
template <typename F>
void with_nb(int nb, F&& f) {
    if (nb <= 2) f(std::integral_constant<int, 2>{});
    else if (nb <= 4) f(std::integral_constant<int, 4>{});
    else if (nb <= 6) f(std::integral_constant<int, 6>{});
    else if (nb <= 8) f(std::integral_constant<int, 8>{});
    else if (nb <= 12) f(std::integral_constant<int, 12>{});
    else if (nb <= 16) f(std::integral_constant<int, 16>{});
    else if (nb <= 24) f(std::integral_constant<int, 24>{});
    else f(std::integral_constant<int, 32>{});
}
template <int NB>
int dot_grid() { return 152 * dot_ctas_per_sm<NB>(); }

}  // namespace

size_t col_partial_doubles(int m) { return (size_t)DOT_CTAS * (NBMAX + 1) * m; }

void spmm64(int mode, int nr, int m, const int* rp, const int* ci, const double* av, const double* X, double* Y,
            const double* B, cudaStream_t s) {
    const int grid = grid_of((long long)nr * (m / 2));
    const double2* X2 = reinterpret_cast<const double2*>(X);
    double2* Y2 = reinterpret_cast<double2*>(Y);
    const double2* B2 = reinterpret_cast<const double2*>(B);
    if (mode == 0) k_spmm64<0><<<grid, 256, 0, s>>>(nr, m, rp, ci, av, X2, Y2, B2);
    else k_spmm64<2><<<grid, 256, 0, s>>>(nr, m, rp, ci, av, X2, Y2, B2);
}

void col_dots(int n, int m, int nb, const double* V, long long ldv, const double* W, double* partial, double* out,
              int sqrt_out, cudaStream_t s) {
    with_nb(nb, [&](auto nbc) {
        constexpr int NB = decltype(nbc)::value;
        k_col_dots<NB><<<dot_grid<NB>(), 256, 0, s>>>(n, m, nb, V, ldv, W, partial);
        k_col_reduce<<<nb, 1024, 0, s>>>(dot_grid<NB>(), m, partial, out, nullptr, 0, sqrt_out);
    });
}

void col_update_dots(int n, int m, int nb, const double* V, long long ldv, const double* H, double* W, double* partial,
                     double* out, double* acc, cudaStream_t s) {
    with_nb(nb, [&](auto nbc) {
        constexpr int NB = decltype(nbc)::value;
        k_col_update_dots<NB><<<dot_grid<NB>(), 256, sizeof(double) * nb * m, s>>>(n, m, nb, V, ldv, H, W, partial);
        k_col_reduce<<<nb + 1, 1024, 0, s>>>(dot_grid<NB>(), m, partial, out, acc, nb, 0);
    });
}

void col_normalise(int n, int m, int nb, const double* V, long long ldv, const double* H, const double* W, double* Vout,
                   double* hn, cudaStream_t s) {
    const int grid = std::min(grid_of((long long)n * m), 152 * 8);
    k_col_normalise<<<grid, 256, sizeof(double) * (nb + 1) * m, s>>>(n, m, nb, V, ldv, H, W, Vout, hn);
}

void col_scale(int n, int m, const double* W, const double* h, double* Vout, cudaStream_t s) {
    const long long nm = (long long)n * m;
    k_col_scale<<<grid_of(nm), 256, 0, s>>>(nm, m, W, h, Vout);
}

void col_givens(int j, int m, int ldh, int n, double* Vn, double* H, const double* hcol, double* hn, double* cs,
                double* sn, double* g, double* resid, cudaStream_t s) {
    k_col_givens<<<m, 256, 0, s>>>(j, m, ldh, n, Vn, H, hcol, hn, cs, sn, g, resid);
}

void col_backsolve(int jend, int m, int ldh, const double* H, const double* g, double* y, cudaStream_t s) {
    k_col_backsolve<<<(m + 63) / 64, 64, 0, s>>>(jend, m, ldh, H, g, y);
}

void col_xupdate(int n, int m, int jend, int ldy, const double* Z, long long ldz, const double* y, double* X,
                 cudaStream_t s) {
    const long long nm = (long long)n * m;
    k_col_xupdate<<<grid_of(nm), 256, 0, s>>>(nm, m, jend, ldy, Z, ldz, y, X);
}

void col_start(int m, int ldg, const double* beta, double* g, cudaStream_t s) {
    k_col_start<<<(m * ldg + 255) / 256, 256, 0, s>>>(m, ldg, beta, g);
}

void pack64(int n, int nrhs, int m, const double* r, double* X, cudaStream_t s) {
    k_pack64<<<grid_of((long long)n * m), 256, 0, s>>>(n, nrhs, m, r, X);
}

void unpack64(int n, int nrhs, int m, const double* X, double* z, cudaStream_t s) {
    k_unpack64<<<grid_of((long long)n * nrhs), 256, 0, s>>>(n, nrhs, m, X, z);
}

void to32(long long nm, const double* x, float* y, cudaStream_t s) { k_to32<<<grid_of(nm), 256, 0, s>>>(nm, x, y); }
void to64(long long nm, const float* x, double* y, cudaStream_t s) { k_to64<<<grid_of(nm), 256, 0, s>>>(nm, x, y); }

}  // namespace sbat
