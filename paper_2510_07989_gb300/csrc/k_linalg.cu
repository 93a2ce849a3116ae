// Kernels of the MOT step other than the history contraction: incidence
// products and FP64 CG solves behind the quasi-Helmholtz projectors
// (paper Section IV-B), the Gram solve and the static preconditioner products
// (Section III, Eq. (CP)), the right-hand side (Section V-C), current recovery
// and running Fourier sums (Eq. (dis_jm)).
//
// Block vectors are row-major [rows][C]: row = edge (or face / vertex),
// column = one right-hand side component (u-part columns 0..B-1, v-part B..2B-1).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "mot_internal.h"

namespace {

namespace cg = cooperative_groups;

// ----------------------------------------------------------------- helpers
__global__ void k_axpby(int n, double a, const double* __restrict__ x, double b, const double* __restrict__ y,
                        double* __restrict__ z) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double v = a * x[i];
        if (y) v += b * y[i];
        z[i] = v;
    }
}

// dst[v][npad][C2]: v=0: [eta u, v/eta], v=1: [eta' u, v/eta'], v=2: [-v, u]
__global__ void k_variants(int npad, int B, const double* __restrict__ x, double* __restrict__ dst, double eta,
                           double etap) {
    const int C2 = 2 * B;
    const size_t ps = (size_t)npad * C2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npad * B; i += gridDim.x * blockDim.x) {
        const int r = i / B, b = i - r * B;
        const double u = x[(size_t)r * C2 + b], v = x[(size_t)r * C2 + B + b];
        dst[(size_t)r * C2 + b] = eta * u;
        dst[(size_t)r * C2 + B + b] = v / eta;
        dst[ps + (size_t)r * C2 + b] = etap * u;
        dst[ps + (size_t)r * C2 + B + b] = v / etap;
        dst[2 * ps + (size_t)r * C2 + b] = -v;
        dst[2 * ps + (size_t)r * C2 + B + b] = u;
    }
}

// f[face][c] = sum over the face's edges of Sigma_{e,face} x[e][c]   (Sigma^T x)
__global__ void k_sigma_t(int nf, int C, const int* __restrict__ fe, const double* __restrict__ fs,
                          const double* __restrict__ x, double* __restrict__ f) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nf * C; i += gridDim.x * blockDim.x) {
        const int r = i / C, c = i - r * C;
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < 3; j++) s += fs[3 * r + j] * x[(size_t)fe[3 * r + j] * C + c];
        f[i] = s;
    }
}

// x[e][c] = z[c+(e)][c] - z[c-(e)][c]   (Sigma z)
__global__ void k_sigma(int ne, int C, const int* __restrict__ ef, const double* __restrict__ z,
                        double* __restrict__ x) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ne * C; i += gridDim.x * blockDim.x) {
        const int r = i / C, c = i - r * C;
        x[i] = z[(size_t)ef[2 * r] * C + c] - z[(size_t)ef[2 * r + 1] * C + c];
    }
}

// x[e][c] = z[v+(e)][c] - z[v-(e)][c]   (Lambda z)
__global__ void k_lambda(int ne, int C, const int* __restrict__ ev, const double* __restrict__ z,
                         double* __restrict__ x) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ne * C; i += gridDim.x * blockDim.x) {
        const int r = i / C, c = i - r * C;
        x[i] = z[(size_t)ev[2 * r + 1] * C + c] - z[(size_t)ev[2 * r] * C + c];
    }
}

// y = A x for a CSR matrix (rows A.n), C columns
__global__ void k_spmv(int n, int C, const int* __restrict__ rp, const int* __restrict__ ci,
                       const double* __restrict__ va, const double* __restrict__ x, double* __restrict__ y) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * C; i += gridDim.x * blockDim.x) {
        const int r = i / C, c = i - r * C;
        double s = 0.0;
        for (int j = rp[r]; j < rp[r + 1]; j++) s = fma(va[j], x[(size_t)ci[j] * C + c], s);
        y[i] = s;
    }
}

// ----------------------------------------------------------------- CG
// Solves A z = f column by column (A SPD, or singular and consistent: the
// Laplacians Sigma^T Sigma and Lambda^T Lambda, whose null space is the
// constants; f = Sigma^T x / Lambda^T x is orthogonal to it up to rounding,
// and its column mean is removed before the iteration). With NORMAL the
// operator is A2 (A x) (CGNR for the Gram matrix: A = G, A2 = G^T).
// One CTA owns CW columns (lane % CW) and all rows; only __syncthreads is used.
struct CsrV {
    const int* rp;
    const int* ci;
    const double* va;
};

template <int CW>
__device__ __forceinline__ double col_reduce(double v, double* red, double* colv) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off >= CW; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane < CW) red[warp * CW + lane] = v;
    __syncthreads();
    if (threadIdx.x < CW) {
        double s = 0.0;
        const int nw = blockDim.x >> 5;
        for (int w = 0; w < nw; w++) s += red[w * CW + threadIdx.x];
        colv[threadIdx.x] = s;
    }
    __syncthreads();
    const double r = colv[lane % CW];
    __syncthreads();
    return r;
}

template <int CW>
__device__ __forceinline__ double col_reduce_max(double v, double* red, double* colv) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off >= CW; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane < CW) red[warp * CW + lane] = v;
    __syncthreads();
    if (threadIdx.x < CW) {
        double m = 0.0;
        const int nw = blockDim.x >> 5;
        for (int w = 0; w < nw; w++) m = fmax(m, red[w * CW + threadIdx.x]);
        colv[threadIdx.x] = m;
    }
    __syncthreads();
    const double r = colv[lane % CW];
    __syncthreads();
    return r;
}

// 2^-e with 2^e the power of two at or below m (1 for m = 0): multiplying by
// it (and later by its inverse) is exact and brings a column to O(1)
__device__ __forceinline__ double pow2_scale(double m) { return m > 0.0 ? ldexp(1.0, -mot_scale_exponent(m)) : 1.0; }

template <int CW, bool NORMAL>
__global__ void __launch_bounds__(1024) k_cg(int N, int C, CsrV A, CsrV A2, const double* __restrict__ f,
                                             double* __restrict__ z, double* __restrict__ r, double* __restrict__ p,
                                             double* __restrict__ q, double* __restrict__ t, double tol, int maxit,
                                             int* __restrict__ it_max, int* __restrict__ noconv) {
    __shared__ double red[32 * CW];
    __shared__ double colv[CW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cl = lane % CW;
    const int c = blockIdx.x * CW + cl;
    const bool cv = c < C;
    const int RPW = 32 / CW;
    const int row0 = warp * RPW + lane / CW;
    const int RS = (blockDim.x >> 5) * RPW;
    double part = 0.0;
    // A graph Laplacian (not NORMAL) is singular with the constants as its null
    // space (connected surface). Its right-hand sides (Sigma^T x, Lambda^T x) sum
    // to zero only up to rounding; when x lies almost entirely in the other
    // subspace, that rounding is a sizeable inconsistent part of f, which CG
    // cannot reduce (the iteration then runs to its limit and drifts along the
    // null space). The column mean is removed first, so the solve is the
    // consistent one whose minimum-norm solution is the pseudo-inverse of
    // Section IV-B applied to f.
    double mean = 0.0;
    if (!NORMAL) {
        for (int row = row0; row < N; row += RS)
            if (cv) part += f[(size_t)row * C + c];
        mean = col_reduce<CW>(part, red, colv) / (double)N;
        part = 0.0;
    }
    // the column is scaled by a power of two to O(1) (exact) and the solution
    // scaled back at the end, so sums of squares neither underflow nor
    // overflow whatever the scale of f (late in a march f decays without bound)
    for (int row = row0; row < N; row += RS)
        if (cv) part = fmax(part, fabs(f[(size_t)row * C + c] - mean));
    const double sc = pow2_scale(col_reduce_max<CW>(part, red, colv));
    part = 0.0;
    for (int row = row0; row < N; row += RS)
        if (cv) {
            const size_t ix = (size_t)row * C + c;
            const double v = (f[ix] - mean) * sc;
            z[ix] = 0.0;
            r[ix] = v;
            p[ix] = v;
            part += v * v;
        }
    double rr = col_reduce<CW>(part, red, colv);
    const double bb = rr;
    bool done = !(bb > 0.0) || !cv;
    int it = 0;
    while (it < maxit) {
        if (__syncthreads_and(done)) break;
        if (NORMAL) {
            for (int row = row0; row < N; row += RS)
                if (cv) {
                    double s = 0.0;
                    for (int j = A.rp[row]; j < A.rp[row + 1]; j++) s = fma(A.va[j], p[(size_t)A.ci[j] * C + c], s);
                    t[(size_t)row * C + c] = s;
                }
            __syncthreads();
        }
        part = 0.0;
        for (int row = row0; row < N; row += RS)
            if (cv) {
                double s = 0.0;
                if (NORMAL) {
                    for (int j = A2.rp[row]; j < A2.rp[row + 1]; j++)
                        s = fma(A2.va[j], t[(size_t)A2.ci[j] * C + c], s);
                } else {
                    for (int j = A.rp[row]; j < A.rp[row + 1]; j++) s = fma(A.va[j], p[(size_t)A.ci[j] * C + c], s);
                }
                q[(size_t)row * C + c] = s;
                part += p[(size_t)row * C + c] * s;
            }
        const double pq = col_reduce<CW>(part, red, colv);
        const double alpha = (done || !(pq > 0.0)) ? 0.0 : rr / pq;
        part = 0.0;
        for (int row = row0; row < N; row += RS)
            if (cv) {
                const size_t ix = (size_t)row * C + c;
                z[ix] += alpha * p[ix];
                const double rv = r[ix] - alpha * q[ix];
                r[ix] = rv;
                part += rv * rv;
            }
        const double rn = col_reduce<CW>(part, red, colv);
        const double beta = done ? 0.0 : rn / rr;
        if (!done) {
            rr = rn;
            if (rr <= tol * tol * bb) done = true;
        }
        for (int row = row0; row < N; row += RS)
            if (cv && !done) {
                const size_t ix = (size_t)row * C + c;
                p[ix] = r[ix] + beta * p[ix];
            }
        __syncthreads();
        it++;
    }
    const double usc = 1.0 / sc;  // exact: sc is a power of two
    for (int row = row0; row < N; row += RS)
        if (cv) z[(size_t)row * C + c] *= usc;
    if (threadIdx.x == 0) {
        atomicMax(it_max, it);
        if (it >= maxit) atomicAdd(noconv, 1);
    }
}

// ----------------------------------------------------------------- dense GEMM
// Y[n][C] = A[n][K] X[K][C] (K a multiple of 32), FP64, for C > 8. Bound by the
// FP64 units (two multiply-adds per clock and SM), so what matters is that all
// of them work: 64-row x TX-column tiles alone are a few dozen CTAs at the
// sizes of the march (576 x 576 x 10: nine), so K is split over gridDim.z as
// well and the splits are summed in a fixed order. TX = 16 for C <= 16 (a
// masked lane of a warp costs what a live one does), else 32.
constexpr int GB_M = 64, GB_K = 32;
template <int TX>
__global__ void __launch_bounds__(256) k_gemm(int n, int K, int C, int kchunk, const double* __restrict__ A,
                                              const double* __restrict__ X, double* __restrict__ Y) {
    constexpr int TY = 256 / TX, RPT = GB_M / TY;
    __shared__ double sa[GB_M][GB_K + 1];
    __shared__ double sx[GB_K][TX];
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    const int row0 = blockIdx.x * GB_M, col0 = blockIdx.y * TX;
    const int kbeg = blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);
    double acc[RPT];
#pragma unroll
    for (int i = 0; i < RPT; i++) acc[i] = 0.0;
    for (int k0 = kbeg; k0 < kend; k0 += GB_K) {
#pragma unroll
        for (int e = threadIdx.x; e < GB_M * GB_K; e += 256) {
            const int r = e / GB_K, k = e - r * GB_K;
            sa[r][k] = (row0 + r < n) ? A[(size_t)(row0 + r) * K + k0 + k] : 0.0;
        }
#pragma unroll
        for (int e = threadIdx.x; e < GB_K * TX; e += 256) {
            const int k = e / TX, cc = e - k * TX;
            sx[k][cc] = (col0 + cc < C) ? X[(size_t)(k0 + k) * C + col0 + cc] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < GB_K; k++) {
            const double xv = sx[k][tx];
#pragma unroll
            for (int i = 0; i < RPT; i++) acc[i] = fma(sa[ty + TY * i][k], xv, acc[i]);
        }
        __syncthreads();
    }
    if (col0 + tx < C) {
        double* out = Y + (size_t)blockIdx.z * n * C;
#pragma unroll
        for (int i = 0; i < RPT; i++) {
            const int r = row0 + ty + TY * i;
            if (r < n) out[(size_t)r * C + col0 + tx] = acc[i];
        }
    }
}

// Y = sum over the S splits of W, in order
__global__ void k_split_sum(long long n, int S, const double* __restrict__ W, double* __restrict__ Y) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double v = 0.0;
        for (int z = 0; z < S; z++) v += W[(size_t)z * n + i];
        Y[i] = v;
    }
}

// Y[n][C] = A[n][K] X[K][C] for C <= 8: one warp per row, lanes over the
// contraction index (coalesced rows of A), warp-shuffle reduction. Bound by
// reading A (C <= 2) or the FP64 units; 16-byte loads, four of A in flight per
// lane (8-byte loads: 57 us at 3840 x 3840, C = 1, 2.0 TB/s).
template <int CC>
__global__ void __launch_bounds__(256) k_gemv_small(int n, int K, const double* __restrict__ A,
                                                    const double* __restrict__ X, double* __restrict__ Y) {
    const int lane = threadIdx.x & 31;
    for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n; row += (gridDim.x * blockDim.x) >> 5) {
        double acc[CC];
#pragma unroll
        for (int c = 0; c < CC; c++) acc[c] = 0.0;
        const double* a = A + (size_t)row * K;
#pragma unroll 4
        for (int k = 2 * lane; k < K; k += 64) {  // K is even, rows 16-byte aligned
            const double2 av = *reinterpret_cast<const double2*>(a + k);
            double2 x[CC];  // X rows k, k + 1
#pragma unroll
            for (int c = 0; c < CC; c++) x[c] = *reinterpret_cast<const double2*>(X + (size_t)k * CC + 2 * c);
            const double* xs = reinterpret_cast<const double*>(x);
#pragma unroll
            for (int c = 0; c < CC; c++) acc[c] = fma(av.x, xs[c], acc[c]);
#pragma unroll
            for (int c = 0; c < CC; c++) acc[c] = fma(av.y, xs[CC + c], acc[c]);
        }
#pragma unroll
        for (int c = 0; c < CC; c++) {
            double v = acc[c];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0) Y[(size_t)row * CC + c] = v;
        }
    }
}

// ----------------------------------------------------------------- RHS
// rho1[e][b] (u-part) / rho1[e][B+b] (v-part): (1/dt) int p_i (e, h) tested;
// rho2: (1/T_max) (d/dt^-1 (e, h))(i dt) tested, 0 after t_trunc.
// Testing with n x f_m gives -<f_m, .>. Section V-C, Eq. (hin).
//
// The incident field's time integral needs two error functions per point and
// wave, FP64 work of a unit that does two operations per clock and SM. A
// triangle's points are those of its three edges' functions, so they are
// evaluated once per distinct point of the quadrature table (a third of it;
// found at load), and beyond |argument| = 6 the error function is 1 to the last
// bit: before the pulse arrives and after it has passed nothing is evaluated.
// F[pt][0][b] = (A/2c) (erf(a1) - erf(a0)),  F[pt][1][b] = (A/2c) (1 + erf(a1))
__global__ void __launch_bounds__(128) k_rhs_points(int npts, int B, const double* __restrict__ pts,
                                                    const double* __restrict__ waves, double ti, double tprev, double c,
                                                    double* __restrict__ F) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= npts * B) return;
    const int pt = i / B, b = i - pt * B;
    const double* wv = waves + 10 * b;
    const double A = wv[0], w = wv[7], t0 = wv[8];
    const double kd = wv[4] * pts[3 * pt] + wv[5] * pts[3 * pt + 1] + wv[6] * pts[3 * pt + 2];
    auto erf_sat = [](double a) { return a >= 6.0 ? 1.0 : a <= -6.0 ? -1.0 : erf(a); };
    const double f = 4.0 / w;
    const double e1 = erf_sat(f * (c * (ti - t0) - kd)), e0 = erf_sat(f * (c * (tprev - t0) - kd));
    const double g = A / (2.0 * c);
    F[((size_t)pt * 2) * B + b] = g * (e1 - e0);
    F[((size_t)pt * 2 + 1) * B + b] = g * (1.0 + e1);
}

__global__ void k_rhs_edges(int ne, int npad, int B, int nq, const int* __restrict__ ptidx,
                            const double* __restrict__ wf, const double* __restrict__ F,
                            const double* __restrict__ waves, double ti, double dt, double tmax, double eta,
                            double* __restrict__ rho1, double* __restrict__ rho2) {
    const int C2 = 2 * B;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npad * B; i += gridDim.x * blockDim.x) {
        const int r = i / B, b = i - r * B;
        if (r >= ne) {
            rho1[(size_t)r * C2 + b] = rho1[(size_t)r * C2 + B + b] = 0.0;
            rho2[(size_t)r * C2 + b] = rho2[(size_t)r * C2 + B + b] = 0.0;
            continue;
        }
        double d[3] = {0, 0, 0}, s[3] = {0, 0, 0};
#pragma unroll 2
        for (int q = 0; q < nq; q++) {
            const double* f = wf + ((size_t)r * nq + q) * 3;
            const double* v = F + (size_t)ptidx[r * nq + q] * 2 * B + b;
            const double ds = v[0], s1 = v[B];
#pragma unroll
            for (int t = 0; t < 3; t++) {
                d[t] = fma(f[t], ds, d[t]);
                s[t] = fma(f[t], s1, s[t]);
            }
        }
        const double* wv = waves + 10 * b;
        const double px = wv[1], py = wv[2], pz = wv[3], kx = wv[4], ky = wv[5], kz = wv[6];
        const double hx = (ky * pz - kz * py) / eta, hy = (kz * px - kx * pz) / eta, hz = (kx * py - ky * px) / eta;
        rho1[(size_t)r * C2 + b] = -(px * d[0] + py * d[1] + pz * d[2]) / dt;
        rho1[(size_t)r * C2 + B + b] = -(hx * d[0] + hy * d[1] + hz * d[2]) / dt;
        const bool on = ti <= wv[9];
        rho2[(size_t)r * C2 + b] = on ? -(px * s[0] + py * s[1] + pz * s[2]) / tmax : 0.0;
        rho2[(size_t)r * C2 + B + b] = on ? -(hx * s[0] + hy * s[1] + hz * s[2]) / tmax : 0.0;
    }
}

// W_a = sum_{k=a}^{kmax-1} variant-2 loop panel of step i-k (steps >= 1), a = 1..amax
__global__ void k_window(int n, int kmax, int amax, long long step_i, int R, size_t pstride,
                         const double* __restrict__ ring, double* __restrict__ win) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int k = kmax - 1; k >= 1; k--) {
            const long long src = step_i - k;
            if (src >= 1) {
                const int slot = (int)(src % R);
                acc += ring[(((size_t)slot * 2 + 0) * 3 + 2) * pstride + i];
            }
            if (k <= amax) win[(size_t)k * pstride + i] = acc;
        }
    }
}

// Current recovery (Eq. (dis_jm)) and running Fourier sums of the four parts.
__global__ void k_recover(int ne, int npad, int B, long long step_i, int R, double scale,
                          const double* __restrict__ ring, double* __restrict__ cur, int nfreq,
                          const double* __restrict__ omega, double dt, double* __restrict__ dft) {
    const int C2 = 2 * B;
    const size_t ps = (size_t)npad * C2;
    const int slot = (int)(step_i % R), slotp = (int)((step_i - 1) % R);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npad * B; i += gridDim.x * blockDim.x) {
        const int r = i / B, b = i - r * B;
        const double* L = ring + ((size_t)slot * 2 + 0) * 3 * ps;
        const double* S = ring + ((size_t)slot * 2 + 1) * 3 * ps;
        const double* Sp = ring + ((size_t)slotp * 2 + 1) * 3 * ps;
        const double lu = L[(size_t)r * C2 + b], lv = L[(size_t)r * C2 + B + b];
        const double su = S[(size_t)r * C2 + b], sv = S[(size_t)r * C2 + B + b];
        const double spu = step_i >= 2 ? Sp[(size_t)r * C2 + b] : 0.0;
        const double spv = step_i >= 2 ? Sp[(size_t)r * C2 + B + b] : 0.0;
        double q[4] = {lu, scale * (su - spu), lv, scale * (sv - spv)};
        const size_t nb = (size_t)npad * B;
        for (int j = 0; j < 4; j++) cur[j * nb + i] = q[j];
        for (int f = 0; f < nfreq; f++) {
            const double w = omega[f];
            double wr, wi;
            if (w == 0.0) {
                wr = dt;
                wi = 0.0;
            } else {
                // e^{-j w i dt} (e^{j w dt} - 1) / (j w)
                double s0, c0, s1, c1;
                sincos(-w * (double)step_i * dt, &s0, &c0);
                sincos(w * dt, &s1, &c1);
                const double ar = c1 - 1.0, ai = s1;          // e^{j w dt} - 1
                const double br = ai / w, bi = -ar / w;       // divided by j w
                wr = c0 * br - s0 * bi;
                wi = c0 * bi + s0 * br;
            }
            double* d = dft + (size_t)f * 4 * nb * 2;
            for (int j = 0; j < 4; j++) {
                d[(j * nb + i) * 2] += q[j] * wr;
                d[(j * nb + i) * 2 + 1] += q[j] * wi;
            }
        }
    }
}

// out[b][part][m] = x[iperm[m]][part*B + b]
__global__ void k_pack_w(int ne, int B, const int* __restrict__ iperm, const double* __restrict__ x,
                         double* __restrict__ out) {
    const int C2 = 2 * B;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * 2 * ne; i += gridDim.x * blockDim.x) {
        const int b = i / (2 * ne), rem = i - b * 2 * ne, part = rem / ne, m = rem - part * ne;
        out[i] = x[(size_t)iperm[m] * C2 + part * B + b];
    }
}

// Per wave b (the u and v columns b and B + b of a block vector): sc[b] =
// 2^-e, 2^e the power of two at or below max |x| over both columns (1 when
// x is zero). One CTA per wave.
__global__ void k_wave_scale(int npad, int B, const double* __restrict__ x, double* __restrict__ sc) {
    __shared__ double red[256];
    const int b = blockIdx.x, C2 = 2 * B;
    double m = 0.0;
    for (int i = threadIdx.x; i < 2 * npad; i += blockDim.x) {
        const int row = i >> 1, col = (i & 1) ? B + b : b;
        m = fmax(m, fabs(x[(size_t)row * C2 + col]));
    }
    red[threadIdx.x] = m;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) sc[b] = red[0] > 0.0 ? ldexp(1.0, -mot_scale_exponent(red[0])) : 1.0;
}

// x[:, b] and x[:, B + b] times sc[b] (inverse: divided by it; exact, powers of two)
__global__ void k_wave_apply(int npad, int B, const double* __restrict__ sc, int inverse, double* __restrict__ x) {
    const int C2 = 2 * B;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npad * C2; i += gridDim.x * blockDim.x) {
        const double f = sc[(i % C2) % B];
        x[i] = inverse ? x[i] / f : x[i] * f;
    }
}

// out[r][0..C) = a[r], out[r][C..2C) = b[r]
__global__ void k_pack2(int n, int C, const double* __restrict__ a, const double* __restrict__ b,
                        double* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * 2 * C; i += gridDim.x * blockDim.x) {
        const int r = i / (2 * C), c = i - r * 2 * C;
        out[i] = c < C ? a[(size_t)r * C + c] : b[(size_t)r * C + c - C];
    }
}

// q1 = X[:, :C] - P[:, :C] (= P^{SH} x1),  q2 = P[:, C:] (= P^L x2)
__global__ void k_unpack_q(int n, int C, const double* __restrict__ X, const double* __restrict__ P,
                           double* __restrict__ q1, double* __restrict__ q2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * C; i += gridDim.x * blockDim.x) {
        const int r = i / C, c = i - r * C;
        q1[i] = X[(size_t)r * 2 * C + c] - P[(size_t)r * 2 * C + c];
        q2[i] = P[(size_t)r * 2 * C + C + c];
    }
}

// out[b][j][m] = cur[j][iperm[m]][b]
__global__ void k_pack_cur(int ne, int npad, int B, const int* __restrict__ iperm, const double* __restrict__ cur,
                           double* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * 4 * ne; i += gridDim.x * blockDim.x) {
        const int b = i / (4 * ne), rem = i - b * 4 * ne, j = rem / ne, m = rem - j * ne;
        out[i] = cur[((size_t)j * npad + iperm[m]) * B + b];
    }
}

// Point currents of a frequency (blockIdx.y): the Fourier sums of j and m (loop
// and star parts summed here, after separate accumulation) times the quadrature's
// weight * basis function, summed over the edges whose tables share the point.
// cur[f][pt][12][b]: j_x re, im, j_y .., then m
__global__ void __launch_bounds__(128) k_point_currents(int npts, int npad, int B, int nq,
                                                        const int* __restrict__ ptr, const int* __restrict__ ent,
                                                        const double* __restrict__ wf, const double* __restrict__ D,
                                                        double* __restrict__ cur) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= npts * B) return;
    const int pt = i / B, b = i - pt * B;
    const size_t nb = (size_t)npad * B;
    D += (size_t)blockIdx.y * 4 * nb * 2;
    cur += (size_t)blockIdx.y * npts * 12 * B;
    double a[12];
#pragma unroll
    for (int k = 0; k < 12; k++) a[k] = 0.0;
    for (int e = ptr[pt]; e < ptr[pt + 1]; e++) {
        const size_t ix = (size_t)(ent[e] / nq) * B + b;
        const double jr = D[ix * 2] + D[(nb + ix) * 2], ji = D[ix * 2 + 1] + D[(nb + ix) * 2 + 1];
        const double mr = D[(2 * nb + ix) * 2] + D[(3 * nb + ix) * 2];
        const double mi = D[(2 * nb + ix) * 2 + 1] + D[(3 * nb + ix) * 2 + 1];
#pragma unroll
        for (int t = 0; t < 3; t++) {
            const double f = wf[(size_t)ent[e] * 3 + t];
            a[2 * t] = fma(jr, f, a[2 * t]);
            a[2 * t + 1] = fma(ji, f, a[2 * t + 1]);
            a[6 + 2 * t] = fma(mr, f, a[6 + 2 * t]);
            a[6 + 2 * t + 1] = fma(mi, f, a[6 + 2 * t + 1]);
        }
    }
#pragma unroll
    for (int k = 0; k < 12; k++) cur[((size_t)pt * 12 + k) * B + b] = a[k];
}

// Far field E_inf(r) = (j k / 4 pi) [eta r x (r x N) + r x L] / S(w); N, L the
// sums of the point currents times e^{j k r.x}. Bound by the FP64 units where
// there is work for all of them: 24 multiply-adds per point, direction, wave and
// frequency, and one sine and cosine per point, direction and frequency, shared
// by the waves (and by the three edges of a point's triangle). A cluster of up to
// eight CTAs takes DT directions and BT waves of one frequency (grid: direction tiles,
// wave tiles, frequencies); its threads are (share of the points, direction,
// wave), the shares are summed in shared memory and then over the cluster, in
// order. BT, DT and the cluster are chosen at the launch. A mot_fields call at 480
// edges: 8 waves, 3 frequencies, 181 directions 697 us, one wave and direction at
// 100 frequencies 135 us; with a launch per frequency over all waves 984 and 7254 us;
// with a CTA per output over its edges, no points or phases shared, 2750 and 157 us.
constexpr int FT = 256, FCL = 8;  // threads a CTA, most CTAs a cluster
template <int CL>
__global__ void __launch_bounds__(FT) k_far_field(int npts, int B, int nfreq, int f0, int ndir, int DT, int BT,
                                                  const double* __restrict__ pts, const double* __restrict__ cur,
                                                  const double* __restrict__ omega, const double* __restrict__ dirs,
                                                  const double* __restrict__ waves, double c, double eta,
                                                  double* __restrict__ E) {
    __shared__ double2 phase[FT];
    __shared__ double sums[FT * 12];  // shares [12][nsub][DT * BT]; their sums in share 0
    cg::cluster_group cl = cg::this_cluster();
    const int rk = (int)cl.block_rank(), t = threadIdx.x, f = f0 + blockIdx.z;
    const int G = DT * BT, nsub = FT / G, sub = t / G, l = t - sub * G, d = l / BT, q = l - d * BT;
    const bool on = sub < nsub;
    const int dir = blockIdx.x / CL * DT + d, b = blockIdx.y * BT + q;
    const bool wave = b < B;
    const double w = omega[f], k = w / c;
    cur += (size_t)blockIdx.z * npts * 12 * B;
    double r[3] = {0, 0, 0};
    if (on && dir < ndir)
        for (int i = 0; i < 3; i++) r[i] = dirs[3 * dir + i];
    double acc[12];
#pragma unroll
    for (int j = 0; j < 12; j++) acc[j] = 0.0;
    // a share takes BT consecutive points at a time: thread (d, q) the phase of point q
    const int step = CL * nsub * BT;
    for (int p0 = 0; p0 < npts; p0 += step) {
        const int first = p0 + (rk * nsub + sub) * BT, n = on ? max(0, min(BT, npts - first)) : 0;
        if (q < n) {
            const double* x = pts + 3 * (size_t)(first + q);
            double sn, cs;
            sincos(k * (r[0] * x[0] + r[1] * x[1] + r[2] * x[2]), &sn, &cs);
            phase[t] = make_double2(cs, sn);
        }
        __syncthreads();
        if (wave)
            for (int i = 0; i < n; i++) {
                const double2 e = phase[t - q + i];
                const double* v = cur + (size_t)(first + i) * 12 * B + b;
#pragma unroll
                for (int j = 0; j < 6; j++) {
                    const double re = v[(2 * j) * B], im = v[(2 * j + 1) * B];
                    acc[2 * j] = fma(re, e.x, fma(-im, e.y, acc[2 * j]));
                    acc[2 * j + 1] = fma(re, e.y, fma(im, e.x, acc[2 * j + 1]));
                }
            }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 12; j++) sums[j * FT + t] = acc[j];
    for (int m = nsub; m > 1;) {  // the upper half of the shares onto the lower
        const int half = (m + 1) / 2;
        __syncthreads();
        if (sub < m - half)
#pragma unroll
            for (int j = 0; j < 12; j++) sums[j * FT + t] += sums[j * FT + t + half * G];
        m = half;
    }
    cl.sync();
    if (t < G && t % CL == rk && dir < ndir && wave) {
        double v[12];
#pragma unroll
        for (int j = 0; j < 12; j++) {
            v[j] = 0.0;
            for (int u = 0; u < CL; u++) v[j] += cl.map_shared_rank(sums, u)[j * FT + t];
        }
        double out[6];
        for (int part = 0; part < 2; part++) {  // real, imag
            double N[3], Lv[3];
            for (int i = 0; i < 3; i++) {
                N[i] = v[2 * i + part];
                Lv[i] = v[6 + 2 * i + part];
            }
            const double rN = r[0] * N[0] + r[1] * N[1] + r[2] * N[2];
            // r x (r x N) = r (r.N) - N ; r x L
            const double rxL[3] = {r[1] * Lv[2] - r[2] * Lv[1], r[2] * Lv[0] - r[0] * Lv[2],
                                   r[0] * Lv[1] - r[1] * Lv[0]};
            for (int i = 0; i < 3; i++) out[2 * i + part] = eta * (r[i] * rN - N[i]) + rxL[i];
        }
        // multiply by j k / (4 pi) and divide by S = (A/c) e^{-j w t0} exp(-(w w_p / 8c)^2)
        const double* wv = waves + 10 * b;
        const double A = wv[0], wp = wv[7], t0 = wv[8];
        const double mag = (A / c) * exp(-(w * wp / (8.0 * c)) * (w * wp / (8.0 * c)));
        double ss, cs;
        sincos(-w * t0, &ss, &cs);
        const double Sr = mag * cs, Si = mag * ss;
        const double den = Sr * Sr + Si * Si;
        const double fac = k / (4.0 * 3.14159265358979323846);
        const size_t o = ((size_t)b * nfreq + f) * ndir + dir;
        for (int i = 0; i < 3; i++) {
            const double vr = -fac * out[2 * i + 1], vi = fac * out[2 * i];  // j k/(4 pi) * (vr + j vi)
            const double er = den > 0 ? (vr * Sr + vi * Si) / den : 0.0;
            const double ei = den > 0 ? (vi * Sr - vr * Si) / den : 0.0;
            E[(o * 3 + i) * 2] = er;
            E[(o * 3 + i) * 2 + 1] = ei;
        }
    }
    cl.sync();  // every read of a CTA's shared memory by the others is done
}

inline int grid_for(long long n, int bs = 256) {
    long long g = (n + bs - 1) / bs;
    if (g > 65535LL * 8) g = 65535LL * 8;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

namespace mot {

void launch_axpby(mot_handle* h, int n, double a, const double* x, double b, const double* y, double* z,
                  cudaStream_t s) {
    k_axpby<<<grid_for(n), 256, 0, s>>>(n, a, x, b, y, z);
    h->launches++;
}

void launch_variants(mot_handle* h, const double* x, double* dst, double eta, double etap, cudaStream_t s) {
    k_variants<<<grid_for((long long)h->npad * h->B), 256, 0, s>>>(h->npad, h->B, x, dst, eta, etap);
    h->launches++;
}

void launch_sigma_t(mot_handle* h, const double* x, int C, double* f, cudaStream_t s) {
    k_sigma_t<<<grid_for((long long)h->nf * C), 256, 0, s>>>(h->nf, C, h->d_face_edges, h->d_face_sgn, x, f);
    h->launches++;
}

void launch_sigma(mot_handle* h, const double* z, int C, double* x, cudaStream_t s) {
    k_sigma<<<grid_for((long long)h->ne * C), 256, 0, s>>>(h->ne, C, h->d_edge_faces, z, x);
    h->launches++;
}

void launch_lambda_t(mot_handle* h, const double* x, int C, double* v, cudaStream_t s) {
    const DCsr& A = h->vtx_edges;
    k_spmv<<<grid_for((long long)A.n * C), 256, 0, s>>>(A.n, C, A.rowptr, A.col, A.val, x, v);
    h->launches++;
}

void launch_lambda(mot_handle* h, const double* z, int C, double* x, cudaStream_t s) {
    k_lambda<<<grid_for((long long)h->ne * C), 256, 0, s>>>(h->ne, C, h->d_edge_verts, z, x);
    h->launches++;
}

void launch_spmv(mot_handle* h, const DCsr& A, const double* x, int C, double* y, cudaStream_t s) {
    k_spmv<<<grid_for((long long)A.n * C), 256, 0, s>>>(A.n, C, A.rowptr, A.col, A.val, x, y);
    h->launches++;
}

int launch_cg(mot_handle* h, const DCsr& A, const DCsr* A2, const double* f, int C, double* z, double* work,
              cudaStream_t s) {
    const int N = A.n;
    double* r = work;
    double* p = r + (size_t)N * C;
    double* q = p + (size_t)N * C;
    double* t = q + (size_t)N * C;
    int cw = 1;
    while (cw < 32 && (C + cw - 1) / cw > 128) cw *= 2;
    const int grid = (C + cw - 1) / cw;
    CsrV a{A.rowptr, A.col, A.val};
    CsrV a2{nullptr, nullptr, nullptr};
    if (A2) a2 = CsrV{A2->rowptr, A2->col, A2->val};
    const double tol = h->opt.cg_tol;
    const int mi = h->opt.cg_maxit;
    int* itmax = h->d_cg_iters;
    int* nc = h->d_cg_iters + 1;
#define MOT_CG_CASE(W)                                                                                         \
    case W:                                                                                                    \
        if (A2)                                                                                                \
            k_cg<W, true><<<grid, 1024, 0, s>>>(N, C, a, a2, f, z, r, p, q, t, tol, mi, itmax, nc);            \
        else                                                                                                   \
            k_cg<W, false><<<grid, 1024, 0, s>>>(N, C, a, a2, f, z, r, p, q, t, tol, mi, itmax, nc);           \
        break;
    switch (cw) {
        MOT_CG_CASE(1)
        MOT_CG_CASE(2)
        MOT_CG_CASE(4)
        MOT_CG_CASE(8)
        MOT_CG_CASE(16)
        MOT_CG_CASE(32)
    }
#undef MOT_CG_CASE
    h->launches++;
    return 0;
}

void launch_gemm_rect(mot_handle* h, int M, int K, const double* A, const double* X, int C, double* Y,
                      cudaStream_t s) {
    if (C <= 8) {
        const int g = grid_for((long long)M * 32);
        switch (C) {
            case 1: k_gemv_small<1><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            case 2: k_gemv_small<2><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            case 3: k_gemv_small<3><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            case 4: k_gemv_small<4><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            case 5: k_gemv_small<5><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            case 6: k_gemv_small<6><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            case 7: k_gemv_small<7><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
            default: k_gemv_small<8><<<g, 256, 0, s>>>(M, K, A, X, Y); break;
        }
        h->launches++;
        return;
    }
    const int tx = C <= 16 ? 16 : 32;
    const int tiles = ((M + GB_M - 1) / GB_M) * ((C + tx - 1) / tx);
    // about four CTAs per SM, each split at least two K blocks long
    int nsm = 148;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->dev);
    int S = std::max(1, std::min(4 * nsm / tiles, K / (2 * GB_K)));
    const int kchunk = ((K + S - 1) / S + GB_K - 1) / GB_K * GB_K;
    S = (K + kchunk - 1) / kchunk;
    double* ws = S > 1 ? split_workspace(h, sizeof(double) * (size_t)S * M * C) : nullptr;
    const bool split = ws != nullptr;
    const dim3 grid((M + GB_M - 1) / GB_M, (C + tx - 1) / tx, split ? S : 1);
    if (tx == 16)
        k_gemm<16><<<grid, 256, 0, s>>>(M, K, C, split ? kchunk : K, A, X, split ? ws : Y);
    else
        k_gemm<32><<<grid, 256, 0, s>>>(M, K, C, split ? kchunk : K, A, X, split ? ws : Y);
    h->launches++;
    if (split) {
        const long long n = (long long)M * C;
        k_split_sum<<<grid_for(n), 256, 0, s>>>(n, S, ws, Y);
        h->launches++;
    }
}

void launch_gemm(mot_handle* h, const double* A, const double* X, int C, double* Y, cudaStream_t s) {
    launch_gemm_rect(h, h->npad, h->npad, A, X, C, Y, s);
}

void launch_rhs(mot_handle* h, long long i, double* rho1, double* rho2, cudaStream_t s) {
    k_rhs_points<<<(h->npts * h->B + 127) / 128, 128, 0, s>>>(h->npts, h->B, h->d_pts, h->d_waves, i * h->dt,
                                                              (i - 1) * h->dt, h->c, h->d_ptfield);
    k_rhs_edges<<<grid_for((long long)h->npad * h->B, 128), 128, 0, s>>>(
        h->ne, h->npad, h->B, h->nq, h->d_ptidx, h->d_rhs_wf, h->d_ptfield, h->d_waves, i * h->dt, h->dt, h->tmax,
        h->eta, rho1, rho2);
    h->launches += 2;
}

void launch_window_sums(mot_handle* h, long long i, cudaStream_t s) {
    if (h->max_tail_lag < 1) return;
    const size_t ps = (size_t)h->npad * 2 * h->B;
    k_window<<<grid_for((long long)ps), 256, 0, s>>>((int)ps, h->kmax, h->max_tail_lag, i, h->R, ps, h->d_ring,
                                                     h->d_win);
    h->launches++;
}

void launch_recover(mot_handle* h, long long i, cudaStream_t s) {
    k_recover<<<grid_for((long long)h->npad * h->B), 256, 0, s>>>(h->ne, h->npad, h->B, i, h->R, h->tmax / h->dt,
                                                                  h->d_ring, h->d_cur, h->nfreq, h->d_omega, h->dt,
                                                                  h->d_dft);
    h->launches++;
}

void launch_pack_w(mot_handle* h, const double* x, double* out, cudaStream_t s) {
    k_pack_w<<<grid_for((long long)h->B * 2 * h->ne), 256, 0, s>>>(h->ne, h->B, h->d_iperm, x, out);
    h->launches++;
}

void launch_wave_scale(mot_handle* h, const double* x, double* sc, cudaStream_t s) {
    k_wave_scale<<<h->B, 256, 0, s>>>(h->npad, h->B, x, sc);
    h->launches++;
}

void launch_wave_apply(mot_handle* h, const double* sc, bool inverse, double* x, cudaStream_t s) {
    const long long n = (long long)h->npad * 2 * h->B;
    k_wave_apply<<<grid_for(n), 256, 0, s>>>(h->npad, h->B, sc, inverse ? 1 : 0, x);
    h->launches++;
}

void launch_pack2(mot_handle* h, const double* a, const double* b, int C, double* out, cudaStream_t s) {
    k_pack2<<<grid_for((long long)h->npad * 2 * C), 256, 0, s>>>(h->npad, C, a, b, out);
    h->launches++;
}

void launch_unpack_q(mot_handle* h, const double* X, const double* P, int C, double* q1, double* q2, cudaStream_t s) {
    k_unpack_q<<<grid_for((long long)h->npad * C), 256, 0, s>>>(h->npad, C, X, P, q1, q2);
    h->launches++;
}

void launch_pack_cur(mot_handle* h, double* out, cudaStream_t s) {
    k_pack_cur<<<grid_for((long long)h->B * 4 * h->ne), 256, 0, s>>>(h->ne, h->npad, h->B, h->d_iperm, h->d_cur, out);
    h->launches++;
}

void launch_far_field(mot_handle* h, int n_dir, const double* dirs, double* E, cudaStream_t s) {
    if (h->B * h->nfreq * n_dir == 0) return;
    const size_t nb = (size_t)h->npad * h->B;
    int nsm = 148;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->dev);
    for (int f0 = 0; f0 < h->nfreq; f0 += h->ptcur_freqs) {
        const int nf = std::min(h->ptcur_freqs, h->nfreq - f0);
        // A cluster takes all waves, for which its phases then serve, unless that leaves SMs idle
        // (one direction and frequency, 64 waves at 480 edges: a call takes 590 us with all of them
        // in eight CTAs, 125 us at eight waves a cluster); then directions, up to a warp of
        // (direction, wave) pairs or eight, which cost no phases but share a cluster's reductions.
        auto ctas = [&](int bt, int dt) {
            return (long long)((h->B + bt - 1) / bt) * ((n_dir + dt - 1) / dt) * nf * FCL;
        };
        int BT = h->B, DT = 1;
        while (BT > 8 && ctas(BT, 1) < 2 * nsm) BT = (BT + 1) / 2;
        while (2 * DT <= std::min(8, n_dir) && DT * BT < 32 && ctas(BT, 2 * DT) >= 2 * nsm) DT *= 2;
        // Shares of a few points are mostly reduction: fewer CTAs a cluster, if the chip stays
        // covered (one wave and direction, 100 frequencies, 480 edges: a call 135 us, with eight 162)
        int CL = FCL;
        while (CL > 2 && h->npts < 4 * CL * (FT / (DT * BT)) && ctas(BT, DT) / FCL * (CL / 2) >= 2 * nsm) CL /= 2;
        k_point_currents<<<dim3((h->npts * h->B + 127) / 128, nf), 128, 0, s>>>(
            h->npts, h->npad, h->B, h->nq, h->d_ptptr, h->d_ptent, h->d_rhs_wf, h->d_dft + (size_t)f0 * 4 * nb * 2,
            h->d_ptcur);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((n_dir + DT - 1) / DT * CL, (h->B + BT - 1) / BT, nf);
        cfg.blockDim = dim3(FT);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, CL == 8 ? k_far_field<8> : CL == 4 ? k_far_field<4> : k_far_field<2>, h->npts, h->B,
                           h->nfreq, f0, n_dir, DT, BT, (const double*)h->d_pts, (const double*)h->d_ptcur,
                           (const double*)h->d_omega, dirs, (const double*)h->d_waves, h->c, h->eta, E);
        h->launches += 2;
    }
}

}  // namespace mot
