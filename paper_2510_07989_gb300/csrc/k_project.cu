// Solves behind the quasi-Helmholtz projectors and the Gram matrix (paper
// Section IV-B, Section III), one launch each:
//   faces    out = Sigma z,  Sigma^T Sigma z = Sigma^T x       (P^Sigma x)
//   vertices out = Lambda z, Lambda^T Lambda z = Lambda^T x    (P^Lambda x)
//   gram     out = z,        G z = x
// A z = f is solved by FP64 iterative refinement with an FP32 dense inverse M
// formed at load (of A + 11^T/N for the graph Laplacians): d = M r, z += d,
// r -= A d until |r| <= cg_tol |f| in every column. d needs no accuracy beyond
// the digits a sweep gains (about six); z, r and A d are FP64, r by recurrence
// as in CG, so three sweeps reach the tolerance CG took 30 to 125 iterations
// for, at two block-wide reductions each (1920 edges, one wave: 1.27 ms a
// Laplacian solve, 2.1 ms a Gram solve).
//
// A cluster of eight CTAs owns CW columns and all rows (each CTA an eighth).
// What bounds a sweep is reading M from L2 once per cluster (6.6 MB at 1280
// faces) at about 60 bytes per clock and SM, and below some 500 rows the
// latency of the cluster barriers, two per sweep. CW is 8 where a batch has the
// columns, since M is read per cluster.
//
// A graph Laplacian is singular with the constants as its null space (connected
// surface); f sums to zero only up to rounding, and its column mean is removed
// first: the solve is the consistent one whose minimum-norm solution is the
// pseudo-inverse of Section IV-B. Every column is scaled by a power of two to
// O(1) (exact) and its solution scaled back, so that a late, decayed march
// neither underflows nor loses digits.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "mot_internal.h"

namespace {

namespace cg = cooperative_groups;

constexpr int PT = 512;  // threads per CTA
constexpr int PW = PT / 32;
constexpr int CL = 8;    // CTAs per cluster
constexpr int REFINE_SMEM = 220 * 1024;

enum { FACES = 0, VERTS = 1, GRAM = 2 };

struct Problem {
    int N;               // rows of A
    int ld;              // leading dimension of M
    int ne, C;
    const float* M;
    const int *rp, *ci;  // A, CSR
    const double* va;
    const int *in_a, *in_c;  // faces: edges [N][3]; vertices: CSR of Lambda^T
    const double* in_v;      //        signs
    const int* out_ab;       // edge -> its two faces (c+, c-) or vertices (v-, v+)
};

// v[0 .. NV) summed over the warp; the lane returns the sum whose index is in
// its high bits (bit 4 chooses the upper half of the values, bit 3 of those, ..),
// the low bits left over hold copies.
template <int NV>
__device__ __forceinline__ float warp_sums(float (&v)[NV]) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1) {
        const bool hi = lane & off;
#pragma unroll
        for (int i = 0; i < n / 2; i++) {
            const float keep = hi ? v[n / 2 + i] : v[i], send = hi ? v[i] : v[n / 2 + i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
        off >>= 1;
    }
    float s = v[0];
    for (; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

__device__ __forceinline__ double pow2_at(double m, int sign) {
    return m > 0.0 && m < INFINITY ? ldexp(1.0, sign * mot_scale_exponent(m)) : 1.0;
}

template <int CW, int MODE>
__global__ void __launch_bounds__(PT) k_refine_solve(Problem Q, const double* __restrict__ x, double* __restrict__ out,
                                                     double* __restrict__ work, double tol, int maxit,
                                                     int* __restrict__ it_max, int* __restrict__ noconv) {
    constexpr int RPW = CW == 8 ? 4 : 8;         // rows of M a warp multiplies together: 16 to 32 loads in flight a lane
    extern __shared__ __align__(16) float rs[];  // [N][CW] r in FP32 (CW = 8: two halves of 4 columns)
    __shared__ double red[PW][CW];
    __shared__ double col[3][CW];                // this CTA's column values of the three reductions
    __shared__ double mean_s[CW], scale_s[CW], thr_s[CW];
    __shared__ int open_s[2];                    // this CTA still has a row above the tolerance (by sweep parity)
    cg::cluster_group cl = cg::this_cluster();
    const int rk = (int)cl.block_rank(), grp = blockIdx.x / CL;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int N = Q.N, C = Q.C;
    const int rows = (N + CL - 1) / CL, r0 = min(N, rk * rows), r1 = min(N, r0 + rows);
    const int c0 = grp * CW, c = t % CW;
    const bool cv = c0 + c < C;
    const int RS = PT / CW, tr = t / CW;
    const size_t slab = (size_t)N * CW;
    double* r = work + (size_t)grp * 3 * slab;
    double* z = r + slab;
    float* d = reinterpret_cast<float*>(z + slab);
    float* rg = d + slab;
    auto sidx = [&](int row, int cc) { return CW == 8 ? ((cc >> 2) * N + row) * 4 + (cc & 3) : row * CW + cc; };
    // the CTA's value of column c (sum, or maximum of non-negative values) into col[slot]
    auto block_value = [&](double v, bool mx, int slot) {
#pragma unroll
        for (int off = 16; off >= CW; off >>= 1) {
            const double o = __shfl_xor_sync(0xffffffffu, v, off);
            v = mx ? fmax(v, o) : v + o;
        }
        if (lane < CW) red[warp][lane] = v;
        __syncthreads();
        if (t < CW) {
            double s = 0.0;
            for (int w = 0; w < PW; w++) s = mx ? fmax(s, red[w][t]) : s + red[w][t];
            col[slot][t] = s;
        }
        cl.sync();
    };
    auto cluster_value = [&](int slot, int cc, bool mx) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < CL; k++) {
            const double o = cl.map_shared_rank(&col[slot][0], k)[cc];
            s = mx ? fmax(s, o) : s + o;
        }
        return s;
    };
    // f, its mean, its scale
    double acc = 0.0;
    for (int row = r0 + tr; row < r1; row += RS) {
        double f = 0.0;
        if (cv) {
            if (MODE == FACES) {
#pragma unroll
                for (int j = 0; j < 3; j++)
                    f += Q.in_v[3 * row + j] * x[(size_t)Q.in_a[3 * row + j] * C + c0 + c];
            } else if (MODE == VERTS) {
                for (int j = Q.in_a[row]; j < Q.in_a[row + 1]; j++)
                    f = fma(Q.in_v[j], x[(size_t)Q.in_c[j] * C + c0 + c], f);
            } else {
                f = x[(size_t)row * C + c0 + c];
            }
        }
        r[(size_t)row * CW + c] = f;
        acc += f;
    }
    double mean = 0.0;
    if (MODE != GRAM) {
        block_value(acc, false, 0);
        if (t < CW) mean_s[t] = cluster_value(0, t, false) / (double)N;
        __syncthreads();
        mean = mean_s[c];
    }
    acc = 0.0;
    for (int row = r0 + tr; row < r1; row += RS) acc = fmax(acc, fabs(r[(size_t)row * CW + c] - mean));
    block_value(acc, true, 1);
    if (t < CW) scale_s[t] = cluster_value(1, t, true);
    __syncthreads();
    const double top = scale_s[c], sc = pow2_at(top, -1);
    acc = 0.0;
    for (int row = r0 + tr; row < r1; row += RS) {
        const size_t ix = (size_t)row * CW + c;
        const double v = (r[ix] - mean) * sc;
        r[ix] = v;
        z[ix] = 0.0;
        rg[ix] = (float)v;
        acc = fma(v, v, acc);
    }
    block_value(acc, false, 2);  // its barrier also publishes rg
    // |r|_inf <= tol |f|_2 / sqrt(N) implies |r|_2 <= tol |f|_2
    if (t < CW) thr_s[t] = tol * sqrt(cluster_value(2, t, false) / (double)N);
    if (t < 2) open_s[t] = 0;
    __syncthreads();
    const double thr = thr_s[c];
    int it = 0;
    // lost: this thread saw a value that is no number (looked at as an integer: the FP64
    // unit's comparisons cost what its multiply-adds do)
    auto no_number = [](double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; };
    bool open = true, lost = no_number(thr);
    while (open && it < maxit) {
        for (int i = t; i < N * CW; i += PT) rs[sidx(i / CW, i % CW)] = __ldcg(rg + i);
        __syncthreads();
        // d = M r, own rows
        for (int row = r0 + warp * RPW; row < r1; row += PW * RPW) {
            float a[RPW * CW];
#pragma unroll
            for (int i = 0; i < RPW * CW; i++) a[i] = 0.f;
            const float* m[RPW];
#pragma unroll
            for (int i = 0; i < RPW; i++) m[i] = Q.M + (size_t)min(row + i, r1 - 1) * Q.ld;
#pragma unroll 4
            for (int k = lane; k < N; k += 32) {
                float v[CW];
                if (CW == 8) {
                    *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(rs + k * 4);
                    *reinterpret_cast<float4*>(v + CW / 2) = *reinterpret_cast<const float4*>(rs + (size_t)(N + k) * 4);
                } else if (CW == 4) {
                    *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(rs + k * 4);
                } else {
                    *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(rs + k * 2);
                }
#pragma unroll
                for (int i = 0; i < RPW; i++) {
                    const float mv = __ldg(m[i] + k);
#pragma unroll
                    for (int q = 0; q < CW; q++) a[i * CW + q] = fmaf(mv, v[q], a[i * CW + q]);
                }
            }
            const float s = warp_sums<RPW * CW>(a);
            constexpr int COPIES = 32 / (RPW * CW);
            const int i = lane / COPIES;  // row + i / CW, column i % CW
            if (lane % COPIES == 0 && row + i / CW < r1) d[(size_t)(row + i / CW) * CW + i % CW] = s;
        }
        cl.sync();
        if (t == 0) open_s[(it + 1) & 1] = 0;  // every CTA has read the last sweep's
        // z += d, r -= A d, own rows
        bool mine = false;
        for (int row = r0 + tr; row < r1; row += RS) {
            const size_t ix = (size_t)row * CW + c;
            double s = 0.0;
            for (int j = Q.rp[row]; j < Q.rp[row + 1]; j++)
                s = fma(Q.va[j], (double)__ldcg(d + (size_t)Q.ci[j] * CW + c), s);
            const double rn = r[ix] - s;
            r[ix] = rn;
            z[ix] += (double)__ldcg(d + ix);
            rg[ix] = (float)rn;
            mine |= fabs(rn) > thr;  // a row or threshold that is no number ends its column's sweeps ..
            lost |= no_number(rn);
        }
        if (mine) open_s[it & 1] = 1;
        cl.sync();
        open = false;
#pragma unroll
        for (int k = 0; k < CL; k++) open |= cl.map_shared_rank(open_s, k)[it & 1] != 0;
        it++;
    }
    if (lost) atomicAdd(noconv, 1);  // .. and counts as not converged
    const double us = pow2_at(top, 1);
    if (MODE == GRAM) {
        for (int row = r0 + tr; row < r1; row += RS)
            if (cv) out[(size_t)row * C + c0 + c] = z[(size_t)row * CW + c] * us;
    } else {
        const int er = (Q.ne + CL - 1) / CL, e0 = rk * er, e1 = min(Q.ne, e0 + er);
        for (int e = e0 + tr; e < e1; e += RS) {
            const int a = Q.out_ab[2 * e], b = Q.out_ab[2 * e + 1];
            const double va = __ldcg(z + (size_t)a * CW + c), vb = __ldcg(z + (size_t)b * CW + c);
            // Sigma: z[c+] - z[c-]; Lambda: z[v+] - z[v-], stored as (v-, v+)
            if (cv) out[(size_t)e * C + c0 + c] = (MODE == FACES ? va - vb : vb - va) * us;
        }
    }
    if (rk == 0 && t == 0) {
        atomicMax(it_max, it);
        if (open) atomicAdd(noconv, 1);
    }
    cl.sync();  // every read of a CTA's shared memory by the others is done
}

template <int CW, int MODE>
void launch(mot_handle* h, const Problem& q, const double* x, double* out, double* work, int maxit, cudaStream_t s) {
    const size_t smem = sizeof(float) * (size_t)q.N * CW;
    static std::atomic<unsigned long long> attr{0};
    mot::once_per_device(attr, h->dev, [] {
        cudaFuncSetAttribute(k_refine_solve<CW, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, REFINE_SMEM);
    });
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((q.C + CW - 1) / CW * CL);
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_refine_solve<CW, MODE>, q, x, out, work, h->opt.cg_tol, maxit, h->d_cg_iters,
                       h->d_cg_iters + 1);
    h->launches++;
}

template <int MODE>
void launch_mode(mot_handle* h, const Problem& q, const double* x, double* out, double* work, int maxit,
                 cudaStream_t s) {
    // as many columns per cluster as there are and as fit in shared memory
    const int cap = (int)(REFINE_SMEM / sizeof(float) / (size_t)q.N);
    if (q.C > 4 && cap >= 8)
        launch<8, MODE>(h, q, x, out, work, maxit, s);
    else if (q.C > 2 && cap >= 4)
        launch<4, MODE>(h, q, x, out, work, maxit, s);
    else
        launch<2, MODE>(h, q, x, out, work, maxit, s);
}

}  // namespace

namespace mot {

// r in FP32 for two columns has to fit in shared memory
bool refine_fits(int N) { return sizeof(float) * 2 * (size_t)N <= REFINE_SMEM; }

// work: 3 N doubles per column, the columns rounded up to the cluster's
void launch_project_refine(mot_handle* h, bool faces, const double* x, int C, double* out, double* work, int maxit,
                           cudaStream_t s) {
    Problem q{};
    q.ne = h->ne;
    q.C = C;
    const DCsr& A = faces ? h->Lf : h->Lv;
    q.N = A.n;
    q.ld = (A.n + 63) / 64 * 64;
    q.M = faces ? h->d_Lfinvf : h->d_Lvinvf;
    q.rp = A.rowptr;
    q.ci = A.col;
    q.va = A.val;
    q.in_a = faces ? h->d_face_edges : h->vtx_edges.rowptr;
    q.in_c = faces ? nullptr : h->vtx_edges.col;
    q.in_v = faces ? h->d_face_sgn : h->vtx_edges.val;
    q.out_ab = faces ? h->d_edge_faces : h->d_edge_verts;
    if (faces)
        launch_mode<FACES>(h, q, x, out, work, maxit, s);
    else
        launch_mode<VERTS>(h, q, x, out, work, maxit, s);
}

void launch_gram_refine(mot_handle* h, const double* y, int C, double* out, double* work, int maxit, cudaStream_t s) {
    Problem q{};
    q.ne = h->ne;
    q.C = C;
    q.N = h->G.n;
    q.ld = (h->npad + 63) / 64 * 64;
    q.M = h->d_Ginvf;
    q.rp = h->G.rowptr;
    q.ci = h->G.col;
    q.va = h->G.val;
    launch_mode<GRAM>(h, q, y, out, work, maxit, s);
}

}  // namespace mot
