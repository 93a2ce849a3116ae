// Batched GMRES of the Q_0 solve (paper Eq. (MOT)): one launch starts a cycle,
// one launch orthogonalises a new Krylov vector and updates the least-squares
// problem, one solves it, one combines the basis.
//
// System b of the batch uses columns b and B + b of a block vector
// [npad][2B]. A thread-block cluster owns G systems (4, so that a row's
// columns fill a 32-byte sector; 1 for B = 1) and all rows: every CTA keeps its
// part of the new vector in registers, and the dot products are summed over
// the cluster through distributed shared memory, in rank order (every CTA
// gets the same sums). What bounds it is the FP64 rate of an SM (two
// multiply-adds per clock) and the latency of the cluster barriers: three
// reductions per iteration.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "mot_internal.h"

namespace {

namespace cg = cooperative_groups;

constexpr int GT = 256;      // threads per CTA
constexpr int NW = GT / 32;
constexpr int MAXE = 12;     // elements per thread kept in registers
constexpr int MAXCL = 8;     // CTAs per cluster (the portable limit)

struct GmState {
    double* H;       // [B][m + 1][m], rotated columns
    double* g;       // [B][m + 1]
    double* cs;      // [B][m]
    double* sn;
    double* bnorm;   // [B]
    double* resid;   // [B] of the current iterate
    double* resid0;  // [B] at the start of the solve
    int* active;     // [B]
    int* jend;       // [B]
    int m;
};

// Elements of group grp (G systems): index (row * 2 + part) * G + q; element e
// of thread t of cluster rank rk is index (e * CL + rk) * GT + t.
template <int G>
struct Part {
    int npad, B, C2, g0, q, rk, cl, t;
    __device__ Part(int npad_, int B_, int rk_, int cl_)
        : npad(npad_), B(B_), C2(2 * B_), rk(rk_), cl(cl_), t(threadIdx.x) {
        g0 = (int)(blockIdx.x / cl_) * G;
        q = t % G;
    }
    __device__ int elements() const { return (2 * npad * G + cl * GT - 1) / (cl * GT); }
    // offset in a block vector, or -1 outside it
    __device__ long long at(int e) const {
        const long long rp = ((long long)(e * cl + rk) * GT + t) / G;
        const long long row = rp >> 1;
        const int part = (int)(rp & 1);
        return row < npad && g0 + q < B ? row * C2 + part * B + g0 + q : -1;
    }
};

// The new vector's elements of a thread: in registers, or (more than MAXE per
// thread) where it stands in global memory.
template <bool REG>
struct Elems {
    double r[REG ? MAXE : 1];
};

// Sums of p[0 .. 3] over the lanes of a warp with the same lane % G: lane
// (i << 3) | .. returns the sum of p[i], i = 0 .. 3 (the first exchange halves
// the values a lane carries, so four sums cost 6 (G = 1) or 4 adds, not 20 or 12).
template <int G>
__device__ __forceinline__ double warp_sum4(const double (&p)[4]) {
    const int lane = threadIdx.x & 31;
    const bool hi = lane & 16, md = lane & 8;
    const double k0 = hi ? p[2] : p[0], s0 = hi ? p[0] : p[2];
    const double k1 = hi ? p[3] : p[1], s1 = hi ? p[1] : p[3];
    const double a = k0 + __shfl_xor_sync(0xffffffffu, s0, 16);
    const double b = k1 + __shfl_xor_sync(0xffffffffu, s1, 16);
    double v = (md ? b : a) + __shfl_xor_sync(0xffffffffu, md ? a : b, 8);
#pragma unroll
    for (int off = 4; off >= G; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// out[i] (i < n * G: sum i / G of system i % G) = the cluster's sums of what the
// warps left in red[warp][i]; part is this CTA's own slot, read by the others
// after the cluster barrier.
__device__ __forceinline__ void cluster_sums(int n, const double* red, double* part, double* out, int cl) {
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += GT) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < NW; w++) s += red[w * n + i];
        part[i] = s;
    }
    cg::cluster_group c = cg::this_cluster();
    c.sync();
    for (int i = threadIdx.x; i < n; i += GT) {
        double s = 0.0;
        for (int r = 0; r < cl; r++) s += c.map_shared_rank(part, r)[i];
        out[i] = s;
    }
    __syncthreads();
}

// red[warp][v * G + q] = this warp's part of <V_v, w>, v < nv
template <int G, bool REG>
__device__ __forceinline__ void dots(const Part<G>& P, int ne, const double* V, size_t vs, int nv, const double* w,
                                     const Elems<REG>& E, double* red) {
    const int lane = P.t & 31, warp = P.t >> 5, n = nv * G;
    for (int v0 = 0; v0 < nv; v0 += 4) {
        double p[4] = {0.0, 0.0, 0.0, 0.0};
        if (REG) {
#pragma unroll
            for (int e = 0; e < MAXE; e++) {
                const long long ix = e < ne ? P.at(e) : -1;
                if (ix < 0) continue;
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (v0 + i < nv) p[i] = fma(V[(size_t)(v0 + i) * vs + ix], E.r[e], p[i]);
            }
        } else {
            for (int e = 0; e < ne; e++) {
                const long long ix = P.at(e);
                if (ix < 0) continue;
                const double x = w[ix];
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (v0 + i < nv) p[i] = fma(V[(size_t)(v0 + i) * vs + ix], x, p[i]);
            }
        }
        const double s = warp_sum4<G>(p);
        const int v = v0 + (((lane >> 4) & 1) << 1 | ((lane >> 3) & 1));
        if ((lane & 7) < G && v < nv) red[warp * n + v * G + (lane & 7)] = s;
    }
}

// w -= sum_v V_v h[v]
template <int G, bool REG>
__device__ __forceinline__ void project_out(const Part<G>& P, int ne, const double* V, size_t vs, int nv, double* w,
                                            Elems<REG>& E, const double* h) {
    if (REG) {
#pragma unroll
        for (int e = 0; e < MAXE; e++) {
            const long long ix = e < ne ? P.at(e) : -1;
            if (ix < 0) continue;
            double s = 0.0;
#pragma unroll 4
            for (int v = 0; v < nv; v++) s = fma(V[(size_t)v * vs + ix], h[v * G + P.q], s);
            E.r[e] -= s;
        }
    } else {
        for (int e = 0; e < ne; e++) {
            const long long ix = P.at(e);
            if (ix < 0) continue;
            double s = 0.0;
#pragma unroll 4
            for (int v = 0; v < nv; v++) s = fma(V[(size_t)v * vs + ix], h[v * G + P.q], s);
            w[ix] -= s;
        }
    }
}

// red[warp][q] = this warp's part of |w|^2
template <int G, bool REG>
__device__ __forceinline__ void square(const Part<G>& P, int ne, const double* w, const Elems<REG>& E, double* red) {
    double p[4] = {0.0, 0.0, 0.0, 0.0};
    if (REG) {
#pragma unroll
        for (int e = 0; e < MAXE; e++)
            if (e < ne) p[0] = fma(E.r[e], E.r[e], p[0]);
    } else {
        for (int e = 0; e < ne; e++) {
            const long long ix = P.at(e);
            const double x = ix >= 0 ? w[ix] : 0.0;
            p[0] = fma(x, x, p[0]);
        }
    }
    const double s = warp_sum4<G>(p);
    const int lane = P.t & 31;
    if (lane < G) red[(P.t >> 5) * G + lane] = s;
}

template <int G, bool REG>
__device__ __forceinline__ void load(const Part<G>& P, int ne, const double* w, Elems<REG>& E) {
    if (!REG) return;
#pragma unroll
    for (int e = 0; e < MAXE; e++) {
        const long long ix = e < ne ? P.at(e) : -1;
        E.r[e] = ix >= 0 ? w[ix] : 0.0;
    }
}

// v = w * f (the group's systems that are live), else 0
template <int G, bool REG>
__device__ __forceinline__ void store_scaled(const Part<G>& P, int ne, const double* w, const Elems<REG>& E, double f,
                                             double* v) {
    if (REG) {
#pragma unroll
        for (int e = 0; e < MAXE; e++) {
            const long long ix = e < ne ? P.at(e) : -1;
            if (ix >= 0) v[ix] = E.r[e] * f;
        }
    } else {
        for (int e = 0; e < ne; e++) {
            const long long ix = P.at(e);
            if (ix >= 0) v[ix] = w[ix] * f;
        }
    }
}

// Below this norm a vector of an O(1) system is a breakdown: its system is done.
constexpr double TINY_NORM = 1e-150;

// Start of a cycle: beta = |r| per system, V_0 = r / beta. On the first cycle
// also the reference norm |b| (b == r: one vector).
template <int G, bool REG>
__global__ void __launch_bounds__(GT) k_gm_begin(int npad, int B, const double* __restrict__ b, int first,
                                                 const double* __restrict__ r, double* __restrict__ V0, GmState S) {
    extern __shared__ double sm[];
    cg::cluster_group c = cg::this_cluster();
    const int cl = (int)c.num_blocks(), rk = (int)c.block_rank();
    const Part<G> P(npad, B, rk, cl);
    const int ne = P.elements();
    double* red = sm;                // NW x G
    double* part = red + NW * G;     // 2 x G (one slot per reduction)
    double* out = part + 2 * G;      // 2 x G
    Elems<REG> E;
    const bool other = first && b != r;
    if (other) {
        load<G, REG>(P, ne, b, E);
        square<G, REG>(P, ne, b, E, red);
        cluster_sums(G, red, part, out, cl);
    }
    load<G, REG>(P, ne, r, E);
    square<G, REG>(P, ne, r, E, red);
    cluster_sums(G, red, part + G, out + G, cl);
    const int sys = P.g0 + P.q;
    const double beta = sqrt(out[G + P.q]);
    double bn = 0.0;
    if (sys < B) bn = first ? (other ? sqrt(out[P.q]) : beta) : S.bnorm[sys];
    const bool live = beta > 0.0 && bn > 0.0;
    store_scaled<G, REG>(P, ne, r, E, live && beta > TINY_NORM ? 1.0 / beta : 0.0, V0);
    if (rk == 0 && P.t < G && sys < B) {
        S.g[(size_t)sys * (S.m + 1)] = beta;
        if (first) S.bnorm[sys] = bn;
        if (first) S.resid0[sys] = bn > 0.0 ? beta / bn : 0.0;
        S.active[sys] = live ? 1 : 0;
        S.jend[sys] = 0;
        S.resid[sys] = bn > 0.0 ? beta / bn : 0.0;
    }
    c.sync();  // every read of a CTA's shared memory by the others is done
}

// Iteration j: w (= Q_0 V_j) orthogonalised against V_0 .. V_j (classical
// Gram-Schmidt twice), V_{j+1} = w / |w|, and the new column of the rotated
// Hessenberg matrix. A system is done at a residual of tol |b|, or of gain times
// its residual at the start. A system that is done writes V_{j+1} = 0 from its next
// iteration on and keeps its state, so iterations past its end change nothing.
template <int G, bool REG>
__global__ void __launch_bounds__(GT) k_gm_iter(int npad, int B, int j, const double* __restrict__ V, size_t vs,
                                                double* __restrict__ w, double* __restrict__ Vnext, double tol,
                                                double gain, GmState S) {
    extern __shared__ double sm[];
    cg::cluster_group c = cg::this_cluster();
    const int cl = (int)c.num_blocks(), rk = (int)c.block_rank();
    const Part<G> P(npad, B, rk, cl);
    const int ne = P.elements(), nv = j + 1, n = nv * G;
    double* red = sm;               // NW x n
    double* part = red + NW * n;    // 2 n + G (one slot per reduction)
    double* h1 = part + 2 * n + G;  // n
    double* h2 = h1 + n;            // n
    double* nr = h2 + n;            // G
    double* rot = nr + G;           // 2 x j x G: cosines, sines of the earlier rotations
    const int sys = P.g0 + P.q;
    const bool valid = sys < B;
    const bool live = valid && S.active[sys] != 0;  // read before the first barrier, written after the last
    if (rk == 0)
        for (int i = P.t; i < j * G; i += GT) {
            const int b = P.g0 + i % G;
            rot[i] = b < B ? S.cs[(size_t)b * S.m + i / G] : 1.0;
            rot[j * G + i] = b < B ? S.sn[(size_t)b * S.m + i / G] : 0.0;
        }
    Elems<REG> E;
    load<G, REG>(P, ne, w, E);
    dots<G, REG>(P, ne, V, vs, nv, w, E, red);
    cluster_sums(n, red, part, h1, cl);
    project_out<G, REG>(P, ne, V, vs, nv, w, E, h1);
    dots<G, REG>(P, ne, V, vs, nv, w, E, red);
    cluster_sums(n, red, part + n, h2, cl);
    project_out<G, REG>(P, ne, V, vs, nv, w, E, h2);
    square<G, REG>(P, ne, w, E, red);
    cluster_sums(G, red, part + 2 * n, nr, cl);
    const double nrm = sqrt(nr[P.q]);
    store_scaled<G, REG>(P, ne, w, E, live && nrm > TINY_NORM ? 1.0 / nrm : 0.0, Vnext);
    if (rk == 0 && P.t < G && live) {
        double* Hb = S.H + (size_t)sys * (S.m + 1) * S.m;
        double* gb = S.g + (size_t)sys * (S.m + 1);
        double a = h1[P.q] + h2[P.q];
        for (int i = 0; i < j; i++) {
            const double x = h1[(i + 1) * G + P.q] + h2[(i + 1) * G + P.q];
            const double cc = rot[i * G + P.q], ss = rot[(j + i) * G + P.q];
            Hb[(size_t)i * S.m + j] = cc * a + ss * x;
            a = -ss * a + cc * x;
        }
        const double d = hypot(a, nrm);
        double cc = 1.0, ss = 0.0;
        if (d > 0.0) {
            cc = a / d;
            ss = nrm / d;
        }
        S.cs[(size_t)sys * S.m + j] = cc;
        S.sn[(size_t)sys * S.m + j] = ss;
        Hb[(size_t)j * S.m + j] = d;
        const double gj = gb[j];
        gb[j + 1] = -ss * gj;
        gb[j] = cc * gj;
        const double rr = fabs(ss * gj) / S.bnorm[sys];
        S.resid[sys] = rr;
        S.jend[sys] = j + 1;
        if (rr <= fmax(tol, gain * S.resid0[sys]) || !(nrm > 0.0)) S.active[sys] = 0;
    }
    c.sync();
}

// y = H^{-1} g (upper triangular, size jend[b]) into y[i][b], i < nv (0 past
// jend). One CTA per system, the triangle staged in shared memory: read entry
// by entry from global memory by one thread per system it took 277 us at 60
// vectors.
__global__ void __launch_bounds__(128) k_gm_back(int B, int nv, GmState S, double* __restrict__ y) {
    extern __shared__ double sm[];
    const int b = blockIdx.x, n = min(S.jend[b], nv);
    const double* Hb = S.H + (size_t)b * (S.m + 1) * S.m;
    double* rhs = sm;       // nv
    double* tri = sm + nv;  // row i at i n
    for (int i = threadIdx.x; i < n; i += 128) rhs[i] = S.g[(size_t)b * (S.m + 1) + i];
    for (int e = threadIdx.x; e < n * n; e += 128) {
        const int i = e / n, k = e - i * n;
        if (k >= i) tri[e] = Hb[(size_t)i * S.m + k];
    }
    __syncthreads();
    for (int i = n - 1; i >= 0; i--) {
        const double d = tri[i * n + i], yi = d != 0.0 ? rhs[i] / d : 0.0;
        __syncthreads();
        for (int k = threadIdx.x; k < i; k += 128) rhs[k] -= tri[k * n + i] * yi;
        if (threadIdx.x == 0) rhs[i] = yi;
        __syncthreads();
    }
    for (int i = threadIdx.x; i < nv; i += 128) y[i * B + b] = i < n ? rhs[i] : 0.0;
}

// x = (add ? x : 0) + sum_v Z_v y[v][b]
__global__ void __launch_bounds__(256) k_gm_combine(int n, int B, const double* __restrict__ Z, size_t zs, int nv,
                                                    const double* __restrict__ y, int add, double* __restrict__ x) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int b = (i % (2 * B)) % B;
        double s = 0.0;
#pragma unroll 4
        for (int v = 0; v < nv; v++) s = fma(Z[(size_t)v * zs + i], y[v * B + b], s);
        x[i] = add ? x[i] + s : s;
    }
}

GmState state_of(mot_handle* h) {
    return GmState{h->d_H, h->d_g, h->d_cs, h->d_sn, h->d_gm_bnorm, h->d_resid, h->d_resid + h->B, h->d_gm_active, h->d_gm_jend, h->gm_m};
}

// Cluster size: about two elements per thread, at most the portable eight CTAs.
int cluster_of(long long elements) {
    int cl = 1;
    while (cl < MAXCL && elements > (long long)cl * GT * 2) cl *= 2;
    return cl;
}

template <class K, class... A>
void launch_cluster(K kernel, int groups, int cl, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(groups * cl);
    cfg.blockDim = dim3(GT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

void set_attributes(mot_handle* h) {
    static std::atomic<unsigned long long> attr{0};
    mot::once_per_device(attr, h->dev, [] {
        const int mx = 200 * 1024;
        cudaFuncSetAttribute(k_gm_iter<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_gm_iter<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_gm_iter<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_gm_iter<4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_gm_back, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    });
}

struct Shape {
    int G, groups, cl;
    bool reg;
};
Shape shape_of(const mot_handle* h) {
    Shape p;
    p.G = h->B == 1 ? 1 : 4;
    p.groups = (h->B + p.G - 1) / p.G;
    const long long el = 2LL * h->npad * p.G;
    p.cl = cluster_of(el);
    p.reg = el <= (long long)p.cl * GT * MAXE;
    return p;
}

}  // namespace

namespace mot {

void launch_gm_begin(mot_handle* h, const double* b, bool first, const double* r, double* V0, cudaStream_t s) {
    const Shape p = shape_of(h);
    auto* k = p.G == 1 ? (p.reg ? k_gm_begin<1, true> : k_gm_begin<1, false>)
                       : (p.reg ? k_gm_begin<4, true> : k_gm_begin<4, false>);
    launch_cluster(k, p.groups, p.cl, sizeof(double) * (NW + 4) * p.G, s, h->npad, h->B, b, first ? 1 : 0, r, V0,
                   state_of(h));
    h->launches++;
}

void launch_gm_iter(mot_handle* h, int j, double* w, double tol, double gain, cudaStream_t s) {
    set_attributes(h);
    const Shape p = shape_of(h);
    const size_t vs = (size_t)h->npad * 2 * h->B;
    const int n = (j + 1) * p.G;
    const size_t smem = sizeof(double) * ((size_t)NW * n + 4 * n + 2 * p.G + 2 * (size_t)j * p.G);
    auto* k = p.G == 1 ? (p.reg ? k_gm_iter<1, true> : k_gm_iter<1, false>)
                       : (p.reg ? k_gm_iter<4, true> : k_gm_iter<4, false>);
    launch_cluster(k, p.groups, p.cl, smem, s, h->npad, h->B, j, (const double*)h->d_V, vs, w,
                   h->d_V + (size_t)(j + 1) * vs, tol, gain, state_of(h));
    h->launches++;
}

void launch_gm_finish(mot_handle* h, const double* Z, int nv, bool add, double* y, double* x, cudaStream_t s) {
    set_attributes(h);
    const long long n = (long long)h->npad * 2 * h->B;
    k_gm_back<<<h->B, 128, sizeof(double) * ((size_t)nv * nv + nv), s>>>(h->B, nv, state_of(h), y);
    const int grid = (int)std::min<long long>((n + 255) / 256, 152 * 16);
    k_gm_combine<<<grid, 256, 0, s>>>((int)n, h->B, Z, (size_t)n, nv, y, add ? 1 : 0, x);
    h->launches += 2;
}

}  // namespace mot
