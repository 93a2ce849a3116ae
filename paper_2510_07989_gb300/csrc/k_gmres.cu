// Batched GMRES of the Q_0 solve (paper Eq. (MOT)): one launch starts a cycle,
// one launch (in long solves eight) orthogonalises a new Krylov vector and updates
// the least-squares problem, one solves it, one combines the basis.
//
// System b of the batch uses columns b and B + b of a block vector
// [npad][2B]. A thread-block cluster owns G systems (4, so that a row's
// columns fill a 32-byte sector; 1 for B = 1) and all rows: every CTA keeps its
// part of the new vector in shared memory, and the dot products are summed over
// the cluster through distributed shared memory, in rank order (every CTA
// gets the same sums). What bounds an iteration is latency: basis vectors from
// L2, two cluster barriers, and chains of FP64 operations of a unit that does
// two multiply-adds per clock and SM (square roots and divisions by one thread
// per system, for the whole cluster).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "mot_internal.h"

namespace {

namespace cg = cooperative_groups;

constexpr int GT = 256;      // threads per CTA
constexpr int NW = GT / 32;
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

// Elements of a group of G systems: index (row * 2 + part) * G + q; local element
// l of cluster rank rk is index ((l / GT) * CL + rk) * GT + l % GT, so a lane's
// elements l = lane + 32 i belong to system lane % G of the group.
template <int G>
struct Part {
    int npad, B, g0, rk, cl;
    __device__ Part(int npad_, int B_, int rk_, int cl_) : npad(npad_), B(B_), rk(rk_), cl(cl_) {
        g0 = (int)(blockIdx.x / cl_) * G;
    }
    __device__ int elements() const { return (2 * npad * G + cl * GT - 1) / (cl * GT) * GT; }
    // offset in a block vector, or -1 outside it
    __device__ int at(int l) const {
        const int idx = (l / GT * cl + rk) * GT + l % GT, rp = idx / G, q = idx % G;
        return rp < 2 * npad && g0 + q < B ? rp * B + g0 + q : -1;
    }
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

// out[i] (i < n: sum i / G of system i % G) = the cluster's sums of what this
// and the other CTAs left in red[0 .. parts)[i]; part is this CTA's own slot,
// read by the others after the cluster barrier.
__device__ __forceinline__ void cluster_sums(int n, int parts, const double* red, double* part, double* out, int cl) {
    __syncthreads();
    double* own = cl == 1 ? out : part;
    for (int i = threadIdx.x; i < n; i += GT) {
        double v[NW];
#pragma unroll
        for (int w = 0; w < NW; w++) v[w] = w < parts ? red[w * n + i] : 0.0;
        own[i] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    if (cl > 1) {
        cg::cluster_group c = cg::this_cluster();
        c.sync();
        for (int i = threadIdx.x; i < n; i += GT) {
            double v[MAXCL];
#pragma unroll
            for (int r = 0; r < MAXCL; r++) v[r] = r < cl ? c.map_shared_rank(part, r)[i] : 0.0;
            out[i] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
    }
    __syncthreads();
}

// Warps that share a group of four sums: all of them for one group, one each
// from NW groups on.
__device__ __forceinline__ int shares(int groups) { return groups >= NW ? 1 : NW / groups; }

// red[share][v * G + q] = the shares' parts of <V_v, w>, v < nv, and with `norm`
// of |w|^2 as one more sum. A warp takes four vectors at a time over its share
// of the elements: sixteen loads in flight a lane. (All warps over the same
// vectors, eight at a time: 46 us an iteration at 1920 edges, B = 1, 17 vectors
// on average.)
template <int G>
__device__ __forceinline__ void dots(const Part<G>& P, int L, const double* V, size_t vs, int nv, bool norm,
                                     const double* ws, double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ns = nv + (norm ? 1 : 0), n = ns * G, ng = (ns + 3) / 4, parts = shares(ng);
    for (int gi = warp; gi < ng * parts; gi += NW) {
        const int v0 = gi % ng * 4, share = gi / ng;
        double p[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int l = share * 32 + lane; l < L; l += parts * 32) {
            // no branch, so that the unrolled loads go out together: past the
            // vector's end x is 0
            const int ix = max(P.at(l), 0);
            const double x = ws[l];
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (v0 + i < ns) p[i] = fma(v0 + i < nv ? V[(size_t)(v0 + i) * vs + ix] : x, x, p[i]);
        }
        const double s = warp_sum4<G>(p);
        const int v = v0 + (((lane >> 4) & 1) << 1 | ((lane >> 3) & 1));
        if ((lane & 7) < G && v < ns) red[share * n + v * G + (lane & 7)] = s;
    }
}

// sum_v V_v[ix] h[v][q]
template <int G>
__device__ __forceinline__ double combine(const double* V, size_t vs, int nv, int ix, const double* h, int q) {
    double s0 = 0.0, s1 = 0.0;
    int v = 0;
#pragma unroll 4
    for (; v + 4 <= nv; v += 4) {
        double a[4];
#pragma unroll
        for (int i = 0; i < 4; i++) a[i] = V[(size_t)(v + i) * vs + ix];
        s0 = fma(a[0], h[v * G + q], s0);
        s1 = fma(a[1], h[(v + 1) * G + q], s1);
        s0 = fma(a[2], h[(v + 2) * G + q], s0);
        s1 = fma(a[3], h[(v + 3) * G + q], s1);
    }
    for (; v < nv; v++) s0 = fma(V[(size_t)v * vs + ix], h[v * G + q], s0);
    return s0 + s1;
}

// Below this squared norm a vector of an O(1) system is a breakdown: its system is done.
constexpr double TINY2 = 1e-300;

// End of iteration j for system sys, whose new column the earlier rotations have
// left at a (and above it in H), with |w| = nrm below: the new rotation, the
// residual, and whether the system is done. gj, ibn, floor_r: g_j, 1 / |b| and the
// residual at which it is done.
__device__ __forceinline__ void new_column(const GmState& S, int sys, int j, double a, double n2, double nrm, double gj,
                                           double ibn, double floor_r) {
    const double d2 = fma(a, a, n2);  // all O(1) or less: b is scaled to O(1)
    double d = 0.0, cc = 1.0, ss = 0.0;
    if (d2 > 0.0) {
        const double id = rsqrt(d2);
        d = d2 * id;
        cc = a * id;
        ss = nrm * id;
    }
    S.cs[(size_t)sys * S.m + j] = cc;
    S.sn[(size_t)sys * S.m + j] = ss;
    S.H[((size_t)sys * (S.m + 1) + j) * S.m + j] = d;
    double* gb = S.g + (size_t)sys * (S.m + 1);
    gb[j + 1] = -ss * gj;
    gb[j] = cc * gj;
    const double rr = fabs(ss * gj) * ibn;
    S.resid[sys] = rr;
    S.jend[sys] = j + 1;
    if (rr <= floor_r || !(nrm > 0.0)) S.active[sys] = 0;
}

// Start of a cycle: beta = |r| per system, V_0 = r / beta. On the first cycle
// also the reference norm |b| (b == r: one vector).
template <int G>
__global__ void __launch_bounds__(GT) k_gm_begin(int npad, int B, const double* __restrict__ b, int first,
                                                 const double* __restrict__ r, double* __restrict__ V0, GmState S) {
    __shared__ double red[NW * 2 * G], part[2 * G], out[2 * G], inv_s[G];
    cg::cluster_group c = cg::this_cluster();
    const int cl = (int)c.num_blocks(), rk = (int)c.block_rank();
    const Part<G> P(npad, B, rk, cl);
    const int L = P.elements(), t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool other = first && b != r;
    double p[4] = {0.0, 0.0, 0.0, 0.0};  // |r|^2, |b|^2
    for (int l = t; l < L; l += GT) {
        const int ix = P.at(l);
        if (ix < 0) continue;
        const double x = r[ix];
        p[0] = fma(x, x, p[0]);
        if (other) {
            const double y = b[ix];
            p[1] = fma(y, y, p[1]);
        }
    }
    const double s = warp_sum4<G>(p);
    if ((lane & 7) < G && lane < 16) red[warp * 2 * G + (lane >> 3) * G + (lane & 7)] = s;
    cluster_sums(2 * G, NW, red, part, out, cl);
    c.barrier_arrive();  // this CTA has read what it needs of the others' shared memory
    if (t < G) {
        const int sys = P.g0 + t;
        const double n2 = out[t], iv = n2 > TINY2 ? rsqrt(n2) : 0.0;
        const double beta = n2 > TINY2 ? n2 * iv : sqrt(n2);
        double bn = 0.0;
        if (sys < B) bn = !first ? S.bnorm[sys] : other ? sqrt(out[G + t]) : beta;
        const bool live = beta > 0.0 && bn > 0.0;
        inv_s[t] = live ? iv : 0.0;
        if (rk == 0 && sys < B) {
            const double rel = bn > 0.0 ? beta / bn : 0.0;
            S.g[(size_t)sys * (S.m + 1)] = beta;
            if (first) S.bnorm[sys] = bn;
            if (first) S.resid0[sys] = rel;
            S.active[sys] = live ? 1 : 0;
            S.jend[sys] = 0;
            S.resid[sys] = rel;
        }
    }
    __syncthreads();
    for (int l = t; l < L; l += GT) {
        const int ix = P.at(l);
        if (ix >= 0) V0[ix] = r[ix] * inv_s[l % G];
    }
    c.barrier_wait();  // ... and they of this one's
}

// Iteration j: w (= Q_0 V_j) orthogonalised against V_0 .. V_j (classical
// Gram-Schmidt twice), V_{j+1} = w / |w|, and the new column of the rotated
// Hessenberg matrix. |w|^2 after the second pass is the sum of squares before
// it less that pass's coefficients (summed with them: two reductions, not
// three), unless it took most of the vector away. A system is done at a residual
// of tol |b|, or of gain times its residual at the start. A system that is done
// writes V_{j+1} = 0 from its next iteration on and keeps its state, so
// iterations past its end change nothing.
template <int G>
__global__ void __launch_bounds__(GT) k_gm_iter(int npad, int B, int j, const double* __restrict__ V, size_t vs,
                                                const double* __restrict__ w, double* __restrict__ Vnext, double tol,
                                                double gain, GmState S) {
    extern __shared__ double sm[];
    __shared__ double inv_s[G], n2_s[G];
    __shared__ int lost_s[G];
    cg::cluster_group c = cg::this_cluster();
    const int cl = (int)c.num_blocks(), rk = (int)c.block_rank();
    const Part<G> P(npad, B, rk, cl);
    const int L = P.elements(), nv = j + 1, n = nv * G, t = threadIdx.x;
    double* red = sm;                // NW (n + G)
    double* part = red + NW * (n + G);  // 2 n + 2 G (one slot per reduction)
    double* h1 = part + 2 * n + 2 * G;  // n
    double* h2 = h1 + n;             // n + G: coefficients, |w|^2
    double* sq = h2 + n + G;         // G
    double* rot = sq + G;            // 2 x j x G: cosines, sines of the earlier rotations
    double* ws = rot + 2 * j * G;    // L: this CTA's part of the new vector
    const int sys = P.g0 + t;        // of threads t < G
    const bool mine = t < G && sys < B;
    // read before the first barrier, written after the last by rank 0
    const bool live = mine && S.active[sys] != 0;
    double gj = 0.0, ibn = 0.0, floor_r = 0.0;
    if (rk == 0) {
        for (int i = t; i < j * G; i += GT) {
            const int b = P.g0 + i % G;
            rot[i] = b < B ? S.cs[(size_t)b * S.m + i / G] : 1.0;
            rot[j * G + i] = b < B ? S.sn[(size_t)b * S.m + i / G] : 0.0;
        }
        if (live) {
            gj = S.g[(size_t)sys * (S.m + 1) + j];
            ibn = 1.0 / S.bnorm[sys];
            floor_r = fmax(tol, gain * S.resid0[sys]);
        }
    }
    for (int l = t; l < L; l += GT) {
        const int ix = P.at(l);
        ws[l] = ix >= 0 ? w[ix] : 0.0;
    }
    __syncthreads();
    dots<G>(P, L, V, vs, nv, false, ws, red);
    cluster_sums(n, shares((nv + 3) / 4), red, part, h1, cl);
    for (int l = t; l < L; l += GT) {
        const int ix = P.at(l);
        if (ix < 0) continue;
        ws[l] -= combine<G>(V, vs, nv, ix, h1, l % G);
    }
    __syncthreads();
    dots<G>(P, L, V, vs, nv, true, ws, red);
    cluster_sums(n + G, shares((nv + 4) / 4), red, part + n, h2, cl);
    if (t < G) {
        double s = h2[n + t], m = s;
        for (int v = 0; v < nv; v++) m -= h2[v * G + t] * h2[v * G + t];
        n2_s[t] = m;
        lost_s[t] = !(m >= 0.5 * s);  // the second pass took most of it away
    }
    __syncthreads();
    bool again = false;
#pragma unroll
    for (int q = 0; q < G; q++) again |= lost_s[q] != 0;
    if (again) {  // the same in every CTA of the cluster: it follows from the sums
        double p[4] = {0.0, 0.0, 0.0, 0.0};
        for (int l = t; l < L; l += GT) {
            const int ix = P.at(l);
            if (ix < 0) continue;
            const double x = ws[l] - combine<G>(V, vs, nv, ix, h2, l % G);
            p[0] = fma(x, x, p[0]);
        }
        const double s = warp_sum4<G>(p);
        if ((t & 31) < G) red[(t >> 5) * G + (t & 31)] = s;
        cluster_sums(G, NW, red, part + 2 * n + G, sq, cl);
        if (t < G) n2_s[t] = sq[t];
    }
    c.barrier_arrive();  // this CTA has read what it needs of the others' shared memory
    if (t < G) inv_s[t] = live && n2_s[t] > TINY2 ? rsqrt(n2_s[t]) : 0.0;
    __syncthreads();
    for (int l = t; l < L; l += GT) {
        const int ix = P.at(l);
        if (ix < 0) continue;
        const double iv = inv_s[l % G];
        const double x = ws[l] - combine<G>(V, vs, nv, ix, h2, l % G);
        Vnext[ix] = iv != 0.0 ? x * iv : 0.0;
    }
    if (rk == 0 && live) {
        double* Hb = S.H + (size_t)sys * (S.m + 1) * S.m;
        double a = h1[t] + h2[t];
        for (int i = 0; i < j; i++) {
            const double x = h1[(i + 1) * G + t] + h2[(i + 1) * G + t];
            const double cc = rot[i * G + t], ss = rot[(j + i) * G + t];
            Hb[(size_t)i * S.m + j] = cc * a + ss * x;
            a = -ss * a + cc * x;
        }
        const double n2 = fmax(n2_s[t], 0.0);
        new_column(S, sys, j, a, n2, n2 > TINY2 ? n2 * inv_s[t] : sqrt(n2), gj, ibn, floor_r);
    }
    c.barrier_wait();  // ... and they of this one's
}

// The same iteration in launches over the whole chip, for long ones (launch_gm_iter).
// partial[chunk][v * B + b] = the chunk of rows' part of <V_v, w>_b, v < nv: four
// vectors a CTA, its threads (row of a stride, system).
constexpr int DT = 256;
__global__ void __launch_bounds__(DT) k_gm_dots(int npad, int B, int rows, const double* __restrict__ V, size_t vs,
                                                int nv, const double* __restrict__ w, double* __restrict__ partial) {
    __shared__ double red[4][DT];
    const int t = threadIdx.x, RS = DT / B, rs = t / B, b = t - rs * B, v0 = blockIdx.y * 4, nl = min(4, nv - v0);
    const int r1 = min(npad, (int)(blockIdx.x + 1) * rows);
    double p[4] = {0.0, 0.0, 0.0, 0.0};
    if (rs < RS)
#pragma unroll 4
        for (int r = blockIdx.x * rows + rs; r < r1; r += RS) {
            const size_t ix = (size_t)r * 2 * B + b;
            const double x = w[ix], y = w[ix + B];
#pragma unroll
            for (int i = 0; i < 4; i++) {  // past the last vector its values again, not used
                const double* v = V + (size_t)(v0 + min(i, nl - 1)) * vs + ix;
                p[i] = fma(v[B], y, fma(v[0], x, p[i]));
            }
        }
#pragma unroll
    for (int i = 0; i < 4; i++) red[i][t] = p[i];
    for (int m = RS; m > 1;) {  // the upper half of the row strides onto the lower
        const int half = (m + 1) / 2;
        __syncthreads();
        if (rs < m - half)
#pragma unroll
            for (int i = 0; i < 4; i++) red[i][t] += red[i][t + half * B];
        m = half;
    }
    __syncthreads();
    for (int i = t; i < nl * B; i += DT)
        partial[(size_t)blockIdx.x * nv * B + v0 * B + i] = red[i / B][i % B];
}

// h[i] = the chunks' partials of sum i, in order
__global__ void __launch_bounds__(128) k_gm_dots_sum(int n, int chunks, const double* __restrict__ partial,
                                                     double* __restrict__ h) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < chunks; c++) s += partial[(size_t)c * n + i];
    h[i] = s;
}

// w -= sum_v V_v h[v][b]
__global__ void __launch_bounds__(128) k_gm_update(int n, int B, const double* __restrict__ V, size_t vs, int nv,
                                                   const double* __restrict__ h, double* __restrict__ w) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    const int b = i % B;
    double s0 = 0.0, s1 = 0.0;
    int v = 0;
#pragma unroll 4
    for (; v + 2 <= nv; v += 2) {
        s0 = fma(V[(size_t)v * vs + i], h[v * B + b], s0);
        s1 = fma(V[(size_t)(v + 1) * vs + i], h[(v + 1) * B + b], s1);
    }
    if (v < nv) s0 = fma(V[(size_t)v * vs + i], h[v * B + b], s0);
    w[i] -= s0 + s1;
}

// |w| of system blockIdx.x, its new column (coefficients h1 + h2) and the factor
// that makes V_{j+1} of w: 0 for a system that is done
__global__ void __launch_bounds__(DT) k_gm_column(int npad, int B, int j, const double* __restrict__ w,
                                                  const double* __restrict__ h1, const double* __restrict__ h2,
                                                  double tol, double gain, GmState S, double* __restrict__ inv) {
    extern __shared__ double sm[];
    double *h = sm, *cs = h + j + 1, *sn = cs + j;  // j + 1, j, j
    __shared__ double red[DT / 32];
    const int b = blockIdx.x, t = threadIdx.x;
    for (int i = t; i <= j; i += DT) h[i] = h1[i * B + b] + h2[i * B + b];
    for (int i = t; i < j; i += DT) {
        cs[i] = S.cs[(size_t)b * S.m + i];
        sn[i] = S.sn[(size_t)b * S.m + i];
    }
    double s = 0.0;
#pragma unroll 8
    for (int r = t; r < 2 * npad; r += DT) {
        const double x = w[(size_t)r * B + b];
        s = fma(x, x, s);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((t & 31) == 0) red[t >> 5] = s;
    __syncthreads();
    if (t > 0) return;
    double n2 = 0.0;
    for (int i = 0; i < DT / 32; i++) n2 += red[i];
    const bool live = S.active[b] != 0;
    const double iv = live && n2 > TINY2 ? rsqrt(n2) : 0.0;
    inv[b] = iv;
    if (!live) return;
    double* Hb = S.H + (size_t)b * (S.m + 1) * S.m;
    double a = h[0];
    for (int i = 0; i < j; i++) {
        const double x = h[i + 1], cc = cs[i], ss = sn[i];
        Hb[(size_t)i * S.m + j] = cc * a + ss * x;
        a = -ss * a + cc * x;
    }
    new_column(S, b, j, a, n2, n2 > TINY2 ? n2 * iv : sqrt(n2), S.g[(size_t)b * (S.m + 1) + j], 1.0 / S.bnorm[b],
               fmax(tol, gain * S.resid0[b]));
}

__global__ void __launch_bounds__(128) k_gm_scale(int n, int B, const double* __restrict__ w,
                                                  const double* __restrict__ inv, double* __restrict__ Vnext) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    const double iv = inv[i % B];
    Vnext[i] = iv != 0.0 ? w[i] * iv : 0.0;
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
        cudaFuncSetAttribute(k_gm_iter<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_gm_iter<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_gm_back, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    });
}

struct Shape {
    int G, groups, cl;
    long long per_cta;  // elements
};
// Cluster size: at most the portable eight CTAs, about 512 elements each, two a
// thread: a cluster barrier costs less than a longer pass over the elements (at
// 2048 an iteration of the first two takes 19.2 us for 14.0 at 216 edges, 8 waves,
// 24.3 for 19.6 at 924 edges, 64 waves; the start of a cycle 5.4 for 4.7).
Shape shape_of(const mot_handle* h) {
    constexpr int per = 512;
    Shape p;
    p.G = h->B == 1 ? 1 : 4;
    p.groups = (h->B + p.G - 1) / p.G;
    const long long el = 2LL * h->npad * p.G;
    p.cl = 1;
    while (p.cl < MAXCL && el > (long long)p.cl * per) p.cl *= 2;
    p.per_cta = (el + p.cl * GT - 1) / (p.cl * GT) * GT;
    return p;
}

}  // namespace

namespace mot {

// An iteration is one cluster launch below LONG elements times vectors a CTA, and
// the eight launches of long_iter from there on: a cluster's groups of four systems
// run on eight SMs each (16 SMs for 8 waves), whose FP64 units and load latency
// grow with elements times vectors (1296 edges, 8 waves: 124 us at 30 vectors),
// where eight launches over the whole chip stay near their 30 us. A step with 38
// to 40 iterations without preconditioner (mixed, 2 / 8 / 64 waves): 1296 edges
// 9.3 / 8.3 / 11.5 ms, in cluster launches only 12.6 / 11.7 / 15.0; 2160 edges 16.5 /
// 12.4 / 17.5 and 24.9 / 20.4 / 25.9. At 8192 the solves of 120 and 270 edges
// (22 to 50 iterations) took 3 to 11 % longer, at 16384 they take as long.
constexpr long long LONG = 16384;

static void long_iter(mot_handle* h, int j, double* w, double tol, double gain, double* work, size_t work_size,
                      cudaStream_t s) {
    const int B = h->B, nv = j + 1, n = nv * B, el = h->npad * 2 * B, groups = (nv + 3) / 4;
    const size_t vs = (size_t)el;
    int nsm = 148;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->dev);
    // chunks of whole row strides, about four CTAs an SM in all, at most 64 to be summed
    const int RS = DT / B, strides = (h->npad + RS - 1) / RS;
    const size_t room = work_size - 2 * (size_t)n - B;
    int chunks = std::max(1, std::min({4 * nsm / groups, 64, strides, (int)(room / n)}));
    const int rows = (strides + chunks - 1) / chunks * RS;
    chunks = (h->npad + rows - 1) / rows;
    double *h1 = work, *h2 = h1 + n, *inv = h2 + n, *partial = inv + B;
    for (double* hh : {h1, h2}) {
        k_gm_dots<<<dim3(chunks, groups), DT, 0, s>>>(h->npad, B, rows, h->d_V, vs, nv, w, partial);
        k_gm_dots_sum<<<(n + 127) / 128, 128, 0, s>>>(n, chunks, partial, hh);
        k_gm_update<<<(el + 127) / 128, 128, 0, s>>>(el, B, h->d_V, vs, nv, hh, w);
    }
    k_gm_column<<<B, DT, sizeof(double) * (3 * (size_t)j + 1), s>>>(h->npad, B, j, w, h1, h2, tol, gain, state_of(h),
                                                                    inv);
    k_gm_scale<<<(el + 127) / 128, 128, 0, s>>>(el, B, w, inv, h->d_V + (size_t)(j + 1) * vs);
    h->launches += 8;
}

void launch_gm_begin(mot_handle* h, const double* b, bool first, const double* r, double* V0, cudaStream_t s) {
    const Shape p = shape_of(h);
    launch_cluster(p.G == 1 ? k_gm_begin<1> : k_gm_begin<4>, p.groups, p.cl, 0, s, h->npad, h->B, b, first ? 1 : 0, r,
                   V0, state_of(h));
    h->launches++;
}

void launch_gm_iter(mot_handle* h, int j, double* w, double tol, double gain, double* work, size_t work_size,
                    cudaStream_t s) {
    set_attributes(h);
    const Shape p = shape_of(h);
    if (p.per_cta * (j + 1) >= LONG) {
        long_iter(h, j, w, tol, gain, work, work_size, s);
        return;
    }
    const size_t vs = (size_t)h->npad * 2 * h->B;
    const int n = (j + 1) * p.G;
    const size_t smem = sizeof(double) * ((size_t)NW * (n + p.G) + 4 * n + 4 * p.G + 2 * (size_t)j * p.G +
                                          (size_t)p.per_cta);  // LONG elements at most: 128 KB, 27 KB of the rest
    launch_cluster(p.G == 1 ? k_gm_iter<1> : k_gm_iter<4>, p.groups, p.cl, smem, s, h->npad, h->B, j, (const double*)h->d_V, vs, (const double*)w,
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
