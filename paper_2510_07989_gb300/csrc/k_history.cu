// Block-sparse history contraction of the MOT step (paper Eq. (MOT)):
//   s1 = sum_k A_k l_{i-k} + A^_k s_{i-k},   s2 = sum_k A~_k l_{i-k} + A_k s_{i-k}
// where each family is the 2x2 PMCHWT block of Section V-B built from stored
// T, T', K + K' matrices. The medium factors (eta, eta') and the block signs of
// the 2x2 structure are folded into three precomputed variants of every
// coefficient panel, so every stored tile is a plain (TILE x TILE) * (TILE x 2B)
// product accumulated into one of two outputs.
//
// FP64 path: one CTA per chunk of tile tasks of a single row block; partial sums
// go to a scratch buffer and a second kernel reduces the chunks of each row
// block in a fixed order (deterministic).
#include "mot_internal.h"

namespace {

constexpr int T = MOT_TILE;
constexpr int NT = 256;                       // threads per CTA
constexpr int MAXO = T * 2 * MOT_MAX_B / NT;  // outputs per thread per target (16)

__device__ __forceinline__ const double* panel_ptr(int mode, const double* ring, const double* win,
                                                   const double* kry, long long step_i, int R, int npad,
                                                   int C2, int k, int part, int variant) {
    const size_t pstride = (size_t)npad * C2;
    if (mode == 1) return kry + ((size_t)part * 3 + variant) * pstride;
    if (part == 2) return win + (size_t)k * pstride;
    long long src = step_i - k;
    int slot = (int)(src % R);
    return ring + (((size_t)slot * 2 + part) * 3 + variant) * pstride;
}

// Bound by the FP64 units (two multiply-adds per clock and SM): at B = 64 a
// task is 131 072 of them when every entry of its tile is multiplied, against
// 40 KB of loads. Only about 30 % of a tile's entries are nonzero, so each
// tile row carries a mask of its nonzeros (built at load) and a warp multiplies
// those: the lanes of a warp are columns of one row (2B a multiple of 32) and
// walk its mask together; in other batches they walk the union of their rows'
// masks. One full-depth launch at 432 edges, 53 lags, B = 64: 20.5 ms with
// every entry multiplied, 8.7 ms with the masks.
__global__ void __launch_bounds__(NT) k_hist_f64(const HistTask* __restrict__ tasks,
                                                 const HistChunk* __restrict__ chunks,
                                                 const double* __restrict__ tiles,
                                                 const uint32_t* __restrict__ masks, const double* __restrict__ ring,
                                                 const double* __restrict__ win, const double* __restrict__ kry,
                                                 int mode, long long step_i, int R, int npad, int C2,
                                                 const int* __restrict__ colidx, double* __restrict__ partial) {
    extern __shared__ double sm[];
    __shared__ uint32_t smask[T];
    double* st = sm;                  // T x (T + 1)
    double* sp = st + T * (T + 1);    // T x C2
    const HistChunk ch = chunks[blockIdx.x];
    const int nout = T * C2;
    const int tid = threadIdx.x;
    double acc0[MAXO], acc1[MAXO];
#pragma unroll
    for (int j = 0; j < MAXO; j++) {
        acc0[j] = 0.0;
        acc1[j] = 0.0;
    }
    auto product = [&](double (&acc)[MAXO]) {
#pragma unroll
        for (int j = 0; j < MAXO; j++) {
            const int o = tid + j * NT;
            if (tid - (tid & 31) + j * NT >= nout) break;  // the whole warp is past the outputs
            const int r = o < nout ? o / C2 : T - 1, c = o < nout ? o - r * C2 : 0;
            const double* sr = st + r * (T + 1);
            double s = acc[j];
            uint32_t m = __reduce_or_sync(0xffffffffu, o < nout ? smask[r] : 0u);
            while (m) {  // two nonzeros at a time: their loads overlap
                const int n0 = __ffs(m) - 1;
                m &= m - 1;
                const bool two = m != 0;
                const int n1 = two ? __ffs(m) - 1 : n0;
                m &= m - 1;
                const double a0 = sr[n0], x0 = sp[n0 * C2 + c], a1 = sr[n1], x1 = sp[n1 * C2 + c];
                s = fma(a0, x0, s);
                if (two) s = fma(a1, x1, s);
            }
            acc[j] = s;
        }
    };
    for (int t = ch.first; t < ch.first + ch.count; t++) {
        const HistTask tk = tasks[t];
        const int part = tk.code & 3, variant = (tk.code >> 2) & 3, out = (tk.code >> 4) & 1;
        if (mode == 0 && step_i - tk.k < 1) continue;  // history before step 1 is zero
        const double* pan = panel_ptr(mode, ring, win, kry, step_i, R, npad, C2, tk.k, part, variant);
        const int* cols = colidx + (size_t)ch.rb * npad + (size_t)tk.cb * T;  // distance-sorted columns
        const double* tl = tiles + (size_t)tk.tile * T * T;
        __syncthreads();
        if (tid < T) smask[tid] = masks[(size_t)tk.tile * T + tid];
        for (int e = tid; e < T * T; e += NT) st[(e / T) * (T + 1) + (e % T)] = tl[e];
        for (int e = tid; e < T * C2; e += NT) {
            const int r = e / C2;
            sp[e] = pan[(size_t)cols[r] * C2 + (e - r * C2)];
        }
        __syncthreads();
        if (out == 0)
            product(acc0);
        else
            product(acc1);
    }
    double* dst = partial + (size_t)blockIdx.x * 2 * nout;
#pragma unroll
    for (int j = 0; j < MAXO; j++) {
        const int o = tid + j * NT;
        if (o < nout) {
            dst[o] = acc0[j];
            dst[nout + o] = acc1[j];
        }
    }
}

// B <= 4 (C2 = 2, 4, 6 or 8 columns): a warp takes eight rows of a tile, its
// lanes the 32 tile columns, and every lane keeps its products' sums over all
// tasks of the chunk in registers -- the lanes are summed once per output and
// chunk, not per tile, and nothing is staged: a tile row is one coalesced
// 256-byte load, a lane gathers its own coefficient row, and the next task's
// loads are in flight during this one's products. Bound by the FP64 units
// (2B multiply-adds per tile entry) with the tile stream close behind. Four
// warps cover a tile; the CTA's other four take every second task.
template <int C2>
__global__ void __launch_bounds__(NT) k_hist_f64_small(const HistTask* __restrict__ tasks,
                                                       const HistChunk* __restrict__ chunks,
                                                       const double* __restrict__ tiles,
                                                       const double* __restrict__ ring, const double* __restrict__ win,
                                                       const double* __restrict__ kry, int mode, long long step_i,
                                                       int R, int npad, const int* __restrict__ colidx,
                                                       double* __restrict__ partial) {
    constexpr int RW = 8, NV = RW * C2;  // rows per warp, sums per lane
    __shared__ double sums[2][2][T * C2];  // [task stream][target][row][column]
    const HistChunk ch = chunks[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row0 = (warp & 3) * RW, half = warp >> 2;
    for (int i = threadIdx.x; i < 4 * T * C2; i += NT) (&sums[0][0][0])[i] = 0.0;
    __syncthreads();
    double acc[RW][C2];
#pragma unroll
    for (int r = 0; r < RW; r++)
#pragma unroll
        for (int c = 0; c < C2; c++) acc[r][c] = 0.0;
    // sums of the lanes into this warp's rows of target `out`
    auto flush = [&](int out) {
#pragma unroll
        for (int r = 0; r < RW; r++)
#pragma unroll
            for (int c = 0; c < C2; c++) {
                double v = acc[r][c];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (lane == 0) sums[half][out][(row0 + r) * C2 + c] += v;
                acc[r][c] = 0.0;
            }
    };
    const int* cols = colidx + (size_t)ch.rb * npad;
    const int end = ch.first + ch.count;
    auto live = [&](int t) {  // the next task of this stream that takes part
        while (t < end && mode == 0 && step_i - tasks[t].k < 1) t += 2;
        return t;
    };
    double a[RW], x[C2];
    int out = 0;
    auto fetch = [&](int t) {
        const HistTask tk = tasks[t];
        out = (tk.code >> 4) & 1;
        const double* pan = panel_ptr(mode, ring, win, kry, step_i, R, npad, C2, tk.k, tk.code & 3, (tk.code >> 2) & 3) +
                            (size_t)cols[tk.cb * T + lane] * C2;
        const double* tl = tiles + (size_t)tk.tile * T * T + row0 * T + lane;
#pragma unroll
        for (int r = 0; r < RW; r++) a[r] = tl[r * T];
#pragma unroll
        for (int c = 0; c < C2; c++) x[c] = pan[c];
    };
    int t = live(ch.first + half), cur = -1;
    if (t < end) fetch(t);
    while (t < end) {
        if (cur >= 0 && out != cur) flush(cur);
        cur = out;
        double ca[RW], cx[C2];
#pragma unroll
        for (int r = 0; r < RW; r++) ca[r] = a[r];
#pragma unroll
        for (int c = 0; c < C2; c++) cx[c] = x[c];
        t = live(t + 2);
        if (t < end) fetch(t);
#pragma unroll
        for (int r = 0; r < RW; r++)
#pragma unroll
            for (int c = 0; c < C2; c++) acc[r][c] = fma(ca[r], cx[c], acc[r][c]);
    }
    if (cur >= 0) flush(cur);
    __syncthreads();
    double* dst = partial + (size_t)blockIdx.x * 2 * T * C2;
    for (int i = threadIdx.x; i < 2 * T * C2; i += NT) dst[i] = (&sums[0][0][0])[i] + (&sums[1][0][0])[i];
}

// masks[tile][r]: bit n set where entry (r, n) of the tile is nonzero; one warp per row
__global__ void k_tile_masks(long long rows, const double* __restrict__ tiles, uint32_t* __restrict__ masks) {
    const int lane = threadIdx.x & 31;
    for (long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; r < rows;
         r += ((long long)gridDim.x * blockDim.x) >> 5) {
        const uint32_t m = __ballot_sync(0xffffffffu, tiles[r * T + lane] != 0.0);
        if (lane == 0) masks[r] = m;
    }
}

// out_s[rb*T + r][c] = sum over the chunks of row block rb of partial[chunk][target][r][c],
// in order; with rho, rho - that sum. One thread per output: with one CTA per row block (a few dozen) the
// chunk loop ran at a fraction of the memory rate (321 us at 432 edges, B = 64).
__global__ void __launch_bounds__(256) k_hist_reduce(const int* __restrict__ chunk_ptr,
                                                     const double* __restrict__ partial, int C2,
                                                     const double* __restrict__ rho1, const double* __restrict__ rho2,
                                                     double* __restrict__ s1, double* __restrict__ s2) {
    const int rb = blockIdx.y;
    const int nout = T * C2;
    const int o = blockIdx.x * 256 + threadIdx.x;  // over both targets
    if (o >= 2 * nout) return;
    const int c1 = chunk_ptr[rb + 1];
    double a = 0.0;
#pragma unroll 4
    for (int c = chunk_ptr[rb]; c < c1; c++) a += partial[(size_t)c * 2 * nout + o];
    const size_t ix = (size_t)rb * nout + (o < nout ? o : o - nout);
    if (rho1) a = (o < nout ? rho1 : rho2)[ix] - a;
    (o < nout ? s1 : s2)[ix] = a;
}

}  // namespace

namespace mot {

void launch_history(mot_handle* h, const TaskList& tl, const double* tiles, const double* ring, const double* win,
                    const double* kry, int mode, long long step_i, const double* rho1, const double* rho2,
                    double* out_s1, double* out_s2, cudaStream_t s) {
    const int C2 = 2 * h->B;
    if (tl.nchunks > 0) {
        size_t smem = sizeof(double) * (T * (T + 1) + T * C2);
        const bool timed = h->opt.timing && mode == 0 && h->ev0 && step_i > h->K;
        if (timed) cudaEventRecord(h->ev0, s);
#define MOT_HIST_SMALL(CV)                                                                                       \
    k_hist_f64_small<CV><<<tl.nchunks, NT, 0, s>>>(tl.tasks, tl.chunks, tiles, ring, win, kry, mode, step_i, h->R, \
                                                   h->npad, h->d_colidx, h->d_partial)
        switch (C2) {
            case 2: MOT_HIST_SMALL(2); break;
            case 4: MOT_HIST_SMALL(4); break;
            case 6: MOT_HIST_SMALL(6); break;
            case 8: MOT_HIST_SMALL(8); break;
            default:
                k_hist_f64<<<tl.nchunks, NT, smem, s>>>(tl.tasks, tl.chunks, tiles, h->d_tmask, ring, win, kry, mode,
                                                        step_i, h->R, h->npad, C2, h->d_colidx, h->d_partial);
        }
#undef MOT_HIST_SMALL
        if (timed) {
            cudaEventRecord(h->ev1, s);
            h->ev_pending = true;
        }
        h->launches++;
    }
    launch_history_reduce(h, tl, C2, rho1, rho2, out_s1, out_s2, s);
}

void launch_history_reduce(mot_handle* h, const TaskList& tl, int C2, const double* rho1, const double* rho2,
                           double* out_s1, double* out_s2, cudaStream_t s) {
    const dim3 grid((2 * T * C2 + 255) / 256, h->nrb);
    k_hist_reduce<<<grid, 256, 0, s>>>(tl.chunk_ptr, h->d_partial, C2, rho1, rho2, out_s1, out_s2);
    h->launches++;
}

void launch_tile_masks(mot_handle* h, int64_t ntiles, const double* tiles, uint32_t* masks, cudaStream_t s) {
    const long long rows = (long long)ntiles * T;
    if (rows == 0) return;
    const int blocks = (int)((rows * 32 + 255) / 256 < 152 * 64 ? (rows * 32 + 255) / 256 : 152 * 64);
    k_tile_masks<<<blocks, 256, 0, s>>>(rows, tiles, masks);
    h->launches++;
}

}  // namespace mot
