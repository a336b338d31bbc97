// lv_mc.cuh -- the Monte Carlo price / pathwise-adjoint kernels (arXiv
// 2002.02481, Sec. III, IV-A..IV-D), templated on the model (the reading of
// the scheme and of the interpolation, see lv_device.cuh). Every translation
// unit that includes this header instantiates its own kernels with internal
// linkage: lv_m<model>c<cell>.cu one model and one way to find the spot cell.
//
// Adjoint kernel: persistent, warp-centric, no block-wide barrier in its
// main loop. Every warp repeatedly either
//   (F) claims a tile of 32 consecutive paths from a global counter and runs
//       their forward passes: normals generated in registers, log-Euler
//       steps under the bilinear grid staged in shared memory, x stored every
//       KCK steps (the checkpoints) into one of kRing groups of 32 slots
//       owned by the warp; payoff and terminal adjoint
//       xbar_N = e^{-rT} 1{phi(S_N - K) > 0} phi S_N; the paths with a
//       nonzero xbar_N (all others have a zero adjoint everywhere) are
//       appended to a per-warp FIFO in shared memory; or
//   (R) takes up to 32 queued paths and runs their reverse sweeps: per
//       checkpoint segment, last to first, recompute KCK steps from the
//       checkpoint with the same Philox counters keeping h_n = d x_{n+1} /
//       d sigma_n, g_n = h_n S_n d sigma / d S, the cell and the weight in
//       registers, then walk back: sigma_bar_n = xbar_{n+1} h_n,
//       xbar_n = xbar_{n+1} (1 + g_n), sigma_bar_n spread over the four
//       corner buckets with the bilinear weights.
// A reverse batch runs when 32 paths are queued, when the oldest queued
// path's checkpoint slots are about to be reused by the next forward tile,
// and at the end; so the reverse sweeps run on full warps. With two paths
// per lane (PPL = 2) a warp claims two consecutive tiles and advances each
// lane's two paths together, their binary32 arithmetic in packed .f32x2
// pairs (forward_path2); the slot groups and the FIFO double, the reverse
// batches stay at 32 paths.
//
// Bucket accumulation: run-length sums in registers while the cell is
// unchanged (level 0); binary32 reductions (one 16-byte red per cell, resolved in
// L2 without a retry loop) into an array of the cells' corner sums in global
// memory, one for every four warps of a block (level 1); every few batches a warp
// drains its array into level 2: the block's binary64 row, one warp at a time under a lock, or in Kahan
// mode a compensated binary32 row the warp owns; at the end each block adds
// what it holds to the call's binary64 sums, and the last block to arrive writes
// the outputs (level 3).
//
// The DBG instantiation additionally writes per-path results and logs
// every forward step whose spot lies within a relative band of its cell's
// nodes, with the cell and inside-grid decision taken there, so that a
// test can hand the same decisions to the binary64 oracle.
#pragma once

#include <math.h>

#include "lv_device.cuh"

namespace lv {

namespace {

constexpr int kTile = 32;      // paths per warp tile (one per lane); the forward-only kernel's hold 32 PPL
constexpr int kRing = 4;       // checkpoint slot groups of kTile per warp

constexpr int kQueue = 64;     // per-warp FIFO capacity per path a lane runs in a forward tile
                               // (entries; < 32 + kTile * ppl never overflows kQueue * ppl)

__host__ __device__ inline size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

constexpr int kStagedTau = 256;   // time nodes (and inverse gaps) staged in shared memory for the time table

// Level-2 accumulator of one value: binary64 or Kahan-compensated binary32.
// The slots live in shared memory (one per thread and value), which keeps
// them out of the registers the reverse sweep needs.
struct AccSlot {
    double d;
    float s, c;
};

struct SmemLayout {
    size_t tab, sig, node, ab, bins, tau, tdt, qslot, qrel, qxb, acc, flag, total;
};

// extra: the adjoint kernel that also sums d V / d r and d V / d T (the time
// slope table and two more accumulators per thread); ppl: paths per lane of
// the adjoint's forward tiles (the FIFO grows with it).
__host__ __device__ inline SmemLayout smem_layout(int I, int J, int N, int n_bins, int block, bool greeks,
                                                  bool grid_smem, bool extra = false, int ppl = 1)
{
    const int W = block / 32, Je = J > 1 ? J : 2;
    SmemLayout L;
    size_t o = 0;
    L.tab = o;   o += align16(sizeof(int4) * (size_t)N);
    L.sig = o;   if (grid_smem) o += align16(sizeof(float2) * (size_t)Je * (I - 1));
    L.node = o;  o += align16(sizeof(float) * (size_t)I);
    L.ab = o;    o += align16(sizeof(float2) * (size_t)I);
    L.bins = o;  o += sizeof(float4) * (size_t)n_bins;
    L.tau = o;   if (J <= kStagedTau) o += align16(2 * sizeof(double) * (size_t)J);
    L.tdt = o;   if (extra) o += align16(sizeof(float) * (size_t)N);
    // the adjoint kernel slices these three per warp from L.qslot: they stay
    // contiguous because each size is a multiple of 16 bytes (kQueue is)
    static_assert(kQueue % 4 == 0, "FIFO arrays must stay contiguous");
    L.qslot = o; if (greeks) o += align16(sizeof(int) * (size_t)W * kQueue * ppl);
    L.qrel = o;  if (greeks) o += align16(sizeof(int) * (size_t)W * kQueue * ppl);
    L.qxb = o;   if (greeks) o += align16(sizeof(float) * (size_t)W * kQueue * ppl);
    L.acc = o;   o += align16(sizeof(AccSlot) * (extra ? 5 : 3) * (size_t)block);
    L.flag = o;  o += 16;
    L.total = o;
    return L;
}

// Adds x to a level-2 slot.
template <int ACC>
__device__ __forceinline__ void acc_add(AccSlot& a, float x)
{
    if (ACC == 1) {
        const float y = x - a.c;
        const float t = a.s + y;
        a.c = (t - a.s) - y;
        a.s = t;
    } else {
        a.d += (double)x;
    }
}

template <int ACC>
__device__ __forceinline__ double acc_value(const AccSlot& a)
{
    return ACC == 1 ? (double)a.s - (double)a.c : a.d;
}

// Asynchronous copy of n elements of SIZE bytes (4, 8 or 16) to shared memory.
template <int SIZE>
__device__ __forceinline__ void copy_async(void* dst, const void* src, int n)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    for (int e = threadIdx.x; e < n; e += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d + SIZE * e),
                     "l"(__cvta_generic_to_global(static_cast<const char*>(src) + (size_t)SIZE * e)), "n"(SIZE)
                     : "memory");
}

// Stages the time table, the spot nodes, the cell coefficients and (when GS)
// the sigma pairs in shared memory; large grids are read from global memory
// through L1 instead, which leaves room for more resident blocks. `clear` runs
// while the copies are in flight: every element is on its way before the first
// is waited for, and the time table's searches read the time nodes from
// shared memory (loads of one thread in turn and searches in global memory took
// 5.4 us at the start of every launch on the 30 x 60 grid with 156 steps).
template <bool GS, bool EXTRA = false, typename F>
__device__ __forceinline__ void stage_grid(const McParams& P, unsigned char* smem, const SmemLayout& L, F&& clear)
{
    const int B = blockDim.x, tid = threadIdx.x;
    int4* s_tab = reinterpret_cast<int4*>(smem + L.tab);
    const double* tau = P.tau;
    const double* rtau = P.tau + P.J;
    if (P.J <= kStagedTau) {
        copy_async<8>(smem + L.tau, P.tau, 2 * P.J);
        tau = reinterpret_cast<const double*>(smem + L.tau);
        rtau = tau + P.J;
    }
    if (GS) copy_async<8>(smem + L.sig, P.sig2, P.Je * (P.I - 1));
    copy_async<4>(smem + L.node, P.node, P.I);
    copy_async<8>(smem + L.ab, P.ab, P.I - 1);
    copy_async<16>(smem + L.bins, P.bins, P.n_bins);
    clear();
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int n = tid; n < P.N; n += B) s_tab[n] = step_time(P, tau, rtau, n);
    if (EXTRA) {
        float* s_tdt = reinterpret_cast<float*>(smem + L.tdt);
        for (int n = tid; n < P.N; n += B) s_tdt[n] = step_tdt(P, tau, n);
    }
    __syncthreads();
}

// The lower node (j I + i) of the cell the paths start in, for the launches whose lanes
// have buckets of their own for it (OWN).
template <bool OWN, int MODEL, int CELL>
__device__ __forceinline__ int start_node(const McParams& P, const SmemGrid& g)
{
    if (!OWN) return 0;
    return g.tab[0].y + start_cell<MODEL, CELL>(P, g) - g.tab[0].x;
}

// The level-1 buckets of a warp. A block has one array for every kBucketWarps of its
// warps, dealt out in turn, so that the warps of one array drain at different times
// (first_drain). With one array for all sixteen warps of a 512-thread block, a
// bucket held four times the paths in binary32 that a 128-thread block's does, and its
// rounding grew with them (relative 2-norm against binary64 sums of the same
// flushes, 104 steps: vegas on 5 x 2 nodes, 2^17 paths 3.9e-8, with four arrays
// 1.2e-8, in 128-thread blocks of node buckets 1.5e-8; second-order buckets on 20 x 10
// nodes 1.1e-7, 4.4e-8 and 7.6e-8). The four arrays' clears and folds take 3-7 us a
// call on 30 x 60 nodes: 2^18 paths 177 -> 183 us, 2^20 509 -> 517, 2^22 1,827 -> 1,842;
// 100 x 100 nodes, 1,260 steps, 2^22 paths 15.38 -> 15.53 ms.
__device__ __forceinline__ float4* warp_buckets(const McParams& P, int warp, int W)
{
    const int G = bucket_arrays(W);
    return P.l1 + (size_t)(blockIdx.x * G + warp % G) * bucket_count(P.I, P.Je);
}

// The level-2 row of the warp: binary64 mode drains into the block's own row
// with binary64 reductions; Kahan pairs cannot be updated atomically, so each
// warp owns one.
template <int ACC>
__device__ __forceinline__ double* level2_row(const McParams& P)
{
    if (ACC == 1)
        return P.warp_rows + (size_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (P.Je * P.I);
    return P.partials + (size_t)blockIdx.x * P.row_words + 3;
}

// Zeroes the block's level-1 buckets and level-2 rows, and the flag that some
// warp drained.
template <int ACC>
__device__ __forceinline__ void clear_buckets(const McParams& P, int* drained)
{
    const int nIJ = P.Je * P.I, B = blockDim.x, W = B >> 5, tid = threadIdx.x;
    const int nc = bucket_arrays(W) * bucket_count(P.I, P.Je);
    float4* l1 = P.l1 + (size_t)blockIdx.x * nc;
    for (int e = tid; e < nc; e += B) l1[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (ACC == 1) {
        double* rows = P.warp_rows + (size_t)blockIdx.x * W * nIJ;
        for (int e = tid; e < W * nIJ; e += B) rows[e] = 0.0;     // zero as a float2 pair too
    } else {
        double* row = P.partials + (size_t)blockIdx.x * P.row_words + 3;
        for (int e = tid; e < nIJ; e += B) row[e] = 0.0;
    }
    if (tid == 0) drained[0] = drained[1] = 0;      // the flag and the drains' lock
}

// Adds the block's sums of the first `n` accumulators (slot k of thread t at
// acc0[k B + t]) to sums[0 .. n-1], one warp per accumulator, after a barrier.
template <int ACC>
__device__ __forceinline__ void add_scalars(const AccSlot* acc0, int n, double* sums)
{
    const int B = blockDim.x, W = B >> 5, lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < n; k += W) {
        double a = acc_value<ACC>(acc0[k * B + lane]);
        for (int w = 1; w < W; ++w) a += acc_value<ACC>(acc0[k * B + 32 * w + lane]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if (lane == 0) atomicAdd(&sums[k], a);
    }
}

// The warp's sums, in lane 0, of its lanes' corner sums.
__device__ __forceinline__ void sum_start(const float4& v, double (&s)[4])
{
    s[0] = v.x;
    s[1] = v.y;
    s[2] = v.z;
    s[3] = v.w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] += __shfl_down_sync(0xffffffffu, s[q], o);
}

// Adds what the block's buckets hold to the call's sums: per node and array the
// corners of the up to four cells around it that were not drained yet and, if some
// warp drained, the block's binary64 row (in Kahan mode its warps' rows). Four nodes
// of a thread are in flight at a time. The four corners of one array are added in
// binary32 (binary64 adds run at 1.7 per SM and cycle: with every corner widened
// first, 2^14 paths on 20 x 10 nodes take 24.4 us a call instead of 23.3 and 2^18 on 30 x 60
// 197 instead of 184, at the same rounding), each a sum of a quarter of the
// contributions that a node's own bucket would hold; everything after in binary64.
template <int ACC, bool OWN>
__device__ __forceinline__ void fold_buckets(const McParams& P, const double* row, bool drained, int start_node)
{
    constexpr int kFly = 4;
    const int I = P.I, nIJ = P.Je * I, B = blockDim.x, W = B >> 5, G = bucket_arrays(W), nc = bucket_count(I, P.Je);
    const float* c0 = reinterpret_cast<const float*>(P.l1 + (size_t)blockIdx.x * G * nc);
    const double* rows0 = P.warp_rows + (size_t)blockIdx.x * W * nIJ;
    // the start cell, a lane's sums each: one warp an array (there are no more arrays than warps)
    const int a0 = (int)(threadIdx.x >> 5);
    const float4 start = OWN && a0 < G ? __ldcg(P.l1 + (size_t)(blockIdx.x * G + a0) * nc + start_bucket(P))
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int e0 = threadIdx.x; e0 < nIJ; e0 += kFly * B) {
        double s[kFly];
#pragma unroll
        for (int q = 0; q < kFly; ++q) s[q] = ACC != 1 && drained && e0 + q * B < nIJ ? __ldcg(row + 3 + e0 + q * B) : 0.0;
        for (int a = 0; a < G; ++a) {
            const float* c = c0 + 4 * (size_t)(a * nc);                  // reductions are resolved in L2: __ldcg
            float f[kFly][4];
#pragma unroll
            for (int q = 0; q < kFly; ++q) {
                const int e = e0 + q * B, j = e / I, i = e - j * I;
                const int cell = 4 * (j * (I - 1) + i);                  // the cell whose lower corner is node e
                const bool in = e < nIJ, up = j < P.Je - 1, rt = i < I - 1;
                f[q][0] = in && up && rt ? __ldcg(c + cell) : 0.0f;
                f[q][1] = in && up && i > 0 ? __ldcg(c + cell - 4 + 1) : 0.0f;
                f[q][2] = in && j > 0 && rt ? __ldcg(c + cell - 4 * (I - 1) + 2) : 0.0f;
                f[q][3] = in && j > 0 && i > 0 ? __ldcg(c + cell - 4 * (I - 1) - 4 + 3) : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kFly; ++q) s[q] += (double)((f[q][0] + f[q][1]) + (f[q][2] + f[q][3]));
        }
#pragma unroll
        for (int q = 0; q < kFly; ++q) {
            const int e = e0 + q * B;
            if (ACC == 1 && drained && e < nIJ) {
                for (int w = 0; w < W; ++w) {
                    const float2 k = reinterpret_cast<const float2*>(rows0 + (size_t)w * nIJ)[e];
                    s[q] += (double)k.x - (double)k.y;
                }
            }
            if (s[q] != 0.0) atomicAdd(&P.sums[3 + e], s[q]);
        }
    }
    if (OWN && a0 < G) {
        double s[4];
        sum_start(start, s);
        if ((threadIdx.x & 31) == 0)
            for (int q = 0; q < 4; ++q) atomicAdd(&P.sums[3 + start_node + (q & 1) + (q >> 1) * I], s[q]);
    }
}

// End of a launch (level 3). Every block has added its sums to P.sums; the last
// one to arrive turns them into the call's outputs and leaves the sums and the
// counters at zero for the next launch. It replaces two launches that summed the
// blocks' rows: where the blocks end at different times their additions hide
// behind the blocks still running, and only the last block's pass over the outputs
// is left. It took 17 us off a call of 2^20 paths on the 30 x 60 grid with 156 steps
// (489 us now), 11 off a forward-only one (223) and 4.4 off 2^14 paths on the 20 x 10 grid
// with 52 steps (23). The divisions by the path count are products with its inverse: a
// binary64 division takes 551 cycles here. A nonzero flag (a vanishing 1 + g_n on a live path of the
// tangent-ratio forms) makes every output NaN. Outputs in the ABI layout (vega
// spot-major); EXTRA: d price / d r and d price / d T after the vegas.
template <bool GREEKS, bool EXTRA = false>
__device__ __forceinline__ void finish_call(const McParams& P)
{
    __shared__ int s_last;
    __threadfence();                      // this thread's additions before the block's arrival
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(P.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();                      // every block's additions before the reads below
    const int B = blockDim.x, tid = threadIdx.x;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const bool bad = P.flag && __ldcg(P.flag) != 0u;
    const int nIJ = P.Je * P.I;
    if (tid == 0) {
        const double s0 = __ldcg(P.sums), s1 = __ldcg(P.sums + 1), s2 = __ldcg(P.sums + 2);
        if (P.want_sums) {
            P.out[0] = bad ? nan : s0;
            P.out[1] = bad ? nan : s1;
            P.out[2] = bad ? nan : s2;
        } else {
            const double mean = s0 * P.inv_paths;
            const double var = (s1 * P.inv_paths - mean * mean) * P.var_scale;
            P.out[LV_OUT_PRICE_DEV] = bad ? nan : mean;
            P.out[LV_OUT_STDERR_DEV] = bad ? nan : (var > 0.0 || var != var) ? sqrt(var * P.inv_paths) : 0.0;
            P.out[LV_OUT_DELTA_DEV] = bad ? nan : s2 * P.inv_delta;
        }
        P.sums[0] = P.sums[1] = P.sums[2] = 0.0;
        *P.tile_counter = 0u;
        *P.done = 0u;
    }
    const double scale = P.want_sums ? 1.0 : P.inv_paths;
    if (GREEKS) {
        double* s = P.sums + 3;           // time-major buckets j I + i
        constexpr int kFly = 8;           // buckets of a thread in flight
        for (int e0 = tid; e0 < nIJ; e0 += kFly * B) {
            double v[kFly];
#pragma unroll
            for (int q = 0; q < kFly; ++q) v[q] = e0 + q * B < nIJ ? __ldcg(s + e0 + q * B) : 0.0;
#pragma unroll
            for (int q = 0; q < kFly; ++q) {
                const int e = e0 + q * B;
                if (e >= nIJ) break;
                s[e] = 0.0;
                const int j = e / P.I, i = e - j * P.I;
                if (j < P.J) P.out[3 + i * P.J + j] = bad ? nan : v[q] * scale;   // not the padding row of one time node
            }
        }
    }
    if (EXTRA && tid < 2) {
        double* s = P.sums + 3 + nIJ + tid;
        P.out[3 + P.I * P.J + tid] = __ldcg(s) * scale;
        *s = 0.0;
    }
    if (P.flag) {
        __syncthreads();                  // every thread has read it
        if (tid == 0) *P.flag = 0u;
    }
}

// Claims the warp's next n consecutive tiles; returns the first. Every warp of
// the grid starts on the tiles of its own index without a claim, so the counter
// gives those after them, and a call with no more than that many claims nothing.
__device__ __forceinline__ int claim_tile(const McParams& P, int n = 1)
{
    const int first = (int)(gridDim.x * (blockDim.x >> 5)) * n;
    if (P.n_tiles <= first) return P.n_tiles;
    int t = 0;
    if ((threadIdx.x & 31) == 0) t = first + (int)atomicAdd(P.tile_counter, (unsigned)n);
    return __shfl_sync(0xffffffffu, t, 0);
}

__device__ __forceinline__ int first_tile(int n = 1)
{
    return (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * n;
}

// Takes a bucket's four sums, leaving zeros. Word by word, as red_add4's reduction is
// atomic per element: an exchange of all 16 bytes beside it would be a race of two
// sizes, for which the memory model promises nothing. At 2^20 paths (30 x 60 nodes, 156
// steps) either took 509-510 us.
__device__ __forceinline__ float4 take4(float4* p)
{
    float* f = reinterpret_cast<float*>(p);
    return make_float4(atomicExch(f, 0.0f), atomicExch(f + 1, 0.0f), atomicExch(f + 2, 0.0f), atomicExch(f + 3, 0.0f));
}

// Where a warp's count of reverse batches starts, so that the block's warps drain
// in turn, every flush_every / W batches of the block's pace, and not all at once: the
// four warps of an array then leave a few hundred live paths in a bucket. The first
// drain comes half a turn later than that (four batches), which spares calls of two
// batches a warp any drain (2^18 paths: 177 us, 190 with the turns from the start).
__device__ __forceinline__ int first_drain(const McParams& P, int warp, int W)
{
    return warp * P.flush_every / W - P.flush_every / 2;
}

// Moves the block's binary32 buckets into its level-2 row (binary64) or the
// warp's (Kahan). A lane takes one column of cells, hands their right corners to
// the next lane and carries the upper corners to the next row, so that every node
// gets one addition; 31 columns a warp at a time (the last lane only receives),
// eight rows of them in flight. A bucket that reads zero is left for a later
// drain. The binary64 row is updated by plain loads and stores under the block's
// lock (flags[1]): as binary64 reductions, two a node, a drain took 28 us of its
// warp's time when every warp drained. Returns false when another warp holds the
// lock: the caller tries again after its next batch.
template <int ACC, bool OWN>
__device__ __forceinline__ bool drain_buckets(const McParams& P, float4* l1, double* wrow, int* flags, int start_node)
{
    constexpr int kFly = 8;
    const int lane = threadIdx.x & 31, I = P.I, C = I - 1, rows = P.Je - 1;
    if (ACC == 0) {
        int got = 0;
        if (lane == 0) got = atomicCAS(&flags[1], 0, 1) == 0;
        if (!__shfl_sync(0xffffffffu, got, 0)) return false;
        __threadfence_block();
    }
    if (lane == 0) flags[0] = 1;
    auto kahan = [&](int e, float f) {
        float2* k = reinterpret_cast<float2*>(wrow) + e;
        float2 p = *k;
        const float y = f - p.y;
        const float t = p.x + y;
        p.y = (t - p.x) - y;
        p.x = t;
        *k = p;
    };
    if (OWN) {                                   // the start cell, a lane's sums each
        double s[4];
        sum_start(take4(l1 + start_bucket(P)), s);
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = start_node + (q & 1) + (q >> 1) * I;
                if (ACC == 1) kahan(e, (float)s[q]);
                else __stcg(wrow + e, __ldcg(wrow + e) + s[q]);
            }
        }
        __threadfence_block();
        __syncwarp();
    }
    for (int i0 = 0; i0 < C; i0 += 31) {
        const int i = i0 + lane;
        const bool cell = lane < 31 && i < C, node = i <= C;
        float carry = 0.0f;
        auto put = [&](int e, double d, float f) {
            if (f == 0.0f) return;
            if (ACC == 1) kahan(e, f);
            else __stcg(wrow + e, d + (double)f);
        };
        for (int j0 = 0; j0 <= rows; j0 += kFly) {          // node rows 0 .. rows
            float4 v[kFly];
            double d[kFly];
#pragma unroll
            for (int q = 0; q < kFly; ++q) {
                v[q] = cell && j0 + q < rows ? __ldcg(l1 + (j0 + q) * C + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                d[q] = ACC == 0 && node && j0 + q <= rows ? __ldcg(wrow + (j0 + q) * I + i) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < kFly; ++q)
                if (v[q].x != 0.0f || v[q].y != 0.0f || v[q].z != 0.0f || v[q].w != 0.0f)
                    v[q] = take4(l1 + (j0 + q) * C + i);
#pragma unroll
            for (int q = 0; q < kFly; ++q) {
                const float y = __shfl_up_sync(0xffffffffu, v[q].y, 1), w = __shfl_up_sync(0xffffffffu, v[q].w, 1);
                const float f = (v[q].x + (lane > 0 ? y : 0.0f)) + carry;
                carry = v[q].z + (lane > 0 ? w : 0.0f);
                if (node && j0 + q <= rows) put((j0 + q) * I + i, d[q], f);
            }
        }
        __threadfence_block();                   // the next columns' first lane updates this one's last node
        __syncwarp();
    }
    if (ACC == 0 && lane == 0) atomicExch(&flags[1], 0);
    return true;
}

// WIDE: one block of 512 threads per SM (choose_launch): the sixteen warps share one copy of
// the sigma pairs in shared memory instead of reading them through L1 (100 x 100 grid,
// 1,260 steps, 2^22 paths: 18.4 -> 16.1 ms; 300 steps, 2^17 paths 342 -> 268 us), and their
// lanes have buckets of their own for the cell that the paths start in (start_bucket).
// Grids that four blocks of 128 stage as well gain a little from the one staging and
// the fewer blocks to fold (30 x 60, 156 steps: 2^20 paths 527 -> 519 us, tangent ratio 587 ->
// 568; 500,000 second-order buckets 362 -> 340), so every call with a tile for each warp
// of the chip runs this form unless its launch shape was chosen otherwise.
//
// Launch bound: the straight-line time loops (time_blocks, reverse_path) want
// registers more than warps. Four blocks per SM at 124-128 registers against
// five at 96 and six at 80, in 128-thread blocks before the bucket reductions of 16 bytes
// (527 us at 2^20 paths now): 615, 643 and 684 us on the 30 x 60 grid with 156
// steps, 2.06, 2.20 and 2.30 ms at 2^22. One path per lane needs 110 registers; held to
// five blocks it gained 1-4 % from 2^20 paths on, where two paths per lane are
// faster still, and lost 4-5 % below.
//
// PPL: paths per lane of a forward tile. With PPL = 2 a warp claims two
// consecutive 32-path tiles and runs them interleaved (forward_path2: two
// independent dependency chains per lane, the per-step time data loaded once);
// each path's arithmetic is that of PPL = 1, the ring groups and the FIFO
// hold twice as many entries, and the reverse batches are unchanged.
template <int KCK, int ACC, bool DBG, bool GS, int MODEL, bool EXTRA, int PPL, int CELL, bool WIDE = false>
__global__ void __launch_bounds__(WIDE ? kWideBlock : 128, WIDE ? 1 : 4) adjoint_kernel(const __grid_constant__ McParams P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kSlots = kTile * PPL;      // checkpoint slots per ring group
    constexpr int kQcap = kQueue * PPL;      // FIFO entries per warp
    const int B = blockDim.x, W = B >> 5;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const SmemLayout L = smem_layout(P.I, P.J, P.N, P.n_bins, B, true, GS, EXTRA, PPL);
    int* const drained = reinterpret_cast<int*>(smem + L.flag);
    AccSlot* const acc0 = reinterpret_cast<AccSlot*>(smem + L.acc);
    AccSlot* acc = acc0 + tid;               // [3][block]: V, V^2, xbar_0; then d V / d r, d V / d T
    stage_grid<GS, EXTRA>(P, smem, L, [&]() {
        clear_buckets<ACC>(P, drained);
        for (int k = 0; k < (EXTRA ? 5 : 3); ++k) acc[k * B] = AccSlot{0.0, 0.0f, 0.0f};
    });
    float4* const l1 = warp_buckets(P, warp, B >> 5);
    // the three FIFO arrays of all warps are contiguous from L.qslot (each
    // W * kQcap words): one base per warp, the others at fixed offsets, which
    // keeps two registers free for the packed forward pass
    int* const q_slot = reinterpret_cast<int*>(smem + L.qslot) + warp * 3 * kQcap;
    int* const q_rel = q_slot + kQcap;
    float* const q_xb = reinterpret_cast<float*>(q_slot + 2 * kQcap);
    const int nIJ = P.Je * P.I;
    const int wid = blockIdx.x * W + warp;                    // global warp id
    const SmemGrid g{ reinterpret_cast<const int4*>(smem + L.tab),
                      GS ? reinterpret_cast<const float2*>(smem + L.sig) : P.sig2,
                      reinterpret_cast<const float*>(smem + L.node), reinterpret_cast<const float2*>(smem + L.ab),
                      reinterpret_cast<const float4*>(smem + L.bins), reinterpret_cast<const float*>(smem + L.tdt) };
    const size_t cks = (size_t)gridDim.x * W * kRing * kSlots;  // checkpoint stride
    float* const ckw = P.ckpt + (size_t)wid * kRing * kSlots;    // this warp's slots

    int q_head = 0, q_count = 0, batches = first_drain(P, warp, B >> 5);
    unsigned fwd_count = 0;
    int tile = first_tile(PPL);

    while (true) {
        const int g_next = (int)(fwd_count % kRing);
        const bool more = tile < P.n_tiles;
        const bool reuse = more && q_count > 0 && q_slot[q_head] / kSlots == g_next;
        if (q_count >= 32 || (!more && q_count > 0) || reuse) {
            // ---------------- reverse batch over up to 32 queued paths
            const int nb = min(32, q_count);
            if (lane < nb) {
                const int e = (q_head + lane) & (kQcap - 1);
                const int slot = q_slot[e];
                const long long rel = q_rel[e];
                float xbar = q_xb[e];
                uint32_t c1, c2;
                path_counter(P, rel, c1, c2);
                float ra = 0.0f, ta = 0.0f;
                xbar = reverse_path<CELL, KCK, MODEL, EXTRA, PPL == 2, WIDE>(
                    P, g, c1, c2, ckw + slot, cks, xbar, l1, &ra, &ta);
                acc_add<ACC>(acc[2 * B], xbar);
                if (EXTRA) {
                    acc_add<ACC>(acc[3 * B], ra);
                    acc_add<ACC>(acc[4 * B], ta);
                }
                if (DBG) P.dbg_xbar0[rel] = xbar;
            }
            q_head = (q_head + nb) & (kQcap - 1);
            q_count -= nb;
            __syncwarp();
            if (++batches >= P.flush_every && drain_buckets<ACC, WIDE>(P, l1, level2_row<ACC>(P), drained, start_node<WIDE, MODEL, CELL>(P, g))) batches = 0;
            continue;
        }
        if (!more) break;

        if constexpr (PPL == 2) {
            // ---------------- forward tiles tile, tile + 1: two paths per lane
            const long long rel_a = (long long)tile * kTile + lane, rel_b = rel_a + kTile;
            const int slot_a = g_next * kSlots + lane, slot_b = slot_a + kTile;
            float xa = 0.0f, xb = 0.0f;
            if (rel_a < P.n_paths) {
                uint32_t c1a, c2a, c1b, c2b;
                path_counter(P, rel_a, c1a, c2a);
                path_counter(P, rel_b, c1b, c2b);
                float ya, yb;
                // packed under every reading (Euler on S, 2^22 paths: 1 % faster than scalar pairs)
                forward_path2<CELL, KCK, true, MODEL, true>(P, g, c1a, c2a, c1b, c2b, ckw + slot_a,
                                                                             ckw + slot_b, cks, ya, yb);
                auto add = [&](float V) {
                    acc_add<ACC>(acc[0], V);
                    acc_add<ACC>(acc[B], V * V);
                    if (EXTRA) {                   // the discount's share: -T V and -r V
                        acc_add<ACC>(acc[3 * B], -P.Tf * V);
                        acc_add<ACC>(acc[4 * B], -P.r_nat * V);
                    }
                };
                float V;
                payoff<MODEL>(P, ya, V, xa);
                add(V);
                if (rel_b < P.n_paths) {
                    payoff<MODEL>(P, yb, V, xb);
                    add(V);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float xbarN = h ? xb : xa;
                const bool live = xbarN != 0.0f;
                const unsigned bal = __ballot_sync(0xffffffffu, live);
                if (live) {
                    const int e = (q_head + q_count + __popc(bal & ((1u << lane) - 1u))) & (kQcap - 1);
                    q_slot[e] = h ? slot_b : slot_a;
                    q_rel[e] = (int)(h ? rel_b : rel_a);
                    q_xb[e] = xbarN;
                }
                q_count += __popc(bal);
            }
            ++fwd_count;
            __syncwarp();
            tile = claim_tile(P, PPL);
            continue;
        }

        // ---------------- forward tile of 32 paths into slot group g_next
        const long long rel = (long long)tile * kTile + lane;
        const bool active = rel < P.n_paths;
        const int slot = g_next * kTile + lane;
        float xbarN = 0.0f;
        if (active) {
            uint32_t c1, c2;
            path_counter(P, rel, c1, c2);
            const float x = forward_path<CELL, KCK, true, DBG, MODEL>(P, g, c1, c2, ckw + slot, cks, rel);
            float V;
            payoff<MODEL>(P, x, V, xbarN);
            acc_add<ACC>(acc[0], V);
            acc_add<ACC>(acc[B], V * V);
            if (EXTRA) {                       // the discount's share: -T V and -r V
                acc_add<ACC>(acc[3 * B], -P.Tf * V);
                acc_add<ACC>(acc[4 * B], -P.r_nat * V);
            }
            if (DBG) {
                P.dbg_xN[rel] = ln_spot<MODEL>(x);
                P.dbg_V[rel] = V;
                P.dbg_xbar0[rel] = 0.0f;
            }
        }
        const bool live = xbarN != 0.0f;
        const unsigned bal = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int e = (q_head + q_count + __popc(bal & ((1u << lane) - 1u))) & (kQcap - 1);
            q_slot[e] = slot;
            q_rel[e] = (int)rel;
            q_xb[e] = xbarN;
        }
        q_count += __popc(bal);
        ++fwd_count;
        __syncwarp();
        tile = claim_tile(P, PPL);
    }

    __syncthreads();                           // after it nothing adds to this block's buckets
    fold_buckets<ACC, WIDE>(P, P.partials + (size_t)blockIdx.x * P.row_words, *drained != 0,
                            start_node<WIDE, MODEL, CELL>(P, g));
    add_scalars<ACC>(acc0, 3, P.sums);
    if (EXTRA) add_scalars<ACC>(acc0 + 3 * B, 2, P.sums + 3 + nIJ);
    finish_call<true, EXTRA>(P);
}

// Tangent-ratio adjoint (LV_ADJ_TANGENT): persistent and warp-centric like
// adjoint_kernel, without checkpoints. A warp claims a tile of 32 paths and
// runs pass 1 (tangent_forward): payoff, xbar_N, and xbar_0 = xbar_N D_N;
// the paths with xbar_N != 0 join the warp's queue with c = xbar_N D_N. At
// 32 queued paths (and at the end) the warp runs pass 2 (tangent_scatter)
// on them as a full-warp batch. Buckets go through the same levels 0-3.
template <int ACC, bool GS, int MODEL, int PPL, int CELL, bool WIDE = false>
__global__ void __launch_bounds__(WIDE ? kWideBlock : 128, WIDE ? 1 : 5) tangent_kernel(const __grid_constant__ McParams P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int B = blockDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kQcap = kQueue * PPL;
    const SmemLayout L = smem_layout(P.I, P.J, P.N, P.n_bins, B, true, GS, false, PPL);
    int* const drained = reinterpret_cast<int*>(smem + L.flag);
    AccSlot* const acc0 = reinterpret_cast<AccSlot*>(smem + L.acc);
    AccSlot* acc = acc0 + tid;               // [3][block]: V, V^2, xbar_0
    stage_grid<GS>(P, smem, L, [&]() {
        clear_buckets<ACC>(P, drained);
        for (int k = 0; k < 3; ++k) acc[k * B] = AccSlot{0.0, 0.0f, 0.0f};
    });
    float4* const l1 = warp_buckets(P, warp, B >> 5);
    int* q_rel = reinterpret_cast<int*>(smem + L.qrel) + warp * kQcap;
    float* q_c = reinterpret_cast<float*>(smem + L.qxb) + warp * kQcap;
    const SmemGrid g{ reinterpret_cast<const int4*>(smem + L.tab),
                      GS ? reinterpret_cast<const float2*>(smem + L.sig) : P.sig2,
                      reinterpret_cast<const float*>(smem + L.node), reinterpret_cast<const float2*>(smem + L.ab),
                      reinterpret_cast<const float4*>(smem + L.bins) };
    int q_head = 0, q_count = 0, batches = first_drain(P, warp, B >> 5);
    int tile = first_tile(PPL);
    while (true) {
        const bool more = tile < P.n_tiles;
        if (q_count >= 32 || (!more && q_count > 0)) {
            const int nb = min(32, q_count);
            if (lane < nb) {
                const int e = (q_head + lane) & (kQcap - 1);
                uint32_t c1, c2;
                path_counter(P, q_rel[e], c1, c2);
                tangent_scatter<CELL, MODEL, WIDE>(P, g, c1, c2, q_c[e], l1);
            }
            q_head = (q_head + nb) & (kQcap - 1);
            q_count -= nb;
            __syncwarp();
            if (++batches >= P.flush_every && drain_buckets<ACC, WIDE>(P, l1, level2_row<ACC>(P), drained, start_node<WIDE, MODEL, CELL>(P, g))) batches = 0;
            continue;
        }
        if (!more) break;
        if constexpr (PPL == 2) {
            // pass 1 on tiles tile, tile + 1: two paths per lane in packed pairs
            const long long rel_a = (long long)tile * kTile + lane, rel_b = rel_a + kTile;
            float xa = 0.0f, xb = 0.0f, ca = 0.0f, cb = 0.0f;
            if (rel_a < P.n_paths) {
                uint32_t c1a, c2a, c1b, c2b;
                path_counter(P, rel_a, c1a, c2a);
                path_counter(P, rel_b, c1b, c2b);
                float ya, yb, Da, Db, V;
                bool ta, tb;
                tangent_forward2<CELL>(P, g, c1a, c2a, c1b, c2b, ya, yb, Da, Db, ta, tb);
                payoff<0>(P, ya, V, xa);
                ca = xa * Da;
                acc_add<ACC>(acc[0], V);
                acc_add<ACC>(acc[B], V * V);
                acc_add<ACC>(acc[2 * B], ca);
                if (ta && xa != 0.0f) atomicAdd(P.flag, 1u);
                if (rel_b < P.n_paths) {
                    payoff<0>(P, yb, V, xb);
                    cb = xb * Db;
                    acc_add<ACC>(acc[0], V);
                    acc_add<ACC>(acc[B], V * V);
                    acc_add<ACC>(acc[2 * B], cb);
                    if (tb && xb != 0.0f) atomicAdd(P.flag, 1u);
                }
            }
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const float x = hh ? xb : xa;
                const bool live = x != 0.0f;
                const unsigned bal = __ballot_sync(0xffffffffu, live);
                if (live) {
                    const int e = (q_head + q_count + __popc(bal & ((1u << lane) - 1u))) & (kQcap - 1);
                    q_rel[e] = (int)(hh ? rel_b : rel_a);
                    q_c[e] = hh ? cb : ca;
                }
                q_count += __popc(bal);
            }
            __syncwarp();
            tile = claim_tile(P, PPL);
            continue;
        }
        const long long rel = (long long)tile * kTile + lane;
        float xbarN = 0.0f, c = 0.0f;
        if (rel < P.n_paths) {
            uint32_t c1, c2;
            path_counter(P, rel, c1, c2);
            float D;
            bool tiny;
            const float y = tangent_forward<CELL, MODEL>(P, g, c1, c2, D, tiny);
            float V;
            payoff<MODEL>(P, y, V, xbarN);
            c = xbarN * D;
            acc_add<ACC>(acc[0], V);
            acc_add<ACC>(acc[B], V * V);
            acc_add<ACC>(acc[2 * B], c);
            if (tiny && xbarN != 0.0f) atomicAdd(P.flag, 1u);
        }
        const bool live = xbarN != 0.0f;
        const unsigned bal = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int e = (q_head + q_count + __popc(bal & ((1u << lane) - 1u))) & (kQcap - 1);
            q_rel[e] = (int)rel;
            q_c[e] = c;
        }
        q_count += __popc(bal);
        __syncwarp();
        tile = claim_tile(P, PPL);
    }
    __syncthreads();
    fold_buckets<ACC, WIDE>(P, P.partials + (size_t)blockIdx.x * P.row_words, *drained != 0,
                            start_node<WIDE, MODEL, CELL>(P, g));
    add_scalars<ACC>(acc0, 3, P.sums);
    finish_call<true>(P);
}

// Second-order buckets (lv_price_greeks_vanna): the tangent-ratio kernel's
// structure with pass 2 replaced by vanna_scatter. Pass 1 (tangent_forward)
// gives the payoff and x_bar_0 = x_bar_N D_N, hence Delta_p = x_bar_0 / S0;
// live paths are queued and scattered in full-warp batches. Main reading,
// binary64 level 2. Rows: price sums as usual, buckets d^2 price / (d S0 d
// sigma_ij) summed over paths.
template <bool GS, int PPL, int CELL, bool WIDE = false>
__global__ void __launch_bounds__(WIDE ? kWideBlock : 128, WIDE ? 1 : 5) vanna_kernel(const __grid_constant__ McParams P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int B = blockDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kQcap = kQueue * PPL;
    const SmemLayout L = smem_layout(P.I, P.J, P.N, P.n_bins, B, true, GS, false, PPL);
    int* const drained = reinterpret_cast<int*>(smem + L.flag);
    AccSlot* const acc0 = reinterpret_cast<AccSlot*>(smem + L.acc);
    AccSlot* acc = acc0 + tid;               // [3][block]: V, V^2, xbar_0
    stage_grid<GS>(P, smem, L, [&]() {
        clear_buckets<0>(P, drained);
        for (int k = 0; k < 3; ++k) acc[k * B] = AccSlot{0.0, 0.0f, 0.0f};
    });
    float4* const l1 = warp_buckets(P, warp, B >> 5);
    int* q_rel = reinterpret_cast<int*>(smem + L.qrel) + warp * kQcap;
    float* q_c = reinterpret_cast<float*>(smem + L.qxb) + warp * kQcap;
    const SmemGrid g{ reinterpret_cast<const int4*>(smem + L.tab),
                      GS ? reinterpret_cast<const float2*>(smem + L.sig) : P.sig2,
                      reinterpret_cast<const float*>(smem + L.node), reinterpret_cast<const float2*>(smem + L.ab),
                      reinterpret_cast<const float4*>(smem + L.bins) };
    int q_head = 0, q_count = 0, batches = first_drain(P, warp, B >> 5);
    int tile = first_tile(PPL);
    while (true) {
        const bool more = tile < P.n_tiles;
        if (q_count >= 32 || (!more && q_count > 0)) {
            const int nb = min(32, q_count);
            if (lane < nb) {
                const int e = (q_head + lane) & (kQcap - 1);
                uint32_t c1, c2;
                path_counter(P, q_rel[e], c1, c2);
                vanna_scatter<CELL, WIDE>(P, g, c1, c2, q_c[e] * P.inv_S0, l1);
            }
            q_head = (q_head + nb) & (kQcap - 1);
            q_count -= nb;
            __syncwarp();
            if (++batches >= P.flush_every && drain_buckets<0, WIDE>(P, l1, level2_row<0>(P), drained, start_node<WIDE, 0, CELL>(P, g))) batches = 0;
            continue;
        }
        if (!more) break;
        if constexpr (PPL == 2) {
            // pass 1 on tiles tile, tile + 1: two paths per lane in packed pairs
            const long long rel_a = (long long)tile * kTile + lane, rel_b = rel_a + kTile;
            float xa = 0.0f, xb = 0.0f, ca = 0.0f, cb = 0.0f;
            if (rel_a < P.n_paths) {
                uint32_t c1a, c2a, c1b, c2b;
                path_counter(P, rel_a, c1a, c2a);
                path_counter(P, rel_b, c1b, c2b);
                float ya, yb, Da, Db, V;
                bool ta, tb;
                tangent_forward2<CELL>(P, g, c1a, c2a, c1b, c2b, ya, yb, Da, Db, ta, tb);
                payoff<0>(P, ya, V, xa);
                ca = xa * Da;
                acc_add<0>(acc[0], V);
                acc_add<0>(acc[B], V * V);
                acc_add<0>(acc[2 * B], ca);
                if (ta && xa != 0.0f) atomicAdd(P.flag, 1u);
                if (rel_b < P.n_paths) {
                    payoff<0>(P, yb, V, xb);
                    cb = xb * Db;
                    acc_add<0>(acc[0], V);
                    acc_add<0>(acc[B], V * V);
                    acc_add<0>(acc[2 * B], cb);
                    if (tb && xb != 0.0f) atomicAdd(P.flag, 1u);
                }
            }
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const float x = hh ? xb : xa;
                const bool live = x != 0.0f;
                const unsigned bal = __ballot_sync(0xffffffffu, live);
                if (live) {
                    const int e = (q_head + q_count + __popc(bal & ((1u << lane) - 1u))) & (kQcap - 1);
                    q_rel[e] = (int)(hh ? rel_b : rel_a);
                    q_c[e] = hh ? cb : ca;
                }
                q_count += __popc(bal);
            }
            __syncwarp();
            tile = claim_tile(P, PPL);
            continue;
        }
        const long long rel = (long long)tile * kTile + lane;
        float xbarN = 0.0f, c = 0.0f;
        if (rel < P.n_paths) {
            uint32_t c1, c2;
            path_counter(P, rel, c1, c2);
            float D;
            bool tiny;
            const float y = tangent_forward<CELL, 0>(P, g, c1, c2, D, tiny);
            float V;
            payoff<0>(P, y, V, xbarN);
            c = xbarN * D;
            acc_add<0>(acc[0], V);
            acc_add<0>(acc[B], V * V);
            acc_add<0>(acc[2 * B], c);
            if (tiny && xbarN != 0.0f) atomicAdd(P.flag, 1u);
        }
        const bool live = xbarN != 0.0f;
        const unsigned bal = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int e = (q_head + q_count + __popc(bal & ((1u << lane) - 1u))) & (kQcap - 1);
            q_rel[e] = (int)rel;
            q_c[e] = c;
        }
        q_count += __popc(bal);
        __syncwarp();
        tile = claim_tile(P, PPL);
    }
    __syncthreads();
    fold_buckets<0, WIDE>(P, P.partials + (size_t)blockIdx.x * P.row_words, *drained != 0,
                          start_node<WIDE, 0, CELL>(P, g));
    add_scalars<0>(acc0, 3, P.sums);
    finish_call<true>(P);
}

// The forward pass alone. Bound by the FMA pipe (its 64-bit integer products
// hold it for four cycles each) and the issue slots. With the straight-line
// time loop, the index without a conversion and the round keys in the parameter
// bank it runs 33 thread instructions per path-step, 43 with a check in every step: 223 us
// a call of 2^20 paths on the 30 x 60 grid with 156 steps, from 291. Every tile takes
// the same time, so the registers are held to nine blocks (12 us less than with eight
// there) and the launcher picks the blocks per SM that leave the last round of tiles
// fullest (make_plan).
template <int ACC, bool GS, int MODEL, int CELL, int PPL>
__global__ void __launch_bounds__(128, 9) price_kernel(const __grid_constant__ McParams P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const SmemLayout L = smem_layout(P.I, P.J, P.N, P.n_bins, blockDim.x, false, GS);
    AccSlot* const acc0 = reinterpret_cast<AccSlot*>(smem + L.acc);
    AccSlot* acc = acc0 + threadIdx.x;
    stage_grid<GS>(P, smem, L, [&]() { acc[0] = acc[blockDim.x] = AccSlot{0.0, 0.0f, 0.0f}; });
    const SmemGrid g{ reinterpret_cast<const int4*>(smem + L.tab),
                      GS ? reinterpret_cast<const float2*>(smem + L.sig) : P.sig2,
                      reinterpret_cast<const float*>(smem + L.node), reinterpret_cast<const float2*>(smem + L.ab),
                      reinterpret_cast<const float4*>(smem + L.bins) };
    const int lane = threadIdx.x & 31;
    for (int tile = first_tile(); tile < P.n_tiles; tile = claim_tile(P)) {
        const long long rel_a = (long long)tile * (kTile * PPL) + lane, rel_b = rel_a + 32;
        if (rel_a < P.n_paths) {
            uint32_t c1a, c2a, c1b, c2b;
            path_counter(P, rel_a, c1a, c2a);
            float ya, yb, V, xb;
            if constexpr (PPL == 1) {
                ya = forward_path<CELL, 4, false, false, MODEL>(P, g, c1a, c2a, nullptr, 0, rel_a);
                payoff<MODEL>(P, ya, V, xb);
                acc_add<ACC>(acc[0], V);
                acc_add<ACC>(acc[blockDim.x], V * V);
                continue;
            }
            path_counter(P, rel_b, c1b, c2b);
            forward_path2<CELL, 4, false, MODEL, true>(P, g, c1a, c2a, c1b, c2b, nullptr, nullptr, 0, ya, yb);
            payoff<MODEL>(P, ya, V, xb);
            acc_add<ACC>(acc[0], V);
            acc_add<ACC>(acc[blockDim.x], V * V);
            if (rel_b < P.n_paths) {
                payoff<MODEL>(P, yb, V, xb);
                acc_add<ACC>(acc[0], V);
                acc_add<ACC>(acc[blockDim.x], V * V);
            }
        }
    }
    __syncthreads();
    add_scalars<ACC>(acc0, 2, P.sums);
    finish_call<false>(P);
}

template <typename K>
cudaError_t set_smem_attr(K kernel)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

template <typename K>
cudaError_t launch_configured(K kernel, bool& configured, const McParams& p, int grid, int block, size_t smem,
                              cudaStream_t s)
{
    if (!configured) {
        cudaError_t e = set_smem_attr(kernel);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    kernel<<<grid, block, smem, s>>>(p);
    return cudaGetLastError();
}

template <typename K>
cudaError_t occupancy(K kernel, int block, size_t smem, int* bps)
{
    cudaError_t e = set_smem_attr(kernel);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, kernel, block, smem);
}

// Calls f(kernel, flag) with the instantiation for (greeks, k, acc, dbg, gs)
// of model MODEL and cell mode CELL: k in {4, 8}, and for model 0 with the search
// also 16 and 32.
template <int MODEL, bool GS, int CELL, typename F>
cudaError_t with_kernel_gs(bool greeks, int k, int acc, bool dbg, int method, bool extra, F&& f, int ppl = 1,
                           bool wide = false)
{
    if (wide) {            // 512-thread blocks: every Greeks kernel, the reverse sweep with checkpoints every 4 steps
        if constexpr (GS && CELL != kCellSearch) {
            static bool cw[12] = {};
            if (!greeks || dbg) return cudaErrorInvalidValue;
            if constexpr (MODEL == 0) {
                if (method == kMethodVanna && acc == 0)
                    return ppl == 2 ? f(vanna_kernel<true, 2, CELL, true>, cw[6]) : f(vanna_kernel<true, 1, CELL, true>, cw[7]);
                if (method == LV_ADJ_TANGENT && ppl == 2)
                    return acc ? f(tangent_kernel<1, true, 0, 2, CELL, true>, cw[8])
                               : f(tangent_kernel<0, true, 0, 2, CELL, true>, cw[9]);
            }
            if (method == LV_ADJ_TANGENT && ppl == 1)
                return acc ? f(tangent_kernel<1, true, MODEL, 1, CELL, true>, cw[10])
                           : f(tangent_kernel<0, true, MODEL, 1, CELL, true>, cw[11]);
            if (method != LV_ADJ_REVERSE || k != 4) return cudaErrorInvalidValue;
            if (extra && acc == 0)
                return ppl == 2 ? f(adjoint_kernel<4, 0, false, true, MODEL, true, 2, CELL, true>, cw[5])
                                : f(adjoint_kernel<4, 0, false, true, MODEL, true, 1, CELL, true>, cw[4]);
            if (extra) return cudaErrorInvalidValue;
            switch (2 * ppl + acc) {
            case 2: return f(adjoint_kernel<4, 0, false, true, MODEL, false, 1, CELL, true>, cw[0]);
            case 3: return f(adjoint_kernel<4, 1, false, true, MODEL, false, 1, CELL, true>, cw[1]);
            case 4: return f(adjoint_kernel<4, 0, false, true, MODEL, false, 2, CELL, true>, cw[2]);
            case 5: return f(adjoint_kernel<4, 1, false, true, MODEL, false, 2, CELL, true>, cw[3]);
            default: break;
            }
        }
        return cudaErrorInvalidValue;
    }
    if (!greeks) {
        static bool c0[2] = {}, c1[2] = {};
        if (ppl == 2) return acc ? f(price_kernel<1, GS, MODEL, CELL, 2>, c1[1]) : f(price_kernel<0, GS, MODEL, CELL, 2>, c0[1]);
        return acc ? f(price_kernel<1, GS, MODEL, CELL, 1>, c1[0]) : f(price_kernel<0, GS, MODEL, CELL, 1>, c0[0]);
    }
    if (ppl == 2) {        // two paths per lane: the reverse sweep (k = 4 or 8) of every reading,
                           // the main reading's tangent-ratio adjoint and second-order buckets
        if (!greeks || dbg || extra) return cudaErrorInvalidValue;
        if constexpr (MODEL == 0) {
            static bool cv2 = false, ct2[2] = {};
            if (method == kMethodVanna)
                return acc == 0 ? f(vanna_kernel<GS, 2, CELL>, cv2) : cudaErrorInvalidValue;
            if (method == LV_ADJ_TANGENT)
                return acc ? f(tangent_kernel<1, GS, 0, 2, CELL>, ct2[1]) : f(tangent_kernel<0, GS, 0, 2, CELL>, ct2[0]);
        }
        if (method != LV_ADJ_REVERSE) return cudaErrorInvalidValue;
        static bool cp[4] = {};
        switch (k * 2 + acc) {
        case 8: return f(adjoint_kernel<4, 0, false, GS, MODEL, false, 2, CELL>, cp[0]);
        case 9: return f(adjoint_kernel<4, 1, false, GS, MODEL, false, 2, CELL>, cp[1]);
        case 16: return f(adjoint_kernel<8, 0, false, GS, MODEL, false, 2, CELL>, cp[2]);
        case 17: return f(adjoint_kernel<8, 1, false, GS, MODEL, false, 2, CELL>, cp[3]);
        default: break;
        }
        return cudaErrorInvalidValue;
    }
    if (ppl != 1) return cudaErrorInvalidValue;
    if (method == kMethodVanna) {     // second-order buckets: main reading, binary64 level 2
        if constexpr (MODEL == 0) {
            static bool cv = false;
            if (!greeks || dbg || extra || acc != 0) return cudaErrorInvalidValue;
            return f(vanna_kernel<GS, 1, CELL>, cv);
        }
        return cudaErrorInvalidValue;
    }
    if (extra) {           // d V / d r and d V / d T: reverse sweep, binary64 level 2, k = 4 or 8
        static bool ce[2] = {};
        if (!greeks || dbg || method != LV_ADJ_REVERSE || acc != 0) return cudaErrorInvalidValue;
        if (k == 4) return f(adjoint_kernel<4, 0, false, GS, MODEL, true, 1, CELL>, ce[0]);
        if (k == 8) return f(adjoint_kernel<8, 0, false, GS, MODEL, true, 1, CELL>, ce[1]);
        return cudaErrorInvalidValue;
    }
    if (method == LV_ADJ_TANGENT && !dbg) {
        static bool t0 = false, t1 = false;
        return acc ? f(tangent_kernel<1, GS, MODEL, 1, CELL>, t1) : f(tangent_kernel<0, GS, MODEL, 1, CELL>, t0);
    }
    if (dbg) {
        if constexpr (CELL == kCellSearch) {
            static bool cd = false;
            if (k != 4) return cudaErrorInvalidValue;       // scratch must be planned with k = 4
            return f(adjoint_kernel<4, 0, true, GS, MODEL, false, 1, CELL>, cd);
        }
        return cudaErrorInvalidValue;
    }
    static bool c[8] = {};
    switch (k * 2 + acc) {
    case 8: return f(adjoint_kernel<4, 0, false, GS, MODEL, false, 1, CELL>, c[0]);
    case 9: return f(adjoint_kernel<4, 1, false, GS, MODEL, false, 1, CELL>, c[1]);
    case 16: return f(adjoint_kernel<8, 0, false, GS, MODEL, false, 1, CELL>, c[2]);
    case 17: return f(adjoint_kernel<8, 1, false, GS, MODEL, false, 1, CELL>, c[3]);
    default: break;
    }
    if constexpr (MODEL == 0 && CELL == kCellSearch) {
        switch (k * 2 + acc) {
        case 32: return f(adjoint_kernel<16, 0, false, GS, 0, false, 1, CELL>, c[4]);
        case 33: return f(adjoint_kernel<16, 1, false, GS, 0, false, 1, CELL>, c[5]);
        case 64: return f(adjoint_kernel<32, 0, false, GS, 0, false, 1, CELL>, c[6]);
        case 65: return f(adjoint_kernel<32, 1, false, GS, 0, false, 1, CELL>, c[7]);
        default: break;
        }
    }
    return cudaErrorInvalidValue;
}

template <int MODEL, int CELL>
cudaError_t launch_model_impl(const McParams& p, int grid, int block, int k, bool greeks, size_t smem,
                              cudaStream_t s)
{
    auto run = [&](auto kernel, bool& configured) {
        return launch_configured(kernel, configured, p, grid, block, smem, s);
    };
    const bool dbg = p.dbg_xN != nullptr;
    const int ppl = p.ppl > 1 ? p.ppl : 1;
    const bool wide = block == kWideBlock;
    return p.grid_smem
               ? with_kernel_gs<MODEL, true, CELL>(greeks, k, p.acc_mode, dbg, p.method, p.extra != 0, run, ppl, wide)
               : with_kernel_gs<MODEL, false, CELL>(greeks, k, p.acc_mode, dbg, p.method, p.extra != 0, run, ppl, wide);
}

template <int MODEL, int CELL>
cudaError_t occupancy_model_impl(int block, int k, bool greeks, int acc, bool dbg, bool gs, int method, bool extra,
                                 size_t smem, int* bps, int ppl = 1)
{
    auto occ = [&](auto kernel, bool&) { return occupancy(kernel, block, smem, bps); };
    const bool wide = block == kWideBlock;
    return gs ? with_kernel_gs<MODEL, true, CELL>(greeks, k, acc, dbg, method, extra, occ, ppl, wide)
              : with_kernel_gs<MODEL, false, CELL>(greeks, k, acc, dbg, method, extra, occ, ppl, wide);
}

}  // namespace

}  // namespace lv

// Defines the launcher and the occupancy query of one model and cell mode.
#define LV_DEFINE_KERNELS(M, C)                                                                                  \
    namespace lv {                                                                                               \
    cudaError_t launch_mc_m##M##c##C(const McParams& p, int grid, int block, int k, bool greeks, size_t smem,     \
                                     cudaStream_t s)                                                             \
    {                                                                                                            \
        return launch_model_impl<M, C>(p, grid, block, k, greeks, smem, s);                                      \
    }                                                                                                            \
    cudaError_t mc_occupancy_m##M##c##C(int block, int k, bool greeks, int acc, bool dbg, bool grid_smem,        \
                                        int method, bool extra, size_t smem, int* bps, int ppl)                  \
    {                                                                                                            \
        return occupancy_model_impl<M, C>(block, k, greeks, acc, dbg, grid_smem, method, extra, smem, bps, ppl); \
    }                                                                                                            \
    }
