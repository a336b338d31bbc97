// lv_internal.h -- interface between the host runtime (lv_api.cu) and the
// device kernels (lv_mc.cuh). Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <vector>

namespace lv {

// Output layout of the finalized result (same values as LV_OUT_* in lv.h).
constexpr int LV_OUT_PRICE_DEV = 0;
constexpr int LV_OUT_DELTA_DEV = 1;
constexpr int LV_OUT_STDERR_DEV = 2;

// The round keys of Philox4x32-10 for one key (seed low, seed high): round r
// xors (k[2r], k[2r + 1]) = key + r (0x9E3779B9, 0xBB67AE85). In the kernel
// parameters they are constant-bank operands of the xors, 20 adds fewer per
// block of normals (0.5 % of the adjoint's and the forward pass's time, 1.6 % of the
// second-order buckets').
struct PhiloxKeys {
    uint32_t k[20];
};

__host__ __device__ inline PhiloxKeys philox_keys(uint32_t k0, uint32_t k1)
{
    PhiloxKeys K{};
    for (int r = 0; r < 10; ++r) {
        K.k[2 * r] = k0 + (uint32_t)r * 0x9E3779B9u;
        K.k[2 * r + 1] = k1 + (uint32_t)r * 0xBB67AE85u;
    }
    return K;
}

// How the loops find the spot cell (lv_device.cuh spot_cell). The two without a
// search need every index of the call bounded (index_bounded).
constexpr int kCellSearch = 0, kCellUniform = 1, kCellBins = 2;
constexpr int kCellAny = 3, kCellNoBins = 4;       // chosen on the device (the book)
constexpr int kCellNodes = 5;                      // the search without bins (the bump kernel, which stages none)

// Whether |cell_scale y + cell_shift| stays below 2^22 on every path of a call,
// y = log2 S. On ln S the path moves by at most |rdt| + hdt sigma^2 +
// sqdt2 sigma |Z| a step, and |Z| <= sqrt(-2 ln 2^-24) < 5.8 (23-bit
// uniforms); under the scheme on S, y is log2 of a binary32 spot clamped from
// below at 1e-30.
__host__ __device__ inline bool index_bounded(bool on_s, int n_steps, double x0, double rdt, double hdt,
                                              double sqdt2, double sig_max, double cell_scale, double cell_shift)
{
    const double step = fabs(rdt) + hdt * sig_max * sig_max + 5.8 * sqdt2 * sig_max;
    const double y = on_s ? 130.0 : fabs(x0) + 1.01 * n_steps * step;
    return fabs(cell_scale) * y + fabs(cell_shift) < 4194304.0 - 2.0;     // false for infinities and NaN
}

// Arrays of level-1 buckets of a block: one for every kBucketWarps warps (lv_mc.cuh warp_buckets).
constexpr int kBucketWarps = 4;
__host__ __device__ inline int bucket_arrays(int warps) { return (warps + kBucketWarps - 1) / kBucketWarps; }
// Buckets of an array: the cells', then one a lane for the cell that the paths start in.
__host__ __device__ inline int bucket_count(int I, int Je) { return (Je - 1) * (I - 1) + 32; }

// Everything a Monte Carlo launch reads, passed by value as a
// __grid_constant__ kernel parameter.
struct McParams {
    // grid (device copies, binary32)
    const float2* sig2;    // [Je][I - 1] time-major pairs (sigma_{i,j}, sigma_{i+1,j} - sigma_{i,j});
                           // Je = max(J, 2), row 1 repeats row 0 when J == 1
    const float* node;     // [I] spot nodes s_i
    const float2* ab;      // [I - 1] (1 / (s_{i+1} - s_i), -s_i / (s_{i+1} - s_i))
    const double* tau;     // [J] time nodes, then [J] inverse gaps 1 / (tau_{j+1} - tau_j) (step_time)
    int I, J, Je;
    int log_uniform;       // spot nodes equally spaced in ln S
    int cell_mode;         // kCellSearch, kCellUniform or kCellBins
    const float4* bins;    // [n_bins] (kCellBins)
    int n_bins;
    float cell_scale;      // ln 2 / d(ln s): cell index from y = log2 S
    float cell_shift;      // -ln(s_0) / d(ln s)
    float s_lo, s_hi;      // s_0, s_{I-1}

    // option and scheme; the path state is y = log2 S (or S when the model
    // runs the Euler scheme on S)
    int model;             // bit 0: spot weight linear in ln S; bit 1: Euler scheme on S
    int extra;             // adjoint also sums d V / d r and d V / d T (rows end with them)
    float x0;              // log2 S0 (S0 on S)
    float rdt;             // log2(e) r dt (r dt on S)
    float hdt;             // log2(e) dt / 2
    float sqdt2;           // log2(e) sqrt(dt)
    float dt;
    float sqdt;            // sqrt(dt) (natural units, for d x_{n+1} / d sigma_n)
    float K;
    float disc;            // e^{-rT}
    float S0f, inv_S0;     // S0, 1 / S0 (the scaled adjoint of the scheme on S)
    float Tf, r_nat;       // T, r (d price / d r and d price / d T)
    float inv_N, half_inv_sqdt;   // 1 / N, 1 / (2 sqrt(dt))
    float phi;             // +1 call, -1 put
    double dt_d;           // dt in binary64 for the time table
    int N;                 // steps

    // random numbers
    PhiloxKeys rk;         // Philox key = seed
    uint32_t stream_id;
    long long path_begin;
    long long n_paths;

    // work decomposition and scratch
    int n_tiles;           // ceil(n_paths / paths_per_tile()): tiles claimed by warps
    int ppl;               // adjoint: paths per lane of a forward tile (1 or 2; a warp claims ppl tiles)
    unsigned int* tile_counter;   // zero before the launch, reset by its last block, as are the next two
    unsigned int* done;    // blocks that have added their sums
    double* sums;          // [5 + Je * I] binary64 sums of the call: V, V^2, x_bar_0, buckets
                           // (time-major), then d V / d r and d V / d T
    double* partials;      // [gridDim.x][row_words] per-block binary64 rows
    int row_words;         // 3 + Je * I (adjoint) or 3 (price only)
    double* warp_rows;     // [gridDim.x * warps][Je * I] per-warp level-2 rows
    float4* l1;            // [gridDim.x][bucket_arrays][bucket_count] level-1 buckets: the corner sums of a cell
                           // (nodes (i, j), (i+1, j), (i, j+1), (i+1, j+1))
    float* ckpt;           // [n_ck][gridDim.x * warps * ring_slots_per_warp() * ppl] checkpoints of x
    int n_ck;
    int flush_every;       // reverse batches between level-1 -> level-2 drains
    int grid_smem;         // 1: sigma pairs staged in shared memory, 0: read through L1
    int acc_mode;          // 0 binary64, 1 Kahan binary32
    int method;            // LV_ADJ_REVERSE or LV_ADJ_TANGENT
    unsigned int* flag;    // tangent-ratio adjoint: count of live paths with a vanishing 1 + g_n

    // results, written by the launch's last block
    double* out;           // device memory or pinned host memory
    int want_sums;         // 1: raw sums, 0: price / delta / stderr / vega
    double inv_paths;      // 1 / n_paths
    double var_scale;      // n_paths / (n_paths - 1) (0 for one path)
    double inv_delta;      // 1 / (n_paths S0)

    // per-path outputs and near-node decision log (debug entry point only;
    // dbg_xN != null selects the logging instantiation)
    float* dbg_xN;
    float* dbg_V;
    float* dbg_xbar0;
    int* dbg_ev;                        // [dbg_ev_cap][3]: path - path_begin, step, 2 i + inside
    unsigned long long* dbg_ev_count;
    long long dbg_ev_cap;
    float dbg_band;                     // relative distance to a node that is logged
};

// Sets cell_mode, and for kCellBins the bins' scale, shift and count in place
// of the cells'; every other field is set. sig_max is the grid's largest sigma.
__host__ __device__ inline void choose_cell_mode(McParams& P, double sig_max, int n_bins, bool bins_two,
                                                 float bin_scale, float bin_shift)
{
    const bool on_s = (P.model & 2) != 0;
    P.cell_mode = kCellSearch;
    P.n_bins = 0;
    if (P.log_uniform) {
        if (index_bounded(on_s, P.N, P.x0, P.rdt, P.hdt, P.sqdt2, sig_max, P.cell_scale, P.cell_shift))
            P.cell_mode = kCellUniform;
    } else if (n_bins > 0 &&
               index_bounded(on_s, P.N, P.x0, P.rdt, P.hdt, P.sqdt2, sig_max, bin_scale, bin_shift)) {
        if (bins_two) P.cell_mode = kCellBins;
        P.n_bins = n_bins;
        P.cell_scale = bin_scale;
        P.cell_shift = bin_shift;
    }
}

// McParams::method of the second-order bucket kernel (besides LV_ADJ_REVERSE
// and LV_ADJ_TANGENT of lv.h).
constexpr int kMethodVanna = 2;

struct FinalizeParams {
    const double* partials;
    int G;                 // rows
    int row_words;
    int I, J;
    long long n_paths;
    double S0;
    double* chunks;        // [finalize_chunks(G)][row_words] stage-1 sums
    double* out;           // [3 + I * J]
    unsigned int* tile_counter;  // reset to 0
    unsigned int* flag;          // nonzero: every output NaN; reset to 0 (may be null)
};

int finalize_chunks(int G);
cudaError_t launch_finalize_sums(const double* sums, int IJ, long long n_paths, double S0, double* out,
                                 cudaStream_t s);

// Batched central bump-and-reprice (lv_bump.cu).
struct BumpParams {
    McParams mc;           // grid, option, random numbers, path tiles, tile counter
    int n_scen;            // 3 + 2 I J
    int n_groups;          // ceil(n_scen / slots per thread)
    float eps_half;        // eps / 2 on sigma
    float x0_up, x0_dn;    // ln(S0 + eps_S / 2), ln(S0 - eps_S / 2)
    double* partials;      // [gridDim.x][row_words] per-block binary64 rows
    int row_words;         // 2 + I J
};

size_t bump_smem_bytes(int I, int Je, int N, int row_words);
int bump_slots_per_thread();
int bump_chunks(int G);
cudaError_t bump_occupancy(int block, size_t smem, int* blocks_per_sm);
cudaError_t launch_bump(const BumpParams& b, int grid, int block, size_t smem, cudaStream_t s);
cudaError_t launch_bump_finalize(const double* partials, int G, int row_words, double* chunks, int IJ,
                                 long long n_paths, double eps, double eps_S, double* out,
                                 unsigned int* tile_counter, cudaStream_t s);

size_t mc_smem_bytes(int I, int J, int N, int n_bins, int block, bool greeks, bool grid_smem, bool extra = false,
                     int ppl = 1);

// Binary64 paths (lv_fp64.cu): the full-FP64 reference adjoint and the
// binary64 bump baseline, main reading only.
struct F64Params {
    const double* spot;    // [I] spot nodes, then [I] inverse gaps 1 / (s_{i+1} - s_i) (0 where infinite)
    bool divide;           // adjoint: some inverse gap is 0
    const double* sig;     // [I * J] sigma, spot-major (as the ABI takes it)
    const double* tau;     // [J] time nodes
    int I, J, N;
    double x0, x0_up, x0_dn;   // ln S0, ln(S0 +- eps_S / 2)
    double r, dt, sqdt, K, disc, phi, eps_half;
    uint32_t k0, k1, stream_id;
    long long path_begin, n_paths;
    double* partials;      // [gridDim.x][row_words]: adjoint 3 + Je I (time-major), bump 2 + I J
    int row_words;
    unsigned int* flag;    // adjoint: live paths with a vanishing 1 + g_n
    double2* tape_hf;      // adjoint, [N][threads]: (h_n, 1 + g_n)
    double* tape_u;        // [N][threads]: spot weight
    int* tape_k;           // [N][threads]: bucket of the cell's lower node
    int n_scen, n_groups;  // bump: 3 + 2 I J scenarios in groups of bump64_slots_per_thread()
};

size_t adjoint64_smem_bytes(int N);
size_t bump64_smem_bytes(int N, int row_words);
int bump64_slots_per_thread();
cudaError_t f64_occupancy(bool bump, size_t smem, int* blocks_per_sm);
cudaError_t launch_adjoint64(const F64Params& P, int grid, int block, size_t smem, cudaStream_t s);
int adjoint64_block();                    // most threads per block
size_t adjoint64_tape_bytes(int N);       // per thread
cudaError_t launch_bump64(const F64Params& P, int grid, size_t smem, cudaStream_t s);

// Pipe-rate probes (lv_probe.cu): out[LV_PIPE_COUNT] operations per second.
cudaError_t measure_pipe_peaks(double* out);

// Test-facing kernels (lv_debug.cu): Philox words and normals for listed
// (path, block) counters; the per-step time table of a call.
cudaError_t launch_debug_normals(uint64_t seed, uint32_t stream_id, const long long* paths, const uint32_t* blocks,
                                 long long n, uint32_t* words, float* z, cudaStream_t s);
cudaError_t launch_debug_time_table(const McParams& P, int* out_j, float* out_v, cudaStream_t s);

// Launchers; return cudaSuccess or the launch error. An adjoint launch with
// p.dbg_xN != null runs the logging instantiation with k = 4 and binary64
// level 2 whatever k and p.acc_mode say: plan its scratch with k = 4.
cudaError_t launch_mc(const McParams& p, int grid, int block, int k, bool greeks, size_t smem,
                      cudaStream_t s);
cudaError_t launch_finalize(const FinalizeParams& f, cudaStream_t s);
cudaError_t mc_occupancy(int block, int k, bool greeks, int acc, bool dbg, bool grid_smem, int method, int model,
                         int cell, bool extra, size_t smem, int* blocks_per_sm, int ppl = 1);

// One translation unit per model and cell mode (lv_m<model>c<cell>.cu, so that
// they compile in parallel). Models 1 to 3 exist for checkpoint intervals k = 4
// and 8, model 0 also for 16 and 32 (kCellSearch only), at one or two paths per
// lane; the logging kernels are kCellSearch.
#define LV_DECLARE_KERNELS(M, C)                                                                             \
    cudaError_t launch_mc_m##M##c##C(const McParams& p, int grid, int block, int k, bool greeks, size_t smem, \
                                     cudaStream_t s);                                                        \
    cudaError_t mc_occupancy_m##M##c##C(int block, int k, bool greeks, int acc, bool dbg, bool grid_smem,    \
                                        int method, bool extra, size_t smem, int* blocks_per_sm, int ppl);
#define LV_DECLARE_MODEL(M) LV_DECLARE_KERNELS(M, 0) LV_DECLARE_KERNELS(M, 1) LV_DECLARE_KERNELS(M, 2)
LV_DECLARE_MODEL(0)
LV_DECLARE_MODEL(1)
LV_DECLARE_MODEL(2)
LV_DECLARE_MODEL(3)
#undef LV_DECLARE_MODEL
#undef LV_DECLARE_KERNELS
constexpr int kModelMaxK = 8;
constexpr int kWideBlock = 512;    // threads of a block that has an SM to itself (adjoint_kernel WIDE)
int ring_slots_per_warp();
int paths_per_tile(bool greeks, int ppl);   // paths of a tile (the adjoint claims ppl tiles at a time)

}  // namespace lv

// Book of options (lv_book.cu): device tables and launch parameters.
namespace lv {

struct BookSurf {
    int I, J, Je, log_uniform;
    float cell_scale, cell_shift, s_lo, s_hi;
    double sig_max;                                  // largest sigma of the grid (index_bounded)
    int n_bins, bins_two;
    float bin_scale, bin_shift;
    long long off_bins;
    long long off_sig2, off_node, off_ab, off_tau;   // offsets into the book's grid arrays
    long long risk_off;                              // first double of this surface's aggregated risk
};

struct BookInst {
    int surf, N, phi, stream_id;
    double K, T;
    long long n_paths;
    long long out_off;                               // first double of this option's sums / outputs
    double w;                                        // position weight (aggregated risk)
    double scale;                                    // w / n_paths
};

struct BookItem {
    int inst, first_tile, n_tiles;                    // tiles of 32 paths
};

struct BookRun {
    double log2_S0, r;
    unsigned long long seed;
};

struct BookParams {
    const BookSurf* surfs;
    const BookInst* insts;
    const BookItem* items;
    int n_items;
    const float2* sig2;
    const float* node;
    const float2* ab;
    const double* tau;
    const float4* bins;
    const BookRun* run;
    unsigned int* item_counter;
    double* sums;          // per option [3 + I J] binary64 sums (zeroed before a run)
    double* risk;          // aggregated runs: per surface [3 + I J], the vega part summed with
                           // weights w / n_paths (zeroed before a run); null: per-option vegas
    float* l1;             // [gridDim.x][max_IJe] binary32 node buckets per block
    float* ckpt;           // [ceil(max_N / k)][gridDim.x * warps * ring slots]
    int max_I, max_Je, max_N, max_IJe, max_bins;
};

// ppl: paths per lane of the forward tiles (1 or 2); the FIFO and the
// checkpoint ring (book_ring_slots_per_warp() * ppl per warp) grow with it.
// Most shared memory of a book's block: 200 KB, and beside them the 144 bytes of the
// option's Philox round keys and output scales, which took no room from the grids.
constexpr size_t kBookSmem = 200 * 1024 + 144;
size_t book_smem_bytes(int maxI, int maxJe, int maxN, int max_bins, int block, int ppl);
int book_ring_slots_per_warp();
cudaError_t book_prepare(int k, int ppl, bool bins);
cudaError_t book_occupancy(int block, int k, int ppl, bool bins, size_t smem, int* blocks_per_sm);
cudaError_t launch_book(const BookParams& b, int grid, int block, int k, int ppl, size_t smem, cudaStream_t s);
cudaError_t launch_book_finalize(const BookParams& b, int n_inst, int max_IJ, double* out, cudaStream_t s);
cudaError_t launch_book_risk_finalize(const BookParams& b, int n_surf, int n_inst, int max_IJ, double* out,
                                      cudaStream_t s);

}  // namespace lv

#include <string>

#include "lv.h"

namespace lv {
// Records the thread-local message lv_last_error() returns; returns s.
lv_status set_error(lv_status s, const std::string& msg);

// Launch-shape cache shared by the autotuners: lines "key v0 v1 v2 v3 ms" in
// the file named by LV_TUNE_CACHE (the last line of a key wins).
bool tune_cache_lookup(const std::string& key, int vals[4]);
void tune_cache_append(const std::string& key, const int vals[4], double ms);
std::string gpu_name(int device);
}  // namespace lv

// Surface handle (host side; shared by the runtime's source files).
struct lv_surface_s {
    int device = 0;
    int num_sms = 0;
    int adj_method = 0;              // LV_ADJ_REVERSE or LV_ADJ_TANGENT
    int interp = 0;                  // LV_INTERP_S or LV_INTERP_LOGS
    int scheme = 0;                  // LV_SCHEME_LOG or LV_SCHEME_S
    int I = 0, J = 0, Je = 0;
    std::vector<double> spot, time;
    float2* d_sig = nullptr;         // [Je][I-1] pairs (sigma_{i,j}, sigma_{i+1,j} - sigma_{i,j})
    float* d_node = nullptr;
    float2* d_ab = nullptr;
    float2* d_abl = nullptr;         // [I] cell coefficients of the ln-S weight, in y = log2 S (behind the bins)
    double* d_tau = nullptr;
    double* d_spot64 = nullptr;      // [I] spot nodes, then [I] inverse gaps, binary64 (the binary64 kernels)
    bool gap_divide = false;         // some gap has no inverse (0 in d_spot64)
    double* d_sig64 = nullptr;       // [I * J] sigma, binary64, spot-major
    double* h_sig64_stage = nullptr; // pinned staging for its uploads
    bool sig64_stale = false;        // d_sig64 behind h_sig64_stage: uploaded by the binary64 calls
    float2* h_sig_stage = nullptr;   // pinned staging for sigma uploads
    int log_uniform = 0;
    double sig_max = 0.0;            // largest sigma of the grid (index_bounded)
    float4* d_bins = nullptr;        // [n_bins] cell table of a grid not log-uniform (lv_api.cu spot_bins)
    bool bins_two = false;           // no bin has more than two nodes
    int n_bins = 0;
    float bin_scale = 0.0f, bin_shift = 0.0f;
    float cell_scale = 0.0f, cell_shift = 0.0f, s_lo = 0.0f, s_hi = 0.0f;
    int phi = 1;
    cudaStream_t stream = nullptr;
    int acc_mode = LV_ACC_FP64;
    int cfg_block = 0, cfg_k = 0, cfg_bps = 0, cfg_ppl = 0;
    void* d_scratch = nullptr;
    size_t scratch_bytes = 0;
    double* d_res = nullptr;         // [3 + I*J] result of the host-output calls
    double* h_res = nullptr;         // pinned copy of it
    cudaEvent_t ev_start = nullptr;  // optional events around the Monte Carlo kernel
    cudaEvent_t ev_end = nullptr;
};
