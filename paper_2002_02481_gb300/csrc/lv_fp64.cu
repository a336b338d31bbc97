// lv_fp64.cu -- the same Monte Carlo estimators with every path in binary64
// (arXiv 2002.02481, Sec. III, IV-A..IV-D), main reading only: log-Euler,
// bilinear sigma linear in S and t. Two kernels:
//
//  - adjoint64_kernel: price, delta and every vega bucket, the reference the
//    binary32 kernels' rounding is measured against on the GPU. One path per
//    thread: forward with a tape, then x_bar_n = x_bar_{n+1} (1 + g_n), g_n = h_n S_n
//    d sigma / d S, h_n = sqrt(dt) Z_n - sigma_n dt, back over it; sigma_bar_n =
//    x_bar_{n+1} h_n spread over the cell's corners with the bilinear weights,
//    run-length sums in registers, binary64 reductions into the block's row.
//  - bump64_kernel: central bump-and-reprice (Sec. III) with binary64 paths,
//    scenario for scenario as the binary32 bump kernel (lv_bump.cu).
//
// The bump kernel's arithmetic follows the FP64 definition step by step with CUDA's
// binary64 functions; the adjoint's takes fewer operations to the same accuracy
// (below). Binary64 runs at a small fraction of the binary32 rate on this part:
// these kernels are references, not the product path.
#include <math.h>

#include "lv_device.cuh"

namespace lv {

namespace {

// Four binary64 normals of Philox block blk: the same words as normals4,
// u = ((w >> 9) + 1/2) 2^-23 (exact), Z_a = sqrt(-2 ln u_a) cos(2 pi u_b),
// Z_b = sqrt(-2 ln u_a) sin(2 pi u_b).
__device__ __forceinline__ void normals4_f64(uint32_t blk, uint32_t c1, uint32_t c2, uint32_t k0, uint32_t k1,
                                             double z[4])
{
    uint32_t w[4] = { blk, c1, c2, 0u };
    philox4x32_10(w[0], w[1], w[2], w[3], philox_keys(k0, k1));
#pragma unroll
    for (int pair = 0; pair < 2; ++pair) {
        const double ua = ((double)(w[2 * pair] >> 9) + 0.5) * 0x1p-23;
        const double ub = ((double)(w[2 * pair + 1] >> 9) + 0.5) * 0x1p-23;
        const double rho = sqrt(-2.0 * log(ua));
        double s, c;
        sincospi(2.0 * ub, &s, &c);
        z[2 * pair] = rho * c;
        z[2 * pair + 1] = rho * s;
    }
}

struct Pt64 {
    int i;
    double u, sigma, dsdS;
};

// Bilinear sigma at (S, time cell j, weight v) and d sigma / d S (0 outside
// [s_0, s_{I-1}]); cell i = the largest i <= I-2 with s_i <= S.
__device__ __forceinline__ Pt64 sigma64(const F64Params& P, double S, int j, double v)
{
    int lo = 0, hi = P.I - 2;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.spot[mid] <= S) lo = mid;
        else hi = mid - 1;
    }
    const int i = lo;
    const double lo_s = P.spot[i], hi_s = P.spot[i + 1];
    double u;
    if (S <= lo_s) u = 0.0;
    else if (S >= hi_s) u = 1.0;
    else u = (S - lo_s) / (hi_s - lo_s);
    const int J = P.J;
    const double s00 = P.sig[i * J + j];
    const double s10 = P.sig[(i + 1) * J + j];
    const double s01 = J > 1 ? P.sig[i * J + j + 1] : 0.0;
    const double s11 = J > 1 ? P.sig[(i + 1) * J + j + 1] : 0.0;
    Pt64 p;
    p.i = i;
    p.u = u;
    const double w0 = (1.0 - u) * (1.0 - v), w1 = u * (1.0 - v), w2 = (1.0 - u) * v, w3 = u * v;
    p.sigma = w0 * s00 + w1 * s10 + w2 * s01 + w3 * s11;
    const bool inside = S >= P.spot[0] && S <= P.spot[P.I - 1];
    p.dsdS = inside ? ((1.0 - v) * (s10 - s00) + v * (s11 - s01)) / (hi_s - lo_s) : 0.0;
    return p;
}

// Time cell and weight of every step (t_n = n dt), in shared memory.
__device__ __forceinline__ void stage_time64(const F64Params& P, int2* s_j, double* s_v)
{
    for (int n = threadIdx.x; n < P.N; n += blockDim.x) {
        const double t = (double)n * P.dt;
        int j = 0;
        double v = 0.0;
        if (P.J > 1) {
            int lo = 0, hi = P.J - 2;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (P.tau[mid] <= t) lo = mid;
                else hi = mid - 1;
            }
            j = lo;
            v = (t - P.tau[j]) / (P.tau[j + 1] - P.tau[j]);
            v = v < 0.0 ? 0.0 : (v > 1.0 ? 1.0 : v);
        }
        s_j[n] = make_int2(j, j * P.I);
        s_v[n] = v;
    }
}

__device__ __forceinline__ void path_words(const F64Params& P, long long rel, uint32_t& c1, uint32_t& c2)
{
    const unsigned long long p = (unsigned long long)(P.path_begin + rel);
    c1 = (uint32_t)p;
    c2 = ((uint32_t)(p >> 32) & 0xffffu) | (P.stream_id << 16);
}

__device__ __forceinline__ void flush64(double* row, int key, int I, double A, double AU, double Bs, double BU)
{
    atomicAdd(row + key, A - AU);
    atomicAdd(row + key + 1, AU);
    atomicAdd(row + key + I, Bs - BU);
    atomicAdd(row + key + I + 1, BU);
}

constexpr double kTiny64 = 0x1p-40;    // |1 + g_n| below this on a live path: the estimate is refused

// ---- binary64 functions of the adjoint kernel, table-driven (P. T. P. Tang,
// "Table-driven implementation of the exponential function", ACM TOMS 15,
// 1989, and "... of the logarithm function", ACM TOMS 16, 1990): a table entry
// and a short polynomial of the residual. The kernel is bound by the binary64
// pipe (1.7 operations per SM and cycle), and these take 10 operations for an
// exponential, 9 for a logarithm and 14 for a sine and a cosine; integer
// instructions do what they can of the rest. The tables come from CUDA's own
// functions, once per block.
constexpr int kTab = 256;

struct Tab64 {
    const double* ex;      // [256] 2^(i / 256)
    const double2* lg;     // [256] (1 / c_i in 13 bits, -ln of that; less ln 2 in the upper half of the octave)
    const double2* cs;     // [256] (cos, sin) of 2 pi (i + 1/2) / 256
    const double* eln2;    // [25] -e ln 2
};

constexpr int kLogSplit = 106;         // 1 + 106 / 256: above sqrt 2 the octave's upper half counts down from 2

__device__ __forceinline__ double log_inv(int i)
{
    // the interval [1 + i / 256, 1 + (i + 1) / 256): its ends at 1 and 2 are exact, so that
    // ln u keeps its relative accuracy at u = 1
    if (i == 0) return 1.0;
    if (i == kTab - 1) return 0.5;
    return rint(4096.0 / (1.0 + (i + 0.5) / 256.0)) / 4096.0;
}

__device__ __forceinline__ void fill_tables(double* ex, double2* lg, double2* cs, double* eln2)
{
    for (int i = threadIdx.x; i < kTab; i += blockDim.x) {
        ex[i] = exp2((double)i / 256.0);
        const double inv = log_inv(i);
        lg[i] = make_double2(inv, i == 0 || i == kTab - 1 ? 0.0
                                  : i >= kLogSplit       ? -log(2.0 * inv)       // -ln inv - ln 2
                                                         : -log(inv));
        double s, c;
        sincospi(2.0 * (i + 0.5) / 256.0, &s, &c);
        cs[i] = make_double2(c, s);
    }
    for (int e = threadIdx.x; e < 25; e += blockDim.x) eln2[e] = -(double)e * 0x1.62e42fefa39efp-1;
}

// e^x for |x| <= 700 (else CUDA's): x = n ln 2 / 256 + r, |r| < 0.00136.
__device__ __forceinline__ double exp64(const Tab64& T, double x)
{
    if ((__double2hiint(x) & 0x7fffffff) > 0x4085e000) return exp(x);
    const double t = fma(x, 369.3299304675746, 0x1.8p52);
    const int n = __double2loint(t);
    const double nd = t - 0x1.8p52;
    double r = fma(nd, -0x1.62e42fcp-9, x);          // ln 2 / 256, high part (27 bits: the product is exact)
    r = fma(nd, -0x1.7d1cf79abc9e4p-36, r);          // low part
    const double q = fma(fma(r, 1.0 / 24.0, 1.0 / 6.0), r, 0.5);
    const double p = fma(q, r * r, r);               // e^r - 1
    const double y = T.ex[n & (kTab - 1)];
    const double v = fma(y, p, y);
    return __hiloint2double(__double2hiint(v) + ((n >> 8) << 20), __double2loint(v));
}

// ln((2 m + 1) 2^-24), m < 2^23: the 24-bit integer normalised to f in [1, 2) by
// integer instructions, f / c - 1 exact, |r| <= 2^-8.
__device__ __forceinline__ double log_unit(const Tab64& T, uint32_t m)
{
    const float w = (float)(2u * m + 1u);            // exact
    const uint32_t b = __float_as_uint(w);
    const int i = (b >> 15) & (kTab - 1);
    const int e = 24 - ((int)(b >> 23) - 127) - (i >= kLogSplit ? 1 : 0);       // u = f 2^-(e + [upper half])
    const double f = __hiloint2double(0x3ff00000 | ((b & 0x7fffffu) >> 3), (b & 7u) << 29);
    const double2 c = T.lg[i];
    const double r = fma(f, c.x, -1.0);
    const double r2 = r * r;
    const double q = fma(fma(fma(fma(r, -1.0 / 6.0, 0.2), r, -0.25), r, 1.0 / 3.0), r, -0.5);
    return (T.eln2[e] + c.y) + fma(q, r2, r);
}

// sqrt(y), y in [1e-8, 40]: a binary32 inverse root refined twice.
__device__ __forceinline__ double sqrt_pos(double y)
{
    const double s = (double)rsqrtf((float)y);
    double g = y * s, h = 0.5 * s;
    double e = fma(-g, h, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    return fma(fma(-g, g, y), h, g);
}

// (cos, sin) of 2 pi (2 m + 1) 2^-24, m < 2^23.
__device__ __forceinline__ double2 cossin_unit(const Tab64& T, uint32_t m)
{
    const double2 a = T.cs[m >> 15];
    const int k = 2 * (int)(m & 0x7fffu) + 1 - 0x8000;                 // residual in 2^-24 turns
    const double d = __hiloint2double(0x43300000, 0x40000000 + k) - __hiloint2double(0x43300000, 0x40000000);
    const double t = d * 0x1.921fb54442d18p-22;                        // |t| < 0.0123
    const double t2 = t * t;
    const double ps = fma(fma(t2, -1.0 / 5040.0, 1.0 / 120.0), t2, -1.0 / 6.0);
    const double pc = fma(fma(t2, -1.0 / 720.0, 1.0 / 24.0), t2, -0.5);
    const double s = fma(t * t2, ps, t), c1 = t2 * pc;                 // sin t, cos t - 1
    return make_double2(fma(a.x, c1, fma(-a.y, s, a.x)), fma(a.y, c1, fma(a.x, s, a.y)));
}

// The normals of normals4_f64 from the tables.
__device__ __forceinline__ void normals4_tab(const Tab64& T, const PhiloxKeys& K, uint32_t blk, uint32_t c1,
                                             uint32_t c2, double z[4])
{
    uint32_t w[4] = { blk, c1, c2, 0u };
    philox4x32_10(w[0], w[1], w[2], w[3], K);
#pragma unroll
    for (int pair = 0; pair < 2; ++pair) {
        const double rho = sqrt_pos(-2.0 * log_unit(T, w[2 * pair] >> 9));
        const double2 c = cossin_unit(T, w[2 * pair + 1] >> 9);
        z[2 * pair] = rho * c.x;
        z[2 * pair + 1] = rho * c.y;
    }
}

struct Smem64 {
    size_t j, v, ex, lg, cs, eln2, xb, list, total;
};

constexpr int kBlock64 = 512;

__host__ __device__ inline Smem64 smem64(int N)
{
    Smem64 L;
    size_t o = 0;
    L.j = o;    o += (sizeof(int2) * (size_t)N + 15) & ~size_t(15);
    L.v = o;    o += sizeof(double) * (size_t)((N + 1) & ~1);
    L.ex = o;   o += sizeof(double) * kTab;
    L.lg = o;   o += sizeof(double2) * kTab;
    L.cs = o;   o += sizeof(double2) * kTab;
    L.eln2 = o; o += sizeof(double) * 26;
    L.xb = o;   o += sizeof(double) * kBlock64;
    L.list = o; o += sizeof(int) * kBlock64;
    L.total = o;
    return L;
}

// Price, delta and vegas with binary64 paths, one path per thread: the forward
// pass leaves (h_n, 1 + g_n, u_n, bucket) of every step on a tape in global memory
// (28 bytes a step, the block's threads side by side); the block then packs its
// live paths onto its first threads, which walk their tapes back: sigma_bar_n =
// x_bar_{n+1} h_n, x_bar_n = x_bar_{n+1} (1 + g_n). Bound by the binary64 pipe: about
// 50 operations per path-step where two forward passes with CUDA's functions, two
// divisions a step and a search by binary64 comparisons took 226. 30 x 60 grid, 156
// steps, 2^16 paths: 5.08 -> 1.05 ms; 2^18 paths 26.8 -> 4.7 ms.
// DIVIDE: some spot gap has no inverse (below 2^-1024), and its cell divides. Both in
// one kernel took 1,097 us instead of 1,056 at 2^16 paths.
template <bool DIVIDE>
__global__ void __launch_bounds__(kBlock64, 1) adjoint64_kernel(const __grid_constant__ F64Params P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_live;
    const Smem64 L = smem64(P.N);
    int2* s_j = reinterpret_cast<int2*>(smem + L.j);
    double* s_v = reinterpret_cast<double*>(smem + L.v);
    double* s_xb = reinterpret_cast<double*>(smem + L.xb);
    int* s_list = reinterpret_cast<int*>(smem + L.list);
    const int tid = threadIdx.x, B = blockDim.x;
    double* row = P.partials + (size_t)blockIdx.x * P.row_words;
    for (int e = tid; e < P.row_words; e += B) row[e] = 0.0;
    fill_tables(reinterpret_cast<double*>(smem + L.ex), reinterpret_cast<double2*>(smem + L.lg),
                reinterpret_cast<double2*>(smem + L.cs), reinterpret_cast<double*>(smem + L.eln2));
    stage_time64(P, s_j, s_v);
    if (tid == 0) s_live = 0;
    __syncthreads();
    const Tab64 T{ reinterpret_cast<const double*>(smem + L.ex), reinterpret_cast<const double2*>(smem + L.lg),
                   reinterpret_cast<const double2*>(smem + L.cs), reinterpret_cast<const double*>(smem + L.eln2) };
    const PhiloxKeys K = philox_keys(P.k0, P.k1);
    const double* gap = P.spot + P.I;                // 1 / (s_{i+1} - s_i), 0 where that overflows
    const size_t threads = (size_t)gridDim.x * B;    // tape stride of a step
    const size_t col0 = (size_t)blockIdx.x * B;
    double2* const t_hf = P.tape_hf + col0;
    double* const t_u = P.tape_u + col0;
    int* const t_k = P.tape_k + col0;
    double* vrow = row + 3;                          // time-major buckets j I + i
    const int I = P.I, J = P.J;
    const long long s_first = __double_as_longlong(P.spot[0]), s_last = __double_as_longlong(P.spot[I - 1]);
    double sV = 0.0, sV2 = 0.0, sX = 0.0;
    for (long long base = (long long)blockIdx.x * B; base < P.n_paths; base += (long long)gridDim.x * B) {
        const long long rel = base + tid;
        if (rel < P.n_paths) {
            uint32_t c1, c2;
            path_words(P, rel, c1, c2);
            double z[4], x = P.x0;
            bool tiny = false;
            for (int n = 0; n < P.N; ++n) {
                if ((n & 3) == 0) normals4_tab(T, K, (uint32_t)(n >> 2), c1, c2, z);
                const double S = exp64(T, x);
                const int2 jr = s_j[n];
                const double v = s_v[n];
                // cell: the largest i <= I-2 with s_i <= S (positive binary64 numbers order like their bits)
                const long long sb = __double_as_longlong(S);
                int i = 0, hi = I - 2;
                while (i < hi) {
                    const int mid = (i + hi + 1) >> 1;
                    if (__double_as_longlong(__ldg(P.spot + mid)) <= sb) i = mid;
                    else hi = mid - 1;
                }
                const double inv = __ldg(gap + i);
                double u = (S - __ldg(P.spot + i)) * inv;
                if (DIVIDE && inv == 0.0) u = (S - __ldg(P.spot + i)) / (__ldg(P.spot + i + 1) - __ldg(P.spot + i));
                if (__double_as_longlong(u) < 0) u = 0.0;                                   // below the grid
                else if (__double_as_longlong(u) > 0x3ff0000000000000ll) u = 1.0;           // above it
                const double* q = P.sig + i * J + jr.x;
                const double s00 = __ldg(q), s10 = __ldg(q + J);
                double top = s10 - s00, sigma, ds;
                if (J > 1) {
                    const double s01 = __ldg(q + 1), d1 = __ldg(q + J + 1) - s01;
                    ds = fma(v, d1 - top, top);
                    top = fma(u, top, s00);
                    sigma = fma(v, fma(u, d1, s01) - top, top);
                } else {
                    ds = top;
                    sigma = fma(u, top, s00);
                }
                const bool inside = sb >= s_first && sb <= s_last;
                const double h = fma(P.sqdt, z[n & 3], -sigma * P.dt);
                double slope = ds * inv;
                if (DIVIDE && inv == 0.0) slope = ds / (__ldg(P.spot + i + 1) - __ldg(P.spot + i));
                const double f = inside ? fma(h, S * slope, 1.0) : 1.0;
                tiny = tiny || (__double2hiint(f) & 0x7fffffff) < 0x3d700000;               // |f| < 2^-40
                const size_t at = (size_t)n * threads + tid;
                t_hf[at] = make_double2(h, f);
                t_u[at] = u;
                t_k[at] = jr.y + i;
                // the definition's order: one rounding of x for the drift, one for the noise
                x = fma(sigma * P.sqdt, z[n & 3], fma(fma(-0.5 * sigma, sigma, P.r), P.dt, x));
            }
            const double SN = exp64(T, x);
            const double itm = P.phi * (SN - P.K);
            const double V = itm > 0.0 ? P.disc * itm : 0.0;
            sV += V;
            sV2 = fma(V, V, sV2);
            if (itm > 0.0 && SN > 0.0) {
                if (tiny) {
                    atomicAdd(P.flag, 1u);
                } else {
                    const int at = atomicAdd(&s_live, 1);
                    s_list[at] = tid;
                    s_xb[at] = P.disc * P.phi * SN;
                }
            }
        }
        __syncthreads();
        const int live = s_live;
        if (tid < live) {
            const int col = s_list[tid];
            double xbar = s_xb[tid];
            int cur = -1;
            double A = 0.0, AU = 0.0, Bs = 0.0, BU = 0.0;
            for (int n0 = P.N - 1; n0 >= 0; n0 -= 4) {
                double2 hf[4];
                double u[4];
                int key[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const size_t at = (size_t)max(n0 - q, 0) * threads + col;
                    hf[q] = t_hf[at];
                    u[q] = t_u[at];
                    key[q] = t_k[at];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (n0 - q < 0) break;
                    const double sbar = xbar * hf[q].x;
                    xbar *= hf[q].y;
                    if (key[q] != cur) {
                        if (cur >= 0) flush64(vrow, cur, I, A, AU, Bs, BU);
                        A = AU = Bs = BU = 0.0;
                        cur = key[q];
                    }
                    const double b = sbar * s_v[n0 - q];
                    const double a = sbar - b;
                    A += a;
                    AU = fma(a, u[q], AU);
                    Bs += b;
                    BU = fma(b, u[q], BU);
                }
            }
            if (cur >= 0) flush64(vrow, cur, I, A, AU, Bs, BU);
            sX += xbar;
        }
        __syncthreads();                  // the tapes and the list are read
        if (tid == 0) s_live = 0;
        __syncthreads();
    }
    // block sums of the scalars
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sV += __shfl_down_sync(0xffffffffu, sV, o);
        sV2 += __shfl_down_sync(0xffffffffu, sV2, o);
        sX += __shfl_down_sync(0xffffffffu, sX, o);
    }
    if ((tid & 31) == 0) {
        atomicAdd(&row[0], sV);
        atomicAdd(&row[1], sV2);
        atomicAdd(&row[2], sX);
    }
}

constexpr int kM64 = 8;   // scenario slots per thread (even: pairs never split)

// Scenario s of 3 + 2 I J as in lv_bump.cu: s = 0, 1 S0 +- eps_S/2; s = 2 + 2e + b
// node e = i J + j at sigma_e + eps/2 (b = 0) or - eps/2 (b = 1); the last one
// unbumped. Each thread prices one path under kM64 consecutive scenarios on the
// same normals; pair differences go to slot s / 2 of the block's row.
__global__ void __launch_bounds__(128) bump64_kernel(const __grid_constant__ F64Params P)
{
    extern __shared__ __align__(16) unsigned char smem[];
    int2* s_j = reinterpret_cast<int2*>(smem);
    double* s_v = reinterpret_cast<double*>(smem + ((sizeof(int2) * (size_t)P.N + 15) & ~size_t(15)));
    double* s_acc = s_v + ((P.N + 1) & ~1);
    for (int e = threadIdx.x; e < P.row_words; e += blockDim.x) s_acc[e] = 0.0;
    stage_time64(P, s_j, s_v);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long n_tiles = (P.n_paths + blockDim.x - 1) / blockDim.x;
    const long long n_items = n_tiles * P.n_groups;
    for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {     // block-uniform
        const int grp = (int)(item % P.n_groups);
        const long long rel = (item / P.n_groups) * blockDim.x + threadIdx.x;
        const int s_first = grp * kM64;
        double x[kM64], V[kM64], bh[kM64];
        int be[kM64];
#pragma unroll
        for (int k = 0; k < kM64; ++k) {
            const int s = s_first + k;
            x[k] = s == 0 ? P.x0_up : (s == 1 ? P.x0_dn : P.x0);
            be[k] = (s >= 2 && s < P.n_scen - 1) ? (s - 2) >> 1 : -1;
            bh[k] = ((s - 2) & 1) ? -P.eps_half : P.eps_half;
            V[k] = 0.0;
        }
        if (rel < P.n_paths) {
            uint32_t c1, c2;
            path_words(P, rel, c1, c2);
            double z[4];
            for (int n = 0; n < P.N; ++n) {
                if ((n & 3) == 0) normals4_f64((uint32_t)(n >> 2), c1, c2, P.k0, P.k1, z);
                const int j = s_j[n].x;
                const double v = s_v[n];
#pragma unroll
                for (int k = 0; k < kM64; ++k) {
                    if (s_first + k >= P.n_scen) continue;
                    const double S = exp(x[k]);
                    const Pt64 pt = sigma64(P, S, j, v);
                    double sig = pt.sigma;
                    if (be[k] >= 0) {       // + or - eps/2 times the bumped node's bilinear weight
                        const int bi = be[k] / P.J, bj = be[k] - bi * P.J;
                        const double ws = bi == pt.i ? 1.0 - pt.u : (bi == pt.i + 1 ? pt.u : 0.0);
                        const double wt = bj == j ? 1.0 - v : (P.J > 1 && bj == j + 1 ? v : 0.0);
                        sig += bh[k] * (ws * wt);
                    }
                    x[k] = x[k] + (P.r - 0.5 * sig * sig) * P.dt + sig * P.sqdt * z[n & 3];
                }
            }
#pragma unroll
            for (int k = 0; k < kM64; ++k) {
                const double itm = P.phi * (exp(x[k]) - P.K);
                V[k] = itm > 0.0 ? P.disc * itm : 0.0;
            }
        }
#pragma unroll
        for (int k = 0; k < kM64; k += 2) {
            const int s = s_first + k;
            if (s < P.n_scen) {
                double d = (s + 1 < P.n_scen) ? V[k] - V[k + 1] : V[k];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
                if (lane == 0) atomicAdd(&s_acc[s >> 1], d);
            }
        }
    }
    __syncthreads();
    double* row = P.partials + (size_t)blockIdx.x * P.row_words;
    for (int e = threadIdx.x; e < P.row_words; e += blockDim.x) row[e] = s_acc[e];
}

size_t f64_time_bytes(int N) { return ((sizeof(int2) * (size_t)N + 15) & ~size_t(15)) + sizeof(double) * ((N + 1) & ~1); }

}  // namespace

size_t adjoint64_smem_bytes(int N) { return smem64(N).total; }
int adjoint64_block() { return kBlock64; }
size_t adjoint64_tape_bytes(int N) { return (sizeof(double2) + sizeof(double) + sizeof(int)) * (size_t)N; }
size_t bump64_smem_bytes(int N, int row_words) { return f64_time_bytes(N) + sizeof(double) * (size_t)row_words; }
int bump64_slots_per_thread() { return kM64; }

cudaError_t f64_occupancy(bool bump, size_t smem, int* bps)
{
    const void* k = bump ? (const void*)bump64_kernel : (const void*)adjoint64_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, k, bump ? 128 : kBlock64, smem);
}

cudaError_t launch_adjoint64(const F64Params& P, int grid, int block, size_t smem, cudaStream_t s)
{
    const auto kernel = P.divide ? adjoint64_kernel<true> : adjoint64_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    kernel<<<grid, block, smem, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_bump64(const F64Params& P, int grid, size_t smem, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(bump64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    bump64_kernel<<<grid, 128, smem, s>>>(P);
    return cudaGetLastError();
}

}  // namespace lv
