// Exact boson sampling by the algorithm the paper's CliffordClifford2017
// back-end implements (Sec. 3.2.3: "adapted Glynn algorithm to efficiently
// compute n simultaneous sub-permanents", O(n 2^n + m n^2) per sample).
//
// With A the m x n matrix of the input photons' columns of U (randomly
// permuted per sample), photon positions are drawn one at a time.  After
// r_1..r_{k-1} have been drawn, the next position i has weight
//     w_i = | sum_{l<k} A[i][l] Perm(A[r_1..r_{k-1}; {0..k-1} \ l]) |^2,
// the Laplace expansion along the new row of Perm(A[r_1..r_{k-1}, i; 0..k-1]).
// The k leave-one-column-out permanents come from one Glynn sum over the
// k-1 rows: with x_j(d) = sum_i d_i M[i][j] and leave-one-out products,
//     Perm(M_{-l}) = 2^{-(k-2)} sum_{d, d_1=+1} (prod d) prod_{j != l} x_j(d).
// The random numbers (column permutation, one uniform per photon) are inputs,
// so a sample is a deterministic function of them.
//
// Two forms of the sub-permanents:
//   subset_sampler_kernel  n <= 15: f_k(S) = Perm(A[r_1..r_k; S]) for every
//                          k-subset S of the n columns, level by level,
//                              f_k(S) = sum_{l in S} A[r_k][l] f_{k-1}(S \ l),
//                          so f_{k-1}({0..k-1} \ l) are the k sub-permanents
//                          of step k: n 2^{n-1} complex multiply-adds for the
//                          whole sample, 4 FP64 instructions each, where the
//                          Glynn sums of the steps take about 14 n 2^{n-1}
//                          (n = 14: 0.46 M against 1.6 M), and no sign
//                          cancellation.  From n = 10 on the levels are in
//                          fixed point on the integer pipe (16,384 samples of
//                          n = 14: 17.3 to 10.6 ms; the FP64 pipe took 12.5 of
//                          it), but for samples that need the range
//                          of FP64.  Two neighbouring levels live in
//                          shared memory (n = 14: 103 KB, two samples per SM;
//                          n = 15: 206 KB), which ends the form at n = 15;
//   sampler_kernel         n = 16: one Glynn sum per step (below), one warp
//                          per sample, lanes splitting the Gray-code sequence.
// Either way the m weights follow, then an inverse-CDF draw with a warp
// prefix sum.

#include <algorithm>

#include <cfloat>
#include <cmath>
#include <type_traits>

#include "fixed30.cuh"
#include "pcv_common.cuh"

namespace pcv {
namespace {

constexpr int kSampWarps = 4;

struct SampArgs {
    const double2* U;         // m x m
    int m, n;
    int cols[PCV_MAX_PHOTONS];
    const uint8_t* perm;      // [count][n] column permutation per sample
    const double* uni;        // [count][n] uniforms in [0, 1)
    int64_t count;
    uint8_t* out;             // [count][m] occupations
};

// Inverse-CDF draw by one warp from the weights of its lanes (wloc[c]: mode
// lane + 32 c; the cumulative order runs lane by lane), u in [0, 1); total: their sum.
__device__ int draw_mode(const double* wloc, int m, double u, double& total)
{
    const int lane = threadIdx.x & 31;
    double part = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) part += wloc[c];
    // total and lane prefix of the per-lane sums
    double incl = part;
    for (int off = 1; off < 32; off <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    const double target = u * total;
    // the lane whose cumulative range holds the target picks within its modes
    const double before = incl - part;
    int pick = -1;
    if (target >= before && target < incl) {
        double acc = before;
        int lastpos = -1;
        for (int c = 0; c < 4; ++c) {
            const int i = lane + 32 * c;
            if (i >= m) break;
            if (wloc[c] > 0.0) lastpos = i;
            acc += wloc[c];
            if (target < acc) { pick = i; break; }
        }
        if (pick < 0) pick = lastpos;          // rounding: this lane's last mode with weight
    }
    const unsigned ball = __ballot_sync(0xffffffffu, pick >= 0);
    if (ball) return __shfl_sync(0xffffffffu, pick, __ffs(ball) - 1);
    int last = -1;                             // rounding at the top end: last mode with weight
    for (int c = 3; c >= 0 && last < 0; --c) {
        const int i = lane + 32 * c;
        if (i < m && wloc[c] > 0.0) last = i;
    }
    for (int off = 16; off > 0; off >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, off));
    return last < 0 ? 0 : last;
}

// Entries of the even and odd levels 1 .. n-1 (C(n, k) at most).
__host__ __device__ inline int subset_level(int n, int odd)
{
    int c = 1, best = 1;
    for (int k = 1; k < n; ++k) {
        c = c * (n + 1 - k) / k;
        if ((k & 1) == odd && c > best) best = c;
    }
    return best;
}

// Shared memory of one sample: two levels, the drawn row, the sub-permanents of
// the step, the weights, the sample's columns, rows and column exponents.
__host__ __device__ inline size_t subset_bytes(int m, int n)
{
    return (size_t)(subset_level(n, 0) + subset_level(n, 1) + 2 * n) * sizeof(double2) +
           (size_t)(m + (m & 1)) * sizeof(double) + 48 * sizeof(int);      // a multiple of 16
}

constexpr int kBinom = 17;

// Position of the lowest bit (15 for none: a valid row of the tables).
__device__ __forceinline__ int low_bit(uint32_t x) { return (__ffs((int)x) - 1) & 15; }

// x 2^e on the integer pipe: 0 below 2^-959, x itself beyond 2^961.
__device__ __forceinline__ double times_pow2(double x, int e)
{
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7FF;
    if (ex < 64) return 0.0;
    return ex < 1984 ? __hiloint2double(hi + e * (1 << 20), __double2loint(x)) : x;
}

// |x| as a float but for its last three bits: 0 below FP32's range, infinity beyond.
__device__ __forceinline__ float abs_float(double x)
{
    const int hi = __double2hiint(x) & 0x7FFFFFFF;
    if (hi < 897 << 20) return 0.0f;
    return hi < 1151 << 20 ? __int_as_float((hi - (896 << 20)) << 3) : INFINITY;
}

// Shift of level k's sums for top 2^29 the largest component of level k - 1.
__device__ __forceinline__ int level_shift(float top, int k)
{
    return min(max(ilogbf(top * sqrtf(2.0f * k) * 1.0001f) - 2, 1), 30);
}

// One sample by a group of T threads, from the table c[t][j] = C(t, j).
//
// FIXED: the levels in fixed point (fixed30.cuh), components at most 2^59.  A
// column is scaled by a power of two to a norm of 1/2 to 1 and a drawn row to 57
// bits of its norm; with M the largest component of level k - 1 a component of
// level k is below 2^57 M sqrt(2 k), which gives the shift back.  A factor common to
// a step's weights cancels in the draw, so no scale is kept but the columns'.
//
// The entries of a level share one absolute error, of variance about
//     var_k = var_{k-1} 4^{27 - sh} |row|^2 k / n + 1/2
// (sh the shift; k of the row's n columns), and the weights' root one of k var.
// Where that passes 2^-96 of their sum, false: nothing is written, and the sample
// is drawn in FP64.  So it is where a column's norm is outside 2^-50 .. 2^50 or a
// drawn row is not finite.  Emulated at n = 10 and 12, rare rows as often as
// likely ones, the summed error of a step's probabilities is at most 2.4 times the
// estimate or 6e-16, so at most 9e-15; Glynn's sums have 1.2e-14.  Haar matrices never
// get there (80,000 samples of n = 10 to 15: 2^-100 at most); 8 samples in 10,000 of
// exp(0.1 i H) at m=16 n=10 do, as a rare row leaves larger entries among the
// columns not yet in use.  Without scales and check inputs with losses down to
// 2^-29 gave other samples, and 1e-5 couplings probabilities off by 0.1 after rare
// rows.
template <int T, bool FIXED>
__device__ __forceinline__ bool draw_sample(const SampArgs& a, int64_t smp, char* mem, const int (*s_c)[kBinom])
{
    const int m = a.m, n = a.n, tid = threadIdx.x % T;
    auto sync = [] {
        if (T == 32) __syncwarp();
        else __syncthreads();
    };
    const int n_even = subset_level(n, 0), n_odd = subset_level(n, 1);
    using Level = std::conditional_t<FIXED, int4, double2>;
    Level* base = (Level*)mem;
    Level* s_a = base + n_even + n_odd;         // A[r_k][.], the drawn row
    double2* s_g = (double2*)(s_a + n);        // entries 0 .. k of level k in FP64
    double* s_w = (double*)(s_g + n);
    int* s_pc = (int*)(s_w + m + (m & 1));               // input mode of each permuted photon
    int* s_rows = s_pc + 15;
    int* s_e = s_rows + 15;                              // exponents of the columns' norms
    unsigned* s_top = (unsigned*)(s_e + 15);             // of the odd and even levels: max |component| >> 29
    unsigned* s_lost = s_top + 2;
    if (FIXED && tid == 0) *s_lost = 0;
    if (tid < n) s_pc[tid] = a.cols[min((int)a.perm[smp * n + tid], n - 1)];   // clamp keeps reads in bounds
    sync();
    if constexpr (FIXED) {
        // squared norms of the columns, sixteen threads a row
        float sum = 0.0f;
        const double2* Uc = a.U + s_pc[tid % 16 < n ? tid % 16 : 0];
#pragma unroll 8
        for (int i = tid / 16; i < m; i += T / 16) {
            const double2 u = __ldg(Uc + (size_t)i * m);
            const float x = abs_float(u.x), y = abs_float(u.y);
            sum = fmaf(x, x, fmaf(y, y, sum));
        }
        sum += __shfl_xor_sync(0xffffffffu, sum, 16);
        float* s_sum = (float*)base;
        if (tid % 32 < 16) s_sum[tid / 32 * 16 + tid % 16] = sum;
        sync();
        if (tid < n) {
            sum = 0.0f;
            for (int w = 0; w < T / 32; ++w) sum += s_sum[w * 16 + tid];
            // 2^e at least the norm; one of 1 but for rounding counts as 1
            s_e[tid] = ((__float_as_int(sum * (1.0f - 0x1p-10f)) >> 23) - 125) >> 1;
            if (!(sum >= 0x1p-100f && sum <= 0x1p100f)) *s_lost = 1;
        }
        sync();
        if (*s_lost) return false;
    }
    float var = 0.0f;                          // warp 0: of level k - 1
    for (int k = 1; k <= n; ++k) {
        // weights: sub-permanent of {0..k-1} \ l is entry k-1-l of level k-1
        const Level* f = base + ((k - 1) & 1 ? n_even : 0);         // level k - 1: even levels first, then odd
        int sh = 1;                            // of level k
        if (FIXED && k > 1) sh = level_shift((float)s_top[(k - 1) & 1] + 1.0f, k);
        if (FIXED && tid == 0) s_top[k & 1] = 0;
        for (int i = tid; i < m; i += T) {
            const double2* Ui = a.U + (size_t)i * m;
            double2 s = make_double2(0.0, 0.0);
            if (k == 1) s = __ldg(Ui + s_pc[0]);
            else
                for (int l = 0; l < k; ++l) {
                    if constexpr (FIXED) cmac(s, __ldg(Ui + s_pc[l]), s_g[k - 1 - l]);
                    else cmac(s, __ldg(Ui + s_pc[l]), f[k - 1 - l]);
                }
            s_w[i] = fma(s.x, s.x, s.y * s.y);
        }
        sync();
        if (tid < 32) {
            double wloc[4], total;
#pragma unroll
            for (int c = 0; c < 4; ++c) wloc[c] = tid + 32 * c < m ? s_w[tid + 32 * c] : 0.0;
            const int r = draw_mode(wloc, m, a.uni[smp * n + k - 1], total);
            if (tid == 0) s_rows[k - 1] = r;
            double2 u = tid < n ? __ldg(a.U + (size_t)r * m + s_pc[tid]) : make_double2(0.0, 0.0);
            if constexpr (FIXED) {
                if (k > 1 && !((float)total * 0x1p-96f >= (float)k * var) && tid == 0) *s_lost = 1;
                if (tid < n) u = make_double2(times_pow2(u.x, -s_e[tid]), times_pow2(u.y, -s_e[tid]));
                double sum = fma(u.x, u.x, u.y * u.y);
                for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
                if (!(sum <= DBL_MAX) && tid == 0) *s_lost = 1;
                // 2^e at least the row's norm but for 2^-17
                const int e = sum > 0.0 ? (((__double2hiint(sum) - 16) >> 20) - 1021) >> 1 : 0;
                const double sc = __hiloint2double((1023 + 57 - e) << 20, 0);
                if (tid < n) s_a[tid] = split30(__double2ll_rn(u.x * sc), __double2ll_rn(u.y * sc));
                if (k > 1) var *= __int_as_float((127 + 2 * (27 - sh)) << 23) * (float)times_pow2(sum, -2 * e) * ((float)k / (float)n);
                var += 0.5f;
            } else if (tid < n) {
                s_a[tid] = u;
            }
        }
        sync();
        if (FIXED && *s_lost) return false;
        if (k == n) break;
        // level k: contiguous runs of subsets (increasing masks) per thread.
        // The rank of S is sum_i C(s_i, i + 1) over its elements in order;
        // without s_j the elements after it move down one place.
        Level* cur = base + (k & 1 ? n_even : 0);
        unsigned top = 0;
        const int cnt = s_c[n][k];
        const int below = s_c[n][k - 1];       // entries of level k - 1
        const int per = (cnt + T - 1) / T;
        const int q0 = tid * per;
        uint32_t mask = 0;
        for (int b = min(q0, cnt - 1), j = k, t = n - 1; j >= 1; --j) {
            while (t > 0 && s_c[t][j] > b) --t;
            mask |= 1u << t;
            b -= s_c[t][j];
        }
        __syncwarp();                          // the search leaves the lanes apart
        for (int q = q0; q < q0 + per; ++q) {
            // every lane runs the same k steps (those past the level redo its
            // last subset and store nothing), so a warp stays together
            int suf = 0;                       // sum over the elements not yet passed, one place down
            uint32_t x = mask;
            for (int i = 0; i < k; ++i, x &= x - 1) suf += s_c[low_bit(x)][i];
            Sum30 re, im;
            double2 acc = make_double2(0.0, 0.0);
            int pre = 0;
            x = mask;
            for (int i = 0; i < k && k > 1; ++i, x &= x - 1) {
                const int l = low_bit(x);
                suf -= s_c[l][i];
                const Level c = f[min((uint32_t)(pre + suf), (uint32_t)(below - 1))];
                if constexpr (FIXED) add_term(re, im, s_a[l], c);
                else cmac(acc, s_a[l], c);
                pre += s_c[l][i + 1];
            }
            if (q < cnt) {
                const Level row = s_a[low_bit(mask)];
                if constexpr (FIXED) {
                    const long long vx = k == 1 ? join30(row.x, row.y) : re.value(sh);
                    const long long vy = k == 1 ? join30(row.z, row.w) : im.value(sh);
                    cur[q] = split30(vx, vy);
                    if (q <= k)                // the subset without column k - q
                        s_g[q] = make_double2(times_pow2((double)vx, -s_e[k - q]), times_pow2((double)vy, -s_e[k - q]));
                    top = max(top, (unsigned)max(llabs(vx) >> 29, llabs(vy) >> 29));
                } else {
                    cur[q] = k == 1 ? row : acc;
                }
            }
            if (q + 1 < cnt) {
                const uint32_t c = mask & (0u - mask), r = mask + c;
                mask = r | (((mask ^ r) >> 2) >> (__ffs(mask) - 1));
            }
        }
        if constexpr (FIXED) {
            top = __reduce_max_sync(0xffffffffu, top);
            if ((tid & 31) == 0) atomicMax(&s_top[k & 1], top);
        }
        sync();
    }
    for (int i = tid; i < m; i += T) {
        int c = 0;
        for (int p = 0; p < n; ++p) c += s_rows[p] == i;
        a.out[smp * m + i] = (uint8_t)c;
    }
    return true;
}

// Not inlined, so that it costs the fixed-point form no registers.
template <int T>
__device__ __noinline__ void draw_sample_fp64(const SampArgs& a, int64_t smp, char* mem, const int (*s_c)[kBinom])
{
    draw_sample<T, false>(a, smp, mem, s_c);
}

// Threads of a block at most.
template <int T, bool FIXED> constexpr int kSubsetThreads = T > 32 ? T : FIXED ? 64 : 256;

// A group of T threads per sample (T = 32: several samples per block); 1024
// threads per SM, where shared memory holds fewer (n = 10, 11) 896.
template <int T, bool FIXED>
__global__ void __launch_bounds__(kSubsetThreads<T, FIXED>, (T == 32 && FIXED ? 896 : 1024) / kSubsetThreads<T, FIXED>)
subset_sampler_kernel(const __grid_constant__ SampArgs a)
{
    extern __shared__ int4 s_mem[];
    __shared__ int s_c[kBinom][kBinom];        // C(t, j)
    for (int q = threadIdx.x; q < kBinom * kBinom; q += blockDim.x) {
        const int t = q / kBinom, j = q % kBinom;
        int c = j <= t ? 1 : 0;
        for (int i = 1; i <= j && j <= t; ++i) c = c * (t + 1 - i) / i;
        s_c[t][j] = c;
    }
    __syncthreads();
    const int64_t smp = (int64_t)blockIdx.x * (blockDim.x / T) + threadIdx.x / T;
    if (smp >= a.count) return;                // whole groups
    char* mem = (char*)s_mem + (size_t)(threadIdx.x / T) * subset_bytes(a.m, a.n);
    if constexpr (FIXED) {
        if (!draw_sample<T, true>(a, smp, mem, s_c)) draw_sample_fp64<T>(a, smp, mem, s_c);
    } else {
        draw_sample<T, false>(a, smp, mem, s_c);
    }
}

template <int NMAX>
__global__ void __launch_bounds__(32 * kSampWarps) sampler_kernel(const SampArgs a)
{
    extern __shared__ double2 sA[];           // A[i][l] = U[i][cols[l]], m x n
    const int m = a.m, n = a.n;
    for (int q = threadIdx.x; q < m * n; q += blockDim.x) {
        const int i = q / n, l = q % n;
        sA[q] = a.U[(size_t)i * m + a.cols[l]];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t smp = (int64_t)blockIdx.x * kSampWarps + warp;
    if (smp >= a.count) return;
    const uint8_t* perm = a.perm + smp * n;
    const double* uni = a.uni + smp * n;
    int rows[NMAX];                            // drawn positions
    int pc[NMAX];                              // permuted column order
#pragma unroll
    for (int l = 0; l < NMAX; ++l) pc[l] = l < n ? min((int)perm[l], n - 1) : 0;   // clamp keeps reads in bounds

    for (int k = 1; k <= n; ++k) {
        // ---- leave-one-out permanents P_l of M = A[rows[0..k-2]; pc[0..k-1]]
        double2 P[NMAX];
#pragma unroll
        for (int l = 0; l < NMAX; ++l) P[l] = make_double2(0.0, 0.0);
        if (k == 1) {
            P[0] = make_double2(lane == 0 ? 1.0 : 0.0, 0.0);
        } else {
            const int R = k - 1;                                // rows of M
            const uint32_t steps = 1u << (R - 1);               // sign vectors with d_0 = +1
            const uint32_t per = steps >= 32 ? steps / 32 : 1;
            const uint32_t k0 = (uint32_t)lane * per;
            if (k0 < steps) {
                uint32_t g = k0 ^ (k0 >> 1);
                double2 x[NMAX];
#pragma unroll
                for (int j = 0; j < NMAX; ++j) {
                    if (j >= k) continue;
                    double2 s = sA[rows[0] * n + pc[j]];
                    for (int i = 1; i < R; ++i) caxpy(s, ((g >> (i - 1)) & 1u) ? -1.0 : 1.0, sA[rows[i] * n + pc[j]]);
                    x[j] = s;
                }
                double par = (__popc(g) & 1) ? -1.0 : 1.0;
                for (uint32_t st = 0; st < per; ++st) {
                    // leave-one-out products of x_0..x_{k-1}
                    double2 pre = make_double2(par, 0.0);
                    double2 pres[NMAX];
#pragma unroll
                    for (int j = 0; j < NMAX; ++j) {
                        if (j >= k) continue;
                        pres[j] = pre;
                        pre = cmul(pre, x[j]);
                    }
                    double2 suf = make_double2(1.0, 0.0);
#pragma unroll
                    for (int j = NMAX - 1; j >= 0; --j) {
                        if (j >= k) continue;
                        const double2 t = cmul(pres[j], suf);
                        P[j] = cadd(P[j], t);
                        suf = cmul(suf, x[j]);
                    }
                    if (st + 1 < per) {
                        const uint32_t kk = k0 + st + 1;
                        const int b = __ffs(kk) - 1;
                        const double sd = ((kk >> (b + 1)) & 1u) ? 2.0 : -2.0;
                        const int rr = rows[b + 1];
#pragma unroll
                        for (int j = 0; j < NMAX; ++j)
                            if (j < k) caxpy(x[j], sd, sA[rr * n + pc[j]]);
                        par = -par;
                    }
                }
            }
            const double sc = ldexp(1.0, -(R - 1));
#pragma unroll
            for (int j = 0; j < NMAX; ++j) {
                if (j >= k) continue;
                for (int off = 16; off > 0; off >>= 1) {
                    P[j].x += __shfl_xor_sync(0xffffffffu, P[j].x, off);
                    P[j].y += __shfl_xor_sync(0xffffffffu, P[j].y, off);
                }
                P[j].x *= sc;
                P[j].y *= sc;
            }
        }
        if (k == 1) {                                   // every lane needs P_0 = 1
            P[0] = make_double2(1.0, 0.0);
        }
        // ---- weights of the m candidate positions, inverse-CDF draw
        double wloc[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int i = lane + 32 * c;
            double w = 0.0;
            if (i < m) {
                double2 s = make_double2(0.0, 0.0);
#pragma unroll
                for (int j = 0; j < NMAX; ++j)
                    if (j < k) cmac(s, sA[i * n + pc[j]], P[j]);
                w = fma(s.x, s.x, s.y * s.y);
            }
            wloc[c] = w;
        }
        double total;
        rows[k - 1] = draw_mode(wloc, m, uni[k - 1], total);
    }
    for (int i = lane; i < m; i += 32) {
        int c = 0;
        for (int p = 0; p < n; ++p) c += rows[p] == i;
        a.out[smp * m + i] = (uint8_t)c;
    }
}

}  // namespace

cudaError_t launch_sampler(const Plan& p, const double2* U, const uint8_t* perm, const double* uni, int64_t count,
                           uint8_t* out, cudaStream_t s)
{
    SampArgs a;
    a.U = U;
    a.m = p.m;
    a.n = p.n;
    for (int j = 0; j < PCV_MAX_PHOTONS; ++j) a.cols[j] = p.cols[j];
    a.perm = perm;
    a.uni = uni;
    a.count = count;
    a.out = out;
    cudaError_t e;
    if (p.n <= 15) {
        // threads per sample: enough for the largest level of a sample, as many
        // samples per SM as shared memory holds
        auto go = [&](auto kernel, int threads, int samples) {
            const size_t smem = (size_t)samples * subset_bytes(p.m, p.n);
            cudaError_t r = allow_dynamic_smem((const void*)kernel, smem);
            if (r != cudaSuccess) return r;
            for (int64_t c0 = 0; c0 < count && r == cudaSuccess; c0 += 1 << 30) {      // grid limit
                SampArgs p1 = a;
                p1.count = std::min<int64_t>(count - c0, 1 << 30);
                p1.perm = perm + c0 * p.n;
                p1.uni = uni + c0 * p.n;
                p1.out = out + c0 * p.m;
                kernel<<<(unsigned)((p1.count + samples - 1) / samples), threads, smem, s>>>(p1);
                note_launches(1);
                r = cudaGetLastError();
            }
            return r;
        };
        // Fixed point and threads, measured on 16,384 samples of n = 14 (m = 60):
        // FP64 with 128 threads 17.3 ms, fixed point with 128, 256, 512 threads
        // 14.4, 11.4, 10.8; n = 12: 4.0, and 2.6, 3.4, 5.7; n = 13: 7.8, and 5.4, 5.2,
        // 7.9; n = 15 (4,096): 9.4 with 256, and 11.3, 7.8, 6.3.  n = 8 (60,000, a warp
        // each): 1.60 in FP64 and 1.96, n = 10 (50,000): 3.10 and 2.41.
        if (p.n <= 8) return go(subset_sampler_kernel<32, false>, 256, 8);
        if (p.n <= 9) return go(subset_sampler_kernel<32, false>, 64, 2);
        if (p.n <= 11) return go(subset_sampler_kernel<32, true>, 64, 2);
        if (p.n <= 12) return go(subset_sampler_kernel<128, true>, 128, 1);
        if (p.n <= 13) return go(subset_sampler_kernel<256, true>, 256, 1);
        return go(subset_sampler_kernel<512, true>, 512, 1);
    }
    const size_t smem = (size_t)p.m * p.n * sizeof(double2);
    const unsigned blocks = (unsigned)((count + kSampWarps - 1) / kSampWarps);
    if ((e = allow_dynamic_smem((const void*)sampler_kernel<16>, smem)) != cudaSuccess) return e;
    sampler_kernel<16><<<blocks, 32 * kSampWarps, smem, s>>>(a);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace pcv
