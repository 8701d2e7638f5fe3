// State expansion of one large distribution on the integer pipe (the sums of
// slos.cu, n <= 12).
//
// What bounds it: the sums of slos.cu are bound by the FP64 pipe, which takes a
// warp instruction per 16 cycles and SM: 64 cycles for the four DFMA of a
// complex term.  Sixteen wide integer multiply-adds of 30-bit halves (fixed30.cuh)
// give the same term in about 16, without any rounding inside a sum; unranking
// then takes as long again, so a thread keeps the first photons of its state.
// m=20 n=10: 2203 us in FP64, 1383 in fixed point, 1118 with the first photons
// kept (relative error against 64 bits 7.6e-16 and 6.3e-16); m=12 n=12: 294, 262,
// 209 and, with the levels' starts overlapped, 168 us (1.2e-15 and 9.5e-16).
// Now (ncu, m=18 n=9): multiplier pipe 49 %, 24 warps an SM, latency of the
// multiply-add chains and of the gathers.
//
// Numbers.  The kernels carry B_k(s) of slos.cu (not C_k: all B_k(s) are of one
// size, so one scale serves a level) as X = B_k(s) 2^S_k, components at most
// 2^59, split as h 2^30 + l with |l| <= 2^29.  The factors U[r][c] sqrt(j), j the
// photons in mode r, are fixed-point numbers of scale 2^(57 - e), 2^e at least
// the 2-norm of column c.  With M the largest component of level k-1 and
// sum_r sqrt(s_r) |U_r| <= sqrt(k) |U|, a component of level k is below
// 2^57 M sqrt(2 k) before it is shifted back to 59 bits: the shift follows from
// M, which every level leaves in the header, so nothing can overflow.  What stays
// unused: level 1 is stored unshifted, 2 + log2(|U| / max |U_r|) of its 59 bits,
// and where a column's entries are of one magnitude a later level's largest
// component is about sqrt(k / m) M, (1 + log2 m) / 2 bits below the bound.  So 2 to 3
// bits at m = 20; 7 of level 1 at m = 1024, n = 2 and 5 of a level at m = 682, n = 3,
// the most modes the tables take.  Sums of half products: with 12 terms the cross
// sum is below 24 2^58 + 2^59 < 2^63, the others are smaller.
//
// A level rounds once, to 2^-52 of the level's typical amplitude or less.  The
// error is one of absolute size, as that of Glynn's sum, so inputs whose outputs
// differ by many orders of magnitude by construction keep the FP64 sums: where a
// column has an entry that is neither zero nor at least 2^-20 of its norm, or a
// norm outside 2^-40 .. 2^40, or an entry that is not finite, or where a mode
// takes all n photons with an amplitude B_n = sqrt(n!) prod_j |U[r][c_j]| below
// 2^-42 of the norms' product (a zero entry counts as the least other one of its
// row: weak couplings between few modes have zeros beside them), the same
// launches run the FP64 form of slos.cu (the first kernel decides, on the
// device).  Single entries do not tell: U = I + 1e-3 Haar at m=19 n=7 has none
// below 2^-17, and 190,797 of its 480,700 amplitudes came out as zero.  The least
// such amplitude of Haar matrices, 300 draws each: m=20 n=10 2^-22 in the median
// and 2^-32 at worst, m=28 n=12 2^-28 and 2^-41.

#include <algorithm>
#include <cmath>

#include "expansion.cuh"
#include "fixed30.cuh"

namespace pcv {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxN = 12;
constexpr int kUBits = 57, kXBits = 59;
constexpr unsigned kBlocks = 152 * 3;          // one wave: a block takes several tiles, its table of factors is built once

struct FixedHeader {
    int fp64;                  // the FP64 form runs
    int colexp[kMaxN];         // e of photon j's column
    unsigned top[kMaxN + 1];   // level k: max |component| >> 29
    int scale[kMaxN + 1];      // S_k
};

struct FixedArgs {
    const double2* U;          // [m][m]
    int m, n, k;
    int col[kMaxN];
    const int64_t* mc;         // [m + 1][n + 1]
    int64_t lo, hi;            // states written
    int steps;                 // of 32 states in a warp's run (K >= 5)
    uint32_t prev_count;
    const int4* prev;
    int4* cur;                 // or null: the last level
    double2* amp;              // last level, at [i - lo]
    double* prob;
    double norm_t;
    FixedHeader* hdr;
    int64_t* status;           // setup: two words zeroed, or null
    float most_bits;           // setup: least log2 of a mode's prod_j |U[r][c_j]| / norm_j, negated
    double sqrtfact[kMaxN + 1];
};

constexpr float kRowBits = 42.0f;

// One warp per photon: its column's norm; then the rows, a thread each: whether
// the fixed-point form applies.
__global__ void fixed_setup_kernel(const __grid_constant__ FixedArgs a)
{
    const int j = threadIdx.x / 32, lane = threadIdx.x & 31;
    extern __shared__ float s_log[];           // [n][m]: -log2 of an entry's larger component, infinity for 0
    __shared__ int s_bad[kMaxN], s_bits;
    __shared__ float s_norm[kMaxN];            // log2 of the norm
    double sum = 0.0, least = INFINITY;
    for (int r = lane; r < a.m; r += 32) {
        const double2 u = a.U[(size_t)r * a.m + a.col[j]];
        sum = fma(u.x, u.x, fma(u.y, u.y, sum));
        const double c = fmax(fabs(u.x), fabs(u.y));
        if (c > 0.0) least = fmin(least, c);
        s_log[j * a.m + r] = -__log2f((float)c);
    }
    for (int d = 16; d; d >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, d);
        least = fmin(least, __shfl_xor_sync(0xffffffffu, least, d));
    }
    const double norm = sqrt(sum);
    // written so that a NaN fails
    const bool ok = norm >= 0x1p-40 && norm <= 0x1p40 && least >= 0x1p-20 * norm;
    if (lane == 0) {
        s_bad[j] = !ok;
        s_norm[j] = __log2f((float)norm);
        int e = 0;
        if (ok) {
            frexp(norm * (1.0 - 0x1p-20), &e);     // a norm of 1 but for rounding counts as 1
        }
        a.hdr->colexp[j] = e;
    }
    if (threadIdx.x <= kMaxN) a.hdr->top[threadIdx.x] = 0;
    if (a.status && threadIdx.x < 2) a.status[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_bits = 0;
    __syncthreads();
    for (int r = threadIdx.x; r < a.m; r += blockDim.x) {
        float bits = 0.0f, most = 0.0f;
        int zeros = 0;
        for (int q = 0; q < a.n; ++q) {
            const float b = s_log[q * a.m + r];
            if (isinf(b)) {
                ++zeros;
            } else {                           // nothing to use where a column is not ok
                bits += fmaxf(b + s_norm[q], 0.0f);
                most = fmaxf(most, b + s_norm[q]);
            }
        }
        if (zeros < a.n) atomicMax(&s_bits, __float_as_int(bits + zeros * most));      // not negative: ordered as integers
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int bad = __int_as_float(s_bits) > a.most_bits;
        for (int q = 0; q < a.n; ++q) bad |= s_bad[q];
        a.hdr->fp64 = bad;
    }
}

// The FP64 form of a level: the sums of slos.cu.  Not inlined, so that it costs
// the fixed-point form no registers.
__device__ __noinline__ void fp64_level(const FixedArgs& a, double2* s_u, const uint32_t* s_mc)
{
    const int m = a.m, k = a.k;
    const double2* prev = (const double2*)a.prev;
    for (int r = threadIdx.x; r < m; r += kThreads) s_u[r] = a.U[(size_t)r * m + a.col[k - 1]];
    __syncthreads();
    for (int64_t i = a.lo + (int64_t)blockIdx.x * kThreads + threadIdx.x; i < a.hi; i += (int64_t)gridDim.x * kThreads) {
        double2 acc = make_double2(0.0, 0.0);
        const double sf = expand_state<kMaxN, uint32_t>(s_mc, k + 1, m, k, (uint32_t)i, a.prev_count, a.sqrtfact,
                                                        [&](int r, uint32_t rk, int) {
                                                            if (k == 1) acc = s_u[r];
                                                            else cmac(acc, s_u[r], prev[rk]);
                                                        });
        if (a.cur) {
            ((double2*)a.cur)[i] = acc;
            continue;
        }
        const double sc = sf * a.norm_t;
        const double2 v = make_double2(acc.x * sc, acc.y * sc);
        if (a.amp) a.amp[i - a.lo] = v;
        if (a.prob) a.prob[i - a.lo] = fma(v.x, v.x, v.y * v.y);
    }
}

// What a block needs before its states: the tables, the shift and the scale.
struct LevelSetup {
    bool fp64;
    int sh;
    double back;
};

__device__ __forceinline__ LevelSetup level_setup(const FixedArgs& a, int k, int4* s_f, uint32_t* s_mc, unsigned& s_top)
{
    const int m = a.m, w1 = k + 1;
    LevelSetup o{};
    if (k == 1) level_below_done();            // the first kernel's header; from level 2 on it is complete
    o.fp64 = a.hdr->fp64;
    for (int q = threadIdx.x; q < (m + 1) * w1; q += kThreads)
        s_mc[q] = (uint32_t)a.mc[(q / w1) * (a.n + 1) + q % w1];
    if (threadIdx.x == 0) s_top = 0;
    if (o.fp64) {
        if (k > 1) level_below_done();
        return o;
    }
    const int e = a.hdr->colexp[k - 1];
    for (int q = threadIdx.x; q < m * k; q += kThreads) {
        const double2 u = a.U[(size_t)(q / k) * m + a.col[k - 1]];
        const double f = ldexp(sqrt((double)(q % k + 1)), kUBits - e);
        s_f[q] = split30(__double2ll_rn(u.x * f), __double2ll_rn(u.y * f));
    }
    if (k > 1) level_below_done();
    // The shift back to kXBits bits; the last level keeps three bits more, as it is not multiplied again.
    const bool last = !a.cur;
    int scale = kUBits - e;
    if (k > 1) {
        const double bound = ((double)a.hdr->top[k - 1] + 1.0) * sqrt(2.0 * k) * (1.0 + 0x1p-18);   // of M sqrt(2k), in 2^29
        o.sh = min(max(ilogb(bound) + 1 + 29 + kUBits - kXBits - 30 - (last ? 3 : 0), 1), 30);
        scale += a.hdr->scale[k - 1] - 30 - o.sh;
    }
    if (!last && blockIdx.x == 0 && threadIdx.x == 0) a.hdr->scale[k] = scale;
    o.back = ldexp(a.norm_t, -scale);
    __syncthreads();
    return o;
}

// State i of the level, x + i y: to the next level, or as an output.
__device__ __forceinline__ void store_state(const FixedArgs& a, int64_t i, long long x, long long y, double back,
                                            unsigned& top)
{
    if (a.cur) {
        a.cur[i] = split30(x, y);
        top = max(top, (unsigned)max(llabs(x) >> 29, llabs(y) >> 29));
        return;
    }
    const double2 v = make_double2((double)x * back, (double)y * back);
    if (a.amp) a.amp[i - a.lo] = v;
    if (a.prob) a.prob[i - a.lo] = fma(v.x, v.x, v.y * v.y);
}

__device__ __forceinline__ void publish_top(const FixedArgs& a, int k, unsigned top, unsigned& s_top)
{
    if (!a.cur) return;
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_top, top);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(&a.hdr->top[k], s_top);
}

// Levels 1 to 4: a thread per state.
__global__ void __launch_bounds__(kThreads) expand_fixed_low_kernel(const __grid_constant__ FixedArgs a)
{
    extern __shared__ int4 s_f[];               // [m][k] factors (FP64 form: [m] entries of U), then the count table
    const int m = a.m, k = a.k;
    uint32_t* s_mc = (uint32_t*)(s_f + m * k);
    __shared__ unsigned s_top;
    const LevelSetup o = level_setup(a, k, s_f, s_mc, s_top);
    if (o.fp64) return fp64_level(a, (double2*)s_f, s_mc);
    unsigned top = 0;
    for (int64_t i = a.lo + (int64_t)blockIdx.x * kThreads + threadIdx.x; i < a.hi; i += (int64_t)gridDim.x * kThreads) {
        Sum30 re, im;
        if (k == 1) {
            const int4 u = s_f[i];
            store_state(a, i, join30(u.x, u.y), join30(u.z, u.w), o.back, top);
            continue;
        }
        expand_state<4, uint32_t>(s_mc, k + 1, m, k, (uint32_t)i, a.prev_count, nullptr, [&](int r, uint32_t rk, int mult) {
            add_term(re, im, s_f[r * k + mult - 1], a.prev[rk]);
        });
        store_state(a, i, re.value(o.sh), im.value(o.sh), o.back, top);
    }
    publish_top(a, k, top, s_top);
}

// Level K >= 5: a warp takes runs of 32 `a.steps` consecutive states.  A thread
// goes through its run 32 states at a time and keeps its first K - 4 photons
// while only the last four change (113 states on average at m=20 n=10): their
// modes, factors and the part of their terms' ranks that the last four do not
// touch; a rank is then one subtraction.
template <int K>
__global__ void __launch_bounds__(kThreads, 3) expand_fixed_kernel(const __grid_constant__ FixedArgs a)
{
    constexpr int P = K - 4, W = K + 1;
    extern __shared__ int4 s_f[];
    const int m = a.m;
    uint32_t* s_mc = (uint32_t*)(s_f + m * K);
    __shared__ unsigned s_top;
    const LevelSetup o = level_setup(a, K, s_f, s_mc, s_top);
    if (o.fp64) return fp64_level(a, (double2*)s_f, s_mc);

    // multisets of size j above mode l
    auto above = [&](int l, int j) { return s_mc[(m - 1 - l) * W + j]; };
    // the next position's mode from v on, `rest` photons behind it
    auto next = [&](int v, int rest, uint32_t& idx) {
        const uint32_t* q = s_mc + (m - v) * W + rest;
        for (uint32_t c = *q; idx >= c; c = *q) {
            idx -= c;
            q -= W;
            ++v;
        }
        return v;
    };

    const uint32_t run = 32u * (uint32_t)a.steps;
    const uint32_t total = (uint32_t)(a.hi - a.lo), runs = (total + run - 1) / run;
    unsigned top = 0;
    for (uint32_t c = blockIdx.x * (kThreads / 32) + threadIdx.x / 32; c < runs; c += gridDim.x * (kThreads / 32)) {
        uint32_t base[P], off = 0, size = 0, after = 0;
        int fac[P], lp = 0, lm = 0;             // factor of a term, -1 where the mode's run goes on
        const uint32_t end = min(total - c * run, run);
        for (uint32_t d = threadIdx.x & 31; d < end; d += 32) {
            const uint32_t out = c * run + d;
            off += 32;
            if (off >= size) {                  // the first photons of this state
                int l[P];
                uint32_t idx = (uint32_t)a.lo + out;
                int v = 0;
#pragma unroll
                for (int p = 0; p < P; ++p) l[p] = v = next(v, K - 1 - p, idx);
                off = idx;
                size = s_mc[(m - v) * W + 4];
                uint32_t suf = 0;
                after = a.prev_count - 1;
#pragma unroll
                for (int p = 1; p < P; ++p) suf += above(l[p], K - p);
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    lm = p > 0 && l[p > 0 ? p - 1 : 0] == l[p] ? lm + 1 : 1;
                    base[p] = after - suf;
                    fac[p] = p + 1 < P && l[p + 1 < P ? p + 1 : p] == l[p] ? -1 : l[p] * K + lm - 1;
                    after -= above(l[p], K - 1 - p);
                    if (p + 1 < P) suf -= above(l[p + 1 < P ? p + 1 : p], K - 1 - p);
                }
                lp = v;
            }
            int x[4];
            {
                uint32_t idx = off;
                x[0] = next(lp, 3, idx);
                x[1] = next(x[0], 2, idx);
                x[2] = next(x[1], 1, idx);
                x[3] = x[2] + (int)idx;
            }
            uint32_t suf = above(x[1], 3) + above(x[2], 2) + above(x[3], 1);
            const uint32_t all = suf + above(x[0], 4);
            Sum30 re, im;
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (p + 1 < P ? fac[p] >= 0 : x[0] != lp) add_term(re, im, s_f[fac[p]], a.prev[base[p] - all]);
            uint32_t pre = after;
            int mult = lm, before = lp;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                mult = x[q] == before ? mult + 1 : 1;
                before = x[q];
                if (q == 3 || x[q < 3 ? q + 1 : q] != x[q]) add_term(re, im, s_f[x[q] * K + mult - 1], a.prev[pre - suf]);
                if (q < 3) {
                    pre -= above(x[q], 3 - q);
                    suf -= above(x[q < 3 ? q + 1 : q], 3 - q);
                }
            }
            store_state(a, a.lo + out, re.value(o.sh), im.value(o.sh), o.back, top);
        }
    }
    publish_top(a, K, top, s_top);
}

cudaError_t launch_level(FixedArgs a, cudaStream_t s)
{
    const size_t smem = (size_t)a.m * a.k * sizeof(int4) + (size_t)(a.m + 1) * (a.k + 1) * sizeof(uint32_t);
    // Runs of up to 16 x 32 states while every warp slot still gets four of them.
    const int64_t n = a.hi - a.lo;
    a.steps = (int)std::min<int64_t>(16, std::max<int64_t>(1, n / (32 * 4 * 8 * (int64_t)kBlocks)));
    const int64_t per_block = (int64_t)kThreads * (a.k <= 4 ? 1 : a.steps);
    const unsigned grid = (unsigned)std::min<int64_t>((n + per_block - 1) / per_block, kBlocks);
    auto go = [&](void (*kernel)(const FixedArgs)) { return launch_level_kernel(kernel, dim3(grid), kThreads, smem, s, a); };
    switch (a.k) {
    case 5: return go(expand_fixed_kernel<5>);
    case 6: return go(expand_fixed_kernel<6>);
    case 7: return go(expand_fixed_kernel<7>);
    case 8: return go(expand_fixed_kernel<8>);
    case 9: return go(expand_fixed_kernel<9>);
    case 10: return go(expand_fixed_kernel<10>);
    case 11: return go(expand_fixed_kernel<11>);
    case 12: return go(expand_fixed_kernel<12>);
    default: return go(expand_fixed_low_kernel);
    }
}

}  // namespace

// By the size of the problem alone, so that a range of outputs takes the form
// of the whole.  The line (both with plain launches): fixed point against FP64 at m=20 n=6 (0.23 M states in
// all) 57 and 50 us, m=46 n=4 (0.25 M) 49 and 36, m=30 n=5 (0.32 M) 54 and 50,
// m=24 n=6 (0.59 M) 69 and 70, m=16 n=8 (0.74 M) 88 and 96, m=16 n=9 140 and 195.  states: of all levels; tables of factors and counts up to 44 KB.
bool expand_fixed_applies(int m, int n, int64_t largest, int64_t states)
{
    return n >= 2 && n <= kMaxN && m * n <= 2048 && largest <= (int64_t)UINT32_MAX && states >= kFixedMinStates;
}

static_assert(sizeof(FixedHeader) <= 256, "the header fits the table that the FP64 form leaves unused");

cudaError_t launch_expand_fixed(const Plan& p, const double2* U, const int64_t* count, int64_t lo, int64_t hi,
                                double* prob, double2* amp, const int64_t* mc, void* header, double2* const* buf,
                                int64_t* status, cudaStream_t s)
{
    ExpandArgs d;
    expand_defaults(&d);
    FixedArgs a{};
    a.U = U;
    a.m = p.m;
    a.n = p.n;
    a.mc = mc;
    a.norm_t = p.norm_t;
    a.hdr = (FixedHeader*)header;
    a.status = status;
    a.most_bits = kRowBits + (float)std::log2(d.sqrtfact[p.n]);
    for (int j = 0; j < p.n; ++j) a.col[j] = p.cols[j];
    for (int j = 0; j <= kMaxN; ++j) a.sqrtfact[j] = d.sqrtfact[j];
    fixed_setup_kernel<<<1, 32 * p.n, (size_t)p.m * p.n * sizeof(float), s>>>(a);      // 8 KB at most
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    for (int k = 1; k <= p.n && e == cudaSuccess; ++k) {
        const bool last = k == p.n;
        a.k = k;
        a.lo = last ? lo : 0;
        a.hi = last ? hi : count[k];
        if (a.hi <= a.lo) break;
        a.prev_count = (uint32_t)count[k - 1];
        a.prev = (const int4*)buf[(k - 1) & 1];
        a.cur = last ? nullptr : (int4*)buf[k & 1];
        a.amp = last ? amp : nullptr;
        a.prob = last ? prob : nullptr;
        e = launch_level(a, s);
    }
    return e;
}

}  // namespace pcv
