// Shared-row-sum Glynn kernels for explicit outputs: one block computes a tile
// of outputs of one (U, input) pair, and a persistent variant pulls tiles of
// many circuits of uneven size from a device work queue.
//
// With Glynn's sign vector d on the input photons (columns of U_{T,S}, Eq.
// eqperm), the row sum of output row i depends only on its output mode:
// y_r(d) = sum_j d_j U[r][c_j].  A block keeps y_r(d) of the modes its outputs
// use, advancing them one Gray step at a time, and each output only forms its
// product a(S) += sigma(d) prod_i y_{r_i}(d).
//
// The products are what bounds the kernel: n - 1 complex ones per output and
// sign vector.  They run on the integer pipe (softc.cuh; about 20 cycles per
// warp and product where FP64 takes 64), with the row sums as fixed-point
// numbers: mode r's columns are rounded once to 2^-61 of a power of two 2^{E_r}
// that bounds sum_j |Re U|, sum_j |Im U|, so the sums themselves are exact
// integers (no drift along the Gray sequence) and an output's scale is
// 2^{sum E_r}, applied once at the end.  Each term is rounded to FP64 and added
// there (8 FP64 instructions, which overlap the integer work).  A mode with a
// non-finite entry in a used column makes its outputs NaN.
//
// Block layout: T = 32 .. 256 outputs x S = 256 / T contiguous ranges of sign
// vectors, walked in chunks of C steps whose row sums are staged in shared
// memory, four steps of a thread's range at a time (four independent chains).
// A sequence may also be split in `parts` over several blocks, whose sums go
// to a buffer and are added in part order: at n = 16 one tile of 64 outputs on
// one SM took 34 ms, and the batch's last items ran alone (48 circuits,
// n <= 16, 512 outputs: 70.8 ms with FP64 products and whole tiles, 3.2 ms
// now; 256 outputs at m=324 n=18: 6.95 ms by the plain block kernel, 1.82 ms).  The S
// partial sums of an output are added in a fixed order at the end, so results
// are deterministic.

#include <algorithm>
#include <cmath>

#include "pcv_common.cuh"
#include "softc.cuh"

namespace pcv {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxModes = 128;       // modes of a batched circuit
constexpr int kMaxChunk = 16;        // Gray steps staged per split and pass
constexpr int kLow = 4;              // columns kept in shared memory (flipped within a chunk)
constexpr int kMinTile = 32;
constexpr int kPack = 512;           // a circuit's tile size and parts in one int: T + kPack parts
constexpr int kItemsPerSm = 12;      // a batched item holds at most 1 / (kItemsPerSm sms) of the tile work
constexpr int kPartSteps = 64;       // sign vectors per split that a part keeps,
constexpr int kLeastSteps = 8;       // or where that leaves SMs idle: parts up to kLightPerSm blocks per SM
constexpr int kLightPerSm = 2;
constexpr float kEntryStart = 2e4f;  // cycles of a multiplicity entry on its warp: at first,
constexpr float kEntryCycles = 100;  // and per FP64 instruction
constexpr int kStage = 2560;         // staged row sums of a batched block (40 KB: three blocks per SM)
constexpr int kStageOne = 3072;      // the same for one circuit (48 KB: eight steps of 324 modes)

// A block's work: outputs and shape of the tile, the part of the sequence.
struct TileShape {
    int T;                           // outputs (a power of two, 32 .. 256)
    int parts;                       // blocks per sequence
    int slots;                       // modes with row sums in shared memory, at most
    int stage;                       // staged row sums
};

// The matrix and the result arrays of a tile's batch entry.
struct TileOut {
    const double2* U;
    double2* amp;
    double* prob;
};

// Shared memory of a block, carved from one dynamic array (the sums of the
// splits at the end reuse the staged row sums).
struct TileMem {
    int4* y;                         // [S][C][slots]
    longlong2* run;                  // [S][slots] running row sums
    longlong2* low;                  // [kLow][slots]: 2 U[r][c_{b+1}]
    int* scale;                      // [slots]: E_r
    int* map;                        // [m]: slot of a mode, -1 unused
    uint16_t* rows;                  // [n][T]: slot of each row
    uint16_t* mode;                  // [slots]
};

__host__ __device__ inline size_t tile_smem(int n, int m, const TileShape& t)
{
    const int S = kThreads / t.T;
    return (size_t)t.stage * 16 + (size_t)(S + kLow) * t.slots * 16 + (size_t)t.slots * 4 + (size_t)(m + (m & 1)) * 4 +
           (size_t)n * t.T * 2 + (size_t)t.slots * 2 + 16;
}

__device__ TileMem tile_mem(unsigned char* base, int n, int m, const TileShape& t)
{
    const int S = kThreads / t.T;
    TileMem k;
    k.y = (int4*)base;
    k.run = (longlong2*)(k.y + t.stage);
    k.low = k.run + S * t.slots;
    k.scale = (int*)(k.low + kLow * t.slots);
    k.map = k.scale + t.slots;
    k.rows = (uint16_t*)(k.map + m + (m & 1));
    k.mode = k.rows + n * t.T;
    return k;
}

constexpr int kBadScale = 1 << 20;   // scale of a mode with a non-finite entry

// 2^{61 - E} u rounded to nearest, for |u| < 2^E, on the integer pipe: the
// 53-bit mantissa moves left by at most 8 places or right with rounding.
__device__ __forceinline__ long long fixed_entry(double u, int E)
{
    const long long b = __double_as_longlong(u);
    const int ef = (int)((b >> 52) & 0x7FF);
    long long m = b & ((1ll << 52) - 1);
    if (ef) m |= 1ll << 52;
    const int sh = (ef ? ef : 1) - 1014 - E;
    if (sh >= 0) {
        m <<= min(sh, 8);
    } else {
        const int r = min(-sh, 60);
        m = (m + (1ll << (r - 1))) >> r;
    }
    return b < 0 ? -m : m;
}

// The products of W consecutive sign vectors of one output (independent
// chains, one row index for all) added to acc; y: their staged row sums, M
// apart; odd: the first one's sign.
template <int W>
__device__ __forceinline__ void tile_products(double2& acc, const int4* y, int M, const uint16_t* rows, int T, int n,
                                              bool odd)
{
    SoftC p[W];
    int r = rows[0];
#pragma unroll
    for (int w = 0; w < W; ++w) p[w] = soft_first(y[w * M + r]);
    for (int i = 1; i < n; ++i) {
        r = rows[i * T];
#pragma unroll
        for (int w = 0; w < W; ++w) soft_mul(p[w], y[w * M + r]);
    }
#pragma unroll
    for (int w = 0; w < W; ++w) soft_add(acc, p[w], odd != ((w & 1) != 0));
}

// One tile of circuit c: positions [tile T, (tile + 1) T) of its output list,
// which is idx[0..count) (or the outputs 0..count-1 themselves when idx is
// null), part `part` of the sign vectors.  With several parts the raw sums go
// to partial[part * count + position].
__device__ void tile_item(const pcv_batch_desc& c, const TileOut& out, const TileShape sh, int64_t tile, int part,
                          unsigned char* smem, const int* idx, int64_t count, double2* partial)
{
    __shared__ int s_used, s_warp[kThreads / 32];
    const int n = c.n, m = c.m, T = sh.T, S = kThreads / T;
    const TileMem k = tile_mem(smem, n, m, sh);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ol = tid % T, s = tid / T;
    const int64_t pos = tile * T + ol;
    const bool live = pos < count;
    const int64_t o = live ? (idx ? (int64_t)idx[pos] : pos) : 0;
    const double2* U = out.U;

    // modes the tile's outputs use, and their slots in mode order
    for (int r = tid; r < m; r += kThreads) k.map[r] = 0;
    __syncthreads();
    bool ok = false;
    if (live) {
        const uint8_t* occ = c.outputs + o * m;
        int cnt = 0;
        for (int r = 0; r < m; ++r) cnt += occ[r];
        ok = cnt == n;
        if (ok && s == 0)
            for (int r = 0; r < m; ++r)
                if (occ[r]) k.map[r] = 1;
    }
    __syncthreads();
    int used = 0;
    for (int r0 = 0; r0 < m; r0 += kThreads) {
        const int r = r0 + tid;
        const bool u = r < m && k.map[r];
        const unsigned bal = __ballot_sync(0xffffffffu, u);
        if (lane == 0) s_warp[wid] = __popc(bal);
        __syncthreads();
        int at = used + __popc(bal & ((1u << lane) - 1));
        for (int w = 0; w < wid; ++w) at += s_warp[w];
        if (r < m) k.map[r] = u ? at : -1;
        if (u) k.mode[at] = (uint16_t)r;
        for (int w = 0; w < kThreads / 32; ++w) used += s_warp[w];
        __syncthreads();
    }
    if (tid == 0) s_used = used;
    __syncthreads();
    const int M = max(1, s_used);

    // rows of each output, and what multiplies its sum: norms and 2^{sum E_r}
    double norm = 1.0;
    if (ok && s == 0) {
        const uint8_t* occ = c.outputs + o * m;
        int cnt = 0;
        double f = 1.0;
        for (int r = 0; r < m; ++r)
            for (int q = 1; q <= occ[r]; ++q) {
                k.rows[cnt++ * T + ol] = (uint16_t)k.map[r];
                f *= q;
            }
        int run = 1;
        for (int j = 1; j < n; ++j) {         // prod t! from the sorted photon -> input-mode list
            run = (c.cols[j] == c.cols[j - 1]) ? run + 1 : 1;
            f *= run;
        }
        norm = 1.0 / sqrt(f);
    }
    // scales, and the columns flipped within a chunk
    for (int q = tid; q < s_used; q += kThreads) {
        const double2* Ur = U + (size_t)k.mode[q] * m;
        double br = 0.0, bi = 0.0;
        for (int j = 0; j < n; ++j) {
            const double2 u = Ur[c.cols[j]];
            br += fabs(u.x);
            bi += fabs(u.y);
        }
        const bool fin = isfinite(br) && isfinite(bi);
        const double b = fmax(br, bi);
        const int E = !fin ? kBadScale : (b > 0.0 ? ilogb(b) + 1 : 0);
        k.scale[q] = E;
        for (int l = 0; l < kLow; ++l) {
            const double2 u = fin && l + 1 < n ? Ur[c.cols[l + 1]] : make_double2(0.0, 0.0);
            k.low[l * sh.slots + q] = make_longlong2(2 * fixed_entry(u.x, E), 2 * fixed_entry(u.y, E));
        }
    }
    __syncthreads();
    // range q = part S + split holds the sign vectors [q steps, (q + 1) steps),
    // cut at 2^{n-1}; steps is a multiple of the chunk
    const int64_t K = 1ll << (n - 1);
    const int64_t ranges = (int64_t)S * sh.parts;
    int64_t steps = (K + ranges - 1) / ranges;
    int C = kMaxChunk;
    while (C > steps || (C > 1 && S * C * M > sh.stage)) C >>= 1;
    steps = (steps + C - 1) / C * C;
    const int64_t k0p = (int64_t)part * S * steps;
    const int active = (int)max((int64_t)0, min((int64_t)S, (K - k0p + steps - 1) / steps));   // splits with work
    const int64_t mine = max((int64_t)0, min(steps, K - k0p - (int64_t)s * steps));            // of this thread's split
    // running row sums of every split at its first sign vector
    for (int q = tid; q < active * s_used; q += kThreads) {
        const int ss = q / s_used, v = q % s_used;
        const int E = k.scale[v];
        long long yr = 0, yi = 0;
        if (E != kBadScale) {
            const int64_t kk = k0p + (int64_t)ss * steps;
            const uint64_t g = (uint64_t)kk ^ ((uint64_t)kk >> 1);
            const double2* Ur = U + (size_t)k.mode[v] * m;
            for (int j = 0; j < n; ++j) {
                const double2 u = Ur[c.cols[j]];
                const long long fr = fixed_entry(u.x, E), fi = fixed_entry(u.y, E);
                const bool neg = j > 0 && ((g >> (j - 1)) & 1u);
                yr += neg ? -fr : fr;
                yi += neg ? -fi : fi;
            }
        }
        k.run[ss * sh.slots + v] = make_longlong2(yr, yi);
    }
    double2 acc = make_double2(0.0, 0.0);
    const uint16_t* rows = k.rows + ol;
    for (int64_t base = 0; base < steps; base += C) {
        __syncthreads();
        // stage C steps of row sums for every split; advance the running sums
        for (int q = tid; q < active * s_used; q += kThreads) {
            const int ss = q / s_used, v = q % s_used;
            longlong2 y = k.run[ss * sh.slots + v];
            int4* dst = k.y + (size_t)ss * C * M + v;
            const int64_t kk0 = k0p + (int64_t)ss * steps + base;
            const int64_t left = min(steps - base, K - kk0);          // steps from here in the range
            for (int st = 0; st < C; ++st) {
                dst[st * M] = soft_split(y.x, y.y);
                if (st + 1 >= left) break;
                const int64_t kk = kk0 + st + 1;
                const int b = __ffsll(kk) - 1;
                longlong2 u;
                if (b < kLow) {
                    u = k.low[b * sh.slots + v];
                } else {
                    const int E = k.scale[v];
                    u = make_longlong2(0, 0);
                    if (E != kBadScale) {
                        const double2 e = U[(size_t)k.mode[v] * m + c.cols[b + 1]];
                        u = make_longlong2(2 * fixed_entry(e.x, E), 2 * fixed_entry(e.y, E));
                    }
                }
                const bool plus = (kk >> (b + 1)) & 1;
                y.x += plus ? u.x : -u.x;
                y.y += plus ? u.y : -u.y;
            }
            k.run[ss * sh.slots + v] = y;
        }
        __syncthreads();
        if (ok && base < mine) {
            // K and steps are multiples of C, so a range holds whole chunks
            const bool odd = (k0p + (int64_t)s * steps + base) & 1;   // sigma(d) alternates along the sequence
            const int4* ys = k.y + (size_t)s * C * M;
            if (C >= 4) {
                for (int st = 0; st < C; st += 4) tile_products<4>(acc, ys + st * M, M, rows, T, n, odd);
            } else if (C == 2) {
                tile_products<2>(acc, ys, M, rows, T, n, odd);
            } else {
                tile_products<1>(acc, ys, M, rows, T, n, odd);
            }
        }
    }
    __syncthreads();
    double2* s_acc = (double2*)k.y;
    if (S > 1) {
        s_acc[tid] = acc;
        __syncthreads();
    }
    if (s == 0 && live) {
        double2 t = acc;
        for (int ss = 1; ss < S; ++ss) t = cadd(t, s_acc[ss * T + ol]);
        double2 v = make_double2(0.0, 0.0);
        if (ok) {
            int e = 0;
            bool bad = false;
            for (int i = 0; i < n; ++i) {
                const int E = k.scale[rows[i * T]];
                bad |= E == kBadScale;
                e += E;
            }
            const double nan = __longlong_as_double(0x7FF8000000000000ll);
            v = bad ? make_double2(nan, nan)
                    : make_double2(scalbn(t.x * norm, e - (n - 1)), scalbn(t.y * norm, e - (n - 1)));
        }
        if (sh.parts > 1) {
            partial[(int64_t)part * count + pos] = v;
        } else {
            if (out.amp) out.amp[o] = v;
            if (out.prob) out.prob[o] = fma(v.x, v.x, v.y * v.y);
        }
    }
    __syncthreads();
}

// Tiles x parts of one circuit (U + b ustride, outputs + b ostride for
// blockIdx.y = b).
struct TileLaunch {
    pcv_batch_desc c;
    TileShape sh;
    int64_t ustride, ostride;
    double2* partial;
};

__global__ void __launch_bounds__(kThreads, 2) glynn_tile_kernel(const __grid_constant__ TileLaunch a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int64_t b = blockIdx.y;
    TileOut out;
    out.U = (const double2*)a.c.U + b * a.ustride;
    out.amp = a.c.amp ? (double2*)a.c.amp + b * a.ostride : nullptr;
    out.prob = a.c.prob ? a.c.prob + b * a.ostride : nullptr;
    tile_item(a.c, out, a.sh, blockIdx.x / a.sh.parts, blockIdx.x % a.sh.parts, smem, nullptr, a.c.n_out, a.partial);
}

// Several parts: an output's sums added in part order.
__device__ void add_parts(const pcv_batch_desc& c, const double2* partial, int parts, const int* idx, int64_t count,
                          int64_t pos)
{
    double2 v = __ldcg(partial + pos);          // of other blocks: not from this SM's cache
    for (int q = 1; q < parts; ++q) v = cadd(v, __ldcg(partial + (int64_t)q * count + pos));
    const int64_t o = idx ? idx[pos] : pos;
    if (c.amp) ((double2*)c.amp)[o] = v;
    if (c.prob) c.prob[o] = fma(v.x, v.x, v.y * v.y);
}

__global__ void __launch_bounds__(kThreads) tile_parts_kernel(const __grid_constant__ TileLaunch a)
{
    const int64_t pos = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (pos < a.c.n_out) add_parts(a.c, a.partial, a.sh.parts, nullptr, a.c.n_out, pos);
}

// Work queue of the batched launch: items (circuit, tile of the circuit's
// tile-routed outputs, part of the sign vectors) in order of decreasing photon
// number; blocks pull the next item with one atomicAdd and never wait for
// another block.
struct Queue {
    int* counter;
    int* total;
    int* item_circ;
    int* item_tile;           // tile * parts + part
    const int64_t* out_off;   // first entry of circuit c in idx
    const int* n_tile;        // tile-routed outputs of circuit c (idx[out_off[c] ...])
    const int* idx;
    int* shape;               // of circuit c: outputs per tile + kPack * parts (blocks per sequence)
    int64_t* slot_off;        // circuit c's first partial sum (parts > 1)
    double2* partial;         // null: every sequence in one part
    int* done;                // finished parts of a tile, at its first item
};

__device__ TileShape batch_shape(const pcv_batch_desc& d, int T, int parts)
{
    TileShape t;
    t.T = T;
    t.parts = parts;
    t.slots = min(d.m, T * d.n);
    t.stage = kStage;
    return t;
}

__global__ void __launch_bounds__(kThreads, 2) glynn_persistent_kernel(const pcv_batch_desc* descs, Queue q)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_item, s_done;
    const int total = *q.total;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(q.counter, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= total) break;
        const int c = q.item_circ[it], T = q.shape[c] % kPack, parts = q.shape[c] / kPack;
        const int tile = q.item_tile[it] / parts, part = q.item_tile[it] % parts;
        const TileOut out{(const double2*)descs[c].U, (double2*)descs[c].amp, descs[c].prob};
        double2* partial = parts > 1 ? q.partial + q.slot_off[c] : nullptr;
        tile_item(descs[c], out, batch_shape(descs[c], T, parts), tile, part, smem, q.idx + q.out_off[c], q.n_tile[c], partial);
        if (parts == 1) continue;
        // the block that finishes a tile's last part adds them all, in part order
        // (a launch of its own for that took 3 us of a small batch's 50)
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_done = atomicAdd(q.done + (it - part), 1);
        __syncthreads();
        if (s_done + 1 < parts) continue;
        __threadfence();
        const int64_t pos = (int64_t)tile * T + threadIdx.x;
        if (threadIdx.x < T && pos < q.n_tile[c])
            add_parts(descs[c], partial, parts, q.idx + q.out_off[c], q.n_tile[c], pos);
    }
}

// A descriptor the kernels cannot run (n or m out of range, an input mode
// outside [0, m) or out of order) gets no work; the binding checks
// descriptors before they reach the device.
__device__ bool desc_ok(const pcv_batch_desc& d)
{
    if (d.n < 1 || d.n > PCV_MAX_PHOTONS || d.m < 1 || d.m > kMaxModes || d.n_out < 0) return false;
    for (int j = 0; j < d.n; ++j)
        if (d.cols[j] < 0 || d.cols[j] >= d.m || (j > 0 && d.cols[j] < d.cols[j - 1])) return false;
    return true;
}

// Block-wide exclusive scan of one value per thread (1024 threads at most);
// returns the thread's offset, *total the sum.  buf holds 64 values.
template <typename T>
__device__ T block_scan(T v, T* buf, T* total)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = (blockDim.x + 31) >> 5;
    T incl = v;
    for (int off = 1; off < 32; off <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
    }
    if (lane == 31) buf[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        T w = lane < nw ? buf[lane] : T(0);
        for (int off = 1; off < 32; off <<= 1) {
            const T t = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += t;
        }
        if (lane < nw) buf[32 + lane] = w;       // inclusive prefix over warps
    }
    __syncthreads();
    const T res = (wid ? buf[32 + wid - 1] : T(0)) + incl - v;
    *total = buf[32 + nw - 1];
    __syncthreads();
    return res;
}

// out_off[c]: exclusive prefix of the output counts of valid circuits, in
// circuit order (one block of 1024 threads).
__global__ void __launch_bounds__(1024) offsets_kernel(const pcv_batch_desc* descs, int n_circ, int64_t* out_off)
{
    __shared__ int64_t buf[64];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < n_circ; b0 += 1024) {
        const int c = b0 + threadIdx.x;
        const int64_t cnt = c < n_circ && desc_ok(descs[c]) ? descs[c].n_out : 0;
        int64_t tot = 0;
        const int64_t ex = block_scan<int64_t>(cnt, buf, &tot);
        if (c < n_circ) out_off[c] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

// Cost of one output in FP64 warp instructions' time (16 cycles of an SM): the
// tile kernel's n - 1 products take about 20 cycles each and the sum's FP64
// instructions overlap them, so 1.25 (n - 1) + 1 per sign vector; Glynn's sum
// with multiplicities spends 2q + 4n - 1 FP64 instructions per term (q
// line-sum updates, n - 1 complex products, the weight and the accumulation).
__device__ double tile_cost(int n) { return ldexp(1.0, n - 1) * (1.25 * (n - 1) + 1.0); }

__device__ double mult_side_cost(const int* mu, int d, int q, int n)
{
    double t = 1.0;
    int odd = -1, big = 0;
    for (int j = 0; j < d; ++j) {
        t *= mu[j] + 1;
        if (odd < 0 && (mu[j] & 1)) odd = j;
        if (mu[j] > mu[big]) big = j;
    }
    const int p = odd >= 0 ? odd : big;
    t = t / (mu[p] + 1) * (mu[p] / 2 + 1);
    return t * (2.0 * q + 4.0 * n - 1.0);
}

// FP64 instructions of output o by Glynn's sum with multiplicities on its
// cheaper side; a negative value for an output outside S_{m,n} (amplitude 0).
__device__ double output_mult_cost(const pcv_batch_desc& c, int64_t o, const int* imu, int d_in)
{
    const uint8_t* occ = c.outputs + o * c.m;
    int omu[PCV_MAX_PHOTONS];
    int d_out = 0, tot = 0;
    for (int r = 0; r < c.m; ++r) {
        const int v = occ[r];
        if (v > 0 && d_out < PCV_MAX_PHOTONS) omu[d_out++] = v;
        tot += v;
    }
    if (tot != c.n) return -1.0;
    return fmin(mult_side_cost(omu, d_out, d_in, c.n), mult_side_cost(imu, d_in, d_out, c.n));
}

// One block per circuit: route each output to the tile kernel or to Glynn's
// sum with multiplicities; idx[out_off[c] ..] lists the tile outputs first
// (in order) and the others after them (in reverse order).  A warp of a tile
// costs as much with one live output as with 32 of them: rest[c] holds what the
// outputs of a last, partly filled warp cost on the multiplicity kernel, all and
// the dearest, and plan_kernel decides about them.
__global__ void __launch_bounds__(256) classify_kernel(const pcv_batch_desc* descs, const int64_t* out_off, int route,
                                                       int64_t cap, int* idx, int* n_tile, int* n_mult, float2* rest)
{
    __shared__ int buf[64];
    __shared__ int s_tile, s_mult;
    const int ci = blockIdx.x;
    const pcv_batch_desc& c = descs[ci];
    const bool valid = desc_ok(c) && out_off[ci] + c.n_out <= cap;
    if (!valid) {
        if (threadIdx.x == 0) {
            n_tile[ci] = n_mult[ci] = 0;
            rest[ci] = make_float2(0.0f, 0.0f);
        }
        return;
    }
    const int n = c.n;
    const int64_t no = c.n_out;
    int* list = idx + out_off[ci];
    // input side: distinct modes and multiplicities
    int imu[PCV_MAX_PHOTONS];
    int d_in = 0;
    for (int j = 0; j < n; ++j) {
        if (j == 0 || c.cols[j] != c.cols[j - 1]) imu[d_in++] = 0;
        imu[d_in - 1] += 1;
    }
    const double ct = tile_cost(n);
    if (threadIdx.x == 0) s_tile = s_mult = 0;
    __syncthreads();
    for (int64_t b0 = 0; b0 < no; b0 += blockDim.x) {
        const int64_t o = b0 + threadIdx.x;
        int to_mult = 0;
        if (o < no) {
            if (route == PCV_ALGO_MULT) {
                to_mult = 1;
            } else if (route == PCV_ALGO_AUTO) {
                const double cm = output_mult_cost(c, o, imu, d_in);
                to_mult = cm < ct;                    // cm < 0: not in S_{m,n}, amplitude 0
            }
        }
        int tot_m = 0;
        const int pm = block_scan<int>(to_mult, buf, &tot_m);
        const int live = o < no ? 1 : 0;
        int tot_t = 0;
        const int pt = block_scan<int>(live - to_mult, buf, &tot_t);
        if (o < no) {
            if (to_mult) list[no - 1 - (s_mult + pm)] = (int)o;
            else list[s_tile + pt] = (int)o;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            s_tile += tot_t;
            s_mult += tot_m;
        }
        __syncthreads();
    }
    if (threadIdx.x < 32) {
        // the last r tile outputs sit just below the multiplicity outputs in the
        // list; moving the boundary re-routes them
        const int r = route == PCV_ALGO_AUTO ? s_tile % kMinTile : 0;
        const float cost = (int)threadIdx.x < r ? (float)output_mult_cost(c, list[s_tile - r + threadIdx.x], imu, d_in) : 0.0f;
        float sum = cost, most = cost;
        for (int off = 16; off > 0; off >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, off);
            most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, off));
        }
        if (threadIdx.x == 0) {
            n_tile[ci] = s_tile;
            n_mult[ci] = s_mult;
            rest[ci] = make_float2(sum, most);
        }
    }
}

// Outputs per tile for `count` outputs: the size with the least work, dead
// lanes and staging included (a staged row sum costs about two thirds of a
// product).
__device__ int pick_tile(int m, int n, int count)
{
    int best = kThreads;
    double least = 0.0;
    for (int T = kThreads; T >= kMinTile; T >>= 1) {
        const double tiles = (double)((count + T - 1) / T);
        const double w = tiles * (T * (double)n + 0.7 * min(m, min(T, count) * n));
        if (T == kThreads || w < least) {
            best = T;
            least = w;
        }
    }
    return best;
}

// Builds both work lists on the device (one block): a counting sort of the
// circuits by n (descending), then tile items and multiplicity entries in
// that order.  A tile's sequence is split in parts so that
// no item holds more than 1 / (kItemsPerSm sms) of all tile work; a part
// keeps at least kPartSteps sign vectors per split, as its start takes some 30 us
// (kLeastSteps everywhere: 31 circuits of 90 outputs, n <= 15, 300 to 400 us), or
// kLeastSteps up to kLightPerSm items per SM (3 circuits of 17 outputs, n = 10:
// 200 to 77 us).
//
// The outputs of a partly filled warp go to the multiplicity kernel when that
// costs less than the warp and takes no longer, each permanent on one warp after
// the tiles are done, than 1/32 of the time of all tiles (kEntryCycles per FP64
// instruction of a lane, kEntryStart at first: n = 10 to 20; a tile product 20
// cycles of an SM).  Decided by the cost alone, 48 circuits of n = 4 to 16 took 4.87
// ms at 100 outputs each (0.91 so), 6.79 at 513 (3.77), and 3.1 at 512.
__global__ void __launch_bounds__(1024) plan_kernel(const pcv_batch_desc* descs, int n_circ, Queue q, MultQueue mq,
                                                    int* order, int* item_off, int* mult_off, int* n_tile, int* n_mult,
                                                    const float2* rest, int* mult_circ, int* mult_out, int max_items,
                                                    int sms)
{
    __shared__ int bucket[PCV_MAX_PHOTONS + 2];
    __shared__ int cursor[PCV_MAX_PHOTONS + 2];
    __shared__ int buf[64];
    __shared__ int64_t buf64[64];
    __shared__ double s_work[32];
    __shared__ float s_total;
    __shared__ int carry_t, carry_m;
    __shared__ int64_t carry_s;
    const int tid = threadIdx.x;
    if (tid < PCV_MAX_PHOTONS + 2) bucket[tid] = 0;
    __syncthreads();
    for (int c = tid; c < n_circ; c += blockDim.x)
        atomicAdd(&bucket[desc_ok(descs[c]) ? descs[c].n : 0], 1);
    // tile sizes and all tile work (n products per lane and sign vector), before
    // and after the partly filled warps' outputs find their kernel; few threads
    // touch FP64, of which an SM issues an instruction per 16 cycles
    auto tile_work = [&] {
        double work = 0.0;
        for (int c = tid; c < n_circ; c += blockDim.x) {
            const int cnt = n_tile[c];
            const int T = cnt > 0 ? pick_tile(descs[c].m, descs[c].n, cnt) : kThreads;
            q.shape[c] = T;
            if (cnt > 0) work += ldexp((double)((cnt + T - 1) / T) * T * descs[c].n, descs[c].n - 1);
        }
        if (tid / 32 * 32 < n_circ)
            for (int off = 16; off > 0; off >>= 1) work += __shfl_xor_sync(0xffffffffu, work, off);
        if ((tid & 31) == 0) s_work[tid >> 5] = work;
        __syncthreads();
        if (tid < 32) {
            work = s_work[tid];
            for (int off = 16; off > 0; off >>= 1) work += __shfl_xor_sync(0xffffffffu, work, off);
            if (tid == 0) s_total = (float)work;
        }
        __syncthreads();
    };
    tile_work();
    const float patience = s_total * (20.0f / 32.0f / 32.0f) / (float)sms;       // cycles
    bool moved = false;
    for (int c = tid; c < n_circ; c += blockDim.x) {
        const float2 r = rest[c];
        if (r.x > 0.0f && kEntryStart + r.y * (kEntryCycles / 32.0f) <= patience && r.x < kMinTile * tile_cost(descs[c].n)) {
            const int cnt = n_tile[c] % kMinTile;
            n_tile[c] -= cnt;
            n_mult[c] += cnt;
            moved = true;
        }
    }
    if (__syncthreads_or(moved)) tile_work();
    if (tid == 0) {
        int acc = 0;
        for (int n = PCV_MAX_PHOTONS; n >= 0; --n) { cursor[n] = acc; acc += bucket[n]; }
        carry_t = carry_m = 0;
        carry_s = 0;
    }
    __syncthreads();
    const float most = s_total / ((float)sms * kItemsPerSm);
    for (int c = tid; c < n_circ; c += blockDim.x) {
        order[atomicAdd(&cursor[desc_ok(descs[c]) ? descs[c].n : 0], 1)] = c;
        int parts = 1;
        if (q.partial && q.n_tile[c] > 0) {
            const int n = descs[c].n;
            const float vectors = ldexpf((float)q.shape[c] / kThreads, n - 1);       // of a split
            const float item = ldexpf((float)(q.shape[c] * n), n - 1) / most;
            parts = (int)fmaxf(1.0f, fmaxf(fminf(vectors / kPartSteps, ceilf(item)),
                                           fminf(vectors / kLeastSteps, item * (kLightPerSm / (float)kItemsPerSm))));       // rounded down: one wave
        }
        q.shape[c] += kPack * parts;
    }
    __syncthreads();
    // exclusive scans of tile items, entries and partial sums over the sorted order
    for (int b0 = 0; b0 < n_circ; b0 += 1024) {
        const int p = b0 + tid;
        int ct = 0, cm = 0;
        int64_t cs = 0;
        if (p < n_circ) {
            const int c = order[p];
            const int T = q.shape[c] % kPack, parts = q.shape[c] / kPack;
            ct = (q.n_tile[c] + T - 1) / T * parts;
            cm = n_mult[c];
            cs = parts > 1 ? (int64_t)q.n_tile[c] * parts : 0;
        }
        int tt = 0, tm = 0;
        int64_t ts = 0;
        const int et = block_scan<int>(ct, buf, &tt);
        const int em = block_scan<int>(cm, buf, &tm);
        const int64_t es = block_scan<int64_t>(cs, buf64, &ts);
        if (p < n_circ) {
            item_off[p] = carry_t + et;
            mult_off[p] = carry_m + em;
            if (q.partial) q.slot_off[order[p]] = carry_s + es;
        }
        __syncthreads();
        if (tid == 0) {
            carry_t += tt;
            carry_m += tm;
            carry_s += ts;
        }
        __syncthreads();
    }
    if (tid == 0) {
        *q.total = carry_t < max_items ? carry_t : max_items;
        *q.counter = 0;
        *mq.total = carry_m;
        *mq.counter = 0;
    }
    __syncthreads();
    // a warp per circuit fills its share of the lists
    const int warp = tid >> 5, lane = tid & 31;
    for (int p = warp; p < n_circ; p += 32) {
        const int c = order[p];
        const int T = q.shape[c] % kPack;
        const int cnt = (q.n_tile[c] + T - 1) / T * (q.shape[c] / kPack);
        for (int t = lane; t < cnt; t += 32) {
            const int it = item_off[p] + t;
            if (it < max_items) {
                q.item_circ[it] = c;
                q.item_tile[it] = t;
                if (q.partial) q.done[it] = 0;
            }
        }
        const int cm = n_mult[c];
        const int* src = q.idx + q.out_off[c] + q.n_tile[c];
        for (int t = lane; t < cm; t += 32) {
            mult_circ[mult_off[p] + t] = c;
            mult_out[mult_off[p] + t] = src[t];
        }
    }
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// The largest block of the persistent kernel.
size_t batch_smem()
{
    size_t b = 0;
    for (int T = kMinTile; T <= kThreads; T *= 2)
        b = std::max(b, tile_smem(PCV_MAX_PHOTONS, kMaxModes, TileShape{T, 1, std::min(kMaxModes, T * PCV_MAX_PHOTONS), kStage}));
    return b;
}

// Tile shape of one circuit (or B unitaries with the same outputs): the tile
// size as the batched planner chooses it, and two blocks per SM (what shared
// memory holds) if the sequences may be split.
TileShape pick_shape(int m, int n, int64_t n_out, int B, bool split)
{
    TileShape t{kThreads, 1, 0, 0};
    double least = 0.0;
    for (int T = kThreads; T >= kMinTile; T >>= 1) {
        const double tiles = (double)((n_out + T - 1) / T);
        const double w = tiles * (T * (double)n + 0.7 * (double)std::min<int64_t>(m, std::min<int64_t>(T, n_out) * n));
        if (T == kThreads || w < least) {
            t.T = T;
            least = w;
        }
    }
    t.slots = (int)std::min<int64_t>(m, (int64_t)t.T * n);
    const int S = kThreads / t.T;
    // the staged sums: up to kMaxChunk steps within 48 KB, one step at least
    t.stage = std::max(std::max(kThreads, S * t.slots), std::min(kStageOne, S * t.slots * kMaxChunk));
    const int64_t tiles = (n_out + t.T - 1) / t.T * B;
    const int64_t room = (1ll << (n - 1)) / ((int64_t)S * kLeastSteps);
    if (split) t.parts = (int)std::max<int64_t>(1, std::min<int64_t>(room, 152 * kLightPerSm / tiles));
    return t;
}

__global__ void store_desc_kernel(const pcv_batch_desc d, pcv_batch_desc* out) { *out = d; }

cudaError_t tile_launch(const pcv_batch_desc& d, int B, const TileShape& sh, double2* partial, cudaStream_t s)
{
    TileLaunch a;
    a.c = d;
    a.sh = sh;
    a.ustride = (int64_t)d.m * d.m;
    a.ostride = d.n_out;
    a.partial = partial;
    const size_t smem = tile_smem(d.n, d.m, sh);
    cudaError_t e = allow_dynamic_smem((const void*)glynn_tile_kernel, smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (d.n_out + sh.T - 1) / sh.T * sh.parts;
    if (blocks > INT32_MAX) return cudaErrorInvalidConfiguration;
    glynn_tile_kernel<<<dim3((unsigned)blocks, (unsigned)B), kThreads, smem, s>>>(a);
    note_launches(1);
    if (sh.parts > 1) {
        tile_parts_kernel<<<(unsigned)((d.n_out + kThreads - 1) / kThreads), kThreads, 0, s>>>(a);
        note_launches(1);
    }
    return cudaGetLastError();
}

}  // namespace

int tile_max_modes() { return kMaxModes; }

cudaError_t launch_store_desc(const pcv_batch_desc& d, pcv_batch_desc* out, cudaStream_t s)
{
    store_desc_kernel<<<1, 1, 0, s>>>(d, out);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_glynn_tile(const pcv_batch_desc& d, cudaStream_t s)
{
    if (d.n_out == 0) return cudaSuccess;
    return tile_launch(d, 1, pick_shape(d.m, d.n, d.n_out, 1, false), nullptr, s);
}

cudaError_t launch_glynn_tile_multi(const pcv_batch_desc& d, int B, cudaStream_t s)
{
    if (d.n_out == 0 || B == 0) return cudaSuccess;
    return tile_launch(d, B, pick_shape(d.m, d.n, d.n_out, B, false), nullptr, s);
}

// The same with the sign vectors of a tile split over blocks; any m whose
// running and staged sums fit in shared memory.
int64_t tile_split_workspace(int m, int n, int64_t n_out)
{
    const TileShape t = pick_shape(m, n, n_out, 1, true);
    if (tile_smem(n, m, t) > 200 * 1024) return -1;
    return t.parts > 1 ? (int64_t)al256((size_t)n_out * t.parts * sizeof(double2)) : 0;
}

cudaError_t launch_glynn_tile_split(const pcv_batch_desc& d, void* ws, cudaStream_t s)
{
    if (d.n_out == 0) return cudaSuccess;
    return tile_launch(d, 1, pick_shape(d.m, d.n, d.n_out, 1, true), (double2*)ws, s);
}

// Workspace of the batched launch: counters, per-circuit arrays, the routed
// output lists and the tile items; then, if there is room, what sequences
// split over several blocks need: more items and the partial sums.  With `most`
// the work per item, a tile of work w is split in at most w / most + 1 parts,
// so there are at most kItemsPerSm sms items more than tiles.
namespace {
constexpr int kPlanSms = 160;          // SMs the plan is sized for
int64_t split_items(int n_circ, int64_t total_outputs)
{
    return (int64_t)kItemsPerSm * kPlanSms + total_outputs / kMinTile + n_circ + 1;
}
int64_t split_slots(int n_circ, int64_t total_outputs)
{
    return ((int64_t)kItemsPerSm * kPlanSms + n_circ) * kThreads + 2 * total_outputs;
}
}  // namespace

int64_t batched_workspace(int n_circ, int64_t total_outputs)
{
    const int64_t max_items = total_outputs / 32 + n_circ + 1;
    return (int64_t)(al256(4 * sizeof(int)) + 6 * al256((size_t)n_circ * sizeof(int)) +
                     al256((size_t)n_circ * sizeof(int64_t)) + 3 * al256((size_t)total_outputs * sizeof(int)) +
                     2 * al256((size_t)max_items * sizeof(int)));
}

int64_t batched_workspace_full(int n_circ, int64_t total_outputs)
{
    return batched_workspace(n_circ, total_outputs) +
           (int64_t)(al256((size_t)n_circ * sizeof(int64_t)) + 3 * al256((size_t)split_items(n_circ, total_outputs) * sizeof(int)) +
                     al256((size_t)split_slots(n_circ, total_outputs) * sizeof(double2)));
}

cudaError_t launch_glynn_batched(const pcv_batch_desc* descs, int n_circ, int64_t total_outputs, void* ws,
                                 int64_t ws_bytes, int sms, int route, cudaStream_t s)
{
    const size_t smem = batch_smem();
    cudaError_t e = allow_dynamic_smem((const void*)glynn_persistent_kernel, smem);
    if (e != cudaSuccess) return e;
    int64_t max_items = total_outputs / 32 + n_circ + 1;
    char* w = (char*)ws;
    int* counters = (int*)w;                          w += al256(4 * sizeof(int));
    int* order = (int*)w;                             w += al256((size_t)n_circ * sizeof(int));
    int* item_off = (int*)w;                          w += al256((size_t)n_circ * sizeof(int));
    int* mult_off = (int*)w;                          w += al256((size_t)n_circ * sizeof(int));
    int* n_tile = (int*)w;                            w += al256((size_t)n_circ * sizeof(int));
    int* n_mult = (int*)w;                            w += al256((size_t)n_circ * sizeof(int));
    int* shapes = (int*)w;                            w += al256((size_t)n_circ * sizeof(int));
    int64_t* out_off = (int64_t*)w;                   w += al256((size_t)n_circ * sizeof(int64_t));
    int* idx = (int*)w;                               w += al256((size_t)total_outputs * sizeof(int));
    int* mult_circ = (int*)w;                         w += al256((size_t)total_outputs * sizeof(int));
    int* mult_out = (int*)w;                          w += al256((size_t)total_outputs * sizeof(int));
    int* item_circ = (int*)w;                         w += al256((size_t)max_items * sizeof(int));
    int* item_tile = (int*)w;                         w += al256((size_t)max_items * sizeof(int));
    Queue q;
    q.counter = counters;
    q.total = counters + 1;
    q.item_circ = item_circ;
    q.item_tile = item_tile;
    q.out_off = out_off;
    q.n_tile = n_tile;
    q.idx = idx;
    q.shape = shapes;
    q.slot_off = nullptr;
    q.partial = nullptr;
    q.done = nullptr;
    if (ws_bytes >= batched_workspace_full(n_circ, total_outputs) && sms <= kPlanSms) {
        max_items = split_items(n_circ, total_outputs);
        q.slot_off = (int64_t*)w;                     w += al256((size_t)n_circ * sizeof(int64_t));
        q.item_circ = (int*)w;                        w += al256((size_t)max_items * sizeof(int));
        q.item_tile = (int*)w;                        w += al256((size_t)max_items * sizeof(int));
        q.done = (int*)w;                             w += al256((size_t)max_items * sizeof(int));
        q.partial = (double2*)w;
    }
    MultQueue mq;
    mq.counter = counters + 2;
    mq.total = counters + 3;
    mq.circ = mult_circ;
    mq.out = mult_out;

    offsets_kernel<<<1, 1024, 0, s>>>(descs, n_circ, out_off);
    // the lists that plan_kernel fills last hold its input until then
    float2* rest = (float2*)item_off;
    classify_kernel<<<n_circ, 256, 0, s>>>(descs, out_off, route, total_outputs, idx, n_tile, n_mult, rest);
    plan_kernel<<<1, 1024, 0, s>>>(descs, n_circ, q, mq, order, item_off, mult_off, n_tile, n_mult, rest, mult_circ,
                                   mult_out, (int)max_items, sms);
    note_launches(3);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, glynn_persistent_kernel, kThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    glynn_persistent_kernel<<<sms * per_sm, kThreads, smem, s>>>(descs, q);
    note_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_glynn_mult_persistent(descs, mq, sms, s);
}

}  // namespace pcv
