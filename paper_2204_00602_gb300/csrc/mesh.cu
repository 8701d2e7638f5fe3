// Clements rectangular MZI mesh: U(phi) and the reverse-mode gradient of a
// real loss with respect to the phases, for a batch of phase sets.
//
// Components (Sec. 2, Eq. bs; the MZI of the Boson-sampling code in Sec. 4.2):
// BS = Rx(theta = pi/2) = (1/sqrt2) [[1, i], [i, 1]] and
//     MZI(phi_a, phi_b) = diag(1, e^{i phi_b}) . BS . diag(e^{i phi_a}, 1) . BS
//                       = diag(1, e^{i phi_b}) . 1/2 [[e - 1, i(e + 1)], [i(e + 1), 1 - e]],  e = e^{i phi_a}.
// Layout (Sec. 2 cites the square decomposition of Clements et al.): m
// columns; column c holds MZIs on modes (k, k+1) for k = c mod 2, c mod 2 + 2,
// ... < m-1, in that order; MZI q uses phases[2q], phases[2q+1].  Later
// components multiply on the left, so U = M_Q ... M_1.
//
// The MZIs of one column act on disjoint pairs of modes, so a phase set takes
// m column steps, not m(m-1)/2 MZI steps.  One block per phase set: all sines
// and cosines first, one phase per thread (FP64 sincos costs tens of FP64
// instructions; formed per MZI by every lane of a warp it was most of the
// time), then a thread per (MZI of the column, column of U) and one barrier
// per step.  U, and in the reverse sweep dL/dU, live in shared memory.
// Measured at m = 12 (before: one warp per phase set, one MZI at a time):
// forward of 64 / 2048 sets 206 / 739 -> 14 / 98 us, backward of 64 sets 569
// -> 31 us.

#include <algorithm>

#include "pcv_common.cuh"

namespace pcv {
namespace {

constexpr int kMaxMeshModes = 64;

__device__ __forceinline__ double2 cexp_i(double phi)
{
    double s, c;
    sincos(phi, &s, &c);
    return make_double2(c, s);
}

__device__ __forceinline__ double2 conj2(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 mul_i(double2 a) { return make_double2(-a.y, a.x); }
__device__ __forceinline__ double2 scale2(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

// Column c: first MZI and number of MZIs.
__device__ __forceinline__ int col_first(int m, int c) { return (c >> 1) * (m - 1) + (c & 1) * (m / 2); }
__device__ __forceinline__ int col_size(int m, int c) { return (c & 1) ? (m - 1) / 2 : m / 2; }

__global__ void mesh_forward_kernel(const double* __restrict__ phases, int m, int nq, double2* __restrict__ Uout)
{
    extern __shared__ double2 sU[];          // [m][m], then the MZIs [nq][4]
    double2* sT = sU + m * m;
    const int b = blockIdx.x;
    const double* ph = phases + (size_t)b * 2 * nq;
    for (int i = threadIdx.x; i < m * m; i += blockDim.x)
        sU[i] = make_double2((i / m) == (i % m) ? 1.0 : 0.0, 0.0);
    for (int q = threadIdx.x; q < 2 * nq; q += blockDim.x) sT[2 * q] = cexp_i(ph[q]);   // e at 4q, f at 4q + 2
    __syncthreads();
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
        const double2 e = sT[4 * q], f = sT[4 * q + 2];
        const double2 t00 = scale2(make_double2(e.x - 1.0, e.y), 0.5);
        const double2 t01 = scale2(mul_i(make_double2(e.x + 1.0, e.y)), 0.5);
        sT[4 * q] = t00;
        sT[4 * q + 1] = t01;
        sT[4 * q + 2] = cmul(f, t01);
        sT[4 * q + 3] = cmul(f, scale2(make_double2(1.0 - e.x, -e.y), 0.5));
    }
    for (int c = 0; c < m; ++c) {
        __syncthreads();
        const int q0 = col_first(m, c), nc = col_size(m, c);
        for (int i = threadIdx.x; i < nc * m; i += blockDim.x) {
            const int u = i / m, j = i % m, k = (c & 1) + 2 * u;
            const double2* t = sT + 4 * (q0 + u);
            const double2 u0 = sU[k * m + j], u1 = sU[(k + 1) * m + j];
            sU[k * m + j] = cadd(cmul(t[0], u0), cmul(t[1], u1));
            sU[(k + 1) * m + j] = cadd(cmul(t[2], u0), cmul(t[3], u1));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m * m; i += blockDim.x) Uout[(size_t)b * m * m + i] = sU[i];
}

// Reverse sweep, column by column: the state after a column is undone with
// the MZIs' inverses and the gradient pulled back with their adjoints (the
// same matrices, MZIs being unitary), through the four factors one at a time.
// With u the rows after the MZI and h the gradient there,
//     dL/dphi_b = sum_j Im-part of conj(i u_1) h_1 = sum_j u_1.x h_1.y - u_1.y h_1.x,
// and after undoing diag(1, e^{i phi_b}) and one BS, with w_0, y_0 the upper
// rows just behind diag(e^{i phi_a}, 1),
//     dL/dphi_a = sum_j w_0.x y_0.y - w_0.y y_0.x.
// So an MZI needs two real sums over the columns of U; a column step leaves
// the terms in shared memory and one thread per phase adds them in order.  BS^H = (1/sqrt2) [[1, -i], [-i, 1]];
// the two factors 1/sqrt2 are applied as one 1/2.
__global__ void mesh_backward_kernel(const double* __restrict__ phases, int m, int nq, const double2* __restrict__ U,
                                     const double2* __restrict__ G, double* __restrict__ gphi)
{
    extern __shared__ double2 sh[];
    double2* sU = sh;                        // [m][m] current state
    double2* sG = sh + m * m;                // [m][m] current gradient
    double2* sE = sG + m * m;                // [nq][2]: e^{i phi_a}, e^{i phi_b}
    double* red = (double*)(sE + 2 * nq);    // [2][m/2][m]: terms of dL/dphi_a, dL/dphi_b
    const int b = blockIdx.x, half = (m / 2) * m;
    const double* ph = phases + (size_t)b * 2 * nq;
    for (int i = threadIdx.x; i < m * m; i += blockDim.x) {
        sU[i] = U[(size_t)b * m * m + i];
        sG[i] = G[(size_t)b * m * m + i];
    }
    for (int q = threadIdx.x; q < 2 * nq; q += blockDim.x) sE[q] = cexp_i(ph[q]);
    for (int c = m - 1; c >= 0; --c) {
        __syncthreads();
        const int q0 = col_first(m, c), nc = col_size(m, c);
        for (int i = threadIdx.x; i < nc * m; i += blockDim.x) {
            const int u = i / m, j = i % m, k = (c & 1) + 2 * u;
            const double2 e = conj2(sE[2 * (q0 + u)]), f = conj2(sE[2 * (q0 + u) + 1]);
            const double2 u0 = sU[k * m + j], u1 = sU[(k + 1) * m + j];
            const double2 h0 = sG[k * m + j], h1 = sG[(k + 1) * m + j];
            red[half + i] = fma(u1.x, h1.y, -(u1.y * h1.x));
            const double2 v1 = cmul(f, u1), g1 = cmul(f, h1);
            // BS^H, without the 1/sqrt2: (a, b) -> (a - i b, b - i a)
            const double2 w0 = make_double2(u0.x + v1.y, u0.y - v1.x), w1 = make_double2(v1.x + u0.y, v1.y - u0.x);
            const double2 y0 = make_double2(h0.x + g1.y, h0.y - g1.x), y1 = make_double2(g1.x + h0.y, g1.y - h0.x);
            red[i] = 0.5 * fma(w0.x, y0.y, -(w0.y * y0.x));
            const double2 a0 = cmul(e, w0), b0 = cmul(e, y0);
            sU[k * m + j] = make_double2(0.5 * (a0.x + w1.y), 0.5 * (a0.y - w1.x));
            sU[(k + 1) * m + j] = make_double2(0.5 * (w1.x + a0.y), 0.5 * (w1.y - a0.x));
            sG[k * m + j] = make_double2(0.5 * (b0.x + y1.y), 0.5 * (b0.y - y1.x));
            sG[(k + 1) * m + j] = make_double2(0.5 * (y1.x + b0.y), 0.5 * (y1.y - b0.x));
        }
        __syncthreads();
        for (int p = threadIdx.x; p < 2 * nc; p += blockDim.x) {
            const double* r = red + (p & 1) * half + (p >> 1) * m;
            double v = r[0];
            for (int j = 1; j < m; ++j) v += r[j];
            gphi[(size_t)b * 2 * nq + 2 * q0 + p] = v;
        }
    }
}

// Threads of a block: one per (MZI, column of U) of a column step, at most 256.
int mesh_threads(int m) { return std::min(256, ((m / 2) * m + 31) / 32 * 32); }

}  // namespace

int mesh_max_modes() { return kMaxMeshModes; }

cudaError_t launch_mesh_forward(const double* phases, int B, int m, double2* U, cudaStream_t s)
{
    const int nq = m * (m - 1) / 2;
    const size_t smem = ((size_t)m * m + 4 * nq) * sizeof(double2);
    const cudaError_t e = allow_dynamic_smem((const void*)mesh_forward_kernel, smem);
    if (e != cudaSuccess) return e;
    mesh_forward_kernel<<<B, mesh_threads(m), smem, s>>>(phases, m, nq, U);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_mesh_backward(const double* phases, int B, int m, const double2* U, const double2* G,
                                 double* gphi, cudaStream_t s)
{
    const int nq = m * (m - 1) / 2;
    const size_t smem = ((size_t)2 * m * m + 2 * nq) * sizeof(double2) + (size_t)2 * (m / 2) * m * sizeof(double);
    const cudaError_t e = allow_dynamic_smem((const void*)mesh_backward_kernel, smem);
    if (e != cudaSuccess) return e;
    mesh_backward_kernel<<<B, mesh_threads(m), smem, s>>>(phases, m, nq, U, G, gphi);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace pcv
