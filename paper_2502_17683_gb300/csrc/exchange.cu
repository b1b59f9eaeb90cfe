// The CPD+THC LT-MP2 exchange energy (Sec. 2.2): the consumer of the CPD factors that ALS
// produces. Per Laplace quadrature point alpha (Eq. lt_D, factors Lam (occupied) and Gam
// (virtual) of Eq. mp1_t):
//   single CPD (Eq. cpd_single_k):  U1 = (Lam o Xo)^T A1, U3 = (Lam o Xo)^T A3,
//       U2 = (Gam o Xv)^T A2, U4 = (Gam o Xv)^T A4, Y = Z (U3 o U2),
//       E_single = - sum_{P,r} lam_r U1[P,r] U4[P,r] Y[P,r]             O(R_thc^2 R)
//   double CPD:  M1 = A1^T diag(Lam) A1, M3 = A3^T diag(Lam) A3, N = A2^T diag(Gam) A4,
//       E_double = - lam^T (M1 o N o M3 o N^T) lam                       O(N R^2)
//   robust (Eq. rob_K):  E_robust = 2 E_single - E_double (no first-order CPD error).
// The quadrature points are independent, so a group of them (as many as 1 GB of intermediates
// holds) goes through every step as one product over the stacked points, (alpha, P) as rows of U and
// (alpha, r) as columns of Y, M1, M3 and N: 20 launches for all points instead of 20 for each. At
// (o, v, R_thc, R_cp) = (20, 100, 480, 720) with 12 points a product per point fills a fraction of
// the SMs (12 us for 14 to 70 MFLOP).
// The products run on the FP64 pipes or, from a size on (oz_worth, of a whole group) or on request,
// as the FP64-accurate products of the BF16 tensor cores; the reductions are fixed-order.
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <vector>

#include "f64.cuh"
#include "oz.cuh"
#include "prof.cuh"
#include "thc_cpd.h"

namespace thc {
namespace {

constexpr int XR_THREADS = 256;
constexpr int XR_BLOCKS = 304;

__device__ double xr_block_sum(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
    if (w == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    return v;
}

// out[r][al n + c] = s[al rows + r] X[r][c] for al < g: the rows scaled by the factors of g points,
// the points' results side by side
__global__ void k_scale_rows(int rows, int n, int g, const double* __restrict__ s, const double* __restrict__ X,
                             double* __restrict__ out) {
    const long total = (long)rows * g * n;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
        const int c = (int)(e % n);
        const long t = e / n;
        const int al = (int)(t % g), r = (int)(t / g);
        out[e] = s[(size_t)al * rows + r] * X[(size_t)r * n + c];
    }
}

// partial sums of lam_r U1 U4 Y over the Rt x R grid of point blockIdx.y (U: its Rt x R block, Y: its
// R columns of g R; one per block, fixed order)
__global__ void __launch_bounds__(XR_THREADS)
k_single_partials(int Rt, int R, int g, const double* __restrict__ U1, const double* __restrict__ U4,
                  const double* __restrict__ Y, const double* __restrict__ lam, double* __restrict__ part) {
    __shared__ double sh[32];
    const long n = (long)Rt * R;
    const size_t off = (size_t)blockIdx.y * n, gR = (size_t)g * R;
    U1 += off;
    U4 += off;
    Y += (size_t)blockIdx.y * R;
    double s = 0.0;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
        const int P = (int)(e / R), r = (int)(e % R);
        s = fma(lam[r] * U1[e], U4[e] * Y[P * gR + r], s);
    }
    s = xr_block_sum(s, sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * XR_BLOCKS + blockIdx.x] = s;
}

// partial sums of lam_r lam_s M1[r,s] N[r,s] M3[r,s] N[s,r] of point blockIdx.y (its R columns of
// g R) over 32 x 32 tiles (N^T through shared memory so that both reads are coalesced)
__global__ void __launch_bounds__(XR_THREADS)
k_double_partials(int R, int g, const double* __restrict__ M1, const double* __restrict__ N,
                  const double* __restrict__ M3, const double* __restrict__ lam, double* __restrict__ part) {
    __shared__ double nt[32][33];
    __shared__ double sh[32];
    const size_t ld = (size_t)g * R, off = (size_t)blockIdx.y * R;
    M1 += off;
    M3 += off;
    N += off;
    const int tiles = (R + 31) / 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
    double s = 0.0;
    for (int t = blockIdx.x; t < tiles * tiles; t += gridDim.x) {
        const int r0 = (t / tiles) * 32, c0 = (t % tiles) * 32;
        __syncthreads();
        for (int k = ty; k < 32; k += 8) {  // nt[k][tx] = N[c0 + k][r0 + tx]
            const int rr = c0 + k, cc = r0 + tx;
            nt[k][tx] = (rr < R && cc < R) ? N[rr * ld + cc] : 0.0;
        }
        __syncthreads();
        for (int k = ty; k < 32; k += 8) {
            const int r = r0 + k, c = c0 + tx;
            if (r < R && c < R) {
                const size_t e = r * ld + c;
                s = fma(lam[r] * lam[c], M1[e] * N[e] * M3[e] * nt[tx][k], s);
            }
        }
    }
    s = xr_block_sum(s, sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * XR_BLOCKS + blockIdx.x] = s;
}

// out[2 al + slot] = -sum of point al's partials (block al, fixed order)
__global__ void __launch_bounds__(XR_THREADS)
k_neg_final(const double* __restrict__ part, int nb, double* __restrict__ out) {
    __shared__ double sh[32];
    part += (size_t)blockIdx.x * nb;
    double s = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) s += part[i];
    s = xr_block_sum(s, sh);
    if (threadIdx.x == 0) out[2 * blockIdx.x] = -s;
}

thc_cpd_status xerr(thc_cpd_status s, const char* m) { return (thc_cpd_status)set_error(s, m); }

}  // namespace
}  // namespace thc

extern "C" thc_cpd_status thc_cpd_exchange(int o, int v, int Rt, int R, int nalpha, const double* Xo,
                                           const double* Xv, const double* Z, const double* const A[4],
                                           const double* lam, const double* Lam, const double* Gam,
                                           double* e_single, double* e_double, double* e_robust,
                                           const thc_cpd_opts* opts) {
    using namespace thc;
    const int chk = check_problem_args(o, v, Rt, R, Xo, Xv, Z, A);
    if (chk != THC_CPD_OK) return (thc_cpd_status)chk;
    if (nalpha < 1 || nalpha > 1024) return xerr(THC_CPD_ERR_SHAPE, "need 1 <= nalpha <= 1024");
    if (!lam || !Lam || !Gam) return xerr(THC_CPD_ERR_ARG, "lam, Lam and Gam must be non-null");
    cudaStream_t st = opts ? (cudaStream_t)opts->stream : (cudaStream_t)0;
    const size_t RtR = (size_t)Rt * R, RR = (size_t)R * R;
    const int nmax = std::max(o, v);
    // points per group: at most 1 GB of intermediates, and 32-bit extents of the stacked products
    const size_t per = 8 * (5 * RtR + 3 * RR + (size_t)(o + v) * (Rt + R) + (size_t)o * R) + 16 * ((size_t)cdiv(Rt, 128) * 128 * R);
    int g = (int)std::min<size_t>(nalpha, std::max<size_t>(1, (size_t(1) << 30) / per));
    while (g > 1 && ((long)g * std::max(Rt, R) * std::max(std::max(Rt, R), nmax) >= 0x7fffffffL)) --g;
    // products from digits: all on request, else those of a group that are faster there
    bool ozd = oz_available() && !fp64_pipes(opts) && Rt <= 8192 && R <= 8192 && nmax <= 8192;
    bool tc_z, tc_u[2], tc_m, tc_n, emu;
    size_t part_cap, bytes;
    void* block = nullptr;
    // where a group's block does not fit, half the points, at last one without digits: what one point
    // takes on the FP64 pipes is what the call needs
    for (;;) {
        const bool all = ozd && opts && opts->ldl == THC_CPD_LDL_EMULATED;
        auto on_tc = [&](int M, int N, int K) { return all || (ozd && oz_worth_flops(2.0 * g * M * (double)N * K)); };
        tc_z = on_tc(Rt, R, Rt);
        tc_u[0] = on_tc(Rt, R, o);
        tc_u[1] = on_tc(Rt, R, v);
        tc_m = on_tc(R, R, o);
        tc_n = on_tc(R, R, v);
        emu = tc_z || tc_u[0] || tc_u[1] || tc_m || tc_n;
        part_cap = std::max(dgemm_part_need(Rt, R, Rt),
                            std::max(dgemm_part_need(g * Rt, R, nmax), dgemm_part_need(R, g * R, nmax)));
        bytes = Arena::need<double>((size_t)o * g * Rt) + Arena::need<double>((size_t)v * g * Rt) +
                5 * Arena::need<double>(g * RtR) + 2 * Arena::need<double>((size_t)o * g * R) +
                Arena::need<double>((size_t)v * g * R) + 3 * Arena::need<double>(g * RR) +
                Arena::need<double>((size_t)XR_BLOCKS * g) + Arena::need<double>(2 * (size_t)nalpha) +
                Arena::need<double>(part_cap);
        if (emu)
            bytes += 2 * ozmat_bytes(R, o) + 2 * ozmat_bytes(R, v) + ozmat_bytes(g * Rt, o) + ozmat_bytes(g * Rt, v) +
                     ozmat_bytes(Rt, Rt) + ozmat_bytes(g * R, Rt) + ozmat_bytes(g * R, nmax);
        if (alloc_block(&block, bytes, st)) break;
        if (g == 1 && !ozd) return xerr(THC_CPD_ERR_ALLOC, "workspace allocation failed");
        if (g == 1)
            ozd = false;
        else
            g = (g + 1) / 2;
    }
    Arena ar;
    ar.base = (char*)block;
    ar.cap = bytes;
    double* XoL = ar.take<double>((size_t)o * g * Rt);
    double* XvG = ar.take<double>((size_t)v * g * Rt);
    double* U[4];
    for (int k = 0; k < 4; ++k) U[k] = ar.take<double>(g * RtR);
    double* Y = ar.take<double>(g * RtR);
    double* A1L = ar.take<double>((size_t)o * g * R);
    double* A3L = ar.take<double>((size_t)o * g * R);
    double* A4G = ar.take<double>((size_t)v * g * R);
    double* M1 = ar.take<double>(g * RR);
    double* M3 = ar.take<double>(g * RR);
    double* N = ar.take<double>(g * RR);
    double* part = ar.take<double>((size_t)XR_BLOCKS * g);
    double* res = ar.take<double>(2 * (size_t)nalpha);
    double* gpart = ar.take<double>(part_cap);
    OzMat dA[4], dX[2], dZ, dP, dS;
    if (emu) {
        for (int k = 0; k < 4; ++k) ozmat_carve(dA[k], ar, R, (k & 1) ? v : o);
        ozmat_carve(dX[0], ar, g * Rt, o);
        ozmat_carve(dX[1], ar, g * Rt, v);
        ozmat_carve(dZ, ar, Rt, Rt);
        ozmat_carve(dP, ar, g * R, Rt);
        ozmat_carve(dS, ar, g * R, nmax);
        // the digits of what no point changes
        for (int k = 0; k < 4; ++k)
            if (tc_u[k & 1] || ((k & 1) ? (tc_n && k == 1) : tc_m)) oz_split_cols(st, A[k], nullptr, R, dA[k]);
        if (tc_z) oz_split_rows(st, Z, Rt, dZ);
    }
    cudaError_t e = cudaSuccess;  // the first failure (a launcher that reports one has cleared CUDA's record of it)
    auto ck = [&](cudaError_t x) {
        if (e == cudaSuccess) e = x;
    };
    auto scale = [&](int rows, int n, int gg, const double* s, const double* X, double* out) {
        const long total = (long)rows * n * gg;
        k_scale_rows<<<(int)std::min<long>(cdiv(total, 256), 4L * num_sms()), 256, 0, st>>>(rows, n, gg, s, X, out);
        count_launch();
    };
    {
        ProfScope prof(st, emu ? KC_OZ : KC_DGEMM,
                       (double)nalpha * (4.0 * (o + v) * RtR + 2.0 * Rt * RtR + (4.0 * o + 2.0 * v) * RR));
        for (int a0 = 0; a0 < nalpha; a0 += g) {
            const int gg = std::min(g, nalpha - a0), gRt = gg * Rt, gR = gg * R;
            const double* lA = Lam + (size_t)a0 * o;
            const double* gA = Gam + (size_t)a0 * v;
            // single CPD: U1, U3 from Lam o Xo, U2, U4 from Gam o Xv, Y = Z (U3 o U2)
            for (int h = 0; h < 2; ++h) {
                const int n = h ? v : o;
                double* XS = h ? XvG : XoL;
                scale(n, Rt, gg, h ? gA : lA, h ? Xv : Xo, XS);
                OzMat d = dX[h];
                d.rows = gRt;
                if (tc_u[h]) oz_split_cols(st, XS, nullptr, gRt, d);
                for (int k = h; k < 4; k += 2) {
                    if (tc_u[h])
                        ck(oz_mul(st, d, dA[k], U[k], R, 1.0, 0));
                    else
                        dgemm(st, true, gRt, R, n, XS, gRt, A[k], nullptr, R, U[k], R, nullptr, false, gpart, part_cap);
                }
            }
            if (tc_z) {
                OzMat d = dP;
                d.rows = gR;
                oz_split_cols_stack(st, U[2], U[1], R, R, gg, d);
                ck(oz_mul(st, dZ, d, Y, gR, 1.0, 0));
            } else {
                for (int al = 0; al < gg; ++al)
                    dgemm(st, false, Rt, R, Rt, Z, Rt, U[2] + al * RtR, U[1] + al * RtR, R, Y + (size_t)al * R, gR,
                          nullptr, false, gpart, part_cap);
            }
            k_single_partials<<<dim3(XR_BLOCKS, gg), XR_THREADS, 0, st>>>(Rt, R, gg, U[0], U[3], Y, lam, part);
            k_neg_final<<<gg, XR_THREADS, 0, st>>>(part, XR_BLOCKS, res + 2 * a0);
            // double CPD: M1 = A1^T (Lam o A1), M3 = A3^T (Lam o A3), N = A2^T (Gam o A4)
            auto pair = [&](const double* Al, const OzMat& dl, const double* As, const double* s, int n, double* AS,
                            double* out, bool tc) {
                scale(n, R, gg, s, As, AS);
                if (tc) {
                    OzMat d = dS;
                    d.rows = gR;
                    d.K = n;
                    oz_split_cols(st, AS, nullptr, gR, d);
                    ck(oz_mul(st, dl, d, out, gR, 1.0, 0));
                } else {
                    dgemm(st, true, R, gR, n, Al, R, AS, nullptr, gR, out, gR, nullptr, false, gpart, part_cap);
                }
            };
            pair(A[0], dA[0], A[0], lA, o, A1L, M1, tc_m);
            pair(A[2], dA[2], A[2], lA, o, A3L, M3, tc_m);
            pair(A[1], dA[1], A[3], gA, v, A4G, N, tc_n);
            k_double_partials<<<dim3(XR_BLOCKS, gg), XR_THREADS, 0, st>>>(R, gg, M1, N, M3, lam, part);
            k_neg_final<<<gg, XR_THREADS, 0, st>>>(part, XR_BLOCKS, res + 2 * a0 + 1);
            count_launch(4);
        }
    }
    std::vector<double> h(2 * (size_t)nalpha);
    ck(cudaGetLastError());
    ck(cudaMemcpyAsync(h.data(), res, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, st));
    ck(cudaStreamSynchronize(st));
    // freed after the synchronisation, which gives what the pool holds unused back to the device: the
    // next call finds the block in the pool (mapping 650 MB anew took 1.9 ms)
    cudaFreeAsync(block, st);
    if (e != cudaSuccess) {
        char msg[256];
        snprintf(msg, sizeof msg, "exchange energy failed: %s", cudaGetErrorString(e));
        return xerr(THC_CPD_ERR_CUDA, msg);
    }
    if (emu) {
        if (int te = oz_take_error()) {
            char msg[128];
            snprintf(msg, sizeof msg, "emulated-product kernel wait gave up (code %d)", te);
            return xerr(THC_CPD_ERR_TIMEOUT, msg);
        }
    }
    double e1 = 0.0, e2 = 0.0;
    for (int al = 0; al < nalpha; ++al) {
        e1 += h[2 * al];
        e2 += h[2 * al + 1];
    }
    if (!isfinite(e1) || !isfinite(e2)) return xerr(THC_CPD_ERR_NONFINITE, "exchange energy is not finite");
    if (e_single) *e_single = e1;
    if (e_double) *e_double = e2;
    if (e_robust) *e_robust = 2.0 * e1 - e2;
    return THC_CPD_OK;
}
