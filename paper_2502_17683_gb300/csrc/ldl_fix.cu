// LDL^T of the normal matrix in blocks of 128 columns, for matrices whose FP64 pivot chain
// would otherwise run on the FP64 pipe: a one-CTA kernel factorises the diagonal block and a
// second kernel substitutes every row below it, both in 64-bit fixed point on the integer
// pipe; the trailing update is an emulated product on the tensor cores (oz_gemm.cu) from the
// digits that the second kernel leaves behind.
//
// Why fixed point: GB300 issues one FP64 warp-instruction per SM sub-partition every 64 clocks
// (latency the same; two FMA per clock and SM), so problems that share the GPU queue for its FP64
// pipes. A 62-bit multiply-add on the integer pipe is ~12 instructions of 32 bits (~45 clocks per
// warp), runs beside the FP64 work of others, and a one-CTA kernel of it carries a pivot column in
// ~500 clocks (a dataflow panel ~1300 on its four kinds of CTA, ldl_flow.cu). Measured: 12 problems
// of R = 144 .. 1080, two sweeps: 35.6 ms with the blocked FP64 kernels, 22.8 ms with these from
// R = 400 on. Alone, a solve takes 155 us at R = 80 (15 rows; the dataflow kernel 149) and 1.33 ms at
// R = 1080 (dataflow panels with emulated updates 1.21): the chain of one CTA (67 us per 128
// columns, half of it the block's own trailing update) bounds it, so it runs in batches only.
// Accuracy: the block is scaled symmetrically by powers of two so that its diagonal lies in
// [1/4, 1): every entry of a positive definite matrix and of its Schur complements is then below 1
// in magnitude. All quantities are held with 62 fraction bits (l = x' / d' <= 2: 61); each product
// is rounded there and each multi-term update at 2^-58, against the 2^-53 relative rounding of every
// FP64 operation on numbers of the same size (backward errors measured equal to the dataflow
// kernel's, 2e-16 .. 9e-16 for R = 80 .. 1800). A value that leaves its range proves that the matrix
// is not positive definite (rows of H) and sets the failed-pivot bit; an appended row (M) is then
// done again with a larger exponent, and sets the bit once no larger one is left.
//
// With A = S A' S (S the diagonal of 2^e), A' = C C^T, the rows' digits are those of C; the result
// is left in the layout of the other factorisations:
// L (unit lower) and D in H, D^-1 in dinv, Y = M L^-T D^-1 in the appended rows.
#include <float.h>

#include <algorithm>

#include "f64.cuh"
#include "fixed.cuh"
#include "ldl_common.cuh"
#include "oz.cuh"
#include "prof.cuh"

namespace thc {

namespace {

constexpr int NB = kOzPanel;   // 128 columns per block
constexpr int TB = 16;         // tile
constexpr int NT = NB / TB;    // tiles per side
constexpr int TP = TB + 1;     // tile row pitch (conflict-free row accesses)
constexpr int kOff = NT * (NT - 1) / 2;
constexpr int kDiagWarps = 16;
constexpr int kPanelWarps = 4;  // two rows each

// What the row kernel reads of a factorised block.
struct BlockTab {
    int2 ct[kOff][TB][TB];   // l(16 tr + i, 16 tq + q), tr > tq: [tr (tr - 1) / 2 + tq][q][i], 29-bit limbs
    int2 ls[NT][TB][TB];     // -l(16 t + i, 16 t + q): [t][q][i], 31-bit halves
    long long rs[NB];        // 1 / sqrt(d') in Q61, d' = d 4^k in [1/4, 1)
    int k[NB];
    int e[NB];               // scaling exponents
};
static_assert(sizeof(BlockTab) % 16 == 0, "copied in 16-byte pieces");

struct DiagSmem {
    long long T[NT * (NT + 1) / 2][TB * TP];  // lower tiles (tr, tc) at tr (tr + 1) / 2 + tc: Q62, l (Q61) when finished
    int2 xl[2][TB][NB];      // limbs of the panel's x' and l, [panel & 1][column][row]
    int2 ll[2][TB][NB];
    int2 xs[TB][TB];         // the diagonal tile's x' as they are finished, [column][row], 31-bit halves
    long long inv[NB], dq[NB];
    long long dg[NB];        // what is left of each row's diagonal entry (Q61, to about 2^-22), plus kDiagSlack
    int k[NB], e[NB];
    int bad;
    volatile int done;       // columns finished by the chain warp
};

struct PanelSmem {
    BlockTab tab;
    int2 xl[kPanelWarps][2][NB];
    long long yq[kPanelWarps][2][NB];
};

// a = x 2^31 + y, 0 <= y < 2^31 (|a| < 2^62)
__device__ __forceinline__ int2 split31(long long a) {
    return make_int2((int)(a >> 31), (int)(a & 0x7FFFFFFFLL));
}

// a ~ (x 2^29 + y) 2^4 with |y| <= 2^28: limbs whose products can be summed 16 times in 64 bits
__device__ __forceinline__ int2 split29(long long a) {
    const long long v = (a + 8) >> 4;
    const int x = (int)((v + (1LL << 28)) >> 29);
    return make_int2(x, (int)(v - ((long long)x << 29)));
}

// 32 x 32 -> 64 multiply(-add)
__device__ __forceinline__ long long mulw(int a, int b) {
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ long long madw(int a, int b, long long c) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// (a b) 2^-62 and 2^-61 of 31-bit halves. The low product (below one unit) is left out; the
// constants round to nearest and stand for its mean, so that the errors of a sum do not add up
// (a zero factor gives 0).
__device__ __forceinline__ long long mul62(int2 a, int2 b) {
    return mulw(a.x, b.x) + (madw(a.x, b.y, madw(a.y, b.x, 3LL << 29)) >> 31);
}
__device__ __forceinline__ long long mul61(int2 a, int2 b) {
    return (mulw(a.x, b.x) << 1) + (madw(a.x, b.y, madw(a.y, b.x, (1LL << 30) - 1)) >> 30);
}

__device__ __forceinline__ long long shfl64(long long v, int src) {
    return __shfl_sync(0xffffffffu, v, src);
}

// |a| >= 2^bits
__device__ __forceinline__ bool beyond(long long a, int bits) {
    const long long t = a >> bits;
    return ((t + 1) >> 1) != 0;
}

// 1 / sqrt(d 4^k) in Q61 for d > 0 in Q62, with k such that d 4^k lies in [1/4, 1): the
// hardware's 23-bit single-precision estimate refined by one third-order step
// y (1 + e/2 + 3 e^2 / 8), e = 1 - d' y^2, in integer arithmetic (relative error below 2^-60).
__device__ __forceinline__ long long rsqrt_fix(long long d, int& k) {
    const int lz = __clzll(d);  // >= 1
    k = (lz - 2) >> 1;
    const unsigned long long dp = (unsigned long long)d << (2 * k);
    const unsigned mant = (unsigned)(((unsigned long long)d << lz) >> 40) & 0x7FFFFFu;
    const float f = __uint_as_float(((unsigned)(126 - (lz & 1)) << 23) | mant);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    const unsigned b = __float_as_uint(y);
    const int y0 = (int)(((b & 0x7FFFFFu) | 0x800000u) << ((b >> 23) - 121));  // Q29, in (1, 2]
    const unsigned long long y2 = (unsigned long long)mulw(y0, y0);  // Q58
    const long long e = (1LL << 61) - (long long)__umul64hi(dp << 2, y2 << 3);  // Q61
    const int eh = (int)(e >> 20);
    const long long u = (e >> 1) + ((3 * (long long)eh * eh) >> 24);
    const long long r = ((long long)y0 << 32) + (((u >> 20) * y0) >> 9) + (((u & 0xFFFFF) * y0) >> 29);
    return min(r, (1LL << 62) - 1);
}

// The reciprocal of d' = d 4^k in [1/4, 1) for d > 0 in Q62, in two parts: y0 in Q28, the
// hardware's single-precision estimate of 1 / d' (the exponent of the truncated single-precision
// value of d gives k without a leading-zero count), and u in Q61 with 1 / d' = y0 (1 + u): u = e + e^2,
// e = 1 - d' y0 (|e| < 2^-21, so the third order is below 2^-62).
struct Recip {
    int y0, k;
    long long u;
};
__device__ __forceinline__ Recip recip_fix(long long d) {
    Recip r;
    // truncated at every step (a 64-bit conversion takes 80 clocks, two 32-bit ones 10)
    const float f = __fmaf_rz(__uint2float_rz((unsigned)(d >> 32)), 4294967296.f, __uint2float_rz((unsigned)d));
    r.k = (61 + 127 - (int)(__float_as_uint(f) >> 23)) >> 1;
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    const unsigned b = __float_as_uint(y);
    r.y0 = (int)(((b & 0x7FFFFFu) | 0x800000u) << ((int)(b >> 23) - 60 - 2 * r.k));
    const int2 dp = split31(d << (2 * r.k));
    const long long e = (1LL << 61) - ((mulw(dp.x, r.y0) << 2) + (mulw(dp.y, r.y0) >> 29));
    const int eh = (int)(e >> 20);
    r.u = e + (mulw(eh, eh) >> 21);
    return r;
}
// 1 / d' in Q60 (at most 4 - 2^-60)
__device__ __forceinline__ long long recip_full(const Recip& r) {
    const long long v = ((long long)r.y0 << 32) + (mulw((int)(r.u >> 20), r.y0) >> 9) +
                        (mulw((int)(r.u & 0xFFFFF), r.y0) >> 29);
    return min(v, (1LL << 62) - 1);
}
// q / d' for q in Q62 with q / d' < 1: (q y0) (1 + u), so that the next pivot does not wait for
// the full reciprocal
__device__ __forceinline__ long long times_recip(long long q, const Recip& r) {
    const int2 s = split31(q);
    const long long P = (mulw(s.x, r.y0) << 3) + (mulw(s.y, r.y0) >> 28);
    const int2 p = split31(P);
    const int u1 = (int)(r.u >> 20), u0 = (int)(r.u & 0xFFFFF);
    return P + (mulw(p.x, u1) >> 10) + (mulw(p.x, u0) >> 30) + (mulw(p.y, u1) >> 41);
}

// V 2^e rounded to FP64 (|V| < 2^63): infinite above the normal range, subnormal below it
__device__ __forceinline__ double fix_to_double(long long V, int e) {
    const unsigned long long sgn = (unsigned long long)V & 0x8000000000000000ULL;
    const unsigned long long u = V < 0 ? 0ULL - (unsigned long long)V : (unsigned long long)V;
    if (u == 0) return __longlong_as_double((long long)sgn);
    const int lz = __clzll((long long)u);
    const unsigned long long m = u << lz;
    const int be = 1023 + 63 - lz + e;
    if (be > 2046) return __longlong_as_double((long long)(sgn | 0x7FF0000000000000ULL));
    const int sh = 11 + max(0, 1 - be);  // bits below the result's last one
    if (sh > 64) return __longlong_as_double((long long)sgn);
    unsigned long long mant = sh < 64 ? m >> sh : 0;
    const unsigned long long rem = m << (64 - sh), half = 0x8000000000000000ULL;
    mant += (rem > half || (rem == half && (mant & 1ULL))) ? 1ULL : 0ULL;
    return __longlong_as_double((long long)(sgn | (((unsigned long long)max(be - 1, 0) << 52) + mant)));
}

// scaling exponent of a diagonal entry a > 0: a 4^-e in [1/4, 1)
__device__ __forceinline__ int diag_exp(double a, bool& bad) {
    const int E = dbl_exp(a);
    if (!(a > 0.0) || E == kNanExp) {
        bad = true;
        return 0;
    }
    return (E + 1) >> 1;
}

// ---- the diagonal block ------------------------------------------------------------------
// With x_rc the entry of column c below its pivot d_c once it is final, x' = x 2^k and l = x' / d'
// (|x'| < 1, |l| <= 2): L(r, c) = l 2^k, and the entry (r, s) loses x_rc x_sc / d_c = l_r x'_s.

//
// Range. x' and l are checked entry by entry, but the sums that they go into are held modulo 4: an
// entry that loses more than that comes back into range and would pass. Of a positive definite
// matrix no diagonal entry gets below zero, and while none does every sum stays below 1 (an
// off-diagonal one by Cauchy-Schwarz). So the lane of a row also follows the row's diagonal entry,
// column by column (each takes less than 2 from it, which cannot wrap) and from the upper halves alone
// (one multiply-add; full products cost the batch 1.5 %): the sum of 128 such products is within
// 2^-22, and below -2^-20 the block is not positive definite.
constexpr long long kDiagSlack = 1LL << (61 - 20);

// The chain: warp 0 factorises diagonal tile p in registers, lane (row, column parity) = (lane
// & 15, lane >> 4) holding eight columns, with shuffles only (no barrier, no shared memory on
// the chain), and publishes each finished column for the row warps. The pivots run one column
// ahead of the rest, d_{c+1} = a_{c+1,c+1} - x'^2 / d'_c, so that a column costs one reciprocal
// and one multiplication in sequence while column c's update of the tile goes on beside them.
__device__ void chain_tile(DiagSmem& S, int p, int& bad) {
    const int lane = threadIdx.x & 31, rr = lane & 15, h = lane >> 4;
    long long* T = S.T[p * (p + 1) / 2 + p];
    long long a[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = T[rr * TP + 2 * i + h];
    long long d = shfl64(a[0], 0);          // pivot of the current column
    long long x = shfl64(a[0], rr);         // its entry in this lane's row
    long long xn = shfl64(a[0], 1);         // x(c + 1, c) and a(c + 1, c + 1)
    long long an = shfl64(a[0], 17);
    long long dg = S.dg[p * TB + rr];  // this row's diagonal entry (see the note on range above)
    int drawn = 0;                     // negative once it has been overdrawn
    // a pivot <= 0 (not positive definite) is reported at the end, any value goes on; selections
    // instead of branches keep a column one block of code whose parts the scheduler interleaves
    bool neg = d <= 0;
    d = d <= 0 ? 1LL << 60 : d;
    Recip r = recip_fix(d);
#pragma unroll
    for (int c = 0; c < TB; ++c) {
        const int i0 = c >> 1, hc = c & 1;
        // the next pivot and its reciprocal
        long long d1 = 1LL << 60;
        Recip r1 = r;
        if (c + 1 < TB) {
            const int2 xk = split31(xn << r.k);
            d1 = an - times_recip(mul62(xk, xk), r);
            neg = neg || d1 <= 0;
            d1 = d1 <= 0 ? 1LL << 60 : d1;
            r1 = recip_fix(d1);
        }
        // column c
        const long long inv = recip_full(r);
        const int2 xp = split31(x << r.k);
        const long long l = mul61(xp, split31(inv));
        neg = neg || (rr > c && (beyond(x, 62 - r.k) || beyond(l, 62)));
        const int2 nl = split31(-l);
        const long long dn = madw(nl.x, xp.x, dg);
        dg = rr > c ? dn : dg;
        drawn |= (int)(dg >> 32);
#pragma unroll
        for (int i = i0; i < 8; ++i) {
            if (2 * i + 1 <= c) continue;
            const int s = 2 * i + h;
            int2 xs;
            xs.x = __shfl_sync(0xffffffffu, xp.x, s);
            xs.y = __shfl_sync(0xffffffffu, xp.y, s);
            const long long v = a[i] + mul61(nl, xs);
            a[i] = s > c ? v : a[i];
        }
        if (c + 1 < TB) x = shfl64(a[(c + 1) >> 1], rr | (((c + 1) & 1) << 4));
        if (c + 2 < TB) {
            xn = shfl64(a[(c + 1) >> 1], (c + 2) | (((c + 1) & 1) << 4));
            an = shfl64(a[(c + 2) >> 1], (c + 2) | (((c + 2) & 1) << 4));
        }
        // publish (every lane writes the same pivot data; lanes of the other half the same x')
        if (h == hc && rr > c) T[rr * TP + c] = l;
        S.xs[c][rr] = xp;
        S.inv[p * TB + c] = inv;
        S.dq[p * TB + c] = d;
        S.k[p * TB + c] = r.k;
        __syncwarp();
        __threadfence_block();
        S.done = p * TB + c + 1;
        d = d1;
        r = r1;
    }
    if (neg || drawn < 0) bad = 1;
}

// Rows below diagonal tile p: a lane per row follows the chain column by column (one column
// behind it), then leaves its 16 entries as l (T), limbs of x' and l for the updates and limbs
// of l for the row kernel (tab).
__device__ void follow_rows(DiagSmem& S, BlockTab* tab, int p, int r, int& bad) {
    const bool live = r < NB;  // (rows past the block's last tile are filled in, harmless)
    const int t = min(r, NB - 1) >> 4, ri = r & 15;
    long long* T = S.T[t * (t + 1) / 2 + p] + ri * TP;
    long long a[TB];
#pragma unroll
    for (int s = 0; s < TB; ++s) a[s] = live ? T[s] : 0;
    int2* ct = &tab->ct[t * (t - 1) / 2 + p][0][ri];
    long long dg = live ? S.dg[r] : 0;
    int drawn = 0;
#pragma unroll
    for (int c = 0; c < TB; ++c) {
        // the chain warp never waits for this one, so the wait ends; bounded all the same
        for (int it = 0; S.done < p * TB + c + 1; ++it)
            if (it > (1 << 22)) {
                bad = 1;
                break;
            }
        __threadfence_block();
        const int k = S.k[p * TB + c];
        const long long x = a[c], xk = x << k;
        const int2 xp = split31(xk);
        const long long l = mul61(xp, split31(S.inv[p * TB + c]));
        const int2 nl = split31(-l);
        dg = madw(nl.x, xp.x, dg);
        drawn |= (int)(dg >> 32);
        bad |= (beyond(x, 62 - k) || beyond(l, 62)) ? 1 : 0;
#pragma unroll
        for (int s = c + 1; s < TB; ++s) a[s] += mul61(nl, S.xs[c][s]);
        if (live) {
            const int2 lm = split29(l);
            S.xl[p & 1][c][r] = split29(xk);
            S.ll[p & 1][c][r] = lm;
            ct[c * TB] = lm;
            T[c] = l;
        }
    }
    if (live) S.dg[r] = dg;
    if (drawn < 0) bad = 1;
}

// Eight rows (half hf) of tile (tr, tc) -= l(tr, p) x'(tc, p)^T: four entries per lane, exact
// 29-bit limb products summed in 64 bits.
__device__ __forceinline__ void update_half(DiagSmem& S, int p, int tr, int tc, int hf) {
    const int lane = threadIdx.x & 31;
    const int ri = 8 * hf + (lane >> 2), ci = 4 * (lane & 3);
    const int2* yr = &S.ll[p & 1][0][tr * TB + ri];
    const int2* yc = &S.xl[p & 1][0][tc * TB + ci];
    long long hh[4] = {0, 0, 0, 0}, mid[4] = {1 << 23, 1 << 23, 1 << 23, 1 << 23};  // (rounding)
#pragma unroll 4
    for (int q = 0; q < TB; ++q) {
        const int2 r = yr[q * NB];
        const int4 c01 = *reinterpret_cast<const int4*>(yc + q * NB);
        const int4 c23 = *reinterpret_cast<const int4*>(yc + q * NB + 2);
        const int cx[4] = {c01.x, c01.z, c23.x, c23.z}, cy[4] = {c01.y, c01.w, c23.y, c23.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            hh[j] = madw(r.x, cx[j], hh[j]);
            mid[j] = madw(r.x, cy[j], madw(r.y, cx[j], mid[j]));
        }
    }
    long long* T = S.T[tr * (tr + 1) / 2 + tc] + ri * TP + ci;
#pragma unroll
    for (int j = 0; j < 4; ++j) T[j] -= (hh[j] << 5) + (mid[j] >> 24);
}

// LDL^T of the nb x nb block at H (ld), nb <= 128 (padded with a diagonal of 1/2). Per 16-column
// panel: warp 0 carries the chain, warps 1-4 the rows below it, the other warps meanwhile the
// rest of the previous panel's update; then all warps update the next panel's tile column.
__global__ void __launch_bounds__(32 * kDiagWarps, 1)
k_fix_diag(double* __restrict__ H, int ld, int nb, int R_tau, double* __restrict__ dinv, DevScalars* sc, int mode,
           BlockTab* __restrict__ tab) {
    extern __shared__ __align__(16) unsigned char smem[];
    DiagSmem& S = *reinterpret_cast<DiagSmem*>(smem);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        S.bad = 0;
        S.done = 0;
    }
    __syncthreads();
    bool bad0 = false;
    if (tid < NB) S.e[tid] = tid < nb ? diag_exp(H[(size_t)tid * ld + tid], bad0) : 0;
    __syncthreads();
    // 36 lower tiles of 256 entries, 18 per thread, all loads in flight before the first is used
    {
        constexpr int PER = NT * (NT + 1) / 2 * TB * TB / (32 * kDiagWarps);
        double h[PER];
        short rc[PER];
        int tr = 0, t0 = 0;  // tile row and its first tile
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int t = 2 * u + (tid >> 8);
            if (t > t0 + tr) t0 += ++tr;
            const int r = tr * TB + ((tid >> 4) & 15), c = (t - t0) * TB + (tid & 15);
            rc[u] = (short)(r << 7 | c);
            h[u] = (r < nb && c <= r) ? H[(size_t)r * ld + c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int t = 2 * u + (tid >> 8), r = rc[u] >> 7, c = rc[u] & 127;
            long long v = r == c ? 1LL << 61 : 0;
            if (r < nb && c <= r) {
                const int er = S.e[r] + S.e[c];
                if (dbl_exp(h[u]) > er) bad0 = true;  // above sqrt(a_rr a_cc), NaN or infinite
                v = fixed62(h[u], er);
            }
            S.T[t][((tid >> 4) & 15) * TP + (tid & 15)] = v;
            if (r == c) S.dg[r] = (v >> 1) + kDiagSlack;
        }
    }
    int bad = bad0 ? 1 : 0;
    // warps 4, 8, 12 share the chain's SM sub-partition and stay out of the way while it runs;
    // of the other twelve, four follow the chain and eight update
    constexpr int kWorkers = 12;
    const int role = (w & 3) ? 3 * (w >> 2) + (w & 3) - 1 : kWorkers;
    __syncthreads();
    const int np = (nb + TB - 1) / TB;  // panels with columns of the block
    for (int p = 0; p < np; ++p) {
        if (w == 0) {
            chain_tile(S, p, bad);
        } else if (role < 4) {
            if (p * TB + TB + 32 * role < np * TB) follow_rows(S, tab, p, p * TB + TB + 32 * role + lane, bad);
        } else if (p > 0 && role < kWorkers) {
            // tiles (tr, tc), tc >= p + 1, of panel p - 1, in halves
            const int n = np - 1 - p;
            for (int u = role - 4; u < n * (n + 1); u += kWorkers - 4) {
                const int t = u >> 1;
                int i = 0;
                while ((i + 1) * (i + 2) / 2 <= t) ++i;
                update_half(S, p - 1, p + 1 + i, p + 1 + t - i * (i + 1) / 2, u & 1);
            }
        }
        __syncthreads();
        if (w < 2 * (np - 1 - p)) update_half(S, p, p + 1 + (w >> 1), p + 1, w & 1);
        __syncthreads();
    }
    // results: L and D in FP64, the row kernel's tables
    const double tau = (double)R_tau * DBL_EPSILON * sc->maxdiag;
    {
        const int i = (tid >> 4) & 15, j = tid & 15;
        int tr = 0, t0 = 0;
#pragma unroll 3
        for (int t = tid >> 8; t < NT * (NT + 1) / 2; t += 2) {
            while (t > t0 + tr) t0 += ++tr;
            const int r = tr * TB + i, c = (t - t0) * TB + j;
            if (c < r && r < nb) H[(size_t)r * ld + c] = fix_to_double(S.T[t][i * TP + j], S.k[c] + S.e[r] - S.e[c] - 61);
        }
    }
#pragma unroll 4
    for (int x = tid; x < NT * TB * TB; x += 32 * kDiagWarps) {
        const int t = x >> 8, q = (x >> 4) & 15, i = x & 15;
        tab->ls[t][q][i] = i > q ? split31(-S.T[t * (t + 1) / 2 + t][i * TP + q]) : make_int2(0, 0);
    }
    if (tid < np * TB) {
        int k;
        tab->rs[tid] = rsqrt_fix(S.dq[tid], k);  // the reciprocal's k
        tab->k[tid] = S.k[tid];
        tab->e[tid] = S.e[tid];
        if (tid < nb) {
            const double D = fix_to_double(S.dq[tid], 2 * S.e[tid] - 62);
            if (!pivot_ok(D, tau)) bad = 1;
            H[(size_t)tid * ld + tid] = D;
            dinv[tid] = recip_nr(D);
        }
    }
    if (bad) S.bad = 1;
    __syncthreads();
    if (tid == 0 && S.bad) atomicOr(&sc->fail_mask, 1 << mode);
}

// ---- the rows below ------------------------------------------------------------------------
// An appended row has no bound like the diagonal of H: its exponent leaves kHeadroom bits over the
// row's largest entry for the growth of the substitution; a value that passes 2^-3 (up to there no
// sum of 128 terms wraps) sends the row through once more with four bits more, so the row's
// largest value keeps at least 55 of its bits. A row that has grown past 2^50 times its largest entry
// after the last try sets the failed-pivot bit like a row of H that leaves its range: what it holds
// has wrapped.
constexpr int kHeadroom = 5;
constexpr int kRowLimit = 59;
constexpr int kRetryBits = 4;
constexpr int kMaxTries = 12;

// Rows i in [nb, nrows) of H (element (0, 0) of the block's columns at H, rows ld apart; the
// first R - j0 of them rows of the matrix, the rest appended rows): L(i, :) or Y(i, :) in FP64 in
// place and, with digits, the digits of C(i, :) for the trailing update. Two rows per warp, a lane
// per column of a 16-column tile; per tile the finished tiles' products run on 29-bit limbs and
// the 16 columns of the tile are substituted one after the other by shuffles.
__global__ void __launch_bounds__(32 * kPanelWarps)
k_fix_rows(double* __restrict__ H, int ld, int nb, int nH, int nrows, DevScalars* sc,
           int mode, const BlockTab* __restrict__ tab, uint16_t* __restrict__ dig,
           int* __restrict__ exps, int digits) {
    extern __shared__ __align__(16) unsigned char smem[];
    PanelSmem& S = *reinterpret_cast<PanelSmem*>(smem);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, l16 = lane & 15, hf = lane >> 4;
    {
        const int4* src = reinterpret_cast<const int4*>(tab);
        int4* dst = reinterpret_cast<int4*>(&S.tab);
#pragma unroll 8
        for (int x = tid; x < (int)(sizeof(BlockTab) / 16); x += 32 * kPanelWarps) dst[x] = src[x];
    }
    const int i = nb + (blockIdx.x * kPanelWarps + w) * 2 + hf;
    const bool live = i < nrows, hrow = i < nH;
    double* row = H + (size_t)min(i, nrows - 1) * ld;
    double v[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        const int c = t * TB + l16;
        v[t] = (live && c < nb) ? row[c] : 0.0;
    }
    const double dg = hrow && live ? row[i] : 1.0;
    __syncthreads();
    int er;           // row exponent: |C(i, :)| < 2^er
    bool out = false;  // out of range: not positive definite (rows of H), too little headroom (appended rows)
    {
        // both rows of the warp take part in the shuffles (one may be a row of H, the other appended)
        int m = kZeroExp;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int E = dbl_exp(v[t]);
            m = max(m, E >= kNanExp || E == kZeroExp ? E : E - S.tab.e[t * TB + l16]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (hrow)
            er = diag_exp(dg, out);
        else
            er = m >= kNanExp ? kNanExp : m == kZeroExp ? 0 : m + kHeadroom;
    }
    const bool nan_row = er == kNanExp;
    const int limit = hrow ? 62 : kRowLimit;
    int2* xl = S.xl[w][hf];
    long long* yq = S.yq[w][hf];
    for (int tries = 0;; ++tries) {
        for (int t = 0; t < NT && t * TB < nb; ++t) {
            const int c = t * TB + l16;
            const int ec = er + S.tab.e[c];
            double vt = 0.0;
#pragma unroll
            for (int u = 0; u < NT; ++u)
                if (u == t) vt = v[u];
            if (!nan_row && dbl_exp(vt) > ec) out = true;
            long long a = nan_row ? 0 : fixed62(vt, ec);
            for (int u = 0; u < t; ++u) {
                const int2* ct = &S.tab.ct[t * (t - 1) / 2 + u][0][l16];
                long long hh = 0, m0 = 1 << 23, m1 = 0;  // (rounding)
#pragma unroll
                for (int q = 0; q < TB; ++q) {
                    const int2 y = xl[u * TB + q], cc = ct[q * TB];
                    hh = madw(y.x, cc.x, hh);
                    m0 = madw(y.x, cc.y, m0);
                    m1 = madw(y.y, cc.x, m1);
                }
                a -= (hh << 5) + ((m0 + m1) >> 24);
            }
            const int2* ls = &S.tab.ls[t][0][l16];
            const int kc = S.tab.k[c];
#pragma unroll
            for (int q = 0; q < TB; ++q) {
                // lane q's entry is final: its x' to every lane (ls is zero for the lanes up to q)
                const int2 xp = split31(a << kc);
                int2 xq;
                xq.x = __shfl_sync(0xffffffffu, xp.x, (lane & 16) | q);
                xq.y = __shfl_sync(0xffffffffu, xp.y, (lane & 16) | q);
                a += mul61(xq, ls[q * TB]);
            }
            const long long xk = a << kc;
            xl[c] = split29(xk);
            const long long y = mul61(split31(xk), split31(S.tab.rs[c]));
            out = out || beyond(a, limit - kc) || beyond(y, limit);
            yq[c] = y;
            __syncwarp();
        }
        const unsigned vote = __ballot_sync(0xffffffffu, out && live);
        const bool row_out = (vote >> (lane & 16)) & 0xFFFFu;
        if (row_out && (hrow || tries == kMaxTries) && l16 == 0) atomicOr(&sc->fail_mask, 1 << mode);
        const bool again = row_out && !hrow;
        if (!__any_sync(0xffffffffu, again) || tries == kMaxTries) break;
        if (again) er += kRetryBits;
        out = false;
    }
    if (live) {
#pragma unroll 4
        for (int t = 0; t < NT; ++t) {
            const int c = t * TB + l16;
            if (c < nb)
                row[c] = nan_row ? __longlong_as_double(0x7FF8000000000000LL)
                                 : fix_to_double(mul62(split31(yq[c]), split31(S.tab.rs[c])),
                                                 S.tab.k[c] + er - S.tab.e[c] - 61);
        }
    }
    __syncwarp();
    if (!digits) return;
    // digits of both rows, four columns per lane
    const size_t rows = nrows - nb;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int ig = nb + (blockIdx.x * kPanelWarps + w) * 2 + g;
        const int eg = __shfl_sync(0xffffffffu, er, 16 * g);
        if (ig >= nrows) break;
        long long x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = S.yq[w][g][4 * lane + j];
        store_fixed4(x, dig + (size_t)(ig - nb) * NB + 4 * lane, rows * NB);
        if (lane == 0) exps[ig - nb] = eg;
    }
}

}  // namespace

size_t ldl_fix_ws_bytes(int R, int n) {
    return Arena::need<BlockTab>(1) + (R > NB ? ozmat_bytes(R + n - NB, NB) : 0);
}

void ldl_fix_carve(FixWs& w, Arena& ar, int R, int n) {
    w.tab = ar.take<BlockTab>(1);
    if (R > NB) ozmat_carve(w.dig, ar, R + n - NB, NB);
}

bool ldl_fix_prepare() {
    if (!oz_available()) return false;
    static PerDevice<bool> ready;
    return ready.get([](int) {
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        return cudaFuncSetAttribute(k_fix_diag, attr, (int)sizeof(DiagSmem)) == cudaSuccess &&
               cudaFuncSetAttribute(k_fix_rows, attr, (int)sizeof(PanelSmem)) == cudaSuccess;
    });
}

cudaError_t ldl_fix(cudaStream_t st, int R, int n, double* Haug, double* dinv, DevScalars* sc, int mode,
                    const FixWs& ws) {
    BlockTab* tab = static_cast<BlockTab*>(ws.tab);
    for (int j0 = 0; j0 < R; j0 += NB) {
        const int nb = std::min(NB, R - j0), below = R + n - j0 - nb, j1 = j0 + nb;
        double* blk = Haug + (size_t)j0 * R + j0;
        const bool more = j1 < R;
        OzMat d = ws.dig;
        d.rows = below;
        d.ld_rows = below;
        d.K = nb;
        {
            ProfScope prof(st, KC_CHOL, (double)nb * nb * nb / 3.0 + (double)below * nb * nb);
            k_fix_diag<<<1, 32 * kDiagWarps, sizeof(DiagSmem), st>>>(blk, R, nb, R, dinv + j0, sc, mode, tab);
            count_launch();
            if (below > 0) {
                k_fix_rows<<<cdiv(below, 2 * kPanelWarps), 32 * kPanelWarps, sizeof(PanelSmem), st>>>(
                    blk, R, nb, R - j0, R - j0 + n, sc, mode, tab, d.d, d.e, more ? 1 : 0);
                count_launch();
            }
        }
        if (more) {
            const int mB = R - j1;
            ProfScope prof(st, KC_OZ, (double)mB * (mB + 1) * nb + 2.0 * (below - mB) * mB * nb);
            OzMat b = d;
            b.rows = mB;
            const cudaError_t e = oz_mul(st, d, b, Haug + (size_t)j1 * R + j1, R, -1.0, OZ_ACC | OZ_LOWER);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaGetLastError();
}

}  // namespace thc
