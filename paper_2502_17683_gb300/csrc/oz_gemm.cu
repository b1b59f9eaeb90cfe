// FP64-accurate emulated products on the BF16 tensor cores (see oz.cuh for the arithmetic).
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "f64.cuh"
#include "fixed.cuh"
#include "oz.cuh"
#include "prof.cuh"
#include "tcgen05.cuh"

namespace thc {

__device__ __managed__ int g_oz_error = 0;  // in managed memory: see take_error_word

namespace {

constexpr int S = kOzSlices;
constexpr int KP = kOzPanel;                 // K elements per operand row (2 x 64)
constexpr int BM = 128;                      // MMA M: rows of the left operand per tile
constexpr int A_TILE = BM * 128;             // bytes of one 128 x 64 BF16 slice (one K half): a ring stage
constexpr int B_STAGES = 2;                  // right operand: all S slices of one K half per stage
constexpr int TMEM_COLS = 512;
constexpr int EPI_WARPS = 16;                // four per TMEM lane quarter, BN / 4 columns each
constexpr int NTHREADS = 64 + 32 * EPI_WARPS + 32;  // warp 0 TMA, warp 1 MMA + TMEM, the epilogue, a look-out
constexpr int STG_BYTES = EPI_WARPS * 1024;  // per epilogue warp: 32 rows x 4 columns of FP64
constexpr uint32_t WAIT_LIMIT = 1u << 22;

// Tile of BN columns: 64 (all 512 TMEM columns hold one set of S accumulators) or 32 (two
// sets, so that the MMAs of the next chunk run while one is drained).
template <int BN>
struct Tile {
    static constexpr int B_HALF = S * BN * 128;
    static constexpr int A_STAGES = BN == 64 ? 5 : 8;
    static constexpr int ACC_SET = S * BN;
    static constexpr int SETS = TMEM_COLS / ACC_SET;
    static constexpr int SMEM = 1024 + A_STAGES * A_TILE + B_STAGES * B_HALF + STG_BYTES + 256;
};
static_assert(Tile<64>::SETS == 1 && Tile<32>::SETS == 2, "TMEM columns");

__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t parity, int code) {
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    atomicExch(&g_oz_error, code);
    return false;
}

// The S digits of four values relative to the row exponent erow (out[a * stride .. + 3]).
__device__ __forceinline__ void store_digits4(const double (&x)[4], int erow, uint16_t* __restrict__ out,
                                              size_t stride) {
    long long X[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) X[i] = fixed62(x[i], erow);
    store_fixed4(X, out, stride);
}

// (hi 2^40 + lo) 2^e rounded once to FP64 (to nearest, ties to even), its sign flipped by neg
// (0 or the sign bit): normalised and assembled in integer arithmetic, so that of each output
// element only the final addition runs on the FP64 pipe (an int64 conversion costs as much
// there as an FMA). |hi| < 2^44, |lo| < 2^62. Below the normal range the term is dropped
// (signed zero; see kTinyExp), above it the result is infinite.
__device__ __forceinline__ double scaled_sum(long long hi, long long lo, int e, unsigned long long neg) {
    // V = hi 2^(40 - sh) + lo 2^-sh within 62 bits; bits below 2^-59 of V are cut only for sh > 0
    const int hb = 64 - __clzll(hi < 0 ? -hi : hi);
    const int sh = max(0, hb - 21);
    const long long V = (sh < 40 ? hi << (40 - sh) : hi >> (sh - 40)) + (lo >> sh);
    const unsigned long long sgn = ((unsigned long long)V & 0x8000000000000000ULL) ^ neg;
    const unsigned long long u = V < 0 ? 0ULL - (unsigned long long)V : (unsigned long long)V;
    if (u == 0) return __longlong_as_double((long long)sgn);
    const int lz = __clzll((long long)u);
    const unsigned long long m = u << lz;   // leading one at bit 63
    unsigned long long mant = m >> 11;      // 53 bits, leading one at bit 52
    const unsigned rem = (unsigned)(m & 0x7FFULL);
    mant += (rem > 0x400u || (rem == 0x400u && (mant & 1ULL))) ? 1ULL : 0ULL;
    const int be = 1023 + 63 - lz + sh + e;  // biased exponent of the result
    if (be < 1) return __longlong_as_double((long long)sgn);
    if (be > 2046) return __longlong_as_double((long long)(sgn | 0x7FF0000000000000ULL));
    // a rounding carry into bit 53 moves into the exponent field
    return __longlong_as_double((long long)(sgn | (((unsigned long long)(be - 1) << 52) + mant)));
}

constexpr int ROWS_PER_BLOCK = 4;  // one warp per row

// Digits of the rows of src (rows x K, ld): wpr warps of a block of four take a row, a chunk of
// KP values at a time each; they find the row's exponent, then cut four consecutive values per
// lane (8-byte stores, a 256-byte line per slice and chunk). The second read of the row comes from
// L1 / L2. VEC: 16-byte loads (even ld, aligned base). Few rows leave an SM a handful of warps, so
// the time is that of one warp's chain of reads and cuts: several warps to a long row shorten it
// (713 x 713: 8.0 -> 5.5 us).
template <bool VEC>
__global__ void __launch_bounds__(32 * ROWS_PER_BLOCK)
k_oz_split_rows(const double* __restrict__ src, int ld, int rows, int K, uint16_t* __restrict__ out,
                int* __restrict__ exps, int wpr) {
    __shared__ int sh[ROWS_PER_BLOCK];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, part = w % wpr;
    const int r = blockIdx.x * (ROWS_PER_BLOCK / wpr) + w / wpr;
    const bool live = r < rows;
    const double* p = src + (size_t)r * ld;
    auto load4 = [&](int k, double (&v)[4]) {
        if (VEC && k + 3 < K) {
            const double2 a = __ldg(reinterpret_cast<const double2*>(p + k));
            const double2 b = __ldg(reinterpret_cast<const double2*>(p + k + 2));
            v[0] = a.x;
            v[1] = a.y;
            v[2] = b.x;
            v[3] = b.y;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = k + i < K ? __ldg(p + k + i) : 0.0;
        }
    };
    int e = kZeroExp;
    const int step = wpr * KP;
#pragma unroll 2
    for (int k = part * KP + 4 * lane; live && k < K; k += step) {
        double v[4];
        load4(k, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) e = max(e, dbl_exp(v[i]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (wpr > 1) {
        if (lane == 0) sh[w] = e;
        __syncthreads();
        for (int i = 0; i < wpr; ++i) e = max(e, sh[w - part + i]);
    }
    if (!live) return;
    if (e == kZeroExp) e = 0;
    if (lane == 0 && part == 0) exps[r] = e;
    const size_t stride = (size_t)rows * KP;
    uint16_t* o = out + (size_t)part * S * stride + (size_t)r * KP + 4 * lane;
    for (int k = part * KP + 4 * lane; k - 4 * lane < K; k += step, o += wpr * S * stride) {
        double v[4];
        load4(k, v);
        store_digits4(v, e, o, stride);
    }
}

constexpr int COLS_PER_BLOCK = 8;   // output rows (source columns) per block, one warp each
constexpr int kColsMaxK = 3072;     // K of one slab of the column split (its shared memory: 193 KB)

// Exponents of the columns of S (K x N, ld), times S2 when given (only for K > kColsMaxK).
__global__ void __launch_bounds__(256)
k_oz_col_exps(const double* __restrict__ S1, const double* __restrict__ S2, int ld, int N, int K,
              int* __restrict__ exps) {
    __shared__ int sh[8][32];
    const int n = blockIdx.x * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
    int e = kZeroExp;
    if (n < N)
        for (int k = w; k < K; k += 8) {
            double v = S1[(size_t)k * ld + n];
            if (S2) v *= S2[(size_t)k * ld + n];
            e = max(e, dbl_exp(v));
        }
    sh[w][threadIdx.x & 31] = e;
    __syncthreads();
    if (w == 0 && n < N) {
        for (int i = 1; i < 8; ++i) e = max(e, sh[i][threadIdx.x]);
        exps[n] = e == kZeroExp ? 0 : e;
    }
}

// Digits of the columns of S1 (K x N row-major, ld), times S2 element by element when given (a
// Hadamard operand): a block brings a K x 8 slab into shared memory once (64-byte row pieces),
// finds its columns' exponents on the way and then cuts a column's chunks on blockDim / 256 warps.
// blockIdx.y: slab of kColsMaxK rows; with several (have_exp) the exponents come from k_oz_col_exps.
// blockIdx.z: matrix of a stack (K ld apart), N of the `rows` output rows each.
// With no more blocks than SMs the time is one block's chain of loads and cuts, not the traffic:
// eight loads a thread (of each operand) are issued before the first is used, whatever K, and a
// block has 256 threads per chunk up to 1024 (713 x 713 times a second matrix: 19.9 -> 9.3 us,
// 713 x 1061: 16.1 -> 9.4, 480 x 720: 10.2 -> 7).
__global__ void __launch_bounds__(1024)
k_oz_split_cols(const double* __restrict__ S1, const double* __restrict__ S2, int ld, int N, int K, int rows,
                uint16_t* __restrict__ out, int* __restrict__ exps, int have_exp) {
    extern __shared__ __align__(16) double slab[];  // [8][pitch]: column n at n * pitch
    __shared__ int sh[32][COLS_PER_BLOCK];
    const int nw = blockDim.x >> 5, cparts = nw / COLS_PER_BLOCK;
    const int n0 = blockIdx.x * COLS_PER_BLOCK, k0 = blockIdx.y * kColsMaxK;
    S1 += (size_t)blockIdx.z * K * ld;
    if (S2) S2 += (size_t)blockIdx.z * K * ld;
    exps += (size_t)blockIdx.z * N;
    const int kn = min(K - k0, kColsMaxK), kpad = (kn + KP - 1) / KP * KP;
    const int pitch = kpad + 4;  // = 4 mod 16 doubles: the 8 x 4 pieces of a warp's stores miss each other's banks
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    {
        const int nn = tid & 7, n = n0 + nn;
        const bool live = n < N;
        const double* p1 = S1 + (size_t)k0 * ld + n;
        const double* p2 = S2 ? S2 + (size_t)k0 * ld + n : nullptr;
        int e = kZeroExp;
        const int step = blockDim.x >> 3;
        for (int kb = tid >> 3; kb < kpad; kb += 8 * step) {
            double v[8], v2[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = kb + u * step;
                const bool in = live && k < kn;
                v[u] = in ? p1[(size_t)k * ld] : 0.0;
                v2[u] = in && p2 ? p2[(size_t)k * ld] : 1.0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = kb + u * step;
                if (p2) v[u] *= v2[u];
                e = max(e, dbl_exp(v[u]));
                if (k < kpad) slab[nn * pitch + k] = v[u];
            }
        }
        e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
        e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
        if (lane < 8) sh[w][lane] = e;
    }
    __syncthreads();
    const int col = w % COLS_PER_BLOCK, part = w / COLS_PER_BLOCK, n = n0 + col;
    if (n >= N) return;
    int e;
    if (have_exp) {
        e = exps[n];
    } else {
        e = kZeroExp;
        for (int i = 0; i < nw; ++i) e = max(e, sh[i][col]);
        if (e == kZeroExp) e = 0;
        if (lane == 0 && part == 0) exps[n] = e;
    }
    const size_t stride = (size_t)rows * KP;
    uint16_t* o = out + (size_t)(k0 / KP + part) * S * stride + ((size_t)blockIdx.z * N + n) * KP + 4 * lane;
    for (int k = part * KP + 4 * lane; k < kpad; k += cparts * KP, o += cparts * S * stride) {
        const double2 a = *reinterpret_cast<const double2*>(&slab[col * pitch + k]);
        const double2 b = *reinterpret_cast<const double2*>(&slab[col * pitch + k + 2]);
        const double v[4] = {a.x, a.y, b.x, b.y};
        store_digits4(v, e, o, stride);
    }
}

__device__ __forceinline__ double pow2(int e) {
    return __longlong_as_double((long long)(e + 1023) << 52);  // e in [-1022, 1023]
}

// The two operands of an LDL^T trailing update from one read of the rows below the panel:
// row r < mA of src (its K entries, K <= 512) gives the left-operand row r, scaled per column k
// by D_k 2^-m_k, and, for r < mB, the right-operand row r, scaled by 2^m_k (m_k =
// floor(E(D_k) / 2), D_k = diag[k * (ldd + 1)]), each cut into its S digit slices. A warp per row.
constexpr int kLdlMaxChunks = 4;
__global__ void __launch_bounds__(32 * ROWS_PER_BLOCK)
k_oz_split_ldl(const double* __restrict__ src, int ld, int mA, int mB, int K,
               const double* __restrict__ diag, int ldd, uint16_t* __restrict__ outA,
               int* __restrict__ expsA, uint16_t* __restrict__ outB, int* __restrict__ expsB) {
    const int lane = threadIdx.x & 31, r = blockIdx.x * ROWS_PER_BLOCK + (threadIdx.x >> 5);
    if (r >= mA) return;
    const bool hasB = r < mB;
    const int nch = (K + KP - 1) / KP;
    int ea = kZeroExp, eb = kZeroExp;
    double a[kLdlMaxChunks][4], b[kLdlMaxChunks][4];
#pragma unroll
    for (int c = 0; c < kLdlMaxChunks; ++c) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = c * KP + 4 * lane + i;
            a[c][i] = b[c][i] = 0.0;
            if (c < nch && k < K) {
                const double v = src[(size_t)r * ld + k];
                const double dk = diag[(size_t)k * (ldd + 1)];
                const int Ek = dbl_exp(dk);
                const int mk = (Ek == kZeroExp || Ek == kNanExp || Ek < -1000) ? 0 : (Ek >> 1);
                a[c][i] = v * (dk * pow2(-mk));
                b[c][i] = v * pow2(mk);
                ea = max(ea, dbl_exp(a[c][i]));
                eb = max(eb, dbl_exp(b[c][i]));
            }
        }
    }
    ea = __reduce_max_sync(0xffffffffu, ea);
    eb = __reduce_max_sync(0xffffffffu, eb);
    if (ea == kZeroExp) ea = 0;
    if (eb == kZeroExp) eb = 0;
    if (lane == 0) {
        expsA[r] = ea;
        if (hasB) expsB[r] = eb;
    }
#pragma unroll
    for (int c = 0; c < kLdlMaxChunks; ++c) {
        if (c >= nch) break;
        store_digits4(a[c], ea, outA + ((size_t)c * S * mA + r) * KP + 4 * lane, (size_t)mA * KP);
        if (hasB) store_digits4(b[c], eb, outB + ((size_t)c * S * mB + r) * KP + 4 * lane, (size_t)mB * KP);
    }
}

struct UpdArgs {
    double* C;     // C[i][j] at C[i * ldc + j]
    int ldc;
    int mA, mB;    // rows of C (left operand rows) and columns (right operand rows)
    const int* eA;
    const int* eB;
    int tiles_m;   // tiles along mA
    int tiles_n;   // tiles along mB
    int lower;     // 1: rows i < mB only on and below the diagonal
    int mirror;    // 1 (with lower, mA == mB): C[j][i] is written with C[i][j]
    double sign;   // C (+)= sign * A B^T; +1 or -1
    int accumulate;  // 0: C is overwritten
    int khalves;      // 64-wide K halves that hold data in the last chunk (1 when its K <= 64)
    int nchunks;      // K chunks of KP; chunk c's slices are planes S c .. S c + S - 1 of the maps
    int nactive;      // active tiles (tile_of's index range)
    int kgroups;      // split K: work item (group g, tile) takes chunks [g cpg, (g + 1) cpg); group 0
    int cpg;          // adds into C, group g > 0 writes its sum to part + (g - 1) mA mB (ld mB)
    double* part;     // (kgroups > 1 only without lower)
    OzSrc srcA, srcB; // where the digits come from
    int K;
};

__device__ __forceinline__ double src_entry(const OzSrc& s, int r, long k, int K) {
    const long i = s.cols ? ((long)(r / s.cols) * K + k) * s.ld + r % s.cols : (long)r * s.ld + k;
    return s.s2 ? s.s1[i] * s.s2[i] : s.s1[i];
}

// Active tiles of row block tm: on a lower-only (symmetric or LDL^T trailing) block, rows
// that lie within the first mB stop at the diagonal; below them every tile is active.
template <int BN>
__host__ __device__ __forceinline__ int row_tiles(int tm, int tiles_n, int mB, bool lower) {
    const int m0 = tm * BM;
    return (lower && m0 + BM - 1 < mB) ? min(tiles_n, (m0 + BM - 1) / BN + 1) : tiles_n;
}

// The active tile of compact index u (row by row, so that the CTAs' shares of a lower block
// differ by at most one tile; tiles above the diagonal are never handed out). Only the rows
// of a lower block that end within its first mB columns (at most mB / BM of them) have
// fewer tiles than tiles_n; they are walked, every later row is full.
template <int BN>
__device__ __forceinline__ void tile_of(const UpdArgs& a, int u, int& m0, int& n0) {
    int tm = 0;
    if (a.lower) {
        for (; tm < a.tiles_m && tm * BM + BM - 1 < a.mB; ++tm) {
            const int c = row_tiles<BN>(tm, a.tiles_n, a.mB, true);
            if (u < c) {
                m0 = tm * BM;
                n0 = u * BN;
                return;
            }
            u -= c;
        }
    }
    tm += u / a.tiles_n;
    m0 = tm * BM;
    n0 = (u % a.tiles_n) * BN;
}

// Between the epilogue's warps and the one that looks out for rows without digits.
__device__ __forceinline__ void epi_barrier() {
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS + 32) : "memory");
}

// Rows whose exponents add up to less may give an element below the normal range (the last unit of
// its sum is 2^(ea + eb - 68)), where the epilogue gives zero.
constexpr int kTinyExp = -954;

// Terms [k0, k1) of element (i, j) in FP64 from the operands. With an infinity or a NaN in its row or
// column: one after the other (nothing changes a NaN: a call on such data is not held up by it). Else
// the rows are tiny: scaled by their exponents (unless these are those of a later K range and say nothing
// of the earlier ones), the products and sums carried with their errors, after Ogita, Rump, Oishi,
// "Accurate sum and dot product", SIAM J. Sci. Comput. 26, 2005: like the digits', the element's only
// rounding is that of the result.
__device__ __forceinline__ double src_dot(const UpdArgs& args, int i, int j, long k0, long k1) {
    int ea = args.eA[i], eb = args.eB[j];
    double s = 0.0, c = 0.0;
    if (max(ea, eb) >= kNanExp) {
        for (long k = k0; k < k1 && !isnan(s); ++k)
            s = fma(src_entry(args.srcA, i, k, args.K), src_entry(args.srcB, j, k, args.K), s);
        return s;
    }
    if (args.srcA.k0 > 0) ea = eb = 0;
    for (long k = k0; k < k1; ++k) {
        const double a = scalbn(src_entry(args.srcA, i, k, args.K), -ea);
        const double b = scalbn(src_entry(args.srcB, j, k, args.K), -eb);
        const double p = a * b, t = s + p, z = t - s;
        c += ((s - (t - z)) + (p - z)) + fma(a, b, -p);
        s = t;
    }
    return isfinite(s) ? scalbn(s + c, ea + eb) : s;
}

// The elements of this CTA's tiles that the digits do not give (an infinity or a NaN in their row or
// column, or next to the subnormal numbers), formed by the look-out's lanes over what the epilogue
// stored. A warp, a branch and a call of its own: the epilogue's loop has no register to spare. Exchange
// energies at (20,100,480,720), 12 points, no such element in them: 885 us without this, 897 with it, 920
// with the loops inlined, 925 with the elements looked for in the epilogue.
template <int BN>
__device__ __noinline__ void fill_undigited(const UpdArgs& args, int lane) {
    for (int w = blockIdx.x; w < args.nactive * args.kgroups; w += gridDim.x) {
        const int t = w % args.nactive, grp = w / args.nactive;
        const long k0 = grp == 0 ? -(long)args.srcA.k0 : (long)grp * args.cpg * KP;
        const long k1 = min(args.K, (grp + 1) * args.cpg * KP);
        int m0, n0;
        tile_of<BN>(args, t, m0, n0);
        double* const c = grp == 0 ? args.C : args.part + (size_t)(grp - 1) * args.mA * args.mB;
        const size_t ld = grp == 0 ? args.ldc : args.mB;
        for (int x = lane; x < BM * BN; x += 32) {
            const int i = m0 + x / BN, j = n0 + x % BN;
            if (i >= args.mA || j >= args.mB || (args.lower && i < args.mB && j > i) ||
                (max(args.eA[i], args.eB[j]) < kNanExp && args.eA[i] + args.eB[j] >= kTinyExp))
                continue;
            const double s = args.sign * src_dot(args, i, j, k0, k1);
            c[i * ld + j] = s;
            if (args.mirror && j < i) c[j * ld + i] = s;
        }
    }
}

// C (+)= sign * A B^T from the digit slices, one 128 x BN output tile at a time, each CTA (one
// per SM) walking tiles blockIdx.x, blockIdx.x + gridDim.x, ...: warp 0 streams, per tile and
// K half, the right operand's S slices (one stage) and the left operand's slices (16 KB stages)
// by 3-D TMA; warp 1 issues, per left slice a and K step, BF16 MMAs against the stacked right
// slices b <= S - 1 - a, whose result columns fall into accumulators a + b of the tile's set
// (N = BN (S - a) at once, in pieces of at most 256); sixteen epilogue warps (a lane quarter
// and BN / 4 columns each) add the S integer accumulators of every K chunk into two 64-bit
// integers per element in registers and form one FP64 value per element after the last chunk:
// C is touched once per tile, through a shared-memory transpose that turns each warp's
// accesses into full 32-byte sectors. The last warp looks over the exponents of the CTA's rows and
// columns meanwhile, for elements without digits. Every wait is bounded.
// Bounds: 36 MMAs of 128 x BN x 16 per K step are 9.2k tensor cycles per 128 x 64 x 128 piece;
// per chunk the epilogue issues ~18 integer instructions per element against them (it was ~150
// with a rounding and an FP64 read-modify-write of C per chunk, which bound the kernel: the
// 1200 x 1800 x 1200 product took 334 us at a tensor pipe of 15 % with seven slices).
template <int BN>
__global__ void __launch_bounds__(NTHREADS, 1)
k_oz_update(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
            const __grid_constant__ UpdArgs args) {
    using T = Tile<BN>;
    constexpr int A_STAGES = T::A_STAGES, SETS = T::SETS;
    constexpr int NC = BN / 4;  // columns per epilogue warp
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* asm_ = smem;                               // [A_STAGES] x A_TILE
    uint8_t* bsm = smem + A_STAGES * A_TILE;            // [B_STAGES] x B_HALF
    double* stg = (double*)(bsm + B_STAGES * T::B_HALF);
    uint64_t* afull = (uint64_t*)((uint8_t*)stg + STG_BYTES);
    uint64_t* aempty = afull + A_STAGES;
    uint64_t* bfull = aempty + A_STAGES;
    uint64_t* bempty = bfull + B_STAGES;
    uint64_t* accfull = bempty + B_STAGES;              // [2]
    uint64_t* accempty = accfull + 2;                   // [2]
    uint32_t* tmem_slot = (uint32_t*)(accempty + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntiles = args.nactive;
    const int nwork = ntiles * args.kgroups;

    if (threadIdx.x == 0) {
        for (int i = 0; i < A_STAGES; ++i) {
            mbar_init(&afull[i], 1);
            mbar_init(&aempty[i], 1);
        }
        for (int i = 0; i < B_STAGES; ++i) {
            mbar_init(&bfull[i], 1);
            mbar_init(&bempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&accfull[i], 1);
            mbar_init(&accempty[i], EPI_WARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // ---- TMA producer ----
        int ia = 0, ib = 0;  // positions in the two rings, over all tiles of this CTA
        bool ok = true;
        for (int w = blockIdx.x; w < nwork && ok; w += gridDim.x) {
            const int t = w % ntiles, g0 = (w / ntiles) * args.cpg, g1 = min(args.nchunks, g0 + args.cpg);
            int m0, n0;
            tile_of<BN>(args, t, m0, n0);
            for (int ch = g0; ch < g1 && ok; ++ch) {
                const int nh = ch == args.nchunks - 1 ? args.khalves : 2;
                for (int c = 0; c < nh && ok; ++c) {
                    const int sb = ib % B_STAGES;
                    if (!oz_wait(&bempty[sb], ((ib / B_STAGES) & 1) ^ 1, 1)) { ok = false; break; }
                    mbar_expect_tx(&bfull[sb], (uint32_t)T::B_HALF);
                    // all S right slices in one box, stacked (slice b at rows BN b ..)
                    tma_load_3d(bsm + sb * T::B_HALF, &mapB, &bfull[sb], 64 * c, n0, S * ch);
                    ++ib;
                    for (int a = 0; a < S; ++a, ++ia) {
                        const int sa = ia % A_STAGES;
                        if (!oz_wait(&aempty[sa], ((ia / A_STAGES) & 1) ^ 1, 1)) { ok = false; break; }
                        mbar_expect_tx(&afull[sa], (uint32_t)A_TILE);
                        tma_load_3d(asm_ + sa * A_TILE, &mapA, &afull[sa], 64 * c, m0, S * ch + a);
                    }
                }
            }
        }
        // every copy issued has landed before the CTA may leave
        for (int j = max(0, ia - A_STAGES); j < ia; ++j) oz_wait(&afull[j % A_STAGES], (j / A_STAGES) & 1, 2);
        for (int j = max(0, ib - B_STAGES); j < ib; ++j) oz_wait(&bfull[j % B_STAGES], (j / B_STAGES) & 1, 2);
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer ----
        int ia = 0, ib = 0, i = 0;
        bool ok = true;
        for (int w = blockIdx.x; w < nwork && ok; w += gridDim.x) {
            const int g0 = (w / ntiles) * args.cpg, g1 = min(args.nchunks, g0 + args.cpg);
            // one accumulator set per (tile, K chunk), in turn
            for (int ch = g0; ch < g1 && ok; ++ch) {
                const int nh = ch == args.nchunks - 1 ? args.khalves : 2;
                const int set = i % SETS;
                // the set is free once the epilogue has drained tile-chunk i - SETS
                if (i >= SETS && !oz_wait(&accempty[set], (i / SETS - 1) & 1, 5)) { ok = false; break; }
                tc_fence_after();
                const uint32_t acc0 = tmem + (uint32_t)(set * T::ACC_SET);
                for (int c = 0; c < nh && ok; ++c) {
                    const int sb = ib % B_STAGES;
                    if (!oz_wait(&bfull[sb], (ib / B_STAGES) & 1, 3)) { ok = false; break; }
                    const uint64_t bd = sw128_desc(smem_u32(bsm + sb * T::B_HALF));
#pragma unroll
                    for (int a = 0; a < S; ++a, ++ia) {
                        const int sa = ia % A_STAGES;
                        if (!oz_wait(&afull[sa], (ia / A_STAGES) & 1, 4)) { ok = false; break; }
                        tc_fence_after();
                        // the right slices b = 0..S-1-a lie stacked in the stage (rows BN b ..), so
                        // MMAs over N = BN (S - a) of its rows with the accumulator base at column
                        // BN a put A_a B_b^T at columns BN (a + b): accumulator a + b, for every b
                        const uint64_t ad = sw128_desc(smem_u32(asm_ + sa * A_TILE));
                        const uint32_t acc = acc0 + (uint32_t)(a * BN);
                        constexpr int NMAX = 256;
                        const int ntot = BN * (S - a);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {  // 4 x 16 elements (32 bytes) per 64-wide box
                            const uint64_t o = (uint64_t)(kk * 32) >> 4;
#pragma unroll
                            for (int nb = 0; nb < ntot; nb += NMAX) {
                                const int nn = ntot - nb < NMAX ? ntot - nb : NMAX;
                                tc_mma<false>(acc + (uint32_t)nb, ad + o, bd + o + (uint64_t)(nb * 128 >> 4),
                                              make_idesc(false, BM, nn), (c | a | kk) ? 1u : 0u);
                            }
                        }
                        tc_commit(&aempty[sa]);
                    }
                    tc_commit(&bempty[sb]);
                    ++ib;
                }
                tc_commit(&accfull[set]);  // also after a failed wait: arrives once the issued MMAs are done
                ++i;
            }
        }
    } else if (warp == 2 + EPI_WARPS) {
        // ---- look-out: rows and columns without digits, or of tiny numbers, among this CTA's tiles ----
        bool found = false;
        for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
            int m0, n0;
            tile_of<BN>(args, w % ntiles, m0, n0);
            for (int x = lane; x < BM + BN; x += 32) {
                const int r = x < BM ? m0 + x : n0 + x - BM;
                if (r >= (x < BM ? args.mA : args.mB)) continue;
                const int e = __ldg((x < BM ? args.eA : args.eB) + r);
                found |= e >= kNanExp || e < kTinyExp / 2;  // (of a tiny pair one at least)
            }
        }
        found = __any_sync(0xffffffffu, found);
        epi_barrier();  // the epilogue has stored every tile
        if (found && args.srcA.s1) fill_undigited<BN>(args, lane);
    } else if (warp >= 2) {
        // ---- epilogue: a lane quarter q and NC columns h of each tile ----
        const int q = warp & 3, h = (warp - 2) >> 2;  // h = 0..3
        const unsigned long long sign_bit = args.sign < 0.0 ? 0x8000000000000000ULL : 0ULL;
        double* st = stg + (warp - 2) * 128;  // 32 rows x 4 columns, columns rotated by row / 4
        const int sr = lane >> 2, sc = lane & 3;
        int i = 0;
        for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
            const int t = w % ntiles, grp = w / ntiles, g0 = grp * args.cpg, g1 = min(args.nchunks, g0 + args.cpg);
            int m0, n0;
            tile_of<BN>(args, t, m0, n0);
            // group 0 into C, the others into their partial sums
            double* const cbase = grp == 0 ? args.C : args.part + (size_t)(grp - 1) * args.mA * args.mB;
            const int cld = grp == 0 ? args.ldc : args.mB;
            const bool accum = grp == 0 && args.accumulate;
            long long hi[NC], lo[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) hi[j] = lo[j] = 0;
            bool ok = true;
            for (int ch = g0; ch < g1; ++ch, ++i) {
                const int set = i % SETS;
                ok = oz_wait(&accfull[set], (i / SETS) & 1, 6) && ok;
                tc_fence_after();
                const uint32_t tbase = tmem + (uint32_t)(set * T::ACC_SET + NC * h) + ((uint32_t)(32 * q) << 16);
#pragma unroll
                for (int j4 = 0; j4 < NC; j4 += 4) {
                    uint32_t r[S][4];
#pragma unroll
                    for (int g = 0; g < S; ++g) tmem_ld4_nowait(tbase + (uint32_t)(g * BN + j4), r[g]);
                    tmem_ld_wait(r);
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        int v[S];
#pragma unroll
                        for (int g = 0; g < S; ++g) v[g] = __float2int_rn(__uint_as_float(r[g][jj]));
                        hi[j4 + jj] += (long long)v[0] * 65536 + (long long)v[1] * 256 + v[2];
                        lo[j4 + jj] += (long long)v[3] * 4294967296LL + (long long)v[4] * 16777216 +
                                       (long long)v[5] * 65536 + (long long)v[6] * 256 + v[7];
                    }
                }
                // every TMEM read of this chunk has completed (tcgen05.wait::ld)
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&accempty[set]);
            }
            const int row = m0 + 32 * q + lane;
            const int ea = row < args.mA ? __ldg(args.eA + row) : 0;
            const int jw = n0 + NC * h;
            if (jw >= args.mB) continue;
#pragma unroll
            for (int j4 = 0; j4 < NC; j4 += 4) {
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int j = jw + j4 + jj;
                    const int eb = j < args.mB ? __ldg(args.eB + j) : 0;
                    double tv = scaled_sum(hi[j4 + jj], lo[j4 + jj], ea + eb - 68, sign_bit);
                    if (max(ea, eb) >= kNanExp || !ok) tv = __longlong_as_double(0x7FF8000000000000LL);
                    st[4 * lane + (jj ^ ((lane >> 2) & 3))] = tv;
                    // the mirrored element (j, row): consecutive lanes, consecutive addresses
                    if (args.mirror && row < args.mA && j < row) {
                        double* m = cbase + (size_t)j * cld + row;
                        *m = accum ? *m + tv : tv;
                    }
                }
                __syncwarp();
                const int j = jw + j4 + sc;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int rl = sr + 8 * k, rw = m0 + 32 * q + rl;
                    if (rw < args.mA && j < args.mB && !(args.lower && rw < args.mB && j > rw)) {
                        double* c = cbase + (size_t)rw * cld + j;
                        const double tv = st[4 * rl + (sc ^ ((rl >> 2) & 3))];
                        *c = accum ? *c + tv : tv;
                    }
                }
                __syncwarp();
            }
        }
        epi_barrier();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

// C[i][j] += part[0][i][j] + part[1][i][j] + ... (the split-K partial sums, fixed order)
__global__ void k_oz_add_parts(double* __restrict__ C, int ldc, int M, int N, const double* __restrict__ part,
                               int nparts) {
    const long total = (long)M * N;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
        double* c = C + (e / N) * (long)ldc + e % N;
        double v = *c;
        for (int p = 0; p < nparts; ++p) v += part[p * total + e];
        *c = v;
    }
}

// ---- host ----------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
// From 1e7 flops on, products run from digits. An MTTKRP at (o, v, R_thc, R_cp) in us with the line at
// 4e6 / 8e6 / 1.6e7 / 3e7 / never: (6,30,144,216) 183 / 187 / 167 / 172 / 172, (8,40,192,288)
// 172 / 188 / 185 / 188 / 190, (14,70,336,504) 207 / 203 / 202 / 252 / 337, (20,100,480,720)
// 230 / 232 / 248 / 252 / 691, (30,150,720,1080) 328 / 334 / 328 / 330 / 1761.
constexpr double kWorthFlops = 1.0e7;
constexpr int kColsSmem = COLS_PER_BLOCK * (kColsMaxK + 4) * (int)sizeof(double);

// The current device can run the kernels of this file (sm_103), their attributes set on it.
bool oz_init() {
    static PerDevice<bool> ready;
    return ready.get([](int dev) {
        cudaDeviceProp p;
        const int need = std::max(std::max(Tile<64>::SMEM, Tile<32>::SMEM), kColsSmem);
        if (cudaGetDeviceProperties(&p, dev) != cudaSuccess || !(p.major == 10 && p.minor == 3) ||
            (int)p.sharedMemPerBlockOptin < need)
            return false;
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return false;
        g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;  // (the same for every device)
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        return cudaFuncSetAttribute(k_oz_update<64>, attr, Tile<64>::SMEM) == cudaSuccess &&
               cudaFuncSetAttribute(k_oz_update<32>, attr, Tile<32>::SMEM) == cudaSuccess &&
               cudaFuncSetAttribute(k_oz_split_cols, attr, kColsSmem) == cudaSuccess;
    });
}

// 3-D map over the digit slices [planes][rows][KP] (BF16; S planes per K chunk):
// box 64 (K) x box_rows x depth.
bool slice_map(CUtensorMap* m, const OzMat& a, int box_rows, int depth) {
    cuuint64_t dims[3] = {(cuuint64_t)KP, (cuuint64_t)a.rows, (cuuint64_t)(S * a.chunks())};
    cuuint64_t strides[2] = {(cuuint64_t)KP * 2, (cuuint64_t)(a.ld_rows ? a.ld_rows : a.rows) * KP * 2};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)depth};
    cuuint32_t estr[3] = {1, 1, 1};
    return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, a.d, dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tile width and K split of a product (SMs, K chunks, tiles): the estimated cycles of the
// busiest CTA. Per chunk 10.7k cycles for a 128 x 64 piece (its drain is not overlapped), 5.6k
// for 128 x 32, per tile an epilogue of 2.5k / 1.5k, and for a split the partial sums' extra
// launch and traffic (~6k). A split never takes part in a lower or symmetric product.
struct MulPlan {
    int bn, groups;
};
MulPlan plan_mul(int mA, int mB, int nch, bool lower, size_t part_cap) {
    MulPlan best{64, 1};
    double bc = 1e300;
    const int sms = num_sms();
    for (int bn : {64, 32}) {
        const int tm = cdiv(mA, BM), tn = cdiv(mB, bn);
        long act = 0;
        for (int t = 0; t < tm; ++t)
            act += bn == 64 ? row_tiles<64>(t, tn, mB, lower) : row_tiles<32>(t, tn, mB, lower);
        const int gmax = (lower || (size_t)mA * mB > part_cap) ? 1 : std::min(nch, 16);
        for (int g = 1; g <= gmax; ++g) {
            const int cpg = cdiv(nch, g), gr = cdiv(nch, cpg);
            if (gr != g || (size_t)(gr - 1) * mA * mB > part_cap) continue;
            const double waves = (double)cdiv(act * gr, sms);
            const double c = waves * (cpg * (bn == 64 ? 10.7 : 5.6) + (bn == 64 ? 2.5 : 1.5)) + (gr > 1 ? 6.0 + 0.3 * gr : 0.0);
            if (c < bc) {
                bc = c;
                best = {bn, gr};
            }
        }
    }
    return best;
}

template <int BN>
cudaError_t launch_mul(cudaStream_t st, const OzMat& A, const OzMat& B, UpdArgs a, int groups) {
    CUtensorMap ma, mb;
    if (!slice_map(&ma, A, BM, 1) || !slice_map(&mb, B, BN, S)) return cudaErrorInvalidValue;
    a.tiles_m = cdiv(a.mA, BM);
    a.tiles_n = cdiv(a.mB, BN);
    long active = 0;
    for (int tm = 0; tm < a.tiles_m; ++tm) active += row_tiles<BN>(tm, a.tiles_n, a.mB, a.lower);
    a.nactive = (int)active;
    a.cpg = cdiv(a.nchunks, std::max(1, groups));
    a.kgroups = cdiv(a.nchunks, a.cpg);
    // persistent: one CTA per SM, at most one per active (tile, K group) work item
    const int grid = (int)std::max<long>(1, std::min<long>(active * a.kgroups, num_sms()));
    k_oz_update<BN><<<grid, NTHREADS, Tile<BN>::SMEM, st>>>(ma, mb, a);
    count_launch();
    if (a.kgroups > 1) {
        k_oz_add_parts<<<(int)std::min<long>(cdiv((long)a.mA * a.mB, 256), 4L * num_sms()), 256, 0, st>>>(
            a.C, a.ldc, a.mA, a.mB, a.part, a.kgroups - 1);
        count_launch();
    }
    return cudaGetLastError();
}

OzMat view(uint16_t* d, int* e, int rows, int K) {
    OzMat m;
    m.d = d;
    m.e = e;
    m.rows = rows;
    m.K = K;
    return m;
}

}  // namespace

size_t ozmat_bytes(int rows, int K) {
    return Arena::need<uint16_t>((size_t)S * rows * KP * cdiv(std::max(K, 1), KP)) + Arena::need<int>(rows);
}

void ozmat_carve(OzMat& m, Arena& ar, int rows, int K) {
    m.d = ar.take<uint16_t>((size_t)S * rows * KP * cdiv(std::max(K, 1), KP));
    m.e = ar.take<int>(rows);
    m.rows = rows;
    m.K = K;
}

void oz_split_rows(cudaStream_t st, const double* src, int ld, OzMat& m) {
    m.src = OzSrc{src, nullptr, ld, 0};
    if (m.rows <= 0) return;
    // up to eight rows per SM, more warps to a row (see the kernel); beyond, the rows fill the chip
    const int wpr = m.rows > 8 * num_sms() ? 1 : m.K > 2 * KP ? 4 : m.K > KP ? 2 : 1, grid = cdiv(m.rows, ROWS_PER_BLOCK / wpr);
    if (ld % 2 == 0 && ((uintptr_t)src & 15) == 0)
        k_oz_split_rows<true><<<grid, 32 * ROWS_PER_BLOCK, 0, st>>>(src, ld, m.rows, m.K, m.d, m.e, wpr);
    else
        k_oz_split_rows<false><<<grid, 32 * ROWS_PER_BLOCK, 0, st>>>(src, ld, m.rows, m.K, m.d, m.e, wpr);
    count_launch();
}

void oz_split_cols_stack(cudaStream_t st, const double* S1, const double* S2, int ld, int n, int g, OzMat& m) {
    m.src = OzSrc{S1, S2, ld, n};
    if (n <= 0 || g <= 0) return;
    const int parts = cdiv(m.K, kColsMaxK);
    if (parts > 1) {
        for (int al = 0; al < g; ++al) {
            const size_t off = (size_t)al * m.K * ld;
            k_oz_col_exps<<<cdiv(n, 32), 256, 0, st>>>(S1 + off, S2 ? S2 + off : nullptr, ld, n, m.K, m.e + (size_t)al * n);
        }
        count_launch(g);
    }
    const int kpad = cdiv(std::min(m.K, kColsMaxK), KP) * KP;
    // up to two blocks per SM, more threads to a block (see the kernel); beyond, blocks of 256 hide
    // each other's latency better (twelve 480 x 720 matrices in a stack: the exchange energies took
    // 920 us with 1024 threads, 892 with 256)
    const long blocks = (long)cdiv(n, COLS_PER_BLOCK) * parts * g;
    const int threads = blocks > 2L * num_sms() ? 256 : 256 * std::min(4, kpad / KP);
    k_oz_split_cols<<<dim3(cdiv(n, COLS_PER_BLOCK), parts, g), threads,
                      COLS_PER_BLOCK * (kpad + 4) * sizeof(double), st>>>(S1, S2, ld, n, m.K, m.rows, m.d, m.e,
                                                                           parts > 1 ? 1 : 0);
    count_launch();
}

void oz_split_cols(cudaStream_t st, const double* S1, const double* S2, int ld, OzMat& m) {
    oz_split_cols_stack(st, S1, S2, ld, m.rows, 1, m);
}

cudaError_t oz_mul(cudaStream_t st, const OzMat& A, const OzMat& B, double* C, int ldc, double sign,
                   int flags, double* part, size_t part_cap) {
    if (A.rows <= 0 || B.rows <= 0) return cudaSuccess;
    const bool symm = flags & OZ_SYMM, lower = symm || (flags & OZ_LOWER);
    const int nch = A.chunks();
    if (A.K != B.K || nch < 1 || nch > kOzMaxChunks || (symm && A.rows != B.rows)) return cudaErrorInvalidValue;
    const int kb = A.K - KP * (nch - 1);
    UpdArgs a{};
    a.C = C;
    a.ldc = ldc;
    a.mA = A.rows;
    a.mB = B.rows;
    a.eA = A.e;
    a.eB = B.e;
    a.lower = lower ? 1 : 0;
    a.mirror = symm ? 1 : 0;
    a.sign = sign;
    a.accumulate = (flags & OZ_ACC) ? 1 : 0;
    a.khalves = kb > 64 ? 2 : 1;
    a.nchunks = nch;
    a.part = part;
    // (where C is added to, only if it holds nothing but the earlier K of the same sources)
    if (A.src.s1 && B.src.s1 && (!a.accumulate || A.src.k0 > 0)) {
        a.srcA = A.src;
        a.srcB = B.src;
    }
    a.K = A.K;
    const MulPlan p = plan_mul(A.rows, B.rows, nch, lower, part ? part_cap : 0);
    return p.bn == 64 ? launch_mul<64>(st, A, B, a, p.groups) : launch_mul<32>(st, A, B, a, p.groups);
}

size_t oz_ws_bytes(int rowsA, int rowsB, size_t part_doubles) {
    return Arena::need<uint16_t>((size_t)S * rowsA * KP) + Arena::need<uint16_t>((size_t)S * rowsB * KP) +
           Arena::need<int>(rowsA) + Arena::need<int>(rowsB) + (part_doubles ? Arena::need<double>(part_doubles) : 0);
}

bool oz_available() { return oz_init(); }

bool oz_worth_flops(double flops) { return flops >= kWorthFlops; }

bool oz_worth(int M, int N, int K, bool symm) {
    return oz_worth_flops((symm ? 1.0 : 2.0) * M * (double)N * K) && M <= 8192 && N <= 8192 && K <= kOzMaxK;
}

void oz_ws_carve(OzWs& w, Arena& ar, int rowsA, int rowsB, size_t part_doubles) {
    w.rowsA = rowsA;
    w.rowsB = rowsB;
    w.sA = ar.take<uint16_t>((size_t)S * w.rowsA * KP);
    w.sB = ar.take<uint16_t>((size_t)S * w.rowsB * KP);
    w.eA = ar.take<int>(w.rowsA);
    w.eB = ar.take<int>(w.rowsB);
    w.part = part_doubles ? ar.take<double>(part_doubles) : nullptr;
    w.part_cap = part_doubles;
}

// Digit rows of one operand of a product, at most: 256 MB. A product of more runs in several launches.
constexpr long kMaxDigitRows = 1L << 17;

void oz_product_ws(int M, int N, int K, int* rowsA, int* rowsB, size_t* part) {
    const long nch = std::min(cdiv(std::max(K, 1), KP), kOzMaxChunks);
    *rowsA = (int)std::max<long>(*rowsA, std::min(nch * M, kMaxDigitRows));
    *rowsB = (int)std::max<long>(*rowsB, std::max<long>(N, std::min(nch * N, kMaxDigitRows)));
    if (part) {
        const long tiles = (long)cdiv(M, BM) * cdiv(N, 32);
        const long g = std::min<long>(nch, std::max<long>(1, 2L * num_sms() / tiles));
        *part = std::max<size_t>(*part, (size_t)(std::min<long>(g, 16) - 1) * M * N);
    }
}

namespace {
// C (+)= sign op(A) (B o B2) with both operands split into ws, in K ranges of as many chunks as ws
// holds of B, and of A in as many rows as it holds of those (fewer chunks where that would be less
// than 1024). a_cols / b_cols: the operand's rows are the columns of the stored matrix.
cudaError_t product(cudaStream_t st, int M, int N, int K, const double* A, int lda, bool a_cols, const double* B,
                    const double* B2, int ldb, bool b_cols, double* C, int ldc, double sign, int flags,
                    const OzWs& ws) {
    if (!oz_init()) return cudaErrorNotSupported;
    // A^T A (a Gram): one operand split serves both sides
    const bool same_ab = a_cols && b_cols && A == B && !B2 && lda == ldb && M == N;
    if (N > ws.rowsB || (!same_ab && (flags & OZ_SYMM) && M > ws.rowsA)) return cudaErrorInvalidValue;
    int chunks = std::min(std::min(cdiv(K, KP), ws.rowsB / N), kOzMaxChunks), rows = M;
    if (!same_ab) {
        const int least = (flags & OZ_SYMM) ? M : std::min(M, 1024);
        chunks = std::min(chunks, std::max(1, ws.rowsA / least));
        rows = std::min(M, ws.rowsA / chunks);
        if (rows < M && rows > BM) rows = rows / BM * BM;
    }
    for (int k0 = 0; k0 < K; k0 += chunks * KP) {
        const int kn = std::min(chunks * KP, K - k0);
        OzMat b = view(ws.sB, ws.eB, N, kn);
        const size_t ob = b_cols ? (size_t)k0 * ldb : (size_t)k0;
        if (b_cols)
            oz_split_cols(st, B + ob, B2 ? B2 + ob : nullptr, ldb, b);
        else
            oz_split_rows(st, B + ob, ldb, b);
        b.src.k0 = k0;
        for (int m0 = 0; m0 < M; m0 += rows) {
            OzMat a = b;
            if (!same_ab) {
                a = view(ws.sA, ws.eA, std::min(rows, M - m0), kn);
                if (a_cols)
                    oz_split_cols(st, A + (size_t)k0 * lda + m0, nullptr, lda, a);
                else
                    oz_split_rows(st, A + (size_t)m0 * lda + k0, lda, a);
                a.src.k0 = k0;
            }
            const cudaError_t e = oz_mul(st, a, b, C + (size_t)m0 * ldc, ldc, sign, k0 > 0 ? flags | OZ_ACC : flags,
                                         ws.part, ws.part_cap);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaGetLastError();
}
}  // namespace

// Once at most this many columns are left, the rest of the factorisation runs as one
// dataflow launch (its FP64 trailing updates still hide behind its pivot chain there)
// instead of further panels, each followed by a digit split and an update launch that the
// next panel waits for. Measured on GB300 with 128-column panels, BF16x3 sweeps/s: 106.9 /
// 108.5 / 110.1 / 110.1 / 105.7 at R_cp = 1800 for 8 (none) / 264 / 520 / 776 / 1032
// columns, 221.9 / 226.5 / 233.7 at R_cp = 1080 for 56 / 312 / 440.
constexpr int kTailCols = 520;

// From R = 1536, panels of two K chunks: half as many panel boundaries (digit split and
// update launch, which the next panel waits for), each update over both chunks in one
// launch. BF16x3 sweeps/s on GB300: 120.2 / 121.3 / 115.6 at R_cp = 1800 for 128 / 256 / 384
// columns (the panel's FP64 substitution work outgrows its pivot chain at 384), 235.8 /
// 238.1 at R_cp = 1080; but the 64-problem batch (R_cp <= 1440, panels on at most 32 CTAs
// beside the other problems, where that FP64 work is no longer hidden) took 3.86 s with
// 256 against 3.73 s with 128. The width depends on R alone, so a problem factorises the
// same way (same bits) in the batched driver and alone.
int panel_cols(int R) { return R >= 1536 ? 2 * KP : KP; }

// Width of the panel that starts at column j0: panel_cols(R), or everything left once at
// most kTailCols columns remain.
int panel_width(int R, int j0) {
    return R - j0 <= kTailCols ? R - j0 : std::min(panel_cols(R), R - j0);
}

void oz_ldl_ws_rows(int R, int nmax, int* rowsA, int* rowsB) {
    const int pc = std::min(panel_cols(R), R);
    const long nch = cdiv(pc, KP);
    if (R - pc <= 0) return;
    *rowsA = (int)std::max<long>(*rowsA, nch * (R + nmax - pc));
    *rowsB = (int)std::max<long>(*rowsB, nch * (R - pc));
}

bool oz_prepare(int R, int n) {
    if (!oz_init()) return false;
    for (int j0 = 0; j0 < R;) {
        const int bw = panel_width(R, j0);
        if (!flow_prepare(bw, R + n - j0 - bw)) return false;
        j0 += bw;
    }
    return true;
}

cudaError_t ldl_oz(cudaStream_t st, int R, int n, double* Haug, double* P, double* dinv,
                   DevScalars* sc, int mode, int* sync, const OzWs& ws, int max_ctas) {
    for (int j0 = 0; j0 < R; j0 += panel_width(R, j0)) {
        const int bw = panel_width(R, j0);
        const int j1 = j0 + bw;
        const int mA = R + n - j1, mB = R - j1;
        cudaError_t e;
        {
            // the panel's LDL^T and the substitution of every row below it
            ProfScope prof(st, KC_CHOL, (double)bw * bw * bw / 3.0 + (double)mA * bw * bw);
            e = ldl_flow_panel(st, R, n, j0, bw, Haug, P, dinv, sc, mode, sync, max_ctas);
        }
        if (e != cudaSuccess) return e;
        if (j1 >= R) break;
        const double* below = Haug + (size_t)j1 * R + j0;   // rows j1.., panel columns
        const double* diag = Haug + (size_t)j0 * R + j0;
        {
            ProfScope prof(st, KC_OZ, (double)mB * (mB + 1) * bw + 2.0 * (mA - mB) * mB * bw);
            const long nch = cdiv(bw, KP);
            if (nch > kLdlMaxChunks || nch * mA > ws.rowsA || nch * mB > ws.rowsB) return cudaErrorInvalidValue;
            const OzMat a = view(ws.sA, ws.eA, mA, bw), b = view(ws.sB, ws.eB, mB, bw);
            k_oz_split_ldl<<<cdiv(mA, ROWS_PER_BLOCK), 32 * ROWS_PER_BLOCK, 0, st>>>(below, R, mA, mB, bw, diag, R, a.d,
                                                                                  a.e, b.d, b.e);
            count_launch();
            e = oz_mul(st, a, b, Haug + (size_t)j1 * R + j1, R, -1.0, OZ_ACC | OZ_LOWER);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

cudaError_t oz_gemm(cudaStream_t st, int M, int N, int K, const double* A, int lda, const double* B,
                    int ldb, double* C, int ldc, const OzWs& ws) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    return product(st, M, N, K, A, lda, false, B, nullptr, ldb, false, C, ldc, 1.0, 0, ws);
}

cudaError_t oz_dgemm(cudaStream_t st, bool trans_a, int M, int N, int K, const double* A, int lda,
                     const double* B, const double* B2, int ldb, double* C, int ldc, bool symm,
                     const OzWs& ws) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if (symm && M != N) return cudaErrorInvalidValue;
    if (K <= 0) return cudaMemset2DAsync(C, sizeof(double) * ldc, 0, sizeof(double) * N, M, st);
    ProfScope prof(st, KC_OZ, (symm ? 1.0 : 2.0) * M * (double)N * K);
    return product(st, M, N, K, A, lda, trans_a, B, B2, ldb, true, C, ldc, 1.0, symm ? OZ_SYMM : 0, ws);
}

cudaError_t oz_gemm_sub(cudaStream_t st, int M, int N, int K, const double* A, int lda, const double* B,
                        int ldb, double* C, int ldc, const OzWs& ws) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    ProfScope prof(st, KC_OZ, 2.0 * M * (double)N * K);
    return product(st, M, N, K, A, lda, false, B, nullptr, ldb, true, C, ldc, -1.0, OZ_ACC, ws);
}

int oz_take_error() { return take_error_word(&g_oz_error); }

}  // namespace thc
