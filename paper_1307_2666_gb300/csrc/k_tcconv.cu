// Direct sum y = K v on a uniform grid (the residual operator of the
// refinement, Sec. 5; K as assembled in Sec. 3.1, Eq. (3.1)) on the tcgen05
// tensor cores, in exact integer digits.
//
// Every table entry t and every source value v is written as a short sum of
// signed 8-bit digits against a power-of-two scale,
//     t = 2^eT sum_s dT_s 2^-8(s+1),  v = 2^eX sum_t dX_t 2^-8(t+1),
// |dT_s|, |dX_t| <= 128 (round-to-nearest digit extraction in FP64, exact).
// Digits are BF16 integers, so dT_s * dX_t is exact in the tensor core and
// a sum of up to 1024 of them (<= 2^24) is exact in its FP32 accumulator.
// Products of digit pairs (s, t) of the same class k = s + t carry the same
// weight 2^(eT + eX - 8(k + 2)), so they share one accumulator column: the
// MMA of table digit s writes the columns of classes s .. s + t_max.  The
// columns are converted to integers and added into 64-bit integer class sums,
// so the only rounding is the dropped digits (below 2^-55 of max|t| max|v|)
// and the final FP64
// combination of eight class sums.  Table digits 0..6 and source digits
// 0..7 are kept, and pairs with s + t >= 8 are not formed.
//
// Shorter digit sets serve the residuals of the refinement that are not the
// last one (their error only enters the next correction, which the last,
// full-digit residual then measures): with KD classes (4, 5 or 6) the kernel
// keeps table and source digits 0..KD-1 and the pairs with s + t < KD.  Per
// term the dropped part is below (KD + 1) 2^(-2 - 8 KD) of 2^(eT + eX) <= 16
// max|t| max|v|, and it behaves like a sum of independent terms of mean zero
// (round-to-nearest digits): on the 2D log-kernel grid with Gaussian sources
// the relative error of y is ~6e-9 with KD = 4, ~2e-11 with KD = 5 and ~1e-13
// with KD = 6, at every N from 4096 to 262144 (exact integer convolutions of
// the digits).
//
// On a grid K_ij depends only on the offset i - j, so the kernel block of a
// tile of 128 targets on one grid line against 128 sources on another line is
// a Toeplitz matrix in the last coordinate.  With the target rows taken in
// reverse order it is a Hankel matrix A[i][q] = v[i + q], whose 8 x 8 core
// matrices depend only on the sum of their block indices: the shared-memory
// operand stores the 31 distinct core matrices of each digit slice once and
// the MMA descriptor walks them with equal leading and stride offsets (144 B:
// a 16-B gap after every core matrix keeps the builders' stores free of
// shared-memory bank conflicts).
//
// The block also depends only on the distance d along the slowest axis, so
// the two source lines at i0 - d and i0 + d of a target line i0 meet the same
// block and are added before the product: the sum of two 8-bit digits has
// magnitude at most 256, which BF16 still holds exactly.  That halves the
// MMAs of the sum over all pairs.  The blocks of several target lines i0,
// i0 + 1, ... at the same d are the same too: one MMA takes 32 columns
// (target line, right-hand side) per source digit, four lines of eight
// right-hand sides up to 32 lines of one, so that few right-hand sides cost
// few MMAs.
//
// What bounds it: an M = 128 MMA takes N / 2 cycles of the tensor pipe and
// reads 4 KB of A and 32 N bytes of B from shared memory at 128 B per clock,
// so a slot (7 table digits x 128 sources) is 4,096 cycles of math, ~3,850 of
// shared-memory reads by the MMAs and ~1,850 of loads and stores by the
// builders on the same L1 data path: that path is full (ncu: 49% + 55% of its
// wavefronts), the tensor pipe is not.  Folding the mirror lines leaves the
// cost of a slot nearly as it was and halves the slots; the folded operand is
// built by threads from L2 (two loads, an add and a store per 16 bytes).
// Measured on a GB300, whole matvec, before (one MMA quarter per source line,
// 8-column padding, whole tiles per CTA) and after: n = 1024 x 8 right-hand
// sides 458 -> 272 ms (classes 6, 5, 4: 357, 290, 248 -> 222, 190, 152 ms; with
// two drains per slot, see below, 281, 236, 208 and 162), n = 512 x 8 30.8 ->
// 17.5 ms, n = 64 x 1 0.29 -> 0.16 ms, 3D n = 24 x 3 2.8 -> 0.94 ms.
//
// The epilogue's conversions of column sums to integers run at 16 per clock, so
// how often a column is drained matters (a drain per 64 sources is 4,096
// cycles a slot at 8 classes).  A column sums products of a table digit (at most
// 128) and a folded source digit; over the 128 sources of a slot that is below
// 2^24, exact in FP32, whenever the digits of every source chunk satisfy
// sum_t sum_q |d_t[q]| <= 2^16 (kFullSlot).  Random digits do (mean 57,300 of 7
// digits, spread 1,100); the digit kernel finds the largest sum, and the two
// accumulators then take a slot each.  Otherwise (coherent sources) they take
// half a slot each: 7 pairs x 64 sources x 2^15 < 2^24 for any digits.  The
// epilogue drains one while the MMAs fill the other.
//
// The slots of all tiles form one sequence (tile, middle source coordinate,
// source chunk, distance) that is cut into equal ranges, one per CTA, so
// every size fills the chip whatever its number of tiles; a tile cut by a
// range boundary leaves its integer class sums, which are exact and therefore
// independent of the cut, in a partial buffer that fixup_kernel adds up.
//
// CTA roles (800 threads, persistent, one CTA per SM, TMEM 512 columns):
//   warps 0-15   epilogue: TMEM -> integer class sums -> FP64 y (one thread
//                per target row and 8 of the 32 columns),
//   warp 16      one thread: the MMAs,
//   warps 17-24  builders: the folded source digits and the Hankel operand
//                from mirrored digit rows.
// Slots flow through a 2-stage shared-memory ring (3 stages for the short
// sums, whose stages are smaller).  Four neighbouring classes are kept as one
// 64-bit sum.  Every wait is bounded; on time-out the kernel sets *status = 1,
// drains its own MMAs, frees TMEM and returns.
#include <cuda_bf16.h>
#include <algorithm>
#include <cstdlib>
#include <mutex>
#include <utility>
#include <vector>
#include <cstdint>
#include "hif_types.h"
#include "launch.h"
#include "tc_ptx.cuh"

namespace hif {
namespace {

constexpr int TM = 128;                         // targets per tile (TMEM lanes)
constexpr int KC = 128;                         // sources per chunk
constexpr int ST = 7;                           // table digits stored
constexpr int SX = 8;                           // source digits stored per chunk
constexpr int NR = 8;                           // right-hand sides per launch
constexpr int NBLK = (TM + KC) / 8 - 1;         // distinct Hankel core matrices per slice (31)
constexpr int CM = 144;                         // core-matrix stride: 128 B + 16 B so that the
                                                // builders' 16-B row stores of consecutive core
                                                // matrices fall in different bank groups
constexpr int A_SLICE = NBLK * CM;              // bytes
constexpr int CHUNK = SX * NR * KC * 2;         // bytes of one source chunk: (digit, rhs) rows x KC, BF16
constexpr int NCOL = 32;                        // columns per class: (target line, rhs)
constexpr int DBLK = NCOL * KC * 2;             // the B rows of one digit
constexpr int NST_MAX = 3;                      // deepest ring of the variants below
constexpr int ACCB = NCOL * 8;                  // TMEM columns of one accumulator: (class, column)
constexpr int NACC = 2;                         // accumulators: the two halves of a slot's sources
constexpr int ACC = ACCB * NACC;                // TMEM columns allocated
constexpr int NEPI = 512;                       // epilogue threads: 4 column groups x 128 rows
constexpr int NBUILD = 256;                     // builder threads
constexpr int NTHR = NEPI + 32 + NBUILD;
constexpr int NGRP = 2;                         // 64-bit class sums (classes 4 g .. 4 g + 3)
constexpr int CARRY = 4096;                     // slots between carries of the class sums
constexpr int PART = NGRP * 8 * NEPI;           // int64 values of one partial tile
constexpr long long WAIT_CYCLES = 4000000000LL; // ~2 s at GB300 clocks

static_assert(7 * (KC / NACC) * 128 * 256 <= (1 << 24), "exact FP32 accumulation of half a slot");
// largest sum of |digit| over a source chunk's digits (the first SUMT) for
// which a whole slot is exact: two chunks are added, table digits are <= 128
constexpr unsigned kFullSlot = (1u << 24) / 2 / 128;
constexpr int SUMT = 7;                         // most digit pairs of a class
// S[1] gains less than 2 x 2^24 x (2^24 + 2^17) per slot
static_assert(4294967296.0 * 65536.0 * 2.1 * CARRY < 9.2e18, "64-bit class sums between carries");

// The variant with KD digit classes (8: every class, the full sum; 4, 5 or
// 6: the short sums).  Columns of table digit s: B rows (source digit t,
// line, rhs) for t below nt(s) = ncols(s) / 32, written to the accumulator
// columns (class s + t, line, rhs), i.e. from column 32 s on; the full sum
// takes s + t <= 7 except for the odd counts rounded down, a short one every
// pair with s + t < KD.
template <int KD>
struct Digits {
    static constexpr int ST = KD == 8 ? 7 : KD;          // table digits read
    static constexpr int SX = KD;                        // source digits read
    static constexpr int A_BYTES = ST * A_SLICE;
    static constexpr int B_BYTES = SX * DBLK;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int NST = KD == 8 ? 2 : 3;         // ring depth within 227 KB of shared memory
    static constexpr int NPAIR = ST * NBLK;             // (slice, core matrix) build items per slot
    __host__ __device__ static constexpr int ncols(int s) {
        return KD == 8 ? (s == 0 ? 256 : s <= 2 ? 192 : s <= 4 ? 128 : 64) : 32 * (KD - s);
    }
    static constexpr int NG = (KD + 3) / 4;             // 64-bit class sums kept
    static_assert(STAGE % 16 == 0 && A_BYTES % 16 == 0 && NPAIR <= NBUILD, "stage layout");
    static_assert(NST <= NST_MAX && NST * STAGE + 1024 + 256 <= 232448, "shared memory");
    static_assert(ncols(0) == 32 * KD && ncols(ST - 1) >= 32, "column map");
};
__host__ __device__ constexpr int coloff(int s) { return 32 * s; }
static_assert(coloff(6) + Digits<8>::ncols(6) <= ACCB && Digits<8>::ncols(0) == ACCB, "column map");

__device__ __forceinline__ int scale_exp(unsigned long long maxbits) {
    const double m = __longlong_as_double((long long)maxbits);
    return m > 0.0 ? ilogb(m) + 2 : 0;             // |x| 2^-e < 1/2
}

// digits of u in [-1/2, 1/2): d_k = rint(256 r_k), r_{k+1} = 256 r_k - d_k
__device__ __forceinline__ void digits8(double u, float (&d)[8]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const double x = u * 256.0;
        const double dk = rint(x);
        d[k] = (float)dk;
        u = x - dk;
    }
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&p);
}

struct Bars {
    uint64_t full[NST_MAX];     // both operands built (NBUILD arrivals)
    uint64_t mma_done[NST_MAX];
    uint64_t acc_full[NACC];    // accumulator written (1 commit); taken in turn
    uint64_t acc_empty[NACC];   // accumulator drained (NEPI arrivals)
    uint64_t drain;
    uint32_t tmem;
    int abort;
};

__device__ __forceinline__ bool wait_bounded(uint64_t* bar, uint32_t parity, volatile int* abort) {
    const long long t0 = clock64();
    while (true) {
        if (tc::mbar_try_wait(bar, parity)) return true;
        if (*abort) return false;
        if (clock64() - t0 > WAIT_CYCLES) {
            *abort = 1;
            return false;
        }
    }
}

}  // namespace

// ---- digit tables ---------------------------------------------------------

__global__ void tc_maxabs_kernel(const double* x, int64_t n, int cols, int64_t ld,
                                 unsigned long long* out) {
    for (int c = 0; c < cols; ++c) {
        double m = 0.0;
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
            m = fmax(m, fabs(x[e + ld * c]));
        for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(out + c, (unsigned long long)__double_as_longlong(m));
    }
}

// Mirrored table rows: R[s][dl][idx] = digit s of T(dl, |Z0 - idx|) (0 where
// |Z0 - idx| >= n), idx in [0, RL), Z0 = 128 nc - 1, RL = 256 nc; dl indexes
// the offsets of all but the last coordinate.
__global__ void tc_table_rows_kernel(const double* table, int n, int64_t lines, int nc,
                                     const unsigned long long* tmax, __nv_bfloat16* R) {
    const int64_t RL = 256LL * nc, Z0 = 128LL * nc - 1;
    const int eT = scale_exp(*tmax);
    const int64_t tot = lines * RL;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t dl = e / RL, idx = e % RL;
        const int64_t z = Z0 - idx, az = z < 0 ? -z : z;
        float d[8];
        if (az < n) {
            digits8(ldexp(table[dl + lines * az], -eT), d);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) d[k] = 0.f;
        }
#pragma unroll
        for (int s = 0; s < ST; ++s) R[((int64_t)s * lines + dl) * RL + idx] = __float2bfloat16_rn(d[s]);
    }
}

// Source digits chunk by chunk for nrv = 2^lg right-hand sides (nr of them in
// use): element (digit t, rhs r, source q) of chunk ch at
// (((ch * SX + t) * (KC/8) + q/8) * nrv + r) * 8 + q % 8 (BF16 units).
__global__ void tc_source_digits_kernel(const double* v, int64_t N, int n, int64_t lines, int nc, int r0, int nr,
                                        int lg, int sx, int xshift, const unsigned long long* xmax, uint4* XB,
                                        unsigned* chunk_max) {
    const int64_t tot = (lines * nc * (KC / 8)) << lg;
    __shared__ unsigned sums[256];               // sum of |digit| per (chunk, rhs) of this block
    unsigned most = 0;
    for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x; e0 < tot; e0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = e0 + threadIdx.x;
        sums[threadIdx.x] = 0;
        __syncthreads();
        if (e < tot) {
            const int r = (int)(e & ((1 << lg) - 1));
            const int kb = (int)((e >> lg) % (KC / 8));
            const int64_t ch = (e >> lg) / (KC / 8);
            const int64_t J = ch / nc;
            const int c = (int)(ch % nc);
            float d[8][8];                       // [source][digit]
            const int ex = (r < nr ? scale_exp(xmax[r]) : 0) + xshift;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int64_t jl = (int64_t)KC * c + 8 * kb + q;
                if (r < nr && jl < n) {
                    digits8(ldexp(v[J * n + jl + N * (r0 + r)], -ex), d[q]);
                } else {
#pragma unroll
                    for (int t = 0; t < 8; ++t) d[q][t] = 0.f;
                }
            }
            float sum = 0.f;
#pragma unroll
            for (int t = 0; t < SX; ++t) {
                if (t >= sx) break;
                uint4 w;
                w.x = pack2(d[0][t], d[1][t]);
                w.y = pack2(d[2][t], d[3][t]);
                w.z = pack2(d[4][t], d[5][t]);
                w.w = pack2(d[6][t], d[7][t]);
                XB[(((ch * SX + t) * (KC / 8) + kb) << lg) + r] = w;
                if (t < SUMT)
#pragma unroll
                    for (int q = 0; q < 8; ++q) sum += fabsf(d[q][t]);
            }
            // (chunk in the block, rhs): a chunk's 16 << lg threads are neighbours
            atomicAdd(&sums[((threadIdx.x >> lg) / (KC / 8) << lg) + r], (unsigned)sum);
        }
        __syncthreads();
        most = max(most, sums[threadIdx.x]);
        __syncthreads();
    }
    for (int o = 16; o; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    if (threadIdx.x % 32 == 0 && most > 0) atomicMax(chunk_max, most);
}

// ---- the tensor-core sum ----------------------------------------------------

struct TcConvArgs {
    const __nv_bfloat16* R;     // mirrored table digit rows
    const unsigned char* XB;    // source digit chunks
    const unsigned long long* tmax;
    const unsigned long long* xmax;   // NR entries, then the largest chunk sum of |digit|
    double* ybuf;               // N x nrhs, grid order
    long long* part;            // two partial tiles per CTA
    int64_t N;
    int n;
    int64_t lines;              // n^(dim-1)
    int dim;
    int nc;                     // target chunks = source chunks per line
    int lg;                     // log2 of the right-hand sides per line in the 32 columns
    int64_t slots;              // slots of all tiles
    int r0, nr;
    int xshift;                 // sources scaled to |u| < 2^-(1 + xshift)
    int* status;
    int stall;                  // test of the bounded waits: issue no MMA at all
};

namespace {

// A tile is NL = 32 / 2^lg target lines i0 .. i0 + NL - 1 along the slowest
// axis (with the middle coordinate i1 in 3D) and one chunk b of 128 targets
// along the last.  Its slots are (j1, c, d): middle source coordinate (3D),
// source chunk, distance along the slowest axis 0 .. dmax, d fastest, so
// consecutive slots read neighbouring source lines.
struct Tiles {
    int n, mid, nc, NL, ngrp;
    __host__ __device__ explicit Tiles(const TcConvArgs& a)
        : n(a.n), mid(a.dim == 3 ? a.n : 1), nc(a.nc), NL(NCOL >> a.lg), ngrp((a.n + NL - 1) / NL) {}
    __host__ __device__ int dmax(int g) const {
        const int lo = g * NL, hi = (lo + NL < n ? lo + NL : n) - 1;
        return hi > n - 1 - lo ? hi : n - 1 - lo;
    }
    __host__ __device__ int64_t tile_slots(int g) const { return (int64_t)(dmax(g) + 1) * mid * nc; }
    __host__ __device__ int64_t group_slots(int g) const { return tile_slots(g) * mid * nc; }
};

int64_t total_slots(const TcConvArgs& a) {
    const Tiles t(a);
    int64_t s = 0;
    for (int g = 0; g < t.ngrp; ++g) s += t.group_slots(g);
    return s;
}

__device__ __forceinline__ int64_t range_start(const TcConvArgs& a, int cta, int ctas) {
    return a.slots / ctas * cta + a.slots % ctas * cta / ctas;
}

// Position in the slot sequence: tile q of group g and slot `off` inside it;
// q = middle target coordinate i1 * nc + target chunk b.
struct Place {
    int g, q;
    int64_t off;
    __device__ Place(const Tiles& t, int64_t slot) {
        g = 0;
        for (int64_t s; g < t.ngrp - 1 && slot >= (s = t.group_slots(g)); ++g) slot -= s;
        const int64_t per = t.tile_slots(g);
        q = (int)(slot / per);
        off = slot % per;
    }
    __device__ void next_tile(const Tiles& t) {
        off = 0;
        if (++q == t.mid * t.nc) {
            q = 0;
            ++g;
        }
    }
};

// Class sums of one (row, column): S[0] = sum_k v_k 2^(8 (3 - k)) over classes
// 0..3, S[1] the same over classes 4..7, 2^-32 of S[0]'s unit.  The carry
// leaves 32 bits in S[1]; S[0] then stays below N 2^38 (1 + 2^-6).
__device__ __forceinline__ void carry(long long (&S)[NGRP]) {
    S[0] += S[1] >> 32;
    S[1] &= 0xffffffffLL;
}
__device__ __forceinline__ double from_sums(const long long (&S)[NGRP], int e2) {
    return ldexp((double)S[0] + (double)S[1] * (1.0 / 4294967296.0), e2 - 40);
}

__device__ __forceinline__ void store_row(const TcConvArgs& a, int i0, int i1, int b, int row, int col, double y) {
    const int l = col >> a.lg, r = col & ((1 << a.lg) - 1);
    const int il = TM * b + TM - 1 - row, line = i0 + l;
    if (il >= a.n || line >= a.n || r >= a.nr) return;
    const int64_t L = a.dim == 3 ? (int64_t)line * a.n + i1 : line;
    a.ybuf[L * a.n + il + a.N * (a.r0 + r)] = y;
}

// 16 bytes of read-only data, zero when !on.  Volatile: the builders keep a
// fixed number of loads in flight; hoisting more of them spills registers,
// and spills go through the same L1 data path that the MMAs read from.
__device__ __forceinline__ uint4 load16(const uint4* p, bool on) {
    uint4 v;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
        "mov.u32 %0, 0;\n\tmov.u32 %1, 0;\n\tmov.u32 %2, 0;\n\tmov.u32 %3, 0;\n\t"
        "@p ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w)
        : "l"(p), "r"((uint32_t)on));
    return v;
}

__device__ __forceinline__ uint32_t add2(uint32_t x, uint32_t y) {
    const __nv_bfloat162 s =
        __hadd2(*reinterpret_cast<const __nv_bfloat162*>(&x), *reinterpret_cast<const __nv_bfloat162*>(&y));
    return *reinterpret_cast<const uint32_t*>(&s);
}

}  // namespace

template <int KD>
__global__ void __launch_bounds__(NTHR, 1) tc_conv_kernel(TcConvArgs a) {
    using C = Digits<KD>;
    constexpr int NST = C::NST, STAGE = C::STAGE, A_BYTES = C::A_BYTES, NG = C::NG;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    Bars* bars = (Bars*)(smem + NST * STAGE);
    volatile int* abort = &bars->abort;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

    if (threadIdx.x == 0) {
        for (int i = 0; i < NST; ++i) {
            tc::mbar_init(&bars->full[i], NBUILD);
            tc::mbar_init(&bars->mma_done[i], 1);
        }
        for (int i = 0; i < NACC; ++i) {
            tc::mbar_init(&bars->acc_full[i], 1);
            tc::mbar_init(&bars->acc_empty[i], NEPI);
        }
        tc::mbar_init(&bars->drain, 1);
        bars->abort = 0;
        tc::fence_mbar_init();
    }
    if (warp == 0) tc::tmem_alloc(&bars->tmem, ACC);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = bars->tmem;
    const int64_t first = range_start(a, blockIdx.x, gridDim.x);
    const int64_t count = range_start(a, blockIdx.x + 1, gridDim.x) - first;
    // a whole slot per accumulator, or half of one
    const bool whole = *reinterpret_cast<const unsigned*>(a.xmax + NR) <= kFullSlot;

    if (warp == NEPI / 32) {
        // ---------------------------------------------------------- issuer
        // (counters are stepped, not divided, and the thread does nothing
        // but wait and issue: its scalar work between MMA batches shows up
        // as tensor-pipe idle time)
        if (lane == 0) {
            int st = 0;
            uint32_t ph = 0;
            bool ok = true;
            int64_t use = 0;                     // accumulators filled
            for (int64_t si = 0; si < (a.stall ? 0 : count); ++si) {
                if (!wait_bounded(&bars->full[st], ph, abort)) {
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                // descriptors of the stage; moving the start address by 16 B
                // adds 1 to the descriptor (addresses stay below 256 KB)
                const uint32_t a_st = tc::smem_addr(smem + st * STAGE);
                const uint64_t a0 = tc::sdesc(a_st, CM, CM);
                const uint64_t b0 = tc::sdesc(a_st + A_BYTES, 128, (KC / 8) * 128);
                // slice by slice: consecutive MMAs of one slice read
                // overlapping Hankel windows and keep N and D fixed, which
                // the tensor core streams faster than alternating slices
                // (the first MMA, slice 0 with every column, initializes
                // the accumulator; the others add into it)
                auto fill = [&](int k0, int k1) {
                    const int ab = (int)(use & 1);
                    if (use >= NACC && !wait_bounded(&bars->acc_empty[ab], (uint32_t)((use / NACC - 1) & 1), abort))
                        return false;
                    tc::tc_fence_after();
#pragma unroll
                    for (int s = 0; s < C::ST; ++s) {
                        const uint64_t as = a0 + (uint64_t)(s * A_SLICE / 16);
                        const uint32_t dst = tmem + ACCB * ab + coloff(s);
#pragma unroll 4
                        for (int kk = k0; kk < k1; ++kk)
                            tc::mma_bf16(dst, as + (uint64_t)(2 * CM / 16) * kk, b0 + (uint64_t)16 * kk,
                                         tc::idesc_bf16_f32(TM, C::ncols(s)), !(s == 0 && kk == k0));
                    }
                    tc::mma_commit(&bars->acc_full[ab]);
                    ++use;
                    return true;
                };
                ok = whole ? fill(0, KC / 16) : fill(0, KC / 32) && fill(KC / 32, KC / 16);
                if (!ok) break;
                tc::mma_commit(&bars->mma_done[st]);
                if (++st == NST) {
                    st = 0;
                    ph ^= 1;
                }
            }
            // drain: every MMA issued so far
            tc::mma_commit(&bars->drain);
            const long long t0 = clock64();
            while (!tc::mbar_try_wait(&bars->drain, 0) && clock64() - t0 < WAIT_CYCLES) {}
            if (!ok) *abort = 1;
        }
    } else if (warp > NEPI / 32) {
        // ------------------------------------------------------- builders
        // source operand: thread bt builds the 16-byte units (digit t, column
        // 8 (2 hi + p) + row8, source octet kb) for every t and p = 0, 1: the
        // digits of source lines i - d and i + d added; a missing line is
        // zero.  table operand: threads below NPAIR build one (slice, core
        // matrix) item each.
        const int bt = threadIdx.x - (NEPI + 32);
        const int row8 = bt & 7, kb = (bt >> 3) & 15, hi = bt >> 7;
        const int64_t Z0 = 128LL * a.nc - 1, RL = 256LL * a.nc;
        const int64_t dig = (int64_t)(KC / 8) << a.lg;                   // uint4 per digit of a chunk
        const int64_t chunk = SX * dig, line = (a.dim == 3 ? a.n : 1) * (int64_t)a.nc * chunk;
        const int as = bt / NBLK, am = bt % NBLK;                        // table item
        int lp[2], up[2];                                                // target line and unit inside a digit
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int col = 8 * (2 * hi + p) + row8;
            lp[p] = col >> a.lg;
            up[p] = (kb << a.lg) + (col & ((1 << a.lg) - 1));
        }
        unsigned char* const bdst = smem + A_BYTES + (2 * hi) * (KC / 8) * 128 + kb * 128 + row8 * 16;
        const int64_t dp = (int64_t)(lp[1] - lp[0]) * line + up[1] - up[0];
        const Tiles tl(a);
        Place pl(tl, first);
        int st = 0, gs = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int left = (int)count; left > 0 && ok;) {
            // the slots of one (tile, j1, c): distances d .. dmax, pointers stepped
            const int dmax = tl.dmax(pl.g), i0 = pl.g * tl.NL, i1 = pl.q / tl.nc, b = pl.q % tl.nc;
            const int c = (int)(pl.off / (dmax + 1) % tl.nc), j1 = (int)(pl.off / (dmax + 1) / tl.nc);
            int d = (int)(pl.off % (dmax + 1));
            const int dend = min(dmax + 1, d + left);
            left -= dend - d;
            pl.off += dend - d;
            if (pl.off == tl.tile_slots(pl.g)) pl.next_tile(tl);
            const int64_t dl = d + (int64_t)(a.dim == 3 ? a.n : 0) * (i1 > j1 ? i1 - j1 : j1 - i1);
            const uint4* tsrc = reinterpret_cast<const uint4*>(
                a.R + ((int64_t)as * a.lines + dl) * RL + (Z0 - ((int64_t)TM * b + TM - 1 - (int64_t)KC * c)) + 8 * am);
            const uint4* pm =
                reinterpret_cast<const uint4*>(a.XB) + ((int64_t)j1 * a.nc + c) * chunk + up[0] + (i0 + lp[0] - d) * line;
            const uint4* pp = pm + 2 * d * line;
            for (; d < dend; ++d, tsrc += RL / 8, pm -= line, pp += line) {
                const uint4 t0 = load16(tsrc, bt < C::NPAIR), t1 = load16(tsrc + 1, bt < C::NPAIR);
                if (gs >= NST && !wait_bounded(&bars->mma_done[st], ph ^ 1, abort)) {
                    ok = false;
                    break;
                }
                ++gs;
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int i = i0 + lp[p];
                    const bool vm = i < a.n && i >= d, vp = d > 0 && i + d < a.n;
                    unsigned char* dst = bdst + st * STAGE + p * (KC / 8) * 128;
                    constexpr int TB = (C::SX + 1) / 2;                                // digits in flight
#pragma unroll
                    for (int t0 = 0; t0 < C::SX; t0 += TB) {
                        uint4 um[TB], uq[TB];
#pragma unroll
                        for (int t = 0; t < TB; ++t) {
                            if (t0 + t < C::SX) {
                                um[t] = load16(pm + p * dp + (t0 + t) * dig, vm);
                                uq[t] = load16(pp + p * dp + (t0 + t) * dig, vp);
                            }
                        }
#pragma unroll
                        for (int t = 0; t < TB; ++t)
                            if (t0 + t < C::SX)
                                *reinterpret_cast<uint4*>(dst + (t0 + t) * DBLK) =
                                    make_uint4(add2(um[t].x, uq[t].x), add2(um[t].y, uq[t].y),
                                               add2(um[t].z, uq[t].z), add2(um[t].w, uq[t].w));
                    }
                }
                if (bt < C::NPAIR) {
                    const uint32_t wd[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
                    uint4* dst = reinterpret_cast<uint4*>(smem + st * STAGE + as * A_SLICE + am * CM);
#pragma unroll
                    for (int rho = 0; rho < 8; ++rho) {
                        uint32_t o[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            o[q] = (rho & 1) ? __funnelshift_r(wd[rho / 2 + q], wd[rho / 2 + q + 1], 16)
                                             : wd[rho / 2 + q];
                        dst[rho] = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                }
                tc::fence_proxy_async_smem();
                tc::mbar_arrive(&bars->full[st]);
                if (++st == NST) {
                    st = 0;
                    ph ^= 1;
                }
            }
        }
    } else {
        // ------------------------------------------------------- epilogue
        // warp w: columns 8 (w / 4) .. + 7 of every class, TMEM lane quarter w % 4
        const int quad = warp & 3, cg = warp >> 2;
        const int row = 32 * quad + lane;
        long long S[8][NGRP];
        const int nh = whole ? 1 : NACC;
        unsigned use = 0;                        // accumulators drained (mod 2^32)
        bool ok = true;
        const Tiles tl(a);
        Place pl(tl, first);
        for (int left = (int)count; left > 0 && ok;) {
            const int64_t per = tl.tile_slots(pl.g);
            const int nsl = (int)(per - pl.off < left ? per - pl.off : left);
#pragma unroll
            for (int e = 0; e < 8; ++e)
#pragma unroll
                for (int g = 0; g < NGRP; ++g) S[e][g] = 0;
            for (int s = 0; s < nsl && ok; ++s) {
#pragma unroll 1                                // (unrolled, the sums spill)
                for (int h = 0; h < nh; ++h, ++use) {
                    // (a warp gives up as one: the TMEM loads below are collective)
                    if (!__all_sync(0xffffffffu, wait_bounded(&bars->acc_full[use & 1], (uint32_t)(use >> 1) & 1, abort))) {
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after();
                    const uint32_t tbase = tmem + ACCB * (use & 1) + 8 * cg + ((uint32_t)(32 * quad) << 16);
#pragma unroll
                    for (int k = 0; k < KD; k += 2) {
                        float v[2][8];
                        if (k + 1 < KD) tc::tmem_ld8x2(tbase + NCOL * k, tbase + NCOL * (k + 1), v[0], v[1]);
                        else tc::tmem_ld8(tbase + NCOL * k, v[0]);
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            if (k + u < KD) {
                                const int g = (k + u) / 4, sh = 8 * (3 - (k + u) % 4);
#pragma unroll
                                for (int e = 0; e < 8; ++e)
                                    S[e][g] += (long long)__float2int_rn(v[u][e]) * (1 << sh);
                            }
                    }
                    tc::tc_fence_before();
                    tc::mbar_arrive(&bars->acc_empty[use & 1]);
                }
                if (s % CARRY == CARRY - 1 || s == nsl - 1) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) carry(S[e]);
                }
            }
            if (!ok) break;
            if (nsl == per) {
                const int eT = scale_exp(*a.tmax);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int col = 8 * cg + e, r = col & ((1 << a.lg) - 1);
                    store_row(a, pl.g * tl.NL, pl.q / tl.nc, pl.q % tl.nc, row, col,
                              from_sums(S[e], eT + scale_exp(a.xmax[r]) + a.xshift));
                }
            } else {
                // a tile begun by an earlier CTA (0) or left to the next one (1)
                long long* part = a.part + (int64_t)(2 * blockIdx.x + (pl.off == 0 ? 1 : 0)) * PART;
#pragma unroll
                for (int g = 0; g < NG; ++g)
#pragma unroll
                    for (int e = 0; e < 8; ++e) part[(g * 8 + e) * NEPI + threadIdx.x] = S[e][g];
            }
            left -= nsl;
            pl.next_tile(tl);
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && bars->abort) atomicExch(a.status, 1);
    if (warp == 0) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, ACC);
    }
}

// The tiles cut by range boundaries: block x adds up the partial class sums
// of the tile in which CTA x + 1 starts, if CTA x is the one that began it.
__global__ void __launch_bounds__(256) tc_fixup_kernel(TcConvArgs a, int ctas, int ng) {
    const Tiles t(a);
    const int cta = blockIdx.x + 1;
    const int64_t start = range_start(a, cta, ctas);
    const Place p(t, start);
    if (p.off == 0 || start - p.off < range_start(a, cta - 1, ctas)) return;
    const int64_t end = start - p.off + t.tile_slots(p.g);
    const int eT = scale_exp(*a.tmax);
    int last = cta;
    while (last < ctas && range_start(a, last, ctas) < end) ++last;
    const int e = blockIdx.y * blockDim.x + threadIdx.x;       // (column of 8, epilogue thread)
    long long S[NGRP] = {0, 0};
#pragma unroll
    for (int g = 0; g < NGRP; ++g) {
        if (g >= ng) continue;
        const long long* src = a.part + (int64_t)g * 8 * NEPI + e;
        long long s = src[(int64_t)(2 * (cta - 1) + 1) * PART];
#pragma unroll 8
        for (int q = cta; q < last; ++q) s += src[(int64_t)(2 * q) * PART];
        S[g] = s;
    }
    carry(S);
    const int th = e % NEPI, col = 8 * (th >> 7) + e / NEPI, r = col & ((1 << a.lg) - 1);
    store_row(a, p.g * t.NL, p.q / t.nc, p.q % t.nc, th & 127, col,
              from_sums(S, eT + scale_exp(a.xmax[r]) + a.xshift));
}

// ---- host side ----------------------------------------------------------------

namespace {
std::mutex g_tm_mu;
bool g_tm_on = false;
std::vector<std::pair<cudaEvent_t, cudaEvent_t>> g_tm_ev;
}  // namespace

void tc_timing_set(bool enable) {
    std::lock_guard<std::mutex> lk(g_tm_mu);
    g_tm_on = enable;
}

cudaError_t tc_timing_collect(double* ms, int64_t* launches) {
    std::lock_guard<std::mutex> lk(g_tm_mu);
    double tot = 0.0;
    cudaError_t err = cudaSuccess;
    for (auto& e : g_tm_ev) {
        float t = 0.f;
        cudaError_t r = cudaEventSynchronize(e.second);
        if (r == cudaSuccess) r = cudaEventElapsedTime(&t, e.first, e.second);
        if (r != cudaSuccess && err == cudaSuccess) err = r;
        tot += t;
        cudaEventDestroy(e.first);
        cudaEventDestroy(e.second);
    }
    if (ms) *ms = tot;
    if (launches) *launches = (int64_t)g_tm_ev.size();
    g_tm_ev.clear();
    return err;
}

size_t tc_table_rows_bytes(int n, int dim) {
    const int nc = (n + KC - 1) / KC;
    const int64_t lines = dim == 2 ? (int64_t)n : (int64_t)n * n;
    return sizeof(__nv_bfloat16) * (size_t)ST * lines * 256 * nc;
}

size_t tc_source_digits_bytes(int n, int dim, int num_sms) {
    const int nc = (n + KC - 1) / KC;
    const int64_t lines = dim == 2 ? (int64_t)n : (int64_t)n * n;
    // + two partial tiles per CTA of the launch
    return (size_t)(lines * nc) * CHUNK + (size_t)2 * std::max(num_sms, 1) * PART * sizeof(long long);
}

cudaError_t launch_tc_table(const double* table, int n, int dim, unsigned long long* tmax, void* R,
                            cudaStream_t st) {
    const int nc = (n + KC - 1) / KC;
    const int64_t lines = dim == 2 ? (int64_t)n : (int64_t)n * n;
    const int64_t tot = lines * n;
    cudaError_t e = cudaMemsetAsync(tmax, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    note_launch();
    tc_maxabs_kernel<<<(int)std::min<int64_t>((tot + 255) / 256, 1024), 256, 0, st>>>(table, tot, 1, tot, tmax);
    note_launch();
    const int64_t rows = lines * 256LL * nc;
    tc_table_rows_kernel<<<(int)std::min<int64_t>((rows + 255) / 256, 152 * 16), 256, 0, st>>>(
        table, n, lines, nc, tmax, (__nv_bfloat16*)R);
    return cudaGetLastError();
}

namespace {
// the kernel variant of KD digit classes and its shared-memory size (the
// opt-in above 48 KB is set once per variant)
template <int KD>
cudaError_t tc_variant(void (**fn)(TcConvArgs), size_t* smem) {
    static bool attr_set = false;
    *fn = tc_conv_kernel<KD>;
    *smem = (size_t)Digits<KD>::NST * Digits<KD>::STAGE + sizeof(Bars) + 1024;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(tc_conv_kernel<KD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)*smem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    return cudaSuccess;
}
}  // namespace

cudaError_t launch_direct_grid_tc(const GridDirectArgs& a, const void* R, const unsigned long long* tmax,
                                  void* XB, unsigned long long* xmax, int* status, int num_sms, int classes,
                                  cudaStream_t st) {
    const int64_t N = a.dim == 2 ? (int64_t)a.n * a.n : (int64_t)a.n * a.n * a.n;
    if (N == 0) return cudaSuccess;
    if (classes < 4 || classes == 7 || classes > 8) return cudaErrorInvalidValue;
    const int nc = (a.n + KC - 1) / KC;
    const int64_t lines = a.dim == 2 ? (int64_t)a.n : (int64_t)a.n * a.n;
    const int eb = (int)std::min<int64_t>((N * a.nrhs + 255) / 256, 152 * 16);
    void (*kfn)(TcConvArgs) = nullptr;
    size_t smem = 0;
    {
        cudaError_t e = classes == 8   ? tc_variant<8>(&kfn, &smem)
                        : classes == 6 ? tc_variant<6>(&kfn, &smem)
                        : classes == 5 ? tc_variant<5>(&kfn, &smem)
                                       : tc_variant<4>(&kfn, &smem);
        if (e != cudaSuccess) return e;
    }
    grid_scatter_kernel_launch(a, N, eb, st);
    // the 64-bit class sums hold N 2^38 for N <= 2^24; larger sums start from
    // smaller top digits
    int xshift = 0;
    while ((N >> xshift) > ((int64_t)1 << 24)) ++xshift;
    for (int r0 = 0; r0 < a.nrhs; r0 += NR) {
        const int nr = std::min(NR, a.nrhs - r0);
        cudaError_t e = cudaMemsetAsync(xmax, 0, (NR + 1) * sizeof(unsigned long long), st);
        if (e != cudaSuccess) return e;
        note_launch();
        tc_maxabs_kernel<<<(int)std::min<int64_t>((N + 255) / 256, 1024), 256, 0, st>>>(a.vbuf + N * r0, N, nr, N,
                                                                                       xmax);
        // right-hand sides of this launch, rounded up to a power of two; the
        // rest of the 32 columns per class are target lines
        const int lg = nr > 4 ? 3 : nr > 2 ? 2 : nr > 1 ? 1 : 0;
        const int64_t items = (lines * nc * (KC / 8)) << lg;
        note_launch();
        tc_source_digits_kernel<<<(int)std::min<int64_t>((items + 255) / 256, 152 * 16), 256, 0, st>>>(
            a.vbuf, N, a.n, lines, nc, r0, nr, lg, classes, xshift, xmax, (uint4*)XB,
            (unsigned*)(xmax + NR));
        TcConvArgs t{};
        t.R = (const __nv_bfloat16*)R;
        t.XB = (const unsigned char*)XB;
        t.tmax = tmax;
        t.xmax = xmax;
        t.ybuf = a.ybuf;
        t.N = N;
        t.n = a.n;
        t.lines = lines;
        t.dim = a.dim;
        t.nc = nc;
        t.lg = lg;
        t.part = (long long*)((unsigned char*)XB + lines * nc * (int64_t)CHUNK);
        t.slots = total_slots(t);
        t.xshift = xshift;
        t.r0 = r0;
        t.nr = nr;
        t.status = status;
        {
            // test of the bounded waits (HIF_TC_TEST_STALL=1): the MMA thread
            // issues nothing, the builders' stage-reuse waits run out after
            // ~2 s and the call returns HIF_ETIMEOUT with the context intact
            const char* e = getenv("HIF_TC_TEST_STALL");
            t.stall = (e && atoi(e) != 0) ? 1 : 0;
        }
        const int grid = (int)std::min<int64_t>(t.slots, num_sms);
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        {
            std::lock_guard<std::mutex> lk(g_tm_mu);
            if (g_tm_on && classes == 8 && cudaEventCreate(&e0) == cudaSuccess &&
                cudaEventCreate(&e1) == cudaSuccess) {
                cudaEventRecord(e0, st);
                g_tm_ev.emplace_back(e0, e1);
            } else {
                e1 = nullptr;
            }
        }
        note_launch();
        kfn<<<grid, NTHR, smem, st>>>(t);
        if (grid > 1) {
            note_launch();
            tc_fixup_kernel<<<dim3(grid - 1, 8 * NEPI / 256), 256, 0, st>>>(t, grid, (classes + 3) / 4);
        }
        if (e1) cudaEventRecord(e1, st);
    }
    grid_finish_kernel_launch(a, N, eb, st);
    return cudaGetLastError();
}

}  // namespace hif
