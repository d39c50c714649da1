// oz_gemm.cu - FP64 stage GEMMs on the FP16 tensor cores (tcgen05).
//
//   D[z][row][col] = sum_k A[z][row][k] B[z][col][k], FP64 in and out, results
//   scattered by the stage's index map: the one-index contractions S1-S4 of
//   Eq. (2bse) (arXiv:1905.01180, Sec. III) and of the time-linear history.
//
// GB300 executes two FP64 FMAs per SM and clock, so the plain FP64 GEMM
// (k_gemm64_stage) is bound by them at 1.2 TFLOP/s.  Here every element is
// split into seven 8-bit digits (oz_digits.h), the digit products run as FP16
// MMAs whose FP32 sums are exact integers, and the epilogue puts a result
// together with integer instructions only.  Results whose error that would leave
// large against sum |x y| (graded rows, blocks that hardly couple) are found by an
// eighth MMA and summed again by FMAs, so that the path is as accurate as FMA chains
// for operands of any scaling (oz_accept; tests/test_oz_graded.py).
//
// Whole calls, FMA chain -> here: Heun step at N = 24, 301 points 309 -> 17.2 ms; 40
// self-energies at N = 33 78 -> 3.5 ms; Heun step at N = 10, 501 points 23.8 -> 1.6 ms.
// Without the check of the results: 15.8, 2.8 and 1.4 ms.  What is summed again costs
// most for matrices near a diagonal or nearly real (a propagation's start; three
// time-linear steps at N = 48 137 -> 30 ms, 12 without the check) and at worst, N = 24
// with imaginary parts of 1e-3, takes 0.6 of the FMA chain's time (50 -> 30 ms for 200
// self-energies; 14 ms where rows and columns span 1e-6 .. 1e6).
//
// What bounds it: the latency of two chains of instructions that are each half busy,
// the epilogue's (about 70 a result) and the converter's (about 53 an element).
#include <cuda_fp16.h>

#include <algorithm>

#include "gkba_internal.cuh"
#include "oz_digits.h"
#include "ptx_sm103.cuh"

namespace gkba {

namespace {

constexpr int kOzBM = 128;       // rows per tile (tensor-memory lanes)
constexpr int kOzLbo = kOzBM * 16 + 32;  // bytes between the 8-wide K chunks of a digit plane of A
constexpr int kOzMaxNB = 24;     // columns per accumulator: (8 levels + M) x 24, at most 256 TMEM columns
constexpr int kOzPlanes = kOzSlices + 1;  // of A: digits, magnitudes
constexpr int kOzRows = kOzSlices + 2;    // of B's image, times NB: digits, zeros, magnitudes
constexpr int kOzMaxSub = 6;     // 8-wide K chunks of one B pipeline stage, at most (48 K)
constexpr int kOzRing = 8;       // exponent rings: more than the windows and accumulators in flight
// Warps of the kernel: epilogue, converter, then producer, MMA issuer and two
// that fill the warpgroup.
constexpr int kOzConvWarps = 8;
constexpr int oz_epi_warps(bool multi) { return multi ? 8 : 16; }
constexpr int oz_threads(bool multi) { return 32 * (oz_epi_warps(multi) + kOzConvWarps + (multi ? 2 : 4)); }
constexpr size_t kOzSmemMax = 227 * 1024;
constexpr int kOzMaxCols = 256;  // 2 N, N <= 128
// column offsets, rings of row and column exponents and square sums, barriers
constexpr int kOzMisc = kOzMaxCols * 4 + kOzRing * 2 * (kOzBM + kOzMaxNB) * 4 + 256;

// Shape of one GEMM: column blocks of NB (a multiple of 8, at most 24) and K
// windows of kw (a multiple of 16): one of at most 96, or several of at most 64,
// which leave room for longer B stages (S4 at N = 24 and 48, windows of 96, 80 and
// 64: 2.42, 2.48, 2.26 and 6.43, 6.59, 6.00 ms).
constexpr int kOzLongKw = 64;
struct OzGeom {
    int Nc, NB, nblk, kw, nwin;
    long long K;
    long long win_bytes() const { return (long long)nblk * (kw / 8) * (kOzRows * NB * 16); }  // digits of a window
    long long img_bytes() const { return nwin * win_bytes(); }                               // of one z
    long long exps() const { return 2LL * nwin * nblk * NB; }  // column exponents and square sums
};

OzGeom oz_geom(int Nc, long long K) {
    OzGeom g;
    g.Nc = Nc;
    g.K = K;
    g.nblk = (Nc + kOzMaxNB - 1) / kOzMaxNB;
    g.NB = ((Nc + g.nblk - 1) / g.nblk + 7) / 8 * 8;
    const int most = K <= kOzMaxKw ? kOzMaxKw : kOzLongKw;
    g.nwin = (int)((K + most - 1) / most);
    g.kw = (int)(((K + g.nwin - 1) / g.nwin + 15) / 16 * 16);
    g.nwin = (int)((K + g.kw - 1) / g.kw);
    return g;
}

struct OzParams {
    const double* A;
    long long lda, sAz;
    int M;
    const double* B;     // for the results that are summed again
    long long ldb, sBz;
    const uint8_t* img;  // digit images of B: [z][window][block][chunk][9 NB rows][16 B]
    long long img_z;     // bytes per z (0: shared)
    const int* ecol;     // exponents and c x square sums of B's columns: [z][window][block][2][NB]
    long long ecol_z;
    double* out;
    long long sOz;
    StageMap map;
    int Nc, NB, nblk, nwin;
    long long K;
    int mtiles;          // ceil(M / 128)
    int nitem, wper;     // split K: items per row tile, windows per item
    long long sOitem;
    long long tiles;     // z x item x row tile
    // per plane of A: instruction descriptor, accumulator column, first row of B
    uint32_t mma_id[kOzPlanes], mma_col[kOzPlanes], mma_row[kOzPlanes];
    OzMul mul;
    int na, nbs, sub;    // A and B pipeline stages, chunks of a B stage
    int* err;
};

// c x the square sum of a row, infinite (nothing is accepted) for one at the
// exponent's floor, whose digits lose more than the criterion knows of.
__device__ __forceinline__ float oz_scaled_squares(float sq, uint32_t emax) {
    return emax <= kOzExpMin ? __int_as_float(0x7F800000) : kOzAccept * sq;
}

// ---------------------------------------------------------------------------
// Digit images of B.  One warp per (z, window, column): FP16 digits in the
// K-major core-matrix layout the MMA reads (8 rows x 16 bytes, no swizzle):
// row j NB + c holds digit j of column c of the block, rows 7 NB .. 8 NB - 1
// are zero (they clear the accumulator's last level), rows 8 NB .. 9 NB - 1 its
// magnitudes (oz_magnitude).  A window's K is
// permuted as the converter of A reads it: of the no chunks of the window,
// chunk p holds k = p + no q, q = 0..7 (K odd), or the pairs 2 (p + no q) + {0, 1},
// q = 0..3 (K even, 16-byte loads).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_oz_slice(const double* __restrict__ B, long long ldb, long long sBz,
                                                  int Nc, long long K, int NB, int nblk, int kw, int nwin,
                                                  long long nwarps, uint8_t* __restrict__ img,
                                                  long long img_z, int* __restrict__ ecol,
                                                  long long ecol_z) {
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gw >= nwarps) return;
    const int lane = threadIdx.x & 31;
    const int ncp = nblk * NB;
    const int col = (int)(gw % ncp);
    const long long zw = gw / ncp;
    const int w = (int)(zw % nwin);
    const long long z = zw / nwin;
    const long long k0 = (long long)w * kw;
    const int Kw = (int)(K - k0 < kw ? K - k0 : kw);
    const int no = 2 * ((Kw + 15) / 16);
    const double* b = B + z * sBz + (long long)col * ldb + k0;
    uint2 x[2][2];  // (lo, hi)
    uint32_t emax = kOzExpMin;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = (lane >> 2) + 8 * u, q = lane & 3;
            const int k = (K & 1) ? p + no * (2 * q + h) : 2 * (p + no * q) + h;
            x[u][h] = make_uint2(0u, 0u);
            if (col < Nc && p < no && k < Kw) x[u][h] = *reinterpret_cast<const uint2*>(b + k);
            emax = max(emax, x[u][h].y & kOzExpMask);
        }
    emax = __reduce_max_sync(0xffffffffu, emax);
    const int blk = col / NB, c = col % NB;
    uint8_t* o = img + z * img_z + ((long long)w * nblk + blk) * (kw / 8) * (kOzRows * NB * 16);
    float sq = 0.0f;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int p = (lane >> 2) + 8 * u;
        if (p >= no) continue;
        const uint64_t t0 = oz_digits(x[u][0].y, x[u][0].x, emax), t1 = oz_digits(x[u][1].y, x[u][1].x, emax);
        uint8_t* op = o + (long long)p * (kOzRows * NB * 16) + c * 16 + (lane & 3) * 4;
#pragma unroll
        for (int j = 0; j < kOzSlices; ++j) {
            const __half2 d = __halves2half2(__int2half_rn(oz_digit(t0, j)), __int2half_rn(oz_digit(t1, j)));
            *reinterpret_cast<__half2*>(op + j * NB * 16) = d;
            if (j > 0) continue;
            const uint32_t b = *reinterpret_cast<const uint32_t*>(&d);
            *reinterpret_cast<uint32_t*>(op + (kOzSlices + 1) * NB * 16) =
                oz_magnitude(b, oz_nonzero(x[u][0].y, x[u][0].x)) |
                oz_magnitude(b >> 16, oz_nonzero(x[u][1].y, x[u][1].x)) << 16;
            const float d0 = (float)oz_digit(t0, 0) * (1.0f / 64.0f), d1 = (float)oz_digit(t1, 0) * (1.0f / 64.0f);
            sq = fmaf(d0, d0, fmaf(d1, d1, sq));
        }
        *reinterpret_cast<uint32_t*>(op + kOzSlices * NB * 16) = 0u;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, d);
    if (lane == 0) {
        int* e = ecol + z * ecol_z + ((long long)w * nblk + blk) * (2 * NB) + c;
        e[0] = oz_exponent(emax);
        e[NB] = __float_as_int(oz_scaled_squares(sq, emax));
    }
}

// ---------------------------------------------------------------------------
// The GEMM kernel: one CTA per SM, persistent over 128-row tiles.
//
// Warps: the epilogue (two warps per tensor-memory lane quarter, half of a
// block's columns each; with one K window two such groups drain alternate
// accumulators), 8 converter warps (16 rows each), one producer of B's digit
// images and one MMA issuer.  Epilogue and converter are long chains of integer
// instructions that bound the kernel together; a second epilogue group overlaps
// more of them (N = 33: 78 -> 68 us a self-energy).
//
// A: the converter reads a window's rows (FP64, through L1), takes the row's
// largest exponent, and writes the seven digit planes and the magnitudes
// [chunk][128 rows][16 B] to shared memory (na stages).  The four lanes of a row read 64 contiguous
// bytes; chunks are kOzLbo apart, 32 bytes off a multiple of 128, so that eight
// lanes (two rows, four chunks) store to different banks.  B: bulk copies of pre-split images, one stage
// per 16 to 48 K of a 24-column block (nbs stages).  Digit i of A times the stacked
// digits 0 .. of B is one MMA of N = (digits) x NB columns at column offset
// i NB of the accumulator: level l = i + j lands in columns [l NB, (l+1) NB),
// so 34 digit products take seven MMAs per K step.  N is rounded up to 16, the 8
// columns past level 7 that this adds to are never read.  The first MMA covers all 8 NB columns
// (B's image has NB zero rows) and clears them.  An eighth MMA sums the magnitudes,
// in NB columns from oz_mag_col on.  Two accumulators (TMEM columns 0 and 256).
//
// A result that oz_accept turns down, or that leaves the normal range, is summed
// again by FMAs in the epilogue, from A and B in memory (oz_again: eight lanes a row;
// with every lane on its own row a warp pays for 32 rows whenever one is wanted, and
// the N = 48 propagation took 46 ms instead of 30).
//
// One window (K <= 96, stages S1-S3 up to N = 48): a row tile is converted
// once and multiplied with every column block.  Longer K: per block and
// window, the window results are added in FP64 registers.
// ---------------------------------------------------------------------------
// Bounded wait.  The tries sleep in between (polls without it were a seventh of
// the issued instructions, of a kernel bound by them); the timer is read once in
// 64 tries.
__device__ __forceinline__ bool oz_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err, int code,
                                        unsigned sleep_ns = 40) {
    if (mbar_try(bar, parity)) return true;
    unsigned long long t0 = 0;
    for (uint32_t it = 1;; ++it) {
        __nanosleep(sleep_ns);
        if (mbar_try(bar, parity)) return true;
        if ((it & 63u) == 0) {
            if (*abort_flag) return false;
            const unsigned long long now = gtimer();
            if (t0 == 0) t0 = now;
            if (now - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                atomicCAS(err, 0, code);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool oz_warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err,
                                             int code) {
    const bool r = oz_wait(bar, parity, abort_flag, err, code);
    return __all_sync(0xffffffffu, r);
}

// D[tmem] (+)= A[smem] B[smem], M = 128, K = 16, FP16 in, FP32 out; issued by
// one elected lane of a converged warp.  ad and bd are the low words of the
// operand descriptors, the only ones that differ.
__device__ __forceinline__ void oz_mma(uint32_t d, uint32_t ad, uint32_t bd, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%1, %5};\n\t"
        "mov.b64 b, {%2, %5};\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}" ::"r"(d),
        "r"(ad), "r"(bd), "r"(idesc), "r"(accumulate), "n"((128 >> 4) | (1 << 14))
        : "memory");
}
__device__ __forceinline__ void oz_commit(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr)
                 : "memory");
}
// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, lbo
// bytes apart along K, 128 bytes apart along the rows.  The low word of the
// descriptor (the high one is the row distance and the version).
__device__ __forceinline__ uint32_t desc_plain(uint32_t saddr, uint32_t lbo) {
    return ((saddr & 0x3FFFFu) >> 4) | (lbo >> 4) << 16;
}

// Accumulator column of the magnitudes' sums: past the levels and the columns that
// an MMA of an odd number of 8-column groups adds to.
__host__ __device__ constexpr int oz_mag_col(int NB) { return kOzLevels * NB + (NB & 8); }
static_assert(oz_mag_col(kOzMaxNB) + 32 <= 256, "accumulator columns");

// sum_k A[row][k] B[k] by FMAs for the rows (lanes) of a mask, four at a time: eight
// lanes share a row's K, so that its loads are coalesced and the few rows of a warp do
// not cost as much as all 32.  The result goes to the row's lane.
__device__ __forceinline__ void oz_again(uint32_t rows, int lane, const double* __restrict__ a, long long lda,
                                         const double* __restrict__ b, int Kw, uint64_t& r) {
    while (rows != 0u) {
        uint32_t pick[4], left = rows;
        int mine = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            pick[i] = left != 0u ? (uint32_t)__ffs((int)left) - 1u : 32u;
            left &= left - 1u;
            if ((lane >> 3) == i) mine = (int)min(pick[i], 31u);
        }
        if (((rows >> mine) & 1u) == 0u) mine = (int)pick[0];
        const double* ar = a + (long long)mine * lda;
        double d = 0.0;
#pragma unroll 4
        for (int k = lane & 7; k < Kw; k += 8) d = fma(__ldg(ar + k), __ldg(b + k), d);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double x = __shfl_sync(0xffffffffu, d, 8 * i);
            if (pick[i] == (uint32_t)lane) r = (uint64_t)__double_as_longlong(x);
        }
        rows = left;
    }
}

// Position of a tile in a CTA's range (row tiles fastest, then split-K items,
// then units), advanced without divisions.
struct OzPos {
    long long z;
    int item, mt, w0, nw;
    __device__ __forceinline__ OzPos(const OzParams& p, long long t) {
        mt = (int)(t % p.mtiles);
        const long long r = t / p.mtiles;
        item = (int)(r % p.nitem);
        z = r / p.nitem;
        windows(p);
    }
    __device__ __forceinline__ void windows(const OzParams& p) {
        w0 = item * p.wper;
        nw = min(p.wper, p.nwin - w0);
    }
    __device__ __forceinline__ void next(const OzParams& p) {
        if (++mt < p.mtiles) return;
        mt = 0;
        if (++item == p.nitem) {
            item = 0;
            ++z;
        }
        windows(p);
    }
};

// 8-wide K chunks of window w (an even number, NO but for a short last window).
template <int NO, bool MULTI>
__device__ __forceinline__ int oz_chunks(const OzParams& p, int w) {
    if (!MULTI) return NO;
    const long long left = p.K - (long long)w * (8 * NO);
    return left >= 8 * NO ? NO : 2 * (((int)left + 15) >> 4);
}

// Register split of the one-window kernel (28 warps, 72 registers a thread at
// launch): 16 x 64 + 8 x 104 + 4 x 40 = 28 x 72, each by the whole of a warpgroup.
// Other splits of the same kernel are slower (us per self-energy at N = 32 and
// 33; this one 37.9 and 70.1): 56 / 104 / 72 41.9 and 77.2, 8 epilogue warps 42.1
// and 78.5, 8 + 16 warps of 88 / 72 40.9 and 75.7.  The auxiliary warps live with
// 40 because the MMA role keeps its per-digit operands among the parameters, its
// descriptors in one word each and its stages as counters.
template <int N>
__device__ __forceinline__ void regs_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

template <int NO, bool MULTI, bool VEC>
__global__ void __launch_bounds__(oz_threads(MULTI), 1) k_oz_gemm(const __grid_constant__ OzParams p) {
    // used as declared, without integer casts: those would lose the address space
    // and turn every access into a generic one (four times the latency)
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int kEpi = oz_epi_warps(MULTI), kWorkers = kEpi + kOzConvWarps;
    constexpr int KW = 8 * NO;                                    // K of a window
    constexpr uint32_t kPlane = (uint32_t)(NO * kOzLbo);          // one digit plane of A
    constexpr uint32_t kAStage = kOzPlanes * kPlane;
    const uint32_t brow = (uint32_t)(kOzRows * p.NB * 16);        // one 8-wide K chunk of a block's image
    const uint32_t bstage = (uint32_t)p.sub * brow;
    uint8_t* sA = smem;
    uint8_t* sB = sA + (size_t)p.na * kAStage;
    uint32_t* sCol = (uint32_t*)(sB + (size_t)p.nbs * bstage);  // output offset of each column
    int* sExp = (int*)(sCol + kOzMaxCols);
    float* sSq = (float*)(sExp + kOzRing * kOzBM);        // c x square sums of the rows
    int* sEcol = (int*)(sSq + kOzRing * kOzBM);           // column exponents and square sums of an accumulator
    uint64_t* bars = (uint64_t*)(sEcol + kOzRing * 2 * kOzMaxNB);
    constexpr int AFULL = 0, AEMPTY = 2, BFULL = 4, BEMPTY = 8, ACCF = 12, ACCE = 14, DRAIN = 16, NBARS = 17;
    uint32_t* tmem_slot = (uint32_t*)(bars + NBARS);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    auto bar = [&](int i) { return smem_u32(bars + i); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar(AFULL + s), kOzConvWarps);
            mbar_init(bar(AEMPTY + s), 1);
            mbar_init(bar(ACCF + s), 1);
            mbar_init(bar(ACCE + s), 8);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(bar(BFULL + s), 1);
            mbar_init(bar(BEMPTY + s), 1);
        }
        mbar_init(bar(DRAIN), 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    for (int col = threadIdx.x; col < p.Nc; col += oz_threads(MULTI))
        sCol[col] = (uint32_t)((long long)(col / p.map.Dy) * p.map.SC + (long long)(col % p.map.Dy) * p.map.SY);
    if (warp == kWorkers + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const long long t0 = p.tiles * blockIdx.x / gridDim.x;
    const int ntile = (int)(p.tiles * (blockIdx.x + 1) / gridDim.x - t0);
    OzPos T(p, t0);

    if (warp < kEpi) {
        // ---------------- epilogue ----------------
        if (!MULTI) regs_dec<64>();
        const int q = warp & 3, h = (warp >> 2) & 1, grp = warp >> 3;
        const int half = p.NB / 2, cb = h * half;  // this warp's columns of a block (a multiple of 4)
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
        const OzMul mul = p.mul;
        uint32_t aseq = 0, accseq = 0;
        bool ok = true;
        // row = (ra Db + rb) Dx + rx of the output map; a tile further is 128 rows
        // = (ia, ib, ix) further, with carries (a division is 20 instructions)
        const int Dx = p.map.Dx, Db = p.map.Db;
        const int ix = kOzBM % Dx, ib = (kOzBM / Dx) % Db, ia = kOzBM / Dx / Db;
        int rx = 0, rb = 0, ra = 0;
        for (int t = 0; t < ntile && ok; ++t, T.next(p)) {
            const int row = T.mt * kOzBM + q * 32 + lane;
            const bool rok = row < p.M;
            if (t == 0 || T.mt == 0) {
                rx = row % Dx;
                rb = (row / Dx) % Db;
                ra = row / Dx / Db;
            } else {
                rx += ix;
                rb += ib;
                ra += ia;
                if (rx >= Dx) {
                    rx -= Dx;
                    ++rb;
                }
                if (rb >= Db) {
                    rb -= Db;
                    ++ra;
                }
            }
            double* o = p.out + T.z * p.sOz + T.item * p.sOitem + ra * p.map.SA + rb * p.map.SB + rx * p.map.SX;
            const int nouter = MULTI ? p.nblk * T.nw : 1, ninner = MULTI ? 1 : p.nblk;
            double sum[kOzMaxNB / 2];
            int blk = 0, wi = 0;
            for (int ao = 0; ao < nouter && ok; ++ao, ++aseq) {
                for (int bi = 0; bi < ninner; ++bi, ++accseq) {
                    const int ab = (int)(accseq & 1);
                    const int col0 = blk * p.NB + cb;
                    if (!MULTI) ++blk;
                    if (!MULTI && ab != grp) continue;
                    const int* ec = sEcol + (accseq % kOzRing) * 2 * kOzMaxNB + cb;
                    if (!oz_warp_wait(bar(ACCF + ab), (accseq >> 1) & 1, abort_flag, p.err, 41)) { ok = false; break; }
                    tc_fence_after();
                    const int Ea = sExp[(aseq % kOzRing) * kOzBM + q * 32 + lane] - 1014;
                    const float sqa = sSq[(aseq % kOzRing) * kOzBM + q * 32 + lane];
                    uint32_t tc[kOzLevels + 1];
#pragma unroll
                    for (int l = 0; l <= kOzLevels; ++l)
                        tc[l] = lane_base + (uint32_t)(ab * 256 + cb + (l < kOzLevels ? l * p.NB : oz_mag_col(p.NB)));
#pragma unroll(MULTI ? kOzMaxNB / 8 : 1)
                    for (int j = 0; j < (MULTI ? kOzMaxNB / 2 : half); j += 4) {  // four columns at a time
                        if (MULTI && j >= half) continue;
                        uint32_t v[kOzLevels + 1][4];
#pragma unroll
                        for (int l = 0; l <= kOzLevels; ++l) tmem_ld4(tc[l] + (uint32_t)j, v[l]);
                        const int4 e4 = *reinterpret_cast<const int4*>(ec + j);
                        const float4 s4 = *reinterpret_cast<const float4*>(ec + p.NB + j);
                        const int Es[4] = {Ea + e4.x, Ea + e4.y, Ea + e4.z, Ea + e4.w};
                        const float cs[4] = {sqa + s4.x, sqa + s4.y, sqa + s4.z, sqa + s4.w};
                        tmem_wait_ld();
                        // four independent chains; the rare cases in a second pass
                        uint32_t bad = 0u;
                        uint64_t r[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float a[kOzLevels];
#pragma unroll
                            for (int l = 0; l < kOzLevels; ++l) a[l] = __uint_as_float(v[l][k]);
                            uint32_t hi, lo, ha, e1;
                            oz_sum(a, mul, hi, lo);
                            r[k] = oz_pack(hi, lo, Es[k], mul, ha, e1);
                            if (!(oz_packed(ha, e1) && oz_accept(__uint_as_float(v[kOzLevels][k]), cs[k]))) bad |= 1u << k;
                        }
                        if (!rok) bad = 0u;
                        if (__any_sync(0xffffffffu, bad != 0u)) {
                            const long long k0 = MULTI ? (long long)(T.w0 + wi) * KW : 0;
                            const int Kw = MULTI ? (int)min((long long)KW, p.K - k0) : (int)p.K;
                            const double* ar = p.A + T.z * p.sAz + (long long)(T.mt * kOzBM + q * 32) * p.lda + k0;
                            const double* br = p.B + T.z * p.sBz + (long long)(col0 + j) * p.ldb + k0;
#pragma unroll
                            for (int k = 0; k < 4; ++k, br += p.ldb) {
                                bool again = ((bad >> k) & 1u) != 0u && col0 + j + k < p.Nc;
                                // M = 0: no two nonzero elements meet
                                if (again && v[kOzLevels][k] == 0u && Es[k] < kOzNonFinite / 2) {
                                    r[k] = 0ull;
                                    again = false;
                                }
                                oz_again(__ballot_sync(0xffffffffu, again), lane, ar, p.lda, br, Kw, r[k]);
                            }
                        }
                        if (MULTI) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const double d = __longlong_as_double((long long)r[k]);
                                sum[j + k] = wi == 0 ? d : sum[j + k] + d;
                            }
                        } else {
                            const uint4 off = *reinterpret_cast<const uint4*>(sCol + col0 + j);
                            const int ncol = rok ? p.Nc - (col0 + j) : 0;
                            if (ncol > 0) o[off.x] = __longlong_as_double((long long)r[0]);
                            if (ncol > 1) o[off.y] = __longlong_as_double((long long)r[1]);
                            if (ncol > 2) o[off.z] = __longlong_as_double((long long)r[2]);
                            if (ncol > 3) o[off.w] = __longlong_as_double((long long)r[3]);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(ACCE + ab));
                    if (MULTI && wi == T.nw - 1) {
#pragma unroll
                        for (int j = 0; j < kOzMaxNB / 2; ++j)
                            if (j < half && rok && col0 + j < p.Nc) o[sCol[col0 + j]] = sum[j];
                    }
                }
                if (MULTI && ++wi == T.nw) {
                    wi = 0;
                    ++blk;
                }
            }
        }
    } else if (warp < kWorkers) {
        // ---------------- converter: FP64 rows of A -> digit planes ----------------
        // A warp owns 16 rows as two groups of 8 (lane / 4).  Up to 6 chunks a
        // window, the 2 no (group, chunk) tasks of both groups are dealt over
        // the four lanes s of a row in one pass; longer windows take one pass per
        // row group (at most three tasks a lane either way).  The loads of the
        // next pass are in flight while the warp waits for its stage, and the
        // lines of the tile (or windows) after it are on their way to L2.
        constexpr bool kBoth = NO <= 6;
        constexpr int NT = kBoth ? NO / 2 : (NO + 3) / 4, NPASS = kBoth ? 1 : 2;
        if (!MULTI) regs_inc<104>();
        const int cw = warp - kEpi, r8 = lane >> 2, s = lane & 3;
        uint2 x[NT][8];  // (lo, hi), then digits
        int t = 0, blk = 0, wi = 0, pass = 0;
        uint32_t aseq = 0;
        OzPos P2 = T;  // the tile after the one being loaded
        P2.next(p);
        auto load = [&]() {
            const int w = T.w0 + wi;
            const long long k0 = (long long)w * KW;
            const int no = oz_chunks<NO, MULTI>(p, w);
            const int Kw = MULTI ? (int)min((long long)KW, p.K - k0) : (int)p.K;
            const int ntask = kBoth ? 2 * no : no;
            const int row0 = T.mt * kOzBM + 16 * cw, rmax = p.M - 1 - row0;  // rmax < 0: past the end
            const double* a = p.A + T.z * p.sAz + (long long)row0 * p.lda + k0;
            // rows, chunks and K past the end are clamped: their products meet
            // zero digits of B or are not stored
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                const int c = min(s + 4 * i, ntask - 1);
                const int rg = kBoth ? (c >= no ? 1 : 0) : pass;
                const int pc = kBoth ? c - rg * no : c;
                const double* ar = a + (long long)min(8 * rg + r8, rmax) * p.lda;
                if (VEC) {
                    const int kp = Kw >> 1;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int k = !MULTI && NO * q + NO - 1 <= 4 * NO - 8 ? pc + NO * q : min(pc + no * q, kp - 1);
                        const uint4 u = __ldg(reinterpret_cast<const uint4*>(ar) + k);
                        x[i][2 * q] = make_uint2(u.x, u.y);
                        x[i][2 * q + 1] = make_uint2(u.z, u.w);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int k = !MULTI && NO * q + NO - 1 <= 8 * NO - 16 ? pc + NO * q : min(pc + no * q, Kw - 1);
                        x[i][q] = __ldg(reinterpret_cast<const uint2*>(ar) + k);
                    }
                }
            }
            if (MULTI) {
                // this warp's rows of the window after the next
                if (pass == 0 && wi + 2 < T.nw) {
                    const int rr = T.mt * kOzBM + 16 * cw + (lane & 15);
                    const char* b = (const char*)(p.A + T.z * p.sAz + (long long)rr * p.lda + k0 + 2 * KW);
                    if (rr < p.M && k0 + 3 * KW <= p.K)
                        for (int o = (lane >> 4) * 128; o < KW * 8; o += 256)
                            asm volatile("prefetch.global.L2 [%0];" ::"l"(b + o));
                }
            } else if (pass == 0 && t + 1 < ntile && P2.mt * kOzBM + 16 * cw + 16 <= p.M) {
                // this warp's rows of the next tile (contiguous up to the row stride)
                const char* b = (const char*)(p.A + P2.z * p.sAz + (long long)(P2.mt * kOzBM + 16 * cw) * p.lda);
                const int bytes = 16 * (int)p.lda * 8;
                for (int o = lane * 128; o < bytes; o += 32 * 128)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(b + o));
            }
        };
        if (ntile > 0) load();
        while (t < ntile) {
            const int no = oz_chunks<NO, MULTI>(p, T.w0 + wi);
            const int ntask = kBoth ? 2 * no : no;
            // row exponents
            uint32_t E0 = kOzExpMin, E1 = kOzExpMin;
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                uint32_t e = kOzExpMin;
#pragma unroll
                for (int q = 0; q < 8; ++q) e = max(e, x[i][q].y & kOzExpMask);
                if (kBoth && s + 4 * i >= no) E1 = max(E1, e);
                else E0 = max(E0, e);
            }
#pragma unroll
            for (int d = 1; d < 4; d <<= 1) {
                E0 = max(E0, __shfl_xor_sync(0xffffffffu, E0, d));
                if (kBoth) E1 = max(E1, __shfl_xor_sync(0xffffffffu, E1, d));
            }
            if (s == 0) {
                int* se = sExp + (aseq % kOzRing) * kOzBM + 16 * cw + r8;
                se[kBoth ? 0 : 8 * pass] = oz_exponent(E0);
                if (kBoth) se[8] = oz_exponent(E1);
            }
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                const uint32_t E = kBoth && s + 4 * i >= no ? E1 : E0;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint64_t d = oz_digits(x[i][q].y, x[i][q].x, E);
                    // the unused last byte says whether the element is zero
                    x[i][q] = make_uint2(((uint32_t)d & 0xFFFFFF00u) | oz_nonzero(x[i][q].y, x[i][q].x), (uint32_t)(d >> 32));
                }
            }
            float S0 = 0.0f, S1 = 0.0f;  // square sums of the rows
            const int as = p.na == 2 ? (int)(aseq & 1) : 0;
            const uint32_t aph = (p.na == 2 ? aseq >> 1 : aseq) & 1;
            if (pass == 0 && !oz_warp_wait(bar(AEMPTY + as), aph ^ 1, abort_flag, p.err, 42)) break;
            uint8_t* ap = sA + (size_t)as * kAStage + 2 * cw * 128 + r8 * 16;
#pragma unroll
            for (int i = 0; i < NT; ++i) {
                const int c = s + 4 * i;
                if (c < ntask) {
                    const int rg = kBoth ? (c >= no ? 1 : 0) : pass;
                    const int pc = kBoth ? c - rg * no : c;
                    uint8_t* o = ap + pc * kOzLbo + rg * 128;
                    uint32_t d0[4];
                    // the same byte of two elements side by side, two digits at a
                    // time, then each digit as FP16 1024 + byte, minus 1152
#pragma unroll
                    for (int w2 = 0; w2 < 4; ++w2) {  // bytes (7,6) (5,4) (3,2) (1,-)
                        uint32_t v[2][4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t a0 = w2 < 2 ? x[i][2 * q].y : x[i][2 * q].x;
                            const uint32_t a1 = w2 < 2 ? x[i][2 * q + 1].y : x[i][2 * q + 1].x;
                            const uint32_t pr = __byte_perm(a0, a1, (w2 & 1) ? 0x4051 : 0x6273);
                            v[0][q] = __byte_perm(pr, 0x64646464u, 0x4140);
                            v[1][q] = __byte_perm(pr, 0x64646464u, 0x4342);
                        }
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            uint32_t d[4];
                            if (2 * w2 + k == kOzSlices) {  // magnitudes
#pragma unroll
                                for (int q = 0; q < 4; ++q) d[q] = (d0[q] & 0x7FFF7FFFu) | (v[k][q] & 0x00010001u);
                                *reinterpret_cast<uint4*>(o + kOzSlices * kPlane) = make_uint4(d[0], d[1], d[2], d[3]);
                                continue;
                            }
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const __half2 hd = __hsub2(*reinterpret_cast<const __half2*>(&v[k][q]),
                                                           __half2half2(__ushort_as_half(0x6480)));
                                d[q] = *reinterpret_cast<const uint32_t*>(&hd);
                                if (2 * w2 + k == 0) d0[q] = d[q];
                            }
                            *reinterpret_cast<uint4*>(o + (2 * w2 + k) * kPlane) = make_uint4(d[0], d[1], d[2], d[3]);
                        }
                    }
                    __half2 sq = __float2half2_rn(0.0f);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const __half2 h = *reinterpret_cast<const __half2*>(&d0[q]);
                        sq = __hfma2(__hmul2(h, __float2half2_rn(1.0f / 4096.0f)), h, sq);
                    }
                    const float f = __low2float(sq) + __high2float(sq);
                    if (kBoth && rg) S1 += f;
                    else S0 += f;
                }
            }
#pragma unroll
            for (int d = 1; d < 4; d <<= 1) {
                S0 += __shfl_xor_sync(0xffffffffu, S0, d);
                if (kBoth) S1 += __shfl_xor_sync(0xffffffffu, S1, d);
            }
            if (s == 0) {
                float* ss = sSq + (aseq % kOzRing) * kOzBM + 16 * cw + r8;
                ss[kBoth ? 0 : 8 * pass] = oz_scaled_squares(S0, E0);
                if (kBoth) ss[8] = oz_scaled_squares(S1, E1);
            }
            // next pass
            if (pass == NPASS - 1) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(AFULL + as));
                ++aseq;
                pass = 0;
                bool done = true;  // all windows and blocks of the tile
                if (MULTI) {
                    if (++wi == T.nw) {
                        wi = 0;
                        ++blk;
                    }
                    done = blk == p.nblk;
                }
                if (done) {
                    blk = 0;
                    ++t;
                    T.next(p);
                    P2.next(p);
                }
            } else {
                ++pass;
            }
            if (t < ntile) load();
        }
    } else {
        if (!MULTI) regs_dec<40>();
        if (warp == kWorkers) {
            if (lane == 0) {
                // ---------------- producer of B's digit images ----------------
                uint32_t bseq = 0, accseq = 0;
                bool ok = true;
                for (int t = 0; t < ntile && ok; ++t, T.next(p)) {
                    const int nacc = MULTI ? p.nblk * T.nw : p.nblk;
                    int blk = 0, wi = 0;
                    for (int a = 0; a < nacc && ok; ++a, ++accseq) {
                        const int w = T.w0 + wi;
                        const int no = oz_chunks<NO, MULTI>(p, w);
                        const uint8_t* src = p.img + T.z * p.img_z + ((long long)w * p.nblk + blk) * NO * brow;
                        for (int c0 = 0; c0 < no; c0 += p.sub, ++bseq) {
                            const int st = (int)(bseq % (uint32_t)p.nbs);
                            if (!oz_wait(bar(BEMPTY + st), ((bseq / (uint32_t)p.nbs) & 1) ^ 1, abort_flag, p.err, 43, 300)) {
                                ok = false;
                                break;
                            }
                            const uint32_t bytes = (uint32_t)min(p.sub, no - c0) * brow;
                            mbar_expect_tx(bar(BFULL + st), bytes + (c0 == 0 ? p.NB * 8u : 0u));
                            if (c0 == 0)
                                bulk_load(smem_u32(sEcol + (accseq % kOzRing) * 2 * kOzMaxNB),
                                          p.ecol + T.z * p.ecol_z + ((long long)w * p.nblk + blk) * (2 * p.NB), p.NB * 8u,
                                          bar(BFULL + st));
                            bulk_load(smem_u32(sB + (size_t)st * bstage), src + (size_t)c0 * brow, bytes, bar(BFULL + st));
                        }
                        if (!MULTI || ++wi == T.nw) {
                            wi = 0;
                            ++blk;
                        }
                    }
                }
                if (*abort_flag) {
                    // copies in flight must land before the CTA leaves
                    for (uint32_t st = 0; st < (uint32_t)p.nbs; ++st) {
                        if (bseq > st) {
                            const uint32_t last = bseq - 1 - ((bseq - 1 - st) % (uint32_t)p.nbs);
                            const unsigned long long g0 = gtimer();
                            while (!mbar_try(bar(BFULL + st), (last / (uint32_t)p.nbs) & 1) && gtimer() - g0 < kWaitLimitNs) {}
                        }
                    }
                }
            }
        } else if (warp == kWorkers + 1) {
            // ---------------- MMA issuer ----------------
            // stage counters with their phases: few registers, no divisions
            uint32_t as = 0, aph = 0, st = 0, bph = 0, accseq = 0;
            const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB);
            bool ok = true;
            for (int t = 0; t < ntile && ok; ++t, T.next(p)) {
                const int nouter = MULTI ? p.nblk * T.nw : 1, ninner = MULTI ? 1 : p.nblk;
                int wi = 0;
                for (int ao = 0; ao < nouter && ok; ++ao) {
                    const int no = oz_chunks<NO, MULTI>(p, T.w0 + wi);
                    if (MULTI && ++wi == T.nw) wi = 0;
                    if (!oz_warp_wait(bar(AFULL + as), aph, abort_flag, p.err, 44)) { ok = false; break; }
                    for (int bi = 0; bi < ninner && ok; ++bi, ++accseq) {
                        const int ab = (int)(accseq & 1);
                        if (!oz_warp_wait(bar(ACCE + ab), ((accseq >> 1) & 1) ^ 1, abort_flag, p.err, 45)) { ok = false; break; }
#pragma unroll 1
                        for (int c0 = 0; c0 < no; c0 += p.sub) {
                            if (!oz_warp_wait(bar(BFULL + st), bph, abort_flag, p.err, 46)) { ok = false; break; }
                            tc_fence_after();
                            const uint32_t ad = desc_plain(sA0 + as * kAStage + (uint32_t)c0 * kOzLbo, kOzLbo);
                            const uint32_t bd = desc_plain(sB0 + st * bstage, brow);
                            const uint32_t acc = tmem + (uint32_t)(ab * 256);
                            const int ns = min(p.sub, no - c0) / 2;
#pragma unroll
                            for (int i = 0; i < kOzPlanes; ++i) {
                                // digits of B this digit of A meets (digit 0's first step also
                                // meets the zero rows, clearing level 7), then the magnitudes
                                const int later = c0 | (i == kOzSlices ? 0 : i);
#pragma unroll 1
                                for (int ks = 0; ks < ns; ++ks)
                                    oz_mma(acc + p.mma_col[i], ad + (i * kPlane >> 4) + (uint32_t)ks * (2 * kOzLbo >> 4),
                                           bd + p.mma_row[i] + (uint32_t)ks * (brow >> 3), p.mma_id[i],
                                           (later | ks) ? 1u : 0u);
                            }
                            oz_commit(bar(BEMPTY + st));
                            if (++st == (uint32_t)p.nbs) {
                                st = 0;
                                bph ^= 1;
                            }
                        }
                        if (!ok) break;
                        oz_commit(bar(ACCF + ab));
                    }
                    if (!ok) break;
                    oz_commit(bar(AEMPTY + as));
                    if (++as == (uint32_t)p.na) {
                        as = 0;
                        aph ^= 1;
                    }
                }
            }
            // closing commit: no MMA reads this CTA's memory after it
            oz_commit(bar(DRAIN));
            const unsigned long long g0 = gtimer();
            while (!mbar_try(bar(DRAIN), 0) && gtimer() - g0 < kWaitLimitNs) {}
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWorkers + 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

using OzKernel = void (*)(const OzParams);
// The kernel of a window of kw K (16 .. 96).
template <bool MULTI, bool VEC>
OzKernel oz_kernel(int kw) {
    switch (kw / 16) {
        case 1: return k_oz_gemm<2, MULTI, VEC>;
        case 2: return k_oz_gemm<4, MULTI, VEC>;
        case 3: return k_oz_gemm<6, MULTI, VEC>;
        case 4: return k_oz_gemm<8, MULTI, VEC>;
        case 5: return k_oz_gemm<10, MULTI, VEC>;
        default: return k_oz_gemm<12, MULTI, VEC>;
    }
}
OzKernel oz_kernel(int kw, bool multi, bool vec) {
    if (multi) return vec ? oz_kernel<true, true>(kw) : oz_kernel<true, false>(kw);
    return vec ? oz_kernel<false, true>(kw) : oz_kernel<false, false>(kw);
}

// A stages (1 or 2), chunks of a B stage and B stages (2 to 4) that fit the shared
// memory: two A stages if two whole B stages fit next to them, then the longest B
// stage of which three fit (kw = 48, two A stages with B stages of 16 K or one with
// 48 K: 2.55, 2.19 ms for S2 at N = 24).
void oz_stages(const OzGeom& g, int* na, int* nbs, int* sub, size_t* smem) {
    const size_t a = (size_t)kOzPlanes * (g.kw / 8) * kOzLbo, row = (size_t)kOzRows * g.NB * 16;
    const size_t room = kOzSmemMax - kOzMisc - 128;
    int c = std::min(kOzMaxSub, g.kw / 8);
    *na = 2 * a + 2 * c * row <= room ? 2 : 1;
    while (c > 2 && *na * a + 3 * c * row > room) c -= 2;
    int n = 2;
    while (n < 4 && *na * a + (n + 1) * c * row <= room) ++n;
    *nbs = n;
    *sub = c;
    *smem = *na * a + n * c * row + kOzMisc + 128;
}

}  // namespace

size_t oz_img_bytes(int Nc, long long K) {
    const OzGeom g = oz_geom(Nc, K);
    return (size_t)g.img_bytes() + (size_t)g.exps() * 4;
}

gkba_status oz_prepare(gkba_ctx* c) {
    for (int kw = 16; kw <= kOzMaxKw; kw += 16)
        for (int m = 0; m < 4; ++m)
            GKBA_CUDA(c, cudaFuncSetAttribute(oz_kernel(kw, (m & 1) != 0, (m & 2) != 0),
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kOzSmemMax));
    return GKBA_OK;
}

gkba_status oz_slice(gkba_ctx* c, const double* B, long long ldb, long long sBz, int Nc, long long K, int nz,
                     void* img) {
    const OzGeom g = oz_geom(Nc, K);
    const long long nwarps = (long long)nz * g.nwin * g.nblk * g.NB;
    int* ecol = (int*)((char*)img + g.img_bytes() * nz);
    const long long blocks = (nwarps * 32 + 255) / 256;
    if (blocks > 0x7fffffffLL) return fail(c, GKBA_EINVAL, "digit images of %d units: too many columns", nz);
    auto t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_oz_slice<<<(unsigned)blocks, 256, 0, c->stream>>>(B, ldb, sBz, Nc, K, g.NB, g.nblk, g.kw, g.nwin, nwarps,
                                                        (uint8_t*)img, g.img_bytes(), ecol, g.exps());
    return launch_end(c, t);
}

// Eight windows an item, three below 64 windows (N < 16: S4 of few units at N = 13,
// eight and three 41 and 21 us), more where that were over 144 items (one an SM for
// a single unit's one row tile, N >= 42).  By K alone: a unit's result does not depend
// on the units it is computed with, nor on the memory that is free.  The partial sums
// add 5 % to the traffic of X3 at N = 24 and 6 % at N = 48; splitting only where row
// tiles were few took 2.27 instead of 1.77 ms for S4 at N = 24, 301 points.
constexpr int kOzMaxItems = 144;
int oz_items(long long K) {
    const int nwin = oz_geom(1, K).nwin, windows = nwin < 64 ? 3 : 8;
    const int want = std::min(kOzMaxItems, (nwin + windows - 1) / windows);
    const int per = (nwin + want - 1) / want;
    return (nwin + per - 1) / per;
}

gkba_status oz_gemm(gkba_ctx* c, int cls, const double* A, long long lda, long long sAz, const double* B,
                    long long ldb, long long sBz, const void* img, int img_nz, int Nc, long long K, double* out, long long sOz, int M, int nz, int nitem,
                    long long sOitem, StageMap map, double flops, double bytes) {
    const OzGeom g = oz_geom(Nc, K);
    if (Nc > kOzMaxCols) return fail(c, GKBA_EINVAL, "oz_gemm: %d columns", Nc);
    // 16-byte loads of A (the digit images have the matching order, by K's parity)
    const bool vec = (K & 1) == 0;
    if (vec && ((lda & 1) || (sAz & 1) || ((uintptr_t)A & 15)))
        return fail(c, GKBA_EINVAL, "oz_gemm: rows of even K must be 16-byte aligned");
    if ((unsigned long long)(Nc / map.Dy) * map.SC + (unsigned long long)map.Dy * map.SY >= 1ull << 32)
        return fail(c, GKBA_EINVAL, "oz_gemm: column offsets past 32 bits");
    OzParams p{};
    p.A = A;
    p.lda = lda;
    p.sAz = sAz;
    p.M = M;
    p.B = B;
    p.ldb = ldb;
    p.sBz = sBz;
    p.img = (const uint8_t*)img;
    p.img_z = img_nz > 1 ? g.img_bytes() : 0;
    p.ecol = (const int*)((const char*)img + g.img_bytes() * img_nz);
    p.ecol_z = img_nz > 1 ? g.exps() : 0;
    p.out = out;
    p.sOz = sOz;
    p.map = map;
    p.Nc = Nc;
    p.NB = g.NB;
    p.nblk = g.nblk;
    p.nwin = g.nwin;
    p.K = K;
    p.mtiles = (M + kOzBM - 1) / kOzBM;
    p.wper = (g.nwin + nitem - 1) / nitem;
    p.nitem = (g.nwin + p.wper - 1) / p.wper;
    if (p.nitem != nitem) return fail(c, GKBA_EINVAL, "oz_gemm: %d items for %d windows", nitem, g.nwin);
    p.sOitem = sOitem;
    p.mul = kOzMul;
    for (int i = 0; i < kOzPlanes; ++i) {
        const bool mag = i == kOzSlices;
        const int cnt = mag ? 1 : i == 0 ? 8 : std::min(kOzSlices, kOzLevels - i);
        const uint32_t n = (uint32_t)((cnt * p.NB + 15) & ~15);
        p.mma_id[i] = (1u << 4) | ((n >> 3) << 17) | ((uint32_t)(kOzBM >> 4) << 24);
        p.mma_col[i] = (uint32_t)(mag ? oz_mag_col(p.NB) : i * p.NB);
        p.mma_row[i] = mag ? (uint32_t)((kOzSlices + 1) * p.NB) : 0u;  // x 16 bytes, as the descriptor counts
    }
    p.tiles = (long long)nz * p.nitem * p.mtiles;
    if (p.tiles >= 1LL << 31) return fail(c, GKBA_EINVAL, "oz_gemm: %lld tiles", p.tiles);
    p.err = c->dint + 1;
    size_t smem = 0;
    oz_stages(g, &p.na, &p.nbs, &p.sub, &smem);
    const unsigned grid = (unsigned)std::min<long long>(p.tiles, c->num_sms);
    auto t = launch_begin(c, cls, flops, bytes);
    oz_kernel(g.kw, g.nwin > 1, vec)<<<grid, oz_threads(g.nwin > 1), smem, c->stream>>>(p);
    return launch_end(c, t);
}

}  // namespace gkba
