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
// together with integer instructions only.  The result is closer to the exact
// sum than the FMA chain's (tests/test_oz_digits.py; whole Heun steps and
// self-energies: 1.1-2.0e-15 from 64-bit references where the FMA chain had
// 1.8-3.3e-15).  Whole calls, FMA chain -> here: Heun step at N = 24, 301 points
// 309 -> 36 ms; 40 self-energies at N = 33 78 -> 5.8 ms; Heun step at N = 10, 501
// points 23.8 -> 3.6 ms; three time-linear steps at N = 48 137 -> 20 ms.
#include <cuda_fp16.h>

#include <algorithm>

#include "gkba_internal.cuh"
#include "oz_digits.h"
#include "ptx_sm103.cuh"

namespace gkba {

namespace {

constexpr int kOzBM = 128;       // rows per tile (tensor-memory lanes)
constexpr int kOzMaxNB = 32;     // columns per accumulator: 8 levels x 32 = 256 TMEM columns
constexpr int kOzSub = 6;        // 8-wide K chunks of one B pipeline stage (48 K)
constexpr int kOzRing = 8;       // row-exponent ring (windows in flight)
constexpr int kOzEpiWarps = 8, kOzConvWarps = 8;
constexpr int kOzThreads = 32 * (kOzEpiWarps + kOzConvWarps + 2);
constexpr size_t kOzSmemMax = 227 * 1024;
constexpr int kOzMisc = kOzRing * kOzBM * 4 + 256;  // row exponents, barriers

// Shape of one GEMM: column blocks of NB (a multiple of 8, at most 32) and K
// windows of kw (a multiple of 16, at most 96).
struct OzGeom {
    int Nc, NB, nblk, kw, nwin;
    long long K;
    long long win_bytes() const { return (long long)nblk * (kw / 8) * (8 * NB * 16); }  // digits of a window
    long long img_bytes() const { return nwin * win_bytes(); }                        // of one z
    long long exps() const { return (long long)nwin * nblk * NB; }                    // column exponents
};

OzGeom oz_geom(int Nc, long long K) {
    OzGeom g;
    g.Nc = Nc;
    g.K = K;
    g.nblk = (Nc + kOzMaxNB - 1) / kOzMaxNB;
    g.NB = ((Nc + g.nblk - 1) / g.nblk + 7) / 8 * 8;
    g.nwin = (int)((K + kOzMaxKw - 1) / kOzMaxKw);
    g.kw = (int)(((K + g.nwin - 1) / g.nwin + 15) / 16 * 16);
    g.nwin = (int)((K + g.kw - 1) / g.kw);
    return g;
}

struct OzParams {
    const double* A;
    long long lda, sAz;
    int M;
    const uint8_t* img;  // digit images of B: [z][window][block][chunk][8 NB rows][16 B]
    long long img_z;     // bytes per z (0: shared)
    const int* ecol;     // exponents of B's columns: [z][window][block NB]
    long long ecol_z;
    double* out;
    long long sOz;
    StageMap map;
    int Nc, NB, nblk, kw, nwin;
    long long K;
    int mtiles;          // ceil(M / 128)
    int nitem, wper;     // split K: items per row tile, windows per item
    long long sOitem;
    long long tiles;     // z x item x row tile
    int na, nbs;         // A and B pipeline stages
    int* err;
};

// ---------------------------------------------------------------------------
// Digit images of B.  One warp per (z, window, column): FP16 digits in the
// K-major core-matrix layout the MMA reads (8 rows x 16 bytes, no swizzle):
// row j NB + c holds digit j of column c of the block, rows 7 NB .. 8 NB - 1
// are zero (they clear the accumulator's last level).  A window's K is
// permuted, chunk p holding k = p + no q (q = 0..7, no the window's chunks), as
// the converter of A does.
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
    uint64_t x[2][2];
    int E = 1;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = (lane >> 2) + 8 * u, k = p + no * (2 * (lane & 3) + h);
            x[u][h] = (col < Nc && p < no && k < Kw) ? (uint64_t)__double_as_longlong(b[k]) : 0ull;
            E = max(E, oz_exponent((uint32_t)(x[u][h] >> 32)));
        }
    E = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
    if (lane == 0) ecol[z * ecol_z + (long long)w * ncp + col] = E;
    const int blk = col / NB, c = col % NB;
    uint8_t* o = img + z * img_z + ((long long)w * nblk + blk) * (kw / 8) * (8 * NB * 16);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int p = (lane >> 2) + 8 * u;
        if (p >= no) continue;
        const uint64_t t0 = oz_digits(x[u][0], E), t1 = oz_digits(x[u][1], E);
        uint8_t* op = o + (long long)p * (8 * NB * 16) + c * 16 + (lane & 3) * 4;
#pragma unroll
        for (int j = 0; j < kOzSlices; ++j) {
            const __half2 d = __halves2half2(__int2half_rn(oz_digit(t0, j)), __int2half_rn(oz_digit(t1, j)));
            *reinterpret_cast<__half2*>(op + j * NB * 16) = d;
        }
        *reinterpret_cast<uint32_t*>(op + kOzSlices * NB * 16) = 0u;
    }
}

// ---------------------------------------------------------------------------
// The GEMM kernel: one CTA per SM, persistent over 128-row tiles.
//
// Warps 0-7 epilogue (two per tensor-memory lane quarter, half of a block's
// columns each), 8-15 converter (16 rows each), 16 TMA producer of B's digit
// images, 17 MMA issuer.
//
// A: the converter reads a window's rows (FP64, through L1), takes the row's
// largest exponent, and writes the seven digit planes [chunk][128 rows][16 B]
// to shared memory (na stages).  B: bulk copies of pre-split images, one stage
// per 48 K of a 32-column block (nbs stages).  Digit i of A times the stacked
// digits 0 .. of B is one MMA of N = (digits) x NB columns at column offset
// i NB of the accumulator: level l = i + j lands in columns [l NB, (l+1) NB),
// so 34 digit products take seven MMAs per K step, none narrower than 32.
// N is rounded up to 16, the columns past level 7 are never read.  The first
// MMA covers all 8 NB columns (B's image ends in NB zero rows) and clears the
// accumulator.  Two accumulators (TMEM columns 0 and 256).
//
// One window (K <= 96, stages S1-S3 up to N = 48): a row tile is converted
// once and multiplied with every column block.  Longer K: per block and
// window, the window results are added in FP64 registers.
// ---------------------------------------------------------------------------
__device__ bool oz_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err, int code) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 63u) == 0) {
            if (*abort_flag) return false;
            if (gtimer() - t0 > kWaitLimitNs) {
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
// one elected lane of a converged warp.
__device__ __forceinline__ void oz_mma(uint32_t d, unsigned long long ad, unsigned long long bd, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
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
// bytes apart along K, 128 bytes apart along the rows.
__device__ __forceinline__ unsigned long long desc_plain(uint32_t saddr, uint32_t lbo) {
    return (unsigned long long)((saddr & 0x3FFFFu) >> 4) | (unsigned long long)(lbo >> 4) << 16 |
           (unsigned long long)(128 >> 4) << 32 | 1ull << 46;
}

// The position of a tile: unit z, split-K item and row tile.
struct OzTile {
    long long z;
    int item, mt, w0, nw;
    __device__ OzTile(const OzParams& p, long long t) {
        mt = (int)(t % p.mtiles);
        const long long r = t / p.mtiles;
        item = (int)(r % p.nitem);
        z = r / p.nitem;
        w0 = item * p.wper;
        nw = min(p.wper, p.nwin - w0);
    }
};

template <bool MULTI>
__global__ void __launch_bounds__(kOzThreads, 1) k_oz_gemm(const __grid_constant__ OzParams p) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    const uint32_t plane = (uint32_t)(kOzBM * p.kw * 2);          // one digit plane of A
    const uint32_t brow = (uint32_t)(8 * p.NB * 16);              // one 8-wide K chunk of a block's image
    const int no_full = p.kw / 8;
    const uint32_t bstage = (uint32_t)min(kOzSub, no_full) * brow;
    uint8_t* sA = smem;
    uint8_t* sB = sA + (size_t)p.na * kOzSlices * plane;
    int* sExp = (int*)(sB + (size_t)p.nbs * bstage);
    uint64_t* bars = (uint64_t*)(sExp + kOzRing * kOzBM);
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
            mbar_init(bar(ACCE + s), kOzEpiWarps);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(bar(BFULL + s), 1);
            mbar_init(bar(BEMPTY + s), 1);
        }
        mbar_init(bar(DRAIN), 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 17) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const long long t0 = p.tiles * blockIdx.x / gridDim.x, t1 = p.tiles * (blockIdx.x + 1) / gridDim.x;

    if (warp < kOzEpiWarps) {
        // ---------------- epilogue ----------------
        const int q = warp & 3, h = warp >> 2;
        const int half = p.NB / 2, cb = h * half;  // this warp's columns of a block (a multiple of 4)
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
        uint32_t aseq = 0, accseq = 0;
        bool ok = true;
        for (long long t = t0; t < t1 && ok; ++t) {
            const OzTile T(p, t);
            const uint32_t row = (uint32_t)T.mt * kOzBM + q * 32 + lane;
            const bool rok = row < (uint32_t)p.M;
            const uint32_t x = row % (uint32_t)p.map.Dx, rb = row / (uint32_t)p.map.Dx;
            double* o = p.out + T.z * p.sOz + T.item * p.sOitem + (long long)(rb / (uint32_t)p.map.Db) * p.map.SA +
                        (long long)(rb % (uint32_t)p.map.Db) * p.map.SB + (long long)x * p.map.SX;
            const int nouter = MULTI ? p.nblk * T.nw : 1, ninner = MULTI ? 1 : p.nblk;
            double sum[kOzMaxNB / 2];
            for (int ao = 0; ao < nouter && ok; ++ao, ++aseq) {
                const int wi = MULTI ? ao % T.nw : 0;
                for (int bi = 0; bi < ninner; ++bi, ++accseq) {
                    const int blk = MULTI ? ao / T.nw : bi;
                    const int ab = (int)(accseq & 1);
                    const int* ec = p.ecol + T.z * p.ecol_z + (long long)(T.w0 + wi) * p.nblk * p.NB + blk * p.NB + cb;
                    if (!oz_warp_wait(bar(ACCF + ab), (accseq >> 1) & 1, abort_flag, p.err, 41)) { ok = false; break; }
                    tc_fence_after();
                    const int Ea = sExp[(aseq % kOzRing) * kOzBM + q * 32 + lane];
                    const uint32_t col0 = lane_base + (uint32_t)(ab * 256 + cb);
#pragma unroll
                    for (int c4 = 0; c4 < kOzMaxNB / 8; ++c4) {
                        if (4 * c4 < half) {
                            uint32_t v[kOzLevels][4];
#pragma unroll
                            for (int l = 0; l < kOzLevels; ++l) tmem_ld4(col0 + (uint32_t)(l * p.NB + 4 * c4), v[l]);
                            const int4 e4 = *reinterpret_cast<const int4*>(ec + 4 * c4);
                            const int Eb[4] = {e4.x, e4.y, e4.z, e4.w};
                            tmem_wait_ld();
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                int a[kOzLevels];
#pragma unroll
                                for (int l = 0; l < kOzLevels; ++l) a[l] = __float2int_rn(__uint_as_float(v[l][j]));
                                const double r = __longlong_as_double((long long)oz_combine(a, Ea, Eb[j]));
                                if (MULTI) {
                                    sum[4 * c4 + j] = wi == 0 ? r : sum[4 * c4 + j] + r;
                                } else {
                                    const int col = blk * p.NB + cb + 4 * c4 + j;
                                    const int cc = col >= p.map.Dy ? 1 : 0;
                                    if (rok && col < p.Nc)
                                        o[cc * p.map.SC + (long long)(col - cc * p.map.Dy) * p.map.SY] = r;
                                }
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(ACCE + ab));
                    if (MULTI && wi == T.nw - 1) {
#pragma unroll
                        for (int j = 0; j < kOzMaxNB / 2; ++j) {
                            const int col = blk * p.NB + cb + j;
                            const int cc = col >= p.map.Dy ? 1 : 0;
                            if (j < half && rok && col < p.Nc)
                                o[cc * p.map.SC + (long long)(col - cc * p.map.Dy) * p.map.SY] = sum[j];
                        }
                    }
                }
            }
        }
    } else if (warp < kOzEpiWarps + kOzConvWarps) {
        // ---------------- converter: FP64 rows of A -> digit planes ----------------
        // A warp owns 16 rows as two groups of 8 (lane & 7).  The 2 no (group,
        // chunk) tasks of a pass are dealt over the four lane groups s; windows
        // of more than 8 chunks take one pass per row group.  The loads of the
        // next pass are in flight while the warp waits for its stage.
        const int cw = warp - kOzEpiWarps, r8 = lane & 7, s = lane >> 3;
        uint64_t x[4][8];
        // pass position
        long long t = t0;
        int ao = 0, pass = 0;
        uint32_t aseq = 0;
        auto load = [&]() {
            const OzTile T(p, t);
            const int w = T.w0 + (MULTI ? ao % T.nw : 0);
            const long long k0 = (long long)w * p.kw;
            const int Kw = (int)(p.K - k0 < p.kw ? p.K - k0 : p.kw);
            const int no = 2 * ((Kw + 15) >> 4);
            const int ntask = no <= 8 ? 2 * no : no;
            const int row0 = T.mt * kOzBM + 16 * cw + r8;
            const double* a = p.A + T.z * p.sAz + (long long)row0 * p.lda + k0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = s + 4 * i;
                const int rg = no <= 8 ? (c >= no ? 1 : 0) : pass;
                const int pc = no <= 8 ? c - rg * no : c;
                const bool ok = c < ntask && row0 + 8 * rg < p.M;
                const double* ar = a + (long long)(8 * rg) * p.lda;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int k = pc + no * q;
                    x[i][q] = ok && k < Kw ? (uint64_t)__double_as_longlong(__ldg(ar + k)) : 0ull;
                }
            }
        };
        bool ok = true;
        if (t < t1) load();
        while (t < t1 && ok) {
            const OzTile T(p, t);
            const int w = T.w0 + (MULTI ? ao % T.nw : 0);
            const long long k0 = (long long)w * p.kw;
            const int Kw = (int)(p.K - k0 < p.kw ? p.K - k0 : p.kw);
            const int no = 2 * ((Kw + 15) >> 4);
            const bool two = no <= 8;  // both row groups in one pass
            const int ntask = two ? 2 * no : no;
            const int npass = two ? 1 : 2;
            // row exponents
            int E0 = 1, E1 = 1;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                int e = 1;
#pragma unroll
                for (int q = 0; q < 8; ++q) e = max(e, oz_exponent((uint32_t)(x[i][q] >> 32)));
                const bool g1 = two ? s + 4 * i >= no : pass != 0;
                if (g1) E1 = max(E1, e);
                else E0 = max(E0, e);
            }
#pragma unroll
            for (int d = 8; d < 32; d <<= 1) {
                E0 = max(E0, __shfl_xor_sync(0xffffffffu, E0, d));
                E1 = max(E1, __shfl_xor_sync(0xffffffffu, E1, d));
            }
            int* se = sExp + (aseq % kOzRing) * kOzBM + 16 * cw + r8;
            if (s == 0) {
                if (two || pass == 0) se[0] = E0;
                if (two || pass == 1) se[8] = E1;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool g1 = two ? s + 4 * i >= no : pass != 0;
                const int E = g1 ? E1 : E0;
#pragma unroll
                for (int q = 0; q < 8; ++q) x[i][q] = oz_digits(x[i][q], E);
            }
            const int as = (int)(aseq % (uint32_t)p.na);
            if (pass == 0 &&
                !oz_warp_wait(bar(AEMPTY + as), ((aseq / (uint32_t)p.na) & 1) ^ 1, abort_flag, p.err, 42)) {
                ok = false;
                break;
            }
            uint8_t* ap = sA + (size_t)as * kOzSlices * plane;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = s + 4 * i;
                if (c < ntask) {
                    const int rg = two ? (c >= no ? 1 : 0) : pass;
                    const int pc = two ? c - rg * no : c;
                    uint8_t* o = ap + pc * (kOzBM * 16) + (2 * cw + rg) * 128 + r8 * 16;
#pragma unroll
                    for (int d = 0; d < kOzSlices; ++d) {
                        // byte 7 - d of each element -> 1024 + byte as FP16, minus 1152
                        const int byte = 7 - d;
                        const uint32_t sel = (uint32_t)((byte & 3) | ((4 + (byte & 3)) << 8));
                        uint32_t v[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t a0 = byte >= 4 ? (uint32_t)(x[i][2 * q] >> 32) : (uint32_t)x[i][2 * q];
                            const uint32_t a1 =
                                byte >= 4 ? (uint32_t)(x[i][2 * q + 1] >> 32) : (uint32_t)x[i][2 * q + 1];
                            const uint32_t b = (__byte_perm(a0, a1, sel) & 0x00FF00FFu) | 0x64006400u;
                            const __half2 hd = __hsub2(*reinterpret_cast<const __half2*>(&b),
                                                       __half2half2(__ushort_as_half(0x6480)));
                            v[q] = *reinterpret_cast<const uint32_t*>(&hd);
                        }
                        *reinterpret_cast<uint4*>(o + (size_t)d * plane) = make_uint4(v[0], v[1], v[2], v[3]);
                    }
                }
            }
            // next pass
            if (pass == npass - 1) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(AFULL + as));
                ++aseq;
                pass = 0;
                if (++ao == (MULTI ? p.nblk * T.nw : 1)) {
                    ao = 0;
                    ++t;
                }
            } else {
                ++pass;
            }
            if (t < t1) load();
        }
    } else if (warp == 16) {
        if (lane == 0) {
            // ---------------- producer of B's digit images ----------------
            uint32_t bseq = 0;
            bool ok = true;
            for (long long t = t0; t < t1 && ok; ++t) {
                const OzTile T(p, t);
                const int nacc = MULTI ? p.nblk * T.nw : p.nblk;
                for (int a = 0; a < nacc && ok; ++a) {
                    const int blk = MULTI ? a / T.nw : a, w = T.w0 + (MULTI ? a % T.nw : 0);
                    const long long k0 = (long long)w * p.kw;
                    const int no = 2 * (int)(((p.K - k0 < p.kw ? p.K - k0 : p.kw) + 15) >> 4);
                    const uint8_t* src = p.img + T.z * p.img_z + ((long long)w * p.nblk + blk) * no_full * brow;
                    for (int c0 = 0; c0 < no; c0 += kOzSub, ++bseq) {
                        const int st = (int)(bseq % (uint32_t)p.nbs);
                        if (!oz_wait(bar(BEMPTY + st), ((bseq / (uint32_t)p.nbs) & 1) ^ 1, abort_flag, p.err, 43)) {
                            ok = false;
                            break;
                        }
                        const uint32_t bytes = (uint32_t)min(kOzSub, no - c0) * brow;
                        mbar_expect_tx(bar(BFULL + st), bytes);
                        bulk_load(smem_u32(sB + (size_t)st * bstage), src + (size_t)c0 * brow, bytes, bar(BFULL + st));
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
    } else {
        // ---------------- MMA issuer ----------------
        uint32_t aseq = 0, bseq = 0, accseq = 0;
        const uint32_t lboB = brow;
        bool ok = true;
        for (long long t = t0; t < t1 && ok; ++t) {
            const OzTile T(p, t);
            const int nouter = MULTI ? p.nblk * T.nw : 1, ninner = MULTI ? 1 : p.nblk;
            for (int ao = 0; ao < nouter && ok; ++ao, ++aseq) {
                const int w = T.w0 + (MULTI ? ao % T.nw : 0);
                const long long k0 = (long long)w * p.kw;
                const int no = 2 * (int)(((p.K - k0 < p.kw ? p.K - k0 : p.kw) + 15) >> 4);
                const int as = (int)(aseq % (uint32_t)p.na);
                if (!oz_warp_wait(bar(AFULL + as), (aseq / (uint32_t)p.na) & 1, abort_flag, p.err, 44)) { ok = false; break; }
                const unsigned long long ad = desc_plain(smem_u32(sA + (size_t)as * kOzSlices * plane), kOzBM * 16);
                for (int bi = 0; bi < ninner && ok; ++bi, ++accseq) {
                    const int ab = (int)(accseq & 1);
                    if (!oz_warp_wait(bar(ACCE + ab), ((accseq >> 1) & 1) ^ 1, abort_flag, p.err, 45)) { ok = false; break; }
                    const uint32_t acc = tmem + (uint32_t)(ab * 256);
                    for (int c0 = 0; c0 < no; c0 += kOzSub, ++bseq) {
                        const int st = (int)(bseq % (uint32_t)p.nbs);
                        if (!oz_warp_wait(bar(BFULL + st), (bseq / (uint32_t)p.nbs) & 1, abort_flag, p.err, 46)) { ok = false; break; }
                        tc_fence_after();
                        const unsigned long long bd = desc_plain(smem_u32(sB + (size_t)st * bstage), lboB);
                        const int ns = min(kOzSub, no - c0) / 2;
#pragma unroll
                        for (int i = 0; i < kOzSlices; ++i) {
                            // digits of B this digit of A meets (digit 0's first step also
                            // meets the zero rows, clearing level 7)
                            const int cnt = i == 0 ? 8 : min(kOzSlices, kOzLevels - i);
                            const uint32_t n = (uint32_t)((cnt * p.NB + 15) & ~15);
                            const uint32_t id = (1u << 4) | ((n >> 3) << 17) | ((uint32_t)(kOzBM >> 4) << 24);
                            for (int ks = 0; ks < ns; ++ks)
                                oz_mma(acc + (uint32_t)(i * p.NB),
                                       ad + (((unsigned long long)i * plane + (unsigned long long)(c0 + 2 * ks) * (kOzBM * 16)) >> 4),
                                       bd + (((unsigned long long)(2 * ks) * brow) >> 4), id, (c0 | i | ks) ? 1u : 0u);
                        }
                        oz_commit(bar(BEMPTY + st));
                    }
                    if (!ok) break;
                    oz_commit(bar(ACCF + ab));
                }
                if (!ok) break;
                oz_commit(bar(AEMPTY + as));
            }
        }
        // closing commit: no MMA reads this CTA's memory after it
        oz_commit(bar(DRAIN));
        const unsigned long long g0 = gtimer();
        while (!mbar_try(bar(DRAIN), 0) && gtimer() - g0 < kWaitLimitNs) {}
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 17) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// A stages (1 or 2) and B stages (2 to 4) that fit the shared memory.
void oz_stages(const OzGeom& g, int* na, int* nbs, size_t* smem) {
    const size_t a = (size_t)kOzSlices * kOzBM * g.kw * 2;
    const size_t b = (size_t)std::min(kOzSub, g.kw / 8) * 8 * g.NB * 16;
    *na = 2 * a + 2 * b + kOzMisc + 128 <= kOzSmemMax ? 2 : 1;
    int n = 2;
    while (n < 4 && *na * a + (n + 1) * b + kOzMisc + 128 <= kOzSmemMax) ++n;
    *nbs = n;
    *smem = *na * a + n * b + kOzMisc + 128;
}

}  // namespace

size_t oz_img_bytes(int Nc, long long K) {
    const OzGeom g = oz_geom(Nc, K);
    return (size_t)g.img_bytes() + (size_t)g.exps() * 4;
}

gkba_status oz_prepare(gkba_ctx* c) {
    GKBA_CUDA(c, cudaFuncSetAttribute(k_oz_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmemMax));
    GKBA_CUDA(c, cudaFuncSetAttribute(k_oz_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmemMax));
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

int oz_items(gkba_ctx* c, int M, int Nc, long long K, long long max_items) {
    const OzGeom g = oz_geom(Nc, K);
    const long long mt = (M + kOzBM - 1) / kOzBM;
    // about two items per SM: K is split only while there are fewer row tiles
    const long long want = std::max(1LL, std::min({2LL * c->num_sms / mt, max_items, (long long)g.nwin}));
    const long long per = (g.nwin + want - 1) / want;
    return (int)((g.nwin + per - 1) / per);
}

gkba_status oz_gemm(gkba_ctx* c, int cls, const double* A, long long lda, long long sAz, const void* img,
                    int img_nz, int Nc, long long K, double* out, long long sOz, int M, int nz, int nitem,
                    long long sOitem, StageMap map, double flops, double bytes) {
    const OzGeom g = oz_geom(Nc, K);
    OzParams p{};
    p.A = A;
    p.lda = lda;
    p.sAz = sAz;
    p.M = M;
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
    p.kw = g.kw;
    p.nwin = g.nwin;
    p.K = K;
    p.mtiles = (M + kOzBM - 1) / kOzBM;
    p.wper = (g.nwin + nitem - 1) / nitem;
    p.nitem = (g.nwin + p.wper - 1) / p.wper;
    if (p.nitem != nitem) return fail(c, GKBA_EINVAL, "oz_gemm: %d items for %d windows", nitem, g.nwin);
    p.sOitem = sOitem;
    p.tiles = (long long)nz * p.nitem * p.mtiles;
    p.err = c->dint + 1;
    size_t smem = 0;
    oz_stages(g, &p.na, &p.nbs, &smem);
    const unsigned grid = (unsigned)std::min<long long>(p.tiles, c->num_sms);
    auto t = launch_begin(c, cls, flops, bytes);
    if (g.nwin == 1) k_oz_gemm<false><<<grid, kOzThreads, smem, c->stream>>>(p);
    else k_oz_gemm<true><<<grid, kOzThreads, smem, c->stream>>>(p);
    return launch_end(c, t);
}

}  // namespace gkba
