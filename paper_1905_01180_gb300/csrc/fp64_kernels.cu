// fp64_kernels.cu - FP64 kernels of the GKBA second-Born path:
//  * the chained-contraction stage GEMM for the FP64 path (Eq. 2bse evaluated
//    as four one-index contractions, see gkba_api.cu for the stage list),
//  * GKBA reconstruction P_k = T(t,t_k) rho_k, Q_k = T(t,t_k) - P_k (Eq. gkba),
//  * split-K reduction and the weighted history sum of Eq. (collint),
//  * the time-local pieces of Eq. (equalt): Sigma_HF, h_HF, commutator,
//    U_n = exp(-i dt h) by scaling and squaring with a Taylor polynomial,
//    the propagator recursion T(t_{n+1},t_k) = U_n T(t_n,t_k), Heun updates.
#include <algorithm>
#include <type_traits>
#include <cmath>
#include <cstdarg>
#include <mutex>

#include "gkba_internal.cuh"

namespace gkba {

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
// acc += a b in four FMAs (a multiply followed by an add takes six FP64
// instructions, and the FP64 rate, two a clock and SM, bounds these kernels).
__device__ __forceinline__ void cmac(double2& acc, double2 a, double2 b) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.y, b.x, acc.y);
}
// a b in a fixed form, rounded by itself.  The N x N products of split-TF32 contexts
// add such terms in the order of k (dot_seq): their results become FP32 operands,
// and one that falls on the other side of an FP32 rounding boundary moves a
// collision integral by up to 1e-8.
__device__ __forceinline__ double2 cmul_seq(double2 a, double2 b) {
    return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.y, b.x, __dmul_rn(a.x, b.y)));
}
__device__ __forceinline__ double flip(double a, int s) {
    return __hiloint2double(__double2hiint(a) ^ s, __double2loint(a));
}
// Re (comp 0, sgn the sign bit) or Im (comp 1, sgn 0) of a b.
__device__ __forceinline__ double prod_seq(double2 a, double2 b, int comp, int sgn) {
    const double u = comp ? a.y : a.x, w = comp ? a.x : a.y;
    return __fma_rn(u, b.x, flip(__dmul_rn(w, b.y), sgn));
}
// The whole sum over k of a[k da] b[k db]: COMP 2 both components (of one lane), else
// acc.x takes the component comp.  The products of eight terms are formed before they
// are added: one chain of load, multiply, FMA and add a term has four latencies.
template <int COMP>
__device__ __forceinline__ void dot_seq(double2& acc, const double2* a, int da, int sa, const double2* b, int db,
                                        int sb, int n, int comp) {
    constexpr int U = 8;
    const int sgn = comp ? 0 : (int)0x80000000;
    auto chunk = [&](int k0, auto count) {
        constexpr int C = decltype(count)::value;
        double2 x[C], y[C];
        double p[C], q[C];
#pragma unroll
        for (int i = 0; i < C; ++i) {
            x[i] = a[(k0 + i) * da];
            y[i] = b[(k0 + i) * db];
        }
#pragma unroll
        for (int i = 0; i < C; ++i) {
            x[i].y = flip(x[i].y, sa);
            y[i].y = flip(y[i].y, sb);
            p[i] = prod_seq(x[i], y[i], COMP == 2 ? 0 : comp, COMP == 2 ? (int)0x80000000 : sgn);
            if (COMP == 2) q[i] = prod_seq(x[i], y[i], 1, 0);
        }
#pragma unroll
        for (int i = 0; i < C; ++i) {
            acc.x = __dadd_rn(acc.x, p[i]);
            if (COMP == 2) acc.y = __dadd_rn(acc.y, q[i]);
        }
    };
    int k = 0;
    for (; k + U <= n; k += U) chunk(k, std::integral_constant<int, U>{});
    for (; k + 2 <= n; k += 2) chunk(k, std::integral_constant<int, 2>{});
    if (k < n) chunk(k, std::integral_constant<int, 1>{});
}

// ---------------------------------------------------------------------------
// Stage GEMM (FP64, CUDA cores; the allocation-free entry point only, whose
// fixed scratch has no room for digit images): D[row][col] = sum_k A[row*lda+k] *
// B[col*ldb+k]; the result is scattered by the stage's index map.  64x64 output tile, 16-wide
// K slices staged in shared memory, 4x4 outputs per thread.
// ---------------------------------------------------------------------------
constexpr int G64_BM = 64, G64_BN = 64, G64_BK = 16;

__global__ void __launch_bounds__(256) k_gemm64_stage(const double* __restrict__ A, long long lda,
                                                      long long sAz, const double* __restrict__ B,
                                                      long long ldb, long long sBz,
                                                      double* __restrict__ out, long long sOz, int M,
                                                      int Nc, long long Ktot, int splitk,
                                                      long long Kc, StageMap map) {
    const int z = blockIdx.z;
    long long K = Ktot;
    if (splitk) {
        const long long k0 = (long long)z * Kc;
        K = Ktot - k0 < Kc ? Ktot - k0 : Kc;
        A += k0;
        B += k0;
        out += (long long)z * sOz;
    } else {
        A += (long long)z * sAz;
        B += (long long)z * sBz;
        out += (long long)z * sOz;
    }
    const long long m0 = (long long)blockIdx.y * G64_BM;
    const int n0 = blockIdx.x * G64_BN;
    __shared__ double As[G64_BK][G64_BM + 1];
    __shared__ double Bs[G64_BK][G64_BN + 1];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;

    for (long long kb = 0; kb < K; kb += G64_BK) {
        for (int e = tid; e < G64_BM * G64_BK; e += 256) {
            const int r = e / G64_BK, kk = e % G64_BK;
            const long long gr = m0 + r, gk = kb + kk;
            As[kk][r] = (gr < M && gk < K) ? A[gr * lda + gk] : 0.0;
        }
        for (int e = tid; e < G64_BN * G64_BK; e += 256) {
            const int cidx = e / G64_BK, kk = e % G64_BK;
            const long long gc = n0 + cidx, gk = kb + kk;
            Bs[kk][cidx] = (gc < Nc && gk < K) ? B[gc * ldb + gk] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < G64_BK; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long row = m0 + ty + 16 * i;
        if (row >= M) continue;
        const long long x = row % map.Dx;
        const long long rb = row / map.Dx;
        const long long b = rb % map.Db;
        const long long a = rb / map.Db;
        const long long roff = a * map.SA + b * map.SB + x * map.SX;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int col = n0 + tx + 16 * j;
            if (col >= Nc) continue;
            const int cc = col / map.Dy, y = col % map.Dy;
            out[roff + cc * map.SC + (long long)y * map.SY] = acc[i][j];
        }
    }
}

// ---------------------------------------------------------------------------
// Complex batched GEMM for N x N matrices (FP64):
//   C = alpha op(A) op(B) + beta C + poly, op in {N, C = conj-transpose},
//   poly = p.c0 I + p.c1 X1 + p.c2 X2 + p.c3 X3 (the terms whose matrix is set).
// Matrices from ident_b on are set to the identity instead.  When skip_ge is
// given and idx >= *skip_ge the launch does nothing (the data-dependent number
// of squarings in the exponential).
//
// Bound by the FP64 rate (two FMAs a clock and SM: 4 n^3 of them a matrix), so
// outputs are summed without padding to a tile, read through L1, in an order that
// is fixed whatever the other matrices of the launch.  SEQ (split-TF32 contexts):
// rounded products added in the order of k, by one lane an output or, where the
// launch has few outputs, by two, its real and its imaginary part.  Else FMA chains:
// eight, one a lane, from n = 32 on (single matrices, of the exponential, count
// most there: at n = 48 3.7 us each, 7.4 by two lanes); below, of even and of odd k,
// by one lane or by two.  Measured, 16 x 16 tiles -> here: the five
// products of a Heun step at n = 10 (over 2501 points, two of them over 5002
// matrices) 914 -> 204 us together; one matrix of n = 48 16.5 -> 3.7 us.  SEQ takes
// six FP64 instructions a term where FMAs take four: the five products at n = 24,
// 501 points, 619 us (FMAs 426).
// ---------------------------------------------------------------------------
// Imaginary part's sign bit flipped by s (conjugation on the integer pipe).
__device__ __forceinline__ double2 zsign(double2 a, int s) { return make_double2(a.x, flip(a.y, s)); }

struct ZPoly {
    double c0 = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;
    const double2 *X1 = nullptr, *X2 = nullptr, *X3 = nullptr;
};

template <int LANES, bool SEQ>
__global__ void __launch_bounds__(128) k_zgemm(int n, int opA, int opB, double2 alpha,
                                               const double2* __restrict__ A, long long sA,
                                               const double2* __restrict__ B, long long sB,
                                               double2 beta, double2* __restrict__ C, long long sC,
                                               uint32_t total, int ident_b, const ZPoly p,
                                               const int* skip_ge, int idx) {
    if (skip_ge != nullptr && idx >= *skip_ge) return;
    const uint32_t gid = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t o = min(gid / LANES, total - 1u);
    const int sub = (int)(gid % LANES);
    const uint32_t nn = (uint32_t)(n * n);
    const int b = (int)(o / nn), e = (int)(o - (uint32_t)b * nn);
    const int row = e / n, col = e - row * n;
    double2 acc = make_double2(0.0, 0.0);
    if (b < ident_b) {
        const double2* a = A + (long long)b * sA + (opA ? row : row * n);
        const double2* bb = B + (long long)b * sB + (opB ? col * n : col);
        const int da = opA ? n : 1, db = opB ? 1 : n;
        const int sa = opA ? (int)0x80000000 : 0, sb = opB ? (int)0x80000000 : 0;
        if (SEQ) {
            dot_seq<LANES == 1 ? 2 : 1>(acc, a, da, sa, bb, db, sb, n, sub);
        } else {
            // the chains of k = 0 .. CH - 1 (mod CH), in as many lanes, or both of two in one
            constexpr int CH = LANES == 1 ? 2 : LANES;
            double2 acc2 = make_double2(0.0, 0.0);
            int k = sub;
#pragma unroll 2
            for (; k + CH - LANES < n; k += CH) {
                cmac(acc, zsign(a[k * da], sa), zsign(bb[k * db], sb));
                if (LANES == 1) cmac(acc2, zsign(a[(k + 1) * da], sa), zsign(bb[(k + 1) * db], sb));
            }
            if (LANES == 1) {
                if (k < n) cmac(acc, zsign(a[k * da], sa), zsign(bb[k * db], sb));
                acc = cadd(acc, acc2);
            }
        }
    }
    if (SEQ) {
        if (LANES == 2) acc.y = __shfl_xor_sync(0xffffffffu, acc.x, 1);  // the other lane's part
    } else {
#pragma unroll
        for (int d = LANES / 2; d > 0; d >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, d);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, d);
        }
    }
    if (sub != 0 || gid / LANES >= total) return;
    double2* c = C + (long long)b * sC + e;
    if (b >= ident_b) {
        *c = make_double2(row == col ? 1.0 : 0.0, 0.0);
        return;
    }
    double2 r = cmul_seq(alpha, acc);
    if (beta.x != 0.0 || beta.y != 0.0) r = cadd(r, cmul_seq(beta, *c));
    if (row == col) r.x += p.c0;
    if (p.X1) r = make_double2(fma(p.c1, p.X1[e].x, r.x), fma(p.c1, p.X1[e].y, r.y));
    if (p.X2) r = make_double2(fma(p.c2, p.X2[e].x, r.x), fma(p.c2, p.X2[e].y, r.y));
    if (p.X3) r = make_double2(fma(p.c3, p.X3[e].x, r.x), fma(p.c3, p.X3[e].y, r.y));
    *c = r;
}

// Sigma_HF(rho)_ij = sum_{l,k} hfK[(i,j),(l,k)] rho_lk, plus h + E d when add_h.
// One warp per (i, j); lanes stride over (l, k).
__global__ void k_mean_field(int N, const double* __restrict__ hfK, const double2* __restrict__ rho,
                             const double2* __restrict__ h, const double2* __restrict__ d, double E,
                             int add_h, double2* __restrict__ out) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int NN = N * N;
    if (warp >= NN) return;
    const double* row = hfK + (long long)warp * NN;
    double re = 0.0, im = 0.0;
    for (int e = lane; e < NN; e += 32) {
        const double kv = row[e];
        const double2 r = rho[e];
        re = fma(kv, r.x, re);
        im = fma(kv, r.y, im);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        if (add_h) {
            re += h[warp].x + E * d[warp].x;
            im += h[warp].y + E * d[warp].y;
        }
        out[warp] = make_double2(re, im);
    }
}

// One stage of Heun's method, every element by four lanes, the two components of
// h rho and of rho h (fixed order of k, rounded products: see dot_seq):
//   k = -i [h, rho] - (I + I^+);  y = base + a (k + kprev)
// with k written to k_out and y also to y2 when given (kprev may be null).
__global__ void __launch_bounds__(64) k_heun_stage(int N, const double2* __restrict__ h,
                                                   const double2* __restrict__ rho,
                                                   const double2* __restrict__ I,
                                                   const double2* __restrict__ base,
                                                   const double2* __restrict__ kprev, double a,
                                                   double2* __restrict__ k_out, double2* __restrict__ y,
                                                   double2* __restrict__ y2) {
    const int gid = blockIdx.x * 64 + threadIdx.x, sub = gid & 3, comp = sub & 1;
    const int e = min(gid >> 2, N * N - 1), i = e / N, j = e % N;
    const double2 *l = (sub & 2 ? rho : h) + i * N, *r = (sub & 2 ? h : rho) + j;
    double2 acc = make_double2(0.0, 0.0);
    dot_seq<1>(acc, l, 1, 0, r, N, 0, N, comp);
    double s = acc.x;
    s = __dadd_rn(s, -__shfl_xor_sync(0xffffffffu, s, 2));
    const double2 c = make_double2(s, __shfl_xor_sync(0xffffffffu, s, 1));  // of lane 0
    if (sub != 0 || (gid >> 2) >= N * N) return;
    const double2 x = I[e], xt = I[j * N + i];
    // -i c = (c.y, -c.x); I + I^+ at (i,j) = I_ij + conj(I_ji)
    double2 k = make_double2(c.y - (x.x + xt.x), -c.x - (x.y - xt.y));
    if (k_out) k_out[e] = k;
    if (kprev) k = cadd(kprev[e], k);
    const double2 b = base[e];
    const double2 v = make_double2(__dadd_rn(b.x, __dmul_rn(a, k.x)), __dadd_rn(b.y, __dmul_rn(a, k.y)));
    y[e] = v;
    if (y2) y2[e] = v;
}

// y = a x + b z (elementwise complex, real a and b).
__global__ void k_lincomb(long long n, double2* __restrict__ y, const double2* __restrict__ x,
                          const double2* __restrict__ z, double a, double b) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double2 xv = x[e];
    const double2 zv = z ? z[e] : make_double2(0.0, 0.0);
    y[e] = make_double2(a * xv.x + b * zv.x, a * xv.y + b * zv.y);
}

__global__ void k_set_identity(int N, int count, double2* __restrict__ A) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * count) return;
    const long long r = e % NN;
    A[e] = make_double2((r / N) == (r % N) ? 1.0 : 0.0, 0.0);
}

// Halvings of an exponential's argument, and squarings of its result, at most: every
// exponential takes as many of the one as of the other (with 30 and 16, arguments of a
// norm above 2^15 gave a root of the exponential).  An argument left larger than 1/2
// keeps the polynomial's accuracy up to a norm of 2^16 (0.5^19 / 19! becomes 1 / 19!).
constexpr int kMaxSquarings = 16;

// expm set-up: A = -i dt (hA + hB)/2; writes A into X, its 1-norm (max column
// sum of |A_ij|) and the number of squarings s so that ||A||/2^s <= 1/2, then
// scales X by 2^-s.  One block.
__global__ void k_expm_setup(int N, double dt, const double2* __restrict__ hA,
                             const double2* __restrict__ hB, double2* __restrict__ X,
                             double* __restrict__ norm_out, int* __restrict__ s_out) {
    __shared__ double colmax[1024];
    const int tid = threadIdx.x;
    double best = 0.0;
    for (int j = tid; j < N; j += blockDim.x) {
        double s = 0.0;
        for (int i = 0; i < N; ++i) {
            const long long e = (long long)i * N + j;
            const double hr = 0.5 * (hA[e].x + hB[e].x), hi = 0.5 * (hA[e].y + hB[e].y);
            s += dt * sqrt(hr * hr + hi * hi);
        }
        best = fmax(best, s);
    }
    colmax[tid] = best;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (tid < o) colmax[tid] = fmax(colmax[tid], colmax[tid + o]);
        __syncthreads();
    }
    const double nrm = colmax[0];
    int s = 0;
    while (s < kMaxSquarings && ldexp(nrm, -s) > 0.5) ++s;
    const double scale = ldexp(1.0, -s);
    for (int e = tid; e < N * N; e += blockDim.x) {
        const double hr = 0.5 * (hA[e].x + hB[e].x), hi = 0.5 * (hA[e].y + hB[e].y);
        // -i dt h = (dt*hi, -dt*hr)
        X[e] = make_double2(scale * dt * hi, -scale * dt * hr);
    }
    if (tid == 0) {
        *norm_out = nrm;
        *s_out = s;
    }
}

// The whole exponential of a matrix of n <= 32 rows in one launch: the argument
// (-i dt (hA + hB)/2, or a general matrix Z) scaled by 2^-s so that its 1-norm is
// at most 1/2, the degree-18 Taylor polynomial as four Horner steps in X^4
// (Paterson and Stockmeyer, SIAM J. Comput. 2, 1973: seven products instead of
// eighteen), s squarings.  From kExpmOneN + 1 rows on a cluster of eight
// CTAs shares every product: each keeps all matrices in shared memory, computes
// an eighth and writes it to all eight (distributed shared memory, one cluster
// barrier a product); below, one CTA is faster than the barriers.  One SM's FP64
// rate bounds a single CTA (n = 24, eighteen products: 520 us; here, cluster:
// 44 us; n = 10: 62 -> 24).
// SEQ (split-TF32 contexts): the propagator feeds FP32 operands and keeps its
// value to the last bit: the polynomial by Horner's scheme, Y = I + X Y / k for
// k = 18 .. 1, every sum in the order of k by one lane a component (dot_seq); 116 us
// at n = 24.
constexpr int kExpmSmallN = 32, kExpmOneN = 12;
constexpr int kExpmLanes = 4;
struct ExpmCoef {  // 1 / k!
    double f[19];
    constexpr ExpmCoef() : f() {
        f[0] = 1.0;
        for (int k = 1; k < 19; ++k) f[k] = f[k - 1] / k;
    }
};
__device__ constexpr ExpmCoef kExpmCoef{};

// C = A B, plus (poly >= 0) sum_{i=0..3} X^i / (4 poly + i)!, into all CTAs' C.
// SEQ: C = A B / poly + I (poly > 0) or A B, one lane a component.
template <int CTAS, bool SEQ>
__device__ void expm_product(int n, int rank, const double2* A, const double2* B, double2* C, int poly,
                             const double2* X1, const double2* X2, const double2* X3) {
    constexpr int kLanes = SEQ ? 2 : kExpmLanes;
    const int nn = n * n, per = (nn + CTAS - 1) / CTAS;
    const int e0 = rank * per, e1 = min(nn, e0 + per), sub = threadIdx.x % kLanes;
    for (int eb = e0; eb < e1; eb += 256 / kLanes) {
        const int et = eb + (int)threadIdx.x / kLanes, e = min(et, e1 - 1), i = e / n, j = e % n;
        double2 acc = make_double2(0.0, 0.0);
        if (SEQ) {
            dot_seq<1>(acc, A + i * n, 1, 0, B + j, n, 0, n, sub);
            const double t = __shfl_xor_sync(0xffffffffu, acc.x, 1);
            acc = sub ? make_double2(t, acc.x) : make_double2(acc.x, t);
        } else {
            for (int k = sub; k < n; k += kLanes) cmac(acc, A[i * n + k], B[k * n + j]);
#pragma unroll
            for (int o = kLanes / 2; o > 0; o >>= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            }
        }
        if (SEQ) {
            if (poly > 0) {
                const double al = 1.0 / poly;
                acc = make_double2(__dmul_rn(al, acc.x), __dmul_rn(al, acc.y));
                if (i == j) acc.x = __dadd_rn(acc.x, 1.0);
            }
        } else if (poly >= 0) {
            const double* c = kExpmCoef.f + 4 * poly;
            if (i == j) acc.x += c[0];
            acc.x = fma(c[1], X1[e].x, fma(c[2], X2[e].x, fma(c[3], X3[e].x, acc.x)));
            acc.y = fma(c[1], X1[e].y, fma(c[2], X2[e].y, fma(c[3], X3[e].y, acc.y)));
        }
        if (CTAS == 1) {
            if (et < e1 && sub == 0) C[e] = acc;
        } else if (et < e1) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(C + e);
            for (int r = sub; r < CTAS; r += kLanes) {
                uint32_t remote;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(dst), "r"(r));
                asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(remote), "d"(acc.x), "d"(acc.y)
                             : "memory");
            }
        }
    }
    if (CTAS == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
template <int CTAS, bool SEQ>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(256)
    k_expm_small(int n, double dt, const double2* __restrict__ hA, const double2* __restrict__ hB,
                 const double2* __restrict__ Z, double2* __restrict__ U, double2* __restrict__ U2) {
    extern __shared__ __align__(16) double2 expm_sm[];
    // the norm only selects s: FP32, with a margin for its rounding, where the last
    // bits of the result may depend on s
    using TN = typename std::conditional<SEQ, double, float>::type;
    __shared__ TN mod[kExpmSmallN * kExpmSmallN], colsum[kExpmSmallN];
    const int tid = threadIdx.x, nn = n * n;
    int rank = 0;
    if (CTAS > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    double2 *X = expm_sm, *X2 = X + nn, *X3 = X2 + nn, *X4 = X3 + nn, *Y = X4 + nn, *W = Y + nn;
    for (int e = tid; e < nn; e += 256) {
        double re, im;  // -i dt (re + i im), or Z
        if (Z) {
            re = Z[e].x;
            im = Z[e].y;
            X[e] = Z[e];
        } else {
            re = 0.5 * (hA[e].x + hB[e].x);
            im = 0.5 * (hA[e].y + hB[e].y);
            X[e] = make_double2(dt * im, -dt * re);
        }
        if (SEQ) mod[e] = (TN)(Z ? hypot(re, im) : sqrt(re * re + im * im));
        else mod[e] = (TN)sqrtf((float)X[e].x * (float)X[e].x + (float)X[e].y * (float)X[e].y);
    }
    __syncthreads();
    if (tid < n) {
        const TN f = SEQ && !Z ? (TN)dt : (TN)1;
        TN sum = 0;
        for (int i = 0; i < n; ++i) sum = fma(f, mod[i * n + tid], sum);
        colsum[tid] = sum;
    }
    __syncthreads();
    TN nrm = 0;
    for (int j = 0; j < n; ++j) nrm = nrm < colsum[j] ? colsum[j] : nrm;
    if (!SEQ) nrm *= (TN)1.0001;
    int s = 0;
    for (; s < kMaxSquarings && nrm > (TN)0.5; ++s) nrm *= (TN)0.5;
    const double scale = __hiloint2double((1023 - s) << 20, 0);
    for (int e = tid; e < nn; e += 256) {
        X[e] = make_double2(scale * X[e].x, scale * X[e].y);
        // the first step of Horner's scheme, X I / 18 + I
        if (SEQ)
            Y[e] = make_double2(__dadd_rn(__dmul_rn(1.0 / 18, X[e].x), e / n == e % n ? 1.0 : 0.0),
                                __dmul_rn(1.0 / 18, X[e].y));
    }
    if (CTAS == 1) {
        __syncthreads();
    } else {
        // every CTA of the cluster has started before remote stores begin
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    double2 *y = Y, *z = W;
    if (SEQ) {
        for (int k = 17; k >= 1; --k) {
            expm_product<CTAS, SEQ>(n, rank, X, y, z, k, nullptr, nullptr, nullptr);
            double2* t = y; y = z; z = t;
        }
    } else {
        expm_product<CTAS, SEQ>(n, rank, X, X, X2, -1, nullptr, nullptr, nullptr);
        expm_product<CTAS, SEQ>(n, rank, X, X2, X3, -1, nullptr, nullptr, nullptr);
        expm_product<CTAS, SEQ>(n, rank, X2, X2, X4, -1, nullptr, nullptr, nullptr);
        // sum_{k=16..18} X^{k-16} / k!
        for (int e = tid; e < nn; e += 256)
            Y[e] = make_double2(fma(kExpmCoef.f[17], X[e].x, kExpmCoef.f[18] * X2[e].x) +
                                    (e / n == e % n ? kExpmCoef.f[16] : 0.0),
                                fma(kExpmCoef.f[17], X[e].y, kExpmCoef.f[18] * X2[e].y));
        __syncthreads();
        for (int j = 3; j >= 0; --j) {
            expm_product<CTAS, SEQ>(n, rank, y, X4, z, j, X, X2, X3);
            double2* t = y; y = z; z = t;
        }
    }
    for (int q = 0; q < s; ++q) {
        expm_product<CTAS, SEQ>(n, rank, y, y, z, -1, nullptr, nullptr, nullptr);
        double2* t = y; y = z; z = t;
    }
    if (rank == 0)
        for (int e = tid; e < nn; e += 256) {
            U[e] = y[e];
            if (U2) U2[e] = y[e];
        }
}
// Y = c16 I + c17 X + c18 X^2
__global__ void k_expm_lead(int n, double c16, double c17, double c18, const double2* __restrict__ X,
                            const double2* __restrict__ X2, double2* __restrict__ Y) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n) return;
    Y[e] = make_double2(fma(c17, X[e].x, c18 * X2[e].x) + (e / n == e % n ? c16 : 0.0),
                        fma(c17, X[e].y, c18 * X2[e].y));
}
// The result of *s squarings that alternated between two buffers.
__global__ void k_expm_select(long long n, const int* __restrict__ s, const double2* __restrict__ even,
                              const double2* __restrict__ odd, double2* __restrict__ U, double2* __restrict__ U2) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double2 x = (*s & 1) ? odd[e] : even[e];
    U[e] = x;
    if (U2) U2[e] = x;
}

// Diagnostics at t_n: {Tr rho, E_total, E_corr, Re Tr I}.
// E_total = 1/2 (Tr[(h+E d) rho] + Tr[h_HF rho]) + 1/2 Im Tr I.
__global__ void k_diagnostics(int N, double E, const double2* __restrict__ h,
                              const double2* __restrict__ d, const double2* __restrict__ hhf,
                              const double2* __restrict__ rho, const double2* __restrict__ I,
                              double* __restrict__ out) {
    __shared__ double s0[256], s1[256], s2[256];
    const int tid = threadIdx.x;
    double t1 = 0.0, t2 = 0.0, tr = 0.0;
    for (int e = tid; e < N * N; e += blockDim.x) {
        const int i = e / N, j = e % N;
        const double2 r = rho[j * N + i];
        const double2 a = make_double2(h[e].x + E * d[e].x, h[e].y + E * d[e].y);
        t1 += a.x * r.x - a.y * r.y;
        t2 += hhf[e].x * r.x - hhf[e].y * r.y;
        if (i == j) tr += rho[e].x;
    }
    s0[tid] = t1;
    s1[tid] = t2;
    s2[tid] = tr;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (tid < o) {
            s0[tid] += s0[tid + o];
            s1[tid] += s1[tid + o];
            s2[tid] += s2[tid + o];
        }
        __syncthreads();
    }
    if (tid == 0) {
        double trI_re = 0.0, trI_im = 0.0;
        for (int i = 0; i < N; ++i) {
            trI_re += I[i * N + i].x;
            trI_im += I[i * N + i].y;
        }
        const double ec = 0.5 * trI_im;
        out[0] = s2[0];
        out[1] = 0.5 * (s0[0] + s1[0]) + ec;
        out[2] = ec;
        out[3] = trI_re;
    }
}

// ---------------------------------------------------------------------------
// GKBA unit forms (FP64 path).  Unit u of a batch holds (G_u, Gb_u); the
// stage-1 operand is B1[u][(c,r)][s] = Gb_c[s][r] (2N x N), the stage-2/3
// operand is the real form of G: Gr[u][(c',p)][(c,q)] with blocks
// [[Re G, -Im G], [Im G, Re G]] (2N x 2N).
// ---------------------------------------------------------------------------
__global__ void k_forms64(int N, int nb, const double2* __restrict__ G, const double2* __restrict__ Gb,
                          double* __restrict__ B1, double* __restrict__ Gr) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * nb) return;
    const int u = (int)(e / NN);
    const int rr = (int)(e % NN);
    const int a = rr / N, b = rr % N;
    // stage-1 operand: entry (s = a, r = b); skipped when only the G forms are wanted
    if (B1 != nullptr) {
        const double2 gb = Gb[u * NN + rr];  // Gb[s][r]
        double* b1 = B1 + (long long)u * 2 * NN;
        b1[(long long)(0 * N + b) * N + a] = gb.x;
        b1[(long long)(1 * N + b) * N + a] = gb.y;
    }
    // stage-2/3 operand: entry (p = a, q = b)
    const double2 g = G[u * NN + rr];
    double* gr = Gr + (long long)u * 4 * NN;
    const long long ld = 2 * N;
    gr[(long long)(0 * N + a) * ld + 0 * N + b] = g.x;
    gr[(long long)(0 * N + a) * ld + 1 * N + b] = -g.y;
    gr[(long long)(1 * N + a) * ld + 0 * N + b] = g.y;
    gr[(long long)(1 * N + a) * ld + 1 * N + b] = g.x;
}

// Units of history point k (batch-local kk = k - k0): u = 2 kk + comp,
//   comp 0 (Sigma^<): G = P_k, Gb = Q_k^+, coefficient -c_k,
//   comp 1 (Sigma^>): G = Q_k, Gb = P_k^+, coefficient +c_k,
// so that I = sum_u coef_u S(G_u, Gb_u) Gb_u (first line of Eq. collint).
// Writes G_u into Gout, Gb_u into Mb and the coefficients.
__global__ void k_gkba_units(int N, int nk, int k0, int L, double dt, const double2* __restrict__ P,
                             const double2* __restrict__ T, const double* __restrict__ w,
                             double2* __restrict__ Gout, double2* __restrict__ Mb,
                             double* __restrict__ coef) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * nk) return;
    const int kk = (int)(e / NN);
    const int rr = (int)(e % NN);
    const int i = rr / N, j = rr % N;
    const long long base = (long long)kk * NN;
    const long long tr = base + (long long)j * N + i;
    const double2 p = P[base + rr], pt = P[tr], t = T[base + rr], tt = T[tr];
    const double2 q = make_double2(t.x - p.x, t.y - p.y), qt = make_double2(tt.x - pt.x, tt.y - pt.y);  // Q = T - P
    Gout[(2 * kk + 0) * NN + rr] = p;
    Gout[(2 * kk + 1) * NN + rr] = q;
    Mb[(2 * kk + 0) * NN + rr] = make_double2(qt.x, -qt.y);  // (Q^+)_ij = conj(Q_ji)
    Mb[(2 * kk + 1) * NN + rr] = make_double2(pt.x, -pt.y);
    if (rr == 0) {
        const int k = k0 + kk;
        double c;
        if (w != nullptr) c = w[k];
        else if (L <= 1) c = 0.0;
        else c = (k == 0 || k == L - 1) ? 0.5 * dt : dt;
        coef[2 * kk + 0] = -c;
        coef[2 * kk + 1] = c;
    }
}

// S_u[i][j] = sum_z part[z][i][u*2N + j] + i part[z][i][u*2N + N + j]
// (split-K partials of the last contraction, rows (u, c, j)).  Two passes with
// a fixed summation order (deterministic): pass 1 sums z-range zc of each
// element into tmp[zc], pass 2 adds the z-ranges in order.  Partials are FP64
// (FP64 path) or FP32 (tensor-core path); all sums are FP64.
// FP32 partials are added in FP32 with compensation (Kahan): the error stays at a
// few ulps of the sum whatever the number of terms, and FP32 adds run at full rate
// (GB300's FP64 rate is low).  The few FP64 partials (oz_items) are plainly added.
template <typename TP>
struct PartialSum {
    TP s = 0, c = 0;
    __device__ __forceinline__ void add(TP x) {
        if (sizeof(TP) == 8) {
            s += x;
            return;
        }
        const TP y = x - c;
        const TP t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

template <typename TP>
__global__ void k_reduce_partials_p1(int N, int Np, int nb, int nz, int zper, long long zstride,
                                     long long Rld, const TP* __restrict__ part,
                                     double2* __restrict__ tmp) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * nb) return;
    const int zc = blockIdx.y;
    const int u = (int)(e / NN);
    const int rr = (int)(e % NN);
    const int i = rr / N, j = rr % N;
    const long long r_re = (long long)u * 2 * Np + j, r_im = r_re + Np;
    const int z0 = zc * zper, z1 = min(nz, z0 + zper);
    PartialSum<TP> re[2], im[2];
    const TP* base = part + (long long)i * Rld;
    int z = z0;
    for (; z + 2 <= z1; z += 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const TP* pz = base + (long long)(z + q) * zstride;
            re[q].add(pz[r_re]);
            im[q].add(pz[r_im]);
        }
    }
    if (z < z1) {
        const TP* pz = base + (long long)z * zstride;
        re[0].add(pz[r_re]);
        im[0].add(pz[r_im]);
    }
    const double sre = ((double)re[0].s - (double)re[0].c) + ((double)re[1].s - (double)re[1].c);
    const double sim = ((double)im[0].s - (double)im[0].c) + ((double)im[1].s - (double)im[1].c);
    tmp[(long long)zc * NN * nb + e] = make_double2(sre, sim);
}

__global__ void k_reduce_partials_p2(long long n, int nzc, const double2* __restrict__ tmp,
                                     double2* __restrict__ S) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    double re = 0.0, im = 0.0;
    for (int zc = 0; zc < nzc; ++zc) {
        const double2 t = tmp[(long long)zc * n + e];
        re += t.x;
        im += t.y;
    }
    S[e] = make_double2(re, im);
}

// I_acc[e] += sum_u coef[u] * Y[u][e] in two passes with a fixed order
// (deterministic): pass 1 sums the contiguous unit range z of every element
// into tmp[z][e] (blockIdx.y = z), pass 2 adds the ranges in order.  Small
// bases have few elements and many units (N = 10: 100 elements, up to 10^4
// units per batch), so the units are spread over the grid, not looped by one
// thread per element.
constexpr int kWsumRanges = 256;
__global__ void k_weighted_sum_p1(int NN, int nb, int per, const double* __restrict__ coef,
                                  const double2* __restrict__ Y, double2* __restrict__ tmp) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NN) return;
    const int u0 = blockIdx.y * per;
    const int u1 = min(nb, u0 + per);
    double re = 0.0, im = 0.0;
    for (int u = u0; u < u1; ++u) {
        const double c = coef[u];
        const double2 y = Y[(long long)u * NN + e];
        re = fma(c, y.x, re);
        im = fma(c, y.y, im);
    }
    tmp[(long long)blockIdx.y * NN + e] = make_double2(re, im);
}
// One warp per element (a thread per element that loads as it adds took 31 us a
// call at N = 10, here 4).
__global__ void __launch_bounds__(256) k_weighted_sum_p2(int NN, int nz, const double2* __restrict__ tmp,
                                                         double2* __restrict__ I_acc) {
    const int e = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (e >= NN) return;
    double re = 0.0, im = 0.0;
    for (int z = lane; z < nz; z += 32) {
        const double2 t = tmp[(long long)z * NN + e];
        re += t.x;
        im += t.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        I_acc[e].x += re;
        I_acc[e].y += im;
    }
}
// The ranges in order, for split-TF32 contexts (I feeds rho~, which becomes FP32
// operands): a block loads the ranges of eight components to shared memory, a thread
// per component adds them (256 ranges of N = 24: 14 us, in the tree above 5).
__global__ void __launch_bounds__(256) k_weighted_sum_p2_seq(int NN2, int nz, const double* __restrict__ tmp,
                                                             double* __restrict__ I_acc) {
    __shared__ double part[8][kWsumRanges + 1];
    const int c = threadIdx.x & 7, e = blockIdx.x * 8 + c;
    for (int z = threadIdx.x >> 3; z < nz; z += 32) part[c][z] = e < NN2 ? tmp[(long long)z * NN2 + e] : 0.0;
    __syncthreads();
    if (threadIdx.x >= 8 || e >= NN2) return;
    double s = 0.0;
#pragma unroll 16
    for (int z = 0; z < nz; ++z) s = __dadd_rn(s, part[c][z]);
    I_acc[e] = __dadd_rn(I_acc[e], s);
}
static void launch_weighted_sum_p2(gkba_ctx* c, int NN, int nz, double2* I) {
    if (tensor_core_path(c))
        k_weighted_sum_p2_seq<<<(unsigned)((2 * NN + 7) / 8), 256, 0, c->stream>>>(2 * NN, nz, (const double*)c->red_tmp,
                                                                                  (double*)I);
    else
        k_weighted_sum_p2<<<(unsigned)((NN * 32LL + 255) / 256), 256, 0, c->stream>>>(NN, nz, c->red_tmp, I);
}

// hfK[(i*N + j)*N*N + l*N + k] = 2 v_iklj - v_ikjl  (Sigma_HF as a matrix-vector product)
__global__ void k_build_hfK(int N, const double* __restrict__ v, double* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = N, N4 = n * n * n * n;
    if (e >= N4) return;
    const long long k = e % n, l = (e / n) % n, j = (e / n / n) % n, i = e / n / n / n;
    out[e] = 2.0 * v[((i * n + k) * n + l) * n + j] - v[((i * n + k) * n + j) * n + l];
}

// wS[j][m][q][s] = w_mqsj = 2 v_mqsj - v_qmsj (the direct and exchange terms of
// Eq. (2bse) after relabelling m <-> q in the exchange term).
__global__ void k_build_wS64(int N, const double* __restrict__ v, double* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = N, N4 = n * n * n * n;
    if (e >= N4) return;
    const long long s = e % n, q = (e / n) % n, m = (e / n / n) % n, j = e / n / n / n;
    out[e] = 2.0 * v[((m * n + q) * n + s) * n + j] - v[((q * n + m) * n + s) * n + j];
}

// vK[i][n][r][p] = v_irpn (K index (n, r, p) of the last contraction).
__global__ void k_build_vK64(int N, const double* __restrict__ v, double* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = N, N4 = n * n * n * n;
    if (e >= N4) return;
    const long long p = e % n, r = (e / n) % n, nn = (e / n / n) % n, i = e / n / n / n;
    out[e] = v[((i * n + r) * n + p) * n + nn];
}

inline unsigned grid1(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// ---------------------------------------------------------------------------
// Structured interactions (Sec. III A, B): the self-energy without the N^5
// contraction chain.
// ---------------------------------------------------------------------------
// Diagonal basis, Eq. (2b-diag): S_ij = U_i U_j G_ij Gb_ji G_ij
// (the entrywise form diag(V) o diag(V) o G o Gb^T o G of Eq. (2b-diag-opt)).
__global__ void k_sigma_diag(int N, int nb, const double* __restrict__ U,
                             const double2* __restrict__ G, const double2* __restrict__ Gb,
                             double2* __restrict__ S) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * nb) return;
    const long long u = e / NN;
    const int rr = (int)(e % NN);
    const int i = rr / N, j = rr % N;
    const double2 g = G[e];
    const double2 x = cmul(cmul(g, g), Gb[u * NN + (long long)j * N + i]);
    const double s = U[i] * U[j];
    S[e] = make_double2(s * x.x, s * x.y);
}

// Symmetric basis, Eq. (2b-symm), bubble and exchange together:
//   S_ij = sum_kl V_ik V_jl (2 G_ij Gb_lk G_kl - G_il Gb_lk G_kj)
//        = sum_l V_jl (2 G_ij r_l - G_il W_lj)
// with, for the row i of the block,
//   r_l  = sum_k V_ik Gb_lk G_kl   (the bubble's [V x (Gb^T o G)]_il, Eq. bubble-contract)
//   W_lj = sum_k V_ik Gb_lk G_kj   (N^3 per row: the exchange term has no
//                                   matrix-product form for the full matrix).
// One block per (row i, unit u); r_l in shared memory; a thread per column j
// (the Gb_lk loads are the same for all threads of a warp, the G_kj loads are
// consecutive in j).  N^4 per unit.
__global__ void k_sigma_symm(int N, const double* __restrict__ V, const double2* __restrict__ G,
                             const double2* __restrict__ Gb, double2* __restrict__ S) {
    extern __shared__ double2 r_sh[];
    const int i = blockIdx.x;
    const long long NN = (long long)N * N;
    const double2* g = G + (long long)blockIdx.y * NN;
    const double2* gb = Gb + (long long)blockIdx.y * NN;
    const double* vi = V + (long long)i * N;
    for (int l = threadIdx.x; l < N; l += blockDim.x) {
        double2 acc = make_double2(0.0, 0.0);
        for (int k = 0; k < N; ++k) {
            const double2 a = gb[(long long)l * N + k];
            cmac(acc, make_double2(vi[k] * a.x, vi[k] * a.y), g[(long long)k * N + l]);
        }
        r_sh[l] = acc;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        const double2 gij = g[(long long)i * N + j];
        double2 s = make_double2(0.0, 0.0);
        for (int l = 0; l < N; ++l) {
            double2 w = make_double2(0.0, 0.0);
            for (int k = 0; k < N; ++k) {
                const double2 a = gb[(long long)l * N + k];
                cmac(w, make_double2(vi[k] * a.x, vi[k] * a.y), g[(long long)k * N + j]);
            }
            const double2 b = cmul(gij, r_sh[l]);
            const double2 x = cmul(g[(long long)i * N + l], w);
            const double vjl = V[(long long)j * N + l];
            s = cadd(s, make_double2(vjl * (2.0 * b.x - x.x), vjl * (2.0 * b.y - x.y)));
        }
        S[(long long)blockIdx.y * NN + (long long)i * N + j] = s;
    }
}

// Same for N <= 24 with G, Gb, V and r in shared memory, several units a block
// (64 threads of work: finer blocks balance the SMs better than 128):
//   r[i][l] = sum_k V_ik Gb_lk G_kl = [V x (Gb^T o G)]_il   (N^3)
//   S_ij    = sum_l V_jl (2 G_ij r[i][l] - G_il sum_k V_ik Gb_lk G_kj)   (N^2 per (i, j))
// Bound by the FP64 rate.  A thread holds one row i and kSymmJ columns j, so that
// V_ik Gb_lk is formed once for all of them: 4.4 FP64 instructions a term of the
// N^4 sum (8 with one column a thread and multiplies kept apart from adds).
// Measured at N = 10, 2002 units: 493 -> 270 us.
constexpr int kSymmSmallN = 24, kSymmJ = 5, kSymmMaxUnits = 16, kSymmThreads = 64;
inline int symm_units(int N) {  // units a block
    const int per = N * ((N + kSymmJ - 1) / kSymmJ);
    return std::max(1, std::min(kSymmMaxUnits, kSymmThreads / per));
}
inline size_t symm_smem(int N) { return (size_t)N * N * (8 + symm_units(N) * 3 * 16); }
__global__ void __launch_bounds__(kSymmThreads) k_sigma_symm_small(int N, int nb, int upb, const double* __restrict__ V,
                                                           const double2* __restrict__ G,
                                                           const double2* __restrict__ Gb,
                                                           double2* __restrict__ S) {
    extern __shared__ __align__(16) double2 symm_sm[];
    const int NN = N * N, u0 = blockIdx.x * upb, nu = min(upb, nb - u0);
    double2 *g_s = symm_sm, *gb_s = g_s + upb * NN, *r_s = gb_s + upb * NN;
    double* vs = (double*)(r_s + upb * NN);
    const long long base = (long long)u0 * NN;
    for (int e = threadIdx.x; e < NN; e += blockDim.x) vs[e] = V[e];
    for (int e = threadIdx.x; e < nu * NN; e += blockDim.x) {
        g_s[e] = G[base + e];
        gb_s[e] = Gb[base + e];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nu * NN; e += blockDim.x) {
        const int u = e / NN, rr = e - u * NN, i = rr / N, l = rr - i * N;
        const double2 *g = g_s + u * NN, *gb = gb_s + u * NN;
        double2 acc = make_double2(0.0, 0.0);
        for (int k = 0; k < N; ++k) {
            const double2 a = gb[l * N + k];
            const double v = vs[i * N + k];
            cmac(acc, make_double2(v * a.x, v * a.y), g[k * N + l]);
        }
        r_s[e] = acc;
    }
    __syncthreads();
    const int njb = (N + kSymmJ - 1) / kSymmJ, per = N * njb;
    for (int t = threadIdx.x; t < nu * per; t += blockDim.x) {
        const int u = t / per, q = t - u * per, i = q / njb, j0 = (q - i * njb) * kSymmJ;
        const double2 *g = g_s + u * NN, *gb = gb_s + u * NN, *r = r_s + u * NN;
        double2 s[kSymmJ];
        int jc[kSymmJ];
#pragma unroll
        for (int m = 0; m < kSymmJ; ++m) {
            s[m] = make_double2(0.0, 0.0);
            jc[m] = min(j0 + m, N - 1);
        }
        for (int l = 0; l < N; ++l) {
            double2 w[kSymmJ];
#pragma unroll
            for (int m = 0; m < kSymmJ; ++m) w[m] = make_double2(0.0, 0.0);
            for (int k = 0; k < N; ++k) {
                const double2 a = gb[l * N + k];
                const double v = vs[i * N + k];
                const double2 va = make_double2(v * a.x, v * a.y);
#pragma unroll
                for (int m = 0; m < kSymmJ; ++m) cmac(w[m], va, g[k * N + jc[m]]);
            }
            const double2 gil = g[i * N + l], ril = r[i * N + l];
#pragma unroll
            for (int m = 0; m < kSymmJ; ++m) {
                const double2 b = cmul(g[i * N + jc[m]], ril), x = cmul(gil, w[m]);
                const double vjl = vs[jc[m] * N + l];
                s[m] = cadd(s[m], make_double2(vjl * (2.0 * b.x - x.x), vjl * (2.0 * b.y - x.y)));
            }
        }
#pragma unroll
        for (int m = 0; m < kSymmJ; ++m)
            if (j0 + m < N) S[base + u * NN + i * N + j0 + m] = s[m];
    }
}

// ---------------------------------------------------------------------------
// Adjoint of the collision integral: per-unit elementwise steps.
// ---------------------------------------------------------------------------
// out_u = op(in_u) for N x N units: conjugate and/or transpose.
__global__ void k_unit_xform(int N, long long n_el, const double2* __restrict__ in,
                             double2* __restrict__ out, int conj, int transpose) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_el) return;
    const long long NN = (long long)N * N, u = e / NN;
    const int rr = (int)(e % NN), i = rr / N, j = rr % N;
    double2 x = in[u * NN + (transpose ? (long long)j * N + i : rr)];
    if (conj) x.y = -x.y;
    out[e] = x;
}
// y_u += x_u (or x_u^T)
__global__ void k_unit_acc(int N, long long n_el, double2* __restrict__ y,
                           const double2* __restrict__ x, int transpose) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_el) return;
    const long long NN = (long long)N * N, u = e / NN;
    const int rr = (int)(e % NN), i = rr / N, j = rr % N;
    const double2 a = x[u * NN + (transpose ? (long long)j * N + i : rr)];
    y[e].x += a.x;
    y[e].y += a.y;
}
// Ybar_u = coef_u Ibar (I = sum_u coef_u Y_u with real coefficients)
__global__ void k_scale_units(int N, int nb, const double* __restrict__ coef,
                              const double2* __restrict__ Ibar, double2* __restrict__ Y) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * nb) return;
    const double c = coef[e / NN];
    const double2 b = Ibar[e % NN];
    Y[e] = make_double2(c * b.x, c * b.y);
}
// Per history point k (units 2k: G = P, Gb = Q^+; 2k+1: G = Q, Gb = P^+):
//   Pbar = Gbar_(2k) + (Gbbar_(2k+1))^+,  Qbar = Gbar_(2k+1) + (Gbbar_(2k))^+
__global__ void k_vjp_points(int N, int nk, const double2* __restrict__ Gbar,
                             const double2* __restrict__ Gbbar, double2* __restrict__ Pbar,
                             double2* __restrict__ Qbar) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long NN = (long long)N * N;
    if (e >= NN * nk) return;
    const long long k = e / NN;
    const int rr = (int)(e % NN), i = rr / N, j = rr % N;
    const long long tr = (long long)j * N + i;
    const double2 g0 = Gbar[(2 * k) * NN + rr], g1 = Gbar[(2 * k + 1) * NN + rr];
    const double2 b0 = Gbbar[(2 * k) * NN + tr], b1 = Gbbar[(2 * k + 1) * NN + tr];
    Pbar[e] = make_double2(g0.x + b1.x, g0.y - b1.y);
    Qbar[e] = make_double2(g1.x + b0.x, g1.y - b0.y);
}

// ---------------------------------------------------------------------------
// Adjoint of the Heun step: small N x N helpers.
// ---------------------------------------------------------------------------
// y += i s (a - b)
__global__ void k_add_i_diff(long long n, double2* __restrict__ y, const double2* __restrict__ a,
                             const double2* __restrict__ b, double s) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double re = a[e].x - b[e].x, im = a[e].y - b[e].y;
    y[e].x += -s * im;
    y[e].y += s * re;
}
// Ibar = -(kbar + kbar^+)   (k = ... - (I + I^+))
__global__ void k_ibar_from_kbar(int N, const double2* __restrict__ kb, double2* __restrict__ Ib) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N * N) return;
    const int i = e / N, j = e % N;
    const double2 a = kb[e], b = kb[j * N + i];
    Ib[e] = make_double2(-(a.x + b.x), -(a.y - b.y));
}
// rho_bar[l][k] += sum_ij hfK[(i,j)][(l,k)] hbar[i][j]  (adjoint of the mean field, hfK real)
__global__ void k_mean_field_adj(int N, const double* __restrict__ hfK, const double2* __restrict__ hb,
                                 double2* __restrict__ rb) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int NN = N * N;
    if (warp >= NN) return;
    double re = 0.0, im = 0.0;
    for (int e = lane; e < NN; e += 32) {
        const double kv = hfK[(long long)e * NN + warp];
        re = fma(kv, hb[e].x, re);
        im = fma(kv, hb[e].y, im);
    }
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        rb[warp].x += re;
        rb[warp].y += im;
    }
}
// out += Re sum_ij conj(hbar_ij) d_ij   (dL/dE for h = ... + E d, E real); one block
__global__ void k_field_grad(int N, const double2* __restrict__ hb, const double2* __restrict__ d,
                             double* __restrict__ out) {
    __shared__ double part[256];
    double acc = 0.0;
    for (int e = threadIdx.x; e < N * N; e += blockDim.x) acc += hb[e].x * d[e].x + hb[e].y * d[e].y;
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out += part[0];
}
// Fréchet block for the adjoint of U = exp(X), X = -i dt (hA + hB)/2:
//   Z = [[X^+, Ubar / nu], [0, X^+]] (2N x 2N), nu = max(1, ||Ubar||_1) so that
// the scaling of the exponential stays small; the top-right block of exp(Z)
// times nu is L_exp(X^+, Ubar) = Xbar.  One block.
__global__ void k_frechet_block(int N, double dt, const double2* __restrict__ hA,
                                const double2* __restrict__ hB, const double2* __restrict__ Ub,
                                double2* __restrict__ Z, double* __restrict__ nu_out) {
    __shared__ double colmax[256];
    double best = 0.0;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        double sum = 0.0;
        for (int i = 0; i < N; ++i) sum += hypot(Ub[i * N + j].x, Ub[i * N + j].y);
        best = fmax(best, sum);
    }
    colmax[threadIdx.x] = best;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) colmax[threadIdx.x] = fmax(colmax[threadIdx.x], colmax[threadIdx.x + o]);
        __syncthreads();
    }
    const double nu = fmax(1.0, colmax[0]);
    const int M = 2 * N;
    for (int e = threadIdx.x; e < M * M; e += blockDim.x) {
        const int r = e / M, c = e % M;
        double2 z = make_double2(0.0, 0.0);
        if ((r < N && c < N) || (r >= N && c >= N)) {
            // X^+ with X = -i dt h, h = (hA + hB)/2 Hermitian: X^+ = i dt h
            const int i = r % N, j = c % N;
            const double hr = 0.5 * (hA[i * N + j].x + hB[i * N + j].x);
            const double hi = 0.5 * (hA[i * N + j].y + hB[i * N + j].y);
            z = make_double2(-dt * hi, dt * hr);
        } else if (r < N && c >= N) {
            const double2 u = Ub[r * N + (c - N)];
            z = make_double2(u.x / nu, u.y / nu);
        }
        Z[e] = z;
    }
    if (threadIdx.x == 0) *nu_out = nu;
}
// hbar_A += (i dt / 2) nu W[0:N, N:2N];  hbar_B += same  (X = -i dt (hA + hB)/2)
__global__ void k_frechet_apply(int N, double dt, const double2* __restrict__ W,
                                const double* __restrict__ nu, double2* __restrict__ hA_b,
                                double2* __restrict__ hB_b) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N * N) return;
    const int i = e / N, j = e % N;
    const double2 w = W[i * (2 * N) + N + j];
    const double s = 0.5 * dt * (*nu);
    const double2 a = make_double2(-s * w.y, s * w.x);  // i s w
    hA_b[e].x += a.x;
    hA_b[e].y += a.y;
    hB_b[e].x += a.x;
    hB_b[e].y += a.y;
}
// exp(Z) for a general complex n x n matrix: scaling set-up (1-norm, number of
// squarings s with ||Z||_1 / 2^s <= 1/2, Z scaled by 2^-s into X).  One block.
__global__ void k_expm_setup_general(int n, const double2* __restrict__ Z, double2* __restrict__ X,
                                     int* __restrict__ s_out) {
    __shared__ double colmax[256];
    double best = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double sum = 0.0;
        for (int i = 0; i < n; ++i) sum += hypot(Z[i * n + j].x, Z[i * n + j].y);
        best = fmax(best, sum);
    }
    colmax[threadIdx.x] = best;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) colmax[threadIdx.x] = fmax(colmax[threadIdx.x], colmax[threadIdx.x + o]);
        __syncthreads();
    }
    const double nrm = colmax[0];
    int s = 0;
    while (s < kMaxSquarings && ldexp(nrm, -s) > 0.5) ++s;
    const double scale = ldexp(1.0, -s);
    for (int e = threadIdx.x; e < n * n; e += blockDim.x)
        X[e] = make_double2(scale * Z[e].x, scale * Z[e].y);
    if (threadIdx.x == 0) *s_out = s;
}

// dst = sum_u src_u over nb N x N units (fixed order)
__global__ void k_sum_units(long long NN, int nb, const double2* __restrict__ src,
                            double2* __restrict__ dst) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NN) return;
    double re = 0.0, im = 0.0;
    for (int u = 0; u < nb; ++u) {
        re += src[u * NN + e].x;
        im += src[u * NN + e].y;
    }
    dst[e] = make_double2(re, im);
}

// ---------------------------------------------------------------------------
// Gradient with respect to the Coulomb integrals (FP64 path).
// ---------------------------------------------------------------------------
// out[a][K] += sum_{u, c, b} S_c(u, a, b) X[u][c][b][K]   (K < N^3)
// with S_c the real (c = 0) / imaginary (c = 1) part of Sbar_u[a][b], or of
// Sbar_u[b][a] when transposeS; X planar complex [u][c][N][N^3] (unit stride
// 2 N^4), i.e. out = Re sum conj(Sbar) X over the contracted index.
__global__ void k_vbar_slot(int N, int nb, const double2* __restrict__ Sbar, int transposeS,
                            const double* __restrict__ X, double* __restrict__ out) {
    const long long N3 = (long long)N * N * N;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N3 * N) return;
    const int a = (int)(e / N3);
    const long long K = e % N3;
    const long long NN = (long long)N * N;
    double acc = 0.0;
    for (int u = 0; u < nb; ++u) {
        const double* xu = X + (long long)u * 2 * N * N3;
        const double2* su = Sbar + (long long)u * NN;
        for (int b = 0; b < N; ++b) {
            const double2 sv = transposeS ? su[(long long)b * N + a] : su[(long long)a * N + b];
            acc = fma(sv.x, xu[(long long)b * N3 + K], acc);
            acc = fma(sv.y, xu[N3 * N + (long long)b * N3 + K], acc);
        }
    }
    out[e] += acc;
}
// vbar[a][b][c][d] += vslot[a][(d, b, c)] + 2 wslot[d][(a, c, b)] - wslot[d][(b, c, a)]
// (vslot[i][(n,r,p)] = dL/dv_irpn; wslot[j][(m,s,q)] = dL/dw_mqsj, w_mqsj = 2 v_mqsj - v_qmsj)
__global__ void k_fold_vbar(int N, const double* __restrict__ vslot, const double* __restrict__ wslot,
                            double* __restrict__ vbar) {
    const long long n = N;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n * n * n) return;
    const long long d = e % n, c = (e / n) % n, b = (e / n / n) % n, a = e / n / n / n;
    const long long N3 = n * n * n;
    double x = vslot[a * N3 + (d * n + b) * n + c];
    x += 2.0 * wslot[d * N3 + (a * n + c) * n + b];
    x -= wslot[d * N3 + (b * n + c) * n + a];
    vbar[e] += x;
}
// Mean-field part, for h = ... + Sigma_HF(rho), Sigma_HF_ij = sum_kl (2 v_iklj - v_ikjl) rho_lk:
// vbar[a][b][c][d] += 2 Re(conj(hbar_ad) rho_cb) - Re(conj(hbar_ac) rho_db)
__global__ void k_vbar_mean_field(int N, const double2* __restrict__ hb, const double2* __restrict__ rho,
                                  double* __restrict__ vbar) {
    const long long n = N;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n * n * n) return;
    const long long d = e % n, c = (e / n) % n, b = (e / n / n) % n, a = e / n / n / n;
    const double2 h1 = hb[a * n + d], r1 = rho[c * n + b];
    const double2 h2 = hb[a * n + c], r2 = rho[d * n + b];
    vbar[e] += 2.0 * (h1.x * r1.x + h1.y * r1.y) - (h2.x * r2.x + h2.y * r2.y);
}
// omega layout for the w-slot chain: wO[i][n][p][r] = v_irpn
__global__ void k_build_vomega64(int N, const double* __restrict__ v, double* __restrict__ out) {
    const long long n = N;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n * n * n) return;
    const long long r = e % n, p = (e / n) % n, nn = (e / n / n) % n, i = e / n / n / n;
    out[e] = v[((i * n + r) * n + p) * n + nn];
}

}  // namespace

// ---------------------------------------------------------------------------
// Host wrappers
// ---------------------------------------------------------------------------

gkba_status fp64_prepare_model(gkba_ctx* c) {
    const long long n = c->N, N4 = n * n * n * n;
    for (auto kfn : {k_expm_small<8, false>, k_expm_small<8, true>})
        GKBA_CUDA(c, cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(6 * kExpmSmallN * kExpmSmallN * sizeof(double2))));
    auto t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_build_hfK<<<grid1(N4, 256), 256, 0, c->stream>>>(c->N, c->v, c->hfK);
    GKBA_TRY(launch_end(c, t));
    if (c->prec != GKBA_FP64 || c->kind != GKBA_V_GENERAL) return GKBA_OK;
    t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_build_wS64<<<grid1(N4, 256), 256, 0, c->stream>>>(c->N, c->v, c->wS64);
    GKBA_TRY(launch_end(c, t));
    t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_build_vK64<<<grid1(N4, 256), 256, 0, c->stream>>>(c->N, c->v, c->vK64);
    GKBA_TRY(launch_end(c, t));
    GKBA_TRY(oz_prepare(c));
    return oz_slice(c, c->vK64, n * n * n, 0, c->N, n * n * n, 1, c->vKimg);
}

gkba_status gemm64_stage(gkba_ctx* c, int cls, const double* A, long long lda, long long sAz,
                         const double* B, long long ldb, long long sBz, double* out,
                         long long sOz, int M, int Nc, long long Ktot, int nz, StageMap map,
                         double flops, double bytes) {
    const long long fit = (long long)(c->ozimg_bytes / oz_img_bytes(Nc, Ktot));
    if (fit < 1) return fail(c, GKBA_ESTATE, "the digit image of an operand of %d x %lld does not fit", Nc, Ktot);
    const int most = sBz ? (int)std::min<long long>(fit, nz) : nz;
    for (int z = 0; z < nz; z += most) {
        const int n = std::min(most, nz - z), nB = sBz ? n : 1;
        GKBA_TRY(oz_slice(c, B + z * sBz, ldb, sBz, Nc, Ktot, nB, c->ozimg));
        GKBA_TRY(oz_gemm(c, cls, A + z * sAz, lda, sAz, B + z * sBz, ldb, sBz, c->ozimg, nB, Nc, Ktot, out + z * sOz, sOz,
                         M, n, 1, 0, map, flops * n / nz, bytes * n / nz));
    }
    return GKBA_OK;
}

static gkba_status zgemm_impl(gkba_ctx* c, int cls, int n, char opA, char opB, double2 alpha,
                              const double2* A, long long sA, const double2* B, long long sB,
                              double2 beta, double2* C, long long sC, int batch, int n_ident,
                              const ZPoly& p, const int* skip_ge, int idx) {
    const double flops = 8.0 * n * (double)n * n;
    const long long nn = (long long)n * n;
    const int all = batch + n_ident;
    const int most = (int)std::min<long long>(1LL << 30, (1LL << 31) / (8 * nn));  // 32-bit thread index
    for (int b0 = 0; b0 < all; b0 += most) {
        const int nb = std::min(most, all - b0), nid = std::max(0, std::min(nb, batch - b0));
        const uint32_t total = (uint32_t)(nb * nn);
        // one lane an output once the launch has about a warp for every SM's scheduler
        const bool seq = tensor_core_path(c), few = total <= 32u * (unsigned)c->num_sms;
        const int lanes = !seq && n >= 32 ? 8 : few ? 2 : 1;
        auto kfn = seq          ? (few ? k_zgemm<2, true> : k_zgemm<1, true>)
                   : lanes == 8 ? k_zgemm<8, false>
                   : lanes == 2 ? k_zgemm<2, false>
                                : k_zgemm<1, false>;
        const int bs = (long long)total * lanes >= 512LL * c->num_sms ? 128 : 32;
        auto t = launch_begin(c, cls, flops * nid, 0.0);
        kfn<<<grid1((long long)total * lanes, bs), bs, 0, c->stream>>>(n, opA == 'C', opB == 'C', alpha, A + b0 * sA, sA, B + b0 * sB, sB,
                                                    beta, C + b0 * sC, sC, total, nid, p, skip_ge, idx);
        GKBA_TRY(launch_end(c, t));
    }
    return GKBA_OK;
}

gkba_status zgemm_batched(gkba_ctx* c, int cls, int n, char opA, char opB, double2 alpha,
                          const double2* A, long long sA, const double2* B, long long sB,
                          double2 beta, double2* C, long long sC, int batch, int n_ident) {
    if (batch + n_ident <= 0) return GKBA_OK;
    return zgemm_impl(c, cls, n, opA, opB, alpha, A, sA, B, sB, beta, C, sC, batch, n_ident, ZPoly{}, nullptr, 0);
}

gkba_status mean_field(gkba_ctx* c, const double2* rho, double2* out) {
    const int NN = c->N * c->N;
    auto t = launch_begin(c, K_STEP, 8.0 * NN * (double)NN, 8.0 * NN * (double)NN);
    k_mean_field<<<grid1((long long)NN * 32, 256), 256, 0, c->stream>>>(c->N, c->hfK, rho, c->h,
                                                                         c->d, 0.0, 0, out);
    return launch_end(c, t);
}

gkba_status h_hf(gkba_ctx* c, double E, const double2* rho, double2* out) {
    const int NN = c->N * c->N;
    auto t = launch_begin(c, K_STEP, 8.0 * NN * (double)NN, 8.0 * NN * (double)NN);
    k_mean_field<<<grid1((long long)NN * 32, 256), 256, 0, c->stream>>>(c->N, c->hfK, rho, c->h,
                                                                         c->d, E, 1, out);
    return launch_end(c, t);
}

gkba_status heun_stage(gkba_ctx* c, const double2* hhf, const double2* rho, const double2* I, const double2* base,
                       const double2* kprev, double a, double2* k_out, double2* y, double2* y2) {
    const long long NN = (long long)c->N * c->N;
    auto t = launch_begin(c, K_STEP, 16.0 * NN * c->N, 0.0);
    k_heun_stage<<<grid1(NN * 4, 64), 64, 0, c->stream>>>(c->N, hhf, rho, I, base, kprev, a, k_out, y, y2);
    return launch_end(c, t);
}

// exp(X) by products spread over all SMs: the degree-18 Taylor polynomial in the
// form that k_expm_small takes (Horner for split-TF32 contexts, else Paterson and
// Stockmeyer), then kMaxSquarings squarings of which the device-side count
// c->dint[0] runs.  X: the scaled argument; X2, X3, X4, Y, W: n x n scratch; the result goes
// to U (and U2).
static gkba_status expm_products(gkba_ctx* c, int n, const double2* X, double2* X2, double2* X3, double2* X4,
                                 double2* Y, double2* W, double2* U, double2* U2) {
    const long long nn = (long long)n * n;
    const double2 one = make_double2(1.0, 0.0), zero = make_double2(0.0, 0.0);
    auto prod = [&](const double2* A, const double2* B, double2* C, const ZPoly& p) {
        return zgemm_impl(c, K_STEP, n, 'N', 'N', one, A, 0, B, 0, zero, C, 0, 1, 0, p, nullptr, 0);
    };
    double2 *y = Y, *z = W;
    if (tensor_core_path(c)) {
        ZPoly p;
        p.c0 = 1.0;
        GKBA_TRY(zgemm_impl(c, K_STEP, n, 'N', 'N', one, X, 0, X, 0, zero, y, 0, 0, 1, ZPoly{}, nullptr, 0));  // I
        for (int k = 18; k >= 1; --k) {
            GKBA_TRY(zgemm_impl(c, K_STEP, n, 'N', 'N', make_double2(1.0 / k, 0.0), X, 0, y, 0, zero, z, 0, 1, 0, p,
                                nullptr, 0));
            std::swap(y, z);
        }
    } else {
        GKBA_TRY(prod(X, X, X2, ZPoly{}));
        GKBA_TRY(prod(X, X2, X3, ZPoly{}));
        GKBA_TRY(prod(X2, X2, X4, ZPoly{}));
        double f[19];
        f[0] = 1.0;
        for (int k = 1; k <= 18; ++k) f[k] = f[k - 1] / k;
        {
            auto t = launch_begin(c, K_STEP, 0.0, 0.0);
            k_expm_lead<<<grid1(nn, 256), 256, 0, c->stream>>>(n, f[16], f[17], f[18], X, X2, Y);
            GKBA_TRY(launch_end(c, t));
        }
        for (int j = 3; j >= 0; --j) {
            ZPoly p;
            p.c0 = f[4 * j];
            p.c1 = f[4 * j + 1];
            p.c2 = f[4 * j + 2];
            p.c3 = f[4 * j + 3];
            p.X1 = X;
            p.X2 = X2;
            p.X3 = X3;
            GKBA_TRY(prod(y, X4, z, p));
            std::swap(y, z);
        }
    }
    // X3 is free now: squarings alternate between y and it
    double2* sq[2] = {y, X3};
    for (int i = 0; i < kMaxSquarings; ++i)
        GKBA_TRY(zgemm_impl(c, K_STEP, n, 'N', 'N', one, sq[i & 1], 0, sq[i & 1], 0, zero, sq[(i + 1) & 1], 0, 1, 0,
                            ZPoly{}, c->dint + 0, i));
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_expm_select<<<grid1(nn, 256), 256, 0, c->stream>>>(nn, c->dint + 0, sq[0], sq[1], U, U2);
    return launch_end(c, t);
}

static gkba_status expm_small(gkba_ctx* c, int n, const double2* hA, const double2* hB, const double2* Z,
                                double2* U, double2* U2) {
    const size_t smem = 6 * (size_t)n * n * sizeof(double2);
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    const int ctas = n <= kExpmOneN ? 1 : 8;
    auto kfn = tensor_core_path(c) ? (ctas == 1 ? k_expm_small<1, true> : k_expm_small<8, true>)
                                   : (ctas == 1 ? k_expm_small<1, false> : k_expm_small<8, false>);
    kfn<<<ctas, 256, smem, c->stream>>>(n, c->dt, hA, hB, Z, U, U2);
    return launch_end(c, t);
}

gkba_status expm_step(gkba_ctx* c, const double2* hA, const double2* hB, double2* U, double2* U2) {
    // Scaling and squaring with a degree-18 Taylor polynomial (Moler & Van Loan,
    // "Nineteen dubious ways to compute the exponential of a matrix"): with
    // ||A/2^s||_1 <= 1/2 the truncation error is below 0.5^19/19! ~ 1e-23.
    const int N = c->N;
    if (N <= kExpmSmallN) return expm_small(c, N, hA, hB, nullptr, U, U2);
    {
        auto t = launch_begin(c, K_STEP, 0.0, 0.0);
        k_expm_setup<<<1, 256, 0, c->stream>>>(N, c->dt, hA, hB, c->ex0, c->dscal + 8, c->dint + 0);
        GKBA_TRY(launch_end(c, t));
    }
    return expm_products(c, N, c->ex0, c->ex1, c->ex2, c->tmp0, c->tmp1, U, U, U2);
}

gkba_status axpy_c(gkba_ctx* c, double2* y, const double2* x, const double2* z, double a, double b,
                   int n) {
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_lincomb<<<grid1(n, 256), 256, 0, c->stream>>>(n, y, x, z, a, b);
    return launch_end(c, t);
}

gkba_status set_identity(gkba_ctx* c, double2* A, int count) {
    const long long n = (long long)c->N * c->N * count;
    if (n == 0) return GKBA_OK;
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_set_identity<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, count, A);
    return launch_end(c, t);
}

gkba_status diagnostics(gkba_ctx* c, double E_n, const double2* rho, const double2* I, double* out4) {
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_diagnostics<<<1, 256, 0, c->stream>>>(c->N, E_n, c->h, c->d, c->hhf_n, rho, I, out4);
    return launch_end(c, t);
}

// P_k = T_k rho_k for k in [k0, k0+nk), then the unit list.
// The G_u are staged in Su (free until the reduction of this batch).
gkba_status build_forms_gkba(gkba_ctx* c, int k0, int nk, int L, const double2* rho,
                             const double2* T, const double* w) {
    const int N = c->N;
    const long long NN = (long long)N * N;
    GKBA_TRY(units_from_history(c, N, k0, nk, L, c->dt, rho, T, w, c->Su, c->Mb, c->coef));
    return build_forms(c, 2 * nk, c->Su, NN, c->Mb, NN, 0);
}

// Units of history points k0 .. k0+nk-1 of one system (history of L points,
// trapezoid weights with dt when w is null) written to G / Gb / coef (unit
// stride N*N), with c->PQ as scratch.  Used by stacked batches of systems.
gkba_status units_from_history(gkba_ctx* c, int N, int k0, int nk, int L, double dt,
                               const double2* rho, const double2* T, const double* w, double2* G,
                               double2* Gb, double* coef) {
    const long long NN = (long long)N * N;
    double2* P = c->PQ;
    GKBA_TRY(zgemm_batched(c, K_PREP, N, 'N', 'N', make_double2(1.0, 0.0), T + k0 * NN, NN,
                           rho + k0 * NN, NN, make_double2(0.0, 0.0), P, NN, nk, 0));
    auto t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_gkba_units<<<grid1(nk * NN, 256), 256, 0, c->stream>>>(N, nk, k0, L, dt, P, T + k0 * NN, w, G, Gb, coef);
    return launch_end(c, t);
}

// I += sum_u coef[u] Y[u] over nb units of one system (N x N), two passes.
gkba_status weighted_sum_units(gkba_ctx* c, int N, int nb, const double* coef, const double2* Y,
                               double2* I) {
    const long long NN = (long long)N * N;
    const int nz = nb < kWsumRanges ? nb : kWsumRanges;
    const int per = (nb + nz - 1) / nz;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_weighted_sum_p1<<<dim3(grid1(NN, 128), nz), 128, 0, c->stream>>>((int)NN, nb, per, coef, Y,
                                                                       c->red_tmp);
    GKBA_TRY(launch_end(c, t));
    t = launch_begin(c, K_RED, 0.0, 0.0);
    launch_weighted_sum_p2(c, (int)NN, nz, I);
    return launch_end(c, t);
}

gkba_status unit_xform(gkba_ctx* c, int nb, const double2* in, double2* out, int conj, int transpose) {
    const long long n = (long long)nb * c->N * c->N;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_unit_xform<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, n, in, out, conj, transpose);
    return launch_end(c, t);
}
gkba_status unit_acc(gkba_ctx* c, int nb, double2* y, const double2* x, int transpose) {
    const long long n = (long long)nb * c->N * c->N;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_unit_acc<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, n, y, x, transpose);
    return launch_end(c, t);
}
gkba_status scale_units(gkba_ctx* c, int nb, const double* coef, const double2* Ibar, double2* Y) {
    const long long n = (long long)nb * c->N * c->N;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_scale_units<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, nb, coef, Ibar, Y);
    return launch_end(c, t);
}
gkba_status vjp_points(gkba_ctx* c, int nk, const double2* Gbar, const double2* Gbbar, double2* Pbar,
                       double2* Qbar) {
    const long long n = (long long)nk * c->N * c->N;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_vjp_points<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, nk, Gbar, Gbbar, Pbar, Qbar);
    return launch_end(c, t);
}

gkba_status add_i_diff(gkba_ctx* c, double2* y, const double2* a, const double2* b, double s) {
    const long long n = (long long)c->N * c->N;
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_add_i_diff<<<grid1(n, 256), 256, 0, c->stream>>>(n, y, a, b, s);
    return launch_end(c, t);
}
gkba_status ibar_from_kbar(gkba_ctx* c, const double2* kb, double2* Ib) {
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_ibar_from_kbar<<<grid1((long long)c->N * c->N, 256), 256, 0, c->stream>>>(c->N, kb, Ib);
    return launch_end(c, t);
}
gkba_status mean_field_adj(gkba_ctx* c, const double2* hb, double2* rb) {
    const int NN = c->N * c->N;
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_mean_field_adj<<<grid1((long long)NN * 32, 256), 256, 0, c->stream>>>(c->N, c->hfK, hb, rb);
    return launch_end(c, t);
}
gkba_status field_grad(gkba_ctx* c, const double2* hb, double* out) {
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_field_grad<<<1, 256, 0, c->stream>>>(c->N, hb, c->d, out);
    return launch_end(c, t);
}
// exp(Z) of a general complex n x n matrix into W; Z is overwritten, S: 4 n x n
// scratch matrices.
static gkba_status expm_general(gkba_ctx* c, int n, double2* Z, double2* S, double2* W) {
    if (n <= kExpmSmallN) return expm_small(c, n, nullptr, nullptr, Z, W, nullptr);
    const long long nn = (long long)n * n;
    {
        auto t = launch_begin(c, K_STEP, 0.0, 0.0);
        k_expm_setup_general<<<1, 256, 0, c->stream>>>(n, Z, S, c->dint + 0);
        GKBA_TRY(launch_end(c, t));
    }
    return expm_products(c, n, S, Z, S + nn, S + 2 * nn, S + 3 * nn, W, W, nullptr);
}
// Adjoint of U = exp(-i dt (hA + hB)/2): hA_bar, hB_bar += (i dt / 2) L_exp(X^+, Ubar).
// scratch: 6 blocks of (2N)^2 entries.
gkba_status expm_adj(gkba_ctx* c, const double2* hA, const double2* hB, const double2* Ubar,
                     double2* hA_bar, double2* hB_bar, double2* scratch) {
    const int N = c->N, M = 2 * N;
    const long long MM = (long long)M * M;
    double2 *Z = scratch, *S = scratch + MM, *W = scratch + 5 * MM;
    {
        auto t = launch_begin(c, K_STEP, 0.0, 0.0);
        k_frechet_block<<<1, 256, 0, c->stream>>>(N, c->dt, hA, hB, Ubar, Z, c->dscal + 12);
        GKBA_TRY(launch_end(c, t));
    }
    GKBA_TRY(expm_general(c, M, Z, S, W));
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_frechet_apply<<<grid1((long long)N * N, 256), 256, 0, c->stream>>>(N, c->dt, W, c->dscal + 12,
                                                                         hA_bar, hB_bar);
    return launch_end(c, t);
}

gkba_status sum_units(gkba_ctx* c, int nb, const double2* src, double2* dst) {
    const long long NN = (long long)c->N * c->N;
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_sum_units<<<grid1(NN, 256), 256, 0, c->stream>>>(NN, nb, src, dst);
    return launch_end(c, t);
}

gkba_status vbar_slot(gkba_ctx* c, int nb, const double2* Sbar, int transposeS, const double* X,
                      double* out) {
    const long long n = (long long)c->N * c->N * c->N * c->N;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_vbar_slot<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, nb, Sbar, transposeS, X, out);
    return launch_end(c, t);
}
gkba_status fold_vbar(gkba_ctx* c, const double* vslot, const double* wslot, double* vbar) {
    const long long n = (long long)c->N * c->N * c->N * c->N;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_fold_vbar<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, vslot, wslot, vbar);
    return launch_end(c, t);
}
gkba_status vbar_mean_field(gkba_ctx* c, const double2* hb, const double2* rho, double* vbar) {
    const long long n = (long long)c->N * c->N * c->N * c->N;
    auto t = launch_begin(c, K_STEP, 0.0, 0.0);
    k_vbar_mean_field<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, hb, rho, vbar);
    return launch_end(c, t);
}
gkba_status build_vomega64(gkba_ctx* c, double* out) {
    const long long n = (long long)c->N * c->N * c->N * c->N;
    auto t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_build_vomega64<<<grid1(n, 256), 256, 0, c->stream>>>(c->N, c->v, out);
    return launch_end(c, t);
}

gkba_status build_forms_fp64(gkba_ctx* c, int nb, const double2* G, const double2* Gb) {
    const long long NN = (long long)c->N * c->N;
    auto t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_forms64<<<grid1(nb * NN, 256), 256, 0, c->stream>>>(c->N, nb, G, Gb, (double*)c->formsB1,
                                                          (double*)c->formsG);
    return launch_end(c, t);
}

// G forms of stage S3 from a separate matrix A (trilinear S3(A, B, C)).
gkba_status build_forms3_fp64(gkba_ctx* c, int nb, const double2* A) {
    const long long NN = (long long)c->N * c->N;
    auto t = launch_begin(c, K_PREP, 0.0, 0.0);
    k_forms64<<<grid1(nb * NN, 256), 256, 0, c->stream>>>(c->N, nb, A, nullptr, nullptr,
                                                          (double*)c->formsG3);
    return launch_end(c, t);
}

gkba_status reduce_partials_launch(gkba_ctx* c, int nb, int nz, long long zstride, long long Rld,
                                   const void* part, bool fp32, double2* S) {
    const long long NN = (long long)c->N * c->N;
    const int nzc = nz < kReduceSplit ? nz : kReduceSplit;
    const int zper = (nz + nzc - 1) / nzc;
    const int Np = tensor_core_path(c) ? c->Np : c->N;
    dim3 g1(grid1(nb * NN, 256), nzc);
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    if (fp32)
        k_reduce_partials_p1<float><<<g1, 256, 0, c->stream>>>(c->N, Np, nb, nz, zper, zstride, Rld,
                                                               (const float*)part, c->red_tmp);
    else
        k_reduce_partials_p1<double><<<g1, 256, 0, c->stream>>>(c->N, Np, nb, nz, zper, zstride,
                                                                Rld, (const double*)part, c->red_tmp);
    GKBA_TRY(launch_end(c, t));
    t = launch_begin(c, K_RED, 0.0, 0.0);
    k_reduce_partials_p2<<<grid1(nb * NN, 256), 256, 0, c->stream>>>(nb * NN, nzc, c->red_tmp, S);
    return launch_end(c, t);
}

// Y_u = S_u Gb_u, I_acc += sum_u coef_u Y_u (fixed order).  When S_out is
// non-null the S_u are copied out instead (gkba_sigma).
gkba_status reduce_batch(gkba_ctx* c, int nb, double2* I_acc, double2* S_out) {
    const int N = c->N;
    const long long NN = (long long)N * N;
    if (S_out != nullptr) {
        GKBA_CUDA(c, cudaMemcpyAsync(S_out, c->Su, nb * NN * sizeof(double2),
                                     cudaMemcpyDeviceToDevice, c->stream));
        return GKBA_OK;
    }
    GKBA_TRY(zgemm_batched(c, K_RED, N, 'N', 'N', make_double2(1.0, 0.0), c->Su, NN, c->Mb, NN,
                           make_double2(0.0, 0.0), c->Yu, NN, nb, 0));
    // nz <= nb <= ub ranges of N*N entries: red_tmp holds 16 ub of them
    const int nz = nb < kWsumRanges ? nb : kWsumRanges;
    const int per = (nb + nz - 1) / nz;
    auto t = launch_begin(c, K_RED, 0.0, 0.0);
    k_weighted_sum_p1<<<dim3(grid1(NN, 128), nz), 128, 0, c->stream>>>((int)NN, nb, per, c->coef,
                                                                       c->Yu, c->red_tmp);
    GKBA_TRY(launch_end(c, t));
    t = launch_begin(c, K_RED, 0.0, 0.0);
    launch_weighted_sum_p2(c, (int)NN, nz, I_acc);
    return launch_end(c, t);
}

// FP64 contraction of one batch (units 0..nb-1 with forms built):
//   S1  X1[j][r][m][c][q] = sum_s wS[j][m][q][s] B1[(c,r)][s]
//   S2  X2[j][r][p][c'][m] = sum_(c,q) X1[(j,r,m)][(c,q)] Gr[(c',p)][(c,q)]
//   S3  X3[c'][j][n][r][p] = sum_(c,m) X2[(j,r,p)][(c,m)] Gr[(c',n)][(c,m)]
//   S4  D[(u,c,j)][i] = sum_(n,r,p) X3[u][(c,j)][(n,r,p)] vK[i][(n,r,p)], split-K
// i.e. W1 = w x_s Gb, W2 = G x_q W1, W3 = G x_m W2, Sigma = v . W3.
// Stages S1-S3 of the FP64 chain into X13 = X3[u][c'][j][n][r][p], with A1
// the stage-S1 operand (w in the [j][m][q][s] layout, or any tensor in it).
// m3 / sOz3, when given, replace the output scatter of S3 (rows (j, r, p),
// columns (c', n), unit offset sOz3).
gkba_status fp64_chain_x3(gkba_ctx* c, int nb, const double* A1, const StageMap* m3,
                          long long sOz3) {
    const int N = c->N;
    const long long N2 = (long long)N * N, N3 = N2 * N, N4 = N3 * N;
    double* X13 = (double*)c->X13;
    double* X2 = (double*)c->X2;
    const double fl_cr = 4.0 * (double)N4 * N;   // complex x real stage, per unit
    const double fl_cc = 8.0 * (double)N4 * N;   // complex x complex stage, per unit
    {
        StageMap m{2 * N3, 2 * N, 1, N, 2 * N2, N, N, N};
        GKBA_TRY(gemm64_stage(c, K_W1, A1, N, 0, (const double*)c->formsB1, N, 2 * N2, X13,
                              2 * N4, (int)N3, 2 * N, N, nb, m, fl_cr * nb,
                              8.0 * (N4 + 2 * N4 * nb)));
    }
    {
        StageMap m{2 * N3, 2 * N2, 1, N, 2 * N, N, N, N};
        GKBA_TRY(gemm64_stage(c, K_W2, X13, 2 * N, 2 * N4, (const double*)c->formsG, 2 * N, 4 * N2,
                              X2, 2 * N4, (int)N3, 2 * N, 2 * N, nb, m, fl_cc * nb,
                              8.0 * 4 * N4 * nb));
    }
    {
        const StageMap m = m3 ? *m3 : StageMap{N3, N, 1, N4, N2, N, N, N};
        GKBA_TRY(gemm64_stage(c, K_W3, X2, 2 * N, 2 * N4,
                              (const double*)(c->sep_A ? c->formsG3 : c->formsG), 2 * N, 4 * N2,
                              X13, m3 ? sOz3 : 2 * N4, (int)N3, 2 * N, 2 * N, nb, m,
                              fl_cc * nb, 8.0 * 4 * N4 * nb));
    }
    return GKBA_OK;
}

// Stage S4, D[(u,c,j)][i], split over K, and the reduction of its partial sums.
gkba_status fp64_final(gkba_ctx* c, int nb) {
    const int N = c->N;
    const long long N2 = (long long)N * N, N3 = N2 * N, N4 = N3 * N;
    const double* X13 = (const double*)c->X13;
    const double fl = 4.0 * (double)N4 * N * nb, by = 8.0 * (2 * N4 * nb + N4);
    const long long R = 2LL * N * nb;
    const StageMap m{0, 0, 1, 0, R, (int)R, 1, N};
    const int nz = oz_items(N3);
    if ((size_t)(8 * N * R * nz) > c->part_bytes) return fail(c, GKBA_ESTATE, "partial sums of %d units do not fit", nb);
    GKBA_TRY(oz_gemm(c, K_FIN, X13, N3, 0, c->vK64, N3, 0, c->vKimg, 1, N, N3, (double*)c->part, 0, (int)R, 1, nz, N * R, m, fl, by));
    return reduce_partials_launch(c, nb, nz, N * R, R, c->part, false, c->Su);
}

gkba_status contract_batch_fp64(gkba_ctx* c, int nb) {
    GKBA_TRY(fp64_chain_x3(c, nb, c->wS64));
    return fp64_final(c, nb);
}

// Self-energy of a structured interaction for nb units (G_u, Gb_u device
// pointers with stride N*N) into c->Su; the kernels write c->PQ (free at this
// point of a batch) because G may alias c->Su.
gkba_status contract_structured(gkba_ctx* c, int nb, const double2* G, const double2* Gb) {
    const int N = c->N;
    const long long NN = (long long)N * N;
    const double n = N;
    if (c->kind == GKBA_V_DIAGONAL) {
        auto t = launch_begin(c, K_W1, 6.0 * n * n * nb, 48.0 * n * n * nb);
        k_sigma_diag<<<grid1(nb * NN, 256), 256, 0, c->stream>>>(N, nb, c->vm, G, Gb, c->PQ);
        GKBA_TRY(launch_end(c, t));
    } else if (N <= kSymmSmallN) {
        auto t = launch_begin(c, K_W1, 8.0 * n * n * n * n * nb, 48.0 * n * n * nb);
        const int upb = symm_units(N);
        k_sigma_symm_small<<<(nb + upb - 1) / upb, kSymmThreads, symm_smem(N), c->stream>>>(N, nb, upb, c->vm, G, Gb, c->PQ);
        GKBA_TRY(launch_end(c, t));
    } else {
        const int bs = N >= 128 ? 128 : ((N + 31) / 32) * 32;
        auto t = launch_begin(c, K_W1, 8.0 * n * n * n * n * nb, 48.0 * n * n * nb);
        k_sigma_symm<<<dim3(N, nb), bs, N * sizeof(double2), c->stream>>>(N, c->vm, G, Gb, c->PQ);
        GKBA_TRY(launch_end(c, t));
    }
    GKBA_CUDA(c, cudaMemcpyAsync(c->Su, c->PQ, nb * NN * sizeof(double2), cudaMemcpyDeviceToDevice,
                                 c->stream));
    return GKBA_OK;
}

}  // namespace gkba

namespace gkba {

// ---------------------------------------------------------------------------
// Allocation-free FP64 self-energy (gkba_sigma_noalloc, include/gkba.h).
//
// For callers that cannot allocate device memory (code that runs while a
// CUDA graph is being captured, inside a host framework that owns every
// allocation, or under a fixed memory budget), this entry point evaluates the
// same FP64 contraction as gkba_sigma without a context and without any
// allocation: its scratch is the file-scope array below, which every GPU that
// loads the library holds until the process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocScratchBytes = (size_t)32 << 20;  // 32 MiB per device
constexpr int kNoAllocMaxN = 24;
constexpr int kNoAllocMaxDevices = 64;

__device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of g_noalloc_scratch per device ordinal (null until set up).
void* g_noalloc_addr[kNoAllocMaxDevices] = {};
std::mutex g_noalloc_mu;

gkba_status noalloc_fail(char* err, size_t err_len, gkba_status st, const char* fmt, ...) {
    if (err != nullptr && err_len > 0) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(err, err_len, fmt, ap);
        va_end(ap);
    }
    return st;
}

size_t round256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

}  // namespace gkba

extern "C" gkba_status gkba_sigma_noalloc(int N, int n_units, const double* v, const double* G,
                                          const double* Gbar, double* S_out, void* cuda_stream,
                                          char* err, size_t err_len) {
    using namespace gkba;
    if (err != nullptr && err_len > 0) err[0] = '\0';
    if (N < 1 || N > kNoAllocMaxN)
        return noalloc_fail(err, err_len, GKBA_EINVAL,
                            "gkba_sigma_noalloc: N=%d outside [1, %d] (static scratch of %zu bytes)", N,
                            kNoAllocMaxN, kNoAllocScratchBytes);
    if (n_units < 0) return noalloc_fail(err, err_len, GKBA_EINVAL, "gkba_sigma_noalloc: n_units < 0");
    if (n_units == 0) return GKBA_OK;
    if (!v || !G || !Gbar || !S_out)
        return noalloc_fail(err, err_len, GKBA_EINVAL, "gkba_sigma_noalloc: NULL pointer argument");
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    int dev = 0;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess)
        return noalloc_fail(err, err_len, GKBA_ECUDA, "gkba_sigma_noalloc: cudaGetDevice: %s",
                            cudaGetErrorString(ce));
    if (dev < 0 || dev >= kNoAllocMaxDevices)
        return noalloc_fail(err, err_len, GKBA_EUNSUPPORTED, "gkba_sigma_noalloc: device %d", dev);
    void* base = nullptr;
    {
        // Set-up once per device (with that device current): the host-side
        // symbol is a stand-in, so the kernels get the device address.
        std::lock_guard<std::mutex> g(g_noalloc_mu);
        if (g_noalloc_addr[dev] == nullptr) {
            void* p = nullptr;
            ce = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (ce != cudaSuccess || p == nullptr)
                return noalloc_fail(err, err_len, GKBA_ECUDA,
                                    "gkba_sigma_noalloc: cudaGetSymbolAddress: %s",
                                    cudaGetErrorString(ce));
            g_noalloc_addr[dev] = p;
        }
        base = g_noalloc_addr[dev];
    }
    const long long n = N, NN = n * n, N3 = NN * n, N4 = N3 * n;
    const long long Kc = 8192;
    const int nz = (int)((N3 + Kc - 1) / Kc);
    // scratch layout: wS | vK | per-batch: B1 | Gr | X13 | X2 | part | red
    const size_t model_b = 2 * round256((size_t)N4 * 8);
    const size_t unit_b = round256((size_t)2 * NN * 8) + round256((size_t)4 * NN * 8) +
                          2 * round256((size_t)2 * N4 * 8) + round256((size_t)nz * n * 2 * n * 8) +
                          round256((size_t)kReduceSplit * NN * 16);
    if (model_b + unit_b > kNoAllocScratchBytes)
        return noalloc_fail(err, err_len, GKBA_EINVAL, "gkba_sigma_noalloc: N=%d does not fit", N);
    const int ub = (int)std::min<size_t>((kNoAllocScratchBytes - model_b) / unit_b, (size_t)n_units);
    char* s = (char*)base;
    double* wS = (double*)s;
    double* vK = (double*)(s + round256((size_t)N4 * 8));
    char* q = s + model_b;
    double* B1 = (double*)q;
    q += round256((size_t)2 * NN * 8 * ub);
    double* Gr = (double*)q;
    q += round256((size_t)4 * NN * 8 * ub);
    double* X13 = (double*)q;
    q += round256((size_t)2 * N4 * 8 * ub);
    double* X2 = (double*)q;
    q += round256((size_t)2 * N4 * 8 * ub);
    double* part = (double*)q;
    q += round256((size_t)nz * n * 2 * n * 8 * ub);
    double2* red = (double2*)q;
    q += round256((size_t)kReduceSplit * NN * 16 * ub);
    if ((size_t)(q - s) > kNoAllocScratchBytes)
        return noalloc_fail(err, err_len, GKBA_EINVAL, "gkba_sigma_noalloc: scratch layout overflow");

    // An error pending from earlier, unrelated work is reported as such and
    // left in place for its owner; launch errors of this call are checked
    // after every group of launches, so a failed launch stops the rest.
    ce = cudaPeekAtLastError();
    if (ce != cudaSuccess)
        return noalloc_fail(err, err_len, GKBA_ECUDA,
                            "gkba_sigma_noalloc: a CUDA error is pending from earlier work: %s",
                            cudaGetErrorString(ce));
    // model operands (rebuilt on every call; every element is written)
    k_build_wS64<<<grid1(N4, 256), 256, 0, stream>>>(N, v, wS);
    k_build_vK64<<<grid1(N4, 256), 256, 0, stream>>>(N, v, vK);
    ce = cudaGetLastError();
    if (ce != cudaSuccess)
        return noalloc_fail(err, err_len, GKBA_ECUDA, "gkba_sigma_noalloc: launch failed: %s",
                            cudaGetErrorString(ce));
    const double2* Gd = (const double2*)G;
    const double2* Gbd = (const double2*)Gbar;
    double2* Sd = (double2*)S_out;
    for (int u0 = 0; u0 < n_units; u0 += ub) {
        const int nb = std::min(ub, n_units - u0);
        k_forms64<<<grid1(nb * NN, 256), 256, 0, stream>>>(N, nb, Gd + u0 * NN, Gbd + u0 * NN, B1, Gr);
        {
            StageMap m{2 * N3, 2 * n, 1, n, 2 * NN, N, N, N};
            dim3 g((2 * N + G64_BN - 1) / G64_BN, (unsigned)((N3 + G64_BM - 1) / G64_BM), nb);
            k_gemm64_stage<<<g, 256, 0, stream>>>(wS, n, 0, B1, n, 2 * NN, X13, 2 * N4, (int)N3,
                                                  2 * N, n, 0, 0, m);
        }
        {
            StageMap m{2 * N3, 2 * NN, 1, n, 2 * n, N, N, N};
            dim3 g((2 * N + G64_BN - 1) / G64_BN, (unsigned)((N3 + G64_BM - 1) / G64_BM), nb);
            k_gemm64_stage<<<g, 256, 0, stream>>>(X13, 2 * n, 2 * N4, Gr, 2 * n, 4 * NN, X2, 2 * N4,
                                                  (int)N3, 2 * N, 2 * n, 0, 0, m);
        }
        {
            StageMap m{N3, n, 1, N4, NN, N, N, N};
            dim3 g((2 * N + G64_BN - 1) / G64_BN, (unsigned)((N3 + G64_BM - 1) / G64_BM), nb);
            k_gemm64_stage<<<g, 256, 0, stream>>>(X2, 2 * n, 2 * N4, Gr, 2 * n, 4 * NN, X13, 2 * N4,
                                                  (int)N3, 2 * N, 2 * n, 0, 0, m);
        }
        const long long R = 2LL * n * nb;
        {
            StageMap m{0, 0, 1, 0, R, (int)R, 1, N};
            dim3 g((N + G64_BN - 1) / G64_BN, (unsigned)((R + G64_BM - 1) / G64_BM), nz);
            k_gemm64_stage<<<g, 256, 0, stream>>>(X13, N3, 0, vK, N3, 0, part, n * R, (int)R, N, N3,
                                                  1, Kc, m);
        }
        const int nzc = nz < kReduceSplit ? nz : kReduceSplit;
        const int zper = (nz + nzc - 1) / nzc;
        dim3 g1(grid1(nb * NN, 256), nzc);
        k_reduce_partials_p1<double><<<g1, 256, 0, stream>>>(N, N, nb, nz, zper, n * R, R, part, red);
        k_reduce_partials_p2<<<grid1(nb * NN, 256), 256, 0, stream>>>(nb * NN, nzc, red, Sd + u0 * NN);
        ce = cudaGetLastError();
        if (ce != cudaSuccess)
            return noalloc_fail(err, err_len, GKBA_ECUDA, "gkba_sigma_noalloc: launch failed: %s",
                                cudaGetErrorString(ce));
    }
    return GKBA_OK;
}

