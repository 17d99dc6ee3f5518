// k_digits.cu -- sigma = (H - c) psi of real float64 states as exact integer products on the
// tensor cores (the float-float form's place in large sectors; the sums are those of
// expectation variant 5, k_abtc.cu and k_tcgemm.cu, to float64-level accuracy).
//
// Every operand is a fixed-point number of 56 bits under one power of two (that of the largest
// amplitude, of the largest element of Ma and Mb, of the largest alpha-beta table entry), cut into seven
// balanced base-256 digits:
//   x = 2^(e - 7) sum_i d_i 2^(-8 i),  -128 <= d_i <= 127,  error at most 2^(e - 56).
// A digit fits bf16's eight-bit significand, and so does d_i 2^(-8 i); a product of digits has at most 15
// bits, so float32 accumulation in tensor memory of the products of one level i + j is exact while the
// sum stays below 2^24: always for the alpha-beta products (at most 60 nonzero entries of A, 7 pairs), and
// for the same-spin products (at most 501) always in levels 0 and 1, in the others unless hundreds of
// trailing digits conspire (a random sum is 2^18).  (This is the scheme of Ootomo, Ozaki and Yokota,
// "DGEMM on integer matrix multiplication unit", 2024, with bf16 digits.)  The 28 products of levels 0 to
// 6 are formed, of the 49; level 7 adds less than 2^-51 of a largest product in a random sum of 501.  A
// level has an accumulator of its own, but in k_ab_digits 5 and 6 share one, which costs 2^-56 there (in
// the same-spin products' 1,300 accumulations it would cost 2^-49).  The accumulators are integers: they
// are added as such, so G and H hold int64 fixed-point values, and the sum over a row's 53 of them is
// exact as well.  Relative gradient error over 12 problems of 16 to 28 qubits (geometric mean) and the
// largest: 2.6e-15 and 1.9e-14, float-float sums 1.0e-14 and 2.2e-14.
//
//   k_max_word       the largest amplitude's exponent
//   k_phase_digits   digits of X = phi C, as planes [7][Db][lda] (same-spin products, TMA) and as words of
//                    two digits [Db][4][ldx] (alpha-beta products, gathers)
//   k_same_digits    G[0] = Ma X and G[1] = X Mb^T (tiles of 128 x 64; the two products side by side)
//   k_ab_digits      H[b'][j][a], the per-partner-row products of k_abtc.cu
//   k_comb_digits    sigma, the row's energy and norm
// 30 qubits (3,003 strings per spin): 39.1 ms in float-float (k_sigma_ab 22.95, k_sigma_same 16.0), 8.6 so
// (k_same_digits 2.45, k_ab_digits 5.1, the rest 1.05); 24 qubits (495) 668 and 216 us.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "sv_check.cuh"
#include "sv_ff.cuh"
#include "sv_internal.h"
#include "sv_sigma.cuh"
#include "sv_tc.cuh"

namespace svk {

namespace {

constexpr int kDg = 7;         // digits

// The seven digits of x as bf16 bits (d_i 2^(-8 i)); |x| <= 0.994 2^e.  Integer steps only: the FP64
// pipe would take a step per digit at a sixty-fourth of the rate.
__device__ __forceinline__ void digits7(double x, int e, uint32_t (&d)[kDg]) {
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    long long q = ex ? ((bits & 0xfffffffffffffll) | 0x10000000000000ll) : 0;  // (subnormal: 0)
    const int s = ex - 1075 + 55 - e;  // q 2^s in units of 2^(e - 55); s <= 2
    if (s >= 0) q <<= (s > 2 ? 2 : s);
    else q = s < -60 ? 0 : (q + (1ll << (-s - 1))) >> -s;
    if (bits < 0) q = -q;
    const unsigned long long t = (unsigned long long)q + 0x80808080808080ull;
    #pragma unroll
    for (int i = 0; i < kDg; ++i) {
        const int v = (int)((t >> (8 * (kDg - 1 - i))) & 255ull) - 128;
        d[i] = __float_as_uint((float)v * __uint_as_float((uint32_t)(127 - 8 * i) << 23)) >> 16;
    }
}

// e with |x| <= 0.994 2^e for every value, from the largest high word w (k_max_word)
__device__ __forceinline__ int word_exponent(unsigned int w) {
    const int e = (int)((w + 0x3000u) >> 20) - 1022;
    return e < -900 ? -900 : e;
}

__global__ void __launch_bounds__(kThreads) k_max_word(const double *__restrict__ C, size_t n, unsigned int *__restrict__ out) {
    unsigned int m = 0;
    for (size_t i = blockIdx.x * (size_t)kThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kThreads)
        m = max(m, (unsigned int)__double2hiint(C[i]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// Planes Xp [7][Db][ld] (piece stride px) and words Xi [Db][4][ldx] (two digits to a word, the first in
// its low half) of X = phi C (phi(a, b) = (-1)^popc(a & pp(b))).
__global__ void __launch_bounds__(kThreads) k_phase_digits(const double *__restrict__ C, const uint16_t *__restrict__ stra,
                                                           const uint16_t *__restrict__ strb, int Da, int Db, int ld,
                                                           const unsigned int *__restrict__ maxw,
                                                           uint16_t *__restrict__ Xp, size_t px,
                                                           uint32_t *__restrict__ Xi, int ldx) {
    const int e = word_exponent(*maxw);
    for (int Ib = blockIdx.x; Ib < Db; Ib += gridDim.x) {
        const uint32_t ppb = prefix_parity(strb[Ib]);
        for (int Ia = threadIdx.x; Ia < Da; Ia += kThreads) {
            const double c = C[(size_t)Ib * Da + Ia];
            uint32_t d[kDg];
            digits7(par(stra[Ia] & ppb) ? -c : c, e, d);
            #pragma unroll
            for (int i = 0; i < kDg; ++i) Xp[i * px + (size_t)Ib * ld + Ia] = (uint16_t)d[i];
            uint32_t *w = Xi + (size_t)Ib * 4 * ldx + Ia;
            w[0] = d[0] | d[1] << 16;
            w[ldx] = d[2] | d[3] << 16;
            w[2 * ldx] = d[4] | d[5] << 16;
            w[3 * ldx] = d[6];
        }
    }
}

// Xt[c][a][b] = X[c][b][a] over 32 x 32 tiles (z = c; Xt's padding columns stay zero).
__global__ void __launch_bounds__(256) k_transpose_digits(const uint16_t *__restrict__ X, uint16_t *__restrict__ Xt,
                                                          int Da, int Db, int lda, int ldb, size_t px, size_t pt) {
    __shared__ uint16_t t[32][34];
    const int a0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
    X += blockIdx.z * px;
    Xt += blockIdx.z * pt;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int b = b0 + i, a = a0 + threadIdx.x;
        t[i][threadIdx.x] = (b < Db && a < Da) ? X[(size_t)b * lda + a] : (uint16_t)0;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int a = a0 + i, b = b0 + threadIdx.x;
        if (a < Da && b < Db) Xt[(size_t)a * ldb + b] = t[threadIdx.x][i];
    }
}

// digits of n float64 values under the exponent of the word *maxw, at piece stride `piece`
__global__ void __launch_bounds__(256) k_split_digits(const double *__restrict__ x, const unsigned int *__restrict__ maxw,
                                                      uint16_t *__restrict__ out, size_t n, size_t piece) {
    const int e = word_exponent(*maxw);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t d[kDg];
        digits7(x[i], e, d);
        #pragma unroll
        for (int k = 0; k < kDg; ++k) out[k * piece + i] = (uint16_t)d[k];
    }
}

// The B table of k_abtc.cu (k_ab_table) in float64.
__global__ void __launch_bounds__(256) k_ab_table64(const double *__restrict__ eri, const double *__restrict__ Jt,
                                                    const uint16_t *__restrict__ strb, int N, int Db,
                                                    double *__restrict__ B) {
    const int row = blockIdx.x, kap = threadIdx.x, NN = N * N, Ktot = N * (N + 1) / 2;
    double v = 0.0;
    if (kap < Ktot) {
        int p = 0, q = 0;
        if (kap < N) {
            p = q = kap;
        } else {
            int pi = kap - N;
            while (pi >= N - 1 - p) { pi -= N - 1 - p; ++p; }
            q = p + 1 + pi;
        }
        if (row < NN) {
            v = eri[(size_t)(q * N + p) * NN + row];
        } else if (row < NN + Db && p != q) {
            for (uint32_t o = strb[row - NN]; o; o &= o - 1u) v += Jt[(size_t)(q * N + p) * N + __ffs(o) - 1];
        }
    }
    B[(size_t)row * 256 + kap] = v;
}

// A level's sum (digit products 2^(-8 l)) in units of 2^-s: an integer.
__device__ __forceinline__ long long level(uint32_t w, int s) { return (long long)__float2int_rn(__uint_as_float(w) * __uint_as_float((uint32_t)(127 + s) << 23)); }

// The same of a sum below 2^22 in magnitude, without a conversion (their rate is a sixteenth of an
// addition's): 1.5 2^23 more, it is its own mantissa.  Alpha-beta levels 0 to 3: at most 60 nonzero
// entries of A within the limits (N = 15, 10 electrons), four pairs, 2^14 a product: 2^21.9.
__device__ __forceinline__ int small_level(uint32_t w, int s) {
    return __float_as_int(fmaf(__uint_as_float(w), __uint_as_float((uint32_t)(127 + s) << 23), 12582912.f)) - 0x4B400000;
}

// ---------------------------------------------------------------- same-spin products

constexpr int kDsThreads = 128;
constexpr int kDsN = 64;                               // beta strings per tile: seven accumulators of 64 columns
constexpr int kGUnit = 40;                             // G in units of 2^-40: 501 products of 2^14 fit int64
constexpr int kDsABytes = kTcM * kTcKb * 2, kDsBBytes = kDsN * kTcKb * 2;
constexpr int kDsStage = kDg * (kDsABytes + kDsBBytes);  // 84 KB
constexpr int kDsStages = 2;
constexpr int kDsSmem = kDsStages * kDsStage + 1024;
static_assert(kDg * kDsN <= 512 && kDsN % 16 == 0 && kDsBBytes % 512 == 0, "accumulators, MMA shape, swizzle atoms");

struct DsOut {
    long long *G;  // [2][Db][Da]
    int Da, Db;
    int *err;
    uint32_t spins;
    int stall;  // test hook: no copy is issued
};

// Roles, barriers and bounded waits as in k_same_tc (k_tcgemm.cu).  blockIdx.z = 0: Ma X, 1: X Mb^T.
// Bound by the shared-memory reads of the operands (6 KB for 128 x 64 x 16, 48 cycles where the tensor
// core takes 32).
__global__ void __launch_bounds__(kDsThreads, 1)
    k_same_digits(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb,
                  const __grid_constant__ CUtensorMap x, const __grid_constant__ CUtensorMap xt, DsOut g) {
    extern __shared__ uint8_t ds_smem[];
    __shared__ __align__(8) uint64_t full[kDsStages], empty[kDsStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int s_fail;
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.x * kDsN, m0 = blockIdx.y * kTcM, beta = blockIdx.z;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
        s_fail = 0;
        s_issued = 0;
        s_consumed = 0;
        for (int s = 0; s < kDsStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base, sbase = (smem_u32(ds_smem) + 1023u) & ~1023u;
    const int nIt = ((beta ? g.Db : g.Da) + kTcKb - 1) / kTcKb;
    if (tid == 0) {
        int it = 0;
        for (; it < (g.stall ? 0 : nIt); ++it) {
            const int s = it % kDsStages;
            if (it >= kDsStages && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((it / kDsStages - 1) & 1), g.spins)) {
                s_fail = 1;
                break;
            }
            if (s_fail) break;
            const uint32_t st = sbase + (uint32_t)(s * kDsStage), fb = smem_u32(&full[s]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "n"(kDsStage) : "memory");
            #pragma unroll 1
            for (int c = 0; c < kDg; ++c) {
                // A = Ma rows a, B = X rows b, K = a'; or A = Xt rows a, B = Mb rows b, K = b'
                tma_3d(st + c * kDsABytes, beta ? &xt : &ma, it * kTcKb, m0, c, fb);
                tma_3d(st + kDg * kDsABytes + c * kDsBBytes, beta ? &mb : &x, it * kTcKb, n0, c, fb);
            }
        }
        s_issued = it;
    } else if (warp == 1) {
        // (the whole warp keeps the loop, so its operands are uniform; one lane issues)
        const uint32_t tm = warp_same(tmem), sb = warp_same(sbase);
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kDsN >> 3) << 17) |
                               ((uint32_t)(kTcM >> 4) << 24);
        int it = 0;
        for (; it < nIt; ++it) {
            const int s = it % kDsStages;
            const bool ready = ab_wait(smem_u32(&full[s]), (uint32_t)((it / kDsStages) & 1), g.spins);
            if (!__all_sync(0xffffffffu, ready && !s_fail)) {
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t da = tc_desc(sb + (uint32_t)(s * kDsStage)),
                           db = tc_desc(sb + (uint32_t)(s * kDsStage + kDg * kDsABytes));
            if (elect_one()) {
                #pragma unroll
                for (int l = 0; l < kDg; ++l)
                    #pragma unroll
                    for (int i = 0; i <= l; ++i)
                        #pragma unroll
                        for (int ks = 0; ks < kTcKb / 16; ++ks) {
                            // the first into an accumulator starts it
                            const uint32_t acc = (i == 0 && ks == 0) ? (uint32_t)(it > 0) : 1u;
                            // (start addresses in 16-byte units; the field does not carry: below 256 KB)
                            asm volatile(
                                "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n\t}\n" ::"r"(tm + (uint32_t)(l * kDsN)),
                                "l"(da + (uint64_t)((i * kDsABytes + ks * 32) >> 4)),
                                "l"(db + (uint64_t)(((l - i) * kDsBBytes + ks * 32) >> 4)), "r"(idesc), "r"(acc)
                                : "memory");
                        }
                ab_commit(smem_u32(&empty[s]));
            }
            __syncwarp();
        }
        s_consumed = it;
        if (elect_one()) ab_commit(smem_u32(&done));  // every MMA issued above is done when `done` completes
    }
    __syncwarp();
    bool ok = mbar_wait(smem_u32(&done), 0u, g.spins);
    if (!ok) s_fail = 1;
    __syncthreads();
    if (s_fail && tid == 0) {
        // copies issued but not consumed by the MMAs: let them land before the CTA exits
        for (int it = s_consumed; it < s_issued; ++it)
            mbar_wait(smem_u32(&full[it % kDsStages]), (uint32_t)((it / kDsStages) & 1), g.spins);
    }
    __syncthreads();
    ok = !s_fail;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        const int m = m0 + warp * 32 + lane;  // this thread's tensor-memory lane: alpha string a
        long long *G = g.G + (size_t)beta * g.Db * g.Da;
        #pragma unroll 1
        for (int c = 0; c < kDsN; c += 8) {
            uint32_t v[kDg][8];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c;
            #pragma unroll
            for (int l = 0; l < kDg; ++l)
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                             : "=r"(v[l][0]), "=r"(v[l][1]), "=r"(v[l][2]), "=r"(v[l][3]), "=r"(v[l][4]),
                               "=r"(v[l][5]), "=r"(v[l][6]), "=r"(v[l][7])
                             : "r"(taddr + (uint32_t)(l * kDsN))
                             : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (m < g.Da) {
                #pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int n = n0 + c + j;
                    long long t = 0;
                    #pragma unroll
                    for (int l = 0; l < kDg - 1; ++l) t = (t << 8) + level(v[l][j], 8 * l);
                    t += level(v[kDg - 1][j], kGUnit);  // level 6, rounded to the unit
                    if (n < g.Db) G[(size_t)n * g.Da + m] = t;
                }
            }
        }
    } else if (tid == 0) {
        atomicExch(g.err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ---------------------------------------------------------------- alpha-beta products

constexpr int kDbS = 2;                                      // stages
constexpr int kDbAcc = 6;                                    // accumulators: levels 0 to 4, and 5 with 6
constexpr int kHUnit = 43;                                   // H in units of 2^-43: 60 products of 2^14 fit int64
constexpr int kDbACols = kAbKc / 2;                          // tensor-memory columns of a digit of A
constexpr int kDbAStage = kDg * kDbACols;
constexpr int kDbABase = kDbAcc * kAbMaxN;                   // first A column, after the accumulators
constexpr int kDbPiece = kAbMaxN * kAbKc * 2;                // one digit of a K block's B: 64 rows x 16 K
constexpr int kDbStage = kDg * kDbPiece;                     // 14 KB
static_assert(kDbABase + kDbS * kDbAStage <= 512, "tensor memory: accumulators and A stages in 512 columns");

struct DbArgs {
    const uint32_t *Xi;       // [Db][4][ldx]: X = phi C, words of two digits (d0 d1, d2 d3, d4 d5, d6); entries from Da on zero
    int ldx;                  // a multiple of 4, at least Da + 1
    const uint16_t *stra, *ra;
    const uint16_t *Bp;       // digits [7][rowsB][256] of the B table
    const uint16_t *rowB;     // [Db][64]: the B-table row of each column of a partner row (k_ab_rows)
    size_t pb;
    long long *H;             // [Db][ncols][ldh]
    int ldh;
    int Da, Db, N, ncols, nK, units;
    int *err;
    uint32_t spins;
    int stall;                // test hook: the builders stage and write nothing
};

// The 28 MMAs of one K block in stage S (A from tensor memory, B from shared memory).
template <int S>
__device__ __forceinline__ void db_mma_stage(uint32_t tmem, uint64_t d0, uint32_t idesc, uint32_t first) {
    #pragma unroll
    for (int l = 0; l < kDg; ++l)
        #pragma unroll
        for (int i = 0; i <= l; ++i) {
            const uint32_t ta = tmem + (uint32_t)(kDbABase + S * kDbAStage + i * kDbACols);
            const uint64_t db = d0 + (uint64_t)((S * kDbStage + (l - i) * kDbPiece) >> 4);
            const int d = l < kDbAcc ? l : kDbAcc - 1;
            const uint32_t acc = (l < kDbAcc && i == 0) ? first ^ 1u : 1u;
            asm volatile(
                "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, q;\n\t}\n" ::"r"(tmem + (uint32_t)(d * kAbMaxN)),
                "r"(ta), "l"(db), "r"(idesc), "r"(acc)
                : "memory");
        }
}

// Units, roles and tables as in k_ab_tc (k_abtc.cu); a builder warp gathers one word (two digits) of its
// rows' 16 entries of a K block and stores them to tensor memory in one instruction.  One set of
// accumulators (six of 64 columns): a unit's drain and the next one's products take turns.  Bound by the
// issue and execution of the MMAs (28 to a K block; one of 128 x 64 x 16 alone takes 46 cycles, not 32) and
// the hand-overs between the roles: at 30 qubits 5.7 ms with a lone thread in the issue loop, 5.1 with the
// whole warp in it (its operands are then uniform registers); without the drain 1.1 ms less, without the
// gathers or the B copies 0.1 less.
__global__ void __launch_bounds__(kAbThreadsTc, 1) k_ab_digits(DbArgs g) {
    extern __shared__ uint8_t db_smem[];
    __shared__ __align__(8) uint64_t full[kDbS], empty[kDbS], accf, acce, done;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int s_fail;
    __shared__ uint8_t s_kp[kAbMaxK], s_kq[kAbMaxK];
    const uint32_t raw = su32(db_smem), sbase = (raw + 1023u) & ~1023u;
    uint8_t *ring = db_smem + (sbase - raw);
    const int xstride = 4 * g.ldx;                                     // words per row buffer
    uint32_t *xrow = reinterpret_cast<uint32_t *>(ring + kDbS * kDbStage);   // [2][4][ldx]
    uint16_t *tbl = reinterpret_cast<uint16_t *>(xrow + 2 * (size_t)xstride);  // [128][tstride]
    const int tid = threadIdx.x, warp = tid >> 5;
    const int N = g.N, tstride = ab_tstride(g.nK), Ktot = N * (N + 1) / 2;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(su32(&tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == kAbBuild) {
        s_fail = 0;
        for (int s = 0; s < kDbS; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&full[s])), "n"(kAbBuild / 32) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&empty[s])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&accf)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&acce)), "n"(kAbEpi) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int k = tid; k < kAbMaxK; k += kAbThreadsTc) {  // kappa -> (p, q)
        int p = 0, q = 0;
        if (k < N) {
            p = q = k;
        } else if (k < Ktot) {
            int pi = k - N;
            while (pi >= N - 1 - p) { pi -= N - 1 - p; ++p; }
            q = p + 1 + pi;
        }
        s_kp[k] = (uint8_t)p;
        s_kq[k] = (uint8_t)q;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;

    if (warp < kAbBuild / 32 && g.stall) {
        // test hook: no copy, no tensor-memory store, no arrival
    } else if (warp < kAbBuild / 32) {
        // ------------------------------------------------------------ builders
        const int r = tid & (kAbM - 1), hf = tid >> 7;  // tile row; which word (two digits)
        auto stage_row = [&](int row, int buf) {
            const uint4 *src = reinterpret_cast<const uint4 *>(g.Xi + (size_t)row * xstride);
            uint4 *dst = reinterpret_cast<uint4 *>(xrow + (size_t)buf * xstride);
            for (int i = tid; i < g.ldx; i += kAbBuild)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(su32(dst + i)), "l"(src + i) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        int cur_tile = -1, it = 0, gch = 0;
        // this thread's B copies: entry i = (digit, row, core column)
        constexpr int kCopies = 2, kSet = kDg * kAbMaxN * 2;
        static_assert(kSet <= kCopies * kAbBuild, "two copies a thread");
        const uint16_t *bsrc[kCopies];
        int brow[kCopies];
        auto row_of = [&](int u, int k) {
            const int i = tid + k * kAbBuild;
            return i < kSet ? (int)g.rowB[(size_t)(u % g.Db) * kAbMaxN + ((i % (kAbMaxN * 2)) >> 1)] : 0;
        };
        #pragma unroll
        for (int k = 0; k < kCopies; ++k) brow[k] = row_of((int)blockIdx.x, k);
        stage_row((int)blockIdx.x % g.Db, 0);
        for (int u = blockIdx.x; u < g.units; u += gridDim.x, ++it) {
            const int atile = u / g.Db, buf = it & 1;
            asm volatile("cp.async.wait_all;" ::: "memory");
            // this unit's row has landed; every builder is done with the previous unit
            if (builders_any(tid == 0 && s_fail)) break;
            const int un = u + (int)gridDim.x;
            if (un < g.units) stage_row(un % g.Db, buf ^ 1);
            if (atile != cur_tile) {
                // the tile's table: per row and kappa the byte offset of the partner's word in its plane (that
                // of word Da, a zero, where the entry is zero) | sign << 15
                cur_tile = atile;
                const int Ia = atile * kAbM + r;
                const bool valid = Ia < g.Da;
                const uint32_t a = valid ? g.stra[Ia] : 0u;
                const int part = tstride / (kAbBuild / kAbM);
                for (int k = hf * part; k < (hf + 1) * part; ++k) {
                    uint32_t e = 4u * (uint32_t)g.Da;
                    if (valid && k < Ktot) {
                        const int p = s_kp[k], q = s_kq[k];
                        if (p == q) {
                            if ((a >> p) & 1u) e = 4u * (uint32_t)Ia;
                        } else if (((a >> p) ^ (a >> q)) & 1u) {
                            const uint32_t ap = a ^ (1u << p) ^ (1u << q);
                            e = 4u * (uint32_t)g.ra[ap] | ((uint32_t)ab_par(a & ab_between(p, q)) << 15);
                        }
                    }
                    tbl[r * tstride + k] = (uint16_t)e;
                }
                builders_sync();
            }
            #pragma unroll
            for (int k = 0; k < kCopies; ++k) {
                const int i = tid + k * kAbBuild, piece = i / (kAbMaxN * 2);
                bsrc[k] = g.Bp + (size_t)piece * g.pb + (size_t)brow[k] * 256 + (i & 1) * 8;
                if (un < g.units) brow[k] = row_of(un, k);
            }
            const uint8_t *xr = reinterpret_cast<const uint8_t *>(xrow + (size_t)buf * xstride + hf * g.ldx);
            const uint16_t *trow = tbl + r * tstride;
            uint4 bv[kCopies];
            auto load_b = [&](int c) {
                #pragma unroll
                for (int k = 0; k < kCopies; ++k)
                    if (tid + k * kAbBuild < kSet) bv[k] = *reinterpret_cast<const uint4 *>(bsrc[k] + c * kAbKc);
            };
            load_b(0);
            // this thread's word of the row's 16 entries of a K block, and their table entries (two to a word)
            uint32_t w[kAbKc], tv[kAbKc / 2];
            auto gather = [&](int c) {
                #pragma unroll
                for (int k = 0; k < kAbKc / 4; ++k) {
                    const uint2 t = *reinterpret_cast<const uint2 *>(trow + c * kAbKc + 4 * k);
                    tv[2 * k] = t.x;
                    tv[2 * k + 1] = t.y;
                }
                #pragma unroll
                for (int k = 0; k < kAbKc; ++k) {
                    const uint32_t e = ((k & 1) ? tv[k >> 1] >> 16 : tv[k >> 1]) & 0x7FFFu;
                    // checked build: an offset past the plane reads its zero word
                    w[k] = *reinterpret_cast<const uint32_t *>(
                        xr + (SV_IN_RANGE(e, 4u * (uint32_t)g.ldx, kChkGather) ? e : 4u * (uint32_t)g.Da));
                }
            };
            gather(0);
            for (int c = 0; c < g.nK; ++c, ++gch) {
                const int s = gch % kDbS;
                // the stage is free once the MMAs of K block gch - kDbS are done
                if (gch >= kDbS && !s_fail && !ab_wait(su32(&empty[s]), (uint32_t)(((gch / kDbS) - 1) & 1), g.spins))
                    s_fail = 1;
                uint8_t *st = ring + s * kDbStage;
                __syncwarp();
                // A: this thread's row (its tensor-memory lane), the 8 columns of each of its two digits (the last
                // word has one), in one store; an entry's sign flips its half of a column
                {
                    uint32_t v[kAbKc];
                    #pragma unroll
                    for (int k = 0; k < kAbKc / 2; ++k) {
                        const uint32_t flip = tv[k] & 0x80008000u;
                        v[k] = __byte_perm(w[2 * k], w[2 * k + 1], 0x5410u) ^ flip;
                        v[8 + k] = __byte_perm(w[2 * k], w[2 * k + 1], 0x7632u) ^ flip;
                    }
                    const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) +
                                        (uint32_t)(kDbABase + s * kDbAStage + hf * 2 * kDbACols);
                    if (hf < 3)
                        asm volatile(
                            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                            "%13, %14, %15, %16};" ::"r"(ta),
                            "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
                            "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
                            : "memory");
                    else
                        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(ta),
                                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                                     : "memory");
                }
                #pragma unroll
                for (int k = 0; k < kCopies; ++k) {
                    const int i = tid + k * kAbBuild, rem = i % (kAbMaxN * 2);
                    if (i < kSet)
                        *reinterpret_cast<uint4 *>(st + (i / (kAbMaxN * 2)) * kDbPiece + ab_off(rem >> 1, rem & 1)) = bv[k];
                }
                if (c + 1 < g.nK) {  // in flight over the waits below and the next block's
                    load_b(c + 1);
                    gather(c + 1);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // B, for the MMAs' reads
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");   // A written
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if ((tid & 31) == 0) ab_arrive(su32(&full[s]));  // one arrival a warp
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (tid >= kAbBuild + 32) {
        // ------------------------------------------------------------ epilogue warps
        const int quarter = warp & 3, r = quarter * 32 + (tid & 31), eh = (warp - kAbBuild / 32 - 1) >> 2;
        int it = 0;
        for (int u = blockIdx.x; u < g.units; u += gridDim.x, ++it) {
            const int atile = u / g.Db, bp = u - atile * g.Db, ia = atile * kAbM + r;
            bool bad = false;
            if (tid == kAbBuild + 32) {
                if (!ab_wait(su32(&accf), (uint32_t)(it & 1), g.spins)) s_fail = 1;
                bad = s_fail != 0;
            }
            if (epi_any(bad)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            long long *Hp = g.H + (size_t)bp * g.ncols * g.ldh + ia;
            for (int c = 8 * eh; c < g.ncols; c += 16) {
                uint32_t v[kDbAcc][8];
                #pragma unroll
                for (int l = 0; l < kDbAcc; ++l)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                                 : "=r"(v[l][0]), "=r"(v[l][1]), "=r"(v[l][2]), "=r"(v[l][3]), "=r"(v[l][4]),
                                   "=r"(v[l][5]), "=r"(v[l][6]), "=r"(v[l][7])
                                 : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(l * kAbMaxN + c))
                                 : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (ia < g.Da) {
                    #pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int t01 = small_level(v[0][j], 0) * 256 + small_level(v[1][j], 8),
                                  t23 = small_level(v[2][j], 16) * 256 + small_level(v[3][j], 24);
                        long long t = (long long)t01 * 65536 + t23;
                        t = t * 256 + level(v[4][j], 32);
                        t = (t << (kHUnit - 32)) + level(v[5][j], kHUnit);  // rounded to the unit
                        if (c + j < g.ncols) Hp[(size_t)(c + j) * g.ldh] = t;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            ab_arrive(su32(&acce));
        }
    } else if (warp == kAbBuild / 32) {
        // ------------------------------------------------------------ MMA issuer
        // (the whole warp keeps the loop, so its operands are uniform; one lane issues)
        const uint32_t nn = (uint32_t)((g.ncols + 15) / 16 * 16);  // columns, in the MMA's steps of 16
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((nn >> 3) << 17) | ((uint32_t)(kAbM >> 4) << 24);
        const uint32_t tm = warp_same(tmem);
        const uint64_t d0 = ab_desc(warp_same(sbase));
        int gch = 0, it = 0;
        bool stop = false;
        for (int u = blockIdx.x; u < g.units && !stop; u += gridDim.x, ++it) {
            if (it >= 1 && !__all_sync(0xffffffffu, ab_wait(su32(&acce), (uint32_t)((it - 1) & 1), g.spins))) {
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int c = 0; c < g.nK; ++c, ++gch) {
                const int s = gch % kDbS;
                const bool ready = ab_wait(su32(&full[s]), (uint32_t)((gch / kDbS) & 1), g.spins);
                if (!__all_sync(0xffffffffu, ready && !s_fail)) {
                    s_fail = 1;
                    stop = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                static_assert(kDbS == 2, "one case per stage");
                if (elect_one()) {
                    if (s == 0) db_mma_stage<0>(tm, d0, idesc, c == 0 ? 1u : 0u);
                    else db_mma_stage<1>(tm, d0, idesc, c == 0 ? 1u : 0u);
                    ab_commit(su32(&empty[s]));
                    if (c + 1 == g.nK) ab_commit(su32(&accf));
                }
                __syncwarp();
            }
        }
        if (elect_one()) ab_commit(su32(&done));  // every MMA issued above has completed when `done` does
    }
    __syncwarp();
    const bool ok = ab_wait(su32(&done), 0u, g.spins);
    if (!ok) s_fail = 1;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(g.err, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

constexpr size_t kDbSmemCap = 227 * 1024 - 1024;  // dynamic; the static part takes 352 bytes

int digits_ldx(int Da) { return Da / 4 * 4 + 4; }  // a zero word at least after the last

size_t ab_digits_smem(int Da, int N) {
    const int nK = (N * (N + 1) / 2 + kAbKc - 1) / kAbKc;
    return 1024 + kDbS * kDbStage + 2 * (size_t)digits_ldx(Da) * 16 + (size_t)kAbM * ab_tstride(nK) * 2;
}

// ---------------------------------------------------------------- the sum

// One block per row b: sigma[b][a] = d(a, b) C + phi(a, b) (2^k (G[0] + G[1]) + 2^k' (the beta excitations'
// H entries, with the signs of k_sigma_comb)), exact up to those two conversions; the row's energy and
// norm in float64.  Bound by the read of H and, a quarter of it, the FP64 pipe: sixteen entries in flight
// (kCombBatch), read past L2 (30 qubits 1.26 ms as the compiler batched them, 0.87 so).
constexpr int kCombBatch = 16;
__global__ void __launch_bounds__(kThreads) k_comb_digits(SigmaTables<double> T, const double *__restrict__ C, double *lam,
                                                          double *lamc, const uint32_t *__restrict__ sa_s,
                                                          const uint32_t *__restrict__ sb_s, int Db, SameDigits g,
                                                          double *__restrict__ partial) {
    constexpr int kMaxH = 65;
    __shared__ ff xb[16];
    __shared__ double red[2 * kThreads / 32];
    __shared__ size_t s_hoff[kMaxH];
    __shared__ uint32_t s_hneg[kMaxH];
    const int Ib = blockIdx.x, Da = T.Da, N = T.N;
    const uint32_t b = T.strb[Ib], ppb = prefix_parity(b);
    const int nb = __popc(b), ne = N - nb, nbs = nb * ne, nh = nbs + 1;
    if ((int)threadIdx.x < nbs) {
        const int i = threadIdx.x / ne, j = threadIdx.x - i * ne;
        uint32_t o = b, z = ~b & T.maskN;
        for (int k = 0; k < i; ++k) o &= o - 1u;
        for (int k = 0; k < j; ++k) z &= z - 1u;
        const int r = __ffs(o) - 1, sx = __ffs(z) - 1;
        const uint32_t bp = b ^ (1u << r) ^ (1u << sx);
        // column of (s occupied, r empty) among b''s excitations
        const int col = __popc(bp & ((1u << sx) - 1u)) * ne + __popc(~bp & T.maskN & ((1u << r) - 1u));
        s_hoff[threadIdx.x] = ((size_t)T.rb[bp] * g.ncols + col) * g.ldh;
        s_hneg[threadIdx.x] = (uint32_t)par(b & between(r, sx));
    } else if ((int)threadIdx.x == nbs) {
        s_hoff[nbs] = ((size_t)Ib * g.ncols + nbs) * g.ldh;
        s_hneg[nbs] = 0u;
    }
    if ((int)threadIdx.x < N) {
        const int k = 2 * (int)threadIdx.x;
        double sx = 0.0;
        for (uint32_t o = b; o; o &= o - 1u) {
            const int l = 2 * (__ffs(o) - 1) + 1;
            sx += T.Jp[min(k, l) * T.n + max(k, l)];
        }
        xb[threadIdx.x] = ff_from(sx);
    }
    __syncthreads();
    const double db = T.e_shift + g.dB[Ib];
    // a state with an infinity or a NaN: every result a NaN
    const unsigned int mw = g.maxw[0];
    const int ex = word_exponent(mw) - 14;
    const bool finite = (mw >> 20) != 0x7ffu;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const double sg = finite ? scalbn(1.0, ex + word_exponent(g.ham_maxw[0]) - kGUnit) : nan;
    const double sh = finite ? scalbn(1.0, ex + word_exponent(g.ham_maxw[1]) - kHUnit) : nan;
    const size_t plane = (size_t)Da * Db, off = (size_t)Ib * Da;
    double e_acc = 0.0, n_acc = 0.0;
    for (int Ia = threadIdx.x; Ia < Da; Ia += kThreads) {
        const uint32_t a = T.stra[Ia];
        long long hi = 0;            // the sum of the H entries: hi 2^32 + lo
        unsigned long long lo = 0;
        for (int j0 = 0; j0 < nh; j0 += kCombBatch) {
            long long v[kCombBatch];
            #pragma unroll
            for (int j = 0; j < kCombBatch; ++j) {
                // checked build: a term outside the plane is skipped
                const bool ok = j0 + j < nh && SV_IN_RANGE(s_hoff[j0 + j] + Ia, g.hplane, kChkPlane);
                v[j] = ok ? __ldcs(g.H + s_hoff[j0 + j] + Ia) : 0ll;
            }
            #pragma unroll
            for (int j = 0; j < kCombBatch; ++j) {
                const long long h = j0 + j < nh && s_hneg[j0 + j] ? -v[j] : v[j];
                hi += h >> 32;
                lo += (unsigned int)h;
            }
        }
        ff d = ff(0, 0);
        for (uint32_t o = a; o; o &= o - 1u) d += xb[__ffs(o) - 1];
        const double hs = fma((double)hi, 4294967296.0, (double)(long long)lo) * sh;
        double v = fma((double)g.G[off + Ia] + (double)g.G[plane + off + Ia], sg, hs);
        if (par(a & ppb)) v = -v;
        const double c0 = C[off + Ia];
        v = fma(db + g.dA[Ia] + ff_to(d), c0, v);
        e_acc = fma(c0, v, e_acc);
        n_acc = fma(c0, c0, n_acc);
        if (lam) lam[sa_s[Ia] | sb_s[Ib]] = v;
        if (lamc) lamc[off + Ia] = v;
    }
    block_sum2(e_acc, n_acc, red);
    if (threadIdx.x == 0) {
        partial[Ib] = e_acc;
        partial[Db + Ib] = n_acc;
    }
}

}  // namespace

// Whether the digit products' limits hold (real float64 states).
bool digits_fit(int Da, int Db, int nb, int N) {
    if (N > 16 || N < 1 || Da > 4096 || Db > 4096 || Da < 1 || Db < 1 || nb < 0 || nb > N) return false;
    if (nb * (N - nb) + 1 > kAbMaxN) return false;
    return ab_digits_smem(Da, N) <= kDbSmemCap;
}

// The digits of [Ma | Mb] (nm float64 values) and of the B table; B64: room for the table's float64
// values, maxw: two words (largest high words of the two).
cudaError_t launch_ham_digits(const double *M, size_t nm, uint16_t *Mp, const double *eri, const double *Jt,
                              const uint16_t *strb, int N, int Db, double *B64, uint16_t *Bp, unsigned int *maxw,
                              int sm_count, cudaStream_t st) {
    const int rows = N * N + Db + 1, grid = sm_count * 8;
    const size_t nb = (size_t)rows * 256;
    cudaError_t e = cudaMemsetAsync(maxw, 0, 2 * sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    k_max_word<<<grid, kThreads, 0, st>>>(M, nm, maxw);
    k_split_digits<<<grid, 256, 0, st>>>(M, maxw, Mp, nm, nm);
    k_ab_table64<<<rows, 256, 0, st>>>(eri, Jt, strb, N, Db, B64);
    k_max_word<<<grid, kThreads, 0, st>>>(B64, nb, maxw + 1);
    k_split_digits<<<grid, 256, 0, st>>>(B64, maxw + 1, Bp, nb, nb);
    return cudaGetLastError();
}

// sigma of the real float64 state C [Db][Da] into lam (at storage addresses) or lamc; partial:
// 2 Db doubles.  Six launches and a memset.  Operand rules as launch_same_tc's (k_tcgemm.cu).
cudaError_t launch_sigma_digits(const SigmaTables<double> &T, const double *C, double *lam, double *lamc,
                                const uint32_t *sa_s, const uint32_t *sb_s, int Db, int nb, const SameDigits &g,
                                double *partial, int sm_count, cudaStream_t st) {
    const int Da = T.Da, N = T.N;
    if (!digits_fit(Da, Db, nb, N) || g.lda % 8 || g.ldb % 8 || g.pm % 8 || g.px % 8 || g.pt % 8 || (g.pb & 7) ||
        g.spins < 1 || ((uintptr_t)g.Mp & 15) || ((uintptr_t)g.Xp & 15) || ((uintptr_t)g.Xtp & 15) ||
        ((uintptr_t)g.Xi & 15) || ((uintptr_t)g.Bp & 15))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(g.maxw, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    const size_t total = (size_t)Da * Db, want = (total + kThreads * 4 - 1) / (kThreads * 4);
    k_max_word<<<(unsigned)(want < (size_t)sm_count * 8 ? want : (size_t)sm_count * 8), kThreads, 0, st>>>(C, total, g.maxw);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int rows = Db < sm_count * 8 ? Db : sm_count * 8;
    k_phase_digits<<<rows, kThreads, 0, st>>>(C, T.stra, T.strb, Da, Db, g.lda, g.maxw, g.Xp, g.px, g.Xi,
                                              digits_ldx(Da));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (g.ev && (e = cudaEventRecord(g.ev[0], st)) != cudaSuccess) return e;
    k_transpose_digits<<<dim3((Da + 31) / 32, (Db + 31) / 32, kDg), dim3(32, 8), 0, st>>>(g.Xp, g.Xtp, Da, Db, g.lda,
                                                                                          g.ldb, g.px, g.pt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    CUtensorMap ma, mb, mx, mt;
    auto map = [&](CUtensorMap *m, const uint16_t *base, int D0, int D1, int ld, size_t piece, int rows2) {
        const uint64_t dims[3] = {(uint64_t)D0, (uint64_t)D1, (uint64_t)kDg},
                       strides[2] = {(uint64_t)ld * 2, (uint64_t)piece * 2};
        return encode_map(m, base, 3, dims, strides, (uint32_t)rows2);
    };
    if (!map(&ma, g.Mp, Da, Da, g.lda, g.pm, kTcM) || !map(&mb, g.Mp + (size_t)Da * g.lda, Db, Db, g.ldb, g.pm, kDsN) ||
        !map(&mx, g.Xp, Da, Db, g.lda, g.px, kDsN) || !map(&mt, g.Xtp, Db, Da, g.ldb, g.pt, kTcM))
        return cudaErrorInvalidValue;
    if ((e = allow_smem(k_same_digits, kDsSmem)) != cudaSuccess) return e;
    k_same_digits<<<dim3((Db + kDsN - 1) / kDsN, (Da + kTcM - 1) / kTcM, 2), kDsThreads, kDsSmem, st>>>(
        ma, mb, mx, mt, DsOut{g.G, Da, Db, g.err, g.spins, g.stall & 1});
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (g.ev && (e = cudaEventRecord(g.ev[1], st)) != cudaSuccess) return e;
    if (g.ev && (e = cudaEventRecord(g.ev[2], st)) != cudaSuccess) return e;
    DbArgs a;
    a.Xi = g.Xi; a.ldx = digits_ldx(Da); a.stra = T.stra; a.ra = T.ra; a.Bp = g.Bp; a.rowB = g.rowB; a.pb = g.pb;
    a.H = g.H; a.ldh = g.ldh; a.Da = Da; a.Db = Db; a.N = N; a.ncols = g.ncols;
    a.nK = (N * (N + 1) / 2 + kAbKc - 1) / kAbKc;
    a.units = (Da + kAbM - 1) / kAbM * Db;
    a.err = g.err; a.spins = g.spins; a.stall = (g.stall >> 1) & 1;
    const size_t sm = ab_digits_smem(Da, N);
    if ((e = allow_smem(k_ab_digits, kDbSmemCap)) != cudaSuccess) return e;
    k_ab_digits<<<a.units < sm_count ? a.units : sm_count, kAbThreadsTc, sm, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (g.ev && (e = cudaEventRecord(g.ev[3], st)) != cudaSuccess) return e;
    k_comb_digits<<<Db, kThreads, 0, st>>>(T, C, lam, lamc, sa_s, sb_s, Db, g, partial);
    return cudaGetLastError();
}

// This unit's check word (checked build), for sv_check_status.
SV_CHECK_READER(check_word_digits)

}  // namespace svk
