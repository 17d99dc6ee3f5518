// k_tcgemm.cu -- the same-spin products of the string-blocked expectation (variant 4)
// on the tensor cores: tcgen05.mma kind::f16 on bf16 operands with every float32 value
// split into three bf16 pieces (x = x1 + x2 + x3, each the rest of the previous
// rounded to bf16), six products x1 y1 + x1 y2 + x2 y1 + x1 y3 + x2 y2 + x3 y1 (the
// dropped terms are below 2^-24 of a product) accumulated in float32 in tensor memory:
// float32-level accuracy at the bf16 tensor rate.
//
// For plane p (re / im) one output tile, 128 alpha strings a (M) x kTcN beta strings b
// (N), accumulates both products in the same tensor-memory tile:
//   G[p][b][a] = sum_a' Ma[a][a'] X[p][b][a']          (K = D_alpha)
//              + sum_b' Xt[p][a][b'] Mb[b][b']          (K = D_beta)
// (sides = 2: one of the two, G of each side in planes of its own).
// (Ma, Mb symmetric; Xt the transposed planes, so both operands of both products are
// K-contiguous).  Operand tiles (rows x 32 bf16 of K, 64-byte rows) are moved by TMA
// (cp.async.bulk.tensor, 64-byte swizzle; rows and K beyond the matrix read as zero)
// into a ring of kTcStages stages.  Warp roles: lane 0 of warp 0 issues the copies,
// lane 0 of warp 1 the MMAs; a full barrier per stage counts the copied bytes, an
// empty barrier per stage is signalled by tcgen05.commit once the MMAs that read it
// are done, and a last commit releases the four warps to the epilogue (tensor memory
// -> registers -> G).  Every wait is bounded: past the limit the kernel sets *err,
// waits (bounded) for its copies and MMAs in flight, frees its tensor memory and
// returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <type_traits>

#include "sv_internal.h"
#include "sv_tc.cuh"

namespace svk {

namespace {

constexpr int kTcThreads = 128;
constexpr int kTcABytes = kTcM * kTcKb * 2;            // one piece of A in one stage
constexpr int kTcCols = 512;                           // tensor-memory columns: every accumulator

// A tile of TN beta strings.  The tensor core cuts each accumulation to float32 (towards zero), and a sum
// keeps losing bits at the rate of its largest terms; so the five small piece products have an accumulator
// of their own and the first pieces' product x1 y1 the rest, K blocks in turn: one with TN = 256,
// three with 128, seven with 64, fifteen with 32.  Relative gradient error at 24 qubits: 2.1e-6 to
// 2.8e-6 with one accumulator for all six, 0.7e-6 to 1.2e-6 with TN = 256.  Below 2^20 determinants, where the
// sparse float32 sums (variant 3) ran before, a CTA takes the alpha or the beta product alone (sides = 2: half as many
// accumulations, and twice the CTAs), tiles are at most 64 wide, and k_sigma_comb adds up with the rounding kept.
// The error of variant 5's pool gradients against the sparse sums' at 245,025 / 511,225 / 627,264 / 853,776
// determinants (24 problems each, geometric mean): 1.04 / 1.14 / 1.23 / - with tiles of 128 and 64 as they fit
// and both products in one CTA (complex, 627,264: 1.95), 0.69 / 0.87 / 0.93 / 0.97 so.
template <int TN>
struct TcTile {
    static constexpr int kMain = kTcCols / TN - 1;                      // accumulators of x1 y1
    static constexpr int kBBytes = TN * kTcKb * 2;                      // one piece of B in one stage
    static constexpr int kStageBytes = 3 * kTcABytes + 3 * kBBytes;
    static constexpr int kStages = TN == 256 ? 3 : TN == 128 ? 4 : 6;   // 3 x 72 KB, 4 x 48 KB, 6 x 36 or 30 KB
    static constexpr int kSmem = kStages * kStageBytes + 1024;          // + alignment of the ring to 1024 bytes
};

struct TcOut {
    float *G;  // [sides][P][Db][Da]
    int Da, Db;
    int planes, sides;  // sides = 2: the alpha and the beta product in CTAs (and planes) of their own
    int *err;
    uint32_t spins;  // mbarrier polls (each with a short sleep) before a wait gives up
    int stall;       // test hook: the producer issues no copy, so the MMA issuer's first wait runs out
};

// Tensor maps (innermost first): ma {K = Da, rows Da, piece}, mb {K = Db, rows Db, piece},
// x {K = Da, rows Db, plane, piece}, xt {K = Db, rows Da, plane, piece}; box {32, rows of a
// tile, 1, 1}.
template <int TN>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_same_tc(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb,
              const __grid_constant__ CUtensorMap x, const __grid_constant__ CUtensorMap xt, TcOut g) {
    constexpr int kTcN = TN, kMain = TcTile<TN>::kMain, kTcBBytes = TcTile<TN>::kBBytes,
                  kTcStageBytes = TcTile<TN>::kStageBytes, kTcStages = TcTile<TN>::kStages;
    extern __shared__ uint8_t tc_smem[];
    __shared__ __align__(8) uint64_t full[kTcStages], empty[kTcStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int s_fail;
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.x * kTcN, m0 = blockIdx.y * kTcM, side = blockIdx.z / g.planes, p = blockIdx.z - side * g.planes;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "n"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
        s_fail = 0;
        s_issued = 0;
        s_consumed = 0;
        for (int s = 0; s < kTcStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base, sbase = (smem_u32(tc_smem) + 1023u) & ~1023u;
    // K blocks first .. first + nIt of the alpha product's nA and the beta product's nB
    const int nA = (g.Da + kTcKb - 1) / kTcKb, nB = (g.Db + kTcKb - 1) / kTcKb;
    const int first = side ? nA : 0, nIt = side ? nB : g.sides == 2 ? nA : nA + nB;
    if (tid == 0) {
        // producer: K block it into stage it % kTcStages once the MMAs of block it - kTcStages are done
        int it = 0;
        for (; it < (g.stall ? 0 : nIt); ++it) {
            const int s = it % kTcStages;
            if (it >= kTcStages && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((it / kTcStages - 1) & 1), g.spins)) {
                s_fail = 1;
                break;
            }
            if (s_fail) break;
            const uint32_t st = sbase + (uint32_t)(s * kTcStageBytes), fb = smem_u32(&full[s]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "n"(kTcStageBytes)
                         : "memory");
            #pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int kb = first + it;
                if (kb < nA) {  // alpha side: A = Ma rows a, B = X[p] rows b, K = a'
                    tma_3d(st + c * kTcABytes, &ma, kb * kTcKb, m0, c, fb);
                    tma_4d(st + 3 * kTcABytes + c * kTcBBytes, &x, kb * kTcKb, n0, p, c, fb);
                } else {        // beta side: A = Xt[p] rows a, B = Mb rows b, K = b'
                    tma_4d(st + c * kTcABytes, &xt, (kb - nA) * kTcKb, m0, p, c, fb);
                    tma_3d(st + 3 * kTcABytes + c * kTcBBytes, &mb, (kb - nA) * kTcKb, n0, c, fb);
                }
            }
        }
        s_issued = it;
    } else if (tid == 32) {
        // MMA issuer: kind::f16, D float32, A and B bf16, both K-major, N = kTcN, M = kTcM
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                               ((uint32_t)(kTcM >> 4) << 24);
        int it = 0;
        for (; it < nIt; ++it) {
            const int s = it % kTcStages;
            if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((it / kTcStages) & 1), g.spins)) {
                s_fail = 1;
                break;
            }
            if (s_fail) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t base = sbase + (uint32_t)(s * kTcStageBytes);
            // (A piece, B piece) of the six products: x1 y1, x1 y2, x2 y1, x1 y3, x2 y2, x3 y1
            const int pa[6] = {0, 0, 1, 0, 1, 2}, pb[6] = {0, 1, 0, 2, 1, 0};
            #pragma unroll
            for (int t = 0; t < 6; ++t) {
                const uint32_t a = base + pa[t] * kTcABytes, b = base + 3 * kTcABytes + pb[t] * kTcBBytes;
                #pragma unroll
                for (int ks = 0; ks < kTcKb / 16; ++ks) {  // K = 16 per instruction: 32 bytes into the 64-byte rows
                    // the first into an accumulator starts it
                    const uint32_t acc = t == 0 ? (it >= kMain || ks > 0) : (it > 0 || t > 1 || ks > 0);
                    const uint32_t d = tmem + (uint32_t)((t == 0 ? it % kMain : kMain) * kTcN);
                    const uint64_t da = tc_desc(a + ks * 32), db = tc_desc(b + ks * 32);
                    asm volatile(
                        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n\t}\n" ::"r"(d),
                        "l"(da), "l"(db), "r"(idesc), "r"(acc)
                        : "memory");
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&empty[s]))
                         : "memory");
        }
        s_consumed = it;
        // the last commit: every MMA issued above is done when `done` completes
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(&done))
                     : "memory");
    }
    __syncwarp();
    bool ok = mbar_wait(smem_u32(&done), 0u, g.spins);
    if (!ok) s_fail = 1;
    __syncthreads();
    if (s_fail && tid == 0) {
        // copies issued but not consumed by the MMAs: let them land before the CTA exits
        for (int it = s_consumed; it < s_issued; ++it)
            mbar_wait(smem_u32(&full[it % kTcStages]), (uint32_t)((it / kTcStages) & 1), g.spins);
    }
    __syncthreads();
    ok = !s_fail;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        const int m = m0 + warp * 32 + lane;  // this thread's tensor-memory lane: alpha string a
        #pragma unroll 1
        for (int c = 0; c < kTcN; c += 8) {
            uint32_t v[kMain + 1][8];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c;
            #pragma unroll
            for (int x2 = 0; x2 <= kMain; ++x2)
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                             : "=r"(v[x2][0]), "=r"(v[x2][1]), "=r"(v[x2][2]), "=r"(v[x2][3]), "=r"(v[x2][4]),
                               "=r"(v[x2][5]), "=r"(v[x2][6]), "=r"(v[x2][7])
                             : "r"(taddr + (uint32_t)(x2 * kTcN))
                             : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (m < g.Da) {
                #pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int n = n0 + c + j;
                    float sum = __uint_as_float(v[kMain][j]);  // the small products first
                    #pragma unroll
                    for (int x2 = 0; x2 < kMain; ++x2)
                        if (x2 < nIt) sum += __uint_as_float(v[x2][j]);  // (started: one per K block)
                    if (n < g.Db) g.G[((size_t)blockIdx.z * g.Db + n) * g.Da + m] = sum;
                }
            }
        }
    } else if (tid == 0) {
        atomicExch(g.err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTcCols) : "memory");
}

// Three bf16 pieces of n floats (x1 = bf16(x), x2 = bf16(x - x1), x3 = bf16(x - x1 - x2)),
// at piece stride `piece`.
__device__ __forceinline__ void split3(float v, uint16_t &p1, uint16_t &p2, uint16_t &p3) {
    const __nv_bfloat16 a = __float2bfloat16_rn(v);
    const float r = v - __bfloat162float(a);
    const __nv_bfloat16 b = __float2bfloat16_rn(r);
    const __nv_bfloat16 c = __float2bfloat16_rn(r - __bfloat162float(b));
    p1 = __bfloat16_as_ushort(a);
    p2 = __bfloat16_as_ushort(b);
    p3 = __bfloat16_as_ushort(c);
}

__global__ void __launch_bounds__(256) k_split_bf16x3(const float *__restrict__ x, uint16_t *__restrict__ out,
                                                      size_t n, size_t piece) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        split3(x[i], out[i], out[piece + i], out[2 * piece + i]);
}

// Xt[c][p][a][b] = X[c][p][b][a] over 32 x 32 tiles for the three pieces c (z = 3 p + c;
// the padding columns of Xt stay zero: the buffer is zeroed when allocated).
__global__ void __launch_bounds__(256) k_transpose_pieces(const uint16_t *__restrict__ X, uint16_t *__restrict__ Xt,
                                                          int Da, int Db, int lda, int ldb, size_t px, size_t pt) {
    __shared__ uint16_t t[32][34];
    const int p = blockIdx.z / 3, c = blockIdx.z - 3 * p, a0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
    const uint16_t *Xp = X + c * px + (size_t)p * Db * lda;
    uint16_t *Xtp = Xt + c * pt + (size_t)p * Da * ldb;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int b = b0 + i, a = a0 + threadIdx.x;
        t[i][threadIdx.x] = (b < Db && a < Da) ? Xp[(size_t)b * lda + a] : (uint16_t)0;
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int a = a0 + i, b = b0 + threadIdx.x;
        if (a < Da && b < Db) Xtp[(size_t)a * ldb + b] = t[threadIdx.x][i];
    }
}

}  // namespace

// G = the two same-spin products of the planes (see above); err: a device int, set
// to 1 when a wait ran out.  M: the bf16 pieces of [Ma | Mb] (piece stride pm; Mb at
// Da lda), X: the pieces of the phased planes (stride px), Xt: room for the transposed
// pieces (stride pt), written here.  Rows padded to lda / ldb (multiples of 8); the
// pointers 16-byte aligned and the piece strides multiples of 8 elements (TMA's rules).
// spins: polls of each bounded wait; stall: the test hook of TcOut.
cudaError_t launch_same_tc(const uint16_t *M, size_t pm, const uint16_t *X, size_t px, uint16_t *Xt, size_t pt,
                           float *G, int planes, int sides, int Da, int Db, int lda, int ldb, int *err, uint32_t spins,
                           int stall, int sm_count, cudaStream_t st) {
    if (Da < 1 || Db < 1 || lda % 8 || ldb % 8 || pm % 8 || px % 8 || pt % 8 || spins < 1 || ((uintptr_t)M & 15) ||
        ((uintptr_t)X & 15) || ((uintptr_t)Xt & 15))
        return cudaErrorInvalidValue;
    k_transpose_pieces<<<dim3((Da + 31) / 32, (Db + 31) / 32, 3 * planes), dim3(32, 8), 0, st>>>(X, Xt, Da, Db, lda,
                                                                                                 ldb, px, pt);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    CUtensorMap ma, mb, mx, mt;
    const uint64_t P = (uint64_t)planes;
    const uint64_t dma[3] = {(uint64_t)Da, (uint64_t)Da, 3}, sma[2] = {(uint64_t)lda * 2, (uint64_t)pm * 2};
    const uint64_t dmb[3] = {(uint64_t)Db, (uint64_t)Db, 3}, smb[2] = {(uint64_t)ldb * 2, (uint64_t)pm * 2};
    const uint64_t dx[4] = {(uint64_t)Da, (uint64_t)Db, P, 3},
                   sx[3] = {(uint64_t)lda * 2, (uint64_t)Db * lda * 2, (uint64_t)px * 2};
    const uint64_t dt[4] = {(uint64_t)Db, (uint64_t)Da, P, 3},
                   stt[3] = {(uint64_t)ldb * 2, (uint64_t)Da * ldb * 2, (uint64_t)pt * 2};
    // the narrowest tiles of which every one has an SM, at most 64 wide with the sides apart.  In us with the
    // transposes, sides apart and together with 128: 330 strings 19 and 29, 495 23 and 35, 715 33 and 47, 792 54 and 61,
    // 924 58 and 55; sides together, 2,002 strings: 256 tiles of 128 would take two rounds
    const int tm = (Da + kTcM - 1) / kTcM;
    auto fits = [&](int n) { return (long long)((Db + n - 1) / n) * tm * planes * sides <= sm_count; };
    const uint32_t tn = sides == 2 ? (fits(32) ? 32 : 64) : fits(64) ? 64 : fits(128) ? 128 : 256;
    if (!encode_map(&ma, M, 3, dma, sma, kTcM) || !encode_map(&mb, M + (size_t)Da * lda, 3, dmb, smb, tn) ||
        !encode_map(&mx, X, 4, dx, sx, tn) || !encode_map(&mt, Xt, 4, dt, stt, kTcM))
        return cudaErrorInvalidValue;
    const TcOut g{G, Da, Db, planes, sides, err, spins, stall};
    const dim3 grid((Db + tn - 1) / tn, tm, planes * sides);
    auto launch = [&](auto tile) -> cudaError_t {
        constexpr int TN = decltype(tile)::value, smem = TcTile<TN>::kSmem;
        if ((e = allow_smem(k_same_tc<TN>, smem)) != cudaSuccess) return e;
        k_same_tc<TN><<<grid, kTcThreads, smem, st>>>(ma, mb, mx, mt, g);
        return cudaGetLastError();
    };
    if (tn == 32) return launch(std::integral_constant<int, 32>());
    if (tn == 64) return launch(std::integral_constant<int, 64>());
    if (tn == 128) return launch(std::integral_constant<int, 128>());
    return launch(std::integral_constant<int, 256>());
}

// The three bf16 pieces of n floats (piece stride `piece` elements).
cudaError_t launch_split_bf16x3(const float *x, uint16_t *out, size_t n, size_t piece, int sm_count, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    size_t grid = (n + 255) / 256;
    if (grid > (size_t)sm_count * 8) grid = (size_t)sm_count * 8;
    k_split_bf16x3<<<(unsigned)grid, 256, 0, st>>>(x, out, n, piece);
    return cudaGetLastError();
}

}  // namespace svk
