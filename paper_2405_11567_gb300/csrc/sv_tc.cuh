// sv_tc.cuh -- what the tensor-core kernels share (k_tcgemm.cu, k_abtc.cu, k_digits.cu): bounded
// mbarrier waits, TMA copies and their tensor maps, shared-memory matrix descriptors, the builder
// and epilogue groups of the alpha-beta kernels.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <cstdint>

namespace svk {
namespace {

// ---- same-spin products: operand tiles of rows x kTcKb by TMA, 64-byte swizzle
constexpr int kTcM = 128;                              // alpha strings per tile (tensor-memory lanes)
constexpr int kTcKb = 32;                              // K (bf16 elements, 64 bytes) per stage

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a K-major operand tile with 64-byte swizzle: start
// address, stride byte offset 512 (8 rows of 64 bytes), descriptor version 1, swizzle
// mode 4 (64-byte).  The leading byte offset is unused for swizzled K-major tiles.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, uint32_t spins) {
    for (uint32_t it = 0; it < spins; ++it) {
        if (mbar_try(mbar, parity)) return true;
        __nanosleep(32);
    }
    return false;
}

__device__ __forceinline__ void tma_3d(uint32_t dst, const CUtensorMap *map, int k, int row, int c3, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"((uint64_t)map), "r"(k), "r"(row), "r"(c3), "r"(mbar)
        : "memory");
}

__device__ __forceinline__ void tma_4d(uint32_t dst, const CUtensorMap *map, int k, int row, int p, int c,
                                       uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(dst),
        "l"((uint64_t)map), "r"(k), "r"(row), "r"(p), "r"(c), "r"(mbar)
        : "memory");
}

// cuTensorMapEncodeTiled from the driver (through the runtime's entry-point query, so
// the library links no driver library).
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = (PFN_cuTensorMapEncodeTiled_v12000)f;
    }
    return fn;
}

// A bf16 tensor map of `rank` dims (innermost first) with byte strides of dims 1.., box
// {kTcKb, rows, 1, 1}, 64-byte swizzle, zero fill.
bool encode_map(CUtensorMap *m, const void *base, int rank, const uint64_t *dims, const uint64_t *strides,
                uint32_t rows) {
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return false;
    const cuuint32_t box[4] = {(cuuint32_t)kTcKb, rows, 1, 1}, es[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base),
              (const cuuint64_t *)dims, (const cuuint64_t *)strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- alpha-beta products: operand A gathered into tensor memory by the builder warps
constexpr int kAbBuild = 512;                  // builder threads (16 warps): 4 per tile row
constexpr int kAbKpt = 4;                      // K entries of a stage per builder thread (16 / 4)
constexpr int kAbEpi = 256;                    // epilogue threads (8 warps: two per tensor-memory lane quarter)
constexpr int kAbThreadsTc = kAbBuild + 32 + kAbEpi;  // builders, the MMA warp, the epilogue warps
constexpr int kAbM = 128;                      // alpha strings per tile
constexpr int kAbKc = 16;                      // K (orbitals and orbital pairs) per stage
constexpr int kAbMaxN = 64;                    // columns per accumulator: nb (N - nb) + 1 <= 51 within the limits
constexpr int kAbMaxK = 144;                   // N (N + 1) / 2 <= 136 for N <= 16, padded to 16

__device__ __forceinline__ uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One poll: a try-wait that suspends the thread until the phase completes or at most
// kAbPollNs nanoseconds have passed (a thread waiting here wakes as soon as the phase
// completes, and takes no issue slots meanwhile).
constexpr uint32_t kAbPollNs = 64;
__device__ __forceinline__ bool ab_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity), "n"(kAbPollNs)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool ab_wait(uint32_t mbar, uint32_t parity, uint32_t spins) {
    for (uint32_t it = 0; it < spins; ++it)
        if (ab_try(mbar, parity)) return true;
    return false;
}

__device__ __forceinline__ void ab_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void ab_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void builders_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kAbBuild) : "memory"); }

// Barrier over the builder warps (named barrier 1) or the epilogue warps (2) that also
// returns, to every thread of the group, whether any of them passed `v` true: a
// decision the whole group takes the same way.
__device__ __forceinline__ bool builders_any(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(kAbBuild)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ bool epi_any(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 2, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(kAbEpi)
        : "memory");
    return r != 0;
}

// One lane of a converged warp (the same one each time).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}\n" : "=r"(p));
    return p != 0;
}
// A value that is the same in every lane, as one the compiler knows to be.
__device__ __forceinline__ uint32_t warp_same(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// Canonical no-swizzle K-major descriptor: K-adjacent core matrices 128 bytes apart,
// adjacent 8-row groups 256 bytes apart (16 K elements = two 16-byte cores per row).
__device__ __forceinline__ uint64_t ab_desc(uint32_t addr) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)(128u >> 4) << 16;
    d |= (uint64_t)(256u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// byte offset of (row r, 16-byte column kc) in a tile of 16 K
__device__ __forceinline__ uint32_t ab_off(int r, int kc) { return (uint32_t)(((r >> 3) * 2 + kc) * 128 + (r & 7) * 16); }

__device__ __forceinline__ int ab_par(uint32_t x) { return __popc(x) & 1; }

// bits strictly between i and j
__device__ __forceinline__ uint32_t ab_between(int i, int j) {
    const int lo = min(i, j), hi = max(i, j);
    return ((1u << hi) - 1u) & ~((1u << (lo + 1)) - 1u);
}


// K entries per tile row in the table (nK * 16) plus 4: an odd number of 8-byte words
// per row, so the builders' 8-byte reads of 16 consecutive rows hit distinct bank pairs.
__host__ __device__ __forceinline__ int ab_tstride(int nK) { return nK * kAbKc + 4; }

}  // namespace
}  // namespace svk
