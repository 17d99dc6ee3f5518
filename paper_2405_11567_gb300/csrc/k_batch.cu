// k_batch.cu -- many independent small problems (uneven qubit counts) in one
// persistent, graph-captured launch: reference preparation, the fermionic
// ansatz, sigma = (H - c) psi and the energy, and the adjoint sweep for the
// gradient, per instance ("Computational Details": ADAPT-VQE runs on many small
// systems; the emulator's workload for every optimiser step).
//
// Each block takes instances from a work queue (one atomicAdd per instance, no
// device-side waiting) in descending order of estimated cost, and runs the whole
// pipeline for it on a compact state: the amplitudes of the instance's
// (N_alpha, N_beta) sector in the string-row order C[rank(b)][rank(a)] (at 20
// qubits and 6 electrons 14,400 amplitudes instead of 2^20).  Every instance starts
// from a determinant and integrals, generators and angles are real, so the amplitudes
// are real numbers whatever the batch's type.  An instance whose string counts are at
// most kBatchSmax holds psi and lambda interleaved in shared memory (in a per-block
// scratch slot that stays in L2 where they do not fit), sweeps two operators to a step
// (sv_sweep.cuh) and takes sigma in the string-blocked basis; others find a
// determinant's partner by its string ranks, and their sigma element is the closed-form
// X-mask evaluation of the string-row kernel (sv_sigma.cuh).  The gradient sums are
// fixed-order, so an instance's results do not depend on which block ran it.
//
// What is the same for every angle -- string tables, pair lists, same-spin matrices --
// is built once per plan (k_batch_lists, k_batch_mats).
//
// Bound: the longest instance (14,400 determinants) in its one block: in complex amplitudes
// from L2, with a sparse sigma, config 4 took 2.49 ms a batch; its sigma was 9 million gathers
// of three shared-memory words each.
//
// An optional time budget makes every block stop taking new instances once the
// budget is spent (checked with %globaltimer before each instance); the host then
// reports SV_ERR_TIMEOUT and leaves the outputs of skipped instances as NaN.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include "sv_internal.h"
#include "sv_sigma.cuh"
#include "sv_sweep.cuh"

namespace svk {

int plan_groups(const OpDesc *ops, int n_ops, int N, int na, int nb, std::vector<uint8_t> &plans, std::vector<uint8_t> &groups,
                uint64_t *words, long long *most, long long *all);

struct BatchOp {
    uint32_t m, from, sm;  // qubit-space flip mask, "from" pattern, sign mask
    uint32_t mab;          // low 16 bits: alpha-string flip mask, high 16: beta-string flip mask
};

struct BatchInst {
    int n, N, Da, Db, L;
    uint32_t hf;                 // compact index of the reference determinant
    double shift;                // c of lambda = (H - c) psi
    double e_shift;              // E_nuc - c
    long long ops, cs;           // offsets into the op and (cos, sin) arrays
    long long eri, hm, dt, jt;   // offsets into the state-precision integral arena
    long long hd, jp;            // offsets into the float64 arena
    long long sa, sb;            // offsets into the uint32 spread arena
    long long stra, strb, ra, rb;  // offsets into the uint16 string arena
    long long out;               // E at out, gradient at out + 1 ...
    int fast;                    // 1: the string-blocked form (both string counts <= kBatchSmax)
    int na, nb;                  // electrons per spin
    // the string-blocked form
    long long lists, groups;     // offsets of its pair lists (entries) and steps
    int words, n_groups;         // their numbers
    long long ep;                // its integrals by orbital pairs, in the state-precision arena
    long long ma, mb;            // its same-spin matrices, in the matrix arena
    long long da, db;            // its one-spin diagonals, in the diagonal arena
    long long xa, xb;            // its spins' excitation tables, in the uint32 arena
    long long tgt;               // its alpha strings' partners by orbital pair, in the uint16 arena
};

// Largest string count per spin for which an instance's sigma runs from per-block
// dense same-spin matrices and excitation tables (matrices of kBatchSmax^2 values).
constexpr int kBatchSmax = 512;
// Dynamic shared memory of the launch at most (its static part, 1,280 bytes, stays below 2 KB; the
// block limit is 227 KB).
constexpr size_t kBatchSmemCap = 224 * 1024;
// Determinants of an instance that may run on a part of a block: the state and the integrals of the
// largest take less than a quarter of the shared memory.
constexpr int kBatchSmall = 2048;
constexpr int kChunk = 24;       // beta excitations whose partner amplitudes a thread holds at once

template <typename R>
struct BatchArgs {
    const BatchInst *inst;
    const int *order;
    int count;
    const BatchOp *ops;
    const Angle<R> *angles;      // per op
    const R *rarena;
    const double *darena;
    const uint32_t *u32;
    const uint16_t *u16;
    const uint2 *lists;          // the string-blocked form: pair lists, steps, same-spin matrices, diagonals
    const Group *groups;
    const R *mats;
    const double *diag;
    double *out;
    R *scratch;                  // per block: psi and lambda, Dmax each
    double *gsum;                // per block: [Lmax][warps] gradient sums
    int Dmax, Lmax;
    size_t smem;                 // dynamic shared memory of a block
    int small, teams;            // the last `small` of the order run one to a team, `teams` (1, 2, 4) to a block
    int *ctrl;                   // [0] counter of the large instances, [1] timeout flag, [2] counter of the small
    unsigned long long budget_ns;
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------- string-blocked sigma
//
// For an instance whose string counts are at most kBatchSmax, sigma is taken in the
// string-blocked basis (all alpha creators before all beta creators; amplitudes
// C~ = phi C with phi(a, b) = (-1)^popc(a & pp(b)), pp = prefix parity), where an
// alpha excitation's sign depends on the alpha string alone and a beta excitation's
// on the beta string alone:
//   sigma~[b][a] = (E_nuc - c + dA[a] + dB[b]) C~[b][a]
//                + sum_a' Ma[a][a'] C~[b][a'] + sum_b' Mb[b][b'] C~[b'][a]
//                + sum_k sum_j s_j s_k (q_j p_j | s_k r_k) C~[b'_k][a'_j]
// Ma holds the alpha singles' string-only coefficient h_qp + sum_{o in a} ((qp|oo) -
// (qo|op)) and the alpha-alpha doubles (a dense Da x Da matrix: at 20 qubits 84 of
// its 120 entries per row are nonzero), dA the alpha one-spin diagonal energy; Mb and
// dB the same for beta.  j runs over the alpha single excitations p -> q of a and,
// as "diagonal" entries p = q, over the occupied alpha orbitals; k likewise for b.
// A diagonal entry on one side and an excitation on the other gives the singles'
// dependence on the other spin's string (sum_{o in b} (qp|oo)); two diagonal entries
// give the alpha-beta part of the diagonal energy, sum (pp|qq).  With real integrals
// (qp|..) = (pq|..), so they are kept by unordered orbital pairs.  sigma = phi sigma~.
__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) / 16 * 16; }

__host__ __device__ constexpr int pair_count(int N) { return N * (N + 1) / 2; }
// Index of the unordered pair p <= q.
__host__ __device__ constexpr int pair_index(int p, int q) { return q * (q + 1) / 2 + p; }

// Index of the u-th set bit of x (u counts from 0; x has more than u set bits).
__device__ __forceinline__ int nth_bit(uint32_t x, int u) {
    for (; u > 0; --u) x &= x - 1u;
    return __ffs(x) - 1;
}

// One spin's matrix M (D x D, row = output string, zero on entry) and one-spin diagonal dS, by
// the whole block.
template <typename R>
__device__ void build_spin_mats(const SigmaTables<R> &T, int spin, int D, int ne, R *M, double *dS) {
    const uint16_t *str = spin ? T.strb : T.stra, *rk = spin ? T.rb : T.ra;
    const int N = T.N, nv = N - ne, nsg = ne * nv, npo = ne * (ne - 1) / 2, npe = nv * (nv - 1) / 2;
    const int items = nsg + npo * npe;
    for (int t = threadIdx.x; t < D * items; t += blockDim.x) {
        const int I = t / items, u = t - I * items;
        const uint32_t a = str[I], e = ~a & T.maskN, pps = prefix_parity(a);
        if (u < nsg) {  // single p -> q: own-string part
            const int p = nth_bit(a, u / nv), q = nth_bit(e, u % nv);
            const uint32_t m = (1u << p) | (1u << q), sg = (uint32_t)par(pps & m) ^ (uint32_t)(p < q);
            R v = T.hm[q * N + p];
            const R *dt = T.Dt + (q * N + p) * N;
            for (uint32_t o = a; o; o &= o - 1u) v += dt[__ffs(o) - 1];
            M[(size_t)I * D + rk[a ^ m]] = sg ? -v : v;
        } else {  // same-spin double p1 < p2 -> q1 < q2
            int io = (u - nsg) / npe, ie = (u - nsg) % npe, i1 = 0, e1 = 0;
            while (io >= ne - 1 - i1) io -= ne - 1 - i1++;
            while (ie >= nv - 1 - e1) ie -= nv - 1 - e1++;
            const int p1 = nth_bit(a, i1), p2 = nth_bit(a, i1 + 1 + io), q1 = nth_bit(e, e1), q2 = nth_bit(e, e1 + 1 + ie);
            const uint32_t m = (1u << p1) | (1u << p2) | (1u << q1) | (1u << q2);
            const uint32_t sg = (uint32_t)par(pps & m) ^ double_order_sign(p1, p2, q1, q2);
            const R v = eri4<R>(T, q1, p1, q2, p2) - eri4<R>(T, q1, p2, q2, p1);
            M[(size_t)I * D + rk[a ^ m]] = sg ? -v : v;
        }
    }
    for (int I = threadIdx.x; I < D; I += blockDim.x) {
        double d = 0.0;
        for (uint32_t o = str[I]; o; o &= o - 1u) {
            const int k = 2 * (__ffs(o) - 1) + spin;
            d += T.hdiag[k];
            for (uint32_t o2 = o & (o - 1u); o2; o2 &= o2 - 1u) d += T.Jp[k * T.n + 2 * (__ffs(o2) - 1) + spin];
        }
        dS[I] = d;
    }
}

template <typename R>
__device__ __forceinline__ SigmaTables<R> sigma_tables(const BatchArgs<R> &B, const BatchInst &I) {
    SigmaTables<R> T;
    T.sa = B.u32 + I.sa; T.sb = B.u32 + I.sb;
    T.stra = B.u16 + I.stra; T.strb = B.u16 + I.strb; T.ra = B.u16 + I.ra; T.rb = B.u16 + I.rb;
    T.eri = B.rarena + I.eri; T.hm = B.rarena + I.hm; T.Dt = B.rarena + I.dt; T.Jt = B.rarena + I.jt;
    T.hdiag = B.darena + I.hd; T.Jp = B.darena + I.jp; T.e_shift = I.e_shift;
    T.N = I.N; T.n = I.n; T.Da = I.Da; T.maskN = (1u << I.N) - 1u;
    return T;
}

// Plan: block 2 i + spin builds instance i's same-spin matrix and diagonal (mats zero on entry).
template <typename R>
__global__ void __launch_bounds__(kThreads) k_batch_mats(BatchArgs<R> B, R *mats, double *diag) {
    const BatchInst &I = B.inst[blockIdx.x >> 1];
    if (!I.fast) return;
    const int spin = blockIdx.x & 1;
    build_spin_mats<R>(sigma_tables<R>(B, I), spin, spin ? I.Db : I.Da, spin ? I.nb : I.na, mats + (spin ? I.mb : I.ma),
                       diag + (spin ? I.db : I.da));
}

// Plan: block 4 g + 2 p + spin builds the list of operator p of step g for one spin; inst_of: the
// steps' instances.
__global__ void __launch_bounds__(kThreads) k_batch_lists(const BatchInst *__restrict__ inst, const int *__restrict__ inst_of,
                                                          const GroupPlan *__restrict__ plans, const uint32_t *__restrict__ u32,
                                                          const uint16_t *__restrict__ u16, uint2 *__restrict__ lists) {
    const int k = blockIdx.x >> 2, p = (blockIdx.x >> 1) & 1, spin = blockIdx.x & 1;
    const GroupPlan &g = plans[k];
    if (p == 1 && !g.two) return;
    const BatchInst &I = inst[inst_of[k]];
    build_list(g.op[p], g.op[1 - p], g.two, spin, spin ? I.Db : I.Da, u16 + (spin ? I.strb : I.stra), u16 + (spin ? I.rb : I.ra),
               u32 + (spin ? I.sb : I.sa), lists + I.lists + g.off[p][spin], (int)g.len[p][spin], 0);
}

// Two float32 values in a register pair, and acc += a b on both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float sum2(f32x2 v) {
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
    return x + y;
}
__device__ __forceinline__ void fma2(f32x2 &acc, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }

// The threads that run one instance: the whole block, or a half or a quarter of it (small instances,
// whose steps are too short to fill a block), with a named barrier of their own.
struct Team {
    int tid, NT, id;
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(NT) : "memory"); }
};

// Shared memory of sigma: the integrals by orbital pairs, the beta excitation table, and the alpha one
// or (float32) the alpha partners by orbital pair; for float32 also, per warp, a row's integrals
// [orbital pair][kChunk], its sums [Da] and a word per lane that sums without a target go to.
__host__ __device__ constexpr size_t blocked_warp_floats(int N, int Da) { return (size_t)pair_count(N) * kChunk + (Da + 3) / 4 * 4 + 32; }
__host__ __device__ constexpr int excitation_count(int N, int ne) { return ne * (N - ne) + ne; }
template <typename R>
__host__ __device__ constexpr size_t blocked_table_bytes(int N, int na, int nb, int Da, int Db) {
    return align16(sizeof(R) * (size_t)pair_count(N) * pair_count(N)) + align16(4 * (size_t)excitation_count(N, nb) * Db) +
           (sizeof(R) == 4 ? align16(2 * (size_t)pair_count(N) * Da) : align16(4 * (size_t)excitation_count(N, na) * Da));
}

// Diagonal and same-spin part of sigma~ into own[].l: a warp takes four rows and 32 kCols columns, so
// that each word it reads serves several products; the matrices pass through shared memory, as many
// of their rows at a time as fit.
template <typename R, bool SM, int kCols>
__device__ __forceinline__ void same_spin(const BatchArgs<R> &B, const BatchInst &I, PairOf<R> *own, unsigned char *work, size_t rest,
                                          const Team &team) {
    constexpr int kRows = 4;
    const int Da = I.Da, Db = I.Db, tid = team.tid, NT = team.NT, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
    const int quads = (Db + kRows - 1) / kRows, ct = (Da + 32 * kCols - 1) / (32 * kCols), items = quads * ct;
    const double *dA = B.diag + I.da, *dB = B.diag + I.db;
    R *stage = reinterpret_cast<R *>(work);
    for (int spin = 0; spin < 2; ++spin) {
        const int D = spin ? Db : Da;
        const R *M = B.mats + (spin ? I.mb : I.ma);
        const int share = (int)min((size_t)D, rest / (sizeof(R) * (size_t)D));
        for (int j0 = 0; j0 < D; j0 += max(share, 1)) {
            const R *Mj = M + (size_t)j0 * D;
            const int n = share > 0 ? min(share, D - j0) : 1;
            if (share > 0) {
                team.sync();
                #pragma unroll 8
                for (int i = tid; i < n * D; i += NT) stage[i] = Mj[i];
                team.sync();
                Mj = stage;
            }
            for (int t = warp; t < items; t += nw) {
                const int b0 = t / ct * kRows, a0 = t % ct * 32 * kCols;
                R acc[kRows][kCols];
                int ac[kCols], br[kRows];
                #pragma unroll
                for (int r = 0; r < kRows; ++r) br[r] = min(b0 + r, Db - 1);
                #pragma unroll
                for (int m = 0; m < kCols; ++m) {
                    ac[m] = min(a0 + 32 * m + lane, Da - 1);
                    #pragma unroll
                    for (int r = 0; r < kRows; ++r) {
                        const PairOf<R> p = own[br[r] * Da + ac[m]];
                        acc[r][m] = spin == 0 && j0 == 0 ? (R)(I.e_shift + dA[ac[m]] + dB[br[r]]) * p.c : p.l;
                    }
                }
                if (spin == 0) {  // sum_j Ma[j][a] C[b][j] (Ma is symmetric: by row, a along the lanes)
                    #pragma unroll 2
                    for (int j = 0; j < n; ++j) {
                        R w[kCols];
                        #pragma unroll
                        for (int m = 0; m < kCols; ++m) w[m] = Mj[j * D + ac[m]];
                        #pragma unroll
                        for (int r = 0; r < kRows; ++r) {
                            const R c = own[br[r] * Da + j0 + j].c;
                            #pragma unroll
                            for (int m = 0; m < kCols; ++m) acc[r][m] = fma(w[m], c, acc[r][m]);
                        }
                    }
                } else {  // sum_k Mb[k][b] C[k][a]
                    #pragma unroll 2
                    for (int k = 0; k < n; ++k) {
                        R c[kCols];
                        #pragma unroll
                        for (int m = 0; m < kCols; ++m) c[m] = own[(j0 + k) * Da + ac[m]].c;
                        #pragma unroll
                        for (int r = 0; r < kRows; ++r) {
                            const R w = Mj[k * D + br[r]];
                            #pragma unroll
                            for (int m = 0; m < kCols; ++m) acc[r][m] = fma(w, c[m], acc[r][m]);
                        }
                    }
                }
                #pragma unroll
                for (int r = 0; r < kRows; ++r)
                    #pragma unroll
                    for (int m = 0; m < kCols; ++m)
                        if (b0 + r < Db && a0 + 32 * m + lane < Da) own[(b0 + r) * Da + a0 + 32 * m + lane].l = acc[r][m];
            }
        }
    }
    team.sync();
}

// sigma~ into own[].l from C~ in own[].c (own: psi and lambda interleaved), the whole block; `work`:
// `rest` bytes of shared memory beyond own.  Alpha-beta part in float32: a warp takes a row b and holds its kChunk excitations' partner amplitudes of 64 columns a'
// in registers; for every orbital pair it forms sum_k s_k (pq|sr_k) C~[b'_k][a'] (integrals broadcast
// from shared memory, packed multiply-adds) and adds it at the string that a' becomes.  That is 55
// products for the 24 that count at 20 qubits and 6 electrons, on a pipe that the three gathers of
// each of the 24 left idle.  float64: the sparse sums, bound by the FP64 pipe.
template <typename R, bool SM>
__device__ __noinline__ void sigma_blocked(const BatchArgs<R> &B, const BatchInst &I, PairOf<R> *scratch, uint32_t at, size_t rest,
                                           const Team &team) {
    extern __shared__ __align__(16) unsigned char batch_smem[];
    PairOf<R> *own = SM ? reinterpret_cast<PairOf<R> *>(batch_smem + at) : scratch;
    unsigned char *work = batch_smem + at + (SM ? align16(sizeof(PairOf<R>) * (size_t)(I.Da * I.Db)) : 0);
    const int Da = I.Da, Db = I.Db, tid = team.tid, NT = team.NT, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
    const R *ep = B.rarena + I.ep;
    const uint32_t *xa = B.u32 + I.xa, *xb = B.u32 + I.xb;
    const uint16_t *tgt = B.u16 + I.tgt;
    const int np = pair_count(I.N), nxa = excitation_count(I.N, I.na), nxb = excitation_count(I.N, I.nb);
    // diagonal and same-spin part: tiles as wide as the strings fill
    if (Da <= 32) same_spin<R, SM, 1>(B, I, own, work, rest, team);
    else if (Da <= 64) same_spin<R, SM, 2>(B, I, own, work, rest, team);
    else same_spin<R, SM, 4>(B, I, own, work, rest, team);
    const size_t tables = blocked_table_bytes<R>(I.N, I.na, I.nb, Da, Db);
    if (tables <= rest) {  // the tables beside the state
        R *e = reinterpret_cast<R *>(work);
        uint32_t *b = reinterpret_cast<uint32_t *>(work + align16(sizeof(R) * (size_t)np * np));
        uint32_t *a = b + align16(4 * (size_t)nxb * Db) / 4;
        for (int i = tid; i < np * np; i += NT) e[i] = ep[i];
        for (int i = tid; i < nxb * Db; i += NT) b[i] = xb[i];
        ep = e;
        xb = b;
        if constexpr (sizeof(R) == 4) {
            uint16_t *g = reinterpret_cast<uint16_t *>(a);
            for (int i = tid; i < np * Da; i += NT) g[i] = tgt[i];
            tgt = g;
        } else {
            for (int i = tid; i < nxa * Da; i += NT) a[i] = xa[i];
            xa = a;
        }
        work += tables;
        rest -= tables;
    }
    int warps_ab = 0;
    if (sizeof(R) == 4) {
        warps_ab = (int)min((size_t)nw, rest / (4 * blocked_warp_floats(I.N, Da)));
        if (warps_ab < (nw + 1) / 2) warps_ab = 0;  // too little shared memory: the sparse sums use every warp
    }
    team.sync();
    if constexpr (sizeof(R) == 4) {
        if (warps_ab > 0) {
            if (warp >= warps_ab) return;
            float *E = reinterpret_cast<float *>(work) + (size_t)warp * blocked_warp_floats(I.N, Da), *sum = E + (size_t)np * kChunk;
            for (int b = warp; b < Db; b += warps_ab) {
                for (int a = lane; a < Da; a += 32) sum[a] = 0.f;
                for (int k0 = 0; k0 < nxb; k0 += kChunk) {
                    // lane k: the row's k-th excitation of this chunk (past the last: the row itself, weight 0)
                    const bool is = lane < kChunk && k0 + lane < nxb;
                    const uint32_t mine = is ? xb[(k0 + lane) * Db + b] : (uint32_t)b;
                    __syncwarp();
                    for (int k = 0; k < kChunk; ++k) {
                        const uint32_t e = __shfl_sync(0xffffffffu, mine, k);
                        const float sg = k0 + k < nxb ? (((e >> 14) & 1u) ? -1.f : 1.f) : 0.f;
                        const float *col = ep + (e >> 16) * np;  // symmetric: by row
                        for (int q = lane; q < np; q += 32) E[q * kChunk + k] = sg * col[q];
                    }
                    __syncwarp();
                    for (int a0 = 0; a0 < Da; a0 += 64) {
                        f32x2 v[kChunk / 2][2];
                        #pragma unroll
                        for (int k = 0; k < kChunk; k += 2) {
                            const PairOf<float> *p0 = own + (__shfl_sync(0xffffffffu, mine, k) & 0x3FFFu) * Da,
                                                *p1 = own + (__shfl_sync(0xffffffffu, mine, k + 1) & 0x3FFFu) * Da;
                            #pragma unroll
                            for (int m = 0; m < 2; ++m) {
                                const int a = min(a0 + 32 * m + lane, Da - 1);
                                v[k / 2][m] = pack2(p0[a].c, p1[a].c);
                            }
                        }
                        // two orbital pairs at a time: their sums, then their additions one after the other (the
                        // targets of one pair are distinct); without a target: the lane's spare word, no branch
                        const int spare = (Da + 3) / 4 * 4 + lane;
                        uint32_t gn[2][2];
                        auto targets = [&](int q) {
                            #pragma unroll
                            for (int p = 0; p < 2; ++p)
                                #pragma unroll
                                for (int m = 0; m < 2; ++m) {
                                    const int a = a0 + 32 * m + lane;
                                    gn[p][m] = q + p < np && a < Da ? tgt[(q + p) * Da + a] : 0u;
                                }
                        };
                        targets(0);
                        for (int q = 0; q < np; q += 2) {
                            f32x2 t[2][2][2] = {};
                            int to[2][2];
                            uint32_t neg[2][2];
                            #pragma unroll
                            for (int p = 0; p < 2; ++p)
                                #pragma unroll
                                for (int m = 0; m < 2; ++m) {
                                    to[p][m] = gn[p][m] >> 15 ? (int)(gn[p][m] & 0x3FFFu) : spare;
                                    neg[p][m] = gn[p][m] >> 14 & 1u;
                                }
                            const ulonglong2 *er = reinterpret_cast<const ulonglong2 *>(E + q * kChunk);
                            const ulonglong2 *eq = q + 1 < np ? er + kChunk / 4 : er;
                            #pragma unroll
                            for (int k = 0; k < kChunk / 4; ++k) {
                                const ulonglong2 e = er[k], f = eq[k];
                                #pragma unroll
                                for (int m = 0; m < 2; ++m) {
                                    fma2(t[0][m][0], v[2 * k][m], e.x);
                                    fma2(t[0][m][1], v[2 * k + 1][m], e.y);
                                    fma2(t[1][m][0], v[2 * k][m], f.x);
                                    fma2(t[1][m][1], v[2 * k + 1][m], f.y);
                                }
                            }
                            targets(q + 2);
                            #pragma unroll
                            for (int p = 0; p < 2; ++p) {
                                float had[2];
                                #pragma unroll
                                for (int m = 0; m < 2; ++m) had[m] = sum[to[p][m]];
                                #pragma unroll
                                for (int m = 0; m < 2; ++m)
                                    sum[to[p][m]] = had[m] + flip(sum2(t[p][m][0]) + sum2(t[p][m][1]), neg[p][m]);
                                __syncwarp();
                            }
                        }
                    }
                }
                __syncwarp();
                for (int a = lane; a < Da; a += 32) own[b * Da + a].l += sum[a];
                __syncwarp();
            }
            return;
        }
    }
    for (int Ib = warp; Ib < Db; Ib += nw) {
        for (int Ia = lane; Ia < Da; Ia += 32) {
            R acc = 0;
            for (int k = 0; k < nxb; ++k) {
                const uint32_t eb = xb[k * Db + Ib];
                const PairOf<R> *prow = own + (size_t)(eb & 0x3FFFu) * Da;
                const R *er = ep + (eb >> 16) * np;
                R t = 0;
                #pragma unroll 4
                for (int j = 0; j < nxa; ++j) {
                    const uint32_t ea = xa[j * Da + Ia];
                    t = fma(flip(er[ea >> 16], ea >> 14 & 1u), prow[ea & 0x3FFFu].c, t);
                }
                acc += flip(t, eb >> 14 & 1u);
            }
            own[Ib * Da + Ia].l += acc;
        }
    }
}

// Sums of products for the energy and the norm.  float32: no FP64 work, and no less than its precision: a
// product is two words exactly, the sum three that pass their rounding on (about 72 bits).
template <typename R> struct DotSum;
template <> struct DotSum<float> {
    float a = 0.f, b = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        float e, f;
        two_sum(a, x, a, e);
        two_sum(b, e, b, f);
        c += f;
    }
    __device__ __forceinline__ void add(const DotSum &o) {
        add(o.a);
        add(o.b);
        add(o.c);
    }
    __device__ __forceinline__ void add_product(float x, float y) {
        const float p = x * y;
        add(p);
        add(fmaf(x, y, -p));
    }
    __device__ __forceinline__ DotSum xor_lane(int m) const {
        DotSum o;
        o.a = __shfl_xor_sync(0xffffffffu, a, m);
        o.b = __shfl_xor_sync(0xffffffffu, b, m);
        o.c = __shfl_xor_sync(0xffffffffu, c, m);
        return o;
    }
    __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};
template <> struct DotSum<double> {
    double a = 0.0;
    __device__ __forceinline__ void add(const DotSum &o) { a += o.a; }
    __device__ __forceinline__ void add_product(double x, double y) { a = fma(x, y, a); }
    __device__ __forceinline__ DotSum xor_lane(int m) const {
        DotSum o;
        o.a = __shfl_xor_sync(0xffffffffu, a, m);
        return o;
    }
    __device__ __forceinline__ double value() const { return a; }
};
// A gradient sum (GradSum::bits) as float64.
__device__ __forceinline__ double sum_value(double bits, float) {
    return (double)__int_as_float(__double2hiint(bits)) + (double)__int_as_float(__double2loint(bits));
}
__device__ __forceinline__ double sum_value(double bits, double) { return bits; }

// The string-blocked form of one instance: psi and lambda interleaved at byte `at` of the block's shared
// memory (SM) or in `scratch`, `rest` bytes of shared memory after them (from `at`).
template <typename R, bool SM>
__device__ __noinline__ void run_blocked(const BatchArgs<R> &B, const BatchInst &I, PairOf<R> *scratch, uint32_t at, size_t rest,
                                         double *red, double *gsum, const Team &team) {
    extern __shared__ __align__(16) unsigned char batch_smem[];
    PairOf<R> *own = SM ? reinterpret_cast<PairOf<R> *>(batch_smem + at) : scratch;
    unsigned char *work = batch_smem + at + (SM ? align16(sizeof(PairOf<R>) * (size_t)(I.Da * I.Db)) : 0);
    const int Da = I.Da, D = I.Da * I.Db, tid = team.tid, NT = team.NT, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
    const uint16_t *stra = B.u16 + I.stra, *strb = B.u16 + I.strb;
    const uint2 *lists = B.lists + I.lists;
    const Group *groups = B.groups + I.groups;
    const Angle<R> *angles = B.angles + I.cs;
    // the lists, steps and angles beside the state while a sweep runs: a step is shorter than a read of L2
    const size_t lw = align16(8 * (size_t)I.words), gw = align16(sizeof(Group) * (size_t)I.n_groups),
                 aw = align16(sizeof(Angle<R>) * (size_t)I.L);
    const bool staged = lw + gw + aw <= rest;
    auto stage = [&] {
        if (!staged) return;
        const uint32_t *src[3] = {(const uint32_t *)(B.lists + I.lists), (const uint32_t *)(B.groups + I.groups),
                                  (const uint32_t *)(B.angles + I.cs)};
        uint32_t *dst[3] = {(uint32_t *)work, (uint32_t *)(work + lw), (uint32_t *)(work + lw + gw)};
        const int n[3] = {2 * I.words, (int)(sizeof(Group) / 4) * I.n_groups, (int)(sizeof(Angle<R>) / 4) * I.L};
        for (int p = 0; p < 3; ++p)
            for (int i = tid; i < n[p]; i += NT) dst[p][i] = src[p][i];
        lists = (const uint2 *)dst[0];
        groups = (const Group *)dst[1];
        angles = (const Angle<R> *)dst[2];
    };
    for (int i = tid; i < D; i += NT) own[i] = PairOf<R>{(uint32_t)i == I.hf ? (R)1 : (R)0, (R)0};
    stage();
    team.sync();
    auto sync = [&](int) {
        team.sync();
        return true;
    };
    run_steps<R, false, 1>(lists, groups, angles, I.n_groups, Da, (size_t)D, tid, NT, warp, nw, 1, nullptr,
                           [&](uint32_t at) { return own[at].c; }, [&](uint32_t at, R v) { own[at].c = v; }, sync);
    team.sync();
    // phi of element (b, a), as a sign flip: the parity of the alpha string under the beta string's prefix parity
    for (int b = warp; b < I.Db; b += nw) {
        const uint32_t pb = prefix_parity(strb[b]);
        for (int a = lane; a < Da; a += 32) own[b * Da + a].c = flip(own[b * Da + a].c, parity32(stra[a] & pb));
    }
    team.sync();
    sigma_blocked<R, SM>(B, I, scratch, at, rest, team);
    team.sync();
    stage();  // sigma worked where the lists were
    DotSum<R> e, n;
    for (int b = warp; b < I.Db; b += nw) {
        const uint32_t pb = prefix_parity(strb[b]);
        for (int a = lane; a < Da; a += 32) {
            const uint32_t f = parity32(stra[a] & pb);
            const PairOf<R> p = own[b * Da + a];
            e.add_product(p.c, p.l);
            n.add_product(p.c, p.c);
            own[b * Da + a] = PairOf<R>{flip(p.c, f), flip(p.l, f)};
        }
    }
    // energy (lower half warp) and norm (upper) in one tree, then the warps in order
    DotSum<R> mine = lane < 16 ? e : n, other = lane < 16 ? n : e;
    mine.add(other.xor_lane(16));
    #pragma unroll
    for (int o = 8; o > 0; o >>= 1) mine.add(mine.xor_lane(o));
    if ((lane & 15) == 0) red[2 * warp + (lane >> 4)] = mine.value();
    team.sync();
    double se = 0.0, sn = 0.0;
    for (int w = 0; w < nw; ++w) {
        se += red[2 * w];
        sn += red[2 * w + 1];
    }
    if (tid == 0) B.out[I.out] = I.shift + se / sn;
    run_steps<R, true, 1>(lists, groups, angles, I.n_groups, Da, (size_t)D, tid, NT, warp, nw, 1, gsum,
                          [&](uint32_t at) { return own[at]; }, [&](uint32_t at, const PairOf<R> &v) { own[at] = v; }, sync);
    team.sync();
    for (int k = tid; k < I.L; k += NT) {
        double g = 0.0;
        for (int w = 0; w < nw; ++w) g += sum_value(gsum[(size_t)k * nw + w], (R)0);
        B.out[I.out + 1 + k] = 2.0 * g / sn;
    }
}

// Every instance's angles as the rotations take them, from float64 cosines and sines: the first node
// of the batch graph (the host only copies the angles).
template <typename R>
__global__ void __launch_bounds__(kThreads) k_batch_sincos(const double *__restrict__ theta, Angle<R> *__restrict__ angles,
                                                          long long n) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double sn, cn;
        sincos(theta[k], &sn, &cn);
        angles[k] = Angle<R>{(R)cn, (R)sn, (R)(cn > 0.0 ? sn / (1.0 + cn) : 2.0)};
    }
}

// The next instance of a queue (its counter at ctrl[0], entries order[first .. first + count)), or -1; every
// thread of the team gets it.
template <typename R>
__device__ __forceinline__ int take(const BatchArgs<R> &B, int *ctrl, int first, int count, unsigned long long t0, volatile int *slot,
                                    const Team &team) {
    if (team.tid == 0) {
        int next = -1;
        if (B.budget_ns && global_ns() - t0 > B.budget_ns) {
            atomicExch(&B.ctrl[1], 1);
        } else {
            const int k = atomicAdd(ctrl, 1);
            if (k < count) next = B.order[first + k];
        }
        *slot = next;
    }
    team.sync();
    const int got = *slot;
    team.sync();
    return got;
}

__device__ __forceinline__ void load_instance(BatchInst &to, const BatchInst &from, const Team &team) {
    static_assert(sizeof(BatchInst) % 4 == 0, "copied by words");
    for (int i = team.tid; i < (int)(sizeof(BatchInst) / 4); i += team.NT)
        reinterpret_cast<uint32_t *>(&to)[i] = reinterpret_cast<const uint32_t *>(&from)[i];
    team.sync();
}

template <typename R, int NT>
__global__ void __launch_bounds__(NT, 1) k_batch(BatchArgs<R> B) {
    __shared__ int s_inst[4];
    __shared__ BatchInst s_I[4];  // the instances in work (in registers they would crowd out the sums)
    __shared__ double red[2 * NT / 32];
    __shared__ unsigned long long s_t0;
    R *psi = B.scratch + (size_t)blockIdx.x * 2 * B.Dmax;
    R *lam = psi + B.Dmax;
    double *gsum = B.gsum + (size_t)blockIdx.x * B.Lmax * (NT / 32);
    if (threadIdx.x == 0) s_t0 = global_ns();
    __syncthreads();
    // the large instances, a block each, then the small ones, a team each
    const Team block = {(int)threadIdx.x, NT, 0};
    for (;;) {
        const int ii = take(B, &B.ctrl[0], 0, B.count - B.small, s_t0, &s_inst[0], block);
        if (ii < 0) break;
        load_instance(s_I[0], B.inst[ii], block);
        const BatchInst &I = s_I[0];
        const int Da = I.Da, D = I.Da * I.Db;
        if (I.fast) {
            const size_t state = align16(sizeof(PairOf<R>) * (size_t)D);
            if (state <= B.smem)
                run_blocked<R, true>(B, I, nullptr, 0, B.smem - state, red, gsum, block);
            else
                run_blocked<R, false>(B, I, reinterpret_cast<PairOf<R> *>(psi), 0, B.smem, red, gsum, block);
            __syncthreads();
            continue;
        }
        const SigmaTables<R> T = sigma_tables<R>(B, I);
        // reference determinant
        for (int i = threadIdx.x; i < D; i += blockDim.x) psi[i] = (uint32_t)i == I.hf ? (R)1 : (R)0;
        __syncthreads();
        // forward sweep
        for (int k = 0; k < I.L; ++k) {
            const BatchOp op = B.ops[I.ops + k];
            const Angle<R> ak = B.angles[I.cs + k];
            for (int i = threadIdx.x; i < D; i += blockDim.x) {
                const int Ib = i / Da, Ia = i - Ib * Da;
                const uint32_t x = T.sa[Ia] | T.sb[Ib];
                if ((x & op.m) != op.from) continue;
                const int j = (int)T.rb[T.strb[Ib] ^ (op.mab >> 16)] * Da + T.ra[T.stra[Ia] ^ (op.mab & 0xFFFFu)];
                const R ss = par(x & op.sm) ? -ak.s : ak.s;
                const R u = psi[i], v = psi[j];
                psi[i] = ak.c * u - ss * v;
                psi[j] = ak.c * v + ss * u;
            }
            __syncthreads();
        }
        // sigma and the energy
        double e_acc = 0.0, n_acc = 0.0;
        for (int i = threadIdx.x; i < D; i += blockDim.x) {
            const int Ib = i / Da, Ia = i - Ib * Da;
            const R c0 = psi[i];
            const R s = sigma_at<R>(T, psi, Ia, Ib, c0);
            lam[i] = s;
            e_acc += (double)c0 * (double)s;
            n_acc += (double)c0 * (double)c0;
        }
        block_sum2_nt<NT>(e_acc, n_acc, red);  // contains the barrier that publishes lambda
        __shared__ double s_norm;
        if (threadIdx.x == 0) {
            s_norm = n_acc;
            B.out[I.out] = I.shift + e_acc / n_acc;
        }
        __syncthreads();
        const double nrm = s_norm;
        // reverse sweep
        for (int k = I.L - 1; k >= 0; --k) {
            const BatchOp op = B.ops[I.ops + k];
            const Angle<R> ak = B.angles[I.cs + k];
            double g = 0.0;
            for (int i = threadIdx.x; i < D; i += blockDim.x) {  // every determinant, with the op's "from" test
                const int Ib = i / Da, Ia = i - Ib * Da;
                const uint32_t x = T.sa[Ia] | T.sb[Ib];
                if ((x & op.m) != op.from) continue;
                const int j = (int)T.rb[T.strb[Ib] ^ (op.mab >> 16)] * Da + T.ra[T.stra[Ia] ^ (op.mab & 0xFFFFu)];
                const bool neg = par(x & op.sm);
                const R u = psi[i], v = psi[j], lu = lam[i], lv = lam[j];
                const R t = lv * u - lu * v;
                g += (double)(neg ? -t : t);
                const R ss = neg ? -ak.s : ak.s;
                psi[i] = ak.c * u + ss * v;
                psi[j] = ak.c * v - ss * u;
                lam[i] = ak.c * lu + ss * lv;
                lam[j] = ak.c * lv - ss * lu;
            }
            const double gs = block_sum_nt<NT>(g, red);
            if (threadIdx.x == 0) B.out[I.out + 1 + k] = 2.0 * gs / nrm;
        }
        __syncthreads();
    }
    const int tn = NT / B.teams, who = threadIdx.x / tn;
    const Team team = {(int)threadIdx.x % tn, tn, 1 + who};
    const size_t share = B.smem / B.teams / 16 * 16;
    for (;;) {
        const int ii = take(B, &B.ctrl[2], B.count - B.small, B.small, s_t0, &s_inst[who], team);
        if (ii < 0) break;
        load_instance(s_I[who], B.inst[ii], team);
        const BatchInst &I = s_I[who];
        const size_t state = align16(sizeof(PairOf<R>) * (size_t)(I.Da * I.Db));  // at most a team's share (the host's choice)
        run_blocked<R, true>(B, I, nullptr, (uint32_t)(who * share), share - state, red + who * 2 * (tn / 32),
                             gsum + (size_t)who * B.Lmax * (tn / 32), team);
        team.sync();
    }
}

}  // namespace svk

using namespace svk;

namespace svk {
void set_thread_error(const std::string &m);  // sv_api.cu: the message sv_last_error(NULL) returns
}

namespace {
sv_status bfail(sv_status s, const std::string &m) {
    set_thread_error(m);
    return s;
}

}  // namespace

struct sv_batch {
    int n_inst = 0;
    sv_dtype dtype = SV_C64;
    cudaStream_t stream = nullptr;
    int device = 0, sm_count = 148, grid = 0, grid_max = 0, Dmax = 0;
    int Lmax = 0;                // most operators of an instance in the string-blocked form
    size_t smem = 0;             // dynamic shared memory of the launch
    int small = 0, teams = 1;    // instances that run one to a team of a block, and teams per block
    void *d_lists = nullptr, *d_groups = nullptr, *d_mats = nullptr;
    double *d_diag = nullptr, *d_gsum = nullptr;
    int threads = 384;  // block size of the persistent kernel: 256 or 384
    std::vector<int> L;
    std::vector<long long> cs_off, out_off;
    long long total_ops = 0, total_out = 0;
    std::vector<void *> dev;  // every device allocation
    BatchInst *d_inst = nullptr;
    int *d_order = nullptr, *d_ctrl = nullptr;
    BatchOp *d_ops = nullptr;
    void *d_cs = nullptr, *d_r = nullptr, *d_scratch = nullptr;
    double *d_theta = nullptr;
    double *d_d = nullptr, *d_out = nullptr;
    uint32_t *d_u32 = nullptr;
    uint16_t *d_u16 = nullptr;
    void *h_cs = nullptr;  // pinned: the angles of the next launch (float64)
    double *h_out = nullptr;
    int *h_ctrl = nullptr;
    unsigned long long budget_ns = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    bool own_stream = false;
    uint64_t launches = 0;
};

namespace {

template <typename R>
struct HostArena {
    std::vector<R> r;
    std::vector<double> d;
    std::vector<uint32_t> u32;
    std::vector<uint16_t> u16;
};

// String table set for (N, k electrons of one spin, spin offset 0 alpha / 1 beta): strings, ranks and
// spreads; for at most kBatchSmax strings also the excitation table (entry u of string I at [u][I]:
// partner rank | sign << 14 | orbital pair << 16, the single excitations, then one diagonal entry per
// occupied orbital) and the partners by orbital pair ([pair][I]: rank | sign << 14 | valid << 15).
struct StrSet {
    long long str, rank, spread, x, tgt;
    int count;
};

template <typename R>
BatchArgs<R> batch_args(const sv_batch *b) {
    BatchArgs<R> a;
    a.inst = b->d_inst; a.order = b->d_order; a.count = b->n_inst; a.ops = b->d_ops;
    a.angles = (const Angle<R> *)b->d_cs; a.rarena = (const R *)b->d_r; a.darena = b->d_d;
    a.u32 = b->d_u32; a.u16 = b->d_u16; a.out = b->d_out; a.scratch = (R *)b->d_scratch;
    a.lists = (const uint2 *)b->d_lists; a.groups = (const Group *)b->d_groups; a.mats = (const R *)b->d_mats;
    a.diag = b->d_diag; a.gsum = b->d_gsum; a.Dmax = b->Dmax; a.Lmax = b->Lmax; a.smem = b->smem;
    a.ctrl = b->d_ctrl; a.budget_ns = b->budget_ns; a.small = b->small; a.teams = b->teams;
    return a;
}

template <typename R>
sv_status build_plan(sv_batch *b, int n_inst, const sv_instance *inst) {
    HostArena<R> A;
    std::vector<BatchInst> hi(n_inst);
    std::vector<BatchOp> hops;
    std::vector<double> cost(n_inst);
    std::map<std::string, StrSet> sets;
    auto strset = [&](int N, int k, int spin) -> StrSet {
        std::string key = std::to_string(N) + "/" + std::to_string(k) + "/" + std::to_string(spin);
        auto it = sets.find(key);
        if (it != sets.end()) return it->second;
        StrSet s;
        s.rank = (long long)A.u16.size();
        A.u16.resize(A.u16.size() + ((size_t)1 << N), 0xFFFFu);
        std::vector<uint16_t> strs;
        for (uint32_t v = 0; v < (1u << N); ++v)
            if (__builtin_popcount(v) == k) {
                A.u16[s.rank + v] = (uint16_t)strs.size();
                strs.push_back((uint16_t)v);
            }
        s.str = (long long)A.u16.size();
        A.u16.insert(A.u16.end(), strs.begin(), strs.end());
        s.spread = (long long)A.u32.size();
        for (uint16_t v : strs) {
            uint32_t x = 0;
            for (int p = 0; p < N; ++p)
                if ((v >> p) & 1u) x |= 1u << (2 * p + spin);
            A.u32.push_back(x);
        }
        s.count = (int)strs.size();
        s.x = s.tgt = 0;
        if (s.count <= kBatchSmax) {
            const int D = s.count, nx = k * (N - k) + k, np = pair_count(N);
            s.x = (long long)A.u32.size();
            s.tgt = (long long)A.u16.size();
            A.u32.resize(A.u32.size() + (size_t)nx * D);
            A.u16.resize(A.u16.size() + (size_t)np * D, 0);
            for (int I = 0; I < D; ++I) {
                const uint32_t a = strs[I];
                int u = 0;
                auto put = [&](int p, int q, int J, uint32_t sg) {
                    const int pi = pair_index(std::min(p, q), std::max(p, q));
                    A.u32[s.x + (size_t)u++ * D + I] = (uint32_t)J | (sg << 14) | ((uint32_t)pi << 16);
                    A.u16[s.tgt + (size_t)pi * D + I] = (uint16_t)((uint32_t)J | (sg << 14) | 0x8000u);
                };
                for (int p = 0; p < N; ++p)
                    for (int q = 0; q < N; ++q) {
                        if (!((a >> p) & 1u) || ((a >> q) & 1u)) continue;
                        const uint32_t m = (1u << p) | (1u << q);
                        put(p, q, A.u16[s.rank + (a ^ m)], (uint32_t)__builtin_parity(a & bits_between(p, q)));
                    }
                for (int p = 0; p < N; ++p)
                    if ((a >> p) & 1u) put(p, p, I, 0u);
            }
        }
        sets[key] = s;
        return s;
    };
    std::vector<GroupPlan> plans;
    std::vector<Group> groups;
    std::vector<int> inst_of;
    long long words = 0, mats = 0, diags = 0;
    std::vector<std::function<size_t(int)>> need(n_inst);
    long long cs = 0, out = 0;
    b->L.resize(n_inst);
    b->cs_off.resize(n_inst);
    b->out_off.resize(n_inst);
    b->Dmax = 1;
    for (int t = 0; t < n_inst; ++t) {
        const sv_instance &in = inst[t];
        const int n = in.n_qubits, N = n / 2;
        if (n < 2 || n > 32 || (n & 1)) return bfail(SV_ERR_ARG, "instance qubit count must be even, 2..32");
        if (N > 16) return bfail(SV_ERR_ARG, "instance too large for the batched kernel");
        if (!in.h || !in.eri || (in.n_ops > 0 && !in.ops) || in.n_ops < 0 || in.n_occ < 0 || in.n_occ > n ||
            (in.n_occ > 0 && !in.occ))
            return bfail(SV_ERR_ARG, "bad instance description");
        uint32_t ref = 0;
        int na = 0, nb = 0;
        for (int k = 0; k < in.n_occ; ++k) {
            int j = in.occ[k];
            if (j < 0 || j >= n || ((ref >> j) & 1u)) return bfail(SV_ERR_ARG, "bad reference occupation");
            ref |= 1u << j;
            (j & 1) ? ++nb : ++na;
        }
        StrSet sa = strset(N, na, 0), sb = strset(N, nb, 1);
        const long long D = (long long)sa.count * sb.count;
        if (D > (1 << 22)) return bfail(SV_ERR_ARG, "instance sector too large for the batched kernel");
        b->Dmax = std::max<int>(b->Dmax, (int)D);
        BatchInst I{};
        I.n = n; I.N = N; I.Da = sa.count; I.Db = sb.count; I.L = in.n_ops;
        I.na = na; I.nb = nb;
        I.fast = sa.count <= kBatchSmax && sb.count <= kBatchSmax;
        I.sa = sa.spread; I.sb = sb.spread; I.stra = sa.str; I.strb = sb.str; I.ra = sa.rank; I.rb = sb.rank;
        // reference index
        uint32_t ra_str = 0, rb_str = 0;
        for (int p = 0; p < N; ++p) {
            if ((ref >> (2 * p)) & 1u) ra_str |= 1u << p;
            if ((ref >> (2 * p + 1)) & 1u) rb_str |= 1u << p;
        }
        I.hf = (uint32_t)A.u16[sb.rank + rb_str] * sa.count + A.u16[sa.rank + ra_str];
        // integrals: validated like sv_ham_create, then cast
        sv_ham H;
        H.n_orb = N;
        H.e_nuc = in.e_nuc;
        H.h.assign(in.h, in.h + (size_t)N * N);
        H.eri.assign(in.eri, in.eri + (size_t)N * N * N * N);
        for (int p = 0; p < N; ++p)
            for (int q = 0; q < N; ++q)
                if (std::fabs(H.h[p * N + q] - H.h[q * N + p]) > 1e-12 * std::max(1.0, std::fabs(H.h[p * N + q])))
                    return bfail(SV_ERR_ARG, "instance h is not symmetric");
        auto E = [&](int p, int q, int r, int s) { return H.eri[(((size_t)p * N + q) * N + r) * N + s]; };
        for (int p = 0; p < N; ++p)
            for (int q = 0; q < N; ++q)
                for (int r = 0; r < N; ++r)
                    for (int s = 0; s < N; ++s) {
                        double v = E(p, q, r, s), tol = 1e-12 * std::max(1.0, std::fabs(v));
                        if (!std::isfinite(v) || std::fabs(v - E(q, p, r, s)) > tol || std::fabs(v - E(p, q, s, r)) > tol ||
                            std::fabs(v - E(r, s, p, q)) > tol)
                            return bfail(SV_ERR_ARG, "instance eri lacks the 8-fold symmetry");
                    }
        I.shift = diag_energy(H, ref, n);
        I.e_shift = in.e_nuc - I.shift;
        I.eri = (long long)A.r.size();
        for (double v : H.eri) A.r.push_back((R)v);
        I.hm = (long long)A.r.size();
        for (double v : H.h) A.r.push_back((R)v);
        I.dt = (long long)A.r.size();
        for (int q = 0; q < N; ++q)
            for (int p = 0; p < N; ++p)
                for (int k = 0; k < N; ++k) A.r.push_back((R)(E(q, p, k, k) - E(q, k, k, p)));
        I.jt = (long long)A.r.size();
        for (int q = 0; q < N; ++q)
            for (int p = 0; p < N; ++p)
                for (int k = 0; k < N; ++k) A.r.push_back((R)E(q, p, k, k));
        HostTables<double> ht;
        build_tables<double>(H, n, ht);
        I.hd = (long long)A.d.size();
        A.d.insert(A.d.end(), ht.hdiag.begin(), ht.hdiag.end());
        I.jp = (long long)A.d.size();
        A.d.insert(A.d.end(), ht.Jp.begin(), ht.Jp.end());
        if (I.fast) {  // the integrals by orbital pairs
            const int np = pair_count(N);
            I.ep = (long long)A.r.size();
            A.r.resize(A.r.size() + (size_t)np * np);
            for (int q = 0; q < N; ++q)
                for (int p = 0; p <= q; ++p)
                    for (int s2 = 0; s2 < N; ++s2)
                        for (int r2 = 0; r2 <= s2; ++r2)
                            A.r[I.ep + (size_t)pair_index(p, q) * np + pair_index(r2, s2)] = (R)E(q, p, s2, r2);
            I.xa = sa.x; I.xb = sb.x; I.tgt = sa.tgt;
            I.ma = mats; mats += (long long)sa.count * sa.count;
            I.mb = mats; mats += (long long)sb.count * sb.count;
            I.da = diags; diags += sa.count;
            I.db = diags; diags += sb.count;
        }
        // operators, qubit space
        std::vector<OpDesc> descs;
        I.ops = (long long)hops.size();
        const int ident[32] = {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15,
                               16, 17, 18, 19, 20, 21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31};
        for (int k = 0; k < in.n_ops; ++k) {
            OpDesc d;
            std::string why;
            if (!make_op(in.ops[k], n, ident, d, why)) return bfail(SV_ERR_ARG, "instance op: " + why);
            uint32_t ma = 0, mb = 0;
            for (int p = 0; p < N; ++p) {
                if ((d.m >> (2 * p)) & 1u) ma |= 1u << p;
                if ((d.m >> (2 * p + 1)) & 1u) mb |= 1u << p;
            }
            hops.push_back(BatchOp{d.m, d.from, d.sm, ma | (mb << 16)});
            descs.push_back(d);
        }
        if (I.fast) {
            std::vector<uint8_t> pb, gb;
            uint64_t w = 0;
            long long most = 0, all = 0;
            const int ng = plan_groups(descs.data(), in.n_ops, N, na, nb, pb, gb, &w, &most, &all);
            if (w > (uint64_t)INT32_MAX) return bfail(SV_ERR_ARG, "instance operator lists too long");
            I.lists = words;
            I.words = (int)w;
            I.groups = (long long)groups.size();
            I.n_groups = ng;
            words += (long long)w;
            plans.insert(plans.end(), (const GroupPlan *)pb.data(), (const GroupPlan *)pb.data() + ng);
            groups.insert(groups.end(), (const Group *)gb.data(), (const Group *)gb.data() + ng);
            inst_of.insert(inst_of.end(), ng, t);
            b->Lmax = std::max(b->Lmax, in.n_ops);
            need[t] = [=](int warps) {  // its shared memory: the state, beside it the larger of its lists and sigma's work
                const size_t state = align16(sizeof(PairOf<R>) * (size_t)D),
                             lists = align16(8 * w) + align16(sizeof(Group) * (size_t)ng) + align16(sizeof(Angle<R>) * (size_t)in.n_ops),
                             ab = sizeof(R) == 4 ? 4 * (size_t)warps * blocked_warp_floats(N, sa.count) : 0;
                return state + std::max(lists, blocked_table_bytes<R>(N, na, nb, sa.count, sb.count) + ab);
            };
        }
        I.cs = cs;
        b->cs_off[t] = cs;
        cs += in.n_ops;
        I.out = out;
        b->out_off[t] = out;
        out += 1 + in.n_ops;
        b->L[t] = in.n_ops;
        hi[t] = I;
        // cost: sector size x (connections + 3 sweeps over the operators)
        const double conn = (double)na * (N - na) + (double)nb * (N - nb);
        cost[t] = (double)D * (conn * conn + 3.0 * in.n_ops + 1.0);
    }
    b->total_ops = cs;
    b->total_out = out;
    std::vector<int> order(n_inst);
    for (int t = 0; t < n_inst; ++t) order[t] = t;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    // Small instances (kBatchSmall determinants at most) run one to a team: four to a block where there
    // are at least four for each SM, so that one's barriers and latencies pass under another's work; in
    // blocks of 256 threads where there are no others.
    for (int t = n_inst; t-- > 0;) {
        const BatchInst &I = hi[order[t]];
        if (!I.fast || I.Da * I.Db > kBatchSmall) break;
        b->small++;
    }
    b->teams = b->small >= 4 * b->sm_count ? 4 : b->small >= 2 * b->sm_count ? 2 : 1;
    b->threads = b->small == n_inst && b->teams == 1 ? 256 : 384;
    for (int t = 0; t < n_inst; ++t) {
        if (!hi[order[t]].fast) continue;
        const bool s = t >= n_inst - b->small;
        const size_t w = need[order[t]](b->threads / 32 / (s ? b->teams : 1)), state = sizeof(PairOf<R>) * (size_t)hi[order[t]].Da * hi[order[t]].Db;
        b->smem = std::max(b->smem, std::min(kBatchSmemCap, s ? (w + 15) / 16 * 16 * b->teams : state <= kBatchSmemCap ? w : w - state));
    }
    // device arenas
    auto up = [&](void **dst, const void *src, size_t bytes) -> sv_status {
        cudaError_t e = cudaMalloc(dst, std::max<size_t>(bytes, 16));
        if (e != cudaSuccess) {
            cudaGetLastError();
            return bfail(SV_ERR_OOM, "batch arena allocation failed");
        }
        b->dev.push_back(*dst);
        if (bytes && src) {
            e = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
            if (e != cudaSuccess) return bfail(SV_ERR_CUDA, cudaGetErrorString(e));
        }
        return SV_OK;
    };
    sv_status s;
    if ((s = up((void **)&b->d_inst, hi.data(), hi.size() * sizeof(BatchInst))) != SV_OK) return s;
    if ((s = up((void **)&b->d_order, order.data(), order.size() * sizeof(int))) != SV_OK) return s;
    if ((s = up((void **)&b->d_ops, hops.data(), hops.size() * sizeof(BatchOp))) != SV_OK) return s;
    if ((s = up(&b->d_r, A.r.data(), A.r.size() * sizeof(R))) != SV_OK) return s;
    if ((s = up((void **)&b->d_d, A.d.data(), A.d.size() * sizeof(double))) != SV_OK) return s;
    if ((s = up((void **)&b->d_u32, A.u32.data(), A.u32.size() * sizeof(uint32_t))) != SV_OK) return s;
    if ((s = up((void **)&b->d_u16, A.u16.data(), A.u16.size() * sizeof(uint16_t))) != SV_OK) return s;
    if ((s = up(&b->d_cs, nullptr, std::max<long long>(cs, 1) * sizeof(Angle<R>))) != SV_OK) return s;
    if ((s = up((void **)&b->d_theta, nullptr, std::max<long long>(cs, 1) * sizeof(double))) != SV_OK) return s;
    if ((s = up((void **)&b->d_out, nullptr, std::max<long long>(out, 1) * sizeof(double))) != SV_OK) return s;
    if ((s = up((void **)&b->d_ctrl, nullptr, 4 * sizeof(int))) != SV_OK) return s;
    // scratch slots for the largest grid sv_batch_autotune may try (4 blocks per SM)
    b->grid_max = std::max(1, std::min(n_inst, b->sm_count * 4));
    b->grid = std::max(1, std::min(n_inst, b->sm_count * 2));
    if ((s = up(&b->d_scratch, nullptr, (size_t)b->grid_max * 2 * b->Dmax * sizeof(R))) != SV_OK) return s;
    if ((s = up(&b->d_lists, nullptr, (size_t)words * sizeof(uint2))) != SV_OK) return s;
    if ((s = up(&b->d_groups, groups.data(), groups.size() * sizeof(Group))) != SV_OK) return s;
    if ((s = up(&b->d_mats, nullptr, (size_t)mats * sizeof(R))) != SV_OK) return s;
    if ((s = up((void **)&b->d_diag, nullptr, (size_t)diags * sizeof(double))) != SV_OK) return s;
    if ((s = up((void **)&b->d_gsum, nullptr, (size_t)b->grid_max * b->Lmax * 32 * sizeof(double))) != SV_OK) return s;
    if (!plans.empty() || mats > 0) {  // what is the same for every angle
        void *d_plans = nullptr, *d_of = nullptr;
        if ((s = up(&d_plans, plans.data(), plans.size() * sizeof(GroupPlan))) != SV_OK) return s;
        if ((s = up(&d_of, inst_of.data(), inst_of.size() * sizeof(int))) != SV_OK) return s;
        cudaError_t e = mats > 0 ? cudaMemsetAsync(b->d_mats, 0, (size_t)mats * sizeof(R), b->stream) : cudaSuccess;
        if (e == cudaSuccess && !plans.empty()) {
            k_batch_lists<<<(unsigned)(4 * plans.size()), kThreads, 0, b->stream>>>(
                b->d_inst, (const int *)d_of, (const GroupPlan *)d_plans, b->d_u32, b->d_u16, (uint2 *)b->d_lists);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && mats > 0) {
            k_batch_mats<R><<<2 * n_inst, kThreads, 0, b->stream>>>(batch_args<R>(b), (R *)b->d_mats, b->d_diag);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return bfail(SV_ERR_CUDA, std::string("batch plan: ") + cudaGetErrorString(e));
        }
    }
    if (cudaMallocHost(&b->h_cs, std::max<long long>(cs, 1) * sizeof(double)) != cudaSuccess ||
        cudaMallocHost((void **)&b->h_out, std::max<long long>(out, 1) * sizeof(double)) != cudaSuccess ||
        cudaMallocHost((void **)&b->h_ctrl, 2 * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return bfail(SV_ERR_OOM, "pinned host allocation failed");
    }
    return SV_OK;
}

template <typename R>
sv_status capture(sv_batch *b) {
    const BatchArgs<R> a = batch_args<R>(b);
    cudaStream_t st = b->stream;
    cudaError_t e = cudaSuccess;
    // always: the default limit on dynamic shared memory is 48 KB less the kernel's static part
    e = b->threads == 384 ? allow_smem(k_batch<R, 384>, kBatchSmemCap) : allow_smem(k_batch<R, 256>, kBatchSmemCap);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return bfail(SV_ERR_CUDA, std::string("batch shared memory: ") + cudaGetErrorString(e));
    }
    e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return bfail(SV_ERR_CUDA, std::string("capture: ") + cudaGetErrorString(e));
    // the first of its nodes that is refused ends the capture: a graph without it would return what is in d_out
    auto add = [&](cudaError_t x) {
        if (e == cudaSuccess) e = x;
    };
    add(cudaMemcpyAsync(b->d_theta, b->h_cs, std::max<long long>(b->total_ops, 1) * sizeof(double), cudaMemcpyHostToDevice, st));
    if (b->total_ops > 0) {
        const long long g = std::min<long long>((b->total_ops + kThreads - 1) / kThreads, (long long)b->sm_count * 4);
        k_batch_sincos<R><<<(int)g, kThreads, 0, st>>>(b->d_theta, (Angle<R> *)b->d_cs, b->total_ops);
        add(cudaGetLastError());
    }
    add(cudaMemsetAsync(b->d_ctrl, 0, 4 * sizeof(int), st));
    if (b->threads == 384) k_batch<R, 384><<<b->grid, 384, b->smem, st>>>(a);
    else k_batch<R, 256><<<b->grid, 256, b->smem, st>>>(a);
    add(cudaGetLastError());
    add(cudaMemcpyAsync(b->h_out, b->d_out, std::max<long long>(b->total_out, 1) * sizeof(double), cudaMemcpyDeviceToHost, st));
    add(cudaMemcpyAsync(b->h_ctrl, b->d_ctrl, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
    cudaGraph_t graph = nullptr;
    const cudaError_t end = cudaStreamEndCapture(st, &graph);
    add(end);
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, graph, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (graph) cudaGraphDestroy(graph);
        b->exec = nullptr;
        return bfail(SV_ERR_CUDA, std::string("batch capture: ") + cudaGetErrorString(e));
    }
    b->graph = graph;
    return SV_OK;
}

template <typename R>
void fill_cs(sv_batch *b, const double *theta) {
    if (b->total_ops > 0) std::memcpy(b->h_cs, theta, (size_t)b->total_ops * sizeof(double));
}

}  // namespace

extern "C" {

sv_status sv_batch_create(int n_inst, const sv_instance *inst, sv_dtype dtype, void *cuda_stream,
                          sv_batch_handle *out) {
    if (!out) return bfail(SV_ERR_ARG, "NULL output handle pointer");
    *out = nullptr;
    if (n_inst < 1 || !inst) return bfail(SV_ERR_ARG, "need at least one instance");
    if (dtype != SV_C64 && dtype != SV_C128) return bfail(SV_ERR_ARG, "bad dtype");
    sv_batch *b = new sv_batch();
    b->n_inst = n_inst;
    b->dtype = dtype;
    b->stream = (cudaStream_t)cuda_stream;
    if (cudaGetDevice(&b->device) != cudaSuccess) {
        cudaGetLastError();
        delete b;
        return bfail(SV_ERR_CUDA, "no CUDA device");
    }
    if (!b->stream) {  // graph capture needs a stream other than the legacy default stream
        if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
            cudaGetLastError();
            delete b;
            return bfail(SV_ERR_CUDA, "stream creation failed");
        }
        b->own_stream = true;
    }
    cudaDeviceGetAttribute(&b->sm_count, cudaDevAttrMultiProcessorCount, b->device);
    sv_status s = dtype == SV_C64 ? build_plan<float>(b, n_inst, inst) : build_plan<double>(b, n_inst, inst);
    if (s != SV_OK) {
        sv_batch_destroy(b);
        return s;
    }
    *out = b;
    return SV_OK;
}

sv_status sv_batch_set_time_limit(sv_batch_handle b, double ms) {
    if (!b || !(ms >= 0.0) || !std::isfinite(ms)) return bfail(SV_ERR_ARG, "bad time limit");
    b->budget_ns = (unsigned long long)(ms * 1e6);
    if (b->exec) {
        cudaGraphExecDestroy(b->exec);
        b->exec = nullptr;
    }
    if (b->graph) {
        cudaGraphDestroy(b->graph);
        b->graph = nullptr;
    }
    return SV_OK;
}

sv_status sv_batch_energy_grad(sv_batch_handle b, const double *theta, double *e_out, double *grad_out) {
    if (!b) return bfail(SV_ERR_ARG, "NULL batch handle");
    if (b->total_ops > 0 && !theta) return bfail(SV_ERR_ARG, "NULL theta");
    for (long long k = 0; k < b->total_ops; ++k)
        if (!std::isfinite(theta[k])) return bfail(SV_ERR_ARG, "non-finite theta");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != b->device) cudaSetDevice(b->device);
    sv_status s = SV_OK;
    if (b->dtype == SV_C64) fill_cs<float>(b, theta);
    else fill_cs<double>(b, theta);
    for (long long k = 0; k < b->total_out; ++k) b->h_out[k] = std::nan("");
    if (!b->exec) s = b->dtype == SV_C64 ? capture<float>(b) : capture<double>(b);
    if (s == SV_OK) {
        cudaError_t e = cudaGraphLaunch(b->exec, b->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        if (e != cudaSuccess) {
            cudaGetLastError();
            s = bfail(SV_ERR_CUDA, std::string("batch launch: ") + cudaGetErrorString(e));
        } else {
            b->launches += b->total_ops > 0 ? 2 : 1;
        }
    }
    if (s == SV_OK) {
        for (int t = 0; t < b->n_inst; ++t) {
            const double *o = b->h_out + b->out_off[t];
            if (e_out) e_out[t] = o[0];
            if (grad_out)
                for (int k = 0; k < b->L[t]; ++k) grad_out[b->cs_off[t] + k] = o[1 + k];
        }
        if (b->h_ctrl[1]) s = bfail(SV_ERR_TIMEOUT, "batch time limit reached; unfinished instances are NaN");
    }
    if (prev >= 0 && prev != b->device) cudaSetDevice(prev);
    return s;
}

uint64_t sv_batch_launch_count(sv_batch_handle b) { return b ? b->launches : 0; }

static void drop_graph(sv_batch_handle b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
}

sv_status sv_batch_autotune(sv_batch_handle b, const double *theta, int *grid_out) {
    if (!b) return bfail(SV_ERR_ARG, "NULL batch handle");
    if (b->total_ops > 0 && !theta) return bfail(SV_ERR_ARG, "NULL theta");
    for (long long k = 0; k < b->total_ops; ++k)
        if (!std::isfinite(theta[k])) return bfail(SV_ERR_ARG, "non-finite theta");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != b->device) cudaSetDevice(b->device);
    if (b->dtype == SV_C64) fill_cs<float>(b, theta);
    else fill_cs<double>(b, theta);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    sv_status s = SV_OK;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) s = bfail(SV_ERR_CUDA, "event creation failed");
    const int keep = b->grid, keep_t = b->threads;
    int best = keep, best_threads = keep_t;
    float best_t = -1.f;
    // (threads per block, blocks per SM): at most 2048 resident threads per SM
    const int cands[][2] = {{256, 1}, {256, 2}, {256, 4}, {384, 1}, {384, 2}};
    for (const auto &cd : cands) {
        if (s != SV_OK) break;
        const int g = std::max(1, std::min(b->n_inst, b->sm_count * cd[1]));
        if (g > b->grid_max) continue;
        drop_graph(b);
        b->grid = g;
        b->threads = cd[0];
        s = b->dtype == SV_C64 ? capture<float>(b) : capture<double>(b);
        float ms = 0.f;
        for (int r = 0; s == SV_OK && r < 2; ++r) {  // the second run is timed
            cudaError_t e = cudaEventRecord(e0, b->stream);
            if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, b->stream);
            if (e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e != cudaSuccess) {
                cudaGetLastError();
                s = bfail(SV_ERR_CUDA, std::string("batch autotune launch: ") + cudaGetErrorString(e));
            } else {
                b->launches += b->total_ops > 0 ? 2 : 1;
            }
        }
        if (s == SV_OK && (best_t < 0.f || ms < best_t)) {
            best_t = ms;
            best = g;
            best_threads = cd[0];
        }
    }
    drop_graph(b);
    b->grid = s == SV_OK ? best : keep;
    b->threads = s == SV_OK ? best_threads : keep_t;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (grid_out) *grid_out = b->grid;
    if (prev >= 0 && prev != b->device) cudaSetDevice(prev);
    return s;
}

sv_status sv_batch_destroy(sv_batch_handle b) {
    if (!b) return SV_OK;
    if (b->stream) cudaStreamSynchronize(b->stream);
    else cudaDeviceSynchronize();
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (void *p : b->dev) cudaFree(p);
    if (b->h_cs) cudaFreeHost(b->h_cs);
    if (b->h_out) cudaFreeHost(b->h_out);
    if (b->h_ctrl) cudaFreeHost(b->h_ctrl);
    if (b->own_stream) cudaStreamDestroy(b->stream);
    cudaGetLastError();
    delete b;
    return SV_OK;
}

}  // extern "C"
