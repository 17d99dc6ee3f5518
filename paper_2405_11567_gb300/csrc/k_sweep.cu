// k_sweep.cu -- whole sector sweeps (the steps of sv_sweep.cuh) as one launch each.
//
// Three forms of one kernel, by what separates the steps:
//   block    the sector fits in one block's shared memory and stays there: __syncthreads
//   cluster  sixteen blocks on amplitudes in L2, the cluster's hardware barrier
//   grid     every SM, amplitudes in L2, a counter in global memory; launched cooperatively, and
//            each wait bounded: past the limit the block sets *err and stops
// The reverse sweep works on psi and lambda interleaved (one access moves both) and takes the
// gradient terms of both operators; each warp's sum leaves the chip (float32 states: as two words hi + lo,
// 48 bits, since GB300 adds float64 at 1/64 of its float32 rate), and k_sweep_grad adds the warps' in order.
#include <algorithm>
#include <vector>

#include "sv_internal.h"
#include "sv_sweep.cuh"

namespace svk {

namespace {

// Block (group, op, spin).
__global__ void __launch_bounds__(kThreads) k_build_groups(const GroupPlan *__restrict__ plans, const uint32_t *__restrict__ sa,
                                                           const uint32_t *__restrict__ sb, const uint16_t *__restrict__ stra,
                                                           const uint16_t *__restrict__ strb, const uint16_t *__restrict__ ra,
                                                           const uint16_t *__restrict__ rb, int Da, int Db,
                                                           uint2 *__restrict__ out, int sorted) {
    const GroupPlan &g = plans[blockIdx.x >> 2];
    const int p = (blockIdx.x >> 1) & 1, spin = blockIdx.x & 1;
    if (p == 1 && !g.two) return;
    build_list(g.op[p], g.op[1 - p], g.two, spin, spin ? Db : Da, spin ? strb : stra, spin ? rb : ra, spin ? sb : sa,
               out + g.off[p][spin], (int)g.len[p][spin], sorted);
}

// A value of 4 to 32 bytes from L2 (other SMs write these addresses between the steps).
template <typename P>
__device__ __forceinline__ P l2_load(const P *p) {
    constexpr int W = sizeof(P) / 4;
    union U {
        P p;
        uint32_t w[W];
        __device__ U() {}
    } u;
    if constexpr (W == 1) {
        u.w[0] = __ldcg(reinterpret_cast<const unsigned int *>(p));
    } else if constexpr (W == 2) {
        const uint2 t = __ldcg(reinterpret_cast<const uint2 *>(p));
        u.w[0] = t.x;
        u.w[1] = t.y;
    } else {
        #pragma unroll
        for (int v = 0; v < W / 4; ++v) {
            const uint4 t = __ldcg(reinterpret_cast<const uint4 *>(p) + v);
            u.w[4 * v] = t.x;
            u.w[4 * v + 1] = t.y;
            u.w[4 * v + 2] = t.z;
            u.w[4 * v + 3] = t.w;
        }
    }
    return u.p;
}

}  // namespace

struct SweepPlan {
    const uint2 *lists;
    const Group *groups;
    const void *angles;      // per operator: Angle in the state's precision
    int n_groups, n_ops, Da, Db;
    uint32_t words;          // block form: list words staged in shared memory (0: read from global memory)
    long long init;          // forward: compact index of the reference determinant, or -1 (psi is there)
    void *work;              // cluster and grid form, reverse: the interleaved matrix
    unsigned int *bar;       // grid form: barrier arrivals, zero at launch
    int *err;
    uint32_t spins;
    int once;                // 1 (run_steps)
    double *partial;         // reverse: [operators][warps] gradient sums (GradSum::bits)
};

enum { kBlock = 0, kCluster = 1, kGrid = 2 };

namespace {

// Separates two steps (number gen = 0, 1, ... of the launch); false: a bounded wait ran out.
template <int FORM>
__device__ __forceinline__ bool step_sync(const SweepPlan &g, unsigned int gen, volatile int *s_ok) {
    if constexpr (FORM == kBlock) {
        __syncthreads();
        return true;
    } else if constexpr (FORM == kCluster) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return true;
    } else {
        __syncthreads();
        if (threadIdx.x == 0) {
            // the block's writes, ordered before this thread by the block barrier, are released
            // with the arrival and the others' acquired with the count
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(g.bar), "r"(1u) : "memory");
            const unsigned int target = (gen + 1u) * gridDim.x;
            bool ok = true;
            for (uint32_t it = 0;; ++it) {
                unsigned int seen;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(g.bar) : "memory");
                if (seen >= target) break;
                if (it >= g.spins) {
                    ok = false;
                    atomicExch(g.err, 1);
                    break;
                }
            }
            *s_ok = ok;
        }
        __syncthreads();
        return *s_ok;
    }
}

}  // namespace

template <typename A, bool ADJ, int FORM>
__global__ void __launch_bounds__(FORM == kGrid ? 256 : 512, FORM == kGrid ? 2 : 1) k_sweep(A *__restrict__ psi, const A *__restrict__ lam, SweepPlan g) {
    using R = real_of<A>;
    using P = std::conditional_t<ADJ, PairOf<A>, A>;
    constexpr int kB = FORM == kGrid && sizeof(P) <= 8 ? 2 : 1;  // components of each operator in flight
    extern __shared__ __align__(16) uint8_t sweep_smem[];
    __shared__ volatile int s_ok;
    P *own = reinterpret_cast<P *>(sweep_smem);
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, nblk = FORM == kBlock ? 1 : (int)gridDim.x;
    // warps dealt to the blocks in turn, so that a step with few pairs still uses every block
    const int T = nblk * NT, gw = (tid >> 5) * nblk + (FORM == kBlock ? 0 : (int)blockIdx.x), gt = gw * 32 + lane, W = T >> 5;
    const size_t count = (size_t)g.Da * g.Db;
    const uint2 *lists = g.lists;
    const Group *groups = g.groups;
    const Angle<R> *angles = reinterpret_cast<const Angle<R> *>(g.angles);
    if constexpr (FORM == kBlock) {
        for (size_t e = tid; e < count; e += NT) {
            if constexpr (ADJ) {
                P p;
                p.c = psi[e];
                p.l = lam[e];
                own[e] = p;
            } else {
                own[e] = g.init >= 0 ? mka<A>((long long)e == g.init ? (R)1 : (R)0, (R)0) : psi[e];
            }
        }
        if (g.words > 0) {
            // lists, steps and angles too: a step is shorter than a read of L2
            uint2 *sl = reinterpret_cast<uint2 *>(sweep_smem + (count * sizeof(P) + 15) / 16 * 16);
            for (uint32_t e = tid; e < g.words; e += NT) sl[e] = g.lists[e];
            lists = sl;
            uint32_t *sg = reinterpret_cast<uint32_t *>(sl + g.words);
            const uint32_t ng = (uint32_t)(g.n_groups * sizeof(Group) / 4), na = (uint32_t)(g.n_ops * sizeof(Angle<R>) / 4);
            for (uint32_t e = tid; e < ng; e += NT) sg[e] = reinterpret_cast<const uint32_t *>(g.groups)[e];
            groups = reinterpret_cast<const Group *>(sg);
            sg += (ng + 1) / 2 * 2;
            for (uint32_t e = tid; e < na; e += NT) sg[e] = reinterpret_cast<const uint32_t *>(g.angles)[e];
            angles = reinterpret_cast<const Angle<R> *>(sg);
            __syncthreads();
        }
    } else {
        own = ADJ ? reinterpret_cast<P *>(g.work) : reinterpret_cast<P *>(psi);
        for (size_t e = (size_t)blockIdx.x * NT + tid; e < count; e += (size_t)T) {
            if constexpr (ADJ) {
                P p;
                p.c = psi[e];
                p.l = lam[e];
                own[e] = p;
            } else if (g.init >= 0) {
                psi[e] = mka<A>((long long)e == g.init ? (R)1 : (R)0, (R)0);
            }
        }
    }
    auto load = [&](uint32_t at) -> P {
        if constexpr (FORM == kBlock) return own[at];
        else return l2_load<P>(own + at);
    };
    auto store = [&](uint32_t at, const P &p) { own[at] = p; };
    auto sync = [&](int n) { return step_sync<FORM>(g, (unsigned int)n, &s_ok); };
    if (!run_steps<A, ADJ, kB>(lists, groups, angles, g.n_groups, g.Da, count, gt, T, gw, W, g.once, g.partial, load, store, sync)) return;
    if constexpr (FORM == kBlock && !ADJ) {
        __syncthreads();
        for (size_t e = tid; e < count; e += NT) psi[e] = own[e];
    }
}

// out[k] = the sum of op k's gradient sums over the W warps, in order.
template <bool SINGLE>
__global__ void __launch_bounds__(kThreads) k_sweep_grad(const double *__restrict__ partial, int W, double *__restrict__ out) {
    __shared__ double red[kThreads / 32];
    const double *row = partial + (size_t)blockIdx.x * W;
    double s = 0.0;
    if constexpr (SINGLE) {
        ff acc(0);
        for (int t = threadIdx.x; t < W; t += kThreads) {
            const double b = row[t];
            acc = acc + ff(__int_as_float(__double2hiint(b)), __int_as_float(__double2loint(b)));
        }
        s = ff_to(acc);
    } else {
        for (int t = threadIdx.x; t < W; t += kThreads) s += row[t];
    }
    s = block_sum(s, red);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// ---------------------------------------------------------------- host side

size_t sweep_angle_bytes(int dtype);

static uint64_t choose(int n, int k) {
    if (k < 0 || k > n) return 0;
    uint64_t r = 1;
    for (int i = 1; i <= k; ++i) r = r * (uint64_t)(n - k + i) / (uint64_t)i;
    return r;
}

static StrOp str_op(const OpDesc &d, int N) {
    StrOp o = {d.sm, {0, 0}, {0, 0}};
    for (int q = 0; q < N; ++q)
        for (int s = 0; s < 2; ++s) {
            o.m[s] |= ((d.m >> (2 * q + s)) & 1u) << q;
            o.f[s] |= ((d.from >> (2 * q + s)) & 1u) << q;
        }
    return o;
}

// The steps of an operator list: plans and groups (bytes of GroupPlan and Group), the list words
// they take, the most pairs of an operator and the pairs of all of them.
int plan_groups(const OpDesc *ops, int n_ops, int N, int na, int nb, std::vector<uint8_t> &plans, std::vector<uint8_t> &groups,
                uint64_t *words, long long *most, long long *all) {
    plans.clear();
    groups.clear();
    uint64_t off = 0;
    *most = *all = 0;
    const int ne[2] = {na, nb};
    int count = 0;
    for (int k = 0; k < n_ops; ++count) {
        const bool two = k + 1 < n_ops && ops[k].m != ops[k + 1].m;
        GroupPlan p = {};
        Group g = {};
        p.two = two;
        for (int j = 0; j < (two ? 2 : 1); ++j) {
            const StrOp o = p.op[j] = str_op(ops[k + j], N);
            long long pairs = 1;
            for (int s = 0; s < 2; ++s) {
                const uint32_t len =
                    (uint32_t)choose(N - __builtin_popcount(o.m[s]), ne[s] - __builtin_popcount(o.f[s]));
                p.off[j][s] = g.off[j][s] = (uint32_t)off;
                p.len[j][s] = g.len[j][s] = len;
                off += len;
                pairs *= len;
            }
            g.magic[j] = g.len[j][0] > 1 ? (uint32_t)((1ull << 32) / g.len[j][0]) + 1u : 0u;
            *most = std::max(*most, pairs);
            *all += pairs;
        }
        g.k[0] = k;
        g.k[1] = two ? k + 1 : -1;
        g.over = 2;
        if (two) {
            const uint32_t mA = ops[k].m, mB = ops[k + 1].m, o = mA & mB;
            g.over = o == 0 ? 0u : o == mA ? 1u : 2u;
            g.cab = (uint32_t)__builtin_parity(mB & ops[k].sm);
            g.cba = (uint32_t)__builtin_parity(mA & ops[k + 1].sm);
        }
        plans.insert(plans.end(), (uint8_t *)&p, (uint8_t *)&p + sizeof p);
        groups.insert(groups.end(), (uint8_t *)&g, (uint8_t *)&g + sizeof g);
        k += two ? 2 : 1;
    }
    *words = off;
    return count;
}

cudaError_t launch_build_groups(const void *plans, int n_groups, const uint32_t *sa, const uint32_t *sb, const uint16_t *stra,
                                const uint16_t *strb, const uint16_t *ra, const uint16_t *rb, int Da, int Db, int sorted, void *out,
                                cudaStream_t st) {
    if (n_groups <= 0) return cudaSuccess;
    k_build_groups<<<4 * n_groups, kThreads, 0, st>>>((const GroupPlan *)plans, sa, sb, stra, strb, ra, rb, Da, Db,
                                                      (uint2 *)out, sorted);
    return cudaGetLastError();
}

// Shared memory of the block form without its staged lists.
size_t sweep_block_smem(int dtype, bool adjoint, int Da, int Db) {
    return ((size_t)Da * Db * amp_size(dtype) * (adjoint ? 2 : 1) + 15) / 16 * 16;
}

// What its lists, steps and angles take beside it.
size_t sweep_stage_bytes(int dtype, uint64_t words, int n_groups, int n_ops) {
    return 8 * (size_t)words + (sizeof(Group) * n_groups + 7) / 8 * 8 + sweep_angle_bytes(dtype) * n_ops;
}

// The angles of an operator list as the kernels take them (sweep_angle_bytes each).
size_t sweep_angle_bytes(int dtype) { return single_prec(dtype) ? sizeof(Angle<float>) : sizeof(Angle<double>); }
void sweep_angles(const OpDesc *ops, int n_ops, int dtype, void *out) {
    for (int k = 0; k < n_ops; ++k) {
        if (single_prec(dtype)) ((Angle<float> *)out)[k] = {(float)ops[k].c, (float)ops[k].s, 0.f};
        else ((Angle<double> *)out)[k] = {ops[k].c, ops[k].s, ops[k].c > 0.0 ? ops[k].s / (1.0 + ops[k].c) : 2.0};
    }
}

namespace {

template <typename A, bool ADJ, int FORM>
cudaError_t sweep_launch(A *psi, const A *lam, SweepPlan g, int blocks, int threads, size_t smem, cudaStream_t st) {
    auto *kernel = k_sweep<A, ADJ, FORM>;
    cudaError_t e = cudaSuccess;
    if (FORM == kBlock) e = allow_smem(kernel, kSweepSmemCap);
    if (FORM == kCluster) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    if (FORM == kCluster) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = blocks;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = FORM == kBlock ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, psi, lam, g);
}

template <typename A, bool ADJ>
cudaError_t sweep_form(A *psi, const A *lam, SweepPlan g, int form, int blocks, int threads, size_t smem, cudaStream_t st) {
    if (form == kBlock) return sweep_launch<A, ADJ, kBlock>(psi, lam, g, 1, threads, smem, st);
    if (form == kCluster) return sweep_launch<A, ADJ, kCluster>(psi, lam, g, blocks, threads, 0, st);
    return sweep_launch<A, ADJ, kGrid>(psi, lam, g, blocks, threads, 0, st);
}

}  // namespace

// Blocks of the grid form: at most bps per SM, and no more than can be resident at once.
int sweep_grid_blocks(int dtype, bool adjoint, int sm_count, int bps) {
    int per_sm = 0;
    cudaError_t e = cudaErrorInvalidValue;
    SV_DISPATCH_AMP(dtype, e = adjoint ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep<A, true, kGrid>, 256, 0)
                                       : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep<A, false, kGrid>, 256, 0));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return std::min(per_sm, bps) * sm_count;
}

cudaError_t launch_sweep(void *psi, const void *lam, int dtype, bool adjoint, int form, int blocks, int threads, uint32_t words,
                         const void *lists, const void *groups, int n_groups, const void *angles, int n_ops, int Da, int Db,
                         long long init, void *work, unsigned int *bar, int *err, uint32_t spins, double *partial, cudaStream_t st) {
    SweepPlan g;
    g.lists = (const uint2 *)lists; g.groups = (const Group *)groups; g.angles = angles; g.n_ops = n_ops;
    g.n_groups = n_groups; g.Da = Da; g.Db = Db; g.words = words; g.init = init; g.work = work; g.bar = bar; g.err = err;
    g.spins = spins; g.once = 1; g.partial = partial;
    const size_t smem = form == kBlock ? sweep_block_smem(dtype, adjoint, Da, Db) +
                                             (words ? sweep_stage_bytes(dtype, words, n_groups, n_ops) : 0) : 0;
    cudaError_t e = cudaErrorInvalidValue;
    SV_DISPATCH_AMP(dtype, e = adjoint ? sweep_form<A, true>((A *)psi, (const A *)lam, g, form, blocks, threads, smem, st)
                                       : sweep_form<A, false>((A *)psi, (const A *)lam, g, form, blocks, threads, smem, st));
    return e;
}

cudaError_t launch_sweep_grad(const double *partial, int dtype, int n_ops, int warps, double *out, cudaStream_t st) {
    if (n_ops <= 0) return cudaSuccess;
    if (single_prec(dtype)) k_sweep_grad<true><<<n_ops, kThreads, 0, st>>>(partial, warps, out);
    else k_sweep_grad<false><<<n_ops, kThreads, 0, st>>>(partial, warps, out);
    return cudaGetLastError();
}

SV_CHECK_READER(check_word_sweep)

}  // namespace svk
