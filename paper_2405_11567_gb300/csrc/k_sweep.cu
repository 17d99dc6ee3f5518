// k_sweep.cu -- whole sector sweeps, two operators to a step.
//
// A sweep is bound by the latency of one step -- a barrier and a round trip of a few
// scattered amplitudes -- times the number of steps: with one operator to a step, 2.5 us
// forward and 3.4 us in reverse even where an operator has 36 pairs.  Two consecutive
// operators A, B (A first) with different flip masks are one step here.  A pairs x with
// x ^ mA and B pairs x with x ^ mB, so the determinants that the two connect are at most the
// four of a coset
//   e0 = x, e1 = x ^ mA, e2 = x ^ mB, e3 = x ^ mA ^ mB,
// and cosets are independent: one thread loads a component's two, three or four amplitudes,
// applies both operators in order and stores them.  Each rotation's arithmetic is that of one
// operator at a time, so the amplitudes are the same bits.
//
// A component is found from A's pair (x matches A's "from" pattern) or, where neither element
// of a pair of B touches A, from B's pair.  With F (T) true where x & mB is B's from (to)
// pattern, F', T' the same at x ^ mA, and o = mA & mB:
//   B pairs e0 with e2 where F or T holds, e1 with e3 where F' or T' holds;
//   A pairs e2 with e3 too where o = 0 (e2 has A's from pattern: the same component is met from
//   e0 and from e2, and taken where T does not hold) or o = mA (e3 has it: met from e0 and from
//   e3, and taken where F' and T' do not hold); any other overlap spoils A's pattern at e2 and e3.
// Every condition and sign is a product over the alpha and the beta string, so it comes from one
// word per string and list (k_build_groups): the four ranks, the string's parity under both
// operators' sign masks and its F, T, F', T'.
//
// Three forms of one kernel, by what separates the steps:
//   block    the sector fits in one block's shared memory and stays there: __syncthreads
//   cluster  sixteen blocks on amplitudes in L2, the cluster's hardware barrier
//   grid     every SM, amplitudes in L2, a counter in global memory; launched cooperatively, and
//            each wait bounded: past the limit the block sets *err and stops
// The reverse sweep works on psi and lambda interleaved (one access moves both) and takes the
// gradient terms of both operators; each warp's sum leaves the chip (float32 states: as an
// error-free sum of hi + lo words, since GB300 adds float64 at 1/64 of its float32 rate), and
// k_sweep_grad adds the warps' in order.
#include <algorithm>
#include <type_traits>

#include "sv_internal.h"
#include "sv_check.cuh"
#include "sv_ff.cuh"

namespace svk {

// One operator's string-space masks.
struct StrOp {
    uint32_t sm;              // sign mask (qubit space)
    uint32_t m[2], f[2];      // flip mask and from pattern of the alpha [0] and beta [1] string
};

// A step as the host plans it: its operators, and the offsets of its lists.
struct GroupPlan {
    StrOp op[2];              // A, B
    uint32_t off[2][2];       // [op][spin] offset of the list
    uint32_t len[2][2];       // its length
    int two;                  // 0: A alone
};

// A step as the sweep kernels read it.
struct Group {
    uint32_t off[2][2], len[2][2];  // [op][spin] offset and length of the lists
    uint32_t magic[2];        // floor(2^32 / len[op][0]) + 1 (0 where that length is 1)
    int k[2];                 // operator indices
    uint32_t over;            // 0: o = 0; 1: o = mA; 2: any other overlap, or one operator
    uint32_t cab, cba;        // parity of mB under A's sign mask, of mA under B's
    uint32_t pad;
};

namespace {

// A list entry, P the list's operator and Q the other, two words:
//   x: rank of the string s, of s ^ mP (14 bits each: at most C(16, 8) = 12,870 strings), F, T, F', T'
//   y: rank of s ^ mQ, of s ^ mP ^ mQ, the string's parity under P's sign mask, under Q's
constexpr int kRank = 14, kFlags = 28;
constexpr uint32_t kRankMask = (1u << kRank) - 1u;

__device__ __forceinline__ uint32_t parity32(uint32_t x) { return __popc(x) & 1u; }

// Block (group, op, spin): the list of the strings that match the operator's from pattern, by
// class (F, T, F', T') and in rank order within one: the components of a warp are then mostly of
// one shape, so that its lanes rotate together (GB300's FP64 pipe spends as long on one lane as
// on all; with the lists in rank order the 30-qubit float64 sweeps took 1.9 / 4.6 ms).
__global__ void __launch_bounds__(kThreads) k_build_groups(const GroupPlan *__restrict__ plans, const uint32_t *__restrict__ sa,
                                                           const uint32_t *__restrict__ sb, const uint16_t *__restrict__ stra,
                                                           const uint16_t *__restrict__ strb, const uint16_t *__restrict__ ra,
                                                           const uint16_t *__restrict__ rb, int Da, int Db,
                                                           uint2 *__restrict__ out, int sorted) {
    __shared__ int wcount[kThreads / 32];
    __shared__ unsigned int s_seen;
    const GroupPlan &g = plans[blockIdx.x >> 2];
    const int p = (blockIdx.x >> 1) & 1, spin = blockIdx.x & 1;
    if (p == 1 && !g.two) return;
    const StrOp P = g.op[p], Q = g.op[1 - p];
    const int D = spin ? Db : Da;
    const uint16_t *str = spin ? strb : stra, *rk = spin ? rb : ra;
    const uint32_t *spr = spin ? sb : sa;
    const uint32_t mp = P.m[spin], fp = P.f[spin], mq = Q.m[spin], fq = Q.f[spin];
    uint2 *dst = out + g.off[p][spin];
    const int cap = (int)g.len[p][spin];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const bool two = g.two;
    auto cls = [&](uint32_t s) {
        if (!two) return 0u;
        const uint32_t t = s ^ mp;
        return (uint32_t)((s & mq) == fq) | (uint32_t)((s & mq) == (mq ^ fq)) << 1 | (uint32_t)((t & mq) == fq) << 2 |
               (uint32_t)((t & mq) == (mq ^ fq)) << 3;
    };
    if (threadIdx.x == 0) s_seen = 0;
    __syncthreads();
    for (int I = threadIdx.x; I < D; I += blockDim.x)
        if ((str[I] & mp) == fp) atomicOr(&s_seen, 1u << cls(str[I]));
    __syncthreads();
    int total = 0;
    for (unsigned int seen = sorted ? s_seen : (s_seen != 0u); seen; seen &= seen - 1u) {
        const uint32_t want = __ffs(seen) - 1;
        for (int base = 0; base < D; base += blockDim.x) {
            const int I = base + threadIdx.x;
            uint32_t s = 0;
            bool hit = false;
            if (I < D) {
                s = str[I];
                hit = (s & mp) == fp && (!sorted || cls(s) == want);
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, hit);
            if (lane == 0) wcount[warp] = __popc(bal);
            __syncthreads();
            int off = total, sum = 0;
            for (int w = 0; w < nw; ++w) {
                const int c = wcount[w];
                if (w < warp) off += c;
                sum += c;
            }
            const int at = off + __popc(bal & lt);
            if (hit && at < cap) {
                auto rank = [&](uint32_t t) {  // 0 where there is no such string: never used
                    return rk[t] == 0xFFFFu ? 0u : (uint32_t)rk[t];
                };
                uint2 e = make_uint2((uint32_t)I | rank(s ^ mp) << kRank, parity32(spr[I] & P.sm) << kFlags);
                if (two) {
                    e.x |= cls(s) << kFlags;
                    e.y |= rank(s ^ mq) | rank(s ^ mp ^ mq) << kRank | parity32(spr[I] & Q.sm) << (kFlags + 1);
                }
                dst[at] = e;
            }
            total += sum;
            __syncthreads();
        }
    }
}

template <typename A>
struct alignas(2 * sizeof(A)) PairOf {
    A c, l;
};

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

// Sums of a thread's gradient terms: float32 terms error-free (hi + lo), float64 terms as they are.
template <typename R> struct GradSum;
template <> struct GradSum<float> {
    ff v = ff(0);
    __device__ __forceinline__ void add(float t) {
        float s, e;
        two_sum(v.hi, t, s, e);
        v = ff(s, v.lo + e);
    }
    __device__ __forceinline__ void add(const GradSum &o) { v = v + o.v; }
    __device__ __forceinline__ GradSum xor_lane(int m) const {
        GradSum o;
        o.v = ff(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
        return o;
    }
    __device__ __forceinline__ double bits() const { return __hiloint2double(__float_as_int(v.hi), __float_as_int(v.lo)); }
};
template <> struct GradSum<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double t) { v += t; }
    __device__ __forceinline__ void add(const GradSum &o) { v += o.v; }
    __device__ __forceinline__ GradSum xor_lane(int m) const {
        GradSum o;
        o.v = __shfl_xor_sync(0xffffffffu, v, m);
        return o;
    }
    __device__ __forceinline__ double bits() const { return v; }
};

// One operator's angle, as its rotations take it: c = cos, s = sin, and t = tan(theta / 2) for
// float64 states, 2 where the three-shear form does not apply (cos <= 0).
template <typename R> struct Angle {
    R c, s, t;
};

// exp(theta G) on the pair (u from, v to): (u, v) <- (c u - s v, c v + s u), sg the pair's sign
// (+-1 as a flip).  float64: three shears (Paeth), u1 = u - t v, v' = v + s u1, u' = u1 - t v',
// three multiply-adds a component instead of four operations (the FP64 pipe bounds these states).
__device__ __forceinline__ float flip(float x, uint32_t neg) { return __int_as_float(__float_as_int(x) ^ (int)(neg << 31)); }
__device__ __forceinline__ double flip(double x, uint32_t neg) {
    return __hiloint2double(__double2hiint(x) ^ (int)(neg << 31), __double2loint(x));
}
__device__ __forceinline__ void shear3(double &u, double &v, double s, double t) {
    u = fma(-t, v, u);
    v = fma(s, u, v);
    u = fma(-t, v, u);
}
__device__ __forceinline__ void shear3(double2 &u, double2 &v, double s, double t) {
    shear3(u.x, v.x, s, t);
    shear3(u.y, v.y, s, t);
}
template <bool SHEAR, typename A>
__device__ __forceinline__ void rotate2(A &u, A &v, const Angle<real_of<A>> &a, uint32_t neg) {
    const real_of<A> s = flip(a.s, neg);
    if constexpr (SHEAR && sizeof(real_of<A>) == 8) {
        if (__double2hiint(a.t) < 0x40000000) {  // t < 2, compared on the integer pipe
            shear3(u, v, s, flip(a.t, neg));
            return;
        }
    }
    const A w = u;
    u = lin2<A>(a.c, u, -s, v);
    v = lin2<A>(a.c, v, s, w);
}
// The gradient term of the pair, lam_v . u - lam_u . v with the pair's sign, and the inverse rotation of both.
template <typename A>
__device__ __forceinline__ void adjoint2(PairOf<A> &u, PairOf<A> &v, const Angle<real_of<A>> &a, uint32_t neg,
                                         GradSum<real_of<A>> &g) {
    g.add(flip(re_dot(v.l, u.c) - re_dot(u.l, v.c), neg));
    rotate2<true, A>(u.c, v.c, a, neg ^ 1u);
    rotate2<true, A>(u.l, v.l, a, neg ^ 1u);
}

// A thread's walk over an operator's pairs: flattened r n_a + i, every T-th from g.
struct ListWalk {
    int r, i, dr, di, na, nb;
    const uint2 *al, *bl;
    __device__ __forceinline__ void start(const Group &G, int op, const uint2 *lists, int g, int T) {
        al = lists + G.off[op][0];
        bl = lists + G.off[op][1];
        na = (int)G.len[op][0];
        nb = na > 0 ? (int)G.len[op][1] : 0;
        const uint32_t m = G.magic[op];  // exact for g, T with g na < 2^32
        r = m ? (int)__umulhi((uint32_t)g, m) : g;
        dr = m ? (int)__umulhi((uint32_t)T, m) : T;
        i = g - r * na;
        di = T - dr * na;
    }
    __device__ __forceinline__ bool more() const { return r < nb; }
    __device__ __forceinline__ bool next(uint2 &ea, uint2 &eb) {
        const bool ok = r < nb;
        ea = ok ? al[i] : make_uint2(0, 0);
        eb = ok ? bl[r] : make_uint2(0, 0);
        r += dr;
        i += di;
        if (i >= na) {
            i -= na;
            ++r;
        }
        return ok;
    }
};

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
    const int dir = ADJ ? -1 : 1, first = ADJ ? g.n_groups - 1 : 0;
    // the entries of a step's first components are loaded while the step before it is in flight
    ListWalk w[2];
    uint2 ea[2][kB], eb[2][kB];
    bool ok[2][kB];
    Group G, N;
    auto begin = [&](const Group &X) {
        #pragma unroll
        for (int p = 0; p < 2; ++p) {
            w[p].start(X, p, lists, gt, T);
            #pragma unroll
            for (int v = 0; v < kB; ++v) ok[p][v] = w[p].next(ea[p][v], eb[p][v]);
        }
    };
    Angle<R> nA = {1, 0, 0}, nB = {1, 0, 0};
    auto fetch = [&](int n) {
        N = groups[first + dir * n];
        nA = angles[N.k[0]];
        if (N.k[1] >= 0) nB = angles[N.k[1]];
    };
    if (g.n_groups > 0) {
        fetch(0);
        begin(N);
    }
    for (int n = 0; n < g.n_groups; ++n) {
        G = N;
        const Angle<R> aA = nA, aB = nB;
        const bool two = G.k[1] >= 0;
        if (n + 1 < g.n_groups) fetch(n + 1);
        if (!step_sync<FORM>(g, (unsigned int)n, &s_ok)) return;
        GradSum<R> gA, gB;
        for (;;) {
            // A's components, of which e0 and e1 are always there, and B's own pairs (no element touches A)
            P e[kB][4], p0[kB], p1[kB];
            uint32_t at[kB][4], q0[kB], q1[kB], fl[kB], sg[kB], sq[kB];
            bool use[kB], useB[kB], b0[kB], b1[kB], a2[kB];
            auto place = [&](uint32_t a, uint32_t b) { return (b & kRankMask) * (uint32_t)g.Da + (a & kRankMask); };
            #pragma unroll
            for (int v = 0; v < kB; ++v) {
                const uint2 x = ea[0][v], y = eb[0][v];
                fl[v] = (x.x & y.x) >> kFlags;
                sg[v] = (x.y ^ y.y) >> kFlags;
                use[v] = ok[0][v] && !(fl[v] & (G.over == 0 ? 2u : G.over == 1 ? 12u : 0u));
                at[v][0] = place(x.x, y.x);
                at[v][1] = place(x.x >> kRank, y.x >> kRank);
                // checked build: skip the component
                if (!SV_IN_RANGE(at[v][0], count, kChkPair) || !SV_IN_RANGE(at[v][1], count, kChkPair)) use[v] = false;
                at[v][2] = place(x.y, y.y);
                at[v][3] = place(x.y >> kRank, y.y >> kRank);
                if (!SV_IN_RANGE(at[v][2], count, kChkPair) || !SV_IN_RANGE(at[v][3], count, kChkPair)) use[v] = false;
                b0[v] = fl[v] & 3u;
                b1[v] = fl[v] & 12u;
                a2[v] = b0[v] && G.over < 2u;
                if (use[v]) {
                    e[v][0] = load(at[v][0]);
                    e[v][1] = load(at[v][1]);
                    if (b0[v]) e[v][2] = load(at[v][2]);
                    if (b1[v] || a2[v]) e[v][3] = load(at[v][3]);
                }
                const uint2 xb = ea[1][v], yb = eb[1][v];
                useB[v] = ok[1][v] && !((xb.x & yb.x) >> kFlags);
                q0[v] = place(xb.x, yb.x);
                q1[v] = place(xb.x >> kRank, yb.x >> kRank);
                sq[v] = (xb.y ^ yb.y) >> kFlags & 1u;
                if (!SV_IN_RANGE(q0[v], count, kChkPair) || !SV_IN_RANGE(q1[v], count, kChkPair)) useB[v] = false;
                if (useB[v]) {
                    p0[v] = load(q0[v]);
                    p1[v] = load(q1[v]);
                }
            }
            const bool more = w[0].more() || w[1].more();
            if (more) {
                #pragma unroll
                for (int p = 0; p < 2; ++p)
                    #pragma unroll
                    for (int v = 0; v < kB; ++v) ok[p][v] = w[p].next(ea[p][v], eb[p][v]);
            }
            #pragma unroll
            for (int v = 0; v < kB; ++v) {
                auto turn = [&](P &u, P &x, const Angle<R> &a, uint32_t neg, GradSum<R> &gs) {
                    if constexpr (ADJ) adjoint2<A>(u, x, a, neg, gs);
                    else rotate2<false, A>(u, x, a, neg);
                };
                if (use[v]) {
                    // A from e0, and from e2 where o = 0 or e3 where o = mA; B from e0 (e1) where F (F') holds, else
                    // from e2 (e3).  With the two elements exchanged a rotation is that of the opposite sign.
                    const uint32_t a0 = sg[v] & 1u, a1 = a0 ^ G.cab ^ (G.over == 1 ? 1u : 0u);
                    const uint32_t s0 = (sg[v] >> 1 ^ fl[v] ^ 1u) & 1u, s1 = (sg[v] >> 1 ^ G.cba ^ fl[v] >> 2 ^ 1u) & 1u;
                    auto opA = [&] {
                        turn(e[v][0], e[v][1], aA, a0, gA);
                        if (a2[v]) turn(e[v][2], e[v][3], aA, a1, gA);
                    };
                    auto opB = [&] {
                        if (b0[v]) turn(e[v][0], e[v][2], aB, s0, gB);
                        if (b1[v]) turn(e[v][1], e[v][3], aB, s1, gB);
                    };
                    if constexpr (ADJ) {
                        opB();
                        opA();
                    } else {
                        opA();
                        opB();
                    }
                    own[at[v][0]] = e[v][0];
                    own[at[v][1]] = e[v][1];
                    if (b0[v]) own[at[v][2]] = e[v][2];
                    if (b1[v] || a2[v]) own[at[v][3]] = e[v][3];
                }
                if (useB[v]) {
                    turn(p0[v], p1[v], aB, sq[v], gB);
                    own[q0[v]] = p0[v];
                    own[q1[v]] = p1[v];
                }
            }
            if (!more) break;
        }
        if (n + 1 < g.n_groups) begin(N);
        if constexpr (ADJ) {
            // both sums in one tree: the lower half warp takes A's, the upper B's
            GradSum<R> mine = lane < 16 ? gA : gB, other = lane < 16 ? gB : gA;
            mine.add(other.xor_lane(16));
            #pragma unroll
            for (int o = 8; o > 0; o >>= 1) mine.add(mine.xor_lane(o));
            if (lane == 0) g.partial[(size_t)G.k[0] * W + gw] = mine.bits();
            if (lane == 16 && two) g.partial[(size_t)G.k[1] * W + gw] = mine.bits();
        }
    }
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
    if (FORM == kBlock) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
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
    g.spins = spins; g.partial = partial;
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
