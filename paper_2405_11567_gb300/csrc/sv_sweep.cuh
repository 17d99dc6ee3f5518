// sv_sweep.cuh -- the steps of a sector sweep, two operators to a step: their lists, the
// rotations, and the walk that the whole-sweep kernels (k_sweep.cu) and the batched launch
// (k_batch.cu) share.
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
#pragma once

#include <type_traits>

#include "sv_check.cuh"
#include "sv_device.cuh"
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

// A list entry, P the list's operator and Q the other, two words:
//   x: rank of the string s, of s ^ mP (14 bits each: at most C(16, 8) = 12,870 strings), F, T, F', T'
//   y: rank of s ^ mQ, of s ^ mP ^ mQ, the string's parity under P's sign mask, under Q's
constexpr int kRank = 14, kFlags = 28;
constexpr uint32_t kRankMask = (1u << kRank) - 1u;

__device__ __forceinline__ uint32_t parity32(uint32_t x) { return __popc(x) & 1u; }

// The list of an operator P (of the other, Q) over one spin's strings, by a whole block: that of the strings that match the operator's from pattern, by
// class (F, T, F', T') and in rank order within one: the components of a warp are then mostly of
// one shape, so that its lanes rotate together (GB300's FP64 pipe spends as long on one lane as
// on all; with the lists in rank order the 30-qubit float64 sweeps took 1.9 / 4.6 ms).
// sorted = 0: in rank order alone (float32 states: longer runs of neighbouring amplitudes).
__device__ __forceinline__ void build_list(const StrOp &P, const StrOp &Q, bool two, int spin, int D, const uint16_t *str,
                                           const uint16_t *rk, const uint32_t *spr, uint2 *dst, int cap, int sorted) {
    __shared__ int wcount[kThreads / 32];
    __shared__ unsigned int s_seen;
    const uint32_t mp = P.m[spin], fp = P.f[spin], mq = Q.m[spin], fq = Q.f[spin];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
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

// Sums of a thread's gradient terms: float32 terms in two words (hi + lo, 48 bits: lo takes the rounding
// of hi and rounds itself, at 2^-24 of a term's own rounding), float64 terms as they are.
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
    if constexpr (sizeof(A) == 8 && !AmpT<A>::kCplx) {  // float64: two multiply-adds into the sum
        g.v = fma(flip(v.l, neg), u.c, g.v);
        g.v = fma(flip(u.l, neg ^ 1u), v.c, g.v);
    } else {
        g.add(flip(re_dot(v.l, u.c) - re_dot(u.l, v.c), neg));
    }
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

// A whole sweep's steps by T threads (this one number gt, of warp gw of W): amplitudes through
// load(at) and store(at, value) (P: with lambda in reverse), sync(n) before step n (false: a wait
// ran out, and so does this function return); gradient sums [operator][warp] into partial.
// KB: components of each operator that a thread has in flight.  once: 1.  Forward rotations of real float64
// amplitudes that a component may not have are loops of `once` turns, because a plain condition becomes
// predicated or selected arithmetic: every warp then ran four or five rotations for the one or two that it had,
// on the pipe that bounds it (30 qubits, 20 operators: 3.0 million FP64 instructions for 1.4; 200 operators 2.27 ms
// so, 1.52 with the loops, 1.56 one operator to a step; 28 qubits 676 and 480 us, 16 qubits 115 and 102).  Complex
// float64 gains nothing (22 qubits 195 and 197 us), and the reverse rotations branch by themselves.
template <typename A, bool ADJ, int KB, class Load, class Store, class Sync>
__device__ __forceinline__ bool run_steps(const uint2 *lists, const Group *groups, const Angle<real_of<A>> *angles, int n_groups,
                                          int Da, size_t count, int gt, int T, int gw, int W, int once, double *partial, Load load,
                                          Store store, Sync sync) {
    using R = real_of<A>;
    using P = std::conditional_t<ADJ, PairOf<A>, A>;
    const int lane = threadIdx.x & 31;
    const int dir = ADJ ? -1 : 1, first = ADJ ? n_groups - 1 : 0;
    // the entries of a step's first components are loaded while the step before it is in flight
    ListWalk w[2];
    uint2 ea[2][KB], eb[2][KB];
    bool ok[2][KB];
    Group G, N;
    auto begin = [&](const Group &X) {
        #pragma unroll
        for (int p = 0; p < 2; ++p) {
            w[p].start(X, p, lists, gt, T);
            #pragma unroll
            for (int v = 0; v < KB; ++v) ok[p][v] = w[p].next(ea[p][v], eb[p][v]);
        }
    };
    Angle<R> nA = {1, 0, 0}, nB = {1, 0, 0};
    auto fetch = [&](int n) {
        N = groups[first + dir * n];
        nA = angles[N.k[0]];
        if (N.k[1] >= 0) nB = angles[N.k[1]];
    };
    if (n_groups > 0) {
        fetch(0);
        begin(N);
    }
    for (int n = 0; n < n_groups; ++n) {
        G = N;
        const Angle<R> aA = nA, aB = nB;
        const bool two = G.k[1] >= 0;
        if (n + 1 < n_groups) fetch(n + 1);
        if (!sync(n)) return false;
        GradSum<R> gA, gB;
        bool did = false;
        #pragma unroll
        for (int v = 0; v < KB; ++v) did = did || ok[0][v] || ok[1][v];
        for (;;) {
            // A's components, of which e0 and e1 are always there, and B's own pairs (no element touches A)
            P e[KB][4], p0[KB], p1[KB];
            uint32_t at[KB][4], q0[KB], q1[KB], fl[KB], sg[KB], sq[KB];
            bool use[KB], useB[KB], b0[KB], b1[KB], a2[KB];
            auto place = [&](uint32_t a, uint32_t b) { return (b & kRankMask) * (uint32_t)Da + (a & kRankMask); };
            #pragma unroll
            for (int v = 0; v < KB; ++v) {
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
                    for (int v = 0; v < KB; ++v) ok[p][v] = w[p].next(ea[p][v], eb[p][v]);
            }
            #pragma unroll
            for (int v = 0; v < KB; ++v) {
                auto turn = [&](P &u, P &x, const Angle<R> &a, uint32_t neg, GradSum<R> &gs) {
                    if constexpr (ADJ) adjoint2<A>(u, x, a, neg, gs);
                    else rotate2<false, A>(u, x, a, neg);
                };
                auto turn_if = [&](bool c, P &u, P &x, const Angle<R> &a, uint32_t neg, GradSum<R> &gs) {
                    if constexpr (!ADJ && std::is_same<A, double>::value) {
                        #pragma unroll 1
                        for (int r = c ? once : 0; r > 0; --r) turn(u, x, a, neg, gs);
                    } else {
                        if (c) turn(u, x, a, neg, gs);
                    }
                };
                if (use[v]) {
                    // A from e0, and from e2 where o = 0 or e3 where o = mA; B from e0 (e1) where F (F') holds, else
                    // from e2 (e3).  With the two elements exchanged a rotation is that of the opposite sign.
                    const uint32_t a0 = sg[v] & 1u, a1 = a0 ^ G.cab ^ (G.over == 1 ? 1u : 0u);
                    const uint32_t s0 = (sg[v] >> 1 ^ fl[v] ^ 1u) & 1u, s1 = (sg[v] >> 1 ^ G.cba ^ fl[v] >> 2 ^ 1u) & 1u;
                    auto opA = [&] {
                        turn(e[v][0], e[v][1], aA, a0, gA);
                        turn_if(a2[v], e[v][2], e[v][3], aA, a1, gA);
                    };
                    auto opB = [&] {
                        turn_if(b0[v], e[v][0], e[v][2], aB, s0, gB);
                        turn_if(b1[v], e[v][1], e[v][3], aB, s1, gB);
                    };
                    if constexpr (ADJ) {
                        opB();
                        opA();
                    } else {
                        opA();
                        opB();
                    }
                    store(at[v][0], e[v][0]);
                    store(at[v][1], e[v][1]);
                    if (b0[v]) store(at[v][2], e[v][2]);
                    if (b1[v] || a2[v]) store(at[v][3], e[v][3]);
                }
                if (useB[v]) {
                    turn_if(true, p0[v], p1[v], aB, sq[v], gB);
                    store(q0[v], p0[v]);
                    store(q1[v], p1[v]);
                }
            }
            if (!more) break;
        }
        if (n + 1 < n_groups) begin(N);
        if constexpr (ADJ) {
            // both sums in one tree: the lower half warp takes A's, the upper B's (no tree, but zeros, where
            // the warp had no pair)
            GradSum<R> mine;
            if (__any_sync(0xffffffffu, did)) {
                mine = lane < 16 ? gA : gB;
                const GradSum<R> other = lane < 16 ? gB : gA;
                mine.add(other.xor_lane(16));
                #pragma unroll
                for (int o = 8; o > 0; o >>= 1) mine.add(mine.xor_lane(o));
            }
            if (lane == 0) partial[(size_t)G.k[0] * W + gw] = mine.bits();
            if (lane == 16 && two) partial[(size_t)G.k[1] * W + gw] = mine.bits();
        }
    }
    return true;
}

}  // namespace svk
