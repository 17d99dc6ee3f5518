// k_sector.cu -- kernels for sector storage: the state held as only the
// amplitudes of its (N_alpha, N_beta) sector, in the string-row order
// C[rank(b)][rank(a)] (x = spread_alpha(a) | spread_beta(b)); 9,018,009 amplitudes
// (72 MB in complex64) at 30 qubits and 10 electrons instead of 2^30.  Every
// operator of the method conserves both electron numbers, so nothing outside the
// sector is ever needed.
//
// An excitation (or a density-matrix element a+_p a_q) acts on the determinants
// whose alpha string matches its alpha "from" pattern and whose beta string
// matches its beta pattern; its partner is found through the string ranks.  The
// rotation kernels spread an operator's pairs (its alpha list x beta list) over the
// whole grid, so a launch touches only the pairs it rotates:
//   k_rotate_l   psi'[x] = c psi[x] - s sn psi[x'],  psi'[x'] = c psi[x'] + s sn psi[x]
//                over the op's pairs (alpha list x beta list, built by k_build_lists)
//   k_adjoint_l  g += s (Re conj(lam[x']) psi[x] - Re conj(lam[x]) psi[x']), then U^dagger
//                on psi and lambda (float64 per block, fixed-order sums)
//   k_rdm_rows   groups of rows, then of columns: every density-matrix element's share
// with s = (-1)^popc(x & sm), the Jordan-Wigner sign (sm = 0 for qubit
// excitations).
#include <cstring>
#include <vector>

#include "sv_internal.h"
#include "sv_check.cuh"
#include "sv_ff.cuh"
#include "sv_sigma.cuh"

namespace svk {

// An op's sign mask and its alpha / beta string flip masks and "from" patterns.
struct SectOp {
    uint32_t sm;
    uint32_t ma, fa, mb, fb;
};

struct SectTabs {
    const uint32_t *sa, *sb;       // qubit-space spreads
    const uint16_t *stra, *strb;   // strings
    const uint16_t *ra, *rb;       // ranks
    int Da, Db;
};

// Per-operator lists.  An operator acts on the determinants whose alpha string
// matches its alpha pattern and whose beta string matches its beta pattern, so its
// pairs are the product of an alpha list and a beta list.  Both are built once per
// operator list (k_build_lists) and kept on the device: one uint32 per string,
//   rank | sign << 15 | partner rank << 16,
// with sign = parity of the string's spread under the operator's sign mask (the
// Jordan-Wigner sign of the pair is the XOR of the alpha and beta entries).
// Ranks fit in 15 bits: at most C(16, 8) = 12,870 strings.
struct ListOp {
    uint32_t sm, ma, fa, mb, fb;
    uint32_t a_off, b_off;  // entry offsets of the op's alpha and beta lists
    uint32_t a_n, b_n;      // their lengths (C(N - |m|, n - |f|) per spin)
};

// Block 2k builds op k's alpha list, block 2k+1 its beta list, in rank order
// (ordered compaction with warp ballots).
__global__ void __launch_bounds__(kThreads) k_build_lists(const ListOp *__restrict__ ops, SectTabs T,
                                                          uint32_t *__restrict__ out) {
    __shared__ int wcount[kThreads / 32];
    const ListOp op = ops[blockIdx.x >> 1];
    const bool beta = blockIdx.x & 1;
    const int D = beta ? T.Db : T.Da;
    const uint16_t *str = beta ? T.strb : T.stra, *rk = beta ? T.rb : T.ra;
    const uint32_t *spr = beta ? T.sb : T.sa;
    const uint32_t m = beta ? op.mb : op.ma, f = beta ? op.fb : op.fa;
    uint32_t *dst = out + (beta ? op.b_off : op.a_off);
    const int cap = (int)(beta ? op.b_n : op.a_n);  // the host's count: writes never pass it
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    int total = 0;
    for (int base = 0; base < D; base += blockDim.x) {
        const int I = base + threadIdx.x;
        uint32_t s = 0;
        bool hit = false;
        if (I < D) {
            s = str[I];
            hit = (s & m) == f;
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
        if (hit && off + __popc(bal & lt) < cap)
            dst[off + __popc(bal & lt)] = (uint32_t)I | ((uint32_t)par(spr[I] & op.sm) << 15) |
                                          ((uint32_t)rk[s ^ m] << 16);
        total += sum;
        __syncthreads();
    }
}

// The op's pairs (beta entry r, alpha entry i) in flattened order r na + i, spread
// over the whole grid: thread t takes pairs t, t + T, ... (T = threads in the grid),
// four at a time so their loads are in flight together.  Pair (r, i) is (I, J) with
//   I = rank_b(r) Da + rank_a(i),  J = partner_b(r) Da + partner_a(i),
// and the Jordan-Wigner sign the XOR of the two entries' sign bits.
struct PairWalk {
    int r, i, dr, di, na;
    __device__ __forceinline__ PairWalk(int na_l) : na(na_l) {
        const int T = (int)(gridDim.x * blockDim.x), g = (int)(blockIdx.x * blockDim.x + threadIdx.x);
        r = g / na_l;
        i = g - r * na_l;
        dr = T / na_l;
        di = T - dr * na_l;
    }
    __device__ __forceinline__ void next() {
        r += dr;
        i += di;
        if (i >= na) {
            i -= na;
            ++r;
        }
    }
};

constexpr int kPairBatch = 4;

// psi <- exp(theta G) psi over the op's pairs.
template <typename A>
__global__ void __launch_bounds__(kThreads) k_rotate_l(A *__restrict__ psi, const uint32_t *__restrict__ al,
                                                       int na_l, const uint32_t *__restrict__ bl, int nb_l, int Da,
                                                       real_of<A> c, real_of<A> sn) {
    using R = real_of<A>;
    if (na_l <= 0) return;
    PairWalk w(na_l);
    while (w.r < nb_l) {
        size_t I[kPairBatch], J[kPairBatch];
        bool ok[kPairBatch];
        R ss[kPairBatch];
        #pragma unroll
        for (int v = 0; v < kPairBatch; ++v) {
            ok[v] = w.r < nb_l;
            const uint32_t eb = ok[v] ? bl[w.r] : 0u, ea = ok[v] ? al[w.i] : 0u;  // 0: rank 0, in bounds
            I[v] = (size_t)(eb & 0x7FFFu) * Da + (ea & 0x7FFFu);
            J[v] = (size_t)(eb >> 16) * Da + (ea >> 16);
            ss[v] = ((ea ^ eb) & 0x8000u) ? -sn : sn;
            w.next();
        }
        A u[kPairBatch], x[kPairBatch];
        #pragma unroll
        for (int v = 0; v < kPairBatch; ++v) {
            u[v] = psi[I[v]];
            x[v] = psi[J[v]];
        }
        #pragma unroll
        for (int v = 0; v < kPairBatch; ++v) {
            if (!ok[v]) continue;
            psi[I[v]] = lin2<A>(c, u[v], -ss[v], x[v]);
            psi[J[v]] = lin2<A>(c, x[v], ss[v], u[v]);
        }
    }
}

// Adjoint step over the op's pairs: the gradient term, then U^dagger on psi and
// lambda; one float64 partial per block (fixed order: every block writes its entry).
template <typename A>
__global__ void __launch_bounds__(kThreads) k_adjoint_l(A *__restrict__ psi, A *__restrict__ lam,
                                                        const uint32_t *__restrict__ al, int na_l,
                                                        const uint32_t *__restrict__ bl, int nb_l, int Da,
                                                        real_of<A> c, real_of<A> sn, double *__restrict__ partial) {
    using R = real_of<A>;
    __shared__ double red[kThreads / 32];
    double acc = 0.0;
    if (na_l > 0) {
        PairWalk w(na_l);
        while (w.r < nb_l) {
            size_t I[kPairBatch], J[kPairBatch];
            bool ok[kPairBatch], neg[kPairBatch];
            #pragma unroll
            for (int v = 0; v < kPairBatch; ++v) {
                ok[v] = w.r < nb_l;
                const uint32_t eb = ok[v] ? bl[w.r] : 0u, ea = ok[v] ? al[w.i] : 0u;
                I[v] = (size_t)(eb & 0x7FFFu) * Da + (ea & 0x7FFFu);
                J[v] = (size_t)(eb >> 16) * Da + (ea >> 16);
                neg[v] = ((ea ^ eb) & 0x8000u) != 0u;
                w.next();
            }
            A u[kPairBatch], x[kPairBatch], lu[kPairBatch], lx[kPairBatch];
            #pragma unroll
            for (int v = 0; v < kPairBatch; ++v) {
                u[v] = psi[I[v]];
                x[v] = psi[J[v]];
                lu[v] = lam[I[v]];
                lx[v] = lam[J[v]];
            }
            R t = 0;
            #pragma unroll
            for (int v = 0; v < kPairBatch; ++v) {
                if (!ok[v]) continue;
                const R ti = re_dot(lx[v], u[v]) - re_dot(lu[v], x[v]);
                t += neg[v] ? -ti : ti;
                const R ss = neg[v] ? -sn : sn;
                psi[I[v]] = lin2<A>(c, u[v], ss, x[v]);
                psi[J[v]] = lin2<A>(c, x[v], -ss, u[v]);
                lam[I[v]] = lin2<A>(c, lu[v], ss, lx[v]);
                lam[J[v]] = lin2<A>(c, lx[v], -ss, lu[v]);
            }
            acc += (double)t;
        }
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// The same adjoint step on the interleaved matrix CL[2 e] = psi[e], CL[2 e + 1] = lam[e]:
// one vector load / store per amplitude moves both, so each pair costs two scattered
// accesses instead of four and every 32-byte L2 sector it touches carries twice the
// useful bytes.  Same arithmetic in the same order as k_adjoint_l.
template <typename A>
struct alignas(2 * sizeof(A)) AmpPair {
    A c, l;
};

template <typename A>
__global__ void __launch_bounds__(kThreads) k_adjoint_li(A *__restrict__ CL, const uint32_t *__restrict__ al, int na_l,
                                                         const uint32_t *__restrict__ bl, int nb_l, int Da,
                                                         real_of<A> c, real_of<A> sn, double *__restrict__ partial) {
    using R = real_of<A>;
    __shared__ double red[kThreads / 32];
    AmpPair<A> *P = reinterpret_cast<AmpPair<A> *>(CL);
    double acc = 0.0;
    if (na_l > 0) {
        PairWalk w(na_l);
        while (w.r < nb_l) {
            size_t I[kPairBatch], J[kPairBatch];
            bool ok[kPairBatch], neg[kPairBatch];
            #pragma unroll
            for (int v = 0; v < kPairBatch; ++v) {
                ok[v] = w.r < nb_l;
                const uint32_t eb = ok[v] ? bl[w.r] : 0u, ea = ok[v] ? al[w.i] : 0u;
                I[v] = (size_t)(eb & 0x7FFFu) * Da + (ea & 0x7FFFu);
                J[v] = (size_t)(eb >> 16) * Da + (ea >> 16);
                neg[v] = ((ea ^ eb) & 0x8000u) != 0u;
                w.next();
            }
            AmpPair<A> pu[kPairBatch], px[kPairBatch];
            #pragma unroll
            for (int v = 0; v < kPairBatch; ++v) {
                pu[v] = P[I[v]];
                px[v] = P[J[v]];
            }
            R t = 0;
            #pragma unroll
            for (int v = 0; v < kPairBatch; ++v) {
                if (!ok[v]) continue;
                const A u = pu[v].c, x = px[v].c, lu = pu[v].l, lx = px[v].l;
                const R ti = re_dot(lx, u) - re_dot(lu, x);
                t += neg[v] ? -ti : ti;
                const R ss = neg[v] ? -sn : sn;
                AmpPair<A> ou, ox;
                ou.c = lin2<A>(c, u, ss, x);
                ox.c = lin2<A>(c, x, -ss, u);
                ou.l = lin2<A>(c, lu, ss, lx);
                ox.l = lin2<A>(c, lx, -ss, lu);
                P[I[v]] = ou;
                P[J[v]] = ox;
            }
            acc += (double)t;
        }
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// The row sums' arithmetic: float32 or float64 for those states, float-float (hi + lo
// float32 words, error-free transformations) for float64 states converted to it.
__device__ __forceinline__ double to_double(float x) { return (double)x; }
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(ff x) { return ff_to(x); }
__device__ __forceinline__ ff re_dot(ffc u, ffc v) { return ff_fma(u.y, v.y, u.x * v.x); }
__device__ __forceinline__ ff im_dot(ffc u, ffc v) { return ff_fma(u.x, v.y, -(u.y * v.x)); }
__device__ __forceinline__ ff re_dot(ff u, ff v) { return u * v; }
__device__ __forceinline__ ff im_dot(ff, ff) { return ff(0, 0); }
// fixed shuffle tree as warp_sum, each step a float-float addition
__device__ __forceinline__ ff warp_sum(ff v) {
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ff w;
        w.hi = __shfl_down_sync(0xffffffffu, v.hi, o);
        w.lo = __shfl_down_sync(0xffffffffu, v.lo, o);
        v = v + w;
    }
    return v;
}

// Density matrix by rows.  A block takes RW rows b of C at a time (alpha pairs), then RW columns a
// (beta pairs), and holds them in shared memory string by string, so that one list entry serves RW
// products and a string's amplitudes are one or two 16-byte words:
//   norm (alpha part) and the spin's occupations   sum |C|^2 (string holds p)
//   pairs p < q   sum over the strings x with q, without p of
//                 conj(C[x']) C[x] (-1)^popc(spread(x) & between), x' = x - q + p (the pair's list),
//                 times each row's own sign (-1)^popc(spread(other string) & between)
// in the element order norm, n occupations (j = 2p + sigma), alpha pairs, beta pairs.  Each pair belongs
// to one warp.  Its lanes' sums are reduced row by row (row_sums) and added, in float64, to the pair's
// slot of that row; the occupations are summed in float-float (float64 for float64 rows).  partial[e]
// [blockIdx.x] at the end: fixed-order sums.
// Bound by shared memory (16-byte words at list order: four cycles a warp and more where strings share
// a bank); float-float states by the FP32 pipe.  One row to a warp's pass, from L1, with the list read
// again for every row: 30 qubits (5, 5) float32 900 us, float64 1,250; so: 230 and 590 (28 qubits float32
// 478 and 153, 24 qubits 45 and 27).
template <typename R> struct RdmSum { using T = R; };
template <> struct RdmSum<float> { using T = ff; };
__device__ __forceinline__ void sum_to(ff &acc, float w) {
    float s, e;
    two_sum(acc.hi, w, s, e);
    acc = ff_make(s, acc.lo + e);
}
__device__ __forceinline__ void sum_to(ff &acc, ff w) { acc += w; }
__device__ __forceinline__ void sum_to(double &acc, double w) { acc += w; }
template <typename T> __device__ __forceinline__ T lane_xor(T v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ ff lane_xor(ff v, int o) {
    return ff_make(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
// Sums v[r] over the lanes, each of the RW sums on 32 / RW lanes: lane l returns that of r = l RW / 32.
template <int RW, typename R>
__device__ __forceinline__ R row_sums(R (&v)[RW], int lane) {
    int o = 16;
    #pragma unroll
    for (int h = RW / 2; h > 0; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
        #pragma unroll
        for (int j = 0; j < h; ++j) {
            const R send = up ? v[j] : v[j + h], keep = up ? v[j + h] : v[j];
            v[j] = keep + lane_xor(send, o);
        }
    }
    for (; o > 0; o >>= 1) v[0] += lane_xor(v[0], o);
    return v[0];
}

__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ ff mad(ff a, ff b, ff c) { return ff_fma(a, b, c); }

// NV: 16-byte words to a string, RW = 16 NV / sizeof(A) rows.  Two, which halve the list reads, while
// the rows still make two groups per SM and two blocks fit on it, and for complex float64 amplitudes,
// whose word holds one row alone (22 qubits 69 us with one, 48 with two); else one.  At most
// 64 registers: two blocks (30 qubits float32 272 us with one, 229 with two).  NT threads: 512, but 256
// up to kRdmFew strings, where a block's few lists leave half the warps idle at its barriers (8 qubits float32
// 14.8 and 13.0 us, 18 qubits, 84 strings, no difference).
constexpr int kRdmFew = 64;
template <typename A, int NV> constexpr int kRdmRows = 16 * NV / (int)sizeof(A);
template <typename A, int NV, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_rdm_rows(const A *__restrict__ C, SectTabs T, int N,
                                                          const uint32_t *__restrict__ lists,
                                                          const int4 *__restrict__ info,
                                                          double *__restrict__ partial) {
    using R = real_of<A>;
    using S = typename RdmSum<R>::T;
    constexpr int RW = kRdmRows<A, NV>, NC = AmpT<A>::kCplx ? 2 : 1, NW = NT / 32;
    struct alignas(16) Word { A v[RW / NV]; };
    extern __shared__ __align__(16) uint8_t rdm_s[];  // [strings][RW] amplitudes, then the pairs' float64 slots
    __shared__ double s_occ[NW][17];
    const int n = 2 * N, npair = N * (N - 1) / 2, Dm = T.Da > T.Db ? T.Da : T.Db;
    Word *buf = reinterpret_cast<Word *>(rdm_s);
    double *slot = reinterpret_cast<double *>(buf + (size_t)Dm * NV);  // [2 npair][RW][NC]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 2 * npair * RW * NC; i += NT) slot[i] = 0.0;
    auto put = [&](int e, double v) {
        partial[(size_t)(2 * e) * gridDim.x + blockIdx.x] = v;
        partial[(size_t)(2 * e + 1) * gridDim.x + blockIdx.x] = 0.0;
    };
    const int na_items = (T.Db + RW - 1) / RW, nb_items = (T.Da + RW - 1) / RW;
    int item = blockIdx.x;  // row groups, then column groups
    for (int s = 0; s < 2; ++s) {
        const int D = s ? T.Db : T.Da, rows = s ? T.Da : T.Db;  // strings of the pairs' spin; rows of them
        const uint16_t *str = s ? T.strb : T.stra;
        const uint32_t *other = s ? T.sa : T.sb;
        const int first = s ? na_items : 0, last = s ? na_items + nb_items : na_items;
        if (item >= last) {  // no group of this pass
            if (threadIdx.x < N) put(1 + 2 * threadIdx.x + s, 0.0);
            if (threadIdx.x == 0 && s == 0) put(0, 0.0);
            continue;
        }
        if (lane < 17) s_occ[warp][lane] = 0.0;
        for (; item < last; item += (int)gridDim.x) {
            const int r0 = (item - first) * RW;
            __syncthreads();  // the last group's reads of buf are done
            if (s == 0) {
                for (int x = threadIdx.x; x < D; x += NT) {
                    #pragma unroll
                    for (int w = 0; w < NV; ++w) {
                        Word v;
                        #pragma unroll
                        for (int j = 0; j < RW / NV; ++j) {
                            const int r = r0 + w * (RW / NV) + j;
                            v.v[j] = r < rows ? C[(size_t)r * T.Da + x] : mka<A>(R(0), R(0));
                        }
                        buf[w * Dm + x] = v;
                    }
                }
            } else {
                A *flat = reinterpret_cast<A *>(buf);
                for (int i = threadIdx.x; i < D * RW; i += NT) {
                    constexpr int WV = RW / NV;
                    const int j = i % RW, r = r0 + j;
                    flat[((j / WV) * Dm + i / RW) * WV + j % WV] = r < rows ? C[(size_t)(i / RW) * T.Da + r] : mka<A>(R(0), R(0));
                }
            }
            __syncthreads();
            // this spin's occupations (and the norm)
            S occ[16], nrm[1] = {S(0)};
            #pragma unroll
            for (int p = 0; p < 16; ++p) occ[p] = S(0);
            for (int x = threadIdx.x; x < D; x += NT) {
                const uint32_t bits = str[x];
                R w = R(0);
                #pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const Word v = buf[k * Dm + x];
                    #pragma unroll
                    for (int j = 0; j < RW / NV; ++j) w += re_dot(v.v[j], v.v[j]);
                }
                sum_to(nrm[0], w);
                #pragma unroll
                for (int p = 0; p < 16; ++p)
                    if ((bits >> p) & 1u) sum_to(occ[p], w);
            }
            const S so = row_sums<16>(occ, lane), sn = row_sums<1>(nrm, lane);
            if (lane % 2 == 0) s_occ[warp][lane / 2] += to_double(so);
            if (lane == 0) s_occ[warp][16] += to_double(sn);
            const uint32_t xo = lane * RW / 32 + r0 < rows ? other[lane * RW / 32 + r0] : 0u;  // this lane's row's string
            // pair k of this spin to warp k % NW
            int p = 0, q = 0;
            for (int k = 0; k < npair; ++k) {
                if (++q == N) { ++p; q = p + 1; }
                if (k % NW != warp) continue;
                // list entry: rank | parity of the string's own bits between << 15 | partner rank << 16
                const int4 li = info[k];
                const uint32_t *L = lists + (s ? li.z : li.x);
                const int cnt = s ? li.w : li.y;
                R acc[RW], ai[RW];
                #pragma unroll
                for (int j = 0; j < RW; ++j) acc[j] = ai[j] = R(0);
                #pragma unroll 2
                for (int i = lane; i < cnt; i += 32) {
                    const uint32_t ea = L[i];
                    if (!(SV_IN_RANGE(ea & 0x7FFFu, D, kChkRank) && SV_IN_RANGE(ea >> 16, D, kChkRank)))
                        continue;  // checked build: skip the entry
                    const bool neg = ((ea >> 15) & 1u) != 0u;
                    #pragma unroll
                    for (int w = 0; w < NV; ++w) {
                        const Word wu = buf[w * Dm + (ea & 0x7FFFu)], wv = buf[w * Dm + (ea >> 16)];
                        #pragma unroll
                        for (int j = 0; j < RW / NV; ++j) {
                            // conj(v) u, the sign on u
                            const A v = wv.v[j], u0 = wu.v[j];
                            const R ux = neg ? -re(u0) : re(u0);
                            const int r = w * (RW / NV) + j;
                            acc[r] = mad(re(v), ux, acc[r]);
                            if constexpr (NC == 2) {
                                const R uy = neg ? -im(u0) : im(u0);
                                acc[r] = mad(im(v), uy, acc[r]);
                                ai[r] = mad(re(v), uy, ai[r]);
                                ai[r] = mad(-im(v), ux, ai[r]);
                            }
                        }
                    }
                }
                const bool flip = par(xo & between(2 * p + s, 2 * q + s)) != 0;
                double *my = slot + ((size_t)(s * npair + k) * RW + lane * RW / 32) * NC;
                const R sr = row_sums<RW>(acc, lane);
                if (lane % (32 / RW) == 0) my[0] += to_double(flip ? -sr : sr);
                if constexpr (NC == 2) {
                    const R si = row_sums<RW>(ai, lane);
                    if (lane % (32 / RW) == 0) my[1] += to_double(flip ? -si : si);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < 17) {
            double t = 0.0;
            for (int w = 0; w < NW; ++w) t += s_occ[w][threadIdx.x];
            if (threadIdx.x < N) put(1 + 2 * threadIdx.x + s, t);
            if (threadIdx.x == 16 && s == 0) put(0, t);
        }
        __syncthreads();
    }
    __syncthreads();  // (a block without groups: the slots were zeroed by other threads)
    for (int e = threadIdx.x; e < 2 * npair; e += NT) {
        double re = 0.0, im = 0.0;
        for (int r = 0; r < RW; ++r) {
            re += slot[((size_t)e * RW + r) * NC];
            if constexpr (NC == 2) im += slot[((size_t)e * RW + r) * NC + 1];
        }
        partial[(size_t)(2 * (1 + n + e)) * gridDim.x + blockIdx.x] = re;
        partial[(size_t)(2 * (1 + n + e) + 1) * gridDim.x + blockIdx.x] = im;
    }
}

// out[i] = C[idx[i]] or 0 when idx[i] is 0xFFFFFFFF (a basis state outside the sector)
template <typename A>
__global__ void k_gather_c(const A *__restrict__ psi, const uint32_t *__restrict__ idx, int count,
                           A *__restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        out[i] = idx[i] == 0xFFFFFFFFu ? mka<A>(0, 0) : psi[idx[i]];
}

// A handle's vector from its compute core's compact amplitudes (Out the handle's type, In the
// core's: the same, or its real one): string pair (a, b) of the core, at ca[a] + cb[b] of the
// vector (dense storage: the storage-space spreads; sector storage: the ranks in its order).
// Without C, zeros.
// Bound: dense, one partly written 32-byte DRAM sector per scattered amplitude.
template <typename Out, typename In>
__global__ void __launch_bounds__(kThreads) k_core_publish(const In *__restrict__ C, Out *__restrict__ psi,
                                                           const uint32_t *__restrict__ ca,
                                                           const uint32_t *__restrict__ cb, int Da, int Db) {
    using R = real_of<Out>;
    for (int Ib = blockIdx.x; Ib < Db; Ib += gridDim.x) {
        const size_t row = (size_t)Ib * Da;
        const uint32_t xb = cb[Ib];
        for (int Ia = blockIdx.y * kThreads + threadIdx.x; Ia < Da; Ia += gridDim.y * kThreads) {
            const In c = C ? C[row + Ia] : In{};
            psi[xb + ca[Ia]] = mka<Out>((R)re(c), (R)im(c));
        }
    }
}

// The other way: the compact amplitudes (their real parts for a real core) of a stored reference.
template <typename Out, typename In>
__global__ void __launch_bounds__(kThreads) k_core_gather(const In *__restrict__ psi, Out *__restrict__ C,
                                                          const uint32_t *__restrict__ ca,
                                                          const uint32_t *__restrict__ cb, int Da, int Db) {
    using R = real_of<Out>;
    for (int Ib = blockIdx.x; Ib < Db; Ib += gridDim.x) {
        const size_t row = (size_t)Ib * Da;
        const uint32_t xb = cb[Ib];
        for (int Ia = blockIdx.y * kThreads + threadIdx.x; Ia < Da; Ia += gridDim.y * kThreads) {
            const In c = psi[xb + ca[Ia]];
            C[row + Ia] = mka<Out>((R)re(c), (R)im(c));
        }
    }
}

// ---------------------------------------------------------------- launchers

// publish: core (core_dtype; NULL: zeros) -> handle (dtype); else the handle's vector -> core.
cudaError_t launch_core_move(void *handle_vec, int dtype, void *core_vec, int core_dtype, bool publish,
                             const uint32_t *ca, const uint32_t *cb, int Da, int Db, int sm_count, cudaStream_t st) {
    if (Da <= 0 || Db <= 0) return cudaSuccess;
    // rows over the grid's x, a row's columns over its y: enough blocks for few long or many short rows
    const int gy = (Da + kThreads - 1) / kThreads, cap = sm_count * 16;
    const dim3 grid(Db < cap ? Db : cap, gy < 8 ? gy : 8);
    if (dtype == core_dtype) {
        SV_DISPATCH_AMP(dtype,
                        if (publish) k_core_publish<A, A><<<grid, kThreads, 0, st>>>((const A *)core_vec, (A *)handle_vec, ca, cb, Da, Db);
                        else k_core_gather<A, A><<<grid, kThreads, 0, st>>>((const A *)handle_vec, (A *)core_vec, ca, cb, Da, Db));
    } else {  // a complex handle with a real core of the same precision
        SV_DISPATCH_AMP(dtype, if constexpr (AmpT<A>::kCplx) {
            using B = real_of<A>;
            if (publish) k_core_publish<A, B><<<grid, kThreads, 0, st>>>((const B *)core_vec, (A *)handle_vec, ca, cb, Da, Db);
            else k_core_gather<B, A><<<grid, kThreads, 0, st>>>((const A *)handle_vec, (B *)core_vec, ca, cb, Da, Db);
        });
    }
    return cudaGetLastError();
}

static SectTabs tabs(const uint32_t *sa, const uint32_t *sb, const uint16_t *stra, const uint16_t *strb,
                     const uint16_t *ra, const uint16_t *rb, int Da, int Db) {
    SectTabs t;
    t.sa = sa; t.sb = sb; t.stra = stra; t.strb = strb; t.ra = ra; t.rb = rb; t.Da = Da; t.Db = Db;
    return t;
}

// Alpha / beta string parts of a qubit-space op.
static void sect_op_from(const OpDesc &d, int N, SectOp *dst) {
    SectOp o;
    o.sm = d.sm;
    o.ma = o.fa = o.mb = o.fb = 0;
    for (int q = 0; q < N; ++q) {
        if ((d.m >> (2 * q)) & 1u) o.ma |= 1u << q;
        if ((d.from >> (2 * q)) & 1u) o.fa |= 1u << q;
        if ((d.m >> (2 * q + 1)) & 1u) o.mb |= 1u << q;
        if ((d.from >> (2 * q + 1)) & 1u) o.fb |= 1u << q;
    }
    *dst = o;
}

// Blocks of the list kernels: one per beta-list entry, at most bps per SM (8 by default).
int sector_grid(int Db, int sm_count, int bps) {
    const int cap = sm_count * (bps > 0 ? bps : 8);
    return Db < cap ? Db : cap;
}

// Host side of the lists: counts from the patterns, offsets, and the build launch.
static uint64_t choose(int n, int k) {
    if (k < 0 || k > n) return 0;
    uint64_t r = 1;
    for (int i = 1; i <= k; ++i) r = r * (uint64_t)(n - k + i) / (uint64_t)i;
    return r;
}

size_t list_op_bytes() { return sizeof(ListOp); }

// Fill the ListOp of op d (qubit-space masks) for a sector with na / nb electrons
// among N orbitals: its alpha list at entry a_off, its beta list right after it.
// Returns the alpha and beta list lengths through na_l, nb_l.
void list_op_from(const OpDesc &d, int N, int na, int nb, uint32_t a_off, void *dst, int *na_l, int *nb_l) {
    SectOp s;
    sect_op_from(d, N, &s);
    *na_l = (int)choose(N - __builtin_popcount(s.ma), na - __builtin_popcount(s.fa));
    *nb_l = (int)choose(N - __builtin_popcount(s.mb), nb - __builtin_popcount(s.fb));
    ListOp o;
    o.sm = s.sm; o.ma = s.ma; o.fa = s.fa; o.mb = s.mb; o.fb = s.fb;
    o.a_off = a_off;
    o.b_off = a_off + (uint32_t)*na_l;
    o.a_n = (uint32_t)*na_l;
    o.b_n = (uint32_t)*nb_l;
    *(ListOp *)dst = o;
}

cudaError_t launch_build_lists(const void *ops, int n_ops, const uint32_t *sa, const uint32_t *sb,
                               const uint16_t *stra, const uint16_t *strb, const uint16_t *ra, const uint16_t *rb,
                               int Da, int Db, uint32_t *out, cudaStream_t st) {
    if (n_ops <= 0) return cudaSuccess;
    SectTabs T = tabs(sa, sb, stra, strb, ra, rb, Da, Db);
    k_build_lists<<<2 * n_ops, kThreads, 0, st>>>((const ListOp *)ops, T, out);
    return cudaGetLastError();
}

cudaError_t launch_rotate_l(void *psi, int dtype, const uint32_t *al, int na_l, const uint32_t *bl, int nb_l, int Da,
                            double c, double s, int grid, cudaStream_t st) {
    if (na_l <= 0 || nb_l <= 0) return cudaSuccess;
    SV_DISPATCH_AMP(dtype, k_rotate_l<A><<<grid, kThreads, 0, st>>>((A *)psi, al, na_l, bl, nb_l, Da,
                                                                     (real_of<A>)c, (real_of<A>)s));
    return cudaGetLastError();
}

// partial: grid doubles (every block writes its entry, zero when it has no rows).
cudaError_t launch_adjoint_l(void *psi, void *lam, int dtype, const uint32_t *al, int na_l, const uint32_t *bl,
                             int nb_l, int Da, double c, double s, int grid, double *partial, cudaStream_t st) {
    SV_DISPATCH_AMP(dtype, k_adjoint_l<A><<<grid, kThreads, 0, st>>>((A *)psi, (A *)lam, al, na_l, bl, nb_l, Da,
                                                                      (real_of<A>)c, (real_of<A>)s, partial));
    return cudaGetLastError();
}

// CL: the interleaved (psi, lam) matrix (launch_interleave), 16-byte aligned.
cudaError_t launch_adjoint_li(void *CL, int dtype, const uint32_t *al, int na_l, const uint32_t *bl, int nb_l, int Da,
                              double c, double s, int grid, double *partial, cudaStream_t st) {
    SV_DISPATCH_AMP(dtype, k_adjoint_li<A><<<grid, kThreads, 0, st>>>((A *)CL, al, na_l, bl, nb_l, Da,
                                                                       (real_of<A>)c, (real_of<A>)s, partial));
    return cudaGetLastError();
}

int rdm_rows_elements(int n) { return 1 + n + (n / 2) * (n / 2 - 1); }

namespace {

// 12,870 strings of 16 bytes and the sums of 16 orbitals' pairs of four rows: 209 KB;
// the static part takes 2,176 bytes.
constexpr size_t kRdmSmemCap = 222 * 1024;

// Words to a string of the sector's amplitudes (of `amp` bytes).
int rdm_words(int amp, int Dm, int sm_count) {
    if (amp == 16) return Dm <= 3 * 1024 ? 2 : 1;
    return Dm <= 3 * 1024 && Dm * amp / 32 >= 2 * sm_count ? 2 : 1;  // two blocks per SM: about 100 KB each
}

template <typename A, int NV>
cudaError_t rdm_rows_nv(const void *C, const SectTabs &T, int N, int grid, const uint32_t *lists, const int *info,
                        double *partial, cudaStream_t st) {
    constexpr int RW = kRdmRows<A, NV>, NC = AmpT<A>::kCplx ? 2 : 1;
    const size_t smem = (size_t)(T.Da > T.Db ? T.Da : T.Db) * 16 * NV + sizeof(double) * (size_t)N * (N - 1) * RW * NC;
    const bool few = (T.Da > T.Db ? T.Da : T.Db) <= kRdmFew;
    const cudaError_t e = few ? allow_smem(k_rdm_rows<A, NV, 256>, kRdmSmemCap) : allow_smem(k_rdm_rows<A, NV, 512>, kRdmSmemCap);
    if (e != cudaSuccess) return e;
    if (few) k_rdm_rows<A, NV, 256><<<grid, 256, smem, st>>>((const A *)C, T, N, lists, (const int4 *)info, partial);
    else k_rdm_rows<A, NV, 512><<<grid, 512, smem, st>>>((const A *)C, T, N, lists, (const int4 *)info, partial);
    return cudaGetLastError();
}

template <typename A>
cudaError_t rdm_rows_of(const void *C, const SectTabs &T, int N, int grid, const uint32_t *lists, const int *info,
                        double *partial, int sm_count, cudaStream_t st) {
    if (rdm_words((int)sizeof(A), T.Da > T.Db ? T.Da : T.Db, sm_count) == 2)
        return rdm_rows_nv<A, 2>(C, T, N, grid, lists, info, partial, st);
    return rdm_rows_nv<A, 1>(C, T, N, grid, lists, info, partial, st);  // at most 12,870 strings: 214 KB
}

}  // namespace

// Blocks: at most bps per SM, one to a group of rows or columns, but no fewer than the strings (28 qubits float32:
// 502 groups on 608 blocks 165 us, on 502 170).  A float64 state's float-float form has its size.
int rdm_rows_grid(int dtype, int Da, int Db, int sm_count, int bps) {
    const int Dm = Da > Db ? Da : Db, amp = (int)amp_size(dtype), rw = 16 * rdm_words(amp, Dm, sm_count) / amp;
    const int cap = sm_count * (bps > 0 ? bps : 4), items = (Da + rw - 1) / rw + (Db + rw - 1) / rw;
    const int want = items > Dm ? items : Dm;
    return want < cap ? want : cap;
}

// partial: [2 n_el][grid] doubles (n_el = rdm_rows_elements(n)), reduced by launch_reduce_rows.
// lists / info: the pair lists and their int4 records, one list op per pair p < q in (p, q) order (for
// each spin flip mask {p, q}, "from" pattern {q}, sign mask the orbitals between).
// ff_form: C holds the float-float form of a float64 state (ffc for complex128, ff for
// float64), as launch_to_ff writes it.
cudaError_t launch_rdm_rows(const void *C, int dtype, int ff_form, int n, const uint32_t *sa, const uint32_t *sb,
                            const uint16_t *stra, const uint16_t *strb, const uint16_t *ra, const uint16_t *rb, int Da,
                            int Db, int grid, const uint32_t *lists, const int *info, double *partial, int sm_count,
                            cudaStream_t st) {
    const SectTabs T = tabs(sa, sb, stra, strb, ra, rb, Da, Db);
    if (ff_form) {
        if (dtype == SV_C128) return rdm_rows_of<ffc>(C, T, n / 2, grid, lists, info, partial, sm_count, st);
        if (dtype == SV_R64) return rdm_rows_of<ff>(C, T, n / 2, grid, lists, info, partial, sm_count, st);
        return cudaErrorInvalidValue;  // single-precision states have no float-float form
    }
    cudaError_t e = cudaErrorInvalidValue;
    SV_DISPATCH_AMP(dtype, e = rdm_rows_of<A>(C, T, n / 2, grid, lists, info, partial, sm_count, st));
    return e;
}

cudaError_t launch_gather_c(const void *psi, int dtype, const uint32_t *idx, int count, void *out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    int grid = (count + kThreads - 1) / kThreads;
    if (grid > 1024) grid = 1024;
    SV_DISPATCH_AMP(dtype, k_gather_c<A><<<grid, kThreads, 0, st>>>((const A *)psi, idx, count, (A *)out));
    return cudaGetLastError();
}

// This unit's check word (checked build), for sv_check_status.
SV_CHECK_READER(check_word_sector)

}  // namespace svk
