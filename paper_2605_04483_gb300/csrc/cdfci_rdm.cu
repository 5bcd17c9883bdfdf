// Sums over pairs of stored determinants a single or double excitation apart:
// spin-summed reduced density matrices of the stored vector, the energy's
// derivatives (Sec. "Optimal Orbital Selections") and the exact Rayleigh
// quotient.
//
//   gamma_pq   = sum_s  <a+_ps a_qs> / c.c
//   Gamma_pqrs = sum_st <a+_ps a+_rt a_st a_qs> / c.c       (chemists' order)
//
// so that E = sum h_pq gamma_pq + 1/2 sum (pq|rs) Gamma_pqrs (Eq. general-ham
// with v_PQRS = (pr|qs)).  A pair J -> I (both with c != 0) contributes
// c_I c_J <I|op|J> to the entries the excitation reaches:
//   I = J                 gamma_pp, Gamma_pprr (direct), Gamma_prrp (exchange)
//   single i -> a         gamma_ai; with every other occupied spin-orbital r:
//                         Gamma_airr, Gamma_rrai, and for the same spin
//                         -Gamma_arri, -Gamma_riar
//   double i->a, j->b     Gamma_aibj, Gamma_bjai; same spin also -Gamma_ajbi,
//                         -Gamma_biaj
// and the reversed pair I -> J to the images under i <-> a, j <-> b.  The
// results are averaged over exactly these symmetries at the end, so each
// unordered pair is met once, in the direction I > J, and adds its four-fold
// weight to one image (twice to gamma).  I > J compares the changed strings,
// the alpha one first, and a string's change raises it exactly when its highest
// changed orbital becomes occupied: a > i for a single, b > j for a double with
// i < j, a < b; so half of the enumeration is never produced.
// The sign <I|a+_a a+_b a_j a_i|J> is that of the sequential excitation i->a,
// j->b.
#include <cuda_runtime.h>

#include <algorithm>

#include "cdfci_internal.cuh"
#include "cdfci_kernels.h"

namespace cdfci {
namespace {

__device__ __forceinline__ int occ_orbital(const ColLists &L, int na, int t) { return t < na ? L.occA[t] : L.occB[t - na]; }

// ---------------------------------------------------------------------------
// The determinants with c != 0 in a hash table of their own, and a bit filter.
//
// Most excitations of a stored determinant are absent or have c = 0, and in the
// solver's table a probe that misses reads more than two random slots at a usual
// load, a warp of 32 probes as many as its unluckiest lane.  So the sums copy the
// nonzeros into a table at most half full (records {A, B, c}, one 32-byte request
// a probe) and test a bit before asking it.  Both go by an exclusive-or hash z,
// one 64-bit word per spin-orbital: z of an excited determinant is that of J
// with two or four words exchanged, so testing an element costs a handful of
// integer instructions.
//   filter 1 (low half of z): in each SM's shared memory;
//   the table (high half): open addressing;
//   filter 2 (high half): in L2, for more determinants than filter 1 can tell.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long orb_word(int t) {      // t: alpha p, 64 + beta p
    return mix64(0x632be59bd9b4e019ull + (unsigned long long)(t + 1) * 0x9e3779b97f4a7c15ull);
}
__device__ __forceinline__ unsigned f1_index(unsigned long long z, unsigned nb1) { return __umulhi((unsigned)z, nb1); }
__device__ __forceinline__ unsigned f2_index(unsigned long long z, unsigned mask2) { return (unsigned)(z >> 32) & mask2; }

__device__ __forceinline__ void ld_slot_cg(const Slot *s, unsigned long long &a, unsigned long long &b, double &c) {
    unsigned long long cb;
    [[maybe_unused]] unsigned long long bb;
    asm volatile("ld.global.cg.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(cb), "=l"(bb) : "l"(s));
    c = __longlong_as_double((long long)cb);
}

// a record {A, B, c}, in one 32-byte request
__device__ __forceinline__ void ld_rec(const PairRec *r, unsigned long long &a, unsigned long long &b, double &c) {
    unsigned long long cb;
    [[maybe_unused]] unsigned long long pad;
    asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(cb), "=l"(pad) : "l"(r));
    c = __longlong_as_double((long long)cb);
}

__global__ void __launch_bounds__(256) k_pair_list(Problem P, IterState *st, PairList L) {
    __shared__ unsigned long long s_z[128];
    if (threadIdx.x < 128) s_z[threadIdx.x] = orb_word(threadIdx.x);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x; i0 < P.capacity; i0 += stride) {
        const long long i = i0 + threadIdx.x;
        unsigned long long a = 0ull, b = 0ull;
        double c = 0.0;
        if (i < P.capacity) ld_slot_cg(P.table + i, a, b, c);
        b &= kKeyMaskB;
        const bool on = (a | b) != 0ull && !is_zero(c);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (!m) continue;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(L.n, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (!on) continue;
        const unsigned long long pos = base + (unsigned)__popc(m & ((1u << lane) - 1u));
        if (pos >= L.cap) continue;                     // the caller sees n > cap and lists again
        unsigned long long z = 0ull;
        for (unsigned long long x = a; x; x &= x - 1) z ^= s_z[__ffsll((long long)x) - 1];
        for (unsigned long long x = b; x; x &= x - 1) z ^= s_z[64 + __ffsll((long long)x) - 1];
        if (L.nb1) {
            const unsigned k = f1_index(z, L.nb1);
            atomicOr(L.f1 + (k >> 5), 1u << (k & 31));
        }
        if (!L.nb1) {
            const unsigned k2 = f2_index(z, L.mask2);
            atomicOr(L.f2 + (k2 >> 5), 1u << (k2 & 31));
        }
        unsigned at = (unsigned)(z >> 32) & L.imask, probe = 0;
        for (; probe <= L.imask; ++probe) {
            if (atomicCAS(&L.rec[at].tag, 0ull, 1ull) == 0ull) break;   // claimed: read by later launches only
            at = (at + 1) & L.imask;
        }
        if (probe <= L.imask) {
            L.rec[at].a = a;
            L.rec[at].b = b;
            L.rec[at].c = c;
            L.pos[pos] = at;
        }
        if (probe > L.imask) set_status(st, kErrInternal);
    }
}

// The number of determinants with c != 0.
__global__ void __launch_bounds__(256) k_count_nonzero(Problem P, unsigned long long *n) {
    unsigned long long mine = 0ull;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P.capacity; i += (long long)gridDim.x * blockDim.x) {
        unsigned long long a, b;
        double c;
        ld_slot_cg(P.table + i, a, b, c);
        mine += ((a | b) != 0ull && !is_zero(c)) ? 1 : 0;
    }
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(n, mine);
}

// visit(A, B, c) for every determinant with c != 0 of this warp's share: of the list, or where there is none
// of the solver's table (32 slots a load).  The whole warp calls it together.
template <bool kListed, class Visit>
__device__ __forceinline__ void for_each_nonzero(const Problem &P, const PairList &Q, const Visit &visit) {
    const int lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const unsigned w0 = blockIdx.x * nwarps + (threadIdx.x >> 5), step = gridDim.x * nwarps;
    if (kListed) {
        const unsigned n = (unsigned)(*Q.n < Q.cap ? *Q.n : Q.cap);
        for (unsigned at = w0; at < n; at += step) {
            const PairRec J = Q.rec[Q.pos[at]];
            visit(J.a, J.b, J.c);
        }
        return;
    }
    for (long long s0 = 32ll * w0; s0 < P.capacity; s0 += 32ll * step) {
        unsigned long long a = 0ull, b = 0ull;
        double c = 0.0;
        if (s0 + lane < P.capacity) ld_slot_cg(P.table + s0 + lane, a, b, c);
        b &= kKeyMaskB;
        for (unsigned m = __ballot_sync(0xffffffffu, (a | b) != 0ull && !is_zero(c)); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            visit(__shfl_sync(0xffffffffu, a, src), __shfl_sync(0xffffffffu, b, src), __shfl_sync(0xffffffffu, c, src));
        }
    }
}

// An excitation met with both determinants stored.
struct PairHit {
    int kind;                          // 0 single alpha, 1 single beta, 2 double aa, 3 double bb, 4 double ab
    int i, a, j, b;
    unsigned parity;                   // 1: the sign is negative
};

// What a pair adds to the density matrices (raw sums, see the head of this file).
struct RdmSink {
    double *g1, *g2;
    __device__ __forceinline__ void start(const Problem &, const ColLists &, double) {}
    __device__ __forceinline__ void hit(const Problem &P, const ColLists &L, const PairHit &x, double cJ, double cI) {
        const int N = P.N, N2 = N * N;
        const double v = apply_parity(cI * cJ, x.parity);
        const int i = x.i, a = x.a;
        const double v4 = 4.0 * v;
        if (x.kind <= 1) {
            atomicAdd(&g1[a * N + i], 2.0 * v);
            const int ne = P.na + P.nb;
            for (int t = 0; t < ne; ++t) {
                const int ts = t < P.na ? 0 : 1;
                const int r = occ_orbital(L, P.na, t);
                if (ts == x.kind && r == i) continue;
                atomicAdd(&g2[(a * N + i) * N2 + r * N + r], v4);
                if (ts == x.kind) atomicAdd(&g2[(a * N + r) * N2 + r * N + i], -v4);
            }
        } else {
            atomicAdd(&g2[(a * N + i) * N2 + x.b * N + x.j], v4);
            if (x.kind <= 3) atomicAdd(&g2[(a * N + x.j) * N2 + x.b * N + i], -v4);
        }
    }
    __device__ __forceinline__ void finish(int, int) {}
};

// c^T H c and c.c: each lane's share of sum_J c_J (H_JJ c_J + 2 sum_{I > J} H_IJ c_I)
struct QuotientSink {
    double *partial;                   // per warp: its sums
    double num, den;
    __device__ __forceinline__ void start(const Problem &P, const ColLists &L, double cJ) {
        const double d = diag_warp(P, L);
        if ((threadIdx.x & 31) == 0) {
            num = fma(cJ, d * cJ, num);
            den = fma(cJ, cJ, den);
        }
    }
    __device__ __forceinline__ void hit(const Problem &P, const ColLists &L, const PairHit &x, double cJ, double cI) {
        const int N = P.N;
        double v;
        if (x.kind <= 1) {
            const size_t at = (size_t)(x.i * N + x.a) * N;
            const double *tA = (x.kind == 0 ? P.W3 : P.V3) + at, *tB = (x.kind == 0 ? P.V3 : P.W3) + at;
            v = __ldg(P.h + x.i * N + x.a);
            for (int k = 0; k < P.na; ++k) v += __ldg(tA + L.occA[k]);
            for (int k = 0; k < P.nb; ++k) v += __ldg(tB + L.occB[k]);
        } else if (x.kind <= 3) {
            v = gi(P.g, N, x.i, x.a, x.j, x.b) - gi(P.g, N, x.i, x.b, x.j, x.a);
        } else {
            v = gi(P.g, N, x.i, x.a, x.j, x.b);
        }
        num = fma(2.0 * cJ * cI, apply_parity(v, x.parity), num);
    }
    __device__ __forceinline__ void finish(int slot, int lane) {
        double a = num, b = den;
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
        if (lane == 0) {
            partial[2 * slot] = a;
            partial[2 * slot + 1] = b;
        }
    }
};

// Shared memory of k_pairs: filter 1, the orbital words, then per warp the
// single excitations (half of the hash that the filter of the loop uses, and
// sign | i << 8 | a << 16 | (a > i) << 24) of the alpha string that raise it and
// of the beta string, the orbital lists and the queue.
constexpr int kPairU = 8;               // alpha singles, or occupied pairs, per item
constexpr int kPairQ = 32 * kPairU + 32;
__host__ __device__ __forceinline__ size_t pair_warp_bytes(int nsA, int nsB) {
    return (((size_t)(nsA + nsB) * 8 + 15) & ~(size_t)15) + sizeof(ColLists) + kPairQ * 4;
}

// One warp per determinant J of the list.  Its excitations I > J are produced
// in items of up to 32 x kPairU elements (opposite-spin doubles: one beta single
// per lane times kPairU alpha singles; same-spin doubles: one virtual pair per
// lane times kPairU occupied pairs; singles: one per lane); the ones whose bit
// is set join the warp's queue as (kind, x, y), and the queue is looked up 32 at
// a time, every lane its own element.
// How an element is found: by filter 1 (shared memory) in the loop, then the
// list's table; by filter 2 (L2) in the loop, then that table; or, where there is
// no room for a list, without a filter in the solver's table.
enum { kFindF1, kFindF2, kFindSlots };
template <class Sink, int kFind>
__global__ void __launch_bounds__(1024, 1) k_pairs(Problem P, IterState *st, PairList Q, Sink sink, int singles_only) {
    constexpr bool kF1 = kFind == kFindF1;
    extern __shared__ __align__(16) unsigned char s_raw[];
    unsigned *s_f = reinterpret_cast<unsigned *>(s_raw);
    const unsigned nw1 = kF1 ? Q.nb1 / 32 : 0;
    unsigned long long *s_z = reinterpret_cast<unsigned long long *>(s_raw + (((size_t)nw1 * 4 + 15) & ~(size_t)15));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nsA = P.na * P.va, nsB = P.nb * P.vb;
    unsigned char *mine = reinterpret_cast<unsigned char *>(s_z + 128) + (size_t)warp * pair_warp_bytes(nsA, nsB);
    unsigned *hs = reinterpret_cast<unsigned *>(mine), *info = hs + (nsA + nsB);
    ColLists &L = *reinterpret_cast<ColLists *>(mine + (((size_t)(nsA + nsB) * 8 + 15) & ~(size_t)15));
    unsigned *queue = reinterpret_cast<unsigned *>(&L + 1);
    for (unsigned t = threadIdx.x; t < nw1; t += blockDim.x) s_f[t] = Q.f1[t];
    if (threadIdx.x < 128) s_z[threadIdx.x] = orb_word(threadIdx.x);
    __syncthreads();
    const int N = P.N;
    auto half = [](unsigned long long z) { return kF1 ? (unsigned)z : (unsigned)(z >> 32); };
    auto zA = [&](int p) { return half(s_z[p]); };
    auto zB = [&](int p) { return half(s_z[64 + p]); };
    auto maybe = [&](unsigned h) {                      // the filter bit of an element
        if (kFind == kFindSlots) return true;
        const unsigned k = kF1 ? __umulhi(h, Q.nb1) : (h & Q.mask2);
        const unsigned w = kF1 ? s_f[k >> 5] : __ldg(Q.f2 + (k >> 5));
        return ((w >> (k & 31)) & 1u) != 0u;
    };
    for_each_nonzero<kFind != kFindSlots>(P, Q, [&](unsigned long long A, unsigned long long B, double cJ) {
        unsigned long long zJ = 0ull;
        for (int t = lane; t < N; t += 32) {
            const int ra = __popcll(A & low_mask(t)), rb = __popcll(B & low_mask(t));
            if ((A >> t) & 1ull) { L.occA[ra] = (unsigned char)t; zJ ^= s_z[t]; } else L.virA[t - ra] = (unsigned char)t;
            if ((B >> t) & 1ull) { L.occB[rb] = (unsigned char)t; zJ ^= s_z[64 + t]; } else L.virB[t - rb] = (unsigned char)t;
        }
        for (int o = 16; o > 0; o >>= 1) zJ ^= __shfl_xor_sync(0xffffffffu, zJ, o);
        __syncwarp();
        sink.start(P, L, cJ);
        // the single excitations: alpha ones with a > i (compacted), then every beta one
        int nA = 0;
        for (int s0 = 0; s0 < nsA; s0 += 32) {
            const int s = s0 + lane;
            int i = 0, a = -1;
            if (s < nsA) {
                const int o = (int)fdiv((unsigned)s, P.mg_va);
                i = L.occA[o];
                a = L.virA[s - o * P.va];
            }
            const unsigned up = __ballot_sync(0xffffffffu, a > i);
            if (a > i) {
                const int k = nA + __popc(up & ((1u << lane) - 1u));
                hs[k] = zA(i) ^ zA(a);
                info[k] = (unsigned)(__popcll(A & between_mask(i, a)) & 1) | (unsigned)i << 8 | (unsigned)a << 16;
            }
            nA += __popc(up);
        }
        for (int s = lane; s < nsB; s += 32) {
            const int o = (int)fdiv((unsigned)s, P.mg_vb);
            const int i = L.occB[o], a = L.virB[s - o * P.vb];
            hs[nsA + s] = zB(i) ^ zB(a);
            info[nsA + s] = (unsigned)(__popcll(B & between_mask(i, a)) & 1) | (unsigned)i << 8 | (unsigned)a << 16 |
                            (a > i ? 1u << 24 : 0u);
        }
        __syncwarp();
        const unsigned hJ = half(zJ);
        int qn = 0;
        auto push = [&](bool on, unsigned code) {
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if (on) queue[qn + __popc(m & ((1u << lane) - 1u))] = code;
            qn += __popc(m);
        };
        // items: type 0 singles, 1 aa, 2 bb, 3 ab; `row` the first lane's element, `col` the looped factor
        int type = 0, row = 0, col = 0;
        while (true) {
            if (type == 0) {
                if (row < nA + nsB) {
                    const int s = row + lane;
                    const bool al = s < nA, in = s < nA + nsB;
                    const int e = al ? s : nsA + s - nA;
                    const bool on = in && (al || (info[in ? e : 0] >> 24)) && maybe(hJ ^ hs[in ? e : 0]);
                    push(on, al ? (unsigned)s << 12 : (1u << 24) | (unsigned)(s - nA));
                    row += 32;
                } else {
                    type = singles_only ? 4 : 1;
                    row = col = 0;
                }
            } else if (type <= 2) {
                const bool alpha = type == 1;
                const int cv2 = alpha ? P.cva2 : P.cvb2, co2 = alpha ? P.ca2 : P.cb2;
                if (row < cv2 && co2 > 0) {
                    const int vp = row + lane;
                    const bool in = vp < cv2;
                    const unsigned pv = __ldg((alpha ? P.pair_va : P.pair_vb) + (in ? vp : 0));
                    const unsigned char *occ = alpha ? L.occA : L.occB, *vir = alpha ? L.virA : L.virB;
                    const int va = vir[pv & 0xff], vb = vir[pv >> 8];
                    const unsigned hv = hJ ^ (alpha ? zA(va) ^ zA(vb) : zB(va) ^ zB(vb));
#pragma unroll
                    for (int u = 0; u < kPairU; ++u) {
                        const int op = col + u;
                        if (op >= co2) break;           // uniform
                        const unsigned po = __ldg((alpha ? P.pair_oa : P.pair_ob) + op);
                        const int oi = occ[po & 0xff], oj = occ[po >> 8];
                        push(in && vb > oj && maybe(hv ^ (alpha ? zA(oi) ^ zA(oj) : zB(oi) ^ zB(oj))),
                             (alpha ? 2u << 24 : 3u << 24) | (unsigned)op << 12 | (unsigned)vp);
                    }
                    col += kPairU;
                    if (col >= co2) { col = 0; row += 32; }
                } else {
                    ++type;
                    row = col = 0;
                }
            } else if (type == 3) {
                if (row < nsB && nA > 0) {
                    const int sb = row + lane;
                    const bool in = sb < nsB;
                    const unsigned hb = hJ ^ hs[nsA + (in ? sb : 0)];
#pragma unroll
                    for (int u = 0; u < kPairU; ++u) {
                        const int sa = col + u;
                        if (sa >= nA) break;            // uniform
                        push(in && maybe(hb ^ hs[sa]), (4u << 24) | (unsigned)sa << 12 | (unsigned)sb);
                    }
                    col += kPairU;
                    if (col >= nA) { col = 0; row += 32; }
                } else {
                    type = 4;
                }
            }
            // the queue's lookups
            while (qn >= 32 || (type == 4 && qn > 0)) {
                __syncwarp();
                const int cnt = min(qn, 32);
                qn -= cnt;
                if (lane < cnt) {
                    const unsigned code = queue[qn + lane];
                    const int cx = (int)((code >> 12) & 0xfffu), cy = (int)(code & 0xfffu);
                    PairHit x;
                    x.kind = (int)(code >> 24);
                    unsigned long long oa = A, ob = B;
                    unsigned long long z = zJ;
                    if (x.kind == 2 || x.kind == 3) {
                        const bool alpha = x.kind == 2;
                        const unsigned po = __ldg((alpha ? P.pair_oa : P.pair_ob) + cx);
                        const unsigned pv = __ldg((alpha ? P.pair_va : P.pair_vb) + cy);
                        const unsigned char *occ = alpha ? L.occA : L.occB, *vir = alpha ? L.virA : L.virB;
                        x.i = occ[po & 0xff]; x.j = occ[po >> 8];
                        x.a = vir[pv & 0xff]; x.b = vir[pv >> 8];
                        const unsigned long long X = alpha ? A : B;
                        const unsigned long long X1 = X ^ (1ull << x.i) ^ (1ull << x.a);
                        const unsigned long long X2 = X1 ^ (1ull << x.j) ^ (1ull << x.b);
                        x.parity = (unsigned)(__popcll(X & between_mask(x.i, x.a)) + __popcll(X1 & between_mask(x.j, x.b))) & 1u;
                        if (alpha) oa = X2; else ob = X2;
                        const int o = alpha ? 0 : 64;
                        z ^= s_z[o + x.i] ^ s_z[o + x.a] ^ s_z[o + x.j] ^ s_z[o + x.b];
                    } else {
                        x.parity = 0u;
                        x.i = x.a = x.j = x.b = 0;
                        if (x.kind != 1) {              // an alpha single
                            const unsigned f = info[cx];
                            x.i = (f >> 8) & 0xff; x.a = (f >> 16) & 0xff;
                            x.parity = f & 1u;
                            oa ^= (1ull << x.i) | (1ull << x.a);
                            z ^= s_z[x.i] ^ s_z[x.a];
                        }
                        if (x.kind != 0) {              // a beta single
                            const unsigned f = info[nsA + cy];
                            const int j = (f >> 8) & 0xff, b = (f >> 16) & 0xff;
                            x.parity ^= f & 1u;
                            ob ^= (1ull << j) | (1ull << b);
                            z ^= s_z[64 + j] ^ s_z[64 + b];
                            if (x.kind == 1) { x.i = j; x.a = b; } else { x.j = j; x.b = b; }
                        }
                    }
                    double cI = 0.0;
                    if (kFind == kFindSlots) {
                        bool ins = false;
                        const long long at = table_find(P, st, oa, ob, false, &ins);
                        if (at >= 0) cI = __ldcg(&P.table[at].c);
                    } else {
                        unsigned pos = (unsigned)(z >> 32) & Q.imask;
                        for (unsigned probe = 0; probe <= Q.imask; ++probe) {
                            unsigned long long ka, kb;
                            double c;
                            ld_rec(Q.rec + pos, ka, kb, c);
                            if (ka == oa && kb == ob) { cI = c; break; }
                            if ((ka | kb) == 0ull) break;
                            pos = (pos + 1) & Q.imask;
                        }
                    }
                    if (!is_zero(cI)) sink.hit(P, L, x, cJ, cI);
                }
                __syncwarp();
            }
            if (type == 4) break;
        }
        __syncwarp();
    });
    sink.finish((int)(blockIdx.x * nwarps + warp), lane);
}

// The number-operator terms: S_PQ = sum_J c_J^2 n_P n_Q over the pairs P <= Q
// of spin-orbitals (alpha p, then beta p), which give gamma_pp, Gamma_pprr and
// Gamma_prrp, and c.c.  A warp adds the occupied pairs of its determinants to an
// array of its own in shared memory: one lane per pair, so no two lanes of a
// determinant meet, and the FP64 pipe (two lanes a cycle here) sees only the
// pairs that are occupied (testing every pair of spin-orbitals in registers took
// 540 us for 300 k determinants of 10 electrons in 32 spin-orbitals).
__host__ __device__ __forceinline__ size_t diag_warp_bytes(int N) { return ((size_t)N * (2 * N + 1) + 16) * sizeof(double); }
template <bool kListed>
__global__ void __launch_bounds__(256) k_rdm_diag(Problem P, PairList Q, double *g1, double *g2, double *norm) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int N = P.N, NS = 2 * N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int npairs = NS * (NS + 1) / 2, ne = P.na + P.nb, nep = ne * (ne + 1) / 2;
    double *s = reinterpret_cast<double *>(s_raw + (size_t)warp * diag_warp_bytes(N));
    unsigned char *occ = reinterpret_cast<unsigned char *>(s + npairs);            // 128 bytes
    unsigned short *uv = reinterpret_cast<unsigned short *>(s_raw + (size_t)nwarps * diag_warp_bytes(N));
    for (int t = threadIdx.x; t < nep; t += blockDim.x) {                          // pairs u <= v of occupied positions
        int v = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
        while (v * (v + 1) / 2 > t) --v;
        while ((v + 1) * (v + 2) / 2 <= t) ++v;
        uv[t] = (unsigned short)((t - v * (v + 1) / 2) | v << 8);
    }
    for (int t = lane; t < npairs; t += 32) s[t] = 0.0;
    __syncthreads();
    double nrm = 0.0;
    for_each_nonzero<kListed>(P, Q, [&](unsigned long long A, unsigned long long B, double cJ) {
        const double c2 = cJ * cJ;
        nrm += c2;
        for (int t = lane; t < N; t += 32) {
            if ((A >> t) & 1ull) occ[__popcll(A & low_mask(t))] = (unsigned char)t;
            if ((B >> t) & 1ull) occ[P.na + __popcll(B & low_mask(t))] = (unsigned char)(N + t);
        }
        __syncwarp();
        for (int t = lane; t < nep; t += 32) {
            const int p = occ[uv[t] & 0xff], q = occ[uv[t] >> 8];                  // p <= q
            s[q * (q + 1) / 2 + p] += c2;
        }
        __syncwarp();
    });
    if (lane == 0 && nrm != 0.0) atomicAdd(norm, nrm);
    // the block's sums, each pair once
    __syncthreads();
    for (int t = threadIdx.x; t < npairs; t += blockDim.x) {
        double v = 0.0;
        for (int w = 0; w < nwarps; ++w) v += reinterpret_cast<const double *>(s_raw + (size_t)w * diag_warp_bytes(N))[t];
        if (v == 0.0) continue;
        int Q0 = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
        while (Q0 * (Q0 + 1) / 2 > t) --Q0;
        while ((Q0 + 1) * (Q0 + 2) / 2 <= t) ++Q0;
        const int P0 = t - Q0 * (Q0 + 1) / 2;
        const int p = P0 < N ? P0 : P0 - N, r = Q0 < N ? Q0 : Q0 - N;
        if (P0 == Q0) {
            atomicAdd(&g1[p * N + p], v);
            continue;
        }
        // both orders of the pair: (pp|rr) and (rr|pp), for one spin also the exchange
        atomicAdd(&g2[(size_t)(p * N + p) * N * N + r * N + r], 2.0 * v);
        if ((P0 < N) == (Q0 < N)) atomicAdd(&g2[(size_t)(p * N + r) * N * N + r * N + p], -2.0 * v);
    }
}

// the warps' sums added in a fixed order (thread-strided, then a tree), and the quotient
__global__ void __launch_bounds__(1024) k_rq_final(const double *partial, int n, double *out) {
    __shared__ double s_a[32], s_b[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        a += partial[2 * i];
        b += partial[2 * i + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) { s_a[warp] = a; s_b[warp] = b; }
    __syncthreads();
    if (warp != 0) return;
    a = s_a[lane];
    b = s_b[lane];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) out[0] = a / b;
}

// gamma and Gamma divided by c.c, averaged over the symmetries a real
// wavefunction gives them exactly (gamma_pq = gamma_qp; Gamma_pqrs = Gamma_rspq
// = Gamma_qpsr = Gamma_srqp), which removes the rounding asymmetry of the sums.
__global__ void k_rdm_finalize(int N, const double *g1, const double *g2, const double *norm, double *o1, double *o2) {
    const double inv = 1.0 / *norm;
    const int N2 = N * N;
    const long long N4 = (long long)N2 * N2;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < N4 + N2; t += (long long)gridDim.x * blockDim.x) {
        if (t < N2) {
            const int p = (int)t / N, q = (int)t - p * N;
            o1[t] = 0.5 * (g1[p * N + q] + g1[q * N + p]) * inv;
            continue;
        }
        const long long u = t - N2;
        const int s = (int)(u % N), r = (int)((u / N) % N), q = (int)((u / N2) % N), p = (int)(u / ((long long)N2 * N));
        const double v = (g2[((p * N + q) * N + r) * N + s] + g2[((r * N + s) * N + p) * N + q]) +
                         (g2[((q * N + p) * N + s) * N + r] + g2[((s * N + r) * N + q) * N + p]);
        o2[u] = 0.25 * v * inv;
    }
}

// dE/dh = gamma; dE/dg = 1/2 Gamma averaged over the 8-fold permutation
// group of (pq|rs) (the derivative along 8-fold symmetric perturbations);
// F_pq = sum_r h_pr gamma_qr + sum_rst (pr|st) Gamma_qrst, one block per
// (p, q) with a fixed-order block sum; dE/dkappa = 2 (F - F^T) in a second pass.
__global__ void k_grad_dg(int N, const double *G2, double *dg) {
    const int N2 = N * N;
    const long long N4 = (long long)N2 * N2;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < N4; u += (long long)gridDim.x * blockDim.x) {
        const int s = (int)(u % N), r = (int)((u / N) % N), q = (int)((u / N2) % N), p = (int)(u / ((long long)N2 * N));
        auto at = [&](int a, int b, int c, int d) { return G2[((a * N + b) * N + c) * N + d]; };
        const double v = ((at(p, q, r, s) + at(q, p, r, s)) + (at(p, q, s, r) + at(q, p, s, r))) +
                         ((at(r, s, p, q) + at(s, r, p, q)) + (at(r, s, q, p) + at(s, r, q, p)));
        dg[u] = 0.0625 * v;
    }
}

__global__ void __launch_bounds__(256) k_grad_F(int N, const double *h, const double *g, const double *G1,
                                                const double *G2, double *F) {
    __shared__ double red[256];
    const int p = blockIdx.x / N, q = blockIdx.x - (blockIdx.x / N) * N;
    const int N3 = N * N * N;
    double acc = 0.0;
    for (int t = threadIdx.x; t < N3; t += blockDim.x) acc = fma(g[(size_t)p * N3 + t], G2[(size_t)q * N3 + t], acc);
    if (threadIdx.x < N) acc = fma(h[p * N + threadIdx.x], G1[q * N + threadIdx.x], acc);
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) F[blockIdx.x] = red[0];
}

__global__ void k_grad_kappa(int N, const double *F, double *dk) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < N * N; t += gridDim.x * blockDim.x) {
        const int p = t / N, q = t - p * N;
        dk[t] = 2.0 * (F[p * N + q] - F[q * N + p]);
    }
}

}  // namespace

// Blocks of k_pairs: as many warps as fit beside the filter, one block per SM
// (or fewer when the list is short).
struct PairShape {
    int warps, blocks;
    size_t smem;
};
constexpr size_t kPairSmem = 224 * 1024, kPairWarpSmem = 112 * 1024;
static int pair_warps(const Problem &P) {
    const size_t per = pair_warp_bytes(P.na * P.va, P.nb * P.vb);
    int w = 32;
    while (w > 1 && (size_t)w * per > kPairWarpSmem) w >>= 1;
    return w;
}
static PairShape pair_shape(const Problem &P, const PairList &Q) {
    PairShape s;
    s.warps = pair_warps(P);
    s.smem = (((size_t)Q.nb1 / 8 + 15) & ~(size_t)15) + 128 * sizeof(unsigned long long) +
             (size_t)s.warps * pair_warp_bytes(P.na * P.va, P.nb * P.vb);
    s.blocks = (int)std::max<long long>(1, std::min<long long>(152, ((long long)Q.est + s.warps - 1) / s.warps));
    return s;
}

// Sizes for about `est` determinants.  Filter 1 takes 32 bits a determinant up
// to what shared memory leaves; below one bit a determinant (two of three
// elements would pass) filter 2 takes its place, with 32 bits a determinant, at
// most 2^28.  The table has at least 2 records a determinant.
void pair_sizes(const Problem &P, long long est, PairList *Q) {
    const size_t used = 128 * sizeof(unsigned long long) + (size_t)pair_warps(P) * pair_warp_bytes(P.na * P.va, P.nb * P.vb);
    const long long room = used + 4096 < kPairSmem ? (long long)(kPairSmem - used - 16) / 128 * 1024 : 0;
    const long long want = std::max<long long>(1024, (32 * est + 1023) / 1024 * 1024);
    const long long b1 = std::min(want, room);
    Q->nb1 = b1 >= est ? (unsigned)b1 : 0u;
    unsigned long long b2 = 1ull << 15;
    while (b2 < 32ull * (unsigned long long)est && b2 < (1ull << 28)) b2 <<= 1;
    Q->mask2 = Q->nb1 ? 31u : (unsigned)(b2 - 1);
    unsigned long long ni = 1024;
    while (ni < 2ull * (unsigned long long)est) ni <<= 1;
    Q->imask = (unsigned)(ni - 1);
    Q->cap = Q->est = (unsigned)est;
}

cudaError_t launch_count_nonzero(const Problem &P, unsigned long long *n, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(n, 0, sizeof(*n), s);
    if (e != cudaSuccess) return e;
    k_count_nonzero<<<(unsigned)std::min<long long>((P.capacity + 255) / 256, 152 * 8), 256, 0, s>>>(P, n);
    return cudaGetLastError();
}

// (everything that starts at zero, up to `end`, in one call: six took a sixth of the RDMs of 20 determinants)
static cudaError_t launch_pair_list(const Problem &P, IterState *st, const PairList &Q, const void *end, cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(Q.zero, 0, (size_t)(static_cast<const unsigned char *>(end) - Q.zero), s);
    if (e != cudaSuccess || !Q.rec) return e;
    long long grid = (P.capacity + 255) / 256;
    if (grid > 152 * 8) grid = 152 * 8;
    k_pair_list<<<(unsigned)grid, 256, 0, s>>>(P, st, Q);
    return cudaGetLastError();
}

template <class Sink>
static cudaError_t launch_pairs(const Problem &P, IterState *st, const PairList &Q, const Sink &sink, int singles_only,
                                cudaStream_t s) {
    const PairShape g = pair_shape(P, Q);
    auto kernel = !Q.rec ? k_pairs<Sink, kFindSlots> : (Q.nb1 ? k_pairs<Sink, kFindF1> : k_pairs<Sink, kFindF2>);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem);
    if (e != cudaSuccess) return e;
    kernel<<<g.blocks, 32 * g.warps, g.smem, s>>>(P, st, Q, sink, singles_only);
    return cudaGetLastError();
}

cudaError_t launch_rdm(const Problem &P, IterState *st, const PairList &Q, double *g1_raw, double *g2_raw,
                       double *norm, double *g1, double *g2, cudaStream_t s) {
    const int N = P.N;
    const size_t n2 = (size_t)N * N, n4 = n2 * n2;
    if (reinterpret_cast<unsigned char *>(g1_raw) != Q.zero_end || g2_raw != g1_raw + n2 || norm != g2_raw + n4)
        return cudaErrorInvalidValue;
    cudaError_t e = launch_pair_list(P, st, Q, norm + 1, s);
    if (e == cudaSuccess) e = launch_pairs(P, st, Q, RdmSink{g1_raw, g2_raw}, 0, s);
    if (e != cudaSuccess) return e;
    int dw = 8;                                         // warps a block: their arrays within 100 KB (200 KB for one)
    while (dw > 1 && dw * diag_warp_bytes(N) > 100 * 1024) --dw;
    const size_t dsm = dw * diag_warp_bytes(N) + (size_t)(P.na + P.nb) * (P.na + P.nb + 1);
    auto diag = Q.rec ? k_rdm_diag<true> : k_rdm_diag<false>;
    e = cudaFuncSetAttribute(diag, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    const long long dblocks = std::max<long long>(1, std::min<long long>(152 * 2, ((long long)Q.est + 8 * dw - 1) / (8 * dw)));
    diag<<<(unsigned)dblocks, 32 * dw, dsm, s>>>(P, Q, g1_raw, g2_raw, norm);
    k_rdm_finalize<<<152 * 4, 256, 0, s>>>(N, g1_raw, g2_raw, norm, g1, g2);
    return cudaGetLastError();
}

size_t rq_partials(const Problem &P) { return 152 * (size_t)pair_warps(P); }

cudaError_t launch_rq(const Problem &P, IterState *st, const PairList &Q, double *partial, double *out, cudaStream_t s) {
    cudaError_t e = launch_pair_list(P, st, Q, Q.zero_end, s);
    if (e == cudaSuccess) e = launch_pairs(P, st, Q, QuotientSink{partial, 0.0, 0.0}, P.doubles_vanish, s);
    if (e != cudaSuccess) return e;
    const PairShape g = pair_shape(P, Q);
    k_rq_final<<<1, 1024, 0, s>>>(partial, g.blocks * g.warps, out);
    return cudaGetLastError();
}

cudaError_t launch_gradient(int N, const double *h, const double *g, const double *G1, const double *G2, double *F,
                            double *dh, double *dg, double *dk, cudaStream_t s) {
    const size_t n2 = (size_t)N * N;
    cudaError_t e = cudaSuccess;
    if (dh) e = cudaMemcpyAsync(dh, G1, n2 * sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    if (dg) k_grad_dg<<<152 * 4, 256, 0, s>>>(N, G2, dg);
    if (dk) {
        k_grad_F<<<N * N, 256, 0, s>>>(N, h, g, G1, G2, F);
        k_grad_kappa<<<1, 256, 0, s>>>(N, F, dk);
    }
    return cudaGetLastError();
}

}  // namespace cdfci
