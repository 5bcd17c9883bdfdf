// xCDFCI (Algorithm 3): K + 1 states, one row of C per iteration.
//
// Per iteration two launches (captured in a CUDA graph), each with its serial
// part in the block that finishes last:
//   k_x_choose    argmax over the candidates of ||G_j||_inf, G_j = 4 B_j + 4 C_j S
//                 (ties: the smaller key), by a block argmax and a last-block
//                 reduction in block order, clearing the candidates' marks; then
//                 H_ii, the quartic of problem choose-eta (appendix "Determining
//                 Step Size") and its minimiser eta, C_i += eta G_i;
//   k_x_column    B_j += eta H_ji G_i for the column of i with the row compression
//                 rule, insertion of absent rows, the gather sum_j H_ji C_j per
//                 block, the rows it updated become the next candidates; then
//                 B_i = H_ii C_i + the gather (Eq. recalculate-b, per state) and
//                 the counters.  A block of its own updates S and M
//                 (double-double, one entry per lane) beside it: they are first
//                 read by the next choice.
// What bounds an iteration is the latency of its dependent memory requests and
// FP64 chains (a column of the N = 24 problem is one element a thread).  As four
// launches (selection, preparation with S and M, column, recalculation) it took
// 55.4 us with K + 1 = 4 (N = 24, 6 + 5 electrons), as two 34.1 us; now 29.6 us, with a warp
// for each scheduler's FP64 pipe, H_ii beside the gradient in the step, independent sums over the
// lanes and the loads that start a kernel ahead of its flags.
// The energies (the pencil (M, S)) are computed on request by k_x_energies.
// Each row j occurs once in a column, so B_j is updated by plain loads and
// stores, and every reduction has a fixed order: the iteration is
// deterministic.
#include <algorithm>

#include "cdfci_internal.cuh"
#include "cdfci_kernels.h"

namespace cdfci {

namespace {

struct XBest {
    unsigned long long gbits, a, b;
    long long slot;
};

// |x| as its bit pattern (monotone in |x| for non-negative doubles)
__device__ __forceinline__ unsigned long long x_abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

__device__ __forceinline__ bool x_better(const XBest &x, const XBest &y) {
    if (x.slot < 0) return false;
    if (y.slot < 0) return true;
    return x.gbits > y.gbits || (x.gbits == y.gbits && key_less(x.a, x.b, y.a, y.b));
}


// max_a |B_a + (C S)_a| as a bit pattern (||G_j||_inf / 4, G_j = 4 B_j + 4 C_j S; the
// factor changes no rounding and no order), from the row's C and B halves; a NaN
// counts as zero.  Every FP64 instruction takes its scheduler 64 cycles, so the
// maximum is taken over the bits.
__device__ __forceinline__ unsigned long long x_gnorm(const double (&c)[kXMax], const double (&bb)[kXMax],
                                                      const double *S, int k1) {
    unsigned long long m = 0ull;
#pragma unroll
    for (int a = 0; a < kXMax; ++a) {
        if (a >= k1) break;
        double s = 0.0;
#pragma unroll
        for (int b = 0; b < kXMax; ++b) {
            if (b >= k1) break;
            s = fma(c[b], S[b * k1 + a], s);
        }
        const unsigned long long x = x_abs_bits(bb[a] + s);
        if (x <= 0x7ff0000000000000ull && x > m) m = x;
    }
    return m;
}

// Sums of the k1 values over the warp, the values halved with the lanes: 6 FP64
// additions for up to 4 values and 9 for 8, instead of 5 a value.  Lane l returns
// the sum of value x_sum_of(l, k1); its copies are the lanes of equal result.
__device__ __forceinline__ int x_sum_of(int lane, int k1) {
    return k1 > 4 ? (lane >> 2) : (lane >> 3);
}
__device__ __forceinline__ double x_warp_sums(double (&v)[kXMax], int k1) {
    const int lane = threadIdx.x & 31;
    const unsigned all = 0xffffffffu;
    double x[4];
    int o = 16;
    if (k1 > 4) {                                                    // uniform
        const bool up = lane & 16;
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = (up ? v[q + 4] : v[q]) + __shfl_xor_sync(all, up ? v[q] : v[q + 4], 16);
        o = 8;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = v[q];
    }
    bool up = lane & o;
    const double y0 = (up ? x[2] : x[0]) + __shfl_xor_sync(all, up ? x[0] : x[2], o);
    const double y1 = (up ? x[3] : x[1]) + __shfl_xor_sync(all, up ? x[1] : x[3], o);
    o >>= 1;
    up = lane & o;
    double z = (up ? y1 : y0) + __shfl_xor_sync(all, up ? y0 : y1, o);
    for (o >>= 1; o > 0; o >>= 1) z += __shfl_xor_sync(all, z, o);
    return z;
}

}  // namespace

// Four warps a block, one for each scheduler of an SM: a column of the N = 24
// problem (14.5 k elements) is then a warp a scheduler, where eight warps on half
// the SMs shared their FP64 pipes.
constexpr int kXThreads = 128;

// Row j of C and of B (k1 values each) into cv and bv, all loads in flight
// together: 16-byte loads when k1 is even (each half is then whole pairs, and
// a row starts at a multiple of 16 bytes), else 8-byte ones.  The scatter is
// bound by the number of memory requests its elements make at once.
__device__ __forceinline__ void x_ld32(const double *p, double &a, double &b, double &c, double &d) {
    asm volatile("ld.global.cg.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(p));
}
__device__ __forceinline__ void x_load_row(const double *rows, long long j, int k1, double (&cv)[kXMax],
                                           double (&bv)[kXMax]) {
    const double *r = rows + j * 2 * k1;
    if ((k1 & 3) == 0) {                                             // uniform: 32-byte loads (halves 32-byte aligned)
#pragma unroll
        for (int q = 0; q < kXMax / 4; ++q) {
            double c0 = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0, b0 = 0.0, b1 = 0.0, b2 = 0.0, b3 = 0.0;
            if (4 * q < k1) {
                x_ld32(r + 4 * q, c0, c1, c2, c3);
                x_ld32(r + k1 + 4 * q, b0, b1, b2, b3);
            }
            cv[4 * q] = c0; cv[4 * q + 1] = c1; cv[4 * q + 2] = c2; cv[4 * q + 3] = c3;
            bv[4 * q] = b0; bv[4 * q + 1] = b1; bv[4 * q + 2] = b2; bv[4 * q + 3] = b3;
        }
        return;
    }
    if ((k1 & 1) == 0) {                                             // uniform
        const double2 *r2 = reinterpret_cast<const double2 *>(r);
#pragma unroll
        for (int q = 0; q < kXMax / 2; ++q) {
            double2 c2 = make_double2(0.0, 0.0), b2 = c2;
            if (2 * q < k1) {
                c2 = __ldcg(r2 + q);
                b2 = __ldcg(r2 + k1 / 2 + q);
            }
            cv[2 * q] = c2.x; cv[2 * q + 1] = c2.y;
            bv[2 * q] = b2.x; bv[2 * q + 1] = b2.y;
        }
        return;
    }
#pragma unroll
    for (int a = 0; a < kXMax; ++a) {
        cv[a] = a < k1 ? __ldcg(r + a) : 0.0;
        bv[a] = a < k1 ? __ldcg(r + k1 + a) : 0.0;
    }
}

// H_ii exactly as diag_warp(P, L) computes it (the same terms, per-lane sums
// in the same order, the same tree), with every lane's loads issued before the
// first addition: one round trip for the integrals of up to 16 electrons.
__device__ __forceinline__ double x_diag(const Problem &P, const ColLists &L) {
    const int lane = threadIdx.x & 31;
    const int N = P.N, n = P.na + P.nb, n2 = n * n;
    if (n > 16) return diag_warp(P, L);                               // more than two rounds per lane
    const int ph = lane < n ? (lane < P.na ? L.occA[lane] : L.occB[lane - P.na]) : 0;
    const double hv = lane < n ? __ldg(P.h + ph * (N + 1)) : 0.0;
    double tv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {                                     // t = lane + 128 (k / 4) + 32 (k % 4)
        const int t = lane + 128 * (k >> 2) + 32 * (k & 3);
        tv[k] = 0.0;
        if (t < n2) {
            const int u = t / n, w = t - u * n;
            if (u != w) {
                const bool ua = u < P.na, wa = w < P.na;
                const int p = ua ? L.occA[u] : L.occB[u - P.na];
                const int q = wa ? L.occA[w] : L.occB[w - P.na];
                const double jv = P.J[p * N + q];
                tv[k] = (ua == wa) ? (jv - P.K[p * N + q]) : jv;
            }
        }
    }
    double x = 0.0;
    if (lane < n) x += hv;
    double y4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int t = lane + 128 * (k >> 2) + 32 * (k & 3);
        if (t < n2) {
            const int u = t / n, w = t - u * n;
            if (u != w) y4[k & 3] += tv[k];
        }
    }
    x = fma(0.5, (y4[0] + y4[1]) + (y4[2] + y4[3]), x);
    for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
    return __shfl_sync(0xffffffffu, x, 0);
}

// The step of the chosen row (warps 0 and 1 of a block): H_ii, the quartic and
// eta, the scatter weights, C_i += eta g; c and b of the row as they were are left
// for the update of S and M.  forced >= 0: the start step of row {fA, fB} with g =
// e_forced and eta = 1.  Warp 1 computes H_ii beside the gradient and its products
// and keeps the books beside the update of C; independent sums are spread over
// the lanes (an FP64 instruction costs its issue, not its lanes).
struct XStepShared {
    ColLists L;
    double c[kXMax], g[kXMax], b[kXMax], t[kXMax];
    double eta, gn, Hii;
    int stop;
};
__device__ __forceinline__ void x_pair_sync() { asm volatile("bar.sync 1, 64;" ::: "memory"); }
__device__ void x_step(const Problem &P, XState *xs, IterState *st, double *rows, const double *sS, XStepShared &W,
                       long long s, unsigned long long A, unsigned long long B, int forced) {
    const int k1 = xs->k1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned all = 0xffffffffu;
    double c0 = 0.0, b0 = 0.0, g0 = 0.0;
    if (warp == 1) {
        for (int t = lane; t < P.N; t += 32) {
            const int ra = __popcll(A & low_mask(t)), rb = __popcll(B & low_mask(t));
            if ((A >> t) & 1ull) W.L.occA[ra] = (unsigned char)t; else W.L.virA[t - ra] = (unsigned char)t;
            if ((B >> t) & 1ull) W.L.occB[rb] = (unsigned char)t; else W.L.virB[t - rb] = (unsigned char)t;
        }
        __syncwarp();
        const double Hii = x_diag(P, W.L);
        if (lane == 0) W.Hii = Hii;
        x_pair_sync();
        x_pair_sync();                                                // the step is known
        if (W.stop) return;
        if (lane == 0) {
            xs->slot = s; xs->A = A; xs->B = B;
            xs->eta = W.eta;
            xs->Hii = Hii;
            xs->go = 1;
            if (forced < 0) {
                const double dx = P.theta * xs->dx + (1.0 - P.theta) * fabs(W.eta) * W.gn;   // W.gn = ||g||
                xs->dx = dx;
                xs->iterations += 1;
                if (P.dx_threshold > 0.0 && dx < P.dx_threshold) xs->done = 1;
            }
        }
        return;
    }
    if (lane < k1) {
        c0 = __ldcg(rows + s * 2 * k1 + lane);
        b0 = __ldcg(rows + s * 2 * k1 + k1 + lane);
        W.c[lane] = c0;
        W.b[lane] = b0;
    }
    if (lane == 0) W.stop = 0;
    __syncwarp();
    if (lane < k1) {                                                  // G_a, lane a
        double m = 0.0;
        for (int b = 0; b < k1; ++b) m = fma(W.c[b], sS[b * k1 + lane], m);
        g0 = forced >= 0 ? (lane == forced ? 1.0 : 0.0) : 4.0 * b0 + 4.0 * m;
        W.g[lane] = g0;
    }
    __syncwarp();
    if (lane < k1 && forced < 0) {                                    // (S g)_a, lane a: the term of g S g^T
        double t = 0.0;
        for (int b = 0; b < k1; ++b) t = fma(sS[lane * k1 + b], W.g[b], t);
        W.t[lane] = t;
    }
    __syncwarp();
    // h(eta) = f(C + eta e_i g) - f(C) = w4 eta^4 + w3 eta^3 + w2 eta^2 + w1 eta with w4 = ||g||^4,
    // w3 = 4 ||g||^2 c.g, w2 = 2 H_ii ||g||^2 + 2 (c.g)^2 + 2 ||c||^2 ||g||^2 + 2 g S g^T,
    // w1 = ||g||^2 (the directional derivative).  Lane 0 sums g.g, 1 c.g, 2 c.c, 3 g.(S g).
    const double *x = (lane & 3) == 0 || (lane & 3) == 3 ? W.g : W.c;
    const double *y = (lane & 3) == 3 ? W.t : ((lane & 3) == 2 ? W.c : W.g);
    double d = 0.0;
    if (forced < 0)
        for (int a = 0; a < k1; ++a) d = fma(x[a], y[a], d);
    const double gg = __shfl_sync(all, d, 0), cg = __shfl_sync(all, d, 1), cc = __shfl_sync(all, d, 2);
    const double gSg = __shfl_sync(all, d, 3);
    // In t = eta ||g|| the quartic is monic with O(1) coefficients (w / w4 would grow like
    // 1 / ||g||^2 near convergence and overflow the single-precision root stage):
    // t^4 + 4 (c.u) t^3 + (2 H_ii + 2 (c.u)^2 + 2 ||c||^2 + 2 u S u^T) t^2 + ||g|| t, u = g / ||g||.
    double ign = 1.0, gn = 1.0, v3 = 0.0, part = 0.0, us = 0.0;
    if (forced < 0) {
        ign = rsqrt(gg);
        gn = gg * ign;
        const double cu = cg * ign;
        v3 = 4.0 * cu;
        part = 2.0 * cu * cu;
        us = 2.0 * (gSg * ign) * ign;
    }
    x_pair_sync();
    const double Hii = W.Hii;
    double eta = 1.0;
    bool stop = false;
    if (forced < 0) {
        if (!(gn > 0.0)) {
            // a zero gradient ends the run; gn is NaN where g.g is, or has overflowed (inf times 1 / inf)
            stop = true;
            if (lane == 0) {
                if (gg == 0.0) xs->done = 1;
                else set_status(st, kErrNonfinite);
            }
        } else {
            const double v2 = 2.0 * Hii + part + 2.0 * cc + us;
            eta = line_search_lanes((float)gn, (float)v2, (float)v3, gn, v2, v3) * ign;
            if (!isfinite(eta)) {
                stop = true;
                if (lane == 0) set_status(st, kErrNonfinite);
            }
        }
    }
    if (lane == 0) {
        W.eta = eta;
        W.gn = gn;
        W.stop = stop ? 1 : 0;
    }
    x_pair_sync();
    if (stop) return;                                                 // uniform
    // C_i += eta g (lane a), the scatter weights eta g and their largest magnitude
    const bool on = lane < k1;
    double cn = 0.0, wa = 0.0;
    if (on) {
        cn = fma(eta, g0, c0);
        rows[s * 2 * k1 + lane] = cn;
        wa = eta * g0;
        xs->wv[lane] = wa;
        xs->g[lane] = g0;
        xs->c_old[lane] = c0;
        xs->b_old[lane] = b0;
    }
    const unsigned was = __ballot_sync(all, on && !is_zero(c0));
    const unsigned now = __ballot_sync(all, on && !is_zero(cn));
    unsigned long long wb = x_abs_bits(wa);                           // (finite: eta is, and g with it)
#pragma unroll
    for (int off = kXMax / 2; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(all, wb, off);
        wb = o > wb ? o : wb;
    }
    if (lane == 0) {
        const double wmax = __longlong_as_double((long long)wb);
        xs->nnz_c += (now ? 1 : 0) - (was ? 1 : 0);
        xs->thr = wmax > 0.0 ? (P.tau > 0.0 ? P.tau / wmax : 0.0) : 1.0e308;
    }
}

__global__ void __launch_bounds__(kXThreads) k_x_choose(Problem P, XState *xs, IterState *st, const long long *cand,
                                                        long long cap_cand, double *rows, XBest *bbest,
                                                        unsigned int *counter, int forced, unsigned long long fA,
                                                        unsigned long long fB) {
    __shared__ double sS[kXMax * kXMax];
    __shared__ XBest wb[kXThreads / 32], s_best;
    __shared__ XStepShared W;
    __shared__ bool s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // every load that needs no other first: the flags, S, the count, this thread's first candidate
    const int t0 = blockIdx.x * blockDim.x + tid;
    const dd Sx = tid < kXMax * kXMax ? xs->S[tid] : dd{0.0, 0.0};
    const int k1 = xs->k1, n = xs->n_cand, done = xs->done, status = st->status;
    long long s = t0 < cap_cand ? cand[t0] : 0;
    if (done || status) {
        if (blockIdx.x == 0 && tid == 0) xs->go = 0;                 // no step this iteration
        return;
    }
    if (forced >= 0) {                                               // one block
        if (tid < k1 * k1) sS[tid] = Sx.hi + Sx.lo;
        if (tid == 0) {
            xs->go = 0;
            xs->eta = 0.0;
            bool ins = false;
            const long long at = table_find(P, st, fA, fB, true, &ins);
            if (at >= 0 && ins) { xs->n_slots += 1; xs->inserted += 1; }
            s_best.slot = at;
        }
        __syncthreads();
        if (s_best.slot >= 0 && warp <= 1) x_step(P, xs, st, rows, sS, W, s_best.slot, fA, fB, forced);
        return;
    }
    XBest best{0ull, ~0ull, ~0ull, -1};
    double rc[kXMax], rb[kXMax];
    ulonglong2 key = make_ulonglong2(0ull, 0ull);
    if (t0 < n) {
        x_load_row(rows, s, k1, rc, rb);
        key = __ldcg(reinterpret_cast<const ulonglong2 *>(P.table + s));
    }
    if (tid < k1 * k1) sS[tid] = Sx.hi + Sx.lo;
    __syncthreads();
    for (int t = t0; t < n;) {
        P.table[s].b = key.y & kKeyMaskB;                            // no longer a candidate
        const XBest x{x_gnorm(rc, rb, sS, k1), key.x, key.y & kKeyMaskB, s};
        if (x_better(x, best)) best = x;
        t += gridDim.x * blockDim.x;
        if (t < n) {
            s = cand[t];
            x_load_row(rows, s, k1, rc, rb);
            key = __ldcg(reinterpret_cast<const ulonglong2 *>(P.table + s));
        }
    }
    auto warp_best = [&](XBest b) {
        for (int off = 16; off > 0; off >>= 1) {
            XBest y;
            y.gbits = __shfl_xor_sync(0xffffffffu, b.gbits, off);
            y.a = __shfl_xor_sync(0xffffffffu, b.a, off);
            y.b = __shfl_xor_sync(0xffffffffu, b.b, off);
            y.slot = __shfl_xor_sync(0xffffffffu, b.slot, off);
            if (x_better(y, b)) b = y;
        }
        return b;
    };
    best = warp_best(best);
    if (lane == 0) wb[warp] = best;
    __syncthreads();
    if (tid == 0) {
        XBest b = wb[0];
        for (int w = 1; w < kXThreads / 32; ++w)
            if (x_better(wb[w], b)) b = wb[w];
        bbest[blockIdx.x] = b;
        __threadfence();
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || warp > 1) return;
    __threadfence();
    // the last block's warp 0 reduces the blocks' winners (lane l takes blocks l, l + 32, ...), and
    // warps 0 and 1 take the step
    if (warp == 0) {
        XBest b{0ull, ~0ull, ~0ull, -1};
        for (int k = lane; k < (int)gridDim.x; k += 32) {
            const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(bbest + k);
            const ulonglong2 x = __ldcg(q), y = __ldcg(q + 1);
            const XBest z{x.x, x.y, y.x, (long long)y.y};
            if (x_better(z, b)) b = z;
        }
        b = warp_best(b);
        if (lane == 0) {
            *counter = 0u;
            xs->n_cand = 0;
            xs->go = 0;
            xs->eta = 0.0;
            if (b.slot < 0) xs->done = 1;                            // nothing left to choose
            s_best = b;
        }
    }
    x_pair_sync();
    if (s_best.slot >= 0) x_step(P, xs, st, rows, sS, W, s_best.slot, s_best.a, s_best.b, -1);
}

// The slot of key {a, b} by linear probing from pos (no insert), whose first key
// the caller has loaded: -1 absent (pos: the empty slot), -2 error (status set);
// kbo receives the slot's b word, candidate mark included.
__device__ __forceinline__ long long x_find(const Problem &P, IterState *st, unsigned long long a, unsigned long long b,
                                            ulonglong2 k, unsigned long long &pos, unsigned long long &kbo) {
    const bool both_nonzero = (P.na > 0) && (P.nb > 0);
    for (int probe = 0; probe < P.max_probe; ++probe) {
        const Slot *s = P.table + pos;
        if (probe > 0) k = __ldcg(reinterpret_cast<const ulonglong2 *>(s));      // the key in one request
        int spins = 0;
        while (both_nonzero && ((k.x == 0ull) != (k.y == 0ull))) {   // an insert in flight
            if (++spins > (1 << 20)) { set_status(st, kErrTimeout); return -2; }
            k = __ldcg(reinterpret_cast<const ulonglong2 *>(s));
        }
        if (k.x == a && (k.y & kKeyMaskB) == b) { kbo = k.y; return (long long)pos; }
        if (k.x == 0ull && k.y == 0ull) return -1;
        pos = (pos + 1) & P.mask;
    }
    set_status(st, kErrTableFull);
    return -2;
}
// Claims an empty slot for a key that no other thread inserts (each row occurs
// once in a column), from pos on; -1 (status set) when there is none.
__device__ __forceinline__ long long x_claim(const Problem &P, IterState *st, unsigned long long a, unsigned long long b,
                                             unsigned long long pos) {
    for (int probe = 0; probe < P.max_probe; ++probe) {
        unsigned long long oa, ob;
        cas128(&P.table[pos].a, 0ull, 0ull, a, b, oa, ob);
        if (oa == 0ull && ob == 0ull) return (long long)pos;
        pos = (pos + 1) & P.mask;
    }
    set_status(st, kErrTableFull);
    return -1;
}

// S += eta (c^T g + g^T c) + eta^2 g^T g,  M += eta (b^T g + g^T b) + eta^2 H_ii g^T g (one entry per thread)
__device__ void x_update_sm(XState *xs) {
    const int k1 = xs->k1;
    const double eta = xs->eta, Hii = xs->Hii;
    for (int t = threadIdx.x; t < 2 * k1 * k1; t += blockDim.x) {
        const bool isM = t >= k1 * k1;
        const int e = isM ? t - k1 * k1 : t, a = e / k1, b = e - a * k1;
        const double *v = isM ? xs->b_old : xs->c_old;
        const dd e2 = dd_two_prod(eta, eta);
        const dd gab = dd_two_prod(xs->g[a], xs->g[b]);
        const dd q = dd_mul(e2, gab);
        const dd d = dd_add(dd_mul_d(dd_add(dd_two_prod(v[a], xs->g[b]), dd_two_prod(xs->g[a], v[b])), eta),
                            isM ? dd_mul_d(q, Hii) : q);
        dd *to = isM ? xs->M : xs->S;
        to[e] = dd_add(to[e], d);
    }
}

// A single excitation's element as element_value gives it (the same terms in the
// same order) from the tables W3 and V3, eight loads in flight before their adds.
__device__ __forceinline__ double x_single(const Problem &P, unsigned long long A, unsigned long long B, const ElemIdx &x) {
    const size_t row = (size_t)(x.i * P.N + x.a) * P.N;
    const double *tA = (x.kind == 0 ? P.W3 : P.V3) + row, *tB = (x.kind == 0 ? P.V3 : P.W3) + row;
    double v = __ldg(P.h + x.i * P.N + x.a);
    for (unsigned long long mA = A, mB = B; mA | mB;) {
        double t[8];
        bool in[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool fa = mA != 0ull;
            const unsigned long long mm = fa ? mA : mB;
            in[u] = mm != 0ull;
            t[u] = in[u] ? __ldg((fa ? tA : tB) + (__ffsll((long long)mm) - 1)) : 0.0;
            if (fa) mA &= mA - 1; else mB &= mB - 1;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (in[u]) v += t[u];
    }
    return apply_parity(v, x.sgn);
}

__global__ void __launch_bounds__(kXThreads) k_x_column(Problem P, XState *xs, IterState *st, double *rows,
                                                        long long *cand, long long cap_cand, double *gathp,
                                                        unsigned int *counter) {
    __shared__ ColLists L;
    __shared__ double sw[kXMax];
    __shared__ double sg[kXThreads / 32][kXMax];
    __shared__ unsigned int s_cnt[4][kXThreads / 32];
    __shared__ bool s_last;
    if (!xs->go) return;                                             // no step this iteration
    const int nb = (int)gridDim.x - 1;                               // blocks of the column; one more for S and M
    if ((int)blockIdx.x == nb) {
        x_update_sm(xs);
        return;
    }
    const int k1 = xs->k1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long A = xs->A, B = xs->B;
    build_lists(L, P.N, A, B);
    if (tid < kXMax) sw[tid] = tid < k1 ? xs->wv[tid] : 0.0;
    __syncthreads();
    const double thr = xs->thr;
    const long long nh = P.doubles_vanish ? P.seg[2] : P.seg[5];
    double gat[kXMax];
#pragma unroll
    for (int a = 0; a < kXMax; ++a) gat[a] = 0.0;
    unsigned int c0 = 0, c1 = 0, c2 = 0, c3 = 0;                     // elements, applied, dropped, inserted
    // (whole warps take every round, and the append below is the whole warp's: lanes that inserted and
    // lanes that found their row come here at different times, and each such group used to wait for
    // an atomic of its own, a microsecond after the other)
    for (long long e0 = 1 + (long long)blockIdx.x * blockDim.x + 32 * warp; e0 < nh; e0 += (long long)nb * blockDim.x) {
        const long long e = e0 + lane;
        long long s = -1;                                            // the row, where its mark is new
        if (e < nh) {
            unsigned long long oa, ob;
            ElemIdx ix;
            decode_element(P, L, A, B, e, oa, ob, ix);
            // the key at its first probe position and the row there (it is usually found there) load
            // beside the integrals; no other thread of this launch writes row j or the mark of j (each
            // row occurs once in a column), so the values loaded here are current
            const unsigned long long pos = key_hash(oa, ob) & P.mask;
            double rc[kXMax], rb[kXMax];
            x_load_row(rows, (long long)pos, k1, rc, rb);
            const ulonglong2 k0 = __ldcg(reinterpret_cast<const ulonglong2 *>(P.table + pos));
            const double H = ix.kind <= 1 ? x_single(P, A, B, ix) : element_value(P, L, ix);
            long long at = -2;                                       // -2: nothing to do
            unsigned long long kb = 0ull;
            if (!is_zero(H)) {
                ++c0;
                unsigned long long empty = pos;
                at = x_find(P, st, oa, ob, k0, empty, kb);           // -1: absent, the empty slot known
                if (at >= 0 && at != (long long)pos) x_load_row(rows, at, k1, rc, rb);
                bool cnz = false;
#pragma unroll
                for (int a = 0; a < kXMax; ++a) {
                    if (at < 0) rc[a] = rb[a] = 0.0;                 // a row that is not there yet is zero
                    cnz = cnz || (a < k1 && !is_zero(rc[a]));
                }
                if (at != -2 && !cnz && !(fabs(H) >= thr)) {
                    ++c2;
                    at = -2;
                } else if (at == -1) {
                    at = x_claim(P, st, oa, ob, empty);              // -1: table full, status set
                    if (at < 0) at = -2; else { ++c3; kb = ob; }
                }
            }
            if (at >= 0) {
                ++c1;
                double *br = rows + at * 2 * k1 + k1;
                double bn[kXMax];
#pragma unroll
                for (int a = 0; a < kXMax; ++a) {
                    bn[a] = 0.0;
                    if (a < k1) {                                    // uniform
                        bn[a] = fma(H, sw[a], rb[a]);
                        gat[a] = fma(H, rc[a], gat[a]);
                    }
                }
                if ((k1 & 3) == 0) {                                 // 32-byte stores (see x_load_row)
#pragma unroll
                    for (int q = 0; q < kXMax / 4; ++q)
                        if (4 * q < k1)
                            asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(br + 4 * q), "d"(bn[4 * q]),
                                         "d"(bn[4 * q + 1]), "d"(bn[4 * q + 2]), "d"(bn[4 * q + 3])
                                         : "memory");
                } else if ((k1 & 1) == 0) {                          // 16-byte stores (see x_load_row)
#pragma unroll
                    for (int q = 0; q < kXMax / 2; ++q)
                        if (2 * q < k1) reinterpret_cast<double2 *>(br)[q] = make_double2(bn[2 * q], bn[2 * q + 1]);
                } else {
#pragma unroll
                    for (int a = 0; a < kXMax; ++a)
                        if (a < k1) br[a] = bn[a];
                }
                if (!(kb & kMarkB)) {
                    P.table[at].b = kb | kMarkB;
                    s = at;
                }
            }
        }
        __syncwarp();
        const unsigned m = __ballot_sync(0xffffffffu, s >= 0);
        if (m) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&xs->n_cand, __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (s >= 0) {
                const int to = base + __popc(m & ((1u << lane) - 1u));
                if (to < cap_cand) cand[to] = s;
                else set_status(st, kErrInternal);
            }
        }
    }
    // gather: warp sums, then warps in order (fixed order)
    {
        const double v = x_warp_sums(gat, k1);
        const int a = x_sum_of(lane, k1);
        if (a < k1 && (lane & (k1 > 4 ? 3 : 7)) == 0) sg[warp][a] = v;
    }
    // counters: warp sums (no shared-memory atomics), then the warps in order
    c0 = __reduce_add_sync(0xffffffffu, c0); c1 = __reduce_add_sync(0xffffffffu, c1);
    c2 = __reduce_add_sync(0xffffffffu, c2); c3 = __reduce_add_sync(0xffffffffu, c3);
    if (lane == 0) { s_cnt[0][warp] = c0; s_cnt[1][warp] = c1; s_cnt[2][warp] = c2; s_cnt[3][warp] = c3; }
    __syncthreads();
    if (tid < k1) {
        double v = sg[0][tid];
        for (int w = 1; w < kXThreads / 32; ++w) v += sg[w][tid];
        gathp[(size_t)blockIdx.x * k1 + tid] = v;
    }
    if (tid < 4) {
        unsigned long long t = 0;
        for (int w = 0; w < kXThreads / 32; ++w) t += s_cnt[tid][w];
        if (t) atomicAdd(&xs->cnt[tid], t);
    }
    // the last block: B_i recalculated, the row's mark, the counters
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(counter, 1u) == (unsigned)nb - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) *counter = 0u;
    if (st->status) return;
    const long long s = xs->slot;
    const double Hii = xs->Hii;
    const double cs = tid < k1 ? __ldcg(rows + s * 2 * k1 + tid) : 0.0;
    // per state: the thread's blocks in order, the warp's sums, the warps in order
    double v[kXMax];
#pragma unroll
    for (int a = 0; a < kXMax; ++a) v[a] = 0.0;
    for (int k = tid; k < nb; k += blockDim.x) {
#pragma unroll
        for (int a = 0; a < kXMax; ++a)
            if (a < k1) v[a] += __ldcg(gathp + (size_t)k * k1 + a);
    }
    {
        const double t = x_warp_sums(v, k1);
        const int a = x_sum_of(lane, k1);
        if (a < k1 && (lane & (k1 > 4 ? 3 : 7)) == 0) sg[warp][a] = t;
    }
    __syncthreads();
    if (tid < k1) {
        double t = sg[0][tid];
        for (int w = 1; w < kXThreads / 32; ++w) t += sg[w][tid];
        rows[s * 2 * k1 + k1 + tid] = fma(Hii, cs, t);
    }
    if (tid == 0) {
        const unsigned long long kb = P.table[s].b;
        if (!(kb & kMarkB)) {
            P.table[s].b = kb | kMarkB;
            const int pos = atomicAdd(&xs->n_cand, 1);
            if (pos < cap_cand) cand[pos] = s;
            else set_status(st, kErrInternal);
        }
        const long long nd = Hii != 0.0 ? 1 : 0;
        const long long n0 = (long long)__ldcg(&xs->cnt[0]), n1 = (long long)__ldcg(&xs->cnt[1]);
        const long long n2 = (long long)__ldcg(&xs->cnt[2]), n3 = (long long)__ldcg(&xs->cnt[3]);
        xs->elements += n0 + nd;
        xs->applied += n1 + nd;
        xs->dropped += n2;
        xs->inserted += n3;
        xs->n_slots += n3;
        xs->last_column = n0 + nd;
        for (int k = 0; k < 4; ++k) xs->cnt[k] = 0ull;
        if (xs->n_slots > P.max_entries) set_status(st, kErrTableFull);
    }
}

// Energies: the k1 eigenvalues of the pencil (M, S), ascending: S = L L^T
// (Cholesky), the symmetric A = L^-1 M L^-T, cyclic Jacobi rotations (Golub &
// Van Loan, Sec. 8.5) until the off-diagonal mass is below 1e-30 of the total.
// One thread; also the host-visible snapshot.
__global__ void k_x_energies(XState *xs, IterState *st) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int n = xs->k1;
    double L[kXMax * kXMax], T[kXMax * kXMax], A[kXMax * kXMax];
    bool ok = true;
    for (int i = 0; i < n * n; ++i) L[i] = 0.0;
    for (int i = 0; i < n && ok; ++i)
        for (int j = 0; j <= i; ++j) {
            double s = xs->S[i * n + j].hi + xs->S[i * n + j].lo;
            for (int k = 0; k < j; ++k) s -= L[i * n + k] * L[j * n + k];
            if (i == j) {
                if (!(s > 0.0)) { ok = false; break; }
                L[i * n + i] = sqrt(s);
            } else {
                L[i * n + j] = s / L[j * n + j];
            }
        }
    if (ok) {
        for (int col = 0; col < n; ++col)
            for (int i = 0; i < n; ++i) {
                double s = xs->M[i * n + col].hi + xs->M[i * n + col].lo;
                for (int k = 0; k < i; ++k) s -= L[i * n + k] * T[k * n + col];
                T[i * n + col] = s / L[i * n + i];
            }
        for (int row = 0; row < n; ++row)
            for (int i = 0; i < n; ++i) {
                double s = T[row * n + i];
                for (int k = 0; k < i; ++k) s -= L[i * n + k] * A[row * n + k];
                A[row * n + i] = s / L[i * n + i];
            }
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < i; ++j) {
                const double v = 0.5 * (A[i * n + j] + A[j * n + i]);
                A[i * n + j] = v; A[j * n + i] = v;
            }
        for (int sweep = 0; sweep < 64; ++sweep) {
            double off = 0.0, tot = 0.0;
            for (int i = 0; i < n; ++i)
                for (int j = 0; j < n; ++j) {
                    tot += A[i * n + j] * A[i * n + j];
                    if (i != j) off += A[i * n + j] * A[i * n + j];
                }
            if (off <= 1e-30 * tot) break;
            for (int p = 0; p < n; ++p)
                for (int q = p + 1; q < n; ++q) {
                    const double apq = A[p * n + q];
                    if (apq == 0.0) continue;
                    const double theta = (A[q * n + q] - A[p * n + p]) / (2.0 * apq);
                    const double t = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                    const double c = 1.0 / sqrt(t * t + 1.0), sn = t * c;
                    for (int k = 0; k < n; ++k) {
                        const double akp = A[k * n + p], akq = A[k * n + q];
                        A[k * n + p] = c * akp - sn * akq;
                        A[k * n + q] = sn * akp + c * akq;
                    }
                    for (int k = 0; k < n; ++k) {
                        const double apk = A[p * n + k], aqk = A[q * n + k];
                        A[p * n + k] = c * apk - sn * aqk;
                        A[q * n + k] = sn * apk + c * aqk;
                    }
                }
        }
        double E[kXMax];
        for (int i = 0; i < n; ++i) E[i] = A[i * n + i];
        for (int i = 0; i < n; ++i)
            for (int j = i + 1; j < n; ++j)
                if (E[j] < E[i]) { const double t = E[i]; E[i] = E[j]; E[j] = t; }
        for (int i = 0; i < n; ++i) xs->E[i] = E[i];
    } else {
        for (int i = 0; i < n; ++i) xs->E[i] = nan("");
    }
    st->iterations = xs->iterations; st->nnz_c = xs->nnz_c; st->n_slots = xs->n_slots;
    st->elements = xs->elements; st->applied = xs->applied; st->dropped = xs->dropped; st->inserted = xs->inserted;
    st->last_column = xs->last_column;
    st->mu = xs->S[0]; st->alpha = xs->M[0];
    st->dx = xs->dx; st->energy = xs->E[0]; st->last_eta = xs->eta;
    st->last_a = xs->A; st->last_b = xs->B; st->done = xs->done;
}

// Diagonal elements H_DD of a list of determinants (one warp each): picks the
// start rows of xCDFCI.
__global__ void k_x_diag_list(Problem P, const unsigned long long *keys, long long n, double *out) {
    __shared__ ColLists Ls[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ColLists &L = Ls[warp];
    for (long long k = (long long)blockIdx.x * 8 + warp; k < n; k += (long long)gridDim.x * 8) {
        const unsigned long long A = keys[2 * k], B = keys[2 * k + 1];
        for (int t = lane; t < P.N; t += 32) {
            const int ra = __popcll(A & low_mask(t)), rb = __popcll(B & low_mask(t));
            if ((A >> t) & 1ull) L.occA[ra] = (unsigned char)t; else L.virA[t - ra] = (unsigned char)t;
            if ((B >> t) & 1ull) L.occB[rb] = (unsigned char)t; else L.virB[t - rb] = (unsigned char)t;
        }
        __syncwarp();
        const double d = diag_warp(P, L);
        if (lane == 0) out[k] = d;
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
cudaError_t launch_x_diag_list(const Problem &P, const unsigned long long *keys, long long n, double *out,
                               cudaStream_t s) {
    const long long blocks = std::min<long long>((n + 7) / 8, 1024);
    k_x_diag_list<<<(int)std::max<long long>(blocks, 1), 256, 0, s>>>(P, keys, n, out);
    return cudaGetLastError();
}

// blocks of a column: an element per thread, at most four blocks per SM; of the choice: a candidate
// per thread, at most two blocks per SM
int x_scatter_blocks(const Problem &P) {
    const long long nh = P.doubles_vanish ? P.seg[2] : P.seg[5];
    return (int)std::max<long long>(1, std::min<long long>(152 * 4, (nh - 1 + kXThreads - 1) / kXThreads));
}
int x_select_blocks(const Problem &P) { return std::min(152 * 2, x_scatter_blocks(P)); }

size_t x_block_bytes() { return sizeof(XBest); }

static cudaError_t launch_x_column(const Problem &P, const XBuffers &b, cudaStream_t s) {
    k_x_column<<<b.nscatter + 1, kXThreads, 0, s>>>(P, b.xs, b.st, b.rows, b.cand, b.cap_cand, b.gathp, b.counter + 1);
    return cudaGetLastError();
}

cudaError_t launch_x_start(const Problem &P, const XBuffers &b, unsigned long long A, unsigned long long B, int k,
                           cudaStream_t s) {
    k_x_choose<<<1, kXThreads, 0, s>>>(P, b.xs, b.st, b.cand, b.cap_cand, b.rows, static_cast<XBest *>(b.bbest), b.counter, k, A, B);
    return launch_x_column(P, b, s);
}

cudaError_t launch_x_iteration(const Problem &P, const XBuffers &b, cudaStream_t s) {
    k_x_choose<<<b.nselect, kXThreads, 0, s>>>(P, b.xs, b.st, b.cand, b.cap_cand, b.rows, static_cast<XBest *>(b.bbest), b.counter,
                                               -1, 0ull, 0ull);
    return launch_x_column(P, b, s);
}

cudaError_t launch_x_energies(const XBuffers &b, cudaStream_t s) {
    k_x_energies<<<1, 32, 0, s>>>(b.xs, b.st);
    return cudaGetLastError();
}

}  // namespace cdfci
