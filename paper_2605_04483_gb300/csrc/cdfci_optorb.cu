// OptOrbFCI (Algorithm 4, Sec. "Optimal Orbital Selections"): device kernels of
// the orbital subproblem.  Every array is FP64 and row-major; U is M x N with
// orthonormal columns, the integrals h (M x M) and g (M^4, chemists' order) are
// in the large basis, the RDMs (N x N, N^4) in the small one.
//   k_oo_contract   out[a][n][b] = sum_m in[a][m][b] U[m][n] (one index of a tensor)
//   k_oo_grad       G = 2 (h U) gamma + 2 sum_bcd g''_pbcd Gamma_abcd
//   k_oo_objective  P = h'.gamma + g'.Gamma / 2, and U kept where P is the lowest so far
//   k_oo_move       U <- orth(U - t G) with the Barzilai-Borwein step t
// The descent runs on the device from the RDMs to the last basis: the host
// launches nine kernels a step and reads nothing before the end.  (The step's
// scalars and every Newton-Schulz iteration's Gram matrix used to be read by the
// host, 11 synchronisations and about 35 launches a step: 12 orbitals to 9, two
// outer iterations of 10 steps, 400 inner iterations: 15.4 -> 8.4 ms.)
#include <cooperative_groups.h>

#include <algorithm>

#include "cdfci_internal.cuh"
#include "cdfci_kernels.h"

namespace cg = cooperative_groups;

namespace cdfci {

__global__ void k_oo_contract(const double *in, const double *U, double *out, long long A, int M, int N, long long B) {
    const long long total = A * N * B;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long b = i % B;
        const int n = (int)((i / B) % N);
        const long long a = i / (B * N);
        double s = 0.0;
        for (int m = 0; m < M; ++m) s = fma(in[(a * M + m) * B + b], U[m * N + n], s);
        out[i] = s;
    }
}

// One block per element (p, a): a sum of N^3 products, strided over the threads,
// then a tree.  (One thread an element, a chain of N^3 dependent operations:
// 54 us for 12 x 9 elements, now 2.8.)
constexpr int kGradThreads = 128;
__global__ void __launch_bounds__(kGradThreads) k_oo_grad(const double *hU, const double *g1, const double *g3,
                                                          const double *g2, double *G, int N) {
    __shared__ double red[kGradThreads / 32];
    const int n3 = N * N * N, p = blockIdx.x / N, a = blockIdx.x - p * N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *x = g3 + (size_t)p * n3, *y = g2 + (size_t)a * n3;
    double s = 0.0;
    if (threadIdx.x < N) s = hU[p * N + threadIdx.x] * g1[threadIdx.x * N + a];
#pragma unroll 4
    for (int t = threadIdx.x; t < n3; t += kGradThreads) s = fma(x[t], y[t], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) G[blockIdx.x] = 2.0 * ((red[0] + red[1]) + (red[2] + red[3]));
}

// The objective P; where it is below *best (or first), *best = P and Ub = U.
// Sums strided over the grid, the blocks' parts added in block order by the one
// that finishes last.
__global__ void __launch_bounds__(256) k_oo_objective(const double *h2, const double *r1, const double *g4,
                                                      const double *r2, int N, double *part, unsigned int *counter,
                                                      double *best, const double *U, double *Ub, int MN, int first) {
    __shared__ double red[8];
    __shared__ double s_P;
    __shared__ bool s_last, s_keep;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long n2 = (long long)N * N, n4 = n2 * n2, step = (long long)gridDim.x * blockDim.x;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
#pragma unroll 4
    for (long long t = t0; t < n4; t += step) s = fma(g4[t], r2[t], s);
    s *= 0.5;
    for (long long t = t0; t < n2; t += step) s = fma(h2[t], r1[t], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = red[0];
        for (int w = 1; w < 8; ++w) v += red[w];
        part[blockIdx.x] = v;
        __threadfence();
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (warp == 0) {
        double v = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(part + b);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) s_P = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s_keep = first || s_P < *best;
        if (s_keep) *best = s_P;
        *counter = 0u;
    }
    __syncthreads();
    if (s_keep)
        for (int i = threadIdx.x; i < MN; i += blockDim.x) Ub[i] = U[i];
}

// One step of the descent: t (the first step 0.1 / max(1, |G|); then S.S / |S.Y|
// and |S.Y| / Y.Y in turn with S = U - Uo, Y = G - Go, the last t where they
// vanish), Uo = U, Go = G, U <- orth(U - t G) by Newton-Schulz iterations
// X <- X (3 I - X^T X) / 2 from X / |X|_F until |X^T X - I| < 4e-16 N.
// Sums as 256 strided parts and a tree.  A cluster of C CTAs of 256 threads holds
// X and X^T X in every CTA's shared memory; each computes its share of the
// entries and writes it to all.  What bounds it is the FP64 pipe of the SMs used
// (two operations a cycle each) for large bases and the barriers for small ones;
// oo_move says where the line lies.
__global__ void __launch_bounds__(256) k_oo_move(double *U, const double *G, double *Uo, double *Go, double *tstate,
                                                 int *failed, int k, int M, int N) {
    extern __shared__ __align__(16) double s_x[];
    __shared__ double red[3][256];
    __shared__ double s_err[8];
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, MN = M * N, NN = N * N;
    double *X = s_x, *Xn = s_x + MN, *Gm = s_x + 2 * MN;
    auto sync_all = [&]() { if (C > 1) cl.sync(); else __syncthreads(); };
    auto put = [&](double *p, double v) {               // p: an address in this CTA, written in every CTA
        if (C == 1) *p = v;
        else
            for (int r = 0; r < C; ++r) *cl.map_shared_rank(p, r) = v;
    };
    auto tree = [&]() {                                 // the three sums of red, in every thread's reach
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (tid < w)
                for (int q = 0; q < 3; ++q) red[q][tid] += red[q][tid + w];
            __syncthreads();
        }
    };
    // t
    double d0 = 0.0, d1 = 0.0, d2 = 0.0;
    for (int i = tid; i < MN; i += 256) {
        if (k == 0) {
            d0 = fma(G[i], G[i], d0);
        } else {
            const double S = U[i] - Uo[i], Y = G[i] - Go[i];
            d0 = fma(S, S, d0); d1 = fma(S, Y, d1); d2 = fma(Y, Y, d2);
        }
    }
    red[0][tid] = d0; red[1][tid] = d1; red[2][tid] = d2;
    tree();
    double t;
    if (k == 0) {
        const double gn = sqrt(red[0][0]);
        t = 0.1 / (1.0 < gn ? gn : 1.0);
    } else {
        t = *tstate;
        const double sy = fabs(red[1][0]), yy = red[2][0];
        if (sy > 0.0 && yy > 0.0) t = (k & 1) ? red[0][0] / sy : sy / yy;
        t = t < 1e-10 ? 1e-10 : t;
        t = 1e10 < t ? 1e10 : t;
    }
    __syncthreads();
    // X = (U - t G) / |U - t G|_F
    d0 = 0.0;
    for (int i = tid; i < MN; i += 256) {
        const double x = U[i] - t * G[i];
        X[i] = x;
        d0 = fma(x, x, d0);
    }
    red[0][tid] = d0;
    red[1][tid] = red[2][tid] = 0.0;
    tree();
    const double f = red[0][0] > 0.0 ? 1.0 / sqrt(red[0][0]) : 1.0;
    for (int i = tid; i < MN; i += 256) X[i] *= f;
    sync_all();                                         // (every CTA has read U, Uo, G, Go, *tstate)
    bool ok = false;
    for (int it = 0; it < 200; ++it) {
        for (int i = rank * 256 + tid; i < NN; i += C * 256) {
            const int a = i / N, b = i - a * N;
            double s = 0.0;
            for (int p = 0; p < M; ++p) s = fma(X[p * N + a], X[p * N + b], s);
            put(Gm + i, s);
        }
        sync_all();
        double e = 0.0;
        for (int i = tid; i < NN; i += 256) e = fmax(e, fabs(Gm[i] - (i % (N + 1) == 0 ? 1.0 : 0.0)));
        for (int o = 16; o > 0; o >>= 1) e = fmax(e, __shfl_xor_sync(0xffffffffu, e, o));
        if (lane == 0) s_err[warp] = e;
        __syncthreads();
        for (int w = 0; w < 8; ++w) e = fmax(e, s_err[w]);
        if (e < 4e-16 * N) { ok = true; break; }        // the same in every CTA
        for (int i = rank * 256 + tid; i < MN; i += C * 256) {
            const int p = i / N, a = i - p * N;
            double s = 0.0;
            for (int b = 0; b < N; ++b) s = fma(X[p * N + b], Gm[b * N + a], s);
            put(Xn + i, 0.5 * (3.0 * X[i] - s));
        }
        sync_all();
        double *y = X; X = Xn; Xn = y;
    }
    if (rank != 0) return;
    if (!ok && tid == 0) *failed = 1;
    if (tid == 0) *tstate = t;
    for (int i = tid; i < MN; i += 256) {
        Uo[i] = U[i];
        Go[i] = G[i];
        U[i] = X[i];
    }
}

// ---------------------------------------------------------------------------
// host wrappers
// ---------------------------------------------------------------------------
static int oo_grid(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152 * 8)); }

cudaError_t oo_contract(const double *in, const double *U, double *out, long long A, int M, int N, long long B,
                        cudaStream_t s) {
    k_oo_contract<<<oo_grid(A * N * B), 256, 0, s>>>(in, U, out, A, M, N, B);
    return cudaGetLastError();
}
cudaError_t oo_grad(const double *hU, const double *g1, const double *g3, const double *g2, double *G, int M, int N,
                    cudaStream_t s) {
    k_oo_grad<<<M * N, kGradThreads, 0, s>>>(hU, g1, g3, g2, G, N);
    return cudaGetLastError();
}
cudaError_t oo_objective(const double *h2, const double *r1, const double *g4, const double *r2, const OoState &st,
                         const double *U, double *Ub, int M, int N, int first, cudaStream_t s) {
    const long long n4 = (long long)N * N * N * N;
    const int blocks = (int)std::max<long long>(1, std::min<long long>(kOoParts, (n4 + 1023) / 1024));
    k_oo_objective<<<blocks, 256, 0, s>>>(h2, r1, g4, r2, N, st.part, st.counter, st.best, U, Ub, M * N, first);
    return cudaGetLastError();
}
// One CTA up to M N^2 = kOoOneCta (a product's operations), eight above.  M = N = 12: 36.6 us with
// one, 44.4 with eight; 16: 50.6, 59.5; 18: 73.4, 65.8; 24: 117, 73.8; 63: 1399, 260.
constexpr long long kOoOneCta = 4096;
cudaError_t oo_move(double *U, const double *G, double *Uo, double *Go, const OoState &st, int k, int M, int N,
                    cudaStream_t s) {
    const size_t smem = (2 * (size_t)M * N + (size_t)N * N) * sizeof(double);    // at most 95 KB
    cudaError_t e = cudaFuncSetAttribute(k_oo_move, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         3 * kMaxN * kMaxN * (int)sizeof(double));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    const unsigned C = (long long)M * N * N <= kOoOneCta ? 1 : 8;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_oo_move, U, G, Uo, Go, st.t, st.failed, k, M, N);
}

}  // namespace cdfci
