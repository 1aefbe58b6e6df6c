// K2 (SIMT): mu-mode contraction Y = X x_mu M on the FP64 / FP32 FMA pipes, with the
// pointwise phi_k scaling (K3) and the stage axpy (K4) fused into the epilogue.
//
// The mu-mode product of Section 1 (e^{A_d (+) ... (+) A_1} v = vec(V x_1 e^{A_1} ...
// x_d e^{A_d})) is a strided batched GEMM. Viewing the state as [P][n_mu][Q] (P the
// directions slower than mu, Q the faster ones):
//   mode 1 (Q = 1):  Y (P x n) = X (P x n) * M^T
//   mode mu > 1:     Y_p (n x Q) = M (n x n) * X_p (n x Q)   for each p
// The host passes element strides for A, B, C so one kernel serves every mode.
#include <cuda_runtime.h>

#include <algorithm>

#include "adr_internal.h"
#include "launch.cuh"
#include "phi_device.cuh"
#include "smem_limit.h"

namespace adr {
namespace {

// The phi factor of node off: from the table, or evaluated where the context keeps none.
template <typename T>
__device__ __forceinline__ T phi_of(const ContractArgs<T>& p, long long off) {
    if (p.phi) return p.phi[off];
    const int i1 = int(off % p.n1);
    const long long t = off / p.n1;
    const int i2 = int(t % p.n2);
    const int i3 = int(t / p.n2);
    double ls = p.lam[0][i1] + p.lam[1][i2];
    if (p.lam[2]) ls += p.lam[2][i3];
    return phi_eval(p.phik, T(p.ctau * ls));
}

// Small passes: a block takes W x W outputs and loads its two panels (all of K) at once, so one trip to
// memory and one barrier stand before the products instead of one per 16 of K. KS lanes share an output's sum: in
// FP64 four, each a quarter of K, so the chain of dependent FMAs is a quarter as long; in FP32 one, which adds
// the products in the order of the tiled kernel. A context's factor is loaded before the kernel waits for its
// predecessor.
// What bounds it is latency: of a launch of 8 us the 32^2 FP64 products need 0.1 us of the FP64 pipe. A launch inside a 32^2
// FP64 ETD2RK step, tiled kernel -> this one: 8.2 -> 6.1 us; the step, three runs at a time, 18.5 -> 7.7 us (10.7 without
// the early start). FP64 takes it wherever 32 x 32 tiles would not give every SM two blocks (100 x 90 Lawson4 1.55x,
// 500 x 30 2.1x, 20 x 24 x 16 ETD2RK 1.9x); FP32, where 16 x 16 tiles are few, at most a sixth of the SMs (64^2 1.54x,
// 80 x 70 1.38x, 150 x 30 1.27x; at 36 blocks, 96^2, 0.99x, at 54, 24^3, 0.91x).
constexpr int kSmallK = 512;

template <typename T, int W, int KS>
__global__ void __launch_bounds__(W * W * KS) contract_small_kernel(ContractArgs<T> p) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    constexpr int NT = W * W * KS;
    const int pitch = p.K + 1;
    T* As = reinterpret_cast<T*>(small_smem);                // [W][pitch]
    T* Bs = As + W * pitch;                                  // [W][pitch]
    const int tid = threadIdx.x, ks = tid % KS, tx = tid / KS % W, ty = tid / KS / W;
    const int b = blockIdx.z, m0 = blockIdx.y * W, n0 = blockIdx.x * W;
    auto load = [&](T* dst, const T* src, int rows, long long srow, long long sk) {
        for (int e = tid; e < W * p.K; e += NT) {            // neighbouring threads along the contiguous index
            const int r = sk == 1 ? e / p.K : e % W, k = sk == 1 ? e % p.K : e / W;
            dst[r * pitch + k] = r < rows ? src[r * srow + k * sk] : T(0);
        }
    };
    auto load_a = [&] { load(As, p.A + (long long)b * p.sab + (long long)m0 * p.sam, p.M - m0, p.sam, p.sak); };
    auto load_b = [&] { load(Bs, p.B + (long long)b * p.sbb + (long long)n0 * p.sbn, p.N - n0, p.sbn, p.sbk); };
    pdl_trigger();
    if (p.factor == 1) load_a();
    if (p.factor == 2) load_b();
    pdl_wait();
    if (p.factor != 1) load_a();
    if (p.factor != 2) load_b();
    __syncthreads();
    T acc = T(0);
#pragma unroll 4
    for (int k = ks; k < p.K; k += KS) acc = fma(As[ty * pitch + k], Bs[tx * pitch + k], acc);
#pragma unroll
    for (int d = 1; d < KS; d <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    const int gm = m0 + ty, gn = n0 + tx;
    if (ks != 0 || gm >= p.M || gn >= p.N) return;
    const long long off = (long long)b * p.scb + (long long)gm * p.scm + (long long)gn * p.scn;
    if (p.epi == EPI_PHI) acc *= phi_of(p, off);
    else if (p.epi == EPI_AXPY) acc = p.base[off] + T(p.alpha) * acc;
    p.C[off] = acc;
}

template <typename T, int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
contract_kernel(ContractArgs<T> p) {
    constexpr int NT = (BM / TM) * (BN / TN);
    constexpr int NX = BN / TN;   // threads along n
    constexpr int NY = BM / TM;   // threads along m
    __shared__ T As[BK][BM + 1];
    __shared__ T Bs[BK][BN + 1];

    const int tid = threadIdx.x;
    const int tx = tid % NX, ty = tid / NX;
    const int b = blockIdx.z;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const T* A = p.A + (long long)b * p.sab;
    const T* B = p.B + (long long)b * p.sbb;
    const bool a_kfast = (p.sak == 1);
    const bool b_kfast = (p.sbk == 1);

    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);

    for (int k0 = 0; k0 < p.K; k0 += BK) {
        // global -> shared, consecutive threads along the contiguous global index
        for (int e = tid; e < BM * BK; e += NT) {
            int mm, kk;
            if (a_kfast) { kk = e % BK; mm = e / BK; } else { mm = e % BM; kk = e / BM; }
            const int gm = m0 + mm, gk = k0 + kk;
            As[kk][mm] = (gm < p.M && gk < p.K) ? A[(long long)gm * p.sam + (long long)gk * p.sak] : T(0);
        }
        for (int e = tid; e < BN * BK; e += NT) {
            int nn, kk;
            if (b_kfast) { kk = e % BK; nn = e / BK; } else { nn = e % BN; kk = e / BN; }
            const int gn = n0 + nn, gk = k0 + kk;
            Bs[kk][nn] = (gn < p.N && gk < p.K) ? B[(long long)gk * p.sbk + (long long)gn * p.sbn] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T ra[TM], rb[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) ra[i] = As[kk][ty + i * NY];
#pragma unroll
            for (int j = 0; j < TN; ++j) rb[j] = Bs[kk][tx + j * NX];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(ra[i], rb[j], acc[i][j]);
        }
        __syncthreads();
    }

    // epilogue: the C offset is the element's linear index in the state array
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int gm = m0 + ty + i * NY;
        if (gm >= p.M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int gn = n0 + tx + j * NX;
            if (gn >= p.N) continue;
            const long long off = (long long)b * p.scb + (long long)gm * p.scm + (long long)gn * p.scn;
            T v = acc[i][j];
            if (p.epi == EPI_PHI) {
                v *= phi_of(p, off);
            } else if (p.epi == EPI_AXPY) {
                v = p.base[off] + T(p.alpha) * v;
            }
            p.C[off] = v;
        }
    }
}

template <typename T, int BM, int BN, int BK, int TM, int TN>
cudaError_t launch_tiled(const ContractArgs<T>& p, cudaStream_t s) {
    dim3 grid((p.N + BN - 1) / BN, (p.M + BM - 1) / BM, p.batch);
    if (grid.y > 65535u || grid.z > 65535u) return cudaErrorInvalidConfiguration;
    contract_kernel<T, BM, BN, BK, TM, TN><<<grid, (BM / TM) * (BN / TN), 0, s>>>(p);
    return cudaGetLastError();
}

template <typename T, int W, int KS>
cudaError_t launch_small(const ContractArgs<T>& p, cudaStream_t s) {
    static SmemLimit smem;
    const cudaError_t e = smem.allow(reinterpret_cast<const void*>(contract_small_kernel<T, W, KS>),
                                     int(2 * W * (kSmallK + 1) * sizeof(T)));
    if (e != cudaSuccess) return e;
    const dim3 grid((p.N + W - 1) / W, (p.M + W - 1) / W, p.batch);
    return launch_pdl(contract_small_kernel<T, W, KS>, grid, W * W * KS, size_t(2 * W) * (p.K + 1) * sizeof(T), s, p);
}

template <typename T>
__global__ void phi_nodes_kernel(T* tab, ContractArgs<T> p, size_t N) {
    for (size_t o = blockIdx.x * size_t(blockDim.x) + threadIdx.x; o < N; o += size_t(gridDim.x) * blockDim.x)
        tab[o] = phi_of(p, (long long)o);
}

int g_sms = 0;

// Output tiles of a bm x bn tiling of the pass.
template <typename T>
long long ctas(const ContractArgs<T>& p, int bm, int bn) {
    return (long long)((p.N + bn - 1) / bn) * ((p.M + bm - 1) / bm) * p.batch;
}

int sm_count() {
    if (g_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

}  // namespace

cudaError_t launch_phi_nodes(double* tab, const ContractArgs<double>& p, size_t N, cudaStream_t s) {
    phi_nodes_kernel<<<unsigned(std::min<size_t>((N + 255) / 256, 65535)), 256, 0, s>>>(tab, p, N);
    return cudaGetLastError();
}
cudaError_t launch_phi_nodes(float* tab, const ContractArgs<float>& p, size_t N, cudaStream_t s) {
    phi_nodes_kernel<<<unsigned(std::min<size_t>((N + 255) / 256, 65535)), 256, 0, s>>>(tab, p, N);
    return cudaGetLastError();
}

// The largest tile that still gives every SM work: a small grid in one big tile would run on
// one SM (and mostly on padding), which the FP64 pipes of this GPU make very slow. Every
// output of the tiled kernel, and of the small one in FP32, accumulates its K products in the same order.
cudaError_t launch_contract(const ContractArgs<double>& p, cudaStream_t s) {
    const long long want = 2LL * sm_count();
    if (ctas(p, 64, 64) >= want) return launch_tiled<double, 64, 64, 16, 4, 4>(p, s);
    if (ctas(p, 32, 32) >= want) return launch_tiled<double, 32, 32, 16, 2, 2>(p, s);
    if (p.K <= kSmallK) return launch_small<double, 8, 4>(p, s);
    if (ctas(p, 16, 16) >= want / 2) return launch_tiled<double, 16, 16, 16, 1, 1>(p, s);
    return launch_tiled<double, 8, 8, 16, 1, 1>(p, s);
}

cudaError_t launch_contract(const ContractArgs<float>& p, cudaStream_t s) {
    const long long want = 2LL * sm_count();
    if (ctas(p, 128, 128) >= want) return launch_tiled<float, 128, 128, 8, 8, 8>(p, s);
    if (ctas(p, 64, 64) >= want) return launch_tiled<float, 64, 64, 16, 4, 4>(p, s);
    if (ctas(p, 32, 32) >= want) return launch_tiled<float, 32, 32, 16, 2, 2>(p, s);
    if (p.K <= kSmallK && ctas(p, 16, 16) <= sm_count() / 6) return launch_small<float, 16, 1>(p, s);
    return launch_tiled<float, 16, 16, 16, 1, 1>(p, s);
}

}  // namespace adr
