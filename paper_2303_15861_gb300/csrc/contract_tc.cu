// K2 (tensor cores, mixed precision): mu-mode contraction Y = X x_mu M of an FP32 state (optionally a hi + lo pair)
// with an FP64 factor, as exact sums of BF16 products.
//
// The exact-slice split. The FP32 state gets one power-of-two scale 2^es from a max-abs its producer
// recorded, each factor row its own; x = 2^(es-7) sum_j 2^(-8j) S_j, f = 2^(e-7) sum_j 2^(-8j) F_j with integer
// slices of at most 128, four of each. Ten products go to four TMEM accumulators,
//     D0 = S0.F0,  D1 = S0.F1 + S1.F0,  D2 = S0.F2 + S1.F1 + S2.F0,
//     D3 = S0.F3 + S1.F2 + S2.F1 + S3.F0,
// integer terms of magnitude at most 2^14. For K <= 256 all four stay within 2^24 even in the
// worst case (D0 and D1 for K <= 512), so they are exact whatever rounding the tensor cores
// apply; beyond that D2 and D3 could pass 2^24 only if hundreds of residual-slice products
// shared the largest magnitude and one sign, and their rounding would weigh 2^-16 and 2^-24 of
// a unit of D0. x.f = D0 + 2^-8 D1 + 2^-16 D2 + 2^-24 D3 up to the products below 2^-32,
// combined once in the epilogue. A time integration applies the same factor to a
// slowly varying state in every step, so any bias of a pass adds up. Measured on the 40-step
// 256^3 Lawson4 run (relative error and mean drift against the FP64 path): six products into
// two accumulators 1.5e-6 / -1.0e-6; seven into three exact accumulators with a 32-bit factor
// but without the 2^-24 cross products S1.F2, S2.F1, S3.F0 2.8e-6 / -1.7e-6; all ten 2.6e-7 /
// +1e-9. With EPI_STORE2 the result is a double-float pair: for the one exponential whose result feeds
// the stencil that no later exponential smooths.
//
// Work split. The factor is the A operand, 128 outputs (TMEM lanes) a tile, and N = 64 lines the B
// operand (32 where 64 would leave SMs without a tile): four accumulators of 64 columns are half of TMEM, so
// the epilogue of a tile overlaps the next tile's MMAs. With 128 columns the four fill TMEM and the epilogue and the
// MMAs of a tile take turns; that form, its state brought by TMA and so only for extents that are multiples of 4, took 84, 95 and
// 93 us at 256^3 in modes 1, 2, 3 where this one takes 78, 80 and 79 (at 384^3 358, 402 and 504 against 336, 342 and
// 343); the form without TMA for the other extents took 15 to 41 us at 129 x 100 x 75 where this one takes 14 to 20. For
// modes >= 2 the lines are consecutive positions, p and q flattened, so a short q leaves no empty columns. Warps 0-7 are
// producers: they load FP32 from global memory (no alignment rules, so every shape takes this kernel) and store the
// slices; warps 8-15 are the epilogue; warp 16 issues the MMAs, warp 17 copies the pre-sliced factor.
//
// What bounds it, at 256^3: the MMAs alone take 45 us, with their epilogue 49, the ring's handshakes 60, the slicing
// 64, and with the loads 79. The ring therefore has one barrier pair for both operands of a stage (a pair each: 90 us).
#include <cuda_runtime.h>

#include <cstdint>

#include "adr_internal.h"
#include "phi_device.cuh"
#include "smem_limit.h"
#include "tc_common.cuh"

namespace adr {
namespace {
using namespace tc;

constexpr int kSl = 4;                   // slices per operand, accumulators
constexpr int kM = 128;                  // UMMA M, TMEM lanes
constexpr int kKc = 32;                  // K per stage: one 64-byte bf16 row (64-byte swizzle)
constexpr int kProducerWarps = 8;
constexpr int kGroups = 2;               // of producer warps, taking the K chunks in turn
constexpr int kGroupWarps = kProducerWarps / kGroups;
constexpr int kEpiWarps = 8;
constexpr int kMmaWarp = kProducerWarps + kEpiWarps;
constexpr int kLoadWarp = kMmaWarp + 1;
constexpr int kThreads = (kLoadWarp + 1) * 32;

template <int N>
struct Cfg {
    static constexpr int FTILE = kM * kKc * 2, STILE = N * kKc * 2;   // one slice tile of either operand
    static constexpr int SBYTES = kSl * STILE, FBYTES = kSl * FTILE;  // one stage: 16 KB (N = 64) and 32 KB
    static constexpr int NS = 4;                                      // stages of the ring
    static constexpr int SMEM = NS * (SBYTES + FBYTES) + 1024;
    static constexpr int SETS = 2;                                    // accumulator sets of 4 N columns
    static constexpr uint32_t TMEM = N == 64 ? 512 : 256;
    static constexpr int COLS = N / (kEpiWarps / 4);                  // columns per epilogue warp
    static constexpr int KV = N * kKc / (kGroupWarps * 32);           // K values a producer thread slices of its chunk
    static constexpr int KG = kKc / KV;                               // threads per line
    static_assert(KV % 8 == 0, "whole 16-byte chunks of a slice row");
    static_assert(COLS <= 32 && COLS % 8 == 0, "one lane per column finds its offset");
    static_assert(SMEM <= 227 * 1024, "shared memory budget");
};

__device__ __forceinline__ uint32_t idesc_of(int ncols) {   // FP32 accumulator, BF16 operands, M = 128
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(ncols >> 3) << 17) | (uint32_t(kM >> 4) << 24);
}

__device__ __forceinline__ void tmem_ld8x4(uint32_t t0, uint32_t stride, float (&d)[4][8]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(t0), "r"(t0 + stride), "r"(t0 + 2 * stride), "r"(t0 + 3 * stride)
        : "memory");
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 8; ++j) d[k][j] = __uint_as_float(r[8 * k + j]);
}

// Integer slices of y + ylo: the residuals y - s0 and y1 - s1 are exact, and the low part enters once,
// after the leading slice.
__device__ __forceinline__ void split(float y, float ylo, float (&s)[kSl]) {
    s[0] = rint_small(y);
    const float y1 = ((y - s[0]) + ylo) * 256.f;
    s[1] = rint_small(y1);
    const float y2 = (y1 - s[1]) * 256.f;
    s[2] = rint_small(y2);
    s[3] = rint_small((y2 - s[2]) * 256.f);
}

// Slice KV values along K (low parts vl, if LO) and store them at K position k (a multiple of 8) of row r of the four slice
// tiles.
template <int TILE, int KV, bool LO>
__device__ __forceinline__ void slice_store(const float (&v)[KV], const float (&vl)[KV], float sc, uint32_t tile0, int r, int k) {
#pragma unroll
    for (int h = 0; h < KV; h += 8) {
        uint32_t w[kSl][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float a[kSl], b[kSl];
            split(v[h + 2 * e] * sc, LO ? vl[h + 2 * e] * sc : 0.f, a);
            split(v[h + 2 * e + 1] * sc, LO ? vl[h + 2 * e + 1] * sc : 0.f, b);
#pragma unroll
            for (int q = 0; q < kSl; ++q) w[q][e] = __byte_perm(__float_as_uint(a[q]), __float_as_uint(b[q]), 0x7632);
        }
        const uint32_t dst = tile0 + swz64(r, (k + h) >> 3);
#pragma unroll
        for (int q = 0; q < kSl; ++q) st_shared_v4(dst + q * TILE, make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]));
    }
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// 32-byte (256-bit) accesses: eight consecutive floats.
__device__ __forceinline__ void ld8(const float* p, float (&v)[8]) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st8(float* p, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

// The phi factor of node o, where the context keeps no table.
__device__ __noinline__ float phi_at(const TcArgs& p, unsigned o) {
    float z = p.zt[0][o % p.n1] + p.zt[1][(o / p.n1) % p.n2];
    if (p.zt[2]) z += p.zt[2][o / p.n1 / p.n2];
    return phi_eval(p.phik, z);
}

template <bool MODE1, int N, int EPI, bool LO>
__global__ void __launch_bounds__(kThreads, 1) tc_contract_kernel(const __grid_constant__ TcArgs p) {
    using C = Cfg<N>;
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t kF = 0, kE = kF + 8 * C::NS, kAF = kE + 8 * C::NS, kAE = kAF + 8 * C::SETS, kDR = kAE + 8 * C::SETS;
    __shared__ __align__(8) uint64_t bars[kDR / 8 + 1];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;     // state slices of the stages
    const uint32_t fbase = sbase + C::NS * C::SBYTES;                   // factor slices of the stages
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto full = [&](int s) { return bar0 + kF + 8u * s; };
    auto empty = [&](int s) { return bar0 + kE + 8u * s; };
    auto accf = [&](int a) { return bar0 + kAF + 8u * a; };
    auto acce = [&](int a) { return bar0 + kAE + 8u * a; };
    const uint32_t drain_bar = bar0 + kDR;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(full(s), kGroupWarps + 1);             // a warp of the chunk's group each, and the loader's expect_tx
            mbar_init(empty(s), 1);                          // tcgen05.commit
        }
        for (int a = 0; a < C::SETS; ++a) {
            mbar_init(accf(a), 1);
            mbar_init(acce(a), kEpiWarps);                   // one arrival per epilogue warp
        }
        mbar_init(drain_bar, 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                     "r"(C::TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;

    const float amax = __uint_as_float(*p.amax_in);
    int es = 0;
    if (amax > 0.f) frexpf(amax, &es);
    const float sc = ldexpf(1.f, 7 - es);
    const float sback = ldexpf(1.f, es - 7);
    const int n = p.n;
    const unsigned Q = MODE1 ? 1u : p.Q;
    const int items = (p.ntiles - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x) * p.nK;   // (tile, K chunk) in order

    if (warp == kLoadWarp) {
        // ------------------------------------------------------------ factor loader (bulk copies)
        if (lane == 0) {
            int s = 0, issued = 0;
            uint32_t ph = 1;
            for (int tile = blockIdx.x; tile < p.ntiles && !abort_s; tile += gridDim.x) {
                const uint8_t* src = p.fimg + size_t(tile % p.nOut) * p.nK * C::FBYTES;
                for (int c = 0; c < p.nK; ++c, src += C::FBYTES, ++issued) {
                    if (!mbar_wait(empty(s), ph, p.err, 64, &abort_s, 32)) break;
                    mbar_arrive_expect_tx(full(s), C::FBYTES);
                    bulk_g2s(fbase + s * C::FBYTES, src, C::FBYTES, full(s));
                    if (++s == C::NS) { s = 0; ph ^= 1; }
                }
            }
            // no copy may land after the CTA has gone (they have, unless a wait gave up)
            const long long t0 = clock64();
            for (int k = max(issued - C::NS, 0); k < issued; ++k)
                while (!mbar_try_wait(full(k % C::NS), uint32_t(k / C::NS) & 1u) && clock64() - t0 < kWaitCycles) {}
        }
    } else if (warp < kProducerWarps) {
        // ------------------------------------------------------------ producers (global -> slices)
        // Two groups of four warps take the chunks in turn: what a chunk costs besides its arithmetic (the wait for its
        // slot, the proxy fence, the arrivals) then passes while the other group slices (256^3: 79 us, 89 with one group of
        // eight). KG threads a line, each KV consecutive K values: neighbouring lanes along K for
        // mode 1, along the positions otherwise, so that a warp reads whole sectors.
        constexpr int KV = C::KV, KG = C::KG;
        const int t = threadIdx.x & (kGroupWarps * 32 - 1), group = warp / kGroupWarps;
        const int row = MODE1 ? t / KG : t % N, kofs = KV * (MODE1 ? t % KG : t / N);
        // the (tile, chunk) whose values are loaded next, and this thread's line of that tile
        int ltile = blockIdx.x, lc = 0;
        bool lrow = false;
        const float* xrow = nullptr;
        const float* xlo = nullptr;
        auto line = [&] {
            const unsigned pos = unsigned(ltile / p.nOut) * N + row;
            lrow = ltile < p.ntiles && pos < p.npos;
            const size_t off = MODE1 ? size_t(pos) * n + kofs : size_t(pos / Q) * n * Q + pos % Q + size_t(kofs) * Q;
            xrow = p.X + off;
            xlo = LO ? p.Xlo + off : nullptr;
        };
        auto advance = [&](int by) {
            lc += by;
            if (lc < p.nK) return;
            for (; lc >= p.nK; lc -= p.nK) ltile += gridDim.x;
            line();
        };
        auto load1 = [&](const float* x, float (&w)[KV]) {
            const int k0 = lc * kKc + kofs;
            x += size_t(lc * kKc) * Q;
            if (MODE1 && p.vec4) {
#pragma unroll
                for (int e = 0; e < KV; e += 4) {
                    const float4 u = ld4_or_0(x + e, lrow && k0 + e < n);
                    w[e] = u.x; w[e + 1] = u.y; w[e + 2] = u.z; w[e + 3] = u.w;
                }
            } else {
#pragma unroll
                for (int e = 0; e < KV; ++e) w[e] = ld1_or_0(x + size_t(e) * Q, lrow && k0 + e < n);
            }
        };
        // chunks held in registers while the ones before them are sliced: 79 us at 256^3, 90 with one (two with low parts would not fit)
        constexpr int DEPTH = LO ? 1 : 2;
        float v[DEPTH][KV], vl[KV];
        line();
        advance(group);
#pragma unroll
        for (int b = 0; b < DEPTH; ++b) {
            if (b > 0) advance(kGroups);
            load1(xrow, v[b]);
            if (LO) load1(xlo, vl);
        }
        bool ok = true;
        for (int it0 = group; it0 < items && ok; it0 += kGroups * DEPTH)
#pragma unroll
            for (int b = 0; b < DEPTH; ++b) {
                const int it = it0 + b * kGroups, s = it % C::NS;
                if (it >= items || !ok) break;
                // waits decide warp-uniformly: the per-warp arrivals need every lane
                ok = __all_sync(0xffffffffu, mbar_wait(empty(s), (uint32_t(it / C::NS) & 1u) ^ 1u, p.err, 1, &abort_s, 32));
                if (!ok) break;
                slice_store<C::STILE, KV, LO>(v[b], vl, sc, sbase + s * C::SBYTES, row, kofs);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(full(s));
                advance(kGroups);
                load1(xrow, v[b]);                           // in flight for DEPTH rounds of both groups
                if (LO) load1(xlo, vl);
            }
    } else if (warp < kMmaWarp) {
        // ------------------------------------------------------------ epilogue
        const int ew = (warp - kProducerWarps) & 3;          // TMEM lane quarter (warp % 4)
        const int part = (warp - kProducerWarps) >> 2;       // column part
        const int jlo = part * C::COLS;
        float vmax = 0.f;
        int tl = 0;
        for (int tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++tl) {
            const int a = tl % C::SETS;
            const int pt = tile / p.nOut, ot = tile % p.nOut;
            const int irow = ot * kM + ew * 32 + lane;       // this lane's output
            const bool rvalid = irow < n, warp_on = ot * kM + ew * 32 < n;
            const float scale = sback * __ldg(p.fscale + irow);   // padded to whole tiles
            const unsigned ioff = unsigned(irow) * Q;
            const int ncol = min(N, int(p.npos - unsigned(pt) * N));
            // lane c: the offset of column jlo + c (one division a tile)
            const unsigned cpos = unsigned(pt) * N + jlo + lane;
            const unsigned coff = MODE1 ? cpos * n : (cpos / Q) * n * Q + cpos % Q;
            auto off_of = [&](int j) { return __shfl_sync(0xffffffffu, coff, j) + ioff; };   // column jlo + j
            // the axpy's base or the phi table's values of eight columns, one group ahead
            auto load_side = [&](int j0, float (&b)[8]) {
                if (EPI != EPI_AXPY && EPI != EPI_PHI) return;
                const float* src = EPI == EPI_PHI ? p.phi : p.base;
                if (!MODE1 && p.vec8 && src && jlo + j0 + 8 <= ncol) {
                    const unsigned o = off_of(j0);           // every lane takes part in the shuffles
                    if (rvalid) ld8(src + o, b);
                    return;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const unsigned o = off_of(j0 + j);
                    b[j] = 0.f;
                    if (rvalid && jlo + j0 + j < ncol) b[j] = EPI == EPI_AXPY || src ? src[o] : phi_at(p, o);
                }
            };
            float side[2][8];
            if (warp_on) load_side(0, side[0]);
            const bool waited = mbar_wait(accf(a), uint32_t(tl / C::SETS) & 1u, p.err, 2, &abort_s, 32);
            if (!__all_sync(0xffffffffu, waited)) break;
            tc_fence_after();
            if (!warp_on) {
                if (lane == 0) mbar_arrive(acce(a));
                continue;
            }
            const uint32_t tbase = tmem + (uint32_t(ew * 32) << 16) + uint32_t(a * kSl * N + jlo);
#pragma unroll(EPI == EPI_AXPY || EPI == EPI_PHI ? C::COLS / 8 : 1)
            for (int j0 = 0; j0 < C::COLS; j0 += 8) {
                float d[4][8];
                const float (&bcur)[8] = side[(j0 >> 3) & 1];
                if (j0 + 8 < C::COLS) load_side(j0 + 8, side[((j0 >> 3) + 1) & 1]);
                __syncwarp();
                tmem_ld8x4(tbase + j0, uint32_t(N), d);
                if (j0 + 8 >= C::COLS) {                     // the last columns are in registers: the set is free
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acce(a));
                }
                float v[8], vl[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float tail = fmaf(d[3][j], 5.9604644775390625e-08f, d[2][j] * 1.52587890625e-05f);
                    if (EPI == EPI_STORE2) {                 // double-float result: D0 + 2^-8 D1 exactly, then the tail
                        float hi, lo;
                        two_sum(d[0][j], d[1][j] * 0.00390625f, hi, lo);
                        lo += tail;
                        const float s = hi + lo;
                        v[j] = s * scale;
                        vl[j] = (lo - (s - hi)) * scale;
                    } else {                                 // one FP32 result: the smaller terms first, D0 last
                        v[j] = (d[0][j] + fmaf(d[1][j], 0.00390625f, tail)) * scale;
                        if (EPI == EPI_PHI) v[j] *= bcur[j];
                        if (EPI == EPI_AXPY) v[j] = fmaf(p.alpha, v[j], bcur[j]);
                    }
                }
                if (!MODE1 && p.vec8 && jlo + j0 + 8 <= ncol) {
                    const unsigned o = off_of(j0);
                    if (rvalid) {
                        st8(p.Y + o, v);
                        if (EPI == EPI_STORE2) st8(p.Ylo + o, vl);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const unsigned o = off_of(j0 + j);
                        if (rvalid && jlo + j0 + j < ncol) {
                            p.Y[o] = v[j];
                            if (EPI == EPI_STORE2) p.Ylo[o] = vl[j];
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (rvalid && jlo + j0 + j < ncol) vmax = fmaxf(vmax, fabsf(v[j]));
            }
        }
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if (lane == 0 && p.amax_out && vmax > 0.f) atomicMax(p.amax_out, __float_as_uint(vmax));
    } else if (warp == kMmaWarp && lane == 0) {
        // ------------------------------------------------------------ MMA issuer
        // F_i.S_j adds to D_(i+j). The S tiles lie one after another, as do the accumulators, so F_i takes
        // S_0..S_(3-i) in one MMA of up to 256 columns: four MMAs per K step instead of ten, and F_i is
        // read from shared memory once.
        uint32_t ph = 0;
        int s = 0, tl = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < p.ntiles && !abort_s && ok; tile += gridDim.x, ++tl) {
            const int a = tl % C::SETS;
            if (!mbar_wait(acce(a), (uint32_t(tl / C::SETS) & 1u) ^ 1u, p.err, 4, &abort_s)) break;
            tc_fence_after();
            const uint32_t d = tmem + uint32_t(a * kSl * N);
            for (int c = 0; c < p.nK; ++c) {
                if (!mbar_wait(full(s), ph, p.err, 8, &abort_s)) { ok = false; break; }
                tc_fence_after();
                const uint64_t a0 = sdesc64(fbase + s * C::FBYTES), b0 = sdesc64(sbase + s * C::SBYTES);
#pragma unroll
                for (int kk = 0; kk < kKc / 16; ++kk) {
                    const uint64_t adv = uint64_t(kk * 32) >> 4;
#pragma unroll
                    for (int i = 0; i < kSl; ++i)
                        tc_mma(d + i * N, a0 + adv + uint64_t(i * C::FTILE >> 4), b0 + adv, idesc_of((kSl - i) * N),
                               (c == 0 && kk == 0 && i == 0) ? 0u : 1u);
                }
                tc_commit(empty(s));
                if (++s == C::NS) { s = 0; ph ^= 1; }
            }
            if (ok) tc_commit(accf(a));
        }
        tc_commit(drain_bar);
        const long long t0 = clock64();
        while (!mbar_try_wait(drain_bar, 0) && clock64() - t0 < kWaitCycles) {}
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM) : "memory");
    }
}

__global__ void phi_table_kernel(float* tab, int k, const float* z1, const float* z2, const float* z3, int n1, int n2, size_t N) {
    for (size_t o = blockIdx.x * size_t(blockDim.x) + threadIdx.x; o < N; o += size_t(gridDim.x) * blockDim.x) {
        float z = z1[o % n1] + z2[(o / n1) % n2];
        if (z3) z += z3[o / n1 / n2];
        tab[o] = phi_eval(k, z);
    }
}

int sm_count() {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 1;
    }();
    return sms;
}

template <bool MODE1, int N, int EPI, bool LO>
cudaError_t launch_variant(const TcArgs& a, cudaStream_t s) {
    static SmemLimit smem;
    const cudaError_t e = smem.allow(reinterpret_cast<const void*>(tc_contract_kernel<MODE1, N, EPI, LO>), Cfg<N>::SMEM);
    if (e != cudaSuccess) return e;
    const int grid = a.ntiles < sm_count() ? a.ntiles : sm_count();
    tc_contract_kernel<MODE1, N, EPI, LO><<<unsigned(grid), kThreads, Cfg<N>::SMEM, s>>>(a);
    return cudaGetLastError();
}

template <bool MODE1, int N>
cudaError_t launch_epi(const TcArgs& a, cudaStream_t s) {
    if (a.Xlo) return a.epi == EPI_STORE2 ? launch_variant<MODE1, N, EPI_STORE2, true>(a, s) : cudaErrorInvalidValue;
    switch (a.epi) {
    case EPI_STORE2: return launch_variant<MODE1, N, EPI_STORE2, false>(a, s);
    case EPI_AXPY: return launch_variant<MODE1, N, EPI_AXPY, false>(a, s);
    case EPI_PHI:                                            // always fused into the last direction's pass
        if constexpr (MODE1) return cudaErrorInvalidValue;
        else return launch_variant<false, N, EPI_PHI, false>(a, s);
    default: return launch_variant<MODE1, N, EPI_STORE, false>(a, s);
    }
}

}  // namespace

cudaError_t launch_phi_table(float* tab, int k, const float* const zt[3], int n1, int n2, size_t N, cudaStream_t s) {
    const unsigned blocks = unsigned((N + 255) / 256 < 65535 ? (N + 255) / 256 : 65535);
    phi_table_kernel<<<blocks, 256, 0, s>>>(tab, k, zt[0], zt[1], zt[2], n1, n2, N);
    return cudaGetLastError();
}

cudaError_t launch_contract_tc(TcArgs a, cudaStream_t s) {
    if (a.n > 512 || a.n < 1) return cudaErrorInvalidValue;
    if (a.npos == 0) return cudaSuccess;
    const bool mode1 = a.Q == 1;
    a.nK = (a.n + kKc - 1) / kKc;
    a.nOut = (a.n + kM - 1) / kM;
    auto aligned = [](const void* q, uintptr_t to) { return reinterpret_cast<uintptr_t>(q) % to == 0; };
    a.vec4 = a.n % 4 == 0 && aligned(a.X, 16) && aligned(a.Xlo, 16);
    // groups of eight columns are eight consecutive nodes: modes >= 2, q a multiple of 8
    a.vec8 = !mode1 && a.Q % 8 == 0 && aligned(a.Y, 32) && aligned(a.Ylo, 32) && aligned(a.base, 32) && aligned(a.phi, 32);
    const bool wide = (a.npos + 63) / 64 * a.nOut >= unsigned(sm_count());
    a.ntiles = int((a.npos + (wide ? 63 : 31)) / (wide ? 64 : 32) * a.nOut);
    if (mode1) return wide ? launch_epi<true, 64>(a, s) : launch_epi<true, 32>(a, s);
    return wide ? launch_epi<false, 64>(a, s) : launch_epi<false, 32>(a, s);
}

}  // namespace adr
