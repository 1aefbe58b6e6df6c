// K2 on the tensor cores for batched 2-D contexts in mixed precision: the mu-mode products
// of Section 1 / Section 5.2 for every instance of a batch in one persistent launch, with
// compensated (hi + lo) FP32 inputs and outputs, the pointwise phi_k scaling (K3) and the
// stage axpy (K4) fused into the epilogue.
//
// Exact-slice split with five state slices. The input x = hi + lo of instance i gets the
// scale 2^(es_i - 7) from max|x| over that instance (recorded by the kernel that produced
// it); each factor row r its own 2^(e_r - 7):
//     x = 2^(es-7) (S0 + 2^-8 S1 + 2^-16 S2 + 2^-24 S3 + 2^-32 S4)   up to 2^-40 of max|x|,
//     f = 2^(e-7)  (F0 + 2^-8 F1 + 2^-16 F2 + 2^-24 F3)              up to 2^-32 of the row max,
// integer slices |S_j|, |F_j| <= 128, exact in BF16. The fourteen products with i + j <= 4
// go into four TMEM accumulators per output:
//     D0 = S0 F0,   D1 = S0 F1 + S1 F0,   D2 = S0 F2 + S1 F1 + S2 F0,
//     D3 = S0 F3 + S1 F2 + S2 F1 + S3 F0 + 2^-8 (S1 F3 + S2 F2 + S3 F1 + S4 F0),
// the 2^-8 terms through pre-scaled tiles (2^-8 F1, F2, F3 sliced on the host, 2^-8 S4 by the
// producers; exact scalings). For K <= 256 D0, D1 and D2 are sums of integers below 2^24 and
// exact whatever rounding the tensor cores apply; D3 rounds at 2^-24 of itself, some 2^-48 of
// the result. The epilogue forms D0 + 2^-8 D1 + 2^-16 D2 + 2^-24 D3 in double-float
// arithmetic. With four slices of the state (ten products), or without the cross products
// at 2^-32, an FP64 emulation of the batched ETD2RK workload ends at 1.5e-4 on its worst
// instance; with these fourteen at 1.0e-6.
//
// CTA (persistent, one per SM). The factor is the A operand, 128 outputs (TMEM lanes) a tile, and 64 lines of one
// instance (x2 rows in mode 1, x1 positions in mode 2) are the B operand; two TMEM accumulator sets (2 x 4 x 64
// columns) let the epilogue of a tile overlap the next tile's MMAs. Warps 0-7 load the FP32 pairs two K chunks ahead, slice
// them and store 64-byte-swizzled K-major BF16 tiles; warps 8-15 are the epilogue; warp 16 issues the MMAs, warp 17
// copies the pre-sliced factor tiles, warp 18 looks up what each tile is (instance, offsets, scales: three dependent loads
// a tile, 32 tiles at a time) into a ring that all the others read. Every mbarrier wait is bounded; on a
// timeout the CTA records an error code, drains its MMAs and frees TMEM.
// On the 512-instance ETD2RK workload a pass (mode 1 store, mode 2 phi, mode 2 store, mode 1 axpy) takes 90, 119, 102 and
// 129 us; 98, 186, 160 and 129 with 128 positions x 64 outputs in mode 2 (each state tile sliced once per 64
// outputs), a rounding instruction in the slicing, one chunk ahead, and every role looking its tile up itself.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#include "adr_internal.h"
#include "smem_limit.h"
#include "tc_common.cuh"

namespace adr {
namespace {
using namespace tc;

constexpr int kM = 128;                 // UMMA M, TMEM lanes: outputs
constexpr int kN = 64;                  // UMMA N: lines, columns of each accumulator
constexpr int kKc = 32;                 // K per stage: one 64-byte BF16 row
constexpr int kSS = 5;                  // state slice tiles: S0..S3, 2^-8 S4
constexpr int kFS = 7;                  // factor slice tiles: F0..F3, 2^-8 F1..F3
static_assert(kM == kBatchTcRows1 && kKc == kBatchTcChunk && kFS == kBatchTcFactorTiles,
              "the host slicing (host_setup.cpp) writes the tiles this kernel reads");
constexpr int kNacc = 4;
constexpr int kProducerWarps = 8;
constexpr int kEpiWarps = 8;
constexpr int kMmaWarp = kProducerWarps + kEpiWarps;
constexpr int kLoadWarp = kMmaWarp + 1;
constexpr int kDescWarp = kMmaWarp + 2;
constexpr int kThreads = (kDescWarp + 1) * 32;
constexpr uint32_t kTmemCols = 512;     // two sets of kNacc x kN columns
static_assert(2 * kNacc * kN <= int(kTmemCols), "TMEM");
constexpr int kSTile = kN * kKc * 2, kFTile = kM * kKc * 2;      // one slice tile
constexpr int kSBytes = kSS * kSTile, kFBytes = kFS * kFTile;    // one stage: 20 KB and 56 KB
constexpr int kNS = 4, kNF = 2;                                   // ring stages
constexpr int kSmem = kNS * kSBytes + kNF * kFBytes + 1024;
static_assert(kSmem <= 222 * 1024, "shared memory budget");
constexpr int kCols = kN / (kEpiWarps / 4);                       // columns per epilogue warp
constexpr int kKV = kN * kKc / (kProducerWarps * 32);             // K values a producer thread slices per chunk
static_assert(kKV == 8, "one 16-byte chunk of a slice row per producer thread");

// What a tile is, as the roles read it.
struct Desc {
    long long off;                      // the instance's elements in the packed arrays
    long long img;                      // its factor image (bytes), at this output tile
    long long fsc;                      // its row scales
    int n1, n2, inst, line0, out0, nK, vec;
    int es;                             // max|x| < 2^es
};
constexpr int kDescs = 8;
constexpr int kDescReaders = kProducerWarps + kEpiWarps + 2;      // + MMA issuer, loader

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void quick_two_sum(float a, float b, float& s, float& e) {   // |a| >= |b|
    s = a + b;
    e = b - (s - a);
}
// (ah + al) (bh + bl) in double-float arithmetic
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float& h, float& l) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, fmaf(al, bh, e));
    quick_two_sum(p, e, h, l);
}
__device__ __forceinline__ void df_add(float ah, float al, float bh, float bl, float& h, float& l) {
    float s, e;
    two_sum(ah, bh, s, e);
    e += al + bl;
    quick_two_sum(s, e, h, l);
}

// Five integer slices of y + ylo (|y + ylo| <= 128 + a rounding), as FP32 patterns whose upper
// halves are the exact BF16 values: S0..S3 and 2^-8 S4. The steps y - rint(y) and the scalings
// by 256 are exact; the low part enters once through an exact TwoSum, its rounding error at
// the last slice, where only products below 2^-40 of the scale are left out.
__device__ __forceinline__ void split5(float y, float ylo, uint32_t (&b)[kSS]) {
    const float s0 = rint_small(y);
    float a = (y - s0) * 256.f;
    const float s1 = rint_small(a);
    a = (a - s1) * 256.f;
    float t, e;
    two_sum(a, ylo * 65536.f, t, e);
    const float s2 = rint_small(t);
    a = (t - s2) * 256.f;
    const float s3 = rint_small(a);
    a = fmaf(e, 65536.f, (a - s3) * 256.f);
    const float s4 = rint_small(a);
    b[0] = __float_as_uint(s0);
    b[1] = __float_as_uint(s1);
    b[2] = __float_as_uint(s2);
    b[3] = __float_as_uint(s3);
    b[4] = __float_as_uint(s4 * 0.00390625f);
}

// Slice 8 consecutive K values (+ low parts) into 16-byte chunk j of row r of the five state tiles.
__device__ __forceinline__ void slice_store8(const float (&v)[8], const float (&vl)[8], float sc, uint32_t tile0, int r, int j) {
    uint32_t w[kSS][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        uint32_t a[kSS], c[kSS];
        split5(v[2 * e] * sc, vl[2 * e] * sc, a);
        split5(v[2 * e + 1] * sc, vl[2 * e + 1] * sc, c);
#pragma unroll
        for (int q = 0; q < kSS; ++q) w[q][e] = __byte_perm(a[q], c[q], 0x7632);
    }
    const uint32_t off = swz64(r, j);
#pragma unroll
    for (int q = 0; q < kSS; ++q) st_shared_v4(tile0 + q * kSTile + off, make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]));
}

// Scale of an instance's input from its recorded max|x| (< 2^es): x * 2^(7 - es) in [-128, 128].
__device__ __forceinline__ int input_exponent(const unsigned* amax, int inst) {
    const float m = __uint_as_float(__ldg(amax + inst));
    int es = 0;
    if (m > 0.f) frexpf(m, &es);
    return es;
}

// Instruction descriptor of an M = 128 product of N columns (BF16 inputs, FP32 accumulate).
constexpr uint32_t idesc_n(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(n >> 3) << 17) | (uint32_t(kM >> 4) << 24);
}

// One K step of 16 of the fourteen products. The accumulators D0..D3 sit in consecutive kN-column
// blocks of TMEM and the slice tiles of each operand in consecutive shared-memory tiles, so one
// factor slice against r consecutive state slices is one product of r kN columns that adds each pair to
// its own accumulator: eight MMAs (N = 256, 192, 128 and five of 64) instead of fourteen of
// N = 64: F0.[S0..S3] -> D0..D3, F1.[S0..S2] -> D1..D3, F2.[S0 S1] -> D2 D3, and
// into D3: F0 (2^-8 S4), F3 S0, (2^-8 F1) S3, (2^-8 F2) S2, (2^-8 F3) S1.
__device__ __forceinline__ void mma_kstep(uint32_t d, uint64_t F, uint64_t S, uint32_t first) {
    auto mma = [&](int acc, int f, int s, int nacc, uint32_t accumulate) {
        tc_mma(d + uint32_t(acc * kN), F + uint64_t(f * kFTile >> 4), S + uint64_t(s * kSTile >> 4), idesc_n(nacc * kN), accumulate);
    };
    mma(0, 0, 0, 4, first ? 0u : 1u);
    mma(1, 1, 0, 3, 1u);
    mma(2, 2, 0, 2, 1u);
    mma(3, 0, 4, 1, 1u);
    mma(3, 3, 0, 1, 1u);
    mma(3, 4, 3, 1, 1u);
    mma(3, 5, 2, 1, 1u);
    mma(3, 6, 1, 1, 1u);
}

// Load 4 columns of the four accumulators (kN columns apart) for this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld4x4(uint32_t t0, float (&d)[4][4]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%16];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%17];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%18];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%19];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(t0), "r"(t0 + uint32_t(kN)), "r"(t0 + uint32_t(2 * kN)), "r"(t0 + uint32_t(3 * kN))
        : "memory");
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) d[k][j] = __uint_as_float(r[4 * k + j]);
}

__device__ __forceinline__ void ldv4(const float* p, float (&v)[4]) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}

template <bool MODE1, int EPI>
__global__ void __launch_bounds__(kThreads, 1) batch_tc_kernel(const __grid_constant__ BatchTcArgs p) {
    extern __shared__ uint8_t smem_raw[];
    // barriers: sfull[NS] sempty[NS] ffull[NF] fempty[NF] accf[2] acce[2] drain dfull[kDescs] dempty[kDescs]
    constexpr int kB = 2 * kNS + 2 * kNF + 5;
    __shared__ __align__(8) uint64_t bars[kB + 2 * kDescs];
    __shared__ Desc descs[kDescs];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;   // state-slice ring
    const uint32_t fbase = sbase + kNS * kSBytes;                     // factor ring
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto sfull = [&](int s) { return bar0 + 8u * s; };
    auto sempty = [&](int s) { return bar0 + 8u * (kNS + s); };
    auto ffull = [&](int s) { return bar0 + 8u * (2 * kNS + s); };
    auto fempty = [&](int s) { return bar0 + 8u * (2 * kNS + kNF + s); };
    const uint32_t acc0 = bar0 + 8u * (2 * kNS + 2 * kNF);
    auto accf = [&](int a) { return acc0 + 8u * a; };
    auto acce = [&](int a) { return acc0 + 8u * (2 + a); };
    const uint32_t drain_bar = acc0 + 8u * 4;
    auto dfull = [&](int s) { return bar0 + 8u * (kB + s); };
    auto dempty = [&](int s) { return bar0 + 8u * (kB + kDescs + s); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kNS; ++s) {
            mbar_init(sfull(s), kProducerWarps);                // one arrival per producer warp
            mbar_init(sempty(s), 1);                            // tcgen05.commit
        }
        for (int s = 0; s < kNF; ++s) {
            mbar_init(ffull(s), 1);                             // the loader's expect_tx arrival
            mbar_init(fempty(s), 1);                            // tcgen05.commit
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(accf(a), 1);                              // tcgen05.commit
            mbar_init(acce(a), kEpiWarps);                      // one arrival per epilogue warp
        }
        mbar_init(drain_bar, 1);
        for (int s = 0; s < kDescs; ++s) {
            mbar_init(dfull(s), 1);
            mbar_init(dempty(s), kDescReaders);                 // one arrival per role's warp
        }
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    constexpr int dir = MODE1 ? 0 : 1;               // direction of the factor (mode - 1)
    const int ntiles = (p.nitems - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x);   // of this CTA

    if (warp == kDescWarp) {
        // ------------------------------------------------------------ tile descriptors
        bool ok = true;
        for (int t0 = 0; t0 < ntiles && ok; t0 += 32) {
            Desc d = {};
            if (t0 + lane < ntiles) {
                const int4 item = __ldg(p.items + blockIdx.x + (long long)(t0 + lane) * gridDim.x);
                const BatchTcInst& in = p.inst[item.x];
                d.off = in.off;
                d.n1 = in.n1;
                d.n2 = in.n2;
                d.inst = item.x;
                d.line0 = item.y * kN;
                d.out0 = item.z * kM;
                d.nK = ((MODE1 ? in.n1 : in.n2) + kKc - 1) / kKc;
                d.img = in.img_off[p.role][dir] + (long long)item.z * d.nK * kFBytes;
                d.fsc = in.fsc_off[p.role][dir];
                d.vec = in.vec;
                d.es = input_exponent(p.amax_in, item.x);
            }
            for (int i = 0; i < 32 && t0 + i < ntiles && ok; ++i) {
                const int t = t0 + i, s = t % kDescs;
                ok = __all_sync(0xffffffffu, mbar_wait(dempty(s), (uint32_t(t / kDescs) & 1u) ^ 1u, p.err, 64, &abort_s, 64));
                if (ok && lane == i) {
                    descs[s] = d;
                    mbar_arrive(dfull(s));
                }
                __syncwarp();
            }
        }
    } else if (warp < kProducerWarps) {
        // ------------------------------------------------------------ producers
        // Four threads a line, each 8 consecutive K values of a chunk: neighbouring lanes along K in mode 1, along the
        // positions in mode 2, so that a warp reads whole sectors.
        const int t = threadIdx.x;
        const int row = MODE1 ? t >> 2 : t & (kN - 1), kg = MODE1 ? t & 3 : t / kN;
        // the (tile, chunk) loaded next
        int lt = 0, lc = 0, nK = 0, len = 0;
        bool lrow = false, vec = false;
        long long step = 1;
        const float* xh = nullptr;
        const float* xl = nullptr;
        float lsc = 0.f;
        bool ok = true;
        auto open = [&]() {                                     // warp-uniform
            if (lt >= ntiles || !ok) { ok = ok && lt < ntiles; return; }
            const int s = lt % kDescs;
            ok = __all_sync(0xffffffffu, mbar_wait(dfull(s), uint32_t(lt / kDescs) & 1u, p.err, 64, &abort_s, 32));
            if (!ok) return;
            const Desc& d = descs[s];
            nK = d.nK;
            const int line = d.line0 + row;
            lrow = line < (MODE1 ? d.n2 : d.n1);
            len = MODE1 ? d.n1 : d.n2;
            step = MODE1 ? 1 : d.n1;
            vec = MODE1 && d.vec;
            const long long o = d.off + (MODE1 ? (long long)line * d.n1 : (long long)line) + 8 * kg * step;
            xh = p.X + o;
            xl = p.Xlo ? p.Xlo + o : nullptr;
            lsc = ldexpf(1.f, 7 - d.es);
            __syncwarp();
            if (lane == 0) mbar_arrive(dempty(s));
        };
        auto load1 = [&](const float* x, float (&w)[8]) {
            const int k0 = lc * kKc + 8 * kg;
            x += (long long)(lc * kKc) * step;
            if (MODE1 && vec && lrow && k0 + 8 <= len) {
                const float4 a = ld4_or_0(x, true), b = ld4_or_0(x + 4, true);
                w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
                w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) w[e] = ld1_or_0(x + (long long)e * step, lrow && k0 + e < len);
            }
        };
        auto load = [&](float (&w)[8], float (&wl)[8], float& sc) -> bool {   // false: no chunk left
            if (!ok) return false;
            sc = lsc;
            load1(xh, w);
            if (xl) {
                load1(xl, wl);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) wl[e] = 0.f;
            }
            if (++lc == nK) {
                lc = 0;
                ++lt;
                open();
            }
            return true;
        };
        int ss = 0;
        uint32_t sph = 1;
        auto put = [&](float (&w)[8], float (&wl)[8], float sc) -> bool {
            // warp-uniform decision: the per-warp arrival below needs every lane
            if (!__all_sync(0xffffffffu, mbar_wait(sempty(ss), sph, p.err, 1, &abort_s, 32))) return false;
            slice_store8(w, wl, sc, sbase + ss * kSBytes, row, kg);
            // one arrival per warp once every lane's slices are visible to the tensor cores
            // (256 single-thread arrivals on one barrier word serialise)
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(sfull(ss));
            if (++ss == kNS) { ss = 0; sph ^= 1; }
            return true;
        };
        float va[8], la[8], vb[8], lb[8], sa = 0.f, sb = 0.f;
        open();
        bool ha = load(va, la, sa), hb = load(vb, lb, sb);
        while (ha) {                                            // the loads of two chunks are in flight
            if (!put(va, la, sa)) break;
            ha = load(va, la, sa);
            if (!hb) break;
            if (!put(vb, lb, sb)) break;
            hb = load(vb, lb, sb);
        }
    } else if (warp < kMmaWarp) {
        // ------------------------------------------------------------ epilogue
        const int ew = (warp - kProducerWarps) & 3;             // TMEM lane quarter (warp % 4)
        const int jlo = ((warp - kProducerWarps) >> 2) * kCols;
        const float ah = float(p.alpha);
        const float al = float(p.alpha - double(ah));
        for (int tl = 0; tl < ntiles; ++tl) {
            const int a = tl & 1, ds = tl % kDescs;
            if (!__all_sync(0xffffffffu, mbar_wait(dfull(ds), uint32_t(tl / kDescs) & 1u, p.err, 64, &abort_s, 32))) break;
            const Desc d = descs[ds];
            __syncwarp();
            if (lane == 0) mbar_arrive(dempty(ds));
            const int out = d.out0 + ew * 32 + lane;            // this lane's output
            const int nout = MODE1 ? d.n1 : d.n2, ncol = min(kN, (MODE1 ? d.n2 : d.n1) - d.line0);
            const bool rvalid = out < nout, warp_on = d.out0 + ew * 32 < nout && jlo < ncol;
            const float scale = rvalid ? ldexpf(1.f, d.es - 7) * __ldg(p.fscale + d.fsc + out) : 0.f;
            // column j of this lane: mode 1 x2 row line0 + j, output along x1; mode 2 the other way
            const long long off0 = d.off + (MODE1 ? (long long)d.line0 * d.n1 + out : (long long)out * d.n1 + d.line0);
            const long long cstep = MODE1 ? d.n1 : 1;
            const bool vec = !MODE1 && d.vec && p.al16;         // four columns are 16 aligned bytes
            // the phi table's pairs or the axpy's base of four columns, one group ahead
            auto load_ops = [&](int j0, float (&x)[4], float (&y)[4]) {
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = y[j] = 0.f;
                if (EPI == EPI_STORE || !rvalid) return;
                const long long o = off0 + (long long)j0 * cstep;
                if (vec && j0 + 4 <= ncol) {
                    if (EPI == EPI_PHI) {
                        float u[4], w[4];
                        ldv4(reinterpret_cast<const float*>(p.phi + o), u);
                        ldv4(reinterpret_cast<const float*>(p.phi + o) + 4, w);
                        x[0] = u[0]; y[0] = u[1]; x[1] = u[2]; y[1] = u[3];
                        x[2] = w[0]; y[2] = w[1]; x[3] = w[2]; y[3] = w[3];
                    } else {
                        ldv4(p.base + o, x);
                        if (p.base_lo) ldv4(p.base_lo + o, y);
                    }
                    return;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j0 + j >= ncol) continue;
                    const long long oj = o + (long long)j * cstep;
                    if (EPI == EPI_PHI) {
                        const float2 f = __ldg(p.phi + oj);
                        x[j] = f.x;
                        y[j] = f.y;
                    } else {
                        x[j] = p.base[oj];
                        if (p.base_lo) y[j] = p.base_lo[oj];
                    }
                }
            };
            float xs[2][4], ys[2][4];
            if (warp_on) load_ops(jlo, xs[0], ys[0]);
            const bool waited = mbar_wait(accf(a), uint32_t(tl >> 1) & 1u, p.err, 2, &abort_s, 32);
            if (!__all_sync(0xffffffffu, waited)) break;        // warp-uniform: TMEM loads are .sync.aligned
            tc_fence_after();
            if (!warp_on) {
                if (lane == 0) mbar_arrive(acce(a));
                continue;
            }
            float vmax = 0.f;
            const uint32_t tbase = tmem + (uint32_t(ew * 32) << 16) + uint32_t(a * kNacc * kN);
            const int jhi = min(jlo + kCols, (ncol + 3) & ~3);
            // in pairs of groups, so that no register move waits for a load (a group past jhi is skipped whole)
#pragma unroll 1
            for (int jp = jlo; jp < jhi; jp += 8)
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                const int j0 = jp + 4 * h2;
                if (j0 >= jhi) break;
                const float (&xc)[4] = xs[h2];
                const float (&yc)[4] = ys[h2];
                float c[4][4];
                if (j0 + 4 < jhi) load_ops(j0 + 4, xs[h2 ^ 1], ys[h2 ^ 1]);
                __syncwarp();
                tmem_ld4x4(tbase + j0, c);
                if (j0 + 4 >= jhi) {                            // the last columns are in registers: the set is free
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acce(a));
                }
                float h[4], l[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // D0 + 2^-8 D1 + 2^-16 D2 + 2^-24 D3 in double-float arithmetic
                    float hi, lo;
                    two_sum(c[0][j], c[1][j] * 0.00390625f, hi, lo);
                    lo += fmaf(c[3][j], 5.9604644775390625e-08f, c[2][j] * 1.52587890625e-05f);
                    quick_two_sum(hi, lo, hi, lo);
                    hi *= scale;                                // a power of two: exact
                    lo *= scale;
                    if (EPI == EPI_PHI) {
                        df_mul(hi, lo, xc[j], yc[j], hi, lo);
                    } else if (EPI == EPI_AXPY) {
                        float th, tl2;
                        df_mul(ah, al, hi, lo, th, tl2);
                        df_add(xc[j], yc[j], th, tl2, hi, lo);
                    }
                    if (!p.Ylo) hi = hi + lo;
                    h[j] = hi;
                    l[j] = lo;
                }
                if (!rvalid) continue;
                const long long o = off0 + (long long)j0 * cstep;
                if (vec && j0 + 4 <= ncol) {
                    const float4 hv = make_float4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<float4*>(p.Y + o) = hv;
                    if (p.Ylo) *reinterpret_cast<float4*>(p.Ylo + o) = make_float4(l[0], l[1], l[2], l[3]);
                    if (p.Yhs) *reinterpret_cast<float4*>(p.Yhs + o) = hv;
                    vmax = fmaxf(vmax, fmaxf(fmaxf(fabsf(h[0]), fabsf(h[1])), fmaxf(fabsf(h[2]), fabsf(h[3]))));
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (j0 + j >= ncol) continue;
                        const long long oj = o + (long long)j * cstep;
                        p.Y[oj] = h[j];
                        if (p.Ylo) p.Ylo[oj] = l[j];
                        if (p.Yhs) p.Yhs[oj] = h[j];
                        vmax = fmaxf(vmax, fabsf(h[j]));
                    }
                }
            }
            for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
            if (lane == 0 && p.amax_out && vmax > 0.f) atomicMax(p.amax_out + d.inst, __float_as_uint(vmax));
        }
    } else if (warp == kLoadWarp) {
        // ------------------------------------------------------------ factor loader
        // The CTA's chunks in the same order as the MMA issuer; a ring slot frees when the MMAs
        // of the chunk kNF earlier retire.
        if (lane == 0) {
            int s = 0, issued = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (int tl = 0; tl < ntiles && ok && !abort_s; ++tl) {
                const int ds = tl % kDescs;
                if (!mbar_wait(dfull(ds), uint32_t(tl / kDescs) & 1u, p.err, 64, &abort_s, 32)) break;
                const uint8_t* src = p.fimg + descs[ds].img;
                const int nK = descs[ds].nK;
                mbar_arrive(dempty(ds));
                for (int c = 0; c < nK; ++c, ++issued, src += kFBytes) {
                    if (!mbar_wait(fempty(s), ph, p.err, 32, &abort_s, 32)) { ok = false; break; }
                    mbar_arrive_expect_tx(ffull(s), kFBytes);
                    bulk_g2s(fbase + s * kFBytes, src, kFBytes, ffull(s));   // the seven tiles are contiguous
                    if (++s == kNF) { s = 0; ph ^= 1; }
                }
            }
            // no copy may land after the CTA has gone (they have, unless a wait gave up)
            const long long t0 = clock64();
            for (int k = max(issued - kNF, 0); k < issued; ++k)
                while (!mbar_try_wait(ffull(k % kNF), uint32_t(k / kNF) & 1u) && clock64() - t0 < kWaitCycles) {}
        }
    } else if (warp == kMmaWarp && lane == 0) {
        // ------------------------------------------------------------ MMA issuer
        int s = 0, fs = 0;
        uint32_t sph = 0, fph = 0;
        bool ok = true;
        for (int tl = 0; tl < ntiles && ok && !abort_s; ++tl) {
            const int ds = tl % kDescs, a = tl & 1;
            if (!mbar_wait(dfull(ds), uint32_t(tl / kDescs) & 1u, p.err, 64, &abort_s)) break;
            const int nK = descs[ds].nK;
            mbar_arrive(dempty(ds));
            if (!mbar_wait(acce(a), (uint32_t(tl >> 1) & 1u) ^ 1u, p.err, 4, &abort_s)) break;
            tc_fence_after();
            const uint32_t d = tmem + uint32_t(a * kNacc * kN);
            for (int c = 0; c < nK; ++c) {
                if (!mbar_wait(ffull(fs), fph, p.err, 16, &abort_s)) { ok = false; break; }
                if (!mbar_wait(sfull(s), sph, p.err, 8, &abort_s)) { ok = false; break; }
                tc_fence_after();
                const uint64_t S = sdesc64(sbase + s * kSBytes), F = sdesc64(fbase + fs * kFBytes);
#pragma unroll
                for (int kk = 0; kk < kKc / 16; ++kk)
                    mma_kstep(d, F + (uint64_t(kk * 32) >> 4), S + (uint64_t(kk * 32) >> 4), (c == 0 && kk == 0) ? 1u : 0u);
                tc_commit(sempty(s));
                tc_commit(fempty(fs));
                if (++s == kNS) { s = 0; sph ^= 1; }
                if (++fs == kNF) { fs = 0; fph ^= 1; }
            }
            if (ok) tc_commit(accf(a));
        }
        // wait for every MMA this thread issued before TMEM is released
        tc_commit(drain_bar);
        const long long t0 = clock64();
        while (!mbar_try_wait(drain_bar, 0) && clock64() - t0 < kWaitCycles) {}
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

int g_sms = 0;

template <bool MODE1, int EPI>
cudaError_t launch_variant(const BatchTcArgs& a, unsigned grid, cudaStream_t s) {
    static SmemLimit smem;
    const cudaError_t e = smem.allow(reinterpret_cast<const void*>(batch_tc_kernel<MODE1, EPI>), kSmem);
    if (e != cudaSuccess) return e;
    batch_tc_kernel<MODE1, EPI><<<grid, kThreads, kSmem, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ small kernels
__global__ void keep_lo_kernel(const float* __restrict__ u, const float* __restrict__ hs, float* __restrict__ lo,
                               long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        if (u[i] != hs[i]) lo[i] = 0.f;
}

// One warp per row of one instance (rows located through the row prefix), lanes along x1.
__global__ void __launch_bounds__(256) batch_amax_kernel(BatchStencilArgs<float> g, const float* __restrict__ x,
                                                         unsigned* amax) {
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < g.rows; r += warps) {
        int lo = 0, hi = g.ninst - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(g.row_start + mid) <= r) lo = mid; else hi = mid - 1;
        }
        const BatchInst<float>& in = g.inst[lo];
        const float* row = x + in.off + (r - in.row0) * in.n1;
        float m = 0.f;
        for (int i1 = lane; i1 < in.n1; i1 += 32) m = fmaxf(m, fabsf(__ldg(row + i1)));
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0 && m > 0.f) atomicMax(amax + lo, __float_as_uint(m));
    }
}

}  // namespace

cudaError_t launch_batch_tc(BatchTcArgs a, cudaStream_t s) {
    if (a.nitems <= 0) return cudaSuccess;
    if (!a.inst || !a.items || !a.fimg || !a.fscale || !a.X || !a.Y || !a.amax_in || (a.mode != 1 && a.mode != 2))
        return cudaErrorInvalidValue;
    if (a.role < 0 || a.role >= kBatchRoles) return cudaErrorInvalidValue;
    if (a.epi == EPI_PHI && (!a.phi || a.mode != 2)) return cudaErrorInvalidValue;
    if (a.epi == EPI_AXPY && !a.base) return cudaErrorInvalidValue;
    if (a.epi != EPI_STORE && a.epi != EPI_PHI && a.epi != EPI_AXPY) return cudaErrorInvalidValue;
    // the mode-1 producers read 16-byte vectors where an instance's rows allow it
    if (reinterpret_cast<uintptr_t>(a.X) % 16 != 0 || (a.Xlo && reinterpret_cast<uintptr_t>(a.Xlo) % 16 != 0))
        return cudaErrorMisalignedAddress;
    if (g_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    long long grid = a.grid > 0 ? a.grid : g_sms;
    if (grid > a.nitems) grid = a.nitems;
    const unsigned g = unsigned(grid);
    a.al16 = true;
    for (const void* q : {(const void*)a.Y, (const void*)a.Ylo, (const void*)a.Yhs, (const void*)a.base, (const void*)a.base_lo,
                          (const void*)a.phi})
        a.al16 = a.al16 && reinterpret_cast<uintptr_t>(q) % 16 == 0;
    if (a.mode == 2) {
        if (a.epi == EPI_PHI) return launch_variant<false, EPI_PHI>(a, g, s);
        if (a.epi == EPI_AXPY) return launch_variant<false, EPI_AXPY>(a, g, s);
        return launch_variant<false, EPI_STORE>(a, g, s);
    }
    if (a.epi == EPI_AXPY) return launch_variant<true, EPI_AXPY>(a, g, s);
    if (a.epi == EPI_PHI) return cudaErrorInvalidValue;
    return launch_variant<true, EPI_STORE>(a, g, s);
}

cudaError_t launch_batch_keep_lo(const float* u, const float* hs, float* lo, long long n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (!u || !hs || !lo) return cudaErrorInvalidValue;
    long long blocks = (n + 255) / 256;
    if (blocks > 8192) blocks = 8192;
    keep_lo_kernel<<<unsigned(blocks), 256, 0, s>>>(u, hs, lo, n);
    return cudaGetLastError();
}

cudaError_t launch_batch_amax(const BatchStencilArgs<float>& geom, const float* x, unsigned* amax, cudaStream_t s) {
    if (geom.rows <= 0) return cudaSuccess;
    if (!geom.inst || !geom.row_start || !x || !amax) return cudaErrorInvalidValue;
    long long blocks = (geom.rows + 7) / 8;
    if (blocks > 8192) blocks = 8192;
    batch_amax_kernel<<<unsigned(blocks), 256, 0, s>>>(geom, x, amax);
    return cudaGetLastError();
}

}  // namespace adr
