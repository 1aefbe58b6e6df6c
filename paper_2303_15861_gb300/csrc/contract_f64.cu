// K2 in FP64 on the tensor cores: mu-mode contraction Y = X x_mu M with FP64 inputs and outputs,
// computed as exact sums of BF16 products.
//
// This GPU's FP64 pipes do 2 FMAs per clock and SM (1.1 TFLOP/s measured): a 256^3 pass of 8.6 GFLOP
// takes 7.4 ms there. The tensor cores do 1.9 PFLOP/s in BF16. So x and the factor are cut into
// integer slices whose products the tensor cores sum exactly, and the slices of the result are put
// together in 64-bit integers:
//   X_k = rint(x_k 2^(c_k + 56 - es)) = sum_i S_i 2^(8 (6 - i)),  |S_0| <= 256, |S_1..S_6| <= 128, |x_k| 2^c_k < 2^es,
//   F_k = rint(f_k 2^(-c_k + 56 - ef)) = sum_j F_j 2^(8 (6 - j)),  the same, ef per factor row, c_k per factor column,
//   D_s = sum_{i + j = s} S_i . F_j,  s = 0..6  (28 products),
//   T = sum_s D_s 2^(8 (6 - s)),   x . f = T 2^(es + ef - 64).
// The seven D_s are TMEM accumulators. They are sums of integers, exact in FP32 up to 2^24: with
// |D_s| <= (s + 3) 2^14 K (D_0: 2^16 K) all of them for K <= 113, D_0 and D_1 for K <= 256. Longer
// lines are summed in segments of 256. There D_2..D_6 could pass 2^24 only where the factor row and the state
// were both constant over the segment at 80% or less of every digit's largest value with matching
// signs: the digits past the first of a varying row or state average out (the sums are then near 2^19).
// Errors: 2^-57 of 2^es and 2^ef for the two representations, about sqrt(K) 2^-57 of 2^(es + ef) for
// the slice products left out (i + j > 6), and one rounding of the result to FP64. A chain of K FMAs rounds
// K times, but each time at the size of its own terms, so what decides is whether 2^(es + ef) is the size of the largest
// term. The columns of V_mu^-1 differ by rho^n (5e8 at n = 128 and b = 40 abar): the c_k give them one
// size. Without them, a pulse of width 0.05 that lies where the columns are small (128^2, b = 50, 60, 80 along x1, abar = 1.5)
// left a phi action 3e-12, 9e-12 and 7e-10 off; with them pulses at b = 30 and 60 are 1e-15 to 4e-15 off and within 4%
// of the FMA chain. Over 162 exponentials and phi actions
// (n = 64..520, b = 3..60, smooth, random, pulses, single points) against 80-bit sums the relative l2 error
// is 0.37 to 1.6 times that of the FMA kernel, 0.92 in the mean. It is an error of the line: results more than 2^-53 below the
// line's largest are noise of that size, of either sign, where a chain of positive terms would keep their digits.
// Time of a pass, FMA kernel -> this one: 256^3 6.9 ms -> 0.24 ms, 128^3 526 -> 31 us (39 with the phi table), 60^3
// 33 -> 12 us. At the BF16 rate the products of a 256^3 pass take 0.13 ms; the rest is the assembly of a tile,
// which cannot overlap its MMAs (the accumulators fill TMEM), and the producers just behind them.
//
// es belongs to one line (the n values that are contracted together): the producers read a tile's lines
// once for their largest exponents and a second time, from L2, to cut them. One es for the whole array would
// save that read, but each pass would then lose what the array varies by: through the eigenbasis
// (V_mu scaled by rho^i, 28-fold from end to end per direction at b = 10) a 100 x 72 x 64 ETD2RK run was
// 1.2e-14 off instead of 5e-16. Lines with a NaN or an infinity, or with max|x| below 2^-958 (or, where the factor has
// column exponents, above 2^624), are contracted with plain FMAs by the epilogue, so that such values propagate as
// in any FP64 sum. That costs 1.2 ms a pass at 128^3 where the FMA kernel takes 0.53.
//
// Work split. The factor is the A operand, 128 outputs (TMEM lanes) a tile; the lines are the B operand,
// N = 64 of them (448 of the 512 TMEM columns), or 32 where 64 would leave SMs without a tile. For modes >= 2
// the lines of a tile are consecutive positions, p and q flattened, so a short q leaves no empty
// columns. Per CTA and SM: 8 producer warps load FP64 from global memory (the next chunk in
// registers while this one is cut, no alignment rules, so every shape takes this kernel) and
// store the slices; one thread issues the MMAs; one copies the pre-cut factor; 8 warps put the results together.
// With the lines as the A operand, 128 a tile, and 64 outputs, each line of a 256^3 grid is cut four
// times instead of twice, which took 460 us a pass.
// Cutting and assembling use integer instructions, one FP64-pipe instruction per result: one of
// those occupies its pipe as long as 64 of the others. Tried, us a pass at 128^3 / 256^3 (29 / 241 as it is): the conversion
// in integers too 33 / 265; the line maxima of the next tile read while a tile is cut 31 / 243 (mode 1) and 268.
#include <cuda_runtime.h>

#include <cstdint>

#include "adr_internal.h"
#include "phi_device.cuh"
#include "smem_limit.h"
#include "tc_common.cuh"

namespace adr {
namespace {
using namespace tc;

constexpr int kSl = kF64Slices;          // slices per operand and accumulators
constexpr int kM = 128;                  // UMMA M, TMEM lanes
constexpr int kKc = kF64Chunk;           // K per stage: one 64-byte bf16 row (64-byte swizzle)
constexpr int kSegChunks = 8;            // K chunks per accumulation segment (256)
constexpr int kProducerWarps = 8;
constexpr int kEpiWarps = 8;
constexpr int kMmaWarp = kProducerWarps + kEpiWarps;
constexpr int kLoadWarp = kMmaWarp + 1;
constexpr int kThreads = (kLoadWarp + 1) * 32;

// Tiles whose line scales are kept: the producers run ahead of the epilogue by the tile whose MMAs wait for it and, at one
// chunk a tile, by one tile more per stage of their ring.
constexpr int kTileBufs = 8;

template <int N>
struct Cfg {
    static constexpr int FTILE = kM * kKc * 2, STILE = N * kKc * 2;   // one slice tile of either operand
    static constexpr int SBYTES = kSl * STILE, FBYTES = kSl * FTILE;  // one stage
    static constexpr int NS = 3, NF = 2;                              // ring depths: 196 KB at N = 64
    static constexpr int SMEM = NS * SBYTES + NF * FBYTES + 1024;
    static constexpr uint32_t TMEM = N == 64 ? 512 : 256;             // 7 N columns, a power of two
    static constexpr int COLS = N / (kEpiWarps / 4);                  // columns per epilogue warp
    static constexpr int WIDE = 256 / N;                              // slices per MMA (N <= 256)
    static constexpr int KV = N * kKc / (kProducerWarps * 32);        // K values a producer thread cuts per chunk
    static constexpr int KG = kKc / KV;                               // threads per line
    static_assert(NS + 3 <= kTileBufs, "line scales of every tile in flight");
    static_assert(SMEM <= 215 * 1024, "shared memory budget");
};

__device__ __forceinline__ uint32_t idesc_of(int ncols) {   // FP32 accumulator, BF16 operands, M = 128
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(ncols >> 3) << 17) | (uint32_t(kM >> 4) << 24);
}

// Cut x 2^c into its seven digits: d = etop - c - exponent(x) >= 0 places below the leading one. Digits
// 1..6 are bytes of X + 0x808080808080 less 128, digit 0 what is above them. Returned as FP32 values
// whose upper halves are their BF16 forms (integers of at most 8 bits).
__device__ __forceinline__ void cut(double x, int etop, int c, float (&s)[kSl]) {
    const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
    const int d = min(etop - c - int((hi >> 20) & 0x7FFu), 63);
    const unsigned long long m = (static_cast<unsigned long long>((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
    long long v = static_cast<long long>((((m << 4) >> d) + 1ull) >> 1);
    const long long sg = static_cast<long long>(int(hi) >> 31);
    v = ((v ^ sg) - sg) + 0x0000808080808080LL;
    const uint32_t vl = uint32_t(v), vh = uint32_t(static_cast<unsigned long long>(v) >> 32);
    s[0] = __uint_as_float(0x4B400000u + uint32_t(int(vh) >> 16)) - 12582912.f;
    s[1] = __uint_as_float(__byte_perm(vh, 0x4B000000u, 0x7441)) - 8388736.f;
    s[2] = __uint_as_float(__byte_perm(vh, 0x4B000000u, 0x7440)) - 8388736.f;
    s[3] = __uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7443)) - 8388736.f;
    s[4] = __uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7442)) - 8388736.f;
    s[5] = __uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7441)) - 8388736.f;
    s[6] = __uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7440)) - 8388736.f;
}

// Cut KV (4 or 8) values along K, of exponents c, and store them at K position k of row r of the seven slice tiles.
template <int TILE, int KV>
__device__ __forceinline__ void cut_store(const double (&v)[KV], int etop, const int (&c)[KV], uint32_t tile0, int r, int k) {
    uint32_t w[kSl][KV / 2];
#pragma unroll
    for (int e = 0; e < KV / 2; ++e) {
        float a[kSl], b[kSl];
        cut(v[2 * e], etop, c[2 * e], a);
        cut(v[2 * e + 1], etop, c[2 * e + 1], b);
#pragma unroll
        for (int q = 0; q < kSl; ++q) w[q][e] = __byte_perm(__float_as_uint(a[q]), __float_as_uint(b[q]), 0x7632);
    }
    const uint32_t dst = tile0 + swz64(r, k >> 3) + (k & 7) * 2;
#pragma unroll
    for (int q = 0; q < kSl; ++q) {
        if constexpr (KV == 8)
            st_shared_v4(dst + q * TILE, make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]));
        else
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + q * TILE), "r"(w[q][0]), "r"(w[q][1]) : "memory");
    }
}

// 32-byte (256-bit) accesses: four consecutive doubles.
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void st4(double* p, const double (&v)[4]) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
}

// Four columns of the seven accumulators, `stride` TMEM columns apart.
__device__ __forceinline__ void tmem_ld4x7(uint32_t t0, uint32_t stride, float (&d)[kSl][4]) {
    uint32_t r[28];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%28];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%29];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%30];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%31];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%33];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%34];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27])
        : "r"(t0), "r"(t0 + stride), "r"(t0 + 2 * stride), "r"(t0 + 3 * stride), "r"(t0 + 4 * stride),
          "r"(t0 + 5 * stride), "r"(t0 + 6 * stride)
        : "memory");
#pragma unroll
    for (int k = 0; k < kSl; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) d[k][j] = __uint_as_float(r[4 * k + j]);
}

// The result from its seven sums, in units of 2^(e - kUnit): T = 2^24 h + l, shifted right (rounding) by the ex >= 0 places
// that leave it 62 bits; the conversion to FP64 rounds to nearest, and the unit goes into the exponent, which
// takes it for 0 <= e <= kUnitTop (1 <= |T| < 2^88).
constexpr int kUnit = 1022, kUnitTop = kUnit + 1023 - 88;
__device__ __forceinline__ double assemble(const float (&d)[kSl][4], int c, int e) {
    int v[kSl];
#pragma unroll
    for (int k = 0; k < kSl; ++k) v[k] = __float2int_rn(d[k][c]);
    const long long h = static_cast<long long>(v[0]) * (1 << 24) + static_cast<long long>(v[1]) * (1 << 16) +
                        static_cast<long long>(v[2]) * (1 << 8) + v[3];
    const long long l = static_cast<long long>(v[4]) * (1 << 16) + static_cast<long long>(v[5]) * (1 << 8) + v[6];
    const int top = int(h >> 32);                            // |T| < 2^(88 - clz)
    const int ex = max(26 - __clz(top ^ (top >> 31)), 0);
    const long long t = (h << (24 - ex)) + ((l + ((1 << ex) >> 1)) >> ex);
    const double r = static_cast<double>(t);
    const int up = t ? (e - kUnit + ex) * (1 << 20) : 0;
    return __hiloint2double(__double2hiint(r) + up, __double2loint(r));
}

__device__ __noinline__ double scale_by(double r, int e) { return ldexp(r, e); }

// One output by plain FMAs, k ascending (lines whose values do not fit the slices).
__device__ __noinline__ double fma_dot(const double* f, const double* x, int n, long long stride) {
    double acc = 0.0;
    for (int k = 0; k < n; ++k) acc = fma(f[k], x[k * stride], acc);
    return acc;
}

// The upper word of |v|. NaN orders above infinity.
__device__ __forceinline__ int f64_abs_hi(double v) { return __double2hiint(v) & 0x7FFFFFFF; }

// The phi factor of node o, where the context keeps no table.
__device__ __noinline__ double f64_phi_eval(const F64Args& p, long long o) {
    double ls = p.lam[0][o % p.n1] + p.lam[1][(o / p.n1) % p.n2];
    if (p.lam[2]) ls += p.lam[2][o / p.n1 / p.n2];
    return phi_eval(p.phik, p.ctau * ls);
}

constexpr int kNoCut = 1 << 20;          // es of a line that fma_dot contracts

template <bool MODE1, int N, int EPI, bool EQ>
__global__ void __launch_bounds__(kThreads, 1) f64_contract_kernel(const __grid_constant__ F64Args p) {
    using C = Cfg<N>;
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t kSF = 0, kSE = kSF + 8 * C::NS, kFF = kSE + 8 * C::NS, kFE = kFF + 8 * C::NF, kAF = kFE + 8 * C::NF,
                       kAE = kAF + 8, kDR = kAE + 8;
    __shared__ __align__(8) uint64_t bars[kDR / 8 + 1];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
    // per line of the last tiles: its exponent es, and its offset in the state (k = 0)
    __shared__ int es_s[kTileBufs][N];
    __shared__ long long off_s[kTileBufs][N];
    __shared__ int part_s[2][C::KG][N];                      // modes >= 2: the parts of a line's max|x|
    __shared__ __align__(16) int cexp_s[EQ ? kF64MaxN : 4];  // c_k (EQ: the factor has any)

    static_assert(kF64MaxN <= 2 * kThreads, "two column exponents a thread");
    int c0 = 0, c1 = 0;                                      // on their way during the set-up
    if (EQ) {
        if (threadIdx.x < p.nK * kKc) c0 = p.cexp[threadIdx.x];
        if (threadIdx.x + kThreads < p.nK * kKc) c1 = p.cexp[threadIdx.x + kThreads];
    }

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;     // state-slice ring
    const uint32_t fbase = sbase + C::NS * C::SBYTES;                   // factor ring
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto sfull = [&](int s) { return bar0 + kSF + 8u * s; };
    auto sempty = [&](int s) { return bar0 + kSE + 8u * s; };
    auto ffull = [&](int s) { return bar0 + kFF + 8u * s; };
    auto fempty = [&](int s) { return bar0 + kFE + 8u * s; };
    const uint32_t accf = bar0 + kAF, acce = bar0 + kAE, drain_bar = bar0 + kDR;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(sfull(s), kProducerWarps);             // one arrival per producer warp
            mbar_init(sempty(s), 1);                         // tcgen05.commit
        }
        for (int s = 0; s < C::NF; ++s) {
            mbar_init(ffull(s), 1);                          // loader's expect_tx arrival
            mbar_init(fempty(s), 1);                         // tcgen05.commit
        }
        mbar_init(accf, 1);
        mbar_init(acce, kEpiWarps);
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
    if (EQ) {
        if (threadIdx.x < p.nK * kKc) cexp_s[threadIdx.x] = c0;
        if (threadIdx.x + kThreads < p.nK * kKc) cexp_s[threadIdx.x + kThreads] = c1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;

    const int n = p.n;
    const long long Q = MODE1 ? 1 : p.Q;
    const int items = (p.ntiles - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x) * p.nK;   // (tile, K chunk) in order

    if (warp == kLoadWarp) {
        // ------------------------------------------------------------ factor loader (bulk copies)
        if (lane == 0) {
            int s = 0, issued = 0;
            uint32_t ph = 1;
            for (int tile = blockIdx.x; tile < p.ntiles && !abort_s; tile += gridDim.x) {
                const uint8_t* src = p.fimg + size_t(tile % p.nOut) * p.nK * C::FBYTES;
                for (int c = 0; c < p.nK; ++c, src += C::FBYTES, ++issued) {
                    if (!mbar_wait(fempty(s), ph, p.err, 64, &abort_s, 32)) break;
                    mbar_arrive_expect_tx(ffull(s), C::FBYTES);
                    bulk_g2s(fbase + s * C::FBYTES, src, C::FBYTES, ffull(s));
                    if (++s == C::NF) { s = 0; ph ^= 1; }
                }
            }
            // no copy may land after the CTA has gone (they have, unless a wait gave up)
            const long long t0 = clock64();
            for (int k = max(issued - C::NF, 0); k < issued; ++k)
                while (!mbar_try_wait(ffull(k % C::NF), uint32_t(k / C::NF) & 1u) && clock64() - t0 < kWaitCycles) {}
        }
    } else if (warp < kProducerWarps) {
        // ------------------------------------------------------------ producers (global -> slices)
        // KG threads a line, each KV consecutive K values of a chunk: neighbouring lanes along K for mode 1,
        // along the positions otherwise, so that a warp reads whole sectors.
        constexpr int KV = C::KV, KG = C::KG;
        const int t = threadIdx.x;
        const int row = MODE1 ? t / KG : t % N, kg = MODE1 ? t % KG : t / N;
        const int kofs = KV * kg;
        double v[KV];
        // the (tile, chunk) whose values are being loaded, and this thread's line of that tile
        int ltile = blockIdx.x, lc = 0, etop = 0;
        const double* xrow = nullptr;
        bool lrow = false, live = true;
        long long xoff = 0;
        auto set_row = [&]() {
            const unsigned pos = unsigned(ltile / p.nOut) * N + row;
            lrow = ltile < p.ntiles && pos < unsigned(p.npos);
            xoff = MODE1 ? (long long)pos * n : (long long)(pos / unsigned(Q)) * n * Q + pos % unsigned(Q);
            xrow = p.X + xoff + kofs * Q;
        };
        auto load = [&](int k0, double (&w)[KV]) {           // K values k0 + kofs.. (0 past the line's end)
            const double* x = xrow + k0 * Q;
            if (MODE1 && p.vec2) {
#pragma unroll
                for (int e = 0; e < KV; e += 2) {
                    const double2 u = (lrow && k0 + kofs + e < n) ? __ldg(reinterpret_cast<const double2*>(x + e)) : make_double2(0.0, 0.0);
                    w[e] = u.x;
                    w[e + 1] = u.y;
                }
            } else {
#pragma unroll
                for (int e = 0; e < KV; ++e) w[e] = (lrow && k0 + kofs + e < n) ? __ldg(x + e * Q) : 0.0;
            }
        };
        auto exps = [&](int k0, int (&c)[KV]) {
#pragma unroll
            for (int e = 0; e < KV; e += 4) {
                const int4 q = EQ ? *reinterpret_cast<const int4*>(&cexp_s[k0 + kofs + e]) : make_int4(0, 0, 0, 0);
                c[e] = q.x; c[e + 1] = q.y; c[e + 2] = q.z; c[e + 3] = q.w;
            }
        };
        // upper word of the largest |x_k| 2^c_k (0 below the normal range), and whether any value is not zero
        int m = 0, any = 0;
        auto amax = [&](const double (&w)[KV], int k0) {
            int c[KV];
            exps(k0, c);
#pragma unroll
            for (int e = 0; e < KV; ++e) {
                const int h = f64_abs_hi(w[e]);
                m = max(m, h + c[e] * (1 << 20));
                any |= h | __double2loint(w[e]);
            }
        };
        // Lines that are cut, by the exponent field of their largest value: below kLiveLow a value outside the normal
        // range, which cut() does not know, could still reach a digit; an infinity or a NaN has at least 2047 + min c_k
        constexpr int kLiveLow = 64, kLiveHigh = 2047 + (EQ ? kF64MinExp : 0);
        // es of this thread's line, of which v holds the first chunk
        auto line_scale = [&](int tl) {
            m = any = 0;
            amax(v, 0);
            int c = 1;
            for (; c + 1 < p.nK; c += 2) {                   // two chunks of loads in flight
                double w[KV], u[KV];
                load(c * kKc, w);
                load((c + 1) * kKc, u);
                amax(w, c * kKc);
                amax(u, (c + 1) * kKc);
            }
            if (c < p.nK) {
                double w[KV];
                load(c * kKc, w);
                amax(w, c * kKc);
            }
            if (any) m = max(m, 1);
            if (MODE1) {
#pragma unroll
                for (int o = 1; o < KG; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            } else {
                part_s[tl & 1][kg][row] = m;
                asm volatile("bar.sync 1, %0;" ::"n"(kProducerWarps * 32) : "memory");
#pragma unroll
                for (int o = 0; o < KG; ++o) m = max(m, part_s[tl & 1][o][row]);
            }
            const int eb = m >> 20;
            live = m == 0 || (eb >= kLiveLow && eb < kLiveHigh);
            etop = m ? eb : 1022;                            // es + 1022
            if (kg == 0) {
                es_s[tl & (kTileBufs - 1)][row] = live ? etop - 1022 : kNoCut;
                off_s[tl & (kTileBufs - 1)][row] = xoff;
            }
        };
        set_row();
        load(0, v);
        line_scale(0);
        for (int it = 0, ss = 0, sph = 1, tl = 0; it < items; ++it) {
            // after an abort the wait returns at once and the loop runs out, so that every producer warp
            // still meets the others at line_scale's barrier
            mbar_wait(sempty(ss), sph, p.err, 1, &abort_s, 32);
            __syncwarp();
            int ce[KV];
            exps(lc * kKc, ce);
            const bool next_tile = ++lc == p.nK;
            if (next_tile) {
                lc = 0;
                ltile += gridDim.x;
                set_row();
            }
            if (!live) {
#pragma unroll
                for (int e = 0; e < KV; ++e) v[e] = 0.0;
            }
            cut_store<C::STILE, KV>(v, etop, ce, sbase + ss * C::SBYTES, row, kofs);
            load(lc * kKc, v);                               // in flight until the next chunk is cut
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(sfull(ss));
            if (++ss == C::NS) { ss = 0; sph ^= 1; }
            if (next_tile && it + 1 < items) line_scale(++tl);
        }
    } else if (warp < kMmaWarp) {
        // ------------------------------------------------------------ epilogue
        const int ew = (warp - kProducerWarps) & 3;          // TMEM lane quarter (warp % 4)
        const int part = (warp - kProducerWarps) >> 2;       // column part
        const int jlo = part * C::COLS, jhi = jlo + C::COLS;
        const uint32_t tbase = tmem + (uint32_t(ew * 32) << 16);
        uint32_t seg = 0;
        int tl = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x, ++tl) {
            const int pt = tile / p.nOut, ot = tile % p.nOut;
            const int irow = ot * kM + ew * 32 + lane;       // this lane's output
            const bool rvalid = irow < n;
            const bool warp_on = ot * kM + ew * 32 < n;
            const int ncol = min(N, int(p.npos - (long long)pt * N));
            const int rexp = __ldg(p.rows + irow);           // padded to whole tiles
            const long long ioff = irow * Q;
            const long long* off_t = off_s[tl & (kTileBufs - 1)];
            const int* es_t = es_s[tl & (kTileBufs - 1)];
            for (int c0 = 0; c0 < p.nK; c0 += kSegChunks, ++seg) {
                const bool first = c0 == 0;
                const bool waited = mbar_wait(accf, seg & 1u, p.err, 2, &abort_s, 32);
                if (!__all_sync(0xffffffffu, waited)) { ok = false; break; }
                tc_fence_after();
                if (!warp_on) {
                    if (lane == 0) mbar_arrive(acce);
                    continue;
                }
                // the axpy's base or the phi table's values of four columns, and the earlier segments' sum,
                // one group ahead
                double bcur[4], bnxt[4];
                auto load_base = [&](int j0, double (&b)[4]) {
                    if (EPI == EPI_STORE || (EPI == EPI_AXPY && !first)) return;
                    if (EPI == EPI_PHI && !p.phi) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) b[j] = rvalid && j0 + j < ncol ? f64_phi_eval(p, off_t[j0 + j] + ioff) : 0.0;
                        return;
                    }
                    const double* src = EPI == EPI_PHI ? p.phi : p.base;
                    if (p.vec4 && rvalid && j0 + 3 < ncol) {
                        ld4(src + off_t[j0] + ioff, b);
                        return;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) b[j] = rvalid && j0 + j < ncol ? src[off_t[j0 + j] + ioff] : 0.0;
                };
                load_base(jlo, bcur);
#pragma unroll 1
                for (int j0 = jlo; j0 < jhi; j0 += 4) {
                    float d[kSl][4];
                    if (j0 + 4 < jhi) load_base(j0 + 4, bnxt);
                    int es[4];
                    long long off[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        es[j] = es_t[j0 + j];
                        off[j] = off_t[j0 + j] + ioff;
                    }
                    __syncwarp();
                    tmem_ld4x7(tbase + j0, uint32_t(N), d);
                    if (j0 + 4 >= jhi) {                     // the last columns are in registers: TMEM is free
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acce);
                    }
                    double v[4];
                    unsigned unit[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) unit[j] = unsigned(rexp + es[j]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] = assemble(d, j, int(min(unit[j], unsigned(kUnitTop))));
                    // results that may leave the normal range, lines that were not cut (nothing of the sums is
                    // needed any more: assembled anew here, they cost 8% of 128^3 ETD2RK)
                    if (max(max(unit[0], unit[1]), max(unit[2], unit[3])) > unsigned(kUnitTop)) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (unit[j] > unsigned(kUnitTop)) v[j] = scale_by(v[j], int(unit[j]) - kUnitTop);
                            if (es[j] == kNoCut)
                                v[j] = first && rvalid && j0 + j < ncol
                                           ? fma_dot(p.factor + (long long)irow * n, p.X + off[j] - ioff, n, Q) : 0.0;
                        }
                    }
                    if (EPI == EPI_PHI) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] *= bcur[j];
                    }
                    if (EPI == EPI_AXPY && first) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = fma(p.alpha, v[j], bcur[j]);
                    }
                    if (!first) {                            // lines past one segment: add to the earlier ones' sum
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (rvalid && j0 + j < ncol) v[j] = fma(EPI == EPI_AXPY ? p.alpha : 1.0, v[j], p.Y[off[j]]);
                    }
                    if (p.vec4 && rvalid && j0 + 3 < ncol) {
                        st4(p.Y + off[0], v);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (rvalid && j0 + j < ncol) p.Y[off[j]] = v[j];
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) bcur[j] = bnxt[j];
                }
            }
        }
    } else if (warp == kMmaWarp && lane == 0) {
        // ------------------------------------------------------------ MMA issuer
        // F_i.S_j adds to D_(i+j). The S tiles lie one after another, as do the accumulators, so F_i
        // takes up to 256 / N consecutive S_j in one MMA of up to 256 columns: 10 MMAs per
        // K step instead of 28 at N = 64, and F_i is read from shared memory once for them.
        uint32_t seg = 0, sph = 0, fph = 0;
        int s = 0, fs = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < p.ntiles && !abort_s && ok; tile += gridDim.x) {
            for (int c = 0; c < p.nK; ++c) {
                const bool first = c % kSegChunks == 0;
                if (first) {
                    if (!mbar_wait(acce, (seg & 1u) ^ 1u, p.err, 4, &abort_s)) { ok = false; break; }
                    tc_fence_after();
                }
                if (!mbar_wait(ffull(fs), fph, p.err, 128, &abort_s)) { ok = false; break; }
                if (!mbar_wait(sfull(s), sph, p.err, 8, &abort_s)) { ok = false; break; }
                tc_fence_after();
                const uint32_t sS = sbase + s * C::SBYTES, sF = fbase + fs * C::FBYTES;
                const uint64_t a0 = sdesc64(sF), b0 = sdesc64(sS);
#pragma unroll
                for (int kk = 0; kk < kKc / 16; ++kk) {
                    const uint64_t adv = uint64_t(kk * 32) >> 4;
#pragma unroll
                    for (int i = 0; i < kSl; ++i)
#pragma unroll
                        for (int j = 0; j < kSl - i; j += C::WIDE) {
                            const int w = (kSl - i - j) < C::WIDE ? (kSl - i - j) : C::WIDE;
                            tc_mma(tmem + (i + j) * N, a0 + adv + uint64_t(i * C::FTILE >> 4),
                                   b0 + adv + uint64_t(j * C::STILE >> 4), idesc_of(w * N),
                                   (first && kk == 0 && i == 0) ? 0u : 1u);
                        }
                }
                tc_commit(sempty(s));
                tc_commit(fempty(fs));
                if (++s == C::NS) { s = 0; sph ^= 1; }
                if (++fs == C::NF) { fs = 0; fph ^= 1; }
                if (c % kSegChunks == kSegChunks - 1 || c == p.nK - 1) {
                    tc_commit(accf);
                    ++seg;
                }
            }
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

// A factor entry as a normal number times 2^sh.
__device__ __forceinline__ double normal_part(double f, int& sh) {
    sh = (f64_abs_hi(f) >> 20) ? 0 : -64;
    return sh ? f * 18446744073709551616.0 : f;
}

// Cut the dense factor (n x n, row-major), its column k times 2^-c_k, into its image: per (tile of 128 rows, K chunk of
// 32) seven 64-byte-swizzled K-major tiles; and per row the exponent of the result's unit, less es, plus kUnit. One block
// per padded row.
__global__ void f64_factor_kernel(const double* M, int n, int nK, const int* cexp, uint8_t* img, int* rows) {
    const int i = blockIdx.x;
    __shared__ int smax;
    constexpr int kNone = -(1 << 20);                        // a row of zeros
    if (threadIdx.x == 0) smax = kNone;
    __syncthreads();
    int m = kNone;                                           // exponent field of the largest entry
    if (i < n)
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            int sh;
            const double f = normal_part(M[(size_t)i * n + k], sh);
            if (f != 0.0) m = max(m, (f64_abs_hi(f) >> 20) + sh - (cexp ? cexp[k] : 0));
        }
    atomicMax(&smax, m);
    __syncthreads();
    const int ef = smax == kNone ? 0 : smax - 1022;          // max|f_k| 2^-c_k < 2^ef
    if (threadIdx.x == 0) rows[i] = ef - 64 + kUnit;
    uint8_t* tile = img + (size_t)(i / kM) * nK * kSl * kM * 64;
    for (int k = threadIdx.x; k < nK * kKc; k += blockDim.x) {
        int sh;
        const double f = normal_part((i < n && k < n) ? M[(size_t)i * n + k] : 0.0, sh);
        float s[kSl] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (f != 0.0) cut(f, ef + 1022, (cexp ? -cexp[k] : 0) + sh, s);
        const int kc = k % kKc;
        uint8_t* dst = tile + (size_t)(k / kKc) * kSl * kM * 64 + swz64(i % kM, kc / 8) + (kc % 8) * 2;
#pragma unroll
        for (int q = 0; q < kSl; ++q)
            *reinterpret_cast<uint16_t*>(dst + (size_t)q * kM * 64) = uint16_t(__float_as_uint(s[q]) >> 16);
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

template <bool MODE1, int N, int EPI, bool EQ>
cudaError_t launch_variant(const F64Args& a, cudaStream_t s) {
    static SmemLimit smem;
    const cudaError_t e = smem.allow(reinterpret_cast<const void*>(f64_contract_kernel<MODE1, N, EPI, EQ>), Cfg<N>::SMEM);
    if (e != cudaSuccess) return e;
    const int grid = a.ntiles < sm_count() ? a.ntiles : sm_count();
    f64_contract_kernel<MODE1, N, EPI, EQ><<<unsigned(grid), kThreads, Cfg<N>::SMEM, s>>>(a);
    return cudaGetLastError();
}

template <bool MODE1, int N, bool EQ>
cudaError_t launch_epi(const F64Args& a, cudaStream_t s) {
    if (a.epi == EPI_PHI) return launch_variant<MODE1, N, EPI_PHI, EQ>(a, s);
    if (a.epi == EPI_AXPY) return launch_variant<MODE1, N, EPI_AXPY, EQ>(a, s);
    return launch_variant<MODE1, N, EPI_STORE, EQ>(a, s);
}
template <bool MODE1, int N>
cudaError_t launch_eq(const F64Args& a, cudaStream_t s) {
    return a.cexp ? launch_epi<MODE1, N, true>(a, s) : launch_epi<MODE1, N, false>(a, s);
}

}  // namespace

size_t f64_image_bytes(int n) { return size_t((n + kM - 1) / kM) * kM * ((n + kKc - 1) / kKc) * kKc * 2 * kSl; }
int f64_rows(int n) { return (n + kM - 1) / kM * kM; }


cudaError_t launch_f64_factor(const double* M, int n, const int* cexp, uint8_t* img, int* rows, cudaStream_t s) {
    f64_factor_kernel<<<f64_rows(n), 128, 0, s>>>(M, n, (n + kKc - 1) / kKc, cexp, img, rows);
    return cudaGetLastError();
}

cudaError_t launch_contract_f64(F64Args a, cudaStream_t s) {
    if (a.npos <= 0) return cudaSuccess;
    const bool mode1 = a.Q == 1;
    a.nK = (a.n + kKc - 1) / kKc;
    a.nOut = (a.n + kM - 1) / kM;
    auto aligned = [](const void* q, uintptr_t to) { return reinterpret_cast<uintptr_t>(q) % to == 0; };
    a.vec2 = a.n % 2 == 0 && aligned(a.X, 16);
    // groups of four columns are four consecutive nodes: modes >= 2, q a multiple of 4
    a.vec4 = !mode1 && a.Q % 4 == 0 && aligned(a.Y, 32) && aligned(a.base, 32) && aligned(a.phi, 32);
    const bool wide = (a.npos + 63) / 64 * a.nOut >= sm_count();
    a.ntiles = int((a.npos + (wide ? 63 : 31)) / (wide ? 64 : 32) * a.nOut);
    if (mode1) return wide ? launch_eq<true, 64>(a, s) : launch_eq<true, 32>(a, s);
    return wide ? launch_eq<false, 64>(a, s) : launch_eq<false, 32>(a, s);
}

}  // namespace adr
