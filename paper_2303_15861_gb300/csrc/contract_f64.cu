// K2 in FP64 on the tensor cores: mu-mode contraction Y = X x_mu M with FP64 inputs and outputs,
// computed as exact sums of BF16 products.
//
// This GPU's FP64 pipes do 2 FMAs per clock and SM (1.1 TFLOP/s measured): a 256^3 pass of 8.6 GFLOP
// takes 7.4 ms there. The tensor cores do 1.9 PFLOP/s in BF16. So x and the factor are cut into
// integer slices whose products the tensor cores sum exactly, and the slices of the result are put
// together in 64-bit integers:
//   X = rint(x 2^(56 - es)) = sum_i S_i 2^(8 (6 - i)),  |S_0| <= 256, |S_1..S_6| <= 128, |x| < 2^es,
//   F = rint(f 2^(56 - ef)) = sum_j F_j 2^(8 (6 - j)),  the same, ef per factor row,
//   D_s = sum_{i + j = s} S_i . F_j,  s = 0..6  (28 products),
//   T = sum_s D_s 2^(8 (6 - s)),   x . f = T 2^(es + ef - 64).
// The seven D_s are TMEM accumulators. They are sums of integers, exact in FP32 up to 2^24: with
// |D_s| <= (s + 3) 2^14 K (D_0: 2^16 K) all of them for K <= 113, D_0 and D_1 for K <= 256. Longer
// lines are summed in segments of 256. There D_2..D_6 could pass 2^24 only where the factor row and the state
// were both constant over the segment at 80% or less of every digit's largest value with matching
// signs: the digits past the first of a varying row or state average out (the sums are then near 2^19).
// Errors: 2^-57 of 2^es and 2^ef for the two representations, about sqrt(K) 2^-57 of 2^(es + ef) for
// the slice products left out (i + j > 6), and one rounding of the result to FP64. A chain of K FMAs rounds
// K times. Against exact sums, e^{c tau A}, V and V^-1 for n = 24..300, b = 1..50, smooth and random
// states: relative l2 4e-17 to 1.6e-16, where the FMA kernel has 9e-17 to 6.3e-16, and the smaller of the two in every case.
// Time of a pass, FMA kernel -> this one: 256^3 6.9 ms -> 0.33 (mode 1) and 0.47 ms, 128^3 526 -> 42 to 62 us,
// 60^3 33 -> 15 to 18 us.
//
// es belongs to one line (the n values that are contracted together): the producers read a tile's lines
// once for their largest exponents and a second time, from L2, to cut them. One es for the whole array would
// save that read, but each pass would then lose what the array varies by: through the eigenbasis
// (V_mu scaled by rho^i, 28-fold from end to end per direction at b = 10) a 100 x 72 x 64 ETD2RK run was
// 1.2e-14 off instead of 5e-16. Lines with a NaN or an infinity, or with max|x| outside
// 2^-500..2^500, are contracted with plain FMAs by the epilogue, so that such values propagate as
// in any FP64 sum.
//
// Work split. 128 rows (TMEM lanes) lie along the contiguous direction: for modes >= 2 they are 128
// positions (q fastest, p and q flattened, so a short q leaves no empty rows) and the columns are outputs; for mode 1
// they are outputs and the columns are fibres. N = 64 columns (448 of the 512 TMEM columns), or 32 where 64 would leave
// SMs without a tile. Per CTA and SM: 8 producer warps load FP64 from global memory (the next chunk in
// registers while this one is cut, no alignment rules, so every shape takes this kernel) and
// store the slices; one thread issues the MMAs; one copies the pre-cut factor; 8 warps put the results together.
// Cutting and assembling use integer instructions throughout (about 40 each): one FP64 instruction
// occupies its pipe as long as 64 of the others.
#include <cuda_runtime.h>

#include <cstdint>

#include "adr_internal.h"
#include "phi_device.cuh"
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

template <bool SA, int N>
struct Cfg {
    static constexpr int ATILE = kM * kKc * 2, BTILE = N * kKc * 2;   // one slice tile of either operand
    static constexpr int STILE = SA ? ATILE : BTILE, FTILE = SA ? BTILE : ATILE;
    static constexpr int SBYTES = kSl * STILE, FBYTES = kSl * FTILE;  // one stage
    static constexpr int NS = SA ? 2 : 3, NF = SA ? 3 : 2;            // ring depths: 196 KB at N = 64
    static constexpr int SMEM = NS * SBYTES + NF * FBYTES + 1024;
    static constexpr uint32_t TMEM = N == 64 ? 512 : 256;             // 7 N columns, a power of two
    static constexpr int COLS = N / (kEpiWarps / 4);                  // columns per epilogue warp
    static constexpr int WIDE = 256 / N;                              // slices per MMA (N <= 256)
    static_assert(SMEM <= 227 * 1024, "shared memory budget");
};

__device__ __forceinline__ uint32_t idesc_of(int ncols) {   // FP32 accumulator, BF16 operands, M = 128
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(ncols >> 3) << 17) | (uint32_t(kM >> 4) << 24);
}

// Cut x into its seven digits: d = es + 1022 - exponent(x) >= 0 places below the leading one. Digits
// 1..6 are bytes of X + 0x808080808080 less 128, digit 0 what is above them. Returned as FP32 values
// whose upper halves are their BF16 forms (integers of at most 8 bits).
__device__ __forceinline__ void cut(double x, int etop, float (&s)[kSl]) {
    const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
    const int d = min(etop - int((hi >> 20) & 0x7FFu), 63);
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

// Cut 8 values along K and store them as 16-byte chunk j of row r of the seven slice tiles.
template <int TILE>
__device__ __forceinline__ void cut_store8(const double (&v)[8], int etop, uint32_t tile0, int r, int j) {
    uint32_t w[kSl][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        float a[kSl], b[kSl];
        cut(v[2 * e], etop, a);
        cut(v[2 * e + 1], etop, b);
#pragma unroll
        for (int q = 0; q < kSl; ++q) w[q][e] = __byte_perm(__float_as_uint(a[q]), __float_as_uint(b[q]), 0x7632);
    }
    const uint32_t off = swz64(r, j);
#pragma unroll
    for (int q = 0; q < kSl; ++q)
        st_shared_v4(tile0 + q * TILE + off, make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]));
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

// The result from its seven sums: T = t 2^sh + r with |t| < 2^51 and 0 <= r < 2^sh, in units of 2^e.
// t goes into the mantissa of 1.5 2^52 2^(e + sh) and r into that of 2^52 2^e; the difference of
// the first to 1.5 2^52 2^(e + sh) + 2^52 2^e is exact, adding the second rounds once: two FP64
// instructions.
__device__ __forceinline__ double assemble(const float (&d)[kSl][4], int c, int sh, int e) {
    int v[kSl];
#pragma unroll
    for (int k = 0; k < kSl; ++k) v[k] = __float2int_rn(d[k][c]);
    const long long h = static_cast<long long>(v[0]) * (1 << 24) + static_cast<long long>(v[1]) * (1 << 16) +
                        static_cast<long long>(v[2]) * (1 << 8) + v[3];
    const long long l = static_cast<long long>(v[4]) * (1 << 16) + static_cast<long long>(v[5]) * (1 << 8) + v[6];
    const long long t = (h << (24 - sh)) + (l >> sh);
    const long long top = static_cast<long long>(((1075 + e + sh) << 20) | 0x80000) << 32;
    const double hi = __longlong_as_double(top + t) - __longlong_as_double(top + (1LL << (52 - sh)));
    return hi + __hiloint2double((1075 + e) << 20, int(l) & ((1 << sh) - 1));
}

// One output by plain FMAs, k ascending (lines whose values do not fit the slices).
__device__ __noinline__ double fma_dot(const double* f, const double* x, int n, long long stride) {
    double acc = 0.0;
    for (int k = 0; k < n; ++k) acc = fma(f[k], x[k * stride], acc);
    return acc;
}

// |v| as an unsigned that orders like |v|: the upper word, with its last bit set where the lower
// word is not zero (so it is 0 only for v = 0). NaN orders above infinity.
__device__ __forceinline__ unsigned f64_amax_bits(double v) {
    return (unsigned(__double2hiint(v)) & 0x7FFFFFFFu) | (__double2loint(v) != 0 ? 1u : 0u);
}

// The phi factor of node o: from the table, or evaluated where the context keeps none.
__device__ __forceinline__ double f64_phi(const F64Args& p, long long o) {
    if (p.phi) return __ldg(p.phi + o);
    double ls = p.lam[0][o % p.n1] + p.lam[1][(o / p.n1) % p.n2];
    if (p.lam[2]) ls += p.lam[2][o / p.n1 / p.n2];
    return phi_eval(p.phik, p.ctau * ls);
}

constexpr int kNoCut = 1 << 20;          // es of a line that fma_dot contracts

template <bool SA, int N, int EPI>
__global__ void __launch_bounds__(kThreads, 1) f64_contract_kernel(const __grid_constant__ F64Args p) {
    using C = Cfg<SA, N>;
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t kSF = 0, kSE = kSF + 8 * C::NS, kFF = kSE + 8 * C::NS, kFE = kFF + 8 * C::NF, kAF = kFE + 8 * C::NF,
                       kAE = kAF + 8, kDR = kAE + 8;
    __shared__ __align__(8) uint64_t bars[kDR / 8 + 1];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
    __shared__ int es_s[4][kM];                              // per line of the last four tiles
    __shared__ unsigned half_s[2][2][kM];                    // SA: the two halves of a line's max|x|

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
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;

    const int n = p.n;
    const long long Q = p.Q;
    const int items = (p.ntiles - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x) * p.nK;   // (tile, K chunk) in order

    if (warp == kLoadWarp) {
        // ------------------------------------------------------------ factor loader (bulk copies)
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 1;
            for (int tile = blockIdx.x; tile < p.ntiles && !abort_s; tile += gridDim.x) {
                const uint8_t* src = p.fimg + size_t(tile % p.nOut) * p.nK * C::FBYTES;
                for (int c = 0; c < p.nK; ++c, src += C::FBYTES) {
                    if (!mbar_wait(fempty(s), ph, p.err, 64, &abort_s, 32)) break;
                    mbar_arrive_expect_tx(ffull(s), C::FBYTES);
                    bulk_g2s(fbase + s * C::FBYTES, src, C::FBYTES, ffull(s));
                    if (++s == C::NF) { s = 0; ph ^= 1; }
                }
            }
        }
    } else if (warp < kProducerWarps) {
        // ------------------------------------------------------------ producers (global -> slices)
        // SA: a thread cuts 16 K values of one position (two chunks of 8); mode 1: 8 of one fibre
        // (N = 32: the upper half of the warps has no rows).
        constexpr int NV = SA ? 2 : 1;
        const int t = threadIdx.x;
        const int row = SA ? (t & (kM - 1)) : (t >> 2);
        const int kofs = SA ? 16 * (t >> 7) : 8 * (t & 3);
        const bool busy = SA || row < N;
        double v[NV][8];
        // the (tile, chunk) whose values are being loaded, and this thread's row of that tile
        int ltile = blockIdx.x, lc = 0;
        const double* xrow = nullptr;
        bool lrow = false, live = true;
        auto set_row = [&]() {
            const unsigned pos = unsigned(ltile / p.nOut) * (SA ? kM : N) + row;
            lrow = ltile < p.ntiles && busy && pos < unsigned(p.npos);
            const unsigned q = SA ? pos % unsigned(Q) : 0u;
            xrow = SA ? p.X + (long long)(pos / unsigned(Q)) * n * Q + q : p.X + (long long)pos * n;
        };
        auto load8 = [&](int h) {
            const int k0 = lc * kKc + kofs + 8 * h;
            const double* x = xrow + (SA ? (long long)k0 * Q : (long long)k0);
            if (SA) {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[h][e] = (lrow && k0 + e < n) ? __ldg(x + e * Q) : 0.0;
            } else if (p.vec2) {
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const double2 w = (lrow && k0 + e < n) ? __ldg(reinterpret_cast<const double2*>(x + e)) : make_double2(0.0, 0.0);
                    v[h][e] = w.x;
                    v[h][e + 1] = w.y;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[h][e] = (lrow && k0 + e < n) ? __ldg(x + e) : 0.0;
            }
        };
        // es of this thread's line: the chunk in v and the line's other chunks
        int etop = 0;
        auto line_scale = [&](int tl) {
            unsigned m = 0;
#pragma unroll
            for (int h = 0; h < NV; ++h)
#pragma unroll
                for (int e = 0; e < 8; ++e) m = max(m, f64_amax_bits(v[h][e]));
            for (int k0 = kKc + kofs; k0 < n; k0 += kKc) {
                const double* x = xrow + (SA ? (long long)k0 * Q : (long long)k0);
#pragma unroll
                for (int e = 0; e < 8 * NV; ++e)
                    if (lrow && k0 + e < n) m = max(m, f64_amax_bits(__ldg(x + (SA ? e * Q : (long long)e))));
            }
            if (SA) {                                        // two threads a line, in different warps
                half_s[tl & 1][t >> 7][row] = m;
                asm volatile("bar.sync 1, %0;" ::"n"(kProducerWarps * 32) : "memory");
                m = max(m, half_s[tl & 1][1 - (t >> 7)][row]);
            } else {                                         // four neighbouring lanes a line
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
            }
            const int eb = int(m >> 20);
            const bool cut_it = m == 0u || (eb >= 1023 - 500 && eb <= 1023 + 500);
            etop = m ? eb : 1022;                            // es + 1022
            if (busy && kofs == 0) es_s[tl & 3][row] = cut_it ? etop - 1022 : kNoCut;
            live = cut_it;
        };
        set_row();
#pragma unroll
        for (int h = 0; h < NV; ++h) load8(h);
        line_scale(0);
        for (int it = 0, ss = 0, sph = 1, tl = 0; it < items; ++it) {
            // waits decide warp-uniformly: the per-warp arrivals below need every lane
            if (!__all_sync(0xffffffffu, mbar_wait(sempty(ss), sph, p.err, 1, &abort_s, 32))) break;
            const bool next_tile = ++lc == p.nK;
            if (next_tile) {
                lc = 0;
                ltile += gridDim.x;
                set_row();
            }
#pragma unroll
            for (int h = 0; h < NV; ++h) {
                if (!live) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[h][e] = 0.0;
                }
                if (busy) cut_store8<C::STILE>(v[h], etop, sbase + ss * C::SBYTES, row, kofs / 8 + h);
                load8(h);                                    // in flight until the next chunk is cut
            }
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
        const int row = ew * 32 + lane;
        const uint32_t tbase = tmem + (uint32_t(ew * 32) << 16);
        uint32_t seg = 0;
        int tl = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x, ++tl) {
            const int pt = tile / p.nOut, ot = tile % p.nOut;
            bool rvalid;
            long long off0, cstep;
            int ncol, rsh = 16, rexp = 0;
            const double* xline = nullptr;                   // SA: this position's line; mode 1: the first fibre's
            if (SA) {
                const unsigned pos = unsigned(pt) * kM + row;
                rvalid = pos < unsigned(p.npos);
                off0 = ((long long)(pos / unsigned(Q)) * n + (long long)ot * N) * Q + pos % unsigned(Q);
                xline = p.X + (long long)(pos / unsigned(Q)) * n * Q + pos % unsigned(Q);
                cstep = Q;
                ncol = min(N, n - ot * N);
            } else {
                const int irow = ot * kM + row;
                rvalid = irow < n;
                const int2 rp = __ldg(p.rows + irow);        // padded to whole tiles
                rsh = rp.y;
                rexp = rp.x;
                xline = p.X + (long long)pt * N * n;
                off0 = (long long)pt * N * n + irow;
                cstep = n;
                ncol = min(N, int(p.npos) - pt * N);
            }
            for (int c0 = 0; c0 < p.nK; c0 += kSegChunks, ++seg) {
                const bool first = c0 == 0;
                const int jlo = part * C::COLS, jhi = jlo + C::COLS;
                // the axpy's base, the phi table's values or the earlier segments' sum, one group ahead
                double bcur[4], bnxt[4];
                double ycur[4], ynxt[4];
                auto load_side = [&](int j0, double (&b)[4], double (&y)[4]) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool in = rvalid && j0 + j < ncol;
                        const long long o = off0 + (long long)(j0 + j) * cstep;
                        b[j] = y[j] = 0.0;
                        if (EPI == EPI_AXPY && in && first) b[j] = p.base[o];
                        if (EPI == EPI_PHI && in) b[j] = f64_phi(p, o);
                        if (in && !first) y[j] = p.Y[o];
                    }
                };
                load_side(jlo, bcur, ycur);
                const bool waited = mbar_wait(accf, seg & 1u, p.err, 2, &abort_s, 32);
                if (!__all_sync(0xffffffffu, waited)) { ok = false; break; }
                tc_fence_after();
                const int* es_t = es_s[tl & 3];
                const int esrow = SA ? es_t[row] : 0;
#pragma unroll 1
                for (int j0 = jlo; j0 < jhi; j0 += 4) {
                    float d[kSl][4];
                    if (j0 + 4 < jhi) load_side(j0 + 4, bnxt, ynxt);
                    int es4[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) es4[j] = SA ? esrow : es_t[j0 + j];
                    __syncwarp();
                    tmem_ld4x7(tbase + j0, uint32_t(N), d);
                    if (j0 + 4 >= jhi) {                     // the last columns are in registers: TMEM is free
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acce);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        int sh = rsh, e = rexp;
                        if (SA) {
                            const int2 cp = __ldg(p.rows + ot * N + j0 + j);
                            sh = cp.y;
                            e = cp.x;
                        }
                        double v = 0.0;
                        if (es4[j] != kNoCut) v = assemble(d, j, sh, e + es4[j]);
                        else if (first && rvalid && j0 + j < ncol)
                            v = SA ? fma_dot(p.factor + (long long)(ot * N + j0 + j) * n, xline, n, Q)
                                   : fma_dot(p.factor + (long long)(ot * kM + row) * n, xline + (long long)(j0 + j) * n, n, 1);
                        if (EPI == EPI_PHI) v *= bcur[j];
                        if (EPI == EPI_AXPY) v = first ? fma(p.alpha, v, bcur[j]) : fma(p.alpha, v, ycur[j]);
                        else if (!first) v += ycur[j];
                        if (rvalid && j0 + j < ncol) p.Y[off0 + (long long)(j0 + j) * cstep] = v;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) { bcur[j] = bnxt[j]; ycur[j] = ynxt[j]; }
                }
            }
        }
    } else if (warp == kMmaWarp && lane == 0) {
        // ------------------------------------------------------------ MMA issuer
        // With X the slices of the A operand and Y those of B (X = S, Y = F for SA, else the other way),
        // X_i.Y_j adds to D_(i+j). The Y tiles lie one after another, as do the accumulators, so X_i
        // takes up to 256 / N consecutive Y_j in one MMA of up to 256 columns: 10 MMAs per
        // K step instead of 28 at N = 64, and X_i is read from shared memory once for them.
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
                const uint64_t a0 = sdesc64(SA ? sS : sF), b0 = sdesc64(SA ? sF : sS);
#pragma unroll
                for (int kk = 0; kk < kKc / 16; ++kk) {
                    const uint64_t adv = uint64_t(kk * 32) >> 4;
#pragma unroll
                    for (int i = 0; i < kSl; ++i)
#pragma unroll
                        for (int j = 0; j < kSl - i; j += C::WIDE) {
                            const int w = (kSl - i - j) < C::WIDE ? (kSl - i - j) : C::WIDE;
                            tc_mma(tmem + (i + j) * N, a0 + adv + uint64_t(i * C::ATILE >> 4),
                                   b0 + adv + uint64_t(j * C::BTILE >> 4), idesc_of(w * N),
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

// Cut the dense factor (n x n, row-major) into its image: per (tile of `rows` rows, K chunk of 32)
// seven 64-byte-swizzled K-major tiles, and per row {ef, sh}. One block per padded row.
__global__ void f64_factor_kernel(const double* M, int n, int rows, int nK, uint8_t* img, int2* rp) {
    const int i = blockIdx.x;
    __shared__ unsigned smax;
    __shared__ double ssum;
    if (threadIdx.x == 0) { smax = 0; ssum = 0.0; }
    __syncthreads();
    unsigned m = 0;
    if (i < n)
        for (int k = threadIdx.x; k < n; k += blockDim.x) m = max(m, f64_amax_bits(M[(size_t)i * n + k]));
    atomicMax(&smax, m);
    __syncthreads();
    const int e = int(smax >> 20);
    // max|f| < 2^ef; rows below 2^-500 keep that scale (their digits are then smaller)
    const int ef = smax ? max(e - 1022, -500) : 0;
    double sum = 0.0;
    if (i < n)
        for (int k = threadIdx.x; k < n; k += blockDim.x) sum += fabs(M[(size_t)i * n + k]);
    atomicAdd(&ssum, sum);
    __syncthreads();
    if (threadIdx.x == 0) {
        // |T| <= 2^64 sum|f| 2^-ef: sh so that T / 2^sh stays below 2^51 (n <= 1024: sh <= 24)
        int q = 0;
        const double s = ldexp(ssum, -ef) * (1.0 + 1e-6);
        if (s > 0.0) frexp(s, &q);
        rp[i] = make_int2(ef - 64, min(max(13 + q, 1), 24));
    }
    uint8_t* tile = img + (size_t)(i / rows) * nK * kSl * rows * 64;
    for (int k = threadIdx.x; k < nK * kKc; k += blockDim.x) {
        const double f = (i < n && k < n) ? M[(size_t)i * n + k] : 0.0;
        float s[kSl];
        cut(f, ef + 1022, s);
        const int kc = k % kKc;
        uint8_t* dst = tile + (size_t)(k / kKc) * kSl * rows * 64 + swz64(i % rows, kc / 8) + (kc % 8) * 2;
#pragma unroll
        for (int q = 0; q < kSl; ++q)
            *reinterpret_cast<uint16_t*>(dst + (size_t)q * rows * 64) = uint16_t(__float_as_uint(s[q]) >> 16);
    }
}

__global__ void f64_phi_kernel(double* tab, int k, double ctau, const double* l1, const double* l2, const double* l3, int n1,
                               int n2, size_t N) {
    for (size_t o = blockIdx.x * size_t(blockDim.x) + threadIdx.x; o < N; o += size_t(gridDim.x) * blockDim.x) {
        double ls = l1[o % n1] + l2[(o / n1) % n2];
        if (l3) ls += l3[o / n1 / n2];
        tab[o] = phi_eval(k, ctau * ls);
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

template <bool SA, int N, int EPI>
cudaError_t launch_variant(const F64Args& a, cudaStream_t s) {
    static const cudaError_t attr = cudaFuncSetAttribute(f64_contract_kernel<SA, N, EPI>,
                                                         cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<SA, N>::SMEM);
    if (attr != cudaSuccess) return attr;
    const long long grid = a.ntiles < sm_count() ? a.ntiles : sm_count();
    f64_contract_kernel<SA, N, EPI><<<unsigned(grid), kThreads, Cfg<SA, N>::SMEM, s>>>(a);
    return cudaGetLastError();
}

template <bool SA, int N>
cudaError_t launch_epi(const F64Args& a, cudaStream_t s) {
    if (a.epi == EPI_PHI) return launch_variant<SA, N, EPI_PHI>(a, s);
    if (a.epi == EPI_AXPY) return launch_variant<SA, N, EPI_AXPY>(a, s);
    return launch_variant<SA, N, EPI_STORE>(a, s);
}

}  // namespace

F64Tiles f64_tiles(int n, long long npos, bool mode1) {
    F64Tiles t;
    t.nK = (n + kKc - 1) / kKc;
    // 64 columns, or 32 where 64 would give fewer tiles than SMs
    for (int cols : {64, 32}) {
        t.cols = cols;
        t.rows = mode1 ? kM : cols;                          // factor rows per tile
        t.nOut = (n + t.rows - 1) / t.rows;
        t.ntiles = (mode1 ? (npos + cols - 1) / cols : (npos + kM - 1) / kM) * t.nOut;
        if (t.ntiles >= sm_count()) break;
    }
    return t;
}

size_t f64_image_bytes(const F64Tiles& t) { return size_t(t.nOut) * t.rows * t.nK * kKc * 2 * kSl; }

cudaError_t launch_f64_factor(const double* M, int n, const F64Tiles& t, uint8_t* img, int2* rows, cudaStream_t s) {
    f64_factor_kernel<<<t.nOut * t.rows, 128, 0, s>>>(M, n, t.rows, t.nK, img, rows);
    return cudaGetLastError();
}

cudaError_t launch_f64_phi(double* tab, int k, double ctau, const double* const lam[3], int n1, int n2, size_t N, cudaStream_t s) {
    const unsigned blocks = unsigned((N + 255) / 256 < 65535 ? (N + 255) / 256 : 65535);
    f64_phi_kernel<<<blocks, 256, 0, s>>>(tab, k, ctau, lam[0], lam[1], lam[2], n1, n2, N);
    return cudaGetLastError();
}

cudaError_t launch_contract_f64(const F64Args& a, bool mode1, int cols, cudaStream_t s) {
    if (a.ntiles <= 0) return cudaSuccess;
    if (mode1) return cols == 64 ? launch_epi<false, 64>(a, s) : launch_epi<false, 32>(a, s);
    return cols == 64 ? launch_epi<true, 64>(a, s) : launch_epi<true, 32>(a, s);
}

}  // namespace adr
