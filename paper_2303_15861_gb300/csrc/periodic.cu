// Periodic Fourier pseudospectral contexts: the discretisation of the paper's two-dimensional
// experiment (Section 5.1, Eq. (ad2d)), where A of Eq. (linop) is diagonal in Fourier space and
// its matrix functions are multipliers on the Fourier coefficients (Section 5.1).
//
// Every nodal array is real, so Fourier space holds half of it: k_1 = 0 .. n_1/2, H = n_1/2 + 1
// columns (x1 fastest, then x2, x3 as in the nodal arrays), the other half being its conjugate. A row of n real
// nodes is transformed as m = n/2 complex points z_j = x_2j + i x_(2j+1): with Z their transform, Z~_k = conj(Z_(m-k)) and
// w = e^{-2 pi i / n}, the row's coefficients are X_k = (E - i w^k O) / 2, E = Z + Z~, O = Z - Z~, and back Z = ((X + X~) +
// i w^-k (X - X~)) / 2. The divisions by 2 are left out (half arrays hold twice the coefficients) and taken with the
// 1/n of the inverse transforms where a row comes back to real space. (Two rows as the real and imaginary parts of one
// line take as many operations, but round equal rows differently.)
//
// FFT: complex radix-4 transforms (one radix-2 stage first when log2 n is odd) along one axis at
// a time in the Stockham autosort form (each stage reads one shared-memory buffer and writes the
// other in natural order, so no bit reversal is needed), twiddles e^{-2 pi i j / n}, j < n/2,
// from a host FP64 table. A block takes G neighbouring lines of one axis, of one or several arrays at
// once, into shared memory.
//
// Fusion. A d-dimensional transform is d passes. The last axis d is the pivot: there all other
// axes are already transformed, so the pivot pass does the forward transform, the pointwise
// work in Fourier space and the inverse transform in one kernel. The passes along x1 take the
// real-space prologue (a real input) or epilogue (the stage combination). i k_mu is constant along the
// other axes, so a derivative D_mu u needs only the transforms along the axes up to mu, and the divergence is
// added up as the axes are transformed: D_1 u and i k_1 f_1^ belong to the passes along x1.
//   Multiplier y = base + alpha Re F^-1(M F x):   x1 fwd | (x2 fwd) | pivot: F, M, F^-1 |
//                                                (x2 inv) | x1 inv + axpy.          2-D: 3 kernels
//   Right-hand side, F(u) = sum_mu D_mu (a_mumu D_mu u + b_mu u) + r(u), g = F - A u, with the
//   spectral first derivative D_mu = F^-1 i k_mu F (Nyquist wavenumber 0):
//     x1 fwd u | (x2: fwd, i k_2 back) | pivot: u^, i k_d u^ back | (x2 inv) |
//     x1: D_mu u -> flux f_mu = a_mumu D_mu u + b_mu u -> forward, G = i k_1 f_1^ |
//     (x2 fwd, G += i k_2 f_2^) | pivot: S = G^ + i k_d f_d^, O_j = (cg_j + cF_j) S - cg_j s u^ | (x2 inv) |
//     x1 inv + out_j = cu_j u + sum_e cx_je X_e + Re O_j + (cg_j + cF_j) r(u).      2-D: 5 kernels
//   A stage kept in Fourier space (2-D; see PeriodicStage): the first three passes as above, with r(u) (and
//   the a Lap u product) transformed in the third one and added to G; the pivot then forms F^, combines it
//   with u^, a saved array Z and the multipliers, saves
//   Ms (zu u^ + zF F^ - zg s u^) for a later stage, and transforms back; the last x1 pass
//   writes y.                                                                           2-D: 5 kernels
//   When the next stage's input is this y, the last x1 pass also transforms y forward along x1
//   into Cx, and the next stage starts at its pivot pass.                       2-D: 4 kernels more
// Transforms along one axis per 2-D stage, in units of one of all n_1 n_2 complex points: 6 (x1 1/2, pivot 1, fluxes 5/2,
// pivot 3/2, x1 1/2) instead of 14 on whole complex arrays with every derivative taken to Fourier space. FP64 is bounded
// by its FP64 instructions: 256^2 Lawson2a 163 -> 79 us a step, 1024^2 2.59 -> 1.11 ms, 64^3 494 -> 217 us. FP32 on
// small grids is bounded by the latency of a pass (loads, barriers of log_4 n stages, stores): 256^2 ETD2RK 36.6 -> 19.2 us a step,
// 64^3 Lawson4 222 -> 144 us, 32^2 Lawson4 (32 passes a step) 42.0 -> 41.6 us.
#include <cuda_runtime.h>

#include <algorithm>

#include "adr_internal.h"

namespace adr {
namespace {

template <typename T>
__device__ __forceinline__ Cplx<T> cmul(Cplx<T> a, Cplx<T> b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T>
__device__ __forceinline__ Cplx<T> mul_i(T k, Cplx<T> a) {   // i k a
    return {-k * a.y, k * a.x};
}

enum PassMode {
    // along x1
    PM_FWD_REAL = 0,     // C[0] = F_1 x (x real)
    PM_FINAL_AXPY = 1,   // y = base + alpha F_1^-1 C[0]  (y = F_1^-1 C[0] without base)
    PM_FINAL_FWD = 2,    // y = F_1^-1 C[0]; Cx = F_1 y (the next stage's first pass)
    PM_FLUX = 3,         // f_mu = a_mumu D_mu u + b_mu u; C[0] = i k_1 F_1 f_1 (+ F_1 of the pointwise part),
                         // C[mu] = F_1 f_mu
    PM_FINAL_OUT = 4,    // out_j = cu_j u + sum cx_je X_e + F_1^-1 C[j] + cgF_j r(u)
    // along another axis
    PM_PLAIN = 5,        // C[a] = F_mu C[a] or F_mu^-1 C[a], a < na
    PM_DERIV = 6,        // Cu = F_mu src; C[mu] = F_mu^-1 (i k_mu Cu)
    PM_MID_DIV = 7,      // 3-D, x2: C[0] = F_2 C[0] + i k_2 F_2 C[1]; C[2] = F_2 C[2]
    PM_PIVOT_MULT = 8,   // C[0] = F_d^-1 (M F_d C[0])
    PM_PIVOT_DIV = 9,    // S = F_d C[0] + i k_d F_d C[d-1]; C[j] = F_d^-1 (cgF_j S - cg_j M Cu)
    PM_PIVOT_STAGE = 10, // F^ = S, H = cgF F^ - cg s u^;
                         // C[0] = F_d^-1 (Mu (cu u^) + Mg (H + cgz Z) + cz Z);
                         // Zs = Ms (zu u^ + zF F^ - zg s u^)
};

constexpr int kPassThreads = 256;
constexpr size_t kPassSmemMax = 200 * 1024;

template <typename T>
struct Pass {
    // the pass: length n of its axis, 2^llen complex points a line (n/2 along x1), twiddle stride 2^tshift, G =
    // 2^logG lines of each array per block, nb arrays in shared memory at once, shared-memory row pitch
    int axis, n, llen, tshift, G, logG, nb, pitch;
    int H;                    // columns of a half array
    long long Q;              // other axes: stride of the axis = lines per outer index
    long long per_outer;      // ... line groups per outer index
    long long groups;         // line groups in the grid
    int dim;
    const Cplx<T>* tw;
    const T* k;               // wavenumbers of the axis
    // arrays
    Cplx<T>* Cu;
    Cplx<T>* Cx;
    Cplx<T>* C[3];
    const Cplx<T>* src;       // PM_DERIV
    int na, inverse;
    const Cplx<T>* M;         // multiplier (PM_PIVOT_MULT) or symbol of A
    const T* x;               // real input: x (PM_FWD_REAL) or the stage input u
    T* y;
    const T* base;
    T alpha;
    T sc[3];                  // scale of a line of array a that comes back to real space
    const T* a[3];
    const T* b[3];
    int nout, nx;
    const T* X[kMaxExtra];
    T* out[kMaxOut];
    T cu[kMaxOut], cx[kMaxOut][kMaxExtra], cgF[kMaxOut], cg[kMaxOut], r[4];
    int adelta;               // a Lap u form (see PeriodicArgs)
    T* dif;                   // adelta: sum_mu a_mumu D_mu D_mu u
    // fused stages: r(u) and the a Lap u product transformed with the fluxes (PM_FLUX); the stage's
    // multipliers and saved array (PM_PIVOT_STAGE)
    int nonflux;
    const Cplx<T>* Mu;
    const Cplx<T>* Mg;
    const Cplx<T>* Ms;
    const Cplx<T>* Z;
    Cplx<T>* Zs;
    T scu, scgF, scg, scgz, scz;
    T szu, szF, szg;
};

// Call f(smem offset, global index in a half array, position along the axis) for every element of the
// block's G lines of one array, in the order that makes consecutive threads touch consecutive global elements.
template <typename T, typename F>
__device__ __forceinline__ void col_elems(const Pass<T>& P, long long grp, F f) {
    const long long p = grp / P.per_outer, q0 = (grp % P.per_outer) << P.logG;
    const long long base = p * P.n * P.Q + q0;
    for (int idx = threadIdx.x; idx < (P.G << P.llen); idx += blockDim.x) {
        const int g = idx & (P.G - 1), j = idx >> P.logG;
        if (q0 + g < P.Q) f(g * P.pitch + j, base + (long long)j * P.Q + g, j);
    }
}

// Passes along x1: f(smem offset, index of the first of two neighbouring nodes), and the Fourier columns k and
// m - k, f(line, k, index of column k, index of column m - k), k = 0 .. m/2.
template <typename T, typename F>
__device__ __forceinline__ void row_nodes(const Pass<T>& P, long long grp, F f) {
    for (int idx = threadIdx.x; idx < (P.G << P.llen); idx += blockDim.x) {
        const int g = idx >> P.llen, j = idx & ((1 << P.llen) - 1);
        f(g * P.pitch + j, ((grp << P.logG) + g) * P.n + 2 * j);
    }
}
template <typename T, typename F>
__device__ __forceinline__ void row_cols(const Pass<T>& P, long long grp, F f) {
    const int m = 1 << P.llen, lh = P.llen > 0 ? P.llen - 1 : 0;
    for (int idx = threadIdx.x; idx < (P.G << lh); idx += blockDim.x) {
        const int g = idx >> lh, k = idx & ((1 << lh) - 1);
        const long long row = ((grp << P.logG) + g) * P.H;
        f(g, k, row + k, row + m - k);
        if (k == 0 && m > 1) f(g, m >> 1, row + (m >> 1), row + (m >> 1));
    }
}

// A row's coefficients (times 2) of columns k and m - k from its line's transform R.
template <typename T>
__device__ __forceinline__ void split(const Pass<T>& P, const Cplx<T>* tws, const Cplx<T>* R, int k, Cplx<T>& A, Cplx<T>& B) {
    const int m = 1 << P.llen;
    if (k == 0) {
        const Cplx<T> z = R[0];
        A = {T(2) * (z.x + z.y), T(0)};
        B = {T(2) * (z.x - z.y), T(0)};
        return;
    }
    const Cplx<T> z = R[k], y = R[m - k];
    const Cplx<T> E = {z.x + y.x, z.y - y.y};
    const Cplx<T> V = cmul(tws[k], Cplx<T>{z.y + y.y, y.x - z.x});   // -i w^k O
    A = {E.x + V.x, E.y + V.y};
    B = {E.x - V.x, V.y - E.y};
}
// The line to transform back from the row's coefficients of columns k and m - k.
template <typename T>
__device__ __forceinline__ void join(const Pass<T>& P, const Cplx<T>* tws, Cplx<T>* R, int k, Cplx<T> A, Cplx<T> B) {
    const int m = 1 << P.llen;
    if (k == 0) {                                         // both are real
        R[0] = {A.x + B.x, A.x - B.x};
        return;
    }
    const Cplx<T> E = {A.x + B.x, A.y - B.y};
    const Cplx<T> V = cmul({tws[k].x, -tws[k].y}, Cplx<T>{-(A.y + B.y), A.x - B.x});   // i w^-k O
    R[k] = {E.x + V.x, E.y + V.y};
    if (2 * k != m) R[m - k] = {E.x - V.x, V.y - E.y};
}

// Stockham transform of nl lines in src (destroys src and dst); returns the buffer that holds
// the result (unscaled). Radix-4 stages, after one radix-2 stage when log2 n is odd: a stage over
// sub-transforms of length Ns takes the four points j + q n/4 (q = 0..3) of butterfly j,
// r = j mod Ns, scales point q by e^{-2 pi i q r / (4 Ns)} (conjugated for the inverse), forms
// their 4-point DFT V_k and writes V_k to 4 (j - r) + r + k Ns.
template <typename T>
__device__ Cplx<T>* fft_lines(const Pass<T>& P, const Cplx<T>* tws, Cplx<T>* src, Cplx<T>* dst, int nl, bool inverse) {
    const int half = (1 << P.llen) >> 1, quarter = (1 << P.llen) >> 2, thalf = P.n >> 1;
    int s = 0, Ns = 1;
    if (P.llen & 1) {                                     // radix 2 with Ns = 1: all twiddles are 1
        for (int bf = threadIdx.x; bf < nl * half; bf += blockDim.x) {
            const int g = bf >> (P.llen - 1), jj = bf & (half - 1);
            const Cplx<T>* sl = src + g * P.pitch;
            Cplx<T>* dl = dst + g * P.pitch;
            const Cplx<T> v0 = sl[jj], v1 = sl[jj + half];
            dl[2 * jj] = {v0.x + v1.x, v0.y + v1.y};
            dl[2 * jj + 1] = {v0.x - v1.x, v0.y - v1.y};
        }
        __syncthreads();
        Cplx<T>* t = src;
        src = dst;
        dst = t;
        s = 1;
        Ns = 2;
    }
    for (; s < P.llen; s += 2, Ns <<= 2) {
        const int lstep = P.llen - 2 - s + P.tshift;      // table steps of n / (4 Ns) points
        for (int bf = threadIdx.x; bf < nl * quarter; bf += blockDim.x) {
            const int g = bf >> (P.llen - 2), jj = bf & (quarter - 1);
            const int r = jj & (Ns - 1);
            const Cplx<T>* sl = src + g * P.pitch;
            Cplx<T>* dl = dst + g * P.pitch;
            Cplx<T> v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = sl[jj + q * quarter];
            if (Ns > 1) {
#pragma unroll
                for (int q = 1; q < 4; ++q) {             // e^{-2 pi i m / n}, m = q r n / (4 Ns) < 3n/4
                    const int m = (q * r) << lstep;
                    Cplx<T> w = m < thalf ? tws[m] : Cplx<T>{-tws[m - thalf].x, -tws[m - thalf].y};
                    if (inverse) w.y = -w.y;
                    v[q] = cmul(v[q], w);
                }
            }
            const Cplx<T> a0 = {v[0].x + v[2].x, v[0].y + v[2].y}, a1 = {v[0].x - v[2].x, v[0].y - v[2].y};
            const Cplx<T> a2 = {v[1].x + v[3].x, v[1].y + v[3].y}, a3 = {v[1].x - v[3].x, v[1].y - v[3].y};
            // -i a3 = (a3.y, -a3.x) for the forward transform, +i a3 for the inverse
            const Cplx<T> ia3 = inverse ? Cplx<T>{-a3.y, a3.x} : Cplx<T>{a3.y, -a3.x};
            const int o = ((jj - r) << 2) + r;
            dl[o] = {a0.x + a2.x, a0.y + a2.y};
            dl[o + Ns] = {a1.x + ia3.x, a1.y + ia3.y};
            dl[o + 2 * Ns] = {a0.x - a2.x, a0.y - a2.y};
            dl[o + 3 * Ns] = {a1.x - ia3.x, a1.y - ia3.y};
        }
        __syncthreads();
        Cplx<T>* t = src;
        src = dst;
        dst = t;
    }
    return src;
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kPassThreads) fourier_pass_kernel(const __grid_constant__ Pass<T> P) {
    extern __shared__ __align__(16) unsigned char fourier_smem[];
    Cplx<T>* tws = reinterpret_cast<Cplx<T>*>(fourier_smem);
    Cplx<T>* B0 = tws + (P.n >> 1);
    const int lsize = P.G * P.pitch;                      // the lines of one array
    Cplx<T>* B1 = B0 + P.nb * lsize;
    for (int j = threadIdx.x; j < (P.n >> 1); j += blockDim.x) tws[j] = P.tw[j];
    __syncthreads();

    for (long long grp = blockIdx.x; grp < P.groups; grp += gridDim.x) {
        if (MODE == PM_FWD_REAL) {
            row_nodes(P, grp, [&](int o, long long i) { B0[o] = {P.x[i], P.x[i + 1]}; });
            __syncthreads();
            const Cplx<T>* R = fft_lines(P, tws, B0, B1, P.G, false);
            row_cols(P, grp, [&](int g, int k, long long c0, long long c1) {
                Cplx<T> A, B;
                split(P, tws, R + g * P.pitch, k, A, B);
                P.C[0][c0] = A;
                if (c0 != c1) P.C[0][c1] = B;
            });
        } else if (MODE == PM_FINAL_AXPY || MODE == PM_FINAL_FWD) {
            row_cols(P, grp, [&](int g, int k, long long c0, long long c1) {
                join(P, tws, B0 + g * P.pitch, k, P.C[0][c0], P.C[0][c1]);
            });
            __syncthreads();
            Cplx<T>* R = fft_lines(P, tws, B0, B1, P.G, true);
            row_nodes(P, grp, [&](int o, long long i) {
                const Cplx<T> v = {R[o].x * P.sc[0], R[o].y * P.sc[0]};
                if (MODE == PM_FINAL_FWD) {               // the same values PM_FWD_REAL would read
                    P.y[i] = v.x;
                    P.y[i + 1] = v.y;
                    R[o] = v;
                } else {
                    P.y[i] = P.base ? P.base[i] + P.alpha * v.x : v.x;
                    P.y[i + 1] = P.base ? P.base[i + 1] + P.alpha * v.y : v.y;
                }
            });
            if (MODE == PM_FINAL_FWD) {
                __syncthreads();
                const Cplx<T>* R2 = fft_lines(P, tws, R, R == B0 ? B1 : B0, P.G, false);
                row_cols(P, grp, [&](int g, int k, long long c0, long long c1) {
                    Cplx<T> A, B;
                    split(P, tws, R2 + g * P.pitch, k, A, B);
                    P.Cx[c0] = A;
                    if (c0 != c1) P.Cx[c1] = B;
                });
            }
        } else if (MODE == PM_FLUX) {
            // the d fluxes and the pointwise part: all at once where they fit the shared memory (nb arrays), else
            // one after another
            const int na = P.dim + (P.nonflux ? 1 : 0), m = 1 << P.llen;
            for (int a0 = 0; a0 < na; a0 += P.nb) {
                const int a1 = min(a0 + P.nb, na), nd = min(a1, P.dim) - a0;
                const bool all = P.nb == na;
                for (int a = a0; a < a0 + nd; ++a) {
                    Cplx<T>* L = B0 + (a - a0) * lsize;
                    row_cols(P, grp, [&](int g, int k, long long c0, long long c1) {
                        Cplx<T> A, B;
                        if (a == 0) {                     // D_1 u (or D_1 D_1 u) from the transform along x1
                            const T ka = P.k[k], kb = P.k[m - k];
                            A = P.Cx[c0];
                            B = P.Cx[c1];
                            if (P.adelta) {
                                A = {-ka * ka * A.x, -ka * ka * A.y};
                                B = {-kb * kb * B.x, -kb * kb * B.y};
                            } else {
                                A = mul_i(ka, A);
                                B = mul_i(kb, B);
                            }
                        } else {
                            A = P.C[a][c0];
                            B = P.C[a][c1];
                        }
                        join(P, tws, L + g * P.pitch, k, A, B);
                    });
                }
                __syncthreads();
                Cplx<T>* R = nd > 0 ? fft_lines(P, tws, B0, B1, nd * P.G, true) : B0;
                row_nodes(P, grp, [&](int o, long long i) {
                    const T u0 = P.x[i], u1 = P.x[i + 1];
                    T d0 = T(0), d1 = T(0);               // adelta: sum_mu a_mumu D_mu D_mu u
                    if (P.adelta && !all && a0 > 0) {
                        d0 = P.dif[i];
                        d1 = P.dif[i + 1];
                    }
                    for (int a = a0; a < a0 + nd; ++a) {
                        Cplx<T>& L = R[o + (a - a0) * lsize];
                        const T v0 = P.a[a][i] * (L.x * P.sc[a]), v1 = P.a[a][i + 1] * (L.y * P.sc[a]);
                        if (P.adelta) {                   // D_mu D_mu u is complete here; the flux is b_mu u
                            d0 += v0;
                            d1 += v1;
                            L = {P.b[a][i] * u0, P.b[a][i + 1] * u1};
                        } else {
                            L = {v0 + P.b[a][i] * u0, v1 + P.b[a][i + 1] * u1};
                        }
                    }
                    if (P.adelta && nd > 0 && !(all && P.nonflux)) {
                        P.dif[i] = d0;
                        P.dif[i + 1] = d1;
                    }
                    if (a1 > P.dim)
                        R[o + (P.dim - a0) * lsize] = {
                            P.r[0] + u0 * (P.r[1] + u0 * (P.r[2] + u0 * P.r[3])) + d0,
                            P.r[0] + u1 * (P.r[1] + u1 * (P.r[2] + u1 * P.r[3])) + d1};
                });
                __syncthreads();
                const Cplx<T>* R2 = fft_lines(P, tws, R, R == B0 ? B1 : B0, (a1 - a0) * P.G, false);
                row_cols(P, grp, [&](int g, int k, long long c0, long long c1) {
                    for (int a = a0; a < a1; ++a) {
                        if (all && a == P.dim) break;     // added to array 0 below
                        Cplx<T> A, B;
                        split(P, tws, R2 + (a - a0) * lsize + g * P.pitch, k, A, B);
                        Cplx<T>* D = P.C[a == P.dim ? 0 : a];
                        if (a == 0) {
                            A = mul_i(P.k[k], A);
                            B = mul_i(P.k[m - k], B);
                        }
                        if (a == P.dim || (all && a == 0 && P.nonflux)) {
                            Cplx<T> rA, rB;
                            if (a == P.dim) {
                                rA = D[c0];
                                rB = D[c1];
                            } else {
                                split(P, tws, R2 + P.dim * lsize + g * P.pitch, k, rA, rB);
                            }
                            A = {A.x + rA.x, A.y + rA.y};
                            B = {B.x + rB.x, B.y + rB.y};
                        }
                        D[c0] = A;
                        if (2 * k != m) D[c1] = B;
                    }
                });
                __syncthreads();
            }
        } else if (MODE == PM_FINAL_OUT) {
            for (int jo = 0; jo < P.nout; ++jo) {
                row_cols(P, grp, [&](int g, int k, long long c0, long long c1) {
                    join(P, tws, B0 + g * P.pitch, k, P.C[jo][c0], P.C[jo][c1]);
                });
                __syncthreads();
                const Cplx<T>* R = fft_lines(P, tws, B0, B1, P.G, true);
                T* out = P.out[jo];
                auto finish = [&](long long i, T w) {
                    const T u = P.x[i];
                    T v = P.cu[jo] * u + w + P.cgF[jo] * (P.r[0] + u * (P.r[1] + u * (P.r[2] + u * P.r[3])));
                    if (P.adelta) v += P.cgF[jo] * P.dif[i];
                    for (int e = 0; e < P.nx; ++e) v += P.cx[jo][e] * P.X[e][i];
                    out[i] = v;
                };
                row_nodes(P, grp, [&](int o, long long i) {
                    finish(i, R[o].x * P.sc[0]);
                    finish(i + 1, R[o].y * P.sc[0]);
                });
                __syncthreads();
            }
        } else if (MODE == PM_PLAIN) {
            for (int a = 0; a < P.na; ++a) {
                Cplx<T>* A = P.C[a];
                col_elems(P, grp, [&](int o, long long i, int) { B0[o] = A[i]; });
                __syncthreads();
                const Cplx<T>* R = fft_lines(P, tws, B0, B1, P.G, P.inverse != 0);
                col_elems(P, grp, [&](int o, long long i, int) { A[i] = R[o]; });
                __syncthreads();
            }
        } else if (MODE == PM_DERIV) {
            col_elems(P, grp, [&](int o, long long i, int) { B0[o] = P.src[i]; });
            __syncthreads();
            Cplx<T>* U = fft_lines(P, tws, B0, B1, P.G, false);
            col_elems(P, grp, [&](int o, long long i, int j) {
                const Cplx<T> v = U[o];
                const T k = P.k[j];
                P.Cu[i] = v;
                U[o] = P.adelta ? Cplx<T>{-k * k * v.x, -k * k * v.y} : mul_i(k, v);
            });
            __syncthreads();
            const Cplx<T>* R = fft_lines(P, tws, U, U == B0 ? B1 : B0, P.G, true);
            Cplx<T>* D = P.C[P.axis];
            col_elems(P, grp, [&](int o, long long i, int) { D[i] = R[o]; });
        } else if (MODE == PM_MID_DIV) {
            for (int a = 0; a < 3; ++a)
                col_elems(P, grp, [&](int o, long long i, int) { B0[o + a * lsize] = P.C[a][i]; });
            __syncthreads();
            const Cplx<T>* R = fft_lines(P, tws, B0, B1, 3 * P.G, false);
            col_elems(P, grp, [&](int o, long long i, int j) {
                const Cplx<T> d = mul_i(P.k[j], R[o + lsize]);
                P.C[0][i] = {R[o].x + d.x, R[o].y + d.y};
                P.C[2][i] = R[o + 2 * lsize];
            });
        } else if (MODE == PM_PIVOT_MULT) {
            col_elems(P, grp, [&](int o, long long i, int) { B0[o] = P.C[0][i]; });
            __syncthreads();
            Cplx<T>* R = fft_lines(P, tws, B0, B1, P.G, false);
            col_elems(P, grp, [&](int o, long long i, int) { R[o] = cmul(R[o], P.M[i]); });
            __syncthreads();
            const Cplx<T>* R2 = fft_lines(P, tws, R, R == B0 ? B1 : B0, P.G, true);
            col_elems(P, grp, [&](int o, long long i, int) { P.C[0][i] = R2[o]; });
        } else if (MODE == PM_PIVOT_STAGE) {
            col_elems(P, grp, [&](int o, long long i, int) {
                B0[o] = P.C[0][i];
                B0[o + lsize] = P.C[P.axis][i];
            });
            __syncthreads();
            Cplx<T>* R = fft_lines(P, tws, B0, B1, 2 * P.G, false);
            col_elems(P, grp, [&](int o, long long i, int j) {
                const Cplx<T> d = mul_i(P.k[j], R[o + lsize]);
                const Cplx<T> fh = {R[o].x + d.x, R[o].y + d.y};
                const Cplx<T> uh = P.Cu[i];
                const Cplx<T> au = cmul(P.M[i], uh);
                const Cplx<T> z = P.Z ? P.Z[i] : Cplx<T>{T(0), T(0)};
                if (P.Zs) {
                    const Cplx<T> w = {P.szu * uh.x + P.szF * fh.x - P.szg * au.x,
                                       P.szu * uh.y + P.szF * fh.y - P.szg * au.y};
                    P.Zs[i] = P.Ms ? cmul(P.Ms[i], w) : w;
                }
                Cplx<T> h = {P.scgF * fh.x - P.scg * au.x + P.scgz * z.x,
                             P.scgF * fh.y - P.scg * au.y + P.scgz * z.y};
                if (P.Mg) h = cmul(P.Mg[i], h);
                Cplx<T> v = {P.scu * uh.x, P.scu * uh.y};
                if (P.Mu) v = cmul(P.Mu[i], v);
                R[o] = {v.x + h.x + P.scz * z.x, v.y + h.y + P.scz * z.y};
            });
            __syncthreads();
            const Cplx<T>* R2 = fft_lines(P, tws, R, R == B0 ? B1 : B0, P.G, true);
            col_elems(P, grp, [&](int o, long long i, int) { P.C[0][i] = R2[o]; });
        } else if (MODE == PM_PIVOT_DIV) {
            col_elems(P, grp, [&](int o, long long i, int) {
                B0[o] = P.C[0][i];
                B0[o + lsize] = P.C[P.axis][i];
            });
            __syncthreads();
            Cplx<T>* R = fft_lines(P, tws, B0, B1, 2 * P.G, false);
            Cplx<T>* O = R == B0 ? B1 : B0;
            for (int jo = 0; jo < P.nout; ++jo) {          // S stays in the first lines of R
                const T cgF = P.cgF[jo], cg = P.cg[jo];
                col_elems(P, grp, [&](int o, long long i, int j) {
                    if (jo == 0) {
                        const Cplx<T> d = mul_i(P.k[j], R[o + lsize]);
                        R[o] = {R[o].x + d.x, R[o].y + d.y};
                    }
                    const Cplx<T> au = cmul(P.M[i], P.Cu[i]);
                    R[o + lsize] = {cgF * R[o].x - cg * au.x, cgF * R[o].y - cg * au.y};
                });
                __syncthreads();
                const Cplx<T>* R2 = fft_lines(P, tws, R + lsize, O + lsize, P.G, true);
                Cplx<T>* D = P.C[jo];
                col_elems(P, grp, [&](int o, long long i, int) { D[i] = R2[o]; });
                __syncthreads();
            }
        }
        __syncthreads();
    }
}

int ilog2(long long v) {
    int l = 0;
    while ((1LL << l) < v) ++l;
    return l;
}

int g_sms = 0;
int sms() {
    if (g_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

// Arrays a mode transforms at once (PM_FLUX: the fluxes and the pointwise part, or one where that
// does not fit).
int mode_arrays(int mode, int dim, bool nonflux) {
    if (mode == PM_FLUX) return dim + (nonflux ? 1 : 0);
    if (mode == PM_MID_DIV) return 3;
    return mode == PM_PIVOT_DIV || mode == PM_PIVOT_STAGE ? 2 : 1;
}

size_t pass_smem(int n, int G, int pitch, int nb, size_t cs) { return (size_t(n / 2) + 2 * size_t(nb) * G * pitch) * cs; }

// Geometry of a pass along `axis`: G lines per block, as many as keep at least two blocks per
// SM busy and fit the shared memory (and up to a 32-byte sector while every SM keeps a block).
template <typename T>
Pass<T> make_pass(const PeriodicArgs<T>& A, int axis, int mode, bool nonflux = false) {
    Pass<T> P{};
    P.axis = axis;
    P.dim = A.dim;
    P.H = A.n[0] / 2 + 1;
    for (int m = 0; m < A.dim; ++m) {
        P.a[m] = A.a[m];
        P.b[m] = A.b[m];
        P.C[m] = A.C[m];
    }
    P.n = A.n[axis];
    P.tshift = axis == 0 ? 1 : 0;
    P.llen = ilog2(P.n) - P.tshift;
    P.k = A.k[axis];
    const size_t cs = sizeof(Cplx<T>);
    P.nonflux = nonflux ? 1 : 0;
    P.nb = mode_arrays(mode, A.dim, nonflux);
    P.pitch = axis == 0 ? P.n / 2 : P.n + 1;
    if (pass_smem(P.n, 1, P.pitch, P.nb, cs) > kPassSmemMax) P.nb = 1;
    long long lines, limit;                               // lines of an array in all and per outer index
    if (axis == 0) {
        lines = limit = A.N / P.n;
    } else {
        P.Q = P.H;
        for (int m = 1; m < axis; ++m) P.Q *= A.n[m];
        limit = P.Q;
        lines = A.N / A.n[0] * P.H / P.n;
    }
    int G = 1;
    auto fits = [&](int g2) { return g2 <= limit && pass_smem(P.n, g2, P.pitch, P.nb, cs) <= kPassSmemMax; };
    while (fits(2 * G) && lines / (2 * G) >= 2LL * sms()) G *= 2;
    while (axis > 0 && size_t(G) * cs < 32 && fits(2 * G) && lines / (2 * G) >= sms()) G *= 2;
    P.G = G;
    P.logG = ilog2(G);
    if (axis == 0) {
        P.groups = lines / G;
    } else {
        P.per_outer = (P.Q + G - 1) / G;
        P.groups = P.per_outer * (lines / P.Q);
    }
    P.tw = A.tw[axis];
    P.Cu = A.Cu;
    P.Cx = A.Cx;
    for (int i = 0; i < 4; ++i) P.r[i] = T(A.r[i]);
    // lines that come back to real space: 1/n of every axis transformed back, and the 1/2 of split()
    T all = T(0.5);
    for (int m = 0; m < A.dim; ++m) all /= T(A.n[m]);
    for (int m = 0; m < 3; ++m) P.sc[m] = all;
    if (mode == PM_FLUX) {                                // D_mu u: axes 1 and 2..mu
        P.sc[0] = T(0.5) / T(A.n[0]);
        for (int m = 1; m < A.dim; ++m) P.sc[m] = P.sc[m - 1] / T(A.n[m]);
    }
    P.adelta = A.adelta ? 1 : 0;
    P.dif = A.dif;
    return P;
}

template <typename T, int MODE>
cudaError_t launch_pass_on(const Pass<T>& P, cudaStream_t st) {
    const size_t smem = pass_smem(P.n, P.G, P.pitch, P.nb, sizeof(Cplx<T>));
    // two threads per radix-4 butterfly: the loads, stores and pointwise work between the transforms take them all
    const int work = std::max(P.nb * P.G * ((1 << P.llen) >> 1), 1);
    const int threads = std::min(kPassThreads, (work + 31) / 32 * 32);
    const long long grid = std::min<long long>(P.groups, 64LL * sms());
    fourier_pass_kernel<T, MODE><<<unsigned(grid), threads, smem, st>>>(P);
    return cudaGetLastError();
}

template <typename T>
cudaError_t prepare_impl() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void* f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kPassSmemMax));
    };
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_FWD_REAL>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_PLAIN>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_PIVOT_MULT>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_FINAL_AXPY>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_DERIV>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_MID_DIV>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_FLUX>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_PIVOT_DIV>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_FINAL_OUT>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_PIVOT_STAGE>));
    set(reinterpret_cast<const void*>(fourier_pass_kernel<T, PM_FINAL_FWD>));
    sms();
    return e;
}

// The x2 pass of a 3-D grid on na arrays.
template <typename T>
cudaError_t middle_pass(const PeriodicArgs<T>& A, Cplx<T>* const* arrays, int na, int inverse, cudaStream_t st) {
    if (A.dim != 3) return cudaSuccess;
    Pass<T> P = make_pass(A, 1, PM_PLAIN);
    for (int a = 0; a < na; ++a) P.C[a] = arrays[a];
    P.na = na;
    P.inverse = inverse;
    return launch_pass_on<T, PM_PLAIN>(P, st);
}

// Cx = F_1 u (unless it is there already), u^ and the derivatives' lines ready for the flux pass.
template <typename T>
cudaError_t derivatives(const PeriodicArgs<T>& A, const T* u, bool have_cx, cudaStream_t st) {
    cudaError_t e;
    if (!have_cx) {
        Pass<T> P = make_pass(A, 0, PM_FWD_REAL);
        P.x = u;
        P.C[0] = A.Cx;
        if ((e = launch_pass_on<T, PM_FWD_REAL>(P, st)) != cudaSuccess) return e;
    }
    for (int axis = 1; axis < A.dim; ++axis) {
        Pass<T> P = make_pass(A, axis, PM_DERIV);
        P.src = axis == 1 ? A.Cx : A.Cu;
        if ((e = launch_pass_on<T, PM_DERIV>(P, st)) != cudaSuccess) return e;
    }
    Cplx<T>* d3[1] = {A.C[2]};
    return middle_pass(A, d3, 1, 1, st);
}

template <typename T>
cudaError_t rhs_impl(const PeriodicArgs<T>& A, const StencilArgs<T>& s, cudaStream_t st) {
    if (s.nout < 1 || s.nout > kMaxOut || s.nout > A.dim || s.nx < 0 || s.nx > kMaxExtra || !s.u)
        return cudaErrorInvalidValue;
    const int last = A.dim - 1;
    cudaError_t e;
    if ((e = derivatives(A, s.u, false, st)) != cudaSuccess) return e;
    {   // fluxes, forward along x1
        Pass<T> P = make_pass(A, 0, PM_FLUX);
        P.x = s.u;
        if ((e = launch_pass_on<T, PM_FLUX>(P, st)) != cudaSuccess) return e;
    }
    if (A.dim == 3) {
        Pass<T> P = make_pass(A, 1, PM_MID_DIV);
        if ((e = launch_pass_on<T, PM_MID_DIV>(P, st)) != cudaSuccess) return e;
    }
    {   // divergence and the stage outputs in Fourier space, back along the pivot axis
        Pass<T> P = make_pass(A, last, PM_PIVOT_DIV);
        P.M = A.sym;
        P.nout = s.nout;
        for (int j = 0; j < s.nout; ++j) {
            P.cgF[j] = T(s.cg[j] + s.cF[j]);
            P.cg[j] = T(s.cg[j]);
        }
        if ((e = launch_pass_on<T, PM_PIVOT_DIV>(P, st)) != cudaSuccess) return e;
    }
    if ((e = middle_pass(A, A.C, s.nout, 1, st)) != cudaSuccess) return e;
    {   // stage outputs in real space
        Pass<T> P = make_pass(A, 0, PM_FINAL_OUT);
        P.x = s.u;
        P.nout = s.nout;
        P.nx = s.nx;
        for (int x = 0; x < kMaxExtra; ++x) P.X[x] = s.X[x];
        for (int j = 0; j < s.nout; ++j) {
            P.out[j] = s.out[j];
            P.cgF[j] = T(s.cg[j] + s.cF[j]);
            state_coefs<T>(s.cu[j], s.cx[j], P.cu[j], P.cx[j]);
        }
        if ((e = launch_pass_on<T, PM_FINAL_OUT>(P, st)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t multiplier_impl(const PeriodicArgs<T>& A, const Cplx<T>* M, const T* x, T* y, const T* base, double alpha,
                            cudaStream_t st) {
    if (!M || !x || !y) return cudaErrorInvalidValue;
    const int last = A.dim - 1;
    cudaError_t e;
    {
        Pass<T> P = make_pass(A, 0, PM_FWD_REAL);
        P.x = x;
        if ((e = launch_pass_on<T, PM_FWD_REAL>(P, st)) != cudaSuccess) return e;
    }
    Cplx<T>* c0[1] = {A.C[0]};
    if ((e = middle_pass(A, c0, 1, 0, st)) != cudaSuccess) return e;
    {
        Pass<T> P = make_pass(A, last, PM_PIVOT_MULT);
        P.M = M;
        if ((e = launch_pass_on<T, PM_PIVOT_MULT>(P, st)) != cudaSuccess) return e;
    }
    if ((e = middle_pass(A, c0, 1, 1, st)) != cudaSuccess) return e;
    {
        Pass<T> P = make_pass(A, 0, PM_FINAL_AXPY);
        P.y = y;
        P.base = base;
        P.alpha = T(alpha);
        if ((e = launch_pass_on<T, PM_FINAL_AXPY>(P, st)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// One fused stage of a 2-D periodic context, kept in Fourier space from the state's transform to
// the stage's result: y = F^-1 (Mu (cu u^) + Mg (cgF F(u)^ ... ) + cz Z), see
// PeriodicStage. Five launches: x1 forward of u | pivot: u^ and i k_2 u^ back | x1: fluxes and
// the pointwise part forward | pivot: the combination and its multipliers, back | x1 inverse.
template <typename T>
cudaError_t stage_impl(const PeriodicArgs<T>& A, const PeriodicStage<T>& s, cudaStream_t st) {
    if (A.dim != 2 || !s.x || !s.y) return cudaErrorInvalidValue;
    cudaError_t e;
    // take_over: the previous stage's last pass left F_1 x in Cx
    if ((e = derivatives(A, s.x, s.take_over, st)) != cudaSuccess) return e;
    {
        Pass<T> P = make_pass(A, 0, PM_FLUX, true);
        P.x = s.x;
        if ((e = launch_pass_on<T, PM_FLUX>(P, st)) != cudaSuccess) return e;
    }
    {
        Pass<T> P = make_pass(A, 1, PM_PIVOT_STAGE);
        P.M = A.sym;
        P.Mu = s.Mu;
        P.Mg = s.Mg;
        P.Ms = s.Ms;
        P.Z = s.Z;
        P.Zs = s.Zs;
        P.scu = T(s.cu);
        P.scgF = T(s.cgF);
        P.scg = T(s.cg);
        P.scgz = T(s.cgz);
        P.scz = T(s.cz);
        P.szu = T(s.zu);
        P.szF = T(s.zF);
        P.szg = T(s.zg);
        if ((e = launch_pass_on<T, PM_PIVOT_STAGE>(P, st)) != cudaSuccess) return e;
    }
    if (s.hand_on) {
        Pass<T> P = make_pass(A, 0, PM_FINAL_FWD);
        P.y = s.y;
        if ((e = launch_pass_on<T, PM_FINAL_FWD>(P, st)) != cudaSuccess) return e;
    } else {
        Pass<T> P = make_pass(A, 0, PM_FINAL_AXPY);
        P.y = s.y;
        P.base = nullptr;
        if ((e = launch_pass_on<T, PM_FINAL_AXPY>(P, st)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

int periodic_stage_launches(int dim, bool take_over) { return dim == 2 ? (take_over ? 4 : 5) : 0; }
cudaError_t launch_periodic_stage(const PeriodicArgs<double>& P, const PeriodicStage<double>& s, cudaStream_t st) {
    return stage_impl(P, s, st);
}
cudaError_t launch_periodic_stage(const PeriodicArgs<float>& P, const PeriodicStage<float>& s, cudaStream_t st) {
    return stage_impl(P, s, st);
}

cudaError_t periodic_prepare(bool fp64) { return fp64 ? prepare_impl<double>() : prepare_impl<float>(); }

bool periodic_line_fits(int n, int axis, int dim, bool fp64) {
    const int arrays = axis == 0 ? 1 : axis == dim - 1 ? 2 : 3;   // the most lines a pass on that axis holds
    const int pitch = axis == 0 ? n / 2 : n + 1;
    return pass_smem(n, 1, pitch, arrays, fp64 ? sizeof(Cplx<double>) : sizeof(Cplx<float>)) <= kPassSmemMax;
}

int periodic_rhs_launches(int dim, int nout) { (void)nout; return 5 + 4 * (dim - 2); }
int periodic_multiplier_launches(int dim) { return 3 + 2 * (dim - 2); }

cudaError_t launch_periodic_rhs(const PeriodicArgs<double>& P, const StencilArgs<double>& s, cudaStream_t st) {
    return rhs_impl(P, s, st);
}
cudaError_t launch_periodic_rhs(const PeriodicArgs<float>& P, const StencilArgs<float>& s, cudaStream_t st) {
    return rhs_impl(P, s, st);
}
cudaError_t launch_periodic_multiplier(const PeriodicArgs<double>& P, const Cplx<double>* M, const double* x, double* y,
                                       const double* base, double alpha, cudaStream_t st) {
    return multiplier_impl(P, M, x, y, base, alpha, st);
}
cudaError_t launch_periodic_multiplier(const PeriodicArgs<float>& P, const Cplx<float>* M, const float* x, float* y,
                                       const float* base, double alpha, cudaStream_t st) {
    return multiplier_impl(P, M, x, y, base, alpha, st);
}

}  // namespace adr
