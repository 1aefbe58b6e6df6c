// K1 in FP64 (Eq. (nonlin), Section 3; see stencil.cu for the discretisation): every grid form, 2-D and
// 3-D, Dirichlet or Neumann faces, flux or a Lap u form.
//
// What bounds it. The FP64 pipe: 2 instructions' lanes per clock and SM, so one FP64 instruction per
// node costs as much time as 12 bytes of HBM traffic. The kernel therefore trades memory for
// instructions: the face weights w_mu = (1/2h^2) ((a - abar)_i + (a - abar)_{i+e}) are stored (three arrays
// beside u instead of one: 24 bytes more a node, 6 additions and 9 multiplications less), differences
// are formed once per face and shared (pairs along x1 in a thread, planes along x3 in
// registers), and terms whose coefficient is zero are left out by branches that every thread takes alike.
// Per node and direction: d+ (shared), two FMAs with the face weights; M = u+ - u- and one FMA
// where b - beta is not zero; for F, L = d+ - d- and one FMA with abar / h^2, and one FMA of M with beta / (2h).
// u + tau/2 g in 3-D: 15.6 FP64 instructions a node instead of about 75; F and g: 32 instead of 85 (ncu).
// Time of a launch, per-node kernel -> this one (us): 256^3 2139 -> 504 (one output), 2460 -> 607 and 692 (two outputs, one and two
// stage inputs); 128^3 F and g 379 -> 142, g - G0 283 -> 66; 60^3 Neumann, a Lap u form 39 -> 17; 32^2 12.6 -> 7.3. The FP64 pipe
// is then 86 to 90% busy.
#include <cuda_runtime.h>

#include <type_traits>

#include "adr_internal.h"
#include "launch.cuh"
#include "stencil_core.cuh"

namespace adr {
namespace {

constexpr int kTX = 32, kTY = 8;         // threads of a block along x1 (V nodes each), the most along x2

// Folded per-direction weights.
struct Weights {
    double w2[3];                        // (b - beta) / (2h)
    double wa[3], wb[3];                 // abar / h^2, beta / (2h)
    double ih2[3], hih2[3];              // 1 / h^2, and half of it
    const double* face[3];               // face weights, laid out as StencilArgs::a (NULL: a = abar everywhere, or NODAL)
    // which terms there are: tested as integers, since a comparison of doubles costs an FP64 instruction
    bool adv;                            // a w2, or a wb that F takes, is not zero
    int start[kMaxOut];                  // a term of coefficient one: 1 u, 2 g, 3 F, 4 + e X_e; 0 none
    unsigned terms[kMaxOut];             // the other terms that are not zero: bits kTu, kTg, kTF, kTx + e
};
constexpr unsigned kTu = 0, kTg = 1, kTF = 2, kTx = 3;

template <int V>
__device__ __forceinline__ void ldv(const double* p, double (&v)[V]) {
    if constexpr (V == 2) {
        const double2 t = __ldg(reinterpret_cast<const double2*>(p));
        v[0] = t.x;
        v[1] = t.y;
    } else {
        v[0] = __ldg(p);
    }
}
template <int V>
__device__ __forceinline__ void stv(double* p, const double (&v)[V]) {
    if constexpr (V == 2) *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    else *p = v[0];
}

// A thread owns V consecutive x1 nodes of one row and walks zb planes of x3; u of the planes z - 1 and z
// and the face weights below plane z stay in registers, the neighbours along x1 and x2 come from L1.
// ADV: any first-derivative term; NX: stage inputs; UT: whether an output takes a multiple of u. An instruction under a false predicate still takes its turn on the
// FP64 pipe, and the compiler turns short branches into predicates, so what decides about few instructions is a
// template argument. NODAL: the face weights formed here from the nodal array, to the same bits, for contexts that had no
// memory for them (256^3, one output: 506 -> 1090 us).
template <int DIM, int V, bool ADELTA, bool NEEDF, bool ADV, int NX, bool UT, bool NODAL = false>
__global__ void __launch_bounds__(kTX * kTY) stencil_f64_kernel(StencilArgs<double> p, Coefs<double> c, Weights w, int zb) {
    const int n1 = p.n1, n2 = p.n2, n3 = DIM == 3 ? p.n3 : 1;
    const int i1 = (int(blockIdx.x) * kTX + int(threadIdx.x % kTX)) * V;
    const int i2 = int(blockIdx.y) * int(blockDim.x / kTX) + int(threadIdx.x / kTX);
    pdl_trigger();
    if (i1 >= n1 || i2 >= n2) return;                        // V = 2: n1 is even
    const long long plane_u = (long long)n1 * n2, plane_a = (long long)p.apitch * (n2 + 2);
    const int z0 = DIM == 3 ? int(blockIdx.z) * zb : 0, z1 = DIM == 3 ? min(z0 + zb, n3) : 1;
    const double* u = p.u + (long long)i2 * n1 + i1 + z0 * plane_u;
    const long long ao = (long long)(i2 + 1) * p.apitch + (i1 + 4) + (DIM == 3 ? (z0 + 1) * plane_a : 0);
    const double* aC = (ADELTA || NODAL) && p.a ? p.a + ao : nullptr;
    const bool faces = NODAL || (!ADELTA && w.face[0]);
    const double* f1 = faces && !NODAL ? w.face[0] + ao : nullptr;
    const double* f2 = faces && !NODAL ? w.face[1] + ao : nullptr;
    const double* f3 = faces && !NODAL && DIM == 3 ? w.face[2] + ao : nullptr;

    double uM[V], uC[V], dM[V], fM[V];
    ldv<V>(u, uC);
#pragma unroll
    for (int k = 0; k < V; ++k) uM[k] = fM[k] = 0.0;
    if (DIM == 3) {
        if (z0 > 0) ldv<V>(u - plane_u, uM);
        if (NODAL) {
            double aM[V];
            ldv<V>(aC - plane_a, aM);
            ldv<V>(aC, fM);
#pragma unroll
            for (int k = 0; k < V; ++k) fM[k] = w.hih2[2] * (aM[k] + fM[k]);
        } else if (faces) {
            ldv<V>(f3 - plane_a, fM);
        }
#pragma unroll
        for (int k = 0; k < V; ++k) dM[k] = uC[k] - uM[k];
    }
    long long idx = (long long)i2 * n1 + i1 + z0 * plane_u;
    for (int z = z0; z < z1; ++z) {
        double uP[V], uS[V], uN[V], fS[V], fN[V], fE[V], fP[V], a0[V], x[NX > 0 ? NX : 1][V];
        double uW = 0.0, uE = 0.0, fW = 0.0;
#pragma unroll
        for (int k = 0; k < V; ++k) uP[k] = uS[k] = uN[k] = 0.0;
        if (DIM == 3) {
            if (z + 1 < n3) ldv<V>(u + plane_u, uP);
            else if (p.neumann) {                            // Neumann face: the ghost mirrors plane n3 - 2
#pragma unroll
                for (int k = 0; k < V; ++k) uP[k] = uM[k];
            }
        }
        if (i2 > 0) ldv<V>(u - n1, uS);
        if (i2 + 1 < n2) ldv<V>(u + n1, uN);
        else if (p.neumann) {
#pragma unroll
            for (int k = 0; k < V; ++k) uN[k] = uS[k];
        }
        if (i1 > 0) uW = __ldg(u - 1);
        if (i1 + V < n1) uE = __ldg(u + V);
        else if (p.neumann) uE = V == 2 ? uC[0] : uW;
        if (NODAL) {
            double ac[V];
            ldv<V>(aC, ac);
            ldv<V>(aC - p.apitch, fS);
            ldv<V>(aC + p.apitch, fN);
            const double ae = __ldg(aC + V);
            fW = w.hih2[0] * (__ldg(aC - 1) + ac[0]);
            if (DIM == 3) ldv<V>(aC + plane_a, fP);
#pragma unroll
            for (int k = 0; k < V; ++k) {
                fE[k] = w.hih2[0] * (ac[k] + (k + 1 < V ? ac[V - 1] : ae));
                fS[k] = w.hih2[1] * (fS[k] + ac[k]);
                fN[k] = w.hih2[1] * (ac[k] + fN[k]);
                if (DIM == 3) fP[k] = w.hih2[2] * (ac[k] + fP[k]);
            }
        } else if (faces) {
            fW = __ldg(f1 - 1);
            ldv<V>(f1, fE);
            ldv<V>(f2 - p.apitch, fS);
            ldv<V>(f2, fN);
            if (DIM == 3) ldv<V>(f3, fP);
        }
        if (ADELTA && aC) ldv<V>(aC, a0);
#pragma unroll
        for (int e = 0; e < NX; ++e) ldv<V>(p.X[e] + idx, x[e]);

        double g[V], au[V], F[V];                            // g, A u, F = g + A u
        double dW = uC[0] - uW;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const double uk = uC[k], ue = k + 1 < V ? uC[V - 1] : uE;
            const double dE = ue - uk, dN = uN[k] - uk, dS = uk - uS[k];
            const double dP = DIM == 3 ? uP[k] - uk : 0.0;
            double r = fma(uk, fma(uk, fma(uk, c.r3, c.r2), c.r1), c.r0);
            double l1 = 0.0, l2 = 0.0, l3 = 0.0;             // second differences
            if (ADELTA || NEEDF) {
                l1 = dE - dW;
                l2 = dN - dS;
                if (DIM == 3) l3 = dP - dM[k];
            }
            if (NEEDF) {
                au[k] = fma(w.wa[1], l2, w.wa[0] * l1);
                if (DIM == 3) au[k] = fma(w.wa[2], l3, au[k]);
            }
            if (!ADELTA && faces) {
                r = fma(fE[k], dE, r);
                r = fma(-(k ? fE[0] : fW), dW, r);
                r = fma(fN[k], dN, r);
                r = fma(-fS[k], dS, r);
                if (DIM == 3) {
                    r = fma(fP[k], dP, r);
                    r = fma(-fM[k], dM[k], r);
                }
            }
            if (ADELTA && aC) {
                double s = w.ih2[0] * l1;
                s = fma(w.ih2[1], l2, s);
                if (DIM == 3) s = fma(w.ih2[2], l3, s);
                r = fma(a0[k], s, r);
            }
            g[k] = r;
            if (DIM == 3) dM[k] = dP;
            dW = dE;
        }
        // centred differences, where a term takes them
#pragma unroll
        for (int m = 0; m < (ADV ? DIM : 0); ++m) {
            double md[V];
#pragma unroll
            for (int k = 0; k < V; ++k)
                md[k] = m == 0 ? (k + 1 < V ? uC[V - 1] : uE) - (k ? uC[0] : uW) : m == 1 ? uN[k] - uS[k] : uP[k] - uM[k];
#pragma unroll
            for (int k = 0; k < V; ++k) {
                g[k] = fma(w.w2[m], md[k], g[k]);
                if (NEEDF) au[k] = fma(w.wb[m], md[k], au[k]);
            }
        }
        if (NEEDF) {
#pragma unroll
            for (int k = 0; k < V; ++k) F[k] = g[k] + au[k];
        }
        double res[kMaxOut][V];
#pragma unroll
        for (int j = 0; j < kMaxOut; ++j) {
            if (j >= p.nout) continue;
            const unsigned tm = w.terms[j];
            const int st = w.start[j];
#pragma unroll
            for (int k = 0; k < V; ++k) {
                double v = st == 1 ? uC[k] : st == 2 ? g[k] : NEEDF && st == 3 ? F[k] : 0.0;
#pragma unroll
                for (int e = 0; e < NX; ++e)
                    if (st == 4 + e) v = x[e][k];
                if (UT && (tm & (1u << kTu))) v = fma(c.cu[j], uC[k], v);
                if (tm & (1u << kTg)) v = fma(c.cg[j], g[k], v);
                if (NEEDF && (tm & (1u << kTF))) v = fma(c.cF[j], F[k], v);
#pragma unroll
                for (int e = 0; e < NX; ++e)
                    if (tm & (1u << (kTx + e))) v = fma(c.cx[j][e], x[e][k], v);
                res[j][k] = v;
            }
        }
#pragma unroll
        for (int j = 0; j < kMaxOut; ++j)
            if (j < p.nout) stv<V>(p.out[j] + idx, res[j]);
        if (DIM == 3) {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                uM[k] = uC[k];
                uC[k] = uP[k];
                fM[k] = fP[k];
            }
            u += plane_u;
            idx += plane_u;
            if (faces && !NODAL) { f1 += plane_a; f2 += plane_a; f3 += plane_a; }
            if ((ADELTA || NODAL) && aC) aC += plane_a;
        }
    }
}

// w_mu at every node that has a next one along mu, from the nodal (a - abar).
__global__ void f64_faces_kernel(const double* a, double* w, double half_ih2, long long next, long long total) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i + next < total; i += (long long)gridDim.x * blockDim.x)
        w[i] = half_ih2 * (a[i] + a[i + next]);
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

template <int DIM, int V>
cudaError_t launch_v(const StencilArgs<double>& p, const Coefs<double>& c, const Weights& w, bool needF, cudaStream_t s) {
    const int gx = (p.n1 + kTX * V - 1) / (kTX * V), sms = sm_count();
    int ty = kTY, zb = 1;
    if (DIM == 3) {
        // planes a block walks: about eight blocks per SM in all, and no fewer than 2 planes
        // (each block loads the plane below its first one)
        const int want = (8 * sms + gx * ((p.n2 + ty - 1) / ty) - 1) / (gx * ((p.n2 + ty - 1) / ty));
        zb = p.n3 / (want < 1 ? 1 : want);
        zb = zb < 2 ? 2 : zb > 32 ? 32 : zb;
    }
    const int gz = DIM == 3 ? (p.n3 + zb - 1) / zb : 1;
    // small grids: a block on every SM (32^2 in four blocks of 8 rows: 14.8 us instead of 7.0)
    while (ty > 1 && gx * ((p.n2 + ty - 1) / ty) * gz < 2 * sms) ty /= 2;
    const dim3 grid(gx, (p.n2 + ty - 1) / ty, gz);
    const int threads = kTX * ty;
    const bool nodal = !p.adelta && p.a && !w.face[0];       // has every term
    auto go = [&](auto adelta, auto f, auto adv) {
        constexpr bool AD = decltype(adelta)::value, NF = decltype(f)::value, AV = decltype(adv)::value;
        if constexpr (!AD && AV) {
            if (nodal) {
                stencil_f64_kernel<DIM, V, false, NF, true, kMaxExtra, true, true><<<grid, threads, 0, s>>>(p, c, w, zb);
                return;
            }
        }
        // odd rows and 2-D grids take the form that has every term
        if constexpr (DIM == 2 || V == 1) {
            stencil_f64_kernel<DIM, V, AD, NF, AV, kMaxExtra, true><<<grid, threads, 0, s>>>(p, c, w, zb);
        } else {
            bool ut = false;
            for (int j = 0; j < p.nout; ++j) ut = ut || (w.terms[j] & (1u << kTu));
            switch (p.nx * 2 + (ut ? 1 : 0)) {
            case 0: stencil_f64_kernel<DIM, V, AD, NF, AV, 0, false><<<grid, threads, 0, s>>>(p, c, w, zb); break;
            case 1: stencil_f64_kernel<DIM, V, AD, NF, AV, 0, true><<<grid, threads, 0, s>>>(p, c, w, zb); break;
            case 2: stencil_f64_kernel<DIM, V, AD, NF, AV, 1, false><<<grid, threads, 0, s>>>(p, c, w, zb); break;
            case 3: stencil_f64_kernel<DIM, V, AD, NF, AV, 1, true><<<grid, threads, 0, s>>>(p, c, w, zb); break;
            case 4: stencil_f64_kernel<DIM, V, AD, NF, AV, 2, false><<<grid, threads, 0, s>>>(p, c, w, zb); break;
            default: stencil_f64_kernel<DIM, V, AD, NF, AV, kMaxExtra, true><<<grid, threads, 0, s>>>(p, c, w, zb); break;
            }
        }
    };
    using Yes = std::integral_constant<bool, true>;
    using No = std::integral_constant<bool, false>;
    auto with_adv = [&](auto adelta, auto f) { w.adv || nodal ? go(adelta, f, Yes{}) : go(adelta, f, No{}); };
    if (p.adelta) needF ? with_adv(Yes{}, Yes{}) : with_adv(Yes{}, No{});
    else          needF ? with_adv(No{}, Yes{}) : with_adv(No{}, No{});
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_f64_faces(const double* a, double* w, double inv_h2, long long next, long long total, cudaStream_t s) {
    const long long blocks = (total + 255) / 256;
    f64_faces_kernel<<<unsigned(blocks < 65535 ? blocks : 65535), 256, 0, s>>>(a, w, 0.5 * inv_h2, next, total);
    return cudaGetLastError();
}

cudaError_t launch_stencil(const StencilArgs<double>& p, cudaStream_t s) {
    if (p.nout < 1 || p.nout > kMaxOut || p.nx < 0 || p.nx > kMaxExtra) return cudaErrorInvalidValue;
    Coefs<double> c{};
    Weights w{};
    for (int m = 0; m < p.dim; ++m) {
        w.w2[m] = p.bmb[m] * p.inv_2h[m];
        w.wa[m] = p.abar * p.inv_h2[m];
        w.wb[m] = p.beta[m] * p.inv_2h[m];
        w.ih2[m] = p.inv_h2[m];
        w.hih2[m] = 0.5 * p.inv_h2[m];
        w.face[m] = p.face[m];
    }
    c.r0 = p.r[0]; c.r1 = p.r[1]; c.r2 = p.r[2]; c.r3 = p.r[3];
    bool needF = false;
    for (int j = 0; j < kMaxOut; ++j) {
        c.cg[j] = p.cg[j];
        c.cF[j] = p.cF[j];
        state_coefs<double>(p.cu[j], p.cx[j], c.cu[j], c.cx[j]);
        if (j >= p.nout) continue;
        if (p.cF[j] != 0.0) needF = true;
        w.start[j] = c.cu[j] == 1.0 ? 1 : c.cg[j] == 1.0 ? 2 : c.cF[j] == 1.0 ? 3 : 0;
        for (int e = 0; e < p.nx; ++e)
            if (!w.start[j] && c.cx[j][e] == 1.0) w.start[j] = 4 + e;
        if (c.cu[j] != 0.0 && w.start[j] != 1) w.terms[j] |= 1u << kTu;
        if (c.cg[j] != 0.0 && w.start[j] != 2) w.terms[j] |= 1u << kTg;
        if (c.cF[j] != 0.0 && w.start[j] != 3) w.terms[j] |= 1u << kTF;
        for (int e = 0; e < p.nx; ++e)
            if (c.cx[j][e] != 0.0 && w.start[j] != 4 + e) w.terms[j] |= 1u << (kTx + e);
    }
    for (int m = 0; m < p.dim; ++m) {
        if (w.w2[m] != 0.0 || (needF && w.wb[m] != 0.0)) w.adv = true;
    }
    // inputs that are not there (forms with more of them than p.nx) are read as u, with no term
    StencilArgs<double> q = p;
    for (int e = p.nx; e < kMaxExtra; ++e) q.X[e] = p.u;
    // two nodes a thread where every row starts on 16 bytes and fills a warp
    auto al = [](const void* q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    bool pairs = p.n1 % 2 == 0 && p.n1 >= 2 * kTX && al(p.u);
    for (int e = 0; e < p.nx; ++e) pairs = pairs && al(p.X[e]);
    for (int j = 0; j < p.nout; ++j) pairs = pairs && al(p.out[j]);
    if (p.dim == 3) return pairs ? launch_v<3, 2>(q, c, w, needF, s) : launch_v<3, 1>(q, c, w, needF, s);
    return pairs ? launch_v<2, 2>(q, c, w, needF, s) : launch_v<2, 1>(q, c, w, needF, s);
}

}  // namespace adr
