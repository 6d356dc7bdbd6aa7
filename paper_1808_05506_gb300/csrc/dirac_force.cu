// Link gradient of L = Re <g, D psi> = Re sum_x g(x)^+ (D psi)(x) for the
// operators that couple through single links, with PyTorch's convention for
// a real loss of complex variables, F = dL/dRe V + i dL/dIm V.  A term
// Re tr(V M) of L contributes M^+ to F and a term Re tr(V^+ M) contributes M.
//   Wilson (Sec. 4, def_wils; V_mu(x) enters the forward hop from x and the
//   backward hop from x+mu):
//     F_mu(x) = -1/2 sum_v sum_s [(1 - gamma_mu) g_v(x)]_s psi_v(x+mu)_s^+
//               -1/2 sum_v sum_s psi_v(x)_s [(1 + gamma_mu) g_v(x+mu)]_s^+
//     Each spin sum runs over the two components of the rank-2 projection:
//     sum_s [(1 + S gamma) a]_s b_s^+ = sum_{c=0,1} h_c k_c^+ with
//     h = a_up + S B a_down, k = b_up + S B b_down.
//   staggered (Sec. 3; eta_mu(x + mu) = eta_mu(x)):
//     F_mu(x) = 1/2 eta_mu(x) sum_v [g_v(x) psi_v(x+mu)^+ - psi_v(x) g_v(x+mu)^+]
// One thread owns NM links of one site, gathers both hops that touch each and
// writes it once (no atomics).  The Brillouin gradient, through the composite
// transporters W, is in dirac_force_brillouin.cu.
#include "dirac_handle.h"
#include "dirac_kernels.cuh"

using namespace dirac;

namespace dirac {

// t[a][b] += sum_{comp} u_comp[a] conj(w_comp[b]) for NC 3-vectors
template <int NC, typename A>
__device__ __forceinline__ void outer_products(cx<A>* t, const cx<A>* u, const cx<A>* w)
{
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) t[3 * a + b] = cfma_conj(w[3 * k + b], u[3 * k + a], t[3 * a + b]);
}

// acc += f (u w^+ + u2 w2^+), the two hops of a link with NC components each.  f joins
// each sum, not the end of it, which could leave the range where the result does
// not.  What is summed by itself first, by what rounds least: both hops, or
// (SINGLE) each component.  FP64 takes SINGLE: a sum of both hops, or straight into
// acc, saves a third of its operations and puts the staggered force of one right-hand side
// 8.8e-17 instead of 4.7e-17 from the exact one.  FP32 sums both hops (16 right-hand
// sides: Wilson 1.0e-7 instead of 1.6e-7, staggered 8.7e-8 instead of 1.1e-7), except
// Wilson with one right-hand side, where there is no longer sum to keep short (6.6e-8
// and 6.4e-8).
template <int NC, bool SINGLE, typename A>
__device__ __forceinline__ void outer_sum(cx<A>* acc, A f, const cx<A>* u, const cx<A>* w, const cx<A>* u2, const cx<A>* w2)
{
    cx<A> t[9];
    auto clear = [&]() {
#pragma unroll
        for (int e = 0; e < 9; ++e) t[e] = cx<A>{A(0), A(0)};
    };
    auto join = [&]() {
#pragma unroll
        for (int e = 0; e < 9; ++e) acc[e] = cx<A>{fma(f, t[e].re, acc[e].re), fma(f, t[e].im, acc[e].im)};
    };
    if constexpr (SINGLE) {
#pragma unroll
        for (int k = 0; k < 2 * NC; ++k) {
            clear();
            outer_products<1>(t, k < NC ? u + 3 * k : u2 + 3 * (k - NC), k < NC ? w + 3 * k : w2 + 3 * (k - NC));
            join();
        }
    } else {
        clear();
        outer_products<NC>(t, u, w);
        outer_products<NC>(t, u2, w2);
        join();
    }
}

template <int MU, bool SINGLE, typename A>
__device__ __forceinline__ void wilson_force_hop(cx<A>* acc, const cx<A>* gs, const cx<A>* ps, const cx<A>* gn, const cx<A>* pn)
{
    cx<A> h[6], k[6], h2[6], k2[6];
    wilson_project<MU, -1>(gs, h);
    wilson_project<MU, -1>(pn, k);
    wilson_project<MU, +1>(ps, k2);
    wilson_project<MU, +1>(gn, h2);
    outer_sum<2, SINGLE>(acc, A(-0.5), h, k, k2, h2);
}

// The links mu = m0 .. m0 + NM - 1 of site s.  The four links of a site share
// psi(x) and g(x): NM links in a thread load 2 + 2 NM spinors per right-hand
// side instead of 4 NM.  FP32 and 16-bit: bound by those loads, which come from
// L2 (16 a site at NM = 1; 16^4, Nv = 8, FP32 Wilson: NM = 1 64 us, 4 44).  FP64: bound by
// FP64 arithmetic, 108 operations per link, right-hand side and pair of 3-vectors
// (16^4, Nv = 8: staggered 406 us, Wilson 1052).
template <typename T, int M0, int NM, bool SINGLE>
__device__ __forceinline__ void wilson_force_links(const Geom& g, int Nv, const void* psi, const void* gv, long s,
                                                   const long* fwd, cx<typename Store<T>::A> (&acc)[NM][9])
{
    using A = typename Store<T>::A;
    for (int v = 0; v < Nv; ++v) {
        cx<A> gs[12], ps[12], gn[12], pn[12];
        load_spinor<T, 12>(gv, g.vol, v, s, gs);
        load_spinor<T, 12>(psi, g.vol, v, s, ps);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            load_spinor<T, 12>(gv, g.vol, v, s + fwd[M0 + m], gn);
            load_spinor<T, 12>(psi, g.vol, v, s + fwd[M0 + m], pn);
            if (M0 + m == 0) wilson_force_hop<0, SINGLE>(acc[m], gs, ps, gn, pn);
            else if (M0 + m == 1) wilson_force_hop<1, SINGLE>(acc[m], gs, ps, gn, pn);
            else if (M0 + m == 2) wilson_force_hop<2, SINGLE>(acc[m], gs, ps, gn, pn);
            else wilson_force_hop<3, SINGLE>(acc[m], gs, ps, gn, pn);
        }
    }
}

template <typename T, bool STAG, int NM, bool SINGLE>
__global__ void __launch_bounds__(128) k_force(Geom g, int Nv, const void* psi, const void* gv, void* F)
{
    using A = typename Store<T>::A;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (links of a site, site), site fastest
    if (i >= (4 / NM) * g.vol) return;
    const int q = (int)(i / g.vol), m0 = q * NM;
    const long s = i - q * g.vol;
    long fwd[4], bwd[4];
    int x[4];
    site_offsets(g, s, fwd, bwd, x);
    cx<A> acc[NM][9];
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int e = 0; e < 9; ++e) acc[m][e] = cx<A>{A(0), A(0)};
    if constexpr (STAG) {
        A f[NM];
        long sp[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int mu = m0 + m;
            const int par = (mu > 0 ? x[0] : 0) + (mu > 1 ? x[1] : 0) + (mu > 2 ? x[2] : 0);
            f[m] = (par & 1) ? A(-0.5) : A(0.5);
            sp[m] = s + (mu == 0 ? fwd[0] : (mu == 1 ? fwd[1] : (mu == 2 ? fwd[2] : fwd[3])));
        }
        for (int v = 0; v < Nv; ++v) {
            cx<A> gs[3], ps[3], gn[3], pn[3];
            load_spinor<T, 3>(gv, g.vol, v, s, gs);
            load_spinor<T, 3>(psi, g.vol, v, s, ps);
#pragma unroll
            for (int c = 0; c < 3; ++c) ps[c] = -ps[c];
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                load_spinor<T, 3>(gv, g.vol, v, sp[m], gn);
                load_spinor<T, 3>(psi, g.vol, v, sp[m], pn);
                outer_sum<1, SINGLE>(acc[m], f[m], gs, pn, ps, gn);
            }
        }
    } else {
        if constexpr (NM == 4) wilson_force_links<T, 0, 4, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
        else if constexpr (NM == 2) {
            if (q == 0) wilson_force_links<T, 0, 2, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
            else wilson_force_links<T, 2, 2, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
        } else {
            if (q == 0) wilson_force_links<T, 0, 1, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
            else if (q == 1) wilson_force_links<T, 1, 1, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
            else if (q == 2) wilson_force_links<T, 2, 1, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
            else wilson_force_links<T, 3, 1, SINGLE>(g, Nv, psi, gv, s, fwd, acc);
        }
    }
    if constexpr (sizeof(A) == 4 && NM > 1) {
        // the NM links of a site are 72 NM contiguous bytes, 16-byte aligned for even NM
        float4* out = reinterpret_cast<float4*>(static_cast<float2*>(F) + ((size_t)s * 4 + m0) * 9);
#pragma unroll
        for (int e = 0; e < NM * 9; e += 2) {
            const cx<A> c0 = acc[e / 9][e % 9], c1 = acc[(e + 1) / 9][(e + 1) % 9];
            out[e / 2] = make_float4(c0.re, c0.im, c1.re, c1.im);
        }
    } else {
        using O = typename Store<A>::One;   // float2 or double2
        O* out = reinterpret_cast<O*>(F) + ((size_t)s * 4 + m0) * 9;
#pragma unroll
        for (int e = 0; e < NM * 9; ++e) {
            O o;
            o.x = acc[e / 9][e % 9].re;
            o.y = acc[e / 9][e % 9].im;
            out[e] = o;
        }
    }
}

template <typename T, bool STAG, int NM, bool SINGLE>
static cudaError_t force_go(const Geom& g, int Nv, const void* psi, const void* gv, void* F, cudaStream_t st)
{
    const long n = (4 / NM) * g.vol;
    k_force<T, STAG, NM, SINGLE><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(g, Nv, psi, gv, F);
    return cudaGetLastError();
}

// share of the block slots that a launch of vol / 128 * (4 / NM) blocks keeps busy, `per`
// blocks to an SM (152 SMs)
static double last_wave(long vol, int NM, int per)
{
    const long blocks = ((4 / NM) * vol + 127) / 128, slots = 152L * per;
    return (double)blocks / ((blocks + slots - 1) / slots * slots);
}

// Links per thread NM.  FP64: one (144 registers of sums for four).  Else four read least
// but leave a quarter of the threads, two blocks to an SM (Wilson): small lattices, and
// those whose last wave is mostly empty, take fewer.  The lines lie where the
// next lower NM, or NM = 1, the kernel of one link per thread, is as fast for every Nv
// from 1 to 24 (us for NM = 1, 2, 4, Nv = 12): Wilson F32 10^4 20 29 19, 12^4 27 26 27,
// 16^3 x 8 39 49 27, 16^4 103 93 62, 24^4 533 372 277; BF16 8^4 11 15 19, 12^4 23 25 29, 16^3 x 12 43 41
// 43 (Nv = 24: 92 97 101), 24^4 309 279 253; staggered F32 8^4 9 10 15, 12^4 13 13 20, 16^4 27 23 27,
// 24^4 197 130 131 (Nv = 3: 115 61 51).
static int links_per_thread(int op, bool f32, long vol)
{
    if (op == OP_STAGGERED) return vol < 16384 ? 1 : (vol < 200000 ? 2 : 4);
    if (last_wave(vol, 4, 2) >= (f32 ? 0.6 : 0.75)) return 4;
    return f32 && last_wave(vol, 2, 3) >= 0.7 ? 2 : 1;
}

template <typename T>
static cudaError_t force_T(int op, const Geom& g, int Nv, const void* psi, const void* gv, void* F, cudaStream_t st)
{
    if constexpr (sizeof(T) == 8) {
        if (op == OP_STAGGERED) return force_go<T, true, 1, true>(g, Nv, psi, gv, F, st);
        return force_go<T, false, 1, true>(g, Nv, psi, gv, F, st);
    } else {
        const int nm = links_per_thread(op, sizeof(T) == 4, g.vol);
        if (op == OP_STAGGERED) {
            if (nm == 1) return force_go<T, true, 1, false>(g, Nv, psi, gv, F, st);
            if (nm == 2) return force_go<T, true, 2, false>(g, Nv, psi, gv, F, st);
            return force_go<T, true, 4, false>(g, Nv, psi, gv, F, st);
        }
        if (Nv == 1) return force_go<T, false, 1, true>(g, Nv, psi, gv, F, st);
        if (nm == 1) return force_go<T, false, 1, false>(g, Nv, psi, gv, F, st);
        if constexpr (sizeof(T) == 4)
            if (nm == 2) return force_go<T, false, 2, false>(g, Nv, psi, gv, F, st);
        return force_go<T, false, 4, false>(g, Nv, psi, gv, F, st);
    }
}

cudaError_t launch_force(int op, int prec, const Geom& g, int Nv, const void* psi, const void* gv, void* F,
                         cudaStream_t st)
{
    switch (prec) {
    case P_F64: return force_T<double>(op, g, Nv, psi, gv, F, st);
    case P_F32: return force_T<float>(op, g, Nv, psi, gv, F, st);
    case P_BF16: return force_T<__nv_bfloat16>(op, g, Nv, psi, gv, F, st);
    case P_F16: return force_T<__half>(op, g, Nv, psi, gv, F, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace dirac

// the link gradient from packed fields
static dirac_status force_internal(dirac_handle* h, void* F, const void* pi, const void* gi)
{
    if (h->op != OP_BRILLOUIN)
        return h->cuda(launch_force(h->op, h->prec, h->g, h->Nv, pi, gi, F, h->stream), "force kernel launch");
    if (!h->have_links)   // Wilson and staggered forces need none
        return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_force: the Brillouin gradient needs links: call dirac_set_links first");
    // the transporters are rebuilt from V (not kept from the forward pass): 40
    // planes of W and 81 of G
    const size_t plane = (size_t)h->g.vol * 9 * 16;
    void* scr = nullptr;
    dirac_status st;
    if ((st = h->scratch(121 * plane, true, &scr))) return st;
    auto run = [&](bool f64) {
        return h->cuda(launch_force_brillouin(h->prec, f64, h->g, h->Nv, pi, gi, h->links64, scr,
                                              static_cast<char*>(scr) + 40 * plane, F, h->range_flag, h->stream),
                       "Brillouin force kernels");
    };
    if (h->prec == P_F64) {
        st = run(true);
    } else {
        // in double-float; again in FP64 if a result left the range
        bool again = false;
        st = h->clear_range_flag();
        if (!st) st = run(false);
        if (!st) st = h->read_range_flag(&again);
        if (!st && again) st = run(true);
    }
    h->scratch_done();
    return st;
}

extern "C" DIRAC_API dirac_status dirac_force(dirac_handle* h, void* F, const void* psi, const void* g,
                                              dirac_layout layout)
{
    if (!h) return DIRAC_ERR_INVALID_ARG;
    if (!F || !psi || !g || F == psi || F == g)
        return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_force: NULL or aliased pointers");
    if (layout != DIRAC_CANONICAL && layout != DIRAC_INTERNAL)
        return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_force: unknown layout");
    if (!dirac_check_device_ptr(F) || !dirac_check_device_ptr(psi) || !dirac_check_device_ptr(g))
        return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_force: F, psi and g must be device pointers");
    dirac_status st;
    const void *pi = psi, *gi = g;
    if (layout == DIRAC_CANONICAL) {
        if ((st = h->ensure_workspace())) return st;
        if ((st = dirac_pack(h, h->ws_in, psi))) return st;
        if ((st = dirac_pack(h, h->ws_out, g))) return st;
        pi = h->ws_in;
        gi = h->ws_out;
    }
    return force_internal(h, F, pi, gi);
}

extern "C" DIRAC_API dirac_status dirac_backward(dirac_handle* h, void* gpsi, void* F, const void* psi, const void* g)
{
    if (!h) return DIRAC_ERR_INVALID_ARG;
    if (!gpsi || !F || !psi || !g || gpsi == psi || gpsi == g || F == psi || F == g || F == gpsi)
        return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_backward: NULL or aliased pointers");
    if (!h->have_links) return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_backward: call dirac_set_links first");
    if (!dirac_check_device_ptr(gpsi) || !dirac_check_device_ptr(F) || !dirac_check_device_ptr(psi) ||
        !dirac_check_device_ptr(g))
        return h->fail(DIRAC_ERR_INVALID_ARG, "dirac_backward: need 16-byte aligned device pointers");
    dirac_status st;
    if ((st = h->ensure_workspace())) return st;
    if ((st = dirac_pack(h, h->ws_in, g))) return st;
    if ((st = h->run_apply_canonical(true, gpsi, h->ws_in))) return st;   // may pass through ws_out
    if ((st = dirac_pack(h, h->ws_out, psi))) return st;
    return force_internal(h, F, h->ws_out, h->ws_in);
}
