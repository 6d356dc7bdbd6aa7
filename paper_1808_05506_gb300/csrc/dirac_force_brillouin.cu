// Link gradient of L = Re <g, D_B psi> for the Brillouin operator (Sec. 5,
// Eqs. def_bril, def_der, def_lap at c_SW = 0), PyTorch's convention
// F = dL/dRe V + i dL/dIm V.  The off-axis transporters W_dir are not kept
// between the forward and the backward pass: they are rebuilt here
// from V by the recursion of Tab. tab:off-axis (every ordering of the k hops,
// weight 1/k!, split by the first hop):
//   W_dir(x) = (1/k) sum_{hops a of dir} H_a(x) W_{dir-a}(x+a),
//   H_{+mu}(x) = V_mu(x), H_{-mu}(x) = V_mu(x-mu)^+.
// Steps (all gathers, one write per output element, no atomics):
//   1. G_dir(y) = dL/dW_dir(y) = sum_{v,s} g_v(y)_s (M_dir psi_v(y+dir))_s^+
//      for the 80 directions, M_dir = rho_k (dir . gamma) - lambda_k / 2;
//   2. for k = 4, 3, 2 the (k-1)-hop gradients collect what the k-hop
//      directions pass down: G_{d'}(y) += (1/k) H_a(y-a)^+ G_{d'+a}(y-a) over
//      the hops a on the axes d' does not use;
//   3. F_mu(y) = sum_{dir with +mu} (1/k) G_dir(y) W_{dir-mu}(y+mu)^+
//             + sum_{dir with -mu} (1/k) W_{dir+mu}(y) G_dir(y+mu)^+
//      (W_0 = 1: the one-hop directions).
// Arithmetic: FP64 for FP64 handles; for the others, whose psi and g are exact
// in FP32 and whose F is rounded to FP32, double-float (dirac_transport.cuh), and
// FP64 after all if an entry of F leaves the range on the way.
// All steps are bound by arithmetic (step 1: 36 complex multiply-adds per
// direction and right-hand side, 144 FP64 operations, at a sixtieth of the
// FP32 rate); 12^3 x 16, 8 right-hand sides, FP32 storage, one GB300:
//                 FP64      double-float
//   step 1        9.51 ms   1.43 ms
//   W build       1.12 ms   0.28 ms  (80 directions in FP64, 40 here)
//   step 2        1.26 ms   0.56 ms
//   step 3        1.42 ms   0.54 ms
#include "dirac_handle.h"
#include "dirac_kernels.cuh"
#include "dirac_transport.cuh"

using namespace dirac;

namespace dirac {
namespace {

// h_s of the spin-transformed g: h = (M_dir / rho_k) g = kappa g + (dir . gamma) g with
// kappa = -lambda_k / (2 rho_k) = -27 2^(k-7), exact in FP32; M_dir is hermitian, so
// sum_s g_s (M psi)_s^+ = sum_s (M g)_s psi_s^+, and moving it from psi to g leaves one
// transform by sums of signed components; rho_k goes into the final scale of G.
// chiral basis, (gamma_mu g)_s = phase g_sigma: x: s <-> 3 - s, phases -i -i i i;
// y: s <-> 3 - s, - + + -; z: s <-> s ^ 2, -i i i -i; t: s <-> s ^ 2, 1
// sums of FP32 components in (hi, lo), exact up to the last bits of lo
struct Sum2 {
    float hi, lo;
    __device__ __forceinline__ void start(float kappa, float g)
    {
        hi = df_mul(kappa, g);
        lo = df_fma(kappa, g, -hi);
    }
    __device__ __forceinline__ void add(float t)
    {
        float s, e;
        dd::two_sum(hi, t, s, e);
        hi = s;
        lo = df_add(lo, e);
    }
    __device__ __forceinline__ dfl get() const { return dfl(hi, lo); }
};
struct Sum1 {
    double v;
    __device__ __forceinline__ void start(double kappa, double g) { v = kappa * g; }
    __device__ __forceinline__ void add(double t) { v += t; }
    __device__ __forceinline__ double get() const { return v; }
};

// one: the power of two h is kept times (kappa has it)
template <typename A, typename S>
__device__ __forceinline__ void h_spin(int s, const int (&d)[4], A kappa, A one, const cx<A>* g, S (&re)[3], S (&im)[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        re[c].start(kappa, g[3 * s + c].re);
        im[c].start(kappa, g[3 * s + c].im);
    }
    const cx<A>* gx = g + 3 * (3 - s);
    const cx<A>* gz = g + 3 * (s ^ 2);
    if (d[0]) {   // uniform over the warp: all its threads work on one direction
        const A f = (s < 2) == (d[0] > 0) ? one : -one;   // -i f g
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            re[c].add(f * gx[c].im);
            im[c].add(-f * gx[c].re);
        }
    }
    if (d[1]) {
        const A f = (s == 0 || s == 3) == (d[1] < 0) ? one : -one;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            re[c].add(f * gx[c].re);
            im[c].add(f * gx[c].im);
        }
    }
    if (d[2]) {
        const A f = (s == 0 || s == 3) == (d[2] > 0) ? one : -one;   // -i f g
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            re[c].add(f * gz[c].im);
            im[c].add(-f * gz[c].re);
        }
    }
    if (d[3]) {
        const A f = d[3] > 0 ? one : -one;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            re[c].add(f * gz[c].re);
            im[c].add(f * gz[c].im);
        }
    }
}

// the spinor in the arithmetic A
template <typename T, typename A>
__device__ __forceinline__ void load_as(const void* base, size_t vol, int v, long s, cx<A>* p)
{
    if constexpr (std::is_same<A, typename Store<T>::A>::value) {
        load_spinor<T, 12>(base, vol, v, s, p);
    } else {
        cx<typename Store<T>::A> q[12];
        load_spinor<T, 12>(base, vol, v, s, q);
#pragma unroll
        for (int i = 0; i < 12; ++i) p[i] = cx<A>{(A)q[i].re, (A)q[i].im};
    }
}

// step 1: one thread per (site, direction j = 0..79); F64: in FP64
template <typename T, bool F64>
__global__ void __launch_bounds__(128) k_bri_gradW(Geom g, int Nv, const void* psi, const void* gv, void* G81)
{
    using A = typename std::conditional<F64, double, float>::type;                 // of psi and g
    using B = typename std::conditional<F64, double, dfl>::type;                   // of G
    using S = typename std::conditional<F64, Sum1, Sum2>::type;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (site, j), site fastest
    if (i >= 80 * g.vol) return;
    const long y = i % g.vol;
    const int j = (int)(i / g.vol);
    const int c = j < 40 ? j : j + 1;   // skip the centre code 40
    int d[4];
    dir_of(c, d);
    long fwd[4], bwd[4];
    int x[4];
    site_offsets(g, y, fwd, bwd, x);
    long nb = y;
    int k = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        nb += d[mu] > 0 ? fwd[mu] : (d[mu] < 0 ? bwd[mu] : 0);
        k += d[mu] != 0;
    }
    // G of k hops is kept times 2^(f_exp - (k - 1) v_exp)
    const A one = F64 ? A(1) : A(pow2f(f_exp<B>() - (k - 1) * v_exp<B>()));
    const A kappa = A(-27.0 / 64.0) * A(1 << (k - 1)) * one;
    cx<B> acc[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) acc[e] = cx<B>{B(0), B(0)};
    for (int v = 0; v < Nv; ++v) {
        cx<A> ps[12], gs[12];
        load_as<T>(psi, g.vol, v, nb, ps);
        load_as<T>(gv, g.vol, v, y, gs);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            S hr[3], hi[3];
            h_spin<A, S>(s, d, kappa, one, gs, hr, hi);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const cx<B> h{hr[a].get(), hi[a].get()};
#pragma unroll
                for (int b = 0; b < 3; ++b) cmacc_conj(h, ps[3 * s + b], acc[3 * a + b]);
            }
        }
    }
    const B rho = B((double)(1 << (8 - 2 * k)) / 432.0);
#pragma unroll
    for (int e = 0; e < 9; ++e)
        st_el(G81, ((size_t)c * 9 + e) * g.vol + y, cx<B>{times(settle(acc[e].re), rho), times(settle(acc[e].im), rho)});
}

// step 2 for level k: one thread per (site, direction of k-1 hops)
template <typename A>
__global__ void __launch_bounds__(128) k_bri_back(Geom g, const __grid_constant__ DirList L, const __grid_constant__ DirPlanes P, int k, const void* W, void* G81)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long)L.n * g.vol) return;
    const long y = i % g.vol;
    const int c = L.code[i / g.vol];
    int d[4];
    dir_of(c, d);
    long fwd[4], bwd[4];
    int x[4];
    site_offsets(g, y, fwd, bwd, x);
    cx<A> acc[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) acc[e] = cx<A>{A(0), A(0)};
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        if (d[mu] != 0) continue;
        const int e1[4] = {mu == 0, mu == 1, mu == 2, mu == 3};
        const int pv = P.p[code_of(e1)];   // the plane of V_mu
        cx<A> U[9], Gu[9];
        // a = +mu: V_mu(y-mu)^+ G_{d+mu}(y-mu);  a = -mu: V_mu(y) G_{d-mu}(y+mu)
#pragma unroll 1
        for (int up = 1; up >= -1; up -= 2) {
            int dp[4] = {d[0], d[1], d[2], d[3]};
            dp[mu] = up;
            const long sn = y + (up > 0 ? bwd[mu] : fwd[mu]);
            load_mat<A>(W, g.vol, pv, up > 0 ? sn : y, up > 0, U);
            load_mat<A>(G81, g.vol, code_of(dp), sn, false, Gu);
            mm_acc(U, Gu, acc);
        }
    }
    const A inv = A(1.0 / k);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const size_t o = ((size_t)c * 9 + e) * g.vol + y;
        const cx<A> G0 = ld_el<A>(G81, o);
        st_el(G81, o, cx<A>{plus(G0.re, times(settle(acc[e].re), inv)), plus(G0.im, times(settle(acc[e].im), inv))});
    }
}

// the directions with a hop along mu, ordered by their number of hops
struct DirsOfMu {
    short code[4][54];
};

__device__ __forceinline__ float as_out(dfl a, int* bad) { return scaled_out(a, f_exp<dfl>(), bad); }
__device__ __forceinline__ double as_out(double a, int*) { return a; }

// step 3: one thread per (site, mu); F canonical [site][mu][a][b] in the type O
template <typename A, typename O>
__global__ void __launch_bounds__(128) k_bri_dV(Geom g, const __grid_constant__ DirsOfMu D, const __grid_constant__ DirPlanes P, const void* G81, const void* W, O* F, int* bad)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (site, mu), site fastest
    if (i >= 4 * g.vol) return;
    const long y = i % g.vol;
    const int mu = (int)(i / g.vol);
    long fwd[4], bwd[4];
    int x[4];
    site_offsets(g, y, fwd, bwd, x);
    long fm = fwd[0];
#pragma unroll
    for (int nu = 1; nu < 4; ++nu)
        if (mu == nu) fm = fwd[nu];
    const long yp = y + fm;
    cx<A> F9[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) F9[e] = cx<A>{A(0), A(0)};
    int j = 0;
#pragma unroll 1
    for (int k = 1; k <= 4; ++k) {
        const int nk = k == 1 ? 2 : (k == 2 ? 12 : (k == 3 ? 24 : 16));
        cx<A> acc[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) acc[e] = cx<A>{A(0), A(0)};
#pragma unroll 1
        for (int n = 0; n < nk; ++n, ++j) {
            const int c = D.code[mu][j];
            int d[4];
            dir_of(c, d);
            const int dm = mu == 0 ? d[0] : (mu == 1 ? d[1] : (mu == 2 ? d[2] : d[3]));
            // dir with +mu: G_dir(y) W_rest(y+mu)^+;  with -mu: W_rest(y) G_dir(y+mu)^+;
            // rest = dir without its hop along mu
            cx<A> Gm[9], Wr[9];
            load_mat<A>(G81, g.vol, c, dm > 0 ? y : yp, dm < 0, Gm);
            if (k == 1) {
#pragma unroll
                for (int e = 0; e < 9; ++e) acc[e] = cx<A>{plus(acc[e].re, Gm[e].re), plus(acc[e].im, Gm[e].im)};
                continue;
            }
            long so = 0;   // offset of rest
#pragma unroll
            for (int nu = 0; nu < 4; ++nu)
                if (nu != mu) so += d[nu] > 0 ? fwd[nu] : (d[nu] < 0 ? bwd[nu] : 0);
            const int p3 = mu == 0 ? 1 : (mu == 1 ? 3 : (mu == 2 ? 9 : 27));
            const int pr = P.p[c - dm * p3];
            const long z = dm > 0 ? yp : y;
            // W_rest(z) or its adjoint; rest not stored: W_rest(z) = W_{-rest}(z + rest)^+
            load_mat<A>(W, g.vol, pr >= 0 ? pr : -1 - pr, pr >= 0 ? z : z + so, (dm > 0) == (pr >= 0), Wr);
            if (dm > 0) mm_acc(Gm, Wr, acc);
            else mm_acc(Wr, Gm, acc);
        }
        const A inv = A(1.0 / k);
#pragma unroll
        for (int e = 0; e < 9; ++e)
            F9[e] = cx<A>{plus(F9[e].re, times(settle(acc[e].re), inv)),
                           plus(F9[e].im, times(settle(acc[e].im), inv))};
    }
    O* out = F + ((size_t)y * 4 + mu) * 9;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        O o;
        o.x = as_out(F9[e].re, bad);
        o.y = as_out(F9[e].im, bad);
        out[e] = o;
    }
}

template <typename T, bool F64>
cudaError_t gradW_T(const Geom& g, int Nv, const void* psi, const void* gv, void* G81, cudaStream_t st)
{
    const long n = 80 * g.vol;
    k_bri_gradW<T, F64><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(g, Nv, psi, gv, G81);
    return cudaGetLastError();
}

template <typename A, typename O>
cudaError_t chain_T(const Geom& g, const void* W, void* G, void* F, int* bad, cudaStream_t st)
{
    const DirPlanes P = dir_planes();
    for (int k = 4; k >= 2; --k) {
        const DirList L = dirs_of_hops(k - 1, false);
        const long n = (long)L.n * g.vol;
        k_bri_back<A><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(g, L, P, k, W, G);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    DirsOfMu D;
    int n[4] = {0, 0, 0, 0};
    for (int k = 1; k <= 4; ++k) {
        const DirList L = dirs_of_hops(k, false);
        for (int m = 0; m < L.n; ++m) {
            int d[4];
            dir_of(L.code[m], d);
            for (int mu = 0; mu < 4; ++mu)
                if (d[mu]) D.code[mu][n[mu]++] = L.code[m];
        }
    }
    const unsigned nb = (unsigned)((4 * g.vol + 127) / 128);
    k_bri_dV<A, O><<<nb, 128, 0, st>>>(g, D, P, G, W, static_cast<O*>(F), bad);
    return cudaGetLastError();
}

}   // namespace

cudaError_t launch_force_brillouin(int prec, bool f64, const Geom& g, int Nv, const void* psi, const void* gv,
                                   const void* V64, void* W, void* G, void* F, int* bad, cudaStream_t st)
{
    f64 = f64 || prec == P_F64;
    cudaError_t e = launch_build_W(g, V64, W, !f64, st);
    if (e != cudaSuccess) return e;
    switch (prec) {
    case P_F64: e = gradW_T<double, true>(g, Nv, psi, gv, G, st); break;
    case P_F32: e = f64 ? gradW_T<float, true>(g, Nv, psi, gv, G, st) : gradW_T<float, false>(g, Nv, psi, gv, G, st); break;
    case P_BF16:
        e = f64 ? gradW_T<__nv_bfloat16, true>(g, Nv, psi, gv, G, st) : gradW_T<__nv_bfloat16, false>(g, Nv, psi, gv, G, st);
        break;
    case P_F16: e = f64 ? gradW_T<__half, true>(g, Nv, psi, gv, G, st) : gradW_T<__half, false>(g, Nv, psi, gv, G, st); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    if (prec == P_F64) return chain_T<double, double2>(g, W, G, F, bad, st);
    return f64 ? chain_T<double, float2>(g, W, G, F, bad, st) : chain_T<dfl, float2>(g, W, G, F, bad, st);
}

}  // namespace dirac
