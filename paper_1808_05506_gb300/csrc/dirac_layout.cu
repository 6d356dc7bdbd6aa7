// Layout conversion (canonical <-> internal blocked layout) and the
// Brillouin off-axis link build of Tab. tab:off-axis.
#include "dirac_transport.cuh"

namespace dirac {

// ---------------------------------------------------------------- spinors
// canonical complex numbers c of one (site, rhs): NSC contiguous complex of type CT,
// read and written with the widest aligned vector (float4 = 2 complex when the
// 8 * NSC-byte run is 16-byte aligned, else one complex at a time)
template <int NSC, typename CT, typename A>
__device__ __forceinline__ void canon_load(const CT* src, cx<A>* p)
{
    if constexpr (sizeof(CT) == 4 && NSC % 2 == 0) {
        const float4* q = reinterpret_cast<const float4*>(src);
#pragma unroll
        for (int j = 0; j < NSC / 2; ++j) {
            float4 v = q[j];
            p[2 * j] = cx<A>{(A)v.x, (A)v.y};
            p[2 * j + 1] = cx<A>{(A)v.z, (A)v.w};
        }
    } else if constexpr (sizeof(CT) == 4) {
        const float2* q = reinterpret_cast<const float2*>(src);
#pragma unroll
        for (int j = 0; j < NSC; ++j) {
            float2 v = q[j];
            p[j] = cx<A>{(A)v.x, (A)v.y};
        }
    } else {
        const double2* q = reinterpret_cast<const double2*>(src);
#pragma unroll
        for (int j = 0; j < NSC; ++j) {
            double2 v = q[j];
            p[j] = cx<A>{(A)v.x, (A)v.y};
        }
    }
}

template <int NSC, typename CT, typename A>
__device__ __forceinline__ void canon_store(CT* dst, const cx<A>* p)
{
    if constexpr (sizeof(CT) == 4 && NSC % 2 == 0) {
        float4* q = reinterpret_cast<float4*>(dst);
#pragma unroll
        for (int j = 0; j < NSC / 2; ++j)
            q[j] = make_float4((float)p[2 * j].re, (float)p[2 * j].im, (float)p[2 * j + 1].re, (float)p[2 * j + 1].im);
    } else if constexpr (sizeof(CT) == 4) {
        float2* q = reinterpret_cast<float2*>(dst);
#pragma unroll
        for (int j = 0; j < NSC; ++j) q[j] = make_float2((float)p[j].re, (float)p[j].im);
    } else {
        double2* q = reinterpret_cast<double2*>(dst);
#pragma unroll
        for (int j = 0; j < NSC; ++j) q[j] = make_double2((double)p[j].re, (double)p[j].im);
    }
}

// canon holds the sites site0 .. site0 + nsites - 1 (a t-slab, or the whole lattice)
template <typename T, int NSC, typename CT>
__global__ void k_pack(Geom g, int Nv, const CT* __restrict__ canon, void* internal, long site0, long nsites)
{
    using A = typename Store<T>::A;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (site, v), v fastest
    if (i >= nsites * Nv) return;
    const long s = site0 + i / Nv;
    const int v = (int)(i % Nv);
    cx<A> p[NSC];
    canon_load<NSC, CT, A>(canon + (size_t)i * NSC * 2, p);
    store_spinor<T, NSC>(internal, g.vol, v, s, p);
}

template <typename T, int NSC, typename CT>
__global__ void k_unpack(Geom g, int Nv, const void* internal, CT* __restrict__ canon, long site0, long nsites)
{
    using A = typename Store<T>::A;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nsites * Nv) return;
    const long s = site0 + i / Nv;
    const int v = (int)(i % Nv);
    cx<A> p[NSC];
    load_spinor<T, NSC>(internal, g.vol, v, s, p);
    canon_store<NSC, CT, A>(canon + (size_t)i * NSC * 2, p);
}

template <typename T, int NSC>
static cudaError_t pack_T(const Geom& g, int Nv, const void* canon, bool f64, void* internal,
                          cudaStream_t st, long site0, long nsites)
{
    const long n = nsites * Nv;
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (f64) k_pack<T, NSC, double><<<nb, 256, 0, st>>>(g, Nv, (const double*)canon, internal, site0, nsites);
    else k_pack<T, NSC, float><<<nb, 256, 0, st>>>(g, Nv, (const float*)canon, internal, site0, nsites);
    return cudaGetLastError();
}

template <typename T, int NSC>
static cudaError_t unpack_T(const Geom& g, int Nv, const void* internal, void* canon, bool f64,
                            cudaStream_t st, long site0, long nsites)
{
    const long n = nsites * Nv;
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (f64) k_unpack<T, NSC, double><<<nb, 256, 0, st>>>(g, Nv, internal, (double*)canon, site0, nsites);
    else k_unpack<T, NSC, float><<<nb, 256, 0, st>>>(g, Nv, internal, (float*)canon, site0, nsites);
    return cudaGetLastError();
}

#define DISPATCH_PREC_NSC(FN, ...)                                                        \
    switch (prec) {                                                                       \
    case P_F64: return nsc == 12 ? FN<double, 12>(__VA_ARGS__) : FN<double, 3>(__VA_ARGS__); \
    case P_F32: return nsc == 12 ? FN<float, 12>(__VA_ARGS__) : FN<float, 3>(__VA_ARGS__);   \
    case P_BF16:                                                                          \
        return nsc == 12 ? FN<__nv_bfloat16, 12>(__VA_ARGS__) : FN<__nv_bfloat16, 3>(__VA_ARGS__); \
    case P_F16: return nsc == 12 ? FN<__half, 12>(__VA_ARGS__) : FN<__half, 3>(__VA_ARGS__); \
    default: return cudaErrorInvalidValue;                                                \
    }

cudaError_t launch_pack_spinor(int prec, int nsc, const Geom& g, int Nv, const void* canon,
                               bool canon_f64, void* internal, cudaStream_t st, long site0, long nsites)
{
    if (nsites < 0) nsites = g.vol;
    if (nsites * Nv == 0) return cudaSuccess;
    DISPATCH_PREC_NSC(pack_T, g, Nv, canon, canon_f64, internal, st, site0, nsites)
}

cudaError_t launch_unpack_spinor(int prec, int nsc, const Geom& g, int Nv, const void* internal,
                                 void* canon, bool canon_f64, cudaStream_t st, long site0, long nsites)
{
    if (nsites < 0) nsites = g.vol;
    if (nsites * Nv == 0) return cudaSuccess;
    DISPATCH_PREC_NSC(unpack_T, g, Nv, internal, canon, canon_f64, st, site0, nsites)
}

// one column c of a canonical FP64 field with Nsrc right-hand sides <-> slot v
// of an internal FP64 field (the batched solver's queue of systems)
template <int NSC>
__global__ void k_pack_column(Geom g, int Nsrc, int c, const double* __restrict__ canon, int v, void* internal)
{
    const long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.vol) return;
    const double* src = canon + ((size_t)s * Nsrc + c) * NSC * 2;
    cx<double> p[NSC];
#pragma unroll
    for (int k = 0; k < NSC; ++k) p[k] = cx<double>{src[2 * k], src[2 * k + 1]};
    store_spinor<double, NSC>(internal, g.vol, v, s, p);
}

template <int NSC>
__global__ void k_unpack_column(Geom g, int v, const void* internal, int Nsrc, int c, double* __restrict__ canon)
{
    const long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.vol) return;
    cx<double> p[NSC];
    load_spinor<double, NSC>(internal, g.vol, v, s, p);
    double* dst = canon + ((size_t)s * Nsrc + c) * NSC * 2;
#pragma unroll
    for (int k = 0; k < NSC; ++k) {
        dst[2 * k] = p[k].re;
        dst[2 * k + 1] = p[k].im;
    }
}

cudaError_t launch_pack_column64(int nsc, const Geom& g, int Nsrc, int c, const void* canon, int v, void* internal,
                                 cudaStream_t st)
{
    const unsigned nb = (unsigned)((g.vol + 255) / 256);
    if (nsc == 12) k_pack_column<12><<<nb, 256, 0, st>>>(g, Nsrc, c, (const double*)canon, v, internal);
    else k_pack_column<3><<<nb, 256, 0, st>>>(g, Nsrc, c, (const double*)canon, v, internal);
    return cudaGetLastError();
}

cudaError_t launch_unpack_column64(int nsc, const Geom& g, int v, const void* internal, int Nsrc, int c, void* canon,
                                   cudaStream_t st)
{
    const unsigned nb = (unsigned)((g.vol + 255) / 256);
    if (nsc == 12) k_unpack_column<12><<<nb, 256, 0, st>>>(g, v, internal, Nsrc, c, (double*)canon);
    else k_unpack_column<3><<<nb, 256, 0, st>>>(g, v, internal, Nsrc, c, (double*)canon);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- links
// Canonical links into the FP64 copy [mu][e][site] and, for T not void, the
// storage links (blocked).  A block takes 32 sites through shared memory: it reads
// their 36 complex per site as they lie in memory and writes runs of 32 sites per
// plane (16^4, FP32: the two passes it replaces, the second reading the FP64 copy
// back, took 10.9 and 10.1 us, this one 11.3).
constexpr int LK_SITES = 32;
template <typename CT, typename T>
__global__ void __launch_bounds__(256) k_links_load(long vol, const CT* __restrict__ canon, double2* V64, void* dst)
{
    using C2 = typename std::conditional<sizeof(CT) == 8, double2, float2>::type;
    __shared__ C2 sm[LK_SITES][37];
    const long s0 = (long)blockIdx.x * LK_SITES;
    const int ns = vol - s0 < LK_SITES ? (int)(vol - s0) : LK_SITES;
    const C2* src = reinterpret_cast<const C2*>(canon) + s0 * 36;
    for (int i = threadIdx.x; i < ns * 36; i += 256) sm[i / 36][i % 36] = src[i];
    __syncthreads();
    const int l = threadIdx.x & 31;
    if (l >= ns) return;
    for (int e = threadIdx.x >> 5; e < 36; e += 8) {
        const C2 c = sm[l][e];
        V64[(size_t)e * vol + s0 + l] = make_double2((double)c.x, (double)c.y);
        if constexpr (!std::is_same<T, void>::value) {
            using A = typename Store<T>::A;
            st_one<T>(dst, blk_index((size_t)vol, 9, e / 9, e % 9, s0 + l), cx<A>{(A)c.x, (A)c.y});
        }
    }
}

// prec < 0: the FP64 copy only
template <typename CT>
static cudaError_t links_load_T(const Geom& g, const CT* canon, double2* V64, int prec, void* dst, cudaStream_t st)
{
    const unsigned nb = (unsigned)((g.vol + LK_SITES - 1) / LK_SITES);
    switch (prec) {
    case P_F64: k_links_load<CT, double><<<nb, 256, 0, st>>>(g.vol, canon, V64, dst); break;
    case P_F32: k_links_load<CT, float><<<nb, 256, 0, st>>>(g.vol, canon, V64, dst); break;
    case P_BF16: k_links_load<CT, __nv_bfloat16><<<nb, 256, 0, st>>>(g.vol, canon, V64, dst); break;
    case P_F16: k_links_load<CT, __half><<<nb, 256, 0, st>>>(g.vol, canon, V64, dst); break;
    default: k_links_load<CT, void><<<nb, 256, 0, st>>>(g.vol, canon, V64, nullptr); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_links_load(const Geom& g, const void* canon, bool canon_f64, void* V64, int prec, void* dst,
                              cudaStream_t st)
{
    return canon_f64 ? links_load_T<double>(g, (const double*)canon, (double2*)V64, prec, dst, st)
                     : links_load_T<float>(g, (const float*)canon, (double2*)V64, prec, dst, st);
}

// FP64 links [m][e][site] -> storage-precision links in the blocked layout
template <typename T>
__global__ void k_convert_links(long vol, long n, const double2* __restrict__ src, void* dst)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (m, e, site), site fastest
    if (i >= n) return;
    const long s = i % vol;
    const long me = i / vol;
    double2 v = src[i];
    using A = typename Store<T>::A;
    st_one<T>(dst, blk_index((size_t)vol, 9, (int)(me / 9), (int)(me % 9), s), cx<A>{(A)v.x, (A)v.y});
}

cudaError_t launch_convert_links(int prec, const Geom& g, int nmat, const void* src64, void* dst,
                                 cudaStream_t st)
{
    const long n = g.vol * 9L * nmat;
    const unsigned nb = (unsigned)((n + 255) / 256);
    const double2* s = (const double2*)src64;
    switch (prec) {
    case P_F64: k_convert_links<double><<<nb, 256, 0, st>>>(g.vol, n, s, dst); break;
    case P_F32: k_convert_links<float><<<nb, 256, 0, st>>>(g.vol, n, s, dst); break;
    case P_BF16: k_convert_links<__nv_bfloat16><<<nb, 256, 0, st>>>(g.vol, n, s, dst); break;
    case P_F16: k_convert_links<__half><<<nb, 256, 0, st>>>(g.vol, n, s, dst); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// hops of the 40 stored directions
struct PlaneHops {
    signed char k[40];
};

// double-float W [plane][e][site] -> storage precision (FP32 or 16 bits), rounded to FP32 first
template <typename T>
__global__ void k_convert_W_df(long vol, long n, const __grid_constant__ PlaneHops H, const float4* __restrict__ src, void* dst, int* bad)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (plane, e, site), site fastest
    if (i >= n) return;
    const long s = i % vol;
    const long me = i / vol;
    const float4 v = src[i];
    const int e = DF_V * H.k[me / 9];
    const cx<float> c{scaled_out(dfl(v.x, v.y), e, bad), scaled_out(dfl(v.z, v.w), e, bad)};
    st_one<T>(dst, blk_index((size_t)vol, 9, (int)(me / 9), (int)(me % 9), s), c);
}

cudaError_t launch_convert_W_df(int prec, const Geom& g, const void* W, void* dst, int* bad, cudaStream_t st)
{
    BriDir dirs[80];
    int reps[40];
    brillouin_tables(dirs, reps);
    PlaneHops H;
    for (int r = 0; r < 40; ++r) {
        int d[4];
        dir_of(reps[r], d);
        H.k[r] = (signed char)((d[0] != 0) + (d[1] != 0) + (d[2] != 0) + (d[3] != 0));
    }
    const long n = g.vol * 360L;
    const unsigned nb = (unsigned)((n + 255) / 256);
    const float4* s = (const float4*)W;
    switch (prec) {
    case P_F32: k_convert_W_df<float><<<nb, 256, 0, st>>>(g.vol, n, H, s, dst, bad); break;
    case P_BF16: k_convert_W_df<__nv_bfloat16><<<nb, 256, 0, st>>>(g.vol, n, H, s, dst, bad); break;
    case P_F16: k_convert_W_df<__half><<<nb, 256, 0, st>>>(g.vol, n, H, s, dst, bad); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- W build
// Tab. tab:off-axis defines W_dir(x) as the average of the path products over
// the k! orderings of the k unit hops of dir.  Splitting off the first hop a
// gives the recursion W_dir(x) = (1/k) sum_{hops a of dir} V_a(x) W_{dir-a}(x+a)
// with V_{-mu}(x) = V_mu(x-mu)^+; it is evaluated level by level (k = 1..4)
// for the 40 stored directions, the others being read as adjoints.
// Bound by arithmetic: 104 products of 3x3 matrices per site.  FP64 handles
// take FP64; the others double-float, since their W is rounded to FP32 or 16
// bits (12^3 x 16: 1.12 ms for 80 directions in FP64, 0.28 ms for these).
template <typename A>
__global__ void k_w_level1(Geom g, const __grid_constant__ DirPlanes P, const double2* __restrict__ V64, void* W)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (mu, e, site), site fastest
    if (i >= g.vol * 36) return;
    const long s = i % g.vol;
    const int me = (int)(i / g.vol), mu = me / 9, e = me % 9;
    int d[4] = {mu == 0, mu == 1, mu == 2, mu == 3};
    const double2 v = V64[i];
    const double sc = (double)(1 << v_exp<A>());
    st_el(W, ((size_t)P.p[code_of(d)] * 9 + e) * g.vol + s, cx<A>{A(sc * v.x), A(sc * v.y)});
}

template <typename A>
__global__ void __launch_bounds__(128) k_w_level(Geom g, const __grid_constant__ DirList L, const __grid_constant__ DirPlanes P, void* W)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (site, j), site fastest
    if (i >= g.vol * L.n) return;
    const long s = i % g.vol;
    const int c = L.code[i / g.vol];
    int d[4];
    dir_of(c, d);
    long fwd[4], bwd[4];
    int x[4];
    site_offsets(g, s, fwd, bwd, x);
    long sd = s;   // x + dir
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) sd += d[mu] > 0 ? fwd[mu] : (d[mu] < 0 ? bwd[mu] : 0);
    cx<A> acc[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) acc[e] = cx<A>{A(0), A(0)};
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        if (d[mu] == 0) continue;
        int a[4] = {mu == 0, mu == 1, mu == 2, mu == 3};
        int rest[4] = {d[0], d[1], d[2], d[3]};
        rest[mu] = 0;
        cx<A> H[9], R[9];
        load_mat<A>(W, g.vol, P.p[code_of(a)], d[mu] > 0 ? s : s + bwd[mu], d[mu] < 0, H);
        const int pr = P.p[code_of(rest)];
        if (pr >= 0) load_mat<A>(W, g.vol, pr, s + (d[mu] > 0 ? fwd[mu] : bwd[mu]), false, R);
        else load_mat<A>(W, g.vol, -1 - pr, sd, true, R);
        mm_acc(H, R, acc);
    }
    const A inv = A(1.0 / L.k);
#pragma unroll
    for (int e = 0; e < 9; ++e)
        st_el(W, ((size_t)P.p[c] * 9 + e) * g.vol + s, cx<A>{times(settle(acc[e].re), inv), times(settle(acc[e].im), inv)});
}

template <typename A> static cudaError_t build_W_T(const Geom& g, const void* V64, void* W, cudaStream_t st)
{
    const DirPlanes P = dir_planes();
    const long n1 = g.vol * 36;
    k_w_level1<A><<<(unsigned)((n1 + 255) / 256), 256, 0, st>>>(g, P, (const double2*)V64, W);
    cudaError_t e = cudaGetLastError();
    for (int k = 2; k <= 4 && e == cudaSuccess; ++k) {
        const DirList L = dirs_of_hops(k, true);
        const long n = g.vol * L.n;
        k_w_level<A><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(g, L, P, W);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_build_W(const Geom& g, const void* V64, void* W, bool df, cudaStream_t st)
{
    return df ? build_W_T<dfl>(g, V64, W, st) : build_W_T<double>(g, V64, W, st);
}

}  // namespace dirac

// ---------------------------------------------------------------- link formats
namespace dirac {

// two-row links: planes e = 0..5 of each storage link, in a layout with 6 planes
template <typename T>
__global__ void k_links_2row(long vol, long n, const void* __restrict__ src, void* dst)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (mu, e < 6, site), site fastest
    if (i >= n) return;
    const long s = i % vol;
    const long me = i / vol;
    const int mu = (int)(me / 6), e = (int)(me % 6);
    st_one<T>(dst, blk_index((size_t)vol, 6, mu, e, s), ld_one<T>(src, blk_index((size_t)vol, 9, mu, e, s)));
}

cudaError_t launch_links_2row(int prec, const Geom& g, const void* links, void* out, cudaStream_t st)
{
    const long n = g.vol * 4L * 6;
    const unsigned nb = (unsigned)((n + 255) / 256);
    switch (prec) {
    case P_F32: k_links_2row<float><<<nb, 256, 0, st>>>(g.vol, n, links, out); break;
    case P_BF16: k_links_2row<__nv_bfloat16><<<nb, 256, 0, st>>>(g.vol, n, links, out); break;
    case P_F16: k_links_2row<__half><<<nb, 256, 0, st>>>(g.vol, n, links, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// max over the links of |U_2c - conj(U_0 x U_1)_c| in FP64 (non-negative
// doubles order like their bit patterns, so the maximum is an integer atomic)
__global__ void k_su3_deviation(long vol, const double2* __restrict__ V64, unsigned long long* dev)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (mu, site), site fastest
    double m = 0.0;
    if (i < 4 * vol) {
        const long s = i % vol;
        const int mu = (int)(i / vol);
        cx<double> U[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const double2 v = V64[((size_t)mu * 9 + e) * vol + s];
            U[e] = cx<double>{v.x, v.y};
        }
        cx<double> R[9];
#pragma unroll
        for (int e = 0; e < 6; ++e) R[e] = U[e];
        reconstruct_row2(R);
#pragma unroll
        for (int c = 6; c < 9; ++c) {
            const cx<double> d = R[c] - U[c];
            m = fmax(m, sqrt(d.re * d.re + d.im * d.im));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(dev, (unsigned long long)__double_as_longlong(m));
}

cudaError_t launch_su3_deviation(const Geom& g, const void* V64, double* dev, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(dev, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    const long n = 4 * g.vol;
    k_su3_deviation<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g.vol, (const double2*)V64,
                                                                 (unsigned long long*)dev);
    return cudaGetLastError();
}

struct RepDirs {
    signed char d[40][4];
};

// all 80 Brillouin directions per site: plane j < 40 is the stored W_{d_j}(x),
// plane 40 + j is W_{-d_j}(x) = W_{d_j}(x - d_j)^+ (Tab. tab:off-axis caption),
// both in the storage precision (a copy and a conjugate transpose: no rounding)
// planes j0..79 (j0 = 40 when src and dst are the same array: only the
// adjoint planes are written, read from the stored ones)
template <typename T>
__global__ void k_brillouin_w80(Geom g, RepDirs R, int j0, long n, const void* __restrict__ src, void* dst)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // (plane - j0, e, site), site fastest
    if (i >= n) return;
    const long s = i % g.vol;
    const long pe = i / g.vol;
    const int j = j0 + (int)(pe / 9), e = (int)(pe % 9);
    using A = typename Store<T>::A;
    cx<A> v;
    if (j < 40) {
        v = ld_one<T>(src, blk_index((size_t)g.vol, 9, j, e, s));
    } else {
        const int rep = j - 40;
        long r = s, sn = 0;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const int L = g.L[mu];
            const int x = (int)(r % L);
            r /= L;
            const int xm = (x - R.d[rep][mu] + L) % L;
            sn += (long)xm * g.stride[mu];
        }
        const int a = e / 3, b = e % 3;   // (W^+)_ab = conj(W_ba)
        v = conj(ld_one<T>(src, blk_index((size_t)g.vol, 9, rep, 3 * b + a, sn)));
    }
    st_one<T>(dst, blk_index((size_t)g.vol, 9, j, e, s), v);
}

cudaError_t launch_brillouin_w80(int prec, const Geom& g, const void* links, void* out, cudaStream_t st)
{
    BriDir dirs[80];
    int reps[40];
    brillouin_tables(dirs, reps);
    RepDirs R;
    for (int r = 0; r < 40; ++r) {
        const int c = reps[r];
        R.d[r][0] = (signed char)(c % 3 - 1);
        R.d[r][1] = (signed char)((c / 3) % 3 - 1);
        R.d[r][2] = (signed char)((c / 9) % 3 - 1);
        R.d[r][3] = (signed char)((c / 27) % 3 - 1);
    }
    const int j0 = links == out ? 40 : 0;
    const long n = g.vol * (80L - j0) * 9;
    const unsigned nb = (unsigned)((n + 255) / 256);
    switch (prec) {
    case P_F64: k_brillouin_w80<double><<<nb, 256, 0, st>>>(g, R, j0, n, links, out); break;
    case P_F32: k_brillouin_w80<float><<<nb, 256, 0, st>>>(g, R, j0, n, links, out); break;
    case P_BF16: k_brillouin_w80<__nv_bfloat16><<<nb, 256, 0, st>>>(g, R, j0, n, links, out); break;
    case P_F16: k_brillouin_w80<__half><<<nb, 256, 0, st>>>(g, R, j0, n, links, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dirac
