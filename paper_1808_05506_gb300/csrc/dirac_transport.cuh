// Building blocks of the Brillouin transporters W_dir (Tab. tab:off-axis) and
// of the gradient through them: the direction codes, matrix fields of 16-byte
// elements, and 3x3 products in FP64 or double-float arithmetic.
//
// A matrix field is [plane][9][site].  The transporters take 40 planes, one
// per +-dir (brillouin_tables): the others follow from W_{-dir}(x) =
// W_dir(x - dir)^+ (table caption), so the recursion over the hops forms half
// the products and moves half the bytes of one that keeps all 80.
//
// A = double: FP64 arithmetic.  A = dfl: double-float (dirac_df.cuh), a
// 48-bit significand in FP32 instructions.  FP64 runs at 1/62 of the FP32
// rate on this GPU and these kernels are bound by arithmetic, so for results
// that are rounded to FP32 or less at their end double-float is the cheaper
// arithmetic whose error (1e-14) stays far below that rounding.
//
// Double-float has FP32's exponent range, the result's own, but the sums on the
// way can leave it where the result does not.  So the chain is kept times powers
// of two, V times 2^DF_V, W of k hops times 2^(k DF_V) and the gradient times
// 2^DF_F, which puts what its products lose below FP32's smallest number (2^-149)
// at 2^-165 and less of the result; and a result that is not finite at the end
// is computed again in FP64 (a word in device memory, which the host reads
// where it waits for the stream anyway).
#pragma once

#include "dirac_df.cuh"

namespace dirac {

// directions of k hops: their dir81 codes
struct DirList {
    int n, k;
    short code[32];
};
// plane of a direction: p >= 0: W_dir is stored in plane p; p < 0: W_dir(x) =
// W_{plane -1 - p}(x + dir)^+ (the centre is not used)
struct DirPlanes {
    signed char p[81];
};

HD void dir_of(int c, int d[4])
{
    d[0] = c % 3 - 1;
    d[1] = (c / 3) % 3 - 1;
    d[2] = (c / 9) % 3 - 1;
    d[3] = (c / 27) % 3 - 1;
}
HD int code_of(const int d[4]) { return (d[0] + 1) + 3 * (d[1] + 1) + 9 * (d[2] + 1) + 27 * (d[3] + 1); }

// rep_only: the stored representatives (first nonzero component positive)
inline DirList dirs_of_hops(int k, bool rep_only)
{
    DirList L;
    L.n = 0;
    L.k = k;
    for (int c = 0; c < 81; ++c) {
        int d[4], n = 0, first = 0;
        dir_of(c, d);
        for (int mu = 0; mu < 4; ++mu) {
            n += d[mu] != 0;
            if (!first) first = d[mu];
        }
        if (n == k && (!rep_only || first > 0)) L.code[L.n++] = (short)c;
    }
    return L;
}
inline DirPlanes dir_planes()
{
    BriDir dirs[80];
    int reps[40];
    brillouin_tables(dirs, reps);
    DirPlanes t;
    for (int c = 0; c < 81; ++c) t.p[c] = 0;
    for (int r = 0; r < 40; ++r) {
        t.p[reps[r]] = (signed char)r;
        t.p[80 - reps[r]] = (signed char)(-1 - r);
    }
    return t;
}

#if defined(__CUDACC__)
template <typename A> __device__ __forceinline__ cx<A> ld_el(const void* p, size_t i);
template <> __device__ __forceinline__ cx<double> ld_el<double>(const void* p, size_t i)
{
    const double2 v = static_cast<const double2*>(p)[i];
    return {v.x, v.y};
}
template <> __device__ __forceinline__ cx<dfl> ld_el<dfl>(const void* p, size_t i)
{
    const float4 v = static_cast<const float4*>(p)[i];
    return {dfl(v.x, v.y), dfl(v.z, v.w)};
}
__device__ __forceinline__ void st_el(void* p, size_t i, cx<double> c)
{
    static_cast<double2*>(p)[i] = make_double2(c.re, c.im);
}
__device__ __forceinline__ void st_el(void* p, size_t i, cx<dfl> c)
{
    static_cast<float4*>(p)[i] = make_float4(c.re.hi, c.re.lo, c.im.hi, c.im.lo);
}

// the matrix of a plane at a site, or its adjoint
template <typename A>
__device__ __forceinline__ void load_mat(const void* base, size_t vol, int plane, long s, bool dag, cx<A>* M)
{
    const size_t b = (size_t)plane * 9 * vol + (size_t)s;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            cx<A> v = ld_el<A>(base, b + (size_t)(dag ? 3 * c + a : 3 * a + c) * vol);
            if (dag) v.im = -v.im;
            M[3 * a + c] = v;
        }
}

// powers of two the chain is kept times (1 in FP64)
constexpr int DF_V = 8, DF_F = 48;
template <typename A> __device__ constexpr int v_exp() { return std::is_same<A, dfl>::value ? DF_V : 0; }
template <typename A> __device__ constexpr int f_exp() { return std::is_same<A, dfl>::value ? DF_F : 0; }
// 2^e, |e| <= 126
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }

// acc += x y.  Double-float sums over many terms keep (hi, lo) unnormalised:
// hi follows by exact two-sums, lo collects the rounding errors; settle()
// renormalises once at the end.
__device__ __forceinline__ void macc(double x, double y, double& acc) { acc = fma(x, y, acc); }
__device__ __forceinline__ void macc(dfl x, dfl y, dfl& acc)
{
    const float p = df_mul(x.hi, y.hi);
    float e = df_fma(x.hi, y.hi, -p);
    e = df_fma(x.hi, y.lo, e);
    e = df_fma(x.lo, y.hi, e);
    float s, t;
    dd::two_sum(acc.hi, p, s, t);
    acc.hi = s;
    acc.lo = df_add(acc.lo, df_add(t, e));
}
// y an FP32 number
__device__ __forceinline__ void macc(dfl x, float y, dfl& acc)
{
    const float p = df_mul(x.hi, y);
    float e = df_fma(x.hi, y, -p);
    e = df_fma(x.lo, y, e);
    float s, t;
    dd::two_sum(acc.hi, p, s, t);
    acc.hi = s;
    acc.lo = df_add(acc.lo, df_add(t, e));
}
__device__ __forceinline__ double settle(double a) { return a; }
// a sum beyond FP32's range stays infinite (its lo is not a number), here and
// in the next two
__device__ __forceinline__ bool in_range(float v) { return fabsf(v) <= 3.402823466e38f; }
__device__ __forceinline__ dfl settle(dfl a)
{
    dfl r(a.hi, 0.f);
    if (in_range(a.hi)) dd::fast_two_sum(a.hi, a.lo, r.hi, r.lo);
    return r;
}
__device__ __forceinline__ double times(double a, double b) { return a * b; }
__device__ __forceinline__ dfl times(dfl a, dfl b)
{
    const float p = df_mul(a.hi, b.hi);
    return in_range(p) ? a * b : dfl(p, 0.f);
}
__device__ __forceinline__ double plus(double a, double b) { return a + b; }
__device__ __forceinline__ dfl plus(dfl a, dfl b)
{
    const float s = df_add(a.hi, b.hi);
    return in_range(s) ? a + b : dfl(s, 0.f);
}
// a 2^-e rounded to FP32 (e >= 0; below its normal range from both halves, in a
// call: inlined, the compiler computes its FP64 operations for every value and
// selects, 345 -> 544 us for the links of 12^3 x 16); marks *bad if a left the range
static __device__ __noinline__ float scaled_below(float hi, float lo, int e)
{
    return (float)(((double)hi + (double)lo) * (double)pow2f(-e));
}
__device__ __forceinline__ float scaled_out(dfl a, int e, int* bad)
{
    if (!in_range(a.hi)) *bad = 1;
    const float r = a.hi * pow2f(-e);
    return fabsf(r) < 1.17549435e-38f && a.hi != 0.f ? scaled_below(a.hi, a.lo, e) : r;
}
template <typename A, typename B> __device__ __forceinline__ void cmacc(cx<A> x, cx<B> y, cx<A>& acc)
{
    macc(x.re, y.re, acc.re);
    macc(-x.im, y.im, acc.re);
    macc(x.re, y.im, acc.im);
    macc(x.im, y.re, acc.im);
}
// acc += x conj(y)
template <typename A, typename B> __device__ __forceinline__ void cmacc_conj(cx<A> x, cx<B> y, cx<A>& acc)
{
    macc(x.re, y.re, acc.re);
    macc(x.im, y.im, acc.re);
    macc(x.im, y.re, acc.im);
    macc(-x.re, y.im, acc.im);
}
// acc += X Y (3x3)
template <typename A> __device__ __forceinline__ void mm_acc(const cx<A>* X, const cx<A>* Y, cx<A>* acc)
{
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int m = 0; m < 3; ++m) cmacc(X[3 * a + m], Y[3 * m + b], acc[3 * a + b]);
}
#endif   // __CUDACC__

// the 40 transporters from V64 ([4][9][site], FP64) into W [40][9][site]: FP64,
// or double-float when df (W of k hops times 2^(k DF_V))
cudaError_t launch_build_W(const Geom& g, const void* V64, void* W, bool df, cudaStream_t st);
// the 40 double-float transporters into storage precision (blocked layout); *bad
// is set where one is not finite
cudaError_t launch_convert_W_df(int prec, const Geom& g, const void* W, void* dst, int* bad, cudaStream_t st);

}  // namespace dirac
