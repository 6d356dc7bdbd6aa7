// Brillouin sweep on the tensor cores, for BF16 and FP16 storage: launch
// variant 7.  Sec. 5, Eqs. def_bril, def_der, def_lap at c_SW = 0:
//   D_B psi(x) = (m0 + 15/8) psi(x)
//                + sum_{d != 0} W_d(x) [rho_k (d . gamma) - lambda_k / 2] psi(x + d).
// The colour and spin factors commute, so with the five coefficient classes
//   C_0(d) = -lambda_k / 2,   C_{1+mu}(d) = rho_k d_mu  (k = |d|_1),
// and T_j[c][(s, v)] = sum_{d, c'} C_j(d) W_d(x)[c][c'] psi_v(x + d)[s][c'],
//   D_B psi_v(x)[s] = (m0 + 15/8) psi_v(x)[s] + T_0[s] + sum_mu (gamma_mu T_{1+mu})[s].
// The coefficients are powers of two up to one factor per class kind,
//   C_0 = -(1/16) 2^(1-k),   C_{1+mu} = (4/27) d_mu 4^(1-k),
// so the products C W are formed in 16 bits (the factors go into the epilogue),
// exactly in BF16, so that the only rounding before the FP32 sums is that of the stored
// W.  In FP16 products below 2^-14 (|W| < 2^-8 at four hops, 2^-11 in C_0) are rounded to
// 2^-25, which is at most 2^-19 of W, next to 2^-12 for an entry near 1.
//
// One warp owns a site and up to 16 right-hand sides: a real matrix product
//   T[(j, c, re/im)][(s, v)] = A[(j, c, re/im)][(d, c', re/im)] B[(d, c', re/im)][(s, v)]
// of 30 (padded to 32) rows, on mma.sync m16n8k16 (16-bit operands, FP32
// accumulators in registers), two directions to a step of K = 16, 4 spins x 2
// right-hand sides to a tile of 8 columns.
//   A, the links: a lane reads one 16-byte element (the three rows c of column
//   c' of W_d) per direction and turns it into its eight operand registers by
//   a swap of (re, im) and a product with (+-2^n, +-2^n) from a table; rows are
//   placed so that a lane's rows 0..2 are the colours c of one class and one
//   of re/im.  T_1 and T_3 are kept times i, which makes every spin matrix of
//   the epilogue real.
//   B, the spinors: one 32-bit word of shared memory (the (re, im) of one
//   colour) is one operand register as stored, so the neighbours are copied
//   unchanged by cp.async: the 9 rows (d_y, d_z) of one d_t at a time, with the
//   links of these directions, the next stage in flight while one is used.
// An item is a tile of up to 16 sites of an (x, y) plane, one warp each, for up to
// 16 right-hand sides (the copies of a tile serve its sites' common neighbours).
// What bounds it: the mma rate (598 TFLOP/s measured for m16n8k16, 8 cycles per
// step and tile: 42 steps x 2 row tiles x 8 column tiles take 1344 cycles per
// site and 16 right-hand sides, 0.58 ms at 16^3 x 32), half reached: between the
// steps the 16 warps of an SM meet at the barrier of each stage and the epilogue
// leaves the tensor pipe idle (50 % active; 4900 instructions per site).  The
// same product on tcgen05.mma takes A and B from shared memory in core matrices;
// building those in 4- and 8-byte stores (6900 instructions and 1600 wavefronts per
// site) bounded that kernel.  16^3 x 32, BF16, one GB300: Nv = 16: 1.85 ms
// with tcgen05 and on CUDA cores, 1.17 ms here; Nv = 12: 1.45 ms on CUDA
// cores, 0.95 ms; Nv = 4: 0.54 and 0.51 ms.
#include <algorithm>
#include <mutex>

#include "dirac.h"
#include "dirac_internal.h"

namespace dirac {
namespace {

constexpr int TC_MAXW = 16;                 // sites of an item, one warp each
constexpr int TC_STAGES = 2;
constexpr int TC_SLOTS = 81;                // directions per site in the link copy: 27 x d_t, the centre zero
constexpr int TC_CO = 9;                    // table entries per direction: 8 row groups, then zeros
constexpr size_t TC_TAB = (size_t)(TC_SLOTS + 3) * TC_CO * 8;   // coefficient table in shared memory

// d_t of phase 0, 1, 2: the one with the site itself last, so that the centre
// spinor is still in shared memory in the epilogue
__host__ __device__ constexpr int tc_dt(int ph) { return ph == 0 ? -1 : (ph == 1 ? 1 : 0); }

// (exponent, sign) of the coefficients of a direction, by class
struct TcDir {
    signed char plane;   // W plane at the site (link format 1: rep, or 40 + rep); -1 the centre
    signed char k;       // |d|_1
    signed char d[4];
};
static __constant__ TcDir c_tc_dirs[TC_SLOTS];

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <typename V> __device__ __forceinline__ V tc_lds(const unsigned char* p) { return *reinterpret_cast<const V*>(p); }
// 16 bytes global -> shared; zeros when off
__device__ __forceinline__ void tc_cp16(uint32_t dst, const void* src, bool on)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}

template <typename T> __device__ __forceinline__ uint32_t tc_mul2(uint32_t a, uint32_t b);
template <> __device__ __forceinline__ uint32_t tc_mul2<__nv_bfloat16>(uint32_t a, uint32_t b)
{
    const __nv_bfloat162 r = __hmul2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
}
template <> __device__ __forceinline__ uint32_t tc_mul2<__half>(uint32_t a, uint32_t b)
{
    const __half2 r = __hmul2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
    return *reinterpret_cast<const uint32_t*>(&r);
}

template <typename T>
__device__ __forceinline__ void tc_mma(float (&c)[4], const uint32_t a0, const uint32_t a1, const uint32_t a2,
                                       const uint32_t a3, const uint32_t b0, const uint32_t b1)
{
    if constexpr (std::is_same<T, __half>::value)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                     "{%0,%1,%2,%3};"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                     : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                     "{%0,%1,%2,%3};"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                     : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// one work item: NB right-hand sides from v0 on the sites x0.. x0 + bx - 1, y0..
// y0 + by - 1 of an (x, y) plane
struct TcItem {
    long base;   // first site of the plane
    int x0, bx, y0, by, v0;
};

struct TcGrid {
    long nitems;
    int nvb, nx, ny, bx, by;   // blocks of right-hand sides, tiles per plane, sites per tile
    FDiv fv, fx, fy, fw;       // division by nvb, nx, ny and bx + 2
};

template <int NB>
__device__ __forceinline__ TcItem tc_item(const ApplyArgs& a, const TcGrid& G, long i)
{
    const uint32_t q = fdiv(G.fv, (uint32_t)i), q1 = fdiv(G.fx, q), q2 = fdiv(G.fy, q1);
    TcItem it;
    it.v0 = ((int)i - (int)q * G.nvb) * NB;
    it.x0 = ((int)q - (int)q1 * G.nx) * G.bx;
    it.y0 = ((int)q1 - (int)q2 * G.ny) * G.by;
    it.bx = min(G.bx, a.g.L[0] - it.x0);
    it.by = min(G.by, a.g.L[1] - it.y0);
    it.base = slab_site(a, (long)q2 * a.g.stride[2]);
    return it;
}

// The fill of one stage: the links of the 27 directions of phase ph, [site][27][3
// pieces of 16 bytes], then the spinors at d_t of the tile with its halo of one
// site in x, y and z, [z][y][x][rhs][3 pieces].  A thread keeps its (x, rhs,
// piece) over the rows; consecutive threads take consecutive x (16-byte pieces
// that lie side by side in the field).  start() copies the links and, where a
// row has more pieces than the CTA has threads, the pieces beyond; part(i) copies the thread's
// piece of row i = 3 y + z, so that the parts can be spread over the mma steps
// of the stage in use.
template <int NB>
struct TcFill {
    const uint4* src = nullptr;
    uint32_t dst = 0, rowbytes = 0, zstep = 0;
    int zo0 = 0, zo1 = 0, zo2 = 0, x = 0, y = 0, Lx = 0, Ly = 0, nparts = 0;
    bool on = false;

    __device__ __forceinline__ void setup(const ApplyArgs& a, const TcGrid& G, const TcItem& it, uint32_t buf, int i)
    {
        const int vk = (int)fdiv(G.fw, (uint32_t)i), p = i - vk * (G.bx + 2);
        const int v = vk / 3, k = vk - 3 * v;
        x = it.x0 - 1 + p;
        if (x < 0) x += Lx;
        if (x >= Lx) x -= Lx;
        on = it.v0 + v < a.Nv;
        src = static_cast<const uint4*>(a.in) +
              ((size_t)(on ? it.v0 + v : 0) * (uint32_t)nblk_of((size_t)a.g.vol) * 96 + 32 * k);
        dst = buf + (uint32_t)p * (NB * 48u) + (uint32_t)(v * 48 + k * 16);
        y = it.y0 == 0 ? Ly - 1 : it.y0 - 1;
    }
    __device__ __forceinline__ void start(const ApplyArgs& a, const TcGrid& G, const TcItem& it, int ph, uint32_t lbuf,
                                          uint32_t buf, int tid, int nthr)
    {
        Lx = a.g.L[0];
        Ly = a.g.L[1];
        const int yw = it.by + 2, dt = tc_dt(ph), row = it.bx * 81;
        const uint4* ls =
            static_cast<const uint4*>(a.links) + ((size_t)(it.base + (long)it.y0 * Lx + it.x0) * TC_SLOTS + 27 * ph) * 3;
        for (int yy = 0; yy < it.by; ++yy) {
            for (int i = tid; i < row; i += nthr) tc_cp16(lbuf + 16u * i, ls + (i / 81 * (TC_SLOTS * 3 - 81) + i), true);
            ls += (size_t)Lx * (TC_SLOTS * 3);
            lbuf += 16u * row;
        }
        // z and t of the plane, and the planes z - 1, z, z + 1 at t + d_t
        const int P = (int)a.g.stride[2], Lz = a.g.L[2], T = P * Lz;
        const int zt = (int)fdiv(a.g.fdP, (uint32_t)it.base), t = (int)fdiv(a.g.fd[2], (uint32_t)zt), z = zt - t * Lz;
        int tt = t + dt;
        tt = tt < 0 ? a.g.L[3] - 1 : (tt == a.g.L[3] ? 0 : tt);
        zo0 = tt * T + (z == 0 ? Lz - 1 : z - 1) * P;
        zo1 = tt * T + z * P;
        zo2 = tt * T + (z + 1 == Lz ? 0 : z + 1) * P;
        rowbytes = (uint32_t)(G.bx + 2) * (NB * 48u);
        zstep = (uint32_t)yw * rowbytes;
        const int n = NB * 3 * (G.bx + 2);
        for (int i = tid + nthr; i < n; i += nthr) {
            setup(a, G, it, buf, i);
            nparts = 3 * yw;
            rest<0>();
        }
        nparts = tid < n ? 3 * yw : 0;
        if (tid < n) setup(a, G, it, buf, tid);
    }
    // row z = dz of the current y, then (dz = 2) the next y
    __device__ __forceinline__ void part_at(int dz)
    {
        const uint32_t s = (uint32_t)(y * Lx + x + (dz == 0 ? zo0 : (dz == 1 ? zo1 : zo2)));
        tc_cp16(dst + (uint32_t)dz * zstep, src + ((s >> 5) * 96u + (s & 31u)), on);
        if (dz == 2) {
            dst += rowbytes;
            y = y + 1 == Ly ? 0 : y + 1;
        }
    }
    __device__ __forceinline__ void part(int i)
    {
        if (i < nparts) part_at(i % 3);
    }
    // the parts from I on (nparts is a multiple of 3); rolled up where the sums of
    // 12 and 16 right-hand sides leave no registers for the unrolled form
    template <int I> __device__ __forceinline__ void rest()
    {
        if constexpr (NB >= 12) {
            for (int i = I; i < nparts; ++i) part_at(i % 3);
            return;
        }
        if (nparts <= I) return;
#pragma unroll
        for (int dz = I % 3; dz < (I % 3 ? 3 : 0); ++dz) part_at(dz);
        for (int r = (I + 2) / 3; r < nparts / 3; ++r) {
#pragma unroll
            for (int dz = 0; dz < 3; ++dz) part_at(dz);
        }
    }
};

// the lane's eight A registers of one direction: w the rows c = 0..2 of column c'
// (words (re, im)), co the coefficient pairs of its class (rows c of m = 0..2)
// and of the class T_4 (m = 3, row c = g / 2)
template <typename T>
__device__ __forceinline__ void tc_a(const uint4& w, uint2 co, uint32_t sel, uint32_t sel3, int g, uint32_t (&A)[4])
{
    A[0] = tc_mul2<T>(__byte_perm(w.x, 0, sel), co.x);
    A[1] = tc_mul2<T>(__byte_perm(w.y, 0, sel), co.x);
    A[2] = tc_mul2<T>(__byte_perm(w.z, 0, sel), co.x);
    const uint32_t w3 = g < 2 ? w.x : (g < 4 ? w.y : w.z);
    A[3] = tc_mul2<T>(__byte_perm(w3, 0, sel3), co.y);
}

template <typename T, int NT>
__global__ void __launch_bounds__(TC_MAXW * 32, 1) k_brillouin_tc(ApplyArgs a, TcGrid G, float frho)
{
    constexpr int NB = 2 * NT;   // right-hand sides of an item
    // the copies of the next stage spread over the mma steps of this one; with few
    // tiles per step they only lengthen it (16^3 x 32: Nv = 16 1.29 -> 1.17 ms, 12
    // 1.01 -> 0.95 ms, but 8 0.73 -> 0.76 ms, 4 0.47 -> 0.62 ms)
    constexpr bool SPREAD = NT >= 6;
    extern __shared__ __align__(128) unsigned char tc_smem[];
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, q = lane & 3, j = g >> 1, ri = g & 1;
    // a stage: links, then spinors
    const uint32_t lbytes = (uint32_t)(G.bx * G.by) * (27u * 48u);
    const uint32_t stage = lbytes + 3u * (uint32_t)((G.bx + 2) * (G.by + 2)) * (NB * 48u);

    // coefficient pairs of every direction and row group g = (class j, re/im): the
    // signs of the realified product, (re, -im) for the real row and (im, re) for
    // the imaginary one; rows kept times i: (-im, -re) and (re, -im)
    for (int i = tid; i < (TC_SLOTS + 3) * TC_CO; i += nthr) {
        const int sl = i / TC_CO, gg = i - sl * TC_CO;
        float c[2] = {0.f, 0.f}, c3[2] = {0.f, 0.f};
        if (sl < TC_SLOTS && gg < 8 && c_tc_dirs[sl].plane >= 0) {
            const TcDir& D = c_tc_dirs[sl];
            const int jj = gg >> 1, im = gg & 1;
            const float p2 = 2.f / (float)(1 << D.k), p4 = 4.f / (float)(1 << (2 * D.k));
            const float cj = jj == 0 ? p2 : p4 * (float)D.d[jj - 1];
            const bool ti = jj == 1 || jj == 3;
            c[0] = (ti && !im) ? -cj : cj;
            c[1] = (ti || !im) ? -cj : cj;
            const float c4 = p4 * (float)D.d[3];
            c3[0] = c4;
            c3[1] = im ? c4 : -c4;
        }
        uint32_t* e = reinterpret_cast<uint32_t*>(tc_smem) + 2 * i;
        e[0] = pack2(cx<float>{c[0], c[1]}, (T*)nullptr);
        e[1] = pack2(cx<float>{c3[0], c3[1]}, (T*)nullptr);
    }

    // lane constants: (re, im) order of the two kinds of rows, table entry (lanes
    // q = 3 pad K: coefficient zero), link element, word of B in a spinor pair
    const uint32_t sel = ((ri != 0) != (j == 1 || j == 3)) ? 0x1032u : 0x3210u;
    const uint32_t sel3 = ri ? 0x1032u : 0x3210u;
    const unsigned char* tabl = tc_smem + 8 * (q == 3 ? 8 : g);
    const int qc = q == 3 ? 2 : q;
    const uint32_t boff = 4u * ((g >> 2) * 12 + 3 * (g & 3) + qc);
    const int wy_full = warp / G.bx;

    long i0 = blockIdx.x, i1 = blockIdx.x;   // item and phase of the next fill
    int ph1 = 0, nfill = 0;
    TcFill<NB> F;
    auto fill_next = [&]() {   // begins the next fill; F.part / F.rest and a commit complete it
        F.nparts = 0;
        if (i1 < G.nitems) {
            const TcItem it = tc_item<NB>(a, G, i1);
            const uint32_t b = smem_u32(tc_smem) + (uint32_t)TC_TAB + (uint32_t)(nfill % TC_STAGES) * stage;
            F.start(a, G, it, ph1, b, b + lbytes, tid, nthr);
        }
        ++nfill;
        if (++ph1 == 3) {
            ph1 = 0;
            i1 += gridDim.x;
        }
    };
    fill_next();
    F.template rest<0>();
    cp_async_commit();
    int nuse = 0;
    for (; i0 < G.nitems; i0 += gridDim.x) {
        const TcItem it = tc_item<NB>(a, G, i0);
        const bool on = warp < it.bx * it.by;
        const int wy = it.bx == G.bx ? wy_full : warp / it.bx, wx = warp - wy * it.bx;
        const long s = it.base + (long)(it.y0 + wy) * a.g.L[0] + it.x0 + wx;
        float acc0[NT][4], acc1[NT][4];   // rows m = 0, 1 and m = 2, 3
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc0[t][e] = acc1[t][e] = 0.f;
        const uint32_t ss = NB * 48u, rs = (uint32_t)(G.bx + 2) * ss, rz = (uint32_t)(it.by + 2) * rs;
        const unsigned char* buf = tc_smem;
#pragma unroll 1
        for (int ph = 0; ph < 3; ++ph) {
            cp_async_wait<TC_STAGES - 2>();
            __syncthreads();   // the stage is filled, and the one before it no longer read
            fill_next();
            if (!SPREAD || !on) {
                F.template rest<0>();
                cp_async_commit();
            }
            buf = tc_smem + TC_TAB + (uint32_t)(nuse % TC_STAGES) * stage + lbytes;
            ++nuse;
            if (!on) continue;
            const unsigned char* lk = buf - lbytes + (uint32_t)warp * (27u * 48u) + 16 * qc;
            const unsigned char* bb = buf + (uint32_t)wy * rs + (uint32_t)wx * ss + boff;
            const unsigned char* tb = tabl + ph * (27 * TC_CO * 8);
#pragma unroll
            for (int st = 0; st < 14; ++st) {
                const int e0 = 2 * st, e1 = st == 13 ? 26 : 2 * st + 1;   // (d_x + 1) + 3 (d_y + 1) + 9 (d_z + 1)
                uint32_t A0[4], A1[4];
                tc_a<T>(tc_lds<uint4>(lk + 48 * e0), tc_lds<uint2>(tb + e0 * (TC_CO * 8)), sel, sel3, g, A0);
                if (st < 13) tc_a<T>(tc_lds<uint4>(lk + 48 * e1), tc_lds<uint2>(tb + e1 * (TC_CO * 8)), sel, sel3, g, A1);
                else A1[0] = A1[1] = A1[2] = A1[3] = 0u;   // 27 directions: the last step has one
                if constexpr (SPREAD) F.part(st);
                const unsigned char* p0 = bb + (uint32_t)(e0 / 9) * rz + (uint32_t)(e0 / 3 % 3) * rs + (uint32_t)(e0 % 3) * ss;
                const unsigned char* p1 = bb + (uint32_t)(e1 / 9) * rz + (uint32_t)(e1 / 3 % 3) * rs + (uint32_t)(e1 % 3) * ss;
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    const uint32_t B0 = tc_lds<uint32_t>(p0 + 96 * t), B1 = tc_lds<uint32_t>(p1 + 96 * t);
                    tc_mma<T>(acc0[t], A0[0], A0[1], A1[0], A1[1], B0, B1);
                    tc_mma<T>(acc1[t], A0[2], A0[3], A1[2], A1[3], B0, B1);
                }
            }
            if constexpr (SPREAD) {
                F.template rest<14>();
                cp_async_commit();
            }
        }
        // Epilogue.  The lane holds, for columns (v, s) with v = q / 2 and s = 2 (q & 1)
        // + {0, 1}: rows m = 0..2 the colours of class j (re or im by ri), row 3 the
        // colour j of T_4 (j < 3).  With X = i T:
        //   out[s] = f0 T_0[s] + frho (s1 X_1[3 - s] + s2 T_2[3 - s] + s2 X_3[s ^ 2] + T_4[s ^ 2]),
        //   s1 = (-, -, +, +), s2 = (-, +, +, -): classes 1..4 move to the lane q ^ 1,
        // then the classes are summed over the lanes of j, each of which keeps the
        // colour c = j, and (re, im) are exchanged so that a lane stores one word.
        if (!on) continue;
        const bool low = (q & 1) != 0;   // the columns of the lane are spins 2, 3; the ones it serves 0, 1
        const float sa = low ? -frho : frho;   // s1, and s2 of the first served spin
        const float m0 = j == 0 ? -1.f / 16.f : sa, m1 = j == 0 ? -1.f / 16.f : (j == 1 ? sa : -sa);
        const bool swap = j == 1 || j == 2;                     // 3 - s: the other parity of s
        const int from = j == 0 ? lane : (lane ^ 1);
        const bool hi = j >= 2, odd = (j & 1) != 0;
        const unsigned char* own = buf + rz + (uint32_t)(wy + 1) * rs + (uint32_t)(wx + 1) * ss;   // the site itself
        const int cw = 3 * (2 * (q & 1) + ri) + (j < 3 ? j : 0);   // the word this lane writes: spin, colour j
        const unsigned char* ownw = own + 48 * (q >> 1) + 4 * cw;
        const uint32_t nblk = (uint32_t)nblk_of((size_t)a.g.vol);
        int v = it.v0 + (q >> 1);
        uint32_t* op = static_cast<uint32_t*>(a.out) +
                       4 * (((size_t)v * nblk + (uint32_t)(s >> 5)) * 96 + 32 * (cw >> 2) + (s & 31)) + (cw & 3);
        const size_t ostep = (size_t)nblk * (2 * 96 * 4);
#pragma unroll
        for (int t = 0; t < NT; ++t, v += 2, op += ostep) {
            float u0[3], u1[3];
            const float in0[3] = {acc0[t][0], acc0[t][2], acc1[t][0]}, in1[3] = {acc0[t][1], acc0[t][3], acc1[t][1]};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                u0[c] = __shfl_sync(0xffffffffu, m0 * (swap ? in1[c] : in0[c]), from);
                u1[c] = __shfl_sync(0xffffffffu, m1 * (swap ? in0[c] : in1[c]), from);
            }
            // sum over j, halving: first j and j ^ 2 (colours 0, 1 | 2), then j and j ^ 1
            const float a0 = (hi ? u0[2] : u0[0]) + __shfl_xor_sync(0xffffffffu, hi ? u0[0] : u0[2], 16);
            const float a1 = (hi ? u1[2] : u1[0]) + __shfl_xor_sync(0xffffffffu, hi ? u1[0] : u1[2], 16);
            const float b0 = u0[1] + __shfl_xor_sync(0xffffffffu, u0[1], 16);   // used by j < 2
            const float b1 = u1[1] + __shfl_xor_sync(0xffffffffu, u1[1], 16);
            float k0 = (odd ? b0 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : b0, 8);
            float k1 = (odd ? b1 : a1) + __shfl_xor_sync(0xffffffffu, odd ? a1 : b1, 8);
            // for j = 2 the partner j = 3 sends its a (colour 2)
            k0 = fmaf(frho, __shfl_xor_sync(0xffffffffu, acc1[t][2], 1), k0);
            k1 = fmaf(frho, __shfl_xor_sync(0xffffffffu, acc1[t][3], 1), k1);
            // (re, im) of one spin per lane: ri = 0 keeps its first column, ri = 1 its second
            const float other = __shfl_xor_sync(0xffffffffu, ri ? k0 : k1, 4);
            if (j < 3 && v < a.Nv) {
                const cx<float> pc = unpack2(tc_lds<uint32_t>(ownw + 96 * t), (T*)nullptr);
                const float dg = diag_of<float>(a, v);
                const cx<float> o{fmaf(dg, pc.re, ri ? other : k0), fmaf(dg, pc.im, ri ? k1 : other)};
                st_cs(op, pack2(o, (T*)nullptr));
            }
        }
    }
    cp_async_wait<0>();
}

template <typename T, int NT>
cudaError_t tc_go_nt(bool dag, const ApplyArgs& a, int nvb, cudaStream_t st)
{
    // the tile of at most 16 sites of a plane that fits two stages of shared memory and
    // cuts the plane into the fewest tiles (16 x 16: 8 x 2), the smaller halo at equal counts
    constexpr size_t room = 227 * 1024;
    TcGrid G;
    const int Lx = a.g.L[0], Ly = a.g.L[1];
    long best = 0;
    size_t smem = 0;
    for (int bx = 1; bx <= TC_MAXW && bx <= Lx; ++bx)
        for (int by = 1; bx * by <= TC_MAXW && by <= Ly; ++by) {
            const size_t need = TC_TAB + (size_t)TC_STAGES * (bx * by * 27 * 48 + 3 * (bx + 2) * (by + 2) * (2 * NT * 48));
            if (need > room) continue;
            const long tiles = (long)((Lx + bx - 1) / bx) * ((Ly + by - 1) / by);
            if (smem && (tiles > best || (tiles == best && need >= smem))) continue;
            best = tiles;
            smem = need;
            G.bx = bx;
            G.by = by;
        }
    G.nvb = nvb;
    G.nx = (Lx + G.bx - 1) / G.bx;
    G.ny = (Ly + G.by - 1) / G.by;
    G.fv = make_fdiv((uint32_t)nvb);
    G.fx = make_fdiv((uint32_t)G.nx);
    G.fy = make_fdiv((uint32_t)G.ny);
    G.fw = make_fdiv((uint32_t)(G.bx + 2));
    G.nitems = (a.nsites / a.g.stride[2]) * best * nvb;
    if (G.nitems <= 0) return cudaSuccess;
    if (G.nitems >= (1L << 31)) return cudaErrorInvalidValue;   // item numbers are 31 bits
    const int threads = 32 * G.bx * G.by;
    auto kern = k_brillouin_tc<T, NT>;
    // the attribute is the kernel's, shared by all handles and host threads: always the same
    // value, so that no thread takes back what another is about to launch with
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0, per = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem)) != cudaSuccess) return e;
    const long grid = std::min<long>(G.nitems, (long)nsm * std::max(per, 1));
    const float rho = 64.f / 432.f;   // 4/27
    kern<<<(unsigned)grid, threads, smem, st>>>(a, G, dag ? -rho : rho);
    return cudaGetLastError();
}

// right-hand sides per item: Nv in equal blocks of at most 16, rounded up to 4, 8, 12 or 16
template <typename T>
cudaError_t tc_go(bool dag, const ApplyArgs& a, cudaStream_t st)
{
    const int nb = (a.Nv + 15) / 16, per = (a.Nv + nb - 1) / nb;
    const int nt = (per + 3) / 4;
    const int nvb = (a.Nv + 4 * nt - 1) / (4 * nt);
    switch (nt) {
    case 1: return tc_go_nt<T, 2>(dag, a, nvb, st);
    case 2: return tc_go_nt<T, 4>(dag, a, nvb, st);
    case 3: return tc_go_nt<T, 6>(dag, a, nvb, st);
    default: return tc_go_nt<T, 8>(dag, a, nvb, st);
    }
}

}  // namespace

// the direction table of the tensor-core sweep (once per device, before any capture)
cudaError_t brillouin_tc_prepare(cudaStream_t st)
{
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    BriDir dirs[80];
    int reps[40];
    brillouin_tables(dirs, reps);
    TcDir t[TC_SLOTS];
    int n = 0;
    for (int ph = 0; ph < 3; ++ph)
        for (int r = 0; r < 27; ++r) {
            TcDir& D = t[n++];
            const int d[4] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1, tc_dt(ph)};
            D.plane = -1;
            D.k = 0;
            for (int m = 0; m < 4; ++m) {
                D.d[m] = (signed char)d[m];
                D.k += d[m] != 0;
            }
            for (int j = 0; j < 80; ++j)
                if (dirs[j].d[0] == d[0] && dirs[j].d[1] == d[1] && dirs[j].d[2] == d[2] && dirs[j].d[3] == d[3])
                    D.plane = (signed char)(dirs[j].neg ? 40 + dirs[j].rep : dirs[j].rep);
        }
    e = cudaMemcpyToSymbolAsync(c_tc_dirs, t, sizeof(t), 0, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

// bytes of the site-major link copy
size_t brillouin_tc_link_bytes(const Geom& g) { return (size_t)g.vol * TC_SLOTS * 48; }

// The site-major copy: element (s, slot, c') = the words W[0][c'], W[1][c'],
// W[2][c'], 0 of the direction of the slot (the centre: zeros).  A block takes 32
// sites and a few slots through shared memory: reads along the sites, writes along
// the elements of a site.
constexpr int TCL_SLOTS = 9;
__global__ void __launch_bounds__(256) k_brillouin_tc_links(size_t vol, const uint32_t* __restrict__ w80, uint4* __restrict__ wtc)
{
    __shared__ uint32_t sm[32][TCL_SLOTS * 9 + 1];
    const long s0 = (long)blockIdx.x * 32;
    const int sl0 = blockIdx.y * TCL_SLOTS;
    for (int i = threadIdx.x; i < TCL_SLOTS * 9 * 32; i += 256) {
        const int s = i & 31, se = i >> 5, sl = se / 9, e = se - 9 * sl;
        const int plane = c_tc_dirs[sl0 + sl].plane;
        sm[s][se] = (plane >= 0 && s0 + s < (long)vol) ? w80[blk_index(vol, 9, plane, e, s0 + s)] : 0u;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TCL_SLOTS * 3 * 32; i += 256) {
        const int s = i / (TCL_SLOTS * 3), r = i - s * (TCL_SLOTS * 3), sl = r / 3, q = r - 3 * sl;
        if (s0 + s >= (long)vol) break;
        const uint32_t* w = sm[s] + 9 * sl + q;
        wtc[((size_t)(s0 + s) * TC_SLOTS + sl0 + sl) * 3 + q] = make_uint4(w[0], w[3], w[6], 0u);
    }
}

cudaError_t launch_brillouin_tc_links(const Geom& g, const void* w80, void* wtc, cudaStream_t st)
{
    static_assert(TC_SLOTS % TCL_SLOTS == 0, "whole groups of slots");
    k_brillouin_tc_links<<<dim3((unsigned)nblk_of((size_t)g.vol), TC_SLOTS / TCL_SLOTS), 256, 0, st>>>(
        (size_t)g.vol, static_cast<const uint32_t*>(w80), static_cast<uint4*>(wtc));
    return cudaGetLastError();
}

// a.links: the W of each site, site-major (launch_brillouin_tc_links), 16-bit;
// a.in, a.out 16-bit fields of the storage type
cudaError_t launch_brillouin_tc(int prec, bool dag, const ApplyArgs& a, cudaStream_t st)
{
    if (a.nsites == 0 || a.Nv == 0) return cudaSuccess;
    if (prec == P_BF16) return tc_go<__nv_bfloat16>(dag, a, st);
    if (prec == P_F16) return tc_go<__half>(dag, a, st);
    return cudaErrorInvalidValue;
}

}  // namespace dirac
