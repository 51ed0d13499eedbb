// gfmc_packed.cuh -- the parity-packed recursion: one complex vector per update.
//
// On an even periodic cubic lattice the sites fall into two parity classes and
// Htilde only couples different classes.  The recursion on the proposal's
// vectors |o> and |v> = Delta~|o> (Algorithm 1, Eq. recursive) starts on
// opposite classes (o on its own, v on its neighbours'), so T_n(Htilde)|o> and
// T_n(Htilde)|v> live on opposite classes for every n.  Their sum
//     S_n = T_n(Htilde) (|o> + |v>),   S_{n+1} = 2 Htilde S_n - S_{n-1}
// therefore holds both: the sites of parity(o) + n carry r_n^o, the others
// r_n^v.  One scalar stencil over the lattice advances both vectors, and the
// products that do not vanish by parity are local to a site:
//     |r_m^o|^2 over class A (parity(o) + m),  |r_m^v|^2 over class B,
//     <r_m^o|r_{m+1}^v> over class A.
// Delta Omega needs nothing else: <o|T_n|o> and <v|T_n|v> vanish for odd n and
// <o|T_n|v> for even n.
//
// Tile.  A CTA holds the pencil of whole x-rows y in [y0, y0 + PY),
// z in [z0, z0 + PZ) with a ring of one row on the four sides.  After a step the owner of
// a face value stores it into the neighbour's ring as well, so the stencil reads the CTA's
// own shared memory only.  On a thread-block cluster the ring stores go over
// distributed shared memory and one hardware cluster barrier ends the step.
//
// Bound: FP32 by shared-memory wavefronts and instruction issue on large
// pencils, by the latency of one step (loads, sums, barrier) on small ones;
// FP64, in fixed point, by the latency of a step and its exchange (gfmc_packed64.cuh).  Against
// the two-vector cluster engine, which advances both vectors on every site (half of the
// values are zeros), ms per update at M = 1024: FP32 L = 32 on 16 CTAs 1.44 -> 0.65, on 8 CTAs
// 2.03 -> 1.23, L = 16 on 1 CTA 1.92 -> 1.22, L = 8 on 1 CTA 0.80 -> 0.37; FP64 L = 16 on 16 CTAs
// 3.12 -> 1.66 with FP64 arithmetic, 0.63 in fixed point (below).
#pragma once

#include "gfmc_engine.cuh"

namespace gfmc {

// ---------------------------------------------------------------------------
// sums
// ---------------------------------------------------------------------------

// FP32 terms summed exactly, as integers: x = hi 2^-20 + lo 2^-41 to 2^-42, for |x| < 4 - 2^-20, by four
// additions.  Adding 12 leaves x on the grid of the floats in [8, 16), whose bits count in
// units of 2^-20; the remainder, at most 2^-21, goes the same way.  Sums of up to 2047
// terms (|lo| <= 2^20 each) do not depend on their order.  bad collects the bits that a
// term in range leaves zero.
struct FixTerm {
    int hi, lo;
};
constexpr unsigned kFixBad = 0xbe800000u;
__device__ __forceinline__ FixTerm fix_term(float x, unsigned& bad)
{
    constexpr float kHi = 12.f, kLo = 0x1.8p-18f;
    constexpr int kHiBits = 0x41400000, kLoBits = 0x36c00000;
    const float t = __fadd_rn(x, kHi);
    const float u = __fadd_rn(__fsub_rn(x, __fsub_rn(t, kHi)), kLo);
    bad |= __float_as_uint(t);
    return {__float_as_int(t) - kHiBits, __float_as_int(u) - kLoBits};
}
// the value of a sum of terms, in units of 2^-60
__device__ __forceinline__ long long fix_value(int hi, int lo) { return ((long long)hi << 40) + ((long long)lo << 19); }
// fix_term of x.x and x.y, by packed additions
__device__ __forceinline__ void fix_terms(float2 x, FixTerm& a, FixTerm& b, unsigned& bad)
{
    constexpr float kHi = 12.f, kLo = 0x1.8p-18f;
    constexpr int kHiBits = 0x41400000, kLoBits = 0x36c00000;
    const float2 t = __fadd2_rn(x, make_float2(kHi, kHi)), w = __fadd2_rn(t, make_float2(-kHi, -kHi));
    const float2 u = __fadd2_rn(__ffma2_rn(w, make_float2(-1.f, -1.f), x), make_float2(kLo, kLo));
    bad |= __float_as_uint(t.x) | __float_as_uint(t.y);
    a = {__float_as_int(t.x) - kHiBits, __float_as_int(u.x) - kLoBits};
    b = {__float_as_int(t.y) - kHiBits, __float_as_int(u.y) - kLoBits};
}

// Values kept apart by the lane groups of 8 of a warp: on return lanes 8 v .. 8 v + 7 hold value
// v (v < 4) over four lanes each (scatter), or the warp's sum of it.
template <class T> __device__ __forceinline__ T warp_scatter4(const T (&v)[4], int lane)
{
    const bool u16 = lane & 16, u8 = lane & 8;
    const T a = u16 ? v[2] : v[0], b = u16 ? v[3] : v[1];
    const T sa = u16 ? v[0] : v[2], sb = u16 ? v[1] : v[3];
    const T x = a + __shfl_xor_sync(0xffffffffu, sa, 16), y = b + __shfl_xor_sync(0xffffffffu, sb, 16);
    return (u8 ? y : x) + __shfl_xor_sync(0xffffffffu, u8 ? x : y, 8);
}
template <class T> __device__ __forceinline__ T warp_reduce_scatter4(const T (&v)[4], int lane)
{
    T r = warp_scatter4(v, lane);
    r += __shfl_xor_sync(0xffffffffu, r, 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}

// The four sums of each step by warp, kept until they are flushed: a warp
// writes step m between its arrival at the barrier that ends the step and its
// wait there, so the sums of step m are complete for every warp after the
// barrier of step m + 1.  Every kPkGroup steps as many warps add one step each
// into the chain's sums (at step m = 1 mod kPkGroup the steps m - kPkGroup - 1 .. m - 2; the
// slots are written again kPkRing steps later), which keeps the additions off the
// steps' critical path: one warp flushing one step in every step cost 220-320 cycles of each.
constexpr int kPkGroup = 8, kPkRing = 16;
template <class R, int NW> struct PkSums {
    long long w[kPkRing][NW][4];
};

// Add the warps' sums of step m (run by one warp) into the chain's fixed-point
// Gram sums, in units of 2^-60: entries 0 |r_m^o|^2, 1 |r_m^v|^2, 6 and 7
// <r_m^o|r_{m+1}^v>.  The sums over warps and CTAs are integer sums, so their
// order does not matter; every |sum| <= 1.
constexpr int kPkFrac = 60;
template <class R, int NW>
__device__ __forceinline__ void pk_flush(const Params& p, const PkSums<R, NW>& s, int m, int lane)
{
    const int v = lane >> 3;
    long long q = 0;
#pragma unroll
    for (int w = 0; w < NW; w += 8) q += s.w[m & (kPkRing - 1)][w + (lane & 7)][v];
    q += __shfl_xor_sync(0xffffffffu, q, 4);
    q += __shfl_xor_sync(0xffffffffu, q, 2);
    q += __shfl_xor_sync(0xffffffffu, q, 1);
    if ((lane & 7) == 0)
        atomicAdd(p.gram + (size_t)(m - 1) * kEntries + (v < 2 ? v : v + 4), (unsigned long long)q);
}
template <class R, int NW>
__device__ __forceinline__ void pk_flush_due(const Params& p, const PkSums<R, NW>& s, int m, int warp, int lane)
{
    if ((m & (kPkGroup - 1)) == 1 && m > kPkGroup) {
        if constexpr (sizeof(R) == 8) {
            // lane (step, value) of one warp adds the warps' sums
            const int f = m - kPkGroup - 1 + (lane >> 2), v = lane & 3;
            if (warp == 0 && f > 0) {
                long long q = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) q += s.w[f & (kPkRing - 1)][w][v];
                atomicAdd(p.gram + (size_t)(f - 1) * kEntries + (v < 2 ? v : v + 4), (unsigned long long)q);
            }
        } else if (warp < kPkGroup) {
            const int f = m - kPkGroup - 1 + warp;
            if (f > 0) pk_flush<R, NW>(p, s, f, lane);
        }
    }
}
// The steps that pk_flush_due, last called for step `last`, has not reached;
// the warps have met since the last step's sums were written.
template <class R, int NW>
__device__ __forceinline__ void pk_flush_rest(const Params& p, const PkSums<R, NW>& s, int last, int warp, int lane)
{
    const int done = last > kPkGroup ? ((last - 1) & ~(kPkGroup - 1)) - 1 : 0;  // the last step flushed
    for (int f = max(done, 0) + 1 + warp; f <= p.nsteps; f += NW) pk_flush<R, NW>(p, s, f, lane);
}

// ---------------------------------------------------------------------------
// the tile
// ---------------------------------------------------------------------------
struct PkTile {
    int L, half, PY, PZ, Cy, Cz, cy, cz, y0, z0, C, rank;
    int zstr;          // ring rows per plane, PY + 2
    unsigned ring;     // shared address of the ring buffers
    unsigned bufB;     // bytes of one ring buffer
    unsigned r_ym, r_yp, r_zm, r_zp;  // shared::cluster ring addresses of the four neighbours
    char* ringp;
    char* bonds;       // BX [PZ][PY], BY [PZ][PY + 1] (from y0 - 1), BZ [PZ + 1][PY] (from z0 - 1) rows
    unsigned rowB;     // bytes of a row
    __device__ __forceinline__ int ring_row(int y, int z) const { return (z + 1) * zstr + y + 1; }
    __device__ __forceinline__ int bx_row(int y, int z) const { return z * PY + y; }
    __device__ __forceinline__ int by_row(int y, int z) const { return PY * PZ + z * (PY + 1) + y + 1; }
    __device__ __forceinline__ int bz_row(int y, int z) const
    {
        return PY * PZ + PZ * (PY + 1) + (z + 1) * PY + y;
    }
    __device__ __forceinline__ int bond_rows() const { return 3 * PY * PZ + PZ + PY; }
};

// The pencils of a grid chain may differ by one row in y and z.
template <class R> __device__ __forceinline__ PkTile pk_tile(const Params& p, int rank, char* smem)
{
    PkTile t;
    t.L = p.L;
    t.half = p.L / 2;
    t.C = p.ncta;
    t.rank = rank;
    t.Cy = p.pk_cy;
    t.Cz = t.C / t.Cy;
    t.cy = rank % t.Cy;
    t.cz = rank / t.Cy;
    t.y0 = t.cy * t.L / t.Cy;
    t.z0 = t.cz * t.L / t.Cz;
    t.PY = (t.cy + 1) * t.L / t.Cy - t.y0;
    t.PZ = (t.cz + 1) * t.L / t.Cz - t.z0;
    t.zstr = t.PY + 2;
    t.rowB = (unsigned)(t.L * 2 * sizeof(R));
    t.ringp = smem;
    t.ring = smem_u32(smem);
    t.bufB = (unsigned)(t.zstr * (t.PZ + 2)) * t.rowB;
    t.bonds = smem + pk_work_bytes(t.L, t.PY, t.PZ, p.K, sizeof(R) == 4);
    t.r_ym = cluster_addr(t.ring, (t.cy + t.Cy - 1) % t.Cy + t.cz * t.Cy);
    t.r_yp = cluster_addr(t.ring, (t.cy + 1) % t.Cy + t.cz * t.Cy);
    t.r_zm = cluster_addr(t.ring, t.cy + ((t.cz + t.Cz - 1) % t.Cz) * t.Cy);
    t.r_zp = cluster_addr(t.ring, t.cy + ((t.cz + 1) % t.Cz) * t.Cy);
    return t;
}

// A face value into a neighbour's ring where `on` (predicated: four branches
// per site cost about 300 cycles of a small tile's step).  A pencil that is its
// own neighbour stores to itself the same way.
__device__ __forceinline__ void pk_st(bool on, unsigned a, float4 v)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n @p st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};\n}" ::"r"(a),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((unsigned)on)
                 : "memory");
}
__device__ __forceinline__ void pk_st(bool on, unsigned a, int4 v)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n @p st.shared::cluster.v4.s32 [%0], {%1, %2, %3, %4};\n}" ::"r"(a),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((unsigned)on)
                 : "memory");
}

// End of a step on the chain's cluster: arrive once this thread's stores are
// issued, wait before the next step's loads.
__device__ __forceinline__ void pk_arrive(int C)
{
    __syncwarp();
    if (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void pk_wait(int C)
{
    if (C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
}

__device__ __forceinline__ int4 lds4(unsigned a)
{
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ int2 lds2(unsigned a)
{
    int2 v;
    asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts2(unsigned a, int2 v)
{
    asm volatile("st.shared.v2.s32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void sts4(unsigned a, int4 v)
{
    asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// the limbs of two fixed-point values: value = high 2^30 + low, the low limb in [-2^29, 2^29)
__device__ __forceinline__ int4 pk_limbs(long long re, long long im)
{
    return make_int4((int)((re + (1ll << 29)) >> 30), (int)((unsigned)re << 2) >> 2, (int)((im + (1ll << 29)) >> 30),
                     (int)((unsigned)im << 2) >> 2);
}

// 2 Htilde's forward bonds of the tile's rows (and of the rows below it in y
// and z) into shared memory.  FP32 rows hold the pairs (x = 2j, 2j + 1) as
// (re, re, im, im), FP64 rows the fixed-point limbs, even sites first.
template <class R, int NT> __device__ __forceinline__ void pk_load_bonds(const Params& p, const PkTile& t)
{
    const int L = t.L, PY = t.PY, PZ = t.PZ, n1 = PY * PZ, n2 = PZ * (PY + 1), rows = t.bond_rows();
    for (int e = threadIdx.x; e < rows * L; e += NT) {
        const int row = e / L, x = e - row * L;
        int a, y, z;
        if (row < n1) {
            a = 0;
            z = row / PY;
            y = row - z * PY;
        } else if (row < n1 + n2) {
            a = 1;
            z = (row - n1) / (PY + 1);
            y = row - n1 - z * (PY + 1) - 1;
        } else {
            a = 2;
            z = (row - n1 - n2) / PY;
            y = row - n1 - n2 - z * PY;
            --z;
        }
        const int gy = (t.y0 + y + L) % L, gz = (t.z0 + z + L) % L;
        const size_t at = (size_t)a * p.N + (size_t)(gz * L + gy) * L + x;
        if constexpr (sizeof(R) == 4) {
            const float2 h = ldcg2(p.hop32 + at);
            float* d = (float*)(t.bonds + (size_t)row * t.rowB) + 4 * (x >> 1) + (x & 1);
            d[0] = 2.f * h.x;
            d[2] = 2.f * h.y;
        } else {
            const double2 h = ldcg2(p.hop64 + at);
            ((int4*)(t.bonds + (size_t)row * t.rowB))[(x & 1) * t.half + (x >> 1)] =
                pk_limbs(__double2ll_rn(h.x * 0x1p61), __double2ll_rn(h.y * 0x1p61));
        }
    }
}

// value of S_0 = |o> + |v> at global site i
__device__ __forceinline__ double2 pk_s0(int i, const int* s_loc, const double2* s_c)
{
    double2 r = make_double2(i == s_loc[0] ? 1.0 : 0.0, 0.0);
#pragma unroll
    for (int k = 1; k < 7; ++k)
        if (i == s_loc[k]) r = s_c[k];
    return r;
}

// ---------------------------------------------------------------------------
// FP32 steps
// ---------------------------------------------------------------------------
// A thread advances up to KZ pairs of x-neighbours (x = 2j, 2j + 1) stacked in
// z: both sites of a pair by one packed FMA, the z-neighbours inside the stack
// and S_{m-1} from registers.  BREG: the pairs' bonds stay in registers for the
// whole update (KZ <= 2 at 512 threads); otherwise the y and z bonds are read
// from shared memory in every step.
struct Pk32Bond {
    float2 re, im;
};
__device__ __forceinline__ float4 pk_ld(const char* a) { return *(const float4*)a; }
__device__ __forceinline__ Pk32Bond pk_bond(const char* a)
{
    const float4 b = *(const float4*)a;
    return {make_float2(b.x, b.y), make_float2(b.z, b.w)};
}

// sums of the positive terms (P, Q) and of the negative ones (S, W): re = P - S, im = Q - W
struct Pk32Acc {
    float2 P = {0.f, 0.f}, Q = {0.f, 0.f}, S = {0.f, 0.f}, W = {0.f, 0.f};
    __device__ __forceinline__ void fwd(const Pk32Bond& h, float2 re, float2 im)
    {
        P = __ffma2_rn(h.re, re, P);
        Q = __ffma2_rn(h.re, im, Q);
        S = __ffma2_rn(h.im, im, S);
        Q = __ffma2_rn(h.im, re, Q);
    }
    __device__ __forceinline__ void bwd(const Pk32Bond& h, float2 re, float2 im)
    {
        P = __ffma2_rn(h.re, re, P);
        Q = __ffma2_rn(h.re, im, Q);
        P = __ffma2_rn(h.im, im, P);
        W = __ffma2_rn(h.im, re, W);
    }
};

template <int NT, int KZ, bool BREG>
__device__ __forceinline__ void pk32_steps(const Params& p, const PkTile& t, const int* s_loc, const double2* s_c,
                                           PkSums<float, NT / 32>& sums, int nseg)
{
    const int nsteps = p.nsteps;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int half = t.half, ncol = half * t.PY;
    const int seg = tid / ncol, col = tid - seg * ncol, y = col / half, j = col - y * half;
    const int z0 = seg * KZ;
    const int nz = seg < nseg ? min(KZ, t.PZ - z0) : 0;
    const int jl = j == 0 ? half - 1 : j - 1, jr = j == half - 1 ? 0 : j + 1;
    const unsigned strY = t.rowB, strZ = (unsigned)t.zstr * t.rowB;
    const unsigned own = nz > 0 ? (unsigned)t.ring_row(y, z0) * t.rowB + 16u * (unsigned)j : 0u;
    const int dl = 16 * (jl - j), dr = 16 * (jr - j);
    const bool fy0 = y == 0, fy1 = y == t.PY - 1, fz0 = z0 == 0, fz1 = z0 + nz == t.PZ;
    // where this column's face values go: the neighbour's ring row beyond the far side
    const unsigned p_ym = t.r_ym + own + strY * (unsigned)t.PY;                      // y = PY of the CTA below
    const unsigned p_yp = t.r_yp + own - strY * (unsigned)t.PY;                      // y = -1 of the CTA above
    const unsigned p_zm = t.r_zm + own + strZ * (unsigned)t.PZ;                      // z = PZ of the CTA below
    const unsigned p_zp = t.r_zp + own - strZ * (unsigned)t.PZ;                      // z = -1 of the CTA above
    auto put = [&](unsigned buf, int k, float4 v) {
        const unsigned o = buf + strZ * (unsigned)k;
        *(float4*)(t.ringp + own + o) = v;
        pk_st(fy0, p_ym + o, v);
        pk_st(fy1, p_yp + o, v);
        pk_st(fz0 && k == 0, p_zm + o, v);
        pk_st(fz1 && k == nz - 1, p_zp + o, v);
    };

    // bonds: inner (2j -> 2j + 1), outer (left neighbour's, conjugated, and right), y and z
    float2 bin[KZ];
    Pk32Bond bout[KZ], byf[BREG ? KZ : 1], byb[BREG ? KZ : 1], bz[BREG ? KZ + 1 : 1];
    const char *a_yf = t.bonds, *a_zf = t.bonds;
    if (nz > 0) {
        a_yf += (size_t)t.by_row(y, z0) * t.rowB + 16 * j;
        a_zf += (size_t)t.bz_row(y, z0) * t.rowB + 16 * j;
    }
    const int sYz = (t.PY + 1) * (int)t.rowB, sZz = t.PY * (int)t.rowB;
    if constexpr (BREG) bz[0] = pk_bond(a_zf - (nz > 0 ? sZz : 0));
#pragma unroll
    for (int k = 0; k < KZ; ++k) {
        bin[k] = make_float2(0.f, 0.f);
        bout[k] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (k < nz) {
            const char* bx = t.bonds + (size_t)t.bx_row(y, z0 + k) * t.rowB;
            const Pk32Bond c = pk_bond(bx + 16 * j), l = pk_bond(bx + 16 * jl);
            bin[k] = make_float2(c.re.x, c.im.x);
            bout[k] = {make_float2(l.re.y, c.re.y), make_float2(-l.im.y, c.im.y)};
        }
        if constexpr (BREG) {
            const Pk32Bond z = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            byf[k] = k < nz ? pk_bond(a_yf + k * sYz) : z;
            byb[k] = k < nz ? pk_bond(a_yf + k * sYz - (int)t.rowB) : z;
            bz[k + 1] = k < nz ? pk_bond(a_zf + k * sZz) : z;
        }
    }

    float4 va[KZ], vb[KZ];  // S_m and S_{m-1}, by turns
#pragma unroll
    for (int k = 0; k < KZ; ++k) {
        vb[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        va[k] = vb[k];
        if (k < nz) {
            const int i = 2 * j + t.L * (t.y0 + y + t.L * (t.z0 + z0 + k));
            const double2 e = pk_s0(i, s_loc, s_c), o = pk_s0(i + 1, s_loc, s_c);
            va[k] = make_float4((float)e.x, (float)o.x, (float)e.y, (float)o.y);
            put(0, k, va[k]);
        }
    }
    pk_arrive(t.C);
    pk_wait(t.C);

    const int lo = s_loc[0];
    const int par_o = (lo % t.L + (lo / t.L) % t.L + lo / (t.L * t.L)) & 1;
    const int par_t = (t.y0 + y + t.z0 + z0) & 1;  // parity of the first pair's even site

    // one step: S_m in cur (and the ring), S_{m-1} in prv, which receives S_{m+1}
    auto step = [&](int m, float4 (&cur)[KZ], float4 (&prv)[KZ]) {
        const char* rb = t.ringp + own + (m & 1) * t.bufB;
        const unsigned wb = (unsigned)((m + 1) & 1) * t.bufB;
        float2 U[2] = {}, Xr[2] = {}, Xi[2] = {};
        float4 below = nz > 0 ? pk_ld(rb - strZ) : make_float4(0.f, 0.f, 0.f, 0.f);
        Pk32Bond zb;
        if constexpr (BREG) zb = bz[0];
        else zb = pk_bond(a_zf - (nz > 0 ? sZz : 0));
#pragma unroll
        for (int k = 0; k < KZ; ++k) {
            if (k < nz) {
                const char* r = rb + strZ * (unsigned)k;
                const float4 vl = pk_ld(r + dl), vr = pk_ld(r + dr), yp = pk_ld(r + strY), ym = pk_ld(r - strY);
                const float4 c = cur[k];
                float4 above;
                if (k + 1 < KZ && k + 1 < nz) above = cur[k + 1 < KZ ? k + 1 : k];
                else above = pk_ld(r + strZ);
                Pk32Bond hf, hb, zf;
                if constexpr (BREG) {
                    hf = byf[k];
                    hb = byb[k];
                    zf = bz[k + 1];
                } else {
                    hf = pk_bond(a_yf + k * sYz);
                    hb = pk_bond(a_yf + k * sYz - (int)t.rowB);
                    zf = pk_bond(a_zf + k * sZz);
                }
                Pk32Acc a;
                // even site: odd of the own pair; odd site: even of the own pair (conjugated bond)
                a.fwd({make_float2(bin[k].x, bin[k].x), make_float2(bin[k].y, -bin[k].y)}, make_float2(c.y, c.x),
                      make_float2(c.w, c.z));
                a.bwd(zb, make_float2(below.x, below.y), make_float2(below.z, below.w));
                a.fwd(zf, make_float2(above.x, above.y), make_float2(above.z, above.w));
                a.fwd(bout[k], make_float2(vl.y, vr.x), make_float2(vl.w, vr.z));
                a.fwd(hf, make_float2(yp.x, yp.y), make_float2(yp.z, yp.w));
                a.bwd(hb, make_float2(ym.x, ym.y), make_float2(ym.z, ym.w));
                const float2 m1 = make_float2(-1.f, -1.f);
                // the bonds first, S_{m-1} last: added onto -S_{m-1}, every term rounds at its magnitude
                // (rms error of Delta Omega, L = 16 at M = 256: 2.6e-8 so, 2.2e-8 with the bonds first)
                float2 re = __ffma2_rn(a.S, m1, a.P);
                float2 im = __ffma2_rn(a.W, m1, a.Q);
                re = __ffma2_rn(make_float2(prv[k].x, prv[k].y), m1, re);
                im = __ffma2_rn(make_float2(prv[k].z, prv[k].w), m1, im);
                if (m == 0) {  // S_1 = Htilde S_0
                    re = make_float2(0.5f * re.x, 0.5f * re.y);
                    im = make_float2(0.5f * im.x, 0.5f * im.y);
                }
                const float4 nx = make_float4(re.x, re.y, im.x, im.y);
                if (m < nsteps) put(wb, k, nx);
                const float2 cr = make_float2(c.x, c.y), ci = make_float2(c.z, c.w);
                U[k & 1] = __ffma2_rn(ci, ci, __ffma2_rn(cr, cr, U[k & 1]));
                Xr[k & 1] = __ffma2_rn(ci, im, __ffma2_rn(cr, re, Xr[k & 1]));
                Xi[k & 1] = __ffma2_rn(cr, im, Xi[k & 1]);
                Xi[k & 1] = __ffma2_rn(make_float2(-ci.x, -ci.y), re, Xi[k & 1]);
                below = c;
                zb = zf;
                prv[k] = nx;
            }
        }
        int h = 0, l = 0;  // value lane >> 3 of the step's sums
        if (m > 0) {
            // class A: the sites of parity par_o + m; an even site has the parity of its row
            const bool ea = par_t == ((par_o + m) & 1);
            float v[4];
            v[0] = ea ? U[0].x + U[1].y : U[0].y + U[1].x;
            v[1] = ea ? U[0].y + U[1].x : U[0].x + U[1].y;
            v[2] = ea ? Xr[0].x + Xr[1].y : Xr[0].y + Xr[1].x;
            v[3] = ea ? Xi[0].x + Xi[1].y : Xi[0].y + Xi[1].x;
            // a thread's sums (of up to four pairs) in FP32, the threads' as integers: over the warp
            // in FP32 they cost more than the recursion's rounding (rms error of Delta Omega over 72
            // updates, M = 256, uniform spins: L = 24 on 16 CTAs 2.4e-8, with the bonds first and this 1.3e-8)
            unsigned bad = 0;
            int hi[4], lo[4];
#pragma unroll
            for (int k = 0; k < 4; k += 2) {
                FixTerm a, b;
                fix_terms(make_float2(v[k], v[k + 1]), a, b, bad);
                hi[k] = a.hi;
                lo[k] = a.lo;
                hi[k + 1] = b.hi;
                lo[k + 1] = b.lo;
            }
            if (bad & kFixBad) set_error(p, ERR_NUMERIC, 90, m);
            h = warp_scatter4(hi, lane);
            l = warp_scatter4(lo, lane);
        }
        // these come before the arrival, whose release waits for the remote stores to be
        // acknowledged (400-560 cycles on a cluster); the rest of the sums before the wait
        pk_arrive(t.C);
        if (m > 0) {
#pragma unroll
            for (int b = 4; b > 0; b >>= 1) {
                h += __shfl_xor_sync(0xffffffffu, h, b);
                l += __shfl_xor_sync(0xffffffffu, l, b);
            }
            if ((lane & 7) == 0) sums.w[m & (kPkRing - 1)][warp][lane >> 3] = fix_value(h, l);
        }
        pk_flush_due<float, NW>(p, sums, m, warp, lane);
        pk_wait(t.C);
    };
    int m = 0;
    for (; m + 1 <= nsteps; m += 2) {
        step(m, va, vb);
        step(m + 1, vb, va);
    }
    if (m <= nsteps) step(m, va, vb);
    __syncthreads();
    pk_flush_rest<float, NW>(p, sums, nsteps, warp, lane);
}

// ---------------------------------------------------------------------------
// FP64 chains: the recursion in fixed point with 60 fraction bits
// ---------------------------------------------------------------------------
// GB300's FP64 pipe retires 2 multiply-adds per clock and SM, its integer
// multiplier about 55 32 x 32 + 64-bit multiply-adds (both measured).
// |S_n(i)| <= 1 on every site (|T_n(Htilde)| <= 1, |v| < 0.82: |Delta~|, or v scaled), so FP64
// chains hold S, and 2 Htilde (|2 Htilde| < 0.34; finer than a double above 2^-8), in
// units of 2^-60 as two limbs, x = xh 2^30 + xl with the low limb centred in
// [-2^29, 2^29).  In the same units
//     h s = hh sh + (hh sl + hl sh) 2^-30 + hl sl 2^-60,
// three wide multiply-adds per real product; the last term, below a quarter
// unit and of either sign, is left out.  A step rounds once, by half a unit
// (4.3e-19), and leaves out 12 such terms per component, 0.29 units rms together, as much as
// the rounding; the FP64 recursion rounds 12 times, each by half a unit in the last
// place of its partial sums (4.3e-19 where |S_n(i)| is near 2^-8, more above).
// Bounds: sum over the six bonds of |hh sl| <= 2.9 2^59 and of |hl sh| <= 3.5 2^59
// (Cauchy-Schwarz, |S_n| <= 1 on a class), so a sum of the middle products stays below 2^62.
struct PkBond64 {
    int rh, rl, ih, il;
};
__device__ __forceinline__ long long pk_join(int h, int l) { return ((long long)h << 30) + l; }
// acc += x y, 32 x 32 + 64 bits in one instruction (left to the compiler, a good
// part of the products came out as separate multiplies and additions: a step
// of L = 32 on 128 CTAs 4466 -> 3529 cycles)
__device__ __forceinline__ void pk_wide(long long& acc, int x, int y)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(x), "r"(y));
}
__device__ __forceinline__ void pk_mac(long long& A, long long& B, int hh, int hl, int sh, int sl)
{
    pk_wide(A, hh, sh);
    pk_wide(B, hh, sl);
    pk_wide(B, hl, sh);
}
// value of sums of limb products: A in units, B in units of 2^30
__device__ __forceinline__ long long pk_value(long long A, long long B) { return A + ((B + (1ll << 29)) >> 30); }
// Sums of one step over a thread's sites, in units of 2^-60: |S_m|^2 by class and
// <S_m|S_{m+1}> over class A, as sums of limb products put together once per
// step.  The squares keep the square of the low limb, which does not average
// out; of the products of S_m and S_{m+1} it is left out.  Over the n sites of a thread
// sum |sh| <= 2^30 sqrt(2 n): the middle sums stay below 2^62 and the low
// squares (their upper halves, 32 bits) below 2^31 for n <= 8; threads with more
// sites put their sums together every kPkPut sites.
constexpr int kPkPut = 8;
struct Pk64Sums {
    long long v[4] = {0, 0, 0, 0};
    long long A[2] = {0, 0}, B[2] = {0, 0};        // squares, by class (0: A)
    int C[2] = {0, 0};
    long long RA = 0, RB = 0, IA = 0, IB = 0;      // Re and Im of the products
    template <int K> __device__ __forceinline__ void square(int h, int l)
    {
        pk_wide(A[K], h, h);
        pk_wide(B[K], h, l);
        C[K] += __mulhi(l, l);
    }
    __device__ __forceinline__ void add(int4 c, int4 n, bool a)
    {
        if (a) {
            square<0>(c.x, c.y);
            square<0>(c.z, c.w);
            pk_mac(RA, RB, c.x, c.y, n.x, n.y);
            pk_mac(RA, RB, c.z, c.w, n.z, n.w);
            pk_mac(IA, IB, c.x, c.y, n.z, n.w);
            pk_mac(IA, IB, -c.z, -c.w, n.x, n.y);
        } else {
            square<1>(c.x, c.y);
            square<1>(c.z, c.w);
        }
    }
    __device__ __forceinline__ void put()
    {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            // (h 2^30 + l)^2 2^-60 = h^2 + 2 h l 2^-30 + l^2 2^-60
            v[k] += A[k] + ((B[k] + 2ll * C[k] + (1ll << 28)) >> 29);
            A[k] = B[k] = 0;
            C[k] = 0;
        }
        v[2] += pk_value(RA, RB);
        v[3] += pk_value(IA, IB);
        RA = RB = IA = IB = 0;
    }
};

// Large tiles on a cluster (more sites than gfmc_packed64.cuh takes): whole sites
// per thread, dealt out class by class, everything in shared memory.  A ring
// row holds its even sites first, then the odd ones, so that the sites a warp
// reads are contiguous.
struct Pk64Site {
    int at;          // byte offset of the site in a ring buffer
    int dxp, dxm;    // byte offsets of its x-neighbours
    int bond;        // byte offset of its x bond
    int y, z, x, cls;
};
__device__ __forceinline__ Pk64Site pk64_site(const PkTile& t, int s, int T2)
{
    Pk64Site q;
    q.cls = s >= T2 ? 1 : 0;
    const int g = s - q.cls * T2, r = g / t.half, j = g - r * t.half;
    q.z = r / t.PY;
    q.y = r - q.z * t.PY;
    const int odd = (q.cls + t.y0 + q.y + t.z0 + q.z) & 1;
    q.x = 2 * j + odd;
    const int col = odd * t.half + j, other = (1 - odd) * t.half;
    const int jp = odd ? (j == t.half - 1 ? 0 : j + 1) : j, jm = odd ? j : (j == 0 ? t.half - 1 : j - 1);
    q.at = 16 * (t.ring_row(q.y, q.z) * t.L + col);
    q.dxp = 16 * (other + jp - col);
    q.dxm = 16 * (other + jm - col);
    q.bond = 16 * (r * t.L + col);
    return q;
}
// the six bonds of a site, backward ones conjugated: re += rr sr - ii si, im += rr si + ii sr
__device__ __forceinline__ void pk64_bonds(const PkTile& t, const Pk64Site& q, PkBond64 (&h)[6])
{
    const char* b = t.bonds + q.bond;
    const int rowB = (int)t.rowB, plane = t.PY * t.PZ;
    const char* by = b + (plane + q.z + 1) * rowB;                       // row z (PY + 1) + y + 1 of BY
    const char* bz = b + (plane + t.PZ * (t.PY + 1) + t.PY) * rowB;      // row (z + 1) PY + y of BZ
    const char* at[6] = {b, b + q.dxm, by, by - rowB, bz, bz - t.PY * rowB};
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        const int4 v = *(const int4*)at[d];
        h[d] = (d & 1) ? PkBond64{v.x, v.y, -v.z, -v.w} : PkBond64{v.x, v.y, v.z, v.w};
    }
}
// 2 Htilde S_m - S_{m-1} at a site: re, im hold S_{m-1} and receive the value
__device__ __forceinline__ void pk64_stencil(const int4 (&v)[6], const PkBond64 (&h)[6], long long& re, long long& im)
{
    long long PA = -re, PB = 0, NA = 0, NB = 0, QA = -im, QB = 0;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        pk_mac(PA, PB, h[d].rh, h[d].rl, v[d].x, v[d].y);
        pk_mac(NA, NB, h[d].ih, h[d].il, v[d].z, v[d].w);
        pk_mac(QA, QB, h[d].rh, h[d].rl, v[d].z, v[d].w);
        pk_mac(QA, QB, h[d].ih, h[d].il, v[d].x, v[d].y);
    }
    re = pk_value(PA - NA, PB - NB);
    im = pk_value(QA, QB);
}

template <int NT>
__device__ __noinline__ void pk64_steps(const Params& p, const PkTile& tile, const int* s_loc, const double2* s_c,
                                           PkSums<double, NT / 32>& sums)
{
    const PkTile t = tile;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int L = t.L, T = L * t.PY * t.PZ, T2 = T / 2;
    const int rowB = (int)t.rowB, planeB = t.zstr * rowB;
    const unsigned yB = t.rowB * (unsigned)t.PY, zB = t.rowB * (unsigned)(t.zstr * t.PZ);
    auto put = [&](int buf, const Pk64Site& q, int4 v) {
        const unsigned b = (unsigned)buf * t.bufB + (unsigned)q.at;
        *(int4*)(t.ringp + b) = v;
        pk_st(q.y == 0, t.r_ym + b + yB, v);
        pk_st(q.y == t.PY - 1, t.r_yp + b - yB, v);
        pk_st(q.z == 0, t.r_zm + b + zB, v);
        pk_st(q.z == t.PZ - 1, t.r_zp + b - zB, v);
    };
    for (int s = tid; s < T; s += NT) {
        const Pk64Site q = pk64_site(t, s, T2);
        const double2 v = pk_s0(q.x + L * (t.y0 + q.y + L * (t.z0 + q.z)), s_loc, s_c);
        put(0, q, pk_limbs(__double2ll_rn(v.x * 0x1p60), __double2ll_rn(v.y * 0x1p60)));
    }
    pk_arrive(t.C);
    const int lo = s_loc[0];
    const int par_o = (lo % L + (lo / L) % L + lo / (L * L)) & 1;
    for (int m = 0; m <= p.nsteps; ++m) {
        pk_wait(t.C);
        const int wb = (m + 1) & 1;
        const char* rd = t.ringp + (m & 1) * t.bufB;
        const char* wr = t.ringp + wb * t.bufB;
        const int clsA = (par_o + m) & 1;
        Pk64Sums acc;
        int nadd = 0;
        for (int s = tid; s < T; s += NT) {
            const Pk64Site q = pk64_site(t, s, T2);
            PkBond64 h[6];
            pk64_bonds(t, q, h);
            const int4 pv = *(const int4*)(wr + q.at), c = *(const int4*)(rd + q.at);
            long long a = m == 0 ? 0 : pk_join(pv.x, pv.y), b = m == 0 ? 0 : pk_join(pv.z, pv.w);
            const char* r = rd + q.at;
            const int4 v[6] = {*(const int4*)(r + q.dxp),  *(const int4*)(r + q.dxm),    *(const int4*)(r + rowB),
                               *(const int4*)(r - rowB), *(const int4*)(r + planeB), *(const int4*)(r - planeB)};
            pk64_stencil(v, h, a, b);
            if (m == 0) {  // S_1 = Htilde S_0
                a = (a + 1) >> 1;
                b = (b + 1) >> 1;
            }
            const int4 n = pk_limbs(a, b);
            if (m < p.nsteps) put(wb, q, n);
            acc.add(c, n, q.cls == clsA);
            if (++nadd % kPkPut == 0) acc.put();
        }
        acc.put();
        if (m > 0) {
            const long long s = warp_reduce_scatter4(acc.v, lane);
            if ((lane & 7) == 0) sums.w[m & (kPkRing - 1)][warp][lane >> 3] = s;
        }
        if (m < p.nsteps) pk_arrive(t.C);
        pk_flush_due<double, NW>(p, sums, m, warp, lane);
    }
    __syncthreads();
    pk_flush_rest<double, NW>(p, sums, p.nsteps, warp, lane);
}

// ---------------------------------------------------------------------------
// the tail
// ---------------------------------------------------------------------------
// With <o|T_n|o> and <v|T_n|v> zero for odd n and X_n = <o|T_n|v> zero for
// even n, the four sequences oo, vv, Re X, Im X have K/2 terms each and
//     f(theta) = sum_p a_p e^{-2 i p theta}           (oo, vv; n = 2p)
//     f(theta) = e^{-i theta} sum_p b_p e^{-2 i p theta}   (Re X, Im X; n = 2p + 1)
// at the even nodes k = 2j (theta_k = pi (k + 1/2)/K) is a K/2-point FFT of the
// twisted terms a_p e^{-i pi p / K} (Eqs. green_fft, mu_to_mu_tilde).  With
// s = 2 / sin theta_k the Green's functions are i s f (Eq. green_short),
// G_ov = i s (f_A + i f_B), G_vo = i s (f_A - i f_B) for f_A, f_B of Re X and Im X, and
//     d = (1 + G_ov)(1 + G_vo) - G_oo G_vv
//       = 1 + 2 i s f_A + s^2 (f_oo f_vv - f_A^2 - f_B^2)       (Eq. d_z_green).
// The odd nodes follow from theta_{K-1-k} = pi - theta_k: f -> conj f for oo, vv
// and -conj f for A, B, hence d_{K-1-k} = conj d_k and arg d_{K-1-k} = -arg d_k.

// What an update starts from and ends with, in shared memory.
struct PkHead {
    double2 c[kVec];             // 2^n v = 2^n Delta~ |o> at the local sites
    double chi[8][3];            // spinors of the local sites and of the proposal
    int loc[kVec];
    int mom[kVec];               // moments calls: the local sites, and where their values go
    unsigned row[2][kVec];
    double draw[3];
    double vv0;                  // <v|v>
    double2 ov1;                 // <o|Htilde|v>
    double unit[3];              // twice a unit of the sums oo, vv and ov: the recursion runs on 2^n v (pk_setup)
    int acc;
    int stop;                    // a CTA marked the update as failed
};

// FFT of the chain's sequences: tasks (sequence V, residue r mod Rz of the node
// index j), task = V Rz + r, dealt round robin to the C CTAs; f of the even
// nodes goes to p.gnode[V K + j].  work: room for work_n double2 (at least K/2).
template <int NT>
__device__ __forceinline__ void pk_tail_fft(const Params& p, int rank, int C, double2* work, int work_n, const PkHead& head)
{
    const int tid = threadIdx.x, K = p.K, H = K / 2, MH = p.M / 2;
    int Rz = 1;
    while (4 * Rz * 2 <= C && Rz < 8 && H / (2 * Rz) >= 8) Rz *= 2;
    const int n = H / Rz, ntask = 4 * Rz;
    int lg = 0;
    while ((1 << lg) < n) ++lg;
    const int mine = rank < ntask ? (ntask - 1 - rank) / C + 1 : 0;
    const int g = min(mine, work_n >> lg);
    const double2 tw1 = __ldg(p.twc + 1);
    for (int b = 0; b < mine; b += g) {
        const int nb = min(g, mine - b), tot = nb << lg;
        for (int e = tid; e < tot; e += NT) {
            const int task = rank + (b + (e >> lg)) * C, V = task / Rz, r = task - V * Rz, q = e & (n - 1);
            const double unit = head.unit[min(V, 2)];
            double2 x = make_double2(0.0, 0.0);
            for (int pp = q; pp < MH; pp += n) {
                const int nn = 2 * pp + (V >> 1);
                const double first = V == 0 ? 1.0 : V == 1 ? head.vv0 : V == 2 ? head.ov1.x : head.ov1.y;
                double a = first;
                if (pp > 0) {
                    const long long s = (long long)__ldcg(p.gram + (size_t)(pp - 1) * kEntries + (V < 2 ? V : V + 4));
                    a = fma((double)s, unit, -first);  // 2 <.|.> - mu_0 (or mu_1)
                }
                a *= __ldg(p.gker + nn) * (nn == 0 ? 0.5 : 1.0);
                double2 w = __ldg(p.twc + 2 * pp);
                if (r) {
                    const int at = (2 * pp * r) & (K - 1);
                    const double2 u = __ldg(p.fftw + (at & (H - 1)));
                    w = dmul(w, at >= H ? make_double2(dneg(u.x), dneg(u.y)) : u);
                }
                x.x = fma(a, w.x, x.x);
                x.y = fma(a, w.y, x.y);
            }
            work[(e & ~(n - 1)) + (lg ? (int)(__brev((unsigned)q) >> (32 - lg)) : 0)] = x;
        }
        __syncthreads();
        for (int lh = 0; lh < lg; ++lh) {
            const int hf = 1 << lh;
            for (int e = tid; e < (tot >> 1); e += NT) {
                const int pos = e & (hf - 1), i0 = ((e >> lh) << (lh + 1)) + pos, i1 = i0 + hf;
                const double2 w = __ldg(p.fftw + ((size_t)pos * (K >> (lh + 1))));
                const double2 u = work[i0], tt = dmul(w, work[i1]);
                work[i0] = dadd(u, tt);
                work[i1] = dsub(u, tt);
            }
            __syncthreads();
        }
        for (int e = tid; e < tot; e += NT) {
            const int task = rank + (b + (e >> lg)) * C, V = task / Rz, r = task - V * Rz;
            const int jn = Rz * (e & (n - 1)) + r;
            double2 x = work[e];
            if (V >= 2) x = dmul(x, dmul(__ldg(p.fftw + jn), tw1));  // e^{-i theta_{2j}}
            __stcg(p.gnode + (size_t)V * K + jn, x);
        }
        __syncthreads();
    }
}

// arg d at the even node k = 2j
__device__ __forceinline__ double pk_arg(const Params& p, int jn)
{
    const int K = p.K;
    const double2 oo = __ldcg(p.gnode + jn), vv = __ldcg(p.gnode + (size_t)K + jn);
    const double2 A = __ldcg(p.gnode + 2 * (size_t)K + jn), B = __ldcg(p.gnode + 3 * (size_t)K + jn);
    const double s = 2.0 / __ldg(p.sinth + 2 * jn);
    const double2 t = dsub(dsub(dmul(oo, vv), dmul(A, A)), dmul(B, B));
    const double2 d = make_double2(fma(s * s, t.x, fma(-2.0 * s, A.y, 1.0)), fma(s * s, t.y, 2.0 * s * A.x));
    if (!isfinite(d.x) || !isfinite(d.y)) set_error(p, ERR_NUMERIC, 40, 2 * jn);
    return atan2(d.y, d.x);
}

__device__ __forceinline__ double pk_wrap(double x)
{
    if (x > CUDART_PI) x -= 2.0 * CUDART_PI;
    else if (x <= -CUDART_PI) x += 2.0 * CUDART_PI;
    return x;
}

// The CTA's part of sum_k inc_k C_k (Eq. d_seff2; inc_k = phi_k - phi_{k+1}
// mapped into (-pi, pi], inc_{K-1} = phi_{K-1}) over the nodes 2j, 2j + 1 and
// their mirrors K-1-2j, K-2-2j for its j in [j0, j1) of [0, K/4): with
// E_j = phi_{2j} and j' = K/2 - 1 - j, phi_{2j+1} = -E_{j'}.
template <int NT>
__device__ __forceinline__ void pk_tail_phase(const Params& p, int rank, int C, double* sarg)
{
    const int tid = threadIdx.x, K = p.K, Q = K / 4;
    const int j0 = (int)(((long long)rank * Q) / C), j1 = (int)(((long long)(rank + 1) * Q) / C), n = j1 - j0;
    double* A = sarg;          // E_{j0 .. j1}
    double* B = sarg + n + 1;  // E_{j'} for j = j0 - 1 .. j1 - 1
    for (int e = tid; e < 2 * n + 2 && n > 0; e += NT) {
        const int jn = e <= n ? j0 + e : K / 2 - 1 - (j0 - 1 + e - (n + 1));
        sarg[e] = jn < K / 2 ? pk_arg(p, jn) : 0.0;
    }
    __syncthreads();
    double part = 0.0, mx = 0.0;
    for (int q = tid; q < n; q += NT) {
        const int j = j0 + q;
        const double a = A[q], b = B[q + 1];
        const double i0 = pk_wrap(a + b), i1 = pk_wrap(-b - A[q + 1]);
        const double i3 = j == 0 ? -a : pk_wrap(-a - B[q]);
        part = fma(i0, __ldg(p.cumw + 2 * j), part);
        part = fma(i1, __ldg(p.cumw + 2 * j + 1), part);
        part = fma(i0, __ldg(p.cumw + (K - 2 - 2 * j)), part);
        part = fma(i3, __ldg(p.cumw + (K - 1 - 2 * j)), part);
        mx = fmax(mx, fmax(fabs(i0), fmax(fabs(i1), fabs(i3))));
    }
    double ps, pm;
    block_sum_max<NT>(part, mx, &ps, &pm);
    if (tid == 0) {
        p.qpart[2 * rank] = ps;
        p.qpart[2 * rank + 1] = pm;
    }
}

// the chain's sums have been read: clear them for the next update
template <int NT> __device__ __forceinline__ void pk_tail_clear(const Params& p, int rank, int C)
{
    for (int e = rank * NT + (int)threadIdx.x; e < 4 * p.nsteps; e += C * NT) {
        const int v = e & 3;
        __stcg(p.gram + (size_t)(e >> 2) * kEntries + (v < 2 ? v : v + 4), 0ull);
    }
}

// Local sites, proposal and Delta~ by warp 0, one sincos per lane (lane k the
// polar, lane 8 + k the azimuthal angle): the FP64 pipe takes 64 cycles per
// warp instruction, so seven threads with six sincos each took six times as
// long.  The caller's barrier follows.
__device__ __forceinline__ void pk_setup(const Params& p, PkHead& h, int o, unsigned long long upd)
{
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x, k = lane & 7;
    const int lk = k == 0 ? o : nbr_site(o, min(k, 6) - 1, p.L);
    double th = p.theta_new, ph = p.phi_new, u = 0.0;
    if (p.mode == MODE_SWEEP) draw_update(p.seed, p.chain_id, upd, th, ph, u);
    if (lane == 7) {
        h.draw[0] = th;
        h.draw[1] = ph;
        h.draw[2] = u;
    }
    if (k < 7) {
        th = __ldcg(p.spins + 2 * lk);
        ph = __ldcg(p.spins + 2 * lk + 1);
    }
    double sn, cs;
    sincos((lane & 8) ? ph : 0.5 * th, &sn, &cs);
    const double sp = __shfl_sync(0xffffffffu, sn, k + 8), cp = __shfl_sync(0xffffffffu, cs, k + 8);
    if (lane < 8) {
        h.chi[k][0] = cs;
        h.chi[k][1] = cp * sn;
        h.chi[k][2] = sp * sn;
    }
    if (lane < 7) h.loc[lane] = lk;
    __syncwarp();
    double2 cv = make_double2(0.0, 0.0), hv = cv;
    if (lane > 0 && lane < 7) {
        // Delta~_{l_j,o} = -t (<chi_j|chi'_o> - <chi_j|chi_o>) / a
        const double* cj = h.chi[lane];
        const double2 on = overlap3(cj[0], cj[1], cj[2], h.chi[7][0], h.chi[7][1], h.chi[7][2]);
        const double2 oo = overlap3(cj[0], cj[1], cj[2], h.chi[0][0], h.chi[0][1], h.chi[0][2]);
        cv = make_double2((-p.t * on.x + p.t * oo.x) / p.a, (-p.t * on.y + p.t * oo.y) / p.a);
        hv = hop_of(p.hop64, p.N, o, lane - 1, lk);  // Htilde_{o, l_k}
    }
    // <v|v> and <o|Htilde|v> = sum_k Htilde_{o, l_k} c_k over lanes 1..6
    double v0 = cv.x * cv.x + cv.y * cv.y;
    double2 o1 = dmul(cv, hv);
#pragma unroll
    for (int b = 4; b > 0; b >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, b);
        o1.x += __shfl_xor_sync(0xffffffffu, o1.x, b);
        o1.y += __shfl_xor_sync(0xffffffffu, o1.y, b);
    }
    // small moves: v scaled by 2^n to |v|^2 in [1/8, 1/2), so that the sums, in integers, and fixed-point
    // vectors resolve it like a large one (the two parities do not mix, so nothing else changes)
    const int e = (__double2hiint(v0) >> 20) - 1023, up = e > -800 && e < -3 ? (-2 - e) >> 1 : 0;
    const double by = __hiloint2double((1023 + up) << 20, 0);
    if (lane < 7) h.c[lane] = make_double2(cv.x * by, cv.y * by);
    if (lane < 3) h.unit[lane] = __hiloint2double((1023 - 59 - (lane == 0 ? 0 : lane == 1 ? 2 * up : up)) << 20, 0);
    if (lane == 0) {
        h.vv0 = v0;
        h.ov1 = o1;
    }
}

// Delta Omega from the CTAs' phase sums (added in one order by every CTA; an infinite
// increment marks a failed update) and the Metropolis decision, by warp 0; the caller's barrier follows.
__device__ __forceinline__ void pk_decide(const Params& p, PkHead& h, int rank, long long q)
{
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    double s = 0.0, mx = 0.0;
    for (int c = lane; c < p.ncta; c += 32) {
        s += __ldcg(p.qpart + 2 * c);
        mx = fmax(mx, __ldcg(p.qpart + 2 * c + 1));
    }
#pragma unroll
    for (int b = 16; b > 0; b >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, b);
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, b));
    }
    if (lane == 0) {
        const double dom = p.a / p.K * s;
        int acc = 0;
        if (p.mode == MODE_SWEEP) acc = exp(-p.beta * dom) > h.draw[2];
        h.acc = acc;
        h.stop = isinf(mx);
        if (rank == 0) {
            const long long slot = (p.mode == MODE_SWEEP) ? q : 0;
            p.domega_out[slot] = dom;
            if (p.maxinc_out) p.maxinc_out[slot] = mx;
            if (p.mode == MODE_SWEEP && p.dec_out) p.dec_out[q] = (unsigned char)acc;
        }
    }
}

// |sum_i S_i| / N after a sweep; sync(where): the chain's barrier.
template <int NT, class Sync>
__device__ __forceinline__ bool pk_magnetisation(const Params& p, int rank, long long nmag, Sync& sync)
{
    const int C = p.ncta, N = p.N;
    magnetisation_partial<NT>(p, (int)((long long)rank * N / C), (int)((long long)(rank + 1) * N / C), rank);
    if (!sync(6)) return false;
    if (rank == 0 && threadIdx.x == 0) {
        double X = 0.0, Y = 0.0, Z = 0.0;
        for (int c = 0; c < C; ++c) {
            X += __ldcg(p.magpart + 3 * c);
            Y += __ldcg(p.magpart + 3 * c + 1);
            Z += __ldcg(p.magpart + 3 * c + 2);
        }
        p.mag_out[nmag] = sqrt(X * X + Y * Y + Z * Z) / N;
    }
    return sync(7);  // magpart is read before the next sweep's partials
}

// ---------------------------------------------------------------------------
// one chain on a cluster
// ---------------------------------------------------------------------------
template <class R> constexpr int pk_threads() { return sizeof(R) == 4 ? kPkThreads32 : kPkThreads64; }

template <class R> __device__ __forceinline__ void pk_run_chain(const Params& p, const int rank, char* smem)
{
    constexpr int NT = pk_threads<R>(), NW = NT / 32;
    __shared__ PkSums<R, NW> sums;
    __shared__ PkHead head;
    const int tid = threadIdx.x, N = p.N, C = p.ncta;
    __shared__ PkTile t;
    if (tid == 0) t = pk_tile<R>(p, rank, smem);
    __syncthreads();
    double2* work = (double2*)smem;
    const int work_n = (int)((t.bonds - smem) / (int)sizeof(double2));
    auto sync = [&](int) {
        if (C > 1) cooperative_groups::this_cluster().sync();
        else __syncthreads();
        return true;
    };
    sync(0);  // every CTA of the cluster has started before any remote store

    const long long nupd = (p.mode == MODE_SWEEP) ? p.n_updates : 1;
    long long nmag = 0;
    unsigned long long nacc = 0;
    bool reload = true;
    for (long long q = 0; q < nupd; ++q) {
        const unsigned long long upd = p.upd0 + (unsigned long long)q;
        const int o = (p.mode == MODE_SWEEP) ? (int)(upd % (unsigned long long)N) : (int)p.site;
        pk_setup(p, head, o, upd);
        if (reload) pk_load_bonds<R, NT>(p, t);
        reload = false;
        __syncthreads();
        if constexpr (sizeof(R) == 4) {
            const int ncol = t.half * t.PY, room = NT / ncol;
            const int nseg0 = min(room, t.PZ), S = (t.PZ + nseg0 - 1) / nseg0, nseg = (t.PZ + S - 1) / S;
            if (S == 1) pk32_steps<NT, 1, true>(p, t, head.loc, head.c, sums, nseg);
            else if (S == 2) pk32_steps<NT, 2, true>(p, t, head.loc, head.c, sums, nseg);
            else if (S == 3) pk32_steps<NT, 3, false>(p, t, head.loc, head.c, sums, nseg);
            else pk32_steps<NT, 4, false>(p, t, head.loc, head.c, sums, nseg);
        } else {
            pk64_steps<NT>(p, t, head.loc, head.c, sums);
        }
        sync(1);
        pk_tail_fft<NT>(p, rank, C, work, work_n, head);
        sync(2);
        pk_tail_clear<NT>(p, rank, C);
        pk_tail_phase<NT>(p, rank, C, (double*)work);
        sync(3);
        pk_decide(p, head, rank, q);
        __syncthreads();
        if (p.mode == MODE_DELTA) break;
        if (head.acc) {
            ++nacc;
            reload = true;
            if (rank == 0 && tid < 7) patch_site(p, o, head.loc, head.draw[0], head.draw[1], tid);
            sync(5);
        }
        if ((upd + 1ull) % (unsigned long long)N == 0ull) {
            pk_magnetisation<NT>(p, rank, nmag, sync);
            ++nmag;
        }
    }
    if (rank == 0 && tid == 0 && p.mode == MODE_SWEEP) {
        *p.n_acc = nacc;
        *p.n_mag = nmag;
    }
    sync(0);  // no CTA leaves while another may still write into its shared memory
}

// A batch of chains, one thread-block cluster per chain (cluster size = the
// chains' p.ncta).
template <class R>
__global__ void __launch_bounds__(pk_threads<R>(), 1) gfmc_packed_cluster(const TeamJob* __restrict__ jobs)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params sp;
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int job = (int)(blockIdx.x / cl.dim_blocks().x);
    if (threadIdx.x == 0) sp = jobs[job].p;
    __syncthreads();
    pk_run_chain<R>(sp, (int)cl.block_rank(), (char*)dyn_all);
}

}  // namespace gfmc
