// gfmc_team.cuh -- even lattices on the packed recursion (gfmc_packed.cuh) on one CTA
// or on a team of CTAs, and the kernel of a batch of teams.
//
// Bound: chains of a few sites per thread by the latency of a step -- shared
// loads, the products of the stencil, a store, one CTA barrier -- so bonds and both
// vectors stay in registers, a step's products are formed under the next step's
// loads, and they are added over the threads by the eight steps, not by a warp
// reduction in each.  us per step (a default chain, before the packed recursion on one
// CTA and now): FP32 on a team of one CTA, L = 8 0.97 -> 0.39, L = 4 0.77 -> 0.27 (0.62 in the
// fixed point it takes for its accuracy); FP64
// alone, L = 4 0.82 (a cluster) -> 0.30; the tail of a team's update 49 -> 29 us.
// Larger tiles by the latency of their loads and index arithmetic, two warps per
// sub-partition, with the bonds in shared memory: us per step (an update of M = 1024 over its
// 511 steps) L = 16 on one CTA 4.2, L = 24 on three 6.9, L = 32 on eight 6.9.  Four sites per
// pass spill.
#pragma once

#include "gfmc_packed.cuh"

namespace gfmc {

__device__ __forceinline__ float2 lds_v(unsigned a, float2)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double2 lds_v(unsigned a, double2)
{
    double2 v;
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float4 lds_v(unsigned a, float4)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int4 lds_v(unsigned a, int4) { return lds4(a); }
__device__ __forceinline__ void sts_v(unsigned a, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts_v(unsigned a, double2 v)
{
    asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void sts_v(unsigned a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void sts_v(unsigned a, int4 v) { sts4(a, v); }

// the chain's sums of step m, value v, in units of 2^-60 (as pk_flush)
__device__ __forceinline__ void pk_add(const Params& p, int m, int v, long long q)
{
    atomicAdd(p.gram + (size_t)(m - 1) * kEntries + (v < 2 ? v : v + 4), (unsigned long long)q);
}

// What a site adds to the sums: cur = S_m and nxt = S_{m+1} there.
template <class R, class R2>
__device__ __forceinline__ void add_site(R (&acc)[4], bool class_a, R2 cur, R2 nxt)
{
    const R2 a = class_a ? cur : c_make<R2>(0, 0), b = class_a ? c_make<R2>(0, 0) : cur;
    acc[0] = fma(a.x, a.x, fma(a.y, a.y, acc[0]));
    acc[1] = fma(b.x, b.x, fma(b.y, b.y, acc[1]));
    acc[2] = fma(a.x, nxt.x, fma(a.y, nxt.y, acc[2]));
    acc[3] = fma(a.x, nxt.y, fma(-a.y, nxt.x, acc[3]));
}

// A thread's sums of a step, for tiles of any number of sites: FP64 terms in FP64; of
// FP32, each site's terms (|S_m|^2, Re and Im of the product) as integers (fix_term), so
// that neither the tile, nor the order of its sites, nor the warps change a bit of them.
// Added in FP32 over a tile and a warp they cost more accuracy than the recursion: rms
// error of Delta Omega at M = 256, uniform spins, L = 16 on two CTAs 2.4e-8, so 1.1e-8, L = 32
// on four 2.2e-8 and 1.1e-8.  The twenty instructions per site cost 5 to 15 % of a step.
template <class R> struct SiteSums {
    R v[4] = {0, 0, 0, 0};
    __device__ __forceinline__ void add(bool class_a, double2 cur, double2 nxt) { add_site(v, class_a, cur, nxt); }
    __device__ __forceinline__ R reduce(const Params&, int, int lane) const { return warp_reduce_scatter4(v, lane); }
};
template <> struct SiteSums<float> {
    int hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
    unsigned bad = 0;
    __device__ __forceinline__ void add(bool class_a, float2 cur, float2 nxt)
    {
        const float2 a = class_a ? cur : make_float2(0.f, 0.f);
        const FixTerm u = fix_term(fmaf(cur.x, cur.x, __fmul_rn(cur.y, cur.y)), bad);
        FixTerm x, y;
        fix_terms(make_float2(fmaf(a.x, nxt.x, __fmul_rn(a.y, nxt.y)), fmaf(a.x, nxt.y, -__fmul_rn(a.y, nxt.x))), x, y, bad);
        if (class_a) {
            hi[0] += u.hi;
            lo[0] += u.lo;
        } else {
            hi[1] += u.hi;
            lo[1] += u.lo;
        }
        hi[2] += x.hi;
        lo[2] += x.lo;
        hi[3] += y.hi;
        lo[3] += y.lo;
    }
    __device__ __forceinline__ long long reduce(const Params& p, int m, int lane) const
    {
        if (bad & kFixBad) set_error(p, ERR_NUMERIC, 90, m);
        const long long q[4] = {fix_value(hi[0], lo[0]), fix_value(hi[1], lo[1]), fix_value(hi[2], lo[2]),
                                fix_value(hi[3], lo[3])};
        return warp_reduce_scatter4(q, lane);
    }
};

// ---------------------------------------------------------------------------
// one CTA, a few sites per thread
// ---------------------------------------------------------------------------
// The sites stand class by class: site i at (parity of i) N / 2 + i / 2, so that the
// sites a warp reads are contiguous and its threads mostly of one class.  FP32, or
// FP64 in fixed point.  buf: two vectors of N values; ring: kPkRing steps of one item
// per thread (FP32: its four sums; FP64: one of the four sums over four threads).
template <class R> struct OneCta {
    static constexpr bool kFix = sizeof(R) == 8;
    using V = std::conditional_t<kFix, int4, float2>;
    static constexpr int kItem = kFix ? 8 : 16;
};

// Add the sums of the steps f0 .. f1 (at most kPkGroup) over the threads, a warp per step, as
// integers (FP32: of each thread's up to four sites; eight threads' in FP32 first cost, rms error of
// Delta Omega over 192 updates at L = 8, M = 256, uniform spins, 1.9e-8, now 1.1e-8).
template <class R>
__device__ __forceinline__ void one_cta_flush(const Params& p, unsigned ring, int ntr, int f0, int f1, int warp, int lane)
{
    const int f = f0 + warp;
    if (warp >= kPkGroup || f > f1) return;
    const unsigned at = ring + (unsigned)OneCta<R>::kItem * (unsigned)((f & (kPkRing - 1)) * ntr + lane);
    long long q = 0;
    if constexpr (sizeof(R) == 4) {
        int hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
        unsigned bad = 0;
        for (int j = 0; j < ntr; j += 32) {
            const float4 b = lds_v(at + 16u * j, float4());
            FixTerm t[4];
            fix_terms(make_float2(b.x, b.y), t[0], t[1], bad);
            fix_terms(make_float2(b.z, b.w), t[2], t[3], bad);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                hi[k] += t[k].hi;
                lo[k] += t[k].lo;
            }
        }
        if (bad & kFixBad) set_error(p, ERR_NUMERIC, 90, f);
        const long long s[4] = {fix_value(hi[0], lo[0]), fix_value(hi[1], lo[1]), fix_value(hi[2], lo[2]),
                                fix_value(hi[3], lo[3])};
        q = warp_reduce_scatter4(s, lane);
    } else {
        for (int j = 0; j < ntr; j += 32) {
            const int2 b = lds2(at + 8u * j);
            q += (long long)(((unsigned long long)(unsigned)b.y << 32) | (unsigned)b.x);
        }
        q += __shfl_xor_sync(0xffffffffu, q, 4);
        q += __shfl_xor_sync(0xffffffffu, q, 2);
        q += __shfl_xor_sync(0xffffffffu, q, 1);
    }
    if ((lane & 7) == 0) pk_add(p, f, lane >> 3, q);
}

// FP64: the thread's four sums into its ring item, two rounds of the butterfly: one of the
// four over four threads
__device__ __forceinline__ void one_cta_item(const Pk64Sums& acc, unsigned at, int lane)
{
    const bool u16 = lane & 16, u8 = lane & 8;
    const long long a = (u16 ? acc.v[2] : acc.v[0]) + __shfl_xor_sync(0xffffffffu, u16 ? acc.v[0] : acc.v[2], 16);
    const long long b = (u16 ? acc.v[3] : acc.v[1]) + __shfl_xor_sync(0xffffffffu, u16 ? acc.v[1] : acc.v[3], 16);
    const long long s = (u8 ? b : a) + __shfl_xor_sync(0xffffffffu, u8 ? a : b, 8);
    sts2(at, make_int2((int)(unsigned)s, (int)(unsigned)(s >> 32)));
}

// The site at place pos (class by class), its class and its neighbours' shared addresses.
template <class V>
__device__ __forceinline__ int one_cta_site(const Params& p, int pos, unsigned buf, int& c, int (&n6)[6], unsigned (&nb)[6])
{
    const int L = p.L, H2 = p.N / 2, half = L / 2;
    c = pos >= H2 ? 1 : 0;
    const int g = pos - c * H2;
    const int r = (int)__umulhi((unsigned)(2 * g), p.divL), z = (int)__umulhi((unsigned)r, p.divL), y = r - z * L;
    const int i = r * L + 2 * (g - r * half) + ((c + y + z) & 1);
    site_nbrs(i, L, p.divL, p.divLL, n6);
#pragma unroll
    for (int d = 0; d < 6; ++d) nb[d] = buf + (unsigned)sizeof(V) * (unsigned)((1 - c) * H2 + (n6[d] >> 1));
    return i;
}

// The steps of one update: up to KR sites per thread, site pos = tid + k NT.  Not
// inlined: the registers that live across the tail stay out of the loop.
template <class R, int NT, int KR>
__device__ __noinline__ void one_cta_steps(const Params& p, const PkHead& head, unsigned buf, unsigned ring, int ntr)
{
    static_assert(NT / 32 >= kPkGroup, "a warp per flushed step");
    using V = typename OneCta<R>::V;
    constexpr bool kFix = OneCta<R>::kFix;
    using B = std::conditional_t<kFix, PkBond64, float2>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = p.N, L = p.L, nsteps = p.nsteps;
    const int lo = head.loc[0];
    const int par_o = (lo % L + (lo / L) % L + lo / (L * L)) & 1;
    const unsigned vecB = (unsigned)(sizeof(V) * N);
    V cur[KR], prv[KR];
    B h[KR][6];
    unsigned nb[KR][6];  // shared addresses of the neighbours in buffer 0
    int cls[KR];         // class, counted from o's
#pragma unroll
    for (int k = 0; k < KR; ++k) {
        const int pos = tid + k * NT;
        const bool on = pos < N;
        int c, n6[6];
        const int i = one_cta_site<V>(p, on ? pos : 0, buf, c, n6, nb[k]);
        cls[k] = c ^ par_o;
        const double2 s = pk_s0(i, head.loc, head.c);
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            if constexpr (kFix) {
                const double2 b = hop_of(p.hop64, N, i, d, n6[d]);
                const int4 w = pk_limbs(__double2ll_rn(b.x * 0x1p61), __double2ll_rn(b.y * 0x1p61));
                h[k][d] = on ? PkBond64{w.x, w.y, w.z, w.w} : PkBond64{0, 0, 0, 0};
            } else {
                const float2 b = hop_of(p.hop32, N, i, d, n6[d]);
                h[k][d] = on ? make_float2(2.f * b.x, 2.f * b.y) : make_float2(0.f, 0.f);
            }
        }
        if constexpr (kFix) {
            prv[k] = make_int4(0, 0, 0, 0);
            cur[k] = on ? pk_limbs(__double2ll_rn(s.x * 0x1p60), __double2ll_rn(s.y * 0x1p60)) : prv[k];
        } else {
            prv[k] = make_float2(0.f, 0.f);
            cur[k] = on ? make_float2((float)s.x, (float)s.y) : prv[k];
        }
        if (on) sts_v(buf + (unsigned)sizeof(V) * pos, cur[k]);
    }
    __syncthreads();
    const bool live = (tid & ~31) < N;
    for (int m = 0; m <= nsteps + 1; ++m) {
        // buffers of S_m and (in the place of S_{m-1}) S_{m+1}
        const unsigned rd = (m & 1) ? vecB : 0u, wr = vecB - rd;
        if (live) {
            // at most two sites' loads at a time (registers)
            constexpr int KB = KR < 2 ? KR : 2;
            V v[KB][6];
            auto load = [&](int k0) {
#pragma unroll
                for (int k = 0; k < KB; ++k)
#pragma unroll
                    for (int d = 0; d < 6; ++d) v[k][d] = lds_v(nb[k0 + k][d] + rd, V());
            };
            if (m <= nsteps) load(0);
            if (m >= 2) {
                // the products of step m - 1: S_{m-1} = prv, S_m = cur
                const unsigned at = ring + (unsigned)OneCta<R>::kItem * (unsigned)(((m - 1) & (kPkRing - 1)) * ntr + tid);
                if constexpr (kFix) {
                    Pk64Sums acc;
#pragma unroll
                    for (int k = 0; k < KR; ++k) acc.add(prv[k], cur[k], ((cls[k] ^ (m - 1)) & 1) == 0);
                    acc.put();
                    one_cta_item(acc, at, lane);
                } else {
                    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int k = 0; k < KR; ++k) add_site(acc, ((cls[k] ^ (m - 1)) & 1) == 0, prv[k], cur[k]);
                    sts_v(at, make_float4(acc[0], acc[1], acc[2], acc[3]));
                }
            }
            if (m <= nsteps) {
#pragma unroll
                for (int k = 0; k < KR; ++k) {
                    if (k > 0 && k % KB == 0) load(k);
                    V nx;
                    if constexpr (kFix) {
                        long long re = pk_join(prv[k].x, prv[k].y), im = pk_join(prv[k].z, prv[k].w);
                        pk64_stencil(v[k % KB], h[k], re, im);
                        if (m == 0) {  // S_1 = Htilde S_0
                            re = (re + 1) >> 1;
                            im = (im + 1) >> 1;
                        }
                        nx = pk_limbs(re, im);
                    } else {
                        const float2 s = bond_sum6(h[k], v[k % KB]);
                        nx = m == 0 ? make_float2(0.5f * s.x, 0.5f * s.y) : make_float2(s.x - prv[k].x, s.y - prv[k].y);
                    }
                    const int pos = tid + k * NT;
                    if (pos < N) sts_v(buf + wr + (unsigned)sizeof(V) * pos, nx);
                    prv[k] = cur[k];
                    cur[k] = nx;
                }
            }
        }
        // the steps m - 9 .. m - 2: their sums were written before the last barrier
        if (m > kPkGroup && ((m - 2) & (kPkGroup - 1)) == 0)
            one_cta_flush<R>(p, ring, ntr, m - 1 - kPkGroup, m - 2, warp, lane);
        __syncthreads();
    }
    one_cta_flush<R>(p, ring, ntr, (nsteps - 1) / kPkGroup * kPkGroup + 1, nsteps, warp, lane);
}

// FP64 chains alone on a CTA: NM threads advance the sites, SPL threads per site (SPL = 2: bit
// 0 the real or imaginary part), and eight more warps form the sums.  The sums of a step are
// a third of its instructions; here the step is six shared loads, the stencil's products, a
// store and a barrier of the advancing warps.  S_m stays in a ring of kOneCtaHist vectors: every
// kPkGroup steps all warps meet, and a helper warp per step forms the products of one of the
// last eight while the next eight are computed.
template <int SPL>
__device__ __noinline__ void one_cta_advance(const Params& p, const PkHead& head, unsigned buf, int nm, int nt)
{
    const int tid = threadIdx.x, N = p.N, nsteps = p.nsteps;
    const unsigned vecB = 16u * (unsigned)N;
    const int c = SPL > 1 ? tid & 1 : 0, pos = tid / SPL;
    const bool on = pos < N;
    int cl, n6[6];
    unsigned nb[6];
    const int i = one_cta_site<int4>(p, on ? pos : 0, buf, cl, n6, nb);
    // SPL = 1: the bonds; SPL = 2: the part's factors of the neighbours' real and imaginary parts
    PkBond64 h[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        const double2 b = hop_of(p.hop64, N, i, d, n6[d]);
        const int4 w = pk_limbs(__double2ll_rn(b.x * 0x1p61), __double2ll_rn(b.y * 0x1p61));
        if (SPL == 1) h[d] = PkBond64{w.x, w.y, w.z, w.w};
        else h[d] = c ? PkBond64{w.z, w.w, w.x, w.y} : PkBond64{w.x, w.y, -w.z, -w.w};
    }
    const double2 s0 = pk_s0(i, head.loc, head.c);
    int4 cur = pk_limbs(__double2ll_rn(s0.x * 0x1p60), __double2ll_rn(s0.y * 0x1p60)), prv = make_int4(0, 0, 0, 0);
    if (SPL > 1) cur = c ? make_int4(cur.z, cur.w, 0, 0) : make_int4(cur.x, cur.y, 0, 0);
    const unsigned own = buf + 16u * (unsigned)pos + 8u * (unsigned)c;
    auto put = [&](unsigned at, int4 v) {
        if (!on) return;
        if (SPL == 1) sts4(own + at, v);
        else sts2(own + at, make_int2(v.x, v.y));
    };
    put(0u, cur);
    for (int m = 0; m <= nsteps; ++m) {
        const unsigned rd = (unsigned)(m & (kOneCtaHist - 1)) * vecB, wr = (unsigned)((m + 1) & (kOneCtaHist - 1)) * vecB;
        if (m > kPkGroup && (m & (kPkGroup - 1)) == 1) nbar_sync(2, nt);
        else nbar_sync(1, nm);
        int4 v[6];
#pragma unroll
        for (int d = 0; d < 6; ++d) v[d] = lds4(nb[d] + rd);
        int4 nx;
        if constexpr (SPL == 1) {
            long long re = pk_join(prv.x, prv.y), im = pk_join(prv.z, prv.w);
            pk64_stencil(v, h, re, im);
            if (m == 0) {  // S_1 = Htilde S_0
                re = (re + 1) >> 1;
                im = (im + 1) >> 1;
            }
            nx = pk_limbs(re, im);
        } else {
            long long A = -(long long)prv.y, B = 0, A2 = 0, B2 = 0;
            pk_wide(A, prv.x, -(1 << 30));
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                pk_mac(A, B, h[d].rh, h[d].rl, v[d].x, v[d].y);
                pk_mac(A2, B2, h[d].ih, h[d].il, v[d].z, v[d].w);
            }
            long long s = pk_value(A + A2, B + B2);
            if (m == 0) s = (s + 1) >> 1;
            nx = make_int4((int)((s + (1ll << 29)) >> 30), (int)((unsigned)s << 2) >> 2, 0, 0);
        }
        put(wr, nx);
        prv = cur;
        cur = nx;
    }
    nbar_sync(2, nt);
}

// The helper warps' part, warp w < kPkGroup.
static __device__ __noinline__ void one_cta_products(const Params& p, const PkHead& head, unsigned buf, int w, int nt)
{
    const int lane = threadIdx.x & 31, N = p.N, L = p.L, H2 = N / 2;
    const unsigned vecB = 16u * (unsigned)N;
    const int lo = head.loc[0];
    const int par_o = (lo % L + (lo / L) % L + lo / (L * L)) & 1;
    for (int f0 = 1; f0 <= p.nsteps; f0 += kPkGroup) {
        nbar_sync(2, nt);
        const int f = f0 + w;
        if (f > p.nsteps) continue;
        const unsigned a = buf + (unsigned)(f & (kOneCtaHist - 1)) * vecB, b = buf + (unsigned)((f + 1) & (kOneCtaHist - 1)) * vecB;
        Pk64Sums acc;
        int n = 0;
        for (int q = lane; q < N; q += 32) {
            acc.add(lds4(a + 16u * q), lds4(b + 16u * q), (((q >= H2 ? 1 : 0) ^ par_o ^ f) & 1) == 0);
            if (++n % kPkPut == 0) acc.put();
        }
        acc.put();
        const long long s = warp_reduce_scatter4(acc.v, lane);
        if ((lane & 7) == 0) pk_add(p, f, lane >> 3, s);
    }
}

// ---------------------------------------------------------------------------
// any number of sites on a team of CTAs
// ---------------------------------------------------------------------------
// The sums of a group of kPkGroup steps by step, warp and value; they are added over the
// warps together, a warp per step.
template <class R> struct StepSums {
    std::conditional_t<sizeof(R) == 4, long long, R> w[kPkGroup][kWarps][4];
};

// Add the sums of the steps f0 .. f1 (one group at most) over the warps, in units of 2^-60.
template <class R>
__device__ __forceinline__ void add_step_sums(const Params& p, const StepSums<R>& sums, int f0, int f1, int warp, int lane)
{
    const int f = f0 + warp;
    if (f > f1) return;
    const auto x = sums.w[f & (kPkGroup - 1)][lane & 7][lane >> 3];
    long long q;
    if constexpr (sizeof(R) == 4) {
        q = x;
    } else {
        bool ok;
        q = fixed58(4.0 * x, ok);
        if (!ok) set_error(p, ERR_NUMERIC, 90, f);
        q = ok ? q : 0;
    }
    q += __shfl_xor_sync(0xffffffffu, q, 4);
    q += __shfl_xor_sync(0xffffffffu, q, 2);
    q += __shfl_xor_sync(0xffffffffu, q, 1);
    if ((lane & 7) == 0) pk_add(p, f, lane >> 3, q);
}

// S_0 = e_o + v and S_1 = Htilde S_0 at site i.
template <class R2>
__device__ __forceinline__ void first_vectors(const Params& p, const R2* hop, const int* s_loc, const R2 (&cv6)[6],
                                              int i, R2& r0, R2& r1)
{
    int nb[6];
    site_nbrs(i, p.L, p.divL, p.divLL, nb);
    r0 = c_make<R2>(i == s_loc[0] ? 1 : 0, 0);
    r1 = c_make<R2>(0, 0);
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (i == s_loc[k + 1]) {
            r0.x += cv6[k].x;
            r0.y += cv6[k].y;
        }
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        bool hit = false;
#pragma unroll
        for (int k = 0; k < kVec; ++k) hit |= nb[d] == s_loc[k];
        if (hit) {
            const R2 h = hop_of(hop, p.N, i, d, nb[d]);
            if (nb[d] == s_loc[0]) {
                r1.x += h.x;
                r1.y += h.y;
            }
#pragma unroll
            for (int k = 0; k < 6; ++k)
                if (nb[d] == s_loc[k + 1]) c_fma(r1, h, cv6[k]);
        }
    }
}

template <class R> __device__ __forceinline__ const typename Cx<R>::T* hop_table(const Params& p)
{
    if constexpr (sizeof(R) == 8) return (const double2*)p.hop64;
    else return (const float2*)p.hop32;
}

// A team CTA of any number of sites.
// WIN: S_m and S_{m-1} of the CTA's sites and of the planes before and after
// them stand in shared memory (buf: two buffers of W sites; behind them, in what is
// left of `bytes`, the forward bonds of the tile's first Tb sites and the z bonds of
// the plane before it); only those planes -- 2 L^2 sites -- come from the other
// CTAs' stores each step.  The sites
// within a plane of the tile's ends go first and are published before the
// others are computed, so the neighbours' wait overlaps the rest of the step.
// Without WIN (tiles below a plane, or too large for shared memory) all values
// are read from global memory, in the same order.
template <class R, bool WIN, bool WIDE, bool LATE = false>
__device__ __noinline__ bool team_packed_steps(const Params& p, int cta, unsigned phase, unsigned buf, int bytes,
                                               const PkHead& head, StepSums<R>& sums)
{
    using R2 = typename Cx<R>::T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = p.N, L = p.L, LL = L * L;
    const int s0 = p.tile_start[cta], s1 = p.tile_start[cta + 1], T = s1 - s0;
    const R2* hop = hop_table<R>(p);
    const int* s_loc = head.loc;
    R2 cv6[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) cv6[k] = c_make<R2>((R)head.c[k + 1].x, (R)head.c[k + 1].y);
    const int lo = s_loc[0];
    const int par_o = (lo % L + (lo / L) % L + lo / LL) & 1;
    // whole: the buffers hold the lattice, site i at i; else site s0 - L^2 + w (mod N) at w
    const bool whole = !WIN || T + 2 * LL >= N;
    const int W = whole ? N : T + 2 * LL, base = whole ? 0 : s0 - LL;
    R2* g0 = (R2*)p.rbuf;
    R2* g1 = g0 + N;
    constexpr unsigned kB = sizeof(R2);
    const unsigned b0 = buf, b1 = buf + kB * (unsigned)W;  // WIN
    auto wrap = [&](int i) { return i < 0 ? i + N : i >= N ? i - N : i; };

    // bonds in shared memory: x and y of sites k < Tb at k, z of site k at LLw + k
    const int LLw = whole ? 0 : LL;
    const int Tb = WIN && (!whole || p.ncta == 1)
                       ? max(0, min(T, (bytes - (int)kB * (2 * W + LLw)) / (3 * (int)kB))) : 0;
    const unsigned hx = b0 + 2u * kB * (unsigned)W, hy = hx + kB * (unsigned)Tb, hz = hy + kB * (unsigned)Tb;
    if constexpr (WIN) {
        for (int k = tid; k < Tb; k += kThreads) {
            sts_v(hx + kB * k, ldcg2(hop + (s0 + k)));
            sts_v(hy + kB * k, ldcg2(hop + (N + s0 + k)));
            sts_v(hz + kB * (LLw + k), ldcg2(hop + (2 * N + s0 + k)));
        }
        if (Tb > 0)
            for (int k = tid; k < LLw; k += kThreads) sts_v(hz + kB * k, ldcg2(hop + (2 * N + wrap(s0 - LL + k))));
    }

    const int n0 = WIN ? W : T, f0 = WIN ? base : s0;
    for (int w = tid; w < n0; w += kThreads) {
        R2 r0, r1;
        first_vectors(p, hop, s_loc, cv6, wrap(f0 + w), r0, r1);
        if constexpr (WIN) {
            sts_v(b0 + kB * w, r0);
            sts_v(b1 + kB * w, r1);
        } else {
            stcg2(g0 + s0 + w, r0);
            stcg2(g1 + s0 + w, r1);
        }
    }
    if constexpr (WIN) __syncthreads();
    else publish(p, cta, phase + 1);

    // sites of the tile within a plane of its ends: [0, e0) and [e1, T).  FP64: wherever the vectors
    // stand (which the launch's other chains have a say in), as the order of the sums follows it
    constexpr bool kEnds = WIN || sizeof(R) == 8;
    const int e0 = (kEnds && p.ncta > 1 && T > 2 * LL) ? LL : T, e1 = e0 < T ? T - LL : T;
    const int parts = e0 < e1 ? 2 : 1;
    const int halo = whole ? N - T : 2 * LL;
    for (int m = 1; m <= p.nsteps; ++m) {
        const unsigned rd = (m & 1) ? b1 : b0, wr = (m & 1) ? b0 : b1;
        const R2* gr = (m & 1) ? g1 : g0;
        R2* gw = (m & 1) ? g0 : g1;
        if (!WIN || (p.ncta > 1 && m > 1)) {
            if (!wait_neighbours(p, cta, phase + (unsigned)m, 100 + m)) return false;
        }
        if constexpr (WIN) {
            if (p.ncta > 1 && m > 1) {
                for (int k = tid; k < halo; k += kThreads) {
                    // k-th site after the tile, or (k >= L^2) before it
                    const int i = whole || k < LL ? wrap(s1 + k) : wrap(s0 - 2 * LL + k);
                    const int w = whole ? i : k < LL ? LL + T + k : k - LL;
                    sts_v(rd + kB * w, ldcg2(gr + i));
                }
                __syncthreads();
            }
        }
        SiteSums<R> acc;
        struct Ops {
            R2 h[6], nv[6], cur, pv;
            int i, w, odd;
        };
        // S_m at offset off from site i (at w of the shared buffer)
        auto ld = [&](int i, int w, int off) {
            if constexpr (WIN) return lds_v(rd + kB * (unsigned)(w + off), R2());
            else return ldcg2(gr + (i + off));
        };
        auto load = [&](int k, Ops& q) {
            const int i = s0 + k;
            const int z = (int)__umulhi((unsigned)i, p.divLL), r = (int)__umulhi((unsigned)i, p.divL);
            const int x = i - r * L, y = r - z * L;
            q.i = i;
            q.w = whole ? i : k + LL;
            q.odd = x + y + z;
            const int xp = x == L - 1 ? 1 - L : 1, xm = x == 0 ? L - 1 : -1;
            const int yp = y == L - 1 ? L - LL : L, ym = y == 0 ? LL - L : -L;
            const int zm = z == 0 ? N - LL : -LL;
            const int wzp = whole && z == L - 1 ? LL - N : LL, wzm = whole ? zm : -LL;
            const int kz = whole ? k + zm : k;  // place of the lower z bond
            if (WIN && k < Tb && (unsigned)(k + xm) < (unsigned)Tb && (unsigned)(k + ym) < (unsigned)Tb && kz < LLw + Tb) {
                q.h[0] = lds_v(hx + kB * (unsigned)k, R2());
                q.h[1] = lds_v(hx + kB * (unsigned)(k + xm), R2());
                q.h[2] = lds_v(hy + kB * (unsigned)k, R2());
                q.h[3] = lds_v(hy + kB * (unsigned)(k + ym), R2());
                q.h[4] = lds_v(hz + kB * (unsigned)(LLw + k), R2());
                q.h[5] = lds_v(hz + kB * (unsigned)kz, R2());
            } else {
                q.h[0] = ldcg2(hop + i);
                q.h[1] = ldcg2(hop + (i + xm));
                q.h[2] = ldcg2(hop + (N + i));
                q.h[3] = ldcg2(hop + (N + i + ym));
                q.h[4] = ldcg2(hop + (2 * N + i));
                q.h[5] = ldcg2(hop + (2 * N + i + zm));
            }
            q.nv[0] = ld(i, q.w, xp);
            q.nv[1] = ld(i, q.w, xm);
            q.nv[2] = ld(i, q.w, yp);
            q.nv[3] = ld(i, q.w, ym);
            q.nv[4] = ld(i, q.w, wzp);
            q.nv[5] = ld(i, q.w, wzm);
            q.cur = ld(i, q.w, 0);
            if constexpr (WIN) q.pv = lds_v(wr + kB * (unsigned)q.w, R2());
            else q.pv = ldcg2(gw + i);
        };
        // LATE: the terms of the last pass's sites wait for the next pass's loads, or for the
        // publication, to be added under (tiles in global memory: us per update at M = 1024, L = 34 alone
        // 1567 -> 1496, L = 64 3065 -> 2772; with the bonds in shared memory, L = 16 on one CTA, 2169 -> 2361;
        // in a kernel of their own, kPackedTiles, L = 34 1261, L = 64 2433)
        constexpr bool kLate = LATE && WIDE && sizeof(R) == 4;
        [[maybe_unused]] R2 pc[2], pn[2];
        [[maybe_unused]] bool pa[2];
        auto late = [&]() {
            if constexpr (kLate) {
                acc.add(pa[0], pc[0], pn[0]);
                acc.add(pa[1], pc[1], pn[1]);
            }
        };
        auto step = [&](Ops& q, bool edge, int slot) {
            q.h[1].y = -q.h[1].y;  // backward bonds: the conjugates
            q.h[3].y = -q.h[3].y;
            q.h[5].y = -q.h[5].y;
            const R2 s = bond_sum6(q.h, q.nv);
            const R2 nx = c_make<R2>(fma((R)2, s.x, -q.pv.x), fma((R)2, s.y, -q.pv.y));
            if (m < p.nsteps) {
                if constexpr (WIN) sts_v(wr + kB * (unsigned)q.w, nx);
                if (!WIN || edge) stcg2(gw + q.i, nx);
            }
            const bool a = ((q.odd + par_o + m) & 1) == 0;
            if constexpr (kLate) {
                pa[slot] = a;
                pc[slot] = q.cur;
                pn[slot] = nx;
            } else {
                acc.add(a, q.cur, nx);
            }
        };
        // sites [0, n) of a list: k < j0 at k, the others at k + j1 - j0
        auto sites = [&](int n, int j0, int j1, bool edge) {
            auto at = [&](int k) { return k < j0 ? k : k + (j1 - j0); };
            if constexpr (WIDE && sizeof(R) == 4) {
                // two sites per pass, both sites' loads issued before the first use
                for (int k = tid; k < n; k += 2 * kThreads) {
                    Ops qa, qb;
                    load(at(k), qa);
                    if (k + kThreads < n) load(at(k + kThreads), qb);
                    if (k >= 2 * kThreads) late();
                    step(qa, edge, 0);
                    if (k + kThreads < n) step(qb, edge, 1);
                    else if constexpr (kLate) pc[1] = pn[1] = c_make<R2>(0, 0);
                }
            } else {
                for (int k = tid; k < n; k += kThreads) {
                    Ops q;
                    load(at(k), q);
                    step(q, edge, 0);
                }
            }
        };
        // the tile's ends, read by the other CTAs, then the sites between.  FP32: one loop;
        // with its body twice in the function, one_cta_steps of the same kernel spilled in its steps
        auto part = [&](bool ends) {
            sites(ends ? e0 + T - e1 : e1 - e0, ends ? e0 : 0, ends ? e1 : e0, ends && p.ncta > 1);
            if (ends) publish(p, cta, phase + (unsigned)m + 1u);
        };
        if constexpr (!kEnds) {
            sites(T, T, T, true);
            publish(p, cta, phase + (unsigned)m + 1u);
            if (tid < T) late();
        } else if constexpr (sizeof(R) == 4) {
#pragma unroll 1
            for (int k = 0; k < parts; ++k) part(k == 0);
        } else {
            part(true);
            if (parts > 1) part(false);
        }
        const auto s = acc.reduce(p, m, lane);
        if ((lane & 7) == 0) sums.w[m & (kPkGroup - 1)][warp][lane >> 3] = s;
        if ((m & (kPkGroup - 1)) == 0 || m == p.nsteps) {
            __syncthreads();
            add_step_sums<R>(p, sums, (m - 1) / kPkGroup * kPkGroup + 1, m, warp, lane);
            __syncthreads();
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// one chain
// ---------------------------------------------------------------------------
// A chain on the p.ncta CTAs of a team, this one its CTA `cta`.  smem: room for
// work_n double2 at least; bytes > 0: the vectors stand there too (`bytes`, at least
// team_vec_bytes), the tail's work space in their place after the steps.  USE: kTeam all paths, kOne a chain
// of at most NT sites on one CTA, kServer and kTiles no vectors in shared memory.
enum { kTeam, kOne, kServer, kTiles };
template <bool ONE> __device__ __forceinline__ bool team_sync(const Params& p, int where)
{
    if (!ONE && p.ncta > 1) return grid_barrier(p, where);
    __syncthreads();
    return true;
}

// What an update does besides its steps.
template <int NT, bool ONE>
__device__ __forceinline__ bool team_tail(const Params& p, PkHead& head, int cta, char* smem, int work_n, long long q)
{
    const int C = ONE ? 1 : p.ncta;
    if (!team_sync<ONE>(p, 1)) return false;
    pk_tail_fft<NT>(p, cta, C, (double2*)smem, work_n, head);
    if (!team_sync<ONE>(p, 2)) return false;
    pk_tail_clear<NT>(p, cta, C);
    pk_tail_phase<NT>(p, cta, C, (double*)smem);
    if (!team_sync<ONE>(p, 3)) return false;
    pk_decide(p, head, cta, q);
    __syncthreads();
    return true;
}
// the accepted move, and the magnetisation after a sweep
template <int NT, bool ONE>
__device__ __forceinline__ bool team_accept(const Params& p, PkHead& head, int cta, int o, bool sweep_done, long long nmag)
{
    if (head.acc) {
        if (cta == 0 && threadIdx.x < 7) patch_site(p, o, head.loc, head.draw[0], head.draw[1], (int)threadIdx.x);
        if (!team_sync<ONE>(p, 5)) return false;
    }
    auto sync = [&](int where) { return team_sync<ONE>(p, where); };
    return !sweep_done || pk_magnetisation<NT>(p, cta, nmag, sync);
}
template <class R, int NT, int USE>
__device__ __forceinline__ void pk_team_chain(const Params& p, const int cta, char* smem, int work_n, int bytes)
{
    __shared__ PkHead head;
    [[maybe_unused]] __shared__ StepSums<R> sums;
    const int tid = threadIdx.x, N = p.N;
    const unsigned buf = smem_u32(smem);
    const long long nupd = (p.mode == MODE_SWEEP) ? p.n_updates : 1;
    long long nmag = 0;
    unsigned long long nacc = 0;
    unsigned phase = 0;
    for (long long q = 0; q < nupd; ++q) {
        const unsigned long long upd = p.upd0 + (unsigned long long)q;
        const int o = (p.mode == MODE_SWEEP) ? (int)(upd % (unsigned long long)N) : (int)p.site;
        pk_setup(p, head, o, upd);
        __syncthreads();
        bool done = false;
        if constexpr (USE == kOne || USE == kTeam) {
            if (USE == kOne || (bytes > 0 && p.ncta == 1 && N <= one_cta_sites<R>(NT))) {
                const unsigned ring = buf + 2u * (unsigned)(sizeof(typename OneCta<R>::V) * N);
                const int ntr = one_cta_items(N, NT);
                if constexpr (USE == kOne && sizeof(R) == 8) {
                    const int spl = one_cta_parts(N), nm = (spl * N + 31) / 32 * 32, nt = nm + 32 * kPkGroup;
                    if (tid < nm) {
                        if (spl == 1) one_cta_advance<1>(p, head, buf, nm, nt);
                        else one_cta_advance<2>(p, head, buf, nm, nt);
                    } else if (tid < nt) {
                        one_cta_products(p, head, buf, (tid - nm) >> 5, nt);
                    }
                } else if (sizeof(R) == 4 && USE == kTeam && N <= kOneCtaExact) {
                    // FP32-mixed chains of the smallest lattice in fixed point as well
                    one_cta_steps<double, NT, 1>(p, head, buf, buf + 32u * (unsigned)N, ntr);
                } else if (USE == kOne || N <= NT) {
                    one_cta_steps<R, NT, 1>(p, head, buf, ring, ntr);
                }
                if constexpr (USE == kTeam) {
                    if (N > 2 * NT) {
                        if constexpr (sizeof(R) == 4) one_cta_steps<R, NT, 4>(p, head, buf, ring, ntr);
                    } else if (N > NT) {
                        one_cta_steps<R, NT, 2>(p, head, buf, ring, ntr);
                    }
                }
                done = true;
            }
        }
        if constexpr (USE == kTeam) {
            if (!done && bytes > 0) {
                if (!team_packed_steps<R, true, true>(p, cta, phase, buf, bytes, head, sums)) return;
                done = true;
            }
        }
        if constexpr (USE != kOne) {
            if (!done && !team_packed_steps<R, false, USE != kServer, USE == kTiles>(p, cta, phase, buf, 0, head, sums)) return;
        }
        phase += (unsigned)p.nsteps + 1u;
        if (!team_tail<NT, USE == kOne>(p, head, cta, smem, work_n, q)) return;
        if (p.mode == MODE_DELTA) break;
        const bool sweep_done = (upd + 1ull) % (unsigned long long)N == 0ull;
        if (head.acc || sweep_done) {
            nacc += head.acc;
            if (!team_accept<NT, USE == kOne>(p, head, cta, o, sweep_done, nmag)) return;
            nmag += sweep_done;
        }
    }
    if (cta == 0 && tid == 0 && p.mode == MODE_SWEEP) {
        *p.n_acc = nacc;
        *p.n_mag = nmag;
    }
}

// A single chain of at most NT sites on one CTA.
template <class R, int NT>
__global__ void __launch_bounds__(NT, 1) gfmc_one_cta(const Params p, int work_n)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params sp;
    if (threadIdx.x == 0) sp = p;
    __syncthreads();
    pk_team_chain<R, NT, kOne>(sp, 0, (char*)dyn_all, work_n, 1);
}

// A batch of chains, each on its own team of CTAs (jobs sorted by cta0).
// smem: bytes of dynamic shared memory, shared out chain by chain (team_smem_bytes).
// NV: the recursion of all chains, 0 when they differ; 1: all on the packed recursion; kPackedTiles:
// on it with every vector in global memory.
// With several recursions in one kernel the FP32 steps spill (seven vectors, moments
// of L = 40: 866 us, alone 720; packed, one-CTA chain of L = 8: 0.94 us per step, alone 0.45).
template <class R, int NV, bool COMP = false>
__global__ void __launch_bounds__(kThreads, 1) gfmc_team_engine(const TeamJob* __restrict__ jobs, int njobs, int smem)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params sp;
    __shared__ int s_job, s_cta, s_vs;
    if (threadIdx.x == 0) {
        int j = 0;
        while (j + 1 < njobs && jobs[j + 1].cta0 <= (int)blockIdx.x) ++j;
        // several one-CTA chains may share this CTA (same cta0): start at the first
        while (j > 0 && jobs[j - 1].cta0 == jobs[j].cta0) --j;
        s_job = j;
    }
    __syncthreads();
    using R2 = typename Cx<R>::T;
    // the chains of this CTA's team, one after another: one chain unless the
    // team is a shared one-CTA team
    auto load = [&]() {
        if (threadIdx.x == 0) {
            const int j = s_job;
            s_cta = (int)blockIdx.x - jobs[j].cta0;
            s_vs = jobs[j].vec_smem;
            sp = jobs[j].p;
        }
        __syncthreads();
    };
    auto next = [&]() -> bool {
        __syncthreads();  // every thread is done with sp and the shared memory
        if (threadIdx.x == 0) {
            const int j = s_job + 1;
            s_job = (j < njobs && jobs[j].cta0 == jobs[j - 1].cta0) ? j : -1;
        }
        __syncthreads();
        return s_job >= 0;
    };
    do {
        load();
        [[maybe_unused]] double2* work = dyn_all + s_vs / (int)sizeof(double2);
        [[maybe_unused]] R2* vec = s_vs ? (R2*)dyn_all : nullptr;
        if constexpr (!COMP && NV != kVec) {
            if (NV == kPackedTiles) {
                pk_team_chain<R, kThreads, kTiles>(sp, s_cta, (char*)dyn_all, smem / (int)sizeof(double2), 0);
                continue;
            }
            if (NV == 1 || (sp.nv == 2 && sp.L % 2 == 0)) {
                pk_team_chain<R, kThreads, kTeam>(sp, s_cta, (char*)dyn_all, smem / (int)sizeof(double2), s_vs ? smem : 0);
                continue;
            }
        }
        if constexpr (NV == 2 || NV == kVec) run_chain<R, 1, NV, kThreads, true, COMP>(sp, s_cta, work, vec);
        if constexpr (NV == 0) {
            if (sp.nv == 2) run_chain<R, 1, 2, kThreads, true, COMP>(sp, s_cta, work, vec);
            else run_chain<R, 1, kVec, kThreads, true, COMP>(sp, s_cta, work, vec);
        }
    } while (next());
}

}  // namespace gfmc
