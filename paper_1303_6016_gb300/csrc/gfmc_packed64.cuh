// gfmc_packed64.cuh -- FP64 single chains on the packed recursion, small tiles:
// one chain on one thread-block cluster, or on the whole GPU.
//
// With fixed point on the integer multiplier (gfmc_packed.cuh) a step's
// arithmetic is short, and what is left is latency: the instructions of one site
// (72 multiply-adds), the sums, the exchange.  On the whole GPU a step takes 1.3 us at L = 8 and
// 16 and 1.6 us at L = 32, with 64 times the sites of L = 8: 1.2 us of it do not depend on the
// sites, and 390 instructions per site of L = 32 issue in a quarter of it.  On a cluster a step
// of L = 16 takes 1.2 us, without sums (moments, L = 12) 0.6.  A thread advances one to three
// sites with bonds, S_m and S_{m-1} in registers, or on the smallest tiles 1/2 or 1/4
// of a site (a lane forms the real or the imaginary part, with 1/4 over half of
// the bonds); it stores and sends S_{m+1} first and forms the step's sums from
// registers while the faces are on their way.  One CTA barrier per step.
//
// Exchange.  On a cluster face values go into the neighbours' rings by st.async
// and complete on the receiver's mbarrier: a cluster barrier's release arrival
// waited 400-560 cycles for the acknowledgement of plain remote stores.  On the
// whole GPU they go through global memory as self-validating words: an 8-byte
// word carries one value (62 bits) and one tag bit that alternates with every
// use of the slot, so a receiver polls the data itself and needs neither a
// flag nor a fence.
#pragma once

#include "gfmc_packed.cuh"

namespace gfmc {

constexpr int kPk64Threads = 256;
constexpr int kNoFail = 1 << 30;

// a site of the tile
struct __align__(8) PkRec {
    unsigned short at;             // index in a ring buffer
    unsigned char y, z, col, xp, xm;  // row, and the columns (even sites first) of the site and its x-neighbours
    unsigned char fl;              // 1: y = 0, 2: y = PY - 1, 4: z = 0, 8: z = PZ - 1, 16: odd parity
};

// Face values over distributed shared memory.  mb: this CTA's two mbarriers,
// barrier m & 1 for the faces of S_m; each phase takes one arrival that states
// the bytes of the faces (bytes).  The re-arming for S_{m+2} may come after some of its
// data: the phase cannot complete before the arrival.  A neighbour sends
// S_{m+2} only after it received S_{m+1} from this CTA, which was sent after
// the phase of S_m completed here.
// A wait that runs out records the error.  The thread then neither waits, sends nor
// arms again -- its next wait on the same barrier would be for a phase after the one that
// did not complete, and try_wait reports such a phase as passed -- and so does its
// CTA from the next step = 7 mod 8 on.  The CTA runs the same sequence of barriers as
// the others to the end of the update, where the cluster leaves the launch together.
struct PkAsyncEx {
    static constexpr bool kAbort = false;
    const PkTile& t;
    const Params& p;
    unsigned mb, m_ym, m_yp, m_zm, m_zp;
    unsigned bytes, yB, zB;
    int last;  // the last step whose values are sent
    unsigned ph;  // values sent before this update (an even number)
    unsigned faces;  // the faces that are sent: none from CTA 0 under the stall hook
    bool dead = false;
    __device__ __forceinline__ PkAsyncEx(const PkTile& t_, const Params& p_, unsigned mb_, unsigned ph_)
        : t(t_), p(p_), mb(mb_), ph(ph_)
    {
        m_ym = cluster_addr(mb, (t.cy + t.Cy - 1) % t.Cy + t.cz * t.Cy);
        m_yp = cluster_addr(mb, (t.cy + 1) % t.Cy + t.cz * t.Cy);
        m_zm = cluster_addr(mb, t.cy + ((t.cz + t.Cz - 1) % t.Cz) * t.Cy);
        m_zp = cluster_addr(mb, t.cy + ((t.cz + 1) % t.Cz) * t.Cy);
        bytes = t.rowB * (unsigned)((t.Cy > 1 ? 2 * t.PZ : 0) + (t.Cz > 1 ? 2 * t.PY : 0));
        last = p.nsteps;
        faces = p.stall && bytes && t.rank == 0 ? 0u : 15u;
        yB = t.rowB * (unsigned)t.PY;
        zB = t.rowB * (unsigned)(t.zstr * t.PZ);
    }
    __device__ __forceinline__ void init() const
    {
        for (int b = 0; b < 2; ++b) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb + 8u * b) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        arm(0);
        arm(1);
    }
    __device__ __forceinline__ void arm(int b) const
    {
        if (bytes)
            asm volatile("mbarrier.arrive.expect_tx.relaxed.cta.shared::cta.b64 _, [%0], %1;" ::"r"(mb + 8u * b), "r"(bytes)
                         : "memory");
    }
    // where a site's values go besides its own ring slot: offsets from the
    // neighbours' rings (shared::cluster) or, where the pencil is its own
    // neighbour, from the own ring; faces the site has not are masked
    struct Target {
        unsigned fl, o;
    };
    __device__ __forceinline__ Target target(const PkRec& r, int c) const { return {r.fl & faces, 16u * r.at + 8u * (unsigned)c}; }
    static __device__ __forceinline__ void send(unsigned on, unsigned a, int2 v, unsigned m)
    {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
            " @p st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.s32 [%0], {%1, %2}, [%3];\n}" ::"r"(a),
            "r"(v.x), "r"(v.y), "r"(m), "r"(on)
            : "memory");
    }
    static __device__ __forceinline__ void send(unsigned on, unsigned a, int4 v, unsigned m)
    {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %6, 0;\n"
            " @p st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.s32 [%0], {%1, %2, %3, %4}, [%5];\n}" ::"r"(a),
            "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(m), "r"(on)
            : "memory");
    }
    static __device__ __forceinline__ void keep(unsigned on, unsigned a, int4 v)
    {
        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n @p st.shared.v4.s32 [%0], {%1, %2, %3, %4};\n}" ::"r"(a),
                     "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(on)
                     : "memory");
    }
    static __device__ __forceinline__ void keep(unsigned on, unsigned a, int2 v)
    {
        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p st.shared.v2.s32 [%0], {%1, %2};\n}" ::"r"(a), "r"(v.x),
                     "r"(v.y), "r"(on)
                     : "memory");
    }
    // one part of a site's S_m, or the whole (in the ring buffer at offset buf)
    template <class W> __device__ __forceinline__ void push(int m, unsigned buf, const Target& g, W v) const
    {
        if (g.fl == 0 || dead || m > last) return;  // S_{M/2} is read by no stencil
        const unsigned a = buf + g.o, b = 8u * (unsigned)(m & 1);
        if (t.Cy == 1) {
            keep(g.fl & 1, t.ring + a + yB, v);
            keep(g.fl & 2, t.ring + a - yB, v);
        } else {
            send(g.fl & 1, t.r_ym + a + yB, v, m_ym + b);
            send(g.fl & 2, t.r_yp + a - yB, v, m_yp + b);
        }
        if (t.Cz == 1) {
            keep(g.fl & 4, t.ring + a + zB, v);
            keep(g.fl & 8, t.ring + a - zB, v);
        } else {
            send(g.fl & 4, t.r_zm + a + zB, v, m_zm + b);
            send(g.fl & 8, t.r_zp + a - zB, v, m_zp + b);
        }
    }
    __device__ __forceinline__ void push(int m, unsigned buf, const Target& g, long long, int2 v) const { push(m, buf, g, v); }
    __device__ __forceinline__ void push(int m, unsigned buf, const Target& g, long long, long long, int4 v) const
    {
        push(m, buf, g, v);
    }
    // wait for the faces of S_m; false: the wait ran out
    __device__ __forceinline__ bool receive(int m, unsigned)
    {
        if (!bytes || dead) return true;
        const bool ok = vc_wait(mb + 8u * (unsigned)(m & 1), ((ph + (unsigned)m) >> 1) & 1u, p.budget);
        if (!ok) {
            set_error(p, ERR_TIMEOUT, 400, m);
            dead = true;
        }
        return ok;
    }
    // ok: this thread's wait for S_m ended, so the phase is complete and takes the next arrival
    __device__ __forceinline__ void received(int m, bool ok) const
    {
        if (threadIdx.x == 0 && ok && !dead) arm(m & 1);
    }
    static __device__ __forceinline__ bool vc_wait(unsigned a, unsigned parity, long long budget)
    {
        unsigned done;
        long long t0 = 0;
        for (int n = 0;; ++n) {
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                " selp.u32 %0, 1, 0, p;\n}"
                : "=r"(done)
                : "r"(a), "r"(parity)
                : "memory");
            if (done) return true;
            if (n == 0) t0 = clock64();
            else if (clock64() - t0 > budget) return false;
        }
    }
};

// Face values through global memory (a chain on p.ncta CTAs of the grid).
// CTA c's inbox: [phase & 1][face: y = -1, y = PY, z = -1, z = PZ][row][column]
// of (re, im) words, value 2 + tag.  Phases count the values sent since the
// launch began (S_0 .. S_nsteps of every update; an even number per update); the tag of phase f is
// 1 - (f >> 1) % 2 against the zeros the host wrote.  A slot is written again
// two phases later, by a neighbour that has received this CTA's values of the
// phase between, which were sent after every value of the older phase was read.
// NP: face values a thread receives per step.  NF: sides of its sites that may be
// faces (2 when every pencil has at least two rows in y and in z, else 4).  Every
// pencil has other CTAs on its four sides.
template <int NP, int NF> struct PkGridEx {
    static constexpr bool kAbort = true;
    const Params& p;
    unsigned long long* inbox;
    unsigned half;             // words of a phase's half of an inbox (4 faces)
    unsigned ring, ph;         // ph: first phase of the update
    int L, last;
    bool mute;
    unsigned nb[4];            // word offsets of the neighbours' faces this CTA writes
    unsigned src[NP], dst[NP]; // word offset from inbox in phase 0's half, and ring byte offset; src ~0u: none
    __device__ __forceinline__ PkGridEx(const PkTile& t, const Params& p_, unsigned, unsigned ph_) : p(p_), ph(ph_)
    {
        const unsigned face = 2u * (unsigned)(p.pk_rows * t.L);
        half = 4 * face;
        inbox = p.pk_inbox;
        ring = t.ring;
        L = t.L;
        last = p.nsteps;
        mute = p.stall && t.rank == 0;
        nb[0] = (unsigned)(t.cz * t.Cy + (t.cy + t.Cy - 1) % t.Cy) * 2 * half + face;             // its y = PY
        nb[1] = (unsigned)(t.cz * t.Cy + (t.cy + 1) % t.Cy) * 2 * half;                           // its y = -1
        nb[2] = (unsigned)(((t.cz + t.Cz - 1) % t.Cz) * t.Cy + t.cy) * 2 * half + 3 * face;       // its z = PZ
        nb[3] = (unsigned)(((t.cz + 1) % t.Cz) * t.Cy + t.cy) * 2 * half + 2 * face;              // its z = -1
        const int n = 2 * (t.PZ + t.PY) * t.L;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int e = (int)threadIdx.x + k * kPk64Threads;
            src[k] = ~0u;
            dst[k] = 0;
            if (e < n) {
                const int row = e / t.L, col = e - row * t.L;
                int f, r, y, z;
                if (row < 2 * t.PZ) {
                    f = row / t.PZ;
                    r = row - f * t.PZ;
                    y = f ? t.PY : -1;
                    z = r;
                } else {
                    f = (row - 2 * t.PZ) / t.PY;
                    r = row - 2 * t.PZ - f * t.PY;
                    z = f ? t.PZ : -1;
                    y = r;
                    f += 2;
                }
                src[k] = (unsigned)t.rank * 2 * half + (unsigned)f * face + 2u * (unsigned)(r * t.L + col);
                dst[k] = 16u * (unsigned)(t.ring_row(y, z) * t.L + col);
            }
        }
    }
    // word offsets of a site (part) in the neighbours' inboxes (phase 0's half; ~0u: not a face)
    struct Target {
        unsigned w[NF];
    };
    __device__ __forceinline__ Target target(const PkRec& r, int c) const
    {
        const unsigned h = 2u * r.col + (unsigned)c, ay = h + 2u * (unsigned)(r.z * L), az = h + 2u * (unsigned)(r.y * L);
        const unsigned w0 = (r.fl & 1) && !mute ? nb[0] + ay : ~0u, w1 = (r.fl & 2) && !mute ? nb[1] + ay : ~0u,
                       w2 = (r.fl & 4) && !mute ? nb[2] + az : ~0u, w3 = (r.fl & 8) && !mute ? nb[3] + az : ~0u;
        Target g;
        if constexpr (NF == 4) {
            g.w[0] = w0;
            g.w[1] = w1;
            g.w[2] = w2;
            g.w[3] = w3;
        } else {
            g.w[0] = w0 != ~0u ? w0 : w1;
            g.w[1] = w2 != ~0u ? w2 : w3;
        }
        return g;
    }
    // value and tag: the two top bits of a value (|value| <= 2^60) are equal, the
    // tag is their difference in the word
    __device__ __forceinline__ unsigned long long word(long long s, unsigned f) const
    {
        return (unsigned long long)s ^ ((unsigned long long)(~f >> 1 & 1u) << 63);
    }
    __device__ __forceinline__ void push(int m, unsigned, const Target& g, long long s, int2) const
    {
        if (m > last) return;  // S_{M/2} is read by no stencil
        const unsigned f = ph + (unsigned)m;
        const unsigned long long w = word(s, f);
        unsigned long long* base = inbox + ((f & 1) ? half : 0u);
#pragma unroll
        for (int k = 0; k < NF; ++k)
            asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0xffffffff;\n @p st.relaxed.gpu.global.u64 [%0], %1;\n}" ::"l"(
                             base + g.w[k]),
                         "l"(w), "r"(g.w[k])
                         : "memory");
    }
    __device__ __forceinline__ void push(int m, unsigned, const Target& g, long long re, long long im, int4) const
    {
        if (m > last) return;
        const unsigned f = ph + (unsigned)m;
        const unsigned long long a = word(re, f), b = word(im, f);
        unsigned long long* base = inbox + ((f & 1) ? half : 0u);
#pragma unroll
        for (int k = 0; k < NF; ++k)
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.u32 p, %3, 0xffffffff;\n @p st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n}" ::"l"(
                    base + g.w[k]),
                "l"(a), "l"(b), "r"(g.w[k])
                : "memory");
    }
    __device__ __forceinline__ bool receive(int m, unsigned buf)
    {
        const unsigned f = ph + (unsigned)m, flip = (~f >> 1 & 1u) << 31;
        const unsigned long long* base = inbox + ((f & 1) ? half : 0u);
        unsigned left = 0;
#pragma unroll
        for (int k = 0; k < NP; ++k) left |= src[k] != ~0u ? 1u << k : 0u;
        long long t0 = 0;
        for (int n = 0; left; ++n) {
            int4 w[NP];  // (low, high) words of re and im
#pragma unroll
            for (int k = 0; k < NP; ++k)
                if (left >> k & 1)
                    asm volatile("ld.relaxed.gpu.global.v4.s32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(w[k].x), "=r"(w[k].y), "=r"(w[k].z), "=r"(w[k].w)
                                 : "l"(base + src[k])
                                 : "memory");
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                // with the tag taken off, bits 63 and 62 of a value are equal
                const int a = w[k].y ^ (int)flip, b = w[k].w ^ (int)flip;
                if ((left >> k & 1) && ((a ^ (a << 1)) | (b ^ (b << 1))) >= 0) {
                    const long long re = ((long long)a << 32) | (unsigned)w[k].x, im = ((long long)b << 32) | (unsigned)w[k].z;
                    sts4(ring + buf + dst[k], pk_limbs(re, im));
                    left &= ~(1u << k);
                }
            }
            if ((n & 63) == 63) {
                if (n == 63) t0 = clock64();
                if (ld_relaxed_s32(p.err) != 0) return false;
                if (clock64() - t0 > p.budget) {
                    set_error(p, ERR_TIMEOUT, 100 + m, (int)f);
                    return false;
                }
            }
        }
        return true;
    }
    __device__ __forceinline__ void received(int, bool) const {}
};

// ---------------------------------------------------------------------------
// the steps
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pk64_records(const PkTile& t, PkRec* tab)
{
    // class by class, so that a helper warp's sites are of one class
    const int T = t.L * t.PY * t.PZ, T2 = T / 2;
    for (int s = threadIdx.x; s < T; s += kPk64Threads) {
        const int cls = s >= T2 ? 1 : 0, g = s - cls * T2, r = g / t.half, j = g - r * t.half, z = r / t.PY, y = r - z * t.PY;
        const int odd = (cls + t.y0 + y + t.z0 + z) & 1, col = odd * t.half + j, other = odd ? 0 : t.half;
        PkRec q;
        q.at = (unsigned short)(t.ring_row(y, z) * t.L + col);
        q.y = (unsigned char)y;
        q.z = (unsigned char)z;
        q.col = (unsigned char)col;
        q.xp = (unsigned char)(other + (odd ? (j == t.half - 1 ? 0 : j + 1) : j));
        q.xm = (unsigned char)(other + (odd ? j : (j == 0 ? t.half - 1 : j - 1)));
        q.fl = (unsigned char)((y == 0 ? 1 : 0) | (y == t.PY - 1 ? 2 : 0) | (z == 0 ? 4 : 0) | (z == t.PZ - 1 ? 8 : 0) |
                               (cls ? 16 : 0));
        tab[s] = q;
    }
}

// A thread's part of a site.  SPL = 1: the whole site.  SPL = 2: lane bit 0
// the real (0) or the imaginary (1) part.  SPL = 4: also lane bit 1 the forward (0)
// or backward (1) bonds.  A part is the sum over the bonds of X re + Y im with
// re: (X, Y) = (Re h, -Im h), im: (Im h, Re h), h conjugated for a backward bond;
// a whole site holds (Re h, Im h).
__device__ __forceinline__ unsigned pk64_nbr(const PkTile& t, const PkRec& r, int d)
{
    const unsigned a = 16u * r.at;
    switch (d) {
        case 0: return a + 16u * r.xp - 16u * r.col;
        case 1: return a + 16u * r.xm - 16u * r.col;
        case 2: return a + t.rowB;
        case 3: return a - t.rowB;
        case 4: return a + t.rowB * (unsigned)t.zstr;
        default: return a - t.rowB * (unsigned)t.zstr;
    }
}
__device__ __forceinline__ unsigned pk64_bond_at(const PkTile& t, const PkRec& r, int d)
{
    switch (d) {
        case 0: return (unsigned)t.bx_row(r.y, r.z) * t.rowB + 16u * r.col;
        case 1: return (unsigned)t.bx_row(r.y, r.z) * t.rowB + 16u * r.xm;
        case 2: return (unsigned)t.by_row(r.y, r.z) * t.rowB + 16u * r.col;
        case 3: return (unsigned)(t.by_row(r.y, r.z) - 1) * t.rowB + 16u * r.col;
        case 4: return (unsigned)t.bz_row(r.y, r.z) * t.rowB + 16u * r.col;
        default: return (unsigned)(t.bz_row(r.y, r.z) - t.PY) * t.rowB + 16u * r.col;
    }
}
template <int SPL>
__device__ __forceinline__ void pk64_xy(unsigned bonds, const PkTile& t, const PkRec& r, int d, int c, int (&X)[2], int (&Y)[2])
{
    const int4 h = lds4(bonds + pk64_bond_at(t, r, d));
    const bool back = d & 1;
    const int2 re = make_int2(h.x, h.y), im = back ? make_int2(-h.z, -h.w) : make_int2(h.z, h.w);
    const bool part_im = SPL > 1 && c == 1, part_re = SPL > 1 && c == 0;
    X[0] = part_im ? im.x : re.x;
    X[1] = part_im ? im.y : re.y;
    Y[0] = part_im ? re.x : part_re ? -im.x : im.x;
    Y[1] = part_im ? re.y : part_re ? -im.y : im.y;
}

// The steps of one update.  KI > 0: up to KI parts of sites per thread (KI = 1 but
// for whole sites), their bonds and S_m, S_{m-1} in registers (SPL T <= 256 KI);
// KI = 0: whole sites s, s + 256, ... with bonds and S_{m-1} from shared memory.
// Not inlined: with the tail in one function the registers that live across it
// went to local memory inside the step loop.
// s_fail: the first step whose wait ran out (before it, kNoFail).  False (in every
// thread): a wait of the CTA ran out.
// MOM: no sums; instead the values at the local sites of a moments call, limbs as they
// are, go to head.mom (pk64_moments), S_m to place m of the sites' rows.
template <class Ex, int SPL, int KI, bool MOM = false>
__device__ __noinline__ bool pk64_advance(const Params& p, const PkTile& tile, const PkRec* tab, const PkHead& head,
                                          PkSums<double, kPk64Threads / 32>& sums, unsigned mb, unsigned ph,
                                          int* s_fail)
{
    static_assert(!MOM || KI == 1, "one site per thread");
    static_assert(KI == 1 || SPL == 1, "one part of a site per thread");
    constexpr int NT = kPk64Threads, NW = NT / 32, ND = SPL == 4 ? 3 : 6, KR = KI > 0 ? KI : 1;
    const PkTile t = tile;
    Ex ex(t, p, mb, ph);
    const unsigned bonds = smem_u32(t.bonds);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int T = t.L * t.PY * t.PZ, items = SPL * T;
    const int c = SPL > 1 ? tid & 1 : 0, hf = SPL == 4 ? (tid >> 1) & 1 : 0;
    unsigned own[KR];                       // shared address of the site (its part) in buffer 0
    typename Ex::Target tgt[KR];
    unsigned off[KR][ND];                   // shared addresses of the neighbours in buffer 0
    int X[KR][ND][2], Y[KR][ND][2];         // the bonds
    int4 cur[KR], prv[KR];                  // S_m and S_{m-1}: limbs (a part: x, y)
    bool odd[KR];
    // values into the ring slot and on to the neighbours; returns the limbs
    auto store = [&](unsigned at, unsigned buf, int m, const typename Ex::Target& g, long long re, long long im) {
        if constexpr (SPL == 1) {
            const int4 w = pk_limbs(re, im);
            sts4(at + buf, w);
            ex.push(m, buf, g, re, im, w);
            return w;
        } else {
            const int2 w = make_int2((int)((re + (1ll << 29)) >> 30), (int)((unsigned)re << 2) >> 2);
            if (hf == 0) {
                sts2(at + buf, w);
                ex.push(m, buf, g, re, w);
            }
            return make_int4(w.x, w.y, 0, 0);
        }
    };
    auto start = [&](const PkRec& r) {
        const int col = r.col, od = col >= t.half ? 1 : 0, x = 2 * (col - od * t.half) + od;
        const double2 v = pk_s0(x + t.L * (t.y0 + r.y + t.L * (t.z0 + r.z)), head.loc, head.c);
        return store(t.ring + 16u * r.at + 8u * c, 0, 0, ex.target(r, c), __double2ll_rn((c ? v.y : v.x) * 0x1p60),
                     __double2ll_rn(v.y * 0x1p60));
    };
    // MOM: byte offsets of place 0 of the rows that take this site's S_m, m even and odd; ~0u: none
    [[maybe_unused]] unsigned row[2] = {~0u, ~0u};
    [[maybe_unused]] auto sample = [&](int m, int4 v) {
        const unsigned r = row[m & 1];
        char* a = (char*)p.mom_out + r + 16u * (unsigned)m;
        if constexpr (SPL == 1)
            asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0xffffffff;\n @p st.global.v4.s32 [%0], {%1, %2, %3, %4};\n}" ::"l"(a),
                         "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(r)
                         : "memory");
        else
            asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0xffffffff;\n @p st.global.v2.s32 [%0], {%1, %2};\n}" ::"l"(a), "r"(v.x),
                         "r"(v.y), "r"(r)
                         : "memory");
    };
    if constexpr (KI > 0) {
#pragma unroll
        for (int k = 0; k < KI; ++k) {
            own[k] = 0;
            cur[k] = prv[k] = make_int4(0, 0, 0, 0);
            if (tid + k * NT < items) {
                const PkRec r = tab[(tid + k * NT) / SPL];
                cur[k] = start(r);
                own[k] = t.ring + 16u * r.at + 8u * c;
                tgt[k] = ex.target(r, c);
                odd[k] = (r.fl >> 4) != 0;
                if constexpr (MOM) {
                    const int od = r.col >= t.half ? 1 : 0, x = 2 * (r.col - od * t.half) + od;
                    const int i = x + t.L * (t.y0 + r.y + t.L * (t.z0 + r.z));
                    for (int j = 0; j < kVec; ++j)
                        if (i == head.mom[j] && hf == 0)
                            for (int b = 0; b < 2; ++b)
                                if (head.row[b][j] != ~0u) row[b] = head.row[b][j] + 8u * (unsigned)c;
                    sample(0, cur[k]);
                }
#pragma unroll
                for (int d = 0; d < ND; ++d) {
                    const int e = SPL == 4 ? 2 * d + hf : d;
                    off[k][d] = t.ring + pk64_nbr(t, r, e);
                    pk64_xy<SPL>(bonds, t, r, e, c, X[k][d], Y[k][d]);
                }
            }
        }
    } else {
        for (int s = tid; s < T; s += NT) start(tab[s]);
    }
    const int nsteps = p.nsteps, lo = head.loc[0];
    const bool odd_o = (lo % t.L + (lo / t.L) % t.L + lo / (t.L * t.L)) & 1;
    for (int m = 0; m <= nsteps; ++m) {
        const unsigned b0 = (m & 1) ? t.bufB : 0u, b1 = (m & 1) ? 0u : t.bufB;
        const bool ok = ex.receive(m, b0);
        if (!ok) atomicMin(s_fail, m);
        __syncthreads();
        ex.received(m, ok);
        // a wait that ran out by step m: the same answer in every thread, as one that runs out
        // in a later step (of a thread ahead of this one) records that step
        if ((m & 7) == 7 && *(volatile int*)s_fail <= m) {
            if constexpr (Ex::kAbort) return false;
            else ex.dead = true;
        }
        const bool oddA = odd_o ^ ((m & 1) != 0);  // the parity that holds r_m^o
        Pk64Sums acc;
        // a whole site: S_{m+1} from the neighbours v, the bonds and S_{m-1}
        auto site = [&](const int4 (&v)[6], const int (&hr)[6][2], const int (&hi)[6][2], int4 q, long long& re,
                        long long& im) {
            long long PA = -(long long)q.y, PB = 0, NA = 0, NB = 0, QA = -(long long)q.w, QB = 0;
            pk_wide(PA, q.x, -(1 << 30));
            pk_wide(QA, q.z, -(1 << 30));
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                pk_mac(PA, PB, hr[d][0], hr[d][1], v[d].x, v[d].y);
                pk_mac(NA, NB, hi[d][0], hi[d][1], v[d].z, v[d].w);
                pk_mac(QA, QB, hr[d][0], hr[d][1], v[d].z, v[d].w);
                pk_mac(QA, QB, hi[d][0], hi[d][1], v[d].x, v[d].y);
            }
            re = pk_value(PA - NA, PB - NB);
            im = pk_value(QA, QB);
            if (m == 0) {  // S_1 = Htilde S_0
                re = (re + 1) >> 1;
                im = (im + 1) >> 1;
            }
        };
        if constexpr (KI == 0) {
            for (int s = tid, n = 1; s < T; s += NT, ++n) {
                const PkRec r = tab[s];
                const unsigned at = t.ring + 16u * r.at;
                int4 v[6];
                int hr[6][2], hi[6][2];
                long long re, im;
#pragma unroll
                for (int d = 0; d < 6; ++d) {
                    v[d] = lds4(t.ring + b0 + pk64_nbr(t, r, d));
                    pk64_xy<1>(bonds, t, r, d, 0, hr[d], hi[d]);
                }
                const int4 pv = m > 0 ? lds4(at + b1) : make_int4(0, 0, 0, 0), cv = lds4(at + b0);
                site(v, hr, hi, pv, re, im);
                const int4 w = store(at, b1, m + 1, ex.target(r, 0), re, im);
                acc.add(cv, w, ((r.fl >> 4) != 0) == oddA);
                if (n % kPkPut == 0) acc.put();
            }
        } else if constexpr (SPL == 1) {
            int4 nx[KI];
#pragma unroll
            for (int k = 0; k < KI; ++k) {
                if (tid + k * NT < T) {
                    int4 v[6];
                    long long re, im;
#pragma unroll
                    for (int d = 0; d < 6; ++d) v[d] = lds4(off[k][d] + b0);
                    site(v, X[k], Y[k], prv[k], re, im);
                    nx[k] = store(own[k], b1, m + 1, tgt[k], re, im);
                }
            }
#pragma unroll
            for (int k = 0; k < KI; ++k) {
                if (tid + k * NT < T) {
                    if constexpr (MOM) sample(m + 1, nx[k]);
                    else acc.add(cur[k], nx[k], odd[k] == oddA);
                    prv[k] = cur[k];
                    cur[k] = nx[k];
                }
            }
        } else if ((tid & ~31) < items) {
            // a part of a site (whole warps but for the last: the shuffles run in all lanes)
            const bool on = tid < items;
            long long A = 0, B = 0;
            int2 w = make_int2(0, 0);
            if (on) {
                int4 v[ND];
#pragma unroll
                for (int d = 0; d < ND; ++d) v[d] = lds4(off[0][d] + b0);
                if (hf == 0) {
                    w = lds2(own[0] + b0 + 8u - 16u * c);  // the other part of S_m
                    A = -(long long)prv[0].y;
                    pk_wide(A, prv[0].x, -(1 << 30));
                }
#pragma unroll
                for (int d = 0; d < ND; ++d) {
                    pk_mac(A, B, X[0][d][0], X[0][d][1], v[d].x, v[d].y);
                    pk_mac(A, B, Y[0][d][0], Y[0][d][1], v[d].z, v[d].w);
                }
            }
            if constexpr (SPL == 4) {
                A += __shfl_xor_sync(0xffffffffu, A, 2);
                B += __shfl_xor_sync(0xffffffffu, B, 2);
            }
            long long s = pk_value(A, B);
            if (m == 0) s = (s + 1) >> 1;
            if (on) {
                const int4 nx = store(own[0], b1, m + 1, tgt[0], s, 0);
                if constexpr (MOM) {
                    sample(m + 1, nx);
                } else if (hf == 0) {
                    if (odd[0] == oddA) {
                        acc.square<0>(cur[0].x, cur[0].y);
                        pk_mac(acc.RA, acc.RB, cur[0].x, cur[0].y, nx.x, nx.y);
                        if (c == 0) {
                            w.x = -w.x;
                            w.y = -w.y;
                        }
                        pk_mac(acc.IA, acc.IB, w.x, w.y, nx.x, nx.y);
                    } else {
                        acc.square<1>(cur[0].x, cur[0].y);
                    }
                }
                prv[0] = cur[0];
                cur[0] = nx;
            }
        }
        if (!MOM && m > 0) {
            acc.put();
            const long long w = warp_reduce_scatter4(acc.v, lane);
            if ((lane & 7) == 0) sums.w[m & (kPkRing - 1)][warp][lane >> 3] = w;
        }
        // warps take turns (a barrier lies between the sums of the flushed steps and this)
        if (!MOM && (m & (kPkGroup - 1)) == 1) pk_flush_due<double, NW>(p, sums, m, warp ^ ((m >> 3) & (NW - 1)), lane);
    }
    __syncthreads();
    if (!MOM) pk_flush_rest<double, NW>(p, sums, nsteps, warp, lane);
    return *(volatile int*)s_fail > nsteps;
}

// ---------------------------------------------------------------------------
// one chain
// ---------------------------------------------------------------------------
// GRID: on the p.ncta CTAs of a cooperative grid, pencils of nearly equal size;
// otherwise on one cluster of p.ncta CTAs, pencils of equal size.
template <bool GRID> __device__ __forceinline__ void pk64_run_chain(const Params& p, const int rank, char* smem)
{
    using Ex = std::conditional_t<GRID, PkGridEx<2, 4>, PkAsyncEx>;
    // larger tiles: more face values per thread, each site on at most one face in y and one in z
    using Ex2 = std::conditional_t<GRID, PkGridEx<2, 2>, PkAsyncEx>;
    using Ex3 = std::conditional_t<GRID, PkGridEx<3, 2>, PkAsyncEx>;
    using ExN = std::conditional_t<GRID, PkGridEx<kPkMaxFaces / kPk64Threads, 4>, PkAsyncEx>;
    __shared__ PkSums<double, kPk64Threads / 32> sums;
    __shared__ PkHead head;
    __shared__ int s_fail;
    __shared__ __align__(8) unsigned long long s_mb[2];
    const int tid = threadIdx.x, C = p.ncta, N = p.N;
    __shared__ PkTile t;
    if (tid == 0) t = pk_tile<double>(p, rank, smem);
    __syncthreads();
    PkRec* tab = (PkRec*)(t.bonds + (size_t)t.bond_rows() * t.rowB);
    double2* work = (double2*)smem;
    const int work_n = (int)((t.bonds - smem) / (int)sizeof(double2));
    const int T = t.L * t.PY * t.PZ;
    pk64_records(t, tab);
    if constexpr (!GRID) {
        if (tid == 0) PkAsyncEx(t, p, smem_u32(s_mb), 0).init();
    }
    if (tid == 0) s_fail = kNoFail;
    bool ok = true;  // no wait of the CTA has run out
    auto sync = [&](int where) -> bool {
        if constexpr (GRID) {
            return grid_barrier(p, where);
        } else {
            if (C > 1) cooperative_groups::this_cluster().sync();
            else __syncthreads();
            return true;
        }
    };
    // cluster: every CTA has started and initialised its barriers before any remote store
    if constexpr (GRID) __syncthreads();
    else sync(0);

    const long long nupd = (p.mode == MODE_SWEEP) ? p.n_updates : 1;
    long long nmag = 0;
    unsigned long long nacc = 0;
    bool reload = true;
    for (long long q = 0; q < nupd; ++q) {
        const unsigned long long upd = p.upd0 + (unsigned long long)q;
        const int o = (p.mode == MODE_SWEEP) ? (int)(upd % (unsigned long long)N) : (int)p.site;
        pk_setup(p, head, o, upd);
        if (reload) pk_load_bonds<double, kPk64Threads>(p, t);
        reload = false;
        __syncthreads();
        const unsigned mb = smem_u32(s_mb), ph = (unsigned)(q * (long long)(p.nsteps + 1));
        constexpr int NT = kPk64Threads;
        const int faces = GRID ? 2 * (t.PY + t.PZ) * t.L : 0;
        const bool wide = !GRID || (t.PY >= 2 && t.PZ >= 2);
        if (4 * T <= NT && faces <= 2 * NT) ok = pk64_advance<Ex, 4, 1>(p, t, tab, head, sums, mb, ph, &s_fail);
        else if (2 * T <= NT && faces <= 2 * NT) ok = pk64_advance<Ex, 2, 1>(p, t, tab, head, sums, mb, ph, &s_fail);
        else if (T <= NT && faces <= 2 * NT && wide) ok = pk64_advance<Ex2, 1, 1>(p, t, tab, head, sums, mb, ph, &s_fail);
        else if (T <= 2 * NT && faces <= 3 * NT && wide) ok = pk64_advance<Ex3, 1, 2>(p, t, tab, head, sums, mb, ph, &s_fail);
        else if (T <= 3 * NT && faces <= 3 * NT && wide) ok = pk64_advance<Ex3, 1, 3>(p, t, tab, head, sums, mb, ph, &s_fail);
        else ok = pk64_advance<ExN, 1, 0>(p, t, tab, head, sums, mb, ph, &s_fail);
        if (GRID && !ok) return;
        if (!sync(1)) return;
        pk_tail_fft<kPk64Threads>(p, rank, C, work, work_n, head);
        if (!sync(2)) return;
        pk_tail_clear<kPk64Threads>(p, rank, C);
        pk_tail_phase<kPk64Threads>(p, rank, C, (double*)work);
        // after a wait that ran out on a cluster no CTA accepts the move, and all leave
        if (!GRID && !ok && tid == 0) {
            p.qpart[2 * rank] = CUDART_NAN;
            p.qpart[2 * rank + 1] = CUDART_INF;
        }
        if (!sync(3)) return;
        pk_decide(p, head, rank, q);
        __syncthreads();
        if (p.mode == MODE_DELTA || (!GRID && head.stop)) break;
        if (head.acc) {
            ++nacc;
            // only the bonds of o change: pencils that do not hold or border its row keep theirs
            const int oy = (o / t.L) % t.L, oz = o / (t.L * t.L);
            const int dy = (oy - t.y0 + 1 + t.L) % t.L, dz = (oz - t.z0 + 1 + t.L) % t.L;
            reload = dy <= t.PY + 1 && dz <= t.PZ + 1;
            if (rank == 0 && tid < 7) patch_site(p, o, head.loc, head.draw[0], head.draw[1], tid);
            if (!sync(5)) return;
        }
        if ((upd + 1ull) % (unsigned long long)N == 0ull) {
            if (!pk_magnetisation<kPk64Threads>(p, rank, nmag, sync)) return;
            ++nmag;
        }
    }
    if (rank == 0 && tid == 0 && p.mode == MODE_SWEEP) {
        *p.n_acc = nacc;
        *p.n_mag = nmag;
    }
    if constexpr (!GRID) {
        if (!ok) {  // values still in flight land before any CTA leaves
            const long long t0 = clock64();
            while (clock64() - t0 < (1ll << 21)) __nanosleep(256);
        }
        sync(0);  // no CTA leaves while another may still write into its shared memory
    }
}

// All moments <l_j|T_n(Htilde)|l_k>, n < M, of the seven local sites of p.site, by six
// clusters, each on its own vector through M - 1 steps: cluster v > 0 on l_{v+1}, cluster 0 on
// o + l_1 (opposite parities).  The values at the local sites are the moments, so a step
// has no sums and the clusters do not meet; against the recursion on seven vectors to
// M/2 with the sums of 28 pairs of products (a grid of flags), L = 12, M = 512:
// 1346 -> 362 us per call, bound by the latency of a step (0.57 us).  Up to L = 16, a site
// per thread; FP32-mixed chains take it as well, with the FP64 bonds.
__global__ void __launch_bounds__(kPk64Threads, 1) gfmc_packed64_moments(const Params q)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params p;
    __shared__ PkSums<double, kPk64Threads / 32> sums;
    __shared__ PkHead head;
    __shared__ PkTile t;
    __shared__ int s_fail;
    __shared__ __align__(8) unsigned long long s_mb[2];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int tid = threadIdx.x, rank = (int)cl.block_rank(), C = (int)cl.dim_blocks().x, v = (int)blockIdx.x / C;
    const int kcol = v + 1, M = q.M;  // the column of the cluster's l
    if (tid == 0) {
        p = q;
        p.nsteps = M - 2;  // S_{M-1} is the last vector
        t = pk_tile<double>(p, rank, (char*)dyn_all);
        s_fail = kNoFail;
        const int o = (int)p.site;
        for (int j = 0; j < kVec; ++j) {
            head.mom[j] = j == 0 ? o : nbr_site(o, j - 1, p.L);
            // row (j, k) of the moment matrix, j <= k
            const unsigned rj = 16u * (unsigned)(M * (kVec * j + kcol));
            for (int b = 0; b < 2; ++b) head.row[b][j] = v > 0 && j <= kcol ? rj : ~0u;
            head.loc[j] = -1;
            head.c[j] = make_double2(1.0, 0.0);
        }
        if (v == 0) {
            // at o: T_m|o> for even m, T_m|l_1> for odd m; at l_1: T_m|l_1> for even m
            head.row[0][0] = 0u;
            head.row[1][0] = 16u * (unsigned)M;
            head.row[0][1] = 16u * (unsigned)(M * (kVec + 1));
            head.row[1][1] = ~0u;
            head.loc[0] = o;
            head.loc[1] = head.mom[1];
        } else {
            head.loc[0] = head.mom[kcol];
        }
    }
    __syncthreads();
    PkRec* tab = (PkRec*)(t.bonds + (size_t)t.bond_rows() * t.rowB);
    pk64_records(t, tab);
    if (tid == 0) PkAsyncEx(t, p, smem_u32(s_mb), 0).init();
    pk_load_bonds<double, kPk64Threads>(p, t);
    cl.sync();  // every CTA has initialised its barriers before any remote store
    const int T = t.L * t.PY * t.PZ;
    const unsigned mb = smem_u32(s_mb);
    constexpr int NT = kPk64Threads;
    bool ok;
    if (4 * T <= NT) ok = pk64_advance<PkAsyncEx, 4, 1, true>(p, t, tab, head, sums, mb, 0, &s_fail);
    else if (2 * T <= NT) ok = pk64_advance<PkAsyncEx, 2, 1, true>(p, t, tab, head, sums, mb, 0, &s_fail);
    else ok = pk64_advance<PkAsyncEx, 1, 1, true>(p, t, tab, head, sums, mb, 0, &s_fail);
    if (!ok) {  // values still in flight land before any CTA leaves
        const long long t0 = clock64();
        while (clock64() - t0 < (1ll << 21)) __nanosleep(256);
    }
    __threadfence();
    cl.sync();
    // limbs to values, and the conjugates below the diagonal
    for (int k = v == 0 ? 0 : kcol; k <= kcol; ++k)
        for (int e = rank * NT + tid; e < (k + 1) * M; e += C * NT) {
            const int j = e / M, n = e - j * M;
            double2* a = p.mom_out + (size_t)(kVec * j + k) * M + n;
            const bool live = ((n + (j > 0 ? 1 : 0) + (k > 0 ? 1 : 0)) & 1) == 0;
            double2 m = make_double2(0.0, 0.0);
            if (live) {
                const int4 w = __ldcg((const int4*)a);
                m = make_double2((double)pk_join(w.x, w.y) * 0x1p-60, (double)pk_join(w.z, w.w) * 0x1p-60);
            }
            if (j == k) m.y = 0.0;
            __stcg(a, m);
            if (j < k) __stcg(p.mom_out + (size_t)(kVec * k + j) * M + n, make_double2(m.x, -m.y));
        }
}

__global__ void __launch_bounds__(kPk64Threads, 1) gfmc_packed64_cluster(const TeamJob* __restrict__ jobs)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params sp;
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    if (threadIdx.x == 0) sp = jobs[blockIdx.x / cl.dim_blocks().x].p;
    __syncthreads();
    pk64_run_chain<false>(sp, (int)cl.block_rank(), (char*)dyn_all);
}

// A single chain on one cluster: FP32-mixed, or FP64 with small tiles.
template <class R>
__global__ void __launch_bounds__(sizeof(R) == 4 ? kPkThreads32 : kPk64Threads, 1) gfmc_packed_single(const Params p)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params sp;
    if (threadIdx.x == 0) sp = p;
    __syncthreads();
    const int rank = (int)cooperative_groups::this_cluster().block_rank();
    if constexpr (sizeof(R) == 4) pk_run_chain<float>(sp, rank, (char*)dyn_all);
    else pk64_run_chain<false>(sp, rank, (char*)dyn_all);
}

__global__ void __launch_bounds__(kPk64Threads, 1) gfmc_packed64_grid(const Params p)
{
    extern __shared__ double2 dyn_all[];
    __shared__ Params sp;
    if (threadIdx.x == 0) sp = p;
    __syncthreads();
    pk64_run_chain<true>(sp, (int)blockIdx.x, (char*)dyn_all);
}

}  // namespace gfmc
