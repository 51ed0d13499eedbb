// gfmc_internal.h -- structures shared by the host API and the CUDA kernels.
//
// One chain = one Params block.  All arrays are device memory owned by the
// handle (gfmc_api.cu); the kernels only read these pointers.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace gfmc {

// Let kernel fn take any dynamic shared memory the current device allows (its
// opt-in maximum less fn's static shared memory).  The attribute is raised to
// that bound and never set to a launch's own size, so its value does not
// depend on the order of calls: a kernel node of a captured graph that is
// launched again on its own (as a profiler replays graph nodes one by one) is
// checked against the attribute as it stands then, and a per-launch setting
// would have let a later, smaller launch or occupancy query lower it below
// the node's size.
inline cudaError_t allow_dynamic_smem(const void* fn)
{
    int dev = 0, optin = 0;
    cudaFuncAttributes a;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
        (e = cudaFuncGetAttributes(&a, fn)) != cudaSuccess)
        return e;
    const int room = optin - (int)a.sharedSizeBytes;
    if (a.maxDynamicSharedSizeBytes >= room) return cudaSuccess;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
}

constexpr int kThreads = 256;            // threads per CTA of the persistent engine
constexpr int kWarps = kThreads / 32;
constexpr int kVec = 7;                  // local vectors: o and its 6 neighbours
constexpr int kPairs = 28;               // upper-triangle pairs (j <= k) of the 7x7 block
constexpr int kEntries = 112;            // 2 Gram blocks x 28 pairs x (re, im)
constexpr int kMaxNbrCta = 64;           // neighbour CTAs a tile may depend on
constexpr int kMaxL = 64;                // larger than kThreads x CTAs sites: team variant
constexpr int kStage = kThreads + 1;     // row stride of the staged vectors (bank spread)

enum Mode : int { MODE_MOMENTS = 0, MODE_DELTA = 1, MODE_SWEEP = 2 };

enum ErrCode : int { ERR_NONE = 0, ERR_TIMEOUT = 4, ERR_NUMERIC = 5 };

struct Params {
    // lattice and model
    int L, N, M, nsteps, ncta;
    int K;                 // Chebyshev nodes of G and of the quadrature (M or 2M)
    unsigned divL, divLL;  // ceil(2^32 / L), ceil(2^32 / L^2): exact i / L, i / L^2 for i < N
    unsigned divT;         // cluster variant: ceil(2^32 / (N / ncta)), the owner of a site
    double t, chem, beta, a;

    // chain state
    double* spins;    // [N][2] (theta, phi)
    double2* hop64;   // [3][N]   Htilde_{i, i+e_alpha}, alpha = x, y, z
    float2* hop32;    // [3][N]   the same rounded to FP32 (mixed path)
    void* rbuf;       // [2][7][N] recursion vectors (double2 or float2)

    // constant tables, filled by the set-up kernel
    double* gker;     // [M]     kernel g_n
    double2* twc;     // [M]     e^{-i n pi / (2K)}
    double2* fftw;    // [K/2]   e^{-2 pi i j / K}
    double* sinth;    // [K]     sin theta_k, theta_k = pi (k + 1/2) / K
    double* cumw;     // [K]     C_k = sum_{j<=k} sin theta_j f(a cos theta_j)

    // per-update scratch
    unsigned long long* gram;  // [nsteps][kEntries]  Gram sums over the CTAs, 64-bit fixed point
    double2* fftin;   // [4][M]  damped, twisted combined moments (zero beyond M)
    double2* gnode;   // [4][K]  G_V(w_k) for V = o, v, o+v, o+iv
    double* qpart;    // [ncta][2]  (phase-sum partial, max |increment|)
    double* magpart;  // [ncta][3]
    double2* mom_out; // [7][7][M] full moment matrix (moments mode)
    // vector-cluster engine: the direct moment entries r_n^k[l_j] at [k][j][n]
    float2* mom32;    // [7][7][M]

    // tile partition of the sites over CTAs and the CTAs each tile reads from
    const int* tile_start;  // [ncta + 1]
    const int* nbr_ptr;     // [ncta + 1]
    const int* nbr_idx;     // [nbr_ptr[ncta]]
    // FP64 single-chain engine: the sites a CTA's stencil reads (its tile and
    // the tile's neighbours) as runs of consecutive sites, win[win_ptr[c] ..
    // win_ptr[c+1]) = (first site, length); win_max = the largest total.  With
    // prefetch set, the helper warp copies these runs of r_m into shared
    // memory while the compute warps form the Gram sums of the step before.
    const int* win_ptr;     // [ncta + 1]
    const int2* win;        // [win_ptr[ncta]]
    int win_max;
    int prefetch;
    // FP64 single-chain engine, L even (the periodic cubic lattice is then
    // bipartite): each step advances only the vectors that are nonzero at a
    // site (vector o on one parity, its 6 neighbours' on the other), dealt to
    // the compute threads as (vector, site) items, and forms only the Gram sums
    // that are not zero by parity; 2: tiles of at least 128 sites, the split
    // instantiation (halo-only prefetch, group sums beside the units)
    int bip;
    // FP32-mixed: the Gram dot products of the doubling (Eq. mu2) with
    // compensated FP32 products and warp sums (Dot2) before FP64
    int comp;
    // single-chain engines on 256 threads (FP32 unit vectors, proposal vectors):
    // every tile fits 7 warps, so warp 7 publishes and polls the flags while
    // the other warps form the Gram sums
    int helper7;

    // synchronisation
    unsigned* flags;  // [ncta]  completed stencil phases of each CTA
    unsigned* bar;    // [2]     grid barrier: arrival count, generation
    int* err;         // [4]     code, where, cta, aux
    long long budget; // clock64 cycles a single wait may spin before giving up
    int stall;        // test hook: CTA 0 withholds its completion flags
    int nv;           // recursion vectors of team launches: 7 (unit vectors) or 2 (o and v)
    int pk_cy;        // packed engines: CTAs along y (0: another engine)
    int pk_cz;        // and along z
    int pk_rows;      // packed grid engine: rows per face of an inbox
    unsigned long long* pk_inbox;  // [ncta][2][4][pk_rows][L][2] face values in flight

    // work description
    int mode;
    long long site;            // moments / delta modes
    double theta_new, phi_new; // delta mode
    unsigned long long upd0;   // sweep mode: first update number
    long long n_updates;       // sweep mode
    unsigned long long seed;
    unsigned chain_id;

    // outputs
    unsigned char* dec_out;    // [n_updates]
    double* domega_out;        // [n_updates] (sweep) or [1] (delta)
    double* maxinc_out;        // [n_updates] or [1]
    double* mag_out;           // [n_updates / N + 1]
    unsigned long long* n_acc; // [1]
    long long* n_mag;          // [1]
};

// Shared memory of a CTA of the packed cluster engine (gfmc_packed.cuh) for a
// pencil of PY x PZ rows of L sites: the two ring buffers, which are the tail's
// work area (16 K bytes at least) between recursions; then the forward bonds.
__host__ __device__ inline int pk_work_bytes(int L, int PY, int PZ, int K, bool fp32)
{
    const int ring = 2 * (PY + 2) * (PZ + 2) * L * (fp32 ? 8 : 16), fft = 16 * K;
    return ((ring > fft ? ring : fft) + 127) & ~127;
}
__host__ __device__ inline int pk_smem_bytes(int L, int PY, int PZ, int K, bool fp32)
{
    const int rows = 3 * PY * PZ + PZ + PY;
    return pk_work_bytes(L, PY, PZ, K, fp32) + rows * L * (fp32 ? 8 : 16);
}
// the same for the FP64 engines of gfmc_packed64.cuh: a record per site too
__host__ __device__ inline int pk64_smem_bytes(int L, int PY, int PZ, int K)
{
    return pk_smem_bytes(L, PY, PZ, K, false) + 8 * L * PY * PZ;
}
constexpr int kPkThreads32 = 512, kPkThreads64 = 256;
// The split of an L^3 chain over a cluster of C CTAs into pencils of L / cy x
// L / (C / cy) rows with the smallest ring (the values exchanged per step);
// false when the packed cluster engine does not take the chain (odd L, or more
// pairs per thread than its FP32 kernel holds).
inline bool pk_split(int L, int C, int K, bool fp32, int* cy, int* bytes)
{
    if (L % 2 != 0 || C < 1 || C > 16) return false;
    long long best = -1;
    for (int a = 1; a <= C; ++a) {
        if (C % a != 0 || L % a != 0 || L % (C / a) != 0) continue;
        const int PY = L / a, PZ = L / (C / a);
        if (fp32) {
            const int ncol = (L / 2) * PY;
            if (ncol > kPkThreads32) continue;
            const int nseg = kPkThreads32 / ncol < PZ ? kPkThreads32 / ncol : PZ;
            if ((PZ + nseg - 1) / nseg > 4) continue;
        }
        const long long ring = (a > 1 ? PZ : 0) + (C / a > 1 ? PY : 0);
        if (best >= 0 && ring >= best) continue;
        best = ring;
        *cy = a;
        *bytes = pk_smem_bytes(L, PY, PZ, K, fp32);
    }
    return best >= 0;
}

// The split of an even lattice over at most max_ctas CTAs of the grid into
// pencils of whole x-rows: the fewest rows in the largest pencil, then the
// fewest face values; false when none fits (smem: the room per CTA).
constexpr int kPkMaxFaces = 6 * 256;  // face values a CTA receives per step at most
inline bool pk_grid_split(int L, int K, int max_ctas, int smem, int* cy, int* cz, int* bytes)
{
    if (L % 2 != 0) return false;
    long long best = -1;
    for (int a = 2; a <= L; ++a)
        for (int b = 2; b <= L && a * b <= max_ctas; ++b) {
            const int PY = (L + a - 1) / a, PZ = (L + b - 1) / b;
            const int faces = L * (2 * PZ + 2 * PY);
            const int need = pk64_smem_bytes(L, PY, PZ, K);
            if (faces > kPkMaxFaces || need > smem || (PY + 2) * (PZ + 2) * L > 65535) continue;
            const long long cost = (long long)PY * PZ * 1000000 + faces * 100 + a + b;
            if (best >= 0 && cost >= best) continue;
            best = cost;
            *cy = a;
            *cz = b;
            *bytes = need;
        }
    return best >= 0;
}

// One-CTA chains of a few sites per thread (gfmc_team.cuh): the most sites a CTA of nt
// threads takes (FP32: 4 per thread, FP64 in fixed point: 2), the ring items per
// step, and the shared memory of vectors and ring.
template <class R> __host__ __device__ constexpr int one_cta_sites(int nt) { return sizeof(R) == 4 ? 4 * nt : 2 * nt; }
__host__ __device__ inline int one_cta_items(int N, int nt) { return N < nt ? (N + 31) / 32 * 32 : nt; }
template <class R> __host__ __device__ inline int one_cta_bytes(int N, int nt)
{
    return 4 * (int)sizeof(R) * N + 16 * one_cta_items(N, nt) * (sizeof(R) == 4 ? 16 : 8);
}
// An FP64 chain alone on a CTA: threads per site.  Two (the real and the imaginary part)
// while that is one warp per sub-partition: L = 4 0.30 us per step, with one thread 0.40;
// L = 6 0.69 with two, 0.61 with one.
__host__ __device__ inline int one_cta_parts(int N) { return 2 * N <= 128 ? 2 : 1; }

// One chain of a batch launch: its parameters (ncta = its team size, tile plan
// for that team) and its CTAs [cta0, cta0 + p.ncta) of the grid.
struct TeamJob {
    Params p;
    int cta0;
    int vec_smem;  // bytes of the chain's recursion vectors in the CTA's shared memory, 0: in global memory
    int pad[2];
};

// Shared memory of a launch of teams.  Every CTA runs one chain at a time, which has
// all of it: its vectors first, if they stand there, and the tail's work area behind
// them -- on the packed recursion in their place.  So the launch takes the largest
// need of any chain, and whether a chain's vectors stand there follows from its own
// sizes and the room (the device's limit less the kernel's static part) alone.
struct TeamChainSmem {
    size_t vec;   // bytes of the vectors; SIZE_MAX: they stay in global memory
    size_t work;  // bytes of the work area
    size_t want;  // packed: bytes that more of the chain's data could use
    bool packed;
    int at;       // out: vec_smem of the chain's job
};
inline int team_smem_bytes(TeamChainSmem* c, int n, size_t room)
{
    size_t total = 0, want = 0;
    for (int k = 0; k < n; ++k) {
        const size_t vec = c[k].vec == SIZE_MAX ? 0 : (c[k].vec + 15) & ~(size_t)15;
        const size_t need = c[k].packed ? (vec > c[k].work ? vec : c[k].work) : vec + c[k].work;
        const bool resident = vec > 0 && need <= room;
        c[k].at = resident ? (int)vec : 0;
        const size_t use = resident ? need : c[k].work;
        total = total > use ? total : use;
        if (resident && c[k].packed && c[k].want > want) want = c[k].want;
    }
    want = (want < room ? want : room) & ~(size_t)15;
    return (int)(total > want ? total : want);
}

// Mailbox of one slot of the serving loop (device memory).  The host writes
// [prec, cta0, job] and then seq; the slot's CTA 0 relays seq through cmd.
struct SlotCtl {
    unsigned seq;  // sequence number of the last posted job (host)
    unsigned cmd;  // slot CTA 0 -> the slot's other CTAs: job to run, or exit
    int prec;      // 0 FP64, 1 FP32-mixed
    int cta0;      // first CTA of the slot in the grid
    Params job;
};

struct ServerArgs {
    SlotCtl* slots;
    unsigned* done;           // host-mapped: last completed sequence number per slot
    const unsigned* shutdown; // nonzero: every slot exits when idle
    unsigned* quiesce;        // [0] slots idle for idle_budget, [1] nonzero: the launch ends (host-cleared)
    int nslots;
    long long idle_budget;    // cycles without work after which a slot counts as idle
};

// Launchers (defined in the kernel translation units).
cudaError_t launch_engine_f64(const Params& p, cudaStream_t s);
cudaError_t launch_engine_f32(const Params& p, cudaStream_t s);
// nv = 7: recursion on the 7 unit vectors; nv = 2: on the proposal's vectors o and v
cudaError_t launch_engine_f64(const Params& p, int nv, cudaStream_t s);
cudaError_t launch_engine_f32(const Params& p, int nv, cudaStream_t s);
cudaError_t launch_team_f64(const TeamJob* d_jobs, int njobs, int grid, int smem, cudaStream_t s);
// nv: the vectors of every job's recursion (p.nv), 0 when they differ; 1: even lattices on two vectors only;
// kPackedTiles: those with all vectors in global memory
constexpr int kPackedTiles = 3;
cudaError_t launch_team_f32(const TeamJob* d_jobs, int njobs, int grid, int smem, cudaStream_t s, bool comp, int nv);
// co-resident CTAs of the kernel launch_team_* takes for comp and nv, and its static shared memory
// (bytes); nv < 0: the fewest of any
cudaError_t team_max_ctas(int precision, int smem, bool comp, int nv, int* out);
cudaError_t team_static_smem(int precision, bool comp, int nv, int* out);
// launch_team_* through cudaLaunchKernelEx with the cooperative attribute (capturable in a CUDA graph)
cudaError_t launch_team_ex_f64(const TeamJob* d_jobs, int njobs, int grid, int smem, cudaStream_t s);
cudaError_t launch_team_ex_f32(const TeamJob* d_jobs, int njobs, int grid, int smem, cudaStream_t s, bool comp, int nv);
cudaError_t launch_server(const ServerArgs& a, int grid, int smem, cudaStream_t s);
// one cluster of C CTAs per job (recursion on the proposal's vectors)
cudaError_t launch_cluster_f64(const TeamJob* d_jobs, int njobs, int C, int vec_bytes, int smem, cudaStream_t s);
cudaError_t launch_cluster_f32(const TeamJob* d_jobs, int njobs, int C, int vec_bytes, int smem, cudaStream_t s,
                               bool comp);
cudaError_t cluster_max_active(int precision, int C, int smem, int* out);
// the packed engines (even L; p.pk_cy set): engine 0 FP64 and 1 FP32-mixed, one
// cluster of C CTAs per job; 2 FP64 with small tiles (pk64_smem_bytes)
cudaError_t launch_packed(int engine, const TeamJob* d_jobs, int njobs, int C, int smem, cudaStream_t s);
cudaError_t launch_packed_single(int engine, const Params& p, int smem, cudaStream_t s);
cudaError_t launch_packed64_moments(const Params& p, int smem, cudaStream_t s);
cudaError_t packed_max_active(int engine, int C, int smem, int* out);
cudaError_t packed_static_smem(int engine, int* out);
// a single chain on one CTA: even L, at most kThreads sites (FP32: 2 kThreads)
// (FP64: at most kThreads that advance the sites, and eight warps for the sums)
inline int one_cta_threads(int precision, int N) { return precision != 0 && N <= kThreads ? kThreads : 2 * kThreads; }
// FP32-mixed chains on one CTA up to this size (L = 4) run the FP64 chains' fixed point: their
// few levels stand apart at the resolution of a large M, which magnifies the rounding of FP32
// vectors to 1e-6 t (L = 4, M = 1024; L = 6: 2e-7), and the steps are bound by latency either way.
constexpr int kOneCtaExact = 64;
constexpr int kOneCtaHist = 32;  // vectors an FP64 chain keeps in shared memory
cudaError_t launch_one_cta(int precision, const Params& p, int smem, cudaStream_t s);
bool one_cta_fits(int precision, int N, int smem);
// a single FP64 chain on p.ncta CTAs of a cooperative grid
cudaError_t launch_packed64_grid(const Params& p, int smem, cudaStream_t s);
cudaError_t packed64_grid_max_ctas(int smem, int* out);
// static shared memory of the cluster engine of a precision (bytes)
cudaError_t cluster_static_smem(int precision, int* out);
cudaError_t server_max_ctas(int smem, int* out);
// K: the number of Chebyshev nodes (the FFT buffer of the tail holds K double2)
int engine_smem_bytes(int K);
int single_smem_bytes(int K, int precision, int win_max = 0);
// static shared memory of the FP64 single-chain engine (bytes)
cudaError_t engine_static_smem_f64(int* out);
cudaError_t engine_max_ctas(int precision, int K, int* out);
cudaError_t launch_build_hoppings(const Params& p, cudaStream_t s);
// FP32-mixed single chain on seven thread-block clusters of 16 CTAs, one per
// local unit vector (L = 32 only; p.bar[0..1] are its update counters)
cudaError_t launch_vcluster_f32(const Params& p, cudaStream_t s);
// how many of that engine's clusters can be resident at once for K nodes
cudaError_t vcluster_max_clusters(int K, int* out);
constexpr int kVcLattice = 32;
constexpr int kVcCtas = 16 * 7;
cudaError_t launch_setup_tables(const Params& p, int kernel_kind, double lambda, cudaStream_t s);

}  // namespace gfmc
