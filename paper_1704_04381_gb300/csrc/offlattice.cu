// offlattice.cu -- Rosenbluth growth in real space (Guo & Baulin, Section
// 3.3.3, Algorithm 2): k trial positions on the unit sphere around the chain
// end, scored against every earlier non-bonded bead by hard-sphere overlap or
// a truncated Lennard-Jones energy; W is multiplied by the sum of the trial
// weights and one trial is drawn in proportion to its weight.
//
// GB300 mapping: a group of G lanes (G = 8, 16 or 32) grows one chain, so a
// warp holds 32/G chains; each lane owns T = ceil(k/G) trials.  Each step:
//  1. the group scans the earlier beads G at a time and keeps, in ballot
//     order (ascending bead index), those within 1 + R of the end (R = sigma
//     or the cutoff); only those can reach a trial.  The kept displacement
//     g = end - r_j and c = 1 + |g|^2 go to a shared list;
//  2. every lane draws its trial directions u (Philox, 24-bit uniforms; one
//     call gives two trials) and evaluates d^2 = |g + u|^2 = c + 2 g.u against
//     the list (three FMAs per pair, entries broadcast from shared memory);
//  3. free flags / weights are combined with group ballots and scans, and the
//     selection draw picks the trial.
// Positions are float-float (hi + lo) sums of the FP32 directions, so they
// carry only the directions' own rounding.  Every FP32 decision comes with a
// bound on its distance from the FP64 result (d^2 within G_i of sigma^2 or of
// the cutoff, or the selection draw within E of a prefix-sum boundary); when
// the bound is not met the group replays the chain's positions in FP64 from
// its chosen trials, stores them back (so later steps start from exact
// positions), and re-decides the step with the sequential FP64 arithmetic of
// the definition.  The grown path is the one an FP64 implementation takes.
//
// Scheduling: the grid is what the GPU holds at once, and every group takes
// its next chain from a counter (chains differ in cost by their re-decisions
// and dead ends).  Lennard-Jones chains, and both potentials in a batch, grow
// with the kernels below; hard spheres grow with those of offlattice_wide.cuh,
// which takes the same steps with fewer lanes per chain.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "internal.cuh"
#include "offlattice_chain.cuh"
#include "offlattice_wide.cuh"

namespace rosen {
namespace {


template <int G, int T, bool LJ>
__global__ void __launch_bounds__(256, 4) offlattice_group_kernel(const OffArgs a, int chains_per_block)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *logm = reinterpret_cast<float *>(smem_raw);
    fill_log_table(logm);
    __syncthreads();

    const Group<G> g;
    const int cib = threadIdx.x / G;
    const int64_t c = (int64_t)blockIdx.x * chains_per_block + cib;
    if (c >= a.C) return;     // whole groups leave together
    const ChainSmem w = carve(smem_raw + kTable * sizeof(float) +
                                  (size_t)cib * chain_smem_bytes(a.N, LJ), a.N, LJ);
    off_chain<G, T, LJ>(a, c, w, g, logm);
}

// The same growth with chains handed out one at a time: every group takes
// its next chain from a counter as soon as it is done with the last, so a
// block holds no lanes idle while its slowest chain finishes (chains differ
// in their number of FP64 re-decisions and dead ends).  The grid is what the
// GPU holds at once.
template <int G, int T, bool LJ>
__global__ void __launch_bounds__(256, 4) offlattice_queue_kernel(const OffArgs a,
                                                                  int chains_per_block,
                                                                  unsigned long long *next,
                                                                  int64_t c_lo, int64_t c_hi)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *logm = reinterpret_cast<float *>(smem_raw);
    fill_log_table(logm);
    __syncthreads();

    const Group<G> g;
    const int cib = threadIdx.x / G;
    const ChainSmem w = carve(smem_raw + kTable * sizeof(float) +
                                  (size_t)cib * chain_smem_bytes(a.N, LJ), a.N, LJ);
    for (;;) {
        unsigned long long c = 0;
        if (g.gl == 0) c = (unsigned long long)c_lo + atomicAdd(next, 1ull);
        c = g.bcast(c, 0);
        if (c >= (unsigned long long)c_hi) break;
        off_chain<G, T, LJ>(a, (int64_t)c, w, g, logm);
    }
}

// Persistent batch kernel for one (G, T, potential) class.  The queue holds
// (ensemble, chain range) items of up to chains_per_block chains, sorted by
// decreasing cost; ticket t of a counter is chain t % chains_per_block of
// item t / chains_per_block.  Every group takes its own tickets, keeps the
// arguments of its current ensemble in shared memory, and grows each chain
// with off_chain -- the code of the single-ensemble Lennard-Jones kernels; hard
// spheres alone grow with offlattice_wide_kernel, whose outputs equal off_chain's
// bit for bit.  No group waits for the others of its block.
template <int G, int T, bool LJ>
__global__ void __launch_bounds__(256, 4) offlattice_batch_kernel(const OffArgs *__restrict__ ens,
                                                                  const BatchItem *__restrict__ items,
                                                                  int n_items, int *head,
                                                                  int chains_per_block, int Nmax)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ OffArgs sa[256 / G];
    float *logm = reinterpret_cast<float *>(smem_raw);
    fill_log_table(logm);
    __syncthreads();
    const Group<G> g;
    const int cib = threadIdx.x / G;
    const ChainSmem w = carve(smem_raw + kTable * sizeof(float) +
                                  (size_t)cib * chain_smem_bytes(Nmax, LJ), Nmax, LJ);
    OffArgs &my = sa[cib];
    const unsigned int tickets = (unsigned int)n_items * (unsigned int)chains_per_block;
    unsigned int *next = reinterpret_cast<unsigned int *>(head);
    int cur = -1;     // the ensemble whose arguments are in my
    for (;;) {
        unsigned int t = 0;
        if (g.gl == 0) t = atomicAdd(next, 1u);
        t = g.bcast(t, 0);
        if (t >= tickets) break;
        const BatchItem bi = items[t / (unsigned int)chains_per_block];
        const unsigned int off = t % (unsigned int)chains_per_block;
        if (off >= bi.n) continue;
        if ((int)bi.ens != cur) {
            constexpr int kWords = (int)(sizeof(OffArgs) / 4);
            for (int q = g.gl; q < kWords; q += G)
                reinterpret_cast<uint32_t *>(&my)[q] =
                    reinterpret_cast<const uint32_t *>(&ens[bi.ens])[q];
            __syncwarp(g.mask);
            cur = (int)bi.ens;
        }
        off_chain<G, T, LJ, ChainSmem, true>(my, bi.c0 + off, w, g, logm);
    }
}

// Directions exactly as the growth kernels compute them (for verification).
__global__ void sphere_points_kernel(const uint2 *words, int64_t n, float *out)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const uint2 v = words[q];
    const float3 u = dir32(v.x, v.y);
    out[3 * q + 0] = u.x;
    out[3 * q + 1] = u.y;
    out[3 * q + 2] = u.z;
}

// The hard-sphere kernel's fast directions (twice the unit vectors; halving is
// exact).
__global__ void sphere_points_fast_kernel(const uint2 *words, int64_t n, float *out)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const uint2 v = words[q];
    float2 x, y, z;
    fast_dirs_x2(make_uint4(v.x, v.y, v.x, v.y), x, y, z);
    out[3 * q + 0] = 0.5f * x.x;
    out[3 * q + 1] = 0.5f * y.x;
    out[3 * q + 2] = 0.5f * z.x;
}

// Float-float directions as the Lennard-Jones kernels commit them.
__global__ void sphere_points_ff_kernel(const uint2 *words, int64_t n, float *out)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const uint2 v = words[q];
    float xh, xl, yh, yl, z;
    dir_ff(v.x, v.y, xh, xl, yh, yl, z);
    out[5 * q + 0] = xh;
    out[5 * q + 1] = xl;
    out[5 * q + 2] = yh;
    out[5 * q + 3] = yl;
    out[5 * q + 4] = z;
}

// Chains per block: 256 threads, fewer if the chains' shared memory would
// exceed 96 KB (at least one warp).
int chains_per_block_for(int G, int N, bool lj)
{
    const size_t per_chain = chain_smem_bytes(N, lj);
    int chains = 256 / G;
    while (chains > 32 / G && (size_t)chains * per_chain > 96 * 1024) chains -= 32 / G;
    return chains;
}

// Scratch of a range launch: the chain counter, zeroed by every launch.
// Launches that may run at the same time need counters of their own.
constexpr size_t kScratchHeader = 16;

int set_cuda_error(cudaError_t e)
{
    return set_error(ROSEN_ECUDA, "rosen_offlattice_grow: %s", cudaGetErrorString(e));
}

// ---- Lennard-Jones: a group of G lanes per chain -----------------------------------
// Local chains [c_lo, c_hi): groups take them from the counter, the grid is
// what the GPU holds at once.  Without a counter, one block per
// chains_per_block chains (the same outputs).
template <int G, int T>
int launch_lj(const OffArgs &a, int64_t c_lo, int64_t c_hi, void *counter, cudaStream_t s,
              int64_t *resident)
{
    const int chains = chains_per_block_for(G, a.N, true);
    const size_t smem = kTable * sizeof(float) + (size_t)chains * chain_smem_bytes(a.N, true);
    const int threads = chains * G;
    const int64_t blocks = (c_hi - c_lo + chains - 1) / chains;
    if (!counter && !resident) {
        allow_max_smem(offlattice_group_kernel<G, T, true>);
        offlattice_group_kernel<G, T, true><<<(unsigned)blocks, threads, smem, s>>>(a, chains);
        return check_launch("rosen_offlattice_grow");
    }
    int dev = 0, sms = 0, bps = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = allow_max_smem(offlattice_queue_kernel<G, T, true>);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, offlattice_queue_kernel<G, T, true>,
                                                          threads, smem);
    if (resident) {
        *resident = e == cudaSuccess ? (int64_t)bps * sms * chains : 0;
        if (e != cudaSuccess) cudaGetLastError();
        return ROSEN_OK;
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, kScratchHeader, s);
    if (e == cudaSuccess) {
        int64_t grid = (int64_t)(bps > 0 ? bps : 1) * sms;
        if (grid > blocks) grid = blocks;
        offlattice_queue_kernel<G, T, true><<<(unsigned)grid, threads, smem, s>>>(
            a, chains, static_cast<unsigned long long *>(counter), c_lo, c_hi);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? ROSEN_OK : set_cuda_error(e);
}

// ---- hard spheres: the wide kernel ---------------------------------------------------
using WideFn = void (*)(const OffArgs, const WideShape, unsigned long long *, int64_t, int64_t);

struct WidePlan {
    WideFn fn;
    int G, warps;        // lanes per chain, warps per block
    size_t smem;
    WideShape sh;
};

// Shape for n chains of N beads and k trials whose sums follow gref lanes per
// chain.  G is the fewest lanes that hold k trials (8 each) and whose scan bits
// fit a word (N <= 32 G); with few chains it doubles while the warps stay
// within 9 per SM (k > 16: 12, k > 32: 14, as more trials keep more lanes busy),
// where the lanes would idle otherwise and a step's latency counts.  G = 4 / 8 /
// 16 / 32, us: N = 64, k = 32, 700 chains 151 / 123 / 97 / 95, 2000 153 / 125 /
// 106 / 131, 3500 156 / 133 / 115 / -; k = 64 (8 / 16 / 32), 2000: 162 / 148 /
// 129; N = 129, k = 64 (8 / 16 / 32), 1500 286 / 222 / 198, 2000 336 / 252 / 226;
// k = 16, 2000 (8 / 16 / 32) 197 / 187 / 218.  A block has the warps that fill an
// SM's shared memory best, at most 16 (128 registers a thread), fewer where there
// are not enough chains for every SM.
WidePlan wide_plan(const OffArgs &a, int gref, int64_t n, int sms)
{
    WidePlan w;
    const int N = a.N, k = a.k;
    int G = 4;
    while (8 * G < k || 32 * G < N) G *= 2;
    const int few = k <= 16 ? 9 : (k <= 32 ? 12 : 14);
    while (G < 32 && n * 2 * G <= (int64_t)32 * few * sms) G *= 2;
    const int T = ((k + G - 1) / G + 1) / 2 * 2;
    w.fn = nullptr;
#define ROSEN_WIDE(GG, TT) if (G == GG && T == TT) w.fn = offlattice_wide_kernel<GG, TT>;
    ROSEN_WIDE(4, 2) ROSEN_WIDE(4, 4) ROSEN_WIDE(4, 6) ROSEN_WIDE(4, 8)
    ROSEN_WIDE(8, 2) ROSEN_WIDE(8, 4) ROSEN_WIDE(8, 6) ROSEN_WIDE(8, 8)
    ROSEN_WIDE(16, 2) ROSEN_WIDE(16, 4) ROSEN_WIDE(16, 6) ROSEN_WIDE(16, 8)
    ROSEN_WIDE(32, 2) ROSEN_WIDE(32, 4)
#undef ROSEN_WIDE
    w.G = G;
    w.sh.np = wide_np(N, G);
    w.sh.stride = wide_stride(N, G);
    w.sh.gref = gref;
    // |g|^2 from the hi words alone differs from the float-float value by the
    // lo words (<= 6e-8 N per axis) and FP32 rounding (as in
    // rosen_offlattice_grow_long); doubled.
    const double rf2 = a.rf2, rf = sqrt(rf2), d = 6e-8 * N + 1e-6;
    w.sh.pre2 = (float)(rf2 + 2.0 * (3.5 * (rf + 1.0) * d + 3.0 * d * d + 4e-6 * rf2) + 1e-6);
    const size_t head = kTable * sizeof(float) + kWideSelBytes;
    const size_t per_warp = (size_t)(32 / G) * w.sh.stride * sizeof(float);
    const size_t sm = (size_t)max_dynamic_smem() + 1024;     // (1 KB per block is reserved)
    int best = 0;
    w.warps = 1;
    for (int q = 1; q <= 16; ++q) {
        const int held = std::min((int)(sm / (head + q * per_warp + 1024)), 16 / q) * q;
        if (held > best) {
            best = held;
            w.warps = q;
        }
    }
    const int64_t warps = (n * G + 31) / 32;
    if (warps < (int64_t)w.warps * sms) w.warps = (int)((warps + sms - 1) / sms);
    w.smem = head + w.warps * per_warp;
    return w;
}

int launch_wide(const OffArgs &a, int gref, int64_t c_lo, int64_t c_hi, void *counter,
                cudaStream_t s, int64_t *resident)
{
    int dev = 0, sms = 0, bps = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return set_cuda_error(e);
    const WidePlan w = wide_plan(a, gref, resident ? INT64_MAX / 64 : c_hi - c_lo, sms);
    const int64_t per_block = (int64_t)w.warps * (32 / w.G);
    e = allow_max_smem(w.fn);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, w.fn, w.warps * 32, w.smem);
    if (resident) {
        *resident = e == cudaSuccess ? (int64_t)bps * sms * per_block : 0;
        if (e != cudaSuccess) cudaGetLastError();
        return ROSEN_OK;
    }
    if (e == cudaSuccess && counter) e = cudaMemsetAsync(counter, 0, kScratchHeader, s);
    if (e == cudaSuccess) {
        int64_t grid = (c_hi - c_lo + per_block - 1) / per_block;
        if (counter) grid = std::min(grid, (int64_t)(bps > 0 ? bps : 1) * sms);
        w.fn<<<(unsigned)grid, w.warps * 32, w.smem, s>>>(
            a, w.sh, static_cast<unsigned long long *>(counter), c_lo, c_hi);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? ROSEN_OK : set_cuda_error(e);
}

// Local chains [c_lo, c_hi) with G lanes per chain (hard spheres: sums in that
// order), with or without a chain counter; or the chains the GPU grows at
// once (resident != nullptr).
int launch_range(const OffArgs &a, bool lj, int G, int64_t c_lo, int64_t c_hi, void *counter,
                 cudaStream_t s, int64_t *resident = nullptr)
{
    if (!lj) return launch_wide(a, G, c_lo, c_hi, counter, s, resident);
    const int T = (a.k + G - 1) / G;
#define ROSEN_LAUNCH(GG, TT) return launch_lj<GG, TT>(a, c_lo, c_hi, counter, s, resident);
    if (G == 8) {
        if (T <= 1) ROSEN_LAUNCH(8, 1)
        if (T <= 2) ROSEN_LAUNCH(8, 2)
        ROSEN_LAUNCH(8, 4)
    }
    if (G == 16) {
        if (T <= 1) ROSEN_LAUNCH(16, 1)
        if (T <= 2) ROSEN_LAUNCH(16, 2)
        ROSEN_LAUNCH(16, 4)
    }
    if (T <= 1) ROSEN_LAUNCH(32, 1)
    if (T <= 2) ROSEN_LAUNCH(32, 2)
    ROSEN_LAUNCH(32, 4)
#undef ROSEN_LAUNCH
}

// The batch kernel of class (G, T, LJ) through one function pointer type.
using BatchFn = void (*)(const OffArgs *, const BatchItem *, int, int *, int, int);

template <int G, int T, bool LJ>
BatchFn batch_fn()
{
    return offlattice_batch_kernel<G, T, LJ>;
}

BatchFn pick_batch(int G, int T, bool lj)
{
#define ROSEN_PICK(GG, TT)                                                              \
    if (G == GG && T == TT) return lj ? batch_fn<GG, TT, true>() : batch_fn<GG, TT, false>();
    ROSEN_PICK(8, 1) ROSEN_PICK(8, 2) ROSEN_PICK(8, 4)
    ROSEN_PICK(16, 1) ROSEN_PICK(16, 2) ROSEN_PICK(16, 4)
    ROSEN_PICK(32, 1) ROSEN_PICK(32, 2) ROSEN_PICK(32, 4)
#undef ROSEN_PICK
    return nullptr;
}

}  // namespace

int offlattice_validate(const rosen_offlattice_params *p, const rosen_offlattice_out *o, int nmax,
                        const char *fn)
{
    if (!p || !o) return set_error(ROSEN_EINVAL, "%s: NULL params or outputs", fn);
    if (p->N < 2 || p->N > nmax)
        return set_error(ROSEN_EINVAL, "%s: N = %d outside [2, %d]", fn, p->N,
                         nmax);
    if (p->k < 1 || p->k > ROSEN_KMAX)
        return set_error(ROSEN_EINVAL, "%s: k = %d outside [1, %d]", fn, p->k,
                         ROSEN_KMAX);
    if (p->C < 0 || p->chain0 < 0 || p->chain0 + p->C > (int64_t(1) << 32))
        return set_error(ROSEN_EINVAL,
                         "%s: chains [%lld, %lld) outside [0, 2^32)", fn,
                         (long long)p->chain0, (long long)(p->chain0 + p->C));
    if (p->potential != ROSEN_HARD_SPHERE && p->potential != ROSEN_LJ)
        return set_error(ROSEN_EINVAL, "%s: unknown potential %d", fn, p->potential);
    if (!(p->sigma >= 0.0) || !isfinite(p->sigma) || p->sigma > 4.0)
        return set_error(ROSEN_EINVAL, "%s: sigma must lie in [0, 4]", fn);
    if (p->potential == ROSEN_LJ &&
        (!(p->cutoff > 0.0) || !isfinite(p->cutoff) || p->cutoff > 8.0 || p->sigma <= 0.0))
        return set_error(ROSEN_EINVAL,
                         "%s: LJ needs sigma > 0 and 0 < cutoff <= 8", fn);
    if (!(p->beta_eps >= 0.0) || !isfinite(p->beta_eps))
        return set_error(ROSEN_EINVAL, "%s: beta_eps must be finite and >= 0", fn);
    if (p->flags & ~(ROSEN_STORE_TRACE | ROSEN_STORE_COORDS))
        return set_error(ROSEN_EINVAL, "%s: unknown flags 0x%x", fn, p->flags);
    if ((p->flags & ROSEN_STORE_TRACE) && !o->trace)
        return set_error(ROSEN_EINVAL, "%s: ROSEN_STORE_TRACE without trace", fn);
    if ((p->flags & ROSEN_STORE_COORDS) && !o->coords)
        return set_error(ROSEN_EINVAL, "%s: ROSEN_STORE_COORDS without coords", fn);
    const int G = p->lanes_per_chain;
    if (G != 0 && G != 8 && G != 16 && G != 32)
        return set_error(ROSEN_EINVAL,
                         "%s: lanes_per_chain must be 0, 8, 16 or 32", fn);
    if (G != 0 && (p->k + G - 1) / G > 4)
        return set_error(ROSEN_EINVAL,
                         "%s: k = %d needs more than 4 trials per lane", fn, p->k);
    if (p->max_attempts < 0 || p->max_attempts > ROSEN_MAX_ATTEMPTS)
        return set_error(ROSEN_EINVAL, "%s: max_attempts = %d outside [0, %d]", fn,
                         p->max_attempts, ROSEN_MAX_ATTEMPTS);
    return ROSEN_OK;
}

// Default lanes per chain of off_chain with shared memory (measured on GB300).
// Lennard-Jones at N = 64 runs best with a whole warp per chain once k > 16, with
// 16 lanes below.  Longer chains spend more of each step in the scan of earlier
// beads, which a whole warp does twice as fast: from N = 100 every k takes 32
// lanes (k = 16, N = 128 / 256: 25.9 / 46.0 ms with 32 lanes against 29.3 / 71.8
// with 16, a bead at a time).  For hard spheres in rosen_offlattice_grow the value
// is only the order of the R_g^2 sum (wide_plan picks the lanes); in a batch's
// class kernel it is the shape before tuning (N = 64, k = 32, 16 lanes: two chains
// per warp).  N = 0: the chain length is not known (the long-chain kernel, whose
// near lists come from cells).
int offlattice_default_lanes(int k, bool lj, int N)
{
    if (N >= 100) return 32;
    if (lj) return k <= 16 ? 16 : 32;
    if (k <= 64) return 16;
    return 32;
}

size_t offlattice_args_size() { return sizeof(OffArgs); }

void offlattice_make_args(const rosen_offlattice_params *p, const rosen_offlattice_out *o,
                          unsigned long long *counters, void *out)
{
    OffArgs a;
    memset(&a, 0, sizeof a);
    a.key = philox_keys(p->seed);
    a.ens = p->ensemble;
    a.chain0 = (uint32_t)p->chain0;
    a.N = p->N;
    a.k = p->k;
    a.C = p->C;
    const bool lj = p->potential == ROSEN_LJ;
    const double sig = p->sigma;
    const double R = lj ? p->cutoff : sig;
    a.sig2 = (float)(sig * sig);
    a.rc2 = lj ? (float)(p->cutoff * p->cutoff) : 0.f;
    a.rf2 = (float)((1.0 + R) * (1.0 + R) * 1.001 + 1e-3);
    a.rf = (float)sqrt((double)a.rf2 * 1.0001);
    a.beta4 = lj ? (float)(4.0 * p->beta_eps) : 0.f;
    a.six_sig2 = lj ? 6.f / a.sig2 : 0.f;
    a.dband = (float)(lj ? p->cutoff : sig * 1.001);
    if (lj) {
        const double sc = (sig * sig) / (p->cutoff * p->cutoff), s3 = sc * sc * sc;
        a.ucut2 = (float)(2.0 * fabs(s3 * (s3 - 1.0)));
    }
    a.sig2d = sig * sig;
    a.rc2d = lj ? p->cutoff * p->cutoff : 0.0;
    a.beta_eps = p->beta_eps;
    a.logw = o->logw;
    a.r2 = o->r2;
    a.rg2 = o->rg2;
    a.alive = o->alive;
    a.trace = (p->flags & ROSEN_STORE_TRACE) ? o->trace : nullptr;
    a.coords = (p->flags & ROSEN_STORE_COORDS) ? o->coords : nullptr;
    // Position drift from exact per step for chains that commit float-float
    // directions (1.5e-12 per component) with float-float adds whose rounding
    // grows with |r| <= N (7e-15 N), both with margin; kernels that commit
    // FP32 directions use 4e-7 instead.
    a.drift = (float)(4e-12 + 1e-14 * p->N);
    a.counters = counters;
    a.attempts = o->attempts;
    a.max_att = p->max_attempts > 1 ? (uint32_t)p->max_attempts : 1u;
    memcpy(out, &a, sizeof a);
}

namespace {

int lanes_of(const rosen_offlattice_params *p)
{
    return p->lanes_per_chain
               ? p->lanes_per_chain
               : offlattice_default_lanes(p->k, p->potential == ROSEN_LJ, p->N);
}

}  // namespace

// A whole ensemble: the chain counter comes from the stream-ordered allocator;
// if that fails, the chains grow without one.
int offlattice_launch(const rosen_offlattice_params *p, const rosen_offlattice_out *o,
                      unsigned long long *counters, cudaStream_t s)
{
    OffArgs a;
    offlattice_make_args(p, o, counters, &a);
    void *buf = nullptr;
    if (cudaMallocAsync(&buf, kScratchHeader, s) != cudaSuccess) {
        cudaGetLastError();   // clear the failed allocation
        buf = nullptr;
    }
    const int st = launch_range(a, p->potential == ROSEN_LJ, lanes_of(p), 0, p->C, buf, s);
    const cudaError_t f = buf ? cudaFreeAsync(buf, s) : cudaSuccess;
    if (st != ROSEN_OK) return st;
    if (f != cudaSuccess)
        return set_error(ROSEN_ECUDA, "rosen_offlattice_grow: freeing the work counter: %s",
                         cudaGetErrorString(f));
    return ROSEN_OK;
}

size_t offlattice_range_counter_bytes() { return kScratchHeader; }

int offlattice_grow_range(const rosen_offlattice_params *p, const rosen_offlattice_out *o,
                          int64_t c_lo, int64_t c_hi, void *counter, cudaStream_t s)
{
    if (c_hi <= c_lo) return ROSEN_OK;
    OffArgs a;
    offlattice_make_args(p, o, reinterpret_cast<unsigned long long *>(o->counters), &a);
    return launch_range(a, p->potential == ROSEN_LJ, lanes_of(p), c_lo, c_hi, counter, s);
}

int64_t offlattice_resident_chains(const rosen_offlattice_params *p)
{
    OffArgs a;
    const rosen_offlattice_out none = {};
    offlattice_make_args(p, &none, nullptr, &a);
    int64_t r = 0;
    launch_range(a, p->potential == ROSEN_LJ, lanes_of(p), 0, 0, nullptr, nullptr, &r);
    return r;
}

int offlattice_batch_prepare(int G, int T, bool lj, int Nmax, int *chains_per_block, size_t *smem,
                             int *blocks_per_sm)
{
    const BatchFn fn = pick_batch(G, T, lj);
    if (!fn) return set_error(ROSEN_EINVAL, "no real-space batch kernel for G=%d T=%d", G, T);
    *chains_per_block = chains_per_block_for(G, Nmax, lj);
    *smem = kTable * sizeof(float) + (size_t)(*chains_per_block) * chain_smem_bytes(Nmax, lj);
    cudaError_t e = allow_max_smem(fn);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn,
                                                          (*chains_per_block) * G, *smem);
    if (e != cudaSuccess)
        return set_error(ROSEN_ECUDA, "real-space batch set-up: %s", cudaGetErrorString(e));
    return ROSEN_OK;
}

void offlattice_batch_launch(int G, int T, bool lj, const void *dev_args, const BatchItem *items,
                             int n_items, int *head, int chains_per_block, int Nmax, size_t smem,
                             int grid, cudaStream_t s)
{
    const BatchFn fn = pick_batch(G, T, lj);
    fn<<<grid, chains_per_block * G, smem, s>>>(reinterpret_cast<const OffArgs *>(dev_args), items,
                                               n_items, head, chains_per_block, Nmax);
}

}  // namespace rosen

using namespace rosen;

extern "C" int rosen_offlattice_grow(const rosen_offlattice_params *p,
                                     const rosen_offlattice_out *o, void *stream)
{
    const int st = offlattice_validate(p, o);
    if (st != ROSEN_OK) return st;
    if (p->C == 0) return ROSEN_OK;
    return offlattice_launch(p, o, reinterpret_cast<unsigned long long *>(o->counters),
                             (cudaStream_t)stream);
}

extern "C" int rosen_sphere_points(const uint32_t *words, int64_t n, float *out, void *stream)
{
    if (n < 0) return set_error(ROSEN_EINVAL, "rosen_sphere_points: n < 0");
    if (n > 0 && (!words || !out)) return set_error(ROSEN_EINVAL, "rosen_sphere_points: NULL");
    if (reinterpret_cast<uintptr_t>(words) & 7u)
        return set_error(ROSEN_EINVAL, "rosen_sphere_points: words must be 8-byte aligned");
    if (n == 0) return ROSEN_OK;
    const int threads = 256;
    sphere_points_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0,
                           (cudaStream_t)stream>>>(reinterpret_cast<const uint2 *>(words), n, out);
    return check_launch("rosen_sphere_points");
}

extern "C" int rosen_sphere_points_fast(const uint32_t *words, int64_t n, float *out, void *stream)
{
    if (n < 0) return set_error(ROSEN_EINVAL, "rosen_sphere_points_fast: n < 0");
    if (n > 0 && (!words || !out)) return set_error(ROSEN_EINVAL, "rosen_sphere_points_fast: NULL");
    if (reinterpret_cast<uintptr_t>(words) & 7u)
        return set_error(ROSEN_EINVAL, "rosen_sphere_points_fast: words must be 8-byte aligned");
    if (n == 0) return ROSEN_OK;
    const int threads = 256;
    sphere_points_fast_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0,
                                (cudaStream_t)stream>>>(reinterpret_cast<const uint2 *>(words), n,
                                                        out);
    return check_launch("rosen_sphere_points_fast");
}

extern "C" int rosen_sphere_points_ff(const uint32_t *words, int64_t n, float *out, void *stream)
{
    if (n < 0) return set_error(ROSEN_EINVAL, "rosen_sphere_points_ff: n < 0");
    if (n > 0 && (!words || !out)) return set_error(ROSEN_EINVAL, "rosen_sphere_points_ff: NULL");
    if (reinterpret_cast<uintptr_t>(words) & 7u)
        return set_error(ROSEN_EINVAL, "rosen_sphere_points_ff: words must be 8-byte aligned");
    if (n == 0) return ROSEN_OK;
    const int threads = 256;
    sphere_points_ff_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0,
                              (cudaStream_t)stream>>>(reinterpret_cast<const uint2 *>(words), n,
                                                      out);
    return check_launch("rosen_sphere_points_ff");
}
