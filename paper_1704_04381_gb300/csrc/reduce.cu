// reduce.cu -- FP64 ensemble reduction of Rosenbluth-weighted observables
// (Guo & Baulin, Eq. 2 with W as the importance weight; Eq. 9 for Z_N).
//
// Rosenbluth weights span hundreds of orders of magnitude, so the sums are
// formed in FP64 relative to a maximum (log-sum-exp).  The chains are cut into
// fixed tiles of kTile chains; a cluster of kTileCtas blocks reduces one tile
// to a partial (its max M_t and the sums scaled by exp(-M_t)), and a cluster
// of kFinalCtas blocks merges an ensemble's partials: their maximum first, then
// every partial scaled once.  Tiles, the in-tile order and the merge order
// depend only on C, so the result is bit-for-bit deterministic.
//
// Bound by the FP64 pipe (a warp instruction takes it 16 cycles) for many
// chains and by latency for few.  So a tile is spread over four SMs, the block
// sums go through shared memory (a hundred warp instructions where shuffles
// took 360), the weights' exponential takes 11 FP64 operations, and the merge
// takes one exponential per partial instead of two per pair merged and forms
// the statistics on different lanes.  GB300, one block per tile and a tree of
// pairwise merges before, and now: 10^5 chains 59.5 -> 27.1 us, 10^7 chains
// 0.957 -> 0.730 ms (weights from counts 1.130 -> 0.826 ms).
#include <math.h>
#include <string.h>

#include <mutex>

#include <cooperative_groups.h>

#include "common.cuh"
#include "internal.cuh"

namespace rosen {
namespace {

namespace cg = cooperative_groups;

constexpr int kTile = 2048;
constexpr int kTileCtas = 4;
constexpr int kThreads = 128;
constexpr int kPerThread = kTile / kTileCtas / kThreads;
constexpr int kFinalCtas = 8;
constexpr int kSums = 10;      // the eight sums, live chains, growths

struct Partial {
    double M;          // max log W in the tile (-inf: no live chain)
    double s[8];       // S0 S1 S2 Q0 Q1a Q2a Q1b Q2b, scaled by exp(-M) / exp(-2M)
    double alive;
    double n;          // growths in the tile: chains, or their attempts (restart mode)
    double pad;
};

struct ReduceArgs {
    int32_t kind, N, k, use_counts;
    int64_t C;
    const float *logw;
    const uint4 *counts;
    const int32_t *r2_i;
    const int64_t *n2rg2;
    const float *r2_f;
    const float *rg2_f;
    const uint16_t *attempts;   // optional: growths per chain (restart mode)
    double logm[8];     // log(m) in FP64, m = 0..6
    double inv_n2;      // 1 / N^2
};

__device__ __forceinline__ void load_chain(const ReduceArgs &a, int64_t c, double &lw,
                                           double &A1, double &A2)
{
    if (a.kind == ROSEN_REDUCE_LATTICE) {
        if (a.use_counts) {
            const uint4 v = a.counts[c];
            if (v.x & 0xFFFFu) {
                lw = -INFINITY;
            } else {
                // log W = sum_m counts[m] log m over the primes of m = 2 .. 6,
                // exact up to FP64 rounding.
                const uint32_t c2 = v.y & 0xFFFFu, c3 = v.y >> 16, c4 = v.z & 0xFFFFu,
                               c5 = v.z >> 16, c6 = v.w & 0xFFFFu;
                const double s = fma((double)(c2 + 2u * c4 + c6), a.logm[2],
                                     fma((double)(c3 + c6), a.logm[3], (double)c5 * a.logm[5]));
                lw = s;
            }
        } else {
            lw = (double)a.logw[c];
        }
        A1 = (double)a.r2_i[c];
        A2 = (double)a.n2rg2[c] * a.inv_n2;
    } else {
        lw = (double)a.logw[c];
        A1 = (double)a.r2_f[c];
        A2 = (double)a.rg2_f[c];
    }
}

// exp(x) for the weights, x <= 0: the table-driven method of Tang (ACM Trans.
// Math. Softw. 15 (1989) 144).  x = (64 k + j) ln2 / 64 + r with |r| <= ln2 / 128;
// exp(x) = 2^k 2^(j/64) (1 + p(r)), 2^(j/64) from a table as a sum of two
// doubles, p the Taylor polynomial of e^r - 1 to r^6 with r^6 economised (its
// Chebyshev polynomial of degree 6 left out) to degree 5: within 3e-18.  11 FP64
// operations.  Below -700, and for NaN, the library's exp.
constexpr double kInvStep = 0x1.71547652b82fep+6;        // 64 / ln 2
constexpr double kStepHi = 0x1.62e42fefa0000p-7;         // ln 2 / 64: 38 bits, and the rest
constexpr double kStepLo = 0x1.cf79abc9e3b3ap-46;
constexpr double kRMax2 = (kStepHi / 2.0) * (kStepHi / 2.0);
constexpr double kC4 = 1.0 / 24.0 + 1.5 * kRMax2 / 720.0;
constexpr double kC2 = 0.5 - 0.5625 * kRMax2 * kRMax2 / 720.0;
__device__ const double2 kPow2[64] = {   // 2^(j / 64): the nearest double, and the rest
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b53p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55},
};

// (Against 113-bit values, 4 10^6 arguments in each of [-700, 0], [-30, 0] and
// [-1, 0]: at most 0.53 ulp, 0.250 on average; the library's exp 0.86 and 0.258.)
__device__ __forceinline__ double exp_weight(double x, const double2 *pow2)
{
    if (!(x > -700.0)) return exp(x);
    constexpr double kRound = 0x1.8p52;
    const double t = fma(x, kInvStep, kRound);
    const int n = __double2loint(t);
    const double f = t - kRound;
    const double r = fma(f, -kStepLo, fma(f, -kStepHi, x));
    const double p = fma(r * r, fma(r, fma(r, fma(r, 1.0 / 120.0, kC4), 1.0 / 6.0), kC2), r);
    const double2 y = pow2[n & 63];
    const double e = y.x + fma(y.x, p, y.y);
    // (k >= -1011: the scaled exponent field stays positive.)
    return __hiloint2double(__double2hiint(e) + ((n >> 6) << 20), __double2loint(e));
}

// Merge the sums of chain set b into those of a (same max-shift convention):
// the multi-GPU merge (rosen_stats_merge).
inline void merge(double &Ma, double *sa, double &na, double Mb,
                                               const double *sb, double nb)
{
    const double M = fmax(Ma, Mb);
    if (M == -INFINITY) {
        na += nb;
        return;
    }
    const double fa = (Ma == -INFINITY) ? 0.0 : exp(Ma - M);
    const double fb = (Mb == -INFINITY) ? 0.0 : exp(Mb - M);
#pragma unroll
    for (int q = 0; q < 3; ++q) sa[q] = sa[q] * fa + sb[q] * fb;
#pragma unroll
    for (int q = 3; q < 8; ++q) sa[q] = sa[q] * (fa * fa) + sb[q] * (fb * fb);
    Ma = M;
    na += nb;
}

// The statistics of an ensemble from its merged sums (on the host; finish_warp
// is the device's form): Eq. 9's log Z (mean
// weight over the n growths), Eq. 2's W-weighted means of R_ee^2 and R_g^2,
// their ratio standard errors sqrt(sum w^2 (A - mean)^2) / sum w, and the
// effective sample size (sum w)^2 / sum w^2.
inline rosen_stats finish(double M, const double *S, double alive,
                                                       double n, int N, int k)
{
    rosen_stats r;
    r.n = n;
    r.n_alive = alive;
    r.log_max = M;
    r.S0 = S[0];
    r.S1 = S[1];
    r.S2 = S[2];
    r.Q0 = S[3];
    r.Q1_r2 = S[4];
    r.Q2_r2 = S[5];
    r.Q1_rg2 = S[6];
    r.Q2_rg2 = S[7];
    if (alive == 0.0) {
        r.logZ = -INFINITY;
        r.logZ_norm = -INFINITY;
        r.mean_r2 = r.se_r2 = r.mean_rg2 = r.se_rg2 = NAN;
        r.ess = 0.0;
    } else {
        r.logZ = r.log_max + log(r.S0 / r.n);
        r.logZ_norm = k > 0 ? r.logZ - (double)(N - 1) * log((double)k) : r.logZ;
        const double m1 = r.S1 / r.S0, m2 = r.S2 / r.S0;
        const double v1 = r.Q2_r2 - 2.0 * m1 * r.Q1_r2 + m1 * m1 * r.Q0;
        const double v2 = r.Q2_rg2 - 2.0 * m2 * r.Q1_rg2 + m2 * m2 * r.Q0;
        r.mean_r2 = m1;
        r.se_r2 = sqrt(v1 > 0.0 ? v1 : 0.0) / r.S0;
        r.mean_rg2 = m2;
        r.se_rg2 = sqrt(v2 > 0.0 ? v2 : 0.0) / r.S0;
        r.ess = r.S0 * r.S0 / r.Q0;
    }
    return r;
}

// Sums of the block's kSums values per thread, in a fixed order: thread q of
// sum q / kSegs adds a segment of the threads' values one after another, and
// the segments are added in pairs.  The result is in v[0..kSums) of shared
// memory when the call returns.
constexpr int kSegs = 8;
struct BlockSums {
    double part[kSums][kThreads + kSegs];   // (a word of padding per segment)
    double v[kSums];
};

__device__ __forceinline__ void block_sums(BlockSums &b, const double (&s)[kSums])
{
    constexpr int kSeg = kThreads / kSegs;
    const int t = threadIdx.x;
#pragma unroll
    for (int q = 0; q < kSums; ++q) b.part[q][t + t / kSeg] = s[q];
    __syncthreads();
    if (t < kSums * kSegs) {
        const double *x = &b.part[t / kSegs][(t % kSegs) * (kSeg + 1)];
        double y = x[0];
#pragma unroll
        for (int q = 1; q < kSeg; ++q) y += x[q];
        b.part[t / kSegs][(t % kSegs) * (kSeg + 1)] = y;
    }
    __syncthreads();
    if (t < kSums) {
        const double *x = b.part[t];
        double y[kSegs];
#pragma unroll
        for (int q = 0; q < kSegs; ++q) y[q] = x[q * (kSeg + 1)];
#pragma unroll
        for (int o = kSegs / 2; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < o; ++q) y[q] += y[q + o];
        b.v[t] = y[0];
    }
    __syncthreads();
}

// Maximum over the block, in every thread.
__device__ __forceinline__ double block_max(double m, double *warp_max)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    m = warp_max[0];
#pragma unroll
    for (int w = 1; w < kThreads / 32; ++w) m = fmax(m, warp_max[w]);
    return m;
}

// Reduce tile `tile` of the ensemble a into *out (one cluster; block r of it
// takes the tile's r-th quarter).
__device__ __forceinline__ void reduce_tile(const ReduceArgs &a, int64_t tile, Partial *out)
{
    __shared__ BlockSums b;
    __shared__ double warp_max[kThreads / 32], block_m;
    __shared__ double2 pow2[64];
    if (threadIdx.x < 64) pow2[threadIdx.x] = kPow2[threadIdx.x];
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int64_t c0 = tile * kTile + (int64_t)rank * (kTile / kTileCtas);
    double lw[kPerThread], A1[kPerThread], A2[kPerThread];
    double m = -INFINITY;
    uint32_t growths = 0u;   // Eq. 9's sample size: chains, or attempts in restart mode
#pragma unroll
    for (int q = 0; q < kPerThread; ++q) {
        const int64_t c = c0 + threadIdx.x + (int64_t)q * kThreads;
        if (c < a.C) {
            load_chain(a, c, lw[q], A1[q], A2[q]);
            growths += a.attempts ? a.attempts[c] : 1u;
        } else {
            lw[q] = -INFINITY;
            A1[q] = A2[q] = 0.0;
        }
        m = fmax(m, lw[q]);
    }
    m = block_max(m, warp_max);
    if (threadIdx.x == 0) block_m = m;
    cluster.sync();
    double M = *cluster.map_shared_rank(&block_m, 0);
#pragma unroll
    for (int r = 1; r < kTileCtas; ++r) M = fmax(M, *cluster.map_shared_rank(&block_m, r));
    if (c0 >= a.C) {              // a short tile: no chain in this quarter
        if (threadIdx.x < kSums) b.v[threadIdx.x] = 0.0;
    } else {
        double s[kSums];
#pragma unroll
        for (int q = 0; q < kSums; ++q) s[q] = 0.0;
        uint32_t alive = 0u;
        if (M > -INFINITY) {
#pragma unroll
            for (int q = 0; q < kPerThread; ++q) {
                if (lw[q] == -INFINITY) continue;
                const double w = exp_weight(lw[q] - M, pow2), w2 = w * w;
                const double u = w2 * A1[q], v = w2 * A2[q];
                s[0] += w;
                s[1] += w * A1[q];
                s[2] += w * A2[q];
                s[3] += w2;
                s[4] += u;
                s[5] += u * A1[q];
                s[6] += v;
                s[7] += v * A2[q];
                ++alive;
            }
        }
        s[8] = (double)alive;
        s[9] = (double)growths;
        block_sums(b, s);
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x < kSums) {
        double t = b.v[threadIdx.x];
#pragma unroll
        for (int r = 1; r < kTileCtas; ++r) t += *cluster.map_shared_rank(&b.v[threadIdx.x], r);
        double *field = threadIdx.x < 8 ? &out->s[threadIdx.x]
                                        : (threadIdx.x == 8 ? &out->alive : &out->n);
        *field = t;
        if (threadIdx.x == 0) out->M = M;
    }
    cluster.sync();      // (no block leaves while its sums are read)
}

__global__ void __cluster_dims__(kTileCtas) __launch_bounds__(kThreads)
    reduce_tiles_kernel(const ReduceArgs a, Partial *part)
{
    const int64_t t = blockIdx.x / kTileCtas;
    reduce_tile(a, t, &part[t]);
}

// finish() by one warp: the divisions, logarithms and square roots of
// different statistics on different lanes, so that a chain of four of them is
// waited for and not of ten.  S: S0 .. Q2b, live chains, growths.
__device__ __forceinline__ void finish_warp(double M, const double *S, int N, int k, rosen_stats *out)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const double alive = S[8], n = S[9];
    if (alive == 0.0) {
        if (lane == 0) {
            rosen_stats r;
            r.n = n;
            r.n_alive = alive;
            r.log_max = M;
            r.S0 = r.S1 = r.S2 = r.Q0 = r.Q1_r2 = r.Q2_r2 = r.Q1_rg2 = r.Q2_rg2 = 0.0;
            r.logZ = r.logZ_norm = -INFINITY;
            r.mean_r2 = r.se_r2 = r.mean_rg2 = r.se_rg2 = NAN;
            r.ess = 0.0;
            *out = r;
        }
        return;
    }
    // Lanes 0, 1: mean and standard error of R_ee^2, R_g^2; 2: log Z; 3: ESS.
    const int a = lane & 1;
    const double num = lane == 3 ? S[0] * S[0] : (lane == 2 ? S[0] : S[1 + a]);
    const double den = lane == 3 ? S[3] : (lane == 2 ? n : S[0]);
    const double q = num / den;
    const double v = S[5 + 2 * a] - 2.0 * q * S[4 + 2 * a] + q * q * S[3];
    const double se = sqrt(v > 0.0 ? v : 0.0) / S[0];
    const double lg = log(lane == 3 ? (double)max(k, 1) : q);
    const double logk = __shfl_sync(kAll, lg, 3);
    if (lane < 2) {
        (lane ? out->mean_rg2 : out->mean_r2) = q;
        (lane ? out->se_rg2 : out->se_r2) = se;
    } else if (lane == 2) {
        const double z = M + lg;
        out->logZ = z;
        out->logZ_norm = k > 0 ? z - (double)(N - 1) * logk : z;
    } else if (lane == 3) {
        out->ess = q;
        out->n = n;
        out->n_alive = alive;
        out->log_max = M;
    } else if (lane < 12) {
        (&out->S0)[lane - 4] = S[lane - 4];      // S0 .. Q2_rg2 follow one another
    }
}

// Merge the ntiles partials of one ensemble (one cluster of kCtas blocks): their
// maximum M, then the sum of every partial's sums scaled by exp(M_t - M) (squared
// for the sums of w^2).  Partial t belongs to block t / kThreads % kFinalCtas, so
// that up to kThreads partials one block alone gives the same sums (the others'
// would be zeros).
template <int kCtas>
__device__ __forceinline__ void reduce_final(const Partial *part, int64_t ntiles,
                                             const ReduceArgs &a, rosen_stats *out)
{
    __shared__ BlockSums b;
    __shared__ double warp_max[kThreads / 32], block_m;
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int64_t t0 = (int64_t)rank * kThreads + threadIdx.x;
    constexpr int64_t kStep = (int64_t)kFinalCtas * kThreads;
    double M = -INFINITY;
    for (int64_t t = t0; t < ntiles; t += kStep) M = fmax(M, part[t].M);
    M = block_max(M, warp_max);
    if (threadIdx.x == 0) block_m = M;
    cluster.sync();
#pragma unroll
    for (int r = 0; r < kCtas; ++r) M = fmax(M, *cluster.map_shared_rank(&block_m, r));
    double s[kSums];
#pragma unroll
    for (int q = 0; q < kSums; ++q) s[q] = 0.0;
    for (int64_t t = t0; t < ntiles; t += kStep) {
        const Partial &p = part[t];
        if (p.M > -INFINITY) {
            const double f = exp(p.M - M), f2 = f * f;
#pragma unroll
            for (int q = 0; q < 3; ++q) s[q] += p.s[q] * f;
#pragma unroll
            for (int q = 3; q < 8; ++q) s[q] += p.s[q] * f2;
        }
        s[8] += p.alive;
        s[9] += p.n;
    }
    block_sums(b, s);
    cluster.sync();
    if (rank == 0) {
        if (threadIdx.x < kSums) {
            double t = b.v[threadIdx.x];
            for (int r = 1; r < kCtas; ++r) t += *cluster.map_shared_rank(&b.v[threadIdx.x], r);
            b.part[0][threadIdx.x] = t;
        }
        __syncthreads();
        // The growth count is a sum of integer-valued partials: exact in FP64.
        if (threadIdx.x < 32) finish_warp(M, b.part[0], a.N, a.k, out);
    }
    cluster.sync();      // (no block leaves while its sums are read)
}

template <int kCtas>
__global__ void __cluster_dims__(kCtas) __launch_bounds__(kThreads)
    reduce_final_kernel(const Partial *part, int64_t ntiles, const ReduceArgs a, rosen_stats *out)
{
    reduce_final<kCtas>(part, ntiles, a, out);
}

// Batched: cluster b reduces global tile b; tile_off[e] .. tile_off[e+1]-1 are
// the tiles of ensemble e.
__global__ void __cluster_dims__(kTileCtas) __launch_bounds__(kThreads)
    reduce_tiles_batch_kernel(const ReduceArgs *args, const int64_t *tile_off, int n_ens,
                              Partial *part)
{
    const int64_t b = blockIdx.x / kTileCtas;
    int lo = 0, hi = n_ens;            // largest e with tile_off[e] <= b
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (tile_off[mid] <= b) lo = mid;
        else hi = mid;
    }
    reduce_tile(args[lo], b - tile_off[lo], &part[b]);
}

template <int kCtas>
__global__ void __cluster_dims__(kCtas) __launch_bounds__(kThreads)
    reduce_final_batch_kernel(const Partial *part, const int64_t *tile_off, const ReduceArgs *args,
                              rosen_stats *out)
{
    const int e = blockIdx.x / kCtas;
    reduce_final<kCtas>(part + tile_off[e], tile_off[e + 1] - tile_off[e], args[e], out + e);
}

}  // namespace

// Shared with the other translation units that reduce on the device.
int64_t reduce_tiles(int64_t C) { return (C + kTile - 1) / kTile; }

size_t reduce_args_size() { return sizeof(ReduceArgs); }
size_t reduce_partial_bytes() { return sizeof(Partial); }

void reduce_make_args(const rosen_reduce_in *in, void *out)
{
    ReduceArgs a;
    memset(&a, 0, sizeof a);
    a.kind = in->kind;
    a.N = in->N;
    a.k = in->k;
    a.use_counts = in->use_counts;
    a.C = in->C;
    a.logw = in->logw;
    a.counts = reinterpret_cast<const uint4 *>(in->counts);
    a.r2_i = in->r2_i;
    a.n2rg2 = in->n2rg2;
    a.r2_f = in->r2_f;
    a.rg2_f = in->rg2_f;
    a.attempts = in->attempts;
    for (int q = 0; q < 8; ++q) a.logm[q] = q >= 1 ? log((double)q) : 0.0;
    a.inv_n2 = 1.0 / ((double)in->N * (double)in->N);
    memcpy(out, &a, sizeof a);
}

void reduce_batch_launch(const void *dev_args, const int64_t *dev_tile_off, int n_ens,
                         int64_t total_tiles, int64_t max_tiles, void *part, rosen_stats *out,
                         cudaStream_t s)
{
    const ReduceArgs *args = reinterpret_cast<const ReduceArgs *>(dev_args);
    Partial *p = reinterpret_cast<Partial *>(part);
    reduce_tiles_batch_kernel<<<(unsigned)(total_tiles * kTileCtas), kThreads, 0, s>>>(
        args, dev_tile_off, n_ens, p);
    if (max_tiles <= kThreads)
        reduce_final_batch_kernel<1><<<n_ens, kThreads, 0, s>>>(p, dev_tile_off, args, out);
    else
        reduce_final_batch_kernel<kFinalCtas>
            <<<n_ens * kFinalCtas, kThreads, 0, s>>>(p, dev_tile_off, args, out);
}

int reduce_launch(const rosen_reduce_in *in, rosen_stats *out, void *part_ws, cudaStream_t s)
{
    ReduceArgs a;
    memset(&a, 0, sizeof a);
    a.kind = in->kind;
    a.N = in->N;
    a.k = in->k;
    a.use_counts = in->use_counts;
    a.C = in->C;
    a.logw = in->logw;
    a.counts = reinterpret_cast<const uint4 *>(in->counts);
    a.r2_i = in->r2_i;
    a.n2rg2 = in->n2rg2;
    a.r2_f = in->r2_f;
    a.rg2_f = in->rg2_f;
    a.attempts = in->attempts;
    for (int q = 0; q < 8; ++q) a.logm[q] = q >= 1 ? log((double)q) : 0.0;
    a.inv_n2 = 1.0 / ((double)in->N * (double)in->N);
    const int64_t tiles = reduce_tiles(in->C);
    Partial *part = reinterpret_cast<Partial *>(part_ws);
    reduce_tiles_kernel<<<(unsigned)(tiles * kTileCtas), kThreads, 0, s>>>(a, part);
    if (tiles <= kThreads)
        reduce_final_kernel<1><<<1, kThreads, 0, s>>>(part, tiles, a, out);
    else
        reduce_final_kernel<kFinalCtas><<<kFinalCtas, kThreads, 0, s>>>(part, tiles, a, out);
    return check_launch("rosen_reduce");
}

int reduce_validate(const rosen_reduce_in *in, const rosen_stats *out)
{
    if (!in || !out) return set_error(ROSEN_EINVAL, "rosen_reduce: NULL input or output");
    if (in->C < 1) return set_error(ROSEN_EINVAL, "rosen_reduce: C must be >= 1");
    if (in->N < 1) return set_error(ROSEN_EINVAL, "rosen_reduce: N must be >= 1");
    if (in->k < 0) return set_error(ROSEN_EINVAL, "rosen_reduce: k must be >= 0");
    if (in->kind == ROSEN_REDUCE_LATTICE) {
        if (in->use_counts ? !in->counts : !in->logw)
            return set_error(ROSEN_EINVAL, "rosen_reduce: missing counts/logw");
        if (in->use_counts && (reinterpret_cast<uintptr_t>(in->counts) & 15u))
            return set_error(ROSEN_EINVAL, "rosen_reduce: counts must be 16-byte aligned");
        if (!in->r2_i || !in->n2rg2)
            return set_error(ROSEN_EINVAL, "rosen_reduce: lattice needs r2_i and n2rg2");
    } else if (in->kind == ROSEN_REDUCE_OFFLATTICE) {
        if (!in->logw || !in->r2_f || !in->rg2_f)
            return set_error(ROSEN_EINVAL, "rosen_reduce: real space needs logw, r2_f, rg2_f");
    } else {
        return set_error(ROSEN_EINVAL, "rosen_reduce: unknown kind %d", in->kind);
    }
    return ROSEN_OK;
}

size_t reduce_workspace_bytes(int64_t C)
{
    return (size_t)reduce_tiles(C < 1 ? 1 : C) * sizeof(Partial);
}

}  // namespace rosen

// ---------------------------------------------------------------------------
// Allocation-free variant.  Its scratch (the per-tile partials) lives in a
// fixed array in this file; every GPU that loads the library holds it until
// the process exits.  In host code the array's name is only a stand-in, so
// the device address is looked up with cudaGetSymbolAddress, with the
// device current, on every call made outside stream capture.
// ---------------------------------------------------------------------------
namespace rosen {
namespace {

constexpr int64_t kNoallocTiles = ((int64_t)ROSEN_REDUCE_NOALLOC_MAX_CHAINS + kTile - 1) / kTile;
static __device__ __align__(256) Partial g_noalloc_partials[kNoallocTiles];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kMaxDevices] = {};

// The device address of the scratch on the current device.  A call whose
// stream is not being captured looks it up again every time (cheap), so a
// module reloaded after cudaDeviceReset is followed; a call made while its
// stream is captured uses the address the last uncaptured call on this
// device found.
int noalloc_scratch(cudaStream_t s, void **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return set_error(ROSEN_ECUDA, "rosen_reduce_noalloc: cudaGetDevice: %s",
                         cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices)
        return set_error(ROSEN_EINVAL, "rosen_reduce_noalloc: device %d out of range", dev);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(s, &cs);
    if (e != cudaSuccess)
        return set_error(ROSEN_ECUDA, "rosen_reduce_noalloc: cudaStreamIsCapturing: %s",
                         cudaGetErrorString(e));
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (cs == cudaStreamCaptureStatusNone) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess || !p)
            return set_error(ROSEN_ECUDA, "rosen_reduce_noalloc: cudaGetSymbolAddress: %s",
                             cudaGetErrorString(e));
        g_noalloc_addr[dev] = p;
    } else if (!g_noalloc_addr[dev]) {
        return set_error(ROSEN_EINVAL, "rosen_reduce_noalloc: the first call on device %d must "
                                       "come before any stream capture", dev);
    }
    *out = g_noalloc_addr[dev];
    return ROSEN_OK;
}

}  // namespace
}  // namespace rosen

extern "C" int rosen_reduce_noalloc(const rosen_reduce_in *in, rosen_stats *out, void *stream)
{
    int st = rosen::reduce_validate(in, out);
    if (st != ROSEN_OK) return st;
    if (in->C > (int64_t)ROSEN_REDUCE_NOALLOC_MAX_CHAINS)
        return rosen::set_error(ROSEN_ENOMEM,
                                "rosen_reduce_noalloc: C = %lld exceeds the built-in scratch "
                                "limit of %d chains; use rosen_reduce with a workspace",
                                (long long)in->C, (int)ROSEN_REDUCE_NOALLOC_MAX_CHAINS);
    void *ws = nullptr;
    st = rosen::noalloc_scratch((cudaStream_t)stream, &ws);
    if (st != ROSEN_OK) return st;
    // Every partial the final merge reads is rewritten by this call's tile
    // kernel, so nothing in the shared scratch has to be cleared first.
    return rosen::reduce_launch(in, out, ws, (cudaStream_t)stream);
}

using namespace rosen;

extern "C" size_t rosen_reduce_workspace_size(int64_t C) { return reduce_workspace_bytes(C); }

extern "C" int rosen_reduce(const rosen_reduce_in *in, rosen_stats *out, void *workspace,
                            size_t workspace_bytes, void *stream)
{
    int st = reduce_validate(in, out);
    if (st != ROSEN_OK) return st;
    if (!workspace || workspace_bytes < reduce_workspace_bytes(in->C))
        return set_error(ROSEN_ENOMEM, "rosen_reduce: workspace of %zu bytes < %zu needed",
                         workspace_bytes, reduce_workspace_bytes(in->C));
    if (reinterpret_cast<uintptr_t>(workspace) & 15u)
        return set_error(ROSEN_EINVAL, "rosen_reduce: workspace must be 16-byte aligned");
    return reduce_launch(in, out, workspace, (cudaStream_t)stream);
}

extern "C" int rosen_stats_merge(const rosen_stats *parts, int32_t n, int32_t N, int32_t k,
                                 rosen_stats *out)
{
    if (!parts || !out || n < 1)
        return set_error(ROSEN_EINVAL, "rosen_stats_merge: NULL argument or n < 1");
    if (N < 1 || k < 0) return set_error(ROSEN_EINVAL, "rosen_stats_merge: N >= 1, k >= 0");
    double M = -INFINITY, S[8] = {0, 0, 0, 0, 0, 0, 0, 0}, alive = 0.0, growths = 0.0;
    for (int32_t p = 0; p < n; ++p) {
        const rosen_stats &b = parts[p];
        const double Sb[8] = {b.S0, b.S1, b.S2, b.Q0, b.Q1_r2, b.Q2_r2, b.Q1_rg2, b.Q2_rg2};
        merge(M, S, alive, b.n_alive > 0.0 ? b.log_max : -INFINITY, Sb, b.n_alive);
        growths += b.n;
    }
    *out = finish(M, S, alive, growths, N, k);
    return ROSEN_OK;
}
