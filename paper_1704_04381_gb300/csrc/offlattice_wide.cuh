// offlattice_wide.cuh -- hard-sphere growth with few lanes per chain (Guo &
// Baulin, Section 3.3.3, Algorithm 2), for the chains shared memory holds.
//
// A step of one chain is k directions and their tests against a handful of
// near beads, plus scalar work (selection, commit, loop control) that every
// lane of the chain's group repeats.  With 16 lanes per chain that scalar work
// was over half of the 278 warp instructions of a chain step (N = 64, k = 32).
// So here a warp carries 32/G = 8, 4 or 2 chains (G = 4, 8, 16 or 32 lanes),
// each lane T = 2..8 trials: the scalar work is shared by more chains and T
// independent trials per lane hide latency.  All groups of a warp step
// together, every loop running to the warp's largest trip count with full-warp
// votes and shuffles.
//
// Per step:
//  1. scan: a lane tests four beads per 16-byte load on the hi words alone
//     (beads not placed yet read as far away) and keeps a bit per candidate;
//  2. trials: T Philox words and directions by the special-function unit;
//  3. rounds: every lane puts the exact float-float displacement of its next
//     candidate up, and every trial is tested against the group's G; FP32
//     arithmetic works on pairs of trials (two results per instruction);
//  4. selection; a step the fast directions cannot decide within their error
//     band is decided again by the whole warp (wide_redecide);
//  5. commit of the chosen trial's direction, taken again as off_chain does
//     from the words its lane kept.
// Displacements, bands, draws, sums and the steps re-decided in FP64 are those
// of off_chain with Gref lanes per chain, operation for operation: a chain's
// outputs are the same bit for bit.  (The order of a hard-sphere list does
// not matter: a minimum.)
//
// It is bound by issue (65%) with 16 warps per SM, the most 128 registers and
// 24 bytes a bead leave: 118 warp instructions per chain step.  GB300, before
// (16 or 32 lanes, FP64 re-decision in a second pass or in place) and now, k =
// 32: N = 64, 10^7 chains 171 -> 91 ms; N = 128, 2 10^5: 11.3 -> 5.8; N = 256,
// 6 10^4: 10.4 -> 5.5; N = 512, 2 10^4: 17.7 -> 6.3; N = 1024, 5 10^3: 18.5 ->
// 5.4.  N = 64: k = 16, 5 10^5 chains 7.9 -> 3.7; k = 64, 3 10^5: 8.3 -> 5.0;
// k = 128, 2 10^5: 9.6 -> 6.2; k = 32, 100 chains 0.19 -> 0.08.  (One or two trials
// of N > 128, too few for any lanes to share, take 4 to 9 us longer: k = 2, N = 200,
// 2000 chains 77 -> 84 us.)  Tried and not kept: all trials through dir32x2 (13.5
// ms), per-chain lists ranked by votes (12.5), the next step's trials drawn beside
// the selection (11.4: more registers moved).
#pragma once

#include "offlattice_chain.cuh"

namespace rosen {
namespace {

constexpr float kFar = 1e15f;           // coordinate of a bead not placed yet
constexpr int kWideSelBytes = 256 * 8;  // selection table: n-th set bit of a byte

// Twice the trial directions of words (a, b) and (c, d) by the special-function
// unit, as pairs: the angle in (-pi, pi] from the signed word, sin, cos and
// sqrt approximate.  The chosen trial's direction is taken again with dir32x2.
// As vectors (Euclidean norm) the two differ by less than kFastDir: 7.6e-7 over
// all 2^24 angles at s = 1, 1.2e-7 over all 2^24 polar words at angle 0, and at
// most 1.7e-7 by the rounding of both sides' products with s; z is the same.
// (Largest difference of 2^31 random directions: 9.1e-7.)
constexpr double kFastDir = 1.06e-6;

// What a squared distance d^2 = c + 2u.g at the decision (d^2 <= sigma^2 + 0.01,
// |g| < rf) differs by between fast_dirs_x2 and dir32x2: kFastDir |g|, and on
// either side the rounding of c + 2 uz gz, of that + 2 uy gy and of d^2, which
// are at most d^2 + 2^(3/2) |g|, d^2 + 2 |g| and d^2.  Together below kFastBand rf,
// as rf > 1 + sigma and sigma <= 4 (sigma^2 / rf < 3.2).  A step whose fast
// distances stay out of pair_band plus this is one that off_chain decides in
// FP32, and alike.  (N = 64, k = 32: a band three times as wide costs 0.1%.)
constexpr float kFastBand = 2.8e-6f;
static_assert(kFastBand > kFastDir + 2.0 * 0x1p-24 * (3.0 * (3.2 + 0.01) + 4.83), "fast band");

__device__ __forceinline__ void fast_dirs_x2(const uint4 &w, float2 &x, float2 &y, float2 &z)
{
    const float2 fa = make_float2((float)(w.x >> 8), (float)(w.z >> 8));
    z = __ffma2_rn(make_float2(-0x1p-22f, -0x1p-22f), fa, make_float2(2.f, 2.f));
    const float2 nz = __ffma2_rn(make_float2(0x1p-22f, 0x1p-22f), fa, make_float2(-2.f, -2.f));
    const float2 q = __ffma2_rn(nz, z, make_float2(4.f, 4.f));
    float2 s;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(s.x) : "f"(q.x));
    asm("sqrt.approx.f32 %0, %1;" : "=f"(s.y) : "f"(q.y));
    constexpr float kTurn24 = (float)(2.0 * kPi * 0x1p-24);
    const float2 phi = __fmul2_rn(make_float2((float)((int32_t)w.y >> 8), (float)((int32_t)w.w >> 8)),
                                  make_float2(kTurn24, kTurn24));
    x = __fmul2_rn(s, make_float2(__cosf(phi.x), __cosf(phi.y)));
    y = __fmul2_rn(s, make_float2(__sinf(phi.x), __sinf(phi.y)));
}

__device__ __forceinline__ float min3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

struct WideShape {
    int np;        // beads per coordinate array: N rounded up to 4 G
    int stride;    // words per chain, = 16 (mod 32): two chains' 16-byte loads share no bank
    float pre2;    // coarse test on the hi words (covers the lo words and rounding)
    int gref;      // lanes per chain whose summation order is followed: 8, 16 or 32
};

__host__ __device__ inline int wide_np(int N, int G) { return (N + 4 * G - 1) / (4 * G) * (4 * G); }
__host__ __device__ inline int wide_stride(int N, int G)
{
    int s = 6 * wide_np(N, G) + 8 * G + (N + 3) / 4;
    s = (s + 15) / 16 * 16;
    return (s & 31) == 16 ? s : s + 16;
}

// Word of bead j in a coordinate array: blocks of 4 G beads, bead j of a block
// to lane j % G, so that a lane's 16-byte load brings it four beads and the
// recent beads (the near ones) spread over the lanes.
template <int G>
__device__ __forceinline__ int wide_at(int j)
{
    const unsigned u = (unsigned)j;
    return (int)(u / (4 * G) * (4 * G) + (u % G) * 4 + u / G % 4);
}

// A chain's R_g^2 with the partial sums of Gref lanes: leaf l adds beads l,
// l + Gref, ...; leaves are added in pairs l, l ^ Gref/2, then Gref/4, ...
template <int G, int Gref>
__device__ __forceinline__ float wide_rg2(const Group<G> &g, const float *P, int np, int N)
{
    constexpr int R = Gref > G ? Gref / G : 1;      // leaves per lane
    float acc[R], m[3];
    const float inv = 1.f / (float)N;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float *h = P + q * np, *l = P + (3 + q) * np;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            acc[r] = 0.f;
            for (int s = g.gl + r * G; g.gl < Gref && s < N; s += Gref)
                acc[r] += h[wide_at<G>(s)] + l[wide_at<G>(s)];
        }
#pragma unroll
        for (int o = R / 2; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < o; ++r) acc[r] += acc[r + o];
        m[q] = g.sum(acc[0]) * inv;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        acc[r] = 0.f;
        for (int s = g.gl + r * G; g.gl < Gref && s < N; s += Gref) {
            const int p = wide_at<G>(s);
            const float dx = (P[p] - m[0]) + P[3 * np + p], dy = (P[np + p] - m[1]) + P[4 * np + p],
                        dz = (P[2 * np + p] - m[2]) + P[5 * np + p];
            acc[r] += fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        }
    }
#pragma unroll
    for (int o = R / 2; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < o; ++r) acc[r] += acc[r + o];
    return g.sum(acc[0]) * inv;
}

// Outputs of a chain that ended (dead: at step i), by its group.
template <int G>
__device__ __noinline__ void wide_finish(const OffArgs &a, const Group<G> &g, float *P,
                                         const uint8_t *tr, int np, int gref, int64_t c,
                                         uint32_t att, bool dead, int i, float lw,
                                         unsigned rechecks, unsigned listed, float3 eh, float3 el)
{
    const int N = a.N;
    const int64_t C = a.C;
    const int grown = dead ? i : N;       // beads 0 .. grown-1 exist
    if (g.gl == 0) {                      // the last is not stored yet
        const int p = wide_at<G>(grown - 1);
        P[p] = eh.x;
        P[np + p] = eh.y;
        P[2 * np + p] = eh.z;
        P[3 * np + p] = el.x;
        P[4 * np + p] = el.y;
        P[5 * np + p] = el.z;
    }
    __syncwarp(g.mask);
    if (a.attempts && g.gl == 0) a.attempts[c] = (uint16_t)(att + 1);
    if (a.counters) {
        if (g.gl == 0) {
            if (rechecks) atomicAdd(&a.counters[0], (unsigned long long)rechecks);
            atomicAdd(&a.counters[1], 1ull);
        }
        if (listed) atomicAdd(&a.counters[2], (unsigned long long)listed);
    }
    float r2 = 0.f, gg = 0.f;
    if (!dead) {
        const float xe = eh.x + el.x, ye = eh.y + el.y, ze = eh.z + el.z;
        r2 = fmaf(xe, xe, fmaf(ye, ye, ze * ze));
        gg = gref == 8 ? wide_rg2<G, 8>(g, P, np, N)
                       : (gref == 16 ? wide_rg2<G, 16>(g, P, np, N) : wide_rg2<G, 32>(g, P, np, N));
    }
    if (g.gl == 0) {
        if (a.logw) a.logw[c] = dead ? -INFINITY : lw;
        if (a.r2) a.r2[c] = r2;
        if (a.rg2) a.rg2[c] = gg;
        if (a.alive) a.alive[c] = dead ? 0 : 1;
    }
    if (a.trace)
        for (int s = 1 + g.gl; s < N; s += G)
            a.trace[(int64_t)(s - 1) * C + c] = s < grown ? tr[s] : (s == grown ? 0xFEu : 0xFFu);
    if (a.coords)
        for (int s = g.gl; s < N; s += G) {
            const int p = wide_at<G>(s);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                a.coords[((int64_t)s * 3 + q) * C + c] =
                    s < grown ? P[q * np + p] + P[(3 + q) * np + p] : 0.f;
        }
    __syncwarp(g.mask);
}

// A chain's step i decided again by the whole warp, because the fast directions
// could not: first with dir32x2's directions and off_chain's band; if that
// cannot decide either, in FP64 with the listing, the replay (in the order of
// Gref lanes) and the arithmetic of redecide(): the positions since bead b
// are replayed in FP64 and stored back, and every trial is tested against the
// listed beads.  Returns the end, the number of free trials, the one taken
// and whether FP64 was needed.
struct WideDecision {
    float hx, hy, hz, lx, ly, lz;
    int m, sel;
    bool exact;
};

// The number of free trials (bits of fr[], 32 to a word) and the idx-th of
// them, idx = floor(selw m / 2^32).
__device__ __forceinline__ void wide_select(const uint32_t (&fr)[4], uint32_t selw, WideDecision &d)
{
    d.m = __popc(fr[0]) + __popc(fr[1]) + __popc(fr[2]) + __popc(fr[3]);
    int idx = (int)__umulhi(selw, (uint32_t)d.m);
    d.sel = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int n = __popc(fr[w]);
        if (idx >= 0 && idx < n) {
            uint32_t v = fr[w];
            for (int q = 0; q < idx; ++q) v &= v - 1u;
            d.sel = 32 * w + __ffs(v) - 1;
        }
        idx -= n;
    }
}

template <int G>
__device__ __noinline__ WideDecision wide_redecide(const OffArgs &a, float *P, int np, int gref,
                                                   uint32_t chain, uint32_t aw, int b, int i,
                                                   uint32_t selw, float ehx, float ehy, float ehz,
                                                   float elx, float ely, float elz)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    uint8_t *const tr = reinterpret_cast<uint8_t *>(P + 6 * np + 8 * G);
    // The listed beads (before the replay moves them): bit r of the lane's
    // mask is bead 32 r + lane.
    uint32_t list = 0u;
    int jmin = a.N;
    for (int j = lane; j <= i - 2; j += 32) {
        const int p = wide_at<G>(j);
        const float gx = (ehx - P[p]) + (elx - P[3 * np + p]);
        const float gy = (ehy - P[np + p]) + (ely - P[4 * np + p]);
        const float gz = (ehz - P[2 * np + p]) + (elz - P[5 * np + p]);
        if (fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < a.rf2) {
            list |= 1u << (j >> 5);
            jmin = min(jmin, j);
        }
    }
    jmin = __reduce_min_sync(kAll, jmin);
    WideDecision d;
    uint32_t fr[4];
    {
        const float band = pair_band(a.rf, 1.f + a.rf2, i - 1 - max(jmin, b), a.dband, 4e-7f);
        bool flag = false;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int t = 32 * w + lane;
            fr[w] = 0u;
            if (32 * w >= a.k) continue;
            const uint4 xx =
                philox(make_uint4(chain, a.ens, (uint32_t)i | aw, 1u + (uint32_t)(t >> 1)), a.key);
            uint32_t wa, wb;
            trial_words(xx, t, wa, wb);
            const float3 u = dir32x2(wa, wb);
            float mind = INFINITY;
            for (int r = 0; 32 * r <= i - 2; ++r)
                for (uint32_t v = __ballot_sync(kAll, (list >> r) & 1u); v; v &= v - 1u) {
                    const int p = wide_at<G>(32 * r + __ffs(v) - 1);
                    const float gx = (ehx - P[p]) + (elx - P[3 * np + p]);
                    const float gy = (ehy - P[np + p]) + (ely - P[4 * np + p]);
                    const float gz = (ehz - P[2 * np + p]) + (elz - P[5 * np + p]);
                    const float c = 1.f + fmaf(gx, gx, fmaf(gy, gy, gz * gz));
                    mind = fminf(mind, fmaf(u.x, gx, fmaf(u.y, gy, fmaf(u.z, gz, c))));
                }
            flag |= t < a.k && fabsf(mind - a.sig2) < band;
            fr[w] = __ballot_sync(kAll, t < a.k && mind >= a.sig2);
        }
        d.exact = __any_sync(kAll, flag && jmin < a.N);
    }
    if (!d.exact) {
        d.hx = ehx;
        d.hy = ehy;
        d.hz = ehz;
        d.lx = elx;
        d.ly = ely;
        d.lz = elz;
        wide_select(fr, selw, d);
        return d;
    }
    if (lane == 0) {                      // the end, bead i-1, is not stored yet
        const int p = wide_at<G>(i - 1);
        P[p] = ehx;
        P[np + p] = ehy;
        P[2 * np + p] = ehz;
        P[3 * np + p] = elx;
        P[4 * np + p] = ely;
        P[5 * np + p] = elz;
    }
    __syncwarp();
    const auto pos = [&](int j, int q) {
        const int p = wide_at<G>(j);
        return (double)P[q * np + p] + (double)P[(3 + q) * np + p];
    };
    double cx = pos(b, 0), cy = pos(b, 1), cz = pos(b, 2);
    __syncwarp();
    for (int b0 = b + 1; b0 <= i - 1; b0 += gref) {
        // (For Gref < 32 the warp's halves or quarters do the same work.)
        const int s = b0 + (lane & (gref - 1));
        double x = 0.0, y = 0.0, z = 0.0;
        if (s <= i - 1) {
            const int t = tr[s];
            const uint4 q =
                philox(make_uint4(chain, a.ens, (uint32_t)s | aw, 1u + (uint32_t)(t >> 1)), a.key);
            uint32_t wa, wb;
            trial_words(q, t, wa, wb);
            dir64(wa, wb, x, y, z);
        }
        for (int o = 1; o < gref; o <<= 1) {
            const double ux = __shfl_up_sync(kAll, x, o, gref), uy = __shfl_up_sync(kAll, y, o, gref),
                         uz = __shfl_up_sync(kAll, z, o, gref);
            if ((lane & (gref - 1)) >= o) {
                x += ux;
                y += uy;
                z += uz;
            }
        }
        x += cx;
        y += cy;
        z += cz;
        if (s <= i - 1 && lane < gref) {
            const int p = wide_at<G>(s);
            const float hx = (float)x, hy = (float)y, hz = (float)z;
            P[p] = hx;
            P[np + p] = hy;
            P[2 * np + p] = hz;
            P[3 * np + p] = (float)(x - hx);
            P[4 * np + p] = (float)(y - hy);
            P[5 * np + p] = (float)(z - hz);
        }
        cx = __shfl_sync(kAll, x, gref - 1);
        cy = __shfl_sync(kAll, y, gref - 1);
        cz = __shfl_sync(kAll, z, gref - 1);
    }
    __syncwarp();
    d.hx = (float)cx;
    d.hy = (float)cy;
    d.hz = (float)cz;
    d.lx = (float)(cx - d.hx);
    d.ly = (float)(cy - d.hy);
    d.lz = (float)(cz - d.hz);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int t = 32 * w + lane;
        bool free = t < a.k;
        fr[w] = 0u;
        if (32 * w >= a.k) continue;
        const uint4 xx =
            philox(make_uint4(chain, a.ens, (uint32_t)i | aw, 1u + (uint32_t)(t >> 1)), a.key);
        uint32_t wa, wb;
        trial_words(xx, t, wa, wb);
        double dx, dy, dz;
        dir64(wa, wb, dx, dy, dz);
        const double tx = __dadd_rn(cx, dx), ty = __dadd_rn(cy, dy), tz = __dadd_rn(cz, dz);
        for (int r = 0; 32 * r <= i - 2; ++r)
            for (uint32_t v = __ballot_sync(kAll, (list >> r) & 1u); v; v &= v - 1u) {
                const int j = 32 * r + __ffs(v) - 1;
                const double rx = __dsub_rn(tx, pos(j, 0)), ry = __dsub_rn(ty, pos(j, 1)),
                             rz = __dsub_rn(tz, pos(j, 2));
                const double d2 =
                    __dadd_rn(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)), __dmul_rn(rz, rz));
                if (d2 < a.sig2d) free = false;
            }
        fr[w] = __ballot_sync(kAll, free);
    }
    wide_select(fr, selw, d);
    return d;
}

// Chains [c_lo, c_hi).  Idle groups take chains from the counter *next once at
// least half of the warp's are idle (so the groups of a warp mostly step
// through the same i, and the scan's trip count is theirs); without a counter
// every group grows one chain, the grid's n-th.
template <int G, int T>
__global__ void __launch_bounds__(512, 1) offlattice_wide_kernel(const __grid_constant__ OffArgs a,
                                                                 const WideShape sh,
                                                              unsigned long long *next,
                                                              int64_t c_lo, int64_t c_hi)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kChains = 32 / G;       // chains of a warp
    float *logm = reinterpret_cast<float *>(smem_raw);
    uint8_t *nth = reinterpret_cast<uint8_t *>(smem_raw + kTable * sizeof(float));
    fill_log_table(logm);
    for (int q = threadIdx.x; q < 256; q += blockDim.x) {
        uint64_t row = 0ull;                 // the set bits of byte q, ascending
        int shift = 0;
        for (uint32_t v = (uint32_t)q; v; v &= v - 1u, shift += 8)
            row |= (uint64_t)(__ffs(v) - 1) << shift;
        reinterpret_cast<uint64_t *>(nth)[q] = row;
    }
    __syncthreads();

    const Group<G> g;
    const int lane = threadIdx.x & 31;
    const int np = sh.np;
    float *const P = reinterpret_cast<float *>(smem_raw + kTable * sizeof(float) + kWideSelBytes) +
                     (size_t)(threadIdx.x / G) * sh.stride;
    float4 *const near = reinterpret_cast<float4 *>(P + 6 * np);   // a near bead per lane
    uint8_t *const tr = reinterpret_cast<uint8_t *>(P + 6 * np + 8 * G);
    for (int q = g.gl; q < sh.stride / 4; q += G)           // (what is read is finite)
        reinterpret_cast<float4 *>(P)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();                         // before restart() writes the same words from other lanes
    const int N = a.N, k = a.k;
    const auto put = [&](int j, float hx, float hy, float hz, float lx, float ly, float lz) {
        const int p = wide_at<G>(j);
        P[p] = hx;
        P[np + p] = hy;
        P[2 * np + p] = hz;
        P[3 * np + p] = lx;
        P[4 * np + p] = ly;
        P[5 * np + p] = lz;
    };
    uint32_t tmask = 0u;                  // the lane's trials that exist (t < k)
#pragma unroll
    for (int s = 0; s < T; ++s) tmask |= (T * g.gl + s < k ? 1u : 0u) << s;

    bool more = true;                     // the counter may hold more chains
    int64_t c = -1;                       // the group's chain (-1: none)
    int i = 0;
    int exact_upto = 0;                   // beads 0..exact_upto are exact
    uint32_t att = 0, chain = 0;
    unsigned rechecks = 0u;               // steps re-decided in FP64
    unsigned listed = 0u;                 // this lane's share of the listed beads
    float ehx = 0.f, ehy = 0.f, ehz = 0.f, elx = 0.f, ely = 0.f, elz = 0.f, lw = 0.f;

    // Bead 0 at the origin, no other placed.
    const auto restart = [&]() {
        for (int q = g.gl; q < np / 4; q += G)
            reinterpret_cast<float4 *>(P)[q] = make_float4(kFar, kFar, kFar, kFar);
        ehx = ehy = ehz = elx = ely = elz = lw = 0.f;
        i = 1;
        exact_upto = 0;
    };

    for (;;) {
        // ---- 0. chains for idle groups, once at most half are at work ----------
        const unsigned idle = __ballot_sync(kAll, c < 0 && g.gl == 0);
        if (more && 2 * __popc(idle) >= kChains) {
            unsigned long long first = 0;
            if (lane == 0)
                first = next ? atomicAdd(next, (unsigned long long)__popc(idle))
                             : ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) / G;
            first = __shfl_sync(kAll, first, 0) + (unsigned long long)c_lo;
            more = next && first + (unsigned long long)__popc(idle) < (unsigned long long)c_hi;
            if (c < 0) {
                const unsigned long long n =
                    first + (unsigned long long)__popc(idle & ((1u << g.base) - 1u));
                if (n < (unsigned long long)c_hi) {
                    c = (int64_t)n;
                    chain = a.chain0 + (uint32_t)c;
                    att = 0;
                    listed = rechecks = 0u;
                    restart();
                }
            }
            __syncwarp();
        }
        if (!__any_sync(kAll, c >= 0)) break;
        const bool on = c >= 0;
        const uint32_t step = (uint32_t)i | (att << 16);

        // ---- 1. scan beads 0 .. i-2 on their hi words ----------------------------
        const int imax = __reduce_max_sync(kAll, on ? i : 0);
        const int blocks = (imax - 1 + 4 * G - 1) / (4 * G);
        uint32_t cand = 0u;
        {
            const float2 nx = both(-ehx), ny = both(-ehy), nz = both(-ehz);
#pragma unroll 1
            for (int b = 0; b < blocks; ++b) {
                const float4 x = reinterpret_cast<const float4 *>(P)[b * G + g.gl];
                const float4 y = reinterpret_cast<const float4 *>(P + np)[b * G + g.gl];
                const float4 z = reinterpret_cast<const float4 *>(P + 2 * np)[b * G + g.gl];
                const auto dist2 = [&](float2 px, float2 py, float2 pz) {
                    const float2 dx = __fadd2_rn(px, nx), dy = __fadd2_rn(py, ny),
                                 dz = __fadd2_rn(pz, nz);
                    return __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                };
                const float2 d = dist2(make_float2(x.x, x.y), make_float2(y.x, y.y),
                                       make_float2(z.x, z.y));
                const float2 e = dist2(make_float2(x.z, x.w), make_float2(y.z, y.w),
                                       make_float2(z.z, z.w));
                uint32_t m = d.x < sh.pre2 ? 1u : 0u;
                if (d.y < sh.pre2) m |= 2u;
                if (e.x < sh.pre2) m |= 4u;
                if (e.y < sh.pre2) m |= 8u;
                cand |= m << (4 * b);
            }
        }
        if (!on) cand = 0u;
        // One band for the step: the oldest candidate drifted longest.
        int jmin = N;
        if (cand) {
            const int b = __ffs(cand) - 1;
            jmin = (b >> 2) * (4 * G) + (b & 3) * G + g.gl;
        }
        if constexpr (G == 32) {
            jmin = __reduce_min_sync(kAll, jmin);
        } else {
#pragma unroll
            for (int o = 1; o < G; o <<= 1) jmin = min(jmin, __shfl_xor_sync(kAll, jmin, o));
        }
        const float band =
            fmaf(kFastBand, a.rf, pair_band(a.rf, 1.f + a.rf2, i - 1 - max(jmin, exact_upto), a.dband, 4e-7f));

        // ---- 2. trials -------------------------------------------------------------------
        float2 ux[T / 2], uy[T / 2], uz[T / 2];      // 2u: d^2 = c + (2u).g
        uint4 words[T / 2];
        float mind[T];
        uint32_t selw = 0u;
#pragma unroll
        for (int s = 0; s < T / 2; ++s) {
            const uint4 x = philox(make_uint4(chain, a.ens, step, 1u + (uint32_t)(T / 2 * g.gl + s)),
                                   a.key);
            if (s == 0)
                selw = __byte_perm(__byte_perm(x.x, x.y, 0x0040u), __byte_perm(x.z, x.w, 0x0040u),
                                   0x5410u);
            words[s] = x;
            fast_dirs_x2(x, ux[s], uy[s], uz[s]);
            mind[2 * s] = mind[2 * s + 1] = INFINITY;
        }
        selw = __shfl_sync(kAll, selw, 0, G);

        // ---- 3. rounds: a candidate per lane, then every trial against the group's -----
        while (__any_sync(kAll, cand != 0u)) {
            const int b = cand ? __ffs(cand) - 1 : 0;
            const int p = (b >> 2) * (4 * G) + g.gl * 4 + (b & 3);
            const float gx = (ehx - P[p]) + (elx - P[3 * np + p]);
            const float gy = (ehy - P[np + p]) + (ely - P[4 * np + p]);
            const float gz = (ehz - P[2 * np + p]) + (elz - P[5 * np + p]);
            const float g2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
            const bool in = cand && g2 < a.rf2;
            const float c1 = in ? 1.f + g2 : kNoBead;   // (out of the list: touches no trial)
            listed += in;
            cand &= cand - 1u;
            // Wide groups put their few near beads first and stop after them.
            int slot = g.gl, n = G;
            if constexpr (G > 4) {
                const unsigned v = __ballot_sync(kAll, in);
                n = __popc(v & g.mask);
                slot = in ? __popc(v & g.below) : n + __popc(~v & g.below);
                if constexpr (G < 32) n = __reduce_max_sync(kAll, n);
            }
            near[2 * slot] = make_float4(gx, gx, gy, gy);
            near[2 * slot + 1] = make_float4(gz, gz, c1, c1);
            __syncwarp();
#pragma unroll(G == 4 ? 2 : 1)
            for (int q = 0; q < n; q += 2) {
                const float4 A = near[2 * q], B = near[2 * q + 1], C = near[2 * q + 2],
                             D = near[2 * q + 3];
#pragma unroll
                for (int s = 0; s < T / 2; ++s) {
                    const float2 d = __ffma2_rn(
                        ux[s], make_float2(A.x, A.y),
                        __ffma2_rn(uy[s], make_float2(A.z, A.w),
                                   __ffma2_rn(uz[s], make_float2(B.x, B.y), make_float2(B.z, B.w))));
                    const float2 e = __ffma2_rn(
                        ux[s], make_float2(C.x, C.y),
                        __ffma2_rn(uy[s], make_float2(C.z, C.w),
                                   __ffma2_rn(uz[s], make_float2(D.x, D.y), make_float2(D.z, D.w))));
                    mind[2 * s] = min3(d.x, e.x, mind[2 * s]);
                    mind[2 * s + 1] = min3(d.y, e.y, mind[2 * s + 1]);
                }
            }
            __syncwarp();
        }

        // ---- 4. selection --------------------------------------------------------------
        // (Only the sign and the size of mind - sigma^2 matter.)
        if (k != G * T)
#pragma unroll
            for (int s = 0; s < T; ++s)
                if (T * g.gl + s >= k) mind[s] = INFINITY;
        uint32_t blocked = 0u;
        bool flag = false;
#pragma unroll
        for (int s = T - 1; s >= 0; --s) {
            const float t = mind[s] - a.sig2;
            blocked = __funnelshift_l(__float_as_uint(t), blocked, 1);
            flag |= fabsf(t) < band;
        }
        const uint32_t fr = ~blocked & tmask;
        // Free trials of the group, and of the lanes before this one: T votes or
        // log2 G shuffles, whichever is fewer.
        const int cnt = __popc(fr);
        int m = 0, before = 0;
        if constexpr (T <= 4 && G >= 16) {
#pragma unroll
            for (int s = 0; s < T; ++s) {
                const unsigned v = __ballot_sync(kAll, (fr >> s) & 1u);
                m += __popc(v & g.mask);
                before += __popc(v & g.below);
            }
        } else {
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                const int u = __shfl_up_sync(kAll, incl, o, G);
                if (g.gl >= o) incl += u;
            }
            m = __shfl_sync(kAll, incl, G - 1, G);
            before = incl - cnt;
        }
        const int r = (int)__umulhi(selw, (uint32_t)m) - before;
        const bool mine = r >= 0 && r < cnt;
        const int ss = nth[(fr << 3) | (uint32_t)(mine ? r : 0)];
        const unsigned who = __ballot_sync(kAll, mine) & g.mask;
        const int src = who ? __ffs(who) - 1 : g.base;
        int sel = __shfl_sync(kAll, T * g.gl + ss, src);
        // Its Philox words, kept since the trials were drawn: T selects and two
        // shuffles in place of a ten-round call by every lane (N = 64, k = 32,
        // 10^6 chains: 9.57 -> 9.26 ms, no more registers).
        uint32_t ca = words[0].x, cb = words[0].y;
#pragma unroll
        for (int s = 0; s < T; ++s)
            if (s == ss) trial_words(words[s / 2], s, ca, cb);
        ca = __shfl_sync(kAll, ca, src);
        cb = __shfl_sync(kAll, cb, src);

        // Steps FP32 cannot decide, a chain at a time with the whole warp.
        unsigned amb = __ballot_sync(kAll, on && flag);
        while (amb) {
            const int from = (__ffs(amb) - 1) & ~(G - 1);     // the chain's first lane
            amb &= ~(unsigned)(((1ull << G) - 1ull) << from);
            const auto b = [&](auto v) { return __shfl_sync(kAll, v, from); };
            const WideDecision d = wide_redecide<G>(
                a, P + ((from - g.base) / G) * sh.stride, np, sh.gref, b(chain), b(att << 16),
                b(exact_upto), b(i), b(selw), b(ehx), b(ehy), b(ehz), b(elx), b(ely), b(elz));
            if (g.base == from) {
                ehx = d.hx;
                ehy = d.hy;
                ehz = d.hz;
                elx = d.lx;
                ely = d.ly;
                elz = d.lz;
                m = d.m;
                if (sel != d.sel) {
                    sel = d.sel;
                    const uint4 xs =
                        philox(make_uint4(chain, a.ens, step, 1u + (uint32_t)(sel >> 1)), a.key);
                    trial_words(xs, sel, ca, cb);
                }
                if (d.exact) {
                    exact_upto = i - 1;
                    ++rechecks;
                }
            }
        }

        // ---- 5. commit: the chosen trial's direction, exactly as off_chain ------------
        const float3 u2 = dir32x2(ca, cb);
        const bool dead = m == 0;
        if (on && !dead) {
            if (g.gl == 0) {
                put(i - 1, ehx, ehy, ehz, elx, ely, elz);
                tr[i] = (uint8_t)sel;
            }
            ff_add_half(ehx, elx, u2.x);
            ff_add_half(ehy, ely, u2.y);
            ff_add_half(ehz, elz, u2.z);
            lw += logm[m];
            ++i;
        }
        __syncwarp();

        // ---- 6. chains that end at this step ------------------------------------------
        if (on && (dead || i == N)) {
            if (dead && att + 1 < a.max_att) {
                ++att;
                restart();
            } else {
                wide_finish<G>(a, g, P, tr, np, sh.gref, c, att, dead, i, lw, rechecks, listed,
                               make_float3(ehx, ehy, ehz), make_float3(elx, ely, elz));
                c = -1;
            }
        }
        __syncwarp();
    }
}

}  // namespace
}  // namespace rosen
