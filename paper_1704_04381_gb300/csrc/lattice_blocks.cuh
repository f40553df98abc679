// lattice_blocks.cuh -- cubic-lattice growth of mid-length chains with the
// occupied sites as bitmaps in shared memory (Guo & Baulin, Section 3.3.2,
// Algorithm 1; weight of Eq. 3).
//
// The scan of lattice.cu costs a step O(i) key tests and holds 4 N bytes of
// shared memory per chain: N = 512 runs 3 warps per SM at 1100 instructions a
// step.  Here a lane keeps its chain's sites in a small hash table in shared
// memory: an entry is a 4x4x4 block of sites, a 32-bit tag (8 bits per axis)
// and a 64-bit occupancy bitmap, 12 bytes, linear probing.  A self-avoiding
// walk of 64 / 128 / 256 / 512 monomers lies in 12 / 21 / 38 / 71 such blocks on
// average; site_entries(N) = 19 N / 100 + 14 of them leave about one chain in
// 10^5 out.  A step looks up the one to three blocks (interacting: three to
// six) its neighbourhood reaches besides the end's, which stays in registers,
// and turns them into one 64-bit picture of the sites around the end.  Entries
// lie [entry][lane], so the lanes' accesses share no bank whatever entries
// they take.
//
// Every lane steps through its own chain and takes the next of its warp's
// range when done (a trapped chain in restart mode at once with its next
// growth).  A chain that would fill its table stops there and is grown again by
// its lane alone with the whole warp's table, once the other lanes are done:
// 32 times the entries, more than the blocks of any chain.
//
// Bound by latency: 5 warps per SM at N = 512 (9 at 256), 454 instructions a
// step, issue 33%.  GB300, scan kernel and now: athermal N = 160, 4 10^5 chains
// 1.32 -> 1.12 ms; 224, 2 10^5: 1.56 -> 1.10; 300, 10^5: 1.80 -> 0.81; 512, 5
// 10^5: 26.5 -> 9.7; beta eps = 0.4, N = 160, 3 10^5: 1.75 -> 1.64; 224, 2
// 10^5: 2.69 -> 1.95; 512, 2 10^5: 18.4 -> 7.2.  At N = 128 the scan is faster
// (1.02 against 1.21 ms; 1.08 against 1.35 interacting); between 160 and 208 it
// depends on the call (blocks_win in lattice.cu).  Tried and not kept:
// buckets of four tags in one load (10.7 ms at N = 512), two buckets per block
// without a loop (overflows: 36 ms).
#pragma once

#include "lattice_step.cuh"

namespace rosen {
namespace {

// Table entries per lane for chains of N monomers.
__host__ __device__ inline int site_entries(int N) { return 19 * N / 100 + 14; }

constexpr uint32_t kSiteOrigin = 0x808080u;   // tag of block (0, 0, 0); a tag is never 0
constexpr uint32_t kSiteMul = 0x9E3779B1u;

// A lane's table of H entries: entry h has its tag at tag[h * step] (0: empty)
// and its bitmap at bits[h * step].  Linear probing from the key's place.
struct SiteTable {
    uint32_t *tag;
    uint2 *bits;
    int step;     // 32: a lane's table; 1: the whole warp's
    uint32_t H;
};

__device__ __forceinline__ uint32_t site_place(const SiteTable &t, uint32_t key)
{
    return __umulhi(key * kSiteMul, t.H);
}

// A block found (its bitmap and entry) or not (no bits, the empty entry where
// it would go).
struct SiteRef {
    uint2 bits;
    uint32_t h;
    bool found;
};

// Look up K blocks together; need[q] == false: none.  The probes of a round
// are loaded before any is examined.
template <int K>
__device__ __forceinline__ void find_sites(const SiteTable &t, const uint32_t (&want)[K],
                                           const bool (&need)[K], SiteRef (&ref)[K])
{
    uint32_t tag[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        ref[q].h = site_place(t, want[q]);
        tag[q] = t.tag[ref[q].h * t.step];
    }
    for (;;) {
        bool any = false;
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const bool on = need[q] && tag[q] != want[q] && tag[q] != 0u;
            if (on) {
                ref[q].h = ref[q].h + 1u == t.H ? 0u : ref[q].h + 1u;
                tag[q] = t.tag[ref[q].h * t.step];
            }
            any |= on;
        }
        if (!any) break;
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
        ref[q].found = need[q] && tag[q] == want[q];
        ref[q].bits = t.bits[ref[q].h * t.step];
        if (!ref[q].found) ref[q].bits = make_uint2(0u, 0u);
    }
}

// The bits of a block turned right by n (mod 64): bit d of the result is site
// n + d.
__device__ __forceinline__ uint2 turn(uint2 v, int n)
{
    const uint32_t a = (n & 32) ? v.y : v.x, b = (n & 32) ? v.x : v.y;
    return make_uint2(__funnelshift_r(a, b, n), __funnelshift_r(b, a, n));
}

// a where the mask is clear, b where it is set.
__device__ __forceinline__ uint2 mix(uint2 a, uint2 b, uint2 mask)
{
    return make_uint2((a.x & ~mask.x) | (b.x & mask.x), (a.y & ~mask.y) | (b.y & mask.y));
}

// Sites around the end in the turned frame: offset dx + 4 dy + 16 dz (mod 64).
constexpr uint64_t site_at(int d) { return 1ull << (d & 63); }
constexpr uint64_t site_mask(int s, int u, int v, int two)
{
    // Offsets of the sites one step along s (and one along +-u, +-v) and, with
    // `two`, two steps along s.
    return site_at(s) | site_at(s + u) | site_at(s - u) | site_at(s + v) | site_at(s - v) |
           (two ? site_at(2 * s) : 0ull);
}
// The sites that lie in the neighbouring block when the end's coordinate in its
// block is 0..3, per axis.  (Two steps along z are bit 32 either way: apart.)
__device__ __forceinline__ void fill_site_masks(uint2 *masks)
{
    constexpr uint64_t m[12] = {
        site_mask(-1, 4, 16, 1), site_at(-2), site_at(2), site_mask(1, 4, 16, 1),
        site_mask(-4, 1, 16, 1), site_at(-8), site_at(8), site_mask(4, 1, 16, 1),
        site_mask(-16, 1, 4, 0), 0ull,        0ull,       site_mask(16, 1, 4, 0)};
#pragma unroll
    for (int q = 0; q < 12; ++q)
        if (threadIdx.x == 0) masks[q] = make_uint2((uint32_t)m[q], (uint32_t)(m[q] >> 32));
}

// State of a lane's chain between steps.
struct SiteWalk {
    int ex, ey, ez;            // end
    int sx, sy, sz, sq;        // sums of the coordinates and of their squares
    uint64_t cnt;              // 9-bit field m: steps with m free sites
    LogW lw;
    int p;                     // the end's place in its block: x + 4 y + 16 z
    uint32_t key, h;           // the block: tag and entry
    uint2 cur;                 // and its bitmap
    uint32_t blocks;
};

__device__ __forceinline__ void begin_sites(SiteWalk &w, const SiteTable &t)
{
    for (uint32_t h = 0; h < t.H; ++h) t.tag[h * t.step] = 0u;
    w.ex = w.ey = w.ez = 0;
    w.sx = w.sy = w.sz = w.sq = 0;
    w.cnt = 0ull;
    w.lw = LogW();
    w.p = 0;
    w.key = kSiteOrigin;
    w.cur = make_uint2(1u, 0u);                    // site (0, 0, 0): bit 0
    w.blocks = 1u;
    w.h = site_place(t, w.key);
    t.tag[w.h * t.step] = w.key;
    t.bits[w.h * t.step] = w.cur;
}

// Blocks a step looks up: across the face the end is nearer to on x, y and z;
// interacting chains also across two faces (x y, x z, y z).
template <bool kIsaw>
constexpr int kSiteBlocks = kIsaw ? 6 : 3;

// What lies around the end at place p of its block (bitmap cur), nb[] the
// bitmaps of the neighbouring blocks: bits 0..5, neighbour d is occupied; bits
// 8+3d..10+3d (interacting), the contacts of neighbour d.
template <bool kIsaw>
__device__ __forceinline__ uint32_t sites_around(int p, uint2 cur,
                                                 const uint2 (&nb)[kSiteBlocks<kIsaw>],
                                                 const uint2 *masks)
{
    const int qx = p & 3, qy = (p >> 2) & 3, qz = p >> 4;
    const int tx = qx > 1 ? p - 4 : p + 4, ty = qy > 1 ? p - 16 : p + 16;
    // The sites around the end in one turned bitmap: those of the end's block,
    // those across a face from its neighbours' bitmaps, turned to match.
    const uint2 mx = masks[qx], my = masks[4 + qy], mz = masks[8 + qz];
    uint2 M = turn(cur, p);
    const uint2 X = turn(nb[0], tx), Y = turn(nb[1], ty), Z = turn(nb[2], p);
    uint32_t two_in = 0u, two_out = 0u;    // two steps along z, in the block and across
    if constexpr (kIsaw) {
        two_in = M.y & 1u;
        two_out = Z.y & 1u;
        const uint2 XY = turn(nb[3], qy > 1 ? tx - 16 : tx + 16), XZ = turn(nb[4], tx),
                    YZ = turn(nb[5], ty);
        M = mix(mix(M, X, mx), mix(Y, XY, mx), my);
        M = mix(M, mix(mix(Z, XZ, mx), YZ, my), mz);
    } else {
        M = mix(mix(mix(M, X, mx), Y, my), Z, mz);
    }
    // Neighbour bits in slot order: offsets 1, 4, 16 are bits 1, 4, 16 of the
    // low word and -1, -4, -16 bits 31, 28, 16 of the high word; two multiplies
    // gather them into bits 26, 28, 30 and 27, 29, 31.
    const uint32_t plus = (M.x & 0x00010012u) * ((1u << 25) | (1u << 24) | (1u << 14));
    const uint32_t minus = ((M.y >> 16) & 0x9001u) * ((1u << 12) | (1u << 17) | (1u << 31));
    const uint32_t occ = ((plus & 0x54000000u) | (minus & 0xA8000000u)) >> 26;
    uint32_t acc = occ;
    if constexpr (kIsaw) {
        // Contacts of neighbour d: the sites next to it other than the end.
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            const int s = (d & 1) ? -(1 << (d & 6)) : 1 << (d & 6);
            const int u = d < 2 ? 4 : 1, v = d < 4 ? 16 : 4;
            const uint64_t m = site_mask(s, u, v, d < 4) & ~site_at(s);
            uint32_t cd = __popc(M.x & (uint32_t)m) + __popc(M.y & (uint32_t)(m >> 32));
            if (d >= 4) cd += ((d == 4) == (qz <= 1)) ? two_in : two_out;
            acc |= cd << (8 + 3 * d);
        }
    }
    return acc;
}

// One step from the chain's end with draw x.  Returns the number of free
// neighbours (0: trapped), -1 if the table is full; sel: the neighbour taken.
template <bool kIsaw>
__device__ __forceinline__ int step_sites(SiteWalk &w, const SiteTable &t, uint32_t x,
                                          const uint8_t *seltab, const uint2 *masks,
                                          const float *wt32, const double *wt64, int &sel)
{
    const int p = w.p, qx = p & 3, qy = (p >> 2) & 3, qz = p >> 4;
    // Two bits per axis, + and -: the neighbour lies across a face.
    const uint32_t cx = (0x42u >> (2 * qx)) & 3u, cy = (0x42u >> (2 * qy)) & 3u,
                   cz = (0x42u >> (2 * qz)) & 3u;
    const uint32_t across = cx | (cy << 2) | (cz << 4);
    // The neighbouring block per axis lies on the side the end is nearer to:
    // sites within two steps reach no other.
    const uint32_t ox = qx > 1 ? 1u : 0xFFFFFFFFu, oy = qy > 1 ? 256u : 0xFFFFFF00u,
                   oz = qz > 1 ? 65536u : 0xFFFF0000u;
    constexpr int K = kSiteBlocks<kIsaw>;
    uint32_t want[K];
    bool need[K];
    want[0] = w.key + ox;
    want[1] = w.key + oy;
    want[2] = w.key + oz;
    need[0] = kIsaw || cx;
    need[1] = kIsaw || cy;
    need[2] = kIsaw || cz;
    if constexpr (kIsaw) {
        // Blocks across two faces: x y, x z, y z.
        want[3] = want[0] + oy;
        want[4] = want[0] + oz;
        want[5] = want[1] + oz;
        need[3] = cx && cy;
        need[4] = cx && cz;
        need[5] = cy && cz;
    }
    SiteRef ref[K];
    find_sites<K>(t, want, need, ref);

    uint2 nb[K];
#pragma unroll
    for (int q = 0; q < K; ++q) nb[q] = ref[q].bits;
    const uint32_t acc = sites_around<kIsaw>(p, w.cur, nb, masks), occ = acc & 63u;
    const uint32_t freem = ~occ & 63u;
    const int m = __popc(freem);
    if (m == 0) return 0;
    sel = choose<kIsaw>(freem, m, acc, x, seltab, wt32, wt64, w.lw);
    w.cnt += 1ull << (9 * m);

    // The new site, in the end's block or across a face.
    const int axis2 = sel & 6, s = 1 << axis2;
    const int dir = (sel & 1) ? -1 : 1;
    if ((across >> sel) & 1u) {
        const bool first = axis2 == 0, second = axis2 == 2;
        w.cur.x = first ? ref[0].bits.x : (second ? ref[1].bits.x : ref[2].bits.x);
        w.cur.y = first ? ref[0].bits.y : (second ? ref[1].bits.y : ref[2].bits.y);
        w.h = first ? ref[0].h : (second ? ref[1].h : ref[2].h);
        w.key = first ? want[0] : (second ? want[1] : want[2]);
        w.p = p - 3 * dir * s;
        const bool found = first ? ref[0].found : (second ? ref[1].found : ref[2].found);
        if (!found) {
            // (One entry stays empty: every probe sequence ends.)
            if (++w.blocks >= t.H) return -1;
            t.tag[w.h * t.step] = w.key;
        }
    } else {
        w.p = p + dir * s;
    }
    if (w.p & 32) w.cur.y |= 1u << (w.p & 31);
    else w.cur.x |= 1u << (w.p & 31);
    t.bits[w.h * t.step] = w.cur;
    if (axis2 == 0) w.ex += dir;
    else if (axis2 == 2) w.ey += dir;
    else w.ez += dir;
    w.sx += w.ex;
    w.sy += w.ey;
    w.sz += w.ez;
    w.sq += w.ex * w.ex + w.ey * w.ey + w.ez * w.ez;
    return m;
}

// Outputs of step i of chain c (the trace byte and the new monomer).
__device__ __forceinline__ void store_step(const LatticeArgs &a, int64_t c, int i, int m, int sel,
                                           const SiteWalk &w)
{
    if (a.trace) a.trace[(int64_t)(i - 1) * a.C + c] = (uint8_t)((m << 3) | sel);
    if (a.coords) {
        a.coords[((int64_t)i * 3 + 0) * a.C + c] = w.ex;
        a.coords[((int64_t)i * 3 + 1) * a.C + c] = w.ey;
        a.coords[((int64_t)i * 3 + 2) * a.C + c] = w.ez;
    }
}

// Outputs of a finished chain (dead: trapped at step i).
template <bool kIsaw>
__device__ __forceinline__ void finish_sites(const LatticeArgs &a, int64_t c, uint32_t att, int i,
                                             bool dead, SiteWalk &w)
{
    const int N = a.N;
    const int64_t C = a.C;
    if (a.attempts) a.attempts[c] = (uint16_t)(att + 1);
    uint32_t cm[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) cm[q] = (uint32_t)(w.cnt >> (9 * q)) & 511u;
    if (a.counts)
        a.counts[c] = make_uint4((dead ? 1u : 0u) | (cm[1] << 16), cm[2] | (cm[3] << 16),
                                 cm[4] | (cm[5] << 16), cm[6]);
    float logw = -INFINITY;
    if (!dead) {
        if (kIsaw) {
            logw = w.lw.value();
        } else {
            logw = 0.f;
#pragma unroll
            for (int q = 2; q <= 6; ++q) logw += (float)cm[q] * a.logm[q];
        }
    }
    if (a.logw) a.logw[c] = logw;
    if (a.r2) a.r2[c] = dead ? 0 : w.ex * w.ex + w.ey * w.ey + w.ez * w.ez;
    if (a.n2rg2)
        a.n2rg2[c] = dead ? 0
                          : (int64_t)N * w.sq - ((int64_t)w.sx * w.sx + (int64_t)w.sy * w.sy +
                                                 (int64_t)w.sz * w.sz);
    if (dead) {
        if (a.trace) {
            a.trace[(int64_t)(i - 1) * C + c] = 7u;
            for (int s = i + 1; s < N; ++s) a.trace[(int64_t)(s - 1) * C + c] = 0xFFu;
        }
        if (a.coords)
            for (int s = 3 * i; s < 3 * N; ++s) a.coords[(int64_t)s * C + c] = 0;
    }
}

__device__ __forceinline__ void first_monomer(const LatticeArgs &a, int64_t c)
{
    if (a.coords)
        for (int q = 0; q < 3; ++q) a.coords[(int64_t)q * a.C + c] = 0;
}

// Block w (one warp) grows chains [c_lo + w per_warp, ...) below c_hi.
template <bool kIsaw>
__global__ void __launch_bounds__(32) lattice_blocks_kernel(const LatticeArgs a, int H,
                                                             int64_t per_warp, int64_t c_lo,
                                                             int64_t c_hi)
{
    extern __shared__ __align__(16) uint32_t smem[];
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ uint8_t seltab[kSelBytes];
    __shared__ float wt32[8];
    __shared__ double wt64[8];
    __shared__ uint2 masks[12];
    fill_site_masks(masks);
    for (int q = threadIdx.x; q < kSelBytes; q += blockDim.x)
        seltab[q] = nth_set_bit((uint32_t)q >> 3, (uint32_t)q & 7u);
    if (threadIdx.x < 8) {
        wt32[threadIdx.x] = a.wt32[threadIdx.x];
        wt64[threadIdx.x] = a.wt64[threadIdx.x];
    }
    const int lane = threadIdx.x;
    // The warp's entries: bitmaps, then tags.
    uint2 *const bits = reinterpret_cast<uint2 *>(smem);
    uint32_t *const tags = reinterpret_cast<uint32_t *>(bits + (size_t)H * 32);
    __syncthreads();
    const SiteTable tab = {tags + lane, bits + lane, 32, (uint32_t)H};

    int64_t next = c_lo + blockIdx.x * per_warp;
    const int64_t hi = next + per_warp < c_hi ? next + per_warp : c_hi;
    // Traces and conformations are written a step's row at a time: then the
    // lanes stay in step (a warp's stores are contiguous).
    const bool together = a.trace || a.coords;
    uint32_t att = 0u;
    int64_t c = -1, over = -1;         // the lane's chain; one that filled its table
    int i = 0;
    SiteWalk s;
    for (;;) {
        const unsigned idle = __ballot_sync(kAll, c < 0 && over < 0);
        if (idle && next < hi && (!together || idle == kAll)) {
            const int64_t n = next + __popc(idle & ((1u << lane) - 1u));
            next += __popc(idle);
            if (((idle >> lane) & 1u) && n < hi) {
                c = n;
                att = 0u;
                i = 1;
                begin_sites(s, tab);
                first_monomer(a, c);
            }
        }
        if (!__any_sync(kAll, c >= 0)) {
            // Chains that filled their tables, one after another with the
            // whole warp's (their lane alone; the others' entries are free).
            unsigned full = __ballot_sync(kAll, over >= 0);
            if (!full) break;
            for (; full; full &= full - 1u) {
                __syncwarp();
                if (lane == __ffs(full) - 1) {
                    const SiteTable big = {tags, bits, 1, 32u * (uint32_t)H};
                    for (att = 0u;; ++att) {
                        begin_sites(s, big);
                        first_monomer(a, over);
                        bool dead = false;
                        for (i = 1; i < a.N && !dead; ++i) {
                            const uint32_t x = philox(make_uint4(a.chain0 + (uint32_t)over, a.ens,
                                                                 (uint32_t)i | (att << 16), 0u),
                                                      a.key).x;
                            int sel = 0;
                            const int m = step_sites<kIsaw>(s, big, x, seltab, masks, wt32,
                                                            wt64, sel);
                            dead = m <= 0;
                            if (dead) break;
                            store_step(a, over, i, m, sel, s);
                        }
                        if (dead && att + 1 < a.max_att) continue;
                        finish_sites<kIsaw>(a, over, att, i, dead, s);
                        break;
                    }
                    over = -1;
                }
                __syncwarp();
            }
            continue;
        }
        if (c >= 0) {
            const uint32_t x = philox(make_uint4(a.chain0 + (uint32_t)c, a.ens,
                                                 (uint32_t)i | (att << 16), 0u), a.key).x;
            int sel = 0;
            const int m = step_sites<kIsaw>(s, tab, x, seltab, masks, wt32, wt64, sel);
            if (m > 0) {
                store_step(a, c, i, m, sel, s);
                if (++i == a.N) {
                    finish_sites<kIsaw>(a, c, att, i, false, s);
                    c = -1;
                }
            } else if (m < 0) {
                over = c;
                c = -1;
            } else if (att + 1 < a.max_att) {
                ++att;
                i = 1;
                begin_sites(s, tab);
            } else {
                finish_sites<kIsaw>(a, c, att, i, true, s);
                c = -1;
            }
        }
        __syncwarp();
    }
}

}  // namespace
}  // namespace rosen
