// sd_plane.cu -- Algorithm 1 (Update DHLA) binned by estimator bit: the
// default update of sd_update (tuning mode 6).
//
// For one pair and one direction, Algorithm 1 sets the SAME bit b = H1(elem)
// in each of the r estimators DH_i(key), i < r (Eq. 2): one hash H1 per pair
// and direction, shared by the rows (§3.2).  Call "plane (d, b)" bit b of
// every estimator of direction d: r rows of 2^k bits, one bit per estimator.
// All r bit-sets of a (pair, direction) fall in one plane, at positions that
// depend on the key alone.  So the update is binned by plane with ONE entry
// per pair and direction -- the key itself -- and the rows are hashed where
// the plane is held, in shared memory:
//
//   k_plane_bin    tiles of pairs: the keys sorted by plane in shared memory,
//                  each plane's run appended to its bin with coalesced
//                  stores (one reservation atomic per plane and tile).  The
//                  bins are laid out back to back (each starting on a
//                  16-byte boundary) from the previous round's counts plus
//                  slack; keys beyond a bin's capacity (traffic that shifted
//                  between rounds) set their bits directly with atomic ORs.
//                  The last block cuts each plane's bin into apply units.
//                  A longer round than the one before (of enough pairs to
//                  go by) takes those bins times a power of two.
//   k_plane_layout for a longer round where the bins have not that room:
//                  the previous per-plane counts scaled to this round's
//                  size, plus slack.
//   k_plane_count  for a round with no usable history (the first one, one
//                  over other directions, or one after a small round): the
//                  exact keys of every plane, and a layout without slack.
//   k_plane_direct for a round of few pairs, instead of all the others: every
//                  bit ORed into the plane copy where it lies.
//   k_plane_apply  one unit (a plane and a range of its bin) per block step:
//                  the plane in shared memory, DH_0 and Eq. 2 of every key,
//                  r shared-memory ORs, then one bulk OR of the plane into
//                  the plane-major copy of the DHLA in L2
//                  (cp.reduce.async.bulk ... .or.b32, so units of one plane
//                  may run on several SMs).  The last block lays out the
//                  next round's bins from this round's counts.
//   k_plane_scan   (sd_fold.cu; window close) counts the plane-major copy as
//                  it is and clears it.
//   k_plane_fold   (sd_fold.cu; sd_get_grid, sd_merge, and a close where the
//                  DHLA holds bits of its own) folds the copy into the
//                  estimator-major DHLA (grid |= planes^T) and clears it.
//
// Per pair this moves dirs keys (4 bytes each) through the bins instead of
// r * dirs bit positions, and the plane copy is swept once per round by
// the bulk reduction.  The result equals Algorithm 1's DHLA bit for bit: the
// effective DHLA of a handle is grid | planes^T at all times, and every step
// only ORs bits in.
//
// Plane-major layout: plane (d, b) is plane index d*g + b; its row i starts
// at word i * 2^k/32 and holds estimator c's bit at word c >> 5, bit c & 31;
// planes are ps words apart (r 2^k / 32 rounded up to 4 words).
#include "sd_common.cuh"

namespace sd {

namespace {

constexpr uint32_t kPlaneThreads = 512;   // k_plane_bin / k_plane_count block
constexpr uint32_t kApplyThreads = 512;   // k_plane_apply block (1024 where one plane fills the block's shared memory)
constexpr uint32_t kHeldReservations = 2;  // reservation results a thread holds across the scatter
constexpr uint32_t kBinTilesPerBlock = 8;   // k_plane_bin tiles per block (blocks retire as a round runs)
constexpr uint32_t kDependentPlaneWords = 512;  // narrower planes: k_plane_apply in a plain launch
constexpr uint32_t kDirectThreads = 256;    // k_plane_direct block: a tile of pairs (numbered in 8 bits)
constexpr uint32_t kDirectSlots = 2048;     // hash slots for finding a tile's equal pairs
constexpr uint32_t kApplyUnitsPerBlock = 4; // k_plane_apply units per block, at most

__device__ __forceinline__ uint32_t h1v(uint64_t A1, uint64_t B1, uint32_t lg, uint32_t y) {
    return (uint32_t)((A1 * (uint64_t)y + B1) >> (64u - lg));
}

// 16-byte load that stays in L2 for the next kernel of the round.
__device__ __forceinline__ uint4 ld_l2_v4(const uint4 *p) {
    uint4 v;
    asm("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// Block-wide exclusive scan of get(0..N) written through put(i, prefix);
// put(N, total) as well.  Each thread takes a contiguous chunk of indices.
// Ends with a barrier; s_warp holds 32 words of shared scratch.
template <typename Get, typename Put>
__device__ __forceinline__ void block_scan(uint32_t N, Get get, Put put, uint32_t *s_warp) {
    const uint32_t per = (N + blockDim.x - 1) / blockDim.x;
    const uint32_t i0 = min(threadIdx.x * per, N), i1 = min(i0 + per, N);
    uint32_t sum = 0;
    for (uint32_t i = i0; i < i1; i++) sum += get(i);
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += v;
    }
    __syncthreads();  // s_warp may still be read by an earlier scan
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        uint32_t x = lane < nw ? s_warp[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if ((int)lane >= o) x += v;
        }
        if (lane < nw) s_warp[lane] = x;
    }
    __syncthreads();
    uint32_t run = incl - sum + (wid ? s_warp[wid - 1] : 0u);
    for (uint32_t i = i0; i < i1; i++) {
        const uint32_t v = get(i);
        put(i, run);
        run += v;
    }
    if (threadIdx.x == blockDim.x - 1) put(N, run);
    __syncthreads();
}

// Capacity of a bin for an expected count c: c plus an eighth and 32 slots
// of slack when `slack`, rounded up to 4 entries.
__device__ __forceinline__ uint32_t bin_cap(uint32_t c, bool slack) {
    return (c + (slack ? c / 8u + 32u : 0u) + 3u) & ~3u;
}

// One block: the bins of the next round from this round's per-plane counts
// (cnt, then kept in prev and cleared), bins back to back.  The caller has
// seen every count (last-block pattern).
__device__ __forceinline__ void write_layout(const PlaneArgs &P, bool slack, uint32_t *s_warp) {
    const uint32_t NB = P.nbins;
    auto cap_of = [&](uint32_t i) { return bin_cap(__ldcg(&P.cnt[i]), slack); };
    block_scan(NB, cap_of, [&](uint32_t i, uint32_t v) { P.binoff[i] = v; }, s_warp);
    for (uint32_t b = threadIdx.x; b < NB; b += blockDim.x) {
        const uint32_t c = __ldcg(&P.cnt[b]);
        P.cap[b] = bin_cap(c, slack);
        P.prev[b] = c;
        P.cnt[b] = 0;
    }
}

// First slot and slots of plane b's bin in this round.
__device__ __forceinline__ uint32_t bin_off(const PlaneArgs &P, uint32_t b) { return P.binoff[b] << P.shift; }
__device__ __forceinline__ uint32_t bin_room(const PlaneArgs &P, uint32_t b) { return P.cap[b] << P.shift; }

// The last block to call this (one call per block, counter at *done) gets
// true, after a fence that makes every earlier block's writes visible.
__device__ __forceinline__ bool last_block(uint32_t *done, bool *s_last) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        *s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!*s_last) return false;
    __threadfence();
    return true;
}

// Set the r bits of `key` in plane b of the plane-major copy directly (a
// key its bin had no room for).
template <int DIRS>
__device__ __forceinline__ void set_key_bits(const Geometry &G, const PlaneArgs &P, uint32_t b, uint32_t key) {
    const uint32_t A0 = (DIRS == 2 && (b >> G.lg)) ? G.h[1].A0 : G.h[0].A0;
    const uint32_t rw = (1u << G.k) >> 5;
    uint32_t *pl = P.planes + (uint64_t)b * P.ps;
    const uint32_t c0 = dh0(A0, G.k, key);
    red_or(pl + (c0 >> 5), 1u << (c0 & 31u));
    for (uint32_t i = 1; i < G.r; i++) {
        const uint32_t ci = dh_row(G, i, key, c0);
        red_or(pl + i * rw + (ci >> 5), 1u << (ci & 31u));
    }
}

}  // namespace

// ------------------------------------------------------------------ count
template <int DIRS>
__global__ void __launch_bounds__(kPlaneThreads)
k_plane_count(const uint32_t *__restrict__ pairs, uint64_t n, Geometry G, PlaneArgs P) {
    extern __shared__ uint32_t hist[];  // [nbins]
    __shared__ uint32_t s_warp[32];
    __shared__ bool s_last;
    const uint32_t NB = P.nbins, g = G.g, lg = G.lg;
    const uint64_t A1a = G.h[0].A1, B1a = G.h[0].B1, A1b = G.h[1].A1, B1b = G.h[1].B1;
    for (uint32_t b = threadIdx.x; b < NB; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    auto count = [&](uint32_t s, uint32_t t) {
        atomicAdd(&hist[h1v(A1a, B1a, lg, t)], 1u);
        if (DIRS == 2) atomicAdd(&hist[g + h1v(A1b, B1b, lg, s)], 1u);
    };
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (((uintptr_t)pairs & 15u) == 0) {
        // four 16-byte loads in flight per thread
        const uint4 *v4 = reinterpret_cast<const uint4 *>(pairs);
        const uint64_t n2 = n / 2;
        uint64_t u = first;
        for (; u + 3 * stride < n2; u += 4 * stride) {
            uint4 v[4];
#pragma unroll
            for (int j = 0; j < 4; j++) v[j] = ld_l2_v4(v4 + u + j * stride);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                count(v[j].x, v[j].y);
                count(v[j].z, v[j].w);
            }
        }
        for (; u < n2; u += stride) {
            const uint4 v = ld_l2_v4(v4 + u);
            count(v.x, v.y);
            count(v.z, v.w);
        }
        if ((n & 1) && first == 0) count(pairs[2 * (n - 1)], pairs[2 * (n - 1) + 1]);
    } else {
        for (uint64_t p = first; p < n; p += stride) count(ld_stream_u32(pairs + 2 * p), ld_stream_u32(pairs + 2 * p + 1));
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < NB; b += blockDim.x)
        if (hist[b]) atomicAdd(&P.cnt[b], hist[b]);
    if (!last_block(&P.ctl[0], &s_last)) return;
    // every count is in cnt: bins of exactly this round's sizes
    write_layout(P, false, s_warp);
    if (threadIdx.x == 0) P.ctl[0] = 0;
}

// ----------------------------------------------------------------- layout
// One block: bins for a round of `num` pairs from the per-plane counts of a
// previous round of `den` pairs (prev), each count scaled by num / den
// (rounded up) and given slack.  Their total stays within the bins of a
// round of num pairs: sum ceil(prev num / den) <= keys + nbins.
__global__ void __launch_bounds__(1024) k_plane_layout(PlaneArgs P, uint64_t num, uint64_t den) {
    __shared__ uint32_t s_warp[32];
    auto cap_of = [&](uint32_t i) {
        return bin_cap((uint32_t)(((uint64_t)P.prev[i] * num + den - 1) / den), true);
    };
    block_scan(P.nbins, cap_of, [&](uint32_t i, uint32_t v) { P.binoff[i] = v; }, s_warp);
    for (uint32_t b = threadIdx.x; b < P.nbins; b += blockDim.x) P.cap[b] = cap_of(b);
}

// -------------------------------------------------------------------- bin
// A thread keeps PPT pairs' DIRS entries in registers as (key, plane << 16
// | rank) while the block counts them per plane; the tile is then scattered
// into plane order in shared memory as 64-bit (plane << 32 | key) entries
// and written out one thread per entry, so each plane's run goes to
// consecutive addresses of its bin.
template <int DIRS, int PPT, bool FULL>
__device__ __forceinline__ void bin_hash(uint32_t cnt, const uint32_t (&ps)[PPT], const uint32_t (&pt)[PPT],
                                         uint32_t g, uint32_t lg, uint64_t A1a, uint64_t B1a, uint64_t A1b,
                                         uint64_t B1b, uint32_t *hist, uint32_t (&key)[PPT * DIRS],
                                         uint32_t (&tag)[PPT * DIRS]) {
#pragma unroll
    for (int j = 0; j < PPT / 2; j++) {
        const uint32_t pu = threadIdx.x + (uint32_t)j * blockDim.x;  // 2-pair unit within the tile
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const bool ok = FULL || 2 * pu + q < cnt;
#pragma unroll
            for (int d = 0; d < DIRS; d++) {
                const int e = (2 * j + q) * DIRS + d;
                key[e] = d ? pt[2 * j + q] : ps[2 * j + q];
                const uint32_t b = d ? g + h1v(A1b, B1b, lg, ps[2 * j + q]) : h1v(A1a, B1a, lg, pt[2 * j + q]);
                tag[e] = 0xFFFFFFFFu;
                if (ok) tag[e] = (b << 16) | atomicAdd(&hist[b], 1u);
            }
        }
    }
}

// SHIFTED: the round's bins are the layout times 2^P.shift (a kernel of its
// own: the shifts cost the others 3% through the register allocation).
template <int DIRS, int PPT, int THREADS, bool SHIFTED>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
k_plane_bin(const uint32_t *__restrict__ pairs, uint64_t n, Geometry G, PlaneArgs P, uint32_t head,
            uint32_t tile) {
    constexpr int E = PPT * DIRS;
    dependents_may_start();
    extern __shared__ unsigned long long sm64[];
    __shared__ uint32_t s_warp[32];
    __shared__ bool s_last;
    const uint32_t NB = P.nbins, g = G.g, lg = G.lg;
    const uint32_t TP = blockDim.x * PPT;
    unsigned long long *sent = sm64;                               // [DIRS TP] (plane << 32 | key), plane order
    uint2 *dst = reinterpret_cast<uint2 *>(sent + (size_t)DIRS * TP);  // [NB] (bin index of sorted position 0,
                                                                   //  sorted positions below .y fit the bin)
    uint32_t *hist = reinterpret_cast<uint32_t *>(dst + NB);       // [NB] entries of each plane in the tile
    uint32_t *offs = hist + NB;                                    // [NB] first sorted position of each plane
    const uint64_t A1a = G.h[0].A1, B1a = G.h[0].B1, A1b = G.h[1].A1, B1b = G.h[1].B1;
    const uint64_t ntiles = (n + tile - 1) / tile;  // (tile <= TP pairs each)
    const bool vec = ((uintptr_t)pairs & 15u) == 0;
    // planes owned by this thread in the scan (contiguous chunk)
    const uint32_t per = (NB + blockDim.x - 1) / blockDim.x;
    const uint32_t b0 = min(threadIdx.x * per, NB), b1 = min(b0 + per, NB);
    // this thread's pairs of tile t: 2-pair units threadIdx.x + j blockDim.x
    // (coalesced 16-byte loads where the buffer allows)
    auto load_tile = [&](uint64_t t, uint32_t (&ps)[PPT], uint32_t (&pt)[PPT]) {
        const uint64_t base = t * tile;
        const uint64_t left = t < ntiles ? n - base : 0;
        const uint32_t cnt = left < tile ? (uint32_t)left : tile;
#pragma unroll
        for (int j = 0; j < PPT / 2; j++) {
            const uint32_t pu = threadIdx.x + (uint32_t)j * blockDim.x;
            const uint64_t p = base + 2ull * pu;
            const bool ok0 = 2 * pu < cnt, ok1 = 2 * pu + 1 < cnt;
            ps[2 * j] = pt[2 * j] = ps[2 * j + 1] = pt[2 * j + 1] = 0u;
            if (vec && ok1) {
                const uint4 v = ld_stream_v4(reinterpret_cast<const uint4 *>(pairs + 2 * p));
                ps[2 * j] = v.x; pt[2 * j] = v.y; ps[2 * j + 1] = v.z; pt[2 * j + 1] = v.w;
            } else {
                if (ok0) { ps[2 * j] = ld_stream_u32(pairs + 2 * p); pt[2 * j] = ld_stream_u32(pairs + 2 * p + 1); }
                if (ok1) {
                    ps[2 * j + 1] = ld_stream_u32(pairs + 2 * p + 2);
                    pt[2 * j + 1] = ld_stream_u32(pairs + 2 * p + 3);
                }
            }
        }
    };
    for (uint32_t b = threadIdx.x; b < NB; b += blockDim.x) hist[b] = 0;
    if (head && blockIdx.x == 0 && threadIdx.x == 0) {  // the pair before `pairs`
        const uint32_t s = pairs[-2], t = pairs[-1];
        set_key_bits<DIRS>(G, P, h1v(A1a, B1a, lg, t), s);
        if (DIRS == 2) set_key_bits<DIRS>(G, P, g + h1v(A1b, B1b, lg, s), t);
    }
    __syncthreads();
    uint32_t nps[PPT], npt[PPT];  // the next tile's pairs, loaded while the current one is written out
    load_tile(blockIdx.x, nps, npt);
    for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const uint64_t left = n - t * tile;
        const uint32_t cnt = left < tile ? (uint32_t)left : tile;
        const bool full = cnt == TP;
        uint32_t key[E], tag[E];
        if (full) bin_hash<DIRS, PPT, true>(cnt, nps, npt, g, lg, A1a, B1a, A1b, B1b, hist, key, tag);
        else bin_hash<DIRS, PPT, false>(cnt, nps, npt, g, lg, A1a, B1a, A1b, B1b, hist, key, tag);
        __syncthreads();
        // planes of this thread's chunk: sorted offsets, and their runs
        // reserved in the bins (the first kHeldReservations atomics' results
        // are used after the scatter, so their round trip overlaps it; with
        // more planes per thread the rest are resolved at once)
        uint32_t run = 0;
        {
            uint32_t sum = 0;
            for (uint32_t b = b0; b < b1; b++) sum += hist[b];
            const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if ((int)lane >= o) incl += v;
            }
            if (lane == 31) s_warp[wid] = incl;
            __syncthreads();
            if (wid == 0) {
                uint32_t x = lane < nw ? s_warp[lane] : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, x, o);
                    if ((int)lane >= o) x += v;
                }
                if (lane < nw) s_warp[lane] = x;
            }
            __syncthreads();
            run = incl - sum + (wid ? s_warp[wid - 1] : 0u);
        }
        uint32_t res[kHeldReservations], rrun[kHeldReservations], rcap[kHeldReservations],
            roff[kHeldReservations];
#pragma unroll
        for (uint32_t q = 0; q < kHeldReservations; q++) {
            const uint32_t b = b0 + q;
            res[q] = 0;
            rrun[q] = run;
            rcap[q] = 0;
            roff[q] = 0;
            if (b < b1) {
                const uint32_t h = hist[b];
                offs[b] = run;
                if (h) {
                    res[q] = atomicAdd(&P.cnt[b], h);
                    rcap[q] = SHIFTED ? bin_room(P, b) : P.cap[b];
                    roff[q] = SHIFTED ? bin_off(P, b) : P.binoff[b];
                }
                hist[b] = 0;
                run += h;
            }
        }
        for (uint32_t b = b0 + kHeldReservations; b < b1; b++) {
            const uint32_t h = hist[b];
            offs[b] = run;
            if (h) {
                const uint32_t pos = atomicAdd(&P.cnt[b], h), c = SHIFTED ? bin_room(P, b) : P.cap[b];
                dst[b] = make_uint2((SHIFTED ? bin_off(P, b) : P.binoff[b]) + pos - run, run + (c > pos ? c - pos : 0u));
            }
            hist[b] = 0;
            run += h;
        }
        __syncthreads();
        // scatter into plane order
#pragma unroll
        for (int e = 0; e < E; e++) {
            if (tag[e] == 0xFFFFFFFFu) continue;
            const uint32_t b = tag[e] >> 16;
            sent[offs[b] + (tag[e] & 0xFFFFu)] = ((unsigned long long)b << 32) | key[e];
        }
        load_tile(t + gridDim.x, nps, npt);
#pragma unroll
        for (uint32_t q = 0; q < kHeldReservations; q++) {
            const uint32_t b = b0 + q;
            if (b < b1)
                dst[b] = make_uint2(roff[q] + res[q] - rrun[q], rrun[q] + (rcap[q] > res[q] ? rcap[q] - res[q] : 0u));
        }
        __syncthreads();
        // write-out: sorted entry q of plane b goes to bins[dst[b].x + q]
        // while its bin has room (plain stores: a plane's run is a fraction
        // of a line, and the line is completed by other tiles; streaming
        // stores would push the partial lines to DRAM several times over)
        const uint32_t nent = cnt * DIRS;
#pragma unroll 4
        for (uint32_t q = threadIdx.x; q < nent; q += blockDim.x) {
            const unsigned long long ent = sent[q];
            const uint32_t b = (uint32_t)(ent >> 32);
            const uint2 d = dst[b];
            if (q < d.y) P.bins[(uint32_t)(d.x + q)] = (uint32_t)ent;
            else set_key_bits<DIRS>(G, P, b, (uint32_t)ent);
        }
    }
    // the last block: apply units of the bins' actual contents
    if (!last_block(&P.ctl[0], &s_last)) return;
    const uint32_t U = P.unit;
    block_scan(NB, [&](uint32_t i) { return (min(__ldcg(&P.cnt[i]), SHIFTED ? bin_room(P, i) : P.cap[i]) + U - 1u) / U; },
               [&](uint32_t i, uint32_t v) { P.unit_start[i] = v; }, s_warp);
    if (threadIdx.x == 0) {
        P.ctl[0] = 0;
        P.ctl[1] = 0;
    }
}

// ------------------------------------------------------------------ apply
template <int R>
__device__ __forceinline__ void apply_key(uint32_t *pl, const Geometry &G, uint32_t A0, uint32_t rw, uint32_t key) {
    const uint32_t c0 = dh0(A0, G.k, key);
    atomicOr(&pl[c0 >> 5], 1u << (c0 & 31u));
#pragma unroll
    for (int i = 1; i < R; i++) {
        const uint32_t ci = dh_row(G, (uint32_t)i, key, c0);
        atomicOr(&pl[(uint32_t)i * rw + (ci >> 5)], 1u << (ci & 31u));
    }
}

// With two plane buffers (nbuf = 2, where two planes fit the block's shared
// memory) a unit is applied in one buffer while the bulk reduction of the
// previous unit still reads the other; before a buffer is reused, its
// reduction must have finished reading it (wait_group.read allows one
// reduction, the other buffer's, to stay in flight).  Planes too large for
// two buffers leave one block per SM, which then runs 1024 threads.
template <int R, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_plane_apply(Geometry G, PlaneArgs P, uint32_t nbuf, uint32_t per_block) {
    extern __shared__ uint4 pl4_all[];  // nbuf planes of ps words
    __shared__ uint4 s_unit[kApplyUnitsPerBlock];  // (plane, first entry, entries, -) of the block's units
    __shared__ uint32_t s_warp[32];
    __shared__ bool s_last;
    const uint32_t NB = P.nbins;
    const uint32_t rw = (1u << G.k) >> 5;
    // a block takes per_block consecutive units (the grid holds enough
    // blocks for every unit), so that blocks retire as the round
    // proceeds and other streams' work (a window close) gets SMs in between.
    // Their planes are found at once: every thread looks at its planes'
    // ranges of units, one L2 round trip instead of a search of ten for each
    // unit (2^26 pairs of the core sketch: 270 us, 280 with searches and a
    // shared unit counter; 128 KiB planes, one block per SM: 345 and 362).
    const uint32_t x0 = blockIdx.x * per_block;
    wait_for_previous();
    const uint32_t total = P.unit_start[NB];
    for (uint32_t b = threadIdx.x; b < NB; b += THREADS) {
        const uint32_t u0 = P.unit_start[b], u1 = P.unit_start[b + 1];
        if (u1 <= x0 || u0 >= x0 + per_block) continue;
        const uint32_t off = bin_off(P, b), n = min(P.cnt[b], bin_room(P, b));
#pragma unroll
        for (uint32_t j = 0; j < kApplyUnitsPerBlock; j++) {
            const uint32_t x = x0 + j;
            if (j >= per_block || x < u0 || x >= u1) continue;
            const uint32_t at = (x - u0) * P.unit;
            s_unit[j] = make_uint4(b, off + at, n - at < P.unit ? n - at : P.unit, 0u);
        }
    }
    for (uint32_t it = 0; it < per_block && x0 + it < total; it++) {
        uint4 *pl4 = pl4_all + (size_t)(it % nbuf) * (P.ps / 4);
        uint32_t *pl = reinterpret_cast<uint32_t *>(pl4);
        if (threadIdx.x == 0) {
            if (nbuf == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        __syncthreads();  // this buffer is free again; the units are known
        const uint4 unit = s_unit[it];
        const uint32_t b = unit.x, beg = unit.y, end = beg + unit.z;
        const uint32_t A0 = (b >> G.lg) ? G.h[1].A0 : G.h[0].A0;
        for (uint32_t i = threadIdx.x; i < P.ps / 4; i += blockDim.x) pl4[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        const uint4 *e4 = reinterpret_cast<const uint4 *>(P.bins + beg);  // beg is a multiple of 4
        const uint32_t n4 = (end - beg) / 4;
        uint32_t q = threadIdx.x;
        for (; q + 3 * blockDim.x < n4; q += 4 * blockDim.x) {
            uint4 v[4];
#pragma unroll
            for (int j = 0; j < 4; j++) v[j] = ld_previous_v4(e4 + q + j * blockDim.x);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                apply_key<R>(pl, G, A0, rw, v[j].x); apply_key<R>(pl, G, A0, rw, v[j].y);
                apply_key<R>(pl, G, A0, rw, v[j].z); apply_key<R>(pl, G, A0, rw, v[j].w);
            }
        }
        for (; q < n4; q += blockDim.x) {
            const uint4 a = ld_previous_v4(e4 + q);
            apply_key<R>(pl, G, A0, rw, a.x); apply_key<R>(pl, G, A0, rw, a.y);
            apply_key<R>(pl, G, A0, rw, a.z); apply_key<R>(pl, G, A0, rw, a.w);
        }
        for (uint32_t r = beg + 4 * n4 + threadIdx.x; r < end; r += blockDim.x)
            apply_key<R>(pl, G, A0, rw, __ldcg(P.bins + r));
        __syncthreads();
        if (threadIdx.x == 0) {
            // the plane's bits into the plane-major DHLA copy, ORed in L2
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.or.b32 [%0], [%1], %2;"
                         ::"l"(P.planes + (uint64_t)b * P.ps), "r"((uint32_t)__cvta_generic_to_shared(pl)),
                         "r"(P.ps * 4u)
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    // (shared memory must outlive the reductions' reads; the reductions
    // themselves are complete when the kernel is: what reads the plane copy
    // next is a plain launch, and must stay one)
    if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    // the last block: the next round's bins from this round's counts
    if (!last_block(&P.ctl[1], &s_last)) return;
    write_layout(P, true, s_warp);
}

// ----------------------------------------------------------------- direct
// A short round: every key's bits ORed into the plane copy where they lie,
// one pair per thread, with no bins and no planes in shared memory.  Bound
// by the L2's random reductions; the binned round's floor is the sweep of
// the whole plane copy through shared memory, whatever the pairs.
//
// Reductions of one word are taken one after another, so the packets of one
// flow must not each bring theirs: of the equal pairs of a block's tile one is
// set.  Each thread writes its number to the slot of its pair's hash, and
// skips the pair when the slot then names another thread with an equal one
// (a slot taken by a different pair lets all of the others through: with
// 2048 slots, one block in twenty).  2^19 pairs, none, a fifth and half of
// them one interleaved flow: tiny sketch 24, 22 and 19 us (every pair set but
// a repeat of the one before it: 24, 121 and 179), core sketch 33, 29 and 24
// (35, 93 and 129), 256 MiB copy 36, 35 and 31 (37, 210 and 294).
template <int DIRS>
__global__ void __launch_bounds__(kDirectThreads)
k_plane_direct(const uint32_t *__restrict__ pairs, uint64_t n, Geometry G, PlaneArgs P) {
    __shared__ uint2 s_pair[kDirectThreads];
    __shared__ uint8_t s_slot[kDirectSlots];
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const bool pair8 = ((uintptr_t)pairs & 7u) == 0;
    for (uint64_t p0 = (uint64_t)blockIdx.x * blockDim.x; p0 < n; p0 += stride) {
        const uint64_t p = p0 + threadIdx.x;
        const bool ok = p < n;
        uint2 v = make_uint2(0u, 0u);
        if (ok && pair8) {
            v = __ldg(reinterpret_cast<const uint2 *>(pairs) + p);
        } else if (ok) {
            v.x = ld_stream_u32(pairs + 2 * p);
            v.y = ld_stream_u32(pairs + 2 * p + 1);
        }
        const uint32_t slot = (v.x * 0x9E3779B1u + v.y * 0x85EBCA6Bu) / (uint32_t)((1ull << 32) / kDirectSlots);
        __syncthreads();  // the previous tile's look-ups are done
        s_pair[threadIdx.x] = v;
        if (ok) s_slot[slot] = (uint8_t)threadIdx.x;
        __syncthreads();
        const uint32_t first = s_slot[slot];
        const uint2 f = s_pair[first];
        if (!ok || (first != threadIdx.x && f.x == v.x && f.y == v.y)) continue;
        set_key_bits<DIRS>(G, P, h1v(G.h[0].A1, G.h[0].B1, G.lg, v.y), v.x);
        if (DIRS == 2) set_key_bits<DIRS>(G, P, G.g + h1v(G.h[1].A1, G.h[1].B1, G.lg, v.x), v.y);
    }
}

cudaError_t launch_plane_direct(const uint32_t *pairs, uint64_t n, const Geometry &G, const PlaneArgs &P, int num_sms,
                                cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    auto kern = G.dirs == 2 ? k_plane_direct<2> : k_plane_direct<1>;
    uint64_t blocks = (n + kDirectThreads - 1) / kDirectThreads;
    if (blocks > (uint64_t)num_sms * 32) blocks = (uint64_t)num_sms * 32;
    kern<<<(unsigned)blocks, kDirectThreads, 0, s>>>(pairs, n, G, P);
    return cudaGetLastError();
}

// --------------------------------------------------------------- launchers
size_t plane_bin_smem_bytes(uint32_t tile_pairs, uint32_t dirs, uint32_t nbins) {
    return (size_t)dirs * tile_pairs * 8 + (size_t)nbins * 16;
}

template <int DIRS, int PPT, int THREADS>
static cudaError_t launch_plane_bin(const uint32_t *pairs, uint64_t n, const Geometry &G, const PlaneArgs &P,
                                    uint32_t head, int num_sms, cudaStream_t s) {
    auto kern = P.shift ? k_plane_bin<DIRS, PPT, THREADS, true> : k_plane_bin<DIRS, PPT, THREADS, false>;
    const size_t smem = plane_bin_smem_bytes(P.tile_pairs, DIRS, P.nbins);
    int per_sm = 0;
    cudaError_t e = prepare_launch(reinterpret_cast<const void *>(kern), THREADS, smem, &per_sm);
    if (e != cudaSuccess) return e;
    // about kBinTilesPerBlock tiles per block (not one persistent block per
    // SM), so that blocks retire as the round proceeds and other streams'
    // work gets SMs in between.  A round of few waves of tiles is cut into as
    // many equal ones instead, so that the last wave is not half empty
    // (4,000,000 pairs are 3.2 waves of full tiles: 34 us, 35 with those).
    const uint64_t resident = (uint64_t)num_sms * per_sm;
    uint32_t tile = P.tile_pairs;
    uint64_t tiles = (n + tile - 1) / tile;
    uint64_t blocks = (tiles + kBinTilesPerBlock - 1) / kBinTilesPerBlock;
    if (blocks < resident) {
        const uint64_t waves = (tiles + resident - 1) / resident;
        const uint64_t even = (n + waves * resident - 1) / (waves * resident);
        if (even + 1 < tile) tile = (uint32_t)((even + 1) & ~1ull);
        tiles = (n + tile - 1) / tile;
        blocks = resident;
    }
    if (tiles < blocks) blocks = tiles;
    kern<<<(unsigned)blocks, THREADS, smem, s>>>(pairs, n, G, P, head, tile);
    return cudaGetLastError();
}

// tiles of 1024 to 4096 pairs: 512 threads with 2, 4 or 8 pairs each;
// 8192: 1024 threads with 8 each (one block per SM)
template <int DIRS>
static cudaError_t launch_plane_bin_d(const uint32_t *pairs, uint64_t n, const Geometry &G, const PlaneArgs &P,
                                      uint32_t head, int num_sms, cudaStream_t s) {
    switch (P.tile_pairs) {
        case 1024: return launch_plane_bin<DIRS, 2, 512>(pairs, n, G, P, head, num_sms, s);
        case 2048: return launch_plane_bin<DIRS, 4, 512>(pairs, n, G, P, head, num_sms, s);
        case 4096: return launch_plane_bin<DIRS, 8, 512>(pairs, n, G, P, head, num_sms, s);
        case 8192: return launch_plane_bin<DIRS, 8, 1024>(pairs, n, G, P, head, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}

template <int R>
static cudaError_t launch_plane_apply(const Geometry &G, const PlaneArgs &P, uint64_t n, int num_sms,
                                     cudaStream_t s, bool lanes) {
    // two plane buffers of 512 threads where they fit; one plane of 1024
    // threads per block beyond that
    const bool two = (size_t)P.ps * 8 <= (size_t)100 * 1024;
    auto kern = two ? k_plane_apply<R, kApplyThreads> : k_plane_apply<R, 2 * kApplyThreads>;
    const uint32_t threads = two ? kApplyThreads : 2 * kApplyThreads;
    const size_t plane = (size_t)P.ps * 4;
    int per_sm = 0;
    cudaError_t e = prepare_launch(reinterpret_cast<const void *>(kern), (int)threads, two ? 2 * plane : plane, &per_sm);
    if (e != cudaSuccess) return e;
    // units of the round: at most (keys + slack) / unit + one partial unit per plane
    const uint64_t keys = (uint64_t)(P.nbins / G.g) * n;
    const uint64_t most = (keys + keys / 8 + 40ull * P.nbins) / P.unit + P.nbins;
    // kApplyUnitsPerBlock of them per block, fewer in a round too short for
    // two waves of such blocks; a block of one unit needs one buffer
    const uint64_t waves = most / ((uint64_t)num_sms * per_sm * 2);
    const uint64_t per_block = waves < 1 ? 1 : (waves < kApplyUnitsPerBlock ? waves : kApplyUnitsPerBlock);
    const uint32_t nbuf = two && per_block > 1 ? 2u : 1u;
    const uint64_t blocks = (most + per_block - 1) / per_block;
    if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    uint32_t nb = nbuf, pb = (uint32_t)per_block;
    void *args[] = {const_cast<Geometry *>(&G), const_cast<PlaneArgs *>(&P), &nb, &pb};
    // Narrow planes: a unit's atomics meet on few words, and its block wants an
    // SM of its own.  Set up beside k_plane_bin's blocks, several land on one
    // (700,001 pairs in two directions, update alone: 64-word planes 96 us as
    // dependents and 46 plain, 192 words 45 and 35; 512 words 34 and 36, 8192
    // words 42 and 42, 2^21 pairs 54 and 56).  On the lanes of a batch, blocks
    // that wait for their own lane's binning keep another lane's off the SM
    // (64 core sketches of 500,000 pairs 1.59 ms as dependents, 1.51 plain).
    if (lanes || P.ps < kDependentPlaneWords)
        return cudaLaunchKernel(reinterpret_cast<const void *>(kern), dim3((unsigned)blocks), dim3(threads), args,
                                plane * nbuf, s);
    return launch_dependent(reinterpret_cast<const void *>(kern), dim3((unsigned)blocks), dim3(threads), plane * nbuf, s,
                            args);
}

cudaError_t launch_plane_round(const uint32_t *pairs, uint64_t n, const Geometry &G, const PlaneArgs &P, int num_sms,
                               cudaStream_t s, PlaneLayout layout, uint64_t prev_pairs, bool lanes) {
    if (n == 0) return cudaSuccess;
    // pairs that start 8 bytes past a 16-byte boundary: the first one is set
    // directly, the rest is read in 16-byte loads (4,000,000 of them: bin 35
    // us where 4-byte loads took 40)
    const uint32_t head = ((uintptr_t)pairs & 15u) == 8 && n > 1 ? 1u : 0u;
    pairs += 2 * head;
    n -= head;
    if (layout == kLayoutScale) {
        if (prev_pairs == 0) return cudaErrorInvalidValue;
        k_plane_layout<<<1, 1024, 0, s>>>(P, n, prev_pairs);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    } else if (layout == kLayoutCount) {
        auto kern = G.dirs == 2 ? k_plane_count<2> : k_plane_count<1>;
        const size_t smem = (size_t)P.nbins * 4;
        int per_sm = 0;
        cudaError_t e = prepare_launch(reinterpret_cast<const void *>(kern), (int)kPlaneThreads, smem, &per_sm);
        if (e != cudaSuccess) return e;
        uint64_t blocks = (uint64_t)num_sms * per_sm;
        const uint64_t need = (n / 2 + kPlaneThreads - 1) / kPlaneThreads;
        if (need < blocks) blocks = need ? need : 1;
        kern<<<(unsigned)blocks, kPlaneThreads, smem, s>>>(pairs, n, G, P);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    cudaError_t e = G.dirs == 2 ? launch_plane_bin_d<2>(pairs, n, G, P, head, num_sms, s)
                                : launch_plane_bin_d<1>(pairs, n, G, P, head, num_sms, s);
    if (e != cudaSuccess) return e;
    switch (G.r) {
        case 3: return launch_plane_apply<3>(G, P, n, num_sms, s, lanes);
        case 4: return launch_plane_apply<4>(G, P, n, num_sms, s, lanes);
        case 5: return launch_plane_apply<5>(G, P, n, num_sms, s, lanes);
        case 6: return launch_plane_apply<6>(G, P, n, num_sms, s, lanes);
        case 7: return launch_plane_apply<7>(G, P, n, num_sms, s, lanes);
        case 8: return launch_plane_apply<8>(G, P, n, num_sms, s, lanes);
        default: return cudaErrorInvalidValue;
    }
}


}  // namespace sd
