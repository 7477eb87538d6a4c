// sd_close.cu -- the window-close path (Algorithm 2 and the estimation step
// of §4.2) on the GPU.
//
//   k_row_stats   z_0 = g - popcount for every estimator, ZR(i) per row, the
//                 hot bitmap of each row (z_0 <= zhot, i.e. z_0 < Zmin) and
//                 |HE(i)|.
//   k_compact     sorted lists HE(0) and HE(1) (all HE(i) for the staged
//                 join of sd_join.cu) from their bitmaps.
//   k_restore     the candidate set K = {a : DH_i(a) in HE(i) for all i},
//                 and SZ(a) from ULE(a) = AND of a's r estimators (16-byte
//                 chunks, several candidates per warp), keeping (a, SZ) when
//                 SZ <= szmax.
//   k_close_finish  each direction's hits ordered by address, with the
//                 counters, into host memory.
//   k_estimate, k_sort_small  SZ of a K made by the staged join, and its hits
//                 ordered (bitonic, smem).
//   k_ss_*        the same for up to 2^19 hits: a sample sort (splitters
//                 from a sorted sample, keys scattered to buckets, each
//                 bucket sorted by one block).
//   k_sort_segments + k_merge_rank  longer lists, or a sample sort that fell
//                 short: sorted 2048-key segments, then pairwise merges.
//   k_reset       clears the DHLA and the per-window counters.
//   k_merge_or    dst |= src over whole DHLAs (multi-monitor merge).
//   k_*_many      the same kernels over an array of windows of one shape
//                 (sd_close_many): one launch per phase for all of them.
//
// Restore.  The paper's GPU restore (Algorithms 3 and 4) joins HE(0) x HE(1)
// x HE(2) and extends the surviving partial addresses row by row.  Here the
// join stops after HE(0) x HE(1): with c0 = DH_0(a) and c1 = DH_1(a),
// L = c0 xor c1 is the low k bits of a (Eq. 3 for i = 1), and because
// DH_0(a) = (A0 a mod 2^32) >> (32-k) with A0 odd, the remaining 32-k high
// bits H of a follow from c0 by one multiplication with A0^-1:
//   write A0*L mod 2^32 = Qh*2^k + Ql; then A0*a mod 2^32 = u*2^k + Ql with
//   u = (A0*H + Qh) mod 2^(32-k), and DH_0(a) = c0 fixes u:
//     k >= 16: u = c0 >> (2k-32), provided (Ql >> (32-k)) equals the low
//              2k-32 bits of c0 (otherwise no a exists);
//     k <  16: u = (c0 << (32-2k)) | t for each t < 2^(32-2k).
//   H = A0^-1 (u - Qh) mod 2^(32-k),  a = H*2^k + L.
// Each a found this way has DH_0(a) = c0 and DH_1(a) = c1 by construction and
// is kept when DH_i(a) is hot for i = 2..r-1: exactly K.  The work is
// |HE(0)|*|HE(1)|*2^max(0,32-2k) cheap integer tests instead of a join whose
// intermediate lists grow with |HE|^3.
#include <algorithm>

#include "sd_common.cuh"

namespace sd {

__device__ __forceinline__ uint32_t warp_sum(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// ------------------------------------------------------------- row stats
// One thread per estimator; a warp covers 32 consecutive estimators of one
// row (2^k >= 32 because (r-1)k >= (r-2)alpha + k >= 32 with r <= 8).
__device__ __forceinline__ void row_stats_body(const uint32_t *__restrict__ grid, const Geometry &G, int zhot,
                                               uint32_t *__restrict__ hotmap, StatBlock *__restrict__ st,
                                               uint32_t bx, uint32_t nbx) {
    __shared__ unsigned long long s_zr[2 * kMaxRows];
    __shared__ unsigned s_nhot[2 * kMaxRows];
    if (threadIdx.x < 2 * kMaxRows) {
        s_zr[threadIdx.x] = 0;
        s_nhot[threadIdx.x] = 0;
    }
    __syncthreads();
    const uint64_t ncell = (uint64_t)G.dirs * G.r << G.k;
    const uint64_t stride = (uint64_t)nbx * blockDim.x;
    const uint32_t lane = threadIdx.x & 31u;
    for (uint64_t q = (uint64_t)bx * blockDim.x + threadIdx.x; q < ncell; q += stride) {
        const uint32_t *cell = grid + q * G.wpc;
        uint32_t pop = 0;
        if ((G.wpc & 3u) == 0) {
            const uint4 *c4 = reinterpret_cast<const uint4 *>(cell);
            for (uint32_t w = 0; w < G.wpc / 4; w++) {
                const uint4 v = __ldg(c4 + w);
                pop += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            }
        } else {
            for (uint32_t w = 0; w < G.wpc; w++) pop += __popc(__ldg(cell + w));
        }
        const uint32_t z0 = G.g - pop;
        const unsigned hot = __ballot_sync(0xFFFFFFFFu, (int)z0 <= zhot);
        const uint32_t zsum = warp_sum(z0);
        if (lane == 0) {
            const uint32_t row = (uint32_t)(q >> G.k);  // dir * r + i
            hotmap[q >> 5] = hot;
            atomicAdd(&s_zr[row], (unsigned long long)zsum);
            atomicAdd(&s_nhot[row], (unsigned)__popc(hot));
        }
    }
    __syncthreads();
    // one global atomic per block and row
    for (uint32_t row = threadIdx.x; row < G.dirs * G.r; row += blockDim.x) {
        const uint32_t d = row / G.r, i = row % G.r;
        if (s_zr[row]) atomicAdd(&st->zr[d][i], s_zr[row]);
        if (s_nhot[row]) atomicAdd(&st->nhot[d][i], s_nhot[row]);
    }
}

__global__ void __launch_bounds__(256)
k_row_stats(const uint32_t *__restrict__ grid, Geometry G, int zhot, uint32_t *__restrict__ hotmap,
            StatBlock *__restrict__ st) {
    row_stats_body(grid, G, zhot, hotmap, st, blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------- compact
// One block per (dir, row in {0, 1}): HE(row) in ascending order.
__device__ __forceinline__ void compact_body(const uint32_t *__restrict__ hotmap, const Geometry &G,
                                             uint32_t *__restrict__ he, uint32_t rows, uint32_t bx) {
    const uint32_t dir = bx / rows, row = bx % rows;
    const uint32_t nw = (1u << G.k) >> 5;
    const uint32_t *bm = hotmap + ((uint64_t)dir * G.r + row) * nw;
    uint32_t *out = he + ((uint64_t)dir * rows + row) * (1ull << G.k);
    const uint32_t per = (nw + blockDim.x - 1) / blockDim.x;
    const uint32_t w0 = threadIdx.x * per;
    const uint32_t w1 = min(w0 + per, nw);
    uint32_t cnt = 0;
    for (uint32_t w = w0; w < w1; w++) cnt += __popc(bm[w]);
    // block exclusive scan of cnt
    __shared__ uint32_t warp_tot[32];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += v;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const uint32_t nwarps = blockDim.x >> 5;
        uint32_t t = lane < nwarps ? warp_tot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, t, o);
            if ((int)lane >= o) t += v;
        }
        if (lane < nwarps) warp_tot[lane] = t;  // inclusive over warps
    }
    __syncthreads();
    uint32_t pos = incl - cnt + (wid ? warp_tot[wid - 1] : 0);
    for (uint32_t w = w0; w < w1; w++) {
        uint32_t b = bm[w];
        while (b) {
            const uint32_t bit = __ffs(b) - 1;
            b &= b - 1u;
            out[pos++] = (w << 5) | bit;
        }
    }
}

__global__ void __launch_bounds__(1024)
k_compact(const uint32_t *__restrict__ hotmap, Geometry G, uint32_t *__restrict__ he, uint32_t rows) {
    compact_body(hotmap, G, he, rows, blockIdx.x);
}

// ---------------------------------------------------------------- restore
constexpr uint32_t kRestoreTileMax = 256;  // c0 values per k_restore tile

// Per-warp output buffers of the restore: candidates and hits are reserved
// in the global lists 32 or more at a time (one atomic per flush instead of
// one per finding warp, which serialised on the two counters).
constexpr int kWarpBuf = 64;

__device__ __forceinline__ void flush_hits(const RestoreArgs &A, uint32_t dir, unsigned long long *hbuf,
                                           uint32_t &hcount, uint32_t lane) {
    if (hcount == 0) return;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&A.stats->nhits[dir], (unsigned long long)hcount);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (uint32_t q = lane; q < hcount; q += 32)
        if (base + q < A.hits_cap) A.hits[(uint64_t)dir * A.hits_cap + base + q] = hbuf[q];
    hcount = 0;
    __syncwarp();
}

// SZ of n <= kWarpBuf candidates in x[] (shared memory) by one warp: the zero
// bits of ULE(a), the AND of a's r estimators; those with SZ <= szmax go to
// the hit list.  lpc lanes per candidate, each ANDing 16-byte chunks (4-byte
// words for g < 128) of the r estimators.
__device__ __forceinline__ void estimate_warp(const Geometry &G, const RestoreArgs &A, uint32_t dir, int szmax,
                                              const uint32_t *x_of, uint32_t n, unsigned long long *hbuf,
                                              uint32_t lane) {
    const uint32_t A0 = dir ? G.h[1].A0 : G.h[0].A0;
    const uint32_t *gdir = A.grid + (uint64_t)dir * G.dir_words;
    const uint32_t kmask = (1u << G.k) - 1u;
    const bool wide = G.wpc >= 4;
    const uint32_t chunks = wide ? G.wpc >> 2 : G.wpc;
    const uint32_t lpc = chunks < 32u ? chunks : 32u;
    const uint32_t cpw = 32u / lpc, sub = lane / lpc, sl = lane % lpc;
    uint32_t hcount = 0;
    for (uint32_t q0 = 0; q0 < n; q0 += cpw) {
        const uint32_t q = q0 + sub;
        const bool ok = q < n;
        const uint32_t x = ok ? x_of[q] : 0u;
        const uint32_t c0 = dh0(A0, G.k, x);
        uint32_t ones = 0;
        if (ok) {
            for (uint32_t c = sl; c < chunks; c += lpc) {
                uint4 ule = make_uint4(~0u, wide ? ~0u : 0u, wide ? ~0u : 0u, wide ? ~0u : 0u);
#pragma unroll
                for (uint32_t i = 0; i < 8; i++) {
                    if (i >= G.r) break;
                    const uint32_t ci = i == 0 ? c0 : ((shr_clamp(x, (i - 1u) * G.alpha) & kmask) ^ c0);
                    const uint32_t *cell = gdir + (uint64_t)i * G.row_words + (uint64_t)ci * G.wpc;
                    if (wide) {
                        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(cell) + c);
                        ule.x &= v.x; ule.y &= v.y; ule.z &= v.z; ule.w &= v.w;
                    } else {
                        ule.x &= __ldcg(cell + c);
                    }
                }
                ones += __popc(ule.x) + __popc(ule.y) + __popc(ule.z) + __popc(ule.w);
            }
        }
        for (uint32_t o = lpc >> 1; o > 0; o >>= 1) ones += __shfl_xor_sync(0xFFFFFFFFu, ones, o);
        const bool hit = ok && sl == 0 && (int)(G.g - ones) <= szmax;
        const unsigned hb = __ballot_sync(0xFFFFFFFFu, hit);
        if (hit) hbuf[hcount + __popc(hb & ((1u << lane) - 1u))] = ((unsigned long long)x << 32) | (G.g - ones);
        hcount += __popc(hb);
    }
    __syncwarp();
    flush_hits(A, dir, hbuf, hcount, lane);
}

// A warp's buffered candidates to K, and their SZ and hits at once (the
// estimators are hot, so in the DHLA; the loads hide behind other warps'
// tests).  Hits of a direction whose K overflows are dropped by the host.
// Returns whether K has passed its capacity (with every slot of K taken).
__device__ __forceinline__ bool flush_cands(const Geometry &G, const RestoreArgs &A, uint32_t dir, int szmax,
                                            uint32_t *cbuf, unsigned long long *hbuf, uint32_t &ccount,
                                            uint32_t lane) {
    if (ccount == 0) return false;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&A.stats->ncand[dir], (unsigned long long)ccount);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (uint32_t q = lane; q < ccount; q += 32)
        if (base + q < A.cand_cap) A.cand[(uint64_t)dir * A.cand_cap + base + q] = cbuf[q];
    const bool over = base + ccount > A.cand_cap;
    if (!over) estimate_warp(G, A, dir, szmax, cbuf, ccount, hbuf, lane);
    ccount = 0;
    __syncwarp();
    return over;
}

// 32-bit load from shared memory at byte address `addr`.
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// How the high 32 - k bits of an address follow from (c0, c1): below k = 16
// each t < 2^(32-2k) is one, at 16 there is exactly one, above 16 at most one.
enum RestoreBits { kBelow16 = 0, kIs16 = 1, kAbove16 = 2 };

// What a test needs besides c0, c1 and t.
struct RestoreConsts {
    uint32_t k, kmask, lowbits, lowmask, ulog, A0, A0inv_k, nw, alpha;
    uint32_t hot2s;        // rows 2.. of the hot bitmap in shared memory (byte address)
    const uint32_t *hot2;  // and in global memory
};

// bit `ci` of row i (>= 2) of the hot bitmap
template <bool SMEM>
__device__ __forceinline__ uint32_t hot_bit(const RestoreConsts &C, uint32_t i, uint32_t ci) {
    const uint32_t w = SMEM ? lds_u32(C.hot2s + (i - 2u) * C.nw * 4u + ((ci >> 3) & ~3u))
                            : __ldcg(C.hot2 + (uint64_t)(i - 2u) * C.nw + (ci >> 5));
    return w >> (ci & 31u) & 1u;
}

// Whether a is hot in rows FROM .. R-1 (with k = 16 and a compile-time alpha
// the shifts and masks are constants).
template <int FROM, int R, int KM, int ALPHA, bool SMEM>
__device__ __forceinline__ bool rows_hot(const RestoreConsts &C, uint32_t a, uint32_t c0) {
    uint32_t found = 1u;
#pragma unroll
    for (int i = FROM; i < R; i++) {
        const uint32_t s = ALPHA ? (uint32_t)((i - 1) * ALPHA) : (uint32_t)(i - 1) * C.alpha;
        const uint32_t m = KM == kIs16 ? 0xFFFFu : C.kmask;
        const uint32_t ci = (ALPHA && s >= 32u ? 0u : (ALPHA ? (a >> (s & 31u)) : shr_clamp(a, s))) & m ^ c0;
        if (SMEM) found &= hot_bit<true>(C, i, ci);
        else if (found) found &= hot_bit<false>(C, i, ci);
    }
    return found;
}

// The first stage of one (c0, c1, t) test: a's low k bits are L = c0 ^ c1;
// its high 32 - k bits are A0^-1 (u - (A0 L >> k)) mod 2^(32-k), computed as
// one multiply by A0^-1 2^k, with u = c0 << (32-2k) | t below k = 16 and
// c0 >> (2k-32) from there on.  For k > 16 the low 2k - 32 bits of c0 must
// match the top bits of A0 L mod 2^k (one pair in 2^(2k-32) does); otherwise
// a's row 2 must be hot.
template <int R, int KM, int ALPHA, bool SMEM>
__device__ __forceinline__ bool restore_first(const RestoreConsts &C, uint32_t c0, uint32_t c1, uint32_t t,
                                              uint32_t &a) {
    const uint32_t L = c0 ^ c1;
    const uint32_t Q = C.A0 * L;
    if (KM == kIs16) a = C.A0inv_k * (c0 - (Q >> 16)) + L;
    else if (KM == kBelow16) a = C.A0inv_k * (((c0 << C.ulog) | t) - (Q >> C.k)) + L;
    else a = C.A0inv_k * ((c0 >> C.lowbits) - (Q >> C.k)) + L;
    if (KM == kAbove16) return ((Q & C.kmask) >> (32u - C.k)) == (c0 & C.lowmask);
    return rows_hot<2, 3, KM, ALPHA, SMEM>(C, a, c0);
}

// Per-warp buffers of a block's restore.
constexpr uint32_t kColumn = 16;  // survivors a lane may hold: two for each of kColumn / 2 c0 values
struct WarpBufs {
    uint32_t *column;          // [kColumn][32] a lane's addresses that passed the first stage
    uint32_t *cand;            // [kWarpBuf] members of K
    unsigned long long *hits;  // [kWarpBuf]
    uint32_t ncand;            // (the same in every lane)
    bool over;                 // K has passed its capacity: nothing more to find
};

// The tests of two (c1, t) items per thread against the tile's c0 values.
// Few pass the first stage, so a lane puts its survivors in a column of its
// own and the warp looks up the other rows for all columns after every eight
// c0 values.  Bound by instruction issue (65%).  Measured with the estimates
// that follow in the same launch, against all rows at once and a launch of
// its own for the estimates: core sketch, 18 M tests, 77,000 candidates 48 us
// (56 and the gap); k = 18, 168 M tests 307 us (598 + 15); 64 core sketches
// 90 us (108 + 25); a window with every estimator hot, where each warp stops
// as it sees K pass its capacity, close 1.1 ms less.
template <int R, int KM, int ALPHA, bool SMEM>
__device__ __forceinline__ void restore_x2(const Geometry &G, const RestoreArgs &A, const RestoreConsts &C,
                                           uint32_t dir, int szmax, const uint32_t *s_c0, uint32_t nc0, uint32_t c1a,
                                           uint32_t ta, bool va, uint32_t c1b, uint32_t tb, bool vb, WarpBufs &W,
                                           uint32_t lane) {
    const unsigned below = (1u << lane) - 1u;
    uint32_t *const col = W.column + lane;
    for (uint32_t q0 = 0; q0 < nc0 && !W.over; q0 += kColumn / 2) {
        const uint32_t q1 = min(q0 + kColumn / 2, nc0);
        uint32_t n = 0;
#pragma unroll 4
        for (uint32_t q = q0; q < q1; q++) {
            const uint32_t c0 = s_c0[q];  // same for the whole block
            uint32_t a;
            if (restore_first<R, KM, ALPHA, SMEM>(C, c0, c1a, ta, a) && va) col[32u * n++] = a;
            if (restore_first<R, KM, ALPHA, SMEM>(C, c0, c1b, tb, a) && vb) col[32u * n++] = a;
        }
        const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, n);
        for (uint32_t j = 0; j < most; j++) {
            const uint32_t a = j < n ? col[32u * j] : 0u;
            const bool in = j < n && rows_hot<KM == kAbove16 ? 2 : 3, R, KM, ALPHA, SMEM>(C, a, dh0(C.A0, C.k, a));
            const unsigned b = __ballot_sync(0xFFFFFFFFu, in);
            if (!b) continue;
            if (in) W.cand[W.ncand + __popc(b & below)] = a;
            W.ncand += __popc(b);
            __syncwarp();
            if (W.ncand >= 32 && flush_cands(G, A, dir, szmax, W.cand, W.hits, W.ncand, lane)) W.over = true;
        }
    }
}

// One direction's restore job as a block needs it.
struct RestoreDir {
    uint32_t n0, n1, tile0;
    int szmax;
};

constexpr uint32_t kRestoreThreads = 256;
constexpr uint32_t kRestoreItems = 2 * kRestoreThreads;  // (c1, t) items per tile

__host__ __device__ __forceinline__ uint32_t restore_ulog(const Geometry &G) {
    return G.k >= 16u ? 0u : 32u - 2u * G.k;
}
// c0 values per tile for `tests` tests in all: about tiles_per_block tiles
// for each of (up to) 8 blocks per SM, so that the last wave is short
__host__ __device__ __forceinline__ uint32_t restore_tile0(unsigned long long tests, uint32_t num_sms,
                                                           uint32_t tiles_per_block) {
    const unsigned long long per = tests / ((unsigned long long)num_sms * 8u * kRestoreThreads * tiles_per_block) + 1;
    return (uint32_t)(per < kRestoreTileMax ? per : kRestoreTileMax);
}
// (n1 <= 2^k items of 2^(32-2k) t: below 2^27; tiles: at most 2^31, as tile0
// grows with the tests up to 256)
__host__ __device__ __forceinline__ uint32_t restore_tiles(const Geometry &G, uint32_t n0, uint32_t n1,
                                                           uint32_t tile0) {
    if (!n0 || !n1) return 0;
    const uint32_t items = n1 << restore_ulog(G);
    return ((n0 + tile0 - 1) / tile0) * ((items + kRestoreItems - 1) / kRestoreItems);
}

// The tiles first, first + step, ... below stop of one direction (see
// restore_body), by one way of testing.  A tile's lists are loaded while the
// tile before it is tested.
template <int R, int KM, int ALPHA, bool SMEM>
__device__ __forceinline__ void restore_loop(const Geometry &G, const RestoreArgs &A, const RestoreConsts &C,
                                             uint32_t dir, const RestoreDir &D, uint32_t first, uint32_t stop,
                                             uint32_t step, WarpBufs &W, uint32_t (*s_c0)[kRestoreTileMax],
                                             bool *s_stop) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t *he0 = A.he + (uint64_t)dir * 2 * (1ull << G.k);
    const uint32_t *he1 = he0 + (1ull << G.k);
    const uint32_t J = D.n1 << C.ulog;
    const uint32_t nchunk = (J + kRestoreItems - 1) / kRestoreItems;
    // tile t covers c0 group t / nchunk and item chunk t % nchunk
    uint32_t t0 = first / nchunk, jc = first % nchunk;
    const uint32_t t0_step = step / nchunk, jc_step = step % nchunk, tm = (1u << C.ulog) - 1u;
    // the next tile's c1 values (two (c1, t) items per thread), its c0 value
    // of this thread, and whether K has passed its capacity: once it has, the
    // direction reports nothing but the overload, and the rest of its
    // enumeration is skipped (the same decision for the whole block; a warp
    // that sees it earlier, as it adds to K, skips the rest of its tile)
    uint32_t c1a = 0, c1b = 0, c0 = 0, ja = 0;
    unsigned long long nk = 0;
    auto load = [&]() {
        ja = jc * kRestoreItems + threadIdx.x;
        const uint32_t q = t0 * D.tile0 + threadIdx.x;
        c1a = ja < J ? __ldcg(he1 + (ja >> C.ulog)) : 0u;
        c1b = ja + kRestoreThreads < J ? __ldcg(he1 + ((ja + kRestoreThreads) >> C.ulog)) : 0u;
        c0 = threadIdx.x < D.tile0 && q < D.n0 ? __ldcg(he0 + q) : 0u;
        if (threadIdx.x == 0) nk = *reinterpret_cast<volatile unsigned long long *>(&A.stats->ncand[dir]);
    };
    load();
    uint32_t cur = 0;
    for (uint32_t t = first; t < stop;) {
        s_c0[cur][threadIdx.x] = c0;
        if (threadIdx.x == 0) s_stop[cur] = nk > A.cand_cap;
        __syncthreads();
        if (s_stop[cur]) break;
        const uint32_t nc0 = min(D.tile0, D.n0 - t0 * D.tile0);
        const uint32_t xa = c1a, xb = c1b, xj = ja;
        t += step < stop - t ? step : stop - t;  // (no wrap)
        t0 += t0_step;
        jc += jc_step;
        if (jc >= nchunk) {
            jc -= nchunk;
            t0++;
        }
        if (t < stop) load();
        restore_x2<R, KM, ALPHA, SMEM>(G, A, C, dir, D.szmax, s_c0[cur], nc0, xa, xj & tm, xj < J, xb,
                                       (xj + kRestoreThreads) & tm, xj + kRestoreThreads < J, W, lane);
        cur ^= 1u;
    }
    __syncwarp();
    flush_cands(G, A, dir, D.szmax, W.cand, W.hits, W.ncand, lane);
}

// Tiles t_begin, t_begin + t_step, ... below t_end of direction `dir`.
// `stage`: rows 2.. of the hot bitmap are copied to shared memory first
// (worth it for more than a few tests per thread), where they fit.
template <int R>
__device__ __forceinline__ void restore_body(const Geometry &G, const RestoreArgs &A, uint32_t dir, RestoreDir D,
                                             bool stage, uint32_t t_begin, uint32_t t_end, uint32_t t_step) {
    extern __shared__ uint4 smem4[];  // (filled in 16-byte words)
    uint32_t *const smem = reinterpret_cast<uint32_t *>(smem4);
    __shared__ unsigned long long s_hbuf[kRestoreThreads / 32][kWarpBuf];
    __shared__ uint32_t s_cbuf[kRestoreThreads / 32][kWarpBuf];
    __shared__ uint32_t s_column[kRestoreThreads / 32][kColumn * 32];
    __shared__ uint32_t s_c0[2][kRestoreTileMax];  // (kRestoreTileMax = kRestoreThreads)
    __shared__ bool s_stop[2];
    __syncthreads();  // shared memory may still be in use by a previous call
    const uint32_t ntiles = restore_tiles(G, D.n0, D.n1, D.tile0);
    const uint32_t t_stop = t_end < ntiles ? t_end : ntiles;
    if (t_begin >= t_stop) return;  // no tile of this direction for the block
    RestoreConsts C;
    C.k = G.k;
    C.kmask = (1u << G.k) - 1u;
    C.lowbits = G.k >= 16u ? 2u * G.k - 32u : 0u;
    C.lowmask = (1u << C.lowbits) - 1u;
    C.ulog = restore_ulog(G);
    C.A0 = dir ? G.h[1].A0 : G.h[0].A0;
    C.A0inv_k = (dir ? G.h[1].A0inv : G.h[0].A0inv) << G.k;
    C.nw = (1u << G.k) >> 5;
    C.alpha = G.alpha;
    C.hot2 = A.hotmap + ((uint64_t)dir * G.r + 2u) * C.nw;
    C.hot2s = (uint32_t)__cvta_generic_to_shared(smem);
    // kept in registers: the compiler would form them again from the kernel
    // parameters in every test
    asm volatile("" : "+r"(C.A0), "+r"(C.A0inv_k), "+r"(C.kmask), "+r"(C.lowbits), "+r"(C.lowmask), "+r"(C.k),
                      "+r"(C.hot2s), "+r"(C.ulog));
    if (stage) {
        const uint32_t words = (G.r - 2) * C.nw;
        if ((C.nw & 3u) == 0) {  // (rows of whole 16-byte words: k >= 7)
            uint4 *to = smem4;
            const uint4 *from = reinterpret_cast<const uint4 *>(C.hot2);
#pragma unroll 4
            for (uint32_t w = threadIdx.x; w < words / 4; w += kRestoreThreads) to[w] = __ldcg(from + w);
        } else {
            for (uint32_t w = threadIdx.x; w < words; w += kRestoreThreads) smem[w] = __ldcg(C.hot2 + w);
        }
    }
    const uint32_t wid = threadIdx.x >> 5;
    WarpBufs W{s_column[wid], s_cbuf[wid], s_hbuf[wid], 0u, false};
#define SD_RESTORE(KM, ALPHA, SMEM) \
    restore_loop<R, KM, ALPHA, SMEM>(G, A, C, dir, D, t_begin, t_stop, t_step, W, s_c0, s_stop)
    if (stage) {
        if (R == 4 && G.k == 16u && G.alpha == 8u) SD_RESTORE(kIs16, 8, true);  // the core-link sketch
        else if (G.k == 16u) SD_RESTORE(kIs16, 0, true);
        else if (G.k < 16u) SD_RESTORE(kBelow16, 0, true);
        else SD_RESTORE(kAbove16, 0, true);
    } else {
        if (G.k == 16u) SD_RESTORE(kIs16, 0, false);
        else if (G.k < 16u) SD_RESTORE(kBelow16, 0, false);
        else SD_RESTORE(kAbove16, 0, false);
    }
#undef SD_RESTORE
}

// Largest SZ that Eq. 4 may report, in float, from sum_ln = sum of
// ln(ZR(i) / (g 2^k)): (g - g psi^r) e^(-theta/g) (Eq. 4 solved for SZ; xfac
// is the exponential), raised by a hundredth, above the float's error (at most g r
// 1e-7, 0.004 for g = 4096 and r = 8).  The host recomputes it in double and drops the
// hits above its own, so the report does not depend on this rounding.
__device__ __forceinline__ int szmax_bound(const Geometry &G, float sum_ln, float xfac) {
    const float psi = -expm1f(sum_ln / (float)G.r);
    float pr = psi;
    for (uint32_t i = 1; i < G.r; i++) pr *= psi;
    return (int)fmaxf(0.0f, ((float)G.g - (float)G.g * pr) * xfac + 0.01f);
}

// The restore of a close whose row statistics the host has not seen: the
// directions that run (no saturated row, the work bound within pair_cap),
// the tiles and the SZ bound are worked out by every block from the
// StatBlock.  The tiles of direction 0, then those of direction 1, are dealt
// round-robin to the blocks.
template <int R>
__global__ void __launch_bounds__(kRestoreThreads, 4)
k_restore(const __grid_constant__ Geometry G, const __grid_constant__ RestoreArgs A, uint64_t pair_cap, float xfac,
          uint32_t num_sms) {
    __shared__ uint32_t s_n[2][2];
    __shared__ int s_szmax[2];
    dependents_may_start();
    wait_for_previous();
    if (threadIdx.x < 16) {  // eight lanes per direction, one row each
        const uint32_t d = threadIdx.x >> 3, i = threadIdx.x & 7u;
        const bool live = d < G.dirs && i < G.r;
        const unsigned long long zr = live ? A.stats->zr[d][i] : 1ull;
        uint32_t n0 = d < G.dirs ? A.stats->nhot[d][0] : 0u, n1 = d < G.dirs ? A.stats->nhot[d][1] : 0u;
        float ln = live ? logf((float)zr / ((float)G.g * (float)(1u << G.k))) : 0.0f;
        const bool sat = (__ballot_sync(0xFFFFu, zr == 0ull) >> (8u * d) & 0xFFu) != 0u;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) ln += __shfl_xor_sync(0xFFFFu, ln, o);
        if (sat || ((uint64_t)n0 << (32u - G.k)) > pair_cap) n0 = n1 = 0;
        if (i == 0) {
            const int szmax = n0 && n1 ? szmax_bound(G, ln, xfac) : 0;
            s_n[d][0] = n0;
            s_n[d][1] = n1;
            s_szmax[d] = szmax;
            if (blockIdx.x == 0) A.stats->szmax_used[d] = szmax;
        }
    }
    __syncthreads();
    const uint32_t ulog = restore_ulog(G);
    const unsigned long long tests = ((unsigned long long)s_n[0][0] * s_n[0][1] +
                                      (unsigned long long)s_n[1][0] * s_n[1][1]) << ulog;
    // staging the bitmap costs a block 3 to 4 us, a test looked up without it
    // an L2 round trip per row: stage from two tests per thread on
    const bool stage = A.smem_hot && tests > (unsigned long long)gridDim.x * kRestoreThreads * 2u;
    const uint32_t tile0 = restore_tile0(tests, num_sms, 4);
    uint32_t skip = 0;  // blocks that direction 0's tiles end on
    for (uint32_t d = 0; d < G.dirs; d++) {
        const RestoreDir D{s_n[d][0], s_n[d][1], tile0, s_szmax[d]};
        const uint32_t first = blockIdx.x >= skip ? blockIdx.x - skip : blockIdx.x + gridDim.x - skip;
        restore_body<R>(G, A, d, D, stage, first, 0xFFFFFFFFu, gridDim.x);
        skip = restore_tiles(G, D.n0, D.n1, D.tile0) % gridDim.x;
    }
}

// SZ and hits of a whole K in memory (the staged join's): warps take 32
// candidates at a time.  A direction whose K overflowed its capacity is
// skipped (it reports nothing).
__global__ void __launch_bounds__(256)
k_estimate(Geometry G, RestoreArgs A) {
    __shared__ unsigned long long s_hbuf[8][kWarpBuf];
    const uint32_t dir = blockIdx.y;
    if (!(dir ? A.run[1] : A.run[0])) return;
    const unsigned long long nk = A.stats->ncand[dir];
    if (nk > A.cand_cap) return;
    const uint32_t wid = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint64_t step = (uint64_t)gridDim.x * 8 * 32;
    for (uint64_t q = ((uint64_t)blockIdx.x * 8 + wid) * 32; q < nk; q += step)
        estimate_warp(G, A, dir, dir ? A.szmax[1] : A.szmax[0], A.cand + (uint64_t)dir * A.cand_cap + q,
                      (uint32_t)(nk - q < 32 ? nk - q : 32), s_hbuf[wid], lane);
}

// ------------------------------------------------------------------- sort
__device__ __forceinline__ void cswap(unsigned long long &a, unsigned long long &b, bool up) {
    if ((a > b) == up) {
        const unsigned long long t = a;
        a = b;
        b = t;
    }
}

// Bitonic sort of s[0, P) (P a power of two) by the whole block: each stage
// visits the P/2 compare-exchange pairs (i, i + j) directly.
__device__ __forceinline__ void bitonic_smem(unsigned long long *s, unsigned P) {
    for (unsigned kk = 2; kk <= P; kk <<= 1) {
        for (unsigned j = kk >> 1; j > 0; j >>= 1) {
            for (unsigned t = threadIdx.x; t < P / 2; t += blockDim.x) {
                const unsigned i = 2 * t - (t & (j - 1));  // low index of the t-th pair
                cswap(s[i], s[i + j], (i & kk) == 0);
            }
            __syncthreads();
        }
    }
}

// One block per direction: bitonic sort of up to kSortSmall hits in shared
// memory (padding with all-ones keys, which sort last).
__device__ __forceinline__ void sort_small_body(unsigned long long *hits, uint64_t hits_cap, StatBlock *st,
                                                uint32_t dir) {
    extern __shared__ unsigned long long s[];  // kSortSmall keys
    const unsigned long long n = st->nhits[dir];
    const unsigned long long nn = n < hits_cap ? n : hits_cap;
    if (nn > (unsigned long long)kSortSmall) {
        if (threadIdx.x == 0) st->big_sort[dir] = 1;
        return;
    }
    if (nn <= 1) return;
    unsigned P = 2;
    while (P < nn) P <<= 1;
    unsigned long long *hd = hits + (uint64_t)dir * hits_cap;
    for (unsigned i = threadIdx.x; i < P; i += blockDim.x) s[i] = i < nn ? hd[i] : ~0ull;
    __syncthreads();
    bitonic_smem(s, P);
    for (unsigned i = threadIdx.x; i < nn; i += blockDim.x) hd[i] = s[i];
}

__global__ void __launch_bounds__(1024)
k_sort_small(unsigned long long *hits, uint64_t hits_cap, StatBlock *st, uint2 run) {
    const uint32_t dir = blockIdx.x;
    if (!(dir ? run.y : run.x)) return;
    sort_small_body(hits, hits_cap, st, dir);
}

// The end of a queued close: each direction's hits ordered by address
// straight into pinned host memory, and the StatBlock after them.
//
// A list of n hits is cut at addresses: nb = n / 256 ranges, each sorted by
// one block.  Every block finds its two cuts by itself, as quantiles of the
// same sample of 2 or 4 hits per range, and reads the whole list: it keeps the
// hits of its range in shared memory and counts those below, which is where
// its part of the order begins.  So no block waits for another and one
// launch does it: 29,000 hits in 24 us and 2,400 in 12 us with cold caches,
// where the one-block sort and the sample sort's four launches took 42 and
// 23 us and a host round trip.  Within a block a hit's place is the number
// of smaller addresses (addresses are distinct).  A range with more than
// kRangeKeys hits, or a list of more than kFinishMax, sets big_sort: the
// host sorts it by the longer way.  A range of 2 or 4 sample gaps of 128 hits
// on average is that long in one list of 4,000 at 32,768 hits (reckoned) and
// one of 100 at 65,536 (16 of 1600 counted).  Twice the samples there take 62
// us instead of 39 for every such launch, more than the rare longer way.
constexpr uint32_t kFinishThreads = 1024;
constexpr uint32_t kFinishLoads = 4;       // 16-byte loads in flight per thread
constexpr uint32_t kFinishBlocks = 128;    // ranges at most
constexpr uint32_t kRangeKeys = 2048;

// number of u32 v[j] < x, j < n, v padded to a multiple of 4 with ~0
__device__ __forceinline__ uint32_t count_below(const uint32_t *v, uint32_t n, uint32_t x) {
    uint32_t c = 0;
    const uint4 *v4 = reinterpret_cast<const uint4 *>(v);
    for (uint32_t j = 0; j < (n + 3) / 4; j++) {
        const uint4 q = v4[j];
        c += (q.x < x) + (q.y < x) + (q.z < x) + (q.w < x);
    }
    return c;
}

__global__ void __launch_bounds__(kFinishThreads)
k_close_finish(const unsigned long long *hits, uint64_t hits_cap, StatBlock *st, unsigned long long *out,
               uint64_t out_cap, unsigned long long *spare, StatBlock *st_out) {
    __shared__ unsigned long long s_key[kRangeKeys];
    __shared__ __align__(16) uint32_t s_ip[kRangeKeys + 4];
    __shared__ uint32_t s_cut[2], s_n, s_below;
    __shared__ bool s_last;
    const uint32_t dir = blockIdx.y;
    wait_for_previous();
    const unsigned long long nh = st->nhits[dir];
    const bool fits = nh <= hits_cap && nh <= kFinishMax;
    const uint32_t n = fits ? (uint32_t)nh : 0u;
    uint32_t nb = (n + 255u) / 256u;
    if (nb > kFinishBlocks) nb = kFinishBlocks;
    // a list beyond the host's buffer is left in `spare` on the device
    const bool spared = n > out_cap;
    if ((!fits || spared) && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&st->big_sort[dir], fits ? 2u : 1u);
    if (blockIdx.x < nb) {
        const unsigned long long *h = hits + (uint64_t)dir * hits_cap;
        if (threadIdx.x == 0) {
            s_cut[0] = 0u;
            s_cut[1] = ~0u;
            s_n = 0;
            s_below = 0;
        }
        if (nb > 1) {
            // range b: addresses in [cut b, cut b + 1), cut j the (per j)-th
            // smallest of per nb samples (a range of 256 hits on average may
            // come out eight times as long, one of 512 four times)
            const uint32_t per = n <= 32768u ? 2u : 4u, m = per * nb;
            for (uint32_t i = threadIdx.x; i < ((m + 3u) & ~3u); i += kFinishThreads)
                s_ip[i] = i < m ? (uint32_t)(__ldcg(h + (uint64_t)i * n / m) >> 32) : ~0u;
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < m; i += kFinishThreads) {
                const uint32_t x = s_ip[i], rank = count_below(s_ip, m, x);
                if (rank == per * blockIdx.x && blockIdx.x > 0) s_cut[0] = x;
                if (rank == per * (blockIdx.x + 1)) s_cut[1] = x;
            }
        }
        __syncthreads();
        const uint32_t lo = s_cut[0], hi = s_cut[1];
        const bool tail = blockIdx.x + 1 == nb;  // the last range has no upper cut
        const uint32_t lane = threadIdx.x & 31u;
        uint32_t below = 0;
        // two hits per load (the lists start on 16 bytes and have room for an
        // even number)
        for (uint32_t i0 = 0; i0 < n; i0 += 2u * kFinishThreads * kFinishLoads) {
            uint4 v[kFinishLoads];
#pragma unroll
            for (uint32_t u = 0; u < kFinishLoads; u++) {
                const uint32_t i = i0 + 2u * (u * kFinishThreads + threadIdx.x);
                v[u] = i < n ? __ldcg(reinterpret_cast<const uint4 *>(h + i)) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (uint32_t u = 0; u < kFinishLoads; u++) {
                const uint32_t i = i0 + 2u * (u * kFinishThreads + threadIdx.x);
                const bool l0 = i < n, l1 = i + 1 < n;
                const bool in0 = l0 && v[u].y >= lo && (tail || v[u].y < hi);
                const bool in1 = l1 && v[u].w >= lo && (tail || v[u].w < hi);
                below += (uint32_t)(l0 && v[u].y < lo) + (uint32_t)(l1 && v[u].w < lo);
                if (in0 || in1) {
                    uint32_t at = atomicAdd(&s_n, (uint32_t)in0 + (uint32_t)in1);
                    if (in0 && at < kRangeKeys) s_key[at] = (unsigned long long)v[u].y << 32 | v[u].x;
                    at += in0;
                    if (in1 && at < kRangeKeys) s_key[at] = (unsigned long long)v[u].w << 32 | v[u].z;
                }
            }
        }
        below = warp_sum(below);
        if (lane == 0 && below) atomicAdd(&s_below, below);
        __syncthreads();
        const uint32_t cnt = s_n, first = s_below;
        if (cnt > kRangeKeys) {
            if (threadIdx.x == 0) atomicOr(&st->big_sort[dir], 1u);
        } else {
            for (uint32_t i = threadIdx.x; i < ((cnt + 3u) & ~3u); i += kFinishThreads)
                s_ip[i] = i < cnt ? (uint32_t)(s_key[i] >> 32) : ~0u;
            __syncthreads();
            unsigned long long key[kRangeKeys / kFinishThreads];
            uint32_t at[kRangeKeys / kFinishThreads];
#pragma unroll
            for (uint32_t u = 0; u < kRangeKeys / kFinishThreads; u++) {
                const uint32_t i = u * kFinishThreads + threadIdx.x;
                key[u] = i < cnt ? s_key[i] : 0ull;
                at[u] = i < cnt ? count_below(s_ip, cnt, (uint32_t)(key[u] >> 32)) : 0u;
            }
            __syncthreads();
#pragma unroll
            for (uint32_t u = 0; u < kRangeKeys / kFinishThreads; u++)
                if (u * kFinishThreads + threadIdx.x < cnt) s_key[at[u]] = key[u];
            __syncthreads();
            unsigned long long *o = (spared ? spare + (uint64_t)dir * hits_cap : out + (uint64_t)dir * out_cap) + first;
            for (uint32_t i = threadIdx.x; i < cnt; i += kFinishThreads) o[i] = s_key[i];
        }
    }
    // the last block: the StatBlock to the host, and zero for the next window
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&st->finish_done, 1u) == gridDim.x * gridDim.y - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const volatile uint32_t *from = reinterpret_cast<const volatile uint32_t *>(st);
    uint32_t *to = reinterpret_cast<uint32_t *>(st_out);
    uint32_t *clr = reinterpret_cast<uint32_t *>(st);
    for (uint32_t i = threadIdx.x; i < sizeof(StatBlock) / 4; i += kFinishThreads) {
        to[i] = from[i];
        clr[i] = 0;
    }
}

// Sort every segment keys[j*kSortSmall, (j+1)*kSortSmall) of keys[0, n) in
// shared memory (one block per segment, bitonic, padded with all-ones keys).
__global__ void __launch_bounds__(1024)
k_sort_segments(unsigned long long *keys, uint64_t n) {
    extern __shared__ unsigned long long s[];
    const uint64_t base = (uint64_t)blockIdx.x * kSortSmall;
    if (base >= n) return;
    const uint64_t left = n - base;
    const unsigned len = (unsigned)(left < (uint64_t)kSortSmall ? left : (uint64_t)kSortSmall);
    unsigned P = 1;
    while (P < len) P <<= 1;
    unsigned long long *kd = keys + base;
    for (unsigned i = threadIdx.x; i < P; i += blockDim.x) s[i] = i < len ? kd[i] : ~0ull;
    __syncthreads();
    bitonic_smem(s, P);
    for (unsigned i = threadIdx.x; i < len; i += blockDim.x) kd[i] = s[i];
}

// Merge neighbouring sorted runs of length L (the last may be shorter) from
// src into dst.  Keys are distinct, so an element's place in the merged run
// is its index in its own run plus the number of keys below it in the other
// run (a binary search): every element moves independently.
__global__ void k_merge_rank(const unsigned long long *__restrict__ src, unsigned long long *__restrict__ dst,
                             uint64_t n, uint64_t L) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t run = i / L;
        const uint64_t pb = (run & ~1ull) * L;
        const uint64_t a0 = pb, a1 = (pb + L < n) ? pb + L : n;
        const uint64_t b0 = a1, b1 = (pb + 2 * L < n) ? pb + 2 * L : n;
        const unsigned long long key = src[i];
        uint64_t lo, hi, own;
        if ((run & 1) == 0) {
            lo = b0; hi = b1; own = i - a0;
        } else {
            lo = a0; hi = a1; own = i - b0;
        }
        const uint64_t other0 = lo;
        while (lo < hi) {
            const uint64_t mid = lo + (hi - lo) / 2;
            if (src[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        dst[pb + own + (lo - other0)] = key;
    }
}

// Merge all sorted segments of 2048 keys at once: a key's place in the
// output is its index in its own segment plus, for every other segment, the
// number of keys below it there (keys are distinct).  One launch instead of
// log2(segments) pairwise passes, for a few dozen segments at most.
constexpr uint32_t kMergeAllMaxSegs = 32;

__global__ void k_merge_all(const unsigned long long *__restrict__ src, unsigned long long *__restrict__ dst,
                            uint64_t n) {
    const uint32_t nseg = (uint32_t)((n + kSortSmall - 1) / kSortSmall);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned long long key = src[i];
        const uint32_t own = (uint32_t)(i / kSortSmall);
        uint64_t pos = i - (uint64_t)own * kSortSmall;
        for (uint32_t t = 0; t < nseg; t++) {
            if (t == own) continue;
            uint64_t lo = (uint64_t)t * kSortSmall;
            uint64_t hi = lo + kSortSmall < n ? lo + kSortSmall : n;
            const uint64_t base = lo;
            while (lo < hi) {
                const uint64_t mid = lo + (hi - lo) / 2;
                if (src[mid] < key) lo = mid + 1;
                else hi = mid;
            }
            pos += lo - base;
        }
        dst[pos] = key;
    }
}

// ----------------------------------------------------- sample sort (big)
// Hit lists longer than kSortSmall: nb buckets (a power of two, about 128
// keys each, up to 1024 buckets) split by nb - 1 splitters taken from a
// sorted sample of `over` keys per bucket (evenly spaced positions: 2 per
// bucket of 128, 8 for larger buckets); every key goes to the bucket of the
// splitters around it, and each bucket is sorted by one block in shared
// memory.  A bucket beyond kSortSmall keys (a sample that did not represent
// the keys) raises *overflow, and the host sorts the list again by the
// merge path.  Keys are distinct.

// bucket of `key`: the number of splitters below it
__device__ __forceinline__ uint32_t bucket_of(const unsigned long long *spl, uint32_t nb, unsigned long long key) {
    uint32_t lo = 0, hi = nb - 1;  // splitters spl[0 .. nb-2]
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (spl[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// One block: sort the sample, write the splitters, clear the counters.
__global__ void __launch_bounds__(1024)
k_ss_splitters(const unsigned long long *__restrict__ keys, uint64_t n, uint32_t nb, uint32_t over, SampleSortArgs S) {
    extern __shared__ unsigned long long smp[];  // nb * over keys
    const uint32_t m = nb * over;
    for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) smp[i] = keys[((uint64_t)i * n) / m];
    for (uint32_t i = threadIdx.x; i <= nb; i += blockDim.x) {
        S.count[i] = 0;
        S.cursor[i] = 0;
    }
    if (threadIdx.x == 0) {
        S.ctl[0] = 0;  // count blocks done
        S.ctl[1] = 0;  // overflow
    }
    __syncthreads();
    if (m <= blockDim.x) {
        // a small sample: each thread places its key by counting the keys
        // below it (sample keys are distinct keys of the list)
        unsigned long long key = 0;
        uint32_t rank = 0;
        if (threadIdx.x < m) {
            key = smp[threadIdx.x];
            for (uint32_t j = 0; j < m; j++) rank += smp[j] < key;
        }
        __syncthreads();
        if (threadIdx.x < m) smp[rank] = key;
        __syncthreads();
    } else {
        bitonic_smem(smp, m);
    }
    for (uint32_t j = threadIdx.x; j + 1 < nb; j += blockDim.x) S.spl[j] = smp[(j + 1) * over - 1];
}

// Keys per bucket; the last block turns the counts into bucket offsets.
__global__ void __launch_bounds__(256)
k_ss_count(const unsigned long long *__restrict__ keys, uint64_t n, uint32_t nb, SampleSortArgs S) {
    __shared__ unsigned long long s_spl[kSampleMaxBuckets];
    __shared__ uint32_t s_hist[kSampleMaxBuckets];
    __shared__ bool s_last;
    for (uint32_t j = threadIdx.x; j < nb; j += blockDim.x) {
        if (j + 1 < nb) s_spl[j] = S.spl[j];
        s_hist[j] = 0;
    }
    __syncthreads();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        atomicAdd(&s_hist[bucket_of(s_spl, nb, keys[i])], 1u);
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < nb; j += blockDim.x)
        if (s_hist[j]) atomicAdd(&S.count[j], s_hist[j]);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&S.ctl[0], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // exclusive scan of the nb <= 1024 counts, 4 consecutive ones per thread
    __shared__ uint32_t s_w[8];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const uint32_t j0 = threadIdx.x * 4;
    uint32_t c[4], sum = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        c[q] = j0 + q < nb ? __ldcg(&S.count[j0 + q]) : 0u;
        sum += c[q];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += v;
    }
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
    for (uint32_t w = 0; w < wid; w++) run += s_w[w];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        if (j0 + q < nb) {
            S.off[j0 + q] = run;
            S.cursor[j0 + q] = run;
        }
        run += c[q];
    }
    if (j0 < nb && j0 + 4 >= nb) S.off[nb] = run;
}

// Every key to a free slot of its bucket in `out`: a block takes
// kScatterKeys keys per thread, ranks them per bucket in shared memory and
// reserves each bucket's run with one atomic.
constexpr uint32_t kScatterKeys = 4;
__global__ void __launch_bounds__(256)
k_ss_scatter(const unsigned long long *__restrict__ keys, unsigned long long *__restrict__ out, uint64_t n, uint32_t nb,
             SampleSortArgs S) {
    __shared__ unsigned long long s_spl[kSampleMaxBuckets];
    __shared__ uint32_t s_cnt[kSampleMaxBuckets];
    for (uint32_t j = threadIdx.x; j < nb; j += blockDim.x) {
        if (j + 1 < nb) s_spl[j] = S.spl[j];
        s_cnt[j] = 0;
    }
    __syncthreads();
    const uint64_t per_block = (uint64_t)blockDim.x * kScatterKeys;
    for (uint64_t base = (uint64_t)blockIdx.x * per_block; base < n; base += (uint64_t)gridDim.x * per_block) {
        unsigned long long key[kScatterKeys];
        uint32_t b[kScatterKeys], rank[kScatterKeys];
#pragma unroll
        for (uint32_t u = 0; u < kScatterKeys; u++) {
            const uint64_t i = base + (uint64_t)u * blockDim.x + threadIdx.x;
            b[u] = 0xFFFFFFFFu;
            if (i < n) {
                key[u] = keys[i];
                b[u] = bucket_of(s_spl, nb, key[u]);
                rank[u] = atomicAdd(&s_cnt[b[u]], 1u);
            }
        }
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < nb; j += blockDim.x) {
            const uint32_t c = s_cnt[j];
            s_cnt[j] = c ? atomicAdd(&S.cursor[j], c) : 0u;  // the run's first slot
        }
        __syncthreads();
#pragma unroll
        for (uint32_t u = 0; u < kScatterKeys; u++)
            if (b[u] != 0xFFFFFFFFu) out[s_cnt[b[u]] + rank[u]] = key[u];
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < nb; j += blockDim.x) s_cnt[j] = 0;
        __syncthreads();
    }
}

// One block per bucket: its keys of `in` sorted into the same places of
// `out` (up to 512 keys: each key placed by counting the keys below it;
// more: bitonic).
__global__ void __launch_bounds__(256)
k_ss_buckets(const unsigned long long *__restrict__ in, unsigned long long *__restrict__ out, SampleSortArgs S) {
    extern __shared__ unsigned long long s[];  // kSortSmall keys
    const uint32_t b = blockIdx.x;
    const uint32_t lo = S.off[b], len = S.off[b + 1] - lo;
    if (len > (uint32_t)kSortSmall) {
        if (threadIdx.x == 0) atomicOr(&S.ctl[1], 1u);
        return;
    }
    if (len == 0) return;
    if (len <= 512) {
        for (unsigned i = threadIdx.x; i < len; i += blockDim.x) s[i] = in[lo + i];
        __syncthreads();
        for (unsigned i = threadIdx.x; i < len; i += blockDim.x) {
            const unsigned long long key = s[i];
            uint32_t rank = 0;
            for (uint32_t j = 0; j < len; j++) rank += s[j] < key;
            out[lo + rank] = key;
        }
        return;
    }
    unsigned P = 1;
    while (P < len) P <<= 1;
    for (unsigned i = threadIdx.x; i < P; i += blockDim.x) s[i] = i < len ? in[lo + i] : ~0ull;
    __syncthreads();
    bitonic_smem(s, P);
    for (unsigned i = threadIdx.x; i < len; i += blockDim.x) out[lo + i] = s[i];
}

// ------------------------------------------------------------ reset/merge
__device__ __forceinline__ void reset_body(uint4 *grid4, uint64_t n4, StatBlock *st, uint32_t bx, uint32_t nbx) {
    const uint64_t stride = (uint64_t)nbx * blockDim.x;
    for (uint64_t i = (uint64_t)bx * blockDim.x + threadIdx.x; i < n4; i += stride)
        grid4[i] = make_uint4(0, 0, 0, 0);
    if (bx == 0) {
        uint32_t *w = reinterpret_cast<uint32_t *>(st);
        for (uint32_t i = threadIdx.x; i < sizeof(StatBlock) / 4; i += blockDim.x) w[i] = 0;
    }
}

__global__ void k_reset(uint4 *grid4, uint64_t n4, StatBlock *st) { reset_body(grid4, n4, st, blockIdx.x, gridDim.x); }

__global__ void k_merge_or(uint4 *dst, const uint4 *__restrict__ src, uint64_t n4) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        const uint4 a = dst[i], b = __ldg(src + i);
        dst[i] = make_uint4(a.x | b.x, a.y | b.y, a.z | b.z, a.w | b.w);
    }
}

// ------------------------------------------------------- batched closes
// The same kernels over an array of jobs, one grid dimension per job.
__global__ void __launch_bounds__(256) k_row_stats_many(const CloseJob *__restrict__ J) {
    const CloseJob &j = J[blockIdx.y];
    if (j.stats_done) return;  // the job's fold wrote its statistics
    row_stats_body(j.A.grid, j.G, j.zhot, const_cast<uint32_t *>(j.A.hotmap), j.A.stats, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(1024) k_compact_many(const CloseJob *__restrict__ J) {
    const CloseJob &j = J[blockIdx.y];
    if (j.stats_done == 2) return;  // listed by k_plane_scan
    compact_body(j.A.hotmap, j.G, const_cast<uint32_t *>(j.A.he), 2, blockIdx.x);
}

// Work of all (job, direction) segments laid end to end: segment s = 2 job +
// dir starts at base[s] (non-decreasing, base[2 count] = total).  The last
// segment whose start is at or below x holds item x.
__device__ __forceinline__ uint32_t segment_of(const unsigned long long *base, uint32_t nseg, uint64_t x) {
    uint32_t lo = 0, hi = nseg;  // base[lo] <= x < base[hi]
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (base[mid] <= x) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Every block takes a contiguous run of the jobs' restore tiles (tile_base:
// host-computed tile offsets per segment), so that blocks share the work of
// the jobs in proportion to their tiles.
template <int R>
__global__ void __launch_bounds__(kRestoreThreads, 4)
k_restore_many(const CloseJob *__restrict__ J, const unsigned long long *__restrict__ tile_base, uint32_t count) {
    const uint64_t total = tile_base[2 * count];
    const uint64_t per = (total + gridDim.x - 1) / gridDim.x;
    uint64_t a = (uint64_t)blockIdx.x * per;
    const uint64_t b = a + per < total ? a + per : total;
    while (a < b) {
        const uint32_t sg = segment_of(tile_base, 2 * count, a), d = sg & 1u;
        const uint64_t end = tile_base[sg + 1] < b ? tile_base[sg + 1] : b;
        const CloseJob &j = J[sg >> 1];
        const RestoreDir D{j.A.n0[d], j.A.n1[d], j.A.tile0, j.A.szmax[d]};
        restore_body<R>(j.G, j.A, d, D, j.A.smem_hot && (end - a) * D.tile0 > 2u, (uint32_t)(a - tile_base[sg]),
                        (uint32_t)(end - tile_base[sg]), 1u);
        a = end;
    }
}

__global__ void __launch_bounds__(1024) k_sort_small_many(const CloseJob *__restrict__ J) {
    const CloseJob &j = J[blockIdx.y];
    const uint32_t dir = blockIdx.x;
    if (!(dir ? j.A.run[1] : j.A.run[0])) return;
    sort_small_body(j.A.hits, j.A.hits_cap, j.A.stats, dir);
}

// Every job's StatBlock, and the first min(hits, kSortSmall) hit keys of
// each direction, into contiguous buffers (one copy to the host for all).
__global__ void __launch_bounds__(256)
k_gather_many(const CloseJob *__restrict__ J, StatBlock *__restrict__ st_out, unsigned long long *__restrict__ hits_out) {
    const CloseJob &j = J[blockIdx.x];
    const uint32_t *src = reinterpret_cast<const uint32_t *>(j.A.stats);
    uint32_t *dst = reinterpret_cast<uint32_t *>(st_out + blockIdx.x);
    for (uint32_t i = threadIdx.x; i < sizeof(StatBlock) / 4; i += blockDim.x) dst[i] = src[i];
    for (uint32_t d = 0; d < j.G.dirs; d++) {
        if (!(d ? j.A.run[1] : j.A.run[0])) continue;
        const unsigned long long n = j.A.stats->nhits[d];
        uint64_t m = n < j.A.hits_cap ? n : j.A.hits_cap;
        if (m > (uint64_t)kSortSmall) m = kSortSmall;
        const unsigned long long *h = j.A.hits + (uint64_t)d * j.A.hits_cap;
        unsigned long long *o = hits_out + ((uint64_t)blockIdx.x * 2 + d) * kSortSmall;
        for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) o[i] = h[i];
    }
}

__global__ void k_reset_many(const CloseJob *__restrict__ J, uint64_t n4) {
    const CloseJob &j = J[blockIdx.y];
    // a DHLA that k_plane_scan wrote holds hot estimators' bits only: stale, not to be cleared
    reset_body(reinterpret_cast<uint4 *>(const_cast<uint32_t *>(j.A.grid)), j.stats_done == 2 ? 0 : n4, j.A.stats,
               blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------- launchers
// the hot bitmap rows that k_restore stages in shared memory
constexpr size_t kRestoreHotMax = (size_t)200 * 1024;
static size_t restore_hot_bytes(const Geometry &G) { return (size_t)(G.r - 2) * ((1u << G.k) >> 5) * 4; }

static unsigned grid_for(uint64_t items, unsigned threads, int num_sms, unsigned per_sm) {
    uint64_t b = (items + threads - 1) / threads;
    const uint64_t cap = (uint64_t)num_sms * per_sm;
    if (b > cap) b = cap;
    return (unsigned)(b ? b : 1);
}

cudaError_t launch_row_stats(const uint32_t *grid, const Geometry &G, int zhot, uint32_t *hotmap,
                             StatBlock *st, int num_sms, cudaStream_t s) {
    const uint64_t ncell = (uint64_t)G.dirs * G.r << G.k;
    k_row_stats<<<grid_for(ncell, 256, num_sms, 8), 256, 0, s>>>(grid, G, zhot, hotmap, st);
    return cudaGetLastError();
}

cudaError_t launch_compact(const uint32_t *hotmap, const Geometry &G, uint32_t *he, uint32_t rows,
                           cudaStream_t s) {
    k_compact<<<G.dirs * rows, 1024, 0, s>>>(hotmap, G, he, rows);
    return cudaGetLastError();
}

// c0 values per tile of a batched restore (its own tests, a tile per block).
void prepare_restore(const Geometry &G, RestoreArgs &A, int num_sms, uint32_t tiles_per_block) {
    uint64_t tests = 0;
    for (uint32_t d = 0; d < G.dirs; d++)
        if (A.run[d]) tests += (uint64_t)A.n0[d] * ((uint64_t)A.n1[d] << restore_ulog(G));
    A.tile0 = restore_tile0(tests, (uint32_t)num_sms, tiles_per_block);
    A.smem_hot = restore_hot_bytes(G) <= kRestoreHotMax;
}

// k_restore tiles of direction d (the same count the kernel derives)
static uint64_t restore_tiles_dir(const Geometry &G, const RestoreArgs &A, uint32_t d) {
    return d < G.dirs && A.run[d] ? restore_tiles(G, A.n0[d], A.n1[d], A.tile0) : 0;
}

template <typename F3, typename F4, typename F5, typename F6, typename F7, typename F8>
static const void *by_rows(uint32_t r, F3 f3, F4 f4, F5 f5, F6 f6, F7 f7, F8 f8) {
    const void *f[] = {(const void *)f3, (const void *)f4, (const void *)f5, (const void *)f6, (const void *)f7,
                       (const void *)f8};
    return r >= 3 && r <= 8 ? f[r - 3] : nullptr;
}

cudaError_t launch_restore(const Geometry &G, RestoreArgs A, uint64_t pair_cap, float xfac, int num_sms,
                           cudaStream_t s) {
    const void *kern = by_rows(G.r, k_restore<3>, k_restore<4>, k_restore<5>, k_restore<6>, k_restore<7>,
                               k_restore<8>);
    if (!kern) return cudaErrorInvalidValue;
    A.smem_hot = restore_hot_bytes(G) <= kRestoreHotMax;
    const size_t smem = A.smem_hot ? restore_hot_bytes(G) : 16;
    int per_sm = 0;
    cudaError_t e = prepare_launch(kern, (int)kRestoreThreads, smem, &per_sm);
    if (e != cudaSuccess) return e;
    uint32_t sms = (uint32_t)num_sms;
    void *args[] = {const_cast<Geometry *>(&G), &A, &pair_cap, &xfac, &sms};
    return launch_dependent(kern, dim3((unsigned)(num_sms * per_sm)), dim3(kRestoreThreads), smem, s, args);
}

cudaError_t launch_close_finish(const unsigned long long *hits, uint64_t hits_cap, StatBlock *st,
                                unsigned long long *out, uint64_t out_cap, unsigned long long *spare,
                                StatBlock *st_out, uint32_t dirs, cudaStream_t s) {
    void *args[] = {&hits, &hits_cap, &st, &out, &out_cap, &spare, &st_out};
    return launch_dependent(reinterpret_cast<const void *>(k_close_finish), dim3(kFinishBlocks, dirs),
                            dim3(kFinishThreads), 0, s, args);
}

cudaError_t launch_estimate(const Geometry &G, const RestoreArgs &A, int num_sms, cudaStream_t s) {
    dim3 grid((unsigned)num_sms * 4, G.dirs);
    k_estimate<<<grid, 256, 0, s>>>(G, A);
    return cudaGetLastError();
}

cudaError_t launch_sort_small(unsigned long long *hits, uint64_t hits_cap, StatBlock *st,
                              const uint32_t run[2], uint32_t dirs, cudaStream_t s) {
    const int smem = kSortSmall * (int)sizeof(unsigned long long);
    int per_sm = 0;
    cudaError_t e = prepare_launch(reinterpret_cast<const void *>(k_sort_small), 1024, smem, &per_sm);
    if (e != cudaSuccess) return e;
    k_sort_small<<<dirs, 1024, smem, s>>>(hits, hits_cap, st, make_uint2(run[0], run[1]));
    return cudaGetLastError();
}

cudaError_t launch_sort_big(unsigned long long *keys, unsigned long long *tmp, uint64_t n, void *scratch, int num_sms,
                            cudaStream_t s, unsigned long long **out, int *launches, uint32_t **overflow) {
    const int smem = kSortSmall * (int)sizeof(unsigned long long);
    int per_sm = 0;
    cudaError_t e;
    *overflow = nullptr;
    if (scratch && n <= kSampleMaxKeys) {
        uint32_t nb = 2;
        while ((uint64_t)nb * 128 < n && nb < kSampleMaxBuckets) nb <<= 1;
        const uint32_t over = (uint64_t)nb * 256 >= n ? 2u : 8u;
        SampleSortArgs S;
        S.spl = static_cast<unsigned long long *>(scratch);
        S.count = reinterpret_cast<uint32_t *>(S.spl + kSampleMaxBuckets);
        S.off = S.count + kSampleMaxBuckets + 1;
        S.cursor = S.off + kSampleMaxBuckets + 1;
        S.ctl = S.cursor + kSampleMaxBuckets + 1;
        const int ssmem = (int)(nb * over * sizeof(unsigned long long));
        if ((e = prepare_launch(reinterpret_cast<const void *>(k_ss_splitters), 1024, ssmem, &per_sm)) != cudaSuccess)
            return e;
        if ((e = prepare_launch(reinterpret_cast<const void *>(k_ss_buckets), 256, smem, &per_sm)) != cudaSuccess)
            return e;
        const unsigned blocks = grid_for(n, 256, num_sms, 4);
        k_ss_splitters<<<1, 1024, ssmem, s>>>(keys, n, nb, over, S);
        k_ss_count<<<blocks, 256, 0, s>>>(keys, n, nb, S);
        k_ss_scatter<<<grid_for(n, 256 * kScatterKeys, num_sms, 4), 256, 0, s>>>(keys, tmp, n, nb, S);
        k_ss_buckets<<<nb, 256, smem, s>>>(tmp, keys, S);
        *launches = 4;
        *out = keys;
        *overflow = S.ctl + 1;
        return cudaGetLastError();
    }
    e = prepare_launch(reinterpret_cast<const void *>(k_sort_segments), 1024, smem, &per_sm);
    if (e != cudaSuccess) return e;
    const uint64_t segs = (n + kSortSmall - 1) / kSortSmall;
    k_sort_segments<<<(unsigned)segs, 1024, smem, s>>>(keys, n);
    *launches = 1;
    if (segs <= kMergeAllMaxSegs) {
        k_merge_all<<<grid_for(n, 256, num_sms, 8), 256, 0, s>>>(keys, tmp, n);
        *launches = 2;
        *out = tmp;
        return cudaGetLastError();
    }
    unsigned long long *a = keys, *b = tmp;
    for (uint64_t L = kSortSmall; L < n; L <<= 1) {
        k_merge_rank<<<grid_for(n, 256, num_sms, 8), 256, 0, s>>>(a, b, n, L);
        ++*launches;
        unsigned long long *t = a;
        a = b;
        b = t;
    }
    *out = a;
    return cudaGetLastError();
}

cudaError_t launch_reset(uint32_t *grid, uint64_t words, StatBlock *st, int num_sms, cudaStream_t s) {
    const uint64_t n4 = words / 4;
    k_reset<<<grid_for(n4, 256, num_sms, 8), 256, 0, s>>>(reinterpret_cast<uint4 *>(grid), n4, st);
    return cudaGetLastError();
}

// Batched launchers: the grid's first dimension is shared by all jobs (each
// job strides over its own work with it), the job index is the last one.
cudaError_t launch_stats_many(const CloseJob *J, uint32_t count, const Geometry &G, int num_sms, cudaStream_t s) {
    const uint64_t ncell = (uint64_t)G.dirs * G.r << G.k;
    const unsigned per_job = std::max(1u, grid_for(ncell, 256, num_sms, 8) / std::max(1u, count / 4));
    k_row_stats_many<<<dim3(per_job, count), 256, 0, s>>>(J);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_compact_many<<<dim3(G.dirs * 2, count), 1024, 0, s>>>(J);
    return cudaGetLastError();
}

cudaError_t launch_restore_many(const CloseJob *J, const CloseJob *Jh, uint32_t count, unsigned long long *tile_base_d,
                                unsigned long long *tile_base_h, int num_sms, cudaStream_t s, int *launches) {
    *launches = 0;
    const Geometry &G = Jh[0].G;
    // (of the shape: a job that does not run has no smem_hot of its own)
    const size_t smem = restore_hot_bytes(G) <= kRestoreHotMax ? restore_hot_bytes(G) : 16;
    unsigned long long acc = 0;
    bool any = false;
    for (uint32_t i = 0; i < count; i++) {
        any = any || Jh[i].A.run[0] || Jh[i].A.run[1];
        for (uint32_t d = 0; d < 2; d++) {
            tile_base_h[2 * i + d] = acc;
            if (d < G.dirs) acc += restore_tiles_dir(G, Jh[i].A, d);
        }
    }
    tile_base_h[2 * count] = acc;
    if (!any) return cudaSuccess;
    cudaError_t e = cudaMemcpyAsync(tile_base_d, tile_base_h, (2 * count + 1) * sizeof(unsigned long long),
                                    cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    if (acc > 0) {
        const void *kern = by_rows(G.r, k_restore_many<3>, k_restore_many<4>, k_restore_many<5>, k_restore_many<6>,
                                   k_restore_many<7>, k_restore_many<8>);
        if (!kern) return cudaErrorInvalidValue;
        int per_sm = 0;
        e = prepare_launch(kern, (int)kRestoreThreads, smem, &per_sm);
        if (e != cudaSuccess) return e;
        const uint64_t blocks = std::min<uint64_t>((uint64_t)num_sms * per_sm, acc);
        void *args[] = {&J, &tile_base_d, &count};
        e = cudaLaunchKernel(kern, dim3((unsigned)blocks), dim3(kRestoreThreads), args, smem, s);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    const int ssmem = kSortSmall * (int)sizeof(unsigned long long);
    int per_sm = 0;
    e = prepare_launch(reinterpret_cast<const void *>(k_sort_small_many), 1024, ssmem, &per_sm);
    if (e != cudaSuccess) return e;
    k_sort_small_many<<<dim3(G.dirs, count), 1024, ssmem, s>>>(J);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_gather_many(const CloseJob *J, uint32_t count, StatBlock *st_out, unsigned long long *hits_out,
                               cudaStream_t s) {
    k_gather_many<<<count, 256, 0, s>>>(J, st_out, hits_out);
    return cudaGetLastError();
}

cudaError_t launch_reset_many(const CloseJob *J, uint32_t count, const Geometry &G, int num_sms, cudaStream_t s) {
    const uint64_t n4 = (uint64_t)G.dirs * G.dir_words / 4;
    const unsigned per_job = std::max(1u, grid_for(n4, 256, num_sms, 8) / std::max(1u, count / 4));
    k_reset_many<<<dim3(per_job, count), 256, 0, s>>>(J, n4);
    return cudaGetLastError();
}

cudaError_t launch_merge(uint32_t *dst, const uint32_t *src, uint64_t words, int num_sms, cudaStream_t s) {
    const uint64_t n4 = words / 4;
    k_merge_or<<<grid_for(n4, 256, num_sms, 8), 256, 0, s>>>(reinterpret_cast<uint4 *>(dst),
                                                            reinterpret_cast<const uint4 *>(src), n4);
    return cudaGetLastError();
}

}  // namespace sd
