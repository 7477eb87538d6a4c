// sd_fold.cu -- the fold of the plane-binned update's plane-major DHLA copy
// into the estimator-major DHLA (grid |= planes^T, then planes = 0), run
// before anything reads the DHLA: sd_get_grid, sd_set_grid, sd_merge,
// sd_export_grid, sd_or_grid and the window close (one launch for every
// handle of a batched close) -- except a close whose DHLA is the plane copy
// alone, which counts the copy as it is (k_plane_scan below).
//
// Plane (d, b) holds bit b of every estimator of direction d: its row i
// starts at word i * 2^k/32 and holds estimator c's bit at word c >> 5, bit
// c & 31 (planes are ps words apart).  The DHLA holds estimator c's g bits
// as g/32 consecutive words.  Bit c & 31 of word c >> 5 of row i of plane
// 32 t + j is bit j of word t of estimator c of row i: each 32 x 32 bit block
// (32 planes x 32 estimators) is transposed.
#include "sd_common.cuh"

namespace sd {

// ------------------------------------------------------------------- fold
// One block per tile: TC groups of 32 planes (32 TC consecutive bits of
// every estimator of a row) times W consecutive words of one row of those
// planes (32 W estimators), 32 TC W = 8192 words at most.  The tile is
// copied with coalesced 16-byte asynchronous copies into shared memory (and
// its plane words cleared); each thread (t, w) transposes the 32 x 32 bit
// block of plane group t at word w in registers (32 words of 32 planes ->
// word t of 32 estimators); the results are staged by (t, estimator) and
// each estimator's TC words are written to the DHLA with vector stores.  A
// DHLA known to be all zero ("clean") is written without being read.
//
// Shapes: TC = min(8, g/32), W = min(32, 2^k/32); or, when the fold also
// computes the row statistics, TC = g/32 (8, 16 or 32: the tile holds every
// bit of its estimators) and W = min(2^k/32, 256 / TC).  With statistics each estimator's
// z_0 = g - popcount is tested against zhot, its hot bit goes to the tile's
// W hot bitmap words (written whole), and the tile adds its sum of z_0 and
// its hot count to ZR(i) and |HE(i)| -- what k_row_stats computes.
constexpr uint32_t kFoldThreads = 256;
constexpr uint32_t kFoldTile = 8192;  // words per tile stage (32 TC W)
constexpr size_t kFoldSmem = (size_t)2 * kFoldTile * 4;  // two tile stages

// 32 x 32 bit transpose in registers: afterwards bit j of x[b] is what was
// bit b of x[j] (block swaps of 16, 8, 4, 2 and 1 bits).
__device__ __forceinline__ void transpose32_regs(uint32_t (&x)[32]) {
#pragma unroll
    for (int s = 0; s < 5; s++) {
        const uint32_t j = 16u >> s;
        const uint32_t m = s == 0 ? 0x0000FFFFu : s == 1 ? 0x00FF00FFu : s == 2 ? 0x0F0F0F0Fu
                         : s == 3 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (uint32_t r = 0; r < 32; r++) {
            if (r & j) continue;
            const uint32_t t = ((x[r] >> j) ^ x[r + j]) & m;
            x[r] ^= t << j;
            x[r + j] ^= t;
        }
    }
}

// Where tile `tile` of a fold lies: its job, direction, row, first plane
// group and first plane word.
struct FoldTile {
    FoldJob job;
    uint32_t d, i, tc0, w0;
};
__device__ __forceinline__ FoldTile fold_tile(uint64_t tile, uint64_t per_job, uint32_t tgroups, uint32_t wgroups,
                                              uint32_t TC, uint32_t W, const Geometry &G, const FoldJob &one,
                                              const FoldJob *jobs) {
    FoldTile f;
    const uint32_t jn = (uint32_t)(tile / per_job);
    f.job = jobs ? jobs[jn] : one;
    uint64_t rest = tile - (uint64_t)jn * per_job;
    f.tc0 = (uint32_t)(rest % tgroups) * TC;
    rest /= tgroups;
    f.w0 = (uint32_t)(rest % wgroups) * W;
    rest /= wgroups;
    f.i = (uint32_t)(rest % G.r);
    f.d = (uint32_t)(rest / G.r);
    return f;
}

// The tile shape of a fold (see above).
__host__ __device__ __forceinline__ void fold_shape(const Geometry &G, bool stats, uint32_t &TC, uint32_t &W) {
    const uint32_t rw = (1u << G.k) >> 5;
    TC = stats ? G.wpc : (G.wpc < 8u ? G.wpc : 8u);
    const uint32_t wmax = stats ? 256u / G.wpc : 32u;
    W = rw < wmax ? rw : wmax;
}

// Folds of several handles of one shape run as one launch (the batched
// close): the tiles of job j follow those of job j - 1.  Two tile stages:
// the next tile's plane words are copied in (cp.async) while the current
// one is transposed; the transposed words are staged in place of the
// current tile's input.
__global__ void __launch_bounds__(kFoldThreads, 3)
k_plane_fold(FoldJob one, const FoldJob *__restrict__ jobs, uint32_t njobs, Geometry G, uint32_t ps,
             uint32_t stats) {
    extern __shared__ uint4 fold_smem[];
    __shared__ uint32_t s_hot[32];
    __shared__ unsigned long long s_zr;
    __shared__ uint32_t s_nhot;
    uint32_t *const stage0 = reinterpret_cast<uint32_t *>(fold_smem);
    const uint32_t wpc = G.wpc;
    uint32_t TC, W;
    fold_shape(G, stats != 0, TC, W);
    const uint32_t rw = (1u << G.k) >> 5;  // plane words per row
    const uint32_t wgroups = rw / W, tgroups = wpc / TC;
    const uint64_t per_job = (uint64_t)G.dirs * G.r * wgroups * tgroups;
    const uint64_t tiles = per_job * njobs;
    const uint32_t W4 = W / 4, rows = 32u * TC;
    // rows of one or two words (k < 7) have no 16-byte words: copied and
    // cleared word by word
    const uint32_t words = W4 ? 0u : rows * W;
    const uint32_t tt = threadIdx.x / W, w = threadIdx.x % W;
    const uint32_t lane = threadIdx.x & 31u;
    // a tile's first plane word
    auto plane_base = [&](const FoldTile &f) {
        return f.job.planes + ((uint64_t)f.d * G.g + 32u * f.tc0) * ps + (uint64_t)f.i * rw + f.w0;
    };
    // start copying tile `tile` into stage s (one commit group per call)
    auto issue = [&](uint64_t tile, uint32_t s) {
        if (tile < tiles) {
            const FoldTile f = fold_tile(tile, per_job, tgroups, wgroups, TC, W, G, one, jobs);
            const uint32_t *pb = plane_base(f);
            const uint32_t sa = (uint32_t)__cvta_generic_to_shared(stage0 + s * kFoldTile);
            for (uint32_t q = threadIdx.x; q < words; q += blockDim.x) {
                const uint32_t row = q / W, c = q - row * W;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                             ::"r"(sa + 4u * q), "l"(pb + (uint64_t)row * ps + c)
                             : "memory");
            }
            for (uint32_t q = threadIdx.x; q < rows * W4; q += blockDim.x) {
                const uint32_t row = q / W4, c = q - row * W4;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             ::"r"(sa + 16u * q), "l"(pb + (uint64_t)row * ps + 4u * c)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (threadIdx.x < 32) s_hot[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        s_zr = 0;
        s_nhot = 0;
    }
    uint32_t cur = 0;
    issue(blockIdx.x, 0);
    for (uint64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, cur ^= 1u) {
        issue(tile + gridDim.x, cur ^ 1u);
        asm volatile("cp.async.wait_group 1;" ::: "memory");  // this tile's copies are done
        __syncthreads();
        const FoldTile f = fold_tile(tile, per_job, tgroups, wgroups, TC, W, G, one, jobs);
        uint32_t *in = stage0 + cur * kFoldTile;
        // clear the tile's plane words that hold bits
        uint32_t *pb = plane_base(f);
        for (uint32_t q = threadIdx.x; q < words; q += blockDim.x) {
            const uint32_t row = q / W, c = q - row * W;
            if (in[q]) pb[(uint64_t)row * ps + c] = 0u;
        }
        for (uint32_t q = threadIdx.x; q < rows * W4; q += blockDim.x) {
            const uint4 v = reinterpret_cast<const uint4 *>(in)[q];
            if (v.x | v.y | v.z | v.w) {
                const uint32_t row = q / W4, c = q - row * W4;
                *reinterpret_cast<uint4 *>(pb + (uint64_t)row * ps + 4u * c) = make_uint4(0, 0, 0, 0);
            }
        }
        uint32_t x[32];
        const bool mine = tt < TC;
        if (mine) {
#pragma unroll
            for (uint32_t j = 0; j < 32; j++) x[j] = in[(32u * tt + j) * W + w];
            transpose32_regs(x);
        }
        __syncthreads();  // every read of the input stage is done
        uint32_t *out = in;  // [TC][32 bits][W words]
        if (mine) {
#pragma unroll
            for (uint32_t b = 0; b < 32; b++) out[(tt * 32u + b) * W + w] = x[b];
        }
        __syncthreads();
        // estimator 32 (w0 + w) + b of row i gets words tc0 .. tc0 + TC - 1
        uint32_t *row = f.job.grid + (uint64_t)f.d * G.dir_words + (uint64_t)f.i * G.row_words;
        for (uint32_t e0 = 0; e0 < 32u * W; e0 += blockDim.x) {  // the same trip count for every thread
            const uint32_t e = e0 + threadIdx.x;
            const bool live = e < 32u * W;
            const uint32_t b = e / W, ww = e - b * W;
            uint32_t pop = 0;
            if (live) {
                uint32_t *dst = row + (uint64_t)(32u * (f.w0 + ww) + b) * wpc + f.tc0;
                if ((TC & 3u) == 0) {
                    uint4 *d4 = reinterpret_cast<uint4 *>(dst);
                    for (uint32_t h = 0; h < TC / 4; h++) {
                        uint4 nv = make_uint4(out[((4 * h) * 32u + b) * W + ww], out[((4 * h + 1) * 32u + b) * W + ww],
                                              out[((4 * h + 2) * 32u + b) * W + ww],
                                              out[((4 * h + 3) * 32u + b) * W + ww]);
                        const bool any = (nv.x | nv.y | nv.z | nv.w) != 0;
                        if (!f.job.clean && (any || stats)) {
                            const uint4 c = d4[h];
                            nv.x |= c.x; nv.y |= c.y; nv.z |= c.z; nv.w |= c.w;
                            if (nv.x != c.x || nv.y != c.y || nv.z != c.z || nv.w != c.w) d4[h] = nv;
                        } else if (any) {
                            d4[h] = nv;
                        }
                        pop += __popc(nv.x) + __popc(nv.y) + __popc(nv.z) + __popc(nv.w);
                    }
                } else {
                    for (uint32_t t = 0; t < TC; t++) {
                        uint32_t v = out[(t * 32u + b) * W + ww];
                        if (!f.job.clean && (v || stats)) v |= dst[t];
                        if (out[(t * 32u + b) * W + ww]) dst[t] = v;
                        pop += __popc(v);
                    }
                }
            }
            if (stats) {
                // z_0 of this estimator; hot bits gathered per hot bitmap word
                const uint32_t z0 = G.g - pop;
                const bool hot = live && (int)z0 <= f.job.zhot;
                const unsigned mask = __ballot_sync(0xFFFFFFFFu, hot);
                unsigned long long zs = live ? z0 : 0u;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) zs += __shfl_xor_sync(0xFFFFFFFFu, zs, o);
                if (lane == 0) {
                    atomicAdd(&s_zr, zs);
                    atomicAdd(&s_nhot, (uint32_t)__popc(mask));
                }
                // the warp's estimators: 32 / W values of b (W < 32) or one
                if (lane < W && live) {
                    const uint32_t b0 = (e - lane) / W;
                    uint32_t c = 0;
                    for (uint32_t qq = 0; qq * W < 32u; qq++) c |= ((mask >> (qq * W + lane)) & 1u) << (b0 + qq);
                    atomicOr(&s_hot[lane], c);
                }
            }
        }
        __syncthreads();  // the stage is refilled two tiles on; the tile's statistics are complete
        if (stats) {
            uint32_t *hm = f.job.hotmap + ((uint64_t)f.d * G.r + f.i) * (rw) + f.w0;
            if (threadIdx.x < W) {
                hm[threadIdx.x] = s_hot[threadIdx.x];
                s_hot[threadIdx.x] = 0;
            }
            if (threadIdx.x == 0) {
                atomicAdd(&f.job.st->zr[f.d][f.i], s_zr);
                atomicAdd(&f.job.st->nhot[f.d][f.i], s_nhot);
                s_zr = 0;
                s_nhot = 0;
            }
            __syncthreads();
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

cudaError_t launch_plane_fold(const FoldJob &one, const FoldJob *jobs, uint32_t njobs, const Geometry &G, uint32_t ps,
                              int num_sms, cudaStream_t s) {
    if (njobs == 0) return cudaSuccess;
    const bool stats = one.st != nullptr;
    if (stats && !fold_stats_fit(G)) return cudaErrorInvalidValue;
    int per_sm = 0;
    cudaError_t e = prepare_launch(reinterpret_cast<const void *>(k_plane_fold), kFoldThreads, kFoldSmem, &per_sm);
    if (e != cudaSuccess) return e;
    uint32_t TC, W;
    fold_shape(G, stats, TC, W);
    const uint64_t rw = ((uint64_t)1 << G.k) >> 5;
    const uint64_t tiles = (uint64_t)G.dirs * G.r * (rw / W) * (G.wpc / TC) * (jobs ? njobs : 1u);
    uint64_t blocks = (uint64_t)num_sms * per_sm;
    if (tiles < blocks) blocks = tiles;
    k_plane_fold<<<(unsigned)blocks, kFoldThreads, kFoldSmem, s>>>(one, jobs, jobs ? njobs : 1u, G, ps,
                                                                   stats ? 1u : 0u);
    return cudaGetLastError();
}

// ------------------------------------------------------- fold at a close
// A window close reads the DHLA twice: for every estimator's z_0, and for
// the bits of the hot ones (each candidate's r estimators are hot).  So when
// the DHLA holds nothing but the plane copy, the close does not fold it: it
// counts every estimator's bits in the plane copy as it is, clears the copy,
// and writes only the hot estimators' bits to the DHLA.  The other words of
// the DHLA keep what an earlier close left there and the handle is marked
// stale: the next close writes all that it reads, and any other reader
// clears the DHLA first.  HE(0) and HE(1) are listed by the block that
// counts the last estimators of their row.
//
// Counting: a thread holds one word (32 estimators) of 32 planes and adds
// them bit-sliced (57 full adders of two three-input operations each give
// six words: bit i of word b is bit b of estimator i's count); the g/32
// partial counts of a word are added the same way through shared memory, and
// the hot test z_0 <= zhot, i.e. count >= g - zhot, is a bit-sliced
// comparison.  No transpose, except of the 32 x 32 blocks whose word has a
// hot estimator.  Bound by the plane copy's read and clear: the core
// sketch's 32 MiB take 14 us with few hot estimators and 22 us with 4,200 a
// row (the fold with statistics, the lists and the DHLA's clear took 28 to
// 33, 4 and 6.5 us); 64 of them 0.94 ms (1.4 and 0.3 ms), 4.6 TB/s.
constexpr uint32_t kScanThreads = 256;
constexpr uint32_t kCountBits = 12;  // counts up to 1024

// s = a + b of N-bit sliced numbers, N + 1 bits
template <int N>
__device__ __forceinline__ void add_sliced(const uint32_t (&a)[N], const uint32_t (&b)[N], uint32_t (&s)[N + 1]) {
    uint32_t carry = 0;
#pragma unroll
    for (int i = 0; i < N; i++) {
        s[i] = a[i] ^ b[i] ^ carry;
        carry = (a[i] & b[i]) | (carry & (a[i] ^ b[i]));
    }
    s[N] = carry;
}

// bit-sliced sum of x[at .. at + 2^LOG)
template <int LOG>
__device__ __forceinline__ void count_sliced(const uint32_t (&x)[32], int at, uint32_t (&s)[LOG + 1]) {
    if constexpr (LOG == 0) {
        s[0] = x[at];
    } else {
        uint32_t a[LOG], b[LOG];
        count_sliced<LOG - 1>(x, at, a);
        count_sliced<LOG - 1>(x, at + (1 << (LOG - 1)), b);
        add_sliced<LOG>(a, b, s);
    }
}

// HE(row) of direction d in ascending order from its hot bitmap (one block;
// the bitmap words were written by other blocks).
__device__ __forceinline__ void list_hot(const uint32_t *bm, uint32_t nw, uint32_t *out) {
    __shared__ uint32_t s_tot[kScanThreads / 32];
    const uint32_t per = (nw + blockDim.x - 1) / blockDim.x;
    const uint32_t w0 = min(threadIdx.x * per, nw), w1 = min(w0 + per, nw);
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    uint32_t cnt = 0;
    for (uint32_t w = w0; w < w1; w++) cnt += __popc(__ldcg(bm + w));
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += v;
    }
    if (lane == 31) s_tot[wid] = incl;
    __syncthreads();
    uint32_t pos = incl - cnt;
    for (uint32_t q = 0; q < wid; q++) pos += s_tot[q];
    for (uint32_t w = w0; w < w1; w++) {
        uint32_t b = __ldcg(bm + w);
        while (b) {
            out[pos++] = (w << 5) | (uint32_t)(__ffs(b) - 1);
            b &= b - 1u;
        }
    }
    __syncthreads();
}

// p, with its value hidden from the compiler: a later pass over the same 32
// addresses then forms them again instead of keeping them in 64 registers.
__device__ __forceinline__ uint32_t *opaque(uint32_t *p) {
    asm volatile("" : "+l"(p));
    return p;
}

// TC = g/32 plane groups; a block takes W = 256 / TC words of one row.
template <int TC>
__global__ void __launch_bounds__(kScanThreads, 4)
k_plane_scan(FoldJob one, const FoldJob *__restrict__ jobs, Geometry G, uint32_t ps) {
    constexpr uint32_t W = kScanThreads / TC;
    constexpr int LOG = TC == 8 ? 3 : TC == 16 ? 4 : 5;  // log2 TC
    constexpr int LW = LOG - 3;                          // of them within a warp
    constexpr int S = 6 + LOG;                           // bits of a full count
    __shared__ uint32_t s_part[7][S][W];
    __shared__ uint32_t s_hot[W];
    __shared__ bool s_list;
    dependents_may_start();
    const uint32_t rw = (1u << G.k) >> 5;
    const uint32_t wgroups = (rw + W - 1) / W;
    uint32_t tile = blockIdx.x;
    const uint32_t wg = tile % wgroups;
    tile /= wgroups;
    const uint32_t i = tile % G.r;
    tile /= G.r;
    const uint32_t d = tile % G.dirs;
    const FoldJob job = jobs ? jobs[tile / G.dirs] : one;
    const uint32_t tt = threadIdx.x / W, w = threadIdx.x % W, word = wg * W + w;
    const bool live = word < rw;
    uint32_t *src = job.planes + ((uint64_t)d * G.g + 32u * tt) * ps + (uint64_t)i * rw + word;
    uint32_t acc[S];  // this thread's count, then sums of TC of them
    uint32_t any = 0;  // planes with a bit in this word
    {
        uint32_t x[32], mine[6];
        const uint32_t *p = src;
#pragma unroll
        for (uint32_t j = 0; j < 32; j++, p += ps) x[j] = live ? __ldcg(p) : 0u;
#pragma unroll
        for (uint32_t j = 0; j < 32; j++) any |= (x[j] ? 1u : 0u) << j;
        count_sliced<5>(x, 0, mine);
#pragma unroll
        for (int b = 0; b < S; b++) acc[b] = b < 6 ? mine[b] : 0u;
    }
    // the plane groups within a warp, then the eight warps, pairwise
#pragma unroll
    for (int l = 0; l < LW; l++) {
        uint32_t v[S - 1];
#pragma unroll
        for (int b = 0; b < 6 + l; b++) v[b] = __shfl_xor_sync(0xFFFFFFFFu, acc[b], W << l);
        uint32_t carry = 0;
#pragma unroll
        for (int b = 0; b < 6 + l; b++) {
            const uint32_t a = acc[b];
            acc[b] = a ^ v[b] ^ carry;
            carry = (a & v[b]) | (carry & (a ^ v[b]));
        }
        acc[6 + l] = carry;
    }
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
#pragma unroll
    for (int l = 0; l < 3; l++) {
        const uint32_t half = 4u >> l, at = 8u - 2u * half;  // slots at, at + 1, ... of this level
        if (wid >= half && wid < 2 * half && lane < W) {
#pragma unroll
            for (int b = 0; b < 6 + LW + l; b++) s_part[at + wid - half][b][lane] = acc[b];
        }
        __syncthreads();
        if (wid < half && lane < W) {
            uint32_t carry = 0;
#pragma unroll
            for (int b = 0; b < 6 + LW + l; b++) {
                const uint32_t v = s_part[at + wid][b][lane], a = acc[b];
                acc[b] = a ^ v ^ carry;
                carry = (a & v) | (carry & (a ^ v));
            }
            acc[6 + LW + l] = carry;
        }
    }
    if (threadIdx.x < W) {  // lanes of the first warp
        const uint32_t T = (uint32_t)max((int)G.g - job.zhot, 0);
        uint32_t gt = 0, eq = ~0u, ones = 0;
#pragma unroll
        for (int b = kCountBits - 1; b >= 0; b--) {
            const uint32_t v = b < S ? acc[b < S ? b : 0] : 0u;
            const uint32_t t = (T >> b & 1u) ? ~0u : 0u;
            gt |= eq & v & ~t;
            eq &= ~(v ^ t);
            ones += (uint32_t)__popc(v) << b;
        }
        const uint32_t hot = live ? (gt | eq) : 0u;
        s_hot[w] = hot;
        if (live) job.hotmap[((uint64_t)d * G.r + i) * rw + word] = hot;
        uint32_t z = live ? 32u * G.g - ones : 0u, nh = (uint32_t)__popc(hot);
        constexpr uint32_t mask = W == 32 ? 0xFFFFFFFFu : (1u << W) - 1u;
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) {
            z += __shfl_xor_sync(mask, z, o);
            nh += __shfl_xor_sync(mask, nh, o);
        }
        if (w == 0) {
            atomicAdd(&job.st->zr[d][i], (unsigned long long)z);
            if (nh) atomicAdd(&job.st->nhot[d][i], nh);
        }
    }
    __syncthreads();
    const uint32_t hot = s_hot[w];
    if (hot) {
        uint32_t x[32];
        const uint32_t *p = opaque(src);
#pragma unroll
        for (uint32_t j = 0; j < 32; j++, p += ps) x[j] = __ldcg(p);
        transpose32_regs(x);  // x[b]: word tt of estimator 32 word + b
        uint32_t *dst = job.grid + (uint64_t)d * G.dir_words + (uint64_t)i * G.row_words + (uint64_t)(32u * word) * TC + tt;
#pragma unroll
        for (uint32_t b = 0; b < 32; b++)
            if (hot >> b & 1u) dst[b * TC] = x[b];
    }
    if (any) {
        uint32_t *p = opaque(src);
#pragma unroll
        for (uint32_t j = 0; j < 32; j++, p += ps)
            if (any >> j & 1u) *p = 0u;
    }
    if (i >= 2) return;
    // rows 0 and 1: the block that counts the row's last estimators lists it
    // (its bitmap words were written by the W threads above)
    if (threadIdx.x < W) {
        __threadfence();
        constexpr uint32_t mask = W == 32 ? 0xFFFFFFFFu : (1u << W) - 1u;
        __syncwarp(mask);
        if (threadIdx.x == 0) s_list = atomicAdd(&job.st->rows_done[d][i], 1u) == wgroups - 1;
    }
    __syncthreads();
    if (s_list) {
        __threadfence();
        list_hot(job.hotmap + ((uint64_t)d * G.r + i) * rw, rw, job.he + ((uint64_t)d * 2 + i) * (1ull << G.k));
    }
}

cudaError_t launch_plane_scan(const FoldJob &one, const FoldJob *jobs, uint32_t njobs, const Geometry &G, uint32_t ps,
                              cudaStream_t s) {
    if (jobs && njobs == 0) return cudaSuccess;
    if (!fold_stats_fit(G)) return cudaErrorInvalidValue;
    const uint32_t W = kScanThreads / G.wpc, rw = (1u << G.k) >> 5;
    const uint64_t blocks = (uint64_t)(jobs ? njobs : 1u) * G.dirs * G.r * ((rw + W - 1) / W);
    if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    switch (G.wpc) {
        case 8: k_plane_scan<8><<<(unsigned)blocks, kScanThreads, 0, s>>>(one, jobs, G, ps); break;
        case 16: k_plane_scan<16><<<(unsigned)blocks, kScanThreads, 0, s>>>(one, jobs, G, ps); break;
        case 32: k_plane_scan<32><<<(unsigned)blocks, kScanThreads, 0, s>>>(one, jobs, G, ps); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace sd
