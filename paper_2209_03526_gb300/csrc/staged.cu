// staged.cu -- masked-mode secEval of a launch whose elements share tree nodes.
//
// In the masked mode one predicate's keys are evaluated at x^ = x + r of every element of a
// column, so the walks of all elements run in the same few trees: elements whose x^ agree in
// the first l bits pass through the same node of level l, and equal values are one walk.  A
// server that has opened the column (every server learns x^ of each element, Sec. V-C) can
// therefore visit each node once instead of once per element.  The kernels here do that:
//
//   1. each column the launch reads is opened once (for its first predicate; another
//      predicate's x^ differs by a constant) and sorted, and its distinct values and every
//      element's rank among them are written (k_sort_*, k_uniq_*).  A column whose domain is
//      hardly larger than its table is dense instead: the distinct values are 0 .. 2^n - 1;
//   2. per predicate, the levels are cut into stages (choose_stages).  A run is a maximal set
//      of distinct values that agree in the bits up to a stage's last level; k_run_* list the
//      runs and each one's parent run;
//   3. k_stage evaluates a stage: one walk per (key, run) from the parent's seed, control bit
//      and value sum, which a table in memory holds; k_stage_last walks the remaining levels
//      for every distinct value and sums the halves per server (Eq. predEval);
//   4. k_combine looks up each element's three sums, re-shares and folds them (Sec. III-B,
//      V-D), exactly as the fused kernel does.
//
// For 2^20 uniform 32-bit values a key takes about 13.5 x 2^20 level steps instead of
// 32 x 2^20; skewed columns take far fewer.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <vector>

#include "device_fss.cuh"
#include "ptx_async.cuh"
#include "runtime.h"
#include "staged.h"

namespace ogm {

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
// Keys per thread of a sort tile: 16 (4,096 keys per CTA) where that gives every SM a few CTAs,
// else 4, which shortens the chain of a CTA that has an SM to itself.
constexpr int kSortItemsLarge = 16, kSortItemsSmall = 4;
constexpr uint32_t kRunBlock = 1024;                         // distinct values per CTA of the run kernels
constexpr int kStageThreads = 768;                           // one CTA per SM (the tables take 128 KiB)
constexpr uint32_t kMaxRoundPreds = 64;

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// All launches of an evaluation but the first are programmatic dependents of the one before
// (ptx_async.cuh), since many are a few microseconds long: 100,003 vertices, 3 predicates (27
// launches) 1,759 -> 1,700 us, 12 DCF keys at 65,537 points 631 -> 578 us, triangle + pendant on
// 1M / 10M (200 launches) 17.07 -> 16.66 ms.

// ------------------------------------------------------------------ opened columns, sorted
//
// Least-significant-digit radix sort, 8 bits a pass, of all the launch's sparse columns side
// by side (grid y).  A pass is three launches: digit counts per tile, their sums along the
// tiles, and the stable scatter.  It moves 20 bytes a key and pass.

template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const SgCol* cols, uint32_t pass) {
    __shared__ uint32_t h[256];
    const SgCol& C = cols[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (blockIdx.x >= C.tiles || pass >= C.passes) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t base = (uint64_t)blockIdx.x * (kSortThreads * ITEMS);
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        const uint64_t e = base + (uint32_t)i * kSortThreads + threadIdx.x;
        if (e < C.n) {
            uint32_t k;
            if (pass == 0) {
                // open x^ = <x>_1 + <x>_2 + <x>_3 + r mod 2^n
                k = __ldg(C.share[0] + e);
                if (C.share[1]) k += __ldg(C.share[1] + e) + __ldg(C.share[2] + e) + C.radd;
                k &= C.mask;
                C.key[0][e] = k;
            } else {
                k = C.key[pass & 1][e];
            }
            atomicAdd(&h[(k >> (8 * pass)) & 255u], 1u);
        }
    }
    __syncthreads();
    C.hist[(uint64_t)threadIdx.x * C.tiles + blockIdx.x] = h[threadIdx.x];
}

// exclusive sum of a CTA's 256 values; *total the sum of all
__device__ __forceinline__ uint32_t block_exclusive_256(uint32_t v, uint32_t* warp_sums, uint32_t* total) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t s = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, s, off);
        if (lane >= (uint32_t)off) s += o;
    }
    __syncthreads();
    if (lane == 31) warp_sums[warp] = s;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < 8; w++) {
        const uint32_t x = warp_sums[w];
        before += (uint32_t)w < warp ? x : 0u;
        all += x;
    }
    *total = all;
    return before + s - v;
}

// in-place exclusive sum of row[0 .. n) by one CTA of 256 threads; the sum of all goes to *total
__device__ __forceinline__ void row_scan(uint32_t* row, uint32_t n, uint32_t* total) {
    __shared__ uint32_t ws[8];
    uint32_t carry = 0;
    for (uint32_t b = 0; b < n; b += 256) {
        const uint32_t i = b + threadIdx.x;
        const uint32_t v = i < n ? row[i] : 0u;
        uint32_t all;
        const uint32_t x = block_exclusive_256(v, ws, &all);
        if (i < n) row[i] = carry + x;
        carry += all;
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(256) k_sort_scan(const SgCol* cols, uint32_t pass) {
    const SgCol& C = cols[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (pass >= C.passes) return;
    row_scan(C.hist + (uint64_t)blockIdx.x * C.tiles, C.tiles, C.tot + blockIdx.x);
}

// Lanes of the warp whose 9-bit value equals this lane's, by a ballot per bit: a match
// instruction takes time per distinct value, which are many here.
__device__ __forceinline__ uint32_t same_digit(uint32_t d) {
    uint32_t m = 0xFFFFFFFFu;
#pragma unroll
    for (int b = 0; b < 9; b++) {
        const uint32_t v = __ballot_sync(0xFFFFFFFFu, (d >> b) & 1u);
        m &= (d >> b) & 1u ? v : ~v;
    }
    return m;
}

// The stable scatter.  Each warp ranks its keys among its own of the same digit; the tile's
// keys then go through shared memory in digit order, so that a digit's keys leave as one
// consecutive run of stores (16 of them in the mean at 4,096 keys and 256 digits): storing
// each key straight from its thread took 416 us a pass on 2 x 10M keys (one sector per word).
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads, 3) k_sort_scatter(const SgCol* cols, uint32_t pass) {
    constexpr uint32_t kTile = kSortThreads * ITEMS;
    __shared__ uint32_t cnt[kSortWarps][256];
    __shared__ uint32_t skey[kTile], sidx[kTile];
    __shared__ uint32_t base_of[256];      // output position of a digit's first key, less its place in the tile
    __shared__ uint32_t ws[8];
    const SgCol& C = cols[blockIdx.y];
    grid_trigger();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, shift = 8 * pass;
    for (int w = 0; w < kSortWarps; w++) cnt[w][threadIdx.x] = 0;
    grid_wait();
    if (blockIdx.x >= C.tiles || pass >= C.passes) return;
    __syncthreads();
    const uint32_t* src = C.key[pass & 1];
    const uint32_t* isrc = C.idx[pass & 1];
    const uint64_t tile0 = (uint64_t)blockIdx.x * kTile;
    const uint64_t base = tile0 + warp * (32 * ITEMS) + lane;     // a warp owns 32 ITEMS consecutive keys
    uint32_t k[ITEMS], rk[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        const uint64_t e = base + 32u * i;
        const bool ok = e < C.n;
        k[i] = ok ? src[e] : 0u;
    }
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        const bool ok = base + 32u * i < C.n;
        const uint32_t d = ok ? (k[i] >> shift) & 255u : 256u;
        const uint32_t same = same_digit(d);
        const uint32_t old = ok ? cnt[warp][d] : 0u;
        __syncwarp();
        const uint32_t below = same & lanemask_lt();
        rk[i] = old + __popc(below);
        if (ok && below == 0) cnt[warp][d] = old + __popc(same);
        __syncwarp();
    }
    __syncthreads();
    // thread d: the place of digit d's first key in the tile, and of each warp's first one
    uint32_t mine = 0, total;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) mine += cnt[w][threadIdx.x];
    uint32_t at = block_exclusive_256(mine, ws, &total);
    const uint32_t tile_keys = total;
    const uint32_t out = block_exclusive_256(C.tot[threadIdx.x], ws, &total) +
                         C.hist[(uint64_t)threadIdx.x * C.tiles + blockIdx.x];
    base_of[threadIdx.x] = out - at;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) {
        const uint32_t c = cnt[w][threadIdx.x];
        cnt[w][threadIdx.x] = at;
        at += c;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        const uint64_t e = base + 32u * i;
        if (e < C.n) {
            const uint32_t o = cnt[warp][(k[i] >> shift) & 255u] + rk[i];
            skey[o] = k[i];
            sidx[o] = pass == 0 ? (uint32_t)e : isrc[e];
        }
    }
    __syncthreads();
    uint32_t* dst = C.key[(pass + 1) & 1];
    uint32_t* didx = C.idx[(pass + 1) & 1];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        const uint32_t o = i * kSortThreads + threadIdx.x;
        if (o < tile_keys) {
            const uint32_t key = skey[o], to = base_of[(key >> shift) & 255u] + o;
            dst[to] = key;
            didx[to] = sidx[o];
        }
    }
}

// The sorted keys' distinct values: counts per tile, their sums, then the values and every
// element's rank.  A warp owns 32 ITEMS consecutive keys of its tile.
__device__ __forceinline__ bool starts_value(const uint32_t* key, uint64_t e, uint64_t n) {
    return e < n && (e == 0 || key[e] != key[e - 1]);
}

template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_uniq_count(const SgCol* cols) {
    __shared__ uint32_t ws[kSortWarps];
    const SgCol& C = cols[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (blockIdx.x >= C.tiles || C.passes == 0) return;
    const uint32_t* key = C.key[C.passes & 1];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * (kSortThreads * ITEMS) + warp * (32 * ITEMS) + lane;
    uint32_t c = 0;
#pragma unroll 4
    for (int i = 0; i < ITEMS; i++)
        c += __popc(__ballot_sync(0xFFFFFFFFu, starts_value(key, base + 32u * i, C.n)));
    if (lane == 0) ws[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < kSortWarps; w++) s += ws[w];
        C.hist[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(256) k_uniq_scan(const SgCol* cols) {
    const SgCol& C = cols[blockIdx.x];
    grid_trigger();
    grid_wait();
    if (C.passes == 0) return;
    row_scan(C.hist, C.tiles, C.m);
}

template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_uniq_emit(const SgCol* cols) {
    __shared__ uint32_t ws[kSortWarps];
    const SgCol& C = cols[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (blockIdx.x >= C.tiles || C.passes == 0) return;
    const uint32_t* key = C.key[C.passes & 1];
    const uint32_t* idx = C.idx[C.passes & 1];
    uint32_t* u = C.key[(C.passes + 1) & 1];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * (kSortThreads * ITEMS) + warp * (32 * ITEMS) + lane;
    uint32_t flags = 0, c = 0;     // bit i: this lane's key of step i starts a value
#pragma unroll 4
    for (int i = 0; i < ITEMS; i++) {
        const bool f = starts_value(key, base + 32u * i, C.n);
        flags |= (f ? 1u : 0u) << i;
        c += __popc(__ballot_sync(0xFFFFFFFFu, f));
    }
    if (lane == 0) ws[warp] = c;
    __syncthreads();
    uint32_t at = C.hist[blockIdx.x];
    for (uint32_t w = 0; w < warp; w++) at += ws[w];
#pragma unroll 4
    for (int i = 0; i < ITEMS; i++) {
        const uint64_t e = base + 32u * i;
        const bool f = (flags >> i) & 1u;
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, f);
        const uint32_t r = at + __popc(b & lanemask_lt()) + (f ? 1u : 0u) - 1u;   // values started up to e, less one
        if (e < C.n) {
            if (f) u[r] = key[e];
            C.rank[idx[e]] = r;
        }
        at += __popc(b);
    }
}

// ------------------------------------------------------------------ runs of a predicate

// values of chunk `c` (a dense column has 2^n of them)
__device__ __forceinline__ uint32_t chunk_values(const SgPred& P, uint32_t c) {
    const uint64_t all = P.dense ? (uint64_t)P.mask + 1u : (uint64_t)*P.m, first = (uint64_t)c * P.chunk;
    return all <= first ? 0u : (uint32_t)min((unsigned long long)(all - first), (unsigned long long)P.chunk);
}

// Bits in which value i of the chunk agrees with the one before, from the top; -1 for the first.
// A run of stage s starts at i where that is below lev[s].
__device__ __forceinline__ int common_bits(const SgPred& P, const uint32_t* u, uint32_t i, uint32_t* x) {
    *x = (u[i] + P.delta) & P.mask;
    if (i == 0) return -1;
    const uint32_t d = *x ^ ((u[i - 1] + P.delta) & P.mask);     // nonzero: the values are distinct
    return __clz((int)d) - (32 - (int)P.n);
}

__global__ void __launch_bounds__(kRunBlock) k_run_count(const SgPred* preds, uint32_t chunk) {
    __shared__ uint32_t ws[32][kSgMaxStages];
    const SgPred& P = preds[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (P.dense) return;
    const uint32_t n = chunk_values(P, chunk);
    if ((uint64_t)blockIdx.x * kRunBlock >= n) return;
    const uint32_t i = blockIdx.x * kRunBlock + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x;
    const int cb = i < n ? common_bits(P, P.u + (uint64_t)chunk * P.chunk, i, &x) : 32;
    const uint32_t S = P.stages - 1;
    for (uint32_t s = 0; s < S; s++) {
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, cb < (int)P.lev[s]);
        if (lane == 0) ws[warp][s] = __popc(b);
    }
    __syncthreads();
    if (threadIdx.x < S) {
        uint32_t c = 0;
        for (int w = 0; w < 32; w++) c += ws[w][threadIdx.x];
        P.blk[(uint64_t)threadIdx.x * P.blocks + blockIdx.x] = c;
    }
}

__global__ void __launch_bounds__(256) k_run_scan(const SgPred* preds, uint32_t chunk) {
    const SgPred& P = preds[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (P.dense || blockIdx.x + 1 >= P.stages) return;
    const uint32_t n = chunk_values(P, chunk);
    row_scan(P.blk + (uint64_t)blockIdx.x * P.blocks, (n + kRunBlock - 1) / kRunBlock, P.cnt + blockIdx.x);
}

__global__ void __launch_bounds__(kRunBlock) k_run_emit(const SgPred* preds, uint32_t chunk) {
    __shared__ uint32_t ws[32][kSgMaxStages];
    const SgPred& P = preds[blockIdx.y];
    grid_trigger();
    grid_wait();
    if (P.dense) return;
    const uint32_t n = chunk_values(P, chunk);
    if ((uint64_t)blockIdx.x * kRunBlock >= n) return;
    const uint32_t i = blockIdx.x * kRunBlock + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = 0;
    const int cb = i < n ? common_bits(P, P.u + (uint64_t)chunk * P.chunk, i, &x) : 32;
    const uint32_t S = P.stages - 1;
    for (uint32_t s = 0; s < S; s++) {
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, cb < (int)P.lev[s]);
        if (lane == 0) ws[warp][s] = __popc(b);
    }
    __syncthreads();
    if (threadIdx.x < S) {
        uint32_t at = P.blk[(uint64_t)threadIdx.x * P.blocks + blockIdx.x];
        for (int w = 0; w < 32; w++) {
            const uint32_t c = ws[w][threadIdx.x];
            ws[w][threadIdx.x] = at;
            at += c;
        }
    }
    __syncthreads();
    uint32_t parent = 0;          // the run of the stage before that value i lies in
    for (uint32_t s = 0; s < S; s++) {
        const bool f = cb < (int)P.lev[s];
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, f);
        const uint32_t r = ws[warp][s] + __popc(b & lanemask_lt()) + (f ? 1u : 0u) - 1u;
        if (f) {
            P.pre[P.pre_off[s] + r] = x >> (P.n - P.lev[s]);
            P.par[P.pre_off[s] + r] = parent;
        }
        parent = r;
    }
    if (i < n) P.par_last[i] = parent;
}

// ------------------------------------------------------------------ the walks

struct StageParams {
    AesParams aes;
    const uint32_t* te0;
    const SgPred* preds;
    const DevKey* keys;
    uint32_t n_preds;
    uint32_t stage;
    uint32_t chunk;
};

// Levels a .. b - 1 of one key's walk at x (n bits), from the node's seed s, control bit t
// and, for a DCF, value sum V; the steps are those of dpf_walk / dcf_walk.
template <bool DCF, class Tab>
__device__ __forceinline__ void walk_levels(const Tab& T, const AesParams& A, const DevKey* K, uint32_t x, int n, int a,
                                            int b, uint32_t s[4], uint32_t& t, uint32_t& V) {
    const uint32_t tl = __ldg(&K->tl), tr = __ldg(&K->tr), party = __ldg(&K->party);
#pragma unroll 1
    for (int i = a; i < b; i++) {
        const uint4 cw = __ldg(reinterpret_cast<const uint4*>(K->scw[i]));
        const uint32_t dir = (x >> (n - 1 - i)) & 1u, m = 0u - dir;
        uint32_t o[4];
        aes_sel(T, A.rk_st, A.d_st, m, s, o);
        if (DCF) {
            const uint32_t v0 = aes_sel_w0(T, A.rk_v, A.d_v, m, s);
            const uint32_t term = (v0 ^ s[0]) + (t ? __ldg(&K->vcw[i]) : 0u);
            V += party ? 0u - term : term;
        }
#pragma unroll
        for (int w = 0; w < 4; w++) o[w] ^= s[w];
        uint32_t tn = o[0] & 1u;
        o[0] &= ~1u;
        const uint32_t tm = 0u - t;
        s[0] = o[0] ^ (cw.x & tm);
        s[1] = o[1] ^ (cw.y & tm);
        s[2] = o[2] ^ (cw.z & tm);
        s[3] = o[3] ^ (cw.w & tm);
        tn ^= t & (((dir ? tr : tl) >> i) & 1u);
        t = tn;
    }
}

// first run of a dense stage: the prefix of the chunk's first value
__device__ __forceinline__ uint32_t dense_base(const SgPred& P, uint32_t chunk, uint32_t level) {
    return level == 0 ? 0u : (uint32_t)(((uint64_t)chunk * P.chunk) >> (P.n - level));
}

__device__ __forceinline__ uint32_t stage_runs(const SgPred& P, uint32_t chunk, uint32_t s) {
    const uint32_t n = chunk_values(P, chunk);
    if (n == 0) return 0u;
    if (!P.dense) return P.cnt[s];
    return (uint32_t)(((uint64_t)chunk * P.chunk + n - 1) >> (P.n - P.lev[s])) - dense_base(P, chunk, P.lev[s]) + 1u;
}

__device__ __forceinline__ void load_state(const SgPred& P, uint32_t buf, uint32_t key, uint32_t r, bool dcf,
                                           uint32_t s[4], uint32_t& t, uint32_t& V) {
    const uint64_t at = (uint64_t)key * P.cap[buf] + r;
    const uint4 q = P.st[buf][at];
    t = q.x & 1u;
    s[0] = q.x & ~1u; s[1] = q.y; s[2] = q.z; s[3] = q.w;
    V = dcf ? P.v[buf][at] : 0u;
}

// work units of the launch's predicates, 32 lanes each: first[p] .. first[p + 1] - 1 belong to p
__device__ __forceinline__ void unit_table(unsigned long long* first, uint32_t n_preds, unsigned long long mine) {
    if (threadIdx.x < n_preds) first[threadIdx.x + 1] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        first[0] = 0;
        for (uint32_t p = 0; p < n_preds; p++) first[p + 1] += first[p];
    }
    __syncthreads();
}

// One stage but the last: a warp takes 32 runs of one key.
__global__ void __launch_bounds__(kStageThreads, 1) k_stage(const __grid_constant__ StageParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned long long first[kMaxRoundPreds + 1];
    grid_trigger();
    fill_tables(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    unsigned long long units = 0;
    if (threadIdx.x < P.n_preds) {
        const SgPred& D = P.preds[threadIdx.x];
        if (P.stage + 1 < D.stages)
            units = (unsigned long long)D.n_keys * ((stage_runs(D, P.chunk, P.stage) + 31) / 32);
    }
    unit_table(first, P.n_preds, units);
    const unsigned long long total = first[P.n_preds];
    if (total == 0) return;
    const SmemTab T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t lane = threadIdx.x & 31, st = P.stage;
    const unsigned long long step = (unsigned long long)gridDim.x * (kStageThreads / 32);
    // consecutive units go to different SMs, so a short last wave is spread evenly
    for (unsigned long long w = (unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < total; w += step) {
        uint32_t p = 0;
        while (first[p + 1] <= w) p++;
        const SgPred& D = P.preds[p];
        const uint32_t runs = stage_runs(D, P.chunk, st), per_key = (runs + 31) / 32;
        const uint32_t local = (uint32_t)(w - first[p]), key = local / per_key;
        const uint32_t r = (local - key * per_key) * 32 + lane;
        if (r >= runs) continue;
        const bool dcf = D.kind == OBLIVGM_PRED_RANGE;
        const int a = st ? D.lev[st - 1] : 0, b = D.lev[st], n = (int)D.n;
        const DevKey* K = P.keys + D.key_begin + key;
        uint32_t pre, par;
        if (D.dense) {
            pre = dense_base(D, P.chunk, (uint32_t)b) + r;
            par = st ? (pre >> (b - a)) - dense_base(D, P.chunk, (uint32_t)a) : 0u;
        } else {
            pre = D.pre[D.pre_off[st] + r];
            par = D.par[D.pre_off[st] + r];
        }
        uint32_t s[4], t, V = 0;
        if (st == 0) {
#pragma unroll
            for (int j = 0; j < 4; j++) s[j] = __ldg(&K->seed[j]);
            t = __ldg(&K->party);
        } else {
            load_state(D, (st - 1) & 1, key, par, dcf, s, t, V);
        }
        const uint32_t x = pre << (n - b);      // b >= 1
        if (dcf) walk_levels<true>(T, P.aes, K, x, n, a, b, s, t, V);
        else walk_levels<false>(T, P.aes, K, x, n, a, b, s, t, V);
        const uint64_t at = (uint64_t)key * D.cap[st & 1] + r;
        D.st[st & 1][at] = make_uint4(s[0] | t, s[1], s[2], s[3]);
        if (dcf) D.v[st & 1][at] = V;
    }
}

// The last stage: a warp takes 32 distinct values of one output slot (a server's two key
// halves, or one key of a raw evaluation) and walks the slot's keys one after another, or, in a
// launch of few such units, one of its keys (SgPred::parts): a slot of a range predicate is a
// chain of four walks that leaves most warps without work.
__global__ void __launch_bounds__(kStageThreads, 1) k_stage_last(const __grid_constant__ StageParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned long long first[kMaxRoundPreds + 1];
    grid_trigger();
    fill_tables(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    unsigned long long units = 0;
    if (threadIdx.x < P.n_preds) {
        const SgPred& D = P.preds[threadIdx.x];
        units = (unsigned long long)D.slots * D.parts * ((chunk_values(D, P.chunk) + 31) / 32);
    }
    unit_table(first, P.n_preds, units);
    const unsigned long long total = first[P.n_preds];
    if (total == 0) return;
    const SmemTab T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t lane = threadIdx.x & 31;
    const unsigned long long step = (unsigned long long)gridDim.x * (kStageThreads / 32);
    for (unsigned long long w = (unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < total; w += step) {
        uint32_t p = 0;
        while (first[p + 1] <= w) p++;
        const SgPred& D = P.preds[p];
        const uint32_t vals = chunk_values(D, P.chunk), per_slot = (vals + 31) / 32;
        const uint32_t local = (uint32_t)(w - first[p]), sp = local / per_slot;
        const uint32_t slot = sp / D.parts, part = sp - slot * D.parts;
        const uint32_t i = (local - sp * per_slot) * 32 + lane;
        if (i >= vals) continue;
        const bool dcf = D.kind == OBLIVGM_PRED_RANGE;
        const uint32_t S = D.stages, nk = D.n_keys / D.slots, nk_part = nk / D.parts;
        const int n = (int)D.n, a = S > 1 ? D.lev[S - 2] : 0;
        const uint64_t gi = (uint64_t)P.chunk * D.chunk + i;
        uint32_t x, par = 0;
        if (D.dense) {
            x = (uint32_t)gi;
            if (S > 1) par = (x >> (n - a)) - dense_base(D, P.chunk, (uint32_t)a);
        } else {
            x = (D.u[gi] + D.delta) & D.mask;
            if (S > 1) par = D.par_last[i];
        }
        uint32_t z = 0;
#pragma unroll 1
        for (uint32_t kk = part * nk_part; kk < (part + 1) * nk_part; kk++) {
            const uint32_t key = slot * nk + kk;
            const DevKey* K = P.keys + D.key_begin + key;
            const uint32_t party = __ldg(&K->party);
            uint32_t s[4], t, V = 0;
            if (S == 1) {
#pragma unroll
                for (int j = 0; j < 4; j++) s[j] = __ldg(&K->seed[j]);
                t = party;
            } else {
                load_state(D, (S - 2) & 1, key, par, dcf, s, t, V);
            }
            if (dcf) walk_levels<true>(T, P.aes, K, x, n, a, n, s, t, V);
            else walk_levels<false>(T, P.aes, K, x, n, a, n, s, t, V);
            const uint32_t term = s[1] + (t ? __ldg(&K->cw_final) : 0u);   // Convert(s_n): bytes 4..7
            z += V + (party ? 0u - term : term);
            // RANGE: the public constant c * beta' joins party 0's half once (sub 0 of the half)
            if (dcf && (kk & 1u) == 0 && party == 0) z += D.cbeta;
        }
        D.z[gi * D.z_elem + slot * D.z_slot + 4 * part] = z;
    }
}

// ------------------------------------------------------------------ re-share and fold

struct CombineParams {
    uint32_t rk_prf[3][44];
    const uint32_t* te0;
    const SgGroup* groups;
    const SgFold* folds;
    uint64_t items;             // tiles of blockDim.x * per_thread elements
    uint32_t n_groups;
    uint32_t per_thread;        // elements per thread of a tile
};

// Dynamic shared memory: the tables, then a tile's counter prefixes, (predicate, pass, PRF key,
// 256 elements) each 5 words.
constexpr int kPrefixWords = 5;
constexpr uint32_t kMaxTileSteps = 64;      // predicates of a group entry x elements per thread
static_assert(kMaxTileSteps >= kMaxRoundPreds, "a round's predicates may all be of one group");
constexpr int kMaxPrefixes = (int)kMaxTileSteps * 6 * (kStageThreads / 256);
constexpr int kCombineSmem = kTableBytes + kMaxPrefixes * kPrefixWords * 4;

// index of element e's value in a predicate's sums.  What earlier kernels of the chain wrote is
// read with plain loads: it changes while this kernel waits for them, which the read-only path
// does not allow.
__device__ __forceinline__ uint32_t value_index(const SgGroup& G, const SgFold& D, uint64_t e) {
    if (D.index == kIndexRank) return D.rank[e];
    if (D.index == kIndexElem) return (uint32_t)e;
    const uint64_t row = (uint64_t)D.attr * G.stride + e;
    return (__ldg(G.share[0] + row) + __ldg(G.share[1] + row) + __ldg(G.share[2] + row) + D.radd) & D.mask;
}

// the three servers' sums of value `at`, over their parts
template <bool SPLIT>
__device__ __forceinline__ uint4 load_sums(const SgFold& D, uint32_t at) {
    if (!SPLIT) return reinterpret_cast<const uint4*>(D.z)[at];
    const uint4* z = reinterpret_cast<const uint4*>(D.z) + (uint64_t)at * (D.more + 1);
    uint4 s = z[0];
#pragma unroll 1
    for (uint32_t w = 1; w <= D.more; w++) {
        const uint4 a = z[w];
        s.x += a.x; s.y += a.y; s.z += a.z;
    }
    return s;
}

// One thread per element of a tile: for each of the round's predicates the three servers' sums
// at the element's value (z_i), r_i = z_i + F(k_i) - F(k_{i-1}) (Sec. III-B), and the fold into the
// group's result with its re-share (Sec. V-D).  The PRF words bound it: 3 per predicate and 3
// per fold, from the shared-memory tables.  Two things keep that pipe busy:
//   * the counters' low byte runs over 256 consecutive elements, so a tile first computes what
//     those share (ctr_prefix) and an element's word takes 121 lookups instead of 148;
//   * the two dependent reads of the sums (rank, then a random 16 bytes) are issued one step
//     ahead, the step after a tile's last predicate being the next tile's first.
template <bool SPLIT>
__global__ void __launch_bounds__(kStageThreads, 1) k_combine(const __grid_constant__ CombineParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint4* pre_c = reinterpret_cast<uint4*>(smem + kTableBytes);
    uint32_t* pre_n = reinterpret_cast<uint32_t*>(pre_c + kMaxPrefixes);
    grid_trigger();
    fill_tables(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    __syncthreads();
    const SmemTab T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t tile = blockDim.x * P.per_thread, subs = tile >> 8;   // 256-element parts of a tile
    uint32_t g = 0;
    while (g + 1 < P.n_groups && P.groups[g + 1].item_begin <= blockIdx.x) g++;
    uint4 zq = make_uint4(0, 0, 0, 0);
    {
        const SgGroup& G = P.groups[g];
        const uint64_t e = (blockIdx.x - G.item_begin) * tile + threadIdx.x;
        const SgFold& D = P.folds[G.pred_begin];
        if (e < G.n_elems) zq = load_sums<SPLIT>(D, value_index(G, D, e));
    }
    for (uint64_t w = blockIdx.x; w < P.items;) {
        const SgGroup& G = P.groups[g];
        const uint64_t e0 = (w - G.item_begin) * tile;
        for (uint32_t q = threadIdx.x; q < G.n_preds * 6 * subs; q += blockDim.x) {
            // prefix q = ((predicate * subs + 256 elements) * 2 + pass) * 3 + key
            const uint32_t key = q % 3, pass = q / 3 % 2, k = q / 6 / subs;
            const uint64_t b = e0 + 256u * (q / 6 % subs);
            const uint32_t in[4] = {(uint32_t)b, (uint32_t)(b >> 32),
                                    (P.folds[G.pred_begin + k].step + 64u * pass) | (G.table_id << 16), G.query_id};
            const CtrPrefix c = ctr_prefix(T, P.rk_prf[key], in);
            pre_c[q] = c.c;
            pre_n[q] = c.n0;
        }
        __syncthreads();
        // the tile after this one
        const uint64_t w2 = w + gridDim.x;
        uint32_t g2 = g;
        while (g2 + 1 < P.n_groups && P.groups[g2 + 1].item_begin <= w2) g2++;
        for (uint32_t at_tile = threadIdx.x; at_tile < tile; at_tile += blockDim.x) {
            const uint64_t e = e0 + at_tile;
            const uint32_t sub = at_tile >> 8;
            const bool mine = e < G.n_elems, tile_end = at_tile + blockDim.x >= tile;
            uint32_t acc[3] = {0, 0, 0};
            if (mine && !G.first) {
#pragma unroll
                for (int i = 0; i < 3; i++) acc[i] = G.out[i][e];
            }
            for (uint32_t k = 0; k < G.n_preds; k++) {
                const SgFold& D = P.folds[G.pred_begin + k];
                uint32_t z[3] = {zq.x, zq.y, zq.z};
                // the next step's sums: its index now, the sums themselves after a PRF word
                const bool last = k + 1 == G.n_preds, leave = last && tile_end;
                const SgGroup& G2 = leave ? P.groups[g2] : G;
                const SgFold& D2 = P.folds[G2.pred_begin + (last ? 0u : k + 1)];
                const uint64_t e2 = leave ? (w2 - G2.item_begin) * tile + threadIdx.x : last ? e + blockDim.x : e;
                const bool more = (!leave || w2 < P.items) && e2 < G2.n_elems;
                const uint32_t at2 = more ? value_index(G2, D2, e2) : 0u;
                if (!mine) {
                    if (more) zq = load_sums<SPLIT>(D2, at2);
                    continue;
                }
                const bool fold = !(G.first && k == 0);
#pragma unroll 1
                for (int pass = 0; pass < (fold ? 2 : 1); pass++) {
                    uint32_t r[3] = {z[0], z[1], z[2]};
#pragma unroll 1
                    for (int i = 0; i < 3; i++) {
                        const uint32_t at_pre = ((k * subs + sub) * 2 + pass) * 3 + i;
                        const CtrPrefix c{pre_n[at_pre], pre_c[at_pre]};
                        const uint32_t f = ctr_w0(T, P.rk_prf[i], c, (uint32_t)e);   // F keeps bytes 0..3
                        if (pass == 0 && i == 0 && more) zq = load_sums<SPLIT>(D2, at2);
                        r[0] += i == 0 ? f : (i == 2 ? 0u - f : 0u);
                        r[1] += i == 1 ? f : (i == 0 ? 0u - f : 0u);
                        r[2] += i == 2 ? f : (i == 1 ? 0u - f : 0u);
                    }
                    if (fold && pass == 0) {
#pragma unroll
                        for (int i = 0; i < 3; i++) {
                            const int i1 = (i + 1) % 3;
                            const uint32_t pr = acc[i] * r[i] + acc[i] * r[i1] + acc[i1] * r[i];
                            z[i] = D.lin * (acc[i] + r[i]) + D.prod * pr;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 3; i++) acc[i] = r[i];
                    }
                }
            }
            if (mine) {
#pragma unroll
                for (int i = 0; i < 3; i++) G.out[i][e] = acc[i];
            }
        }
        __syncthreads();
        w = w2;
        g = g2;
    }
}

// ------------------------------------------------------------------ raw evaluation

// out[k * n_points + i] = z of key k at point i's value; grid y strides over the keys
struct GatherParams {
    const SgCol* col;
    const uint32_t* z;
    uint32_t* out;
    uint64_t n_points, vals;
    uint32_t n_keys;
};

__global__ void __launch_bounds__(256) k_gather_raw(const __grid_constant__ GatherParams P) {
    const SgCol& C = *P.col;
    grid_trigger();
    grid_wait();
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < P.n_points; i += (uint64_t)gridDim.x * 256) {
        const uint32_t at = C.passes ? C.rank[i] : __ldg(C.share[0] + i) & C.mask;
        for (uint32_t k = blockIdx.y; k < P.n_keys; k += gridDim.y)
            P.out[k * P.n_points + i] = P.z[k * P.vals + at];
    }
}

// ------------------------------------------------------------------ planning

// GB300 figures the plan weighs: a DPF / DCF level step of one key at the T-table lookup rate,
// a PRF word, a launch (with its table fill) and a key of a sort pass.
constexpr double kDpfStep = 16.7e-12, kDcfStep = 32.2e-12, kPrfWord = 15.5e-12, kLaunch = 4.0e-6;
// a level step of a thread on its own, and what k_filter takes on top (of 564 plans of 1,000 to
// 100,000 elements, one to five predicates and n = 8 to 32, timed both ways, the estimates
// pick the slower one, by 5 % and more, in 25, each by staying fused)
constexpr double kDpfLatency = 0.57e-6, kDcfLatency = 0.92e-6, kFusedFixed = 20e-6;
constexpr double kSortKeyPass = 12e-12;
// what a staged raw evaluation takes beside its launches: scratch, descriptors and their copy
constexpr double kRawFixed = 3.0e-6;
constexpr uint64_t kMaxElems = 1ull << 28;
constexpr int kMaxDenseBits = 24;
// A launch whose last stages have fewer units (32 values of one slot) than this for each SM, one and
// a half for each of its 24 warps, runs a unit per key there: a range of 5,000 values, n = 32,
// 167 -> 135 us, of 2^8 (n = 8) 40 -> 17 us; 2^16 values in 1.7 units a warp lose 3 %.
constexpr uint64_t kSplitUnitsPerSm = 3 * (kStageThreads / 32) / 2;

// distinct l-bit prefixes of n_vals uniform values, the most that a column can be expected to have
double expected_nodes(double n_vals, int l) {
    const double cells = std::ldexp(1.0, l);
    return -cells * std::expm1(-n_vals / cells);
}

// The level boundaries: shortest path over the levels, where a stage a -> b costs one step per
// level and node of level b, plus a state's round trip (about 15 % of a DCF step) and a launch.
// Real columns repeat values and prefixes, and the more so the nearer the root, so deep
// boundaries are worth a little more than uniform values would say.
double choose_stages(double n_vals, bool dense, int n, double step_s, std::vector<uint8_t>* lev) {
    std::vector<double> nodes(n + 1), best(n + 1, 1e300);
    std::vector<int> from(n + 1, 0);
    for (int l = 0; l <= n; l++)
        nodes[l] = dense ? std::ldexp(1.0, l) : expected_nodes(n_vals, l) * (0.75 + 0.25 * l / n);
    best[0] = 0;
    for (int b = 1; b <= n; b++)
        for (int a = 0; a < b; a++) {
            const double c = best[a] + nodes[b] * step_s * ((b - a) + (b < n ? 0.15 : 0.05)) + kLaunch;
            if (c < best[b]) { best[b] = c; from[b] = a; }
        }
    lev->clear();
    for (int b = n; b > 0; b = from[b]) lev->push_back((uint8_t)b);
    std::reverse(lev->begin(), lev->end());
    return best[n];
}

size_t up256(size_t b) { return (b + 255) / 256 * 256; }

// distinct values a predicate's column can have, and those of one chunk
uint64_t max_values(const SgCol& c) {
    const uint64_t domain = (uint64_t)c.mask + 1;
    return c.passes == 0 ? domain : std::min<uint64_t>(c.n, domain);
}

// Runs a chunk can have after stage s.  A sparse chunk's values ascend in u, so in x^ = u + delta
// they wrap once past 2^n: the prefix that holds the first value can come up again at the end.
uint64_t max_runs(const SgPred& p, const SgCol& c, uint32_t s) {
    return std::min<uint64_t>(std::min<uint64_t>(p.chunk, max_values(c)), (1ull << p.lev[s]) + (p.dense ? 0 : 1));
}

// Sort tiles: large ones once the sparse columns fill the SMs' tiles several times over.
void choose_tiles(Staged* sg) {
    uint64_t keys = 0;
    for (const SgCol& C : sg->cols) keys += C.passes ? C.n : 0;
    const uint32_t large = kSortThreads * kSortItemsLarge, small = kSortThreads * kSortItemsSmall;
    sg->sort_large = keys >= 512ull * large;
    sg->sort_tiles = 0;
    for (SgCol& C : sg->cols) {
        C.tiles = (uint32_t)((C.n + (sg->sort_large ? large : small) - 1) / (sg->sort_large ? large : small));
        if (C.passes) sg->sort_tiles = std::max(sg->sort_tiles, C.tiles);
    }
}

// Lays out a sparse column / a predicate from byte `at` on and returns the end; sets the
// pointers when there is a base.
size_t layout_col(SgCol* c, unsigned char* base, size_t at) {
    const auto take = [&](size_t b) { unsigned char* p = base + at; at += up256(b); return reinterpret_cast<uint32_t*>(p); };
    if (c->passes == 0) return at;
    for (int j = 0; j < 2; j++) c->key[j] = take(c->n * 4);
    for (int j = 0; j < 2; j++) c->idx[j] = take(c->n * 4);
    c->rank = take(c->n * 4);
    c->hist = take((size_t)c->tiles * 256 * 4);
    c->tot = take(256 * 4);
    c->m = take(4);
    return at;
}

size_t layout_pred(SgPred* p, const SgCol& c, unsigned char* base, size_t at) {
    const auto take = [&](size_t b) { unsigned char* q = base + at; at += up256(b); return reinterpret_cast<uint32_t*>(q); };
    const uint64_t vals = max_values(c);
    p->z = take(vals * 4 * (p->z_elem > 1 ? p->z_elem : p->n_keys));
    for (int b = 0; b < 2; b++) {
        p->st[b] = reinterpret_cast<uint4*>(take((size_t)p->n_keys * p->cap[b] * 16));
        p->v[b] = p->kind == OBLIVGM_PRED_RANGE ? take((size_t)p->n_keys * p->cap[b] * 4) : nullptr;
    }
    if (p->dense) return at;
    uint64_t runs = 0;
    for (uint32_t s = 0; s + 1 < p->stages; s++) {
        p->pre_off[s] = runs;
        runs += max_runs(*p, c, s);
    }
    p->u = c.key[(c.passes + 1) & 1];
    p->m = c.m;
    p->pre = take(runs * 4);
    p->par = take(runs * 4);
    p->par_last = take(std::min<uint64_t>(p->chunk, vals) * 4);
    p->blk = take((size_t)p->stages * p->blocks * 4);
    p->cnt = take((size_t)p->stages * 4);
    return at;
}

}  // namespace

// Elements per tile of the combine: the CTA width whose waves take the least time (a wave of t
// threads takes as long as its lookups, or at 384 threads and less as long as an element's chain
// of PRF words: 100,003 elements in one wave of 768 threads 35 us, in two of 512 46 us), and
// several elements per thread, so that a tile's barriers are rare, where every SM still gets a
// few tiles.
CombineShape combine_shape(uint64_t elems, uint32_t most_preds, int sm_count) {
    CombineShape c;
    uint64_t best = ~0ull;
    for (uint32_t t = 256; t <= (uint32_t)kStageThreads; t += 256) {
        const uint64_t waves = ((elems + t - 1) / t + sm_count - 1) / sm_count, cost = waves * std::max(t, 384u);
        if (cost <= best) { best = cost; c.threads = t; }
    }
    const uint64_t spread = elems / (6ull * kStageThreads * sm_count);
    c.per_thread = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>({8, spread, kMaxTileSteps / most_preds}));
    return c;
}

uint64_t combine_tiles(const CombineShape& c, SgGroup* groups, uint32_t n_groups) {
    const uint64_t tile = (uint64_t)c.threads * c.per_thread;
    uint64_t items = 0;
    for (uint32_t g = 0; g < n_groups; g++) {
        groups[g].item_begin = items;
        items += (groups[g].n_elems + tile - 1) / tile;
    }
    return items;
}

void launch_combine(oblivgm_ctx* ctx, const CombineShape& c, const SgGroup* groups, uint32_t n_groups,
                    const SgFold* folds, bool split, uint64_t items, cudaStream_t s) {
    CombineParams F{};
    std::memcpy(F.rk_prf, ctx->rk_prf, sizeof F.rk_prf);
    F.te0 = ctx->d_te0;
    F.folds = folds;
    F.groups = groups;
    F.n_groups = n_groups;
    F.items = items;
    F.per_thread = c.per_thread;
    launch_after(split ? k_combine<true> : k_combine<false>, (unsigned)std::min<uint64_t>((uint64_t)ctx->sm_count, items), c.threads, kCombineSmem, s, F);
    ctx->launches++;
}

bool staged_plan(const std::vector<GroupDesc>& groups, const std::vector<PredDesc>& preds, size_t n_keys, int sm_count,
                 const StagedLimits& limits, double fixed, double wp_seconds, Staged* sg) {
    *sg = Staged{};
    sg->n_keys = (uint32_t)n_keys;
    // columns: a share row of the first set
    std::map<const uint32_t*, uint32_t> col_of;
    std::vector<double> col_steps;                      // seconds per node of one level, over its predicates' keys
    std::vector<uint32_t> pred_col(preds.size());
    double fused = 0, combine = 0, chain = 0;
    for (const GroupDesc& G : groups) {
        if (G.n_elems == 0) continue;
        if (G.n_elems > kMaxElems) return false;
        double group_chain = 0;
        for (uint32_t k = 0; k < G.n_preds; k++) {
            const PredDesc& D = preds[G.pred_begin + k];
            const uint64_t row = (uint64_t)D.attr * G.stride;
            const auto ins = col_of.emplace(G.share[0] + row, (uint32_t)sg->cols.size());
            if (ins.second) {
                SgCol c{};
                for (int j = 0; j < 3; j++) c.share[j] = G.share[j] + row;
                c.n = G.n_elems;
                c.radd = D.r[0] + D.r[1] + D.r[2];
                c.mask = D.n_bits >= 32 ? 0xFFFFFFFFu : ((1u << D.n_bits) - 1u);
                c.passes = (D.n_bits + 7) / 8;
                sg->cols.push_back(c);
                col_steps.push_back(0);
            }
            pred_col[G.pred_begin + k] = ins.first->second;
            const double step = D.kind == OBLIVGM_PRED_EQ ? 6 * kDpfStep : 12 * kDcfStep;
            col_steps[ins.first->second] += step;
            fused += step * D.n_bits * (double)G.n_elems;
            combine += (k ? 6 : 3) * kPrfWord * (double)G.n_elems;
            group_chain += D.n_bits * (D.kind == OBLIVGM_PRED_EQ ? 6 * kDpfLatency : 12 * kDcfLatency);
        }
        chain = std::max(chain, group_chain);
    }
    // a column is a row of the sort kernels' grids
    if (sg->cols.empty() || sg->cols.size() > 65535) { *sg = Staged{}; return false; }
    // per column: dense when the whole domain costs no more than its sorted values
    std::vector<std::vector<uint8_t>> lev(sg->cols.size());
    double staged = 0;
    size_t most_stages = 0;
    for (size_t c = 0; c < sg->cols.size(); c++) {
        SgCol& C = sg->cols[c];
        const int n = __builtin_popcount(C.mask);
        std::vector<uint8_t> ld;
        double cd = 1e300;
        if (n <= kMaxDenseBits) cd = choose_stages(0, true, n, col_steps[c], &ld);
        const double sort = (double)C.n * kSortKeyPass * C.passes;
        const double cs = choose_stages((double)C.n, false, n, col_steps[c], &lev[c]) + sort;
        const bool dense = cd <= cs + 6 * kLaunch;
        if (dense) {
            C.passes = 0;
            lev[c] = ld;
        }
        // the columns' launches are shared, so they are counted once below
        staged += (dense ? cd : cs) - kLaunch * (double)lev[c].size();
        most_stages = std::max(most_stages, lev[c].size());
        sg->sort_passes = std::max(sg->sort_passes, C.passes);
    }
    staged += kLaunch * (double)(most_stages + 1 + (sg->sort_passes ? 6 + 3 * sg->sort_passes : 0));
    // further rounds (of predicates; of bytes only where the walks take far longer) launch anew, each
    // launch while the one before runs
    const double more_rounds = (double)((preds.size() - 1) / kMaxRoundPreds);
    staged += 0.5 * kLaunch * more_rounds * (double)(most_stages + 1 + (sg->sort_passes ? 3 : 0));
    // against k_filter, whose threads walk an element's keys one after another (at least its chain),
    // or the walk-parallel kernel's schedule
    const double other = wp_seconds > 0 ? wp_seconds : kFusedFixed + std::max(fused + combine, chain);
    if (fixed + 1.05 * staged + 1.5 * combine > 0.95 * other) { *sg = Staged{}; return false; }

    choose_tiles(sg);
    size_t col_end = 0;
    for (SgCol& C : sg->cols) col_end = layout_col(&C, nullptr, col_end);
    uint64_t last_units = 0;
    for (size_t q = 0; q < preds.size(); q++)
        last_units += 3 * ((max_values(sg->cols[pred_col[q]]) + 31) / 32);
    sg->split = last_units < kSplitUnitsPerSm * (uint64_t)sm_count;
    // predicates in group order, cut into rounds whose states fit limits.round_bytes
    size_t at = col_end, most = col_end;
    StagedRound R{};
    const auto close = [&]() {
        if (R.n_preds) sg->rounds.push_back(R);
        R = StagedRound{};
        R.pred_begin = (uint32_t)sg->preds.size();
        R.group_begin = (uint32_t)sg->groups.size();
        at = col_end;
    };
    for (const GroupDesc& G : groups) {
        if (G.n_elems == 0) continue;
        bool open = false;          // the group has an entry in the current round
        for (uint32_t k = 0; k < G.n_preds; k++) {
            const PredDesc& D = preds[G.pred_begin + k];
            const SgCol& C = sg->cols[pred_col[G.pred_begin + k]];
            SgPred p{};
            p.kind = D.kind; p.n = D.n_bits; p.n_keys = D.n_keys; p.key_begin = D.key_begin;
            p.mask = C.mask;
            p.delta = D.r[0] + D.r[1] + D.r[2] - C.radd;
            p.cbeta = D.cbeta;
            p.dense = C.passes == 0;
            p.col = pred_col[G.pred_begin + k];
            p.slots = 3;
            p.parts = sg->split ? D.n_keys / 3 : 1;
            p.z_elem = 4 * p.parts;
            p.z_slot = 1;
            p.stages = (uint32_t)lev[p.col].size();
            std::copy(lev[p.col].begin(), lev[p.col].end(), p.lev);
            const uint64_t vals = max_values(C);
            p.chunk = kRunBlock;
            while (p.chunk < vals && p.chunk < limits.chunk) p.chunk <<= 1;
            p.blocks = p.chunk / kRunBlock;
            for (uint32_t s = 0; s + 1 < p.stages; s++) p.cap[s & 1] = std::max(p.cap[s & 1], (uint32_t)max_runs(p, C, s));
            if (R.n_preds && (R.n_preds >= kMaxRoundPreds || layout_pred(&p, C, nullptr, at) - col_end > limits.round_bytes)) {
                close();
                open = false;
            }
            at = layout_pred(&p, C, nullptr, at);
            most = std::max(most, at);
            if (!open) {
                SgGroup g{};
                for (int j = 0; j < 3; j++) { g.share[j] = G.share[j]; g.out[j] = G.out[j]; }
                g.stride = G.stride; g.n_elems = G.n_elems;
                g.query_id = G.query_id; g.table_id = G.table_id;
                g.pred_begin = (uint32_t)sg->preds.size();
                g.first = k == 0 ? 1u : 0u;
                sg->groups.push_back(g);
                R.n_groups++;
                open = true;
            }
            sg->groups.back().n_preds++;
            SgFold f{};
            f.step = D.step; f.lin = D.lin; f.prod = D.prod; f.attr = D.attr;
            f.radd = D.r[0] + D.r[1] + D.r[2];
            f.mask = p.mask;
            f.index = p.dense ? kIndexDense : kIndexRank;
            f.more = p.parts - 1;
            sg->preds.push_back(p);
            sg->folds.push_back(f);
            R.n_preds++;
            R.max_stages = std::max(R.max_stages, p.stages);
            R.chunks = std::max<uint32_t>(R.chunks, (uint32_t)((vals + p.chunk - 1) / p.chunk));
            if (!p.dense) {
                R.sparse = 1;
                R.max_blocks = std::max(R.max_blocks, p.blocks);
            }
        }
    }
    close();
    uint32_t most_preds = 1;
    uint64_t elems = 0;
    for (const SgGroup& g : sg->groups) {
        most_preds = std::max(most_preds, g.n_preds);
        elems += g.first ? g.n_elems : 0;
    }
    sg->shape = combine_shape(elems, most_preds, sm_count);
    for (StagedRound& r : sg->rounds) r.items = combine_tiles(sg->shape, sg->groups.data() + r.group_begin, r.n_groups);
    sg->scratch_bytes = most;
    if (sg->scratch_bytes > limits.cap) { *sg = Staged{}; return false; }
    sg->off_preds = up256(sg->cols.size() * sizeof(SgCol));
    sg->off_folds = sg->off_preds + up256(sg->preds.size() * sizeof(SgPred));
    sg->off_groups = sg->off_folds + up256(sg->folds.size() * sizeof(SgFold));
    sg->off_keys = sg->off_groups + up256(sg->groups.size() * sizeof(SgGroup));
    sg->image_bytes = sg->off_keys + up256(n_keys * sizeof(DevKey));
    return true;
}

void staged_image(Staged* sg, const DevKey* keys, unsigned char* scratch, std::vector<unsigned char>* bytes) {
    size_t col_end = 0;
    for (SgCol& C : sg->cols) col_end = layout_col(&C, scratch, col_end);
    for (const StagedRound& R : sg->rounds) {
        size_t at = col_end;
        for (uint32_t q = R.pred_begin; q < R.pred_begin + R.n_preds; q++) {
            SgPred& p = sg->preds[q];
            const SgCol& C = sg->cols[p.col];
            at = layout_pred(&p, C, scratch, at);
            if (sg->raw) continue;
            sg->folds[q].rank = C.rank;
            sg->folds[q].z = p.z;
        }
    }
    bytes->assign(sg->image_bytes, 0);
    std::memcpy(bytes->data(), sg->cols.data(), sg->cols.size() * sizeof(SgCol));
    std::memcpy(bytes->data() + sg->off_preds, sg->preds.data(), sg->preds.size() * sizeof(SgPred));
    std::memcpy(bytes->data() + sg->off_folds, sg->folds.data(), sg->folds.size() * sizeof(SgFold));
    std::memcpy(bytes->data() + sg->off_groups, sg->groups.data(), sg->groups.size() * sizeof(SgGroup));
    if (keys) std::memcpy(bytes->data() + sg->off_keys, keys, sg->n_keys * sizeof(DevKey));
}

namespace {

template <int ITEMS>
void launch_sort_tiles(const Staged& sg, const SgCol* cols, cudaStream_t s) {
    const unsigned nc = (unsigned)sg.cols.size();
    const dim3 grid(sg.sort_tiles, nc);
    for (uint32_t p = 0; p < sg.sort_passes; p++) {
        if (p == 0) k_sort_hist<ITEMS><<<grid, kSortThreads, 0, s>>>(cols, p);
        else launch_after(k_sort_hist<ITEMS>, grid, kSortThreads, 0, s, cols, p);
        launch_after(k_sort_scan, dim3(256, nc), 256, 0, s, cols, p);
        launch_after(k_sort_scatter<ITEMS>, grid, kSortThreads, 0, s, cols, p);
    }
    launch_after(k_uniq_count<ITEMS>, grid, kSortThreads, 0, s, cols);
    launch_after(k_uniq_scan, nc, 256, 0, s, cols);
    launch_after(k_uniq_emit<ITEMS>, grid, kSortThreads, 0, s, cols);
}

uint64_t sort_launches(const Staged& sg) { return sg.sort_passes ? 3ull * sg.sort_passes + 3 : 0; }

uint64_t round_launches(const StagedRound& R) {
    return R.chunks * (R.max_stages + (R.sparse && R.max_stages > 1 ? 3ull : 0ull));
}

uint64_t launch_sort(const Staged& sg, const SgCol* cols, cudaStream_t s) {
    if (!sg.sort_passes) return 0;
    if (sg.sort_large) launch_sort_tiles<kSortItemsLarge>(sg, cols, s);
    else launch_sort_tiles<kSortItemsSmall>(sg, cols, s);
    return sort_launches(sg);
}

// the sums of a round's predicates at every distinct value
uint64_t launch_round(const oblivgm_ctx* ctx, const StagedRound& R, const SgPred* preds, const DevKey* keys,
                      cudaStream_t s) {
    StageParams W{};
    W.aes = ctx->aes;
    W.te0 = ctx->d_te0;
    W.keys = keys;
    W.preds = preds + R.pred_begin;
    W.n_preds = R.n_preds;
    const unsigned sms = (unsigned)ctx->sm_count;
    for (uint32_t c = 0; c < R.chunks; c++) {
        if (R.sparse && R.max_stages > 1) {
            launch_after(k_run_count, dim3(R.max_blocks, R.n_preds), kRunBlock, 0, s, W.preds, c);
            launch_after(k_run_scan, dim3(R.max_stages - 1, R.n_preds), 256, 0, s, W.preds, c);
            launch_after(k_run_emit, dim3(R.max_blocks, R.n_preds), kRunBlock, 0, s, W.preds, c);
        }
        W.chunk = c;
        for (uint32_t st = 0; st + 1 < R.max_stages; st++) {
            W.stage = st;
            launch_after(k_stage, sms, kStageThreads, kTableBytes, s, W);
        }
        launch_after(k_stage_last, sms, kStageThreads, kTableBytes, s, W);
    }
    return round_launches(R);
}

}  // namespace

uint64_t staged_launches(const Staged& sg) {
    uint64_t launches = sort_launches(sg);
    for (const StagedRound& R : sg.rounds) launches += round_launches(R) + 1;
    return launches;
}

oblivgm_status staged_launch(oblivgm_ctx* ctx, const Staged& sg, const unsigned char* image, cudaStream_t s) {
    uint64_t launches = launch_sort(sg, reinterpret_cast<const SgCol*>(image), s);
    for (const StagedRound& R : sg.rounds) {
        launches += launch_round(ctx, R, reinterpret_cast<const SgPred*>(image + sg.off_preds),
                                 reinterpret_cast<const DevKey*>(image + sg.off_keys), s);
        launch_combine(ctx, sg.shape, reinterpret_cast<const SgGroup*>(image + sg.off_groups) + R.group_begin, R.n_groups,
                       reinterpret_cast<const SgFold*>(image + sg.off_folds), sg.split, R.items, s);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "staged launch");
    ctx->launches += launches;
    return OBLIVGM_OK;
}

bool staged_plan_raw(uint32_t kind, uint32_t n_bits, uint32_t n_keys, const uint32_t* points, uint64_t n_points,
                     const StagedLimits& limits, Staged* sg) {
    *sg = Staged{};
    if (n_points > kMaxElems) return false;
    SgCol C{};
    C.share[0] = points;
    C.n = n_points;
    C.mask = n_bits >= 32 ? 0xFFFFFFFFu : ((1u << n_bits) - 1u);
    C.passes = (n_bits + 7) / 8;
    const bool dcf = kind == OBLIVGM_KEY_DCF;
    // at most 64 keys a round; a round's launches are its own, the sort is shared
    const double rounds = (n_keys + 63) / 64, step = n_keys / rounds * (dcf ? kDcfStep : kDpfStep);
    // the per-item kernel's time, less a margin, is what a staged evaluation may take (2 DCF keys at
    // 15,000 points, n = 8: per item 17.5 us, staged 20.3; at 30,000 points 32.9 and 19.2); most
    // small calls are decided by the launches alone
    const double other = 0.95 * rounds * step * n_bits * (double)n_points + kLaunch;
    const bool may_be_dense = (int)n_bits <= kMaxDenseBits;
    const double sort = (double)C.n * kSortKeyPass * C.passes + kLaunch * (3 + 3 * rounds + 3 * C.passes);
    if (kRawFixed + 2 * rounds * kLaunch + (may_be_dense ? 0 : sort) > other) return false;
    std::vector<uint8_t> lev, ld;
    double cs = rounds * choose_stages((double)C.n, false, (int)n_bits, step, &lev) + sort;
    if (may_be_dense) {
        const double cd = rounds * choose_stages(0, true, (int)n_bits, step, &ld);
        if (cd <= cs) {
            cs = cd;
            C.passes = 0;
            lev = ld;
        }
    }
    if (kRawFixed + cs + rounds * kLaunch > other) return false;
    sg->raw = true;
    sg->sort_passes = C.passes;
    sg->cols.push_back(C);
    choose_tiles(sg);
    C = sg->cols[0];
    const size_t col_end = layout_col(&C, nullptr, 0);
    // one predicate per 64 keys at most and per round, fewer where their states would not fit
    SgPred p{};
    p.kind = dcf ? OBLIVGM_PRED_RANGE : OBLIVGM_PRED_EQ;
    p.n = n_bits;
    p.mask = C.mask;
    p.dense = C.passes == 0;
    p.stages = (uint32_t)lev.size();
    std::copy(lev.begin(), lev.end(), p.lev);
    const uint64_t vals = max_values(C);
    p.z_elem = 1;
    p.z_slot = vals;
    p.parts = 1;
    p.chunk = kRunBlock;
    while (p.chunk < vals && p.chunk < limits.chunk) p.chunk <<= 1;
    p.blocks = p.chunk / kRunBlock;
    for (uint32_t s = 0; s + 1 < p.stages; s++) p.cap[s & 1] = std::max(p.cap[s & 1], (uint32_t)max_runs(p, C, s));
    p.n_keys = std::min<uint32_t>(n_keys, 64);
    while (p.n_keys > 1 && layout_pred(&p, C, nullptr, col_end) - col_end > limits.round_bytes) p.n_keys = (p.n_keys + 1) / 2;
    sg->scratch_bytes = layout_pred(&p, C, nullptr, col_end);
    if (sg->scratch_bytes > limits.cap) { *sg = Staged{}; return false; }
    const uint32_t per = p.n_keys;
    for (uint32_t k = 0; k < n_keys; k += per) {
        p.key_begin = k;
        p.n_keys = p.slots = std::min(per, n_keys - k);
        StagedRound R{};
        R.pred_begin = (uint32_t)sg->preds.size();
        R.n_preds = 1;
        R.max_stages = p.stages;
        R.chunks = (uint32_t)((vals + p.chunk - 1) / p.chunk);
        R.sparse = !p.dense;
        R.max_blocks = p.blocks;
        sg->preds.push_back(p);
        sg->rounds.push_back(R);
    }
    sg->off_preds = up256(sizeof(SgCol));
    sg->off_folds = sg->off_groups = sg->off_keys = sg->off_preds + up256(sg->preds.size() * sizeof(SgPred));
    sg->image_bytes = sg->off_keys;
    return true;
}

oblivgm_status staged_launch_raw(oblivgm_ctx* ctx, const Staged& sg, const unsigned char* image, const DevKey* keys,
                                 uint32_t* out, cudaStream_t s) {
    uint64_t launches = launch_sort(sg, reinterpret_cast<const SgCol*>(image), s);
    GatherParams G{};
    G.col = reinterpret_cast<const SgCol*>(image);
    G.n_points = sg.cols[0].n;
    for (const StagedRound& R : sg.rounds) {
        const SgPred& p = sg.preds[R.pred_begin];
        launches += launch_round(ctx, R, reinterpret_cast<const SgPred*>(image + sg.off_preds), keys, s);
        G.z = p.z;
        G.vals = p.z_slot;
        G.n_keys = p.n_keys;
        G.out = out + (uint64_t)p.key_begin * G.n_points;
        const unsigned gx = (unsigned)std::min<uint64_t>((G.n_points + 255) / 256, 8ull * ctx->sm_count);
        launch_after(k_gather_raw, dim3(gx, std::min<uint32_t>(p.n_keys, 8)), 256, 0, s, G);
        launches++;
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "staged evaluation launch");
    ctx->launches += launches;
    return OBLIVGM_OK;
}

oblivgm_status set_staged_attrs() {
    cudaError_t e = cudaFuncSetAttribute(k_stage, cudaFuncAttributeMaxDynamicSharedMemorySize, kTableBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stage_last, cudaFuncAttributeMaxDynamicSharedMemorySize, kTableBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_combine<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCombineSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_combine<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCombineSmem);
    return e == cudaSuccess ? OBLIVGM_OK : cuda_fail(e, "staged kernel attributes");
}

}  // namespace ogm
