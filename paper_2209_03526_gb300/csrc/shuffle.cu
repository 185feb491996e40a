// shuffle.cu -- secShuffle (Alg. 5) with the three servers simulated on one GPU, and
// secFetch case II (Alg. 4) on top of it.
//
//   k_feistel_tab the round function of each pair's Feistel PRP at all 2^h half-words
//   k_shuf_cs1    CS1: X1 = pi31(pi12(D1 + D2 + T12) + T31)
//   k_shuf_cs2    CS2: Y1 = pi12(D3 - T12); C1 = pi23(X1 + T23) - R2; its output share R2
//   k_shuf_cs3    CS3: C2 = pi23(pi31(Y1 - T31) - T23) - R1; R3 = C1 + C2; output shares R1, R3
//
// Each server kernel reads only what that server holds or receives, evaluates its pairs'
// permutations row by row from the round-function tables (4 lookups a pass, cycle walking) and
// makes the masks T and R, AES blocks of the pair's seed, four words per block, where used.
// The mask AES and the rows' out-of-order accesses share the L1 / shared-memory pipe, so both
// are kept small: an AES call starts from what its counters have in common (mask_words), a
// partial last block ends with the columns it needs, and the rows that go between the servers
// are padded to whole 16-byte groups, so that a row moved out of order is one or two 16-byte
// accesses inside its own sectors.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "device_fss.cuh"
#include "host_crypto.h"
#include "oblivgm.h"
#include "ptx_async.cuh"
#include "runtime.h"

namespace ogm {

namespace {

#ifndef OGM_SHUF_THREADS
#define OGM_SHUF_THREADS 768
#endif
constexpr int kShufThreads = OGM_SHUF_THREADS;
constexpr uint32_t kShufMaxWidth = 64;

// What AES calls on counters i < 2^24 (tag, block q fixed) share: three columns after round 1
// without byte 0..2's lookups and the four columns after round 2 without those three
// columns' bytes, 17 lookups of 160.
struct MaskPrefix {
    uint32_t n0, n2, n3, m[4];
};
constexpr int kMaskStreams = 5;              // (s12, T), (s12, R), (s23, T), (s31, T), (s31, R)
constexpr int kT12 = 0, kR2 = 1, kT23 = 2, kT31 = 3, kR1 = 4;
constexpr uint64_t kFastRows = 1ull << 24;   // prefixes, and round tables that fit shared memory

struct ShufParams {
    uint32_t rk[3][44];         // round keys of s12, s23, s31
    const uint32_t* te0;
    const uint32_t* d[3];       // input shares, rows of width words every ds words
    uint32_t* s[3];             // output shares R1, R2, R3, rows every os words
    uint16_t* ftab;             // [which][round][2^h] Feistel round values
    uint32_t* x1;               // rows between the servers, every ps words (a multiple of 4)
    uint32_t* y1;
    uint32_t* c1;
    uint64_t n;
    uint32_t width, group;      // group: OBLIVGM_SHUFFLE_ADD or _XOR
    uint32_t half_bits;         // h of the Feistel network
    uint32_t ds, ps, os;
    uint32_t vec_d, vec_s;      // 16-byte accesses fit the input / output rows
    // secFetch case II: the input rows come straight from columns x, (id), attributes, and word 0
    // of the output rows also goes to columns, which the opening reads
    const uint32_t* cols[3][kShufMaxWidth];
    uint32_t* x_out[3];
    uint32_t from_cols;
    MaskPrefix pre[kMaskStreams][kShufMaxWidth / 4];
};

constexpr int S12 = 0, S23 = 1, S31 = 2;

__device__ __forceinline__ uint32_t op_add(uint32_t g, uint32_t a, uint32_t b) { return g ? a ^ b : a + b; }
__device__ __forceinline__ uint32_t op_sub(uint32_t g, uint32_t a, uint32_t b) { return g ? a ^ b : a - b; }

// words 4 q .. 4 q + need - 1 of row i of stream `str` (a seed's table T, tag 1, or R, tag 2)
template <bool FAST>
__device__ __forceinline__ void mask_words(const SmemTabPair& T, const ShufParams& P, int str, uint64_t i, uint32_t q,
                                           uint32_t need, uint32_t out[4]) {
    const uint32_t* rk = P.rk[str <= kR2 ? S12 : str == kT23 ? S23 : S31];
    uint32_t c[4];
    if (FAST) {
        const MaskPrefix& p = P.pre[str][q];
        const uint32_t c0 = (uint32_t)i ^ rk[0];
        const uint32_t n0 = p.n0 ^ T.lu<0, 0>(c0), n2 = p.n2 ^ T.lu<2, 2>(c0), n3 = p.n3 ^ T.lu<1, 1>(c0);
        c[0] = p.m[0] ^ T.lu<0, 0>(n0) ^ T.lu<2, 2>(n2) ^ T.lu<3, 3>(n3);
        c[1] = p.m[1] ^ T.lu<3, 3>(n0) ^ T.lu<1, 1>(n2) ^ T.lu<2, 2>(n3);
        c[2] = p.m[2] ^ T.lu<2, 2>(n0) ^ T.lu<0, 0>(n2) ^ T.lu<1, 1>(n3);
        c[3] = p.m[3] ^ T.lu<1, 1>(n0) ^ T.lu<3, 3>(n2) ^ T.lu<0, 0>(n3);
    } else {
        const uint32_t tag = str == kR2 || str == kR1 ? 2u : 1u;
        c[0] = (uint32_t)i ^ rk[0];
        c[1] = (uint32_t)(i >> 32) ^ rk[1];
        c[2] = (tag | (q << 16)) ^ rk[2];
        c[3] = rk[3];
        aes_round(T, c, rk[4], rk[5], rk[6], rk[7]);
        aes_round(T, c, rk[8], rk[9], rk[10], rk[11]);
    }
#pragma unroll
    for (int r = 3; r < 10; r++) aes_round(T, c, rk[4 * r], rk[4 * r + 1], rk[4 * r + 2], rk[4 * r + 3]);
    out[0] = last_col(T, c[0], c[1], c[2], c[3]) ^ rk[40];
    out[1] = out[2] = out[3] = 0u;
    if (need > 1) out[1] = last_col(T, c[1], c[2], c[3], c[0]) ^ rk[41];
    if (need > 2) out[2] = last_col(T, c[2], c[3], c[0], c[1]) ^ rk[42];
    if (need > 3) out[3] = last_col(T, c[3], c[0], c[1], c[2]) ^ rk[43];
}

// F_r(R) of the three permutations for every round r and every half-word R: the round
// function sees only h <= 16 bits, so 4 * 2^h AES calls per permutation cover all inputs
__global__ void __launch_bounds__(kShufThreads, 1) k_feistel_tab(const __grid_constant__ ShufParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_trigger();
    fill_tables<true>(reinterpret_cast<uint32_t*>(smem), P.te0);
    __syncthreads();
    const SmemTabPair T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t h = P.half_bits, side = 1u << h, mask = side - 1u;
    const uint64_t total = 12ull * side;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t which = (uint32_t)(t / (4ull * side)), rem = (uint32_t)(t % (4ull * side));
        const uint32_t r = rem / side, R = rem % side;
        const uint32_t in[4] = {R, 0u, 3u | (r << 16), (uint32_t)P.n};
        P.ftab[t] = (uint16_t)(aes_one_w0(T, P.rk[which], in) & mask);
    }
}

// One pair's permutation of [0, n) from its round tables (shared memory, or global for the
// largest tables).  The inverse of a cycle-walking permutation walks the inverse network
// until it re-enters [0, n); the cycle re-enters within the network's domain.
struct Perm {
    const uint16_t* ft;
    uint64_t n;
    uint32_t h;
    template <bool INV>
    __device__ __forceinline__ uint64_t pass(uint64_t x) const {
        const uint32_t side = 1u << h, mask = side - 1u;
        uint32_t L = (uint32_t)(x >> h) & mask, R = (uint32_t)x & mask;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (INV) {        // rounds 3..0, each (L', R') -> (R' xor F_r(L'), L')
                const uint32_t prev = R ^ ft[(uint32_t)(3 - k) * side + L];
                R = L;
                L = prev;
            } else {          // round r: (L, R) -> (R, L xor F_r(R))
                const uint32_t t = L ^ ft[(uint32_t)k * side + R];
                L = R;
                R = t;
            }
        }
        return ((uint64_t)L << h) | R;
    }
    template <bool INV>
    __device__ __forceinline__ uint64_t walk(uint64_t y) const {
        if (n <= 1) return y;
        uint64_t x = pass<INV>(y);
        for (uint64_t guard = 0; x >= n && guard < (1ull << (2 * h)); guard++) x = pass<INV>(x);
        return x < n ? x : y;      // y is unreachable; it keeps every later index inside the table
    }
    __device__ __forceinline__ uint64_t fwd(uint64_t i) const { return walk<false>(i); }
    __device__ __forceinline__ uint64_t inv(uint64_t i) const { return walk<true>(i); }
};

// a server's two permutations: their round tables copied next to the AES tables (FAST)
template <bool FAST>
__device__ __forceinline__ void load_perms(const ShufParams& P, unsigned char* smem, int a, int b, Perm& pa, Perm& pb) {
    const uint32_t words = 4u << P.half_bits;             // 16-bit values of one permutation
    const uint16_t *ga = P.ftab + (uint64_t)a * words, *gb = P.ftab + (uint64_t)b * words;
    if (FAST) {
        uint16_t* sm = reinterpret_cast<uint16_t*>(smem + kTableBytes);
        for (uint32_t w = threadIdx.x; w < words; w += blockDim.x) {
            sm[w] = ga[w];
            sm[words + w] = gb[w];
        }
        ga = sm;
        gb = sm + words;
    }
    pa = Perm{ga, P.n, P.half_bits};
    pb = Perm{gb, P.n, P.half_bits};
}

// words 4 q .. of a row (need of them; with vec the row has room for, and the base alignment of, all four)
__device__ __forceinline__ void load_words(const uint32_t* row, uint32_t q, uint32_t need, bool vec, uint32_t v[4]) {
    if (vec) {
        const uint4 x = *reinterpret_cast<const uint4*>(row + 4 * q);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
        for (uint32_t e = 0; e < 4; e++) v[e] = e < need ? row[4 * q + e] : 0u;
    }
}

__device__ __forceinline__ void store_words(uint32_t* row, uint32_t q, uint32_t need, bool vec, const uint32_t v[4]) {
    if (vec) {
        *reinterpret_cast<uint4*>(row + 4 * q) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (uint32_t e = 0; e < 4; e++)
            if (e < need) row[4 * q + e] = v[e];
    }
}

// words 4 q .. of row i of share set j of the input; a record is (x, id, attributes), the id c
// shared as (c, 0, 0)
__device__ __forceinline__ void load_input(const ShufParams& P, int j, uint64_t i, uint32_t q, uint32_t need,
                                           uint32_t v[4]) {
    if (P.from_cols) {
#pragma unroll
        for (uint32_t e = 0; e < 4; e++) {
            const uint32_t w = 4 * q + e;
            v[e] = w == 1 ? (j == 0 ? (uint32_t)i : 0u) : e < need ? __ldg(P.cols[j][w] + i) : 0u;
        }
    } else {
        load_words(P.d[j] + i * P.ds, q, need, P.vec_d, v);
    }
}

// The input rows are read in order and written, padded, at their permuted place: an unaligned
// or column-wise input never has to be gathered.  (secFetch case II packed CS2's share set into
// rows for a gather before: 16 us of 409 at 2^20 x 6 words.)  The rows that come from another
// server are gathered instead, so that those writes are in order.  A row's words are read
// before the AES calls, which then cover the reads.

// CS1: X1[k] = (D1 + D2 + T12)[i] + T31[j], j = pi12(i), k = pi31(j)
template <bool FAST>
__global__ void __launch_bounds__(kShufThreads, 1) k_shuf_cs1(const __grid_constant__ ShufParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_trigger();
    fill_tables<true>(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    Perm p12, p31;
    load_perms<FAST>(P, smem, S12, S31, p12, p31);
    __syncthreads();
    const SmemTabPair T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t W = P.width, g = P.group;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t j = p12.fwd(i), k = p31.fwd(j);
        for (uint32_t q = 0; q * 4 < W; q++) {
            const uint32_t need = min(4u, W - 4 * q);
            uint32_t a[4], b[4], t12[4], t31[4];
            load_input(P, 0, i, q, need, a);
            load_input(P, 1, i, q, need, b);
            mask_words<FAST>(T, P, kT12, i, q, need, t12);
            mask_words<FAST>(T, P, kT31, j, q, need, t31);
#pragma unroll
            for (int e = 0; e < 4; e++) a[e] = op_add(g, op_add(g, op_add(g, a[e], b[e]), t12[e]), t31[e]);
            store_words(P.x1 + k * P.ps, q, need, true, a);
        }
    }
}

// CS2: items 0..n-1: Y1[j] = D3[i] - T12[i], j = pi12(i);
//      items n..2n-1 (l = item - n): C1[l] = X1[k] + T23[k] - R2[l], k = pi23^-1(l); output R2[l]
template <bool FAST>
__global__ void __launch_bounds__(kShufThreads, 1) k_shuf_cs2(const __grid_constant__ ShufParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_trigger();
    fill_tables<true>(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    Perm p12, p23;
    load_perms<FAST>(P, smem, S12, S23, p12, p23);
    __syncthreads();
    const SmemTabPair T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t W = P.width, g = P.group;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < 2 * P.n;
         t += (uint64_t)gridDim.x * blockDim.x) {
        if (t < P.n) {
            const uint64_t i = t, j = p12.fwd(i);
            for (uint32_t q = 0; q * 4 < W; q++) {
                const uint32_t need = min(4u, W - 4 * q);
                uint32_t a[4], t12[4];
                load_input(P, 2, i, q, need, a);
                mask_words<FAST>(T, P, kT12, i, q, need, t12);
#pragma unroll
                for (int e = 0; e < 4; e++) a[e] = op_sub(g, a[e], t12[e]);
                store_words(P.y1 + j * P.ps, q, need, true, a);
            }
        } else {
            const uint64_t l = t - P.n, k = p23.inv(l);
            for (uint32_t q = 0; q * 4 < W; q++) {
                const uint32_t need = min(4u, W - 4 * q);
                uint32_t a[4], t23[4], r2[4];
                load_words(P.x1 + k * P.ps, q, need, true, a);
                mask_words<FAST>(T, P, kT23, k, q, need, t23);
                mask_words<FAST>(T, P, kR2, l, q, need, r2);
#pragma unroll
                for (int e = 0; e < 4; e++) a[e] = op_sub(g, op_add(g, a[e], t23[e]), r2[e]);
                store_words(P.c1 + l * P.ps, q, need, true, a);
                store_words(P.s[1] + l * P.os, q, need, P.vec_s, r2);
                if (P.from_cols && q == 0) P.x_out[1][l] = r2[0];
            }
        }
    }
}

// CS3: C2[l] = Y1[j] - T31[j] - T23[k] - R1[l], R3[l] = C1[l] + C2[l], with k = pi23^-1(l),
// j = pi31^-1(k); outputs R1[l] and R3[l]
template <bool FAST>
__global__ void __launch_bounds__(kShufThreads, 1) k_shuf_cs3(const __grid_constant__ ShufParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_trigger();
    fill_tables<true>(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    Perm p23, p31;
    load_perms<FAST>(P, smem, S23, S31, p23, p31);
    __syncthreads();
    const SmemTabPair T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t W = P.width, g = P.group;
    for (uint64_t l = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; l < P.n; l += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t k = p23.inv(l), j = p31.inv(k);
        for (uint32_t q = 0; q * 4 < W; q++) {
            const uint32_t need = min(4u, W - 4 * q);
            uint32_t a[4], c[4], t31[4], t23[4], r1[4];
            load_words(P.y1 + j * P.ps, q, need, true, a);
            load_words(P.c1 + l * P.ps, q, need, true, c);
            mask_words<FAST>(T, P, kT31, j, q, need, t31);
            mask_words<FAST>(T, P, kT23, k, q, need, t23);
            mask_words<FAST>(T, P, kR1, l, q, need, r1);
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const uint32_t c2 = op_sub(g, op_sub(g, op_sub(g, a[e], t31[e]), t23[e]), r1[e]);
                a[e] = op_add(g, c[e], c2);
            }
            store_words(P.s[2] + l * P.os, q, need, P.vec_s, a);
            store_words(P.s[0] + l * P.os, q, need, P.vec_s, r1);
            if (P.from_cols && q == 0) {
                P.x_out[0][l] = r1[0];
                P.x_out[2][l] = a[0];
            }
        }
    }
}

// ------------------------------------------------------------------ secFetch case II

constexpr int kCompactRows = 1024;   // rows per block of the open-and-compact pass

// The opening reads word 0 of the shuffled rows from columns that CS2 and CS3 wrote beside them:
// 12 bytes a row instead of three rows' sectors, 16.4 + 19.7 us for the two passes before.
struct CompactParams {
    const uint32_t* x[3];
    const uint32_t* s[3];
    uint32_t* out[3];
    uint32_t* block_count;      // per block: rows with x^ = 1
    uint64_t n, cap;
    uint32_t width, stride, n_blocks;   // rows of width words every stride words
};

__device__ __forceinline__ bool opened_one(const CompactParams& P, uint64_t l) {
    return l < P.n && P.x[0][l] + P.x[1][l] + P.x[2][l] == 1u;
}

// open x^ for a block of rows and count the ones
__global__ void __launch_bounds__(kCompactRows) k_open_count(const __grid_constant__ CompactParams P) {
    __shared__ uint32_t warp_n[kCompactRows / 32];
    grid_trigger();
    grid_wait();
    const uint64_t l = (uint64_t)blockIdx.x * kCompactRows + threadIdx.x;
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, opened_one(P, l));
    if ((threadIdx.x & 31) == 0) warp_n[threadIdx.x >> 5] = __popc(b);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < kCompactRows / 32; w++) s += warp_n[w];
        P.block_count[blockIdx.x] = s;
    }
}

// exclusive scan of the block counts in place (one CTA); the total goes to block_count[n_blocks]
__global__ void __launch_bounds__(1024) k_scan_counts(uint32_t* c, uint32_t n_blocks) {
    __shared__ uint32_t part[1024];
    __shared__ uint32_t carry;
    grid_trigger();
    grid_wait();
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t base = 0; base < n_blocks; base += 1024) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t v = i < n_blocks ? c[i] : 0u;
        part[threadIdx.x] = v;
        __syncthreads();
        for (uint32_t off = 1; off < 1024; off <<= 1) {   // Hillis-Steele inclusive scan
            const uint32_t add = threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
            __syncthreads();
            part[threadIdx.x] += add;
            __syncthreads();
        }
        if (i < n_blocks) c[i] = carry + part[threadIdx.x] - v;
        __syncthreads();
        if (threadIdx.x == 0) carry += part[1023];
        __syncthreads();
    }
    if (threadIdx.x == 0) c[n_blocks] = carry;
}

// write the kept rows (id and attributes of every share set) at their scanned offsets
__global__ void __launch_bounds__(kCompactRows) k_compact(const __grid_constant__ CompactParams P) {
    __shared__ uint32_t warp_off[kCompactRows / 32];
    grid_wait();
    const uint64_t l = (uint64_t)blockIdx.x * kCompactRows + threadIdx.x;
    const bool keep = opened_one(P, l);
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, keep);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_off[warp] = __popc(b);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < kCompactRows / 32; w++) {
            const uint32_t t = warp_off[w];
            warp_off[w] = s;
            s += t;
        }
    }
    __syncthreads();
    if (!keep) return;
    const uint64_t m = (uint64_t)P.block_count[blockIdx.x] + warp_off[warp] + __popc(b & ((1u << lane) - 1u));
    if (m >= P.cap) return;
    const uint32_t W = P.width;
#pragma unroll
    for (int j = 0; j < 3; j++)
        for (uint32_t w = 1; w < W; w++) P.out[j][m * (W - 1) + (w - 1)] = P.s[j][l * P.stride + w];
}

}  // namespace

// host side of mask_words: what the counters i < 2^24 of stream (tag, block q) share
static MaskPrefix mask_prefix(const uint32_t* rk, uint32_t tag, uint32_t q) {
    const uint32_t* te0 = aes_tables().te0;
    const auto lu = [&](int byte, int table, uint32_t col) {
        const uint32_t v = te0[(col >> (8 * byte)) & 0xFFu];
        return table ? (v << (8 * table)) | (v >> (32 - 8 * table)) : v;
    };
    const uint32_t c0 = rk[0], c1 = rk[1], c2 = (tag | (q << 16)) ^ rk[2], c3 = rk[3];
    MaskPrefix p;
    p.n0 = lu(1, 1, c1) ^ lu(2, 2, c2) ^ lu(3, 3, c3) ^ rk[4];
    const uint32_t n1 = lu(0, 0, c1) ^ lu(1, 1, c2) ^ lu(2, 2, c3) ^ lu(3, 3, c0) ^ rk[5];
    p.n2 = lu(0, 0, c2) ^ lu(1, 1, c3) ^ lu(3, 3, c1) ^ rk[6];
    p.n3 = lu(0, 0, c3) ^ lu(2, 2, c1) ^ lu(3, 3, c2) ^ rk[7];
    p.m[0] = lu(1, 1, n1) ^ rk[8];
    p.m[1] = lu(0, 0, n1) ^ rk[9];
    p.m[2] = lu(3, 3, n1) ^ rk[10];
    p.m[3] = lu(2, 2, n1) ^ rk[11];
    return p;
}

// Rows of the shuffle's input and output; secFetch case II has input columns instead of rows, and
// columns for word 0 of the output rows.
struct ShufRows {
    uint32_t ds, os;                            // row strides in words
    const uint32_t* const* cols[3];
    uint32_t* x_out[3];
};

// the shuffle on device buffers; scratch from the stream-ordered pool
oblivgm_status shuffle_device(oblivgm_ctx* ctx, uint32_t group, uint64_t n, uint32_t width, const uint32_t* const in[3],
                              const uint8_t seeds[48], uint32_t* const out[3], const ShufRows& rows, cudaStream_t s) {
    if (n == 0) return OBLIVGM_OK;
    ShufParams P;
    std::memset(&P, 0, sizeof P);
    for (int k = 0; k < 3; k++) {
        const RoundKeys rk = expand_key(seeds + 16 * k);
        std::memcpy(P.rk[k], rk.w, sizeof P.rk[k]);
        P.d[k] = in[k];
        P.s[k] = out[k];
    }
    P.te0 = ctx->d_te0;
    P.n = n;
    P.width = width;
    P.group = group;
    P.ds = rows.ds;
    P.os = rows.os;
    P.ps = (width + 3) / 4 * 4;
    // 16-byte accesses: whole groups of four words in every row, and aligned bases
    P.vec_d = rows.ds % 4 == 0;
    P.vec_s = rows.os % 4 == 0;
    for (int k = 0; k < 3; k++) {
        if (in[k] && reinterpret_cast<uintptr_t>(in[k]) % 16) P.vec_d = 0;
        if (reinterpret_cast<uintptr_t>(out[k]) % 16) P.vec_s = 0;
    }
    if (rows.cols[0]) {
        P.from_cols = 1;
        for (int k = 0; k < 3; k++) {
            P.x_out[k] = rows.x_out[k];
            for (uint32_t w = 0; w < width; w++) P.cols[k][w] = rows.cols[k][w];
        }
    }
    uint32_t bits = 0;
    for (uint64_t v = n - 1; v; v >>= 1) bits++;
    P.half_bits = std::max<uint32_t>(1, (bits + 1) / 2);
    const bool fast = n <= kFastRows;
    if (fast) {
        const int seed_of[kMaskStreams] = {S12, S12, S23, S31, S31};
        const uint32_t tag_of[kMaskStreams] = {1u, 2u, 1u, 1u, 2u};
        for (int k = 0; k < kMaskStreams; k++)
            for (uint32_t q = 0; 4 * q < width; q++) P.pre[k][q] = mask_prefix(P.rk[seed_of[k]], tag_of[k], q);
    }
    const size_t tab_bytes = ((size_t)n * P.ps * 4 + 255) & ~size_t(255);
    const size_t total = 3 * tab_bytes + 12ull * (1ull << P.half_bits) * sizeof(uint16_t);
    uint8_t* scratch = nullptr;
    const oblivgm_status as = ws_alloc(ctx, reinterpret_cast<void**>(&scratch), total, s, "shuffle scratch");
    if (as != OBLIVGM_OK) return as;
    uint32_t** tabs[3] = {&P.x1, &P.y1, &P.c1};
    for (int k = 0; k < 3; k++) *tabs[k] = reinterpret_cast<uint32_t*>(scratch + k * tab_bytes);
    P.ftab = reinterpret_cast<uint16_t*>(scratch + 3 * tab_bytes);
    auto grid = [&](uint64_t items) {
        return (unsigned)std::min<uint64_t>((items + kShufThreads - 1) / kShufThreads, (uint64_t)ctx->sm_count);
    };
    k_feistel_tab<<<grid(12ull << P.half_bits), kShufThreads, kTableBytes, s>>>(P);
    if (fast) {
        const int smem = kTableBytes + (int)((8u << P.half_bits) * sizeof(uint16_t));
        launch_after(k_shuf_cs1<true>, grid(n), kShufThreads, smem, s, P);
        launch_after(k_shuf_cs2<true>, grid(2 * n), kShufThreads, smem, s, P);
        launch_after(k_shuf_cs3<true>, grid(n), kShufThreads, smem, s, P);
    } else {
        launch_after(k_shuf_cs1<false>, grid(n), kShufThreads, kTableBytes, s, P);
        launch_after(k_shuf_cs2<false>, grid(2 * n), kShufThreads, kTableBytes, s, P);
        launch_after(k_shuf_cs3<false>, grid(n), kShufThreads, kTableBytes, s, P);
    }
    ctx->launches += 4;
    cudaError_t ce = cudaGetLastError();
    const cudaError_t fe = cudaFreeAsync(scratch, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "shuffle launch");
    ce = fe;
    return ce == cudaSuccess ? OBLIVGM_OK : cuda_fail(ce, "shuffle scratch release");
}

oblivgm_status set_shuffle_attrs() {
    constexpr int kFastSmem = kTableBytes + (8 << 12) * (int)sizeof(uint16_t);   // h <= 12 up to 2^24 rows
    const struct { const void* fn; int smem; } fns[] = {
        {reinterpret_cast<const void*>(k_feistel_tab), kTableBytes},
        {reinterpret_cast<const void*>(k_shuf_cs1<true>), kFastSmem},
        {reinterpret_cast<const void*>(k_shuf_cs2<true>), kFastSmem},
        {reinterpret_cast<const void*>(k_shuf_cs3<true>), kFastSmem},
        {reinterpret_cast<const void*>(k_shuf_cs1<false>), kTableBytes},
        {reinterpret_cast<const void*>(k_shuf_cs2<false>), kTableBytes},
        {reinterpret_cast<const void*>(k_shuf_cs3<false>), kTableBytes}};
    for (const auto& f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, f.smem);
        if (e != cudaSuccess) return cuda_fail(e, "shuffle kernel attributes");
    }
    return OBLIVGM_OK;
}

}  // namespace ogm

using namespace ogm;

extern "C" oblivgm_status oblivgm_shuffle(oblivgm_ctx* ctx, uint32_t group, uint64_t n_rows, uint32_t width,
                                          const uint32_t* const in[3], const uint8_t seeds[48],
                                          uint32_t* const out[3], void* stream) {
    const NvtxRange nvtx_range("oblivgm_shuffle");
    if (!ctx || !in || !out || !seeds) return fail(OBLIVGM_EINVAL, "NULL argument");
    if (group != OBLIVGM_SHUFFLE_ADD && group != OBLIVGM_SHUFFLE_XOR) return fail(OBLIVGM_EINVAL, "unknown share group");
    if (width < 1 || width > kShufMaxWidth) return fail(OBLIVGM_EINVAL, "width must be 1..64");
    if (n_rows >= (1ull << 31)) return fail(OBLIVGM_EINVAL, "at most 2^31 - 1 rows");
    for (int j = 0; j < 3; j++) {
        if (n_rows && (!in[j] || !out[j])) return fail(OBLIVGM_EINVAL, "NULL share set");
        if (reinterpret_cast<uintptr_t>(in[j]) % 4 || reinterpret_cast<uintptr_t>(out[j]) % 4)
            return fail(OBLIVGM_EINVAL, "share sets must be 4-byte aligned");
    }
    const cudaError_t ce = cudaSetDevice(ctx->device);
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaSetDevice");
    return shuffle_device(ctx, group, n_rows, width, in, seeds, out, ShufRows{width, width, {}, {}},
                          static_cast<cudaStream_t>(stream));
}

extern "C" oblivgm_status oblivgm_fetch_multi(oblivgm_ctx* ctx, uint32_t table_id, const uint32_t* const x[3],
                                              uint32_t n_attrs, const uint32_t* attrs, const uint8_t seeds[48],
                                              uint32_t* const out[3], uint64_t cap, uint64_t* count, void* stream) {
    const NvtxRange nvtx_range("oblivgm_fetch_multi");
    if (!ctx || !x || !out || !seeds || !count || (n_attrs && !attrs)) return fail(OBLIVGM_EINVAL, "NULL argument");
    if (n_attrs + 2 > kShufMaxWidth) return fail(OBLIVGM_EINVAL, "at most 62 attributes");
    cudaError_t ce = cudaSetDevice(ctx->device);
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaSetDevice");
    auto it = ctx->tables.find(table_id);
    if (it == ctx->tables.end()) return fail(OBLIVGM_ENOENT, "no such table");
    const Table& tb = it->second;
    for (uint32_t a = 0; a < n_attrs; a++)
        if (attrs[a] >= tb.n_attrs) return fail(OBLIVGM_EINVAL, "attribute outside the table");
    const uint64_t n = tb.n_elems;
    if (n >= (1ull << 31)) return fail(OBLIVGM_EINVAL, "at most 2^31 - 1 elements");
    for (int j = 0; j < 3; j++)
        if (n && (!x[j] || (cap && !out[j]))) return fail(OBLIVGM_EINVAL, "NULL share set");
    *count = 0;
    if (n == 0) return OBLIVGM_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const uint32_t W = 2 + n_attrs;
    const uint32_t n_blocks = (uint32_t)((n + kCompactRows - 1) / kCompactRows);
    const uint32_t stride = (W + 3) / 4 * 4;      // rows padded to 16-byte groups
    const size_t tab = ((size_t)n * stride * 4 + 255) & ~size_t(255);
    const size_t col = ((size_t)n * 4 + 255) & ~size_t(255);
    const size_t total = 3 * (tab + col) + ((size_t)(n_blocks + 1) * 4 + 255);
    uint8_t* scratch = nullptr;
    {
        const oblivgm_status as = ws_alloc(ctx, reinterpret_cast<void**>(&scratch), total, s, "fetch scratch");
        if (as != OBLIVGM_OK) return as;
    }
    // the records' columns: x, id, attributes
    const uint32_t* cols[3][kShufMaxWidth] = {};
    uint32_t *sh[3], *xs[3];
    for (int j = 0; j < 3; j++) {
        sh[j] = reinterpret_cast<uint32_t*>(scratch + j * tab);
        xs[j] = reinterpret_cast<uint32_t*>(scratch + 3 * tab + j * col);
        cols[j][0] = x[j];
        for (uint32_t a = 0; a < n_attrs; a++)
            cols[j][2 + a] = tb.dev + ((uint64_t)j * tb.n_attrs + attrs[a]) * tb.stride;
    }
    uint32_t* counts = reinterpret_cast<uint32_t*>(scratch + 3 * (tab + col));
    const uint32_t* din[3] = {nullptr, nullptr, nullptr};
    uint32_t* dout[3] = {sh[0], sh[1], sh[2]};
    oblivgm_status st = shuffle_device(ctx, OBLIVGM_SHUFFLE_ADD, n, W, din, seeds, dout,
                                       ShufRows{stride, stride, {cols[0], cols[1], cols[2]}, {xs[0], xs[1], xs[2]}}, s);
    if (st) {
        cudaFreeAsync(scratch, s);
        return st;
    }
    CompactParams C;
    std::memset(&C, 0, sizeof C);
    for (int j = 0; j < 3; j++) {
        C.x[j] = xs[j];
        C.s[j] = sh[j];
        C.out[j] = out[j];
    }
    C.block_count = counts;
    C.n = n;
    C.cap = cap;
    C.width = W;
    C.stride = stride;
    C.n_blocks = n_blocks;
    launch_after(k_open_count, n_blocks, kCompactRows, 0, s, C);
    launch_after(k_scan_counts, 1, 1024, 0, s, counts, n_blocks);
    launch_after(k_compact, n_blocks, kCompactRows, 0, s, C);
    ctx->launches += 3;
    ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        cudaFreeAsync(scratch, s);
        return cuda_fail(ce, "fetch launch");
    }
    uint32_t total_count = 0;
    ce = cudaMemcpyAsync(&total_count, counts + n_blocks, 4, cudaMemcpyDeviceToHost, s);
    if (ce != cudaSuccess) {
        cudaFreeAsync(scratch, s);
        return cuda_fail(ce, "fetch count read");
    }
    ce = cudaFreeAsync(scratch, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "fetch scratch release");
    ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_fail(ce, "fetch synchronize");
    *count = total_count;
    return OBLIVGM_OK;
}
