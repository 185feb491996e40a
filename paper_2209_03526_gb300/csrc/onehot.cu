// onehot.cu -- the one-hot mode of the oblivgm library: secEval exactly as the
// paper writes it (Sec. V-B, V-C, Eq. predEval, Alg. 3).  Attribute values are
// stored as binary-RSS shares of one-hot vectors of length D = 2^n (n <= 16),
// packed 32 positions per word.  Each server evaluates its FSS key halves (Z_2
// outputs, beta = 1) at every public position l and computes
//     x = XOR_l Eval(k, l) AND <e_v>_j[l]
// for the share j its key pair is tied to; it XORs its two results, re-shares them
// in binary RSS and the query element's predicates are folded (AND, XOR or OR) in binary RSS.
//
// Three steps per query:
//  * EvalAll, every key half at every position: the keys stop their trees early (a
//    leaf seed expands into the outputs of 2^min(n,7) consecutive positions, BGI16's
//    early termination for small output groups), and k_onehot_evalall_et gives each
//    (key, leaf) a lane pair that walks the n - 7 levels (seed chain and DCF value
//    chain side by side) and writes the leaf's 128 bits;
//  * the dot pass, one streaming pass over an attribute column's three share rows for
//    up to 4 predicates on that column: k_onehot_dots_pipe (D >= 2^12, persistent,
//    rows staged by per-lane cp.async, warps splitting the rows, each lane holding its
//    slice of the half vectors in registers; parities are XOR-reduced over the warp and
//    each server's bit written packed) or k_onehot_dots (smaller D, a thread per element);
//  * k_onehot_fold: every group in one launch, each element's bits re-shared in
//    binary RSS and folded in token order on whole 32-element words (one PRF AES
//    block from the shared-memory T-tables serves 128 elements); results are packed
//    32 elements per word.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <utility>
#include <vector>

#include "device_fss.cuh"
#include "host_crypto.h"
#include "oblivgm.h"
#include "ptx_async.cuh"
#include "runtime.h"

namespace ogm {

namespace {

constexpr uint32_t kNoKey = 0xFFFFFFFFu;

struct HalfDesc {
    uint32_t key0, key1;   // one DPF key, or two DCF keys (a1, a0); key1 = kNoKey for DPF
    uint32_t cbit;         // public constant XORed in by party 0 of a range half
    uint32_t kind;         // OBLIVGM_KEY_DPF / OBLIVGM_KEY_DCF
};

struct KeySlot {
    uint32_t key;       // index into the keys
    uint32_t half;      // the half vector it is XORed into
    uint32_t cmask;     // all ones where party 0 of a range half adds the public constant
    uint32_t dcf;
};

struct EvalEtParams {
    AesParams aes;
    const uint32_t* te0;
    const EtKey* keys;
    const KeySlot* slots;
    uint32_t* hv;          // [half][words], zeroed before the launch
    uint32_t words;        // max(1, 2^n / 32)
    uint32_t leaves;       // 2^nu leaf seeds per key
    uint32_t n_slots;
};

// AES-128 whose round keys depend on the lane: key A (rkA ^ (m & dA)) where r = 0, key B
// (rkB ^ (m & dB)) where r = ~0.  The four schedules are launch parameters (uniform
// operands); the per-lane choice costs three LOP3s per round-key word.
template <class Tab>
__device__ __forceinline__ void aes_two_keys(const Tab& T, const uint32_t* rkA, const uint32_t* dA,
                                             const uint32_t* rkB, const uint32_t* dB, uint32_t m, uint32_t r,
                                             const uint32_t in[4], uint32_t out[4]) {
    auto key = [&](int w) {
        const uint32_t a = rkA[w] ^ (m & dA[w]), b = rkB[w] ^ (m & dB[w]);
        return a ^ ((a ^ b) & r);
    };
    uint32_t c[4];
#pragma unroll
    for (int j = 0; j < 4; j++) c[j] = in[j] ^ key(j);
#pragma unroll
    for (int rd = 1; rd < 10; rd++) aes_round(T, c, key(4 * rd), key(4 * rd + 1), key(4 * rd + 2), key(4 * rd + 3));
    aes_last(T, c, key(40), key(41), key(42), key(43));
#pragma unroll
    for (int j = 0; j < 4; j++) out[j] = c[j];
}

// Every key at every position.  Work item = (key slot, leaf), taken by a pair of lanes:
// at each of the nu levels the even lane computes the chosen child's seed block and the
// odd lane, for a DCF, its value block H_{K_vdir}(s) on the same seed (for a DPF its
// block is not used); the new seed and control bit reach the odd lane by shuffles.  The
// odd lane then expands the leaf seed into the 2^m output bits of positions
// leaf * 2^m + j,
//   y = V ^ H_{K_vL}(s) ^ t CW,
// and XORs them into the slot's half vector (a range half's two DCF keys land in the same
// words).  At n = 16 a key has 512 leaves of 9 levels: 36 keys are 18,432 items.
constexpr int kEvalEtMaxThreads = 512;

__global__ void __launch_bounds__(kEvalEtMaxThreads, 1) k_onehot_evalall_et(const __grid_constant__ EvalEtParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_trigger();
    fill_tables(reinterpret_cast<uint32_t*>(smem), P.te0);
    __syncthreads();
    const SmemTab T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t lane = threadIdx.x & 31, role = lane & 1u, rmask = 0u - role, even = lane & ~1u;
    const uint64_t items = (uint64_t)P.n_slots * P.leaves;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x / 2;
    // the warp's first pair: the loop bound is the same for every lane of the warp, so the
    // shuffles below always have all 32 lanes; a pair past the end repeats the last item
    // and writes nothing
    const uint64_t warp_first = ((uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) / 2;
    for (uint64_t wf = warp_first; wf < items; wf += stride) {
        const uint64_t idx = wf + lane / 2;
        const bool live = idx < items;
        const uint64_t it = live ? idx : items - 1;
        const uint32_t slot = (uint32_t)(it / P.leaves), leaf = (uint32_t)(it % P.leaves);
        const KeySlot S = P.slots[slot];
        const EtKey& K = P.keys[S.key];
        const int nu = (int)K.levels, m = (int)K.low_bits;
        const uint32_t vmask = S.dcf ? rmask : 0u;    // the value chain runs on the odd lane of a DCF pair
        uint32_t s[4] = {K.seed[0], K.seed[1], K.seed[2], K.seed[3]};
        uint32_t t = K.party, V[4] = {0u, 0u, 0u, 0u};
        for (int i = 0; i < nu; i++) {
            const uint32_t dir = (leaf >> (nu - 1 - i)) & 1u, dm = 0u - dir, tm = 0u - t;
            uint32_t o[4];
            aes_two_keys(T, P.aes.rk_st, P.aes.d_st, P.aes.rk_v, P.aes.d_v, dm, rmask, s, o);
#pragma unroll
            for (int w = 0; w < 4; w++) {
                o[w] ^= s[w];
                V[w] ^= (o[w] ^ (K.vcw[i][w] & tm)) & vmask;
            }
            uint32_t tn = (o[0] & 1u) ^ (t & (((dir ? K.tr : K.tl) >> i) & 1u));
            o[0] &= ~1u;
#pragma unroll
            for (int w = 0; w < 4; w++) s[w] = __shfl_sync(0xFFFFFFFFu, o[w] ^ (K.scw[i][w] & tm), even);
            t = __shfl_sync(0xFFFFFFFFu, tn, even);
        }
        uint32_t c[4];
        aes_sel(T, P.aes.rk_v, P.aes.d_v, 0u, s, c);
        const uint32_t tm = 0u - t;
        const uint32_t bits = 1u << m;
        const uint32_t nw = bits >= 32 ? bits / 32 : 1u;
        const uint32_t keep = bits >= 32 ? 0xFFFFFFFFu : ((1u << bits) - 1u);
        uint32_t* dst = P.hv + (uint64_t)S.half * P.words + (uint64_t)leaf * nw;
        if (live && role) {
#pragma unroll
            for (uint32_t w = 0; w < 4; w++)
                if (w < nw) atomicXor(dst + w, (V[w] ^ c[w] ^ s[w] ^ (K.cw_final[w] & tm) ^ S.cmask) & keep);
        }
    }
}

constexpr int kDotPreds = 4;   // predicates one streaming pass over a column serves

// Pass over one attribute column for up to kDotPreds predicates on it: every element's
// three share rows are read once and ANDed with the six half vectors of each predicate.
// Output: per predicate and server, the bit z_i = x(first half) xor x(second half),
// packed 32 elements per word into zbits[pred][server][word].
struct DotParams {
    const uint32_t* share[3];     // share set j at the column's first element: [elem][words]
    const uint32_t* hv;           // [half][words]
    uint32_t half_base[kDotPreds];
    uint32_t* zbits[kDotPreds];   // [3][ceil(n_elems / 32)] each
    uint64_t n_elems;
    uint32_t words;
    uint32_t n_preds;
    uint32_t pow2[32];            // pow2[i] = 2^i (read at run time by the staged pass)
};

// The pass for rows of W <= 64 words (D < 2^12).  A thread takes one element: its rows are a few
// sectors, the predicates' half vectors come from shared memory (the same word for all lanes),
// every (predicate, server) has one accumulator over the whole row, and a ballot of the parities
// is the packed output word.  A warp per row left most lanes without a word: the query of four
// predicates on 500,000 elements took 311 us at n = 6 and 327 at n = 10, now 42 and 107; 200,000
// at n = 11 152 -> 98 us.  Short rows leave the launches and EvalAll (30 us), longer ones the row
// loads, each lane its own lines.
constexpr int kDotBatch = 8;                  // elements of a step of the staged pass
constexpr int kDotThreads = 256;
constexpr uint32_t kDotMaxWords = 64;

template <int VEC>
__device__ __forceinline__ void load_words(const uint32_t* p, uint32_t v[VEC]) {
    if constexpr (VEC == 4) {
        const uint4 q = *reinterpret_cast<const uint4*>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        v[0] = *p;
    }
}

template <int VEC>     // words per load: 4 where rows are whole 16-byte groups, else 1
__global__ void __launch_bounds__(kDotThreads) k_onehot_dots(const __grid_constant__ DotParams P) {
    __shared__ __align__(16) uint32_t hs[kDotPreds * 6 * kDotMaxWords];    // [predicate][server][half][word]
    const uint32_t W = P.words, np = P.n_preds;
    for (uint32_t t = threadIdx.x; t < np * 6 * W; t += kDotThreads) {
        const uint32_t k = t / (6 * W), r = t - k * 6 * W;
        hs[t] = P.hv[(uint64_t)P.half_base[k] * W + r];
    }
    __syncthreads();
    const uint64_t nwords = (P.n_elems + 31) / 32;
    for (uint64_t first = (uint64_t)blockIdx.x * kDotThreads; first < P.n_elems; first += (uint64_t)gridDim.x * kDotThreads) {
        const uint64_t e = first + threadIdx.x, wd = e / 32;
        uint32_t acc[kDotPreds][3];
#pragma unroll
        for (int k = 0; k < kDotPreds; k++) acc[k][0] = acc[k][1] = acc[k][2] = 0;
        if (e < P.n_elems) {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const uint32_t* row = P.share[j] + e * W;
                // share j meets server j's first half and server j - 1's second
                const uint32_t i0 = (uint32_t)j, i1 = (uint32_t)(j + 2) % 3;
#pragma unroll 2
                for (uint32_t w = 0; w < W; w += VEC) {
                    uint32_t v[VEC];
                    load_words<VEC>(row + w, v);
#pragma unroll
                    for (int k = 0; k < kDotPreds; k++) {
                        if ((uint32_t)k >= np) break;
                        uint32_t ha[VEC], hb[VEC];
                        load_words<VEC>(hs + (k * 6 + 2 * i0) * W + w, ha);
                        load_words<VEC>(hs + (k * 6 + 2 * i1 + 1) * W + w, hb);
#pragma unroll
                        for (int r = 0; r < VEC; r++) {
                            acc[k][i0] ^= v[r] & ha[r];
                            acc[k][i1] ^= v[r] & hb[r];
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kDotPreds; k++) {
            if ((uint32_t)k >= np) break;
#pragma unroll
            for (int i = 0; i < 3; i++) {
                const uint32_t z = __ballot_sync(0xFFFFFFFFu, __popc(acc[k][i]) & 1);
                if ((threadIdx.x & 31) == 0 && wd < nwords) P.zbits[k][(uint64_t)i * nwords + wd] = z;
            }
        }
    }
}

// The same pass for rows of W = 128 * WARPS words (2^12 <= D <= 2^16), persistent, with the
// element rows staged through shared memory so that two batches are always in flight while a
// third is combined, across words too.  Lane l of warp q owns words [128 q + 4 l, 128 q + 4 l + 4)
// of every row: it copies them with its own 16-byte cp.async into its own slots and reads back
// only those, so the pipeline needs no barrier.  A CTA takes a run of 16-element halves of output
// words (a 45th half is 2 % of a CTA's share of 107,614 elements, a 23rd word was 4 %), as
// chunks of 32 elements; a step is 8 elements of one share set.  Two chunks share the
// half-vector slices that their share set needs, loaded into registers a few steps ahead.
// With four predicates the AND / XOR work on the ALU pipe bounds it (4 bytes read are 8 such
// operations), so everything else is kept off that pipe: a compile-time row length makes a
// step's addresses immediates, one warp reduction instruction replaces five shuffle / XOR
// steps, popcounts are placed by multiply-adds.  107,614 elements, n = 16, four predicates:
// 453 -> 412 us, 6.4 TB/s.  (The binary matrix instruction m16n8k256 would do a step's work
// in 4 of them, but takes 127 cycles of an SM each: 3.5 times too slow.)
constexpr int kPipeStages = 3;
constexpr int kGroupChunks = 2;                       // 32-element chunks per load of the half vectors
constexpr int kBatches = 32 / kDotBatch;              // steps per (chunk, share set)
constexpr uint32_t kPipeSmemPerWarp = kPipeStages * kDotBatch * 32 * 16;

__device__ __forceinline__ void load_halves(const DotParams& P, uint32_t W, uint32_t w0, uint32_t np, int j,
                                            uint32_t h[kDotPreds][2][4]) {
#pragma unroll
    for (int k = 0; k < kDotPreds; k++) {
        if ((uint32_t)k < np) {
            // plain loads: a read-only one could move above grid_wait
            const uint4 a = *reinterpret_cast<const uint4*>(P.hv + (uint64_t)(P.half_base[k] + j * 2) * W + w0);
            const uint4 b = *reinterpret_cast<const uint4*>(
                P.hv + (uint64_t)(P.half_base[k] + ((j + 2) % 3) * 2 + 1) * W + w0);
            h[k][0][0] = a.x; h[k][0][1] = a.y; h[k][0][2] = a.z; h[k][0][3] = a.w;
            h[k][1][0] = b.x; h[k][1][1] = b.y; h[k][1][2] = b.z; h[k][1][3] = b.w;
        } else {
#pragma unroll
            for (int r = 0; r < 4; r++) h[k][0][r] = h[k][1][r] = 0;
        }
    }
}

// acc ^ (a & b) in one instruction
__device__ __forceinline__ uint32_t xor_and(uint32_t acc, uint32_t a, uint32_t b) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0x78;" : "=r"(d) : "r"(acc), "r"(a), "r"(b));
    return d;
}

// A CTA's steps in order: groups of kGroupChunks chunks, their share sets, their chunks, their
// batches of kDotBatch elements (a last chunk of one half has two).
struct DotSteps {
    uint32_t chunks, last_batches;     // chunks of the CTA; batches of its last one
    uint32_t group, share, chunk, batch;
    __device__ __forceinline__ uint32_t group_chunks() const {
        return min((uint32_t)kGroupChunks, chunks - group * kGroupChunks);
    }
    __device__ __forceinline__ uint32_t at() const { return group * kGroupChunks + chunk; }
    __device__ __forceinline__ uint32_t batches() const { return at() + 1 == chunks ? last_batches : (uint32_t)kBatches; }
    __device__ __forceinline__ bool done() const { return group * kGroupChunks >= chunks; }
    __device__ __forceinline__ void next() {
        if (++batch < batches()) return;
        batch = 0;
        if (++chunk < group_chunks()) return;
        chunk = 0;
        if (++share < 3) return;
        share = 0;
        group++;
    }
};

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_onehot_dots_pipe(const __grid_constant__ DotParams P) {
    extern __shared__ __align__(16) unsigned char dsmem[];
    constexpr uint32_t W = 128 * WARPS;
    // 2^i for i < 32 from the launch parameters: a runtime factor, so that shifts into place
    // are multiply-adds on the FMA pipe and leave the ALU pipe to the AND / XOR work
    const uint32_t* pw = P.pow2;
    // by group parity: masks per (chunk, share, warp, predicate and half)
    __shared__ __align__(16) uint32_t zs[2][kGroupChunks][3][WARPS][2 * kDotPreds];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t np = P.n_preds;
    const uint64_t nwords = (P.n_elems + 31) / 32, halves = 2 * nwords;
    const uint64_t half0 = blockIdx.x * halves / gridDim.x, half1 = (blockIdx.x + 1) * halves / gridDim.x;
    grid_trigger();
    const uint32_t mine_halves = (uint32_t)(half1 - half0);
    DotSteps F{};                                     // the next step to fetch
    F.chunks = (mine_halves + 1) / 2;
    F.last_batches = mine_halves % 2 ? kBatches / 2 : kBatches;
    const uint32_t w0 = warp * 128 + lane * 4;
    // slot (stage s, element b) of this lane: mine[(s * kDotBatch + b) * 32]
    uint4* const mine = reinterpret_cast<uint4*>(dsmem + (size_t)warp * kPipeSmemPerWarp) + lane;
    uint32_t fetch_stage = 0, stage = 0;
    const auto fetch = [&]() {
        if (!F.done()) {
            const uint64_t e0 = half0 * 16 + F.at() * 32u + F.batch * kDotBatch;
            uint4* dst = mine + fetch_stage * kDotBatch * 32;
            const uint32_t* src = P.share[F.share] + e0 * W + w0;
            if (e0 + kDotBatch <= P.n_elems) {
#pragma unroll
                for (int b = 0; b < kDotBatch; b++) cp_async16(dst + b * 32, src + (size_t)b * W, 16u);
            } else {
                // rows past the table's end are zero-filled, nothing read
#pragma unroll
                for (int b = 0; b < kDotBatch; b++) {
                    const bool ok = e0 + b < P.n_elems;
                    cp_async16(dst + b * 32, ok ? src + (size_t)b * W : P.share[F.share] + w0, ok ? 16u : 0u);
                }
            }
            F.next();
        }
        cp_async_commit();                            // an empty group keeps the count uniform
        fetch_stage = fetch_stage + 1 == kPipeStages ? 0 : fetch_stage + 1;
    };
    for (int d = 0; d < kPipeStages - 1; d++) fetch();    // the table's rows do not depend on EvalAll
    grid_wait();
    uint32_t h[kDotPreds][2][4], hn[kDotPreds][2][4];
    load_halves(P, W, w0, np, 0, h);
    const uint32_t chunks = F.chunks, last_batches = F.last_batches;
#pragma unroll 1
    for (uint32_t c0 = 0; c0 < chunks; c0 += kGroupChunks) {
        const uint32_t nch = min((uint32_t)kGroupChunks, chunks - c0), par = (c0 / kGroupChunks) & 1u;
#pragma unroll 1
        for (int j = 0; j < 3; j++) {
#pragma unroll 1
            for (uint32_t ch = 0; ch < nch; ch++) {
                const uint32_t nb = c0 + ch + 1 == chunks ? last_batches : (uint32_t)kBatches;
                uint32_t pl[kDotPreds][2];
#pragma unroll
                for (int k = 0; k < kDotPreds; k++) pl[k][0] = pl[k][1] = 0;
#pragma unroll
                for (int cb = 0; cb < kBatches; cb++) {
                    if (cb >= kBatches / 2 && cb >= (int)nb) break;
                    fetch();
                    cp_async_wait<kPipeStages - 1>();     // this lane's copies of the step have landed
                    if (cb == 1 && ch + 1 == nch) load_halves(P, W, w0, np, j < 2 ? j + 1 : 0, hn);
                    const uint4* slot = mine + stage * kDotBatch * 32;
                    stage = stage + 1 == kPipeStages ? 0 : stage + 1;
                    uint32_t v[kDotBatch][4];
#pragma unroll
                    for (int b = 0; b < kDotBatch; b++) {
                        const uint4 x = slot[b * 32];
                        v[b][0] = x.x; v[b][1] = x.y; v[b][2] = x.z; v[b][3] = x.w;
                    }
#pragma unroll
                    for (int k = 0; k < kDotPreds; k++) {
                        if ((uint32_t)k >= np) break;
#pragma unroll
                        for (int hh = 0; hh < 2; hh++) {
                            uint32_t cnt[kDotBatch / 4] = {};
#pragma unroll
                            for (int b = 0; b < kDotBatch; b++) {
                                uint32_t a = v[b][0] & h[k][hh][0];
                                a = xor_and(a, v[b][1], h[k][hh][1]);
                                a = xor_and(a, v[b][2], h[k][hh][2]);
                                a = xor_and(a, v[b][3], h[k][hh][3]);
                                // popcount into byte b % 4 by a multiply-add (the FMA pipe, not the ALU)
                                cnt[b / 4] = (uint32_t)__popc(a) * pw[8 * (b % 4)] + cnt[b / 4];
                            }
                            // bit 8 f + q, q = cb * (kDotBatch / 4) + (b / 4): shifted by a multiply
#pragma unroll
                            for (int q = 0; q < kDotBatch / 4; q++) {
                                constexpr uint32_t M = 0x01010101u;
                                const int sh = cb * (kDotBatch / 4) + q;
                                pl[k][hh] = xor_and(pl[k][hh], cnt[q] * pw[sh], M << sh);
                            }
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < kDotPreds; k++) {
                    if ((uint32_t)k >= np) break;
#pragma unroll
                    for (int hh = 0; hh < 2; hh++) {
                        const uint32_t m = __reduce_xor_sync(0xFFFFFFFFu, pl[k][hh]);
                        if (lane == 0) zs[par][ch][j][warp][2 * k + hh] = m;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < kDotPreds; k++)
#pragma unroll
                for (int hh = 0; hh < 2; hh++)
#pragma unroll
                    for (int r = 0; r < 4; r++) h[k][hh][r] = hn[k][hh][r];
        }
        // the group's masks are complete: combine the warps' and write the packed bits, a half
        // word at a time.  zs is double-buffered by group parity, so one barrier per group suffices.
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < nch * np * 3; t += WARPS * 32) {
            const uint32_t ch = t / (np * 3), k = t / 3 % np, i = t % 3;
            uint32_t zp = 0;
#pragma unroll
            for (int q = 0; q < WARPS; q++) zp ^= zs[par][ch][i][q][2 * k] ^ zs[par][ch][(i + 1) % 3][q][2 * k + 1];
            // element c sits at bit 8 (c % 4) + c / 4
            uint32_t z = 0;
#pragma unroll
            for (uint32_t c = 0; c < 32; c++) z |= ((zp >> (8 * (c % 4) + c / 4)) & 1u) << c;
            uint16_t* out = reinterpret_cast<uint16_t*>(P.zbits[k] + (uint64_t)i * nwords) + half0 + 2 * (c0 + ch);
            out[0] = (uint16_t)z;
            if (c0 + ch + 1 < chunks || last_batches == kBatches) out[1] = (uint16_t)(z >> 16);
        }
    }
    cp_async_wait<0>();
}

template <int WARPS>
void launch_dots_pipe(const DotParams& D, uint64_t nwords, int sm_count, cudaStream_t s) {
    // persistent: as many CTAs as fit on the SMs (one of 16 warps per SM at D = 2^16)
    constexpr uint32_t smem = WARPS * kPipeSmemPerWarp;
    const uint32_t per_sm = std::max<uint32_t>(1, std::min<uint32_t>(227u * 1024 / (smem + 4096), 32 / WARPS));
    const uint64_t grid = std::min<uint64_t>(nwords, (uint64_t)sm_count * per_sm);
    launch_after(k_onehot_dots_pipe<WARPS>, (unsigned)grid, WARPS * 32, smem, s, D);
}

void launch_dots(const DotParams& D, uint64_t nwords, int sm_count, cudaStream_t s) {
    switch (D.words / 128) {
        case 1: return launch_dots_pipe<1>(D, nwords, sm_count, s);
        case 2: return launch_dots_pipe<2>(D, nwords, sm_count, s);
        case 4: return launch_dots_pipe<4>(D, nwords, sm_count, s);
        case 8: return launch_dots_pipe<8>(D, nwords, sm_count, s);
        case 16: return launch_dots_pipe<16>(D, nwords, sm_count, s);
        default: {                                     // D < 2^12
            const unsigned grid = (unsigned)std::min<uint64_t>((D.n_elems + kDotThreads - 1) / kDotThreads, 8ull * sm_count);
            if (D.words % 4 == 0) k_onehot_dots<4><<<grid, kDotThreads, 0, s>>>(D);
            else k_onehot_dots<1><<<grid, kDotThreads, 0, s>>>(D);
        }
    }
}

// All groups of a query in one launch: each element's predicate bits are re-shared in
// binary RSS and folded in token order.  The re-share PRF gives the bits of 128
// consecutive elements from one AES block (bit e mod 128 of AES_k(c), c = u64 (e div 128)
// | 2^63 || u16 step || u16 table || u32 query), and word q of that block holds the bits
// of the block's output word q, so a warp takes one (group, 128 elements) item and
// works on whole 32-element words: lane 4 b + q (b < 6) computes PRF block b (the three
// servers' keys at the predicate's step, then at its fold step) and keeps word q; shuffles
// bring each word's six PRF words to lane q, which re-shares, folds and stores word q.
// The AES reads the bank-replicated shared-memory T-tables (one persistent CTA per SM).
struct FoldGroup {
    uint32_t* out[3];
    uint64_t n_elems;
    uint64_t item_begin;     // first item (128-element block) of the group in the launch
    uint32_t first;          // index of the group's first predicate in zoff / steps
    uint32_t n_preds;
    uint32_t table_id;
    uint32_t pad;
};

struct FoldParams {
    uint32_t rk_prf[3][44];
    const uint32_t* te0;
    const uint32_t* zbase;             // the query's packed predicate bits
    const uint64_t* zoff;              // per predicate (group order): word offset of its [3][nwords] block
    const uint32_t* steps;             // per predicate: its index in the token | combine << 16
    const FoldGroup* groups;
    uint64_t total_items;
    uint32_t n_groups;
    uint32_t query_id;
};

constexpr int kFoldThreads = 768;
constexpr uint32_t kFoldBlockElems = 128;

__global__ void __launch_bounds__(kFoldThreads, 1) k_onehot_fold(const __grid_constant__ FoldParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    fill_tables(reinterpret_cast<uint32_t*>(smem), P.te0);
    grid_wait();
    __syncthreads();
    const SmemTab T{reinterpret_cast<const char*>(smem), lane_offset()};
    const uint32_t lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    // this lane's PRF block: b = 0..2 server b's key at the step, 3..5 at the fold step
    // (lanes 24..31 repeat lanes 16..23; they keep a word nobody reads)
    const uint32_t b = lane < 24 ? lane >> 2 : (lane >> 2) - 2, q = lane & 3;
    const uint32_t* rk = P.rk_prf[b % 3];
    for (uint64_t item = (uint64_t)blockIdx.x * warps + (threadIdx.x >> 5); item < P.total_items;
         item += (uint64_t)gridDim.x * warps) {
        uint32_t g = 0;
        while (g + 1 < P.n_groups && P.groups[g + 1].item_begin <= item) g++;
        const FoldGroup& G = P.groups[g];
        const uint64_t nwords = (G.n_elems + 31) / 32;
        const uint64_t blk = item - G.item_begin;
        const uint64_t wd = blk * 4 + q;                  // this lane's output word
        const bool have = wd < nwords;
        const uint64_t rem = have ? G.n_elems - wd * 32 : 0;
        const uint32_t valid = rem >= 32 ? 0xFFFFFFFFu : ((1u << rem) - 1u);
        const uint32_t c0 = (uint32_t)blk, c1 = (uint32_t)(blk >> 32) | 0x80000000u;
        uint32_t acc[3] = {0, 0, 0};
        for (uint32_t k = 0; k < G.n_preds; k++) {
            const uint64_t zo = P.zoff[G.first + k];
            const uint32_t sc = P.steps[G.first + k];
            const uint32_t step = sc & 0xFFFFu, combine = sc >> 16;
            // the predicate's bits of this word, loaded before the PRF's AES so the loads overlap it
            uint32_t z[3], r[3];
#pragma unroll
            for (int i = 0; i < 3; i++) z[i] = have ? P.zbase[zo + (uint64_t)i * nwords + wd] : 0u;
            uint32_t f = 0;
            if (b < 3 || k > 0) {
                const uint32_t ctr[4] = {c0, c1, (b < 3 ? step : 64u + step) | (G.table_id << 16), P.query_id};
                uint32_t o[4];
                aes_one(T, rk, ctr, o);
                f = q == 0 ? o[0] : q == 1 ? o[1] : q == 2 ? o[2] : o[3];
            }
            uint32_t F[6];
#pragma unroll
            for (int s = 0; s < 6; s++) F[s] = __shfl_sync(0xFFFFFFFFu, f, 4 * s + (int)q);
            // binary re-share: r_i = z_i xor F(k_i) xor F(k_{i-1})
#pragma unroll
            for (int i = 0; i < 3; i++) r[i] = z[i] ^ F[i] ^ F[(i + 2) % 3];
            if (k == 0) {
                acc[0] = r[0]; acc[1] = r[1]; acc[2] = r[2];
            } else {
                // fold over Z_2 (Sec. V-D): AND = a b, XOR = a ^ b, OR = a ^ b ^ a b
                const uint32_t lin = combine == OBLIVGM_COMBINE_AND ? 0u : 0xFFFFFFFFu;
                const uint32_t prod = combine == OBLIVGM_COMBINE_XOR ? 0u : 0xFFFFFFFFu;
                uint32_t w[3];
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    const int i1 = (i + 1) % 3;
                    const uint32_t pr = (acc[i] & r[i]) ^ (acc[i] & r[i1]) ^ (acc[i1] & r[i]);
                    w[i] = ((acc[i] ^ r[i]) & lin) ^ (pr & prod);
                }
#pragma unroll
                for (int i = 0; i < 3; i++) acc[i] = w[i] ^ F[3 + i] ^ F[3 + (i + 2) % 3];
            }
        }
        if (lane < 4 && have) {
#pragma unroll
            for (int i = 0; i < 3; i++) G.out[i][wd] = acc[i] & valid;
        }
    }
}

}  // namespace

}  // namespace ogm

// ====================================================================== host side

using namespace ogm;

extern "C" oblivgm_status oblivgm_keygen_onehot(const oblivgm_pred* preds, uint32_t n_preds, uint32_t n_bits,
                                                const uint8_t seed[16], uint8_t* const tok[3], size_t cap,
                                                size_t out_len[3]) {
    const NvtxRange nvtx_range("oblivgm_keygen_onehot");
    std::string err;
    oblivgm_status st = keygen(preds, n_preds, n_bits, seed, tok, cap, out_len, &err, /*onehot=*/true);
    if (st != OBLIVGM_OK) return fail(st, err);
    return OBLIVGM_OK;
}

extern "C" oblivgm_status oblivgm_load_onehot(oblivgm_ctx* ctx, uint32_t table_id, uint64_t n_elems,
                                              uint32_t n_attrs, uint32_t n_bits,
                                              const uint32_t* const share_sets[3], int32_t mem_kind, void* stream) {
    const NvtxRange nvtx_range("oblivgm_load_onehot");
    if (!ctx) return fail(OBLIVGM_EINVAL, "NULL context");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    if (table_id > 0xFFFF || n_attrs == 0 || n_attrs > 65536 || n_bits < 1 || n_bits > (uint32_t)kMaxOnehotBits ||
        !share_sets)
        return fail(OBLIVGM_EINVAL, "bad one-hot table arguments");
    if (mem_kind != OBLIVGM_MEM_HOST && mem_kind != OBLIVGM_MEM_DEVICE) return fail(OBLIVGM_EINVAL, "bad mem_kind");
    for (int j = 0; j < 3; j++)
        if (!share_sets[j] && n_elems) return fail(OBLIVGM_EINVAL, "NULL share set");
    const uint32_t words = n_bits >= 5 ? (1u << n_bits) / 32 : 1u;
    const size_t set_words = (size_t)n_attrs * n_elems * words;
    const size_t bytes = 3 * set_words * sizeof(uint32_t);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    auto it = ctx->onehot_tables.find(table_id);
    if (it != ctx->onehot_tables.end()) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "stream synchronize");
        cudaFree(it->second.dev);
        ctx->onehot_tables.erase(it);
    }
    OnehotTable tb{};
    tb.n_elems = n_elems; tb.n_attrs = n_attrs; tb.n_bits = n_bits; tb.words = words; tb.bytes = bytes;
    e = cudaMalloc(&tb.dev, std::max<size_t>(bytes, 16));
    if (e != cudaSuccess) return cuda_fail(e, "one-hot table allocation");
    ctx->onehot_tables[table_id] = tb;
    const cudaMemcpyKind kind = mem_kind == OBLIVGM_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    for (int j = 0; j < 3 && set_words; j++) {
        e = cudaMemcpyAsync(tb.dev + j * set_words, share_sets[j], set_words * sizeof(uint32_t), kind, s);
        if (e != cudaSuccess) return cuda_fail(e, "one-hot share upload");
    }
    if (mem_kind == OBLIVGM_MEM_HOST) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "stream synchronize");
    }
    return OBLIVGM_OK;
}

extern "C" oblivgm_status oblivgm_filter_onehot(oblivgm_ctx* ctx, uint32_t query_id, const uint8_t* const tok[3],
                                                const size_t tok_len[3], uint32_t n_groups, uint32_t* const* out,
                                                void* stream) {
    const NvtxRange nvtx_range("oblivgm_filter_onehot");
    if (!ctx || !tok || !tok_len || !out) return fail(OBLIVGM_EINVAL, "NULL argument");
    cudaError_t ce = cudaSetDevice(ctx->device);
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaSetDevice");
    ParsedQuery q;
    std::string err;
    oblivgm_status st = parse_tokens(tok, tok_len, &q, &err);
    if (st != OBLIVGM_OK) return fail(st, err);
    if (q.out_group != 1) return fail(OBLIVGM_EINVAL, "a masked-mode token was given to the one-hot evaluation");
    if (n_groups == 0 || n_groups > OBLIVGM_MAX_GROUPS) return fail(OBLIVGM_EINVAL, "n_groups must be 1..64");
    std::vector<std::vector<uint32_t>> members(n_groups);   // predicate indices per group
    for (uint32_t p = 0; p < q.preds.size(); p++) {
        if (q.preds[p].group >= n_groups) return fail(OBLIVGM_EINVAL, "predicate group outside 0..n_groups-1");
        members[q.preds[p].group].push_back(p);
    }
    for (uint32_t g = 0; g < n_groups; g++) {
        if (members[g].empty()) return fail(OBLIVGM_EINVAL, "an AND-group has no predicate");
        const ParsedPred& p0 = q.preds[members[g][0]];
        auto it = ctx->onehot_tables.find(p0.table);
        if (it == ctx->onehot_tables.end()) return fail(OBLIVGM_ENOENT, "predicate on a one-hot table that is not loaded");
        for (uint32_t p : members[g]) {
            const ParsedPred& pp = q.preds[p];
            if (pp.table != p0.table) return fail(OBLIVGM_EINVAL, "an AND-group spans two tables");
            if (pp.attr >= it->second.n_attrs) return fail(OBLIVGM_EINVAL, "predicate attribute outside its table");
            if (pp.n != it->second.n_bits) return fail(OBLIVGM_EINVAL, "predicate domain differs from its table's");
        }
    }
    const uint32_t n = q.n_bits, domain = 1u << n, words = n >= 5 ? domain / 32 : 1u;
    // device keys and half descriptors: six halves per predicate, [server][half]
    std::vector<EtKey> keys;
    std::vector<HalfDesc> halves;
    for (const ParsedPred& pp : q.preds) {
        const bool eq = pp.kind == OBLIVGM_PRED_EQ;
        const uint32_t nsub = eq ? 1 : 2, k0 = (uint32_t)keys.size();
        keys.insert(keys.end(), pp.et_keys.begin(), pp.et_keys.end());
        for (uint32_t hh = 0; hh < 6; hh++) {
            HalfDesc h{};
            h.key0 = k0 + hh * nsub;
            h.key1 = eq ? kNoKey : k0 + hh * nsub + 1;
            h.kind = eq ? OBLIVGM_KEY_DPF : OBLIVGM_KEY_DCF;
            h.cbit = (!eq && pp.et_keys[hh * nsub].party == 0) ? (pp.cbeta & 1u) : 0u;
            halves.push_back(h);
        }
    }
    // packed predicate bits: per predicate [3][ceil(n_elems / 32)] words of its table
    std::vector<uint64_t> zoff(q.preds.size());
    uint64_t zwords = 0;
    for (uint32_t p = 0; p < q.preds.size(); p++) {
        const OnehotTable& tb = ctx->onehot_tables.at(q.preds[p].table);
        zoff[p] = zwords;
        zwords += 3 * ((tb.n_elems + 31) / 32);
    }
    // per group, the word offsets and token steps of its predicates (token order)
    std::vector<uint64_t> gzoff;
    std::vector<uint32_t> gstep;
    std::vector<size_t> gbegin;
    for (uint32_t g = 0; g < n_groups; g++) {
        gbegin.push_back(gzoff.size());
        for (uint32_t p : members[g]) {
            gzoff.push_back(zoff[p]);
            gstep.push_back(q.preds[p].step | q.preds[p].combine << 16);
        }
    }
    const size_t np = gzoff.size();
    // fold descriptors: the groups with elements, each with its first item
    std::vector<FoldGroup> fg;
    uint64_t fold_items = 0;
    for (uint32_t g = 0; g < n_groups; g++) {
        const OnehotTable& tb = ctx->onehot_tables.at(q.preds[members[g][0]].table);
        if (tb.n_elems == 0) continue;
        FoldGroup G{};
        for (int j = 0; j < 3; j++) {
            G.out[j] = out[3 * g + j];
            if (!G.out[j]) return fail(OBLIVGM_EINVAL, "NULL output pointer");
        }
        G.n_elems = tb.n_elems;
        G.item_begin = fold_items;
        G.first = (uint32_t)gbegin[g];
        G.n_preds = (uint32_t)members[g].size();
        G.table_id = q.preds[members[g][0]].table;
        fg.push_back(G);
        fold_items += (tb.n_elems + kFoldBlockElems - 1) / kFoldBlockElems;
    }
    // scratch: keys | halves | group offsets | group steps | key slots | fold groups | half vectors |
    // predicate bits
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t off_h = up(keys.size() * sizeof(EtKey));
    const size_t off_o = off_h + up(halves.size() * sizeof(HalfDesc));
    const size_t off_s = off_o + up(np * sizeof(uint64_t));
    std::vector<KeySlot> slots;             // DPF keys first, then DCF keys
    for (uint32_t kind = 0; kind < 2; kind++)
        for (uint32_t h = 0; h < halves.size(); h++) {
            const HalfDesc& H = halves[h];
            const uint32_t dcf = H.kind == OBLIVGM_KEY_DCF ? 1u : 0u;
            if (dcf != kind) continue;
            slots.push_back(KeySlot{H.key0, h, H.cbit ? 0xFFFFFFFFu : 0u, dcf});
            if (H.key1 != kNoKey) slots.push_back(KeySlot{H.key1, h, 0u, dcf});
        }
    const size_t off_k = off_s + up(np * sizeof(uint32_t));
    const size_t off_g = off_k + up(slots.size() * sizeof(KeySlot));
    const size_t off_v = off_g + up(fg.size() * sizeof(FoldGroup));
    const size_t off_z = off_v + up(halves.size() * words * sizeof(uint32_t));
    const size_t total = off_z + zwords * sizeof(uint32_t);
    std::vector<unsigned char> img(off_v, 0);
    std::memcpy(img.data(), keys.data(), keys.size() * sizeof(EtKey));
    std::memcpy(img.data() + off_h, halves.data(), halves.size() * sizeof(HalfDesc));
    std::memcpy(img.data() + off_o, gzoff.data(), np * sizeof(uint64_t));
    std::memcpy(img.data() + off_s, gstep.data(), np * sizeof(uint32_t));
    std::memcpy(img.data() + off_k, slots.data(), slots.size() * sizeof(KeySlot));
    if (!fg.empty()) std::memcpy(img.data() + off_g, fg.data(), fg.size() * sizeof(FoldGroup));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char* ws = nullptr;
    {
        const oblivgm_status as = ws_alloc(ctx, reinterpret_cast<void**>(&ws), total, s, "one-hot scratch");
        if (as != OBLIVGM_OK) return as;
    }
    ScratchGuard guard(ws, s);
    ce = cudaMemcpyAsync(ws, img.data(), off_v, cudaMemcpyHostToDevice, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "one-hot descriptor upload");
    uint32_t* zbase = reinterpret_cast<uint32_t*>(ws + off_z);
    uint32_t* hv = reinterpret_cast<uint32_t*>(ws + off_v);
    ce = cudaMemsetAsync(hv, 0, halves.size() * words * sizeof(uint32_t), s);
    if (ce != cudaSuccess) return cuda_fail(ce, "half-vector clear");
    {
        EvalEtParams E{};
        E.aes = ctx->aes;
        E.te0 = ctx->d_te0;
        E.keys = reinterpret_cast<const EtKey*>(ws);
        E.slots = reinterpret_cast<const KeySlot*>(ws + off_k);
        E.hv = hv;
        E.words = words;
        E.leaves = 1u << (n - (uint32_t)et_low_bits((int)n));
        E.n_slots = (uint32_t)slots.size();
        const uint64_t items = (uint64_t)E.n_slots * E.leaves;
        // one CTA per SM (the tables take 128 KiB), as many threads as give every item a lane pair
        const uint64_t per_sm = (2 * items + ctx->sm_count - 1) / ctx->sm_count;
        const unsigned threads = (unsigned)std::min<uint64_t>(kEvalEtMaxThreads, std::max<uint64_t>(64, (per_sm + 31) / 32 * 32));
        const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((2 * items + threads - 1) / threads,
                                                                                 (uint64_t)ctx->sm_count));
        k_onehot_evalall_et<<<grid, threads, kTableBytes, s>>>(E);
    }
    ctx->launches++;
    // one streaming pass per (table, attribute) for up to kDotPreds predicates on it
    std::map<std::pair<uint32_t, uint32_t>, std::vector<uint32_t>> by_column;
    for (uint32_t p = 0; p < q.preds.size(); p++) by_column[{q.preds[p].table, q.preds[p].attr}].push_back(p);
    for (auto& col : by_column) {
        const OnehotTable& tb = ctx->onehot_tables.at(col.first.first);
        if (tb.n_elems == 0) continue;
        const size_t set_words = (size_t)tb.n_attrs * tb.n_elems * tb.words;
        const uint64_t nwords = (tb.n_elems + 31) / 32;
        const std::vector<uint32_t>& ps = col.second;
        for (size_t c0 = 0; c0 < ps.size(); c0 += kDotPreds) {
            DotParams D{};
            for (int j = 0; j < 3; j++) D.share[j] = tb.dev + j * set_words + (size_t)col.first.second * tb.n_elems * tb.words;
            D.hv = hv;
            D.n_preds = (uint32_t)std::min<size_t>(kDotPreds, ps.size() - c0);
            for (uint32_t k = 0; k < D.n_preds; k++) {
                D.half_base[k] = 6 * ps[c0 + k];
                D.zbits[k] = zbase + zoff[ps[c0 + k]];
            }
            D.n_elems = tb.n_elems;
            D.words = words;
            for (int i = 0; i < 32; i++) D.pow2[i] = 1u << i;
            launch_dots(D, nwords, ctx->sm_count, s);
            ctx->launches++;
        }
    }
    // every AND-group in one launch: binary re-share and fold, packed outputs
    if (!fg.empty()) {
        FoldParams F{};
        std::memcpy(F.rk_prf, ctx->rk_prf, sizeof F.rk_prf);
        F.te0 = ctx->d_te0;
        F.zbase = zbase;
        F.zoff = reinterpret_cast<const uint64_t*>(ws + off_o);
        F.steps = reinterpret_cast<const uint32_t*>(ws + off_s);
        F.groups = reinterpret_cast<const FoldGroup*>(ws + off_g);
        F.total_items = fold_items;
        F.n_groups = (uint32_t)fg.size();
        F.query_id = query_id;
        // a warp per item: as many warps per CTA as spread the items over every SM (at least 4)
        const uint64_t warps = std::min<uint64_t>(kFoldThreads / 32, std::max<uint64_t>(
                                                      4, (fold_items + ctx->sm_count - 1) / ctx->sm_count));
        const unsigned grid = (unsigned)std::min<uint64_t>((fold_items + warps - 1) / warps, (uint64_t)ctx->sm_count);
        launch_after(k_onehot_fold, grid, (unsigned)(warps * 32), kTableBytes, s, F);
        ctx->launches++;
    }
    ce = cudaGetLastError();
    if (ce != cudaSuccess) return cuda_fail(ce, "one-hot launch");
    guard.done();
    ce = cudaFreeAsync(ws, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "one-hot scratch release");
    return OBLIVGM_OK;
}

namespace ogm {

template <int WARPS>
static cudaError_t dots_pipe_attr() {
    return cudaFuncSetAttribute(k_onehot_dots_pipe<WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                WARPS * (int)kPipeSmemPerWarp);
}

oblivgm_status set_onehot_attrs() {
    cudaError_t e = cudaFuncSetAttribute(k_onehot_evalall_et, cudaFuncAttributeMaxDynamicSharedMemorySize, kTableBytes);
    if (e == cudaSuccess) e = dots_pipe_attr<1>();
    if (e == cudaSuccess) e = dots_pipe_attr<2>();
    if (e == cudaSuccess) e = dots_pipe_attr<4>();
    if (e == cudaSuccess) e = dots_pipe_attr<8>();
    if (e == cudaSuccess) e = dots_pipe_attr<16>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_onehot_fold, cudaFuncAttributeMaxDynamicSharedMemorySize, kTableBytes);
    return e == cudaSuccess ? OBLIVGM_OK : cuda_fail(e, "one-hot kernel attributes");
}

}  // namespace ogm
