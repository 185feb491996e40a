// staged.h -- host side of the staged masked-mode evaluation (staged.cu): the descriptors it
// shares with the fused kernels, its plan and its launch.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "host_crypto.h"
#include "oblivgm.h"

struct oblivgm_ctx;

namespace ogm {

struct StagedLimits;

// One AND-group of a launch.
struct GroupDesc {
    const uint32_t* share[3];   // share set j of the group's table: [attr][stride]
    uint32_t* out[3];           // RSS share sets of the result, n_elems each
    uint64_t stride;
    uint64_t n_elems;
    uint32_t query_id, table_id, pred_begin, n_preds;
    uint32_t vec_out;           // out pointers are 16-byte aligned
    uint32_t tile;              // elements per work item of this group (k_filter_wp; k_filter uses the launch's)
    uint32_t slots;             // k_filter_wp: walk threads per element, 6 (equality predicates only) or 12
    uint32_t pad;
};

// One predicate of a launch.
struct PredDesc {
    uint32_t kind, n_bits, attr, step;
    uint32_t r[3];
    uint32_t cbeta;
    uint32_t key_begin, n_keys;
    // fold into the group's result: w_i = lin (a_i + b_i) + prod (a_i b_i + a_i b_{i+1} + a_{i+1} b_i)
    uint32_t lin, prod;
};

constexpr int kSgMaxStages = 33;

// One opened column of the launch (an attribute of a table, all its elements).
struct SgCol {
    const uint32_t* share[3];   // the column's three share rows (points of a raw evaluation: one row, twice NULL)
    uint64_t n;                 // elements
    uint32_t radd;              // <r>_1 + <r>_2 + <r>_3 of the first predicate on it
    uint32_t mask;              // 2^n_bits - 1
    uint32_t passes;            // radix passes of 8 bits; 0: the column is dense (not sorted)
    uint32_t tiles;             // sort tiles
    uint32_t* key[2];           // opened values, ping-pong; key[(passes + 1) & 1] ends up as the distinct values
    uint32_t* idx[2];           // their elements
    uint32_t* hist;             // [256][tiles] digit counts, then their exclusive sums; [tiles] for the distinct count
    uint32_t* tot;              // [256] digit totals
    uint32_t* rank;             // element -> index of its value among the distinct ones
    uint32_t* m;                // number of distinct values
};

// One predicate of the launch.
struct SgPred {
    uint32_t kind, n, n_keys, key_begin;
    uint32_t mask, delta;       // x^ = (u + delta) & mask for a distinct value u of the column
    uint32_t cbeta;
    uint32_t dense;             // the column's values are 0 .. 2^n - 1, no sort
    uint32_t chunk;             // distinct values evaluated together (a power of two)
    uint32_t stages;            // levels lev[s-1] .. lev[s] - 1 belong to stage s; lev[stages - 1] = n
    uint32_t slots;             // outputs per value: 3 servers, or one per key (raw evaluation)
    uint32_t col;
    uint64_t z_elem, z_slot;    // output word of (value i, slot q): z[i * z_elem + q * z_slot], part w of
                                // it 4 w further
    const uint32_t* u;          // distinct values (sorted), *m of them
    const uint32_t* m;
    uint32_t* z;
    uint4* st[2];               // seeds after a stage, [key][cap], control bit in bit 0 of word 0
    uint32_t* v[2];             // DCF value sums after a stage, [key][cap]
    uint32_t cap[2];
    uint32_t* pre;              // runs: prefix values; stage s at pre_off[s]
    uint32_t* par;              // runs: parent run of the stage before
    uint32_t* par_last;         // parent run of every value of the chunk
    uint32_t* blk;              // [stages - 1][blocks] run counts per block, then exclusive sums
    uint32_t* cnt;              // [stages - 1] runs of each stage
    uint32_t blocks;            // blocks of kRunBlock values in a chunk
    uint32_t parts;             // last stage: work units an output is split into (1, or its keys)
    uint64_t pre_off[kSgMaxStages];
    uint8_t lev[kSgMaxStages + 3];
};

// The predicates of one group that a round combines.
struct SgGroup {
    const uint32_t* share[3];
    uint32_t* out[3];
    uint64_t stride, n_elems;
    uint64_t item_begin;        // first tile of the group in the round
    uint32_t query_id, table_id;
    uint32_t pred_begin, n_preds;   // in the launch's predicate list
    uint32_t first;             // 1: the group's first predicate is among them; 0: the result so far is in out
    uint32_t pad;
};

struct SgFold {                 // per predicate, next to SgPred
    uint32_t step, lin, prod, attr;
    uint32_t radd, mask;
    uint32_t index;             // kIndexRank, kIndexDense or kIndexElem: which sums are element e's
    uint32_t more;              // further parts of the sums
    const uint32_t* rank;
    const uint32_t* z;          // per value and part four words: the three servers' sums
};
constexpr uint32_t kIndexRank = 0;    // those of value rank[e]
constexpr uint32_t kIndexDense = 1;   // those of value x^, opened from the shares
constexpr uint32_t kIndexElem = 2;    // those of element e (fresh keys)

// The re-share and fold over predicates' sums: tile shape for `elems` elements in all with at most
// most_preds predicates in a group entry, the entries' first tiles (returns the tiles), launch.
struct CombineShape {
    uint32_t threads = 0, per_thread = 1;
};
CombineShape combine_shape(uint64_t elems, uint32_t most_preds, int sm_count);
uint64_t combine_tiles(const CombineShape& c, SgGroup* groups, uint32_t n_groups);
void launch_combine(oblivgm_ctx* ctx, const CombineShape& c, const SgGroup* groups, uint32_t n_groups,
                    const SgFold* folds, bool split, uint64_t items, cudaStream_t s);

struct StagedRound {
    uint32_t pred_begin = 0, n_preds = 0;
    uint32_t group_begin = 0, n_groups = 0;
    uint32_t max_stages = 0, chunks = 0, sparse = 0, max_blocks = 0;
    uint64_t items = 0;
};

// Host recipe of a staged launch: sizes first, pointers when the memory is there.
struct Staged {
    std::vector<SgCol> cols;
    std::vector<SgPred> preds;
    std::vector<SgFold> folds;
    std::vector<SgGroup> groups;
    std::vector<StagedRound> rounds;
    uint32_t n_keys = 0, sort_tiles = 0, sort_passes = 0;
    CombineShape shape;
    bool split = false;         // last stages of a unit per key
    bool sort_large = false;    // sort tiles of 4,096 keys instead of 1,024
    bool raw = false;           // a raw evaluation: no combine, its keys are elsewhere on the device
    size_t off_preds = 0, off_folds = 0, off_groups = 0, off_keys = 0, image_bytes = 0;
    size_t scratch_bytes = 0;
};

// Plans the staged evaluation of a launch; false when it does not pay (or does not apply) and
// the fused kernels should run.  fixed: what it takes beside its kernels; wp_seconds: the
// walk-parallel kernel's time where that is the fused kernel of the launch, else 0.
bool staged_plan(const std::vector<GroupDesc>& groups, const std::vector<PredDesc>& preds, size_t n_keys, int sm_count,
                 const StagedLimits& limits, double fixed, double wp_seconds, Staged* out);

// Sets the pointers for scratch at a device address and builds the descriptor image's bytes.
void staged_image(Staged* sg, const DevKey* keys, unsigned char* scratch, std::vector<unsigned char>* bytes);

// Launches it on an image in device memory: no host work beyond the launches, no allocation,
// capturable.
oblivgm_status staged_launch(oblivgm_ctx* ctx, const Staged& sg, const unsigned char* image, cudaStream_t s);
uint64_t staged_launches(const Staged& sg);     // kernels of one launch

// Raw evaluation of n_keys keys of one kind at the same n_points points (OBLIVGM_ALL_PAIRS):
// plan (false: does not pay) and launch; out[k * n_points + i] = Eval(key k, points[i]).
bool staged_plan_raw(uint32_t kind, uint32_t n_bits, uint32_t n_keys, const uint32_t* points, uint64_t n_points,
                     const StagedLimits& limits, Staged* out);
oblivgm_status staged_launch_raw(oblivgm_ctx* ctx, const Staged& sg, const unsigned char* image, const DevKey* keys,
                                 uint32_t* out, cudaStream_t s);

oblivgm_status set_staged_attrs();

}  // namespace ogm
