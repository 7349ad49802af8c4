// Library-internal declarations shared by the esspt .cu translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "esspt.h"

namespace esspt {

// Latched device error bits (status word in the workspace).
enum : uint32_t {
  kErrStale = 1u,     // a read version broke the staleness bound
  kErrRowRange = 2u,  // a GET/INC row id outside [0, n_rows)
  kErrInput = 4u,     // an MF input index outside its range
};

// Word of the context's status block (after the error bits) that receives
// the oldest row version a row-granular GET read.
constexpr int kGetMinWord = 16;

// Counter-generator stream ids of the schedule.
constexpr uint64_t kStreamPhase = 101u;
constexpr uint64_t kStreamDelay = 102u;

// Users with more than kHeavy entries in a minibatch are split in chunks of
// kChunk entries, each a work item of its own.
constexpr int32_t kHeavy = 96;
constexpr int32_t kChunk = 64;
// The work list is sorted by length within tiles of 2^kTileBits users: the
// items that a warp takes together then have (nearly) one length, and a tile's
// rows stay close in memory.  Tiles of 256, 1024 and 4096 users: 2729, 2682 and
// 2672 us per clock on 10M x 1M, K = 64, and the same within 1% on 480k x 18k.
constexpr int kTileBits = 12;
// Cost of an item in a warp's share: its entries plus kItemCost.
constexpr int32_t kItemCost = 5;
// Replica accumulators: an item gets one delta row per kItemRep entries
// (largest minibatch count, rounded up to a power of two); a heavy user one
// per kUserRep chunks.  Replicas spread the fp32 reductions of popular rows
// over many L2 addresses and keep each partial sum short.
#ifndef ESSPT_ITEM_REP
#define ESSPT_ITEM_REP 2048
#endif
constexpr int32_t kItemRep = ESSPT_ITEM_REP;
constexpr int32_t kUserRep = 64;
#ifndef ESSPT_MAX_REP
#define ESSPT_MAX_REP 64
#endif
constexpr int32_t kMaxRep = ESSPT_MAX_REP;

// Rows of 36..64 values: the kHot items with the most entries of each minibatch
// have their updates summed per row group in shared memory and added to the
// replica rows once per warp instead of once per entry.
constexpr int kHot = 2;
inline bool uses_hot(int32_t K) { return K > 32 && K <= 64; }

// Row stride (in float4) of the item delta replicas: K rounded up to a whole
// number of 128-byte lines where that adds at most a third, so that eight
// lanes' 128 bytes of a reduction are one request, else to 32-byte sectors, so
// that they touch the fewest.
inline int32_t dR_stride4(int32_t K) {
  const int32_t lines = (K + 31) / 32 * 8;
  return 3 * lines <= K ? lines : (K + 7) / 8 * 2;
}

struct ScheduleArgs {
  int32_t* v;              // [P] read versions (in: v(c-1), out: v(c))
  int32_t* vslot;          // [P] out: ring slot v mod nslots of each read version
  uint32_t* status;        // latched error bits
  const uint32_t* thr;     // [dmax+1] ESSP delay thresholds, thr[k] = floor((1-p)^k 2^32)
  const uint32_t* vap_norm;  // [s+1] VAP: see launch_vap
  double vap_bound;        // VAP: v0 / sqrt(c)
  int32_t P, c, s, nslots, model, phased, dmax;
  uint64_t seed;
};

// One clock of MF-SGD over the users of minibatch b.
struct SgdArgs {
  float* ring;              // (s+2) * n_rows * K
  int64_t n_rows;
  int32_t K;
  int32_t n_users;
  int32_t nslots;           // s + 2
  int32_t slot_base;        // slot merged from (c-1, or c if INCs already landed there)
  int32_t slot_out;         // slot of version c
  const int32_t* vslot;     // [P] ring slots of the read versions
  const int32_t* uoff;      // [n_users+1] entry offsets of minibatch b (relative)
  float* dR;                // item delta replicas (all zero between clocks)
  int32_t dR_ld;            // float4 per dR row (dR_stride4)
  const int32_t* item_rep;  // see MergeArgs; hot_item: [kHot] hot items of minibatch b, -1 if unused
  const int32_t* hot_item;
  float eta, lambda;
  int32_t cap;
  double* sq_loss;          // optional
  int32_t row_mode;         // row-granular SSP: per-user slots, and offsets of item rows in the whole ring
  const int32_t* user_slot; // [n_users] row mode: ring slot of each user's cached row
  // chg[u] = last clock that changed user row u (written with every user row
  // that changes); an idle row whose slot already holds its current value is
  // not copied forward: clock > copy_all_until and clock - chg[u] >= nslots
  // (unchanged over the whole ring).  chg_item likewise for item rows.
  int32_t* chg;
  int32_t clock, copy_all_until;
};

// The work list of minibatch b: x = user, y = first entry, z = replica row in
// dL of a heavy user's chunk, or -1 for a user with 1..kHeavy entries (its row
// of version c is written directly), w = entries << 16 | worker; sorted by
// length within tiles of 2^kTileBits users.
// Warp w takes items part[w].x .. part[w].y in rounds of gpw (one per row
// group), per_step entries of an item per step, and its steps are part[w].z ..
// part[w].w (unsigned) of the minibatch's stream.  A step has gpw * per_step places, those
// of one group side by side.  Place p holds an entry: x[p] = item * K/4, and in
// yz, per_step y words before per_step z words, y = replica row * dR_stride4
// (both float4 offsets: of the item's row, and of the row in dR that its update
// adds into), or 1 + 2 * hot slot, and z = the value (fp32).  Empty places hold
// kNoRecord.
constexpr uint32_t kNoRecord = 0xffffffffu;
constexpr int kStepAlign = 4;  // a warp's first step is a multiple
struct StreamGeometry {
  int gpw, per_step;
};
// A minibatch of nearly 2^31 entries of users with one each has 2^32 places at two
// entries per step, and steps past 2^31 at one place per step: an item's place
// word is step * gpw + group, and steps and replica offsets are unsigned.
__host__ __device__ inline uint32_t place_word(const StreamGeometry& g, int64_t step, int grp) {
  return (uint32_t)(step * g.gpw + grp);
}
// Place of entry k of an item with place word `at`, and where its y word is (the
// z word follows per_step words later).
__host__ __device__ inline int64_t record_place(const StreamGeometry& g, uint32_t at, int32_t k) {
  return ((int64_t)at + (int64_t)(k / g.per_step) * g.gpw) * g.per_step + k % g.per_step;
}
__host__ __device__ inline int64_t y_word(const StreamGeometry& g, int64_t place) {
  return place / g.per_step * g.per_step * 2 + place % g.per_step;
}
// The most steps of a minibatch: the SGD kernel looks a few past the last.
constexpr int64_t kMaxSteps = (int64_t)UINT32_MAX - 64;
struct StreamArgs {
  SgdArgs a;
  const int4* items;
  const int4* part;
  int64_t n_warps;
  const uint32_t *x, *yz;   // x: in row mode (float4 offset in the ring of the cached version)
  float* dL;                // heavy-user delta replicas (all zero between clocks)
};

// The Clock() merge of the item rows, R^c_j = R^base_j + eta s_j sum of
// replicas, and of the heavy users' rows.
struct MergeArgs {
  float* ring;
  int64_t n_rows;
  int32_t K, n_users, n_items, nslots, slot_base, slot_out;
  const int32_t* item_rep;  // [M+1] prefix of extra replicas: replica 0 of item j is row j of dR,
                            // replica r > 0 row M + item_rep[j] + r - 1
  float* dR;
  int32_t dR_ld;
  const int32_t* item_cnt;  // [M] entries per item in minibatch b
  // Rows with several replicas: x = item or user (and its first replica row),
  // y = second replica row, z = replicas; of a heavy user w = entries.
  const int4 *popular, *heavy;
  int64_t n_popular, n_heavy;
  float* dL;
  float eta;
  int32_t cap;
  int32_t *chg, *chg_item;  // see SgdArgs
  int32_t clock, copy_all_until;
  int32_t do_schedule;      // also compute the next clock's read versions
  int32_t chained;          // start beside the kernel before it
  ScheduleArgs sched;
};

// Blocks for work_items at per_block each, at most max_per_sm per SM, at least one.
int grid_for(int64_t work_items, int64_t per_block, int max_per_sm);

// Launchers (return the launch error, if any).
cudaError_t launch_schedule(const ScheduleArgs& a, cudaStream_t st);
// VAP: norm[k], k = 1..kmax, is within the bound (as fp32 bits) exactly where
// max |X[c-1] - X[c-1-k]| over the table is, down to the stalest such k: the
// norm itself, or 0 / +inf (norm and words, s+1 each, must be zero on entry; a
// NaN difference counts as +inf).
cudaError_t launch_vap(const float* ring, int64_t slot_floats, int32_t nslots, int32_t c, int32_t kmax,
                            double bound, uint32_t* norm, uint32_t* words, cudaStream_t st);
cudaError_t launch_copy_rows(float* dst, const float* src, int64_t n_floats, cudaStream_t st);
// GET; with rowver non-null (row-granular SSP at clock c) each row is read at
// the worker's cached version, refreshed to c-1 first where it is missing or
// older than c-1-s, and *vmin (if non-null) receives the oldest version read.
cudaError_t launch_get(const float* ring, int64_t n_rows, int32_t K, int32_t nslots, const int32_t* v,
                       int32_t worker, const int32_t* ids, int64_t n, float* out, uint32_t* status,
                       int32_t* rowver, int32_t c, int32_t s, int32_t* vmin, cudaStream_t st);
cudaError_t launch_inc(float* slot, int64_t n_rows, int32_t K, const int32_t* ids, const float* d, int64_t n,
                       uint32_t* status, cudaStream_t st);
// The SGD kernel of one clock; the warps it can use at row width K on this
// device, and the shape of its stream.
cudaError_t launch_sgd_stream(const StreamArgs& a, cudaStream_t st);
int64_t stream_max_warps(int32_t K);
// Whether a clock of n_warps warps and n_users users is one block per SM at most.
bool stream_is_small(int32_t K, int64_t n_warps, int64_t n_users);
StreamGeometry stream_geometry(int32_t K);
// Build of the streams of all minibatches (setup), in four launches: the split of
// each one's work items over its warps, the steps of the warps, the records and
// their places (place[i] = item i's place word).  Nothing is written where status
// holds an error or a stream passes its limits, which the caller checks.
struct StreamBuild {
  const int4* items;
  const int64_t *item_base, *entry_base;  // [F+1] first item and entry of each minibatch
  const int64_t* pre;                     // see LayoutBuild
  const uint32_t* status;
  int32_t F;
  int64_t max_items, max_warps;           // of one minibatch at most
  StreamGeometry g;
  const int32_t* rec_j;
  const float* rec_D;
  const int32_t* item_rep;
  const int32_t* hot_item;                // [F][kHot] or null
  int64_t n_items;
  int32_t K, dR_ld;
  int64_t max_places;
  int4* part;
  int64_t *part_base, *place_base, *steps;  // out: [F+1], [F+1] first warp and place, [F] steps
  uint32_t *x, *yz, *place;
};
cudaError_t launch_stream_build(const StreamBuild& b, cudaStream_t st);
// New values for the places of a minibatch.
cudaError_t launch_stream_refill(const int4* items, const uint32_t* place, int64_t n_items, const StreamGeometry& g,
                                 const float* D, uint32_t* yz, cudaStream_t st);
// Row-granular SSP, before the SGD kernels of clock c: refresh the cached
// version of every row a worker reads (rowver[p * n_rows + r], -1 = never
// read) to c-1 where it is missing or older than c-1-s, and write the ring
// slot of each user's row and the place in the ring of each entry's item row.
struct RowRefreshArgs {
  int32_t* rowver;
  const int4* items;       // work list of minibatch b and its places (see StreamArgs)
  const uint32_t* place;
  int64_t n_items;
  StreamGeometry g;
  const int32_t* rec_j;    // item of each entry of minibatch b
  int64_t n_rows;
  int32_t K4, n_users, c, s, nslots;
  int32_t* user_slot;      // out [n_users], for the users of the work list
  uint32_t* x;             // out: the x words of the stream
};
cudaError_t launch_row_refresh(const RowRefreshArgs& a, cudaStream_t st);

// Sequential (read-my-writes) SGD of one clock over minibatch b: the users
// kernel writes every user row of version c, the item merge every item row.
struct SeqArgs {
  SgdArgs a;                // ring, slots, offsets, step sizes (no vslot, dR or work list)
  int32_t P, n_items;
  const int32_t* v;         // [P] read versions
  const int32_t* wuser;     // [n_users] users by worker, ascending within a worker
  const int32_t* wbase;     // [P+1] first of each worker's users
  const int32_t* rec_j;     // item of each entry of minibatch b
  const float* rec_D;
  const int32_t* item_cnt;  // [n_items] entries per item in minibatch b (hot-row cap)
  int32_t* chg_item;        // see SgdArgs
  float* mine;              // [P][n_items][K] each worker's item changes this clock (zero on entry)
};
cudaError_t launch_seq_clock(const SeqArgs& a, cudaStream_t st);
cudaError_t launch_clock_merge(const MergeArgs& a, cudaStream_t st);
// Objective at one table version over the work lists of all F minibatches:
// item_base and entry_base (device, [F+1]) hold each one's first item and entry.
// out[0] = sum e^2 and out[out_stride] = penalised sum; by worker (P at most,
// sums added to what out holds) at out[p] and out[out_stride + p].
struct ObjectiveArgs {
  const float* slot;
  int64_t n_users;
  int32_t K, F, P;
  const int4* items;
  int64_t n_items;
  const int64_t *item_base, *entry_base;
  const int32_t* rec_j;
  const float* rec_D;
  float lambda;
  double* out;
  int64_t out_stride;
  int64_t n_obs;        // entries, and those of the longest item
  int32_t longest;
  int32_t part, parts;  // (set by the launch) entries of a part, and parts of an item
};
cudaError_t launch_objective(const ObjectiveArgs& a, cudaStream_t st);
cudaError_t launch_worker_objective(const ObjectiveArgs& a, cudaStream_t st);

// MF layout build (setup, not per clock).
struct LayoutBuild {
  const int32_t* i;
  const int32_t* j;
  const float* D;
  const uint8_t* mb;
  const int32_t* worker;
  int64_t n_obs, n_users, n_items;
  int32_t F, P;
  // outputs (persistent)
  int32_t* rec_u;
  int32_t* rec_j;
  float* rec_D;
  int32_t* hot_item;    // [F][kHot] hot items of each minibatch, or null
  int32_t* uoff;        // [F][n_users+1]
  int64_t* mb_base;     // [F+1]
  int32_t* item_cnt;    // [F][n_items]
  int32_t* item_rep;    // [n_items+1]
  int4* popular;        // [max_popular] items with extra replicas (see MergeArgs), in no order
  uint32_t* n_popular;  // their number (0 on entry)
  uint32_t* longest;    // entries of the longest work item (0 on entry)
  int4* chunk;          // [max_chunks] work items (see StreamArgs); before that 3 words per item of the build's
  int64_t* chunk_base;  // [F+1]
  int4* heavy;          // [max_heavy]
  int64_t* heavy_base;  // [F+1]
  int32_t* wuser;       // [n_users] users by worker, ascending within a worker
  int32_t* wbase;       // [P+1] first of each worker's users
  int64_t max_chunks, max_heavy;
  // scratch, and the stream's memory, which is free until the stream is filled
  void* scratch;
  size_t scratch_bytes;
  void* stream_mem;     // layout_stage_bytes
  int64_t n_work;       // out: work items
  const int64_t* pre;   // out, in stream_mem: [items+1] summed cost of the items before each
  uint32_t* status;
};

size_t layout_scratch_bytes(int64_t n_obs, int64_t n_users, int64_t n_items, int32_t F);
size_t layout_stage_bytes(int64_t n_obs, int64_t n_users, int32_t F);
size_t layout_chunk_bytes(int64_t n_obs, int64_t n_users, int32_t F);
int64_t layout_max_chunks(int64_t n_obs, int32_t F, int64_t n_users);
int64_t layout_max_heavy(int64_t n_obs, int32_t F);
int64_t layout_max_popular(int64_t n_obs);
int64_t layout_max_item_reps(int64_t n_obs, int64_t n_items);
int64_t layout_max_user_reps(int64_t n_obs);
cudaError_t build_layout(LayoutBuild& b, cudaStream_t st);
// Places that the streams of all minibatches can take, empty ones included.
int64_t layout_max_places(int64_t n_obs, int64_t n_users, int32_t F, const StreamGeometry& g, int64_t max_warps);
cudaError_t launch_validate(const LayoutBuild& b, cudaStream_t st);
// Staged minibatch check: su/sj (n entries) and suoff (n_off offsets) against
// the resident ru/rj/ruoff; a difference latches kErrInput.
cudaError_t launch_stage_check(const int32_t* su, const int32_t* sj, const int32_t* suoff, const int32_t* ru,
                               const int32_t* rj, const int32_t* ruoff, int64_t n, int64_t n_off, uint32_t* status,
                               cudaStream_t st);

// The objective's inputs for a context's loaded entries and table version
// `version` (checked against the live window), all but out and lambda, for
// entry points defined in other translation units; and the context's error
// setter.
esspt_status mf_view(esspt_ctx* ctx, int32_t version, ObjectiveArgs* a, cudaStream_t* st);
esspt_status mf_fail(esspt_ctx* ctx, esspt_status code, const char* msg);

}  // namespace esspt
