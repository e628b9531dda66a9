// Internal declarations of the GB300 parameter manager (not part of the ABI).
//
// Device data layout (all in HBM, owned by the context):
//   main        [K][D] fp32     main copy of every parameter
//   val, acc    [S][D] fp32     replica pool: local value and pending updates
//                               (rows are written only when needed, see the replica states)
//   map         [W][K] int32    worker w's replica of key k: -1 if none, else its
//                               slot, with bit 31 set when slot_owner may hold
//                               a state other than REP_ALIAS (see map_touched)
//   rc          [W][K] uint32   number of w's active intents containing k
//   holders     [K]    uint32   bit w set iff worker w holds a replica of k
//   slot_owner  [S]    uint64   key, worker and state of a live slot (see
//                               owner_word), kEmptySlot if free
//   free_stack  [S]    int32    free slots, top at free_stack[free_top - 1]
//   stamp       [K]    uint32   tag of the last Intent call that listed k
//   dirty       [K]    uint8    versioned refresh only: main[k] written other
//                               than by a sync merge since the last sync of k
//   own         [K]    uint16   relocation mode only: ((owner + 1) << 8) |
//                               number of workers with active intent; owner
//                               -1 is the key's home (no worker held it yet)
//   DevState                    counters and the sticky error bits
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct adapm_ctx;

namespace adapm {

constexpr uint32_t kNoKey = 0xFFFFFFFFu;          // sentinel: skipped element
constexpr uint64_t kEmptySlot = ~0ull;
constexpr int kMaxWorkers = 32;
constexpr int kNumSms = 152;                      // GB300; refreshed at create

enum ErrBits : uint32_t {
  ERR_KEY_RANGE = 1u,   // a key >= K was passed
  ERR_NO_SLOTS = 2u,    // replica capacity exhausted
  ERR_REFCOUNT = 4u,    // refcount over/underflow
  ERR_TIMEOUT = 8u,     // a bounded wait on another block gave up
  ERR_INTERNAL = 16u,   // an index read from the library's own scratch or lists was out of
                        // range: the element was skipped instead of accessed
};

struct DevState {
  int32_t free_top;       // free slots on the stack
  int32_t high_water;     // slots [0, high_water) have been used
  uint32_t n_create;      // keys appended to the create list of this advance (0 between advances)
  uint32_t n_evict;       // slots appended to the evict list of this advance (0 between advances)
  int32_t adv_top;        // free_top before this advance's slots moved
  uint32_t adv_nc;        // creations of this advance (0 if the slots ran out)
  uint32_t errors;        // ErrBits, sticky until read by adapm_wait
  uint32_t last_unique;   // distinct keys of the last push
  uint32_t plan_miss;     // sequence number of the last push whose plan did not match its keys
  uint32_t adv_ne;        // evictions of this advance
  unsigned long long created;
  unsigned long long destroyed;
  int32_t live;
  int32_t live_keys;      // keys with at least one replica
  int32_t sole_keys;      // keys with exactly one replica
  uint32_t par;           // parity of the syncs so far (see the replica states)
  uint32_t sync_done;     // blocks of a sync that finished (0 between syncs)
  uint32_t ev_done;       // blocks of the closing events launch that finished (0 between advances)
  uint32_t loss_done;     // blocks of a training step that finished (0 between steps)
  unsigned long long push_rows;       // rows pushed (cumulative)
  unsigned long long push_unique;     // distinct keys over all pushes (cumulative)
  unsigned long long sync_keys;       // keys merged by sync (cumulative)
  unsigned long long sync_replicas;   // replicas refreshed by sync (cumulative)
  unsigned long long relocations;     // owner changes (relocation mode, cumulative)
  unsigned long long sync_refreshed;  // replica values written by sync (cumulative)
  unsigned long long plan_misses;     // pushes whose plan did not match their keys (cumulative)
  // grid barriers of the sort: blocks arrived, over the context's lifetime
  // (a line of its own, away from the counters above)
  alignas(128) unsigned long long bar_arrivals;
};

// Counters of one worker's early advance events (computed ahead of the
// advance, on a stream of their own): list lengths, and the blocks of the
// evict_create launch that have finished.  Zero between advances.
struct AdvCounts {
  uint32_t nc;     // keys on the create list
  uint32_t ne;     // slots on the evict list
  uint32_t done;   // evict_create blocks finished
  uint32_t pad;
};

// Plain view of the device state passed to kernels by value.
struct Store {
  float* main;
  float* val;
  float* acc;
  int32_t* map;
  uint32_t* rc;
  uint32_t* holders;
  unsigned long long* slot_owner;
  int32_t* free_stack;
  uint32_t* stamp;
  uint16_t* own;    // null unless relocation mode
  uint8_t* dirty;   // null unless versioned refresh
  DevState* st;
  uint64_t K;
  uint64_t S;
  uint32_t D;
  uint32_t W;
  uint32_t par;     // kernels that look at replica states: their copy of st->par
};

// ---- replica states ---------------------------------------------------------
// A replica's value equals its main row until somebody writes either, so its
// rows are not copied when it is created or refreshed; they are written when
// the two first differ.  Its state is three flags:
//   REP_PENDING  acc holds pending updates (else none are pending, acc unset)
//   REP_OWNVAL   the value's base is val (else main[k], val unset)
//   REP_FOLDED   val includes acc (only with both of the above)
// value = base, plus acc when updates are pending and not folded.  0 is an
// alias of the main row.  The first push to a replica after its creation or
// a sync stores its sum in acc and leaves the base alone, later ones fold
// acc into val; whoever writes main[k] while other workers' replicas have it
// as their base (an evicted replica's pending updates, a push of a worker
// without a replica) first copies the old row to their val.  A sync merges
// the pending rows and leaves every replica an alias again.  The values are
// those of replicas that are copied at creation and written by every push
// (the same sums in the same order) with a third of the row traffic: a
// replica that is created, pushed to once, synced and evicted moves 4 rows
// instead of 15, one whose key other workers evict meanwhile 6.
//
// The state lives in slot_owner beside the parity of the syncs made when it
// was written.  The last block of a sync flips the parity, which makes every
// state an alias at once without a write that other blocks of the sync could
// see half done; the states it voids are cleared by the next sync's scan.
// Bit 31 of a map entry says that slot_owner has to be read: an entry without
// it is an alias.
//
// With relocation (s.own set) the main copy of a replicated key is written by
// its owner on every push, so every alias would be detached at once, by the
// push: there replicas are copied at creation, refreshed by every sync and
// always in the state REP_COPIED, which is not stored.  (Measured with
// aliases there: 8 x 2^18 Zipf(1.1) keys of 64 floats, push 461 -> 566 us per
// clock, the clock 1261 -> 1382 us.)
constexpr uint32_t REP_ALIAS = 0u;
constexpr uint32_t REP_PENDING = 1u;
constexpr uint32_t REP_OWNVAL = 2u;
constexpr uint32_t REP_FOLDED = 4u;
constexpr uint32_t REP_COPIED = REP_PENDING | REP_OWNVAL | REP_FOLDED;
__host__ __device__ __forceinline__ bool rep_adds(uint32_t state) {   // acc is added to the base
  return (state & (REP_PENDING | REP_FOLDED)) == REP_PENDING;
}

__host__ __device__ __forceinline__ bool map_none(int32_t e) { return e == -1; }
__host__ __device__ __forceinline__ bool map_touched(int32_t e) { return e < -1; }   // bit 31, not "none"
__host__ __device__ __forceinline__ int32_t map_slot(int32_t e) { return e & 0x7FFFFFFF; }
__host__ __device__ __forceinline__ int32_t map_touch(int32_t slot) { return (int32_t)((uint32_t)slot | 0x80000000u); }

// High word of slot_owner: worker (bits 0-7), state (8-10), parity (11); the
// low word is the key.
__device__ __forceinline__ uint32_t owner_hi(uint32_t w, uint32_t state, uint32_t par) {
  return w | (state << 8) | (par << 11);
}
__device__ __forceinline__ unsigned long long owner_word(uint32_t w, uint32_t k, uint32_t state, uint32_t par) {
  return ((unsigned long long)owner_hi(w, state, par) << 32) | k;
}
__device__ __forceinline__ uint32_t owner_worker(unsigned long long ow) { return (uint32_t)(ow >> 32) & 0xFFu; }
__device__ __forceinline__ uint32_t owner_raw_state(unsigned long long ow) { return (uint32_t)(ow >> 40) & 7u; }
__device__ __forceinline__ uint32_t owner_par(unsigned long long ow) { return (uint32_t)(ow >> 43) & 1u; }
__device__ __forceinline__ uint32_t owner_state(unsigned long long ow, uint32_t par) {
  return owner_par(ow) == par ? owner_raw_state(ow) : REP_ALIAS;
}
__device__ __forceinline__ void set_owner_hi(const Store& s, int32_t slot, uint32_t hi) {
  reinterpret_cast<uint32_t*>(s.slot_owner + slot)[1] = hi;
}
// Whether a map entry is one whose value is not (just) the main row.
__device__ __forceinline__ bool rep_differs(const Store& s, int32_t e) {
  return s.own != nullptr ? !map_none(e) : map_touched(e);
}
// State of the replica behind a map entry that is not -1.
__device__ __forceinline__ uint32_t rep_state(const Store& s, int32_t e) {
  if (s.own != nullptr) return REP_COPIED;
  return map_touched(e) ? owner_state(s.slot_owner[map_slot(e)], s.par) : REP_ALIAS;
}
// The row that holds worker's value of key k under map entry e (main, or the
// replica's own value), and whether the replica's pending row has to be added
// to it (*add: that row, else null).
__device__ __forceinline__ const float4* row_source(const Store& s, int32_t e, uint32_t k, const float4** add) {
  const uint32_t D4 = s.D >> 2;
  const float4* p = reinterpret_cast<const float4*>(s.main) + (uint64_t)k * D4;
  *add = nullptr;
  if (s.own != nullptr) return map_none(e) ? p : reinterpret_cast<const float4*>(s.val) + (uint64_t)e * D4;
  if (map_touched(e)) {
    const uint64_t off = (uint64_t)map_slot(e) * D4;
    const uint32_t state = rep_state(s, e);
    if (state & REP_OWNVAL) p = reinterpret_cast<const float4*>(s.val) + off;
    if (rep_adds(state)) *add = reinterpret_cast<const float4*>(s.acc) + off;
  }
  return p;
}
// Before main[k] changes: worker b's replica of k, if it has the main row as
// its base, becomes one with a value of its own.  Returns the slot whose val
// row the caller then copies the old main row to, -1 if there is none.
__device__ __forceinline__ int32_t take_alias(const Store& s, uint32_t b, uint32_t k) {
  int32_t* me = s.map + (uint64_t)b * s.K + k;
  const int32_t e = *me;
  if (map_none(e)) return -1;
  const uint32_t state = rep_state(s, e);
  if (state & REP_OWNVAL) return -1;
  const int32_t sl = map_slot(e);
  set_owner_hi(s, sl, owner_hi(b, state | REP_OWNVAL, s.par));
  if (!map_touched(e)) *me = map_touch(sl);
  return sl;
}

// Fields of own[k] (relocation mode).
__device__ __forceinline__ uint32_t own_count(uint32_t o) { return o & 0xFFu; }
__device__ __forceinline__ int own_owner(uint32_t o) { return (int)(o >> 8) - 1; }
__device__ __forceinline__ uint16_t own_pack(int owner, uint32_t count) {
  return (uint16_t)(((uint32_t)(owner + 1) << 8) | count);
}

__device__ __forceinline__ void set_error(DevState* st, uint32_t bits) {
  atomicOr(&st->errors, bits);
}

// True once a sort has given up (ERR_TIMEOUT): its output is incomplete and
// the kernels that consume sorted keys return without touching the store.
__device__ __forceinline__ bool sort_failed(const DevState* st) {
  return (*reinterpret_cast<const volatile uint32_t*>(&st->errors) & ERR_TIMEOUT) != 0u;
}

// ---- radix sort / compaction (sort.cu) --------------------------------------
// Stable sort of n uint32 keys by their low `bits` bits in one cooperative
// launch on `stream`.  `raw` (n keys, not modified) is the first pass's
// input; a key >= K is sorted as kNoKey (after every valid key) and sets
// ERR_KEY_RANGE unless allow_nokey and it equals kNoKey.  ka/kb are
// ping-pong space of n keys; with va/vb non-null the positions 0..n-1
// travel with the keys.  The sorted keys (and positions) end in the buffers
// returned through *keys_out / *pos_out.  `scratch` holds
// sort_scratch_words(n, bits, sms) uint32 words.  *bar_base is the host's copy of
// st->bar_arrivals, advanced by the launch.  clear0 / clear1 (may be null)
// are device words the launch sets to zero before any later kernel on the
// stream runs (counters of the consumer).  If a grid-barrier wait gives
// up, the kernel sets ERR_TIMEOUT and returns; every kernel that consumes a
// sort checks that bit first and does nothing while it is set.
//
// Plans (cooperative launch only): with plan_keys and plan_word, the blocks
// first compare raw with plan_keys, the keys a plan was sorted from,
// position by position (out-of-range keys all counting as the sentinel); a
// mismatch stores plan_seq in *plan_word and counts a plan miss.  After one
// more grid barrier the launch sorts only if *plan_word == plan_seq;
// otherwise its blocks account their remaining barriers and return, leaving
// ka/kb/va/vb as they are (the plan holds the result).  Out-of-range keys
// are reported by the check as the sort would.
// `by`: SORT_BY_SIZE sorts few keys in one block (below) and others in the
// cooperative launch, SORT_BY_BARRIERS all in the latter; SORT_BY_LAUNCHES
// runs the sort as ordinary launches (kernel boundaries instead of grid
// barriers, *bar_base untouched): for a stream that runs beside other work,
// where a cooperative launch would wait for the whole GPU, and for a graph.  One for the
// count and two per pass, or one per pass when the blocks are few enough that
// each scans the digit table itself.
enum SortBy { SORT_BY_SIZE, SORT_BY_BARRIERS, SORT_BY_LAUNCHES };
size_t sort_scratch_words(uint64_t n, int bits, int sms);
int sort_passes(int bits);
cudaError_t sort_keys(const uint32_t* raw, uint64_t n, uint64_t K, bool allow_nokey, int bits,
                      uint32_t* ka, uint32_t* kb, uint32_t* va, uint32_t* vb, uint32_t* scratch, int sms,
                      DevState* st, unsigned long long* bar_base, uint32_t* clear0, uint32_t* clear1,
                      cudaStream_t stream, uint32_t** keys_out, uint32_t** pos_out,
                      const uint32_t* plan_keys = nullptr, uint32_t* plan_word = nullptr, uint32_t plan_seq = 0,
                      SortBy by = SORT_BY_SIZE);

// Up to kSmallSort keys are sorted by one block in one ordinary launch
// (sort_small.cu; sort_keys calls it for a push).  keys_out / pos_out: the
// sorted keys and their positions (both or neither); copy_out: the keys as
// given; heads_out / heads_count: the distinct valid ones, ascending, and
// their number; plan_*, clear*, allow_nokey as for sort_keys.  Pointers that
// are null are not written.  The limits: a push of 8000 keys that sorts takes
// 53 us so and 57 us with the grid sort, of 16,384 keys 50 us more; one that
// only checks a plan is done sooner by a block per SM above kSmallPlan keys.
constexpr uint64_t kSmallSort = 8192, kSmallPlan = 4096;
struct SmallSort {
  const uint32_t* raw;
  uint32_t n;
  uint64_t K;
  bool allow_nokey;
  uint32_t* keys_out;
  uint32_t* pos_out;
  uint32_t* copy_out;
  uint32_t* heads_out;
  uint32_t* heads_count;
  DevState* st;
  uint32_t* clear0;
  uint32_t* clear1;
  const uint32_t* plan_keys;
  uint32_t* plan_word;
  uint32_t plan_seq;
};
cudaError_t sort_small(const SmallSort& a, int bits, cudaStream_t stream);

// The distinct valid keys of a sorted array, in no particular order, into out;
// their number is added to *count.
void list_sorted_heads(const uint32_t* sk, uint64_t n, uint32_t* out, uint32_t* count, cudaStream_t stream);

// Stream compaction (a count / scan / write pass), tmp of compact_tmp_words(n).
size_t compact_tmp_words(uint64_t n);

// Keys k < K with a replica (map_w[k] != -1), ascending, into out; count to *count.
void compact_replica_keys(const int32_t* map_w, uint64_t K, uint32_t* out, uint32_t* count,
                          uint32_t* tmp, cudaStream_t stream);

int bits_for(uint64_t num_keys);   // bits covering [0, K] (K itself is the sentinel range)

// Process-wide count of kernels launched by the library (capi.cu).
void note_launches(uint64_t n);

// What an entry point outside capi.cu needs of a context (capi.cu).
struct CtxView {
  Store s;
  DevState* dstate;
  cudaStream_t stream;
  int device;
  int sms;
  int bits;
  bool broken;
  unsigned long long* bar_base;   // the context's copy of dstate->bar_arrivals
};
bool ctx_view(struct ::adapm_ctx* ctx, CtxView* out);
void ctx_set_error(struct ::adapm_ctx* ctx, const char* msg);
void ctx_add_push_rows(struct ::adapm_ctx* ctx, uint64_t n);
// The checks every entry point starts with: a live context (ADAPM_EINVAL for
// null, ADAPM_ECUDA once it is unusable), its last error cleared, its device
// current.  Returns an adapm_status value (0 = ADAPM_OK).
int ctx_begin(struct ::adapm_ctx* ctx);
// How a push of n keys sorts: in ordinary launches while its stream records a
// graph (the grid barriers' arrival count is the host's, per launch) and the
// keys are too many for one block; with the grid barriers, whose first one
// will wait in vain, after adapm_debug_fail_next_barrier (taken once).
SortBy ctx_sort_by(struct ::adapm_ctx* ctx, uint64_t n);
// A CUDA runtime error: records "where: message", marks the context unusable
// (as every entry point does) and returns ADAPM_ECUDA.
int ctx_fail_cuda(struct ::adapm_ctx* ctx, cudaError_t e, const char* where);
// cudaGetLastError() after a call's launches, or the launch failure that
// adapm_debug_fail_next_launch asked for (taken once).
cudaError_t ctx_launch_error(struct ::adapm_ctx* ctx);
// Per-operation timing (adapm_profile_enable): events recorded around an
// operation's work on the context's stream; a no-op while profiling is off.
struct ProfToken {
  int op = -1;
  cudaEvent_t a = nullptr, b = nullptr;
};
ProfToken ctx_prof_start(struct ::adapm_ctx* ctx, int op);
void ctx_prof_stop(struct ::adapm_ctx* ctx, ProfToken& t);

// ---- launches that overlap the end of the kernel before them ----------------
// The kernels of a call, and of one call after another, follow each other on
// one stream, and a kernel of a few thousand rows is not much longer than the
// gap in front of it.  launch_after starts a kernel while the one before it
// drains: its blocks are placed as soon as that kernel's blocks have all left
// (no kernel here lets go earlier, so nothing it keeps in caches is read
// before it is final), and its first statement, after_previous(), waits until
// the other's writes are visible.  Every block makes that wait, so a kernel
// ends after all before it on the stream have, and a kernel or event that
// follows sees them too.  Such a kernel runs from before the other's last
// writes, so it reads with plain loads alone: __ldg and const __restrict__
// parameters promise data that does not change while the kernel runs, and need
// not stay behind the wait.  (Plain loads in their place: between 0.998 and
// 1.02 times as fast over the timed cases.)
// A kernel that a stream runs right after a wait for
// another stream has nothing to overlap and is launched plainly (the
// attribute costs the host more than it gives: follows = false).
//
// Measured, per pass: 1000 keys pulled and pushed 30 -> 21 us, a clock of 8 x
// 16,384 keys 463 -> 400 us, of 8 x 131,072 with windows of four clocks 989 ->
// 945 us, 8 x 65,536 factorisation cells 1190 -> 1129 us, 8 x 2^20 keys 2918 ->
// 2873 us.
template <class... P, class... A>
inline void launch_on(bool follows, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem,
                      cudaStream_t stream, const A&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = stream;
  c.attrs = &at;
  c.numAttrs = follows ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
inline void launch_after(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                         const A&... args) {
  launch_on(true, kernel, grid, block, smem, stream, args...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

}  // namespace adapm
