// Kernels of the parameter manager's hot path that read and write rows
// through the slot maps: pull, sync and the inspection gathers.  The push is
// in push.cu, the intent and advance kernels in advance.cu.
//
//   pull        out[i] = replica of keys[i] at worker w, else main       (Sec. 5.1)
//   sync        main += sum of all holders' pending updates (ascending
//               worker); holders are aliases of main afterwards        (App. B.1.2)
#include "internal.cuh"
#include "rowgroup.cuh"
#include "store_launch.cuh"

namespace adapm {

namespace {

// ---------------------------------------------------------------------------
// pull (and main-only gather for inspection when w < 0)
// ---------------------------------------------------------------------------
// R rows per group and round, software-pipelined so that one round issues
// the row loads of round i, the slot lookups of round i+1 and the key loads
// of round i+2 together: one memory latency per round instead of three.
// With one float4 of a row per lane, four rows per group at five blocks per SM
// do better than eight at three (rows of 64 floats: 9 x 2^18 rows 430 -> 397
// us, 9 x 131,072 291 -> 250 us); wider rows want the bytes in flight (8 float4
// per lane; rows of 200 floats 538 us, with half of that 556 us).
constexpr int pull_rows(int C) { return C == 1 ? 4 : (8 / C > 0 ? 8 / C : 1); }

template <int G, int C, int R>
__global__ void __launch_bounds__(kThreads, C == 1 ? 5 : 1)
pull_kernel(Store s, int w, const uint32_t* keys, uint64_t n, float* __restrict__ out) {
  after_previous();
  const int lane = threadIdx.x & (G - 1);
  const uint64_t g = group_id<G>(), ng = group_count<G>();
  const uint32_t D4 = s.D >> 2;
  const float4* main4 = reinterpret_cast<const float4*>(s.main);
  const float4* val4 = reinterpret_cast<const float4*>(s.val);
  float4* out4 = reinterpret_cast<float4*>(out);
  const int32_t* mapw = w >= 0 ? s.map + (uint64_t)w * s.K : nullptr;
  s.par = s.st->par;
  const uint64_t step = ng * R;
  bool bad = false;
  auto load_keys = [&](uint64_t b, uint32_t (&k)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) k[r] = b + r < n ? keys[b + r] : kNoKey;
  };
  auto load_slots = [&](const uint32_t (&k)[R], int32_t (&sl)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) sl[r] = (mapw != nullptr && k[r] < s.K) ? mapw[k[r]] : -1;
  };
  uint64_t base = g * R;
  uint32_t k0[R], k1[R];
  int32_t sl0[R];
  load_keys(base, k0);
  load_keys(base + step, k1);
  load_slots(k0, sl0);
  for (; base < n; base += step) {
    // this round's rows: main, unless the replica has a value of its own (or
    // one pending push to add, which few have: added in a pass of its own)
    const float4* src[R];
    uint32_t sums = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      src[r] = nullptr;
      if (k0[r] < s.K) {
        src[r] = main4 + (uint64_t)k0[r] * D4;
        if (s.own != nullptr) {
          if (sl0[r] >= 0) src[r] = val4 + (uint64_t)sl0[r] * D4;
        } else if (map_touched(sl0[r])) {
          const uint32_t state = rep_state(s, sl0[r]);
          if (state & REP_OWNVAL) src[r] = val4 + (uint64_t)map_slot(sl0[r]) * D4;
          if (rep_adds(state)) sums |= 1u << r;
        }
      } else if (base + r < n) {
        bad = true;
      }
    }
    float4 v[R][C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = lane + c * G;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r][c] = (src[r] != nullptr && col < D4) ? src[r][col] : f4zero();
    }
    if (sums) {
      const float4* acc4 = reinterpret_cast<const float4*>(s.acc);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if ((sums >> r) & 1u)
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            if (col < D4) v[r][c] = f4add(v[r][c], acc4[(uint64_t)map_slot(sl0[r]) * D4 + col]);
          }
    }
    // next round's slots and the keys of the round after
    int32_t sl1[R];
    uint32_t k2[R];
    load_slots(k1, sl1);
    load_keys(base + 2 * step, k2);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = lane + c * G;
      if (col < D4)
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (base + r < n) __stcs(out4 + (base + r) * D4 + col, v[r][c]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      k0[r] = k1[r];
      sl0[r] = sl1[r];
      k1[r] = k2[r];
    }
  }
  if (bad && lane == 0) set_error(s.st, ERR_KEY_RANGE);
}

// ---------------------------------------------------------------------------
// sync
// ---------------------------------------------------------------------------
// Every replica is an alias of its main row afterwards (REP_ALIAS; with
// relocation, where they are copies, copied.cu), so only pending rows move:
// main[k] += acc for every holder with updates, in ascending worker order.  A warp scans the slots' owner words, up to 32 at a
// time, and lists those with updates; replicas nobody touched since the last
// sync cost their 8-byte word alone.  Once 32 are listed (or the scan ends)
// one lane per listed slot looks up the key's holders, which of them merges
// (the lowest with updates) and, for its key, one lane per holder where the
// pending rows are; rows move last, taken by the warp's row groups.  The
// chain of lookups is as long as a row transfer several times over, so it is
// paid per 32 listed slots, not per scanned word or per holder.  No word that
// decides who merges (states, map slots) is changed by the launch: its last
// block flips the parity, which voids every state.
//
// Measured, copies refreshed by row groups before -> now: 2.45M replicas of
// 64 floats pushed every clock 598 -> 198 us (their rows bound it: 1.6 GB),
// 2.0M of which a fifth are pending (the scan and the lookups) 516 -> 128 us,
// 3.2M of 512 floats, 8% pending, 4833 -> 356 us.
//
// VER: versioned refresh (App. B.1.2: a holder receives only updates it has
// not seen; s.dirty is set): a sole holder's own value (REP_OWNVAL) is left
// alone unless main[k] was written other than by a sync since the last sync
// of k (dirty[k]); keys with several holders are always refreshed.
constexpr uint32_t kSyncPairs = 128;          // (key, holder) pairs a warp looks up at a time
constexpr uint32_t kFold = 0x80000000u;       // Merge slot flag: val += acc too (VER: it keeps its own value)

struct SyncSmem {
  struct Item {
    uint32_t slot, key, hi;     // hi: high word of slot_owner
  };
  struct Merge {
    uint32_t slot, key;
  };
  Item list[kThreads / 32][64];
  Merge sole[kThreads / 32][32];
  uint2 pair[kThreads / 32][kSyncPairs];    // (key, holder), then (key, slot or -1)
};

template <int G, int C, bool VER>
__global__ void __launch_bounds__(kThreads, C >= 8 ? 2 : 4) sync_kernel(Store s) {
  after_previous();
  constexpr int R = 4 / C > 0 ? 4 / C : 1;
  constexpr uint32_t GW = 32 / G;   // row groups per warp
  __shared__ SyncSmem sm;
  const int lane32 = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int lane = threadIdx.x & (G - 1);
  const uint32_t gi = (uint32_t)lane32 / G;
  const unsigned before = (1u << lane32) - 1u;
  const uint32_t D4 = s.D >> 2;
  const uint64_t hw = (uint64_t)s.st->high_water;
  s.par = s.st->par;
  if (s.st->errors & ERR_TIMEOUT) return;   // a sort gave up (read with the words above, in one latency)
  float4* main4 = reinterpret_cast<float4*>(s.main);
  const float4* acc4 = reinterpret_cast<const float4*>(s.acc);
  const uint64_t warps = (uint64_t)gridDim.x * (kThreads / 32);
  const uint64_t warp = (uint64_t)blockIdx.x * (kThreads / 32) + wid;
  // slots per warp and round: all 32 lanes once there are enough to keep every warp busy
  const uint32_t per = hw >= warps * 32 ? 32u : (uint32_t)((hw + warps - 1) / warps);
  uint32_t nref = 0;   // VER: sole holders refreshed
  uint32_t have = 0;   // listed slots of this warp
  auto scan = [&](uint64_t b0) {
    const uint64_t b = b0 + lane32;
    return (uint32_t)lane32 < per && b < hw ? s.slot_owner[b] : kEmptySlot;
  };
  unsigned long long ow = scan(warp * per);
  for (uint64_t b0 = warp * per;; b0 += warps * per) {   // warp-uniform
    const bool more = b0 < hw;
    if (more) {
      const uint64_t b = b0 + lane32;
      const uint32_t k = (uint32_t)ow, hi = (uint32_t)(ow >> 32);
      uint32_t state = ow == kEmptySlot ? REP_ALIAS : owner_raw_state(ow);
      if (state != REP_ALIAS && owner_par(ow) != s.par) {   // voided by the sync before
        set_owner_hi(s, (int32_t)b, owner_hi(owner_worker(ow), REP_ALIAS, s.par));
        state = REP_ALIAS;
      }
      const bool take = VER ? state != REP_ALIAS : (state & REP_PENDING) != 0u;
      // touched, nothing pending: an alias again, no state to look up
      if (!VER && !take && state != REP_ALIAS) s.map[(uint64_t)owner_worker(ow) * s.K + k] = (int32_t)b;
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, take);
      if (take) sm.list[wid][have + __popc(bal & before)] = SyncSmem::Item{(uint32_t)b, k, hi};
      have += __popc(bal);
      ow = scan(b0 + warps * per);
      __syncwarp();
    }
    while (have >= 32u || (!more && have)) {
      const uint32_t cnt = have < 32u ? have : 32u;
      have -= cnt;
      const bool in = (uint32_t)lane32 < cnt;
      const SyncSmem::Item it = in ? sm.list[wid][have + lane32] : SyncSmem::Item{0u, 0u, 0u};
      const uint32_t k = it.key, w = it.hi & 0xFFu, state = (it.hi >> 8) & 7u;
      bool add = in && (state & REP_PENDING);   // rows to add: this slot's, or all of the key's if it merges
      bool own = false;                         // VER: the replica keeps its own value
      uint32_t mask = 0;                        // all holders when the key has several
      if (in) {
        mask = s.holders[k];
        if ((mask & ~(1u << w)) == 0u) {
          mask = 0;
          if (VER) {
            if (s.dirty[k]) {
              s.dirty[k] = 0;
              nref += 1;
            } else {
              own = state & REP_OWNVAL;
            }
          }
        } else {
          if (VER) s.dirty[k] = 0;
          // the lowest holder with pending updates merges all of them
          uint32_t lower = add ? mask & ((1u << w) - 1u) : 0u;
          while (lower) {
            constexpr int Q = 4;
            int32_t e[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              e[q] = -1;
              if (lower) {
                e[q] = s.map[(uint64_t)(__ffs(lower) - 1) * s.K + k];
                lower &= lower - 1;
              }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q)
              if (!map_none(e[q]) && (owner_state(s.slot_owner[map_slot(e[q])], s.par) & REP_PENDING)) add = false;
            if (!add) lower = 0;
          }
        }
        if (own) set_owner_hi(s, (int32_t)it.slot, owner_hi(w, REP_OWNVAL, s.par ^ 1u));
        else s.map[(uint64_t)w * s.K + k] = (int32_t)it.slot;   // an alias: no state to look up
      }
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, add && mask == 0u);
      const uint32_t nsole = __popc(bal);
      if (add && mask == 0u) {
        // (VER: a replica that keeps its own value folds the pending row into it)
        const bool fold = VER && own && rep_adds(state);
        sm.sole[wid][__popc(bal & before)] = SyncSmem::Merge{it.slot | (fold ? kFold : 0u), k};
      }
      __syncwarp();
      for (uint32_t j0 = gi * R; j0 < nsole; j0 += GW * R) {
        uint32_t key[R];
        float4 mv[R][C], av[R][C];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const bool v = j0 + r < nsole;
          const SyncSmem::Merge t = v ? sm.sole[wid][j0 + r] : SyncSmem::Merge{0u, 0u};
          key[r] = t.key;
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            mv[r][c] = v && col < D4 ? main4[(uint64_t)t.key * D4 + col] : f4zero();
            av[r][c] = v && col < D4 ? acc4[(uint64_t)(t.slot & ~kFold) * D4 + col] : f4zero();
          }
        }
        if (VER) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const uint32_t sl = j0 + r < nsole ? sm.sole[wid][j0 + r].slot : 0u;
            if (!(sl & kFold)) continue;
            float4* v4 = reinterpret_cast<float4*>(s.val) + (uint64_t)(sl & ~kFold) * D4;
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const uint32_t col = lane + c * G;
              if (col < D4) v4[col] = f4add(v4[col], av[r][c]);
            }
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (j0 + r < nsole)
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const uint32_t col = lane + c * G;
              if (col < D4) main4[(uint64_t)key[r] * D4 + col] = f4add(mv[r][c], av[r][c]);
            }
      }
      // shared keys: the (key, holder) pairs of as many as fit, one lane per
      // pair for the lookups, then one row group per key
      uint32_t np = add && mask ? __popc(mask) : 0u;
      unsigned rest = __ballot_sync(0xFFFFFFFFu, np != 0u);
      while (rest) {   // warp-uniform
        uint32_t end = ((rest >> lane32) & 1u) ? np : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, end, o);
          if (lane32 >= o) end += y;
        }
        const bool now = ((rest >> lane32) & 1u) && end <= kSyncPairs;   // (32 pairs at most each: at least 4 fit)
        const unsigned batch = __ballot_sync(0xFFFFFFFFu, now);
        rest &= ~batch;
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, end, 31 - __clz(batch));
        if (now) {
          uint32_t at = end - np;
          for (uint32_t mm = mask; mm; mm &= mm - 1) sm.pair[wid][at++] = make_uint2(k, (uint32_t)(__ffs(mm) - 1));
        }
        __syncwarp();
        for (uint32_t p = lane32; p < total; p += 32) {
          const uint2 kb = sm.pair[wid][p];
          const int32_t e = s.map[(uint64_t)kb.y * s.K + kb.x];
          const bool pend = !map_none(e) && (owner_state(s.slot_owner[map_slot(e)], s.par) & REP_PENDING);
          sm.pair[wid][p].y = pend ? (uint32_t)map_slot(e) : 0xFFFFFFFFu;
        }
        __syncwarp();
        const uint32_t keys = __popc(batch);
        for (uint32_t j0 = 0; j0 < keys; j0 += GW) {   // warp-uniform: the shuffles below are the whole warp's
          unsigned bm = batch;
          for (uint32_t t = 0; t < j0 + gi; ++t) bm &= bm - 1;   // the (j0 + gi)-th key of the batch
          const int src = bm ? __ffs(bm) - 1 : 0;
          const uint32_t pe = __shfl_sync(0xFFFFFFFFu, end, src), pn = __shfl_sync(0xFFFFFFFFu, np, src);
          if (!bm) continue;
          const uint32_t p0 = pe - pn;
          float4* m4 = main4 + (uint64_t)sm.pair[wid][p0].x * D4;
          float4 m[C];
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            m[c] = col < D4 ? m4[col] : f4zero();
          }
          constexpr int Q = 8 / C > 0 ? 8 / C : 1;   // pending rows in flight
          for (uint32_t q0 = p0; q0 < pe; q0 += Q) {
            float4 av[Q][C];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const uint32_t sl = q0 + q < pe ? sm.pair[wid][q0 + q].y : 0xFFFFFFFFu;
#pragma unroll
              for (int c = 0; c < C; ++c) {
                const uint32_t col = lane + c * G;
                av[q][c] = sl != 0xFFFFFFFFu && col < D4 ? acc4[(uint64_t)sl * D4 + col] : f4zero();
              }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q)
              if (q0 + q < pe && sm.pair[wid][q0 + q].y != 0xFFFFFFFFu)
#pragma unroll
                for (int c = 0; c < C; ++c) m[c] = f4add(m[c], av[q][c]);
          }
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            if (col < D4) m4[col] = m[c];
          }
        }
        __syncwarp();   // pair is rewritten
      }
      __syncwarp();   // list and sole are rewritten
    }
    if (!more) break;
  }
  if (VER) {
    uint32_t unused = 0;
    block_sum2(nref, unused);
    if (threadIdx.x == 0 && nref) atomicAdd(&s.st->sync_refreshed, (unsigned long long)nref);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&s.st->sync_done, 1u) == gridDim.x - 1) {
      // every replica counts as refreshed; versioned: those of shared keys do (and nref above)
      const int32_t live = s.st->live, keys = s.st->live_keys, sole = s.st->sole_keys;
      s.st->sync_keys += (unsigned long long)keys;
      s.st->sync_replicas += (unsigned long long)live;
      atomicAdd(&s.st->sync_refreshed, (unsigned long long)(VER ? live - sole : live));
      s.st->sync_done = 0u;
      s.st->par = s.par ^ 1u;
    }
  }
}

// ---------------------------------------------------------------------------
// inspection
// ---------------------------------------------------------------------------
__global__ void refcounts_kernel(Store s, uint32_t w, const uint32_t* __restrict__ keys, uint64_t n,
                                 uint32_t* __restrict__ out) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t k = keys[i];
    if (k < s.K) out[i] = s.rc[(uint64_t)w * s.K + k];
    else {
      out[i] = 0;
      set_error(s.st, ERR_KEY_RANGE);
    }
  }
}

// owner of each key: -1 at its home (and always without relocation)
__global__ void owners_kernel(Store s, const uint32_t* __restrict__ keys, uint64_t n, int32_t* __restrict__ out) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t k = keys[i];
    if (k < s.K) out[i] = s.own ? own_owner(s.own[k]) : -1;
    else {
      out[i] = -1;
      set_error(s.st, ERR_KEY_RANGE);
    }
  }
}

__global__ void replica_rows_kernel(Store s, uint32_t w, const uint32_t* __restrict__ keys, uint64_t n,
                                    float* __restrict__ val_out, float* __restrict__ acc_out,
                                    uint8_t* __restrict__ has_out) {
  const uint32_t D = s.D;
  s.par = s.st->par;
  for (uint64_t i = blockIdx.x; i < n; i += gridDim.x) {
    const uint32_t k = keys[i];
    const int32_t e = k < s.K ? s.map[(uint64_t)w * s.K + k] : -1;
    const bool has = !map_none(e);
    const uint32_t state = has ? rep_state(s, e) : REP_ALIAS;
    if (threadIdx.x == 0) {
      has_out[i] = has ? 1 : 0;
      if (k >= s.K) set_error(s.st, ERR_KEY_RANGE);
    }
    for (uint32_t c = threadIdx.x; c < D; c += blockDim.x) {
      const float acc = (state & REP_PENDING) ? s.acc[(uint64_t)map_slot(e) * D + c] : 0.f;
      float val = 0.f;
      if (has) val = (state & REP_OWNVAL) ? s.val[(uint64_t)map_slot(e) * D + c] : s.main[(uint64_t)k * D + c];
      val_out[i * D + c] = rep_adds(state) ? val + acc : val;
      acc_out[i * D + c] = acc;
    }
  }
}

__global__ void init_pool_kernel(int32_t* free_stack, uint64_t S, unsigned long long* owner) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < S;
       i += (uint64_t)gridDim.x * blockDim.x) {
    free_stack[i] = (int32_t)(S - 1 - i);   // top of the stack holds slot 0
    owner[i] = kEmptySlot;
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
void launch_pull(const Store& s, int w, const uint32_t* keys, uint64_t n, float* out, int sms,
                 cudaStream_t stream) {
  if (n == 0) return;
  dispatch_gc(s.D / 4, [&](auto Gc, auto Cc) {
    constexpr int G = decltype(Gc)::value, C = decltype(Cc)::value;
    constexpr int R = pull_rows(C);
    note_launches(1);
    launch_after(pull_kernel<G, C, R>, grid_for((n + R - 1) / R, G, sms), kThreads, 0, stream, s, w, keys, n, out);
  });
}

void launch_sync(const Store& s, uint64_t slot_bound, int sms, cudaStream_t stream) {
  if (slot_bound == 0) return;
  if (s.own != nullptr) return launch_sync_copied(s, slot_bound, sms, stream);
  dispatch_gc(s.D / 4, [&](auto Gc, auto Cc) {
    constexpr int G = decltype(Gc)::value, C = decltype(Cc)::value;
    note_launches(1);
    // at least four slots per warp, at most the blocks that are resident together
    uint64_t blocks = (slot_bound + 4 * (kThreads / 32) - 1) / (4 * (kThreads / 32));
    const uint64_t resident = (uint64_t)sms * (C >= 8 ? 2 : 4);
    if (blocks > resident) blocks = resident;
    const unsigned grid = (unsigned)blocks;
    if (s.dirty != nullptr) launch_after(sync_kernel<G, C, true>, grid, kThreads, 0, stream, s);
    else launch_after(sync_kernel<G, C, false>, grid, kThreads, 0, stream, s);
  });
}

void launch_refcounts(const Store& s, uint32_t w, const uint32_t* keys, uint64_t n, uint32_t* out,
                      cudaStream_t stream) {
  if (n == 0) return;
  note_launches(1);
  refcounts_kernel<<<(unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, stream>>>(
      s, w, keys, n, out);
}

void launch_owners(const Store& s, const uint32_t* keys, uint64_t n, int32_t* out, cudaStream_t stream) {
  if (n == 0) return;
  note_launches(1);
  owners_kernel<<<(unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, stream>>>(s, keys, n,
                                                                                                 out);
}

void launch_replica_rows(const Store& s, uint32_t w, const uint32_t* keys, uint64_t n, float* val,
                         float* acc, uint8_t* has, cudaStream_t stream) {
  if (n == 0) return;
  note_launches(1);
  replica_rows_kernel<<<(unsigned)(n < 4096 ? n : 4096), 128, 0, stream>>>(s, w, keys, n, val, acc, has);
}

void launch_init_pool(int32_t* free_stack, uint64_t S, unsigned long long* owner, cudaStream_t stream) {
  uint64_t b = (S + 255) / 256;
  if (b > 65535) b = 65535;
  if (b == 0) return;
  note_launches(1);
  init_pool_kernel<<<(unsigned)b, 256, 0, stream>>>(free_stack, S, owner);
}

}  // namespace adapm
