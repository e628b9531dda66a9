// Advance and sync of a store with relocation, where replicas are copies of
// their main rows (REP_COPIED): val = main and acc = 0 when a replica is
// created, both written by every push, and val = main, acc = 0 again after
// every sync.  The general kernels (advance.cu, store.cu) leave rows alone
// until a replica and its main row differ, which with relocation they do at
// the owner's next push.  There every replica's rows move in every one of
// these calls, and kernels whose row groups load a slot's words and rows
// themselves, several slots at a time, do better: 98k replicas of 200 floats
// sync in 71 us against 90 us with one lane per slot for the words first;
// 41k created and destroyed replicas take 305 us against 326 us.
#include "internal.cuh"
#include "rowgroup.cuh"
#include "store_launch.cuh"

namespace adapm {

namespace {

// evict_create: entry i of the advance evicts the i-th listed slot (any
// worker's: a relocation destroys another worker's replica) -- main[k] +=
// its pending row, by vector atomic adds since main[k] may receive two
// pending rows in one advance (the leaving worker's and a relocated
// holder's) -- and creates the i-th listed key of worker w, val = main,
// pending = 0, in that same slot when there is one (the thread reads the
// pending row before it overwrites it), else in a slot popped from the
// stack; an evicted slot with no creation to take it is pushed.  A created
// key is never one whose replica this advance destroys (a worker joins or
// leaves a key, not both), so its main row is final.  R entries per row
// group at a time; a round's loads (owner records, pending rows, main rows)
// go out together with the next round's list entries.
template <int G, int C>
__global__ void __launch_bounds__(kThreads, C >= 8 ? 2 : 3) evict_create_copied_kernel(Store s, uint32_t w,
                                                                                     const uint32_t* evict_list,
                                                                                     const uint32_t* create_list) {
  after_previous();
  constexpr int R = 4 / C > 0 ? 4 / C : 1;
  const int lane = threadIdx.x & (G - 1);
  const uint32_t D4 = s.D >> 2;
  const uint32_t ne = s.st->adv_ne, nc = s.st->adv_nc;
  const int32_t top = s.st->adv_top;
  if (s.st->errors & ERR_TIMEOUT) return;   // a sort gave up: the events that fill the lists have returned, too
  const uint64_t n = ne > nc ? ne : nc;
  float4* main4 = reinterpret_cast<float4*>(s.main);
  float4* val4 = reinterpret_cast<float4*>(s.val);
  float4* acc4 = reinterpret_cast<float4*>(s.acc);
  int32_t* mapw = s.map + (uint64_t)w * s.K;
  const uint64_t g = group_id<G>(), ng = group_count<G>();
  const uint64_t step = ng * R;
  // list entries out of range (slots >= S, keys >= K) are skipped and reported
  auto load_entries = [&](uint64_t i0, int32_t (&es)[R], uint32_t (&ck)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t i = i0 + r;
      const uint32_t e = i < ne ? evict_list[i] : 0xFFFFFFFFu;
      es[r] = e < s.S ? (int32_t)e : -1;
      ck[r] = i < nc ? create_list[i] : kNoKey;
      if ((i < ne && e >= s.S) || (i < nc && ck[r] >= s.K)) {
        set_error(s.st, ERR_INTERNAL);
        if (ck[r] >= s.K) ck[r] = kNoKey;
      }
    }
  };
  int32_t es[R];
  uint32_t ck[R];
  load_entries(g * R, es, ck);
  for (uint64_t i0 = g * R; i0 < n; i0 += step) {
    int32_t cs[R];
    unsigned long long ow[R];
    float4 ac[R][C], mv[R][C];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t i = i0 + r;
      // slot of the creation: the paired evicted slot, else popped (top first;
      // a pair whose evicted slot is out of range has none)
      cs[r] = ck[r] == kNoKey || (es[r] < 0 && i < ne)
                  ? -1
                  : (es[r] >= 0 ? es[r] : s.free_stack[top - 1 - (int32_t)(i - ne)]);
      ow[r] = es[r] >= 0 ? s.slot_owner[es[r]] : 0ull;
      const bool bad_slot = ck[r] != kNoKey && (cs[r] < 0 || (uint64_t)cs[r] >= s.S);
      const bool bad_owner = es[r] >= 0 && ((uint32_t)ow[r] >= s.K || (ow[r] >> 32) >= s.W);
      if (bad_slot || bad_owner) {
        set_error(s.st, ERR_INTERNAL);   // a free-stack entry or owner record out of range: skipped
        if (bad_slot) {
          cs[r] = -1;
          ck[r] = kNoKey;
        }
        if (bad_owner) es[r] = -1;
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t col = lane + c * G;
        ac[r][c] = (es[r] >= 0 && col < D4) ? acc4[(uint64_t)es[r] * D4 + col] : f4zero();
        mv[r][c] = (ck[r] != kNoKey && col < D4) ? main4[(uint64_t)ck[r] * D4 + col] : f4zero();
      }
    }
    int32_t es1[R];
    uint32_t ck1[R];
    load_entries(i0 + step, es1, ck1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t i = i0 + r;
      if (es[r] >= 0) {
        const uint32_t k = (uint32_t)ow[r], a = (uint32_t)(ow[r] >> 32);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          if (col < D4) atomicAdd(main4 + (uint64_t)k * D4 + col, ac[r][c]);
        }
        if (lane == 0) {
          if (s.dirty != nullptr) s.dirty[k] = 1;   // versioned refresh: main changed
          s.map[(uint64_t)a * s.K + k] = -1;
          atomicAnd(s.holders + k, ~(1u << a));
          if (ck[r] == kNoKey) {
            s.slot_owner[es[r]] = kEmptySlot;
            s.free_stack[top + (int32_t)(i - nc)] = es[r];
          }
        }
      }
      if (ck[r] != kNoKey) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          if (col < D4) {
            val4[(uint64_t)cs[r] * D4 + col] = mv[r][c];
            acc4[(uint64_t)cs[r] * D4 + col] = f4zero();
          }
        }
        if (lane == 0) {
          // versioned refresh: the new replica has seen every update (a stale
          // replica of another worker is refreshed anyway: the key has two holders)
          if (s.dirty != nullptr) s.dirty[ck[r]] = 0;
          mapw[ck[r]] = cs[r];
          atomicOr(s.holders + ck[r], 1u << w);
          s.slot_owner[cs[r]] = ((unsigned long long)w << 32) | ck[r];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      es[r] = es1[r];
      ck[r] = ck1[r];
    }
  }
}

// ---------------------------------------------------------------------------
// sync
// ---------------------------------------------------------------------------
// VER: versioned refresh (s.dirty is set)
template <int G, int C, bool VER>
__global__ void __launch_bounds__(kThreads, C >= 8 ? 2 : (VER && C == 1 ? 3 : 4)) sync_copied_kernel(Store s) {
  after_previous();
  const int lane = threadIdx.x & (G - 1);
  const uint32_t D4 = s.D >> 2;
  const uint64_t hw = (uint64_t)s.st->high_water;
  if (s.st->errors & ERR_TIMEOUT) return;   // a sort gave up
  float4* main4 = reinterpret_cast<float4*>(s.main);
  float4* val4 = reinterpret_cast<float4*>(s.val);
  float4* acc4 = reinterpret_cast<float4*>(s.acc);
  const uint64_t g = group_id<G>(), ng = group_count<G>();
  uint32_t nkeys = 0, nreps = 0, nref = 0;   // nref: VER only
  __shared__ int32_t hslots[kThreads / G][32];   // holders' slots of the key a group merges (W <= 32)
  const unsigned gmask = G == 32 ? 0xFFFFFFFFu : (((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1)));
  // R slots per group at a time: owners, holder masks, then (for keys held
  // by one worker only, the common case) main and pending rows, each as one
  // round of independent loads.  Versioned refresh (App. B.1.2: a holder
  // receives only updates it has not seen): a sole holder's value is left
  // alone unless main[k] was written other than by a sync since the last
  // sync of k (dirty[k]); keys with several holders are always refreshed.
  constexpr int R = 4 / C > 0 ? 4 / C : 1;
  for (uint64_t b = g * R; b < hw; b += ng * R) {
    unsigned long long own[R];
    uint32_t mk[R];
#pragma unroll
    for (int r = 0; r < R; ++r) own[r] = b + r < hw ? s.slot_owner[b + r] : kEmptySlot;
#pragma unroll
    for (int r = 0; r < R; ++r) mk[r] = own[r] != kEmptySlot ? s.holders[(uint32_t)own[r]] : 0u;
    // a live slot's key is held by this worker alone iff its mask has one bit
    // (its own); such a mask is known, so it is replaced by the refresh flag
    // (1: write the value, 0: leave it), which keeps at most one bit set
    auto is_single = [&](int r) { return own[r] != kEmptySlot && __popc(mk[r]) <= 1; };
    float4 mv[R][C], av[R][C];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool single = is_single(r);
      if (VER && single) mk[r] = (uint32_t)s.dirty[(uint32_t)own[r]];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t col = lane + c * G;
        const bool cv = single && col < D4;
        mv[r][c] = cv ? main4[(uint64_t)(uint32_t)own[r] * D4 + col] : f4zero();
        av[r][c] = cv ? acc4[(b + r) * D4 + col] : f4zero();
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!is_single(r)) continue;
      const uint32_t k = (uint32_t)own[r];
      if (lane == 0) {
        nkeys += 1;
        nreps += 1;
        if (VER && mk[r]) {
          nref += 1;
          s.dirty[k] = 0;
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t col = lane + c * G;
        if (col < D4) {
          const float4 m = f4add(mv[r][c], av[r][c]);
          main4[(uint64_t)k * D4 + col] = m;
          if (!VER || mk[r]) val4[(b + r) * D4 + col] = m;
          acc4[(b + r) * D4 + col] = f4zero();
        }
      }
    }
    // keys with several holders: the lowest holder merges all of them
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (own[r] == kEmptySlot || is_single(r)) continue;
      const uint32_t w = (uint32_t)(own[r] >> 32);
      const uint32_t k = (uint32_t)own[r];
      const uint32_t mask = mk[r];
      if ((uint32_t)(__ffs(mask) - 1) != w) continue;   // the lowest holder merges
      if (lane == 0) {
        nkeys += 1;
        nreps += (uint32_t)__popc(mask);
        if (VER) {
          nref += (uint32_t)__popc(mask);
          s.dirty[k] = 0;
        }
      }
      // Holders that fit in one round of Q rows: their slots are looked up with
      // the sum and again for the writes.  More: each lane looks up one
      // holder's slot (G at a time) into shared memory, so the sum and the
      // writes need no second lookup.  Both add the pending rows to main in
      // ascending worker order.
      if (__popc(mask) <= (4 / C > 0 ? 4 / C : 1)) {
        float4 m[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          m[c] = col < D4 ? main4[(uint64_t)k * D4 + col] : f4zero();
        }
        constexpr int Q = 4 / C > 0 ? 4 / C : 1;
        uint32_t mm = mask;
        while (mm) {
          int32_t hs[Q];
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            hs[q] = -1;
            if (mm) {
              const uint32_t wb = __ffs(mm) - 1;
              mm &= mm - 1;
              hs[q] = s.map[(uint64_t)wb * s.K + k];
            }
          }
          float4 t[Q][C];
#pragma unroll
          for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const uint32_t col = lane + c * G;
              t[q][c] = (hs[q] >= 0 && col < D4) ? acc4[(uint64_t)hs[q] * D4 + col] : f4zero();
            }
#pragma unroll
          for (int q = 0; q < Q; ++q)
            if (hs[q] >= 0)
#pragma unroll
              for (int c = 0; c < C; ++c) m[c] = f4add(m[c], t[q][c]);
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          if (col < D4) main4[(uint64_t)k * D4 + col] = m[c];
        }
        mm = mask;
        while (mm) {
          const uint32_t wb = __ffs(mm) - 1;
          mm &= mm - 1;
          const int32_t h = s.map[(uint64_t)wb * s.K + k];
          if (h < 0) continue;
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            if (col < D4) {
              val4[(uint64_t)h * D4 + col] = m[c];
              acc4[(uint64_t)h * D4 + col] = f4zero();
            }
          }
        }
      } else {
        float4 m[C];   // (loaded with the holders' slots)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          m[c] = col < D4 ? main4[(uint64_t)k * D4 + col] : f4zero();
        }
        // the holders' slots: one slot-map lookup per lane (holder j by lane j,
        // G at a time), kept in shared memory for the sum and the writes
        const int nh = __popc(mask);
        int32_t* hsl = hslots[threadIdx.x / G];
        for (int j = lane; j < nh; j += G) {
          uint32_t mm = mask;   // the j-th set bit (j < nh, so mm stays nonzero)
          for (int t = 0; t < j; ++t) mm &= mm - 1;
          const uint32_t wb = (uint32_t)(__ffs(mm) - 1);
          hsl[j] = s.map[(uint64_t)wb * s.K + k];
        }
        __syncwarp(gmask);
        constexpr int Q = 4 / C > 0 ? 4 / C : 1;
        // pending rows added in ascending worker order, Q rows in flight
        for (int j0 = 0; j0 < nh; j0 += Q) {
          int32_t hs[Q];
#pragma unroll
          for (int q = 0; q < Q; ++q) hs[q] = j0 + q < nh ? hsl[j0 + q] : -1;
          float4 t[Q][C];
#pragma unroll
          for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const uint32_t col = lane + c * G;
              t[q][c] = (hs[q] >= 0 && col < D4) ? acc4[(uint64_t)hs[q] * D4 + col] : f4zero();
            }
#pragma unroll
          for (int q = 0; q < Q; ++q)
            if (hs[q] >= 0)
#pragma unroll
              for (int c = 0; c < C; ++c) m[c] = f4add(m[c], t[q][c]);
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          if (col < D4) main4[(uint64_t)k * D4 + col] = m[c];
        }
        for (int j = 0; j < nh; ++j) {
          const int32_t h = hsl[j];
          if (h < 0) continue;
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            if (col < D4) {
              val4[(uint64_t)h * D4 + col] = m[c];
              acc4[(uint64_t)h * D4 + col] = f4zero();
            }
          }
        }
        __syncwarp(gmask);   // hsl is reused by the group's next key
      }
    }
  }
  block_sum2(nkeys, nreps);
  if (VER) {
    __syncthreads();   // block_sum2's shared words are reused below
    uint32_t unused = 0;
    block_sum2(nref, unused);
  }
  if (threadIdx.x == 0 && nkeys) {
    atomicAdd(&s.st->sync_keys, (unsigned long long)nkeys);
    atomicAdd(&s.st->sync_replicas, (unsigned long long)nreps);
    atomicAdd(&s.st->sync_refreshed, (unsigned long long)(VER ? nref : nreps));
  }
}

}  // namespace

void launch_evict_create_copied(const Store& s, uint32_t w, const uint32_t* create_list, const uint32_t* evict_list,
                                uint64_t max_events, int sms, cudaStream_t stream) {
  dispatch_gc(s.D / 4, [&](auto Gc, auto Cc) {
    constexpr int G = decltype(Gc)::value, C = decltype(Cc)::value;
    constexpr uint64_t R = 4 / C > 0 ? 4 / C : 1;   // list entries per group, as in the kernel
    note_launches(1);
    const unsigned grid = grid_for((max_events + R - 1) / R, G, sms);
    launch_after(evict_create_copied_kernel<G, C>, grid, kThreads, 0, stream, s, w, evict_list, create_list);
  });
}

void launch_sync_copied(const Store& s, uint64_t slot_bound, int sms, cudaStream_t stream) {
  if (slot_bound == 0) return;
  dispatch_gc(s.D / 4, [&](auto Gc, auto Cc) {
    constexpr int G = decltype(Gc)::value, C = decltype(Cc)::value;
    note_launches(1);
    constexpr uint64_t R = 4 / C > 0 ? 4 / C : 1;   // slots per group, as in the kernel
    const unsigned grid = grid_for((slot_bound + R - 1) / R, G, sms);
    if (s.dirty != nullptr) launch_after(sync_copied_kernel<G, C, true>, grid, kThreads, 0, stream, s);
    else launch_after(sync_copied_kernel<G, C, false>, grid, kThreads, 0, stream, s);
  });
}

}  // namespace adapm
