// push: the rows of each distinct key of one call are summed and added to the
// worker's replica (value and pending updates) or to main (Sec. 4,
// App. B.1.2).  Sorted (key, position) pairs are split into fixed chunks,
// a block's groups taking consecutive chunks of one span; each group sums
// the delta rows of every key segment of its chunk in position order and
// adds the sum to its target.  A segment cut by chunk boundaries leaves a
// partial sum per chunk; the block adds those of segments inside its span
// in chunk order and applies them, and the partial sums of segments that run
// past a span are added in span order by push_combine.
//
// Where a delta row comes from (kSrc*): an array (adapm_push, the MF step), or
// a training step's factors.  The ComplEx and SGNS steps' delta rows are a
// scalar times one of a few rows (a triple's product, a centre's vector), or
// the AdaGrad update of such a gradient, so the step writes those rows once
// and a scalar per row occurrence, and the delta rows are formed here, where
// they are summed: they never travel through memory, and the few rows they
// are formed from stay in L2.  Written and read back, they were two thirds of
// the steps' traffic.  Per clock of 8 workers, step + scatter, delta rows and
// as both are now: SGNS, 8192 centres of 261 rows x 300 floats 9.88 + 8.43 and
// 3.64 + 3.11 ms; ComplEx, 4096 triples of 103 rows x 512 floats 3.77 + 2.29
// and 1.10 + 2.42 ms.
#pragma once

#include "internal.cuh"
#include "rowgroup.cuh"
#include "store_launch.cuh"

namespace adapm {

namespace {

// What a push kernel needs to know before its first row: loaded together and
// first, used only once the loads that do not depend on it are under way.
struct PushWords {
  uint32_t errors, miss, live, par;
};
__device__ __forceinline__ PushWords push_words(const Store& s, const PushArgs& a) {
  auto ld = [](const void* p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
  };
  return PushWords{ld(&s.st->errors), ld(a.plan_seq != 0u ? a.plan_word : &s.st->plan_miss), ld(&s.st->live),
                   ld(&s.st->par)};
}
// 0: an earlier sort gave up, nothing may be touched; 1: the sorted keys and
// positions are those in `a` (the plan's); 2: they are the sort's, which `a`
// now names (the plan's check stored a mismatch for this push).
// any_replica: there are replicas that may be aliases of a main row.
__device__ __forceinline__ int push_resolve(Store& s, PushArgs& a, const PushWords& pw, bool& any_replica) {
  any_replica = s.own == nullptr && (int32_t)pw.live > 0;
  s.par = pw.par;
  if (pw.errors & ERR_TIMEOUT) return 0;
  if (a.plan_seq == 0u || pw.miss != a.plan_seq) return 1;
  a.skeys = a.alt_keys;
  a.spos = a.alt_pos;
  return 2;
}

// ---------------------------------------------------------------------------
// push: chunked segmented reduction over key-sorted (key, position) pairs
// ---------------------------------------------------------------------------
// The target of one key's sum: the worker's replica (slot >= 0) in its state
// before this push, or main[k] (slot -1) with the workers that hold replicas
// of k (0: none has to be looked at).
struct Target {
  int32_t slot;
  uint32_t state;
  uint32_t holders;
};

// Looks the target of key k up: the state before this push.
__device__ __forceinline__ Target look_target(const Store& s, uint32_t w, uint32_t k, bool any_replica) {
  const int32_t e = s.map[(uint64_t)w * s.K + k];
  Target t{-1, REP_ALIAS, 0u};
  if (map_none(e)) {
    if (any_replica) t.holders = s.holders[k];
    return t;
  }
  t.slot = map_slot(e);
  t.state = rep_state(s, e);
  return t;
}
// Records the state after this push.  One thread per key and push (the key
// has one segment).
__device__ __forceinline__ void mark_target(const Store& s, uint32_t w, uint32_t k, const Target& t) {
  if (t.slot < 0) {
    if (s.dirty != nullptr) s.dirty[k] = 1;   // versioned refresh: main written by a worker without a replica
    return;
  }
  if (t.state == REP_COPIED) return;
  if (t.state == REP_ALIAS) s.map[(uint64_t)w * s.K + k] = map_touch(t.slot);
  const uint32_t after = (t.state & REP_PENDING) ? REP_PENDING | REP_OWNVAL | REP_FOLDED : t.state | REP_PENDING;
  set_owner_hi(s, t.slot, owner_hi(w, after, s.par));
}

// Adds one key's sum to its target (a whole row group).  The segment is the
// only writer of its targets in this push: a row that is not yet set is
// stored, others take vector atomic adds, which give the plain fp32 sums
// without a round trip of the target row.
template <int G, int C, int SRC>
__device__ __forceinline__ void apply_sum(const Store& s, uint32_t k, const Target& t, const float4 (&sum)[C],
                                          int lane, unsigned gmask) {
  const uint32_t D4 = s.D >> 2;
  // the lane's columns (push_chunks_kernel)
  const uint32_t T4 = SRC == kSrcAda ? D4 / 2 : D4;
  auto col_of = [&](int c) -> uint32_t {   // D4: none
    const uint32_t q = lane + (SRC == kSrcAda ? c % (C / 2 > 0 ? C / 2 : 1) : c) * G;
    return q >= T4 ? D4 : (SRC == kSrcAda && c >= C / 2 ? T4 + q : q);
  };
  float4* main4 = reinterpret_cast<float4*>(s.main) + (uint64_t)k * D4;
  if (t.slot < 0) {
    if (t.holders) {
      detach_aliases<G, C>(s, k, t.holders, lane, gmask);
      // (its lanes copy columns of another layout: all of them before main changes)
      if (SRC == kSrcAda) __syncwarp(gmask);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = col_of(c);
      if (col < D4) atomicAdd(main4 + col, sum[c]);
    }
    return;
  }
  float4* val4 = reinterpret_cast<float4*>(s.val) + (uint64_t)t.slot * D4;
  float4* acc4 = reinterpret_cast<float4*>(s.acc) + (uint64_t)t.slot * D4;
  if (rep_adds(t.state)) {   // the second push: acc is folded into a value of the replica's own
    const float4* base4 = (t.state & REP_OWNVAL) ? val4 : main4;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = col_of(c);
      if (col >= D4) continue;
      const float4 p = acc4[col];
      val4[col] = f4add(f4add(base4[col], p), sum[c]);
      acc4[col] = f4add(p, sum[c]);
    }
    return;
  }
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const uint32_t col = col_of(c);
    if (col >= D4) continue;
    if (t.state & REP_FOLDED) {
      atomicAdd(val4 + col, sum[c]);
      atomicAdd(acc4 + col, sum[c]);
    } else {
      acc4[col] = sum[c];
    }
  }
}

// The same for a segment whose target nobody has looked up yet: lane 0 of the
// group does.
template <int G, int C, int SRC>
__device__ __forceinline__ void take_and_apply(const Store& s, uint32_t w, uint32_t k, const float4 (&sum)[C],
                                               int lane, unsigned gmask, bool any_replica) {
  Target t{-1, REP_ALIAS, 0u};
  if (lane == 0) {
    t = look_target(s, w, k, any_replica);
    mark_target(s, w, k, t);
  }
  t.slot = __shfl_sync(gmask, t.slot, 0, G);
  t.state = __shfl_sync(gmask, t.state, 0, G);
  t.holders = __shfl_sync(gmask, t.holders, 0, G);
  apply_sum<G, C, SRC>(s, k, t, sum, lane, gmask);
}

// Each block stages a span of up to kPushSpan consecutive sorted positions
// (keys and source positions) in shared memory; its groups own consecutive
// chunks of it.  A segment cut by chunk boundaries leaves a partial sum per
// chunk (a tail piece in the chunk it starts in, head pieces in the chunks
// it continues into).
constexpr int kPushSpan = 3072;
constexpr uint32_t kPushCopies = 512;
// push_chunks blocks per SM by its launch bounds, and rows a group keeps in
// flight.  Shared memory fits as many, but for a step's scalars: rows of three
// vectors per lane then take 82 KB a block, of which two fit an SM, rows of
// eight 123 KB, of which one does.  (There the registers are cut for a block
// more than runs, and push_chunk_rows counts its place.)
constexpr int push_blocks_per_sm(int C) { return C >= 4 ? 2 : 3; }
constexpr int push_rows_in_flight(int C) { return C == 3 ? 2 : (4 / C > 0 ? 4 / C : 1); }

// Dynamic shared memory of push_chunks: the head and tail piece of every
// chunk (a row of G * C float4 per group each), then the staged span (with
// the factors of a step's rows: a scalar each).
template <int C, int SRC>
constexpr size_t push_chunks_smem() {
  return 2 * (size_t)kThreads * C * sizeof(float4) + (kPushSpan + 2) * sizeof(uint32_t) +
         kPushSpan * sizeof(uint32_t) + kPushSpan * sizeof(int32_t) + kPushSpan +
         (SRC == kSrcRows ? 0 : kPushSpan * sizeof(float));
}

// AdaGrad deltas of one gradient g under accumulator a.  The products are
// rounded by themselves: the sums that follow see the same delta rows as if
// they had been stored.
__device__ __forceinline__ float ada_theta(float g, float a, float lr, float eps) {
  return __fmul_rn(-lr * g, __frsqrt_rn(a + g * g + eps));   // correctly rounded 1/sqrt
}
__device__ __forceinline__ float4 ada_theta4(float4 g, float4 a, float lr, float eps) {
  return make_float4(ada_theta(g.x, a.x, lr, eps), ada_theta(g.y, a.y, lr, eps), ada_theta(g.z, a.z, lr, eps),
                     ada_theta(g.w, a.w, lr, eps));
}
__device__ __forceinline__ float4 f4mul(float4 a, float s) {
  return make_float4(__fmul_rn(a.x, s), __fmul_rn(a.y, s), __fmul_rn(a.z, s), __fmul_rn(a.w, s));
}
__device__ __forceinline__ float4 f4square(float4 g) {
  return make_float4(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y), __fmul_rn(g.z, g.z), __fmul_rn(g.w, g.w));
}

// Row of x that the delta row at position `pos` of a step's batch is formed
// from (the layouts of the step kernels).
__device__ __forceinline__ uint32_t factor_row(const PushArgs& a, uint32_t pos) {
  const uint32_t n = a.x_n;
  if (a.x_kind == kFactorsComplEx) return pos < 3 * n ? pos : 2 * n + (pos - 3 * n) / a.x_per;
  const uint32_t i = pos / a.x_per;                                 // SGNS: the centre's vector, or its own update
  return pos == i * a.x_per ? n + i : i;
}

// SRC = kSrcAda: a lane owns C / 2 float4 of the theta half of a row and the
// same ones of the accumulator half, so a gradient is loaded once for both.
template <int G, int C, int R, int SRC>
__global__ void __launch_bounds__(kThreads, push_blocks_per_sm(C)) push_chunks_kernel(Store s, PushArgs a) {
  after_previous();
  const PushWords pw = push_words(s, a);
  bool any_replica = false, resolved = false;
  constexpr int NG = kThreads / G;
  const uint32_t CH = (uint32_t)a.chunk;            // rows per group, NG * CH <= kPushSpan
  const uint32_t span = NG * CH;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ uint2 copies[kPushCopies];   // (key, holder), then (key, slot): old main rows to copy first
  __shared__ uint32_t ncopy;
  float4* ph = reinterpret_cast<float4*>(dsm);                    // head piece of each chunk
  float4* pt = ph + kThreads * C;                                 // tail piece of each chunk
  uint32_t* sk = reinterpret_cast<uint32_t*>(pt + kThreads * C);  // sk[0]: key before the span; sk[1+len]: after it
  uint32_t* sp = sk + kPushSpan + 2;                              // source row of each sorted position
  int32_t* ss = reinterpret_cast<int32_t*>(sp + kPushSpan);       // target slot of rows that end a whole segment
  uint8_t* sf = reinterpret_cast<uint8_t*>(ss + kPushSpan);       // row flags (below)
  // flags: bit0 a piece ends at this row, bit1 that piece began inside the
  // row's chunk, bit2 the key's segment ends here, bit3 a piece begins here,
  // bit4 the row holds a key (not a skipped one); a row with bits 0-2 all set
  // ends a segment that lies inside one chunk and carries its target's state
  // in bits 5-7 (main rows: bit 7 when aliases of it are left to detach)
  const unsigned gmask = group_mask<G>();
  const int lane = threadIdx.x & (G - 1);
  const int gi = threadIdx.x / G;
  const uint32_t D4 = s.D >> 2;
  const float4* d4 = reinterpret_cast<const float4*>(a.deltas);
  float4* acc4 = reinterpret_cast<float4*>(s.acc);
  float4* sp4 = reinterpret_cast<float4*>(a.span_parts);
  float* sc = reinterpret_cast<float*>(sf + kPushSpan);           // a step's scalar of each position
  const uint32_t T4 = SRC == kSrcAda ? D4 / 2 : D4;               // float4 of a factor row
  // column of the lane's c-th float4 of a row, and whether it is one
  auto col_of = [&](int c) {
    return SRC == kSrcAda && c >= C / 2 ? T4 + lane + (c - C / 2) * G : (uint32_t)(lane + c * G);
  };
  auto col_ok = [&](int c) { return (uint32_t)(lane + (SRC == kSrcAda ? c % (C / 2 > 0 ? C / 2 : 1) : c) * G) < T4; };
  uint32_t heads = 0;
  for (uint64_t P0 = (uint64_t)blockIdx.x * span; P0 < a.n; P0 += (uint64_t)gridDim.x * span) {
    const uint32_t len = (uint32_t)(a.n - P0 < (uint64_t)span ? a.n - P0 : span);
    __syncthreads();
    if (threadIdx.x == 0) ncopy = 0;
    auto stage = [&]() {
      for (uint32_t i = threadIdx.x; i < len; i += kThreads) {
        sk[1 + i] = a.skeys[P0 + i];
        sp[i] = a.spos[P0 + i];
      }
      if (threadIdx.x == 0) {
        sk[0] = P0 > 0 ? a.skeys[P0 - 1] : kNoKey;
        sk[1 + len] = P0 + len < a.n ? a.skeys[P0 + len] : kNoKey;
      }
    };
    stage();
    if (!resolved) {   // (uniform over the grid)
      resolved = true;
      const int from = push_resolve(s, a, pw, any_replica);
      if (from == 0) return;
      if (from == 2) {
        __syncthreads();
        stage();
      }
    }
    __syncthreads();
    // per-row control, one thread per row, and the target of every whole
    // segment; SU rows per thread and round, whose random accesses (map
    // entries, then states or holder masks) go out together (one row after
    // the other, nine rows per thread at 2^20 rows cost a tenth of the kernel)
    constexpr int SU = C >= 3 ? 2 : 4;
    for (uint32_t i0 = threadIdx.x; i0 < len; i0 += SU * kThreads) {
      uint32_t key[SU];
      uint8_t f[SU];
      int32_t e[SU];
      float coef[SU];
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const uint32_t i = i0 + u * kThreads;
        key[u] = kNoKey;
        f[u] = 0;
        e[u] = -1;
        coef[u] = 0.f;
        if (i >= len) continue;
        const uint32_t k = sk[1 + i];
        key[u] = k;
        // (sorted keys are valid or the skip sentinel; anything else out of
        // range, like a position outside the batch, is an internal error)
        if (k < s.K && sp[i] < a.n) {
          const uint32_t cs = i - i % CH;                          // first row of the chunk
          const uint32_t ce = cs + CH < len ? cs + CH : len;        // end of the chunk
          const bool seg_begin = (P0 + i == 0) || sk[i] != k;       // sk[i] is the key of row i-1
          const bool seg_end = (P0 + i + 1 >= a.n) || sk[1 + i + 1] != k;
          const bool started = (P0 + cs == 0) || sk[cs] != k;       // piece began inside the chunk
          const bool piece_end = seg_end || i + 1 == ce;
          f[u] = (piece_end ? 1 : 0) | (started ? 2 : 0) | (seg_end ? 4 : 0) |
                 ((seg_begin || i == cs) ? 8 : 0) | 16;
          if (seg_begin) ++heads;
          // (AdaGrad sources: also where the accumulators of a piece's first row are)
          if ((f[u] & 7) == 7 || (SRC == kSrcAda && (f[u] & 8))) e[u] = s.map[(uint64_t)a.worker * s.K + k];
          if (SRC != kSrcRows) coef[u] = a.coef[sp[i]];
        } else if (k != kNoKey || sp[i] >= a.n) {
          set_error(s.st, ERR_INTERNAL);
        }
      }
      uint32_t state[SU], holders[SU];
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const bool whole = (f[u] & 7) == 7;
        state[u] = map_none(e[u]) ? REP_ALIAS : rep_state(s, e[u]);
        holders[u] = whole && map_none(e[u]) && any_replica ? s.holders[key[u]] : 0u;
      }
#pragma unroll
      for (int u = 0; u < SU; ++u) {
        const uint32_t i = i0 + u * kThreads;
        if (i >= len) continue;
        const Target t{map_none(e[u]) ? -1 : map_slot(e[u]), state[u], holders[u]};
        const bool whole = (f[u] & 7) == 7;
        if (whole && SRC != kSrcAda) mark_target(s, a.worker, key[u], t);
        f[u] |= (uint8_t)(state[u] << 5);
        // a main row that others replicate: its (key, holder) pairs are
        // listed for the block (as far as the list goes)
        if (t.holders) {
          uint32_t at = atomicAdd(&ncopy, (uint32_t)__popc(t.holders));
          for (uint32_t h = t.holders; h; h &= h - 1, ++at) {
            if (at < kPushCopies) copies[at] = make_uint2(key[u], (uint32_t)(__ffs(h) - 1));
            else f[u] |= 128;
          }
        }
        sf[i] = f[u];
        ss[i] = whole || (SRC == kSrcAda && (f[u] & 8)) ? t.slot : -2;
        if (SRC != kSrcRows) {
          sc[i] = coef[u];
          sp[i] = (f[u] & 16) ? factor_row(a, sp[i]) : 0u;
        }
      }
    }
    __syncthreads();
    if (SRC == kSrcAda) {
      // the states after this push, now that the block has read those before
      // it (a key with a whole segment here has no row in another block)
      for (uint32_t i = threadIdx.x; i < len; i += kThreads)
        if ((sf[i] & 7) == 7) mark_target(s, a.worker, sk[1 + i], Target{ss[i], (uint32_t)(sf[i] >> 5), 0u});
    }
    if (ncopy) {   // block-uniform
      // aliases of the main rows that are about to change get the old rows:
      // one thread per pair for the lookups, then one group per row
      const uint32_t nc = ncopy < kPushCopies ? ncopy : kPushCopies;
      for (uint32_t i = threadIdx.x; i < nc; i += kThreads)
        copies[i].y = (uint32_t)take_alias(s, copies[i].y, copies[i].x);
      __syncthreads();
      float4* val4 = reinterpret_cast<float4*>(s.val);
      const float4* main4 = reinterpret_cast<const float4*>(s.main);
      for (uint32_t i = gi; i < nc; i += NG) {
        const uint2 kc = copies[i];
        if (kc.y == 0xFFFFFFFFu) continue;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          if (col < D4) val4[(uint64_t)kc.y * D4 + col] = main4[(uint64_t)kc.x * D4 + col];
        }
      }
      __syncthreads();
    }
    const uint32_t p0 = gi * CH;
    const uint32_t p1 = p0 + CH < len ? p0 + CH : len;
    float4 run[C];
#pragma unroll
    for (int c = 0; c < C; ++c) run[c] = f4zero();
    float4 cura[SRC == kSrcAda ? C / 2 : 1];   // accumulators of the current key
    // software-pipelined: the delta rows of the next round are in flight
    // while this round's are summed and applied
    auto fetch = [&](uint32_t p, uint8_t (&f)[R], float4 (&d)[R][C]) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool v = p + r < p1;
        f[r] = v ? sf[p + r] : 0;
        const uint32_t src = v ? sp[p + r] : 0u;
        if (SRC != kSrcAda) {
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t col = lane + c * G;
            d[r][c] = ((f[r] & 16) && col < D4) ? d4[(uint64_t)src * D4 + col] : f4zero();
          }
        } else {
          // gradient factor, and (where a piece begins) the key's accumulators
#pragma unroll
          for (int c = 0; c < C / 2; ++c) {
            const uint32_t q = lane + c * G;
            d[r][c] = ((f[r] & 16) && q < T4) ? d4[(uint64_t)src * T4 + q] : f4zero();
          }
          if (f[r] & 8) {
            const uint32_t state = f[r] >> 5;
            const int32_t sl = ss[p + r];
            const uint32_t key = sk[1 + p + r];
            const float4* base = sl >= 0 && (state & REP_OWNVAL)
                                     ? reinterpret_cast<const float4*>(s.val) + (uint64_t)sl * D4
                                     : reinterpret_cast<const float4*>(s.main) + (uint64_t)key * D4;
#pragma unroll
            for (int c = 0; c < C / 2; ++c) {
              const uint32_t q = lane + c * G;
              d[r][C / 2 + c] = q < T4 ? base[T4 + q] : f4zero();
              if (sl >= 0 && rep_adds(state) && q < T4)
                d[r][C / 2 + c] = f4add(d[r][C / 2 + c], acc4[(uint64_t)sl * D4 + T4 + q]);
            }
          }
        }
      }
    };
    uint8_t f[R];
    float4 d[R][C];
    fetch(p0, f, d);
    for (uint32_t p = p0; p < p1; p += R) {
      uint8_t fn[R];
      float4 dn[R][C];
      fetch(p + R, fn, dn);
      if (SRC != kSrcRows) {
        // the delta rows of the round from their factors
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float coef = p + r < p1 ? sc[p + r] : 0.f;
#pragma unroll
          for (int c = 0; c < (SRC == kSrcAda ? C / 2 : C); ++c) {
            const float4 g = f4mul(d[r][c], coef);
            if (SRC == kSrcSgd) {
              d[r][c] = g;
            } else {
              if (f[r] & 8) cura[c] = d[r][C / 2 + c];
              d[r][c] = ada_theta4(g, cura[c], a.lr, a.eps);
              d[r][C / 2 + c] = f4square(g);
            }
          }
        }
      }
      int32_t sl[R];
      uint32_t k[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        sl[r] = (f[r] & 7) == 7 ? ss[p + r] : -2;
        k[r] = p + r < p1 ? sk[1 + p + r] : kNoKey;
      }
      // running sums in position order
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          run[c] = (f[r] & 8) ? d[r][c] : f4add(run[c], d[r][c]);
          d[r][c] = run[c];
        }
      }
      // a whole segment's sum goes to its target; the usual one is a replica
      // that has not been pushed to since its creation or the last sync: the
      // sum becomes its pending row
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const uint32_t state = f[r] >> 5;
        if (sl[r] >= 0 && !(state & REP_PENDING)) {
#pragma unroll
          for (int c = 0; c < C; ++c) {
            if (col_ok(c)) acc4[(uint64_t)sl[r] * D4 + col_of(c)] = d[r][c];
          }
        } else if (sl[r] != -2) {
          const Target t{sl[r], state, (sl[r] < 0 && (f[r] & 128)) ? s.holders[k[r]] : 0u};
          apply_sum<G, C, SRC>(s, k[r], t, d[r], lane, gmask);
        } else if (f[r] & 1) {
          // a piece of a segment cut by a chunk boundary: partial sum, kept
          // in shared memory (a chunk has at most one head and one tail piece)
          float4* dst = (f[r] & 2) ? pt : ph;
#pragma unroll
          for (int c = 0; c < C; ++c) dst[gi * G * C + lane + c * G] = d[r][c];
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        f[r] = fn[r];
#pragma unroll
        for (int c = 0; c < C; ++c) d[r][c] = dn[r][c];
      }
    }
    // Pieces of the span's cut segments are in shared memory, visible to the
    // whole block after the barrier.  A segment that begins in chunk
    // gi and continues is combined here by group gi (its tail piece, then the
    // head pieces of the chunks it covers, in chunk order) and applied when it
    // ends inside the span; one that runs past the span leaves that sum as
    // the span's tail piece, and the rows the span's first segment holds when
    // it continues from the previous span are its head piece (group 0);
    // push_combine adds span pieces up.
    __syncthreads();
    const uint32_t nch = (len + CH - 1) / CH;          // chunks of this span that hold rows
    const uint64_t sidx = P0 / span;
    auto chunk_end = [&](uint32_t m) { return (m + 1) * CH < len ? (m + 1) * CH : len; };
    // last chunk m >= g the segment of key kk covers, given it reaches chunk g;
    // out: it continues past the span
    auto walk = [&](uint32_t g, uint32_t kk, bool& out) {
      while (true) {
        const uint32_t e = chunk_end(g);
        const bool through = sk[e] == kk && sk[1 + e] == kk;   // last row kk, next row kk
        if (!through || g + 1 >= nch) {
          out = through;
          return g;
        }
        ++g;
      }
    };
    if (gi < (int)nch) {
      const uint32_t kl = sk[p1];        // the chunk's last row
      if (kl < s.K && sk[1 + p1] == kl) {
        const bool whole = sk[1 + p0] == kl;
        const bool began = !whole || P0 + p0 == 0 || sk[p0] != kl;
        if (began) {
          bool out = true;
          const uint32_t g1 = (uint32_t)gi + 1 < nch ? walk(gi + 1, kl, out) : (uint32_t)gi;
          float4 tot[C];
#pragma unroll
          for (int c = 0; c < C; ++c) tot[c] = pt[gi * G * C + lane + c * G];
          for (uint32_t m = gi + 1; m <= g1; ++m)
#pragma unroll
            for (int c = 0; c < C; ++c) tot[c] = f4add(tot[c], ph[m * G * C + lane + c * G]);
          if (out) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
              if (col_ok(c)) sp4[(2 * sidx + 1) * D4 + col_of(c)] = tot[c];
            }
          } else {
            take_and_apply<G, C, SRC>(s, a.worker, kl, tot, lane, gmask, any_replica);
          }
        }
      }
    }
    if (gi == 0 && P0 > 0 && sk[1] < s.K && sk[0] == sk[1]) {
      bool out = false;
      const uint32_t g1 = walk(0, sk[1], out);
      float4 tot[C];
#pragma unroll
      for (int c = 0; c < C; ++c) tot[c] = ph[lane + c * G];
      for (uint32_t m = 1; m <= g1; ++m)
#pragma unroll
        for (int c = 0; c < C; ++c) tot[c] = f4add(tot[c], ph[m * G * C + lane + c * G]);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (col_ok(c)) sp4[2 * sidx * D4 + col_of(c)] = tot[c];
      }
    }
  }
  uint32_t unused = 0;
  block_sum2(heads, unused);
  if (threadIdx.x == 0 && heads) {
    atomicAdd(&s.st->last_unique, heads);
    atomicAdd(&s.st->push_unique, (unsigned long long)heads);
  }
}

// Segments that run past a span: the span where one begins owns it; its sum
// is that span's tail piece plus the head pieces of the spans it continues
// into (the spans whose first row holds the key, counted by the block).  The
// groups of the block take those head pieces in strides, in increasing order,
// then group 0 adds the tail piece and the group sums in
// group order: a fixed order, whatever the number of spans.
template <int G, int C>
__global__ void __launch_bounds__(kThreads) push_combine_kernel(Store s, PushArgs a, uint64_t span,
                                                                uint64_t nspans) {
  after_previous();
  const PushWords pw = push_words(s, a);
  bool any_replica = false, resolved = false;
  constexpr int NG = kThreads / G;
  __shared__ float4 part[NG][G * C];
  const int lane = threadIdx.x & (G - 1);
  const int gi = threadIdx.x / G;
  const uint32_t D4 = s.D >> 2;
  const float4* sp4 = reinterpret_cast<const float4*>(a.span_parts);
  const unsigned gmask = group_mask<G>();
  for (uint64_t b = blockIdx.x; b < nspans; b += gridDim.x) {   // block-uniform
    const uint64_t st = b * span;
    const uint64_t en = st + span < a.n ? st + span : a.n;
    // the keys around the span's end and before its start, and the first keys
    // of the spans after it, in one latency
    uint32_t kl, kn, kb, kf;
    auto look = [&]() {
      kl = a.skeys[en - 1];
      kn = en < a.n ? a.skeys[en] : kNoKey;
      kb = st > 0 ? a.skeys[st - 1] : kNoKey;
      kf = b + 1 + threadIdx.x < nspans ? a.skeys[(b + 1 + threadIdx.x) * span] : kNoKey;
    };
    look();
    if (!resolved) {   // (uniform over the grid)
      resolved = true;
      const int from = push_resolve(s, a, pw, any_replica);
      if (from == 0) return;
      if (from == 2) look();
    }
    if (kl >= s.K || kn != kl) continue;
    if (st > 0 && kb == kl) continue;             // it began in an earlier span
    Target target{-1, REP_ALIAS, 0u};
    if (threadIdx.x == 0) target = look_target(s, a.worker, kl, any_replica);
    // the last span whose first row holds kl: the spans after b that do form
    // a prefix (the keys are sorted), so the block tests kThreads of them at
    // once and counts
    uint64_t lo = b;
    for (uint64_t m0 = b + 1; m0 < nspans; m0 += kThreads) {   // block-uniform
      const uint64_t m = m0 + threadIdx.x;
      if (m0 > b + 1) kf = m < nspans ? a.skeys[m * span] : kNoKey;
      const int cnt = __syncthreads_count(m < nspans && kf == kl);
      lo += (uint64_t)cnt;
      if (cnt < kThreads) break;
    }
    float4 acc[C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = f4zero();
    constexpr int UB = 8 / C > 0 ? 8 / C : 1;   // span pieces per group in flight
    for (uint64_t m0 = b + 1 + gi; m0 <= lo; m0 += (uint64_t)NG * UB) {
      float4 t[UB][C];
#pragma unroll
      for (int u = 0; u < UB; ++u)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          const uint64_t m = m0 + (uint64_t)u * NG;
          t[u][c] = (m <= lo && col < D4) ? __ldcg(sp4 + 2 * m * D4 + col) : f4zero();
        }
#pragma unroll
      for (int u = 0; u < UB; ++u)
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = f4add(acc[c], t[u][c]);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) part[gi][lane + c * G] = acc[c];
    __syncthreads();
    if (gi == 0) {
      float4 tot[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t col = lane + c * G;
        tot[c] = col < D4 ? __ldcg(sp4 + (2 * b + 1) * D4 + col) : f4zero();
        for (int g2 = 0; g2 < NG; ++g2) tot[c] = f4add(tot[c], part[g2][lane + c * G]);
      }
      if (lane == 0) mark_target(s, a.worker, kl, target);
      target.slot = __shfl_sync(gmask, target.slot, 0, G);
      target.state = __shfl_sync(gmask, target.state, 0, G);
      target.holders = __shfl_sync(gmask, target.holders, 0, G);
      apply_sum<G, C, kSrcRows>(s, kl, target, tot, lane, gmask);
    }
    __syncthreads();
  }
}

template <int SRC>
void launch_push_source(const Store& s, const PushArgs& a, int sms, cudaStream_t stream) {
  dispatch_push_gc(s.D / 4, SRC == kSrcAda, [&](auto Gc, auto Cc) {
    constexpr int G = decltype(Gc)::value, C = decltype(Cc)::value;
    if constexpr (SRC != kSrcAda || C % 2 == 0) {
      constexpr int R = push_rows_in_flight(C);
      // one block per span: the block scheduler balances spans over the SMs
      const uint64_t span = a.chunk * (kThreads / G);
      const uint64_t spans = (a.n + span - 1) / span;
      note_launches(spans > 1 ? 2 : 1);
      constexpr size_t smem = push_chunks_smem<C, SRC>();
      // the kernel's dynamic shared-memory limit is a per-device attribute
      static bool attr_set[64] = {false};
      int dev = 0;
      cudaGetDevice(&dev);
      if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        cudaFuncSetAttribute(push_chunks_kernel<G, C, R, SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
      }
      launch_after(push_chunks_kernel<G, C, R, SRC>, (unsigned)spans, kThreads, smem, stream, s, a);
      if (spans > 1) {
        const unsigned grid = (unsigned)(spans < (uint64_t)sms * 8 ? spans : (uint64_t)sms * 8);
        launch_after(push_combine_kernel<G, C>, grid, kThreads, 0, stream, s, a, span, spans);
      }
    }
  });
}

}  // namespace
}  // namespace adapm
