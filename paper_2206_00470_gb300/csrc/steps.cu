// Fused training steps of the three sparse workloads (App. C): each reads the
// rows a sample needs straight through the worker's slot map (replica, else
// main copy) and computes loss and gradients in fp32 from those values.  The
// delta row of every row occurrence,
//   AdaGrad rows [theta | a]:  delta = [-lr*g/sqrt(a + g*g + eps) | g*g]
//   (1/sqrt evaluated with the correctly rounded __frsqrt_rn)
//   plain SGD:                 delta = -lr*g
// is written for the push that follows (MF), or formed by it from factors
// written here (ComplEx, SGNS): g is a scalar of the occurrence (coef) times
// one of a few rows (x): a triple's h*r (tails) or its head and relation
// gradients, a centre's vector or its gradient.  So those steps write 4 bytes
// per occurrence and these rows, not the delta rows (per worker: 8192 centres
// of 261 rows x 300 floats: 28 MB instead of 2.5 GB; 4096 triples of 103 rows
// x 512 floats: 14 MB instead of 864 MB), and read no accumulators.
// Losses: MF 1/2 (v - u.w)^2; ComplEx softplus(-y phi), phi = Re(sum h r
// conj(t)) with rows [re | im]; SGNS softplus(-u_o.v_c) + sum softplus(u_n.v_c).
// Every sample's loss is added into a per-block fp64 partial in a fixed order,
// so the batch loss is deterministic.
#include <type_traits>

#include "internal.cuh"
#include "store_launch.cuh"

namespace adapm {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float4 f4zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ float dot4(float4 a, float4 b) {
  return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
}
__device__ __forceinline__ float4 f4fma(float4 a, float s, float4 acc) {
  return make_float4(fmaf(a.x, s, acc.x), fmaf(a.y, s, acc.y), fmaf(a.z, s, acc.z), fmaf(a.w, s, acc.w));
}

__device__ __forceinline__ float softplus_f(float x) { return log1pf(expf(-fabsf(x))) + fmaxf(x, 0.f); }
__device__ __forceinline__ float sigmoid_f(float x) {
  if (x >= 0.f) return 1.f / (1.f + expf(-x));
  const float e = expf(x);
  return e / (1.f + e);
}

// AdaGrad delta of one float of gradient g with accumulator a
__device__ __forceinline__ float ada_theta(float g, float a, float lr, float eps) {
  return -lr * g * __frsqrt_rn(a + g * g + eps);   // correctly rounded 1/sqrt
}
__device__ __forceinline__ float4 ada_theta4(float4 g, float4 a, float lr, float eps) {
  return make_float4(ada_theta(g.x, a.x, lr, eps), ada_theta(g.y, a.y, lr, eps),
                     ada_theta(g.z, a.z, lr, eps), ada_theta(g.w, a.w, lr, eps));
}
__device__ __forceinline__ float4 sq4(float4 g) { return make_float4(g.x * g.x, g.y * g.y, g.z * g.z, g.w * g.w); }
__device__ __forceinline__ float4 f4scale(float4 a, float s) {
  return make_float4(a.x * s, a.y * s, a.z * s, a.w * s);
}

// The derivative of a score's loss: softplus(-x) under label +1, softplus(x)
// under label -1 (softplus_f of the same argument is the loss).
__device__ __forceinline__ float score_coef(float x, bool positive) {
  return positive ? -sigmoid_f(-x) : sigmoid_f(x);
}

// Sums over the warp of U values per lane (U = 1, 2, 4), in 5 + U - 1 shuffles:
// the lanes halve the values they carry before they halve the warp.  The
// caller's lane gets the sum of value summed_row<U>(lane), which lane
// summing_lane<U>(u) has for value u.
template <int U>
__device__ __forceinline__ int summed_row(int lane) {
  return U == 1 ? 0 : (U == 2 ? (lane >> 4) & 1 : ((lane >> 4) & 1) | ((lane >> 2) & 2));
}
template <int U>
__device__ __forceinline__ int summing_lane(int u) {
  return U == 1 ? 0 : (U == 2 ? u << 4 : ((u & 1) << 4) | ((u & 2) << 2));
}
template <int U>
__device__ __forceinline__ float sum_rows(const float (&part)[U], int lane) {
  static_assert(U == 1 || U == 2 || U == 4, "values per lane");
  float v[U];
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = part[u];
  if (U >= 2) {
    const bool hi = lane & 16;
#pragma unroll
    for (int u = 0; u < U / 2; ++u) {
      const float keep = hi ? v[2 * u + 1] : v[2 * u], give = hi ? v[2 * u] : v[2 * u + 1];
      v[u] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, 16);
    }
  }
  if (U == 4) {
    const bool hi = lane & 8;
    const float keep = hi ? v[1 % U] : v[0], give = hi ? v[0] : v[1 % U];
    v[0] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, 8);
  }
#pragma unroll
  for (int o = U == 4 ? 4 : (U == 2 ? 8 : 16); o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
  return v[0];
}

template <int G>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Where a worker's value of a key is read (see the replica states): the row, and the
// pending row to add to it when one push is pending on an alias (few have
// one at a step: a null pointer otherwise).
struct Row {
  const float4* p;
  const float4* add;
};
__device__ __forceinline__ Row row_of(const Store& s, int32_t e, uint32_t k) {
  Row r;
  r.p = row_source(s, e, k, &r.add);
  return r;
}

__device__ __forceinline__ float4 f4add(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// Fixed-order block reduction of one double per thread into
// o.loss_part[blockIdx.x]; with o.loss_out the last block to finish then
// sums the partials (thread t the partials t, t + 256, ... in order, then a
// fixed tree) into *o.loss_out and clears the block counter.
__device__ void block_loss(double v, const StepOut& o) {
  __shared__ double sm[kThreads / 32];
  __shared__ double tree[kThreads];
  __shared__ int last;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, off);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int i = 0; i < kThreads / 32; ++i) t += sm[i];
    o.loss_part[blockIdx.x] = t;
    last = 0;
    if (o.loss_out) {
      __threadfence();
      last = atomicAdd(o.loss_done, 1u) == gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += kThreads) t += __ldcg(o.loss_part + i);
  tree[threadIdx.x] = t;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) tree[threadIdx.x] += tree[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *o.loss_out = tree[0];
    *o.loss_done = 0u;
  }
}

// ---------------------------------------------------------------------------
// matrix factorisation: one cell per group of G lanes
// ---------------------------------------------------------------------------
// The delta rows are written here, unlike the other steps': a batch's rows
// stay in L2 until the push, and a cell's two rows share nothing that would be
// read once for many.  (Formed in the push from theta and accumulator halves:
// step 395 -> 286 us, push 383 -> 536 us per clock of 8 x 65,536 cells of rank
// 100.)  One cell per group: two in flight take the registers of a third of
// the resident warps (step 395 -> 587 us).
template <int G, int C>
__global__ void __launch_bounds__(kThreads)
mf_step_kernel(Store s, uint32_t w, const uint32_t* rows, const uint32_t* cols,
               const float* vals, uint64_t n, uint32_t dim, int adagrad, float lr, float eps,
               StepOut o) {
  after_previous();
  const int lane = threadIdx.x & (G - 1);
  constexpr int GPW = 32 / G;
  const int gi = (threadIdx.x & 31) / G;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t dim4 = dim >> 2, D4 = s.D >> 2;
  const int32_t* mapw = s.map + (uint64_t)w * s.K;
  s.par = s.st->par;
  float4* d4 = reinterpret_cast<float4*>(o.x);
  double lsum = 0.0;
  // software-pipelined: a round loads the rows of its cell, the slots of the
  // next round's cell and the keys of the cell after
  const uint64_t step = nwarps * GPW;
  auto cell_keys = [&](uint64_t i, uint32_t& ku, uint32_t& kw) -> bool {   // both in range
    ku = 0;
    kw = 0;
    if (i >= n) return false;
    ku = rows[i];
    kw = cols[i];
    return ku < s.K && kw < s.K;
  };
  uint32_t ku0, kw0, ku1, kw1;
  bool ok0 = cell_keys(warp * GPW + gi, ku0, kw0);
  bool ok1 = cell_keys(warp * GPW + gi + step, ku1, kw1);
  int32_t su0 = ok0 ? mapw[ku0] : -1, sw0 = ok0 ? mapw[kw0] : -1;
  for (uint64_t b = warp * GPW; b < n; b += step) {
    const uint64_t i = b + gi;
    const bool in = i < n;
    const uint32_t ku = ku0, kw = kw0;
    const bool ok = ok0;
    if (in && !ok && lane == 0) set_error(s.st, ERR_KEY_RANGE);
    float4 tu[C], tw[C], au[C], aw[C];
    {
      const Row ru = row_of(s, su0, ku), rw = row_of(s, sw0, kw);
      const float4 *pu = ru.p, *pw = rw.p;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t col = lane + c * G;
        const bool cv = ok && col < dim4;
        tu[c] = cv ? pu[col] : f4zero();
        tw[c] = cv ? pw[col] : f4zero();
        au[c] = (cv && adagrad) ? pu[dim4 + col] : f4zero();
        aw[c] = (cv && adagrad) ? pw[dim4 + col] : f4zero();
      }
      // the next cell's slots and the keys of the cell after, issued before
      // this cell's rows are used
      su0 = ok1 ? mapw[ku1] : -1;
      sw0 = ok1 ? mapw[kw1] : -1;
      ku0 = ku1;
      kw0 = kw1;
      ok0 = ok1;
      ok1 = cell_keys(i + 2 * step, ku1, kw1);
      if (ru.add || rw.add) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + c * G;
          if (!ok || col >= dim4) continue;
          if (ru.add) tu[c] = f4add(tu[c], ru.add[col]);
          if (rw.add) tw[c] = f4add(tw[c], rw.add[col]);
          if (ru.add && adagrad) au[c] = f4add(au[c], ru.add[dim4 + col]);
          if (rw.add && adagrad) aw[c] = f4add(aw[c], rw.add[dim4 + col]);
        }
      }
    }
    float part = 0.f;
#pragma unroll
    for (int c = 0; c < C; ++c) part += dot4(tu[c], tw[c]);
    const float dot = group_sum<G>(part);
    if (!in) continue;
    if (!ok) {
      if (lane == 0) {
        o.dkeys[i] = kNoKey;
        o.dkeys[n + i] = kNoKey;
      }
      continue;
    }
    const float e = vals[i] - dot;
    if (lane == 0) lsum += 0.5 * (double)e * (double)e;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = lane + c * G;
      if (col < dim4) {
        const float4 gu = f4scale(tw[c], -e);
        const float4 gw = f4scale(tu[c], -e);
        if (adagrad) {
          d4[i * D4 + col] = ada_theta4(gu, au[c], lr, eps);
          d4[i * D4 + dim4 + col] = sq4(gu);
          d4[(n + i) * D4 + col] = ada_theta4(gw, aw[c], lr, eps);
          d4[(n + i) * D4 + dim4 + col] = sq4(gw);
        } else {
          d4[i * D4 + col] = f4scale(gu, -lr);
          d4[(n + i) * D4 + col] = f4scale(gw, -lr);
        }
      }
    }
    if (lane == 0) {
      o.dkeys[i] = ku;
      o.dkeys[n + i] = kw;
    }
  }
  block_loss(lsum, o);
}

// Rows of a sample (tails of a triple, context and negative rows of a centre)
// are taken in batches of 32: lane t looks up row t of the batch (key, map
// entry, where its value is) while the batches before it are being read, up
// to the next sample's first ones, and writes its key and scalar.  The warp
// reads the rows in order, each lane its columns, by 16-byte asynchronous
// copies into a ring of DEPTH rows in shared memory, U rows consumed at a
// time: a lane reads back only what it copied itself, so the ring needs no
// barrier, and the rows in flight take no registers.  (Loaded into registers,
// U rows at a time with two blocks per SM, the SGNS step spent most of its
// issue slots waiting for the next U.)
struct RowBits {   // a Row, passed between lanes; 0: the row is skipped
  unsigned long long p, add;
};
__device__ __forceinline__ RowBits row_bits(const Store& s, int32_t e, uint32_t k) {
  if (k == kNoKey) return RowBits{0ull, 0ull};
  const Row r = row_of(s, e, k);
  return RowBits{reinterpret_cast<unsigned long long>(r.p), reinterpret_cast<unsigned long long>(r.add)};
}

__device__ __forceinline__ void copy_async16(float4* dst, const float4* src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {   // all but the last N groups have landed
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// ComplEx: one triple per warp; lane q holds float4 q of the re and im halves
// ---------------------------------------------------------------------------
template <int CC, int U, int DEPTH>
__global__ void __launch_bounds__(kThreads, 2)
complex_step_kernel(Store s, uint32_t w, const uint32_t* heads, const uint32_t* rels,
                    const uint32_t* tails, const uint32_t* negs, uint64_t n,
                    uint32_t n_neg, uint32_t dim, StepOut o) {
  after_previous();
  static_assert(16 % U == 0 && DEPTH <= 16 && U <= DEPTH, "see the batches' second half");
  extern __shared__ float4 ring_all[];
  const int lane = threadIdx.x & 31;
  float4* const ring = ring_all + (threadIdx.x >> 5) * (DEPTH * 2 * CC * 32) + lane;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t h4 = dim >> 3;          // float4 per half (re or im) of theta
  const uint32_t T4 = 2 * h4;            // float4 of a theta row
  const int32_t* mapw = s.map + (uint64_t)w * s.K;
  s.par = s.st->par;
  float4* x4 = reinterpret_cast<float4*>(o.x);   // head gradients, relation gradients, h*r, n rows each
  // row occurrences in the order the keys of a batch are listed: all heads,
  // all relations, all true tails, then the negatives triple by triple
  const uint64_t rrel = n, rt = 2 * n, rneg = 3 * n;
  // tails: j = 0 is the true tail (label +1), j >= 1 the negatives (label -1)
  const uint32_t J = 1 + n_neg;
  double lsum = 0.0;
  auto tail_key = [&](uint64_t i, uint32_t j) -> uint32_t {   // kNoKey: no such row, or skipped
    if (i >= n || j >= J) return kNoKey;
    const uint32_t k = j == 0 ? tails[i] : negs[i * n_neg + (j - 1)];
    if (k >= s.K) {
      set_error(s.st, ERR_KEY_RANGE);
      return kNoKey;
    }
    return k;
  };
  auto entry = [&](uint32_t k) -> int32_t { return k != kNoKey ? mapw[k] : -1; };
  // this batch's rows, and the next batch's keys
  uint32_t key = 0, k1 = 0;
  RowBits cur{0ull, 0ull};
  auto restart = [&](uint64_t i) {
    key = tail_key(i, lane);
    k1 = J > 32 ? tail_key(i, 32 + lane) : tail_key(i + nwarps, lane);
    cur = row_bits(s, entry(key), key);
  };
  for (int t = 0; t < DEPTH * 2 * CC; ++t) ring[t * 32] = f4zero();   // (columns no copy writes stay zero)
  restart(warp);
  for (uint64_t i = warp; i < n; i += nwarps) {
    const uint32_t kh = heads[i], kr = rels[i], kt = tails[i];
    if (kh >= s.K || kr >= s.K || kt >= s.K) {
      if (lane == 0) set_error(s.st, ERR_KEY_RANGE);
      if (lane < 3) o.dkeys[(uint64_t)lane * n + i] = kNoKey;
      for (uint64_t q = lane; q < n_neg; q += 32) o.dkeys[rneg + i * n_neg + q] = kNoKey;
      restart(i + nwarps);
      continue;
    }
    RowBits nxt{0ull, 0ull};
    uint32_t islot = 0, cslot = 0;   // ring slots of the next row copied, consumed
    auto issue = [&](uint32_t r, uint32_t j0) {   // row r of the triple (in the batch at j0 or the next)
      const float4* pt = reinterpret_cast<const float4*>(
          r < j0 + 32 ? __shfl_sync(0xFFFFFFFFu, cur.p, r & 31) : __shfl_sync(0xFFFFFFFFu, nxt.p, r & 31));
      if (r < J && pt != nullptr) {
#pragma unroll
        for (int c = 0; c < CC; ++c) {
          const uint32_t q = lane + 32 * c;
          if (q < h4) {
            copy_async16(ring + (islot * 2 * CC + 2 * c) * 32, pt + q);
            copy_async16(ring + (islot * 2 * CC + 2 * c + 1) * 32, pt + h4 + q);
          }
        }
      }
      copy_commit();
      islot = islot + 1 == DEPTH ? 0 : islot + 1;
    };
#pragma unroll
    for (int r = 0; r < DEPTH; ++r) issue(r, 0);
    const Row ph = row_of(s, mapw[kh], kh);
    const Row pr = row_of(s, mapw[kr], kr);
    // float4 q of half p (0 re, 1 im) of a theta row
    auto part4 = [&](const Row& row, uint32_t p, uint32_t q) {
      float4 v = q < h4 ? row.p[p * h4 + q] : f4zero();
      if (row.add && q < h4) v = f4add(v, row.add[p * h4 + q]);
      return v;
    };
    float4 xre[CC], xim[CC], Tre[CC], Tim[CC];
#pragma unroll
    for (int c = 0; c < CC; ++c) {
      const uint32_t q = lane + 32 * c;
      const float4 hre = part4(ph, 0, q), him = part4(ph, 1, q), rre = part4(pr, 0, q), rim = part4(pr, 1, q);
      // complex product h*r: d phi / d t
      xre[c] = make_float4(hre.x * rre.x - him.x * rim.x, hre.y * rre.y - him.y * rim.y,
                           hre.z * rre.z - him.z * rim.z, hre.w * rre.w - him.w * rim.w);
      xim[c] = make_float4(hre.x * rim.x + him.x * rre.x, hre.y * rim.y + him.y * rre.y,
                           hre.z * rim.z + him.z * rre.z, hre.w * rim.w + him.w * rre.w);
      Tre[c] = f4zero();
      Tim[c] = f4zero();
      if (q < h4) {
        x4[(rt + i) * T4 + q] = xre[c];
        x4[(rt + i) * T4 + h4 + q] = xim[c];
      }
    }
    for (uint32_t j0 = 0; j0 < J; j0 += 32) {
      const bool any_add = __any_sync(0xFFFFFFFFu, cur.add != 0ull);
      // the next batch's map entries and the keys of the one after
      const int32_t e1 = entry(k1);
      const uint32_t k2 = j0 + 64 < J ? tail_key(i, j0 + 64 + lane)
                          : j0 + 32 < J ? tail_key(i + nwarps, lane)
                          : J > 32 ? tail_key(i + nwarps, 32 + lane) : tail_key(i + 2 * nwarps, lane);
      const unsigned there = __ballot_sync(0xFFFFFFFFu, cur.p != 0ull);   // rows of the batch that are not skipped
      float mycoef = 0.f, myphi = 0.f;
      const uint32_t cnt = J - j0 < 32 ? J - j0 : 32;
#pragma unroll 1
      for (uint32_t u0 = 0; u0 < cnt; u0 += U) {
        if (u0 == 16) nxt = row_bits(s, e1, k1);
        copy_wait<DEPTH - U>();
        float4 tre[U][CC], tim[U][CC];
        float part[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool v = (there >> (u0 + u)) & 1u;   // (uniform; no bit at or above cnt is set)
#pragma unroll
          for (int c = 0; c < CC; ++c) {
            tre[u][c] = f4zero();
            tim[u][c] = f4zero();
            if (v) {
              tre[u][c] = ring[(cslot * 2 * CC + 2 * c) * 32];
              tim[u][c] = ring[(cslot * 2 * CC + 2 * c + 1) * 32];
            }
          }
          cslot = cslot + 1 == DEPTH ? 0 : cslot + 1;
        }
        if (any_add) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const float4* pa = reinterpret_cast<const float4*>(__shfl_sync(0xFFFFFFFFu, cur.add, (u0 + u) & 31));
            if (pa == nullptr || u0 + u >= cnt) continue;
#pragma unroll
            for (int c = 0; c < CC; ++c) {
              const uint32_t q = lane + 32 * c;
              if (q >= h4) continue;
              tre[u][c] = f4add(tre[u][c], pa[q]);
              tim[u][c] = f4add(tim[u][c], pa[h4 + q]);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          part[u] = 0.f;
#pragma unroll
          for (int c = 0; c < CC; ++c) part[u] += dot4(xre[c], tre[u][c]) + dot4(xim[c], tim[u][c]);
        }
        const float phi = sum_rows<U>(part, lane);
        // (the ring slots just read are free)
#pragma unroll
        for (int u = 0; u < U; ++u) issue(j0 + u0 + DEPTH + u, j0);
        // every lane evaluates the derivative of the row it has the score of;
        // lane u0 + u keeps row u's
        const uint32_t ru = u0 + summed_row<U>(lane);
        const float dphi = (there >> ru) & 1u ? score_coef(phi, j0 + ru == 0u) : 0.f;
        const int from = summing_lane<U>((lane - (int)u0) & (U - 1));
        const float s_phi = __shfl_sync(0xFFFFFFFFu, phi, from), s_coef = __shfl_sync(0xFFFFFFFFu, dphi, from);
        if ((uint32_t)lane - u0 < (uint32_t)U) {
          myphi = s_phi;
          mycoef = s_coef;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float coef = __shfl_sync(0xFFFFFFFFu, dphi, summing_lane<U>(u));   // (0 for a skipped row)
#pragma unroll
          for (int c = 0; c < CC; ++c) {
            Tre[c] = f4fma(tre[u][c], coef, Tre[c]);
            Tim[c] = f4fma(tim[u][c], coef, Tim[c]);
          }
        }
      }
      if ((there >> lane) & 1u) lsum += (double)softplus_f(j0 + lane == 0 ? -myphi : myphi);
      if ((uint32_t)lane < cnt) {
        const uint64_t row = j0 + lane == 0 ? rt + i : rneg + i * n_neg + (j0 + lane - 1);
        o.dkeys[row] = key;
        o.coef[row] = mycoef;
      }
      if (cnt <= 16) nxt = row_bits(s, e1, k1);
      cur = nxt;
      key = k1;
      k1 = k2;
    }
    // head and relation: gradients are linear in T = sum_j coef_j t_j (their
    // rows are read again, from the caches, rather than held through the tails)
#pragma unroll
    for (int c = 0; c < CC; ++c) {
      const uint32_t q = lane + 32 * c;
      if (q >= h4) continue;
      const float4 hre = part4(ph, 0, q), him = part4(ph, 1, q), rre = part4(pr, 0, q), rim = part4(pr, 1, q);
      x4[i * T4 + q] = make_float4(rre.x * Tre[c].x + rim.x * Tim[c].x, rre.y * Tre[c].y + rim.y * Tim[c].y,
                                   rre.z * Tre[c].z + rim.z * Tim[c].z, rre.w * Tre[c].w + rim.w * Tim[c].w);
      x4[i * T4 + h4 + q] = make_float4(rre.x * Tim[c].x - rim.x * Tre[c].x, rre.y * Tim[c].y - rim.y * Tre[c].y,
                                        rre.z * Tim[c].z - rim.z * Tre[c].z, rre.w * Tim[c].w - rim.w * Tre[c].w);
      x4[(rrel + i) * T4 + q] = make_float4(hre.x * Tre[c].x + him.x * Tim[c].x, hre.y * Tre[c].y + him.y * Tim[c].y,
                                            hre.z * Tre[c].z + him.z * Tim[c].z, hre.w * Tre[c].w + him.w * Tim[c].w);
      x4[(rrel + i) * T4 + h4 + q] =
          make_float4(hre.x * Tim[c].x - him.x * Tre[c].x, hre.y * Tim[c].y - him.y * Tre[c].y,
                      hre.z * Tim[c].z - him.z * Tre[c].z, hre.w * Tim[c].w - him.w * Tre[c].w);
    }
    if (lane < 2) {
      o.dkeys[(uint64_t)lane * n + i] = lane == 0 ? kh : kr;
      o.coef[(uint64_t)lane * n + i] = 1.f;
    }
  }
  block_loss(lsum, o);
}

// ---------------------------------------------------------------------------
// skip-gram with negative sampling: one centre per warp
// rows per centre: [centre | for each context slot: positive, negatives...]
// ---------------------------------------------------------------------------
template <int C, int U, int DEPTH>
__global__ void __launch_bounds__(kThreads, 2)
sgns_step_kernel(Store s, uint32_t w, const uint32_t* centres, const uint32_t* contexts,
                 const uint32_t* negs, uint64_t n, uint32_t n_ctx, uint32_t n_neg, uint32_t vocab,
                 float lr, StepOut o) {
  after_previous();
  static_assert(16 % U == 0 && DEPTH <= 16 && U <= DEPTH, "see the batches' second half");
  extern __shared__ float4 ring_all[];
  const int lane = threadIdx.x & 31;
  float4* const ring = ring_all + (threadIdx.x >> 5) * (DEPTH * C * 32) + lane;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t D4 = s.D >> 2;
  const int32_t* mapw = s.map + (uint64_t)w * s.K;
  s.par = s.st->par;
  float4* x4 = reinterpret_cast<float4*>(o.x);   // the centres' vectors, then their gradients
  const uint64_t per = 1 + (uint64_t)n_ctx * (1 + n_neg);
  // a centre's rows in one index space t = j * (1 + n_neg) + q (q = 0: the
  // context word, q >= 1: its negatives)
  const uint32_t per_ctx = 1 + n_neg;
  const uint32_t T = n_ctx * per_ctx;
  double lsum = 0.0;
  auto token = [&](uint64_t i, uint32_t t) -> uint32_t {   // the row's key; kNoKey: no such row, or skipped
    if (i >= n || t >= T) return kNoKey;
    const uint32_t j = t / per_ctx, q = t - j * per_ctx;
    const uint32_t oc = contexts[i * n_ctx + j];
    if (oc == kNoKey) return kNoKey;
    if (oc >= vocab) {
      if (q == 0) set_error(s.st, ERR_KEY_RANGE);
      return kNoKey;
    }
    const uint32_t tok = q == 0 ? oc : negs[(i * n_ctx + j) * n_neg + (q - 1)];
    if (tok >= vocab) {
      set_error(s.st, ERR_KEY_RANGE);
      return kNoKey;
    }
    return vocab + tok;
  };
  auto entry = [&](uint32_t k) -> int32_t { return k != kNoKey ? mapw[k] : -1; };
  // this batch's rows, and the next batch's keys
  uint32_t key = 0, k1 = 0;
  RowBits cur{0ull, 0ull};
  auto restart = [&](uint64_t i) {
    key = token(i, lane);
    k1 = T > 32 ? token(i, 32 + lane) : token(i + nwarps, lane);
    cur = row_bits(s, entry(key), key);
  };
  for (int t = 0; t < DEPTH * C; ++t) ring[t * 32] = f4zero();   // (columns no copy writes stay zero)
  restart(warp);
  for (uint64_t i = warp; i < n; i += nwarps) {
    const uint64_t base = i * per;
    const uint32_t kc = centres[i];
    if (kc >= vocab) {
      if (lane == 0) set_error(s.st, ERR_KEY_RANGE);
      for (uint64_t q = lane; q < per; q += 32) o.dkeys[base + q] = kNoKey;
      restart(i + nwarps);
      continue;
    }
    RowBits nxt{0ull, 0ull};
    uint32_t islot = 0, cslot = 0;   // ring slots of the next row copied, consumed
    auto issue = [&](uint32_t r, uint32_t t0) {   // row r of the centre (in the batch at t0 or the next)
      const float4* px = reinterpret_cast<const float4*>(
          r < t0 + 32 ? __shfl_sync(0xFFFFFFFFu, cur.p, r & 31) : __shfl_sync(0xFFFFFFFFu, nxt.p, r & 31));
      if (r < T && px != nullptr) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t col = lane + 32 * c;
          if (col < D4) copy_async16(ring + (islot * C + c) * 32, px + col);
        }
      }
      copy_commit();
      islot = islot + 1 == DEPTH ? 0 : islot + 1;
    };
#pragma unroll
    for (int r = 0; r < DEPTH; ++r) issue(r, 0);
    const Row pv = row_of(s, mapw[kc], kc);
    float4 v[C], gv[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = lane + 32 * c;
      v[c] = col < D4 ? pv.p[col] : f4zero();
      if (pv.add && col < D4) v[c] = f4add(v[c], pv.add[col]);
      gv[c] = f4zero();
      if (col < D4) x4[i * D4 + col] = v[c];
    }
    for (uint32_t t0 = 0; t0 < T; t0 += 32) {
      const bool any_add = __any_sync(0xFFFFFFFFu, cur.add != 0ull);
      // the next batch's map entries and the keys of the one after
      const int32_t e1 = entry(k1);
      const uint32_t k2 = t0 + 64 < T ? token(i, t0 + 64 + lane)
                          : t0 + 32 < T ? token(i + nwarps, lane)
                          : T > 32 ? token(i + nwarps, 32 + lane) : token(i + 2 * nwarps, lane);
      const bool positive = (t0 + lane) % per_ctx == 0;
      const unsigned pos = __ballot_sync(0xFFFFFFFFu, positive);
      const unsigned there = __ballot_sync(0xFFFFFFFFu, cur.p != 0ull);   // rows of the batch that are not skipped
      float mycoef = 0.f, mysc = 0.f;
      const uint32_t cnt = T - t0 < 32 ? T - t0 : 32;
#pragma unroll 1
      for (uint32_t u0 = 0; u0 < cnt; u0 += U) {
        if (u0 == 16) nxt = row_bits(s, e1, k1);
        copy_wait<DEPTH - U>();
        float4 x[U][C];
        float part[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool vx = (there >> (u0 + u)) & 1u;   // (uniform; no bit at or above cnt is set)
#pragma unroll
          for (int c = 0; c < C; ++c) {
            x[u][c] = f4zero();
            if (vx) x[u][c] = ring[(cslot * C + c) * 32];
          }
          cslot = cslot + 1 == DEPTH ? 0 : cslot + 1;
        }
        if (any_add) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const float4* pa = reinterpret_cast<const float4*>(__shfl_sync(0xFFFFFFFFu, cur.add, (u0 + u) & 31));
            if (pa == nullptr || u0 + u >= cnt) continue;
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const uint32_t col = lane + 32 * c;
              if (col < D4) x[u][c] = f4add(x[u][c], pa[col]);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          part[u] = 0.f;
#pragma unroll
          for (int c = 0; c < C; ++c) part[u] += dot4(x[u][c], v[c]);
        }
        const float sc = sum_rows<U>(part, lane);
        // (the ring slots just read are free)
#pragma unroll
        for (int u = 0; u < U; ++u) issue(t0 + u0 + DEPTH + u, t0);
        // every lane evaluates the derivative of the row it has the score of;
        // lane u0 + u keeps row u's
        const uint32_t ru = u0 + summed_row<U>(lane);
        const float dsc = (there >> ru) & 1u ? score_coef(sc, (pos >> ru) & 1u) : 0.f;
        const int from = summing_lane<U>((lane - (int)u0) & (U - 1));
        const float s_sc = __shfl_sync(0xFFFFFFFFu, sc, from), s_coef = __shfl_sync(0xFFFFFFFFu, dsc, from);
        if ((uint32_t)lane - u0 < (uint32_t)U) {
          mysc = s_sc;
          mycoef = s_coef;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float coef = __shfl_sync(0xFFFFFFFFu, dsc, summing_lane<U>(u));   // (0 for a skipped row)
#pragma unroll
          for (int c = 0; c < C; ++c) gv[c] = f4fma(x[u][c], coef, gv[c]);
        }
      }
      if ((there >> lane) & 1u) lsum += (double)softplus_f(positive ? -mysc : mysc);
      if ((uint32_t)lane < cnt) {
        o.dkeys[base + 1 + t0 + lane] = key;
        o.coef[base + 1 + t0 + lane] = -lr * mycoef;
      }
      if (cnt <= 16) nxt = row_bits(s, e1, k1);
      cur = nxt;
      key = k1;
      k1 = k2;
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const uint32_t col = lane + 32 * c;
      if (col < D4) x4[(n + i) * D4 + col] = gv[c];
    }
    if (lane == 0) {
      o.dkeys[base] = kc;
      o.coef[base] = -lr;
    }
    if (T == 0) restart(i + nwarps);   // (no batch moved the lookups on)
  }
  block_loss(lsum, o);
}

// The ring's dynamic shared memory per block; a kernel's limit is a
// per-device attribute, set once.
template <typename Kernel>
void allow_smem(Kernel kernel, size_t bytes, bool (&set)[64]) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && set[dev]) return;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (dev >= 0 && dev < 64) set[dev] = true;
}

}  // namespace

unsigned step_loss_blocks(int sms) { return (unsigned)sms * 4; }

void launch_mf_step(const Store& s, uint32_t w, const uint32_t* rows, const uint32_t* cols,
                    const float* vals, uint64_t n, uint32_t dim, bool adagrad, float lr, float eps,
                    const StepOut& o, int sms, cudaStream_t stream) {
  const unsigned grid = o.loss_blocks;
  note_launches(1);
  const uint32_t dim4 = dim / 4;
  const int a = adagrad ? 1 : 0;
  auto run = [&](auto kernel) {
    launch_after(kernel, grid, kThreads, 0, stream, s, w, rows, cols, vals, n, dim, a, lr, eps, o);
  };
  if (dim4 <= 4) run(mf_step_kernel<4, 1>);
  else if (dim4 <= 8) run(mf_step_kernel<8, 1>);
  else if (dim4 <= 16) run(mf_step_kernel<16, 1>);
  else if (dim4 <= 32) run(mf_step_kernel<32, 1>);
  else if (dim4 <= 64) run(mf_step_kernel<32, 2>);
  else if (dim4 <= 128) run(mf_step_kernel<32, 4>);
  else run(mf_step_kernel<32, 8>);
}

void launch_complex_step(const Store& s, uint32_t w, const uint32_t* heads, const uint32_t* rels,
                         const uint32_t* tails, const uint32_t* negs, uint64_t n, uint32_t n_neg,
                         uint32_t dim, const StepOut& o, int sms, cudaStream_t stream) {
  const unsigned grid = o.loss_blocks;
  note_launches(1);
  const uint32_t h4 = dim / 8;
  auto run = [&](auto CCc, auto Uc, auto Dc) {
    constexpr int CC = decltype(CCc)::value, U = decltype(Uc)::value, DEPTH = decltype(Dc)::value;
    constexpr size_t smem = (size_t)kThreads * DEPTH * 2 * CC * sizeof(float4);
    static bool set[64] = {false};
    allow_smem(complex_step_kernel<CC, U, DEPTH>, smem, set);
    launch_after(complex_step_kernel<CC, U, DEPTH>, grid, kThreads, smem, stream, s, w, heads, rels, tails, negs, n,
                 n_neg, dim, o);
  };
  // ring depths: as many rows as two blocks' rings hold per SM (96 KB each)
  if (h4 <= 32) run(std::integral_constant<int, 1>{}, std::integral_constant<int, 4>{}, std::integral_constant<int, 12>{});
  else run(std::integral_constant<int, 2>{}, std::integral_constant<int, 2>{}, std::integral_constant<int, 6>{});
}

void launch_sgns_step(const Store& s, uint32_t w, const uint32_t* centres, const uint32_t* contexts,
                      const uint32_t* negs, uint64_t n, uint32_t n_ctx, uint32_t n_neg,
                      uint32_t vocab, uint32_t dim, float lr, const StepOut& o, int sms,
                      cudaStream_t stream) {
  const unsigned grid = o.loss_blocks;
  note_launches(1);
  const uint32_t D4 = dim / 4;
  auto run = [&](auto Cc, auto Uc, auto Dc) {
    constexpr int C = decltype(Cc)::value, U = decltype(Uc)::value, DEPTH = decltype(Dc)::value;
    constexpr size_t smem = (size_t)kThreads * DEPTH * C * sizeof(float4);
    static bool set[64] = {false};
    allow_smem(sgns_step_kernel<C, U, DEPTH>, smem, set);
    launch_after(sgns_step_kernel<C, U, DEPTH>, grid, kThreads, smem, stream, s, w, centres, contexts, negs, n, n_ctx,
                 n_neg, vocab, lr, o);
  };
  // ring depths: as many rows as two blocks' rings hold per SM (96 KB each), 16 at most
  if (D4 <= 32) run(std::integral_constant<int, 1>{}, std::integral_constant<int, 4>{}, std::integral_constant<int, 16>{});
  else if (D4 <= 64) run(std::integral_constant<int, 2>{}, std::integral_constant<int, 4>{}, std::integral_constant<int, 12>{});
  else if (D4 <= 96) run(std::integral_constant<int, 3>{}, std::integral_constant<int, 4>{}, std::integral_constant<int, 8>{});
  else run(std::integral_constant<int, 8>{}, std::integral_constant<int, 1>{}, std::integral_constant<int, 3>{});
}

}  // namespace adapm
