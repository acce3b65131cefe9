// Fused four-step inverse transforms of many rows (the basis filter a2 + a3, the template method and the
// folded first stage) for block lengths 2^14..2^20, one persistent launch per call.
//
// With j = j1 + n1 j2 and m = m2 + n2 m1, part A transforms the columns j1 (length n2, over j2), applies
// w_n^(j1 m2) and writes X[row][j1][m2]; part B transforms the columns m2 (length n1, over j1) and keeps the
// valid half m1 >= n1 / 2. X is a ring of a few rows that stays in L2: parts of both kinds are dealt out
// from one ticket counter in an order in which part B of a row follows part A of the row a few rows later,
// so that no launch boundary separates the two and every SM works on a mix of both.
//
// A work item is TP = 2048 WARPS points: CA (CB) whole columns of one row. A CTA's loop: the item's tile was requested with cp.async while the item before was computed; it goes from shared memory into
// registers and through a first stage of radix 32 (a thread holds 32 points of two columns, pair.cuh), the
// results are exchanged through the same shared memory, the next item's tile is requested into it, and the
// second stage of radix L / 32 follows. In part A a warp owns its columns, so its exchange needs no block
// barrier and its results leave as runs of L / 4 contiguous bytes; in part B the lanes span the columns,
// which makes the loads, the stores of beta and the bin sums contiguous.
//
// What bounds it, and what was measured (n = 2^19, 201 rows, w = 8): 520 us against 892 us for two radix-32 launches
// per chunk of 8 rows, which it replaces (132 us are the rows' HBM bytes). The launches lost 512 work items to
// 456 resident CTAs, a gap and a ramp each. Three CTAs of 128 threads fit an SM (168 registers, 74 KB); the issue
// slots are busy 30 % of the time and the long straight-line code of an item (about 2000 instructions a warp) is what
// they wait for: of 3.15 us a row the loads were 0.4 us and the butterflies 0.7 us. Running three items of an SM in
// step, so that they fetch it together, brought the fetch stalls from 2.9 to 0.4 cycles per instruction and as much
// waiting for each other's shared-memory and FP32 phases (3.27 us); two CTAs with 255 registers and a separate
// exchange buffer: 3.2 us; L2 residency hints on X: no change; fewer instructions (no spare cases): 2.75 us, and with
// short copy loops and exchange addresses 2.69 us, without the twiddles' row of ones in shared memory 2.58 us (and at 2^20,
// where that row left room for two CTAs an SM only, 6.63 -> 6.00 us a row).
//
// Order and dependencies. Tickets are taken in increasing order by CTAs that are running, a CTA never
// waits while it holds results that it has not announced, and an item depends on items of lower tickets
// only: the lowest unfinished ticket can always finish, whatever else runs on the GPU. Waits are bounded
// all the same (RB_FLAG_TIMEOUT); a basis filter whose launch gave up fills beta and the bin means with NaN, as not
// every caller of it reads the flag.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "internal.h"
#include "pair.cuh"

namespace rbseries {

using namespace rbpair;

constexpr uint64_t kWaitNs = 2000000000ull;  // a wait for another item gives up after 2 s

// What the rows are and what becomes of the transforms: basis vectors (beta and bin means), templates
// (arg-max of every window against a threshold), or complete folded spectra (every sample against a threshold).
enum { KIND_BANK = 0, KIND_PLAIN = 1, KIND_FOLD = 2 };

// Synchronisation words (unsigned) in the workspace, zero between launches: ticket counter, CTAs done, abort,
// one unused, then per ring slot the finished A items and the finished B items.
constexpr int kSyncHead = 4;

struct Args {
  const float2* rows;  // [nvec][n/2] one-sided spectra (KIND_FOLD: [nvec][n] complete spectra)
  const float2* shat;  // [n/2] (unused by KIND_FOLD)
  float2* X;           // [ring][n1][n2]
  const float2* w2a;   // [32][n2/32 + 1]: exp(2 pi i j r / n2)
  const float2* w4;    // [n1/4]: exp(2 pi i 128 e / n), then [128]: exp(2 pi i e / n)
  unsigned* sync;
  unsigned* flags;
  int nvec, lag, log2ring;
  int64_t vec0;  // number of row 0 (outputs and template numbers count from it)
  int w, log2w;
  float2* beta;
  float2* beta_avg;
  rb_trigger* trig;
  rb_candidate* cand;
  unsigned long long* counter;
  int64_t cap;
  float thr2;
  int64_t sample_offset;
  int block_id;
  int align_rows;  // rows and shat lie on 16-byte boundaries (else on 8-byte ones)
  int align_beta;
  unsigned withhold;  // failure-detection test: part B waits for one count more than there is (rbx_series_withhold)
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_relaxed(unsigned* p) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ uint64_t timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

template <int LOG2N, int WARPS>
struct Shape {
  static constexpr int P = LOG2N;
  static constexpr int N1 = 1 << (P / 2), N2 = 1 << (P - P / 2);
  static constexpr int NT = 32 * WARPS, TP = 64 * NT;  // threads, points of an item
  static constexpr int CA = TP / N2, CB = TP / N1;     // columns of an item
  static constexpr int ITEMS = (1 << P) / TP;          // items per row and part
  static constexpr int SA = N2 / 32, SB = N1 / 32;     // threads per column pair = radix of the second stage
  static_assert(SA >= 4 && SA <= 32 && SB >= 4 && CA >= 8 && CB >= 8, "column lengths 128..1024");
  static constexpr int kPairsA = CA / 2, kPairsB = CB / 2;
  // the tile, then the exchange in its place: 16 bytes (two columns) per point, the points of a run of 32
  // permuted by the run's number, which spreads a quarter warp's stores and loads over all banks in both parts
  static constexpr int kTile = TP * 8;
  // stage-2 twiddles of the powers 1 .. SA - 1 (at 2^20 points the row of ones would cost the third CTA of an SM)
  static constexpr int kTw = (SA - 1) * 32 * 8, kRoots = (N1 / 4 + 128) * 8;
  static constexpr int kSmem = kTile + kTw + kRoots;
  static constexpr int kCtas = WARPS == 4 ? 3 : 1;  // per SM: 228 KB, of which a CTA takes 1 KB and its static variables more
  static_assert(kCtas * (kSmem + 1024 + 256) <= 228 * 1024, "resident CTAs");
  // chunk swizzle of part A's tile (16-byte units, U per row): the eight lanes of a 16-byte load, which
  // read eight consecutive rows of one pair (four rows of two pairs when SA = 4), hit distinct banks
  static constexpr int U = CA / 2;
  __device__ __forceinline__ static int swz(int row) {
    return SA == 4 ? 2 * (row & 3) : U == 4 ? (row >> 1) & 3 : row & 7;
  }
};

// The order of the work: `lag` items of part A, then items of A and B in turn, then the last `lag` of B. Returns
// the part (0: A, 1: B) of ticket t, *item its number within the part.
__device__ __forceinline__ int part_of(unsigned t, unsigned items, unsigned lag, unsigned* item) {
  if (t < lag) {
    *item = t;
    return 0;
  }
  const unsigned u = t - lag;
  if (u < 2 * (items - lag)) {
    *item = (u >> 1) + ((u & 1) ? 0 : lag);
    return (int)(u & 1);
  }
  *item = u - (items - lag);
  return 1;
}

// Sums over the 2^LV lanes of a bin's group, each lane ending with 16 >> LV of the 16 values; returns the
// number of the first one it holds. s[0 .. 16 >> LV) hold them on return.
template <int LV>
__device__ __forceinline__ int reduce_scatter(float2 (&s)[16], int lane) {
  int q0 = 0;
#pragma unroll
  for (int l = 0; l < LV; ++l) {
    const int off = 1 << (LV - 1 - l), keep = 16 >> (l + 1);
    const bool up = (lane & off) != 0;
    q0 += up ? keep : 0;
#pragma unroll
    for (int i = 0; i < keep; ++i) {
      const float2 give = up ? s[i] : s[i + keep], mine = up ? s[i + keep] : s[i];
      s[i].x = mine.x + __shfl_xor_sync(0xffffffffu, give.x, off);
      s[i].y = mine.y + __shfl_xor_sync(0xffffffffu, give.y, off);
    }
  }
  return q0;
}

static __device__ __noinline__ void emit_trigger(const Args& a, float best, int64_t sample, int tmpl, float zr, float zi) {
  const unsigned long long idx = atomicAdd(a.counter, 1ull);
  if ((int64_t)idx >= a.cap) return;
  rb_trigger t;
  t.sample = sample;
  t.tmpl = tmpl;
  t.block = a.block_id;
  t.snr = sqrtf(best);
  t.phase = atan2f(zi, zr);
  a.trig[idx] = t;
}

static __device__ __noinline__ void emit_candidate(const Args& a, float r2, int bin, int tmpl) {
  const unsigned long long idx = atomicAdd(a.counter, 1ull);
  if ((int64_t)idx >= a.cap) return;
  rb_candidate c;
  c.tmpl = tmpl;
  c.bin = bin;
  c.snr_avg = sqrtf(r2);
  c.block = a.block_id;
  a.cand[idx] = c;
}

// The window of one pair of columns and its lanes (all of a warp's windows at once): arg-max, first on ties,
// emitted by the window's first lane when it reaches the threshold. m: block sample of the pair's first column.
static __device__ __noinline__ void plain_window(const Args& a, float2 re, float2 im, int64_t m, int tmpl) {
  const float x = fmaf(re.x, re.x, im.x * im.x), y = fmaf(re.y, re.y, im.y * im.y);
  const float ra = x >= 0.f ? x : -1.f, rb = y >= 0.f ? y : -1.f;  // (a NaN is never the best)
  if (a.log2w == 0) {
    if (ra >= a.thr2) emit_trigger(a, ra, a.sample_offset + m, tmpl, re.x, im.x);
    if (rb >= a.thr2) emit_trigger(a, rb, a.sample_offset + m + 1, tmpl, re.y, im.y);
    return;
  }
  const bool second = rb > ra;
  float best = second ? rb : ra, zr = second ? re.y : re.x, zi = second ? im.y : im.x;
  const int first = 2 * ((int)(threadIdx.x & 31) & ((1 << (a.log2w - 1)) - 1));  // the pair's place in the window
  int at = first + second;
  for (int off = 1; off < (a.w >> 1); off <<= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, off), orr = __shfl_xor_sync(0xffffffffu, zr, off),
                oi = __shfl_xor_sync(0xffffffffu, zi, off);
    const int oa = __shfl_xor_sync(0xffffffffu, at, off);
    if (ob > best || (ob == best && oa < at)) {
      best = ob;
      zr = orr;
      zi = oi;
      at = oa;
    }
  }
  if (first == 0 && best >= a.thr2) emit_trigger(a, best, a.sample_offset + m + at, tmpl, zr, zi);
}

template <int LOG2N, int WARPS, int KIND>
__global__ void __launch_bounds__(32 * WARPS, Shape<LOG2N, WARPS>::kCtas) k_series(const __grid_constant__ Args a) {
  using S = Shape<LOG2N, WARPS>;
  constexpr bool FULL = KIND == KIND_FOLD;
  constexpr int N1 = S::N1, N2 = S::N2, NT = S::NT, TP = S::TP, I = S::ITEMS, SA = S::SA, SB = S::SB;
  constexpr int64_t N = (int64_t)1 << LOG2N, HALF = N / 2;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* const tile = smem;
  float2* const tw = reinterpret_cast<float2*>(smem + S::kTile);  // [r - 1][32]: exp(2 pi i j r / n2)
  float2* const roots = reinterpret_cast<float2*>(smem + S::kTile + S::kTw);
  __shared__ unsigned s_next[2];
  __shared__ int s_ready[2], s_abort;

  // (read anew where they are used: the values of a stage leave no registers for what can be had again)
  auto thread = [&]() {
    unsigned t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return (int)t;
  };
  auto opaque = [](unsigned x) {
    asm volatile("" : "+r"(x));
    return x;
  };
  const unsigned items = (unsigned)I * (unsigned)a.nvec, total = 2 * items;
  unsigned* const done_a = a.sync + kSyncHead;
  unsigned* const done_b = done_a + (1 << a.log2ring);
  const unsigned slot_mask = (1u << a.log2ring) - 1;

  // A ticket starts when the counter of its row has reached a number: B when all of the row's A items are written
  // (one count per warp), A when the ring slot's previous row has been read.
  struct Need {
    const unsigned* at;
    unsigned count;
  };
  auto need_of = [&](unsigned t) -> Need {
    unsigned item;
    const int part = part_of(t, items, (unsigned)a.lag, &item);
    const unsigned vec = item / I, gen = vec >> a.log2ring;
    return {(part ? done_a : done_b) + (vec & slot_mask), part ? (gen + 1) * (unsigned)(I * WARPS) + a.withhold : gen * (unsigned)I};
  };
  // (one thread) until the ticket may start; false when it never will
  auto wait_ready = [&](unsigned t) {
    const uint64_t t0 = timer_ns();
    const Need p = need_of(t);
    while (ld_acquire(p.at) < p.count) {
      if (ld_acquire(a.sync + 2)) return false;
      if (timer_ns() - t0 > kWaitNs) {
        atomicOr(a.flags, (unsigned)RB_FLAG_TIMEOUT);
        atomicExch(a.sync + 2, 1u);
        return false;
      }
      __nanosleep(100);
    }
    return true;
  };
  // (every thread) the tile of ticket t into shared memory; short loops, for the code's sake (2.76 -> 2.71 us a row with them)
  auto request = [&](unsigned t) {
    unsigned item;
    const int part = part_of(t, items, (unsigned)a.lag, &item);
    const unsigned vec = item / I, grp = item % I;
    const int tid = thread();
    const uint32_t tile_s = (uint32_t)__cvta_generic_to_shared(tile);
    if (part == 0) {
      constexpr int U = S::U;
      // a thread's rows lie NT / U apart, a multiple of the swizzle's period, so one offset serves them all
      static_assert((NT / U) % (SA == 4 ? 4 : 8) == 0, "swizzle period");
      const uint32_t dst0 = tile_s + (tid / U * U + (tid % U ^ S::swz(tid / U))) * 16;
      if constexpr (FULL) {
        const float2* src = a.rows + (int64_t)vec * N + grp * S::CA + (int64_t)(tid / U) * N1 + 2 * (tid % U);
#pragma unroll 4
        for (int i = 0; i < TP / 2 / NT; ++i) cp16(dst0 + i * NT * 16, src + (int64_t)i * (NT / U) * N1);
      } else {
        const float2* src = a.rows + (int64_t)vec * HALF + grp * S::CA + (int64_t)(tid / U) * N1 + 2 * (tid % U);
        const float2* sh = a.shat + grp * S::CA + (int64_t)(tid / U) * N1 + 2 * (tid % U);
        if (a.align_rows) {
#pragma unroll 4
          for (int i = 0; i < TP / 4 / NT; ++i) {
            const uint32_t dst = dst0 + i * NT * 16;
            cp16(dst, src + (int64_t)i * (NT / U) * N1);
            cp16(dst + TP * 4, sh + (int64_t)i * (NT / U) * N1);
          }
        } else {
#pragma unroll 1
          for (int i = 0; i < TP / 4 / NT; ++i) {
            const uint32_t dst = dst0 + i * NT * 16;
            const float2 *p = src + (int64_t)i * (NT / U) * N1, *q = sh + (int64_t)i * (NT / U) * N1;
            cp8(dst, p);
            cp8(dst + 8, p + 1);
            cp8(dst + TP * 4, q);
            cp8(dst + TP * 4 + 8, q + 1);
          }
        }
      }
    } else {
      constexpr int U = S::kPairsB;
      const float2* src = a.X + (int64_t)(vec & slot_mask) * N + grp * S::CB + (int64_t)(tid / U) * N2 + 2 * (tid % U);
#pragma unroll 4
      for (int i = 0; i < TP / 2 / NT; ++i) cp16(tile_s + (tid + i * NT) * 16, src + (int64_t)i * (NT / U) * N2);
    }
  };

  // Thread 0 holds two tickets beyond the current one: t1, whose counter (seen) and t2, which itself, are asked for
  // an item before they are needed, so that the round trips are not waited for.
  unsigned t1 = total, t2 = total, seen = 0;
  auto look = [&]() {
    if (t1 < total) {
      seen = ld_relaxed(need_of(t1).at);
      t2 = atomicAdd(a.sync, 1u);
    }
  };
  if (threadIdx.x == 0) s_next[0] = atomicAdd(a.sync, 1u);
  for (int e = threadIdx.x; e < N2 - 32; e += NT) tw[e] = a.w2a[(e & 31) * (SA + 1) + (e >> 5) + 1];
  for (int e = threadIdx.x; e < N1 / 4 + 128; e += NT) roots[e] = a.w4[e];
  if (threadIdx.x == 0) s_abort = s_next[0] < total && !wait_ready(s_next[0]);
  __syncthreads();
  unsigned cur = s_next[0];
  bool asked = false;  // this ticket's tile is on its way
  int pending = -1;    // ring slot of finished A results that are not announced yet
  unsigned turn = 0;
  __syncthreads();  // (s_next[0] is written again below)
  if (threadIdx.x == 0 && cur < total) {
    t1 = atomicAdd(a.sync, 1u);
    look();
  }

#pragma unroll 1
  while (cur < total && !s_abort) {
    if (!asked) request(cur);
    unsigned number;
    const int part = part_of(cur, items, (unsigned)a.lag, &number);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // the tile is there
    unsigned row, grp, slot;
    // (every thread, when it has read the exchange) the announcement of the item before, whose stores have long
    // landed, and the next ticket's tile
    auto advance = [&]() {
      __syncwarp();
      if (thread() % 32 == 0) {
        if (pending >= 0 || threadIdx.x == 0) fence_gpu();  // (thread 0's also orders the counter seen before the reads it allows)
        if (pending >= 0) red_relaxed(done_a + pending);
        if (threadIdx.x == 0) {
          if (part) red_relaxed(done_b + (opaque(number) / I & slot_mask));  // the X tile has been read
          s_next[turn & 1] = t1;
          s_ready[turn & 1] = t1 >= total || seen >= need_of(t1).count;
        }
      }
      pending = -1;
      __syncthreads();
      asked = s_ready[turn & 1] && s_next[turn & 1] < total;
      if (asked) request(s_next[turn & 1]);
      if (threadIdx.x == 0) {
        t1 = t2;
        t2 = total;
        look();
      }
      const unsigned item = opaque(number);
      row = item / I;
      grp = item % I;
      slot = row & slot_mask;
    };
    C2 v[32], y[32];
    const int tid = thread(), lane = tid & 31;
    if (part == 0) {
      const int pr = (tid >> 5) * (32 / SA) + lane / SA, tj = lane % SA;  // pair of columns, thread of the pair
      const float4* t4 = reinterpret_cast<const float4*>(tile) + tj * S::U + (pr ^ S::swz(tj));
      if constexpr (FULL) {
#pragma unroll
        for (int r = 0; r < 32; ++r) {
          const float4 x = t4[r * SA * S::U];
          v[r] = {pack(x.x, x.z), pack(x.y, x.w)};
        }
      } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) {  // s_hat conj(row)
          const float4 x = t4[r * SA * S::U], s = t4[TP / 4 + r * SA * S::U];
          v[r] = {pack(fmaf(s.x, x.x, s.y * x.y), fmaf(s.z, x.z, s.w * x.w)),
                  pack(fmaf(s.y, x.x, -s.x * x.y), fmaf(s.w, x.z, -s.z * x.w))};
        }
      }
      __syncthreads();  // the tile has been read
      dftp<32, 1, !FULL, false>(v, y);
      // exchange within the warp: y1[32 tj + k] out, y1[j + 32 r] in
      // (eight addresses, one per low part of the point's number, and constant offsets from them)
      ulonglong2* const ex = reinterpret_cast<ulonglong2*>(tile) + pr * N2;
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        ulonglong2* const e = ex + 32 * tj + (m ^ (tj & 7));
#pragma unroll
        for (int k2 = m; k2 < 32; k2 += 8) e[k2 - m] = make_ulonglong2(y[k2].re, y[k2].im);
      }
      __syncwarp();
#pragma unroll
      for (int b = 0; b < 32 / SA; ++b)
#pragma unroll
        for (int m = 0; m < (SA < 8 ? SA : 8); ++m) {
          const ulonglong2* const e = ex + ((tj + SA * b) ^ m);
#pragma unroll
          for (int r = m; r < SA; r += 8) {
            const ulonglong2 x = e[32 * r];
            v[b * SA + r] = {x.x, x.y};
          }
        }
      advance();
      // four-step twiddles w_n^(j1 (j + 32 k)), j = tj + SA b: w_n^(j1 tj) (w_n^(SA j1))^b (w_n^(32 j1))^k
      const int j1 = (int)grp * S::CA + 2 * pr;
      auto root = [&](int e) { return cmul(roots[e >> 7], roots[N1 / 4 + (e & 127)]); };  // w_n^e, e < 32 n1
      auto both = [&](int f) -> C2 {
        const float2 p = root(j1 * f), q = root(j1 * f + f);
        return {pack(p.x, q.x), pack(p.y, q.y)};
      };
      constexpr int CH = 4;  // the powers by running products: interleaved chains, of step^4 for radix 8 and more
      C2 base = both(tj);
      const C2 st1 = both(32);
      const u64 nst1 = neg2(st1.im);
      C2 st4 = st1;
      if constexpr (SA > CH) {
        const C2 st2 = cmul2(st1, st1, nst1);
        st4 = cmul2(st2, st2, neg2(st2.im));
      }
      const u64 nst4 = neg2(st4.im);
      float2* const xo = a.X + (int64_t)slot * N + (int64_t)j1 * N2 + tj;
#pragma unroll
      for (int b = 0; b < 32 / SA; ++b) {
#pragma unroll
        for (int r = 1; r < SA; ++r) v[b * SA + r] = cmul_w(v[b * SA + r], tw[(r - 1) * 32 + tj + SA * b]);
        dftp<SA, 1, false, false>(v + b * SA, y + b * SA);
        C2 p[CH];
        p[0] = base;
#pragma unroll
        for (int c = 1; c < CH; ++c) p[c] = cmul2(p[c - 1], st1, nst1);
#pragma unroll
        for (int k2 = 0; k2 < SA; ++k2) {
          const float2 wr2 = unpack(p[k2 % CH].re), wi2 = unpack(p[k2 % CH].im);
          const float2 re = unpack(y[b * SA + k2].re), im = unpack(y[b * SA + k2].im);
          xo[SA * b + 32 * k2] = cmul(make_float2(re.x, im.x), make_float2(wr2.x, wi2.x));
          xo[N2 + SA * b + 32 * k2] = cmul(make_float2(re.y, im.y), make_float2(wr2.y, wi2.y));
          if (k2 + CH < SA) p[k2 % CH] = cmul2(p[k2 % CH], st4, nst4);
        }
        if (b + 1 < 32 / SA) {
          const C2 bs = both(SA);
          base = cmul2(base, bs, neg2(bs.im));
        }
      }
      pending = (int)slot;
    } else {
      constexpr int PB = S::kPairsB;
      const int pr = tid % PB, tj = tid / PB;  // lanes across the pairs
      const float4* t4 = reinterpret_cast<const float4*>(tile) + tid;
#pragma unroll
      for (int r = 0; r < 32; ++r) {
        const float4 x = t4[r * NT];
        v[r] = {pack(x.x, x.z), pack(x.y, x.w)};
      }
      __syncthreads();  // the tile has been read
      dftp<32, 1, false, false>(v, y);
      ulonglong2* const ex = reinterpret_cast<ulonglong2*>(tile) + pr;
      constexpr int X = PB == 4 ? 1 : 0;  // (eight pairs and more: a quarter warp holds one point)
#pragma unroll
      for (int k2 = 0; k2 < 32; ++k2) ex[(32 * tj + (k2 ^ (tj & X))) * PB] = make_ulonglong2(y[k2].re, y[k2].im);
      __syncthreads();
#pragma unroll
      for (int b = 0; b < 32 / SB; ++b)
#pragma unroll
        for (int r = 0; r < SB; ++r) {
          const ulonglong2 x = ex[(32 * r + ((tj + SB * b) ^ (r & X))) * PB];
          v[b * SB + r] = {x.x, x.y};
        }
      advance();
      // the kept outputs: butterfly b, k = SB/2 + kk: row p = tj + SB b + 32 kk of the valid half
      C2 z[16];
#pragma unroll
      for (int b = 0; b < 32 / SB; ++b) {
#pragma unroll
        for (int r = 1; r < SB; ++r) v[b * SB + r] = cmul_w(v[b * SB + r], tw[(r * (N2 / N1) - 1) * 32 + tj + SB * b]);
        dftp<SB, 1, false, true>(v + b * SB, y + b * SB);
#pragma unroll
        for (int kk = 0; kk < SB / 2; ++kk) z[b * (SB / 2) + kk] = y[b * SB + SB / 2 + kk];
      }
      auto row_of = [&](int q) { return tj + SB * (q / (SB / 2)) + 32 * (q % (SB / 2)); };
      const int m2 = (int)grp * S::CB + 2 * pr;
      const int64_t vec = a.vec0 + row;
      if constexpr (KIND == KIND_BANK) {
        if (a.beta) {
          float2* const out = a.beta + vec * HALF + m2;
          if (a.align_beta) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const float2 re = unpack(z[q].re), im = unpack(z[q].im);
              __stcs(reinterpret_cast<float4*>(out + (int64_t)N2 * row_of(q)), make_float4(re.x, im.x, re.y, im.y));
            }
          } else {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const float2 re = unpack(z[q].re), im = unpack(z[q].im);
              out[(int64_t)N2 * row_of(q)] = make_float2(re.x, im.x);
              out[(int64_t)N2 * row_of(q) + 1] = make_float2(re.y, im.y);
            }
          }
        }
        float2* const avg = a.beta_avg + vec * (HALF >> a.log2w) + (m2 >> a.log2w);
        if (a.log2w == 0) {
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float2 re = unpack(z[q].re), im = unpack(z[q].im);
            avg[(int64_t)N2 * row_of(q)] = make_float2(re.x, im.x);
            avg[(int64_t)N2 * row_of(q) + 1] = make_float2(re.y, im.y);
          }
        } else {
          float2 s[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float2 re = unpack(z[q].re), im = unpack(z[q].im);
            s[q] = make_float2(re.x + re.y, im.x + im.y);
          }
          const float inv = 1.0f / (float)a.w;
          auto put = [&](int q0, auto count) {
#pragma unroll
            for (int i = 0; i < decltype(count)::value; ++i)
              avg[(int64_t)(N2 >> a.log2w) * row_of(q0 + i)] = cscale(s[i], inv);
          };
          if (a.log2w == 1) {
            put(0, std::integral_constant<int, 16>{});
          } else if (a.log2w == 2) {
            put(reduce_scatter<1>(s, lane), std::integral_constant<int, 8>{});
          } else if (a.log2w == 3) {
            put(reduce_scatter<2>(s, lane), std::integral_constant<int, 4>{});
          } else {
            put(reduce_scatter<3>(s, lane), std::integral_constant<int, 2>{});
          }
        }
      } else {
        // few samples reach the threshold: a warp looks closer only when one of its samples does (fmaxf
        // passes NaN samples over, as the comparisons further on do)
        float most = 0.f;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const float2 re = unpack(z[q].re), im = unpack(z[q].im);
          most = fmaxf(most, fmaxf(fmaf(re.x, re.x, im.x * im.x), fmaf(re.y, re.y, im.y * im.y)));
        }
        if (__any_sync(0xffffffffu, most >= a.thr2)) {
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float2 re = unpack(z[q].re), im = unpack(z[q].im);
            const int64_t m = HALF + m2 + (int64_t)N2 * row_of(q);
            if constexpr (KIND == KIND_PLAIN) {
              plain_window(a, re, im, m, (int)vec);
            } else {
              const float x = fmaf(re.x, re.x, im.x * im.x), y2 = fmaf(re.y, re.y, im.y * im.y);
              if (x >= a.thr2) emit_candidate(a, x, (int)m, (int)vec);
              if (y2 >= a.thr2) emit_candidate(a, y2, (int)m + 1, (int)vec);
            }
          }
        }
      }
    }
    const unsigned nx = s_next[turn & 1];
    if (!s_ready[turn & 1]) {
      // the next ticket has to wait for others: announce what is done first
      __syncwarp();
      if (pending >= 0 && thread() % 32 == 0) {
        fence_gpu();
        red_relaxed(done_a + pending);
      }
      pending = -1;
      if (threadIdx.x == 0 && !wait_ready(nx)) s_abort = 1;
      __syncthreads();
    }
    cur = nx;
    ++turn;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  if (pending >= 0 && thread() % 32 == 0) {
    fence_gpu();
    red_relaxed(done_a + pending);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // the last CTA leaves the words zero for the next launch (an aborted launch: the next call's set-up does)
    fence_gpu();
    const bool last = atomicAdd(a.sync + 1, 1u) == gridDim.x - 1;
    fence_gpu();
    const bool gave_up = last && ld_acquire(a.sync + 2);
    if (last && !gave_up) {
      for (int i = 0; i < 2 << a.log2ring; ++i) done_a[i] = 0;
      a.sync[0] = 0;
      a.sync[1] = 0;
    }
    s_abort = gave_up;
  }
  if constexpr (KIND == KIND_BANK) {  // (the other kinds' callers read the flag)
    __syncthreads();
    if (s_abort) {
      const float nan = __int_as_float(0x7fffffff);
      const int64_t rows = a.nvec, bins = HALF >> a.log2w;
      for (int64_t i = threadIdx.x; i < rows * bins; i += NT) a.beta_avg[a.vec0 * bins + i] = make_float2(nan, nan);
      if (a.beta)
        for (int64_t i = threadIdx.x; i < rows * HALF; i += NT) a.beta[a.vec0 * HALF + i] = make_float2(nan, nan);
    }
  }
}

// SMs of the current device, asked once per device.
inline int sm_count() {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < kDevices && (sms = known[dev].load()) > 0) return sms;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  if (dev >= 0 && dev < kDevices) known[dev].store(sms);
  return sms;
}

// rows_ws: rows of X that the workspace holds. The ring is as long as the order needs, so that X stays in L2.
template <int LOG2N, int WARPS, int KIND>
int launch(Args a, int rows_ws, cudaStream_t st) {
  using S = Shape<LOG2N, WARPS>;
  auto kern = k_series<LOG2N, WARPS, KIND>;
  RB_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem));
  const int64_t items = (int64_t)S::ITEMS * a.nvec;
  const int grid = (int)std::min<int64_t>(2 * items, sm_count() * S::kCtas);
  // A row is complete one row's items and the items in flight (half of every CTA's current and next) after its
  // first item; the ring holds the rows between the first A item and the last B item in flight.
  const auto rows_of = [&](int64_t t) { return (int)((t + S::ITEMS - 1) / S::ITEMS); };
  a.lag = (int)std::min<int64_t>(items, S::ITEMS + 1 + grid);
  const int want = rows_of(a.lag) + 2 + rows_of(grid / 2);
  // a power of two: of at least nvec rows (no slot is used twice), or of what the workspace holds
  a.log2ring = 0;
  while ((1 << a.log2ring) < a.nvec && (2 << a.log2ring) <= (a.nvec <= rows_ws ? 2 * a.nvec : rows_ws) && (1 << a.log2ring) < want) ++a.log2ring;
  const int ring = 1 << a.log2ring;
  if (ring < a.nvec && rows_of(a.lag) + 2 > ring)  // a short ring: fewer items ahead
    a.lag = (int)std::max<int64_t>(S::ITEMS + 2, (int64_t)(ring - 2) * S::ITEMS);
  kern<<<grid, S::NT, S::kSmem, st>>>(a);
  RB_LAUNCH_CHECK();
  return RB_OK;
}

}  // namespace rbseries
