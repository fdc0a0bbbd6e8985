// gen_resident.cuh — many generations of a population that fits on the chip
// in one cooperative launch (de_run on rows of the row-per-CTA kernel).
//
// A generation of such a population moves a few megabytes through L2 and is a
// chain of dependent steps, not a stream: a launch per generation (1.6-2.1 us)
// plus the loads of the generation number, slot bytes, row and donors, the
// selection's atomics and the close, one after the other. Here every CTA owns
// a block of rows for the whole run and keeps them in shared memory, and rows
// wait only for what they read:
//
//  - Every row has a 32-bit word in global memory, (generation tag, buffer
//    that holds the row now and in the three generations before). The warps of
//    a row poll the words of its three donors, load the donors' genes, and
//    publish the row's own word after the selection. There is no grid barrier
//    on that path: a barrier of 152 CTAs costs 1.4-1.7 us here (an arrival
//    counter; 2.7-5.4 us as an all-gather of words that every CTA polls),
//    a published word 0.6 us.
//  - Four buffers hold each row's versions: the current one, the one that the
//    next trial goes to, and two more that come after it in turn. A trial is
//    stored as soon as it is formed, before its fitness is known; if it loses,
//    nobody reads it. The buffer that a trial of generation h goes to was last
//    current in generation h - 3 at the latest, so the store needs every CTA
//    to have finished that generation.
//    Only the slots that changed are stored: each lane keeps, per buffer, which
//    of its slots that buffer holds from an older version.
//  - Two helper warps per CTA keep all of that off the rows' path: one draws
//    donors and lengths a few generations ahead (pure functions of seed,
//    generation and row), the other counts finished generations on arrival
//    counters (a ring, one per generation); both tell the rows' warps through
//    shared memory which generations are drawn and may be stored. Nothing in
//    the loop synchronises a whole CTA.
//  - NEC and exponential segments change L genes of a row (10 on average at
//    Cr = 0.9): one warp owns a row, keeps the partial sums of gen_kernel's
//    threads and warps in shared memory, and computes again only those whose
//    genes the segment changed, so a generation costs O(L) instructions, not
//    O(D). Binomial rows take a warp per 128 genes and sum all. Both sum in
//    gen_kernel's order, so values, selections and populations are
//    bit-identical to de_step's.
//  - Every wait is bounded (ResidentParams::wait_ns); a CTA that gives up
//    records DE_ETIMEOUT, leaves the loop and still closes, so the launch ends.
//    Its rows stay where their words say; the last CTA, when nobody reads any
//    more, brings every row's last version together and counts the generations
//    that all rows have finished.
//    Whether a wait was met is one answer for a warp, and for the warps of a row
//    one that they agree on at the row's barriers: no plan, word or barrier is
//    used by lanes or warps that went on alone.
//
// What bounds it: latency. A generation is the chain poll a word (L2, 0.5 us on
// a line that another SM has just written), load the genes (0.5 us), some 300
// dependent instructions, fence and publish (0.5 us). Per generation, against
// a launch each: NEC sphere N = 100, D = 30 4.5 -> 2.0 us, Rastrigin N = 1024,
// D = 1000 5.7 -> 2.5 us (exponential at Cr = 0.5 6.6 -> 2.5 us), binomial
// Griewank N = 300, D = 500 5.5 -> 2.9 us. Words that share a line cost twice
// that (5 us at N = 300, D = 500): each has a line of its own. Waits that let the
// lanes of a warp leave one by one cost up to twice as well, for as long as the lanes
// stayed apart: the same binomial run took 3.05 or 6.04 us from one launch to the next.
#pragma once
#include "draws.cuh"
#include "internal.h"
#include "objectives.cuh"
#include "ptx.cuh"
#include "slot_terms.cuh"

namespace de {

// Draws of one row and generation, in shared memory.
struct __align__(16) ResPlan {
  int r[3], jrand;
  // exp and NEC: the slots whose sums the segment changes are a0 .. a0 + n0 - 1
  // and 0 .. n - n0 - 1 (for Rosenbrock the one before the segment is among
  // them), those of the warps `again`; mask: genes that cross in the first,
  // second and last of the slots (four bits each), all in the others
  int L;
  uint16_t a0, n0, n, mask;
  unsigned again;
};
// Generations of plans in shared memory: a draw takes the latency of some 400
// instructions whatever the lanes in use, so few rows are drawn many
// generations at a time.
__host__ __device__ inline int res_depth(int rpc) { return rpc <= 16 ? 16 : 4; }

// Row word: generation tag above eight bits, the buffer of the row at that
// tag (bits 0-1) and one, two and three generations before (2-7).
constexpr uint32_t kResTagMask = 0x00FFFFFFu;

__device__ __forceinline__ float4 ld_l2(const float4* p) {
  float4 v;
  asm volatile("ld.relaxed.gpu.global.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_flag(const int* p) {   // flags in shared memory
  int v;
  asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_flag(int* p, int v) {
  asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void red_release(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Shared memory of one CTA, in bytes from the start of the dynamic block.
struct ResLayout {
  unsigned rows, trial, sums, new_sums, warp_sums, stale, plans, red, first, fit, slot, total;
};
// T threads and V slots per thread as in gen_kernel, ns sums per row; groups
// rows at a time. seg: the layout of the segment kernel.
__host__ __device__ inline ResLayout res_layout(bool seg, int rpc, int D4, int groups, int T, int V, int ns) {
  ResLayout l;
  unsigned o = 0;
  const unsigned R = (unsigned)rpc, G = (unsigned)groups, nw = (unsigned)T / 32u;
  l.rows = o; o += R * D4 * 16u;
  l.trial = o; o += seg ? G * D4 * 16u : 0u;
  l.stale = o; o += R * (seg ? 1u : nw) * 128u;              // four buffers x slots of a lane, as bits
  l.plans = o; o += (unsigned)res_depth(rpc) * R * (unsigned)sizeof(ResPlan);
  l.sums = o; o += seg ? R * ns * T * 4u : 0u;
  l.new_sums = o; o += seg ? G * ns * T * 4u : 0u;
  l.warp_sums = o; o += seg ? R * ns * 32u : 0u;
  l.red = o; o += seg ? 0u : G * 2u * 3u * 32u;              // two sets of three sums of up to 8 warps
  l.first = o; o += seg ? 0u : G * V * 32u;
  l.fit = o; o += (R * 4u + 15u) & ~15u;
  l.slot = o; o += (R * 4u + 15u) & ~15u;
  l.total = o;
  return l;
}

// One slot q of a row (genes 4q ..) added to a thread's sums; nb is gene 4q + 4.
template <int OBJ>
__device__ __forceinline__ void res_slot(Acc& a, const float4& x, float nb, int q, const GenParams& p) {
  const int j0 = 4 * q;
  if constexpr (OBJ == kRosenbrock) {
    if (j0 + 1 < p.D) accum_pair(a, x.x, x.y);
    if (j0 + 2 < p.D) accum_pair(a, x.y, x.z);
    if (j0 + 3 < p.D) accum_pair(a, x.z, x.w);
    if (j0 + 4 < p.D) accum_pair(a, x.w, nb);
  } else if constexpr (OBJ == kGriewank) {
    griewank_slot(a, x, j0, p);
  } else {
    accum_gene<OBJ>(a, x.x, j0, p);
    if (j0 + 1 < p.D) accum_gene<OBJ>(a, x.y, j0 + 1, p);
    if (j0 + 2 < p.D) accum_gene<OBJ>(a, x.z, j0 + 2, p);
    if (j0 + 3 < p.D) accum_gene<OBJ>(a, x.w, j0 + 3, p);
  }
}

// gen_kernel's butterfly over the lanes, strides kFrom, kFrom / 2, .. 1.
template <int NS, int kFrom>
__device__ __forceinline__ void res_butterfly(Acc& s) {
#pragma unroll
  for (int o = kFrom; o > 0; o >>= 1) {
    s.a += __shfl_xor_sync(0xFFFFFFFFu, s.a, o);
    if (NS > 1) s.b += __shfl_xor_sync(0xFFFFFFFFu, s.b, o);
    if (NS > 2) s.c += __shfl_xor_sync(0xFFFFFFFFu, s.c, o);
  }
}

// kSeg: one warp per row that computes again what a segment (exp, NEC) changed
// (V = 1); else binomial, a warp per 128 V genes that computes all of them.
template <bool kSeg, int OBJ, int V>
__global__ void __launch_bounds__(kResThreads, 1) resident_kernel(const __grid_constant__ ResidentParams rp) {
  const GenParams& p = rp.g;
  extern __shared__ __align__(16) unsigned char res_smem[];
  __shared__ int s_dead, s_drawn, s_safe;   // a wait gave up; generations drawn; last generation whose trials may be stored
  __shared__ int s_done[kResWarps];         // per group: generations finished
  __shared__ unsigned long long s_masked, s_wins, s_key, s_hist;
  __shared__ int s_last, s_least;           // this CTA closes; generations that every row has finished

  constexpr int NS = ObjTraits<OBJ>::kSums;
  const int T = rp.row_threads, nw = T >> 5;       // threads and warps of a row in gen_kernel's order
  const int W = kSeg ? 1 : nw, groups = rp.groups; // warps per row, rows at a time
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int grp = wid / W, pw = wid - grp * W;
  const int helper = wid - (int)(blockDim.x >> 5) + kResHelpers + 1;   // 1, 2: the helper warps; below: a row's warp
  const ResLayout lay = res_layout(kSeg, rp.rpc, p.D4, groups, T, V, NS);
  float4* sx = reinterpret_cast<float4*>(res_smem + lay.rows);
  ResPlan* plans = reinterpret_cast<ResPlan*>(res_smem + lay.plans);
  float* sfit = reinterpret_cast<float*>(res_smem + lay.fit);
  uint32_t* sslot = reinterpret_cast<uint32_t*>(res_smem + lay.slot);   // buffers: queue of four in bits 0-7, the row's last three in 8-13
  // per lane and row: which of its slots the buffers 0-3 do not hold as the
  // row has them now, a byte each
  uint32_t* sstale = reinterpret_cast<uint32_t*>(res_smem + lay.stale);
  const int row0 = blockIdx.x * rp.rpc;
  const int rows = min(rp.rpc, p.N - row0);
  const long long gen0 = p.st->gen;
  const uint32_t tag0 = rp.rs->epoch, gave_up = rp.rs->failed;
  auto buffer = [&](uint32_t b) { return b == 0 ? p.pop0 : (b == 1 ? p.pop1 : rp.pop2 + (size_t)(b - 2) * p.N * p.pitch); };

  const uint8_t* slot_in = p.slots + (size_t)(gen0 & 1) * p.N;
  for (int q = tid; q < rows * p.D4; q += blockDim.x) {
    const int l = q / p.D4, i = row0 + l;
    sx[q] = reinterpret_cast<const float4*>((slot_in[i] ? p.pop1 : p.pop0) + (size_t)i * p.pitch)[q - l * p.D4];
  }
  if (gave_up) return;                             // a launch before this one did
  for (int q = tid; q < rows * W * 32; q += blockDim.x)
    sstale[q] = slot_in[row0 + q / (W * 32)] ? 0xFFFF00FFu : 0xFFFFFF00u;
  for (int l = tid; l < rows; l += blockDim.x) {
    const uint32_t c = slot_in[row0 + l] ? 1u : 0u;
    sfit[l] = p.fit[row0 + l];
    sslot[l] = c | ((1u - c) << 2) | (2u << 4) | (3u << 6) | (c * 0x15u) << 8;
    st_release(rp.words + (size_t)(row0 + l) * kResWordStride, (tag0 << 8) | (c * 0x55u));
  }
  if (tid == 0) {
    s_dead = 0;
    s_drawn = 0;
    s_safe = 2;
    s_masked = 0ULL;
    s_wins = 0ULL;
    s_key = ~0ULL;
    s_hist = ~0ULL;
    s_least = rp.gens;
  }
  if (tid < kResWarps) s_done[tid] = 0;
  __syncthreads();

  const int depth = res_depth(rp.rpc);             // a power of two
  auto draw = [&](int k0, int gens) {              // one warp: plans of the run's generations k0 .. k0 + gens - 1
    for (int e = lane; e < gens * rows; e += 32) {
      const int dk = e / rows, l = e - dk * rows, k = k0 + dk;
      const uint32_t g = (uint32_t)(gen0 + k);
      RowDraws d;
      draw_donors(p, g, row0 + l, d);
      int L = 0;
      if constexpr (kSeg) L = rp.xo == kNec ? nec_length(p, g, row0 + l) : exp_walk_length(p, g, row0 + l);
      ResPlan pl{};
      if constexpr (kSeg) {
        const int over = d.jrand + L - p.D;        // genes past the row's end
        const int a0 = max(0, (d.jrand >> 2) - (OBJ == kRosenbrock ? 1 : 0));
        const int b0 = over > 0 ? p.D4 - 1 : (d.jrand + L - 1) >> 2;
        const int b1 = over > 0 ? min((over - 1) >> 2, a0 - 1) : -1;
        auto crossing = [&](int q) {
          unsigned m = 0u;
          for (int e = 0; e < 4; ++e) {
            int de = 4 * q + e - d.jrand;
            if (de < 0) de += p.D;
            m |= (de < L && 4 * q + e < p.D) ? 1u << e : 0u;
          }
          return m;
        };
        for (int w = 0; w < nw; ++w)
          if ((32 * w <= b0 && 32 * w + 31 >= a0) || 32 * w <= b1) pl.again |= 1u << w;
        pl.a0 = (uint16_t)a0;
        pl.n0 = (uint16_t)(b0 - a0 + 1);
        pl.n = (uint16_t)(pl.n0 + b1 + 1);
        pl.mask = (uint16_t)(crossing(a0) | (crossing(a0 < b0 ? a0 + 1 : 0) << 4) | (crossing(b1 >= 0 ? b1 : b0) << 8));
      }
      pl.r[0] = d.r1; pl.r[1] = d.r2; pl.r[2] = d.r3;
      pl.jrand = d.jrand;
      pl.L = L;
      plans[(size_t)(k & (depth - 1)) * rp.rpc + l] = pl;
    }
  };
  // called by a whole warp, with one answer for it
  auto dead = [&] { return __shfl_sync(0xFFFFFFFFu, ld_flag(&s_dead), 0) != 0; };
  auto late = [&](unsigned long long t0) { return __any_sync(0xFFFFFFFFu, global_ns() - t0 > rp.wait_ns) != 0; };
  auto give_up = [&] {
    if (lane == 0) {
      st_flag(&s_dead, 1);
      atomicMax(&p.st->error, 4u);                 // DE_ETIMEOUT
    }
    __syncwarp();
  };
  // generations that every group of this CTA has finished. Each lane acquires its
  // group's flag and the warp's barrier hands that on: what the warp then writes,
  // or lane 0 releases, comes after the groups' reads
  auto finished = [&] {
    const int n = (int)__reduce_min_sync(0xFFFFFFFFu, lane < groups ? (unsigned)ld_flag(&s_done[lane]) : 0x7FFFFFFFu);
    __syncwarp();
    return n;
  };
  if (helper == 1) {                               // draws ahead
    const int batch = max(1, min(32 / max(1, rows), depth / 2));
    unsigned long long t0 = global_ns();
    for (int k = 0; k < rp.gens && !dead();) {
      const int room = min(depth - (k - finished()), rp.gens - k);
      if (room >= min(batch, rp.gens - k)) {
        draw(k, min(room, batch));
        k += min(room, batch);
        __syncwarp();
        if (lane == 0) st_flag(&s_drawn, k);
        t0 = global_ns();
      } else if (late(t0)) {
        give_up();
      } else {
        __nanosleep(200);                          // leaves the issue slots to the rows
      }
    }
  } else if (helper == 2) {                        // counts finished generations: this CTA's, and everyone's
    int arrived = 0, all = 0;
    unsigned long long t0 = global_ns();
    while (all < rp.gens && !dead()) {
      bool moved = false;
      for (const int done = finished(); arrived < done; ++arrived, moved = true)
        if (lane == 0) red_release(&rp.rs->ctr[arrived & 7], 1u);
      const uint32_t have = ld_acquire(&rp.rs->ctr[all & 7]);
      if (__all_sync(0xFFFFFFFFu, have >= (uint32_t)((all >> 3) + 1) * gridDim.x)) {
        __syncwarp();
        ++all;
        if (lane == 0) st_flag(&s_safe, all + 2);
        moved = true;
      }
      if (moved) t0 = global_ns();
      else if (late(t0)) give_up();
      else __nanosleep(64);
    }
  }
  // a worker warp's wait until `flag` (in shared memory) is at least `want`;
  // `seen` is the last value read, so that most waits read nothing. False: the
  // wait, or another one of the CTA, gave up, and what the flag stands for is not there
  int drawn_seen = 0, safe_seen = 2;
  auto wait_flag = [&](const int* flag, int& seen, int want) {
    if (seen >= want) return true;
    const unsigned long long t0 = global_ns();
    for (int n = 0;; ++n) {
      seen = __shfl_sync(0xFFFFFFFFu, ld_flag(flag), 0);
      if (seen >= want) break;
      if (dead()) return false;
      if ((n & 1023) == 1023 && late(t0)) give_up();
    }
    __syncwarp();
    return true;
  };

  // the buffers that hold the rows of a generation's donors: lanes 0-2 wait for
  // the words of row pl.r[lane] and the result is every lane's. False: gave up
  auto donors = [&](const ResPlan& pl, uint32_t tag, const float4*& d1, const float4*& d2, const float4*& d3) {
    uint32_t w = 0u, ahead = 0u;
    const uint32_t* wp = rp.words + (size_t)(lane == 0 ? pl.r[0] : (lane == 1 ? pl.r[1] : pl.r[2])) * kResWordStride;
    if (lane < 3) {
      w = ld_acquire(wp);
      ahead = ((w >> 8) - tag) & kResTagMask;
    }
    if (__any_sync(0xFFFFFFFFu, ahead > 3u)) {
      const unsigned long long t0 = global_ns();
      for (int n = 0;; ++n) {
        if (ahead > 3u) {
          w = ld_acquire(wp);
          ahead = ((w >> 8) - tag) & kResTagMask;
        }
        if (!__any_sync(0xFFFFFFFFu, ahead > 3u)) break;
        if (dead()) return false;
        if ((n & 63) == 63 && late(t0)) give_up();
      }
    }
    __syncwarp();                                  // what lanes 0-2 acquired, the others may read
    const uint32_t buf = (w >> (2u * ahead)) & 3u;
    d1 = reinterpret_cast<const float4*>(buffer(__shfl_sync(0xFFFFFFFFu, buf, 0)) + (size_t)pl.r[0] * p.pitch);
    d2 = reinterpret_cast<const float4*>(buffer(__shfl_sync(0xFFFFFFFFu, buf, 1)) + (size_t)pl.r[1] * p.pitch);
    d3 = reinterpret_cast<const float4*>(buffer(__shfl_sync(0xFFFFFFFFu, buf, 2)) + (size_t)pl.r[2] * p.pitch);
    return true;
  };

  unsigned long long masked = 0, wins = 0, key = ~0ULL, hist = ~0ULL;
  // the decision on row l in generation k, by one thread of its group: the
  // row's word and slot queue, fitness and the run's best
  auto decide = [&](int k, uint32_t tag, int l, uint32_t sl, float f, bool win) {
    const int i = row0 + l;
    const uint32_t c = sl & 3u, past = ((sl >> 6) & 0xFCu) | c;   // the buffers at this tag and before it
    const uint32_t queue = win ? ((sl & 0xFFu) >> 2) | (c << 6) : sl & 0xFFu;
    st_release(rp.words + (size_t)i * kResWordStride, ((tag + 1u) << 8) | ((past << 2) & 0xFCu) | (queue & 3u));
    sslot[l] = queue | (past & 0x3Fu) << 8;
    if (win) {
      sfit[l] = f;
      ++wins;
      key = min(key, best_key_of(f, i));
      hist = min(hist, ((unsigned long long)ordered_bits(f + 0.0f) << 32) | (unsigned)(k + 1));
    }
  };

  if constexpr (kSeg) {
    // a row's warp; group grp's rows are l = grp, grp + groups, ...
    float4* tr = reinterpret_cast<float4*>(res_smem + lay.trial) + (size_t)grp * p.D4;
    float* sums = reinterpret_cast<float*>(res_smem + lay.sums);
    float* nsum = reinterpret_cast<float*>(res_smem + lay.new_sums) + (size_t)grp * NS * T;
    float* wsums = reinterpret_cast<float*>(res_smem + lay.warp_sums);
    // sums of the threads 32 w .. 32 w + 31 of a row whose slots [a0, b0] and
    // [0, b1] are in tr and the others in x; the warp's sum is every lane's
    auto warp_sum = [&](const float4* x, int w, int a0, int b0, int b1, float* to) {
      Acc s{0.0f, 0.0f, 0.0f};
      const int q = 32 * w + lane;
      if (q < p.D4) {
        const float4 xv = ((q >= a0 && q <= b0) || q <= b1) ? tr[q] : x[q];
        float nb = 0.0f;
        if constexpr (OBJ == kRosenbrock) {
          if (q + 1 < p.D4) nb = ((q + 1 >= a0 && q + 1 <= b0) || q + 1 <= b1) ? tr[q + 1].x : x[q + 1].x;
        }
        res_slot<OBJ>(s, xv, nb, q, p);
      }
      to[32 * w + lane] = s.a;
      if (NS > 1) to[T + 32 * w + lane] = s.b;
      if (NS > 2) to[2 * T + 32 * w + lane] = s.c;
      res_butterfly<NS, 16>(s);
      return s;
    };
    if (helper < 1) {
      for (int l = grp; l < rows; l += groups)
        for (int w = 0; w < nw; ++w) {
          const Acc s = warp_sum(sx + (size_t)l * p.D4, w, 1, 0, -1, sums + (size_t)l * NS * T);
          if (lane == 0) {
            wsums[(l * NS) * 8 + w] = s.a;
            if (NS > 1) wsums[(l * NS + 1) * 8 + w] = s.b;
            if (NS > 2) wsums[(l * NS + 2) * 8 + w] = s.c;
          }
        }
      __syncwarp();
    }
    for (int k = 0; k < rp.gens && helper < 1; ++k) {
      const uint32_t tag = (tag0 + (uint32_t)k) & kResTagMask;
      bool ok = wait_flag(&s_drawn, drawn_seen, k + 1);
      for (int l = grp; l < rows && ok; l += groups) {
        const ResPlan pl = plans[(size_t)(k & (depth - 1)) * rp.rpc + l];
        const float fi = sfit[l];
        const uint32_t sl = sslot[l];
        float4* x = sx + (size_t)l * p.D4;
        float4* out = reinterpret_cast<float4*>(buffer((sl >> 2) & 3u) + (size_t)(row0 + l) * p.pitch);
        const int a0 = pl.a0, n0 = pl.n0, n = pl.n, b0 = a0 + n0 - 1, b1 = n - n0 - 1;
        // the slot of lane e of a pass, and the genes of it that cross
        auto slot_of = [&](int e) { return e < n0 ? a0 + e : e - n0; };
        auto crossing_of = [&](int e, int q) {
          unsigned m = q == p.D4 - 1 ? (1u << (p.D - 4 * q)) - 1u : 15u;
          if (e <= 1) m = pl.mask >> (4 * e);
          if (e == n - 1) m = pl.mask >> 8;
          return m & 15u;
        };
        // before the donors are there: what the trial's buffer holds from an older
        // version of the row and the segment leaves as it is
        uint32_t stale = sstale[l * 32 + lane];
        const uint32_t nshift = 8u * ((sl >> 2) & 3u), old = (stale >> nshift) & 0xFFu;
        ok = wait_flag(&s_safe, safe_seen, k);
        if (!ok) break;
#pragma unroll 1
        for (uint32_t todo = __reduce_or_sync(0xFFFFFFFFu, old); todo; todo &= todo - 1u) {
          const int w = __ffs((int)todo) - 1, q = 32 * w + lane;
          if (((old >> w) & 1u) && q < p.D4 && !((q >= a0 && q <= b0) || q <= b1)) __stcg(out + q, x[q]);
        }
        Acc s{0.0f, 0.0f, 0.0f};                   // lane w < nw: the sum of warp w
        if (lane < nw) {
          s.a = wsums[(l * NS) * 8 + lane];
          if (NS > 1) s.b = wsums[(l * NS + 1) * 8 + lane];
          if (NS > 2) s.c = wsums[(l * NS + 2) * 8 + lane];
        }
        float* own = sums + (size_t)l * NS * T;
        uint32_t touched = 0u;                     // this lane's slots in the segment
        const bool brief = n <= 32;                // a slot per lane: all in registers
        const bool mine = brief && lane < n;
        const int qe = mine ? slot_of(lane) : 0;
        const unsigned me = mine ? crossing_of(lane, qe) : 0u;
        float4 te = x[qe];
        Acc es{0.0f, 0.0f, 0.0f};
        const float4 *d1, *d2, *d3;
        ok = donors(pl, tag, d1, d2, d3);
        if (!ok) break;
        if (brief) {
          if (mine) {
            const float4 a1 = ld_l2(d1 + qe), a2 = ld_l2(d2 + qe), a3 = ld_l2(d3 + qe);
            mutate_slot(te, a1, a2, a3, me, p);
            __stcg(out + qe, te);
          }
          float nx = 0.0f;
          if constexpr (OBJ == kRosenbrock) {
            nx = __shfl_down_sync(0xFFFFFFFFu, te.x, 1);
            const float tx0 = __shfl_sync(0xFFFFFFFFu, te.x, 0);
            if (lane == n0 - 1 || lane >= n - 1) nx = qe + 1 < p.D4 ? x[qe + 1].x : 0.0f;
            if (lane == n - 1 && qe + 1 == a0) nx = tx0;   // the slots after the wrap end where the first one begins
          }
          __syncwarp();                            // all lanes compute on
          res_slot<OBJ>(es, te, nx, qe, p);
          __syncwarp();
#pragma unroll 1
          for (uint32_t todo = pl.again; todo; todo &= todo - 1u) {
            const int w = __ffs((int)todo) - 1, q = 32 * w + lane;
            const int e = (q >= a0 && q <= b0) ? q - a0 : (q <= b1 ? n0 + q : -1);
            Acc r;
            r.a = __shfl_sync(0xFFFFFFFFu, es.a, e & 31);
            if (NS > 1) r.b = __shfl_sync(0xFFFFFFFFu, es.b, e & 31);
            if (NS > 2) r.c = __shfl_sync(0xFFFFFFFFu, es.c, e & 31);
            if (e < 0) {
              r.a = own[q];
              if (NS > 1) r.b = own[T + q];
              if (NS > 2) r.c = own[2 * T + q];
            } else {
              touched |= 1u << w;
            }
            res_butterfly<NS, 16>(r);
            if (lane == w) s = r;
          }
        } else {
#pragma unroll 1
          for (int e = lane; e < n; e += 32) {
            const int q = slot_of(e);
            const float4 a1 = ld_l2(d1 + q), a2 = ld_l2(d2 + q), a3 = ld_l2(d3 + q);
            float4 t = x[q];
            mutate_slot(t, a1, a2, a3, crossing_of(e, q), p);
            tr[q] = t;
            __stcg(out + q, t);
          }
          __syncwarp();
#pragma unroll 1
          for (uint32_t todo = pl.again; todo; todo &= todo - 1u) {
            const int w = __ffs((int)todo) - 1;
            const int q = 32 * w + lane;
            if ((q >= a0 && q <= b0) || q <= b1) touched |= 1u << w;
            const Acc r = warp_sum(x, w, a0, b0, b1, nsum);
            if (lane == w) s = r;
          }
        }
        __syncwarp();                              // every store of the trial precedes the row's word
        s.a += 0.0f;
        if (NS > 1) s.b += 0.0f;
        if (NS > 2) s.c += 0.0f;
        const Acc ws = s;
        res_butterfly<NS, 4>(s);                   // lanes 0-7 hold the warps' sums or zero
        float f = finalize_fitness<OBJ>(s, p);
        f = __shfl_sync(0xFFFFFFFFu, f, 0);
        if (f != f) f = __int_as_float(0x7F800000);
        const bool win = f < fi;
        if (lane == 0) {
          decide(k, tag, l, sl, f, win);
          masked += (unsigned)pl.L;
        }
        // a winner's buffer holds the row, the others miss its slots; a loser's
        // buffer misses the slots that it tried
        stale &= ~(0xFFu << nshift);
        stale |= win ? (touched * 0x01010101u) & ~(0xFFu << nshift) : touched << nshift;
        sstale[l * 32 + lane] = stale;
        if (win) {
          if (mine) {
            x[qe] = te;
            own[qe] = es.a;
            if (NS > 1) own[T + qe] = es.b;
            if (NS > 2) own[2 * T + qe] = es.c;
          }
          if (!brief) {
#pragma unroll 1
            for (int e = lane; e < n; e += 32) x[slot_of(e)] = tr[slot_of(e)];
#pragma unroll 1
            for (uint32_t todo = pl.again; todo; todo &= todo - 1u) {
              const int t = 32 * (__ffs((int)todo) - 1) + lane;
              for (int c = 0; c < NS; ++c) own[c * T + t] = nsum[c * T + t];
            }
          }
          if (lane < nw) {
            wsums[(l * NS) * 8 + lane] = ws.a;
            if (NS > 1) wsums[(l * NS + 1) * 8 + lane] = ws.b;
            if (NS > 2) wsums[(l * NS + 2) * 8 + lane] = ws.c;
          }
        }
        __syncwarp();
      }
      if (!ok) break;
      if (lane == 0) st_flag(&s_done[grp], k + 1);
    }
  } else {
    float* red = reinterpret_cast<float*>(res_smem + lay.red) + grp * 2 * 24;
    float* first = reinterpret_cast<float*>(res_smem + lay.first) + grp * V * 8;
    int set = 0;
    // whether every warp of the group has what it waited for; a barrier of them
    auto agree = [&](bool ok) { return W > 1 ? named_bar_and(1 + grp, 32 * W, ok) : ok; };
    for (int k = 0; k < rp.gens && helper < 1; ++k) {
      const uint32_t g = (uint32_t)(gen0 + k), tag = (tag0 + (uint32_t)k) & kResTagMask;
      bool ok = wait_flag(&s_drawn, drawn_seen, k + 1);   // a warp without its plan goes on to the barrier
      for (int l = grp; l < rows; l += groups) {
        const ResPlan pl = ok ? plans[(size_t)(k & (depth - 1)) * rp.rpc + l] : ResPlan{};
        const int i = row0 + l;
        const float fi = sfit[l];
        const uint32_t sl = sslot[l];
        float4* out = reinterpret_cast<float4*>(buffer((sl >> 2) & 3u) + (size_t)i * p.pitch);
        uint32_t m = 0u;                           // crossover masks, four bits per slot
        float4 x[V], a1[V], a2[V], a3[V];
#pragma unroll
        for (int s = 0; s < V; ++s) {
          const int q = pw * 32 + lane + s * T;
          x[s] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (ok && q < p.D4) {
            unsigned b = bin_mask(p, philox_block_rk(p.rk, kStreamBin, p.inst, g, (uint32_t)i, (uint32_t)q), q, pl.jrand);
            b &= (1u << min(4, p.D - 4 * q)) - 1u;
            m |= b << (4 * s);
            x[s] = sx[l * p.D4 + q];
          }
        }
        const float4 *d1 = nullptr, *d2 = nullptr, *d3 = nullptr;
        if (__any_sync(0xFFFFFFFFu, m != 0u)) ok = donors(pl, tag, d1, d2, d3);
        if (!ok) m = 0u;
        uint32_t touched = 0u;
#pragma unroll
        for (int s = 0; s < V; ++s) {
          const int q = pw * 32 + lane + s * T;
          if ((m >> (4 * s)) & 15u) {
            a1[s] = ld_l2(d1 + q);
            a2[s] = ld_l2(d2 + q);
            a3[s] = ld_l2(d3 + q);
            touched |= 1u << s;
          }
        }
#pragma unroll
        for (int s = 0; s < V; ++s)
          if ((touched >> s) & 1u) mutate_slot(x[s], a1[s], a2[s], a3[s], (m >> (4 * s)) & 15u, p);
        // the trial to its buffer: the slots that crossed, and those that the
        // buffer holds from an older version
        uint32_t stale = sstale[(l * W + pw) * 32 + lane];
        const uint32_t nshift = 8u * ((sl >> 2) & 3u), put = ((stale >> nshift) & 0xFFu) | touched;
        ok = ok && wait_flag(&s_safe, safe_seen, k);
        if (ok) {
#pragma unroll
          for (int s = 0; s < V; ++s) {
            const int q = pw * 32 + lane + s * T;
            if (((put >> s) & 1u) && q < p.D4) __stcg(out + q, x[s]);
          }
        }
        // fitness, in block_row_fitness's order
        if constexpr (OBJ == kRosenbrock) {
          if (lane == 0) {
#pragma unroll
            for (int s = 0; s < V; ++s) first[s * 8 + pw] = x[s].x;
          }
          if (W > 1) named_bar_sync(1 + grp, 32 * W);
          else __syncwarp();
        }
        Acc s{0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int v = 0; v < V; ++v) {
          float nb = 0.0f;
          if constexpr (OBJ == kRosenbrock) {
            nb = __shfl_down_sync(0xFFFFFFFFu, x[v].x, 1);
            if (lane == 31) nb = (pw + 1 < nw) ? first[v * 8 + pw + 1] : (v + 1 < V ? first[(v + 1) * 8] : 0.0f);
          }
          const int q = pw * 32 + lane + v * T;
          if (q < p.D4) res_slot<OBJ>(s, x[v], nb, q, p);
        }
        res_butterfly<NS, 16>(s);
        if (W > 1) {
          float* r = red + set * 24;
          if (lane == 0) {
            r[pw] = s.a;
            if (NS > 1) r[8 + pw] = s.b;
            if (NS > 2) r[16 + pw] = s.c;
          }
          ok = agree(ok);                          // and every store of the trial precedes the row's word
          set ^= 1;                                // this set's readers are past the next barrier before it is reused
          const bool in = (lane & 7) < nw;
          s.a = in ? r[lane & 7] : 0.0f;
          if (NS > 1) s.b = in ? r[8 + (lane & 7)] : 0.0f;
          if (NS > 2) s.c = in ? r[16 + (lane & 7)] : 0.0f;
          s.a += 0.0f; s.b += 0.0f; s.c += 0.0f;
          res_butterfly<NS, 4>(s);
        } else {
          s.a += 0.0f; s.b += 0.0f; s.c += 0.0f;
          __syncwarp();
        }
        float f = finalize_fitness<OBJ>(s, p);
        if (f != f) f = __int_as_float(0x7F800000);
        if (!ok) break;
        const bool win = f < fi;
        masked += (unsigned)__popc(m);
        if (pw == 0 && lane == 0) decide(k, tag, l, sl, f, win);
        // a winner's buffer holds the row, the others miss its slots; a loser's
        // buffer misses the slots that it tried
        stale &= ~(0xFFu << nshift);
        stale |= win ? (touched * 0x01010101u) & ~(0xFFu << nshift) : touched << nshift;
        sstale[(l * W + pw) * 32 + lane] = stale;
        if (win) {
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const int q = pw * 32 + lane + v * T;
            if (q < p.D4) sx[l * p.D4 + q] = x[v];
          }
        }
      }
      // the group's reads of generation k are over once its warps are here; they
      // end early together or not at all
      __syncwarp();
      if (!agree(ok)) break;
      if (pw == 0 && lane == 0) st_flag(&s_done[grp], k + 1);
    }
  }

  // the run's state: rows to buffer 0, fitness, slot bytes, counters; the last
  // CTA closes. Unless this CTA gave up, its second helper has seen every CTA
  // finish every generation, and nobody reads the buffers any more
  masked = warp_sum_u64(masked);
  if (masked && lane == 0) atomicAdd(&s_masked, masked);
  if (wins) atomicAdd(&s_wins, wins);
  if (key != ~0ULL) {
    atomicMin(&s_key, key);
    atomicMin(&s_hist, hist);
  }
  __syncthreads();
  if (!s_dead) {
    for (int q = tid; q < rows * p.D4; q += blockDim.x) {
      const int l = q / p.D4;
      reinterpret_cast<float4*>(p.pop0 + (size_t)(row0 + l) * p.pitch)[q - l * p.D4] = sx[q];
    }
  }
  uint8_t* slot_out = p.slots + (size_t)((gen0 + rp.gens) & 1) * p.N;
  for (int l = tid; l < rows; l += blockDim.x) {
    p.fit[row0 + l] = sfit[l];
    slot_out[row0 + l] = 0;
  }
  __syncthreads();
  if (tid == 0) {
    atomicAdd(&p.st->masked, s_masked);
    if (s_wins) {
      atomicAdd(&p.st->accepts, s_wins);
      atomicMin(&p.st->best_key, s_key);
      atomicMin(&rp.rs->hist, s_hist);
    }
    __threadfence();
    s_last = atomicAdd(&p.st->done, 1u) == gridDim.x - 1 ? 1 : 0;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  const bool failed = ld_acquire(&p.st->error) != 0u;
  if (failed) {
    for (int i = tid >> 5; i < p.N; i += (int)blockDim.x >> 5) {   // a warp per row
      const uint32_t w = ld_acquire(rp.words + (size_t)i * kResWordStride);
      const float4* from = reinterpret_cast<const float4*>(buffer(w & 3u) + (size_t)i * p.pitch);
      float4* to = reinterpret_cast<float4*>(p.pop0 + (size_t)i * p.pitch);
      if (w & 3u)
        for (int q = lane; q < p.D4; q += 32) to[q] = ld_l2(from + q);
      if (lane == 0) atomicMin(&s_least, (int)(((w >> 8) - tag0) & kResTagMask));
    }
    for (int i = tid; i < 2 * p.N; i += blockDim.x) p.slots[i] = 0;
    __syncthreads();
  }
  if (tid == 0) {
    const unsigned long long bk = atomicAdd(&p.st->best_key, 0ULL), h = atomicExch(&rp.rs->hist, ~0ULL);
    const float bf = from_ordered_bits((uint32_t)(bk >> 32));
    if (bf < p.st->best_f) {
      p.st->best_f = bf;
      p.st->best_gen = gen0 + min((long long)(uint32_t)h, (long long)s_least);   // the first generation that reached the best value
    }
    p.st->gen = gen0 + s_least;
    p.st->base_row = (int)(uint32_t)(bk & 0xFFFFFFFFull);
    p.st->done = 0u;
    rp.rs->epoch = (tag0 + (uint32_t)rp.gens + 1u) & kResTagMask;
    rp.rs->failed = failed ? 1u : 0u;
    for (int c = 0; c < 8; ++c) rp.rs->ctr[c] = 0u;
  }
}

// The kernel for a crossover kind and objective; vidx indexes VecChoices.
template <int OBJ>
const void* resident_entry_obj(bool seg, int vidx) {
  if (seg) return (const void*)resident_kernel<true, OBJ, 1>;
  return vidx ? (const void*)resident_kernel<false, OBJ, 2> : (const void*)resident_kernel<false, OBJ, 1>;
}

}  // namespace de
