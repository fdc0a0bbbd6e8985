// batch_seg.cu — generations of a batch whose crossovers are segments (NEC,
// classic exponential), within one run: a generation reads and writes what
// the segments touch instead of every row.
//
// A trial differs from its parent in the L genes of its segment (10 on average
// at Cr = 0.9, of up to 2048), and the FP32 fitness is the sum of 32 partial
// sums (virtual lane v: the slots v, v + 32, ... in order) by a butterfly. The
// run starts with one pass over every row (batch_seg_init_kernel) that keeps
// those 32 sums beside the row and makes both of the row's buffers equal. From
// then on (batch_seg_kernel) a generation computes again only the sums that
// hold a changed slot, and a winning trial is written as two short pieces into
// the other buffer, which lacks exactly the segment that won last and the one
// that wins now. Every value is added in the order of the other row kernels, so
// fitness, selections and populations are theirs bit for bit, and a run leaves
// nothing behind that the next call would need.
//
// Work: a warp takes a span of up to 32 rows of one instance. Lane r draws row
// r (donors, length, slot bytes, fitness: one round trip for 32 rows); then four
// rows at a time are processed by 8 lanes each, lane e computing the segment's
// e-th slot and the sum that it belongs to. Segments of more than 8 slots, and
// those that wrap around the end of a row of more than 32 slots (two of its slots
// may share a sum), take the whole warp.
//
// Bound by latency and issue (16 warps per SM, long-scoreboard and fixed-latency
// stalls; DRAM 30 % busy): 128 instances of D log-uniform in [10, 2000] (264 202
// rows, 1.9e8 genes, Cr = 0.9) 559 us per generation with the staged kernel, which
// reads every row, 164 us here; 512 instances 1579 -> 566 us. Steps: sums and
// segments in registers, 8 lanes or the warp per row 269 us; 16 lanes for 9 to 16
// slots 224 us; the slots of a sum by cp.async, all loads of a row in flight
// together 177 us; 4 lanes for up to 4 slots 164 us.
#include <algorithm>

#include "batch_plan.cuh"
#include "draws.cuh"
#include "internal.h"
#include "objectives.cuh"
#include "ptx.cuh"

namespace de {

namespace {

constexpr int kBsWarps = 4, kBsMaxK = kStageMaxD4 / 32;   // slots per sum of the longest rows

// Where a warp's rows land: the slots of each lane's sum and, for Rosenbrock,
// the gene after each.
struct SegSmem {
  float4 x[kBsMaxK][32];
  float nb[kBsMaxK][32];
};

__device__ __forceinline__ void ca4_g2s(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

struct SegCnt {
  unsigned long long kmin, masked;
  unsigned accepts;
};

// Slot q of a row (genes 4q ..) added to a virtual lane's sums; nb is gene 4q + 4.
template <int OBJ>
__device__ __forceinline__ void seg_slot(Acc& a, const float4& x, float nb, int q, const GenParams& p) {
  const int j0 = 4 * q;
  if constexpr (OBJ == kRosenbrock) {
    if (j0 + 1 < p.D) accum_pair(a, x.x, x.y);
    if (j0 + 2 < p.D) accum_pair(a, x.y, x.z);
    if (j0 + 3 < p.D) accum_pair(a, x.z, x.w);
    if (j0 + 4 < p.D) accum_pair(a, x.w, nb);
  } else {
    accum_gene<OBJ>(a, x.x, j0, p);
    if (j0 + 1 < p.D) accum_gene<OBJ>(a, x.y, j0 + 1, p);
    if (j0 + 2 < p.D) accum_gene<OBJ>(a, x.z, j0 + 2, p);
    if (j0 + 3 < p.D) accum_gene<OBJ>(a, x.w, j0 + 3, p);
  }
}

// Genes of slot q that a segment of L genes from jrand takes.
__device__ __forceinline__ unsigned seg_crossing(int q, int jrand, int L, int D) {
  unsigned m = 0u;
  int dd = 4 * q - jrand;
  if (dd < 0) dd += D;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    int de = dd + e;
    if (de >= D) de -= D;
    m |= (de < L && 4 * q + e < D) ? 1u << e : 0u;
  }
  return m;
}

// The slots whose sums a segment changes: a0 .. a0 + n0 - 1 and 0 .. n1 - 1 (for
// Rosenbrock the slot before the segment is among them).
struct SegSlots {
  int a0, n0, n1;
};
template <int OBJ>
__device__ __forceinline__ SegSlots seg_slots(int jrand, int L, const GenParams& p) {
  const int over = jrand + L - p.D;
  SegSlots s;
  s.a0 = max(0, (jrand >> 2) - (OBJ == kRosenbrock ? 1 : 0));
  s.n0 = (over > 0 ? p.D4 - 1 : (jrand + L - 1) >> 2) - s.a0 + 1;
  s.n1 = over > 0 ? min((over - 1) >> 2, s.a0 - 1) + 1 : 0;
  return s;
}

__device__ __forceinline__ bool seg_has(const SegSlots& s, int q) {
  return (q >= s.a0 && q < s.a0 + s.n0) || q < s.n1;
}

// What a lane knows of the row that it drew.
struct SegRow {
  int r1, r2, r3, L, jrand;
  uint32_t slots;                                  // slot bits of the row (0) and its donors (1-3)
  float fit;
};

template <int NS>
__device__ __forceinline__ void seg_store_sums(float* ps, int v, const Acc& a) {
  ps[v] = a.a;
  if (NS > 1) ps[32 + v] = a.b;
  if (NS > 2) ps[64 + v] = a.c;
}
template <int NS>
__device__ __forceinline__ Acc seg_load_sums(const float* ps, int v) {
  Acc a{0.0f, 0.0f, 0.0f};
  a.a = ps[v];
  if (NS > 1) a.b = ps[32 + v];
  if (NS > 2) a.c = ps[64 + v];
  return a;
}
template <int NS>
__device__ __forceinline__ void seg_add(Acc& s, const Acc& t) {
  s.a += t.a;
  if (NS > 1) s.b += t.b;
  if (NS > 2) s.c += t.c;
}
template <int NS>
__device__ __forceinline__ Acc seg_shfl(const Acc& s, int from) {
  Acc r{0.0f, 0.0f, 0.0f};
  r.a = __shfl_sync(0xFFFFFFFFu, s.a, from);
  if (NS > 1) r.b = __shfl_sync(0xFFFFFFFFu, s.b, from);
  if (NS > 2) r.c = __shfl_sync(0xFFFFFFFFu, s.c, from);
  return r;
}
template <int NS>
__device__ __forceinline__ Acc seg_xor(const Acc& s, int o) {
  Acc r{0.0f, 0.0f, 0.0f};
  r.a = __shfl_xor_sync(0xFFFFFFFFu, s.a, o);
  if (NS > 1) r.b = __shfl_xor_sync(0xFFFFFFFFu, s.b, o);
  if (NS > 2) r.c = __shfl_xor_sync(0xFFFFFFFFu, s.c, o);
  return r;
}

__device__ __forceinline__ const float4* seg_row_ptr(const GenParams& p, int buf, int i) {
  return reinterpret_cast<const float4*>((buf ? p.pop1 : p.pop0) + (size_t)i * p.pitch);
}

// Slot q of the trial of a row: the parent's slot with the segment's genes.
__device__ __forceinline__ float4 seg_trial(const GenParams& p, const SegRow& R, const float4* x, int q) {
  float4 t = ld_ro(x + q);
  const unsigned m = seg_crossing(q, R.jrand, R.L, p.D);
  if (m) {
    const float4 a1 = ld_ro(seg_row_ptr(p, (R.slots >> 1) & 1, R.r1) + q);
    const float4 a2 = ld_ro(seg_row_ptr(p, (R.slots >> 2) & 1, R.r2) + q);
    const float4 a3 = ld_ro(seg_row_ptr(p, (R.slots >> 3) & 1, R.r3) + q);
    mutate_slot<0>(t, a1, a2, a3, m, p);
  }
  return t;
}

__device__ __forceinline__ void seg_count(SegCnt& c, const GenParams& p, int i, float f, bool win, int L) {
  c.masked += (unsigned long long)L;
  if (win) {
    c.accepts += 1u;
    p.fit[i] = f;
    const unsigned long long key = best_key_of(f, i);
    c.kmin = key < c.kmin ? key : c.kmin;
  }
}

// One row on the whole warp, any segment. won: the segment that won last (the
// slots that the other buffer lacks).
template <int OBJ>
__device__ __noinline__ void seg_row_warp(const GenParams& p, uint8_t* slot_out, const SegRow R, int i, float* ps,
                                          ushort4* won, int lane, SegCnt& c) {
  constexpr int NS = ObjTraits<OBJ>::kSums;
  const SegSlots S = seg_slots<OBJ>(R.jrand, R.L, p);
  const int si = (int)(R.slots & 1u);
  const float4* x = seg_row_ptr(p, si, i);
  float4* out = const_cast<float4*>(seg_row_ptr(p, 1 - si, i));
  bool mine = false;
  for (int q = lane; q < p.D4; q += 32) mine = mine || seg_has(S, q);
  Acc a{0.0f, 0.0f, 0.0f};
  if (mine) {
    for (int q = lane; q < p.D4; q += 32) {
      float nb = 0.0f;
      if constexpr (OBJ == kRosenbrock) {
        if (q + 1 < p.D4) nb = seg_has(S, q + 1) ? seg_trial(p, R, x, q + 1).x : ld_ro(x + q + 1).x;
      }
      seg_slot<OBJ>(a, seg_has(S, q) ? seg_trial(p, R, x, q) : ld_ro(x + q), nb, q, p);
    }
  } else {
    a = seg_load_sums<NS>(ps, lane);
  }
  __syncwarp();
  Acc s = a;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) seg_add<NS>(s, seg_xor<NS>(s, o));
  float f = finalize_fitness<OBJ>(s, p);
  if (f != f) f = __int_as_float(0x7F800000);
  const bool win = f < R.fit;
  if (win) {
    const ushort4 w = *won;
    const SegSlots W{w.x, w.y, w.z};
    for (int q = lane; q < p.D4; q += 32) {
      if (seg_has(S, q)) out[q] = seg_trial(p, R, x, q);
      else if (seg_has(W, q)) out[q] = ld_ro(x + q);
    }
    if (mine) seg_store_sums<NS>(ps, lane, a);
  }
  __syncwarp();                                    // every lane has read *won
  if (lane == 0) {
    slot_out[i] = (uint8_t)(win ? 1 - si : si);
    if (win) *won = make_ushort4((unsigned short)S.a0, (unsigned short)S.n0, (unsigned short)S.n1, 0);
    seg_count(c, p, i, f, win, R.L);
  }
}

// The rows of `todo` (bit r: row r of the span, drawn by lane r as R), 32 / G at
// a time on G lanes each; their segments have at most G slots, no two of them in
// one sum.
template <int OBJ, int G>
__device__ __forceinline__ void seg_rows(const GenParams& p, uint8_t* slot_out, const BatchSpan& sp, const SegRow& R,
                                         unsigned todo, float* sums, int stride, ushort4* won, int lane, SegSmem& w, SegCnt& c) {
  constexpr int NS = ObjTraits<OBJ>::kSums, kEach = 32 / G;
  const int e = lane & (G - 1), top = lane & ~(G - 1), grp = lane / G;
  while (todo) {
    // group j takes the j-th row that is left
    unsigned left = todo;
    int r = 0;
    bool act = false;
#pragma unroll
    for (int j = 0; j < kEach; ++j) {
      if (grp == j) {
        act = left != 0u;
        r = act ? __ffs((int)left) - 1 : 0;
      }
      left &= left - 1u;
    }
    todo = left;
    SegRow Q;
    Q.r1 = __shfl_sync(0xFFFFFFFFu, R.r1, r);
    Q.r2 = __shfl_sync(0xFFFFFFFFu, R.r2, r);
    Q.r3 = __shfl_sync(0xFFFFFFFFu, R.r3, r);
    Q.L = __shfl_sync(0xFFFFFFFFu, R.L, r);
    Q.jrand = __shfl_sync(0xFFFFFFFFu, R.jrand, r);
    Q.slots = __shfl_sync(0xFFFFFFFFu, R.slots, r);
    Q.fit = __shfl_sync(0xFFFFFFFFu, R.fit, r);
    const int i = sp.row0 + r;
    const SegSlots S = seg_slots<OBJ>(Q.jrand, max(Q.L, 1), p);
    const int n = act ? S.n0 + S.n1 : 0;
    const bool slot = e < n;                       // this lane has a slot of the segment
    const int q = slot ? (e < S.n0 ? S.a0 + e : e - S.n0) : 0, v = q & 31;
    const int si = (int)(Q.slots & 1u);
    const float4* x = seg_row_ptr(p, si, i);
    float4* out = const_cast<float4*>(seg_row_ptr(p, 1 - si, i));
    float* ps = sums + (size_t)(sp.plan0 + r) * stride;
    const unsigned m = slot ? seg_crossing(q, Q.jrand, Q.L, p.D) : 0u;
    // all of a lane's loads before anything is used: the slots of its sum to
    // shared memory, the rest to registers
    if (slot) {
      int k = 0;
      for (int o = v; o < p.D4; o += 32, ++k) {
        ca16_g2s(smem_u32(&w.x[k][lane]), x + o);
        if constexpr (OBJ == kRosenbrock) {
          if (o + 1 < p.D4) ca4_g2s(smem_u32(&w.nb[k][lane]), x + o + 1);
        }
      }
    }
    ca_commit();
    float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f), a1 = t, a2 = t, a3 = t;
    Acc old[kEach];
    ushort4 w4 = make_ushort4(0, 0, 0, 0);
    if (m) {
      a1 = ld_ro(seg_row_ptr(p, (Q.slots >> 1) & 1, Q.r1) + q);
      a2 = ld_ro(seg_row_ptr(p, (Q.slots >> 2) & 1, Q.r2) + q);
      a3 = ld_ro(seg_row_ptr(p, (Q.slots >> 3) & 1, Q.r3) + q);
    }
#pragma unroll
    for (int j = 0; j < kEach; ++j) old[j] = act ? seg_load_sums<NS>(ps, e + G * j) : Acc{0.0f, 0.0f, 0.0f};
    if (act) w4 = won[sp.plan0 + r];
    ca_wait_all();
    if (slot) t = w.x[q >> 5][lane];
    if (m) mutate_slot<0>(t, a1, a2, a3, m, p);
    __syncwarp();
    float nx = __shfl_down_sync(0xFFFFFFFFu, t.x, 1);
    if constexpr (OBJ == kRosenbrock) {
      const float tx0 = __shfl_sync(0xFFFFFFFFu, t.x, top);
      if (slot && (e == S.n0 - 1 || e == n - 1)) nx = w.nb[q >> 5][lane];
      if (e == n - 1 && q + 1 == S.a0) nx = tx0;   // the slots after the wrap end where the first one begins
    }
    // the sum that the slot belongs to, its slots in order
    Acc es{0.0f, 0.0f, 0.0f};
    if (slot) {
      int k = 0;
      for (int o = v; o < p.D4; o += 32, ++k) {
        float nb = 0.0f;
        if constexpr (OBJ == kRosenbrock) nb = o == q ? nx : w.nb[k][lane];   // not used past the row's end
        seg_slot<OBJ>(es, o == q ? t : w.x[k][lane], nb, o, p);
      }
    }
    __syncwarp();
    // lane e holds the sums of virtual lanes e, e + G, ...
#pragma unroll
    for (int j = 0; j < kEach; ++j) {
      const int vj = e + G * j;
      int from = (vj - S.a0) & 31;
      bool changed = from < S.n0 && act;
      if (vj < S.n1) {
        from = S.n0 + vj;
        changed = act;
      }
      const Acc u = seg_shfl<NS>(es, top | (from & (G - 1)));
      if (changed) old[j] = u;
    }
#pragma unroll
    for (int o = kEach / 2; o > 0; o >>= 1)        // strides 16 .. G of the butterfly
#pragma unroll
      for (int j = 0; j < o; ++j) seg_add<NS>(old[j], old[j + o]);
    Acc s0 = old[0];
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) seg_add<NS>(s0, seg_xor<NS>(s0, o));
    float f = finalize_fitness<OBJ>(s0, p);
    if (f != f) f = __int_as_float(0x7F800000);
    const bool win = act && f < Q.fit;
    if (win) {
      const SegSlots W{w4.x, w4.y, w4.z};
      if (slot) {
        out[q] = t;
        seg_store_sums<NS>(ps, v, es);
      }
      for (int k = e; k < W.n0 + W.n1; k += G) {
        const int o = k < W.n0 ? W.a0 + k : k - W.n0;
        if (!seg_has(S, o)) out[o] = ld_ro(x + o);
      }
    }
    if (act && e == 0) {
      slot_out[i] = (uint8_t)(win ? 1 - si : si);
      if (win) won[sp.plan0 + r] = make_ushort4((unsigned short)S.a0, (unsigned short)S.n0, (unsigned short)S.n1, 0);
      seg_count(c, p, i, f, win, Q.L);
    }
    __syncwarp();
  }
}

template <int OBJ>
__device__ __forceinline__ void seg_span(const BatchInst& I, const BatchSpan& sp, float* sums, int stride,
                                         ushort4* won, int lane, SegSmem& w, SegCnt& c) {
  const GenParams& p = I.g;
  const long long gen = p.st->gen;
  uint8_t* slot_out = p.slots + (size_t)((gen + 1) & 1) * p.N;
  SegRow R{};
  if (lane < sp.rows) {
    RowDraws d;
    int L;
    const int i = sp.row0 + lane;
    row_draws(I, gen, i, nullptr, d, L);
    const RowPlan32 pl = row_plan(p, gen, i, d, L);
    R.r1 = pl.r1; R.r2 = pl.r2; R.r3 = pl.r3; R.L = L; R.jrand = pl.jrand;
    R.slots = (pl.slots & 1u) | ((pl.slots >> 7) & 2u) | ((pl.slots >> 14) & 4u) | ((pl.slots >> 21) & 8u);
    R.fit = pl.fit_i;
  }
  // a segment's slots belong to sums of their own unless it wraps and its end
  // reaches, 32 slots apart, into its start
  const SegSlots S = seg_slots<OBJ>(R.jrand, max(R.L, 1), p);
  const bool apart = p.D4 <= 32 || S.n1 == 0 || ((S.a0 >> 5) == ((p.D4 - 1) >> 5) && (S.a0 & 31) >= S.n1);
  const int n = (lane < sp.rows && apart) ? S.n0 + S.n1 : 33;
  const unsigned to4 = __ballot_sync(0xFFFFFFFFu, n <= 4), to8 = __ballot_sync(0xFFFFFFFFu, n <= 8) & ~to4,
                 to16 = __ballot_sync(0xFFFFFFFFu, n <= 16) & ~(to4 | to8);
  seg_rows<OBJ, 4>(p, slot_out, sp, R, to4, sums, stride, won, lane, w, c);
  seg_rows<OBJ, 8>(p, slot_out, sp, R, to8, sums, stride, won, lane, w, c);
  seg_rows<OBJ, 16>(p, slot_out, sp, R, to16, sums, stride, won, lane, w, c);
  for (unsigned rest = __ballot_sync(0xFFFFFFFFu, lane < sp.rows) & ~(to4 | to8 | to16); rest; rest &= rest - 1u) {
    const int r = __ffs((int)rest) - 1;
    SegRow Q;
    Q.r1 = __shfl_sync(0xFFFFFFFFu, R.r1, r);
    Q.r2 = __shfl_sync(0xFFFFFFFFu, R.r2, r);
    Q.r3 = __shfl_sync(0xFFFFFFFFu, R.r3, r);
    Q.L = __shfl_sync(0xFFFFFFFFu, R.L, r);
    Q.jrand = __shfl_sync(0xFFFFFFFFu, R.jrand, r);
    Q.slots = __shfl_sync(0xFFFFFFFFu, R.slots, r);
    Q.fit = __shfl_sync(0xFFFFFFFFu, R.fit, r);
    seg_row_warp<OBJ>(p, slot_out, Q, sp.row0 + r, sums + (size_t)(sp.plan0 + r) * stride, won + sp.plan0 + r, lane, c);
  }
}

__global__ void __launch_bounds__(32 * kBsWarps, 4) batch_seg_kernel(const BatchInst* __restrict__ insts,
                                                                 const BatchSpan* __restrict__ spans, int nspans,
                                                                 float* sums, int stride, ushort4* won,
                                                                 DevState* states, int n_inst, unsigned* done) {
  griddep_wait();                                  // the previous generation has closed
  griddep_launch_dependents();
  extern __shared__ __align__(16) unsigned char seg_smem[];
  SegSmem& w = reinterpret_cast<SegSmem*>(seg_smem)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31, k = blockIdx.x * kBsWarps + (threadIdx.x >> 5);
  if (k < nspans) {
    const BatchSpan sp = spans[k];
    const BatchInst& I = insts[sp.inst];
    SegCnt c{~0ull, 0ull, 0u};
    switch (I.obj) {
      case kSphere: seg_span<kSphere>(I, sp, sums, stride, won, lane, w, c); break;
      case kRastrigin: seg_span<kRastrigin>(I, sp, sums, stride, won, lane, w, c); break;
      case kAckley: seg_span<kAckley>(I, sp, sums, stride, won, lane, w, c); break;
      case kRosenbrock: seg_span<kRosenbrock>(I, sp, sums, stride, won, lane, w, c); break;
      case kGriewank: seg_span<kGriewank>(I, sp, sums, stride, won, lane, w, c); break;
      default: seg_span<kElliptic>(I, sp, sums, stride, won, lane, w, c); break;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long ko = __shfl_xor_sync(0xFFFFFFFFu, c.kmin, o);
      c.kmin = ko < c.kmin ? ko : c.kmin;
      c.masked += __shfl_xor_sync(0xFFFFFFFFu, c.masked, o);
      c.accepts += __shfl_xor_sync(0xFFFFFFFFu, c.accepts, o);
    }
    if (lane == 0) {
      if (c.accepts) {
        atomicMin(&I.g.st->best_key, c.kmin);
        atomicAdd(&I.g.st->accepts, (unsigned long long)c.accepts);
      }
      atomicAdd(&I.g.st->masked, c.masked);
    }
  }
  // the last warp closes every instance
  unsigned last = 0u;
  if (lane == 0) {
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x * kBsWarps - 1u ? 1u : 0u;
  }
  if (__shfl_sync(0xFFFFFFFFu, last, 0)) {
    __threadfence();
    for (int n = lane; n < n_inst; n += 32) close_instance(states[n], 0);
    if (lane == 0) *done = 0u;
  }
}

// Start of a run, one warp per row: the 32 sums of every row, and the row into
// its other buffer.
template <int OBJ>
__device__ __forceinline__ void seg_init_row(const GenParams& p, int i, float* ps, int lane) {
  const int si = p.slots[(size_t)(p.st->gen & 1) * p.N + i];
  const float4* x = seg_row_ptr(p, si, i);
  float4* out = const_cast<float4*>(seg_row_ptr(p, 1 - si, i));
  Acc a{0.0f, 0.0f, 0.0f};
  for (int q = lane; q < p.D4; q += 32) {
    const float4 xv = x[q];
    float nb = 0.0f;
    if constexpr (OBJ == kRosenbrock) nb = q + 1 < p.D4 ? x[q + 1].x : 0.0f;
    out[q] = xv;
    seg_slot<OBJ>(a, xv, nb, q, p);
  }
  seg_store_sums<ObjTraits<OBJ>::kSums>(ps, lane, a);
}

__global__ void __launch_bounds__(32 * kBsWarps) batch_seg_init_kernel(const BatchInst* __restrict__ insts,
                                                                      const BatchSpan* __restrict__ spans, int nspans,
                                                                      float* sums, int stride, ushort4* won) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const BatchSpan sp = spans[blockIdx.x];
  const BatchInst& I = insts[sp.inst];
  for (int r = warp; r < sp.rows; r += kBsWarps) {
    float* ps = sums + (size_t)(sp.plan0 + r) * stride;
    const int i = sp.row0 + r;
    switch (I.obj) {
      case kSphere: seg_init_row<kSphere>(I.g, i, ps, lane); break;
      case kRastrigin: seg_init_row<kRastrigin>(I.g, i, ps, lane); break;
      case kAckley: seg_init_row<kAckley>(I.g, i, ps, lane); break;
      case kRosenbrock: seg_init_row<kRosenbrock>(I.g, i, ps, lane); break;
      case kGriewank: seg_init_row<kGriewank>(I.g, i, ps, lane); break;
      default: seg_init_row<kElliptic>(I.g, i, ps, lane); break;
    }
    if (lane == 0) won[sp.plan0 + r] = make_ushort4(0, 0, 0, 0);
  }
}

}  // namespace

cudaError_t prepare_batch_seg() {
  return cudaFuncSetAttribute(batch_seg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kBsWarps * (int)sizeof(SegSmem));
}

cudaError_t launch_batch_seg_init(const BatchInst* insts, const BatchSeg& b, cudaStream_t s) {
  batch_seg_init_kernel<<<(unsigned)b.nspans, 32 * kBsWarps, 0, s>>>(insts, b.spans, b.nspans, b.sums, b.stride, b.won);
  return cudaGetLastError();
}

cudaError_t launch_batch_seg(const BatchInst* insts, const BatchSeg& b, DevState* states, int n_inst, cudaStream_t s) {
  return launch_pdl(batch_seg_kernel, dim3((unsigned)((b.nspans + kBsWarps - 1) / kBsWarps)), dim3(32 * kBsWarps),
                    kBsWarps * sizeof(SegSmem), s, insts, b.spans, b.nspans, b.sums, b.stride, b.won, states, n_inst, b.done);
}

}  // namespace de
