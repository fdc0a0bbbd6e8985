// sr_kernels.cu — generation of the shifted-rotated objectives.
//
// One generation = sr_trial_kernel (draws, crossover, mutation, clipping as
// in the separable path; the trial row is written to the row's other slot
// buffer, so acceptance is a slot flip; a = u - o and |a|^2, and for the BF16
// path the split operands bf16(a), bf16(a - bf16(a))), then the product
// Z = A R^T with a fused g(z) epilogue (this file: FP32 SIMT; sr_tc.cu:
// tcgen05), then sr_select_kernel (strict '<' decisions, or interval
// decisions with a per-row error bound on the BF16 path: rows whose interval
// straddles the parent's go to an FP32 re-evaluation with this file's GEMM
// and sr_resolve_kernel), then sr_finish_kernel (FP64 incumbent when due, and
// the close of the generation).
//
// The FP32 GEMM accumulates every z_ik in one fixed order (j ascending, one
// FMA per term, one thread per element) and reduces g(z) over each 64-column
// tile in one fixed order, so a row's value does not depend on which other
// rows share its tile: re-evaluating a row reproduces the FP32 path bit for
// bit.
#include "draws.cuh"
#include "gen_kernel.cuh"
#include "internal.h"
#include "sr_common.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace de {

// ---------------------------------------------------------------------------
// trials: one warp per row, 8 rows per CTA. The warp issues its first parent
// loads, lane 0 draws the donors and L (Philox, slot lookups) and broadcasts
// them, then the lanes stream the row 4 genes at a time: crossover mask,
// mutation and clip of masked genes, the trial into the other slot, a = u - o
// with |a|^2, and on the BF16 path the split operands as packed 8-byte
// stores. Mask counts go to the state with one atomic per CTA.
// ---------------------------------------------------------------------------
constexpr int kTrialWarps = 8, kTrialUnroll = 4;

template <int XO>
__global__ void __launch_bounds__(kTrialWarps * 32, 4) sr_trial_kernel(const __grid_constant__ SrParams sp) {
  griddep_wait();                                  // the previous kernel of the generation is done
  griddep_launch_dependents();
  const GenParams& p = sp.g;
  __shared__ int wcnt[kTrialWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * kTrialWarps + warp;
  const long long gen = p.st->gen;
  const uint32_t g = (uint32_t)gen;
  const uint8_t* slot_in = p.slots + (size_t)(gen & 1) * p.N;
  int Lrow = 0;
  if (i < p.N) {                                   // warp-uniform
    const int si = slot_in[i];
    const float4* xrow = reinterpret_cast<const float4*>((si ? p.pop1 : p.pop0) + (size_t)i * p.pitch);
    float4* trow = reinterpret_cast<float4*>((si ? p.pop0 : p.pop1) + (size_t)i * p.pitch);
    float4 x[kTrialUnroll];
#pragma unroll
    for (int u = 0; u < kTrialUnroll; ++u) {
      const int q = lane + 32 * u;
      x[u] = (q < p.D4) ? ld_stream(xrow + q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    RowDraws d{};
    unsigned long long pd1 = 0, pd2 = 0, pd3 = 0;
    if (lane == 0) {
      draw_donors(p, g, i, d);
      if constexpr (XO == kNec) d.L = nec_length(p, g, i);
      else if constexpr (XO == kExp) d.L = exp_walk_length(p, g, i);
      else d.L = 0;
      pd1 = (unsigned long long)((slot_in[d.r1] ? p.pop1 : p.pop0) + (size_t)d.r1 * p.pitch);
      pd2 = (unsigned long long)((slot_in[d.r2] ? p.pop1 : p.pop0) + (size_t)d.r2 * p.pitch);
      pd3 = (unsigned long long)((slot_in[d.r3] ? p.pop1 : p.pop0) + (size_t)d.r3 * p.pitch);
    }
    const int jrand = __shfl_sync(0xFFFFFFFFu, d.jrand, 0);
    const int L = __shfl_sync(0xFFFFFFFFu, d.L, 0);
    const float4* d1 = reinterpret_cast<const float4*>(__shfl_sync(0xFFFFFFFFu, pd1, 0));
    const float4* d2 = reinterpret_cast<const float4*>(__shfl_sync(0xFFFFFFFFu, pd2, 0));
    const float4* d3 = reinterpret_cast<const float4*>(__shfl_sync(0xFFFFFFFFu, pd3, 0));
    int cnt = 0;
    float nrm = 0.0f, amx = 0.0f;
    for (int q0 = 0; q0 < p.D4; q0 += 32 * kTrialUnroll) {
      if (q0 > 0) {
#pragma unroll
        for (int u = 0; u < kTrialUnroll; ++u) {
          const int q = q0 + lane + 32 * u;
          x[u] = (q < p.D4) ? ld_stream(xrow + q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
      }
#pragma unroll
      for (int u = 0; u < kTrialUnroll; ++u) {
        const int q = q0 + lane + 32 * u;
        if (q >= p.D4) continue;
        const int j0 = 4 * q;
        unsigned m = 0u;
        if constexpr (XO == kBin) {
          const uint4 w = philox_block(p.key, kStreamBin, p.inst, g, (uint32_t)i, (uint32_t)q);
          m |= ((unsigned long long)w.x < p.cr_t || j0 + 0 == jrand) ? 1u : 0u;
          m |= ((unsigned long long)w.y < p.cr_t || j0 + 1 == jrand) ? 2u : 0u;
          m |= ((unsigned long long)w.z < p.cr_t || j0 + 2 == jrand) ? 4u : 0u;
          m |= ((unsigned long long)w.w < p.cr_t || j0 + 3 == jrand) ? 8u : 0u;
        } else {
          int dd = j0 - jrand;
          if (dd < 0) dd += p.D;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            int de = dd + e;
            if (de >= p.D) de -= p.D;
            m |= (de < L) ? (1u << e) : 0u;
          }
        }
        m &= (1u << min(4, p.D - j0)) - 1u;
        float4 v = x[u];
        if (m) {
          const float4 a1 = ld_ro(d1 + q), a2 = ld_ro(d2 + q), a3 = ld_ro(d3 + q);
          mutate_slot(v, a1, a2, a3, m, p);
        }
        if constexpr (XO == kBin) cnt += __popc(m);
        st_stream(trow + q, v);
        if (p.dbg_trial) reinterpret_cast<float4*>(p.dbg_trial + (size_t)i * p.pitch)[q] = v;
        float a[4];
        if (j0 + 4 <= p.D) {                       // a full slot: o by one 16-byte load
          const float4 o4 = __ldg(reinterpret_cast<const float4*>(sp.shift) + q);
          a[0] = __fsub_rn(v.x, o4.x);
          a[1] = __fsub_rn(v.y, o4.y);
          a[2] = __fsub_rn(v.z, o4.z);
          a[3] = __fsub_rn(v.w, o4.w);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = j0 + e;
            a[e] = (j < p.D) ? __fsub_rn(lane_of(v, e), sp.shift[j]) : 0.0f;
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          nrm = fmaf(a[e], a[e], nrm);
          amx = fmaxf(amx, fabsf(a[e]));
        }
        if (sp.prec != 0) {                        // D % 256 == 0 on this path: 8-byte aligned
          uint32_t h[4], l[4];
          if (sp.prec == 3) {                      // FP16 halves of 2^sa a (the scaling is exact)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float as = a[e] * sp.a_scale;
              const __half hi = __float2half_rn(as);
              const __half lo = __float2half_rn(__fsub_rn(as, __half2float(hi)));
              h[e] = __half_as_ushort(hi);
              l[e] = __half_as_ushort(lo);
            }
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const __nv_bfloat16 hi = __float2bfloat16_rn(a[e]);
              const __nv_bfloat16 lo = __float2bfloat16_rn(__fsub_rn(a[e], __bfloat162float(hi)));
              h[e] = __bfloat16_as_ushort(hi);
              l[e] = __bfloat16_as_ushort(lo);
            }
          }
          *reinterpret_cast<uint2*>(sp.a_hi + (size_t)i * p.D + j0) = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
          *reinterpret_cast<uint2*>(sp.a_lo + (size_t)i * p.D + j0) = make_uint2(l[0] | (l[1] << 16), l[2] | (l[3] << 16));
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      nrm += __shfl_xor_sync(0xFFFFFFFFu, nrm, o);
      amx = fmaxf(amx, __shfl_xor_sync(0xFFFFFFFFu, amx, o));
      cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
    }
    Lrow = (XO == kBin) ? cnt : L;
    if (lane == 0) {
      sp.norm2[i] = nrm;
      sp.amax[i] = amx;
      if (p.dbg_draws) {
        int* o = p.dbg_draws + 5 * (size_t)i;
        o[0] = d.r1; o[1] = d.r2; o[2] = d.r3; o[3] = d.jrand; o[4] = Lrow;
      }
    }
  }
  if (lane == 0) wcnt[warp] = Lrow;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long c = 0;
    for (int w = 0; w < kTrialWarps; ++w) c += (unsigned long long)wcnt[w];
    atomicAdd(&p.st->masked, c);
  }
}

// ---------------------------------------------------------------------------
// FP32 product with the fitness epilogue
// mode 0: all rows, trial rows (other slot); 1: all rows, parent rows;
// 2: the ambiguous entries (row << 1 | parent flag), partials to part2_*.
//
// Every z_ik is one FMA chain over j ascending (zero padding past D adds
// fma(0, 0, acc) = acc), and every 64-column partial sums g over the column
// tile the same way in both kernels below: each of 16 lanes adds its 4
// consecutive columns in order, then an xor tree over the 16 lanes
// (offsets 8, 4, 2, 1). So a row's partials do not depend on the kernel, the
// tile or the other rows: the re-evaluation kernel reproduces the all-rows
// kernel bit for bit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ const float* sr_row_ptr(const SrParams& sp, int mode, int e, const uint8_t* slot_in) {
  const GenParams& p = sp.g;
  int r = e, parent = (mode == 1);
  if (mode == 2) {
    r = sp.amb[e] >> 1;
    parent = sp.amb[e] & 1;
  }
  const int s = slot_in[r];
  const int buf = parent ? s : 1 - s;
  return (buf ? p.pop1 : p.pop0) + (size_t)r * p.pitch;
}

// One row's 4 columns of a 64-column tile, reduced over the tile's 16 lanes
// (all 32 lanes of the warp call it; lanes 16..31 reduce their own tile row).
__device__ __forceinline__ float sr_tile_reduce(const SrParams& sp, const float z[4], int c0) {
  const GenParams& p = sp.g;
  float sg = 0.0f;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int n = c0 + b;
    if (n < p.D) {
      const float w = sr_weight(sp.obj, n, p.ell_k);
      sg += sr_g(sp.obj, z[b], w);
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    sg += __shfl_xor_sync(0xFFFFFFFFu, sg, o);
  }
  return sg;
}

// All rows (modes 0 and 1): tiles of 8 RT rows x 64 columns, 128 threads, RT
// rows x 4 columns per thread (thread tx of 16 has the columns 4 tx .. 4 tx + 3,
// the lane layout above), K in steps of 16. x and R^T arrive two steps ahead
// by cp.async (read one step ahead through registers, the loads were the first
// stall); a step before its use each thread turns the x it copied itself into
// a = fl(x - o), K-major.
//
// Bound by the FP32 pipe (2 N D^2 flop; 128 FMA per SM and clock, busy 67 % of
// the time here, 50 % before) and, next, by shared-memory loads. The products
// are fma.rn.f32x2 on pairs of rows: the same pipe rate in half the issue slots,
// so that the shared loads and the operand copies issue beside them; each half is
// its element's own fmaf chain over j ascending. N = 4096, D = 1024, a generation:
// 271 us with 128 x 128 tiles of scalar FMAs (256 tiles: two on some SMs, one on
// the others), 189 us with 592 tiles of 112 x 64, four on almost every SM.
constexpr int kGbN = 64, kGbK = 16, kGbThreads = 128, kGbLdB = kGbN + 4;

__device__ __forceinline__ void ffma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}

// VEC: D % 4 == 0, 16-byte copies of x, o and R^T; else single elements.
template <int RT, bool VEC>
__global__ void __launch_bounds__(kGbThreads, 4) sr_gemm_fp32_kernel(const __grid_constant__ SrParams sp, int mode) {
  griddep_wait();                                  // the previous kernel of the generation is done
  griddep_launch_dependents();
  static_assert(RT % 2 == 0 && RT >= 4 && RT <= 16, "pairs of rows");
  constexpr int M = 8 * RT, LdA = M + 4, P = RT / 2, kQuads = RT / 4;
  constexpr int kLoads = (M * 4 + kGbThreads - 1) / kGbThreads;   // four-element pieces of a step's rows per thread
  const GenParams& p = sp.g;
  __shared__ __align__(16) float As[2][kGbK][LdA];
  __shared__ __align__(16) float Bs[3][kGbK][kGbLdB];
  __shared__ __align__(16) float4 Xs[2][kLoads][kGbThreads];
  __shared__ __align__(16) float Os[4][kGbK];
  __shared__ const float* rowp[M];

  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int n0 = blockIdx.x * kGbN, r0 = blockIdx.y * M;
  const long long gen = p.st->gen;
  const uint8_t* slot_in = p.slots + (size_t)(gen & 1) * p.N;
  for (int m = t; m < M; m += kGbThreads) rowp[m] = (r0 + m < p.N) ? sr_row_ptr(sp, mode, r0 + m, slot_in) : nullptr;
  __syncthreads();

  // step k0 to stage `at` of x (two) and `bt` of R^T (three); past D: zeros.
  // Four lanes copy a row's 16 elements, four each
  const int ak = 4 * (t & 3);                      // this thread's elements of every row
  auto issue = [&](int k0, int at, int bt) {
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int m = (t + kGbThreads * u) >> 2, j = k0 + ak;
      const float* xa = m < M ? rowp[m] : nullptr;
      const uint32_t dst = sr_smem_u32(&Xs[at][u][t]);
      if constexpr (VEC) {
        const bool in = xa && j < p.D;
        cp_async16(dst, in ? xa + j : sp.shift, in ? 16u : 0u);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool in = xa && j + e < p.D;
          cp_async4(dst + 4 * e, in ? xa + j + e : sp.shift, in ? 4u : 0u);
        }
      }
    }
    constexpr int kW = VEC ? 4 : 1;
#pragma unroll
    for (int u = 0; u < kGbK * kGbN / kW / kGbThreads; ++u) {
      const int c = t + kGbThreads * u, k = c / (kGbN / kW), n = (c % (kGbN / kW)) * kW;
      const bool in = k0 + k < p.D && n0 + n < p.D;
      const float* src = in ? sp.rot_t + (size_t)(k0 + k) * p.D + n0 + n : sp.rot_t;
      if constexpr (VEC) cp_async16(sr_smem_u32(&Bs[bt][k][n]), src, in ? 16u : 0u);
      else cp_async4(sr_smem_u32(&Bs[bt][k][n]), src, in ? 4u : 0u);
    }
  };
  // o of a step, three steps ahead: other threads read it, so it takes a barrier
  // after it has landed
  auto issue_o = [&](int step) {
    if (t < kGbK) {
      const bool in = step * kGbK + t < p.D;
      cp_async4(sr_smem_u32(&Os[step & 3][t]), in ? sp.shift + step * kGbK + t : sp.shift, in ? 4u : 0u);
    }
  };
  auto form_a = [&](int step, int at, int buf) {   // x and o are zero past D, and so is a
    const float4 o = *reinterpret_cast<const float4*>(&Os[step & 3][ak]);
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int m = (t + kGbThreads * u) >> 2;
      if (m >= M) continue;
      const float4 x = Xs[at][u][t];
      As[buf][ak + 0][m] = __fsub_rn(x.x, o.x);
      As[buf][ak + 1][m] = __fsub_rn(x.y, o.y);
      As[buf][ak + 2][m] = __fsub_rn(x.z, o.z);
      As[buf][ak + 3][m] = __fsub_rn(x.w, o.w);
    }
  };

  // rows of thread ty: 32 i + 4 ty .. + 3 for i < RT / 4, then (RT = 4 i + 2)
  // 32 i + 2 ty, + 1; acc holds them in pairs
  unsigned long long acc[P][4];
#pragma unroll
  for (int a = 0; a < P; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0ULL;

  issue(0, 0, 0);
  issue_o(0);
  issue_o(1);
  cp_async_commit();
  if (kGbK < p.D) issue(kGbK, 1, 1);
  issue_o(2);
  cp_async_commit();
  cp_async_wait<1>();
  __syncthreads();
  form_a(0, 0, 0);
  __syncthreads();
  const int steps = (p.D + kGbK - 1) / kGbK;
  int bt = 0;                                      // stage of R^T of this step
  for (int step = 0; step < steps; ++step) {
    const int buf = step & 1, bt2 = bt == 0 ? 2 : bt - 1;
    if (step + 2 < steps) issue((step + 2) * kGbK, buf, bt2);   // both stages were read before the last barrier
    issue_o(step + 3);
    cp_async_commit();
#pragma unroll
    for (int kk = 0; kk < kGbK; ++kk) {
      unsigned long long a[P];
#pragma unroll
      for (int i = 0; i < kQuads; ++i) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&As[buf][kk][32 * i + 4 * ty]);
        a[2 * i] = v.x;
        a[2 * i + 1] = v.y;
      }
      if constexpr (RT % 4 == 2) a[P - 1] = *reinterpret_cast<const unsigned long long*>(&As[buf][kk][32 * kQuads + 2 * ty]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[bt][kk][4 * tx]);
      const unsigned long long b[4] = {pack2(b4.x, b4.x), pack2(b4.y, b4.y), pack2(b4.z, b4.z), pack2(b4.w, b4.w)};
#pragma unroll
      for (int i = 0; i < P; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) ffma2(acc[i][c], a[i], b[c]);
    }
    cp_async_wait<1>();                            // step + 1 has landed
    if (step + 1 < steps) form_a(step + 1, buf ^ 1, buf ^ 1);
    __syncthreads();
    bt = bt == 2 ? 0 : bt + 1;
  }
  cp_async_wait<0>();

#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int m = (RT % 4 == 2 && i == P - 1) ? 32 * kQuads + 2 * ty : 32 * (i >> 1) + 4 * ty + 2 * (i & 1);
    const float2 z0 = unpack2(acc[i][0]), z1 = unpack2(acc[i][1]), z2 = unpack2(acc[i][2]), z3 = unpack2(acc[i][3]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float z[4] = {h ? z0.y : z0.x, h ? z1.y : z1.x, h ? z2.y : z2.x, h ? z3.y : z3.x};
      const int e = r0 + m + h;
      const float sg = sr_tile_reduce(sp, z, n0 + 4 * tx);
      if (tx == 0 && e < p.N) sp.part_g[(size_t)e * sp.nct2 + blockIdx.x] = sg;
    }
  }
}

// The ambiguous entries (mode 2; split-operand paths only, so D % 256 == 0):
// work items of 4 WE entries x 64 columns, taken by groups of 4 warps: a warp has
// WE entries (WE = 2, 4 or 8), a lane the columns 2 lane and 2 lane + 1 of the
// tile for all of them, so a k costs a broadcast of the entries' a, 8 bytes of R^T
// per lane and 2 WE FMAs. Each group has its own 3-stage cp.async ring of 64-deep
// slices of the entries' rows of x, o and rows of R^T and its own named barrier.
// Once a stage has landed, each warp forms a = fl(x - o) K-major for its own
// entries (so only a warp barrier follows): every z stays one FMA chain over j
// ascending. The list is short (a few hundred entries) and each chain is D FMAs
// long, so the time is set by the busiest SM, and there by the latency of a warp's
// step: about 27, 37 and 52 cycles per k for WE = 2, 4 and 8, one warp per
// scheduler (ls_warp_entries has the rule). Generations by WE = 2, 4, 8, us: 71 rows
// (FP16 Rastrigin, N = 4096, D = 1024) 63.4, 59.2, 62.2 and 58.3 by the rule, which
// follows each list; 141 rows (BF16) 86.3, 71.2, 73.2 and 70.3; 9 rows (N = 1000, D
// = 512) 29.9, 31.7, 36.3; 563 rows (N = 16384) 300, 237, 210. Two groups per CTA and a ring per
// group that needs more than half an SM's shared memory for the pair put exactly
// one CTA on each SM; the grid is one CTA per SM, group g of CTA b takes items b +
// g * grid, b + (2 + g) * grid, ..., so the first items of a short list land on
// distinct SMs whatever order the CTAs are placed in.
constexpr int kLsMaxE = 32, kLsN = 64, kLsK = 64, kLsStages = 3, kLsGroupThreads = 128, kLsGroups = 2;
constexpr int kLsThreads = kLsGroups * kLsGroupThreads;
constexpr int kLsLdX = kLsK + 4, kLsLdB = kLsN + 4;   // floats per row
constexpr int kLsGroupFloats = kLsStages * (kLsMaxE * kLsLdX + kLsK + kLsK * kLsLdB) + kLsK * (kLsMaxE + 4);
constexpr size_t kLsSmem = sizeof(float) * (size_t)kLsGroups * kLsGroupFloats;
static_assert(kLsSmem > 114 * 1024 && kLsSmem <= 227 * 1024, "one CTA per SM");

// Entries per warp for a list of n entries and ct column tiles on `grid` CTAs:
// the least estimated time: a round of items (one group per SM) at the cost above,
// two rounds side by side 1.6 of it.
__device__ __forceinline__ int ls_warp_entries(int n, int ct, int grid) {
  int best = 8;
  float cost = 1e30f;
  const float per_k[3] = {27.0f, 37.0f, 52.0f};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int we = 2 << c, items = (n + 4 * we - 1) / (4 * we) * ct, rounds = (items + grid - 1) / grid;
    const float t = per_k[c] * (1.6f * (float)(rounds / 2) + (float)(rounds % 2));
    if (t < cost) {
      cost = t;
      best = we;
    }
  }
  return best;
}

__device__ __forceinline__ void ls_group_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(kLsGroupThreads) : "memory");
}

template <int WE>
__device__ __forceinline__ void ls_items(const SrParams& sp, float* ls_smem, const float** rowp, int nrows) {
  constexpr int kLsE = 4 * WE, kLsLdA = kLsE + 4;
  const GenParams& p = sp.g;
  const int g = threadIdx.x / kLsGroupThreads, t = threadIdx.x % kLsGroupThreads;
  float* Xs = ls_smem + (size_t)g * kLsGroupFloats;  // [stage][entry][kLsLdX]: raw x
  float* Os = Xs + kLsStages * kLsE * kLsLdX;      // [stage][k]: o
  float* Bs = Os + kLsStages * kLsK;               // [stage][k][kLsLdB]: R^T rows
  float* As = Bs + kLsStages * kLsK * kLsLdB;      // [k][kLsLdA]: a per entry
  const int lane = t & 31, warp = t >> 5;
  const int ebase = warp * WE;               // the warp's first entry in the tile
  const long long gen = p.st->gen;
  const uint8_t* slot_in = p.slots + (size_t)(gen & 1) * p.N;
  const int KS = p.D / kLsK, ctiles = p.D / kLsN;
  const int items = ((nrows + kLsE - 1) / kLsE) * ctiles;
  int n0 = 0;

  // one stage: x 4 WE entries x 16 chunks of 16 bytes, o 16 chunks, R^T 64 rows x
  // 16 chunks (8 per thread); entries past the list read zeros
  auto issue = [&](int step) {
    const int st = step % kLsStages, k0 = step * kLsK;
#pragma unroll
    for (int i = 0; i < (kLsE * kLsK / 4) / kLsGroupThreads; ++i) {
      const int qx = t + kLsGroupThreads * i, m = qx / (kLsK / 4), c = (qx % (kLsK / 4)) * 4;
      const float* xa = rowp[m];
      cp_async16(sr_smem_u32(Xs + (st * kLsE + m) * kLsLdX + c), xa ? xa + k0 + c : sp.shift, xa ? 16u : 0u);
    }
    if (t < kLsK / 4) cp_async16(sr_smem_u32(Os + st * kLsK + 4 * t), sp.shift + k0 + 4 * t, 16u);
#pragma unroll
    for (int i = 0; i < (kLsK * kLsN / 4) / kLsGroupThreads; ++i) {
      const int q = t + kLsGroupThreads * i, kr = q >> 4, c = (q & 15) * 4;
      cp_async16(sr_smem_u32(Bs + (st * kLsK + kr) * kLsLdB + c), sp.rot_t + (size_t)(k0 + kr) * p.D + n0 + c, 16u);
    }
  };

  for (int item = blockIdx.x + g * gridDim.x; item < items; item += kLsGroups * gridDim.x) {
    const int r0 = (item / ctiles) * kLsE, ct = item % ctiles;
    n0 = ct * kLsN;
    ls_group_sync(g);                              // rowp and the stages are reused
    if (t < kLsE) rowp[t] = (r0 + t < nrows) ? sr_row_ptr(sp, 2, r0 + t, slot_in) : nullptr;
    ls_group_sync(g);
#pragma unroll
    for (int s0 = 0; s0 < kLsStages - 1; ++s0) {
      if (s0 < KS) issue(s0);
      cp_async_commit();
    }
    float acc[WE][2];
#pragma unroll
    for (int e = 0; e < WE; ++e) acc[e][0] = acc[e][1] = 0.0f;
    for (int step = 0; step < KS; ++step) {
      cp_async_wait<kLsStages - 2>();
      ls_group_sync(g);                             // this stage landed; every lane is done with the
                                                    // slot refilled next
      if (step + kLsStages - 1 < KS) issue(step + kLsStages - 1);
      cp_async_commit();
      const int st = step % kLsStages;
#pragma unroll
      for (int kk = lane; kk < kLsK; kk += 32) {   // a = fl(x - o): k = kk, the warp's WE entries
        const float* xs = Xs + (st * kLsE + ebase) * kLsLdX + kk;
        const float o = Os[st * kLsK + kk];
#pragma unroll
        for (int e = 0; e < WE; e += 2)
          *reinterpret_cast<float2*>(As + kk * kLsLdA + ebase + e) =
              make_float2(__fsub_rn(xs[e * kLsLdX], o), __fsub_rn(xs[(e + 1) * kLsLdX], o));
      }
      __syncwarp();                                 // a of the warp's entries, written by the warp
      const float* as = As + ebase;
      const float* bs = Bs + st * kLsK * kLsLdB + 2 * lane;
#pragma unroll
      for (int k = 0; k < kLsK; ++k) {
        const float2 bv = *reinterpret_cast<const float2*>(bs + k * kLsLdB);
        float av[WE];
        if constexpr (WE == 2) {
          const float2 a = *reinterpret_cast<const float2*>(as + k * kLsLdA);
          av[0] = a.x; av[1] = a.y;
        } else {
#pragma unroll
          for (int e = 0; e < WE; e += 4) {
            const float4 a = *reinterpret_cast<const float4*>(as + k * kLsLdA + e);
            av[e] = a.x; av[e + 1] = a.y; av[e + 2] = a.z; av[e + 3] = a.w;
          }
        }
#pragma unroll
        for (int e = 0; e < WE; ++e) {
          acc[e][0] = fmaf(av[e], bv.x, acc[e][0]);
          acc[e][1] = fmaf(av[e], bv.y, acc[e][1]);
        }
      }
    }                                               // (the next step's group barrier orders the As reuse)
    cp_async_wait<0>();
    // the layout of the tile reduction: lane tx of each half has the columns 4 tx
    // .. 4 tx + 3, the lower half of one entry and the upper half of the next
    const int tx = lane & 15;
#pragma unroll
    for (int e = 0; e < WE; e += 2) {
      float z[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float a = __shfl_sync(0xFFFFFFFFu, acc[e][c & 1], 2 * tx + (c >> 1));
        const float b = __shfl_sync(0xFFFFFFFFu, acc[e + 1][c & 1], 2 * tx + (c >> 1));
        z[c] = lane < 16 ? a : b;
      }
      const int ent = r0 + ebase + e + (lane >> 4);
      const float sg = sr_tile_reduce(sp, z, n0 + 4 * tx);
      if (tx == 0 && ent < nrows) sp.part2_g[(size_t)ent * sp.nct2 + ct] = sg;
    }
  }
}

__global__ void __launch_bounds__(kLsThreads, 1) sr_gemm_fp32_list_kernel(const __grid_constant__ SrParams sp) {
  griddep_wait();                                  // the previous kernel of the generation is done
  griddep_launch_dependents();
  extern __shared__ __align__(16) float ls_smem[];
  __shared__ const float* rowp[kLsGroups][kLsMaxE];
  const float** mine = rowp[threadIdx.x / kLsGroupThreads];
  const int nrows = (int)*sp.amb_count;
  switch (ls_warp_entries(nrows, sp.g.D / kLsN, (int)gridDim.x)) {
    case 2: ls_items<2>(sp, ls_smem, mine, nrows); break;
    case 4: ls_items<4>(sp, ls_smem, mine, nrows); break;
    default: ls_items<8>(sp, ls_smem, mine, nrows); break;
  }
}

cudaError_t prepare_sr_list(int* ctas) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  *ctas = sms > 0 ? sms : 1;
  return cudaFuncSetAttribute(sr_gemm_fp32_list_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLsSmem);
}

// R^T for the list kernel's contiguous B tiles (once, at set-up).
__global__ void sr_transpose_kernel(const float* __restrict__ rot, float* __restrict__ rot_t, int D) {
  __shared__ float tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = by + r, j = bx + threadIdx.x;
    tile[r][threadIdx.x] = (k < D && j < D) ? rot[(size_t)k * D + j] : 0.0f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int j = bx + r, k = by + threadIdx.x;
    if (j < D && k < D) rot_t[(size_t)j * D + k] = tile[threadIdx.x][r];
  }
}

cudaError_t launch_sr_transpose(const float* rot, float* rot_t, int D, cudaStream_t s) {
  const dim3 grid((unsigned)((D + 31) / 32), (unsigned)((D + 31) / 32)), blk(32, 8);
  sr_transpose_kernel<<<grid, blk, 0, s>>>(rot, rot_t, D);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// decisions
// ---------------------------------------------------------------------------
// The partials of a row are loaded 16 at a time before they are added in order: a
// load per addition was a round trip to L2 per tile in one dependent row (D /
// 256 in the selection, D / 64 twice in the resolution). tsq, if wanted: the sum
// of their squares.
template <bool kSquares = false>
__device__ __forceinline__ float sr_row_value(const float* pg, int nct, float* tsq = nullptr) {
  float f = 0.0f, s = 0.0f;
  for (int c0 = 0; c0 < nct; c0 += 16) {
    float v[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = (c0 + c < nct) ? pg[c0 + c] : 0.0f;
#pragma unroll
    for (int c = 0; c < 16; ++c)
      if (c0 + c < nct) {
        f += v[c];
        if constexpr (kSquares) s = fmaf(v[c], v[c], s);
      }
  }
  if constexpr (kSquares) *tsq = s;
  return (f != f) ? __int_as_float(0x7F800000) : f;
}

// Bound on |f_split - f_FP32path| of one row (BF16 or FP16 split operands)
// from n^2 = |a|_2^2, the row's sum_k w_k |z_k| and its value f.
// Worst case: |dz_k| <= delta = c n + delta_abs for every k; Rastrigin |dg| <=
// delta (2|z| + 20 pi + 3 delta); elliptic |dg_k| <= w_k delta (2|z_k| +
// delta); plus the reductions' relative error.
// Probabilistic: the first-order change sum_k g'(z_k) dz_k is a sum of
// independent zero-mean terms (operand-split residuals, accumulation
// roundings) whose bounds give the standard deviations; the g evaluations and
// the sums over k add theirs (tsq: the sum of the squares of the row's tile
// partials). The tensor cores' FP32 accumulator rounds toward zero, which
// shrinks every |z_k| a little: half an ulp, at most 2^-24 |z_k|, per MMA step
// of the leading product on average bounds that bias, and the correction
// products' steps, on partial sums ~2 u_s smaller, add a term in n H.
// Second-order terms are bounded by the mean of |dz|_2^2 with a factor 2.
__device__ __forceinline__ float sr_bound(int obj, float norm2, float amax, float sumw, float f, float tsq, int D,
                                         const SrBound& b) {
  if (b.mode == 1) {
    const float delta = b.delta_per_norm * sqrtf(norm2) * 1.0001f + b.delta_abs;
    float e;
    if (obj == kSrElliptic) e = delta * (2.0f * sumw + delta * b.sum_w);
    else e = delta * (2.0f * sumw + (float)D * (20.0f * 3.14159274f + 3.0f * delta));
    return (e + b.rel * fabsf(f)) * 1.001f;
  }
  const float n = sqrtf(norm2) * 1.0001f;
  const float af = fabsf(f);
  // |g'(z)| for Rastrigin: 2|z| + 20 pi |sin 2 pi z| <= min(2|z| + 20 pi, (2 + 40 pi^2) |z|)
  const float H = (obj == kSrElliptic) ? 2.0f * sqrtf(b.wmax * af * 1.0001f)
                                       : fminf(2.0002f * n + b.hconst, 396.7843f * n);
  const float rep = fmaf(b.rep_k, amax * 1.0001f, b.rep_f);
  const float s_rep = 1.7320509f * rep * H, s_acc = b.acc_c * n * H;
  const float s_ev = b.eval_c * af + b.sum_u * sqrtf(b.sum_f2 * af * af + b.sum_t2 * tsq);
  const float sig = sqrtf(s_rep * s_rep + s_acc * s_acc + s_ev * s_ev);
  const float bias = b.bias_c * ((obj == kSrElliptic) ? 2.0f * af : n * H) + b.bias_c2 * n * H;
  // A row with a = 0 exactly has z = 0 exactly on both paths: B = 0. Any other
  // row keeps a floor, so that terms underflowing in FP32 never leave B = 0.
  const float B = (b.lambda * sig + bias + b.quad_a * rep * rep + b.quad_b * norm2) * 1.001f;
  return amax > 0.0f ? fmaxf(B, 1e-36f) : B;
}

// Warp-aggregated updates of the generation's counters: one atomic per warp
// instead of one per row (every lane of the warp calls these).
__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xFFFFFFFFu, v, o);
    v = w < v ? w : v;
  }
  return v;
}

__device__ __forceinline__ void warp_note_accepts(DevState* st, bool acc, unsigned long long key) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, acc);
  if (m == 0u) return;                             // uniform across the warp
  const unsigned long long k = warp_min_u64(acc ? key : ~0ull);
  if ((threadIdx.x & 31) == __ffs(m) - 1) {
    atomicMin(&st->best_key, k);
    atomicAdd(&st->accepts, (unsigned long long)__popc(m));
  }
}

// One row per thread (the grid covers N once).
__global__ void sr_select_kernel(const __grid_constant__ SrParams sp, SrBound bnd) {
  griddep_wait();                                  // the previous kernel of the generation is done
  griddep_launch_dependents();
  const GenParams& p = sp.g;
  const long long gen = p.st->gen;
  const uint8_t* slot_in = p.slots + (size_t)(gen & 1) * p.N;
  uint8_t* slot_out = p.slots + (size_t)((gen + 1) & 1) * p.N;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  if (i == 0) *sp.finish_due = (sp.inc_every > 0 && (gen + 1) % sp.inc_every == 0) ? 1 : 0;
  int decision = 0;                                // 1 accept, 0 reject, 2 ambiguous
  float f = 0.0f, bx = 0.0f;
  if (i < p.N) {
    const int si = slot_in[i];
    const float fx = p.fit[i];
    bx = sp.fit_err[i];
    const float norm2 = sp.norm2[i], amax = sp.amax[i];
    float bu = 0.0f, tsq;                          // sum of the tile partials' squares
    f = sr_row_value<true>(sp.part_g + (size_t)i * sp.nct, sp.nct, &tsq);
    if (sp.prec != 0) {
      float sw = 0.0f;
      if (bnd.mode == 1)
        for (int c = 0; c < sp.nct; ++c) sw += sp.part_w[(size_t)i * sp.nct + c];
      bu = sr_bound(sp.obj, norm2, amax, sw, f, tsq * 1.0001f, p.D, bnd);
    }
    if (bu == 0.0f && bx == 0.0f) decision = (f < fx) ? 1 : 0;
    else if (f + bu < fx - bx) decision = 1;
    else if (f - bu >= fx + bx) decision = 0;
    else decision = 2;
    if (decision == 1) {
      slot_out[i] = (uint8_t)(1 - si);
      p.fit[i] = f;
      sp.fit_err[i] = bu;
    } else {
      slot_out[i] = (uint8_t)si;
    }
    if (p.dbg_ftrial) p.dbg_ftrial[i] = f;
    if (p.dbg_accept) p.dbg_accept[i] = (uint8_t)(decision == 1);
  }
  warp_note_accepts(p.st, decision == 1, best_key_of(f, i));
  // ambiguous rows: the trial, and the parent when its stored value is inexact,
  // in consecutive entries; one reservation per warp
  const unsigned need = (decision == 2) ? (bx > 0.0f ? 2u : 1u) : 0u;
  unsigned incl = need;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += v;
  }
  const unsigned total = __shfl_sync(0xFFFFFFFFu, incl, 31);
  if (total > 0u) {                                // uniform across the warp
    const unsigned rows = __popc(__ballot_sync(0xFFFFFFFFu, need > 0u));
    unsigned base = 0u;
    if (lane == 31) {
      base = atomicAdd(sp.amb_count, total);
      atomicAdd(&p.st->reselected, (unsigned long long)rows);
    }
    base = __shfl_sync(0xFFFFFFFFu, base, 31);
    if (need > 0u) {
      const unsigned k = base + incl - need;
      sp.amb[k] = i << 1;                          // the trial
      if (need == 2u) sp.amb[k + 1] = (i << 1) | 1;  // and the parent
    }
  }
}

// Ambiguous rows: decide with FP32-path values of the trial (and the parent).
// One entry per thread (the grid covers 2N entries once).
__global__ void sr_resolve_kernel(const __grid_constant__ SrParams sp) {
  griddep_wait();                                  // the previous kernel of the generation is done
  griddep_launch_dependents();
  const GenParams& p = sp.g;
  const long long gen = p.st->gen;
  const uint8_t* slot_in = p.slots + (size_t)(gen & 1) * p.N;
  uint8_t* slot_out = p.slots + (size_t)((gen + 1) & 1) * p.N;
  const unsigned n = *sp.amb_count;
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x * blockDim.x >= n) return;        // uniform across the CTA
  bool acc = false;
  float fu = 0.0f;
  int i = 0;
  if (e < n && !(sp.amb[e] & 1)) {                 // parents are read by their trial's entry
    i = sp.amb[e] >> 1;
    const int si = slot_in[i];
    const float fp = p.fit[i];
    const bool parent = e + 1 < n && sp.amb[e + 1] == ((i << 1) | 1);
    fu = sr_row_value(sp.part2_g + (size_t)e * sp.nct2, sp.nct2);
    const float fe = parent ? sr_row_value(sp.part2_g + (size_t)(e + 1) * sp.nct2, sp.nct2) : fp;
    if (parent) {
      p.fit[i] = fe;                               // the parent's exact FP32-path value
      sp.fit_err[i] = 0.0f;
    }
    acc = fu < fe;
    if (acc) {
      slot_out[i] = (uint8_t)(1 - si);
      p.fit[i] = fu;
      sp.fit_err[i] = 0.0f;
    }
    if (p.dbg_ftrial) p.dbg_ftrial[i] = fu;
    if (p.dbg_accept) p.dbg_accept[i] = (uint8_t)acc;
  }
  warp_note_accepts(p.st, acc, best_key_of(fu, i));
}

// Initial evaluation (always the FP32 product, whose partials have nct2
// columns): fit = sum of partials, fit_err = 0, best key.
__global__ void sr_store_eval_kernel(const __grid_constant__ SrParams sp) {
  const GenParams& p = sp.g;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.N; i += gridDim.x * blockDim.x) {
    const float f = sr_row_value(sp.part_g + (size_t)i * sp.nct2, sp.nct2);
    p.fit[i] = f;
    sp.fit_err[i] = 0.0f;
    atomicMin(&p.st->best_key, best_key_of(f, i));
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_sr_trial(int xo, int /*vidx*/, const SrParams& sp, int /*block*/, cudaStream_t s) {
  const unsigned grid = (unsigned)((sp.g.N + kTrialWarps - 1) / kTrialWarps);
  if (xo == kBin) return launch_pdl(sr_trial_kernel<kBin>, dim3(grid), dim3(kTrialWarps * 32), 0, s, sp);
  if (xo == kExp) return launch_pdl(sr_trial_kernel<kExp>, dim3(grid), dim3(kTrialWarps * 32), 0, s, sp);
  return launch_pdl(sr_trial_kernel<kNec>, dim3(grid), dim3(kTrialWarps * 32), 0, s, sp);
}

template <int RT>
static cudaError_t launch_gemm_rows(dim3 grid, bool vec, const SrParams& sp, int mode, cudaStream_t s) {
  // Not with programmatic dependent launch: CTAs that start while the trial
  // kernel still fills the SMs are placed where room is left, several to an SM
  // and none on others, and stay there (N = 1000, D = 1024: 65 us alone, 130 us so).
  if (vec) sr_gemm_fp32_kernel<RT, true><<<grid, kGbThreads, 0, s>>>(sp, mode);
  else sr_gemm_fp32_kernel<RT, false><<<grid, kGbThreads, 0, s>>>(sp, mode);
  return cudaGetLastError();
}

cudaError_t launch_sr_gemm_fp32(const SrParams& sp, int mode, int max_rows, cudaStream_t s) {
  const unsigned gx = (unsigned)((sp.g.D + kGbN - 1) / kGbN);
  if (mode == 2) {                                // split-operand paths: D % 256 == 0
    if (sp.g.D % kLsN != 0) return cudaErrorInvalidValue;
    const long long items = (long long)((max_rows + 7) / 8) * (sp.g.D / kLsN);   // of the smallest tiles
    const int grid = (int)std::max(1LL, std::min((long long)sp.list_ctas, items));
    return launch_pdl(sr_gemm_fp32_list_kernel, dim3((unsigned)grid), dim3(kLsThreads), kLsSmem, s, sp);
  }
  // Rows per tile (8 RT): every SM works through ceil(tiles / SMs) of them, each
  // taking about RT + 1.5 (the loads and copies of a step do not shrink with RT).
  // us per generation by RT = 16, 14, 12, 8, 4: N = 4096, D = 1024 204, 190, 194,
  // 191, 248; N = 1000, D = 512 47, 44, 38, 31, 31; N = 16384, D = 1024 657, 687,
  // 646, 687, 921; N = 700, D = 300 34, 32, 28, 24, 20.
  const int sms = sp.sm_count > 0 ? sp.sm_count : 1;
  int best = 16;
  double cost = 1e30;
  for (int rt : {16, 14, 12, 8, 4}) {
    const long long tiles = (long long)gx * ((max_rows + 8 * rt - 1) / (8 * rt));
    const double c = (double)((tiles + sms - 1) / sms) * (rt + 1.5);
    if (c < cost) {
      cost = c;
      best = rt;
    }
  }
  const dim3 grid(gx, (unsigned)((max_rows + 8 * best - 1) / (8 * best)));
  const bool vec = sp.g.D % 4 == 0;
  switch (best) {
    case 16: return launch_gemm_rows<16>(grid, vec, sp, mode, s);
    case 14: return launch_gemm_rows<14>(grid, vec, sp, mode, s);
    case 12: return launch_gemm_rows<12>(grid, vec, sp, mode, s);
    case 8: return launch_gemm_rows<8>(grid, vec, sp, mode, s);
    default: return launch_gemm_rows<4>(grid, vec, sp, mode, s);
  }
}

cudaError_t launch_sr_select(const SrParams& sp, const SrBound& b, cudaStream_t s) {
  return launch_pdl(sr_select_kernel, dim3((sp.g.N + 255) / 256), dim3(256), 0, s, sp, b);
}

cudaError_t launch_sr_resolve(const SrParams& sp, cudaStream_t s) {
  return launch_pdl(sr_resolve_kernel, dim3((2 * sp.g.N + 255) / 256), dim3(256), 0, s, sp);
}

cudaError_t launch_sr_store_eval(const SrParams& sp, cudaStream_t s) {
  sr_store_eval_kernel<<<(sp.g.N + 255) / 256, 256, 0, s>>>(sp);
  return cudaGetLastError();
}

}  // namespace de

namespace de {

// R -> hi(R), lo(R) = the rounded remainder: BF16 halves of R, or FP16
// halves of 2^sr R (scale = 2^sr, exact).
__global__ void sr_split_kernel(const float* rot, uint16_t* hi, uint16_t* lo, size_t n, int fp16, float scale) {
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    const float r = rot[k];
    if (fp16) {
      const float rs = r * scale;
      const __half h = __float2half_rn(rs);
      hi[k] = __half_as_ushort(h);
      lo[k] = __half_as_ushort(__float2half_rn(__fsub_rn(rs, __half2float(h))));
    } else {
      const __nv_bfloat16 h = __float2bfloat16_rn(r);
      hi[k] = __bfloat16_as_ushort(h);
      lo[k] = __bfloat16_as_ushort(__float2bfloat16_rn(__fsub_rn(r, __bfloat162float(h))));
    }
  }
}

cudaError_t launch_sr_split_rotation(const float* rot, uint16_t* hi, uint16_t* lo, size_t n, bool fp16, float scale,
                                     cudaStream_t s) {
  sr_split_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, s>>>(rot, hi, lo, n, fp16 ? 1 : 0,
                                                                                     scale);
  return cudaGetLastError();
}

// The incumbent in FP64 (the only FP64 arithmetic on the GPU), fused with
// the close of the generation. Generation g' = g + 1 when closing (g itself
// for the initial evaluation); every `every` generations the best row's
// objective is recomputed as z = R (x - o) and sum g(z) in FP64: one warp per
// z_k (coalesced reads of row k of R, lanes over j, a fixed shuffle tree),
// g(z_k) to inc_part[k]. The last CTA to finish (a ticket) sums inc_part in a
// fixed order, so the value does not depend on scheduling, and then closes
// the generation: best value and generation, the counter, the ambiguous list.
// Every CTA reads the state before it takes its ticket, and only the last
// one writes it.
constexpr int kIncWarps = 8;

// The close of a generation: best value and its generation, the counter, the
// base row of the next generation, an empty ambiguous list.
__device__ __forceinline__ void sr_close_generation(DevState* st, long long gnext, unsigned* amb_count) {
  const float bf = from_ordered_bits((uint32_t)(st->best_key >> 32));
  if (bf < st->best_f) {
    st->best_f = bf;
    st->best_gen = gnext;
  }
  st->gen = gnext;
  st->base_row = (int)(uint32_t)(st->best_key & 0xFFFFFFFFull);
  *amb_count = 0u;
}

__global__ void __launch_bounds__(kIncWarps * 32) sr_finish_kernel(const __grid_constant__ SrParams sp, int every,
                                                                  int close) {
  griddep_wait();                                  // the previous kernel of the generation is done
  griddep_launch_dependents();
  const GenParams& p = sp.g;
  // Closing a generation: whether the incumbent is due was recorded by this
  // generation's selection kernel, so that CTA 0 may close the generation
  // (write the counter) alone while the other CTAs are still deciding.
  // Without a close nothing writes the counter.
  const bool due = close ? (*sp.finish_due != 0) : (every > 0 && p.st->gen % every == 0);
  if (!due && !close) return;                       // uniform across the grid
  if (!due) {                                       // nothing to re-evaluate: CTA 0 closes alone
    if (blockIdx.x == 0 && threadIdx.x == 0) sr_close_generation(p.st, p.st->gen + 1, sp.amb_count);
    return;
  }
  const long long gen = p.st->gen;                  // written only by the last CTA below
  const long long gnext = close ? gen + 1 : gen;
  const int idx = (int)(uint32_t)(p.st->best_key & 0xFFFFFFFFull);
  const bool have = due && idx >= 0 && idx < p.N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (have) {
    const int si = p.slots[(size_t)(gnext & 1) * p.N + idx];
    const float* x = (si ? p.pop1 : p.pop0) + (size_t)idx * p.pitch;
    const int k = blockIdx.x * kIncWarps + warp;
    if (k < p.D) {
      const float* r = sp.rot + (size_t)k * p.D;
      double z = 0.0;
      for (int j = lane; j < p.D; j += 32) z = fma((double)r[j], (double)x[j] - (double)sp.shift[j], z);
      for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
      if (lane == 0) {
        double gk;
        if (sp.obj == kSrElliptic) {
          const double c = (p.D > 1) ? exp2((double)k * (6.0 * 3.321928094887362 / (double)(p.D - 1))) : 1.0;
          gk = c * z * z;
        } else {
          gk = z * z - 10.0 * cos(2.0 * 3.141592653589793 * z) + 10.0;
        }
        sp.inc_part[k] = gk;
      }
    }
  }
  __shared__ unsigned ticket;
  __shared__ double red[kIncWarps * 32];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) ticket = atomicAdd(sp.inc_count, 1u);
  __syncthreads();
  if (ticket != gridDim.x - 1) return;
  __threadfence();
  if (have) {
    double acc = 0.0;
    for (int q = threadIdx.x; q < p.D; q += blockDim.x) acc += __ldcg(sp.inc_part + q);
    red[threadIdx.x] = acc;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (have) {
      double f = 0.0;
      for (int w = 0; w < (int)blockDim.x; ++w) f += red[w];
      p.st->incumbent_f64 = f;
      p.st->incumbent_gen = gnext;
    }
    if (close) sr_close_generation(p.st, gnext, sp.amb_count);
    *sp.inc_count = 0u;
  }
}

cudaError_t launch_sr_finish(const SrParams& sp, int every, bool close, cudaStream_t s) {
  const unsigned grid = (unsigned)((sp.g.D + kIncWarps - 1) / kIncWarps);
  return launch_pdl(sr_finish_kernel, dim3(grid), dim3(kIncWarps * 32), 0, s, sp, every, close ? 1 : 0);
}

}  // namespace de
