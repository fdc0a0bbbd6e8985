// gen_cluster.cu — many generations of a small population in one cluster.
//
// A population of up to 248 rows of D <= 128 needs 8 SMs: one warp per row, the
// row one float4 per lane in registers, its fitness beside it. The rows that
// donors are read from lie in the shared memory of the cluster's CTAs, one buffer
// per generation parity: in generation g a warp reads its donors' slots from
// buffer g & 1 of their CTAs (distributed shared memory), and stores its winner,
// trial or parent, to buffer (g + 1) & 1 of its own. One cluster barrier per
// generation orders both: a buffer is written again only after the barrier that
// every reader of it has passed. A helper warp per CTA draws donors and lengths
// two generations at a time, a barrier ahead.
//
// Nothing goes through L2 between the first and the last generation, where the
// resident kernel (gen_resident.cuh) pays three round trips and a fence each:
// NEC sphere N = 100, D = 30 2.0 us per generation there (4.5 us with a launch each),
// 1.0 us here, of which a cluster barrier is 0.28 us. What is left is the chain of
// about 200 dependent instructions.
// Sums run in gen_kernel's order, so results are de_step's bit for bit.
#include <algorithm>

#include "draws.cuh"
#include "internal.h"
#include "objectives.cuh"
#include "ptx.cuh"
#include "slot_terms.cuh"

namespace de {

namespace {

constexpr int kClCtas = 8, kClRows = 31;             // CTAs of the cluster; rows (warps) per CTA
constexpr int kClThreads = 32 * (kClRows + 1);
constexpr int kClDepth = 4;                          // generations of plans in shared memory
constexpr int kClTable = 1024;                       // NEC thresholds staged in shared memory

struct __align__(16) ClPlan {
  uint32_t donor[3];                                 // cluster addresses of the donors' rows in buffer 0
  int jrand;
  int L, pad_[3];
};

struct ClSmem {
  float4 row[2][kClRows][32];
  ClPlan plan[kClDepth][kClRows];
  uint32_t tab[kClTable];
};

__device__ __forceinline__ float4 ld_cluster(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();                                      // .aligned: the warp arrives as one
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int OBJ>
__global__ void __launch_bounds__(kClThreads, 1) cluster_kernel(const __grid_constant__ GenParams p, int xo, int gens,
                                                               int rpc, unsigned long long* hist) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  ClSmem& w = *reinterpret_cast<ClSmem*>(cl_smem);
  __shared__ unsigned long long s_masked, s_wins, s_key, s_hist;
  constexpr int NS = ObjTraits<OBJ>::kSums;
  const int lane = threadIdx.x & 31, l = threadIdx.x >> 5;
  const int row0 = blockIdx.x * rpc, rows = max(0, min(rpc, p.N - row0)), i = row0 + l;
  const bool helper = l == (int)(blockDim.x >> 5) - 1, mine = l < rows, used = lane < p.D4;
  const long long gen0 = p.st->gen;
  const bool tab_smem = xo == kNec && p.nT <= kClTable;

  float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float fi = 0.0f;
  if (mine) {
    const uint8_t s = p.slots[(size_t)(gen0 & 1) * p.N + i];
    if (used) x = reinterpret_cast<const float4*>((s ? p.pop1 : p.pop0) + (size_t)i * p.pitch)[lane];
    fi = p.fit[i];
    w.row[0][l][lane] = x;
  }
  if (tab_smem)
    for (int k = threadIdx.x; k < p.nT; k += blockDim.x) w.tab[k] = p.nec_tm1[k];
  if (threadIdx.x == 0) {
    s_masked = 0ULL;
    s_wins = 0ULL;
    s_key = ~0ULL;
    s_hist = ~0ULL;
  }
  __syncthreads();

  auto draw = [&](int k0) {                          // the helper warp: plans of generations k0 and k0 + 1
    for (int e = lane; e < 2 * rows; e += 32) {
      const int k = k0 + (e >= rows ? 1 : 0), r = e >= rows ? e - rows : e;
      const uint32_t g = (uint32_t)(gen0 + k);
      RowDraws d;
      draw_donors(p, g, row0 + r, d);
      int L = 0;
      if (xo == kNec) {
        if (p.cr_mode != kCrGeneral) L = p.cr_mode == kCrZero ? 1 : p.D;
        else if (tab_smem) L = nec_length_of<true>(p, nec_word(p, g, row0 + r), w.tab);
        else L = nec_length_of<false>(p, nec_word(p, g, row0 + r), p.nec_tm1);
      } else if (xo == kExp) {
        L = exp_walk_length(p, g, row0 + r);
      }
      ClPlan pl;
      const int dr[3] = {d.r1, d.r2, d.r3};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int rank = dr[c] / rpc;
        pl.donor[c] = map_rank(smem_u32(&w.row[0][dr[c] - rank * rpc][0]), (uint32_t)rank);
      }
      pl.jrand = d.jrand;
      pl.L = L;
      w.plan[k % kClDepth][r] = pl;
    }
  };
  if (helper) draw(0);

  constexpr uint32_t kParity = (uint32_t)sizeof(w.row[0]);
  unsigned long long masked = 0, wins = 0, key = ~0ULL, best = ~0ULL;
  for (int k = 0; k < gens; ++k) {
    cluster_sync();                                  // rows and plans of generation k are in place
    if (helper) {
      if ((k & 1) == 0 && k + 2 < gens) draw(k + 2);
      continue;
    }
    if (!mine) continue;
    const ClPlan pl = w.plan[k % kClDepth][l];
    const uint32_t at = (uint32_t)(k & 1) * kParity + 16u * (uint32_t)lane;
    unsigned m = 0u;
    const int j0 = 4 * lane;
    if (xo == kBin) {
      m = bin_mask(p, philox_block_rk(p.rk, kStreamBin, p.inst, (uint32_t)(gen0 + k), (uint32_t)i, (uint32_t)lane), lane,
                   pl.jrand);
    } else {
      int dd = j0 - pl.jrand;
      if (dd < 0) dd += p.D;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int de = dd + e;
        if (de >= p.D) de -= p.D;
        m |= (de < pl.L) ? (1u << e) : 0u;
      }
    }
    m = used ? m & ((1u << min(4, p.D - j0)) - 1u) : 0u;
    float4 t = x;
    if (m) {
      const float4 a1 = ld_cluster(pl.donor[0] + at), a2 = ld_cluster(pl.donor[1] + at),
                   a3 = ld_cluster(pl.donor[2] + at);
      mutate_slot(t, a1, a2, a3, m, p);
    }
    // fitness, in block_row_fitness's order for rows of one warp
    const float nb = __shfl_down_sync(0xFFFFFFFFu, t.x, 1);
    Acc s{0.0f, 0.0f, 0.0f};
    if (used) {
      if constexpr (OBJ == kRosenbrock) {
        if (j0 + 1 < p.D) accum_pair(s, t.x, t.y);
        if (j0 + 2 < p.D) accum_pair(s, t.y, t.z);
        if (j0 + 3 < p.D) accum_pair(s, t.z, t.w);
        if (j0 + 4 < p.D) accum_pair(s, t.w, nb);
      } else if constexpr (OBJ == kGriewank) {
        griewank_slot(s, t, j0, p);
      } else {
        accum_gene<OBJ>(s, t.x, j0, p);
        if (j0 + 1 < p.D) accum_gene<OBJ>(s, t.y, j0 + 1, p);
        if (j0 + 2 < p.D) accum_gene<OBJ>(s, t.z, j0 + 2, p);
        if (j0 + 3 < p.D) accum_gene<OBJ>(s, t.w, j0 + 3, p);
      }
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.a += __shfl_xor_sync(0xFFFFFFFFu, s.a, o);
      if (NS > 1) s.b += __shfl_xor_sync(0xFFFFFFFFu, s.b, o);
      if (NS > 2) s.c += __shfl_xor_sync(0xFFFFFFFFu, s.c, o);
    }
    s.a += 0.0f; s.b += 0.0f; s.c += 0.0f;           // the padded butterfly over the warps
    float f = finalize_fitness<OBJ>(s, p);
    if (f != f) f = __int_as_float(0x7F800000);
    const bool win = f < fi;
    if (win) {
      x = t;
      fi = f;
    }
    w.row[(k + 1) & 1][l][lane] = x;
    if (xo == kBin) masked += (unsigned)__popc(m);
    else if (lane == 0) masked += (unsigned)pl.L;
    if (win && lane == 0) {
      ++wins;
      key = min(key, best_key_of(f, i));
      best = min(best, ((unsigned long long)ordered_bits(f + 0.0f) << 32) | (unsigned)(k + 1));
    }
  }
  cluster_sync();                                    // nobody reads this CTA's rows any more

  if (mine) {
    if (used) reinterpret_cast<float4*>(p.pop0 + (size_t)i * p.pitch)[lane] = x;
    if (lane == 0) {
      p.fit[i] = fi;
      p.slots[(size_t)((gen0 + gens) & 1) * p.N + i] = 0;
    }
  }
  masked = warp_sum_u64(masked);
  if (masked && lane == 0) atomicAdd(&s_masked, masked);
  if (wins) {
    atomicAdd(&s_wins, wins);
    atomicMin(&s_key, key);
    atomicMin(&s_hist, best);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(&p.st->masked, s_masked);
    if (s_wins) {
      atomicAdd(&p.st->accepts, s_wins);
      atomicMin(&p.st->best_key, s_key);
      atomicMin(hist, s_hist);
    }
    __threadfence();
    if (atomicAdd(&p.st->done, 1u) == gridDim.x - 1) {
      __threadfence();
      const unsigned long long bk = atomicAdd(&p.st->best_key, 0ULL), h = atomicExch(hist, ~0ULL);
      const float bf = from_ordered_bits((uint32_t)(bk >> 32));
      if (bf < p.st->best_f) {
        p.st->best_f = bf;
        p.st->best_gen = gen0 + (long long)(uint32_t)h;   // the first generation that reached the best value
      }
      p.st->gen = gen0 + gens;
      p.st->base_row = (int)(uint32_t)(bk & 0xFFFFFFFFull);
      p.st->done = 0u;
    }
  }
}

using ClusterKernel = void (*)(GenParams, int, int, int, unsigned long long*);

ClusterKernel kernel_of(int obj) {
  switch (obj) {
    case kSphere: return cluster_kernel<kSphere>;
    case kRastrigin: return cluster_kernel<kRastrigin>;
    case kAckley: return cluster_kernel<kAckley>;
    case kRosenbrock: return cluster_kernel<kRosenbrock>;
    case kGriewank: return cluster_kernel<kGriewank>;
    case kElliptic: return cluster_kernel<kElliptic>;
    default: return nullptr;
  }
}

cudaLaunchConfig_t config(int N, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  const int rpc = (N + kClCtas - 1) / kClCtas;
  cfg.gridDim = dim3(kClCtas);
  cfg.blockDim = dim3(32u * (unsigned)(rpc + 1));
  cfg.dynamicSmemBytes = sizeof(ClSmem);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kClCtas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

// Where the cluster is the faster (us per generation, cluster against resident):
// NEC up to its 248 rows (N = 100, D = 30 1.0 / 2.0, N = 248, D = 128, Ackley 2.1 /
// 2.6). Binomial up to 160 rows, or shorter ones (Ackley, D = 128: N = 60 1.5 /
// 2.3, N = 130 2.1 / 2.3, N = 160 2.3 / 2.3, N = 200 2.8 / 2.3; D = 60: N = 200 2.3 / 2.4,
// N = 248 2.5 / 2.4; D = 30: N = 248 2.3 / 2.4): beyond, 8 SMs have too many genes to
// draw and sum. Exponential while its walk is short: one warp walks for all rows of a
// CTA (D = 128, N = 248: Cr = 0.3 2.4 / 2.5, 0.5 2.3 / 2.2, 0.9 6.5 / 2.2; N = 130, D = 60,
// Cr = 0.5 1.8 / 2.1).
// From two generations on it is not the slower (us per run of 2, 3, 4 generations,
// Rastrigin, cluster / a launch each: N = 100, D = 30 NEC 8.5 / 12.3, 10.3 / 18.5, 12.3 /
// 22.6; N = 248, D = 128, exponential, Cr = 0.5 12.6 / 12.6, 16.4 / 18.5, 17.9 / 22.6; N =
// 150, D = 128, binomial 12.3 / 12.4, 14.4 / 16.5, 16.5 / 21.6).
bool prepare_cluster(int xo, int obj, int vidx, int block, int N, int D4, double CR) {
  if (xo == kBin && N > 160 && D4 > 16) return false;
  if (xo == kExp && CR > 0.5) return false;
  const ClusterKernel fn = kernel_of(obj);
  if (!fn || vidx != 0 || block != 32 || D4 > 32 || N > kClCtas * kClRows) return false;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClSmem)) != cudaSuccess)
    return false;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = config(N, attr, nullptr);
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n >= 1;
}

cudaError_t launch_cluster(int xo, int obj, const GenParams& p, int gens, unsigned long long* hist, cudaStream_t s) {
  const ClusterKernel fn = kernel_of(obj);
  if (!fn) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = config(p.N, attr, s);
  return cudaLaunchKernelEx(&cfg, fn, p, xo, gens, (p.N + kClCtas - 1) / kClCtas, hist);
}

}  // namespace de
