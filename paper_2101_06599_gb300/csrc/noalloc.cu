// noalloc.cu — one DE/rand/1/NEC generation on device buffers the caller
// owns, with every piece of scratch memory in a fixed array compiled into
// the library, so that the call allocates nothing.
//
// Who needs this: callers that cannot call cudaMalloc. Examples are plug-ins
// running inside another framework that owns every device allocation and
// only lends buffers, code that must not implicitly synchronise the device
// (cudaMalloc and cudaFree may), and programs that reserve a fixed memory
// budget at start-up and may not grow it afterwards.
//
// Scratch kept in g_noalloc_scratch (fixed size, held by every GPU that loads
// the library until the process exits): the NEC thresholds T_n - 1, n = 1 ..
// D - 1. They are rewritten only when (Cr, D) differ from the last call's on
// that device (a host-side record per device), since building them takes up to
// D - 1 dependent FP64 products on one thread. Calls that overlap on the GPU
// (two streams, or two host threads) race on the array and must be serialised
// by the caller.
//
// A call whose thresholds are kept is one kernel: every row goes to pop_out,
// the trial or the parent, in the pass that evaluates it (8 bytes per gene plus
// the segment's donors). It was four operations (clear the state, copy the
// fitness, generate, copy the rejected parents): N = 100, D = 30 23.8 -> 16.0 us
// per call, N = 8192, D = 4097 113 -> 60 us (66 % of the copy bandwidth).
#include <algorithm>
#include <cmath>

#include "../../include/de.h"
#include "gen_kernel.cuh"
#include "internal.h"

namespace de {

constexpr int kNoallocMaxN = 65536;
constexpr int kNoallocMaxD = 32768;
constexpr int kNoallocMaxDevices = 64;

}  // namespace de

static __device__ __align__(256) uint32_t g_noalloc_scratch[de::kNoallocMaxD];

namespace de {

// Device address of g_noalloc_scratch per device ordinal, taken once with the
// device current (a host-side name of the array is not a device address).
static void* g_scratch_addr[kNoallocMaxDevices];
static bool g_scratch_ready[kNoallocMaxDevices];
// (Cr, D) of the thresholds the array holds, per device ordinal.
static double g_table_cr[kNoallocMaxDevices];
static int g_table_d[kNoallocMaxDevices];   // 0: no table built yet

// Writes the NEC thresholds T_n - 1 = ceil(c_n 2^32) - 1 with c_1 = Cr, c_n =
// fl(c_{n-1} Cr) in FP64, exactly as de_create computes them, and 0 from the
// first T_n <= 1 on (no word w >= 1 passes those). The products are a chain:
// thread 0 forms them, a chunk at a time, into shared memory, and all threads
// turn each chunk into thresholds.
constexpr int kNoallocChunk = 256;

__global__ void noalloc_table_kernel(uint32_t* tab, int D, double CR, int cr_mode) {
  __shared__ double cbuf[kNoallocChunk];
  __shared__ int s_ended;                           // every entry from this chunk on is 0
  double cn = CR;                                   // c_(base + 1), thread 0's running product
  if (threadIdx.x == 0) s_ended = (cr_mode != kCrGeneral);
  __syncthreads();
  for (int base = 0; base < D - 1; base += kNoallocChunk) {
    const int len = min(kNoallocChunk, D - 1 - base);
    const bool ended = s_ended != 0;
    if (threadIdx.x == 0 && !ended) {
      for (int k = 0; k < len; ++k) {
        cbuf[k] = cn;
        cn = __dmul_rn(cn, CR);
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < len; k += blockDim.x) {
      uint32_t t = 0u;
      if (!ended) {
        const double Tn = ceil(__dmul_rn(cbuf[k], 4294967296.0));
        t = (Tn > 1.0) ? (uint32_t)(Tn - 1.0) : 0u;   // T_n <= 1: no word w >= 1 passes
      }
      tab[base + k] = t;
    }
    // the products only decrease: once one is at most 2^-32, every later T_n is at most 1
    if (threadIdx.x == 0 && !ended && cbuf[len - 1] <= 0x1p-32) s_ended = 1;
    __syncthreads();
  }
}

// One generation of every row, one CTA per row, the row in registers and the
// sums in gen_kernel's order. p.pop0, p.fit: the parents (read only); row i of
// pop_out and fit_out gets the trial and its value or the parent and its own.
// The draws need no memory, so they are made before the wait for the kernel in
// front; the donors' genes are loaded together with the parent's.
template <int OBJ, int V>
__global__ void __launch_bounds__(kMaxThreads) noalloc_kernel(const __grid_constant__ GenParams p, uint32_t g,
                                                              float* __restrict__ pop_out, float* __restrict__ fit_out) {
  __shared__ RowShared sh;
  __shared__ float red[4][32];
  __shared__ float s_first[(OBJ == kRosenbrock) ? V : 1][32];
  const int i = blockIdx.x, t = threadIdx.x, T = blockDim.x;
  if (t == 0) {
    RowDraws d;
    draw_donors(p, g, i, d);
    sh.d1 = reinterpret_cast<const float4*>(p.pop0 + (size_t)d.r1 * p.pitch);
    sh.d2 = reinterpret_cast<const float4*>(p.pop0 + (size_t)d.r2 * p.pitch);
    sh.d3 = reinterpret_cast<const float4*>(p.pop0 + (size_t)d.r3 * p.pitch);
    sh.jrand = d.jrand;
  }
  const bool len = t == (T >= 64 ? 32 : 0);        // L on another warp, at the same time
  uint32_t w = 0;
  if (len) w = nec_word(p, g, i);
  griddep_wait();                                  // what is in front of the call on its stream is done
  griddep_launch_dependents();
  const float4* xrow = reinterpret_cast<const float4*>(p.pop0 + (size_t)i * p.pitch);
  float4 x[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const int q = t + k * T;
    x[k] = (q < p.D4) ? ld_stream(xrow + q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  const float fi = (t == 0) ? p.fit[i] : 0.0f;
  if (len) sh.L = nec_length_of<false>(p, w, p.nec_tm1);
  __syncthreads();

  const int jrand = sh.jrand, L = sh.L;
  unsigned crossed = 0u;                           // slots that took mutant genes
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const int q = t + k * T;
    if (q < p.D4) {
      int dd = 4 * q - jrand;
      if (dd < 0) dd += p.D;
      unsigned m = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int de = dd + e;
        if (de >= p.D) de -= p.D;
        m |= (de < L) ? (1u << e) : 0u;
      }
      m &= (1u << min(4, p.D - 4 * q)) - 1u;
      if (m) {
        const float4 a1 = ld_ro(sh.d1 + q), a2 = ld_ro(sh.d2 + q), a3 = ld_ro(sh.d3 + q);
        mutate_slot<0>(x[k], a1, a2, a3, m, p);
        crossed |= 1u << k;
      }
    }
  }
  int cnt = 0;
  const float f = block_row_fitness<OBJ, V>(x, cnt, p, s_first, red);
  if (t == 0) {
    sh.accept = (f < fi) ? 1 : 0;
    fit_out[i] = sh.accept ? f : fi;
  }
  __syncthreads();
  float4* out = reinterpret_cast<float4*>(pop_out + (size_t)i * p.pitch);
  const bool lost = sh.accept == 0;
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const int q = t + k * T;
    if (q < p.D4) {
      if (lost && ((crossed >> k) & 1u)) x[k] = ld_ro(xrow + q);   // the parent's genes again
      st_stream(out + q, x[k]);
    }
  }
}

template <int OBJ>
static cudaError_t launch_noalloc_obj(int vidx, const GenParams& p, uint32_t g, float* pop_out, float* fit_out,
                                      int block, cudaStream_t s) {
  const dim3 grid((unsigned)p.N), blk((unsigned)block);
  switch (vidx) {
    case 0: return launch_pdl(noalloc_kernel<OBJ, 1>, grid, blk, 0, s, p, g, pop_out, fit_out);
    case 1: return launch_pdl(noalloc_kernel<OBJ, 2>, grid, blk, 0, s, p, g, pop_out, fit_out);
    case 2: return launch_pdl(noalloc_kernel<OBJ, 4>, grid, blk, 0, s, p, g, pop_out, fit_out);
    case 3: return launch_pdl(noalloc_kernel<OBJ, 8>, grid, blk, 0, s, p, g, pop_out, fit_out);
    case 4: return launch_pdl(noalloc_kernel<OBJ, 16>, grid, blk, 0, s, p, g, pop_out, fit_out);
    default: return cudaErrorInvalidValue;
  }
}

static cudaError_t launch_noalloc(int obj, int vidx, const GenParams& p, uint32_t g, float* pop_out, float* fit_out,
                                  int block, cudaStream_t s) {
  switch (obj) {
    case kSphere: return launch_noalloc_obj<kSphere>(vidx, p, g, pop_out, fit_out, block, s);
    case kRastrigin: return launch_noalloc_obj<kRastrigin>(vidx, p, g, pop_out, fit_out, block, s);
    case kAckley: return launch_noalloc_obj<kAckley>(vidx, p, g, pop_out, fit_out, block, s);
    case kRosenbrock: return launch_noalloc_obj<kRosenbrock>(vidx, p, g, pop_out, fit_out, block, s);
    case kGriewank: return launch_noalloc_obj<kGriewank>(vidx, p, g, pop_out, fit_out, block, s);
    case kElliptic: return launch_noalloc_obj<kElliptic>(vidx, p, g, pop_out, fit_out, block, s);
    default: return cudaErrorInvalidValue;
  }
}

// Launch shape of the row-per-CTA kernel: the rule de_create uses by default
// (smallest float4-per-thread count whose thread count fits 256, else 512).
static void noalloc_shape(int D4, int& block, int& vidx) {
  for (int limit : {256, 512}) {
    for (int k = 0; k < 5; ++k) {
      const int V = kVecChoices[k];
      const int T = (((D4 + V - 1) / V) + 31) / 32 * 32;
      if (T <= limit) {
        block = T;
        vidx = k;
        return;
      }
    }
  }
  block = 512;
  vidx = 4;
}

}  // namespace de

using namespace de;

extern "C" int de_nec_step_noalloc(const float* pop_in, const float* fit_in, float* pop_out, float* fit_out,
                                   int32_t N, int32_t D, int32_t pitch, float F, double CR, de_objective obj,
                                   de_bounds b, uint64_t seed, int64_t generation, void* cuda_stream) {
  if (!pop_in || !fit_in || !pop_out || !fit_out) return DE_EINVAL;
  if (N < 4 || N > kNoallocMaxN || D < 1 || D > kNoallocMaxD) return DE_EINVAL;
  if (pitch < D || pitch % 4 != 0) return DE_EINVAL;
  if (((uintptr_t)pop_in | (uintptr_t)pop_out) % 16 != 0) return DE_EINVAL;
  if (pop_in == pop_out || fit_in == fit_out) return DE_EINVAL;
  if (!std::isfinite(F) || !(CR >= 0.0 && CR <= 1.0) || generation < 0) return DE_EINVAL;
  if ((int)obj < DE_OBJ_SPHERE || (int)obj > DE_OBJ_ELLIPTIC) return DE_EINVAL;
  if (!std::isfinite(b.lo) || !std::isfinite(b.hi) || !(b.lo < b.hi)) return DE_EINVAL;

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return DE_ECUDA;
  if (!g_scratch_ready[dev]) {
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_noalloc_scratch) != cudaSuccess || addr == nullptr) {
      cudaGetLastError();
      return DE_ECUDA;
    }
    g_scratch_addr[dev] = addr;
    g_scratch_ready[dev] = true;
  }
  uint32_t* table = static_cast<uint32_t*>(g_scratch_addr[dev]);
  cudaStream_t s = (cudaStream_t)cuda_stream;

  GenParams p{};
  p.pop0 = const_cast<float*>(pop_in);   // read only, as is fit
  p.fit = const_cast<float*>(fit_in);
  p.nec_tm1 = table;
  p.nT = D - 1;
  p.N = N;
  p.D = D;
  p.pitch = pitch;
  p.D4 = (D + 3) / 4;
  p.F = F;
  p.lo = b.lo;
  p.hi = b.hi;
  p.cr_mode = (CR <= 0.0) ? kCrZero : (CR >= 1.0 ? kCrOne : kCrGeneral);
  p.cr_t = (unsigned long long)std::ceil(CR * 4294967296.0);
  p.cr_lt = (uint32_t)std::min<unsigned long long>(p.cr_t, 0xFFFFFFFFull);
  p.cr_all = p.cr_t > 0xFFFFFFFFull ? 1 : 0;
  p.key = Key2{(uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32)};
  p.rk = philox_round_keys(p.key);
  p.inst = 0;
  p.ackley_b = 0.2f;
  p.ell_k = (D > 1) ? (float)(6.0 * std::log2(10.0) / (double)(D - 1)) : 0.0f;
  p.nec_k = (CR > 0.0 && CR < 1.0) ? (float)(1.0 / -std::log2(CR)) : 0.0f;

  int block = 32, vidx = 0;
  noalloc_shape(p.D4, block, vidx);
  const bool build_table = !(g_table_d[dev] == D && g_table_cr[dev] == CR);
  cudaError_t e = cudaSuccess;
  if (build_table) {
    noalloc_table_kernel<<<1, 256, 0, s>>>(table, D, CR, p.cr_mode);
    e = cudaGetLastError();
    // recorded only once the build is queued; a failed launch builds it again next time
    g_table_d[dev] = (e == cudaSuccess) ? D : 0;
    g_table_cr[dev] = CR;
  }
  if (e == cudaSuccess) e = launch_noalloc((int)obj, vidx, p, (uint32_t)generation, pop_out, fit_out, block, s);
  return e == cudaSuccess ? DE_OK : DE_ECUDA;
}
