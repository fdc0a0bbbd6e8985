// gen_resident.cu — launch shape and launch of the resident generation kernel.
#include <algorithm>

#include "gen_resident.cuh"

namespace de {

static const void* entry_of(bool seg, int obj, int vidx) {
  switch (obj) {
    case kSphere: return resident_entry_sphere(seg, vidx);
    case kRastrigin: return resident_entry_rastrigin(seg, vidx);
    case kAckley: return resident_entry_ackley(seg, vidx);
    case kRosenbrock: return resident_entry_rosenbrock(seg, vidx);
    case kGriewank: return resident_entry_griewank(seg, vidx);
    case kElliptic: return resident_entry_elliptic(seg, vidx);
    default: return nullptr;
  }
}

static int sums_of(int obj) {
  return obj == kAckley ? ObjTraits<kAckley>::kSums : (obj == kGriewank ? ObjTraits<kGriewank>::kSums : 1);
}

// Where one launch for many generations is the faster (both sides measured at
// the sizes named, us per generation, resident against a launch each):
//  - exp and NEC: one slot per thread (D <= 1024) and segments that mostly fit
//    a slot per lane, 1 / (1 - Cr) <= 40 genes or rows of at most 32 slots.
//    N = 1024, D = 1000: Cr = 0.9 2.5 / 5.7, Cr = 0.95 (exp) 2.6 / 12.8, Cr =
//    0.975 2.8 / 5.7, 0.99 3.8 / 5.7, 0.999 7.0 / 6.0 (the line is on the safe side); two
//    slots per thread lose (N = 300, D = 1100 6.9 / 5.3).
//  - binomial: rows of one warp (N = 5000, D = 128 7.0 / 11.5), or all rows of
//    a CTA at once: N = 600, D = 500 (16 warps) 2.6 / 5.0. Beyond, a CTA's rows take
//    turns: N = 700 (20 warps) 4.6 / 4.9, N = 500, D = 1000, Ackley (32) 5.2 / 5.4, N =
//    1024, D = 1000 (56) 9.0 / 7.4.
// Populations that shared memory does not hold launch each generation.
//
// The fewest generations that pay for the launch, which loads the rows, forms every
// sum and writes all back: four (us per run of 3, 4, 8 generations, Rastrigin, resident /
// a launch each: N = 250, D = 30 NEC 18.5 / 18.5, 20.6 / 22.8, 29.1 / 43.1; N = 1024, D =
// 1000 22.6 / 20.6, 26.2 / 26.7, 36.3 / 49.2; binomial N = 300, D = 500 18.1 / 16.5, 20.4 /
// 21.7, 29.0 / 40.7; N = 300, D = 1500 20.5 / 20.6, 24.5 / 26.5, 36.6 / 49.1). Three with
// eight rows per CTA or more, where a launch costs more (at 2 and 3: N = 2000, D = 64 NEC
// 16.7 / 16.5, 20.4 / 22.6, D = 128 binomial 16.1 / 15.9, 18.5 / 21.9). Five for segments
// with one row per CTA and more than 128 slots (N = 64, D = 1000 at 4 and 5: 23.3 / 22.5,
// 26.4 / 26.7), and where one warp walks for many rows (exponential, Cr = 0.9, N = 5000, D
// = 120 at 4, 5 and 8: 54.0 / 51.0, 62.0 / 62.1, 84.1 / 96.2).
static int least_generations(int xo, int rpc, int D4, double CR) {
  if (xo != kBin && rpc == 1 && D4 > 128) return 5;
  if (xo == kExp && CR > 0.5 && rpc > 16) return 5;
  return rpc >= 8 ? 3 : 4;
}

bool prepare_resident(int xo, int obj, int vidx, int block, int N, int D4, double CR, int gens, int sm_count,
                      int smem_optin, ResidentShape* out) {
  if (vidx > 1 || block > 256 || sm_count <= 0) return false;
  ResidentShape s{};
  s.rpc = (N + sm_count - 1) / sm_count;
  s.grid = (N + s.rpc - 1) / s.rpc;
  const int nw = block / 32;
  s.seg = xo != kBin;
  if (s.seg && (vidx != 0 || (D4 > 32 && (1.0 - CR) * 40.0 < 1.0))) return false;
  if (!s.seg && nw > 1 && s.rpc * nw > kResWarps) return false;
  if (gens < least_generations(xo, s.rpc, D4, CR)) return false;
  const int W = s.seg ? 1 : nw;
  // 15 named barriers, one per group of more than a warp
  s.groups = std::min(s.rpc, W > 1 ? std::min(kResWarps / W, 15) : kResWarps);
  s.block = 32 * (s.groups * W + kResHelpers);
  s.smem = res_layout(s.seg, s.rpc, D4, s.groups, block, kVecChoices[vidx], sums_of(obj)).total;
  const void* fn = entry_of(s.seg, obj, vidx);
  cudaFuncAttributes a;
  if (!fn || cudaFuncGetAttributes(&a, fn) != cudaSuccess) return false;
  if (s.smem + a.sharedSizeBytes > (size_t)smem_optin || s.block > a.maxThreadsPerBlock) return false;
  int per_sm = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           smem_optin - (int)a.sharedSizeBytes) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, s.block, s.smem) != cudaSuccess)
    return false;
  if (per_sm < 1) return false;
  *out = s;
  return true;
}

cudaError_t launch_resident(int xo, int obj, int vidx, const ResidentShape& sh, ResidentParams rp, cudaStream_t s) {
  const void* fn = entry_of(sh.seg, obj, vidx);
  if (!fn) return cudaErrorInvalidValue;
  rp.rpc = sh.rpc;
  rp.groups = sh.groups;
  rp.xo = xo;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)sh.grid);
  cfg.blockDim = dim3((unsigned)sh.block);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {&rp};
  return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace de
