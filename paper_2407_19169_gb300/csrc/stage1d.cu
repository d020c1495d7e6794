// stage1d.cu — instantiations of the 1D kernels: degrees 1..3, advection / Burgers / Euler, FP64 and the
// FP32 form; the whole-step kernel, and the single-stage kernel for the hybrid limiter and OEDG.
#include "dg_internal.h"
#include "stage1d.cuh"

namespace dgk {

template <int K, int EQ, class PR, bool OE>
static cudaError_t launch1d(const void* args, unsigned grid, unsigned block, size_t smem, cudaStream_t s) {
  stage1d_kernel<K, EQ, PR, OE><<<grid, block, smem, s>>>(*(const Stage1DArgs*)args);
  return cudaGetLastError();
}
template <int K, int EQ, class PR, bool OE>
static cudaError_t smem1d(size_t bytes) {
  return cudaFuncSetAttribute(stage1d_kernel<K, EQ, PR, OE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)bytes);
}
template <int K, int EQ, class PR, bool OE>
static StageLauncher make1d() {
  return StageLauncher{&launch1d<K, EQ, PR, OE>, &smem1d<K, EQ, PR, OE>, 0, nullptr};
}

// the OEDG form (OE) for Burgers and Euler only
template <int K, class PR, bool OE>
static StageLauncher pick_eq(int EQ) {
  switch (EQ) {
    case EQ_ADV:
      if constexpr (!OE) return make1d<K, EQ_ADV, PR, false>();
      break;
    case EQ_BURG: return make1d<K, EQ_BURG, PR, OE>();
    case EQ_EULER: return make1d<K, EQ_EULER, PR, OE>();
  }
  return StageLauncher{nullptr, nullptr, 0, nullptr};
}

template <class PR, bool OE>
static StageLauncher pick_k(int K, int EQ) {
  switch (K) {
    case 1: return pick_eq<1, PR, OE>(EQ);
    case 2: return pick_eq<2, PR, OE>(EQ);
    case 3: return pick_eq<3, PR, OE>(EQ);
  }
  return StageLauncher{nullptr, nullptr, 0, nullptr};
}

template <int K, int EQ, class PR>
static cudaError_t launch_step1(const void* args, unsigned grid, unsigned block, size_t, cudaStream_t s) {
  step1d_kernel<K, EQ, PR><<<grid, block, 0, s>>>(*(const Stage1DArgs*)args);
  return cudaGetLastError();
}
static cudaError_t no_smem(size_t) { return cudaSuccess; }
template <int K, int EQ, class PR>
static int occ_step1(unsigned block, size_t) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, step1d_kernel<K, EQ, PR>, (int)block, 0) != cudaSuccess) return 0;
  return n;
}
template <int K, class PR>
static StageLauncher pick_step(int EQ) {
  switch (EQ) {
    case EQ_ADV: return StageLauncher{&launch_step1<K, EQ_ADV, PR>, &no_smem, 0, &occ_step1<K, EQ_ADV, PR>};
    case EQ_BURG: return StageLauncher{&launch_step1<K, EQ_BURG, PR>, &no_smem, 0, &occ_step1<K, EQ_BURG, PR>};
    case EQ_EULER: return StageLauncher{&launch_step1<K, EQ_EULER, PR>, &no_smem, 0, &occ_step1<K, EQ_EULER, PR>};
  }
  return StageLauncher{nullptr, nullptr, 0, nullptr};
}
StageLauncher step1d_launcher(int K, int EQ, int PREC) {
  const bool f64 = PREC == PREC_F64;
  switch (K) {
    case 1: return f64 ? pick_step<1, PrecF64>(EQ) : pick_step<1, PrecF32M>(EQ);
    case 2: return f64 ? pick_step<2, PrecF64>(EQ) : pick_step<2, PrecF32M>(EQ);
    case 3: return f64 ? pick_step<3, PrecF64>(EQ) : pick_step<3, PrecF32M>(EQ);
  }
  return StageLauncher{nullptr, nullptr, 0, nullptr};
}

// Threads and blocks of the whole-step kernel for n cells. A block of NT threads gives NT - 12 cells. The
// issue slots and the FP64 pipe belong to the quarters of an SM (an FP64 warp instruction holds its
// quarter for 64 cycles), so the time follows the warps of the fullest quarter: the smallest NT of 32,
// 64, 128 and 256 with the fewest (a few cells spread over the SMs, many take wide tiles with little
// halo), then at most the resident blocks, which loop over their tiles. The FP32 form also waits at the
// block's barriers, which the rule leaves out. Euler, us per step with 32 / 64 / 128 / 256 threads, the
// rule's choice in brackets: FP32 form P2 10^4 cells (9.3) 8.3 8.3 9.2, 65536 26.0 13.0 (11.3) 11.3,
// 2 10^5 34.8 20.1 (18.2) 18.5, 10^6 82.6 66.4 59.9 (60.4), P3 65536 26.9 14.4 (12.4) 12.4; FP64 P3 65536
// 222 182 (160) 159.
Step1DGrid step1d_grid(const StageLauncher& L, long long n) {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
    nsm = 152;
  Step1DGrid best{32, 1, 1};
  long long cost = -1;
  for (int nt : {32, 64, 128, STEP_THREADS}) {
    const int bps = L.blocks_per_sm(nt, 0);
    if (bps < 1) continue;
    const long long tiles = tiles_of(n, nt - 2 * STEP_HALO);
    const long long c = (((tiles + nsm - 1) / nsm) * (nt / 32) + 3) / 4;
    if (cost >= 0 && c >= cost) continue;
    cost = c;
    const long long cap = (long long)nsm * bps;
    best = Step1DGrid{(unsigned)nt, (unsigned)(tiles < cap ? tiles : cap), tiles};
  }
  return best;
}

StageLauncher stage1d_launcher(int K, int EQ, int PREC, bool oedg) {
  if (oedg) return PREC == PREC_F64 ? pick_k<PrecF64, true>(K, EQ) : pick_k<PrecF32M, true>(K, EQ);
  return PREC == PREC_F64 ? pick_k<PrecF64, false>(K, EQ) : pick_k<PrecF32M, false>(K, EQ);
}

}  // namespace dgk
