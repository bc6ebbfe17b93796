// One order of the face form (face_kernels.cuh).  The build compiles this file once per RDG_ORDER in
// 1..6, after writing that order's operators face_ops_<N>.h into the build folder (gen_face.cpp).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#ifndef RDG_ORDER
#error "RDG_ORDER must be defined"
#endif

#define RDG_CAT2(a, b) a##b
#define RDG_CAT(a, b) RDG_CAT2(a, b)
#define RDG_STR2(a) #a
#define RDG_STR(a) RDG_STR2(a)

#include "face_kernels.cuh"

namespace rdg {
namespace face {
#include RDG_STR(RDG_CAT(face_ops_, RDG_ORDER).h)
}  // namespace face

int RDG_CAT(launch_face_parts_, RDG_ORDER)(bool alg1, const FaceArgs& a, cudaStream_t s) {
  constexpr int N = RDG_ORDER, BLK = dev::kFaceBlock;
  if (a.k_end <= a.k_begin) return RDG_OK;
  const unsigned grid = (unsigned)((a.k_end - a.k_begin + BLK - 1) / BLK);
  return alg1 ? launch_pdl(dev::face_parts_kernel<N, true>, grid, BLK, s, a)
              : launch_pdl(dev::face_parts_kernel<N, false>, grid, BLK, s, a);
}

// Resident blocks of a kernel on the current device (asked once per device).
template <typename K>
static int resident_blocks(K kernel, std::atomic<int>* cached) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, dev::kFaceBlock, 0) != cudaSuccess || per < 1) per = 1;
    n = per * sm_count();
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// Which kernel runs a stage, by the number of 32-element tiles:
//  - at orders 4..6, up to one tile per SM: four warps to a tile (512 elements, order 4 / 5 / 6: 2.8 / 3.6
//    / 4.5 us per stage against 3.1 / 4.7 / 6.8; at 8192 elements it no longer gains);
//  - the small build while its warps hold all tiles, the large one (more, leaner warps) beyond, as long
//    as few waves of it remain (2 up to order 4, 1 above): with many waves the difference is gone and
//    the small build's early loads win (order 3, 1M elements: 53 against 57 us per stage).
template <bool ALG1>
static int launch_stage(const FaceArgs& a, cudaStream_t s) {
  constexpr int N = RDG_ORDER;
  static std::atomic<int> small_slots[64], large_slots[64];
  const int64_t tiles = (a.K + 31) / 32, blocks = (tiles + dev::kFaceWarps - 1) / dev::kFaceWarps;
  if constexpr (N >= 4) {
    if (tiles <= sm_count()) return launch_pdl(dev::face_team_kernel<N, ALG1>, (unsigned)tiles, 128, s, a);
  }
  auto small = dev::face_stage_kernel<N, ALG1, false>;
  auto large = dev::face_stage_kernel<N, ALG1, true>;
  const int64_t ns = resident_blocks(small, small_slots), nl = resident_blocks(large, large_slots);
  if (blocks > ns && blocks <= (N <= 4 ? 2 : 1) * nl)
    return launch_pdl(large, (unsigned)std::min(blocks, nl), dev::kFaceBlock, s, a);
  return launch_pdl(small, (unsigned)std::min(blocks, ns), dev::kFaceBlock, s, a);
}

int RDG_CAT(launch_face_stage_, RDG_ORDER)(bool alg1, const FaceArgs& a, cudaStream_t s) {
  if (a.K == 0) return RDG_OK;
  return alg1 ? launch_stage<true>(a, s) : launch_stage<false>(a, s);
}

template <bool ALG1>
static int launch_lone(const FaceArgs& a, cudaStream_t s) {
  const unsigned grid = (unsigned)((a.K + dev::kFaceBlock - 1) / dev::kFaceBlock);
  if constexpr (RDG_ORDER == 1) return launch_pdl(dev::face_lone_kernel<RDG_ORDER, ALG1>, grid, dev::kFaceBlock, s, a);
  else return a.mode == 0 ? launch_pdl(dev::face_rhs_kernel<RDG_ORDER, ALG1>, grid, dev::kFaceBlock, s, a) : RDG_EINVAL;
}

int RDG_CAT(launch_face_lone_, RDG_ORDER)(bool alg1, const FaceArgs& a, cudaStream_t s) {
  if (a.K == 0) return RDG_OK;
  return alg1 ? launch_lone<true>(a, s) : launch_lone<false>(a, s);
}

int RDG_CAT(launch_face_ghost_, RDG_ORDER)(bool alg1, const float* G, const float4* gpar, int64_t B, int nghost, float* out,
                                           cudaStream_t s) {
  constexpr int N = RDG_ORDER;
  const int64_t n = B * nghost;
  if (n == 0) return RDG_OK;
  const unsigned grid = (unsigned)((n + 127) / 128);
  if (alg1) dev::face_ghost_kernel<N, true><<<grid, 128, 0, s>>>(G, gpar, B, n, out);
  else dev::face_ghost_kernel<N, false><<<grid, 128, 0, s>>>(G, gpar, B, n, out);
  return cudaGetLastError() == cudaSuccess ? RDG_OK : RDG_ECUDA;
}

}  // namespace rdg
