// One order of the face form (face_kernels.cuh).  The build compiles this file once per RDG_ORDER in
// 1..6, after writing that order's operators face_ops_<N>.h into the build folder (gen_face.cpp).
#include <cuda_runtime.h>

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
  constexpr int N = RDG_ORDER, BLK = dev::face_block<N>();
  if (a.k_end <= a.k_begin) return RDG_OK;
  const unsigned grid = (unsigned)((a.k_end - a.k_begin + BLK - 1) / BLK);
  return alg1 ? launch_pdl(dev::face_parts_kernel<N, true>, grid, BLK, s, a)
              : launch_pdl(dev::face_parts_kernel<N, false>, grid, BLK, s, a);
}

int RDG_CAT(launch_face_stage_, RDG_ORDER)(bool alg1, const FaceArgs& a, cudaStream_t s) {
  constexpr int N = RDG_ORDER, BLK = dev::face_block<N>();
  if (a.K == 0) return RDG_OK;
  const unsigned grid = (unsigned)((a.K + BLK - 1) / BLK);
  return alg1 ? launch_pdl(dev::face_stage_kernel<N, true>, grid, BLK, s, a)
              : launch_pdl(dev::face_stage_kernel<N, false>, grid, BLK, s, a);
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
