// One persistent launch for a chunk of SSP-RK3 steps of many independent problems (meshes of any
// size, orders 1..6, FP32 in the face form).  The work of a launch is one list of items per order,
// phase by phase: in phase 0 every member's items form the face records of its state, in phase p they run its
// stage p - 1 (face_kernels.cuh: fluxes from the records, volume term, LIFT, sources, update and the
// records of the result).  Blocks take items from a list's ticket counter in list order.  A member's
// phase p starts when its phase p - 1 is done (one count of finished items per member).  Because items
// are handed out in list order, every item an item waits on was handed out earlier to a block that is
// running it, so the waits always end (no co-residency needed).  Each wait is bounded: after the wait
// limit the block records kErrWaitTimeout, raises the launch's abort flag and leaves, and every other
// block leaves at its next item.
//
// A block takes items of one order, if it can that of its SM (a share of the SMs by the order's work),
// until that list is used up, then of the others: an order's code is 5 to 70 KB.  With one list for all
// orders the batch named below took 18.3 us per stage, with lists and as many blocks to each as it has
// items 14.5; no ticket is taken before the item ahead of it is done (a block would hold two items of a
// phase while others had none: two members of orders 2 and 3, 8.7 against 5.4 us).
//
// One phase per stage: with per-edge operators a stage took two dependent parts (edge fluxes and volume
// terms, then the element updates) and streamed 584 B per edge; 12 members of orders 2..6 and 200 to
// 27000 triangles, 20 steps: 3405 us then, 866 now.  The paper solves one problem at a time; this has no
// counterpart there.
#include <cuda_runtime.h>

#include <algorithm>

#include "batch_kernel.h"
#include "face_kernels.cuh"

namespace rdg {
namespace face {
#include "face_ops_1.h"
#include "face_ops_2.h"
#include "face_ops_3.h"
#include "face_ops_4.h"
#include "face_ops_5.h"
#include "face_ops_6.h"
}  // namespace face

namespace bk {

constexpr int kBlock = dev::kFaceBlock;
constexpr int kRowFloats = 2 * dev::kFaceWarps * 32 * np_of(6);   // two row slices per warp, or a team's five

__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long count_of(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Bounded wait until *cnt >= target (or the launch is aborted).  false: gave up.  A stage is a few us,
// so the count alone is polled; the abort flag and the clock are looked at every 32nd time.
__device__ bool wait_count(const unsigned long long* cnt, unsigned long long target, const int* abort,
                           uint64_t limit_ns) {
  const volatile int* ab = abort;
  const uint64_t t0 = gtime();
  for (unsigned polls = 1; count_of(cnt) < target; ++polls) {
    if (polls % 32 == 0) {
      if (*ab) return false;
      if (gtime() - t0 > limit_ns) return false;
      if (polls > 256) __nanosleep(polls > 4096 ? 512 : 64);
    }
  }
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  return true;
}

// Elements [k0, k1) of one item: their records (phase 0) or one stage.
template <int N, bool ALG1>
__device__ __noinline__ void run_item(const FaceArgs& a, bool records, bool team, int64_t k0, int64_t k1, float* sh) {
  const int warp = threadIdx.x >> 5;
  if constexpr (N >= 4) {
    if (team && !records) {
      for (int64_t k = k0; k < k1; k += 32) {
        dev::team_tile<N, ALG1, true>(a, k, (int)min((int64_t)32, k1 - k), sh,
                                      reinterpret_cast<float(*)[32 * np_of(N)]>(sh + 32 * np_of(N)));
        __syncthreads();
      }
      return;
    }
  }
  float* s = sh + warp * 64 * np_of(N);
  for (int64_t k = k0 + warp * 32; k < k1; k += kBlock) {
    const int nk = (int)min((int64_t)32, k1 - k);
    if (records) dev::parts_tile<N, ALG1, (N >= 5), true>(a, k, nk, s);
    else dev::stage_tile<N, ALG1, (N <= 4 ? 3 : 0), (N >= 5), true>(a, k, nk, s, s + 32 * np_of(N));
    __syncwarp();
  }
}

template <int N>
__device__ __forceinline__ void run_order(const BMember& b, const FaceArgs& a, bool records, int64_t k0, int64_t k1,
                                          float* sh) {
  if (b.alg1) run_item<N, true>(a, records, b.team, k0, k1, sh);
  else run_item<N, false>(a, records, b.team, k0, k1, sh);
}

__global__ void __launch_bounds__(kBlock, 4) batch_persistent_kernel(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) float smem[];
  // the member descriptors, in shared memory when they fit (searched for every item)
  BMember* smem_m = reinterpret_cast<BMember*>(smem + kRowFloats);
  const bool in_smem = a.nm <= kSmemMembers;
  const BMember* mem = in_smem ? smem_m : a.m;
  __shared__ FaceArgs s_args;
  __shared__ long long s_item;
  __shared__ int s_go, s_list;
  if (in_smem) {
    const int words = a.nm * (int)(sizeof(BMember) / 4);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.m);
    uint32_t* dst = reinterpret_cast<uint32_t*>(smem_m);
    for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = src[i];
  }
  unsigned sm;
  asm volatile("mov.u32 %0, %smid;" : "=r"(sm));
  int q = 0;                                    // this block's list (thread 0), lists used up so far
  while (q + 1 < a.nlist && (int)sm >= a.list[q].sm_end) ++q;
  if (threadIdx.x == 0 && a.nlist > 1) {
    for (int t = 0; t < a.nlist; ++t) {
      if (atomicAdd(a.claim + q * kCountStride, 1ull) < (unsigned long long)a.list[q].blocks) break;
      q = q + 1 < a.nlist ? q + 1 : 0;
    }
  }
  int used = 0;
  long long next = threadIdx.x == 0 ? (long long)atomicAdd(a.ticket + q * kCountStride, 1ull) : 0;
  for (;;) {
    if (threadIdx.x == 0) {
      while (next >= a.list[q].per_phase * a.nphase && ++used < a.nlist) {
        q = q + 1 < a.nlist ? q + 1 : 0;
        next = (long long)atomicAdd(a.ticket + q * kCountStride, 1ull);
      }
      s_item = used < a.nlist ? next : -1;
      s_list = q;
    }
    __syncthreads();
    const long long it = s_item;
    if (it < 0) break;
    const BatchList& list = a.list[s_list];
    const int p = (int)(it / list.per_phase);
    const long long r = it - (long long)p * list.per_phase;
    int lo = list.m0, hi = list.m1 - 1;         // member holding item r of the phase
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (mem[mid].off <= r) lo = mid;
      else hi = mid - 1;
    }
    const BMember& b = mem[lo];
    const int step = p > 0 ? (p - 1) / 3 : 0, stage = p > 0 ? (p - 1) % 3 : 0;
    if (threadIdx.x < (int)(sizeof(FaceArgs) / 4))
      reinterpret_cast<uint32_t*>(&s_args)[threadIdx.x] = reinterpret_cast<const uint32_t*>(&b.base)[threadIdx.x];
    __syncthreads();
    if (threadIdx.x == 0) {
      s_args.us = stage == 0 ? b.u : (stage == 1 ? b.u1 : b.u2);
      s_args.un = b.u;
      s_args.out = stage == 0 ? b.u1 : (stage == 1 ? b.u2 : b.u);
      s_args.fin = b.rec[(p + 1) & 1];
      s_args.fout = p + 1 < a.nphase ? b.rec[p & 1] : nullptr;
      s_args.mode = stage + 1;
      // phase p of the member after its phase p - 1; a held phase never starts
      const bool ok = wait_count(a.done + (size_t)lo * kCountStride, p == b.hold_phase ? ~0ull : (unsigned long long)p * (unsigned long long)b.nitem,
                                 a.abort, a.wait_ns);
      if (!ok) {
        atomicOr(a.err, kErrWaitTimeout);
        atomicExch(a.abort, 1);
      }
      s_go = ok;
    } else if (threadIdx.x >= 32 && threadIdx.x < 32 + 2 * RDG_MAX_FORCING_TERMS) {
      const int m = threadIdx.x - 32, i = m % RDG_MAX_FORCING_TERMS;
      const bool src = m < RDG_MAX_FORCING_TERMS;
      if (i < (src ? b.frc.nsrc : b.frc.nghost)) {
        const double t = b.ts->t0 + ((double)b.ts->n + step + (stage == 0 ? 0.0 : (stage == 1 ? 1.0 : 0.5))) * b.dt;
        s_args.tau[m] = (float)dev::tau_of(src ? b.frc.kind[i] : b.frc.gkind[i], src ? b.frc.omega[i] : b.frc.gomega[i], t);
      }
    }
    __syncthreads();
    if (!s_go) break;
    const int64_t k0 = (r - b.off) * b.per_item, k1 = min(k0 + b.per_item, b.base.K);
    switch (b.N) {
      case 1: run_order<1>(b, s_args, p == 0, k0, k1, smem); break;
      case 2: run_order<2>(b, s_args, p == 0, k0, k1, smem); break;
      case 3: run_order<3>(b, s_args, p == 0, k0, k1, smem); break;
      case 4: run_order<4>(b, s_args, p == 0, k0, k1, smem); break;
      case 5: run_order<5>(b, s_args, p == 0, k0, k1, smem); break;
      default: run_order<6>(b, s_args, p == 0, k0, k1, smem); break;
    }
    // the next ticket, its round trip beside the release's; taken any earlier, a block would hold two
    // items of a phase while another had none
    if (threadIdx.x == 0) next = (long long)atomicAdd(a.ticket + q * kCountStride, 1ull);
    __syncthreads();                            // every thread's writes of the item, then its release
    if (threadIdx.x == 0)
      asm volatile("fence.acq_rel.gpu;\n\tred.relaxed.gpu.global.add.u64 [%0], 1;" ::"l"(a.done + (size_t)lo * kCountStride)
                   : "memory");
  }
}

__global__ void batch_advance_kernel(BMember* m, int nm, long long steps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nm) m[i].ts->n += steps;
}

}  // namespace bk

static_assert(sizeof(FaceArgs) % 4 == 0 && sizeof(FaceArgs) / 4 <= bk::kBlock, "copied one word per thread");
static_assert(sizeof(BMember) % 8 == 0, "copied word by word");

int batch_sms() { return sm_count(); }

size_t batch_smem_bytes(int nm) {
  return bk::kRowFloats * sizeof(float) + (nm <= kSmemMembers ? (size_t)nm * sizeof(BMember) : 0);
}

int batch_grid(size_t smem) {
  static bool attr = false;
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr) {
    if (cudaFuncSetAttribute(bk::batch_persistent_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) !=
        cudaSuccess)
      return -1;
    attr = true;
  }
  int per = 0, nsm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, bk::batch_persistent_kernel, bk::kBlock, smem) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1;
  return std::max(1, per) * nsm;
}

int launch_batch_persistent(const BatchArgs& a, int grid, size_t smem, cudaStream_t s) {
  bk::batch_persistent_kernel<<<grid, bk::kBlock, smem, s>>>(a);
  return cudaGetLastError() == cudaSuccess ? RDG_OK : RDG_ECUDA;
}

int launch_batch_advance(BMember* m, int nm, long long steps, cudaStream_t s) {
  bk::batch_advance_kernel<<<(nm + 127) / 128, 128, 0, s>>>(m, nm, steps);
  return cudaGetLastError() == cudaSuccess ? RDG_OK : RDG_ECUDA;
}

}  // namespace rdg
