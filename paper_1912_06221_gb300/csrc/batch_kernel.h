// Device-side descriptors and host entry points of the persistent batch launch
// (batch_kernel.cu), shared with the batch host code (batch.cpp).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace rdg {

// One member problem as the persistent kernel sees it (face form, SSP-RK3).  Its work of one phase is
// a row of items, each `per_item` elements: in phase 0 the face records of its state, in phase p >= 1
// stage p - 1 of the launch.
struct BMember {
  FaceArgs base;             // everything a stage takes that does not change from stage to stage
  float *u, *u1, *u2;        // state and the two stage buffers
  float* rec[2];             // the two record buffers
  TimeState* ts;             // time origin and steps done before this launch
  Forcing frc;
  double dt;
  int N;
  bool alg1, team;           // team: items of 32-element tiles, four warps to a tile
  int64_t per_item, nitem;   // elements per item, items per phase
  int64_t off;               // first item of this member within a phase of its list
  int64_t hold_phase;        // a phase that is never released (test hook), or -1
};

// The members of one order: a list of items of its own.  Blocks prefer the list of their SM, until as
// many as the list wants have come.
struct BatchList {
  int m0, m1;                // members [m0, m1) of the descriptor array
  int sm_end;                // SMs up to here (exclusive, from the previous list's end) prefer this list
  int blocks;                // blocks wanted
  int64_t per_phase;         // items of one phase, all members of the list
};

struct BatchArgs {
  const BMember* m;          // device array [nm], by ascending order and, within it, ascending off
  int nm, nlist;
  BatchList list[6];
  int nphase;                // 1 + stages of this launch (3 x steps)
  unsigned long long* ticket;  // per list, kCountStride apart (a cache line each)
  unsigned long long* claim;   // blocks that came to each list, likewise
  unsigned long long* done;    // items finished per member, likewise
  int* abort;
  int* err;                  // the batch's device error word
  uint64_t wait_ns;          // bound on every dependency wait
};

constexpr int kCountStride = 16;
constexpr int kSmemMembers = 64;   // descriptors kept in shared memory up to this many
size_t batch_smem_bytes(int nm);
int batch_grid(size_t smem);       // resident blocks of the persistent kernel (-1 on error)
int launch_batch_persistent(const BatchArgs& a, int grid, size_t smem, cudaStream_t s);
int launch_batch_advance(BMember* m, int nm, long long steps, cudaStream_t s);
int batch_sms();                   // SMs of the current device

}  // namespace rdg
