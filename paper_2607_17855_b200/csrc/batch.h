// Batched window kernels: the structures and the once-per-call part shared by the scalar contraction (batch.cu) and
// the one on the float64 matrix instruction (batch_mma.cu).
#pragma once
#include <stdint.h>

#include "bi_internal.h"

// Programmatic dependent launch: the iteration loop queues its kernels so that the next one may be
// scheduled while the previous one drains.  A kernel first does what needs none of its
// predecessor's results (its task, the slice copy, index loads), then waits for the predecessor to
// complete (bi_grid_wait; a no-op when launched without the attribute) and only then lets its own
// successor be scheduled: when a kernel starts, everything before its predecessor is complete.
__device__ __forceinline__ void bi_grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void bi_grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }

// Most (agent, step) units of a call: the kernels and launchers count them in 32 bits.
constexpr long long kMaxUnits = 1LL << 30;

struct BatchMember {
  const void *logA;        // packed [m][P_pad]
  int32_t m, P_pad, modality, shape, rank;
  int32_t offp[BI_MAX_RANK];   // padded belief offsets of the group's axes, packed order
  int32_t dim[BI_MAX_RANK];    // axis sizes, packed order (last one unpadded)
  int32_t ooff[BI_MAX_RANK];   // start of each outer axis in the per-thread shared-memory columns
  int32_t ncp, rows;       // padded last axis; rows = product of the outer axes
  int64_t gstride;         // elements per agent's model (per-agent models), 0 when shared
  int32_t task0;           // first task slot of this member
  int32_t tu, perm0;       // units per task; first entry of its units in perm (task slot s: tu entries from perm0 + (s - task0) tu)
  int32_t split;           // unrolled forms: threads per unit (1, 2 or 4), each taking a range of the first axis
  // Where the messages of each axis go, relative to the unit's row of this member's plane.  (A transition
  // tensor of a model with several parents per transition is a member too: its first axis is the child's state at
  // the next step -- the next unit's beliefs, and messages to the next unit's row of a plane of their own.)
  int32_t edge;            // 0, or 1 + the factor whose transition this is: its "outcome" is the action
  int64_t oout[BI_MAX_RANK];
};

struct BatchParams {
  BatchMember mem[BI_MAX_M + BI_MAX_F];
  int32_t nmem;            // members of rank >= 2
  int32_t task_base;       // first task of this launch
  int32_t NU, Sp, ntask, tu;   // tu: units per contraction CTA
  int32_t sc_off;          // unrolled forms: element offset of the split tasks' scratch columns behind the slice
  int32_t lbuf, so_max;    // any-shape form: elements of the slice staging buffer; most outer states of a member
  const int32_t *perm;     // unit ids, member by member, ordered by observed outcome
  const int4 *task;        // [ntask] (outcome, first entry in perm, count, member)
  void *ellp;              // [nmem][NU][Sp] partial likelihood messages
  void *qbuf;              // [2][NU][Sp] beliefs
  uint32_t *status;        // the handle's status word
  const int32_t *obs;      // [NU][M] (per-agent models: every unit reads its own slice)
  const int32_t *act;      // [N][T-1][F] (transition members)
  int32_t M, T, F;
  int32_t drop_copy;       // testing aid: the contraction announces its slice copy and does not issue it
};

// Queues the kernels that write the starting beliefs and bucket the units: perm and task of P's members (shared
// models; perm and task are P.perm and P.task, writable).  max_m: most outcomes of a member.
int bi_batch_start_f64(const bi_model *md, const BatchParams &P, int max_m, const float *q_init, int32_t *perm, int4 *task,
                       cudaStream_t stream);
