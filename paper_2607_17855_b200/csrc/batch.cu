// Batched window kernels (VMP / MMP) for agents that share one model.
//
// With a shared model, every (agent, step) whose observation of modality i is
// the same outcome o contracts the SAME slice ln A_i[o] against its own
// beliefs.  The calls are therefore organised iteration by iteration over all
// agents at once: (agent, step) units are bucketed by observed outcome per
// modality (once per call), and in each iteration a CTA stages one slice in
// shared memory and 128 units of that bucket contract against it, one thread
// per unit with every accumulator in registers.  A slice row is then one
// broadcast shared-memory load for the whole warp, the row's index arithmetic
// is shared by all units, and the leave-one-out messages of all the group's
// factors (Section IV, marginalisation) come out of a single pass over the
// slice.  A second kernel per iteration adds the transition messages and takes
// the softmax per unit (Jacobi over steps and factors, Appendix A-2).
//
// Float64 calls on shared models run on the matrix instruction (batch_mma.cu); the contractions here serve float32,
// slices per unit, and groups over five factors.  They have two forms: fully unrolled float32 code for the dependency-group
// shapes in BI_BATCH_SHAPES (every accumulator in registers), and a form for any
// shape of rank 2..5 that is compiled only for the padded size of the last axis
// (its accumulators in registers, those of the outer axes in per-thread columns
// of shared memory; a plain loop along the innermost outer axis, one climb of the others per run of rows).
#include <algorithm>
#include <climits>
#include <cstring>

#include <type_traits>

#include <cooperative_groups.h>

#include "batch.h"
#include "tile3.cuh"

namespace {

constexpr int kTU = 128;   // most units per contraction CTA (the call picks 32, 64 or 128)

// packed dims of the compiled group shapes: rank, then the axis sizes (last axis unpadded)
#define BI_BATCH_SHAPES(X) \
  X(0, 4, 10, 10, 6, 8)    \
  X(1, 3, 10, 6, 8, 0)     \
  X(2, 2, 10, 8, 0, 0)     \
  X(3, 2, 10, 10, 0, 0)    \
  X(4, 3, 3, 2, 4, 0)      \
  X(5, 2, 5, 3, 0, 0)

// ---- one unit against one slice: every message of the group in one pass ----
// L: the slice in shared memory, rows of NCP; q / out: this unit's beliefs and
// message area (padded layout); o0..: offsets of the axes' factors.

// SPLIT > 1: the threads of `SPLIT` different warps share a unit, each taking a range of the first
// axis (part = which); a thread writes the first axis' messages of its range, and its partial messages
// of the other axes to the scratch columns sc[i * nt + tid], which the caller adds in a fixed order.
template <typename R, int N1, int NC>
__device__ __forceinline__ void contract2(const R *__restrict__ L, const R *__restrict__ q, R *__restrict__ out,
                                          const int32_t *o) {
  constexpr int NCP = (NC + 3) & ~3;
  R qc[NC], accc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) { qc[c] = q[o[1] + c]; accc[c] = (R)0; }
  for (int s1 = 0; s1 < N1; ++s1) {
    const R q1 = q[o[0] + s1];
    const R *row = L + s1 * NCP;
    R v0 = (R)0, v1 = (R)0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const R x = row[c];
      if (c & 1) v1 = fma(x, qc[c], v1); else v0 = fma(x, qc[c], v0);
      accc[c] = fma(q1, x, accc[c]);
    }
    out[o[0] + s1] = v0 + v1;
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) out[o[1] + c] = accc[c];
}

template <typename R, int N1, int N2, int NC, int SPLIT = 1>
__device__ __forceinline__ void contract3(const R *__restrict__ L, const R *__restrict__ q, R *__restrict__ out,
                                          const int32_t *o, int part = 0, bool wr = true, R *sc = nullptr, int nt = 0) {
  const int sa = part * N1 / SPLIT, sb = (part + 1) * N1 / SPLIT;
  constexpr int NCP = (NC + 3) & ~3;
  R q2[N2], qc[NC], acc2[N2], accc[NC];
#pragma unroll
  for (int i = 0; i < N2; ++i) { q2[i] = q[o[1] + i]; acc2[i] = (R)0; }
#pragma unroll
  for (int c = 0; c < NC; ++c) { qc[c] = q[o[2] + c]; accc[c] = (R)0; }
  R q1n = q[o[0] + sa];   // (the first axis' belief is read one index ahead: its latency hides under the rows)
  for (int s1 = sa; s1 < sb; ++s1) {
    const R q1 = q1n;
    if (s1 + 1 < sb) q1n = q[o[0] + s1 + 1];
    R a1 = (R)0;
#pragma unroll
    for (int s2 = 0; s2 < N2; ++s2) {
      const R *row = L + (s1 * N2 + s2) * NCP;
      const R w = q1 * q2[s2];
      R v0 = (R)0, v1 = (R)0;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const R x = row[c];
        if (c & 1) v1 = fma(x, qc[c], v1); else v0 = fma(x, qc[c], v0);
        accc[c] = fma(w, x, accc[c]);
      }
      const R v = v0 + v1;
      acc2[s2] = fma(q1, v, acc2[s2]);
      a1 = fma(q2[s2], v, a1);
    }
    if (wr) out[o[0] + s1] = a1;
  }
#pragma unroll
  for (int i = 0; i < N2; ++i) {
    if (SPLIT > 1) sc[i * nt] = acc2[i];
    else out[o[1] + i] = acc2[i];
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if (SPLIT > 1) sc[(N2 + c) * nt] = accc[c];
    else out[o[2] + c] = accc[c];
  }
}

template <typename R, int N1, int N2, int N3, int NC, int SPLIT = 1>
__device__ __forceinline__ void contract4(const R *__restrict__ L, const R *__restrict__ q, R *__restrict__ out,
                                          const int32_t *o, int part = 0, bool wr = true, R *sc = nullptr, int nt = 0) {
  const int sa = part * N1 / SPLIT, sb = (part + 1) * N1 / SPLIT;
  constexpr int NCP = (NC + 3) & ~3;
  R q2[N2], q3[N3], qc[NC], acc2[N2], acc3[N3], accc[NC];
#pragma unroll
  for (int i = 0; i < N2; ++i) { q2[i] = q[o[1] + i]; acc2[i] = (R)0; }
#pragma unroll
  for (int i = 0; i < N3; ++i) { q3[i] = q[o[2] + i]; acc3[i] = (R)0; }
#pragma unroll
  for (int c = 0; c < NC; ++c) { qc[c] = q[o[3] + c]; accc[c] = (R)0; }
  R q1n = q[o[0] + sa];   // (read one index ahead, as above)
  for (int s1 = sa; s1 < sb; ++s1) {
    const R q1 = q1n;
    if (s1 + 1 < sb) q1n = q[o[0] + s1 + 1];
    R a1 = (R)0;
#pragma unroll
    for (int s2 = 0; s2 < N2; ++s2) {
      const R w12 = q1 * q2[s2];
      R v2 = (R)0;
#pragma unroll
      for (int s3 = 0; s3 < N3; ++s3) {
        const R *row = L + ((s1 * N2 + s2) * N3 + s3) * NCP;
        const R w = w12 * q3[s3];
        R v0 = (R)0, v1 = (R)0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const R x = row[c];
          if (c & 1) v1 = fma(x, qc[c], v1); else v0 = fma(x, qc[c], v0);
          accc[c] = fma(w, x, accc[c]);
        }
        const R v = v0 + v1;
        acc3[s3] = fma(w12, v, acc3[s3]);
        v2 = fma(q3[s3], v, v2);
      }
      acc2[s2] = fma(q1, v2, acc2[s2]);
      a1 = fma(q2[s2], v2, a1);
    }
    if (wr) out[o[0] + s1] = a1;
  }
#pragma unroll
  for (int i = 0; i < N2; ++i) {
    if (SPLIT > 1) sc[i * nt] = acc2[i];
    else out[o[1] + i] = acc2[i];
  }
#pragma unroll
  for (int i = 0; i < N3; ++i) {
    if (SPLIT > 1) sc[(N2 + i) * nt] = acc3[i];
    else out[o[2] + i] = acc3[i];
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if (SPLIT > 1) sc[(N2 + N3 + c) * nt] = accc[c];
    else out[o[3] + c] = accc[c];
  }
}

template <typename R, int RANK, int D0, int D1, int D2, int D3>
__device__ __forceinline__ void contract_shape(const R *L, const R *q, R *out, const int32_t *o, int split, int part,
                                               bool wr, R *sc, int nt) {
  if constexpr (RANK == 2) contract2<R, D0, D1>(L, q, out, o);
  else if constexpr (RANK == 3) {
    if (split == 1) contract3<R, D0, D1, D2>(L, q, out, o);
    else contract3<R, D0, D1, D2, 2>(L, q, out, o, part, wr, sc, nt);
  } else {
    if (split == 1) contract4<R, D0, D1, D2, D3>(L, q, out, o);
    else if (split == 2) contract4<R, D0, D1, D2, D3, 2>(L, q, out, o, part, wr, sc, nt);
    else contract4<R, D0, D1, D2, D3, 4>(L, q, out, o, part, wr, sc, nt);
  }
}

// ---- bucket the units of one modality by observed outcome (once per call) ----
// A cluster of kBucketCtas CTAs per member, each with a share of the units.  Writes the member's part of perm (unit ids
// grouped by outcome) and its task slots: chunks of at most tu units of one outcome.  A chain of latencies -- load,
// counter, load again, counter, store, for every 1024 units -- so the units are spread over a cluster and the
// counts exchanged through distributed shared memory; with one CTA per member 20 480 units took 30 us.  (One atomic for
// all of a warp's units of an outcome instead of one each: 42 us, the match instruction costs more.)  It runs beside
// the kernel that writes the starting beliefs.
constexpr int kBucketCtas = 8;
__global__ void __cluster_dims__(kBucketCtas, 1, 1) __launch_bounds__(1024)
bi_batch_bucket_kernel(BatchParams P, const int32_t *__restrict__ obs, int M, uint32_t *status,
                       int32_t *perm, int4 *task) {
  namespace cg = cooperative_groups;
  extern __shared__ int32_t sh[];       // count[m] | cursor[m] | total[m] | first task[m]
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), mi = blockIdx.x / kBucketCtas, tid = threadIdx.x, nt = blockDim.x;
  const BatchMember &mm = P.mem[mi];
  const int m = mm.m, NU = P.NU;
  int32_t *count = sh, *cursor = sh + m, *total = sh + 2 * m, *first = sh + 3 * m;
  for (int i = tid; i < m; i += nt) count[i] = 0;
  __syncthreads();
  const int share = (NU + kBucketCtas - 1) / kBucketCtas, ua = rank * share, ub = min(NU, ua + share);
  // the outcome that buckets a unit: the observed one, or for a transition the action taken at the unit's step
  // (a window's last step has none)
  auto outcome = [&](int u) {
    if (!mm.edge) return obs[(size_t)u * M + mm.modality];
    const int a = u / P.T, t = u - a * P.T;
    return t + 1 < P.T ? max(P.act[((size_t)a * (P.T - 1) + t) * P.F + mm.edge - 1], -1) : INT_MIN;
  };
#pragma unroll 4
  for (int u = ua + tid; u < ub; u += nt) {
    const int v = outcome(u);
    if (mm.edge && v == INT_MIN) continue;
    atomicAdd(&count[clamp_flag(v, m, status, mm.edge ? BI_FLAG_ACT_RANGE : BI_FLAG_OBS_RANGE)], 1);
  }
  cl.sync();
  for (int o = tid; o < m; o += nt) {
    int before = 0, all = 0;
#pragma unroll
    for (int r = 0; r < kBucketCtas; ++r) {
      const int n = cl.map_shared_rank(count, r)[o];
      if (r < rank) before += n;
      all += n;
    }
    cursor[o] = before;
    total[o] = all;
  }
  cl.sync();   // (everybody's counts are read; this also orders the block)
  // a member's buckets take whole tasks of tu units, one after the other: the units of a task are found without reading it
  const int tu = mm.tu, slot_end = mm.task0 + (NU + tu - 1) / tu + m;
  if (tid == 0) {
    int slot = mm.task0;
    for (int o = 0; o < m; ++o) {
      first[o] = slot;
      slot += (total[o] + tu - 1) / tu;
    }
    count[0] = slot;   // (the first unused slot)
  }
  __syncthreads();
  if (rank == 0) {
    for (int o = tid >> 5; o < m; o += nt >> 5) {
      const int n = total[o];
      for (int k = tid & 31; k * tu < n; k += 32)
        task[first[o] + k] = make_int4(o, mm.perm0 + (first[o] + k - mm.task0) * tu, min(tu, n - k * tu), mi);
    }
    for (int slot = count[0] + tid; slot < slot_end; slot += nt) task[slot] = make_int4(0, 0, 0, 0);
    __syncthreads();
  }
  int32_t *pm = perm + mm.perm0;
#pragma unroll 4
  for (int u = ua + tid; u < ub; u += nt) {
    int o = outcome(u);
    if (mm.edge && o == INT_MIN) continue;
    o = o < 0 ? 0 : (o >= m ? m - 1 : o);
    pm[(first[o] - mm.task0) * tu + atomicAdd(&cursor[o], 1)] = u;
  }
  bi_grid_wait();   // (the starting beliefs: whoever waits for this kernel finds both)
}

// Per-agent models: no two units share a slice, so the "buckets" are just runs of consecutive units.
__global__ void bi_batch_identity_tasks_kernel(BatchParams P, int32_t *perm, int4 *task) {
  const int mi = blockIdx.y, NU = P.NU, tu = P.tu;
  const int nchunk = (NU + tu - 1) / tu, p0 = P.mem[mi].perm0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NU; i += gridDim.x * blockDim.x)
    perm[p0 + i] = i;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nchunk + P.mem[mi].m; k += gridDim.x * blockDim.x)
    task[P.mem[mi].task0 + k] = k < nchunk ? make_int4(0, p0 + k * tu, min(tu, NU - k * tu), 0) : make_int4(0, 0, 0, 0);
}

// ---- contraction: one task = one slice, up to kTU units, one thread per unit ----
template <typename R>
__global__ void __launch_bounds__(kTU)
bi_batch_contract_kernel(BatchParams P, int cur, int first) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R *L = reinterpret_cast<R *>(smem_raw);
  if (first) {   // the tasks were written by the kernel just before this one
    bi_grid_wait();
    bi_grid_launch_dependents();
  }
  int mi = 0;
  const int slot = (int)blockIdx.x + P.task_base;
  while (mi + 1 < P.nmem && slot >= P.mem[mi + 1].task0) ++mi;
  const BatchMember &mm = P.mem[mi];
  const int4 tk = P.task[slot];
  if (tk.z == 0) {   // an unused task slot (an exiting CTA counts as having released its dependents)
    return;
  }
  // stage the slice of outcome tk.x: one bulk asynchronous copy, global -> shared, issued by one
  // thread; the others meanwhile look up their unit
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) bi_mbar_init(&bar, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (P.drop_copy) bi_mbar_expect(&bar, (uint32_t)(mm.P_pad * sizeof(R)));   // (testing aid: the copy never comes)
    else bi_bulk_load(L, (const R *)mm.logA + (size_t)tk.x * mm.P_pad, (uint32_t)(mm.P_pad * sizeof(R)), &bar);
  }
  // (a heavy member's units are shared by `split` threads, one in each of `split` groups of warps: a
  // warp's threads then still read the same slice row, a broadcast)
  const int upt = (int)blockDim.x / mm.split;   // units per task of this member
  const int ut = (int)threadIdx.x % upt, part = (int)threadIdx.x / upt;
  const bool has_unit = ut < tk.z;
  const int unit = has_unit ? P.perm[tk.y + ut] : 0;
  const R *q = (const R *)P.qbuf + ((size_t)cur * P.NU + unit) * P.Sp;
  R *out = (R *)P.ellp + ((size_t)mi * P.NU + unit) * P.Sp;
  if (!first) {   // beliefs of the previous update, and the right to overwrite the messages it read
    bi_grid_wait();
    bi_grid_launch_dependents();
  }
  // a copy that does not arrive within the probe limit: the block reports it and leaves (nothing of
  // its own is in flight then; the call's outputs are invalid)
  if (!bi_mbar_wait(&bar, 0, P.drop_copy ? 256 : 1 << 18)) {
    if (threadIdx.x == 0) atomicOr(P.status, BI_FLAG_COPY_TIMEOUT);
    return;
  }
  // (in a split task the threads without a unit stay for the barrier below; they contract unit 0's
  // beliefs and write nothing)
  if (!has_unit && mm.split == 1) return;
  R *sc = L + P.sc_off + threadIdx.x;   // scratch columns behind the slice
  switch (mm.shape) {
#define X(ID, RANK, D0, D1, D2, D3) \
  case ID: contract_shape<R, RANK, D0, D1, D2, D3>(L, q, out, mm.offp, mm.split, part, has_unit, sc, (int)blockDim.x); break;
    BI_BATCH_SHAPES(X)
#undef X
    default: break;
  }
  if (mm.split > 1) {   // add the parts' partial messages of the axes after the first, part 0 first
    __syncthreads();
    if (part == 0 && has_unit) {
      const R *col = L + P.sc_off + ut;
      int idx = 0;
      for (int j = 1; j < mm.rank; ++j)
        for (int i = 0; i < mm.dim[j]; ++i, ++idx) {
          R sum = col[(size_t)idx * blockDim.x];
          for (int pp = 1; pp < mm.split; ++pp) sum += col[(size_t)idx * blockDim.x + pp * upt];
          out[mm.offp[j] + i] = sum;
        }
    }
  }
}

// ---- contraction for any shape: compiled for the padded last axis only ----
// Same arithmetic as the unrolled forms.  For a row of the slice (all outer indices fixed)
// v = sum_c L[row][c] q_c[c] and acc_c[c] += W L[row][c], with W the product of the outer beliefs.  Consecutive
// rows run through the innermost outer axis: along it the accumulator of index s receives (prefix product) * v
// and a running sum receives q[s] * v; after its last index that sum climbs the other outer axes the same way.
// All indices are the same for every thread of a warp, so the branches are uniform and a slice row is a broadcast
// load.  qs / as: columns (state-major, thread-minor) holding the outer axes' beliefs per unit and message
// accumulators per thread, one entry longer than the threads, so that they can also be read along the states.
// Two rows a trip and one climb per run of rows: with an odometer over all axes advanced after every row, a warp
// took some 290 cycles per row, nearly all of them latency.
//
// Small batches do not have enough units to fill the machine with one thread
// per unit, so a CTA is tu units x rs row splits: split r contracts the rows of
// a contiguous range of the first axis' indices for the same tu units, and the
// partial messages of the splits are added through shared memory at the end
// (fixed order: deterministic).
// PERUNIT (per-agent models): nothing is shared between units, so nothing is staged; every thread
// reads the rows of its own unit's slice straight from global memory (consecutive rows of one
// thread share cache lines, so L1 serves most of the loads).
template <typename R, int NCP, bool PERUNIT>
__device__ __forceinline__ void contract_rt(const BatchMember &mm, const R *__restrict__ slice, R *Lbuf, int lbuf,
                                            R *qs, R *as, int *unit_s, const BatchParams &P, int cur, int4 tk,
                                            int mi) {
  constexpr int VE = 16 / (int)sizeof(R);
  const int tid = threadIdx.x, nt = blockDim.x, tu = P.tu, rs = nt / tu, nts = nt + 1, tus = tu + 1;
  const int u = tid % tu, r = tid / tu;
  const bool has_unit = u < tk.z;
  const int unit = has_unit ? P.perm[tk.y + u] : 0;
  if (r == 0) unit_s[u] = unit;
  const R *qbase = (const R *)P.qbuf + (size_t)cur * P.NU * P.Sp;
  const int K1 = mm.rank - 1, NC = mm.dim[K1];
  R qc[NCP], accc[NCP];
  {
    const R *q = qbase + (size_t)unit * P.Sp + mm.offp[K1];   // (offsets of factors are multiples of four: whole vectors)
#pragma unroll
    for (int c = 0; c < NCP; c += VE) {
      R v[VE];
      if (c < bi_pad4(NC)) {
        if constexpr (sizeof(R) == 8) { const double2 x = *reinterpret_cast<const double2 *>(q + c); v[0] = x.x; v[1] = x.y; }
        else { const float4 x = *reinterpret_cast<const float4 *>(q + c); v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; }
      }
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        qc[c + e] = (has_unit && c + e < NC) ? v[e] : (R)0;
        accc[c + e] = (R)0;
      }
    }
  }
  constexpr bool stage = !PERUNIT;
  __shared__ __align__(8) unsigned long long bar[8];   // one per split
  if (stage && tid < rs) bi_mbar_init(&bar[tid], 1);
  const int so = mm.ooff[K1];   // outer states of this member
  for (int i = 0; i < so; ++i) as[i * nts + tid] = (R)0;
  __syncthreads();              // (unit_s, the barriers)
  // the outer axes' beliefs, once per unit: consecutive threads read consecutive states of one unit
  for (int j = 0; j < K1; ++j) {
    const int d = mm.dim[j];
    for (int i = tid; i < d * tu; i += nt) {
      const int uu = i / d, sj = i - uu * d;
      qs[(mm.ooff[j] + sj) * tus + uu] = uu < tk.z ? qbase[(size_t)unit_s[uu] * P.Sp + mm.offp[j] + sj] : (R)0;
    }
  }
  __syncthreads();
  // this split's range of the first axis, and of rows
  const int d0 = mm.dim[0], rps = mm.rows / d0;
  const int s0a = (int)((long long)r * d0 / rs), s0b = (int)((long long)(r + 1) * d0 / rs);
  const int row_a = s0a * rps, row_b = s0b * rps;
  const int most = ((d0 + rs - 1) / rs) * rps;   // rows of the largest split: the common trip count
  const int din = mm.dim[K1 - 1], oin = mm.ooff[K1 - 1];   // the innermost outer axis
  int sin = K1 == 1 ? s0a : 0;                             // ... and the current index along it
  int dig[3] = {s0a < d0 ? s0a : 0, 0, 0};                 // indices of the other outer axes
  R p[3] = {(R)0, (R)0, (R)0}, Wp[3] = {(R)1, (R)1, (R)1}, pin = (R)0;
#pragma unroll
  for (int lv = 0; lv < 3; ++lv)
    if (lv < K1 - 1) Wp[lv] = (lv > 0 ? Wp[lv > 0 ? lv - 1 : 0] : (R)1) * qs[(mm.ooff[lv] + dig[lv]) * tus + u];
  R wpre = K1 == 1 ? (R)1 : K1 == 2 ? Wp[0] : K1 == 3 ? Wp[1] : Wp[2];
  const int lrows = PERUNIT ? most : lbuf / rs / NCP;   // rows of one split's staging area (PERUNIT: all at once)
  R *Lr = Lbuf + (size_t)r * (PERUNIT ? 0 : lrows) * NCP;
  uint32_t phase = 0;
  bool failed = false;
  const R *mine = nullptr;   // PERUNIT: this unit's slice
  if (PERUNIT && has_unit) {
    const int o = clamp_flag(P.obs[(size_t)unit * P.M + mm.modality], mm.m, P.status, BI_FLAG_OBS_RANGE);
    mine = (const R *)mm.logA + (size_t)(unit / P.T) * mm.gstride + (size_t)o * mm.P_pad;
  }
  auto one_row = [&](const R *row, int s) {
    const R qv = qs[(oin + s) * tus + u];
    const R wf = wpre * qv;
    R *acc = as + (oin + s) * nts + tid;
    const R before = *acc;
    R v0 = (R)0, v1 = (R)0;
#pragma unroll
    for (int cc = 0; cc < NCP; cc += VE) {
      R x[VE];
      if (PERUNIT) ldg_vec(row + cc, x);
      else lds_vec(row + cc, x);
#pragma unroll
      for (int i = 0; i < VE; ++i) {
        if (i & 1) v1 = fma(x[i], qc[cc + i], v1);
        else v0 = fma(x[i], qc[cc + i], v0);
        accc[cc + i] = fma(wf, x[i], accc[cc + i]);
      }
    }
    const R val = v0 + v1;
    *acc = fma(wpre, val, before);
    pin = fma(qv, val, pin);
  };
  for (int c0 = 0; c0 < most; c0 += lrows) {
    const int ra = row_a + c0;
    const int nr = max(0, min(lrows, row_b - ra));
    if (!PERUNIT) __syncthreads();   // the previous rows are consumed
    if (!PERUNIT && nr > 0) {
      // this split's rows: one bulk asynchronous copy issued by the split's first thread
      if (u == 0) bi_bulk_load(Lr, slice + (size_t)ra * NCP, (uint32_t)(nr * NCP * sizeof(R)), &bar[r]);
      if (!bi_mbar_wait(&bar[r], phase)) {
        if (u == 0) atomicOr(P.status, BI_FLAG_COPY_TIMEOUT);
        failed = true;
      }
      phase ^= 1u;
    }
    if (!has_unit || failed) continue;
    const R *row = PERUNIT ? mine + (size_t)ra * NCP : Lr;
    for (int left = nr; left > 0;) {
      const int run = min(left, din - sin);   // rows to the end of the innermost axis, or of the staged rows
      int i = 0;
      for (; i + 1 < run; i += 2, row += 2 * NCP) {
        one_row(row, sin + i);
        one_row(row + NCP, sin + i + 1);
      }
      if (i < run) { one_row(row, sin + i); row += NCP; }
      left -= run;
      sin += run;
      if (sin < din) continue;
      // the axis is through: its sum climbs the others
      sin = 0;
      R val = pin;
      pin = (R)0;
      bool act = true;
      int top = K1 - 1;
#pragma unroll
      for (int lv = 2; lv >= 0; --lv) {
        if (lv < K1 - 1 && act) {
          const int sj = dig[lv];
          R *acc = as + (mm.ooff[lv] + sj) * nts + tid;
          *acc = fma(lv > 0 ? Wp[lv > 0 ? lv - 1 : 0] : (R)1, val, *acc);
          if (lv > 0) p[lv > 0 ? lv - 1 : 0] = fma(qs[(mm.ooff[lv] + sj) * tus + u], val, p[lv > 0 ? lv - 1 : 0]);
          if (sj + 1 == mm.dim[lv]) {
            dig[lv] = 0;
            if (lv > 0) {
              val = p[lv > 0 ? lv - 1 : 0];
              p[lv > 0 ? lv - 1 : 0] = (R)0;
            }
          } else {
            dig[lv] = sj + 1;
            act = false;
          }
          top = lv;
        }
      }
      // prefix products of the outer beliefs, from the first axis whose index changed
#pragma unroll
      for (int lv = 0; lv < 3; ++lv)
        if (lv < K1 - 1 && lv >= top)
          Wp[lv] = (lv > 0 ? Wp[lv > 0 ? lv - 1 : 0] : (R)1) * qs[(mm.ooff[lv] + dig[lv]) * tus + u];
      wpre = K1 == 1 ? (R)1 : K1 == 2 ? Wp[0] : K1 == 3 ? Wp[1] : Wp[2];
    }
  }
  // ---- add the splits' partial messages and write them out (consecutive threads: consecutive states of one unit):
  // the outer axes' from the accumulator columns, then the last axis' through the same columns (free by then)
  __syncthreads();
  for (int j = 0; j < K1; ++j) {
    const int d = mm.dim[j];
    for (int i = tid; i < d * tu; i += nt) {
      const int uu = i / d, sj = i - uu * d;
      if (uu >= tk.z) continue;
      const R *col = as + (size_t)(mm.ooff[j] + sj) * nts + uu;
      R sum = col[0];
      for (int k = 1; k < rs; ++k) sum += col[k * tu];
      ((R *)P.ellp)[(int64_t)((size_t)mi * P.NU + unit_s[uu]) * P.Sp + mm.oout[j] + sj] = sum;
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < NCP; ++c) as[c * nts + tid] = accc[c];
  __syncthreads();
  for (int i = tid; i < NC * tu; i += nt) {
    const int uu = i / NC, st = i - uu * NC;
    if (uu >= tk.z) continue;
    const R *col = as + (size_t)st * nts + uu;
    R sum = col[0];
    for (int k = 1; k < rs; ++k) sum += col[k * tu];
    ((R *)P.ellp)[(int64_t)((size_t)mi * P.NU + unit_s[uu]) * P.Sp + mm.oout[K1] + st] = sum;
  }
}

// NCPMAX: the largest padded last axis among the model's members.  The forms for longer last axes
// hold that many beliefs and accumulators in registers; a model that needs none of them gets a kernel
// with half the registers, two CTAs of which share an SM.
template <typename R, bool PERUNIT, int NCPMAX>
__global__ void __launch_bounds__(256, NCPMAX <= 16 ? 2 : 1)
bi_batch_contract_rt_kernel(BatchParams P, int cur, int first) {
  // (this form reads beliefs from its first instruction on, so it waits at once)
  bi_grid_wait();
  bi_grid_launch_dependents();
  (void)first;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R *Lbuf = reinterpret_cast<R *>(smem_raw);
  R *qs = Lbuf + P.lbuf;                                   // [so_max][tu + 1] beliefs of the outer axes, per unit
  R *as = qs + (size_t)P.so_max * (P.tu + 1);               // [so_max][threads + 1] message accumulators, per thread
  int *unit_s = reinterpret_cast<int *>(as + (size_t)P.so_max * (blockDim.x + 1));
  int mi = 0;
  const int slot = (int)blockIdx.x + P.task_base;
  while (mi + 1 < P.nmem && slot >= P.mem[mi + 1].task0) ++mi;
  const BatchMember &mm = P.mem[mi];
  const int4 tk = P.task[slot];
  if (tk.z == 0) return;
  const R *slice = (const R *)mm.logA + (size_t)tk.x * mm.P_pad;
  switch (mm.ncp) {
    case 4: contract_rt<R, 4, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 8: contract_rt<R, 8, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 12: contract_rt<R, 12, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 16: contract_rt<R, 16, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 20: if constexpr (NCPMAX > 16) contract_rt<R, 20, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 24: if constexpr (NCPMAX > 16) contract_rt<R, 24, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 28: if constexpr (NCPMAX > 16) contract_rt<R, 28, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    case 32: if constexpr (NCPMAX > 16) contract_rt<R, 32, PERUNIT>(mm, slice, Lbuf, P.lbuf, qs, as, unit_s, P, cur, tk, mi); break;
    default: break;
  }
}

// ---- per unit: sum the partial messages, add rank-1 slices and transition messages, softmax ----
struct UpdateArgs {
  const int32_t *obs, *act;
  float *q_out, *logq_out;
  int32_t *argmax_out;
  int32_t T, cur, final;
  const void *lnprior;        // [N][S] log-priors used in the place of ln D at a window's first step, or NULL
  double lambda;              // damping step; 1 = plain update
  void *xprev;                // [NU][Sp] previous iterate's logits (damped calls only), or NULL
  int32_t first;              // first iteration of the call
  const float *q_init;        // warm start (for the first damped step's ln q), or NULL
  uint32_t fmask[BI_MAX_F];   // members (rank >= 2) whose group contains factor f
  uint32_t r1mask[BI_MAX_F];  // descriptor members (modalities) that depend on factor f alone
  int32_t child_plane;        // transition members: the plane of the messages to the children (-1: none of that kind)
  uint32_t pmask[BI_MAX_F];   // ... and the members with factor f among the parents
};

// Both transition messages' dot products at once: dp = sum_r Mp[r][s] qp[r] and df = sum_r Mf[r][s] qf[r],
// r < n, the matrices read [summation index][own state] from global memory (L1), the beliefs as pairs
// from shared memory (their padding entries are zero); pointers advance by additions only.
template <typename R>
__device__ __forceinline__ void edge_dots_g(const R *__restrict__ mp, const R *__restrict__ mf, int npad,
                                            const R *qp, const R *qf, int n, R &dp, R &df) {
  using V2 = typename std::conditional<sizeof(R) == 8, double2, float2>::type;
  R p0 = (R)0, p1 = (R)0, f0 = (R)0, f1 = (R)0;
  const int st2 = 2 * npad;
  int r = 0;
#pragma unroll 2
  for (; r + 1 < n; r += 2) {
    const V2 x = *reinterpret_cast<const V2 *>(qp + r), y = *reinterpret_cast<const V2 *>(qf + r);
    p0 = fma(__ldg(mp), x.x, p0); p1 = fma(__ldg(mp + npad), x.y, p1);
    f0 = fma(__ldg(mf), y.x, f0); f1 = fma(__ldg(mf + npad), y.y, f1);
    mp += st2;
    mf += st2;
  }
  if (r < n) {
    p0 = fma(__ldg(mp), qp[r], p0);
    f0 = fma(__ldg(mf), qf[r], f0);
  }
  dp = p0 + p1;
  df = f0 + f1;
}

// LW lanes per unit (the smallest power of two that holds the largest factor),
// one lane per state: for each factor in turn the lanes gather the partial
// messages, add the single-factor slices and the two transition messages, and
// normalise with shuffles inside the lane group.
struct FactorInfo {
  int32_t n, np, op, off, U;
  uint32_t fmask, r1mask;
  int32_t pad_;
};

template <int LW, typename R>
__device__ __forceinline__ R lane_group_sum(R v) {
#pragma unroll
  for (int o = LW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <int LW, typename R>
__device__ __forceinline__ R lane_group_max(R v) {
#pragma unroll
  for (int o = LW / 2; o > 0; o >>= 1) v = bi_max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// A first pass gathers, with loads that do not depend on one another (one position of the unit's
// state vector per lane and trip), everything that comes from L2: the sum of the partial messages,
// the single-factor slices, the first step's log-prior, and the two neighbouring steps' beliefs, into
// the unit's part of shared memory.  The per-factor pass then reads shared memory and the transition
// matrices (L1) only.  (With the L2 reads inside the per-factor loop every factor paid several
// dependent round trips: 35 us per launch on 20 480 units, `long_scoreboard` 8.9 stall cycles per issue.)
// FW (small batches, 32 lanes per unit): a CTA is one unit and one warp per factor, so the factors are
// updated side by side instead of one after the other: with a few thousand units the kernel is a chain
// of latencies per unit, not a matter of throughput.
// FINAL: the call's last iteration (the only one that writes outputs); DAMPED: the damped update.  Both
// are instantiations of their own: the plain iteration in between runs sixteen times a call and is
// bound by instruction issue, so it carries none of their code.  BDEP: transitions with several parents, whose
// messages were contracted with the slices (as a run-time test it cost the others a third of their time).
template <typename R, int ALGO, int LW, bool FW, bool FINAL, bool DAMPED, bool BDEP>
__global__ void __launch_bounds__(FW ? 32 * BI_MAX_F : 128)
bi_batch_update_kernel(const BiDev *__restrict__ mdp, BatchParams P, UpdateArgs A) {
  static_assert(!FW || LW == 32, "a warp per factor needs a whole warp per unit");
  __shared__ FactorInfo fi[BI_MAX_F];
  __shared__ unsigned char pfac[BI_MAX_F * 32];   // factor of each padded state position
  extern __shared__ __align__(16) unsigned char upd_smem[];
  const BiDev &md = *mdp;
  constexpr int UPB = 128 / LW;   // units per CTA
  const int F = md.F, Sp = md.Sp, S = md.S, M = md.M, T = A.T, NU = P.NU;
  if ((int)threadIdx.x < F) {
    const int f = threadIdx.x;
    FactorInfo x;
    x.n = md.n[f]; x.np = md.npad[f]; x.op = md.offp[f]; x.off = md.off[f]; x.U = md.U[f];
    x.fmask = A.fmask[f]; x.r1mask = A.r1mask[f]; x.pad_ = 0;
    fi[f] = x;
  }
  for (int p = threadIdx.x; p < Sp; p += blockDim.x) {
    int f = 0;
    while (f + 1 < F && p >= md.offp[f + 1]) ++f;
    pfac[p] = (unsigned char)f;
  }
  __syncthreads();
  bi_grid_wait();   // the contraction's messages (and, for the beliefs, everything before it)
  bi_grid_launch_dependents();
  const int sub = FW ? 0 : threadIdx.x / LW, s = threadIdx.x % LW;
  int unit = FW ? (int)blockIdx.x : blockIdx.x * UPB + sub;
  const bool live = unit < NU;    // dead groups shadow the last unit so that whole warps reach the shuffles
  if (!live) unit = NU - 1;
  const int a = unit / T, t = unit - a * T;
  const int g = md.G == 1 ? 0 : a;   // per-agent models: this agent's matrices and slices
  const R *qc = (const R *)P.qbuf + (size_t)A.cur * NU * Sp;
  R *qn = (R *)P.qbuf + ((size_t)(A.cur ^ 1) * NU + unit) * Sp;
  const int32_t *ob = A.obs + (size_t)unit * M;
  // acp[f]: action into step t (t > 0); acp[F + f]: action out of it (t + 1 < T)
  const int32_t *acp = A.act + ((ptrdiff_t)a * (T - 1) + (t - 1)) * F;
  R *base = reinterpret_cast<R *>(upd_smem) + (size_t)sub * 3 * Sp;   // [Sp] logit constants, [Sp] q(t-1), [Sp] q(t+1)
  R *qprev = base + Sp, *qnext = base + 2 * Sp;
  for (int p = FW ? (int)threadIdx.x : s; p < Sp; p += FW ? (int)blockDim.x : LW) {
    const int f = pfac[p];
    const FactorInfo I = fi[f];
    const int sl = p - I.op;
    R x = (R)0;
    if (sl < I.n) {
      const R *ep = (const R *)P.ellp + (size_t)unit * Sp + p;   // member j's entry: NU * Sp elements further per j
      const size_t mstride = (size_t)NU * Sp;
      for (uint32_t mk = I.fmask; mk; mk &= mk - 1) x += ep[(__ffs(mk) - 1) * mstride];
      if (BDEP) {
        if (t > 0) x += ep[A.child_plane * mstride];
        if (t + 1 < T)
          for (uint32_t mk = A.pmask[f]; mk; mk &= mk - 1) x += ep[(__ffs(mk) - 1) * mstride];
      }
      for (uint32_t mk = I.r1mask; mk; mk &= mk - 1) {   // single-factor modalities: the slice is the message
        const BiMember &mm = md.mem[__ffs(mk) - 1];
        const int o = clamp_flag(ob[mm.modality], mm.m, md.status, BI_FLAG_OBS_RANGE);
        x += __ldg((const R *)mm.logA + (size_t)g * mm.gstride + (size_t)o * mm.P_pad + sl);
      }
      if (t == 0)
        x += A.lnprior ? ((const R *)A.lnprior)[(size_t)a * S + I.off + sl]
                       : ((const R *)md.logD[f])[(size_t)g * md.Dstride[f] + sl];
    }
    base[p] = x;
    qprev[p] = t > 0 ? qc[(size_t)(unit - 1) * Sp + p] : (R)0;
    qnext[p] = t + 1 < T ? qc[(size_t)(unit + 1) * Sp + p] : (R)0;
  }
  if (FW) __syncthreads();
  else __syncwarp();
  for (int f = FW ? (int)(threadIdx.x >> 5) : 0; f < F; f += FW ? BI_MAX_F : 1) {
    const FactorInfo I = fi[f];
    const int n = I.n, np = I.np, op = I.op;
    R x = -bi_inf<R>();
    if (BDEP && s < n) x = base[op + s];
    if (!BDEP && s < n) {
      x = base[op + s];
      // both edges are evaluated (a window's end reads zeros and discards the result)
      const int up = t > 0 ? clamp_flag(acp[f], I.U, md.status, BI_FLAG_ACT_RANGE) : 0;
      const int uf = t + 1 < T ? clamp_flag(acp[F + f], I.U, md.status, BI_FLAG_ACT_RANGE) : 0;
      const R *M0 = (const R *)(ALGO == BI_ALGO_VMP ? md.logBt[f] : md.BfT[f]);   // [previous][next]
      const R *M1 = (const R *)(ALGO == BI_ALGO_VMP ? md.logB[f] : md.BdagT[f]);   // [next][previous]
      const size_t mo = (size_t)g * md.Bstride[f] + s;
      R dp, df;
      edge_dots_g<R>(M0 + mo + up * n * np, M1 + mo + uf * n * np, np, qprev + op, qnext + op, n, dp, df);
      if (ALGO == BI_ALGO_MMP) {
        dp = (R)0.5 * bi_log_inline(bi_max(dp, (R)BI_EPS));
        df = (R)0.5 * bi_log_inline(bi_max(df, (R)BI_EPS));
      }
      x += (t > 0 ? dp : (R)0) + (t + 1 < T ? df : (R)0);
    }
    if (DAMPED) {
      // damped step on the logits; the first one starts from ln q of the starting belief (uniform: a
      // constant, taken as 0)
      R *xp = (R *)A.xprev + (size_t)unit * Sp + op;
      if (s < n) {
        R prev = (R)0;
        if (!A.first) prev = xp[s];
        else if (A.q_init) prev = bi_log(bi_max((R)A.q_init[(size_t)unit * S + I.off + s], (R)BI_EPS));
        x = fma((R)A.lambda, x, ((R)1 - (R)A.lambda) * prev);
        if (live) xp[s] = x;
      }
    }
    // any shift near the maximum keeps the exponentials in range; the last iterate takes the exact one
    const R mx = FINAL ? lane_group_max<LW>(x) : (R)lane_group_max<LW>((float)x);
    const R e = s < n ? bi_exp_inline(x - mx) : (R)0;
    const R z = lane_group_sum<LW>(e);
    const R q = e * bi_rcp(z);
    if (live && s < np) qn[op + s] = q;
    if (FINAL) {
      if (live && s < n) {
        A.q_out[(size_t)unit * S + I.off + s] = (float)q;
        if (A.logq_out) A.logq_out[(size_t)unit * S + I.off + s] = (float)(x - mx - bi_log(z));
      }
      if (A.argmax_out) {
        unsigned b = __ballot_sync(0xffffffffu, s < n && x == mx);
        if (LW < 32) b = (b >> ((threadIdx.x & 31) - s)) & ((1u << (LW & 31)) - 1u);
        if (live && s == 0) A.argmax_out[(size_t)unit * F + f] = __ffs(b) - 1;
      }
    }
  }
}

// The same for batches that fill the machine with one thread per (unit, factor), on shared models.  A CTA takes 32
// consecutive units, a warp per factor and a lane per unit.  The units' rows (messages summed over the members,
// the neighbours' beliefs) are one contiguous run of memory: they come through shared memory with coalesced
// loads, the new beliefs leave the same way.  A lane keeps its unit's states of the factor in registers, so sums and
// softmax need no shuffles; the factors' transition matrices, every action's, sit in shared memory (a pad of
// 16 bytes between actions puts the rows that a warp's units read for different actions on different banks, so
// a 16-byte load serves 32 units with two entries each).  The lane-group form above issues a 16-lane dot product
// per unit and state and waits for it: 20 480 units of 34 states took 38 us.
// NP: states in registers (the model's largest factor, padded).
struct UnitUpdate {   // shared-memory layout, elements
  int32_t mat[BI_MAX_F], xs, qs, stride;   // matrices of each factor; the units' logits; beliefs of units -1 .. 32; row stride
};
template <typename R>
__device__ __forceinline__ void vec_add(R *x, const R *p) {
  if constexpr (sizeof(R) == 8) {
    const double2 v = *reinterpret_cast<const double2 *>(p);
    x[0] += v.x; x[1] += v.y;
  } else {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    x[0] += v.x; x[1] += v.y; x[2] += v.z; x[3] += v.w;
  }
}
template <typename R, int ALGO, int NP, bool FINAL, bool DAMPED>
__global__ void __launch_bounds__(32 * BI_MAX_F)
bi_batch_update_unit_kernel(const BiDev *__restrict__ mdp, BatchParams P, UpdateArgs A, UnitUpdate L) {
  extern __shared__ __align__(16) unsigned char upd_smem[];
  __shared__ unsigned char pfac[BI_MAX_F * 32];   // factor of each padded state position
  R *sm = reinterpret_cast<R *>(upd_smem);
  const BiDev &md = *mdp;
  constexpr int VE = 16 / (int)sizeof(R);
  const int F = md.F, Sp = md.Sp, S = md.S, M = md.M, T = A.T, NU = P.NU;
  const int f = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = md.n[f], np = md.npad[f], op = md.offp[f], off = md.off[f], U = md.U[f];
  const int msz = np * np, mst = msz + VE;   // (rows padded like columns; the padding rows are zero)
  R *M0 = sm + L.mat[f], *M1 = M0 + (size_t)U * mst;
  if (A.child_plane < 0) {
    const R *s0 = (const R *)(ALGO == BI_ALGO_VMP ? md.logBt[f] : md.BfT[f]);   // [previous][next]
    const R *s1 = (const R *)(ALGO == BI_ALGO_VMP ? md.logB[f] : md.BdagT[f]);   // [next][previous]
    for (int u = 0; u < U; ++u)
      for (int e = lane; e < msz; e += 32) {
        const bool in = e < n * np;
        M0[u * mst + e] = in ? __ldg(s0 + (size_t)u * n * np + e) : (R)0;
        M1[u * mst + e] = in ? __ldg(s1 + (size_t)u * n * np + e) : (R)0;
      }
  }
  for (int p = lane; p < np; p += 32) pfac[op + p] = (unsigned char)f;
  __syncthreads();
  bi_grid_wait();   // the contraction's messages (and, for the beliefs, everything before it)
  bi_grid_launch_dependents();
  // ---- rows in: summed messages, and the beliefs of the units from one before to one after
  const int u0 = blockIdx.x * 32, nu = min(32, NU - u0), hv = Sp / VE;
  const size_t mstride = (size_t)NU * Sp;
  for (int i = threadIdx.x; i < nu * hv; i += blockDim.x) {
    const int ul = i / hv, p = (i - ul * hv) * VE, fp = pfac[p];
    const R *ep = (const R *)P.ellp + (size_t)u0 * Sp + (size_t)i * VE;   // member j's entry: NU * Sp elements further per j
    R x[VE];
#pragma unroll
    for (int e = 0; e < VE; ++e) x[e] = (R)0;
    uint32_t mk = A.fmask[fp];
    if (A.child_plane >= 0) {   // transitions with several parents: their messages were contracted with the slices
      const int t = (u0 + ul) % T;
      if (t > 0) vec_add(x, ep + A.child_plane * mstride);
      if (t + 1 < T) mk |= A.pmask[fp];
    }
    for (; mk; mk &= mk - 1) vec_add(x, ep + (__ffs(mk) - 1) * mstride);
#pragma unroll
    for (int e = 0; e < VE; ++e) sm[L.xs + ul * L.stride + p + e] = x[e];
  }
  if (A.child_plane < 0) {
    const R *qc = (const R *)P.qbuf + (size_t)A.cur * NU * Sp;
    for (int i = threadIdx.x; i < (nu + 2) * hv; i += blockDim.x) {
      const int ul = i / hv, p = (i - ul * hv) * VE, u = u0 + ul - 1;
      R x[VE];
#pragma unroll
      for (int e = 0; e < VE; ++e) x[e] = (R)0;
      if (u >= 0 && u < NU) vec_add(x, qc + (size_t)u * Sp + p);
#pragma unroll
      for (int e = 0; e < VE; ++e) sm[L.qs + ul * L.stride + p + e] = x[e];
    }
  }
  __syncthreads();
  // ---- one unit and factor per lane
  const bool live = lane < nu;
  const int ul = live ? lane : 0, unit = u0 + ul;
  const int a = unit / T, t = unit - a * T;
  const bool has_prev = t > 0, has_next = t + 1 < T;
  R *xrow = sm + L.xs + ul * L.stride + op;
  R x[NP];
#pragma unroll
  for (int s = 0; s < NP; ++s) x[s] = (R)0;
  auto add_row = [&](const R *row) {
#pragma unroll
    for (int s = 0; s < NP; s += VE)
      if (s < np) vec_add(x + s, row + s);
  };
  add_row(xrow);
  for (uint32_t mk = A.r1mask[f]; mk; mk &= mk - 1) {
    const BiMember &mm = md.mem[__ffs(mk) - 1];
    const int o = clamp_flag(A.obs[(size_t)unit * M + mm.modality], mm.m, md.status, BI_FLAG_OBS_RANGE);
    add_row((const R *)mm.logA + (size_t)o * mm.P_pad);
  }
  if (!has_prev) {
    if (A.lnprior) {
#pragma unroll
      for (int s = 0; s < NP; ++s)
        if (s < n) x[s] += ((const R *)A.lnprior)[(size_t)a * S + off + s];
    } else {
      add_row((const R *)md.logD[f]);
    }
  }
  // both transition messages: acc[s] += sum_r M[r][s] q[r] (a window's ends add nothing)
  if (A.child_plane < 0) {
    const int32_t *acp = A.act + ((ptrdiff_t)a * (T - 1) + (t - 1)) * F + f;
    auto edge = [&](bool real, const R *Mx, const int32_t *ac, const R *q, R (&acc)[NP]) {
      const int u = real ? clamp_flag(*ac, U, md.status, BI_FLAG_ACT_RANGE) : 0;
      const R *row = Mx + u * mst;
#pragma unroll 2
      for (int r = 0; r < np; r += VE, row += VE * np) {
        R w[VE];
        lds_vec(q + r, w);
#pragma unroll
        for (int k = 0; k < VE; ++k) {
          const R wk = real ? w[k] : (R)0;
#pragma unroll
          for (int s = 0; s < NP; s += VE) {
            if (s < np) {
              R m[VE];
              lds_vec(row + k * np + s, m);
#pragma unroll
              for (int e = 0; e < VE; ++e) acc[s + e] = fma(m[e], wk, acc[s + e]);
            }
          }
        }
      }
    };
    const R *q0 = sm + L.qs + ul * L.stride + op, *q1 = q0 + 2 * L.stride;
    if (ALGO == BI_ALGO_VMP) {
      edge(has_prev, M0, acp, q0, x);
      edge(has_next, M1, acp + F, q1, x);
    } else {
#pragma unroll 1
      for (int d = 0; d < 2; ++d) {
        const bool real = d == 0 ? has_prev : has_next;
        R m[NP];
#pragma unroll
        for (int s = 0; s < NP; ++s) m[s] = (R)0;
        edge(real, d == 0 ? M0 : M1, d == 0 ? acp : acp + F, d == 0 ? q0 : q1, m);
#pragma unroll
        for (int s = 0; s < NP; ++s)
          if (s < n) x[s] += real ? (R)0.5 * bi_log_inline(bi_max(m[s], (R)BI_EPS)) : (R)0;
      }
    }
  }
  if (DAMPED) {   // as in the lane-group form
    R *xp = (R *)A.xprev + (size_t)unit * Sp + op;
#pragma unroll
    for (int s = 0; s < NP; ++s) {
      if (s < n && live) {
        R prev = (R)0;
        if (!A.first) prev = xp[s];
        else if (A.q_init) prev = bi_log(bi_max((R)A.q_init[(size_t)unit * S + off + s], (R)BI_EPS));
        x[s] = fma((R)A.lambda, x[s], ((R)1 - (R)A.lambda) * prev);
        xp[s] = x[s];
      }
    }
  }
  R mx;
  if (FINAL) {
    mx = x[0];
#pragma unroll
    for (int s = 1; s < NP; ++s)
      if (s < n) mx = bi_max(mx, x[s]);
  } else {   // (any shift near the maximum keeps the exponentials in range)
    float m = (float)x[0];
#pragma unroll
    for (int s = 1; s < NP; ++s)
      if (s < n) m = fmaxf(m, (float)x[s]);
    mx = (R)m;
  }
  R e[NP], z0 = (R)0, z1 = (R)0;
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    e[s] = s < n ? bi_exp_inline(x[s] - mx) : (R)0;
    if (s & 1) z1 += e[s];
    else z0 += e[s];
  }
  const R z = z0 + z1, rz = bi_rcp(z);
#pragma unroll
  for (int s = 0; s < NP; ++s)
    if (s < np && live) xrow[s] = e[s] * rz;   // (the lane's own entries: nobody else reads them before the barrier)
  if (FINAL && live) {
    const R lz = A.logq_out ? bi_log(z) : (R)0;
    int am = 0;
    bool found = false;
#pragma unroll
    for (int s = 0; s < NP; ++s) {
      if (s < n) {
        A.q_out[(size_t)unit * S + off + s] = (float)(e[s] * rz);
        if (A.logq_out) A.logq_out[(size_t)unit * S + off + s] = (float)(x[s] - mx - lz);
        if (!found && x[s] == mx) { am = s; found = true; }
      }
    }
    if (A.argmax_out) A.argmax_out[(size_t)unit * F + f] = am;
  }
  if (!FINAL) {   // rows out
    __syncthreads();
    R *qn = (R *)P.qbuf + ((size_t)(A.cur ^ 1) * NU + u0) * Sp;
    for (int i = threadIdx.x; i < nu * hv; i += blockDim.x) {
      const int ul2 = i / hv, p = (i - ul2 * hv) * VE;
      const R *src = sm + L.xs + ul2 * L.stride + p;
      if constexpr (sizeof(R) == 8) *reinterpret_cast<double2 *>(qn + (size_t)i * VE) = *reinterpret_cast<const double2 *>(src);
      else *reinterpret_cast<float4 *>(qn + (size_t)i * VE) = *reinterpret_cast<const float4 *>(src);
    }
  }
}

template <typename R>
__global__ void bi_batch_init_kernel(const BiDev *__restrict__ mdp, R *q, int NU, const float *__restrict__ q_init) {
  bi_grid_launch_dependents();
  const BiDev &md = *mdp;
  const size_t total = (size_t)NU * md.Sp;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int p = (int)(i % md.Sp);
    int f = 0;
    while (f + 1 < md.F && p >= md.offp[f + 1]) ++f;
    const int s = p - md.offp[f];
    R v = (R)0;
    if (s < md.n[f]) v = q_init ? (R)q_init[(i / md.Sp) * md.S + md.off[f] + s] : (R)1 / (R)md.n[f];
    q[i] = v;
  }
}

template <typename R>
int batch_start(const bi_model *md, const BatchParams &P, int max_m, const float *q_init, int32_t *perm, int4 *task,
                cudaStream_t stream) {
  bi_batch_init_kernel<R><<<256, 256, 0, stream>>>(md->d, (R *)P.qbuf, P.NU, q_init);
  if (P.nmem == 0) return BI_OK;
  cudaLaunchAttribute early[1];
  early[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(P.nmem * kBucketCtas));
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = 4 * max_m * sizeof(int32_t);
  if (cfg.dynamicSmemBytes > 48 * 1024 &&
      bi_allow_smem((const void *)bi_batch_bucket_kernel, cfg.dynamicSmemBytes) != cudaSuccess)
    return BI_ERR_CUDA;
  cfg.stream = stream;
  cfg.attrs = early;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, bi_batch_bucket_kernel, P, P.obs, (int)P.M, P.status, perm, task) == cudaSuccess ? BI_OK : BI_ERR_CUDA;
}

int shape_of(const BiGroup &g) {
  const int d[4] = {g.rank > 0 ? g.dim[0] : 0, g.rank > 1 ? g.dim[1] : 0, g.rank > 2 ? g.dim[2] : 0,
                    g.rank > 3 ? g.dim[3] : 0};
#define X(ID, RANK, D0, D1, D2, D3) \
  if (g.rank == RANK && d[0] == D0 && d[1] == D1 && d[2] == D2 && d[3] == D3) return ID;
  BI_BATCH_SHAPES(X)
#undef X
  return -1;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

template <typename R>
int launch_batch_t(const BiCall &c, bi_model *mut) {
  const bi_model *md = c.model;
  const BiDev &h = md->h;
  const int NU = c.N * c.T;
  BatchParams P;
  memset(&P, 0, sizeof(P));
  // units per contraction CTA: small enough that the heaviest member alone gives every SM a CTA
  int tu = kTU;
  while (tu > 32 && NU / tu < md->sm_count) tu >>= 1;
  P.tu = tu;
  UpdateArgs A;
  memset(&A, 0, sizeof(A));
  // members of rank >= 2, largest slices first (their tasks are the longest)
  int order[BI_MAX_M], cnt = 0;
  const bool per_unit = h.G != 1;   // per-agent models: every unit contracts its own slice
  A.child_plane = -1;
  constexpr bool f32 = sizeof(R) == 4;   // (float64 comes here with a slice per unit, groups over five factors or four parents only)
  bool any_shape = per_unit || !f32;     // (also set when some group has no unrolled form)
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank < 2) continue;
    if (g.rank > BI_MAX_RANK) return BI_ERR_UNSUPPORTED;
    if (shape_of(g) < 0) any_shape = true;
    for (int mi = g.mem_begin; mi < g.mem_end; ++mi) order[cnt++] = mi;
  }
  // (cnt == 0: every modality depends on a single factor; the update kernel alone does the work)
  std::sort(order, order + cnt, [&](int x, int y) { return h.mem[x].P_pad > h.mem[y].P_pad; });
  size_t max_slice = 0;
  int max_m = 1, so_max = 1, ncp_max = 4;
  for (int j = 0; j < cnt; ++j) {
    const BiMember &mm = h.mem[order[j]];
    int gi = 0;
    while (!(order[j] >= h.grp[gi].mem_begin && order[j] < h.grp[gi].mem_end)) ++gi;
    const BiGroup &g = h.grp[gi];
    BatchMember &bm = P.mem[j];
    bm.edge = 0;
    bm.logA = mm.logA; bm.m = mm.m; bm.P_pad = mm.P_pad; bm.modality = mm.modality;
    bm.gstride = mm.gstride;
    bm.shape = shape_of(g); bm.rank = g.rank;
    int so = 0, rows = 1;
    for (int k = 0; k < g.rank; ++k) {
      bm.offp[k] = h.offp[g.axis[k]];
      bm.oout[k] = h.offp[g.axis[k]];
      bm.dim[k] = g.dim[k];
      bm.ooff[k] = so;
      if (k + 1 < g.rank) { so += g.dim[k]; rows *= g.dim[k]; }
      A.fmask[g.axis[k]] |= 1u << j;
    }
    bm.ncp = bi_pad4(g.dim[g.rank - 1]);
    bm.rows = rows;
    bm.split = 1;
    if ((long long)rows * bm.ncp != mm.P_pad || bm.ncp > 32) return BI_ERR_UNSUPPORTED;
    so_max = std::max(so_max, so);
    ncp_max = std::max(ncp_max, (int)bm.ncp);
    max_slice = std::max(max_slice, (size_t)mm.P_pad * sizeof(R));
    max_m = std::max(max_m, mm.m);
  }
  // transitions with several parents: members behind the slices, always on the any-shape form
  const int nslice = cnt;
  const size_t max_slice_u = max_slice;
  if (h.has_bdep) A.child_plane = cnt + h.F;   // (also for windows of one step, which have no transitions at all)
  if (h.has_bdep && c.T > 1) {
    for (int f = 0; f < h.F; ++f, ++cnt) {
      BatchMember &bm = P.mem[cnt];
      const int k = h.bdep_len[f], r = k + 1;
      if (r > BI_MAX_RANK || per_unit) return BI_ERR_UNSUPPORTED;
      bm.edge = 1 + f;
      bm.logA = h.logBedge[f]; bm.m = h.U[f];
      bm.modality = 0; bm.gstride = 0;
      bm.shape = -1; bm.rank = r; bm.split = 1;
      // first axis: the child's next state (one unit on), then the parents in list order, the last one padded
      int so = 0, rows = 1;
      for (int j = 0; j < r; ++j) {
        const int fa = j == 0 ? f : h.bdep[f][j - 1];
        bm.dim[j] = h.n[fa];
        bm.offp[j] = h.offp[fa] + (j == 0 ? h.Sp : 0);
        bm.oout[j] = h.offp[fa];
        if (j == 0) bm.oout[j] += ((int64_t)(A.child_plane - cnt) * NU + 1) * h.Sp;
        else A.pmask[fa] |= 1u << cnt;
        bm.ooff[j] = so;
        if (j + 1 < r) { so += bm.dim[j]; rows *= bm.dim[j]; }
      }
      bm.ncp = bi_pad4(bm.dim[r - 1]);
      bm.rows = rows;
      bm.P_pad = rows * bm.ncp;
      so_max = std::max(so_max, so);
      ncp_max = std::max(ncp_max, (int)bm.ncp);
      max_slice = std::max(max_slice, (size_t)bm.P_pad * sizeof(R));
      max_m = std::max(max_m, (int)bm.m);
    }
  }
  const bool edges = cnt > nslice;
  const bool use_rt = any_shape || edges;   // (the unrolled form for the slices, if they have it, beside the any-shape one)
  if (max_m > 4096) return BI_ERR_UNSUPPORTED;
  // shared memory and shape of a contraction CTA
  size_t csmem = max_slice;
  int rs = 1;
  if (use_rt) {
    // row splits: enough warps for about two per scheduler when the batch is small
    if (tu == 32) rs = NU <= 32 * 4 * md->sm_count ? 8 : 4;
    else if (tu == 64) rs = 2;
    // a column per unit (beliefs) and one per thread (message accumulators; at least 32 rows: they also
    // carry the last axis' partial messages to the final sum) for every outer state, and a staging area
    // of whole rows per split: 48 KB at most, and less when that lets a second CTA share the SM (the
    // kernel's loops are chains of shared-memory round trips: with one CTA of eight warps per SM it
    // issued on 29 % of the cycles); fewer splits, then fewer units, when even that does not fit
    P.so_max = std::max(so_max, 32);
    for (;;) {
      const size_t cols = ((size_t)P.so_max * (tu + 1) + (size_t)P.so_max * (tu * rs + 1)) * sizeof(R) + (size_t)tu * sizeof(int);
      size_t stage = std::min<size_t>(max_slice, 48 * 1024);
      const size_t half_sm = ((size_t)md->max_smem_optin + 1024) / 2 - 1024 - 1024;   // two CTAs, their reserved 1 KB each
      if (ncp_max <= 16 && cols + stage > half_sm && cols + 8 * 1024 <= half_sm) stage = half_sm - cols;
      P.lbuf = (int)(stage / sizeof(R));
      P.lbuf = std::max(P.lbuf / (32 * rs) * (32 * rs), 32 * rs);
      csmem = cols + (size_t)P.lbuf * sizeof(R);
      if (csmem <= (size_t)md->max_smem_optin - 1024) break;
      if (rs > 1) rs >>= 1;
      else if (tu > 32) tu >>= 1;
      else break;
    }
    P.tu = tu;
  }
  if (csmem > (size_t)md->max_smem_optin - 1024) return BI_ERR_UNSUPPORTED;
  // Unrolled forms: a member whose contraction is several thousand multiply-adds per unit is shared by
  // two threads per unit (halves of the first axis, in different warps), so that the schedulers that
  // get one more of its warps than the rest do not set the time.  (Measured on a rank-4 group of 4800
  // entries, 20 480 units: 1.32 ms per call unsplit, 1.23 ms in halves, 1.27 ms in quarters; lanes of one
  // warp sharing a unit, which turns the slice rows' broadcast loads into four different rows, 2.3 ms.)
  size_t usmem = max_slice_u;   // the unrolled form's
  if (!any_shape)
    for (int j = 0; j < nslice; ++j) {
      BatchMember &bm = P.mem[j];
      const long long fm = 2LL * bm.P_pad;
      int sp = fm >= 4000 ? 2 : 1;
      if (bm.rank == 3 && sp > 2) sp = 2;
      if (bm.rank < 3) sp = 1;
      while (sp > 1 && (bm.dim[0] < sp || (tu / sp) % 32 != 0)) sp >>= 1;   // (whole warps per part)
      bm.split = sp;
      if (sp > 1) {
        int ns = 0;
        for (int k = 1; k < bm.rank; ++k) ns += bm.dim[k];
        P.sc_off = (int)((max_slice_u / sizeof(R) + 1) & ~(size_t)1);
        usmem = std::max(usmem, ((size_t)P.sc_off + (size_t)ns * tu) * sizeof(R));
      }
    }
  if (std::max(use_rt ? csmem : 0, any_shape ? 0 : usmem) > (size_t)md->max_smem_optin - 1024) return BI_ERR_UNSUPPORTED;
  int ntask = 0;
  long long nperm = 0;
  for (int j = 0; j < cnt; ++j) {
    P.mem[j].task0 = ntask;
    P.mem[j].perm0 = (int)nperm;
    const int tum = P.mem[j].tu = tu / P.mem[j].split;
    const int slots = (NU + tum - 1) / tum + P.mem[j].m;
    ntask += slots;
    nperm += (long long)slots * tum;
  }
  if (nperm > INT_MAX) return BI_ERR_UNSUPPORTED;
  const int ntask_slices = edges ? P.mem[nslice].task0 : ntask;
  P.nmem = cnt; P.NU = NU; P.Sp = h.Sp; P.ntask = ntask;

  // ---- workspace (stream-ordered; kept in the handle and grown on demand)
  const size_t b_perm = up256((size_t)nperm * sizeof(int32_t));
  const size_t b_task = up256((size_t)ntask * sizeof(int4));
  const size_t b_ellp = up256((size_t)(cnt + (edges ? 1 : 0)) * NU * h.Sp * sizeof(R));
  const size_t b_q = up256(2 * (size_t)NU * h.Sp * sizeof(R));
  const size_t b_x = c.lambda != 1.0 ? up256((size_t)NU * h.Sp * sizeof(R)) : 0;
  const size_t need = b_perm + b_task + b_ellp + b_q + b_x;
  if (const int rc = bi_workspace(mut, need, c.stream)) return rc;
  unsigned char *w = static_cast<unsigned char *>(mut->ws);
  int32_t *perm = reinterpret_cast<int32_t *>(w);
  int4 *task = reinterpret_cast<int4 *>(w + b_perm);
  P.perm = perm;
  P.task = task;
  P.ellp = w + b_perm + b_task;
  P.qbuf = w + b_perm + b_task + b_ellp;
  P.status = h.status;
  P.drop_copy = 0;
  if (mut->test_drop_copy > 0) {   // testing aid: this many calls lose their copies
    P.drop_copy = 1;
    mut->test_drop_copy -= 1;
  }
  P.obs = c.obs; P.M = h.M; P.T = c.T; P.F = h.F; P.act = c.act;
  A.obs = c.obs; A.act = c.act; A.q_out = c.q_out; A.logq_out = c.logq_out; A.argmax_out = c.argmax_out;
  A.T = c.T;
  A.lnprior = c.lnprior;
  A.lambda = c.lambda;
  A.xprev = b_x ? w + b_perm + b_task + b_ellp + b_q : nullptr;
  A.q_init = c.q_init;

  if (cnt > 0 && !per_unit) {
    const int rc = batch_start<R>(md, P, max_m, c.q_init, perm, task, c.stream);
    if (rc != BI_OK) return rc;
  } else {
    bi_batch_init_kernel<R><<<256, 256, 0, c.stream>>>(md->d, (R *)P.qbuf, NU, c.q_init);
    if (cnt > 0) bi_batch_identity_tasks_kernel<<<dim3(64, cnt), 256, 0, c.stream>>>(P, perm, task);
  }
  typedef void (*ContractKernel)(BatchParams, int, int);
  const ContractKernel rt = per_unit ? (ncp_max <= 16 ? bi_batch_contract_rt_kernel<R, true, 16> : bi_batch_contract_rt_kernel<R, true, 32>)
                                     : (ncp_max <= 16 ? bi_batch_contract_rt_kernel<R, false, 16> : bi_batch_contract_rt_kernel<R, false, 32>);
  ContractKernel unrolled = nullptr;
  if constexpr (f32) unrolled = bi_batch_contract_kernel<R>;
  if (use_rt && bi_allow_smem((const void *)rt, csmem) != cudaSuccess)
    return BI_ERR_CUDA;
  if (!any_shape && bi_allow_smem((const void *)unrolled, usmem) != cudaSuccess)
    return BI_ERR_CUDA;
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank != 1) continue;
    for (int mi = g.mem_begin; mi < g.mem_end; ++mi) A.r1mask[g.axis[0]] |= 1u << mi;
  }
  int nmax = 1;
  for (int f = 0; f < h.F; ++f) nmax = std::max(nmax, (int)h.n[f]);
  const int lw = nmax <= 8 ? 8 : nmax <= 16 ? 16 : 32, upb = 128 / lw;
  typedef void (*UpdateKernel)(const BiDev *, BatchParams, UpdateArgs);
  const bool fw = lw == 32 && NU <= 64 * md->sm_count;   // a few thousand units: a warp per factor (see the kernel)
  const bool damped = A.xprev != nullptr;
  auto pick = [&](bool fin) -> UpdateKernel {
#define BI_UPD(AL, LWV, FWV, BD) \
    (fin ? (damped ? (UpdateKernel)bi_batch_update_kernel<R, AL, LWV, FWV, true, true, BD>   \
                   : (UpdateKernel)bi_batch_update_kernel<R, AL, LWV, FWV, true, false, BD>) \
         : (damped ? (UpdateKernel)bi_batch_update_kernel<R, AL, LWV, FWV, false, true, BD>  \
                   : (UpdateKernel)bi_batch_update_kernel<R, AL, LWV, FWV, false, false, BD>))
#define BI_UPL(AL, BD) \
    (fw ? BI_UPD(AL, 32, true, BD) : lw == 8 ? BI_UPD(AL, 8, false, BD) \
                                   : lw == 16 ? BI_UPD(AL, 16, false, BD) : BI_UPD(AL, 32, false, BD))
    if (h.has_bdep) return BI_UPL(BI_ALGO_VMP, true);
    if (c.algo == BI_ALGO_VMP) return BI_UPL(BI_ALGO_VMP, false);
    return BI_UPL(BI_ALGO_MMP, false);
#undef BI_UPL
#undef BI_UPD
  };
  const UpdateKernel update_mid = pick(false), update_last = pick(true);
  // a lane per unit and a warp per factor: shared models of up to 16 states per factor whose matrices fit beside
  // the units' rows twice per SM, from about two CTAs and six warps per SM on (below that the form above has
  // more warps: one factor of four states, 12 405 units, 86 against 107 us a call); not in
  // float32 with zeros in A, where the order of sums is kept (see bi_block_serves)
  typedef void (*UnitKernel)(const BiDev *, BatchParams, UpdateArgs, UnitUpdate);
  UnitKernel unit_mid = nullptr, unit_last = nullptr;
  UnitUpdate UL;
  memset(&UL, 0, sizeof(UL));
  size_t unit_smem = 0;
  if constexpr (f32) if (h.G == 1 && nmax <= 16 && NU >= 64 * md->sm_count && (long long)NU * h.F >= 192LL * md->sm_count && !md->has_zeros) {
    constexpr int VE = 16 / (int)sizeof(R);
    size_t o = 0;
    for (int f = 0; f < h.F; ++f) {
      UL.mat[f] = (int)o;
      if (!h.has_bdep) o += 2 * (size_t)h.U[f] * ((size_t)h.npad[f] * h.npad[f] + VE);
      if (o > 100 * 1024) break;
    }
    UL.stride = ((h.Sp / VE) | 1) * VE;   // an odd number of 16-byte units: the lanes' rows on different banks
    UL.xs = (int)o; o += 32 * (size_t)UL.stride;
    UL.qs = (int)o; o += h.has_bdep ? 0 : 34 * (size_t)UL.stride;
    unit_smem = o * sizeof(R);
    if (unit_smem <= 100 * 1024) {
      auto pick_unit = [&](bool fin) -> UnitKernel {
#define BI_UPT(AL, NPV) \
    (fin ? (damped ? (UnitKernel)bi_batch_update_unit_kernel<R, AL, NPV, true, true>   \
                   : (UnitKernel)bi_batch_update_unit_kernel<R, AL, NPV, true, false>) \
         : (damped ? (UnitKernel)bi_batch_update_unit_kernel<R, AL, NPV, false, true>  \
                   : (UnitKernel)bi_batch_update_unit_kernel<R, AL, NPV, false, false>))
        if (c.algo == BI_ALGO_VMP) return nmax <= 8 ? BI_UPT(BI_ALGO_VMP, 8) : nmax <= 12 ? BI_UPT(BI_ALGO_VMP, 12) : BI_UPT(BI_ALGO_VMP, 16);
        return nmax <= 8 ? BI_UPT(BI_ALGO_MMP, 8) : nmax <= 12 ? BI_UPT(BI_ALGO_MMP, 12) : BI_UPT(BI_ALGO_MMP, 16);
#undef BI_UPT
      };
      unit_mid = pick_unit(false);
      unit_last = pick_unit(true);
      for (UnitKernel k : {unit_mid, unit_last})
        if (bi_allow_smem((const void *)k, unit_smem) != cudaSuccess)
          return BI_ERR_CUDA;
    }
  }
  // every launch of the loop may be scheduled while its predecessor drains (see bi_grid_wait)
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  for (int k = 0; k < c.K; ++k) {
    const int cur = k & 1;
    A.cur = cur;
    A.final = (k == c.K - 1);
    A.first = (k == 0);
    cudaLaunchConfig_t cfg = {};
    cfg.stream = c.stream;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    // the slices on their unrolled form where they all have one, everything else on the any-shape form
    const int n_unrolled = any_shape ? 0 : ntask_slices;
    if (n_unrolled > 0) {
      cfg.gridDim = dim3((unsigned)n_unrolled);
      cfg.blockDim = dim3((unsigned)tu);
      cfg.dynamicSmemBytes = usmem;
      P.task_base = 0;
      if (cudaLaunchKernelEx(&cfg, unrolled, P, cur, (int)(k == 0)) != cudaSuccess) return BI_ERR_CUDA;
    }
    if (ntask > n_unrolled) {
      cfg.gridDim = dim3((unsigned)(ntask - n_unrolled));
      cfg.blockDim = dim3((unsigned)(tu * rs));
      cfg.dynamicSmemBytes = csmem;
      P.task_base = n_unrolled;
      if (cudaLaunchKernelEx(&cfg, rt, P, cur, (int)(k == 0)) != cudaSuccess) return BI_ERR_CUDA;
    }
    if (unit_mid) {
      cfg.gridDim = dim3((unsigned)((NU + 31) / 32));
      cfg.blockDim = dim3((unsigned)(32 * h.F));
      cfg.dynamicSmemBytes = unit_smem;
      if (cudaLaunchKernelEx(&cfg, A.final ? unit_last : unit_mid, (const BiDev *)md->d, P, A, UL) != cudaSuccess) return BI_ERR_CUDA;
      continue;
    }
    cfg.gridDim = dim3((unsigned)(fw ? NU : (NU + upb - 1) / upb));
    cfg.blockDim = dim3((unsigned)(fw ? 32 * h.F : 128));
    cfg.dynamicSmemBytes = (size_t)(fw ? 1 : upb) * 3 * h.Sp * sizeof(R);
    if (cudaLaunchKernelEx(&cfg, A.final ? update_last : update_mid, (const BiDev *)md->d, P, A) != cudaSuccess)
      return BI_ERR_CUDA;
  }
  if (cudaGetLastError() != cudaSuccess) return BI_ERR_CUDA;
  mut->launches += 1 + (cnt > 0) + c.K * (1 + (!any_shape && nslice > 0) + (any_shape ? cnt > 0 : edges));
  const bool f64 = sizeof(R) == 8;
  mut->last_kernel = c.algo == BI_ALGO_VMP ? (f64 ? "batch_vmp_f64" : "batch_vmp_f32")
                                           : (f64 ? "batch_mmp_f64" : "batch_mmp_f32");
  return BI_OK;
}

}  // namespace

int bi_batch_start_f64(const bi_model *md, const BatchParams &P, int max_m, const float *q_init, int32_t *perm, int4 *task,
                       cudaStream_t stream) {
  return batch_start<double>(md, P, max_m, q_init, perm, task, stream);
}

int bi_batch_shape(int rank, const int *dim) {
  BiGroup g;
  memset(&g, 0, sizeof(g));
  g.rank = rank;
  for (int k = 0; k < rank && k < BI_MAX_RANK; ++k) g.dim[k] = dim[k];
  return rank >= 2 && rank <= 4 ? shape_of(g) : -1;
}

// Applies to window calls with enough (agent, step) units to fill the machine.  Shared models
// bucket the units by observed outcome and share a staged slice, in float64 on the matrix instruction (batch_mma.cu);
// per-agent models run the any-shape contraction with every unit reading its own slice.
int bi_launch_batch(const BiCall &c, bi_model *mut) {
  const bi_model *md = c.model;
  if (c.algo == BI_ALGO_FILTER) return BI_ERR_UNSUPPORTED;
  if (md->h.has_bdep && (c.algo != BI_ALGO_VMP || md->h.G != 1 || !md->h.logBedge[0] || (md->arith == BI_ARITH_F32 && md->has_zeros)))
    return BI_ERR_UNSUPPORTED;   // (with zeros in A the order of float32 sums is kept, see bi_block_serves)
  if (md->h.G != 1) {
    // per-agent models: the slices are re-read every iteration, which pays only while they stay in L2
    // (measured on a three-factor model with per-step slices: faster than the warp-per-step kernels at
    // 112 MB of slices, slower at 224 MB)
    double bytes = 0;
    for (int gi = 0; gi < md->h.ngroups; ++gi)
      if (md->h.grp[gi].rank >= 2) bytes += (double)md->h.grp[gi].P_pad * (md->h.grp[gi].mem_end - md->h.grp[gi].mem_begin);
    bytes *= (double)c.N * c.T * (md->arith == BI_ARITH_F64 ? 8 : 4);
    if (bytes > 120e6) return BI_ERR_UNSUPPORTED;
  }
  if ((long long)c.N * c.T < 2048 || (long long)c.N * c.T > kMaxUnits) return BI_ERR_UNSUPPORTED;   // (too few to fill the machine this way)
  const int rc = bi_launch_batch_mma(c, mut);
  if (rc != BI_ERR_UNSUPPORTED) return rc;
  return md->arith == BI_ARITH_F64 ? launch_batch_t<double>(c, mut) : launch_batch_t<float>(c, mut);
}
