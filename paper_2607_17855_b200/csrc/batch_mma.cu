// Batched window kernels (VMP / MMP) on the float64 matrix instruction, for agents that share one model.
//
// As in batch.cu the (agent, step) units are bucketed by the observed outcome of every modality, and a task
// contracts one slice of ln A with the beliefs of the units of a bucket.  Seen as a matrix over (first axes) x (last
// axes), R x C, the slice takes part in two products per iteration, both with one column per unit:
//
//   V[r] = sum_c L[r][c] Y[c],   W[c] = sum_r L[r][c] X[r],
//
// X and Y the products of the first and of the last axes' beliefs.  V carries every message of the first axes (each a
// sum over V weighted by the other first axes' beliefs: 2R multiply-adds), W those of the last.  The two products are the 2P
// multiply-adds that all leave-one-out messages take (Section IV, marginalisation); they run as mma.sync.m8n8k4 on
// float64 operands, which has the vector pipe's peak at a sixteenth of its issue slots (measured: 16 cycles per
// instruction and scheduler).  tcgen05 has no float64 form.
//
// The transitions of a step's edge are the same shape -- a matrix per action, the child's state at the next step by
// the parents' at this one -- so they are members too, their units bucketed by the action: V is the message to
// the next step, W the message back.  (MMP: V takes B and W its column-normalised form, and both messages the logarithm.)
// A last kernel per iteration adds up a unit's messages and takes the softmax.
#include <algorithm>
#include <climits>
#include <cstring>

#include "batch.h"
#include "tile3.cuh"

namespace {

constexpr int kWarps = 4;          // warps of a CTA of the pair kernel: two (V and W) for each of two groups of units
constexpr int kPairTiles = 2;      // eights of units that one of its warps takes at a time
constexpr int kTiles = 8;          // most 8-wide tiles of results a warp accumulates at once
constexpr int kChunk = 8 * kTiles;
constexpr int kChunkStride = kChunk + 4;   // (4 modulo 16: a half warp's 4 units x 32 bytes fall on different banks)

struct MmaMember {
  const double *L0, *L1;     // the matrices of V and of W, [outcome][R][C] (the same for all but MMP's transitions)
  int64_t ostride;
  int32_t R, C;
  int32_t logs;              // both messages enter as 1/2 ln max(., eps)
  // up to two axes of each side, slow and fast: 0, 1 rows; 2, 3 columns.  A side of one axis has no slow one: sizes 1, lo -1.
  // (A slow axis that is there may have one state too, in a transition: its messages are summed and written like any other's.)
  int32_t n[4], np[4];       // states; length along its side (the last axis is padded)
  int32_t q[4];              // beliefs, from the unit's row
  int32_t lo[4];             // beliefs in the warp's copy, or -1
  int64_t out[4];            // messages, from the unit's row of the first plane
};

struct MmaParams {
  MmaMember mem[BI_MAX_M + BI_MAX_F];
  int32_t NU, Sp;
  int32_t task0;             // first task slot of this launch
  int32_t one;               // the warp's copy of a unit's beliefs: entry 1.0, then entry 0.0
  int32_t sq;                // its length (4 modulo 8)
  int32_t tabs, lsz;         // entries of the index tables; elements of the staged slice
  const int32_t *perm;
  const int4 *task;
  double *ell;               // planes of messages, [NU][Sp] each
  const double *q;           // [2][NU][Sp]
  uint32_t *status;
  int32_t drop_copy;
};

__device__ __forceinline__ void mma_f64(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1},{%2},{%3},{%0,%1};"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}
__device__ __forceinline__ double half_log(double x) { return 0.5 * bi_log_inline(bi_max(x, BI_EPS)); }

// Fragments of an instruction: lane = 4 g + l holds A[g][l] (unit g, summation index l), B[l][g] and C[g][2l], C[g][2l + 1].

// ---- members over two axes: slices of pairs, transitions with one parent ----
// A warp takes one side (V or W) of a task, 8 UT units at a time, and shares nothing: the matrix (32 x 32 at most) is loaded into
// fragments once, before the wait for the beliefs; those go from memory straight into fragments, and the next units
// are read ahead.  Tasks are as long as lets the launch be one wave.
// after: the launch just before this one is the other contraction kernel, which does not touch what this one reads or
// writes and has waited for the beliefs; so this one starts at once, and its first CTA waits for the other kernel before it
// ends (whoever waits for this kernel finds both complete).  Reads of beliefs and tasks go to L2.
template <int UT, int NK>
__global__ void __launch_bounds__(32 * kWarps) bi_mma_pair_kernel(const __grid_constant__ MmaParams P, int cur, int first, int after) {
  if (first || after) {
    if (!after) bi_grid_wait();
    bi_grid_launch_dependents();
  }
  constexpr int STEP = kWarps / 2 * 8 * UT;   // units of a CTA's trip
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, l = lane & 3;
  const int side = warp & 1;
  int u0 = (warp >> 1) * 8 * UT;
  const int4 tk = __ldcg(P.task + P.task0 + (int)blockIdx.x);   // (of no units: an unused slot)
  const bool some = u0 < tk.z;
  const MmaMember &mm = P.mem[some ? tk.w : 0];
  const int32_t *pm = P.perm + tk.y + g;
  int unit[UT];
#pragma unroll
  for (int i = 0; i < UT; ++i) unit[i] = u0 + 8 * i + g < tk.z ? __ldcg(pm + u0 + 8 * i) : -1;
  // results n (rows for V, columns for W), summed index k; beyond the last of either it is repeated: such results are not
  // used, and such beliefs are zero (rows of beliefs are padded to multiples of four)
  const int R = mm.R, C = mm.C, nn = side == 0 ? R : C, kk = side == 0 ? C : R;
  double x[NK / 2][NK];
  if (some) {
    const double *L = (side == 0 ? mm.L0 : mm.L1) + (size_t)tk.x * mm.ostride;
#pragma unroll
    for (int t = 0; t < NK / 2; ++t)
      if (8 * t < nn) {
        const int n = min(8 * t + g, nn - 1);
#pragma unroll
        for (int k = 0; k < NK; ++k) {
          const int j = min(4 * k + l, kk - 1);
          x[t][k] = 4 * k < kk ? __ldg(L + (side == 0 ? n * C + j : j * C + n)) : 0.0;
        }
      }
  }
  if (!(first || after)) {
    bi_grid_wait();
    bi_grid_launch_dependents();
  }
  const double *qc = P.q + (size_t)cur * P.NU * P.Sp + mm.q[side == 0 ? 3 : 1] + l;
  double *out = P.ell + mm.out[side == 0 ? 1 : 3] + 2 * l;
  const int np = (nn + 3) & ~3;
  const bool logs = mm.logs != 0;
#pragma unroll 1
  for (; u0 < tk.z; u0 += STEP) {
    double a[UT][NK];
#pragma unroll
    for (int i = 0; i < UT; ++i) {
      const double *qr = qc + (size_t)max(unit[i], 0) * P.Sp;
#pragma unroll
      for (int k = 0; k < NK; ++k) a[i][k] = unit[i] >= 0 && 4 * k < kk ? __ldcg(qr + 4 * k) : 0.0;
    }
    int after_unit[UT];
#pragma unroll
    for (int i = 0; i < UT; ++i) after_unit[i] = u0 + STEP + 8 * i + g < tk.z ? __ldcg(pm + u0 + STEP + 8 * i) : -1;
#pragma unroll
    for (int t = 0; t < NK / 2; ++t) {
      if (8 * t < nn) {
        double c[UT][2], d[UT][2];
#pragma unroll
        for (int i = 0; i < UT; ++i) c[i][0] = c[i][1] = d[i][0] = d[i][1] = 0.0;
#pragma unroll
        for (int k = 0; k < NK; k += 2) {
          if (4 * k < kk) {
#pragma unroll
            for (int i = 0; i < UT; ++i) {
              mma_f64(c[i], a[i][k], x[t][k]);
              mma_f64(d[i], a[i][k + 1], x[t][k + 1]);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < UT; ++i) {
          double v0 = c[i][0] + d[i][0], v1 = c[i][1] + d[i][1];
          if (logs) { v0 = half_log(v0); v1 = half_log(v1); }
          if (unit[i] >= 0 && 8 * t + 2 * l < np)
            *reinterpret_cast<double2 *>(out + (size_t)unit[i] * P.Sp + 8 * t) = make_double2(v0, v1);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < UT; ++i) unit[i] = after_unit[i];
  }
  if (after && blockIdx.x == 0) bi_grid_wait();
}

// ---- members over three or four axes ----

// T tiles of eight results for eight units: c[t] += A B.  A: the units' products of beliefs (tab: byte offsets of two
// entries of a unit's beliefs per summation index; q: the lane's unit).  B: tile t's fragment of summation step k is 8 t S + 4 k
// (V) or 8 t + 4 k S (W) from b on; GLOBAL: off[t] + 4 k, or for W the row clamped to the last.
template <int T, bool GLOBAL, int SIDE>
__device__ __forceinline__ void mma_tiles(double (&c)[kTiles][2], const double *__restrict__ b, int S, int R, const int (&off)[kTiles],
                                          const uint32_t *tab, const double *q, int nk, int l) {
#pragma unroll
  for (int t = 0; t < T; ++t) c[t][0] = c[t][1] = 0.0;
  const char *qb = reinterpret_cast<const char *>(q);
  const int kst = SIDE == 0 ? 4 : 4 * S;
#pragma unroll 4
  for (int k = 0; k < nk; ++k) {
    const uint32_t e = tab[4 * k];
    const double a = *reinterpret_cast<const double *>(qb + (e & 0xffff)) * *reinterpret_cast<const double *>(qb + (e >> 16));
    if (GLOBAL && SIDE == 1) b += (min(4 * k + l, R - 1) - (k ? min(4 * k - 4 + l, R - 1) : 0)) * S;
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const double x = GLOBAL ? __ldg(b + off[t] + (SIDE == 0 ? k * kst : 0)) : b[SIDE == 0 ? t * 8 * S + k * kst : t * 8 + k * kst];
      mma_f64(c[t], a, x);
    }
  }
}

// sum_i v[i st] q[i], n terms
__device__ __forceinline__ double dot_strided(const double *v, int st, const double *q, int n) {
  double m0 = 0.0, m1 = 0.0, m2 = 0.0, m3 = 0.0;
  int i = 0;
#pragma unroll 1
  for (; i + 3 < n; i += 4, v += 4 * st) {
    m0 = fma(v[0], q[i], m0);
    m1 = fma(v[st], q[i + 1], m1);
    m2 = fma(v[2 * st], q[i + 2], m2);
    m3 = fma(v[3 * st], q[i + 3], m3);
  }
  if (i < n) m0 = fma(v[0], q[i], m0);
  if (i + 1 < n) m1 = fma(v[st], q[i + 1], m1);
  if (i + 2 < n) m2 = fma(v[2 * st], q[i + 2], m2);
  return (m0 + m1) + (m2 + m3);
}

// One side's messages to eight units: SIDE 0 the rows' (V), 1 the columns' (W).  The results go to the warp's scratch, a row per
// unit, and four lanes per unit sum them along either axis.
template <bool GLOBAL, int SIDE>
__device__ __forceinline__ void mma_side(const MmaParams &P, const MmaMember &mm, const double *L, int S, const uint32_t *tab,
                                         const double *q, double *scr, int unit, int g, int l) {
  const int nx = mm.n[2 * SIDE], ny = mm.n[2 * SIDE + 1], nyp = mm.np[2 * SIDE + 1];
  const int xs = max(1, kChunk / nyp);                 // slow indices of a chunk
  const int len = SIDE == 0 ? mm.R : mm.C;             // results of this side
  const int nk = ((SIDE == 0 ? mm.C : mm.R) + 3) >> 2; // summation steps
  double *ox = P.ell + (int64_t)unit * P.Sp + mm.out[2 * SIDE], *oy = P.ell + (int64_t)unit * P.Sp + mm.out[2 * SIDE + 1];
  const bool live = unit >= 0;
  double *row = scr + g * kChunkStride;
  for (int x0 = 0; x0 < nx; x0 += xs) {
    const int nxc = min(nx - x0, xs), n0 = x0 * nyp, cnt = nxc * nyp, T = (cnt + 7) >> 3;
    int off[kTiles];
#pragma unroll
    for (int t = 0; t < kTiles; ++t) off[t] = GLOBAL ? min(n0 + 8 * t + g, len - 1) * (SIDE == 0 ? S : 1) : 0;
    // (in shared memory rows beyond the last are there to be read, see staged_elements: what comes of them is not used)
    const double *b = GLOBAL ? L + (SIDE == 0 ? l : 0) : L + (SIDE == 0 ? (n0 + g) * S + l : l * S + n0 + g);
    double c[kTiles][2];
    switch (T) {
#define X(TT) case TT: mma_tiles<TT, GLOBAL, SIDE>(c, b, S, mm.R, off, tab + l, q, nk, l); break;
      X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8)
#undef X
      default: break;
    }
    if (mm.lo[2 * SIDE] < 0) {   // one axis: the results are its messages
#pragma unroll
      for (int t = 0; t < kTiles; ++t)
        if (live && 8 * t + 2 * l < ((cnt + 3) & ~3)) *reinterpret_cast<double2 *>(oy + 8 * t + 2 * l) = make_double2(c[t][0], c[t][1]);
      continue;
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kTiles; ++t)
      if (t < T) *reinterpret_cast<double2 *>(row + 8 * t + 2 * l) = make_double2(c[t][0], c[t][1]);
    __syncwarp();
    const double *qx = q + mm.lo[2 * SIDE] + x0, *qy = q + mm.lo[2 * SIDE + 1];
    if (live) {
      if ((nyp & 1) == 0) {   // pairs of neighbours in one 16-byte load (beliefs beyond the last are zero)
        for (int x = l; x < nxc; x += 4) {
          const double2 *v = reinterpret_cast<const double2 *>(row + x * nyp), *w = reinterpret_cast<const double2 *>(qy);
          double m0 = 0.0, m1 = 0.0;
#pragma unroll 2
          for (int j = 0; j < nyp >> 1; ++j) {
            const double2 p = v[j], r = w[j];
            m0 = fma(p.x, r.x, m0);
            m1 = fma(p.y, r.y, m1);
          }
          ox[x0 + x] = m0 + m1;
        }
        for (int y = 2 * l; y < nyp; y += 8) {
          const double *v = row + y;
          double2 m = x0 ? *reinterpret_cast<const double2 *>(oy + y) : make_double2(0.0, 0.0), o = make_double2(0.0, 0.0);   // (this thread's own sums so far)
          int x = 0;
#pragma unroll 2
          for (; x + 1 < nxc; x += 2, v += 2 * nyp) {
            const double2 p = *reinterpret_cast<const double2 *>(v), r = *reinterpret_cast<const double2 *>(v + nyp);
            const double q0 = qx[x], q1 = qx[x + 1];
            m.x = fma(p.x, q0, m.x); m.y = fma(p.y, q0, m.y);
            o.x = fma(r.x, q1, o.x); o.y = fma(r.y, q1, o.y);
          }
          if (x < nxc) {
            const double2 p = *reinterpret_cast<const double2 *>(v);
            m.x = fma(p.x, qx[x], m.x); m.y = fma(p.y, qx[x], m.y);
          }
          *reinterpret_cast<double2 *>(oy + y) = make_double2(m.x + o.x, m.y + o.y);
        }
      } else {
        for (int x = l; x < nxc; x += 4) ox[x0 + x] = dot_strided(row + x * nyp, 1, qy, ny);
        for (int y = l; y < ny; y += 4) {
          const double before = x0 ? oy[y] : 0.0;
          oy[y] = before + dot_strided(row + y, nyp, qx, nxc);
        }
      }
    }
    __syncwarp();
  }
}

// A CTA per task.  The slice is staged in shared memory (GLOBAL: slices that do not fit are read through L1) and its index
// tables made before the wait for the beliefs, and a task is as many units as lets the launch be one wave, so that all of
// that overlaps the kernel before (tasks of 32 units, three waves: 15 of 35 us went into starting them).  The
// warps take eight units at a time, their beliefs gathered by asynchronous copies.  SPLIT: half
// of the warps does V, half W, for batches with fewer units than that fills the machine with.
template <bool GLOBAL, bool SPLIT, int NW>
__global__ void __launch_bounds__(32 * NW, 16 / NW) bi_mma_slice_kernel(const __grid_constant__ MmaParams P, int cur, int first) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bar;
  double *Ls = reinterpret_cast<double *>(smem_raw);
  uint32_t *tab = reinterpret_cast<uint32_t *>(Ls + P.lsz);
  if (first) {   // the tasks were written by the kernel just before this one
    bi_grid_wait();
    bi_grid_launch_dependents();
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, l = lane & 3;
  const int4 tk = __ldcg(P.task + P.task0 + (int)blockIdx.x);
  if (tk.z == 0) return;   // an unused task slot
  const MmaMember &mm = P.mem[tk.w];
  const int R = mm.R, C = mm.C, S = GLOBAL ? C : (C & 4) ? C : C + 4;
  const double *slice = mm.L0 + (size_t)tk.x * mm.ostride;
  if (!GLOBAL) {
    if (tid == 0) {
      bi_mbar_init(&bar, 1);
      bi_mbar_expect(&bar, (uint32_t)(R * C * sizeof(double)));
    }
    __syncthreads();
    if (warp == 0 && !P.drop_copy)
      for (int r = lane; r < (S == C ? 1 : R); r += 32)
        bi_bulk_copy(Ls + (size_t)r * S, slice + (size_t)r * C, (uint32_t)((S == C ? R * C : C) * sizeof(double)), &bar);
    if (warp > 0 && warp <= ((-R) & 3))   // (the last summation step's rows beyond the last: their beliefs are zero, and these must be finite)
      for (int c = lane; c < C; c += 32) Ls[(R + warp - 1) * S + c] = 0.0;
  }
  // index tables: summation index -> two entries of a unit's beliefs
  uint32_t *ctab = tab, *rtab = tab + C;
  for (int c = tid; c < C; c += 32 * NW) {
    const int x = c / mm.np[3], y = c - x * mm.np[3];
    ctab[c] = (uint32_t)((mm.lo[2] >= 0 ? mm.lo[2] + x : P.one) | ((mm.lo[3] + y) << 16)) * 8u;
  }
  for (int r = tid; r < ((R + 3) & ~3); r += 32 * NW) {
    const int x = r / mm.np[1], y = r - x * mm.np[1];
    rtab[r] = (r < R ? (uint32_t)((mm.lo[0] >= 0 ? mm.lo[0] + x : P.one) | ((mm.lo[1] + y) << 16)) : (uint32_t)((P.one + 1) | ((P.one + 1) << 16))) * 8u;
  }
  constexpr int GRP = SPLIT ? NW / 2 : NW;   // groups of units at a time
  const int side = SPLIT ? warp & 1 : 0;
  int u0 = 8 * (SPLIT ? warp >> 1 : warp);
  double *own = reinterpret_cast<double *>(tab + P.tabs) + (size_t)warp * 8 * (P.sq + kChunkStride);
  double *scr = own + 8 * P.sq, *q = own + g * P.sq;
  if (l < 2) q[P.one + l] = l == 0 ? 1.0 : 0.0;
  const int32_t *pm = P.perm + tk.y + g;
  int unit = u0 + g < tk.z ? __ldcg(pm + u0) : -1;
  __syncthreads();
  if (!first) {   // beliefs of the previous update, and the right to overwrite the messages it read
    bi_grid_wait();
    bi_grid_launch_dependents();
  }
  const double *qc = P.q + (size_t)cur * P.NU * P.Sp;
  const double *L = GLOBAL ? slice : Ls;
  bool staged = GLOBAL;
#pragma unroll 1
  for (; u0 < tk.z; u0 += 8 * GRP) {
    const double *qr = qc + (size_t)max(unit, 0) * P.Sp;
    const int size = unit >= 0 ? 16 : 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)   // 16 bytes a copy (rows and offsets are multiples of four entries; zeros where there is no unit)
      if ((j & 1) != 0 || mm.lo[j] >= 0)
        for (int s = 2 * l; s < ((mm.n[j] + 3) & ~3); s += 8)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(bi_smem_addr(q + mm.lo[j] + s)), "l"(qr + mm.q[j] + s), "r"(size) : "memory");
    const int unit2 = u0 + 8 * GRP + g < tk.z ? __ldcg(pm + u0 + 8 * GRP) : -1;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (!staged) {   // a copy that does not arrive within the probe limit: the warp reports it and leaves
      if (!bi_mbar_wait(&bar, 0, P.drop_copy ? 256 : 1 << 18)) {
        if (lane == 0) atomicOr(P.status, BI_FLAG_COPY_TIMEOUT);
        return;
      }
      staged = true;
    }
    if (!SPLIT || side == 0) mma_side<GLOBAL, 0>(P, mm, L, S, ctab, q, scr, unit, g, l);
    if (!SPLIT || side == 1) mma_side<GLOBAL, 1>(P, mm, L, S, rtab, q, scr, unit, g, l);
    __syncwarp();
    unit = unit2;
  }
}

// ---- per unit: add up the messages, softmax ----
struct MmaUpdate {
  const int32_t *obs;
  float *q_out, *logq_out;
  int32_t *argmax_out;
  int32_t T, cur, first;
  const void *lnprior;        // [N][S] log-priors used in the place of ln D at a window's first step, or NULL
  double lambda;              // damping step; 1 = plain update
  double *xprev;              // [NU][Sp] previous iterate's logits (damped calls only)
  const float *q_init;        // warm start (for the first damped step's ln q), or NULL
  // The exponentials need no shift where none of a logit's terms -- one per modality, the prior or past message, the future
  // messages -- is below ln 1e-16 (53.2 binary orders) and there are at most seventeen of them; a model with
  // entries above 1 is marked in the status words.
  int32_t common;
  uint32_t child;             // the plane of the messages over the edge into the step (as a mask)
  uint32_t fmask[BI_MAX_F];   // planes with messages to factor f: from its groups,
  uint32_t emask[BI_MAX_F];   // ... and over the edge out of the step
  uint32_t r1mask[BI_MAX_F];  // modalities (descriptor members) that depend on factor f alone
};

// A thread per two consecutive states (16 bytes) of a unit's padded state vector, all factors side by side: every lane
// has work whatever the factors' sizes, rows of messages and beliefs are read and written as they lie in memory, and a
// factor's normaliser goes through a few words of shared memory.  The kernel is loads from L2: those of four planes
// go out together, and what does not change between the iterations (the slices of single-factor modalities, the prior) is
// added up before the wait for the messages.
constexpr int kUpdThreads = 128;
// PER_SM: CTAs resident on an SM.  Twelve cost some spilled registers and hide more of the loads, which pays where the units are
// more than one wave of nine (20 480 units of 34 states: 751 -> 738 us a call; with fewer it costs up to 6 %).
template <int PER_SM, bool FINAL, bool DAMPED>
__global__ void __launch_bounds__(kUpdThreads, PER_SM) bi_mma_update_kernel(const BiDev *__restrict__ mdp, const __grid_constant__ MmaUpdate A,
                                                                    const double *__restrict__ ell, double *__restrict__ qbuf, int NU, int upb) {
  __shared__ double part[2][kUpdThreads];
  __shared__ double2 logit[FINAL ? kUpdThreads : 1];
  const BiDev &md = *mdp;
  const int F = md.F, Sp = md.Sp, S = md.S, M = md.M, T = A.T, nv = Sp >> 1, tid = threadIdx.x;
  const int ul = tid / nv, v = tid - ul * nv;
  int f = 0;
  while (f + 1 < F && 2 * v >= md.offp[f + 1]) ++f;
  const int n = md.n[f], op = md.offp[f], off = md.off[f], s = 2 * v - op;   // this thread's states: s and s + 1
  const int p0 = (ul < upb ? ul * nv : 0) + (op >> 1), np2 = md.npad[f] >> 1;   // the factor's vectors
  const bool common = A.common && __ldg(md.status + 1) == 0;
  const size_t plane = (size_t)NU * Sp;
  const uint32_t fmask = A.fmask[f], emask = A.emask[f], r1mask = A.r1mask[f];
  bool waited = false;
  for (int u0 = (int)blockIdx.x * upb; u0 < NU; u0 += (int)gridDim.x * upb) {
    const bool live = ul < upb && u0 + ul < NU;
    const int unit = live ? u0 + ul : 0;
    const int a = unit / T, t = unit - a * T;
    const size_t base = (size_t)unit * Sp + 2 * v;
    double2 x = make_double2(0.0, 0.0);
    auto add = [&](const double *p) {
      const double2 w = *reinterpret_cast<const double2 *>(p);
      x.x += w.x; x.y += w.y;
    };
    for (uint32_t mk = r1mask; mk; mk &= mk - 1) {   // single-factor modalities: the slice is the message
      const BiMember &mm = md.mem[__ffs(mk) - 1];
      const int o = clamp_flag(__ldg(A.obs + (size_t)unit * M + mm.modality), mm.m, md.status, BI_FLAG_OBS_RANGE);
      add((const double *)mm.logA + (size_t)o * mm.P_pad + s);
    }
    if (t == 0) {
      if (A.lnprior) {
        const double *p = (const double *)A.lnprior + (size_t)a * S + off;
        if (s < n) x.x += p[s];
        if (s + 1 < n) x.y += p[s + 1];
      } else {
        add((const double *)md.logD[f] + s);
      }
    }
    uint32_t mk = fmask | (t > 0 ? A.child : 0u) | (t + 1 < T ? emask : 0u);
    if (!waited) {
      bi_grid_wait();
      bi_grid_launch_dependents();
      waited = true;
    }
    const double *row = ell + base;
    while (mk) {
      double2 w[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        w[b] = mk ? __ldcg(reinterpret_cast<const double2 *>(row + (size_t)(__ffs(mk) - 1) * plane)) : make_double2(0.0, 0.0);
        mk &= mk - 1;
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) { x.x += w[b].x; x.y += w[b].y; }
    }
    if (DAMPED) {   // a step on the logits; the first one starts from ln q of the starting belief (uniform: a constant, taken as 0)
      double2 prev = make_double2(0.0, 0.0);
      double2 *xp = reinterpret_cast<double2 *>(A.xprev + base);
      if (!A.first) {
        prev = *xp;
      } else if (A.q_init) {
        const float *qi = A.q_init + (size_t)unit * S + md.off[f] + s;
        if (s < n) prev.x = bi_log(bi_max((double)qi[0], BI_EPS));
        if (s + 1 < n) prev.y = bi_log(bi_max((double)qi[1], BI_EPS));
      }
      x.x = fma(A.lambda, x.x, (1.0 - A.lambda) * prev.x);
      x.y = fma(A.lambda, x.y, (1.0 - A.lambda) * prev.y);
      if (live) *xp = x;
    }
    double mx = 0.0;
    if (FINAL || !common) {   // (see MmaUpdate::common; the last iterate takes the exact maximum)
      part[0][tid] = s < n ? (s + 1 < n ? bi_max(x.x, x.y) : x.x) : -bi_inf<double>();
      if (FINAL) logit[tid] = x;
      __syncthreads();
      mx = part[0][p0];
      for (int j = 1; j < np2; ++j) mx = bi_max(mx, part[0][p0 + j]);
    }
    double2 e;
    e.x = s < n ? bi_exp_inline(x.x - mx) : 0.0;
    e.y = s + 1 < n ? bi_exp_inline(x.y - mx) : 0.0;
    part[1][tid] = e.x + e.y;
    __syncthreads();
    double z0 = 0.0, z1 = 0.0;   // (a factor has an even number of vectors)
    for (int j = 0; j < np2; j += 2) { z0 += part[1][p0 + j]; z1 += part[1][p0 + j + 1]; }
    const double z = z0 + z1, rz = bi_rcp(z);
    if (!FINAL) {
      if (live) *reinterpret_cast<double2 *>(qbuf + (size_t)(A.cur ^ 1) * plane + base) = make_double2(e.x * rz, e.y * rz);
    } else if (live) {
      const double lz = A.logq_out ? bi_log(z) : 0.0;
      const size_t o = (size_t)unit * S + off + s;
      if (s < n) {
        A.q_out[o] = (float)(e.x * rz);
        if (A.logq_out) A.logq_out[o] = (float)(x.x - mx - lz);
      }
      if (s + 1 < n) {
        A.q_out[o + 1] = (float)(e.y * rz);
        if (A.logq_out) A.logq_out[o + 1] = (float)(x.y - mx - lz);
      }
      if (A.argmax_out && s == 0) {   // the lowest state that has the maximum
        int am = 0;
        for (int k = n - 1; k >= 0; --k) {
          const double2 y = logit[p0 + (k >> 1)];
          if (((k & 1) ? y.y : y.x) == mx) am = k;
        }
        A.argmax_out[(size_t)unit * F + f] = am;
      }
    }
    __syncthreads();   // (the exchange area is free again)
  }
}

int ceil_div(int a, int b) { return (a + b - 1) / b; }
size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// matrix instructions per eight units of a cut of n axes into the first `rows` and the rest, the last one padded
long long cut_cost(const int *dim, int rank, int rows) {
  int n[4] = {1, 1, 1, 1};
  for (int j = 0; j < rows; ++j) n[2 - rows + j] = dim[j];
  for (int j = rows; j < rank; ++j) n[4 - rank + j] = j == rank - 1 ? bi_pad4(dim[j]) : dim[j];
  long long cost = 0;
  for (int side = 0; side < 2; ++side) {
    const int nx = n[2 * side], ny = n[2 * side + 1], xs = std::max(1, kChunk / ny), other = n[2 - 2 * side] * n[3 - 2 * side];
    for (int x0 = 0; x0 < nx; x0 += xs) cost += (long long)ceil_div(std::min(xs, nx - x0) * ny, 8) * ceil_div(other, 4);
    if (nx > 1) cost += nx * ny / 8;
  }
  return cost;
}

// Elements of a staged slice's buffer: up to the last that either side's tiles read.  A chunk takes whole tiles of eight results
// from its first one on, which need not be a multiple of eight: rows of 8 x 9 states are read as 0 to 63 and 63 to 78.
size_t staged_elements(const MmaMember &mm) {
  const int S = (mm.C & 4) ? mm.C : mm.C + 4, rows = bi_pad4(mm.R);   // (row stride, rows summed over: see the kernel)
  int end[2] = {0, 0};
  for (int side = 0; side < 2; ++side) {
    const int nx = mm.n[2 * side], ny = mm.np[2 * side + 1], xs = std::max(1, kChunk / ny);
    for (int x0 = 0; x0 < nx; x0 += xs) end[side] = std::max(end[side], x0 * ny + 8 * ceil_div(std::min(xs, nx - x0) * ny, 8));
  }
  return std::max((size_t)std::max(rows, end[0]) * S, (size_t)(rows - 1) * S + end[1]);
}

// matrix instructions per eight units of one member
double member_instructions(int R, int C) {
  return (double)ceil_div(R, 8) * ceil_div(C, 4) + (double)ceil_div(C, 8) * ceil_div(R, 4);
}
double axes_instructions(const int *dim, int rank) {
  const int rows = rank == 4 ? 2 : rank == 3 && cut_cost(dim, 3, 2) < cut_cost(dim, 3, 1) ? 2 : 1;
  int R = 1, C = 1;
  for (int j = 0; j < rank; ++j) (j < rows ? R : C) *= j == rank - 1 ? bi_pad4(dim[j]) : dim[j];
  return member_instructions(R, C);
}

}  // namespace

// Microseconds of a call on these kernels, or a negative number where they do not take it.  Linear in the launches, the longest
// task, the instructions, gathers and rows of messages of the units that share an SM; fitted to 139 calls on
// structures of one to five factors, 2 048 to 62 000 units, 6 and 16 iterations (11 % rms error).
double bi_batch_mma_cost(const BiCall &c) {
  const BiDev &h = c.model->h;
  if (c.model->arith != BI_ARITH_F64 || h.G != 1 || (long long)c.N * c.T < 2048 || (long long)c.N * c.T > kMaxUnits) return -1.0;
  double deep = 0, longest = 0, pairs = 0, states = 0;
  int ndeep = 0, npair = 0;
  auto add = [&](const int *dim, int rank) {
    const double n = axes_instructions(dim, rank);
    if (rank > 2) { deep += n; longest = std::max(longest, n); ++ndeep; }
    else { pairs += n; ++npair; }
  };
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank > 4) return -1.0;
    for (int mi = g.mem_begin; mi < g.mem_end && g.rank > 1; ++mi) add(g.dim, g.rank);
  }
  for (int f = 0; f < h.F; ++f) {
    states += h.npad[f];
    if (c.T == 1) continue;
    int dim[4] = {h.n[f], h.n[f], 1, 1};
    const int k = h.has_bdep ? h.bdep_len[f] : 1;
    if (k > 3) return -1.0;
    for (int j = 0; j < k && h.has_bdep; ++j) dim[1 + j] = h.n[h.bdep[f][j]];
    add(dim, 1 + k);
  }
  const double per_sm = (double)c.N * c.T / c.model->sm_count * 1e-3;   // thousands of units
  return 14.5 + c.K * (4.7 + 0.34 * ndeep + (ndeep ? 1.5 : 0.0) + 0.0127 * longest) +
         c.K * per_sm * (0.905 * deep + 12.6 * ndeep + 0.924 * pairs + 4.8 * npair + (0.93 + 0.68 * (c.algo == BI_ALGO_MMP)) * states);
}

int bi_launch_batch_mma(const BiCall &c, bi_model *mut) {
  const bi_model *md = c.model;
  const BiDev &h = md->h;
  if (md->arith != BI_ARITH_F64 || h.G != 1) return BI_ERR_UNSUPPORTED;
  const int NU = c.N * c.T;
  BatchParams B;   // for the bucketing
  MmaParams P;
  MmaUpdate A;
  memset(&B, 0, sizeof(B));
  memset(&P, 0, sizeof(P));
  memset(&A, 0, sizeof(A));
  struct Axes { int rank, fac[4], next; };   // next: the first axis is the step after
  Axes ax[BI_MAX_M + BI_MAX_F];
  int cnt = 0, max_m = 1;
  auto add_member = [&](const double *L0, const double *L1, int m, int modality, int edge, const Axes &x) {
    BatchMember &b = B.mem[cnt];
    b.m = m; b.modality = modality; b.edge = edge; b.split = 1;
    P.mem[cnt].L0 = L0; P.mem[cnt].L1 = L1;
    ax[cnt++] = x;
    max_m = std::max(max_m, m);
  };
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank > 4) return BI_ERR_UNSUPPORTED;
    for (int mi = g.mem_begin; mi < g.mem_end; ++mi) {
      if (g.rank == 1) A.r1mask[g.axis[0]] |= 1u << mi;
      if (g.rank < 2) continue;
      Axes x = {g.rank, {0, 0, 0, 0}, 0};
      for (int j = 0; j < g.rank; ++j) x.fac[j] = g.axis[j];
      add_member((const double *)h.mem[mi].logA, (const double *)h.mem[mi].logA, h.mem[mi].m, h.mem[mi].modality, 0, x);
    }
  }
  const int nslice = cnt;
  if (c.T > 1)
    for (int f = 0; f < h.F; ++f) {
      Axes x = {2, {f, f, 0, 0}, 1};
      if (h.has_bdep) {
        if (h.bdep_len[f] > 3) return BI_ERR_UNSUPPORTED;
        x.rank = 1 + h.bdep_len[f];
        for (int j = 0; j < h.bdep_len[f]; ++j) x.fac[1 + j] = h.bdep[f][j];
        add_member((const double *)h.logBedge[f], (const double *)h.logBedge[f], h.U[f], 0, 1 + f, x);
      } else if (c.algo == BI_ALGO_VMP) {
        add_member((const double *)h.logB[f], (const double *)h.logB[f], h.U[f], 0, 1 + f, x);
      } else {
        add_member((const double *)h.Bf[f], (const double *)h.BdagT[f], h.U[f], 0, 1 + f, x);
      }
    }
  if (max_m > 4096) return BI_ERR_UNSUPPORTED;
  // planes of messages: one per slice member, one for the messages to the children, and for those to the parents
  // one (a factor has one child, itself) or one per child
  const int nplanes = nslice + (cnt > nslice ? (h.has_bdep ? 1 + h.F : 2) : 0);
  A.child = 1u << nslice;
  // ---- cut every member into rows and columns
  bool heavy[BI_MAX_M + BI_MAX_F];
  int nmax = 1;
  size_t tabs = 0, lsz = 0;
  int own = 0;
  for (int j = 0; j < cnt; ++j) {
    const Axes &x = ax[j];
    MmaMember &mm = P.mem[j];
    int dim[4];
    for (int k = 0; k < x.rank; ++k) dim[k] = h.n[x.fac[k]];
    int rows = x.rank == 4 ? 2 : 1;
    if (x.rank == 3 && cut_cost(dim, 3, 2) < cut_cost(dim, 3, 1)) rows = 2;
    for (int k = 0; k < 4; ++k) {
      mm.n[k] = mm.np[k] = 1;
      mm.lo[k] = -1;
    }
    int lo = 0;
    for (int k = 0; k < x.rank; ++k) {
      const int side = k < rows ? 0 : 1, slot = side == 0 ? 2 - rows + k : 4 - x.rank + k, f = x.fac[k];
      mm.n[slot] = dim[k];
      mm.np[slot] = k == x.rank - 1 ? bi_pad4(dim[k]) : dim[k];
      mm.q[slot] = h.offp[f] + (x.next && k == 0 ? h.Sp : 0);
      mm.lo[slot] = lo;
      lo += bi_pad4(dim[k]);
      int64_t plane = j;
      if (x.next) plane = k == 0 ? nslice : h.has_bdep ? nslice + 1 + (B.mem[j].edge - 1) : nslice + 1;
      mm.out[slot] = plane * NU * h.Sp + h.offp[f] + (x.next && k == 0 ? h.Sp : 0);
      if (!x.next) A.fmask[f] |= 1u << plane;
      else if (k > 0) A.emask[f] |= 1u << plane;
    }
    mm.R = mm.np[0] * mm.np[1];
    mm.C = mm.np[2] * mm.np[3];
    mm.ostride = (int64_t)mm.R * mm.C;
    mm.logs = x.next && c.algo == BI_ALGO_MMP;
    heavy[j] = x.rank > 2;
    if (heavy[j]) {
      tabs = std::max(tabs, (size_t)(mm.C + bi_pad4(mm.R)));
      lsz = std::max(lsz, staged_elements(mm));
      own = std::max(own, lo);
    } else {
      for (int k = 0; k < 2; ++k) nmax = std::max(nmax, dim[k]);
    }
  }
  // ---- order: the deep members first, largest first, then the pairs
  int order[BI_MAX_M + BI_MAX_F], nheavy = 0;
  for (int j = 0; j < cnt; ++j) {
    order[j] = j;
    nheavy += heavy[j];
  }
  std::stable_sort(order, order + cnt, [&](int a, int b) { return heavy[a] != heavy[b] ? heavy[a] : P.mem[a].ostride > P.mem[b].ostride; });
  {
    const MmaParams P0 = P;
    const BatchParams B0 = B;
    for (int j = 0; j < cnt; ++j) {
      P.mem[j] = P0.mem[order[j]];
      B.mem[j] = B0.mem[order[j]];
    }
  }
  P.one = own;
  P.sq = (own + 2 + 3) & ~3;
  if (P.sq % 8 == 0) P.sq += 4;
  P.tabs = (int)((tabs + 3) & ~(size_t)3);
  auto slice_smem = [&](int nw, size_t slice) { return (size_t)P.tabs * sizeof(uint32_t) + ((size_t)nw * 8 * (P.sq + kChunkStride) + slice) * sizeof(double); };
  auto fit = [&](int nw, size_t bytes) { return std::max(1, std::min(16 / nw, (int)(((size_t)md->max_smem_optin + 1024) / (bytes + 1024 + 64)))); };
  const bool global = slice_smem(4, lsz) > (size_t)md->max_smem_optin - 1024;
  P.lsz = global ? 0 : (int)((lsz + 1) & ~(size_t)1);
  // Warps of a CTA of the slice kernel, eight units at a time each: four, or eight around one staged slice where that leaves
  // more warps on an SM and the units are enough for them (a slice of 5236 entries, 12 222 units: 713 -> 557 us a call; of 3528,
  // 10 674 units: 750 -> 678; with 2 478 to 7 218 units up to 5 % slower)
  const int nw = !global && NU >= 8192 && slice_smem(8, P.lsz) <= (size_t)md->max_smem_optin - 1024 &&
                         8 * fit(8, slice_smem(8, P.lsz)) > 4 * fit(4, slice_smem(4, P.lsz)) ? 8 : 4;
  const size_t smem = slice_smem(nw, P.lsz);
  if (nheavy && smem > (size_t)md->max_smem_optin - 1024) return BI_ERR_UNSUPPORTED;
  // Units per task: a wave of CTAs is shared out between the members by the cost of a unit, a matrix instruction taking
  // sixteen cycles and the rest of eight units' work about 1500; every outcome may leave one partial task.
  const int per_sm = fit(nw, smem);
  double cost[BI_MAX_M + BI_MAX_F], heavy_cost = 0;
  for (int j = 0; j < cnt; ++j) {
    const MmaMember &mm = P.mem[j];
    cost[j] = 1500.0 + 16.0 * member_instructions(mm.R, mm.C);
    if (j < nheavy) heavy_cost += cost[j];
  }
  // V and W by different warps where the units do not fill a wave with eight to a warp, and the slices are large enough to be worth
  // the second set of beliefs (a slice of 5742 entries, 2560 units: 18.5 against 21.8 us an iteration; of 648, 7500
  // units: 18.5 against 15.6)
  const bool split = NU <= 4 * nw * per_sm * md->sm_count && nheavy && P.mem[0].ostride >= 2048;
  int ntask = 0, ntask_heavy = 0;
  long long nperm = 0;
  for (int j = 0; j < cnt; ++j) {
    const double wave = j < nheavy ? per_sm * md->sm_count * cost[j] / heavy_cost : (nmax <= 16 ? 8.0 : 4.0) * md->sm_count / (cnt - nheavy);
    const int trip = j < nheavy ? 8 * (split ? nw / 2 : nw) : 8 * kPairTiles * kWarps / 2;
    const double tasks = std::max(wave - B.mem[j].m, 0.5 * wave);
    const int unit_step = j < nheavy ? 8 : trip;
    const int tu = std::max(trip, ceil_div((int)std::ceil(NU / std::max(tasks, 1.0)), unit_step) * unit_step);
    B.mem[j].tu = tu;
    B.mem[j].task0 = ntask;
    B.mem[j].perm0 = (int)nperm;
    const int slots = ceil_div(NU, tu) + B.mem[j].m;
    ntask += slots;
    nperm += (long long)slots * tu;
    if (j < nheavy) ntask_heavy = ntask;
  }
  if (nperm > INT_MAX) return BI_ERR_UNSUPPORTED;

  // ---- workspace (stream-ordered; kept in the handle and grown on demand)
  const size_t b_perm = up256((size_t)nperm * sizeof(int32_t));
  const size_t b_task = up256((size_t)ntask * sizeof(int4));
  const size_t b_ell = up256((size_t)nplanes * NU * h.Sp * sizeof(double));
  const size_t b_q = up256(2 * (size_t)NU * h.Sp * sizeof(double));
  const size_t b_x = c.lambda != 1.0 ? up256((size_t)NU * h.Sp * sizeof(double)) : 0;
  const size_t need = b_perm + b_task + b_ell + b_q + b_x;
  int rc = bi_workspace(mut, need, c.stream);
  if (rc != BI_OK) return rc;
  if (mut->test_workspace == BI_WORKSPACE_NAN && cudaMemsetAsync(mut->ws, 0xff, need, c.stream) != cudaSuccess) return BI_ERR_CUDA;
  unsigned char *w = static_cast<unsigned char *>(mut->ws);
  int32_t *perm = reinterpret_cast<int32_t *>(w);
  int4 *task = reinterpret_cast<int4 *>(w + b_perm);
  B.nmem = cnt;
  P.NU = B.NU = NU;
  P.Sp = B.Sp = h.Sp;
  P.perm = B.perm = perm;
  P.task = B.task = task;
  P.ell = reinterpret_cast<double *>(w + b_perm + b_task);
  double *q = reinterpret_cast<double *>(w + b_perm + b_task + b_ell);
  P.q = q;
  B.qbuf = q;
  P.status = B.status = h.status;
  B.obs = c.obs; B.act = c.act; B.M = h.M; B.T = c.T; B.F = h.F;
  if (mut->test_drop_copy > 0) {   // testing aid: this many calls lose their copies
    P.drop_copy = 1;
    mut->test_drop_copy -= 1;
  }
  A.obs = c.obs; A.q_out = c.q_out; A.logq_out = c.logq_out; A.argmax_out = c.argmax_out;
  A.T = c.T;
  A.lnprior = c.lnprior;
  A.lambda = c.lambda;
  A.xprev = b_x ? reinterpret_cast<double *>(w + b_perm + b_task + b_ell + b_q) : nullptr;
  A.q_init = c.q_init;

  rc = bi_batch_start_f64(md, B, max_m, c.q_init, perm, task, c.stream);
  if (rc != BI_OK) return rc;
  typedef void (*SliceKernel)(MmaParams, int, int);
  typedef void (*PairKernel)(MmaParams, int, int, int);
  typedef void (*UpdateKernel)(const BiDev *, MmaUpdate, const double *, double *, int, int);
  const SliceKernel ks = nw == 8 ? (split ? bi_mma_slice_kernel<false, true, 8> : bi_mma_slice_kernel<false, false, 8>)
                         : split ? (global ? bi_mma_slice_kernel<true, true, 4> : bi_mma_slice_kernel<false, true, 4>)
                                 : (global ? bi_mma_slice_kernel<true, false, 4> : bi_mma_slice_kernel<false, false, 4>);
  const PairKernel kp = nmax <= 16 ? bi_mma_pair_kernel<kPairTiles, 4> : bi_mma_pair_kernel<kPairTiles, 8>;
  const bool damped = A.xprev != nullptr;
  int terms = h.M + 3;   // (see MmaUpdate::common; with several parents a future message from every child)
  for (int f = 0; f < h.F; ++f) terms = std::max(terms, h.M + 1 + __builtin_popcount(A.emask[f]));
  const int upb = std::max(1, kUpdThreads / (h.Sp / 2)), upd_threads = (upb * (h.Sp / 2) + 31) / 32 * 32;
  const int upd_per_sm = ceil_div(NU, upb) > 9 * md->sm_count ? 12 : 9;
  auto pick = [&](bool fin) -> UpdateKernel {
#define BI_UPD(PER) (fin ? (damped ? bi_mma_update_kernel<PER, true, true> : bi_mma_update_kernel<PER, true, false>) \
                         : (damped ? bi_mma_update_kernel<PER, false, true> : bi_mma_update_kernel<PER, false, false>))
    return upd_per_sm == 12 ? BI_UPD(12) : BI_UPD(9);
#undef BI_UPD
  };
  const UpdateKernel mid = pick(false), last = pick(true);
  if (nheavy && bi_allow_smem((const void *)ks, smem) != cudaSuccess) return BI_ERR_CUDA;
  // every launch of the loop may be scheduled while its predecessor drains (see bi_grid_wait)
  // ... and they share SMs, so they ask for one split of L1 and shared memory
  cudaLaunchAttribute pdl[2];
  pdl[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  pdl[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  for (int k = 0; k < c.K; ++k) {
    const int cur = k & 1;
    A.cur = cur;
    A.first = k == 0;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = c.stream;
    cfg.attrs = pdl;
    cfg.numAttrs = nheavy && !global ? 2 : 1;
    if (nheavy) {
      cfg.gridDim = dim3((unsigned)ntask_heavy);
      cfg.dynamicSmemBytes = smem;
      cfg.blockDim = dim3((unsigned)(32 * nw));
      P.task0 = 0;
      if (cudaLaunchKernelEx(&cfg, ks, P, cur, (int)(k == 0)) != cudaSuccess) return BI_ERR_CUDA;
    }
    cfg.dynamicSmemBytes = 0;
    cfg.blockDim = dim3(32 * kWarps);
    if (cnt > nheavy) {
      cfg.gridDim = dim3((unsigned)(ntask - ntask_heavy));
      P.task0 = ntask_heavy;
      if (cudaLaunchKernelEx(&cfg, kp, P, cur, (int)(k == 0), (int)(nheavy > 0)) != cudaSuccess) return BI_ERR_CUDA;
    }
    // (the CTAs that are resident at once: twelve an SM where nine fit waited for the last quarter, 762 against 735 us on 20 480 units of 34 states)
    cfg.gridDim = dim3((unsigned)std::min(ceil_div(NU, upb), upd_per_sm * md->sm_count));
    cfg.blockDim = dim3((unsigned)upd_threads);
    A.common = terms * 54 < 960 && !(c.q_init && (k == 0 || damped));   // (starting beliefs are used as given)
    if (cudaLaunchKernelEx(&cfg, k == c.K - 1 ? last : mid, (const BiDev *)md->d, A, (const double *)P.ell, q, NU, upb) != cudaSuccess)
      return BI_ERR_CUDA;
  }
  if (cudaGetLastError() != cudaSuccess) return BI_ERR_CUDA;
  mut->launches += 1 + (cnt > 0) + c.K * (1 + (nheavy > 0) + (cnt > nheavy));
  mut->last_kernel = c.algo == BI_ALGO_VMP ? "batch_vmp_f64" : "batch_mmp_f64";
  return BI_OK;
}
