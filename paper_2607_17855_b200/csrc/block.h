// Block kernels: plan structures shared by the planner (block.cu) and the kernels (block.cuh).
//
// A unit is one (agent, time step).  Everything a unit's update multiplies with beliefs -- the summed
// slices of the dependency groups over two to four factors, and in window calls the transition matrices
// of the two edges -- is cut into blocks of BR x BC entries, one per thread of the unit's team, and each
// thread keeps its block in registers for all iterations.  The plan, made once with the handle, says per
// block where its beliefs are, where its partial messages go, and per lane of the finishing phase which
// state it completes.
#pragma once
#include <stdint.h>

#include "bi_internal.h"

namespace bi_block {

// what a block contributes
enum {
  KIND_V = 1,      // messages to the row axis (weighted by the prefix beliefs)
  KIND_W = 2,      // messages to the column axis
  KIND_U0 = 4,     // message to the prefix factor that q0 points at
  KIND_U1 = 8,     // message to the prefix factor that q1 points at
  KIND_PAST = 16,  // source: a transition of the edge into the step (strided); else a group's slice
  KIND_FUT = 32    // source: a transition of the edge out of the step
};

// One block.  Belief offsets are relative to the unit's own belief slot (a neighbouring step's slot lies
// one slot stride before or after it); message addresses are elements of the unit's message area.
struct alignas(16) Desc {
  int16_t qr, qc, q0, q1;       // row beliefs, column beliefs, the two prefix entries (or the constant 1)
  int32_t yv, yw;               // first row's / first column's message entry
  int32_t yu0, yu1;             // prefix messages
  int16_t sv, sw;               // entries between consecutive rows' / columns' messages
  int32_t kind;
  int32_t grp, base;            // group and block within it, or factor and first element of a strided source
  int32_t rs, cs;               // strided source: row and column strides
  int16_t rlim, clim;           // strided source: rows and columns that exist
  int32_t pad[3];
};

// One lane of the finishing phase: completes state s of a factor, together with the g - 1 lanes beside it.
// A state's message entries are three runs (groups, edge into the step, edge out of it) of whole 16-byte
// vectors, padded with zeros to the longest run of the pass, so that all lanes make the same trips.
struct alignas(16) Lane {
  int32_t ya;                   // first vector of this lane (element offset in the unit's message area)
  int16_t op, of;               // from ya: first vectors of the two edges' runs
  int16_t qa, f;                // belief entry of the state, factor (-1: idle lane)
  int16_t s, p;                 // state, lane within the state
  int16_t g, n;                 // lanes per state, states of the factor
  int16_t e0, pad0;             // first entry of the factor in the exchange area
  int32_t out;                  // entry in an output belief vector
  int32_t pad;
};
struct alignas(16) Pass {       // 32 lanes
  int32_t gmax;                 // most lanes per state
  int32_t nvec;                 // most vectors of a lane in the groups' run
  int32_t nedge;                // ... in an edge's run
  int32_t nz;                   // most exchange vectors of a factor (all three even)
};

constexpr int kMaxVariants = 10;     // team sizes a plan prepares (window calls: for 1, 2, 3, 4, 6, 12 steps per CTA)
// Threads of a CTA by the registers a block takes (32-bit words): what is left of 65536 registers must hold
// the addresses, beliefs and partial messages beside it.
constexpr int max_threads(int block_words) { return block_words > 32 ? 384 : block_words > 16 ? 512 : 640; }
constexpr int regs_per_thread(int block_words) { return 65536 / max_threads(block_words) & ~7; }
constexpr int kMaxRank = 4;

struct Variant {
  int nbpt, LT, npass;
  const Lane *lane;   // device
  const Pass *pass;
};
struct Plan {
  int ok, max_th;
  int BR, BC, NB, SQ, one, Ysz, Esz;   // Esz: doubles of the exchange area
  int qo[BI_MAX_F];            // belief offset of each factor in a slot
  int nv;
  Variant var[kMaxVariants];
  const Desc *desc;            // device
  int g_nb[BI_MAX_GROUPS];     // blocks of each group
  int ydead, ydump;            // message area of zeros that idle lanes read; one that nobody reads
};

struct Params {
  const Desc *desc;
  const Lane *lane;
  const Pass *pass;
  int32_t NB, nbpt, LT, npass, SQ, one, Ysz, Esz;
  int32_t N, T, K, F, M, S, G, mmp, has_bdep;
  int32_t UC, CS, W;           // window: steps per CTA, CTAs per agent; filtering: agents per CTA
  int32_t max_mem, n_max;      // most modalities of a group, most states of a factor
  int32_t g_any;               // a group over several factors (valid to read from)
  int32_t extra;               // blocks beyond one per thread, in whole warps (kept in shared memory)
  uint32_t ones;               // window: factors of one state (no transition blocks: their actions are only checked)
  int32_t common;              // the softmax needs no shift
  double lambda;
  int32_t n[BI_MAX_F], off[BI_MAX_F], qo[BI_MAX_F], npad[BI_MAX_F], U[BI_MAX_F];
  const void *Mp[BI_MAX_F], *Mf[BI_MAX_F], *logD[BI_MAX_F];
  int64_t Bstride[BI_MAX_F], Dstride[BI_MAX_F];
  int32_t r1_begin[BI_MAX_F + 1];
  int32_t r1_mod[BI_MAX_M], r1_m[BI_MAX_M], r1_P[BI_MAX_M];
  const void *r1_logA[BI_MAX_M];
  int64_t r1_gstride[BI_MAX_M];
  int32_t g_nb[BI_MAX_GROUPS], g_beg[BI_MAX_GROUPS + 1];
  int32_t m_mod[BI_MAX_M], m_m[BI_MAX_M];
  const void *m_blk[BI_MAX_M];
  // transitions that read other factors' states (filtering): parents of each factor
  int32_t bdep_len[BI_MAX_F], bdep[BI_MAX_F][BI_MAX_RANK], PB[BI_MAX_F], wpar;
  const void *Bfull[BI_MAX_F];
  int64_t Bfull_stride[BI_MAX_F];
  const double *exp_tab;
  const int32_t *obs, *act, *act_prev;
  const float *q_prev, *q_init;
  const void *carry_in;
  void *carry_out;
  const void *lnprior;
  float *q_out, *logq_out;
  int32_t *argmax_out;
  uint32_t *status;
  // shared-memory layout
  // (bytes)
  int32_t o_unit, unit_sz;     // per unit: messages, then (offsets from the unit's start)
  int32_t o_cst, o_xp, o_e;    // constants of the logits, previous logits, exchange area
  int32_t o_q, o_par, o_L, o_ref, o_lane;   // belief slots; parents' product (filtering); blocks kept in shared memory
                                            // and their descriptions; the lanes' descriptions
};

}  // namespace bi_block
