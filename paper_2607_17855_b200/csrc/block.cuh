// Block kernels: inference on models of any structure (groups over up to four factors), a team of
// threads per (agent, step).
//
// One Jacobi iteration of a unit (Section IV marginalisation, then the softmax of Section III-A) is two
// phases with one team barrier each:
//
//   contract  every thread takes its BR x BC block of one group's summed slice, which stays in
//             registers for all iterations: with the row and column beliefs from shared memory
//               V[i] = sum_j L[i][j] q_col[j],   W[j] = sum_i q_row[i] L[i][j]
//             (two multiply-adds per entry, none of them waiting for memory), weighted by the prefix
//             beliefs of a group of rank 3 or 4, and u = sum_i q_row[i] V[i] for the prefix factors
//             themselves.  The BR + BC + 2 results go to the message area, every state's entries in one
//             contiguous run.  In window calls the transition matrices of the step's two edges are blocks
//             as well, against the neighbouring steps' beliefs.
//   finish    one to sixteen lanes per state add the state's run, the log-prior and the slices of
//             single-factor modalities and exponentiate; a factor's numerators are summed from a small exchange
//             area.  Several small factors share a pass of one warp, large ones have a warp each.
//
// Why this shape: the kernels it replaced re-read the slices from shared memory or L1 in every
// iteration, decoded row indices as they went and reduced column sums with shuffle trees; they ran at
// 0.5 to 1.5 of the 36 TFLOP/s a float64 unit can do, bound by instruction issue and by serial phases
// of single warps.  Here an iteration's shared-memory traffic is (BR + BC + 2) / (BR BC) of the slice
// instead of all of it, and all offsets are loop invariants in registers.  Bound: the latency of the two
// phases' dependent chains where few teams share an SM, issue and shared-memory throughput where many do.  Five
// coupled factors filtered by 256 agents: 2116 -> 414 us; 1000 agents in float32: 1201 -> 435 us.
#pragma once
#include "bi_internal.h"
#include "block.h"
#include "tile3.cuh"

namespace bi_block {

constexpr int EXP_TAB = 512, EXP_BITS = 9;
constexpr int kTabBytes = EXP_TAB * (int)sizeof(double);   // (MMP: the logarithm's 128 pairs (1/c, ln c) follow)

// exp(x), |x| <= 700, good to 3e-16 relative: x = k ln2/512 + r with the constant in two parts, 2^(j/512) from
// the table, a quartic in r (|r| <= ln2/1024: the first dropped term is below 2e-18).  Zero below -700.
__device__ __forceinline__ double exp_tab_full(double x, const double *__restrict__ tab) {
  const double KL = 738.6598609351493, LKH = 0.0013538030870311431, LKL = 4.529388308293554e-20,   // 512 / ln 2, ln 2 / 512
               MAGIC = 6755399441055744.0;   // 1.5 * 2^52: adding it rounds to the nearest integer
  const double t = fma(x, KL, MAGIC);
  const int k = __double2loint(t);
  const double kd = t - MAGIC;
  double r = fma(kd, -LKH, x);
  r = fma(kd, -LKL, r);
  const double T = tab[k & (EXP_TAB - 1)];
  double a = fma(r, 1.0 / 24.0, 1.0 / 6.0);
  const double r2 = r * r;
  a = fma(r, a, 0.5);
  const double p = fma(r2, a, r);
  const double m = fma(T, p, T);
  const double v = __hiloint2double(__double2hiint(m) + ((k >> EXP_BITS) << 20), __double2loint(m));
  return x < -700.0 ? 0.0 : v;
}

// shared memory by byte offset: 32-bit addresses that the compiler can fold into the instructions
extern __shared__ __align__(16) unsigned char block_smem[];
template <typename T>
__device__ __forceinline__ T &at(int byte) { return *reinterpret_cast<T *>(block_smem + byte); }

// N consecutive beliefs (offset a multiple of two elements; of four where N is)
template <int N>
__device__ __forceinline__ void load_q(int q, double (&x)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const double2 v = at<double2>(q + 8 * i);
    x[i] = v.x; x[i + 1] = v.y;
  }
}
template <int N>
__device__ __forceinline__ void load_q(int q, float (&x)[N]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 v = at<float4>(q + 4 * i);
      x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const float2 v = at<float2>(q + 4 * i);
      x[i] = v.x; x[i + 1] = v.y;
    }
  }
}

// what the contraction of one block needs besides the block: byte offsets, beliefs relative to the unit's own
// slot, messages absolute
struct BlockRef {
  int qr, qc, q0, q1, yv, yw, yu0, yu1, sv, sw, kind;
};
template <typename R>
__device__ __forceinline__ BlockRef block_ref(const Desc *d, int ybase) {
  const int4 a = __ldg(reinterpret_cast<const int4 *>(d)), b = __ldg(reinterpret_cast<const int4 *>(d) + 1);
  constexpr int E = (int)sizeof(R);
  BlockRef r;
  r.qr = (int16_t)(a.x & 0xffff) * E; r.qc = (a.x >> 16) * E;
  r.q0 = (int16_t)(a.y & 0xffff) * E; r.q1 = (a.y >> 16) * E;
  r.yv = ybase + a.z * E; r.yw = ybase + a.w * E;
  r.yu0 = ybase + b.x * E; r.yu1 = ybase + b.y * E;
  r.sv = (int16_t)(b.z & 0xffff) * E; r.sw = (b.z >> 16) * E;
  r.kind = b.w;
  return r;
}

// a block in shared memory, described there too ([3][extra] int4 and [vectors][extra] 16-byte vectors)
__device__ __forceinline__ BlockRef extra_ref(int tab, int i, int extra, int ybase) {
  const int4 a = at<int4>(tab + 16 * i), b = at<int4>(tab + 16 * (extra + i)), c = at<int4>(tab + 16 * (2 * extra + i));
  BlockRef r;
  r.qr = a.x; r.qc = a.y; r.q0 = a.z; r.q1 = a.w;
  r.yv = ybase + b.x; r.yw = ybase + b.y; r.yu0 = ybase + b.z; r.yu1 = ybase + b.w;
  r.sv = c.x; r.sw = c.y; r.kind = c.z;
  return r;
}

// The block's messages.  L(v, x): 16-byte vector v of the block (row-major); DV / DW: what any block of the warp
// contributes (KIND_V or KIND_U*, KIND_W); own: byte offset of the unit's belief slot.  A block that lacks one of
// the results has that message address in an area nobody reads: eight conditional stores cost a lone warp more
// than the arithmetic.
template <typename R, int BR, int BC, bool DV, bool DW, bool LOWREG, class LF>
__device__ __forceinline__ void contract(const LF &L, int own, const BlockRef &b) {
  constexpr int VE = 16 / (int)sizeof(R);
  const R w0 = at<R>(own + b.q0), w1 = at<R>(own + b.q1);
  const R wp = w0 * w1;
  R qc[BC], W[BC];
  if (DV) load_q<BC>(own + b.qc, qc);
  if (DW) {
#pragma unroll
    for (int j = 0; j < BC; ++j) W[j] = (R)0;
  }
  R qr[BR];   // (LOWREG: read row by row, beside a block that already fills the registers)
  if (!LOWREG) load_q<BR>(own + b.qr, qr);
  R u = (R)0, v0 = (R)0, v1 = (R)0;
#pragma unroll
  for (int k = 0; k < BR * BC / VE; ++k) {
    R x[VE];
    L(k, x);
#pragma unroll
    for (int e = 0; e < VE; ++e) {
      const int i = (k * VE + e) / BC, j = (k * VE + e) % BC;
      if (LOWREG && j == 0) qr[i] = at<R>(own + b.qr + i * (int)sizeof(R));
      if (DV) {
        if (j == 0) v0 = x[e] * qc[j];
        else if (j == 1) v1 = x[e] * qc[j];
        else if (j & 1) v1 = fma(x[e], qc[j], v1);
        else v0 = fma(x[e], qc[j], v0);
      }
      if (DW) W[j] = fma(qr[i], x[e], W[j]);
      if (DV && j == BC - 1) {
        const R v = v0 + v1;
        u = fma(qr[i], v, u);
        at<R>(b.yv + i * b.sv) = wp * v;
      }
    }
  }
  if (DV) {
    at<R>(b.yu0) = u * w1;
    at<R>(b.yu1) = u * w0;
  }
  if (DW) {
#pragma unroll
    for (int j = 0; j < BC; ++j) at<R>(b.yw + j * b.sw) = wp * W[j];
  }
}
template <typename R, int BR, int BC, bool LOWREG, class LF>
__device__ __forceinline__ void contract_any(const LF &L, int own, const BlockRef &b, int any) {
  const bool dv = (any & (KIND_V | KIND_U0 | KIND_U1)) != 0, dw = (any & KIND_W) != 0;
  if (dv && dw) contract<R, BR, BC, true, true, LOWREG>(L, own, b);
  else if (dw) contract<R, BR, BC, false, true, LOWREG>(L, own, b);
  else if (dv) contract<R, BR, BC, true, false, LOWREG>(L, own, b);
}
template <typename R>
__device__ __forceinline__ void lds16(int byte, R (&x)[16 / sizeof(R)]) {
  if constexpr (sizeof(R) == 8) {
    const double2 v = at<double2>(byte);
    x[0] = v.x; x[1] = v.y;
  } else {
    const float4 v = at<float4>(byte);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  }
}
// all blocks of the thread: its own in registers, every LT-th of the rest from shared memory
template <typename R, int BR, int BC, bool HASS>
__device__ __forceinline__ void contract_all(const Params &p, const R (&L)[BR * BC], int own, const BlockRef &b0, int any0, int lt, int LT,
                                             int unit, int lbase) {
  constexpr int VE = 16 / (int)sizeof(R);
  contract_any<R, BR, BC, (BR * BC * (int)sizeof(R) > 256)>([&](int v, R (&x)[VE]) {
#pragma unroll
    for (int i = 0; i < VE; ++i) x[i] = L[v * VE + i];
  }, own, b0, any0);
  if (HASS) {
#pragma unroll 1
    for (int i = lt; i < p.extra; i += LT) {
      const BlockRef b = extra_ref(p.o_ref, i, p.extra, unit);
      const int any = (int)__reduce_or_sync(0xffffffffu, (unsigned)b.kind);
      const int src = lbase + 16 * i, st = 16 * p.extra;
      contract_any<R, BR, BC, true>([&](int v, R (&x)[VE]) { lds16<R>(src + v * st, x); }, own, b, any);
    }
  }
}
// the descriptions of the blocks in shared memory (once per launch, for all teams of the CTA)
template <typename R>
__device__ __forceinline__ void stage_refs(const Params &p) {
  for (int i = threadIdx.x; i < p.extra; i += blockDim.x) {
    const int blk = p.LT + i;
    const BlockRef r = block_ref<R>(p.desc + min(blk, p.NB), 0);
    at<int4>(p.o_ref + 16 * i) = make_int4(r.qr, r.qc, r.q0, r.q1);
    at<int4>(p.o_ref + 16 * (p.extra + i)) = make_int4(r.yv, r.yw, r.yu0, r.yu1);
    at<int4>(p.o_ref + 16 * (2 * p.extra + i)) = make_int4(r.sv, r.sw, r.kind, 0);
  }
}

// ---- finishing one pass (32 lanes) ----
// n (even) vectors from y on, st bytes apart.  Eight, four or two loads go out together: one after the other a
// trip of two costs a lone warp about a hundred cycles, most of them latency.
template <int N>
__device__ __forceinline__ void add_vecs(double (&a)[4], int y, int st) {
  double2 v[N];
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = at<double2>(y + i * st);
#pragma unroll
  for (int i = 0; i < N; ++i) { a[(2 * i) & 3] += v[i].x; a[(2 * i + 1) & 3] += v[i].y; }
}
template <int N>
__device__ __forceinline__ void add_vecs(float (&a)[4], int y, int st) {
  float4 v[N];
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = at<float4>(y + i * st);
#pragma unroll
  for (int i = 0; i < N; ++i) { a[0] += v[i].x; a[1] += v[i].y; a[2] += v[i].z; a[3] += v[i].w; }
}
template <typename R>
__device__ __forceinline__ double sum_run(int y, int n, int st) {
  R a[4] = {(R)0, (R)0, (R)0, (R)0};
#pragma unroll 1
  for (; n >= 8; n -= 8, y += 8 * st) add_vecs<8>(a, y, st);
  if (n & 4) { add_vecs<4>(a, y, st); y += 4 * st; }
  if (n & 2) add_vecs<2>(a, y, st);
  return (double)((a[0] + a[1]) + (a[2] + a[3]));
}

struct LaneRef {     // byte offsets, absolute unless said otherwise
  int y, p, fo, st;  // first vectors of the three runs; bytes between a lane's vectors
  int qa, ca;        // belief entry within a slot; the same entry in the (double) arrays of constants and logits
  int e, ez;         // own exchange entry, the factor's first
  int g;
  int4 pass;
  bool writes;
};
// The lanes' descriptions, in shared memory for all teams of the CTA (16 bytes each; a pass' own 16 bytes behind
// them): read again in every iteration just before the barrier between the phases, so that they take no
// registers beside the blocks; the filtering kernel keeps a warp's first one where the blocks are small (see kKeepLanes).
template <typename R>
__device__ __forceinline__ void stage_lanes(const Params &p) {
  const int n = p.npass * 32;
  auto lo = [](int x) { return x & 0xffff; };
  auto hi = [](int x) { return (x >> 16) & 0xffff; };
  constexpr int VE = 16 / (int)sizeof(R);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int4 a = __ldg(reinterpret_cast<const int4 *>(p.lane + i)), b = __ldg(reinterpret_cast<const int4 *>(p.lane + i) + 1);
    const int qa = lo(a.z), f = (int)(int16_t)hi(a.z), s = lo(a.w), q = hi(a.w), g = lo(b.x), e0 = lo(b.y);
    const int y = a.x / VE, op = lo(a.y) / VE, of = hi(a.y) / VE;   // in vectors
    at<int4>(p.o_lane + 16 * i) = make_int4(y | op << 16, of | (g | (f >= 0 && q == 0 ? 0x8000 : 0)) << 16, qa | e0 << 16, s);
  }
  for (int i = threadIdx.x; i < p.npass; i += blockDim.x)
    at<int4>(p.o_lane + 16 * (n + i)) = __ldg(reinterpret_cast<const int4 *>(p.pass) + i);
}
template <typename R>
__device__ __forceinline__ LaneRef lane_ref(const Params &p, int pass, int lane, int unit, int ex) {
  const int4 a = at<int4>(p.o_lane + 16 * (pass * 32 + lane));
  LaneRef r;
  r.pass = at<int4>(p.o_lane + 16 * (p.npass * 32 + pass));
  r.y = unit + (a.x & 0xffff) * 16;
  r.p = r.y + (a.x >> 16) * 16;
  r.fo = r.y + (a.y & 0xffff) * 16;
  r.g = (a.y >> 16) & 0x7fff;
  r.st = r.g * 16;
  r.writes = a.y < 0;
  r.qa = (a.z & 0xffff) * (int)sizeof(R);
  r.ca = (a.z & 0xffff) * 8;
  r.ez = ex + (a.z >> 16) * 8;
  r.e = r.ez + a.w * 8;
  return r;
}

// store into another CTA of the cluster (a shared::cluster address)
__device__ __forceinline__ void st_cluster(uint32_t a, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ void st_cluster(uint32_t a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }

struct StepOut {          // where a unit's results go (pointers already at the unit), and what is wanted
  float *q, *logq;
  int32_t *argmax;
  void *carry;            // [S] of the unit's agent, or NULL
  bool store;             // idle units store nothing
};

// The sum of the numerators is taken by every lane itself from the exchange area (in shared memory, one
// 16-byte load and two additions per two states, all lanes of a factor reading one address): states need no
// alignment to powers of two within a pass, and nothing is shuffled.
// The exponentials need no shift where the logits are sums of at most seventeen logarithms of probabilities (`common`,
// decided by the launcher): none is above zero and none below -640, so the numerators and their sum are normal
// numbers.  Otherwise they are relative to the factor's largest logit (starting beliefs are used as
// given, which counts for the first iteration, and under damping for all).
template <typename R, bool WIN, bool FINAL>
__device__ __forceinline__ void finish(const Params &p, const LaneRef &l, int cst, int xp, int qslot, bool common,
                                       bool has_prev, bool has_next, const StepOut &o, const Lane *cold, uint32_t halo0,
                                       uint32_t halo1) {
  const bool mmp = WIN && p.mmp;
  const int4 ps = l.pass;
  double v = sum_run<R>(l.y, ps.y, l.st);
  double vp = 0.0, vf = 0.0;
  if (WIN) {
    vp = sum_run<R>(l.p, ps.z, l.st);
    vf = sum_run<R>(l.fo, ps.z, l.st);
    if (!mmp) v += vp + vf;
  }
#pragma unroll 1
  for (int d = 1; d < ps.x; d <<= 1) {   // the lanes of one state
    const double a = __shfl_xor_sync(0xffffffffu, v, d);
    v += d < l.g ? a : 0.0;
    if (mmp) {
      const double b = __shfl_xor_sync(0xffffffffu, vp, d), c = __shfl_xor_sync(0xffffffffu, vf, d);
      vp += d < l.g ? b : 0.0;
      vf += d < l.g ? c : 0.0;
    }
  }
  double x = v + at<double>(cst + l.ca);
  if (mmp) {
    double lp, lf;
    if constexpr (sizeof(R) == 8) {
      const double2 *lt = reinterpret_cast<const double2 *>(block_smem + kTabBytes);
      lp = 0.5 * bi_log_fast(bi_max(vp, BI_EPS), lt); lf = 0.5 * bi_log_fast(bi_max(vf, BI_EPS), lt);
    } else {
      lp = 0.5f * logf(fmaxf((float)vp, (float)BI_EPS)); lf = 0.5f * logf(fmaxf((float)vf, (float)BI_EPS));
    }
    x += (has_prev ? lp : 0.0) + (has_next ? lf : 0.0);
  }
  if (xp >= 0) x = fma(p.lambda, x, (1.0 - p.lambda) * at<double>(xp + l.ca));   // damped step on the logits
  double xs = x;
  if (!common) {
    if (l.writes) at<double>(l.e) = xs;
    __syncwarp();
    const int n = __ldg(&cold->n);
    double m = -CUDART_INF;
#pragma unroll 4
    for (int r = 0; r < 2 * ps.w; ++r) m = bi_max(m, at<double>(l.ez + 8 * min(r, n - 1)));
    __syncwarp();
    xs -= m;
  }
  const double e = exp_tab_full(xs, reinterpret_cast<const double *>(block_smem));
  if (l.writes) at<double>(l.e) = e;
  __syncwarp();
  double za[4] = {0.0, 0.0, 0.0, 0.0};   // (two, four, eight or sixteen vectors, zeros behind the states)
  if (ps.w <= 2) add_vecs<2>(za, l.ez, 16);
  else if (ps.w <= 4) add_vecs<4>(za, l.ez, 16);
  else if (ps.w <= 8) add_vecs<8>(za, l.ez, 16);
  else {
    add_vecs<8>(za, l.ez, 16);
    add_vecs<8>(za, l.ez + 128, 16);
  }
  const double z = (za[0] + za[1]) + (za[2] + za[3]);
  const R q = (R)(e * bi_rcp(z));
  if (l.writes) {
    at<R>(qslot + l.qa) = q;
    if (WIN) {
      if (halo0) st_cluster(halo0 + l.qa, q);
      if (halo1) st_cluster(halo1 + l.qa, q);
    }
    if (xp >= 0) at<double>(xp + l.ca) = x;
  }
  if (FINAL) {
    const int out = __ldg(&cold->out), f = __ldg(&cold->f), s = __ldg(&cold->s);
    if (l.writes && o.store) {
      o.q[out] = (float)q;
      if (o.logq) o.logq[out] = (float)(xs - log(z));
      if (o.carry) ((R *)o.carry)[out] = q;
    }
    if (o.argmax) {   // lowest index among equals: the factor's logits through the exchange area
      __syncwarp();
      if (l.writes) at<double>(l.e) = x;
      __syncwarp();
      const int n = __ldg(&cold->n);
      double best = -CUDART_INF;
      int idx = 0;
      for (int r = 0; r < 32; ++r) {
        const double y = at<double>(l.ez + 8 * min(r, n - 1));
        if (y > best) { best = y; idx = min(r, n - 1); }
      }
      if (l.writes && s == 0 && o.store) o.argmax[f] = idx;
      __syncwarp();
    }
  }
}

// How a team synchronises: one warp; the whole CTA; one of several teams of a CTA (named barriers -- a kernel
// of its own, because one that names barriers at run time reserves all sixteen and then only four CTAs fit an SM)
enum { SYNC_WARP = 0, SYNC_CTA = 1, SYNC_NAMED = 2 };
template <int SYNC>
__device__ __forceinline__ void team_sync(int LT, int team) {
  if (SYNC == SYNC_WARP) __syncwarp();
  else if (SYNC == SYNC_CTA) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(LT) : "memory");
}

// this thread's block of a group's summed slice, from the block-ordered copies of the group's modalities
// (16-byte vector v of block b at v * nb + b: consecutive lanes read consecutive vectors)
template <typename R, int BR, int BC>
__device__ __forceinline__ void gather_group(const Params &p, R (&L)[BR * BC], int grp, int blk, int g, const int32_t *obs_t) {
  constexpr int VE = 16 / (int)sizeof(R), NV = BR * BC / VE;
  const int nb = p.g_nb[grp], beg = p.g_beg[grp], cnt = p.g_beg[grp + 1] - beg;
  const size_t st = (size_t)nb * VE;
  // (No branch and no trip count here differs between the lanes -- one with fewer modalities adds zeros --
  // because a warp split in the set-up stays split through the step's iterations: measured, 2.6 times the
  // instructions per iteration.)
#pragma unroll
  for (int e = 0; e < BR * BC; ++e) L[e] = (R)0;
  for (int k = 0; k < p.max_mem; ++k) {
    const int mi = beg + min(k, cnt - 1);
    const int o = clamp_flag(__ldg(obs_t + p.m_mod[mi]), p.m_m[mi], p.status, BI_FLAG_OBS_RANGE);
    const R *src = (const R *)p.m_blk[mi] + (((size_t)g * p.m_m[mi] + o) * NV * nb + blk) * VE;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      R x[VE];
      ldg_vec(src + v * st, x);
#pragma unroll
      for (int i = 0; i < VE; ++i) L[v * VE + i] += k < cnt ? x[i] : (R)0;
    }
  }
}
// factor of entry i of an output belief vector
__device__ __forceinline__ int factor_of(const Params &p, int i) {
  int f = 0;
#pragma unroll
  for (int k = 1; k < BI_MAX_F; ++k) f += k < p.F && i >= p.off[k] ? 1 : 0;
  return f;
}
// the slices of factor f's own modalities at state s (the same trips in every lane, see gather_group)
template <typename R>
__device__ __forceinline__ R single_factor_slices(const Params &p, int f, int s, int g, const int32_t *obs_t) {
  R c = (R)0;
  const int n1 = p.r1_begin[p.F], beg = p.r1_begin[f], end = p.r1_begin[f + 1];
  for (int j = 0; j < n1; ++j) {
    const int o = clamp_flag(__ldg(obs_t + p.r1_mod[j]), p.r1_m[j], p.status, BI_FLAG_OBS_RANGE);
    const bool mine = j >= beg && j < end;
    const R x = __ldg((const R *)p.r1_logA[j] + (size_t)g * p.r1_gstride[j] + (size_t)o * p.r1_P[j] + (mine ? s : 0));
    c += mine ? x : (R)0;
  }
  return c;
}

// ---- filtering: W agents per CTA (teams of one warp) or one agent per CTA ----
// HASS: teams with more blocks than threads keep a thread's further blocks in shared memory.
template <typename R, int BR, int BC, int SYNC, bool HASS>
__global__ void __launch_bounds__(SYNC == SYNC_WARP ? 128 : max_threads(BR * BC * (int)sizeof(R) / 4),
                                  SYNC == SYNC_WARP ? max_threads(BR * BC * (int)sizeof(R) / 4) / 128 : 1)
bi_block_filter_kernel(const __grid_constant__ Params p) {
  constexpr int E = (int)sizeof(R), VE = 16 / E, NV = BR * BC / VE;
  const int LT = p.LT, team = (int)threadIdx.x / LT, lt = (int)threadIdx.x - team * LT, lane = lt & 31;
  const int warp = lt >> 5, NW = LT >> 5;
  for (int j = threadIdx.x; j < EXP_TAB / 2; j += blockDim.x)
    at<double2>(16 * j) = __ldg(reinterpret_cast<const double2 *>(p.exp_tab) + j);
  const int unit = p.o_unit + team * p.unit_sz, cst = unit + p.o_cst, ex = unit + p.o_e;
  const int xp = p.lambda != 1.0 ? unit + p.o_xp : -1;
  const int own = p.o_q + team * p.SQ * E;
  for (int i = lt; i < p.SQ; i += LT) {
    at<R>(own + i * E) = i == p.one ? (R)1 : (R)0;
    at<double>(cst + i * 8) = 0.0;
  }
  for (int i = lt; i < p.Ysz; i += LT) at<R>(unit + i * E) = (R)0;   // (the runs' closing vectors and padding stay zero)
  for (int i = lt; i < p.Esz; i += LT) at<double>(ex + 8 * i) = 0.0;
  if (HASS) stage_refs<R>(p);
  stage_lanes<R>(p);
  __syncthreads();
  const int a = (int)blockIdx.x * p.W + team;
  if (a >= p.N) return;   // (only teams of one warp: nothing below synchronises more than a team)
  const int g = p.G == 1 ? 0 : a;

  // ---- this thread's block and this lane's state, for the whole call
  const bool has = lt < p.NB;
  const BlockRef b0 = block_ref<R>(p.desc + min(lt, p.NB), unit);   // (entry NB: no block)
  const int2 src0 = __ldg(reinterpret_cast<const int2 *>(&(p.desc + (has ? lt : 0))->grp));
  const int any0 = (int)__reduce_or_sync(0xffffffffu, (unsigned)b0.kind);
  const bool lanes0 = warp < p.npass;
  // the description of the warp's first pass, kept where the blocks are small enough to leave the registers for it
  // (a description read again in every iteration is 40 instructions and a round trip to shared memory; 1000 agents, [7,9,5],
  // float32, 8 x 4 blocks: 436 -> 414 us; 585 agents, [8,5], 4 x 4: 262 -> 246 us; beside 8 x 6 in float64 it spills)
  constexpr bool kKeepLanes = BR * BC * E <= 256;
  const LaneRef l0 = lane_ref<R>(p, lanes0 ? warp : 0, lane, unit, ex);
  const bool common = p.common != 0 && __ldg(p.status + 1) == 0;

  const bool from_prev = p.q_prev != nullptr || p.carry_in != nullptr;
  if (from_prev) {
    for (int i0 = 0; i0 < p.S; i0 += LT) {
      const int i = min(i0 + lt, p.S - 1), f = factor_of(p, i);
      const size_t src = (size_t)a * p.S + i;
      at<R>(own + (p.qo[f] + i - p.off[f]) * E) = p.carry_in ? ((const R *)p.carry_in)[src] : (R)p.q_prev[src];   // (q_prev may alias q_out)
    }
    team_sync<SYNC>(LT, team);
  }
  for (int t = 0; t < p.T; ++t) {
    const int32_t *obs_t = p.obs + ((size_t)a * p.T + t) * p.M;
    // ---- the step's blocks (those for shared memory first: the own one's registers are still free)
    if (HASS) {
      for (int i = lt; i < p.extra; i += LT) {
        const int2 src = __ldg(reinterpret_cast<const int2 *>(&(p.desc + min(LT + i, p.NB - 1))->grp));
        R X[BR * BC];
        gather_group<R, BR, BC>(p, X, src.x, src.y, g, obs_t);
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int e = 0; e < VE; ++e) at<R>(p.o_L + (v * p.extra + i) * 16 + e * E) = X[v * VE + e];
      }
    }
    R L[BR * BC];
#pragma unroll
    for (int i = 0; i < BR * BC; ++i) L[i] = (R)0;
    if (p.NB > 0) gather_group<R, BR, BC>(p, L, src0.x, src0.y, g, obs_t);   // (threads without a block read the first one)
    // ---- constants of the logits: ln prior (D, or B_u times the previous belief) and the slices of
    // modalities that depend on one factor
    if (p.has_bdep && (t > 0 || from_prev)) {
      const int par = p.o_par + team * p.wpar * E;
      for (int f = 0; f < p.F; ++f) {
        const int n = p.n[f], PB = p.PB[f], k = p.bdep_len[f];
        for (int e0 = 0; e0 < PB; e0 += LT) {   // the parents' product, last parent fastest
          const int e = min(e0 + lt, PB - 1);
          int rem = e;
          R w = (R)1;
          for (int j = k - 1; j >= 0; --j) {
            const int gq = p.bdep[f][j], nj = p.n[gq];
            const int dgt = rem % nj;
            rem /= nj;
            w *= at<R>(own + (p.qo[gq] + dgt) * E);
          }
          at<R>(par + e * E) = w;
        }
        team_sync<SYNC>(LT, team);
        const int ur = t == 0 ? __ldg(p.act_prev + (size_t)a * p.F + f) : __ldg(p.act + ((size_t)a * (p.T - 1) + (t - 1)) * p.F + f);
        const int u = clamp_flag(ur, p.U[f], p.status, BI_FLAG_ACT_RANGE);
        const R *Xu = (const R *)p.Bfull[f] + (size_t)g * p.Bfull_stride[f] + (size_t)u * n * PB;
        // eight lanes per next state, four states to a warp (with one warp per state a lone warp spends its time in
        // reductions)
        for (int s0 = 4 * warp; s0 < n; s0 += 4 * NW) {
          const int s = min(s0 + (lane >> 3), n - 1), e8 = lane & 7;
          const R *row = Xu + (size_t)s * PB;
          R acc = (R)0;
#pragma unroll 4
          for (int e0 = 0; e0 < PB; e0 += 8) {
            const int e = min(e0 + e8, PB - 1);
            acc = fma(__ldg(row + e), e0 + e8 < PB ? at<R>(par + e * E) : (R)0, acc);
          }
          acc += __shfl_xor_sync(0xffffffffu, acc, 1);
          acc += __shfl_xor_sync(0xffffffffu, acc, 2);
          acc += __shfl_xor_sync(0xffffffffu, acc, 4);
          if (e8 == 0) at<double>(cst + (p.qo[f] + s) * 8) = (double)bi_log(bi_max(acc, (R)BI_EPS));
        }
        team_sync<SYNC>(LT, team);
      }
    }
    for (int i0 = 0; i0 < p.S; i0 += LT) {   // (lanes beyond the last state repeat it and store nothing)
      const int i = min(i0 + lt, p.S - 1);
      const int f = factor_of(p, i);
      const int s = i - p.off[f], n = p.n[f], np = p.npad[f];
      R c;
      if (t == 0 && !from_prev) {
        c = __ldg((const R *)p.logD[f] + (size_t)g * p.Dstride[f] + s);
      } else if (p.has_bdep) {
        c = (R)at<double>(cst + (p.qo[f] + s) * 8);
      } else {
        const int ur = t == 0 ? __ldg(p.act_prev + (size_t)a * p.F + f) : __ldg(p.act + ((size_t)a * (p.T - 1) + (t - 1)) * p.F + f);
        const int u = clamp_flag(ur, p.U[f], p.status, BI_FLAG_ACT_RANGE);
        // [previous][next]: the lanes of consecutive states read consecutive addresses
        const R *col = (const R *)p.Mp[f] + (size_t)g * p.Bstride[f] + (size_t)u * n * np + s;
        const int q = own + p.qo[f] * E;
        R c0 = (R)0, c1 = (R)0;
#pragma unroll 4
        for (int r = 0; r < p.n_max; r += 2) {   // (trips of the largest factor for every lane, see gather_group)
          const int r0 = min(r, n - 1), r1 = min(r + 1, n - 1);
          const R q0 = at<R>(q + r0 * E), q1 = at<R>(q + r1 * E);
          c0 = fma(__ldg(col + (size_t)r0 * np), r < n ? q0 : (R)0, c0);
          c1 = fma(__ldg(col + (size_t)r1 * np), r + 1 < n ? q1 : (R)0, c1);
        }
        c = bi_log_inline(bi_max(c0 + c1, (R)BI_EPS));
      }
      const double cc = (double)c + (double)single_factor_slices<R>(p, f, s, g, obs_t);
      if (p.has_bdep) team_sync<SYNC>(LT, team);   // (the threads that repeat the last state have read its constant)
      if (i0 + lt < p.S) at<double>(cst + (p.qo[f] + s) * 8) = cc;
    }
    team_sync<SYNC>(LT, team);
    // ---- uniform start
    for (int i0 = 0; i0 < p.S; i0 += LT) {
      const int i = min(i0 + lt, p.S - 1);
      const int f = factor_of(p, i);
      const int q = p.qo[f] + i - p.off[f];
      at<R>(own + q * E) = (R)1 / (R)p.n[f];
      if (xp >= 0) at<double>(xp + q * 8) = 0.0;   // logits of the uniform start: a constant
    }
    team_sync<SYNC>(LT, team);
    StepOut o;
    o.q = nullptr; o.logq = nullptr; o.argmax = nullptr; o.carry = nullptr;
    o.store = true;
#pragma unroll 1
    for (int k = 0; k < p.K; ++k) {
      contract_all<R, BR, BC, HASS>(p, L, own, b0, any0, lt, LT, unit, p.o_L);
      LaneRef l = kKeepLanes ? l0 : lane_ref<R>(p, lanes0 ? warp : 0, lane, unit, ex);
      team_sync<SYNC>(LT, team);
      if (k < p.K - 1) {
        if (lanes0) {
#pragma unroll 1
          for (int ps = warp;;) {
            finish<R, false, false>(p, l, cst, xp, own, common, false, false, o, p.lane + ps * 32 + lane, 0u, 0u);
            ps += NW;
            if (ps >= p.npass) break;
            l = lane_ref<R>(p, ps, lane, unit, ex);
          }
        }
      } else {
        o.q = p.q_out + ((size_t)a * p.T + t) * p.S;
        o.logq = p.logq_out ? p.logq_out + ((size_t)a * p.T + t) * p.S : nullptr;
        o.argmax = p.argmax_out ? p.argmax_out + ((size_t)a * p.T + t) * p.F : nullptr;
        o.carry = p.carry_out && t == p.T - 1 ? (void *)((R *)p.carry_out + (size_t)a * p.S) : nullptr;
#pragma unroll 1
        for (int ps = warp; ps < p.npass; ps += NW) {
          finish<R, false, true>(p, lane_ref<R>(p, ps, lane, unit, ex), cst, xp, own, common, false, false, o,
                                 p.lane + ps * 32 + lane, 0u, 0u);
        }
      }
      team_sync<SYNC>(LT, team);
    }
  }
}

// ---- windows (VMP / MMP): a team per time step, UC steps per CTA, CS CTAs (a cluster) per agent ----
// Beliefs are double-buffered in shared memory, a slot per step plus one halo slot at either end; at a CTA
// boundary the finishing lanes also store into the neighbouring CTA's halo (distributed shared memory),
// so every read is local.  One barrier over the CTA (or cluster) per iteration (Appendix A-2 runs the
// window's steps side by side; Section IV's transition messages read the neighbours' previous iterate).
template <typename R, int BR, int BC, int SYNC, bool HASS>
__global__ void __launch_bounds__(max_threads(BR * BC * (int)sizeof(R) / 4), 1) bi_block_window_kernel(const __grid_constant__ Params p) {
  constexpr int E = (int)sizeof(R), VE = 16 / E, NV = BR * BC / VE;
  const int LT = p.LT, team = (int)threadIdx.x / LT, lt = (int)threadIdx.x - team * LT, lane = lt & 31;
  const int warp = lt >> 5, NW = LT >> 5;
  for (int j = threadIdx.x; j < EXP_TAB / 2 + (p.mmp ? BI_LOG_TAB : 0); j += blockDim.x)
    at<double2>(16 * j) = __ldg(reinterpret_cast<const double2 *>(p.exp_tab) + j);
  const bool cluster = p.CS > 1;
  const int agent = (int)blockIdx.x / p.CS, rank = (int)blockIdx.x - agent * p.CS;
  const int g = p.G == 1 ? 0 : agent;
  const int t_raw = rank * p.UC + team, T = p.T;
  const bool live = t_raw < T;
  const int t = live ? t_raw : T - 1;   // idle teams shadow the last step; they store and publish nothing that is read
  const int unit = p.o_unit + team * p.unit_sz, cst = unit + p.o_cst, ex = unit + p.o_e;
  const int xp = p.lambda != 1.0 ? unit + p.o_xp : -1;
  const int slot_sz = p.SQ * E, bufsz = (p.UC + 2) * slot_sz;
  const int32_t *obs_t = p.obs + ((size_t)agent * T + t) * p.M;

  // ---- belief slots: zero padding, the constant 1, the starting beliefs of every step (halos too)
  for (int i = threadIdx.x; i < 2 * (p.UC + 2) * p.SQ; i += blockDim.x) at<R>(p.o_q + i * E) = (i % p.SQ) == p.one ? (R)1 : (R)0;
  for (int i = lt; i < p.SQ; i += LT) {
    at<double>(cst + i * 8) = 0.0;
    if (xp >= 0) at<double>(xp + i * 8) = 0.0;
  }
  for (int i = lt; i < p.Ysz; i += LT) at<R>(unit + i * E) = (R)0;   // (the runs' closing vectors and padding stay zero)
  for (int i = lt; i < p.Esz; i += LT) at<double>(ex + 8 * i) = 0.0;
  if (HASS) stage_refs<R>(p);
  stage_lanes<R>(p);
  __syncthreads();
  for (int i0 = 0; i0 < (p.UC + 2) * p.S; i0 += blockDim.x) {
    const int i = min(i0 + (int)threadIdx.x, (p.UC + 2) * p.S - 1);
    const int slot = i / p.S, e = i - slot * p.S, ts = rank * p.UC + slot - 1;
    const bool real = ts >= 0 && ts < T;
    const int f = factor_of(p, e);
    R q = (R)1 / (R)p.n[f];
    if (p.q_init) q = (R)__ldg(p.q_init + ((size_t)agent * T + (real ? ts : 0)) * p.S + e);
    if (real) at<R>(p.o_q + slot * slot_sz + (p.qo[f] + e - p.off[f]) * E) = q;
  }
  // ---- this team's constants
  for (int i0 = 0; i0 < p.S; i0 += LT) {   // (lanes beyond the last state repeat it and store nothing)
    const int i = min(i0 + lt, p.S - 1);
    const bool real = i0 + lt < p.S;
    const int f = factor_of(p, i);
    const int s = i - p.off[f];
    R c = (R)0;
    if (t == 0)
      c = p.lnprior ? __ldg((const R *)p.lnprior + (size_t)agent * p.S + i)
                    : __ldg((const R *)p.logD[f] + (size_t)g * p.Dstride[f] + s);
    const double cc = (double)c + (double)single_factor_slices<R>(p, f, s, g, obs_t);
    if (real) at<double>(cst + (p.qo[f] + s) * 8) = cc;
    // (the damped update starts from the logarithms of the given beliefs; the uniform start's are a constant)
    if (xp >= 0 && p.q_init && real)
      at<double>(xp + (p.qo[f] + s) * 8) = (double)bi_log(bi_max((R)__ldg(p.q_init + ((size_t)agent * T + t) * p.S + i), (R)BI_EPS));
  }
  if (t > 0)
    for (uint32_t mk = p.ones; mk; mk &= mk - 1) {
      const int f = __ffs(mk) - 1;
      clamp_flag(__ldg(p.act + ((size_t)agent * (T - 1) + (t - 1)) * p.F + f), p.U[f], p.status, BI_FLAG_ACT_RANGE);
    }
  // ---- this thread's block: a group's summed slice, or part of an edge's transition (both are read and one
  // is taken where a warp holds blocks of both kinds: see gather_group on why the warp must not split)
  const bool has_prev = t > 0, has_next = t + 1 < T;
  auto gather = [&](const Desc *d, R (&L)[BR * BC]) {
    const int4 c = __ldg(reinterpret_cast<const int4 *>(d) + 2);   // grp, base, rs, cs
    const int4 e = __ldg(reinterpret_cast<const int4 *>(d) + 3);   // rlim | clim << 16
    const int kind = __ldg(&d->kind);
    const bool edge = (kind & (KIND_PAST | KIND_FUT)) != 0;
    const bool any_edge = __any_sync(0xffffffffu, edge), any_group = __any_sync(0xffffffffu, !edge);
#pragma unroll
    for (int i = 0; i < BR * BC; ++i) L[i] = (R)0;
    if (any_group && p.max_mem > 0) {
      const int grp = edge ? p.g_any : c.x, blk = edge ? 0 : c.y;
      gather_group<R, BR, BC>(p, L, grp, blk, g, obs_t);
    }
    if (any_edge) {
      const bool past = (kind & KIND_PAST) != 0;
      const bool real = edge && (past ? has_prev : has_next);
      const int f = edge ? c.x : 0, tt = past ? t - 1 : t;
      const int ua = real ? __ldg(p.act + ((size_t)agent * (T - 1) + tt) * p.F + f) : 0;
      const int u = clamp_flag(ua, p.U[f], p.status, BI_FLAG_ACT_RANGE);
      const R *src = p.has_bdep ? (const R *)p.Mp[f] + (size_t)g * p.Bfull_stride[f] + (size_t)u * p.n[f] * p.PB[f]
                                : (const R *)(past ? p.Mp[f] : p.Mf[f]) + (size_t)g * p.Bstride[f] + (size_t)u * p.n[f] * p.npad[f];
      if (edge) src += c.y;
      const int rlim = real ? (int16_t)(e.x & 0xffff) : 0, clim = real ? e.x >> 16 : 0;
#pragma unroll
      for (int i = 0; i < BR; ++i)
#pragma unroll
        for (int j = 0; j < BC; ++j) {
          const bool in = i < rlim && j < clim;
          const R x = __ldg(src + (in ? (size_t)i * c.z + (size_t)j * c.w : 0));
          L[i * BC + j] = edge ? (in ? x : (R)0) : L[i * BC + j];
        }
    }
  };
  const bool has = lt < p.NB;
  const BlockRef b0 = block_ref<R>(p.desc + min(lt, p.NB), unit);   // (entry NB: no block)
  const int lbase = p.o_L + team * p.extra * BR * BC * E;
  if (HASS) {
    for (int i = lt; i < p.extra; i += LT) {
      R X[BR * BC];
      gather(p.desc + min(LT + i, p.NB - 1), X);
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int e = 0; e < VE; ++e) at<R>(lbase + (v * p.extra + i) * 16 + e * E) = X[v * VE + e];
    }
  }
  R L[BR * BC];
  gather(p.desc + (has ? lt : 0), L);
  const int any0 = (int)__reduce_or_sync(0xffffffffu, (unsigned)b0.kind);
  const bool lanes0 = warp < p.npass;
  const bool common_all = p.common != 0 && __ldg(p.status + 1) == 0;

  // halo slots of the neighbouring CTAs that this team feeds (buffer 0)
  uint32_t h_prev = 0, h_next = 0;   // (0: none; the exponential table sits at the start of shared memory)
  if (cluster) {
    auto remote = [&](int r, int slot) -> uint32_t {   // address of a slot in another CTA of the cluster
      uint32_t out;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(bi_smem_addr(block_smem + p.o_q + slot * slot_sz)), "r"(r));
      return out;
    };
    if (live && team == 0 && rank > 0) h_prev = remote(rank - 1, p.UC + 1);
    if (live && team == p.UC - 1 && rank + 1 < p.CS) h_next = remote(rank + 1, 0);
  }
  auto all_sync = [&]() {
    if (cluster) {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
      __syncthreads();
    }
  };
  StepOut o;
  o.q = nullptr; o.logq = nullptr; o.argmax = nullptr; o.carry = nullptr;
  o.store = live;
  all_sync();
  int own = p.o_q + (team + 1) * slot_sz, dst = own + bufsz;   // this step's slot in the current and the next buffer
  int hoff = bufsz;                                           // ... and the halos' next buffer
#pragma unroll 1
  for (int k = 0; k < p.K; ++k) {
    const bool common = common_all && (k > 0 || !p.q_init);
    contract_all<R, BR, BC, HASS>(p, L, own, b0, any0, lt, LT, unit, lbase);
    LaneRef l = lane_ref<R>(p, lanes0 ? warp : 0, lane, unit, ex);
    team_sync<SYNC>(LT, team);
    const uint32_t h0 = h_prev ? h_prev + hoff : 0u, h1 = h_next ? h_next + hoff : 0u;
    if (k < p.K - 1) {
      if (lanes0) {
#pragma unroll 1
        for (int ps = warp;;) {
          finish<R, true, false>(p, l, cst, xp, dst, common, has_prev, has_next, o, p.lane + ps * 32 + lane, h0, h1);
          ps += NW;
          if (ps >= p.npass) break;
          l = lane_ref<R>(p, ps, lane, unit, ex);
        }
      }
    } else {
      o.q = p.q_out + ((size_t)agent * T + t) * p.S;
      o.logq = p.logq_out ? p.logq_out + ((size_t)agent * T + t) * p.S : nullptr;
      o.argmax = p.argmax_out ? p.argmax_out + ((size_t)agent * T + t) * p.F : nullptr;
#pragma unroll 1
      for (int ps = warp; ps < p.npass; ps += NW) {
        finish<R, true, true>(p, lane_ref<R>(p, ps, lane, unit, ex), cst, xp, dst, common, has_prev, has_next, o,
                              p.lane + ps * 32 + lane, h0, h1);
      }
    }
    { const int tmp = own; own = dst; dst = tmp; }
    hoff = bufsz - hoff;
    all_sync();
  }
}

// ---- launching (instantiated once per arithmetic type) ----
template <typename R>
const void *pick_kernel(int BR, int BC, bool window, int sync, bool hass) {
#define BI_BLK_W(A, B, S) \
  (hass ? (const void *)bi_block_window_kernel<R, A, B, S, true> : (const void *)bi_block_window_kernel<R, A, B, S, false>)
#define BI_BLK(A, B)                                                                                       \
  if (BR == A && BC == B) {                                                                                \
    if (window) return sync == SYNC_WARP ? BI_BLK_W(A, B, SYNC_WARP) : sync == SYNC_CTA ? BI_BLK_W(A, B, SYNC_CTA) : BI_BLK_W(A, B, SYNC_NAMED); \
    if (sync == SYNC_WARP) return (const void *)bi_block_filter_kernel<R, A, B, SYNC_WARP, false>;         \
    return hass ? (const void *)bi_block_filter_kernel<R, A, B, SYNC_CTA, true> : (const void *)bi_block_filter_kernel<R, A, B, SYNC_CTA, false>; \
  }
  BI_BLK(4, 4)
  BI_BLK(8, 4)
  BI_BLK(8, 6)
#undef BI_BLK
#undef BI_BLK_W
  return nullptr;
}

}  // namespace bi_block
