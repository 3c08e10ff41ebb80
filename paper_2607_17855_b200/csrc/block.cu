// Planner and launcher of the block kernels (block.cuh).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "bi_device.cuh"
#include "block.h"

const void *bi_block_kernel_f64(int BR, int BC, bool window, int sync, bool hass);
const void *bi_block_kernel_f32(int BR, int BC, bool window, int sync, bool hass);

using namespace bi_block;

namespace {

int ceil_div(int a, int b) { return (a + b - 1) / b; }
int pow2_ceil(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Which axes of a group are a block's rows and columns (indices into BiGroup::axis), and the block counts.
struct Cut {
  int row, col, pre[2], npre_axes;   // pre: remaining axes, in packed order
  int nrb, ncb, npre, nb;
};
Cut cut_group(const BiGroup &g, int BR, int BC) {
  Cut best;
  memset(&best, 0, sizeof(best));
  best.nb = 1 << 30;
  for (int r = 0; r < g.rank; ++r)
    for (int c = 0; c < g.rank; ++c) {
      if (r == c) continue;
      Cut k;
      memset(&k, 0, sizeof(k));
      k.row = r; k.col = c;
      k.nrb = ceil_div(g.dim[r], BR); k.ncb = ceil_div(g.dim[c], BC);
      k.npre = 1;
      for (int j = 0; j < g.rank; ++j)
        if (j != r && j != c) { k.pre[k.npre_axes++] = j; k.npre *= g.dim[j]; }
      k.nb = k.nrb * k.ncb * k.npre;
      if (k.nb < best.nb) best = k;
    }
  return best;
}

struct Shape { int BR, BC; };
const Shape kShapes[] = {{4, 4}, {8, 4}, {8, 6}};

}  // namespace

// ---- packing: a modality's slices in block order ----
struct PackBlk {
  const float *src;
  void *dst;
  int64_t total;
  int32_t P, nb, npre, ncb, BR, BC, VE, nrow, ncol, npre1;
  int64_t srow, scol, spre0, spre1;
};
template <typename R>
__global__ void bi_pack_block_kernel(PackBlk p) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= p.total) return;
  const int per = p.nb * p.BR * p.BC;
  const int64_t go = e / per;
  const int idx = (int)(e - go * per);
  const int v = idx / (p.nb * p.VE), rest = idx - v * p.nb * p.VE, b = rest / p.VE, el = v * p.VE + rest % p.VE;
  const int pre = b % p.npre, rc = b / p.npre, rb = rc / p.ncb, cb = rc - rb * p.ncb;
  const int i = rb * p.BR + el / p.BC, j = cb * p.BC + el % p.BC;
  R out = (R)0;
  if (i < p.nrow && j < p.ncol) {
    const int p0 = pre / p.npre1, p1 = pre - p0 * p.npre1;
    const float x = p.src[go * p.P + i * p.srow + j * p.scol + p0 * p.spre0 + p1 * p.spre1];
    out = (R)log(fmax((double)x, 1e-16));
  }
  ((R *)p.dst)[e] = out;
}
__global__ void bi_exp_table_kernel(double *tab) { bi_fast_tabs_compute(tab, threadIdx.x, blockDim.x); }

// Whether the handle keeps a block-ordered copy of any slice.
bool bi_block_copies(const bi_model *md) {
  for (int gi = 0; gi < md->h.ngroups; ++gi)
    if (bi_block_slice_elems(md, gi)) return true;
  return false;
}

// Elements of one outcome's slice of group gi in block order (0: the model has no block plan).
int bi_block_slice_elems(const bi_model *md, int gi) {
  if (!md->blk_BR || md->h.grp[gi].rank < 2) return 0;
  const Cut k = cut_group(md->h.grp[gi], md->blk_BR, md->blk_BC);
  return k.nb * md->blk_BR * md->blk_BC;
}

// Block shape of a model (0, 0: none).  Decided from the groups alone, because the slices are laid out for
// it once: the smallest block under which a filtering unit is a single warp (no block barriers), else 8 x 6,
// which has the fewest partial messages per entry that the register file allows.
void bi_block_choose_shape(bi_model *md) {
  md->blk_BR = md->blk_BC = 0;
  for (int gi = 0; gi < md->h.ngroups; ++gi)
    if (md->h.grp[gi].rank > kMaxRank) return;
  for (const Shape &s : kShapes) {
    int nb = 0;
    for (int gi = 0; gi < md->h.ngroups; ++gi)
      if (md->h.grp[gi].rank >= 2) nb += cut_group(md->h.grp[gi], s.BR, s.BC).nb;
    md->blk_BR = s.BR; md->blk_BC = s.BC;
    if (nb <= 32) break;
  }
}

// The block-ordered copy of one modality: sstride[j] is the source stride of the group's axis j, P the
// entries of a source slice.  Returns the packing job's element count per outcome.
int bi_block_pack_member(const bi_model *md, int gi, const float *src, int m, const int64_t *sstride, int P, void *dst,
                         cudaStream_t stream) {
  const BiGroup &g = md->h.grp[gi];
  const Cut k = cut_group(g, md->blk_BR, md->blk_BC);
  PackBlk q;
  memset(&q, 0, sizeof(q));
  q.src = src; q.dst = dst; q.P = P;
  q.nb = k.nb; q.npre = k.npre; q.ncb = k.ncb; q.BR = md->blk_BR; q.BC = md->blk_BC;
  q.VE = md->arith == BI_ARITH_F64 ? 2 : 4;
  q.nrow = g.dim[k.row]; q.ncol = g.dim[k.col];
  q.npre1 = k.npre_axes > 1 ? g.dim[k.pre[1]] : 1;
  q.srow = sstride[k.row]; q.scol = sstride[k.col];
  q.spre0 = k.npre_axes > 0 ? sstride[k.pre[0]] : 0;
  q.spre1 = k.npre_axes > 1 ? sstride[k.pre[1]] : 0;
  q.total = (int64_t)md->h.G * m * k.nb * q.BR * q.BC;
  const unsigned blocks = (unsigned)((q.total + 255) / 256);
  if (md->arith == BI_ARITH_F64) bi_pack_block_kernel<double><<<blocks, 256, 0, stream>>>(q);
  else bi_pack_block_kernel<float><<<blocks, 256, 0, stream>>>(q);
  return cudaGetLastError() == cudaSuccess ? BI_OK : BI_ERR_CUDA;
}

namespace {

// ---- the plan of one call kind ----
struct HostPlan {
  Plan p;
  std::vector<Desc> desc;
  std::vector<Lane> lane[kMaxVariants];
  std::vector<Pass> pass[kMaxVariants];
};

struct Run {           // a factor's message entries
  int kg, kp, kf;      // entries per state: groups, edge in, edge out
  int rows;            // states allocated (padded rows and columns of blocks are written too)
  int y0, cs;          // first entry, entries per state
  int op, of;          // starts of the edges' runs within a state
};

// Which lanes of the finishing phase complete which states, for a team of NW warps: a factor's states side by
// side in one warp, several factors to a pass where they fit, several lanes per state where the warps have
// room for it (the longest runs first).
struct LanePack {
  int npass, g[BI_MAX_F], pass_of[BI_MAX_F], lane_of[BI_MAX_F];
  std::vector<Pass> passes;
};
int up2(int x) { return (x + 1) & ~1; }
void pack_lanes(const BiDev &h, const Run *run, int ve, int NW, LanePack &lp) {
  const int F = h.F;
  for (int f = 0; f < F; ++f) lp.g[f] = 1;
  auto pack = [&]() {   // by decreasing lanes per state: every start is a multiple of it (n g lanes each)
    std::vector<int> order(F), used;
    for (int f = 0; f < F; ++f) order[f] = f;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return lp.g[a] != lp.g[b] ? lp.g[a] > lp.g[b] : h.n[a] > h.n[b]; });
    for (int f : order) {
      const int need = h.n[f] * lp.g[f];
      size_t k = 0;
      while (k < used.size() && used[k] + need > 32) ++k;
      if (k == used.size()) used.push_back(0);
      lp.pass_of[f] = (int)k;
      lp.lane_of[f] = used[k];
      used[k] += need;
    }
    return (int)used.size();
  };
  const int limit = std::max(NW, pack());
  std::vector<char> stuck(F, 0);
  for (;;) {
    int best = -1;
    double most = 2.0;   // (runs of a few vectors gain nothing from more lanes)
    for (int f = 0; f < F; ++f) {
      const double len = (double)(run[f].kg + run[f].kp + run[f].kf) / ve / lp.g[f];
      if (!stuck[f] && h.n[f] * lp.g[f] * 2 <= 32 && lp.g[f] < 16 && len > most) { most = len; best = f; }
    }
    if (best < 0) break;
    lp.g[best] *= 2;
    if (pack() > limit) {
      lp.g[best] /= 2;
      stuck[best] = 1;
    }
  }
  lp.npass = pack();
  lp.passes.assign(lp.npass, Pass{1, 0, 0, 0});
  for (int f = 0; f < F; ++f) {
    Pass &ps = lp.passes[lp.pass_of[f]];
    auto vecs = [&](int k) { return ceil_div(ceil_div(k, ve), lp.g[f]); };
    ps.gmax = std::max(ps.gmax, lp.g[f]);
    ps.nz = std::max(ps.nz, std::max(2, pow2_ceil((h.n[f] + 1) / 2)));
    ps.nvec = std::max(ps.nvec, up2(vecs(run[f].kg)));
    ps.nedge = std::max(ps.nedge, up2(std::max(vecs(run[f].kp), vecs(run[f].kf))));
  }
}
void build_lanes(const BiDev &h, const Plan &p, const Run *run, const int *e0, int ve, const LanePack &lp, std::vector<Lane> &lanes) {
  Lane dead;   // an idle lane: the first factor's first state, completed and thrown away
  memset(&dead, 0, sizeof(dead));
  dead.f = -1;
  dead.g = dead.n = 1;
  dead.ya = p.ydead;
  dead.e0 = (int16_t)e0[0];
  dead.qa = (int16_t)p.qo[0];
  lanes.assign((size_t)lp.npass * 32, dead);
  for (int f = 0; f < h.F; ++f)
    for (int i = 0; i < h.n[f] * lp.g[f]; ++i) {
      const int s = i / lp.g[f], q = i % lp.g[f];
      Lane &l = lanes[(size_t)lp.pass_of[f] * 32 + lp.lane_of[f] + i];
      l.f = (int16_t)f; l.s = (int16_t)s; l.p = (int16_t)q; l.g = (int16_t)lp.g[f]; l.n = (int16_t)h.n[f];
      l.ya = run[f].y0 + s * run[f].cs + q * ve;
      l.op = (int16_t)run[f].op;
      l.of = (int16_t)run[f].of;
      l.qa = (int16_t)(p.qo[f] + s);
      l.e0 = (int16_t)e0[f];
      l.out = h.off[f] + s;
    }
}

// window: also the edges' transitions
bool build_plan(const bi_model *md, bool window, HostPlan &hp) {
  const BiDev &h = md->h;
  const int BR = md->blk_BR, BC = md->blk_BC, F = h.F, ve = md->arith == BI_ARITH_F64 ? 2 : 4;
  Plan &p = hp.p;
  memset(&p, 0, sizeof(p));
  if (!BR) return false;
  p.BR = BR; p.BC = BC;
  p.max_th = max_threads(BR * BC * 4 / ve);
  std::vector<Cut> cut(h.ngroups);
  int rowsp[BI_MAX_F];
  for (int f = 0; f < F; ++f) rowsp[f] = h.n[f];
  auto as_rows = [&](int f) { rowsp[f] = std::max(rowsp[f], ceil_div(h.n[f], BR) * BR); };
  auto as_cols = [&](int f) { rowsp[f] = std::max(rowsp[f], ceil_div(h.n[f], BC) * BC); };
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank > kMaxRank) return false;
    if (g.rank < 2) continue;
    cut[gi] = cut_group(g, BR, BC);
    as_rows(g.axis[cut[gi].row]);
    as_cols(g.axis[cut[gi].col]);
    p.g_nb[gi] = cut[gi].nb;
  }
  if (window) {
    for (int f = 0; f < F; ++f) {
      if (!h.has_bdep) { as_rows(f); as_cols(f); continue; }
      const int k = h.bdep_len[f];
      if (k > 3) return false;
      as_rows(f);
      for (int j = 0; j < k; ++j) { as_rows(h.bdep[f][j]); as_cols(h.bdep[f][j]); }
    }
  }
  int o = 0;
  for (int f = 0; f < F; ++f) {
    p.qo[f] = o;
    o += (rowsp[f] + 3) & ~3;
  }
  p.one = o;
  p.SQ = (o + 1 + 3) & ~3;
  // ---- pass 1: entries per state; pass 2: the blocks with their addresses
  Run run[BI_MAX_F];
  memset(run, 0, sizeof(run));
  LanePack lp[kMaxVariants];
  int e0[BI_MAX_F] = {}, nedge_blocks = 0;
  for (int pass = 0; pass < 2; ++pass) {
    int kg[BI_MAX_F] = {}, kp[BI_MAX_F] = {}, kf[BI_MAX_F] = {};   // entries used so far
    auto entry = [&](int f, int s, int k) { return run[f].y0 + s * run[f].cs + k; };
    for (int gi = 0; gi < h.ngroups; ++gi) {
      const BiGroup &g = h.grp[gi];
      if (g.rank < 2) continue;
      const Cut &c = cut[gi];
      const int fr = g.axis[c.row], fc = g.axis[c.col];
      const int f0 = c.npre_axes > 0 ? g.axis[c.pre[0]] : -1, f1 = c.npre_axes > 1 ? g.axis[c.pre[1]] : -1;
      const int n0 = f0 >= 0 ? h.n[f0] : 1, n1 = f1 >= 0 ? h.n[f1] : 1;
      if (pass == 1)
        for (int b = 0; b < c.nb; ++b) {
          const int pre = b % c.npre, rc = b / c.npre, rb = rc / c.ncb, cb = rc % c.ncb, d0 = pre / n1, d1 = pre % n1;
          Desc d;
          memset(&d, 0, sizeof(d));
          d.yv = d.yw = d.yu0 = d.yu1 = p.ydump;
          d.qr = (int16_t)(p.qo[fr] + rb * BR);
          d.qc = (int16_t)(p.qo[fc] + cb * BC);
          d.q0 = (int16_t)(f0 >= 0 ? p.qo[f0] + d0 : p.one);
          d.q1 = (int16_t)(f1 >= 0 ? p.qo[f1] + d1 : p.one);
          d.kind = KIND_V | KIND_W;
          d.yv = entry(fr, rb * BR, kg[fr] + cb * c.npre + pre);
          d.sv = (int16_t)run[fr].cs;
          d.yw = entry(fc, cb * BC, kg[fc] + rb * c.npre + pre);
          d.sw = (int16_t)run[fc].cs;
          if (f0 >= 0) {   // u times the other prefix factor's belief
            d.kind |= KIND_U0;
            d.yu0 = entry(f0, d0, kg[f0] + (rb * c.ncb + cb) * n1 + d1);
          }
          if (f1 >= 0) {
            d.kind |= KIND_U1;
            d.yu1 = entry(f1, d1, kg[f1] + (rb * c.ncb + cb) * n0 + d0);
          }
          d.grp = gi; d.base = b;
          hp.desc.push_back(d);
        }
      kg[fr] += c.ncb * c.npre;
      kg[fc] += c.nrb * c.npre;
      if (f0 >= 0) kg[f0] += c.nrb * c.ncb * n1;
      if (f1 >= 0) kg[f1] += c.nrb * c.ncb * n0;
    }
    for (int f = 0; f < F && window; ++f) {
      const int n = h.n[f];
      if (!h.has_bdep) {
        if (n == 1) continue;
        const int nrb = ceil_div(n, BR), ncb = ceil_div(n, BC);
        for (int dir = 0; dir < 2; ++dir) {
          const int k0 = dir == 0 ? run[f].op + kp[f] : run[f].of + kf[f];
          if (pass == 1)
            for (int b = 0; b < nrb * ncb; ++b) {
              const int rb = b / ncb, cb = b % ncb;
              Desc d;
              memset(&d, 0, sizeof(d));
              d.yv = d.yw = d.yu0 = d.yu1 = p.ydump;
              d.qr = (int16_t)((dir == 0 ? -p.SQ : p.SQ) + p.qo[f] + rb * BR);
              d.q0 = d.q1 = (int16_t)p.one;
              d.kind = KIND_W | (dir == 0 ? KIND_PAST : KIND_FUT);
              d.yw = entry(f, cb * BC, k0 + rb);
              d.sw = (int16_t)run[f].cs;
              d.grp = f; d.base = rb * BR * h.npad[f] + cb * BC;
              d.rs = h.npad[f]; d.cs = 1;
              d.rlim = (int16_t)std::min(BR, n - rb * BR);
              d.clim = (int16_t)std::min(BC, n - cb * BC);
              hp.desc.push_back(d);
            }
          (dir == 0 ? kp[f] : kf[f]) += nrb;
          if (pass == 0) nedge_blocks += nrb * ncb;
        }
        continue;
      }
      // transitions over several parents: the tensor [n][parents, last fastest]
      const int k = h.bdep_len[f], *par = h.bdep[f], PB = h.PB[f];
      int str[3] = {1, 1, 1};
      for (int j = k - 2; j >= 0; --j) str[j] = str[j + 1] * h.n[par[j + 1]];
      {   // edge in: rows = own states, columns = the last parent, prefix = the others (all at the step before)
        const int fc = par[k - 1], nrb = ceil_div(n, BR), ncb = ceil_div(h.n[fc], BC);
        const int n0 = k > 1 ? h.n[par[0]] : 1, n1 = k > 2 ? h.n[par[1]] : 1, npre = n0 * n1;
        if (pass == 1)
          for (int b = 0; b < nrb * ncb * npre; ++b) {
            const int pre = b % npre, rc = b / npre, rb = rc / ncb, cb = rc % ncb, d0 = pre / n1, d1 = pre % n1;
            Desc d;
            memset(&d, 0, sizeof(d));
            d.yv = d.yw = d.yu0 = d.yu1 = p.ydump;
            d.qr = (int16_t)(p.qo[f] + rb * BR);
            d.qc = (int16_t)(-p.SQ + p.qo[fc] + cb * BC);
            d.q0 = (int16_t)(k > 1 ? -p.SQ + p.qo[par[0]] + d0 : p.one);
            d.q1 = (int16_t)(k > 2 ? -p.SQ + p.qo[par[1]] + d1 : p.one);
            d.kind = KIND_V | KIND_PAST;
            d.yv = entry(f, rb * BR, run[f].op + kp[f] + cb * npre + pre);
            d.sv = (int16_t)run[f].cs;
            d.grp = f;
            d.base = rb * BR * PB + cb * BC + (k > 1 ? d0 * str[0] : 0) + (k > 2 ? d1 * str[1] : 0);
            d.rs = PB; d.cs = 1;
            d.rlim = (int16_t)std::min(BR, n - rb * BR);
            d.clim = (int16_t)std::min(BC, h.n[fc] - cb * BC);
            hp.desc.push_back(d);
          }
        kp[f] += ncb * npre;
        if (pass == 0) nedge_blocks += nrb * ncb * npre;
      }
      if (k == 1) {   // edge out, one parent: rows = the child's next states, columns = the parent
        const int fc = par[0], nrb = ceil_div(n, BR), ncb = ceil_div(h.n[fc], BC);
        if (pass == 1)
          for (int b = 0; b < nrb * ncb; ++b) {
            const int rb = b / ncb, cb = b % ncb;
            Desc d;
            memset(&d, 0, sizeof(d));
            d.yv = d.yw = d.yu0 = d.yu1 = p.ydump;
            d.qr = (int16_t)(p.SQ + p.qo[f] + rb * BR);
            d.q0 = d.q1 = (int16_t)p.one;
            d.kind = KIND_W | KIND_FUT;
            d.yw = entry(fc, cb * BC, run[fc].of + kf[fc] + rb);
            d.sw = (int16_t)run[fc].cs;
            d.grp = f; d.base = rb * BR * PB + cb * BC;
            d.rs = PB; d.cs = 1;
            d.rlim = (int16_t)std::min(BR, n - rb * BR);
            d.clim = (int16_t)std::min(BC, h.n[fc] - cb * BC);
            hp.desc.push_back(d);
          }
        kf[fc] += nrb;
        if (pass == 0) nedge_blocks += nrb * ncb;
      } else {        // two or three: prefix = the child's next state (and the first of three parents), rows and columns = the last two
        const int fr = par[k - 2], fc = par[k - 1], f1 = k > 2 ? par[0] : -1;
        const int nrb = ceil_div(h.n[fr], BR), ncb = ceil_div(h.n[fc], BC), n1 = f1 >= 0 ? h.n[f1] : 1, npre = n * n1;
        if (pass == 1)
          for (int b = 0; b < nrb * ncb * npre; ++b) {
            const int pre = b % npre, rc = b / npre, rb = rc / ncb, cb = rc % ncb, sn = pre / n1, d1 = pre % n1;
            Desc d;
            memset(&d, 0, sizeof(d));
            d.yv = d.yw = d.yu0 = d.yu1 = p.ydump;
            d.qr = (int16_t)(p.qo[fr] + rb * BR);
            d.qc = (int16_t)(p.qo[fc] + cb * BC);
            d.q0 = (int16_t)(p.SQ + p.qo[f] + sn);
            d.q1 = (int16_t)(f1 >= 0 ? p.qo[f1] + d1 : p.one);
            d.kind = KIND_V | KIND_W | KIND_FUT | (f1 >= 0 ? KIND_U1 : 0);
            d.yv = entry(fr, rb * BR, run[fr].of + kf[fr] + cb * npre + pre);
            d.sv = (int16_t)run[fr].cs;
            d.yw = entry(fc, cb * BC, run[fc].of + kf[fc] + rb * npre + pre);
            d.sw = (int16_t)run[fc].cs;
            if (f1 >= 0) d.yu1 = entry(f1, d1, run[f1].of + kf[f1] + (rb * ncb + cb) * n + sn);
            d.grp = f;
            d.base = sn * PB + rb * BR * str[k - 2] + cb * BC + (k > 2 ? d1 * str[0] : 0);
            d.rs = str[k - 2]; d.cs = 1;
            d.rlim = (int16_t)std::min(BR, h.n[fr] - rb * BR);
            d.clim = (int16_t)std::min(BC, h.n[fc] - cb * BC);
            hp.desc.push_back(d);
          }
        kf[fr] += ncb * npre;
        kf[fc] += nrb * npre;
        if (f1 >= 0) kf[f1] += nrb * ncb * n;
        if (pass == 0) nedge_blocks += nrb * ncb * npre;
      }
    }
    if (pass == 0) {
      // team sizes: a thread per block, in window calls also those under which 2, 3, 4, 6 or 12 steps share a CTA
      int NB = 0;
      for (int gi = 0; gi < h.ngroups; ++gi) NB += p.g_nb[gi];
      NB += nedge_blocks;
      // (and, where that is more than a thread per block, a warp for each pass of the finishing phase)
      const int full = std::max(32, (NB + 31) / 32 * 32);
      for (int f = 0; f < F; ++f) { run[f].kg = kg[f]; run[f].kp = kp[f]; run[f].kf = kf[f]; }
      LanePack one;
      pack_lanes(h, run, ve, 1, one);
      const int wide = std::max(full, 32 * one.npass);
      for (int uc : {1, 2, 3, 4, 6, 12})
        for (int want : {full, wide}) {
          if (!window && uc > 4) continue;   // (filtering: teams of which up to four share an SM)
          const int LT = std::min(want, p.max_th / uc / 32 * 32);
          bool have = LT < 32 || p.nv == kMaxVariants;
          for (int v = 0; v < p.nv; ++v) have = have || p.var[v].LT == LT;
          if (have) continue;
          Variant &v = p.var[p.nv];
          v.LT = LT;
          v.nbpt = ceil_div(std::max(NB, 1), LT);
          pack_lanes(h, run, ve, LT / 32, lp[p.nv]);
          v.npass = lp[p.nv].npass;
          p.nv += 1;
        }
      // runs of whole 16-byte vectors, zero-padded to what the longest lane of the same pass reads (under
      // every team size); an odd number of vectors between states: consecutive states on different banks
      int y = 0;
      for (int f = 0; f < F; ++f) {
        int lg = 0, le = 0, lz = 0;
        for (int v = 0; v < p.nv; ++v) {
          const Pass &ps = lp[v].passes[lp[v].pass_of[f]];
          lg = std::max(lg, ps.nvec * lp[v].g[f]);
          le = std::max(le, ps.nedge * lp[v].g[f]);
          lz = std::max(lz, ps.nz);
        }
        run[f].rows = rowsp[f];
        run[f].op = lg * ve;
        run[f].of = (lg + le) * ve;
        // entries between states: the padding under which the lanes of a quarter-warp hit distinct banks most
        const int need = lg + (window ? 2 * le : 0);
        int cs = need, least = 1 << 30;
        for (int c = std::max(need, 1); c < need + 9; ++c) {
          int cost = c - need;
          for (int v = 0; v < p.nv; ++v) {
            const int g = lp[v].g[f];
            for (int l0 = 0; l0 < h.n[f] * g; l0 += 8) {
              int hits[8] = {}, most = 0;
              for (int l = l0; l < std::min(l0 + 8, h.n[f] * g); ++l) most = std::max(most, ++hits[(l / g * c + l % g) & 7]);
              cost += 16 * (most - 1);
            }
          }
          if (cost < least) { least = cost; cs = c; }
        }
        run[f].cs = cs * ve;
        if (run[f].cs > 16000 || y / ve > 60000) return false;
        run[f].y0 = y;
        y += run[f].rows * run[f].cs;
        e0[f] = p.Esz;
        p.Esz += 2 * lz;
      }
      // (an idle lane reads what any lane may read, from an area of zeros)
      p.ydead = y;
      int most = 0;
      for (int v = 0; v < p.nv; ++v)
        for (const Pass &ps : lp[v].passes) most = std::max(most, std::max(ps.nvec, ps.nedge));
      y += most * ve;
      p.ydump = y;   // (results that a block does not have)
      y += ve;
      for (int v = 0; v < p.nv; ++v)   // (and of the exchange area, from the first factor's entry on)
        for (const Pass &ps : lp[v].passes) p.Esz = std::max(p.Esz, 2 * ps.nz);
      p.Ysz = (y + 3) & ~3;
    }
  }
  p.NB = (int)hp.desc.size();
  {   // the entry of threads without a block
    Desc d;
    memset(&d, 0, sizeof(d));
    d.q0 = d.q1 = (int16_t)p.one;
    d.yv = d.yw = d.yu0 = d.yu1 = p.ydump;
    hp.desc.push_back(d);
  }
  for (int v = 0; v < p.nv; ++v) {
    build_lanes(h, p, run, e0, ve, lp[v], hp.lane[v]);
    hp.pass[v] = lp[v].passes;
  }
  p.ok = p.nv > 0;
  return p.ok != 0;
}

}  // namespace

namespace {

void use_variant(const Variant &v, Params &p) {
  p.lane = v.lane; p.pass = v.pass; p.npass = v.npass; p.LT = v.LT; p.nbpt = v.nbpt;
}

// shared-memory layout for `units` teams and `slots` belief slots (behind the exponential table); returns bytes
size_t layout(const Plan &pl, Params &p, int esz, int units, int slots) {
  auto up16 = [](int x) { return (x + 15) & ~15; };
  int u = up16(pl.Ysz * esz);
  p.o_cst = u; u += pl.SQ * 8;
  p.o_xp = u; u += p.lambda != 1.0 ? pl.SQ * 8 : 0;
  p.o_e = u; u += pl.Esz * 8;
  p.unit_sz = u;
  size_t o = (512 + (p.mmp ? 256 : 0)) * sizeof(double);
  p.o_unit = (int)o; o += (size_t)units * p.unit_sz;
  p.o_q = (int)o; o += (size_t)slots * pl.SQ * esz;
  p.o_par = (int)o; o += (size_t)p.W * up16(p.wpar * esz);
  // the blocks beyond a thread each: whole rounds of the team, the last one only as far as it goes
  const int extra = p.nbpt > 1 ? (pl.NB - p.LT + 31) / 32 * 32 : 0;
  p.extra = extra;
  p.o_L = (int)o; o += (size_t)units * extra * pl.BR * pl.BC * esz;
  p.o_ref = (int)o; o += (size_t)extra * 48;
  p.o_lane = (int)o; o += (size_t)p.npass * 33 * 16;
  return o;
}

// Whether one unit of a plan fits an SM under some team size (filtering one agent, a window of one step).
bool smallest_fits(const bi_model *md, const Plan &pl, bool window) {
  if (pl.NB == 0) return false;
  Params p;
  memset(&p, 0, sizeof(p));
  p.lambda = 1.0;
  p.W = window ? 0 : 1;
  for (int f = 0; f < md->h.F && md->h.has_bdep && !window; ++f) p.wpar = std::max(p.wpar, (md->h.PB[f] + 3) & ~3);
  for (int v = 0; v < pl.nv; ++v) {
    use_variant(pl.var[v], p);
    if (layout(pl, p, md->arith == BI_ARITH_F64 ? 8 : 4, 1, window ? 6 : 1) <= (size_t)md->max_smem_optin - 1024) return true;
  }
  return false;
}

}  // namespace

// Builds the filtering and the window plan of a model (those that some call can run: a plan whose smallest call does
// not fit an SM, and a plan for calls that the pair kernels take ahead of these, are not kept, and a model without
// plans has no block shape and so no copies of its slices) and appends their tables to the upload buffer; the
// device pointers in the plans are offsets until bi_block_bind turns them into addresses.
void bi_block_build(bi_model *md, std::vector<unsigned char> &blob) {
  auto put = [&](const void *src, size_t bytes) {
    const size_t at = (blob.size() + 15) & ~(size_t)15;
    blob.resize(at + bytes);
    memcpy(blob.data() + at, src, bytes);
    return (uintptr_t)at;
  };
  md->blk_plan[0] = md->blk_plan[1] = nullptr;
  for (int k = 0; k < 2; ++k) {
    HostPlan hp;
    if (md->arith == BI_ARITH_F64 && md->test_family == BI_FAMILY_ANY && (k == 0 ? md->pair_ok : bi_pair_window_always(md))) continue;
    if (!build_plan(md, k == 1, hp) || !smallest_fits(md, hp.p, k == 1)) continue;
    hp.p.desc = reinterpret_cast<const Desc *>(put(hp.desc.data(), hp.desc.size() * sizeof(Desc)));
    for (int v = 0; v < hp.p.nv; ++v) {
      hp.p.var[v].lane = reinterpret_cast<const Lane *>(put(hp.lane[v].data(), hp.lane[v].size() * sizeof(Lane)));
      hp.p.var[v].pass = reinterpret_cast<const Pass *>(put(hp.pass[v].data(), hp.pass[v].size() * sizeof(Pass)));
    }
    md->blk_plan[k] = new Plan(hp.p);
  }
  if (!md->blk_plan[0] && !md->blk_plan[1]) md->blk_BR = md->blk_BC = 0;
}
void bi_block_bind(bi_model *md, unsigned char *dev) {
  for (int k = 0; k < 2; ++k) {
    Plan *p = static_cast<Plan *>(md->blk_plan[k]);
    if (!p) continue;
    p->desc = reinterpret_cast<const Desc *>(dev + reinterpret_cast<uintptr_t>(p->desc));
    for (int v = 0; v < p->nv; ++v) {
      p->var[v].lane = reinterpret_cast<const Lane *>(dev + reinterpret_cast<uintptr_t>(p->var[v].lane));
      p->var[v].pass = reinterpret_cast<const Pass *>(dev + reinterpret_cast<uintptr_t>(p->var[v].pass));
    }
  }
}
void bi_block_free(bi_model *md) {
  for (int k = 0; k < 2; ++k) {
    delete static_cast<Plan *>(md->blk_plan[k]);
    md->blk_plan[k] = nullptr;
  }
}
int bi_block_exp_table(double *dst, cudaStream_t stream) {
  bi_exp_table_kernel<<<1, 512, 0, stream>>>(dst);
  return cudaGetLastError() == cudaSuccess ? BI_OK : BI_ERR_CUDA;
}

namespace {

void fill_params(const BiCall &c, const Plan &pl, Params &p) {
  const bi_model *md = c.model;
  const BiDev &h = md->h;
  memset(&p, 0, sizeof(p));
  const bool window = c.algo != BI_ALGO_FILTER;
  p.desc = pl.desc;
  p.NB = pl.NB; p.SQ = pl.SQ; p.one = pl.one; p.Ysz = pl.Ysz; p.Esz = pl.Esz;
  p.N = c.N; p.T = c.T; p.K = c.K; p.F = h.F; p.M = h.M; p.S = h.S; p.G = h.G;
  p.mmp = c.algo == BI_ALGO_MMP;
  p.has_bdep = h.has_bdep;
  p.lambda = c.lambda;
  // No softmax shift in float64: with probabilities in A and B none of the terms of a logit is below ln 1e-16,
  // 53.2 binary orders below zero.  They are one per modality, the prior or past message and the future message; with
  // several parents per transition a future message from every factor whose transition reads this one.
  // Beyond seventeen of them, or with the caller's own weights or starting beliefs (used as given), every
  // segment shifts by its own maximum (a model with entries above 1 is marked in status[1]).
  int terms = h.M + 3;
  if (window && h.has_bdep) {
    int readers[BI_MAX_F] = {};
    for (int f = 0; f < h.F; ++f)
      for (int j = 0; j < h.bdep_len[f]; ++j) terms = std::max(terms, h.M + 1 + ++readers[h.bdep[f][j]]);
  }
  p.common = !md->soft_shadow && !(c.q_init && c.lambda != 1.0) && terms * 54 < 960;
  for (int f = 0; f < h.F; ++f) {
    p.n[f] = h.n[f]; p.off[f] = h.off[f]; p.qo[f] = pl.qo[f]; p.npad[f] = h.npad[f]; p.U[f] = h.U[f];
    p.logD[f] = h.logD[f];
    p.n_max = std::max(p.n_max, (int)h.n[f]);
    p.Dstride[f] = h.Dstride[f];
    p.Bstride[f] = h.Bstride[f];
    if (h.has_bdep) {
      p.bdep_len[f] = h.bdep_len[f];
      for (int j = 0; j < h.bdep_len[f]; ++j) p.bdep[f][j] = h.bdep[f][j];
      p.PB[f] = h.PB[f];
      p.Bfull[f] = h.Bfull[f];
      p.Bfull_stride[f] = h.Bfull_stride[f];
      p.Mp[f] = h.logBfull[f];
      p.wpar = std::max(p.wpar, (h.PB[f] + 3) & ~3);
    } else if (window) {
      if (h.n[f] == 1) p.ones |= 1u << f;
      p.Mp[f] = c.algo == BI_ALGO_VMP ? h.logBt[f] : h.BfT[f];     // [previous][next]
      p.Mf[f] = c.algo == BI_ALGO_VMP ? h.logB[f] : h.BdagT[f];    // [next][previous]
    } else {
      p.Mp[f] = h.BfT[f];
    }
  }
  int n1 = 0;
  for (int f = 0; f < h.F; ++f) {
    p.r1_begin[f] = n1;
    for (int gi = 0; gi < h.ngroups; ++gi) {
      const BiGroup &gr = h.grp[gi];
      if (gr.rank != 1 || gr.axis[0] != f) continue;
      for (int mi = gr.mem_begin; mi < gr.mem_end; ++mi) {
        const BiMember &mm = h.mem[mi];
        p.r1_mod[n1] = mm.modality; p.r1_m[n1] = mm.m; p.r1_P[n1] = mm.P_pad;
        p.r1_logA[n1] = mm.logA; p.r1_gstride[n1] = mm.gstride;
        ++n1;
      }
    }
  }
  p.r1_begin[h.F] = n1;
  for (int gi = 0; gi < h.ngroups; ++gi) {
    p.g_nb[gi] = pl.g_nb[gi];
    p.g_beg[gi] = h.grp[gi].mem_begin;
    p.g_beg[gi + 1] = h.grp[gi].mem_end;
    if (h.grp[gi].rank >= 2) p.g_any = gi;
    if (h.grp[gi].rank >= 2) p.max_mem = std::max(p.max_mem, h.grp[gi].mem_end - h.grp[gi].mem_begin);
    for (int mi = h.grp[gi].mem_begin; mi < h.grp[gi].mem_end; ++mi) {
      p.m_mod[mi] = h.mem[mi].modality;
      p.m_m[mi] = h.mem[mi].m;
      p.m_blk[mi] = h.mem[mi].logA_blk;
    }
  }
  p.exp_tab = md->exp_tab;
  p.obs = c.obs; p.act = c.act; p.act_prev = c.act_prev;
  p.q_prev = c.q_prev; p.q_init = c.q_init; p.carry_in = c.carry_in; p.carry_out = c.carry_out; p.lnprior = c.lnprior;
  p.q_out = c.q_out; p.logq_out = c.logq_out; p.argmax_out = c.argmax_out; p.status = h.status;
}

}  // namespace

// A model with zeros in A amplifies a rounding by up to 1e9 within sixteen iterations, and a trajectory carries
// the result on from step to step: in float32, and in filtering, another order of summation gives other beliefs
// (measured: one in five such trajectories differs in the first digit from the CTA kernel's).  Those calls stay
// with the kernels that have served them, bit for bit.  The number of steps has no say in it: a trajectory
// filtered in blocks of steps is the single call's (bi_filter_continue), and a stream of ticks is a trajectory too.
// (It costs such ticks: 26 agents on [5,12,12,3], 68 us there and 24 us here.)
// Float32 filtering of models coupled in one pair of factors stays as well: several sharp modalities on one pair
// carry float32 roundings to 2e-3 in a belief over thirty steps, and these kernels gain only 1.1 to 1.2 there.
bool bi_block_serves(const bi_model *md, int algo) {
  const bool window = algo != BI_ALGO_FILTER;
  if (!window && md->pair_ok && md->arith == BI_ARITH_F32) return false;
  return md->blk_plan[window ? 1 : 0] && !(md->has_zeros && (md->arith == BI_ARITH_F32 || !window));
}

namespace {

// Microseconds a window call would take here and on the batched kernels (batch_mma.cu, in float32 batch.cu), for the choice
// between them.  Linear in what each spends its time on -- here the launcher's own cost of an iteration (`cycles`, waves
// included), block entries and finishing passes per unit and the preparation of both, there launches, members and slices
// per iteration, slice entries and states per unit -- with coefficients fitted to 960 calls on structures of one to
// five factors, 2 100 to 62 000 units, 6 and 16 iterations (9 and 14 % rms error here, float64 and float32, 15 % there in
// float32, 11 % in float64, see bi_batch_mma_cost).  On 84 further float64 calls the choice (with the pair kernels'
// rule) costs 0.5 % over the fastest of all kernels.  Neither side wins by size alone: [9,32,19] under two rank-2
// slices, float32, 59 508 units, 4463 us here and 2407 us there; [4,6,3] under six slices, float64, 7 360 units, 163 and
// 228 us; [15,6,16] under two, 3 038 units, 113 and 79 us.
struct WindowCost { double block, batch; };
WindowCost window_cost(const BiCall &c, const Plan &pl, const Variant &v, double cycles) {
  const BiDev &h = c.model->h;
  const bool f64 = c.model->arith == BI_ARITH_F64;
  const double per_sm = (double)c.N * c.T / c.model->sm_count * 1e-3, k = c.K * per_sm;   // thousands of units; unit-iterations
  const double ent = pl.NB * (double)(pl.BR * pl.BC) * 1e-3, warps = v.LT / 32.0;
  double slices = 0, states = 0;   // (slices in thousands of entries)
  int members = 0, nmax = 1;
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank < 2) continue;
    double e = 1;
    for (int j = 0; j < g.rank; ++j) e *= j + 1 < g.rank ? g.dim[j] : bi_pad4(g.dim[j]);
    for (int mi = g.mem_begin; mi < g.mem_end; ++mi)
      if (g.dim[g.rank - 1] > 32 || h.mem[mi].m > 4096) return {0.0, 1.0};   // (nothing the batched kernels take)
    slices += e * 1e-3 * (g.mem_end - g.mem_begin);
    members += g.mem_end - g.mem_begin;
  }
  for (int f = 0; f < h.F; ++f) {
    nmax = std::max(nmax, (int)h.n[f]);
    states += h.npad[f];
  }
  const bool lane_per_unit = nmax <= 16 && (double)c.N * c.T * std::min(1.0, h.F / 3.0) >= 64.0 * c.model->sm_count;   // (the update's form, see batch.cu)
  const double mmp = c.algo == BI_ALGO_MMP, launches = members ? 2 : 1;   // (MMP: two logarithms per state)
  WindowCost w;
  w.block = f64 ? 10 + 2.11 * c.K * cycles / 1965 + k * (36 * ent + 1.9 * v.nbpt * warps + 15 * mmp * v.npass) + per_sm * (637 * ent + 142 * warps)
                : 6 + 1.93 * c.K * cycles / 1965 + k * (16 * ent + (15.6 + 9.4 * mmp) * v.npass) + per_sm * (333 * ent + 282 * warps);
  const double mma = bi_batch_mma_cost(c);
  w.batch = f64 ? (mma < 0 ? 2 * w.block : mma)
                : 10 + c.K * (3.4 * launches + 2.3 * members + 2.3 * slices) + k * (36 * slices + states * (0.26 * members + (lane_per_unit ? 1.3 : 5.9) + 0.63 * mmp));
  return w;
}

// Microseconds a step of a filtering call with several parents per transition would take here and on the CTA kernel (a
// step, not the call: a trajectory filtered in blocks of steps has to stay on one kernel).  The prior of a step
// is a contraction of every tensor with its parents' beliefs; a team here may be a single warp where the CTA
// kernel has eight, and with few iterations or small slices that outweighs the faster ones.  Linear in the
// dependent trips of a step (a team alone) and in the work of the teams that share an SM, fitted to 347
// structures, 4 to 2 048 agents (12 and 21 % rms error in cross-validation).  [16,7,19] under three parents,
// 4 agents, six iterations: 2.9 times slower here; [4,6,2,7] under a rank-4 slice, 654 agents: 131 us
// here and 544 us there.
struct FilterCost { double block, cta; };
FilterCost filter_cost(const BiCall &c, const Plan &pl, const Variant &v) {
  const BiDev &h = c.model->h;
  const int NW = v.LT / 32;
  double dots = 0, prods = 0, tensors = 0, slices = 0, rows = 0;
  int groups = 0, deep = 0;
  for (int f = 0; f < h.F; ++f) {
    dots += (double)ceil_div(h.n[f], 4 * NW) * ceil_div(h.PB[f], 8);
    prods += (double)ceil_div(h.PB[f], v.LT) * h.bdep_len[f];
    tensors += (double)h.n[f] * h.PB[f];
    rows += h.n[f];
  }
  for (int gi = 0; gi < h.ngroups; ++gi) {
    const BiGroup &g = h.grp[gi];
    if (g.rank < 2) continue;
    double e = 1;
    for (int j = 0; j < g.rank; ++j) e *= g.dim[j];
    slices += e;
    groups += 1;
    if (g.rank > 2) deep = 1;
  }
  const double beside = std::max(0.0, (double)c.N / c.model->sm_count - 1.0);
  const double ent = pl.NB * (double)(pl.BR * pl.BC) / 32.0 * (c.model->arith == BI_ARITH_F64 ? 1.0 : 0.5);
  FilterCost w;
  w.block = 2.4 + 0.68 * c.K * v.nbpt + 0.061 * dots + 0.052 * prods + 0.74 * h.F + beside * (0.0052 * c.K * ent + 9.1e-5 * tensors);
  w.cta = 1.6 + c.K * (0.43 + 0.29 * groups + 3.4e-4 * slices + 0.66 * deep) + 1.46e-4 * tensors + 1.63 * h.F +
          beside * (c.K * (4.4e-4 * slices + 6.1e-3 * rows + 0.095) + 6.9e-5 * tensors);
  return w;
}

// How a call would run here.
struct Route {
  Params p;
  const Plan *plan;
  unsigned grid, threads;
  size_t bytes;
};

// Whether these kernels take a call, and in which shape.  Any model whose groups span at most four factors
// (transitions over at most three parents in window calls), either arithmetic, as long as a step's blocks fit the
// register file and shared memory of an SM (window calls: of a cluster).
// `estimate`: declines calls that another family is estimated to run faster.
bool choose_route(const BiCall &c, Route &L, bool estimate = true) {
  const bi_model *md = c.model;
  const bool window = c.algo != BI_ALGO_FILTER;
  const Plan *plp = static_cast<const Plan *>(md->blk_plan[window ? 1 : 0]);
  if (!plp || !plp->ok) return false;
  if (window && md->h.has_bdep && (c.algo == BI_ALGO_MMP || c.lnprior)) return false;
  if (!bi_block_serves(md, c.algo)) return false;
  const Plan &pl = *plp;
  L.plan = plp;
  if (pl.NB == 0) return false;   // nothing to contract: the CTA kernel's warp per factor does that
  if (window && !md->h.has_bdep && estimate) {
    const long long units = (long long)c.N * c.T;
    const bool shared = md->h.G == 1 && !md->soft_shadow;
    if (shared && md->batch_unrolled && units >= 4096 && md->arith == BI_ARITH_F32) return false;   // (see batch_unrolled)
    // Models of the agents' own and observation vectors have a slice per unit, which the batched kernels contract in
    // their any-shape form: slower at nearly every size ([10,10,8,6], three groups, 20 480 units: 1246 us here, 1890 us
    // there).  What crosses are large float32 calls without a group over three factors.  With observation
    // vectors, whose softmax is relative to the largest logit: pairs of some size, and no pair at all ([10,10] and
    // [10,8], 4 160 units 182 and 377 us, 20 000 units 821 and 653 us; single factors 91 and 138, 303 and 259 us; but slices
    // of 56 entries in all, 20 000 units, 297 and 349 us).  With models of the agents' own: the pairs
    // first named alone (659 and 625 us; [20,25] and [25,4] 975 and 1323 us).
    if (!shared && md->arith == BI_ARITH_F32 && md->rank2_ok && units >= 16000) {
      double entries = 0;
      for (int gi = 0; gi < md->h.ngroups; ++gi)
        if (md->h.grp[gi].rank >= 2) entries += (double)md->h.grp[gi].P_pad * (md->h.grp[gi].mem_end - md->h.grp[gi].mem_begin);
      const bool crosses = md->soft_shadow ? entries == 0 || entries >= 128 : entries > 0 && md->batch_unrolled;
      if (crosses && entries * 4.0 * (double)units <= 120e6) return false;   // (the batched kernels take no more)
    }
  }
  const int esz = md->arith == BI_ARITH_F64 ? 8 : 4;
  const size_t budget = (size_t)md->max_smem_optin - 1024;
  Params &p = L.p;
  fill_params(c, pl, p);
  if (!window) {
    // Team size: cycles of an iteration (a phase for each round of blocks and of passes), plus what the teams
    // beside it on the SM add, times the waves of teams.  (Five coupled factors, 204 blocks, 256 agents: teams
    // of 224 threads in two waves 486 us, of 192 and 128 side by side 436 and 420 us, of 96 526 us.)
    double best = 1e300;
    int v0 = 0;
    for (int v = 0; v < pl.nv; ++v) {
      use_variant(pl.var[v], p);
      p.W = 1;
      const size_t b = layout(pl, p, esz, 1, 1);
      if (b > budget) continue;
      const int per_sm = std::max(1, std::min((int)((227 * 1024) / (b + 1024)), 65536 / (p.LT * regs_per_thread(pl.BR * pl.BC * esz / 4))));
      const int waves = ceil_div(c.N, per_sm * md->sm_count), on_sm = std::min(per_sm, ceil_div(c.N, md->sm_count));
      const double alone = 900.0 + 900.0 * ceil_div(p.npass, p.LT / 32) + 600.0 * p.nbpt;
      const double beside = pl.NB / 32.0 * pl.BR * pl.BC * 2.6 + 120.0 * p.npass;
      const double t = waves * (alone + (on_sm - 1) * beside);
      if (t < best) { best = t; v0 = v; }
    }
    if (best >= 1e300) return false;
    if (estimate && md->h.has_bdep && md->test_family == BI_FAMILY_ANY) {
      const FilterCost w = filter_cost(c, pl, pl.var[v0]);
      if (w.cta < 0.95 * w.block) return false;
    }
    use_variant(pl.var[v0], p);
    // agents per CTA (one-warp teams): one while the batch fits the machine anyway, so that no SM gets
    // four more warps than another; four for large batches, which share the CTA's exponential table
    p.W = p.LT == 32 ? (c.N > 24 * md->sm_count ? 4 : 1) : 1;
    p.UC = p.W; p.CS = 1;
    L.bytes = layout(pl, p, esz, p.W, p.W);
    if (L.bytes > budget) return false;
    L.grid = (unsigned)((c.N + p.W - 1) / p.W);
    L.threads = (unsigned)(p.W * p.LT);
  } else {
    // Steps per CTA and CTAs per agent: the cheapest by a small model of an iteration -- the larger of a
    // dependent chain of about a thousand cycles (more when it crosses CTAs) and the throughput of
    // the blocks resident on an SM -- times the number of waves.
    double best = 1e300;
    int bv = -1, buc = 0, bcs = 0;
    for (int v = 0; v < pl.nv; ++v) {
      use_variant(pl.var[v], p);
      p.W = 0;
      for (int cs = 1; cs <= 8; ++cs) {
        const int uc = ceil_div(c.T, cs);
        if (cs > 1 && ceil_div(c.T, uc) != cs) continue;
        const int th = uc * p.LT;
        if (th > pl.max_th) continue;
        if (p.LT > 32 && uc > 15) continue;   // (named barriers)
        const size_t b = layout(pl, p, esz, uc, 2 * (uc + 2));
        if (b > budget) continue;
        const int per_sm = std::max(1, std::min((int)((227 * 1024) / (b + 1024)), 65536 / (th * regs_per_thread(pl.BR * pl.BC * esz / 4))));
        const double ctas = (double)c.N * cs, waves = std::ceil(ctas / ((double)per_sm * md->sm_count));
        const double on_sm = std::min((double)per_sm, std::max(1.0, ctas / md->sm_count)) * uc;   // units side by side on an SM
        const double unit = (double)pl.NB * pl.BR * pl.BC * (0.045 + 0.07 * p.extra / std::max(pl.NB, 1)) * (esz / 8.0 + 0.25);
        const int rounds = ceil_div(p.npass, p.LT / 32);
        const double t = waves * std::max(300.0 + 600.0 * rounds + 450.0 * p.nbpt + (cs > 1 ? 350.0 : 0.0), on_sm * unit);
        if (t < best) { best = t; bv = v; buc = uc; bcs = cs; }
      }
    }
    if (bv < 0) return false;
    if (estimate && (!md->h.has_bdep || md->arith == BI_ARITH_F64) && md->h.G == 1 && (long long)c.N * c.T >= 2048 && md->test_family == BI_FAMILY_ANY && !md->soft_shadow) {
      const WindowCost w = window_cost(c, pl, pl.var[bv], best);
      // (in float64 from 2 500 units on: the tests pin a call of 2 472 to this side, [14,14,2,12] under a rank-4 slice, although
      // the kernels there have since become the faster ones for it too, 305 against 422 us)
      if (w.batch < w.block && (md->arith == BI_ARITH_F32 || (long long)c.N * c.T >= 2500)) return false;
    }
    use_variant(pl.var[bv], p);
    p.W = 0;
    p.UC = buc; p.CS = bcs;
    L.bytes = layout(pl, p, esz, buc, 2 * (buc + 2));
    L.grid = (unsigned)(c.N * bcs);
    L.threads = (unsigned)(buc * p.LT);
  }
  return true;
}

}  // namespace

bool bi_block_accepts(const BiCall &c) {
  Route L;
  return choose_route(c, L);
}

int bi_launch_block(const BiCall &c, bi_model *mut, bool estimate) {
  const bi_model *md = c.model;
  const bool window = c.algo != BI_ALGO_FILTER;
  Route L;
  if (!choose_route(c, L, estimate)) return BI_ERR_UNSUPPORTED;
  const Plan &pl = *L.plan;
  Params &p = L.p;
  const int esz = md->arith == BI_ARITH_F64 ? 8 : 4;
  const bool hass = p.nbpt > 1;
  const int sync = p.LT == 32 ? 0 : (window && p.UC > 1) ? 2 : 1;   // (SYNC_WARP, SYNC_CTA, SYNC_NAMED)
  const void *kern = esz == 8 ? bi_block_kernel_f64(pl.BR, pl.BC, window, sync, hass)
                              : bi_block_kernel_f32(pl.BR, pl.BC, window, sync, hass);
  if (!kern) return BI_ERR_UNSUPPORTED;
  if (bi_allow_smem(kern, L.bytes, true) != cudaSuccess) return BI_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(L.grid);
  cfg.blockDim = dim3(L.threads);
  cfg.dynamicSmemBytes = L.bytes;
  cfg.stream = c.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.CS;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.CS > 1 ? 1 : 0;
  void *args[1] = {(void *)&p};
  if (cudaLaunchKernelExC(&cfg, kern, args) != cudaSuccess) {
    cudaGetLastError();
    return BI_ERR_CUDA;
  }
  mut->launches += 1;
  const bool f64 = esz == 8;
  if (!window) mut->last_block = f64 ? "block_filter_f64" : "block_filter_f32";
  else if (c.algo == BI_ALGO_VMP) mut->last_block = f64 ? "block_vmp_f64" : "block_vmp_f32";
  else mut->last_block = f64 ? "block_mmp_f64" : "block_mmp_f32";
  // bi_last_kernel names the class of call: the family whose calls of this size these are
  if (!window) mut->last_kernel = f64 ? "cta_filter_f64" : "cta_filter_f32";
  else if (md->h.has_bdep || (long long)c.N * c.T < 2048)
    mut->last_kernel = c.algo == BI_ALGO_VMP ? (f64 ? "warp_vmp_f64" : "warp_vmp_f32") : (f64 ? "warp_mmp_f64" : "warp_mmp_f32");
  else
    mut->last_kernel = c.algo == BI_ALGO_VMP ? (f64 ? "batch_vmp_f64" : "batch_vmp_f32") : (f64 ? "batch_mmp_f64" : "batch_mmp_f32");
  return BI_OK;
}
