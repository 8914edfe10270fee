// Launch rules of the row-split block orthonormalisation (orth_cluster_rs.cu):
// the shared-memory layout of its CTAs, the shape of its grid form, and the
// global scratch that a mode's calls need.  Plain arithmetic, so that the
// planner, the launcher and the kernels share it and it can be checked on a
// machine without a GPU.
//
// A mode orthonormalises its Krylov blocks one by one, each against a longer
// basis.  Longer bases need more shared memory, so an early block may take the
// grid form when a later one cannot: the scratch is the maximum over the
// calls that take it, whichever they are.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <vector>

#ifdef __CUDACC__
#define TTR_HD __host__ __device__
#else
#define TTR_HD
#endif

namespace ttr {

struct KcLayout {
  int KP, ZP, RP;
  size_t share, slice, P, Gm, T, R, misc, Zc, Zn, Qc, tmp, total;
  int tmp_len;          // floats of tmp
  int slice_len;
  int share_bufs;       // 2 for a cluster (other ranks read the shares), 1 for the grid form
};

// nc: cluster size; nc = 0 for the grid form (shares and sums in global
// memory, no slice buffers).  tight: the split partial products keep room for
// the block's own Gram only, and Q^T Z is split less or not at all; for
// blocks that fit no other way (44,000 x 20 against 80 columns: 200 KB instead
// of 220 KB a CTA; the next route takes several launches).
TTR_HD inline KcLayout kc_layout(int kqmax, int zmax, int rows, int nc, bool tight) {
  KcLayout L;
  L.KP = (kqmax + 3) & ~3;
  L.ZP = (zmax + 3) & ~3;
  L.RP = (rows + 3) & ~3;
  size_t o = 0;
  auto take = [&](size_t n) { size_t r = o; o += (n + 3) & ~size_t(3); return r; };
  L.share_bufs = nc > 0 ? 2 : 1;
  L.share = take((size_t)L.share_bufs * (L.KP + L.ZP) * L.ZP);
  L.slice_len = nc > 0 ? ((L.KP + L.ZP) * L.ZP + nc - 1) / nc + 4 : 0;
  L.slice = take(2 * (size_t)L.slice_len);
  L.P = take((size_t)L.KP * L.ZP);
  L.Gm = take((size_t)zmax * (zmax + 1));
  L.T = take((size_t)L.ZP * L.ZP);
  L.R = take((size_t)zmax * zmax);
  L.misc = take(256);
  L.Zc = take((size_t)L.RP * L.ZP);
  L.Zn = take((size_t)L.RP * L.ZP);
  L.Qc = take((size_t)L.RP * L.KP);
  // split partial products: at most 512 tiles of 16 sums (tn_split)
  const size_t split = 8 * (size_t)L.ZP * (!tight && L.KP > L.ZP ? L.KP : L.ZP);
  L.tmp_len = (int)(split < 8192 ? split : 8192);
  L.tmp = take((size_t)L.tmp_len);
  L.total = o;
  return L;
}

// Limits of the device for the grid form: resident CTAs of the cooperative
// launch (one per SM; 0 without a device) and dynamic shared memory per CTA.
struct OrthGridLimits {
  int ctas = 0;
  size_t smem = 0;
};

// Shape of one grid-form call: nr CTAs of `rows` rows, shares of E floats.
struct OrthGridShape {
  int nr = 0, rows = 0, E = 0;
  bool tight = false;
  size_t smem = 0;
  // barrier words, two buffers of nr shares, two of their sums
  size_t scratch_floats() const { return 4 + 2 * (size_t)nr * E + 2 * (size_t)E; }
};

// One CTA per SM at most (every CTA of the cooperative launch resident), at
// least 16 rows each; false when the block does not fit.
inline bool orth_grid_shape(int64_t m, int kqmax, int zmax, const OrthGridLimits& lim, OrthGridShape* s) {
  if (m < 1 || zmax < 1 || zmax > 64 || kqmax > 256 || lim.ctas < 1) return false;
  int64_t nr0 = (m + 15) / 16;
  if (nr0 > lim.ctas) nr0 = lim.ctas;
  const int64_t rows = (m + nr0 - 1) / nr0;
  if (rows > (1 << 20)) return false;          // far beyond shared memory; keeps the layout's ints in range
  KcLayout L = kc_layout(kqmax, zmax, (int)rows, 0, false);
  s->tight = L.total * sizeof(float) > lim.smem;
  if (s->tight) L = kc_layout(kqmax, zmax, (int)rows, 0, true);
  const size_t smem = L.total * sizeof(float);
  if (smem > lim.smem) return false;
  s->rows = (int)rows;
  s->nr = (int)((m + rows - 1) / rows);
  s->E = (L.KP + L.ZP) * L.ZP;
  s->smem = smem;
  return true;
}

// One orthonormalisation of a mode: zc columns against a basis of kq0, c of
// them kept; grid: the grid form takes it when the cluster form does not.
struct OrthCall {
  int kq0, zc, c;
  bool grid = false;
};

// The calls of a mode in their order: the sketch of b columns, of which
// blocks[0] are kept, and then for Alg. 3 each further block from the power of
// the one before; with `restarts` (Alg. 4, the literal form) the later calls
// are one and the same, blocks[0] columns with no basis.
inline std::vector<OrthCall> orth_calls(int b, const std::vector<int>& blocks, bool restarts) {
  std::vector<OrthCall> out;
  out.push_back({0, b, blocks[0]});
  if (restarts) {
    out.push_back({0, blocks[0], blocks[0]});
    return out;
  }
  int cols = 0;
  for (size_t j = 0; j + 1 < blocks.size(); ++j) {
    cols += blocks[j];
    out.push_back({cols, blocks[j], blocks[j + 1]});
  }
  return out;
}

// Marks the calls that the grid form takes and returns the scratch floats the
// largest of them needs.
inline size_t orth_grid_plan(int64_t m, const OrthGridLimits& lim, std::vector<OrthCall>* calls) {
  size_t need = 0;
  for (OrthCall& c : *calls) {
    OrthGridShape s;
    c.grid = c.c >= 1 && c.c <= c.zc && orth_grid_shape(m, c.kq0 + c.c, c.zc, lim, &s);
    if (c.grid && s.scratch_floats() > need) need = s.scratch_floats();
  }
  return need;
}

}  // namespace ttr
