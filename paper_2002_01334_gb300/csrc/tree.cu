// Input validation, per-group octrees (Morton keys + radix sort) and interaction lists.
// Tree rule (Sec. 3.5, before Algorithm 1): the root cube of target group (l, a) is bisected by its interface
// (d_l for a = 1, d_{l-1} for a = 2), so every box of level >= 1 has its centre on the
// side of the points it holds; all trees here have uniform depth D.
#include "internal.h"
#include "prims.cuh"

#include <algorithm>

namespace lpb {

// ---------------------------------------------------------------------------------------
// scan / sort wrappers
// ---------------------------------------------------------------------------------------
void scan_u32(Ctx &c, const uint32_t *in, uint32_t *out, int64_t n, uint32_t *d_total) {
  if (n <= 8192) {  // one launch, one chunk
    k_scan_one<<<1, 1024, 0, c.stream>>>(in, out, n, d_total);
    LPB_LAUNCH();
    c.launches++;
    return;
  }
  const int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  uint32_t *sums = c.arena.get<uint32_t>(tiles + 1);
  if (n > 0) {
    k_scan_tiles<<<(unsigned)tiles, SCAN_THREADS, 0, c.stream>>>(in, out, sums, n);
    LPB_LAUNCH();
  }
  k_scan_sums<<<1, 1024, 0, c.stream>>>(sums, tiles, d_total);
  LPB_LAUNCH();
  if (tiles > 1) {
    k_scan_add<<<(unsigned)tiles, SCAN_THREADS, 0, c.stream>>>(out, sums, n);
    LPB_LAUNCH();
  }
  c.launches += 2 + (tiles > 1) + (n > 0 ? 0 : -1);
}

// the scans of several arrays
static void scan_batch(Ctx &c, ScanJobs &J, int nj) {
  int64_t nmax = 0;
  for (int k = 0; k < nj; ++k) nmax = std::max(nmax, J.j[k].n);
  if (!nj || !nmax) return;
  if (nmax <= 8192) {
    k_scan_one_b<<<nj, 1024, 0, c.stream>>>(J);
    LPB_LAUNCH();
    c.launches++;
    return;
  }
  const unsigned tiles = (unsigned)((nmax + SCAN_TILE - 1) / SCAN_TILE);
  for (int k = 0; k < nj; ++k) J.j[k].sums = c.arena.get<uint32_t>((size_t)(J.j[k].n + SCAN_TILE - 1) / SCAN_TILE + 1);
  k_scan_tiles_b<<<dim3(tiles, nj), SCAN_THREADS, 0, c.stream>>>(J);
  LPB_LAUNCH();
  k_scan_sums_b<<<nj, 1024, 0, c.stream>>>(J);
  LPB_LAUNCH();
  k_scan_add_b<<<dim3(tiles, nj), SCAN_THREADS, 0, c.stream>>>(J);
  LPB_LAUNCH();
  c.launches += 3;
}

// stable sorts of several arrays by key bits [lo, bits) of each: lower bits must not matter for the order
// (zero, or a field equal within a run that the caller does not need sorted)
struct SortReq {
  uint64_t **keys;
  uint32_t **vals;
  int64_t n;
  int bits, lo;
};
static void sort_batch(Ctx &c, const std::vector<SortReq> &reqs) {
  SortJobs small{}, large{};
  ScanJobs sc{};
  std::vector<const SortReq *> rs, rl;
  for (const SortReq &r : reqs) {
    if (r.n <= 1) continue;
    SortJob j{};
    j.k = *r.keys; j.v = *r.vals; j.n = r.n; j.lo = r.lo; j.bits = r.bits;
    j.ok = c.arena.get<uint64_t>(r.n);
    j.ov = c.arena.get<uint32_t>(r.n);
    if (r.n <= RS_SMALL) {
      small.j[rs.size()] = j;
      rs.push_back(&r);
    } else {
      j.nblocks = (int)((r.n + RS_TILE - 1) / RS_TILE);
      j.hist = c.arena.get<uint32_t>((size_t)256 * j.nblocks);
      j.offs = c.arena.get<uint32_t>((size_t)256 * j.nblocks);
      large.j[rl.size()] = j;
      rl.push_back(&r);
    }
  }
  if (!rs.empty()) {
    k_radix_small<<<(unsigned)rs.size(), 1024, 0, c.stream>>>(small);
    LPB_LAUNCH();
    c.launches++;
    for (size_t k = 0; k < rs.size(); ++k)
      if (((rs[k]->bits - rs[k]->lo + 7) / 8) & 1) {
        *rs[k]->keys = small.j[k].ok;
        *rs[k]->vals = small.j[k].ov;
      }
  }
  for (int pass = 0; !rl.empty(); ++pass) {
    SortJobs J{};
    std::vector<int> who;
    unsigned nb = 0;
    for (size_t k = 0; k < rl.size(); ++k)
      if (large.j[k].lo + 8 * pass < large.j[k].bits) {
        J.j[who.size()] = large.j[k];
        sc.j[who.size()] = ScanJob{large.j[k].hist, large.j[k].offs, nullptr, (int64_t)256 * large.j[k].nblocks};
        who.push_back((int)k);
        nb = std::max(nb, (unsigned)large.j[k].nblocks);
      }
    if (who.empty()) break;
    const int nj = (int)who.size();
    k_radix_hist<<<dim3(nb, nj), RS_THREADS, 0, c.stream>>>(J, pass);
    LPB_LAUNCH();
    scan_batch(c, sc, nj);
    k_radix_scatter<<<dim3(nb, nj), RS_THREADS, 0, c.stream>>>(J, pass);
    LPB_LAUNCH();
    c.launches += 2;
    for (int k : who) {
      SortJob &j = large.j[k];
      uint64_t *tk = const_cast<uint64_t *>(j.k);
      uint32_t *tv = const_cast<uint32_t *>(j.v);
      j.k = j.ok; j.ok = tk;
      j.v = j.ov; j.ov = tv;
    }
  }
  for (size_t k = 0; k < rl.size(); ++k) {
    *rl[k]->keys = const_cast<uint64_t *>(large.j[k].k);
    *rl[k]->vals = const_cast<uint32_t *>(large.j[k].v);
  }
}

// ---------------------------------------------------------------------------------------
// validation: finite, off the interfaces, layer_id consistent with z; counts and extents
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long ord_of(double v) {
  unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ unsigned long long wmin(unsigned long long v) {
  for (int o = 16; o; o >>= 1) { unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o); v = w < v ? w : v; }
  return v;
}
__device__ __forceinline__ unsigned long long wmax(unsigned long long v) {
  for (int o = 16; o; o >>= 1) { unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o); v = w > v ? w : v; }
  return v;
}

// Grid-stride validation: every thread keeps its own extremes (order-preserving integers of
// the FP64 coordinates) and per-layer counts; they are reduced per warp by shuffles, per block
// in shared memory, and merged into the global statistics with one atomic per block and field.
constexpr int VAL_THREADS = 256;
__global__ void __launch_bounds__(VAL_THREADS) k_validate(int64_t n, const double *q, const double *q2, const double *xyz,
                                                          const int32_t *layer, Medium md, double thr, Stats *st) {
  const unsigned long long HI = ~0ull, LO = 0ull;
  unsigned long long xlo = HI, xhi = LO, ylo = HI, yhi = LO, zlo[MAXLAYER], zhi[MAXLAYER];
  unsigned cnt[MAXLAYER];
#pragma unroll
  for (int k = 0; k < MAXLAYER; ++k) {
    zlo[k] = HI;
    zhi[k] = LO;
    cnt[k] = 0;
  }
  int code_seen = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
    const double qq = q[i];
    const int lay = layer[i];
    int code = 0;
    if (!isfinite(x) || !isfinite(y) || !isfinite(z) || !isfinite(qq) || (q2 && !isfinite(q2[i]))) {
      code = LPBFMM_ERR_NONFINITE;
    } else {
      int l = 0;
      while (l < md.L && z < md.d[l]) ++l;
      for (int k = 0; k < md.L; ++k)
        if (fabs(z - md.d[k]) < thr) code = LPBFMM_ERR_ON_INTERFACE;
      if (!code && l != lay) code = LPBFMM_ERR_LAYER_MISMATCH;
    }
    if (code) {
      if (!code_seen) atomicCAS(&st->status, 0, code);
      code_seen = 1;
      continue;
    }
    const unsigned long long ox = ord_of(x), oy = ord_of(y), oz = ord_of(z);
    xlo = min(xlo, ox); xhi = max(xhi, ox);
    ylo = min(ylo, oy); yhi = max(yhi, oy);
#pragma unroll
    for (int k = 0; k < MAXLAYER; ++k)
      if (k == lay) {
        zlo[k] = min(zlo[k], oz);
        zhi[k] = max(zhi[k], oz);
        ++cnt[k];
      }
  }
  __shared__ unsigned long long red[VAL_THREADS / 32][4 + 3 * MAXLAYER];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long v[4 + 3 * MAXLAYER];
  v[0] = wmin(xlo); v[1] = wmax(xhi); v[2] = wmin(ylo); v[3] = wmax(yhi);
#pragma unroll
  for (int k = 0; k < MAXLAYER; ++k) {
    v[4 + k] = wmin(zlo[k]);
    v[4 + MAXLAYER + k] = wmax(zhi[k]);
    unsigned c = cnt[k];
#pragma unroll
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    v[4 + 2 * MAXLAYER + k] = c;
  }
  if (lane == 0)
    for (int f = 0; f < 4 + 3 * MAXLAYER; ++f) red[warp][f] = v[f];
  __syncthreads();
  if (threadIdx.x < 4 + 3 * MAXLAYER) {
    const int f = threadIdx.x;
    const bool is_min = f == 0 || f == 2 || (f >= 4 && f < 4 + MAXLAYER);
    const bool is_cnt = f >= 4 + 2 * MAXLAYER;
    unsigned long long a = is_min ? HI : LO;
    for (int w2 = 0; w2 < nw; ++w2) {
      const unsigned long long b = red[w2][f];
      a = is_cnt ? a + b : (is_min ? min(a, b) : max(a, b));
    }
    unsigned long long *dst = f == 0 ? &st->xlo : f == 1 ? &st->xhi : f == 2 ? &st->ylo : f == 3 ? &st->yhi
                            : f < 4 + MAXLAYER ? &st->zlo[f - 4]
                            : f < 4 + 2 * MAXLAYER ? &st->zhi[f - 4 - MAXLAYER]
                            : &st->cnt[f - 4 - 2 * MAXLAYER];
    if (is_cnt) { if (a) atomicAdd(dst, a); }
    else if (is_min) { if (a != HI) atomicMin(dst, a); }
    else if (a != LO) atomicMax(dst, a);
  }
}

void launch_validate(Ctx &c, int64_t n, const double *q, const double *q2, const double *xyz, const int32_t *layer,
                     Stats *st) {
  double scale = 1.0;
  for (int k = 0; k < c.md.L; ++k) scale = fmax(scale, fabs(c.md.d[k]));
  const double thr = 1e-12 * scale;
  const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + VAL_THREADS - 1) / VAL_THREADS, 152 * 4));
  k_validate<<<blocks, VAL_THREADS, 0, c.stream>>>(n, q, q2, xyz, layer, c.md, thr, st);
  LPB_LAUNCH();
  c.launches++;
}

// flags of every layer present (f[k] may be null)
__global__ void k_flag_layers(int64_t n, const int32_t *layer, int nl, RankPtrs f) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int lay = layer[i];
  for (int k = 0; k < nl; ++k)
    if (f.r[k]) f.r[k][i] = lay == k ? 1u : 0u;
}
// stable rank of every charge within its layer (layers without charges: null)
void layer_ranks(Ctx &c, int64_t n, const int32_t *layer, const int64_t *cnt, RankPtrs &rank) {
  RankPtrs f{};
  ScanJobs J{};
  int nj = 0;
  for (int k = 0; k <= c.md.L; ++k) {
    rank.r[k] = nullptr;
    if (!cnt[k]) continue;
    f.r[k] = c.arena.get<uint32_t>(n);
    rank.r[k] = c.arena.get<uint32_t>(n);
    J.j[nj++] = ScanJob{f.r[k], rank.r[k], nullptr, n};
  }
  k_flag_layers<<<(unsigned)((n + 255) / 256), 256, 0, c.stream>>>(n, layer, c.md.L + 1, f);
  LPB_LAUNCH();
  c.launches++;
  scan_batch(c, J, nj);
}

// ---------------------------------------------------------------------------------------
// points and Morton keys
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
  uint64_t x = v & 0x3ffu;  // 10 bits
  x = (x | (x << 16)) & 0x30000ffull;
  x = (x | (x << 8)) & 0x300f00full;
  x = (x | (x << 4)) & 0x30c30c3ull;
  x = (x | (x << 2)) & 0x9249249ull;
  return x;
}
__device__ __forceinline__ uint32_t compact3(uint64_t x) {
  x &= 0x9249249ull;
  x = (x ^ (x >> 2)) & 0x30c30c3ull;
  x = (x ^ (x >> 4)) & 0x300f00full;
  x = (x ^ (x >> 8)) & 0x30000ffull;
  x = (x ^ (x >> 16)) & 0x3ffull;
  return (uint32_t)x;
}
// cell index i = floor((x - x0) * s) clamped to [0, 2^DMAX - 1]; rounded ops, no contraction
__device__ __forceinline__ uint32_t cell_of(double x, double x0, double s) {
  double t = floor(__dmul_rn(__dsub_rn(x, x0), s));
  t = fmin(fmax(t, 0.0), double((1 << DMAX) - 1));
  return (uint32_t)t;
}
__device__ __forceinline__ uint64_t morton_of(double x, double y, double z, const double *o, double s) {
  return (spread3(cell_of(x, o[0], s)) << 2) | (spread3(cell_of(y, o[1], s)) << 1) | spread3(cell_of(z, o[2], s));
}

struct GroupGeom {
  double o[3];  // lower corner of the root cube
  double s;     // 2^DMAX / (2H)
  int l, a, D;
  int64_t type_off[2 * MAXLAYER];
  uint64_t *key;
  uint32_t *src;
};
struct GroupGeoms {
  GroupGeom g[MAXJOB];
};
struct GatherJob {
  int64_t np;
  const uint64_t *key;
  const uint32_t *src;
  int l, a;
  double *x, *y, *z, *q;
  uint32_t *cnt;  // targets: non-empty boxes per level (null: not counted)
};
struct GatherJobs {
  GatherJob j[MAXJOB];
};

__global__ void k_make_targets(int64_t n, const double *xyz, const int32_t *layer, RankPtrs rk, int ng,
                               const __grid_constant__ GroupGeoms G) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int lay = layer[i];
  const double x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
  for (int k = 0; k < ng; ++k) {
    const GroupGeom &gg = G.g[k];
    if (lay != gg.l) continue;
    const uint32_t pos = rk.r[gg.l][i];
    gg.key[pos] = morton_of(x, y, z, gg.o, gg.s) << 4;
    gg.src[pos] = (uint32_t)i;
  }
}

__global__ void k_make_images(int64_t n, const double *xyz, const int32_t *layer, Medium md, RankPtrs rk, int ng,
                              const __grid_constant__ GroupGeoms G) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int lp = layer[i];
  const double x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
  const uint32_t rank = rk.r[lp][i];
  for (int k = 0; k < ng; ++k) {
    const GroupGeom &gg = G.g[k];
    for (int b = 1; b <= 2; ++b) {
      if ((b == 1 && lp == md.L) || (b == 2 && lp == 0)) continue;
      const int t = type_index(lp, b);
      const int64_t pos = gg.type_off[t] + rank;
      const double zi = image_z(md, gg.l, gg.a, lp, b, z);
      gg.key[pos] = ((morton_of(x, y, zi, gg.o, gg.s) >> (3 * (DMAX - gg.D))) << 4) | (uint64_t)t;
      gg.src[pos] = (uint32_t)i;
    }
  }
}

// sorted points of every group; with cnt, also the number of non-empty target boxes at every level
// 2..DMAX (automatic depth rule)
__global__ void k_gather_points(const double *q, const double *xyz, Medium md, int images,
                                const __grid_constant__ GatherJobs J) {
  const GatherJob &j = J.j[blockIdx.y];
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j.cnt)
    for (int l = 2; l <= DMAX; ++l) {
      bool f = false;
      if (k < j.np) {
        const int sh = 4 + 3 * (DMAX - l);
        f = (k == 0) || ((j.key[k] >> sh) != (j.key[k - 1] >> sh));
      }
      const unsigned b = __popc(__ballot_sync(0xffffffffu, f));
      if ((threadIdx.x & 31) == 0 && b) atomicAdd(&j.cnt[l], b);
    }
  if (k >= j.np) return;
  const uint32_t i = j.src[k];
  j.x[k] = xyz[3 * (size_t)i];
  j.y[k] = xyz[3 * (size_t)i + 1];
  double z = xyz[3 * (size_t)i + 2];
  if (images) {
    int lp, b;
    type_decode((int)(j.key[k] & 15ull), lp, b);
    z = image_z(md, j.l, j.a, lp, b, z);
  }
  j.z[k] = z;
  j.q[k] = q[i];
}

static GroupGeom group_geom(Ctx &c, const Group &g, const int64_t *cnt) {
  GroupGeom gg;
  const double H = g.root[3];
  gg.o[0] = g.root[0] - H;
  gg.o[1] = g.root[1] - H;
  gg.o[2] = g.root[2] - H;
  gg.s = double(1 << DMAX) / (2.0 * H);
  gg.l = g.l;
  gg.a = g.a;
  gg.D = g.D;
  int64_t off = 0;
  for (int t = 0; t < 2 * c.md.L; ++t) {
    int lp, b;
    type_decode(t, lp, b);
    gg.type_off[t] = off;
    off += cnt[lp];
  }
  return gg;
}

static void gather(Ctx &c, std::vector<Group> &groups, int images, const double *q, const double *xyz, uint32_t *dc) {
  GatherJobs J{};
  int nj = 0;
  int64_t nmax = 0;
  for (size_t k = 0; k < groups.size(); ++k) {
    Group &g = groups[k];
    PointSet &P = images ? g.I : g.T;
    P.x = c.arena.get<double>(P.np);
    P.y = c.arena.get<double>(P.np);
    P.z = c.arena.get<double>(P.np);
    P.q = c.arena.get<double>(P.np);
    if (!P.np) continue;
    J.j[nj++] = GatherJob{P.np, P.key, P.src, g.l, g.a, P.x, P.y, P.z, P.q, dc ? dc + k * (DMAX + 1) : nullptr};
    nmax = std::max(nmax, P.np);
  }
  if (!nj) return;
  k_gather_points<<<dim3((unsigned)((nmax + 255) / 256), nj), 256, 0, c.stream>>>(q, xyz, c.md, images, J);
  LPB_LAUNCH();
  c.launches++;
}

struct ChargeJob {
  int64_t np;
  const uint32_t *src;
  double *q;
};
struct ChargeJobs {
  ChargeJob j[2 * MAXJOB];
};
__global__ void k_recharge(const double *q, const __grid_constant__ ChargeJobs J) {
  const ChargeJob &j = J.j[blockIdx.y];
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < j.np) j.q[k] = q[j.src[k]];
}
void recharge_points(Ctx &c, std::vector<Group> &groups, const double *q) {
  ChargeJobs J{};
  int nj = 0;
  int64_t nmax = 0;
  for (auto &g : groups)
    for (PointSet *P : {&g.T, &g.I}) {
      if (!P->np) continue;
      J.j[nj++] = ChargeJob{P->np, P->src, P->q};
      nmax = std::max(nmax, P->np);
    }
  if (!nj) return;
  k_recharge<<<dim3((unsigned)((nmax + 255) / 256), nj), 256, 0, c.stream>>>(q, J);
  LPB_LAUNCH();
  c.launches++;
}

// targets of every group, sorted by their depth-DMAX Morton keys (every coarser key is a prefix); dc (may be
// null): non-empty boxes per group and level [G][DMAX + 1]
void build_targets(Ctx &c, std::vector<Group> &groups, int64_t n, const double *q, const double *xyz,
                   const int32_t *layer, const RankPtrs &rank, const int64_t *cnt, uint32_t *dc) {
  if (groups.empty()) return;
  GroupGeoms G{};
  std::vector<SortReq> reqs;
  for (size_t k = 0; k < groups.size(); ++k) {
    Group &g = groups[k];
    g.T.np = cnt[g.l];
    g.T.key = c.arena.get<uint64_t>(g.T.np);
    g.T.src = c.arena.get<uint32_t>(g.T.np);
    G.g[k] = group_geom(c, g, cnt);
    G.g[k].key = g.T.key;
    G.g[k].src = g.T.src;
    reqs.push_back(SortReq{&g.T.key, &g.T.src, g.T.np, DMAX * 3 + 4, 4});  // the low 4 bits are zero
  }
  k_make_targets<<<(unsigned)((n + 255) / 256), 256, 0, c.stream>>>(n, xyz, layer, rank, (int)groups.size(), G);
  LPB_LAUNCH();
  c.launches++;
  sort_batch(c, reqs);
  gather(c, groups, 0, q, xyz, dc);
}

// images of every group, sorted by (depth-D leaf key, type, input order): every (leaf box,
// type) pair is one contiguous run
void build_images(Ctx &c, std::vector<Group> &groups, int64_t n, const double *q, const double *xyz,
                  const int32_t *layer, const RankPtrs &rank, const int64_t *cnt) {
  if (groups.empty()) return;
  int64_t tot = 0;
  for (int t = 0; t < 2 * c.md.L; ++t) {
    int lp, b;
    type_decode(t, lp, b);
    tot += cnt[lp];
  }
  GroupGeoms G{};
  std::vector<SortReq> reqs;
  for (size_t k = 0; k < groups.size(); ++k) {
    Group &g = groups[k];
    g.I.np = tot;
    g.I.key = c.arena.get<uint64_t>(g.I.np);
    g.I.src = c.arena.get<uint32_t>(g.I.np);
    G.g[k] = group_geom(c, g, cnt);
    G.g[k].key = g.I.key;
    G.g[k].src = g.I.src;
    reqs.push_back(SortReq{&g.I.key, &g.I.src, g.I.np, g.D * 3 + 4, 0});
  }
  k_make_images<<<(unsigned)((n + 255) / 256), 256, 0, c.stream>>>(n, xyz, layer, c.md, rank, (int)groups.size(), G);
  LPB_LAUNCH();
  c.launches++;
  sort_batch(c, reqs);
  gather(c, groups, 1, q, xyz, nullptr);
}

// ---------------------------------------------------------------------------------------
// boxes of every level of every point set.  The points are sorted by key, so the boxes of a level are
// the runs of equal key prefix: for each (set, level) a scan of the run starts numbers the boxes
// (k_box_tiles, k_box_sums), every run start writes its box, every point keeps its box number
// (k_box_fill), and the links between levels follow from the box numbers of the run starts (k_box_links).
// Four launches for all sets and levels.  Image sets also number their (leaf box, type) segments.
// ---------------------------------------------------------------------------------------
struct BoxJob {
  const uint64_t *pkey;
  int64_t np, tile0, box0, cap;  // first tile / first box slot of this job in the flattened launches
  int sh, seg;                   // key prefix: key >> sh; seg: (leaf box, type) segments
  uint32_t *idx, *sums, *total;  // box of every point, per-tile counts, number of boxes
  uint64_t *key;
  uint32_t *pstart, *pcount;     // segments: seg_start, seg_count
  uint32_t *start, *count;       // children (null at the leaf level)
  const uint32_t *cidx, *ctotal; // the finer level's box numbers and total
  uint32_t *parent;              // (null at level 2)
  const uint32_t *pidx;          // the coarser level's box numbers
  uint32_t *sbox, *stype;        // segments: leaf box (cidx: the leaf level's numbers), type
};
__device__ __forceinline__ bool box_starts(const BoxJob &j, int64_t k) {
  return k == 0 || (j.pkey[k] >> j.sh) != (j.pkey[k - 1] >> j.sh);
}
template <int64_t BoxJob::*M>
__device__ __forceinline__ int box_find(const BoxJob *jobs, int nj, int64_t g) {
  int lo = 0, hi = nj - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].*M <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}
__global__ void k_box_tiles(const BoxJob *jobs, int nj) {
  const BoxJob j = jobs[box_find<&BoxJob::tile0>(jobs, nj, blockIdx.x)];
  __shared__ uint32_t sm[32];
  const int64_t tile = (int64_t)blockIdx.x - j.tile0;
  const int64_t base = tile * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  uint32_t f = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k)
    if (base + k < j.np && box_starts(j, base + k)) f |= 1u << k;
  uint32_t tot;
  uint32_t run = block_exclusive_scan(__popc(f), sm, &tot);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    run += (f >> k) & 1u;
    if (base + k < j.np) j.idx[base + k] = run;  // run starts of the tile up to and including this point
  }
  if (threadIdx.x == 0) j.sums[tile] = tot;
}
__global__ void k_box_sums(const BoxJob *jobs) {
  const BoxJob &j = jobs[blockIdx.x];
  __shared__ uint32_t sm[32];
  const int64_t m = (j.np + SCAN_TILE - 1) / SCAN_TILE;
  uint32_t carry = 0;
  for (int64_t c = 0; c < m; c += blockDim.x) {
    const int64_t i = c + threadIdx.x;
    const uint32_t v = i < m ? j.sums[i] : 0u;
    uint32_t tot;
    const uint32_t ex = block_exclusive_scan(v, sm, &tot);
    if (i < m) j.sums[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) *j.total = carry;
}
__global__ void k_box_fill(const BoxJob *jobs, int nj) {
  const BoxJob j = jobs[box_find<&BoxJob::tile0>(jobs, nj, blockIdx.x)];
  const int64_t tile = (int64_t)blockIdx.x - j.tile0;
  const uint32_t before = j.sums[tile];
  for (int x = threadIdx.x; x < SCAN_TILE; x += blockDim.x) {
    const int64_t k = tile * SCAN_TILE + x;
    if (k >= j.np) break;
    const uint32_t b = before + j.idx[k] - 1u;
    j.idx[k] = b;
    if (!box_starts(j, k)) continue;
    j.pstart[b] = (uint32_t)k;
    if (j.seg) j.stype[b] = (uint32_t)(j.pkey[k] & 15ull);
    else j.key[b] = j.pkey[k] >> j.sh;
  }
}
__global__ void k_box_links(const BoxJob *jobs, int nj, int64_t ntot) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ntot) return;
  const BoxJob &j = jobs[box_find<&BoxJob::box0>(jobs, nj, g)];
  const int64_t b = g - j.box0;
  const uint32_t n = *j.total;
  if (b >= n || b >= j.cap) return;
  const uint32_t s = j.pstart[b], e = b + 1 < n ? j.pstart[b + 1] : (uint32_t)j.np;
  j.pcount[b] = e - s;
  if (j.seg) {
    j.sbox[b] = j.cidx[s];
    return;
  }
  if (j.start) {
    const uint32_t c0 = j.cidx[s], c1 = b + 1 < n ? j.cidx[e] : *j.ctotal;
    j.start[b] = c0;
    j.count[b] = c1 - c0;
  }
  if (j.parent) j.parent[b] = j.pidx[s];
}

static int64_t level_cap(int64_t np, int l) {
  int64_t c = 1;
  for (int k = 0; k < l && c < np; ++k) c *= 8;
  return c < np ? c : np;
}

// the box arrays of every group; *dcounts, *ncounts: the device array of box counts in the order of
// read_box_counts
void build_boxes(Ctx &c, std::vector<Group> &groups, uint32_t **dcounts, size_t *ncounts) {
  std::vector<BoxJob> jobs;
  size_t nc = 0;
  for (auto &g : groups) nc += 2 * (size_t)(g.D - 1) + 1;
  uint32_t *counts = c.arena.get<uint32_t>(nc);
  LPB_CUDA(cudaMemsetAsync(counts, 0, sizeof(uint32_t) * nc, c.stream));
  *dcounts = counts;
  *ncounts = nc;
  int64_t tiles = 0, boxes = 0;
  size_t at = 0;
  for (auto &g : groups)
    for (int which = 0; which < 2; ++which) {
      PointSet &P = which ? g.I : g.T;
      const int64_t np = P.np, nt = (np + SCAN_TILE - 1) / SCAN_TILE;
      for (int l = 0; l <= DMAX; ++l) P.lev[l] = Level();
      for (int l = 2; l <= g.D; ++l, ++at) {
        if (!np) continue;
        Level &L = P.lev[l];
        BoxJob j{};
        j.pkey = P.key; j.np = np; j.tile0 = tiles; j.box0 = boxes; j.cap = level_cap(np, l);
        // targets carry depth-DMAX keys, images depth-D keys (both shifted by 4 type bits)
        j.sh = 4 + 3 * ((which ? g.D : DMAX) - l);
        j.idx = c.arena.get<uint32_t>(np);
        j.sums = c.arena.get<uint32_t>(nt);
        j.total = L.d_n = counts + at;
        j.key = L.key = c.arena.get<uint64_t>(j.cap);
        j.pstart = L.pstart = c.arena.get<uint32_t>(j.cap);
        j.pcount = L.pcount = c.arena.get<uint32_t>(j.cap);
        if (l < g.D) {
          j.start = L.start = c.arena.get<uint32_t>(j.cap);
          j.count = L.count = c.arena.get<uint32_t>(j.cap);
        } else {
          L.start = L.pstart;
          L.count = L.pcount;
        }
        if (l > 2) {
          j.parent = L.parent = c.arena.get<uint32_t>(j.cap);
          j.pidx = jobs.back().idx;
          jobs.back().cidx = j.idx;
          jobs.back().ctotal = j.total;
        }
        jobs.push_back(j);
        tiles += nt;
        boxes += j.cap;
        if (l == g.D) P.pbox = j.idx;
      }
      if (which) {
        if (np) {
          BoxJob j = jobs.back();  // the leaf level's keys with their type bits
          j.tile0 = tiles; j.box0 = boxes; j.cap = np; j.sh = 0; j.seg = 1;
          j.cidx = j.idx;
          j.idx = c.arena.get<uint32_t>(np);
          j.sums = c.arena.get<uint32_t>(nt);
          j.total = P.d_nseg = counts + at;
          j.pstart = P.seg_start = c.arena.get<uint32_t>(np);
          j.pcount = P.seg_count = c.arena.get<uint32_t>(np);
          j.sbox = P.seg_box = c.arena.get<uint32_t>(np);
          j.stype = P.seg_type = c.arena.get<uint32_t>(np);
          j.start = j.count = j.parent = nullptr;
          jobs.push_back(j);
          tiles += nt;
          boxes += np;
        }
        ++at;
      }
    }
  if (jobs.empty()) return;
  const int nj = (int)jobs.size();
  BoxJob *dj = c.arena.get<BoxJob>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(BoxJob) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
  k_box_tiles<<<(unsigned)tiles, SCAN_THREADS, 0, c.stream>>>(dj, nj);
  LPB_LAUNCH();
  k_box_sums<<<nj, 1024, 0, c.stream>>>(dj);
  LPB_LAUNCH();
  k_box_fill<<<(unsigned)tiles, SCAN_THREADS, 0, c.stream>>>(dj, nj);
  LPB_LAUNCH();
  k_box_links<<<(unsigned)((boxes + 255) / 256), 256, 0, c.stream>>>(dj, nj, boxes);
  LPB_LAUNCH();
  c.launches += 4;
}

// source types present in every image box: each segment marks its leaf and climbs until an ancestor is marked
// already (whoever marked it climbs on)
struct MaskJob {
  const uint32_t *sbox, *stype;
  int64_t nseg, item0;
  int D;
  const uint32_t *parent[DMAX + 1];
  uint32_t *mask[DMAX + 1];
};
__global__ void k_type_masks(const MaskJob *jobs, int nj, int64_t ntot) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ntot) return;
  int lo = 0, hi = nj - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].item0 <= g) lo = mid; else hi = mid - 1;
  }
  const MaskJob &J = jobs[lo];
  const int64_t s = g - J.item0;
  if (s >= J.nseg) return;
  uint32_t b = J.sbox[s];
  const uint32_t bit = 1u << J.stype[s];
  for (int l = J.D; l >= 2; --l) {
    if ((l < J.D && (*(volatile uint32_t *)&J.mask[l][b] & bit)) || (atomicOr(&J.mask[l][b], bit) & bit)) return;
    if (l > 2) b = J.parent[l][b];
  }
}
void build_type_masks(Ctx &c, std::vector<Group> &groups) {
  std::vector<MaskJob> jobs;
  int64_t segs = 0, boxes = 0;
  for (auto &g : groups)
    if ((g.parts & 2) && g.I.np)
      for (int l = 2; l <= g.D; ++l) boxes += g.I.lev[l].n;
  if (!boxes) return;
  uint32_t *m = c.arena.get<uint32_t>(boxes);
  LPB_CUDA(cudaMemsetAsync(m, 0, sizeof(uint32_t) * boxes, c.stream));
  for (auto &g : groups) {
    if (!((g.parts & 2) && g.I.np)) continue;
    MaskJob j{};
    j.sbox = g.I.seg_box; j.stype = g.I.seg_type; j.nseg = g.I.nseg; j.item0 = segs; j.D = g.D;
    segs += j.nseg;
    for (int l = 2; l <= g.D; ++l) {
      g.tmask[l] = j.mask[l] = m;
      j.parent[l] = g.I.lev[l].parent;
      m += g.I.lev[l].n;
    }
    jobs.push_back(j);
  }
  if (!segs) return;
  MaskJob *dj = c.arena.get<MaskJob>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(MaskJob) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
  k_type_masks<<<(unsigned)((segs + 255) / 256), 256, 0, c.stream>>>(dj, (int)jobs.size(), segs);
  LPB_LAUNCH();
  c.launches++;
}

// the counts of build_boxes, on the host, into the groups
void read_box_counts(std::vector<Group> &groups, const uint32_t *h) {
  for (auto &g : groups) {
    for (int which = 0; which < 2; ++which) {
      PointSet &P = which ? g.I : g.T;
      for (int l = 2; l <= g.D; ++l) P.lev[l].n = P.np ? *h : 0, ++h;
    }
    g.I.nseg = g.I.np ? *h : 0;
    ++h;
  }
}

// ---------------------------------------------------------------------------------------
// interaction lists with separation ws.  Far list (multipole-to-local, V): source boxes at
// offset d with |d|_inf > ws whose parent lies within ws of the target's parent.  Near list
// (U): |d|_inf <= ws.  Dense layout: [target box][offset slot] -> source box index or -1, with
// the slots of WS_MAX (offsets of a smaller ws leave the outer slots at -1).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ int64_t find_key(const uint64_t *keys, int64_t n, uint64_t k) {
  int64_t lo = 0, hi = n - 1;
  while (lo <= hi) {
    const int64_t m = (lo + hi) >> 1;
    const uint64_t v = keys[m];
    if (v == k) return m;
    if (v < k) lo = m + 1; else hi = m - 1;
  }
  return -1;
}

// dense box index of a level: grid[Morton key] = box index or -1 (levels up to GRID_LEV_MAX)
constexpr int GRID_LEV_MAX = 8;
struct GridJob {
  const uint64_t *key;
  int32_t *grid;
  int64_t n, box0;
};
__global__ void k_grid_fill(const GridJob *jobs, int nj, int64_t ntot) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ntot) return;
  int lo = 0, hi = nj - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].box0 <= g) lo = mid; else hi = mid - 1;
  }
  const GridJob &j = jobs[lo];
  const int64_t b = g - j.box0;
  if (b < j.n) j.grid[j.key[b]] = (int32_t)b;
}

// One list of one level: far = 1: V list over NOFF slots; far = 0: near list over NNEAR slots; react:
// targets against images (the far list also records the classes in use and sorts the target boxes into
// their rows, box layers k_t = 0 .. 2 ws from the interface).  One block per target box, every list of
// every group in one launch.
struct ListJob {
  const uint64_t *tkey, *skey;
  const int32_t *sgrid;  // dense box index of the source level (nullptr: binary search in skey)
  int64_t nt, ns, box0;
  int lev, far, react, a;
  int32_t *out;
  uint8_t *used;
  int32_t *rows, *ktrow;
  uint32_t *nrows;
};
constexpr int LIST_THREADS = 128;
__global__ void __launch_bounds__(LIST_THREADS) k_lists(const ListJob *jobs, int nj, int ws) {
  int lo = 0, hi = nj - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].box0 <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const ListJob &J = jobs[lo];
  const int64_t t = (int64_t)blockIdx.x - J.box0, ns = J.ns;
  const int nslot = J.far ? NOFF : NNEAR, lev = J.lev, far = J.far, a = J.a;
  const uint64_t *skey = J.skey;
  const int32_t *sgrid = J.sgrid;
  uint8_t *used = J.used;
  int32_t *out = J.out + t * nslot;
  const uint64_t k = J.tkey[t];
  const int ix = compact3(k >> 2), iy = compact3(k >> 1), iz = compact3(k), nc = 1 << lev, half = nc >> 1;
  const int kt = a == 1 ? iz - half : half - 1 - iz;
  const bool react_far = J.react && far;
  if (react_far && threadIdx.x == 0) {
    J.ktrow[t] = kt;
    if (kt >= 0 && kt < 2 * ws + 1) {
      const uint32_t pos = atomicAdd(&J.nrows[kt], 1u);
      J.rows[kt * J.nt + pos] = (int32_t)t;
    }
  }
  // images lie across the interface: a box more than 2 ws layers from it has no image box in reach
  const bool none = ns <= 0 || (J.react && kt > 2 * ws);
  // classes in use are gathered per block and written once where they are new: a global store per found source
  // box kept every block's stores on the same few lines (139,000 leaf boxes of four layers: lists 0.93 -> 0.51 ms)
  __shared__ uint8_t seen[NREACT_CLS];
  if (react_far && !none) {
    for (int e = threadIdx.x; e < NREACT_CLS; e += LIST_THREADS) seen[e] = 0;
    __syncthreads();
  }
  for (int o = threadIdx.x; o < nslot; o += LIST_THREADS) {
    int32_t res = -1;
    if (!none) {
      int dx, dy, dz;
      if (far) off_decode(o, dx, dy, dz);
      else near_decode(o, dx, dy, dz);
      const int jx = ix + dx, jy = iy + dy, jz = iz + dz;
      const int cheb = cheb3(dx, dy, dz);
      bool ok = jx >= 0 && jy >= 0 && jz >= 0 && jx < nc && jy < nc && jz < nc;
      if (far) {
        ok = ok && cheb > ws && abs((jx >> 1) - (ix >> 1)) <= ws && abs((jy >> 1) - (iy >> 1)) <= ws &&
             abs((jz >> 1) - (iz >> 1)) <= ws;
      } else {
        ok = ok && cheb <= ws;
      }
      if (ok) {
        const uint64_t sk = (spread3(jx) << 2) | (spread3(jy) << 1) | spread3(jz);
        const int64_t s = sgrid ? (int64_t)sgrid[sk] : find_key(skey, ns, sk);
        if (s >= 0) {
          res = (int32_t)s;
          if (react_far) {
            const int ks = (a == 1) ? half - 1 - jz : jz - half;
            const int kk = kk_index(kt, ks);
            if (kk >= 0) seen[rho_index(dx, dy) * NKK + kk] = 1;
          }
        }
      }
    }
    out[o] = res;
  }
  if (react_far && !none) {
    __syncthreads();
    for (int e = threadIdx.x; e < NREACT_CLS; e += LIST_THREADS)
      if (seen[e] && !used[e]) used[e] = 1;
  }
}

void build_lists(Ctx &c, std::vector<Group> &groups) {
  std::vector<GridJob> gj;
  std::vector<ListJob> lj;
  int64_t gboxes = 0, lboxes = 0;
  size_t cells = 0, zb = 0;
  // pass 0 sizes the grids and the zeroed records, pass 1 hands them out
  int32_t *grids = nullptr;
  uint8_t *zero = nullptr;
  for (int pass = 0; pass < 2; ++pass) {
    if (pass) {
      grids = c.arena.get<int32_t>(cells);
      zero = c.arena.get<uint8_t>(zb);
      if (cells) LPB_CUDA(cudaMemsetAsync(grids, 0xff, sizeof(int32_t) * cells, c.stream));
      if (zb) LPB_CUDA(cudaMemsetAsync(zero, 0, zb, c.stream));
      cells = zb = 0;
    }
    auto grid = [&](const Level &L, int lev) -> const int32_t * {
      if (lev > GRID_LEV_MAX || !L.n) return nullptr;
      int32_t *g = pass ? grids + cells : nullptr;
      cells += (size_t)1 << (3 * lev);
      if (pass) {
        gj.push_back(GridJob{L.key, g, L.n, gboxes});
        gboxes += L.n;
      }
      return g;
    };
    for (auto &g : groups) {
      const bool fr = g.is_free && (g.parts & 1), re = g.parts & 2;
      const int32_t *tgf = nullptr, *igd = nullptr;  // grids of the leaf levels
      auto list = [&](int lev, const Level &S, const int32_t *sg, int far, int react, int32_t *&out) {
        const Level &T = g.T.lev[lev];
        ListJob j{};
        if (far && react) {
          uint8_t *z = zero + zb;
          zb += (NREACT_CLS + 3) / 4 * 4 + NKT * sizeof(uint32_t);
          zb = (zb + 15) / 16 * 16;
          if (pass) {
            g.used[lev] = j.used = z;
            g.nrows[lev] = j.nrows = (uint32_t *)(z + (NREACT_CLS + 3) / 4 * 4);
            g.rows[lev] = j.rows = c.arena.get<int32_t>((size_t)NKT * T.n);
            g.ktrow[lev] = j.ktrow = c.arena.get<int32_t>(T.n);
          }
        }
        if (!pass) return;
        out = c.arena.get<int32_t>((size_t)T.n * (far ? NOFF : NNEAR));
        j.tkey = T.key; j.skey = S.key; j.sgrid = sg; j.nt = T.n; j.ns = S.n; j.box0 = lboxes;
        j.lev = lev; j.far = far; j.react = react; j.a = g.a; j.out = out;
        lj.push_back(j);
        lboxes += T.n;
      };
      for (int l = 2; l <= g.D; ++l) {
        const Level &T = g.T.lev[l], &I = g.I.lev[l];
        if (!T.n) continue;
        if (fr && l <= g.Df) {
          const int32_t *tg = grid(T, l);
          if (l == g.Df) tgf = tg;
          list(l, T, tg, 1, 0, g.vfree[l]);
        }
        if (re && I.n) {
          const int32_t *ig = grid(I, l);
          if (l == g.D) igd = ig;
          list(l, I, ig, 1, 1, g.vreact[l]);
        }
      }
      if (fr && g.T.lev[g.Df].n) list(g.Df, g.T.lev[g.Df], tgf, 0, 0, g.ufree);
      if (re && g.T.lev[g.D].n && g.I.lev[g.D].n) list(g.D, g.I.lev[g.D], igd, 0, 1, g.ureact);
    }
  }
  if (!gj.empty()) {
    GridJob *dg = c.arena.get<GridJob>(gj.size());
    LPB_CUDA(cudaMemcpyAsync(dg, gj.data(), sizeof(GridJob) * gj.size(), cudaMemcpyHostToDevice, c.stream));
    k_grid_fill<<<(unsigned)((gboxes + 255) / 256), 256, 0, c.stream>>>(dg, (int)gj.size(), gboxes);
    LPB_LAUNCH();
    c.launches++;
  }
  if (!lj.empty()) {
    ListJob *dl = c.arena.get<ListJob>(lj.size());
    LPB_CUDA(cudaMemcpyAsync(dl, lj.data(), sizeof(ListJob) * lj.size(), cudaMemcpyHostToDevice, c.stream));
    k_lists<<<(unsigned)lboxes, LIST_THREADS, 0, c.stream>>>(dl, (int)lj.size(), c.ws);
    LPB_LAUNCH();
    c.launches++;
  }
}

}  // namespace lpb

namespace lpb {

// ---------------------------------------------------------------------------------------
// Adaptive dual-tree lists of a group's free-space target tree with itself (Sec. 3.5 builds the
// method on the adaptive FMM framework; diagnostic for now, the evaluation uses uniform trees).
// A box of level l >= 3 exists in the adaptive tree when its parent exists and holds more than s
// targets (every box of level 2 exists); a box is a leaf when it holds at most s or l = D.  The
// dual traversal starts from every pair of level-2 boxes and runs level-synchronously over
// frontiers of box pairs: a pair that is not near (separation ws: the coarser box grown by ws - 1
// of its sides meets the finer one) is V (same level), W (target leaf, finer source) or X (source
// leaf, finer target); a near pair of two leaves is U; any other near pair is replaced by its
// child pairs (both boxes refined when both have children, else the one that has).
// ---------------------------------------------------------------------------------------
struct APair {
  uint32_t bt, bs;  // box indices in their levels
  int32_t lt, ls;   // levels
};
struct ALevel {
  const uint64_t *key;
  const uint32_t *start, *count, *pcount, *parent;
  const uint8_t *flag;  // bit 0: the box exists in the adaptive tree; bit 1: it is a leaf
  uint32_t n;
};

__global__ void k_adapt_flags(int l, int D, int s, ALevel cur, const uint8_t *pflag, uint8_t *flag) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= cur.n) return;
  bool present = true;
  if (l > 2) {
    const uint8_t pf = pflag[cur.parent[b]];
    present = (pf & 1) && !(pf & 2);
  }
  const bool leaf = present && (cur.pcount[b] <= (uint32_t)s || l == D);
  flag[b] = (uint8_t)((present ? 1 : 0) | (leaf ? 2 : 0));
}

__global__ void k_adapt_init(uint32_t n2, APair *pairs) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n2 * n2) return;
  pairs[i] = APair{(uint32_t)(i / n2), (uint32_t)(i % n2), 2, 2};
}

// boxes (la, ka) and (lb, kb) near for separation ws (integer geometry at the finer level)
__device__ bool adapt_near(int la, uint64_t ka, int lb, uint64_t kb, int ws) {
  const int L = max(la, lb);
  const int64_t sa = (int64_t)1 << (L - la), sb = (int64_t)1 << (L - lb);
  const int64_t ga = la <= lb ? (ws - 1) * sa : 0, gb = lb < la ? (ws - 1) * sb : 0;
  for (int d = 0; d < 3; ++d) {
    const int64_t u = compact3(ka >> (2 - d)), v = compact3(kb >> (2 - d));
    if ((u + 1) * sa + ga < v * sb - gb || (v + 1) * sb + gb < u * sa - ga) return false;
  }
  return true;
}

// classify every frontier pair; nchild[i] = its child pairs (0 when classified).  Records of
// 5 int64: kind (0 V, 1 U, 2 W, 3 X), lt, key t, ls, key s; at most one per pair
__global__ void k_adapt_step(const APair *pairs, uint32_t np, const ALevel *lv, int ws, uint32_t *nchild,
                             int64_t *rec, uint32_t *nrec) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  const APair P = pairs[i];
  const ALevel &T = lv[P.lt], &S = lv[P.ls];
  if (P.bt >= T.n || P.bs >= S.n) {  // cannot happen for pairs built below; checked all the same
    nchild[i] = 0;
    return;
  }
  const uint64_t kt = T.key[P.bt], ks = S.key[P.bs];
  const bool tl = T.flag[P.bt] & 2, sl = S.flag[P.bs] & 2;
  int kind = -1;
  uint32_t nc = 0;
  if (!adapt_near(P.lt, kt, P.ls, ks, ws)) kind = P.lt == P.ls ? 0 : (P.ls > P.lt ? 2 : 3);
  else if (tl && sl) kind = 1;
  else nc = (tl ? 1u : T.count[P.bt]) * (sl ? 1u : S.count[P.bs]);
  nchild[i] = nc;
  if (kind >= 0) {
    const uint32_t r = atomicAdd(nrec, 1u);
    if (r < np) {
      int64_t *o = rec + (size_t)r * 5;
      o[0] = kind; o[1] = P.lt; o[2] = (int64_t)kt; o[3] = P.ls; o[4] = (int64_t)ks;
    }
  }
}

__global__ void k_adapt_children(const APair *pairs, uint32_t np, const ALevel *lv, const uint32_t *nchild,
                                 const uint32_t *off, APair *next, uint32_t cap) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np || !nchild[i]) return;
  const APair P = pairs[i];
  const ALevel &T = lv[P.lt], &S = lv[P.ls];
  const bool tl = T.flag[P.bt] & 2, sl = S.flag[P.bs] & 2;
  const uint32_t nt = tl ? 1u : T.count[P.bt], ns = sl ? 1u : S.count[P.bs];
  for (uint32_t a = 0; a < nt; ++a)
    for (uint32_t b = 0; b < ns; ++b) {
      const uint64_t o = (uint64_t)off[i] + (uint64_t)a * ns + b;
      if (o >= cap) continue;
      next[o] = APair{tl ? P.bt : T.start[P.bt] + a, sl ? P.bs : S.start[P.bs] + b, tl ? P.lt : P.lt + 1,
                      sl ? P.ls : P.ls + 1};
    }
}

void adaptive_lists(Ctx &c, Group &g, int s, int ws, std::vector<int64_t> &rec) {
  rec.clear();
  PointSet &P = g.T;
  const int D = g.Df;
  if (!P.np || D < 2) return;
  // flags, top down
  std::vector<ALevel> hl(DMAX + 1);
  for (int l = 2; l <= D; ++l) {
    const Level &L = P.lev[l];
    uint8_t *f = c.arena.get<uint8_t>((size_t)std::max<int64_t>(L.n, 1));
    hl[l] = ALevel{L.key, L.start, L.count, L.pcount, L.parent, f, (uint32_t)L.n};
    if (L.n)
      k_adapt_flags<<<(unsigned)((L.n + 255) / 256), 256, 0, c.stream>>>(l, D, s, hl[l], l > 2 ? hl[l - 1].flag : nullptr,
                                                                         f);
    LPB_LAUNCH();
  }
  ALevel *dl = c.arena.get<ALevel>(DMAX + 1);
  LPB_CUDA(cudaMemcpyAsync(dl, hl.data(), sizeof(ALevel) * (DMAX + 1), cudaMemcpyHostToDevice, c.stream));
  const uint32_t n2 = (uint32_t)P.lev[2].n;
  uint64_t F = (uint64_t)n2 * n2;
  constexpr uint64_t FMAX = (uint64_t)1 << 26;  // frontier pairs this diagnostic handles
  if (F > FMAX) throw StatusError{LPBFMM_ERR_UNSUPPORTED};
  APair *pairs = c.arena.get<APair>((size_t)std::max<uint64_t>(F, 1));
  if (F) k_adapt_init<<<(unsigned)((F + 255) / 256), 256, 0, c.stream>>>(n2, pairs);
  LPB_LAUNCH();
  uint32_t *hp = (uint32_t *)c.h_pinned;
  for (int step = 0; F > 0; ++step) {
    if (step > 4 * DMAX) throw StatusError{LPBFMM_ERR_UNSUPPORTED};
    uint32_t *nchild = c.arena.get<uint32_t>(F), *off = c.arena.get<uint32_t>(F), *d2 = c.arena.get<uint32_t>(2);
    int64_t *drec = c.arena.get<int64_t>((size_t)F * 5);
    LPB_CUDA(cudaMemsetAsync(d2, 0, 2 * sizeof(uint32_t), c.stream));
    k_adapt_step<<<(unsigned)((F + 255) / 256), 256, 0, c.stream>>>(pairs, (uint32_t)F, dl, ws, nchild, drec, d2);
    LPB_LAUNCH();
    scan_u32(c, nchild, off, (int64_t)F, d2 + 1);
    LPB_CUDA(cudaMemcpyAsync(hp, d2, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, c.stream));
    LPB_CUDA(cudaStreamSynchronize(c.stream));
    const uint32_t nr = std::min<uint64_t>(hp[0], F), nnext = hp[1];
    const size_t base = rec.size();
    rec.resize(base + (size_t)nr * 5);
    if (nr) LPB_CUDA(cudaMemcpy(rec.data() + base, drec, sizeof(int64_t) * nr * 5, cudaMemcpyDeviceToHost));
    if (nnext > FMAX) throw StatusError{LPBFMM_ERR_UNSUPPORTED};
    APair *next = nnext ? c.arena.get<APair>(nnext) : nullptr;
    if (nnext)
      k_adapt_children<<<(unsigned)((F + 255) / 256), 256, 0, c.stream>>>(pairs, (uint32_t)F, dl, nchild, off, next,
                                                                         nnext);
    LPB_LAUNCH();
    pairs = next;
    F = nnext;
  }
  LPB_CUDA(cudaStreamSynchronize(c.stream));
}

}  // namespace lpb
