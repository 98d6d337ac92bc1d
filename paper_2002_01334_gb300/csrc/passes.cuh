// Upward and downward passes (included by fmm.cu): P2M, M2M, L2L, L2P of every target group.  One
// launch per pass and level for all groups (job records, a block finds its job by the first work item);
// group by group they were a chain of small launches.
#pragma once

template <typename J>
__device__ __forceinline__ const J &job_of(const J *jobs, int nj, int64_t item) {
  int lo = 0, hi = nj - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].item0 <= item) lo = mid; else hi = mid - 1;
  }
  return jobs[lo];
}
template <typename J>
static const J *upload_jobs(Ctx &c, const std::vector<J> &jobs) {
  J *d = c.arena.get<J>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(d, jobs.data(), sizeof(J) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
  return d;
}

// ---------------------------------------------------------------------------------------
// P2M.  A segment is the points of one (leaf box, source type).
//   k_p2m: one warp per segment, a lane per point; the coefficients of 32 points are summed over the lanes by
//     halving exchanges of 32 values at a time (31 shuffles for 32 sums; a butterfly per value took 160 and
//     was the kernel's bound).
//   k_p2m_sparse: one lane per segment, for trees whose segments hold a few points (a warp per segment ran
//     with one or two lanes in work there: N = 200,000 four layers, 1.9 points a segment).
// ---------------------------------------------------------------------------------------
struct P2MJob {
  const uint32_t *sst, *scnt, *sbox, *styp;  // segments (sbox, styp null: box = segment, type 0)
  int64_t nseg, item0;                       // item0: first block
  int ntypes;
  const uint64_t *bkey;
  const double *x, *y, *z, *q;
  Geo geo;
  double lam[2 * MAXLAYER];                  // per type
  void *M;
};
constexpr int P2M_SPARSE = 6;  // mean points per segment below which a lane takes a segment

template <typename T>
__device__ __forceinline__ T halve(T a, T b, bool hi, int o) {  // hi lanes keep b, the others a; the rest is exchanged
  const T send = hi ? a : b, keep = hi ? b : a;
  return keep + __shfl_xor_sync(0xffffffffu, send, o);
}

template <typename T, int PT>
__global__ void __launch_bounds__(128) k_p2m(const P2MJob *jobs, int nj, int p, int K) {
  typedef typename C2<T>::t T2;
  constexpr int NV = (PT + 1) * (PT + 2), NB = (NV + 31) / 32;  // values (Re, Im), m outer, n inner; blocks of 32
  const P2MJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t seg = ((int64_t)blockIdx.x - J.item0) * 4 + warp;
  if (seg >= J.nseg) return;
  const uint32_t st = J.sst[seg], cnt = J.scnt[seg];
  const uint32_t box = J.sbox ? J.sbox[seg] : (uint32_t)seg;
  const uint32_t type = J.styp ? J.styp[seg] : 0u;
  double cx, cy, cz;
  box_center(J.bkey[box], J.geo, cx, cy, cz);
  const double ih = 1.0 / J.geo.h;
  const T lh = (T)(J.lam[type] * J.geo.h);
  T acc[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) acc[b] = T(0);
  for (uint32_t b0 = 0; b0 < cnt; b0 += 32) {
    const uint32_t j = b0 + lane;
    const bool valid = j < cnt;
    const uint32_t k = st + (valid ? j : 0);
    const T rx = (T)((J.x[k] - cx) * ih), ry = (T)((J.y[k] - cy) * ih), rz = (T)((J.z[k] - cz) * ih);
    const T qq = valid ? (T)(J.q[k] * 4.0 * PI) : T(0);
    const T r2 = rx * rx + ry * ry + rz * rz;
    T it[PT + 2];
    itilde_all<T, PT + 1>(lh * lh * r2, it);
    T2 Rmm = T2{(T)(0.5 / sqrt(PI)), T(0)};
    T v[32];
    int at = 0;
    auto push = [&](T val) {
      v[at & 31] = val;
      ++at;
      if ((at & 31) == 0 || at == NV) {
        const int blk = (at - 1) >> 5;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i > ((at - 1) & 31)) v[i] = T(0);
#pragma unroll
        for (int o = 16; o; o >>= 1)
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (i < o) v[i] = halve(v[i], v[i + o], (lane & o) != 0, o);
        acc[blk] += v[0];  // lane L: value 32 blk + L
      }
    };
#pragma unroll
    for (int m = 0; m <= PT; ++m) {
      if (m > 0) {
        const T s = CK<T>::sect(m);
        const T2 t = T2{Rmm.x * rx - Rmm.y * ry, Rmm.x * ry + Rmm.y * rx};
        Rmm = T2{s * t.x, s * t.y};
      }
      T2 p1 = T2{0, 0}, p2 = T2{0, 0};
#pragma unroll
      for (int n = m; n <= PT; ++n) {
        T2 R;
        if (n == m) R = Rmm;
        else if (n == m + 1) { const T s = CK<T>::sub(m) * rz; R = T2{s * p1.x, s * p1.y}; }
        else {
          const T a = CK<T>::A(n, m) * rz, b = CK<T>::B(n, m) * r2;
          R = T2{a * p1.x - b * p2.x, a * p1.y - b * p2.y};
        }
        p2 = p1;
        p1 = R;
        const T c = qq * it[n];
        push(c * R.x);
        push(-c * R.y);
      }
    }
  }
  T *out = (T *)((T2 *)J.M + ((size_t)box * J.ntypes + type) * K);
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int val = 32 * b + lane;
    int e = val >> 1, m = 0;
    while (m <= PT && e >= PT + 1 - m) e -= PT + 1 - m++;
    const int n = m + e;
    if (val < NV && n <= p) out[2 * hidx(n, m) + (val & 1)] = acc[b];
  }
}

template <typename T, int PT>
__global__ void __launch_bounds__(128) k_p2m_sparse(const P2MJob *jobs, int nj, int p, int K) {
  typedef typename C2<T>::t T2;
  const P2MJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int64_t seg = ((int64_t)blockIdx.x - J.item0) * 128 + threadIdx.x;
  if (seg >= J.nseg) return;
  const uint32_t st = J.sst[seg], cnt = J.scnt[seg];
  const uint32_t box = J.sbox ? J.sbox[seg] : (uint32_t)seg;
  const uint32_t type = J.styp ? J.styp[seg] : 0u;
  double cx, cy, cz;
  box_center(J.bkey[box], J.geo, cx, cy, cz);
  const double ih = 1.0 / J.geo.h;
  const T lh = (T)(J.lam[type] * J.geo.h);
  T2 *out = (T2 *)J.M + ((size_t)box * J.ntypes + type) * K;
  for (uint32_t j = 0; j < cnt; ++j) {
    const uint32_t k = st + j;
    const T rx = (T)((J.x[k] - cx) * ih), ry = (T)((J.y[k] - cy) * ih), rz = (T)((J.z[k] - cz) * ih);
    const T qq = (T)(J.q[k] * 4.0 * PI);
    const T r2 = rx * rx + ry * ry + rz * rz;
    T it[PT + 2];
    itilde_all<T, PT + 1>(lh * lh * r2, it);
    T2 Rmm = T2{(T)(0.5 / sqrt(PI)), T(0)};
#pragma unroll
    for (int m = 0; m <= PT; ++m) {
      if (m > p) break;
      if (m > 0) {
        const T s = CK<T>::sect(m);
        const T2 t = T2{Rmm.x * rx - Rmm.y * ry, Rmm.x * ry + Rmm.y * rx};
        Rmm = T2{s * t.x, s * t.y};
      }
      T2 p1 = T2{0, 0}, p2 = T2{0, 0};
#pragma unroll
      for (int n = m; n <= PT; ++n) {
        if (n > p) break;
        T2 R;
        if (n == m) R = Rmm;
        else if (n == m + 1) { const T s = CK<T>::sub(m) * rz; R = T2{s * p1.x, s * p1.y}; }
        else {
          const T a = CK<T>::A(n, m) * rz, b = CK<T>::B(n, m) * r2;
          R = T2{a * p1.x - b * p2.x, a * p1.y - b * p2.y};
        }
        p2 = p1;
        p1 = R;
        const T c = qq * it[n];
        T2 &d = out[hidx(n, m)];
        if (j == 0) d = T2{c * R.x, -c * R.y};
        else d = T2{d.x + c * R.x, d.y - c * R.y};
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// M2M (children -> parent) and L2L (parent -> child): azimuth-factored dense operators, stored with
// the output row fastest so that a warp's operator reads coalesce.
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void rot_of_octant(uint64_t ckey, int m, const T *rot4, T &c, T &s) {
  const int oct = (int)(ckey & 7ull);
  const int dir = ((oct >> 2) & 1) * 2 + ((oct >> 1) & 1);
  c = rot4[(dir * (PMAX + 1) + m) * 2];
  s = rot4[(dir * (PMAX + 1) + m) * 2 + 1];
}

// One CTA per parent: for every source type present in it (pmask; a box holds an expansion of type t if bit t
// of its mask is set, other rows are neither written nor read), all children's rotated
// multipoles are staged at once; a thread owns an output row, reads each operator entry once per z-half
// (child octant bit cz) and applies it to the (at most four) children with that cz.
struct M2MJob {
  const uint32_t *pstart, *pcount;  // children of every parent
  const uint64_t *ckey;
  const uint32_t *pmask, *cmask;    // types present (null: type 0 everywhere)
  const void *Mc, *ops;
  void *Mp;
  int64_t np, item0;
  int ntypes;
};
template <typename T>
__global__ void k_m2m(const M2MJob *jobs, int nj, const T *rot4, int K) {
  typedef typename C2<T>::t T2;
  __shared__ T xr[8][KHALF_MAX], xi[8][KHALF_MAX];
  __shared__ uint64_t ck_s[8];
  __shared__ uint32_t cm_s[8];
  const M2MJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int64_t box = (int64_t)blockIdx.x - J.item0;
  if (box >= J.np) return;
  const size_t KK = (size_t)K * K;
  const int ntypes = J.ntypes;
  const uint32_t c0 = J.pstart[box], nc = min(J.pcount[box], 8u);
  if (threadIdx.x < nc) {
    ck_s[threadIdx.x] = J.ckey[c0 + threadIdx.x];
    cm_s[threadIdx.x] = J.cmask ? J.cmask[c0 + threadIdx.x] : 1u;
  }
  const T2 *Mc = (const T2 *)J.Mc;
  for (uint32_t todo = J.pmask ? J.pmask[box] : 1u; todo; todo &= todo - 1) {
    const int type = __ffs(todo) - 1;
    __syncthreads();
    // children of the type, by z-half
    int slot[2][4], ns[2] = {0, 0};
#pragma unroll
    for (int j = 0; j < 4; ++j) slot[0][j] = slot[1][j] = 0;
    for (uint32_t c = 0; c < nc; ++c)
      if ((cm_s[c] >> type) & 1u) {
#pragma unroll
        for (int cz = 0; cz < 2; ++cz) {
          if ((int)(ck_s[c] & 1ull) != cz) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j >= ns[cz]) slot[cz][j] = (int)c;  // unfilled slots repeat the last child
          ++ns[cz];
        }
      }
    for (uint32_t e = threadIdx.x; e < nc * (uint32_t)K; e += blockDim.x) {
      const int c = (int)(e / K), k = (int)(e % K);
      if (!((cm_s[c] >> type) & 1u)) continue;
      T cs, sn;
      rot_of_octant(ck_s[c], cK.mof[k], rot4, cs, sn);
      const T2 v = Mc[((size_t)(c0 + c) * ntypes + type) * K + k];
      xr[c][k] = cs * v.x - sn * v.y;
      xi[c][k] = sn * v.x + cs * v.y;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      const int m = cK.mof[i];
      T ar = 0, ai = 0;
#pragma unroll
      for (int cz = 0; cz < 2; ++cz) {
        const int n = ns[cz];
        if (n == 0) continue;
        const T *P = (const T *)J.ops + ((size_t)type * 2 + cz) * 2 * KK + i, *Q = P + KK;
        T yr[4] = {0, 0, 0, 0}, yi[4] = {0, 0, 0, 0};
        if (n == 1) {
          const T *x0 = xr[slot[cz][0]], *x1 = xi[slot[cz][0]];
#pragma unroll 4
          for (int k = 0; k < K; ++k) {
            yr[0] += P[(size_t)k * K] * x0[k];
            yi[0] += Q[(size_t)k * K] * x1[k];
          }
        } else {
#pragma unroll 2
          for (int k = 0; k < K; ++k) {
            const T pv = P[(size_t)k * K], qv = Q[(size_t)k * K];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              yr[j] += pv * xr[slot[cz][j]][k];
              yi[j] += qv * xi[slot[cz][j]][k];
            }
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j >= n) break;
          T cs, sn;
          rot_of_octant(ck_s[slot[cz][j]], m, rot4, cs, sn);
          ar += cs * yr[j] + sn * yi[j];
          ai += cs * yi[j] - sn * yr[j];
        }
      }
      ((T2 *)J.Mp)[((size_t)box * ntypes + type) * K + i] = T2{ar, ai};
    }
  }
}

struct L2LJob {
  const uint32_t *cparent;
  const uint64_t *ckey;
  const void *Lp, *ops;
  void *Lc;
  int64_t nc, item0;
};
template <typename T>
__global__ void k_l2l(const L2LJob *jobs, int nj, const T *rot4, int K) {
  typedef typename C2<T>::t T2;
  __shared__ T xr[KHALF_MAX], xi[KHALF_MAX];
  const L2LJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int64_t c = (int64_t)blockIdx.x - J.item0;
  if (c >= J.nc) return;
  const uint64_t ck = J.ckey[c];
  const int cz = (int)(ck & 1ull);
  const size_t KK = (size_t)K * K;
  const T *P = (const T *)J.ops + (size_t)cz * 2 * KK, *Q = P + KK;
  const uint32_t par = J.cparent[c];
  const T2 *Lp = (const T2 *)J.Lp;
  for (int e = threadIdx.x; e < K; e += blockDim.x) {
    T cs, sn;
    rot_of_octant(ck, cK.mof[e], rot4, cs, sn);
    const T2 v = Lp[(size_t)par * K + e];
    xr[e] = cs * v.x - sn * v.y;
    xi[e] = sn * v.x + cs * v.y;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    T yr = 0, yi = 0;
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      yr += P[(size_t)k * K + i] * xr[k];
      yi += Q[(size_t)k * K + i] * xi[k];
    }
    T cs, sn;
    rot_of_octant(ck, cK.mof[i], rot4, cs, sn);
    T2 &dst = ((T2 *)J.Lc)[(size_t)c * K + i];
    dst.x += cs * yr + sn * yi;
    dst.y += cs * yi - sn * yr;
  }
}

// ---------------------------------------------------------------------------------------
// L2P with field: one warp per leaf box, or (SPARSE) one lane per target where leaves hold a few
// ---------------------------------------------------------------------------------------
struct L2PJob {
  const uint64_t *bkey;
  const uint32_t *bstart, *bcount, *pbox;  // leaf ranges; leaf of every point
  const double *x, *y, *z;
  const uint32_t *src;
  const void *L;
  Geo geo;
  double lam;
  int64_t n, item0;  // boxes (SPARSE: points); first block
};
template <typename T, int PT, bool SPARSE>
__global__ void __launch_bounds__(128) k_l2p(const L2PJob *jobs, int nj, int p, int K, double *phi, double *field) {
  typedef typename C2<T>::t T2;
  __shared__ T2 Ls[SPARSE ? 1 : 4][KHALF_MAX];
  const L2PJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t item = ((int64_t)blockIdx.x - J.item0) * (SPARSE ? 128 : 4) + (SPARSE ? (int)threadIdx.x : warp);
  if (item >= J.n) return;
  const int64_t box = SPARSE ? (int64_t)J.pbox[item] : item;
  const T2 *Lw = (const T2 *)J.L + (size_t)box * K;
  if (!SPARSE) {
    for (int e = lane; e < K; e += 32) Ls[warp][e] = Lw[e];
    __syncwarp();
    Lw = Ls[warp];
  }
  double cx, cy, cz;
  box_center(J.bkey[box], J.geo, cx, cy, cz);
  const double lam = J.lam, h = J.geo.h, ih = 1.0 / h;
  const T lh = (T)(lam * h);
  const uint32_t st = SPARSE ? (uint32_t)item : J.bstart[box], cnt = SPARSE ? 1u : J.bcount[box];
  for (uint32_t j = SPARSE ? 0 : lane; j < cnt; j += 32) {
    const uint32_t k = st + j;
    const T rx = (T)((J.x[k] - cx) * ih), ry = (T)((J.y[k] - cy) * ih), rz = (T)((J.z[k] - cz) * ih);
    const T r2 = rx * rx + ry * ry + rz * rz;
    T it[PT + 3];
    itilde_all<T, PT + 2>(lh * lh * r2, it);
    T ph = 0, S1 = 0, Gz = 0, Gpr = 0, Gpi = 0;
    T2 Rmm = T2{(T)(0.5 / sqrt(PI)), T(0)};
#pragma unroll
    for (int m = 0; m <= PT; ++m) {
      if (m > p) break;
      if (m > 0) {
        const T s = CK<T>::sect(m);
        const T2 t = T2{Rmm.x * rx - Rmm.y * ry, Rmm.x * ry + Rmm.y * rx};
        Rmm = T2{s * t.x, s * t.y};
      }
      const T wm = m ? T(2) : T(1);
      T2 p1 = T2{0, 0}, p2 = T2{0, 0};
#pragma unroll
      for (int n = m; n <= PT; ++n) {
        if (n > p) break;
        T2 R;
        if (n == m) R = Rmm;
        else if (n == m + 1) { const T s = CK<T>::sub(m) * rz; R = T2{s * p1.x, s * p1.y}; }
        else {
          const T a = CK<T>::A(n, m) * rz, b = CK<T>::B(n, m) * r2;
          R = T2{a * p1.x - b * p2.x, a * p1.y - b * p2.y};
        }
        p2 = p1;
        p1 = R;
        const T2 Lnm = Lw[hidx(n, m)];
        const T re = Lnm.x * R.x - Lnm.y * R.y;
        ph += wm * it[n] * re;
        S1 += wm * it[n + 1] / T(2 * n + 3) * re;
        if (n < p) {
          const T in1 = it[n + 1];
          const T2 Lz = Lw[hidx(n + 1, m)];
          Gz += wm * in1 * CK<T>::gz(n, m) * (Lz.x * R.x - Lz.y * R.y);
          if (m >= 1) {
            const T2 La = Lw[hidx(n + 1, m - 1)];
            const T ca = in1 * CK<T>::ga(n, m);
            Gpr += ca * (La.x * R.x - La.y * R.y);
            Gpi += ca * (La.x * R.y + La.y * R.x);
          }
          const T2 Lb = Lw[hidx(n + 1, m + 1)];
          const T cb = in1 * CK<T>::gb(n, m);
          // - conj(Lb R)
          Gpr -= cb * (Lb.x * R.x - Lb.y * R.y);
          Gpi += cb * (Lb.x * R.y + Lb.y * R.x);
        }
      }
    }
    const uint32_t i = J.src[k];
    phi[i] += (double)ph;
    if (field) {
      const double l2h = lam * lam * h;  // lambda^2 r = lambda^2 h r_u
      field[3 * (size_t)i] -= l2h * (double)rx * (double)S1 + (double)Gpr * ih;
      field[3 * (size_t)i + 1] -= l2h * (double)ry * (double)S1 + (double)Gpi * ih;
      field[3 * (size_t)i + 2] -= l2h * (double)rz * (double)S1 + (double)Gz * ih;
    }
  }
}
