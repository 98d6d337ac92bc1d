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
// Mean points per segment below which a lane takes a segment; us by warps / by lanes: FP32 (N = 100,000) 8.9 points a segment
// 179 / 406, 6.5: 316 / 507, 1.8: 810 / 452; FP64 (N = 20,000, p = 10; 3,000, p = 12) 13.1: 662 / 947, 11.7: 268 / 1,028, 2.3: 3,480 / 579,
// 2.0: 1,349 / 334.  L2P takes the same line for points per leaf, although a lane per target was the faster form at
// every occupancy measured there (FP32, N = 100,000, 65 points a leaf 48 / 24, 1.8: 203 / 34; FP64, N = 20,000, 104: 538 / 109).
constexpr int P2M_SPARSE = 6;

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
//
// One CTA per parent (M2M: and per source type where parents are few): the operator of a z-half serves its (at most
// four) children, whose columns lie side by side in shared memory.  Rows are real: K real parts by P, then the
// K - p - 1 imaginary parts of m > 0 by Q (the m = 0 ones vanish for real charges).  A thread owns one row of one
// z-half and one of OCT_SPLIT parts of its columns.
// Bound: latency where parents are few, L2 reads of the operators (or the FP64 pipe) where they are many.  A thread per
// row that walked both z-halves of every type in turn took 255 us for the 56 parents of a level, as long as for 448;
// now 16 us.  M2M of three layers N = 1M (p = 10, 56 / 448 / 3,584 parents) 869 -> 209 us, L2L 307 -> 118; four layers
// N = 200,000 (p = 8, 24,576 sparse parents) M2M 2.28 -> 1.28 ms an evaluation, L2L 0.57 -> 0.28.
// ---------------------------------------------------------------------------------------
constexpr int OCT_SPLIT = 2;
// parents of a level up to which each source type takes a CTA of its own; far beyond it the set-up that every CTA
// repeats costs more than the types in turn.  us in turn / apart: FP32 448 parents (p = 10) 57 / 28, 3,584: 158 / 147, 5,120 (p = 8)
// 222 / 200, 26,649 (p = 10) 755 / 827, 40,177 (p = 8) 935 / 1,119; FP64 448 (p = 10) 224 / 161, 3,574: 1,132 / 961, 4,596 (p = 12)
// 921 / 876.  The two meet between 5,000 and 27,000 parents; the line is on the low side of that.
constexpr int M2M_TSPLIT_MAX = 2048;
// CTAs of a level up to which a CTA takes one group of threads per z-half and column part (latency counts);
// beyond it one group does all, so that a half without children idles no threads and more parents are in flight.  us with the
// groups / with one: FP32 (p = 10) 152 CTAs 16 / 29, 384 (L2L, p = 8) 25 / 31, 1,216: 48 / 28, 26,649: 1,424 / 755; FP64 (p = 10) 152 CTAs
// 32 / 82, 384 (L2L, p = 12) 111 / 114, 1,216: 164 / 160, 3,574: 1,053 / 1,110, 4,596 (p = 12) 1,343 / 942.
constexpr int OCT_WIDE = 512;
static __host__ __device__ __forceinline__ int oct_rows(int K, int p) { return (2 * K - (p + 1) + 31) / 32 * 32; }
static int oct_threads(int K, int p, int64_t ctas) {
  const int r = oct_rows(K, p);
  if (ctas > OCT_WIDE) return r;
  return 2 * r * OCT_SPLIT <= 1024 ? 2 * r * OCT_SPLIT : 2 * r;  // p = 16: two parts of 320 rows exceed a block
}
template <typename T>
static size_t oct_smem(int K, int p) {
  const int R = 2 * K - (p + 1);
  return sizeof(T) * ((size_t)R * 8 + 4 * (PMAX + 1) * 2) + sizeof(int) * (R + K);
}
__device__ __forceinline__ void ld4(const float *p, float *v) {
  const float4 a = *(const float4 *)p;
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void ld4(const double *p, double *v) {
  const double2 a = *(const double2 *)p, b = *(const double2 *)(p + 2);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
template <int NJ, typename T>
__device__ __forceinline__ void oct_dot(T *acc, const T *__restrict__ W, const int *row, const T *x, int q0, int q1, int K) {
#pragma unroll 8
  for (int q = q0; q < q1; ++q) {
    const T w = __ldg(W + row[q] * K);
    T v[4];
    if (NJ == 4) ld4(x + q * 8, v);
    else
#pragma unroll
      for (int j = 0; j < NJ; ++j) v[j] = x[q * 8 + j];
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] += w * v[j];
  }
}
// shared state of a CTA: the children's columns, the azimuthal factors of the four (x, y) octants, indices
template <typename T>
struct OctCta {
  T *x;      // [R][8]: row, z-half * 4 + slot
  T *rt;     // [4][PMAX + 1][2]
  int *row;  // [R] coefficient of each real row
  int *nm;   // [K] n | m << 8
  int K, KI;
  __device__ __forceinline__ OctCta(unsigned char *sm, const T *rot4, int K_, int p) : K(K_), KI(K_ - (p + 1)) {
    const int R = K + KI;
    x = (T *)sm;
    rt = x + R * 8;
    row = (int *)(rt + 4 * (PMAX + 1) * 2);
    nm = row + R;
    for (int e = threadIdx.x; e < 4 * (PMAX + 1) * 2; e += blockDim.x) rt[e] = rot4[e];
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
      int n = (int)((sqrtf(8.0f * (float)k + 1.0f) - 1.0f) * 0.5f);
      while (n * (n + 1) / 2 > k) --n;
      while ((n + 1) * (n + 2) / 2 <= k) ++n;
      const int m = k - n * (n + 1) / 2;
      nm[k] = n | m << 8;
      row[k] = k;
      if (m) row[K + k - n - 1] = k;  // k - n - 1: position among the m > 0 coefficients
    }
  }
  __device__ __forceinline__ void put(int k, int dir, int slot, T re, T im) {  // rotated into the operator's frame
    const int n = nm[k] & 255, m = nm[k] >> 8;
    const T cs = rt[(dir * (PMAX + 1) + m) * 2], sn = rt[(dir * (PMAX + 1) + m) * 2 + 1];
    x[k * 8 + slot] = cs * re - sn * im;
    if (m) x[(K + k - n - 1) * 8 + slot] = sn * re + cs * im;
  }
  __device__ __forceinline__ void add(int k, int dir, int slot, T &re, T &im) const {  // rotated back
    const int n = nm[k] & 255, m = nm[k] >> 8;
    const T cs = rt[(dir * (PMAX + 1) + m) * 2], sn = rt[(dir * (PMAX + 1) + m) * 2 + 1];
    const T yr = x[k * 8 + slot], yi = m ? x[(K + k - n - 1) * 8 + slot] : (T)0;
    re += cs * yr + sn * yi;
    im += cs * yi - sn * yr;
  }
  // x <- [P 0; 0 Q] x for the n0, n1 slots in use of the two z-halves; ops: [z-half][P, Q][K][K].  A group of threads
  // (one per row) takes one z-half and one part of the columns, or, where it is the only one, all of both.
  __device__ __forceinline__ void product(const T *ops, int n0, int n1) {
    const int R = K + KI, Rp = (R + 31) / 32 * 32, grp = threadIdx.x / Rp, r = threadIdx.x - grp * Rp;
    const int ngrp = blockDim.x / Rp, parts = ngrp > 1 ? ngrp >> 1 : 1, part = grp >> 1;
    const int im = r >= K;
    T acc[2][4] = {};
    if (r < R) {
      const int len = im ? KI : K, per = (len + parts - 1) / parts, b = im ? K : 0;
      const int q0 = b + part * per, q1 = b + min(len, (part + 1) * per);
#pragma unroll
      for (int cz = 0; cz < 2; ++cz) {
        const int n = cz ? n1 : n0;
        if (n == 0 || (ngrp > 1 && (grp & 1) != cz)) continue;
        const T *W = ops + (size_t)(cz * 2 + im) * K * K + row[r];
        if (n == 1) oct_dot<1>(acc[cz], W, row, x + cz * 4, q0, q1, K);
        else if (n == 2) oct_dot<2>(acc[cz], W, row, x + cz * 4, q0, q1, K);
        else oct_dot<4>(acc[cz], W, row, x + cz * 4, q0, q1, K);  // a fourth, unused slot is not read back
      }
    }
    for (int t = 0; t < parts; ++t) {
      __syncthreads();
      if (r >= R || part != t) continue;
#pragma unroll
      for (int cz = 0; cz < 2; ++cz) {
        const int n = cz ? n1 : n0;
        if (ngrp > 1 && (grp & 1) != cz) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < n) x[r * 8 + cz * 4 + j] = t ? x[r * 8 + cz * 4 + j] + acc[cz][j] : acc[cz][j];
      }
    }
    __syncthreads();
  }
};
// slot of child c among the children in `have` (bit per child; zm: bit set for the upper z-half)
__device__ __forceinline__ int oct_slot(uint32_t have, uint32_t zm, int c) {
  const int cz = (zm >> c) & 1;
  return cz * 4 + __popc(have & (cz ? zm : ~zm) & ((1u << c) - 1u));
}

// A box holds an expansion of type t if bit t of its mask is set; other rows are neither written nor read.
// tsplit CTAs share the types present in a parent.
struct M2MJob {
  const uint32_t *pstart, *pcount;  // children of every parent
  const uint64_t *ckey;
  const uint32_t *pmask, *cmask;    // types present (null: type 0 everywhere)
  const void *Mc, *ops;
  void *Mp;
  int64_t np, item0;
  int ntypes, tsplit;
};
template <typename T>
__global__ void __launch_bounds__(1024) k_m2m(const M2MJob *jobs, int nj, const T *rot4, int K, int p) {
  typedef typename C2<T>::t T2;
  extern __shared__ __align__(16) unsigned char oct_sm[];
  __shared__ uint32_t cm_s[8];
  __shared__ uint32_t oc_s[8];
  const M2MJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int64_t it = (int64_t)blockIdx.x - J.item0, box = it / J.tsplit;
  const int part = (int)(it - box * J.tsplit);
  if (box >= J.np) return;
  uint32_t todo = J.pmask ? J.pmask[box] : 1u;
  if (__popc(todo) <= part) return;
  const int ntypes = J.ntypes;
  const uint32_t c0 = J.pstart[box], nc = min(J.pcount[box], 8u);
  OctCta<T> S(oct_sm, rot4, K, p);
  if (threadIdx.x < 8) {
    const bool in = threadIdx.x < nc;
    oc_s[threadIdx.x] = in ? (uint32_t)(J.ckey[c0 + threadIdx.x] & 7ull) : 0u;
    cm_s[threadIdx.x] = in ? (J.cmask ? J.cmask[c0 + threadIdx.x] : 1u) : 0u;
  }
  const T2 *Mc = (const T2 *)J.Mc;
  for (int w = 0; todo; todo &= todo - 1, ++w) {
    if (w % J.tsplit != part) continue;
    const int type = __ffs(todo) - 1;
    __syncthreads();
    uint32_t have = 0, zm = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      have |= ((cm_s[c] >> type) & 1u) << c;
      zm |= (oc_s[c] & 1u) << c;
    }
    for (uint32_t e = threadIdx.x; e < nc * (uint32_t)K; e += blockDim.x) {
      const int c = (int)(e / K), k = (int)(e - c * K);
      if (!((have >> c) & 1u)) continue;
      const T2 v = Mc[((size_t)(c0 + c) * ntypes + type) * K + k];
      S.put(k, oc_s[c] >> 1, oct_slot(have, zm, c), v.x, v.y);
    }
    __syncthreads();
    S.product((const T *)J.ops + (size_t)type * 4 * K * K, __popc(have & ~zm), __popc(have & zm));
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      T ar = 0, ai = 0;
      for (int c = 0; c < (int)nc; ++c)
        if ((have >> c) & 1u) S.add(i, oc_s[c] >> 1, oct_slot(have, zm, c), ar, ai);
      ((T2 *)J.Mp)[((size_t)box * ntypes + type) * K + i] = T2{ar, ai};
    }
  }
}

struct L2LJob {
  const uint32_t *pstart, *pcount;  // children of every parent
  const uint64_t *ckey;
  const void *Lp, *ops;
  void *Lc;
  int64_t np, item0;
};
template <typename T>
__global__ void __launch_bounds__(1024) k_l2l(const L2LJob *jobs, int nj, const T *rot4, int K, int p) {
  typedef typename C2<T>::t T2;
  extern __shared__ __align__(16) unsigned char oct_sm[];
  __shared__ uint32_t oc_s[8];
  const L2LJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int64_t box = (int64_t)blockIdx.x - J.item0;
  if (box >= J.np) return;
  const uint32_t c0 = J.pstart[box], nc = min(J.pcount[box], 8u);
  OctCta<T> S(oct_sm, rot4, K, p);
  if (threadIdx.x < 8) oc_s[threadIdx.x] = threadIdx.x < nc ? (uint32_t)(J.ckey[c0 + threadIdx.x] & 7ull) : 0u;
  __syncthreads();
  const uint32_t have = (1u << nc) - 1u;
  uint32_t zm = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) zm |= (oc_s[c] & 1u) << c;
  const T2 *Lp = (const T2 *)J.Lp + (size_t)box * K;
  for (uint32_t e = threadIdx.x; e < nc * (uint32_t)K; e += blockDim.x) {
    const int c = (int)(e / K), k = (int)(e - c * K);
    const T2 v = Lp[k];
    S.put(k, oc_s[c] >> 1, oct_slot(have, zm, c), v.x, v.y);
  }
  __syncthreads();
  S.product((const T *)J.ops, __popc(have & ~zm), __popc(have & zm));
  for (uint32_t e = threadIdx.x; e < nc * (uint32_t)K; e += blockDim.x) {
    const int c = (int)(e / K), k = (int)(e - c * K);
    T2 &dst = ((T2 *)J.Lc)[(size_t)(c0 + c) * K + k];
    T re = dst.x, im = dst.y;
    S.add(k, oc_s[c] >> 1, oct_slot(have, zm, c), re, im);
    dst = T2{re, im};
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
