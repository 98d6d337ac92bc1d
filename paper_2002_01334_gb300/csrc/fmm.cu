// FMM passes of one target group (Algorithm 1 for the reaction components of group (l, a),
// the free-space Yukawa FMM of layer l when the group carries it, Algorithm 2 around them):
// P2M, M2M, M2L (free + reaction), L2L, L2P with field, near-field P2P.
// Expansions use the half representation (m >= 0) and the scaling described in ops.cu:
//   M~_nm = sum_j q_j 4 pi itilde_n(lambda r_j) conj(R_n^m(r_j / h)),
//   phi(r) = sum_n [L~_n0 itilde_n R_n^0 + 2 Re sum_{m>0} L~_nm itilde_n R_n^m](r / h).
#include "internal.h"
#include "tc.cuh"

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>

namespace lpb {

// recurrence and gradient constants (index [n][m], n <= PMAX + 1)
struct Consts {
  double A[PMAX + 2][PMAX + 2], B[PMAX + 2][PMAX + 2];
  double sect[PMAX + 2], sub[PMAX + 2];
  double gz[PMAX + 2][PMAX + 2], ga[PMAX + 2][PMAX + 2], gb[PMAX + 2][PMAX + 2];
  int mof[KHALF_MAX];
};
__constant__ Consts cK;
// FP32 copies of the recurrence constants: the FP32 kernels read these directly (a conversion
// from FP64 runs on the FP64 pipe, ~2 lanes per clock per SM on this GPU)
struct ConstsF {
  float A[PMAX + 2][PMAX + 2], B[PMAX + 2][PMAX + 2];
  float sect[PMAX + 2], sub[PMAX + 2];
  float gz[PMAX + 2][PMAX + 2], ga[PMAX + 2][PMAX + 2], gb[PMAX + 2][PMAX + 2];
};
__constant__ ConstsF cKf;
template <typename T> struct CK;
template <> struct CK<float> {
  static __device__ __forceinline__ float A(int n, int m) { return cKf.A[n][m]; }
  static __device__ __forceinline__ float B(int n, int m) { return cKf.B[n][m]; }
  static __device__ __forceinline__ float sect(int m) { return cKf.sect[m]; }
  static __device__ __forceinline__ float sub(int m) { return cKf.sub[m]; }
  static __device__ __forceinline__ float gz(int n, int m) { return cKf.gz[n][m]; }
  static __device__ __forceinline__ float ga(int n, int m) { return cKf.ga[n][m]; }
  static __device__ __forceinline__ float gb(int n, int m) { return cKf.gb[n][m]; }
};
template <> struct CK<double> {
  static __device__ __forceinline__ double A(int n, int m) { return cK.A[n][m]; }
  static __device__ __forceinline__ double B(int n, int m) { return cK.B[n][m]; }
  static __device__ __forceinline__ double sect(int m) { return cK.sect[m]; }
  static __device__ __forceinline__ double sub(int m) { return cK.sub[m]; }
  static __device__ __forceinline__ double gz(int n, int m) { return cK.gz[n][m]; }
  static __device__ __forceinline__ double ga(int n, int m) { return cK.ga[n][m]; }
  static __device__ __forceinline__ double gb(int n, int m) { return cK.gb[n][m]; }
};

void upload_consts(cudaStream_t s) {
  static Consts h;
  for (int n = 0; n <= PMAX + 1; ++n)
    for (int m = 0; m <= PMAX + 1; ++m) {
      h.A[n][m] = h.B[n][m] = h.gz[n][m] = h.ga[n][m] = h.gb[n][m] = 0.0;
      if (m <= n && n >= m + 2) {
        h.A[n][m] = sqrt((4.0 * n * n - 1.0) / (double(n) * n - double(m) * m));
        h.B[n][m] = sqrt(((n - 1.0) * (n - 1.0) - double(m) * m) * (2.0 * n + 1.0) /
                         ((2.0 * n - 3.0) * (double(n) * n - double(m) * m)));
      }
      if (m <= n) {
        const double c1 = sqrt((2.0 * (n + 1) + 1.0) / (2.0 * (n + 1) - 1.0));
        h.gz[n][m] = c1 * sqrt(double(n + 1 + m) * (n + 1 - m));
        h.ga[n][m] = c1 * sqrt(double(n + 2 - m) * (n + 1 - m));
        h.gb[n][m] = c1 * sqrt(double(n + 2 + m) * (n + 1 + m));
      }
    }
  for (int m = 0; m <= PMAX + 1; ++m) {
    h.sect[m] = m ? -sqrt((2.0 * m + 1.0) / (2.0 * m)) : 1.0;
    h.sub[m] = sqrt(2.0 * m + 3.0);
  }
  for (int n = 0; n <= PMAX; ++n)
    for (int m = 0; m <= n; ++m) h.mof[hidx(n, m)] = m;
  LPB_CUDA(cudaMemcpyToSymbolAsync(cK, &h, sizeof(Consts), 0, cudaMemcpyHostToDevice, s));
  static ConstsF hf;
  for (int n = 0; n <= PMAX + 1; ++n) {
    for (int m = 0; m <= PMAX + 1; ++m) {
      hf.A[n][m] = (float)h.A[n][m];
      hf.B[n][m] = (float)h.B[n][m];
      hf.gz[n][m] = (float)h.gz[n][m];
      hf.ga[n][m] = (float)h.ga[n][m];
      hf.gb[n][m] = (float)h.gb[n][m];
    }
    hf.sect[n] = (float)h.sect[n];
    hf.sub[n] = (float)h.sub[n];
  }
  LPB_CUDA(cudaMemcpyToSymbolAsync(cKf, &hf, sizeof(ConstsF), 0, cudaMemcpyHostToDevice, s));
  LPB_CUDA(cudaStreamSynchronize(s));
}

template <typename T> struct C2;
template <> struct C2<float> { typedef float2 t; };
template <> struct C2<double> { typedef double2 t; };

struct Geo {
  double o[3];  // lower corner of the root cube
  double h;     // box size at the level
};

__device__ __forceinline__ uint32_t compact3_(uint64_t x) {
  x &= 0x9249249ull;
  x = (x ^ (x >> 2)) & 0x30c30c3ull;
  x = (x ^ (x >> 4)) & 0x300f00full;
  x = (x ^ (x >> 8)) & 0x30000ffull;
  x = (x ^ (x >> 16)) & 0x3ffull;
  return (uint32_t)x;
}
__device__ __forceinline__ void box_center(uint64_t key, const Geo &g, double &cx, double &cy, double &cz) {
  cx = g.o[0] + (compact3_(key >> 2) + 0.5) * g.h;
  cy = g.o[1] + (compact3_(key >> 1) + 0.5) * g.h;
  cz = g.o[2] + (compact3_(key) + 0.5) * g.h;
}

template <typename T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

#include "passes.cuh"

// ---------------------------------------------------------------------------------------
// M2L: one launch for every (group, level, free / reaction row) job.  A work item is
// (job, tile of target boxes, slice dx of the NOFF offsets).  For every offset of its slice
// the class operator (P, Q) and the phase-rotated multipoles of the tile's sources are staged
// in shared memory in K-chunks and multiplied as a small GEMM (rows = output coefficients,
// columns = target boxes); each target's partial local expansion of the slice is written to
// its own slot [box][slot] and the slots are summed in a fixed order (k_m2l_reduce), so the
// result does not depend on scheduling.  (Mixed mode with p > 11; k_m2l_f32 serves p = 11, k_m2l_tc
// p <= 10, and the FP64 mode runs the operator-sorted lists of m2l_pairs.cuh.)
// ---------------------------------------------------------------------------------------
constexpr int M2L_KC = 32;
constexpr int M2L_NSLICE = NSLICE;  // offsets with dx = -OFF_R..OFF_R, SLICE_OFFS each

struct XJob {
  const int32_t *tlist;   // target box indices (nullptr: 0..ntb-1)
  const uint32_t *d_ntl;  // number of entries of tlist (device)
  int64_t ntb;
  const int32_t *vlist;   // [ntb][NOFF] source box or -1
  const int32_t *cls_of;  // [NOFF] operator class or -1
  const void *M;          // [nsb][ntypes][K]
  const void *ops;        // [ncls][ntypes][2][K][K]
  void *L;                // partial sums [ntb][M2L_NSLOT][K]: slot = slot0 + dx-slice
  int ntypes, slot0;
  int64_t item0;          // first work item of this job
  // octant tiles (free-space jobs at levels >= 3): tile = (octant, run of parents); its slot j
  // holds the child of parent j with that octant.  Boxes of one octant share their far offsets.
  const uint32_t *pstart; // parents' first child (nullptr: plain tiles over tlist / 0..ntb-1)
  const uint32_t *pcount;
  const uint64_t *ckey;   // keys of the target level
  int64_t npar;
};

__host__ __device__ __forceinline__ int64_t m2l_tiles(const XJob &J, int TT) {
  return J.pstart ? 8 * ((J.npar + TT - 1) / TT) : (J.ntb + TT - 1) / TT;
}

// target box of slot j of tile ti, or -1
__device__ __forceinline__ int m2l_target(const XJob &J, int64_t ti, int j, int TT, int64_t ntl) {
  if (J.pstart) {
    const int oct = (int)(ti & 7);
    const int64_t P = (ti >> 3) * TT + j;
    if (P >= J.npar) return -1;
    const uint32_t s0 = J.pstart[P], n = J.pcount[P];
    for (uint32_t k = 0; k < n; ++k)
      if ((int)(J.ckey[s0 + k] & 7ull) == oct) return (int)(s0 + k);
    return -1;
  }
  const int64_t t = ti * TT + j;
  return t < ntl ? (J.tlist ? J.tlist[t] : (int)t) : -1;
}
constexpr int M2L_NSLOT = 2 * M2L_NSLICE;  // free-space slices, then reaction slices

template <typename T, int TPT, int NR>
__global__ void __launch_bounds__(256) k_m2l(const XJob *jobs, int njobs, const T *rot, int K) {
  typedef typename C2<T>::t T2;
  constexpr int TT = 16 * TPT, KR = 16 * NR;
  extern __shared__ __align__(16) unsigned char smraw[];
  T *Pm = (T *)smraw;                 // [KR][KC]
  T *Qm = Pm + KR * M2L_KC;           // [KR][KC]
  T *Xr = Qm + KR * M2L_KC;           // [KC][TT]
  T *Xi = Xr + M2L_KC * TT;           // [KC][TT]
  int *sidx = (int *)(Xi + M2L_KC * TT);  // [TT]
  int *tid_ = sidx + TT;                  // [TT]
  // find the job of this item (jobs sorted by item0)
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].item0 <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const XJob J = jobs[lo];
  const int64_t local = (int64_t)blockIdx.x - J.item0;
  const int slice = (int)(local % M2L_NSLICE);
  const int64_t ti = local / M2L_NSLICE;
  const int64_t ntl = J.tlist ? (int64_t)*J.d_ntl : J.ntb;
  if (J.pstart ? (ti >> 3) * TT >= J.npar : ti * TT >= ntl) return;
  const T2 *M = (const T2 *)J.M;
  const T *ops = (const T *)J.ops;
  T2 *L = (T2 *)J.L;
  const int ntypes = J.ntypes;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if (threadIdx.x < TT) tid_[threadIdx.x] = m2l_target(J, ti, threadIdx.x, TT, ntl);
  T Lr[NR][TPT], Li[NR][TPT];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int j = 0; j < TPT; ++j) Lr[r][j] = Li[r][j] = 0;
  const size_t KK = (size_t)K * K;
  bool any = false;
  __syncthreads();
  for (int o = slice * SLICE_OFFS; o < slice * SLICE_OFFS + SLICE_OFFS; ++o) {
    const int cls = J.cls_of[o];
    if (cls < 0) continue;
    int has = 0;
    if (threadIdx.x < TT) {
      const int t = tid_[threadIdx.x];
      const int s = (t >= 0) ? J.vlist[(size_t)t * NOFF + o] : -1;
      sidx[threadIdx.x] = s;
      has = s >= 0;
    }
    if (!__syncthreads_or(has)) continue;
    any = true;
    T Yr[NR][TPT], Yi[NR][TPT];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int j = 0; j < TPT; ++j) Yr[r][j] = Yi[r][j] = 0;
    const T *rc = rot + (size_t)o * (PMAX + 1) * 2;
    for (int tau = 0; tau < ntypes; ++tau) {
      const T *P = ops + ((size_t)cls * ntypes + tau) * 2 * KK, *Q = P + KK;
      for (int kc = 0; kc < K; kc += M2L_KC) {
        for (int e = threadIdx.x; e < KR * M2L_KC; e += blockDim.x) {
          const int r = e / M2L_KC, k = e % M2L_KC;
          const bool ok = r < K && kc + k < K;
          Pm[e] = ok ? P[(size_t)r * K + kc + k] : T(0);
          Qm[e] = ok ? Q[(size_t)r * K + kc + k] : T(0);
        }
        for (int e = threadIdx.x; e < M2L_KC * TT; e += blockDim.x) {
          const int k = e / TT, j = e % TT;
          const int s = sidx[j];
          T vr = 0, vi = 0;
          if (s >= 0 && kc + k < K) {
            const int m = cK.mof[kc + k];
            const T c = rc[2 * m], sn = rc[2 * m + 1];
            const T2 v = M[((size_t)s * ntypes + tau) * K + kc + k];
            vr = c * v.x - sn * v.y;
            vi = sn * v.x + c * v.y;
          }
          Xr[e] = vr;
          Xi[e] = vi;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < M2L_KC; ++k) {
          T xr[TPT], xi[TPT];
#pragma unroll
          for (int j = 0; j < TPT; ++j) {
            xr[j] = Xr[k * TT + tx + 16 * j];
            xi[j] = Xi[k * TT + tx + 16 * j];
          }
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            const T pv = Pm[(ty + 16 * r) * M2L_KC + k], qv = Qm[(ty + 16 * r) * M2L_KC + k];
#pragma unroll
            for (int j = 0; j < TPT; ++j) {
              Yr[r][j] += pv * xr[j];
              Yi[r][j] += qv * xi[j];
            }
          }
        }
        __syncthreads();
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int row = ty + 16 * r;
      if (row >= K) break;
      const int m = cK.mof[row];
      const T c = rc[2 * m], sn = rc[2 * m + 1];
#pragma unroll
      for (int j = 0; j < TPT; ++j) {
        Lr[r][j] += c * Yr[r][j] + sn * Yi[r][j];
        Li[r][j] += c * Yi[r][j] - sn * Yr[r][j];
      }
    }
  }
  if (!any) return;
#pragma unroll
  for (int j = 0; j < TPT; ++j) {
    const int t = tid_[tx + 16 * j];
    if (t < 0) continue;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int row = ty + 16 * r;
      if (row >= K) break;
      L[((size_t)t * M2L_NSLOT + J.slot0 + slice) * K + row] = T2{Lr[r][j], Li[r][j]};
    }
  }
}

// FP32 multipole-to-local with asynchronous double-buffered staging.  A work item (job, tile of
// 96 target boxes, dx-slice) first lists its (offset, type) steps that have at least one source;
// every step copies the class operator (P, Q, K x K) and the tile's source multipoles into a
// shared-memory stage with cp.async while the previous step is multiplied.  After a stage lands
// the multipoles are rotated by e^{i mu phi} in place; the product is rotated by e^{-i m phi}
// into the register accumulators, which are written to the slice's partial slots at the end.
constexpr int F32_TPT = 6, F32_TT = 16 * F32_TPT, F32_NR = 5, F32_KR = 16 * F32_NR;
constexpr int F32_MAXSTEP = SLICE_OFFS * 2 * (MAXLAYER - 1);  // offsets x source types (2L, L <= 8)
constexpr int HASW = (SLICE_OFFS + 31) / 32;  // words of a per-slice offset mask

__device__ __forceinline__ void cp_async8(void *smem, const void *gmem, bool valid) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

static size_t m2l_f32_smem(int K) {
  const size_t op = (size_t)2 * F32_KR * K * 4, xs = (size_t)F32_TT * (K + 1) * 8;
  return 2 * (op + xs) + sizeof(int) * (F32_TT + F32_MAXSTEP + 2 * F32_TT + F32_KR) + 2 * (PMAX + 1) * 8 * 2;
}

__global__ void __launch_bounds__(256, 1) k_m2l_f32(const XJob *jobs, int njobs, const float *rot, int K) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const size_t opsz = (size_t)2 * F32_KR * K, xsz = (size_t)F32_TT * (K + 1) * 2;  // floats
  float *stage[2];
  stage[0] = (float *)smraw;
  stage[1] = stage[0] + opsz + xsz;
  int *tid_ = (int *)(stage[1] + opsz + xsz);
  int *steps = tid_ + F32_TT;                // (o << 4) | tau
  int *srcs = steps + F32_MAXSTEP;           // [2][TT] source box per stage
  int *mofs = srcs + 2 * F32_TT;              // [KR] m of each half-representation index
  float *rotc = (float *)(mofs + F32_KR);     // [2][PMAX+1][2]
  __shared__ int nsteps;
  __shared__ unsigned hasmask[HASW];
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].item0 <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const XJob J = jobs[lo];
  const int64_t local = (int64_t)blockIdx.x - J.item0;
  const int slice = (int)(local % M2L_NSLICE);
  const int64_t ti = local / M2L_NSLICE;
  const int64_t ntl = J.tlist ? (int64_t)*J.d_ntl : J.ntb;
  if (J.pstart ? (ti >> 3) * F32_TT >= J.npar : ti * F32_TT >= ntl) return;
  const float2 *M = (const float2 *)J.M;
  const float *ops = (const float *)J.ops;
  float2 *L = (float2 *)J.L;
  const int ntypes = J.ntypes;
  const size_t KK = (size_t)K * K;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if (threadIdx.x < F32_TT) tid_[threadIdx.x] = m2l_target(J, ti, threadIdx.x, F32_TT, ntl);
  if (threadIdx.x < HASW) hasmask[threadIdx.x] = 0u;
  if (threadIdx.x < F32_KR) mofs[threadIdx.x] = threadIdx.x < K ? cK.mof[threadIdx.x] : 0;
  // zero the operator padding rows K..KR-1 of both stages once
  for (int s2 = 0; s2 < 2; ++s2)
    for (int e = threadIdx.x; e < 2 * (F32_KR - K) * K; e += blockDim.x) {
      const int half = e / ((F32_KR - K) * K), r = e % ((F32_KR - K) * K);
      stage[s2][half * F32_KR * K + K * K + r] = 0.0f;
    }
  __syncthreads();
  // offsets of the slice with at least one source in the tile
  if (threadIdx.x < F32_TT) {
    const int t = tid_[threadIdx.x];
    if (t >= 0)
      for (int k = 0; k < SLICE_OFFS; ++k) {
        const int o = slice * SLICE_OFFS + k;
        if (J.cls_of[o] >= 0 && J.vlist[(size_t)t * NOFF + o] >= 0) atomicOr(&hasmask[k >> 5], 1u << (k & 31));
      }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int n = 0;
    for (int k = 0; k < SLICE_OFFS; ++k)
      if (hasmask[k >> 5] & (1u << (k & 31)))
        for (int tau = 0; tau < ntypes; ++tau) steps[n++] = ((slice * SLICE_OFFS + k) << 4) | tau;
    nsteps = n;
  }
  __syncthreads();
  const int ns = nsteps;
  if (ns == 0) return;
  // --- staging helpers (explicit, see below)
  auto stage_step = [&](int st, int buf) {
    const int o = steps[st] >> 4, tau = steps[st] & 15;
    const int cls = J.cls_of[o];
    float *opP = stage[buf], *opQ = opP + F32_KR * K;
    float *xs = opP + opsz;
    const float *P = ops + ((size_t)cls * ntypes + tau) * 2 * KK, *Q = P + KK;
    if (KK & 1) {  // Q is only 4-byte aligned: 4-byte granules
      for (int e = threadIdx.x; e < (int)KK; e += blockDim.x) {
        cp_async4(opP + e, P + e);
        cp_async4(opQ + e, Q + e);
      }
    } else {
      const int halfKK = (int)(KK / 2);
      for (int e = threadIdx.x; e < halfKK; e += blockDim.x) {
        cp_async8(opP + 2 * e, P + 2 * e, true);
        cp_async8(opQ + 2 * e, Q + 2 * e, true);
      }
    }
    int *sb = srcs + buf * F32_TT;
    if (threadIdx.x < F32_TT) {
      const int t = tid_[threadIdx.x];
      sb[threadIdx.x] = t >= 0 ? J.vlist[(size_t)t * NOFF + o] : -1;
    }
    if (threadIdx.x < 2 * (PMAX + 1)) {
      float *rc = rotc + buf * 2 * (PMAX + 1);
      rc[threadIdx.x] = rot[(size_t)o * (PMAX + 1) * 2 + threadIdx.x];
    }
    __syncthreads();
    // multipoles: row j (K float2, padded to K+1) of source sb[j]; 8-byte granules
    for (int e = threadIdx.x; e < F32_TT * K; e += blockDim.x) {
      const int j = e / K, k = e % K;
      const int s = sb[j];
      const float2 *src = s >= 0 ? M + ((size_t)s * ntypes + tau) * K + k : M;
      cp_async8(xs + 2 * ((size_t)j * (K + 1) + k), src, s >= 0);
    }
    cp_commit();
  };
  float Lr[F32_NR][F32_TPT], Li[F32_NR][F32_TPT];
#pragma unroll
  for (int r = 0; r < F32_NR; ++r)
#pragma unroll
    for (int j = 0; j < F32_TPT; ++j) Lr[r][j] = Li[r][j] = 0.f;
  stage_step(0, 0);
  for (int st = 0; st < ns; ++st) {
    const int buf = st & 1;
    if (st + 1 < ns) {
      stage_step(st + 1, buf ^ 1);
      cp_wait1();
    } else {
      cp_wait0();
    }
    __syncthreads();
    float *opP = stage[buf], *opQ = opP + F32_KR * K;
    float *xs = opP + opsz;
    const float *rc = rotc + buf * 2 * (PMAX + 1);
    // rotate the staged multipoles by e^{i mu phi}
    for (int e = threadIdx.x; e < F32_TT * K; e += blockDim.x) {
      const int j = e / K, k = e % K;
      float2 *v = (float2 *)(xs + 2 * ((size_t)j * (K + 1) + k));
      const int m = mofs[k];
      const float c = rc[2 * m], sn = rc[2 * m + 1];
      const float2 a = *v;
      *v = make_float2(c * a.x - sn * a.y, sn * a.x + c * a.y);
    }
    __syncthreads();
    float Yr[F32_NR][F32_TPT], Yi[F32_NR][F32_TPT];
#pragma unroll
    for (int r = 0; r < F32_NR; ++r)
#pragma unroll
      for (int j = 0; j < F32_TPT; ++j) Yr[r][j] = Yi[r][j] = 0.f;
    const float2 *xv = (const float2 *)xs;
#pragma unroll 2
    for (int k = 0; k < K; ++k) {
      float2 x[F32_TPT];
#pragma unroll
      for (int j = 0; j < F32_TPT; ++j) x[j] = xv[(size_t)(tx + 16 * j) * (K + 1) + k];
#pragma unroll
      for (int r = 0; r < F32_NR; ++r) {
        const float pv = opP[(ty + 16 * r) * K + k], qv = opQ[(ty + 16 * r) * K + k];
#pragma unroll
        for (int j = 0; j < F32_TPT; ++j) {
          Yr[r][j] = fmaf(pv, x[j].x, Yr[r][j]);
          Yi[r][j] = fmaf(qv, x[j].y, Yi[r][j]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < F32_NR; ++r) {
      const int row = ty + 16 * r;
      const int m = mofs[row];
      const float c = rc[2 * m], sn = rc[2 * m + 1];
#pragma unroll
      for (int j = 0; j < F32_TPT; ++j) {
        Lr[r][j] += c * Yr[r][j] + sn * Yi[r][j];
        Li[r][j] += c * Yi[r][j] - sn * Yr[r][j];
      }
    }
    __syncthreads();  // the stage is refilled two steps later
  }
#pragma unroll
  for (int j = 0; j < F32_TPT; ++j) {
    const int t = tid_[tx + 16 * j];
    if (t < 0) continue;
#pragma unroll
    for (int r = 0; r < F32_NR; ++r) {
      const int row = ty + 16 * r;
      if (row >= K) break;
      L[((size_t)t * M2L_NSLOT + J.slot0 + slice) * K + row] = make_float2(Lr[r][j], Li[r][j]);
    }
  }
}

// L[box][k] += sum over the box's written partial slots, in slot order (deterministic)
template <typename T>
__global__ void k_m2l_reduce(const RJob *jobs, int njobs, int K) {
  typedef typename C2<T>::t T2;
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].e0 <= g) lo = mid; else hi = mid - 1;
  }
  const RJob J = jobs[lo];
  const int64_t e = g - J.e0;
  if (e < 0 || e >= J.n) return;
  const int64_t box = e / K, k = e % K;
  const T2 *P = (const T2 *)J.part + box * M2L_NSLOT * K + k;
  T sx = 0, sy = 0;
  for (uint32_t m = J.smask ? J.smask[box] : (1u << M2L_NSLOT) - 1u; m; m &= m - 1) {
    const int s = __ffs(m) - 1;
    sx += P[(size_t)s * K].x;
    sy += P[(size_t)s * K].y;
  }
  T2 &d = ((T2 *)J.L)[e];
  d.x += sx;
  d.y += sy;
}

// ---------------------------------------------------------------------------------------
// free-space P2P over the near list (the boxes within the separation, incl. the box itself).  A
// pair of zero distance (the charge itself, or another at the same point) contributes nothing.
// ---------------------------------------------------------------------------------------
constexpr int P2P_THREADS = 128;  // reaction near field

__device__ __forceinline__ float fexp(float x) { return __expf(x); }
__device__ __forceinline__ double fexp(double x) { return exp(x); }

// FP64 near field: one CTA of P64_WARPS warps per leaf, every group of the evaluation in one launch.
// Bound: the FP64 pipe (half an FMA per clock and SM quarter), so the kernel minimises FP64
// operations per pair and idle lanes and leaves everything else to the other pipes:
//  * 28 FP64 operations per pair (21 without the field): 1/r from the special-function unit's
//    approximation y by one third-order step (5 operations): with e = 1 - x y^2, x^{-1/2} = y (1 - e)^{-1/2} =
//    y (1 + e/2 + 3 e^2/8 + ...), the binomial series to second order, whose next term 5 e^3/16 is below 2^-58 for an
//    approximation good to 2^-20; e^{-lambda r} by the table method (Tang,
//    ACM TOMS 15, 1989: 2^(n/2048) from a table, a cubic for the remainder below 2^-12; 7 operations).
//    The library's rsqrt and exp take about 45 in all.
//  * no idle lanes in a leaf's last, partial group of targets: a group of 2^b targets gives each of
//    them 32 / 2^b lanes, which split the sources; cnt targets take the full groups of 32 and one
//    group per set bit of the rest.  The warps of the CTA split the sources once more.
//  * coordinates are read as they are (no shared-memory tiles: a pair's 32 bytes cost nothing beside
//    its FP64 time) and differences of them are the exact inputs of r.
// Sums: per lane over its sources, then over the lanes and warps of a target in a fixed order.
constexpr int P64_WARPS = 8;
constexpr int EXP_TAB_BITS = 11, EXP_TAB = 1 << EXP_TAB_BITS;
__device__ double g_exp2_tab[EXP_TAB];  // 2^(j / EXP_TAB)

void upload_exp2(cudaStream_t s) {
  static double h[EXP_TAB];
  for (int j = 0; j < EXP_TAB; ++j) h[j] = (double)exp2l((long double)j / EXP_TAB);
  LPB_CUDA(cudaMemcpyToSymbolAsync(g_exp2_tab, h, sizeof h, 0, cudaMemcpyHostToDevice, s));
}

struct P64Job {
  const uint32_t *bstart, *bcount;  // leaf point ranges
  const int32_t *ulist;             // [nb][NNEAR] near leaves or -1
  const double *x, *y, *z, *q;      // sorted points
  const uint32_t *src;              // input index of each point
  double lam, scale, ce;            // screening; 1 / (4 pi eps); -lambda log2(e) EXP_TAB
  uint32_t hi_max;                  // high word of the largest r^2 that counts: lambda r <= 700
  uint32_t nb;
  int64_t block0;
};

template <bool FIELD>
__device__ __forceinline__ void p64_pair(double dx, double dy, double dz, double q, double lam, double ce,
                                         uint32_t hi_max, double &p, double &fx, double &fy, double &fz) {
  const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
  double y0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(r2));
  // normal r^2 up to the cut (beyond it e^{-lambda r} < 1e-304); else 1/r = 0 and the pair drops out
  const uint32_t hi = (uint32_t)__double2hiint(r2) - 0x00100000u;
  y0 = hi <= hi_max ? y0 : 0.0;
  const double e = fma(-(r2 * y0), y0, 1.0);
  const double ri = fma(y0 * e, fma(0.375, e, 0.5), y0);
  const double r = r2 * ri;
  const double magic = 6755399441055744.0;  // 1.5 * 2^52: the sum's low word is the rounded integer
  const double kd = fma(r, ce, magic);
  const int n = __double2loint(kd);
  const double f = fma(r, ce, magic - kd);
  constexpr double u = 0.693147180559945309417 / EXP_TAB;
  const double pm = f * fma(f, fma(f, u * u * u / 6.0, u * u / 2.0), u);
  const double t0 = g_exp2_tab[n & (EXP_TAB - 1)];
  const double t = __hiloint2double(__double2hiint(t0) + ((n >> EXP_TAB_BITS) << 20), __double2loint(t0));
  const double w = fma(t, pm, t) * ri;
  p = fma(q, w, p);
  if (FIELD) {
    const double g = (q * w) * (ri * (ri + lam));
    fx = fma(g, dx, fx);
    fy = fma(g, dy, fy);
    fz = fma(g, dz, fz);
  }
}

template <bool FIELD>
__global__ void __launch_bounds__(32 * P64_WARPS) k_p2p_free_f64(const P64Job *jobs, int njobs, double *phi,
                                                                 double *field) {
  __shared__ uint32_t nb_start[NNEAR], nb_cnt[NNEAR];
  __shared__ double part[P64_WARPS][4][32];
  __shared__ int s_nnb;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].block0 <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const P64Job &J = jobs[lo];
  const uint32_t box = (uint32_t)((int64_t)blockIdx.x - J.block0);
  if (box >= J.nb) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tst = J.bstart[box], tcnt = J.bcount[box];
  if (warp == 0) {  // the non-empty near boxes, in slot order
    int nnb = 0;
    for (int o0 = 0; o0 < NNEAR; o0 += 32) {
      const int o = o0 + lane;
      const int sb = o < NNEAR ? J.ulist[(size_t)box * NNEAR + o] : -1;
      const uint32_t cnt = sb >= 0 ? J.bcount[sb] : 0u;
      const unsigned m = __ballot_sync(0xffffffffu, cnt > 0);
      if (cnt > 0) {
        const int k = nnb + __popc(m & ((1u << lane) - 1u));
        nb_start[k] = J.bstart[sb];
        nb_cnt[k] = cnt;
      }
      nnb += __popc(m);
    }
    if (lane == 0) s_nnb = nnb;
  }
  __syncthreads();
  const int nnb = s_nnb;
  const double *X = J.x, *Yc = J.y, *Z = J.z, *Q = J.q;
  const double lam = J.lam, ce = J.ce;
  const uint32_t hi_max = J.hi_max;
  for (uint32_t t0 = 0; t0 < tcnt;) {
    const uint32_t left = tcnt - t0;
    const int lb = left >= 32 ? 5 : 31 - __clz((int)left);  // 2^lb targets in this group
    const int sub = lane >> lb, nsub = 32 >> lb;            // this lane's share of the sources
    const uint32_t tk = tst + t0 + (lane & ((1 << lb) - 1));
    const double px = X[tk], py = Yc[tk], pz = Z[tk];
    double p = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
    // sources first + stride i of the concatenated near boxes
    const uint32_t stride = (uint32_t)(nsub * P64_WARPS);
    uint32_t off = (uint32_t)(warp * nsub + sub);
    int k = 0;
    for (;; off += stride) {
      while (k < nnb && off >= nb_cnt[k]) off -= nb_cnt[k++];
      if (k >= nnb) break;
      const uint32_t j = nb_start[k] + off;
      p64_pair<FIELD>(px - X[j], py - Yc[j], pz - Z[j], Q[j], lam, ce, hi_max, p, fx, fy, fz);
    }
    for (int o = 16; o >= (1 << lb); o >>= 1) {  // lanes of one target differ in the bits above lb
      p += __shfl_xor_sync(0xffffffffu, p, o);
      if (FIELD) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
        fz += __shfl_xor_sync(0xffffffffu, fz, o);
      }
    }
    __syncthreads();  // the previous group's sums have been read
    part[warp][0][lane] = p;
    if (FIELD) {
      part[warp][1][lane] = fx;
      part[warp][2][lane] = fy;
      part[warp][3][lane] = fz;
    }
    __syncthreads();
    const int v = threadIdx.x >> lb, t = threadIdx.x & ((1 << lb) - 1);  // value, target
    if (v < (FIELD ? 4 : 1)) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < P64_WARPS; ++w) s += part[w][v][t];
      const uint32_t i = J.src[tst + t0 + t];
      if (v == 0) phi[i] += J.scale * s;
      else field[3 * (size_t)i + v - 1] += J.scale * s;
    }
    t0 += 1u << lb;
  }
}

#include "p2p_f32.cuh"

// ---------------------------------------------------------------------------------------
// reaction near field: target leaf box vs adjacent image leaf boxes across the interface,
// Sommerfeld integral by the precomputed node rule, truncated per pair at exp(-36)
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float fj0(float x) { return j0f(x); }
__device__ __forceinline__ double fj0(double x) { return j0(x); }
__device__ __forceinline__ float fj1(float x) { return j1f(x); }
__device__ __forceinline__ double fj1(double x) { return j1(x); }

template <typename T>
__global__ void __launch_bounds__(P2P_THREADS) k_p2p_react(
    const uint32_t *d_nb, const uint64_t *tkey, const uint32_t *tstart, const uint32_t *tcount, const int32_t *ulist,
    const double *tx, const double *ty, const double *tz, const uint32_t *tsrc, const uint32_t *istart,
    const uint32_t *icount, const double *ix, const double *iy, const double *iz, const double *iq,
    const uint64_t *ikey, Geo geo, double dI, double sa, const double *nodes, int nq, double *phi, double *field) {
  __shared__ T sx[P2P_THREADS], sy[P2P_THREADS], szs[P2P_THREADS], sq[P2P_THREADS];
  __shared__ int st[P2P_THREADS];
  const uint32_t box = blockIdx.x;
  if (box >= *d_nb) return;
  bool any = false;
  for (int o = 0; o < NNEAR; ++o) any |= ulist[(size_t)box * NNEAR + o] >= 0;
  if (!any) return;
  double cx, cy, cz;
  box_center(tkey[box], geo, cx, cy, cz);
  const uint32_t tst = tstart[box], tcnt = tcount[box];
  for (uint32_t t0 = 0; t0 < tcnt; t0 += P2P_THREADS) {
    const uint32_t tj = t0 + threadIdx.x;
    const bool tv = tj < tcnt;
    const uint32_t tk = tst + (tv ? tj : 0);
    const T px = (T)(tx[tk] - cx), py = (T)(ty[tk] - cy);
    const T zt = (T)fabs(tz[tk] - dI);
    double aphi = 0, ax = 0, ay = 0, az = 0;
    for (int o = 0; o < NNEAR; ++o) {
      const int s = ulist[(size_t)box * NNEAR + o];
      if (s < 0) continue;
      const uint32_t sst = istart[s], scnt = icount[s];
      for (uint32_t s0 = 0; s0 < scnt; s0 += P2P_THREADS) {
        __syncthreads();
        if (s0 + threadIdx.x < scnt) {
          const uint32_t k = sst + s0 + threadIdx.x;
          sx[threadIdx.x] = (T)(ix[k] - cx);
          sy[threadIdx.x] = (T)(iy[k] - cy);
          szs[threadIdx.x] = (T)fabs(iz[k] - dI);
          sq[threadIdx.x] = (T)iq[k];
          st[threadIdx.x] = (int)(ikey[k] & 15ull);
        }
        __syncthreads();
        const uint32_t nn = min((uint32_t)P2P_THREADS, scnt - s0);
        if (!tv) continue;
        for (uint32_t jj = 0; jj < nn; ++jj) {
          const T dx = px - sx[jj], dy = py - sy[jj];
          const T rho = sqrt(dx * dx + dy * dy);
          const T zs = szs[jj];
          const T xcut = T(36) / (zt + zs);
          const double *nd = nodes + (size_t)st[jj] * nq * 4;
          T v = 0, vr = 0, vz = 0;
          for (int k = 0; k < nq; ++k) {
            const T lr = (T)nd[4 * k];
            if (lr > xcut) break;
            const T E = (T)nd[4 * k + 1] * fexp(-(T)nd[4 * k + 2] * zt - (T)nd[4 * k + 3] * zs);
            const T a = lr * rho;
            const T J0 = fj0(a);
            const T J1r = rho > T(0) ? fj1(a) / rho : T(0.5) * lr;
            v += E * J0;
            vr += E * lr * J1r;
            vz += E * J0 * (T)nd[4 * k + 2];
          }
          const T qq = sq[jj];
          aphi += (double)(qq * v);
          ax += (double)(qq * dx * vr);
          ay += (double)(qq * dy * vr);
          az += (double)(qq * vz);
        }
      }
    }
    if (tv) {
      const uint32_t i = tsrc[tk];
      phi[i] += aphi;
      if (field) {
        field[3 * i] += ax;
        field[3 * i + 1] += ay;
        field[3 * i + 2] += sa * az;
      }
    }
  }
}

#include "m2l_pairs.cuh"
#include "m2l_tc.cuh"

// ---------------------------------------------------------------------------------------
// driver for one group
// ---------------------------------------------------------------------------------------
struct Tables {
  int32_t *cls_free, *cls_react;  // [NOFF], [2][NKT][NOFF]
  int32_t *tc_free, *tc_react;    // the same for the tensor-core operators (per canonical pair)
  void *rot, *rot4;               // per precision
};
Tables g_tab_d[LPB_MAX_DEVICES], g_tab_f[LPB_MAX_DEVICES];  // per device
static std::atomic<uint64_t> g_tab_ready{0};

static void make_tables(Ctx &c) {
  if (!not_done_on_device(g_tab_ready)) return;
  // operator class of every offset that can appear in a far list (|d|_inf >= 2); which offsets
  // do appear is decided by the list builder for the context's separation
  std::vector<int32_t> cf(NOFF, -1), cr(2 * NKT * NOFF, -1), tf(NOFF, -1), tr(2 * NKT * NOFF, -1);
  std::vector<double> rot(NOFF * (PMAX + 1) * 2), rot4(4 * (PMAX + 1) * 2);
  for (int o = 0; o < NOFF; ++o) {
    int dx, dy, dz;
    off_decode(o, dx, dy, dz);
    const int cheb = cheb3(dx, dy, dz);
    int kq;
    bool refl;
    const int ci = can_of(dx, dy, kq, refl);
    if (cheb >= 2) {
      cf[o] = rho_index(dx, dy) * NDZ + dz + OFF_R;
      tf[o] = ci * NDZ + dz + OFF_R;
    }
    for (int a = 1; a <= 2; ++a)
      for (int kt = 0; kt < NKT; ++kt) {
        const int ks = (a == 1) ? -dz - 1 - kt : dz - 1 - kt;
        const int kk = kk_index(kt, ks);
        if (cheb < 2 || kk < 0) continue;
        cr[((a - 1) * NKT + kt) * NOFF + o] = rho_index(dx, dy) * NKK + kk;
        tr[((a - 1) * NKT + kt) * NOFF + o] = ci * NKK + kk;
      }
    const double ph = (dx == 0 && dy == 0) ? 0.0 : atan2(-(double)dy, -(double)dx);
    for (int m = 0; m <= PMAX; ++m) {
      rot[(o * (PMAX + 1) + m) * 2] = cos(m * ph);
      rot[(o * (PMAX + 1) + m) * 2 + 1] = sin(m * ph);
    }
  }
  for (int dir = 0; dir < 4; ++dir) {
    const int bx = dir >> 1, by = dir & 1;
    const double ph = atan2(2.0 * by - 1.0, 2.0 * bx - 1.0);
    for (int m = 0; m <= PMAX; ++m) {
      rot4[(dir * (PMAX + 1) + m) * 2] = cos(m * ph);
      rot4[(dir * (PMAX + 1) + m) * 2 + 1] = sin(m * ph);
    }
  }
  int32_t *dcf, *dcr, *dtf, *dtr;
  LPB_CUDA(cudaMalloc(&dtf, sizeof(int32_t) * NOFF));
  LPB_CUDA(cudaMalloc(&dtr, sizeof(int32_t) * 2 * NKT * NOFF));
  LPB_CUDA(cudaMemcpy(dtf, tf.data(), sizeof(int32_t) * NOFF, cudaMemcpyHostToDevice));
  LPB_CUDA(cudaMemcpy(dtr, tr.data(), sizeof(int32_t) * 2 * NKT * NOFF, cudaMemcpyHostToDevice));
  LPB_CUDA(cudaMalloc(&dcf, sizeof(int32_t) * NOFF));
  LPB_CUDA(cudaMalloc(&dcr, sizeof(int32_t) * 2 * NKT * NOFF));
  LPB_CUDA(cudaMemcpy(dcf, cf.data(), sizeof(int32_t) * NOFF, cudaMemcpyHostToDevice));
  LPB_CUDA(cudaMemcpy(dcr, cr.data(), sizeof(int32_t) * 2 * NKT * NOFF, cudaMemcpyHostToDevice));
  std::vector<float> rotf(rot.begin(), rot.end()), rot4f(rot4.begin(), rot4.end());
  void *rd, *r4d, *rf, *r4f;
  LPB_CUDA(cudaMalloc(&rd, sizeof(double) * rot.size()));
  LPB_CUDA(cudaMalloc(&r4d, sizeof(double) * rot4.size()));
  LPB_CUDA(cudaMalloc(&rf, sizeof(float) * rot.size()));
  LPB_CUDA(cudaMalloc(&r4f, sizeof(float) * rot4.size()));
  LPB_CUDA(cudaMemcpy(rd, rot.data(), sizeof(double) * rot.size(), cudaMemcpyHostToDevice));
  LPB_CUDA(cudaMemcpy(r4d, rot4.data(), sizeof(double) * rot4.size(), cudaMemcpyHostToDevice));
  LPB_CUDA(cudaMemcpy(rf, rotf.data(), sizeof(float) * rotf.size(), cudaMemcpyHostToDevice));
  LPB_CUDA(cudaMemcpy(r4f, rot4f.data(), sizeof(float) * rot4f.size(), cudaMemcpyHostToDevice));
  g_tab_d[c.device] = Tables{dcf, dcr, dtf, dtr, rd, r4d};
  g_tab_f[c.device] = Tables{dcf, dcr, dtf, dtr, rf, r4f};
  mark_done_on_device(g_tab_ready);
}

void upload_gl();
void upload_an();
void upload_trig(cudaStream_t s);
void init_fmm_tables(Ctx &c) {
  static std::mutex mu;
  std::lock_guard<std::mutex> lk(mu);
  upload_gl();
  upload_an();
  make_tables(c);
  upload_exp2(c.stream);
  upload_trig(c.stream);
  upload_consts(c.stream);
}

template <typename T, int PT>
static void launch_p2m(Ctx &c, const std::vector<P2MJob> &dense, const std::vector<P2MJob> &sparse, int64_t nd,
                       int64_t ns) {
  if (nd) {
    k_p2m<T, PT><<<(unsigned)nd, 128, 0, c.stream>>>(upload_jobs(c, dense), (int)dense.size(), c.p, c.K);
    LPB_LAUNCH();
    c.launches++;
  }
  if (ns) {
    k_p2m_sparse<T, PT><<<(unsigned)ns, 128, 0, c.stream>>>(upload_jobs(c, sparse), (int)sparse.size(), c.p, c.K);
    LPB_LAUNCH();
    c.launches++;
  }
}
template <typename T, int PT>
static void launch_l2p(Ctx &c, const std::vector<L2PJob> &dense, const std::vector<L2PJob> &sparse, int64_t nd,
                       int64_t ns, double *phi, double *field) {
  if (nd) {
    k_l2p<T, PT, false><<<(unsigned)nd, 128, 0, c.stream>>>(upload_jobs(c, dense), (int)dense.size(), c.p, c.K, phi,
                                                            field);
    LPB_LAUNCH();
    c.launches++;
  }
  if (ns) {
    k_l2p<T, PT, true><<<(unsigned)ns, 128, 0, c.stream>>>(upload_jobs(c, sparse), (int)sparse.size(), c.p, c.K, phi,
                                                           field);
    LPB_LAUNCH();
    c.launches++;
  }
}

template <typename T, int TPT, int NR>
static void launch_m2l_t(Ctx &c, const std::vector<XJob> &jobs, int64_t items) {
  constexpr int TT = 16 * TPT, KR = 16 * NR;
  const size_t smem = sizeof(T) * (2 * KR * M2L_KC + 2 * M2L_KC * TT) + sizeof(int) * 2 * TT;
  LPB_ATTR_ONCE((k_m2l<T, TPT, NR>), smem);
  XJob *dj = c.arena.get<XJob>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(XJob) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
  const Tables &tb = sizeof(T) == 8 ? g_tab_d[c.device] : g_tab_f[c.device];
  k_m2l<T, TPT, NR><<<(unsigned)items, 256, smem, c.stream>>>(dj, (int)jobs.size(), (const T *)tb.rot, c.K);
  LPB_LAUNCH();
  c.launches++;
}

#define PT_DISPATCH(F, ...)                                   \
  do {                                                        \
    if (c.p <= 5) F<T, 5>(__VA_ARGS__);                       \
    else if (c.p <= 8) F<T, 8>(__VA_ARGS__);                  \
    else if (c.p <= 10) F<T, 10>(__VA_ARGS__);                \
    else if (c.p <= 12) F<T, 12>(__VA_ARGS__);                \
    else F<T, 16>(__VA_ARGS__);                               \
  } while (0)

template <typename T>
static Geo geo_at(const Group &g, int l) {
  Geo G;
  G.o[0] = g.root[0] - g.root[3];
  G.o[1] = g.root[1] - g.root[3];
  G.o[2] = g.root[2] - g.root[3];
  G.h = g.h(l);
  return G;
}

// P2M and M2M of every group; local expansions of every level zeroed
template <typename T>
static void upward_t(Ctx &c, std::vector<Group> &groups) {
  typedef typename C2<T>::t T2;
  const int K = c.K;
  const Tables &tb = sizeof(T) == 8 ? g_tab_d[c.device] : g_tab_f[c.device];
  int64_t nl = 0;
  int Dmax = 2;
  for (auto &g : groups)
    for (int l = 2; l <= g.D; ++l) nl += g.T.lev[l].n;
  T2 *Lt = c.arena.get<T2>(nl * K);
  LPB_CUDA(cudaMemsetAsync(Lt, 0, sizeof(T2) * nl * K, c.stream));
  // absent (box, type) rows are neither written nor read; the SIMT M2L of the mixed mode (p > 10) reads them all
  const bool zero_img = sizeof(T) == 4 && tc_chunks(c.p) > 4;
  std::vector<P2MJob> dense, sparse;
  int64_t nd = 0, ns = 0;
  auto p2m = [&](const Group &g, const PointSet &P, int lev, const uint32_t *sst, const uint32_t *scnt,
                 const uint32_t *sbox, const uint32_t *styp, int64_t nseg, int ntypes, void *M) {
    P2MJob j;
    j.sst = sst; j.scnt = scnt; j.sbox = sbox; j.styp = styp; j.nseg = nseg; j.ntypes = ntypes;
    j.bkey = P.lev[lev].key; j.x = P.x; j.y = P.y; j.z = P.z; j.q = P.q; j.geo = geo_at<T>(g, lev); j.M = M;
    for (int t = 0; t < 2 * MAXLAYER; ++t) j.lam[t] = c.md.lam[g.l];
    if (styp)
      for (int t = 0; t < ntypes; ++t) {
        int lp, b;
        type_decode(t, lp, b);
        j.lam[t] = c.md.lam[lp];
      }
    if (P.np < P2M_SPARSE * nseg) {
      j.item0 = ns;
      ns += (nseg + 127) / 128;
      sparse.push_back(j);
    } else {
      j.item0 = nd;
      nd += (nseg + 3) / 4;
      dense.push_back(j);
    }
  };
  for (auto &g : groups) {
    const bool dofree = g.is_free && (g.parts & 1), doreact = (g.parts & 2) && g.I.np > 0;
    Dmax = std::max(Dmax, g.D);
    for (int l = 2; l <= g.D; ++l) {
      const int64_t ntb = g.T.lev[l].n, nib = g.I.lev[l].n;
      g.Lt[l] = Lt;
      Lt += ntb * K;
      if (dofree && l <= g.Df) g.Mfree[l] = c.arena.get<T2>(ntb * K);
      if (doreact) {
        g.Mimg[l] = c.arena.get<T2>(nib * g.ntypes * K);
        if (zero_img) LPB_CUDA(cudaMemsetAsync(g.Mimg[l], 0, sizeof(T2) * nib * g.ntypes * K, c.stream));
      }
    }
    // free-space P2M at the free-space leaves (level Df; their point ranges)
    const Level &Lf = g.T.lev[g.Df];
    if (dofree && Lf.n) p2m(g, g.T, g.Df, Lf.pstart, Lf.pcount, nullptr, nullptr, Lf.n, 1, g.Mfree[g.Df]);
    if (doreact && g.I.nseg)
      p2m(g, g.I, g.D, g.I.seg_start, g.I.seg_count, g.I.seg_box, g.I.seg_type, g.I.nseg, g.ntypes, g.Mimg[g.D]);
  }
  PT_DISPATCH(launch_p2m, c, dense, sparse, nd, ns);
  for (int l = Dmax; l >= 3; --l) {
    std::vector<M2MJob> jobs;
    auto m2m = [&](const PointSet &P, const uint32_t *const *mask, int ntypes, const void *Mc, void *Mp, const void *ops) {
      if (!P.lev[l - 1].n) return;
      M2MJob j;
      j.pstart = P.lev[l - 1].start; j.pcount = P.lev[l - 1].count; j.ckey = P.lev[l].key;
      j.pmask = mask ? mask[l - 1] : nullptr; j.cmask = mask ? mask[l] : nullptr;
      j.Mc = Mc; j.Mp = Mp; j.ops = ops; j.np = P.lev[l - 1].n; j.ntypes = ntypes;
      jobs.push_back(j);
    };
    for (auto &g : groups) {
      if (l > g.D) continue;
      if (g.is_free && (g.parts & 1) && l <= g.Df) m2m(g.T, nullptr, 1, g.Mfree[l], g.Mfree[l - 1], g.op_m2m_t[l]);
      if ((g.parts & 2) && g.I.np > 0) m2m(g.I, g.tmask, g.ntypes, g.Mimg[l], g.Mimg[l - 1], g.op_m2m_i[l]);
    }
    if (jobs.empty()) continue;
    int64_t np = 0, items = 0;
    for (auto &j : jobs) np += j.np;
    for (auto &j : jobs) {
      j.tsplit = np <= M2M_TSPLIT_MAX ? j.ntypes : 1;
      j.item0 = items;
      items += j.np * j.tsplit;
    }
    k_m2m<T><<<(unsigned)items, oct_threads(K, c.p, items), oct_smem<T>(K, c.p), c.stream>>>(
        upload_jobs(c, jobs), (int)jobs.size(), (const T *)tb.rot4, K, c.p);
    LPB_LAUNCH();
    c.launches++;
  }
}

// FP64: every multipole-to-local translation of every group and level, sorted by operator
static void m2l_all_f64(Ctx &c, std::vector<Group> &groups) {
  const Tables &tb = g_tab_d[c.device];
  std::vector<PairJob> jobs;
  std::vector<int> ncls;
  for (int kind = 0; kind < 2; ++kind)  // free-space jobs, then reaction jobs
    for (auto &g : groups) {
      const bool react_far = (g.parts & 2) && g.I.np > 0 && !(g.parts & 8);
      for (int l = 2; l <= g.D; ++l) {
        const int64_t ntb = g.T.lev[l].n;
        if (!ntb) continue;
        PairJob j;
        j.L = (double2 *)g.Lt[l];
        j.ntb = (int32_t)ntb;
        j.t0 = 0;
        j.bin0 = 0;
        if (kind == 0 && g.is_free && (g.parts & 1) && l <= g.Df) {
          j.vlist = g.vfree[l]; j.cls = tb.cls_free; j.ktrow = nullptr; j.tmask = nullptr;
          j.M = (const double2 *)g.Mfree[l]; j.ops = (const double *)g.op_free[l];
          j.ntypes = 1; j.nkt = 0;
          jobs.push_back(j);
          ncls.push_back(NFREE_CLS);
        }
        if (kind == 1 && react_far && g.vreact[l]) {
          j.vlist = g.vreact[l]; j.cls = tb.cls_react + (size_t)(g.a - 1) * NKT * NOFF; j.ktrow = g.ktrow[l];
          j.tmask = g.tmask[l]; j.M = (const double2 *)g.Mimg[l]; j.ops = (const double *)g.op_react[l];
          j.ntypes = g.ntypes; j.nkt = 2 * c.ws + 1;
          jobs.push_back(j);
          ncls.push_back(NREACT_CLS);
        }
      }
    }
  if (jobs.empty()) return;
  prof_mark(c, "m2l_prep");
  launch_pair_m2l(c, jobs, ncls, (const double *)tb.rot);
}

template <int P>
static void launch_pack_w_p(const PackWJob *jobs, int njobs, int64_t items, int ws, cudaStream_t st) {
  constexpr int K = (P + 1) * (P + 2) / 2;
  k_tc_pack_w<P><<<(unsigned)items, PACKW_THREADS, sizeof(float) * 2 * K * K, st>>>(jobs, njobs, ws);
}
static void launch_pack_w(int p, const PackWJob *jobs, int njobs, int64_t items, int ws, cudaStream_t st) {
  switch (p) {
#define LPB_TC_CASE(P) case P: launch_pack_w_p<P>(jobs, njobs, items, ws, st); break;
    LPB_TC_CASE(2) LPB_TC_CASE(3) LPB_TC_CASE(4) LPB_TC_CASE(5) LPB_TC_CASE(6) LPB_TC_CASE(7) LPB_TC_CASE(8)
    LPB_TC_CASE(9) LPB_TC_CASE(10)
#undef LPB_TC_CASE
  }
}
template <int P>
static void launch_tc_p(const TJob *jobs, int njobs, int64_t items, int *status, cudaStream_t st) {
  LPB_ATTR_ONCE(k_m2l_tc<P>, tc_smem(tc_chunks(P)));
  k_m2l_tc<P><<<(unsigned)items, TC_THREADS, tc_smem(tc_chunks(P)), st>>>(jobs, njobs, status);
}
static void launch_tc(int p, const TJob *jobs, int njobs, int64_t items, int *status, cudaStream_t st) {
  switch (p) {
#define LPB_TC_CASE(P) case P: launch_tc_p<P>(jobs, njobs, items, status, st); break;
    LPB_TC_CASE(2) LPB_TC_CASE(3) LPB_TC_CASE(4) LPB_TC_CASE(5) LPB_TC_CASE(6) LPB_TC_CASE(7) LPB_TC_CASE(8)
    LPB_TC_CASE(9) LPB_TC_CASE(10)
#undef LPB_TC_CASE
  }
}

void reserve_images(Ctx &c, std::vector<Group> &groups) {
  c.images_ready = false;
  const int NC = tc_chunks(c.p), N = 32 * NC;
  if (c.opts.precision == LPBFMM_FP64 || NC > 4) return;
  for (auto &g : groups)
    for (int l = 2; l <= g.D; ++l)
      for (int kind = 0; kind < 2; ++kind) {
        if (!g.T.lev[l].n) continue;
        if (kind == 0 ? !(g.is_free && (g.parts & 1) && l <= g.Df)
                      : !((g.parts & 2) && g.I.np > 0 && !(g.parts & 8) && g.vreact[l])) continue;
        const size_t n = kind ? (size_t)TC_NREACT * g.ntypes : (size_t)TC_NFREE;
        g.wimg[kind][l] = c.arena.get<unsigned char>(n * N * N * 4);
        g.wscale[kind][l] = c.arena.get<float>(n);
      }
}

// mixed mode: every multipole-to-local translation of every group and level in one launch
static void m2l_all_f32(Ctx &c, std::vector<Group> &groups) {
  typedef float T;
  constexpr int TPT = 4, TT = 16 * TPT;
  const Tables &tb = g_tab_f[c.device];
  std::vector<XJob> jobs;
  int64_t items = 0;
  typedef C2<T>::t T2;
  std::vector<RJob> rjobs;
  int64_t relem = 0;
  // tensor-core path: 2K - (p+1) <= 128 real coordinates
  const int tc_nc = tc_chunks(c.p);
  const bool use_tc = tc_nc <= 4;  // p <= 10
  std::vector<TJob> tjobs;
  int64_t titems = 0;
  std::vector<PackRowJob> prow;
  std::vector<PackWJob> pw;
  int64_t row_items = 0, img_items = 0;
  uint32_t *smasks = nullptr;
  if (use_tc) {
    int64_t nb = 0;
    for (auto &g : groups)
      for (int l = 2; l <= g.D; ++l) nb += g.T.lev[l].n;
    smasks = c.arena.get<uint32_t>(nb);
    LPB_CUDA(cudaMemsetAsync(smasks, 0, sizeof(uint32_t) * nb, c.stream));
  }
  auto add = [&](const int32_t *tlist, const uint32_t *d_ntl, int64_t ntb, const int32_t *vlist,
                 const int32_t *cls_of, const void *M, const void *ops, void *part, int ntypes, int slot0,
                 const Level *par, const Level *lev) {
    XJob j;
    j.tlist = tlist; j.d_ntl = d_ntl; j.ntb = ntb; j.vlist = vlist; j.cls_of = cls_of;
    j.M = M; j.ops = ops; j.L = part; j.ntypes = ntypes; j.slot0 = slot0; j.item0 = items;
    j.pstart = par ? par->start : nullptr;
    j.pcount = par ? par->count : nullptr;
    j.ckey = par ? lev->key : nullptr;
    j.npar = par ? par->n : 0;
    jobs.push_back(j);
    items += m2l_tiles(j, TT) * M2L_NSLICE;
  };
  for (auto &g : groups) {
    const int parts = g.parts;
    const bool react_far = (parts & 2) && g.I.np > 0 && !(parts & 8);
    for (int l = 2; l <= g.D; ++l) {
      const bool dofree = g.is_free && (parts & 1) && l <= g.Df;
      const int64_t ntb = g.T.lev[l].n;
      if (!ntb || !(dofree || (react_far && g.vreact[l]))) continue;
      T2 *part = c.arena.get<T2>((size_t)ntb * M2L_NSLOT * c.K);
      uint32_t *smask = nullptr;  // partial slots written (the SIMT kernels write or leave zero every slot)
      if (use_tc) {
        smask = smasks;
        smasks += ntb;
      } else {
        LPB_CUDA(cudaMemsetAsync(part, 0, sizeof(T2) * ntb * M2L_NSLOT * c.K, c.stream));
      }
      RJob r;
      r.part = part; r.L = g.Lt[l]; r.n = ntb * c.K; r.e0 = relem; r.smask = smask;
      rjobs.push_back(r);
      relem += r.n;
      const int N = 32 * tc_nc;
      // split source rows; operator images (once per evaluation, also for several charge vectors)
      auto pack = [&](TJob &j, const void *M, const Level &sl, const uint32_t *mask, int side, const void *ops, int kind,
                      int ntypes, const uint8_t *used, int ncls) {
        PackRowJob r;
        r.M = (const float2 *)M; r.nrows = sl.n * ntypes; r.item0 = row_items; r.ntypes = ntypes; r.mask = mask;
        r.bkey = sl.key; r.lev = l; r.side = side;
        r.rows = c.arena.get<__half>((size_t)r.nrows * 2 * N);
        r.rscale = c.arena.get<float>((size_t)r.nrows);
        row_items += (r.nrows + 7) / 8;
        prow.push_back(r);
        if (!c.images_ready) {
          pw.push_back(PackWJob{(const float *)ops, used, g.wimg[kind][l], g.wscale[kind][l], img_items, kind, ntypes});
          img_items += (int64_t)ncls * ntypes;
        }
        j.rows = r.rows; j.rscale = r.rscale; j.tmask = mask; j.ntypes = ntypes;
        j.wimg = g.wimg[kind][l]; j.wscale = g.wscale[kind][l];
        j.L = (float2 *)part; j.smask = smask; j.ntb = ntb;
      };
      if (dofree && use_tc) {
        TJob j;
        pack(j, g.Mfree[l], g.T.lev[l], nullptr, 0, g.op_free[l], 0, 1, nullptr, TC_NFREE);
        j.vlist = g.vfree[l]; j.cls_of = tb.tc_free; j.tlist = nullptr; j.d_ntl = nullptr;
        j.item0 = titems; j.slot0 = 0;
        const Level *par = l >= 3 ? &g.T.lev[l - 1] : nullptr;
        j.pstart = par ? par->start : nullptr;
        j.pcount = par ? par->count : nullptr;
        j.ckey = par ? g.T.lev[l].key : nullptr;
        j.npar = par ? par->n : 0;
        j.ntiles = par ? 8 * ((j.npar + TC_ROWS - 1) / TC_ROWS) : (ntb + TC_ROWS - 1) / TC_ROWS;
        titems += j.ntiles * M2L_NSLICE;
        tjobs.push_back(j);
      } else if (dofree) {
        add(nullptr, nullptr, ntb, g.vfree[l], tb.cls_free, g.Mfree[l], g.op_free[l], part, 1, 0,
            l >= 3 ? &g.T.lev[l - 1] : nullptr, &g.T.lev[l]);
      }
      if (react_far && g.vreact[l] && use_tc && g.ntypes <= 16) {
        TJob j;
        pack(j, g.Mimg[l], g.I.lev[l], g.tmask[l], g.a, g.op_react[l], 1, g.ntypes, g.used[l], TC_NREACT);
        j.vlist = g.vreact[l]; j.slot0 = M2L_NSLICE;
        j.pstart = nullptr; j.pcount = nullptr; j.ckey = nullptr; j.npar = 0;
        // a row is one layer of boxes: at most 4^l of them
        j.ntiles = (std::min<int64_t>(ntb, (int64_t)1 << (2 * l)) + TC_ROWS - 1) / TC_ROWS;
        for (int kt = 0; kt < 2 * c.ws + 1; ++kt) {
          j.cls_of = tb.tc_react + ((g.a - 1) * NKT + kt) * NOFF;
          j.tlist = g.rows[l] + (size_t)kt * ntb; j.d_ntl = g.nrows[l] + kt;
          j.item0 = titems;
          titems += j.ntiles * M2L_NSLICE;
          tjobs.push_back(j);
        }
      } else if (react_far && g.vreact[l]) {
        for (int kt = 0; kt < 2 * c.ws + 1; ++kt)
          add(g.rows[l] + (size_t)kt * ntb, g.nrows[l] + kt, ntb, g.vreact[l],
              tb.cls_react + ((g.a - 1) * NKT + kt) * NOFF, g.Mimg[l], g.op_react[l], part, g.ntypes, M2L_NSLICE,
              nullptr, nullptr);
      }
    }
  }
  if (jobs.empty() && tjobs.empty()) return;
  if (!prow.empty()) {
    k_tc_pack_rows<<<(unsigned)row_items, 256, 0, c.stream>>>(upload_jobs(c, prow), (int)prow.size(), c.K, c.p, tc_nc, c.ws);
    LPB_LAUNCH();
    c.launches++;
    if (!pw.empty()) {
      launch_pack_w(c.p, upload_jobs(c, pw), (int)pw.size(), img_items, c.ws, c.stream);
      LPB_LAUNCH();
      c.launches++;
      c.images_ready = true;
    }
  }
  prof_mark(c, "m2l_prep");
  if (c.def.on && !tjobs.empty() && jobs.empty()) {
    // batched evaluation: the tensor-core M2L and the slot sums join a grouped launch
    c.def.nc = tc_nc;
    c.def.tc = tjobs;
    c.def.tc_items = titems;
    c.def.red = rjobs;
    c.def.red_elems = relem;
    return;
  }
  if (!tjobs.empty()) {
    TJob *dj = c.arena.get<TJob>(tjobs.size());
    LPB_CUDA(cudaMemcpyAsync(dj, tjobs.data(), sizeof(TJob) * tjobs.size(), cudaMemcpyHostToDevice, c.stream));
    launch_tc(c.p, dj, (int)tjobs.size(), titems, c.status, c.stream);
    LPB_LAUNCH();
    c.launches++;
    prof_mark(c, "m2l_tc");
  }
  auto launch_reduce = [&]() {
    RJob *dr = c.arena.get<RJob>(rjobs.size());
    LPB_CUDA(cudaMemcpyAsync(dr, rjobs.data(), sizeof(RJob) * rjobs.size(), cudaMemcpyHostToDevice, c.stream));
    k_m2l_reduce<T><<<(unsigned)((relem + 255) / 256), 256, 0, c.stream>>>(dr, (int)rjobs.size(), c.K);
    LPB_LAUNCH();
    c.launches++;
  };
  if (jobs.empty()) {
    launch_reduce();
    return;
  }
  if (c.K <= F32_KR) {
    // re-count items with the larger tile of the asynchronous FP32 kernel
    int64_t it = 0;
    for (auto &j : jobs) {
      j.item0 = it;
      it += m2l_tiles(j, F32_TT) * M2L_NSLICE;
    }
    const size_t smem = m2l_f32_smem(c.K);
    // the largest K of this kernel, p = 11; the K = 80 that its rows are padded to would ask for more than a block has
    LPB_ATTR_ONCE(k_m2l_f32, m2l_f32_smem(12 * 13 / 2));
    XJob *dj = c.arena.get<XJob>(jobs.size());
    LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(XJob) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
    k_m2l_f32<<<(unsigned)it, 256, smem, c.stream>>>(dj, (int)jobs.size(), (const float *)tb.rot, c.K);
    LPB_LAUNCH();
    c.launches++;
    prof_mark(c, "m2l_simt");
    launch_reduce();
    return;
  }
  if (c.K <= 128) launch_m2l_t<T, TPT, 8>(c, jobs, items);
  else launch_m2l_t<T, TPT, 10>(c, jobs, items);
  launch_reduce();
}

// the FP64 free-space near field of every group, one launch
static void near_free_f64(Ctx &c, std::vector<Group> &groups, double *phi, double *field) {
  std::vector<P64Job> jobs;
  int64_t blocks = 0;
  for (auto &g : groups) {
    if (!(g.is_free && (g.parts & 1))) continue;
    const Level &Lf = g.T.lev[g.Df];
    if (!Lf.n) continue;
    P64Job j;
    j.bstart = Lf.pstart; j.bcount = Lf.pcount; j.ulist = g.ufree;
    j.x = g.T.x; j.y = g.T.y; j.z = g.T.z; j.q = g.T.q; j.src = g.T.src;
    j.lam = c.md.lam[g.l];
    j.scale = 1.0 / (4.0 * PI * c.md.eps[g.l]);
    j.ce = (double)(-(long double)j.lam * 1.44269504088896340736L * EXP_TAB);
    const double rmax = 700.0 / j.lam, r2 = std::min(rmax * rmax, 1e300);
    uint64_t u;
    std::memcpy(&u, &r2, sizeof u);
    // (high word - 0x00100000) <= hi_max: normal numbers up to the cut
    j.hi_max = std::max((uint32_t)(u >> 32), 0x00100000u) - 0x00100000u;
    j.nb = (uint32_t)Lf.n;
    j.block0 = blocks;
    jobs.push_back(j);
    blocks += Lf.n;
  }
  if (jobs.empty()) return;
  P64Job *dj = c.arena.get<P64Job>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(P64Job) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
  if (field) k_p2p_free_f64<true><<<(unsigned)blocks, 32 * P64_WARPS, 0, c.stream>>>(dj, (int)jobs.size(), phi, field);
  else k_p2p_free_f64<false><<<(unsigned)blocks, 32 * P64_WARPS, 0, c.stream>>>(dj, (int)jobs.size(), phi, field);
  LPB_LAUNCH();
  c.launches++;
}

// L2L (adding the parent's shifted expansion), L2P and the reaction near field of every group
template <typename T>
static void downward_t(Ctx &c, std::vector<Group> &groups, double *phi, double *field) {
  const int K = c.K;
  const Tables &tb = sizeof(T) == 8 ? g_tab_d[c.device] : g_tab_f[c.device];
  int Dmax = 2;
  for (auto &g : groups) Dmax = std::max(Dmax, g.D);
  for (int l = 3; l <= Dmax; ++l) {
    std::vector<L2LJob> jobs;
    int64_t items = 0;
    for (auto &g : groups) {
      if (l > g.D || !g.T.lev[l].n) continue;
      const Level &P = g.T.lev[l - 1];
      jobs.push_back(L2LJob{P.start, P.count, g.T.lev[l].key, g.Lt[l - 1], g.op_l2l[l], g.Lt[l], P.n, items});
      items += P.n;
    }
    if (jobs.empty()) continue;
    k_l2l<T><<<(unsigned)items, oct_threads(K, c.p, items), oct_smem<T>(K, c.p), c.stream>>>(
        upload_jobs(c, jobs), (int)jobs.size(), (const T *)tb.rot4, K, c.p);
    LPB_LAUNCH();
    c.launches++;
  }
  // the two groups of a layer add into the same outputs: one side after the other
  for (int a = 1; a <= 2; ++a) {
    std::vector<L2PJob> dense, sparse;
    int64_t nd = 0, ns = 0;
    for (auto &g : groups) {
      const Level &Lv = g.T.lev[g.D];
      if (g.a != a || !Lv.n) continue;
      L2PJob j;
      j.bkey = Lv.key; j.bstart = Lv.start; j.bcount = Lv.count; j.pbox = g.T.pbox;
      j.x = g.T.x; j.y = g.T.y; j.z = g.T.z; j.src = g.T.src; j.L = g.Lt[g.D]; j.geo = geo_at<T>(g, g.D);
      j.lam = c.md.lam[g.l];
      if (g.T.np < P2M_SPARSE * Lv.n) {
        j.n = g.T.np;
        j.item0 = ns;
        ns += (j.n + 127) / 128;
        sparse.push_back(j);
      } else {
        j.n = Lv.n;
        j.item0 = nd;
        nd += (j.n + 3) / 4;
        dense.push_back(j);
      }
    }
    PT_DISPATCH(launch_l2p, c, dense, sparse, nd, ns, phi, field);
  }
  for (auto &g : groups) {
    const bool react_near = (g.parts & 2) && g.I.np > 0 && !(g.parts & 4);
    if (!react_near || !g.ureact || !g.nodes) continue;
    const int D = g.D;
    k_p2p_react<T><<<(unsigned)g.T.lev[D].n, P2P_THREADS, 0, c.stream>>>(
        g.T.lev[D].d_n, g.T.lev[D].key, g.T.lev[D].start, g.T.lev[D].count, g.ureact, g.T.x, g.T.y, g.T.z, g.T.src,
        g.I.lev[D].start, g.I.lev[D].count, g.I.x, g.I.y, g.I.z, g.I.q, g.I.key, geo_at<T>(g, D), g.dI,
        g.a == 1 ? 1.0 : -1.0, g.nodes, g.nq, phi, field);
    LPB_LAUNCH();
    c.launches++;
  }
}

// one launch of the FP32 free-space near field over the jobs (block0 renumbered from 0)
static void launch_p2p(Ctx &c, const std::vector<P2PJob> &jobs, int64_t blocks, cudaStream_t st) {
  if (jobs.empty() || blocks <= 0) return;
  P2PJob *dj = c.arena.get<P2PJob>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(P2PJob) * jobs.size(), cudaMemcpyHostToDevice, st));
  if (jobs[0].field) k_p2p_free_f32<true><<<(unsigned)blocks, 32 * P2P_WARPS, 0, st>>>(dj, (int)jobs.size());
  else k_p2p_free_f32<false><<<(unsigned)blocks, 32 * P2P_WARPS, 0, st>>>(dj, (int)jobs.size());
  LPB_LAUNCH();
  c.launches++;
}

void run_fmm_front(Ctx &c, std::vector<Group> &groups) {
  c.def.nc = 0;
  c.def.tc.clear();
  c.def.red.clear();
  c.def.tc_items = c.def.red_elems = 0;
  const bool d = c.opts.precision == LPBFMM_FP64;
  // the free-space operators (far stream) are complete before the upward pass
  if (c.ev_free) LPB_CUDA(cudaStreamWaitEvent(c.stream, c.ev_free, 0));
  d ? upward_t<double>(c, groups) : upward_t<float>(c, groups);
  prof_mark(c, "upward");
  // the reaction tables and operators (side stream) are complete before any M2L
  if (c.ev_join) LPB_CUDA(cudaStreamWaitEvent(c.stream, c.ev_join, 0));
  d ? m2l_all_f64(c, groups) : m2l_all_f32(c, groups);
  prof_mark(c, "m2l");
}

void run_near_free(Ctx &c, std::vector<Group> &groups, double *phi, double *field, cudaStream_t st) {
  c.def.p2p.clear();
  c.def.p2p_blocks = 0;
  c.p2p_timed = false;
  if (c.opts.precision == LPBFMM_FP64) return;
  OnStream on(c, st);
  for (auto &g : groups) {
    if (!(g.is_free && (g.parts & 1))) continue;
    const Level &Lf = g.T.lev[g.Df];
    const unsigned nb = (unsigned)Lf.n;
    if (!nb) continue;
    const int64_t np = g.T.np;
    float *pts = c.arena.get<float>((size_t)np * 7);
    k_split_points<<<nb, 64, 0, c.stream>>>(Lf.d_n, Lf.key, Lf.pstart, Lf.pcount, g.T.x, g.T.y, g.T.z, g.T.q,
                                             geo_at<float>(g, g.Df), pts, np);
    LPB_LAUNCH();
    c.launches++;
    const double hD = g.h(g.Df);
    P2PJob j;
    j.d_nb = Lf.d_n; j.bkey = Lf.key; j.bstart = Lf.pstart; j.bcount = Lf.pcount; j.ulist = g.ufree;
    j.pts = pts; j.ld = np; j.src = g.T.src; j.phi = phi; j.field = field;
    j.scale = 1.0 / (4.0 * PI * c.md.eps[g.l]);
    j.hh = (float)hD; j.hl = (float)(hD - (double)j.hh); j.lam = (float)c.md.lam[g.l];
    j.block0 = c.def.p2p_blocks;
    c.def.p2p.push_back(j);
    c.def.p2p_blocks += nb;
  }
  if (!c.def.on && !c.def.p2p.empty()) {
    LPB_CUDA(cudaEventRecord(c.ev_p2p[0], c.stream));
    launch_p2p(c, c.def.p2p, c.def.p2p_blocks, c.stream);
    LPB_CUDA(cudaEventRecord(c.ev_p2p[1], c.stream));
    c.p2p_timed = true;
    c.def.p2p.clear();
    c.def.p2p_blocks = 0;
  }
}

void run_fmm_back(Ctx &c, std::vector<Group> &groups, double *phi, double *field) {
  const bool d = c.opts.precision == LPBFMM_FP64;
  // the far field (its own stream) and the free-space near field, which adds into the same
  // outputs, are complete first
  if (c.far_async) LPB_CUDA(cudaStreamWaitEvent(c.stream, c.ev_far, 0));
  if (c.near_async) LPB_CUDA(cudaStreamWaitEvent(c.stream, c.ev_near, 0));
  d ? downward_t<double>(c, groups, phi, field) : downward_t<float>(c, groups, phi, field);
  if (d) near_free_f64(c, groups, phi, field);
  prof_mark(c, "downward");
}

void launch_deferred(const std::vector<Ctx *> &cs, int stage, cudaStream_t st) {
  if (cs.empty()) return;
  Ctx &c0 = *cs[0];
  if (stage == 0) {
    // per truncation order (the kernels take K and p as arguments): one tensor-core M2L launch,
    // then one launch of the slot sums (FP32 partials: the tensor-core path runs in mixed mode)
    std::vector<int> orders;
    for (Ctx *c : cs)
      if (c->def.nc && std::find(orders.begin(), orders.end(), c->p) == orders.end()) orders.push_back(c->p);
    for (int p : orders) {
      std::vector<TJob> tj;
      std::vector<RJob> red;
      int64_t items = 0, relem = 0;
      Ctx *lead = nullptr;
      for (Ctx *c : cs) {
        if (!c->def.nc || c->p != p) continue;
        if (!lead) lead = c;
        for (TJob j : c->def.tc) {
          j.item0 += items;
          tj.push_back(j);
        }
        items += c->def.tc_items;
        for (RJob r : c->def.red) {
          r.e0 += relem;
          red.push_back(r);
        }
        relem += c->def.red_elems;
      }
      TJob *dj = c0.arena.get<TJob>(tj.size());
      LPB_CUDA(cudaMemcpyAsync(dj, tj.data(), sizeof(TJob) * tj.size(), cudaMemcpyHostToDevice, st));
      launch_tc(p, dj, (int)tj.size(), items, c0.status, st);
      LPB_LAUNCH();
      c0.launches++;
      if (!red.empty()) {
        RJob *dr = c0.arena.get<RJob>(red.size());
        LPB_CUDA(cudaMemcpyAsync(dr, red.data(), sizeof(RJob) * red.size(), cudaMemcpyHostToDevice, st));
        k_m2l_reduce<float><<<(unsigned)((relem + 255) / 256), 256, 0, st>>>(dr, (int)red.size(), lead->K);
        LPB_LAUNCH();
        c0.launches++;
      }
    }
  } else {
    std::vector<P2PJob> pj;
    int64_t blocks = 0;
    for (Ctx *c : cs) {
      for (P2PJob j : c->def.p2p) {
        j.block0 += blocks;
        pj.push_back(j);
      }
      blocks += c->def.p2p_blocks;
    }
    launch_p2p(c0, pj, blocks, st);
  }
}

}  // namespace lpb
