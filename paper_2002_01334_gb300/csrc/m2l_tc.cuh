// Tensor-core multipole-to-local of the mixed mode (included by fmm.cu).
#pragma once

// ---------------------------------------------------------------------------------------
// M2L on the tensor cores (tcgen05), free space and reaction, mixed mode, p <= 10.
//
// Every translation of this library has the azimuth-factored form
//     X = e^{i m phi} M,   Y_nm = sum P_{nm,nu mu} Re X_{nu mu} + i sum Q_{nm,nu mu} Im X_{nu mu},
//     L_nm += e^{-i m phi} Y_nm
// with real class operators P, Q that do not depend on the azimuth phi of the offset.  Write
// phi = s phi_c + k pi / 2 with s = +-1 and phi_c in [0, pi/4] the azimuth of (a, b), 0 <= b <= a (the
// offset's |dx|, |dy| in order).  Then with M' = i^{mk} M, conjugated if s < 0,
//     Z = D(-phi_c) (P, Q) D(phi_c) M',   L += i^{-mk} (Z, conjugated if s < 0),
// so one real matrix W per canonical pair (a, b) serves all eight azimuths of the pair, and what is left
// of the rotations are exchanges and sign changes of real and imaginary parts: exact, and the same
// on the two halves of a split number.  In real form: R = 2K - (p+1) coordinates, for m > 0 the pair
// (Re, Im) in adjacent columns, then the real parts of the m = 0 coefficients (their imaginary
// parts vanish for real charges), padded to N = 32 NC columns.
//
// Operands are FP16 pairs, value = 2^-e (hi + lo): 11 significand bits each, 22 in all, as in a TF32 pair, in
// half the bytes and at twice the tensor rate.  FP16's short exponent is met by one power of
// two per source row and per operator that brings the largest entry to [2^13, 2^14): an entry keeps
// its 22 bits down to 2^-17 of the largest, and below that errs by 2^-39 of it.  The product is
// hi hi + hi lo + lo hi, accumulated in FP32 in a fresh TMEM accumulator per (offset, source type) and
// folded into FP32 registers (the tensor core's accumulation loses digits over long chains, measured; a dot
// product of 32 NC terms does not).
// ---------------------------------------------------------------------------------------
// Column order.  A quarter turn acts on a coefficient by i^m, so columns are ordered by m mod 4, in the same
// segments in each half of the N columns: pairs (Re, Im) with m = 1, 2, 3, 0 mod 4 (m > 0), then pairs
// of m = 0 real parts, each segment of seg pairs per half (its last ones may be padding).  The fold then needs two scalars
// per segment and step, known at compile time for every column.
__host__ __device__ constexpr int tc_count(int p, int c) {  // coefficients 1 <= m <= n <= p with m = c mod 4
  int k = 0;
  for (int m = 1; m <= p; ++m)
    if (m % 4 == c) k += p - m + 1;
  return k;
}
// pairs per half of segment g = 0..4 (m = 1, 2, 3, 0 mod 4; m = 0)
__host__ __device__ constexpr int tc_seg(int p, int g) {
  return g < 4 ? (tc_count(p, (g + 1) & 3) + 1) / 2 : ((p + 2) / 2 + 1) / 2;
}
__host__ __device__ constexpr int tc_chunks(int p) { return ((p + 1) * (p + 1) + 31) / 32; }  // R = (p + 1)^2
// segment of pair j of a half; 5: padding
__host__ __device__ constexpr int tc_segment(int p, int j) {
  int g = 0;
  while (g < 5 && j >= tc_seg(p, g)) j -= tc_seg(p, g++);
  return g;
}
// column c -> half-representation index: >= 0 real part, <= -2 imaginary part of index (-code - 2),
// -1 padding
__host__ __device__ __forceinline__ int tc_remap(int c, int p) {
  const int half = 16 * tc_chunks(p), h = c / half;
  int j = (c % half) >> 1, g = 0;
  while (g < 5 && j >= tc_seg(p, g)) j -= tc_seg(p, g++);
  if (g == 5) return -1;
  int i = h * tc_seg(p, g) + j;  // index in the segment's list
  if (g == 4) {
    const int n = 2 * i + (c & 1);
    return n <= p ? n * (n + 1) / 2 : -1;
  }
  for (int m = g < 3 ? g + 1 : 4; m <= p; m += 4) {
    if (i < p - m + 1) {
      const int n = m + i, k = n * (n + 1) / 2 + m;
      return (c & 1) ? -k - 2 : k;
    }
    i -= p - m + 1;
  }
  return -1;
}

// canonical pairs (a, b), 0 <= b <= a <= OFF_R: index a (a + 1) / 2 + b
constexpr int NCAN = (OFF_R + 1) * (OFF_R + 2) / 2;
constexpr int TC_NFREE = NCAN * NDZ, TC_NREACT = NCAN * NKK;  // operator images of a level (per type)
__host__ __device__ __forceinline__ void can_decode(int ci, int &a, int &b) {
  a = 0;
  while ((a + 1) * (a + 2) / 2 <= ci) ++a;
  b = ci - a * (a + 1) / 2;
}
// (dx, dy) -> canonical pair index, quarter turns k and reflection (s < 0): the translation vector
// (-dx, -dy) turned back by k quarter turns is (a, s b)
__host__ __device__ __forceinline__ int can_of(int dx, int dy, int &k, bool &refl) {
  int x = -dx, y = -dy;
  for (k = 0; k < 3; ++k) {
    if (x >= (y < 0 ? -y : y)) break;
    const int t = x;  // a quarter turn back
    x = y;
    y = -t;
  }
  refl = y < 0;
  const int b = refl ? -y : y;
  return x * (x + 1) / 2 + b;
}
__constant__ float c_trig[NCAN][PMAX + 1][2];  // cos, sin of m phi_c
void upload_trig(cudaStream_t s) {
  static float h[NCAN][PMAX + 1][2];
  for (int ci = 0; ci < NCAN; ++ci) {
    int a, b;
    can_decode(ci, a, b);
    const double ph = b ? atan2((double)b, (double)a) : 0.0;
    for (int m = 0; m <= PMAX; ++m) {
      h[ci][m][0] = (float)cos(m * ph);
      h[ci][m][1] = (float)sin(m * ph);
    }
  }
  LPB_CUDA(cudaMemcpyToSymbolAsync(c_trig, h, sizeof h, 0, cudaMemcpyHostToDevice, s));
}

// exponent e with v 2^e in [2^13, 2^14); 0 for zero and for what is not finite
__device__ __forceinline__ int tc_exponent(float v) { return v > 0.f && v < INFINITY ? 13 - ilogbf(v) : 0; }
__device__ __forceinline__ void tc_split(float x, int e, __half &h, __half &l) {
  const float s = scalbnf(x, e);
  h = __float2half_rn(s);
  l = __float2half_rn(s - __half2float(h));
}

// W of one (canonical class, type) as the shared-memory image the MMA reads: NC K-chunks of 32
// columns, each N rows of 128 bytes [32 hi | 32 lo] in the 128-byte swizzled K-major layout, so that one
// bulk copy moves a chunk.  One CTA per image; classes that no far list uses are skipped.
// kind 0: free space (class (a, b), dz), 1: reaction (class (a, b), kk; used[] per (rho^2, kk)).  Every
// level of every group in one launch.
struct PackWJob {
  const float *ops;
  const uint8_t *used;
  unsigned char *wimg;
  float *wscale;
  int64_t item0;
  int kind, ntypes;
};
constexpr int PACKW_THREADS = 256;
template <int P>
__global__ void __launch_bounds__(PACKW_THREADS) k_tc_pack_w(const PackWJob *jobs, int nj, int ws) {
  constexpr int NC = tc_chunks(P), N = 32 * NC, K = (P + 1) * (P + 2) / 2;
  extern __shared__ float pq[];  // P, Q
  __shared__ int code[N];
  __shared__ float tc_[N], ts_[N];  // cos, sin of m phi_c of every column's coefficient
  __shared__ float red[PACKW_THREADS / 32];
  const PackWJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int kind = J.kind, ntypes = J.ntypes;
  const int ct = (int)((int64_t)blockIdx.x - J.item0), cls = ct / ntypes, tau = ct % ntypes;
  const int per = kind ? NKK : NDZ, ci = cls / per, sub = cls % per;
  int a, b;
  can_decode(ci, a, b);
  const int src = rho_index(a, b) * per + sub;  // the (rho^2, ...) class of the operators
  if (kind ? !J.used[src] : max(a, abs(sub - OFF_R)) <= ws) return;
  const float *op = J.ops + ((size_t)src * ntypes + tau) * 2 * K * K;
  float mx = 0.f;
  for (int e = threadIdx.x; e < 2 * K * K; e += blockDim.x) {
    const float v = op[e];
    pq[e] = v;
    mx = fmaxf(mx, fabsf(v));
  }
  for (int c = threadIdx.x; c < N; c += blockDim.x) {
    const int cd = tc_remap(c, P);
    const int m = cd == -1 ? 0 : cK.mof[cd >= 0 ? cd : -cd - 2];
    code[c] = cd;
    tc_[c] = c_trig[ci][m][0];
    ts_[c] = c_trig[ci][m][1];
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < PACKW_THREADS / 32; ++w) mx = fmaxf(mx, red[w]);
  // the entries of W are bounded by the largest of P and Q
  const int e2 = tc_exponent(mx);
  if (threadIdx.x == 0) J.wscale[ct] = scalbnf(1.f, -e2);
  // 2^e2 in two factors, each an ordinary number
  const float f1 = scalbnf(1.f, e2 / 2), f2 = scalbnf(1.f, e2 - e2 / 2);
  const float *Pm = pq, *Qm = pq + K * K;
  unsigned char *img = J.wimg + (size_t)ct * N * NC * 128;
  for (int e = threadIdx.x; e < N * (N / 2); e += blockDim.x) {
    const int r = e / (N / 2), cp = 2 * (e % (N / 2));  // row, first column of the pair
    const int ro = code[r], k0 = code[cp], k1 = code[cp + 1];
    float w0 = 0.f, w1 = 0.f;
    if (ro != -1 && k0 != -1) {
      const int i = ro >= 0 ? ro : -ro - 2;
      const float c_i = tc_[r], s_i = ts_[r];
      if (k1 <= -2) {  // (Re, Im) of coefficient k0
        const float c_k = tc_[cp], s_k = ts_[cp];
        const float Pv = Pm[i * K + k0], Qv = Qm[i * K + k0];
        if (ro >= 0) {
          w0 = c_i * Pv * c_k + s_i * Qv * s_k;
          w1 = s_i * Qv * c_k - c_i * Pv * s_k;
        } else {
          w0 = c_i * Qv * s_k - s_i * Pv * c_k;
          w1 = c_i * Qv * c_k + s_i * Pv * s_k;
        }
      } else {  // two m = 0 coefficients (or one and padding)
        const float f = ro >= 0 ? c_i : -s_i;
        w0 = f * Pm[i * K + k0];
        if (k1 >= 0) w1 = f * Pm[i * K + k1];
      }
    }
    w0 = w0 * f1 * f2;
    w1 = w1 * f1 * f2;
    const __half2 h = __floats2half2_rn(w0, w1);
    const float2 hf = __half22float2(h);
    const __half2 l = __floats2half2_rn(w0 - hf.x, w1 - hf.y);
    unsigned char *row = img + ((size_t)(cp >> 5) * N + r) * 128;
    const int by = (cp & 31) * 2;  // byte of the hi pair in the row
    *(__half2 *)(row + ((((by >> 4)) ^ (r & 7)) << 4) + (by & 15)) = h;
    *(__half2 *)(row + ((((by >> 4) + 4) ^ (r & 7)) << 4) + (by & 15)) = l;
  }
}

// source rows as split FP16 (per 32-column chunk [32 hi | 32 lo]), with the row's inverse power of two; rows
// of absent types are neither written nor read.  One warp per (box, type) row, every level of every group in one
// launch.  side: 0 free space; 1, 2 reaction side a: only image boxes within 2 ws box layers of the
// interface can be in a far list, the others are skipped.
struct PackRowJob {
  const float2 *M;
  const uint32_t *mask;  // types present (nullptr: all)
  const uint64_t *bkey;
  __half *rows;
  float *rscale;
  int64_t nrows, item0;
  int ntypes, lev, side;
};
__global__ void __launch_bounds__(256) k_tc_pack_rows(const PackRowJob *jobs, int nj, int K, int p, int NC, int ws) {
  __shared__ int code[128];
  const int N = 32 * NC, lane = threadIdx.x & 31;
  for (int c = threadIdx.x; c < N; c += blockDim.x) code[c] = tc_remap(c, p);
  __syncthreads();
  const PackRowJob &J = job_of(jobs, nj, (int64_t)blockIdx.x);
  const int64_t row = ((int64_t)blockIdx.x - J.item0) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= J.nrows) return;
  const int64_t box = row / J.ntypes;
  if (J.mask && !((J.mask[box] >> (int)(row % J.ntypes)) & 1u)) return;
  if (J.side) {
    const int iz = (int)compact3_(J.bkey[box]), half = 1 << (J.lev - 1);
    if ((J.side == 1 ? half - 1 - iz : iz - half) > 2 * ws) return;
  }
  float v[4], mx = 0.f;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    v[ch] = 0.f;
    if (ch < NC) {
      const int cd = code[ch * 32 + lane];
      if (cd != -1) {
        const float2 m = J.M[row * K + (cd >= 0 ? cd : -cd - 2)];
        v[ch] = cd >= 0 ? m.x : m.y;
      }
    }
    mx = fmaxf(mx, fabsf(v[ch]));
    if (v[ch] != v[ch]) mx = INFINITY;  // a NaN row stays one
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int e2 = tc_exponent(mx);
  __half *out = J.rows + row * 2 * N;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    if (ch >= NC) break;
    __half h, l;
    tc_split(v[ch], e2, h, l);
    out[ch * 64 + lane] = h;
    out[ch * 64 + 32 + lane] = l;
  }
  if (lane == 0) J.rscale[row] = scalbnf(1.f, -e2);
}

constexpr int TC_MAXSTEP = SLICE_OFFS * 2 * (MAXLAYER - 1);

constexpr int TC_ROWS = 128, TC_WORKERS = 256, TC_THREADS = TC_WORKERS + 64;
constexpr int TC_WAIT = 1 << 22;  // mbarrier polls before the kernel reports a timeout
constexpr int TC_NST = 6;         // stages of one K-chunk (A and W tiles)
constexpr int TC_SCL = TC_NST + 2;

__host__ __device__ constexpr size_t tc_stage_bytes(int NC) { return (size_t)(TC_ROWS + 32 * NC) * 128; }
static size_t tc_smem(int NC) { return TC_NST * tc_stage_bytes(NC) + 1024; }

__device__ __forceinline__ uint64_t to_global(const void *p) {
  uint64_t g;
  asm("cvta.to.global.u64 %0, %1;" : "=l"(g) : "l"(p));
  return g;
}
// one arrival that also announces tx bytes to come by bulk copies
__device__ __forceinline__ void mbar_expect_tx(uint64_t *mbar, uint32_t bytes) {
  asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(
                   tc::smem_u32(mbar)),
               "r"(bytes)
               : "memory");
}
// bulk copy of bytes (multiple of 16, both addresses 16-byte aligned) global -> shared, completing
// on mbar
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   tc::smem_u32(dst)),
               "l"(to_global(src)), "r"(bytes), "r"(tc::smem_u32(mbar))
               : "memory");
}

// A CTA owns 128 target boxes (an octant tile, or a run of a target list) and one dx-slice of the offsets;
// its steps are the (offset, source type) pairs that some row of the tile needs.  8 worker warps stage
// the source rows (global -> registers, exchange and signs, -> the swizzled A tile; eight lanes read one
// row's 128-byte chunk, a warp 16 rows) a whole step at a time, and fold the previous step's
// accumulator while the next step's rows are on their way; warp 8 issues the MMAs, warp 9 the bulk
// copies of the operator chunks.
template <int P>
__global__ void __launch_bounds__(TC_THREADS, 1) k_m2l_tc(const TJob *jobs, int njobs, int *status) {
  constexpr int NC = tc_chunks(P), N = 32 * NC, NST = TC_NST, K = (P + 1) * (P + 2) / 2;
  constexpr int TCOLS = 2 * N <= 32 ? 32 : (2 * N <= 64 ? 64 : (2 * N <= 128 ? 128 : 256));
  static_assert(2 * N <= 256, "two accumulators of N columns");
  static_assert(NC <= NST, "a step's chunks stay staged until its last products");
  constexpr uint32_t SA = TC_ROWS * 128, SB = N * 128;  // bytes of one A / W chunk tile
  extern __shared__ __align__(16) unsigned char tcsm[];  // base rounded up to 1024 below
  unsigned char *sbase = (unsigned char *)(((uintptr_t)tcsm + 1023) & ~(uintptr_t)1023);
  __shared__ int tid_[TC_ROWS];
  __shared__ int steps[TC_MAXSTEP];  // (offset << 4) | source type
  __shared__ int remap_s[N], mcol[N];  // coordinate -> half index code; m of that coefficient
  __shared__ int nsteps;
  __shared__ unsigned tmk[SLICE_OFFS];  // per offset of the slice: the source types some row needs
  // exchange and signs of every column pair on the way in, for the slice's 11 (dx, dy): a byte
  // permutation and an XOR of the FP16 pair
  __shared__ __align__(16) uint2 win[OFF_D][N / 2];
  __shared__ int quarter[OFF_D], reflect[OFF_D], cls_s[SLICE_OFFS];
  // row scale x operator scale of the steps in flight: a warp stages at most NST chunks ahead of the
  // slowest warp, whose fold is one step behind (7 steps at one chunk per step)
  __shared__ float scl[TC_SCL][TC_ROWS];
  // full[b]: the worker warps have staged buffer b; wfull[b]: its operator chunk has landed; empty[b]: its
  // MMAs are done; accbar[a]: a step's MMAs into accumulator a are done; foldbar[a]: the workers have read it; done: every MMA
  __shared__ uint64_t full[NST], empty[NST], accbar[2], foldbar[2], wfull[NST], done;
  __shared__ uint32_t tbase;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].item0 <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const TJob &J = jobs[lo];
  // the fields the pipeline reads, in registers: the inline-assembly memory clobbers of the
  // barrier and copy instructions would otherwise make the compiler reload them from global
  // memory after every one
  const unsigned char *const Jrows = (const unsigned char *)J.rows, *const Jwimg = (const unsigned char *)J.wimg;
  const float *const Jrs = J.rscale, *const Jws = J.wscale;
  const int32_t *const Jvlist = J.vlist, *const Jcls = J.cls_of;
  const uint32_t *const Jtm = J.tmask;
  const int64_t local = (int64_t)blockIdx.x - J.item0;
  // slice-major: the CTAs resident at one time share a dx-slice, hence the operator classes of
  // its offsets, which then stay in L2 (a level's reaction operators alone exceed it)
  const int64_t ntiles = J.ntiles;
  const int slice = (int)(local / ntiles);
  const int64_t ti = local % ntiles;
  const int64_t ntl = J.tlist ? (int64_t)*J.d_ntl : J.ntb;
  if (J.pstart ? (ti >> 3) * TC_ROWS >= J.npar : ti * TC_ROWS >= ntl) return;
  // worker thread (tid < TC_WORKERS) in the fold = (row, half): row = target slot and TMEM lane, half =
  // which half of the accumulator columns
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = tid & (TC_ROWS - 1), hf = (tid >> 7) & 1;
  const bool worker = tid < TC_WORKERS;
  const int ntypes = J.ntypes;
  for (int c = tid; c < N; c += TC_THREADS) {
    const int code = tc_remap(c, P);
    remap_s[c] = code;
    mcol[c] = code == -1 ? 0 : cK.mof[code >= 0 ? code : -code - 2];
  }
  if (tid < TC_ROWS) {
    int t = -1;
    if (J.tlist) {
      const int64_t j = ti * TC_ROWS + tid;
      if (j < ntl) t = J.tlist[j];
    } else if (J.pstart) {
      const int oct = (int)(ti & 7);
      const int64_t par = (ti >> 3) * TC_ROWS + tid;
      if (par < J.npar) {
        const uint32_t s0 = J.pstart[par], n = J.pcount[par];
        for (uint32_t k = 0; k < n; ++k)
          if ((int)(J.ckey[s0 + k] & 7ull) == oct) t = (int)(s0 + k);
      }
    } else {
      const int64_t j = ti * TC_ROWS + tid;
      if (j < J.ntb) t = (int)j;
    }
    tid_[tid] = t;
  }
  for (int k = tid; k < SLICE_OFFS; k += TC_THREADS) {
    tmk[k] = 0u;
    cls_s[k] = Jcls[slice * SLICE_OFFS + k];
  }
  __syncthreads();
  // which types each offset of the slice needs: a warp reads whole list rows
  constexpr int KB = (SLICE_OFFS + 31) / 32;
  {
    unsigned acc[KB];
#pragma unroll
    for (int b = 0; b < KB; ++b) acc[b] = 0u;
#pragma unroll 2
    for (int r = warp; r < TC_ROWS; r += TC_THREADS / 32) {
      const int t = tid_[r];
      if (t < 0) continue;
#pragma unroll
      for (int b = 0; b < KB; ++b) {
        const int k = 32 * b + lane;
        const int sb = k < SLICE_OFFS ? Jvlist[(size_t)t * NOFF + slice * SLICE_OFFS + k] : -1;
        if (sb >= 0) acc[b] |= Jtm ? Jtm[sb] : 1u;
      }
    }
#pragma unroll
    for (int b = 0; b < KB; ++b) {
      const int k = 32 * b + lane;
      if (acc[b] && cls_s[k] >= 0) atomicOr(&tmk[k], acc[b]);
    }
  }
  for (int e = tid; e < OFF_D * (N / 2); e += TC_THREADS) {
    const int dyi = e / (N / 2), j = e % (N / 2), m = mcol[2 * j];
    int k;
    bool refl;
    can_of(slice - OFF_R, dyi - OFF_R, k, refl);
    const int q = (m * k) & 3;
    const bool pair = m > 0;
    // in: i^q (re, im), then conjugated: q = 1 (-im, re), 2 (-re, -im), 3 (im, -re)
    const unsigned x = (q == 1 ? 0x8000u : q == 2 ? 0x80008000u : q == 3 ? 0x80000000u : 0u) ^
                       (pair && refl ? 0x80000000u : 0u);
    win[dyi][j] = make_uint2((q & 1) ? 0x1032u : 0x3210u, x);
    if (j == 0) {
      quarter[dyi] = k;
      reflect[dyi] = refl;
    }
  }
  __syncthreads();
  if (warp == 0) {  // the step list, in (offset, type) order
    int n = 0;
    for (int b = 0; b < KB; ++b) {
      const int k = 32 * b + lane;
      const unsigned m = k < SLICE_OFFS ? tmk[k] & ((1u << ntypes) - 1u) : 0u;
      int x = __popc(m);
      const int c = x;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      int at = n + x - c;
      for (unsigned r = m; r; r &= r - 1) steps[at++] = ((slice * SLICE_OFFS + k) << 4) | (__ffs(r) - 1);
      n += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) nsteps = n;
  }
  __syncthreads();
  const int ns = nsteps;
  if (ns == 0) return;
  if (warp == 0) tc::tmem_alloc(&tbase, TCOLS);
  if (tid == 0) {
    for (int b = 0; b < NST; ++b) {
      tc::mbar_init(&full[b], TC_WORKERS / 32);
      tc::mbar_init(&empty[b], 1);
      tc::mbar_init(&wfull[b], 1);
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(&accbar[a], 1);
      tc::mbar_init(&foldbar[a], TC_WORKERS / 32);
    }
    tc::mbar_init(&done, 1);
    tc::mbar_fence_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  // a warp reads the TMEM lanes of its quarter, 32 (warp % 4) .. + 31
  const uint32_t tmem = tbase, lanebase = (uint32_t)((warp & 3) * 32) << 16;
  const int S = ns * NC;  // stages: (step, K-chunk)
  bool fail = false;
  if (worker) {
    const int myt = tid_[row];
    constexpr int NH = N / 2;  // accumulator columns per thread
    float racc[NH];
#pragma unroll
    for (int j = 0; j < NH; ++j) racc[j] = 0.f;
    // racc += the accumulator of step i, scaled, after the exchange and signs of the way out:
    // i^{-q} of (zr, s zi), q = m k mod 4: q = 1 (s zi, -zr), 2 (-zr, -s zi), 3 (-s zi, zr)
    auto fold = [&](int i) -> bool {
      // warp-uniform, so that the barriers below are met by whole warps also after a timeout
      const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&accbar[i & 1], (uint32_t)((i >> 1) & 1), TC_WAIT));
      if (!ok) return false;
      tc::fence_after();
      const int dyi = (steps[i] >> 4) / OFF_D % OFF_D, k = quarter[dyi];
      const float sc = scl[i % TC_SCL][row], s = reflect[dyi] ? -sc : sc;
      // per segment: factor into the real and the imaginary part (exchanged for odd m and odd k)
      const float sg = k & 2 ? -1.f : 1.f;  // k = 2, 3
      float fr[5], fi[5];
      if (k & 1) {
        fr[0] = sg * s; fi[0] = -sg * sc;   // m = 1: q = k
        fr[1] = -sc; fi[1] = -s;            // m = 2: q = 2
        fr[2] = -sg * s; fi[2] = sg * sc;   // m = 3: q = 3 k
      } else {
        fr[0] = fr[2] = sg * sc; fi[0] = fi[2] = sg * s;
        fr[1] = sc; fi[1] = s;
      }
      fr[3] = sc; fi[3] = s;
      fr[4] = fi[4] = sc;
      const uint32_t at = tmem + lanebase + (uint32_t)((i & 1) * N + hf * NH);
      auto sweep = [&](auto odd) {
#pragma unroll
        for (int c1 = 0; c1 < NH; c1 += 16) {
          uint32_t v[16];
          tc::tmem_ld16(at + (uint32_t)c1, v);
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const int g = tc_segment(P, (c1 + j) / 2);
            if (g == 5) continue;
            const float vr = __uint_as_float(v[j]), vi = __uint_as_float(v[j + 1]);
            const bool x = decltype(odd)::value && (g == 0 || g == 2);
            racc[c1 + j] = fmaf(fr[g], x ? vi : vr, racc[c1 + j]);
            racc[c1 + j + 1] = fmaf(fi[g], x ? vr : vi, racc[c1 + j + 1]);
          }
        }
      };
      if (k & 1) sweep(std::true_type());
      else sweep(std::false_type());
      tc::fence_before();
      return true;
    };
    // staging: lane = (row of a group of 4, 16-byte unit); lanes 0..15 also look up the sources of the warp's
    // 16 rows, the list entry two steps and the type mask one step ahead of use
    const int r4 = lane >> 3, un = lane & 7, row0 = warp * 16;
    const int lt = tid_[row0 + (lane & 15)];
    const int32_t *const lrow = Jvlist + (size_t)(lt >= 0 ? lt : 0) * NOFF;
    auto src_of = [&](int i) { return i < ns && lt >= 0 ? lrow[steps[i] >> 4] : -1; };
    int s1 = src_of(0), s2 = src_of(1);                // sources of the next step and the one after
    unsigned m1 = s1 >= 0 ? (Jtm ? Jtm[s1] : 1u) : 0u;              // type mask of the next step's source
    float rs = 0.f, wsc = 0.f;                         // scales of the loaded step (lanes 0..15)
    uint4 buf[NC][4];                                  // the loaded step: per chunk, one unit of four rows
    auto load = [&](int i) {
      const int tau = steps[i] & 15;
      const int rr = s1 >= 0 && ((m1 >> tau) & 1u) ? s1 * ntypes + tau : -1;
      rs = rr >= 0 ? Jrs[rr] : 0.f;
      wsc = Jws[(size_t)cls_s[(steps[i] >> 4) - slice * SLICE_OFFS] * ntypes + tau];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int r = __shfl_sync(0xffffffffu, rr, 4 * g + r4);
        const uint4 *const at = (const uint4 *)(Jrows + (size_t)(r >= 0 ? r : 0) * (NC * 128)) + un;
#pragma unroll
        for (int kc = 0; kc < NC; ++kc) buf[kc][g] = r >= 0 ? __ldg(at + kc * 8) : make_uint4(0u, 0u, 0u, 0u);
      }
      s1 = s2;
      m1 = s1 >= 0 ? (Jtm ? Jtm[s1] : 1u) : 0u;
      s2 = src_of(i + 2);
    };
    load(0);
    for (int i = 0; i < ns; ++i) {
      // exchange, signs, store into the A tiles.  One proxy fence per step, before the next step's loads are
      // issued: the fence waits for the thread's loads in flight (a fence per chunk beside prefetched
      // loads cost an L2 latency per chunk, 8.3k clocks a step at N = 1M)
      const uint4 *wi = (const uint4 *)&win[(steps[i] >> 4) / OFF_D % OFF_D][(un & 3) * 4];
#pragma unroll
      for (int kc = 0; kc < NC; ++kc) {
        const int s = i * NC + kc, b = s % NST;
        if (s >= NST && !fail)
          fail = !__all_sync(0xffffffffu, tc::mbar_wait(&empty[b], (uint32_t)((s / NST - 1) & 1), TC_WAIT));
        if (fail) break;
        unsigned char *A = sbase + (size_t)b * tc_stage_bytes(NC);
        const uint4 c0 = wi[kc * 8], c1 = wi[kc * 8 + 1];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint4 x = buf[kc][g];
          x.x = __byte_perm(x.x, 0u, c0.x) ^ c0.y;
          x.y = __byte_perm(x.y, 0u, c0.z) ^ c0.w;
          x.z = __byte_perm(x.z, 0u, c1.x) ^ c1.y;
          x.w = __byte_perm(x.w, 0u, c1.z) ^ c1.w;
          *(uint4 *)(A + tc::swz16(row0 + 4 * g + r4, un)) = x;
        }
      }
      if (fail) break;
      if (lane < 16) scl[i % TC_SCL][row0 + lane] = rs * wsc;
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) {
#pragma unroll
        for (int kc = 0; kc < NC; ++kc) tc::mbar_arrive(&full[(i * NC + kc) % NST]);
      }
      if (i + 1 < ns) load(i + 1);
      if (i >= 1) {  // the accumulator of step i - 1 is reused by step i + 1
        if (!fold(i - 1)) {
          fail = true;
          break;
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&foldbar[(i - 1) & 1]);
      }
    }
    if (!fail && !fold(ns - 1)) fail = true;
    if (!fail && myt >= 0) {
      float2 *Lrow = J.L + ((size_t)myt * M2L_NSLOT + J.slot0 + slice) * K;
      if (hf == 0) atomicOr(&J.smask[myt], 1u << (J.slot0 + slice));
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        const int code = remap_s[hf * NH + j];
        if (code >= 0) {
          Lrow[code].x = racc[j];
          if (mcol[hf * NH + j] == 0) Lrow[code].y = 0.f;
        } else if (code <= -2) {
          Lrow[-code - 2].y = racc[j];
        }
      }
    }
  } else if (tid == TC_WORKERS) {
    // the MMA thread: a step's cross products (hi lo, lo hi) of every chunk as it is filled, by the workers and the bulk
    // copy, then its hi hi ones; a step starts once the workers have read the accumulator two steps back
    constexpr uint32_t IDESC = tc::idesc_f16(TC_ROWS, N);
    for (int si = 0; si < ns && !fail; ++si) {
      if (si >= 2 && !tc::mbar_wait(&foldbar[si & 1], (uint32_t)(((si - 2) >> 1) & 1), TC_WAIT)) {
        fail = true;
        break;
      }
      const uint32_t dacc = tmem + (uint32_t)((si & 1) * N);
      for (int kc = 0; kc < NC; ++kc) {
        const int sc = si * NC + kc, b = sc % NST;
        if (!tc::mbar_wait(&full[b], (uint32_t)((sc / NST) & 1), TC_WAIT) ||
            !tc::mbar_wait(&wfull[b], (uint32_t)((sc / NST) & 1), TC_WAIT)) {
          fail = true;
          break;
        }
        tc::fence_after();
        const uint32_t ah = tc::smem_u32(sbase + (size_t)b * tc_stage_bytes(NC)), wh = ah + SA;
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {  // 16 columns: 32 bytes of hi, their lo 64 bytes on
          const uint32_t o = kk * 32;
          tc::mma_f16(dacc, tc::sdesc(ah + o), tc::sdesc(wh + 64 + o), IDESC, (kc | kk) ? 1u : 0u);
          tc::mma_f16(dacc, tc::sdesc(ah + 64 + o), tc::sdesc(wh + o), IDESC, 1u);
        }
      }
      if (fail) break;
      for (int kc = 0; kc < NC; ++kc) {
        const int sc = si * NC + kc, b = sc % NST;
        const uint32_t ah = tc::smem_u32(sbase + (size_t)b * tc_stage_bytes(NC)), wh = ah + SA;
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) tc::mma_f16(dacc, tc::sdesc(ah + kk * 32), tc::sdesc(wh + kk * 32), IDESC, 1u);
        tc::commit(&empty[b]);
      }
      tc::commit(&accbar[si & 1]);
    }
    // no MMA may be in flight when the tensor memory is freed, also those of a step that a timeout cut short, whose chunks
    // no other barrier covers
    tc::commit(&done);
    if (!tc::mbar_wait(&done, 0u, TC_WAIT)) fail = true;
  } else if (tid == TC_WORKERS + 32) {
    // the operator chunks, one bulk copy per stage
    int issued = 0;
    for (int s = 0; s < S; ++s) {
      const int b = s % NST;
      if (s >= NST && !tc::mbar_wait(&empty[b], (uint32_t)((s / NST - 1) & 1), TC_WAIT)) {
        fail = true;
        break;
      }
      const int st = steps[s / NC];
      const size_t ct = (size_t)cls_s[(st >> 4) - slice * SLICE_OFFS] * ntypes + (st & 15);
      mbar_expect_tx(&wfull[b], SB);
      bulk_g2s(sbase + (size_t)b * tc_stage_bytes(NC) + SA, Jwimg + (ct * NC + s % NC) * SB, SB, &wfull[b]);
      issued = s + 1;
    }
    // no bulk copy may still be writing this CTA's shared memory when it exits
    for (int s = issued > NST ? issued - NST : 0; s < issued; ++s)
      tc::mbar_wait(&wfull[s % NST], (uint32_t)((s / NST) & 1), TC_WAIT);
  }
  if (fail) atomicExch(status, LPBFMM_ERR_TIMEOUT);
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, TCOLS);
}
